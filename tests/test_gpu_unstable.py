"""A string whose state became non-finite (SFD_EUNSTABLE) is not stepped any
further: later blocks are zeros and leave its time level, its sweep counts and
its state as they were, and no sample is written outside the block, in every
instance of the step function and in the shared-memory path.

The unstable bit is set in a checkpoint of an ordinary string (Scalars: two
floats, the time level, the next sample, the status), so the state itself is
finite and would go on giving samples if it were stepped."""

import struct

import numpy as np
import pytest

from paper_2311_18505_gb300 import workloads as W
from test_gpu_instances import string

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GUARD = 256   # floats on either side of a block, more than a block


@pytest.fixture(scope="module")
def sfd():
    from paper_2311_18505_gb300 import build as B
    B.build()
    from paper_2311_18505_gb300 import sfd as S
    return S


def state_offset(blob):
    """Where a checkpoint's Scalars begin (header, set-up record, descriptor)."""
    header = struct.calcsize("<8sIIQIIIIQQiiii")
    desc, _, record = struct.unpack_from("<III", blob, 28)
    return header + record + desc


def guarded_block(sfd, s, n):
    """The status code of the next n samples, the samples, and whether the
    memory on both sides is untouched."""
    buf = torch.full((2 * GUARD + n,), 7.0, device="cuda")
    out = buf[GUARD:GUARD + n]
    torch.cuda.synchronize()
    rc = sfd.lib().sfd_synthesize(s, n, out.data_ptr(), 1)
    torch.cuda.synchronize()
    y = buf.cpu().numpy()
    return rc, y[GUARD:GUARD + n], bool(np.all(y[:GUARD] == 7.0) and np.all(y[GUARD + n:] == 7.0))


@pytest.mark.parametrize("n_t,n_l,kind,factored,groups", [
    (90, 0, "bow", False, True),          # linear
    (90, 1, "hammer", False, True),       # nonlinear, no longitudinal grid
    (31, 33, "pluck", False, True),       # longitudinal rows in registers
    (90, 96, "bow", False, True),
    (150, 200, "bow", False, False),      # ... in shared memory, one warp
    (150, 200, "bow", False, True),       # ... a group of 4
    (288, 420, "hammer", False, True),    # ... a group of 8
    (160, 190, "pluck", True, True),      # factored longitudinal matrix
    (300, 100, "pluck", False, True),     # shared-memory path
])
def test_an_unstable_string_is_not_stepped_again(sfd, n_t, n_l, kind, factored, groups):
    ctx = sfd.sfd_ctx_create(0, None, 64 << 20)
    try:
        sfd.sfd_ctx_set_warp_pairs(ctx, groups)
        s = sfd.string_from_dict(ctx, string(n_t, n_l, kind, factored))
        sfd.sfd_synthesize(s, 40)
        blob = bytearray(sfd.sfd_string_save(s))
        sfd.sfd_string_destroy(s)
        struct.pack_into("<i", blob, state_offset(blob) + 24, 1)
        s = sfd.sfd_string_load(ctx, bytes(blob))
        level, first = sfd.sfd_string_position(s)
        stats, state = sfd.sfd_string_stats(s), sfd.sfd_string_delta_state(s)
        done = 0
        for n in (33, 64, 1):
            rc, y, clean = guarded_block(sfd, s, n)
            assert rc == sfd.SFD_EUNSTABLE and clean and np.all(y == 0.0)
            done += n
            assert sfd.sfd_string_position(s) == (level, first + done)
            assert sfd.sfd_string_stats(s)[1:] == stats[1:]
            assert all(np.array_equal(a, b) for a, b in zip(sfd.sfd_string_delta_state(s), state))
        sfd.sfd_string_destroy(s)
    finally:
        sfd.sfd_ctx_destroy(ctx)


def test_blocks_after_the_one_that_became_unstable(sfd):
    """The printed grid (N_t of the theta = 1 rule with theta = 0.70) grows
    without bound: the samples up to the failure, then zeros; the blocks that
    follow leave the time level of the failure."""
    d = W.make(grid_rule=1, sigma0=0.0, sigma1=0.0, n_samples=4000)
    ctx = sfd.sfd_ctx_create(0, None, 64 << 20)
    try:
        s = sfd.string_from_dict(ctx, d)
        rc, y, clean = guarded_block(sfd, s, 4000)
        assert rc == sfd.SFD_EUNSTABLE and clean and y[0] != 0.0 and y[-1] == 0.0
        level, stats = sfd.sfd_string_position(s)[0], sfd.sfd_string_stats(s)
        assert level < 4000
        for k in (1, 2):
            rc, y, clean = guarded_block(sfd, s, 100)
            assert rc == sfd.SFD_EUNSTABLE and clean and np.all(y == 0.0)
            assert sfd.sfd_string_position(s) == (level, 4000 + 100 * k)
            assert sfd.sfd_string_stats(s) == stats
        sfd.sfd_string_destroy(s)
    finally:
        sfd.sfd_ctx_destroy(ctx)
