"""Which adjoint kernel takes a string, and the edges of each kernel's range: a
tape whose strings alternate between the two kernels (one thread per row: up to
255 rows and a folded longitudinal matrix; four warps per string: the rest),
each string against the FP64 oracle's exact derivatives (complex step) and
against the same string in a tape of its own.

Tolerances, relative to |w| |dy/dp|, the largest the component can be for
weights w of that norm (random ones give some 1 / sqrt(N) of it).  Against the
oracle 1e-3: the adjoint differentiates the FP32 trajectory (rel-L2 1e-6 and
less), whose phase drifts by at most that times the 240 steps; a wrong row,
offset or entry of the job table is of order 1 / sqrt(N).  Against the string
alone 1e-7: the block's thread count changes the order of double-float sums,
and the solves end at a relative change of 1e-13."""

import numpy as np
import pytest

import oracle
from test_gpu_instances import string

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 240


def third_level(n_t, n_l, kind):
    """A longitudinal coupling just below the 1 % up to which it is folded: the
    reduction of that matrix takes all three levels."""
    d = string(n_t, n_l, kind)
    d["sigma1"] = 0.0049 * d["fs"] / n_l ** 2
    assert oracle.grid(d)[:2] == (n_t, n_l)
    return d


def strings():
    return [string(31, 33, "pluck"),              # row kernel, 30 rows
            string(300, 200, "pluck"),            # four warps: 299 rows
            string(256, 190, "hammer"),           # row kernel at its 255 rows
            string(160, 190, "pluck", True),      # four warps: factored longitudinal matrix
            string(130, 195, "hammer"),           # row kernel, 194 longitudinal rows on 160 threads (alone)
            string(257, 120, "pluck"),            # four warps: 256 rows
            third_level(100, 140, "pluck"),       # row kernel, three reduction levels
            string(120, 0, "hammer"),             # row kernel, linear
            third_level(200, 290, "hammer"),
            string(2, 2, "pluck"),                # one row of each grid
            string(290, 430, "hammer", True)]     # four warps, both reasons


def gradient(sfd, ctx, dicts, w, K, record):
    tape = sfd.sfd_tape_create(ctx, dicts, N, K)
    try:
        sfd.sfd_tape_set_record_forward(tape, record)
        y = torch.empty(len(dicts), N, device="cuda")
        sfd.sfd_tape_forward(tape, y)
        return y.cpu().numpy(), sfd.sfd_tape_backward(tape, w, len(dicts))
    finally:
        sfd.sfd_tape_destroy(tape)


@pytest.fixture(scope="module")
def reference():
    """The oracle's derivatives dy/dp of every string, and weights dJ/dy."""
    rng = np.random.default_rng(11)
    ds = strings()
    D = [np.array([oracle.complex_step(d, k, n=N, n_t=oracle.grid(d)[0], n_l=oracle.grid(d)[1])[1] for k in range(5)])
         for d in ds]
    return ds, D, rng.standard_normal((len(ds), N)).astype(np.float32)


@pytest.mark.parametrize("K,record", [(512, True), (100, False)])
def test_a_tape_of_both_kernels(reference, K, record):
    from paper_2311_18505_gb300 import sfd
    torch.cuda.init()
    ds, D, w = reference
    ctx = sfd.sfd_ctx_create(0, None, 128 << 20)
    try:
        y, g = gradient(sfd, ctx, ds, torch.from_numpy(w).cuda(), K, record)
        for i, d in enumerate(ds):
            ref = D[i] @ w[i].astype(np.float64)
            most = np.linalg.norm(w[i]) * np.linalg.norm(D[i], axis=1)
            assert np.all(np.abs(g[i] - ref) <= 1e-3 * most), (i, g[i], ref)
            y1, g1 = gradient(sfd, ctx, [d], torch.from_numpy(w[i:i + 1]).cuda(), K, record)
            assert np.array_equal(y1[0], y[i]), i
            assert np.all(np.abs(g1[0] - g[i]) <= 1e-7 * most), (i, g[i], g1)
    finally:
        sfd.sfd_ctx_destroy(ctx)
