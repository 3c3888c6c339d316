"""The forward pass of a tape records the trajectory while it synthesizes.  For
strings stepped by a warp group (5 and more longitudinal rows per lane: 4
warps; 13 to 24: 8 warps) its samples equal plain synthesis bit for bit, in
every run, and the gradient from the recorded levels equals the one from
replayed segments bit for bit.  (A step that read a longitudinal transfer slot
which another warp's sweep had already rewritten gave samples that differed
from run to run.)"""

import numpy as np
import pytest

from test_gpu_instances import string

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 1500


@pytest.mark.parametrize("n_t,n_l,kind", [
    (110, 160, "pluck"), (150, 200, "bow"), (180, 260, "hammer"),     # 5, 7, 9 rows per lane: groups of 4
    (270, 400, "bow"), (288, 420, "hammer"),                          # 13, 15: groups of 8
])
def test_recorded_groups_equal_plain_synthesis(n_t, n_l, kind):
    from paper_2311_18505_gb300 import sfd
    torch.cuda.init()
    d = string(n_t, n_l, kind)
    m_z = (n_l + 31) // 32 | 1
    assert m_z >= 5
    dicts = [d] * 24
    w = torch.randn(len(dicts), N, generator=torch.Generator().manual_seed(3)).cuda()
    ctx = sfd.sfd_ctx_create(0, None, 128 << 20)
    try:
        s = sfd.string_from_dict(ctx, d)
        plain = sfd.sfd_synthesize(s, N)
        sfd.sfd_string_destroy(s)
        grads = []
        for record in (True, True, False):
            tape = sfd.sfd_tape_create(ctx, dicts, N, 512)
            sfd.sfd_tape_set_record_forward(tape, record)
            y = torch.empty(len(dicts), N, device="cuda")
            sfd.sfd_tape_forward(tape, y)
            for row in y.cpu().numpy():
                assert np.array_equal(row.view(np.int32), plain.view(np.int32))
            grads.append(sfd.sfd_tape_backward(tape, w, len(dicts)))
            sfd.sfd_tape_destroy(tape)
        assert np.array_equal(grads[0], grads[1]) and np.array_equal(grads[0], grads[2])
    finally:
        sfd.sfd_ctx_destroy(ctx)
