"""The launch plan's division of the SMs (sfd_api.cu, make_plan): batches whose
CTAs just fit the device with an SM for each, and just do not, with and
without warp groups, give every string the samples it has alone, bit for bit."""

import numpy as np
import pytest

from paper_2311_18505_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kinds,f0,fs,counts", [
    (("bow",), (40.0, 80.0), 48000.0, (2, 3, 5, 33)),                      # groups, few CTAs
    (("pluck", "hammer", "bow"), (60.0, 1500.0), 48000.0, (2, 7, 64, 143, 145, 160, 300)),
    (("pluck", "hammer", "bow"), (27.5, 60.0), 96000.0, (4, 40, 150)),     # groups of 4 and 8, their number near the SMs
])
def test_batches_around_one_cta_per_sm(kinds, f0, fs, counts):
    import torch
    from paper_2311_18505_gb300 import sfd
    rng = np.random.Generator(np.random.PCG64(4242))
    n = 48
    ds = [W.random_string(rng, f0[0], f0[1], kinds, fs=fs) for _ in range(max(counts))]
    ctx = sfd.sfd_ctx_create(0, None, 256 << 20)
    probe = range(0, max(counts), max(1, max(counts) // 24))
    alone = {}
    for i in probe:
        s = sfd.string_from_dict(ctx, ds[i])
        y = torch.zeros(n, device="cuda")
        torch.cuda.synchronize()
        sfd.sfd_synthesize(s, n, y)
        alone[i] = y.cpu().numpy()
        sfd.sfd_string_destroy(s)
    for count in counts:
        hs = [sfd.string_from_dict(ctx, d) for d in ds[:count]]
        b = sfd.sfd_batch_create(ctx, hs)
        y = torch.zeros(count, n, device="cuda")
        torch.cuda.synchronize()
        sfd.sfd_batch_synthesize(b, [n] * count, y, np.arange(count) * n)
        torch.cuda.synchronize()
        y = y.cpu().numpy()
        for i in probe:
            if i < count:
                assert np.array_equal(y[i].view(np.int32), alone[i].view(np.int32)), (count, i)
        sfd.sfd_batch_destroy(b)
        for h in hs:
            sfd.sfd_string_destroy(h)
    sfd.sfd_ctx_destroy(ctx)
