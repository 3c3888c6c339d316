"""Every instance of the register-path step function (rows per lane of both
grids, excitation, linear, folded or factored longitudinal matrix) at the
edges of its range: the smallest and largest grid of each class against the
FP64 oracle, and the same samples alone, in one launch with all the others
(segments of several strings per CTA) and on one warp or a warp group.

Tolerances are the repository's for these excitations: relative L2 1e-4
plucked and struck, 1e-3 bowed (300 samples)."""

import numpy as np
import pytest

import oracle
from paper_2311_18505_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 300
EXC = {"pluck": {"kind": "pluck", "amp": 1e-3, "pos": 0.3},
       "hammer": {"kind": "hammer", "mass": 3e-3, "vel": 1.0, "pos": 0.27, "omega": 3000.0, "alpha": 2.5},
       "bow": {"kind": "bow", "vel": 0.2, "force": 0.8, "pos": 0.21, "a": 100.0, "eps": 0.1, "release": -1.0}}


def string(n_t, n_l, kind, factored=False, output="transverse"):
    """A string without stiffness whose grids are n_t and n_l intervals (n_l 0: linear)."""
    d = W.make(kappa=0.0, excitation=EXC[kind], n_samples=N, sigma1=1e-5, output=output)
    f0 = np.sqrt(2 * d["theta"] - 1) * d["fs"] / 2 / (n_t + 0.5)
    d.update(f0=f0, alpha=1.0 if n_l == 0 else d["fs"] / (2 * f0 * (n_l + 0.5)))
    # a coarse longitudinal grid means a large alpha: less motion, so that the coupling stays as in practice
    gentle = min(1.0, 4.0 / d["alpha"])
    for key in ("amp", "vel", "force"):
        if key in d["excitation"]:
            d["excitation"][key] *= gentle
    if factored:   # above the ratio of 1 % at which the off-diagonal is folded into the sweeps
        d["sigma1"] = 0.012 * d["fs"] / n_l ** 2
    got = oracle.grid(d)
    assert got[0] == n_t and (n_l == 0 or got[1] == n_l)
    return d


def cases():
    out = []
    for m_u in (1, 3, 5, 7, 9):
        least, most = (2 if m_u == 1 else 32 * (m_u - 2) + 1), 32 * m_u
        for n_t in (least, most):
            sizes = {0, 1, 2, 32, 33, 96, 97, 160, int(1.5 * n_t)}   # m_z: none, 1, 3, 5 and the largest
            for n_l in sorted(s for s in sizes if s <= 1.5 * n_t):
                for kind in EXC:
                    out.append((n_t, n_l, kind, False))
        out.append((most, int(1.2 * most), "bow", True))
        out.append((most, int(1.2 * most), "pluck", True))
    return out


@pytest.fixture(scope="module")
def rendered():
    from paper_2311_18505_gb300 import sfd
    strings = [string(*c, output="longitudinal" if i % 7 == 3 and c[0] > 2 and c[1] > 1 else "transverse")
               for i, c in enumerate(cases())]
    torch.cuda.init()
    out = {}
    for groups in (True, False):
        ctx = sfd.sfd_ctx_create(0, None, 128 << 20)
        try:
            sfd.sfd_ctx_set_warp_pairs(ctx, groups)
            alone = []
            for d in strings:
                s = sfd.string_from_dict(ctx, d)
                alone.append(sfd.sfd_synthesize(s, N))
                sfd.sfd_string_destroy(s)
            copies = strings * (1 if groups else 9)   # more than one string per warp slot without groups
            hs = [sfd.string_from_dict(ctx, d) for d in copies]
            b = sfd.sfd_batch_create(ctx, hs)
            ys, _ = sfd.sfd_batch_synthesize_host(b, [N] * len(hs))
            sfd.sfd_batch_destroy(b)
            for h in hs:
                sfd.sfd_string_destroy(h)
            out[groups] = (alone, ys)
        finally:
            sfd.sfd_ctx_destroy(ctx)
    return strings, out


def test_instances_match_the_oracle(rendered):
    strings, out = rendered
    worst = {}
    for d, y, c in zip(strings, out[True][0], cases()):
        ref = oracle.run(d, N)
        scale = np.linalg.norm(ref)
        err = np.linalg.norm(y - ref) / scale if scale > 0 else float(np.abs(y).max())
        worst[c] = err / (1e-3 if c[2] == "bow" else 1e-4)
    bad = {c: w for c, w in worst.items() if not w <= 1.0}
    assert not bad, bad


def test_instances_give_the_same_bits_however_they_are_launched(rendered):
    strings, out = rendered
    ref = out[True][0]
    n = len(strings)
    for alone, batch in out.values():
        for i, y in enumerate(list(alone) + list(batch)):
            assert np.array_equal(y, ref[i % n]), (i, cases()[i % n])
