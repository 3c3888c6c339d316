"""A context makes its side streams when it is created: a first synthesis, of
one string or of a batch with one launch per kernel class, makes none (the
driver numbers streams as they are made, so a gap in the numbers shows one)."""

import ctypes

import pytest

from test_gpu_instances import string

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def made_by(fn):
    """How many streams fn makes (None if the driver's numbers do not tell)."""
    cuda = ctypes.CDLL("libcuda.so.1")
    handles = []

    def number():
        h, n = ctypes.c_void_p(), ctypes.c_ulonglong()
        assert cuda.cuStreamCreate(ctypes.byref(h), 1) == 0
        handles.append(h)
        assert cuda.cuStreamGetId(h, ctypes.byref(n)) == 0
        return n.value

    try:
        a, b = number(), number()
        fn()
        c = number()
        return c - b - 1 if b - a == 1 else None
    finally:
        for h in handles:
            cuda.cuStreamDestroy_v2(h)


@pytest.mark.parametrize("grids", [[(90, 60)], [(31, 31), (90, 60), (150, 90), (210, 90), (280, 90)]])
def test_a_first_synthesis_makes_no_stream(grids):
    from paper_2311_18505_gb300 import sfd
    torch.cuda.init()
    torch.zeros(1, device="cuda")
    ctx = sfd.sfd_ctx_create(0, None, 64 << 20)
    hs = [sfd.string_from_dict(ctx, string(*g, "pluck")) for g in grids]
    b = sfd.sfd_batch_create(ctx, hs)

    def first():
        if len(hs) == 1:
            sfd.sfd_synthesize(hs[0], 64)
        else:
            sfd.sfd_batch_synthesize_host(b, [64] * len(hs))
        assert sfd.sfd_last_launch_count(ctx) == len(hs)

    try:
        made = made_by(first)
    finally:
        sfd.sfd_batch_destroy(b)
        for h in hs:
            sfd.sfd_string_destroy(h)
        sfd.sfd_ctx_destroy(ctx)
    if made is None:
        pytest.skip("stream numbers are not consecutive here")
    assert made == 0
