"""Contexts side by side on one GPU: a call of one context is not held up by a
batch that another context (on a stream of its own) is stepping, as long as
the batch leaves warps free; its samples are those it has alone."""

import threading
import time

import numpy as np
import pytest

from test_gpu_instances import string

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 16384     # samples of the batch: 30 ms and more
NOTE = 64     # samples of the call beside it: 0.2 to 0.5 ms alone

# strings of the batch (count, grid, excitation): some of it on every SM, with
# two launches; and groups of 4 warps beside CTAs of 8
BATCHES = {"spread": [(128, (90, 60), "pluck"), (128, (31, 31), "pluck")],
           "full": [(80, (150, 200), "pluck"), (760, (90, 60), "pluck")]}
# strings of the call: one note; two launches; groups of 4 and of 8 among them
NOTES = {"note": [(100, 80, "bow")],
         "pair": [(31, 33, "pluck"), (90, 96, "bow")],
         "chord": [(31, 33, "pluck"), (90, 96, "bow"), (150, 200, "bow")],
         "wide": [(90, 60, "pluck"), (288, 420, "hammer")]}


class Batch:
    def __init__(self, sfd, dicts, n):
        self.sfd, self.stream = sfd, torch.cuda.Stream()
        self.ctx = sfd.sfd_ctx_create(0, self.stream.cuda_stream, 64 << 20)
        self.strings = [sfd.string_from_dict(self.ctx, d) for d in dicts]
        self.batch = sfd.sfd_batch_create(self.ctx, self.strings)
        self.out = torch.zeros(len(dicts), n, device="cuda")
        torch.cuda.synchronize()
        sfd.sfd_batch_prepare(self.batch, [n] * len(dicts), self.out, np.arange(len(dicts)) * n)

    def launch(self):
        self.sfd.sfd_batch_launch(self.batch)

    def timed(self):
        t = time.perf_counter()
        self.launch()
        self.stream.synchronize()
        return time.perf_counter() - t

    def close(self):
        torch.cuda.synchronize()
        self.sfd.sfd_batch_destroy(self.batch)
        for s in self.strings:
            self.sfd.sfd_string_destroy(s)
        self.sfd.sfd_ctx_destroy(self.ctx)


@pytest.mark.parametrize("batch,notes", [("spread", "note"), ("spread", "chord"), ("spread", "wide"),
                                         ("full", "note"), ("full", "pair")])
def test_a_call_beside_another_contexts_batch(batch, notes):
    from paper_2311_18505_gb300 import sfd
    big = Batch(sfd, [string(*grid, kind) for count, grid, kind in BATCHES[batch] for _ in range(count)], N)
    dicts = [string(*c) for c in NOTES[notes]]
    alone = Batch(sfd, dicts, NOTE)
    alone.timed()
    ref = alone.out.cpu().numpy()
    alone.close()
    try:
        big.timed()
        t_big = big.timed()
        best = float("inf")
        # (a stream may share a hardware queue with one of the batch's, and the
        # host may be late: the best of the tries that met the batch running)
        for _ in range(5):
            call = Batch(sfd, dicts, NOTE)
            big.launch()
            time.sleep(0.1 * t_big)
            t = call.timed()
            if not big.stream.query():
                best = min(best, t)
            assert np.array_equal(call.out.cpu().numpy(), ref)
            call.close()
        assert best < 0.25 * t_big, (best, t_big)
    finally:
        big.close()


def test_a_call_beside_another_contexts_tape():
    """One note while another context's tape runs its reverse sweep on every SM
    (blocks of 192 threads and 100 KB, which leave warps and memory free)."""
    from paper_2311_18505_gb300 import sfd
    n = 1024
    dicts = [string(188, 280, "pluck")] * torch.cuda.get_device_properties(0).multi_processor_count
    note = [string(100, 80, "bow")]
    alone = Batch(sfd, note, NOTE)
    alone.timed()
    ref = alone.out.cpu().numpy()
    alone.close()
    stream = torch.cuda.Stream()
    ctx = sfd.sfd_ctx_create(0, stream.cuda_stream, 256 << 20)
    tape = sfd.sfd_tape_create(ctx, dicts, n, n)
    try:
        with torch.cuda.stream(stream):
            y = torch.empty(len(dicts), n, device="cuda")
            w = torch.ones(len(dicts), n, device="cuda")
        torch.cuda.synchronize()
        sfd.sfd_tape_forward(tape, y)
        backward = lambda: sfd.sfd_tape_backward(tape, w, len(dicts))
        backward()
        t = time.perf_counter()
        backward()
        t_back = time.perf_counter() - t
        best = float("inf")
        for _ in range(5):
            call = Batch(sfd, note, NOTE)
            thread = threading.Thread(target=backward)
            thread.start()
            time.sleep(0.3 * t_back)
            t = call.timed()
            if thread.is_alive():
                best = min(best, t)
            thread.join()
            assert np.array_equal(call.out.cpu().numpy(), ref)
            call.close()
        assert best < 0.25 * t_back, (best, t_back)
    finally:
        sfd.sfd_tape_destroy(tape)
        sfd.sfd_ctx_destroy(ctx)
