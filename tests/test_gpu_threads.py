"""Calls of several threads with rows of different lengths: a launch never finds its kernel's shared
memory limit lowered by another thread's call."""
import sys
import threading

import pytest
import torch

from paper_2002_09049_gb300 import binding

pytestmark = pytest.mark.gpu


def calls(kind, d, dev, stream):
    """The C call on 2 channels of d elements, its arguments ready (and kept)."""
    lib, p = binding.load(), lambda t: t.data_ptr()
    W, X = torch.randn(2, d, device=dev), torch.randn(2, 3, d, device=dev)
    codes = torch.zeros((4, 2, d), dtype=torch.int8, device=dev)
    scales, err = torch.zeros((2, 4), device=dev), torch.zeros((2, 5), device=dev)
    best = torch.zeros(2, dtype=torch.int32, device=dev)
    keep = (W, X, codes, scales, err, best)
    fn, args = {
        "adaptive": (lib.mpq_quantize_layer_adaptive,
                     (p(W), 2, d, 3, 1, binding.ETA, 10 ** 15, p(codes), p(scales), None, None)),
        "clip": (lib.mpq_clip_search,
                 (p(X), 3, 2, p(W), 2, d, 4, 4, binding.MPQ_CLIP_PER_CHANNEL, p(scales), p(err), p(best))),
        "grouped": (lib.mpq_output_error,
                    (p(X), 3, 2, p(W), p(codes), p(scales), None, 2, d, 4, p(err))),
    }[kind]
    return fn, args + (stream.cuda_stream,), keep


@pytest.mark.parametrize("kind,long,short", [("clip", 7000, 40), ("grouped", 4096, 40),
                                             ("adaptive", 8192, 40)])
def test_rows_of_different_lengths(gpu, kind, long, short):
    failed, start = [], threading.Barrier(4)

    def work(d, n):
        torch.cuda.set_device(gpu)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            fn, args, keep = calls(kind, d, gpu, stream)
        stream.synchronize()
        start.wait()
        for i in range(n):
            status = fn(*args)
            if status != 0:
                failed.append((d, status, binding.load().mpq_last_error()))
                break
            if i % 64 == 63:
                stream.synchronize()
        stream.synchronize()

    interval = sys.getswitchinterval()
    sys.setswitchinterval(1e-6)
    try:
        threads = [threading.Thread(target=work, args=(d, n))
                   for d, n in ((long, 1500), (short, 3000), (long, 1500), (short, 3000))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    finally:
        sys.setswitchinterval(interval)
    assert not failed, failed
