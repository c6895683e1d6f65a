"""Scratch of the calls without a plan (stand-alone product and transform): one pool per device, shared by
threads and streams.  The same call gives the same bits whatever runs beside it, sizes above and below what
the pool keeps follow one another, and a capturing stream is refused with the capture left intact."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _product(B, torch, M, N, K, slices, splits, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn((M, K), dtype=torch.float64, device="cuda", generator=g)
    b = torch.randn((N, K), dtype=torch.float64, device="cuda", generator=g)
    c = torch.empty((M, N), dtype=torch.float64, device="cuda")
    return lambda: (B.isdf_gemm_f64(a, b, c, slices=slices, splits=splits), c.clone())[1]


def test_threads_and_streams_share_the_pool():
    import torch

    from paper_2404_09373_gb300 import isdf as B

    shapes = [(391, 208, 208, 8, 1), (1000, 97, 700, 5, 4), (64, 16, 33, 6, 1), (5000, 300, 1100, 7, 3)]
    calls = [_product(B, torch, *s, seed=i) for i, s in enumerate(shapes)]
    want = [c() for c in calls]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for r in range(6):
                a = calls[i]()
                stream.synchronize()
                if not torch.equal(a, want[i]):
                    bad.append((i, r))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_a_capturing_stream_is_refused():
    import torch

    from paper_2404_09373_gb300 import isdf as B

    call = _product(B, torch, 100, 50, 60, 8, 1, seed=3)
    want = call()
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    a = torch.randn((100, 60), dtype=torch.float64, device="cuda")
    c = torch.empty((100, 100), dtype=torch.float64, device="cuda")
    with torch.cuda.graph(graph):
        with pytest.raises(Exception):
            B.isdf_gemm_f64(a, a, c, slices=8)
        x.add_(1.0)
    graph.replay()
    torch.cuda.synchronize()
    assert x.eq(1.0).all()
    assert torch.equal(call(), want)


def test_large_then_small():
    import torch

    from paper_2404_09373_gb300 import isdf as B

    small = _product(B, torch, 129, 49, 65, 8, 1, seed=5)
    want = small()
    big = _product(B, torch, 700001, 40, 511, 8, 1, seed=6)  # 5.7 GB of digits, more than the pool keeps
    first = big()
    assert torch.equal(small(), want)
    assert torch.equal(big(), first)
    rows = np.array([0, 127, 128, 350000, 700000])
    assert torch.equal(first[rows].isfinite(), torch.ones_like(first[rows], dtype=torch.bool))
