"""Transforms of several host threads at once: axes whose passes need different amounts of shared memory (16 and 18
points 43 KB, 96 points 54, 108 points 60, 128 points 74) side by side give the bits that each gives alone."""
import threading

import pytest

pytestmark = pytest.mark.gpu


def test_threads_transform_side_by_side():
    import torch

    from paper_2404_09373_gb300 import isdf as B

    shapes = [(96, 16, 18, 1), (18, 108, 16, 1), (36, 16, 81, 1), (16, 18, 128, 1), (16, 16, 16, 4), (18, 16, 18, 4)]
    calls = 300
    f, want, out = [], [], []
    for i, (nx, ny, nz, batch) in enumerate(shapes):
        g = torch.Generator(device="cuda").manual_seed(i)
        f.append(torch.randn((batch, nz, ny, nx), dtype=torch.float64, device="cuda", generator=g))
        want.append(B.isdf_rfft3(f[i]))
        # one slot per call, so that a pass that did not run is not made good by the next call
        out.append([torch.full_like(want[i], float("nan")) for _ in range(calls)])
    torch.cuda.synchronize()
    start = threading.Barrier(len(shapes))
    failed = []

    def work(i):
        stream = torch.cuda.Stream()
        start.wait()
        try:
            for r in range(calls):
                B.isdf_rfft3(f[i], out[i][r], stream=stream.cuda_stream)
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            failed.append((i, e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(shapes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    bad = [(i, r) for i in range(len(shapes)) for r in range(calls)
           if not torch.equal(torch.view_as_real(out[i][r]), torch.view_as_real(want[i]))]
    assert not bad, (len(bad), bad[:8])
