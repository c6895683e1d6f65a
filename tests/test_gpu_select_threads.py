"""Selections of several host threads at once whose speculative sets need different amounts of shared memory (16 KB to
216 KB, and above 108 members none): each gives the points and values that it gives alone."""
import threading

import numpy as np
import pytest

from paper_2404_09373_gb300 import isdf as B
from paper_2404_09373_gb300 import systems as S

pytestmark = pytest.mark.gpu


def test_plans_of_different_set_size_select_side_by_side():
    import torch

    sizes = (108, 16, 64, 96, 40, 109)
    sysd = S.make_system((1, 1, 1), 0.05, np.random.default_rng(12), ((24, 24, 24), (12, 12, 12), (6, 6, 6)),
                         S.LEVEL_EDGES_3)
    streams = [torch.cuda.Stream() for _ in sizes]
    plans = [B.isdf_plan(sysd, {"precision": 1, "prefilter": 1, "select_block": n}, stream=s.cuda_stream)
             for n, s in zip(sizes, streams)]
    try:
        want = [B.isdf_select_points(p, 240) for p in plans]
        for piv, _ in want[1:]:
            assert np.array_equal(piv, want[0][0])
        start = threading.Barrier(len(sizes))
        bad = []

        def work(i):
            start.wait()
            for r in range(8):
                try:
                    piv, val = B.isdf_select_points(plans[i], 240)
                except Exception as e:  # noqa: BLE001 - reported by the main thread
                    bad.append((sizes[i], r, e))
                    return
                if not (np.array_equal(piv, want[i][0]) and np.array_equal(val, want[i][1])):
                    bad.append((sizes[i], r))

        threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not bad
    finally:
        for p in plans:
            p.close()
