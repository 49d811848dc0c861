"""Handles of several threads at once, with lists of different lengths: the
kernels' limit of dynamic shared memory is one value per process and device."""
import threading

import numpy as np
import pytest

from synth import make_dataset

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2201_03331_gb300 as fcm
    from paper_2201_03331_gb300 import build
    build.build()
    return fcm


@pytest.mark.parametrize("k,S,samples", [(2, 60, (300, 4000)), (2, 1100, (300, 4000)), (3, 200, (300, 4000)),
                                         (4, 64, (300, 3000))])
def test_lists_of_different_lengths(fc, k, S, samples):
    sets = [make_dataset("thr%d" % i, seed=1600 + i, S=S, cases=M // 2, controls=M // 2, k=k, top_n=10)
            for i, M in enumerate(samples)]
    work = [(sets[0], 10), (sets[1], 1600), (sets[1], 200), (sets[0], 700)]
    handles = [fc.fc_load(d.genotypes, d.phenotype) for d, _ in work]
    want = [fc.fc_search(h, k, n) for h, (_, n) in zip(handles, work)]
    start, wrong = threading.Barrier(len(work)), []

    def run(i):
        start.wait()
        try:
            for _ in range(150):
                idx, s = fc.fc_search(handles[i], k, work[i][1])
                if not (np.array_equal(idx, want[i][0]) and np.array_equal(s, want[i][1])):
                    raise AssertionError("another list")
        except Exception as e:   # (reported by the test's own thread)
            wrong.append((i, repr(e)))
    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
