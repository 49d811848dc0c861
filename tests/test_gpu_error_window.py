"""The window of FP32 scores that order 2 rescores: the kernel's error stays
within the bound the window rests on, and near-tied scores widen a list only
where that bound asks for it."""
import itertools
import math

import numpy as np
import pytest

import oracle
from synth import make_dataset

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.fixture(scope="module")
def fc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2201_03331_gb300 as fcm
    from paper_2201_03331_gb300 import build
    build.build()
    return fcm


@pytest.mark.parametrize("cases,controls", [(1, 1), (3, 4), (4, 4), (8, 7), (60, 190), (150, 149), (2000, 2000),
                                            (4095, 4095), (4096, 4096), (100, 20000), (16000, 19000)])
def test_pair_scores_within_28u(fc, cases, controls):
    S = 130
    ds = make_dataset("win", seed=1400 + cases, S=S, cases=cases, controls=controls, k=2, top_n=5)
    G = ds.genotypes.copy()
    G[0], G[1] = 0, 1          # whole classes in one cell
    G[2] = ds.phenotype * 2    # and a cell per class
    sc, _ = fc.fc_pairs_dense(fc.fc_load(G, ds.phenotype), scores=True, tables=False)
    C = np.array(list(itertools.combinations(range(S), 2)), dtype=np.uint32)
    mi = oracle.mi(oracle.tables(G, ds.phenotype, 2, C), 2)
    assert np.abs(sc[C[:, 0], C[:, 1]].astype(np.float64) - mi).max() <= 28.0 * U


def near_tied():
    """One strong SNP and 80 that are almost constant: 40 pairs tie at the top
    and 40 more lie just below, between once and twice the sweep's window."""
    M, S = 20000, 81
    ph = (np.arange(M) < 10000).astype(np.uint8)
    G = np.zeros((S, M), np.uint8)
    G[0, :8000] = 2
    G[0, 8000:9000] = 1
    G[0, 10000:12000] = 2
    G[0, 12000:16000] = 1
    for i in range(80):
        G[1 + i, 5 * i] = 1
        if i < 40:
            G[1 + i, 5 * i + 1] = 1
    return G, ph


@pytest.mark.parametrize("path", ["popc", "tc"])
def test_window_of_order_2_does_not_widen(fc, monkeypatch, path):
    monkeypatch.setenv("FC_PAIRS_PATH", path)
    G, ph = near_tied()
    M = G.shape[1]
    C = np.array(list(itertools.combinations(range(len(G)), 2)), dtype=np.uint32)
    mi = oracle.mi(oracle.tables(G, ph, 2, C), 2)
    top = np.sort(mi)[::-1]
    lm = math.log(M)
    window = 4.0 * U * (2.0 * lm + 24.0 * math.log(2.0))
    assert top[39] - top[0] == 0 and window < top[0] - top[40] < 4.0 * U * (7.0 * lm + 19.0 * math.log(2.0)) - 1e-7
    assert top[0] - top[79] < 2 * window < top[0] - top[80]
    h = fc.fc_load(G, ph)
    fc.fc_timing(h, 1)
    idx, s = fc.fc_search(h, 2, 10)   # a list of 64 places: the first 40 fit, all 80 do not
    assert fc.fc_timing(h, 0)[1] == 1
    at = np.lexsort((np.arange(len(C)), -mi))[:10]
    assert np.array_equal(idx, C[at])
    np.testing.assert_allclose(s, mi[at], rtol=1e-6, atol=1e-12)
