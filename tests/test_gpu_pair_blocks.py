"""Edges of the order-2 tensor-core tiles: SNP counts around the 56 and 112
SNPs j and the 64 and 128 SNPs i of a tile, classes that end inside, at and
past a 256-sample chunk, accumulators near 2^24, classes beyond one
accumulator, and rank ranges."""
import itertools
import math

import numpy as np
import pytest

import oracle
from synth import make_dataset
from tests.parity_util import assert_topn_equal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2201_03331_gb300 as fcm
    from paper_2201_03331_gb300 import build
    build.build()
    return fcm


@pytest.mark.parametrize("S,cases,controls", [(2, 1, 1), (56, 128, 128), (57, 129, 127), (64, 127, 129), (65, 256, 257),
                                              (112, 257, 256), (113, 384, 128), (128, 128, 385), (129, 511, 70),
                                              (241, 200, 130), (20, 4095, 4095), (70, 4096, 100), (130, 90, 4200),
                                              (40, 16500, 300)])
def test_tile_edges(fc, monkeypatch, S, cases, controls):
    """Every table equals the oracle's, every FP32 score is within u (7 ln M +
    19 ln 2) of its FP64 value, and the lists of the search and of ranges are
    the oracle's.  Two SNPs without variation put whole classes into one
    cell."""
    monkeypatch.setenv("FC_PAIRS_PATH", "tc")
    ds = make_dataset("blk", seed=1200 + S, S=S, cases=cases, controls=controls, k=2, top_n=5)
    G = ds.genotypes.copy()
    G[0], G[S - 1] = 0, 1
    h = fc.fc_load(G, ds.phenotype)
    sc, tab = fc.fc_pairs_dense(h, scores=True, tables=True)
    C = np.array(list(itertools.combinations(range(S), 2)), dtype=np.uint32)
    ref = oracle.tables(G, ds.phenotype, 2, C)
    assert np.array_equal(tab[C[:, 0], C[:, 1]], ref)
    assert not tab[np.tril_indices(S)].any()
    mi = oracle.mi(ref, 2)
    bound = 2.0 ** -24 * (7.0 * math.log(max(ds.M, 2)) + 19.0 * math.log(2.0))
    assert np.abs(sc[C[:, 0], C[:, 1]].astype(np.float64) - mi).max() <= bound

    def score_of(c):
        return float(oracle.mi(oracle.tables(G, ds.phenotype, 2, [c]), 2)[0])
    T = len(C)
    for r0, r1 in ((0, T), (0, (T + 2) // 3), (T // 3, T // 3 + 1), (T // 2, T)):
        n = min(40, r1 - r0)
        order = np.lexsort((np.arange(r0, r1), -mi[r0:r1]))[:n] + r0
        idx, s = fc.fc_search_range(h, 2, n, r0, r1)
        assert fc.fc_last_search_kind(h) == 2
        assert_topn_equal(idx, s, C[order], mi[order], score_of)
