"""Edges of the order-3 tensor-core tiles: SNP counts around the 28 and 56
pairs and the 64 and 128 SNPs of a tile, classes that end inside, at and past
a 256-sample chunk, accumulators near 2^24, and batches that mix both forms."""
import itertools
import math

import numpy as np
import pytest

import oracle
from synth import make_dataset, permuted_phenotypes
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


def combos(S):
    return np.array(list(itertools.combinations(range(S), 3)), dtype=np.uint32)


@pytest.mark.parametrize("enc", ["1", "0"])
@pytest.mark.parametrize("S,cases,controls", [(4, 1, 1), (28, 128, 128), (29, 129, 127), (30, 127, 129),
                                              (57, 256, 257), (58, 257, 256), (64, 384, 128), (65, 128, 385),
                                              (66, 511, 1), (130, 1, 130), (12, 4095, 4095)])
def test_tile_edges(fc, monkeypatch, S, cases, controls, enc):
    """Every table equals the oracle's, every FP32 score is within u (7 ln M +
    37 ln 2) of its FP64 value, and the search's list is the oracle's.  Two
    SNPs without variation put whole classes into one cell."""
    monkeypatch.setenv("FC_TRIPLES_ENC", enc)
    monkeypatch.setenv("FC_TRIPLES_PATH", "tc")
    ds = make_dataset("edge", seed=900 + S, S=S, cases=cases, controls=controls, k=3, top_n=5)
    G = ds.genotypes.copy()
    G[0], G[1], G[S - 1] = 0, 1, 0
    h = fc.fc_load(G, ds.phenotype)
    sc, tab = fc.fc_triples_dense(h, scores=True, tables=True)
    C = combos(S)
    ref = oracle.tables(G, ds.phenotype, 3, C)
    assert np.array_equal(tab, ref)
    mi = oracle.mi(ref, 3)
    bound = 2.0 ** -24 * (7.0 * math.log(max(ds.M, 2)) + 37.0 * math.log(2.0))
    assert np.abs(sc.astype(np.float64) - mi).max() <= bound
    n = min(33, len(C))
    order = np.lexsort((np.arange(len(C)), -mi))[:n]
    # Candidate lists grow 128, 512, 2048: more ties than that are refused.
    if np.count_nonzero(mi >= mi[order[-1]] - bound) > 2048:
        with pytest.raises(fc.FiunchoError, match="4096 candidates"):
            fc.fc_search(h, 3, n)
        return
    idx, s = fc.fc_search(h, 3, n)

    def score_of(c):
        return float(oracle.mi(oracle.tables(G, ds.phenotype, 3, [c]), 3)[0])
    assert_topn_equal(idx, s, C[order], mi[order], score_of)


def test_batch_of_both_forms(fc, monkeypatch):
    """Jobs of both forms, several SNP and sample counts in one batch, with
    slabs built in one group and in several."""
    monkeypatch.setenv("FC_TRIPLES_PATH", "tc")
    sets = [make_dataset("m%d" % i, seed=930 + i, S=S, cases=a, controls=b, k=3, top_n=7)
            for i, (S, a, b) in enumerate([(57, 300, 260), (66, 4200, 100), (29, 129, 127), (130, 256, 513)])]
    phs = [permuted_phenotypes(ds.phenotype, 2, seed=940 + i) for i, ds in enumerate(sets)]
    for mb in (None, "1"):
        if mb:
            monkeypatch.setenv("FC_BATCH_SLAB_MB", mb)
        h = fc.fc_load_batch([ds.genotypes for ds in sets], phs)
        idx, score, cnt = fc.fc_search_batch(h, 3, 7)
        for j in range(8):
            ds, ph = sets[j // 2], phs[j // 2][j % 2]
            o_idx, o_s, _ = oracle.search(ds.genotypes, ph, 3, 7)

            def score_of(c, ds=ds, ph=ph):
                return float(oracle.mi(oracle.tables(ds.genotypes, ph, 3, [c]), 3)[0])
            assert cnt[j] == 7
            assert_topn_equal(idx[j], score[j], o_idx, o_s, score_of)


@pytest.mark.parametrize("S,kind", [(191, 3), (192, 6)])
def test_default_path_by_snps(fc, monkeypatch, S, kind):
    """From 192 SNPs the tensor cores by default; both sides give the sweep's
    list."""
    monkeypatch.delenv("FC_TRIPLES_PATH", raising=False)
    ds = make_dataset("path", seed=960, S=S, cases=260, controls=301, k=3, top_n=40)
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    a = fc.fc_search(h, 3, 40)
    assert fc.fc_last_search_kind(h) == kind
    monkeypatch.setenv("FC_TRIPLES_PATH", "popc")
    b = fc.fc_search(h, 3, 40)
    assert fc.fc_last_search_kind(h) == 3
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
