"""Edges of the packed 4-bit tuple kernel of orders 4-6: accumulators near
2^24, class boundaries inside a 256-sample chunk, cells on both sides of the
small-count table's limit, and rank ranges that build their own left rows."""
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


def combos(S, k):
    return np.array(list(itertools.combinations(range(S), k)), dtype=np.uint32)


@pytest.mark.parametrize("k", [4, 5, 6])
@pytest.mark.parametrize("cases,controls", [(4095, 4095), (1, 4095), (128, 129), (129, 127), (127, 128), (128, 127)])
def test_one_accumulator_limits(fc, monkeypatch, k, cases, controls):
    """SNPs without variation put whole classes into one cell: the
    accumulator n_case + 4096 n_ctrl reaches 2^24 - 1, and counts of 127 and
    128 take either side of the small-count table.  128- and 129-sample
    classes end inside, at and just past a chunk."""
    monkeypatch.setenv("FC_QUADS_ENC", "1")
    S = k + 3
    ds = make_dataset("lim", seed=40 + k, S=S, cases=cases, controls=controls, k=k, top_n=5)
    G = ds.genotypes.copy()
    G[: k - 1] = 0
    G[k - 1] = 2
    h = fc.fc_load(G, ds.phenotype)
    sc, tab = fc.fc_tuples_dense(h, k, scores=True, tables=True)
    ref = oracle.tables(G, ds.phenotype, k, combos(S, k))
    assert np.array_equal(tab, ref)
    u = 2.0 ** -24
    bound = 2.0 * u * (2.0 * math.log(ds.M) + (2.0 * 3 ** k + 6.0) * math.log(2.0))
    assert np.abs(sc.astype(np.float64) - oracle.mi(ref, k)).max() <= bound


@pytest.mark.parametrize("enc", ["1", "0"])
@pytest.mark.parametrize("k,S", [(4, 31), (5, 20), (6, 17)])
def test_ranges_match_oracle(fc, monkeypatch, k, S, enc):
    """Short ranges (few left tuples: their rows are built again, close
    together), long ones (the resident rows), and single combinations."""
    monkeypatch.setenv("FC_QUADS_PATH", "tc")
    monkeypatch.setenv("FC_QUADS_ENC", enc)
    ds = make_dataset("rng", seed=60 + k, S=S, cases=300, controls=333, k=k, top_n=5)
    all_c = combos(S, k)
    mi = oracle.mi(oracle.tables(ds.genotypes, ds.phenotype, k, all_c), k)
    total = len(all_c)
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    for r0, r1 in ((0, total // 64), (total // 3, total // 3 + total // 50), (total // 2, total), (0, total - 1),
                   (total // 5, total // 5 + 1), (total - 7, total), (total // 7, total // 2)):
        idx, s = fc.fc_search_range(h, k, 20, r0, r1)
        assert fc.fc_last_search_kind(h) == 7
        order = np.lexsort((np.arange(r0, r1), -mi[r0:r1]))[:20] + r0

        def score_of(c):
            return float(oracle.mi(oracle.tables(ds.genotypes, ds.phenotype, k, [c]), k)[0])
        assert_topn_equal(idx, s, all_c[order], mi[order], score_of)
