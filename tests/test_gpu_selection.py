"""The merge of the candidate lists, the rescoring and the final order: list
lengths on both sides of the counted and the sorted orders, fewer combinations
than places, and ties of more combinations than a list holds."""
import itertools

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


def check(fc, G, ph, k, n):
    C = np.array(list(itertools.combinations(range(len(G)), k)), dtype=np.uint32)
    mi = oracle.mi(oracle.tables(G, ph, k, C), k)
    order = np.lexsort((np.arange(len(C)), -mi))[:n]
    idx, s = fc.fc_search(fc.fc_load(G, ph), k, n)

    def score_of(c):
        return float(oracle.mi(oracle.tables(G, ph, k, [c]), k)[0])
    assert_topn_equal(idx, s, C[order], mi[order], score_of)


@pytest.mark.parametrize("k,S", [(1, 500), (2, 2), (2, 90), (3, 30), (4, 16)])
@pytest.mark.parametrize("n", [1, 32, 33, 205, 206, 819, 2048])
def test_list_lengths(fc, k, S, n):
    ds = make_dataset("sel", seed=1000 + 10 * S + k, S=S, cases=300, controls=280, k=max(k, 2), top_n=5)
    check(fc, ds.genotypes, ds.phenotype, k, n)


@pytest.mark.parametrize("k,S", [(2, 64), (3, 24)])
@pytest.mark.parametrize("n", [1, 40, 900, 2048])
def test_all_scores_tie(fc, k, S, n):
    """Equal SNPs: every list is full of one score, and the first
    combinations are the best."""
    ds = make_dataset("tie", seed=1100, S=S, cases=200, controls=230, k=k, top_n=5)
    check(fc, np.repeat(ds.genotypes[:1], S, axis=0), ds.phenotype, k, n)
