"""A search that fails part of the way through building its operands leaves
nothing half built behind: the same handle then searches as a new one does.
The failures are made on the host (FC_FAULT_ALLOC, FC_FAULT_LAUNCH)."""
import ctypes
import math

import numpy as np
import pytest

import oracle
from synth import make_dataset, permuted_phenotypes
from tests.parity_util import assert_topn_equal

pytestmark = pytest.mark.gpu
TC = {"FC_PAIRS_PATH": "tc", "FC_TRIPLES_PATH": "tc", "FC_QUADS_PATH": "tc"}


@pytest.fixture(scope="module")
def fc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2201_03331_gb300 as fcm
    from paper_2201_03331_gb300 import build
    build.build()
    return fcm


def fail_each(fc, monkeypatch, variable, load, search, check):
    """Makes the 1st, 2nd, .. allocation or launch of a first search fail until
    none is left to fail; the search after it has to be right.  A search of
    other data in between leaves other contents in the memory handed out."""
    reset = ctypes.CDLL(fc._binding.LIB_PATH)._ZN2fc20fault_counters_resetEv
    failed = 0
    for n in range(1, 60):
        h = load(1)
        search(h)
        fc.fc_free(h)
        h = load(0)
        reset()
        monkeypatch.setenv(variable, str(n))
        try:
            result = search(h)
        except fc.FiunchoError as e:
            assert e.status == (fc.FC_ENOMEM if variable == "FC_FAULT_ALLOC" else fc.FC_ECUDA)
            failed += 1
            result = None
        finally:
            monkeypatch.delenv(variable)
        check(search(h))
        if result is not None:
            check(result)
            return failed
    raise AssertionError("still failing")


@pytest.mark.parametrize("variable", ["FC_FAULT_ALLOC", "FC_FAULT_LAUNCH"])
@pytest.mark.parametrize("k,S,part,slab_mb", [(2, 60, None, None), (3, 40, None, None), (4, 24, None, None),
                                              (4, 24, (3, 8), None), (5, 18, None, "6"), (6, 14, None, None)])
def test_search_after_a_failed_one(fc, monkeypatch, variable, k, S, part, slab_mb):
    for name, value in TC.items():
        monkeypatch.setenv(name, value)
    if slab_mb:
        monkeypatch.setenv("FC_TUPLES_SLAB_MB", slab_mb)
    sets = [make_dataset("retry", seed=1300 + 10 * k + i, S=S, cases=300, controls=290, k=k, top_n=12) for i in (0, 1)]
    total = math.comb(S, k)
    lo, hi = (total * part[0] // part[1], total * (part[0] + 1) // part[1]) if part else (0, total)
    G, ph = sets[0].genotypes, sets[0].phenotype
    o_idx, o_s, _ = oracle.search(G, ph, k, 12) if not part else (None, None, None)
    if part:
        C = np.array([fc.fc_unrank(S, k, r) for r in range(lo, hi)], dtype=np.uint32)
        mi = oracle.mi(oracle.tables(G, ph, k, C), k)
        at = np.lexsort((np.arange(len(C)), -mi))[:12]
        o_idx, o_s = C[at], mi[at]

    def check(r):
        assert_topn_equal(r[0], r[1], o_idx, o_s, lambda c: float(oracle.mi(oracle.tables(G, ph, k, [c]), k)[0]))
    failed = fail_each(fc, monkeypatch, variable, lambda i: fc.fc_load(sets[i].genotypes, sets[i].phenotype),
                       lambda h: fc.fc_search_range(h, k, 12, lo, hi) if part else fc.fc_search(h, k, 12), check)
    assert failed >= 2


@pytest.mark.parametrize("variable", ["FC_FAULT_ALLOC", "FC_FAULT_LAUNCH"])
def test_batch_after_a_failed_one(fc, monkeypatch, variable):
    for name, value in TC.items():
        monkeypatch.setenv(name, value)
    sets = [make_dataset("retryb", seed=1390 + i, S=40, cases=300, controls=290, k=3, top_n=7) for i in (0, 1)]
    phs = [permuted_phenotypes(s.phenotype, 2, seed=1395) for s in sets]
    want = [oracle.search(sets[0].genotypes, ph, 3, 7) for ph in phs[0]]

    def check(r):
        for j, (o_idx, o_s, _) in enumerate(want):
            assert r[2][j] == 7
            assert_topn_equal(r[0][j], r[1][j], o_idx, o_s, lambda c: float(
                oracle.mi(oracle.tables(sets[0].genotypes, phs[0][j], 3, [c]), 3)[0]))
    failed = fail_each(fc, monkeypatch, variable, lambda i: fc.fc_load_batch([sets[i].genotypes], [phs[i]]),
                       lambda h: fc.fc_search_batch(h, 3, 7), check)
    assert failed >= 2
