"""The lines between the sweep and the tensor cores on the default path, from
both sides: rank ranges and the jobs of a batch at order 3; and sample counts
whose shared memory once did not fit at orders 2 and 4."""
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


@pytest.fixture(autouse=True)
def default_paths(monkeypatch):
    for name in ("FC_PAIRS_PATH", "FC_TRIPLES_PATH", "FC_QUADS_PATH"):
        monkeypatch.delenv(name, raising=False)


@pytest.mark.parametrize("S,kind", [(383, 3), (384, 6)])
@pytest.mark.parametrize("part,parts", [(0, 64), (1, 2)])
def test_rank_ranges(fc, monkeypatch, S, kind, part, parts):
    ds = make_dataset("line", seed=1500, S=S, cases=260, controls=301, k=3, top_n=40)
    total = math.comb(S, 3)
    lo, hi = total * part // parts, total * (part + 1) // parts
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    a = fc.fc_search_range(h, 3, 40, lo, hi)
    assert fc.fc_last_search_kind(h) == kind
    monkeypatch.setenv("FC_TRIPLES_PATH", "popc")
    b = fc.fc_search_range(h, 3, 40, lo, hi)
    assert fc.fc_last_search_kind(h) == 3
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("replicates", [2, 8])
def test_batch_jobs(fc, monkeypatch, replicates):
    """(SNPs, cases, controls, 128-sample words; path in a batch of few jobs
    and of 48 or more that are short)."""
    sizes = [(255, 200, 200, 4, 3, 3), (256, 200, 200, 4, 8, 3), (287, 200, 200, 4, 8, 3), (288, 200, 200, 4, 8, 8),
             (256, 128, 129, 3, 8, 3), (351, 128, 129, 3, 8, 3), (352, 128, 129, 3, 8, 8),
             (256, 128, 128, 2, 8, 3), (383, 128, 128, 2, 8, 3), (384, 128, 128, 2, 8, 8), (256, 300, 250, 5, 8, 8)]
    kinds = [s[4 if replicates == 2 else 5] for s in sizes]
    sets = [make_dataset("lineb%d" % i, seed=1510 + i, S=s[0], cases=s[1], controls=s[2], k=3, top_n=9)
            for i, s in enumerate(sizes)]
    phs = [permuted_phenotypes(d.phenotype, replicates, seed=1530) for d in sets]
    h = fc.fc_load_batch([d.genotypes for d in sets], phs)
    a = fc.fc_search_batch(h, 3, 9)
    assert [fc.fc_batch_job_kind(h, replicates * i) for i in range(len(sets))] == kinds
    monkeypatch.setenv("FC_BATCH_TC", "0")
    h = fc.fc_load_batch([d.genotypes for d in sets], phs)
    b = fc.fc_search_batch(h, 3, 9)
    assert {fc.fc_batch_job_kind(h, j) for j in range(replicates * len(sets))} == {3}
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("k,S,kind", [(2, 1024, 2), (4, 64, 7)])
@pytest.mark.parametrize("M", [2399, 2450, 2500, 2550, 2600])
@pytest.mark.parametrize("n", [10, 1000])
def test_around_2500_samples(fc, monkeypatch, k, S, kind, M, n):
    """The static arrays count beside the table and the stages."""
    ds = make_dataset("mid", seed=1540, S=S, cases=M // 2, controls=M - M // 2, k=k, top_n=n)
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    a = fc.fc_search(h, k, n)
    assert fc.fc_last_search_kind(h) == kind and len(a[1]) == n
    monkeypatch.setenv("FC_PAIRS_PATH", "popc")
    monkeypatch.setenv("FC_QUADS_PATH", "popc")
    b = fc.fc_search(h, k, n)
    assert fc.fc_last_search_kind(h) != kind
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    if n == 10:
        o_idx, o_s, _ = oracle.search(ds.genotypes, ds.phenotype, k, n)
        assert_topn_equal(a[0], a[1], o_idx, o_s, lambda c: float(
            oracle.mi(oracle.tables(ds.genotypes, ds.phenotype, k, [c]), k)[0]))


@pytest.mark.parametrize("M,tc", [(36223, True), (36224, True), (39295, True), (39296, False)])
def test_order_4_at_its_sample_limit(fc, monkeypatch, M, tc):
    """What fits is asked of the table and the list as they are launched."""
    ds = make_dataset("most", seed=1550, S=64, cases=M // 2, controls=M - M // 2, k=4, top_n=10)
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    a = fc.fc_search(h, 4, 10)
    assert (fc.fc_last_search_kind(h) == 7) == tc
    monkeypatch.setenv("FC_QUADS_PATH", "popc")
    b = fc.fc_search(h, 4, 10)
    assert fc.fc_last_search_kind(h) != 7
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


def test_static_search_keeps_the_form_of_its_operands(fc, monkeypatch):
    """fc_search_static takes the order-3 operands as they were built, in
    whichever form, and allocates nothing."""
    ds = make_dataset("form", seed=1560, S=200, cases=300, controls=330, k=3, top_n=20)
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    want = fc.fc_search(h, 3, 20)
    for form in ("0", "1"):
        monkeypatch.setenv("FC_TRIPLES_ENC", form)
        monkeypatch.setenv("FC_FAULT_ALLOC_ALL", "1")
        got = fc.fc_search_static(h, 3, 20)
        assert fc.fc_last_search_kind(h) == 6
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
        monkeypatch.delenv("FC_FAULT_ALLOC_ALL")
        got = fc.fc_search(h, 3, 20)   # builds the operands of that form
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
