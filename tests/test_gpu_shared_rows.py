"""Orders 2 and 3 share one copy of the packed SNP rows on the tensor cores,
whichever is searched first, and whether or not order 3 keeps its operands."""
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


@pytest.fixture(autouse=True)
def tensor_cores(monkeypatch):
    monkeypatch.setenv("FC_PAIRS_PATH", "tc")
    monkeypatch.setenv("FC_TRIPLES_PATH", "tc")


def launches(fc, h, k):
    fc.fc_timing(h, 1)
    fc.fc_search(h, k, 10)
    return fc.fc_timing(h, 0)[2]


def test_rows_are_built_once(fc):
    """The second order's first search launches three kernels fewer than on a
    handle of its own: the rows, the genotype counts and the x log2 x table."""
    ds = make_dataset("rows", seed=1800, S=70, cases=300, controls=290, k=3, top_n=10)
    for first, second in ((2, 3), (3, 2)):
        alone, both = fc.fc_load(ds.genotypes, ds.phenotype), fc.fc_load(ds.genotypes, ds.phenotype)
        fc.fc_search(both, first, 10)
        assert launches(fc, alone, second) - launches(fc, both, second) == 3


@pytest.mark.parametrize("slab_mb", [None, "1"])
@pytest.mark.parametrize("cases,controls", [(300, 290), (4200, 100)])
def test_any_order_of_searches(fc, monkeypatch, slab_mb, cases, controls):
    """1 MB: order 3 in several slabs, which gives its operands back."""
    if slab_mb:
        monkeypatch.setenv("FC_TRIPLES_SLAB_MB", slab_mb)
    ds = make_dataset("rows2", seed=1801, S=90, cases=cases, controls=controls, k=3, top_n=15)
    want = {k: oracle.search(ds.genotypes, ds.phenotype, k, 15)[:2] for k in (2, 3)}
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    for k in (3, 2, 3, 3, 2):
        idx, s = fc.fc_search(h, k, 15)
        assert fc.fc_last_search_kind(h) == (2 if k == 2 else 6)
        assert_topn_equal(idx, s, *want[k], lambda c: float(
            oracle.mi(oracle.tables(ds.genotypes, ds.phenotype, k, [c]), k)[0]))
    for enc in ("0", "1"):   # operands of the other form
        monkeypatch.setenv("FC_TRIPLES_ENC", enc)
        for k in (3, 2):
            assert np.array_equal(fc.fc_search(h, k, 15)[0], want[k][0])
