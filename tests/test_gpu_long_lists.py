"""Order 3 with the longest lists beside the tables of the most samples: the
tensor cores (from 31,616 samples with shorter candidate buffers) and the
sweep's list."""
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


@pytest.mark.parametrize("cases,controls", [(15000, 15336), (15232, 16383), (15233, 16383), (16383, 16383)])
@pytest.mark.parametrize("n", [820, 1638])
def test_lists_of_2048(fc, monkeypatch, cases, controls, n):
    ds = make_dataset("long", seed=1700, S=200, cases=cases, controls=controls, k=3, top_n=n)
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    try:
        a = fc.fc_search(h, 3, n)
    except fc.FiunchoError as e:
        # More candidates within the error window than the longest list holds
        # are refused on either path.
        assert n == 1638 and e.status == fc.FC_ERANGE
        monkeypatch.setenv("FC_TRIPLES_PATH", "popc")
        with pytest.raises(fc.FiunchoError, match="4096 candidates"):
            fc.fc_search(h, 3, n)
        return
    assert fc.fc_last_search_kind(h) == 6 and len(a[1]) == n
    monkeypatch.setenv("FC_TRIPLES_PATH", "popc")
    b = fc.fc_search(h, 3, n)
    assert fc.fc_last_search_kind(h) == 3
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
