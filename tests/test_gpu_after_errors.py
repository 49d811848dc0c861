"""A call that the CUDA runtime refused (no launch configuration, no memory) is
reported once: the next call of the thread starts without its error."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from synth import make_dataset

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2201_03331_gb300 as fcm
    from paper_2201_03331_gb300 import build
    build.build()
    return fcm


@pytest.fixture(scope="module")
def small(fc):
    ds = make_dataset("aft", seed=1900, S=40, cases=200, controls=210, k=2, top_n=10)
    want = oracle.search(ds.genotypes, ds.phenotype, 2, 10)[0]

    def check():
        h = fc.fc_load(ds.genotypes, ds.phenotype)
        assert np.array_equal(fc.fc_search(h, 2, 10)[0], want)
    return check


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
def test_after_a_search_that_fits_nowhere(fc, small, k):
    """60,000 samples: the sweep's table alone exceeds shared memory."""
    ds = make_dataset("aft2", seed=1901, S=12, cases=30000, controls=30000, k=max(k, 2), top_n=10)
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    with pytest.raises(fc.FiunchoError):
        fc.fc_search(h, k, 10)
    small()


def test_after_an_allocation_that_fails(fc, small):
    """A bit table (24,576 bytes a SNP at 65,535 cases) of one and a half times
    the device's memory: the load ends at its allocation, before any genotype
    is read."""
    ph = torch.ones(65535, dtype=torch.uint8, device="cuda")
    S = int(1.5 * torch.cuda.mem_get_info()[1] / 24576)
    out = ctypes.c_void_p()
    assert fc.library().fc_load_device(ph.data_ptr(), S, len(ph), ph.data_ptr(), ctypes.byref(out)) == fc.FC_ENOMEM
    small()
