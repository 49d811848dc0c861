"""Sample limits of the dense outputs: what fits in shared memory by the
kernels' own size functions, and the calls at those limits."""
import ctypes
import itertools
import math

import numpy as np
import pytest

import oracle
from synth import make_dataset

SMEM = 232448   # bytes of shared memory a block may opt in to
LAST = 41471    # most samples the order-2 dense output takes


def size_functions():
    from paper_2201_03331_gb300 import build
    lib = ctypes.CDLL(build.build())
    stages = lib._ZN2fc12pairs_stagesEiim      # fc::pairs_stages(int M, int L, size_t cap)
    stages.argtypes, stages.restype = [ctypes.c_int, ctypes.c_int, ctypes.c_size_t], ctypes.c_int
    size = lib._ZN2fc16pairs_smem_bytesEiii    # fc::pairs_smem_bytes(int stages, int M, int L)
    size.argtypes, size.restype = [ctypes.c_int] * 3, ctypes.c_size_t
    return stages, size


@pytest.mark.parametrize("L", [0, 64, 1024, 2048])
def test_pair_stages_fit(L):
    """Two stages or more that fit, or none; a dump takes up to LAST samples."""
    stages, size = size_functions()
    for M in itertools.chain(range(2, 30000, 97), range(30000, 131071)):
        st = stages(M, L, SMEM)
        assert st == 0 or 2 <= st <= 6
        if st:
            assert size(st, M, L) <= SMEM
        if L == 0:
            assert (st > 0) == (M <= LAST), M


@pytest.fixture(scope="module")
def fc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2201_03331_gb300 as fcm
    from paper_2201_03331_gb300 import build
    build.build()
    return fcm


@pytest.mark.gpu
@pytest.mark.parametrize("M", [38271, 38272, 40000, LAST])
def test_pairs_dense_up_to_the_limit(fc, M):
    ds = make_dataset("lim", seed=1200, S=5, cases=M // 3, controls=M - M // 3, k=2, top_n=5)
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    sc, tab = fc.fc_pairs_dense(h, scores=True, tables=True)
    C = np.array(list(itertools.combinations(range(5), 2)), dtype=np.uint32)
    ref = oracle.tables(ds.genotypes, ds.phenotype, 2, C)
    assert np.array_equal(tab[C[:, 0], C[:, 1]], ref)
    bound = 2.0 ** -24 * (7.0 * math.log(M) + 19.0 * math.log(2.0))
    assert np.abs(sc[C[:, 0], C[:, 1]].astype(np.float64) - oracle.mi(ref, 2)).max() <= bound


@pytest.mark.gpu
@pytest.mark.parametrize("M", [LAST + 1, 41600, 131070])
def test_pairs_dense_refuses_more(fc, M):
    ds = make_dataset("lim", seed=1201, S=4, cases=M // 2, controls=M - M // 2, k=2, top_n=5)
    h = fc.fc_load(ds.genotypes, ds.phenotype)
    with pytest.raises(fc.FiunchoError) as e:
        fc.fc_pairs_dense(h)
    assert e.value.status == fc.FC_ERANGE
    if M < 50000:   # (the sweep takes over in searches while its table fits)
        assert len(fc.fc_search(h, 2, 3)[0]) == 3


@pytest.mark.gpu
@pytest.mark.parametrize("k,cases,controls,fits", [(3, 16383, 16383, True), (3, 16384, 100, False),
                                                   (4, 20736, 20735, True), (4, 30000, 30000, False)])
def test_higher_orders_at_their_limits(fc, k, cases, controls, fits):
    ds = make_dataset("lim", seed=1202, S=6, cases=cases, controls=controls, k=k, top_n=5)
    h = fc.fc_load(ds.genotypes, ds.phenotype)

    def dense():
        return fc.fc_triples_dense(h, scores=False, tables=True)[1] if k == 3 else \
            fc.fc_tuples_dense(h, k, scores=False, tables=True)[1]
    if not fits:
        with pytest.raises(fc.FiunchoError) as e:
            dense()
        assert e.value.status == fc.FC_ERANGE
        return
    C = np.array(list(itertools.combinations(range(6), k)), dtype=np.uint32)
    assert np.array_equal(dense(), oracle.tables(ds.genotypes, ds.phenotype, k, C))
