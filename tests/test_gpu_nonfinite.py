"""A non-finite element of H0, or one beyond FP32, in a single block: reported by every submatrix that holds the block,
also where it lies outside the centre columns, and by no other.

One cluster of molecules on either side of 192 rows (operands kept on the SM or streamed), each followed by the same one
without the element; every submatrix of a cluster holds all of its blocks. The element makes A_J = T_J(S)^-1 T_J(H0) non-finite
in FP32, the sign iteration reports it, and so does the FP64 path that the submatrix is handed to. 1e39 is finite there, but
beyond the FP32 Gershgorin interval that scales the iteration."""
import numpy as np
import pytest

from test_gpu_tile_edges import MU, clusters, lattice_pair

pytestmark = pytest.mark.gpu

SIZES = (100, 100, 230, 230)


@pytest.fixture(scope="module")
def nl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_08245_gb300 import build
    build.build()
    import paper_2104_08245_gb300 as nl
    return nl


def with_element(value):
    """The system, its molecules per cluster, and the two molecules whose block holds the element in clusters 0 and 2."""
    sysm, _ = clusters(SIZES, lattice_pair, 0.5)
    of = np.repeat(np.arange(len(SIZES)), [int(np.sum(np.cumsum(sysm.nbf) <= e)) - int(np.sum(np.cumsum(sysm.nbf) <= e - n))
                                           for n, e in zip(SIZES, np.cumsum(SIZES))])
    owners = []
    for c in (0, 2):
        I, J = np.flatnonzero(of == c)[[2, 6]]
        owners += [I, J]
        for a, b in ((I, J), (J, I)):
            p = sysm.H.row_ptr[a] + int(np.flatnonzero(sysm.H.col_idx[sysm.H.row_ptr[a]:sysm.H.row_ptr[a + 1]] == b)[0])
            sysm.H.vals[sysm.H.blk_off[p]] = value
    return sysm, of, owners


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e39])
@pytest.mark.parametrize("prec,inverse", [("bf16x3", 0), ("bf16x3", 1), ("fp32", 1), ("fp16", 1), ("fp64", 0)])
def test_every_submatrix_that_holds_the_element_reports_it(nl, prec, inverse, value):
    sysm, of, owners = with_element(value)
    plan = nl.nolsm_build_submatrices(nl.DeviceSystem(sysm))
    o = nl.options(prec, inverse=inverse)
    r = nl.nolsm_solve_batch(plan, MU, o, check=False)
    st = r.sub_status.cpu().numpy()
    print(f"{prec} ({inverse}), {value}: {np.unique(st[of == 0])} {np.unique(st[of == 1])} {np.unique(st[of == 2])} {np.unique(st[of == 3])}")
    assert np.all(st[(of == 1) | (of == 3)] == 0)
    assert np.all(st[(of == 0) | (of == 2)] != 0)
    if not np.isfinite(value):
        assert np.all(st[(of == 0) | (of == 2)] == nl._abi.ERR_NONFINITE)
    assert r.status != 0
    plan.close()


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e39])
def test_a_range_without_the_owners_of_the_block_reports_it(nl, value):
    sysm, of, owners = with_element(value)
    plan = nl.nolsm_build_submatrices(nl.DeviceSystem(sysm))
    for c in (0, 2):
        first = int(np.flatnonzero(of == c)[0])
        r = nl.nolsm_solve_batch(plan, MU, nl.options("bf16x3", inverse=1, sub_begin=first, sub_end=first + 2), check=False)
        assert r.status != 0 and np.all(r.sub_status.cpu().numpy()[first:first + 2] != 0)
    plan.close()
