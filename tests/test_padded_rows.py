"""Rows are padded only for the grids that the TMA-pipelined kernel serves
(host-side sizes; no GPU)."""
import pytest

import paper_1904_12553_gb300 as P
from paper_1904_12553_gb300 import workloads as W


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1904_12553_gb300 import build
    build.build()


def nbytes(nx, ny, rho):
    return P.lbm_nphase_workspace_bytes(
        W.base_params(3, nx, ny, 0.01, rho=rho, precision="fp32"))


@pytest.mark.parametrize("nx,ny", [(1, 200000), (9, 20000), (33, 5000), (57, 40000), (63, 20000),
                                   (301, 203), (20001, 9)])
def test_narrow_and_small_grids_stay_dense(nx, ny):
    """As many bytes as the same grid with unequal densities, whose rows are
    never padded."""
    assert nbytes(nx, ny, None) == nbytes(nx, ny, [3.0, 1.0, 2.0])


@pytest.mark.parametrize("nx,ny", [(1501, 997), (97, 5000)])
def test_large_grids_are_padded(nx, ny):
    dense = nbytes(nx, ny, [3.0, 1.0, 2.0])
    assert dense < nbytes(nx, ny, None) <= dense * 1.1
