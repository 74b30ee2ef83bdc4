"""GPU: the FP32 sweeps of the mixed factors as products over levels (rank above 32), at
the edges of their blocks (1, 31, 33, 127, 128, 129 and more eliminated columns, none),
of the column counts (4, 8, 16) and on two refinement lanes."""
import numpy as np
import pytest

from oracle import ulv as O
from paper_2311_00921_gb300 import hss
from paper_2311_00921_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf,rank,nrhs,lanes", [
    (34, 33, 1, 1), (64, 33, 4, 1), (72, 39, 5, 1), (40, 40, 3, 1), (161, 34, 8, 1), (163, 35, 9, 2),
    (164, 35, 16, 1), (300, 130, 17, 1), (420, 64, 7, 2)])
def test_mixed_sweeps_against_oracle(leaf, rank, nrhs, lanes):
    h = I.random_hss(3, leaf, rank, seed=leaf + rank, orthonormal=False)
    b = I.rhs(h.n, nrhs, 5)
    x_ref = O.solve(O.factor(h), b).reshape(b.shape)
    dev = hss.HSS(h)
    dev.factorize("fp32", ir_lanes=lanes)
    x = dev.solve(hss.colmajor(b)).cpu().numpy().reshape(b.shape)
    err = np.linalg.norm(x - x_ref, axis=0) / np.linalg.norm(x_ref, axis=0)
    assert err.max() <= 1e-10
    # a sound FP32 solve leaves 1e-3 of the error at most, so that four corrections
    # reach the tolerance of 1e-12; a wrong block would not contract
    assert dev.last_info()["ir_iters"] <= 4
