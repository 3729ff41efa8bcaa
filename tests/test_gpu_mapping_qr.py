"""The mapping's factorisation at the edges of its register tiles: the smallest and largest
row counts (3 N_s, with the Tikhonov rows 3 N_s + 192 up to 960) and a count that is no
multiple of the block, against the oracle's SVD-based least squares.  Bound: the framework's
1e-7 per row (kappa eps64 of each side)."""
import numpy as np
import pytest

import oracle
import paper_2501_04684_gb300 as ie
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_samples,radius,tikhonov", [(64, 1.0, 1e-5), (86, 1.5, 0.0), (86, 1.5, 1e-4), (128, 1.5, 1e-5),
                                                       (256, 1.5, 1e-5)])
def test_rows_at_the_row_count_limits(n_samples, radius, tikhonov):
    a = W.BOX_EDGE
    fun_off, pos, mom = W.point_dipole_basis(np.full(3, 3), 960 + n_samples, a=a)
    P, res = ie.ie_map_basis(W.K0, W.ETA0, a, fun_off, pos, mom, n_samples=n_samples, sample_radius=radius,
                             tikhonov=tikhonov)
    Pr, rr = oracle.map_basis(W.K0, W.ETA0, a, 4, n_samples, radius, fun_off, pos, mom, tikhonov=tikhonov)
    err = np.linalg.norm(P - Pr, axis=1) / np.linalg.norm(Pr, axis=1)
    assert err.max() <= 1e-7
    assert np.allclose(res, rr, rtol=1e-6, atol=1e-12)
