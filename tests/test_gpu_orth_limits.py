"""Orthogonalisation at its documented limits (ranks to 64, r n = 4096): the largest interior cores, whose
rows fill a CTA's share of the working region to the last element, and the sizes just below them.
FP64 output against the FP64 oracle, with the bound of the smaller shapes: the square boundary
unfoldings (64 x 64 Gaussian) have condition numbers below 1e4, so the factors agree to condition x
rounding x sqrt(columns) x chain < 1e4 * 1.1e-16 * 8 * 8 = 7e-11 < 1e-10."""
import numpy as np
import pytest

import oracle as O
from tests._util import objects, rel_err_cores, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,r", [
    ([64, 64, 64], [1, 64, 64, 1]),
    ([64, 64, 64, 64], [1, 64, 64, 64, 1]),
    ([64, 63, 64], [1, 64, 64, 1]),   # 4032 rows
    ([64, 64, 64], [1, 63, 64, 1]),   # 4032 rows, 64 columns
    ([64, 64, 64], [1, 64, 63, 1]),   # 4096 rows, 63 columns
])
def test_orthogonalize_limits(lib, n, r):
    rng = np.random.default_rng(940)
    X = round32([rng.normal(0.0, 1.0 / np.sqrt(r[k + 1]), size=(1, r[k], n[k], r[k + 1])) for k in range(len(n))])
    U, V = lib.orthogonalize(lib.TT.from_cores([np.asarray(c, np.float32) for c in X], device="cuda"), dtype=torch.float64)
    Ur, Vr, rr = O.orthogonalize(objects(X)[0])
    assert U.ranks == rr and V.ranks == rr
    Ug = objects([c.cpu().numpy() for c in U.cores()])[0]
    Vg = objects([c.cpu().numpy() for c in V.cores()])[0]
    for k in range(len(n)):
        assert rel_err_cores([Ug[k]], [Ur[k]]) < 1e-10, ("U", k)
        assert rel_err_cores([Vg[k]], [Vr[k]]) < 1e-10, ("V", k)
    for k in range(len(n) - 1):
        M = Ug[k].reshape(-1, Ug[k].shape[-1])
        assert np.abs(M.T @ M - np.eye(M.shape[1])).max() < 1e-11, k
