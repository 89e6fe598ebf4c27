"""Orthogonalisation over both of its factorisations: tall unfoldings of up to 32 columns (two
exchanges, an FP32 preconditioner corrected in FP64), the same made ill-conditioned step by step
(second-order terms in FP64, then the Householder columns), 33 columns and wide unfoldings
(Householder columns), rows that do not divide over the cluster, inputs scaled out of FP32's range
for squares. FP64 output against the FP64 oracle: with condition numbers up to ~1e5 the factors
agree to ~1e-11 (condition x rounding x chain); Q is orthonormal to the same."""
import numpy as np
import pytest

import oracle as O
from tests._util import objects, rel_err_cores, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _cores(rng, n, r, near=None, scale=1.0):
    cores = [rng.normal(0.0, 1.0 / np.sqrt(r[k + 1]), size=(1, r[k], n[k], r[k + 1])) for k in range(len(n))]
    if near is not None:  # the last columns of every interior rank nearly repeat the first
        for c in cores[:-1]:
            c[..., -1] = c[..., 0] + near * c[..., -1]
    cores[0] = cores[0] * scale
    return round32(cores)


@pytest.mark.parametrize("n,r,near,scale", [
    ([40, 7, 9, 40], [1, 32, 32, 31, 1], None, 1.0),
    ([50, 5, 50], [1, 33, 33, 1], None, 1.0),          # 33 columns
    ([10, 10, 10, 10], [1, 8, 8, 8, 1], None, 1.0),    # 80 rows over 16 CTAs
    ([37, 3, 37], [1, 7, 7, 1], None, 1.0),            # odd columns, 21 rows
    ([4, 4, 4, 4], [1, 16, 20, 16, 1], None, 1.0),     # wide unfoldings, reduced ranks
    ([40, 8, 40], [1, 24, 24, 1], 1e-1, 1.0),
    ([40, 8, 40], [1, 24, 24, 1], 1e-2, 1.0),
    ([40, 8, 40], [1, 24, 24, 1], 1e-4, 1.0),
    ([40, 8, 40], [1, 24, 24, 1], None, 2.0 ** 80),
    ([40, 8, 40], [1, 24, 24, 1], None, 2.0 ** -90),
])
def test_orthogonalize_paths(lib, n, r, near, scale):
    X = _cores(np.random.default_rng(930), n, r, near, scale)
    Xd = lib.TT.from_cores([np.asarray(c, np.float32) for c in X], device="cuda")
    U, V = lib.orthogonalize(Xd, dtype=torch.float64)
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
