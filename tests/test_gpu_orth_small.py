"""Orthogonalisation on both sides of its rule for small unfoldings (Householder columns up to three and for
square ones up to five, two exchanges above), with batches, reduced ranks and modes that leave CTAs without
rows. FP64 output against the FP64 oracle: condition numbers below 1e4, rounding and chains of at most eight
cores, so 1e-10."""
import numpy as np
import pytest

import oracle as O
from tests._util import objects, rel_err_cores, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("batch,n,r", [
    (1, [5, 3, 8], [1, 1, 1, 1]),
    (3, [8, 8, 8, 8], [1, 2, 2, 2, 1]),
    (2, [20, 3, 20], [1, 3, 3, 1]),
    (1, [30, 4, 30], [1, 4, 3, 1]),
    (2, [4, 4, 4], [1, 4, 4, 1]),          # square boundary unfoldings of four columns
    (2, [5, 6, 5], [1, 5, 5, 1]),
    (2, [6, 4, 6], [1, 6, 6, 1]),          # square, six columns: two exchanges
    (3, [4, 40], [1, 39, 1]),              # ranks reduced to four
    (1, [2] * 8, [1, 2, 3, 4, 5, 4, 3, 2, 1]),
])
def test_orthogonalize_small(lib, batch, n, r):
    rng = np.random.default_rng(941)
    X = round32([rng.normal(0.0, 1.0 / np.sqrt(r[k + 1]), size=(batch, r[k], n[k], r[k + 1])) for k in range(len(n))])
    U, V = lib.orthogonalize(lib.TT.from_cores([np.asarray(c, np.float32) for c in X], device="cuda"), dtype=torch.float64)
    Uh, Vh = (objects([c.cpu().numpy() for c in t.cores()]) for t in (U, V))
    for b, x in enumerate(objects(X)):
        Ur, Vr, rr = O.orthogonalize(x)
        assert U.ranks == rr and V.ranks == rr
        for k in range(len(n)):
            assert rel_err_cores([Uh[b][k]], [Ur[k]]) < 1e-10, ("U", b, k)
            assert rel_err_cores([Vh[b][k]], [Vr[k]]) < 1e-10, ("V", b, k)
