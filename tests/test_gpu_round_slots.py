"""Rounding at the heights where its columns take another number of register slots (32, 64, 128, 256 rows and
one more) and W R^T another number of row groups, with one kept column too (a 1 x 1 eigenproblem), against the
FP64 oracle. FP64 arithmetic and FP32 output: the FP32 tolerance holds per core."""
import numpy as np
import pytest

import oracle as O
from tests._util import TOL, objects, rel_err_cores, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,r,maxr", [
    ([32, 4, 9], [1, 9, 8, 1], 3),       # 32 rows, 32 rows of W
    ([97, 3, 11], [1, 20, 11, 1], 5),    # 33, 97
    ([96, 8, 8], [1, 30, 8, 1], 18),     # 64, 96; 18 kept rows
    ([33, 5, 13], [1, 30, 13, 1], 7),    # 65
    ([12, 16, 8], [1, 12, 8, 1], 4),     # 128
    ([12, 3, 43], [1, 12, 43, 1], 4),    # 129
    ([12, 32, 8], [1, 11, 8, 1], 4),     # 256
    ([12, 257, 3], [1, 5, 1, 1], 2),     # 257, rank 1
    ([5, 4, 3, 2], [1, 1, 1, 1, 1], 1),
])
def test_round_slots(lib, n, r, maxr):
    rng = np.random.default_rng(931)
    X = round32([rng.normal(0.0, 1.0 / np.sqrt(r[k + 1]), size=(2, r[k], n[k], r[k + 1])) for k in range(len(n))])
    Y = lib.round_tt(lib.TT.from_cores([np.asarray(c, np.float32) for c in X], device="cuda"), maxr)
    got = objects([c.double().cpu().numpy() for c in Y.cores()])
    assert Y.ranks == O.round_ranks(n, r, maxr)
    for j, Xo in enumerate(objects(X)):
        ref, _ = O.round_tt(Xo, maxr)
        assert rel_err_cores(got[j], ref) < TOL["fp32"], j
