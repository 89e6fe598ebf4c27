"""Rounding at the edges of its kernel's paths: columns of 512 rows (the longest held in
registers) and longer ones, panels and column pairs with remainders, wide unfoldings, odd and
largest eigenproblems, each against the FP64 oracle. The arithmetic is FP64 and only the output
is FP32, so the FP32 tolerance holds element by element."""
import numpy as np
import pytest

import oracle as O
import synth as S
from tests._util import TOL, objects, rel_err_cores, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("case", [
    # seed, modes, ranks, max_rank
    (920, [8, 8, 8, 9], [1, 8, 64, 9, 1], 7),        # 512-row columns; 64 columns = 8 full panels
    (921, [8, 9, 9, 8], [1, 8, 58, 8, 1], 9),        # 522-row columns (through memory); 58 = 7 panels + 2
    (922, [2, 3, 5], [1, 30, 40, 1], 3),             # wide unfoldings (5 x 40, 15 x 30)
    (923, [10, 10, 10, 10], [1, 10, 120, 10, 1], 37),  # eigenproblem of side 100, odd kept rank
    (924, [3, 11, 3, 2], [1, 3, 6, 2, 1], 1),        # 33-row tail of a 32-row slot; rank 1
    (925, [5, 7, 5], [1, 5, 5, 1], 5),               # odd eigenproblems, nothing truncated
])
def test_round_edges(lib, case):
    seed, n, r, maxr = case
    rng = np.random.default_rng(seed)
    X = round32([rng.normal(0.0, 1.0 / np.sqrt(r[k + 1]), size=(2, r[k], n[k], r[k + 1])) for k in range(len(n))])
    Xd = lib.TT.from_cores([np.asarray(c, np.float32) for c in X], device="cuda")
    Y = lib.round_tt(Xd, maxr)
    got = objects([c.detach().double().cpu().numpy() for c in Y.cores()])
    for j, Xo in enumerate(objects(X)):
        ref, _ = O.round_tt(Xo, maxr)
        assert Y.ranks == O.round_ranks(n, r, maxr)
        assert rel_err_cores(got[j], ref) < TOL["fp32"], j


def test_round_zero_core(lib):
    # an all-zero core: every reflector of its unfolding is the identity, the result is zero
    rng = np.random.default_rng(926)
    X = round32(S.random_tt(rng, 1, [3, 4, 3], [1, 3, 3, 1]))
    X[1] = np.zeros_like(X[1])
    Y = lib.round_tt(lib.TT.from_cores([np.asarray(c, np.float32) for c in X], device="cuda"), 2)
    full = O.full(objects([c.detach().double().cpu().numpy() for c in Y.cores()])[0])
    assert np.all(full == 0.0)
