"""The low-rank FP32 Gram forward on both sides of its rules for many pairs: ranks to 4 with the row test,
ranks to 2 and unequal high ranks handed to the general kernel, ranks 11 and 12. FP32 against an FP64
transfer-matrix sweep: sums of 2 d products a chain, within 1e-5 normwise."""
import numpy as np
import pytest

import synth as S
from tests._util import TOL, rel_err, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bA,bB,n,rA,rB", [
    (151, 150, [2, 3, 2], [1, 3, 3, 1], [1, 2, 3, 1]),    # just below 150 pairs an SM
    (152, 151, [2, 3, 2], [1, 3, 3, 1], [1, 2, 3, 1]),    # row test
    (275, 276, [2, 3, 2], [1, 2, 2, 1], [1, 2, 1, 1]),    # 500 pairs an SM
    (277, 277, [2, 3, 2], [1, 2, 2, 1], [1, 1, 2, 1]),
    (676, 675, [2, 2], [1, 2, 1], [1, 2, 1]),             # 3000 pairs an SM
    (174, 174, [2, 3, 2], [1, 5, 4, 1], [1, 4, 4, 1]),    # 200 pairs an SM, sides 5 and 4
    (175, 174, [2, 3, 2], [1, 5, 4, 1], [1, 4, 4, 1]),
    (83, 84, [3, 2, 2], [1, 12, 11, 1], [1, 11, 12, 1]),  # 46 pairs an SM
    (84, 84, [3, 2, 2], [1, 12, 11, 1], [1, 11, 12, 1]),
    (98, 100, [2, 2, 2], [1, 14, 12, 1], [1, 13, 14, 1]),  # an inner core of rank 12
    (98, 100, [2, 2, 2], [1, 14, 13, 1], [1, 13, 14, 1]),
])
def test_gram_low_routes(lib, bA, bB, n, rA, rB):
    rng = np.random.default_rng(955)
    A, B = round32(S.random_tt(rng, bA, n, rA, 0.5)), round32(S.random_tt(rng, bB, n, rB, 0.5))
    M = np.ones((bA, bB, 1, 1))
    for a, b in zip(A, B):
        M = sum(np.einsum("abix,aij->abjx", np.einsum("abix,bxy->abiy", M, b[:, :, i], optimize=True), a[:, :, i],
                          optimize=True) for i in range(a.shape[2]))
    Ad, Bd = (lib.TT.from_cores([np.asarray(c, np.float32) for c in X], device="cuda") for X in (A, B))
    assert rel_err(lib.gram(Ad, Bd).cpu().numpy(), M[:, :, 0, 0]) < TOL["fp32"]
