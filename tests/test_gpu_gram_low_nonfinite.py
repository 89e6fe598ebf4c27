"""Infinities through the low-rank FP32 Gram sweep and adjoint, at ranks that fill the compiled rank, ranks
padded up to it and unequal sides: partials that overflow FP32 on the way (half of A's objects are
scaled by 1e10 to 1e12 a core, d = 4), and one infinite core entry. All entries are positive, so an exact
product is inf or finite and never NaN: the infinities have to be those of the FP64 oracle cut to
FP32, and the finite entries within the stated 1e-5 normwise."""
import numpy as np
import pytest

import oracle as O
import synth as S
from tests._util import TOL, objects, rel_err, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _same(got, want):
    got = np.asarray(got, np.float64)
    want = np.where(np.abs(want) > np.finfo(np.float32).max, np.inf, want)
    assert not np.isnan(got).any() and not np.isnan(want).any()
    assert np.array_equal(np.isinf(got), np.isinf(want))
    fin = np.isfinite(want)
    assert not fin.any() or rel_err(got[fin], want[fin]) < TOL["fp32"]


@pytest.mark.parametrize("kind", ["overflow", "entry"])
@pytest.mark.parametrize("b,n,rA,rB", [
    (6, [2, 2, 2, 2], 1, 1),
    (6, [3, 2, 2, 3], 3, 2),
    (5, [3, 2, 2, 3], 5, 5),
    (6, [2, 3, 2, 2], 7, 6),
    (6, [2, 3, 2, 2], 9, 9),
    (7, [2, 3, 2, 2], 10, 7),
    (6, [2, 2, 2, 2], 12, 11),   # forward only above rank 10
    (6, [2, 2, 2, 2], 16, 13),
])
def test_gram_low_infinities(lib, b, n, rA, rB, kind):
    rng = np.random.default_rng(960)
    d = len(n)
    A, B = ([np.abs(c) for c in round32(S.random_tt(rng, b, n, [1] + [r] * (d - 1) + [1], 0.5))] for r in (rA, rB))
    if kind == "overflow":
        for c in A:
            c[: b // 2] *= 1e12 if rA == 1 else 1e10
        A = round32(A)
    else:
        B[1][0, 0, 0, 0] = np.inf
    Ad, Bd = (lib.TT.from_cores([np.asarray(c, np.float32) for c in X], device="cuda") for X in (A, B))
    _same(lib.gram(Ad, Bd).cpu().numpy(), O.gram(objects(A), objects(B)))
    if max(rA, rB) > 10:
        return
    g = np.ones((b, b), np.float32)
    dA, dB = lib.gram_backward(Ad, Bd, torch.tensor(g, device="cuda"))
    for got, want in zip((dA, dB), O.gram_vjp(objects(A), objects(B), g.astype(np.float64))):
        for k, c in enumerate(got.cores()):
            _same(c.cpu().numpy(), np.stack([o[k] for o in want]))
