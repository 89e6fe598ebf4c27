"""The bucketed completion adjoint over its chunk rules: four, two and one CTA per SM, both forms of the chains
(ranks to 4 and to 8), slices whose parts fill a warp, span warps or have one lane, warps whose items see no
tuple. FP32 against the FP64 oracle: sums of N products of d factors, within 1e-5 normwise."""
import numpy as np
import pytest

import oracle as O
import synth as S
from tests._util import TOL, objects, rel_err, rel_err_cores, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,r,N,riemannian", [
    ([4, 1, 1], 2, 4, False),        # one slice with hundreds of parts, four tuples
    ([4, 1, 1], 2, 5000, False),
    ([3, 2, 3], 8, 700, False),      # parts over several warps
    ([8, 8, 8], 5, 4, False),        # most warps see no tuple
    ([8, 8, 8], 4, 6000, True),
    ([10] * 8, 3, 2500, False),      # four CTAs per SM
    ([30, 20, 30, 20], 4, 900, True),
    ([4] * 30, 4, 600, False),       # one CTA per SM
    ([4] * 20, 6, 600, True),
    ([200, 3, 150], 1, 40000, False),
])
def test_completion_routes(lib, n, r, N, riemannian):
    rng = np.random.default_rng(945)
    d = len(n)
    X = round32(S.random_tt(rng, 1, n, [1] + [r] * (d - 1) + [1], 1.0))
    idx = np.stack([rng.integers(0, m, N) for m in n]).astype(np.int32)
    y = rng.standard_normal(N).astype(np.float32)
    it, yt = torch.tensor(idx, device="cuda"), torch.tensor(y, device="cuda")
    Xd = lib.TT.from_cores([np.asarray(c, np.float32) for c in X], device="cuda")
    host = lambda t: objects([c.double().cpu().numpy() for c in t.cores()])[0]
    if riemannian:
        U, V = lib.orthogonalize(Xd)
        dU, loss = lib.gather_backward(None, it, y=yt, want_loss=True, riemannian=True, U=U, V=V)
        L, want = O.riemannian_grad_completion(host(U), host(V), idx, y.astype(np.float64))
        assert rel_err_cores(host(dU), want) < TOL["fp32"]
    else:
        dX, loss = lib.gather_backward(Xd, it, y=yt, want_loss=True)
        w = O.gather(objects(X)[0], idx) - y
        L = 0.5 * np.sum(w * w)
        assert rel_err_cores(host(dX), O.gather_vjp(objects(X)[0], idx, w)) < TOL["fp32"]
    assert rel_err(loss.cpu().numpy(), np.array([L])) < TOL["fp32"]
