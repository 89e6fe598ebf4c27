"""The bucketed completion adjoint at the edges of its chunks: tuple counts around a chunk and a
full round of CTAs, one and two cores, more than 32 slices (the scan takes two passes), modes that
differ by core, all tuples in one slice, given weights, both rank paddings and the Riemannian form.
FP32 against the FP64 oracle: sums of N products of d factors, within 1e-5 normwise."""
import numpy as np
import pytest

import oracle as O
import synth as S
from tests._util import TOL, objects, rel_err, rel_err_cores, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _dev(lib, cores):
    return lib.TT.from_cores([np.asarray(c, np.float32) for c in cores], device="cuda")


def _host(tt):
    return objects([c.detach().double().cpu().numpy() for c in tt.cores()])[0]


@pytest.mark.parametrize("n,r,N,kind", [
    ([10] * 5, [1, 8, 8, 8, 8, 1], 127, "y"),
    ([10] * 5, [1, 8, 8, 8, 8, 1], 128, "y"),
    ([10] * 5, [1, 7, 8, 5, 3, 1], 257, "w"),
    ([6, 5, 6], [1, 4, 4, 1], 304 * 256 + 33, "y"),
    ([9], [1, 1], 500, "y"),
    ([7, 3], [1, 3, 1], 333, "w"),
    ([40, 3, 33], [1, 6, 5, 1], 1000, "y"),
    ([12, 2, 5, 30], [1, 2, 4, 8, 1], 777, "y"),
    ([10] * 6, [1, 8, 8, 8, 8, 8, 1], 3000, "one slice"),
    ([10] * 10, [1] + [8] * 9 + [1], 4001, "riemannian"),
    ([5, 13, 4], [1, 5, 4, 1], 129, "riemannian"),
])
def test_completion_edges(lib, n, r, N, kind):
    rng = np.random.default_rng(940)
    X = round32(S.random_tt(rng, 1, n, r, 1.0))
    idx = np.stack([rng.integers(0, m, N) for m in n]).astype(np.int32)
    if kind == "one slice":
        idx[:] = idx[:, :1]
    y = rng.standard_normal(N).astype(np.float32)
    it, yt = torch.tensor(idx, device="cuda"), torch.tensor(y, device="cuda")
    Xo = objects(X)[0]
    if kind == "riemannian":
        U, V = lib.orthogonalize(_dev(lib, X))
        dU, loss = lib.gather_backward(None, it, y=yt, want_loss=True, riemannian=True, U=U, V=V)
        Uh, Vh = _host(U), _host(V)
        L, want = O.riemannian_grad_completion(Uh, Vh, idx, y.astype(np.float64))
        assert rel_err_cores(_host(dU), want) < TOL["fp32"]
        assert rel_err(loss.cpu().numpy(), np.array([L])) < TOL["fp32"]
        return
    Xd = _dev(lib, X)
    if kind == "w":
        dX, _ = lib.gather_backward(Xd, it, w=yt)
        w = y.astype(np.float64)
    else:
        dX, loss = lib.gather_backward(Xd, it, y=yt, want_loss=True)
        w = O.gather(Xo, idx) - y
        assert rel_err(loss.cpu().numpy(), np.array([0.5 * np.sum(w * w)])) < TOL["fp32"]
    assert rel_err_cores(_host(dX), O.gather_vjp(Xo, idx, w)) < TOL["fp32"]
    again, _ = lib.gather_backward(Xd, it, **({"w": yt} if kind == "w" else {"y": yt}))
    assert rel_err(again.data.cpu().numpy(), dX.data.double().cpu().numpy()) < 1e-6
