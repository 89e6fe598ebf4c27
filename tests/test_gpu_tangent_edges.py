"""The one-kernel batched projection and the triangular tangent Gram at the edges of their tiles:
ranks 1 off the 8 / 16 / 32 paddings, unfoldings whose rows do not divide into eights or over a
cluster, more units than CTAs, batches of one 8-row block, one short of and at the full tile, and one
past it (the general kernel), coordinates that are no multiple of 4. FP32 against FP64: the
projection is a chain of 2 d products and a sum over at most r n rows, the Gram matrix a sum over the
coordinates whose terms' errors average out, both inside 1e-5 normwise."""
import numpy as np
import pytest

import oracle as O
import synth as S
from tests._util import TOL, batched, objects, rel_err, rel_err_cores, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _dev(lib, cores):
    return lib.TT.from_cores([np.asarray(c, np.float32) for c in cores], device="cuda")


def _host(tt):
    return [c.detach().double().cpu().numpy() for c in tt.cores()]


@pytest.mark.parametrize("batch,d,n,rX,rZ", [
    (120, 4, 16, 32, 8),   # 480 units over the SMs, full blocks
    (9, 4, 5, 31, 7),      # rows 155, columns 31
    (8, 3, 3, 17, 1),
    (127, 3, 4, 9, 8),
    (128, 3, 3, 8, 3),
    (129, 2, 3, 3, 2),     # past one tile
    (1, 5, 7, 16, 5),
    (3, 1, 6, 4, 3),       # d = 1
])
def test_projection_and_tangent_gram(lib, batch, d, n, rX, rZ):
    cfg = S.config5(seed=88, batch=batch, d=d, n=n, rX=rX, rZ=rZ)
    X, Z = round32(cfg.X), round32(cfg.Z)
    c = cfg.c.astype(np.float32)
    U, V = lib.orthogonalize(_dev(lib, X))
    Uh, Vh = objects(_host(U))[0], objects(_host(V))[0]
    P = lib.project(U, V, _dev(lib, Z), torch.tensor(c, device="cuda"))
    ref = O.project_batch(Uh, Vh, objects(Z), c.astype(np.float64))
    assert rel_err_cores(_host(P), batched(ref)) < TOL["fp32"]
    G = lib.tangent_gram(P, P).cpu().numpy()
    assert rel_err(G, O.tangent_gram(ref, ref)) < TOL["fp32"]
    # gauge projection on its own (the cluster kernel): the adjoint's first step
    rng = np.random.default_rng(89)
    bar = [rng.standard_normal(u.shape).astype(np.float32) for u in Uh]
    dZ, _ = lib.project_sum_backward(U, V, _dev(lib, Z), torch.tensor(c, device="cuda"),
                                     _dev(lib, [b[None] for b in bar]))
    rZb, _ = O.project_sum_vjp(Uh, Vh, objects(Z), c.astype(np.float64), [b.astype(np.float64) for b in bar])
    assert rel_err_cores(_host(dZ), batched(rZb)) < TOL["fp32"]
