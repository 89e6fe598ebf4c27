"""project_sum, its adjoint and the batched projection over the block shapes of their sweeps:
few and many objects per CTA (the rule changes at four per SM), ranks at the edges of the 8 / 16 /
32 paddings, more slices at a time than the mode has, modes that do not divide them. FP32 against
the FP64 oracle: every output is a chain of at most 2 d rank-32 products, so the stated FP32
tolerance (1e-5 normwise) holds."""
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
    (500, 3, 5, 32, 8),    # 8 x 8 / 8 x 4 blocks, 8 slices at a time over 5
    (470, 4, 3, 13, 3),    # padded to 16, ranks that are no multiple of 4
    (610, 3, 4, 7, 8),     # padded to 8, 5 objects per CTA
    (160, 4, 7, 32, 8),    # 4 x 4 blocks, 2 objects per CTA
    (1, 3, 17, 20, 6),     # one object, more slices than fit at a time
    (2, 3, 33, 8, 5),
    (5, 1, 6, 4, 3),       # d = 1
])
def test_psweep_shapes(lib, batch, d, n, rX, rZ):
    cfg = S.config5(seed=77, batch=batch, d=d, n=n, rX=rX, rZ=rZ)
    X, Z = round32(cfg.X), round32(cfg.Z)
    c = cfg.c.astype(np.float32)
    U, V = lib.orthogonalize(_dev(lib, X))
    Uh, Vh = objects(_host(U))[0], objects(_host(V))[0]
    Zd, ct = _dev(lib, Z), torch.tensor(c, device="cuda")
    dU = lib.project_sum(U, V, Zd, ct)
    assert rel_err_cores(_host(dU), [r[None] for r in O.project_sum(Uh, Vh, objects(Z), c.astype(np.float64))]) < TOL["fp32"]
    rng = np.random.default_rng(78)
    bar = [rng.standard_normal(u.shape).astype(np.float32) for u in Uh]
    dZ, dc = lib.project_sum_backward(U, V, Zd, ct, _dev(lib, [b[None] for b in bar]))
    rZb, rc = O.project_sum_vjp(Uh, Vh, objects(Z), c.astype(np.float64), [b.astype(np.float64) for b in bar])
    assert rel_err_cores(_host(dZ), batched(rZb)) < TOL["fp32"]
    assert rel_err(dc.cpu().numpy(), rc) < TOL["fp32"]
    few = objects(Z)[:3]
    P = lib.project(U, V, _dev(lib, batched(few)), ct[:len(few)].contiguous())
    ref = O.project_batch(Uh, Vh, few, c[:len(few)].astype(np.float64))
    for j, got in enumerate(objects(_host(P))):
        assert rel_err_cores(got, ref[j]) < TOL["fp32"], j
