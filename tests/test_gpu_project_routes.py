"""The batched projection on both sides of its rule (one kernel for large cores, two for small ones, the
line moving with the number of objects), and the sweeps on both sides of theirs (8 x 8 blocks where they
make four warps, else 4 x 4). FP32 against the FP64 oracle: chains of at most 2 d products of ranks to 32,
within the stated 1e-5 normwise."""
import numpy as np
import pytest

import oracle as O
import synth as S
from tests._util import TOL, objects, rel_err_cores, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("batch,d,n,rX,rZ", [
    (500, 3, 2, 12, 8),    # many small cores
    (310, 3, 16, 16, 4),   # 4096 elements a core, many
    (310, 3, 17, 16, 4),   # just above
    (40, 3, 8, 16, 5),     # 2048 elements a core, few
    (40, 3, 9, 15, 5),     # nine modes, few
    (650, 4, 1, 6, 3),     # one mode
    (620, 3, 8, 32, 8),    # 8 x 8 blocks
    (620, 3, 6, 30, 7),    # 8 x 8 blocks in the fused sweep alone
    (620, 3, 2, 32, 8),    # too few warps that way
])
def test_project_routes(lib, batch, d, n, rX, rZ):
    cfg = S.config5(seed=79, batch=batch, d=d, n=n, rX=rX, rZ=rZ)
    X, Z, c = round32(cfg.X), round32(cfg.Z), cfg.c.astype(np.float32)
    dev = lambda cs: lib.TT.from_cores([np.asarray(x, np.float32) for x in cs], device="cuda")
    host = lambda t: [x.double().cpu().numpy() for x in t.cores()]
    U, V = lib.orthogonalize(dev(X))
    Uh, Vh = objects(host(U))[0], objects(host(V))[0]
    Zd, ct, zo = dev(Z), torch.tensor(c, device="cuda"), objects(Z)
    got = objects(host(lib.project(U, V, Zd, ct)))
    some = [0, 1, batch // 2, batch - 1]
    for j, want in zip(some, O.project_batch(Uh, Vh, [zo[j] for j in some], c[some].astype(np.float64))):
        assert rel_err_cores(got[j], want) < TOL["fp32"], j
    want = O.project_sum(Uh, Vh, zo, c.astype(np.float64))
    assert rel_err_cores(host(lib.project_sum(U, V, Zd, ct)), [w[None] for w in want]) < TOL["fp32"]
