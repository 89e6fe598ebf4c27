"""Grouped FP32 Gram of more than 256 objects on both sides of the rule for the default tile caps (few tiles:
the small caps, many: the large ones), forward and adjoint, prepared with the default table left out and used
with it given by value. Against an FP64 transfer-matrix sweep: sums of 2 d products a chain, within 1e-5."""
import numpy as np
import pytest

from tests._util import TOL, assert_gram_blocks, rel_err

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("groups,size,rlo,rhi", [(2, 130, 2, 4), (65, 4, 2, 40), (3, 90, 2, 33)])
def test_default_caps(lib, groups, size, rlo, rhi):
    rng = np.random.default_rng(990)
    n, d = [2, 3, 2], 3
    ranks = [[1] + [int(v) for v in rng.integers(rlo, rhi + 1, d - 1)] + [1] for _ in range(groups * size)]
    objs = [[rng.normal(0, 1 / np.sqrt(r[k + 1]), (r[k], n[k], r[k + 1])).astype(np.float32) for k in range(d)] for r in ranks]
    X = lib.RaggedTT.from_objects(objs)
    gs = [size * g for g in range(groups + 1)]
    ws = lib.gram_groups_prepare(X, gs)
    out, norms = lib.gram_groups(X, gs, ws, tiles=lib.DEFAULT_TILES)
    full = [np.einsum("aib,bjc,ckd->aijkd", *[c.astype(np.float64) for c in o]).ravel() for o in objs]
    want = [np.stack(full[gs[g]:gs[g + 1]]) for g in range(groups)]
    G = np.concatenate([(w @ w.T).ravel() for w in want])
    assert_gram_blocks(out.cpu().numpy(), G, [size] * groups, TOL["fp32"])
    assert rel_err(norms.cpu().numpy(), np.concatenate([np.linalg.norm(w, axis=1) for w in want])) < TOL["fp32"]
    # the adjoint: <dX, X> summed over one core is the cotangent applied to the Gram, symmetrised
    dout = rng.standard_normal(G.size).astype(np.float32)
    dX = lib.gram_groups_backward(X, gs, ws, torch.tensor(dout, device="cuda")).double().cpu().numpy()
    for o in (0, size, groups * size - 1):
        g = o // size
        D = dout[g * size * size:(g + 1) * size * size].reshape(size, size).astype(np.float64)
        w = (D + D.T)[o - gs[g]] @ want[g]
        c = [x.astype(np.float64) for x in objs[o]]
        ref = np.einsum("ijk,aib,bjc->ckc".replace("ckc", "ck"), w.reshape(n), c[0], c[1])
        off = X.offsets[o] + c[0].size + c[1].size
        assert rel_err(dX[off:off + c[2].size], ref) < TOL["fp32"], o
