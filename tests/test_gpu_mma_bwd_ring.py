"""Tensor-core Gram adjoint of uniform batches with many gradient items per thread block: the items of
a block follow one another without a barrier, so buffers, phases and tables carry over from item to
item. Cores of one mode (one slice an item), both sides or one, rank classes 16, 32 and 64 on either
side. Against the FP64 oracle at the math's stated tolerance, each object on its own."""
import numpy as np
import pytest

import oracle as O
import synth as S
from tests._util import TOL, objects, rel_err_cores, round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("math_", ["tf32", "bf16"])
@pytest.mark.parametrize("bA,bB,n,rA,rB,sides", [
    (27, 25, [1, 2, 3, 1], [1, 40, 33, 20, 1], [1, 45, 64, 50, 1], "AB"),
    (41, 40, [2, 1, 2], [1, 30, 7, 1], [1, 12, 16, 1], "A"),
    (33, 47, [1, 1, 5], [1, 5, 11, 1], [1, 35, 21, 1], "B"),
])
def test_gram_backward_many_items(lib, bA, bB, n, rA, rB, sides, math_):
    rng = np.random.default_rng(1150)
    A = round32(S.random_tt(rng, bA, n, rA, 1.0 / np.sqrt(max(rA))))
    B = round32(S.random_tt(rng, bB, n, rB, 1.0 / np.sqrt(max(rB))))
    dG = rng.normal(size=(bA, bB)).astype(np.float32)
    dev = lambda c: lib.TT.from_cores([torch.tensor(np.asarray(x)) for x in c], dtype=torch.float32, device="cuda")
    tA, tB = dev(A), dev(B)
    ws = lib.workspace("gram_bwd_tc", tA, tB)
    got = lib.gram_backward(tA, tB, torch.tensor(dG, device="cuda"), math=math_, ws=ws, need_A="A" in sides,
                            need_B="B" in sides)
    assert lib.device_status(ws) == 0
    for side, g, want in zip("AB", got, O.gram_vjp(objects(A), objects(B), dG.astype(np.float64))):
        assert (g is not None) == (side in sides)
        if g is not None:
            h = objects([c.double().cpu().numpy() for c in g.cores()])
            for o, w in zip(h, want):
                assert rel_err_cores(o, w) < TOL[math_]
