"""The low-rank FP32 Gram sweep and adjoint (ranks to 16) over every compiled rank and the ranks just
below it, unequal sides, core-dependent ranks, tiles cut at the batch's end and shrunk for few objects,
one and two cores, and the neighbours that stay on the general kernels (rank 17, sides far apart,
the adjoint of few pairs above rank 10, BF16 storage). Against the FP64 oracle: sums of up to bB (bA) chains of 2 d products in FP32, within
the stated 1e-5 normwise."""
import numpy as np
import pytest

import oracle as O
import synth as S
from tests._util import TOL, objects, rel_err, rel_err_cores, round32, round_bf16

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bA,bB,n,rA,rB,bf16", [
    (100, 90, [3, 2, 4], [1, 3, 4, 1], [1, 4, 2, 1], False),
    (23, 41, [2, 3, 2], [1, 5, 6, 1], [1, 6, 5, 1], False),
    (33, 17, [3, 2, 2], [1, 8, 7, 1], [1, 7, 8, 1], False),
    (37, 44, [2, 2, 3], [1, 9, 10, 1], [1, 10, 7, 1], False),
    (9, 14, [2, 3, 2], [1, 11, 12, 1], [1, 12, 8, 1], False),
    (5, 3, [3, 2, 2], [1, 13, 14, 1], [1, 14, 10, 1], False),
    (18, 21, [2, 2, 2, 2], [1, 15, 16, 11, 1], [1, 16, 16, 16, 1], False),
    (37, 20, [3, 2, 2], [1, 12, 11, 1], [1, 9, 12, 1], False),
    (66, 64, [2, 3, 2], [1, 13, 16, 1], [1, 14, 15, 1], False),
    (60, 70, [2, 2, 2], [1, 14, 13, 1], [1, 13, 14, 1], False),
    (1, 1, [4, 3], [1, 10, 1], [1, 9, 1], False),
    (2, 300, [5], [1, 1], [1, 1], False),
    (150, 160, [2, 1], [1, 10, 1], [1, 10, 1], False),
    (5, 6, [3, 3, 2], [1, 15, 10, 1], [1, 16, 9, 1], True),
    (5, 6, [3, 3, 2], [1, 17, 10, 1], [1, 16, 9, 1], False),
    (5, 6, [3, 3, 2], [1, 5, 4, 1], [1, 16, 9, 1], False),
])
def test_gram_low(lib, bA, bB, n, rA, rB, bf16):
    rng = np.random.default_rng(950)
    rnd = round_bf16 if bf16 else round32
    A, B = rnd(S.random_tt(rng, bA, n, rA, 0.5)), rnd(S.random_tt(rng, bB, n, rB, 0.5))
    dt = torch.bfloat16 if bf16 else torch.float32
    Ad, Bd = lib.TT.from_cores(A, dtype=dt, device="cuda"), lib.TT.from_cores(B, dtype=dt, device="cuda")
    g = rng.standard_normal((bA, bB)).astype(np.float32)
    want = O.gram(objects(A), objects(B))
    assert rel_err(lib.gram(Ad, Bd).cpu().numpy(), want) < TOL["fp32"]
    dA, dB = lib.gram_backward(Ad, Bd, torch.tensor(g, device="cuda"))
    rdA, rdB = O.gram_vjp(objects(A), objects(B), g.astype(np.float64))
    for got, want in ((dA, rdA), (dB, rdB)):
        h = objects([c.double().cpu().numpy() for c in got.cores()])
        err = rel_err_cores([x for o in h for x in o], [x for o in want for x in o])
        assert err < TOL["fp32"], err
    # one side alone
    only, none = lib.gram_backward(Ad, Bd, torch.tensor(g, device="cuda"), need_B=False)
    assert none is None
    assert torch.allclose(only.data, dA.data, rtol=1e-4, atol=1e-5 * float(dA.data.abs().max()))
