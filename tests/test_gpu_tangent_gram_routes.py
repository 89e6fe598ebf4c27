"""The self Gram matrix of tangent vectors on both sides of its rule (upper triangle, or the full tile for few
coordinates and for one team of threads), with coordinate counts that are no multiple of four. FP32 against
FP64 inner products of the same coordinates: sums of at most 10^5 products, within 1e-5 of the norms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,r,batch", [
    ([8, 8, 8], [1, 24, 24, 1], 25),          # 312 chunks: the tile
    ([8, 9, 8], [1, 24, 24, 1], 25),          # 348 chunks: the triangle
    ([10, 7, 9, 11], [1, 13, 31, 13, 1], 120),
    ([10, 7, 9, 11], [1, 13, 31, 13, 1], 121),
    ([16] * 8, [1] + [32] * 7 + [1], 128),    # 20 chunks a CTA: the triangle by one team
    ([3], [1, 1], 128),
    ([2, 2], [1, 1, 1], 1),
])
def test_tangent_gram_routes(lib, n, r, batch):
    g = torch.Generator(device="cuda")
    g.manual_seed(980)
    size = sum(r[k] * n[k] * r[k + 1] for k in range(len(n)))
    D = lib.TT(torch.randn(size * batch, generator=g, device="cuda"), n, r, batch)
    got = lib.tangent_gram(D, D).double()
    want = torch.zeros(batch, batch, dtype=torch.float64, device="cuda")
    for c in D.cores():
        m = c.reshape(batch, -1).double()
        want += m @ m.T
    scale = torch.sqrt(torch.outer(want.diagonal(), want.diagonal()))
    assert float(((got - want).abs() / scale).max()) < 1e-5
    assert torch.equal(got, got.T)
