"""The error word of t3f_project's workspace is this call's: whatever a workspace held before, a call whose
waits all end leaves 0 there (register-tiled sweeps and the general ones)."""
import ctypes

import pytest

import synth as S
from tests._util import round32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("rx,rz", [(4, 3), (9, 8), (33, 3), (5, 9)])
def test_project_clears_its_error_word(lib, rx, rz):
    import numpy as np
    b = lib._binding
    n, batch = [8, 9, 8], 5
    rng = np.random.default_rng(970)
    tt = lambda bt, r: lib.TT.from_cores([np.asarray(c, np.float32) for c in round32(S.random_tt(rng, bt, n, [1, r, r, 1], 0.5))],
                                         device="cuda")
    X, Z = tt(1, rx), tt(batch, rz)
    U, V = lib.orthogonalize(X)
    want = lib.project(U, V, Z)
    ws = b.workspace("project", U, Z)
    ws[:4].view(torch.int32).fill_(-6)
    out = lib.TT.empty(U.n, U.ranks, batch, device="cuda")
    st = lib.load().t3f_project(b._ref(U), b._ref(V), b._ref(Z), None, b._ref(out), b._ptr(ws), ws.numel(),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    assert lib.device_status(ws) == 0
    assert torch.equal(out.data, want.data)
