"""Performance cases of the TT-sweep library: what its users call, at the sizes they call it.

Every case is one pass through public entry points (`autograd.gram`, `autograd.completion_loss`,
`autograd.project_sum`, `gather_backward`, `matvec`, `orthogonalize`, `gram_groups`, `project`,
`tangent_gram`, `round_tt`, ...) on synthetic TT objects with cores N(0, 1/sqrt(r)), the
distribution of the repository's own benchmark. `draw` spreads the sizes of each kind of call over
its whole range. The references of `exact` are plain torch / numpy in FP64.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1801_01928_gb300 as t3f
from paper_1801_01928_gb300 import autograd as t3f_ad

DEV = "cuda"


def listed():
    return [
        # a handful of small tensors: the call an interactive user makes; launch latency
        {"name": "gram_tiny", "kind": "gram", "bA": 8, "bB": 8, "d": 4, "n": 3, "r": 2, "grad": False},
        # all pairwise inner products of two batches of 100 and their gradient (kernel learning
        # on TT features; the paper's 'gram' row with its batch of 100 and rank 10)
        {"name": "gram_train", "kind": "gram", "bA": 100, "bB": 100, "d": 10, "n": 10, "r": 10, "grad": True},
        # stochastic tensor completion: a mini-batch with odd sizes (loss and core gradient)
        {"name": "completion_minibatch", "kind": "completion", "N": 20011, "d": 7, "n": 13, "r": 5},
        # tensor completion over all observed entries: loss and gradient per optimiser step
        {"name": "completion_full", "kind": "completion", "N": 1000000, "d": 10, "n": 10, "r": 8},
        # Riemannian gradient descent on the same problem: orthogonal forms at the iterate, then
        # the projected gradient and the loss
        {"name": "riemannian_step", "kind": "riemannian", "N": 1000000, "d": 10, "n": 10, "r": 8},
        # 100 TT-matrix by TT-vector products and their gradient (the paper's 'matvec' row)
        {"name": "matvec_train", "kind": "matvec", "batch": 100, "d": 10, "m": 4, "n": 4, "rA": 10, "rx": 10},
        # 512 objects of uneven order, mode size and rank: Gram matrices within groups of 64,
        # norms and gradient, FP32 throughout
        {"name": "uneven_fp32", "kind": "uneven", "groups": 8, "per_group": 64, "shape_seed": 5, "math": "fp32"},
        # the same collection stored in BF16, on the tensor cores
        {"name": "uneven_bf16", "kind": "uneven", "groups": 8, "per_group": 64, "shape_seed": 5, "math": "bf16"},
        # weighted sum of 1000 TTs projected on the tangent space of a rank-32 point, and its
        # gradient w.r.t. the 1000 objects and the weights
        {"name": "project_sum_train", "kind": "psum", "batch": 1000, "d": 20, "n": 16, "rX": 32, "rZ": 8},
        # left- and right-orthogonal forms of one rank-32 object (the start of every Riemannian
        # operation at that point)
        {"name": "orthogonalize", "kind": "orth", "d": 20, "n": 16, "r": 32},
        # 100 tangent vectors of one tangent space and their Gram matrix
        {"name": "tangent_gram", "kind": "tangent", "batch": 100, "d": 20, "n": 16, "rX": 32, "rZ": 8},
        # recompression of 100 rank-100 objects (products of rank-10 TT-matrices and TT-vectors)
        # to rank 10
        {"name": "round", "kind": "round", "batch": 100, "d": 10, "n": 4, "rA": 10, "rx": 10, "max_rank": 10},
    ]


# ---------------------------------------------------------------------------------------------
# drawn cases
# ---------------------------------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_gram(rng):
    while True:
        c = {"kind": "gram", "bA": _log_int(rng, 4, 128), "bB": _log_int(rng, 4, 128), "d": rng.randint(3, 16),
             "n": rng.randint(2, 16), "r": _log_int(rng, 2, 48), "grad": rng.random() < 0.7}
        if work(c)["flops"] <= 2e10:
            return c


def _draw_completion(rng):
    while True:
        c = {"kind": rng.choice(["completion", "riemannian"]), "N": _log_int(rng, 1000, 1000000),
             "d": rng.randint(3, 12), "n": rng.randint(3, 20), "r": rng.randint(2, 8)}
        # the cores of the model stay in one thread block's shared memory
        if c["d"] * c["n"] <= 130:
            return c


def _draw_matvec(rng):
    return {"kind": "matvec", "batch": _log_int(rng, 4, 100), "d": rng.randint(3, 10), "m": rng.randint(2, 5),
            "n": rng.choice([2, 3, 4, 5]), "rA": rng.randint(2, 10), "rx": rng.randint(2, 10)}


def _draw_uneven(rng):
    return {"kind": "uneven", "groups": rng.randint(1, 8), "per_group": rng.randint(8, 64),
            "shape_seed": rng.randint(0, 10 ** 6), "math": rng.choice(["fp32", "bf16"])}


def _draw_psum(rng):
    return {"kind": "psum", "batch": _log_int(rng, 10, 1000), "d": rng.randint(4, 20), "n": rng.randint(3, 16),
            "rX": rng.randint(8, 32), "rZ": rng.randint(2, 8)}


def _draw_orth(rng):
    return {"kind": "orth", "d": rng.randint(4, 20), "n": rng.randint(4, 16), "r": rng.randint(4, 32)}


def _draw_tangent(rng):
    return {"kind": "tangent", "batch": _log_int(rng, 8, 100), "d": rng.randint(4, 20), "n": rng.randint(3, 16),
            "rX": rng.randint(8, 32), "rZ": rng.randint(2, 8)}


def _draw_round(rng):
    return {"kind": "round", "batch": _log_int(rng, 8, 100), "d": rng.randint(4, 10), "n": rng.randint(3, 5),
            "rA": rng.randint(3, 10), "rx": rng.randint(3, 10), "max_rank": rng.randint(4, 12)}


_DRAWS = [_draw_gram, _draw_completion, _draw_matvec, _draw_uneven, _draw_psum, _draw_orth, _draw_tangent, _draw_round]


def draw(rng):
    return rng.choice(_DRAWS)(rng)


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------

def _ranks(d, r):
    return [1] + [r] * (d - 1) + [1]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _tt_cores(gen, batch, d, n, r, m=None):
    """d core blocks [batch][r0][(m)][n][r1], N(0, 1/sqrt(r)), FP32."""
    rk = _ranks(d, r)
    mid = [n] if m is None else [m, n]
    return [torch.randn([batch, rk[k]] + mid + [rk[k + 1]], generator=gen, device=DEV) / math.sqrt(r) for k in range(d)]


def _pack(cores):
    return torch.cat([c.reshape(-1) for c in cores])


def _chains(cores, idx):
    """X(i_t) of a batch-1 TT, and the prefix rows it goes through."""
    v = torch.ones(idx.shape[1], 1, dtype=cores[0].dtype, device=DEV)
    pre = [v]
    for k, c in enumerate(cores):
        v = torch.bmm(v[:, None, :], c[0].permute(1, 0, 2)[idx[k].long()])[:, 0]
        pre.append(v)
    return v[:, 0], pre


def _qr_pos(w):
    q, r = np.linalg.qr(w)
    s = np.where(np.diagonal(r) < 0, -1.0, 1.0)
    return q * s, r * s[:, None]


def _right_sweep(cores):
    cores = list(cores)
    for k in range(len(cores) - 1, 0, -1):
        r0, n, r1 = cores[k].shape
        q, r = _qr_pos(cores[k].reshape(r0, n * r1).T)
        cores[k] = q.T.reshape(-1, n, r1)
        cores[k - 1] = cores[k - 1] @ r.T
    return cores


def _left_sweep(cores):
    cores = list(cores)
    for k in range(len(cores) - 1):
        r0, n, r1 = cores[k].shape
        q, r = _qr_pos(cores[k].reshape(r0 * n, r1))
        cores[k] = q.reshape(r0, n, -1)
        cores[k + 1] = np.einsum("ab,bnc->anc", r, cores[k + 1])
    return cores


def _orth_forms(cores):
    """Left- and right-orthogonal forms (FP64 numpy lists) of a batch-1 TT."""
    u = _left_sweep(_right_sweep([c[0].double().cpu().numpy() for c in cores]))
    return u, _right_sweep(u)


def _group_shapes(case):
    """Per group (d, n, ranks of its objects): d in [4, 16], n in [2, 16], ranks log-uniform in [2, 64]."""
    rng = random.Random(case["shape_seed"])
    return [(rng.randint(4, 16), rng.randint(2, 16), [_log_int(rng, 2, 64) for _ in range(case["per_group"])])
            for _ in range(case["groups"])]


def _inputs(case, seed):
    """The call's inputs as plain tensors, from the seed alone."""
    gen, kind = _gen(seed), case["kind"]
    if kind == "gram":
        a = _tt_cores(gen, case["bA"], case["d"], case["n"], case["r"])
        b = _tt_cores(gen, case["bB"], case["d"], case["n"], case["r"])
        return a, b, torch.randn(case["bA"], case["bB"], generator=gen, device=DEV)
    if kind in ("completion", "riemannian"):
        target = _tt_cores(gen, 1, case["d"], case["n"], 4)
        x = _tt_cores(gen, 1, case["d"], case["n"], case["r"])
        idx = torch.randint(0, case["n"], (case["d"], case["N"]), generator=gen, device=DEV, dtype=torch.int32)
        noise = 0.01 * torch.randn(case["N"], generator=gen, device=DEV)
        return x, idx, _chains(target, idx)[0] + noise
    if kind == "matvec":
        a = _tt_cores(gen, case["batch"], case["d"], case["n"], case["rA"], m=case["m"])
        x = _tt_cores(gen, case["batch"], case["d"], case["n"], case["rx"])
        dc = _tt_cores(gen, case["batch"], case["d"], case["m"], case["rA"] * case["rx"])
        return a, x, dc
    if kind == "uneven":
        objs, couts = [], []
        for d, n, ranks in _group_shapes(case):
            objs += [[c[0] for c in _tt_cores(gen, 1, d, n, r)] for r in ranks]
            couts.append(torch.randn(len(ranks), len(ranks), generator=gen, device=DEV))
        if case["math"] == "bf16":
            objs = [[c.bfloat16() for c in o] for o in objs]
        return objs, couts
    if kind in ("psum", "tangent"):
        x = _tt_cores(gen, 1, case["d"], case["n"], case["rX"])
        u, v = ([torch.from_numpy(c)[None].float().to(DEV) for c in f] for f in _orth_forms(x))
        z = _tt_cores(gen, case["batch"], case["d"], case["n"], case["rZ"])
        c = torch.randn(case["batch"], generator=gen, device=DEV)
        return u, v, z, c, [torch.randn(t.shape, generator=gen, device=DEV) for t in u]
    if kind == "orth":
        return _tt_cores(gen, 1, case["d"], case["n"], case["r"])
    # round: the unrounded products of TT-matrices and TT-vectors
    a = _tt_cores(gen, case["batch"], case["d"], case["n"], case["rA"], m=case["n"])
    x = _tt_cores(gen, case["batch"], case["d"], case["n"], case["rx"])
    return [torch.einsum("paijq,pbjs->pabiqs", s, t).reshape(case["batch"], s.shape[1] * t.shape[1], case["n"], -1)
            for s, t in zip(a, x)]


def _tt(cores, grad=False):
    data = _pack(cores)
    if grad:
        data.requires_grad_(True)
    ranks = [cores[0].shape[1]] + [c.shape[-1] for c in cores]
    m = [c.shape[2] for c in cores] if cores[0].dim() == 5 else None
    return t3f.TT(data, [c.shape[-2] for c in cores], ranks, cores[0].shape[0], m)


def prepare(case, seed):
    kind, inp = case["kind"], _inputs(case, seed)
    s = {"case": case}
    if kind == "gram":
        s.update(A=_tt(inp[0], case["grad"]), B=_tt(inp[1], case["grad"]), dG=inp[2])
    elif kind == "completion":
        s.update(X=_tt(inp[0], True), idx=inp[1], y=inp[2])
    elif kind == "riemannian":
        s.update(X=_tt(inp[0]), idx=inp[1], y=inp[2])
    elif kind == "matvec":
        s.update(A=_tt(inp[0]), x=_tt(inp[1]), dC=_tt(inp[2]))
    elif kind == "uneven":
        objs, couts = inp
        dims = [len(o) for o in objs]
        sizes = [sum(c.numel() for c in o) for o in objs]
        data = torch.cat([c.reshape(-1) for o in objs for c in o])
        X = t3f.RaggedTT(data, dims, [[c.shape[1] for c in o] for o in objs],
                         [[1] + [c.shape[2] for c in o] for o in objs],
                         np.concatenate([[0], np.cumsum(sizes)[:-1]]))
        gstart = [g * case["per_group"] for g in range(case["groups"] + 1)]
        # the work list and workspace a program keeps for a collection of these shapes
        ws = t3f.gram_groups_prepare(X, gstart, backward_math=case["math"])
        s.update(X=X, gstart=gstart, ws=ws, dout=torch.cat([c.reshape(-1) for c in couts]))
    elif kind in ("psum", "tangent"):
        u, v, z, c, dub = inp
        if kind == "psum":
            c.requires_grad_(True)
        s.update(U=_tt(u), V=_tt(v), Z=_tt(z, kind == "psum"), c=c, dUbar=_pack(dub))
    else:
        s.update(X=_tt(inp))
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gram":
        A, B = state["A"], state["B"]
        if not case["grad"]:
            return t3f.gram(A, B)
        G = t3f_ad.gram(A, B)
        dA, dB = torch.autograd.grad(G, [A.data, B.data], state["dG"])
        return [G.detach(), dA, dB]
    if kind == "completion":
        X = state["X"]
        loss = t3f_ad.completion_loss(X, state["idx"], state["y"])
        (dX,) = torch.autograd.grad(loss, [X.data])
        return [loss.detach(), dX]
    if kind == "riemannian":
        U, V = t3f.orthogonalize(state["X"])
        dU, loss = t3f.gather_backward(None, state["idx"], y=state["y"], want_loss=True, riemannian=True, U=U, V=V)
        return [U.data, V.data, dU.data, loss]
    if kind == "matvec":
        A, x = state["A"], state["x"]
        C = t3f.matvec(A, x)
        dA, dx = t3f.matvec_backward(A, x, state["dC"])
        return [C.data, dA.data, dx.data]
    if kind == "uneven":
        X, gs, ws = state["X"], state["gstart"], state["ws"]
        G, norms = t3f.gram_groups(X, gs, ws, math=case["math"])
        dX = t3f.gram_groups_backward(X, gs, ws, state["dout"], math=case["math"])
        return [G, norms, dX]
    if kind == "psum":
        Z, c = state["Z"], state["c"]
        S = t3f_ad.project_sum(state["U"], state["V"], Z, c)
        dZ, dc = torch.autograd.grad(S.data, [Z.data, c], state["dUbar"])
        return [S.data.detach(), dZ, dc]
    if kind == "tangent":
        dU = t3f.project(state["U"], state["V"], state["Z"], state["c"])
        return [dU.data, t3f.tangent_gram(dU, dU)]
    if kind == "orth":
        U, V = t3f.orthogonalize(state["X"])
        return [U.data, V.data]
    return t3f.round_tt(state["X"], case["max_rank"]).data


# ---------------------------------------------------------------------------------------------
# bytes and operations a pass cannot do without (FP32 storage unless the case says otherwise)
# ---------------------------------------------------------------------------------------------

def _numel(d, n, r):
    return sum(a * n * b for a, b in zip(_ranks(d, r)[:-1], _ranks(d, r)[1:]))


def _pair_flops(d, n, ra, rb):
    """One left sweep of a pair: T = M B_i, M' += A_i^T T."""
    A, B = _ranks(d, ra), _ranks(d, rb)
    return sum(2.0 * n * A[k] * B[k + 1] * (B[k] + A[k + 1]) for k in range(d))


def work(case):
    kind = case["kind"]
    if kind == "gram":
        d, n, r = case["d"], case["n"], case["r"]
        pairs, cores = case["bA"] * case["bB"], (case["bA"] + case["bB"]) * _numel(d, n, r)
        f = pairs * _pair_flops(d, n, r, r)
        if not case["grad"]:
            return {"bytes": 4 * (cores + pairs), "flops": f}
        # forward and right sweep share their halves; the gradients take two products a side
        return {"bytes": 4 * (2 * cores + 2 * pairs), "flops": 4 * f}
    if kind in ("completion", "riemannian"):
        d, n, r, N = case["d"], case["n"], case["r"], case["N"]
        chain = sum(2.0 * a * b for a, b in zip(_ranks(d, r)[:-1], _ranks(d, r)[1:]))
        cores = _numel(d, n, r)
        if kind == "completion":
            return {"bytes": 4 * (N * (d + 1) + 2 * cores), "flops": 3 * N * chain}
        orth = work({"kind": "orth", "d": d, "n": n, "r": r})["flops"]
        return {"bytes": 4 * (N * (d + 1) + 4 * cores), "flops": 3 * N * chain + orth}
    if kind == "matvec":
        d, m, n, ra, rx, b = (case[k] for k in ("d", "m", "n", "rA", "rx", "batch"))
        C, A, x = b * _numel(d, m, ra * rx), b * _numel(d, m * n, ra), b * _numel(d, n, rx)
        return {"bytes": 4 * (2 * C + 3 * A + 3 * x), "flops": 3 * 2.0 * n * C}
    if kind == "uneven":
        size = 2 if case["math"] == "bf16" else 4
        flops = elems = pairs = 0.0
        for d, n, ranks in _group_shapes(case):
            for i, ra in enumerate(ranks):
                elems += _numel(d, n, ra)
                flops += sum(_pair_flops(d, n, ra, rb) for rb in ranks[i:])
            pairs += len(ranks) ** 2
        # forward once per unordered pair; the adjoint's two sweeps and its gradients
        return {"bytes": size * 2 * elems + 4 * elems + 8 * pairs, "flops": 4.5 * flops}
    if kind in ("psum", "tangent"):
        d, n, rx, rz, b = (case[k] for k in ("d", "n", "rX", "rZ", "batch"))
        Z, U = b * _numel(d, n, rz), _numel(d, n, rx)
        sweep = b * _pair_flops(d, n, rx, rz)
        if kind == "psum":
            return {"bytes": 4 * (2 * Z + 4 * U + 3 * b), "flops": 8 * sweep}
        return {"bytes": 4 * (Z + 2 * U + b * U + b * b), "flops": 4 * sweep + b * U * b}
    if kind == "orth":
        d, n, r = case["d"], case["n"], case["r"]
        rk = _ranks(d, r)
        # three sweeps of Householder factors, orthogonal factors and products with R
        flops = 3 * sum(5.0 * max(a * n * b * b, b * n * a * a) for a, b in zip(rk[:-1], rk[1:]))
        return {"bytes": 4 * 3 * _numel(d, n, r), "flops": flops}
    d, n, r, b, mr = case["d"], case["n"], case["rA"] * case["rx"], case["batch"], case["max_rank"]
    rk = _ranks(d, r)
    flops = sum(4.0 * n * c * a * min(a, n * c) for a, c in zip(rk[:-1], rk[1:]))
    return {"bytes": 4 * b * (_numel(d, n, r) + _numel(d, n, min(r, mr))), "flops": b * flops}


# ---------------------------------------------------------------------------------------------
# FP64 values
# ---------------------------------------------------------------------------------------------

def _gram64(a, b):
    m = torch.ones(a[0].shape[0], b[0].shape[0], 1, 1, dtype=torch.float64, device=DEV)
    for s, t in zip(a, b):
        w = torch.einsum("pqxy,qyiz->pqixz", m, t)
        m = torch.einsum("pixu,pqixz->pquz", s.transpose(1, 2), w)
    return m[:, :, 0, 0]


def _grad64(y, ins, cot):
    return torch.autograd.grad(y, ins, cot)


def _leaf64(cores):
    return [c.detach().double().clone().requires_grad_(True) for c in cores]


def _tangent64(u, v, z):
    """Per object the unprojected tangent cores: L_{k-1} Z_k R_{k+1}^T, as lists of factors."""
    b = z[0].shape[0]
    one = torch.ones(b, 1, 1, dtype=torch.float64, device=DEV)
    left, right = [one], [one]
    for k in range(len(u) - 1):
        w = torch.einsum("jxp,jpiq->jxiq", left[-1], z[k])
        left.append(torch.einsum("xiy,jxiq->jyq", u[k][0], w))
    for k in range(len(u) - 1, 0, -1):
        w = torch.einsum("jpiq,jyq->jpiy", z[k], right[-1])
        right.append(torch.einsum("xiy,jpiy->jxp", v[k][0], w))
    right.reverse()
    return [(torch.einsum("jxp,jpiq->jxiq", left[k], z[k]), right[k]) for k in range(len(u))]


def _gauge64(uk, zk, last):
    """(I - U U^T) Z on the left unfoldings [batch, r0 n, r1]."""
    if last:
        return zk
    w = uk.reshape(-1, uk.shape[-1])
    q = zk.reshape(zk.shape[0], -1, zk.shape[-1])
    return (q - w @ (w.T @ q)).reshape(zk.shape)


def _exact_uneven(objs, couts, shapes):
    outs, norms, grads, o = [], [], [], 0
    for (d, n, ranks), cot in zip(shapes, couts):
        S = len(ranks)
        # objects of similar rank are padded together (to at most 25 % above the smallest)
        order = sorted(range(S), key=lambda j: ranks[j])
        runs = []
        for j in order:
            if runs and ranks[j] <= 1.25 * ranks[runs[-1][0]]:
                runs[-1].append(j)
            else:
                runs.append([j])
        packs = []
        for run_ in runs:
            rm = max(ranks[j] for j in run_)
            pads = []
            for k in range(d):
                shape = (len(run_), 1 if k == 0 else rm, n, 1 if k == d - 1 else rm)
                t = torch.zeros(shape, dtype=torch.float64, device=DEV)
                for q, j in enumerate(run_):
                    c = objs[o + j][k].double()
                    t[q, :c.shape[0], :, :c.shape[2]] = c
                pads.append(t)
            packs.append(pads)
        G = torch.empty(S, S, dtype=torch.float64, device=DEV)
        gp = [[torch.zeros_like(t) for t in p] for p in packs]
        sym = cot.double()
        for x, rx in enumerate(runs):
            ix = torch.tensor(rx, device=DEV)
            for y in range(x + 1):
                iy = torch.tensor(runs[y], device=DEV)
                a, b = _leaf64(packs[x]), _leaf64(packs[y])
                g = _gram64(a, b)
                G[ix[:, None], iy] = g.detach()
                G[iy[:, None], ix] = g.detach().T
                w = sym[ix[:, None], iy]
                if y != x:
                    w = w + sym[iy[:, None], ix].T
                ga = _grad64(g, a + b, w)
                for k in range(d):
                    gp[x][k] += ga[k]
                    gp[y][k] += ga[d + k]
        slot = {j: (x, q) for x, rx in enumerate(runs) for q, j in enumerate(rx)}
        for j in range(S):
            x, q = slot[j]
            grads += [gp[x][k][q, :c.shape[0], :, :c.shape[2]].reshape(-1) for k, c in enumerate(objs[o + j])]
        outs.append(G.reshape(-1))
        norms.append(torch.sqrt(torch.diagonal(G)))
        o += S
    return [torch.cat(outs), torch.cat(norms), torch.cat(grads)]


def _exact_round(cores, max_rank):
    w = [c.double().cpu().numpy() for c in cores]
    b = w[0].shape[0]
    for k in range(len(w) - 1, 0, -1):
        r0, n, r1 = w[k].shape[1:]
        q, r = np.linalg.qr(w[k].reshape(b, r0, n * r1).transpose(0, 2, 1))
        w[k] = q.transpose(0, 2, 1).reshape(b, -1, n, r1)
        w[k - 1] = np.einsum("paic,pjc->paij", w[k - 1], r, optimize=True)
    for k in range(len(w) - 1):
        r0, n, r1 = w[k].shape[1:]
        u, s, vt = np.linalg.svd(w[k].reshape(b, r0 * n, r1), full_matrices=False)
        keep = min(max_rank, s.shape[1])
        u, sv = u[:, :, :keep], s[:, :keep, None] * vt[:, :keep]
        top = np.take_along_axis(u, np.abs(u).argmax(axis=1)[:, None, :], axis=1)
        sign = np.where(top < 0, -1.0, 1.0)
        w[k] = (u * sign).reshape(b, r0, n, keep)
        nxt = w[k + 1]
        w[k + 1] = ((sv * sign.transpose(0, 2, 1)) @ nxt.reshape(b, nxt.shape[1], -1)).reshape(b, keep, nxt.shape[2], nxt.shape[3])
    return np.concatenate([c.reshape(-1) for c in w])


def exact(case, seed):
    kind, inp = case["kind"], _inputs(case, seed)
    if kind == "gram":
        a, b = _leaf64(inp[0]), _leaf64(inp[1])
        G = _gram64(a, b)
        if not case["grad"]:
            return G.detach()
        g = _grad64(G, a + b, inp[2].double())
        return [G.detach(), _pack(g[:len(a)]), _pack(g[len(a):])]
    if kind == "completion":
        x = _leaf64(inp[0])
        loss = 0.5 * ((_chains(x, inp[1])[0] - inp[2].double()) ** 2).sum()
        return [loss.detach(), _pack(_grad64(loss, x, None))]
    if kind == "riemannian":
        x, idx, y = inp
        u, v = ([torch.from_numpy(c)[None].to(DEV) for c in f] for f in _orth_forms(x))
        val, pre = _chains(u, idx)
        res = val - y.double()
        out, suf = [], torch.ones(len(val), 1, dtype=torch.float64, device=DEV)
        for k in range(len(u) - 1, -1, -1):
            r0, n, r1 = u[k].shape[1:]
            z = torch.zeros(n, r0, r1, dtype=torch.float64, device=DEV)
            for i in range(n):
                sel = idx[k] == i
                z[i] = (pre[k][sel] * res[sel, None]).T @ suf[sel]
            out.append(_gauge64(u[k], z.permute(1, 0, 2)[None].contiguous(), k == len(u) - 1))
            suf = torch.bmm(v[k][0].permute(1, 0, 2)[idx[k].long()], suf[:, :, None])[:, :, 0]
        return [_pack(u), _pack(v), _pack(out[::-1]), 0.5 * (res ** 2).sum().reshape(1)]
    if kind == "matvec":
        a, x = _leaf64(inp[0]), _leaf64(inp[1])
        C = torch.cat([torch.einsum("paijq,pbjs->pabiqs", s, t).reshape(-1) for s, t in zip(a, x)])
        g = _grad64(C, a + x, _pack(inp[2]).double())
        return [C.detach(), _pack(g[:len(a)]), _pack(g[len(a):])]
    if kind == "uneven":
        return _exact_uneven(inp[0], inp[1], _group_shapes(case))
    if kind in ("psum", "tangent"):
        u, v = [c.double() for c in inp[0]], [c.double() for c in inp[1]]
        d = len(u)
        if kind == "psum":
            z, c = _leaf64(inp[2]), inp[3].double().requires_grad_(True)
            hat = [torch.einsum("jxiq,jyq->xiy", w * c[:, None, None, None], r)[None] for w, r in _tangent64(u, v, z)]
            S = _pack([_gauge64(u[k], hat[k], k == d - 1) for k in range(d)])
            g = _grad64(S, z + [c], _pack(inp[4]).double())
            return [S.detach(), _pack(g[:d]), g[d]]
        c = inp[3].double()
        hat = [torch.einsum("jxiq,jyq->jxiy", w * c[:, None, None, None], r)
               for w, r in _tangent64(u, v, [t.double() for t in inp[2]])]
        dU = [_gauge64(u[k], hat[k], k == d - 1) for k in range(d)]
        flat = [t.reshape(t.shape[0], -1) for t in dU]
        return [_pack(dU), sum(f @ f.T for f in flat)]
    if kind == "orth":
        return [torch.from_numpy(np.concatenate([c.reshape(-1) for c in f])) for f in _orth_forms(inp)]
    return torch.from_numpy(_exact_round(inp, case["max_rank"]))
