"""Performance cases of the codec: the work a program has it do, through api.py.

A case names one call ("op") and its sizes.  The sizes span what the codec is used
at: from a tiny scene of 10,000 Gaussians with 256 atoms to scenes of millions with
512 to 2048 atoms, 4 to 16 nonzeros per Gaussian, at every precision and storage
format that the calls offer.  Inputs are drawn on the GPU from the seed with the
distributions of the synthetic workload (synth.py); exact() restates each call in
plain 64-bit torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_30396_gb300 import api, synth

DEV = "cuda"
D_SH = 45
CODE_NOISE = 0.02  # a learned dictionary's distance from the one that made the signals


def listed():
    return [
        # The smallest scene: one wave of tiles, launches and latency count.
        {"name": "encode_tiny", "op": "encode", "N": 10_000, "K": 256, "s": 8, "prec": "fp32", "eps": 0.0},
        # A whole scene at the usual sparsity, the codec's main call.
        {"name": "encode_scene", "op": "encode", "N": 3_000_000, "K": 1024, "s": 8, "prec": "fp32", "eps": 0.0},
        # A large dictionary and long codes that stop at an error tolerance; a ragged last tile.
        {"name": "encode_s16_eps", "op": "encode", "N": 400_009, "K": 2048, "s": 16, "prec": "fp32", "eps": 0.2},
        # Low-precision correlations with FP32 re-scoring.
        {"name": "encode_bf16", "op": "encode", "N": 1_000_000, "K": 1024, "s": 8, "prec": "bf16", "eps": 0.0},
        # Dictionary update of the learning loop: a whole scene, and the smallest one.
        {"name": "mod_scene", "op": "mod", "N": 3_000_000, "K": 1024, "s": 8, "ragged": False},
        {"name": "mod_tiny", "op": "mod", "N": 10_000, "K": 256, "s": 8, "ragged": False},
        # The other dictionary update, on codes of uneven length.
        {"name": "ksvd_mid", "op": "ksvd", "N": 400_003, "K": 512, "s": 8, "ragged": True},
        # Colours of a whole scene from one camera; and of a scene whose dictionary outgrows shared memory,
        # along given directions with the DC term.
        {"name": "decode_scene", "op": "decode", "N": 3_000_000, "K": 1024, "s": 8, "store": "fp32", "view": "camera",
         "dc": False, "ragged": False},
        {"name": "decode_k2048", "op": "decode", "N": 777_777, "K": 2048, "s": 16, "store": "fp32", "view": "dirs",
         "dc": True, "ragged": True},
        # The renderer's preprocess with the colours from compact codes.
        {"name": "preprocess_compact", "op": "preprocess", "N": 2_000_003, "K": 1024, "s": 8, "store": "compact",
         "inside": False, "ragged": True},
        # Forward and backward of the support-proposal network on a training batch.
        {"name": "mlp_gradients", "op": "gradients", "N": 8_192, "K": 1024, "s": 8},
        # Its inference: 16 candidate atoms for every signal.
        {"name": "propose", "op": "propose", "N": 500_001, "K": 1024, "m": 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# Largest N * K * s of the encoder's and N * s of the other calls' drawn cases.
ENCODE_MOST = 3_000_000 * 1024 * 8
CODES_MOST = 3_000_000 * 8


def draw(rng):
    op = rng.choice(["encode", "encode", "mod", "ksvd", "decode", "decode", "preprocess", "gradients", "propose"])
    K = rng.choice([256, 512, 1024, 2048, _log_int(rng, 64, 2048)])
    s = rng.choice([4, 8, 16, rng.randint(1, 16)])
    ragged = rng.random() < 0.5
    if op == "encode":
        prec = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp8"])
        # the codes of more than 8 atoms and the low precisions cost more per signal
        most = ENCODE_MOST // (1 if s <= 8 and prec == "fp32" else 4)
        N = _log_int(rng, 1_000, max(2_000, min(3_000_000, most // (K * s))))
        return {"op": op, "N": N, "K": K, "s": s, "prec": prec, "eps": rng.choice([0.0, 0.0, 0.2])}
    if op == "mod":
        return {"op": op, "N": _log_int(rng, 5_000, min(3_000_000, CODES_MOST // s)), "K": K, "s": s,
                "ragged": ragged}
    if op == "ksvd":
        return {"op": op, "N": _log_int(rng, 5_000, min(1_000_000, CODES_MOST // (2 * s))), "K": min(K, 512), "s": s,
                "ragged": ragged}
    if op in ("decode", "preprocess"):
        N = _log_int(rng, 10_000, min(3_000_000, CODES_MOST // s))
        if op == "decode":
            store = rng.choice(["fp32", "fp32", "compact"])
            return {"op": op, "N": N, "K": min(K, 1200) if store == "compact" else K, "s": s, "store": store,
                    "view": rng.choice(["camera", "dirs"]), "dc": rng.random() < 0.5, "ragged": ragged}
        store = rng.choice(["sh", "fp32", "compact"])
        return {"op": op, "N": N, "K": min(K, 900), "s": s, "store": store, "inside": rng.random() < 0.3, "ragged": ragged}
    if op == "gradients":
        return {"op": op, "N": _log_int(rng, 512, 16_384), "K": K, "s": min(s, 8)}
    return {"op": op, "N": _log_int(rng, 10_000, 500_000), "K": max(K, 128), "m": rng.choice([8, 16, 32])}


# ---- inputs ---------------------------------------------------------------------------

def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 16 + salt)
    return g


def _atoms(case, seed):
    """The atoms behind the signals, and the learned dictionary (unit rows near them), FP32."""
    A = synth.hidden_dictionary(case["K"], int(seed) % (1 << 31), rho=0.6)
    r = np.random.default_rng(int(seed) + 1).standard_normal(A.shape)
    D = A + CODE_NOISE * r
    D /= np.linalg.norm(D, axis=1, keepdims=True)
    return A, torch.from_numpy(D.astype(np.float32)).to(DEV)


def _codes(case, seed):
    """ELL codes: distinct uniform atoms, Laplace coefficients, nnz = s or uneven; slots past nnz are zero."""
    N, K, s = case["N"], case["K"], case["s"]
    g = _gen(seed, 1)
    idx = torch.randint(0, K, (N, s), generator=g, device=DEV)
    while True:
        srt = torch.sort(idx, dim=1)[0]
        bad = (srt[:, 1:] == srt[:, :-1]).any(dim=1).nonzero().flatten()
        if bad.numel() == 0:
            break
        idx[bad] = torch.randint(0, K, (bad.numel(), s), generator=g, device=DEV)
    u = (torch.rand((N, s), generator=g, device=DEV) - 0.5).clamp(-0.4999999, 0.4999999)
    coef = -torch.sign(u) * torch.log1p(-2.0 * u.abs())
    nnz = torch.full((N,), s, dtype=torch.uint8, device=DEV)
    if case.get("ragged"):
        nnz = torch.randint(0, s + 1, (N,), generator=g, device=DEV).to(torch.uint8)
        pad = torch.arange(s, device=DEV)[None, :] >= nnz[:, None]
        idx[pad] = 0
        coef[pad] = 0.0
    return idx, coef, nnz


def _dense(D, idx, coef, step=1 << 18):
    """sum_t coef[:, t] D[idx[:, t]], in D's type."""
    out = torch.empty((idx.shape[0], D.shape[1]), dtype=D.dtype, device=DEV)
    for lo in range(0, idx.shape[0], step):
        i, c = idx[lo:lo + step], coef[lo:lo + step].to(D.dtype)
        out[lo:lo + step] = torch.einsum("ns,nsd->nd", c, D[i])
    return out


def _signals(case, seed):
    A, D = _atoms(case, seed)
    s = min(case.get("s", 8), case["K"])
    return D, synth.signals_device(case["N"], A, s, int(seed) + 2)


def _mlp_params(case, seed):
    return synth.mlp_params(case["K"], int(seed) % (1 << 31))


def _splat(case, seed):
    """Means, scales, rotations and DC colours of a scene's Gaussians."""
    g, N = _gen(seed, 3), case["N"]
    rand = lambda *n: torch.randn(n, generator=g, device=DEV)  # noqa: E731
    means = 2.0 * torch.rand((N, 3), generator=g, device=DEV) - 1.0
    return means, torch.exp(math.log(0.01) + 0.5 * rand(N, 3)), rand(N, 4), rand(N, 3)


IMAGE = (1920, 1080)
FOCAL = 1100.0
Z_NEAR = 0.2


def _pose(case):
    if case["inside"]:
        return synth.look_at((0.15, -0.1, 0.05), (1.0, 0.4, -0.3))
    return synth.look_at((0.4, -3.2, 1.1))


def _store(case, idx, coef):
    """The codes as a program keeps them: int16 bits and FP32, or the compact form."""
    if case["store"] == "compact":
        return idx.to(torch.uint8 if case["K"] <= 256 else torch.int16), coef.to(torch.float16)
    return idx.to(torch.int16), coef


def prepare(case, seed):
    op = case["op"]
    st = {"case": case}
    if op == "encode":
        st["D"], st["X"] = _signals(case, seed)
    elif op in ("mod", "ksvd"):
        A, st["D"] = _atoms(case, seed)
        idx, coef, st["nnz"] = _codes(case, seed)
        X = _dense(torch.from_numpy(A.astype(np.float32)).to(DEV), idx, coef)
        X += 1e-3 * torch.randn(X.shape, generator=_gen(seed, 2), device=DEV)
        st["resid"] = (X - _dense(st["D"], idx, coef)).square().sum(dim=1)
        st["X"], st["idx"], st["coef"] = X, idx.to(torch.int16), coef
    elif op == "decode":
        _, st["D"] = _atoms(case, seed)
        idx, coef, st["nnz"] = _codes(case, seed)
        st["idx"], st["coef"] = _store(case, idx, coef)
        st["view"] = _view(case, seed)
        st["dc"] = torch.randn((case["N"], 3), generator=_gen(seed, 5), device=DEV) if case["dc"] else None
    elif op == "preprocess":
        st["g"] = _splat(case, seed)
        R, t = _pose(case)
        st["cam"] = api.camera(R, t, FOCAL, FOCAL, IMAGE[0], IMAGE[1], Z_NEAR)
        if case["store"] == "sh":
            st["colour"] = {"sh": 0.2 * torch.randn((case["N"], D_SH), generator=_gen(seed, 4), device=DEV)}
        else:
            _, D = _atoms(case, seed)
            idx, coef, nnz = _codes(case, seed)
            idx, coef = _store(case, idx, coef)
            st["colour"] = {"D": D, "idx": idx, "coef": coef, "nnz": nnz}
    else:
        _, st["X"] = _signals(case, seed)
        st["mlp"] = api.MLP(case["K"], _mlp_params(case, seed))
        if op == "gradients":
            idx, _, st["nnz"] = _codes(case, seed)
            st["idx"] = idx.to(torch.int16)
    return st


def _view(case, seed):
    g = _gen(seed, 4)
    if case["view"] == "dirs":
        v = torch.randn((case["N"], 3), generator=g, device=DEV)
        return {"dirs": v / v.norm(dim=1, keepdim=True)}
    cam = 4.0 * synth.unit_directions(1, int(seed) % (1 << 31))[0]
    return {"means": 2.0 * torch.rand((case["N"], 3), generator=g, device=DEV) - 1.0, "cam": cam}


# ---- the calls ------------------------------------------------------------------------

def run(st):
    case = st["case"]
    op = case["op"]
    if op == "encode":
        return api.encode(st["D"], st["X"], case["s"], eps=case["eps"], precision=case["prec"])
    if op == "mod":
        return api.mod_update(st["X"], st["D"], st["idx"], st["coef"], st["nnz"], st["resid"])
    if op == "ksvd":  # the sweep refits the coefficients in place; the next pass goes on from both
        st["D"] = api.ksvd_update(st["X"], st["D"], st["idx"], st["coef"], st["nnz"], st["resid"])
        return st["D"], st["coef"]
    if op == "decode":
        f = api.decode_compact if case["store"] == "compact" else api.decode
        return f(st["D"], st["idx"], st["coef"], st["nnz"], dc=st["dc"], **st["view"])
    if op == "preprocess":
        return api.preprocess(st["cam"], *st["g"], **st["colour"])
    if op == "gradients":
        return st["mlp"].gradients(st["X"], st["idx"], st["nnz"])
    return st["mlp"].propose(st["X"], case["m"])


def work(case):
    """Each input read once, each output written once; the operations of the method itself."""
    op, N, K = case["op"], case["N"], case["K"]
    s = case.get("s", 0)
    signal, atoms = 4 * D_SH * N, 4 * D_SH * K
    if op == "encode":  # correlations with every atom per selected atom
        return {"bytes": signal + atoms + N * (6 * s + 5), "flops": 2.0 * D_SH * K * s * N}
    if op == "mod":  # Gram matrix and right-hand side from the codes, factorisation, two triangular solves
        return {"bytes": signal + 2 * atoms + N * (6 * s + 5), "flops": 2.0 * N * s * (s + D_SH) + K ** 3 / 3 + 2.0 * D_SH * K * K}
    if op == "ksvd":  # residual, one power step and the residual's update per entry
        return {"bytes": signal + 2 * atoms + N * (10 * s + 5), "flops": 2.0 * D_SH * N * s * 4}
    if op in ("decode", "preprocess"):
        code = 4 * D_SH if case["store"] == "sh" else s * (6 if case["store"] == "fp32" else 3 if K <= 256 else 4) + 1
        fixed = 24 + (12 if case.get("dc") else 0) if op == "decode" else 52 + 40
        return {"bytes": N * (code + fixed) + (0 if case["store"] == "sh" else atoms), "flops": 2.0 * D_SH * N * (s + 1)}
    layers = D_SH * 256 + 256 * 256 + 256 * K
    params = 4 * (layers + 512 + K)
    if op == "gradients":
        return {"bytes": signal + N * (2 * s + 1) + 2 * params, "flops": 2.0 * N * (3 * layers - D_SH * 256)}
    return {"bytes": signal + params / 2 + 2 * N * case["m"], "flops": 2.0 * N * layers}


# ---- the same in 64 bits ----------------------------------------------------------------

def exact(case, seed):
    op = case["op"]
    if op == "propose":  # atom indices only
        return None
    st = prepare(case, seed)
    if op == "encode":
        coef, resid = _exact_omp(st["D"].double(), st["X"], case["s"], case["eps"])
        return None, coef, None, resid
    if op == "mod":
        return _exact_mod(st)
    if op == "ksvd":
        return _exact_ksvd(st)
    if op == "decode":
        return _exact_decode(case, st)
    if op == "preprocess":
        return _exact_preprocess(case, st)
    return _exact_gradients(case, seed, st)


def _exact_omp(D, X, s, eps, step=1 << 16):
    N, K = X.shape[0], D.shape[0]
    G = D @ D.T
    coef = torch.zeros((N, s), dtype=torch.float64, device=DEV)
    resid = torch.empty((N,), dtype=torch.float64, device=DEV)
    for lo in range(0, N, step):
        x = X[lo:lo + step].double()
        n = x.shape[0]
        rows = torch.arange(n, device=DEV)
        xn = x.norm(dim=1)
        b = x @ D.T
        sel = torch.zeros((n, s), dtype=torch.int64, device=DEV)
        L = torch.zeros((n, s, s), dtype=torch.float64, device=DEV)
        y = torch.zeros((n, s), dtype=torch.float64, device=DEV)
        gam = torch.zeros((n, s), dtype=torch.float64, device=DEV)
        r, live = x.clone(), torch.ones(n, dtype=torch.bool, device=DEV)
        for t in range(s):
            live = live & (r.norm(dim=1) > eps)
            c = (r @ D.T).abs_()
            c.scatter_(1, sel[:, :t], -1.0)
            best, j = c.max(dim=1)
            live = live & (best > 1e-7 * xn)
            w = torch.zeros((n, t), dtype=torch.float64, device=DEV)
            for m in range(t):
                w[:, m] = (G[j, sel[:, m]] - (L[:, m, :m] * w[:, :m]).sum(dim=1)) / L[:, m, m]
            ell2 = G[j, j] - w.square().sum(dim=1)
            live = live & (ell2 > 1e-6 * G[j, j])
            ell = ell2.clamp_min(1e-300).sqrt()
            L[:, t, :t], L[:, t, t], sel[:, t] = w, ell, j
            y[:, t] = (b[rows, j] - (w * y[:, :t]).sum(dim=1)) / ell
            g = torch.zeros((n, t + 1), dtype=torch.float64, device=DEV)
            for m in range(t, -1, -1):
                g[:, m] = (y[:, m] - (L[:, m + 1:t + 1, m] * g[:, m + 1:]).sum(dim=1)) / L[:, m, m]
            new = x - torch.einsum("nt,ntd->nd", g, D[sel[:, :t + 1]])
            gam[:, :t + 1] = torch.where(live[:, None], g, gam[:, :t + 1])
            r = torch.where(live[:, None], new, r)
            if not bool(live.any()):
                break
        coef[lo:lo + step] = gam
        resid[lo:lo + step] = r.square().sum(dim=1)
    return coef, resid


def _live(st):
    idx = st["idx"].to(torch.int64)
    return idx, torch.arange(idx.shape[1], device=DEV)[None, :] < st["nnz"][:, None]


def _exact_mod(st):
    D, X = st["D"].double(), st["X"]
    K = D.shape[0]
    idx, live = _live(st)
    a = st["coef"].double() * live
    G = torch.zeros(K * K, dtype=torch.float64, device=DEV)
    B = torch.zeros((K, D_SH), dtype=torch.float64, device=DEV)
    for t in range(idx.shape[1]):
        for u in range(idx.shape[1]):
            G.index_add_(0, idx[:, t] * K + idx[:, u], a[:, t] * a[:, u])
        for lo in range(0, X.shape[0], 1 << 19):
            B.index_add_(0, idx[lo:lo + (1 << 19), t], a[lo:lo + (1 << 19), t, None] * X[lo:lo + (1 << 19)].double())
    G = G.view(K, K)
    tr = float(G.diagonal().sum())
    lam = 1e-6 * tr / K if tr > 0 else 1e-6
    Z = torch.linalg.solve(G + lam * torch.eye(K, dtype=torch.float64, device=DEV), B + lam * D)
    out = Z / Z.norm(dim=1, keepdim=True)
    used = torch.zeros(K, dtype=torch.bool, device=DEV)
    used[idx[live]] = True
    return out if bool(used.all()) else _refilled(st, out, used)


def _refilled(st, D, used):
    """Unused atoms, in order, from the signals of largest residual."""
    D = D.clone()
    dead = (~used).nonzero().flatten()
    order = torch.sort(st["resid"], descending=True, stable=True)[1]
    order = order[st["X"].norm(dim=1)[order] > 0][:dead.numel()]
    x = st["X"][order].double()
    D[dead[:order.numel()]] = x / x.norm(dim=1, keepdim=True)
    return D


def _exact_ksvd(st):
    D = st["D"].double()
    K = D.shape[0]
    idx, live = _live(st)
    s = idx.shape[1]
    A = st["coef"].double()
    R = st["X"].double() - _dense(D, idx, A * live)
    # entries grouped by atom, in signal order
    key = torch.where(live, idx, torch.full_like(idx, K)).flatten()
    srt, order = torch.sort(key, stable=True)
    start = torch.searchsorted(srt, torch.arange(K + 1, device=DEV)).tolist()
    A = A.flatten()
    for j in range(K):
        e = order[start[j]:start[j + 1]]
        if e.numel() == 0:
            continue
        i, g = e // s, A[e]
        E = R[i] + g[:, None] * D[j]
        d = E.T @ g
        d = d / d.norm()
        new = E @ d
        R[i] = E - new[:, None] * d
        D[j], A[e] = d, new
    used = torch.zeros(K, dtype=torch.bool, device=DEV)
    used[idx[live]] = True
    return (D if bool(used.all()) else _refilled(st, D, used)), A.view(-1, s)


def _sh(v):
    """Real spherical harmonics of degree 1..3 (Condon-Shortley phase), basis l*l + l + m - 1."""
    x, y, z = v.unbind(dim=1)
    p = math.pi
    c1 = math.sqrt(3 / (4 * p))
    a2, b2, c2 = math.sqrt(15 / (4 * p)), math.sqrt(5 / (16 * p)), math.sqrt(15 / (16 * p))
    a3, b3, c3 = math.sqrt(35 / (32 * p)), math.sqrt(105 / (4 * p)), math.sqrt(21 / (32 * p))
    d3, e3 = math.sqrt(7 / (16 * p)), math.sqrt(105 / (16 * p))
    return torch.stack([
        -c1 * y, c1 * z, -c1 * x,
        a2 * x * y, -a2 * y * z, b2 * (3 * z * z - 1), -a2 * x * z, c2 * (x * x - y * y),
        -a3 * y * (3 * x * x - y * y), b3 * x * y * z, -c3 * y * (5 * z * z - 1), d3 * z * (5 * z * z - 3),
        -c3 * x * (5 * z * z - 1), e3 * z * (x * x - y * y), -a3 * x * (x * x - 3 * y * y)], dim=1)


def _colour(Y, v):
    return torch.einsum("nb,ncb->nc", _sh(v), Y.view(-1, 3, 15))


def _code_sh(case, D, idx, coef, nnz):
    """Dense 45 coefficients from stored codes; the compact form rounds D and the coefficients to FP16."""
    if case["store"] == "compact":
        D = D.half()
    idx = idx.to(torch.int64)
    live = torch.arange(idx.shape[1], device=DEV)[None, :] < nnz[:, None]
    return _dense(D.double(), idx, coef.double() * live)


Y00 = 0.5 / math.sqrt(math.pi)


def _exact_decode(case, st):
    if "dirs" in st["view"]:
        v = st["view"]["dirs"].double()
    else:
        v = st["view"]["means"].double() - torch.from_numpy(st["view"]["cam"]).to(DEV).double()
        v = v / v.norm(dim=1, keepdim=True)
    rgb = _colour(_code_sh(case, st["D"], st["idx"], st["coef"], st["nnz"]), v)
    return rgb if st["dc"] is None else (Y00 * st["dc"].double() + rgb + 0.5).clamp_min(0.0)


def _exact_preprocess(case, st):
    mu, scale, q, dc = (t.double() for t in st["g"])
    # the pose as the camera holds it, in FP32
    R, t = (torch.from_numpy(np.asarray(a, dtype=np.float32)).to(DEV).double() for a in _pose(case))
    W, H = IMAGE
    pc = mu @ R.T + t
    z = pc[:, 2]
    zn = float(np.float32(Z_NEAR))
    zs = torch.where(z > zn, z, torch.ones_like(z))
    ux, uy = pc[:, 0] / zs, pc[:, 1] / zs
    cx, cy = ux.clamp(-0.65 * W / FOCAL, 0.65 * W / FOCAL), uy.clamp(-0.65 * H / FOCAL, 0.65 * H / FOCAL)
    zero = torch.zeros_like(z)
    J = torch.stack([FOCAL / zs, zero, -FOCAL * cx / zs, zero, FOCAL / zs, -FOCAL * cy / zs], dim=1).view(-1, 2, 3)
    w, x, y, k = (q / q.norm(dim=1, keepdim=True)).unbind(dim=1)
    rot = torch.stack([1 - 2 * (y * y + k * k), 2 * (x * y - w * k), 2 * (x * k + w * y),
                       2 * (x * y + w * k), 1 - 2 * (x * x + k * k), 2 * (y * k - w * x),
                       2 * (x * k - w * y), 2 * (y * k + w * x), 1 - 2 * (x * x + y * y)], dim=1).view(-1, 3, 3)
    M = torch.einsum("nij,jk,nkl,nl->nil", J, R, rot, scale)
    S = torch.einsum("nij,nkj->nik", M, M)
    a, b, c = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det = a * c - b * b
    mid = 0.5 * (a + c)
    radius = torch.ceil(3.0 * (mid + (mid * mid - det).clamp_min(0.1).sqrt()).sqrt())
    px, py = FOCAL * ux + 0.5 * W, FOCAL * uy + 0.5 * H
    vis = (z > zn) & (det > 0) & (px + radius > 0) & (px - radius < W) & (py + radius > 0) & (py - radius < H)
    v = mu + t @ R  # mu - C with C = -R^T t
    v = v / v.norm(dim=1, keepdim=True)
    col = st["colour"]
    Y = col["sh"].double() if "sh" in col else _code_sh(case, col["D"], col["idx"], col["coef"], col["nnz"])
    rgb = (Y00 * dc + _colour(Y, v) + 0.5).clamp_min(0.0)
    seen = lambda u: torch.where(vis.view(-1, *[1] * (u.dim() - 1)), u, torch.zeros_like(u))  # noqa: E731
    return {"xy": seen(torch.stack([px, py], dim=1)), "depth": seen(z), "radius": None, "rgb": seen(rgb),
            "conic": seen(torch.stack([c / det, -b / det, a / det], dim=1))}


def _exact_gradients(case, seed, st):
    """Gradients of the mean BCE loss by 64-bit autograd, on weights in BF16 as every GEMM reads them."""
    K, N = case["K"], case["N"]
    p = {k: torch.from_numpy(np.asarray(v, dtype=np.float32)).to(DEV) for k, v in _mlp_params(case, seed).items()}
    p = {k: (v.bfloat16() if k.startswith("W") else v).double().requires_grad_() for k, v in p.items()}
    x = st["X"].double()
    h = x / x.norm(dim=1, keepdim=True)
    gelu = lambda u: 0.5 * u * (1.0 + torch.erf(u / math.sqrt(2.0)))  # noqa: E731
    h = gelu(h @ p["W1"].T + p["b1"])
    h = gelu(h @ p["W2"].T + p["b2"])
    zl = h @ p["W3"].T + p["b3"]
    idx, live = _live(st)
    target = torch.zeros((N, K + 1), dtype=torch.float64, device=DEV)
    target.scatter_(1, torch.where(live, idx, torch.full_like(idx, K)), 1.0)
    loss = torch.nn.functional.binary_cross_entropy_with_logits(zl, target[:, :K])
    loss.backward()
    w1 = torch.nn.functional.pad(p["W1"].grad, (0, api.X_IN - D_SH))
    parts = [w1] + [p[k].grad for k in ("b1", "W2", "b2", "W3", "b3")]
    return torch.cat([g.reshape(-1) for g in parts]), float(loss)
