"""Step a5: the MOD dictionary update on the GPU vs the FP64 oracle, same codes."""
import numpy as np
import pytest
import torch

from oracle import mod as omod, omp as oomp
from paper_2605_30396_gb300 import synth

pytestmark = pytest.mark.gpu


def _inputs(N, K, s, seed=0):
    Dh = synth.hidden_dictionary(K, seed + 1)
    X = synth.signals(N, Dh, s, seed + 2)
    D0 = synth.hidden_dictionary(K, seed + 3).astype(np.float32)
    ref = oomp.omp(D0.astype(np.float64), X.astype(np.float64), s)
    idx = ref["idx"].astype(np.uint16)
    coef = ref["coef"].astype(np.float32)
    nnz = ref["nnz"].astype(np.uint8)
    resid = ref["resid_sq"].astype(np.float32)
    return X, D0, idx, coef, nnz, resid


def _gpu(lib, X, D0, idx, coef, nnz, resid):
    c = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return lib.mod_update(c(X), c(D0), c(idx.view(np.int16)), c(coef), c(nnz),
                          c(resid) if resid is not None else None, sync=True).cpu().numpy()


@pytest.mark.parametrize("N,K,s", [(5000, 128, 6), (3000, 256, 8), (20000, 1024, 8), (700, 64, 16),
                                   (4000, 300, 4), (30000, 2048, 8), (1000, 20, 4), (12000, 4096, 8)])
def test_mod_matches_oracle(lib, N, K, s):
    X, D0, idx, coef, nnz, resid = _inputs(N, K, s)
    got = _gpu(lib, X, D0, idx, coef, nnz, resid)
    ref, info = omod.mod_update(X.astype(np.float64), D0.astype(np.float64), idx.astype(np.int64),
                                coef.astype(np.float64), nnz, resid.astype(np.float64))
    np.testing.assert_allclose(got, ref, atol=3e-6, rtol=0)


def test_mod_on_nearly_dependent_atoms(lib):
    """K = 1024 with the atoms in pairs that are always used together, with coefficients
    1 % apart (the scaled Gram matrix has a condition of 6e4): the refined solution is
    FP64's rounded to FP32, below 2^-24 in the norm."""
    N, K, s = 60_000, 1024, 8
    rng = np.random.default_rng(21)
    h = synth.distinct_supports(rng, N, K // 2, s // 2)
    idx = np.stack([2 * h, 2 * h + 1], axis=2).reshape(N, s)
    c = rng.laplace(0, 1, h.shape)
    coef = np.stack([c, c * (1 + 1e-2 * rng.standard_normal(c.shape))], axis=2).reshape(N, s).astype(np.float32)
    X = synth.signals(N, synth.hidden_dictionary(K, 22), 4, 23)
    D0 = synth.hidden_dictionary(K, 24).astype(np.float32)
    nnz = np.full(N, s, dtype=np.uint8)
    got = _gpu(lib, X, D0, idx.astype(np.uint16), coef, nnz, None)
    ref, _ = omod.mod_update(X.astype(np.float64), D0.astype(np.float64), idx, coef.astype(np.float64), nnz)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 2.0**-24


@pytest.mark.parametrize("N,K,s,skip", [(513, 40, 1, 0), (9000, 1500, 8, 0), (65537, 128, 17, 0), (33000, 96, 32, 2),
                                        (330_000, 300, 3, 2), (311_297, 64, 8, 0)])
def test_mod_on_random_codes(lib, N, K, s, skip):
    """Uneven code lengths and codes that name an atom twice, at the edges of the
    sort's tiles (512 and, from 311,296 signals on, 1024 signals), chunks and
    segments; skip > 0 hands in arrays that start off 16-byte alignment.  Atoms
    within 3e-6 as above (FP32 output of an FP64-accurate solve)."""
    D = synth.hidden_dictionary(K, 11)
    idx, coef, nnz = synth.random_codes(N + skip, K, s, 12)
    X = np.einsum("ns,nsd->nd", coef.astype(np.float64), D[idx]) if N < 100_000 else sum(
        coef[:, t, None].astype(np.float64) * D[idx[:, t]] for t in range(s))
    X = (X + 0.05 * np.random.default_rng(13).standard_normal(X.shape)).astype(np.float32)
    D0 = synth.hidden_dictionary(K, 14).astype(np.float32)
    c = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()[skip:]  # noqa: E731
    got = lib.mod_update(c(X), torch.from_numpy(D0).cuda(), c(idx.view(np.int16)), c(coef), c(nnz),
                         sync=True).cpu().numpy()
    ref, info = omod.mod_update(X[skip:].astype(np.float64), D0.astype(np.float64), idx[skip:].astype(np.int64),
                                coef[skip:].astype(np.float64), nnz[skip:], np.zeros(N))
    np.testing.assert_allclose(got, ref, atol=3e-6, rtol=0)


def test_dead_atoms_refilled_in_order(lib):
    N, K, s = 4000, 64, 4
    X, D0, idx, coef, nnz, resid = _inputs(N, K, s, seed=5)
    # make atoms 7, 20 and 63 unused by zeroing their coefficients out of the codes
    for j in (7, 20, 63):
        m = idx == j
        idx[m] = 0
        coef[m] = 0.0
    keep = np.zeros_like(idx, dtype=bool)
    for i in range(N):
        sel = [t for t in range(nnz[i]) if not (idx[i, t] == 0 and coef[i, t] == 0.0)]
        row_i, row_c = idx[i, sel], coef[i, sel]
        idx[i] = 0
        coef[i] = 0.0
        idx[i, :len(sel)] = row_i
        coef[i, :len(sel)] = row_c
        nnz[i] = len(sel)
    del keep
    resid = resid + np.arange(N, dtype=np.float32) * 1e-7  # distinct residual keys
    got = _gpu(lib, X, D0, idx, coef, nnz, resid)
    ref, info = omod.mod_update(X.astype(np.float64), D0.astype(np.float64), idx.astype(np.int64),
                                coef.astype(np.float64), nnz, resid.astype(np.float64))
    assert set(info["dead"].tolist()) >= {7, 20, 63}
    np.testing.assert_allclose(got, ref, atol=3e-6, rtol=0)


def test_mod_deterministic(lib):
    X, D0, idx, coef, nnz, resid = _inputs(30000, 512, 8, seed=9)
    a = _gpu(lib, X, D0, idx, coef, nnz, resid)
    b = _gpu(lib, X, D0, idx, coef, nnz, resid)
    np.testing.assert_array_equal(a, b)


def test_learn_loop_matches_oracle_trajectory(lib):
    """Config 1: N=10,000, K=256 learned with s=8 for 10 alternating iterations.
    The first coding pass must match to 1e-4; later passes are chaotic in the
    support flips that near-ties allow, so the trajectory is compared loosely."""
    N, K, s, iters = 10000, 256, 8, 10
    Dh = synth.hidden_dictionary(K, 0)
    X = synth.signals(N, Dh, s, 0)
    init = synth.init_atom_indices(N, K, 0)
    D, idx, coef, nnz, rmse = lib.learn_dictionary(torch.from_numpy(X).cuda(), K, s, iters, init,
                                                   sync=True)
    rmse = rmse.cpu().numpy().astype(np.float64)
    Dref, codes, hist = omod.learn(X.astype(np.float64), K, s, iters, init)
    hist = np.array(hist)
    assert abs(rmse[0] - hist[0]) <= 1e-4 * hist[0], (rmse[0], hist[0])
    assert np.all(np.abs(rmse - hist) <= 0.05 * hist), (rmse, hist)
    assert rmse[-1] < rmse[0]
    Dg = D.cpu().numpy().astype(np.float64)
    np.testing.assert_allclose(np.linalg.norm(Dg, axis=1), 1.0, atol=1e-5)
    rec_g = np.mean(np.abs(Dg @ Dh.T).max(axis=1) > 0.99)
    rec_o = np.mean(np.abs(Dref @ Dh.T).max(axis=1) > 0.99)
    assert abs(rec_g - rec_o) <= 0.1, (rec_g, rec_o)


def test_csc_export(lib):
    rng = np.random.default_rng(0)
    N, s, K = 10007, 8, 300
    idx = synth.distinct_supports(rng, N, K, s).astype(np.uint16)
    coef = rng.standard_normal((N, s)).astype(np.float32)
    nnz = rng.integers(0, s + 1, N).astype(np.uint8)
    c = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    cp, ri, va = lib.csc_from_ell(c(idx.view(np.int16)), c(coef), c(nnz), sync=True)
    cp = cp.cpu().numpy()
    ri = ri.cpu().numpy().view(np.uint16)
    va = va.cpu().numpy()
    np.testing.assert_array_equal(cp, np.concatenate([[0], np.cumsum(nnz)]))
    for i in range(0, N, 97):
        np.testing.assert_array_equal(ri[cp[i]:cp[i + 1]], idx[i, :nnz[i]])
        np.testing.assert_array_equal(va[cp[i]:cp[i + 1]], coef[i, :nnz[i]])


def test_mod_under_graph_capture(lib):
    """The whole update (counting sort, accumulation, the cooperative
    factorisation, the refinement) is enqueued without host synchronisation, so
    it can be captured once and replayed; the replay matches the eager call bit
    for bit (the update is deterministic)."""
    X, D0, idx, coef, nnz, resid = _inputs(20000, 256, 8, seed=11)
    c = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    Xt, Dt, it, ct, nt, rt = c(X), c(D0), c(idx.view(np.int16)), c(coef), c(nnz), c(resid)
    eager = lib.mod_update(Xt, Dt, it, ct, nt, rt, sync=True).cpu().numpy()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        lib.mod_update(Xt, Dt, it, ct, nt, rt)  # warm-up: workspace and attributes exist
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        out = lib.mod_update(Xt, Dt, it, ct, nt, rt)
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy(), eager)
