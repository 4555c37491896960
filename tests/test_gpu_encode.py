"""Steps a1-a4: GPU Batch-OMP vs the FP64 oracle OMP."""
import numpy as np
import pytest
import torch

from gpu_common import embed45, well_separated
from oracle import omp as oomp
from paper_2605_30396_gb300 import synth

pytestmark = pytest.mark.gpu


def run(lib, D, X, s, prec="fp32", eps=0.0):
    idx, coef, nnz, resid = lib.encode(torch.from_numpy(D.astype(np.float32)).cuda(),
                                       torch.from_numpy(X.astype(np.float32)).cuda(), s, eps=eps,
                                       precision=prec, sync=True)
    return (lib.idx_as_long(idx).cpu().numpy(), coef.cpu().numpy(), nnz.cpu().numpy().astype(int),
            resid.cpu().numpy())


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("n,s", [(16, 2), (32, 3)])
def test_exact_recovery_erc(lib, prec, n, s):
    """Planted s-sparse signals over [I | H/sqrt n] (mu (2s-1) < 1): exact support."""
    D = embed45(synth.erc_dictionary(n))
    rng = np.random.default_rng(n + s)
    X, sup, coef = synth.planted_sparse(rng, D, 777, s)
    idx, cf, nnz, resid = run(lib, D, X, s, prec)
    assert (nnz == s).all()
    np.testing.assert_array_equal(np.sort(idx, 1), np.sort(sup, 1))
    for i in range(50):
        got = dict(zip(idx[i], cf[i]))
        for j, c in zip(sup[i], coef[i]):
            assert abs(got[j] - c) <= 1e-4 * (abs(c) + 1)
    assert resid.max() <= 1e-8 * np.max(np.sum(X * X, 1))


def test_orthonormal_dictionary_is_hard_thresholding(lib):
    rng = np.random.default_rng(3)
    Q, _ = np.linalg.qr(rng.standard_normal((45, 45)))
    D = Q.T
    X = rng.standard_normal((400, 45))
    s = 6
    idx, cf, nnz, _ = run(lib, D, X, s)
    c = X @ D.T
    top = np.argsort(-np.abs(c), axis=1, kind="stable")[:, :s]
    srt = -np.sort(-np.abs(c), axis=1)
    sep = (srt[:, :s] - srt[:, 1:s + 1]).min(axis=1) > 1e-4
    assert sep.mean() > 0.9
    np.testing.assert_array_equal(idx[sep], top[sep])
    np.testing.assert_allclose(cf[sep], np.take_along_axis(c, top, 1)[sep], atol=2e-5)


@pytest.mark.parametrize("N,K,s", [(3000, 256, 8), (1111, 300, 4), (2000, 1024, 16),
                                   (700, 2048, 8), (129, 64, 1)])
def test_plain_fp32_matches_oracle(lib, N, K, s):
    """Configuration-1 generator; supports identical wherever the oracle's every
    selection margin exceeds 1e-4; RMSE within 1e-4 relative; coefficients close."""
    Dh = synth.hidden_dictionary(K, 0)
    X = synth.signals(N, Dh, min(s, 8), 1).astype(np.float64)
    D = synth.hidden_dictionary(K, 7)  # an unrelated dictionary: nontrivial selections
    ref = oomp.omp(D.astype(np.float32).astype(np.float64), X, s)
    idx, cf, nnz, resid = run(lib, D, X, s)
    sep = well_separated(ref["topc"], ref["nnz"], 1e-4)
    assert sep.mean() > 0.8
    np.testing.assert_array_equal(idx[sep], ref["idx"][sep])
    np.testing.assert_array_equal(nnz[sep], ref["nnz"][sep])
    scale = np.abs(ref["coef"][sep]).max(axis=1, keepdims=True) + 1e-12
    assert (np.abs(cf[sep] - ref["coef"][sep]) / scale).max() <= 1e-3
    r_got = np.sqrt(resid.sum() / (N * 45))
    r_ref = np.sqrt(ref["resid_sq"].sum() / (N * 45))
    assert abs(r_got - r_ref) <= 1e-4 * r_ref, (r_got, r_ref)


def in_top4_by_margin(topc, nnz, delta, fp32_margin=1e-4):
    """Signals whose every oracle selection step had its winner ahead of the
    fifth-largest |c| by more than 2 delta (so it is inside any low-precision top
    4 whose error is below delta) and ahead of the runner-up by more than the
    FP32 re-score's margin."""
    gap04 = topc[:, :, 0] - topc[:, :, 4]
    gap01 = topc[:, :, 0] - topc[:, :, 1]
    s = topc.shape[1]
    steps = np.arange(s)[None, :] < np.asarray(nnz)[:, None]
    ok = np.where(steps, (gap04 > 2 * delta) & (gap01 > fp32_margin), True)
    return ok.all(axis=1)


@pytest.mark.parametrize("prec,delta,K,s,N,min_ok", [
    ("bf16", 6e-3, 256, 4, 3000, 50), ("bf16", 6e-3, 300, 8, 3000, 50),
    ("bf16", 6e-3, 1024, 8, 3000, 50), ("bf16", 6e-3, 1024, 16, 3000, 20),
    ("bf16", 6e-3, 2048, 8, 3000, 20),
    # FP8's error bound is ten times BF16's: few signals clear it at every step
    # (none in 20,000 at s = 8), so FP8 is pinned at s = 4
    ("fp8", 6e-2, 256, 4, 20000, 20)])
def test_low_precision_top4_rescore_picks_the_oracle_winner(lib, prec, delta, K, s, N, min_ok):
    """BF16 / FP8 correlation with each row's exact low-precision top 4 re-scored
    in FP32 before every commit (Sec. 2.1's argmax, in the precision reading).
    delta bounds the low-precision correlation error relative to ||r||.  Wherever
    the oracle's winner clears the fifth-largest correlation by more than 2 delta
    at every step, it is inside the low-precision top 4, so the FP32 re-score
    must pick it: the whole support equals the oracle's."""
    Dh = synth.hidden_dictionary(K, 0)
    X = synth.signals(N, Dh, min(s, 8), 1).astype(np.float64)
    D = synth.hidden_dictionary(K, 7)  # an unrelated dictionary: near-tied selections occur
    ref = oomp.omp(D.astype(np.float32).astype(np.float64), X, s)
    idx, cf, nnz, resid = run(lib, D, X, s, prec)
    ok = in_top4_by_margin(ref["topc"], ref["nnz"], delta)
    assert ok.sum() >= min_ok, ok.sum()
    np.testing.assert_array_equal(idx[ok], ref["idx"][ok])
    np.testing.assert_array_equal(nnz[ok], ref["nnz"][ok])
    r_got = np.sqrt(resid.sum() / (N * 45))
    r_ref = np.sqrt(ref["resid_sq"].sum() / (N * 45))
    assert abs(r_got - r_ref) <= 2e-2 * r_ref, (prec, r_got, r_ref)


@pytest.mark.parametrize("prec,delta", [("bf16_qw", 6e-3), ("fp8_qw", 6e-2)])
@pytest.mark.parametrize("K,s", [(256, 4), (300, 8), (1024, 16)])
def test_low_precision_with_rescore(lib, prec, delta, K, s):
    """BF16 / FP8 correlation with the cheaper candidate set: the low-precision
    winner of each column group (quarters of 128-atom chunks for s > 8, halves
    of 64-atom chunks for s <= 8) is re-scored in FP32.  delta bounds the
    low-precision correlation error relative to ||r|| (the a1 tests measure it);
    wherever the oracle's winner clears the runner-up by more than 2 delta at
    every step, it wins its group in low precision and the re-score must pick
    it exactly."""
    N = 3000
    D = synth.hidden_dictionary(K, 7)
    X = synth.signals(N, D, s, 1).astype(np.float64)  # codes over D itself: large margins
    ref = oomp.omp(D.astype(np.float32).astype(np.float64), X, s)
    idx, cf, nnz, resid = run(lib, D, X, s, prec)
    ok = well_separated(ref["topc"], ref["nnz"], 2 * delta)
    if s <= 8:
        assert ok.sum() >= 20, ok.sum()
    np.testing.assert_array_equal(idx[ok], ref["idx"][ok])
    # the first selection (empty support on both sides) wherever its margin clears 2 delta
    first = (ref["nnz"] > 0) & (ref["topc"][:, 0, 0] - ref["topc"][:, 0, 1] > 2 * delta)
    assert first.sum() >= 100, first.sum()
    np.testing.assert_array_equal(idx[first, 0], ref["idx"][first, 0])
    r_got = np.sqrt(resid.sum() / (N * 45))
    r_ref = np.sqrt(ref["resid_sq"].sum() / (N * 45))
    agree = (idx == ref["idx"]).all(axis=1).mean()
    if s <= 8:  # every one of s selections must agree: a strong check at small s
        # (for s <= 8 the candidates are the two column-half winners; FP8's
        # three mantissa bits leave near-ties to more complete supports)
        assert agree > (0.9 if prec == "bf16_qw" else 0.85), agree
    assert abs(r_got - r_ref) <= 5e-2 * r_ref, (prec, agree, r_got, r_ref)


def test_tolerance_stop_zero_and_ragged(lib):
    D = embed45(synth.erc_dictionary(16))
    rng = np.random.default_rng(5)
    X, sup, _ = synth.planted_sparse(rng, D, 200, 2)
    X = np.concatenate([X, np.zeros((3, 45))])
    idx, cf, nnz, resid = run(lib, D, X, 6, eps=1e-3)
    assert (nnz[:200] == 2).all()
    assert (nnz[200:] == 0).all() and (cf[200:] == 0).all() and (idx[200:] == 0).all()
    # pads after nnz are zero
    assert (cf[:200, 2:] == 0).all() and (idx[:200, 2:] == 0).all()


def test_empty_and_single(lib):
    D = synth.hidden_dictionary(64, 1)
    idx, cf, nnz, resid = run(lib, D, np.zeros((0, 45)), 4)
    assert idx.shape == (0, 4)
    X = synth.signals(1, D, 3, 2)
    idx, cf, nnz, resid = run(lib, D, X, 4)
    ref = oomp.omp(D.astype(np.float32).astype(np.float64), X.astype(np.float64), 4)
    np.testing.assert_array_equal(idx, ref["idx"])


def test_residual_orthogonality_and_lstsq(lib):
    N, K, s = 500, 512, 8
    D = synth.hidden_dictionary(K, 3).astype(np.float32).astype(np.float64)
    X = synth.signals(N, synth.hidden_dictionary(K, 4), s, 5).astype(np.float64)
    idx, cf, nnz, resid = run(lib, D, X, s)
    for i in range(0, N, 7):
        I = idx[i, :nnz[i]]
        DI = D[I].T
        r = X[i] - DI @ cf[i, :nnz[i]]
        assert np.abs(DI.T @ r).max() <= 1e-5 * np.linalg.norm(X[i])
        g, *_ = np.linalg.lstsq(DI, X[i], rcond=None)
        np.testing.assert_allclose(cf[i, :nnz[i]], g, rtol=1e-3, atol=1e-5 * np.abs(g).max())
        assert abs(resid[i] - r @ r) <= 1e-4 * (X[i] @ X[i])


def test_deterministic(lib):
    D = synth.hidden_dictionary(1024, 3)
    X = synth.signals(5000, D, 8, 4)
    a = run(lib, D, X, 8)
    b = run(lib, D, X, 8)
    for u, v in zip(a, b):
        np.testing.assert_array_equal(u, v)


@pytest.mark.parametrize("variant", [2, 3, 4, 5, 6, 7, 64, 128])
@pytest.mark.parametrize("N,K,s", [(3000, 256, 8), (2000, 1024, 8), (1500, 300, 4), (777, 64, 1)])
def test_fp32_kernel_variants_match_oracle(lib, variant, N, K, s):
    """Every FP32 encoder the autotuner can pick (two tiles on two warp groups,
    two tiles served in turn, two tiles with selection and solver warps as three
    TF32 or three FP16 products, three such tiles with FP16 products, one tile
    with FP16 products or with 64- or 128-atom TF32 chunks): supports
    identical to the oracle's wherever its every selection margin exceeds 1e-4,
    RMSE within 1e-4 relative."""
    Dh = synth.hidden_dictionary(K, 0)
    X = synth.signals(N, Dh, min(s, 8), 1).astype(np.float64)
    D = synth.hidden_dictionary(K, 7)
    ref = oomp.omp(D.astype(np.float32).astype(np.float64), X, s)
    sc = [{"D": torch.from_numpy(D.astype(np.float32)).cuda(),
           "X": torch.from_numpy(X.astype(np.float32)).cuda(), "s": s}]
    idx, cf, nnz, resid = lib.encode_multi(sc, precision="fp32", bn=variant, sync=True)[0]
    idx = lib.idx_as_long(idx).cpu().numpy()
    nnz = nnz.cpu().numpy().astype(int)
    sep = well_separated(ref["topc"], ref["nnz"], 1e-4)
    assert sep.mean() > 0.8
    np.testing.assert_array_equal(idx[sep], ref["idx"][sep])
    np.testing.assert_array_equal(nnz[sep], ref["nnz"][sep])
    r_got = np.sqrt(resid.cpu().numpy().astype(np.float64).sum() / (N * 45))
    r_ref = np.sqrt(ref["resid_sq"].sum() / (N * 45))
    assert abs(r_got - r_ref) <= 1e-4 * r_ref, (r_got, r_ref)


@pytest.mark.parametrize("variant", [3, 4, 5, 6])
def test_multi_tile_fp32_encoders_over_several_rounds(lib, variant):
    """75,077 signals are 587 tiles: on 152 CTAs of two tile slots, CTAs 131
    and up have a second round with slot 0 only; with three slots, CTAs below
    131 have a second round with slot 0 only and the others one round of three
    tiles; the last tile is ragged.  Supports as the oracle's wherever every
    selection margin exceeds 1e-4, residuals within 2e-4 relative per signal."""
    N, K, s = 75077, 256, 8
    Dh = synth.hidden_dictionary(K, 0)
    X = synth.signals(N, Dh, s, 3).astype(np.float64)
    D = synth.hidden_dictionary(K, 7)
    ref = oomp.omp(D.astype(np.float32).astype(np.float64), X, s)
    sc = [{"D": torch.from_numpy(D.astype(np.float32)).cuda(),
           "X": torch.from_numpy(X.astype(np.float32)).cuda(), "s": s}]
    idx, cf, nnz, resid = lib.encode_multi(sc, precision="fp32", bn=variant, sync=True)[0]
    idx = lib.idx_as_long(idx).cpu().numpy()
    nnz = nnz.cpu().numpy().astype(int)
    sep = well_separated(ref["topc"], ref["nnz"], 1e-4)
    assert sep.mean() > 0.8
    np.testing.assert_array_equal(idx[sep], ref["idx"][sep])
    np.testing.assert_array_equal(nnz[sep], ref["nnz"][sep])
    r = resid.cpu().numpy().astype(np.float64)
    np.testing.assert_allclose(r[sep], ref["resid_sq"][sep], rtol=2e-4, atol=1e-9)


@pytest.mark.parametrize("K,s,prec", [(256, 8, "fp32"), (1024, 4, "fp32"), (130, 1, "fp32"), (512, 16, "fp32"),
                                      (300, 9, "fp32"), (200, 12, "fp32"), (1100, 10, "fp32"), (256, 8, "bf16"),
                                      (500, 5, "fp8"), (130, 3, "bf16_qw"), (100, 4, "bf16"), (130, 3, "fp8"),
                                      (256, 8, "fp8_qw")])
def test_small_calls_match_large_ones(lib, K, s, prec):
    """Up to one tile per SM the FP32 encoder takes tiles of 64 signals instead of
    128, BF16/FP8 give each CTA one tile instead of two, and with s > 8 the kernel
    itself depends on K and N: a signal's code does not depend on any of it, so the
    first N signals alone give bitwise the codes they have in a call of 20,000 (152
    SMs: 64-signal tiles up to 19,456)."""
    n = 20_000
    D = torch.from_numpy(synth.hidden_dictionary(K, 1).astype(np.float32)).cuda()
    X = torch.from_numpy(synth.signals(n, synth.hidden_dictionary(K, 2), min(s, 4), 3)).cuda()
    whole = lib.encode(D, X, s, precision=prec, sync=True)
    for N in (1, 63, 64, 65, 129, 9728, 9729, 19_456, 19_457):
        part = lib.encode(D, X[:N].contiguous(), s, precision=prec, sync=True)
        for a, b in zip(part, whole):
            assert torch.equal(a, b[:N]), N


@pytest.mark.parametrize("K,s", [(200, 12), (64, 16)])
def test_long_codes_around_atoms_without_a_correlation(lib, K, s):
    """s > 8 with atoms that hold a NaN, an infinity, or values beyond the FP16 parts
    (each takes its 32 columns out of the selection): a call of half tiles, two per
    CTA, and one of a whole tile per CTA on the one-tile kernel give the same bits,
    and most signals still get codes."""
    D = synth.hidden_dictionary(K, 1).astype(np.float32)
    D[3], D[5, 2], D[7, 1], D[9] = 0.0, np.nan, np.inf, D[9] * 1e30
    Dt = torch.from_numpy(D).cuda()
    X = torch.from_numpy(synth.signals(14_000, synth.hidden_dictionary(K, 2), 8, 3)).cuda()
    whole = lib.encode(Dt, X, s, sync=True)
    part = lib.encode(Dt, X[:3000].contiguous(), s, sync=True)
    for a, b in zip(part, whole):
        a, b = a.cpu().numpy(), b[:3000].cpu().numpy()
        np.testing.assert_array_equal(a, b)
    assert (part[2].cpu().numpy() > 0).mean() > 0.9


@pytest.mark.parametrize("N,K,s,eps", [(100_003, 300, 12, 0.2), (45_000, 1024, 9, 0.0), (79_000, 640, 16, 0.3)])
def test_long_codes_over_several_rounds(lib, N, K, s, eps):
    """s > 8 on whole tiles, two per CTA, K > 256 and more than 256 signals per SM (one to
    three rounds per CTA, ragged last tiles, tolerance stops), with the bounds of the
    test below."""
    test_codes_of_nine_to_sixteen_atoms(lib, N, K, s, eps)


@pytest.mark.parametrize("N,K,s,eps", [(40_000, 129, 9, 0.0), (2500, 640, 13, 0.3), (300, 2048, 16, 0.0),
                                       (20_100, 64, 16, 0.05)])
def test_codes_of_nine_to_sixteen_atoms(lib, N, K, s, eps):
    """s = 9..16 on two tiles per CTA: whole and half tiles, ragged last tiles,
    several rounds per CTA, tolerance stops.  Supports as the oracle's wherever
    every selection margin exceeds 1e-4 and no residual norm is within 1e-4 of
    the tolerance; coefficients there within 1e-3 (FP32 least squares on up to 16
    atoms), residuals of all signals within 1e-3 in the RMSE."""
    n = min(N, 600)
    rows = np.sort(np.random.default_rng(5).choice(N, n, replace=False))
    D = synth.hidden_dictionary(K, 7)
    X = synth.signals(N, synth.hidden_dictionary(K, 0), 8, 1)
    idx, coef, nnz, resid = lib.encode(torch.from_numpy(D.astype(np.float32)).cuda(), torch.from_numpy(X).cuda(), s,
                                       eps=eps, sync=True)
    Xd, Dd = X[rows].astype(np.float64), D.astype(np.float32).astype(np.float64)
    ref = oomp.omp(Dd, Xd, s, eps)
    ok = well_separated(ref["topc"], ref["nnz"], 1e-4)
    if eps > 0:
        res = np.linalg.norm(ref["resid"], axis=1)
        ok &= np.abs(res - eps) > 1e-4
    gi = lib.idx_as_long(idx).cpu().numpy()[rows]
    gn = nnz.cpu().numpy()[rows].astype(np.int64)
    same = (gn == ref["nnz"]) & (gi == ref["idx"]).all(axis=1)
    assert ok.mean() > 0.5 and same[ok].mean() > 0.995, (ok.mean(), same[ok].mean())
    np.testing.assert_allclose(coef.cpu().numpy()[rows][ok & same], ref["coef"][ok & same], rtol=1e-3, atol=1e-3)
    a = np.sqrt(resid.cpu().numpy()[rows].astype(np.float64).sum())
    b = np.sqrt(ref["resid_sq"].sum())
    assert abs(a - b) <= 1e-3 * b + 1e-4, (a, b)
