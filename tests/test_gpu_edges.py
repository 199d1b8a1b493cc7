"""Edges of the tiles, slices and splits of the CUDA kernels against the
float64 oracle or exact arithmetic: sizes around each boundary, odd counts,
odd strides, the smallest and the largest of a range."""
import numpy as np
import pytest
import torch

from oracle import spsvm as O

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.fixture(scope="module")
def sp():
    import paper_1404_1066_gb300 as m
    return m


def _kmat(sp, K, fmt, odd_plane=False):
    """A stored kernel matrix of K's values (exact in the format)."""
    rows, n = K.shape
    ld = (n + 127) // 128 * 128
    K32 = _t(K.astype(np.float32))
    if fmt == "fp32":
        buf = torch.zeros(rows * ld, dtype=torch.float32, device=DEV)
        buf.view(rows, ld)[:, :n] = K32
        return sp.KMat(buf, sp.SPSVM_FP32, n, rows, ld, 0), K32.double().cpu().numpy()
    plane = rows * ld + (1 if odd_plane else 0)
    buf = torch.zeros(2 * plane, dtype=torch.bfloat16, device=DEV)
    hi = K32.to(torch.bfloat16)
    lo = (K32 - hi.float()).to(torch.bfloat16)
    buf[:rows * ld].view(rows, ld)[:, :n] = hi
    buf[plane:plane + rows * ld].view(rows, ld)[:, :n] = lo
    return sp.KMat(buf, sp.SPSVM_BF16SPLIT, n, rows, ld, plane), (hi.double() + lo.double()).cpu().numpy()


# columns taken 128 at a time, at least 1,024 points per slice, rows 4 per warp
# and 32 per block
@pytest.mark.parametrize("fmt,kc_fmt", [("fp32", "fp32"), ("fp32", "bf16split"), ("bf16split", "bf16split")])
@pytest.mark.parametrize("n,m,ns", [(2050, 33, 1025), (2050, 31, 2049), (1024, 4, 1), (4097, 65, 127),
                                    (4097, 3, 4097), (130, 1, 0), (9001, 5, 129)])
def test_compaction_edges(sp, fmt, kc_fmt, n, m, ns):
    """Copies are exact, the tail to 128 is zero, and the weighted sums of ns
    products are within 32 FP32 roundings of their terms."""
    g = np.random.default_rng(n + m)
    km, Kref = _kmat(sp, np.exp(-3 * g.random((m, n))), fmt)
    S = np.zeros(n, dtype=bool)
    S[g.choice(n, ns, replace=False)] = True
    w1, w2 = g.standard_normal((2, n)).astype(np.float32)
    kc, _ = _kmat(sp, np.zeros((m, km.ld)), kc_fmt, odd_plane=m % 2 == 1)
    kc.buf.fill_(7.0)
    a, b, count, pos = sp.spsvm_compact_active(km, _t(S.astype(np.uint8)), _t(w1), _t(w2), kc)
    assert int(count.item()) == ns
    np.testing.assert_array_equal(pos.cpu().numpy(), np.cumsum(S) - S)
    got = kc.to_float().double().cpu().numpy()
    want = Kref[:, S]
    if kc_fmt != fmt:
        w32 = _t(want.astype(np.float32))
        hi = w32.to(torch.bfloat16)
        want = (hi.double() + (w32 - hi.float()).to(torch.bfloat16).double()).cpu().numpy()
    np.testing.assert_array_equal(got[:, :ns], want)
    end = (ns + 127) // 128 * 128
    assert np.all(got[:, ns:end] == 0) and np.all(got[:, end:] >= 7.0)
    for out, w in ((a, w1), (b, w2)):
        terms = np.abs(Kref[:, S]) @ np.abs(w[S].astype(np.float64))
        err = np.abs(out.cpu().numpy() - Kref[:, S] @ w[S].astype(np.float64))
        assert np.all(err <= 32 * 2.0 ** -24 * terms + 1e-300)


def _points(n, d, seed, pad):
    """n x d points whose rows are 16-byte aligned, or (pad) are not."""
    g = np.random.default_rng(seed)
    X = g.standard_normal((n, d)).astype(np.float32)
    ld = (d + 3) // 4 * 4 + (1 if pad else 0)
    buf = torch.zeros((n, ld), dtype=torch.float32, device=DEV)
    buf[:, :d] = _t(X)
    return X, buf[:, :d]


# four features a lane, 128 a warp step; planes padded to 64 columns
@pytest.mark.parametrize("pad", [False, True])
@pytest.mark.parametrize("n,d", [(1, 1), (9, 3), (8, 64), (7, 127), (33, 129), (5, 260)])
def test_points_norms_and_planes(sp, n, d, pad):
    """Norms are the FP64 sums rounded once; hi + mid + lo is x exactly."""
    X, Xt = _points(n, d, n + d, pad)
    P = sp.spsvm_prepare_points(Xt, "bf16split")
    want = (X.astype(np.float64) ** 2).sum(1)
    got = P.norms.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - want) <= 2.0 ** -24 * want * (1 + 2.0 ** -20))
    planes = [p.float().cpu().numpy() for p in (P.hi, P.mid, P.lo)]
    np.testing.assert_array_equal(planes[0].astype(np.float64)[:, :d] + planes[1][:, :d] + planes[2][:, :d], X)
    assert all(np.all(p[:, d:] == 0) for p in planes)
    np.testing.assert_array_equal(planes[0][:, :d], _t(X).to(torch.bfloat16).float().cpu().numpy())


# tiles of 64 or 32 rows by 128 points, 16 features a step; the wide tile needs
# 456 tiles of 64 rows
@pytest.mark.parametrize("pad", [False, True])
@pytest.mark.parametrize("n,d,m", [(127, 15, 31), (129, 17, 33), (1, 1, 1), (300, 784, 64), (58_500, 33, 65)])
def test_fp32_block_and_score_edges(sp, n, d, m, pad):
    """FP32 kernel values, and the scores' sums over 128 points in FP32 terms
    of four, against float64 from direct differences."""
    X, Xt = _points(n, d, n + m, pad)
    g = np.random.default_rng(m)
    J = g.choice(n, min(m, n), replace=False)
    gamma = 0.7 / d
    P = sp.spsvm_prepare_points(Xt, "fp32")
    out = sp.kmat_empty(n, len(J), "fp32")
    sp.spsvm_kernel_block(P, _t(J), gamma, "fp32", out)
    K = O.rbf_kernel(X, X[J], gamma)                # n x m
    sq = (X.astype(np.float64) ** 2).sum(1)
    bound = 4 * 2.0 ** -24 * gamma * (sq[:, None] + sq[J][None, :]) + 2e-6
    assert np.all(np.abs(out.to_float().cpu().numpy().T - K) <= bound)

    y = np.where(g.random(n) < 0.5, 1.0, -1.0).astype(np.float32)
    o = (y * (1 + 0.5 * g.standard_normal(n))).astype(np.float32)
    gs, hs, delta = (v.cpu().numpy() for v in sp.spsvm_score_candidates(P, _t(y), _t(o), _t(J), gamma, 1e-3, "fp32"))
    S = (y * o < 1).astype(np.float64)
    r = S * (o.astype(np.float64) - y)
    tol = 4 * 2.0 ** -24
    assert np.all(np.abs(gs - (1e-3 * o[J] + K.T @ r)) <= (bound + tol * K).T @ np.abs(r) + 1e-9)
    assert np.all(np.abs(hs - (1e-3 + (K * K).T @ S)) <= (2 * bound * K + tol * K * K).T @ S + 1e-9)
    np.testing.assert_allclose(delta, gs * gs / (2 * hs), rtol=1e-14)


# query tiles of 128, or 32 with the basis split over 1, 2, 4 or 8 blocks and the
# features over four groups of threads
@pytest.mark.parametrize("pad", [False, True])
@pytest.mark.parametrize("nq,m,d", [(1, 1, 1), (33, 63, 15), (32, 65, 17), (31, 129, 64), (100, 300, 65),
                                    (129, 520, 31), (58_400, 64, 5)])
def test_fp32_decision_edges(sp, nq, m, d, pad):
    """beta_j in FP64 over 12 decades: each kernel value carries its FP32
    bound, and the sum one FP32 rounding."""
    X, Xt = _points(nq + m, d, nq, pad)
    g = np.random.default_rng(d)
    beta = g.standard_normal(m) * 10.0 ** g.uniform(-6, 6, m)
    gamma = 0.7 / d
    f = sp.spsvm_decision(Xt[:m], _t(beta), Xt[m:], gamma, "fp32").cpu().numpy()
    K = O.rbf_kernel(X[m:], X[:m], gamma)
    sq = (X.astype(np.float64) ** 2).sum(1)
    bound = 4 * 2.0 ** -24 * gamma * (sq[m:, None] + sq[None, :m]) + 2e-6
    ref = K @ beta
    assert np.all(np.abs(f - ref) <= bound @ np.abs(beta) + 2.0 ** -24 * np.abs(ref))


# tiles of 128 rows, or of 256 by pairs of CTAs, by 64 or 128 columns; 64
# features a step; score sums kept over a CTA's tiles of one block of candidates
@pytest.mark.parametrize("pad", [False, True])
@pytest.mark.parametrize("n,d,m", [(1, 1, 1), (128, 64, 64), (129, 65, 65), (257, 63, 129), (300, 130, 128),
                                   (20_000, 33, 64), (40_001, 100, 257), (60_000, 7, 300), (600, 33, 300), (5000, 20, 600),
                                   (3000, 9, 2000), (33_000, 12, 1100)])
def test_split_block_score_and_decision_edges(sp, n, d, m, pad):
    """Kernel values: three dropped products and the norms, and d / 16
    truncating accumulations of the large terms; then sums of at most 32 FP32
    terms in chains of 8, beta rounded to FP32."""
    X, Xt = _points(n + m, d, n + d, pad)
    X, Xt, B, Bt = X[:n], Xt[:n], X[n:], Xt[n:]
    g = np.random.default_rng(m)
    J = g.choice(n, min(m, n), replace=False)
    gamma = 0.7 / d
    P = sp.spsvm_prepare_points(Xt, "bf16split")
    out = sp.kmat_empty(n, len(J), "fp32")
    sp.spsvm_kernel_block(P, _t(J), gamma, "bf16split", out)
    K = O.rbf_kernel(X, X[J], gamma)                # n x m
    sq = (X.astype(np.float64) ** 2).sum(1)
    eps = (d / 16 + 8) * 2.0 ** -23 * gamma
    bound = eps * (sq[:, None] + sq[J][None, :]) + 2e-6
    assert np.all(np.abs(out.to_float().cpu().numpy().T - K) <= bound)

    y = np.where(g.random(n) < 0.5, 1.0, -1.0).astype(np.float32)
    o = (y * (1 + 0.5 * g.standard_normal(n))).astype(np.float32)
    gs, hs, delta = (v.cpu().numpy() for v in
                     sp.spsvm_score_candidates(P, _t(y), _t(o), _t(J), gamma, 1e-3, "bf16split"))
    S = (y * o < 1).astype(np.float64)
    r = S * (o.astype(np.float64) - y)
    tol = 12 * 2.0 ** -24
    assert np.all(np.abs(gs - (1e-3 * o[J] + K.T @ r)) <= (bound + tol * K).T @ np.abs(r) + 1e-9)
    assert np.all(np.abs(hs - (1e-3 + (K * K).T @ S)) <= (2 * bound * K + tol * K * K).T @ S + 1e-9)
    np.testing.assert_allclose(delta, gs * gs / (2 * hs), rtol=1e-14)

    beta = g.standard_normal(m) * 10.0 ** g.uniform(-6, 6, m)
    f = sp.spsvm_decision(Bt, _t(beta), Xt, gamma, "bf16split").cpu().numpy()
    K = O.rbf_kernel(X, B, gamma)
    bound = eps * (sq[:, None] + (B.astype(np.float64) ** 2).sum(1)[None, :]) + 2e-6
    assert np.all(np.abs(f - K @ beta) <= (bound + tol * K) @ np.abs(beta) + 1e-30)


def test_split_decision_sums_in_pairs(sp):
    """Partials that cancel: 1,024 basis rows (32 partials a query), beta of
    +-1e6 in pairs on the same point; each partial's 32 terms are FP32."""
    g = np.random.default_rng(3)
    B = np.repeat(g.standard_normal((512, 16)), 2, axis=0).astype(np.float32)
    Q = g.standard_normal((70, 16)).astype(np.float32)
    beta = np.tile([1e6, -1e6], 512) + g.standard_normal(1024)
    f = sp.spsvm_decision(_t(B), _t(beta), _t(Q), 0.05, "bf16split").cpu().numpy()
    K = O.rbf_kernel(Q, B, 0.05)
    assert np.all(np.abs(f - K @ beta) <= 1e6 * K.sum(1) * 8 * 2.0 ** -24)


# 1,024 points a block of the step and the scan, which sum up to 1,024 blocks'
# counts by themselves
@pytest.mark.parametrize("n", [5, 1024, 1025, 1_048_577])
def test_step_stats_and_scan(sp, n):
    """A fit's last record against its outputs: counts exact, the loss (FP32
    pairs of exact terms) to 1e-10; the compaction's positions and count."""
    g = np.random.default_rng(n)
    X = g.standard_normal((n, 2)).astype(np.float32)
    y = np.where(X[:, 0] + 0.7 * g.standard_normal(n) > 0, 1.0, -1.0).astype(np.float32)
    J = g.choice(n, 3, replace=False)
    mdl = sp.spsvm_fit(_t(X), _t(y), 0.8, 0.1, 3, 1e-8, precision="fp32", initial_basis=J, fixed_basis=True)
    o = mdl.outputs(n).astype(np.float64)
    last = mdl.history()[-1]
    S = y * o < 1
    assert len(mdl.history()) > 1 and last["active"] == S.sum() and last["errors"] == (y * o <= 0).sum()
    loss = 0.5 * ((1 - y * o)[S] ** 2).sum()
    assert abs(last["loss"] - loss) <= 1e-10 * loss

    km, _ = _kmat(sp, np.zeros((1, n)), "fp32")
    kc, _ = _kmat(sp, np.zeros((1, km.ld)), "fp32")
    _, _, count, pos = sp.spsvm_compact_active(km, _t(S.astype(np.uint8)), None, None, kc)
    assert int(count.item()) == S.sum()
    np.testing.assert_array_equal(pos.cpu().numpy(), np.cumsum(S) - S)


# FP32: 64 x 32 or 64 x 128 tiles, split form: 256 x 256 tiles of CTA pairs;
# points in splits of at least 128, FP32 sums of 2,048 (8,192) points
@pytest.mark.parametrize("prec,kfmt", [("fp32", "fp32"), ("fp32", "bf16split"), ("bf16split", "bf16split")])
@pytest.mark.parametrize("m,ns", [(1, 1), (65, 127), (64, 129), (129, 0), (255, 2049), (257, 2177), (300, 40_000),
                                  (513, 8193)])
def test_gram_edges(sp, prec, kfmt, m, ns):
    """H against float64, the first rows being the basis; symmetric.  FP32:
    2,048 sequential roundings; split: the products are exact and the tensor
    cores' FP32 accumulation truncates, 8,192 x 4 / 16 times."""
    g = np.random.default_rng(m + ns)
    n = max(ns, m) + 3
    K = np.exp(-2 * g.random((m, n)))
    km, Kref = _kmat(sp, K, kfmt)
    S = np.zeros(n, dtype=bool)
    S[g.choice(n, ns, replace=False)] = True
    kc, _ = _kmat(sp, np.zeros((m, km.ld)), kfmt)
    _, _, count, _ = sp.spsvm_compact_active(km, _t(S.astype(np.uint8)), None, None, kc)
    J = np.arange(m)
    H = sp.spsvm_gram(kc, count, n, km, _t(J), 0.3, prec).cpu().numpy()
    Ks, KJ = Kref[:, S], Kref[:, J]
    ref = 0.3 * 0.5 * (KJ + KJ.T) + Ks @ Ks.T
    assert np.all(np.abs(H - ref) <= 2048 * 2.0 ** -24 * (Ks @ Ks.T) + 1e-12)
    np.testing.assert_array_equal(H, H.T)


# a cluster of up to 8 blocks per 512 points, each with whole chunks of 32 rows
@pytest.mark.parametrize("fmt", ["fp32", "bf16split"])
@pytest.mark.parametrize("n,m", [(1, 1), (511, 33), (513, 257), (1025, 64), (3000, 1000), (80_001, 97)])
def test_products_over_a_cluster(sp, fmt, n, m):
    """u = K v (added to u or not) and o = K beta with the flags and stats of
    the stored o; FP32 chunks of 32 terms, the rest FP64."""
    g = np.random.default_rng(n + m)
    km, Kref = _kmat(sp, np.exp(-3 * g.random((m, n))), fmt)
    v = g.standard_normal(m)
    u0 = g.standard_normal(n).astype(np.float32)
    y = np.where(g.random(n) < 0.5, 1.0, -1.0).astype(np.float32)
    ref, terms = v @ Kref, np.abs(v) @ Kref
    tol = 33 * 2.0 ** -24 * terms + 2.0 ** -24 * (np.abs(ref) + np.abs(u0))
    for add in (False, True):
        u = _t(u0)
        sp.spsvm_gemv(km, _t(v), u, accumulate=add)
        assert np.all(np.abs(u.cpu().numpy() - ref - (u0 if add else 0)) <= tol)
    o = torch.empty(n, dtype=torch.float32, device=DEV)
    active, stats = sp.spsvm_outputs(km, _t(v), _t(y), o)
    oh = o.cpu().numpy()
    assert np.all(np.abs(oh - ref) <= tol)
    margin = y * oh
    np.testing.assert_array_equal(active.cpu().numpy(), margin < 1)
    want = [0.5 * np.sum(np.maximum(0, 1 - margin.astype(np.float64)) ** 2), np.sum(margin <= 0), np.sum(margin < 1)]
    np.testing.assert_allclose(stats.cpu().numpy(), want, rtol=1e-12)


# one CTA up to 2,048 points, four points a thread in registers and the rest
# read again, at most one CTA per SM; the first bracket is [0, 2]
@pytest.mark.parametrize("n", [1, 2048, 2049, 40_001, 400_003])
@pytest.mark.parametrize("scale", [1.0, 0.13, 0.011, 3.7, 1e-4])
def test_line_search_finds_the_root(sp, n, scale):
    """phi'(t) by sorted breakpoints in float64 from the same o and u: its root
    (t near 1 / scale: inside the first bracket, or past it by up to 8^5) to a
    few FP32 roundings of its terms over the slope there."""
    g = np.random.default_rng(n)
    m = min(n, 40)
    y = np.where(g.random(n) < 0.5, 1.0, -1.0).astype(np.float32)
    o = (y * (1 + 0.5 * g.standard_normal(n)) - 0.9 * y * (np.arange(n) == 0)).astype(np.float32)
    step = np.where(y * o < 1, (y - o) * (1 + 0.3 * g.standard_normal(n)), 0.2 * g.standard_normal(n))
    u = (scale * step).astype(np.float32)
    J = np.arange(m)
    d = scale * 1e-3 * np.abs(g.standard_normal(m)) * np.sign(u[J])   # d' K_JJ d >= 0
    lam = 1e-3
    a0, a1 = lam * d @ o[J].astype(np.float64), lam * d @ u[J].astype(np.float64)
    mm = 1 - (y * o).astype(np.float64)
    v = (y * u).astype(np.float64)
    f = lambda t: a0 + a1 * t - np.sum(v * np.maximum(0, mm - t * v))  # noqa: E731
    t = sp.spsvm_line_search(_t(o), _t(u), _t(y), _t(d), _t(J), lam)
    if not f(0.0) < 0:
        assert t == 0.0
        return
    lo, hi = 0.0, 2.0 * 8.0 ** 12
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if f(mid) < 0 else (lo, mid)
    slope = a1 + np.sum(np.where(mm - hi * v > 0, v * v, 0))
    noise = abs(a0) + abs(a1) * hi + np.sum(np.abs(v) * np.maximum(0, np.abs(mm) + hi * np.abs(v)))
    assert abs(t - hi) <= 8 * 2.0 ** -24 * noise / slope + 1e-6 * hi


# diagonal blocks of 64 rows inverted directly, of 256 by columns, merged to
# 1,024; more than one such block; 16 columns a tile and 8 rows a CTA
@pytest.mark.parametrize("m", [2, 64, 66, 129, 255, 256, 257, 320, 513, 1023, 1024, 1025, 1100, 2049, 2500])
@pytest.mark.parametrize("ldx,shift", [(0, 0.0), (1, 0.5)])
def test_mixed_solve_over_block_inverses(sp, m, ldx, shift):
    """Backward error 1e-13 as asked, from H with an even and an odd pitch, H
    untouched, and the 64 x 64 blocks' inverses beside the factor."""
    g = np.random.default_rng(m)
    A = g.standard_normal((m, m + 8)) / np.sqrt(m)
    Hn = A @ A.T + 0.2 * np.eye(m)
    buf = torch.zeros((m, m + ldx), dtype=torch.float64, device=DEV)
    buf[:, :m] = _t(Hn)
    H, b = buf[:, :m], _t(g.standard_normal(m))
    info, status, x, iters, be = sp.spsvm_solve_mixed(H, b, shift=shift)
    assert info == 0 and status == 0 and be <= 1e-13
    np.testing.assert_array_equal(H.cpu().numpy(), Hn)
    Hs = Hn + shift * np.eye(m)
    xn, bn = x.cpu().numpy(), b.cpu().numpy()
    r = np.max(np.abs(bn - Hs @ xn))
    assert r <= 2e-13 * (np.max(np.abs(Hs).sum(1)) * np.max(np.abs(xn)) + np.max(np.abs(bn)))
    info, Lw = sp.spsvm_cholesky_mixed(H, shift=shift)
    Lw = Lw.cpu().numpy().astype(np.float64)
    for k in {0, (m - 1) // 64}:
        D = Lw[64 * k:64 * k + 64, 64 * k:min(m, 64 * k + 64)]
        low, inv = np.tril(D), np.triu(D, 1).T + np.diag(1 / np.diag(D))
        c = np.abs(np.linalg.inv(low)) @ np.abs(low)
        assert np.all(np.abs(inv @ low - np.eye(len(D))) <= 64 * 2.0 ** -24 * c @ c + 1e-12)
