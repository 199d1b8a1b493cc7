"""Inputs that the entry points accept beside the usual ones: kernel matrices
whose planes lie an odd number of elements apart, active flags of any nonzero
byte, coefficients past FP32's range, requests of any size."""
import numpy as np
import pytest
import torch

from oracle import spsvm as O

pytestmark = pytest.mark.gpu


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.fixture(scope="module")
def sp():
    import paper_1404_1066_gb300 as m
    return m


def _split_kmat(sp, K, gap):
    """hi / lo planes of K, `gap` elements between them; and the values held."""
    rows, n = K.shape
    ld = (n + 7) // 8 * 8
    plane = rows * ld + gap
    buf = torch.zeros(2 * plane, dtype=torch.bfloat16, device="cuda")
    K32 = _t(K.astype(np.float32))
    hi = K32.to(torch.bfloat16)
    lo = (K32 - hi.float()).to(torch.bfloat16)
    buf[:rows * ld].view(rows, ld)[:, :n] = hi
    buf[plane:plane + rows * ld].view(rows, ld)[:, :n] = lo
    return sp.KMat(buf, sp.SPSVM_BF16SPLIT, n, rows, ld, plane), (hi.double() + lo.double()).cpu().numpy()


# planes an even and an odd number of elements apart; one block of 512 points,
# clusters, and more blocks than six per SM
@pytest.mark.parametrize("gap", [0, 1, 2, 5])
@pytest.mark.parametrize("n,m", [(1, 1), (7, 3), (515, 70), (3001, 129), (500_001, 3)])
def test_products_with_planes_any_distance_apart(sp, gap, n, m):
    """u = K v and o = K beta: FP32 chunks of 32 terms, then one rounding."""
    g = np.random.default_rng(n + gap)
    km, Kref = _split_kmat(sp, np.exp(-3 * g.random((m, n))), gap)
    v = g.standard_normal(m)
    y = np.where(g.random(n) < 0.5, 1.0, -1.0).astype(np.float32)
    ref = v @ Kref
    tol = 33 * 2.0 ** -24 * (np.abs(v) @ Kref) + 2.0 ** -24 * np.abs(ref)
    u = torch.empty(n, dtype=torch.float32, device="cuda")
    sp.spsvm_gemv(km, _t(v), u)
    assert np.all(np.abs(u.cpu().numpy() - ref) <= tol)
    o = torch.empty(n, dtype=torch.float32, device="cuda")
    active, _ = sp.spsvm_outputs(km, _t(v), _t(y), o)
    np.testing.assert_array_equal(o.cpu().numpy(), u.cpu().numpy())
    np.testing.assert_array_equal(active.cpu().numpy(), y * o.cpu().numpy() < 1)


# flags of one set written as 1, 255 and a mix; up to and past the points that
# the writers of the list count by themselves
@pytest.mark.parametrize("n", [1, 1025, 40_000, 1_048_577 + 3])
def test_active_flags_are_any_nonzero_byte(sp, n):
    """Count, positions, copies and sums are those of the set; flags that
    differ only as bytes are no change."""
    g = np.random.default_rng(n)
    S = g.random(n) < 0.4
    K = np.exp(-g.random((2, n)))
    km = sp.kmat_empty(n, 2, "fp32")
    km.buf.view(2, km.ld)[:, :n] = _t(K.astype(np.float32))
    w = _t(g.standard_normal(n).astype(np.float32))
    outs = []
    for values in ([1], [255], [1, 2, 128, 255]):
        act = (S * g.choice(values, n)).astype(np.uint8)
        kc = sp.kmat_empty(km.ld, 2, "fp32")
        a, b, count, pos = sp.spsvm_compact_active(km, _t(act), w, w, kc)
        assert int(count.item()) == S.sum()
        np.testing.assert_array_equal(pos.cpu().numpy(), np.cumsum(S) - S)
        outs.append((a.cpu().numpy(), kc.to_float().cpu().numpy()))
        ref = (S * g.choice([1, 3, 255], n)).astype(np.uint8)
        changed = g.choice(n, min(n, 3), replace=False)
        ref[changed] = np.where(S[changed], 0, 255)
        k, Wt, sign = sp.spsvm_active_diff(km, _t(act), _t(ref), 8)
        changed.sort()
        assert k == len(changed)
        np.testing.assert_array_equal(sign.cpu().numpy(), np.where(S[changed], 1.0, -1.0))
        np.testing.assert_array_equal(Wt.cpu().numpy(), km.to_float().cpu().numpy()[:, changed])
    np.testing.assert_array_equal(outs[0][1][:, :S.sum()], K.astype(np.float32)[:, S])
    for o in outs[1:]:
        np.testing.assert_array_equal(o[0], outs[0][0])
        np.testing.assert_array_equal(o[1], outs[0][1])


# one block of 64 rows, several, and more than one inverse of 1,024 rows
@pytest.mark.parametrize("m", [3, 130, 1100])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_solve_of_what_is_not_finite_does_not_converge(sp, m, bad):
    """A NaN or an infinity in b is no solution with backward error zero; b of
    zeros has one."""
    SPSVM_ERR_NO_CONVERGE = -4
    g = np.random.default_rng(m)
    A = g.standard_normal((m, m + 8)) / np.sqrt(m)
    H = _t(A @ A.T + 0.5 * np.eye(m))
    for k in (0, m - 1):
        b = g.standard_normal(m)
        b[k] = bad
        info, status, x, iters, be = sp.spsvm_solve_mixed(H, _t(b))
        assert info == 0 and status == SPSVM_ERR_NO_CONVERGE and not be <= 1e-13
    info, status, x, iters, be = sp.spsvm_solve_mixed(H, _t(np.zeros(m)))
    assert info == 0 and status == 0 and be == 0.0 and torch.all(x == 0)


# single CTAs and pairs of them, tiles of 64 and 128 basis rows, a last partial
# tile, two passes of queries; SIMT tiles of 32 and 128 queries, clusters of 1 to
# 8 blocks, one to four shares of the features
@pytest.mark.parametrize("precision", ["fp32", "bf16split"])
@pytest.mark.parametrize("m,d", [(1, 3), (40, 17), (65, 64), (300, 130), (600, 784), (2100, 33)])
def test_decision_value_is_the_same_in_any_request(sp, precision, m, d):
    """A query's value has the same bits alone, in a small and in a large
    request, wherever it stands in it."""
    g = np.random.default_rng(m + d)
    nq = 40_000
    Q = _t(g.standard_normal((nq, d)).astype(np.float32))
    B = _t(g.standard_normal((m, d)).astype(np.float32))
    beta = _t(g.standard_normal(m) * 10.0 ** g.uniform(-3, 3, m))
    f = sp.spsvm_decision(B, beta, Q, 0.5 / d, precision).cpu().numpy()
    for a, b in [(0, 1), (17, 18), (127, 160), (100, 229), (0, 1000), (5, 3005), (20_000, 32_769),
                 (39_999, 40_000), (3, 40_000)]:
        part = sp.spsvm_decision(B, beta, Q[a:b], 0.5 / d, precision).cpu().numpy()
        np.testing.assert_array_equal(part, f[a:b])


# one tile and several lanes of tiles, the small and the wide tile
@pytest.mark.parametrize("nq", [5, 60_000])
@pytest.mark.parametrize("m", [3, 70, 700])
def test_coefficients_beyond_fp32(sp, m, nq):
    """beta_j past FP32's range where the kernel value brings the term back, and
    as small as FP64 goes, beside ordinary ones.  Kernel values carry the
    rounding of their exponent (FP32 norms and product) and of the exponential;
    sums are FP64, or FP32 pairs, then rounded once."""
    g = np.random.default_rng(m)
    d, gamma = 4, 1.0
    B = g.standard_normal((m, d)).astype(np.float32)
    Q = g.standard_normal((nq, d)).astype(np.float32)
    beta = g.standard_normal(m)
    far = g.choice(m, max(1, m // 5), replace=False)
    B[far] += 4.0 * np.sign(B[far])     # exp(-d2) about 1e-20 to 1e-60
    beta[far] *= 10.0 ** g.uniform(38, 42, len(far))
    beta[g.choice(m, m // 4, replace=False)] *= 1e-200
    f = sp.spsvm_decision(_t(B), _t(beta), _t(Q), gamma, "fp32").cpu().numpy().astype(np.float64)
    K = O.rbf_kernel(Q, B, gamma)
    sq = (Q.astype(np.float64) ** 2).sum(1)[:, None] + (B.astype(np.float64) ** 2).sum(1)[None, :]
    rel = 8 * 2.0 ** -24 * gamma * sq + 2.0 ** -20
    err = (rel * K + 2.0 ** -149) @ np.abs(beta)
    ref = K @ beta
    inside = np.abs(ref) < 1e38
    assert inside.mean() > 0.5 and np.all(np.isfinite(f[inside]))
    assert np.all(np.abs(f - ref)[inside] <= (err + 2.0 ** -23 * np.abs(ref) + 1e-44)[inside])
