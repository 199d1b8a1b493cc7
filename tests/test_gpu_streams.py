"""Calls that fill the GPU by themselves (cooperative launches of a CTA per SM)
on several streams at once, and the mixed solve between well conditioned and
hopeless."""
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_cooperative_launches_on_several_streams():
    """Line searches over 400,000 points and solves of 1,300 unknowns from four
    threads, each on its own stream: the bits of the same calls alone."""
    import paper_1404_1066_gb300 as sp
    sp.load()
    g = torch.Generator(device="cuda").manual_seed(3)
    n, m = 400_000, 1300
    jobs = []
    for k in range(4):
        y = torch.where(torch.rand(n, device="cuda", generator=g) < 0.5, 1.0, -1.0)
        o = y * (1 + 0.5 * torch.randn(n, device="cuda", generator=g))
        u = (y - o) * (1 + 0.3 * torch.randn(n, device="cuda", generator=g))
        d = 1e-3 * torch.rand(40, dtype=torch.float64, device="cuda", generator=g) * torch.sign(u[:40])
        A = torch.randn(m, m + 8, dtype=torch.float64, device="cuda", generator=g) / m ** 0.5
        H = A @ A.T + 0.5 * torch.eye(m, dtype=torch.float64, device="cuda")
        b = torch.randn(m, dtype=torch.float64, device="cuda", generator=g)
        jobs.append((o, u, y, d, torch.arange(40, device="cuda"), H, b))

    def work(job):
        o, u, y, d, J, H, b = job
        t = sp.spsvm_line_search(o, u, y, d, J, 1e-3)
        info, status, x, iters, be = sp.spsvm_solve_mixed(H, b)
        assert info == 0 and status == 0
        return t, x.cpu().numpy()

    want = [work(j) for j in jobs]
    torch.cuda.synchronize()
    got, errors = [None] * 4, []

    def run(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(10):
                    got[k] = work(jobs[k])
        except Exception as e:   # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for (t0, x0), (t1, x1) in zip(want, got):
        assert t0 == t1
        np.testing.assert_array_equal(x0, x1)


# inverses of 256, 512 and 1,024 rows, one and more of them
@pytest.mark.parametrize("m", [256, 700, 1024, 1500])
@pytest.mark.parametrize("cond,most", [(1e3, 4), (1e5, 6), (1e6, 11)])
def test_mixed_solve_of_ill_conditioned_systems(m, cond, most):
    """Eigenvalues spread evenly over the logarithm: the residual shrinks by the FP32
    solve's error, about 2^-24 cond, a step, from 1 to 1e-13."""
    import paper_1404_1066_gb300 as sp
    g = torch.Generator(device="cuda").manual_seed(m)
    Q, _ = torch.linalg.qr(torch.randn(m, m, dtype=torch.float64, device="cuda", generator=g))
    lam = torch.logspace(0, -np.log10(cond), m, dtype=torch.float64, device="cuda")
    H = (Q * lam) @ Q.T
    H = 0.5 * (H + H.T).contiguous()
    b = torch.randn(m, dtype=torch.float64, device="cuda", generator=g)
    info, status, x, iters, be = sp.spsvm_solve_mixed(H, b)
    assert info == 0 and status == 0 and be <= 1e-13 and iters <= most
    r = (b - H @ x).abs().max()
    assert r <= 2e-13 * (H.abs().sum(1).max() * x.abs().max() + b.abs().max())
