"""Tensor-core kernels whose waits give up at once (spsvm_set_wait_limit(1)):
the call ends with OK or TIMEOUT on its stream, with nothing of it left in
flight, and the same call afterwards gives the same bits as before.  Waits on
shared-memory barriers may also succeed in their one poll, so either outcome is
right; no fault or unbounded wait is involved."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SPSVM_ERR_TIMEOUT = -6


def _calls(sp):
    g = torch.Generator(device="cuda").manual_seed(5)
    n, d, m = 40_000, 96, 300
    X = torch.randn(n, d, device="cuda", generator=g)
    y = torch.where(torch.rand(n, device="cuda", generator=g) < 0.5, 1.0, -1.0)
    o = y * (1 + 0.5 * torch.randn(n, device="cuda", generator=g))
    beta = torch.randn(m, dtype=torch.float64, device="cuda", generator=g)
    P = sp.spsvm_prepare_points(X, "bf16split")
    J = torch.arange(m, device="cuda")

    def block():
        return sp.spsvm_kernel_block(P, J, 0.01, "bf16split", sp.kmat_empty(n, m, "fp32")).to_float()

    def score():
        return torch.stack(sp.spsvm_score_candidates(P, y, o, J, 0.01, 1e-3, "bf16split"))

    def decide():
        return sp.spsvm_decision(X[:m], beta, X[:20_000], 0.01, "bf16split")

    def gram(rows, cols):
        K = sp.kmat_empty(cols, rows, "bf16split")
        K.buf.copy_(torch.rand(K.buf.shape, device="cuda", generator=g))
        ns = torch.tensor([cols], device="cuda")
        return lambda: sp.spsvm_gram(K, ns, cols, K, torch.arange(rows, device="cuda"), 0.1, "bf16split")

    A = torch.randn(1024, 1100, dtype=torch.float64, device="cuda", generator=g)
    H = A @ A.T + torch.eye(1024, dtype=torch.float64, device="cuda")

    def factor():
        L = H.clone()
        sp.spsvm_cholesky(L)
        return torch.tril(L)

    return {"block": block, "score": score, "decide": decide, "gram_single": gram(200, 20_000),
            "gram_pair": gram(1500, 40_000), "factor": factor}


@pytest.mark.parametrize("name", ["block", "score", "decide", "gram_single", "gram_pair", "factor"])
def test_recovers_from_waits_that_give_up(name):
    import paper_1404_1066_gb300 as sp
    lib = sp.load()
    run = _calls(sp)[name]
    want = run()
    torch.cuda.synchronize()
    code = ctypes.c_int32(-9)
    assert lib.spsvm_device_status(ctypes.byref(code)) == 0
    for _ in range(3):
        try:
            lib.spsvm_set_wait_limit(1)
            run()
            torch.cuda.synchronize()
        finally:
            lib.spsvm_set_wait_limit(0)
        rc = lib.spsvm_device_status(ctypes.byref(code))
        assert rc in (0, SPSVM_ERR_TIMEOUT) and (rc == 0) == (code.value == 0)
        got = run()
        torch.cuda.synchronize()
        assert lib.spsvm_device_status(ctypes.byref(code)) == 0
        np.testing.assert_array_equal(got.cpu().numpy(), want.cpu().numpy())
