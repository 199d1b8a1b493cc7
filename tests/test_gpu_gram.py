"""The masked Gram matrix over all of its kernels and splits: single CTAs on 128 x
128 tiles, pairs of CTAs on 256 x 256, the choice between them from the points
on the device, and matrices of few tiles on many points."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _split(K):
    hi = K.to(torch.bfloat16)
    return hi, (K - hi.float()).to(torch.bfloat16)


# m: one row of tiles, remainders of 128 and 256, and (2,049) more tiles of 128
# than SMs, which only pairs take.  ns: none, one point, around one slice of
# 8,192 and around as many as a wave of single CTAs takes (one for m = 1,409, ten
# for 513), a remainder of the 64-point steps, more slices than 16 splits.
@pytest.mark.parametrize("prec", ["fp32", "bf16split"])
@pytest.mark.parametrize("m,n,counts", [
    (64, 200_003, (0, 131_073, 200_000)),
    (130, 150_000, (1, 140_001)),
    (513, 100_000, (64 * 7 + 1, 81_920, 81_921)),
    (1409, 40_000, (0, 1, 8192, 8193, 16_385, 40_000)),
    (2049, 20_000, (0, 65, 8193, 20_000))])
def test_gram_over_kernels_and_splits(m, n, counts, prec):
    """H = lambda K_JJ + K_S K_S' against float64 from the stored values,
    symmetric.  FP32: 2,048 sequential roundings; split: the products are exact
    and the tensor cores' FP32 accumulation truncates, 8,192 x 4 / 16 times."""
    import paper_1404_1066_gb300 as sp
    g = torch.Generator(device="cuda").manual_seed(m)
    cols = (n + 127) // 128 * 128
    kc = sp.kmat_empty(cols, m, prec)
    vals = torch.exp(-2 * torch.rand(m, cols, device="cuda", generator=g))
    if prec == "bf16split":
        hi, lo = _split(vals)
        kc.buf[:m * kc.ld].view(m, kc.ld)[:, :cols] = hi
        kc.buf[kc.plane:kc.plane + m * kc.ld].view(m, kc.ld)[:, :cols] = lo
        vals = hi.float() + lo.float()
    else:
        kc.buf.view(m, kc.ld)[:, :cols] = vals
    K = sp.KMat(kc.buf, kc.format, cols, m, kc.ld, kc.plane)
    J = torch.arange(m, device="cuda")
    KJ = vals[:, :m].double()
    for ns in counts:
        # columns from ns up to the next multiple of 128 are zero, as the compaction leaves them
        end = (ns + 127) // 128 * 128
        Kz = sp.kmat_empty(cols, m, prec)
        Kz.buf.copy_(kc.buf)
        for off in (0,) if prec == "fp32" else (0, kc.plane):
            Kz.buf[off:off + m * kc.ld].view(m, kc.ld)[:, ns:end] = 0
        H = sp.spsvm_gram(Kz, torch.tensor([ns], device="cuda"), n, K, J, 0.3, prec)
        Ks = vals[:, :ns].double()
        S = Ks @ Ks.T
        ref = 0.3 * 0.5 * (KJ + KJ.T) + S
        assert torch.all((H - ref).abs() <= 2048 * 2.0 ** -24 * S + 1e-12), (ns, (H - ref).abs().max())
        np.testing.assert_array_equal(H.cpu().numpy(), H.T.cpu().numpy())
