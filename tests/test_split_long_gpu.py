"""The split of B in the split-BF16 product where a long inner dimension and few
columns meet an odd leading dimension (tiles instead of one CTA a strip): the
same numbers at an even leading dimension take the strips and must give the
same bits, in columns that are scaled, zero and non-finite too, on both sides
of the line between the two."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(3, 1, 16383), (3, 1, 16384), (5, 17, 16385), (2, 65, 16447), (3, 511, 16384),
                                   (2, 513, 16384)])
def test_tiles_equal_strips(m, n, k):
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo
    pkg_build.build()
    g = torch.Generator(device="cuda").manual_seed(k + n)
    A = torch.rand(m, k, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
    B = torch.rand(k, n, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
    B[:, n // 2] *= 2.0 ** 50   # scaled
    if n > 16:
        B[:, 3] *= 2.0 ** -30   # scaled
        B[:, 5] = 0.0
        B[k - 1, 7] = float("inf")
    ctx = oo.oo_create(0)
    try:
        got = []
        for pad in (1 - n % 2, n % 2):  # odd, then even
            dB = torch.zeros(k, n + pad, dtype=torch.float64, device="cuda")
            dB[:, :n] = B
            C = torch.empty(m, n, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            oo.oo_gemm_f64_dev(ctx, m, n, k, A, k, dB, n + pad, C, n, prec=oo.OO_PREC_SPLIT3_BF16)
            oo.oo_sync(ctx)
            got.append(C)
    finally:
        oo.oo_destroy(ctx)
    assert torch.equal(got[0].view(torch.int64), got[1].view(torch.int64))
    finite = torch.isfinite(B).all(0)
    assert torch.isnan(got[0][:, ~finite]).all()
    err = (got[0] - A @ B).abs()[:, finite] / (A.abs() @ B.abs())[:, finite].clamp_min(1e-300)
    assert float(err.max()) <= 1e-4
