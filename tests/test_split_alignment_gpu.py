"""The digit splits of the split-BF16 and split-TF32 products with operands that
16-byte loads can and cannot read: odd and even leading dimensions of A and B
and bases 8 bytes off a 16-byte boundary, at row, column and inner sizes around
the strips (16 columns, 256 rows) and blocks (32 columns, 128 rows).  The same
numbers must give the same bits whichever loads are taken, and stay within the
splits' error of the FP64 product."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def placed(M, pad, off):
    """M on the device, row pitch M's width + pad, base off elements into its buffer."""
    r, c = M.shape
    buf = torch.zeros(r * (c + pad) + off, dtype=torch.float64, device="cuda")
    view = buf[off:].view(r, c + pad)
    view[:, :c] = torch.from_numpy(M).cuda()
    return buf[off:], c + pad


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (3, 15, 127), (5, 17, 129), (33, 31, 256), (130, 66, 258)])
def test_loads_give_the_same_bits(m, n, k):
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo
    pkg_build.build()
    rng = np.random.default_rng(17)
    A, B = rng.uniform(-1, 1, (m, k)), rng.uniform(-1, 1, (k, n))
    B[:, n // 2] *= 2.0 ** 50  # a column that the BF16 split scales
    bound = np.abs(A) @ np.abs(B)
    ctx = oo.oo_create(0, torch.cuda.Stream())
    try:
        for prec, tol in ((oo.OO_PREC_SPLIT3_BF16, 1e-4), (oo.OO_PREC_SPLIT3_TF32, 1e-5)):
            got = []
            for pa, oa in ((k % 2, 0), (1 - k % 2, 0), (k % 2, 1)):
                for pb, ob in ((n % 2, 0), (1 - n % 2, 0), (n % 2, 1)):
                    dA, lda = placed(A, pa, oa)
                    dB, ldb = placed(B, pb, ob)
                    C = torch.full((m, n), np.nan, dtype=torch.float64, device="cuda")
                    torch.cuda.synchronize()
                    oo.oo_gemm_f64_dev(ctx, m, n, k, dA, lda, dB, ldb, C, n, prec=prec)
                    oo.oo_sync(ctx)
                    got.append(C.cpu().numpy())
            assert np.all(np.abs(got[0] - A @ B) <= tol * bound)
            for g in got[1:]:
                assert np.array_equal(g, got[0])
    finally:
        oo.oo_destroy(ctx)
