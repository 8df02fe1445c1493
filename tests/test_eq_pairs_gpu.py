"""The pair scheme (k > 512) at the edges of its K-blocks, tiles and C store:
inner dimensions around one, two and three K-blocks of at most 1024 terms (all
about as long), rows and columns around the 128- and 256-row tiles and the
8-column groups in which C is written, odd leading dimensions.  Entries are
integers below 2^10 times a power of two, so every product sum is an integer
below 2500 * 2^20 < 2^32 of that unit: cut into digits without remainder, exact
in the float-float sums, and FP64 gives it exactly; the result must equal it,
in the middle of the range and at both ends (results down among the
subnormals are rounded once, as ldexp rounds)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 513), (7, 9, 577), (127, 129, 1024), (129, 127, 1025), (256, 8, 1088), (257, 255, 1300),
          (300, 33, 2048), (64, 300, 2049), (513, 261, 2113),
          (2001, 1101, 577)]  # the last in wide tiles (one wave of CTA pairs), the others in narrow ones


@pytest.mark.parametrize("ea,eb", [(0, 0), (-600, -455), (500, 480)])
def test_edges_exact_alone_and_batched(ea, eb):
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo
    pkg_build.build()
    rng = np.random.default_rng(7)
    ctx = oo.oo_create(0, torch.cuda.Stream())
    try:
        reqs, want = [], []
        for m, n, k in SHAPES:
            A = rng.integers(-1023, 1024, (m, k)).astype(np.float64)
            B = rng.integers(-1023, 1024, (k, n)).astype(np.float64)
            want.append(np.ldexp(A @ B, ea + eb))
            A, B = np.ldexp(A, ea), np.ldexp(B, eb)
            got = oo.oo_gemm_f64(ctx, A, B, prec=oo.OO_PREC_FP64EQ)
            assert np.array_equal(got, want[-1]), (m, n, k)
            reqs.append(dict(kind="gemm", prec=oo.OO_PREC_FP64EQ, m=m, n=n, k=k, A=torch.from_numpy(A).cuda(),
                             B=torch.from_numpy(B).cuda(),
                             C=torch.full((m, n), np.nan, dtype=torch.float64, device="cuda")))
        torch.cuda.synchronize()
        b = oo.oo_batch_create(ctx, reqs)
        try:
            oo.oo_batch_run(ctx, b, 0)
            oo.oo_batch_check(ctx, b)
            for r, w in zip(reqs, want):
                assert np.array_equal(r["C"].cpu().numpy(), w), (r["m"], r["n"], r["k"])
        finally:
            oo.oo_batch_destroy(b)
    finally:
        oo.oo_destroy(ctx)
