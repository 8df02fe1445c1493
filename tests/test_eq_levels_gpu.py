"""The level-scheme kernel of FP64-equivalent products (k <= 512) at the edges
of its tiles, boxes and K steps: row counts around 32, 64 and 128 (TMA boxes,
partial tiles), column counts around 32 and 64 (tile widths, odd and even
leading dimensions of C), inner dimensions around the K step and the change of
digit width (128).  Entries are integers below 2^10, so every product sum is an
integer below 512 * 2^20 = 2^29: representable, cut into digits without
remainder in the levels kept, and FP64 gives it exactly; the result must equal
it.  Alone and all in one batch, so that tiles of both digit widths and both
tile widths follow one another on an SM."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (31, 32, 63), (32, 33, 64), (33, 31, 65), (64, 64, 128), (65, 65, 129), (63, 66, 512),
          (127, 95, 127), (128, 96, 130), (129, 97, 200), (200, 1, 511), (1, 200, 512), (257, 130, 448), (300, 161, 5)]


@pytest.fixture(scope="module")
def oo_mod():
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo
    pkg_build.build()
    return oo


def integers(rng, *shape):
    return rng.integers(-1023, 1024, shape).astype(np.float64)


def test_edges_exact_alone_and_batched(oo_mod):
    oo = oo_mod
    rng = np.random.default_rng(3)
    ctx = oo.oo_create(0, torch.cuda.Stream())
    try:
        reqs, want = [], []
        for rep in range(12):  # several tiles for every SM
            for m, n, k in SHAPES:
                A, B = integers(rng, m, k), integers(rng, k, n)
                want.append(A @ B)
                if rep == 0:
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


def test_leading_dimensions_and_range(oo_mod):
    """C inside a wider matrix whose other columns stay, and scales at both
    ends of the exponent range (the epilogue's general conversion): within the
    pattern's bound 2^-42 of k max|a| max|b| (k = 70), or half a subnormal's
    spacing, 2^-1075, for results that small."""
    oo = oo_mod
    rng = np.random.default_rng(4)
    m, n, k, ldc = 70, 45, 70, 61
    ctx = oo.oo_create(0, torch.cuda.Stream())
    try:
        for ea, eb in ((0, 0), (500, 490), (-520, -530), (-600, -440)):
            A, B = rng.uniform(-1, 1, (m, k)), rng.uniform(-1, 1, (k, n))
            exact = A @ B
            dA = torch.from_numpy(np.ldexp(A, ea)).cuda()
            dB = torch.from_numpy(np.ldexp(B, eb)).cuda()
            C = torch.full((m, ldc), 7.0, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            oo.oo_gemm_f64_dev(ctx, m, n, k, dA, k, dB, n, C, ldc, prec=oo.OO_PREC_FP64EQ)
            oo.oo_gemm_check(ctx, m, n, k)
            got = C.cpu().numpy()
            assert np.all(got[:, n:] == 7.0)
            bound = np.ldexp(k * 2.0 ** -42, ea + eb) + 2.0 ** -1074
            assert np.all(np.abs(got[:, :n] - np.ldexp(exact, ea + eb)) <= bound), (ea, eb)
    finally:
        oo.oo_destroy(ctx)
