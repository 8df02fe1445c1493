"""The pair scheme's error over many K-blocks.  What a long product adds to the
digits' own truncation is the rounding of its running float-float sums.  The
yardstick is the plain order: the products D_pq of a K-block in pairs of
neighbouring q of one p, smallest contributions first, each added by itself and
renormalised, replayed here in FP32 from digits cut in FP64.  However the
kernels group the products, their error against the exact product must not be
larger than that (rms over a 256 x 256 product of uniform entries, the
reference in pairs of doubles)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

BETA, LEVELS, SLICES, KB = 7, 8, 7, 1024


def two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def halves(a):
    c = a * 134217729.0
    h = c - (c - a)
    return h, a - h


def exact(A, B):
    """A B in pairs of doubles."""
    s = torch.zeros(A.shape[0], B.shape[1], dtype=torch.float64, device="cuda")
    e = torch.zeros_like(s)
    Ah, Al = halves(A)
    Bh, Bl = halves(B)
    for j in range(A.shape[1]):
        ah, al, bh, bl = Ah[:, j:j + 1], Al[:, j:j + 1], Bh[j:j + 1], Bl[j:j + 1]
        p = A[:, j:j + 1] * B[j:j + 1]
        s, d = two_sum(s, p)
        e += d + (((ah * bh - p) + ah * bl + al * bh) + al * bl)
    return s, e


def digits(M, dim):
    e = torch.frexp(M.abs().amax(dim, keepdim=True))[1]
    x, out = torch.ldexp(M.abs(), -e), []
    for _ in range(SLICES):
        x = x * 2.0 ** BETA
        out.append(torch.floor(x) * M.sign())
        x = x - torch.floor(x)
    return out, e


def plain_order(A, B):
    dA, ea = digits(A, 1)
    dB, eb = digits(B, 0)
    units = [(p, q) for p in range(1, SLICES + 1) for q in range(1, LEVELS - p + 1, 2)]
    units.sort(key=lambda u: -(u[0] + u[1]))
    order = [(p, x) for p, q in units for x in (q, q + 1) if p + x <= LEVELS]
    h = torch.zeros(A.shape[0], B.shape[1], dtype=torch.float32, device="cuda")
    l = torch.zeros_like(h)
    for k0 in range(0, A.shape[1], KB):
        for p, q in order:
            d = dA[p - 1][:, k0:k0 + KB] @ dB[q - 1][k0:k0 + KB] * 2.0 ** (-BETA * (p + q))
            s, e = two_sum(h, d.float())
            l = l + e
            h = s + l
            l = l - (h - s)
    return torch.ldexp(h.double(), ea + eb), torch.ldexp(l.double(), ea + eb)


@pytest.mark.parametrize("k", [4096, 8192])
def test_error_not_above_plain_order(k):
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo
    pkg_build.build()
    g = torch.Generator(device="cuda").manual_seed(k)
    A = torch.rand(256, k, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
    B = torch.rand(k, 256, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
    C = torch.empty(256, 256, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    ctx = oo.oo_create(0)
    try:
        oo.oo_gemm_f64_dev(ctx, 256, 256, k, A, k, B, 256, C, 256, prec=oo.OO_PREC_FP64EQ)
        oo.oo_sync(ctx)
    finally:
        oo.oo_destroy(ctx)
    s, e = exact(A, B)
    h, l = plain_order(A, B)
    scale = A.abs() @ B.abs()
    got = float((((C - s) - e) / scale).square().mean().sqrt())
    plain = float((((h - s) + (l - e)) / scale).square().mean().sqrt())
    print("k %d: rms %.4e, plain order %.4e, ratio %.4f" % (k, got, plain, got / plain))
    assert got <= plain
