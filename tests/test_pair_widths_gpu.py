"""The split-BF16 product at every tile width that the rule can choose (64 to 224
columns; the context option pins 160 and wider only): shapes whose cheapest
width by the rule's own costs is the wanted one, ragged against it, must give
the bits of the single-CTA kernel."""
import itertools

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def rule(m, n, k, clusters):
    """The width with the least waves x K steps x (56 + w) + 15 w, the widest on a tie."""
    slabs, steps = -(-m // 256), -(-k // 64)
    return min(range(256, 63, -32), key=lambda w: -(-slabs * -(-n // w) // clusters) * steps * (56 + w) + 15 * w)


@pytest.mark.parametrize("width", [64, 96, 128, 160, 192, 224])
def test_chosen_width_gives_the_same_bits(width):
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo
    pkg_build.build()
    clusters = torch.cuda.get_device_properties(0).multi_processor_count // 2
    shapes = sorted((m * n * k, m, n, k)
                    for m, n, k in itertools.product((100, 276, 600, 1100), range(33, 4000, 61), (129, 394, 1000, 2000))
                    if rule(m, n, k, clusters) == width)
    # last tiles of one column to a full one: as full as can be, as empty as can be, in between
    picks = {min(shapes, key=lambda s: (s[2] - 1) % width), max(shapes, key=lambda s: (s[2] - 1) % width), shapes[0]}
    pair, single = oo.oo_create(0), oo.oo_create(0)
    try:
        oo.oo_set_option(single, oo.OO_OPT_GEMM_PAIR, 0)
        for _, m, n, k in sorted(picks):
            g = torch.Generator(device="cuda").manual_seed(m + n + k)
            A = torch.rand(m, k, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
            B = torch.rand(k, n, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
            C = [torch.full((m, n), np.nan, dtype=torch.float64, device="cuda") for _ in range(2)]
            torch.cuda.synchronize()
            for ctx, c in zip((pair, single), C):
                oo.oo_gemm_f64_dev(ctx, m, n, k, A, k, B, n, c, n, prec=oo.OO_PREC_SPLIT3_BF16)
                oo.oo_sync(ctx)
                oo.oo_gemm_check(ctx, m, n, k)
            assert torch.equal(C[0], C[1]), (m, n, k)
            assert float(((C[0] - A @ B).abs() / (A.abs() @ B.abs())).max()) <= 1e-4
    finally:
        oo.oo_destroy(pair)
        oo.oo_destroy(single)
