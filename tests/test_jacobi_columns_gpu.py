"""Sweeps over grids with more (k, j) tile columns than CTAs: rounds of whole
columns, with and without columns left over for segments and tails, in every
tile variant; p and wrk2 exchanged over three iterations.  p must be the
oracle's bits, the residuals within the stencil's 1e-9 of the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

# columns at 128 x 8 (the default where K - 1 fills 128 columns): 8 x 25 = 200, 8 x
# 19 = 152 (as many as SMs), 16 x 19 = 304, 1 x 153
SHAPES = [(30, 200, 1000), (5, 154, 1000), (4, 154, 2000), (6, 1226, 66)]


@pytest.mark.parametrize("shape", SHAPES)
def test_whole_columns(shape):
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo
    pkg_build.build()
    I, J, K = shape
    iters = 3
    ref_res, ref_p = oracle.jacobi_run(I, J, K, iters, mode=1)
    ctx = oo.oo_create(0)
    try:
        oo.oo_set_option(ctx, oo.OO_OPT_JACOBI_FUSED, 0)
        for variant in range(-1, oo.OO_STENCIL_VARIANTS):
            oo.oo_set_option(ctx, oo.OO_OPT_STENCIL_VARIANT, variant)
            p, res = np.empty(I * J * K, np.float32), np.empty(iters)
            st = oo.oo_run_pattern(ctx, 63, 1, oo.jacobi(I, J, K, iters), p, res)
            assert st["n_launches"] == 2 + 2 * iters
            assert np.array_equal(p, ref_p.reshape(-1).astype(np.float32)), variant
            assert np.max(np.abs(res - ref_res) / ref_res) <= 1e-9, variant
    finally:
        oo.oo_destroy(ctx)
