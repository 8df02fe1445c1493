"""N3 + N4 + N5 in one pass behind a stencil on the CPU (with the stencil on the
GPU, p and wrk2 exchange roles and nothing is copied back) against the three
nest kernels, which per-nest timing keeps apart: p and the residuals are
bit-identical, and p is the float-store oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,iters", [((3, 3, 3), 3), ((4, 4, 4), 2), ((5, 7, 5), 4), ((5, 7, 9), 3),
                                         ((9, 10, 131), 3), ((18, 66, 34), 2), ((6, 40, 517), 2)])
def test_one_pass_equals_separate_nests(shape, iters):
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo
    pkg_build.build()
    I, J, K = shape
    ctx = oo.oo_create(0)
    try:
        out = []
        for timing, per_iteration in ((False, 1), (True, 3)):
            p, res = np.empty(I * J * K, np.float32), np.empty(iters)
            st = oo.oo_run_pattern(ctx, 0b111011, 1, oo.jacobi(I, J, K, iters, timing=timing), p, res)
            assert st["n_launches"] == 2 + per_iteration * iters
            out.append((p, res))
    finally:
        oo.oo_destroy(ctx)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    _, ref_p = oracle.jacobi_run(I, J, K, iters, mode=1)
    assert np.array_equal(out[0][0], ref_p.reshape(-1).astype(np.float32))
