"""Runs in which p and wrk2 exchange roles (every iteration nest on the GPU, no
copy in the loop): the cooperative all-iterations kernel and the per-iteration
sweeps against each other at the sizes where their work splits change.  Both
use the same float-float arithmetic per point, so p is bit-identical; the
residuals differ in summation order only: a float-float sum of n terms is
within n 2^-47 of them, and the longest run of terms here is below 2000, so
2000 * 2^-47 = 1.4e-11 bounds the difference."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def oo_mod():
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo
    pkg_build.build()
    return oo


def run(oo, shape, iters, fused):
    I, J, K = shape
    ctx = oo.oo_create(0)
    try:
        oo.oo_set_option(ctx, oo.OO_OPT_JACOBI_FUSED, fused)
        p, res = np.empty(I * J * K, np.float32), np.empty(iters)
        st = oo.oo_run_pattern(ctx, 63, 1, oo.jacobi(I, J, K, iters), p, res)
        assert st["n_launches"] == (3 if fused else 2 + 2 * iters)
        return p, res
    finally:
        oo.oo_destroy(ctx)


@pytest.mark.parametrize("shape,iters", [
    # iterations around the residual chunks of the cooperative kernel (64)
    ((7, 8, 9), 1), ((7, 8, 9), 63), ((7, 8, 9), 64), ((7, 8, 9), 65), ((7, 8, 9), 129),
    # fewer points than CTAs x 256, one CTA, rows shorter and longer than a CTA's threads
    ((3, 3, 3), 5), ((3, 3, 1200), 4), ((40, 3, 3), 4), ((9, 40, 517), 3),
    # a CTA's points within and beyond its shared-memory coefficients
    ((90, 90, 92), 3), ((91, 93, 97), 3),
    # several i slabs of the sweeps (p above 80 MB), ranges crossing columns
    ((211, 301, 322), 3), ((150, 5, 131), 3)])
def test_exchanged_runs_agree(oo_mod, shape, iters):
    one, many = run(oo_mod, shape, iters, 1), run(oo_mod, shape, iters, 0)
    assert np.array_equal(one[0], many[0])
    assert np.all(np.abs(one[1] - many[1]) <= 1.4e-11 * np.abs(many[1]))
