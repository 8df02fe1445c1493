"""The tile-width autotuner where two widths are the same launch (the level
schemes run 128-wide entries as 64-wide tiles): their times are one number, and
the choice between them is the built-in table's, not the noise's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_one_launch_is_timed_once():
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo
    pkg_build.build()
    ctx = oo.oo_create(0)
    try:
        builtin = oo.oo_get_gemm_tiles(ctx).copy()
        widths, ms = oo.oo_tune_gemm_tiles(ctx)
        assert np.array_equal(oo.oo_get_gemm_tiles(ctx), widths)
    finally:
        oo.oo_destroy(ctx)
    builtin, widths, ms = builtin.reshape(6, 5), widths.reshape(6, 5), ms.reshape(6, 5, 3)
    assert np.all(ms > 0)
    assert np.array_equal(ms[:, :4, 2], ms[:, :4, 1])  # k <= 512
    wide = np.maximum(64, builtin[:, :4])
    assert np.array_equal(widths[:, :4], np.where(ms[:, :4, 1] < ms[:, :4, 0], wide, 32))
