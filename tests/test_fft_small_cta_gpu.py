"""Transforms in small CTAs (calls with few columns) against the grouped
items, which always use full ones: the arithmetic of a column does not depend
on its CTA, so the results are the same bits; and against numpy's FFT within
the block's 1e-12."""
import numpy as np
import pytest
import torch

from paper_2011_03602_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log2n", list(range(1, 21)))
def test_small_ctas_equal_grouped_items(log2n):
    from paper_2011_03602_gb300 import oo
    n = 1 << log2n
    ctx = oo.oo_create(0, torch.cuda.Stream())
    try:
        for batch, direction in ((1, -1), (3, 1), (17, -1)):
            if batch * n > (1 << 20):
                continue
            x = synth.complex_normal(log2n * 100 + batch, batch * n).reshape(batch, n)
            dx = torch.from_numpy(x).cuda()
            one, many = torch.empty_like(dx), torch.empty_like(dx)
            torch.cuda.synchronize()
            oo.oo_fft_c128_dev(ctx, n, batch, direction, dx, one)
            b = oo.oo_batch_create(ctx, [dict(kind="fft", n=n, x=dx[i], X=many[i], dir=direction)
                                         for i in range(batch)])
            try:
                oo.oo_batch_run(ctx, b, 0)
                oo.oo_batch_check(ctx, b)
            finally:
                oo.oo_batch_destroy(b)
            assert torch.equal(torch.view_as_real(one), torch.view_as_real(many)), batch
            ref = np.fft.fft(x) if direction < 0 else np.fft.ifft(x)
            assert np.linalg.norm(one.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref), batch
    finally:
        oo.oo_destroy(ctx)
