"""A time-out of an earlier sweep outlasts the sweeps queued behind it: with
the next sweep on other arrays, or on another grid, oo_stencil_check still
reports it (once), and the sweeps behind it are whole."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def arrays(oo, synth, shape, seed):
    I, J, K = shape
    pitch = oo.oo_jacobi_pitch(K)

    def pad(a):
        t = torch.zeros((I, J, pitch), dtype=torch.float32, device="cuda")
        t[:, :, :K] = torch.from_numpy(np.ascontiguousarray(a)).cuda()
        return t

    coef = [pad(synth.field(seed + a, shape, -1.0, 1.0)) for a in range(12)]
    p = pad(synth.field(seed + 20, shape, 0.0, 1.0))
    return pitch, coef, p, torch.zeros_like(p), torch.zeros(1, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("second", [(12, 19, 70), (40, 37, 200), (3, 3, 3)])
def test_earlier_time_out_is_reported(second):
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo, synth
    pkg_build.build()
    first = (12, 19, 70)
    a, b = arrays(oo, synth, first, 100), arrays(oo, synth, second, 200)
    torch.cuda.synchronize()
    ctx = oo.oo_create(0)

    def sweep(shape, s):
        oo.oo_stencil_dev(ctx, *shape, s[0], s[1], s[2], 0.8, s[3], s[4])

    try:
        sweep(second, b)
        oo.oo_stencil_check(ctx)
        want = (b[3].clone(), b[4].item())
        b[3].zero_()
        torch.cuda.synchronize()
        oo.oo_inject_wait_timeout(ctx, oo.OO_INJECT_STENCIL_LOAD)
        sweep(first, a)
        sweep(second, b)
        with pytest.raises(oo.OOError) as e:
            oo.oo_stencil_check(ctx)
        assert e.value.status == oo.OO_ETIMEOUT
        assert torch.equal(b[3], want[0]) and b[4].item() == want[1]
        oo.oo_stencil_check(ctx)  # reported once
        sweep(first, a)
        oo.oo_stencil_check(ctx)
    finally:
        oo.oo_destroy(ctx)
