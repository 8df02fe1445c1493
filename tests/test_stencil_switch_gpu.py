"""Sweeps on the caller's arrays that change arrays and grid from call to call
share one scratch of the context, ordered by its stream: queued one after
another without waiting they must give what each gives alone, bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(12, 19, 70), (40, 37, 200), (6, 40, 517), (3, 3, 3)]


def arrays(oo, synth, shape, seed):
    I, J, K = shape
    pitch = oo.oo_jacobi_pitch(K)

    def pad(a):
        t = torch.zeros((I, J, pitch), dtype=torch.float32, device="cuda")
        t[:, :, :K] = torch.from_numpy(np.ascontiguousarray(a)).cuda()
        return t

    coef = [pad(synth.field(seed + a, shape, -1.0, 1.0)) for a in range(12)]
    return pitch, coef, pad(synth.field(seed + 20, shape, 0.0, 1.0))


def test_queued_sweeps_equal_single_ones():
    from paper_2011_03602_gb300 import build as pkg_build
    from paper_2011_03602_gb300 import oo, synth
    pkg_build.build()
    sets = [(s, *arrays(oo, synth, s, 100 * i)) for i, s in enumerate(SHAPES + SHAPES[:1])]
    out = []
    for alone in (True, False):
        ctx = oo.oo_create(0)
        got = []
        try:
            for rep in range(1 if alone else 3):
                for (I, J, K), pitch, coef, p in sets:
                    w = torch.zeros((I, J, pitch), dtype=torch.float32, device="cuda")
                    r = torch.zeros(1, dtype=torch.float64, device="cuda")
                    got.append((w, r))
            torch.cuda.synchronize()
            for n, (w, r) in enumerate(got):
                (I, J, K), pitch, coef, p = sets[n % len(sets)]
                oo.oo_stencil_dev(ctx, I, J, K, pitch, coef, p, 0.8, w, r)
                if alone:
                    oo.oo_stencil_check(ctx)
            oo.oo_stencil_check(ctx)
            out.append([(w.cpu().numpy(), r.item()) for w, r in got])
        finally:
            oo.oo_destroy(ctx)
    for n, (w, r) in enumerate(out[1]):
        assert np.array_equal(w, out[0][n % len(sets)][0]) and r == out[0][n % len(sets)][1], n
