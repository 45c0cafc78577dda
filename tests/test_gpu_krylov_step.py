"""The fused Krylov-step kernels at the edges of their shapes: one to sixteen CTAs, one
to sixteen entries a thread, and vectors beyond their largest sizes (FP32 131072
entries, FP64 16384), which take the separate kernels.

A mixed solve (FP32 smoothers) and an FP64 solve of one hierarchy: the true residual
meets the tolerance (1.0001: its own rounding), and the outer counts agree within one,
as the two paths do at every size they share."""
import numpy as np
import pytest

import synth
from oracle import dirac
from gpu_util import dev, host

pytestmark = pytest.mark.gpu

M0 = -0.03
TOL = 1e-10


# fine entries: 512, 7680, 15360, 16896, 32768, 131072, 139264; intermediate: 384 to 104448
@pytest.mark.parametrize("Lx,Lt", [(16, 16), (80, 48), (96, 80), (176, 48), (128, 128), (256, 256), (256, 272)])
def test_krylov_step_shapes(cuda_lib, Lx, Lt):
    import torch
    import paper_1912_02868_gb300 as mg
    U = synth.heatbath(Lx, Lt, 6.0, 60, 79 + Lx + 1000 * Lt)
    b = synth.complex_gaussian((2, Lt, Lx, 2), 9600, Lx, Lt)
    outer = []
    for prec in (mg.MG_FP64, mg.MG_MIXED):
        g = mg.mg_setup(dev(U), Lx, Lt, M0, params=mg.default_params(seed=5, precision=prec))
        try:
            x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
            _, it, _, _ = mg.mg_solve(g, dev(b), x, 2, TOL)
        finally:
            g.close()
        xv = host(x)
        for i in range(2):
            r = np.linalg.norm(dirac.wilson(U, xv[i], M0) - b[i]) / np.linalg.norm(b[i])
            assert r <= 1.0001 * TOL
        outer.append(it)
    assert all(abs(a - c) <= 1 for a, c in zip(*outer))
