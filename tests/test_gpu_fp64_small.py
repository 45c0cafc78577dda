"""FP64 stencils of grids below and at the size where a CTA takes one site (2048 sites),
dense and with rank-4 hop factors: D and D^+ against the stencil blocks in numpy, 1e-12
relative in the max norm, the bound of the FP64 operator applies."""
import numpy as np
import pytest

import synth
from oracle import dirac
from gpu_util import dev, host, rel

pytestmark = pytest.mark.gpu


# intermediate sites: 16, 240, 1920, 2048; coarsest: 1, 15, 120, 128
@pytest.mark.parametrize("Lx,Lt", [(16, 16), (80, 48), (128, 240), (128, 256)])
@pytest.mark.parametrize("lowrank", [0, 1])
def test_fp64_stencils(cuda_lib, Lx, Lt, lowrank):
    import torch
    import paper_1912_02868_gb300 as mg
    U = synth.heatbath(Lx, Lt, 6.0, 10, 78 + Lx + 1000 * Lt)
    v0 = synth.complex_gaussian((12, Lt, Lx, 2), 9500, Lx, Lt)
    v1 = synth.complex_gaussian((12, Lt // 4, Lx // 4, 24), 9501, Lx, Lt)
    g = mg.mg_setup_from_vectors(dev(U), Lx, Lt, -0.03, dev(v0), dev(v1),
                                 params=mg.default_params(lowrank_hops=lowrank))
    try:
        for level in (1, 2):
            A = mg.mg_get_stencil(g, level)
            v = synth.complex_gaussian(A.shape[:2] + (24,), 9502 + level, Lx, Lt)
            sign = np.where(np.arange(24) < 12, 1.0, -1.0)
            for dagger in (False, True):
                want = dirac.stencil_apply(A, v * sign) * sign if dagger else dirac.stencil_apply(A, v)
                y = torch.empty(v.shape, dtype=torch.complex128, device="cuda")
                mg.mg_apply(g, level, dev(v), y, dagger=dagger, precision=mg.MG_F64)
                assert rel(host(y), want) <= 1e-12
    finally:
        g.close()
