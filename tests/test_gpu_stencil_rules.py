"""The intermediate stencil at the sizes where its kernels change: FP32 hop factors staged in
shared memory (few sites an SM, or an operator larger than L2) or loaded where they are used,
FP64 one CTA a site or blocks of eight, factored and dense.  Against the dense blocks of
mg_get_stencil in FP64, max norm 2e-6 (FP32) and 1e-12 (FP64), the bounds of the operator
applies; D and D^+.
"""
import pytest

import synth
from gpu_util import dev

pytestmark = pytest.mark.gpu


def _apply(A, x, dagger):
    """D x (D^+ x) from the dense blocks [t][x][5][k][l], in FP64 on the GPU."""
    import torch
    sign = torch.ones(24, dtype=torch.float64, device="cuda")
    if dagger:
        sign[12:] = -1.0
    v = x * sign
    y = torch.zeros_like(v)
    for d, nb in enumerate((v, torch.roll(v, -1, 1), torch.roll(v, 1, 1), torch.roll(v, -1, 0), torch.roll(v, 1, 0))):
        y += torch.einsum("txkl,txl->txk", A[:, :, d], nb)
    return y * sign


# sites (a GB300 has 152 SMs): 16, 1728 and 1920 (FP32: staged to 12 an SM, 1824), 10000 and 10400
# (107.5 and 111.8 MB of FP32 factors); FP64, sites an SM: 864 (6), 1024 (7), 1152 (8), 1600 (11),
# 1760 (12), 2112 (14), 2304 (16)
@pytest.mark.parametrize("nx,nt", [(4, 4), (36, 48), (40, 48), (100, 100), (104, 100), (36, 24), (32, 32), (32, 36),
                                   (40, 40), (40, 44), (44, 48), (48, 48)])
def test_kernel_boundaries(cuda_lib, nx, nt):
    import torch
    import paper_1912_02868_gb300 as mg
    Lx, Lt = 4 * nx, 4 * nt
    U = dev(synth.heatbath(Lx, Lt, 6.0, 20, 79 + Lx + 1000 * Lt))
    nv = [dev(synth.complex_gaussian((12, Lt, Lx, 2), 9800, Lx, Lt)), dev(synth.complex_gaussian((12, nt, nx, 24), 9801, Lx, Lt))]
    for lowrank in (1, 0):
        p = mg.default_params(precision=mg.MG_MIXED, lowrank_hops=lowrank)
        g = mg.mg_setup_from_vectors(U, Lx, Lt, -0.03, *nv, params=p)
        try:
            assert bool(mg.mg_stencil_info(g, 1)[0]) == bool(lowrank)
            A = torch.from_numpy(mg.mg_get_stencil(g, 1)).cuda()
            x = dev(synth.complex_gaussian((nt, nx, 24), 9802, Lx, Lt))
            for dagger in (False, True):
                for dt, prec, tol in ((torch.complex128, mg.MG_F64, 1e-12), (torch.complex64, mg.MG_F32, 2e-6)):
                    xs = x.to(dt)
                    want = _apply(A, xs.to(torch.complex128), dagger)
                    y = torch.empty_like(xs)
                    mg.mg_apply(g, 1, xs, y, dagger=dagger, precision=prec)
                    err = (y.to(torch.complex128) - want).abs().max() / want.abs().max()
                    assert float(err) <= tol
        finally:
            g.close()
