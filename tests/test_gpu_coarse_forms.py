"""Shapes of the coarsest-grid kernels and of the restriction where their splits
have edges: one to sixteen sites a CTA with ragged last CTAs, the grid-wide form
beyond one cluster's 256 sites, the FP64 apply's column groups, and vectors that
start on any entry.

* FP32 (tensor-core apply, FP16 operator) against the general kernel (FP32 FMAs on
  the same operator, deflation space and right-hand side): step counts within 2%
  (at least 2), solutions within 1e-4, the bound both keep against the oracle.
* FP64: the true residual with the handle's own stencil meets the tolerance.
* Restriction: against P^+ formed from the handle's prolongator in FP64, 2e-6
  (FP32) and 1e-12 (FP64) in the max norm, the bounds of the operator applies.
"""
import numpy as np
import pytest

import synth
from oracle import dirac
from gpu_util import dev, host, rel, rel2

pytestmark = pytest.mark.gpu

M0 = -0.03


@pytest.fixture(scope="module")
def mgmod(cuda_lib):
    import paper_1912_02868_gb300 as mg
    return mg


def _setup(mgmod, Lx, Lt, **params):
    U = synth.heatbath(Lx, Lt, 6.0, 60, 77 + Lx + 1000 * Lt)
    return mgmod.mg_setup(dev(U), Lx, Lt, M0, params=mgmod.default_params(seed=5, **params))


def _with_deflation(mgmod, Lx, Lt, **params):
    import torch
    g = _setup(mgmod, Lx, Lt, **params)
    b = dev(synth.complex_gaussian((Lt, Lx, 2), 9100, Lx, Lt))
    mgmod.mg_solve(g, b, torch.empty_like(b), 1, 1e-6)
    return g


# coarse sites: 1, 2, 15, 32 (2 a CTA), 42 (3), 72 (5, last 2), 247 (16, last 7), 272 and 399 (grid)
@pytest.mark.parametrize("Lx,Lt", [(16, 16), (32, 16), (80, 48), (128, 64), (96, 112), (144, 128), (208, 304),
                                   (272, 256), (336, 304)])
def test_coarse_tensor_forms(mgmod, Lx, Lt):
    import torch
    n2 = (Lx // 16) * (Lt // 16) * 24
    b = dev(synth.complex_gaussian((n2,), 9200, Lx, Lt), torch.complex64)
    got = {}
    for mma in (1, 0):
        g = _with_deflation(mgmod, Lx, Lt, precision=mgmod.MG_MIXED, coarse_mma=mma)
        try:
            x = torch.zeros_like(b)
            st, it, conv, info = mgmod.mg_coarse_solve(g, b, x, 1e-5, mgmod.MG_F32)
            y = torch.zeros_like(b)
            _, it2, _, _ = mgmod.mg_coarse_solve(g, b, y, 1e-5, mgmod.MG_F32)
        finally:
            g.close()
        assert conv[0] and info["timeouts"] == 0 and info["tensor_apply"] == mma
        assert it == it2 and torch.equal(x, y)  # the reductions' order is fixed
        got[mma] = (it[0], host(x))
    assert abs(got[1][0] - got[0][0]) <= max(2, 0.02 * got[0][0])
    assert rel2(got[1][1], got[0][1]) <= 1e-4


# sites a CTA 1, 2 (last 1), 3, 5 (last 2), 9: 20, 10, 6, 4 and 2 column groups
@pytest.mark.parametrize("Lx,Lt", [(80, 48), (80, 80), (96, 112), (144, 128), (192, 192)])
def test_coarse_fp64_groups(mgmod, Lx, Lt):
    import torch
    tol = 1e-10
    g = _with_deflation(mgmod, Lx, Lt)
    try:
        A = mgmod.mg_get_stencil(g, 2)
        nt, nx = A.shape[:2]
        b = synth.complex_gaussian((nt * nx * 24,), 9300, Lx, Lt)
        x = torch.zeros(b.size, dtype=torch.complex128, device="cuda")
        st, it, conv, info = mgmod.mg_coarse_solve(g, dev(b), x, tol, mgmod.MG_F64)
    finally:
        g.close()
    assert conv[0] and info["dataflow"] == 1 and info["timeouts"] == 0
    r = dirac.stencil_apply(A, host(x).reshape(nt, nx, 24)).ravel() - b
    assert np.linalg.norm(r) <= 1.05 * tol * np.linalg.norm(b)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("Lx,Lt", [(16, 16), (80, 48)])
def test_restriction_edges(mgmod, Lx, Lt, offset):
    import torch
    g = _setup(mgmod, Lx, Lt)
    try:
        for level in (0, 1):
            Q = mgmod.mg_get_prolongator(g, level)
            bt, bx, _, _, _, h = Q.shape
            v = synth.complex_gaussian((bt * 4, bx * 4, 2 * h), 9400 + level, Lx, Lt)
            w = v.reshape(bt, 4, bx, 4, 2, h).transpose(0, 2, 4, 1, 3, 5).reshape(bt, bx, 2, 16, h)
            want = np.einsum("xycjla,xycla->xycj", Q.conj(), w)
            for dt, prec, tol in ((torch.complex64, mgmod.MG_F32, 2e-6), (torch.complex128, mgmod.MG_F64, 1e-12)):
                buf = torch.zeros(v.size + offset, dtype=dt, device="cuda")
                fine = buf[offset:]  # offset 1: aligned to one entry only
                fine.copy_(dev(v).reshape(-1))
                out = torch.empty(want.size, dtype=dt, device="cuda")
                mgmod.mg_restrict(g, level, fine, out, precision=prec)
                assert rel(host(out), want) <= tol
    finally:
        g.close()
