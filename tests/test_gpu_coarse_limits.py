"""The tensor-core form of the coarsest-grid solve at the ends of what it takes, in one
cluster (64^2) and over the whole GPU (272 x 256: more than 256 coarse sites).

* Right-hand sides whose squared norm leaves FP32's range (it overflows at entries of 1e22,
  and is zero at entries of 1e-30 and at zero): the solve ends with the projection onto the
  deflation space, as the general kernel (coarse_mma = 0) does, to the 1e-4 that both keep
  against the oracle.
* A bounded wait that gives up (the probe: nothing ends it) makes the call return MG_ETIMEOUT
  with every CTA counted, and the next solve is bitwise the one before the probe.
"""
import numpy as np
import pytest

import synth
from gpu_util import dev, host, rel2

pytestmark = pytest.mark.gpu

SIZES = [(64, 64), (272, 256)]


@pytest.fixture(scope="module")
def mgmod(cuda_lib):
    import paper_1912_02868_gb300 as mg
    return mg


def _handle(mgmod, Lx, Lt, **params):
    import torch
    U = synth.heatbath(Lx, Lt, 6.0, 60, 77 + Lx + 1000 * Lt)
    g = mgmod.mg_setup(dev(U), Lx, Lt, -0.03, params=mgmod.default_params(seed=5, precision=mgmod.MG_MIXED, **params))
    b = dev(synth.complex_gaussian((Lt, Lx, 2), 9100, Lx, Lt))
    mgmod.mg_solve(g, b, torch.empty_like(b), 1, 1e-6)
    return g


def _rhs(Lx, Lt, scale=1.0):
    import torch
    return dev(scale * synth.complex_gaussian(((Lx // 16) * (Lt // 16) * 24,), 9200, Lx, Lt), torch.complex64)


@pytest.mark.parametrize("Lx,Lt", SIZES)
def test_norms_beyond_fp32(mgmod, Lx, Lt):
    import torch
    got = {}
    for mma in (1, 0):
        g = _handle(mgmod, Lx, Lt, coarse_mma=mma)
        try:
            for scale in (1e22, 1e-30, 0.0):
                b = _rhs(Lx, Lt, scale)
                x = torch.zeros_like(b)
                _, it, conv, info = mgmod.mg_coarse_solve(g, b, x, 1e-5, mgmod.MG_F32)
                assert info["tensor_apply"] == mma and info["timeouts"] == 0
                got[mma, scale] = (it[0], conv[0], host(x).astype(np.complex128))
        finally:
            g.close()
    for scale in (1e22, 1e-30, 0.0):
        (it1, conv1, x1), (it0, conv0, x0) = got[1, scale], got[0, scale]
        assert (it1, conv1) == (it0, conv0) == (0, True)
        assert np.isfinite(x1).all() and rel2(x1, x0) <= 1e-4


@pytest.mark.parametrize("Lx,Lt", SIZES)
def test_probe_gives_up(mgmod, Lx, Lt):
    import torch
    g = _handle(mgmod, Lx, Lt)
    try:
        b = _rhs(Lx, Lt)
        x, y, z = (torch.zeros_like(b) for _ in range(3))
        _, it, conv, info = mgmod.mg_coarse_solve(g, b, x, 1e-5, mgmod.MG_F32)
        assert conv[0] and info["tensor_apply"] == 1 and info["timeouts"] == 0
        st, _, _, info = mgmod.mg_coarse_solve(g, b, y, 1e-5, mgmod.MG_F32, flags=mgmod.MG_COARSE_PROBE_TIMEOUT,
                                               spin=64, allow=(mgmod.MG_OK, mgmod.MG_ETIMEOUT))
        assert st == mgmod.MG_ETIMEOUT and info["timeouts"] == info["ctas"] >= 16
        _, it2, conv2, info = mgmod.mg_coarse_solve(g, b, z, 1e-5, mgmod.MG_F32)
        assert it2 == it and conv2[0] and info["timeouts"] == 0 and torch.equal(x, z)
    finally:
        g.close()
