"""Concurrent mixed solves beyond 256 coarse sites: the form of the coarsest solve by the
number of solves that run at once (mg_params.parallel).

380 sites: grids of eight sites a CTA (48 CTAs) while they all fit on the GPU's SMs, then of
16 (24 CTAs), and clusters of 16 CTAs with FP32 FMAs for more solves than grids that fit.
Each right-hand side meets its tolerance, repeats bit for bit, alone and beside the others,
and solutions of different forms agree to the tolerance that both keep (1e-10 on the
residual, M0 leaves a condition number below 1e4).
"""
import numpy as np
import pytest

import synth
from gpu_util import dev, host, rel2
from oracle import dirac

pytestmark = pytest.mark.gpu

LX, LT, M0, TOL = 320, 304, -0.03, 1e-10


def test_forms_by_concurrent_solves(cuda_lib):
    import torch
    import paper_1912_02868_gb300 as mg
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    U = synth.heatbath(LX, LT, 6.0, 60, 77 + LX + 1000 * LT)
    n2 = (LX // 16) * (LT // 16) * 24
    c = dev(synth.complex_gaussian((n2,), 9700, LX, LT), torch.complex64)
    B = synth.complex_gaussian((8, LT, LX, 2), 9701, LX, LT)
    grids = {8: 48, 16: 24}
    many = sms // grids[16] + 1
    sol, low = {}, {}
    for par in (1, sms // grids[8], sms // grids[8] + 1, many):
        g = mg.mg_setup(dev(U), LX, LT, M0, params=mg.default_params(seed=5, precision=mg.MG_MIXED, parallel=par))
        try:
            x0 = torch.empty((1, LT, LX, 2), dtype=torch.complex128, device="cuda")
            mg.mg_solve(g, dev(B[:1]), x0, 1, 1e-6)
            y = torch.zeros_like(c)
            _, _, conv, info = mg.mg_coarse_solve(g, c, y, 1e-5, mg.MG_F32)
            assert conv[0] and info["timeouts"] == 0
            if par < many:
                assert info["tensor_apply"] == 1 and info["ctas"] * par <= sms
                assert info["ctas"] == grids[8 if grids[8] * par <= sms else 16]
            else:
                assert info["tensor_apply"] == 0 and info["ctas"] <= 16
            low[par] = host(y)
            X, Y, Z = (torch.empty(B.shape, dtype=torch.complex128, device="cuda") for _ in range(3))
            _, it, rr, _ = mg.mg_solve(g, dev(B), X, len(B), TOL)
            _, it2, _, _ = mg.mg_solve(g, dev(B), Y, len(B), TOL)
            for i in range(len(B)):
                mg.mg_solve(g, dev(B[i:i + 1]), Z[i:i + 1], 1, TOL)
            assert max(rr) <= TOL and it == it2 and torch.equal(X, Y) and torch.equal(X, Z)
            sol[par] = host(X)
        finally:
            g.close()
    r = dirac.wilson(U, sol[1][3], M0) - B[3]
    assert np.linalg.norm(r) <= 1.0001 * TOL * np.linalg.norm(B[3])
    for par in sol:
        assert rel2(low[par], low[1]) <= 1e-4 and rel2(sol[par], sol[1]) <= 1e4 * TOL
