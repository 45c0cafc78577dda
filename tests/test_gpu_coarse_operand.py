"""Coarse solves on tensor cores, in one cluster and over the whole GPU: the vector enters the
apply with at least 22 bits of its entries, small ones beside large ones too.

One GMRES cycle of two steps (m - k = 2, one cycle) on a right-hand side of one entry of 1 and
entries of about 2^-24 elsewhere, with a deflation space on three other entries of that site.
Away from it x is d_0 v_0 + d_1 v_1, v_1 proportional to (A - h) v_0: it shows the small
entries' own error.  Against the general kernel (FP32 FMAs on the same FP16 operator): both
round a sum of 240 products in FP32, about 3e-7 of its size each, and the operand's 22 bits
are 1.2e-7: with the dozen operations around them below 2e-6.  An operand of two FP16 parts
on one scale keeps 2^-35, about 5e-4 of these entries.
"""
import numpy as np
import pytest

import synth
from gpu_util import dev, host, rel2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Lt", [(128, 64), (192, 192), (256, 256), (272, 256), (640, 512)])
def test_small_entries_keep_their_bits(cuda_lib, Lx, Lt):
    import torch
    import paper_1912_02868_gb300 as mg
    nx, nt = Lx // 16, Lt // 16
    U = synth.heatbath(Lx, Lt, 6.0, 60, 77 + Lx + 1000 * Lt)
    nv = [dev(synth.complex_gaussian((12, Lt, Lx, 2), 9600, Lx, Lt)),
          dev(synth.complex_gaussian((12, Lt // 4, Lx // 4, 24), 9601, Lx, Lt))]
    big = 3 * nx + 5  # site (5, 3)
    W = np.zeros((3, nt * nx, 24), complex)
    for i in range(3):
        W[i, big, i] = 1.0
    f = 2.0 ** -24 * synth.complex_gaussian((nt * nx, 24), 9602, Lx, Lt)
    f[big] = 0.0
    f[big, 5] = 1.0
    far = np.array([min(abs(s % nx - 5), nx - abs(s % nx - 5)) + min(abs(s // nx - 3), nt - abs(s // nx - 3)) > 2
                    for s in range(nt * nx)])
    got = {}
    for mma in (1, 0):
        p = mg.default_params(precision=mg.MG_MIXED, coarse_mma=mma, dr_m=4, dr_k=2, proj_max_cycles=1)
        g = mg.mg_setup_from_vectors(dev(U), Lx, Lt, -0.03, *nv, params=p)
        try:
            mg.mg_set_deflation(g, W.reshape(3, -1), np.eye(3, 2, dtype=complex))
            b = dev(f.reshape(-1), torch.complex64)
            x = torch.zeros_like(b)
            _, it, _, info = mg.mg_coarse_solve(g, b, x, 1e-5, mg.MG_F32)
        finally:
            g.close()
        assert it[0] == 2 and info["timeouts"] == 0 and info["tensor_apply"] == mma
        got[mma] = host(x).reshape(nt * nx, 24).astype(np.complex128)
    assert np.isfinite(got[1]).all()
    # the second step counts: x is not just a multiple of f there
    y = got[0][far].ravel()
    v = f[far].ravel()
    assert rel2(v * (np.vdot(v, y) / np.vdot(v, v)), y) > 1e-2
    assert rel2(got[1][far], got[0][far]) <= 2e-6
