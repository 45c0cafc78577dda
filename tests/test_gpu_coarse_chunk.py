"""Batched coarse GMRES-Proj at the sizes where its split into site chunks and
tiles of eight right-hand sides has edges: chunks of 4, 8, 14 and 16 sites with
ragged last ones, one chunk only, more than 32 chunks, one to eight tiles, the
last tile ragged.

Each right-hand side against the single-right-hand-side kernel on the same FP16
operator and deflation space: step counts within 2% (at least 2), solutions within
2e-4 (both keep 1e-4 against the oracle).  A second run gives the same bits.
"""
import pytest

import synth
from gpu_util import dev, host, rel2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mgmod(cuda_lib):
    import paper_1912_02868_gb300 as mg
    return mg


# coarse sites and right-hand sides: 1 x 3, 15 x 5 (chunks of 4, last 3), 42 x 16 (4, last 2),
# 247 x 20 (8, last 7), 256 x 64 (14, last 4), 399 x 48 (16, last 15), 1024 x 9 (74 chunks)
@pytest.mark.parametrize("Lx,Lt,nrhs", [(16, 16, 3), (80, 48, 5), (96, 112, 16), (208, 304, 20), (256, 256, 64),
                                        (336, 304, 48), (512, 512, 9)])
def test_chunked_cycle_against_single(mgmod, Lx, Lt, nrhs):
    import torch
    n2 = (Lx // 16) * (Lt // 16) * 24
    U = synth.heatbath(Lx, Lt, 6.0, 60, 77 + Lx + 1000 * Lt)
    g = mgmod.mg_setup(dev(U), Lx, Lt, -0.03, params=mgmod.default_params(seed=5, precision=mgmod.MG_MIXED))
    try:
        f = dev(synth.complex_gaussian((Lt, Lx, 2), 9100, Lx, Lt))
        mgmod.mg_solve(g, f, torch.empty_like(f), 1, 1e-6)
        b = dev(synth.complex_gaussian((nrhs, n2), 9500, Lx, Lt), torch.complex64)
        x, y = torch.zeros_like(b), torch.zeros_like(b)
        _, it, conv, info = mgmod.mg_coarse_solve(g, b, x, 1e-5, mgmod.MG_F16, nrhs=nrhs)
        _, it2, _, _ = mgmod.mg_coarse_solve(g, b, y, 1e-5, mgmod.MG_F16, nrhs=nrhs)
        assert all(conv) and info["timeouts"] == 0
        assert it == it2 and torch.equal(x, y)  # the sums' order is fixed
        for r in {0, nrhs // 2, nrhs - 1}:
            z = torch.zeros_like(b[r])
            _, it1, conv1, _ = mgmod.mg_coarse_solve(g, b[r].contiguous(), z, 1e-5, mgmod.MG_F32)
            assert conv1[0] and abs(it[r] - it1[0]) <= max(2, 0.02 * it1[0])
            assert rel2(host(x[r]), host(z)) <= 2e-4
    finally:
        g.close()
