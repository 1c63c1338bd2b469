"""FP64 Legendre transforms at the edges of their split: ring pairs just below, at and above a
warp (npairs = 2 nside) and 256 (two pairs per lane from there on in the analysis), band limits
around a table block of 32 l, a band limit below the plan's, both directions against the oracle
(1e-10 of the largest value, the FP64 bound of the other tests), and the analysis twice in a row
(its sums start from zero each time)."""
import numpy as np
import pytest

import oracle
import wf_inputs as gen
from gpu_util import T, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax,L", [(1, 2, 2), (2, 4, 3), (15, 30, 30), (16, 31, 31), (16, 32, 30), (17, 33, 33),
                                          (24, 48, 47), (33, 64, 64), (40, 80, 65), (64, 128, 128), (127, 33, 33),
                                          (128, 40, 39), (145, 60, 60)])
def test_fp64_legendre_edges(nside, lmax, L):
    import torch

    import paper_1210_4931_gb300 as wf

    wf.load()
    rng = np.random.default_rng(5000 + 100 * nside + L)
    a = gen.alm_unit_gaussian(rng, lmax)
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision="fp64")
    m = torch.empty(plan.npix, dtype=torch.float64, device="cuda")
    wf.wf_alm2map(plan, T(a), L, m)
    assert rel(m.cpu().numpy(), oracle.synthesis(nside, lmax, L, a)) < 1e-10
    x = rng.standard_normal(plan.npix)
    ref = oracle.adjoint_synthesis(nside, lmax, L, x)
    out = torch.full((plan.nalm,), float("nan"), dtype=torch.complex128, device="cuda")
    for _ in range(2):
        wf.wf_map2alm_adjoint(plan, T(x), L, out)
        assert rel(out.cpu().numpy(), ref) < 1e-10
    plan.close()
