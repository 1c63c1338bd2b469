"""Grids of short rings: quarter-ring lengths up to 8 take direct sums, 9 is the first FFT.  Band
limits at and below the ring lengths (one alias per bin) and at 2 nside (many), both directions,
against the oracle's direct sums; 1e-12 (some 10 roundings of FP64) and 2e-6 (of FP32) of the largest value."""
import numpy as np
import pytest

import oracle
import wf_inputs as gen
from gpu_util import T, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 2e-6)])
@pytest.mark.parametrize("nside,lmax,L", [(1, 2, 2), (2, 4, 4), (2, 2, 2), (3, 6, 5), (5, 10, 10), (7, 14, 3), (7, 14, 14),
                                          (8, 16, 16), (8, 9, 9), (9, 18, 18)])
def test_short_rings(nside, lmax, L, precision, tol):
    import torch

    import paper_1210_4931_gb300 as wf

    wf.load()
    rng = np.random.default_rng(4300 + 10 * nside + L)
    a = gen.alm_unit_gaussian(rng, lmax)
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision=precision)
    m = torch.empty(plan.npix, dtype=torch.float64, device="cuda")
    wf.wf_alm2map(plan, T(a), L, m)
    assert rel(m.cpu().numpy(), oracle.synthesis(nside, lmax, L, a)) < tol
    f = rng.standard_normal(plan.npix)
    b = torch.empty(plan.nalm, dtype=torch.complex128, device="cuda")
    wf.wf_map2alm_adjoint(plan, T(f), L, b)
    assert rel(b.cpu().numpy(), oracle.adjoint_synthesis(nside, lmax, L, f)) < tol
    plan.close()
