"""Mixed temperature solves up to nside 256 repeat bit for bit: each sum of the analysis has at
most two addends in no fixed order (two groups of ring pairs), the others one order."""
import numpy as np
import pytest

import wf_inputs as gen
from gpu_util import T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax", [(64, 128), (129, 200), (160, 320), (192, 384), (227, 454), (256, 512), (256, 300)])
@pytest.mark.parametrize("precision", ["mixed", "tf32"])
def test_repeated_solve_is_identical(nside, lmax, precision):
    import torch

    import paper_1210_4931_gb300 as wf

    wf.load()
    npix = 12 * nside * nside
    rng = np.random.default_rng(41)
    cl = gen.cmb_like_cl(lmax, 4 * 3438.0 / lmax)
    nv = 0.05 * cl.max() * rng.uniform(0.5, 50.0, npix)
    d = T(rng.standard_normal(npix) * np.sqrt(nv))
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision=precision)
    lam, L = [9.0, 4.0, 2.0, 1.0, 1.0], [lmax // 3, lmax // 2, lmax, lmax, lmax]
    wf.wf_set_schedule(plan, lam, L)
    s = torch.empty(npix, dtype=torch.float64, device="cuda")
    a = torch.empty(plan.nalm, dtype=torch.complex128, device="cuda")
    first = None
    for _ in range(4):
        rep = wf.wf_solve(plan, d, T(nv), None, T(cl), 1e-12, s, a, trace_cap=8)
        got = (s.clone(), a.clone(), np.array(rep["chi2_trace"]), rep["final_residual"])
        if first is None:
            first = got
            continue
        assert torch.equal(got[0], first[0]) and torch.equal(got[1], first[1])
        np.testing.assert_array_equal(got[2], first[2])
        assert got[3] == first[3]
    plan.close()
