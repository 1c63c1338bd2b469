"""Pixel setup: inverse noise, source and least noise variance over noise scales from 2^-200 to
2^200 (reciprocals near the ends of FP32's range and beyond them), and for polarised plans the
least eigenvalue where Gershgorin's bound is tight, loose (strong correlations) or useless, with
the minimum in the first, a middle and the last pixel.  One FP64 iteration agrees with the oracle
to its roundings (1e-10); tau to 1e-12 of the trigonometric eigenvalue's own accuracy."""
import numpy as np
import pytest

import oracle
import wf_inputs as gen
from gpu_util import T, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wf():
    import paper_1210_4931_gb300 as lib

    lib.load()
    return lib


@pytest.mark.parametrize("precision,log2scale,tol", [("fp64", -200, 1e-10), ("fp64", 200, 1e-10), ("mixed", -60, 2e-5),
                                                     ("mixed", 0, 2e-5), ("mixed", 60, 2e-5)])
def test_noise_scales(wf, precision, log2scale, tol):
    import torch

    nside, lmax = 8, 16
    P = gen.healpix_problem(nside, lmax, seed=gen.seed_for(2, 900))
    f = 2.0 ** log2scale
    rng = np.random.default_rng(17)
    nv = P["noise_var"] * f * rng.uniform(0.5, 2.0, P["noise_var"].size)
    cl = P["c_ell"] * f
    d = np.sqrt(f) * (oracle.synthesis(nside, lmax, lmax, P["a_signal"]) + P["noise"])
    basis = oracle.HealpixBasis(nside, lmax)
    obs = P["mask"] > 0
    nu = np.where(obs, 1.0 / nv, 0.0)
    tau = float(nv[obs].min())
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision=precision)
    wf.wf_set_schedule(plan, [3.0, 1.0])
    s = torch.empty(plan.npix, dtype=torch.float64, device="cuda")
    rep = wf.wf_solve(plan, T(d), T(nv), T(P["mask"]), T(cl), 1e-6, s)
    ref = oracle.messenger_solve(basis, nu * d, nu, basis.per_mode(cl), tau, replay=[(3.0, lmax), (1.0, lmax)], d=d)
    assert rep["tau"] == tau
    assert rel(s.cpu().numpy(), ref["s"]) < tol
    assert rep["chi2_over_ndof"] == pytest.approx(ref["chi2_final"] / ref["n_dof"], rel=100 * tol)
    plan.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("corr,scale,where", [(0.05, 1.0, 0), (0.9, 1.0, 311), (0.5, 1e-40, -1), (0.5, 1e40, 5)])
def test_polarised_least_eigenvalue(wf, precision, corr, scale, where):
    import torch

    nside, lmax = 8, 16
    npix = 12 * nside * nside
    rng = np.random.default_rng(23)
    B = rng.standard_normal((npix, 3, 3)) * np.array([1.0, corr, corr])[:, None]
    N = (B @ B.transpose(0, 2, 1) + np.eye(3)) * rng.uniform(2.0, 20.0, npix)[:, None, None]
    N[where] *= 1.5 / np.linalg.eigvalsh(N[where])[0]
    N *= scale
    mask = np.ones(npix, dtype=np.uint8)
    mask[7] = mask[40] = 0
    N[7] = np.nan
    tau = float(np.linalg.eigvalsh(N[mask > 0])[:, 0].min())
    N6 = np.stack([N[:, 0, 0], N[:, 1, 1], N[:, 2, 2], N[:, 0, 1], N[:, 0, 2], N[:, 1, 2]])
    C = np.zeros((4, lmax + 1))
    C[:3, 2:] = scale
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision=precision, ncomp=3)
    wf.wf_set_schedule(plan, [1.0])
    s = torch.empty(3 * npix, dtype=torch.float64, device="cuda")
    d = np.sqrt(scale) * rng.standard_normal((3, npix))
    args = (plan, T(d.ravel()), T(N6.ravel()), T(mask), T(C.ravel()), 1e-6, s)
    if precision == "mixed" and scale != 1.0:  # N^-1 does not fit FP32: refused as divergence
        with pytest.raises(wf.WfError) as e:
            wf.wf_solve(*args)
        assert e.value.status == wf.WF_EDIVERGE
    else:
        rep = wf.wf_solve(*args)
        assert rep["tau"] == pytest.approx(tau, rel=1e-12)
    plan.close()
