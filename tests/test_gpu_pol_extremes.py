"""Polarised plans at the ends of the FP64 range: the least eigenvalue of noise blocks whose
entries are FP32 subnormals (FP64 plans take them; FP32 cannot bound them), and priors and noise
blocks whose 2 x 2 determinants are FP64 subnormals, so that 1 / det overflows where the quotient
by det does not."""
import numpy as np
import pytest

import wf_inputs as gen
from gpu_util import T, healpix_pol_case, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wf():
    import paper_1210_4931_gb300 as lib

    lib.load()
    return lib


def _worst_block(scale, rng):
    """(a, d, 1 - (a - d)) of a block [[a, d], [d, a]] whose least eigenvalue a - d lies below 1, while
    Gershgorin's bound of the scaled entries in FP32, less 1e-5 of the trace, lies above FP32(scale);
    where there is none, one that lies 1e-9 below."""
    f32 = np.float32
    a = rng.uniform(1.4, 1.6, 400000)
    below = 10.0 ** rng.uniform(-9, -0.5, a.size)
    d = a - (1.0 - below)
    fa, fd, fc = f32(a * scale), f32(d * scale), f32(1.6 * scale)
    bad = np.minimum(fa - fd, fc) - f32(1e-5) * (fa + fa + fc) > f32(scale)
    k = np.argmax(np.where(bad, below, -1.0)) if bad.any() else np.argmin(below)
    return a[k], d[k], below[k]


@pytest.mark.parametrize("scale", [1e-30, 1e-36, 1e-38, 1e-41, 1e-42, 1e-43, 1e-44, 1e-46])
def test_least_eigenvalue_of_tiny_blocks(wf, scale):
    """Every block but one has the least eigenvalue 1 x scale or more, the last pixel's a little
    less.  tau to 1e-12, the accuracy of the eigenvalue's closed form."""
    import torch

    nside, lmax = 256, 4  # more pixels than threads of the setup: the last are looked at last
    npix = 12 * nside * nside
    rng = np.random.default_rng(31)
    a, d, below = _worst_block(scale, rng)
    f = rng.uniform(2.0, 20.0, npix)
    f[:256] = 1.0
    one = np.array([1.5, 1.5, 1.6, 0.5, 0.0, 0.0])
    N6 = one[:, None] * f * scale
    N6[:, -1] = np.array([a, a, 1.6, d, 0.0, 0.0]) * scale
    tau = float(np.linalg.eigvalsh(np.array([[N6[0, -1], N6[3, -1], 0], [N6[3, -1], N6[1, -1], 0], [0, 0, N6[2, -1]]]) / scale)[0]) * scale
    assert tau < scale * (1.0 - 0.5 * below)
    C = np.zeros((4, lmax + 1))
    C[:3, 2:] = scale
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision="fp64", ncomp=3)
    wf.wf_set_schedule(plan, [1.0])
    s = torch.empty(3 * npix, dtype=torch.float64, device="cuda")
    dm = np.sqrt(scale) * rng.standard_normal((3, npix))
    rep = wf.wf_solve(plan, T(dm.ravel()), T(N6.ravel()), None, T(C.ravel()), 1e-6, s)
    assert rep["tau"] / scale == pytest.approx(tau / scale, rel=1e-12)
    plan.close()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-4)])
def test_prior_with_subnormal_determinants(wf, precision, tol):
    """A beam takes TT and EE of the highest l to 1e-155 each: those modes contribute 1e-155 of a
    map, the same as modes held at zero, and leave chi^2 and the residual finite."""
    import torch

    nside, lmax = 8, 16
    P, basis, d, nu, obs, N6, C4 = healpix_pol_case(nside, lmax, gen.seed_for(4, 77))
    npix = 12 * nside * nside
    out = {}
    for name, f in (("tiny", 1.0), ("zero", 0.0)):
        C = C4.copy()
        C[0, 11:], C[1, 11:], C[3, 11:] = 1e-155 * f, 3e-156 * f, 1e-156 * f
        if name == "tiny":
            det = C[0, 11:] * C[1, 11:] - C[3, 11:] ** 2
            assert np.all((det > 0) & (det < 1.0 / np.finfo(float).max))
        plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision=precision, ncomp=3)
        wf.wf_set_schedule(plan, [4.0, 1.0, 1.0])
        s = torch.empty(3 * npix, dtype=torch.float64, device="cuda")
        rep = wf.wf_solve(plan, T(d.ravel()), T(N6.ravel()), T(P["mask"]), T(C.ravel()), 1e-9, s, trace_cap=3)
        out[name] = s.cpu().numpy(), rep
        plan.close()
    assert rel(out["tiny"][0], out["zero"][0]) < tol
    rep = out["tiny"][1]
    assert np.all(np.isfinite(rep["chi2_trace"])) and np.isfinite(rep["final_residual"])
    assert rep["chi2_over_ndof"] == pytest.approx(out["zero"][1]["chi2_over_ndof"], rel=100 * tol)


def test_noise_blocks_with_subnormal_determinants(wf):
    """A few Q, U pixels with variances of 2^-515 (their determinants keep 44 bits, 6e-14) among
    ordinary ones: the first iteration's map, which these pixels alone make, against the oracle."""
    import torch

    from oracle.messenger_pol import messenger_solve_pol, pol_inverse_noise, pol_tau

    nside, lmax = 8, 16
    P, basis, d, _, _, N6, C4 = healpix_pol_case(nside, lmax, gen.seed_for(4, 78))
    npix = 12 * nside * nside
    mask = P["mask"].copy()
    few = np.array([0, 100, 500, npix - 1])
    mask[few] = 3
    N = P["noise_cov"].copy()
    N[few, 1, 1], N[few, 2, 2] = 2.0 ** -515, 1.5 * 2.0 ** -515
    N[few, 1, 2] = N[few, 2, 1] = 0.25 * 2.0 ** -515
    N6 = np.stack([N[:, 0, 0], N[:, 1, 1], N[:, 2, 2], N[:, 0, 1], N[:, 0, 2], N[:, 1, 2]])
    det = N6[1, few] * N6[2, few] - N6[5, few] ** 2
    assert np.all((det > 0) & (det < 1.0 / np.finfo(float).max))
    d = 1e-6 * d
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision="fp64", ncomp=3)
    wf.wf_set_schedule(plan, [1.0])
    s = torch.empty(3 * npix, dtype=torch.float64, device="cuda")
    rep = wf.wf_solve(plan, T(d.ravel()), T(N6.ravel()), T(mask), T(C4.ravel()), 1e-9, s, trace_cap=1)
    nu = pol_inverse_noise(N, mask)
    tau = pol_tau(N, mask)
    ref = messenger_solve_pol(basis, np.einsum("nij,jn->in", nu, d), nu, basis.per_mode(P["c_ell"]), tau,
                              replay=[(1.0, lmax)])
    assert rep["tau"] / 2.0 ** -515 == pytest.approx(tau / 2.0 ** -515, rel=1e-12)
    assert rel(s.cpu().numpy().reshape(3, npix), ref["s"]) < 1e-10
    assert np.isfinite(rep["final_residual"]) and np.isfinite(rep["chi2_over_ndof"])
    plan.close()
