"""Polarised plans at the ends of the FP64 range: the least eigenvalue of noise blocks whose
entries are FP32 subnormals (FP64 plans take them; FP32 cannot bound them)."""
import numpy as np
import pytest

from gpu_util import T

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
