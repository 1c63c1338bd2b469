"""The two-step Legendre forms of the mixed plans (belt and polar cap, blocks of four k =
(l - m)/2) where they can go wrong: grids of one to a few ring pairs per part, band limits
that end on every remainder of the blocks and on both parities of l - m, FP64 blocks l < l_c
that end at every remainder of a block of four k, and every tile, in both directions against
the oracle.  Tolerance: the FP32 basis change's 2e-5 of the largest value."""
import numpy as np
import pytest

import oracle
import wf_inputs as gen
from gpu_util import T, rel

pytestmark = pytest.mark.gpu
TOL = 2e-5


@pytest.fixture(scope="module")
def wf():
    import paper_1210_4931_gb300 as lib

    lib.load()
    return lib


def _both_directions(wf, plan, nside, lmax, L, rng):
    import torch

    a = gen.alm_unit_gaussian(rng, lmax)
    m = torch.empty(plan.npix, dtype=torch.float64, device="cuda")
    wf.wf_alm2map(plan, T(a), L, m)
    assert rel(m.cpu().numpy(), oracle.synthesis(nside, lmax, L, a)) < TOL
    f = rng.standard_normal(plan.npix)
    b = torch.empty(plan.nalm, dtype=torch.complex128, device="cuda")
    for _ in range(2):  # the sums are cleared for the next call
        wf.wf_map2alm_adjoint(plan, T(f), L, b)
        assert rel(b.cpu().numpy(), oracle.adjoint_synthesis(nside, lmax, L, f)) < TOL


@pytest.mark.parametrize("nside,lmax", [(1, 2), (2, 4), (3, 5), (5, 10), (16, 31), (33, 66)])
def test_band_limits(wf, nside, lmax):
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision="mixed")
    for L in sorted({0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, lmax - 1, lmax}):
        if L <= lmax:
            _both_directions(wf, plan, nside, lmax, L, np.random.default_rng(60 + L))
    plan.close()


@pytest.mark.parametrize("lc", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 17, 40])
def test_fp64_block_ends(wf, lc):
    nside, lmax = 20, 40
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision="mixed")
    wf.wf_set_options(plan, mixed_lc=lc)
    for L in (lmax, lc, lc + 3):
        _both_directions(wf, plan, nside, lmax, min(L, lmax), np.random.default_rng(70 + lc))
    plan.close()


@pytest.mark.parametrize("tile", [2, 4, 8])
@pytest.mark.parametrize("nside,lmax", [(63, 126), (65, 100), (130, 131), (257, 64)])
def test_tiles_and_partial_groups(wf, nside, lmax, tile):
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision="mixed")
    wf.wf_set_options(plan, tile_syn=tile, tile_ana=tile, mixed_lc=5)
    _both_directions(wf, plan, nside, lmax, lmax, np.random.default_rng(80 + nside))
    plan.close()
