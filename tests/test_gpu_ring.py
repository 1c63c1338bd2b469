"""Ring DFTs at the edges of their FFT lengths: every quarter-ring length k of the polar
caps up to nside, and belts whose k = nside just passes a power of two (Bluestein of
length 32 to 4096) or is one (direct FFTs), against the oracle's direct sums, both
directions.  Small band limits keep the oracle's sums cheap; lmax = 2 nside (rings shorter
than the band limit, many aliases per bin) runs on the small grids.  Tolerances as in the
full-size tests' FP64 (1e-10 of the largest value) and the FP32 basis change (2e-5)."""
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


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 2e-5)])
@pytest.mark.parametrize("nside,lmax", [(3, 6), (9, 18), (16, 32), (17, 34), (33, 66), (65, 130), (130, 40), (257, 40),
                                        (256, 300), (520, 24), (1024, 16), (1030, 16)])
def test_ring_lengths_at_fft_edges(wf, nside, lmax, precision, tol):
    import torch

    rng = np.random.default_rng(4000 + nside)
    a = gen.alm_unit_gaussian(rng, lmax)
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision=precision)
    m = torch.empty(plan.npix, dtype=torch.float64, device="cuda")
    wf.wf_alm2map(plan, T(a), lmax, m)
    got = m.cpu().numpy()
    if nside < 300:
        assert rel(got, oracle.synthesis(nside, lmax, lmax, a)) < tol
    else:  # sampled rings: the first and last of each cap FFT length, the belt's ends, the equator
        off = np.concatenate([[0], np.cumsum(gen.ring_layout(nside)[2])])
        ks = sorted({1, nside - 1, nside, nside + 1, 2 * nside} | {k for b in range(2, 11) for k in (1 << b, (1 << b) + 1)
                                                                  if k < nside})
        for r in [k - 1 for k in ks] + [4 * nside - 1 - nside // 3, 4 * nside - 2]:
            sl = slice(off[r], off[r + 1])
            ref = oracle.synthesis(nside, lmax, lmax, a, rings=(r, r + 1))[sl]
            assert rel(got[sl], ref) < tol, r
    f = rng.standard_normal(plan.npix) + got
    b = torch.empty(plan.nalm, dtype=torch.complex128, device="cuda")
    wf.wf_map2alm_adjoint(plan, T(f), lmax, b)
    assert rel(b.cpu().numpy(), oracle.adjoint_synthesis(nside, lmax, lmax, f)) < tol
    plan.close()
