"""Flat-grid solve with a prior that falls to 1e-307 at the highest wavenumbers (a Gaussian beam):
1/S is still an FP64 number, so chi^2 and the residual are too.  Against the oracle; 1e-10 for
what is made of the map, 1e-6 for the residual of the last iterate (differences of close values)."""
import numpy as np
import pytest

import oracle
import wf_inputs as gen
from gpu_util import T, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 32, 128])
def test_prior_down_to_the_least_normal_numbers(n):
    import torch

    import paper_1210_4931_gb300 as wf

    wf.load()
    P = gen.flat_problem(n, seed=gen.seed_for(1, 160 + n), band_rows=(n // 2 - 2, n // 2 + 2), n_disks=3,
                         disk_radius=2.0)
    k = gen.flat_kabs(n, n)
    S = P["S"] * np.exp(-707.0 * (k / k.max()) ** 2) / P["S"].min()
    assert 5e-308 < S.min() < 1e-306
    B = oracle.FlatBasis(n, n)
    nu = np.where(P["mask"] > 0, 1.0 / P["noise_var"], 0.0)
    tau = float(P["noise_var"][P["mask"] > 0].min())
    d = B.synth(P["a_signal"]) + P["noise"]
    plan = wf.wf_plan_create("flat", n=n)
    s = torch.empty(n * n, dtype=torch.float64, device="cuda")
    lam = [100.0, 7.0, 1.0, 1.0, 1.0]
    wf.wf_set_schedule(plan, lam)
    rep = wf.wf_solve(plan, T(d.ravel()), T(P["noise_var"].ravel()), T(P["mask"].ravel()), T(S), 1e-9, s, trace_cap=100)
    ref = oracle.messenger_solve(B, nu * d, nu, S, tau, replay=[(x, None) for x in lam], d=d)
    assert rel(s.cpu().numpy().reshape(n, n), ref["s"]) < 1e-10
    np.testing.assert_allclose(rep["chi2_trace"], ref["chi2"], rtol=1e-10, atol=1e-10 * np.max(np.abs(ref["chi2"])))
    fin = ~np.isnan(ref["resid"])
    np.testing.assert_allclose(rep["resid_trace"][fin], ref["resid"][fin], rtol=1e-6)
    assert rep["chi2_over_ndof"] == pytest.approx(ref["chi2_final"] / ref["n_dof"], rel=1e-10)
    plan.close()
