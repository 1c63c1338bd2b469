"""Flat-grid solve at every size its FFT distinguishes (n = 16, 64: radix-4 passes only; 32, 128:
a last radix-2 pass; 16: fewer values than a warp): a replayed schedule, its traces, the
fluctuation term and the input checks of the first and the last pixel, against the oracle.
Tolerance: FP64 iterations that contract, ~50 roundings each of 1.1e-16 (1e-10)."""
import numpy as np
import pytest

import oracle
import wf_inputs as gen
from gpu_util import T, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 32, 64, 128])
def test_flat_grid_sizes(n):
    import torch

    import paper_1210_4931_gb300 as wf

    wf.load()
    P = gen.flat_problem(n, seed=gen.seed_for(1, 60 + n), band_rows=(n // 2 - 2, n // 2 + 2), n_disks=3,
                         disk_radius=2.0)
    P["mask"][0, 0] = P["mask"][-1, -1] = 1
    B = oracle.FlatBasis(n, n)
    nu = np.where(P["mask"] > 0, 1.0 / P["noise_var"], 0.0)
    tau = float(P["noise_var"][P["mask"] > 0].min())
    d = B.synth(P["a_signal"]) + P["noise"]
    plan = wf.wf_plan_create("flat", n=n)
    nv, mk, S = T(P["noise_var"].ravel()), T(P["mask"].ravel()), T(P["S"].ravel())
    s = torch.empty(n * n, dtype=torch.float64, device="cuda")
    lam = [100.0, 100.0, 7.0, 3.0, 1.0, 1.0, 1.0]
    for r, out in ((nu * d, "solve"), (oracle.fluct_source(B, nu, P["S"], P["g1"], P["g2"]), "fluct")):
        if out == "solve":
            wf.wf_set_schedule(plan, lam)
            rep = wf.wf_solve(plan, T(d.ravel()), nv, mk, S, 1e-6, s, trace_cap=100)
            used = lam
        else:
            wf.wf_set_schedule(plan, [])
            rep = wf.wf_fluct(plan, nv, mk, S, T(P["g1"].ravel()), T(P["g2"].ravel()), 1e-6, s, trace_cap=20000)
            used = rep["lambda_trace"]
        ref = oracle.messenger_solve(B, r, nu, P["S"], tau, replay=[(x, None) for x in used],
                                     d=d if out == "solve" else None)
        np.testing.assert_array_equal(rep["lambda_trace"], used)
        assert rel(s.cpu().numpy().reshape(n, n), ref["s"]) < 1e-10
        np.testing.assert_allclose(rep["chi2_trace"], ref["chi2"], rtol=1e-10,
                                   atol=1e-10 * np.max(np.abs(ref["chi2"])))
        fin = ~np.isnan(ref["resid"])
        np.testing.assert_allclose(rep["resid_trace"][fin], ref["resid"][fin], rtol=1e-6)
    for at in (0, n * n - 1):  # the setup's first and last block report a bad variance
        bad = P["noise_var"].ravel().copy()
        bad[at] = np.nan
        with pytest.raises(wf.WfError) as e:
            wf.wf_solve(plan, T(d.ravel()), T(bad), mk, S, 1e-6, s)
        assert e.value.status == wf.WF_EINVAL
    plan.close()
