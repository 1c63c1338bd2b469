"""Solves of several threads at once, each with its own plan and stream: the flat solve's CTAs wait for
one another (a cooperative launch), and a temperature solve's next synthesis runs ahead of the host.
Each result has the bits of the same solve alone (both repeat exactly at these sizes)."""
import threading

import numpy as np
import pytest

import wf_inputs as gen
from gpu_util import T, healpix_case

pytestmark = pytest.mark.gpu


class _Solve:
    def __init__(self, wf, kind, size, seed):
        import torch

        self.wf, self.stream = wf, torch.cuda.Stream()
        if kind == "flat":
            P = gen.flat_problem(size, seed=seed)
            d, cov = np.random.default_rng(seed).standard_normal((size, size)).ravel(), P["S"]
            self.plan = wf.wf_plan_create("flat", n=size, stream=self.stream)
        else:
            P, _, d, _, _ = healpix_case(size, 2 * size, seed)
            cov = P["c_ell"]
            self.plan = wf.wf_plan_create("healpix", nside=size, lmax=2 * size, precision="mixed", stream=self.stream)
            wf.wf_set_options(self.plan, ell0=8, band_margin=8, ell_step_max=12)
        self.args = (T(d), T(P["noise_var"].ravel()), T(P["mask"].ravel()), T(cov), 1e-4)
        self.s = torch.empty(d.size, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()

    def run(self, times):
        for _ in range(times):
            self.rep = self.wf.wf_solve(self.plan, *self.args, self.s)


@pytest.mark.parametrize("mix", [[("flat", 128)] * 8, [("flat", 128), ("flat", 32), ("flat", 16), ("flat", 64)] * 2,
                                 [("flat", 128), ("healpix", 32), ("flat", 64), ("healpix", 16), ("healpix", 32)]])
def test_threads_get_the_results_of_solves_alone(mix):
    import torch

    import paper_1210_4931_gb300 as wf

    wf.load()
    solves = [_Solve(wf, kind, size, gen.seed_for(6, 200 + i)) for i, (kind, size) in enumerate(mix)]
    alone = []
    for x in solves:
        x.run(1)
        alone.append((x.s.clone(), x.rep["iters"], x.rep["final_residual"]))
    torch.cuda.synchronize()
    threads = [threading.Thread(target=x.run, args=(5,)) for x in solves]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for x, (s, iters, resid) in zip(solves, alone):
        assert torch.equal(x.s, s)
        assert x.rep["iters"] == iters and x.rep["final_residual"] == resid
        x.plan.close()
