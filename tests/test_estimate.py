"""Size of a plan as the request loop's admission sees it (host only): a small grid does not pay for the
ring FFT tables of the largest.  The bounds are the budgets that held these plans when rings took
other FFTs, plus 0.1 %."""
import pytest


@pytest.mark.parametrize("precision,nside,bytes_", [("mixed", 8, 1143496), ("fp64", 8, 1161904), ("mixed", 64, 6433720),
                                                    ("fp64", 64, 7829776), ("mixed", 512, 401605560)])
def test_small_plans_keep_their_size(precision, nside, bytes_):
    import paper_1210_4931_gb300 as wf
    from paper_1210_4931_gb300 import build

    build.build()
    assert wf.wf_plan_estimate_bytes("healpix", nside=nside, lmax=2 * nside, precision=precision) <= 1.001 * bytes_
