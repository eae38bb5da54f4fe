"""The device power iteration against the host's at sizes around a CTA's 256 rows,
with rows longer than the four entries loaded at once, and where it stops early."""
import pytest

import ucgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_03627_gb300 as pkg
    pkg.build()
    from paper_2607_03627_gb300 import binding
    return binding


# steps times the rounding of a step's sums (2 k eps for k steps, the sums' own
# rounding aside, which both sides have): 500 steps stay below 1e-12
@pytest.mark.parametrize("buses,periods,units", [(2, 1, 1), (3, 2, 1), (10, 8, 2), (16, 8, 1), (64, 24, 8), (1100, 24, 132)])
@pytest.mark.parametrize("angles", [False, True])
@pytest.mark.parametrize("steps,tol", [(1, 1e-10), (500, 1e-10), (500, 1e-3)])
def test_device_norm_equals_host_norm(B, buses, periods, units, angles, steps, tol):
    P = ucgen.make_problem(buses, B=buses, L=min(buses * (buses - 1) // 2, int(1.32 * buses)), G=units, T=periods, lo=0.4,
                           hi=0.8, noise=0.05, zero_pmin_frac=0.1)
    lp = B.uc_build_lp(P)
    kw = dict(power_max_iter=steps, power_tol=tol, eliminate_angles=int(angles))
    h = B.uc_presolved_export(B.uc_presolve(lp, **kw))
    d = B.uc_presolved_export(B.uc_presolve(lp, power_device=1, **kw))
    assert d["norm_A"] == pytest.approx(h["norm_A"], rel=1e-12)
