"""The Halpern row kernels with period-strided slots, which run LPs and batches that
do not fit into the SMs' shared memory, on LPs that do: n_eval above
UC_RESIDENT_MAX_EVAL selects them.  Against the resident kernel and the CSR-only row
kernels bit for bit, against the oracle, for every row split; and which kernels a
session runs, by its launches."""
import numpy as np
import pytest

import ucgen
from gpu_common import ITERATE_RTOL, oracle_pipeline, oracle_trace, rel_inf

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


@pytest.fixture(scope="module")
def rows(B):
    return B.UC_RESIDENT_MAX_EVAL + 2        # n_eval of the row kernels


def _grid(seed, buses, periods, units):
    return ucgen.make_problem(seed, B=buses, L=min(buses * (buses - 1) // 2, int(1.32 * buses)), G=units, T=periods, lo=0.4, hi=0.8,
                              noise=0.05, zero_pmin_frac=0.1)


def _iterates(B, res, ps):
    n, m, _, _ = B.uc_presolved_dims(ps)
    return [v for which in (0, 1, 2) for v in B.uc_get_iterate(res, which, n, m)]


def _equal(B, ra, rb, ps, stats=()):
    for a, b in zip(_iterates(B, ra, ps), _iterates(B, rb, ps)):
        np.testing.assert_array_equal(a, b)
    sa, sb = B.uc_get_stats(ra), B.uc_get_stats(rb)
    assert [sa[k] for k in stats] == [sb[k] for k in stats]


STATS = ("status", "iters", "restarts", "evals", "omega", "rel_primal", "rel_dual", "rel_gap")
LPS = {"two_buses": (2, 2, 1, 1), "ragged": (7, 37, 5, 11), "31_periods": (3, 40, 31, 7), "groups": (5, 300, 24, 36)}


@pytest.mark.parametrize("name", LPS)
@pytest.mark.parametrize("value_bits", [64, 32])
@pytest.mark.parametrize("cta,rpt", [(0, 1), (128, 4), (256, 2), (512, 1), (512, 4)])
def test_strided_row_kernels_equal_csr_and_resident(B, rows, name, value_bits, cta, rpt):
    ps = B.uc_presolve(B.uc_build_lp(_grid(*LPS[name])), value_bits=value_bits, power_max_iter=20)
    kw = dict(tol=0.0, cta_rows=cta, rows_per_thread=[rpt])
    for budget in (1, 2, 63, 200, 1024, rows, rows + 75):
        r = B.uc_solve(ps, max_iter=budget, n_eval=rows, **kw)[0]
        assert B.uc_get_stats(r)["kernel_launches"] > 2 * budget
        _equal(B, B.uc_solve(ps, max_iter=budget, n_eval=rows, spmv_kernel=1, **kw)[0], r, ps, STATS)
        if budget < 1024:                    # before the first evaluation of either
            res = B.uc_solve(ps, tol=0.0, max_iter=budget, n_eval=rows - 2)[0]
            assert B.uc_get_stats(res)["kernel_launches"] < 16
            _equal(B, res, r, ps)


def test_row_kernels_with_long_columns(B, rows):
    ps = B.uc_presolve(B.uc_build_lp(_grid(3, 500, 24, 60)), eliminate_angles=1, power_max_iter=20)
    for rpt in (1, 2, 4):
        for budget in (1, 200, rows + 75):
            r = B.uc_solve(ps, tol=0.0, max_iter=budget, n_eval=rows, rows_per_thread=[rpt])[0]
            _equal(B, B.uc_solve(ps, tol=0.0, max_iter=budget, n_eval=rows, spmv_kernel=1)[0], r, ps, STATS)
            if budget < 1024:
                _equal(B, B.uc_solve(ps, tol=0.0, max_iter=budget, n_eval=rows - 2)[0], r, ps)


@pytest.mark.parametrize("use_graph", [True, False])
def test_row_kernels_match_the_oracle(B, rows, use_graph):
    # non-expansive steps of about 1e-16 relative difference each: 1e-9 leaves the
    # same wide margin over 1,101 of them as over 200
    P = _grid(7, 37, 5, 11)
    _, _, S = oracle_pipeline(P)
    ks = [1, 65, 200, rows, rows + 75]
    ref = oracle_trace(S, ks, n_eval=rows)
    ps = B.uc_presolve(B.uc_build_lp(P))
    for k in ks:
        res = B.uc_solve(ps, tol=0.0, max_iter=k, n_eval=rows, use_graph=use_graph)[0]
        x, y, _, _, xm, ym = _iterates(B, res, ps)
        for got, want in ((x, ref[k][0]), (y, ref[k][1]), (xm, ref[k][4]), (ym, ref[k][5])):
            assert rel_inf(got, want) <= ITERATE_RTOL, (k, rel_inf(got, want))
        assert B.uc_get_stats(res)["restarts"] == ref[k][2]


def test_row_kernel_batch_equals_single_solves(B, rows):
    # uneven LPs, groups of 16 rows that belong to two of them, every row split, tables
    # rebuilt as LPs end
    pss = [B.uc_presolve(B.uc_build_lp(_grid(*LPS[k])), power_max_iter=20) for k in ("ragged", "31_periods", "groups", "two_buses")]
    kw = dict(tol=1e-3, max_iter=40_000, n_eval=rows)
    batch = B.uc_solve_batch(pss, rows_per_thread=[4, 2, 1, 4], **kw)[0]
    for ps, r in zip(pss, batch):
        _equal(B, B.uc_solve(ps, spmv_kernel=1, **kw)[0], r, ps, STATS)


# a few rows, one tile per warp, 24 warps, 28 warps with staged constants
@pytest.mark.parametrize("buses,periods,units", [(2, 1, 1), (100, 24, 12), (1500, 24, 180), (2000, 48, 240)])
@pytest.mark.parametrize("value_bits", [64, 32])
def test_launches_show_the_kernels_of_a_session(B, rows, buses, periods, units, value_bits):
    base = _grid(buses, buses, periods, units)
    ps = B.uc_presolve(B.uc_build_lp(base), value_bits=value_bits, power_max_iter=20)
    launches = lambda r: B.uc_get_stats(r)["kernel_launches"]
    # resident: block, evaluation (three) and restart per 64 iterations, up to two more blocks queued
    assert launches(B.uc_solve(ps, tol=0.0, max_iter=640)[0]) <= 3 + 12 * 5
    assert launches(B.uc_solve(ps, tol=0.0, max_iter=640, n_eval=rows - 2)[0]) <= 3 + 2 * 5
    for kw in (dict(n_eval=rows), dict(spmv_kernel=1), dict(algorithm="average")):
        assert launches(B.uc_solve(ps, tol=0.0, max_iter=640, **kw)[0]) >= 2 * 640
    pair = [ps, B.uc_presolve_reuse(ps, B.uc_build_lp(ucgen.served_request(base, buses, 1)))]
    for lanes in (False, True):
        assert launches(B.uc_solve_batch(pair, tol=0.0, max_iter=640, lanes=lanes)[0][0]) <= 3 + 12 * 5
        assert launches(B.uc_solve_batch(pair, tol=0.0, max_iter=640, lanes=lanes, n_eval=rows)[0][0]) >= 2 * 640
