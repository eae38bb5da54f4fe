"""The resident block kernel (default for LPs that fit into the SMs' shared
memory) against the row kernels (spmv_kernel = 1), bit for bit: tile edges, budgets
that end inside a block, batches rebuilt as LPs finish, long
columns, FP32 values, several streams at once."""
import numpy as np
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


def _grid(seed, buses, periods, units):
    return ucgen.make_problem(seed, B=buses, L=min(buses * (buses - 1) // 2, int(1.32 * buses)), G=units, T=periods, lo=0.4, hi=0.8, noise=0.05,
                              zero_pmin_frac=0.1)


def _same(B, ra, rb, ps):
    n, m, _, _ = B.uc_presolved_dims(ps)
    sa, sb = B.uc_get_stats(ra), B.uc_get_stats(rb)
    for key in ("status", "iters", "restarts", "evals", "omega", "rel_primal", "rel_dual", "rel_gap"):
        assert sa[key] == sb[key], (key, sa[key], sb[key])
    for which in (0, 1, 2):
        for a, b in zip(B.uc_get_iterate(ra, which, n, m), B.uc_get_iterate(rb, which, n, m)):
            np.testing.assert_array_equal(a, b)


# one and two buses (a tile of a few rows), sizes around a tile's 32 rows, one tile
# per warp, several tiles per warp (1,500 buses: about two)
@pytest.mark.parametrize("buses,periods,units", [(2, 1, 1), (5, 3, 2), (16, 2, 3), (33, 8, 1), (40, 31, 7), (300, 24, 36),
                                                 (700, 24, 84), (1500, 24, 180)])
@pytest.mark.parametrize("value_bits", [64, 32])
def test_resident_kernel_equals_row_kernels(B, buses, periods, units, value_bits):
    ps = B.uc_presolve(B.uc_build_lp(_grid(buses, buses, periods, units)), value_bits=value_bits, power_max_iter=20)
    for budget in (1, 2, 63, 64, 65, 200):
        _same(B, B.uc_solve(ps, tol=0.0, max_iter=budget, spmv_kernel=1)[0], B.uc_solve(ps, tol=0.0, max_iter=budget)[0], ps)
    a, b = B.uc_solve(ps, tol=0.0, max_iter=100, n_eval=2, spmv_kernel=1)[0], B.uc_solve(ps, tol=0.0, max_iter=100, n_eval=2)[0]
    _same(B, a, b, ps)
    _same(B, a, B.uc_solve(ps, tol=0.0, max_iter=100, n_eval=2, use_graph=False)[0], ps)


# runs of rows with shared entries that begin on tile and group edges (8, 16, 32 periods)
# and off them (10, 31), and the largest CTAs (2,000 buses of 48 periods: more than five tiles per warp)
@pytest.mark.parametrize("buses,periods,units", [(70, 8, 9), (60, 10, 9), (50, 16, 6), (45, 32, 6), (64, 31, 8), (2000, 48, 240)])
@pytest.mark.parametrize("value_bits", [64, 32])
def test_resident_kernel_with_shared_entries(B, buses, periods, units, value_bits):
    ps = B.uc_presolve(B.uc_build_lp(_grid(buses, buses, periods, units)), value_bits=value_bits, power_max_iter=20)
    for budget in (1, 64, 130):
        _same(B, B.uc_solve(ps, tol=0.0, max_iter=budget, spmv_kernel=1)[0], B.uc_solve(ps, tol=0.0, max_iter=budget)[0], ps)


def test_resident_kernel_with_long_columns(B):
    ps = B.uc_presolve(B.uc_build_lp(_grid(3, 500, 24, 60)), eliminate_angles=1, power_max_iter=20)
    for budget in (1, 64, 150):
        _same(B, B.uc_solve(ps, tol=0.0, max_iter=budget, spmv_kernel=1)[0], B.uc_solve(ps, tol=0.0, max_iter=budget)[0], ps)


def test_resident_batch_rebuilt_as_it_shrinks(B):
    # LPs finish at different times and the session is rebuilt for the others
    lps = [_grid(1, 30, 24, 6), _grid(2, 60, 24, 7), _grid(4, 37, 5, 11)]
    pss = [B.uc_presolve(B.uc_build_lp(P)) for P in lps]
    outs = {}
    for kernel in (1, 0):
        s = B.Session(pss, tol=1e-4, max_iter=20_000, spmv_kernel=kernel)
        s.reset(-1)
        s.run()
        outs[kernel] = [s.result(i)[0] for i in range(len(pss))]
        s.reset(1)                       # one LP again, alone
        s.run()
        outs[kernel].append(s.result(1)[0])
        s.close()
    for i, (a, b) in enumerate(zip(outs[1], outs[0])):
        _same(B, a, b, pss[i if i < 3 else 1])
    for i, ps in enumerate(pss):         # and a batch's result is the single solve's
        _same(B, B.uc_solve(ps, tol=1e-4, max_iter=20_000)[0], outs[0][i], ps)


@pytest.mark.parametrize("slots", [2, 4])
@pytest.mark.parametrize("value_bits", [64, 32])
def test_shared_matrix_session_resident_equals_interleaved(B, slots, value_bits):
    # LPs of one grid: in shared memory one beside another, or interleaved (spmv_kernel 1)
    base = _grid(5, 60, 24, 8)
    ps0 = B.uc_presolve(B.uc_build_lp(base), value_bits=value_bits, power_max_iter=20)
    pss = [B.uc_presolve_reuse(ps0, B.uc_build_lp(ucgen.served_request(base, 5, r))) for r in range(slots + 1)]
    for n_eval, budget in ((64, 1), (64, 130), (2, 64)):
        kw = dict(tol=0.0, max_iter=budget, n_eval=n_eval, lanes=True)
        for ps, ra, rb in zip(pss, B.uc_solve_batch(pss[:slots], spmv_kernel=1, **kw)[0], B.uc_solve_batch(pss[:slots], **kw)[0]):
            _same(B, ra, rb, ps)
    outs = []
    for kernel in (1, 0):                # to the end at different times, then one slot refilled alone
        s = B.Session(pss[:slots], tol=1e-3, max_iter=20_000, lanes=True, spmv_kernel=kernel)
        s.reset(-1)
        s.run()
        outs.append([s.result(i)[0] for i in range(slots)])
        s.update_lp(1, pss[slots])
        s.reset(1)
        s.run()
        outs[-1].append(s.result(1)[0])
        s.close()
    for i, (ra, rb) in enumerate(zip(*outs)):
        _same(B, ra, rb, pss[i])


# one host thread and several, the slots' largest LP and a smaller one
@pytest.mark.parametrize("buses", [(40, 20), (500, 30)])
@pytest.mark.parametrize("reorder", [True, False])
def test_slot_takes_another_lp(B, buses, reorder):
    grids = [_grid(s, b, 24, 4) for s, b in enumerate(buses)]
    firsts = [B.uc_presolve(B.uc_build_lp(P), power_max_iter=20) for P in grids]
    s = B.Session(firsts, tol=0.0, max_iter=130, reorder=reorder)
    s.reset(-1)
    s.run()
    for slot in (0, 1):
        other = B.uc_presolve_reuse(firsts[slot], B.uc_build_lp(ucgen.served_request(grids[slot], slot, 3)))
        with pytest.raises(B.UCError):
            s.update_lp(1 - slot, other)
        s.update_lp(slot, other)
        s.reset(slot)
        s.run()
        got = s.result(slot)[0]
        _same(B, B.uc_solve(other, tol=0.0, max_iter=130, reorder=reorder)[0], got, other)
        _, yw = B.uc_get_iterate(got, 2, *B.uc_presolved_dims(other)[:2])
        s.set_start(slot, None, yw, 0.5)     # a start of the new LP's
        s.reset(slot)
        s.run()
        _same(B, B.uc_solve(other, tol=0.0, max_iter=130, reorder=reorder, warm_y=yw, warm_omega=0.5)[0], s.result(slot)[0], other)
    s.close()


def test_resident_sessions_on_several_streams(B):
    import concurrent.futures as cf

    import torch
    pss = [B.uc_presolve(B.uc_build_lp(_grid(s, b, 24, b // 8))) for s, b in ((1, 40), (2, 300), (3, 700), (4, 90))]
    alone = [B.uc_solve(ps, tol=0.0, max_iter=1280)[0] for ps in pss]

    def one(ps):
        with torch.cuda.stream(torch.cuda.Stream()):
            return [B.uc_solve(ps, tol=0.0, max_iter=1280)[0] for _ in range(3)]
    with cf.ThreadPoolExecutor(4) as ex:
        for ps, ref, got in zip(pss, alone, ex.map(one, pss)):
            for r in got:
                _same(B, ref, r, ps)
