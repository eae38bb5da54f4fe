"""The resident block kernel at its limits: a wait that runs out, blocks too short for
the timed iteration, what a session uploads, sessions that device memory holds only
without it, tables rebuilt, sessions that fill the SMs side by side."""
import ctypes

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


def _presolved(B, seed, buses, periods, units, **kw):
    return B.uc_presolve(B.uc_build_lp(ucgen.make_problem(
        seed, B=buses, L=int(1.32 * buses), G=units, T=periods, lo=0.4, hi=0.8, noise=0.05, zero_pmin_frac=0.1)),
        power_max_iter=20, **kw)


def _same(B, ra, rb, ps):
    n, m, _, _ = B.uc_presolved_dims(ps)
    sa, sb = B.uc_get_stats(ra), B.uc_get_stats(rb)
    for key in ("status", "iters", "restarts", "evals", "omega", "rel_primal", "rel_dual", "rel_gap"):
        assert sa[key] == sb[key], (key, sa[key], sb[key])
    for which in (0, 1, 2):
        for a, b in zip(B.uc_get_iterate(ra, which, n, m), B.uc_get_iterate(rb, which, n, m)):
            np.testing.assert_array_equal(a, b)


def test_a_wait_that_runs_out_is_an_error_status_and_the_session_goes_on(B):
    # every wait gives up after its second look: the kernel ends, the LP is reported as
    # failed, and with the usual limit the session solves as ever
    ps = _presolved(B, 6, 100, 24, 12)
    limit = B.lib.uc_session_wait_limit
    limit.argtypes, limit.restype = [ctypes.c_void_p, ctypes.c_uint], ctypes.c_int
    s = B.Session([ps], tol=0.0, max_iter=640)
    assert limit(s.ptr, 0) == B.UC_OK
    s.reset(-1)
    s.run()
    _, rc = s.result(0)
    assert rc == B.UC_ECUDA and b"stopped waiting" in B.lib.uc_last_error()
    assert limit(s.ptr, 1 << 25) == B.UC_OK
    s.reset(-1)
    s.run()
    _same(B, B.uc_solve(ps, tol=0.0, max_iter=640, spmv_kernel=1)[0], s.result(0)[0], ps)
    s.close()


# every block of n_eval iterations times one of them; a block that the budget ends
# before it times none
@pytest.mark.parametrize("n_eval,budget,timed", [(2, 64, True), (4, 64, True), (64, 640, True), (64, 20, False)])
def test_kernel_timing_of_short_blocks(B, n_eval, budget, timed):
    ps = _presolved(B, 1, 60, 24, 8)
    st = B.uc_get_stats(B.uc_solve(ps, tol=0.0, max_iter=budget, n_eval=n_eval, kernel_timing=True)[0])
    assert st["kernel_launches"] < budget * 5            # the resident kernel: five launches a block
    if not timed:
        assert st["timed_launches"] == 0
        return
    # the last block ends the solve and is not read
    assert budget // n_eval - 2 <= st["timed_launches"] <= budget // n_eval
    assert 0 < st["primal_kernel_ms"] + st["dual_kernel_ms"] < 1


def test_upload_has_no_packed_entries(B):
    # against a session on the row kernels (n_eval above the resident kernel's limit): only
    # the tiles (32 bytes per 32 rows or columns of a kind) and the warps' lists come along
    ps = _presolved(B, 2, 300, 24, 36)
    n, m, _, _ = B.uc_presolved_dims(ps)
    sent = [B.uc_get_stats(B.uc_solve(ps, tol=0.0, max_iter=64, n_eval=e)[0])["h2d_bytes"] for e in (64, 1026)]
    assert 0 < sent[0] - sent[1] < 2 * (n + m) + 64 * 1024


# device memory for the row kernels' session but not for the resident kernel's: the
# session runs on the row kernels; for less: refused as ever
@pytest.mark.parametrize("kind", ["one", "batch", "lanes"])
def test_session_that_fits_only_without_the_resident_kernel(B, monkeypatch, kind):
    base = ucgen.make_problem(5, B=60, L=79, G=8, T=24, lo=0.4, hi=0.8, noise=0.05, zero_pmin_frac=0.1)
    ps0 = B.uc_presolve(B.uc_build_lp(base), power_max_iter=20)
    pss, kw = [ps0], dict(tol=0.0, max_iter=130)
    if kind == "batch":
        pss = [ps0, _presolved(B, 7, 40, 24, 5), _presolved(B, 8, 30, 5, 4)]
    if kind == "lanes":
        pss = [B.uc_presolve_reuse(ps0, B.uc_build_lp(ucgen.served_request(base, 5, r))) for r in range(2)]
        kw["lanes"] = True
    rows = B.Session(pss, **dict(kw, n_eval=1026))
    limit = rows.device_bytes()
    rows.close()

    class Limited(B._TorchAllocator):
        def _alloc(self, nbytes, stream, ctx):
            return super()._alloc(nbytes, stream, ctx) if nbytes <= self.limit else None
    small = Limited()
    B._torch_stream_and_allocator()
    monkeypatch.setattr(B, "_allocator", small)
    small.limit = limit
    s = B.Session(pss, **kw)
    assert s.device_bytes() == limit
    s.reset(-1)
    s.run()
    for i, ps in enumerate(pss):
        small.limit = 1 << 40
        _same(B, B.uc_solve(ps, spmv_kernel=1, tol=0.0, max_iter=130)[0], s.result(i)[0], ps)
    s.close()
    small.limit = limit - 1
    with pytest.raises(B.UCError, match="allocator returned NULL"):
        B.Session(pss, **kw)


def test_tables_are_rebuilt_without_a_pass_over_the_matrices(B):
    # a reset that brings LPs back into the launch tables deals their tiles anew; the
    # tiles themselves are cut once, with the session.  About 1 % of the session's
    # creation; cut again each time they take 10 %.
    import time

    import torch
    pss = [_presolved(B, s, 1500, 48, 180) for s in range(3)]
    for _ in range(2):                       # the first is not timed
        t0 = time.perf_counter()
        s = B.Session(pss, tol=0.0, max_iter=640)
        torch.cuda.synchronize()
        create = time.perf_counter() - t0
    took = []
    for _ in range(7):
        for i in (0, -1):                    # one alone: the tables shrink to it between its blocks; then all again
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            s.reset(i)
            torch.cuda.synchronize()
            if i < 0:
                took.append(time.perf_counter() - t0)
            s.run()
            [s.result(q) for q in range(3)]
    assert sorted(took)[3] < 0.04 * create
    s.close()


def test_sessions_that_each_fill_the_sms_run_side_by_side(B):
    # three resident sessions with one CTA of 28 warps on every SM, whose registers leave no
    # room for another's, on streams of both priorities, beside a session on the row kernels: their launches
    # take turns, and every result is that of the session alone
    import concurrent.futures as cf

    import torch
    pss = [_presolved(B, s, 3000, 48, 360) for s in range(2)]
    kw = dict(tol=0.0, max_iter=1280)
    alone = [B.uc_solve(ps, **kw)[0] for ps in pss]
    jobs = [(0, 0, {}), (1, -1, {}), (0, -1, {}), (1, 0, dict(spmv_kernel=1))]

    def one(job):
        i, priority, more = job
        with torch.cuda.stream(torch.cuda.Stream(priority=priority)):
            return [B.uc_solve(pss[i], **kw, **more)[0] for _ in range(3)]
    with cf.ThreadPoolExecutor(len(jobs)) as ex:
        for (i, _, _), got in zip(jobs, ex.map(one, jobs)):
            for r in got:
                _same(B, alone[i], r, pss[i])
