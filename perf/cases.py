"""Measured workloads of the unit-commitment LP solver.

Every case is one call sequence a user of the package makes, on seeded
synthetic grids (``ucgen``) between the 30-bus and the 6,049-bus size:

kind "kkt"       uc_kkt_noalloc: relative KKT of a point already on the device
kind "solve"     uc_solve: session set-up, cold solve to 1e-4, result
kind "session"   a device-resident session: reset, run to an iteration budget, result
kind "batch"     several uneven LPs in one block-diagonal session
kind "served"    a shared-matrix session: new loads into its slots, reset, run, results
kind "presolve"  uc_presolve with the power iteration for ||A|| on the device

Sizes: ``buses`` with 1.32 lines and 0.12 units per bus (the batch recipe of
``ucgen``) over ``periods`` periods; the 30-bus and 6,049-bus grids have the
line and unit counts of ``ucgen.tiny`` and ``ucgen.paper_scale``.  Iteration
budgets end a solve after a fixed amount of work, as a user with a time limit
does (max_iter); every restart and stopping test before that runs as in a full
solve.

``exact`` evaluates the same formulas in FP64 with numpy and torch alone: its
own LP builder, scaling, power iteration and restarted Halpern PDHG.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import ucgen
from paper_2607_03627_gb300 import binding as B

N_EVAL = 64          # iterations between evaluations (the library's default)
TOL = 1e-4
POWER_STEPS = 500    # the presolve's default limit of the power iteration
POWER_TOL = 1e-10
SOLUTION = ("p", "u", "v", "theta", "f", "shed", "lmp")


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _case(kind, buses, periods, iters=0, value_bits=64, angles=False, slots=1):
    return dict(kind=kind, buses=buses, periods=periods, iters=iters, value_bits=value_bits, angles=angles,
                slots=slots)


def listed():
    cases = {
        # monitoring a 30-bus point kept on the device: two launches, latency only
        "kkt_30": _case("kkt", 30, 24),
        # the same check on the largest grid: one sweep over A, A^T and all vectors
        "kkt_6049": _case("kkt", 6049, 48),
        # a 30-bus LP solved from the host arrays' presolve to 1e-4, set-up included
        "solve_30": _case("solve", 30, 24, iters=100_000),
        # the smallest grid of the uneven batch, re-solved on a resident session
        "session_300": _case("session", 300, 24, iters=6_400),
        # a mid-size grid with FP32 matrix values, a budget that ends inside a block
        "session_1441_fp32": _case("session", 1441, 24, iters=6_437, value_bits=32),
        # the headline LP: 6,049 buses, 48 periods, FP64
        "session_6049": _case("session", 6049, 48, iters=12_800),
        # bus angles substituted out, PD gains on the primal weight: long rows and columns
        "angles_2000": _case("session", 2000, 48, iters=3_200, angles=True),
        # eight LPs of different grids and horizons solved together
        "batch_8": _case("batch", 500, 48, iters=3_200, slots=8),
        # two load variants of one grid admitted to a two-slot server session
        "served_1500x2": _case("served", 1500, 48, iters=3_200, slots=2),
        # four slots of a smaller grid
        "served_600x4": _case("served", 600, 24, iters=3_200, slots=4),
        # presolve of a new grid, norm estimate on the device
        "presolve_3000": _case("presolve", 3000, 48),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["kkt", "solve", "session", "session", "session", "batch", "served", "presolve"])
    periods = rng.choice([24, 48])
    if kind == "kkt":
        return _case(kind, _log_uniform(rng, 30, 6049), periods)
    if kind == "presolve":
        return _case(kind, _log_uniform(rng, 300, 4000), periods)
    if kind == "solve":
        return _case(kind, _log_uniform(rng, 30, 200), 24, iters=rng.randrange(2_000, 16_000))
    if kind == "batch":
        return _case(kind, _log_uniform(rng, 300, 600), periods, iters=rng.randrange(500, 3_000),
                     slots=rng.randrange(2, 9))
    if kind == "served":
        return _case(kind, _log_uniform(rng, 300, 1500), periods, iters=rng.randrange(500, 3_000),
                     slots=rng.choice([2, 4]), value_bits=rng.choice([64, 64, 32]))
    angles = rng.random() < 0.25
    buses = _log_uniform(rng, 60, 2500 if angles else 6049)
    return _case(kind, buses, periods, iters=rng.randrange(500, 6_000), angles=angles,
                 value_bits=rng.choice([64, 64, 32]))


def _grid_sizes(buses):
    if buses == 30:
        return 41, 6
    if buses == 6049:
        return 8000, 700
    return int(round(1.32 * buses)), max(1, int(round(0.12 * buses)))


def _batch_shape(case, i):
    """Buses and periods of LP i of a batch: uneven, up to 3x the first, alternating horizons."""
    return int(round(case["buses"] * (1.0 + 2.0 * ((i * 5) % 8) / 7.0))), case["periods"] // (1 + i % 2)


def _problem(buses, periods, seed):
    lines, units = _grid_sizes(buses)
    if buses == 30:
        P = ucgen.make_problem(seed, B=buses, L=lines, G=units, T=periods, lo=0.4, hi=0.8)
    else:
        P = ucgen.make_problem(seed, B=buses, L=lines, G=units, T=periods, lo=0.5, hi=0.85, noise=0.05,
                               zero_pmin_frac=0.10)
    # a leaf bus as the angle reference: its columns leave the LP with their
    # entries, so the presolved sizes are the same for every seed
    P.ref_bus = int(np.argmin(np.bincount(np.concatenate([P.line_from, P.line_to]), minlength=buses)))
    return P


def _problems(case, seed):
    """The UC problems of a case, one per LP."""
    if case["kind"] == "batch":
        return [_problem(*_batch_shape(case, i), 97 * seed + i) for i in range(case["slots"])]
    base = _problem(case["buses"], case["periods"], seed)
    if case["kind"] == "served":
        return [ucgen.served_request(base, seed % 1000, r) for r in range(case["slots"])]
    return [base]


def _presolve_options(case):
    return dict(value_bits=case["value_bits"], power_device=1, eliminate_angles=int(case["angles"]))


def _solve_options(case):
    o = dict(tol=TOL, max_iter=case["iters"])
    if case["angles"]:
        o["pw_gains"] = (0.5, 0.0, 0.5)
    return o


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    problems = _problems(case, seed)
    if kind == "kkt":
        return _prepare_kkt(problems[0], seed)
    lps = [B.uc_build_lp(p) for p in problems]
    state = dict(case=case, problems=problems, lps=lps)
    if kind == "presolve":
        return state
    options = _presolve_options(case)
    if kind == "served":
        # the server's base LP fixes the scaling; each request reuses it
        base = B.uc_presolve(B.uc_build_lp(_problem(case["buses"], case["periods"], seed)), **options)
        state["ps"] = [B.uc_presolve_reuse(base, lp) for lp in lps]
        state["session"] = B.Session([base] * case["slots"], lanes=True, **_solve_options(case))
        return state
    state["ps"] = [B.uc_presolve(lp, **options) for lp in lps]
    if kind != "solve":
        state["session"] = B.Session(state["ps"], **_solve_options(case))
    return state


def _prepare_kkt(problem, seed):
    lp = _scaled(_reference_lp(problem, False), 64)
    x, y, omega = _kkt_point(lp, seed)
    dev = {"q": lp["q"] / lp["Dr"], "c": lp["c"] / lp["Dc"]}     # unscaled, for the relative parts
    A, AT = lp["A"], lp["AT"]
    arrays = [A.crow_indices().int(), A.col_indices().int(), A.values(), AT.crow_indices().int(),
              AT.col_indices().int(), AT.values(), lp["c"], lp["l"], lp["u"], lp["Dc"], lp["q"], lp["Dr"]]
    arrays = [a.cuda().contiguous() for a in arrays]
    names = ("A_rowptr", "A_colidx", "A_val", "AT_rowptr", "AT_colidx", "AT_val", "c", "l", "u", "Dc", "q", "Dr")
    d = B.uc_device_lp(n=lp["c"].numel(), m=lp["q"].numel(), m_eq=lp["m_eq"],
                       q_inf=float(dev["q"].abs().max()), c_inf=float(dev["c"].abs().max()))
    for name, a in zip(names, arrays):
        setattr(d, name, ctypes.c_void_p(a.data_ptr()))
    return dict(case=dict(kind="kkt"), lp=d, arrays=arrays, x=x.cuda(), y=y.cuda(), omega=omega,
                out=torch.zeros(8, dtype=torch.float64, device="cuda"))


def run(state):
    kind = state["case"]["kind"]
    if kind == "kkt":
        rc = B.uc_kkt_noalloc(state["lp"], state["x"].data_ptr(), state["y"].data_ptr(), state["omega"],
                              state["out"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if rc != B.UC_OK:
            raise B.UCError(rc, "uc_kkt_noalloc")
        return state["out"]
    if kind == "presolve":
        return B.uc_presolved_export(B.uc_presolve(state["lps"][0], **_presolve_options(state["case"])))
    if kind == "solve":
        res, _ = B.uc_solve(state["ps"][0], **_solve_options(state["case"]))
        return _solution(res, state["problems"][0])
    session = state["session"]
    if kind == "served":
        for slot, ps in enumerate(state["ps"]):
            session.update_lp(slot, ps)
    session.reset(-1)
    session.run()
    return [_solution(session.result(i)[0], p) for i, p in enumerate(state["problems"])]


def _solution(res, P):
    d = B.uc_get_solution(res, P.T, P.B, P.L, P.G)
    out = {k: d[k] for k in SOLUTION}
    out["iters"] = d["stats"]["iters"]
    return out


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _sizes(case, buses, periods):
    """Columns, rows and entries of the presolved LP."""
    L, G = _grid_sizes(buses)
    T = periods
    Gp = G if buses == 30 else G - int(round(0.10 * G))     # units with a minimum output
    n = T * (3 * G + 2 * buses - 1 + L)
    m = T * (buses + L + 2 * G + Gp) + 2 * (T - 1) * G
    nnz = T * (G + buses + 2 * L + 3 * L - 1 + 2 * G + 2 * Gp) + (3 * T - 1) * G + 4 * (T - 1) * G
    if case["angles"]:      # no angle columns, no tree rows; cycle rows grow with the grid's depth
        n -= T * (buses - 1)
        m -= T * (buses - 1)
        nnz += T * (int(2.65 * math.log(buses) - 3.3) * (L - buses + 1) - 3 * L)
    return n, m, nnz


def work(case):
    """Bytes and operations of one pass: the LP read and the solution written
    once (a chip with room for the iterates moves nothing else), and per
    iteration the products with A and A^T (an FMA per entry each) and the update
    of every column and row (3 FMAs and a product).  A solve that may stop at
    its tolerance is counted with 8,448 iterations (the 30-bus LP's)."""
    kind = case["kind"]
    if kind == "batch":
        shapes = [_batch_shape(case, i) for i in range(case["slots"])]
    else:
        shapes = [(case["buses"], case["periods"])] * (case["slots"] if kind == "served" else 1)
    nbytes = flops = 0
    for buses, periods in shapes:
        n, m, nnz = _sizes(case, buses, periods)
        matrix = nnz * (4 + case["value_bits"] // 8)
        if kind == "kkt":
            nbytes += 2 * matrix + 8 * (5 * n + 3 * m)
            flops += 4 * nnz + 10 * n + 6 * m
        elif kind == "presolve":
            nbytes += 2 * matrix + 8 * (4 * n + 2 * m)
            flops += POWER_STEPS * (4 * nnz + 3 * n)
        else:
            iters = min(case["iters"], 8_448) if kind == "solve" else case["iters"]
            nbytes += 2 * matrix + 8 * (4 * n + 2 * m)
            flops += iters * (4 * nnz + 7 * n + 7 * m)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same computation in plain FP64 numpy / torch
# ---------------------------------------------------------------------------
def _spanning_tree(P):
    """Breadth-first tree from the reference bus, each bus's lines in order:
    parent[bus] = (parent bus, line, +1 when the bus is the line's from end)."""
    adj = [[] for _ in range(P.B)]
    for l in range(P.L):
        a, b = int(P.line_from[l]), int(P.line_to[l])
        adj[a].append((b, l))
        adj[b].append((a, l))
    parent = {P.ref_bus: None}
    order = [P.ref_bus]
    for v in order:
        for w, l in adj[v]:
            if w not in parent:
                parent[w] = (v, l, 1.0 if int(P.line_from[l]) == w else -1.0)
                order.append(w)
    return parent, order


def _reference_lp(P, angles):
    """Presolved LP of a UC problem in the library's row and column order: COO
    entries, q, c, l, u, equality rows, and the (kind, period, entity) maps."""
    G, Bn, L, T = P.G, P.B, P.L, P.T
    nc = 3 * G + 2 * Bn + L
    op, ou, ov, oth, of, os_ = 0, G, 2 * G, 3 * G, 3 * G + Bn, 3 * G + Bn + L
    g, b, ln, t = np.arange(G), np.arange(Bn), np.arange(L), np.arange(T)[:, None]
    ge = T * (Bn + L)                         # first ">=" row
    inv = 1.0 / P.x_pu
    rows, cols, vals = [], [], []

    def put(r, c, v):
        r, c, v = np.broadcast_arrays(r, c, v)
        rows.append(r.ravel()); cols.append(c.ravel()); vals.append(v.ravel().astype(np.float64))

    bal = t * (Bn + L)
    put(bal + P.gen_bus, t * nc + op + g, 1.0)
    put(bal + b, t * nc + os_ + b, 1.0)
    put(bal + P.line_from, t * nc + of + ln, -1.0)
    put(bal + P.line_to, t * nc + of + ln, 1.0)
    flow = t * (Bn + L) + Bn
    if angles:
        parent, _ = _spanning_tree(P)
        tree_lines = {e[1] for e in parent.values() if e is not None}

        def path(v):
            out = []
            while parent[v] is not None:
                out.append(parent[v])
                v = parent[v][0]
            return out
        for l in range(L):
            if l in tree_lines:
                continue
            pa, pb = path(int(P.line_from[l])), path(int(P.line_to[l]))
            while pa and pb and pa[-1] == pb[-1]:
                pa.pop()
                pb.pop()
            put(flow + l, t * nc + of + l, 1.0)
            for side, edges in ((-1.0, pa), (1.0, pb)):
                for _, e, s in edges:
                    put(flow + l, t * nc + of + e, side * s * inv[l] / inv[e])
    else:
        put(flow + ln, t * nc + of + ln, 1.0)
        put(flow + ln, t * nc + oth + P.line_from, -inv)
        put(flow + ln, t * nc + oth + P.line_to, inv)
    r = ge + t * 5 * G
    put(r + g, t * nc + op + g, -1.0)
    put(r + g, t * nc + ou + g, P.pmax)
    gm = g[P.pmin > 0.0]                       # p >= 0 is a bound, not a row
    put(r + G + gm, t * nc + op + gm, 1.0)
    put(r + G + gm, t * nc + ou + gm, -P.pmin[gm])
    put(r + 2 * G + g, t * nc + ou + g, -1.0)
    put(r + 2 * G + g, t * nc + ov + g, 1.0)
    put((r + 2 * G + g)[1:], (t * nc + ou + g)[:-1], 1.0)
    for k, s in ((3, 1.0), (4, -1.0)):
        put((r + k * G + g)[1:], (t * nc + op + g)[:-1], s)
        put((r + k * G + g)[1:], (t * nc + op + g)[1:], -s)
    rows, cols, vals = np.concatenate(rows), np.concatenate(cols), np.concatenate(vals)
    keep = cols % nc != oth + P.ref_bus        # the reference angle is fixed at 0
    rows, cols, vals = rows[keep], cols[keep], vals[keep]

    zeros = np.zeros(T * nc)
    c, lo, up = zeros.reshape(T, nc).copy(), zeros.reshape(T, nc).copy(), zeros.reshape(T, nc).copy()
    c[:, op:ou], c[:, ou:ov], c[:, ov:oth], c[:, os_:] = P.c_lin, P.c_nl, P.c_su, P.voll
    up[:, op:ou], up[:, ou:oth] = P.pmax, 1.0
    lo[:, oth:of], up[:, oth:of] = -np.inf, np.inf
    lo[:, of:os_], up[:, of:os_] = -P.fmax, P.fmax
    up[:, os_:] = P.load
    q = np.zeros(ge + T * 5 * G)
    q[:ge].reshape(T, Bn + L)[:, :Bn] = P.load
    ineq = q[ge:].reshape(T, 5, G)
    ineq[0, 2] = -P.u0
    ineq[1:, 3:] = -P.ramp

    order = np.lexsort((cols, rows))
    rows, cols, vals = rows[order], cols[order], vals[order]
    row_map, rows = np.unique(rows, return_inverse=True)
    col_map, cols = np.unique(cols, return_inverse=True)
    pick = lambda a: a.ravel()[col_map]
    return dict(rows=rows, cols=cols, vals=vals, q=q[row_map], c=pick(c), l=pick(lo), u=pick(up),
                m_eq=int(np.count_nonzero(row_map < ge)), row_map=row_map, col_map=col_map)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _scaled(R, value_bits):
    """10 Ruiz passes and one Pock-Chambolle pass; CSR matrices on the GPU."""
    dev = _device()
    rows, cols = torch.as_tensor(R["rows"], device=dev), torch.as_tensor(R["cols"], device=dev)
    v = torch.as_tensor(R["vals"], device=dev)
    q, c, l, u = (torch.as_tensor(np.ascontiguousarray(R[k]), device=dev) for k in ("q", "c", "l", "u"))
    m, n = q.numel(), c.numel()
    Dr, Dc = torch.ones_like(q), torch.ones_like(c)
    for it in range(11):
        how = "amax" if it < 10 else "sum"
        rf = torch.zeros_like(q).scatter_reduce(0, rows, v.abs(), how).sqrt()
        cf = torch.zeros_like(c).scatter_reduce(0, cols, v.abs(), how).sqrt()
        v = v / rf[rows] / cf[cols]
        Dr, Dc = Dr / rf, Dc / cf

    def csr(r, k, val, shape):
        ptr = torch.zeros(shape[0] + 1, dtype=torch.int64, device=dev)
        ptr[1:] = torch.bincount(r, minlength=shape[0]).cumsum(0)
        return torch.sparse_csr_tensor(ptr, k, val, shape)

    vs = v.float().double() if value_bits == 32 else v
    order = torch.argsort(cols * m + rows)
    return dict(A=csr(rows, cols, vs, (m, n)), AT=csr(cols[order], rows[order], vs[order], (n, m)), val=v,
                q=q * Dr, c=c * Dc, l=l / Dc, u=u / Dc, Dr=Dr, Dc=Dc, m_eq=R["m_eq"],
                q_inf=float(np.abs(R["q"]).max()), c_inf=float(np.abs(R["c"]).max()))


def _power_norm(S):
    n = S["c"].numel()
    v = torch.full_like(S["c"], 1.0 / math.sqrt(n))
    lam = prev = 0.0
    for _ in range(POWER_STEPS):
        w = S["AT"] @ (S["A"] @ v)
        lam = float(w.norm())
        if lam == 0.0 or abs(lam - prev) <= POWER_TOL * lam:
            break
        prev = lam
        v = w / lam
    return math.sqrt(lam)


def _omega0(S):
    cn, qn = float(S["c"].norm()), float(S["q"].norm())
    return cn / qn if cn > 1e-10 and qn > 1e-10 else 1.0


def _kkt(S, x, y):
    """Residual norms, objectives and relative parts of a scaled point."""
    rp = S["A"] @ x - S["q"]
    rp[S["m_eq"]:].clamp_(max=0.0)
    lam = S["c"] - S["AT"] @ y
    lf, uf = torch.isfinite(S["l"]), torch.isfinite(S["u"])
    zero = torch.zeros_like(lam)
    proj = torch.where(lf & uf, lam, torch.where(lf, lam.clamp(min=0.0), torch.where(uf, lam.clamp(max=0.0), zero)))
    rd = lam - proj
    bound = (torch.where(lf, S["l"], zero) * proj.clamp(min=0.0)).sum()
    bound = bound + (torch.where(uf, S["u"], zero) * proj.clamp(max=0.0)).sum()
    parts = torch.stack([(rp * rp).sum(), (rp.abs() / S["Dr"]).max(), (rd * rd).sum(), (rd.abs() / S["Dc"]).max(),
                         (S["c"] * x).sum(), (S["q"] * y).sum() + bound])
    rp2, rpu, rd2, rdu, pobj, dobj = parts.tolist()
    rel = (rpu / (1.0 + S["q_inf"]), rdu / (1.0 + S["c_inf"]),
           abs(pobj - dobj) / (1.0 + abs(pobj) + abs(dobj)))
    return rp2, rd2, pobj - dobj, rel, pobj, dobj, rpu


def _weighted(k, w):
    return math.sqrt(w * w * k[0] + k[1] / (w * w) + k[2] * k[2])


def _kkt_point(S, seed):
    """A point such as a solve in progress holds: inside the bounds, y_I >= 0."""
    gen = np.random.default_rng(seed + 1)
    x = torch.as_tensor(gen.standard_normal(S["c"].numel()), device=S["c"].device)
    y = torch.as_tensor(gen.standard_normal(S["q"].numel()), device=S["c"].device)
    y[S["m_eq"]:].clamp_(min=0.0)
    return torch.minimum(torch.maximum(x, S["l"]), S["u"]), y, _omega0(S)


def _halpern(S, max_iter, gains):
    """Restarted reflected Halpern PDHG with the constant step 0.998 (the scaled
    matrix has norm at most 1): last map output and iterations."""
    x = torch.zeros_like(S["c"]).clamp(min=S["l"], max=S["u"])
    y = torch.zeros_like(S["q"])
    x0, y0, w, eta = x, y, _omega0(S), 0.998
    anchor, prev, e_prev = _weighted(_kkt(S, x, y), w), math.inf, None
    j = k = 0
    tau, sigma = eta / w, eta * w
    while k < max_iter:
        a = (j + 1.0) / (j + 2.0)
        xh = (x - tau * (S["c"] - S["AT"] @ y)).clamp(min=S["l"], max=S["u"])
        xr = 2.0 * xh - x
        yh = y + sigma * (S["q"] - S["A"] @ xr)
        yh[S["m_eq"]:].clamp_(min=0.0)
        x = a * xr + (1.0 - a) * x0
        y = a * (2.0 * yh - y) + (1.0 - a) * y0
        j += 1
        k += 1
        if k % N_EVAL:
            continue
        kkt = _kkt(S, xh, yh)
        if max(kkt[3]) <= TOL:
            break
        r = _weighted(kkt, w)
        if r <= 0.2 * anchor or (r <= 0.8 * anchor and r > prev) or j >= 0.36 * k:
            dx, dy = float((xh - x0).norm()), float((yh - y0).norm())
            if dx > 1e-10 and dy > 1e-10:
                if gains is None:
                    w = math.exp(0.5 * math.log(dy / dx) + 0.5 * math.log(w))
                else:                        # proportional and derivative gains
                    e = math.log(w * dx / dy)
                    w = math.exp(math.log(w) - gains[0] * e - gains[2] * (e - (e if e_prev is None else e_prev)))
                    e_prev = e
            tau, sigma = eta / w, eta * w
            anchor, prev, j = _weighted(kkt, w), math.inf, 0
            x = x0 = xh
            y = y0 = yh
        else:
            prev = r
    return xh, yh, k


def _exact_solution(case, P, S, R):
    xh, yh, iters = _halpern(S, case["iters"], _solve_options(case).get("pw_gains"))
    G, Bn, L, T = P.G, P.B, P.L, P.T
    nc = 3 * G + 2 * Bn + L
    x, y = np.zeros(T * nc), np.zeros(T * (Bn + L + 5 * G))
    x[R["col_map"]] = (xh * S["Dc"]).cpu().numpy()
    y[R["row_map"]] = (yh * S["Dr"]).cpu().numpy()
    x = x.reshape(T, nc)
    out, at = {}, 0
    for name, size in (("p", G), ("u", G), ("v", G), ("theta", Bn), ("f", L), ("shed", Bn)):
        out[name] = x[:, at:at + size].copy()
        at += size
    if case["angles"]:
        parent, order = _spanning_tree(P)
        for bus in order[1:]:
            up, line, s = parent[bus]
            out["theta"][:, bus] = out["theta"][:, up] + s * out["f"][:, line] * P.x_pu[line]
    out["lmp"] = y[:T * (Bn + L)].reshape(T, Bn + L)[:, :Bn].copy()
    out["iters"] = iters
    return out


def exact(case, seed):
    kind = case["kind"]
    problems = _problems(case, seed)
    if kind == "kkt":
        S = _scaled(_reference_lp(problems[0], False), 64)
        x, y, omega = _kkt_point(S, seed)
        k = _kkt(S, x, y)
        return torch.tensor([*k[3], _weighted(k, omega), k[4], k[5], k[6], 0.0], dtype=torch.float64)
    if kind == "presolve":
        R = _reference_lp(problems[0], False)
        S = _scaled(R, 64)
        norm = _power_norm(S)
        host = lambda v: v.cpu().numpy()
        P = problems[0]
        first = P.T * (P.B + P.L) + 5 * P.G     # the ramp rows start in the second period
        row_map = R["row_map"] - 2 * P.G * (R["row_map"] >= first)
        return dict(rowptr=host(S["A"].crow_indices()).astype(np.int32), colidx=R["cols"].astype(np.int32),
                    val=host(S["val"]), q=host(S["q"]), c=host(S["c"]), l=host(S["l"]), u=host(S["u"]),
                    Dr=host(S["Dr"]), Dc=host(S["Dc"]), col_map=R["col_map"].astype(np.int32),
                    row_map=row_map.astype(np.int32), n=S["c"].numel(), m=S["q"].numel(), m_eq=S["m_eq"],
                    eta=0.998 / max(1.0, norm), omega0=_omega0(S), norm_A=norm, obj_const=0.0, q_inf=S["q_inf"],
                    c_inf=S["c_inf"], norm_bound=max(1.0, norm))
    outs = []      # a served request takes the base LP's scaling, which does not depend on the load
    for P in problems:
        R = _reference_lp(P, case["angles"])
        outs.append(_exact_solution(case, P, _scaled(R, case["value_bits"]), R))
    return outs[0] if kind == "solve" else outs
