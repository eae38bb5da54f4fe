"""uc_kkt_noalloc at the edges of its CTAs, groups and row splits, against the
same formulas in torch FP64 on random sparse LPs."""
import ctypes

import numpy as np
import pytest

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


def _csr(torch, rows, cols, width, gen):
    """Random CSR, up to `width` entries per row (empty rows among them)."""
    length = torch.as_tensor(gen.integers(0, width + 1, rows) if cols else np.zeros(rows, int))
    ptr = torch.zeros(rows + 1, dtype=torch.int64)
    ptr[1:] = length.cumsum(0)
    nnz = int(ptr[-1])
    ci = torch.as_tensor(gen.integers(0, max(cols, 1), nnz))
    return length.cuda(), ptr.int().cuda(), ci.int().cuda(), torch.as_tensor(gen.standard_normal(nnz)).cuda()


def _mul(torch, M, rows, v):
    length, _, ci, val = M
    r = torch.repeat_interleave(torch.arange(rows, device="cuda"), length)
    z = torch.zeros(rows, dtype=torch.float64, device="cuda")
    terms = val * v[ci.long()]
    return z.index_add(0, r, terms), z.index_add(0, r, terms.abs())


# m, n: no rows / columns, one, the CTA's 256 and neighbours, a group's 64 CTAs and
# neighbours, several groups, and sizes that take 512 and 1024 rows per CTA
@pytest.mark.parametrize("m,n,m_eq", [(0, 0, 0), (0, 5, 0), (3, 0, 1), (1, 1, 0), (255, 257, 255), (256, 256, 100),
                                      (257, 511, 0), (8192, 8192, 8192), (8192, 8193, 17), (40_000, 70_001, 20_000), (155_000, 160_001, 9),
                                      (1_000_000, 1_097_153, 900_000), (1_100_001, 1_300_000, 3)])
def test_kkt_sizes_match_fp64_formulas(B, m, n, m_eq):
    import torch
    gen = np.random.default_rng(m + 7 * n)
    A, AT = _csr(torch, m, n, 9, gen), _csr(torch, n, m, 9, gen)   # two matrices: the entry takes both as given
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64).cuda()
    c, q = t(gen.standard_normal(n) * (gen.random(n) < 0.5)), t(gen.standard_normal(m) * (gen.random(m) < 0.5))
    lo = t(np.where(gen.random(n) < 0.4, -np.inf, -gen.random(n)))
    up = t(np.where(gen.random(n) < 0.4, np.inf, gen.random(n)))
    Dc, Dr = t(np.exp(gen.standard_normal(n))), t(np.exp(gen.standard_normal(m)))
    x, y = t(gen.standard_normal(n)), t(gen.standard_normal(m))
    out = torch.zeros(8, dtype=torch.float64, device="cuda")
    d = B.uc_device_lp(n=n, m=m, m_eq=m_eq, q_inf=1.5, c_inf=2.5)
    for name, a in dict(A_rowptr=A[1], A_colidx=A[2], A_val=A[3], AT_rowptr=AT[1], AT_colidx=AT[2], AT_val=AT[3],
                        c=c, l=lo, u=up, Dc=Dc, q=q, Dr=Dr).items():
        setattr(d, name, ctypes.c_void_p(a.data_ptr()))
    one = torch.zeros(1, dtype=torch.float64, device="cuda")    # a valid address where a vector is empty
    for _ in range(2):                                          # the second call finds the counters back at zero
        out.fill_(float("nan"))
        assert B.uc_kkt_noalloc(d, (x if n else one).data_ptr(), (y if m else one).data_ptr(), 0.7,
                                out.data_ptr(), torch.cuda.current_stream().cuda_stream) == B.UC_OK
        got = out.cpu().numpy()
        Ax, Aabs = _mul(torch, A, m, x)
        r = Ax - q
        r[m_eq:] = torch.clamp(r[m_eq:], max=0.0)
        ATy, Tabs = _mul(torch, AT, n, y)
        lam = c - ATy
        lf, uf = torch.isfinite(lo), torch.isfinite(up)
        z = torch.zeros_like(lam)
        proj = torch.where(lf & uf, lam, torch.where(lf, lam.clamp(min=0), torch.where(uf, lam.clamp(max=0), z)))
        rd = lam - proj
        bnd = torch.where(lf, lo, z) * proj.clamp(min=0) + torch.where(uf, up, z) * proj.clamp(max=0)
        s = lambda v: float(v.sum()) if v.numel() else 0.0
        top = lambda v: float(v.max()) if v.numel() else 0.0
        pobj, dobj = s(c * x), s(q * y) + s(bnd)
        rp, rdu = top(r.abs() / Dr), top(rd.abs() / Dc)
        gap = pobj - dobj
        want = np.array([rp / 2.5, rdu / 3.5, abs(gap) / (1 + abs(pobj) + abs(dobj)),
                         (0.49 * s(r * r) + s(rd * rd) / 0.49 + gap * gap) ** 0.5, pobj, dobj, rp, 0.0])
        # a row's sum has up to 10 roundings of its absolute terms; the sums over rows
        # are trees of at most 64 levels and terms in a row
        eps = 2.0 ** -52
        row = 10 * eps * max(top((Aabs + q.abs()) / Dr), top((Tabs + c.abs()) / Dc))
        obj = 64 * eps * (s((c * x).abs()) + s((q * y).abs()) + s(bnd.abs())) + 10 * eps * s(Tabs * torch.where(lf | uf, torch.ones_like(z), z))
        tol = np.array([row, row, obj, 0.0, obj, obj, row, 0.0]) + 1e-300
        tol[3] = 100 * eps * want[3] + 2 * obj
        assert (np.abs(got - want) <= tol).all(), (got, want, tol)
