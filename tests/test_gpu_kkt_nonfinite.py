"""uc_kkt_noalloc where a value is not finite or a quotient leaves FP32's range,
against the formulas in numpy FP64: a residual or bound term of an infinity is what
inf - inf and 0 inf give, whatever the other columns of the warp hold."""
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


def _call(B, c, l, u, Dc, q, Dr, m_eq, x, y, at_val):
    """A without entries; A^T with one entry per column, column j's in row j mod m."""
    import torch
    n, m = len(c), len(q)
    t = lambda a, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=dt).cuda()
    d = B.uc_device_lp(n=n, m=m, m_eq=m_eq, q_inf=1.5, c_inf=2.5)
    i32 = torch.int32
    keep = dict(A_rowptr=t(np.zeros(m + 1), i32), A_colidx=t([0], i32), A_val=t([0.0]),
                AT_rowptr=t(np.arange(n + 1), i32), AT_colidx=t(np.arange(n) % m, i32), AT_val=t(at_val),
                c=t(c), l=t(l), u=t(u), Dc=t(Dc), q=t(q), Dr=t(Dr))
    for k, a in keep.items():
        setattr(d, k, ctypes.c_void_p(a.data_ptr()))
    out = torch.full((8,), 7.0, dtype=torch.float64, device="cuda")
    xd, yd = t(x), t(y)
    assert B.uc_kkt_noalloc(d, xd.data_ptr(), yd.data_ptr(), 0.7, out.data_ptr(),
                            torch.cuda.current_stream().cuda_stream) == B.UC_OK
    return out.cpu().numpy()


def _want(c, l, u, Dc, q, Dr, m_eq, x, y, at_val):
    with np.errstate(all="ignore"):
        r = 0.0 - q
        r[m_eq:] = np.where(r[m_eq:] > 0, 0.0, r[m_eq:])
        lm = c - at_val * y[np.arange(len(c)) % len(q)]
        lf, uf = np.isfinite(l), np.isfinite(u)
        lp = np.where(lf & uf, lm, np.where(lf, np.fmax(lm, 0.0), np.where(uf, np.fmin(lm, 0.0), 0.0)))
        rd = lm - lp
        bnd = np.where(lf, np.where(lf, l, 0.0) * np.fmax(lp, 0.0), 0.0) + np.where(uf, np.where(uf, u, 0.0) * np.fmin(lp, 0.0), 0.0)
        pobj, dobj = np.sum(c * x), np.sum(q * y) + np.sum(bnd)
        rp, rdu = np.max(np.abs(r) / Dr), np.max(np.abs(rd) / Dc)
        gap = pobj - dobj
        w = np.sqrt(0.49 * np.sum(r * r) + np.sum(rd * rd) / 0.49 + gap * gap)
        return np.array([rp / 2.5, rdu / 3.5, np.abs(gap) / (1 + np.abs(pobj) + np.abs(dobj)), w, pobj, dobj, rp, 0.0])


def _check(got, want):
    np.testing.assert_array_equal(np.isnan(got), np.isnan(want), err_msg=f"{got} {want}")
    # few hundred terms of one sign or the value itself: a generous multiple of their rounding
    np.testing.assert_allclose(got, want, rtol=1e-12, atol=1e-300)


FREE, LOWER, UPPER, BOX = (-np.inf, np.inf), (1.0, np.inf), (-np.inf, 1.0), (1.0, 2.0)
ZERO_LOWER, ZERO_UPPER, ZERO_BOX = (0.0, np.inf), (-np.inf, 0.0), (0.0, 0.0)


# one column's reduced cost is +-inf or NaN: from an infinite y, or from a finite y whose
# product overflows; the other columns of its warp need the bound term or do not
@pytest.mark.parametrize("bounds", [FREE, LOWER, UPPER, BOX, ZERO_LOWER, ZERO_UPPER, ZERO_BOX])
@pytest.mark.parametrize("bad", ["inf", "-inf", "nan", "overflow", "-overflow"])
@pytest.mark.parametrize("others", [ZERO_LOWER, LOWER])
def test_reduced_cost_that_is_not_finite(B, bounds, bad, others):
    n, m, j = 300, 300, 77
    gen = np.random.default_rng(1)
    c, x = gen.random(n) + 0.5, gen.random(n)
    l, u = np.full(n, others[0]), np.full(n, others[1])
    l[j], u[j] = bounds
    y, at_val, q = np.zeros(m), np.ones(n), np.zeros(m)
    y[j] = {"inf": -np.inf, "-inf": np.inf, "nan": np.nan, "overflow": -1e200, "-overflow": 1e200}[bad]
    if "overflow" in bad:
        at_val[j] = 1e200
    args = (c, l, u, np.exp(gen.standard_normal(n)), q, np.exp(gen.standard_normal(m)), 100, x, y, at_val)
    _check(_call(B, *args), _want(*args))


# an infinite x or y beside a zero or a nonzero cost
@pytest.mark.parametrize("value", [np.inf, -np.inf])
@pytest.mark.parametrize("cost", [0.0, 1.0, -2.0])
@pytest.mark.parametrize("where", ["x", "y"])
def test_infinite_x_or_y_beside_a_cost(B, value, cost, where):
    n, m, j = 260, 520, 259
    c, q, x, y = np.zeros(n), np.zeros(m), np.ones(n), np.zeros(m)
    if where == "x":
        x[j], c[j] = value, cost
    else:
        y[m - 1], q[m - 1] = value, cost     # no column reads the last rows
    args = (c, np.zeros(n), np.full(n, np.inf), np.ones(n), q, np.ones(m), 520, x, y, np.ones(n))
    _check(_call(B, *args), _want(*args))


# a NaN with its sign set, as the device makes of inf - inf, wins the largest residual too
@pytest.mark.parametrize("sign", [0x7ff8 << 48, 0xfff8 << 48])
@pytest.mark.parametrize("where", ["x", "y"])
def test_nan_of_either_sign_wins_the_largest_residual(B, sign, where):
    n, m, j = 300, 300, 131
    nan = np.array([sign], np.uint64).view(np.float64)[0]
    gen = np.random.default_rng(3)
    x, y, q = np.zeros(n), gen.random(m), gen.random(m)
    if where == "y":
        y[j] = nan
    else:
        q[j] = nan          # A has no entries: the row's residual is -q
    args = (gen.random(n), np.full(n, -np.inf), np.full(n, np.inf), np.ones(n), q, np.ones(m), m, x, y, np.ones(n))
    got = _call(B, *args)
    assert np.isnan(got[1 if where == "y" else 0]) and np.isnan(got[3])
