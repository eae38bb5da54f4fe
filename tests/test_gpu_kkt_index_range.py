"""uc_kkt_noalloc on row pointers up to 2^31 - 1: the entries of one warp's rows, which
differ in length, are read in bounds and none twice.  The arrays hold the last entries
only; the addresses handed over lie before them by the first entry's index."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

END = 2 ** 31 - 1


@pytest.mark.parametrize("lengths", [(207, 0, 7), (1, 400, 3), (5,), (64, 1, 2, 3, 4)])
def test_rows_that_end_at_the_largest_index(lengths):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_03627_gb300 as pkg
    pkg.build()
    from paper_2607_03627_gb300 import binding as B
    k, nnz = len(lengths), sum(lengths)
    gen = np.random.default_rng(nnz)
    first = END - nnz
    ptr = first + np.concatenate([[0], np.cumsum(lengths)])
    ci, val = gen.integers(0, k, nnz), gen.standard_normal(nnz)
    t = lambda a, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=dt).cuda()
    i32 = torch.int32
    rp_d, ci_d, val_d = t(ptr, i32), t(ci, i32), t(val)
    x, y, c, q = (gen.standard_normal(k) for _ in range(4))
    vec = dict(c=t(c), q=t(q), l=t(np.full(k, -np.inf)), u=t(np.full(k, np.inf)), Dc=t(np.ones(k)), Dr=t(np.ones(k)))
    d = B.uc_device_lp(n=k, m=k, m_eq=k, q_inf=0.0, c_inf=0.0)
    for name, a in vec.items():
        setattr(d, name, ctypes.c_void_p(a.data_ptr()))
    for side in ("A", "AT"):
        setattr(d, side + "_rowptr", ctypes.c_void_p(rp_d.data_ptr()))
        setattr(d, side + "_colidx", ctypes.c_void_p(ci_d.data_ptr() - 4 * first))
        setattr(d, side + "_val", ctypes.c_void_p(val_d.data_ptr() - 8 * first))
    out = torch.zeros(8, dtype=torch.float64, device="cuda")
    xd, yd = t(x), t(y)
    assert B.uc_kkt_noalloc(d, xd.data_ptr(), yd.data_ptr(), 1.0, out.data_ptr(),
                            torch.cuda.current_stream().cuda_stream) == B.UC_OK
    got = out.cpu().numpy()
    rows = np.repeat(np.arange(k), lengths)
    mul = lambda v: np.bincount(rows, weights=val * v[ci], minlength=k)
    pobj, dobj = float(c @ x), float(q @ y)
    rp, rd = np.abs(mul(x) - q).max(), np.abs(c - mul(y)).max()
    # a row's sum of at most 400 terms of at most 10 in size
    np.testing.assert_allclose(got[[0, 1, 4, 5, 6]], [rp, rd, pobj, dobj, rp], rtol=0, atol=400 * 400 * 10 * 2.0 ** -52)
