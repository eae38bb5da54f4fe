"""The autotuner's trials run the kernels its choices are for: the row kernels, also
for an LP that alone would run the resident kernel."""
import pytest

import ucgen

pytestmark = pytest.mark.gpu


def test_trials_run_the_row_kernels(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_03627_gb300 as pkg
    pkg.build()
    from paper_2607_03627_gb300 import binding as B, tune
    seen = []

    class Recorded(B.Session):
        def close(self):
            if self.ptr:
                st = B.uc_get_stats(self.result(0)[0])
                seen.append((st["kernel_launches"], st["iters"]))
            super().close()
    monkeypatch.setattr(tune.B, "Session", Recorded)
    ps = B.uc_presolve(B.uc_build_lp(ucgen.tiny(0)), power_max_iter=20)
    t = tune.Tuner(cache_path=None)
    ms = {(c, r): t.time_choice(ps, r, c) for c in tune.CTA_CHOICES for r in tune.CHOICES}
    nnz = B.uc_presolved_dims(ps)[3]
    assert t.choose(ps, 64, 5 * nnz) in tune.CHOICES         # three trials of four copies
    assert len(seen) == 9 and all(v > 0 for v in ms.values())
    for launches, iters in seen:         # a primal and a dual launch per iteration
        assert iters >= 64 * t.trial_replays and launches >= 2 * iters
