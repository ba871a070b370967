"""The autotuner and the block elimination's grid: it is timed, and stored, only where regions go
there; a grid that an earlier version stored without that is not read."""
import numpy as np
import pytest

from paper_2101_01231_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _solver(R, **kw):
    w = dict(I.burgers_ensemble(1)[0], n=(24, 20), M=3)
    s = R.Solver(2, w["n"], w["M"], flux="burgers", cfl=w["cfl"], precision=R.RIDG_PREC_MIXED_FP32, **kw)
    return s, I.initial_state(w)


def test_grid_is_tuned_only_for_listed_regions(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    family = f"nb4 m1 flux{R.RIDG_FLUX_BURGERS} prec{R.RIDG_PREC_MIXED_FP32}"
    s, q = _solver(R)
    largest = s.tuning()["newton_grid"]
    s.close()
    f = tmp_path / "old.txt"
    f.write_text(f"newton.grid {family} 1\n")
    R.ridg_tune_load(str(f))
    s, q = _solver(R)
    assert s.tuning()["newton_grid"] == largest
    s.set_state(q)
    s.step(1)
    assert s.sync() == R.RIDG_OK        # (every region by the iterative solver)
    s.set_state(q)
    s.autotune()
    assert s.tuning()["newton_grid"] == largest
    assert R.ridg_tune_lookup(f"newton.list_grid {family}") is None
    s.close()
    # a tolerance that no region meets: all of them are eliminated, and the grid is timed
    s, q = _solver(R, newton_tol=1e-30)
    s.set_state(q)
    s.autotune()
    g = s.tuning()["newton_grid"]
    assert 1 <= g <= largest
    assert R.ridg_tune_lookup(f"newton.list_grid {family}") in (1, 2, 4, 8)
    assert np.array_equal(s.get_state(), q)
    s.close()
    s, _ = _solver(R)
    assert s.tuning()["newton_grid"] == g
    s.set_state(q)
    s.autotune()
    assert s.tuning()["newton_grid"] == g       # (nothing listed: a stored choice stays)
    s.close()
