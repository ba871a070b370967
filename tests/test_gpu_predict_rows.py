"""3D degree 4: four or five rows of the operator per thread, whichever leaves the busiest SM fewer
(152 SMs: five at 9 x 10 x 8 and 11^3 cells, four at 3^3 and 16^3; the whole prediction of 5^3: five).
Both are the same sums: time means and whole predictions against the oracle, and every launch form
against each other bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(3, 3, 3), (5, 5, 5), (9, 10, 8), (11, 11, 11), (16, 16, 16)])
@pytest.mark.parametrize("vel", [(0.8, -0.5, 0.3), (0.0, 0.6, 0.0)])
def test_rows_per_thread_3d_q4(n, vel):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from oracle import linear as OL
    from paper_2101_01231_gb300 import inputs as I
    from paper_2101_01231_gb300 import ridg as R
    w = I.workload("adv3d_n96_q2", n=n, M=4, vel=vel, cfl=0.2)
    rng = np.random.default_rng(4)
    cells = int(np.prod(n))
    q0 = rng.standard_normal((cells, 125))
    s = R.Solver(3, n, 4, vel=vel, cfl=0.2)
    s.set_state(q0)
    W = s.predict()
    dt = s.info()["dt"]
    some = np.unique(rng.integers(0, cells, 12))
    ref = OL.step_cells(q0, w, dt, some)
    # sums of up to 1000 products of O(1) terms
    s.step(1)
    q1 = s.get_state()
    assert np.abs(q1[some] - ref).max() <= 2e-12 * np.abs(ref).max()
    s.set_state(q0)
    s.predict()
    s.correct()
    assert np.array_equal(s.get_state(), q1)     # the whole prediction's rows are the step's
    s.close()
    assert np.isfinite(W).all()


def test_rows_per_thread_cost_no_step():
    """A mesh where five rows leave a third, nearly empty wave of blocks costs no more per cell than
    a larger one."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    ms = {}
    for n in (20, 24):
        s = R.Solver(3, (n, n, n), 4, vel=(0.8, -0.5, 0.3), cfl=0.2)
        s.set_state(np.random.default_rng(1).standard_normal((n ** 3, 125)))
        s.profile_step(2)
        ms[n] = min(s.profile_step(3)["predict_ms"] for _ in range(3))
        s.close()
    # (five rows: 2.27 against 3.13 ms, four: 1.79 against 3.10)
    assert ms[20] <= ms[24] * (20 / 24) ** 3 * 1.12
