"""The 2D nonlinear correction with one cell per block up to a full block's, as the mesh's size asks
(152 SMs: one cell up to 152, all from 16 x 152 at Burgers Q1): the oracle's correction of the same
prediction."""
import numpy as np
import pytest

from oracle import nonlinear as NL
from paper_2101_01231_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flux,M,n", [("burgers", 1, (19, 8)), ("burgers", 1, (17, 9)), ("burgers", 1, (31, 29)),
                                      ("burgers", 1, (53, 47)), ("burgers", 2, (23, 22)), ("burgers", 3, (31, 26)),
                                      ("burgers", 4, (22, 19)), ("euler", 1, (21, 22)), ("euler", 1, (37, 33)),
                                      ("euler", 2, (13, 24))])
def test_cells_per_block(flux, M, n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    w = I.workload("euler2d_n512_q2", n=n, M=M) if flux == "euler" else dict(I.burgers_ensemble(1)[0], M=M, n=n)
    m, ths = (4 if flux == "euler" else 1), (M + 1) ** 2
    q = 1e-5 * np.random.default_rng(M).standard_normal((n[0] * n[1], m, ths))
    q[:, :, 0] += np.array([1.0, 0.3, -0.2, 2.5])[:m]
    q = q.reshape(n[0] * n[1], -1)
    s = R.Solver(2, n, M, flux=flux, cfl=0.2, lo=w["lo"], hi=w["hi"], precision=R.RIDG_PREC_MIXED_FP32)
    s.set_state(q)
    W = s.predict()
    dt = s.info()["dt"]
    s.correct()
    q1 = s.get_state()
    s.close()
    ref = NL.correct(q, W, w, dt)
    # FP64 sums of a few hundred terms of size |Q| on both sides
    assert np.abs(q1 - ref).max() <= 1e-13 * np.abs(ref).max()
    assert np.abs(q1 - q).max() > 1e-7
