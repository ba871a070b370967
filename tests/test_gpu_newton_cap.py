"""The iteration cap of the mixed precisions: FP32 solves make at most 1 + 3 solves per
linearisation, so a region that needs five from one linearisation is reported as unconverged at
newton_max_iters = 1, whichever solver takes it."""
import numpy as np
import pytest

from oracle import linear as OL
from oracle import nonlinear as NL
from paper_2101_01231_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _chord_updates(q, w, dt, solves):
    """max |dW| / max(1, max |W|) of every region after each solve with the first Jacobian."""
    tb, fl = NL.Tables(2, w["M"]), NL.flux_model(w)
    lam, n = dt / OL.cell_sizes(w), q.shape[0]
    QR = OL.gather_cells(q, w, np.arange(n)).reshape(n, 9, fl.m, tb.thS)
    W = np.zeros((n, 9, fl.m, tb.thT))
    W[..., :tb.thS] = QR
    _, al = NL.residual(W, QR, fl, tb, lam)
    J = NL.jacobian(W, QR, fl, tb, lam, al, "qqf")
    out = []
    for _ in range(solves):
        r, _ = NL.residual(W, QR, fl, tb, lam, frozen=al)
        d = np.linalg.solve(J, r.reshape(n, -1, 1)).reshape(r.shape)
        W -= d
        out.append(np.abs(d).reshape(n, -1).max(1) / np.maximum(1, np.abs(W).reshape(n, -1).max(1)))
    return np.array(out)


@pytest.mark.parametrize("amp", [0.05, 0.1])
def test_fp32_cap_of_one_linearisation(amp):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    w = dict(I.burgers_ensemble(1)[0], M=2, n=(5, 4))
    f = lambda x, y: 0.5 + amp * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    q = np.ascontiguousarray(I.project_tensor(f, w, 3).reshape(-1, 9))
    dt, _ = OL.time_step(w, NL.max_speed(q, w))
    upd = _chord_updates(q, w, dt, 4)
    assert (upd[3] > 1e-9).all()        # ten times the tolerance: no region is done after four
    for cap in (1, 2):
        s = R.Solver(2, w["n"], 2, flux="burgers", cfl=w["cfl"], lo=w["lo"], hi=w["hi"],
                     precision=R.RIDG_PREC_MIXED_FP32, newton_max_iters=cap)
        s.set_state(q)
        s.predict()
        info = s.info()
        s.close()
        assert s.last_status == (R.RIDG_ENOCONV if cap == 1 else R.RIDG_OK)
        assert info["newton_unconverged"] == (20 if cap == 1 else 0)
        assert info["newton_iters_max"] <= cap
