"""Newton predictions of states far below the solvers' FP32 range, against the oracle at the same
scale."""
import numpy as np
import pytest

from oracle import linear as OL
from oracle import nonlinear as NL
from paper_2101_01231_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg
    return ridg


def _problem(dim, n):
    if dim == 2:
        w = dict(I.burgers_ensemble(1)[0], M=2, n=n)
        f = lambda x, y: 0.5 + 0.05 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    else:
        w = dict(flux="burgers", dim=3, n=n, M=1, lo=(0.0,) * 3, hi=(1.0,) * 3, cfl=0.3)
        f = lambda x, y, z: 0.5 + 0.05 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * (y - z))
    q = np.ascontiguousarray(I.project_tensor(f, w, w["M"] + 1).reshape(int(np.prod(n)), -1))
    return w, q


def _predict(R, w, q, prec):
    s = R.Solver(w["dim"], w["n"], w["M"], flux="burgers", cfl=w["cfl"], lo=w["lo"], hi=w["hi"],
                 precision={"fp64": R.RIDG_PREC_FP64, "fp32": R.RIDG_PREC_MIXED_FP32,
                            "tf32": R.RIDG_PREC_MIXED_TF32}[prec])
    s.set_state(q)
    dt = s.info()["dt"]
    try:
        W = s.predict()
        assert s.last_status == R.RIDG_OK
    finally:
        s.close()
    return W, dt


@pytest.mark.parametrize("dim,n", [(2, (5, 4)), (3, (3, 4, 3))])
@pytest.mark.parametrize("e", [0, -60, -100, -130, -500])
def test_fp64_states_of_any_scale(R, dim, n, e):
    w, q = _problem(dim, n)
    q = np.ldexp(q, e)
    W, dt = _predict(R, w, q, "fp64")
    # (below the absolute tolerance both sides stop after one iteration)
    ref = NL.newton_predict(q, w, dt)
    assert np.abs(W - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("prec", ["fp32", "tf32"])
def test_mixed_states_below_fp32_are_refused(R, prec):
    """lambda and the state leave FP32's range: as by the block elimination, an error, no result."""
    w, q = _problem(2, (5, 4))
    with pytest.raises(R.RidgError) as err:
        _predict(R, w, np.ldexp(q, -500), prec)
    assert err.value.status == R.RIDG_ENONFINITE
