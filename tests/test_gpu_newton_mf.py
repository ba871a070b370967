"""The matrix-free Newton solver of the mixed precisions (k_newton_mf.cuh) at the edges of its
range: the smallest meshes (every region wraps onto itself), every degree and both fluxes,
and the hand-over of regions that it leaves to the block elimination."""
import numpy as np
import pytest

from paper_2101_01231_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# both precisions stop when the last update is below 1e-10 and contract by at least 10 per
# solve, as the FP64 form does: the same fixed point to the tolerance of the existing parity
# tests
TOL = 1e-11


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg
    return ridg


def _smooth(flux, n, M):
    """A well-resolved state on a small mesh (low wave numbers, small amplitude)."""
    if flux == "euler":
        w = I.workload("euler2d_n512_q2", n=n, M=M)
        c = np.array([1.0, 0.3, -0.2, 2.5])

        def f(x, y):
            p = 0.02 * np.sin(2 * np.pi * x / 10) + 0.01 * np.cos(2 * np.pi * y / 10)
            return np.stack([c[j] + (1 + 0.3 * j) * p for j in range(4)])
        return w, np.ascontiguousarray(I.project_tensor(f, w, M + 1, m=4).reshape(-1, 4 * (M + 1) ** 2))
    w = dict(I.burgers_ensemble(1)[0], M=M, n=n)
    f = lambda x, y: 0.5 + 0.05 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    return w, np.ascontiguousarray(I.project_tensor(f, w, M + 1).reshape(-1, (M + 1) ** 2))


def _predict(R, w, q, prec, **kw):
    s = R.Solver(2, w["n"], w["M"], flux=w["flux"], cfl=w["cfl"], lo=w["lo"], hi=w["hi"],
                 gamma=w.get("gamma", 1.4), precision=prec, **kw)
    s.set_state(q)
    W = s.predict()
    info, status = s.info(), s.last_status
    s.close()
    return W, info, status


@pytest.mark.parametrize("flux,M", [("burgers", 1), ("burgers", 2), ("burgers", 3), ("burgers", 4),
                                    ("euler", 1), ("euler", 2)])
@pytest.mark.parametrize("n", [(3, 3), (5, 17)])
def test_matrix_free_matches_fp64(R, flux, M, n):
    w, q = _smooth(flux, n, M)
    ref, _, st = _predict(R, w, q, R.RIDG_PREC_FP64)
    assert st == R.RIDG_OK
    for prec in (R.RIDG_PREC_MIXED_FP32, R.RIDG_PREC_MIXED_TF32):
        W, info, st = _predict(R, w, q, prec)
        assert st == R.RIDG_OK and info["newton_unconverged"] == 0
        assert sum(info["newton_hist"]) == n[0] * n[1]
        assert np.abs(W - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("flux,M", [("burgers", 1), ("burgers", 2), ("burgers", 3), ("burgers", 4),
                                    ("euler", 1), ("euler", 2)])
@pytest.mark.parametrize("scale", [1.0, 1e-3])
def test_fp64_newton_path_is_the_block_eliminations(R, flux, M, scale):
    """FP64: with a tolerance that no iterate meets, every region goes to the block elimination
    and stops at the cap; the matrix-free Newton's own iterates, stopped by the default
    tolerance, count the same iterations as the oracle and agree to round-off (the linear
    systems are solved to FP64 accuracy whatever the state's scale)."""
    from oracle import nonlinear as NL
    w, q = _smooth(flux, (4, 5), M)
    if flux == "burgers":
        q = scale * q
    W, info, st = _predict(R, w, q, R.RIDG_PREC_FP64)
    direct, dinfo, dst = _predict(R, w, q, R.RIDG_PREC_FP64, newton_tol=1e-30)
    assert st == R.RIDG_OK and dst == R.RIDG_ENOCONV and dinfo["newton_hist"][4] == 20
    assert np.abs(W - direct).max() <= 1e-12 * np.abs(direct).max()
    cells = np.arange(20)[:: 1 if M < 3 else 7]
    _, it, conv = NL.newton_predict(q, w, info["dt"], cells=cells, return_iters=True, chunk=4)
    assert conv.all()
    assert info["newton_iters_max"] >= it.max() and info["newton_hist"][it.max()] >= 1


@pytest.mark.parametrize("flux,M", [("burgers", 2), ("burgers", 4), ("euler", 2)])
def test_regions_left_over_are_block_eliminated(R, flux, M):
    # a tolerance below round-off: no region converges, every one goes through the list to the
    # block elimination, which stops them at its cap
    w, q = _smooth(flux, (7, 5), M)
    ref, _, _ = _predict(R, w, q, R.RIDG_PREC_FP64)
    for prec in (R.RIDG_PREC_MIXED_FP32, R.RIDG_PREC_MIXED_TF32):
        W, info, st = _predict(R, w, q, prec, newton_tol=1e-30)
        assert st == R.RIDG_ENOCONV
        assert info["newton_unconverged"] == 35 and info["newton_hist"][4] == 35
        assert np.abs(W - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("flux,M", [("burgers", 1), ("burgers", 2), ("burgers", 3), ("burgers", 4),
                                    ("euler", 1), ("euler", 2)])
@pytest.mark.parametrize("n", [(3, 3), (7, 11)])
def test_correction_matches_oracle(R, flux, M, n):
    """The sum-factorised correction from a given prediction, on meshes that leave its last block
    partly empty.  Both sides are FP64 sums of a few hundred terms of size |Q|: 1e-13."""
    from oracle import nonlinear as NL
    w, q = _smooth(flux, n, M)
    s = R.Solver(2, w["n"], M, flux=w["flux"], cfl=w["cfl"], lo=w["lo"], hi=w["hi"],
                 gamma=w.get("gamma", 1.4), precision=R.RIDG_PREC_MIXED_FP32)
    s.set_state(q)
    W = s.predict()
    dt = s.info()["dt"]
    s.correct()
    q1 = s.get_state()
    s.close()
    ref = NL.correct(q, W, w, dt)
    assert np.abs(q1 - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("flux,M", [("burgers", 2), ("euler", 1)])
def test_first_call_of_a_step_count_equals_its_replay(R, flux, M):
    """The steps of a call are launched one by one the first time and replayed as a graph from
    the second: the same kernels in the same order, so the same bits."""
    w, q = _smooth(flux, (6, 5), M)
    s = R.Solver(2, w["n"], M, flux=flux, cfl=w["cfl"], lo=w["lo"], hi=w["hi"],
                 gamma=w.get("gamma", 1.4))
    s.set_state(q)
    for _ in range(3):                  # direct, captured, replayed
        s.step(2)
    assert s.sync() == R.RIDG_OK
    t = R.Solver(2, w["n"], M, flux=flux, cfl=w["cfl"], lo=w["lo"], hi=w["hi"],
                 gamma=w.get("gamma", 1.4))
    t.set_state(q)
    t.step(6)
    assert t.sync() == R.RIDG_OK
    np.testing.assert_array_equal(s.get_state(), t.get_state())
    s.close()
    t.close()


@pytest.mark.parametrize("flux,M,dim", [("burgers", 2, 2), ("euler", 1, 2), ("burgers", 1, 3)])
def test_fp64_regions_at_the_cap_keep_newtons_iterate(R, flux, M, dim):
    """FP64 regions stopped by the iteration cap are kept as the matrix-free solver leaves them:
    the oracle's iterate after as many steps (tolerance as the converged parity), all counted
    as unconverged."""
    from oracle import nonlinear as NL
    if dim == 2:
        w, q = _smooth(flux, (3, 4), M)
    else:
        w = dict(flux=flux, dim=3, n=(3, 3, 4), M=M, lo=(0.0,) * 3, hi=(1.0,) * 3, cfl=0.3)
        f = lambda x, y, z: 0.3 + 0.1 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * (y - z))
        q = np.ascontiguousarray(I.project_tensor(f, w, 2)[:, 0, :])
    s = R.Solver(dim, w["n"], M, flux=flux, cfl=w["cfl"], lo=w["lo"], hi=w["hi"],
                 gamma=w.get("gamma", 1.4), newton_max_iters=2)
    s.set_state(q)
    dt = s.info()["dt"]
    cells = int(np.prod(w["n"]))
    Wd = s.predict()
    assert s.last_status == R.RIDG_ENOCONV
    info = s.info()
    s.close()
    ref = NL.newton_predict(q, w, dt, max_iters=2)
    assert info["newton_unconverged"] == cells and info["newton_iters_max"] == 2
    assert np.abs(Wd - ref).max() <= 1e-12 * np.abs(ref).max()
