"""1D steps in chunks (several steps per launch): the states are the two step kernels' bit for
bit, for every launch count (one, odd, even), chunks that wrap around the whole mesh, meshes
that do not divide into chunks, every velocity sign and degrees up to the largest."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vel", [1.0, -0.6, 0.0])
@pytest.mark.parametrize("n,M,steps", [(3, 0, 1), (3, 3, 17), (5, 11, 2), (31, 1, 33), (601, 7, 14),
                                       (9001, 2, 5), (153, 4, 48)])
def test_chunked_steps_are_the_step_kernels(n, M, steps, vel):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    q0 = np.random.default_rng(7).standard_normal((n, M + 1))
    out = []
    for chunked in (True, False):
        s = R.Solver(1, (n,), M, vel=(vel,), cfl=0.45)
        s.set_state(q0)
        if chunked:
            s.step(steps)
            s.step(1)
        else:
            s.profile_step(steps + 1)
        out.append(s.get_state())
        s.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("dim,n,M", [(2, (5, 7), 1), (2, (83, 83), 2), (2, (84, 82), 5), (3, (19, 19, 19), 1),
                                     (3, (19, 18, 20), 3), (3, (4, 3, 5), 4)])
def test_fp64_steps_at_the_dispatch_edges(dim, n, M):
    """FP64 linear steps on meshes to both sides of 45 cells per SM (152 SMs: 6840 cells), where
    the correction changes from a thread per mode to a thread per cell, and of every block size
    of the prediction, with velocities of both signs: the oracle's states."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from oracle import linear as OL
    from paper_2101_01231_gb300 import inputs as I
    from paper_2101_01231_gb300 import ridg as R
    vel = (0.8, -0.5, 0.3)[:dim]
    w = I.workload("adv2d_n256_q3" if dim == 2 else "adv3d_n96_q2", n=n, M=M, vel=vel, cfl=0.2)
    q0 = np.random.default_rng(3).standard_normal((int(np.prod(n)), (M + 1) ** dim))
    s = R.Solver(dim, n, M, vel=vel, cfl=0.2)
    s.set_state(q0)
    dt = s.info()["dt"]
    s.step(2)
    q = s.get_state()
    s.close()
    ref = OL.run(q0, w, dt, 2)
    # two steps of sums of up to theta_S 2^d products of O(1) terms
    assert np.abs(q - ref).max() <= 2e-12 * np.abs(ref).max()
