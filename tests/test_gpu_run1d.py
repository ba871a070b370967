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
