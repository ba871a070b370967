"""1D runs: in chunks of several steps per launch, in one block, or as two kernels per step, whichever
is the faster.  The states are the two kernels' bit for bit on both sides of every rule, and a run
takes no longer than its steps one kernel at a time."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _solver(n, M, vel=1.0):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    return R.Solver(1, (n,), M, vel=(vel,), cfl=0.45)


@pytest.mark.parametrize("vel", [1.0, -0.6])
@pytest.mark.parametrize("n,M,steps", [(3, 11, 1), (16, 3, 2), (60, 11, 1), (62, 11, 1), (63, 11, 1),
                                       (190, 3, 1), (191, 3, 1), (150, 2, 3), (16, 0, 5), (45599, 3, 6),
                                       (45601, 3, 6), (30001, 7, 3), (20011, 5, 1), (300007, 1, 4)])
def test_runs_are_the_step_kernels(n, M, steps, vel):
    q0 = np.random.default_rng(7).standard_normal((n, M + 1))
    out = []
    for run in (True, False):
        s = _solver(n, M, vel)
        s.set_state(q0)
        if run:
            s.step(steps)
            s.step(1)
            s.step(2)
        else:
            s.profile_step(steps + 3)
        out.append(s.get_state())
        s.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("n,M", [(100000, 11), (300000, 6), (600, 7)])
def test_runs_are_no_slower_than_their_kernels(n, M):
    import torch
    s = _solver(n, M)
    s.set_state(np.random.default_rng(2).standard_normal((n, M + 1)))
    s.profile_step(2)
    apart = min(s.profile_step(10)["step_ms"] for _ in range(3))
    s.step(20)
    s.sync()
    times = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(s.stream)
        s.step(20)
        b.record(s.stream)
        b.synchronize()
        times.append(a.elapsed_time(b) / 20)
    s.close()
    # (chunks took 1.5 times as long at 100000 cells Q11, twice at 300000 Q6)
    assert min(times) <= 1.1 * apart, (min(times), apart)


def test_long_runs_replay_one_graph():
    """A run of many steps takes the states of short ones and no device memory for its launches."""
    import torch
    q0 = np.random.default_rng(7).standard_normal((16, 3))
    s, t = _solver(16, 2), _solver(16, 2)
    for x in (s, t):
        x.set_state(q0)
        x.step(100)
        x.sync()
    s.step(40000)                       # 4 x 8192 and a rest
    for _ in range(400):
        t.step(100)
    assert s.info()["steps"] == t.info()["steps"] == 40100
    assert s.info()["t"] == 100 * s.info()["dt"] + 40000 * s.info()["dt"]
    np.testing.assert_array_equal(s.get_state(), t.get_state())
    free = torch.cuda.mem_get_info()[0]
    s.step(400000)
    s.sync()
    assert free - torch.cuda.mem_get_info()[0] < 64 << 20      # (one graph: 230 MB)
    s.close()
    t.close()
