"""States and predictions in the caller's device memory: every address that a copy takes is taken
(doubles at 4 and 8 bytes past a 16-byte boundary), and a correction after such a prediction does
not depend on the caller's buffer."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,M,prec", [(1, (33,), 4, "fp64"), (1, (200003,), 2, "fp64"),
                                          (2, (9, 7), 3, "bf16"), (2, (131, 129), 3, "fp64"),
                                          (2, (131, 129), 3, "bf16"), (3, (5, 4, 6), 2, "fp64"),
                                          (3, (9, 7, 8), 1, "bf16"), (3, (31, 33, 35), 1, "bf16"),
                                          (3, (31, 29, 27), 2, "bf16")])
@pytest.mark.parametrize("offset", [0, 4, 8])
def test_any_device_address_gives_the_host_bits(dim, n, M, prec, offset):
    """The prediction of a state handed over from a device address into another one, and the state
    after the correction, have the bits of the same calls on host arrays; the caller overwrites
    the prediction before the correction."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    p = {"fp64": R.RIDG_PREC_FP64, "bf16": R.RIDG_PREC_MIXED_BF16}[prec]
    cells, ths, tht = int(np.prod(n)), (M + 1) ** dim, (M + 1) ** (dim + 1)
    q = np.random.default_rng(11).standard_normal((cells, ths))

    def solver():
        return R.Solver(dim, n, M, vel=(0.7, -0.4, 0.3)[:dim], cfl=0.2, precision=p)
    s = solver()
    s.set_state(q)
    W = s.predict()
    s.correct()
    q1 = s.get_state()
    s.close()

    s = solver()
    src = torch.empty(q.nbytes + 16, dtype=torch.uint8, device="cuda")
    dst = torch.empty(8 * cells * tht + 16, dtype=torch.uint8, device="cuda")
    src[offset:offset + q.nbytes] = torch.from_numpy(q.view(np.uint8).reshape(-1)).cuda()
    torch.cuda.synchronize()
    assert R._lib.ridg_set_state(s.h, C.c_void_p(src.data_ptr() + offset), 1) == R.RIDG_OK
    assert R._lib.ridg_predict(s.h, C.c_void_p(dst.data_ptr() + offset), 1) == R.RIDG_OK
    s.sync()
    got = dst[offset:offset + 8 * cells * tht].cpu().numpy().view(np.float64).reshape(cells, tht)
    np.testing.assert_array_equal(got, W)
    dst.fill_(255)                      # (NaN)
    torch.cuda.synchronize()
    s.correct()
    np.testing.assert_array_equal(s.get_state(), q1)
    s.close()


def test_a_prediction_that_stays_is_one_kernel():
    """Without a buffer of the caller's a linear prediction is its kernel alone (the correction reads
    it in place); at degree 0 in 1D that is the step's prediction kernel."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    s = R.Solver(1, (1000000,), 0, vel=(0.7,), cfl=0.2)
    s.set_state(np.random.default_rng(1).standard_normal((s.cells, 1)))
    s.profile_step(2)
    kernel = min(s.profile_step(5)["predict_ms"] for _ in range(3))
    times = []
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(s.stream)
        R.ridg_predict(s.h)
        b.record(s.stream)
        b.synchronize()
        times.append(a.elapsed_time(b))
    s.close()
    # (with a pass over the prediction for its time means: twice as long)
    assert min(times) <= 1.4 * kernel, (min(times), kernel)
