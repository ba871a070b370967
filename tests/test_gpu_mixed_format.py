"""The corrections' digit format is a constant of the kernel (or read at run time): both formats take
the same steps bit for bit at every digit count, on meshes to both sides of each rule (3D Q2 at six
slices: 816 bytes per cell within L2 or beyond; 2D Q3: one or two threads per cell), and stay with
the FP64 path."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,M,slices", [(2, (9, 7), 1, 2), (2, (65, 3), 2, 5), (2, (9, 7), 3, 7),
                                            (2, (283, 281), 3, 2), (2, (283, 281), 3, 5),
                                            (2, (283, 281), 3, 6), (3, (9, 7, 8), 1, 4),
                                            (3, (9, 7, 8), 2, 2), (3, (9, 7, 8), 2, 4),
                                            (3, (9, 7, 8), 2, 6), (3, (57, 55, 59), 2, 6)])
def test_formats_take_the_same_steps(dim, n, M, slices):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    q0 = torch.from_numpy(np.random.default_rng(5).standard_normal((int(np.prod(n)), (M + 1) ** dim)))
    out = []
    for p in (R.RIDG_PREC_MIXED_BF16, R.RIDG_PREC_MIXED_FP16, R.RIDG_PREC_FP64):
        s = R.Solver(dim, n, M, vel=(0.7, -0.4, 0.5)[:dim], cfl=0.2, precision=p, slices=slices)
        s.set_state(q0.cuda())
        s.step(3)
        assert s.sync() == R.RIDG_OK
        out.append(s.get_state())
        s.close()
    assert np.array_equal(out[0], out[1])
    # digits of 8 bits: 2^(-8 slices) of the state's maximum per product, sums of up to theta_S 2^d
    # of them, three steps
    terms = (M + 1) ** dim * 2 ** dim
    bound = 3 * terms * 2.0 ** (1 - 8 * slices) + 1e-13
    assert np.abs(out[0] - out[2]).max() <= bound * np.abs(q0.numpy()).max()


def test_3d_six_slices_at_64_cubed_takes_less_than_scaled_from_96():
    """Per cell, a step of a mesh just beyond L2 costs no more than one far beyond."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    us = {}
    for n in (64, 96):
        s = R.Solver(3, (n, n, n), 2, vel=(0.8, -0.5, 0.3), cfl=0.2,
                     precision=R.RIDG_PREC_MIXED_BF16, slices=6)
        s.set_state(torch.randn(n ** 3, 27, dtype=torch.float64, device="cuda"))
        s.profile_step(4)
        us[n] = min(s.profile_step(6)["correct_ms"] for _ in range(4)) / n ** 3
        s.close()
    # (the runtime flag: 176 us at 64^3 against 474 at 96^3, 1.25 per cell; the constant: 147, 444)
    assert us[64] <= 1.18 * us[96]
