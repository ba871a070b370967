"""The 2D mixed correction's two thread layouts (two threads per cell up to 512 cells per SM at
Q3, one above) and the groups of modes that hold none: meshes on both sides and with partly
empty last blocks, against the FP64 path."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M", [((9, 7), 3), ((273, 285), 3), ((279, 281), 3), ((9, 7), 1), ((65, 3), 2)])
@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_mixed_2d_layouts_match_fp64(n, M, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    q0 = np.random.default_rng(5).standard_normal((n[0] * n[1], (M + 1) ** 2))
    out = []
    for p in (R.RIDG_PREC_FP64, R.RIDG_PREC_MIXED_BF16 if prec == "bf16" else R.RIDG_PREC_MIXED_FP16):
        s = R.Solver(2, n, M, vel=(0.7, -0.4), cfl=0.3, precision=p)
        s.set_state(q0)
        s.step(3)
        s.sync()
        out.append(s.get_state())
        s.close()
    # six digits of 8 bits: 2^-48 of the state's maximum per product, sums of up to 64, 3 steps
    assert np.abs(out[1] - out[0]).max() <= 3 * 64 * 2.0 ** -47 * np.abs(q0).max()
