"""The first call of a step count, which a nonlinear flux launches directly: it refuses the streams
that the captured calls refuse, and a batch's is its replay's bits."""
import ctypes as C

import numpy as np
import pytest

from paper_2101_01231_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg
    return ridg


@pytest.mark.parametrize("batch", [False, True])
def test_legacy_stream_is_refused_from_the_first_call(R, batch):
    w = dict(I.burgers_ensemble(1)[0], n=(5, 4), M=1)
    q = I.initial_state(w)
    opt = R.make_options(stream=C.c_void_p(1))          # cudaStreamLegacy
    mesh, flux = R.make_mesh(2, w["n"]), R.make_flux("burgers")
    if batch:
        b = R.ridg_batch_create([mesh], [1], flux, w["cfl"], opt)
        h = R.ridg_batch_instance(b, 0)
    else:
        h = R.ridg_create(mesh, 1, flux, w["cfl"], opt)
    R.ridg_set_state(h, q)
    for _ in range(2):
        with pytest.raises(R.RidgError):
            R.ridg_batch_step(b, 1) if batch else R.ridg_step(h, 1)
    out = np.empty_like(q)
    R.ridg_get_state(h, out)
    assert np.array_equal(out, q)                       # no step was taken
    R.ridg_batch_destroy(b) if batch else R.ridg_destroy(h)


def _state(w):
    if w["flux"] == "euler":
        return I.initial_state(w)
    f = lambda x, y: 0.5 + 0.05 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    return np.ascontiguousarray(I.project_tensor(f, w, w["M"] + 1).reshape(-1, (w["M"] + 1) ** 2))


@pytest.mark.parametrize("flux,degrees", [("burgers", (1, 2, 4, 2)), ("euler", (1, 2, 1))])
@pytest.mark.parametrize("prec", ["fp64", "tf32"])
def test_batch_first_call_equals_its_replay(R, flux, degrees, prec):
    if flux == "burgers":
        ws = [dict(x, n=(6 + i, 5), M=M) for i, (x, M) in enumerate(zip(I.burgers_ensemble(), degrees))]
    else:
        ws = [I.workload("euler2d_n512_q2", n=(6 + i, 5), M=M) for i, M in enumerate(degrees)]
    p = R.RIDG_PREC_FP64 if prec == "fp64" else R.RIDG_PREC_MIXED_TF32
    out = []
    for calls in ((2, 2, 2), (6,)):                     # direct, captured, replayed; direct
        b = R.ridg_batch_create([R.make_mesh(2, w["n"], w["lo"], w["hi"]) for w in ws],
                                [w["M"] for w in ws], R.make_flux(flux, gamma=1.4), ws[0]["cfl"],
                                R.make_options(precision=p))
        for i, w in enumerate(ws):
            R.ridg_batch_set_state(b, i, _state(w))
        for n in calls:
            R.ridg_batch_step(b, n)
        R.ridg_batch_sync(b)
        qs = []
        for i, w in enumerate(ws):
            q = np.empty_like(_state(w))
            R.ridg_batch_get_state(b, i, q)
            qs.append(q)
        R.ridg_batch_destroy(b)
        out.append(qs)
    for a, c in zip(*out):
        np.testing.assert_array_equal(a, c)
