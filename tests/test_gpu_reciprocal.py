"""The Newton residual's reciprocal against CUDA's correctly rounded one, and the states outside its
range, which end with the solvers that divide."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2101_01231_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    so = str(tmp_path_factory.mktemp("rcp") / "librcp.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-shared", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(ROOT, "paper_2101_01231_gb300", "csrc"),
                    "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "host", "reciprocal_check.cu"), "-o", so], check=True)
    lib = C.CDLL(so)

    def run(x):
        xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        r, ref = torch.empty_like(xd), torch.empty_like(xd)
        torch.cuda.synchronize()
        assert lib.reciprocal_check(C.c_void_p(xd.data_ptr()), C.c_void_p(r.data_ptr()),
                                    C.c_void_p(ref.data_ptr()), C.c_longlong(x.size)) == 0
        return r.cpu().numpy(), ref.cpu().numpy()
    return run


@pytest.mark.parametrize("emin,emax", [(-1022, 1021), (-40, 40), (-1, 1)])
def test_reciprocal_is_correctly_rounded_but_for_ties(check, emin, emax):
    """Two steps from a seed of 20 bits leave 2^-80 relative ahead of the last rounding, 2^-27 of a
    unit: another value than the correctly rounded one only where 1 / x lies that close to the
    middle of two, one x in some 2^26, and then its neighbour."""
    n = 1 << 25
    rng = np.random.default_rng(emax)
    x = np.ldexp(1.0 + rng.random(n), rng.integers(emin, emax + 1, n))
    x[::3] *= -1
    r, ref = check(x)
    off = np.abs(r.view(np.int64) - ref.view(np.int64))
    assert off.max() <= 1
    assert np.count_nonzero(off) <= 16          # (2^25 values: 0.5 expected)


def test_reciprocal_at_the_ends_of_its_range(check):
    x = np.array([2.0 ** -1022, np.ldexp(2.0 - 2.0 ** -52, 1021), 1.0, np.nextafter(1.0, 2.0),
                  np.nextafter(1.0, 0.0)])
    r, ref = check(x)
    # (the values below a power of two have reciprocals 2^-54 of a unit from the middle of two)
    assert np.abs(r.view(np.int64) - ref.view(np.int64)).max() <= 1
    r, _ = check(np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 2.0 ** -1023]))
    assert np.isnan(r).all()
    r, _ = check(np.array([1.5 * 2.0 ** 1022, 1.7e308]))
    assert (r == 0.0).all()


@pytest.mark.parametrize("e,tol", [(0, 1e-13), (1015, 1e-13), (-1022, 1e-13), (-1030, 1e-9)])
def test_states_of_any_scale(e, tol):
    """The Euler fluxes are homogeneous: a constant state stays constant at any density, also where
    its reciprocal leaves the range of the residual's (2^-1030: 44 bits of a subnormal density)."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2101_01231_gb300 import ridg as R
    w = I.workload("euler2d_n512_q2", n=(5, 4), M=1)
    q = np.zeros((20, 16))
    q[:, ::4] = np.ldexp(np.array([1.0, 0.25, -0.125, 2.5]), e)
    s = R.Solver(2, w["n"], 1, flux="euler", cfl=w["cfl"], lo=w["lo"], hi=w["hi"])
    s.set_state(q)
    s.step(2)
    assert s.sync() == R.RIDG_OK
    assert np.abs(s.get_state() - q).max() <= tol * np.abs(q).max()
    s.close()
