"""The list of regions that the matrix-free Newton solver leaves to the block elimination: empty,
partly filled and full, for one mesh and for a batch in both schedules.  The lists are read in
device memory, which the tests allocate themselves."""
import numpy as np
import pytest

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


class Memory:
    """Allocator callbacks that keep their blocks as tensors."""

    def __init__(self, R):
        import torch
        self.blocks = {}

        @R.ALLOC_FN
        def alloc(nbytes, user):
            t = torch.empty(max(int(nbytes), 4), dtype=torch.uint8, device="cuda")
            self.blocks[t.data_ptr()] = (int(nbytes), t)
            return t.data_ptr()

        @R.FREE_FN
        def free(ptr, user):
            self.blocks.pop(ptr, None)

        self.callbacks = (alloc, free)

    def listed(self, cells):
        """The counts of every list with room for `cells` regions."""
        import torch
        torch.cuda.synchronize()
        return [int(t[:4].view(torch.int32)[0]) for n, t in self.blocks.values() if n == 4 * (cells + 1)]


def _prec(R, name):
    return {"fp64": R.RIDG_PREC_FP64, "fp32": R.RIDG_PREC_MIXED_FP32,
            "tf32": R.RIDG_PREC_MIXED_TF32}[name]


def _burgers(n, M, scale=1.0):
    """A smooth state whose cell means lie between 0.45 and 0.55 of scale; at twice 1e30 about half of
    the regions hold an entry above 1e30, where the iterative solver refuses them."""
    w = dict(I.burgers_ensemble(1)[0], n=n, M=M)
    f = lambda x, y: 0.5 + 0.05 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    return w, scale * np.ascontiguousarray(I.project_tensor(f, w, M + 1).reshape(-1, (M + 1) ** 2))


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-10), ("tf32", 1e-10)])
@pytest.mark.parametrize("M", [1, 2, 3, 4])
def test_partly_filled_list(R, prec, tol, M):
    n = (14, 5)
    w, q = _burgers(n, M, 2e30)
    mem = Memory(R)
    h = R.ridg_create(R.make_mesh(2, n), M, R.make_flux("burgers"), w["cfl"],
                      R.make_options(_prec(R, prec), allocator=mem.callbacks))
    R.ridg_set_state(h, q)
    W = np.empty((70, (M + 1) ** 3))
    assert R.ridg_predict(h, W) == R.RIDG_OK
    info = R.ridg_info(h)
    count, = mem.listed(70)
    assert 0 < count < 70
    assert sum(info["newton_hist"]) == 70 and info["newton_unconverged"] == 0
    R.ridg_destroy(h)
    # (Burgers scales: the prediction is 2e30 times that of the state at scale one)
    w1, q1 = _burgers(n, M)
    s = R.Solver(2, n, M, flux="burgers", cfl=w["cfl"])
    s.set_state(q1)
    ref = 2e30 * s.predict()
    s.close()
    cells = np.arange(70)[::1 if M < 3 else 9]
    oracle = NL.newton_predict(q, w, info["dt"], cells=cells)
    assert np.abs(W - ref).max() <= tol * np.abs(ref).max()
    assert np.abs(W[cells] - oracle).max() <= tol * np.abs(oracle).max()


@pytest.mark.parametrize("prec", ["fp64", "fp32", "tf32"])
@pytest.mark.parametrize("schedule", [0, 1])
@pytest.mark.parametrize("newton_tol", [0.0, 1e-30])
def test_batch_lists(R, prec, schedule, newton_tol, tmp_path):
    """(Even numbers of cells per degree: no other block has a list's size.)  Three degrees, two
    instances each, one of them at the scale where about half of its regions go
    on the list; or every region, at a tolerance that none meets: each degree's list holds the
    regions of the right instance, and the states after a step are those of single handles."""
    p = _prec(R, prec)
    f = tmp_path / "schedule.txt"
    f.write_text(f"batch.schedule flux{R.RIDG_FLUX_BURGERS} prec{p} {schedule}\n")
    R.ridg_tune_load(str(f))
    big = 1.0 if newton_tol else 2e30
    shapes = [((7, 5), 1, 1.0), ((14, 5), 2, big), ((6, 7), 3, 1.0), ((13, 5), 1, big),
              ((4, 9), 2, 1.0), ((13, 6), 3, big)]
    cases = [_burgers(*x) for x in shapes]
    mem = Memory(R)
    opt = R.make_options(p, newton_tol=newton_tol, allocator=mem.callbacks)
    b = R.ridg_batch_create([R.make_mesh(2, n) for n, _, _ in shapes], [M for _, M, _ in shapes],
                            R.make_flux("burgers"), cases[0][0]["cfl"], opt)
    assert R.ridg_batch_schedule(b)["schedule"] == schedule
    for i, (_, q) in enumerate(cases):
        R.ridg_batch_set_state(b, i, q)
    R.ridg_batch_step(b, 1)
    st = R.ridg_batch_sync(b)
    assert st == (R.RIDG_ENOCONV if newton_tol else R.RIDG_OK)
    for M in (1, 2, 3):
        cells = [n[0] * n[1] for n, m, _ in shapes if m == M]
        count, = mem.listed(sum(cells))
        assert count == sum(cells) if newton_tol else 0 < count < max(cells), M
    for i, ((n, M, scale), (w, q)) in enumerate(zip(shapes, cases)):
        out = np.empty_like(q)
        R.ridg_batch_get_state(b, i, out)
        info = R.ridg_info(R.ridg_batch_instance(b, i))
        assert sum(info["newton_hist"]) == n[0] * n[1]
        assert info["newton_unconverged"] == (n[0] * n[1] if newton_tol else 0)
        s = R.Solver(2, n, M, flux="burgers", cfl=w["cfl"], precision=p)
        s.set_state(q / scale)
        s.step(1)
        assert s.sync() == R.RIDG_OK
        ref = s.get_state()
        s.close()
        # both are within the Newton tolerance of the regions' fixed points
        assert np.abs(out / scale - ref).max() <= 1e-10, (i, M)
    R.ridg_batch_destroy(b)


@pytest.mark.parametrize("dim,instance", [(2, 6), (2, 7), (2, 0), (2, 10), (3, 2)])
def test_stalled_solves_start_anew(R, dim, instance):
    """States some of whose linear solves stall: without the restart from a residual orthogonal to the
    shadow vector 2, 1 and (3D) 5 regions went to the list (instances 6, 7; 3D), without the second
    shadow vector 1 each of instances 0 and 10.  None does."""
    if dim == 2:
        w = dict(I.burgers_ensemble()[instance], M=4, n=(72, 72))
        q, prec = I.initial_state(w), "fp64"
    else:
        w = dict(flux="burgers", dim=3, n=(10, 11, 9), M=1, lo=(0.0,) * 3, hi=(1.0,) * 3, cfl=0.3)
        rng = np.random.default_rng(instance)
        a, ph, ks = rng.uniform(.1, .5, 3), rng.uniform(0, 6, 3), rng.integers(-2, 3, (3, 3))
        f = lambda x, y, z: 0.3 + sum(a[j] / 2 * np.cos(2 * np.pi * (ks[j, 0] * x + ks[j, 1] * y + ks[j, 2] * z)
                                                       + ph[j]) for j in range(3))
        q, prec = np.ascontiguousarray(I.project_tensor(f, w, 2)[:, 0, :]), "fp32"
    cells = int(np.prod(w["n"]))
    mem = Memory(R)
    h = R.ridg_create(R.make_mesh(dim, w["n"], w["lo"], w["hi"]), w["M"], R.make_flux("burgers"), w["cfl"],
                      R.make_options(_prec(R, prec), allocator=mem.callbacks))
    R.ridg_set_state(h, q)
    assert R.ridg_predict(h) == R.RIDG_OK
    assert mem.listed(cells) == [0]
    R.ridg_destroy(h)
