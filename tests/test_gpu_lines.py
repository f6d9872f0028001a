"""Sweeps of lines of any length (one line per thread in registers) against the
FP64 oracle at the lengths where those kernels can go wrong: one and two cells,
the last length of each register size and the first of the next, the longest
they take and one beyond (the shared-memory kernels), lines of both directions
in a warp, last CTAs that are not full, both boundary rules, and shifts of a
cell or more beside sub-cell ones."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

from oracle import vp_oracle as O  # noqa: E402
from paper_1206_6152_gb300 import inputs as I  # noqa: E402

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1206_6152_gb300 import build as B
    B.build()


def compare_sweep(w, axis, taus, seed):
    """One sweep per tau against the oracle; f has zeros and a wide range."""
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    rng = np.random.default_rng(seed)
    np_t = np.float32 if w.dtype == "f32" else np.float64
    f0 = (rng.random(w.shape) * np.exp(-8 * rng.random(w.shape)) * (rng.random(w.shape) > 0.1)).astype(np_t)
    acc = rng.normal(size=(3,) + w.n)
    grid, per = O.Grid.of(w), w.space_bc == "periodic"
    f = torch.from_numpy(f0).to(DEV)
    with VlasovPoisson(config_of(w), f) as sim:
        sim.set_accel(torch.from_numpy(acc))
        for tau in taus:
            f.copy_(torch.from_numpy(f0))
            lost0 = sim.energy()["M_out"]
            sim.sweep(axis, tau)
            ref = f0.astype(np.float64)
            if axis < 3:
                lost = O.sweep(ref, axis, grid.vc(axis), tau, grid.dx[axis], per)
            else:
                lost = O.sweep(ref, axis, acc[axis - 3], tau, grid.dv[axis - 3], False)
            got = f.cpu().numpy().astype(np.float64)
            # one rounding of each flux and update in the storage type
            tol = 1e-12 if w.dtype == "f64" else 2e-6
            assert np.abs(got - ref).max() <= tol * f0.max(), (axis, tau)
            assert got.min() >= 0.0
            lost_g = (sim.energy()["M_out"] - lost0) / (grid.dvol_x * grid.dvol_v)
            assert abs(lost_g - lost) <= 50 * tol * max(lost, f0.sum() * 1e-3), (axis, tau)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("space_bc", ["periodic", "outflow"])
@pytest.mark.parametrize("n", [1, 2, 15, 18, 33, 63, 65])
def test_drift_lines_match_oracle(n, space_bc, dtype):
    for axis in range(3):
        shape = [2, 3, 2]
        shape[axis] = n
        nv = (5, 7, 6)                  # 210 velocity cells: the last CTA is not full
        w = I.small_maxwell(n=tuple(shape), nv=nv, dtype=dtype, space_bc=space_bc)
        h, v = w.dx[axis], max(abs(w.vlo[axis]), abs(w.vhi[axis]))
        compare_sweep(w, axis, (0.7 * h / v, -0.97 * h / v, 2.3 * h / v), 10 * n + axis)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 32, 33, 64, 65])
def test_kick_lines_match_oracle(n, dtype):
    for axis in range(3):
        nv = [5, 6, 7]
        nv[axis] = n
        w = I.small_maxwell(n=(3, 2, 5), nv=tuple(nv), dtype=dtype)
        # accelerations of both signs: |shift| below a cell, and up to several
        h = w.dv[axis]
        compare_sweep(w, 3 + axis, (0.25 * h, -0.3 * h, 1.7 * h), 100 * n + axis)


@pytest.mark.gpu
@pytest.mark.parametrize("n,nv", [((16, 16, 10), (3, 2, 2)), ((2, 2, 3), (17, 16, 16))])
def test_fp64_density_matches_oracle(n, nv):
    """One warp per cube (many cubes) and one CTA per cube (few)."""
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    w = I.small_maxwell(n=n, nv=nv, dtype="f64")
    f0 = np.random.default_rng(3).random(w.shape) ** 20        # widely spread values
    with VlasovPoisson(config_of(w), torch.from_numpy(f0).to(DEV)) as sim:
        rho = sim.density().cpu().numpy()
    ref = O.density(f0, O.Grid.of(w))
    assert np.abs(rho - ref).max() <= 4e-16 * ref.max()


@pytest.mark.gpu
@pytest.mark.parametrize("whole_cell", [False, True])
@pytest.mark.parametrize("nv", [
    (7, 6, 5),          # one warp of lines
    (24, 28, 26),       # whole cubes, several CTAs per SM
    (37, 38, 39),       # whole cubes, one CTA per SM
    (63, 40, 30),       # blocks of vx planes, the last one not full
    (9, 64, 64), (50, 41, 37),
    # vx planes of a compile-time size, the last block of planes not full
    (37, 40, 40), (25, 48, 48), (19, 56, 56), (15, 64, 64),
])
def test_fp32_steps_of_any_cube_match_oracle(nv, whole_cell):
    """Half kicks and the fused six-sweep kick (two steps); with whole_cell
    the fixed step moves some of the cubes by more than a cell."""
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    w = I.small_maxwell(n=(4, 2, 3), nv=nv, dtype="f32", amp=0.5, G=20.0)
    ref = O.Simulation(I.initial_condition(w, np.float64), O.Grid.of(w), O.Params.of(w))
    if whole_cell:
        shift = max(np.abs(ref.g[a]).max() / w.dv[a] for a in range(3)) / 2
        w = w.replace(dt_fixed=1.6 / shift)
    f0 = I.initial_condition(w)
    ref = O.Simulation(f0.astype(np.float64), O.Grid.of(w), O.Params.of(w))
    f = torch.from_numpy(f0).to(DEV)
    with VlasovPoisson(config_of(w), f) as sim:
        sim.step(2)
        got = f.cpu().numpy().astype(np.float64)
    ref.step(2)
    # 18 sweeps, one FP32 rounding of about 6e-8 each
    assert np.abs(got - ref.f).sum() <= 4e-6 * np.abs(ref.f).sum()
    assert got.min() >= 0.0


@pytest.mark.gpu
@pytest.mark.parametrize("space_bc", ["periodic", "outflow"])
@pytest.mark.parametrize("n", [15, 18, 33, 64])
def test_fp64_many_lines_match_oracle(n, space_bc):
    """Lines that fill the GPU in whole rounds (19008 of 19456 lanes): one thread
    per line; the tests above have few lines in FP64, one thread per cell."""
    w = I.small_maxwell(n=(n, 4, 4), nv=(12, 11, 9), dtype="f64", space_bc=space_bc)
    h, v = w.dx[0], max(abs(w.vlo[0]), abs(w.vhi[0]))
    compare_sweep(w, 0, (0.7 * h / v, -0.97 * h / v), n)
    if space_bc == "outflow":
        return
    w = I.small_maxwell(n=(16, 8, 8), nv=(5, 6, n), dtype="f64")
    compare_sweep(w, 5, (0.25 * w.dv[2], -1.1 * w.dv[2]), n + 1)
    w = I.small_maxwell(n=(16, 8, 8), nv=(n, 5, 6), dtype="f64")
    compare_sweep(w, 3, (0.25 * w.dv[0], -1.1 * w.dv[0]), n + 2)


@pytest.mark.gpu
@pytest.mark.parametrize("nv", [(13, 16, 14), (14, 14, 15), (18, 18, 18), (18, 18, 19)])
def test_fp64_kick_at_the_shared_memory_limits(nv):
    """Cubes whose buffers lie around the 48 KB of shared memory a launch has
    without asking, and around the 96 KB up to which cubes take one thread per
    cell."""
    w = I.small_maxwell(n=(2, 2, 3), nv=nv, dtype="f64")
    compare_sweep(w, 3, (0.25 * w.dv[0], -1.1 * w.dv[0]), sum(nv))
