"""Adjoint sweeps of lines of any length (one line per thread in registers)
against the FP64 oracle: the shortest and longest lines they take and one
beyond on each side (the shared-memory kernel), the last length of each register
size and the first of the next (that the Poisson solver takes, for drifts), even row pitches, last CTAs that are not full,
lines of both directions in a warp, both boundary rules, and lines shifted by a
cell or more beside the others."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

from oracle import vp_oracle as O  # noqa: E402
from paper_1206_6152_gb300 import inputs as I  # noqa: E402

DEV = "cuda:0"


def compare(w, axis, taus, seed):
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    rng = np.random.default_rng(seed)
    npdt = np.float32 if w.dtype == "f32" else np.float64
    f0 = (rng.random(w.shape) + 0.05).astype(npdt)
    acc = rng.normal(size=(3,) + w.n)
    grid, per = O.Grid.of(w), w.space_bc == "periodic"
    fin = torch.from_numpy(f0).to(DEV)
    with VlasovPoisson(config_of(w), fin.clone()) as sim:
        sim.set_accel(torch.from_numpy(acc))
        for tau in taus:
            lam0 = rng.normal(size=w.shape).astype(npdt)
            lam = torch.from_numpy(lam0).to(DEV)
            lg = torch.zeros((3,) + w.n, dtype=torch.float64, device=DEV)
            sim.sweep_adjoint(axis, tau, fin, lam, lg)
            ref = lam0.astype(np.float64)
            ds = np.zeros(int(np.prod(w.n)))
            f64 = f0.astype(np.float64)
            if axis < 3:
                O.sweep_adjoint(f64, ref, axis, grid.vc(axis), tau, grid.dx[axis], per, None)
            else:
                O.sweep_adjoint(f64, ref, axis, acc[axis - 3], tau, grid.dv[axis - 3], False, ds)
            # a few roundings of each term in the storage type; an arm that a rounding
            # flips (odds of one rounding per cell) changes its cell by its own size
            err = np.abs(lam.cpu().numpy().astype(np.float64) - ref).sum() / np.abs(ref).sum()
            assert err <= (1e-14 if w.dtype == "f64" else 1e-6), (axis, tau, err)
            if axis >= 3:
                gg = lg.cpu().numpy()[axis - 3].reshape(-1)
                errg = np.abs(gg - ds).sum() / np.abs(ds).sum()
                assert errg <= (1e-12 if w.dtype == "f64" else 1e-5), (axis, tau, errg)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("n", [2, 3, 16, 18, 33, 64, 65])
def test_drift_adjoint_lines_match_oracle(n, dtype):
    for axis in range(3):
        for bc in ("periodic", "outflow"):
            shape = [2, 1, 3]
            shape[axis] = n
            w = I.small_maxwell(n=tuple(shape), nv=(5, 7, 6), dtype=dtype, space_bc=bc)
            vm = max(abs(v) for v in w.vhi)
            dx = (w.box_hi[axis] - w.box_lo[axis]) / n
            compare(w, axis, [0.9 * dx / vm, -1.6 * dx / vm], seed=n + axis)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("n", [2, 3, 16, 17, 33, 64, 65])
def test_kick_adjoint_lines_match_oracle(n, dtype):
    for axis in range(3, 6):
        nv = [10, 18, 14]
        nv[axis - 3] = n
        w = I.small_maxwell(n=(3, 2, 4), nv=tuple(nv), dtype=dtype)
        dv = (w.vhi[axis - 3] - w.vlo[axis - 3]) / n
        # accelerations of both signs, up to about 2.5: with the second tau some
        # cubes shift by a cell or more
        compare(w, axis, [0.3 * dv, -0.8 * dv], seed=n + axis)
