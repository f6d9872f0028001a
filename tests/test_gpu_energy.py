"""M, K and U (vp_energy) and the functionals' values against FP64 sums of the
same array: velocity cubes whose rows do and do not take 16-byte loads, one
warp or one CTA per cell, single-cell axes, empty cells, and values so small or
large that FP32 partial sums would under- or overflow."""
import math

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


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e36])
@pytest.mark.parametrize("n,nv", [((16, 16, 10), (3, 5, 8)), ((16, 16, 10), (7, 2, 3)),
                                  ((2, 3, 2), (12, 9, 20)), ((4, 1, 1), (33, 1, 1))])
def test_energy_matches_fp64_sums(n, nv, scale, dtype):
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    w = I.small_maxwell(n=n, nv=nv, dtype=dtype, G=1.0 / scale)
    rng = np.random.default_rng(9)
    f0 = (rng.random(w.shape) * np.exp(-6 * rng.random(w.shape)) * scale)
    f0[rng.random(n) < 0.2] = 0.0                                   # empty cells
    f0 = f0.astype(np.float32 if dtype == "f32" else np.float64)
    f = torch.from_numpy(f0).to(DEV)
    grid = O.Grid.of(w)
    f64 = f0.astype(np.float64)
    v2 = sum(np.square(grid.vc(a)).reshape([-1 if b == a else 1 for b in range(3)]) for a in range(3))
    dV = grid.dvol_x * grid.dvol_v
    M = math.fsum(f64.ravel()) * dV
    K = 0.5 * math.fsum((f64 * v2).ravel()) * dV
    ref = O.Simulation(f64, grid, O.Params.of(w))
    U = 0.5 * float((ref.rho * ref.phi).sum()) * grid.dvol_x
    with VlasovPoisson(config_of(w), f) as sim:
        e = sim.energy()
        lam = torch.empty_like(f)
        J0 = sim.functional(0, lam)
        target = torch.from_numpy(ref.rho * 0.5).to(DEV)
        J1 = sim.functional(1, lam, target)
    # FP64 totals of exact (or double-float) partial sums
    assert abs(e["M"] - M) <= 1e-14 * M
    assert abs(e["K"] - K) <= 1e-14 * K
    assert abs(e["U"] - U) <= 1e-12 * abs(U)
    if scale == 1.0:
        # (the functionals take the density of the step, whose FP32 sums have no
        # FP64 path for values near the ends of the FP32 range)
        assert abs(J0 - U) <= 1e-12 * abs(U)
        assert abs(J1 - 0.125 * float((ref.rho ** 2).sum()) * grid.dvol_x) <= 1e-13 * J1
