"""The x drift with the fused density on lines of 48 and 64 cells (one line per
thread, density sums by lane pairs) against the FP64 oracle: fewer pairs of
velocity cells than a CTA takes, several turns with the last not full, both
boundary rules, velocity rows that a pair straddles."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

from oracle import vp_oracle as O  # noqa: E402
from paper_1206_6152_gb300 import inputs as I  # noqa: E402

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("nx,n,nv,space_bc", [
    (48, (2, 1), (2, 3, 6), "periodic"), (48, (2, 1), (2, 3, 6), "outflow"),
    (64, (1, 2), (6, 5, 11), "periodic"), (64, (1, 2), (6, 5, 11), "outflow"),
    (48, (50, 50), (5, 18, 3), "periodic")])
def test_step_with_fused_density_matches_oracle(nx, n, nv, space_bc):
    from paper_1206_6152_gb300 import build as B
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    B.build()
    w = I.small_maxwell(n=(nx,) + n, nv=nv, dtype="f32", amp=0.3, space_bc=space_bc)
    # one step of less than a cell on every axis
    grid = O.Grid.of(w)
    w = w.replace(dt_fixed=0.45 * min(h / max(abs(a), abs(b)) for h, a, b in zip(grid.dx, w.vlo, w.vhi)))
    f0 = I.initial_condition(w)
    ref = O.Simulation(f0.astype(np.float64), grid, O.Params.of(w))
    ref.step(1)
    f = torch.from_numpy(f0).to(DEV)
    with VlasovPoisson(config_of(w), f) as sim:
        sim.step(1)
        rho = sim.field()[0].cpu().numpy()
        # nine sweeps, one rounding of each flux and update in FP32 per sweep
        assert np.abs(f.cpu().numpy() - ref.f).max() <= 9 * 2e-6 * f0.max()
        # (the kicks before and after move nothing between positions)
        assert np.abs(rho - ref.rho).max() <= 2e-6 * ref.rho.max()
