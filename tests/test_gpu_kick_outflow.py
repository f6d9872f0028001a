"""The mass that leaves through the velocity faces (M_out) in FP32 kicks of cubes
whose vx planes have a kernel of a compile-time edge, against the FP64 oracle:
edges whose pairs of planes are (48, 64) and are not (40, 56) a whole number of
warps of lines, a last block of one plane, sweeps below a cell, of more, and past
the whole line."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

from oracle import vp_oracle as O  # noqa: E402
from paper_1206_6152_gb300 import inputs as I  # noqa: E402

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("cells", [0.7, 1.6, 3.3, 70.0])
@pytest.mark.parametrize("nv", [(37, 40, 40), (25, 48, 48), (19, 56, 56), (15, 64, 64)])
def test_outflow_of_plane_kicks_matches_oracle(nv, cells):
    from paper_1206_6152_gb300 import build as B
    from paper_1206_6152_gb300._lib import check
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    B.build()
    w = I.small_maxwell(n=(3, 2, 1), nv=nv, dtype="f32")
    grid = O.Grid.of(w)
    rng = np.random.default_rng(sum(nv))
    f0 = rng.random(w.shape).astype(np.float32)              # mass in every face cell
    acc = rng.choice([-1.0, 1.0], size=(3,) + w.n) * rng.uniform(0.6, 1.0, size=(3,) + w.n)
    tau = cells * min(grid.dv)
    f = torch.from_numpy(f0).to(DEV)
    with VlasovPoisson(config_of(w), f) as sim:
        sim.set_accel(torch.from_numpy(acc))
        got = []
        for axes in ((4,), (5,), (3, 4, 5)):
            f.copy_(torch.from_numpy(f0))
            lost0 = sim.energy()["M_out"]
            if len(axes) == 1:
                sim.sweep(axes[0], tau)
            else:
                check(sim.lib.vp_kick(sim._ctx, tau, 0.0), "vp_kick")
            got.append((sim.energy()["M_out"] - lost0) / (grid.dvol_x * grid.dvol_v))
    for axes, lost_g in zip(((4,), (5,), (3, 4, 5)), got):
        ref = f0.astype(np.float64)
        lost = sum(O.sweep(ref, a, acc[a - 3], tau, grid.dv[a - 3], False) for a in axes)
        # every cell that leaves carries at most three sweeps' roundings in FP32,
        # each 2e-6 of the largest value (here the values are of its order)
        assert abs(lost_g - lost) <= 1e-5 * lost, axes
