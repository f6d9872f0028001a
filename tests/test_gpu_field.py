"""The field chain of a split step (density -> potential -> g, the timestep and
the kick tables from it) against the FP64 oracle at the grids where its line
kernels can go wrong: every radix, several stages of one odd radix, axes of one
cell, more lines than one CTA takes, lines that do not fill their CTAs, and the
zero-padded rows and planes of the isolated solve."""
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
@pytest.mark.parametrize("bc,n", [
    ("periodic", (1, 9, 4)), ("periodic", (27, 1, 2)), ("periodic", (128, 1, 1)),
    ("periodic", (3, 11, 7)), ("periodic", (26, 25, 14)), ("periodic", (48, 40, 36)),
    ("isolated", (2, 2, 2)), ("isolated", (5, 6, 7)), ("isolated", (16, 13, 22)),
])
def test_field_and_timestep_match_oracle(bc, n):
    h = 0.5 * np.array(n) / max(n)                       # cubic cells
    w = I.small_maxwell(n=n, nv=(4, 4, 4), dtype="f64", amp=0.0, modes=(), G=30.0,
                        box_lo=tuple(-h), box_hi=tuple(h), poisson_bc=bc,
                        space_bc="outflow" if bc == "isolated" else "periodic")
    f0 = I.initial_condition(w) * np.random.default_rng(5).uniform(0.5, 1.5, n + (1, 1, 1))
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    f = torch.from_numpy(f0).to(DEV)
    ref = O.Simulation(f0, O.Grid.of(w), O.Params.of(w))
    with VlasovPoisson(config_of(w), f) as sim:
        for steps in (0, 1, 2):
            # FP64 throughout: rounding of the sums and of up to 4 stages
            if steps:
                t = sim.step(steps, sync=True)
                ref.step(steps)
                assert abs(t - ref.t) <= 1e-12 * ref.t
                assert np.abs(f.cpu().numpy() - ref.f).max() <= 1e-12 * ref.f.max()
            _, phi, g = (x.cpu().numpy() for x in sim.field())
            phi_o = O.potential_in_box(ref.phi, ref.grid)
            assert np.abs(phi - phi_o).max() <= 1e-12 * np.abs(ref.phi).max()
            assert np.abs(g - ref.g).max() <= 1e-11 * np.abs(ref.g).max()
