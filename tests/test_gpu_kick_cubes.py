"""Kicks of FP32 cubes of edge 48 and 32 against the FP64 oracle with more work
than the device has SMs, so that a CTA takes several slabs or cubes in turn and
fetches ahead, a last turn that is not full, and cubes shifted by a cell or more
among them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

from oracle import vp_oracle as O  # noqa: E402
from paper_1206_6152_gb300 import inputs as I  # noqa: E402

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("edge,n,halves", [(48, (1, 1, 1), 1), (48, (5, 4, 3), 1), (48, (5, 4, 3), 2),
                                           (32, (1, 1, 1), 2), (32, (5, 8, 4), 2)])
def test_kick_of_cubes_matches_oracle(edge, n, halves):
    from paper_1206_6152_gb300 import build as B
    from paper_1206_6152_gb300._lib import check
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    B.build()
    w = I.small_maxwell(n=n, nv=(edge,) * 3, dtype="f32")
    grid = O.Grid.of(w)
    rng = np.random.default_rng(5)
    f0 = (rng.random(w.shape) * (rng.random(w.shape) > 0.1)).astype(np.float32)
    acc = rng.uniform(-1, 1, size=(3,) + w.n)
    acc.reshape(3, -1)[:, ::7] *= 1.9
    tau = 0.95 * min(grid.dv)
    f = torch.from_numpy(f0).to(DEV)
    with VlasovPoisson(config_of(w), f) as sim:
        sim.set_accel(torch.from_numpy(acc))
        check(sim.lib.vp_kick(sim._ctx, tau, 0.8 * tau * (halves - 1)), "vp_kick")
        got = f.cpu().numpy().astype(np.float64)
    ref = f0.astype(np.float64)
    for half, axis in [(h, a) for h in range(halves) for a in (3, 4, 5)]:
        O.sweep(ref, axis, acc[axis - 3], (1.0, 0.8)[half] * tau, grid.dv[axis - 3], False)
    # one rounding of each flux and update per sweep
    assert np.abs(got - ref).max() <= halves * 3 * 2e-6 * f0.max()
    assert got.min() >= 0.0
