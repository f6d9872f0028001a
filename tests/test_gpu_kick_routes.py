"""FP64 kicks, whose kernel is chosen by the estimated cost of the whole call: a half
kick and a fused kick are bit for bit the vx, vy and vz sweeps one by one, whichever
kernels these take, and lose the same mass; whole cubes, lines and cells are the
cheapest in turn, below and above a whole cell's shift."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("cells", [0.8, 2.6])
@pytest.mark.parametrize("n,nv", [((4, 4, 4), (9, 10, 11)), ((8, 8, 8), (6, 7, 8)), ((4, 4, 4), (6, 6, 6)),
                                  ((3, 3, 3), (33, 2, 2)), ((128, 1, 1), (64, 1, 1)), ((16, 16, 10), (12, 9, 10)),
                                  ((4, 1, 1), (70, 5, 3)), ((2, 1, 1), (1, 1, 1))])
def test_kicks_are_their_sweeps(n, nv, cells):
    from paper_1206_6152_gb300 import build as B
    from paper_1206_6152_gb300._lib import check
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, make_config
    B.build()
    cfg = make_config(n, nv, (0,) * 3, n, (-1,) * 3, (1,) * 3, G=1e-3, dtype=torch.float64)
    rng = np.random.default_rng(8)
    f0 = torch.from_numpy(rng.random(n + nv) * (rng.random(n + nv) > 0.1)).to(DEV)
    # shifts of up to `cells` cells along each axis, both directions
    acc = rng.uniform(-1, 1, size=(3,) + n) * np.array([2 * cells / k for k in nv]).reshape(3, 1, 1, 1)
    f = f0.clone()
    with VlasovPoisson(cfg, f) as sim:
        sim.set_accel(torch.from_numpy(acc))
        for tau2 in (0.0, 0.7):
            f.copy_(f0)
            m0 = sim.energy()["M_out"]
            for tau in (1.0, tau2) if tau2 else (1.0,):
                for axis in (3, 4, 5):
                    sim.sweep(axis, tau)
            want, m1 = f.clone(), sim.energy()["M_out"]
            f.copy_(f0)
            check(sim.lib.vp_kick(sim._ctx, 1.0, tau2), "vp_kick")
            assert torch.equal(f, want)
            # the same losses, added up in another order
            m2 = sim.energy()["M_out"]
            assert abs((m2 - m1) - (m1 - m0)) <= 1e-13 * m2
