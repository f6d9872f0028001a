"""The x drift with the fused density on lines of 48 in the form that long runs take
(line pairs, CTAs of more than a hundred turns): f bit for bit that of the drift
without the density, columns of it against the FP64 oracle, the density against FP64
sums of that f, and the mass that leaves through outflow faces."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

from oracle import vp_oracle as O  # noqa: E402

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("space_bc", ["periodic", "outflow"])
def test_pairs_of_long_runs(space_bc):
    from paper_1206_6152_gb300 import build as B
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, make_config
    B.build()
    n, nv = (48, 49, 50), (30, 31, 28)              # 12 GB of f: one CTA per (y, z) column
    parts = -(-16 * torch.cuda.get_device_properties(0).multi_processor_count // (n[1] * n[2]))
    if int(np.prod(nv)) // 2 // parts <= 100 * 128:
        pytest.skip("more SMs than this size is meant for")
    dx, vb, tau = 1.0, (3.0, 3.1, 2.8), 0.21
    cfg = make_config(n, nv, (0,) * 3, [k * dx for k in n], [-v for v in vb], vb, G=1e-300, dt_fixed=tau,
                      space_bc=space_bc, dtype=torch.float32)
    gen = torch.Generator(device=DEV).manual_seed(6)
    f0 = torch.rand(n + nv, device=DEV, generator=gen)
    f0 *= torch.rand(n + (1, 1, 1), device=DEV, generator=gen) > 0.1       # empty cells
    f = f0.clone()
    dv = [2 * v / k for v, k in zip(vb, nv)]
    w = dv[0] * dv[1] * dv[2]
    cells = [(0, 0), (31, 17), (48, 49)]
    with VlasovPoisson(cfg, f) as sim:
        none = torch.zeros((3,) + n, dtype=torch.float64, device=DEV)
        sim.set_accel(none)
        sim.sweep(2, tau)
        sim.sweep(1, tau)
        before = [f[:, j, k].double().cpu().numpy() for j, k in cells]
        sim.sweep(0, tau)
        swept, lost = f.clone(), sim.energy()["M_out"]
        f.copy_(f0)
        del f0
        sim.set_accel(none)
        sim.step(1)
        lost_step = sim.energy()["M_out"] - lost
        assert torch.equal(f, swept)
        rho = sim.field()[0]
        assert torch.allclose(rho, f.flatten(3).sum(-1, dtype=torch.float64) * w, rtol=1e-13, atol=0.0)
    vx = -vb[0] + (np.arange(nv[0]) + 0.5) * dv[0]
    for (j, k), line in zip(cells, before):
        ref = np.ascontiguousarray(line.reshape((n[0], 1, 1) + nv))
        O.sweep(ref, 0, vx, tau, dx, space_bc == "periodic")
        # one rounding of each flux and update in FP32
        assert np.abs(swept[:, j, k].cpu().numpy() - ref[:, 0, 0]).max() <= 2e-6
    # (each thread adds the losses of its 102 turns of two lines in FP32)
    assert abs(lost_step - lost) <= 204 * 6e-8 * lost if space_bc == "outflow" else lost_step == 0.0
