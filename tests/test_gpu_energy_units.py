"""M and K (vp_energy) do not depend on the unit of velocity: boxes whose |v|^2, or
its product with f, lies far outside the FP32 range, single-cell velocity axes at
v = 0, against sums of long doubles."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

DEV = "cuda:0"


def moments(f, vc, dvol):
    """sum f dV and sum f |v|^2 dV / 2 in long double."""
    L = np.longdouble
    f = f.astype(L)
    v2 = sum((v.astype(L) ** 2).reshape([-1 if b == a else 1 for b in range(3)]) for a, v in enumerate(vc))
    return f.sum() * dvol, (f * v2).sum() * dvol / 2


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("unit,scale", [(1e-18, 1.0), (1e15, 1.0), (1e25, 1e-3), (1e7, 1e24), (1e-9, 1e-9),
                                        (1e-9, 1e20)])
@pytest.mark.parametrize("n,nv", [((16, 16, 10), (7, 5, 8)), ((2, 3, 1), (9, 12, 10)), ((4, 1, 1), (33, 1, 1))])
def test_energy_in_any_unit_of_velocity(n, nv, unit, scale, dtype):
    from paper_1206_6152_gb300 import build as B
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, make_config
    B.build()
    np_t = np.float32 if dtype == "f32" else np.float64
    rng = np.random.default_rng(2)
    f0 = (rng.random(n + nv) * np.exp(-6 * rng.random(n + nv)) * scale).astype(np_t)
    f0[0] = 0.0                                                      # empty cells
    vb = [5.0 * unit if k > 1 else 0.5 * unit for k in nv]
    # (the field plays no part: a G that keeps U finite)
    cfg = make_config(n, nv, (0,) * 3, n, [-v for v in vb], vb, G=1e-30,
                      dtype=torch.float32 if dtype == "f32" else torch.float64)
    with VlasovPoisson(cfg, torch.from_numpy(f0).to(DEV)) as sim:
        e = sim.energy()
    dv = [2 * v / k for v, k in zip(vb, nv)]
    vc = [-v + (np.arange(k) + 0.5) * d for v, k, d in zip(vb, nv, dv)]
    M, K = moments(f0, vc, dv[0] * dv[1] * dv[2])
    assert abs(e["M"] - M) <= 1e-14 * M
    assert abs(e["K"] - K) <= 1e-14 * K
