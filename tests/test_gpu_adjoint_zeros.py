"""Adjoint sweeps of FP64 lines whose empty cells are stored as +0 or -0: equal
numbers, so the same arms and the same cotangent."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

from paper_1206_6152_gb300 import inputs as I  # noqa: E402

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("space_bc", ["periodic", "outflow"])
def test_the_sign_of_zero_does_not_matter(space_bc, dtype):
    from paper_1206_6152_gb300 import build as B
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    B.build()
    w = I.small_maxwell(n=(6, 5, 4), nv=(7, 9, 6), dtype=dtype, space_bc=space_bc)
    npdt = np.float32 if dtype == "f32" else np.float64
    rng = np.random.default_rng(4)
    f0 = (rng.random(w.shape) * (rng.random(w.shape) > 0.6)).astype(npdt)
    signed = np.where((f0 == 0) & (rng.random(w.shape) < 0.5), npdt(-0.0), f0)
    lam0 = rng.normal(size=w.shape).astype(npdt)
    acc = rng.normal(size=(3,) + w.n)
    out = []
    for f in (f0, signed):
        fin = torch.from_numpy(f).to(DEV)
        with VlasovPoisson(config_of(w), fin.clone()) as sim:
            sim.set_accel(torch.from_numpy(acc))
            for axis in range(6):
                h = w.dx[axis] if axis < 3 else w.dv[axis - 3]
                v = max(abs(w.vlo[axis]), abs(w.vhi[axis])) if axis < 3 else 1.0
                lam = torch.from_numpy(lam0).to(DEV)
                sim.sweep_adjoint(axis, 0.4 * h / v, fin, lam)
                out.append(lam.cpu().numpy())
    for a, b in zip(out[:6], out[6:]):
        assert np.array_equal(a, b)
