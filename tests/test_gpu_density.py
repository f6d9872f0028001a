"""The FP32 density of a state against NumPy's FP64 sums at the cube sizes where
its loads change: one load per thread, the first size whose loads are batched
(with and without a multiple of 4), remainders after whole batches."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

from paper_1206_6152_gb300 import inputs as I  # noqa: E402


@pytest.mark.gpu
@pytest.mark.parametrize("nv", [(3, 5, 7), (12, 13, 13), (23, 89, 1), (25, 82, 1), (31, 33, 47), (16, 16, 31),
                                (16, 16, 32), (41, 50, 4), (48, 48, 48)])
def test_density_matches_fp64_sum(nv):
    from paper_1206_6152_gb300 import build as B
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, config_of
    B.build()
    w = I.small_maxwell(n=(3, 2, 4), nv=nv, dtype="f32")
    rng = np.random.default_rng(math.prod(nv))
    f0 = (rng.random(w.shape) * np.exp(-12 * rng.random(w.shape))).astype(np.float32)
    dv = math.prod((b - a) / n for a, b, n in zip(w.vlo, w.vhi, nv))
    with VlasovPoisson(config_of(w), torch.from_numpy(f0).to("cuda:0")) as sim:
        rho = sim.density().cpu().numpy()
    ref = f0.astype(np.float64).sum(axis=(3, 4, 5)) * dv
    # pairs of floats carry about 44 bits through the sum
    assert np.abs(rho - ref).max() <= 1e-12 * ref.max()
