"""How exactly vp_energy sums: grids with few columns (vy, vz), where nothing averages
out, against sums of long doubles; and values spread so widely that a plain addition
of two threads' or two warps' sums in FP64 loses part of them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = pytest.mark.skip(reason="needs a CUDA GPU")

DEV = "cuda:0"


def energy(f0, n, nv, vb):
    from paper_1206_6152_gb300 import build as B
    from paper_1206_6152_gb300.vlasov import VlasovPoisson, make_config
    B.build()
    cfg = make_config(n, nv, (0,) * 3, n, [-v for v in vb], vb, G=1.0,
                      dtype=torch.float32 if f0.dtype == np.float32 else torch.float64)
    with VlasovPoisson(cfg, torch.from_numpy(f0).to(DEV)) as sim:
        return sim.energy()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n,nv", [((1, 1, 1), (64, 1, 1)), ((128, 1, 1), (128, 1, 1)), ((1, 1, 1), (16, 16, 16)),
                                  ((2, 1, 1), (32, 32, 32)), ((1, 1, 1), (1, 1, 64)), ((4, 1, 1), (5, 1, 7)),
                                  ((16, 16, 10), (6, 7, 8)), ((16, 16, 10), (9, 5, 3))])
def test_few_columns_are_summed_to_fp64_rounding(n, nv, dtype):
    L = np.longdouble
    vb = [5.0 if k > 1 else 0.5 for k in nv]
    dv = [2 * v / k for v, k in zip(vb, nv)]
    vc = [-v + (np.arange(k) + 0.5) * d for v, k, d in zip(vb, nv, dv)]
    v2 = sum((v.astype(L) ** 2).reshape([-1 if b == a else 1 for b in range(3)]) for a, v in enumerate(vc))
    for seed in range(4):
        rng = np.random.default_rng(seed)
        f0 = (rng.random(n + nv) * np.exp(-6 * rng.random(n + nv))).astype(dtype)
        e = energy(f0, n, nv, vb)
        w = dv[0] * dv[1] * dv[2]
        M, K = f0.astype(L).sum() * w, (f0.astype(L) * v2).sum() * w / 2
        # a cell's sum and its factors dv_x dv_y dv_z, the 1/2 and |v|^2: five or six
        # roundings of 1.1e-16
        assert abs(e["M"] - M) <= 6e-16 * M
        assert abs(e["K"] - K) <= 6e-16 * K


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n,nv", [((1, 1, 1), (1, 16, 16)), ((2, 1, 1), (4, 32, 32)), ((16, 16, 16), (1, 4, 8)),
                                  ((16, 16, 16), (2, 1, 31))])
def test_threads_sums_are_merged_without_loss(n, nv, dtype):
    """One cell of 1 and the rest 2^-54: the sum is that of exact arithmetic, rounded
    once (dV is a power of two, and so is the number of cubes)."""
    f0 = np.full(n + nv, 2.0 ** -54, dtype=dtype)
    f0[..., 0, 0, 0] = 1.0
    e = energy(f0, n, nv, [k * 0.5 for k in nv])                     # dv = 1
    cells = int(np.prod(nv))
    one = 1.0 + float(np.round((cells - 1) / 4)) * 2.0 ** -52        # 1 + (cells - 1) 2^-54
    assert e["M"] == one * float(np.prod(n))


@pytest.mark.gpu
def test_cells_sums_are_added_without_loss():
    """2^-5 and 2^-58 in each of 48 runs of 128 cells, the runs that one CTA adds up:
    1.5 and three quarters of its last place, which no run's own rounded sum keeps."""
    f0 = np.zeros((16, 16, 24, 1, 1, 2))
    cells = f0.reshape(48, 128, 2)
    cells[:, 3, 0] = 2.0 ** -5
    cells[:, 90, 1] = 2.0 ** -58
    e = energy(f0, (16, 16, 24), (1, 1, 2), [0.5, 0.5, 1.0])
    assert e["M"] == 1.5 + 2.0 ** -52
