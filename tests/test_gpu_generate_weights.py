"""Grain assignment with strongly unequal semi-axes (ratios 1e2 to 1e6, inside the FP32 screen) against
the brute-force oracle: the heavy seed lies just outside a tile, beside the corner voxel that is farthest
from the light seed within, so that it wins that voxel by less than the rounding of its FP32 bound."""
import numpy as np
import pytest

from paper_2602_07354_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS = (16, 16, 16)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07354_gb300 import build

    build.build()


def _pair(rng, ratio):
    """A seed of axes 1 about the centre of the tile [0, 8)^3 and one of axes 1 / ratio outside a corner."""
    off = rng.uniform(-1, 1, 3) * rng.choice([0.0, 1.0])
    corner, out = np.where(off > 0, 0.5, 7.5), np.where(off > 0, -1.0, 1.0)
    n = np.abs(rng.normal(size=3)) * (rng.random(3) < 0.6) + (0, 0, 1e-9)
    gap = np.linalg.norm(corner - 4.0 - off) / ratio * (1.0 - np.exp(rng.uniform(np.log(1e-7), np.log(1e-3))))
    return np.stack([4.0 + off, np.mod(corner + out * n / np.linalg.norm(n) * gap, 16.0)])


def _check(oracle, seeds, semi):
    ph = B.elas_assign_grains(DIMS, seeds, semi)
    torch.cuda.synchronize()
    assert np.array_equal(ph.cpu().numpy(), oracle.assign_grains(DIMS, seeds, semi))


def test_a_heavy_seed_beyond_a_tile_keeps_its_voxel(oracle):
    seeds = np.array([[4.0, 4.0, 4.0], [7.500606182903449, 7.5, 7.5]])
    semi = np.array([[1.0, 1.0], [1e-4, 1e-4]])
    assert oracle.assign_grains(DIMS, seeds, semi).reshape(16, 16, 16)[7, 7, 7] == 1
    _check(oracle, seeds, semi)


@pytest.mark.parametrize("ratio", [1e2, 1e3, 5e3, 1e4, 1e5, 1e6])
@pytest.mark.parametrize("extra", [0, 30])
def test_unequal_weights_equal_the_oracle(oracle, ratio, extra):
    rng = np.random.default_rng(int(np.log10(ratio) * 10) + extra)
    for _ in range(25):
        seeds, semi = _pair(rng, ratio), np.array([[1.0, 1.0], [1.0 / ratio, 1.0 / ratio]])
        if rng.random() < 0.3:
            semi[1, rng.integers(2)] = np.exp(-rng.uniform(0, np.log(ratio)))
        if extra:  # seeds of every weight around
            seeds = np.concatenate([seeds, rng.random((extra, 3)) * 16.0])
            semi = np.concatenate([semi, np.exp(-rng.uniform(0, np.log(ratio), (extra, 2)))])
        _check(oracle, seeds, semi)
