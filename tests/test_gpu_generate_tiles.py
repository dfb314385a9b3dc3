"""Grain assignment by tiles (pruned candidate lists, FP32 screen) against the brute-force oracle at
the edges of its branches: ragged tiles, cells narrower than a tile, more candidates than a tile's
list holds, windows that miss the nearest seed, near ties, and weights outside the screen's range;
and the pore overwrite at box edges, flat ellipsoids and frames that are not rotations."""
import numpy as np
import pytest

from paper_2602_07354_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07354_gb300 import build

    build.build()


def _seeds(kind, dims, rng):
    n = np.array(dims, float)
    if kind == "dense":  # about one seed per 3 voxels
        return rng.random((int(n.prod() / 3), 3)) * n
    if kind == "cluster":  # 3,000 seeds within one voxel's width, and a few elsewhere
        return np.concatenate([rng.random((3000, 3)) + np.floor(0.4 * n), rng.random((5, 3)) * n])
    if kind == "corner":  # all seeds in one corner: most tiles must look at every seed
        return rng.random((1500, 3)) * 0.2 * n
    if kind == "lattice":  # exact ties everywhere
        return np.stack(np.meshgrid(*[np.arange(0, d, 4.0) for d in dims], indexing="ij"), -1).reshape(-1, 3)
    if kind == "near":  # pairs a few 1e-9 apart: the FP32 screen cannot tell them
        s = rng.random((40, 3)) * n
        return np.concatenate([s, np.mod(s + 1e-9 * rng.standard_normal(s.shape), n)])
    return rng.random((max(1, int(n.prod() / 500)), 3)) * n


@pytest.mark.parametrize("dims", [(8, 8, 8), (9, 17, 25), (1, 40, 7), (61, 5, 33)])
@pytest.mark.parametrize("kind", ["plain", "dense", "cluster", "corner", "lattice", "near"])
@pytest.mark.parametrize("spread", [None, 0.2, 3.0, 40.0])
def test_tiles_equal_the_oracle(oracle, dims, kind, spread):
    rng = np.random.default_rng(sum(dims) + len(kind))
    seeds = _seeds(kind, dims, rng)
    semi = None if spread is None else np.exp(spread * rng.uniform(-1, 1, (len(seeds), 2)))
    ph = B.elas_assign_grains(dims, seeds, semi)
    torch.cuda.synchronize()
    assert np.array_equal(ph.cpu().numpy(), oracle.assign_grains(dims, seeds, semi))


@pytest.mark.parametrize("dims", [(20, 24, 28), (9, 40, 11), (33, 33, 33)])
def test_pore_boxes_equal_the_oracle(oracle, dims):
    rng = np.random.default_rng(sum(dims))
    n, most = np.array(dims, float), 0.4999 * min(dims)
    pores = []
    for q in range(60):
        a = np.array([most, most, most]) if q % 6 == 0 else np.minimum(most, np.exp(rng.uniform(np.log(0.05), np.log(most), 3)))
        c = np.floor(rng.random(3) * n) + (0.5 if q % 4 == 0 else rng.random())
        R = np.linalg.qr(rng.normal(size=(3, 3)))[0] if q % 3 else np.eye(3)
        if q % 10 == 7:
            R = 3.0 * rng.normal(size=(3, 3))  # any matrix is accepted
        pores.append(np.concatenate([np.minimum(c, n - 1e-3), a, R.ravel()]))
    pores = np.array(pores)
    for p in range(0, len(pores), 5):  # a few at a time, so that one wrong voxel is not covered by another pore
        ph = torch.zeros(int(n.prod()), dtype=torch.int32, device="cuda")
        got = B.elas_stamp_pores(dims, pores[p:p + 5], ph)
        ref = np.zeros(int(n.prod()), np.int32)
        for one in pores[p:p + 5]:  # voxels are looked for in the pore's box, which holds every voxel of a rotated one
            hit = np.zeros(int(n.prod()), np.int32)
            oracle.stamp_pores(dims, one[None], hit)
            ref[(hit < 0) & _box(dims, one)] = -1
        assert got == np.count_nonzero(ref)
        assert np.array_equal(ph.cpu().numpy(), ref)


def _box(dims, pore):
    """The voxels within ceil(largest semi-axis) + 1 of the centre's voxel in every dimension (periodic)."""
    ext = int(np.ceil(pore[3:6].max())) + 1
    inside = []
    for d in range(3):
        m = np.zeros(dims[d], bool)
        m[np.mod(np.arange(-ext, ext + 1) + int(np.floor(pore[d])), dims[d])] = True
        inside.append(m)
    return (inside[2][:, None, None] & inside[1][None, :, None] & inside[0][None, None, :]).ravel()
