"""The pore overwrite where a voxel lies half a cell from the pore's centre to within FP32 rounding: its
minimum image is the FP64 one, also in frames that are not rotations, whose sum depends on the image."""
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


@pytest.mark.parametrize("dims", [(8, 8, 8), (8, 9, 10), (24, 20, 22)])
@pytest.mark.parametrize("gap", [0.0, 1e-9, -1e-9, 1e-7, -1e-7, 1e-5])
def test_half_cell_images_equal_the_oracle(oracle, dims, gap):
    rng = np.random.default_rng(sum(dims) + int(1e10 * abs(gap)))
    n, most = np.array(dims, float), 0.4999 * min(dims)
    for q in range(20):
        c = np.floor(rng.random(3) * (n - 1)) + 0.5 - gap  # voxels at n/2 + gap
        a = most * np.array([0.5, 1.0, 1.0])               # (the box of ceil(max a) + 1 covers the short sides)
        R = np.zeros((3, 3))
        if q == 0:
            c, R[0, 0], R[1, 0], R[2, 2] = np.array([0.5 - gap, 0.0, 0.0]), 0.5, 0.5, 1.0
        elif q % 2:
            R = rng.uniform(-1, 1, (3, 3))  # sheared: the image of one component changes the sum
        else:
            R = np.linalg.qr(rng.normal(size=(3, 3)))[0]
        pore = np.concatenate([c, a[rng.permutation(3)] if q else a, R.ravel()])[None]
        ph = torch.zeros(int(n.prod()), dtype=torch.int32, device="cuda")
        got = B.elas_stamp_pores(dims, pore, ph)
        ref = np.zeros(int(n.prod()), np.int32)
        oracle.stamp_pores(dims, pore, ref)
        ref[~_box(dims, pore[0])] = 0
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
