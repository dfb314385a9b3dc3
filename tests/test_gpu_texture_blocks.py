"""Seeding and orientations of more grains than one launch has one-warp blocks for: every grain has the bits
that it has in a call of its own part."""
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


@pytest.mark.parametrize("n", [4096 * 32, 4096 * 32 + 1, 1_500_001])
def test_large_calls_equal_their_parts(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    z = torch.randn(n, 2, generator=g, device="cuda", dtype=torch.float64)
    u = torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64)
    args = ([0.0, 0.0, 0.0], [50.0, 60.0, 70.0], 11.0, 2.75, 3.18, 0.6)
    seeds, semi = B.elas_seed_grains(*args, z, u)
    rho = [B.elas_orientations(t, u) for t in (B.TEXTURE_RANDOM, B.TEXTURE_FIBER)]
    for lo, hi in ((0, 5), (4096 * 32 - 40, min(n, 4096 * 32 + 40)), (n - 333, n)):
        part = B.elas_seed_grains(*args, z[lo:hi].contiguous(), u[lo:hi].contiguous())
        assert torch.equal(part[0], seeds[lo:hi]) and torch.equal(part[1], semi[lo:hi])
        for t, full in zip((B.TEXTURE_RANDOM, B.TEXTURE_FIBER), rho):
            assert torch.equal(B.elas_orientations(t, u[lo:hi].contiguous()), full[lo:hi])
