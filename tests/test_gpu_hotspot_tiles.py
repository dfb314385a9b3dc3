"""Maximum-stress extraction at the edges of its tiles against the oracle, bitwise: ragged tiles and
z chunks, grids narrower than the kernel, every radius, windows without a solid voxel, plateaus, and
magnitudes at which the division by the full weight sum takes its general form."""
import numpy as np
import pytest

from paper_2602_07354_gb300 import binding as B
from paper_2602_07354_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07354_gb300 import build

    build.build()


def _field(kind, N, rng):
    vm = np.abs(rng.normal(size=N))
    if kind == "plateau":
        return np.round(vm * 2) / 2
    if kind == "tiny":
        return vm * 10.0 ** rng.uniform(-320, -270, N)
    if kind == "huge":
        return vm * 10.0 ** rng.uniform(270, 305, N)
    return vm


@pytest.mark.parametrize("dims", [(2, 3, 2), (70, 33, 9), (5, 4, 131), (129, 2, 3)])
@pytest.mark.parametrize("s", [0.3, 0.5, 0.8, 1.3, 2.0])
@pytest.mark.parametrize("kind,pores", [("rough", 0.02), ("rough", 0.97), ("plateau", 0.3), ("tiny", 0.05), ("huge", 0.0)])
def test_tiles_equal_the_oracle(oracle, dims, s, kind, pores):
    rng = np.random.default_rng(sum(dims) + int(100 * s))
    ms = synth.random_problem(dims, 2, rng, pore_prob=pores)
    vm = _field(kind, ms.N, rng)
    ctx = B.create_from_micro(ms)
    r = min(4, max(1, int(np.ceil(2 * s))))
    for solid in (False, True):
        smax, at, sm = B.elas_hotspot(ctx, torch.from_numpy(vm).cuda(), s, neighbours=B.HOTSPOT_SOLID if solid else B.HOTSPOT_ALL)
        best, at_ref, sm_ref = oracle.hotspot(dims, ms.phase, vm, s=s, r=r, solid_only=solid)
        assert np.array_equal(sm.cpu().numpy(), sm_ref)
        assert smax == best and at == at_ref
