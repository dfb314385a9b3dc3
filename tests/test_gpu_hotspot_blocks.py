"""Smoothing and hotspot of small grids against the oracle, bitwise: the grids take blocks of 128, 256 and
512 columns and items of one layer and of several (fewer and more than the kernel's radius), so that the
planes beside an item reach only some of its outputs."""
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


@pytest.mark.parametrize("dims", [(13, 11, 12), (24, 25, 23), (40, 37, 41), (64, 64, 64), (90, 17, 133)])
@pytest.mark.parametrize("s", [0.4, 0.8, 1.2, 1.9])
@pytest.mark.parametrize("pores", [0.0, 0.01, 0.6])
def test_small_grids_equal_the_oracle(oracle, dims, s, pores):
    rng = np.random.default_rng(sum(dims) + int(100 * s))
    ms = synth.random_problem(dims, 2, rng, pore_prob=pores)
    vm = np.abs(rng.normal(size=ms.N))
    smax, at, sm = B.elas_hotspot(B.create_from_micro(ms), torch.from_numpy(vm).cuda(), s, neighbours=B.HOTSPOT_ALL)
    best, at_ref, ref = oracle.hotspot(dims, ms.phase, vm, s=s, r=min(4, max(1, int(np.ceil(2 * s)))), solid_only=False)
    assert np.array_equal(sm.cpu().numpy(), ref)
    assert smax == best and at == at_ref
