"""Stress kernel at the edges of its tiles against the oracle: ragged tiles, grids narrower than a
tile, one-layer and many-layer items, with and without each output.  Bound: the centroid gradient and
C eps are sums of at most 24 and 6 rounded terms, so a relative error of 1e-13 leaves two digits."""
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


@pytest.mark.parametrize("dims", [(2, 2, 2), (2, 3, 200), (67, 5, 3), (33, 70, 9), (130, 2, 17), (40, 41, 43)])
def test_tiles_match_the_oracle(oracle, dims):
    rng = np.random.default_rng(sum(dims))
    ms = synth.random_problem(dims, 4, rng, pore_prob=0.15)
    p = oracle.Problem.from_micro(ms)
    e6 = np.array([2e-4, -1e-4, 1e-3, 3e-4, -2e-4, 5e-4])
    w = 1e-3 * rng.normal(size=3 * p.N)
    s_ref, vm_ref, macro_ref = p.stress(e6, w)
    ctx = B.create_from_micro(ms)
    wd = torch.from_numpy(w).cuda()
    s, vm = (torch.full((k * p.N,), float("nan"), dtype=torch.float64, device="cuda") for k in (6, 1))
    macro = B.elas_stress(ctx, e6, wd, s, vm)
    close = lambda a, b: np.linalg.norm(np.ravel(a) - np.ravel(b)) <= 1e-13 * np.linalg.norm(np.ravel(b))  # noqa: E731
    assert close(s.cpu().numpy(), s_ref) and close(vm.cpu().numpy(), vm_ref)
    assert np.abs(macro - macro_ref).max() <= 1e-13 * np.abs(s_ref).max()
    only = torch.empty_like(vm)
    assert B.elas_stress(ctx, e6, wd, None, only, want_macro=False) is None
    assert torch.equal(only, vm) and np.array_equal(B.elas_stress(ctx, e6, wd), macro)
