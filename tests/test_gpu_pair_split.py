"""The double-float operator on operands whose split into float pairs is delicate, against the oracle:
leading parts that round up into the next power of two, exact halves of the leading part's last bit,
isolated non-zeros, and a wide range of magnitudes.  The pairs keep 48 bits, so a product is within
1e-12 of the oracle's in relative L2 norm, as everywhere."""
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


def _operand(kind, n, rng):
    s = rng.choice([-1.0, 1.0], n)
    if kind == "carry":  # all leading bits set: rounding carries into the exponent
        return s * (1.0 - 2.0 ** -rng.integers(24, 53, n).astype(float)) * 2.0 ** rng.integers(-3, 4, n)
    if kind == "tie":  # exactly half a unit of the leading float's last bit
        return s * (1.0 + rng.integers(0, 2 ** 23, n) * 2.0 ** -23 + 2.0 ** -24)
    if kind == "sparse":
        return np.where(rng.random(n) < 0.01, s * rng.random(n), 0.0)
    return s * 10.0 ** rng.uniform(-25, 0, n)


@pytest.mark.parametrize("dims", [(11, 9, 7), (40, 21, 13)])
@pytest.mark.parametrize("kind", ["carry", "tie", "sparse", "range"])
def test_products_match_the_oracle(oracle, dims, kind):
    rng = np.random.default_rng(sum(dims) + len(kind))
    ms = synth.random_problem(dims, 5, rng, pore_prob=0.1)
    p = oracle.Problem.from_micro(ms)
    u = _operand(kind, 3 * p.N, rng)
    ctx = B.create_from_micro(ms)
    y = torch.empty(3 * p.N, dtype=torch.float64, device="cuda")
    B.elas_apply(ctx, torch.from_numpy(u).cuda(), y)
    ref = p.apply(u)
    assert np.linalg.norm(y.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
    w = 1e-3 * u / np.abs(u).max()
    e6 = np.array([1e-3, 0, 2e-4, 0, -3e-4, 0])
    g = torch.empty_like(y)
    B.elas_residual(ctx, e6, torch.from_numpy(w).cuda(), g)
    ref = p.apply(w) + p.rhs(e6)
    assert np.linalg.norm(g.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
