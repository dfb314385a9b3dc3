"""The double-float product on one-layer tiles (both voxel layers side by side) against the oracle under
forced tilings: the narrowest, one that fills half a block exactly, wider than the grid and ragged; and a
batch of thin and thick problems against single solves, bitwise."""
import numpy as np
import pytest

from paper_2602_07354_gb300 import binding as B
from paper_2602_07354_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS = (13, 11, 6)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07354_gb300 import build

    build.build()


@pytest.mark.parametrize("tx,ty", [(4, 2), (5, 7), (13, 11), (15, 11), (31, 5)])
def test_thin_tiles_match_the_oracle(oracle, tx, ty):
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    B.elas_tuning_import(f"{DIMS[0]} {DIMS[1]} {DIMS[2]} 8 {sm} {tx} {ty} 1\n")
    ms = synth.random_problem(DIMS, 4, np.random.default_rng(tx + ty), pore_prob=0.15)
    p = oracle.Problem.from_micro(ms)
    u = np.random.default_rng(5).normal(size=3 * p.N)
    ctx = B.create_from_micro(ms)
    y = torch.empty(3 * p.N, dtype=torch.float64, device="cuda")
    B.elas_apply(ctx, torch.from_numpy(u).cuda(), y)
    ref = p.apply(u)
    assert np.linalg.norm(y.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
    e6 = np.array([0.0, 4e-4, 1e-3, 0.0, 2e-4, 0.0])
    ref = p.pcg(e6, 1e-10, 3000)
    w = torch.empty_like(y)
    info = B.elas_pcg_solve(ctx, e6, 1e-10, 3000, w_out=w, stop_rule=B.STOP_PRECOND)
    assert info["status"] == B.CONVERGED and abs(info["iters"] - ref["iters"]) <= 1
    assert np.linalg.norm(w.cpu().numpy() - ref["w"]) <= 1e-7 * np.linalg.norm(ref["w"])


def test_thin_tiles_give_the_bits_of_thick_ones():
    # the same sums in the same order: a column's two voxels in mode space, then four corners a node
    dims = (12, 14, 9)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    ms = synth.random_problem(dims, 5, np.random.default_rng(21), pore_prob=0.15)
    u = torch.from_numpy(np.random.default_rng(22).normal(size=3 * ms.N)).cuda()
    out = []
    for tile in ("6 7 1", "12 14 3", "12 14 1", "5 3 1"):
        B.elas_tuning_import(f"{dims[0]} {dims[1]} {dims[2]} 8 {sm} {tile}\n")
        y = torch.empty_like(u)
        B.elas_apply(B.create_from_micro(ms), u, y)
        out.append(y)
    assert all(torch.equal(y, out[1]) for y in out)


def test_thin_and_thick_problems_in_one_batch():
    rng = np.random.default_rng(8)
    micros = [synth.random_problem(d, 3, rng, pore_prob=0.1) for d in [(18, 17, 19), (40, 41, 42), (20, 20, 20)]]
    load = synth.UNIT_LOAD_CASES[2]
    b = B.elas_batch_create(micros, 1, B.PREC_FP64)
    B.elas_batch_solve(b, np.tile(load, len(micros)), 0.0, 9)
    for i, ms in enumerate(micros):
        w, ref = (torch.empty(3 * ms.N, dtype=torch.float64, device="cuda") for _ in range(2))
        B.elas_batch_fluctuation(b, i, 0, w)
        B.elas_pcg_solve(B.create_from_micro(ms), load, 0.0, 9, w_out=ref)
        assert torch.equal(w, ref)
