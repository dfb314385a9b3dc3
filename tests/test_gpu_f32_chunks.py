"""The FP32 product's items of several z-chunks: problems that share launches march merged chunks and
must give bitwise what they give alone (one chunk an item), at chunk counts that do not divide, ragged
tiles and grids of one chunk; and tiles recorded for wider blocks are kept in the tuning text but not
launched."""
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


@pytest.mark.parametrize("iters", [1, 7])
def test_merged_chunks_equal_single_solves(iters):
    dims = [(33, 31, 70), (17, 9, 5), (40, 44, 37), (64, 20, 3), (2, 3, 90)]
    rng = np.random.default_rng(3)
    micros = [synth.random_problem(d, 4, rng, pore_prob=0.1) for d in dims]
    loads = synth.UNIT_LOAD_CASES[:2]
    b = B.elas_batch_create(micros, 2, B.PREC_MIXED)
    B.elas_batch_solve(b, np.tile(loads.reshape(-1), len(dims)), 0.0, iters)
    for i, ms in enumerate(micros):
        ctx = B.create_from_micro(ms, B.PREC_MIXED)
        for r in range(2):
            w, ref = (torch.empty(3 * ms.N, dtype=torch.float64, device="cuda") for _ in range(2))
            B.elas_batch_fluctuation(b, i, r, w)
            B.elas_pcg_solve(ctx, loads[r], 0.0, iters, w_out=ref)
            assert torch.equal(w, ref)


def test_wide_tiles_of_earlier_records_are_kept_but_not_launched(oracle):
    dims, sm = (37, 26, 11), torch.cuda.get_device_properties(0).multi_processor_count
    line = f"{dims[0]} {dims[1]} {dims[2]} 4 {sm} 17 20 4"  # 378 columns
    B.elas_tuning_import(line + "\n")
    assert line in B.elas_tuning_export().splitlines()
    ms = synth.random_problem(dims, 3, np.random.default_rng(4), pore_prob=0.1)
    u = np.random.default_rng(5).normal(size=3 * ms.N).astype(np.float32)
    y = torch.empty(3 * ms.N, dtype=torch.float32, device="cuda")
    B.elas_apply_f32(B.create_from_micro(ms, B.PREC_MIXED), torch.from_numpy(u).cuda(), y)
    ref = oracle.Problem.from_micro(ms).apply(u.astype(np.float64))
    assert np.linalg.norm(y.cpu().numpy() - ref) <= 2e-6 * np.linalg.norm(ref)
