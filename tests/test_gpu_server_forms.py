"""FP64 servers whose requests come in the product's thin form (one-layer tiles of small grids) and in the
general one: alone, together and one after the other, each request has the bits of a plain solve."""
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


@pytest.mark.parametrize("first,later", [(20, 40), (40, 20), (20, 18)])
def test_small_and_large_requests_equal_plain_solves(first, later):
    rng = np.random.default_rng(first)
    micros = [synth.random_problem((n, n + 1, n - 1), 3, rng, pore_prob=0.1) for n in (first, later, first)]
    load = synth.UNIT_LOAD_CASES[4]
    srv = B.elas_server_create(1 << 30, 4, B.PREC_FP64, iters_per_step=4)
    ids = [B.elas_server_submit(srv, micros[0], load, 0.0, 21)]
    B.elas_server_step(srv)  # alone
    ids.append(B.elas_server_submit(srv, micros[1], load, 0.0, 9))
    ids.append(B.elas_server_submit(srv, micros[2], load, 0.0, 30))
    left, got = set(range(3)), {}
    for _ in range(40):
        B.elas_server_step(srv)
        for k in list(left):
            w = torch.empty(3 * micros[k].N, dtype=torch.float64, device="cuda")
            info = B.elas_server_poll(srv, ids[k], w)
            if info is not None:
                got[k] = (info, w)
                left.discard(k)
    srv.close()
    assert not left
    for k, ms in enumerate(micros):
        w = torch.empty(3 * ms.N, dtype=torch.float64, device="cuda")
        info = B.elas_pcg_solve(B.create_from_micro(ms), load, 0.0, (21, 9, 30)[k], w_out=w)
        assert got[k][0]["iters"] == info["iters"] and got[k][0]["relres_true"] == info["relres_true"]
        assert torch.equal(got[k][1], w)
