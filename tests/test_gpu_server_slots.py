"""Server slots that are used again: every request of a one-slot server, not only its first, must return
the w and the true residual of a plain solve, bit for bit, however it stops: converged in its update
(FP64), converged in a residual replacement (mixed), out of iterations between two replacements, or
cancelled."""
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


def _f64(n):
    return torch.empty(n, dtype=torch.float64, device="cuda")


def _collect(srv, rid, N, steps=400):
    w = _f64(3 * N)
    for _ in range(steps):
        B.elas_server_step(srv)
        info = B.elas_server_poll(srv, rid, w)
        if info is not None:
            return info, w
    raise AssertionError("server did not finish")


def _plain(ms, prec, strain, tol, max_iter):
    w = _f64(3 * ms.N)
    return B.elas_pcg_solve(B.create_from_micro(ms, prec), strain, tol, max_iter, w_out=w), w


def _same(got, ref):
    assert got[0]["iters"] == ref[0]["iters"] and got[0]["relres_true"] == ref[0]["relres_true"] > 0.0
    assert torch.equal(got[1], ref[1])


MICROS = [((20, 18, 22), 0.02), ((24, 24, 24), 0.0), ((15, 21, 17), 0.02)]


@pytest.mark.parametrize("prec", [B.PREC_FP64, B.PREC_MIXED])
@pytest.mark.parametrize("tol,max_iter", [(1e-8, 5000), (0.0, 7)])
def test_requests_in_a_used_slot_equal_plain_solves(prec, tol, max_iter):
    srv = B.elas_server_create(1 << 30, 1, prec)
    for k, (dims, pores) in enumerate(MICROS):
        ms = synth.polycrystal(0, 6, pore_frac=pores, seed=70 + k, dims=dims)
        strain = synth.random_symmetric_strain(np.random.default_rng(k))
        got = _collect(srv, B.elas_server_submit(srv, ms, strain, tol, max_iter), ms.N)
        assert got[0]["status"] == (B.CONVERGED if tol else B.MAX_ITER)
        _same(got, _plain(ms, prec, strain, tol, max_iter))
    srv.close()


@pytest.mark.parametrize("prec", [B.PREC_FP64, B.PREC_MIXED])
def test_cancelled_requests_in_a_used_slot_hold_their_last_iterate(prec):
    srv = B.elas_server_create(1 << 30, 1, prec, iters_per_step=8)
    for k, (dims, pores) in enumerate(MICROS):
        ms = synth.polycrystal(0, 6, pore_frac=pores, seed=80 + k, dims=dims)
        strain = synth.random_symmetric_strain(np.random.default_rng(k))
        rid = B.elas_server_submit(srv, ms, strain, 0.0, 5000)
        B.elas_server_step(srv)
        B.elas_server_step(srv)
        B.elas_server_cancel(srv, rid)
        got = _collect(srv, rid, ms.N)
        assert got[0]["status"] == B.CANCELLED and got[0]["iters"] == 16
        _same(got, _plain(ms, prec, strain, 0.0, 16))
    srv.close()
