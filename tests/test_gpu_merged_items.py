"""Items of several chunks: batches large enough that the vector kernels take four chunks an item and the FP32
product several z-chunks of several layers, with ragged last items, against single solves (one chunk an item),
bitwise.  The merge factors are computed here as the engine computes them, and must exceed 1."""
import numpy as np
import pytest

from paper_2602_07354_gb300 import binding as B
from paper_2602_07354_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# grids (one whose size is no multiple of four, one no multiple of two), FP32 tiles and their layers
GRIDS = [((70, 71, 71), (15, 14, 5)), ((47, 45, 51), (15, 14, 3)), ((48, 44, 40), (11, 14, 4))]
LOADS = 6


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_07354_gb300 import build

    build.build()


def _chunks(N, mixed):
    """Number of chunks of the vector kernels."""
    up = lambda a, b: -(-a // b)  # noqa: E731
    full, chunk = (768, 768) if mixed else (512, 512 if N >= 1 << 16 else 256 if N >= 1 << 14 else 128)
    for per in range(3 if mixed else 4, 0, -1):
        wave = 152 * per
        c = up(up(N, wave * up(N, wave * 4096)), 4) * 4
        if c >= full:
            chunk = c
            break
    return up(N, chunk)


def _merge(most, count, sm):
    """The largest merge target (halved from `most`) that leaves four items an SM."""
    while most > 1 and count(most) < 4 * sm:
        most //= 2
    return most


@pytest.mark.parametrize("prec,iters", [(B.PREC_MIXED, 6), (B.PREC_MIXED, 51), (B.PREC_FP64, 9)])
def test_items_of_several_chunks_equal_single_solves(prec, iters):
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    up = lambda a, b: -(-a // b)  # noqa: E731
    n = [_chunks(int(np.prod(d)), prec == B.PREC_MIXED) for d, _ in GRIDS]
    v = _merge(4, lambda m: LOADS * sum(up(c, m) for c in n), sm)
    assert v > 1 and any(c % v for c in n)
    if prec == B.PREC_MIXED:
        xy = [up(d[0], t[0]) * up(d[1], t[1]) for d, t in GRIDS]
        z = [up(d[2], t[2]) for d, t in GRIDS]
        f = lambda m: [max(1, min(c, up(m, t[2]))) for c, (_, t) in zip(z, GRIDS)]  # noqa: E731
        fm = f(_merge(32, lambda m: LOADS * sum(a * up(c, q) for a, c, q in zip(xy, z, f(m))), sm))
        assert min(fm) > 1 and any(c % q for c, q in zip(z, fm))
    for d, t in GRIDS:
        B.elas_tuning_import(f"{d[0]} {d[1]} {d[2]} 4 {sm} {t[0]} {t[1]} {t[2]}\n")
    rng = np.random.default_rng(11)
    micros = [synth.random_problem(d, 4, rng, pore_prob=0.1) for d, _ in GRIDS]
    loads = synth.UNIT_LOAD_CASES[:LOADS]
    b = B.elas_batch_create(micros, LOADS, prec)
    infos = B.elas_batch_solve(b, np.tile(loads.reshape(-1), len(micros)), 0.0, iters)
    assert all(i["iters"] == iters for i in infos)
    for i, ms in enumerate(micros):
        ctx = B.create_from_micro(ms, prec)
        for r in range(LOADS):
            w, ref = (torch.empty(3 * ms.N, dtype=torch.float64, device="cuda") for _ in range(2))
            B.elas_batch_fluctuation(b, i, r, w)
            info = B.elas_pcg_solve(ctx, loads[r], 0.0, iters, w_out=ref)
            assert infos[LOADS * i + r]["relres_true"] == info["relres_true"]
            assert torch.equal(w, ref)
