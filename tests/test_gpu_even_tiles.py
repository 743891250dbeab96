"""Token tiles of the tensor-memory GEMM that share an expert's rows out evenly (gathered rows, fp32 sums, a short K): rows around the edges of
one, two and three tiles against the oracle, and the choice of the tile where rows are uneven."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_19438_b200 import binding as qg, synth
from tests import util

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _restore_schedule():
    yield
    qg.set_schedule(0, -1)


SIZES = [(129, 0, 193, 16), (257, 385, 1), (128, 192, 256, 17), (513, 400)]


@pytest.mark.parametrize("tile", [128, 192, 256])
@pytest.mark.parametrize("sizes", SIZES, ids=["-".join(map(str, s)) for s in SIZES])
@pytest.mark.parametrize("qbits", [8, 4])
def test_rows_around_the_edges(qbits, sizes, tile):
    """All modes, rows sorted and gathered; rows that belong to no tile of their own would show as sentinels."""
    E, R, N, K, k = len(sizes), sum(sizes), 384, 256, 4
    rng = np.random.default_rng(11)
    off = np.concatenate(([0], np.cumsum(sizes))).astype(np.int32)
    M = (R + k - 1) // k
    pairs, w = rng.permutation(M * k)[:R].astype(np.int32), rng.uniform(0.1, 1.0, M * k).astype(np.float32)
    X, Wq, Ws = synth.dense_problem(qbits, M, E * N, K, seed=41)
    Wq, Ws = Wq.reshape(E, N, -1), Ws.reshape(E, N, -1)
    A = np.ascontiguousarray(X[pairs // k])
    plain = orc.grouped_gemm(qbits, orc.bf16_to_f64(A), off, Wq, Ws)
    weighted = plain * w[pairs].astype(np.float64)[:, None]
    sums = np.zeros((M, N))
    np.add.at(sums, pairs // k, weighted)
    refs = {qg.MODE_PLAIN: plain, qg.MODE_GATE_UP_SILU: orc.silu_mul(plain), qg.MODE_DOWN_WEIGHTED: weighted, qg.MODE_DOWN_ACCUM_F32: sums}
    dev = [util.dev(off), util.dev(Wq), util.dev_f16(Ws)]
    dX, dA, dp, dw = util.dev_bf16(X), util.dev_bf16(A), util.dev(pairs), util.dev(w)
    qg.set_schedule(tile, 0)
    for mode, ref in refs.items():
        f32 = mode == qg.MODE_DOWN_ACCUM_F32
        for gathered in (False, True):
            g = util.Guarded(ref.shape, torch.float32 if f32 else torch.bfloat16, fill_inside=not f32)
            if gathered:
                qg.moe_grouped_qgemm_gather(mode, qbits, dX, dp, k, *dev, topk_w=dw, out=g.t)
            else:
                qg.moe_grouped_qgemm(mode, qbits, dA, *dev, topk_w=dw, row_pair=dp, k=k, out=g.t)
            qg.poll_status()
            assert g.intact() and (f32 or not bool(g.untouched_inside().any().item()))
            util.assert_close(g.t.double().cpu().numpy(), ref, f"mode {mode}, gathered {gathered}")


@pytest.mark.parametrize("mode,gathered,N,K", [(qg.MODE_GATE_UP_SILU, True, 1536, 2048), (qg.MODE_DOWN_WEIGHTED, True, 2048, 768),
                                               (qg.MODE_DOWN_ACCUM_F32, True, 2048, 768), (qg.MODE_DOWN_ACCUM_F32, False, 2048, 768)],
                         ids=["gate-up-gathered", "weighted-gathered", "sums-gathered", "sums"])
@pytest.mark.parametrize("qbits", [8, 4])
def test_uneven_rows_take_a_tile_that_suits_them(qbits, mode, gathered, N, K):
    """32 experts, 80 rows each on average, a quarter of them preferred: the call's own choice is within 1.1 times the faster of both tiles (192
    tokens took 1.25 to 1.31 times as long as 128; two timings of one launch differ by 2 %)."""
    E, R, k = 32, 80 * 32, 8
    p = np.where(np.arange(E) % 4 == 0, 4.5, 1.0)
    off = np.concatenate(([0], np.cumsum(np.random.default_rng(3).multinomial(R, p / p.sum())))).astype(np.int32)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    X = torch.randn((R // k if gathered else R, K), device="cuda", generator=gen).to(torch.bfloat16)
    Wq = torch.randint(-127, 128, (E, N, K), dtype=torch.int8, device="cuda", generator=gen) if qbits == 8 else \
        torch.randint(0, 256, (E, N, K // 2), dtype=torch.uint8, device="cuda", generator=gen)
    Ws = (torch.rand((E, N, K // 32), device="cuda", generator=gen) * 0.002).to(torch.float16)
    w, pairs = torch.rand(R, device="cuda", generator=gen), torch.randperm(R, device="cuda", generator=gen).to(torch.int32)
    f32 = mode == qg.MODE_DOWN_ACCUM_F32
    out = torch.zeros((R // k if f32 else R, N // 2 if mode == qg.MODE_GATE_UP_SILU else N), dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    dev = (util.dev(off), Wq, Ws)

    def call():
        if gathered:
            qg.moe_grouped_qgemm_gather(mode, qbits, X, pairs, k, *dev, topk_w=w, out=out)
        else:
            qg.moe_grouped_qgemm(mode, qbits, X, *dev, topk_w=w, row_pair=pairs, k=k, out=out)

    graphs, times = {}, {0: 1e9, 128: 1e9, 192: 1e9}
    for tile in times:
        qg.set_schedule(tile, -1)
        call()
        torch.cuda.synchronize()
        graphs[tile] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graphs[tile]):
            for _ in range(10):
                call()
    for _ in range(12):
        for tile, graph in graphs.items():
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(); graph.replay(); b.record()
            torch.cuda.synchronize()
            times[tile] = min(times[tile], a.elapsed_time(b) * 100)
    qg.poll_status()
    assert times[0] <= 1.1 * min(times.values()), times
