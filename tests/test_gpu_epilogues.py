"""Epilogues of the tensor-memory GEMM at every token tile: SiLU(gate) * up in registers, alone and shared with the converting warps
(single accumulator, last tile), and routing weights that are fetched two tiles ahead."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_19438_b200 import binding as qg, synth
from tests import util

pytestmark = pytest.mark.gpu


@pytest.fixture(params=[128, 192, 256])
def tile(request):
    qg.set_schedule(request.param, 0)
    yield request.param
    qg.set_schedule(0, -1)


@pytest.mark.parametrize("qbits", [8, 4])
@pytest.mark.parametrize("M,F", [(1, 64), (15, 192), (17, 64), (129, 192), (193, 128), (257, 64), (400, 320)])
def test_gate_up(tile, qbits, M, F):
    """Tokens around the edges of 16-token blocks and of the tiles, odd numbers of row tiles (a pair's second one is past the end)."""
    A, Wq, Ws = synth.dense_problem(qbits, M, 2 * F, 512, seed=31)
    g = util.Guarded((M, F), torch.bfloat16)
    qg.qgemm_dense_gate_up_silu(qbits, util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws), out=g.t)
    qg.poll_status()
    assert g.intact() and not bool(g.untouched_inside().any().item())
    util.assert_close(util.host_bf16_f64(g.t), orc.silu_mul(orc.qgemm_dense(qbits, A, Wq, Ws)), "gate/up")


@pytest.mark.parametrize("qbits", [8, 4])
@pytest.mark.parametrize("sizes", [(0, 1, 130, 0, 200, 391), (16, 15, 17), (500,)], ids=["ragged", "blocks", "one"])
def test_routing_weights_over_many_tiles_per_pair(tile, qbits, sizes):
    """One to five tiles per pair (N = 10240 and 264): weights of tiles j, j + 1 and pairs of tile j + 2 are on their way together, and a
    tile may belong to another expert than the one before."""
    E, R, K = len(sizes), sum(sizes), 256
    rng = np.random.default_rng(5)
    off = np.concatenate(([0], np.cumsum(sizes))).astype(np.int32)
    pairs, w = rng.permutation(R).astype(np.int32), rng.random(R).astype(np.float32)
    for N in (10240, 264):
        A, Wq, Ws = synth.dense_problem(qbits, R, E * N, K, seed=37)
        Wq, Ws = Wq.reshape(E, N, -1), Ws.reshape(E, N, -1)
        g = util.Guarded((R, N), torch.bfloat16)
        qg.moe_grouped_qgemm(qg.MODE_DOWN_WEIGHTED, qbits, util.dev_bf16(A), util.dev(off), util.dev(Wq), util.dev_f16(Ws),
                             topk_w=util.dev(w), row_pair=util.dev(pairs), out=g.t)
        qg.poll_status()
        assert g.intact() and not bool(g.untouched_inside().any().item())
        ref = orc.grouped_gemm(qbits, orc.bf16_to_f64(A), off, Wq, Ws) * w[pairs][:, None].astype(np.float64)
        util.assert_close(util.host_bf16_f64(g.t), ref, f"weighted, N = {N}")
