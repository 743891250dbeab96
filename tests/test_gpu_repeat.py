"""Sums of the GEMM calls have a fixed order: a call gives the same bits every time, whole or in slices or by stream-K, and the gathering form those
of the form for sorted rows.  (Mode 3 of the grouped call adds with atomics and is not part of this.)"""
import numpy as np
import pytest
import torch

from paper_2607_19438_b200 import binding as qg, synth
from tests import util

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _restore_schedule():
    yield
    qg.set_schedule(0, -1)


def same_every_time(call, times=6):
    outs = [call() for _ in range(times)]
    qg.poll_status()
    assert all(torch.equal(o, outs[0]) for o in outs)
    return outs[0]


@pytest.mark.parametrize("tile,streamk", [(0, -1), (128, 0), (192, 0), (256, 0), (128, 1), (192, 1), (256, 1)],
                         ids=lambda v: str(v))
@pytest.mark.parametrize("qbits,M,N,K", [(8, 700, 2560, 2048), (4, 333, 3072, 3072), (8, 300, 1032, 4096)], ids=lambda v: str(v))
def test_dense(qbits, M, N, K, tile, streamk):
    A, Wq, Ws = synth.dense_problem(qbits, M, N, K, seed=51)
    args = (util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws))
    qg.set_schedule(tile, streamk)
    same_every_time(lambda: qg.qgemm_dense(qbits, *args))


@pytest.mark.parametrize("qbits,M,N,K", [(8, 40, 2048, 4096), (4, 20, 3072, 3072), (8, 192, 512, 8192)], ids=lambda v: str(v))
def test_slices(qbits, M, N, K):
    assert qg.plan_slices(qbits, M, N, K) > 1
    A, Wq, Ws = synth.dense_problem(qbits, M, N, K, seed=52)
    args = (util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws))
    same_every_time(lambda: qg.qgemm_dense(qbits, *args))


@pytest.mark.parametrize("tile", [0, 128, 192, 256])
@pytest.mark.parametrize("qbits", [8, 4])
def test_gate_up(qbits, tile):
    A, Wq, Ws = synth.dense_problem(qbits, 517, 2 * 1088, 2048, seed=53)
    args = (util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws))
    qg.set_schedule(tile, -1)
    same_every_time(lambda: qg.qgemm_dense_gate_up_silu(qbits, *args))


@pytest.mark.parametrize("tile", [0, 128, 192, 256])
@pytest.mark.parametrize("K", [512, 1280])
@pytest.mark.parametrize("qbits", [8, 4])
def test_sorted_and_gathered_rows(qbits, K, tile):
    """K = 512: tiles of sorted rows are equally long too; K = 1280: full ones against equally long ones of the gathering form."""
    sizes, N, k = (200, 0, 130, 17, 391, 1), 768, 4
    E, R = len(sizes), sum(sizes)
    rng = np.random.default_rng(7)
    off = util.dev(np.concatenate(([0], np.cumsum(sizes))).astype(np.int32))
    M = (R + k - 1) // k
    pairs = util.dev(rng.permutation(M * k)[:R].astype(np.int32))
    w = util.dev(rng.uniform(0.1, 1.0, M * k).astype(np.float32))
    X, Wq, Ws = synth.dense_problem(qbits, M, E * N, K, seed=54)
    X, W = util.dev_bf16(X), (util.dev(Wq.reshape(E, N, -1)), util.dev_f16(Ws.reshape(E, N, -1)))
    A = X[(pairs // k).long()]
    qg.set_schedule(tile, -1)
    for mode in (qg.MODE_PLAIN, qg.MODE_GATE_UP_SILU, qg.MODE_DOWN_WEIGHTED):
        a = same_every_time(lambda: qg.moe_grouped_qgemm(mode, qbits, A, off, *W, topk_w=w, row_pair=pairs))
        b = same_every_time(lambda: qg.moe_grouped_qgemm_gather(mode, qbits, X, pairs, k, off, *W, topk_w=w))
        assert torch.equal(a, b)
