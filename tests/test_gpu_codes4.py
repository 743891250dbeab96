"""4-bit codes: every code times every finite fp16 scale, as the GEMM kernels form it, is the exact product rounded once to bf16.

One-hot activations make each output one weight, so there is nothing to sum and nothing else to round."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_19438_b200 import binding as qg
from tests import util

pytestmark = pytest.mark.gpu


def scales():
    bits = np.arange(65536, dtype=np.uint32).astype(np.uint16)
    return bits[np.isfinite(bits.view(np.float16))]


@pytest.mark.parametrize("rows", [256, 16], ids=["tensor_memory", "block"])
def test_all_codes_times_all_scales(rows):
    K = 256                                         # qgemm_dense; K = 256 sends qgemm_small_m to the block kernel
    s = scales()
    N = len(s) // 8
    Ws = np.ascontiguousarray(s[:N * 8].reshape(N, 8))
    codes = np.arange(K, dtype=np.uint8) % 16       # each 32-block holds every code twice
    Wq = np.broadcast_to((codes[0::2] | (codes[1::2] << 4)).astype(np.uint8), (N, K // 2)).copy()
    A = np.zeros((rows, K), np.uint16)
    i = np.arange(rows)
    A[i, i * (K // rows) + i % (K // rows)] = 0x3F80
    call = qg.qgemm_dense if rows > 16 else qg.qgemm_small_m
    out = util.host_bf16_bits(call(4, util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws)))
    qg.poll_status()
    k = np.argmax(A != 0, axis=1)
    w = (codes[k].astype(np.float64) - 8)[:, None] * Ws.view(np.float16).astype(np.float64)[:, k // 32].T
    ref = orc.f64_to_bf16(w)
    zero = (out & 0x7FFF) == 0                      # a zero's sign is not part of the contract
    assert np.array_equal(zero, (ref & 0x7FFF) == 0)
    assert np.array_equal(out[~zero], ref[~zero])


@pytest.mark.parametrize("shift", range(16))
def test_every_code_with_every_scale_in_the_block_kernel(shift):
    """Sixteen tokens show each scale two codes; moved on by one sixteen times, all of them."""
    K = 256
    s = scales()
    N = len(s) // 8
    Ws = np.ascontiguousarray(s[:N * 8].reshape(N, 8))
    codes = np.arange(K, dtype=np.uint8) % 16
    Wq = np.broadcast_to((codes[0::2] | (codes[1::2] << 4)).astype(np.uint8), (N, K // 2)).copy()
    k = np.arange(16) * 16 + (np.arange(16) + shift) % 16
    A = np.zeros((16, K), np.uint16)
    A[np.arange(16), k] = 0x3F80
    out = util.host_bf16_bits(qg.qgemm_small_m(4, util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws)))
    qg.poll_status()
    ref = orc.f64_to_bf16((codes[k].astype(np.float64) - 8)[:, None] * Ws.view(np.float16).astype(np.float64)[:, k // 32].T)
    zero = (out & 0x7FFF) == 0                      # a zero's sign is not part of the contract
    assert np.array_equal(zero, (ref & 0x7FFF) == 0)
    assert np.array_equal(out[~zero], ref[~zero])
