"""qgemm_dense with K cut into slices that a thread-block cluster adds (few tiles): two to four slices, token tiles of 128 and 192
rows in both formats, ragged rows and tokens, against the oracle.  Each case first asks whether the call will be sliced, and
afterwards that the GPU has not refused the launch."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_19438_b200 import binding as qg, synth
from tests import util

pytestmark = pytest.mark.gpu

# slices of equal and unequal length (K = 1280: 5 units of four k-blocks), one row tile and an odd number of them, rows past
# the end in the last tile, tokens around the edges of the 16-token blocks and of the 128- and 192-token tiles
SHAPES = [(8, 17, 256, 2048), (4, 20, 3072, 3072), (8, 128, 2184, 2560), (4, 129, 1152, 1280), (8, 127, 136, 8192),
          (4, 192, 2048, 2048), (8, 333, 2048, 2048), (4, 500, 2560, 2048), (8, 193, 4096, 4096), (4, 64, 5120, 3072),
          (8, 1, 512, 1024), (4, 16, 8, 512), (8, 500, 2560, 2048), (8, 64, 136, 8192), (8, 64, 8192, 512)]
WHOLE = (8, 64, 8192, 512)                               # 32 row tiles and two units of K: two slices would fill the GPU
# (8 x 127 x 136 x 8192 was expected whole, by stream-K: 57 us there, 30 data-parallel and 13 in four slices.)


@pytest.mark.parametrize("qbits,M,N,K", SHAPES, ids=[f"q{q}-{m}x{n}x{k}" for q, m, n, k in SHAPES])
def test_slices_match_the_oracle(qbits, M, N, K):
    A, Wq, Ws = synth.dense_problem(qbits, M, N, K, seed=23)
    g = util.Guarded((M, N), torch.bfloat16)
    args = (util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws))
    planned = qg.plan_slices(qbits, M, N, K)
    assert (planned > 1) == ((qbits, M, N, K) != WHOLE)
    for _ in range(3):                                   # back to back: a launch's start overlaps the end of the one before
        qg.qgemm_dense(qbits, *args, out=g.t)
    qg.poll_status()
    assert qg.plan_slices(qbits, M, N, K) == planned     # a refused launch would not be planned again
    assert g.intact() and not bool(g.untouched_inside().any().item())
    rows = np.unique(np.concatenate([np.arange(0, N, max(1, N // 500)), np.arange(max(0, N - 140), N)]))
    util.assert_close(util.host_bf16_f64(g.t)[:, rows], orc.qgemm_dense(qbits, A, Wq[rows], Ws[rows]), "slices")


def test_a_wait_that_runs_out_in_one_slice():
    qbits, M, N, K = 8, 40, 2048, 4096
    assert qg.plan_slices(qbits, M, N, K) > 1
    A, Wq, Ws = synth.dense_problem(qbits, M, N, K, seed=24)
    args = (util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws))
    try:
        qg.test_inject(wait_limit_polls=2048, skip_kblock=K // 64 - 2)      # a k-block of the last slice
        qg.qgemm_dense(qbits, *args)
        assert qg.poll_status_code() == -7
    finally:
        qg.test_inject(0, -1)
    out = qg.qgemm_dense(qbits, *args)
    qg.poll_status()
    util.assert_close(util.host_bf16_f64(out), orc.qgemm_dense(qbits, A, Wq, Ws), "after a timeout")


def test_a_plan_needs_no_current_device_and_leaves_it_alone():
    """Planning on a fresh context, before any launch; with a second GPU, while that one is current: the plan is the same, and
    the sliced launch that follows is not refused (the plan then still names its slices)."""
    import ctypes as C
    lib, shape = qg.load(), (8, 20, 2048, 4096)
    want = qg.plan_slices(*shape)
    assert want > 1
    for dev in range(min(2, torch.cuda.device_count())):
        h, n = C.c_void_p(), C.c_int(0)
        assert lib.qg_create(C.byref(h), 0) == 0
        with torch.cuda.device(dev):
            assert lib.qg_plan_slices(h, *shape, C.byref(n)) == 0 and n.value == want
            assert torch.cuda.current_device() == dev
        A, Wq, Ws = synth.dense_problem(*shape, seed=25)
        dA, dWq, dWs, out = util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws), torch.empty((20, 2048), dtype=torch.bfloat16, device="cuda")
        assert lib.qgemm_dense(h, *shape, dA.data_ptr(), dWq.data_ptr(), dWs.data_ptr(), out.data_ptr(), None) == 0
        assert lib.qg_poll_status(h, None) == 0
        util.assert_close(util.host_bf16_f64(out), orc.qgemm_dense(8, A, Wq, Ws), "a context of its own")
        assert lib.qg_plan_slices(h, *shape, C.byref(n)) == 0 and n.value == want
        lib.qg_destroy(h)
    assert lib.qg_plan_slices(qg.context(), 8, 20, 2044, 4096, C.byref(C.c_int(0))) == -2
    assert lib.qg_plan_slices(qg.context(), *shape, None) == -1


@pytest.mark.parametrize("N,K", [(8192, 1024), (8192, 512), (6144, 1024)], ids=lambda v: str(v))
@pytest.mark.parametrize("M", [17, 128])
def test_short_k_over_many_tiles_is_not_sliced(M, N, K):
    """24 and 32 row tiles with a short K: two slices fill the GPU and the next launch cannot start early (8.8 us against 7.9
    whole, 10.1 against 8.5 at 128 tokens)."""
    assert qg.plan_slices(8, M, N, K) == 1 and qg.plan_slices(4, M, N, K) == 1
    assert qg.plan_slices(8, M, 4096, 4096) > 1 and qg.plan_slices(8, M, 5120, 3072) > 1


@pytest.mark.parametrize("qbits,M,N,K", [(8, 128, 512, 16384), (4, 192, 136, 14336), (8, 17, 1024, 16384), (4, 333, 512, 8192), (8, 150, 4096, 14336)],
                         ids=lambda v: str(v))
def test_long_k_over_few_tiles_is_sliced(qbits, M, N, K):
    """Under stream-K, whose tiles of up to 64 parts are added by one pair each, these took 71, 119, 36, 52 and 34 us; in slices 21, 19, 19,
    14 and 29."""
    assert qg.plan_slices(qbits, M, N, K) > 1


def test_the_cases_cover_every_instantiation():
    """Both formats with both token tiles, and two, three and four slices."""
    plans = {(q, qg.plan_dense(q, m, n, k)[0]) for q, m, n, k in SHAPES if (q, m, n, k) != WHOLE}
    assert plans == {(8, 128), (8, 192), (4, 128), (4, 192)}
    assert {qg.plan_slices(*s) for s in SHAPES} == {1, 2, 3, 4}
