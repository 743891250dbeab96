"""The weight-streaming kernel (a few rows per expert, or one matrix and up to sixteen tokens): the edges of its tiles, stages,
row groups and K slices, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_19438_b200 import binding as qg, synth
from tests import util

pytestmark = pytest.mark.gpu


def problem(counts, N, K, seed):
    E = len(counts)
    offsets = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    R = int(offsets[-1])
    A = synth.activations(R, K, seed, 61)
    Wq = synth.weights_q4(E * N, K, seed, 62).reshape(E, N, K // 2)
    Ws = synth.scales(E * N, K // 32, 7, seed, 63).reshape(E, N, K // 32)
    return offsets, A, Wq, Ws


# one row; the row groups of eight and the tile of sixteen from both sides; a segment cut into three tiles; empty experts first,
# in between and last; an odd number of stages, a single one, and more stages than the ring holds; ragged rows of weights
SEGMENTS = [([1], 128, 256), ([0, 7, 8, 9, 0], 384, 512), ([15, 16, 17, 0, 1, 40], 256, 768),
            ([0, 0, 3, 0, 33, 1, 0, 2], 640, 2048), ([1] * 9, 1408, 1280), ([2, 0, 5], 136, 256), ([4, 12, 6], 8, 1024)]


@pytest.mark.parametrize("mode", [qg.MODE_PLAIN, qg.MODE_GATE_UP_SILU, qg.MODE_DOWN_WEIGHTED], ids=["plain", "gateup", "weighted"])
@pytest.mark.parametrize("counts,N,K", SEGMENTS, ids=["-".join(map(str, c)) + f"_{n}_{k}" for c, n, k in SEGMENTS])
def test_short_segments(counts, N, K, mode):
    if mode == qg.MODE_GATE_UP_SILU and N % 128:
        N = (N + 127) // 128 * 128
    offsets, A, Wq, Ws = problem(counts, N, K, 4)
    R = int(offsets[-1])
    rng = np.random.default_rng(6)
    row_pair, w = rng.permutation(R).astype(np.int32), rng.uniform(0.1, 1.0, R).astype(np.float32)
    g = util.Guarded((R, N // 2 if mode == qg.MODE_GATE_UP_SILU else N), torch.bfloat16)
    out = qg.moe_grouped_qgemm(mode, 4, util.dev_bf16(A), util.dev(offsets), util.dev(Wq), util.dev_f16(Ws), topk_w=util.dev(w),
                               row_pair=util.dev(row_pair), out=g.t)
    qg.poll_status()
    ref = orc.grouped_gemm(4, orc.bf16_to_f64(A), offsets, Wq, Ws)
    if mode == qg.MODE_GATE_UP_SILU:
        ref = orc.silu_mul(ref)
    elif mode == qg.MODE_DOWN_WEIGHTED:
        ref = ref * w[row_pair].astype(np.float64)[:, None]
    util.assert_close(util.host_bf16_f64(out), ref, "short segments")
    assert g.intact()


def test_infinities_and_nan_stay_in_their_rows():
    """A row with an infinity gives what the plain sum gives (an infinity of the weight's sign where the weight is not
    zero), and no other row notices."""
    counts, N, K = [3, 2, 9], 256, 512
    offsets, A, Wq, Ws = problem(counts, N, K, 5)
    clean = qg.moe_grouped_qgemm(qg.MODE_PLAIN, 4, util.dev_bf16(A), util.dev(offsets), util.dev(Wq), util.dev_f16(Ws))
    dA = util.dev_bf16(A)
    dA[4, 77], dA[11, 3] = float("inf"), float("nan")
    out = qg.moe_grouped_qgemm(qg.MODE_PLAIN, 4, dA, util.dev(offsets), util.dev(Wq), util.dev_f16(Ws))
    qg.poll_status()
    rest = [r for r in range(14) if r not in (4, 11)]
    assert torch.equal(out[rest], clean[rest])
    assert bool(torch.isnan(out[11]).all())
    q = ((Wq[1, :, 77 // 2] >> 4).astype(np.int64) - 8) * np.sign(Ws[1, :, 77 // 32].view(np.float16).astype(np.float64))
    got, nz = out[4].float().cpu().numpy(), q != 0
    assert np.array_equal(got[nz], np.sign(q[nz]) * np.inf)


def test_a_wait_that_runs_out_is_reported_and_the_next_call_is_correct():
    counts, N, K = [5, 9, 2, 12], 512, 1024
    offsets, A, Wq, Ws = problem(counts, N, K, 7)
    args = (util.dev_bf16(A), util.dev(offsets), util.dev(Wq), util.dev_f16(Ws))
    try:
        qg.test_inject(wait_limit_polls=2048, skip_kblock=6)         # the second stage's rows are never loaded
        qg.moe_grouped_qgemm(qg.MODE_PLAIN, 4, *args)
        assert qg.poll_status_code() == -7
    finally:
        qg.test_inject(0, -1)
    out = qg.moe_grouped_qgemm(qg.MODE_PLAIN, 4, *args)
    qg.poll_status()
    util.assert_close(util.host_bf16_f64(out), orc.grouped_gemm(4, orc.bf16_to_f64(A), offsets, Wq, Ws), "after a timeout")


# one stage and an odd number of them; a slice of a single stage; ragged rows; more tiles than CTAs (tiles taken over)
# with one stage, with an odd number and with more stages than the ring holds; eight and sixteen tokens from both sides
DENSE = [(8, 1, 64, 4096), (8, 8, 72, 768), (8, 9, 264, 1280), (4, 16, 136, 256 * 7), (4, 8, 2048, 512), (8, 16, 19016, 256),
         (8, 3, 19136, 768), (4, 9, 38024, 256), (4, 7, 38144, 1280), (8, 2, 4096, 4096), (4, 1, 3072, 8192)]


@pytest.mark.parametrize("mode", [2, 3], ids=["slices", "whole-k"])
@pytest.mark.parametrize("qbits,M,N,K", DENSE, ids=[f"q{q}-{m}x{n}x{k}" for q, m, n, k in DENSE])
def test_one_matrix(qbits, M, N, K, mode):
    A, Wq, Ws = synth.dense_problem(qbits, M, N, K, seed=15)
    dA, dWq, dWs = util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws)
    g = util.Guarded((M, N), torch.bfloat16)
    qg.test_gemv_mode(mode)
    try:
        qg.qgemm_small_m(qbits, dA, dWq, dWs, out=g.t)
        again = [qg.qgemm_small_m(qbits, dA, dWq, dWs) for _ in range(3)]
        qg.poll_status()
    finally:
        qg.test_gemv_mode(0)
    assert g.intact() and not bool(g.untouched_inside().any().item())
    assert all(torch.equal(g.t, a) for a in again)
    rows = np.unique(np.concatenate([np.arange(0, N, max(1, N // 700)), np.arange(max(0, N - 140), N)]))
    util.assert_close(util.host_bf16_f64(g.t)[:, rows], orc.qgemm_dense(qbits, A, Wq[rows], Ws[rows]), "one matrix")


def test_every_8_bit_code_is_exact():
    """Unit tokens and unit scales: the output is the code itself, for all 256 codes at every position of a 32-block."""
    N, K = 256, 1024
    Wq = ((np.arange(N)[:, None] + 37 * np.arange(K)[None, :]) % 256 - 128).astype(np.int8)
    Ws = np.full((N, K // 32), np.float16(1).view(np.uint16))
    for k0 in range(0, 32, 16):
        A = torch.zeros((16, K), dtype=torch.bfloat16, device="cuda")
        ks = [(k0 + m) + 32 * ((5 * m + k0) % 32) for m in range(16)]
        for m, k in enumerate(ks):
            A[m, k] = 1.0
        out = qg.qgemm_small_m(8, A, util.dev(Wq), util.dev_f16(Ws))
        qg.poll_status()
        assert np.array_equal(util.host_bf16_f64(out), Wq[:, ks].T.astype(np.float64))


def test_an_infinite_token_gives_infinities_of_the_codes_signs():
    M, N, K = 3, 512, 1024
    A, Wq, Ws = synth.dense_problem(8, M, N, K, seed=16)
    dA = util.dev_bf16(A)
    clean = qg.qgemm_small_m(8, dA, util.dev(Wq), util.dev_f16(Ws))
    dA[1, 500] = float("-inf")
    out = qg.qgemm_small_m(8, dA, util.dev(Wq), util.dev_f16(Ws))
    qg.poll_status()
    assert torch.equal(out[[0, 2]], clean[[0, 2]])
    q = Wq[:, 500].astype(np.int64) * np.sign(Ws[:, 500 // 32].view(np.float16).astype(np.float64))
    assert np.array_equal(out[1].float().cpu().numpy()[q != 0], -np.sign(q[q != 0]) * np.inf)


def test_expert_gemms_on_two_streams_at_once():
    """Launches that overlap deal out their tiles independently."""
    counts, N, K = [3, 7, 1, 12, 0, 5] * 8, 1536, 1024
    offsets, A, Wq, Ws = problem(counts, N, K, 9)
    args = (util.dev_bf16(A), util.dev(offsets), util.dev(Wq), util.dev_f16(Ws))
    want = qg.moe_grouped_qgemm(qg.MODE_PLAIN, 4, *args)
    streams, outs = [torch.cuda.Stream(), torch.cuda.Stream()], []
    torch.cuda.synchronize()
    for i in range(40):
        with torch.cuda.stream(streams[i % 2]):
            outs.append(qg.moe_grouped_qgemm(qg.MODE_PLAIN, 4, *args))
    torch.cuda.synchronize()
    qg.poll_status()
    assert all(torch.equal(o, want) for o in outs)


@pytest.mark.parametrize("dense", [False, True], ids=["grouped", "one-matrix"])
def test_launches_share_nothing_however_they_overlap(dense):
    """Launches queued behind a long kernel on one stream, many more issued on a second one meanwhile, and replays of a captured
    launch on a third: all write what a launch alone writes."""
    if dense:
        A, Wq, Ws = synth.dense_problem(8, 5, 38016, 512, seed=19)            # 594 tiles: more than CTAs
        args = (util.dev_bf16(A), util.dev(Wq), util.dev_f16(Ws))
        call = lambda out: qg.qgemm_small_m(8, *args, out=out)
        shape = (5, 38016)
    else:
        counts, N, K = [3, 7, 1, 12, 0, 5] * 8, 1536, 1024
        offsets, A, Wq, Ws = problem(counts, N, K, 9)
        args = (util.dev_bf16(A), util.dev(offsets), util.dev(Wq), util.dev_f16(Ws))
        call = lambda out: qg.moe_grouped_qgemm(qg.MODE_PLAIN, 4, *args, out=out)
        shape = (int(offsets[-1]), N)
    fresh = lambda: torch.full(shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    want = call(fresh())
    held, busy, replay = (torch.cuda.Stream() for _ in range(3))
    captured, graph = fresh(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(captured)
    outs = [fresh() for _ in range(170)]
    torch.cuda.synchronize()
    with torch.cuda.stream(held):
        torch.cuda._sleep(2_000_000)                                          # about a millisecond
        for o in outs[:20]:
            call(o)
    for i, o in enumerate(outs[20:]):
        with torch.cuda.stream(busy):
            call(o)
        if i % 3 == 0:
            with torch.cuda.stream(replay):
                graph.replay()
    torch.cuda.synchronize()
    qg.poll_status()
    assert torch.equal(captured, want) and all(torch.equal(o, want) for o in outs)


def huge_tokens(M, K, seed):
    """Ordinary token rows, then in some 256-k stages values up to the largest bf16; the first row is the largest number for
    which no unscaled block sum overflows, and the second an ordinary one throughout."""
    x = synth.bf16_bits_to_f32(synth.activations(M, K, seed, 64)).copy()
    rng = np.random.default_rng(seed)
    for st in range(0, K // 256, 2):
        blk = slice(256 * st, 256 * st + 256)
        x[2:, blk] = rng.choice([-1.0, 1.0], (M - 2, 256)) * rng.uniform(0.5, 1.0, (M - 2, 256)).astype(np.float32) * np.float32(3.38e38)
    x[0, :] = np.float32(2.0 ** 116 * (1 - 2.0 ** -8))
    return synth.f32_to_bf16_bits(x.astype(np.float32))


@pytest.mark.parametrize("qbits,M,N,K", [(8, 4, 1024, 768), (8, 16, 1032, 1024), (4, 5, 1024, 768), (4, 16, 2056, 256), (8, 9, 38016, 256)],
                         ids=lambda v: str(v))
def test_tokens_up_to_the_largest_number_stay_finite(qbits, M, N, K):
    """Weights scaled beforehand give finite sums of huge tokens, so the exact integer products have to as well, and a zero
    scale gives zero.  An ordinary row beside them keeps its bits."""
    _, Wq, Ws = synth.dense_problem(qbits, M, N, K, seed=21)
    Wq = Wq.copy()
    Wq[:64] = -128 if qbits == 8 else 0                          # the most negative code throughout
    Ws = np.abs(Ws.view(np.float16)).astype(np.float32)
    Ws = (Ws / Ws.max() * 2.0 ** -15).astype(np.float16)
    Ws[5], Ws[N - 3] = 0, 0
    Ws = Ws.view(np.uint16)
    xb = huge_tokens(M, K, 3)
    args = (util.dev(Wq), util.dev_f16(Ws))
    out = util.host_bf16_f64(qg.qgemm_small_m(qbits, util.dev_bf16(xb), *args))
    alone = util.host_bf16_f64(qg.qgemm_small_m(qbits, util.dev_bf16(np.repeat(xb[1:2], M, 0)), *args))
    qg.poll_status()
    assert np.all(out[:, [5, N - 3]] == 0) and np.array_equal(out[1], alone[1])
    rows = np.unique(np.concatenate([np.arange(0, N, max(1, N // 512)), np.arange(64)]))
    ref = orc.qgemm_dense(qbits, xb, Wq[rows], Ws[rows])
    inside = np.abs(ref) < 3.3e38                                # (rows of one sign and one code may leave the format's range)
    assert inside[:, 64:].all() and inside[0].all()
    for m in range(M):                                           # row by row: the rows differ by 38 orders of magnitude
        util.assert_close(out[m, rows][inside[m]], ref[m][inside[m]], f"row {m}")


@pytest.mark.parametrize("mode", [qg.MODE_PLAIN, qg.MODE_GATE_UP_SILU, qg.MODE_DOWN_WEIGHTED], ids=["plain", "gateup", "weighted"])
def test_huge_tokens_in_short_segments(mode):
    counts, N, K = [0, 7, 16, 1, 23], 256, 768
    offsets, _, Wq, Ws = problem(counts, N, K, 22)
    R = int(offsets[-1])
    Ws = (np.abs(Ws.view(np.float16)).astype(np.float32) * 2.0 ** -7).astype(np.float16)
    if mode == qg.MODE_GATE_UP_SILU:
        Ws[:, N // 2:] *= np.float16(2.0 ** 7)                   # the up projection sees the ordinary stage only: the gate is huge already
        Ws[:, N // 2:, :8], Ws[:, N // 2:, 16:] = 0, 0
    Ws = Ws.view(np.uint16)
    xb = huge_tokens(R, K, 5)
    w = np.full(R, 0.5, np.float32)
    row_pair = np.arange(R, dtype=np.int32)
    out = qg.moe_grouped_qgemm(mode, 4, util.dev_bf16(xb), util.dev(offsets), util.dev(Wq), util.dev_f16(Ws), topk_w=util.dev(w),
                               row_pair=util.dev(row_pair))
    qg.poll_status()
    ref = orc.grouped_gemm(4, orc.bf16_to_f64(xb), offsets, Wq, Ws)
    if mode == qg.MODE_GATE_UP_SILU:
        g, u = ref[:, :N // 2], ref[:, N // 2:]
        ref = np.where(g > 0, g * u, 0.0)                        # |g| is beyond 100 wherever it is not the ordinary row
        keep = (np.abs(g) > 100) & (np.abs(ref) < 3.3e38)
    else:
        ref = ref * (0.5 if mode == qg.MODE_DOWN_WEIGHTED else 1.0)
        keep = np.abs(ref) < 3.3e38
    got = util.host_bf16_f64(out)
    for r in range(R):
        if keep[r].sum() > 8:
            util.assert_close(got[r][keep[r]], ref[r][keep[r]], f"row {r}")
    assert keep.mean() > (0.3 if mode == qg.MODE_GATE_UP_SILU else 0.99)


@pytest.mark.parametrize("mode", [qg.MODE_PLAIN, qg.MODE_GATE_UP_SILU, qg.MODE_DOWN_WEIGHTED], ids=["plain", "gateup", "weighted"])
@pytest.mark.parametrize("M,E,k,N,K", [(1, 4, 1, 128, 256), (3, 8, 2, 256, 512), (37, 5, 2, 384, 768), (70, 40, 8, 256, 1280), (100, 128, 8, 1536, 1024)],
                         ids=lambda v: str(v))
def test_gathered_rows_give_the_bits_of_sorted_rows(M, E, k, N, K, mode):
    """Fewer rows than a copy of four, a tile of eight, a tile of sixteen; tokens used more than once; more tiles than CTAs."""
    X, Wq, Ws = synth.activations(M, K, 31), synth.weights_q4(E * N, K, 31).reshape(E, N, K // 2), synth.scales(E * N, K // 32, 7, 31).reshape(E, N, K // 32)
    dX, dWq, dWs = util.dev_bf16(X), util.dev(Wq), util.dev_f16(Ws)
    r = qg.moe_route(util.dev(synth.router_logits(M, E, 31)), k, X=dX)
    w = r["topk_w"].view(-1)
    a = qg.moe_grouped_qgemm(mode, 4, r["Xperm"], r["offsets"], dWq, dWs, topk_w=w, row_pair=r["row_pair"])
    g = util.Guarded(a.shape, torch.bfloat16)
    qg.moe_grouped_qgemm_gather(mode, 4, dX, r["row_pair"], k, r["offsets"], dWq, dWs, topk_w=w, out=g.t)
    qg.poll_status()
    assert torch.equal(a, g.t) and g.intact()
    dX[M // 2, K // 2] = float("inf")                      # and so they do in the rows of a token that is not finite
    a = qg.moe_grouped_qgemm(mode, 4, qg.moe_permute(dX, r["row_pair"], k), r["offsets"], dWq, dWs, topk_w=w, row_pair=r["row_pair"])
    b = qg.moe_grouped_qgemm_gather(mode, 4, dX, r["row_pair"], k, r["offsets"], dWq, dWs, topk_w=w)
    qg.poll_status()
    assert torch.equal(a.nan_to_num(7.0), b.nan_to_num(7.0))


def spread(kind, R, E):
    """R rows over E experts: evenly, preferring a few, all with one (not the first)."""
    counts = np.zeros(E, np.int64)
    if kind == "even":
        counts[:] = R // E
        counts[:R % E] += 1
    elif kind == "few":
        counts[::E // 4] = R // 4
        counts[E - 1] += R - counts.sum()
    else:
        counts[E // 2] = R
    return counts.tolist()


@pytest.mark.parametrize("mode", [qg.MODE_PLAIN, qg.MODE_GATE_UP_SILU, qg.MODE_DOWN_WEIGHTED], ids=["plain", "gateup", "weighted"])
@pytest.mark.parametrize("kind", ["even", "few", "one"])
@pytest.mark.parametrize("R,E,N,K", [(449, 32, 3072, 3072), (160, 32, 6144, 3072), (320, 32, 2944, 3072)], ids=lambda v: str(v))
def test_either_kernel_serves_uneven_segments(R, E, N, K, kind, mode):
    """Sizes around which both kernels are launched and the offsets decide."""
    counts = spread(kind, R, E)
    offsets, A, _, _ = problem(counts, 8, K, 41)
    Wq, Ws = synth.weights_q4(N, K, 41, 62), synth.scales(N, K // 32, 7, 41, 63)
    Wq, Ws = np.stack([np.roll(Wq, e, 0) for e in range(E)]), np.stack([np.roll(Ws, e, 0) for e in range(E)])
    rng = np.random.default_rng(42)
    row_pair, w = rng.permutation(R).astype(np.int32), rng.uniform(0.1, 1.0, R).astype(np.float32)
    X = np.empty_like(A)
    X[row_pair] = A                                        # token order: row r is token row_pair[r]
    dW, dO, dw, drp = (util.dev(Wq), util.dev_f16(Ws)), util.dev(offsets), util.dev(w), util.dev(row_pair)
    g = util.Guarded((R, N // 2 if mode == qg.MODE_GATE_UP_SILU else N), torch.bfloat16)
    for _ in range(3):                                     # back to back: a call's kernels overlap the next one's
        qg.moe_grouped_qgemm(mode, 4, util.dev_bf16(A), dO, *dW, topk_w=dw, row_pair=drp, out=g.t)
    b = qg.moe_grouped_qgemm_gather(mode, 4, util.dev_bf16(X), drp, 1, dO, *dW, topk_w=dw)
    qg.poll_status()
    assert g.intact() and not bool(g.untouched_inside().any().item())
    cols = np.unique(np.concatenate([np.arange(0, N // 2, 29), np.arange(N // 2 - 130, N // 2)]))
    if mode != qg.MODE_GATE_UP_SILU:
        cols = np.concatenate([cols, cols + N // 2])
    es = [e for e in range(E) if counts[e]][:: max(1, E // 8)]
    for e in es:
        seg = slice(int(offsets[e]), int(offsets[e + 1]))
        rows = np.concatenate([cols, cols + N // 2]) if mode == qg.MODE_GATE_UP_SILU else cols
        ref = orc.qgemm_dense(4, A[seg], np.ascontiguousarray(Wq[e][rows]), np.ascontiguousarray(Ws[e][rows]))
        if mode == qg.MODE_GATE_UP_SILU:
            ref = orc.silu_mul(ref)
        elif mode == qg.MODE_DOWN_WEIGHTED:
            ref = ref * w[row_pair[seg]].astype(np.float64)[:, None]
        util.assert_close(util.host_bf16_f64(g.t[seg])[:, cols], ref, f"expert {e}")
        util.assert_close(util.host_bf16_f64(b[seg])[:, cols], ref, f"expert {e}, gathered")


def test_several_tiles_per_block():
    """More tiles than a launch has blocks: a block's second tile, and blocks beyond the last tile."""
    R, E, N, K = 64, 8, 131072, 256
    A = util.dev_bf16(synth.activations(R, K, 44))
    Wq = torch.randint(0, 256, (E, N, K // 2), dtype=torch.uint8, device="cuda")
    Ws = torch.rand((E, N, K // 32), device="cuda").mul_(0.01).to(torch.float16)
    for counts in (spread("even", R, E), spread("one", R, E)):
        offsets = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
        g = util.Guarded((R, N), torch.bfloat16)
        qg.moe_grouped_qgemm(qg.MODE_PLAIN, 4, A, util.dev(offsets), Wq, Ws, out=g.t)
        qg.poll_status()
        assert g.intact() and not bool(g.untouched_inside().any().item())
        for e in range(E):
            q = torch.stack((Wq[e] & 15, Wq[e] >> 4), -1).flatten(-2).to(torch.float32) - 8
            w = (q.unflatten(-1, (-1, 32)) * Ws[e].float()[..., None]).flatten(-2)
            seg = slice(int(offsets[e]), int(offsets[e + 1]))
            if counts[e]:
                util.assert_close(util.host_bf16_f64(g.t[seg]), (A[seg].double() @ w.double().T).cpu().numpy(), f"expert {e}")


@pytest.mark.parametrize("R,E,N,K", [(2304, 128, 1536, 2048), (1024, 256, 4096, 2048), (128, 8, 28672, 4096)], ids=lambda v: str(v))
@pytest.mark.parametrize("kind", ["few", "one"])
def test_uneven_segments_do_not_fall_behind_the_tensor_memory_kernel(R, E, N, K, kind):
    """Rows that crowd into a few experts: the call takes about the time of the kernel that suits them, whatever their average
    (1.5 times and 16 us are the cost of launching both, with room; the wrong kernel takes 2.7 to 4 times as long)."""
    counts = spread(kind, R, E)
    offsets, A, Wq, Ws = problem([R], 8, K, 43)            # random rows; any codes will do
    offsets = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    Wq = torch.randint(0, 256, (E, N, K // 2), dtype=torch.uint8, device="cuda")
    Ws = torch.full((E, N, K // 32), 0.01, dtype=torch.float16, device="cuda")
    args = (util.dev_bf16(A), util.dev(offsets), Wq, Ws)
    out = torch.empty((R, N), dtype=torch.bfloat16, device="cuda")

    def best():
        graph = torch.cuda.CUDAGraph()
        qg.moe_grouped_qgemm(qg.MODE_PLAIN, 4, *args, out=out)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            for _ in range(10):
                qg.moe_grouped_qgemm(qg.MODE_PLAIN, 4, *args, out=out)
        times = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(); graph.replay(); b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 100)
        return min(times)

    own = best()
    qg.set_schedule(128, -1)
    try:
        forced = best()
    finally:
        qg.set_schedule(0, -1)
    qg.poll_status()
    assert own <= 1.5 * forced + 16.0, (own, forced)
