// Block-quantised weight x bf16 activation GEMM for sm_100a: dense and grouped (MoE) in one kernel.
//
// Operation (paper Sec. 3.1: dense GEMM in 4-/8-bit quantisation, MoE expert GEMM, fused gate/up+SiLU):
//   Out[t, n] = sum_k X[t, k] * q[n, k] * scale[n, k/32], per expert segment in the grouped case.
//
// Mapping onto the tensor cores.  The weight rows are the UMMA "M" side and the tokens the "N" side.  Two CTAs
// on neighbouring SMs form a pair (cluster of 2, tcgen05 cta_group::2): the pair's tile is 256 weight rows x BT
// tokens (BT = 128, 192 or 256).  Each CTA dequantises its own 128 weight rows straight into tensor memory, where
// the MMA reads them as its A operand, and stages half of the token tile in shared memory as its half of the B
// operand, so per SM only half of the activation bytes cross L2 -> SM and shared memory.
//
// Persistent CTA of 24 warps, one tile at a time.  BT <= 192: two TMEM accumulators (the epilogue of tile j overlaps
// the main loop of tile j+1); BT = 256: one accumulator and eight TMEM weight stages, the exposed epilogue is shared
// with the dequantising warps.
//   warp 0      TMA producer of this CTA's half activation tile, 2 x X[BT/2, 64] (128-byte swizzle) -> x ring
//   warp 2      TMA producer of packed weights [128, 64] (+ scales every 4 k-blocks)              -> raw ring
//   warps 8-23  dequantise raw -> bf16, written with tcgen05.st into TMEM weight stages (4 groups x 4 warps,
//               group g converts every 4th k-block)
//   warp 1      (even CTA only) issues tcgen05.mma.cta_group::2, two k-blocks at a time, and commits to both CTAs
//   warps 4-7   epilogue: tcgen05.ld, fused activation / routing weight, staged 16-byte bf16 stores
//   warp 3      allocates and frees TMEM
// Barriers the MMA waits on live in the even CTA and also collect the odd CTA's arrivals (remote mbarrier
// arrive, TMA completion bytes); barriers that free a stage are signalled in both CTAs by the commit.
// Dense calls with few tiles cut K into slices, one per CTA pair of a larger cluster (qgemm_slices_kernel): every pair leaves
// its fp32 tile in shared memory and the cluster adds them in slice order.
// Every mbarrier wait is bounded; when one expires the CTA records QG_ERR_TIMEOUT and leaves.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "qg_internal.h"
#include "qg_ptx.cuh"
#include "qg_profile.cuh"
#include "qg_dequant.cuh"

namespace qg {

constexpr int BW = 128;        // weight rows per CTA tile (one UMMA M half)
constexpr int BK = 64;         // k per pipeline stage (one 128-byte swizzle row of bf16)
constexpr int NTHREADS = 768;
constexpr int MAX_E = 1024;

struct GemmParams {
    int mode, R, N, K, E, k;
    int n_wt;                   // 128-row weight tiles per expert (64 gate + 64 up rows each in gate/up mode)
    int gather_k;               // > 0: input row r is X[row_pair[r] / gather_k] (token gather folded into the loads)
    int even_tiles;             // an expert's rows are shared out evenly among its token tiles (to 16 rows); else all but the last are full
    const int32_t* offsets;     // device expert offsets [E+1]; nullptr: one segment [0, R)
    void* out;
    const float* topk_w;
    const int32_t* row_pair;
    int streamk;                // dense plain calls only: the k-blocks of all tiles are dealt out evenly over the CTA
                                // pairs; tiles cut in the middle are summed through sk_partial
    float* sk_partial;          // [CTAs][BT * 128] fp32: the partial accumulator of each CTA's unfinished first tile
    int* sk_flags;              // [CTAs][2]: 16-token blocks of the partial written / consumed; zero between launches
    int slices, kc;             // dense plain calls with few tiles: K cut into `slices` parts of kc k-blocks, one per CTA
                                // pair of a cluster; the cluster adds the parts through distributed shared memory
    int* status;
    uint32_t wait_limit;        // polls per bounded wait (an unsatisfied poll lasts about 4 us)
    int skip_kb;                // test hook: k-block of the first tile whose activation load is left out (-1: none)
#ifdef QG_PROFILE
    long long* stats;           // per-CTA cycle counters of a profiling build
#endif
};

template <int QBITS, int BT>
struct Cfg {
    static constexpr int SX = 8;                                   // k-block stages: ring of the activation tile (smem)
    static constexpr int SP = SX / 2;                              // ... in pairs: what the full/done barriers count
    static constexpr int SR = (QBITS == 4 && BT <= 192) ? 16 : 8;  // packed-weight stages (smem, refilled four at a time):
                                                                   // twice as deep for 4-bit tiles where shared memory allows
    static constexpr int NACC = (BT > 192) ? 1 : 2;                // accumulators in tensor memory
    static constexpr int SA = ((512 - NACC * BT) / 32 >= 8) ? 8 : (512 - NACC * BT) / 32;   // dequantised-weight stages in
                                                                   // tensor memory (8, or what two accumulators leave)
    // With a single accumulator the epilogue is exposed, so the dequantising warps share it (they would idle at the
    // tile boundary); with two accumulators it overlaps the next main loop and the dequantising warps stay on theirs.
    static constexpr bool HELP = (NACC == 1);
    static constexpr int NSB = SR / 4 + 1;                         // scale buffers (one per 4 k-blocks)
    static constexpr int XH_ROWS = BT / 2;                         // token rows this CTA stages per k-block
    static constexpr int X_BYTES = XH_ROWS * 128;
    static constexpr int RAW_ROW = (QBITS == 8) ? 64 : 32;         // packed bytes per row per stage
    static constexpr int RAW_BYTES = BW * RAW_ROW;
    static constexpr int SC_BYTES = BW * 16;                       // 8 fp16 scales per row
    // transposition buffers: 1 KB for each dequantising warp, then the epilogue warps'; theirs are 2 KB, used in turn, where they
    // drain most tiles alone
    static constexpr int EPI_ST = HELP ? 1024 : 2048;
    static constexpr int STG_BYTES = 16 * 1024 + 4 * EPI_ST;
    static constexpr int WT_BYTES = HELP ? 0 : 2 * BT * 4;         // routing weights of a tile's tokens, two tiles in turn
    static constexpr int OFF_X = 0;
    static constexpr int OFF_RAW = OFF_X + SX * X_BYTES;
    static constexpr int OFF_SC = OFF_RAW + SR * RAW_BYTES;
    static constexpr int OFF_STG = OFF_SC + NSB * SC_BYTES;
    static constexpr int OFF_WT = OFF_STG + STG_BYTES;
    static constexpr int OFF_PREFIX = OFF_WT + WT_BYTES;
    static constexpr int TAB_N = 128;                              // decoded tiles of this pair kept in shared memory
    static constexpr int OFF_TAB = OFF_PREFIX + (MAX_E + 4) * 4;
    static constexpr int OFF_BAR = OFF_TAB + TAB_N * 16;
    static constexpr int NBAR = 2 * SP + 2 * SR + 5;
    static constexpr int OFF_MISC = OFF_BAR + NBAR * 8;
    static constexpr int SMEM_BYTES = OFF_MISC + 32 + 1024;        // + slack for 1024-byte alignment
    static constexpr int TMEM_COLS = 512;                          // accumulator(s) + SA weight stages
    static constexpr int A_COL0 = NACC * BT;                       // first column of the weight stages
    static constexpr int A_COLS = 32;                              // 64 bf16 per lane = 32 columns per stage
    static_assert(NACC * BT + SA * 32 <= 512, "tensor memory budget");
    static_assert(X_BYTES % 1024 == 0, "swizzled stages must stay 1024-byte aligned");
    static_assert(SX == 8, "stage arithmetic below assumes a ring of eight");
    static_assert(SA >= 4 && SA % 2 == 0 && (!HELP || SA == 8), "weight stages");
};

struct __align__(16) Tile {
    int e, pw, tok0, tok_end;   // expert, pair weight tile (weight tiles 2 pw and 2 pw + 1), token range
};

// The part of a tile one CTA pair computes: k-blocks [kb0, kb1), the first of which has ring index i0 in this pair's
// sequence.  nsrc: 0 the whole tile; -1 a part that does not start at k = 0 (its fp32 partial goes to this CTA's slot
// of sk_partial); n > 0 the part that starts at k = 0 but stops early: the n following pairs hold the rest, their
// partials are added in pair order before the tile is rounded and stored.
struct __align__(16) Piece {
    int kb0, kb1, i0, nsrc;
};

template <bool GROUPED>          // false: stream-K and K slices, one segment
__device__ __forceinline__ Tile decode_tile(int t, const int* prefix, const GemmParams& p, int BT) {
    int lo = 0, hi = p.E - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= t) lo = mid; else hi = mid - 1;
    }
    const int seg0 = p.offsets ? p.offsets[lo] : 0;
    const int seg1 = p.offsets ? p.offsets[lo + 1] : p.R;
    const int n_tt = (seg1 - seg0 + BT - 1) / BT;
    const int local = t - prefix[lo];
    int rows = BT;
    if (GROUPED && p.even_tiles) {
        // the fewest rows, in steps of 16, with which as many tiles do: BT - 16 floor(spare / (16 n_tt)); the quotient of two numbers below 17
        // by a float reciprocal (an integer division here costs every call 0.13 us)
        const int spare = (n_tt * BT - (seg1 - seg0)) >> 4;
        rows -= 16 * static_cast<int>(__fdividef(static_cast<float>(spare) + 0.5f, static_cast<float>(n_tt)));
    }
    Tile r;
    r.e = lo;
    r.pw = local / n_tt;
    r.tok0 = seg0 + (local % n_tt) * rows;
    r.tok_end = min(seg1, r.tok0 + rows);
    return r;
}

// Bounded wait on an mbarrier phase, first without suspending: a phase that is complete already is the common case, and the
// plain test tells it sooner (3 % of a grouped GEMM).  Returns false if the CTA is giving up.
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag, const GemmParams& p) {
    const uint32_t limit = p.wait_limit;
    if (mbar_test_wait(bar, parity)) return true;
    for (uint32_t it = 0; it < limit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 255u && *abort_flag) return false;
    }
    *abort_flag = 1;
    atomicCAS(p.status, 0, QG_ERR_TIMEOUT);
    return false;
}

// Same for the MMA warp: a short non-blocking spin first (the barrier is usually complete or about to be), then
// the bounded blocking wait.
__device__ __forceinline__ bool spin_wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag, const GemmParams& p) {
    for (int it = 0; it < 64; ++it)
        if (mbar_test_wait(bar, parity)) return true;
    return wait_bar(bar, parity, abort_flag, p);
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

// Plain / routing-weighted epilogue of one warp: drains the 16-column (token) blocks b = pid, pid + npart, ... of
// its 32 TMEM lanes (weight rows).  The block is read in accumulator-fragment layout (thread T: rows T/4 + 8 m,
// token pairs), scaled, packed to bf16x2 and written with two transposing matrix stores into a private
// [16 tokens][32 rows] buffer (16-byte chunks XOR-swizzled by the token pair, conflict-free both ways), from which
// every thread moves two 16-byte pieces to global memory (64 contiguous bytes per token).  The next block's TMEM
// loads are in flight while the current one is stored.  Called by the four epilogue warps (TWO: with two buffers in turn, so
// that a block need not wait until the one before it has left) and by the sixteen dequantising warps: for a
// single-accumulator tile, and for a pair's last tile, when they would otherwise idle.
// WS: the tile's routing weights are in shared memory (wts, by token); otherwise every warp fetches them, two dependent loads from
// global memory in front of its first block (with 12 k-blocks a tile, 1500 of the 6500 cycles of an epilogue that was the pace).
template <bool SK, bool WS, bool TWO>
__device__ __forceinline__ void drain_plain(const GemmParams& p, int tok0, int tok_end, int n_base, uint32_t taddr,
                                            int n_epi, int pid, int npart, __nv_bfloat16* st, const float* wts, int lane, int nsrc_in,
                                            int quarter, int slot_floats, volatile int* abort_flag) {
    const int nsrc = SK ? nsrc_in : 0;       // without stream-K all of the partial-tile handling below compiles away
    // The loop is issue-bound (five warps of a scheduler drain together), so everything that does not depend on the
    // block is computed once: the lane's two shared-memory read addresses, its global pointer and its token limit.
    const int nblk = n_epi >> 4;
    int b = pid;
    if (b >= nblk) return;
    const bool weighted = (p.mode == QG_MODE_DOWN_WEIGHTED);
    // Stream-K parts of a tile.  A part that does not start at k = 0 leaves its raw fp32 fragments in this CTA's slot
    // (register r of 16-token block b and lane quarter q at ((b 4 + q) 16 + r) 32 + lane: 128-byte rows) and counts its
    // blocks in the slot's first flag.  The part that starts at k = 0 waits until every block of each of the nsrc
    // following pairs' slots is there, adds them in pair order and goes on as for a whole tile; the second flag
    // counts what has been read, and whoever reads last clears both for the next launch.
    const int mine = SK ? (nblk - pid + npart - 1) / npart : 0;     // blocks this warp drains
    const int slot = static_cast<int>(blockIdx.x);
    if (SK && nsrc > 0) {
        for (int c = 1; c <= nsrc; ++c) {
            const int* f = p.sk_flags + 2 * (slot + 2 * c);
            bool there = false;
            for (uint32_t it = 0; it < p.wait_limit * 16u && !there; ++it) {
                int v;
                asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
                there = (v >= nblk * 4);
                if (!there) {
                    if ((it & 1023u) == 1023u && *abort_flag) break;
                    __nanosleep(200);
                }
            }
            if (!there) {        // give up: the launch reports a timeout, the host clears the flags
                *abort_flag = 1;
                atomicCAS(p.status, 0, QG_ERR_TIMEOUT);
                return;
            }
        }
    }
    uint32_t v0[8], v1[8];                       // TMEM lanes 0-15 / 16-31 of this warp's quarter
    tmem_ld_16x256_x2(taddr + 16 * b, v0);
    tmem_ld_16x256_x2(taddr + (16u << 16) + 16 * b, v1);
    // Routing weights of the whole tile, fetched once (two dependent global loads, all in flight together): lane l
    // holds the weights of tokens l, l + 32, ... of the tile.
    float wt8[8];
    if (!WS && weighted) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int tokl = tok0 + 32 * j + lane;
            wt8[j] = (32 * j < n_epi && tokl < tok_end) ? p.topk_w[p.row_pair[tokl]] : 0.f;
        }
    }
    uint32_t st_row = smem_u32(st) + (lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) << 4);   // matrix lane>>3, token lane&7
    const int c = 2 * (lane & 3);                // this thread's token pairs: c, c + 1 and 8 + c, 9 + c of the block
    // store side: this lane moves tokens tk and 8 + tk of every block, 16 bytes (8 rows from n) each
    const int tk = lane >> 2, c4 = lane & 3;
    const int n = n_base + c4 * 8;
    uint32_t s_lo = smem_u32(st) + tk * 64 + ((c4 ^ ((tk >> 1) & 3)) << 4);      // token 8 + tk: 512 bytes on, same swizzle
    int flip = 1024;                             // to the other buffer and back
    const size_t row8 = static_cast<size_t>(8) * p.N;
    __nv_bfloat16* g = static_cast<__nv_bfloat16*>(p.out) + static_cast<size_t>(tok0 + 16 * b + tk) * p.N + n;
    const size_t g_step = 2 * row8 * npart;
    int left = (n < p.N) ? (tok_end - tok0 - 16 * b - tk) : 0;   // tokens tk, 8 + tk of the block are stored if 0, 8 < left
    const int left_step = 16 * npart;
    while (b < nblk) {
        tmem_ld_wait();
        if (SK && nsrc != 0) {
            const size_t at = (static_cast<size_t>(b * 4 + quarter) * 16) * 32 + lane;
            if (nsrc < 0) {
                float* dst = p.sk_partial + static_cast<size_t>(slot) * slot_floats + at;
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    dst[r * 32] = __uint_as_float(v0[r]);
                    dst[(8 + r) * 32] = __uint_as_float(v1[r]);
                }
                const int bn = b + npart;
                if (bn < nblk) {
                    tmem_ld_16x256_x2(taddr + 16 * bn, v0);
                    tmem_ld_16x256_x2(taddr + (16u << 16) + 16 * bn, v1);
                }
                b = bn;
                continue;
            }
            for (int c = 1; c <= nsrc; ++c) {
                const float* src = p.sk_partial + static_cast<size_t>(slot + 2 * c) * slot_floats + at;
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    v0[r] = __float_as_uint(__uint_as_float(v0[r]) + __ldcg(src + r * 32));
                    v1[r] = __float_as_uint(__uint_as_float(v1[r]) + __ldcg(src + (8 + r) * 32));
                }
            }
        }
        uint32_t pk[8];
        if (weighted) {
            float w0, w1, w2, w3;                // weights of tokens 16 b + c, + 1, + 8, + 9
            if constexpr (WS) {
                const float2 wa = *reinterpret_cast<const float2*>(wts + 16 * b + c), wb = *reinterpret_cast<const float2*>(wts + 16 * b + 8 + c);
                w0 = wa.x; w1 = wa.y; w2 = wb.x; w3 = wb.y;
            } else {
                const int j = b >> 1;            // tokens 16 b .. 16 b + 15 live in register j, lanes 16 (b & 1) ..
                float wv = wt8[0];
#pragma unroll
                for (int jj = 1; jj < 8; ++jj) wv = (j == jj) ? wt8[jj] : wv;
                const int src = 16 * (b & 1) + c;
                w0 = __shfl_sync(0xFFFFFFFFu, wv, src); w1 = __shfl_sync(0xFFFFFFFFu, wv, src + 1);
                w2 = __shfl_sync(0xFFFFFFFFu, wv, src + 8); w3 = __shfl_sync(0xFFFFFFFFu, wv, src + 9);
            }
#pragma unroll
            for (int gq = 0; gq < 2; ++gq) {     // tokens 8 gq .. 8 gq + 7
                const float wa = gq ? w2 : w0, wb = gq ? w3 : w1;
                pk[4 * gq + 0] = bf16x2(__uint_as_float(v0[4 * gq + 0]) * wa, __uint_as_float(v0[4 * gq + 1]) * wb);
                pk[4 * gq + 1] = bf16x2(__uint_as_float(v0[4 * gq + 2]) * wa, __uint_as_float(v0[4 * gq + 3]) * wb);
                pk[4 * gq + 2] = bf16x2(__uint_as_float(v1[4 * gq + 0]) * wa, __uint_as_float(v1[4 * gq + 1]) * wb);
                pk[4 * gq + 3] = bf16x2(__uint_as_float(v1[4 * gq + 2]) * wa, __uint_as_float(v1[4 * gq + 3]) * wb);
            }
        } else {
#pragma unroll
            for (int gq = 0; gq < 2; ++gq) {
                pk[4 * gq + 0] = bf16x2(__uint_as_float(v0[4 * gq + 0]), __uint_as_float(v0[4 * gq + 1]));
                pk[4 * gq + 1] = bf16x2(__uint_as_float(v0[4 * gq + 2]), __uint_as_float(v0[4 * gq + 3]));
                pk[4 * gq + 2] = bf16x2(__uint_as_float(v1[4 * gq + 0]), __uint_as_float(v1[4 * gq + 1]));
                pk[4 * gq + 3] = bf16x2(__uint_as_float(v1[4 * gq + 2]), __uint_as_float(v1[4 * gq + 3]));
            }
        }
        const int bn = b + npart;
        if (bn < nblk) {                         // next block, overlapped with the stores below
            tmem_ld_16x256_x2(taddr + 16 * bn, v0);
            tmem_ld_16x256_x2(taddr + (16u << 16) + 16 * bn, v1);
        }
        stmatrix_x4_trans(st_row, pk[0], pk[1], pk[2], pk[3]);
        stmatrix_x4_trans(st_row + 512, pk[4], pk[5], pk[6], pk[7]);
        __syncwarp();
        if (left > 0) *reinterpret_cast<uint4*>(g) = lds128(s_lo);
        if (left > 8) *reinterpret_cast<uint4*>(g + row8) = lds128(s_lo + 512);
        if constexpr (TWO) {
            st_row += flip;
            s_lo += flip;
            flip = -flip;
        } else {
            __syncwarp();
        }
        g += g_step;
        left -= left_step;
        b = bn;
    }
    __syncwarp();                                // the buffers may be written again
    if (SK && nsrc < 0) {
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicAdd(p.sk_flags + 2 * slot, mine);
    } else if (SK && nsrc > 0) {
        __syncwarp();
        if (lane == 0) {
            for (int c = 1; c <= nsrc; ++c) {
                int* f = p.sk_flags + 2 * (slot + 2 * c);
                if (atomicAdd(f + 1, mine) + mine == nblk * 4) { f[1] = 0; __threadfence(); f[0] = 0; }
            }
        }
    }
}

// Gate/up epilogue of one warp.  The tile's weight rows were dequantised into such an order (see the dequantising warps) that the
// lanes 0-15 of a quarter are gate rows and lanes 16-31 the up rows that belong to them, so the two fragments of a 16-token block hold
// a thread's gates and ups in the same places: SiLU(gate) * up in registers, one transposing matrix store into a [16 tokens][16
// rows] buffer, 32 contiguous bytes per token from there.  Blocks as in drain_plain; two buffers of 512 bytes in turn.  (Gates and ups in
// different warps met through a [32 tokens][128 rows] fp32 buffer and two barriers of all four: 8000 cycles a tile of 192 tokens.)
__device__ __forceinline__ void drain_gate_up(const GemmParams& p, int tok0, int tok_end, int f_base, uint32_t taddr, int n_epi, int pid,
                                              int npart, __nv_bfloat16* st, int lane) {
    const int nblk = n_epi >> 4, F = p.N >> 1;
    int b = pid;
    if (b >= nblk) return;
    uint32_t v0[8], v1[8];
    tmem_ld_16x256_x2(taddr + 16 * b, v0);
    tmem_ld_16x256_x2(taddr + (16u << 16) + 16 * b, v1);
    // write side: matrix m = lane / 8 holds rows 8 (m % 2) .. of tokens 8 (m / 2) ..; this lane names token 8 (m / 2) + lane % 8
    const int wtok = ((lane >> 4) << 3) + (lane & 7), whalf = (lane >> 3) & 1;
    uint32_t st_row = smem_u32(st) + wtok * 32 + ((whalf ^ ((wtok >> 2) & 1)) << 4);
    const int tk = lane >> 1, half = lane & 1;   // store side: 16 bytes (8 rows) of one token
    uint32_t s_at = smem_u32(st) + tk * 32 + ((half ^ ((tk >> 2) & 1)) << 4);
    __nv_bfloat16* g = static_cast<__nv_bfloat16*>(p.out) + static_cast<size_t>(tok0 + 16 * b + tk) * F + f_base + 8 * half;
    const size_t g_step = static_cast<size_t>(16 * npart) * F;
    int left = tok_end - tok0 - 16 * b - tk, flip = 512;
    while (b < nblk) {
        tmem_ld_wait();
        float h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float gt = __uint_as_float(v0[i]);
            h[i] = __fdividef(gt, 1.0f + __expf(-gt)) * __uint_as_float(v1[i]);
        }
        const int bn = b + npart;
        if (bn < nblk) {                         // next block, overlapped with the rest of this one
            tmem_ld_16x256_x2(taddr + 16 * bn, v0);
            tmem_ld_16x256_x2(taddr + (16u << 16) + 16 * bn, v1);
        }
        stmatrix_x4_trans(st_row, bf16x2(h[0], h[1]), bf16x2(h[2], h[3]), bf16x2(h[4], h[5]), bf16x2(h[6], h[7]));
        __syncwarp();
        if (left > 0) *reinterpret_cast<uint4*>(g) = lds128(s_at);
        st_row += flip;
        s_at += flip;
        flip = -flip;
        g += g_step;
        left -= 16 * npart;
        b = bn;
    }
    __syncwarp();
}

// K slices (SK = 2): a warp leaves the raw fp32 fragments of its 16-token blocks in this CTA's shared memory (the idle ring of
// the activation tile, exactly as large): register r of block b and lane quarter q at ((b 4 + q) 16 + r) 32 + lane.
__device__ __forceinline__ void dump_partial(float* part, uint32_t taddr, int n_epi, int pid, int npart, int quarter, int lane) {
    for (int b = pid; b < (n_epi >> 4); b += npart) {
        uint32_t v0[8], v1[8];
        tmem_ld_16x256_x2(taddr + 16 * b, v0);
        tmem_ld_16x256_x2(taddr + (16u << 16) + 16 * b, v1);
        tmem_ld_wait();
        float* dst = part + ((b * 4 + quarter) * 16) * 32 + lane;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            dst[r * 32] = __uint_as_float(v0[r]);
            dst[(8 + r) * 32] = __uint_as_float(v1[r]);
        }
    }
}

// Then one warp adds a block's fragments over the slices, in slice order, and stores it (the layout and the transposition of
// drain_plain).  part: shared::cluster-mappable address of the fragments, r_cta: which CTA of each pair holds these rows.
__device__ __forceinline__ void sum_block(const GemmParams& p, uint32_t part, uint32_t r_cta, int unit, int tok0, int tok_end,
                                          int n_tile, __nv_bfloat16* st, int lane) {
    const int b = unit >> 2, quarter = unit & 3;
    float v[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = 0.f;
    for (int sl = 0; sl < p.slices; ++sl) {
        const uint32_t src = map_to_cta(part + (unit * 16 * 32 + lane) * 4, 2 * sl + r_cta);
        float x[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x[r]) : "r"(src + r * 128));
#pragma unroll
        for (int r = 0; r < 16; ++r) v[r] += x[r];
    }
    uint32_t pk[8];
#pragma unroll
    for (int gq = 0; gq < 2; ++gq) {
        pk[4 * gq + 0] = bf16x2(v[4 * gq + 0], v[4 * gq + 1]);
        pk[4 * gq + 1] = bf16x2(v[4 * gq + 2], v[4 * gq + 3]);
        pk[4 * gq + 2] = bf16x2(v[8 + 4 * gq + 0], v[8 + 4 * gq + 1]);
        pk[4 * gq + 3] = bf16x2(v[8 + 4 * gq + 2], v[8 + 4 * gq + 3]);
    }
    const uint32_t st_row = smem_u32(st) + (lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) << 4);
    const int tk = lane >> 2, c4 = lane & 3, n = n_tile + quarter * 32 + c4 * 8, left = tok_end - tok0 - 16 * b - tk;
    stmatrix_x4_trans(st_row, pk[0], pk[1], pk[2], pk[3]);
    stmatrix_x4_trans(st_row + 512, pk[4], pk[5], pk[6], pk[7]);
    __syncwarp();
    const uint4* s_lo = reinterpret_cast<const uint4*>(st + tk * 32 + ((c4 ^ ((tk >> 1) & 3)) << 3));
    __nv_bfloat16* g = static_cast<__nv_bfloat16*>(p.out) + static_cast<size_t>(tok0 + 16 * b + tk) * p.N + n;
    if (n < p.N && left > 0) *reinterpret_cast<uint4*>(g) = *s_lo;
    if (n < p.N && left > 8) *reinterpret_cast<uint4*>(g + static_cast<size_t>(8) * p.N) = s_lo[32];
    __syncwarp();
}

// SK: 0 every tile is computed whole, 1 stream-K, 2 K slices of one tile on the CTA pairs of a cluster (grid = one cluster
// per tile).
// EPI: 0 plain / routing-weighted bf16 store, 1 gate/up + SiLU, 2 weighted fp32 atomic accumulate (compiled apart so
// that each instantiation carries one epilogue only).
template <int QBITS, int BT, int EPI, int SK>
__device__ __forceinline__ void gemm_body(const CUtensorMap& tm_x, const CUtensorMap& tm_w, const CUtensorMap& tm_s,
                                          const GemmParams& p) {
    using C = Cfg<QBITS, BT>;
    extern __shared__ uint8_t smem_dyn[];
    const uint32_t sbase = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    uint8_t* sgen = smem_dyn + (sbase - smem_u32(smem_dyn));
    int* prefix = reinterpret_cast<int*>(sgen + C::OFF_PREFIX);
    __nv_bfloat16* stg16 = reinterpret_cast<__nv_bfloat16*>(sgen + C::OFF_STG);
    float* wts = reinterpret_cast<float*>(sgen + C::OFF_WT);
    volatile int* misc = reinterpret_cast<volatile int*>(sgen + C::OFF_MISC);  // [0] tmem base, [1] abort, [2..3] epilogue go/stop
    const uint32_t bar0 = sbase + C::OFF_BAR;
    // full[s]   (even CTA): the two k-blocks of stage pair s are ready: both halves of the activation tile have landed (TMA
    //           bytes) and all sixteen dequantising warps of the pair (4 per CTA and k-block) have written their weights to TMEM.
    // done[s]   (both CTAs, by commit): the MMAs of the two k-blocks in stage pair s have completed.
    // r_full / r_empty: this CTA's packed-weight ring.   acc_full (both CTAs) / acc_empty (even CTA): accumulators.
    auto full = [&](int s) { return bar0 + 8u * s; };
    auto done = [&](int s) { return bar0 + 8u * (C::SP + s); };
    auto r_full = [&](int s) { return bar0 + 8u * (2 * C::SP + s); };
    auto r_empty = [&](int s) { return bar0 + 8u * (2 * C::SP + C::SR + s); };
    auto acc_full = [&](int s) { return bar0 + 8u * (2 * C::SP + 2 * C::SR + s); };
    auto acc_empty = [&](int s) { return bar0 + 8u * (2 * C::SP + 2 * C::SR + 2 + s); };
    // last_full (this CTA, one phase): the epilogue warps, which consume every accumulator phase in order, have seen the
    // last tile's accumulator complete.  The dequantising warps that help with that last epilogue wait here instead
    // of on acc_full, whose parity they cannot tell apart from the phase two tiles earlier when K is short.
    const uint32_t last_full = bar0 + 8u * (2 * C::SP + 2 * C::SR + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t crank = cluster_ctarank();
    const uint32_t rank = (SK == 2) ? (crank & 1u) : crank;            // 0: issues the MMAs, 1: its peer
    const uint32_t leader = (SK == 2) ? (crank & ~1u) : 0u;            // the pair's even CTA
    const int slice = (SK == 2) ? static_cast<int>(crank >> 1) : 0;
    const int kb_first = (SK == 2) ? slice * p.kc : 0;                 // this pair's first k-block
    // The next kernel in the stream may be scheduled as this grid's CTAs leave their SMs.  This kernel in turn may
    // have started before the previous one finished: whatever that kernel may have written (activations, expert
    // offsets, routing tables) or may still read (the output buffer) is touched only after pdl_wait().  The weights
    // are constants of the model, so in the dense case their producer and the dequantising warps start at once.
    pdl_launch_dependents();
    if (warp == 0) { QG_MARK(0); }
    QG_SPAN(0);
    const bool grouped = (p.offsets != nullptr);
    const int pair = (SK == 2) ? static_cast<int>(blockIdx.x) / (2 * p.slices) : static_cast<int>(blockIdx.x) >> 1;
    const int n_pairs = (SK == 2) ? static_cast<int>(gridDim.x) / (2 * p.slices) : static_cast<int>(gridDim.x) >> 1;
    volatile int* abort_flag = misc + 1;
    float* partial = reinterpret_cast<float*>(sgen + C::OFF_X);          // K slices: where the ring of the activation tile was

    if (warp == 0) {   // barrier initialisation spread over the lanes of one warp (a single thread needs ~50 steps)
        if (lane < C::SP) { mbar_init(full(lane), 1 + 16); mbar_init(done(lane), 1); }
        // an accumulator is released by the 4 epilogue + 16 dequantising warps of both CTAs
        if (lane >= 16 && lane < 18) { mbar_init(acc_full(lane - 16), 1); mbar_init(acc_empty(lane - 16), C::HELP ? 40 : 8); }
        if (lane == 31) { misc[1] = 0; mbar_init(last_full, 1); }
        fence_mbar_init();
        fence_proxy_async_smem();
        if (lane == 30) prefetch_tmap(&tm_x);
        if (lane == 29) prefetch_tmap(&tm_w);
        if (lane == 28) prefetch_tmap(&tm_s);
    }
    if (warp == 3) {
        tmem_alloc_pair(sbase + C::OFF_MISC, C::TMEM_COLS);
        tmem_relinquish_pair();
    }
    const int n_pw = (p.n_wt + 1) >> 1;
    // The packed-weight ring is private to this CTA and to warp 2, its producer: that warp initialises the ring's
    // barriers itself and, as soon as it knows the pair's first tile, sends the first four k-blocks of weights on
    // their way, so that they travel while the pair synchronises and the tile tables are built.
    bool w_pre_issued = false;
    // One copy fetches this CTA's 128 weight rows of a k-block (or their scales): a 128-row box, or in gate/up mode a
    // box of 64 rows x 2 planes of a 3-D map whose planes are the gate and the up halves of the experts' matrices.
    auto load_w = [&](uint32_t dst, const CUtensorMap* tm, int x, int e, int wt, uint32_t bar) {
        if constexpr (EPI == 1) tma_load_3d(dst, tm, x, wt * 64, 2 * e, bar);
        else tma_load_2d(dst, tm, x, e * p.N + wt * 128, bar);
    };
    if (warp == 2) {  // prefix[e] = pair tiles before expert e; prefix[E] = total
        // one barrier pair per batch of four stages (the batch's first stage carries it): 16 converting warps release it
        if (lane < C::SR) { mbar_init(r_full(lane), 1); mbar_init(r_empty(lane), 16); }
        fence_mbar_init();
        fence_proxy_async_smem();
        if (grouped) pdl_wait();
        int carry = 0;
        constexpr int PB = 4;                    // experts per lane whose offsets travel together
        for (int e0 = 0; e0 < p.E; e0 += 32 * PB) {
            int cnt[PB];
#pragma unroll
            for (int i = 0; i < PB; ++i) {
                const int e = e0 + 32 * i + lane;
                cnt[i] = (e >= p.E) ? 0 : p.offsets ? p.offsets[e + 1] - p.offsets[e] : p.R;
            }
#pragma unroll
            for (int i = 0; i < PB; ++i) {
                const int e = e0 + 32 * i + lane;
                if (e0 + 32 * i >= p.E) break;
                const int n = ((cnt[i] + BT - 1) / BT) * n_pw;
                int inc = n;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int v = __shfl_up_sync(0xFFFFFFFFu, inc, off);
                    if (lane >= off) inc += v;
                }
                if (e < p.E) prefix[e] = carry + inc - n;
                carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
            }
        }
        if (lane == 0) prefix[p.E] = carry;
        __syncwarp();
        if (SK != 1 && pair < carry) {
            const Tile tl = decode_tile<SK == 0>(pair, prefix, p, BT);
            const int wt = 2 * tl.pw + static_cast<int>(rank);
            if (elect_one()) {
                mbar_arrive_expect_tx(r_full(0), 4 * C::RAW_BYTES + C::SC_BYTES);
                load_w(sbase + C::OFF_SC, &tm_s, (kb_first >> 2) * 8, tl.e, wt, r_full(0));
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    load_w(sbase + C::OFF_RAW + j * C::RAW_BYTES, &tm_w, (kb_first + j) * C::RAW_ROW, tl.e, wt, r_full(0));
            }
            w_pre_issued = true;
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();          // both CTAs' barriers are initialised and both halves of TMEM are allocated
    tc_fence_after_sync();
    if (grouped || warp == 0 || (warp >= 4 && warp < 8)) pdl_wait();   // dense: the other roles wait when they must
    const uint32_t tmem_base = static_cast<uint32_t>(misc[0]);
    const int total_tiles = prefix[p.E];
    const int nkb = p.K / BK;     // a multiple of 4
    // The pair's j-th tile is tile pair + j n_pairs.  Decoding one costs a binary search and two global loads, far
    // too much for the control warps to repeat at every tile boundary, so the first TAB_N are decoded once, here.
    Tile* tab = reinterpret_cast<Tile*>(sgen + C::OFF_TAB);
    // stream-K (dense only, so the prefix array needs two entries and the piece table takes the rest of its space)
    Piece* ptab = reinterpret_cast<Piece*>(sgen + C::OFF_PREFIX + 16);
    const int nk4 = nkb >> 2;
    int my_tiles;
    uint32_t own_kb4;            // this pair's k-blocks / 4
    if constexpr (SK == 1) {
        // Units of four k-blocks, U = tiles * nk4 in all; pair q owns units [U q / P, U (q + 1) / P).  Piece j of this
        // pair lies in tile t_first + j (the host keeps the number of pieces within the table).
        const long long U = static_cast<long long>(total_tiles) * nk4;
        const long long u0 = U * pair / n_pairs, u1 = U * (pair + 1) / n_pairs;
        const int t_first = static_cast<int>(u0 / nk4);
        my_tiles = (u1 > u0) ? static_cast<int>((u1 - 1) / nk4) - t_first + 1 : 0;
        own_kb4 = static_cast<uint32_t>(u1 - u0);
        for (int j = threadIdx.x; j < my_tiles; j += NTHREADS) {
            const int t = t_first + j;
            const long long tb = static_cast<long long>(t) * nk4;
            const long long a = (u0 > tb) ? u0 : tb, b = (u1 < tb + nk4) ? u1 : tb + nk4;
            Piece pc;
            pc.kb0 = static_cast<int>(a - tb) * 4;
            pc.kb1 = static_cast<int>(b - tb) * 4;
            pc.i0 = static_cast<int>(a - u0) * 4;
            pc.nsrc = 0;
            if (pc.kb0 > 0) {
                pc.nsrc = -1;
            } else if (pc.kb1 < nkb) {
                int q = pair + 1;                                   // owner of the tile's last unit
                while (q + 1 < n_pairs && U * (q + 1) / n_pairs <= tb + nk4 - 1) ++q;
                pc.nsrc = q - pair;
            }
            ptab[j] = pc;
            tab[j] = decode_tile<SK == 0>(t, prefix, p, BT);
        }
    } else if constexpr (SK == 2) {
        my_tiles = 1;                                       // one cluster per tile
        own_kb4 = static_cast<uint32_t>(min(p.kc, nkb - kb_first)) >> 2;
        if (threadIdx.x == 0) tab[0] = decode_tile<SK == 0>(pair, prefix, p, BT);
    } else {
        my_tiles = (total_tiles > pair) ? (total_tiles - pair + n_pairs - 1) / n_pairs : 0;
        own_kb4 = static_cast<uint32_t>(my_tiles) * static_cast<uint32_t>(nk4);
        for (int j = threadIdx.x; j < min(my_tiles, C::TAB_N); j += NTHREADS)
            tab[j] = decode_tile<SK == 0>(pair + j * n_pairs, prefix, p, BT);
    }
    __syncthreads();
    if (warp == 0) { QG_MARK(1); }
    auto tile_at = [&](int j) -> Tile {
        return (j < C::TAB_N) ? tab[j] : decode_tile<SK == 0>(pair + j * n_pairs, prefix, p, BT);
    };
    auto piece_at = [&](int j) -> Piece {
        if constexpr (SK == 1) return ptab[j];
        Piece pc;
        pc.kb0 = kb_first; pc.kb1 = (SK == 2) ? kb_first + 4 * static_cast<int>(own_kb4) : nkb; pc.i0 = j * nkb; pc.nsrc = 0;
        return pc;
    };

    // Control warps walk their loops with all 32 lanes (converged) and issue behind elect.sync.  Each shares its scheduler with
    // four converting warps, so an iteration of a few dozen dependent instructions lasts some hundred cycles, the price of a wait
    // that succeeds at once (200) among them: a k-block at a time the activation producer was the pace of the kernel (128
    // experts, 1536 x 2048, 512 tokens: 116 us).  So it hands over two k-blocks at a time, as one copy and one barrier, the
    // packed-weight producer four.
    if (warp == 0) {
        // ------------------------------------------------ activation producer (this CTA's half of the token tile)
        uint32_t s = 0, ph = 0;      // next stage pair and the parity of its next "done" phase
        uint32_t sent = 0;           // pairs sent so far: the first ones find the ring empty and need no wait
        const uint32_t full_leader = map_to_cta(full(0), leader);
        bool ok = true;
        QG_DECL();
        for (int jt = 0; jt < my_tiles && ok; ++jt) {
            const Tile tl = tile_at(jt);
            const Piece pc = piece_at(jt);
            const int n_mma = min(BT, (tl.tok_end - tl.tok0 + 15) & ~15);
            const int row0 = tl.tok0 + static_cast<int>(rank) * (n_mma >> 1);   // B rows split at N / 2
            // Gathered input: lane l fetches rows 4 l .. 4 l + 3 of this CTA's half tile from the token rows the
            // routing table names (rows past the segment end fetch token 0: computed, never stored).
            const int groups = n_mma >> 3;                                      // (n_mma / 2) / 4
            int g0 = 0, g1 = 0, g2 = 0, g3 = 0;
            if (p.gather_k > 0 && lane < groups) {
                const int r = row0 + 4 * lane;
                if (r < tl.tok_end) g0 = p.row_pair[r] / p.gather_k;
                if (r + 1 < tl.tok_end) g1 = p.row_pair[r + 1] / p.gather_k;
                if (r + 2 < tl.tok_end) g2 = p.row_pair[r + 2] / p.gather_k;
                if (r + 3 < tl.tok_end) g3 = p.row_pair[r + 3] / p.gather_k;
            }
            for (int kb = pc.kb0; kb < pc.kb1; kb += 2) {
                QG_T0();
                // a stage pair is free once the MMAs that read it eight k-blocks ago are done
                if (sent >= C::SP && !wait_bar(done(s), ph ^ 1u, abort_flag, p)) { ok = false; break; }
                ++sent;
                QG_ACC(0);
                if (jt == 0 && kb == pc.kb0) { QG_MARK(7); }
                const uint32_t dst = sbase + C::OFF_X + s * (2 * C::X_BYTES);
                if (!(jt == 0 && kb == (p.skip_kb & ~1))) {                 // test hook: that pair never fills
                    if (p.gather_k > 0) {
                        if (lane == 0 && rank == 0) mbar_arrive_expect_tx(full(s), 4u * groups * 512u);
                        if (lane < groups) {
                            tma_gather4_pair(dst + lane * 512, &tm_x, kb * BK, g0, g1, g2, g3, full_leader + 8u * s);
                            tma_gather4_pair(dst + C::X_BYTES + lane * 512, &tm_x, (kb + 1) * BK, g0, g1, g2, g3, full_leader + 8u * s);
                        }
                    } else if (elect_one()) {
                        if (rank == 0) mbar_arrive_expect_tx(full(s), 4 * C::X_BYTES);
                        tma_load_3d_pair(dst, &tm_x, 0, row0, kb, full_leader + 8u * s);
                    }
                }
                __syncwarp();
                s = (s + 1u) % C::SP;
                if (s == 0) ph ^= 1u;
            }
        }
        __syncwarp();
        if (lane == 0) QG_FLUSH();
    } else if (warp == 2) {
        // ------------------------------------------------ packed weight + scale producer (local ring)
        uint32_t s = 0, ph = 0, sg = 0;     // first raw stage of the batch (0 or 4), parity, scale buffer
        uint32_t batches = 0;               // batches sent so far: the first SR / 4 find the ring empty and need no wait
        bool ok = true;
        QG_DECL();
        for (int jt = 0; jt < my_tiles && ok; ++jt) {
            const Tile tl = tile_at(jt);
            const Piece pc = piece_at(jt);
            const int wt = 2 * tl.pw + static_cast<int>(rank);
            for (int kb = pc.kb0; kb < pc.kb1; kb += 4) {
                QG_T0();
                if (batches >= C::SR / 4 && !wait_bar(r_empty(s), ph ^ 1u, abort_flag, p)) { ok = false; break; }
                QG_ACC(1);
                if (jt == 0 && kb == pc.kb0) { QG_MARK(8); }
                const bool sent = (batches == 0 && w_pre_issued);       // the first batch left in the prologue
                ++batches;
                if (!sent && elect_one()) {
                    // five copies and one barrier per batch: the 8 scales per row that cover these four k-blocks,
                    // then the packed codes of each k-block
                    mbar_arrive_expect_tx(r_full(s), 4 * C::RAW_BYTES + C::SC_BYTES);
                    load_w(sbase + C::OFF_SC + sg * C::SC_BYTES, &tm_s, (kb >> 2) * 8, tl.e, wt, r_full(s));
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        load_w(sbase + C::OFF_RAW + (s + j) * C::RAW_BYTES, &tm_w, (kb + j) * C::RAW_ROW, tl.e, wt, r_full(s));
                }
                __syncwarp();
                if (++sg == C::NSB) sg = 0;
                s = (s + 4u) & (C::SR - 1);
                if (s == 0) ph ^= 1u;
            }
        }
        __syncwarp();
        if (lane == 0) QG_FLUSH();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer (even CTA of the pair only)
        // Two k-blocks per barrier.  Four MMAs take 120 cycles to issue and the commit 113, about 350 for a pair, and the tensor cores
        // 8 (15 + N / 2) for its eight MMAs, more than that from 64 tokens on (with the test of the next pair's barrier, in a profiling
        // build, 430 to 500).  One issuing thread also fixes the order in which a tile's k-blocks are added.
        if (rank == 0) {
            bool ok = true;
            QG_DECL();
            const uint32_t b_hi = (1024u >> 4) | (1u << 14) | (2u << 29);   // stride, version, 128-byte swizzle
            const uint32_t b_lo0 = ((sbase + C::OFF_X) >> 4) | (1u << 16);
            for (uint32_t j = 0; static_cast<int>(j) < my_tiles && ok; ++j) {
                const Tile tl = tile_at(static_cast<int>(j));
                const Piece pc = piece_at(static_cast<int>(j));
                const int n_mma = min(BT, (tl.tok_end - tl.tok0 + 15) & ~15);
                const uint32_t idesc = umma_idesc_bf16(2 * BW, n_mma);
                const uint32_t a = (C::NACC == 2) ? (j & 1u) : 0u;
                const uint32_t aph = (C::NACC == 2) ? ((j >> 1) & 1u) : (j & 1u);
                QG_T0();
                if (!spin_wait_bar(acc_empty(a), aph ^ 1u, abort_flag, p)) { ok = false; break; }
                QG_ACC(2);
                const uint32_t d_tmem = tmem_base + a * BT;
                uint32_t i = static_cast<uint32_t>(pc.i0);                    // ring index of k-block kb
                bool ready = mbar_test_wait(full((i >> 1) % C::SP), (i >> 3) & 1u);
                for (int kb = pc.kb0; kb < pc.kb1; kb += 2, i += 2) {
                    const uint32_t sp = (i >> 1) % C::SP;
                    QG_T0();
                    if (!ready && !spin_wait_bar(full(sp), (i >> 3) & 1u, abort_flag, p)) { ok = false; break; }
                    QG_ACC(3);
                    if (j == 0 && kb == pc.kb0) { QG_MARK(2); }
                    tc_fence_after_sync();
                    // start the wait for the next pair before issuing, so its latency is hidden
                    ready = (kb + 2 < pc.kb1) && mbar_test_wait(full((sp + 1) % C::SP), ((i + 2) >> 3) & 1u);
                    if (elect_one()) {
                        const uint32_t ta = tmem_base + C::A_COL0 + (i % C::SA) * C::A_COLS;     // TMEM weight stage
                        const uint32_t b_lo = b_lo0 + sp * (2 * C::X_BYTES >> 4);
                        umma_kblock_ts_pair(d_tmem, ta, b_lo, b_hi, idesc, kb != pc.kb0 ? 1u : 0u);
                        umma_kblock_ts_pair(d_tmem, ta + C::A_COLS, b_lo + (C::X_BYTES >> 4), b_hi, idesc, 1u);
                        umma_commit_pair(done(sp), 3u << leader);
                        if (kb + 2 >= pc.kb1) umma_commit_pair(acc_full(a), 3u << leader);
                    }
                    __syncwarp();
                    QG_ACC(10);
                }
                if (static_cast<int>(j) == my_tiles - 1) { QG_MARK(3); }
            }
            __syncwarp();
            if (lane == 0) QG_FLUSH();
        }
    } else if (warp >= 8) {
        // ------------------------------------------------ dequantise: raw ring -> TMEM weight stages
        // Four groups of four warps; group g owns TMEM weight stage g and converts the k-blocks i = g (mod 4), so
        // a warp has four k-block periods for one round of waits, loads, arithmetic and tensor-memory stores.
        // Warp (g, q) covers weight rows 32 q .. 32 q + 31 (a warp may only touch the TMEM lanes of its quarter);
        // thread = one row, all 64 k of the k-block: 64 bytes (Q8) or 32 bytes (Q4) of packed codes, read from the
        // swizzled raw tile without bank conflicts, 2 scales, 32 TMEM columns out.
        const int g = (warp - 8) >> 2, q = warp & 3;
        // In gate/up mode lanes 0-15 of a quarter take gate rows and lanes 16-31 the up rows that belong to them (the raw tile is 64
        // gate rows, then 64 up rows).
        const int row = (EPI == 1) ? ((lane >> 4) << 6) + q * 16 + (lane & 15) : q * 32 + lane;
        const uint32_t swz = (QBITS == 8) ? ((row >> 1) & 3u) : ((row >> 2) & 1u);
        const uint32_t raw_row = row * C::RAW_ROW;
        const uint32_t a_taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + C::A_COL0;
        const uint32_t full_leader = map_to_cta(full(0), leader);
        const uint32_t n_own = own_kb4;
        QG_DECL();
        // Helping with the epilogue.  Before this warp waits for the MMAs of own k-block n - 2 (to reuse their TMEM
        // stage) it must have released every accumulator of an earlier tile, otherwise a single-accumulator pipeline
        // would wait for itself; at that point it has filled the ring for the next tile and would idle anyway.
        auto per_tile = [&](uint32_t t) -> uint32_t {                  // own k-blocks of the pair's t-th tile (piece)
            if constexpr (SK == 0) return static_cast<uint32_t>(nk4);
            if constexpr (SK == 2) return own_kb4;
            const Piece pc = ptab[t];
            return static_cast<uint32_t>(pc.kb1 - pc.kb0) >> 2;
        };
        uint32_t helped = 0;                                           // tiles whose accumulator this warp released
        uint32_t t2 = 0, in2 = 0;                                      // tile of own k-block n - 2, position in it
        const uint32_t acc_empty_leader = map_to_cta(acc_empty(0), leader);
        constexpr bool shared_ep = (EPI < 2);
        __nv_bfloat16* my_st = stg16 + (warp - 8) * 512;               // private 1 KB transposition buffer
        uint32_t ta = static_cast<uint32_t>(g) % C::SA;                 // TMEM weight stage of own k-block i = i % SA
        bool dq_ok = true;
        auto help_tile = [&](uint32_t jt, bool release) -> bool {
            pdl_wait();          // these warps store to the output from here on (returns at once after the first time)
            const Tile tl = tile_at(static_cast<int>(jt));
            const int wt = 2 * tl.pw + static_cast<int>(rank);
            const uint32_t a = (C::NACC == 2) ? (jt & 1u) : 0u;
            const uint32_t aph = (C::NACC == 2) ? ((jt >> 1) & 1u) : (jt & 1u);
            // single accumulator: every tile is helped, so the phases of acc_full are consumed in order; two
            // accumulators: only the last tile is helped, through the one-shot barrier
            if (!wait_bar(C::HELP ? acc_full(a) : last_full, C::HELP ? aph : 0u, abort_flag, p)) return false;
            tc_fence_after_sync();
            if (shared_ep && wt < p.n_wt) {
                const int n_mma = min(BT, (tl.tok_end - tl.tok0 + 15) & ~15);
                if constexpr (EPI == 1)
                    drain_gate_up(p, tl.tok0, tl.tok_end, wt * 64 + q * 16, tmem_base + (static_cast<uint32_t>(q * 32) << 16) + a * BT, n_mma,
                                  1 + g, 5, my_st, lane);
                else if constexpr (SK == 2)
                    dump_partial(partial, tmem_base + (static_cast<uint32_t>(q * 32) << 16) + a * BT, n_mma, 1 + g, 5, q, lane);
                else
                    drain_plain<SK == 1, !C::HELP, false>(p, tl.tok0, tl.tok_end, wt * BW + q * 32,
                            tmem_base + (static_cast<uint32_t>(q * 32) << 16) + a * BT, n_mma, 1 + g, 5, my_st,
                            C::HELP ? nullptr : wts + (jt & 1u) * BT, lane,
                            piece_at(static_cast<int>(jt)).nsrc, q, BT * 128, abort_flag);
            }
            tc_fence_before_sync();
            __syncwarp();
            if (release && lane == 0) mbar_arrive_cluster(acc_empty_leader + 8u * a);
            return true;
        };
        for (uint32_t n = 0; n < n_own && dq_ok; ++n) {       // own k-block i = 4 n + g
            constexpr uint32_t NB = C::SR / 4;                     // batches of four stages in the packed-weight ring
            const uint32_t sr = ((n % NB) << 2) + g;               // ring stage i % SR
            const uint32_t phr = (n / NB) & 1u;                    // parity of (i / SR)
            // (t2 = tile of own k-block n - 2.)  The release must come before this iteration's wait for the MMAs of
            // own k-block n - 2, or the single-accumulator pipeline would wait for itself; it is done first, while
            // no converted weights are held in registers.
            if (C::HELP && n >= 2) {
                while (dq_ok && helped < t2) dq_ok = help_tile(helped++, true);
                if (!dq_ok) break;
                if (++in2 == per_tile(t2)) { in2 = 0; ++t2; }
            }
            QG_T0();
            // the four k-blocks of a batch and their scales arrive on the barrier of the batch's first stage
            if (!wait_bar(r_full((n % NB) << 2), phr, abort_flag, p)) break;
            QG_ACC(5);
            if (n == 0 && warp == 8) { QG_MARK(10); }
            const uint32_t raw = sbase + C::OFF_RAW + sr * C::RAW_BYTES + raw_row;
            const uint32_t scw = *reinterpret_cast<const uint32_t*>(
                sgen + C::OFF_SC + (n % C::NSB) * C::SC_BYTES + row * 16 + g * 4);
            const float s0 = __half2float(__ushort_as_half(static_cast<unsigned short>(scw & 0xFFFFu)));
            const float s1 = __half2float(__ushort_as_half(static_cast<unsigned short>(scw >> 16)));
            uint32_t o[32];
#pragma unroll
            for (int h = 0; h < 2; ++h) {            // k = 32 h .. 32 h + 31 share one scale
                const float sc = h ? s1 : s0;
                uint32_t* oh = o + 16 * h;
                if constexpr (QBITS == 8) {
                    const uint4 v0 = lds128(raw + (((2 * h) ^ swz) << 4));
                    const uint4 v1 = lds128(raw + (((2 * h + 1) ^ swz) << 4));
                    uint64_t m, c;
                    dq8_consts(sc, m, c);
                    dq8_word(v0.x, m, c, DQ_MAGIC, oh[0], oh[1]);
                    dq8_word(v0.y, m, c, DQ_MAGIC, oh[2], oh[3]);
                    dq8_word(v0.z, m, c, DQ_MAGIC, oh[4], oh[5]);
                    dq8_word(v0.w, m, c, DQ_MAGIC, oh[6], oh[7]);
                    dq8_word(v1.x, m, c, DQ_MAGIC, oh[8], oh[9]);
                    dq8_word(v1.y, m, c, DQ_MAGIC, oh[10], oh[11]);
                    dq8_word(v1.z, m, c, DQ_MAGIC, oh[12], oh[13]);
                    dq8_word(v1.w, m, c, DQ_MAGIC, oh[14], oh[15]);
                } else {
                    const uint4 v = lds128(raw + ((h ^ swz) << 4));
                    uint32_t hi2, lo2;
                    dq4_consts(sc, hi2, lo2);
                    dq4_word(v.x, hi2, lo2, oh);
                    dq4_word(v.y, hi2, lo2, oh + 4);
                    dq4_word(v.z, hi2, lo2, oh + 8);
                    dq4_word(v.w, hi2, lo2, oh + 12);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(r_empty((n % NB) << 2));  // the packed codes are in registers now
            QG_ACC(7);
            // its TMEM stage (i % SA) is free once the MMAs of k-block i - SA have completed
            {
                const uint32_t i = 4u * n + g;
                if (i >= C::SA && !wait_bar(done(((i - C::SA) >> 1) % C::SP), ((i - C::SA) >> 3) & 1u, abort_flag, p)) break;
            }
            QG_ACC(6);
            tc_fence_after_sync();
            {
                uint32_t (&o0)[16] = *reinterpret_cast<uint32_t (*)[16]>(o);
                uint32_t (&o1)[16] = *reinterpret_cast<uint32_t (*)[16]>(o + 16);
                tmem_st_32x32_x16(a_taddr + ta * C::A_COLS, o0);
                tmem_st_32x32_x16(a_taddr + ta * C::A_COLS + 16, o1);
            }
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(full_leader + 8u * (((n & 1u) << 1) + (g >> 1)));   // stage pair (i / 2) % 4
            if (n == 0 && warp == 8) { QG_MARK(9); }
            ta += 4;
            if (ta >= C::SA) ta -= C::SA;
            QG_ACC(7);
        }
        while (C::HELP && dq_ok && helped < static_cast<uint32_t>(my_tiles)) dq_ok = help_tile(helped++, true);
        // With two accumulators the epilogues overlap the main loops, except the last one: these warps have nothing
        // left to do then and take four fifths of it (nobody waits for that accumulator again: no release).
        if (!C::HELP && shared_ep && dq_ok && my_tiles > 0) help_tile(static_cast<uint32_t>(my_tiles - 1), false);
        __syncwarp();
        if (warp == 8 && lane == 0) QG_FLUSH();
    } else if (warp >= 4) {
        // ------------------------------------------------ epilogue (warps 4..7 <-> TMEM lanes 32 (warp-4) ..)
        const int qd = warp - 4;
        const int et = threadIdx.x - 128;
        float* outf = static_cast<float*>(p.out);
        const uint32_t acc_empty_base = map_to_cta(acc_empty(0), leader);
        uint32_t j = 0;
        // Routing weights are fetched ahead, a thread the token et (and et + 128) of a tile: the pairs' numbers two tiles ahead, the
        // weights they name one tile ahead.
        const bool weighted = EPI == 0 && !C::HELP && p.mode == QG_MODE_DOWN_WEIGHTED;
        int pr0 = -1, pr1 = -1;
        float w0 = 0.f, w1 = 0.f;
        auto fetch_pairs = [&](int jt) {
            pr0 = pr1 = -1;
            if (jt >= my_tiles) return;
            const Tile tn = tile_at(jt);
            if (tn.tok0 + et < tn.tok_end) pr0 = p.row_pair[tn.tok0 + et];
            if (BT > 128 && tn.tok0 + 128 + et < tn.tok_end) pr1 = p.row_pair[tn.tok0 + 128 + et];
        };
        auto fetch_weights = [&]() {
            w0 = pr0 >= 0 ? p.topk_w[pr0] : 0.f;
            w1 = (BT > 128 && pr1 >= 0) ? p.topk_w[pr1] : 0.f;
        };
        if (weighted) {
            fetch_pairs(0);
            fetch_weights();
            fetch_pairs(1);
        }
        QG_DECL();
        for (; static_cast<int>(j) < my_tiles; ++j) {
            const Tile tl = tile_at(static_cast<int>(j));
            const int wt = 2 * tl.pw + static_cast<int>(rank);     // may be one past the last tile: nothing is stored
            if (weighted) {
                if (et < BT) wts[(j & 1u) * BT + et] = w0;
                if (BT > 128 && et + 128 < BT) wts[(j & 1u) * BT + 128 + et] = w1;
                fetch_weights();
                fetch_pairs(static_cast<int>(j) + 2);
            }
            const uint32_t a = (C::NACC == 2) ? (j & 1u) : 0u;
            const uint32_t aph = (C::NACC == 2) ? ((j >> 1) & 1u) : (j & 1u);
            const uint32_t fl = j & 1u;       // flag slot: alternates so a slow warp never reads a newer flag
            QG_T0();
            if (et == 0) misc[2 + fl] = wait_bar(acc_full(a), aph, abort_flag, p) ? 1 : 0;
            tc_fence_before_sync();
            named_bar_sync(1, 128);
            if (!misc[2 + fl]) break;
            tc_fence_after_sync();
            if (!C::HELP && et == 0 && static_cast<int>(j) == my_tiles - 1) mbar_arrive(last_full);
            QG_ACC(8);
            if (qd == 0 && static_cast<int>(j) == my_tiles - 1) { QG_MARK(4); }
            const int n_mma = min(BT, (tl.tok_end - tl.tok0 + 15) & ~15);
            const uint32_t taddr = tmem_base + (static_cast<uint32_t>(qd * 32) << 16) + a * BT;
            const int n_epi = (wt < p.n_wt) ? n_mma : 0;
            if constexpr (EPI == 0) {
                // shared with the dequantising warps (participants 1..4 of this lane quarter) when they help
                if constexpr (SK == 2) dump_partial(partial, taddr, n_epi, 0, 5, qd, lane);
                else drain_plain<SK == 1, !C::HELP, !C::HELP>(p, tl.tok0, tl.tok_end, wt * BW + qd * 32, taddr, n_epi, 0,
                            (C::HELP || static_cast<int>(j) == my_tiles - 1) ? 5 : 1,
                            stg16 + 16 * 512 + qd * (C::EPI_ST / 2), C::HELP ? nullptr : wts + (j & 1u) * BT, lane,
                            piece_at(static_cast<int>(j)).nsrc, qd, BT * 128, abort_flag);
            } else if constexpr (EPI == 1) {
                drain_gate_up(p, tl.tok0, tl.tok_end, wt * 64 + qd * 16, taddr, n_epi, 0,
                              (C::HELP || static_cast<int>(j) == my_tiles - 1) ? 5 : 1, stg16 + 16 * 512 + qd * (C::EPI_ST / 2), lane);
            } else {
                for (int c = 0; c < n_epi; c += 32) {
                    uint32_t v[32];
                    tmem_ld_32x32(taddr + c, v);
                    tmem_ld_wait();
                    // y[token, n] += w * acc: lanes are consecutive n, so each warp-wide red covers 128 bytes
                    const int n = wt * BW + qd * 32 + lane;
                    const int tokl = tl.tok0 + c + lane;
                    int trow = 0;
                    float wv = 0.f;
                    if (tokl < tl.tok_end) {
                        const int pr = p.row_pair[tokl];
                        wv = p.topk_w[pr];
                        trow = pr / p.k;
                    }
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj) {
                        const float w = __shfl_sync(0xFFFFFFFFu, wv, jj);
                        const int tr = __shfl_sync(0xFFFFFFFFu, trow, jj);
                        if (tl.tok0 + c + jj < tl.tok_end && n < p.N)
                            atomicAdd(outf + static_cast<size_t>(tr) * p.N + n, w * __uint_as_float(v[jj]));
                    }
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(acc_empty_base + 8u * a);
            QG_ACC(9);
            if (qd == 0 && static_cast<int>(j) == my_tiles - 1) { QG_MARK(5); }
        }
        if (et == 0) QG_FLUSH();
    }

    // ---------------------------------------------------- K slices: sum over the cluster
    if constexpr (SK == 2) {
        __syncthreads();
        cluster_sync_all();          // every slice's fragments are in place
        const Tile tl = tab[0];
        const int wt = 2 * tl.pw + static_cast<int>(rank);
        if (warp >= 4 && wt < p.n_wt && !*abort_flag) {
            pdl_wait();
            const int units = ((tl.tok_end - tl.tok0 + 15) >> 4) * 4;
            for (int u = (warp - 4) * p.slices + slice; u < units; u += 20 * p.slices)
                sum_block(p, smem_u32(partial), rank, u, tl.tok0, tl.tok_end, wt * BW,
                          stg16 + (warp >= 8 ? (warp - 8) * 512 : 16 * 512 + (warp - 4) * (C::EPI_ST / 2)), lane);
        }
    }

    // ---------------------------------------------------- teardown
    __syncthreads();
    if (warp == 0) { QG_MARK(6); }
    if (*abort_flag) {
        // copies may still be in flight towards this CTA's shared memory: give them time to land
        for (int i = 0; i < 64; ++i) __nanosleep(2000);
    }
    tc_fence_before_sync();
    cluster_sync_all();          // the peer no longer reads this CTA's shared memory or signals its barriers
    tc_fence_after_sync();
    if (warp == 3) tmem_dealloc_pair(tmem_base, C::TMEM_COLS);
    QG_SPAN(1);
}

template <int QBITS, int BT, int EPI, int SK>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NTHREADS, 1)
qgemm_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
             const __grid_constant__ CUtensorMap tm_s, const GemmParams p) {
    gemm_body<QBITS, BT, EPI, SK>(tm_x, tm_w, tm_s, p);
}
// Grouped, behind a launch of the streaming kernel: whether this one has the work follows from the offsets.
template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NTHREADS, 1)
qgemm_choice_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                    const __grid_constant__ CUtensorMap tm_s, const GemmParams p, const GroupedChoice choice) {
    pdl_launch_dependents();
    // The kernel in front lets this one start only when the offsets are there (it has waited for them), so they are read before its
    // end, past the L1 cache, by every warp for itself: a launch that is not wanted ends before it has set anything up.
    int chunks = 0, wide = 0;
    for (int e = threadIdx.x & 31; e < p.E; e += 32) {
        const int cnt = __ldcg(p.offsets + e + 1) - __ldcg(p.offsets + e);
        chunks += (cnt + choice.chunk - 1) / choice.chunk;
        wide += (cnt + 127) >> 7;
    }
    if (choice.streams(__reduce_add_sync(0xFFFFFFFFu, chunks), __reduce_add_sync(0xFFFFFFFFu, wide))) {
        // the kernel behind this one waits for this one alone, so one pair waits for the kernel in front; the others leave their
        // SMs to the kernel behind
        if (blockIdx.x < 2) pdl_wait();
        return;
    }
    gemm_body<4, 128, EPI, 0>(tm_x, tm_w, tm_s, p);
}
// K slices: the launch names the cluster size (two CTAs per slice)
template <int QBITS, int BT>
__global__ void __launch_bounds__(NTHREADS, 1)
qgemm_slices_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                    const __grid_constant__ CUtensorMap tm_s, const GemmParams p) {
    gemm_body<QBITS, BT, 0, 2>(tm_x, tm_w, tm_s, p);
}
// clusters of 2 * slices CTAs of the kernel above that fit on the GPU at once (asked once per context, kernel and size)
template <int QBITS, int BT>
static int slices_capacity(qg_ctx* ctx, int slices) {
    constexpr int inst = (QBITS == 4 ? 2 : 0) + (BT == 128 ? 0 : 1);
    int& cached = ctx->slice_clusters[inst][slices];
    if (cached == 0) {
        constexpr int smem = Cfg<QBITS, BT>::SMEM_BYTES;
        auto kern = qgemm_slices_kernel<QBITS, BT>;
        cudaLaunchConfig_t q = {};
        cudaLaunchAttribute ca;
        ca.id = cudaLaunchAttributeClusterDimension;
        ca.val.clusterDim.x = 2 * slices; ca.val.clusterDim.y = 1; ca.val.clusterDim.z = 1;
        q.gridDim = dim3(2 * slices); q.blockDim = dim3(NTHREADS); q.dynamicSmemBytes = smem; q.attrs = &ca; q.numAttrs = 1;
        int n = 0;
        // a plan may be asked for with another device current: attribute and answer are those of the context's device
        const OnDevice here(ctx->device);
        if (!here.ok || cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kern, &q) != cudaSuccess) { cudaGetLastError(); n = 0; }
        cached = n > 0 ? n : -1;
    }
    return cached;
}

template <int QBITS, int BT, int EPI, int SK>
static int launch_gemm(qg_ctx* ctx, const GemmParams& p, const void* X, int x_rows, const void* Wq, const void* Ws,
                       cudaStream_t st, const GroupedChoice* choice = nullptr) {
    using C = Cfg<QBITS, BT>;
    static_assert(C::SMEM_BYTES <= 232448, "shared memory budget");
    CUtensorMap tm_x, tm_w, tm_s;       // cached in the context: the same buffers recur every layer and step
    const uint64_t wrows = static_cast<uint64_t>(p.E) * p.N;
    // activations: a box of half a token tile and two k-blocks, which land one after the other (a view [K / 64][rows][64]), or
    // of a single row when the rows are gathered four at a time
    int rc = p.gather_k > 0 ? get_tmap_2d(ctx, &tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, X, p.K, x_rows, BK, 1, CU_TENSOR_MAP_SWIZZLE_128B)
                            : get_tmap_3d(ctx, &tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, X, BK, x_rows, p.K / BK, 2 * BK, BK,
                                          C::XH_ROWS, 2, CU_TENSOR_MAP_SWIZZLE_128B, 2ull * p.K);
    // weights and scales: a box of this CTA's 128 rows; in gate/up mode 64 gate rows + 64 up rows, as two planes of a
    // 3-D view (k, row within a half, half of an expert's matrix)
    const uint64_t kbytes = (QBITS == 8) ? p.K : p.K / 2;
    const CUtensorMapSwizzle wswz = (QBITS == 8) ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
    if (rc == QG_OK)
        rc = (EPI == 1) ? get_tmap_3d(ctx, &tm_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, kbytes, p.N / 2, 2ull * p.E,
                                      kbytes * (p.N / 2), C::RAW_ROW, 64, 2, wswz)
                        : get_tmap_2d(ctx, &tm_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, kbytes, wrows, C::RAW_ROW, 128, wswz);
    if (rc == QG_OK)
        rc = (EPI == 1) ? get_tmap_3d(ctx, &tm_s, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, Ws, p.K / 32, p.N / 2, 2ull * p.E,
                                      static_cast<uint64_t>(p.K / 32) * 2 * (p.N / 2), 8, 64, 2, CU_TENSOR_MAP_SWIZZLE_NONE)
                        : get_tmap_2d(ctx, &tm_s, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, Ws, p.K / 32, wrows, 8, 128,
                                      CU_TENSOR_MAP_SWIZZLE_NONE);
    if (rc != QG_OK) return rc;
    if constexpr (SK == 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * p.slices * static_cast<unsigned>(((p.n_wt + 1) / 2) * ((p.R + BT - 1) / BT)));
        cfg.blockDim = dim3(NTHREADS); cfg.dynamicSmemBytes = C::SMEM_BYTES; cfg.stream = st;
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2 * p.slices; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at; cfg.numAttrs = ctx->pdl ? 2 : 1;
        if (cudaLaunchKernelEx(&cfg, qgemm_slices_kernel<QBITS, BT>, tm_x, tm_w, tm_s, p) == cudaSuccess) return QG_OK;
        // refused although the occupancy query allowed it: remember that and leave K whole
        cudaGetLastError();
        ctx->slice_clusters[(QBITS == 4 ? 2 : 0) + (BT == 128 ? 0 : 1)][p.slices] = -1;
        GemmParams whole = p;
        whole.slices = 1;
        return launch_gemm<QBITS, BT, EPI, 0>(ctx, whole, X, x_rows, Wq, Ws, st);
    } else {
        auto kern = qgemm_kernel<QBITS, BT, EPI, SK>;
        // the shared-memory attribute belongs to the function on one device: set once per context and instantiation
        constexpr int inst = SK == 1 ? ATTR_GEMM_SK + ((QBITS == 4) ? 3 : 0) + ((BT == 128) ? 0 : (BT == 192) ? 1 : 2)
                                : ATTR_GEMM + ((QBITS == 4) ? 9 : 0) + ((BT == 128) ? 0 : (BT == 192) ? 3 : 6) + EPI;
        if (!ctx->attr_set[inst]) {
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES) != cudaSuccess) {
                cudaGetLastError();
                return QG_ERR_CUDA;
            }
            ctx->attr_set[inst] = true;
        }
        // Upper bound on the number of pair tiles (the exact count lives on the device for grouped calls).
        long long max_tiles =
            (static_cast<long long>((p.R + BT - 1) / BT) + (p.offsets ? p.E : 0)) * ((p.n_wt + 1) / 2);
        if (p.streamk) max_tiles *= p.K / (4 * BK);      // units of four k-blocks: every pair gets at least one
        const long long pairs_hw = ctx->sm_count / 2;
        const int grid = 2 * static_cast<int>(max_tiles < pairs_hw ? max_tiles : pairs_hw);
        cudaError_t e = cudaSuccess;
        if constexpr (QBITS == 4 && BT == 128 && SK == 0 && EPI < 2) {
            if (choice) {
                if (!ctx->attr_set[ATTR_GEMM_CHOICE + EPI]) {
                    e = cudaFuncSetAttribute(qgemm_choice_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
                    ctx->attr_set[ATTR_GEMM_CHOICE + EPI] = e == cudaSuccess;
                }
                if (e == cudaSuccess)
                    e = launch_kernel(ctx, qgemm_choice_kernel<EPI>, dim3(grid), dim3(NTHREADS), C::SMEM_BYTES, st, tm_x, tm_w, tm_s, p, *choice);
                if (e != cudaSuccess) cudaGetLastError();
                return e == cudaSuccess ? QG_OK : QG_ERR_CUDA;
            }
        }
        e = launch_kernel(ctx, kern, dim3(grid), dim3(NTHREADS), C::SMEM_BYTES, st, tm_x, tm_w, tm_s, p);
        if (e != cudaSuccess) cudaGetLastError();
        return e == cudaSuccess ? QG_OK : QG_ERR_CUDA;
    }
}

// Token tile and schedule of a dense call: the candidate with the smallest modelled time in ns, fitted to 1300 calls timed back to back on
// B200 (Q8 and Q4, plain and gate/up, N from 136 to 28672, K from 512 to 16384, 17 to 4096 tokens; every candidate of each).  There the choice
// takes 1.004 of the time of the fastest candidate on average, 1.12 at worst; over 904 unsliced calls of 24 layers timed afterwards, five of
// them new to the model, 1.008 and 1.17 (4096 x 14336, 4 bit, 1800 tokens: 195 us, by stream-K 167).
// Data-parallel: a tile costs nkb k-blocks of `period` plus, for the single-accumulator 256-token tile, an exposed epilogue;
// tiles come in waves of one per SM pair, but a ragged last wave costs less than a full one (the pairs that are done leave L2,
// HBM and power to the others), so the wave count is taken about half-way between the rounded-up and the fractional one, and of a
// single wave as 0.77 + 0.23 of the share of the pairs that have a tile.  16384 x 3072 gate/up, 4 bit, 200 tokens: 29.4 us with 192-token
// tiles, 20.3 with 256; 1024 tokens 80.1 and 74.8; 4096 x 4096, 8 bit, 4096 tokens: 92.7 and 99.9.
// Stream-K: every pair gets the same share of all k-blocks; the pair with a tile's first k-block adds the parts of all pairs that have
// others one after another, 930 ns and 5.6 a token for each.  4096 x 14336: at 2500 tokens (2.2 waves) 244 us against 293 data-parallel, at
// 1500 (1.7) 154 and 154.  Few tiles have many parts each: 512 x 16384 at 128 tokens, 37 parts, 73 us against 60 whole and 21 in four slices.
// Not from 5.5 waves on: what a ragged last one leaves idle is a tenth of the call at most, and its idle pairs leave their power to the others.
// 28672 x 4096, 8 bit: 1024 tokens (6.05 waves of 256-token tiles) 195 us by stream-K, 179 data-parallel, 2500 tokens 466 and 425; 14336 x 4096,
// 2048 tokens 179 and 170; three waves (28672 x 4096, 400 tokens) 91.7 and 106.
struct DensePlan {
    int bt, streamk;
    int slices, kc;      // > 1: K slices of kc k-blocks on the CTA pairs of a cluster
};
static int slices_capacity(qg_ctx* ctx, int qbits, int bt, int slices) {
    if (qbits == QG_Q8) return bt == 128 ? slices_capacity<8, 128>(ctx, slices) : slices_capacity<8, 192>(ctx, slices);
    return bt == 128 ? slices_capacity<4, 128>(ctx, slices) : slices_capacity<4, 192>(ctx, slices);
}
// Few tiles leave most SM pairs idle behind a serial walk over K.  Cutting K into two to four slices, one per pair of a
// cluster that adds its partial tiles through distributed shared memory, divides the walk; the sum costs 525 + 620 (slices - 2) ns and
// 9.5 + 2.4 (slices - 2) per token of the tile (a k-block of such a short walk being 245 ns with up to 128 tokens and 286 with 192, and 271
// of a whole walk of several 128-token tiles).  Unless the alternative is stream-K, slices take SMs that the next launch could start on:
// 380 ns from a quarter of the SM pairs on and 1430 from 0.45 of them on (two slices, K = 1024, 17 tokens: 24 tiles 8.0 us against 7.5 whole,
// 32 tiles 8.8 against 7.9, 16 tiles 6.7 against 7.4).  All clusters have to be resident at once: 33 / 22 / 15 with two / three / four
// slices, so this is for at most 33 tiles.  Measured, 20 / 128 tokens: 3072 x 3072 16.5 / 17.3 us whole, 10.0 / 12.3 in four
// slices; 5120 x 3072 16.7 / 17.7, 11.3 / 13.3 in three; 2048 x 8192 24.8 / 30.1 (stream-K), 14.1 / 16.8 in four; 4096 x 14336
// 29.2 / 34.1 (stream-K), 26.7 / 29.6 in three.
constexpr double PLAN_START = 5000.0;        // start and end of any call
// `whole_ns`: the time of the plan as it is, PLAN_START included
static void plan_slices(qg_ctx* ctx, int qbits, int M, int n_wt, int K, double whole_ns, DensePlan& plan) {
    if (ctx->force_bt || ctx->streamk_mode != -1) return;
    const long long pairs = ctx->sm_count / 2, n_pw = (n_wt + 1) / 2;
    const int nk4 = K / (4 * BK);
    const long long tiles0 = n_pw * ((M + plan.bt - 1) / plan.bt);
    if (tiles0 > pairs) return;
    auto period = [](int bt) { return bt == 128 ? 245.0 : bt == 192 ? 286.0 : 343.0; };
    const bool streamk = plan.streamk != 0;
    double best = 0.97 * (streamk ? whole_ns - PLAN_START : nk4 * 4.0 * (plan.bt == 128 && M > 128 ? 271.0 : period(plan.bt)));
    for (int bt = 128; bt <= 192; bt += 64) {
        if (bt > 128 && M <= 128) break;
        const long long tiles = n_pw * ((M + bt - 1) / bt);
        for (int sl = 2; sl <= 4 && sl <= nk4 && tiles * sl <= pairs; ++sl) {
            const int per = (nk4 + sl - 1) / sl;
            if ((nk4 + per - 1) / per != sl) continue;             // the same cut as a smaller count
            const double cost = per * 4.0 * period(bt) + 525.0 + 620.0 * (sl - 2) + (9.5 + 2.4 * (sl - 2)) * (M < bt ? M : bt) +
                                (streamk || 4 * tiles * sl < pairs ? 0.0 : 20 * tiles * sl < 9 * pairs ? 380.0 : 1430.0);
            if (cost < best && slices_capacity(ctx, qbits, bt, sl) >= tiles) {
                best = cost;
                plan = DensePlan{bt, 0, sl, 4 * per};
            }
        }
    }
}
static DensePlan plan_whole(const qg_ctx* ctx, int qbits, int M, int n_wt, int K, bool streamk, double* ns = nullptr) {
    const int cand[3] = {128, 192, 256};
    // 128-token tiles: with 4 bit 0.90 to 1.06 of the time of 192-token ones where both are a single wave, with 8 bit 0.02 less.  4 bit, 3072 x 3072,
    // 512 tokens 18.4 us with 128, 17.5 with 192; 8 bit, 8192 x 8192, 256 tokens 37.0 whole with 128, 38.8 by stream-K with 256.
    const double period[3] = {!streamk ? 285.0 : qbits == QG_Q8 ? 279.0 : 288.0, 300.0, 377.0};
    const double epilogue[3] = {0.0, 0.0, 2200.0}, start[3] = {PLAN_START, PLAN_START, PLAN_START - 1750.0};
    const double sk_period[3] = {295.0, 311.0, 394.0}, sk_start[3] = {8400.0, 8400.0, 11000.0};
    const long long pairs = ctx->sm_count / 2, n_pw = (n_wt + 1) / 2;
    const int nk4 = K / (4 * BK);
    DensePlan best{256, 0, 1, 0};
    double best_cost = 1e300;
    for (int c = 0; c < 3; ++c) {
        if (M <= 128 && cand[c] > 128) break;
        const long long tiles = n_pw * ((M + cand[c] - 1) / cand[c]);
        const double frac = static_cast<double>(tiles) / pairs;
        const double waves = tiles <= pairs ? 0.77 + 0.23 * frac : 0.55 * static_cast<double>((tiles + pairs - 1) / pairs) + 0.45 * frac;
        // (gate/up: the single accumulator has to be clearly faster; at 3000 tokens and more the two are level within the clock's drift)
        const double dp = (start[c] + waves * ((K / BK) * period[c] + epilogue[c])) * (!streamk && cand[c] == 256 ? 1.03 : 1.0);
        if (!streamk || ctx->streamk_mode != 1 || tiles % pairs == 0)
            if (dp < best_cost) { best_cost = dp; best = DensePlan{cand[c], 0, 1, 0}; }
    }
    // Below K = 4096 the exchange never paid in the measurements (K = 2048 and 3072, 64 to 1024 tokens: 2 to 10 us slower).
    const double whole_cost = best_cost;
    for (int c = 0; c < 3; ++c) {
        if (!streamk || ctx->streamk_mode == 0 || (ctx->streamk_mode != 1 && nk4 < 16)) break;
        if (M <= 128 && cand[c] > 128) break;
        const long long tiles = n_pw * ((M + cand[c] - 1) / cand[c]);
        if (tiles % pairs == 0 || (ctx->streamk_mode != 1 && 2 * tiles > 11 * pairs)) continue;
        const long long units = tiles * nk4;
        const long long P = units < pairs ? units : pairs;
        const long long share = (units + P - 1) / P;                        // units of the busiest pair
        if (share / nk4 + 2 > 120) continue;                                // the piece table has 128 entries
        const double sk = sk_start[c] + share * 4.0 * sk_period[c] + static_cast<double>(P) / tiles * (930.0 + 5.6 * (M < cand[c] ? M : cand[c]));
        if (ctx->streamk_mode == 1 ? (best.streamk == 0 || sk < best_cost) : (sk < best_cost && sk < 0.96 * whole_cost)) {
            best_cost = sk;
            best = DensePlan{cand[c], 1, 1, 0};
        }
    }
    if (ns) *ns = best_cost;
    return best;
}
static DensePlan plan_dense(qg_ctx* ctx, int qbits, int M, int n_wt, int K) {
    double ns = 0.0;
    DensePlan plan = plan_whole(ctx, qbits, M, n_wt, K, true, &ns);
    plan_slices(ctx, qbits, M, n_wt, K, ns, plan);
    return plan;
}

static int dispatch_gemm(qg_ctx* ctx, int qbits, int bt, const GemmParams& p_in, const void* X, int x_rows,
                         const void* Wq, const void* Ws, cudaStream_t st, const GroupedChoice* choice = nullptr) {
    GemmParams p = p_in;
    if (ctx->force_bt) bt = ctx->force_bt;       // QG_FORCE_BT, read when the context was created (tile-shape sweeps)
    p.status = ctx->d_status;
    p.wait_limit = ctx->wait_limit;
    p.skip_kb = ctx->skip_kb;
    ctx->skip_kb = -1;                           // the test hook acts on one launch
#ifdef QG_PROFILE
    p.stats = ctx->stats;
#endif
    const int epi = (p.mode == QG_MODE_GATE_UP_SILU) ? 1 : (p.mode == QG_MODE_DOWN_ACCUM_F32) ? 2 : 0;
#define QG_LAUNCH(Q, B)                                                                 \
    do {                                                                                \
        if (epi == 0 && p.streamk) return launch_gemm<Q, B, 0, 1>(ctx, p, X, x_rows, Wq, Ws, st);       \
        if (epi == 0) return launch_gemm<Q, B, 0, 0>(ctx, p, X, x_rows, Wq, Ws, st, choice);            \
        if (epi == 1) return launch_gemm<Q, B, 1, 0>(ctx, p, X, x_rows, Wq, Ws, st, choice);            \
        return launch_gemm<Q, B, 2, 0>(ctx, p, X, x_rows, Wq, Ws, st);                                  \
    } while (0)
    if (p.slices > 1) {
        if (qbits == QG_Q8)
            return (bt == 128) ? launch_gemm<8, 128, 0, 2>(ctx, p, X, x_rows, Wq, Ws, st) : launch_gemm<8, 192, 0, 2>(ctx, p, X, x_rows, Wq, Ws, st);
        return (bt == 128) ? launch_gemm<4, 128, 0, 2>(ctx, p, X, x_rows, Wq, Ws, st) : launch_gemm<4, 192, 0, 2>(ctx, p, X, x_rows, Wq, Ws, st);
    }
    if (qbits == QG_Q8) {
        if (bt == 256) QG_LAUNCH(8, 256);
        if (bt == 192) QG_LAUNCH(8, 192);
        QG_LAUNCH(8, 128);
    }
    if (bt == 256) QG_LAUNCH(4, 256);
    if (bt == 192) QG_LAUNCH(4, 192);
    QG_LAUNCH(4, 128);
#undef QG_LAUNCH
}

}  // namespace qg

extern "C" {

int qg_plan_dense(qg_ctx* ctx, int qbits, int M, int N, int K, int* token_tile, int* streamk) {
    if (!ctx) return QG_ERR_NULL;
    if (qbits != QG_Q8 && qbits != QG_Q4) return QG_ERR_SHAPE;
    if (M < 1 || N < 8 || N % 8 || K < 256 || K % 256) return QG_ERR_SHAPE;
    const qg::DensePlan plan = qg::plan_dense(ctx, qbits, M, (N + qg::BW - 1) / qg::BW, K);
    if (token_tile) *token_tile = ctx->force_bt ? ctx->force_bt : plan.bt;
    if (streamk) *streamk = (ctx->force_bt == 0 || ctx->streamk_mode == 1) ? plan.streamk : 0;
    return QG_OK;
}

int qg_plan_slices(qg_ctx* ctx, int qbits, int M, int N, int K, int* slices) {
    if (!ctx || !slices) return QG_ERR_NULL;
    if (qbits != QG_Q8 && qbits != QG_Q4) return QG_ERR_SHAPE;
    if (M < 1 || N < 8 || N % 8 || K < 256 || K % 256) return QG_ERR_SHAPE;
    *slices = qg::plan_dense(ctx, qbits, M, (N + qg::BW - 1) / qg::BW, K).slices;
    return QG_OK;
}

int qgemm_dense(qg_ctx* ctx, int qbits, int M, int N, int K, const void* A, const void* Wq, const void* Wscale,
                void* Cout, void* stream) {
    if (!ctx) return QG_ERR_NULL;
    if (qbits != QG_Q8 && qbits != QG_Q4) return QG_ERR_SHAPE;
    if (M < 0 || N < 8 || N % 8 || K < 256 || K % 256) return QG_ERR_SHAPE;
    if (M == 0) return QG_OK;     // nothing to do: empty tensors may carry null pointers
    if (!A || !Wq || !Wscale || !Cout) return QG_ERR_NULL;
    if (!qg::aligned16(A) || !qg::aligned16(Wq) || !qg::aligned16(Wscale) || !qg::aligned16(Cout)) return QG_ERR_ALIGN;
    if (const int rc = qg::check_device(ctx)) return rc;
    qg::GemmParams p{};
    p.mode = QG_MODE_PLAIN; p.R = M; p.N = N; p.K = K; p.E = 1; p.k = 1;
    p.n_wt = (N + qg::BW - 1) / qg::BW;
    p.offsets = nullptr; p.out = Cout; p.topk_w = nullptr; p.row_pair = nullptr;
    const qg::DensePlan plan = qg::plan_dense(ctx, qbits, M, p.n_wt, K);
    p.streamk = (ctx->force_bt == 0 || ctx->streamk_mode == 1) ? plan.streamk : 0;
    p.slices = plan.slices; p.kc = plan.kc;
    p.sk_partial = ctx->sk_partial; p.sk_flags = ctx->sk_flags;
    return qg::dispatch_gemm(ctx, qbits, plan.bt, p, A, M, Wq, Wscale, static_cast<cudaStream_t>(stream));
}

int qgemm_dense_gate_up_silu(qg_ctx* ctx, int qbits, int M, int F, int K, const void* A, const void* Wq,
                             const void* Wscale, void* Out, void* stream) {
    if (!ctx) return QG_ERR_NULL;
    if (qbits != QG_Q8 && qbits != QG_Q4) return QG_ERR_SHAPE;
    if (M < 0 || F < 64 || F % 64 || K < 256 || K % 256) return QG_ERR_SHAPE;
    if (M == 0) return QG_OK;
    if (!A || !Wq || !Wscale || !Out) return QG_ERR_NULL;
    if (!qg::aligned16(A) || !qg::aligned16(Wq) || !qg::aligned16(Wscale) || !qg::aligned16(Out)) return QG_ERR_ALIGN;
    if (const int rc = qg::check_device(ctx)) return rc;
    qg::GemmParams p{};      // one segment [0, M), the gate/up epilogue of the grouped kernel
    p.mode = QG_MODE_GATE_UP_SILU; p.R = M; p.N = 2 * F; p.K = K; p.E = 1; p.k = 1;
    p.n_wt = (2 * F) / 128;
    p.offsets = nullptr; p.out = Out; p.topk_w = nullptr; p.row_pair = nullptr;
    const int bt = qg::plan_whole(ctx, qbits, M, p.n_wt, K, false).bt;
    return qg::dispatch_gemm(ctx, qbits, bt, p, A, M, Wq, Wscale, static_cast<cudaStream_t>(stream));
}

static int grouped_impl(qg_ctx* ctx, int mode, int qbits, int R, int E, int N, int K, const void* Ain, int in_rows,
                        int gather_k, const int32_t* expert_offsets, const void* Wq, const void* Wscale,
                        const float* topk_w, const int32_t* row_pair, int k, void* Out, void* stream) {
    if (!ctx) return QG_ERR_NULL;
    if (R == 0) return QG_OK;     // nothing to do: empty tensors may carry null pointers
    if (!Ain || !expert_offsets || !Wq || !Wscale || !Out) return QG_ERR_NULL;
    if (qbits != QG_Q8 && qbits != QG_Q4) return QG_ERR_SHAPE;
    if (mode < QG_MODE_PLAIN || mode > QG_MODE_DOWN_ACCUM_F32) return QG_ERR_SHAPE;
    if (R < 0 || E < 1 || E > qg::MAX_E || N < 8 || N % 8 || K < 256 || K % 256) return QG_ERR_SHAPE;
    if (mode == QG_MODE_GATE_UP_SILU && (N % 128)) return QG_ERR_SHAPE;  // F % 64 == 0
    if ((mode >= QG_MODE_DOWN_WEIGHTED || gather_k > 0) && !row_pair) return QG_ERR_NULL;
    if (mode >= QG_MODE_DOWN_WEIGHTED && !topk_w) return QG_ERR_NULL;
    if ((mode == QG_MODE_DOWN_ACCUM_F32 || gather_k > 0) && k < 1) return QG_ERR_SHAPE;
    if (gather_k > 0 && in_rows < 1) return QG_ERR_SHAPE;
    if (static_cast<long long>(E) * N > 0x7FFFFFFF) return QG_ERR_SHAPE;
    if (!qg::aligned16(Ain) || !qg::aligned16(Wq) || !qg::aligned16(Wscale) || !qg::aligned16(Out)) return QG_ERR_ALIGN;
    if (const int rc = qg::check_device(ctx)) return rc;
    qg::GemmParams p{};
    p.mode = mode; p.R = R; p.N = N; p.K = K; p.E = E; p.k = (k < 1) ? 1 : k;
    p.n_wt = (mode == QG_MODE_GATE_UP_SILU) ? (N / 128) : (N + qg::BW - 1) / qg::BW;
    p.gather_k = gather_k;
    p.offsets = expert_offsets; p.out = Out; p.topk_w = topk_w; p.row_pair = row_pair;
    // Expected rows per expert decide the token tile: a 192-token tile spares an expert with 129 to 192 rows the second conversion of its
    // weights.  192 against 128 tokens over eight layers of 8 to 512 experts, rows drawn evenly / with a quarter of the experts preferred:
    // 4 bit, 19 rows per expert 0.98 / 0.98, 64 rows 1.00 / 0.83, 96 rows 1.00 / 0.99, 128 rows 0.76 / 0.88; 8 bit 19 rows 1.01 / 1.01, 48 rows
    // 1.01 / 0.99, 64 rows 1.01 / 0.88, 80 rows 1.01 / 0.95, 96 rows 1.02 / 1.03, 128 rows 0.81 / 0.92.  (Behind the streaming kernel the tile
    // is 128 tokens, so the 4-bit line is where that kernel ends: GroupedChoice::MAX_ROWS.)
    //   Gathered rows and fp32 sums cost a tile time by the row where sorted rows are bound by the conversion, and so do the stores of a short
    // K (the epilogue is the pace): there a tile of few rows is as dear as one of about 100, and 230 rows in 192 + 38 dearer than in 128 + 102, so
    // an expert's tiles are made equally long.  200 rows per expert, 128 experts, 4 bit, gathered 1536 x 2048 584 -> 444 us, fp32 sums
    // 2048 x 768 271 -> 204, weighted 2048 x 768 105 -> 99; sorted rows of K = 1024 on 1.00 (K = 4096, 450 rows 1.04: not for them).  Between 65
    // and 100 rows 128-token tiles are the better ones for the first two (a quarter preferred, 80 rows: 0.83 to 0.98 of the time of 192; evenly
    // drawn 1.00), for fp32 sums up to K = 1536 (0.85 to 1.02 there, 1.11 at K = 3072).
    const int rows = R / E;
    const bool by_row = gather_k > 0 || mode == QG_MODE_DOWN_ACCUM_F32;
    p.even_tiles = by_row || K <= 768;
    const bool short_tiles = (gather_k > 0 || (by_row && K <= 1536)) && rows > 64 && rows <= 100;
    const int bt = (rows > (qbits == QG_Q4 ? qg::GroupedChoice::MAX_ROWS : 50) && !short_tiles) ? 192 : 128;
    // a few rows per expert (4-bit weights, no accumulation) the streaming kernel is faster; the gathering form takes the same
    // kernel as the form for sorted rows, so that they give the same numbers
    qg::GroupedChoice choice{};
    if (qbits == QG_Q4 && mode <= QG_MODE_DOWN_WEIGHTED && ctx->force_bt == 0) {
        const int rc = qg::launch_moe_stream(ctx, mode, R, E, N, K, Ain, in_rows, gather_k, expert_offsets, Wq, Wscale, topk_w, row_pair, Out,
                                             choice, static_cast<cudaStream_t>(stream));
        if (rc != QG_ERR_WORKSPACE && (rc != QG_OK || !choice.on)) return rc;
    }
    return qg::dispatch_gemm(ctx, qbits, bt, p, Ain, in_rows, Wq, Wscale, static_cast<cudaStream_t>(stream), choice.on ? &choice : nullptr);
}

int moe_grouped_qgemm(qg_ctx* ctx, int mode, int qbits, int R, int E, int N, int K, const void* Ain,
                      const int32_t* expert_offsets, const void* Wq, const void* Wscale, const float* topk_w,
                      const int32_t* row_pair, int k, void* Out, void* stream) {
    return grouped_impl(ctx, mode, qbits, R, E, N, K, Ain, R, 0, expert_offsets, Wq, Wscale, topk_w, row_pair, k, Out,
                        stream);
}

int moe_grouped_qgemm_gather(qg_ctx* ctx, int mode, int qbits, int M, int R, int E, int N, int K, const void* X,
                             const int32_t* row_pair, int k, const int32_t* expert_offsets, const void* Wq,
                             const void* Wscale, const float* topk_w, void* Out, void* stream) {
    if (M < 1 && R > 0) return QG_ERR_SHAPE;
    return grouped_impl(ctx, mode, qbits, R, E, N, K, X, M, k, expert_offsets, Wq, Wscale, topk_w, row_pair, k, Out,
                        stream);
}

}  // extern "C"
