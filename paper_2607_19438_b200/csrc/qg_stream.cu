// The weight-streaming GEMM: one matrix and up to sixteen tokens (qgemm_small_m), or the 4-bit expert matrices of a routed
// layer with a few rows per expert (moe_grouped_qgemm and its gathering form: plain, gate/up + SiLU, routing-weighted).
//
// Every weight byte is used for a handful of token rows only, so the call is a streaming read of the packed weights: 39
// 4-bit or 21 8-bit weights per clock and SM at HBM speed.  The tensor-memory kernel of the long segments (qg_gemm.cu)
// passes 13 weights per clock and SM from stage to stage whatever the row count; here mma.sync takes them directly.
//
// A CTA (eight consumer warps, a producer warp and one that prepares the rows; two CTAs per SM, so that the next kernel's
// first loads travel while this one ends) works on tiles of 128 weight rows (8-bit codes: 64) x 8 or 16 token rows.  The
// producer keeps a ring of stages (256 k: 16 KB of codes, 1 or 2 KB of scales, 4 KB per eight token rows) filled by TMA.
// The consumers are two sets of four warps; set 0 takes the even stages, set 1 the odd ones, a warp 32 (16) weight rows of
// each, so that with 4-bit codes a fragment of token rows read from shared memory serves two MMAs (with 16 rows per warp
// shared memory was the limit; 8-bit codes are twice the bytes per MMA).  The set with a tile's last stage adds the
// other's sums and writes the result.  In gate/up mode an MMA tile is eight gate rows and the eight up rows that belong
// to them: a thread ends up with both values of its outputs.
//   More tiles than CTAs fit: the grid has a block per tile, or per few tiles, and a CTA that is done with its block takes over
// one that has not been started (cluster launch control; dealt out beforehand, the tiles left an SM up to 16 % more than its
// share: nine tiles are too few to round).  The hardware keeps the count, nothing outlives the launch, so launches may
// overlap on the GPU in any way.
//   One matrix with fewer tiles: K is cut into slices, the slices of a tile are a thread-block cluster, and each of its CTAs sends its
// sums to the one that adds them, in slice order.  All sums have a fixed order: results are reproducible.
//
// Arithmetic.  A weight costs as few instructions as possible: a nibble becomes the bf16 number 128 + code by a byte
// permute (0x43 above the code), in the order in which byte operations deliver them, and half a packed subtraction makes
// it the integer code - 8.  The tenth warp brings the segment rows of a stage into the same order once for all consumers
// (two permutes per eight weights otherwise).  The products are integers times bf16, exact in fp32; a 32-block's result is
// multiplied by its scale in fp32 and added to the running sum.  The scaled weight is never rounded, which is closer to
// the exact sum than a product of rounded weights (2.9e-3 against 4.0e-3 relative error of a layer).  (Starting the MMAs
// from -136 times the rows' block sums saves the subtractions but turns an infinity into a NaN, and gained 3 % at eight
// rows and lost 6 % at sixteen.)
//
// 8-bit codes: the low seven bits above 0x43 are the bf16 number 128 + bits, the sign bit above 0x43 is 128 or 256, and the
// difference is the code (42 instructions per 512 weights and eight rows, against 68 slots of the permute, packed fma and
// round chain that produces scaled weights).
//
// Range.  A 32-block's unscaled sum is up to 2^12 (4-bit codes: 2^8) times its largest token value: from 2^116 (2^120) on it may
// leave fp32 although the scaled sum would not.  Such a sum ends as an infinity or a NaN whatever is added, and so does the
// output; a warp that has stored one computes its outputs that are not finite again, from weights scaled beforehand, unless their
// token row is not finite itself (ms_again).  (Looking for huge values where the rows are prepared, and shrinking them by a
// power of two, costs every stage something: 128 tokens, 128 experts 144 us against 127.  As a called function, with a stack frame,
// the repair costs short launches 0.6 us: inlined, 1 % over 1086 shapes.)
//
// Measured, 128 experts x (1536 x 2048 gate/up, 2048 x 768 down), against the tensor-memory kernel: 1 token of eight
// experts 13.3 / 9.1 us against 16 / 12, 4 tokens 22 / 13 against 33 / 21, 32 tokens 48 / 30 (3.9 / 3.2 TB/s of codes and
// scales) against 85 / 49, 128 tokens 64 / 39 against 101 / 56, 256 tokens 91 / 54 against 102 / 57.
// One matrix (rotating copies larger than L2), 1 / 16 tokens, against a ring kernel with one CTA of 20 warps per SM that
// rounded scaled 8-bit weights, a block kernel and the tensor-memory kernel, whichever was fastest: 28672 x 4096 8 bit
// 32.3 / 38.2 us (3.9 / 3.3 TB/s) against 34.3 / 39.5; 4096 x 14336 16.4 / 19.8 against 19.0 / 28.7; 4096 x 4096 8.0 / 9.6
// against 8.6 / 13.2; 2048 x 2048 5.6 / 6.6 against 5.9 / 7.0; 3072 x 8192 4 bit 9.0 / 12.1 against 15.4 / 26.3.
// K slices send their sums to the CTA that adds them (st.async); while they met, read each other's and met again, 1 / 16 tokens back
// to back in a graph: 2048 x 2048 8 bit 4.8 / 5.9 us, now 4.35 / 4.95; 3072 x 8192 4 bit 8.7 / 10.75, now 7.7 / 9.8; 5120 x 3072
// 6.7 / 8.3, now 6.1 / 7.3.
// What bounds it: without its arithmetic the 28672 x 4096 launch takes 26.4 us, with the codes' loads alone 22.1 (5.65 TB/s);
// supply and arithmetic overlap, but with 16 consumer warps per SM neither hides the other fully.
// Every mbarrier wait is bounded.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "qg_internal.h"
#include "qg_ptx.cuh"
#include "qg_dequant.cuh"
#include "qg_mma.cuh"

namespace qg {

constexpr int MS_SK = 256;                            // k per stage
constexpr int MS_W_BYTES = 16384;                     // codes per stage: 128 rows of 4-bit codes, 64 rows of 8-bit codes
__host__ __device__ constexpr int ms_rows(int qbits) { return qbits == 4 ? 128 : 64; }        // weight rows per tile
__host__ __device__ constexpr int ms_s_bytes(int qbits) { return ms_rows(qbits) * 16; }       // eight scales per row
constexpr int MS_X_BYTES = 8 * MS_SK * 2;             // eight token rows
// Room for the fragments that a CTA adds, of all slices: each slice sends a share of 4 x 32 fragments of 16 bytes per MMA tile.
__host__ __device__ constexpr int ms_recv_bytes(int mma_tiles) { return (4 * 32 * mma_tiles + 8 * 7) * 16; }
constexpr int MS_CONS_WARPS = 8, MS_THREADS = 32 * (MS_CONS_WARPS + 2);
constexpr int MS_NT = 2;                              // most groups of eight segment rows per tile
constexpr int MS_MAX_ST = 6;
// Most blocks of a launch, per SM: above that many tiles a block has several.  A CTA that runs out of tiles takes the blocks
// beyond the last tile one by one, 0.33 us each, and with a block per tile there may be 50 for each of them (all rows with one
// of 256 experts: 75 us against 60).  Fewer blocks are dealt out less evenly (8 per SM: 1946 us against 1506 for 17000 tiles).
constexpr int MS_BLOCKS_PER_SM = 64;
constexpr size_t MS_SMEM_MAX = 115712;                // half of an SM's shared memory: two CTAs per SM

struct StreamParams {
    int R, N, K, E;
    int n_wt;                   // weight tiles per expert (gate/up mode: 64 gate + 64 up rows each)
    int n_stages, stage_bytes;
    int kc;                     // k per CTA: K, or a slice of it when the CTAs of a cluster share a tile
    int dynamic;                // more blocks than fit at once: a CTA goes on with the tiles of blocks not yet started
    GroupedChoice choice;       // grouped: whether this launch has the work or the one behind it
    const int32_t* offsets;     // grouped: device expert offsets [E + 1]
    __nv_bfloat16* out;
    const __nv_bfloat16* x;     // token rows, codes and scales once more, for ms_again
    const uint8_t* wq;
    const __half* ws;
    const float* topk_w;        // grouped: routing weights, applied to the rows named by row_pair (nullptr: none)
    const int32_t* row_pair;
    int gather_k;               // gathered: row r of the input is token row_pair[r] / gather_k
    int* status;
    uint32_t wait_limit;
    int skip_stage;             // test hook: stage of the first CTA whose token rows are never loaded (-1: none)
};

template <bool CLUSTER = false>         // other CTAs' stores are read after the wait
__device__ __forceinline__ bool ms_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, const StreamParams& p) {
    if (CLUSTER ? mbar_test_wait_cluster(bar, parity) : mbar_test_wait(bar, parity)) return true;
    for (uint32_t it = 0; it < p.wait_limit; ++it) {
        if (CLUSTER ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 255u && *abort_flag) return false;
    }
    *abort_flag = 1;
    atomicCAS(p.status, 0, QG_ERR_TIMEOUT);
    return false;
}

struct __align__(16) StreamTile {
    int e, wt, tok0, n;         // expert, weight tile, first row and rows (0: no more tiles)
};

// One stage (eight 32-blocks): this warp's MMA tiles of 16 weight rows (g and the row HI further; 4-bit codes: a second tile
// STEP rows on) x 8 NT token rows.  wl: this lane's code word of block 0 in its lowest row; x: its fragments of the token
// rows; sc: the scales of its lowest row.
template <int QBITS, int NT, int HI, int STEP, int NTM, int MT>
__device__ __forceinline__ void ms_stage(float (&acc)[NTM][MT][4], uint32_t wl, uint32_t x, uint32_t sc) {
#pragma unroll
    for (int b2 = 0; b2 < 4; ++b2) {               // two 32-blocks share a word of scales
        uint32_t s_lo[MT], s_hi[MT];
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            s_lo[m] = lds_u1(sc + b2 * 4 + m * STEP * 16);
            s_hi[m] = lds_u1(sc + b2 * 4 + (m * STEP + HI) * 16);
        }
#pragma unroll
        for (int bb = 0; bb < 2; ++bb) {
            const int b = 2 * b2 + bb;
            uint32_t pl[MT][4], ph[MT][4];
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                if constexpr (QBITS == 4) {
                    const uint32_t a = (wl ^ (b << 4)) + m * STEP * 128;
                    q4_spread(lds_u1(a), pl[m]);
                    q4_spread(lds_u1(a + HI * 128), ph[m]);
                } else {                           // the lane's words of the block's two 16-byte chunks
                    const uint32_t a = (wl ^ ((b & 3) << 5)) + (b >> 2) * (MS_W_BYTES / 2), a2 = a ^ 16;
                    q8_spread(lds_u1(a), pl[m][0], pl[m][1]);
                    q8_spread(lds_u1(a2), pl[m][2], pl[m][3]);
                    q8_spread(lds_u1(a + HI * 128), ph[m][0], ph[m][1]);
                    q8_spread(lds_u1(a2 + HI * 128), ph[m][2], ph[m][3]);
                }
            }
            float fl[MT], fh[MT];
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const float2 l2 = __half22float2(*reinterpret_cast<const __half2*>(&s_lo[m]));
                const float2 h2 = __half22float2(*reinterpret_cast<const __half2*>(&s_hi[m]));
                fl[m] = bb ? l2.y : l2.x;
                fh[m] = bb ? h2.y : h2.x;
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const uint4 xv = lds_u4(x + nt * MS_X_BYTES + b * 512);
                float t[MT][4];
#pragma unroll
                for (int m = 0; m < MT; ++m) mma_w16_first(t[m], pl[m][0], ph[m][0], pl[m][1], ph[m][1], xv.x, xv.y);
#pragma unroll
                for (int m = 0; m < MT; ++m) mma_w16(t[m], pl[m][2], ph[m][2], pl[m][3], ph[m][3], xv.z, xv.w);
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    acc[nt][m][0] = fmaf(fl[m], t[m][0], acc[nt][m][0]);
                    acc[nt][m][1] = fmaf(fl[m], t[m][1], acc[nt][m][1]);
                    acc[nt][m][2] = fmaf(fh[m], t[m][2], acc[nt][m][2]);
                    acc[nt][m][3] = fmaf(fh[m], t[m][3], acc[nt][m][3]);
                }
            }
        }
    }
}

__device__ __forceinline__ float silu_mul(float g, float u) { return __fdividef(g, 1.0f + __expf(-g)) * u; }

// Token row x times weight row `row` (over all experts), each weight scaled before it is multiplied, in the order of k.
template <int QBITS>
__device__ __forceinline__ float ms_dot(const StreamParams& p, const __nv_bfloat16* x, long long row) {
    const uint8_t* q = p.wq + row * (static_cast<long long>(p.K) * QBITS / 8);
    const __half* s = p.ws + row * (p.K >> 5);
    float acc = 0.f;
#pragma unroll 1
    for (int k = 0; k < p.K; k += 2) {
        const float sc = __half2float(s[k >> 5]);
        int q0, q1;
        if constexpr (QBITS == 8) {
            q0 = static_cast<int8_t>(q[k]); q1 = static_cast<int8_t>(q[k + 1]);
        } else {
            q0 = (q[k >> 1] & 15) - 8; q1 = (q[k >> 1] >> 4) - 8;
        }
        acc = fmaf(__bfloat162float(x[k]), q0 * sc, acc);
        acc = fmaf(__bfloat162float(x[k + 1]), q1 * sc, acc);
    }
    return acc;
}
__device__ __forceinline__ bool ms_finite(__nv_bfloat16 v) { return (__bfloat16_as_ushort(v) & 0x7F80) != 0x7F80; }
// The outputs of token row `tok` in columns c and c + 8 (gate/up: column c only) again, where they are not finite.
template <int QBITS, bool GATE_UP, bool GATHER>
__device__ __forceinline__ void ms_again(const StreamParams& p, int e, int tok, int c) {
    const __nv_bfloat16* x = p.x + static_cast<size_t>(GATHER ? p.row_pair[tok] / p.gather_k : tok) * p.K;
    const int width = GATE_UP ? p.N >> 1 : p.N;
    __nv_bfloat16* o = p.out + static_cast<size_t>(tok) * width;
    bool scanned = false;
#pragma unroll 1
    for (int h = 0; h < (GATE_UP ? 1 : 2); ++h, c += 8) {
        if (c >= width || ms_finite(o[c])) continue;
#pragma unroll 1
        for (int k = 0; !scanned && k < p.K; ++k)
            if (!ms_finite(x[k])) return;             // what the products gave stands
        scanned = true;
        const long long row = static_cast<long long>(e) * p.N + c;
        float v = ms_dot<QBITS>(p, x, row);
        if (GATE_UP) v = silu_mul(v, ms_dot<QBITS>(p, x, row + width));
        else if (p.topk_w) v *= p.topk_w[p.row_pair[tok]];
        o[c] = __float2bfloat16_rn(v);
    }
}
// 0, or NaN if one of the four is an infinity or a NaN
__device__ __forceinline__ float zero_if_finite(float z, float a, float b, float c, float d) {
    return fmaf(a, 0.f, fmaf(b, 0.f, fmaf(c, 0.f, fmaf(d, 0.f, z))));
}

// tm_w: packed codes, box 128 bytes x the tile's rows (gate/up: 64 rows x 2 planes), 128-byte swizzle; tm_s: scales, box 8 x
// the same rows; tm_x: token rows as [K / 32][R][32], box 32 k x 8 rows x 8 blocks, so that the 16 bytes a lane of an MMA
// fragment needs follow one another in lane order.  Rows past the end arrive as zeros.  Gathered rows: [M][K], box 256 k x one
// row, four rows per copy, which land row after row.
// grid = (tiles, K slices); the slices of a tile are one cluster.
template <int QBITS, bool GROUPED, bool GATE_UP, int NTM, bool GATHER, bool SLICED = false>
__global__ void __launch_bounds__(MS_THREADS, 2)
stream_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_s,
              const __grid_constant__ CUtensorMap tm_x, const StreamParams p) {
    constexpr int ROWS = ms_rows(QBITS), MT = ROWS / 64, TN = 8 * NTM;
    constexpr int OFF_S = MS_W_BYTES, OFF_X = MS_W_BYTES + ms_s_bytes(QBITS);
    extern __shared__ uint8_t ms_smem[];
    const uint32_t ring = (smem_u32(ms_smem) + 1023u) & ~1023u;
    uint8_t* after = ms_smem + (ring - smem_u32(ms_smem)) + p.n_stages * p.stage_bytes;
    const uint32_t xch = smem_u32(after);              // [4 warps][NTM][MT][32 lanes] float4: sums handed from set to set
    after += 4 * NTM * MT * 512;
    const uint32_t recv = smem_u32(after);             // K slices: [slices][fragments this CTA adds] float4, written by the cluster's CTAs
    if (SLICED) after += ms_recv_bytes(NTM * MT);
    // full: stage i's barrier is number i mod 2 n_stages (twice the slots), so that one set waits on it every time it is used:
    // with one barrier per slot and an odd number of slots a set would see every other phase only, and a wait by parity
    // passes too early while the phase in between is not complete.
    const uint32_t full0 = smem_u32(after), empty0 = full0 + 16u * MS_MAX_ST, xfull0 = empty0 + 8u * MS_MAX_ST;
    const uint32_t hfull0 = xfull0 + 8u * MS_MAX_ST, hempty0 = hfull0 + 32u;      // the hand-over of each pair of warps
    after += 32 * MS_MAX_ST + 64;
    const uint32_t taken = smem_u32(after), taken_bar = taken + 16;      // the hardware's answer to a request for a tile
    const uint32_t recv_bar = taken + 24;              // the fragments of all slices are there
    after += 32;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(after);
    volatile StreamTile* tiles = reinterpret_cast<volatile StreamTile*>(after + 16);   // per stage: the tile it belongs to
    int* off = reinterpret_cast<int*>(after + 16 + 16 * MS_MAX_ST);      // grouped: [E + 1] segment offsets
    int* prefix = off + p.E + 1;                                         // grouped: [E + 1] tiles before an expert
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (!GROUPED || !p.choice.on) pdl_launch_dependents();
    if (warp == 0) {
        if (lane < 2 * p.n_stages) mbar_init(full0 + 8u * lane, 2);
        if (lane < p.n_stages) { mbar_init(empty0 + 8u * lane, MS_CONS_WARPS / 2); mbar_init(xfull0 + 8u * lane, 1); }
        if (lane >= 16 && lane < 24) mbar_init(hfull0 + 8u * (lane - 16), 1);
        if (lane == 31) { *abort_flag = 0; mbar_init(taken_bar, 1); mbar_init(recv_bar, 1); }
        fence_mbar_init();
        fence_proxy_async_smem();
    }
    if (threadIdx.x == 256) { prefetch_tmap(&tm_w); prefetch_tmap(&tm_s); prefetch_tmap(&tm_x); }
    int total = p.n_wt;
    if constexpr (GROUPED) {
        pdl_wait();
        if (p.choice.on) pdl_launch_dependents();      // the kernel behind this one reads the offsets as soon as it runs
        for (int e = threadIdx.x; e <= p.E; e += MS_THREADS) off[e] = p.offsets[e];
        __syncthreads();
        if (warp == 0) {
            int carry = 0, wide = 0;
            for (int e0 = 0; e0 < p.E; e0 += 32) {
                const int e = e0 + lane;
                const int n = (e < p.E) ? (off[e + 1] - off[e] + TN - 1) / TN * p.n_wt : 0;
                wide += (e < p.E) ? (off[e + 1] - off[e] + 127) >> 7 : 0;
                int inc = n;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int v = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                    if (lane >= d) inc += v;
                }
                if (e < p.E) prefix[e] = carry + inc - n;
                carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
            }
            if (p.choice.on && !p.choice.streams(carry / p.n_wt, __reduce_add_sync(0xFFFFFFFFu, wide))) carry = 0;     // nothing to do
            if (lane == 0) prefix[p.E] = carry;
        }
        __syncthreads();
        total = prefix[p.E];
    } else {
        __syncthreads();
        if (warp != MS_CONS_WARPS) pdl_wait();         // the weights are constants of the model: their producer starts at once
    }
    const int k0 = static_cast<int>(blockIdx.y) * p.kc;
    const int nst = min(p.kc, p.K - k0) / MS_SK;       // stages of a tile
    // K slices (SLICED: p.kc < p.K, and a CTA has one tile): the CTAs of a cluster hold one slice's sums of the same tile each.  Every
    // CTA adds a share of the tile's fragments (16 bytes: rows lo / hi x two tokens): the others send theirs to its shared memory, and
    // a barrier there counts the bytes.
    const uint32_t n_frag = 4 * MT * 32 * ((p.R + 7) >> 3), share = (n_frag + gridDim.y - 1) / gridDim.y, rank = blockIdx.y;
    const uint32_t my_frags = rank * share < n_frag ? min(share, n_frag - rank * share) : 0;
    if constexpr (SLICED) {
        if (threadIdx.x == 0) mbar_arrive_expect_tx(recv_bar, my_frags * gridDim.y * 16);
        __syncwarp();
        cluster_arrive();
        if (warp < MS_CONS_WARPS) cluster_wait();      // the others' barriers are set up
    }

    if (warp == MS_CONS_WARPS) {
        // ------------------------------------------------ producer
        if (elect_one()) {
            uint32_t slot = 0, phase = 0, fslot = 0;
            int sent = 0, ahead = 0;                   // stages filled, stages whose weights are on their way
            uint32_t asked = 0;                        // answers to requests for a block so far, each a phase of taken_bar
            bool more = p.dynamic, waiting = false;    // there may be blocks that have not been started; a request is on its way
            const int skip = (blockIdx.x == 0 && blockIdx.y == 0) ? p.skip_stage : -1;
            bool ok = true;
            auto load_weights = [&](uint32_t at, uint32_t bar, int st, const StreamTile& tl) {
                const uint32_t dst = ring + at * p.stage_bytes;
                mbar_arrive_expect_tx(bar, MS_W_BYTES + ms_s_bytes(QBITS));
                if constexpr (GATE_UP) {
                    tma_load_3d(dst, &tm_w, st * 128, tl.wt * 64, 2 * tl.e, bar);
                    tma_load_3d(dst + OFF_S, &tm_s, st * 8, tl.wt * 64, 2 * tl.e, bar);
                } else {
                    const int row = tl.e * p.N + tl.wt * ROWS, ks = k0 / MS_SK + st;
                    if (QBITS == 8) tma_load_3d(dst, &tm_w, 0, row, 2 * ks, bar);
                    else tma_load_2d(dst, &tm_w, ks * 128, row, bar);
                    tma_load_2d(dst + OFF_S, &tm_s, ks * 8, row, bar);
                }
            };
            if (!GROUPED) {
                const StreamTile tl{0, static_cast<int>(blockIdx.x), 0, p.R};
                for (; ahead < min(nst, p.n_stages); ++ahead) load_weights(ahead, full0 + 8u * ahead, ahead, tl);
                pdl_wait();
            }
            for (int t = blockIdx.x; ok; ) {
                if (more && !waiting) {                // asked for early, used at the end of this block's tiles
                    mbar_arrive_expect_tx(taken_bar, 16);
                    clc_try_cancel(taken, taken_bar);
                    waiting = true;
                }
                if (more && t >= total) {              // (blocks past the last tile are taken as well: started, they would cost more)
                    uint32_t block = 0;
                    ok = ms_wait(taken_bar, asked & 1u, abort_flag, p);
                    ++asked;
                    waiting = false;
                    more = ok && clc_block(taken, block);
                    if (more) t = static_cast<int>(block);
                    continue;
                }
                StreamTile tl{0, 0, 0, 0};
                if (t < total) {
                    if constexpr (GROUPED) {
                        int lo = 0, hi = p.E - 1;            // the last expert whose tiles start at or before t
                        while (lo < hi) {
                            const int mid = (lo + hi + 1) >> 1;
                            if (prefix[mid] <= t) lo = mid; else hi = mid - 1;
                        }
                        // chunks of the segment fastest: the second chunk finds its weights in L2
                        const int n_ch = (off[lo + 1] - off[lo] + TN - 1) / TN, local = t - prefix[lo];
                        tl.e = lo;
                        tl.wt = local / n_ch;
                        tl.tok0 = off[lo] + (local - tl.wt * n_ch) * TN;
                        tl.n = min(TN, off[lo + 1] - tl.tok0);
                    } else {
                        tl.wt = t;
                        tl.n = p.R;
                    }
                }
                const int nt = (tl.n + 7) >> 3;
                int rows[TN];                          // gathered: the tile's token rows (past its end the first one: computed, never stored)
                if (GATHER && tl.n > 0) {
#pragma unroll
                    for (int i = 0; i < TN; ++i) rows[i] = p.row_pair[tl.tok0 + (i < tl.n ? i : 0)];
#pragma unroll
                    for (int i = 0; i < TN; ++i) rows[i] /= p.gather_k;
                }
                for (int st = 0; st < (tl.n ? nst : 2); ++st, ++sent) {     // no more tiles: two empty stages, one for each set, say so
                    if (sent >= p.n_stages && !ms_wait(empty0 + 8u * slot, phase ^ 1u, abort_flag, p)) { ok = false; break; }
                    const uint32_t xbar = xfull0 + 8u * slot;
                    volatile StreamTile* d = tiles + slot;
                    d->e = tl.e; d->wt = tl.wt; d->tok0 = tl.tok0; d->n = tl.n;
                    if (tl.n == 0) {
                        mbar_arrive(xbar);
                        mbar_arrive(full0 + 8u * fslot);
                    } else {
                        mbar_arrive_expect_tx(xbar, nt * MS_X_BYTES);
                        if (sent == skip) {
                        } else if (GATHER) {
#pragma unroll
                            for (int i = 0; i < TN; i += 4)
                                if (i < 8 * nt)
                                    tma_gather4(ring + slot * p.stage_bytes + OFF_X + i * 512, &tm_x, st * MS_SK, rows[i], rows[i + 1], rows[i + 2],
                                                rows[i + 3], xbar);
                        } else
                            for (int i = 0; i < nt; ++i)
                                tma_load_3d(ring + slot * p.stage_bytes + OFF_X + i * MS_X_BYTES, &tm_x, 0, tl.tok0 + 8 * i, k0 / 32 + st * 8, xbar);
                        if (sent >= ahead) load_weights(slot, full0 + 8u * fslot, st, tl);
                    }
                    if (++slot == static_cast<uint32_t>(p.n_stages)) { slot = 0; phase ^= 1u; }
                    if (++fslot == 2u * p.n_stages) fslot = 0;
                }
                if (tl.n == 0) break;
                t += gridDim.x;
            }
        }
    } else if (warp == MS_CONS_WARPS + 1) {
        // ------------------------------------------------ token rows: every 32-block into the order of q4_spread (a lane's eight
        // k as 0, 2, 4, 6, 1, 3, 5, 7) or q8_spread (four k of each half of the block, each as 0, 2, 1, 3), in place
        uint32_t slot = 0, phase = 0, fslot = 0;
        int ends = 0;
        const int g = lane >> 2, j = lane & 3;
        while (ends < 2 && __all_sync(0xFFFFFFFFu, ms_wait(xfull0 + 8u * slot, phase, abort_flag, p))) {
            const int nt = (tiles[slot].n + 7) >> 3;
            ends += (nt == 0);
            const uint32_t x = ring + slot * p.stage_bytes + OFF_X;
            for (int i = 0; i < nt; ++i) {
                const uint32_t xi = x + i * MS_X_BYTES;
                uint4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if constexpr (QBITS == 4) {
                        const uint4 r = lds_u4(GATHER ? xi + g * 512 + u * 64 + j * 16 : xi + u * 512 + lane * 16);
                        v[u] = make_uint4(__byte_perm(r.x, r.y, 0x5410), __byte_perm(r.z, r.w, 0x5410),
                                          __byte_perm(r.x, r.y, 0x7632), __byte_perm(r.z, r.w, 0x7632));
                    } else {
                        const uint2 a = lds_u2(xi + u * 512 + g * 64 + j * 8), c = lds_u2(xi + u * 512 + g * 64 + 32 + j * 8);
                        v[u] = make_uint4(__byte_perm(a.x, a.y, 0x5410), __byte_perm(a.x, a.y, 0x7632),
                                          __byte_perm(c.x, c.y, 0x5410), __byte_perm(c.x, c.y, 0x7632));
                    }
                }
                if (QBITS == 8 || GATHER) __syncwarp();      // everything is read before anything is written
#pragma unroll
                for (int u = 0; u < 8; ++u) sts_u4(xi + u * 512 + lane * 16, v[u]);
            }
            fence_proxy_async_smem();              // the slot's next load comes after these writes
            __syncwarp();
            if (lane == 0) mbar_arrive(full0 + 8u * fslot);
            if (++slot == static_cast<uint32_t>(p.n_stages)) { slot = 0; phase ^= 1u; }
            if (++fslot == 2u * p.n_stages) fslot = 0;
        }
    } else {
        // ------------------------------------------------ consumers: two sets of four warps, set 0 takes the even stages and
        // set 1 the odd ones, a warp 16 MT weight rows of each
        constexpr int HI = GATE_UP ? 64 : 8, STEP = GATE_UP ? 8 : 16;     // distance of a tile's two halves, and of the two tiles
        const int set = warp >> 2, w4 = warp & 3;
        const int g = lane >> 2, j = lane & 3;
        const uint32_t row = (GATE_UP ? 16 : 16 * MT) * w4 + g;
        const uint32_t wl0 = ring + row * 128 + (g << 4) + 4 * j;         // 16-byte chunk c of the row lies at c ^ g
        const uint32_t sc0 = ring + OFF_S + row * 16;
        const uint32_t x0 = ring + OFF_X + lane * 16;
        const uint32_t my_xch = xch + (w4 * NTM * MT * 32 + lane) * 16, hfull = hfull0 + 8u * w4, hempty = hempty0 + 8u * w4;
        uint32_t slot = set, fslot = set, fphase = 0;
        float wl = 0.f;                       // routing weight of row `lane` of the chunk
        int have = -1;                        // first row of the chunk wl belongs to
        for (uint32_t q = 0, base = 0; ; ++q, base += nst) {              // tile and its first stage, both counted from 0
            const uint32_t first = base + ((base ^ set) & 1u);            // this set's first stage of the tile
            if (first >= base + nst) {                                    // a tile of one stage: every other one is the other set's
                if (SLICED) break;
                continue;
            }
            if (!__all_sync(0xFFFFFFFFu, ms_wait(full0 + 8u * fslot, fphase, abort_flag, p))) break;
            const int wt = tiles[slot].wt, tok0 = tiles[slot].tok0, n = tiles[slot].n;
            if (n == 0) break;
            const int nt_n = (n + 7) >> 3;
            const bool mine = ((base + nst - 1 - set) & 1u) == 0;         // the set with the last stage finishes the tile
            if (GROUPED && mine && p.topk_w && have != tok0) {
                wl = (lane < n) ? p.topk_w[p.row_pair[tok0 + lane]] : 0.f;
                have = tok0;
            }
            float acc[NTM][MT][4];
#pragma unroll
            for (int nt = 0; nt < NTM; ++nt)
#pragma unroll
                for (int e = 0; e < 4 * MT; ++e) acc[nt][e >> 2][e & 3] = 0.f;
            bool ok = true;
            for (uint32_t st = first; st < base + nst; st += 2) {
                ok = __all_sync(0xFFFFFFFFu, ms_wait(full0 + 8u * fslot, fphase, abort_flag, p));
                if (!ok) break;
                const uint32_t o = slot * p.stage_bytes;
                if (NTM == 1 || nt_n == 1) ms_stage<QBITS, 1, HI, STEP>(acc, wl0 + o, x0 + o, sc0 + o);
                else ms_stage<QBITS, NTM, HI, STEP>(acc, wl0 + o, x0 + o, sc0 + o);
                __syncwarp();
                if (lane == 0) mbar_arrive(empty0 + 8u * slot);
                slot += 2;
                if (slot >= static_cast<uint32_t>(p.n_stages)) slot -= p.n_stages;
                fslot += 2;
                if (fslot >= 2u * p.n_stages) { fslot -= 2u * p.n_stages; fphase ^= 1u; }
            }
            if (!ok) break;
            if (nst > 1 && !mine) {           // hand the sums to the other set's warp of the same rows
                if (q > 0 && !__all_sync(0xFFFFFFFFu, ms_wait(hempty, (q & 1u) ^ 1u, abort_flag, p))) break;
#pragma unroll
                for (int nt = 0; nt < NTM; ++nt)
#pragma unroll
                    for (int m = 0; m < MT; ++m)
                        if (nt < nt_n)
                            sts_u4(my_xch + (nt * MT + m) * 512, make_uint4(__float_as_uint(acc[nt][m][0]), __float_as_uint(acc[nt][m][1]),
                                                                            __float_as_uint(acc[nt][m][2]), __float_as_uint(acc[nt][m][3])));
                __syncwarp();
                if (lane == 0) mbar_arrive(hfull);
                continue;
            }
            if (nst > 1 && !__all_sync(0xFFFFFFFFu, ms_wait(hfull, q & 1u, abort_flag, p))) break;
            float z = 0.f;
#pragma unroll
            for (int nt = 0; nt < NTM; ++nt) {
                if (nt >= nt_n) break;
                const int t = 8 * nt + 2 * j;
                float w0 = 1.f, w1 = 1.f;
                if (GROUPED && !GATE_UP && p.topk_w) { w0 = __shfl_sync(0xFFFFFFFFu, wl, t); w1 = __shfl_sync(0xFFFFFFFFu, wl, t + 1); }
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    float c0 = acc[nt][m][0], c1 = acc[nt][m][1], c2 = acc[nt][m][2], c3 = acc[nt][m][3];   // rows lo / hi x token rows t, t + 1
                    const uint32_t at = my_xch + (nt * MT + m) * 512;
                    if (nst > 1) {
                        const uint4 v = lds_u4(at);
                        c0 += __uint_as_float(v.x); c1 += __uint_as_float(v.y); c2 += __uint_as_float(v.z); c3 += __uint_as_float(v.w);
                    }
                    if constexpr (SLICED) {   // this slice's sum: to the CTA that adds this fragment
                        const uint32_t i = ((nt * 4 + w4) * MT + m) * 32 + lane, to = i / share;
                        st_async_v4(map_to_cta(recv + (rank * share + i - to * share) * 16, to), c0, c1, c2, c3, map_to_cta(recv_bar, to));
                        continue;
                    }
                    z = zero_if_finite(z, c0, c1, c2, c3);
                    __nv_bfloat16* o = p.out;
                    if constexpr (GATE_UP) {
                        const int F = p.N >> 1;
                        o += static_cast<size_t>(tok0 + t) * F + wt * 64 + 16 * w4 + 8 * m + g;
                        if (t < n) o[0] = __float2bfloat16_rn(silu_mul(c0, c2));
                        if (t + 1 < n) o[F] = __float2bfloat16_rn(silu_mul(c1, c3));
                    } else {
                        if (GROUPED && p.topk_w) { c0 *= w0; c1 *= w1; c2 *= w0; c3 *= w1; }
                        const int r = wt * ROWS + 16 * (MT * w4 + m);        // N % 8 == 0: a half's eight rows are all inside or all outside
                        o += static_cast<size_t>(tok0 + t) * p.N + r + g;
                        if (t < n) {
                            if (r < p.N) o[0] = __float2bfloat16_rn(c0);
                            if (r + 8 < p.N) o[8] = __float2bfloat16_rn(c2);
                        }
                        if (t + 1 < n) {
                            if (r < p.N) o[p.N] = __float2bfloat16_rn(c1);
                            if (r + 8 < p.N) o[p.N + 8] = __float2bfloat16_rn(c3);
                        }
                    }
                }
            }
            if (SLICED) break;
            if (nst > 1) {
                __syncwarp();
                if (lane == 0) mbar_arrive(hempty);
            }
            if (z != 0.f) {                   // a NaN: one of this thread's sums is not finite
                int e = 0;
                if (GROUPED)
                    while (off[e + 1] <= tok0) ++e;
#pragma unroll 1
                for (int i = 0; i < 2 * MT * nt_n; ++i) {
                    const int t = 8 * (i / (2 * MT)) + 2 * j + (i & 1), m = (i >> 1) % MT;
                    if (t < n) ms_again<QBITS, GATE_UP, GATHER>(p, e, tok0 + t, GATE_UP ? wt * 64 + 16 * w4 + 8 * m + g : wt * ROWS + 16 * (MT * w4 + m) + g);
                }
            }
        }
    }
    if constexpr (SLICED) {
        // A fragment's slices are added in order, so results are reproducible.  Nobody leaves before everybody has sent, which this CTA
        // waits for anyway.  (Until all had met, read each other's sums and met again: 0.9 us of 5 to 9.)
        if (warp >= MS_CONS_WARPS) cluster_wait();
        cluster_arrive();
        if (threadIdx.x < my_frags && ms_wait<true>(recv_bar, 0u, abort_flag, p)) {
            const uint32_t i = rank * share + threadIdx.x;               // (((token group) 4 + warp) MT + MMA tile) 32 + lane
            const uint32_t l = i & 31u, m = (i >> 5) % MT, w4 = (i / (32u * MT)) & 3u, nt = i / (128u * MT);
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            for (uint32_t sl = 0; sl < gridDim.y; ++sl) {
                const uint4 v = lds_u4(recv + (sl * share + threadIdx.x) * 16);
                c[0] += __uint_as_float(v.x); c[1] += __uint_as_float(v.y); c[2] += __uint_as_float(v.z); c[3] += __uint_as_float(v.w);
            }
            const int t = 8 * nt + 2 * (l & 3), r = blockIdx.x * ROWS + 16 * (MT * w4 + m);
            __nv_bfloat16* o = p.out + static_cast<size_t>(t) * p.N + r + (l >> 2);
            if (t < p.R) {
                if (r < p.N) o[0] = __float2bfloat16_rn(c[0]);
                if (r + 8 < p.N) o[8] = __float2bfloat16_rn(c[2]);
            }
            if (t + 1 < p.R) {
                if (r < p.N) o[p.N] = __float2bfloat16_rn(c[1]);
                if (r + 8 < p.N) o[p.N + 8] = __float2bfloat16_rn(c[3]);
            }
            if (zero_if_finite(0.f, c[0], c[1], c[2], c[3]) != 0.f)
#pragma unroll 1
                for (int u = t; u < min(t + 2, p.R); ++u) ms_again<QBITS, false, false>(p, 0, u, r + (l >> 2));
        }
        cluster_wait();
    }
    __syncthreads();
    if (*abort_flag) {
        for (int i = 0; i < 64; ++i) __nanosleep(2000);       // copies still in flight land before the memory is released
    }
}

// Ring depth and shared memory of a launch; false if not even two stages fit.
static bool ms_layout(StreamParams& p, int qbits, int ntm, int n_exp, size_t& smem) {
    p.stage_bytes = (MS_W_BYTES + ms_s_bytes(qbits) + ntm * MS_X_BYTES + 1023) & ~1023;      // the codes' swizzle wants 1 KB
    const int mma_tiles = ntm * (ms_rows(qbits) / 64);
    const size_t fixed = 1024 + 4 * mma_tiles * 512 + (n_exp ? 0 : ms_recv_bytes(mma_tiles)) + 32 * MS_MAX_ST + 64 + 32 + 16 +
                         16 * MS_MAX_ST + (2 * static_cast<size_t>(n_exp) + 2) * sizeof(int);
    p.n_stages = static_cast<int>((MS_SMEM_MAX - fixed) / p.stage_bytes);
    if (p.n_stages > MS_MAX_ST) p.n_stages = MS_MAX_ST;
    smem = fixed + static_cast<size_t>(p.n_stages) * p.stage_bytes;
    return p.n_stages >= 2;
}
using StreamKernel = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const StreamParams);
static int ms_set_smem(qg_ctx* ctx, StreamKernel kern, int inst) {
    if (ctx->attr_set[inst]) return QG_OK;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(MS_SMEM_MAX)) != cudaSuccess) {
        cudaGetLastError();
        return QG_ERR_CUDA;
    }
    ctx->attr_set[inst] = true;
    return QG_OK;
}

// The grouped call, alone or (choice.on) with the other kernel behind it.  Returns QG_ERR_WORKSPACE if the shape does not suit
// this kernel (the caller takes the other one).
int launch_moe_stream(qg_ctx* ctx, int mode, int R, int E, int N, int K, const void* Ain, int in_rows, int gather_k, const int32_t* offsets,
                      const void* Wq, const void* Ws, const float* topk_w, const int32_t* row_pair, void* Out, GroupedChoice& choice, cudaStream_t st) {
    const bool gate_up = mode == QG_MODE_GATE_UP_SILU;
    StreamParams p{};
    p.R = R; p.N = N; p.K = K; p.E = E; p.kc = K;
    p.n_wt = gate_up ? N / 128 : (N + 127) / 128;
    // Rows per tile: eight up to five rows per expert, sixteen above.  The wider tile's ring is a stage shorter (56.1 us
    // against 53.0 at four rows per expert, gate/up); cutting a segment in two costs more from six on (60.4 with eight and
    // 61.4 with sixteen at six rows, 68.2 and 63.9 at eight, 79.4 and 68.1 at ten).  24 and 32 rows were slower throughout.
    const int ntm = (R <= 5LL * E) ? 1 : MS_NT;
    size_t smem = 0;
    if (!ms_layout(p, 4, ntm, E, smem)) return QG_ERR_WORKSPACE;
    // at most one chunk per 8 ntm rows and one more per expert that has rows
    const long long max_tiles = static_cast<long long>(R / (8 * ntm) + (R < E ? R : E)) * p.n_wt;
    if (max_tiles > 0x3FFFFFFF) return QG_ERR_WORKSPACE;
    p.choice.chunk = 8 * ntm; p.choice.n_wt = p.n_wt; p.choice.stages = K / MS_SK; p.choice.sm_count = ctx->sm_count;
    const int way = p.choice.plan(R, E);
    if (way == GroupedChoice::OTHER) return QG_ERR_WORKSPACE;
    p.choice.on = way == GroupedChoice::BOTH;
    choice = p.choice;
    p.offsets = offsets; p.out = static_cast<__nv_bfloat16*>(Out);
    p.x = static_cast<const __nv_bfloat16*>(Ain); p.wq = static_cast<const uint8_t*>(Wq); p.ws = static_cast<const __half*>(Ws);
    p.topk_w = (mode == QG_MODE_DOWN_WEIGHTED) ? topk_w : nullptr; p.row_pair = row_pair;
    p.gather_k = gather_k;
    p.status = ctx->d_status; p.wait_limit = ctx->wait_limit;
    p.skip_stage = ctx->skip_kb < 0 ? -1 : ctx->skip_kb / (MS_SK / 64);
    CUtensorMap tm_w, tm_s, tm_x;
    const uint64_t kb = K / 2, ks = K / 32, wrows = static_cast<uint64_t>(E) * N;
    int rc = gate_up ? get_tmap_3d(ctx, &tm_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, kb, N / 2, 2ull * E, kb * (N / 2), 128, 64, 2,
                                   CU_TENSOR_MAP_SWIZZLE_128B)
                     : get_tmap_2d(ctx, &tm_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, kb, wrows, 128, 128, CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc == QG_OK)
        rc = gate_up ? get_tmap_3d(ctx, &tm_s, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, Ws, ks, N / 2, 2ull * E, ks * 2 * (N / 2), 8, 64, 2,
                                   CU_TENSOR_MAP_SWIZZLE_NONE)
                     : get_tmap_2d(ctx, &tm_s, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, Ws, ks, wrows, 8, 128, CU_TENSOR_MAP_SWIZZLE_NONE);
    if (rc == QG_OK)
        rc = gather_k > 0 ? get_tmap_2d(ctx, &tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Ain, K, in_rows, MS_SK, 1, CU_TENSOR_MAP_SWIZZLE_NONE)
                          : get_tmap_3d(ctx, &tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Ain, 32, R, K / 32, 64, 32, 8, 8,
                                        CU_TENSOR_MAP_SWIZZLE_NONE, static_cast<uint64_t>(K) * 2);
    if (rc != QG_OK) return rc;
    const StreamKernel kerns[8] = {
        stream_kernel<4, true, false, 1, false>, stream_kernel<4, true, false, MS_NT, false>, stream_kernel<4, true, true, 1, false>,
        stream_kernel<4, true, true, MS_NT, false>, stream_kernel<4, true, false, 1, true>, stream_kernel<4, true, false, MS_NT, true>,
        stream_kernel<4, true, true, 1, true>, stream_kernel<4, true, true, MS_NT, true>};
    const int which = (gather_k > 0 ? 4 : 0) + (gate_up ? 2 : 0) + ntm - 1;
    const StreamKernel kern = kerns[which];
    rc = ms_set_smem(ctx, kern, ATTR_STREAM + which);
    if (rc != QG_OK) return rc;
    ctx->skip_kb = -1;                                        // the test hook acts on one launch
    const long long max_blocks = static_cast<long long>(MS_BLOCKS_PER_SM) * ctx->sm_count;
    const int grid = static_cast<int>(max_tiles < max_blocks ? max_tiles : max_blocks);
    p.dynamic = grid > 2 * ctx->sm_count;
    if (launch_kernel(ctx, kern, dim3(grid), dim3(MS_THREADS), smem, st, tm_w, tm_s, tm_x, p) != cudaSuccess) {
        cudaGetLastError();
        return QG_ERR_CUDA;
    }
    return QG_OK;
}

// The dense call for up to sixteen tokens.
int launch_dense_stream(qg_ctx* ctx, int qbits, int M, int N, int K, const void* A, const void* Wq, const void* Ws, void* Cout,
                        cudaStream_t st) {
    const int rows = ms_rows(qbits), ntm = (M > 8) ? 2 : 1, variant = (qbits == 8 ? 0 : 2) + ntm - 1;
    StreamParams p{};
    size_t smem = 0;
    if (!ms_layout(p, qbits, ntm, 0, smem)) return QG_ERR_WORKSPACE;
    const StreamKernel whole[4] = {stream_kernel<8, false, false, 1, false>, stream_kernel<8, false, false, 2, false>,
                                   stream_kernel<4, false, false, 1, false>, stream_kernel<4, false, false, 2, false>};
    const StreamKernel cut[4] = {stream_kernel<8, false, false, 1, false, true>, stream_kernel<8, false, false, 2, false, true>,
                                 stream_kernel<4, false, false, 1, false, true>, stream_kernel<4, false, false, 2, false, true>};
    int rc = ms_set_smem(ctx, whole[variant], ATTR_DENSE_STREAM + variant);
    if (rc == QG_OK) rc = ms_set_smem(ctx, cut[variant], ATTR_DENSE_STREAM + 4 + variant);
    if (rc != QG_OK) return rc;
    // clusters of `ns` CTAs of this kernel that fit on the GPU at once (asked once per context, variant and size)
    auto cluster_capacity = [&](int ns) {
        int& cached = ctx->gemv_max_clusters[variant][ns];
        if (cached == 0) {
            cudaLaunchConfig_t q = {};
            cudaLaunchAttribute ca;
            ca.id = cudaLaunchAttributeClusterDimension;
            ca.val.clusterDim.x = 1; ca.val.clusterDim.y = ns; ca.val.clusterDim.z = 1;
            q.gridDim = dim3(1, ns); q.blockDim = dim3(MS_THREADS); q.dynamicSmemBytes = smem; q.attrs = &ca; q.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, cut[variant], &q) != cudaSuccess) { cudaGetLastError(); n = 0; }
            cached = n > 0 ? n : -1;
        }
        return cached;
    };
    // K slices.  A CTA streams at its own pace as long as it has an SM to itself and at 0.8 of that with a second one beside
    // it, so more and shorter slices are faster until the sum over the cluster (about 60 k of a tile per slice) takes it
    // back.  4096 x 14336, 8 bit, one token: 36.8 / 24.7 / 19.1 / 16.4 us with one to four slices; 2048 x 2048: 6.6 / 6.3 /
    // 5.6 / 6.2 with one, two, four and eight; 3072 x 8192, 4 bit: 22.0 / 16.7 / 12.1 / 9.0.  Clusters of eight that fill the GPU
    // start late behind one another, and seven or six slices are faster then (32 tiles of 8 bit, K = 8192: 9.0 us with eight, 8.2
    // with seven; 4 bit, K = 4096: 7.8 with eight, 7.1 with six).  All clusters have to be resident at once.
    const int tiles = (N + rows - 1) / rows, blocks = K / MS_SK;
    int slices = 1, kc = K;
    long long best = -1;
    for (int ns = 1; ns <= 8 && ns <= blocks; ++ns) {
        const int per = (blocks + ns - 1) / ns;
        if ((blocks + per - 1) / per != ns) continue;          // the same cut as a smaller count
        if (ns > 1 && (ctx->gemv_mode & 1 || cluster_capacity(ns) < tiles)) continue;
        const long long alone = static_cast<long long>(per) * MS_SK;
        const long long ctas = static_cast<long long>(tiles) * ns;
        const int beside = ctas <= ctx->sm_count ? 100 : ns == 8 && 5 * ctas > 8 * ctx->sm_count ? 170 : 125;     // percent
        const long long cost = alone * beside / 100 + (ns > 1 ? 60 * ns : 0);
        if (best < 0 || cost < best) { best = cost; slices = ns; kc = per * MS_SK; }
    }
    p.R = M; p.N = N; p.K = K; p.E = 0; p.kc = kc; p.n_wt = tiles;
    p.out = static_cast<__nv_bfloat16*>(Cout);
    p.x = static_cast<const __nv_bfloat16*>(A); p.wq = static_cast<const uint8_t*>(Wq); p.ws = static_cast<const __half*>(Ws);
    p.status = ctx->d_status; p.wait_limit = ctx->wait_limit;
    p.skip_stage = ctx->skip_kb;
    CUtensorMap tm_w, tm_s, tm_x;
    // 8-bit codes as [K / 128][N][128]: both halves of a stage are one box (an instruction less per stage for the producer)
    rc = (qbits == 8) ? get_tmap_3d(ctx, &tm_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, 128, N, K / 128, 128, 128, rows, 2,
                                    CU_TENSOR_MAP_SWIZZLE_128B, static_cast<uint64_t>(K))
                      : get_tmap_2d(ctx, &tm_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, static_cast<uint64_t>(K) / 2, N, 128, rows,
                                    CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc == QG_OK) rc = get_tmap_2d(ctx, &tm_s, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, Ws, K / 32, N, 8, rows, CU_TENSOR_MAP_SWIZZLE_NONE);
    if (rc == QG_OK)
        rc = get_tmap_3d(ctx, &tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, A, 32, M, K / 32, 64, 32, 8, 8, CU_TENSOR_MAP_SWIZZLE_NONE,
                         static_cast<uint64_t>(K) * 2);
    if (rc != QG_OK) return rc;
    ctx->skip_kb = -1;
    p.dynamic = slices == 1 && tiles > 2 * ctx->sm_count;
    const int blocks_x = tiles < MS_BLOCKS_PER_SM * ctx->sm_count ? tiles : MS_BLOCKS_PER_SM * ctx->sm_count;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks_x, slices); cfg.blockDim = dim3(MS_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute at[2];
    int n_at = 0;
    if (ctx->pdl) {
        at[n_at].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n_at].val.programmaticStreamSerializationAllowed = 1;
        ++n_at;
    }
    if (slices > 1) {
        at[n_at].id = cudaLaunchAttributeClusterDimension;
        at[n_at].val.clusterDim.x = 1; at[n_at].val.clusterDim.y = slices; at[n_at].val.clusterDim.z = 1;
        ++n_at;
    }
    cfg.attrs = at; cfg.numAttrs = n_at;
    if (cudaLaunchKernelEx(&cfg, slices > 1 ? cut[variant] : whole[variant], tm_w, tm_s, tm_x, p) != cudaSuccess) {
        cudaGetLastError();
        if (slices == 1) return QG_ERR_CUDA;
        // the cluster launch was refused although the occupancy query allowed it: remember that and leave K whole
        ctx->gemv_max_clusters[variant][slices] = -1;
        return launch_dense_stream(ctx, qbits, M, N, K, A, Wq, Ws, Cout, st);
    }
    return QG_OK;
}

}  // namespace qg
