// Grouped 4-bit GEMM for short expert segments: the weight-streaming end of the expert projections.
//
// Operation: moe_grouped_qgemm's (plain, gate/up + SiLU, routing-weighted), for segments of a few rows.  There every
// weight byte is used for a handful of rows only, so the call is a streaming read of the experts' packed weights.  The
// tensor-memory kernel of the long segments (qg_gemm.cu) passes 13 weights per clock and SM from stage to stage whatever
// the row count, a third of what HBM delivers (42 4-bit weights per clock and SM); here mma.sync takes them directly.
//
// A CTA (eight consumer warps, a producer warp and one that prepares the rows; two CTAs per SM) takes tile after tile from
// a counter in global memory, a tile being 128 weight rows of one expert x 8 or 16 rows of its segment.  (Dealt out
// beforehand, the tiles left an SM up to 16 % more than its share: nine tiles are too few to round.)  The producer keeps a
// ring of stages (256 k: 16 KB of codes, 2 KB of scales, 4 KB per eight segment rows) filled by TMA.  The consumers are two
// sets of four warps; set 0 takes the even stages, set 1 the odd ones, a warp 32 weight rows of each, so that a fragment
// of segment rows read from shared memory serves two MMAs (with 16 rows per warp shared memory was the limit).  The set
// with a tile's last stage adds the other's sums and writes the result.  In gate/up mode an MMA tile is eight gate rows
// and the eight up rows that belong to them: a thread ends up with both values of its outputs.
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
// Measured, 128 experts x (1536 x 2048 gate/up, 2048 x 768 down), against the tensor-memory kernel: 1 token of eight
// experts 13.3 / 9.1 us against 16 / 12, 4 tokens 22 / 13 against 33 / 21, 32 tokens 48 / 30 (3.9 / 3.2 TB/s of codes and
// scales) against 85 / 49, 128 tokens 64 / 39 against 101 / 56, 256 tokens 91 / 54 against 102 / 57.  Without its
// arithmetic the 32-token gate/up launch takes 35 us: supply and arithmetic overlap, but neither hides the other fully.
// Every mbarrier wait is bounded.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "qg_internal.h"
#include "qg_ptx.cuh"
#include "qg_dequant.cuh"
#include "qg_mma.cuh"

namespace qg {

constexpr int MS_ROWS = 128;                          // weight rows per tile
constexpr int MS_SK = 256;                            // k per stage: 128 bytes of codes per row
constexpr int MS_W_BYTES = MS_ROWS * 128, MS_S_BYTES = MS_ROWS * 16;
constexpr int MS_X_BYTES = 8 * MS_SK * 2;             // eight segment rows
constexpr int MS_CONS_WARPS = 8, MS_THREADS = 32 * (MS_CONS_WARPS + 2);
constexpr int MS_NT = 2;                              // most groups of eight segment rows per tile
constexpr int MS_MAX_ST = 6;
// Rows per expert, on average, up to which this kernel is the faster one (both projections: 145 us against 158 at sixteen
// rows, 166 against 160 at twenty).
constexpr int MS_MAX_ROWS = 18;
constexpr size_t MS_SMEM_MAX = 115712;                // half of an SM's shared memory: two CTAs per SM

struct StreamParams {
    int R, N, K, E;
    int n_wt;                   // 128-row weight tiles per expert (64 gate + 64 up rows each in gate/up mode)
    int nt_max, n_stages, stage_bytes;
    int* sched;                 // [0] tiles taken beyond the first of each CTA, [1] CTAs that are done; zero between launches
    const int32_t* offsets;     // device expert offsets [E + 1]
    __nv_bfloat16* out;
    const float* topk_w;        // routing weights, applied to the rows named by row_pair (nullptr: none)
    const int32_t* row_pair;
    int* status;
    uint32_t wait_limit;
    int skip_kb;                // test hook: k-block (of 64) of the first tile whose activation load is left out (-1: none)
};

__device__ __forceinline__ bool ms_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, const StreamParams& p) {
    if (mbar_test_wait(bar, parity)) return true;
    for (uint32_t it = 0; it < p.wait_limit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 255u && *abort_flag) return false;
    }
    *abort_flag = 1;
    atomicCAS(p.status, 0, QG_ERR_TIMEOUT);
    return false;
}

struct __align__(16) StreamTile {
    int e, wt, tok0, n;         // expert, weight tile, first row and rows (0: no more tiles)
};

// One stage (eight 32-blocks): this warp's two MMA tiles of weight rows (g, the row HI further, and both STEP rows on) x
// 8 NT segment rows.  wl: this lane's code word of block 0 in its lowest row; x, xs: its fragments of the segment rows and of
// their sums; sc: the scales of its lowest row.
template <int NT, int HI, int STEP, int NTM>
__device__ __forceinline__ void ms_stage(float (&acc)[NTM][2][4], uint32_t wl, uint32_t x, uint32_t sc) {
#pragma unroll
    for (int b2 = 0; b2 < 4; ++b2) {               // two 32-blocks share a word of scales
        uint32_t s_lo[2], s_hi[2];
        s_lo[0] = lds_u1(sc + b2 * 4); s_hi[0] = lds_u1(sc + b2 * 4 + HI * 16);
        s_lo[1] = lds_u1(sc + b2 * 4 + STEP * 16); s_hi[1] = lds_u1(sc + b2 * 4 + (STEP + HI) * 16);
#pragma unroll
        for (int bb = 0; bb < 2; ++bb) {
            const int b = 2 * b2 + bb;
            uint32_t pl[2][4], ph[2][4];
            const uint32_t a = wl ^ (b << 4);
            q4_spread(lds_u1(a), pl[0]);
            q4_spread(lds_u1(a + HI * 128), ph[0]);
            q4_spread(lds_u1(a + STEP * 128), pl[1]);
            q4_spread(lds_u1(a + (STEP + HI) * 128), ph[1]);
            float fl[2], fh[2];
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const float2 l2 = __half22float2(*reinterpret_cast<const __half2*>(&s_lo[m]));
                const float2 h2 = __half22float2(*reinterpret_cast<const __half2*>(&s_hi[m]));
                fl[m] = bb ? l2.y : l2.x;
                fh[m] = bb ? h2.y : h2.x;
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const uint4 xv = lds_u4(x + nt * MS_X_BYTES + b * 512);
                float t[2][4];
#pragma unroll
                for (int m = 0; m < 2; ++m) mma_w16_first(t[m], pl[m][0], ph[m][0], pl[m][1], ph[m][1], xv.x, xv.y);
#pragma unroll
                for (int m = 0; m < 2; ++m) mma_w16(t[m], pl[m][2], ph[m][2], pl[m][3], ph[m][3], xv.z, xv.w);
#pragma unroll
                for (int m = 0; m < 2; ++m) {
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

// tm_w: packed codes, box 128 bytes x 128 rows (gate/up: 64 rows x 2 planes), 128-byte swizzle; tm_s: scales, box 8 x the
// same rows; tm_x: segment rows as [K / 32][R][32], box 32 k x 8 rows x 8 blocks, so that the 16 bytes a lane of an MMA
// fragment needs follow one another in lane order.  Rows past the end arrive as zeros.
template <bool GATE_UP, int NTM>
__global__ void __launch_bounds__(MS_THREADS, 2)
moe_stream_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_s,
                  const __grid_constant__ CUtensorMap tm_x, const StreamParams p) {
    extern __shared__ uint8_t ms_smem[];
    const uint32_t ring = (smem_u32(ms_smem) + 1023u) & ~1023u;
    uint8_t* after = ms_smem + (ring - smem_u32(ms_smem)) + p.n_stages * p.stage_bytes;
    const uint32_t xch = smem_u32(after);                                // [4 warps][NTM][2][32 lanes] float4: sums handed from set to set
    after += 4 * NTM * 2 * 512;
    const uint32_t full0 = smem_u32(after), empty0 = full0 + 8u * MS_MAX_ST, xfull0 = empty0 + 8u * MS_MAX_ST;
    const uint32_t hfull0 = xfull0 + 8u * MS_MAX_ST, hempty0 = hfull0 + 32u;      // the hand-over of each pair of warps
    after += 24 * MS_MAX_ST + 64;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(after);
    volatile StreamTile* tiles = reinterpret_cast<volatile StreamTile*>(after + 16);   // per stage: the tile it belongs to
    int* off = reinterpret_cast<int*>(after + 16 + 16 * MS_MAX_ST);      // [E + 1] segment offsets
    int* prefix = off + p.E + 1;                                         // [E + 1] tiles before an expert
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tn = 8 * p.nt_max;
    pdl_launch_dependents();
    if (warp == 0) {
        if (lane < p.n_stages) { mbar_init(full0 + 8u * lane, 2); mbar_init(empty0 + 8u * lane, MS_CONS_WARPS / 2); mbar_init(xfull0 + 8u * lane, 1); }
        if (lane >= 16 && lane < 24) mbar_init(hfull0 + 8u * (lane - 16), 1);
        if (lane == 31) *abort_flag = 0;
        fence_mbar_init();
        fence_proxy_async_smem();
    }
    if (threadIdx.x == 256) { prefetch_tmap(&tm_w); prefetch_tmap(&tm_s); prefetch_tmap(&tm_x); }
    pdl_wait();
    for (int e = threadIdx.x; e <= p.E; e += MS_THREADS) off[e] = p.offsets[e];
    __syncthreads();
    if (warp == 0) {
        int carry = 0;
        for (int e0 = 0; e0 < p.E; e0 += 32) {
            const int e = e0 + lane;
            const int n = (e < p.E) ? (off[e + 1] - off[e] + tn - 1) / tn * p.n_wt : 0;
            int inc = n;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                if (lane >= d) inc += v;
            }
            if (e < p.E) prefix[e] = carry + inc - n;
            carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
        }
        if (lane == 0) prefix[p.E] = carry;
    }
    __syncthreads();
    const int total = prefix[p.E];
    const int nst = p.K / MS_SK;

    if (warp == MS_CONS_WARPS) {
        // ------------------------------------------------ producer
        if (lane == 0) {
            uint32_t slot = 0, phase = 0;
            int sent = 0, skip = (blockIdx.x == 0) ? p.skip_kb : -1;
            bool ok = true;
            for (int t = blockIdx.x; ok; ) {
                StreamTile tl{0, 0, 0, 0};
                int next = 0;
                if (t < total) {
                    next = static_cast<int>(gridDim.x) + atomicAdd(p.sched, 1);       // asked for early, used at the end of this tile
                    int lo = 0, hi = p.E - 1;                // the last expert whose tiles start at or before t
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (prefix[mid] <= t) lo = mid; else hi = mid - 1;
                    }
                    // chunks of the segment fastest: the second chunk finds its weights in L2
                    const int n_ch = (off[lo + 1] - off[lo] + tn - 1) / tn, local = t - prefix[lo];
                    tl.e = lo;
                    tl.wt = local / n_ch;
                    tl.tok0 = off[lo] + (local - tl.wt * n_ch) * tn;
                    tl.n = min(tn, off[lo + 1] - tl.tok0);
                }
                const int nt = (tl.n + 7) >> 3;
                for (int st = 0; st < (tl.n ? nst : 2); ++st, ++sent) {     // no more tiles: two empty stages, one for each set, say so
                    if (sent >= p.n_stages && !ms_wait(empty0 + 8u * slot, phase ^ 1u, abort_flag, p)) { ok = false; break; }
                    const uint32_t dst = ring + slot * p.stage_bytes, bar = full0 + 8u * slot, xbar = xfull0 + 8u * slot;
                    volatile StreamTile* d = tiles + slot;
                    d->e = tl.e; d->wt = tl.wt; d->tok0 = tl.tok0; d->n = tl.n;
                    if (tl.n == 0) {
                        mbar_arrive(xbar);
                        mbar_arrive(bar);
                        if (++slot == static_cast<uint32_t>(p.n_stages)) { slot = 0; phase ^= 1u; }
                        continue;
                    }
                    mbar_arrive_expect_tx(xbar, nt * MS_X_BYTES);
                    if (st != skip)
                        for (int i = 0; i < nt; ++i)
                            tma_load_3d(dst + MS_W_BYTES + MS_S_BYTES + i * MS_X_BYTES, &tm_x, 0, tl.tok0 + 8 * i, st * 8, xbar);
                    mbar_arrive_expect_tx(bar, MS_W_BYTES + MS_S_BYTES);
                    if constexpr (GATE_UP) {
                        tma_load_3d(dst, &tm_w, st * 128, tl.wt * 64, 2 * tl.e, bar);
                        tma_load_3d(dst + MS_W_BYTES, &tm_s, st * 8, tl.wt * 64, 2 * tl.e, bar);
                    } else {
                        tma_load_2d(dst, &tm_w, st * 128, tl.e * p.N + tl.wt * MS_ROWS, bar);
                        tma_load_2d(dst + MS_W_BYTES, &tm_s, st * 8, tl.e * p.N + tl.wt * MS_ROWS, bar);
                    }
                    if (++slot == static_cast<uint32_t>(p.n_stages)) { slot = 0; phase ^= 1u; }
                }
                if (tl.n == 0) break;
                t = next;
                skip = -1;
            }
        }
    } else if (warp == MS_CONS_WARPS + 1) {
        // ------------------------------------------------ segment rows: each group of eight k into the order 0, 2, 4, 6, 1, 3,
        // 5, 7 of q4_spread, in place
        uint32_t slot = 0, phase = 0;
        int ends = 0;
        while (ends < 2 && __all_sync(0xFFFFFFFFu, ms_wait(xfull0 + 8u * slot, phase, abort_flag, p))) {
            const int nt = (tiles[slot].n + 7) >> 3;
            ends += (nt == 0);
            const uint32_t x = ring + slot * p.stage_bytes + MS_W_BYTES + MS_S_BYTES;
            for (int i = 0; i < nt; ++i) {
                const uint32_t xi = x + i * MS_X_BYTES;
                uint4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = lds_u4(xi + u * 512 + lane * 16);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const uint4 o = make_uint4(__byte_perm(v[u].x, v[u].y, 0x5410), __byte_perm(v[u].z, v[u].w, 0x5410),
                                               __byte_perm(v[u].x, v[u].y, 0x7632), __byte_perm(v[u].z, v[u].w, 0x7632));
                    sts_u4(xi + u * 512 + lane * 16, o);
                }
            }
            fence_proxy_async_smem();              // the slot's next load comes after these writes
            __syncwarp();
            if (lane == 0) mbar_arrive(full0 + 8u * slot);
            if (++slot == static_cast<uint32_t>(p.n_stages)) { slot = 0; phase ^= 1u; }
        }
    } else {
        // ------------------------------------------------ consumers: two sets of four warps, set 0 takes the even stages and
        // set 1 the odd ones, a warp 32 weight rows of each
        constexpr int HI = GATE_UP ? 64 : 8, STEP = GATE_UP ? 8 : 16;     // distance of a tile's two halves, and of the two tiles
        const int set = warp >> 2, w4 = warp & 3;
        const int g = lane >> 2, j = lane & 3;
        const uint32_t row = (GATE_UP ? 16 : 32) * w4 + g;
        const uint32_t wl0 = ring + row * 128 + (g << 4) + 4 * j;         // block b of the row: 16-byte chunk b ^ g
        const uint32_t sc0 = ring + MS_W_BYTES + row * 16;
        const uint32_t x0 = ring + MS_W_BYTES + MS_S_BYTES + lane * 16;
        const uint32_t my_xch = xch + (w4 * NTM * 2 * 32 + lane) * 16, hfull = hfull0 + 8u * w4, hempty = hempty0 + 8u * w4;
        uint32_t slot = set, phase = 0;
        float wl = 0.f;                       // routing weight of row `lane` of the chunk
        int have = -1;                        // first row of the chunk wl belongs to
        for (uint32_t q = 0, base = 0; ; ++q, base += nst) {              // tile and its first stage, both counted from 0
            const uint32_t first = base + ((base ^ set) & 1u);            // this set's first stage of the tile
            if (first >= base + nst) continue;                            // (K = 256: every other tile is the other set's)
            if (!__all_sync(0xFFFFFFFFu, ms_wait(full0 + 8u * slot, phase, abort_flag, p))) break;
            const int wt = tiles[slot].wt, tok0 = tiles[slot].tok0, n = tiles[slot].n;
            if (n == 0) break;
            const int nt_n = (n + 7) >> 3;
            const bool mine = ((base + nst - 1 - set) & 1u) == 0;         // the set with the last stage finishes the tile
            if (mine && p.topk_w && have != tok0) {
                wl = (lane < n) ? p.topk_w[p.row_pair[tok0 + lane]] : 0.f;
                have = tok0;
            }
            float acc[NTM][2][4];
#pragma unroll
            for (int nt = 0; nt < NTM; ++nt)
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[nt][e >> 2][e & 3] = 0.f;
            bool ok = true;
            for (uint32_t st = first; st < base + nst; st += 2) {
                ok = __all_sync(0xFFFFFFFFu, ms_wait(full0 + 8u * slot, phase, abort_flag, p));
                if (!ok) break;
                const uint32_t o = slot * p.stage_bytes;
                if (NTM == 1 || nt_n == 1) ms_stage<1, HI, STEP>(acc, wl0 + o, x0 + o, sc0 + o);
                else ms_stage<NTM, HI, STEP>(acc, wl0 + o, x0 + o, sc0 + o);
                __syncwarp();
                if (lane == 0) mbar_arrive(empty0 + 8u * slot);
                slot += 2;
                if (slot >= static_cast<uint32_t>(p.n_stages)) { slot -= p.n_stages; phase ^= 1u; }
            }
            if (!ok) break;
            if (nst > 1 && !mine) {           // hand the sums to the other set's warp of the same rows
                if (q > 0 && !__all_sync(0xFFFFFFFFu, ms_wait(hempty, (q & 1u) ^ 1u, abort_flag, p))) break;
#pragma unroll
                for (int nt = 0; nt < NTM; ++nt)
#pragma unroll
                    for (int m = 0; m < 2; ++m)
                        if (nt < nt_n)
                            sts_u4(my_xch + (nt * 2 + m) * 512, make_uint4(__float_as_uint(acc[nt][m][0]), __float_as_uint(acc[nt][m][1]),
                                                                           __float_as_uint(acc[nt][m][2]), __float_as_uint(acc[nt][m][3])));
                __syncwarp();
                if (lane == 0) mbar_arrive(hfull);
                continue;
            }
            if (nst > 1 && !__all_sync(0xFFFFFFFFu, ms_wait(hfull, q & 1u, abort_flag, p))) break;
#pragma unroll
            for (int nt = 0; nt < NTM; ++nt) {
                if (nt >= nt_n) break;
                const int t = 8 * nt + 2 * j;
                float w0 = 1.f, w1 = 1.f;
                if (!GATE_UP && p.topk_w) { w0 = __shfl_sync(0xFFFFFFFFu, wl, t); w1 = __shfl_sync(0xFFFFFFFFu, wl, t + 1); }
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    float c0 = acc[nt][m][0], c1 = acc[nt][m][1], c2 = acc[nt][m][2], c3 = acc[nt][m][3];   // rows lo / hi x segment rows t, t + 1
                    if (nst > 1) {
                        const uint4 v = lds_u4(my_xch + (nt * 2 + m) * 512);
                        c0 += __uint_as_float(v.x); c1 += __uint_as_float(v.y); c2 += __uint_as_float(v.z); c3 += __uint_as_float(v.w);
                    }
                    __nv_bfloat16* o = p.out;
                    if constexpr (GATE_UP) {
                        const int F = p.N >> 1;
                        o += static_cast<size_t>(tok0 + t) * F + wt * 64 + 16 * w4 + 8 * m + g;
                        if (t < n) o[0] = __float2bfloat16_rn(silu_mul(c0, c2));
                        if (t + 1 < n) o[F] = __float2bfloat16_rn(silu_mul(c1, c3));
                    } else {
                        if (p.topk_w) { c0 *= w0; c1 *= w1; c2 *= w0; c3 *= w1; }
                        const int r = wt * MS_ROWS + 32 * w4 + 16 * m;       // N % 8 == 0: a half's eight rows are all inside or all outside
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
            if (nst > 1) {
                __syncwarp();
                if (lane == 0) mbar_arrive(hempty);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {                    // whoever is last leaves the counters ready for the next launch
        __threadfence();
        if (atomicAdd(p.sched + 1, 1) == static_cast<int>(gridDim.x) - 1) { p.sched[0] = 0; p.sched[1] = 0; }
    }
    if (*abort_flag) {
        for (int i = 0; i < 64; ++i) __nanosleep(2000);       // copies still in flight land before the memory is released
    }
}

// The host side.  Returns QG_ERR_WORKSPACE if the shape does not fit this kernel (the caller takes the other one).
int launch_moe_stream(qg_ctx* ctx, int mode, int R, int E, int N, int K, const void* Ain, const int32_t* offsets,
                      const void* Wq, const void* Ws, const float* topk_w, const int32_t* row_pair, void* Out, cudaStream_t st) {
    const bool gate_up = mode == QG_MODE_GATE_UP_SILU;
    if (R > static_cast<long long>(MS_MAX_ROWS) * E) return QG_ERR_WORKSPACE;
    StreamParams p{};
    p.R = R; p.N = N; p.K = K; p.E = E;
    p.n_wt = gate_up ? N / 128 : (N + MS_ROWS - 1) / MS_ROWS;
    // Rows per tile: eight up to five rows per expert, sixteen above.  The wider tile's ring is a stage shorter (56.1 us
    // against 53.0 at four rows per expert, gate/up); cutting a segment in two costs more from six on (60.4 with eight and
    // 61.4 with sixteen at six rows, 68.2 and 63.9 at eight, 79.4 and 68.1 at ten).  24 and 32 rows were slower throughout.
    p.nt_max = (R <= 5LL * E) ? 1 : MS_NT;
    p.stage_bytes = (MS_W_BYTES + MS_S_BYTES + p.nt_max * MS_X_BYTES + 1023) & ~1023;      // the codes' swizzle wants 1 KB
    const size_t fixed = 1024 + 4 * p.nt_max * 2 * 512 + 24 * MS_MAX_ST + 64 + 16 + 16 * MS_MAX_ST + (2 * static_cast<size_t>(E) + 2) * sizeof(int);
    p.n_stages = static_cast<int>((MS_SMEM_MAX - fixed) / p.stage_bytes);
    if (p.n_stages > MS_MAX_ST) p.n_stages = MS_MAX_ST;
    // An even number, so that a slot's stages all belong to one set: with an odd one a set would see every other phase of a
    // slot's barrier only, and a wait by parity passes too early when the phase in between is not complete yet.
    p.n_stages &= ~1;
    if (p.n_stages < 2) return QG_ERR_WORKSPACE;
    const size_t smem = fixed + static_cast<size_t>(p.n_stages) * p.stage_bytes;
    p.offsets = offsets; p.out = static_cast<__nv_bfloat16*>(Out);
    p.topk_w = (mode == QG_MODE_DOWN_WEIGHTED) ? topk_w : nullptr; p.row_pair = row_pair;
    p.sched = ctx->gemv_tickets + ctx->gemv_ticket_count;
    p.status = ctx->d_status; p.wait_limit = ctx->wait_limit;
    p.skip_kb = ctx->skip_kb < 0 ? -1 : ctx->skip_kb / (MS_SK / 64);
    CUtensorMap tm_w, tm_s, tm_x;
    const uint64_t kb = K / 2, ks = K / 32, wrows = static_cast<uint64_t>(E) * N;
    int rc = gate_up ? get_tmap_3d(ctx, &tm_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, kb, N / 2, 2ull * E, kb * (N / 2), 128, 64, 2,
                                   CU_TENSOR_MAP_SWIZZLE_128B)
                     : get_tmap_2d(ctx, &tm_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, Wq, kb, wrows, 128, MS_ROWS, CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc == QG_OK)
        rc = gate_up ? get_tmap_3d(ctx, &tm_s, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, Ws, ks, N / 2, 2ull * E, ks * 2 * (N / 2), 8, 64, 2,
                                   CU_TENSOR_MAP_SWIZZLE_NONE)
                     : get_tmap_2d(ctx, &tm_s, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, Ws, ks, wrows, 8, MS_ROWS, CU_TENSOR_MAP_SWIZZLE_NONE);
    if (rc == QG_OK)
        rc = get_tmap_3d(ctx, &tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Ain, 32, R, K / 32, 64, 32, 8, 8, CU_TENSOR_MAP_SWIZZLE_NONE,
                         static_cast<uint64_t>(K) * 2);
    if (rc != QG_OK) return rc;
    auto kern = (p.nt_max == 1) ? (gate_up ? moe_stream_kernel<true, 1> : moe_stream_kernel<false, 1>)
                                : (gate_up ? moe_stream_kernel<true, MS_NT> : moe_stream_kernel<false, MS_NT>);
    const int inst = ATTR_MOE_STREAM + (gate_up ? 2 : 0) + p.nt_max - 1;
    if (!ctx->attr_set[inst]) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(MS_SMEM_MAX)) != cudaSuccess) {
            cudaGetLastError();
            return QG_ERR_CUDA;
        }
        ctx->attr_set[inst] = true;
    }
    ctx->skip_kb = -1;                                        // the test hook acts on one launch
    // at most one chunk per eight rows nt_max and one more per expert that has rows
    const long long chunks = R / (8 * p.nt_max) + (R < E ? R : E);
    const long long max_tiles = chunks * p.n_wt;
    const int grid = static_cast<int>(max_tiles < 2LL * ctx->sm_count ? max_tiles : 2LL * ctx->sm_count);
    if (launch_kernel(ctx, kern, dim3(grid), dim3(MS_THREADS), smem, st, tm_w, tm_s, tm_x, p) != cudaSuccess) {
        cudaGetLastError();
        return QG_ERR_CUDA;
    }
    return QG_OK;
}

}  // namespace qg
