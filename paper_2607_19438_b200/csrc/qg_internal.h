// Internal declarations shared by the translation units of the library (not part of the ABI).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "../../include/qgemm.h"

namespace qg {
// One cached tensor map: the key is everything cuTensorMapEncodeTiled was given.
struct TmapEntry {
    const void* base;
    uint64_t inner, rows, row_stride;
    uint32_t box_inner, box_rows;
    uint64_t planes, plane_stride;   // third dimension of a 3-D map (0 for 2-D maps)
    uint32_t box_planes;
    int dt, elem_bytes, swz;
    CUtensorMap map;
};
constexpr int TMAP_CACHE = 2048, TMAP_WAYS = 8;   // entries, entries per hashed set
constexpr uint32_t DEFAULT_WAIT_LIMIT = 1u << 18;   // polls; an unsatisfied try_wait poll lasts about 4 us: about a second
// Slots of qg_ctx::attr_set, one per kernel instantiation that needs the dynamic shared-memory attribute.
enum AttrSlot {
    ATTR_GEMM = 0,          // 18 slots: format (2) x token tile (3) x epilogue (3)
    ATTR_GEMV = 18,         // 2: Q8, Q4
    ATTR_ATTN = 20,         // 3: head dimensions
    ATTR_ROUTER_1 = 23,
    ATTR_GEMM_SK = 24,      // 6: format (2) x token tile (3), stream-K
    ATTR_MX_192 = 30,
    ATTR_ROUTER_4 = 31,
    ATTR_MX_MOE = 32,       // 2: down, gate/up
    ATTR_MX_256 = 34,
    ATTR_STREAM = 35,       // 8: sorted, gathered rows x down, gate/up x rows per tile (2)
    ATTR_DENSE_STREAM = 43, // 8: K whole, in slices x format (2) x more than eight tokens (2)
    ATTR_GEMM_CHOICE = 51,  // 2: epilogue
    ATTR_SLOTS = 53
};
}  // namespace qg

struct qg_ctx {
    int device;
    int sm_count;
    int* d_status;  // device status word: 0, or the first QG_ERR_* a kernel recorded
    CUresult (*encode_tiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                             const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                             CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    int force_bt;              // QG_FORCE_BT at creation (0: heuristic)
    uint32_t wait_limit;       // polls per bounded device wait
    int skip_kb;               // test hook, consumed by the next GEMM launch (-1: none)
    bool attr_set[qg::ATTR_SLOTS];        // per kernel instantiation: dynamic shared-memory attribute set on this device
    qg::TmapEntry tmaps[qg::TMAP_CACHE];   // tensor maps of recent calls (weights and buffers recur every layer)
    unsigned tmap_next;        // replacement counter
    bool pdl;                  // launch kernels with programmatic stream serialization (QG_NO_PDL=1 turns it off)
    float* sk_partial;         // stream-K: one fp32 partial tile (256 tokens x 128 rows) per CTA
    int* sk_flags;             // stream-K: two counters per CTA, zero between launches
    int streamk_mode;          // QG_STREAMK at creation: -1 heuristic (default), 0 never, 1 whenever legal
    float* gemv_partial;       // K-slice partial sums of qgemm_small_m's block kernel, [slices][16][N] fp32
    size_t gemv_partial_bytes;
    int* gemv_tickets;         // one arrival counter per 64-row tile, zero between launches
    int gemv_ticket_count;
    int slice_clusters[4][5];      // dense GEMM with K slices, per format x token tile and slices: clusters that fit at once (0 unknown, -1 none)
    int gemv_mode;             // test hook (qg_test_gemv_mode): bit 0 no clusters, bit 1 always the streaming kernel, bit 2 never
    int gemv_max_clusters[4][9];   // streaming kernel, per instantiation and cluster size: clusters that fit at once (0 unknown, -1 none)
    long long* stats;          // profiling builds only
};

namespace qg {
// Launches `kern`; with ctx->pdl the launch carries the programmatic-serialization attribute, so the kernel's prologue
// may overlap the tail of the kernel before it in the stream.  Every kernel of this library calls pdl_wait() before it reads
// or writes anything an earlier kernel may touch, except quantised weights, which no kernel of this library writes: the GEMMs
// that take codes and scales request their first ones before the wait.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(const qg_ctx* ctx, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                 cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = ctx->pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
// QG_OK if the calling thread's current device is the context's, else QG_ERR_DEVICE.
int check_device(const qg_ctx* ctx);
// Makes the context's device the current one for a question about it, and leaves the caller's as it was.
struct OnDevice {
    int prev = -1;
    bool ok;
    explicit OnDevice(int device) {
        ok = cudaGetDevice(&prev) == cudaSuccess && (prev == device || cudaSetDevice(device) == cudaSuccess);
        if (prev == device) prev = -1;
        if (!ok) cudaGetLastError();
    }
    ~OnDevice() { if (prev >= 0) cudaSetDevice(prev); }
};
// A 2-D row-major tensor map (inner = contiguous extent in elements, box in elements, row_stride_bytes = distance
// between rows, 0 = packed): looked up in the context's cache, encoded on a miss, and copied to *out (the caller's own
// copy: a later lookup may replace the cached entry).
int get_tmap_2d(qg_ctx* ctx, CUtensorMap* out, CUtensorMapDataType dt, int elem_bytes, const void* base,
                uint64_t inner, uint64_t rows, uint32_t box_inner, uint32_t box_rows, CUtensorMapSwizzle swz,
                uint64_t row_stride_bytes = 0);
// The same with a third dimension: `planes` planes of `rows` rows, plane_stride_bytes apart; box = box_inner x box_rows x
// box_planes, which lands in shared memory plane after plane.
int get_tmap_3d(qg_ctx* ctx, CUtensorMap* out, CUtensorMapDataType dt, int elem_bytes, const void* base,
                uint64_t inner, uint64_t rows, uint64_t planes, uint64_t plane_stride_bytes, uint32_t box_inner,
                uint32_t box_rows, uint32_t box_planes, CUtensorMapSwizzle swz, uint64_t row_stride_bytes = 0);
// Which of its two kernels serves a grouped call with 4-bit weights: the streaming kernel when every expert has a few rows, the
// tensor-memory kernel when they crowd into few experts, and how the rows are spread only the device knows.  By the times below the faster
// kernel is chosen in 758 of 780 calls or missed by less than 5 % (eight layers of 8 to 512 experts, a quarter of a row to 32 rows per
// expert; rows spread evenly, with a quarter of the experts preferred, over eight experts, all with one); 1.004 of the faster one's time on
// average, 1.27 at worst.  (The times of the other kernel lie 7 % above what it takes by now.  Fitted anew, 773 of the 780 calls are within
// 5 %, but the host's choice, which knows the averages only, is no better: 1.011 and 1.012 of the fastest with even and uneven rows, now 1.012
// and 1.011, and its worst uneven call 1.39 instead of 1.20.)
//   The host weighs three calls with evenly spread rows against one with all rows in one segment: the streaming kernel alone,
// the other alone, or both, in which case each works out the same answer from the offsets and the one that is not wanted ends at
// once.  That costs every such call 3 to 14 us (the unwanted launch keeps the next one from starting early).  128 experts,
// 1536 x 2048: alone up to 12 rows per expert (even 62 us against 91, one segment 39 against 16 at eight rows), both up to 17,
// the other from there (even 100 against 91, one segment 71 against 25 at eighteen).  256 experts, 4096 x 7168, eight rows: both
// (even 1009 us against 1680 of the other alone; eight segments 173 against 562 of the streaming kernel and 126 of the other).
struct GroupedChoice {
    enum Way { STREAM, OTHER, BOTH };
    int on;                    // both kernels are launched
    int chunk;                 // rows per tile of the streaming kernel, 8 or 16
    int n_wt, stages;          // its weight tiles per expert and 256-k stages per tile
    int sm_count;
    // ns of each kernel; chunks: row tiles of all experts, wide: their tiles of 128 rows
    __host__ __device__ long long stream_ns(long long chunks) const {
        const long long ctas = 2 * sm_count, tiles = chunks * n_wt, waves = (tiles + ctas - 1) / ctas;
        const long long halves = waves > 2 ? tiles + waves * ctas : 2 * waves * ctas;        // waves, in units of 1 / (2 ctas)
        return 1300 + halves * stages * (chunk == 8 ? 1000 : 1300) / (2 * ctas) + waves * 1500;
    }
    __host__ __device__ long long other_ns(long long wide) const {
        const long long pairs = sm_count / 2;
        return 8000 + (wide * ((n_wt + 1) / 2) + pairs - 1) / pairs * stages * (4 * 271);
    }
    __host__ __device__ bool streams(long long chunks, long long wide) const { return stream_ns(chunks) <= other_ns(wide); }
    // Rows per expert, on average.  Evenly spread and sorted, the streaming kernel takes 0.94 of the other one's time at 14, 1.05 at 16 and
    // 1.13 at 18 (eight layers); gathered, 0.93 at 16 and 0.96 at 18, and both forms take the same kernel.
    static constexpr int MAX_ROWS = 18;
    Way plan(long long R, long long E) const {
        if (R > MAX_ROWS * E) return OTHER;
        // rows drawn evenly (Poisson): a tile per expert up to 5/8 of a tile's rows, then 3/8 of a tile more than the rows fill
        const long long used = R < E ? R : E, even = 8 * R <= 5 * chunk * E ? used : R / chunk + 3 * E / 8;
        const long long gain = other_ns(used) - stream_ns(even), loss = stream_ns((R + chunk - 1) / chunk) - other_ns((R + 127) / 128);
        const long long stream = loss > 0 ? loss : 0, other = gain > 0 ? 3 * gain : 0, both = 4 * (6000 + 10 * E);
        if (stream <= other && stream <= both) return STREAM;
        return other <= both ? OTHER : BOTH;
    }
};
// The streaming kernel of the grouped GEMM (4-bit weights, modes 0 to 2), for a few rows per expert; QG_ERR_WORKSPACE if the
// shape does not suit it.  choice.on: the other kernel has to be launched behind it.
int launch_moe_stream(qg_ctx* ctx, int mode, int R, int E, int N, int K, const void* Ain, int in_rows, int gather_k, const int32_t* offsets,
                      const void* Wq, const void* Ws, const float* topk_w, const int32_t* row_pair, void* Out, GroupedChoice& choice, cudaStream_t st);
// The same kernel for one matrix and up to sixteen tokens.
int launch_dense_stream(qg_ctx* ctx, int qbits, int M, int N, int K, const void* A, const void* Wq, const void* Ws, void* Cout,
                        cudaStream_t st);
}  // namespace qg
