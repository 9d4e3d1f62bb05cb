// lmhead.cu -- row statistics straight from the LM head (rps_lmhead_row_stats).
//
// Each scored row's logits are z = h W^T: its hidden state h (d bf16) against
// the unembedding W (one row of d bf16 weights per token). The paper's p_i is
// the softmax of that row (Sec. 2 notation), and the statistics of Eq. 1 and
// Eq. 3 follow from it. Here the contraction runs on the tensor cores and the
// statistics are folded in its epilogue, so the logits never reach HBM.
//
// Contraction. A CTA owns one tile of 128 hidden rows and one contiguous range
// of the vocabulary (a "split"), walked in tiles of 256 tokens; the CTAs of
// every row tile take the same splits, so they stream the same unembedding
// tiles at the same pace and each tile comes from HBM once, the other row tiles
// finding it in L2. Two row tiles can share a CTA pair (cta_group::2): M = 256
// over both, half of each unembedding tile in either CTA.
//   warp 0      TMA producer: per stage, the hidden tile's and the unembedding
//               tile's 64-wide slices of d (one, or several of a narrow
//               tile), 128-byte swizzle, into a ring of shared-memory stages
//               (mbarrier completion, bounded waits). A
//               pair takes two slices per stage and one copy per operand: with
//               a copy per 64 rows and slice the one issuing thread set the pace
//               (512 rows: 329 us against 309);
//   warp 1      MMA issuer (the pair's first CTA): tcgen05.mma kind::f16 (bf16 x
//               bf16 -> f32), M = 128 or 256, N = 256, K = 16, four per slice,
//               into one of two TMEM accumulators (128 lanes x 256 columns each),
//               so that the epilogue of one tile overlaps the contraction of the
//               next; it also allocates and frees the 512 TMEM columns;
//   warps 2-5   epilogue: thread = row (TMEM lane). tcgen05.ld brings its 256
//               logits; pass 1 finds the tile maximum, pass 2 folds the
//               logits into the row's base-2 online softmax record (B, S, T
//               with S = sum 2^u, T = sum u 2^u, u = z log2(e) - B), the
//               running maximum and argmax, and, in top-k mode, a sorted
//               register list of the KMAX largest logits. A warp inserts as
//               often as its busiest lane, so few columns may enter: the first
//               tile's group maxima bound the k-th logit before any does (200
//               rows, V 32,000, d 1,024, k 10: 72 -> 36 us with the pairs).
// At the end of its range each epilogue thread leaves its row's record and
// list in the workspace; a second launch (one warp per row) merges the splits
// and writes the statistics, with the same formulas as the streaming kernel.
//
// Every mbarrier wait is bounded (%globaltimer). A role whose wait runs out
// flags RPS_DEVERR_TIMEOUT, marks the workspace unhealthy and raises a CTA
// abort flag that ends the other roles' waits; the producer then waits,
// bounded, for the copies it issued, the MMA issuer for the MMAs it issued,
// and TMEM is freed before the CTA exits.
#include <cuda.h>  // CUtensorMap and the tensor-map encoder's signature (no link against the driver)
#include <cudaTypedefs.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <cstring>
#include <mutex>

#include "lmhead_split.h"
#include "rps_internal.cuh"
#include "topk_device.cuh"
#include "umma_desc.h"

namespace rps {
namespace {

constexpr int kTileK = 64;                  // d per stage: one 128-byte swizzle row of bf16
constexpr int kMmaK = 16;                   // K of one tcgen05.mma kind::f16
constexpr int kABytes = kTileM * kTileK * 2;  // 16 KB
constexpr int kBBytes = kTileN * kTileK * 2;  // 32 KB
constexpr int kEpiWarps = 4;
constexpr int kMaxStages = 5;
constexpr int kCopyRows = kTileN / 4;       // unembedding rows per copy of a narrow tile (single CTAs)
constexpr int kLineRows = 16;               // packed rows (128 bytes each) per line of the pair's tensor map
// Shape of the contraction by CTA group: one CTA (CG 1) with the whole
// unembedding tile in its stages, or a pair (CG 2) with half of it each.
template <int CG>
struct Shape {
    static constexpr int stages = CG == 1 ? 4 : 3;
    static constexpr int slices = CG == 1 ? 1 : 2;              // 64-wide slices of d per stage
    static constexpr int stage_bytes = slices * (kABytes + kBBytes / CG);
    // the ring, 32 logits per epilogue thread, and slack to align the ring to 1024 bytes
    static constexpr int ring_bytes = stages * stage_bytes;
    static constexpr int smem_bytes = ring_bytes + kEpiWarps * 32 * 32 * 4 + 1024;
    static_assert(stages <= kMaxStages, "");
};
// A single CTA's ring cut by its rows (FLEX): with few rows a fifth stage fits, and
// a narrow last tile takes several slices of d per stage, since each stage costs
// its barriers and commit whatever it holds. 32 rows of V 126,464, d 4,096 172 -> 164 us
// (with the fifth stage alone 167); 53 rows of V 8,723, d 3,456 35 -> 31. Twelve stages of
// one slice instead of four of three: 38.5.
__host__ __device__ constexpr int slice_rows_bytes(int rows) { return (rows * kTileK * 2 + 1023) / 1024 * 1024; }  // (the swizzle's period)
__host__ __device__ __forceinline__ int tile_slices(int n_cols, int a_bytes, int stage_bytes) {
    const int n = stage_bytes / (a_bytes + n_cols * kTileK * 2);
    return n < 4 ? n : 4;
}
constexpr int kThreads = 192;               // warp 0 TMA, warp 1 MMA, warps 2-5 epilogue
constexpr uint32_t kTmemCols = 2 * kTileN;  // two accumulators
constexpr int kMergeThreads = 128;
constexpr uint64_t kDrainNs = 200ull * 1000 * 1000;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// One split's record of a row.
struct __align__(16) LmPartial {
    float B;   // base-2 reference
    float s;   // sum 2^u
    float t;   // sum u 2^u
    float mx;  // largest logit
    int32_t amax;
    int32_t pad[3];
};

struct LmArgs {
    int32_t n_rows, d, splits, kmax, k;
    int32_t granule, n_gran;  // tokens the splits are cut at, granules of the vocabulary
    int32_t h_rows;  // rows of a hidden copy: a tile's, or all of fewer
    int32_t stages, stage_bytes;  // the ring (CG 1)
    const uint8_t *w_packed;  // unembedding in the packed tile layout, or nullptr (tensor map)
    int64_t vocab;
    LmPartial *part;   // [n_rows][splits]
    float2 *lists;     // [n_rows][splits][kmax]: (logit, token id as int bits)
    float *logits_out; // optional [n_rows][vocab]
    uint32_t *health;
    uint32_t *err;
    uint64_t wait_ns;
    float *zmax, *lse, *H, *pmax, *mu, *htrunc, *topk_logit;
    int32_t *argmax, *topk_idx;
};

// ---------------------------------------------------------------- PTX
__device__ __forceinline__ uint32_t saddr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(bar)), "r"(bytes) : "memory");
}
// (a pair: cluster scope, the arrival may come from the other CTA)
template <int CG>
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t done;
    if constexpr (CG == 1)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(saddr(bar)), "r"(parity)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(saddr(bar)), "r"(parity)
            : "memory");
    return done != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int c0, int c1, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            saddr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(saddr(bar))
        : "memory");
}
// The same as half of a CTA pair: `bar` is a cluster address, in either CTA of the pair.
__device__ __forceinline__ void tma_load_3d_pair(void *dst, const CUtensorMap *map, int c0, int c1, int c2,
                                                 uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
        "%3, %4}], [%5];" ::"r"(saddr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}
// Cluster address of `p`'s counterpart in CTA 0 of the cluster.
__device__ __forceinline__ uint32_t leader_addr(const void *p) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(saddr(p)));
    return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// Plain bulk copy of `bytes` contiguous bytes into shared memory, completing on `bar`.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     saddr(dst)),
                 "l"(src), "r"(bytes), "r"(saddr(bar))
                 : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

template <int CG>
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {
    if constexpr (CG == 1)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(slot)), "r"(ncols)
                     : "memory");
    else
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(slot)), "r"(ncols)
                     : "memory");
}
template <int CG>
__device__ __forceinline__ void tmem_relinquish() {
    if constexpr (CG == 1) asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    else asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
template <int CG>
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    if constexpr (CG == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
    else
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] x B[smem]^T, bf16 inputs, f32 accumulator; accumulate != 0
// adds to D. CG 2: A, B and D are spread over the pair, half in each CTA at the
// same addresses.
template <int CG>
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
    if constexpr (CG == 1)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
            "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
            "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
            : "memory");
}
// Arrives on `bar` once every tcgen05 operation this thread issued before has
// completed; CG 2: on the barrier's counterpart in both CTAs of the pair.
template <int CG>
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    if constexpr (CG == 1)
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar))
                     : "memory");
    else
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                saddr(bar)),
            "h"(static_cast<uint16_t>(3))
            : "memory");
}

// 32 consecutive f32 columns of this thread's TMEM lane (the warp's 32 lanes at once).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---------------------------------------------------------------- bounded waits
struct Ctl {
    uint64_t full[kMaxStages], empty[kMaxStages], acc_full[2], acc_empty[2], mma_done;
    uint32_t tmem_base;
    int abort_flag;
    int skip;
};

// Waits for phase `parity` of `bar`. False when the CTA aborts: this wait ran
// out (then it flags the timeout, marks the workspace and raises the abort
// flag) or another role already aborted.
template <int CG>
__device__ bool wait_or_abort(uint64_t *bar, uint32_t parity, Ctl &c, const LmArgs &a) {
    if (a.wait_ns != 0 && mbar_try_wait<CG>(bar, parity)) return true;
    const uint64_t start = global_ns();
    while (a.wait_ns != 0) {
        if (mbar_try_wait<CG>(bar, parity)) return true;
        if (*reinterpret_cast<volatile int *>(&c.abort_flag)) return false;
        if (global_ns() - start > a.wait_ns) break;
    }
    flag_error(a.err, RPS_DEVERR_TIMEOUT);
    atomicExch(a.health, 1u);
    *reinterpret_cast<volatile int *>(&c.abort_flag) = 1;
    return false;
}

// wait_or_abort for every lane of a warp that goes on to warp-wide tcgen05
// instructions: the warp leaves together, on the same answer.
template <int CG, typename Ctl_, typename Args_>
__device__ __forceinline__ bool warp_wait_or_abort(uint64_t *bar, uint32_t parity, Ctl_ &c, const Args_ &a) {
    return __all_sync(kFull, wait_or_abort<CG>(bar, parity, c, a));
}

// A wait that only ends early when the phase completes (drains before exit).
template <int CG>
__device__ void wait_drain(uint64_t *bar, uint32_t parity) {
    if (mbar_try_wait<CG>(bar, parity)) return;
    const uint64_t start = global_ns();
    while (global_ns() - start < kDrainNs)
        if (mbar_try_wait<CG>(bar, parity)) return;
}

// ---------------------------------------------------------------- epilogue state
template <int KMAX>
struct RowState {
    float B, s, t, mx;
    int amx;
    float lv[KMAX > 0 ? KMAX : 1];
    int li[KMAX > 0 ? KMAX : 1];
};

// Inserts (z, id) into the sorted list (logit desc; ids arrive in increasing
// order, so equal logits keep the lower id first). Called for z > lv[KMAX-1].
// Every entry is formed from the old list (itself, its neighbour or z), so the
// steps do not wait for one another.
template <int KMAX>
__device__ __forceinline__ void list_insert(RowState<KMAX> &st, float z, int id) {
#pragma unroll
    for (int i = KMAX - 1; i > 0; --i) {
        const float cur = st.lv[i], up = st.lv[i - 1];
        const int cur_i = st.li[i], up_i = st.li[i - 1];
        const float v = z > up ? up : z;
        const int vi = z > up ? up_i : id;
        st.lv[i] = z > cur ? v : cur;
        st.li[i] = z > cur ? vi : cur_i;
    }
    const float top = st.lv[0];
    const int top_i = st.li[0];
    st.lv[0] = z > top ? z : top;
    st.li[0] = z > top ? id : top_i;
}

// Sorts v descending (bitonic network over registers).
template <int N>
__device__ __forceinline__ void sort_desc(float (&v)[N]) {
#pragma unroll
    for (int size = 2; size <= N; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int j = i ^ stride;
                if (j > i) {
                    const float hi = fmaxf(v[i], v[j]), lo = fminf(v[i], v[j]);
                    v[i] = (i & size) == 0 ? hi : lo;
                    v[j] = (i & size) == 0 ? lo : hi;
                }
            }
        }
    }
}

// The float below x (-inf and NaN stay).
__device__ __forceinline__ float next_below(float x) {
    if (!(x > -INFINITY)) return x;
    if (x == 0.f) return __uint_as_float(0x80000001u);
    const uint32_t b = __float_as_uint(x);
    return __uint_as_float(x > 0.f ? b - 1 : b + 1);
}

// FLEX: the ring cut by the launch's rows (CG 1)
template <int KMAX, int CG, bool FLEX>
__global__ void __launch_bounds__(kThreads, 1)
    lmhead_kernel(const __grid_constant__ CUtensorMap tm_h, const __grid_constant__ CUtensorMap tm_w,
                  const __grid_constant__ CUtensorMap tm_w_half, const LmArgs a) {
    using Sh = Shape<CG>;
    const int n_stages = FLEX ? a.stages : Sh::stages;
    const int stage_bytes = FLEX ? a.stage_bytes : Sh::stage_bytes;
    // Bytes of a slice's hidden tile in a stage. The MMA reads 16 KB from its start:
    // what lies there beyond fewer rows (inside the dynamic shared memory: 16 KB
    // follow the ring) are rows past the last, whose results nobody uses.
    const int a_bytes = FLEX ? slice_rows_bytes(a.h_rows) : kABytes;
    extern __shared__ uint8_t dyn_smem[];
    __shared__ Ctl c;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = CG == 1 ? 0 : static_cast<int>(cluster_rank());
    const int unit = static_cast<int>(blockIdx.x) / CG;  // CTA or pair
    const int rt = unit / a.splits * CG + rank, split = unit % a.splits;
    const int col_begin = static_cast<int>(lm_range(split, a.n_gran, a.splits, a.granule));
    const int64_t col_end = lm_range(split + 1, a.n_gran, a.splits, a.granule);
    const int n_tiles = static_cast<int>((col_end - col_begin + kTileN - 1) / kTileN);
    const int kblocks = a.d / kTileK;
    // With fewer rows than a tile the hidden copies are that high: filling most of
    // a tile from outside so small a tensor is slow (V 126,464, d 4,096, k 10: 4 rows
    // 235 -> 164 us; V 32,000, d 1,024: 28.4 -> 22.5). A last tile of several is filled
    // with zeros at no cost, and a pair's empty half is zeroed once.
    const int row0 = rt * kTileM;
    const bool has_rows = row0 < a.n_rows;
    const int h_bytes = a.h_rows * kTileK * 2;  // of one slice
    // the ring starts on a 1024-byte boundary (the 128-byte swizzle's period)
    uint8_t *ring = dyn_smem + ((1024u - (saddr(dyn_smem) & 1023u)) & 1023u);

    if (threadIdx.x == 0) {
        for (int s = 0; s < n_stages; ++s) {
            mbar_init(&c.full[s], 1);
            mbar_init(&c.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&c.acc_full[b], 1);
            mbar_init(&c.acc_empty[b], kEpiWarps * CG);
        }
        mbar_init(&c.mma_done, 1);
        c.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0 && lane == 0) {
        prefetch_map(&tm_h);
        prefetch_map(&tm_w);
    }
    if (warp == 1) {
        tmem_alloc<CG>(&c.tmem_base, kTmemCols);
        tmem_relinquish<CG>();
    }
    if (CG == 2 && !has_rows) {
        for (int i = threadIdx.x; i < Sh::stages * Sh::slices * kABytes / 16; i += kThreads) {
            constexpr int kPerStage = Sh::slices * kABytes / 16;
            *reinterpret_cast<uint4 *>(ring + i / kPerStage * Sh::stage_bytes + i % kPerStage * 16) = make_uint4(0, 0, 0, 0);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    // the hidden rows may come from the previous kernel on the stream
    pdl_wait();
    pdl_launch_next();
    if (threadIdx.x == 0) c.skip = __ldcg(a.health) != 0;
    tc_fence_before();
    __syncthreads();
    if constexpr (CG == 2) {
        cluster_sync();  // the pair's barriers are initialised
        __syncwarp();
    }
    tc_fence_after();
    const uint32_t tmem = c.tmem_base;
    if (c.skip) {  // a workspace an earlier launch gave up on: write nothing
        if (threadIdx.x == 0) flag_error(a.err, RPS_DEVERR_WORKSPACE);
    } else if (warp == 0) {
        if (lane == 0) {  // ---------------------------------------- TMA producer
            uint32_t it = 0;  // stages filled
            const int pair_tiles = (rt | 1) * kTileM < a.n_rows ? 2 : 1;  // row tiles of the pair (CG 2)
            uint32_t ph = 0;
            int s = 0;
            bool ok = true;
            for (int t = 0; t < n_tiles && ok; ++t) {
                const int col0 = col_begin + t * kTileN;
                const int n_cols = static_cast<int>(min(static_cast<int64_t>(kTileN), col_end - col0));  // 256, or whole granules in a range's last tile
                const int slices = FLEX ? tile_slices(n_cols, a_bytes, stage_bytes) : Sh::slices;
                // packed (CG 1): the rest of a 32 KB block, already in the swizzled
                // image, and the start of the next tile's
                const int off = col0 % kTileN, head = min(n_cols, kTileN - off);
                const uint8_t *blk = a.w_packed + static_cast<int64_t>(col0 / kTileN) * kblocks * kBBytes +
                                     static_cast<int64_t>(off) * kTileK * 2;
                const int64_t next_blk = static_cast<int64_t>(kblocks) * kBBytes - static_cast<int64_t>(off) * kTileK * 2;
                for (int kb = 0; kb < kblocks; kb += slices) {
                    if (!wait_or_abort<CG>(&c.empty[s], ph ^ 1, c, a)) {
                        ok = false;
                        break;
                    }
                    uint8_t *sa = ring + s * stage_bytes;
                    if constexpr (CG == 1) {
                        uint64_t *bar = &c.full[s];
                        const int n_sl = min(slices, kblocks - kb);
                        mbar_expect_tx(bar, n_sl * (h_bytes + n_cols * kTileK * 2));
                        uint8_t *sb = sa + slices * a_bytes;
                        int j = 0;
                        do {
                            tma_load_2d(sa, &tm_h, (kb + j) * kTileK, row0, bar);
                            if (a.w_packed) {
                                bulk_load(sb, blk, head * (kTileK * 2), bar);
                                if (head < n_cols)
                                    bulk_load(sb + head * (kTileK * 2), blk + next_blk, (n_cols - head) * (kTileK * 2), bar);
                                blk += kBBytes;
                            } else if (n_cols == kTileN) {
                                tma_load_2d(sb, &tm_w, (kb + j) * kTileK, col0, bar);
                            } else {  // (tm_w_half: kCopyRows a copy)
                                for (int g = 0; g < n_cols; g += kCopyRows)
                                    tma_load_2d(sb + g * (kTileK * 2), &tm_w_half, (kb + j) * kTileK, col0 + g, bar);
                            }
                            sa += a_bytes;
                            sb += n_cols * (kTileK * 2);
                        } while (++j < n_sl);
                    } else {
                        // both CTAs' copies complete on the leader's barrier, which
                        // expects the bytes of both
                        const uint32_t bar = leader_addr(&c.full[s]);
                        if (rank == 0)
                            mbar_expect_tx(&c.full[s], Sh::slices * (h_bytes * pair_tiles + n_cols * kTileK * 2));
                        // one copy per operand for all slices of the stage (past the last
                        // slice of d it brings values that no MMA reads)
                        if (has_rows) tma_load_3d_pair(sa, &tm_h, 0, row0, kb, bar);
                        const int tok = col0 + rank * (n_cols / 2);  // this CTA's half of the tile's tokens
                        const CUtensorMap *map = n_cols == kTileN ? &tm_w : &tm_w_half;
                        uint8_t *sb = sa + Sh::slices * kABytes;
                        // packed: 16 rows of the swizzled image per 2 KB line of the map
                        if (a.w_packed)
                            tma_load_3d_pair(sb, map, 0, tok % kTileN / kLineRows, tok / kTileN * kblocks + kb, bar);
                        else
                            tma_load_3d_pair(sb, map, 0, tok, kb, bar);
                    }
                    ++it;
                    if (++s == n_stages) {
                        s = 0;
                        ph ^= 1;
                    }
                }
            }
            // every copy issued lands before the CTA leaves, whichever role
            // aborted (in a normal run these phases have long completed). The
            // second CTA of a pair sees it by its stages being consumed.
            const uint32_t ring_len = n_stages;
            for (uint32_t j = it > ring_len ? it - ring_len : 0; j < it; ++j)
                wait_drain<CG>(rank == 0 ? &c.full[j % ring_len] : &c.empty[j % ring_len], (j / ring_len) & 1);
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {  // --------------------------- MMA issuer
            uint32_t ph = 0;
            int s = 0;
            bool ok = true;
            const uint64_t ring_desc = umma::smem_desc_kmajor_sw128(saddr(ring));
            for (int t = 0; t < n_tiles && ok; ++t) {
                const int buf = t & 1;
                const uint32_t use = static_cast<uint32_t>(t >> 1);
                if (!wait_or_abort<CG>(&c.acc_empty[buf], (use & 1) ^ 1, c, a)) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem + static_cast<uint32_t>(buf * kTileN);
                const int n_cols = static_cast<int>(min(static_cast<int64_t>(kTileN), col_end - (col_begin + t * kTileN)));
                const uint32_t idesc = umma::instr_desc_bf16(kTileM * CG, n_cols);
                const int slices = FLEX ? tile_slices(n_cols, a_bytes, stage_bytes) : Sh::slices;
                const uint32_t a_step = a_bytes / 16, b_step = n_cols / CG * kTileK * 2 / 16, b_off = slices * a_step;
                for (int kb = 0; kb < kblocks; kb += slices) {
                    if (!wait_or_abort<CG>(&c.full[s], ph, c, a)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    // (a descriptor's low bits are the address in 16-byte units)
                    uint64_t ad = ring_desc + static_cast<uint32_t>(s * stage_bytes) / 16;
                    uint64_t bd = ad + b_off;
                    const auto slice_mmas = [&](bool first) {
#pragma unroll
                        for (int k = 0; k < kTileK / kMmaK; ++k)
                            mma_bf16<CG>(d_tmem, umma::advance_k16(ad, k), umma::advance_k16(bd, k), idesc,
                                         k != 0 || !first ? 1u : 0u);
                        ad += a_step;
                        bd += b_step;
                    };
                    slice_mmas(kb == 0);
                    if constexpr (FLEX)
                        for (int j = 1; j < slices && kb + j < kblocks; ++j) slice_mmas(false);
                    else if (Sh::slices > 1 && kb + 1 < kblocks) slice_mmas(false);
                    mma_commit<CG>(&c.empty[s]);  // the stage is free once these MMAs have read it
                    if (++s == n_stages) {
                        s = 0;
                        ph ^= 1;
                    }
                }
                if (ok) mma_commit<CG>(&c.acc_full[buf]);
            }
            // every MMA issued has completed before TMEM is freed
            mma_commit<CG>(&c.mma_done);
            wait_drain<CG>(&c.mma_done, 0);
        }
        __syncwarp();
    } else {  // ---------------------------------------------------- epilogue
        const int q = warp & 3;  // this warp's quarter of the TMEM lanes
        const int row = row0 + q * 32 + lane;
        const bool live = row < a.n_rows;
        RowState<KMAX> st;
        st.B = -INFINITY;
        st.s = 0.f;
        st.t = 0.f;
        st.mx = -INFINITY;
        st.amx = INT_MAX;
#pragma unroll
        for (int i = 0; i < (KMAX > 0 ? KMAX : 1); ++i) {
            st.lv[i] = -INFINITY;
            st.li[i] = INT_MAX;
        }
        float floor_thr = -INFINITY;  // logits up to this never enter the list
        float *pick = reinterpret_cast<float *>(ring + Sh::ring_bytes) + (warp - 2) * 32 + lane;
        bool ok = true;
        for (int t = 0; t < n_tiles; ++t) {
            const int buf = t & 1;
            const uint32_t use = static_cast<uint32_t>(t >> 1);
            if (!warp_wait_or_abort<CG>(&c.acc_full[buf], use & 1, c, a)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t tbase = tmem + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(buf * kTileN);
            const int col0 = col_begin + t * kTileN;
            const int ncol = static_cast<int>(min(static_cast<int64_t>(kTileN), min(col_end, a.vocab) - col0));
            const int n_ch = (ncol + 31) / 32;
            // pass 1: the tile's maximum and its lowest column. In the first tile
            // of a list, the maxima of its groups of columns bound the row's k-th
            // logit from below (k groups each hold one at least that large), so
            // that few columns enter the list (see pass 2).
            constexpr int kGroup = 8, kGroups = kTileN / kGroup;  // 32: at least KMAX, and more bound closer
            float tm = -INFINITY;
            int ta = INT_MAX;
            for (int ch = 0; ch < n_ch; ++ch) {
                float v[32];
                tmem_ld32(tbase + ch * 32, v);
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int cc = ch * 32 + i;
                    if (cc < ncol && v[i] > tm) {
                        tm = v[i];
                        ta = col0 + cc;
                    }
                }
                if (KMAX > 0 && t == 0) {
#pragma unroll
                    for (int g = 0; g < 32 / kGroup; ++g) {
                        float gm = -INFINITY;
#pragma unroll
                        for (int i = g * kGroup; i < (g + 1) * kGroup; ++i)
                            if (ch * 32 + i < ncol) gm = fmaxf(gm, v[i]);
                        pick[(ch * (32 / kGroup) + g) * (kEpiWarps * 32)] = gm;
                    }
                }
            }
            if (KMAX > 0 && t == 0) {
                float gm[kGroups];
#pragma unroll
                for (int g = 0; g < kGroups; ++g)
                    gm[g] = g < n_ch * (32 / kGroup) ? pick[g * (kEpiWarps * 32)] : -INFINITY;
                sort_desc(gm);
                float kth = -INFINITY;
#pragma unroll
                for (int g = 0; g < kGroups; ++g) kth = fmaxf(kth, g >= a.k - 1 ? gm[g] : -INFINITY);  // (entry k - 1)
                floor_thr = next_below(kth);
            }
            if (tm > st.mx) {
                st.mx = tm;
                st.amx = ta;
            }
            // the base-2 reference follows the running maximum
            const float nb = fmaxf(st.B, tm * kLog2e);
            if (nb > st.B) {
                if (st.s > 0.f) {
                    const float dl = st.B - nb;
                    const float f = ex2(dl);
                    st.t = f * fmaf(dl, st.s, st.t);
                    st.s *= f;
                }
                st.B = nb;
            }
            // pass 2: the sums, the top-k list, and (testing only) the logits
            for (int ch = 0; ch < n_ch; ++ch) {
                float v[32];
                tmem_ld32(tbase + ch * 32, v);
                const int nv = min(32, ncol - ch * 32);  // valid columns of this chunk (32 but in the last tile)
                if (nv < 32) {
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (i >= nv) v[i] = -INFINITY;  // contributes 2^-inf = 0 and never enters the list
                }
                float ps[2] = {0.f, 0.f}, pt[2] = {0.f, 0.f};
                uint32_t cand = 0;  // columns that pass the list's last entry
                const float thr = KMAX > 0 ? fmaxf(st.lv[KMAX > 0 ? KMAX - 1 : 0], floor_thr) : INFINITY;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const float u = fmaf(v[i], kLog2e, -st.B);
                    const float e = ex2(u);
                    ps[i & 1] += e;
                    pt[i & 1] = fmaf(e > 0.f ? u : 0.f, e, pt[i & 1]);
                    if (KMAX > 0 && v[i] > thr) cand |= 1u << i;
                }
                st.s += ps[0] + ps[1];
                st.t += pt[0] + pt[1];
                // the few candidates, one copy of the insertion (the list only
                // grows stricter, so each is checked again against it), their
                // logits picked by index from shared memory
                if (!live) cand = 0;  // (rows past the last: equal logits, all of them candidates)
                if (KMAX > 0 && __any_sync(kFull, cand != 0)) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) pick[i * (kEpiWarps * 32)] = v[i];
#pragma unroll 1
                    while (cand) {
                        const int i = __ffs(cand) - 1;
                        cand &= cand - 1;
                        const float x = pick[i * (kEpiWarps * 32)];
                        if (x > st.lv[KMAX > 0 ? KMAX - 1 : 0]) list_insert<KMAX>(st, x, col0 + ch * 32 + i);
                    }
                    __syncwarp();
                }
                if (a.logits_out && live) {
                    float *dst = a.logits_out + static_cast<int64_t>(row) * a.vocab + col0 + ch * 32;
                    for (int i = 0; i < 32; ++i)
                        if (ch * 32 + i < ncol) dst[i] = v[i];
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if constexpr (CG == 1) mbar_arrive(&c.acc_empty[buf]);
                else mbar_arrive_cluster(leader_addr(&c.acc_empty[buf]));
            }
        }
        if (ok && live) {
            const int64_t slot = static_cast<int64_t>(row) * a.splits + split;
            LmPartial p;
            p.B = st.B;
            p.s = st.s;
            p.t = st.t;
            p.mx = st.mx;
            p.amax = st.amx;
            p.pad[0] = p.pad[1] = p.pad[2] = 0;
            a.part[slot] = p;
            if (KMAX > 0) {
                float2 *l = a.lists + slot * KMAX;
#pragma unroll
                for (int i = 0; i < (KMAX > 0 ? KMAX : 1); ++i) l[i] = make_float2(st.lv[i], __int_as_float(st.li[i]));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (CG == 2) {
        // neither CTA leaves while the other's copies, MMAs or arrivals may reach
        // it: the last commit arrives in both
        if (rank != 0 && threadIdx.x == 0 && !c.skip) wait_drain<CG>(&c.mma_done, 0);
        __syncwarp();
        cluster_sync();
        __syncwarp();
    }
    tc_fence_after();
    if (warp == 1) tmem_dealloc<CG>(tmem, kTmemCols);
}

// ---------------------------------------------------------------- merge
// One warp per row: the splits' records give zmax, lse, H, P^max and argmax; in
// top-k mode the splits' sorted lists give T_i, mu and the truncated entropy
// (Eq. 3). Lane l owns splits l, l + 32, ...
//
// Latency bound: a few hundred bytes to 20 KB per row, one chain of dependent
// round trips, so the chain is kept to two. The records come in one round, and
// bound the row's k-th logit from below: of the splits' (t + 1)-th logits,
// t = (k - 1) / splits, the m-th largest with m (t + 1) >= k is reached by m
// lists of t + 1 logits each. Only lists whose largest logit reaches the bound
// (about k of them) are read, all their entries at once, and the entries that
// reach it are ranked by shuffles. V 126,464, k = 10, LM head and merge: 32 rows
// (152 splits) 213.6 -> 184.6 us, 256 rows (76 splits) 258.4 -> 244.8, against a
// merge that took one round of loads and shuffles per rank (19 and 13 us alone).
constexpr int kMergeCand = 256;   // candidates buffered per row before they are ranked
constexpr int kMergeLoads = 4;    // list loads a lane keeps in flight

// Ranks the n buffered candidates into the warp's list, 32 at a time.
__device__ __forceinline__ void rank_candidates(float &tv, int &ti, const float2 *buf, int n, int k, int lane,
                                                float2 *scratch, bool &empty) {
    for (int b = 0; b < n; b += kCandBatch) {
        const float2 e = b + lane < n ? buf[b + lane] : make_float2(-INFINITY, __int_as_float(INT_MAX));
        if (empty) warp_rank_into_list(tv, ti, e.x, __float_as_int(e.y), k, lane, scratch);
        else warp_merge_batch(tv, ti, e.x, __float_as_int(e.y), k, lane);
        empty = false;
    }
    __syncwarp();
}

template <int KMAX>
__global__ void __launch_bounds__(kMergeThreads) lmhead_merge_kernel(const LmArgs a) {
    constexpr int kPerLane = kMaxSplits / 32;
    constexpr int kWarps = kMergeThreads / 32;
    __shared__ int16_t hit_all[KMAX > 0 ? kWarps : 1][kMaxSplits];
    __shared__ float2 cand_all[KMAX > 0 ? kWarps : 1][kMergeCand + 64];
    __shared__ float2 scratch_all[KMAX > 0 ? kWarps : 1][kCandBatch];
    pdl_wait();
    pdl_launch_next();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    if (__ldcg(a.health) != 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) flag_error(a.err, RPS_DEVERR_WORKSPACE);
        return;
    }
    const int warps = gridDim.x * kWarps;
    for (int row = blockIdx.x * kWarps + wib; row < a.n_rows; row += warps) {
        const LmPartial *pr = a.part + static_cast<int64_t>(row) * a.splits;
        const float2 *ls = a.lists + static_cast<int64_t>(row) * a.splits * KMAX;
        const int t = KMAX > 0 && a.k > 0 ? (a.k - 1) / a.splits : 0;  // depth of the bound (below KMAX: k <= KMAX)
        float4 p[kPerLane];   // B, s, t, largest logit
        int pam[kPerLane];
        float deep[kPerLane]; // the (t + 1)-th logit
#pragma unroll
        for (int m = 0; m < kPerLane; ++m) {
            const int j = lane + 32 * m;
            p[m] = make_float4(-INFINITY, 0.f, 0.f, -INFINITY);
            pam[m] = INT_MAX;
            deep[m] = -INFINITY;
            if (j < a.splits) {
                p[m] = *reinterpret_cast<const float4 *>(pr + j);
                pam[m] = pr[j].amax;
                if (KMAX > 0 && t > 0) deep[m] = ls[j * KMAX + t].x;
            }
        }
        // the largest reference of the row's live records
        float M = -INFINITY, mx = -INFINITY;
        int am = INT_MAX;
        bool nan = false;
#pragma unroll
        for (int m = 0; m < kPerLane; ++m) {
            if (p[m].y > 0.f) M = fmaxf(M, p[m].x);
            if (p[m].y != p[m].y) nan = true;
            if (p[m].w > mx || (p[m].w == mx && pam[m] < am)) {
                mx = p[m].w;
                am = pam[m];
            }
        }
        M = warp_max(M);
        float S = 0.f, T = 0.f;
#pragma unroll
        for (int m = 0; m < kPerLane; ++m) {
            if (p[m].y > 0.f) {
                const float dl = p[m].x - M;
                const float f = ex2(dl);
                S = fmaf(f, p[m].y, S);
                T = fmaf(f, fmaf(dl, p[m].y, p[m].z), T);
            }
        }
        S = warp_sum(S);
        T = warp_sum(T);
        nan = __any_sync(kFull, nan);
        const float rmx = warp_max(mx);
        const int ram = warp_min_int(mx == rmx ? am : INT_MAX);
        const bool ok = !nan && rmx > -INFINITY && S > 0.f && !(T != T) && ram != INT_MAX;
        float lse = NAN, H = NAN, pmax = NAN, lnS = NAN, invS = NAN;
        if (ok) {
            lnS = logf(S);
            invS = 1.f / S;
            lse = fmaf(M, kLn2, lnS);
            H = fmaxf(lnS - kLn2 * T * invS, 0.f);
            pmax = ex2(fmaf(rmx, kLog2e, -M)) * invS;
        }
        if (lane == 0) {
            a.zmax[row] = ok ? rmx : NAN;
            a.lse[row] = lse;
            a.H[row] = H;
            a.pmax[row] = pmax;
            a.argmax[row] = ok ? ram : -1;
            if (!ok) flag_error(a.err, RPS_DEVERR_NONFINITE);
        }
        if constexpr (KMAX > 0) {  // (the statistics-only form has no lists)
            if (a.k == 0) continue;
            int16_t *hit = hit_all[wib];
            float2 *cand = cand_all[wib];
            float2 *scratch = scratch_all[wib];
            // the bound: the m-th largest of the lanes' largest (t + 1)-th logits
            float dmax = -INFINITY;
#pragma unroll
            for (int m = 0; m < kPerLane; ++m) dmax = fmaxf(dmax, t > 0 ? deep[m] : p[m].w);
            const float theta = warp_kth_largest(dmax, (a.k + t) / (t + 1), lane);
            int n_hit = 0;
#pragma unroll
            for (int m = 0; m < kPerLane; ++m) {
                const bool h = lane + 32 * m < a.splits && p[m].w >= theta;
                const unsigned hm = __ballot_sync(kFull, h);
                if (h) hit[n_hit + __popc(hm & ((1u << lane) - 1u))] = static_cast<int16_t>(lane + 32 * m);
                n_hit += __popc(hm);
            }
            __syncwarp();
            float tv = -INFINITY;
            int ti = INT_MAX;
            bool empty = true;
            int pending = 0;
            const int items = n_hit * (KMAX / 2);  // two entries each
            for (int i0 = 0; i0 < items; i0 += 32 * kMergeLoads) {
                float4 e[kMergeLoads];
#pragma unroll
                for (int u = 0; u < kMergeLoads; ++u) {
                    const int i = i0 + u * 32 + lane;
                    e[u] = make_float4(-INFINITY, __int_as_float(INT_MAX), -INFINITY, __int_as_float(INT_MAX));
                    if (i < items)
                        e[u] = reinterpret_cast<const float4 *>(ls + hit[i / (KMAX / 2)] * KMAX)[i % (KMAX / 2)];
                }
#pragma unroll
                for (int u = 0; u < kMergeLoads; ++u) {
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        const float v = half ? e[u].z : e[u].x;
                        const float id = half ? e[u].w : e[u].y;
                        const bool in = v >= theta && __float_as_int(id) != INT_MAX;
                        const unsigned im = __ballot_sync(kFull, in);
                        if (in) cand[pending + __popc(im & ((1u << lane) - 1u))] = make_float2(v, id);
                        pending += __popc(im);
                    }
                    __syncwarp();
                    if (pending >= kMergeCand) {
                        rank_candidates(tv, ti, cand, pending, a.k, lane, scratch, empty);
                        pending = 0;
                    }
                }
            }
            rank_candidates(tv, ti, cand, pending, a.k, lane, scratch, empty);
            // mu and the truncated entropy against the row's reference, as the streaming kernel forms them
            float pr_v = 0.f, h = 0.f;
            if (ok && lane < a.k && ti != INT_MAX) {
                const float u = fmaf(tv, kLog2e, -M);
                pr_v = ex2(u) * invS;
                if (pr_v > 0.f) h = -pr_v * (u * kLn2 - lnS);
            }
            const float mu = warp_sum(pr_v), ht = warp_sum(h);
            if (lane == 0) {
                a.mu[row] = ok ? mu : NAN;
                a.htrunc[row] = ok ? ht : NAN;
            }
            if (lane < a.k) {
                a.topk_idx[static_cast<int64_t>(row) * a.k + lane] = ti == INT_MAX ? -1 : ti;
                a.topk_logit[static_cast<int64_t>(row) * a.k + lane] = ti == INT_MAX ? NAN : tv;
            }
        }
    }
}

// ---------------------------------------------------------------- packed unembedding
// The packed layout holds, for vocabulary tile vt and d slice kb, the 256 x 64
// block W[256 vt + n][64 kb + k] as the 32 KB image a TMA load with 128-byte
// swizzle would leave in shared memory: row n at byte 128 n, its 16-byte
// chunk c at chunk position c ^ (n % 8). Rows past the vocabulary are zero.
// One thread per 16-byte chunk of the packed tensor.
__global__ void pack_unembed_kernel(const uint4 *w, int64_t vocab, int32_t d, int64_t stride_elems, uint4 *out,
                                    int64_t n_chunks) {
    const int kblocks = d / kTileK;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n_chunks;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t blk = i / (kBBytes / 16);
        const int in = static_cast<int>(i - blk * (kBBytes / 16));  // chunk within the block image
        const int n = in >> 3, pos = in & 7, c = pos ^ (n & 7);     // row, stored position, source chunk
        const int64_t vt = blk / kblocks;
        const int kb = static_cast<int>(blk - vt * kblocks);
        const int64_t row = vt * kTileN + n;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (row < vocab) v = w[(row * stride_elems + static_cast<int64_t>(kb) * kTileK) / 8 + c];
        out[i] = v;
    }
}

// ---------------------------------------------------------------- host
struct LmDevice {
    bool ready = false;
    int sm_count = 0;
    int pairs = 0;  // CTA pairs resident at once
};

// Tensor maps of one launch: hidden rows, unembedding tiles, half tiles (pairs).
struct LmMaps {
    CUtensorMap h, w, w_half;
};

template <int CG>
void lm_config(cudaLaunchConfig_t *cfg, cudaLaunchAttribute (&attr)[2], dim3 grid, cudaStream_t stream) {
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = grid;
    cfg->blockDim = dim3(kThreads);
    cfg->dynamicSmemBytes = Shape<CG>::smem_bytes;
    cfg->stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = CG;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = CG == 1 ? 1 : 2;
}

template <int KMAX, int CG, bool FLEX>
cudaError_t launch_lm(int grid, cudaStream_t stream, const LmMaps &m, const LmArgs &a) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    lm_config<CG>(&cfg, attr, dim3(grid), stream);
    return cudaLaunchKernelEx(&cfg, lmhead_kernel<KMAX, CG, FLEX>, m.h, m.w, m.w_half, a);
}

template <int CG, bool FLEX>
cudaError_t launch_lm_k(int grid, cudaStream_t stream, const LmMaps &m, const LmArgs &a) {
    return a.kmax == 0    ? launch_lm<0, CG, FLEX>(grid, stream, m, a)
           : a.kmax == 12 ? launch_lm<12, CG, FLEX>(grid, stream, m, a)
           : a.kmax == 16 ? launch_lm<16, CG, FLEX>(grid, stream, m, a)
           : a.kmax == 20 ? launch_lm<20, CG, FLEX>(grid, stream, m, a)
                          : launch_lm<32, CG, FLEX>(grid, stream, m, a);
}

template <int KMAX>
cudaError_t set_smem() {
    cudaError_t e = cudaFuncSetAttribute(lmhead_kernel<KMAX, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         Shape<1>::smem_bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(lmhead_kernel<KMAX, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 Shape<1>::smem_bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(lmhead_kernel<KMAX, 2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 Shape<2>::smem_bytes);
    return e;
}

// Resident CTA pairs of the widest form (the others need no more).
cudaError_t count_pairs(int *pairs) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    lm_config<2>(&cfg, attr, dim3(2), nullptr);
    cfg.attrs = attr + 1;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(pairs, lmhead_kernel<32, 2, false>, &cfg);
}
constexpr int kMaxDevices = 64;
std::mutex g_lm_mutex;
LmDevice g_lm_devices[kMaxDevices];
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

rps_status lm_device(LmDevice *out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return RPS_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_lm_mutex);
    if (!g_encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return RPS_ERR_CUDA;
        g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    LmDevice &d = g_lm_devices[dev];
    if (!d.ready) {
        if (cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return RPS_ERR_CUDA;
        if (set_smem<0>() != cudaSuccess || set_smem<12>() != cudaSuccess || set_smem<16>() != cudaSuccess ||
            set_smem<20>() != cudaSuccess || set_smem<32>() != cudaSuccess)
            return RPS_ERR_CUDA;
        int counted = 0;
        const cudaError_t e = count_pairs(&counted);
        if (e != cudaSuccess) cudaGetLastError();  // (not the next call's error)
        d.pairs = lm_pairs(e == cudaSuccess, counted);
        d.ready = true;
    }
    *out = d;
    return RPS_OK;
}

rps_status encode(CUtensorMap *m, CUtensorMapDataType type, int rank, const void *base, const cuuint64_t *dims,
                  const cuuint64_t *strides, const cuuint32_t *box, bool swizzle) {
    const cuuint32_t es[3] = {1, 1, 1};
    const CUresult r = g_encode(m, type, rank, const_cast<void *>(base), dims, strides, box, es,
                                CU_TENSOR_MAP_INTERLEAVE_NONE,
                                swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? RPS_OK : RPS_ERR_CUDA;
}

// 2-D bf16 tensor map over rows x d (d contiguous), box of 64 x box_rows, 128-byte swizzle.
rps_status make_map(CUtensorMap *m, const void *base, int64_t rows, int32_t d, int64_t stride_elems, int box_rows) {
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(d), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(stride_elems) * 2};
    const cuuint32_t box[2] = {static_cast<cuuint32_t>(kTileK), static_cast<cuuint32_t>(box_rows)};
    return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, true);
}

// The same rows x d as 64 x rows x (d / 64): a box holds `box_rows` rows of a
// stage's slices, slice after slice, 128-byte swizzle.
rps_status make_slice_map(CUtensorMap *m, const void *base, int64_t rows, int32_t d, int64_t stride_elems,
                          int box_rows) {
    const cuuint64_t dims[3] = {kTileK, static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(d / kTileK)};
    const cuuint64_t strides[2] = {static_cast<cuuint64_t>(stride_elems) * 2, kTileK * 2};
    const cuuint32_t box[3] = {kTileK, static_cast<cuuint32_t>(box_rows), Shape<2>::slices};
    return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, true);
}

// The packed unembedding as 2 KB lines (16 of its 128-byte rows, 256 64-bit
// words) x 16 lines x blocks, no swizzle (the blocks hold the swizzled image).
rps_status make_packed_map(CUtensorMap *m, const void *base, int64_t blocks, int box_rows) {
    const cuuint64_t dims[3] = {256, kTileN / kLineRows, static_cast<cuuint64_t>(blocks)};
    const cuuint64_t strides[2] = {2048, kBBytes};
    const cuuint32_t box[3] = {256, static_cast<cuuint32_t>(box_rows / kLineRows), Shape<2>::slices};
    return encode(m, CU_TENSOR_MAP_DATA_TYPE_INT64, 3, base, dims, strides, box, false);
}

// Entries of the splits' lists. An insertion costs about as many instructions as
// six times the length, and a CTA with one or two tiles little else: 100 rows of V
// 32,000, d 1,024 at k = 20: 34.7 us with 20 entries, 41.5 with 32; k = 10: 12 for 16.
int list_len(int32_t k) { return k == 0 ? 0 : k <= 12 ? 12 : k <= 16 ? 16 : k <= 20 ? 20 : 32; }

struct LmLayout {
    size_t health, part, lists, total;
};

// Splits the workspace is laid out for. One row tile takes every SM, also with
// fewer vocabulary tiles than SMs.
int64_t splits_cap(int32_t n_rows, int64_t vocab) {
    const int tokens = n_rows <= kTileM ? kQuarter : kTileN;
    return std::min<int64_t>((vocab + tokens - 1) / tokens, kMaxSplits);
}

LmLayout lm_layout(int32_t n_rows, int64_t splits, int32_t k) {
    const size_t cap = static_cast<size_t>(n_rows) * static_cast<size_t>(splits);
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    LmLayout l;
    l.health = 0;
    l.part = 256;
    l.lists = l.part + up(cap * sizeof(LmPartial));
    l.total = l.lists + up(cap * static_cast<size_t>(list_len(k)) * sizeof(float2));
    return l;
}

}  // namespace
}  // namespace rps

using namespace rps;

extern "C" {

size_t rps_lmhead_packed_bytes(int64_t vocab, int32_t d) {
    if (vocab < 1 || vocab > INT32_MAX || d < kTileK || d % kTileK) return 0;
    return static_cast<size_t>((vocab + kTileN - 1) / kTileN) * (d / kTileK) * kBBytes;
}

rps_status rps_lmhead_pack_unembed(const void *unembed, int64_t vocab, int32_t d, int64_t stride, void *packed,
                                   size_t packed_bytes, rps_stream_t stream) {
    if (!unembed || !packed || reinterpret_cast<uintptr_t>(unembed) % 16 || reinterpret_cast<uintptr_t>(packed) % 16)
        return RPS_ERR_INVALID_ARG;
    const size_t need = rps_lmhead_packed_bytes(vocab, d);
    if (need == 0 || stride < d || stride % 8 || packed_bytes < need) return RPS_ERR_INVALID_ARG;
    const int64_t n_chunks = static_cast<int64_t>(need / 16);
    const int grid = static_cast<int>(std::min<int64_t>((n_chunks + 255) / 256, 152 * 16));
    pack_unembed_kernel<<<grid, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        static_cast<const uint4 *>(unembed), vocab, d, stride, static_cast<uint4 *>(packed), n_chunks);
    return cudaGetLastError() == cudaSuccess ? RPS_OK : RPS_ERR_CUDA;
}

size_t rps_lmhead_workspace_bytes(int32_t n_rows, int64_t vocab, int32_t k_max) {
    if (n_rows < 1 || vocab < 1 || vocab > INT32_MAX || k_max < 0 || k_max > RPS_MAX_K) return 0;
    // one row tile may need more than a few rows of the next: a workspace queried for
    // the largest row count has to do for every smaller one
    size_t need = lm_layout(n_rows, splits_cap(n_rows, vocab), k_max).total;
    if (n_rows > kTileM) need = std::max(need, lm_layout(kTileM, splits_cap(kTileM, vocab), k_max).total);
    return need;
}

rps_status rps_lmhead_row_stats(const rps_lmhead *lm, const rps_params *prm, const rps_row_stats *out,
                                float *d_logits_out, void *d_ws, size_t ws_bytes, rps_stream_t stream) {
    if (!lm || !lm->hidden || !lm->unembed || !out) return RPS_ERR_INVALID_ARG;
    if (lm->n_rows < 1 || lm->vocab < 1 || lm->vocab > INT32_MAX || lm->d < kTileK || lm->d % kTileK != 0)
        return RPS_ERR_INVALID_ARG;
    if (lm->hidden_stride < lm->d || lm->hidden_stride % 8) return RPS_ERR_INVALID_ARG;
    if (!lm->unembed_packed && (lm->unembed_stride < lm->d || lm->unembed_stride % 8)) return RPS_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(lm->hidden) % 16 || reinterpret_cast<uintptr_t>(lm->unembed) % 16)
        return RPS_ERR_INVALID_ARG;
    if (!out->zmax || !out->lse || !out->H || !out->pmax || !out->argmax) return RPS_ERR_INVALID_ARG;
    int32_t k = 0;
    if (out->topk_idx) {
        if (!prm || prm->k_max < 1) return RPS_ERR_INVALID_ARG;
        if (prm->k_max > RPS_MAX_K) return RPS_ERR_UNSUPPORTED;
        if (prm->k_max > lm->vocab || !out->topk_logit || !out->mu || !out->htrunc) return RPS_ERR_INVALID_ARG;
        k = prm->k_max;
    }
    // The least workspace has room for a split per vocabulary tile; with less than
    // the queried size there are no more splits than that.
    const int n_vt = static_cast<int>((lm->vocab + kTileN - 1) / kTileN);
    int64_t cap = splits_cap(lm->n_rows, lm->vocab);
    if (ws_bytes < lm_layout(lm->n_rows, cap, k).total) cap = std::min(n_vt, kMaxSplits);
    const LmLayout w = lm_layout(lm->n_rows, cap, k);
    if (!d_ws || ws_bytes < w.total || reinterpret_cast<uintptr_t>(d_ws) % 16) return RPS_ERR_INVALID_ARG;
    LmDevice dev;
    rps_status st = lm_device(&dev);
    if (st != RPS_OK) return st;
    uint32_t *err = device_error_word();
    if (!err) return RPS_ERR_CUDA;

    const int n_rt = (lm->n_rows + kTileM - 1) / kTileM;
    const int kblocks = lm->d / kTileK;
    const int64_t packed_blocks = static_cast<int64_t>(n_vt) * kblocks;
    const LmSplit sp = lm_split(n_rt, lm->vocab, kblocks, cap, dev.sm_count, dev.pairs);
    const bool pair = sp.pair;
    const int units = sp.units, granule = sp.granule, n_gran = sp.n_gran, splits = sp.splits, longest = sp.longest;
    LmMaps maps;
    std::memset(&maps, 0, sizeof maps);
    if (pair) {
        st = make_slice_map(&maps.h, lm->hidden, lm->n_rows, lm->d, lm->hidden_stride, kTileM);  // (n_rows > kTileM)
        for (int half = 0; half < 2 && st == RPS_OK; ++half) {
            CUtensorMap *m = half ? &maps.w_half : &maps.w;
            const int rows = kTileN / 2 >> half;  // one CTA's tokens
            st = lm->unembed_packed ? make_packed_map(m, lm->unembed, packed_blocks, rows)
                                    : make_slice_map(m, lm->unembed, lm->vocab, lm->d, lm->unembed_stride, rows);
        }
        if (st != RPS_OK) return st;
    } else {
        st = make_map(&maps.h, lm->hidden, lm->n_rows, lm->d, lm->hidden_stride, std::min<int32_t>(lm->n_rows, kTileM));
        if (st != RPS_OK) return st;
        maps.w = maps.w_half = maps.h;  // (single CTAs read the packed unembedding without a tensor map)
        for (int part = 0; part < 2 && !lm->unembed_packed && st == RPS_OK; ++part)
            st = make_map(part ? &maps.w_half : &maps.w, lm->unembed, lm->vocab, lm->d, lm->unembed_stride,
                          part ? kCopyRows : kTileN);
        if (st != RPS_OK) return st;
    }

    LmArgs a;
    std::memset(&a, 0, sizeof a);
    a.n_rows = lm->n_rows;
    a.h_rows = std::min<int32_t>(lm->n_rows, kTileM);
    a.d = lm->d;
    a.splits = splits;
    a.kmax = list_len(k);
    a.k = k;
    a.vocab = lm->vocab;
    char *ws = static_cast<char *>(d_ws);
    a.health = reinterpret_cast<uint32_t *>(ws + w.health);
    a.part = reinterpret_cast<LmPartial *>(ws + w.part);
    a.lists = reinterpret_cast<float2 *>(ws + w.lists);
    a.logits_out = d_logits_out;
    a.w_packed = lm->unembed_packed ? static_cast<const uint8_t *>(lm->unembed) : nullptr;
    a.err = err;
    a.wait_ns = ring_wait_limit_ns();
    a.zmax = out->zmax;
    a.lse = out->lse;
    a.H = out->H;
    a.pmax = out->pmax;
    a.argmax = out->argmax;
    a.mu = out->mu;
    a.htrunc = out->htrunc;
    a.topk_idx = out->topk_idx;
    a.topk_logit = out->topk_logit;

    const cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    a.granule = granule;
    a.n_gran = n_gran;
    // A single CTA's ring by its rows (FLEX), where that gives a fifth stage or
    // several slices in the last tile's stages; otherwise its code only costs (607
    // rows of V 15,010, d 2,432: 38.2 us without, 39.6 with).
    const int64_t range = static_cast<int64_t>(longest) * granule;  // of the longest split
    const int a_bytes = slice_rows_bytes(a.h_rows), last_cols = static_cast<int>((range - 1) % kTileN) + 1;
    a.stage_bytes = range < kTileN ? Shape<1>::stage_bytes : a_bytes + kBBytes;
    a.stages = std::min(kMaxStages, Shape<1>::ring_bytes / a.stage_bytes);
    const bool flex = a.stages > Shape<1>::stages || tile_slices(last_cols, a_bytes, a.stage_bytes) > 1;
    cudaError_t e = pair   ? launch_lm_k<2, false>(units * splits * 2, s, maps, a)
                    : flex ? launch_lm_k<1, true>(units * splits, s, maps, a)
                           : launch_lm_k<1, false>(units * splits, s, maps, a);
    if (e != cudaSuccess) return RPS_ERR_CUDA;
    const dim3 mgrid(std::min((lm->n_rows + kMergeThreads / 32 - 1) / (kMergeThreads / 32), dev.sm_count * 8));
    if (a.kmax == 0) e = launch_pdl(lmhead_merge_kernel<0>, mgrid, dim3(kMergeThreads), 0, s, a);
    else if (a.kmax == 12) e = launch_pdl(lmhead_merge_kernel<12>, mgrid, dim3(kMergeThreads), 0, s, a);
    else if (a.kmax == 16) e = launch_pdl(lmhead_merge_kernel<16>, mgrid, dim3(kMergeThreads), 0, s, a);
    else if (a.kmax == 20) e = launch_pdl(lmhead_merge_kernel<20>, mgrid, dim3(kMergeThreads), 0, s, a);
    else e = launch_pdl(lmhead_merge_kernel<32>, mgrid, dim3(kMergeThreads), 0, s, a);
    return e == cudaSuccess ? RPS_OK : RPS_ERR_CUDA;
}

}  // extern "C"
