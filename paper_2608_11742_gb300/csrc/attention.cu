// attention.cu -- branch-isolating attention of the packed lookahead forward
// pass (rps_packed_attention_fwd; Sec. 3.1 "Lookahead scoring", Fig. 2 right).
//
// The lookahead pass scores every candidate branch of a step in one forward
// pass over a packed sequence [context | branch 0 | branch 1 | ... ] (branch 0
// is the anchor: the normal sequence's own generation region). A branch's
// queries attend to the context and to their own branch, the context's
// queries to the normal sequence (context and branch 0). The mask is
// block-structured, so no mask is ever formed: a query tile walks exactly the
// key tiles of its two visible segments, and the last tile of a segment masks
// the keys past its end.
//
// One persistent CTA per SM takes work items (batch, head, 128-query tile);
// branches of at most 64 tokens share a tile, as many as fit, each row masking
// the other branches' keys in the tile's own key tile. The CTA's key tiles are
// numbered through all its items; even and odd ones go to two independent
// halves of the softmax, each with its own S / P buffer, its own running
// maximum and sum and its own output accumulator, merged when the item ends:
//   warp 0      TMA producer of Q (128 x 128, two 64-wide swizzle atoms) and,
//               per key tile, K (128 keys x 128), 128-byte swizzle, two stages;
//   warp 2      TMA producer of V^T (128 dims x 128 keys: V is stored
//               transposed so that both MMA operands are K-major), two stages
//               of their own, so that K runs ahead of V (K is free once S is
//               computed, V only once P V is);
//   warp 1      MMA issuer: S = Q K^T (M 128, N 128, K 128) into TMEM buffer t % 2 and
//               O[t % 2] += P V^T, P read from TMEM, in one thread and in the
//               order PV(t), S(t + 2), PV(t + 1), ...: the tensor pipe runs them in
//               order, so S may overwrite the P just read with no wait, and the
//               commit of S(t + 2) stands for all that PV(t) frees but V. It also
//               allocates and frees TMEM;
//   warps 4-7   softmax of even tiles, warps 8-11 of odd ones: thread = query
//               row, its 128 scores in registers (these warps take registers
//               from the others with setmaxnreg). The base-2 reference m is
//               raised only when a score passes it by more than 8 (then O and
//               the running sum are rescaled in TMEM); P = 2^(s c - m) is written
//               as bf16 over the S it came from. One half's softmax runs while
//               the other's MMAs do.
//   warps 12-15 read-out: at the end of an item the halves' accumulators are
//               weighted by 2^(m_half - m) / l, added and written as bf16, while the
//               softmax goes on with the next item.
// What bounds it: the MMA issue and the issuer's waits, in turn. Of about 2,090 cycles
// of a key tile the issuer spends 1,490 on its 16 instructions of N 128 (1,024 cycles of
// work; back to back, batches of 16 with one commit take 1,230, each further commit
// about 50) and 600 waiting: for the read-out at the items' ends 213, P 136, K 107, V 103,
// Q 41. A half of the softmax waits for S most of the time: it takes 1,330 to 1,540
// cycles, and two run at once. Shared-memory traffic is not the limit: pairs of CTAs
// that share K and V (160 -> 96 KB per tile) took the same time. 8 x 32 heads, context
// 512, 9 branches of 256: 262 -> 248 us; 32 heads, context 328, 9 branches of 32: 20.3 ->
// 13.9 us (against two halves of each row in turn with separate S and P V issuers, and
// a tile per branch).
// Every wait is bounded; a role whose wait runs out flags RPS_DEVERR_TIMEOUT
// and raises the CTA's abort flag, copies and MMAs in flight are drained and
// TMEM is freed before the CTA exits.
#include <cuda.h>  // CUtensorMap and the tensor-map encoder's signature (no link against the driver)
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "rps_internal.cuh"
#include "umma_desc.h"

namespace rps {
namespace {

constexpr int kD = 128;                      // head dimension
constexpr int kBQ = 128;                     // queries per tile (TMEM lanes)
constexpr int kBK = 128;                     // keys per tile
constexpr int kAtom = 64 * 128 * 2;          // one 128-row x 64-column bf16 swizzle atom: 16 KB
constexpr int kQBytes = 2 * kAtom;           // Q tile: two atoms along d
constexpr int kKBytes = 2 * kAtom;           // K tile: two atoms along d
constexpr int kVBytes = 2 * kAtom;           // V^T tile: two atoms along the keys
constexpr int kKvStages = 2;
constexpr int kQBufs = 2;                    // the next item's Q loads while this item runs
constexpr int kHalves = 2;                   // key tile t: softmax half, S / P buffer and O of t % 2
constexpr int kStageBytes = 32 * 128;          // per read-out warp: 32 rows x 64 bf16 of O on their way out
constexpr int kSmemBytes = kQBufs * kQBytes + kKvStages * (kKBytes + kVBytes) + 4 * kStageBytes + 1024;
constexpr int kThreads = 512;                // warps 0 and 2 TMA, 1 MMA, 4-11 softmax, 12-15 read-out
constexpr int kVWarp = 2;
constexpr int kOutWarps = 4;
// Registers per thread after the split: 128 x 56 + 256 x 176 + 128 x 104 = 65,536
// of the 65,536 the block is launched with (512 threads of 128).
constexpr int kCtlRegs = 56;
constexpr int kSoftRegs = 176;
constexpr int kOutRegs = 104;
static_assert(kKvStages == kHalves, "a tile's stages and buffers go by its parity");
static_assert(128 * kCtlRegs + 256 * kSoftRegs + 128 * kOutRegs <= 512 * 128, "the split fits the launch's registers");
constexpr uint32_t kTmemCols = 512;          // S buffers at columns 0 and 128, O at 256 and 384
constexpr uint32_t kOCol = kHalves * kBK;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kRescale = 8.0f;             // base-2 units a score may pass the reference by
constexpr uint64_t kDrainNs = 200ull * 1000 * 1000;

struct AttnArgs {
    int32_t n_bh, n_heads, n_tokens, n_context, n_branch, branch_len;
    int32_t q_tiles_ctx, q_tiles_branch, items;  // query tiles of the context, of one branch; work items
    int32_t group, groups;                       // branches per query tile (1: a branch has its own tiles), tiles or branches
    float c;                                     // scale * log2(e)
    __nv_bfloat16 *out;
    uint32_t *err;
    uint64_t wait_ns;
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
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
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
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(slot)), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// D[tmem] (+)= A[smem] x B[smem]^T. Executed by the whole warp, issued by the one
// lane with `issue` set, so that the warp stays converged.
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate, uint32_t issue) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(issue)
        : "memory");
}
// D[tmem] (+)= A[tmem] x B[smem]^T: the A operand (128 rows x 16 bf16, two per
// 32-bit column, lane = row) read from tensor memory.
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate, uint32_t issue) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(issue)
        : "memory");
}
// 32 columns without waiting (tmem_wait_st before they are handed on).
__device__ __forceinline__ void tmem_st32_u(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]),
        "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]),
        "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr)
                 : "memory");
    return v;
}
__device__ __forceinline__ void mma_commit(uint64_t *bar, uint32_t issue) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(saddr(bar)),
        "r"(issue)
        : "memory");
}
// 32 columns without waiting: the registers are valid only after tmem_wait_dep on them.
__device__ __forceinline__ void tmem_ld32_async(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
// Waits for this thread's outstanding tcgen05.ld; naming the registers as
// operands keeps every later use of them after the wait.
__device__ __forceinline__ void tmem_wait_dep(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                   "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}

// 16 columns without waiting, and the wait that names them.
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_dep(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15])
                 :
                 : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}

// Packed fp32 pairs (one instruction for two lanes of work).
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// ---------------------------------------------------------------- work items
// Item w = (bh, query tile); query tiles: the context's, then each branch's, or
// each group of branches. Its key tiles: the context's, then those of the one
// visible branch, or the group's own tile.
struct Item {
    int bh, q_start, q_len;     // queries [q_start, q_start + q_len) of the packed sequence (q_len <= 128)
    int k_start, k_len;         // keys after the context's
    bool grouped;               // each row sees its own branch's keys among them only
    int n_ctx_tiles, n_tiles;   // key tiles: context tiles first
};

// The CTA's items w = blockIdx.x + n * gridDim.x, walked in order: (bh, index
// within bh) moves on by the grid's quotient and remainder, so the walk needs
// no division per item (one at the start).
struct ItemWalk {
    int per_bh, step_bh, step_t;  // items per (batch, head); gridDim.x = step_bh * per_bh + step_t
    int bh, t;                    // the current item
    float inv_qtb;                // 1 / query tiles per branch
};

__device__ __forceinline__ ItemWalk item_walk(const AttnArgs &a) {
    ItemWalk wk;
    wk.per_bh = a.q_tiles_ctx + a.groups * a.q_tiles_branch;
    wk.bh = static_cast<int>(blockIdx.x) / wk.per_bh;
    wk.t = static_cast<int>(blockIdx.x) - wk.bh * wk.per_bh;
    wk.step_bh = static_cast<int>(gridDim.x) / wk.per_bh;
    wk.step_t = static_cast<int>(gridDim.x) - wk.step_bh * wk.per_bh;
    wk.inv_qtb = 1.f / static_cast<float>(a.q_tiles_branch);
    return wk;
}

__device__ __forceinline__ void item_next(ItemWalk &wk) {
    wk.t += wk.step_t;
    wk.bh += wk.step_bh;
    if (wk.t >= wk.per_bh) {
        wk.t -= wk.per_bh;
        ++wk.bh;
    }
}

// item_of for the walk's current item; the branch index is the float quotient
// moved to the exact floor (it is off by at most one for these sizes; the
// loops make the result exact regardless)
__device__ __forceinline__ Item item_at(const AttnArgs &a, const ItemWalk &wk) {
    Item it;
    it.bh = wk.bh;
    it.grouped = false;
    int t = wk.t;
    if (t < a.q_tiles_ctx) {
        it.q_start = t * kBQ;
        it.q_len = min(kBQ, a.n_context - it.q_start);
        it.k_start = a.n_context;
        it.k_len = a.branch_len;
    } else if (a.group > 1) {
        const int b0 = (t - a.q_tiles_ctx) * a.group;
        it.grouped = true;
        it.q_start = it.k_start = a.n_context + b0 * a.branch_len;
        it.q_len = it.k_len = min(a.group, a.n_branch - b0) * a.branch_len;
    } else {
        t -= a.q_tiles_ctx;
        int b = __float2int_rz(static_cast<float>(t) * wk.inv_qtb);
        while (b > 0 && b * a.q_tiles_branch > t) --b;
        while ((b + 1) * a.q_tiles_branch <= t) ++b;
        const int qt = t - b * a.q_tiles_branch;
        it.k_start = a.n_context + b * a.branch_len;
        it.k_len = a.branch_len;
        it.q_start = it.k_start + qt * kBQ;
        it.q_len = min(kBQ, a.branch_len - qt * kBQ);
    }
    it.n_ctx_tiles = a.q_tiles_ctx;
    it.n_tiles = a.q_tiles_ctx + a.q_tiles_branch;
    return it;
}

// First key and number of valid keys of key tile j of an item.
__device__ __forceinline__ void key_tile(const AttnArgs &a, const Item &it, int j, int &k0, int &valid) {
    if (j < it.n_ctx_tiles) {
        k0 = j * kBK;
        valid = min(kBK, a.n_context - k0);
    } else {
        const int jj = j - it.n_ctx_tiles;
        k0 = it.k_start + jj * kBK;
        valid = min(kBK, it.k_len - jj * kBK);
    }
}

// Moves (item n, key tile j) of the CTA's key-tile sequence one tile on:
// the loops walk the sequence in order, with no division per tile.
__device__ __forceinline__ void next_tile(int &n, int &j, int T) {
    if (++j == T) {
        j = 0;
        ++n;
    }
}

struct Ctl {
    // A commit per tile after S of tile t + 2, which follows the product of tile t in
    // the tensor pipe. s_full[t % 2]: S of tile t is computed and the product of
    // tile t - 2 is done, so K stage t % 2 and Q of the items before t's are free.
    // V stage t % 2 has a commit of its own right after the product (v_empty):
    // its next tile is then on its way while S of tile t + 2 is computed, which
    // is worth more than the 50 cycles of a second commit per tile (the first
    // takes about 200; 8 x 32 heads, context 512, 9 branches of 256: 258 -> 254 us). No wait sees a barrier two phases on: each
    // waits for every phase in turn. (The read-out waits once an item, on a
    // barrier of its own: o_ready.)
    uint64_t q_full[kQBufs], k_full[kKvStages], v_full[kKvStages], v_empty[kKvStages];
    uint64_t s_full[kHalves], p_full[kHalves], o_ready, o_free, mma_done;
    // a half's reference and sum of a row at the end of item n, in slot n % 4: it
    // is written before the half's last P of the item is handed on, read once
    // O is ready, and written again for item n + 4, whose P needs the
    // products of item n + 2 and so the read-out of item n + 1
    float2 ml[4][kHalves][kBQ];
    uint32_t tmem_base;
    int abort_flag;
};

__device__ bool wait_or_abort(uint64_t *bar, uint32_t parity, Ctl &c, const AttnArgs &a) {
    if (a.wait_ns != 0 && mbar_try_wait(bar, parity)) return true;
    const uint64_t start = global_ns();
    while (a.wait_ns != 0) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*reinterpret_cast<volatile int *>(&c.abort_flag)) return false;
        if (global_ns() - start > a.wait_ns) break;
    }
    flag_error(a.err, RPS_DEVERR_TIMEOUT);
    *reinterpret_cast<volatile int *>(&c.abort_flag) = 1;
    return false;
}

// wait_or_abort for every lane of a warp that goes on to warp-wide tcgen05
// instructions: the warp leaves together, on the same answer.
template <typename Ctl_, typename Args_>
__device__ __forceinline__ bool warp_wait_or_abort(uint64_t *bar, uint32_t parity, Ctl_ &c, const Args_ &a) {
    return __all_sync(kFull, wait_or_abort(bar, parity, c, a));
}

__device__ void wait_drain(uint64_t *bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return;
    const uint64_t start = global_ns();
    while (global_ns() - start < kDrainNs)
        if (mbar_try_wait(bar, parity)) return;
}

// Steps of the softmax over 32 of a row's scores: -inf outside keys [lo, hi); the
// running maxima; P as bf16 pairs pk[at..at+15] and the sums.
// (The mask as one word, whose bits become predicates eight at a time: two
// comparisons per score cost a masked tile 600 cycles. 7 x 28 heads, context 88, 10
// branches of 200: 134 -> 112 us; 60 shapes of other sizes: 8 % on average.)
__device__ __forceinline__ uint32_t low_bits(int n) { return n >= 32 ? ~0u : n <= 0 ? 0u : (1u << n) - 1; }
__device__ __forceinline__ void mask_scores(uint32_t (&s)[32], int lo, int hi) {
    const uint32_t keep = low_bits(hi) & ~low_bits(lo);
#pragma unroll
    for (int i = 0; i < 32; ++i)
        if (!(keep >> i & 1u)) s[i] = __float_as_uint(-INFINITY);
}
__device__ __forceinline__ void max_scores(const uint32_t (&s)[32], float (&mx)[8]) {
#pragma unroll
    for (int i = 0; i < 32; ++i) mx[i & 7] = fmaxf(mx[i & 7], __uint_as_float(s[i]));
}
__device__ __forceinline__ void exp_scores(const uint32_t (&s)[32], f2 cc, f2 mm, f2 (&lsum)[4], uint32_t (&pk)[32],
                                           int at) {
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
        const f2 u = fma2(pack2(__uint_as_float(s[i]), __uint_as_float(s[i + 1])), cc, mm);
        float u0, u1;
        unpack2(u, u0, u1);
        const float p0 = ex2(u0), p1 = ex2(u1);
        lsum[(i >> 1) & 3] = add2(lsum[(i >> 1) & 3], pack2(p0, p1));
        pk[at + i / 2] = pack_bf16(p0, p1);
    }
}

// O / l of this thread's row of item n, bf16, to global memory, once the item's
// last product is done (o_ready, one phase per item); then O is released to the
// MMA (o_free). The halves' accumulators are weighted by 2^(m_half - m) / l; one
// that took no tile of the item (one-tile items) is not read.
// The warp's 32 rows go out through its shared-memory stage, 64 columns at a
// time: written a row per thread, read back so that each store instruction
// covers 128 contiguous bytes of 4 rows (a row per thread would touch 32 lines
// per instruction). The 16-byte chunk index is XORed with the row's low three
// bits, so that neither the writes nor the reads put two threads of a
// quarter-warp in one bank group.
__device__ bool read_out(const Item &it, int n, int T, uint32_t tmem, int q, int lane, uint32_t stage, Ctl &c,
                         const AttnArgs &a) {
    if (!warp_wait_or_abort(&c.o_ready, n & 1, c, a)) return false;
    tc_fence_after();
    const int r = q * 32 + lane;
    const bool both = T > 1;
    const int only = n & 1;  // the half of a one-tile item's tile
    const float2 e = c.ml[n & 3][both ? 0 : only][r];
    float w0 = 1.f / e.y, w1 = 0.f;
    if (both) {
        const float2 f = c.ml[n & 3][1][r];
        const float m = fmaxf(e.x, f.x);
        const float x0 = ex2(e.x - m), x1 = ex2(f.x - m);
        const float inv = 1.f / (x0 * e.y + x1 * f.y);
        w0 = x0 * inv;
        w1 = x1 * inv;
    }
    const uint32_t col = tmem + (static_cast<uint32_t>(q * 32) << 16) + kOCol;
    __nv_bfloat16 *dst = a.out + (static_cast<int64_t>(it.bh) * a.n_tokens + it.q_start + q * 32) * kD;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
            uint32_t o0[32], o1[32];
            const uint32_t cc = col + half * 64 + ch * 32;
            tmem_ld32_async(cc + (both ? 0 : only * kBK), o0);
            if (both) {
                tmem_ld32_async(cc + kBK, o1);
                tmem_wait_dep(o0);
                tmem_wait_dep(o1);
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    o0[i] = __float_as_uint(fmaf(__uint_as_float(o1[i]), w1, __uint_as_float(o0[i]) * w0));
            } else {
                tmem_wait_dep(o0);
#pragma unroll
                for (int i = 0; i < 32; ++i) o0[i] = __float_as_uint(__uint_as_float(o0[i]) * w0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                uint32_t pk[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    pk[i] = pack_bf16(__uint_as_float(o0[8 * u + 2 * i]), __uint_as_float(o0[8 * u + 2 * i + 1]));
                st_shared_v4(stage + lane * 128 + (((ch * 4 + u) ^ (lane & 7)) << 4), make_uint4(pk[0], pk[1], pk[2], pk[3]));
            }
        }
        if (half == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&c.o_free);  // O may take the next item
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int rr = i * 4 + (lane >> 3), cc = lane & 7;
            const uint4 v = ld_shared_v4(stage + rr * 128 + ((cc ^ (rr & 7)) << 4));
            if (q * 32 + rr < it.q_len)
                *reinterpret_cast<uint4 *>(dst + static_cast<int64_t>(rr) * kD + half * 64 + cc * 8) = v;
        }
        __syncwarp();  // the stage is rewritten next
    }
    return true;
}

__global__ void __launch_bounds__(kThreads, 1)
    packed_attention_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                            const __grid_constant__ CUtensorMap tm_vt, const AttnArgs a) {
    extern __shared__ uint8_t dyn_smem[];
    __shared__ Ctl c;
    // (from lane 0, so that the compiler knows the role branches and what they
    // compute to be uniform over the warp)
    const int warp = __shfl_sync(kFull, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    uint8_t *base = dyn_smem + ((1024u - (saddr(dyn_smem) & 1023u)) & 1023u);
    uint8_t *sq = base;                          // Q buffers
    uint8_t *sk = sq + kQBufs * kQBytes;         // K stages
    uint8_t *sv = sk + kKvStages * kKBytes;      // V^T stages
    uint8_t *so = sv + kKvStages * kVBytes;      // output stages of the read-out warps
    // Every item has the same number of key tiles (the context's and one
    // branch's), so the CTA's key tiles are numbered globally: tile t is tile
    // t % T of the CTA's item t / T.
    const int T = a.q_tiles_ctx + a.q_tiles_branch;
    const int my_items = blockIdx.x < static_cast<unsigned>(a.items)
                             ? (a.items - 1 - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x) + 1
                             : 0;
    const uint32_t tiles = static_cast<uint32_t>(my_items) * T;

    if (threadIdx.x == 0) {
        for (int b = 0; b < kQBufs; ++b) mbar_init(&c.q_full[b], 1);
        for (int s = 0; s < kKvStages; ++s) {
            mbar_init(&c.k_full[s], 1);
            mbar_init(&c.v_full[s], 1);
            mbar_init(&c.v_empty[s], 1);
        }
        for (int b = 0; b < kHalves; ++b) {
            mbar_init(&c.s_full[b], 1);
            mbar_init(&c.p_full[b], 4);  // a half's four warps
        }
        mbar_init(&c.o_ready, 1);
        mbar_init(&c.o_free, kOutWarps);
        mbar_init(&c.mma_done, 1);
        c.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc(&c.tmem_base, kTmemCols);
        tmem_relinquish();
    }
    pdl_wait();
    pdl_launch_next();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = c.tmem_base;
    constexpr uint32_t idesc = umma::instr_desc_bf16(kBQ, kBK);

    if (warp < 4) {  // (setmaxnreg: each warpgroup as a whole, before its warps part)
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kCtlRegs));
    if (warp == 0) {
        if (lane == 0) {  // -------------------------------------------- Q and K producer
            uint32_t t = 0;  // key tiles issued
            int n_q = 0;     // Q tiles issued
            Item it{};
            ItemWalk wk = item_walk(a);
            for (int n = 0, j = 0; t < tiles; ++t, next_tile(n, j, T)) {
                // S of tile t - 2 is computed: K stage t % 2 is free, and at an item's
                // first tile the Q buffer of item n - 2, whose last tile is no later
                const int s = t % kKvStages;
                if (t >= kKvStages && !wait_or_abort(&c.s_full[s], (t / kKvStages - 1) & 1, c, a)) break;
                if (j == 0) {  // this item's Q, into buffer n % 2
                    if (n > 0) item_next(wk);
                    it = item_at(a, wk);
                    const int b = n & 1;
                    mbar_expect_tx(&c.q_full[b], kQBytes);
                    const int qrow = it.bh * a.n_tokens + it.q_start;
                    tma_load_2d(sq + b * kQBytes, &tm_q, 0, qrow, &c.q_full[b]);
                    tma_load_2d(sq + b * kQBytes + kAtom, &tm_q, 64, qrow, &c.q_full[b]);
                    ++n_q;
                }
                int k0, valid;
                key_tile(a, it, j, k0, valid);
                uint8_t *dst = sk + s * kKBytes;
                mbar_expect_tx(&c.k_full[s], kKBytes);
                const int krow = it.bh * a.n_tokens + k0;
                tma_load_2d(dst, &tm_k, 0, krow, &c.k_full[s]);
                tma_load_2d(dst + kAtom, &tm_k, 64, krow, &c.k_full[s]);
            }
            // every copy issued lands before the CTA leaves
            for (uint32_t x = t > kKvStages ? t - kKvStages : 0; x < t; ++x)
                wait_drain(&c.k_full[x % kKvStages], (x / kKvStages) & 1);
            for (int n = n_q > kQBufs ? n_q - kQBufs : 0; n < n_q; ++n) wait_drain(&c.q_full[n & 1], (n >> 1) & 1);
        }
    } else if (warp == kVWarp) {
        if (lane == 0) {  // -------------------------------------------- V producer
            uint32_t t = 0;
            Item it{};
            ItemWalk wk = item_walk(a);
            for (int n = 0, j = 0; t < tiles; ++t, next_tile(n, j, T)) {
                if (j == 0) {
                    if (n > 0) item_next(wk);
                    it = item_at(a, wk);
                }
                const int s = t % kKvStages;
                if (!wait_or_abort(&c.v_empty[s], ((t / kKvStages) & 1) ^ 1, c, a)) break;
                int k0, valid;
                key_tile(a, it, j, k0, valid);
                uint8_t *dst = sv + s * kVBytes;
                mbar_expect_tx(&c.v_full[s], kVBytes);
                tma_load_2d(dst, &tm_vt, k0, it.bh * kD, &c.v_full[s]);
                tma_load_2d(dst + kAtom, &tm_vt, k0 + 64, it.bh * kD, &c.v_full[s]);
            }
            for (uint32_t x = t > kKvStages ? t - kKvStages : 0; x < t; ++x)
                wait_drain(&c.v_full[x % kKvStages], (x / kKvStages) & 1);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------- MMA issuer (lane 0, the warp converged)
        {
            const uint32_t issue = lane == 0;
            // S of the first two tiles, then per tile the product P V and S two
            // tiles on, into the buffer whose P the product has read: the tensor
            // pipe runs them in order, so nothing waits in between.
            bool ok = true;
            int n = 0, j = 0;    // the product's item and tile
            int sn = 0, sj = 0;  // the scores'
            const auto scores = [&](uint32_t t) -> bool {  // S_t = Q K_t^T into buffer t % 2
                const int qb = sn & 1, s = t % kKvStages;
                if ((sj == 0 && !warp_wait_or_abort(&c.q_full[qb], (sn >> 1) & 1, c, a)) ||
                    !warp_wait_or_abort(&c.k_full[s], (t / kKvStages) & 1, c, a))
                    return false;
                tc_fence_after();
                const uint64_t qd = umma::smem_desc_kmajor_sw128(saddr(sq + qb * kQBytes));
                const uint64_t qd1 = umma::smem_desc_kmajor_sw128(saddr(sq + qb * kQBytes + kAtom));
                const uint64_t kd = umma::smem_desc_kmajor_sw128(saddr(sk + s * kKBytes));
                const uint64_t kd1 = umma::smem_desc_kmajor_sw128(saddr(sk + s * kKBytes + kAtom));
                const uint32_t sbuf = tmem + (t % kHalves) * kBK;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    mma_bf16(sbuf, umma::advance_k16(k < 4 ? qd : qd1, k & 3), umma::advance_k16(k < 4 ? kd : kd1, k & 3),
                             idesc, k != 0, issue);
                mma_commit(&c.s_full[t % kHalves], issue);
                next_tile(sn, sj, T);
                return true;
            };
            for (uint32_t t = 0; t < min(tiles, static_cast<uint32_t>(kHalves)) && ok; ++t) ok = scores(t);
            for (uint32_t t = 0; t < tiles && ok; ++t, next_tile(n, j, T)) {  // O[t % 2] += P_t V_t
                // the first product of an item overwrites O: the previous item's read-out must be done
                if ((j == 0 && !warp_wait_or_abort(&c.o_free, (n & 1) ^ 1, c, a)) ||
                    !warp_wait_or_abort(&c.p_full[t % kHalves], (t / kHalves) & 1, c, a) ||
                    !warp_wait_or_abort(&c.v_full[t % kKvStages], (t / kKvStages) & 1, c, a)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint8_t *vb = sv + (t % kKvStages) * kVBytes;
                const uint64_t vd = umma::smem_desc_kmajor_sw128(saddr(vb));
                const uint64_t vd1 = umma::smem_desc_kmajor_sw128(saddr(vb + kAtom));
                // P of keys 16k..16k+15: columns 8k..8k+7 of S buffer t % 2; the half's
                // first product of an item overwrites its O
                const uint32_t b = t % kHalves, pcol = tmem + b * kBK, ocol = tmem + kOCol + b * kBK;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    mma_bf16_ts(ocol, pcol + k * 8, umma::advance_k16(k < 4 ? vd : vd1, k & 3), idesc,
                                (j >= kHalves || k != 0) ? 1u : 0u, issue);
                mma_commit(&c.v_empty[t % kKvStages], issue);
                if (j == T - 1) mma_commit(&c.o_ready, issue);  // the item's O is complete
                if (t + kHalves < tiles) ok = scores(t + kHalves);
            }
            mma_commit(&c.mma_done, issue);
            if (lane == 0) wait_drain(&c.mma_done, 0);
        }
        __syncwarp();
    }
    } else if (warp < 12) {  // ------------------------------------- softmax (warps 4-11)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftRegs));
        const int q = warp & 3, h = (warp >> 2) - 1;  // TMEM lane quarter; half
        const int r = q * 32 + lane;                  // query row in the tile (TMEM lane)
        const uint32_t lane_off = static_cast<uint32_t>(q * 32) << 16;
        const uint32_t sbuf = tmem + lane_off + h * kBK, obuf = tmem + lane_off + kOCol + h * kBK;
        const int own0 = a.group > 1 ? r / a.branch_len * a.branch_len : 0;  // the row's branch in a group
        ItemWalk wk = item_walk(a);
        bool ok = true;
        for (int n = 0; n < my_items && ok; ++n) {
            if (n > 0) item_next(wk);
            const Item it = item_at(a, wk);
            float m = -INFINITY, l = 0.f;
            for (int j = (h ^ (n * T)) & 1; j < T; j += kHalves) {
                const uint32_t t = static_cast<uint32_t>(n) * T + j;
                if (!warp_wait_or_abort(&c.s_full[h], (t / kHalves) & 1, c, a)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                uint32_t s0[32], s1[32], s2[32], s3[32];  // the row's 128 scores
                tmem_ld32_async(sbuf, s0);
                tmem_ld32_async(sbuf + 32, s1);
                tmem_ld32_async(sbuf + 64, s2);
                tmem_ld32_async(sbuf + 96, s3);
                tmem_wait_dep(s0);
                tmem_wait_dep(s1);
                tmem_wait_dep(s2);
                tmem_wait_dep(s3);
                int k0, valid;
                key_tile(a, it, j, k0, valid);
                const bool own = it.grouped && j >= it.n_ctx_tiles;
                if (valid < kBK || own) {  // keys past the segment's end, or of other branches, take no weight
                    const int lo = own ? min(own0, valid - a.branch_len) : 0;  // (rows past q_len: the last branch)
                    const int hi = own ? lo + a.branch_len : valid;
                    mask_scores(s0, lo, hi);
                    mask_scores(s1, lo - 32, hi - 32);
                    mask_scores(s2, lo - 64, hi - 64);
                    mask_scores(s3, lo - 96, hi - 96);
                }
                // the row's largest score (eight independent chains)
                float mx8[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) mx8[i] = -INFINITY;
                max_scores(s0, mx8);
                max_scores(s1, mx8);
                max_scores(s2, mx8);
                max_scores(s3, mx8);
                const float tm = fmaxf(fmaxf(fmaxf(mx8[0], mx8[1]), fmaxf(mx8[2], mx8[3])),
                                       fmaxf(fmaxf(mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7]))) * a.c;
                float f = 1.f;
                bool rescale = false;
                if (m == -INFINITY) {
                    m = tm;
                } else if (tm > m + kRescale) {
                    f = ex2(m - tm);
                    m = tm;
                    rescale = true;
                }
                // tcgen05.ld / st are warp-wide (.sync.aligned): the warp rescales
                // its O together when any of its rows needs it, the other rows
                // by f = 1. The half's previous product (tile t - 2) is done: S of
                // this tile was issued after it.
                if (__any_sync(kFull, rescale)) {
#pragma unroll 1
                    for (int ch = 0; ch < kBK / 16; ++ch) {
                        uint32_t o[16];
                        tmem_ld16_async(obuf + ch * 16, o);
                        tmem_wait_dep(o);
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
                        tmem_st16(obuf + ch * 16, o);
                    }
                }
                l *= f;
                // P = 2^(s c - m) (a masked key gives 2^-inf = 0), bf16 pairs, over
                // the first 64 columns of S (already in registers). Scores of -inf in
                // all of the half's tiles so far leave m there: P = 0, and the sum 0.
                const float mr = m == -INFINITY ? 0.f : -m;
                const f2 cc = pack2(a.c, a.c), mm = pack2(mr, mr);
                f2 lsum[4] = {pack2(0.f, 0.f), pack2(0.f, 0.f), pack2(0.f, 0.f), pack2(0.f, 0.f)};
                uint32_t pk[32];
                exp_scores(s0, cc, mm, lsum, pk, 0);
                exp_scores(s1, cc, mm, lsum, pk, 16);
                tmem_st32_u(sbuf, pk);
                uint32_t pk2[32];
                exp_scores(s2, cc, mm, lsum, pk2, 0);
                exp_scores(s3, cc, mm, lsum, pk2, 16);
                tmem_st32_u(sbuf + 32, pk2);
                {
                    float l0, l1;
                    unpack2(add2(add2(lsum[0], lsum[1]), add2(lsum[2], lsum[3])), l0, l1);
                    l += l0 + l1;
                }
                if (j + kHalves >= T) c.ml[n & 3][h][r] = make_float2(m, l);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&c.p_full[h]);
            }
        }
    } else {  // ---------------------------------------------------- read-out (warps 12-15)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOutRegs));
        ItemWalk wk = item_walk(a);
        for (int n = 0; n < my_items; ++n) {
            if (n > 0) item_next(wk);
            const Item it = item_at(a, wk);
            if (!read_out(it, n, T, tmem, warp & 3, lane, saddr(so + (warp - 12) * kStageBytes), c, a)) break;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

// ---------------------------------------------------------------- host
std::mutex g_attn_mutex;
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
bool g_attr_set[64] = {};
int g_sm_count[64] = {};

rps_status attn_setup(int *sm_count) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return RPS_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_attn_mutex);
    if (!g_encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return RPS_ERR_CUDA;
        g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    if (!g_attr_set[dev]) {
        if (cudaDeviceGetAttribute(&g_sm_count[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return RPS_ERR_CUDA;
        if (cudaFuncSetAttribute(packed_attention_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) !=
            cudaSuccess)
            return RPS_ERR_CUDA;
        g_attr_set[dev] = true;
    }
    *sm_count = g_sm_count[dev];
    return RPS_OK;
}

rps_status map_2d(CUtensorMap *m, const void *base, int64_t rows, int64_t cols) {
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(cols) * 2};
    const cuuint32_t box[2] = {64, 128};
    const cuuint32_t es[2] = {1, 1};
    const CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? RPS_OK : RPS_ERR_CUDA;
}

}  // namespace
}  // namespace rps

using namespace rps;

extern "C" rps_status rps_packed_attention_fwd(const rps_packed_attention *p, rps_stream_t stream) {
    if (!p || !p->q || !p->k || !p->vt || !p->out) return RPS_ERR_INVALID_ARG;
    if (p->head_dim != kD) return RPS_ERR_UNSUPPORTED;
    if (p->n_batch < 1 || p->n_heads < 1 || p->n_context < 0 || p->n_branch < 1 || p->branch_len < 1)
        return RPS_ERR_INVALID_ARG;
    if (p->n_context % 8 || p->branch_len % 8) return RPS_ERR_INVALID_ARG;
    if (!(p->scale > 0.f) || !std::isfinite(p->scale)) return RPS_ERR_INVALID_ARG;
    for (const void *x : {p->q, p->k, p->vt, static_cast<const void *>(p->out)})
        if (reinterpret_cast<uintptr_t>(x) % 16) return RPS_ERR_INVALID_ARG;
    const int64_t n_tokens = static_cast<int64_t>(p->n_context) + static_cast<int64_t>(p->n_branch) * p->branch_len;
    const int64_t n_bh = static_cast<int64_t>(p->n_batch) * p->n_heads;
    if (n_tokens > INT32_MAX / 2 || n_bh * n_tokens > INT32_MAX || n_bh * kD > INT32_MAX) return RPS_ERR_UNSUPPORTED;
    int sm_count = 0;
    rps_status st = attn_setup(&sm_count);
    if (st != RPS_OK) return st;
    uint32_t *err = device_error_word();
    if (!err) return RPS_ERR_CUDA;
    CUtensorMap tq, tk, tv;
    if ((st = map_2d(&tq, p->q, n_bh * n_tokens, kD)) != RPS_OK) return st;
    if ((st = map_2d(&tk, p->k, n_bh * n_tokens, kD)) != RPS_OK) return st;
    if ((st = map_2d(&tv, p->vt, n_bh * kD, n_tokens)) != RPS_OK) return st;
    AttnArgs a;
    std::memset(&a, 0, sizeof a);
    a.n_bh = static_cast<int32_t>(n_bh);
    a.n_heads = p->n_heads;
    a.n_tokens = static_cast<int32_t>(n_tokens);
    a.n_context = p->n_context;
    a.n_branch = p->n_branch;
    a.branch_len = p->branch_len;
    a.q_tiles_ctx = (p->n_context + kBQ - 1) / kBQ;
    a.q_tiles_branch = (p->branch_len + kBQ - 1) / kBQ;
    // Branches of at most half a tile share query tiles: 9 branches of 32 take three
    // tiles instead of nine that are three quarters empty. Longer ones would not fit
    // twice.
    a.group = std::min(kBQ / std::min(p->branch_len, kBQ), p->n_branch);
    a.groups = (p->n_branch + a.group - 1) / a.group;
    const int64_t items = n_bh * (a.q_tiles_ctx + static_cast<int64_t>(a.groups) * a.q_tiles_branch);
    if (items > INT32_MAX) return RPS_ERR_UNSUPPORTED;
    a.items = static_cast<int32_t>(items);
    a.c = p->scale * kLog2e;
    a.out = static_cast<__nv_bfloat16 *>(p->out);
    a.err = err;
    a.wait_ns = ring_wait_limit_ns();
    const int grid = static_cast<int>(std::min<int64_t>(items, sm_count));
    const cudaError_t e = launch_pdl(packed_attention_kernel, dim3(grid), dim3(kThreads), kSmemBytes,
                                     reinterpret_cast<cudaStream_t>(stream), tq, tk, tv, a);
    return e == cudaSuccess ? RPS_OK : RPS_ERR_CUDA;
}
