// (a3)-(a6) Layers of the learned recursion (Eq. mlsp2) for every active
// (instance, chain) of a grouped launch, on the 5th-generation tensor cores:
// one layer per launch, or consecutive layers of the main format in one
// persistent cooperative launch (below).
//
// The product of a layer is the symmetric square Z^2 of the centred state.
// Output tiles are 256 x 256 or 256 x 128 (CTA pairs) or 128 x 128 or 128 x 64
// (single CTAs), chosen per call, and only those touching the upper triangle are computed; each
// element (r, c) with r <= c is produced once.  Since Z is
// symmetric, (Z^2)_{rc} = sum_k Z_{rk} Z_{ck}: both MMA operands are row
// panels of the same matrix, loaded by TMA with 128-byte swizzle.  The next
// operands are stored for the upper triangle plus the diagonal tile blocks
// (the mirror (c, r) everywhere only before a layer that reads full
// matrices); K-slices left of a panel's diagonal block are loaded as
// transposed 64 x 64 panels of the upper triangle (MN-major operands).
//
// Split precision (Sec. IV A, Eq. emulated matmul, generalised): Z is stored as
// NSPLIT low-precision planes Z = sum_s Z_s and the products Z_s Z_t with
// s + t small enough are accumulated in FP32:
//   FP16X2: (0,0) (0,1) (1,0)    TF32X3: same      BF16X3: + (0,2) (2,0) (1,1)
// (the paper's two GEMMs plus a transpose-add become three products on the
// triangle: 1.5 n^3 MACs instead of 2 n^3).
//
// Tile shapes.  CTA pairs (cta_group::2): a cluster of two CTAs computes one
// 256 x 256 or 256 x 128 tile with M = 256 MMAs issued by the even CTA.  CTA r
// loads its own 128 rows of the A panel and its half of the B panel, so each SM
// fills and reads half of B.  Both CTAs' TMA loads complete on the even CTA's
// "full" barrier; the MMA commit is multicast to both CTAs' "empty" and "tfull"
// barriers; the odd CTA's epilogue warps release accumulators on the even CTA's
// "tempty".  Single CTAs (cta_group::1) run the same pipeline on 128 x 128 tiles
// with M = 128 MMAs: the least padding on the diagonal and at ragged edges, but
// an MMA whose two panels come from one shared memory takes 119 clocks for 64
// (a pair's 256 x 128 one: 71).  128 x 64 tiles of single CTAs, for calls of few
// tiles, where a layer is one tile's latency: half the columns of an epilogue warp
// and twice the SMs at work, an MMA of about 80 clocks for the 32 that it runs.
// Per solve against the best of the others: n = 256 239 -> 214 us, mu search at
// 512 1380 -> 1253, n = 1024 BF16X3 553 -> 519, n = 384 TF32X3 428 -> 330.  One
// choice per call (shape_cost in ftsp2_api.cu).
//
// Chunked accumulation.  Every 128 elements of K (CK slices; a launch may ask
// for shorter chunks) the MMAs switch to the next of the TMEM chunk
// accumulators (two of 256 columns, four of 128) and the epilogue adds the
// finished chunk into FP32 registers; the tensor core's internal accumulation
// then spans 128 products per chunk instead of all n.  Measured at n = 4096 with
// the printed table (density, FP16X2): chunks of 256 / 128 / 64 elements give
// max|D - D_ref| = 1.85e-6 / 9.0e-7 / 6.9e-7 at layer times 0.235 / 0.251 /
// 0.314 ms (an earlier kernel); 128 is the default.
//
// layer_tc_kernel (persistent over the unit's items):
//   warp 0     : TMA producer (ring of 128-byte K-slices)
//   warp 1     : TMEM allocation; MMA issuer (even CTA)
//   warps 2 .. : epilogue warps; warp w reads TMEM lane quarter w % 4 and a column
//                group of the CTA's 128-row accumulator, adds the chunks in FP32
//                registers and runs the final epilogue (Z_{k+1}, A_{k+1}, next
//                operands).  It is a chain of short dependent steps (a warp issues
//                an instruction every eleven clocks), so FP16X2 operands of
//                128-column tiles have 16 warps of 32 columns (96 registers) and
//                256-column tiles 16 warps of 64; the others have 8 warps of 64
//                columns (168 registers): the wider formats' planes spill in 96.  8 -> 16 warps, FP16X2: n = 256
//                277 -> 261 us, 60 fragments 411 -> 380, ragged batch 22.8 ->
//                22.1 ms, n = 1501 unchanged; BF16X3 and TF32X3 on 128 columns
//                0.7 % slower at n = 1024 and 2048.  256 x 256 tiles, inline, 8 ->
//                16 warps with the state 16 columns ahead: n = 2200 TF32X3
//                (density) 2173 -> 2038 us, n = 2700 FP16X2 1526 -> 1456, n = 2816
//                FP16X2 (density + entropy) 2716 -> 2546; their last layer at n =
//                4096 440 -> 332.
//   last warp  : context warp (below)
// The loops of warps 0 and 1 run on the whole warp with one elected lane issuing:
// their values are then uniform, and a copy or an MMA takes no moves from vector
// registers to uniform ones (110 against 71 clocks per 128-column MMA, 150
// against 50 per copy).
// On 128-column tiles an epilogue warp keeps its sums in registers and releases
// every chunk buffer at once; a 256-column tile's sums are written back to the
// last buffer, which stays held.  Where a launch has one tile per unit, Z and A
// of that tile stay in TMEM from layer to layer.
// One lattice, density + entropy, FP16X2, per solve, before (single CTAs, 576
// threads, operands written by plain stores) and now, the rest of a solve
// included: n = 256: 402 -> 208 us; n = 1501 (entropy): 789 -> 498 us; n = 1024
// BF16X3 (density): 814 -> 520 us; n = 2048 TF32X3 (density): 2567 -> 2208 us.
//
// layer_defer_kernel (640 threads; 256 x 256 tiles with long K).  Sixteen
// accumulating warps store a tile's sums to a per-CTA scratch in global memory
// and go on with the next tile at once; two store warps stream scratch, Z_k and
// A_k through a small shared ring (cp.async) and run the final epilogue while the
// next tile's MMAs run.  A unit's last tile runs inline, so no store-warp tail
// follows the last MMAs.  At 96 registers a thread (640 threads) the epilogue has
// 16 columns of the state at a time and its context in shared memory; with 32
// columns and a context in registers it spilled 640 bytes for 390 (FP16X2), and
// n = 2816 (density + entropy, deferred) took 2810 us, 2431 now, n = 5000 TF32X3
// (density) 11585, 11340 now.
//
// Multi-layer launches (a.nlayers > 1).  The work items are (layer, tile) in
// layer order; every role walks the same item sequence.  An item of layer g
// waits (producer) until all tiles of layer g - 1 of its instance and chain
// have finished their epilogues: each CTA counts its epilogue (accumulating)
// warps' completions per tile in the instance's counter, released after the
// warp's stores and acquired by the readers, with a proxy fence before the TMA
// loads of the new operands.  Dependencies point only to earlier items and a
// unit takes its items in order, so the waits end; the CTAs of such a launch are
// co-resident (cooperative launch).
// Every wait is bounded (a.wait_ns).  A dependency wait that runs out records
// FTSP2_E_TIMEOUT in the status word of the call; from then on every role of
// every CTA that sees the failure runs the rest of its work items in skip
// mode: the same barrier arrivals, waits and commits in the same order, but no
// TMA loads and no epilogue stores.  layer_tc_kernel's MMAs still run, on whatever
// their stage holds (one CTA of a pair may skip while its peer loads): they write
// only TMEM, their sums are not stored, and their commits complete the phases as
// usual; layer_defer_kernel leaves them out.  Every barrier phase therefore still
// completes and nothing is in flight when the work list ends; the MMA issuer
// also waits for a last commit of its own before the CTAs free TMEM.  A
// pipeline wait that runs out twice (a broken protocol, not expected) leaves
// its loop after a bounded grace period for the copies in flight.
#include <atomic>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "epilogue.cuh"
#include "ftsp2_internal.h"

namespace ftsp2 {

template <int MODE>
struct TcCfg;

template <>
struct TcCfg<FTSP2_FP16X2> {
    static constexpr int NSPLIT = 2, ESIZE = 2, STAGES = 3, NPROD = 3, CK = 2;
    static constexpr uint32_t ATYPE = 0;      // f16
    static constexpr bool TF32 = false;
};
template <>
struct TcCfg<FTSP2_BF16X3> {
    static constexpr int NSPLIT = 3, ESIZE = 2, STAGES = 2, NPROD = 6, CK = 2;
    static constexpr uint32_t ATYPE = 1;      // bf16
    static constexpr bool TF32 = false;
};
template <>
struct TcCfg<FTSP2_TF32X3> {
    static constexpr int NSPLIT = 2, ESIZE = 4, STAGES = 3, NPROD = 3, CK = 4;
    static constexpr uint32_t ATYPE = 2;      // tf32
    static constexpr bool TF32 = true;
};

// Tile geometry.  SHAPE_SINGLE: one CTA, 128 x 128 tiles, M = 128 MMAs.
// SHAPE_PAIR / SHAPE_PAIR128: clusters of two CTAs, M = 256 MMAs on 256 x 256 or
// 256 x 128 tiles.  SHAPE_SINGLE64: one CTA, 128 x 64 tiles.  A CTA owns 128 rows of
// its tile in every shape.
template <int SHAPE>
struct Geo {
    static constexpr int NCTA = tc_pair(SHAPE) ? 2 : 1;
    static constexpr int TM = 128 * NCTA;                      // rows of a tile
    // columns of a tile
    static constexpr int TN = SHAPE == SHAPE_PAIR ? 256 : SHAPE == SHAPE_SINGLE64 ? 64 : 128;
    static constexpr int BROWS = TN / NCTA;                    // rows of the B panel a CTA loads
    // TMEM chunk accumulators of TN columns (512 columns in all)
    static constexpr int NBUF = 512 / TN;
};
constexpr int kCtaRows = 128;
// Epilogue warps of layer_tc_kernel, followed by the context warp.
template <int OUTFMT, int SHAPE>
constexpr int epi_warps() {
    if (SHAPE == SHAPE_SINGLE64) return OUTFMT == -1 ? 4 : 8;     // last layer: a 32 x 64 block of partial sums a warp
    return SHAPE == SHAPE_PAIR || OUTFMT == OP_F16X2 ? 16 : 8;
}
template <int OUTFMT, int SHAPE>
constexpr int tc_threads() { return 32 * (2 + epi_warps<OUTFMT, SHAPE>() + 1); }
// Deferred final epilogue: store warps, their shared-memory staging ring
// (entries of 16 columns x 32 rows: sums, Z_k, A_k) and the per-CTA scratch
// of finished tile sums in global memory (one 32-row x 64-column block per
// accumulating warp, in the blocked layout of the state).
constexpr int kDeferWarps = 16;
constexpr int kStoreWarps = 2;
constexpr int kRing = 2;
constexpr int kEntryBytes = 3 * 2048;
constexpr int kItemFloats = 2048;
static_assert(kDeferWarps * kItemFloats == kEpiScratchFloats, "scratch of one CTA");
// multi-layer launches: the store warps' shares of a tile's completions add up
// to the kDeferWarps that the accumulating warps give for an inline tile
static_assert(kDeferWarps % kStoreWarps == 0, "completion shares of the store warps");
constexpr int kDeferThreads = 64 + 32 * (kDeferWarps + kStoreWarps);

// split planes (s, t) of the products Z_s Z_t, in issue order
__host__ __device__ constexpr int prod_a(int p) { return p == 2 ? 1 : (p == 4 ? 2 : (p == 5 ? 1 : 0)); }
__host__ __device__ constexpr int prod_b(int p) { return p == 1 ? 1 : (p == 3 ? 2 : (p == 5 ? 1 : 0)); }

// Instruction descriptor of tcgen05.mma kind::f16 / kind::tf32: D in FP32,
// A and B K-major, M x N.
__host__ __device__ constexpr uint32_t make_idesc(uint32_t atype, int M, int N) {
    return (1u << 4)                       // D format: F32
           | (atype << 7) | (atype << 10)  // A, B formats
           | ((uint32_t)(N >> 3) << 17)    // N >> 3
           | ((uint32_t)(M >> 4) << 24);   // M >> 4
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, rows of 128 bytes,
// 8-row swizzle atoms of 1024 bytes (stride byte offset), version bits 46-48 = 1.
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;                 // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset
    d |= (uint64_t)1 << 46;                 // descriptor version
    d |= (uint64_t)2 << 61;                 // SWIZZLE_128B
    return d;
}

// MN-major (transposed) operand panel, 128-byte swizzle: atoms of 8 K-rows x
// 64 MN elements (1 KB), the K atoms of one 64-wide MN half consecutive, the
// second MN half 8 KB further.
constexpr uint32_t kMnLbo = 8192, kMnSbo = 1024;
__device__ __forceinline__ uint64_t sdesc_mn_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(kMnLbo >> 4) << 16;     // leading byte offset
    d |= (uint64_t)(kMnSbo >> 4) << 32;     // stride byte offset
    d |= (uint64_t)1 << 46;                 // descriptor version
    d |= (uint64_t)2 << 61;                 // SWIZZLE_128B
    return d;
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// shared::cluster address of the same shared variable in CTA `rank`
__device__ __forceinline__ uint32_t map_to(uint32_t local, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// Arrivals on a barrier of either CTA of the pair.  The barriers only order
// asynchronous-proxy work (TMA completion, tcgen05 commits, TMEM reads fenced
// with tcgen05.fence), so CTA-scope semantics suffice and no cluster-wide
// memory fence is issued per arrival.
__device__ __forceinline__ void remote_arrive(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void remote_expect_tx(uint32_t cluster_addr, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%0], %1;" ::"r"(cluster_addr), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool try_wait_cluster(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Has the call failed (a wait ran out in this or another CTA)?
__device__ __forceinline__ bool call_failed(const LayerArgs& a) {
    return *reinterpret_cast<volatile int*>(a.status) != 0;
}
__device__ __forceinline__ void record_timeout(const LayerArgs& a) { atomicCAS(a.status, 0, (int)FTSP2_E_TIMEOUT); }

// Wait on a pipeline mbarrier phase.  A failure elsewhere never ends such a
// wait: after a failure every role keeps the barrier protocol of its work list
// (arrivals and commits in the usual order, without loads or stores), so every
// phase still completes.  The wait gives up only on its own clock: after
// a.wait_ns it records FTSP2_E_TIMEOUT (the call has failed), and after twice
// that it returns false, which only a broken protocol can cause; the caller
// then leaves its loop and the kernel drains before it frees TMEM.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, const LayerArgs& a) {
    if (try_wait_cluster(bar, parity)) return true;
    const unsigned long long t0 = globaltimer();
    bool recorded = false;
    for (uint32_t it = 1;; ++it) {
        if (try_wait_cluster(bar, parity)) return true;
        if ((it & 63u) == 0) {
            const unsigned long long dt = globaltimer() - t0;
            if (!recorded && dt > a.wait_ns) {
                record_timeout(a);
                recorded = true;
            }
            if (dt > 2 * a.wait_ns) return false;
        }
    }
}

// ... of a whole warp; the result is uniform
__device__ __forceinline__ bool all_wait(uint64_t* bar, uint32_t parity, const LayerArgs& a) {
    return __all_sync(0xffffffffu, wait_bar(bar, parity, a));
}
// lane 0's value as a uniform one
__device__ __forceinline__ uint32_t uniform32(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ uint64_t uniform64(uint64_t v) {
    return ((uint64_t)uniform32((uint32_t)(v >> 32)) << 32) | uniform32((uint32_t)v);
}
__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e != 0;
}

// TMA 2-D tile load into this CTA's shared memory, completing on an mbarrier
// that may live in the peer CTA of the pair.
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar_cluster, int x,
                                              int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
        "%4}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster), "r"(x), "r"(y)
        : "memory");
}

template <bool TF32>
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc,
                                          uint32_t accumulate) {
    if constexpr (TF32) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
            "l"(da), "l"(db), "r"(idesc), "r"(accumulate));
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
            "l"(da), "l"(db), "r"(idesc), "r"(accumulate));
    }
}

// arrive (once) on the barrier at this shared offset in both CTAs of the pair
// when all previously issued MMAs of this thread have completed
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
    const uint16_t mask = 0x3;
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
        "h"(mask)
        : "memory");
}

// arrive on this CTA's barrier only, when all previously issued MMAs of this
// thread (on both CTAs of the pair) have completed
__device__ __forceinline__ void umma_commit_local_pair(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 32 lanes x 16 columns of FP32 from TMEM into registers (no wait)
// single-CTA counterparts
__device__ __forceinline__ void tma_load_one(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
        : "memory");
}
template <bool TF32>
__device__ __forceinline__ void umma_one(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc,
                                         uint32_t accumulate) {
    if constexpr (TF32) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
            "l"(da), "l"(db), "r"(idesc), "r"(accumulate));
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
            "l"(da), "l"(db), "r"(idesc), "r"(accumulate));
    }
}
__device__ __forceinline__ void umma_commit_one(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void local_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void local_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
        "%12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float* x) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
                 "r"(__float_as_uint(x[0])), "r"(__float_as_uint(x[1])), "r"(__float_as_uint(x[2])),
                 "r"(__float_as_uint(x[3])), "r"(__float_as_uint(x[4])), "r"(__float_as_uint(x[5])),
                 "r"(__float_as_uint(x[6])), "r"(__float_as_uint(x[7]))
                 : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* x) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16};" ::"r"(taddr),
        "r"(__float_as_uint(x[0])), "r"(__float_as_uint(x[1])), "r"(__float_as_uint(x[2])), "r"(__float_as_uint(x[3])),
        "r"(__float_as_uint(x[4])), "r"(__float_as_uint(x[5])), "r"(__float_as_uint(x[6])), "r"(__float_as_uint(x[7])),
        "r"(__float_as_uint(x[8])), "r"(__float_as_uint(x[9])), "r"(__float_as_uint(x[10])),
        "r"(__float_as_uint(x[11])), "r"(__float_as_uint(x[12])), "r"(__float_as_uint(x[13])),
        "r"(__float_as_uint(x[14])), "r"(__float_as_uint(x[15]))
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Split formats of the next layer's operands: planes, bytes of an element.
template <int FMT>
struct OpFmtT;
template <>
struct OpFmtT<OP_F16X2> {
    static constexpr int NPL = 2, ESZ = 2;
};
template <>
struct OpFmtT<OP_BF16X3> {
    static constexpr int NPL = 3, ESZ = 2;
};
template <>
struct OpFmtT<OP_TF32X3> {
    static constexpr int NPL = 2, ESZ = 4;
};
template <>
struct OpFmtT<OP_F32> {
    static constexpr int NPL = 1, ESZ = 4;
};

constexpr int kLastLayer = -1;

// The 8 state values of a row past the L1 (no reuse, and in multi-layer launches
// other CTAs write them) and in program order with the waits around it.
__device__ __forceinline__ void ld_state8(const float* S, float* x) {
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3])
                 : "l"(S));
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7])
                 : "l"(S + 128));
}

// The persistent loop of a unit visits tiles t, t + nunits, ...: is there an
// active tile after t?  (The last tile of a unit runs its final epilogue inline,
// so that no store-warp tail follows the last MMAs.)
// Work items of a launch: item f is (global layer gl + f / ntiles, tile
// f % ntiles); a one-layer launch has ntiles items.
__device__ __forceinline__ int n_items(const LayerArgs& a) { return a.ntiles * a.nlayers; }
__device__ __forceinline__ void item_of(const LayerArgs& a, int f, int& g, int& t) {
    const int l = f / a.ntiles;
    g = a.gl + l;
    t = f - l * a.ntiles;
}

// Does the unit have an active item after item f?
__device__ __forceinline__ bool has_next_tile(const LayerArgs& a, int f, int nunits) {
    const int nf = n_items(a);
    for (int u = f + nunits; u < nf; u += nunits) {
        int g, t, k;
        item_of(a, u, g, t);
        if (tile_active_g(a, a.tiles[t], g, k)) return true;
    }
    return false;
}

// Completion counters of multi-layer launches, one per (layer, instance,
// chain): an epilogue warp adds its share after its stores (release: fence,
// then the atomic); a reader acquires.  (A counter shared by a whole layer
// took 16 atomics per tile from every CTA on one address, which serialised
// ragged batches of ten thousand tiles per layer.)
__device__ __forceinline__ int* inst_counter(const LayerArgs& a, int g, int inst, int chain) {
    return a.done_inst + ((size_t)g * a.nb + inst) * kMaxChains + chain;
}
__device__ __forceinline__ void done_add(int* counter, int v) {
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(counter), "r"(v) : "memory");
}
__device__ __forceinline__ int acquire_load(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Wait until the counter at p reaches target.  False when the call has failed
// (this wait ran out after a.wait_ns, which records FTSP2_E_TIMEOUT, or another
// wait of this launch did): the producer then runs its remaining items in skip
// mode, without loads.
__device__ __forceinline__ bool wait_counter(const LayerArgs& a, const int* p, int target) {
    if (acquire_load(p) >= target) return true;
    const unsigned long long t0 = globaltimer();
    for (uint32_t it = 0;; ++it) {
        // a layer of a small instance ends within a few microseconds of the first
        // look: poll without pause at first, a few loads in flight, and acquire
        // once the count is there
        int v = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int x;
            asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(x) : "l"(p));
            v = max(v, x);
        }
        if (v >= target && acquire_load(p) >= target) return true;
        if (it >= 64) __nanosleep(128);
        if ((it & 7u) == 7u) {
            if (call_failed(a)) return false;
            if (globaltimer() - t0 > a.wait_ns) {
                record_timeout(a);
                return false;
            }
        }
    }
}

// ----------------------------------------------------------------------------------
// Work items.  The context warp of a CTA walks the unit's items (layer, tile),
// leaves out the inactive ones and describes each of the others to the roles of
// its CTA through a small ring in shared memory (ctx_full / ctx_empty): the
// coordinates of the TMA boxes, the dependency counter, and the constants and
// pointers of the final epilogue.  The description of an item takes a chain of
// three or four dependent global loads (tile, instance, layer constants), which
// the epilogue warps used to make themselves between the last MMA and the first
// state load of every tile (about 4000 of the 12000 clocks that a 32 x 32 block's
// epilogue took); here it is ready before the item starts.
// ----------------------------------------------------------------------------------
constexpr int kCtxSlots = 4;
struct __align__(16) ItemCtx {
    // final epilogue
    float* Z;                 // state slab of Z (blocked layout); A = Z + plane_elems
    long long doff;           // offset of D (last layer)
    float mul, bp, d, os;     // DevLayer constants
    float p, q, d2, g;
    float cdiag;              // last layer: f0, or 1 - f0 when flipped
    int simple;               // Eq. mlsp2 constants: d2 = 0, p = 1, q = 0
    int flip, dout;           // last layer: flipped output; D is written
    int n, nk, ck;            // order, K slices, K slices per accumulation chunk (nk = 0: end of the list)
    int row0, col0;           // first row of the CTA's block, first column of the tile
    int mirror;               // operands (c, r) are written too
    int inst;                 // instance
    // TMA producer
    int slab_row;             // first row of the instance's slab in the operand maps
    int chain, maps;          // chain; tensor-map set
    int panA, panB;           // first rows of the A panel and of the B panel that this CTA loads
    int lowA, lowB;           // K slices below: not stored there, loaded transposed from the upper triangle
    int same;                 // both panels are the same rows: B is read from A's planes
    // dependencies of multi-layer launches (null: none)
    const int* dep;           // completions of the previous layer of this instance and chain
    int target;
    int* done;                // this item's counter
    int first, final;         // first / last item of a unit that keeps its tile's state in TMEM
};

// Final epilogue of a non-last layer on the warp's rows R0 .. R0 + 31 (lane = row),
// one 32-column block at a time, of the blocks that touch the triangle and the
// order:
//   A_{k+1} = A_k + d_k Z_k (+ d2 xh),  Z_{k+1} = p xh + q A_k,  xh = mul S + bp Z_k,
// then the operands of Z_{k+1} (times the FP16 scale 2^e_{k+1}) for the next
// layer.  The state of the next block is loaded as soon as this one's is used (the
// first block's before the last chunk is waited for), so that its latency overlaps
// the chunk or the block's stores; a resident tile's state stays in TMEM columns
// of its own (kStateZ, kStateA).
// Operands of a block: staged plane by plane as rows of 64 bytes and written by
// TMA, one box of 32 rows x 64 bytes (two boxes of 16 columns for the 4-byte
// formats) at (r, c) and, where the next layer reads it, the transposed box at
// (c, r); a block on the diagonal is made symmetric in shared memory.  Rows and
// columns from n on are written as zeros.  The TMA unit writes 32 bytes a clock:
// 2000 clocks for the 64 KB of a 128 x 128 tile's FP16X2 operands.
constexpr int kStageBytes = 4096;                // operand staging of a store warp
constexpr int kStagingBytes = 32768;             // ... of the epilogue warps of layer_tc_kernel
constexpr int kStateZ = 256, kStateA = 384;      // TMEM columns of a resident tile's state

// State of row r, columns c .. c + 15 (c % 16 == 0): the 8-column groups below the
// order of a block that touches the triangle.
__device__ __forceinline__ void load16(const LayerArgs& a, const float* Zs, int n, int R0, int r, int c, float* z,
                                       float* x) {
    if (!(c < n && c + 15 >= R0)) return;            // warp-uniform
    const float* const Zg = Zs + state_off(a.P, r, c);
    ld_state8(Zg, z);
    ld_state8(Zg + a.plane_elems, x);
    if (c + 8 < n) {
        ld_state8(Zg + 256, z + 8);
        ld_state8(Zg + 256 + a.plane_elems, x + 8);
    }
}

// The planes of a split are formed one after the other, each rounded to nearest
// from what the planes before left of z (TF32X3: the low part too, since the tensor
// core would cut its low 13 bits): 32 columns of one plane as packed words (two
// columns a word for the 16-bit formats).
template <int FMT>
struct PlaneWords {
    static constexpr int ESZ = OpFmtT<FMT>::ESZ, N = 8 * ESZ;
    uint32_t w[N];
    __device__ __forceinline__ void round(const float (&v)[32]) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if constexpr (FMT == OP_F16X2) {
                const __half2 h = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
                w[i] = *reinterpret_cast<const uint32_t*>(&h);
            } else if constexpr (FMT == OP_BF16X3) {
                const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                w[i] = *reinterpret_cast<const uint32_t*>(&h);
            } else if constexpr (FMT == OP_TF32X3) {
                asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(w[i]) : "f"(v[i]));
            } else {
                w[i] = __float_as_uint(v[i]);
            }
        }
    }
    // v less the plane
    __device__ __forceinline__ void residual(float (&v)[32]) const {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if constexpr (FMT == OP_F16X2) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
                v[2 * i] -= f.x;
                v[2 * i + 1] -= f.y;
            } else if constexpr (FMT == OP_BF16X3) {
                v[2 * i] -= __uint_as_float(w[i] << 16);
                v[2 * i + 1] -= __uint_as_float(w[i] & 0xffff0000u);
            } else {
                v[i] -= __uint_as_float(w[i]);
            }
        }
    }
};

// The warp's staging: boxes of 32 rows x 64 bytes, written in turn, in the layout
// of TMA's 64-byte swizzle (the 16-byte chunk index is XORed with bits 1-2 of the
// row).  One or two boxes of its own, or, where the unit keeps one tile for all
// layers, its share of kRingBytes in the operand ring: its MMAs have all completed when the epilogue
// starts, and the loads of the next layer wait for the completions that the
// epilogue warps count after their stores.
constexpr int kRingBytes = 144 * 1024;
struct Stager {
    uint32_t base;                                   // boxes of 2 KB, 1024-byte aligned
    int lane, used;                                  // lane; boxes sent so far
    int cap;                                         // boxes
    __device__ __forceinline__ uint32_t box() const { return base + (uint32_t)(used % cap) * 2048u; }
    // the next box may be written: the store that last used it has read it
    __device__ __forceinline__ void next() const {
        if (used < cap) return;
        if (lane == 0) {
            if (cap == 2) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            else asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
        __syncwarp();
    }
    // 64 bytes of row `lane`, words w[0 .. 15]
    __device__ __forceinline__ void put_row(const uint32_t* w) const {
        const uint32_t at = box() + 64u * lane, x = 16u * ((lane >> 1) & 3);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + ((16u * j) ^ x)), "r"(w[4 * j]),
                         "r"(w[4 * j + 1]), "r"(w[4 * j + 2]), "r"(w[4 * j + 3])
                         : "memory");
    }
    // elements (u, col), u = from .. 31, of the words w of 32 elements
    template <int ESZ>
    __device__ __forceinline__ void put_column(int col, int from, const uint32_t* w) const {
        const uint32_t chunk = 16u * ((col * ESZ) >> 4), off = box() + ((col * ESZ) & 15);
#pragma unroll
        for (int u = 0; u < 32; ++u) {
            const uint32_t at = off + 64u * u + (chunk ^ (16u * ((u >> 1) & 3)));
            if (u >= from) {
                if constexpr (ESZ == 2)
                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(at), "h"((uint16_t)((u & 1) ? w[u / 2] >> 16 : w[u / 2]))
                                 : "memory");
                else asm volatile("st.shared.u32 [%0], %1;" ::"r"(at), "r"(w[u]) : "memory");
            }
        }
    }
    // the box is complete: write it at column x, row y of the plane
    __device__ __forceinline__ void send(const CUtensorMap* map, int x, int y) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                             reinterpret_cast<uint64_t>(map)),
                         "r"(box()), "r"(x), "r"(y)
                         : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        ++used;
    }
    // every store is complete; they and the warp's other stores may be published
    __device__ __forceinline__ void finish() {
        if (lane == 0) {
            asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
            asm volatile("fence.proxy.async.global;" ::: "memory");
        }
        used = 0;
    }
};

// Write one plane of the 32 x 32 block at (R0, c0); lane = row, words w.
template <int FMT>
__device__ __forceinline__ void store_plane(const CUtensorMap* map, Stager& st, int R0, int c0, int slab_row,
                                            bool mirror, const PlaneWords<FMT>& pw) {
    constexpr int ESZ = OpFmtT<FMT>::ESZ;
    constexpr int BOXES = ESZ == 4 ? 2 : 1, BC = 32 / BOXES;   // boxes per plane, their columns
    const bool diag = R0 == c0;
#pragma unroll
    for (int h = 0; h < BOXES; ++h) {
        st.next();
        st.put_row(pw.w + 16 * h);
        if (diag) {
            // a block on the diagonal: the part below it from the part above
            __syncwarp();
            if (BOXES == 1 || (st.lane >> 4) == h) st.put_column<ESZ>(st.lane - h * BC, st.lane + 1, pw.w);
        }
        st.send(map, c0 + h * BC, slab_row + R0);
    }
    if (mirror && !diag) {
#pragma unroll
        for (int h = 0; h < BOXES; ++h) {
            st.next();
            if (BOXES == 1 || (st.lane >> 4) == h) st.put_column<ESZ>(st.lane - h * BC, 0, pw.w);
            st.send(map, R0 + h * BC, slab_row + c0);
        }
    }
}

// The state of 16 H columns of a row, loaded ahead.
template <int H>
struct State {
    float z[H][16], x[H][16];
};
using State32 = State<2>;

// One 32 x 32 block: v holds the sums S of the lane's row, s the state of its 32
// columns (H = 2) or of the first 16 (H = 1).  After the use of half h the same half
// of the next block (at column c_next; -1: none) is loaded (H = 2), or fetch(h) loads
// the second half of this block (h = 0) and the first one of the next (h = 1).
template <int FMT, bool CAN_RESIDE, int H, class Fetch>
__device__ __forceinline__ void epi_block32(const LayerArgs& a, const ItemCtx& c, const CUtensorMap* wmaps, Stager& st,
                                            int R0, int c0, uint32_t tstate, bool from_tmem, bool to_tmem,
                                            float (&v)[32], State<H>& s, int c_next, Fetch&& fetch) {
    constexpr int NPL = OpFmtT<FMT>::NPL;
    const int n = c.n, r = R0 + st.lane;
    const float mul = c.mul, bp = c.bp, d = c.d;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int cc = c0 + 16 * h, hs = H == 2 ? h : 0;
        if (cc < n) {
            if (CAN_RESIDE && from_tmem) {
                tmem_ld16(tstate + 16 * h, reinterpret_cast<uint32_t*>(s.z[hs]));
                tmem_ld16(tstate + (kStateA - kStateZ) + 16 * h, reinterpret_cast<uint32_t*>(s.x[hs]));
                tmem_wait_ld();
            }
            if (c.simple) {
                // Eq. mlsp2: d2 = 0, p = 1, q = 0
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    v[16 * h + u] = fmaf(mul, v[16 * h + u], bp * s.z[hs][u]);
                    s.x[hs][u] = fmaf(d, s.z[hs][u], s.x[hs][u]);
                }
            } else {
                const float d2 = c.d2, p1 = c.p, q1 = c.q;
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    const float xh = fmaf(mul, v[16 * h + u], bp * s.z[hs][u]);
                    const float an = fmaf(d2, xh, fmaf(d, s.z[hs][u], s.x[hs][u]));
                    v[16 * h + u] = fmaf(p1, xh, q1 * s.x[hs][u]);
                    s.x[hs][u] = an;
                }
            }
            if (CAN_RESIDE && to_tmem) {
                tmem_st16(tstate + 16 * h, v + 16 * h);
                tmem_st16(tstate + (kStateA - kStateZ) + 16 * h, s.x[hs]);
            } else if (r < n) {
                float* const Zg = c.Z + state_off(a.P, r, cc);
                store_state8(Zg, v + 16 * h);
                store_state8(Zg + a.plane_elems, s.x[hs]);
                if (cc + 8 < n) {
                    store_state8(Zg + 256, v + 16 * h + 8);
                    store_state8(Zg + 256 + a.plane_elems, s.x[hs] + 8);
                }
            }
        }
        if constexpr (H == 2) {
            if (!from_tmem && c_next >= 0) load16(a, c.Z, n, R0, r, c_next + 16 * h, s.z[h], s.x[h]);
        } else {
            fetch(h);
        }
    }
    if (!(R0 + 31 < n && c0 + 31 < n)) {
        // zeros in the padding
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] = r < n && c0 + u < n ? v[u] : 0.f;
    }
    if constexpr (FMT == OP_F16X2) {
        const float os = c.os;
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] *= os;
    }
    const bool mirror = c.mirror != 0;
#pragma unroll
    for (int p = 0; p < NPL; ++p) {
        PlaneWords<FMT> pw;
        pw.round(v);
        store_plane<FMT>(wmaps + p, st, R0, c0, c.slab_row, mirror, pw);
        if (p + 1 < NPL) pw.residual(v);
    }
}

// Last layer on the warp's 32 x COLS block, 8 columns at a time: G = A + d Z + g xh with
// xh = mul v + bp Z (Eq. mlsp2: A_L + Z_L, A_L = A_{L-1} + d Z_{L-1},
// Z_L = a v + b' Z_{L-1}; Skip-SP2: A_L + gamma_L x_L), then D = G + f0 I (or
// (1 - f0) I - G when flipped) at (r, c) and (c, r), and the sums of the
// diagonal and of the squares of G.  The diagonal element is added in FP64.  A
// group's 8 squares are summed without rounding error in pairs of FP32 numbers
// (the product's error by an FMA, each addition's by TwoSum, Knuth), the high
// part is added in FP64 and the low part in FP32 into `lo`, which is added once
// per block: per-element FP64 arithmetic would run on the FP64 pipe, the slowest
// unit of this GPU.  The direct row (r, c .. c + 7) is written as two 16-byte
// vectors when the whole group lies in the triangle and is aligned; the mirror
// (c, r) is one element per lane, a contiguous run of row c across the warp.
struct LastSums {
    double tr, sq;
    float lo;
};
template <int COLS>
__device__ __forceinline__ void epi_last(const LayerArgs& a, const ItemCtx& c, int R0, int lane, int c0,
                                         const float* v, const float* zs, const float* xs, LastSums& b) {
    const int n = c.n, r = R0 + lane;
    const float mul = c.mul, bp = c.bp, d = c.d, g1 = c.g, cdiag = c.cdiag;
    const bool flip = c.flip != 0, dout = c.dout != 0;
    float* const Db = a.D + c.doff;
    float* const drow = Db + (int64_t)r * n;
    if (r >= n) return;
    double tr = b.tr, sq = b.sq;
    float lo = b.lo;
#pragma unroll
    for (int h = 0; h < COLS / 8; ++h) {
        const int cc0 = c0 + 8 * h;
        if (cc0 >= n) break;
        float dv[8];
        float sh = 0.f, sl = 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int cc = cc0 + u;
            const float z = zs[8 * h + u], x = xs[8 * h + u];
            const float g = fmaf(g1, fmaf(mul, v[8 * h + u], bp * z), fmaf(d, z, x));
            const bool diag = r == cc;
            if (flip) dv[u] = (diag ? cdiag : 0.f) - g;
            else dv[u] = g + (diag ? cdiag : 0.f);
            if (cc < n && r <= cc) {
                if (diag) tr += (double)g;
                const float w = diag ? g : 2.f * g;            // (r, c) and (c, r)
                const float p = __fmul_rn(w, g);
                const float pe = fmaf(w, g, -p);               // w g - p, exact
                const float t = __fadd_rn(sh, p);
                const float bb = __fsub_rn(t, sh);
                const float te = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bb)), __fsub_rn(p, bb));   // sh + p - t, exact
                sh = t;
                sl = __fadd_rn(sl, __fadd_rn(te, pe));
            }
        }
        sq += (double)sh;
        lo = __fadd_rn(lo, sl);
        if (!dout) continue;
        if (cc0 >= r && cc0 + 8 <= n && (reinterpret_cast<uintptr_t>(drow + cc0) & 15u) == 0) {
            reinterpret_cast<float4*>(drow + cc0)[0] = make_float4(dv[0], dv[1], dv[2], dv[3]);
            reinterpret_cast<float4*>(drow + cc0)[1] = make_float4(dv[4], dv[5], dv[6], dv[7]);
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (cc0 + u < n && r <= cc0 + u) drow[cc0 + u] = dv[u];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (cc0 + u < n && r < cc0 + u) Db[(int64_t)(cc0 + u) * n + r] = dv[u];
    }
    b.tr = tr;
    b.sq = sq;
    b.lo = lo;
}

// L2 prefetch of the Z and A state that the CTA's epilogue warps read at the
// end of an item: 128 rows from row0, columns from the diagonal (or the tile's
// first column) to the order n; each 32-row block row of the blocked layout is
// one contiguous run.  Issued by the TMA producer a few K-slices before the
// tile ends.
template <int TN>
__device__ __forceinline__ void prefetch_state(const LayerArgs& a, const float* Z, int row0, int col0, int n) {
    const int cend = min(n, col0 + TN);
#pragma unroll 1
    for (int R = row0; R < row0 + kCtaRows && R < n; R += 32) {
        const int cs = max(col0, R) & ~7;
        if (cs >= cend) continue;
        const uint32_t bytes = (uint32_t)((cend - cs + 7) / 8) * 1024u;
        const float* const src = Z + state_off(a.P, R, cs);
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src + a.plane_elems), "r"(bytes) : "memory");
    }
}

template <int MODE, int SHAPE>
struct Stage {
    using C = TcCfg<MODE>;
    static constexpr int APLANE = kCtaRows * 128;              // bytes of one 128-byte K slice of the A panel
    static constexpr int BPLANE = Geo<SHAPE>::BROWS * 128;
    static constexpr int BYTES = C::NSPLIT * (APLANE + BPLANE);
    // as many stages as fit beside the operand staging of the epilogue warps:
    // 192 KB, or 144 KB (BF16X3 on 256 x 128 tiles; 216 KB where the staging is
    // in the ring)
    static constexpr int N = (192 * 1024) / BYTES;
    static constexpr int NMAX = (222 * 1024) / BYTES;
    static constexpr int SMEM = NMAX * BYTES > N * BYTES + kStagingBytes ? NMAX * BYTES : N * BYTES + kStagingBytes;
    static_assert(N * BYTES >= kRingBytes, "ring staging");
};

// Blocks of the deferred epilogue: block e of a tile is the half e & 1 of the
// 32 x 64 sums of accumulating warp 2 + e / 2, i.e. 32 rows x 32 columns; those
// that touch the triangle and the order are written.  Store warp sw takes the
// warps' sums sw, sw + kStoreWarps, ...
struct DeferBlock {
    int R0, c0;
    bool live;
};
__device__ __forceinline__ DeferBlock defer_block(const ItemCtx& c, int e) {
    const int i = e >> 1;
    DeferBlock d;
    d.R0 = c.row0 + ((i + 2) & 3) * 32;
    d.c0 = c.col0 + (i >> 2) * 64 + (e & 1) * 32;
    d.live = d.c0 >= d.R0 && d.c0 < c.n && d.R0 < c.n;
    return d;
}
__device__ __forceinline__ bool next_block(const ItemCtx& c, int sw, int& e) {
    // e = 2 i + half with i = sw, sw + kStoreWarps, ...
    for (;;) {
        e = e < 0 ? 2 * sw : (e & 1) ? e - 1 + 2 * kStoreWarps : e + 1;
        if (e >= 2 * kDeferWarps) return false;
        if (defer_block(c, e).live) return true;
    }
}

// What the final epilogue of tile tl needs: instance w, layer constants L.
template <int MODE, int OUTFMT, int SHAPE>
__device__ __forceinline__ void fill_epilogue(const LayerArgs& a, const Tile& tl, const InstWork& w, const DevLayer& L,
                                              int rank, ItemCtx& c) {
    using G = Geo<SHAPE>;
    c.Z = a.Z[tl.chain] + (size_t)tl.inst * a.P * a.P;
    c.os = OUTFMT == OP_F16X2 ? L.out_scale : 1.f;
    c.mul = MODE == FTSP2_FP16X2 ? L.acc_mul : L.a;
    c.bp = L.bp;
    c.d = L.d;
    c.p = L.p;
    c.q = L.q;
    c.d2 = L.d2;
    c.g = L.g;
    c.simple = L.d2 == 0.f && L.p == 1.f && L.q == 0.f;
    c.doff = w.doff;
    c.cdiag = w.cdiag;
    c.flip = w.flip;
    c.dout = a.chain_kind[tl.chain] == CHAIN_FERMI && a.D != nullptr;
    c.n = w.n;
    c.row0 = tl.I * G::TM + rank * kCtaRows;
    c.col0 = tl.J * G::TN;
    c.mirror = a.mirror_all || (tl.J * G::TN) / G::TM == tl.I;   // inside the diagonal block, or everywhere
    c.inst = tl.inst;
    c.slab_row = tl.inst * a.P;
}

template <int MODE, int OUTFMT, int SHAPE>
__global__ void __launch_bounds__((tc_threads<OUTFMT, SHAPE>()), 1)
    layer_tc_kernel(const __grid_constant__ LayerArgs a, const __grid_constant__ TmaMaps maps0,
                    const __grid_constant__ TmaMaps maps1, const __grid_constant__ WriteMaps wmaps0,
                    const __grid_constant__ WriteMaps wmaps1) {
    using C = TcCfg<MODE>;
    using G = Geo<SHAPE>;
    using St = Stage<MODE, SHAPE>;
    constexpr bool PAIR = G::NCTA == 2;
    constexpr bool LAST = OUTFMT == kLastLayer;
    constexpr int TM = G::TM, TN = G::TN;
    constexpr int EW = epi_warps<OUTFMT, SHAPE>(), CTX_WARP = 2 + EW;
    constexpr int EPI_COLS = TN / (EW / 4);            // columns per epilogue warp
    constexpr int BKE = 128 / C::ESIZE;                // K elements per 128-byte slice
    constexpr int KSTEPS = 4;                          // 128-byte slice / 32 bytes per MMA
    constexpr uint32_t IDESC = make_idesc(C::ATYPE, TM, TN);
    constexpr uint32_t TMEM_COLS = 512;
    // a unit that keeps its tile's state in TMEM has two chunk buffers there
    constexpr bool CAN_RESIDE = TN <= 128 && !LAST;

    // A launch whose layers all lie below the first layer any instance starts
    // at (models with fewer layers than the set's maximum start late) has no
    // active item: every thread of both CTAs of a pair leaves at once.
    grid_wait();
    const int first_layer = *reinterpret_cast<volatile const int*>(a.status + 1);
    if (a.gl + a.nlayers <= first_layer) return;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full_bar[St::NMAX];
    __shared__ __align__(8) uint64_t empty_bar[St::NMAX];
    __shared__ __align__(8) uint64_t tfull_bar[G::NBUF];
    __shared__ __align__(8) uint64_t tempty_bar[G::NBUF];
    __shared__ __align__(8) uint64_t ctx_full[kCtxSlots];
    __shared__ __align__(8) uint64_t ctx_empty[kCtxSlots];
    __shared__ ItemCtx ctx[kCtxSlots];
    // drain: the MMA issuer's last commit (all of its MMAs complete)
    __shared__ __align__(8) uint64_t drain_bar;
    __shared__ uint32_t tmem_slot;
    // skip mode: set once this CTA has seen the call fail; the roles then keep
    // the barrier protocol of their work items without loads or stores
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? cluster_rank() : 0u;
    const int unit = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;     // pair or CTA
    const int nunits = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
    const bool resident = CAN_RESIDE && a.resident != 0;
    const int nbuf = resident ? kStateZ / TN : G::NBUF;
    const int nst = (resident || LAST) ? St::NMAX : St::N;     // stages of the operand ring
    if (threadIdx.x == 0) {
        for (int s = 0; s < St::NMAX; ++s) {
            mbar_init(&full_bar[s], G::NCTA);      // one expect_tx arrival per CTA
            mbar_init(&empty_bar[s], 1);
        }
        for (int s = 0; s < G::NBUF; ++s) {
            mbar_init(&tfull_bar[s], 1);
            mbar_init(&tempty_bar[s], G::NCTA * EW);
        }
        for (int s = 0; s < kCtxSlots; ++s) {
            mbar_init(&ctx_full[s], 1);
            // read by the epilogue warps, the producer and, on the even CTA, the MMA issuer
            mbar_init(&ctx_empty[s], EW + 1 + (rank == 0 ? 1 : 0));
        }
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        if constexpr (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&tmem_slot)),
                         "r"(TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&tmem_slot)),
                         "r"(TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == CTX_WARP) {
        // ---------------- context warp: the unit's active items ----------------
        // 32 items are looked up at a time, a lane each (a model with few layers
        // starts late: many items of a ragged batch are inactive).
        const int nf = a.ntiles * a.nlayers;
        // the items of layers before the first active one are left out
        const int f0 = max(0, first_layer - a.gl) * a.ntiles + unit;
        int it = 0;
        bool ok = true;
        for (int fb = f0; fb < nf && ok; fb += 32 * nunits) {
            const int f = fb + lane * nunits;
            const int l = f / a.ntiles, g = a.gl + l, t = f - l * a.ntiles;
            Tile tl = {0, 0, 0, 0};
            int k = -1;
            if (f < nf) {
                tl = a.tiles[t];
                const InstWork& w = a.iw[tl.inst];
                if (w.active) k = g - ((w.start_layer >> (16 * tl.chain)) & 0xffff);
            }
            unsigned active = __ballot_sync(0xffffffffu, k >= 0);
            for (; active && ok; active &= active - 1) {
                if (lane == __ffs(active) - 1) {
                    const InstWork& w = a.iw[tl.inst];
                    const DevLayer L = a.layers[w.layer_off[tl.chain] + k];
                    const int slot = it % kCtxSlots;
                    ok = wait_bar(&ctx_empty[slot], ((it / kCtxSlots) & 1) ^ 1u, a);
                    if (ok) {
                        ItemCtx& c = ctx[slot];
                        const int odd = l & 1;
                        fill_epilogue<MODE, OUTFMT, SHAPE>(a, tl, w, L, (int)rank, c);
                        const int n = c.n;
                        c.nk = (n + BKE - 1) / BKE;
                        const int ce = g >= a.tail_from ? a.chunk_tail : a.chunk_elems;
                        c.ck = max(1, (ce > 0 ? ce : C::CK * BKE) / BKE);
                        const int blkB = (tl.J * TN) / TM;             // diagonal block of the B panel
                        c.chain = tl.chain;
                        c.maps = odd;
                        c.panA = c.row0;
                        c.panB = c.col0 + (int)rank * G::BROWS;
                        c.lowA = (!C::TF32 && a.lower_t) ? tl.I * TM / BKE : 0;
                        c.lowB = (!C::TF32 && a.lower_t) ? blkB * TM / BKE : 0;
                        c.same = SHAPE == SHAPE_SINGLE && tl.I == tl.J;
                        // operands and state written by other CTAs of this launch
                        const bool dep = g > a.gl && k > 0;
                        c.dep = dep ? inst_counter(a, g - 1, tl.inst, tl.chain) : nullptr;
                        c.target = EW * G::NCTA * w.tile_count[a.dtab][tl.chain] + (g == a.stall_layer ? 1 : 0);
                        c.done = inst_counter(a, g, tl.inst, tl.chain);
                        c.first = it == 0;
                        c.final = l == a.nlayers - 1;
                        mbar_arrive(&ctx_full[slot]);
                    }
                }
                ok = __all_sync(0xffffffffu, ok);
                ++it;
            }
        }
        if (lane == 0) {
            const int slot = it % kCtxSlots;
            if (ok && wait_bar(&ctx_empty[slot], ((it / kCtxSlots) & 1) ^ 1u, a)) {
                ctx[slot].nk = 0;                    // the end of the list
                mbar_arrive(&ctx_full[slot]);
            }
        }
        __syncwarp();
    } else if (warp == 0) {
        // ---------------- TMA producer ----------------
        // The whole warp runs the loop and one elected lane issues (coordinates,
        // maps and barriers are uniform values): issued from a single-lane loop a
        // copy took some 150 clocks, six to eight of them a K-slice.
        const bool leader = elect_one();
        int stage = 0;
        uint32_t phase = 0;
        uint64_t known0 = 0, known1 = 0;         // per chain: predecessor known complete
        bool skip = false;                       // the call has failed: no more loads
        bool broken = false;                     // a pipeline wait ran out twice
        const uint32_t smem0 = uniform32(smem_u32(smem));
        const uint32_t full0 = uniform32(PAIR ? map_to(smem_u32(&full_bar[0]), 0) : smem_u32(&full_bar[0]));
        for (int it = 0; !broken; ++it) {
            const int slot = it % kCtxSlots;
            if (!all_wait(&ctx_full[slot], (it / kCtxSlots) & 1, a)) {
                broken = true;
                break;
            }
            const ItemCtx& c = ctx[slot];
            const int nk = uniform32(c.nk);
            if (nk == 0) break;
            const int lowA = uniform32(c.lowA), lowB = uniform32(c.lowB), panA = uniform32(c.panA),
                      panB = uniform32(c.panB), slab = uniform32(c.slab_row), chain = uniform32(c.chain);
            const int row0 = c.row0, col0 = c.col0, n = c.n, target = c.target;
            const bool same = SHAPE == SHAPE_SINGLE && uniform32(c.same) != 0;
            const uint64_t dep = reinterpret_cast<uint64_t>(c.dep);
            const float* const Z = c.Z;
            const TmaMaps& maps = uniform32(c.maps) ? maps1 : maps0;
            __syncwarp();
            if (leader) local_arrive(smem_u32(&ctx_empty[slot]));
            if (!skip && dep && dep != (chain ? known1 : known0)) {
                // wait for the previous layer of the item's own instance only,
                // so a small instance need not wait for a large one
                bool done = true;
                if (leader) {
                    done = wait_counter(a, reinterpret_cast<const int*>(dep), target);
                    if (done) asm volatile("fence.proxy.async.global;" ::: "memory");
                }
                if (__all_sync(0xffffffffu, done)) {
                    if (chain) known1 = dep;
                    else known0 = dep;
                } else {
                    skip = true;
                }
            }
            if (skip && leader) *reinterpret_cast<volatile int*>(&abort_flag) = 1;
            for (int kb = 0; kb < nk; ++kb) {
                // K-slices left of a panel's diagonal block: not stored below
                // the diagonal, loaded from the transposed upper block
                const bool tA = kb < lowA, tB = kb < lowB;
                if (!all_wait(&empty_bar[stage], phase ^ 1u, a)) {
                    broken = true;
                    break;
                }
                if (leader) {
                    const uint32_t fb = full0 + 8u * stage;
                    if (skip) {
                        // the stage's arrival without data: the phase completes
                        // with the peer's loads (if any), and the sums of the MMAs
                        // that read it are not used
                        if constexpr (PAIR) remote_arrive(fb);
                        else local_arrive(fb);
                    } else {
                        if (!resident && kb == max(0, nk - 3)) prefetch_state<TN>(a, Z, row0, col0, n);
                        const uint32_t bytes = same ? C::NSPLIT * St::APLANE : St::BYTES;
                        if constexpr (PAIR) remote_expect_tx(fb, bytes);
                        else local_expect_tx(fb, bytes);
                        auto load = [&](uint32_t dst, const CUtensorMap* m, int x, int y) {
                            if constexpr (PAIR) tma_load_pair(dst, m, fb, x, y);
                            else tma_load_one(dst, m, fb, x, y);
                        };
                        const uint32_t sb = smem0 + stage * St::BYTES;
                        const int kx = kb * BKE, ky = slab + kb * BKE;
#pragma unroll
                        for (int s = 0; s < C::NSPLIT; ++s) {
                            const uint32_t dA = sb + s * St::APLANE;
                            const uint32_t dB = sb + C::NSPLIT * St::APLANE + s * St::BPLANE;
                            if (tA) {
                                load(dA, &maps.t[chain][s], panA, ky);
                                load(dA + 8192, &maps.t[chain][s], panA + 64, ky);
                            } else {
                                load(dA, &maps.a[chain][s], kx, slab + panA);
                            }
                            if (same) continue;
                            if (tB) {
                                load(dB, &maps.t[chain][s], panB, ky);
                                if constexpr (G::BROWS == 128) load(dB + 8192, &maps.t[chain][s], panB + 64, ky);
                            } else {
                                // a panel of 64 rows: the 64-row box
                                load(dB, G::BROWS == 128 ? &maps.a[chain][s] : &maps.t[chain][s], kx, slab + panB);
                            }
                        }
                    }
                }
                __syncwarp();
                if (++stage == nst) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
        if (broken) {
            // The barrier protocol failed, so the completion of the loads
            // already issued cannot be observed: give them a bounded grace
            // period (a load of one stage takes microseconds) before the
            // CTA releases its shared memory.
            *reinterpret_cast<volatile int*>(&abort_flag) = 1;
            const unsigned long long t0 = globaltimer();
            while (globaltimer() - t0 < 2000000ull) __nanosleep(1000);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (rank == 0) {
            // ---------------- MMA issuer (the even CTA of a pair) ----------------
            // The whole warp runs the loop and one elected lane issues: loop state
            // and descriptors are then uniform values.  With the loop in a single
            // lane every descriptor went through vector registers, and the issue of
            // a 128-column MMA took 110 clocks for the 64 that it runs.
            // On single CTAs the completed waits of the next slice (and of the next
            // chunk's buffer) are seen while this slice's last products are queued:
            // a completed wait, the choice of the descriptors and a commit each take
            // 100 to 150 clocks of this warp, 900 a slice where a chunk is one
            // slice.  Ragged batch 22.12 -> 21.85 ms, 60 fragments 380 -> 373 us;
            // on pairs, whose producer is rarely a slice ahead, the extra look
            // cost 1.6 % (n = 1501) and 3.5 % (n = 2048 TF32X3).
            const bool leader = elect_one();
            int stage = 0;
            uint32_t phase = 0;
            int buf = 0;
            uint32_t aphase = 0;
            bool ok = true;
            // descriptors differ only in the start-address field (bits 0-13,
            // address >> 4); all operand slices lie inside this CTA's window
            const uint64_t desc0 = uniform64(sdesc_sw128(smem_u32(smem)));
            const uint64_t descT = uniform64(sdesc_mn_sw128(smem_u32(smem)));   // transposed panels
            const uint32_t tm = uniform32(tmem);
            for (int it = 0; ok; ++it) {
                const int slot = it % kCtxSlots;
                if (!all_wait(&ctx_full[slot], (it / kCtxSlots) & 1, a)) break;
                const ItemCtx& c = ctx[slot];
                const int nk = uniform32(c.nk);
                if (nk == 0) break;
                const int ck = uniform32(c.ck), lowA = uniform32(c.lowA), lowB = uniform32(c.lowB);
                const bool same = SHAPE == SHAPE_SINGLE && uniform32(c.same) != 0;
                if (leader) local_arrive(smem_u32(&ctx_empty[slot]));
                bool have_full = false, have_buf = false;
                for (int kc = 0; kc < nk && ok; kc += ck) {
                    if (!have_buf && !all_wait(&tempty_bar[buf], aphase ^ 1u, a)) {
                        ok = false;
                        break;
                    }
                    have_buf = false;
                    const uint32_t dt = tm + (uint32_t)(buf * TN);
                    const int kend = min(nk, kc + ck);
                    const int nbuf_next = buf + 1 == nbuf ? 0 : buf + 1;
                    const uint32_t aphase_next = nbuf_next == 0 ? aphase ^ 1u : aphase;
                    for (int kb = kc; kb < kend; ++kb) {
                        if (!have_full && !all_wait(&full_bar[stage], phase, a)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        // In skip mode the stage holds no new data; its MMAs only keep
                        // the protocol, their sums are not used.
                        // The producer's classification of this K-slice (transposed
                        // panels: MN-major operand, K steps of two 1 KB atoms per 64 columns)
                        const bool tA = kb < lowA, tB = kb < lowB;
                        const uint32_t so = (uint32_t)((stage * St::BYTES) >> 4);
                        const uint64_t baseA = (tA ? descT : desc0) + so, baseB = (tB ? descT : desc0) + so;
                        const uint32_t idesc = IDESC | (tA ? 1u << 15 : 0u) | (tB ? 1u << 16 : 0u);
                        const uint32_t stepA = tA ? 2048u >> 4 : 32u >> 4, stepB = tB ? 2048u >> 4 : 32u >> 4;
                        const uint32_t planeB = (same ? 0 : C::NSPLIT * St::APLANE) >> 4;
                        const uint32_t strideB = (same ? St::APLANE : St::BPLANE) >> 4;
                        // The small products (index sum >= 1) of the slice go first and
                        // the leading one (p = 0) last: in a chunk's first slice the
                        // small products are added while the accumulator holds only
                        // small values, so fewer additions land on a large partial sum
                        // (the tensor core's FP32 accumulation is not round-to-nearest).
                        // Measured: 15-30 % smaller errors in D and S at the same speed.
                        auto product = [&](int p) {
#pragma unroll
                            for (int kk = 0; kk < KSTEPS; ++kk) {
                                const uint64_t da = baseA + (uint32_t)(prod_a(p) * (St::APLANE >> 4)) + kk * stepA;
                                const uint64_t db = baseB + planeB + prod_b(p) * strideB + kk * stepB;
                                const uint32_t accum = (kk == 0 && p == C::NPROD - 1) ? (kb == kc ? 0u : 1u) : 1u;
                                if constexpr (PAIR) umma_pair<C::TF32>(dt, da, db, idesc, accum);
                                else umma_one<C::TF32>(dt, da, db, idesc, accum);
                            }
                        };
                        if (leader) {
#pragma unroll
                            for (int p = C::NPROD - 1; p > 0; --p) product(p);
                        }
                        const int stage_next = stage + 1 == nst ? 0 : stage + 1;
                        const uint32_t phase_next = stage_next == 0 ? phase ^ 1u : phase;
                        if constexpr (!PAIR) {
                            have_full = kb + 1 < nk &&
                                        __all_sync(0xffffffffu, try_wait_cluster(&full_bar[stage_next], phase_next));
                            if (kb + 1 == kend && kend < nk)
                                have_buf = __all_sync(0xffffffffu,
                                                      try_wait_cluster(&tempty_bar[nbuf_next], aphase_next ^ 1u));
                        }
                        if (leader) {
                            product(0);
                            if constexpr (PAIR) umma_commit_pair(smem_u32(&empty_bar[stage]));
                            else umma_commit_one(smem_u32(&empty_bar[stage]));
                            if (kb == kend - 1) {
                                if constexpr (PAIR) umma_commit_pair(smem_u32(&tfull_bar[buf]));
                                else umma_commit_one(smem_u32(&tfull_bar[buf]));
                            }
                        }
                        __syncwarp();
                        stage = stage_next;
                        phase = phase_next;
                    }
                    if (!ok) break;
                    buf = nbuf_next;
                    aphase = aphase_next;
                }
            }
            // Drain: every MMA this warp issued (they write TMEM of both CTAs
            // of a pair and read both CTAs' stages) has completed before the
            // final barrier, after which the CTAs free TMEM and shared memory.
            if (leader) {
                if constexpr (PAIR) umma_commit_local_pair(smem_u32(&drain_bar));
                else umma_commit_one(smem_u32(&drain_bar));
            }
            __syncwarp();
            if (!all_wait(&drain_bar, 0, a)) {
                const unsigned long long t0 = globaltimer();
                while (globaltimer() - t0 < 2000000ull) __nanosleep(1000);
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue (warps 2 .. 1 + EW) ----------------
        const int q = warp & 3;                  // TMEM lane quarter
        const int cq = (warp - 2) >> 2;          // column group of the tile
        // "tempty" barriers of the even CTA (consecutive 8-byte words)
        const uint32_t tempty0 = PAIR ? map_to(smem_u32(&tempty_bar[0]), 0) : smem_u32(&tempty_bar[0]);
        const uint32_t tlane = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cq * EPI_COLS);
        constexpr int RING_BOXES = kRingBytes / EW / 2048, BOXES = kStagingBytes / EW / 2048;
        Stager st{resident ? smem_u32(smem) + (uint32_t)((warp - 2) * (RING_BOXES * 2048))
                           : smem_u32(smem + St::N * St::BYTES) + (uint32_t)((warp - 2) * (BOXES * 2048)),
                  lane, 0, resident ? RING_BOXES : BOXES};
        int buf = 0;
        uint32_t aphase = 0;
        auto release = [&]() {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if constexpr (PAIR) remote_arrive(tempty0 + 8u * (uint32_t)buf);
                else local_arrive(tempty0 + 8u * (uint32_t)buf);
            }
            if (++buf == nbuf) {
                buf = 0;
                aphase ^= 1u;
            }
        };
        bool ok = true;
        for (int it = 0; ok; ++it) {
            const int slot = it % kCtxSlots;
            if (!wait_bar(&ctx_full[slot], (it / kCtxSlots) & 1, a)) break;
            const ItemCtx& c = ctx[slot];
            const int nk = c.nk;
            if (nk == 0) break;
            const int n = c.n, nch = (nk + c.ck - 1) / c.ck;
            const int R0 = c.row0 + q * 32, C0 = c.col0 + cq * EPI_COLS;
            // the 32-column blocks that touch the triangle and the order: [cb0, cb1)
            const int cb0 = max(0, min(EPI_COLS, R0 - C0)), cb1 = R0 < n ? max(0, min(EPI_COLS, (n - C0 + 31) & ~31)) : 0;
            const bool live = cb0 < cb1;
            const int* const dep = resident ? nullptr : c.dep;
            // the state of the first block, loaded ahead of the last chunk
            constexpr int AH = EW == 16 ? 1 : 2;
            State<AH> ahead;
            const bool state_global = live && (!resident || c.first);
            auto load_first = [&](State<AH>& s) {
#pragma unroll
                for (int h = 0; h < AH; ++h) load16(a, c.Z, n, R0, R0 + lane, C0 + cb0 + 16 * h, s.z[h], s.x[h]);
            };
            // Chunk drain: every chunk is added into acc and its buffer released.
            // The columns of a 256-column tile's warp leave no registers for
            // the final epilogue: there the finished sum is written back into the
            // last chunk's buffer, which stays held, and read from it block by
            // block; the MMAs of the next tile meanwhile fill the other buffer.
            constexpr bool HOLD = TN > 128;
            float acc[EPI_COLS];
#pragma unroll
            for (int i = 0; i < EPI_COLS; ++i) acc[i] = 0.f;
            for (int j = 0; j < nch; ++j) {
                if (!HOLD && j > 0 && j == nch - 1 && state_global) load_first(ahead);
                if (!wait_bar(&tfull_bar[buf], aphase, a)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                if (j == 0 && dep) {
                    // the state of the previous layer, written by other CTAs
                    if (lane == 0) acquire_load(dep);
                    __syncwarp();
                }
                if (!HOLD && nch == 1 && state_global) load_first(ahead);
                const uint32_t ta = tlane + (uint32_t)(buf * TN);
                if (live) {
                    constexpr int W = HOLD ? 8 : 16;
#pragma unroll
                    for (int g = 0; g < EPI_COLS / W; ++g) {
                        uint32_t v[W];
                        if constexpr (HOLD) tmem_ld8(ta + W * g, v);
                        else tmem_ld16(ta + W * g, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int jj = 0; jj < W; ++jj) acc[W * g + jj] += __uint_as_float(v[jj]);
                    }
                    if (HOLD && j == nch - 1) {
#pragma unroll
                        for (int g = 0; g < EPI_COLS / 16; ++g) tmem_st16(ta + 16 * g, &acc[16 * g]);
                        tmem_wait_st();
                    }
                }
                if (HOLD && j == nch - 1) break;
                release();
            }
            if (!ok) break;
            // skip mode (warp-uniform): the protocol without the memory work
            const bool work = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&abort_flag) == 0 ? 1 : 0, 0) != 0;
            const bool from_tmem = CAN_RESIDE && resident && !c.first, to_tmem = CAN_RESIDE && resident && !c.final;
            // every block of the warp: its sums in v, the state loaded ahead in s
            auto blocks = [&](auto&& block) {
                if constexpr (HOLD) {
                    State<AH> s;
                    load_first(s);
                    const uint32_t tfin = tlane + (uint32_t)(buf * TN);
#pragma unroll 1
                    for (int cb = cb0; cb < cb1; cb += 32) {
                        float v[32];
                        tmem_ld32(tfin + cb, reinterpret_cast<uint32_t*>(v));
                        tmem_wait_ld();
                        block(cb, v, s);
                    }
                } else {
                    float(&v0)[32] = *reinterpret_cast<float(*)[32]>(acc);
                    if constexpr (EPI_COLS == 32) {
                        block(0, v0, ahead);
                        return;
                    }
                    float(&v1)[32] = *reinterpret_cast<float(*)[32]>(acc + EPI_COLS - 32);
                    if (cb0 == 0) block(0, v0, ahead);
                    if (cb1 == EPI_COLS) block(EPI_COLS - 32, v1, ahead);
                }
            };
            auto next_of = [&](int cb) { return cb + 32 < cb1 ? C0 + cb + 32 : -1; };
            if constexpr (!LAST) {
                if (live && work) {
                    const CUtensorMap* const wm = (c.maps ? wmaps1 : wmaps0).w[c.chain];
                    blocks([&](int cb, float (&v)[32], State<AH>& s) {
                        const int cn = next_of(cb);
                        epi_block32<OUTFMT, CAN_RESIDE, AH>(
                            a, c, wm, st, R0, C0 + cb, tlane + kStateZ + cb, from_tmem, to_tmem, v, s, cn, [&](int h) {
                                if (from_tmem) return;
                                if (h == 0) load16(a, c.Z, n, R0, R0 + lane, C0 + cb + 16, s.z[0], s.x[0]);
                                else if (EPI_COLS > 32 && cn >= 0) load16(a, c.Z, n, R0, R0 + lane, cn, s.z[0], s.x[0]);
                            });
                    });
                    if (CAN_RESIDE && to_tmem) tmem_wait_st();
                }
            }
            if constexpr (LAST) {
                // the sums of every 32 x 64 block of the matrix apart (the same
                // ones whatever the tiles), in the order of their position
                LastSums lb;
                lb.tr = lb.sq = 0.0;
                lb.lo = 0.f;
                auto flush = [&](int col) {
                    double tr = lb.tr, sq = lb.sq + (double)lb.lo;
                    for (int o = 16; o > 0; o >>= 1) {
                        tr += __shfl_xor_sync(0xffffffffu, tr, o);
                        sq += __shfl_xor_sync(0xffffffffu, sq, o);
                    }
                    if (lane == 0) store_partial(a, c.inst, c.chain, R0 >> 5, col >> 6, tr, sq);
                    lb.tr = lb.sq = 0.0;
                    lb.lo = 0.f;
                };
                if constexpr (HOLD) {
                    if (live && work) {
                        // a warp's 32 x 64 block, 8 columns at a time: the registers of
                        // sixteen warps hold no more without spills (16 columns 359 us a
                        // layer of n = 4096, D + S; with the next 16 ahead 365; 332 so)
                        const uint32_t tfin = tlane + (uint32_t)(buf * TN);
                        const float* Zg = c.Z + state_off(a.P, R0 + lane, C0 + cb0);
#pragma unroll 2
                        for (int cb = cb0; cb < cb1 && C0 + cb < n; cb += 8, Zg += 256) {
                            float v[8], z[8], x[8];
                            tmem_ld8(tfin + cb, reinterpret_cast<uint32_t*>(v));
                            ld_state8(Zg, z);
                            ld_state8(Zg + a.plane_elems, x);
                            tmem_wait_ld();
                            epi_last<8>(a, c, R0, lane, C0 + cb, v, z, x, lb);
                            __syncwarp();
                        }
                        flush(C0 + cb0);
                    }
                } else if (live && work) {
                    blocks([&](int cb, float (&v)[32], State32& s) {
                        epi_last<32>(a, c, R0, lane, C0 + cb, v, s.z[0], s.x[0], lb);
                        if (next_of(cb) >= 0) {
                            load16(a, c.Z, n, R0, R0 + lane, next_of(cb), s.z[0], s.x[0]);
                            load16(a, c.Z, n, R0, R0 + lane, next_of(cb) + 16, s.z[1], s.x[1]);
                        }
                        __syncwarp();
                        if ((cb & 32) || cb + 32 >= cb1) flush(C0 + cb);
                    });
                }
            }
            if constexpr (HOLD) release();
            else __syncwarp();
            // count the item's completion (release: the warp's stores come first)
            // and hand back the context
            if constexpr (!LAST) st.finish();
            if (lane == 0 && a.nlayers > 1) done_add(c.done, 1);
            __syncwarp();
            if (lane == 0) local_arrive(smem_u32(&ctx_empty[slot]));
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync();
    if (warp == 1) {
        tc_fence_after();
        if constexpr (PAIR)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS)
                         : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS)
                         : "memory");
    }
}

template <int MODE, int OUTFMT>
__global__ void __launch_bounds__(kDeferThreads, 1)
    layer_defer_kernel(const __grid_constant__ LayerArgs a, const __grid_constant__ TmaMaps maps0,
                       const __grid_constant__ TmaMaps maps1, const __grid_constant__ WriteMaps wmaps0,
                       const __grid_constant__ WriteMaps wmaps1) {
    using C = TcCfg<MODE>;
    using G = Geo<SHAPE_PAIR>;
    static_assert(OUTFMT != kLastLayer, "the last layer runs its epilogue inline");
    constexpr int TILE = G::TN;
    constexpr int EPI_COLS = TILE / (kDeferWarps / 4);   // columns per accumulating warp (64)
    constexpr int BKE = 128 / C::ESIZE;                // K elements per 128-byte slice
    constexpr int PLANE = kCtaRows * 128;              // bytes of one 128-row slice
    constexpr int STAGE_BYTES = C::NSPLIT * 2 * PLANE; // A and B planes (B: this CTA's half)
    constexpr int KSTEPS = 4;                          // 128-byte slice / 32 bytes per MMA
    constexpr uint32_t IDESC = make_idesc(C::ATYPE, TILE, TILE);
    constexpr int NBUF = G::NBUF;
    constexpr uint32_t TMEM_COLS = NBUF * TILE;

    // A launch whose layers all lie below the first layer any instance starts
    // at (models with fewer layers than the set's maximum start late) has no
    // active item: every thread of both CTAs of a pair leaves at once.
    grid_wait();
    const int first_layer = *reinterpret_cast<volatile const int*>(a.status + 1);
    if (a.gl + a.nlayers <= first_layer) return;
    // the items of layers before the first active one are skipped by every role
    const int f0 = max(0, first_layer - a.gl) * a.ntiles;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full_bar[C::STAGES];
    __shared__ __align__(8) uint64_t empty_bar[C::STAGES];
    __shared__ __align__(8) uint64_t tfull_bar[NBUF];
    __shared__ __align__(8) uint64_t tempty_bar[NBUF];
    // deferred epilogue: scratch full / empty
    __shared__ __align__(8) uint64_t sfull_bar, sempty_bar;
    // drain: the MMA issuer's last commit (all of its MMAs complete)
    __shared__ __align__(8) uint64_t drain_bar;
    __shared__ ItemCtx dctx[kStoreWarps];
    __shared__ uint32_t tmem_slot;
    // skip mode: set once this CTA has seen the call fail; the roles then keep
    // the barrier protocol of their work items without loads, MMAs or stores
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    // K slices per accumulation chunk at global layer g: the default 128
    // elements, or a shorter chunk requested for the layer
    auto ck_of = [&](int g) {
        const int ce = g >= a.tail_from ? a.chunk_tail : a.chunk_elems;
        return max(1, (ce > 0 ? ce : C::CK * BKE) / BKE);
    };
    const int unit = (int)(blockIdx.x >> 1), nunits = (int)(gridDim.x >> 1);     // pairs
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(&full_bar[s], G::NCTA);      // one expect_tx arrival per CTA
            mbar_init(&empty_bar[s], 1);
        }
        for (int s = 0; s < NBUF; ++s) {
            mbar_init(&tfull_bar[s], 1);
            mbar_init(&tempty_bar[s], G::NCTA * kDeferWarps);
        }
        mbar_init(&sfull_bar, kDeferWarps);
        mbar_init(&sempty_bar, kStoreWarps);
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == 0) {
        // ---------------- TMA producer (the warp runs the loop, one lane issues) ----------------
        const bool leader = elect_one();
        int stage = 0;
        uint32_t phase = 0;
        // (layer, instance) of each chain whose predecessor is known complete
        int known_g[kMaxChains] = {-1, -1}, known_i[kMaxChains] = {-1, -1};
        bool skip = false;                       // the call has failed: no more loads
        bool broken = false;                     // a pipeline wait ran out twice
        const uint32_t smem0 = uniform32(smem_u32(smem));
        const uint32_t full0 = uniform32(map_to(smem_u32(&full_bar[0]), 0));
        const int nf = n_items(a);
        for (int f = f0 + unit; f < nf && !broken; f += nunits) {
            int g, t;
            item_of(a, f, g, t);
            const Tile tl = a.tiles[t];
            int k;
            if (!tile_active_g(a, tl, g, k)) {
                // an inactive item counts as finished for the layer's completion
                if (a.nlayers > 1 && leader) atomicAdd(inst_counter(a, g, tl.inst, tl.chain), kDeferWarps);
                continue;
            }
            if (!skip && g > a.gl && g - 1 >= first_layer &&
                !(tl.chain ? g == known_g[1] && tl.inst == known_i[1] : g == known_g[0] && tl.inst == known_i[0])) {
                // Operands and state of this item were written by other CTAs:
                // wait for the previous layer of its own instance only, so a
                // small instance need not wait for a large one.
                bool done = true;
                if (leader) {
                    const int tgt = kDeferWarps * G::NCTA * a.iw[tl.inst].tile_count[a.dtab][tl.chain] +
                                    (g == a.stall_layer ? 1 : 0);
                    done = wait_counter(a, inst_counter(a, g - 1, tl.inst, tl.chain), tgt);
                    if (done) asm volatile("fence.proxy.async.global;" ::: "memory");
                }
                if (__all_sync(0xffffffffu, done)) {
                    if (tl.chain) {
                        known_g[1] = g;
                        known_i[1] = tl.inst;
                    } else {
                        known_g[0] = g;
                        known_i[0] = tl.inst;
                    }
                } else {
                    skip = true;
                }
            }
            if (skip && leader) *reinterpret_cast<volatile int*>(&abort_flag) = 1;
            const TmaMaps& maps = ((g - a.gl) & 1) ? maps1 : maps0;
            const int n = uniform32(a.inst[tl.inst].n), chain = uniform32(tl.chain);
            const int nk = (n + BKE - 1) / BKE;
            const int slab = uniform32(tl.inst * a.P), I0 = uniform32(tl.I * TILE), J0 = uniform32(tl.J * TILE);
            const int panA = I0 + (int)rank * kCtaRows, panB = J0 + (int)rank * kCtaRows;
            const int lowA = (!C::TF32 && a.lower_t) ? I0 / BKE : 0, lowB = (!C::TF32 && a.lower_t) ? J0 / BKE : 0;
            for (int kb = 0; kb < nk; ++kb) {
                // K-slices left of a panel's diagonal block: not stored below
                // the diagonal, loaded from the transposed upper block
                const bool tA = kb < lowA, tB = kb < lowB;
                if (!all_wait(&empty_bar[stage], phase ^ 1u, a)) {
                    broken = true;
                    break;
                }
                if (leader) {
                    const uint32_t fb = full0 + 8u * stage;
                    if (skip) {
                        // the stage's arrival without data: the phase completes
                        // with the peer's loads (if any) and no MMA reads it
                        remote_arrive(fb);
                    } else {
                        if (kb == max(0, nk - 3))
                            prefetch_state<TILE>(a, a.Z[tl.chain] + (size_t)tl.inst * a.P * a.P, panA, J0, n);
                        remote_expect_tx(fb, STAGE_BYTES);
                        const uint32_t sb = smem0 + stage * STAGE_BYTES;
                        const int kx = kb * BKE, ky = slab + kb * BKE;
#pragma unroll
                        for (int s = 0; s < C::NSPLIT; ++s) {
                            const uint32_t dA = sb + s * PLANE, dB = sb + (C::NSPLIT + s) * PLANE;
                            if (tA) {
                                tma_load_pair(dA, &maps.t[chain][s], fb, panA, ky);
                                tma_load_pair(dA + PLANE / 2, &maps.t[chain][s], fb, panA + 64, ky);
                            } else {
                                tma_load_pair(dA, &maps.a[chain][s], fb, kx, slab + panA);
                            }
                            if (tB) {
                                tma_load_pair(dB, &maps.t[chain][s], fb, panB, ky);
                                tma_load_pair(dB + PLANE / 2, &maps.t[chain][s], fb, panB + 64, ky);
                            } else {
                                tma_load_pair(dB, &maps.a[chain][s], fb, kx, slab + panB);
                            }
                        }
                    }
                }
                __syncwarp();
                if (++stage == C::STAGES) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
        if (broken) {
            // The barrier protocol failed, so the completion of the loads
            // already issued cannot be observed: give them a bounded grace
            // period (a load of one stage takes microseconds) before the
            // CTA releases its shared memory.
            *reinterpret_cast<volatile int*>(&abort_flag) = 1;
            const unsigned long long t0 = globaltimer();
            while (globaltimer() - t0 < 2000000ull) __nanosleep(1000);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (rank == 0) {
            // ---------------- MMA issuer (the even CTA of a pair; as in layer_tc_kernel) ----------------
            const bool leader = elect_one();
            int stage = 0;
            uint32_t phase = 0;
            int buf = 0;
            uint32_t aphase = 0;
            bool ok = true;
            const uint64_t desc0 = uniform64(sdesc_sw128(smem_u32(smem)));
            const uint64_t descT = uniform64(sdesc_mn_sw128(smem_u32(smem)));   // transposed panels
            const uint32_t tm = uniform32(tmem);
            const int nf = n_items(a);
            for (int f = f0 + unit; f < nf && ok; f += nunits) {
                int g, t;
                item_of(a, f, g, t);
                const Tile tl = a.tiles[t];
                int k;
                if (!tile_active_g(a, tl, g, k)) continue;
                const int n = uniform32(a.inst[tl.inst].n);
                const int nk = (n + BKE - 1) / BKE;
                const int ck = ck_of(g);
                const int I0 = uniform32(tl.I * TILE), J0 = uniform32(tl.J * TILE);
                const int lowA = (!C::TF32 && a.lower_t) ? I0 / BKE : 0, lowB = (!C::TF32 && a.lower_t) ? J0 / BKE : 0;
                for (int kc = 0; kc < nk && ok; kc += ck) {
                    if (!all_wait(&tempty_bar[buf], aphase ^ 1u, a)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t dt = tm + (uint32_t)(buf * TILE);
                    const int kend = min(nk, kc + ck);
                    for (int kb = kc; kb < kend; ++kb) {
                        if (!all_wait(&full_bar[stage], phase, a)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        // skip mode: the stage holds no new data; the commits below
                        // keep the protocol
                        const bool mma = uniform32(*reinterpret_cast<volatile int*>(&abort_flag)) == 0;
                        const bool tA = kb < lowA, tB = kb < lowB;
                        const uint32_t so = (uint32_t)((stage * STAGE_BYTES) >> 4);
                        const uint64_t baseA = (tA ? descT : desc0) + so, baseB = (tB ? descT : desc0) + so;
                        const uint32_t idesc = IDESC | (tA ? 1u << 15 : 0u) | (tB ? 1u << 16 : 0u);
                        const uint32_t stepA = tA ? 2048u >> 4 : 32u >> 4, stepB = tB ? 2048u >> 4 : 32u >> 4;
                        if (leader) {
                            if (mma) {
#pragma unroll
                                for (int q = 0; q < C::NPROD; ++q) {
                                    const int p = C::NPROD - 1 - q;      // the small products first
#pragma unroll
                                    for (int kk = 0; kk < KSTEPS; ++kk) {
                                        const uint64_t da = baseA + (uint32_t)(prod_a(p) * (PLANE >> 4)) + kk * stepA;
                                        const uint64_t db =
                                            baseB + (uint32_t)((C::NSPLIT + prod_b(p)) * (PLANE >> 4)) + kk * stepB;
                                        umma_pair<C::TF32>(dt, da, db, idesc,
                                                           (kk == 0 && q == 0) ? (kb == kc ? 0u : 1u) : 1u);
                                    }
                                }
                            }
                            umma_commit_pair(smem_u32(&empty_bar[stage]));
                            if (kb == kend - 1) umma_commit_pair(smem_u32(&tfull_bar[buf]));
                        }
                        __syncwarp();
                        if (++stage == C::STAGES) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                    if (!ok) break;
                    if (++buf == NBUF) {
                        buf = 0;
                        aphase ^= 1u;
                    }
                }
            }
            // Drain: every MMA this warp issued has completed before the final
            // barrier, after which the CTAs free TMEM and shared memory.
            if (leader) umma_commit_local_pair(smem_u32(&drain_bar));
            __syncwarp();
            if (!all_wait(&drain_bar, 0, a)) {
                const unsigned long long t0 = globaltimer();
                while (globaltimer() - t0 < 2000000ull) __nanosleep(1000);
            }
        }
        __syncwarp();
    } else if (warp >= 2 + kDeferWarps) {
        // ---------------- deferred final epilogue (store warps) ----------------
        // Tile t's finished sums arrive in the CTA's scratch while the MMAs and
        // the accumulating warps already work on tile t + 1.  Each lane streams
        // its rows of the blocks, 16 columns (sums, Z_k, A_k) at a time, into a
        // two-deep shared ring with cp.async; the warp computes Z_{k+1} and
        // A_{k+1} and writes the next operands block by block.
        const int sw = warp - 2 - kDeferWarps;
        Stager st{smem_u32(smem + C::STAGES * STAGE_BYTES) + (uint32_t)(sw * kStageBytes), lane, 0, 2};
        uint8_t* const ring = smem + C::STAGES * STAGE_BYTES + kStoreWarps * kStageBytes + sw * (kRing * kEntryBytes);
        const float* const scr = a.escr + (size_t)blockIdx.x * kEpiScratchFloats;
        ItemCtx& c = dctx[sw];
        uint32_t sp = 0;
        bool ok = true;
        const int nf = n_items(a);
        for (int f = f0 + unit; f < nf && ok; f += nunits) {
            int g, t;
            item_of(a, f, g, t);
            const Tile tl = a.tiles[t];
            int k;
            if (!tile_active_g(a, tl, g, k)) continue;
            if (!has_next_tile(a, f, nunits)) continue;     // inline in the accumulating warps
            if (lane == 0) {
                const InstWork& w = a.iw[tl.inst];
                fill_epilogue<MODE, OUTFMT, SHAPE_PAIR>(a, tl, w, a.layers[w.layer_off[tl.chain] + k], (int)rank, c);
            }
            __syncwarp();
            if (!wait_bar(&sfull_bar, sp, a)) {
                ok = false;
                break;
            }
            sp ^= 1u;
            // skip mode (warp-uniform): hand the scratch back without the work
            const bool work = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&abort_flag) == 0 ? 1 : 0, 0) != 0;
            if (work) {
                if (a.nlayers > 1 && g > a.gl) {
                    // the state of layer g - 1 of this instance, written by other CTAs
                    if (lane == 0) acquire_load(inst_counter(a, g - 1, tl.inst, tl.chain));
                    __syncwarp();
                }
                const CUtensorMap* const wm = (((g - a.gl) & 1) ? wmaps1 : wmaps0).w[tl.chain];
                // each lane copies exactly the 16-byte runs it reads later (its row
                // of the 8-column groups), so its own cp.async.wait_group suffices
                auto issue = [&](int e, int h, uint32_t slot) {
                    const DeferBlock d = defer_block(c, e);
                    const uint32_t dst = smem_u32(ring + slot * kEntryBytes) + 16u * lane;
                    const float* ssrc = scr + (e >> 1) * kItemFloats + ((e & 1) * 4 + 2 * h) * 256 + lane * 4;
                    const float* zsrc = c.Z + state_off(a.P, d.R0, d.c0 + 16 * h) + lane * 4;
#pragma unroll
                    for (int o = 0; o < 512; o += 128) {
                        cp_async16(dst + 4u * o, ssrc + o);
                        cp_async16(dst + 4u * (512 + o), zsrc + o);
                        cp_async16(dst + 4u * (1024 + o), zsrc + a.plane_elems + o);
                    }
                    cp_async_commit();
                };
                int e = -1;
                bool more = next_block(c, sw, e);
                if (more) {
                    issue(e, 0, 0);
                    issue(e, 1, 1);
                }
                while (more) {
                    const DeferBlock d = defer_block(c, e);
                    int en = e;
                    const bool next = next_block(c, sw, en);
                    float v[32];
                    State<1> s;
                    // half h of the block from the ring, whose entry takes that of the next one
                    auto take = [&](int h) {
                        // oldest copy group first: the other half, or the next block's first half
                        if (h == 0 || next) cp_async_wait<1>();
                        else cp_async_wait<0>();
                        const float* const src = reinterpret_cast<const float*>(ring + h * kEntryBytes) + lane * 4;
                        load_state8(src, v + 16 * h);
                        load_state8(src + 256, v + 16 * h + 8);
                        load_state8(src + 512, s.z[0]);
                        load_state8(src + 768, s.z[0] + 8);
                        load_state8(src + 1024, s.x[0]);
                        load_state8(src + 1280, s.x[0] + 8);
                        if (next) issue(en, h, h);
                    };
                    take(0);
                    epi_block32<OUTFMT, false>(a, c, wm, st, d.R0, d.c0, 0u, false, false, v, s, -1, [&](int h) {
                        if (h == 0) take(1);
                    });
                    e = en;
                    more = next;
                }
            }
            __syncwarp();
            st.finish();
            if (lane == 0) {
                // this warp's share of the tile's kDeferWarps completions
                if (a.nlayers > 1) done_add(inst_counter(a, g, tl.inst, tl.chain), kDeferWarps / kStoreWarps);
                local_arrive(smem_u32(&sempty_bar));
            }
            __syncwarp();
        }
        __syncwarp();
    } else {
        // ---------------- epilogue (warps 2..17) ----------------
        const int q = warp & 3;                  // TMEM lane quarter
        const int cq = (warp - 2) >> 2;          // column quarter of the tile
        // "tempty" barriers of the even CTA (consecutive 8-byte words)
        const uint32_t tempty0 = map_to(smem_u32(&tempty_bar[0]), 0);
        int buf = 0;
        uint32_t aphase = 0;
        uint32_t sp = 0;                         // scratch parity (deferred epilogue)
        bool ok = true;
        const int nf = n_items(a);
        for (int f = f0 + unit; f < nf && ok; f += nunits) {
            int g, t;
            item_of(a, f, g, t);
            // Only the chunk count and the liveness of the warp's block are
            // carried through the drain loop; the tile's descriptor and the
            // rest of the context are fetched again for the final epilogue, into
            // shared memory (the 64 accumulators leave 32 registers).
            int nch;
            bool warp_live, defer_tile;
            {
                const Tile tl = a.tiles[t];
                int k;
                if (!tile_active_g(a, tl, g, k)) continue;
                const int n = a.inst[tl.inst].n;
                const int R0 = tl.I * TILE + (int)rank * kCtaRows + q * 32;
                const int C0 = tl.J * TILE + cq * EPI_COLS;
                warp_live = C0 < n && C0 + EPI_COLS - 1 >= R0 && R0 < n;
                const int ck = ck_of(g);
                nch = ((n + BKE - 1) / BKE + ck - 1) / ck;
                defer_tile = has_next_tile(a, f, nunits);
            }
            float acc[EPI_COLS];
#pragma unroll
            for (int i = 0; i < EPI_COLS; ++i) acc[i] = 0.f;
            // Chunk drain.  Chunks 0 .. nch - 2 are added into acc and their
            // buffer released at once.  The last chunk is added too, and the
            // finished sum is written back into that chunk's TMEM buffer, which
            // stays held through the final epilogue: the epilogue then reads
            // its 8-column groups from TMEM, so the 64 accumulator registers of
            // a pair tile are free for the memory work.  The MMAs of the next
            // tile meanwhile fill the other buffers.
            const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cq * EPI_COLS);
            for (int j = 0; j < nch; ++j) {
                if (!wait_bar(&tfull_bar[buf], aphase, a)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t ta = tbase + (uint32_t)(buf * TILE);
                if (warp_live) {
#pragma unroll
                    for (int g = 0; g < EPI_COLS / 16; ++g) {
                        uint32_t v[16];
                        tmem_ld16(ta + 16 * g, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int jj = 0; jj < 16; ++jj) acc[16 * g + jj] += __uint_as_float(v[jj]);
                    }
                }
                if (j == nch - 1 && !defer_tile) {
                    if (warp_live) {
#pragma unroll
                        for (int g = 0; g < EPI_COLS / 8; ++g) tmem_st8(ta + 8 * g, &acc[8 * g]);
                        tmem_wait_st();
                    }
                    break;                            // buffer released after the final epilogue
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    remote_arrive(tempty0 + 8u * (uint32_t)buf);
                }
                if (++buf == NBUF) {
                    buf = 0;
                    aphase ^= 1u;
                }
            }
            if (!ok) break;
            // skip mode (warp-uniform): the protocol without the memory work
            const bool work = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&abort_flag) == 0 ? 1 : 0, 0) != 0;
            if (defer_tile) {
                // hand the finished sums to the store warps through the scratch
                // (its previous tile must have been read), then go on to the next tile
                if (!wait_bar(&sempty_bar, sp ^ 1u, a)) break;
                sp ^= 1u;
                if (warp_live && work) {
                    float* const dst = a.escr + (size_t)blockIdx.x * kEpiScratchFloats + (warp - 2) * kItemFloats + lane * 4;
#pragma unroll
                    for (int g = 0; g < EPI_COLS / 8; ++g) store_state8(dst + 256 * g, &acc[8 * g]);
                }
                __syncwarp();
                if (lane == 0) local_arrive(smem_u32(&sfull_bar));
                continue;
            }
            const uint32_t tfin = tbase + (uint32_t)(buf * TILE);   // the held buffer
            const Tile tl = a.tiles[t];
            int k;
            tile_active_g(a, tl, g, k);
            if (a.nlayers > 1 && g > a.gl) {
                // the state of layer g - 1 of this instance, written by other CTAs
                if (lane == 0) acquire_load(inst_counter(a, g - 1, tl.inst, tl.chain));
                __syncwarp();
            }
            if (warp_live && work) {
                // The unit's last tile: its MMAs have all completed and no loads
                // follow, so the blocks are staged in the operand ring, with the
                // warp's context behind them.
                ItemCtx& c = *reinterpret_cast<ItemCtx*>(smem + kDeferWarps * kStageBytes + (warp - 2) * 256);
                static_assert(sizeof(ItemCtx) <= 256 && kDeferWarps * (kStageBytes + 256) <= C::STAGES * STAGE_BYTES,
                              "staging and contexts in the ring");
                if (lane == 0) {
                    const InstWork& w = a.iw[tl.inst];
                    fill_epilogue<MODE, OUTFMT, SHAPE_PAIR>(a, tl, w, a.layers[w.layer_off[tl.chain] + k], (int)rank, c);
                }
                __syncwarp();
                Stager st{smem_u32(smem) + (uint32_t)((warp - 2) * kStageBytes), lane, 0, 2};
                const CUtensorMap* const wm = (((g - a.gl) & 1) ? wmaps1 : wmaps0).w[tl.chain];
                const int R0 = c.row0 + q * 32;
#pragma unroll 1
                for (int cb = 0; cb < EPI_COLS; cb += 32) {
                    const int c0 = c.col0 + cq * EPI_COLS + cb;
                    if (!(c0 >= R0 && c0 < c.n)) continue;
                    float v[32];
                    State<1> s;
                    load16(a, c.Z, c.n, R0, R0 + lane, c0, s.z[0], s.x[0]);
                    tmem_ld32(tfin + cb, reinterpret_cast<uint32_t*>(v));
                    tmem_wait_ld();
                    epi_block32<OUTFMT, false>(a, c, wm, st, R0, c0, 0u, false, false, v, s, -1, [&](int h) {
                        if (h == 0) load16(a, c.Z, c.n, R0, R0 + lane, c0 + 16, s.z[0], s.x[0]);
                    });
                }
                st.finish();
            }
            // release the held accumulator buffer
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                remote_arrive(tempty0 + 8u * (uint32_t)buf);
                if (a.nlayers > 1) done_add(inst_counter(a, g, tl.inst, tl.chain), 1);
            }
            if (++buf == NBUF) {
                buf = 0;
                aphase ^= 1u;
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

int tc_block_m(int shape) { return tc_pair(shape) ? 256 : 128; }
int tc_block_n(int shape) { return shape == SHAPE_PAIR ? 256 : shape == SHAPE_SINGLE64 ? 64 : 128; }

// One kernel variant: its function, threads, dynamic shared memory and CTAs per unit.
template <int MODE, int OUTFMT, int SHAPE, bool DEFER>
struct Variant {
    static auto fn() {
        if constexpr (DEFER) return layer_defer_kernel<MODE, OUTFMT>;
        else return layer_tc_kernel<MODE, OUTFMT, SHAPE>;
    }
    static constexpr int threads = DEFER ? kDeferThreads : tc_threads<OUTFMT, SHAPE>();
    static constexpr int smem = 1024 + (DEFER ? TcCfg<MODE>::STAGES * TcCfg<MODE>::NSPLIT * 2 * kCtaRows * 128 +
                                                    kStoreWarps * (kStageBytes + kRing * kEntryBytes)
                                              : Stage<MODE, SHAPE>::SMEM);
    static constexpr int ncta = Geo<SHAPE>::NCTA;

    static cudaError_t prepare() {
        static std::atomic<bool> done{false};
        if (done.load(std::memory_order_acquire)) return cudaSuccess;
        const cudaError_t e = cudaFuncSetAttribute(fn(), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) done.store(true, std::memory_order_release);
        return e;
    }
    static void config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int units) {
        cfg = cudaLaunchConfig_t{};
        cfg.gridDim = dim3(ncta * units, 1, 1);
        cfg.blockDim = dim3(threads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = attr;
        if (ncta > 1) {
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = ncta;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.numAttrs = 1;
        }
    }
    // A multi-layer launch (a.nlayers > 1) is cooperative: its CTAs wait on one
    // another, so all of them must be resident at once.
    static cudaError_t launch(const LayerArgs& a, const LayerMaps& m, int units,
                              cudaStream_t s) {
        cudaError_t e = prepare();
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[2];
        config(cfg, attr, units);
        cfg.stream = s;
        if (a.nlayers > 1) {
            attr[cfg.numAttrs].id = cudaLaunchAttributeCooperative;
            attr[cfg.numAttrs].val.cooperative = 1;
        } else {
            attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
        }
        ++cfg.numAttrs;
        e = cudaLaunchKernelEx(&cfg, fn(), a, *m.rd[0], *m.rd[1], *m.wr[0], *m.wr[1]);
        count_launch();
        return e;
    }
    // units that can be resident at once (0 if unknown)
    static int max_units() {
        if (prepare() != cudaSuccess) return 0;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[1];
        config(cfg, attr, 1);
        if (ncta == 1) {
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.numAttrs = 1;
        }
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, fn(), &cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return n;
    }
};

template <int MODE, int MAINFMT, int SHAPE>
static cudaError_t launch_shape(const LayerArgs& a, const LayerMaps& m, int units,
                                cudaStream_t s) {
    if (a.last) return Variant<MODE, kLastLayer, SHAPE, false>::launch(a, m, units, s);
    if (a.next_fmt == OP_F32) return Variant<MODE, OP_F32, SHAPE, false>::launch(a, m, units, s);
    if constexpr (MAINFMT != OP_BF16X3) {
        // the layer before BF16X3 refinement layers (FTSP2_REFINE_TC)
        if (a.next_fmt == OP_BF16X3) return Variant<MODE, OP_BF16X3, SHAPE, false>::launch(a, m, units, s);
    }
    // the layers of the main format: the final epilogue inline or deferred to
    // store warps (a.escr set: a scratch slot for each CTA of the grid)
    if constexpr (SHAPE == SHAPE_PAIR) {
        if (a.escr) return Variant<MODE, MAINFMT, SHAPE, true>::launch(a, m, units, s);
    }
    return Variant<MODE, MAINFMT, SHAPE, false>::launch(a, m, units, s);
}

template <int MODE, int MAINFMT>
static cudaError_t launch_mode(const LayerArgs& a, const LayerMaps& m, int units, int shape,
                               cudaStream_t s) {
    switch (shape) {
        case SHAPE_SINGLE: return launch_shape<MODE, MAINFMT, SHAPE_SINGLE>(a, m, units, s);
        case SHAPE_PAIR: return launch_shape<MODE, MAINFMT, SHAPE_PAIR>(a, m, units, s);
        case SHAPE_PAIR128: return launch_shape<MODE, MAINFMT, SHAPE_PAIR128>(a, m, units, s);
        case SHAPE_SINGLE64: return launch_shape<MODE, MAINFMT, SHAPE_SINGLE64>(a, m, units, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_layer_tc(int mode, const LayerArgs& a, const LayerMaps& m, int units,
                            int shape, cudaStream_t s) {
    switch (mode) {
        case FTSP2_FP16X2: return launch_mode<FTSP2_FP16X2, OP_F16X2>(a, m, units, shape, s);
        case FTSP2_BF16X3: return launch_mode<FTSP2_BF16X3, OP_BF16X3>(a, m, units, shape, s);
        case FTSP2_TF32X3: return launch_mode<FTSP2_TF32X3, OP_TF32X3>(a, m, units, shape, s);
    }
    return cudaErrorInvalidValue;
}

template <int MODE, int MAINFMT>
static int max_units_mode(int shape, bool defer) {
    switch (shape) {
        case SHAPE_SINGLE: return Variant<MODE, MAINFMT, SHAPE_SINGLE, false>::max_units();
        case SHAPE_PAIR:
            return defer ? Variant<MODE, MAINFMT, SHAPE_PAIR, true>::max_units()
                         : Variant<MODE, MAINFMT, SHAPE_PAIR, false>::max_units();
        case SHAPE_PAIR128: return Variant<MODE, MAINFMT, SHAPE_PAIR128, false>::max_units();
        case SHAPE_SINGLE64: return Variant<MODE, MAINFMT, SHAPE_SINGLE64, false>::max_units();
    }
    return 0;
}

int layer_tc_max_units(int mode, int shape, bool defer) {
    switch (mode) {
        case FTSP2_FP16X2: return max_units_mode<FTSP2_FP16X2, OP_F16X2>(shape, defer);
        case FTSP2_BF16X3: return max_units_mode<FTSP2_BF16X3, OP_BF16X3>(shape, defer);
        case FTSP2_TF32X3: return max_units_mode<FTSP2_TF32X3, OP_TF32X3>(shape, defer);
    }
    return 0;
}

}  // namespace ftsp2
