// Bidirectional block-query attention on the tcgen05 tensor cores (head dim HD, 64 or 128): the refresh prefill and
// the decode step over several block copies.
//
// Work item: up to 128 consecutive query rows x one head (x one key split in a decode step).
//   refresh: keys = every row of the sequence (fresh q/k/v of the same forward; nothing is read from the
//            cache, the refresh is what writes it); the output is final.
//   step:    the rows of all copies of one block (a StepTile).  Key splits 0 .. ks-2 stream the cached
//            K/V of the positions outside the block, visible to every row; the last split takes the fresh
//            rows: the item's own rows as they lie, the copies one behind the other, and for an item without
//            copy 0 in the decoded-share layout that copy's rows.  A row sees its own copy's rows and, in the
//            decoded-share layout, the decoded ones of copy 0.  Copies stay mutually invisible through this
//            per-row key mask, no mask tensor exists.  Outputs are per-split (max, sum, unnormalised
//            output) partials merged in split order by the merge kernel of attention.cu.
// No causal mask.  One pass over the key tiles of 64; per tile S = Q K^T is one 128 x 64 x HD tcgen05.mma group
// whose fp32 result lives in TMEM, and thread r owns TMEM lane r = query row r (no cross-thread reduction):
//   the tile's largest visible score moves the row's shift M - an INTEGER in the log2 domain - only when it exceeds
//   M by more than a slack of 4 (so P < 16); then O (in TMEM) and the row sum are multiplied by the exact power of two
//   2^(M_old - M_new), once the previous P V has been added;
//   P = exp2(S - M), row sums, P rounded to a two-term bf16 sum (value + remainder, as in the
//   mma.sync kernel) and written over S in TMEM, as the A operand of O += P V
//   (128 x HD x 64, V taken MN-major straight from its [key][dim] tile), O in TMEM.
// Exact softmax (rescaling by powers of two changes no bit of a normal number).  Warp-specialised: warps 0..3 = softmax (one query row per thread),
// warp 4 lane 0 = MMA issuer, warp 5 lane 0 = loader (TMA: boxes of 64 rows x 64 columns with the 128-byte
// swizzle land in the canonical operand layout, one 64-column atom per 64 dims).  Rows of a tile behind its last key are other
// sequences' or what a slot's earlier occupant left in the cache: the softmax masks their scores and sets their V to zero, for a
// zero of P times an infinity or NaN there would be a NaN in this sequence's output.  (Copies of one sequence share their tiles: there a
// row that is not finite reaches the block's other copies, as in a dense softmax under a mask.)  The roles meet only through mbarriers.  Two CTAs share an SM
// (256 TMEM columns each, 112 or 64 KB of shared memory).  Every mbarrier wait is bounded; on expiry the CTA records
// ODB_ERR_TIMEOUT, every role stops, the CTA releases its TMEM and exits.
//
// What bounds it is the chain of a tile: softmax (about 1000 cycles with an SM's sub-partition to itself: 170 for the read and
// the maximum, 720 for the exponentials - 512 is what the special-function unit takes for 64 - and 70 for the store), and
// from P to the S that takes its place about 2600 with head dim 128 (P V, S, and the hand-overs).  With three S / P buffers, for
// which head dim 64 leaves room, the second is hidden; with two a tile takes 1800 cycles on an SM of its own, 2300 with two
// CTAs.  The form before this one (P through shared memory, a select per key, one row stored per thread) took 2200 and 2800.
// us per launch, before / now: refresh of 768 rows 31.9 / 23.8, of 25568 rows in 16 sequences 1122 / 872, step of 16 sequences
// x 256 rows 221 / 167, of 128 rows 17.1 / 14.3; head dim 64, 1118 rows x 16 heads, 26.0 (mma.sync) / 16.3.
#include "odb_internal.cuh"

namespace odb {

namespace {

constexpr int kTQ = 128;   // query rows per work item (MMA M)
constexpr int kTK = 64;    // keys per tile
constexpr int kThreads = 192;   // 4 softmax warps, MMA warp, loader warp

// shared memory, HD = 128 / 64: Q 32 / 16 KB (one atom of 128 rows x 128 B per 64 columns), a ring of five / six K / V tiles of
// 16 / 8 KB (atoms of 64 rows x 128 B); the dynamic region starts 1024-aligned
template <int HD> constexpr uint32_t kQBytes = kTQ * HD * 2;
template <int HD> constexpr uint32_t kKBytes = kTK * HD * 2;
template <int HD> constexpr int kSlots = HD == 128 ? 5 : 6;
template <int HD> constexpr uint32_t kSmemBytes = kQBytes<HD> + kSlots<HD> * kKBytes<HD> + 256;
constexpr uint32_t kPatchBytes = 4096;               // per softmax warp, in the Q buffer: 32 rows x 128 bytes of output
// TMEM, 256 columns so that two CTAs share an SM: O takes the last HD, the S / P buffers 64 each of the others
template <int HD> constexpr int kSBuffers = HD == 128 ? 2 : 3;
constexpr uint32_t kTmemCols = 256;

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// one box of 64 rows x 64 columns (8 KB): rows row0.., columns col0..
__device__ __forceinline__ void tma_box(uint32_t dst, const CUtensorMap* tmap, uint64_t* bar, int col0, int row0) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(bar)), "r"(col0), "r"(row0)
        : "memory");
}

// asks L2 for the same box (no shared-memory destination, nothing to wait for)
__device__ __forceinline__ void tma_prefetch_box(const CUtensorMap* tmap, int col0, int row0) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(reinterpret_cast<uint64_t>(tmap)),
                 "r"(col0), "r"(row0)
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

// Bounded wait (shared implementation): false if the CTA has been aborted or the limit expired.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* cta_abort, int* status) {
    return mbar_wait_bounded(bar, parity, cta_abort, status);
}

// K-major operand, rows of 128 bytes, 128-byte swizzle, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t desc_k_major(uint32_t saddr) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>(1) << 16;                   // leading byte offset (unused with swizzle)
    d |= static_cast<uint64_t>(1024 >> 4) << 32;           // stride byte offset between 8-row groups
    d |= static_cast<uint64_t>(1) << 46;                   // descriptor version of this architecture
    d |= static_cast<uint64_t>(2) << 61;                   // 128-byte swizzle
    return d;
}

// MN-major operand: 64 contiguous elements (128 bytes) of the N dimension per K row, 128-byte swizzle;
// 8-K-row groups 1024 bytes apart (stride offset), 64-element N groups `n_group_bytes` apart (leading offset)
__device__ __forceinline__ uint64_t desc_mn_major(uint32_t saddr, uint32_t n_group_bytes) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>(n_group_bytes >> 4) << 16;
    d |= static_cast<uint64_t>(1024 >> 4) << 32;
    d |= static_cast<uint64_t>(1) << 46;
    d |= static_cast<uint64_t>(2) << 61;
    return d;
}

// bf16 x bf16 -> fp32, A K-major, B K-major or MN-major
__host__ __device__ constexpr uint32_t instr_desc(int m, int n, int b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(b_mn_major) << 16) |
           (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(m >> 4) << 24);
}

__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// the same with the A operand in TMEM: lane = row, two bf16 per column
__device__ __forceinline__ void umma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// The wait belongs to the instruction: as a statement of its own nothing would keep a use of the values behind it.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, uint32_t (&v)[64]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, "
        "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, "
        "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31]), "=r"(v[32]),
          "=r"(v[33]), "=r"(v[34]), "=r"(v[35]), "=r"(v[36]), "=r"(v[37]), "=r"(v[38]), "=r"(v[39]), "=r"(v[40]),
          "=r"(v[41]), "=r"(v[42]), "=r"(v[43]), "=r"(v[44]), "=r"(v[45]), "=r"(v[46]), "=r"(v[47]), "=r"(v[48]),
          "=r"(v[49]), "=r"(v[50]), "=r"(v[51]), "=r"(v[52]), "=r"(v[53]), "=r"(v[54]), "=r"(v[55]), "=r"(v[56]),
          "=r"(v[57]), "=r"(v[58]), "=r"(v[59]), "=r"(v[60]), "=r"(v[61]), "=r"(v[62]), "=r"(v[63])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]),
        "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]),
        "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]),
        "r"(v[31])
        : "memory");
}

// two fp32 values in one 64-bit register: the packed forms round each value as the plain ones do
__device__ __forceinline__ uint64_t pack2f(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ uint64_t pack2u(uint32_t a, uint32_t b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2f(uint64_t x) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

struct alignas(8) TcShared {
    uint64_t q_full;       // Q tile landed                                   (loader -> MMA)
    uint64_t full[6];      // K or V tile landed in the ring's slot            (loader -> MMA, softmax)
    uint64_t empty[6];     // the MMAs have read the slot                      (MMA -> loader)
    uint64_t s_full[3];    // S = Q K^T into S buffer i has completed          (MMA -> softmax)
    uint64_t p_full[3];    // P has taken its place                           (softmax -> MMA, 4 arrivals)
    uint64_t pv_done[2];   // O += P V of an even / odd tile has completed     (MMA -> MMA, softmax)
    uint64_t o_full;       // the last one has                                 (MMA -> softmax)
    uint32_t tmem_base;
    int abort;
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// 2^x for x <= 0 on the special-function unit (flushes to zero far below zero, which is the wanted value)
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One key tile of a work item: 64 consecutive rows of a [rows][HD]-column view starting at row0, of which
// the first `valid` are keys.  src: 0 = fresh k / v rows of this forward, 1 = the K/V cache.
struct KeyTile {
    int src, row0, v_row0, valid;
    int copy;          // fresh tile of a step: the source copy, or kPacked; -1 otherwise (visible to every row)
};

constexpr int kPacked = -2;   // consecutive rows of the item's own copies

struct TcArgs {
    const QTile* qtiles;          // refresh work items
    const StepTile* stiles;       // step work items
    const int32_t* row_flags;
    __nv_bfloat16* o;             // refresh: final output [M][H * HD]
    float* part_o; float* part_ml;   // step: split partials [ks][M][H][HD], [ks][M][H][2]
    int layer, n_layers, H, max_seq, M;
    int any_order;                // step: the order of sums is free
};

// 128-byte pieces of a warp's 32 rows, turned in its patch of shared memory (16-byte chunks, XOR-swizzled) so that eight lanes
// store one row's 128 bytes: w = the lane's own row, sink(row of the warp, 16-byte chunk, value).
template <class Sink>
__device__ __forceinline__ void turn_rows(uint32_t patch, int lane, const uint32_t (&w)[32], Sink&& sink) {
    __syncwarp();   // the previous piece has been taken
#pragma unroll
    for (int c = 0; c < 8; ++c)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(patch + lane * 128 + ((c ^ (lane & 7)) << 4)), "r"(w[4 * c]),
                     "r"(w[4 * c + 1]), "r"(w[4 * c + 2]), "r"(w[4 * c + 3])
                     : "memory");
    __syncwarp();
    const int c = lane & 7;
#pragma unroll
    for (int it = 0; it < 8; ++it) {
        const int r = it * 4 + (lane >> 3);
        uint4 x;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
                     : "r"(patch + r * 128 + ((c ^ (r & 7)) << 4))
                     : "memory");
        sink(r, c, x);
    }
}

template <int HD, bool STEP>
__global__ void __launch_bounds__(kThreads, 2) attention_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                                                                   const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_c,
                                                                   TcArgs a, int* status) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    constexpr uint32_t kK = kKBytes<HD>;
    constexpr int kAtoms = HD / 64;       // 64-column atoms of a row
    uint8_t* sQ = smem_raw;
    uint8_t* ring = sQ + kQBytes<HD>;     // K and V tiles in the order the MMAs take them
    constexpr int kRing = kSlots<HD>, kBufs = kSBuffers<HD>, kFirst = kBufs - 1;
    TcShared* sh = reinterpret_cast<TcShared*>(ring + kRing * kK);
    static_assert(sizeof(TcShared) <= 256 && kRing <= 6 && kBufs <= 3, "the barriers end inside the allocation");
    static_assert(kBufs * kTK + HD <= static_cast<int>(kTmemCols) && 4 * kPatchBytes <= kQBytes<HD>, "TMEM columns, output patches");

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int* cta_abort = &sh->abort;

    if ((smem_u32(smem_raw) & 1023u) != 0) {                // the swizzled tiles need 1024-byte alignment
        if (tid == 0) atomicExch(status, ODB_ERR_CUDA);
        pdl_wait();
        return;
    }
    if (tid == 0) {
        mbar_init(&sh->q_full, 1);
        for (int i = 0; i < kRing; ++i) {
            mbar_init(&sh->full[i], 1);
            mbar_init(&sh->empty[i], 1);
        }
        for (int b = 0; b < kBufs; ++b) {
            mbar_init(&sh->s_full[b], 1);
            mbar_init(&sh->p_full[b], 4);
        }
        for (int i = 0; i < 2; ++i) mbar_init(&sh->pv_done[i], 1);
        mbar_init(&sh->o_full, 1);
        sh->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh->tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_launch_dependents();                                // behind the TMEM allocation: the successor allocates for pairs
    const uint32_t tmem_s = sh->tmem_base;                          // kBufs x 64 columns: a tile's S, then its P
    const uint32_t tmem_o = sh->tmem_base + kTmemCols - HD;

    // q, k, v of this layer come from the preceding kernel.  A step's work items were complete before anything behind its first
    // norm could start, its K/V cache before the step: the loader asks for cached tiles before it waits.
    if (!STEP || warp != 5) pdl_wait();
    const int head = blockIdx.y;
    const int z = blockIdx.z, ks = gridDim.z;
    // ---- the work item: query rows and key tiles ----
    int q_row0, nq, ntiles;
    int f0 = 0, NK = 0;                                     // refresh: keys = fresh rows [f0, f0 + NK)
    int cA = 0, cB0 = 0, cB1 = 0, nA_t = 0, t_first = 0;    // step, cached split: positions [0, cA) and [cB0, cB1)
    int c_row = 0;                                          // step: row of position 0 of this head's keys in the cache view
    bool fresh_split = false;
    const bool single = STEP && ks == 1;                    // step without key splits
    int n_cached = 0;                                       // step: cached key tiles of this CTA (they come first)
    const StepTile* stp = nullptr;
    int n_own = 0;                                          // step: packed tiles of the item's own rows; 0: a tile per source copy
    if constexpr (!STEP) {
        const QTile t = a.qtiles[blockIdx.x];
        q_row0 = t.q_row0; nq = t.nq; f0 = t.f0; NK = t.n0;
        ntiles = (NK + kTK - 1) / kTK;
    } else {
        stp = a.stiles + blockIdx.x;
        q_row0 = stp->slab_row0[0];
        nq = stp->slab_row0[stp->n_slabs - 1] + stp->slab_n[stp->n_slabs - 1] - q_row0;   // the slabs are consecutive rows
        cA = stp->cA; cB0 = stp->cB0; cB1 = stp->cB1;
        nA_t = (cA + kTK - 1) / kTK;
        const int nct = nA_t + (cB1 - cB0 + kTK - 1) / kTK;
        // Fresh keys in tiles of 64 rows as they lie, not a tile per copy (four copies of 32: two tiles, not four; eight of the
        // decoded-share layout, 24 + 7 x 9 rows: two or three, not eight).  Where the order of sums has to stay, only with
        // copies of 16, 32 or 64 rows: their keys then fall into the same groups of sixteen and halves of a tile.
        fresh_split = z == ks - 1;                          // also the only one
        int nf = 0;
        if (fresh_split) {
            const int n0 = stp->src_n[0];
            const bool other0 = stp->stage2 && stp->slab_copy[0] != 0;   // copy 0 belongs to another item: its tile comes last
            nf = stp->n_src;
            if (a.any_order || (!stp->stage2 && n0 >= 16 && (n0 & (n0 - 1)) == 0)) {
                n_own = (nq + kTK - 1) / kTK;
                nf = n_own + (other0 ? 1 : 0);
            }
        }
        if (single) {
            // one CTA takes every key of the item: the cached tiles, then the fresh ones; its output is final
            n_cached = nct;
            ntiles = nct + nf;
        } else {
            const int tp = (nct + ks - 2) / (ks - 1);
            t_first = fresh_split ? 0 : z * tp;
            n_cached = fresh_split ? 0 : max(0, min(nct, t_first + tp) - t_first);
            ntiles = fresh_split ? nf : n_cached;
        }
        c_row = ((stp->seq * a.n_layers + a.layer) * 2 * a.H + head) * a.max_seq;   // K; V is H * max_seq rows further
    }
    auto key_tile = [&](int i) {
        KeyTile kt;
        kt.copy = -1;
        if constexpr (!STEP) {
            kt.src = 0; kt.row0 = f0 + i * kTK; kt.v_row0 = kt.row0; kt.valid = min(kTK, NK - i * kTK);
        } else if (i >= n_cached) {
            const int fi = i - n_cached, f = n_own ? stp->n_src - 1 : fi;
            if (fi < n_own) {
                kt.src = 0; kt.row0 = q_row0 + fi * kTK; kt.v_row0 = kt.row0; kt.valid = min(kTK, nq - fi * kTK); kt.copy = kPacked;
                return kt;
            }
            kt.src = 0; kt.row0 = stp->src_row0[f]; kt.v_row0 = kt.row0; kt.valid = stp->src_n[f]; kt.copy = stp->src_copy[f];
        } else {
            const int j = t_first + i;
            const int pos0 = j < nA_t ? j * kTK : cB0 + (j - nA_t) * kTK;
            const int end = j < nA_t ? cA : cB1;
            kt.src = 1; kt.row0 = c_row + pos0; kt.v_row0 = kt.row0 + a.H * a.max_seq; kt.valid = min(kTK, end - pos0);
        }
        return kt;
    };
    const float scale_log2 = rsqrtf(static_cast<float>(HD)) * 1.4426950408889634f;
    auto wait = [&](uint64_t* bar, uint32_t parity) { return mbar_wait(bar, parity, cta_abort, status); };
    auto wait_pv = [&](int tile) { return wait(&sh->pv_done[tile & 1], static_cast<uint32_t>(tile >> 1) & 1u); };

    if (warp == 5) {
        // ================= loader =================
        if (lane == 0 && ntiles > 0) {
            const int col0 = head * HD;
            const int n_loads = 2 * ntiles;
            // 64 rows x HD columns: one box per 64-column atom (the cache view has HD columns per row)
            auto boxes = [&](const KeyTile& kt, bool v, auto&& box) {
                const CUtensorMap* map = kt.src ? &tm_c : v ? &tm_v : &tm_k;
#pragma unroll
                for (int at = 0; at < kAtoms; ++at) box(at, map, (kt.src ? 0 : col0) + 64 * at, v ? kt.v_row0 : kt.row0);
            };
            // Load i: K(0) .. K(kFirst - 1), then K(t + kFirst), V(t) by turns, then the last V (the order of the MMAs).
            const int head_k = min(kFirst, ntiles), turns = 2 * (ntiles - head_k);
            auto load_of = [&](int i, int& tile) {               // true: V
                if (i < head_k) { tile = i; return false; }
                const int j = i - head_k;
                const bool v = j >= turns || (j & 1);
                tile = j >= turns ? j - turns / 2 : (j >> 1) + (v ? 0 : kFirst);
                return v;
            };
            // The ring covers little of a load's latency from HBM: every load also asks L2 for the tile kAhead tiles
            // further on, so that the load that later fills a slot comes from L2.
            constexpr int kAhead = 3;
            int slot = 0;
            auto load = [&](int i) {
                int tile;
                const bool v = load_of(i, tile);
                const uint32_t dst = smem_u32(ring) + slot * kK;
                uint64_t* bar = &sh->full[slot];
                mbar_expect_tx(bar, kK);
                boxes(key_tile(tile), v, [&](int at, const CUtensorMap* map, int col, int row) { tma_box(dst + at * kTK * 128, map, bar, col, row); });
                if (tile + kAhead < ntiles)
                    boxes(key_tile(tile + kAhead), v, [&](int, const CUtensorMap* map, int col, int row) { tma_prefetch_box(map, col, row); });
                if (++slot == kRing) slot = 0;
            };
            int i = 0;
            if (STEP) {
                for (int tile; i < n_loads && i < kRing && (load_of(i, tile), tile < n_cached); ++i) load(i);
                pdl_wait();
            }
            // Q: rows 0..63 and 64..127 of each atom
            mbar_expect_tx(&sh->q_full, kQBytes<HD>);
#pragma unroll
            for (int at = 0; at < kAtoms; ++at) {
                tma_box(smem_u32(sQ) + at * kTQ * 128, &tm_q, &sh->q_full, col0 + 64 * at, q_row0);
                tma_box(smem_u32(sQ) + at * kTQ * 128 + 64 * 128, &tm_q, &sh->q_full, col0 + 64 * at, q_row0 + 64);
            }
            uint32_t ph = 1;                                         // a slot's first load waits for nothing
            for (; i < n_loads; ++i) {
                if (i >= kRing) {
                    if (slot == 0) ph ^= 1u;
                    if (!wait(&sh->empty[slot], ph)) break;
                }
                load(i);
            }
            if (*cta_abort) {   // let the copies still in flight land before the CTA's shared memory goes away
                const long long t0 = clock64();
                auto land = [&](uint64_t* bar, uint32_t parity) {
                    while (!mbar_try_wait_parity(bar, parity) && clock64() - t0 < kWaitLimitCycles / 8) {
                    }
                };
                land(&sh->q_full, 0);
                for (int j = max(0, i - kRing); j < i; ++j) land(&sh->full[j % kRing], static_cast<uint32_t>(j / kRing) & 1u);
            }
        } else if (STEP) {
            pdl_wait();
        }
    } else if (warp == 4) {
        // ================= MMA issuer =================
        // S(0) .. S(kFirst - 1), then S(t + kFirst), P V(t) by turns: a warp that has finished its rows of a tile finds the next
        // scores ready.  S(t + kFirst) takes the buffer of P(t - 1), so it is issued when P V(t - 1) has completed: MMAs of
        // different shapes and accumulators have no order among themselves.
        if (lane == 0 && ntiles > 0) {
            constexpr uint32_t idesc_s = instr_desc(kTQ, kTK, 0);
            constexpr uint32_t idesc_o = instr_desc(kTQ, HD, 1);
            int slot = 0, sb = 0;                                    // ring slot, S buffer of the next S
            uint32_t ph = 0;
            auto next_slot = [&]() {
                umma_commit(&sh->empty[slot]);
                if (++slot == kRing) { slot = 0; ph ^= 1u; }
            };
            // S = Q K^T of the next tile over the head dim: MMAs of K = 16
            // (a descriptor's address field counts 16 bytes and no tile crosses its end: offsets are added to the descriptor)
            const uint64_t q_desc = desc_k_major(smem_u32(sQ)), ring_k = desc_k_major(smem_u32(ring)),
                           ring_v = desc_mn_major(smem_u32(ring), kTK * 128);
            auto issue_s = [&](int after_pv) {
                if (!wait(&sh->full[slot], ph)) return false;
                if (after_pv >= 0 && !wait_pv(after_pv)) return false;
                tc_fence_after();
                const uint64_t k_desc = ring_k + static_cast<uint32_t>(slot) * (kK >> 4);
#pragma unroll
                for (int kk = 0; kk < HD / 16; ++kk) {
                    const uint32_t atom = kk >> 2, within = (kk & 3) * 32;
                    umma(tmem_s + sb * kTK, q_desc + ((atom * (kTQ * 128) + within) >> 4), k_desc + ((atom * (kTK * 128) + within) >> 4),
                         idesc_s, kk > 0 ? 1u : 0u);
                }
                next_slot();
                umma_commit(&sh->s_full[sb]);
                if (++sb == kBufs) sb = 0;
                return true;
            };
            bool ok = wait(&sh->q_full, 0);
            for (int tile = 0; tile < kFirst && tile < ntiles && ok; ++tile) ok = issue_s(-1);
            int b = 0;
            uint32_t round = 0;                                      // S buffer of `tile`, parity of its use
            for (int tile = 0; tile < ntiles && ok; ++tile) {
                if (tile + kFirst < ntiles) ok = issue_s(tile - 1);
                if (ok) ok = wait(&sh->full[slot], ph);
                if (ok) ok = wait(&sh->p_full[b], round);
                if (!ok) break;
                tc_fence_after();
                const uint32_t p = tmem_s + b * kTK;
                const uint64_t v_desc = ring_v + static_cast<uint32_t>(slot) * (kK >> 4);
#pragma unroll
                for (int kk = 0; kk < kTK / 16; ++kk) {             // 16 keys per MMA: rounded values, then remainders
                    umma_ts(tmem_o, p + kk * 8, v_desc + kk * (2048 >> 4), idesc_o, (tile > 0 || kk > 0) ? 1u : 0u);
                    umma_ts(tmem_o, p + kTK / 2 + kk * 8, v_desc + kk * (2048 >> 4), idesc_o, 1u);
                }
                next_slot();
                umma_commit(&sh->pv_done[tile & 1]);
                if (++b == kBufs) { b = 0; round ^= 1u; }
            }
            if (ok) umma_commit(&sh->o_full);
        }
    } else {
        // ================= softmax: thread r = query row r = TMEM lane r =================
        const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;   // this warp's TMEM lanes
        bool ok = true;
        int my_copy = -1, stage2 = 0;
        int my_row0 = 0, my_n = 0;                                  // the rows of this row's copy
        int n_copy0 = 0;                                            // rows of copy 0 at the front of the item
        if (STEP && fresh_split) {                                  // the splits of cached keys need no copies
            stage2 = stp->stage2;
            const int grow = q_row0 + tid;
            for (int sl = 0; sl < stp->n_slabs; ++sl)
                if (grow >= stp->slab_row0[sl] && grow < stp->slab_row0[sl] + stp->slab_n[sl]) my_copy = stp->slab_copy[sl];
            if (my_copy >= 0) {
                const int f = my_copy - stp->src_copy[0];           // an item's copies are consecutive
                my_row0 = stp->src_row0[f];
                my_n = stp->src_n[f];
            }
            if (stage2 && stp->src_copy[0] == 0) n_copy0 = stp->src_n[0];
        }
        // which of the tile's 64 keys this row sees (bit j = key j).  Every lane of a warp calls this for the
        // same tile: the branch that uses the ballots is uniform.
        auto tile_mask = [&](const KeyTile& kt) -> unsigned long long {
            const unsigned long long all = kt.valid >= 64 ? ~0ull : ((1ull << kt.valid) - 1ull);
            if (kt.copy == -1) return all;                          // cached keys, or a refresh
            unsigned long long shared = 0ull;
            if constexpr (STEP) {
                // decoded rows of copy 0, shared with every copy
                const int n_shared = kt.copy == kPacked ? min(kt.valid, q_row0 + n_copy0 - kt.row0) : stage2 && kt.copy == 0 ? kt.valid : 0;
                if (n_shared > 0) {
                    const bool d0 = lane < n_shared && (a.row_flags[kt.row0 + lane] & kRowDecoded);
                    const bool d1 = lane + 32 < n_shared && (a.row_flags[kt.row0 + lane + 32] & kRowDecoded);
                    const unsigned lo = __ballot_sync(0xffffffffu, d0), hi = __ballot_sync(0xffffffffu, d1);
                    shared = (static_cast<unsigned long long>(hi) << 32 | lo) & all;
                }
                if (kt.copy == kPacked) {
                    const int k0 = max(0, my_row0 - kt.row0), k1 = min(kt.valid, my_row0 + my_n - kt.row0);
                    return k1 <= k0 ? shared : shared | ((k1 >= 64 ? ~0ull : (1ull << k1) - 1ull) & ~((1ull << k0) - 1ull));
                }
            }
            return kt.copy == my_copy ? all : shared;
        };
        // ---- one pass over the key tiles: online softmax.  The row's shift M is an INTEGER in the log2 domain, so
        // that moving it rescales O and the row sum by an exact power of two; it moves only when a tile's maximum
        // exceeds it by more than kSlack (P then stays below 2^kSlack), which after the first tiles is rare. ----
        constexpr float kSlack = 4.0f;
        float M_row = -INFINITY;                                     // no visible key yet
        float l_row = 0.f;
        const uint64_t scale2 = pack2f(scale_log2, scale_log2), minus1 = pack2f(-1.0f, -1.0f);
        int b = 0;
        uint32_t round = 0;                                          // S buffer of `tile`, parity of its use
        for (int tile = 0; tile < ntiles; ++tile) {
            const uint32_t ts = tmem_s + lane_base + b * kTK;
            const KeyTile kt = key_tile(tile);
            // a whole tile of cached keys (or of a refresh) is seen by every row
            const bool full = kt.copy == -1 && kt.valid >= 64;
            const unsigned long long mask = full ? ~0ull : tile_mask(kt);
            ok = wait(&sh->s_full[b], round);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            uint32_t sv[64];                                         // the row's scores
            tmem_ld64(ts, sv);
            if (!full) {                                             // keys the row does not see: exp2 gives exactly 0
#pragma unroll
                for (int j = 0; j < 64; ++j)
                    if (!((mask >> j) & 1ull)) sv[j] = 0xff800000u;
            }
            float m0 = __uint_as_float(sv[0]), m1 = __uint_as_float(sv[32]);   // largest visible score of the tile
#pragma unroll
            for (int j = 1; j < 31; j += 2) {
                m0 = max3(m0, __uint_as_float(sv[j]), __uint_as_float(sv[j + 1]));
                m1 = max3(m1, __uint_as_float(sv[32 + j]), __uint_as_float(sv[33 + j]));
            }
            m0 = max3(m0, m1, __uint_as_float(sv[31]));
            m0 = fmaxf(m0, __uint_as_float(sv[63]));
            float factor = 1.0f;                                     // what O and the row sum so far are multiplied by
            const float mt_log2 = m0 * scale_log2;                   // -inf: the row sees no key of this tile
            if (mt_log2 > M_row + kSlack) {                          // also the first visible key (M_row = -inf)
                const float M_new = ceilf(mt_log2);
                if (M_row != -INFINITY) factor = exp2f(M_row - M_new);   // an exact power of two
                M_row = M_new;
            }
            // The exponentials take a score's exact product with scale_log2, the shift comes from the rounded one: from 2^22 on they lie up
            // to 0.25 and more apart (from 2^31 on P overflowed or vanished), and the scores are rounded first.
            const bool far = fabsf(mt_log2) >= 0x1p22f && mt_log2 != -INFINITY;
            bool rescale = false;
            uint64_t mult2 = scale2;
            if (__any_sync(0xffffffffu, factor != 1.0f || far)) {
                rescale = __any_sync(0xffffffffu, factor != 1.0f);
                if (__any_sync(0xffffffffu, far)) {
#pragma unroll
                    for (int j = 0; j < 64; ++j) sv[j] = __float_as_uint(__uint_as_float(sv[j]) * scale_log2);
                    mult2 = pack2f(1.0f, 1.0f);
                }
            }
            const float m_log2 = M_row == -INFINITY ? 0.f : M_row;   // a row that has seen no key: every P is 0
            const uint64_t shift2 = pack2f(-m_log2, -m_log2);
            float l_tile = 0.f;
            uint32_t hi[32], lo[32];                                 // the row's P: 64 keys as bf16 pairs, value + remainder
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint64_t sum = 0ull;
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    // arguments are <= kSlack: the hardware exponential needs no range handling (far below zero it returns 0)
                    const float2 x = unpack2f(fma2(pack2u(sv[half * 32 + 2 * u], sv[half * 32 + 2 * u + 1]), mult2, shift2));
                    const float p0 = ex2_approx(x.x), p1 = ex2_approx(x.y);
                    const uint64_t p = pack2f(p0, p1);
                    sum = add2(sum, p);
                    const __nv_bfloat162 h = __floats2bfloat162_rn(p0, p1);
                    const uint32_t hb = *reinterpret_cast<const uint32_t*>(&h);
                    // the bf16 halves widened back to fp32 are the bit patterns themselves, shifted into place
                    const float2 r = unpack2f(fma2(pack2u(hb << 16, hb & 0xffff0000u), minus1, p));
                    const __nv_bfloat162 l = __floats2bfloat162_rn(r.x, r.y);
                    hi[half * 16 + u] = hb;
                    lo[half * 16 + u] = *reinterpret_cast<const uint32_t*>(&l);
                }
                const float2 t = unpack2f(sum);
                l_tile += t.x + t.y;
            }
            tmem_st32(ts, hi);
            tmem_st32(ts + kTK / 2, lo);
            if (kt.valid < kTK) {
                // V's rows behind the keys, once it has landed.  i: V(tile)'s place in the loader's order.  The parity is not ambiguous:
                // the load before it in this slot is a K or V tile multiplied before S(tile) was, the one behind it waits for P V(tile).
                // us per call, without / with: 8B step of four sequences (three such tiles an item) 141.2 / 142.6, d 1024 refresh of two layers
                // 177.8 / 178.9, 8B refresh of 768 rows equal.  Only non-finite rows, or the rest of a group of 16 alone (P V of the
                // others left out), takes as long: it is the wait in front of P's arrival.  By the MMA warp's other lanes 142.0 and 180.4.
                const int i = tile < ntiles - kFirst ? kFirst + 2 * tile + 1 : ntiles + tile, slot = i % kRing;
                ok = __all_sync(0xffffffffu, wait(&sh->full[slot], static_cast<uint32_t>(i / kRing) & 1u));
                if (!ok) break;
                const uint32_t v = smem_u32(ring) + slot * kK;
#pragma unroll
                for (int at = 0; at < kAtoms; ++at)
                    for (uint32_t off = kt.valid * 128 + tid * 16; off < kTK * 128; off += 128 * 16)
                        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(v + at * kTK * 128 + off), "r"(0) : "memory");
                proxy_fence();
            }
            if (rescale) {                                           // warp-uniform; rows that keep their shift multiply by 1
                // P V(tile - 1) has been added to O.  The parity is not ambiguous: S(tile) was issued behind P V(tile - kBufs), so
                // P V(tile - 3), which the same barrier counts, has completed; P V(tile + 1) cannot have, it is behind this P.
                ok = __all_sync(0xffffffffu, tile == 0 || wait_pv(tile - 1));
                if (!ok) break;
                tc_fence_after();
                if (tile > 0) {
#pragma unroll 1
                    for (int c = 0; c < HD / 32; ++c) {
                        uint32_t v[32];
                        tmem_ld32(tmem_o + lane_base + c * 32, v);
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) * factor);
                        tmem_st32(tmem_o + lane_base + c * 32, v);
                    }
                }
            }
            l_row = l_row * factor + l_tile;
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->p_full[b]);
            if (++b == kBufs) { b = 0; round ^= 1u; }
        }
        const float m_log2 = M_row == -INFINITY ? 0.f : M_row;      // the shift the row's sum and output carry
        if (ok && ntiles > 0) ok = __all_sync(0xffffffffu, wait(&sh->o_full, 0));
        if (ok) {
            tc_fence_after();
            const int d = a.H * HD;
            const int row_w = q_row0 + warp * 32;                   // the warp's first row
            const int left = nq - warp * 32;                        // rows of the item from there on
            const uint32_t patch = smem_u32(sQ) + warp * kPatchBytes;   // every MMA that reads Q has completed
            if (!STEP || single) {
                const float inv = l_row > 0.f ? 1.0f / l_row : 0.f;
                __nv_bfloat16* out = a.o + static_cast<size_t>(row_w) * d + head * HD;
#pragma unroll 1
                for (int c = 0; c < HD / 64; ++c) {
                    uint32_t v[64], w[32];
                    tmem_ld64(tmem_o + lane_base + c * 64, v);
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const __nv_bfloat162 x = __floats2bfloat162_rn(__uint_as_float(v[2 * j]) * inv, __uint_as_float(v[2 * j + 1]) * inv);
                        w[j] = *reinterpret_cast<const uint32_t*>(&x);
                    }
                    turn_rows(patch, lane, w, [&](int r, int ch, const uint4& x) {
                        if (r < left) *reinterpret_cast<uint4*>(out + static_cast<size_t>(r) * d + c * 64 + ch * 8) = x;
                    });
                }
            } else {
                // split partial: unnormalised output, (max in the log2 domain, sum); a split that saw no key has sum 0
                const size_t pr = (static_cast<size_t>(z) * a.M + row_w) * a.H + head;   // of the warp's first row
                if (lane < left) *reinterpret_cast<float2*>(a.part_ml + (pr + static_cast<size_t>(lane) * a.H) * 2) = make_float2(m_log2, l_row);
                if (ntiles > 0) {
                    float* po = a.part_o + pr * HD;
#pragma unroll 1
                    for (int c = 0; c < HD / 32; ++c) {
                        uint32_t v[32];
                        tmem_ld32(tmem_o + lane_base + c * 32, v);
                        turn_rows(patch, lane, v, [&](int r, int ch, const uint4& x) {
                            if (r < left) *reinterpret_cast<uint4*>(po + static_cast<size_t>(r) * d + c * 32 + ch * 4) = x;
                        });
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sh->tmem_base), "r"(kTmemCols) : "memory");
    }
}

template <int HD, bool STEP>
cudaError_t launch_tc(dim3 grid, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v, const __nv_bfloat16* cache,
                      size_t cache_rows, const TcArgs& ta, int* status, cudaStream_t st) {
    static std::atomic<unsigned long long> attr_done{0};
    cudaError_t e = set_smem_limit_once(attr_done, attention_tc_kernel<HD, STEP>, static_cast<int>(kSmemBytes<HD>));
    if (e != cudaSuccess) return e;
    // the fresh q / k / v of this forward: [M][H * HD] bf16, rows beyond M read as zero; the cache as rows of HD
    CUtensorMap tq, tk, tv, tc;
    const int d = ta.H * HD;
    e = make_rows_tmap(&tq, q, ta.M, d, 64);
    if (e == cudaSuccess) e = make_rows_tmap(&tk, k, ta.M, d, 64);
    if (e == cudaSuccess) e = make_rows_tmap(&tv, v, ta.M, d, 64);
    if (e == cudaSuccess) e = STEP ? make_rows_tmap(&tc, cache, static_cast<int>(cache_rows), HD, 64) : make_rows_tmap(&tc, k, ta.M, d, 64);
    if (e != cudaSuccess) return e;
    return launch_kernel(attention_tc_kernel<HD, STEP>, grid, dim3(kThreads), kSmemBytes<HD>, st, tq, tk, tv, tc, ta, status);
}

}  // namespace

// Refresh attention on the tensor cores: a.tiles = work items of up to 128 query rows whose keys are the
// fresh rows [f0, f0 + n0) (cA = cB0 = cB1 = n1 = 0).
cudaError_t launch_attention_tc(const AttnArgs& a, int* status, cudaStream_t st) {
    if (a.n_tiles == 0) return cudaSuccess;
    TcArgs ta{};
    ta.qtiles = a.tiles;
    ta.row_flags = a.row_flags;
    ta.o = a.o;
    ta.layer = a.layer; ta.n_layers = a.n_layers; ta.H = a.H; ta.max_seq = a.max_seq; ta.M = a.M;
    const dim3 grid(a.n_tiles, a.H);
    return a.hd == 128 ? launch_tc<128, false>(grid, a.q, a.k, a.v, nullptr, 0, ta, status, st)
                       : launch_tc<64, false>(grid, a.q, a.k, a.v, nullptr, 0, ta, status, st);
}

// Decode-step attention over StepTiles on the tensor cores; cache_rows = rows of the K/V cache viewed as
// [rows][head dim] (batch x layers x 2 x heads x max_seq).  ksplit = 1: every work item is one CTA over all of its
// keys and writes the final output; ksplit >= 2: partials only, the caller merges them.
cudaError_t launch_step_attention_tc(const StepAttnArgs& a, size_t cache_rows, int* status, cudaStream_t st) {
    if (a.n_tiles == 0) return cudaSuccess;
    if (a.ksplit < 1 || a.ksplit > 8) return cudaErrorInvalidValue;
    TcArgs ta{};
    ta.stiles = a.tiles;
    ta.row_flags = a.row_flags;
    ta.any_order = a.any_order;
    ta.o = a.o;                                            // written when there is no key split
    ta.part_o = a.part_o; ta.part_ml = a.part_ml;
    ta.layer = a.layer; ta.n_layers = a.n_layers; ta.H = a.H; ta.max_seq = a.max_seq; ta.M = a.M;
    const dim3 grid(a.n_tiles, a.H, a.ksplit);
    return a.hd == 128 ? launch_tc<128, true>(grid, a.q, a.k, a.v, a.cache, cache_rows, ta, status, st)
                       : launch_tc<64, true>(grid, a.q, a.k, a.v, a.cache, cache_rows, ta, status, st);
}

}  // namespace odb
