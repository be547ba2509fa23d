// Many-row projections (more than 128 activation rows): persistent CTA pairs with the ACTIVATION rows on the M side of
// the tensor-core tile.
//
// The kernel of gemm_tcgen05.cu gives the M side to the weights (as the pair kernel before this one did); its
// accumulator then has one weight row per TMEM lane and an epilogue thread owns one output FEATURE of many rows:
// SwiGLU has to fetch the matching up value from another warp through shared memory behind a block barrier, the
// confidence statistics need a transpose, and every bf16 store is a 2-byte store.  Here the two operands of the MMA change
// places: a cluster of two CTAs issues one tcgen05.mma.cta_group::2 of 256 activation rows x 256 weight rows, each
// CTA staging 128 activation rows (A) and one packed weight tile of 128 rows (its half of B), so the bytes staged and
// the MMA rate are the ones of the other kernel, and lane r of a CTA's accumulator is its activation row r with 256
// features in consecutive columns.  A thread owns a row: gate and up (a packed gate/up tile is 64 gate then 64 up
// rows), rotate-half partners, the row's RMSNorm scalar and a whole vocabulary tile's logits are its own; the eight
// epilogue warps (two per 32 TMEM lanes, one packed weight tile each) share no data and meet at no barrier.  Results
// leave through a 4 KB patch of shared memory per warp, so that stores are 16 bytes wide and cover whole 64- or
// 128-byte lines.  The sums are the same products in the same order.
//
// One pair per two SMs walks over the output tiles (6 stages x 32 KB, two accumulators in TMEM): the epilogue of a tile
// runs under the main loop of the next.  With 227 KB of shared memory no other kernel that allocates TMEM fits beside a
// CTA, and no second pair either: an allocation for a pair needs the same columns in both SMs, so two of them meeting on
// one pair of SMs, or one meeting single-SM allocations of a successor, could wait for each other.
//
// Measured against the kernels this replaces (8B shape, one launch each, 768 / 4096 / 25600 rows):
//   SwiGLU                                154 -> 106, 793 -> 515 us, 4.52 -> 3.34 ms (1.46, 1.60, 1.54 PFLOP/s; 1.68 is the peak)
//   QKV + RoPE + cache scatter             72 -> 59, 330 -> 273 us, 2.17 -> 1.71 ms (projection and RoPE kernel before)
//   LM head + statistics at 256 rows      321 -> 205 us
// Tensor pipe busy in 86 % (SwiGLU), 80 % (QKV) of the cycles at 4096 rows.
#include "odb_internal.cuh"
#include "tcgen05_common.cuh"

namespace odb {

namespace {

constexpr int kRowsN = 256;                              // weight rows of a pair's tile (two packed tiles)
constexpr uint32_t kTileBytes = kBM * kBK * 2;           // 16 KB: a packed weight tile, and 128 activation rows
constexpr uint32_t kRowsStageBytes = 2 * kTileBytes;
constexpr int kRowsStages = 6;
constexpr uint32_t kRowsTmemCols = 2 * kRowsN;           // two accumulators
constexpr int kRowsThreads = 320;                        // TMA warp, MMA warp, eight epilogue warps
constexpr uint32_t kPatchBytes = 4096;                   // per epilogue warp: 32 rows x 128 bytes

constexpr int ROWS_SWIGLU = 0, ROWS_CONF = 1, ROWS_ADD = 2, ROWS_PARTIAL = 3, ROWS_QKV64 = 4, ROWS_QKV128 = 5;

struct alignas(8) RowsShared {
    uint64_t full[kRowsStages];
    uint64_t empty[kRowsStages];
    uint64_t acc_full[2];
    uint64_t acc_empty[2];       // the leader's counts the 16 epilogue warps of both CTAs
    uint32_t tmem_base;
    int abort;
};

struct RowsArgs {
    float* partial;              // ROWS_PARTIAL: fp32 [splits][M][N]
    __nv_bfloat16* act_out;      // ROWS_SWIGLU: bf16 [M][N = F]
    ConfEpilogue ce;             // ROWS_CONF
    float* add_to;               // ROWS_ADD: fp32 [M][N], the residual stream
    QkvRopeArgs qkv;             // ROWS_QKV64 / ROWS_QKV128 (head dim)
    RowScale rs;
    int M, N, nkb_total, nkb_per_split;
    int n_pairs, m_tiles, group;           // pairs of weight tiles, tiles of 256 rows, row tiles that are walked side by side
    int whole, n_items;          // the items from `whole` on are single weight tiles
    uint64_t w_hint;             // L2 policy of the weight tiles
    int wide;                    // ROWS_PARTIAL: output rows start on 16-byte boundaries
    int* status;
};

// The tiles in the order they are handed out, round robin, to the pairs: the row tiles of a group side by side on one
// weight-tile pair (its weights come from HBM once, from L2 for the other row tiles), then the next weight-tile pair
// (the group's activation rows stay in L2: 17 MB at K 4096, 50 MB at K 12288), then the next group, then the next K split.
//
// HALVES: the items that do not fill a last round of the pairs are two items each, of one packed weight tile (256 x 128;
// either CTA stages half of its rows).
struct RowsItem {
    int m_tile, tile, split, kb0, nkb;   // tile: packed weight tile, the first of two unless half
    bool half;
};
template <bool HALVES>
__device__ __forceinline__ RowsItem rows_item(const RowsArgs& a, int item) {
    RowsItem w;
    int second = 0;
    w.half = HALVES && item >= a.whole;
    if (w.half) {
        second = (item - a.whole) & 1;
        item = a.whole + ((item - a.whole) >> 1);
    }
    const int per_split = a.m_tiles * a.n_pairs;
    w.split = item / per_split;
    item -= w.split * per_split;
    const int g = item / (a.group * a.n_pairs), m_first = g * a.group;
    const int in_group = min(a.group, a.m_tiles - m_first);
    item -= m_first * a.n_pairs;
    const int pair = item / in_group;
    w.m_tile = m_first + item - pair * in_group;
    w.tile = 2 * pair + second;
    w.kb0 = w.split * a.nkb_per_split;
    w.nkb = min(a.nkb_per_split, a.nkb_total - w.kb0);   // >= 1: the launcher refuses empty splits
    return w;
}

// 128-byte pieces of 32 rows, turned in shared memory (16-byte chunks, XOR-swizzled: no bank conflicts either way):
// lane r puts its row's chunks, then eight lanes take one row's 128 bytes, so that a store covers whole lines.
__device__ __forceinline__ void put_chunk(uint8_t* buf, int lane, int c, uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(smem_u32(buf) + lane * 128 + ((c ^ (lane & 7)) << 4)), "r"(x0), "r"(x1),
                 "r"(x2), "r"(x3)
                 : "memory");
}
// sink(row of the warp, 16-byte chunk of the piece, value); every lane calls it eight times
template <class Sink>
__device__ __forceinline__ void take_rows(uint8_t* buf, int lane, Sink&& sink) {
    const uint32_t base = smem_u32(buf);
    const int c = lane & 7;
#pragma unroll
    for (int it = 0; it < 8; ++it) {
        const int r = it * 4 + (lane >> 3);
        uint4 x;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
                     : "r"(base + r * 128 + ((c ^ (r & 7)) << 4))
                     : "memory");
        sink(r, c, x);
    }
}
// four fp32 sums added to memory without a read back; every element has exactly one such add per launch, so the
// result is the rounded sum whatever the order of the CTAs
__device__ __forceinline__ void red_add4(float* p, const uint4& x) {
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(__uint_as_float(x.x)),
                 "f"(__uint_as_float(x.y)), "f"(__uint_as_float(x.z)), "f"(__uint_as_float(x.w))
                 : "memory");
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 y = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&y);
}

// tcgen05.ld is a whole-warp instruction: the lanes meet first, whatever the code in front made of them (lanes without a
// row or a column leave the piece before early).
__device__ __forceinline__ void tmem_read32(uint32_t taddr, uint32_t (&v)[32]) {
    __syncwarp();
    tmem_ld32(taddr, v);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// two pieces of 16 columns; the wait is part of the statement, so that no use of the values can come in front of it
__device__ __forceinline__ void tmem_read16x2(uint32_t t0, uint32_t t1, uint32_t (&a)[16], uint32_t (&b)[16]) {
    __syncwarp();
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%33];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]), "=r"(a[9]),
          "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]), "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]),
          "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]),
          "=r"(b[14]), "=r"(b[15])
        : "r"(t0), "r"(t1)
        : "memory");
}

__device__ __forceinline__ uint32_t leader_address(uint64_t* bar) {   // shared::cluster address of the leader's copy of `bar`
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(bar)));
    return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}

template <int EPI, bool HALVES>
__global__ void __launch_bounds__(kRowsThreads, 1)
gemm_rows_kernel(const __grid_constant__ WeightMaps maps, const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ RowsArgs a,
                 const __grid_constant__ PeerOut po) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* patches = ring + kRowsStages * kRowsStageBytes;
    RowsShared* sh = reinterpret_cast<RowsShared*>(patches + 8 * kPatchBytes);
    const uint32_t rank = cluster_ctarank();
    const bool leader = rank == 0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int first = static_cast<int>(blockIdx.x) >> 1, step = static_cast<int>(gridDim.x) >> 1;
    const int n_items = a.n_items;
    static_assert(!(HALVES && EPI == ROWS_CONF), "the statistics belong to whole tiles");
    volatile int* cta_abort = &sh->abort;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kRowsStages; ++i) {
            mbar_init(&sh->full[i], 1);
            mbar_init(&sh->empty[i], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sh->acc_full[b], 1);
            mbar_init(&sh->acc_empty[b], 16);
        }
        sh->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps.tile)) : "memory");
        if (HALVES) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps.half)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmap_x)) : "memory");
    }
    if (warp == 1) {   // the same warp of both CTAs allocates the same columns in both SMs
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh->tmem_base)),
                     "r"(kRowsTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    cluster_barrier();         // the peer's barriers are initialised before anything signals them
    // Behind the allocation: no successor's allocation can come before it.  Not in front of the attention: its CTAs would take
    // the SMs that this launch leaves free (or leaves first), five on each, and run there side by side (two layers of d 1024,
    // 1118 rows: 236 -> 232 us; d 256, 2200 rows: 169 -> 126).
    if (EPI != ROWS_QKV64 && EPI != ROWS_QKV128) pdl_launch_dependents();
    const uint32_t tmem_acc = sh->tmem_base;

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer: weight tiles of the first stages first (they do not depend on the preceding kernel) ----
            RowsItem w = rows_item<HALVES>(a, first);
            const int pre = w.nkb < kRowsStages ? w.nkb : kRowsStages;
            int wt, wrow, mrow;
            auto begin = [&]() {
                wt = (w.tile + (w.half ? 0 : static_cast<int>(rank))) * a.nkb_total + w.kb0;
                wrow = w.half ? static_cast<int>(rank) * (kBM / 2) : 0;
                mrow = w.m_tile * 2 * kBM + static_cast<int>(rank) * kBM;
            };
            auto load_w = [&](int i, int st) {   // the loads of both CTAs report to the leader
                if (leader) mbar_expect_tx(&sh->full[st], w.half ? 3 * kTileBytes : 2 * kRowsStageBytes);
                tma_load_3d_pair(ring + st * kRowsStageBytes, w.half ? &maps.half : &maps.tile, &sh->full[st], 0, wrow, wt + i, a.w_hint);
            };
            begin();
            for (int i = 0; i < pre; ++i) load_w(i, i);
            pdl_wait();
            for (int i = 0; i < pre; ++i)
                tma_load_2d_pair(ring + i * kRowsStageBytes + kTileBytes, &tmap_x, &sh->full[i], (w.kb0 + i) * kBK, mrow, kEvictLast);
            int st = pre == kRowsStages ? 0 : pre;
            uint32_t ph = pre == kRowsStages ? 1u : 0u;   // parity of the ring's current round
            long long issued = pre;
            bool ok = true;
            int i = pre;
            for (int item = first;;) {
                for (; i < w.nkb && ok; ++i) {
                    ok = mbar_wait(&sh->empty[st], ph ^ 1u, cta_abort, a.status);   // the first round's stages are free
                    if (!ok) break;
                    load_w(i, st);
                    tma_load_2d_pair(ring + st * kRowsStageBytes + kTileBytes, &tmap_x, &sh->full[st], (w.kb0 + i) * kBK, mrow, kEvictLast);
                    ++issued;
                    if (++st == kRowsStages) { st = 0; ph ^= 1u; }
                }
                item += step;
                if (!ok || item >= n_items) break;
                w = rows_item<HALVES>(a, item);
                begin();
                i = 0;
            }
            if (*cta_abort && leader) {
                // aborted: let the copies still in flight land before the CTA's shared memory goes away (the
                // peer cannot observe its own copies; it is held by the cluster barrier at the end)
                for (long long j = issued > kRowsStages ? issued - kRowsStages : 0; j < issued; ++j) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait_parity(&sh->full[j % kRowsStages], static_cast<uint32_t>(j / kRowsStages) & 1u) &&
                           clock64() - t0 < kWaitLimitCycles / 8) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && leader) {
            // ---- MMA issuer (the leader's, for both CTAs): A = activation rows, B = weight rows ----
            bool ok = true;
            int st = 0, n = 0;
            uint32_t ph = 0;
            for (int item = first; item < n_items && ok; item += step, ++n) {
                const RowsItem w = rows_item<HALVES>(a, item);
                const int nkb = w.nkb, b = n & 1;
                const uint32_t idesc = w.half ? make_instr_desc(2 * kBM, kRowsN / 2) : make_instr_desc(2 * kBM, kRowsN);
                const uint32_t acc = tmem_acc + static_cast<uint32_t>(b * kRowsN);
                ok = mbar_wait(&sh->acc_empty[b], ((n >> 1) & 1) ^ 1u, cta_abort, a.status);   // free at first
                tc_fence_after();
                for (int i = 0; i < nkb && ok; ++i) {
                    ok = mbar_wait(&sh->full[st], ph, cta_abort, a.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t w_addr = smem_u32(ring + st * kRowsStageBytes), x_addr = w_addr + kTileBytes;
#pragma unroll
                    for (int k = 0; k < kBK / kUmmaK; ++k)
                        umma_bf16_pair(acc, make_smem_desc(x_addr + k * kUmmaK * 2), make_smem_desc(w_addr + k * kUmmaK * 2), idesc,
                                       (i > 0 || k > 0) ? 1u : 0u);
                    umma_commit_pair(&sh->empty[st]);   // frees the stage in both CTAs once these MMAs have read it
                    if (++st == kRowsStages) { st = 0; ph ^= 1u; }
                }
                if (ok) umma_commit_pair(&sh->acc_full[b]);
            }
        }
    } else {
        // ---- epilogue: warps 2..9 own TMEM lanes 32 * (warp % 4) .. + 31 = activation rows; group t of four warps owns the
        // 128 columns of an item's packed weight tile t, or half t of the columns of its only one ----
        const int q = warp & 3, t = (warp - 2) >> 2;
        uint8_t* patch = patches + (warp - 2) * kPatchBytes;
        const uint32_t free_bar = leader_address(&sh->acc_empty[0]);
        pdl_wait();   // the previous reader of the output buffer has finished; the predecessor's results are visible
        int n_done = 0;
        for (int item = first; item < n_items; item += step, ++n_done) {
            const RowsItem w = rows_item<HALVES>(a, item);
            const int b = n_done & 1;
            const int mw = w.m_tile * 2 * kBM + static_cast<int>(rank) * kBM + q * 32;   // the warp's first row
            const int m = mw + lane;
            const int tile = w.half ? w.tile : w.tile + t;
            const uint32_t tmem = tmem_acc + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(b * kRowsN + (w.half ? 0 : t * kBM));
            const float sc = m < a.M ? row_scale_of(a.rs, m) : 1.0f;
            int pos = 0, seq = 0;
            // QKV: quarters of the tile's columns that are this warp's, and the (cos, sin) of the first
            const int first_quarter = w.half ? 2 * t : 0, last_quarter = w.half ? 2 * t + 2 : 4;
            float2 next_cs[16];
            auto load_cs = [&](int u) {
                constexpr int HD = EPI == ROWS_QKV128 ? 128 : 64;
                const int c = HD == 128 ? u * 16 : (u & 1) * 16;
                if (tile * (kBM / HD) + (HD == 128 ? 0 : u >> 1) >= 2 * a.qkv.H) return;   // v is not rotated
#pragma unroll
                for (int j = 0; j < 16; ++j) next_cs[j] = a.qkv.rope_t[static_cast<size_t>(c + j) * a.qkv.max_seq + pos];
            };
            if constexpr (EPI == ROWS_QKV64 || EPI == ROWS_QKV128) {
                if (m < a.M) { pos = a.qkv.row_pos[m]; seq = a.qkv.row_seq[m]; }
                load_cs(first_quarter);
            }
            if (!__all_sync(0xffffffffu, mbar_wait(&sh->acc_full[b], (n_done >> 1) & 1, cta_abort, a.status))) break;
            tc_fence_after();
            if constexpr (EPI == ROWS_SWIGLU) {
#pragma unroll
                for (int c = 0; c < 64; c += 16) {
                    if (w.half && c / 32 != t) continue;
                    uint32_t g[16], u[16];
                    __syncwarp();
                    tmem_ld16(tmem + c, g);
                    tmem_ld16(tmem + 64 + c, u);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    float gate[16], up[16], x[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) { gate[j] = __uint_as_float(g[j]) * sc; up[j] = __uint_as_float(u[j]) * sc; }
                    silu_product(gate, up, x);
                    uint32_t out[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) out[j] = pack2(x[2 * j], x[2 * j + 1]);
                    put_chunk(patch, lane, c / 8, out[0], out[1], out[2], out[3]);
                    put_chunk(patch, lane, c / 8 + 1, out[4], out[5], out[6], out[7]);
                }
                __syncwarp();
                take_rows(patch, lane, [&](int r, int ch, const uint4& x) {
                    const int f = tile * 64 + ch * 8;
                    if (w.half && ch / 4 != t) return;
                    if (mw + r < a.M && f < a.N)             // F % 16 == 0
                        *reinterpret_cast<uint4*>(a.act_out + static_cast<size_t>(mw + r) * a.N + f) = x;
                });
            } else if constexpr (EPI == ROWS_ADD || EPI == ROWS_PARTIAL) {
                const size_t split_off = static_cast<size_t>(w.split) * a.M * a.N;
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    if (w.half && c / 2 != t) continue;
                    const int nc = tile * kBM + c * 32;
                    if (nc >= a.N) break;
                    uint32_t v[32];
                    tmem_read32(tmem + c * 32, v);           // the warp meets: the previous piece has been taken
                    if (EPI == ROWS_PARTIAL && a.rs.ssq) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) * sc);
                    }
#pragma unroll
                    for (int ch = 0; ch < 8; ++ch) put_chunk(patch, lane, ch, v[4 * ch], v[4 * ch + 1], v[4 * ch + 2], v[4 * ch + 3]);
                    __syncwarp();
                    if (EPI == ROWS_ADD || (a.wide && po.n == 0)) {
                        take_rows(patch, lane, [&](int r, int ch, const uint4& x) {
                            const int n = nc + ch * 4;
                            if (mw + r >= a.M || n >= a.N) return;       // N % 4 == 0
                            const size_t off = static_cast<size_t>(mw + r) * a.N + n;
                            if (EPI == ROWS_ADD) red_add4(a.add_to + off, x);
                            else *reinterpret_cast<uint4*>(a.partial + split_off + off) = x;
                        });
                    } else {
                        // tensor-parallel partial sums (the tile goes to the receive buffer of every rank), and rows of any
                        // length on any 4-byte boundary; apart from the code above, which that made 2 % of a step slower
                        take_rows(patch, lane, [&](int r, int ch, const uint4& x) {
                            const int n = nc + ch * 4;
                            if (mw + r >= a.M || n >= a.N) return;
                            const size_t off = split_off + static_cast<size_t>(mw + r) * a.N + n;
#pragma unroll 1
                            for (int p = 0; p < (po.n ? po.n : 1); ++p) {
                                float* out = (po.n ? po.partial[p] : a.partial) + off;
                                if (a.wide) {
                                    *reinterpret_cast<uint4*>(out) = x;
                                } else {
                                    out[0] = __uint_as_float(x.x);
                                    if (n + 1 < a.N) out[1] = __uint_as_float(x.y);
                                    if (n + 2 < a.N) out[2] = __uint_as_float(x.z);
                                    if (n + 3 < a.N) out[3] = __uint_as_float(x.w);
                                }
                            }
                        });
                    }
                }
            } else if constexpr (EPI == ROWS_QKV64 || EPI == ROWS_QKV128) {
                // QKV projection: a head's q, k or v of this row is the thread's own, rotate-half partners included.
                // The RMSNorm scalar, RoPE (q and k), bf16 rows and - in a refresh - the K/V cache.  The (cos, sin) table
                // is read transposed ([pair][position]): the lanes' positions are neighbours, mostly.  A quarter is 16
                // dims of a head's lower half and the 16 they rotate with, two of them a piece; the table's entries of the
                // next quarter are asked for in front of the work on this one.
                constexpr int HD = EPI == ROWS_QKV128 ? 128 : 64, kHalf = HD / 2;
                const QkvRopeArgs& e = a.qkv;
                const long long crow = (static_cast<long long>(seq) * e.n_layers + e.layer) * 2 * e.H * e.max_seq + pos;
#pragma unroll 1
                for (int u = first_quarter; u < last_quarter; ++u) {
                    const int grp = HD == 128 ? 0 : u >> 1, c = HD == 128 ? u * 16 : (u & 1) * 16;
                    const int g = tile * (kBM / HD) + grp;             // head of [Wq; Wk; Wv]
                    if (g >= 3 * e.H) break;
                    const int sec = g / e.H, head = g - sec * e.H;
                    uint32_t lo[16], hi[16];
                    if (!(u & 1)) __syncwarp();                        // the previous piece has been taken
                    tmem_read16x2(tmem + grp * HD + c, tmem + grp * HD + kHalf + c, lo, hi);
                    float2 cs[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) cs[j] = next_cs[j];
                    if (u + 1 < last_quarter) load_cs(u + 1);
                    uint32_t pl[8], ph[8];
#pragma unroll
                    for (int j = 0; j < 16; j += 2) {
                        float x0 = __uint_as_float(lo[j]) * sc, y0 = __uint_as_float(hi[j]) * sc;
                        float x1 = __uint_as_float(lo[j + 1]) * sc, y1 = __uint_as_float(hi[j + 1]) * sc;
                        if (sec < 2) {
                            const float a0 = x0 * cs[j].x - y0 * cs[j].y, b0 = y0 * cs[j].x + x0 * cs[j].y;
                            const float a1 = x1 * cs[j + 1].x - y1 * cs[j + 1].y, b1 = y1 * cs[j + 1].x + x1 * cs[j + 1].y;
                            x0 = a0; y0 = b0; x1 = a1; y1 = b1;
                        }
                        pl[j / 2] = pack2(x0, x1);
                        ph[j / 2] = pack2(y0, y1);
                    }
                    const int ch = (u & 1) * 2;
                    put_chunk(patch, lane, ch, pl[0], pl[1], pl[2], pl[3]);
                    put_chunk(patch, lane, ch + 1, pl[4], pl[5], pl[6], pl[7]);
                    put_chunk(patch, lane, ch + 4, ph[0], ph[1], ph[2], ph[3]);
                    put_chunk(patch, lane, ch + 5, ph[4], ph[5], ph[6], ph[7]);
                    if (!(u & 1)) continue;
                    __syncwarp();
                    const int c0 = c - 16;
                    __nv_bfloat16* fresh = (sec == 0 ? e.q : sec == 1 ? e.k : e.v) + head * HD;
                    const long long chead = static_cast<long long>((sec - 1) * e.H + head) * e.max_seq;
                    take_rows(patch, lane, [&](int r, int ch, const uint4& x) {
                        const long long cr = __shfl_sync(0xffffffffu, crow, r);
                        if (mw + r >= a.M) return;
                        const int dim = c0 + (ch & 3) * 8 + (ch >> 2) * kHalf;
                        *reinterpret_cast<uint4*>(fresh + static_cast<size_t>(mw + r) * (e.H * HD) + dim) = x;
                        if (e.cache && sec > 0) *reinterpret_cast<uint4*>(e.cache + (cr + chead) * HD + dim) = x;
                    });
                }
            } else {
                // LM head: softmax statistics of each 128-entry vocabulary tile of this thread's row: maximum and argmax
                // (ascending ids, strict: lowest id on ties) in one pass over the tile, the sum of exponentials in a second
                const int n0 = tile * kBM, id0 = n0 + a.ce.tile0 * kBM;
                // ids the statistics leave out: the padding behind the vocabulary, [MASK]
                const bool whole = n0 + kBM <= a.N && (a.ce.mask_id < id0 || a.ce.mask_id >= id0 + kBM);
                auto skip = [&](int i) { return !whole && (n0 + i >= a.N || id0 + i == a.ce.mask_id); };
                float mx = -INFINITY, sum = 0.f;
                int idx = 0x7fffffff;
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    uint32_t v[32];
                    tmem_read32(tmem + c * 32, v);
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float l = __uint_as_float(v[j]) * sc;
                        if (l > mx && !skip(c * 32 + j)) { mx = l; idx = id0 + c * 32 + j; }
                    }
                }
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    uint32_t v[32];
                    tmem_read32(tmem + c * 32, v);
                    float s = 0.f;
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float l = __uint_as_float(v[j]) * sc;
                        const float e = l == mx ? 1.0f : expf(l - mx);      // also for an infinite maximum
                        if (!skip(c * 32 + j)) s += e;
                    }
                    sum += s;
                }
                if (m < a.M) {
                    ConfPartial p;
                    p.m = mx; p.s = sum; p.idx = idx;
                    if (po.n == 0) {
                        a.ce.part[static_cast<size_t>(m) * (2 * a.n_pairs) + tile] = p;
                    } else {
                        for (int r = 0; r < po.n; ++r) po.conf[r][static_cast<size_t>(m) * a.ce.tiles_total + a.ce.tile0 + tile] = p;
                    }
                }
            }
            // the accumulator has been read: the next but one tile may overwrite it
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(free_bar + b * 8);
        }
        if ((EPI == ROWS_CONF || EPI == ROWS_PARTIAL) && po.n > 0) {   // uniform: the stores of all eight warps, then one arrival for the CTA
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (threadIdx.x == 64) tp_arrive_and_signal(po, gridDim.x);
        }
    }
    pdl_wait();   // every thread: keeps completion of the launch chain transitive
    tc_fence_before();
    __syncthreads();
    cluster_barrier();   // neither CTA's shared memory or TMEM goes away while its peer may touch it
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_acc), "r"(kRowsTmemCols) : "memory");
    }
}

int sm_pairs() {
    static std::atomic<int> n{0};
    int v = n.load(std::memory_order_relaxed);
    if (!v) {
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess) v = sms / 2;
        if (v < 1) v = 74;
        n.store(v, std::memory_order_relaxed);
    }
    return v;
}

// Launches of up to this many rounds hand out single weight tiles in their last one.  Such an item takes about 0.7 of a whole
// one, and a launch that knows both kinds is 3 to 4 % slower on the whole ones.  Measured (us; without / with): one round or
// less, refresh of 160 rows at d 256 82 / 74, d 1024 98 / 89, of 1100 rows at d 1024 157 / 142; up to two, refresh at d 2048 350 rows
// 150 / 143.5, 500 rows 153 / 147, at d 4096 160 rows 180 / 174; O and down of 4096 rows at d 4096 (3.5 rounds) 106 / 107, 292 / 296.
constexpr int kHalvesRounds = 2;

// items handed out as single weight tiles, of `items` whole ones: the last round's, if they still are one round as halves
int half_items(long long items, int pairs) {
    const int left = static_cast<int>(items % pairs);
    return 2 * left <= pairs && items <= static_cast<long long>(kHalvesRounds) * pairs ? left : 0;
}

template <int EPI>
cudaError_t launch_rows(const GemmArgs& g, int n_tiles, cudaStream_t st) {
    CUtensorMap tmx;
    cudaError_t e = make_rows_tmap(&tmx, g.x, g.M, g.K, kBM);
    if (e != cudaSuccess) return e;
    RowsArgs a;
    a.partial = g.partial; a.act_out = g.act_out; a.ce = g.conf; a.rs = g.row_scale; a.add_to = g.add_to;
    a.qkv = g.qkv ? *g.qkv : QkvRopeArgs();
    a.M = g.M; a.N = g.N;
    a.nkb_total = (g.K + kBK - 1) / kBK;
    a.nkb_per_split = (a.nkb_total + g.splits - 1) / g.splits;
    if (a.nkb_per_split * (g.splits - 1) >= a.nkb_total) return cudaErrorInvalidValue;   // an empty split
    uintptr_t low = static_cast<uintptr_t>(4 * g.N) | reinterpret_cast<uintptr_t>(g.partial);
    for (int r = 0; r < g.peers.n; ++r) low |= reinterpret_cast<uintptr_t>(g.peers.partial[r]);
    a.wide = (low & 15) == 0;
    a.n_pairs = n_tiles / 2;
    a.m_tiles = (g.M + 2 * kBM - 1) / (2 * kBM);
    // row tiles per group: 8 x 256 rows x K x 2 B stay in L2 (refresh of one layer over 25568 rows with groups of 4 / 8 / 16:
    // 10.7 / 10.2 / 10.25 ms)
    a.group = a.m_tiles < 8 ? a.m_tiles : 8;
    a.status = g.status;
    // with several row tiles a weight tile is read once per row tile of its group, by pairs a few microseconds apart:
    // marked "first to be evicted", as in the single-pass kernels, it came from HBM 4.5 times per group (25568 rows,
    // SwiGLU: 11.5 GB; refresh of 16 sequences 11.2 ms against 10.2)
    a.w_hint = a.m_tiles > 1 ? kEvictNormal : kEvictFirst;
    const long long items = static_cast<long long>(a.n_pairs) * a.m_tiles * g.splits;
    if (items > (1ll << 30)) return cudaErrorInvalidValue;
    const int pairs = sm_pairs(), left = EPI == ROWS_CONF ? 0 : half_items(items, pairs);
    const bool halves = left > 0;
    a.whole = static_cast<int>(items) - left;
    a.n_items = static_cast<int>(items) + left;
    constexpr int smem = kRowsStages * kRowsStageBytes + 8 * kPatchBytes + sizeof(RowsShared) + 1024;
    static_assert(smem <= 227 * 1024, "one CTA per SM");
    void (*kernel)(WeightMaps, CUtensorMap, RowsArgs, PeerOut) = gemm_rows_kernel<EPI, false>;
    if constexpr (EPI != ROWS_CONF) {
        if (halves) kernel = gemm_rows_kernel<EPI, true>;
    }
    static std::atomic<unsigned long long> attr_done[2];
    e = set_smem_limit_once(attr_done[halves], kernel, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * static_cast<unsigned>(a.n_items < pairs ? a.n_items : pairs));
    cfg.blockDim = dim3(kRowsThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, g.w, tmx, a, g.peers);
}

}  // namespace

// K splits of the O and down projections of a forward over more than 128 rows without LM head: the cheapest by two terms, the rounds of the CTA
// pairs (0.45 us per k-block of 256 x 256; a last round of single weight tiles counts 0.68) and the sums themselves (1 us per split
// and million of them: written, and read by the norm behind; an unsplit product's go into the residual stream, which is
// as much).  At least eight k-blocks each.  Fitted to and checked against 60 sweeps of one projection's splits, d 1024, 2048 and
// 4096 and 160 to 3600 rows: on average 0.12 % of the refresh behind the best split, 1.3 % at worst.  Against as many splits as
// make 296 tiles, the rule of gemm_pick_splits (us per refresh, before / now; one layer at d 4096, two below): d 4096 900 rows, O 2 -> 1
// splits 449 / 437, down 2 -> 1 449 / 437; 1200 rows, down 1 -> 4 601 / 573 (three 569); d 2048 512
// rows, down 7 -> 4 240 / 232, 2000 rows, O 2 -> 1 528 / 506; d 1024 3600 rows, down 2 -> 1 369 / 353.
// Beyond 2048 rows, or two rounds of unsplit tiles, none: the power cap makes the sums' traffic dearer than idle pairs.  By the two terms
// alone d 4096, 4096 rows would take two for down (step of 16 sequences 1724, unsplit 1708), 3000 three (1269, 1227), 2600 two for O (1166,
// 1142); d 2048, 2800 three for down (743, 725).
int gemm_rows_splits(int M, int N, int K) {
    const int pairs = sm_pairs(), nkb = (K + kBK - 1) / kBK;
    const long long tiles = static_cast<long long>((N + 2 * kBM - 1) / (2 * kBM)) * ((M + 2 * kBM - 1) / (2 * kBM));
    int best = 1;
    double least = 0.;
    if (M > 2048 || tiles > 2 * pairs) return 1;
    for (int sp = 1; sp <= kMaxKSplits && (sp == 1 || 8 * sp <= nkb); ++sp) {
        if (gemm_whole_splits(sp, nkb) != sp) continue;
        const long long items = tiles * sp;
        const double rounds = half_items(items, pairs) ? items / pairs + 0.68 : static_cast<double>((items + pairs - 1) / pairs);
        const double cost = rounds * 0.45 * ((nkb + sp - 1) / sp) + 1e-6 * sp * M * N;
        if (sp == 1 || cost < least) { best = sp; least = cost; }
    }
    return best;
}

// More than 128 rows and an even number of weight tiles.  Inside a model every row starts on a 16-byte boundary (d and F
// are multiples of 16, heads have 64 or 128 dims); the GEMM entry points take any N.
cudaError_t launch_gemm_rows(const GemmArgs& a, int n_tiles, cudaStream_t st) {
    if (a.act_out) return launch_rows<ROWS_SWIGLU>(a, n_tiles, st);
    if (a.qkv) return a.qkv->hd == 128 ? launch_rows<ROWS_QKV128>(a, n_tiles, st) : launch_rows<ROWS_QKV64>(a, n_tiles, st);
    if (a.add_to) return launch_rows<ROWS_ADD>(a, n_tiles, st);
    if (a.conf.part) return launch_rows<ROWS_CONF>(a, n_tiles, st);
    return launch_rows<ROWS_PARTIAL>(a, n_tiles, st);
}

}  // namespace odb
