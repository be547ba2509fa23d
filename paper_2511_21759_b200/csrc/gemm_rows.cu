// Many-row projection (more than 128 activation rows) as CTA pairs, with the ACTIVATION rows on the M side of the
// tensor-core tile.
//
// The pair kernel of gemm_tcgen05.cu gives the M side to the weights; its accumulator then has one weight row per
// TMEM lane and an epilogue thread owns one output FEATURE of many rows: SwiGLU has to fetch the matching up value
// from another warp through shared memory behind block barriers (half of the epilogue warps idle), the confidence
// statistics need a transpose, and every bf16 store is a 2-byte store.  Here the two operands of the same MMA change
// places: a cluster of two CTAs issues one tcgen05.mma.cta_group::2 of 256 activation rows x 256 weight rows, each
// CTA staging 128 activation rows (A) and one packed weight tile of 128 rows (its half of B), so the bytes staged and
// the MMA rate are the ones of the other kernel, and lane r of a CTA's accumulator is its activation row r with 256
// features in consecutive columns.  A thread owns a row: gate and up (a packed gate/up tile is 64 gate then 64 up
// rows), the row's RMSNorm scalar and a whole vocabulary tile's logits are its own, the four epilogue warps share no
// data and meet at no barrier.  Results leave through a 4 KB patch of the (then idle) stage ring per warp, so that
// stores are 16 bytes wide and cover whole 128-byte lines.  The sums are the same products in the same order.
//
// Bound: tensor cores (operand staging 131 FLOP per byte).  Two CTAs per SM, 3 stages x 32 KB each.
// Measured against the other kernel (8B shape, one launch): SwiGLU at 768 / 4096 / 25568 rows 154 -> 118, 793 -> 603
// and 4523 -> 3640 us (1.31, 1.37 and 1.41 PFLOP/s); LM head with statistics at 256 rows 321 -> 268 us.
#include <stdlib.h>

#include "odb_internal.cuh"
#include "tcgen05_common.cuh"

namespace odb {

namespace {

constexpr int kRowsN = 256;                              // weight rows of a pair's tile (two packed tiles)
constexpr uint32_t kTileBytes = kBM * kBK * 2;           // 16 KB: a packed weight tile, and 128 activation rows
constexpr uint32_t kRowsStageBytes = 2 * kTileBytes;
constexpr int kRowsStages = 3;                           // 96 KB: two CTAs per SM
constexpr uint32_t kRowsTmemCols = kRowsN;

constexpr int ROWS_SWIGLU = 0, ROWS_CONF = 1;

struct alignas(8) RowsShared {
    uint64_t full[kRowsStages];
    uint64_t empty[kRowsStages];
    uint64_t acc_full;
    uint32_t tmem_base;
    int abort;
};

struct RowsArgs {
    __nv_bfloat16* act_out;      // ROWS_SWIGLU: bf16 [M][N = F]
    ConfEpilogue ce;             // ROWS_CONF
    RowScale rs;
    int M, N, nkb;
    int n_pairs, m_tiles;        // pairs of weight tiles, tiles of 256 rows
    int* status;
};

// One 128-byte piece of 32 rows: lane r holds row r's piece in v.  It is turned in shared memory (16-byte chunks,
// XOR-swizzled: no bank conflicts either way) so that eight lanes store one row's 128 bytes; sink(row of the warp,
// 16-byte chunk of the piece, value) stores.  buf alternates between two patches, so one barrier per piece is enough.
template <class Sink>
__device__ __forceinline__ void store_rows(uint8_t* buf, const uint32_t (&v)[32], int lane, Sink&& sink) {
    const uint32_t base = smem_u32(buf);
#pragma unroll
    for (int c = 0; c < 8; ++c)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(base + lane * 128 + ((c ^ (lane & 7)) << 4)), "r"(v[4 * c]),
                     "r"(v[4 * c + 1]), "r"(v[4 * c + 2]), "r"(v[4 * c + 3])
                     : "memory");
    __syncwarp();
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

__device__ __forceinline__ void tmem_read32(uint32_t taddr, uint32_t (&v)[32]) {
    tmem_ld32(taddr, v);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

template <int EPI>
__global__ void __launch_bounds__(kThreads, 2)
gemm_rows_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ RowsArgs a,
                 const __grid_constant__ PeerOut po) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    RowsShared* sh = reinterpret_cast<RowsShared*>(ring + kRowsStages * kRowsStageBytes);
    const uint32_t rank = cluster_ctarank();
    const bool leader = rank == 0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // grid (2, row tiles of a group, weight-tile pairs x row-tile groups), scheduled in that order: the row
    // tiles of a group run side by side on one weight-tile pair (its weights come from HBM once) and a group's
    // activation rows (a few MB) stay in L2 while every weight-tile pair passes over them
    const int pair = static_cast<int>(blockIdx.z) % a.n_pairs;
    const int m_tile = static_cast<int>(blockIdx.z) / a.n_pairs * static_cast<int>(gridDim.y) + static_cast<int>(blockIdx.y);
    if (m_tile >= a.m_tiles) {   // ragged last group: both CTAs of the pair leave together
        if (po.n > 0 && threadIdx.x == 0) {
            pdl_wait();   // the arrival counter is shared with the previous exchanging launch: count only once that one is complete
            tp_arrive_and_signal(po, gridDim.x * gridDim.y * gridDim.z);
        }
        return;
    }
    const int nkb = a.nkb;
    const int m0 = m_tile * 2 * kBM + static_cast<int>(rank) * kBM;   // first activation row of this CTA
    const int wtile0 = (2 * pair + static_cast<int>(rank)) * nkb;
    volatile int* cta_abort = &sh->abort;

    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        for (int i = 0; i < kRowsStages; ++i) {
            mbar_init(&sh->full[i], 1);
            mbar_init(&sh->empty[i], 1);
        }
        mbar_init(&sh->acc_full, 1);
        sh->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmap_w)) : "memory");
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
    cluster_barrier();   // the peer's barriers are initialised before anything signals them
    const uint32_t tmem_acc = sh->tmem_base;

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer: weight tiles first (they do not depend on the preceding kernel), then the rows ----
            const int pre = nkb < kRowsStages ? nkb : kRowsStages;
            for (int i = 0; i < pre; ++i) {
                if (leader) mbar_expect_tx(&sh->full[i], 2 * kRowsStageBytes);   // the loads of both CTAs report to the leader
                tma_load_3d_pair(ring + i * kRowsStageBytes, &tmap_w, &sh->full[i], 0, 0, wtile0 + i, kEvictFirst);
            }
            pdl_wait();
            for (int i = 0; i < pre; ++i)
                tma_load_2d_pair(ring + i * kRowsStageBytes + kTileBytes, &tmap_x, &sh->full[i], i * kBK, m0, kEvictLast);
            int st = 0, issued = pre;
            uint32_t ph = 0;   // fills of the ring completed so far, parity
            for (int i = pre; i < nkb; ++i) {
                if (!mbar_wait(&sh->empty[st], ph, cta_abort, a.status)) break;
                uint8_t* dst = ring + st * kRowsStageBytes;
                if (leader) mbar_expect_tx(&sh->full[st], 2 * kRowsStageBytes);
                tma_load_3d_pair(dst, &tmap_w, &sh->full[st], 0, 0, wtile0 + i, kEvictFirst);
                tma_load_2d_pair(dst + kTileBytes, &tmap_x, &sh->full[st], i * kBK, m0, kEvictLast);
                issued = i + 1;
                if (++st == kRowsStages) { st = 0; ph ^= 1u; }
            }
            if (*cta_abort && leader) {
                // aborted: let the copies still in flight land before the CTA's shared memory goes away (the
                // peer cannot observe its own copies; it is held by the cluster barrier at the end)
                const int first = issued > kRowsStages ? issued - kRowsStages : 0;
                for (int i = first; i < issued; ++i) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait_parity(&sh->full[i % kRowsStages], static_cast<uint32_t>(i / kRowsStages) & 1u) &&
                           clock64() - t0 < kWaitLimitCycles / 8) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && leader) {
            // ---- MMA issuer (the leader's, for both CTAs): A = activation rows, B = weight rows ----
            constexpr uint32_t idesc = make_instr_desc(2 * kBM, kRowsN);
            bool ok = true;
            int st = 0;
            uint32_t ph = 0;
            for (int i = 0; i < nkb; ++i) {
                ok = mbar_wait(&sh->full[st], ph, cta_abort, a.status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t w_addr = smem_u32(ring + st * kRowsStageBytes), x_addr = w_addr + kTileBytes;
#pragma unroll
                for (int k = 0; k < kBK / kUmmaK; ++k)
                    umma_bf16_pair(tmem_acc, make_smem_desc(x_addr + k * kUmmaK * 2), make_smem_desc(w_addr + k * kUmmaK * 2), idesc,
                                   (i > 0 || k > 0) ? 1u : 0u);
                umma_commit_pair(&sh->empty[st]);   // frees the stage in both CTAs once these MMAs have read it
                if (++st == kRowsStages) { st = 0; ph ^= 1u; }
            }
            if (ok) umma_commit_pair(&sh->acc_full);
        }
    } else {
        // ---- epilogue: warps 2..5 own TMEM lanes 32 * (warp % 4) .. + 31 = activation rows ----
        const int q = warp & 3;
        const int mw = m0 + q * 32;                          // the warp's first row
        const int m = mw + lane;
        const uint32_t tmem = tmem_acc + (static_cast<uint32_t>(q * 32) << 16);
        pdl_wait();   // the previous reader of the output buffer has finished; the predecessor's results are visible
        const float sc = m < a.M ? row_scale_of(a.rs, m) : 1.0f;
        const bool ok = __all_sync(0xffffffffu, mbar_wait(&sh->acc_full, 0, cta_abort, a.status));
        if (ok) {
            tc_fence_after();
            // every MMA of both CTAs has completed, so the stage ring is free
            uint8_t* patch = ring + q * 8192;
            if constexpr (EPI == ROWS_SWIGLU) {
#pragma unroll 1
                for (int t = 0; t < 2; ++t) {
                    const int f0 = (2 * pair + t) * 64;
                    uint32_t out[32];                        // 64 features of this row
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        uint32_t g[32], u[32];
                        tmem_ld32(tmem + t * 128 + half * 32, g);
                        tmem_ld32(tmem + t * 128 + 64 + half * 32, u);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int j = 0; j < 32; j += 2) {
                            const float g0 = __uint_as_float(g[j]) * sc, g1 = __uint_as_float(g[j + 1]) * sc;
                            const float u0 = __uint_as_float(u[j]) * sc, u1 = __uint_as_float(u[j + 1]) * sc;
                            const __nv_bfloat162 y = __floats2bfloat162_rn(g0 / (1.0f + expf(-g0)) * u0, g1 / (1.0f + expf(-g1)) * u1);
                            out[half * 16 + j / 2] = *reinterpret_cast<const uint32_t*>(&y);
                        }
                    }
                    store_rows(patch + t * 4096, out, lane, [&](int r, int ch, const uint4& x) {
                        const int f = f0 + ch * 8;
                        if (mw + r < a.M && f < a.N)         // F % 16 == 0
                            *reinterpret_cast<uint4*>(a.act_out + static_cast<size_t>(mw + r) * a.N + f) = x;
                    });
                }
            } else {
                // LM head: softmax statistics of each 128-entry vocabulary tile of this thread's row: maximum and argmax
                // (ascending ids, strict: lowest id on ties) in one pass over the tile, the sum of exponentials in a second
#pragma unroll 1
                for (int t = 0; t < 2; ++t) {
                    const int tile = 2 * pair + t, n0 = tile * kBM, id0 = n0 + a.ce.tile0 * kBM;
                    // ids the statistics leave out: the padding behind the vocabulary, [MASK]
                    const bool whole = n0 + kBM <= a.N && (a.ce.mask_id < id0 || a.ce.mask_id >= id0 + kBM);
                    auto skip = [&](int i) { return !whole && (n0 + i >= a.N || id0 + i == a.ce.mask_id); };
                    float mx = -INFINITY, sum = 0.f;
                    int idx = 0x7fffffff;
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        uint32_t v[32];
                        tmem_read32(tmem + t * 128 + c * 32, v);
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const float l = __uint_as_float(v[j]) * sc;
                            if (l > mx && !skip(c * 32 + j)) { mx = l; idx = id0 + c * 32 + j; }
                        }
                    }
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        uint32_t v[32];
                        tmem_read32(tmem + t * 128 + c * 32, v);
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
            }
        }
        if (EPI != ROWS_SWIGLU && po.n > 0) {   // uniform: the stores of all four warps, then one arrival for the CTA
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (threadIdx.x == 64) tp_arrive_and_signal(po, gridDim.x * gridDim.y * gridDim.z);
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

template <int EPI>
cudaError_t launch_rows(const GemmArgs& g, int n_tiles, cudaStream_t st) {
    CUtensorMap tmx;
    cudaError_t e = make_rows_tmap(&tmx, g.x, g.M, g.K, kBM);
    if (e != cudaSuccess) return e;
    RowsArgs a;
    a.act_out = g.act_out; a.ce = g.conf; a.rs = g.row_scale;
    a.M = g.M; a.N = g.N;
    a.nkb = (g.K + kBK - 1) / kBK;
    a.n_pairs = n_tiles / 2;
    a.m_tiles = (g.M + 2 * kBM - 1) / (2 * kBM);
    a.status = g.status;
    constexpr int smem = kRowsStages * kRowsStageBytes + sizeof(RowsShared) + 1024;
    static std::atomic<unsigned long long> attr_done{0};
    e = set_smem_limit_once(attr_done, gemm_rows_kernel<EPI>, smem);
    if (e != cudaSuccess) return e;
    // row tiles per group: 8 x 256 rows x K x 2 B stay in L2 (measured at 128 row tiles: groups of 2 / 4 / 8 / 16
    // give 430 / 414 / 404 / 407 ms of GEMM time per refresh, no grouping 475, one row tile per weight pass 462)
    const int group = a.m_tiles < 8 ? a.m_tiles : 8;
    const int m_groups = (a.m_tiles + group - 1) / group;
    const size_t z = static_cast<size_t>(a.n_pairs) * m_groups;
    if (z > 65535) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2, group, static_cast<unsigned>(z));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;   // neighbouring weight tiles form the pair
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, gemm_rows_kernel<EPI>, g.tmap_w, tmx, a, g.peers);
}

}  // namespace

// SwiGLU and LM-head projections with an even number of weight tiles (pairs) and more than 128 rows.  fp32 partial sums
// stay with gemm_kernel: its epilogue (a feature per thread) stores them without a detour and measured 3 % faster.
bool gemm_rows_supported(const GemmArgs& a, int n_tiles) {
    if (a.M <= 128 || (n_tiles & 1) || a.splits != 1) return false;
    if (a.act_out) return (a.N & 7) == 0 && (reinterpret_cast<uintptr_t>(a.act_out) & 15) == 0;   // 16-byte stores
    return a.conf.part != nullptr;
}

cudaError_t launch_gemm_rows(const GemmArgs& a, int n_tiles, cudaStream_t st) {
    if (a.act_out) return launch_rows<ROWS_SWIGLU>(a, n_tiles, st);
    return launch_rows<ROWS_CONF>(a, n_tiles, st);
}

}  // namespace odb
