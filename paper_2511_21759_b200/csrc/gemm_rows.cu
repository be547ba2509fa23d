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
// rows), the row's RMSNorm scalar and a whole vocabulary tile's logits are its own, the epilogue warps share no data
// and meet at no barrier.  Results leave through a 4 KB patch of the (then idle) stage ring per warp, so that
// stores are 16 bytes wide and cover whole 128-byte lines.  The sums are the same products in the same order.
//
// Bound: tensor cores (operand staging 131 FLOP per byte).  Two CTAs per SM, 3 stages x 32 KB each.
// Eight epilogue warps (two per 32 TMEM lanes, one packed weight tile each): with four, the QKV epilogue below took 20 us
// longer at 768 rows, where the single wave of CTAs leaves it exposed (59 against 76 us).
// Measured against the other kernel (8B shape, one launch each):
//   SwiGLU at 768 / 4096 / 25568 rows        154 -> 111, 793 -> 573, 4523 -> 3604 us (1.39, 1.44, 1.43 PFLOP/s)
//   LM head + statistics at 256 rows          321 -> 245 us
//   QKV + RoPE + cache scatter, same rows      72 -> 59, 330 -> 300, 2170 -> 1868 us (projection and RoPE kernel before)
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
constexpr int kRowsThreads = 320;                        // TMA warp, MMA warp, eight epilogue warps (two per 32 TMEM lanes)

constexpr int ROWS_SWIGLU = 0, ROWS_CONF = 1, ROWS_ADD = 2, ROWS_QKV64 = 3, ROWS_QKV128 = 4;

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
    float* add_to;               // ROWS_ADD: fp32 [M][N], the residual stream
    QkvRopeArgs qkv;             // ROWS_QKV64 / ROWS_QKV128 (head dim)
    RowScale rs;
    int M, N, nkb;
    int n_pairs, m_tiles;        // pairs of weight tiles, tiles of 256 rows
    int* status;
};

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
// put, meet, take.  Callers alternate between two buffers, so that one warp barrier per piece is enough.
template <class Sink>
__device__ __forceinline__ void store_rows(uint8_t* buf, const uint32_t (&v)[32], int lane, Sink&& sink) {
#pragma unroll
    for (int c = 0; c < 8; ++c) put_chunk(buf, lane, c, v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
    __syncwarp();
    take_rows(buf, lane, sink);
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

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void tmem_read32(uint32_t taddr, uint32_t (&v)[32]) {
    tmem_ld32(taddr, v);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

template <int EPI>
__global__ void __launch_bounds__(kRowsThreads, 2)
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
        // ---- epilogue: warps 2..9 own TMEM lanes 32 * (warp % 4) .. + 31 = activation rows, and the 128 columns of
        // packed weight tile 2 * pair + t ----
        const int q = warp & 3, t = (warp - 2) >> 2;
        const int mw = m0 + q * 32;                          // the warp's first row
        const int m = mw + lane;
        const int tile = 2 * pair + t;
        const uint32_t tmem = tmem_acc + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(t * kBM);
        pdl_wait();   // the previous reader of the output buffer has finished; the predecessor's results are visible
        const float sc = m < a.M ? row_scale_of(a.rs, m) : 1.0f;
        const bool ok = __all_sync(0xffffffffu, mbar_wait(&sh->acc_full, 0, cta_abort, a.status));
        if (ok) {
            tc_fence_after();
            // every MMA of both CTAs has completed, so the stage ring is free
            uint8_t* patch = ring + (warp - 2) * 8192;
            if constexpr (EPI == ROWS_SWIGLU) {
#pragma unroll 1
                for (int c = 0; c < 64; c += 16) {
                    uint32_t g[16], u[16];
                    tmem_ld16(tmem + c, g);
                    tmem_ld16(tmem + 64 + c, u);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    uint32_t out[8];
#pragma unroll
                    for (int j = 0; j < 16; j += 2) {
                        const float g0 = __uint_as_float(g[j]) * sc, g1 = __uint_as_float(g[j + 1]) * sc;
                        const float u0 = __uint_as_float(u[j]) * sc, u1 = __uint_as_float(u[j + 1]) * sc;
                        out[j / 2] = pack2(g0 / (1.0f + expf(-g0)) * u0, g1 / (1.0f + expf(-g1)) * u1);
                    }
                    put_chunk(patch, lane, c / 8, out[0], out[1], out[2], out[3]);
                    put_chunk(patch, lane, c / 8 + 1, out[4], out[5], out[6], out[7]);
                }
                __syncwarp();
                take_rows(patch, lane, [&](int r, int ch, const uint4& x) {
                    const int f = tile * 64 + ch * 8;
                    if (mw + r < a.M && f < a.N)             // F % 16 == 0
                        *reinterpret_cast<uint4*>(a.act_out + static_cast<size_t>(mw + r) * a.N + f) = x;
                });
            } else if constexpr (EPI == ROWS_ADD) {
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    const int nc = tile * kBM + c * 32;
                    if (nc >= a.N) break;
                    uint32_t v[32];
                    tmem_read32(tmem + c * 32, v);
                    store_rows(patch + (c & 1) * 4096, v, lane, [&](int r, int ch, const uint4& x) {
                        const int n = nc + ch * 4;
                        if (mw + r < a.M && n < a.N) red_add4(a.add_to + static_cast<size_t>(mw + r) * a.N + n, x);   // N % 4 == 0
                    });
                }
            } else if constexpr (EPI == ROWS_QKV64 || EPI == ROWS_QKV128) {
                // QKV projection: a head's q, k or v of this row is the thread's own, rotate-half partners included.
                // The RMSNorm scalar, RoPE (q and k), bf16 rows and - in a refresh - the K/V cache.  The (cos, sin) table
                // is read transposed ([pair][position]): the lanes' positions are neighbours, mostly.
                constexpr int HD = EPI == ROWS_QKV128 ? 128 : 64, kHalf = HD / 2;
                const QkvRopeArgs& e = a.qkv;
                const int pos = m < a.M ? e.row_pos[m] : 0, seq = m < a.M ? e.row_seq[m] : 0;
                const long long crow = (static_cast<long long>(seq) * e.n_layers + e.layer) * 2 * e.H * e.max_seq + pos;
                const float2* rope = e.rope_t + pos;
#pragma unroll 1
                for (int grp = 0; grp < kBM / HD; ++grp) {
                    const int g = tile * (kBM / HD) + grp;             // head of [Wq; Wk; Wv]
                    if (g >= 3 * e.H) break;
                    const int sec = g / e.H, head = g - sec * e.H;
                    uint8_t* buf = patch + grp * 4096;                 // one group of two pieces, or two of one
#pragma unroll 1
                    for (int c = 0; c < kHalf; c += 16) {
                        uint32_t lo[16], hi[16];
                        tmem_ld16(tmem + grp * HD + c, lo);
                        tmem_ld16(tmem + grp * HD + kHalf + c, hi);
                        float2 cs[16];
                        if (sec < 2) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) cs[j] = rope[static_cast<size_t>(c + j) * e.max_seq];
                        }
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
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
                        uint8_t* bh = HD == 128 ? buf + 4096 : buf;    // where the upper half of the head goes
                        const int ch = c / 8, chh = HD == 128 ? ch : ch + 4;
                        put_chunk(buf, lane, ch, pl[0], pl[1], pl[2], pl[3]);
                        put_chunk(buf, lane, ch + 1, pl[4], pl[5], pl[6], pl[7]);
                        put_chunk(bh, lane, chh, ph[0], ph[1], ph[2], ph[3]);
                        put_chunk(bh, lane, chh + 1, ph[4], ph[5], ph[6], ph[7]);
                    }
                    __syncwarp();
                    __nv_bfloat16* fresh = (sec == 0 ? e.q : sec == 1 ? e.k : e.v) + head * HD;
                    const long long chead = static_cast<long long>((sec - 1) * e.H + head) * e.max_seq;
#pragma unroll
                    for (int piece = 0; piece < HD / 64; ++piece)
                        take_rows(buf + piece * 4096, lane, [&](int r, int ch, const uint4& x) {
                            const long long cr = __shfl_sync(0xffffffffu, crow, r);
                            if (mw + r >= a.M) return;
                            *reinterpret_cast<uint4*>(fresh + static_cast<size_t>(mw + r) * (e.H * HD) + piece * 64 + ch * 8) = x;
                            if (e.cache && sec > 0) *reinterpret_cast<uint4*>(e.cache + (cr + chead) * HD + piece * 64 + ch * 8) = x;
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
        }
        if (EPI == ROWS_CONF && po.n > 0) {   // uniform: the stores of all eight warps, then one arrival for the CTA
            asm volatile("bar.sync 1, 256;" ::: "memory");
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
    a.add_to = g.add_to;
    if (g.qkv) a.qkv = *g.qkv;
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
    cfg.blockDim = dim3(kRowsThreads);
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

// Projections with an even number of weight tiles (pairs) and more than 128 rows whose epilogue gains from owning rows.
// fp32 partial sums (K splits) stay with gemm_kernel: its epilogue (a feature per thread) stores them without a detour
// and measured 3 % faster.  All row starts are 16-byte aligned: d, F multiples of 16, heads of 64 or 128.
bool gemm_rows_supported(const GemmArgs& a, int n_tiles) {
    return a.M > 128 && (n_tiles & 1) == 0 && a.splits == 1 && (a.act_out || a.conf.part || a.qkv || a.add_to);
}

cudaError_t launch_gemm_rows(const GemmArgs& a, int n_tiles, cudaStream_t st) {
    if (a.act_out) return launch_rows<ROWS_SWIGLU>(a, n_tiles, st);
    if (a.qkv) return a.qkv->hd == 128 ? launch_rows<ROWS_QKV128>(a, n_tiles, st) : launch_rows<ROWS_QKV64>(a, n_tiles, st);
    if (a.add_to) return launch_rows<ROWS_ADD>(a, n_tiles, st);
    return launch_rows<ROWS_CONF>(a, n_tiles, st);
}

}  // namespace odb
