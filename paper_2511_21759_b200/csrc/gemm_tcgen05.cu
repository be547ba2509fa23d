// Weight-streaming GEMM for sm_100a: TMA -> shared memory -> tcgen05.mma -> TMEM -> registers.
//
// Computes, for every K split s,   partial[s][m][n] = sum_{k in split s} x[m][k] * w[n][k]
// with x the bf16 activations [M][K] (few rows: block_len * copies in a decode step; all
// positions in a refresh) and w a bf16 weight matrix [N][K].  The 128-row side of the tensor
// core tile is given to the WEIGHTS (they are the large, streamed operand) and the activation
// rows ride on the MMA's N dimension (32..128), so a 32-row decode step wastes no tensor-core
// rows and every weight byte is fetched from HBM exactly once.  Projections of more than 128 rows with
// an even number of weight tiles run as CTA pairs in gemm_rows.cu.
//
// Weights are stored PACKED: tile (n-tile of 128 rows, k-block of 64 columns) is one contiguous
// 16 KB chunk, tiles of a row of tiles consecutive in k.  A CTA therefore reads one sequential
// stream of whole DRAM pages; with the plain row-major layout each TMA box gathers 128 separate
// 128-byte pieces 2K bytes apart and HBM delivers little more than half its bandwidth (measured).
//
// One CTA = one 128 x BN output tile over one K range.  Warp 0 lane 0 issues TMA loads into two
// rings of shared-memory stages (weights, activation rows), warp 1 lane 0 issues the MMAs (accumulator in TMEM) and
// frees stages through tcgen05.commit, the other warps read the accumulator back (tcgen05.ld) and store
// fp32 partials.  Splits are reduced later in a fixed order by the consumer kernel, so results
// are run-to-run identical.  Every mbarrier wait is bounded: on expiry the CTA records
// ODB_ERR_TIMEOUT, stops issuing work, releases its TMEM and exits.
#include <stdlib.h>

#include "norm_common.cuh"
#include "tcgen05_common.cuh"

namespace odb {

namespace {

constexpr int kMaxStages = 5;

struct alignas(8) GemmShared {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t acc_full;
    uint32_t tmem_base;
    int abort;
    float scale[128];      // RowScale of the tile's activation rows
};

// BN: activation rows per tile (MMA N): 32, 64 or 128, or as many less as a launch of a single row tile has (x_rows).
// SWIGLU: the weight is the gate/up matrix packed with gate and up rows interleaved in groups of
// 64 (tile t = gate rows [64t, 64t+64) then up rows [64t, 64t+64)); the epilogue pairs TMEM lane r
// (gate) with lane r + 64 (up) through shared memory and stores bf16(silu(gate) * up) to
// g[m][64 t + r]; N is then the FFN width F and there is no K split.
constexpr int EPI_PARTIAL = 0, EPI_SWIGLU = 1, EPI_CONF = 3;
constexpr int kMinStages = 3;

// Groups of four epilogue warps; group g takes the activation rows [g, g + 1) * BN / groups of the tile.  Every CTA of a
// one-wave launch ends at the same time, so an epilogue is paid in full: with four warps the gate/up projection of 128 rows had
// 14 us that did not grow with K, of 32 rows 7.  Measured (8B shape, us): gate/up at 128 rows 46.5 with one group, 41.3 with
// two, 41.0 with four; at 64 rows 38.5 -> 36.1; LM head at 128 rows 220 / 190 / 175, at 64 rows 184 -> 163 (32 rows: 161).
// The partial sums' epilogue is stores alone: more warps make it slower (QKV at 128 rows 21.3 -> 22.4).
__host__ __device__ constexpr int epilogue_groups(int bn, int epi) {
    return bn == 32 || epi == EPI_PARTIAL ? 1 : bn == 128 && epi == EPI_CONF ? 4 : 2;
}
__host__ __device__ constexpr int gemm_threads(int bn, int epi) { return 64 + 128 * epilogue_groups(bn, epi); }

template <int BN, int EPI>
__global__ void __launch_bounds__(gemm_threads(BN, EPI), 2)
gemm_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
            float* __restrict__ partial, __nv_bfloat16* __restrict__ act_out, RowScale rs,
            ConfEpilogue ce, int M, int N, int nkb_total, int nkb_per_split, int x_rows, int w_stages, int x_stages,
            int l2_prefetch, int* status, const __grid_constant__ PeerOut po, const __grid_constant__ NormOut no) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    constexpr uint32_t kABytes = kBM * kBK * 2;
    // x_rows <= BN: activation rows that are loaded and multiplied; the accumulator's columns behind them are never stored
    const uint32_t x_bytes = static_cast<uint32_t>(x_rows) * (kBK * 2);
    const uint32_t stage_bytes = kABytes + x_bytes;
    constexpr uint32_t kLeastStageBytes = kABytes + (BN == 32 ? 16 : BN / 2 + 16) * kBK * 2;
    constexpr uint32_t kTmemCols = BN;
    // the epilogues exchange values through the stage ring, which holds at least kMinStages stages
    constexpr int kGroups = epilogue_groups(BN, EPI), kGroupRows = BN / kGroups;
    constexpr int kNormPitch = 132;                       // floats of a row in the norm's exchange buffer
    static_assert(32 * kNormPitch * 4 <= kMinStages * kABytes, "the norm's exchange buffer must end inside the ring");
    constexpr uint32_t kExchangeBytes = EPI == EPI_SWIGLU ? 2 * 64 * (kGroupRows / 2 + 1) * 4 : EPI == EPI_CONF ? 32 * 129 * 4 : 0;
    static_assert(kGroups * kExchangeBytes <= kMinStages * kLeastStageBytes, "the exchange buffer must end inside the ring");

    // Two rings, not one of whole stages: the weights come from HBM and need more bytes in flight than the activation rows,
    // which come from L2.  No slack for an alignment: the rings end where the second CTA of the SM begins.
    uint8_t* tiles = smem_raw;                                                  // [w_stages][128][64] weights
    uint8_t* xring = tiles + static_cast<size_t>(w_stages) * kABytes;           // [x_stages][x_rows][64] activation rows
    GemmShared* sh = reinterpret_cast<GemmShared*>(xring + static_cast<size_t>(x_stages) * x_bytes);
    if ((smem_u32(smem_raw) & 1023u) != 0) {                // the swizzled tiles need 1024-byte alignment
        if (threadIdx.x == 0) atomicExch(status, ODB_ERR_CUDA);
        pdl_wait();
        return;
    }

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    // work unit of this CTA: grid (weight tiles, row tiles, K splits)
    const int n_tile = static_cast<int>(blockIdx.x), n_tiles = static_cast<int>(gridDim.x);
    const int m_tile = static_cast<int>(blockIdx.y);
    const int n0 = n_tile * kBM;
    const int m0 = m_tile * BN;
    const int split = static_cast<int>(blockIdx.z);
    const int kb0 = split * nkb_per_split;
    int nkb = nkb_total - kb0;
    if (nkb > nkb_per_split) nkb = nkb_per_split;
    volatile int* cta_abort = &sh->abort;
    // packed weights: tile (n-tile, k-block) is the contiguous 16 KB chunk number n_tile * nkb_total + k_block
    const int wtile0 = n_tile * nkb_total + kb0;

    if (threadIdx.x == 0) {
        for (int i = 0; i < w_stages; ++i) {
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
    if (warp == 1) {   // whole warp: allocate the accumulator's TMEM columns
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh->tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        pdl_launch_dependents();   // behind the allocation, as in every kernel that makes one; one thread's word is the CTA's
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_acc = sh->tmem_base;

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer ----
            // The weights do not depend on the preceding kernel: fill the ring with weight tiles
            // first, then wait for the predecessor and fetch the activation tiles.
            const int pre = nkb < w_stages ? nkb : w_stages, xpre = nkb < x_stages ? nkb : x_stages;
            auto load_w = [&](int i, int st) {   // arms the barrier of k-block i for its weights and its activation rows
                mbar_expect_tx(&sh->full[st], stage_bytes);
                tma_load_3d(tiles + static_cast<size_t>(st) * kABytes, &tmap_w, &sh->full[st], 0, 0, wtile0 + i, kEvictFirst);
            };
            auto load_x = [&](int i, int st, int slot) {
                tma_load_2d(xring + static_cast<size_t>(slot) * x_bytes, &tmap_x, &sh->full[st], (kb0 + i) * kBK, m0, kEvictLast);
            };
            for (int i = 0; i < pre; ++i) load_w(i, i);
            // and ask L2 for the weight tiles that follow, so that HBM keeps streaming while the
            // predecessor (a short elementwise kernel) is still running
            int pf = nkb - pre;
            if (pf > l2_prefetch) pf = l2_prefetch;
            for (int i = pre; i < pre + pf; ++i)
                asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(
                                 reinterpret_cast<uint64_t>(&tmap_w)),
                             "r"(0), "r"(0), "r"(wtile0 + i)
                             : "memory");
            pdl_wait();
            for (int i = 0; i < xpre; ++i) load_x(i, i, i);
            // the MMAs of k-block i free its weight stage for k-block i + w_stages and its activation stage for i + x_stages
            int st = 0, slot = 0, xst = x_stages;   // weight stage and activation slot of i; weight stage of i + x_stages
            if (xst >= w_stages) xst -= w_stages;
            uint32_t ph = 0;
            int issued = pre;
            for (int i = 0; i + x_stages < nkb; ++i) {
                if (!mbar_wait(&sh->empty[st], ph, cta_abort, status)) break;
                if (i + w_stages < nkb) {
                    load_w(i + w_stages, st);
                    issued = i + w_stages + 1;
                }
                load_x(i + x_stages, xst, slot);
                if (++st == w_stages) { st = 0; ph ^= 1u; }
                if (++xst == w_stages) xst = 0;
                if (++slot == x_stages) slot = 0;
            }
            if (*cta_abort) {
                // aborted: let the copies still in flight land before the CTA's shared memory goes away (a k-block whose
                // activation rows were never asked for takes its wait's whole limit)
                const int first = issued > w_stages ? issued - w_stages : 0;
                for (int i = first; i < issued; ++i) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait_parity(&sh->full[i % w_stages], static_cast<uint32_t>(i / w_stages) & 1u) &&
                           clock64() - t0 < kWaitLimitCycles / 8) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMA issuer ----
            const uint32_t idesc = make_instr_desc(kBM, x_rows);
            bool ok = true;
            int st = 0, slot = 0;
            uint32_t ph = 0;
            for (int i = 0; i < nkb; ++i) {
                ok = mbar_wait(&sh->full[st], ph, cta_abort, status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a_addr = smem_u32(tiles + static_cast<size_t>(st) * kABytes);
                const uint32_t b_addr = smem_u32(xring + static_cast<size_t>(slot) * x_bytes);
#pragma unroll
                for (int k = 0; k < kBK / kUmmaK; ++k)
                    umma_bf16(tmem_acc, make_smem_desc(a_addr + k * kUmmaK * 2), make_smem_desc(b_addr + k * kUmmaK * 2), idesc,
                              (i > 0 || k > 0) ? 1u : 0u);
                umma_commit(&sh->empty[st]);   // frees both stages once these MMAs have read them
                if (++st == w_stages) { st = 0; ph ^= 1u; }
                if (++slot == x_stages) slot = 0;
            }
            if (ok) umma_commit(&sh->acc_full);
        }
    } else {
        // ---- epilogue: the four warps of a group own TMEM lanes 32*(warp%4) .. +31, and the group's activation rows ----
        const int q = warp & 3;
        const int grp = kGroups == 1 ? 0 : (warp - 2) >> 2, gthread = static_cast<int>(threadIdx.x) - 64 - 128 * grp;
        const int g0 = grp * kGroupRows;                                   // the group's first row within the tile
        auto group_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory"); };
        pdl_wait();   // the previous reader of the output buffer has finished; the predecessor's results are visible
        if (rs.ssq) {   // uniform: row scalars of this tile's activation rows, computed while the main loop runs
            for (int i = g0 + gthread; i < g0 + kGroupRows; i += 128) sh->scale[i] = m0 + i < M ? row_scale_of(rs, m0 + i) : 1.0f;
            group_sync();
        }
        const bool ok = nkb > 0 && mbar_wait(&sh->acc_full, 0, cta_abort, status);   // nkb == 0: empty K split
        if (ok) tc_fence_after();
        if (EPI == EPI_PARTIAL && BN == 32 && no.h) {
            // The whole product of an unsplit projection of one row tile, added to the residual stream here and normalised: what
            // rmsnorm_kernel does, the sums of squares per 128 columns, which is what a warp of that kernel adds up.  One kernel less in
            // the chain.
            float* xch = reinterpret_cast<float*>(tiles);                       // [32 rows][kNormPitch]
            const int col = n0 + lane * 4;                                      // of this lane's four, once a row is a warp's
            const bool in = col < N;                                            // N % 16 == 0
            const bool warp_ok = __all_sync(0xffffffffu, ok);
            const float4 gain = in ? *reinterpret_cast<const float4*>(no.gain + col) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (warp_ok) {
                uint32_t v[32];
                __syncwarp();
                tmem_ld32(tmem_acc + (static_cast<uint32_t>(q * 32) << 16), v);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int j = 0; j < 32; ++j) xch[j * kNormPitch + q * 32 + lane] = __uint_as_float(v[j]);
            }
            group_sync();                                                       // every warp, whether or not its wait succeeded
            float4 x[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int m = r * 4 + q;
                if (in && m < M && warp_ok) x[r] = *reinterpret_cast<const float4*>(no.h + static_cast<size_t>(m) * N + col);
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int m = r * 4 + q;
                float ss = 0.f;
                if (in && m < M && warp_ok) {
                    const float4 t = *reinterpret_cast<const float4*>(xch + m * kNormPitch + lane * 4);
                    x[r].x += t.x; x[r].y += t.y; x[r].z += t.z; x[r].w += t.w;
                    *reinterpret_cast<float4*>(no.h + static_cast<size_t>(m) * N + col) = x[r];
                    *reinterpret_cast<uint2*>(no.out + static_cast<size_t>(m) * N + col) =
                        pack4_bf16(x[r].x * gain.x, x[r].y * gain.y, x[r].z * gain.z, x[r].w * gain.w);
                    ss = squares4<true>(x[r]);
                }
                ss = warp_sum(ss);
                if (lane == 0 && m < M) no.ssq[static_cast<size_t>(m) * n_tiles + n_tile] = ss;
            }
        } else if constexpr (EPI == EPI_PARTIAL) {
            const int n = n0 + q * 32 + lane;
            if (ok) {
                const size_t split_off = static_cast<size_t>(split) * M * N;
                float* out = partial + split_off;
#pragma unroll 1
                for (int c = g0 / 32; c < (g0 + kGroupRows) / 32; ++c) {
                    uint32_t v[32];
                    __syncwarp();   // tcgen05.ld is a whole-warp instruction, and the stores before are some lanes' only
                    tmem_ld32(tmem_acc + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(c * 32), v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (po.n == 0) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const int m = m0 + c * 32 + j;
                            const float sc = rs.ssq ? sh->scale[c * 32 + j] : 1.0f;
                            if (n < N && m < M) out[static_cast<size_t>(m) * N + n] = __uint_as_float(v[j]) * sc;
                        }
                    } else {
                        // tensor-parallel partial sums: the tile goes to the receive buffer of every rank
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const int m = m0 + c * 32 + j;
                            if (n < N && m < M) {
                                const size_t off = split_off + static_cast<size_t>(m) * N + n;
#pragma unroll 1
                                for (int r = 0; r < po.n; ++r) po.partial[r][off] = __uint_as_float(v[j]);
                            }
                        }
                    }
                }
            }
            if (po.n > 0) {   // uniform: the tile's stores of all epilogue warps, then one arrival for the CTA
                asm volatile("bar.sync 15, %0;" ::"n"(128 * kGroups) : "memory");
                if (threadIdx.x == 64) tp_arrive_and_signal(po, gridDim.x * gridDim.y * gridDim.z);
            }
        } else if constexpr (EPI == EPI_CONF) {
            // LM head fused with the confidence reduction: the logits of this tile (128 vocabulary
            // entries x BN rows) never leave the SM.  They are transposed through shared memory so that
            // four threads scan one row's 128 logits (32 each, ascending ids, online max / sum of exp /
            // argmax); the four are merged in id order and one (max, sum, argmax) triple per (row, tile)
            // is stored.  The RMSNorm scalar of the row is applied first; [MASK] and padding are skipped.
            float* xch = reinterpret_cast<float*>(tiles + grp * kExchangeBytes);   // [32 rows][129]
            const int t = gthread;                                     // 0..127
#pragma unroll 1
            for (int c = g0 / 32; c < (g0 + kGroupRows) / 32; ++c) {
                uint32_t v[32];
                if (ok) {
                    tmem_ld32(tmem_acc + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(c * 32), v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                }
#pragma unroll
                for (int j = 0; j < 32; ++j) xch[j * 129 + q * 32 + lane] = ok ? __uint_as_float(v[j]) : 0.f;
                group_sync();
                const int m_l = t >> 2, part = t & 3;
                const int m = m0 + c * 32 + m_l;
                const float sc = rs.ssq ? sh->scale[c * 32 + m_l] : 1.0f;
                float mx = -INFINITY, sum = 0.f;
                int idx = 0x7fffffff;
#pragma unroll 8
                for (int i = 0; i < 32; ++i) {
                    const int n = n0 + part * 32 + i;
                    const int id = n + ce.tile0 * kBM;                  // vocabulary id (a shard starts at tile0)
                    const float l = xch[m_l * 129 + part * 32 + i] * sc;
                    if (n < N && id != ce.mask_id) {
                        if (l > mx) {
                            sum = sum * expf(mx - l) + 1.0f;            // first element: 0 * exp(-inf) + 1
                            mx = l;
                            idx = id;
                        } else {
                            sum += expf(l - mx);
                        }
                    }
                }
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                    const float om = __shfl_down_sync(0xffffffffu, mx, o, 4);
                    const float os = __shfl_down_sync(0xffffffffu, sum, o, 4);
                    const int oi = __shfl_down_sync(0xffffffffu, idx, o, 4);
                    if (part + o < 4) conf_merge(mx, sum, idx, om, os, oi);
                }
                if (ok && part == 0 && m < M) {
                    ConfPartial p;
                    p.m = mx; p.s = sum; p.idx = idx;
                    if (po.n == 0) {
                        ce.part[static_cast<size_t>(m) * n_tiles + n_tile] = p;
                    } else {
                        for (int r = 0; r < po.n; ++r) po.conf[r][static_cast<size_t>(m) * ce.tiles_total + ce.tile0 + n_tile] = p;
                    }
                }
                group_sync();
            }
            if (po.n > 0) {
                asm volatile("bar.sync 15, %0;" ::"n"(128 * kGroups) : "memory");
                if (threadIdx.x == 64) tp_arrive_and_signal(po, gridDim.x * gridDim.y * gridDim.z);
            }
        } else {
            // All MMAs have completed, so the stage ring is free: the warps that own gate features hand the values of the
            // tile's second half of rows to the warps that own the matching up features, and get the up values of the
            // first half; behind one barrier every warp then finishes its half.  (Up values handed over chunk by chunk
            // behind two barriers each, the up warps idle, in CTA pairs: 50 us for the 8B shape's gate/up projection at
            // 128 rows; this way 47, and 36 instead of 38 at 32 rows.)
            constexpr int kHalfRows = kGroupRows / 2, kPitch = kHalfRows + 1;
            float* xch = reinterpret_cast<float*>(tiles + grp * kExchangeBytes);   // [gate | up][64 features][kPitch]
            const int fl = (q & 1) * 32 + lane;                       // feature of this lane within the tile
            const int f = n_tile * 64 + fl;
            const bool is_gate = q < 2;
            const uint32_t tm_lane = tmem_acc + (static_cast<uint32_t>(q * 32) << 16);
            float* give = xch + (is_gate ? 0 : 64 * kPitch) + fl * kPitch;
            const float* take = xch + (is_gate ? 64 * kPitch : 0) + fl * kPitch;
            if (ok) {
#pragma unroll 1
                for (int c = 0; c < kHalfRows; c += 16) {
                    uint32_t v[16];
                    tmem_ld16(tm_lane + static_cast<uint32_t>(g0 + (is_gate ? kHalfRows : 0) + c), v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 16; ++j) give[c + j] = __uint_as_float(v[j]);
                }
            }
            group_sync();                                             // every epilogue warp, whether or not its wait succeeded
            if (ok) {
                const int r0 = g0 + (is_gate ? 0 : kHalfRows);
#pragma unroll 1
                for (int c = 0; c < kHalfRows; c += 16) {
                    uint32_t v[16];
                    __syncwarp();
                    tmem_ld16(tm_lane + static_cast<uint32_t>(r0 + c), v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    float gate[16], up[16], x[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float sc = rs.ssq ? sh->scale[r0 + c + j] : 1.0f;
                        const float own = __uint_as_float(v[j]) * sc, other = take[c + j] * sc;
                        gate[j] = is_gate ? own : other;
                        up[j] = is_gate ? other : own;
                    }
                    silu_product(gate, up, x);
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const int m = m0 + r0 + c + j;
                        if (m < M && f < N) act_out[static_cast<size_t>(m) * N + f] = __float2bfloat16_rn(x[j]);
                    }
                }
            }
        }
    }
    pdl_wait();   // every thread: keeps completion of the launch chain transitive
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_acc), "r"(kTmemCols) : "memory");
    }
}

__global__ void reduce_partials_kernel(const float* __restrict__ partial, int splits, size_t stride,
                                       float* __restrict__ out, size_t n) {
    const size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float acc = partial[i];
    for (int s = 1; s < splits; ++s) acc += partial[s * stride + i];
    out[i] = acc;
}

// ---- tensor maps -----------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// bf16 [rows][K] row-major, box = 64 K-elements x box_rows rows, 128-byte swizzle, zero fill.
cudaError_t make_tmap_2d(CUtensorMap* out, const void* base, int rows, int K, int box_rows) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return cudaErrorNotSupported;
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(rows)};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(K) * 2};
    cuuint32_t box[2] = {static_cast<cuuint32_t>(kBK), static_cast<cuuint32_t>(box_rows)};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Packed weight [n_tiles * k_blocks][128][64] bf16: one tile = 16 KB contiguous, rows of 128 bytes; box = box_rows rows of a tile.
cudaError_t make_tmap_packed(CUtensorMap* out, const void* base, int N, int K, int box_rows) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t ntiles = static_cast<cuuint64_t>((N + kBM - 1) / kBM) * ((K + kBK - 1) / kBK);
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(kBK), static_cast<cuuint64_t>(kBM), ntiles};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(kBK) * 2, static_cast<cuuint64_t>(kBK) * kBM * 2};
    cuuint32_t box[3] = {static_cast<cuuint32_t>(kBK), static_cast<cuuint32_t>(box_rows), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// dst[((tn * KB + kb) * 128 + r) * 64 + c] = src[(tn * 128 + r) * K + kb * 64 + c], zero beyond N or K
__global__ void pack_weight_kernel(const __nv_bfloat16* __restrict__ src, __nv_bfloat16* __restrict__ dst, int N, int K,
                                   int KB) {
    const size_t chunk = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;   // 8 elements (16 bytes) each
    const size_t total = static_cast<size_t>((N + kBM - 1) / kBM) * KB * kBM * (kBK / 8);
    if (chunk >= total) return;
    const int c8 = static_cast<int>(chunk % (kBK / 8));
    const int r = static_cast<int>((chunk / (kBK / 8)) % kBM);
    const size_t tile = chunk / (kBK / 8) / kBM;
    const int kb = static_cast<int>(tile % KB);
    const int tn = static_cast<int>(tile / KB);
    const int n = tn * kBM + r, k = kb * kBK + c8 * 8;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (n < N && k < K) v = *reinterpret_cast<const uint4*>(src + static_cast<size_t>(n) * K + k);   // K % 8 == 0
    reinterpret_cast<uint4*>(dst)[chunk] = v;
}

// Gate/up variant: src is [2F][K] = gate rows then up rows; packed tile t holds gate rows
// [64t, 64t+64) in its rows 0..63 and up rows [64t, 64t+64) in its rows 64..127.
__global__ void pack_gate_up_kernel(const __nv_bfloat16* __restrict__ src, __nv_bfloat16* __restrict__ dst, int F, int K,
                                    int KB) {
    const size_t chunk = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const size_t total = static_cast<size_t>((F + 63) / 64) * KB * kBM * (kBK / 8);
    if (chunk >= total) return;
    const int c8 = static_cast<int>(chunk % (kBK / 8));
    const int r = static_cast<int>((chunk / (kBK / 8)) % kBM);
    const size_t tile = chunk / (kBK / 8) / kBM;
    const int kb = static_cast<int>(tile % KB);
    const int t = static_cast<int>(tile / KB);
    const int f = t * 64 + (r & 63), k = kb * kBK + c8 * 8;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (f < F && k < K) v = *reinterpret_cast<const uint4*>(src + (static_cast<size_t>(r < 64 ? 0 : F) + f) * K + k);
    reinterpret_cast<uint4*>(dst)[chunk] = v;
}

// ODB_GEMM_PAIR=0 in the environment: no CTA pairs, many rows run as single CTAs.
bool pair_enabled() {
    static int v = -1;
    if (v < 0) {
        const char* e = getenv("ODB_GEMM_PAIR");
        v = e ? atoi(e) : 1;
    }
    return v != 0;
}

// activation rows per tile of a single CTA; two CTAs share an SM (one's epilogue overlaps the other's main loop)
int pick_bn(int M) {
    static int max_bn = -1;
    if (max_bn < 0) {
        const char* e = getenv("ODB_GEMM_MAX_BN");
        max_bn = e ? atoi(e) : 0;
    }
    const int bn = M <= 32 ? 32 : M <= 64 ? 64 : 128;
    return max_bn > 0 && bn > max_bn ? (max_bn < 64 ? 32 : 64) : bn;
}

template <int BN, int EPI>
cudaError_t launch_bn(const GemmArgs& a, cudaStream_t st) {
    // The rows that there are, in steps of the MMA's sixteen: at 128 an SM takes in as many bytes of activation rows, again and
    // again from L2, as of weights, and gate/up, 44 SMs of which have two tiles, is as long as that takes.  Layer steps, us, a full tile /
    // the rows: d 4096, 96 rows 134.6 / 132.2, 87 rows 137.6 / 136.3; d 2048, two layers, 96 rows 152 / 147, 112 rows 155 / 150;
    // d 1024 96 rows 114.6 / 111.1.  A fourth activation stage in the room of the third of 96 or less rows changes nothing.
    const int x_rows = a.M < BN ? (a.M + 15) / 16 * 16 : BN;
    CUtensorMap tmx;
    cudaError_t e = make_tmap_2d(&tmx, a.x, a.M, a.K, x_rows);
    if (e != cudaSuccess) return e;
    const int nkb_total = (a.K + kBK - 1) / kBK;
    const int nkb_per_split = (nkb_total + a.splits - 1) / a.splits;
    // Two CTAs per SM, up to 112 KB of stages each.  Weight x activation stages at 128 rows, us per layer step of 87 rows: 3 x 3
    // (whole stages) 158.6, 4 x 3 155.5, 4 x 2 162; at 32 rows 4 x 2 131, 5 x 2 127, 5 x 4 121.5, 6 x 4 122.8; at 64 rows 5 x 4
    // 127.9, 4 x 4 126.2, 5 x 3 127.4, 4 x 3 126.5 (d 2048, two layers: 136.3, 136.1, 133.2, 132.6), but a request through
    // the LM head with 47 rows 310.7, 315.3, 315.7, 317.4.  With whole tiles of 64 and 128 rows the two CTAs leave less
    // than a kilobyte of the SM's shared memory, with fewer rows up to 40 KB: either way no successor's CTA that needs the rings is
    // resident there, prefetching its weights, before one of them ends.
    constexpr int kWStages = BN == 128 ? 4 : 5, kXStages = BN == 128 ? 3 : 4;
    constexpr int kWBytes = kBM * kBK * 2, kXBytes = BN * kBK * 2;   // kXBytes: a full tile's
    static_assert(kWStages * kWBytes + kXStages * kXBytes + sizeof(GemmShared) <= 113 * 1024, "two CTAs share an SM");
    const int least = nkb_per_split < kMinStages ? kMinStages : nkb_per_split;
    const int w_stages = kWStages < least ? kWStages : least, x_stages = kXStages < least ? kXStages : least;
    const size_t smem = static_cast<size_t>(w_stages) * kWBytes + static_cast<size_t>(x_stages) * x_rows * (kBK * 2) + sizeof(GemmShared);
    static std::atomic<unsigned long long> attr_done{0};
    e = set_smem_limit_once(attr_done, gemm_kernel<BN, EPI>, 227 * 1024);
    if (e != cudaSuccess) return e;
    // EPI_SWIGLU: N is the FFN width and a weight tile holds 64 gate + 64 up rows
    dim3 grid(EPI == EPI_SWIGLU ? (a.N + 63) / 64 : (a.N + kBM - 1) / kBM, (a.M + BN - 1) / BN, a.splits);
    static int l2_prefetch = -1;
    if (l2_prefetch < 0) {
        const char* env = getenv("ODB_GEMM_L2_PREFETCH");
        l2_prefetch = env ? atoi(env) : 0;   // measured: prefetching into L2 slows the step down
    }
    return launch_kernel(gemm_kernel<BN, EPI>, grid, dim3(gemm_threads(BN, EPI)), smem, st, a.w.tile, tmx, a.partial, a.act_out, a.row_scale, a.conf,
                         a.M, a.N, nkb_total, nkb_per_split, x_rows, w_stages, x_stages, pdl_enabled() ? l2_prefetch : 0, a.status, a.peers, a.norm);
}

template <int EPI>
cudaError_t launch_epi(const GemmArgs& a, cudaStream_t st) {
    switch (pick_bn(a.M)) {
        case 32: return launch_bn<32, EPI>(a, st);
        case 64: return launch_bn<64, EPI>(a, st);
        default: return launch_bn<128, EPI>(a, st);
    }
}

// Whether a projection of M activation rows with n_tiles weight tiles runs as CTA pairs (gemm_rows.cu).  Measured on
// the 8B shape: with many rows (refresh, 768..1024 rows: tensor/L2 bound) pairs with 256-row tiles are 11 %
// faster than single CTAs with 128-row tiles; up to 128 rows (decode steps: HBM bound) the pair's extra
// synchronisation costs more than the halved activation traffic saves (3.55 vs 3.41 ms at 32 rows).
bool use_pair(int M, int n_tiles) { return pair_enabled() && M > 128 && (n_tiles & 1) == 0; }

}  // namespace

int gemm_tiled_rows(int M, int N, int plan_rows) {
    const int bn = use_pair(plan_rows, (N + kBM - 1) / kBM) ? 2 * kBM : pick_bn(M);
    return (M + bn - 1) / bn * bn;
}

bool gemm_rows_usable(int M, int N) { return use_pair(M, (N + kBM - 1) / kBM); }

cudaError_t make_weight_maps(WeightMaps* out, const void* w, int N, int K) {
    const cudaError_t e = make_tmap_packed(&out->tile, w, N, K, kBM);
    return e == cudaSuccess ? make_tmap_packed(&out->half, w, N, K, kBM / 2) : e;
}

cudaError_t make_rows_tmap(CUtensorMap* out, const void* base, int rows, int cols, int box_rows) {
    return make_tmap_2d(out, base, rows, cols, box_rows);
}

size_t packed_weight_bytes(int N, int K) {
    return static_cast<size_t>((N + kBM - 1) / kBM) * ((K + kBK - 1) / kBK) * kBM * kBK * 2;
}

size_t packed_gate_up_bytes(int F, int K) {
    return static_cast<size_t>((F + 63) / 64) * ((K + kBK - 1) / kBK) * kBM * kBK * 2;
}

cudaError_t make_gate_up_maps(WeightMaps* out, const void* w, int F, int K) {
    return make_weight_maps(out, w, ((F + 63) / 64) * kBM, K);
}

cudaError_t launch_pack_gate_up(const void* src, void* dst, int F, int K, cudaStream_t st) {
    const int KB = (K + kBK - 1) / kBK;
    const size_t chunks = packed_gate_up_bytes(F, K) / 16;
    pack_gate_up_kernel<<<static_cast<unsigned>((chunks + 255) / 256), 256, 0, st>>>(
        static_cast<const __nv_bfloat16*>(src), static_cast<__nv_bfloat16*>(dst), F, K, KB);
    return cudaGetLastError();
}

cudaError_t launch_pack_weight(const void* src, void* dst, int N, int K, cudaStream_t st) {
    const int KB = (K + kBK - 1) / kBK;
    const size_t chunks = packed_weight_bytes(N, K) / 16;
    pack_weight_kernel<<<static_cast<unsigned>((chunks + 255) / 256), 256, 0, st>>>(
        static_cast<const __nv_bfloat16*>(src), static_cast<__nv_bfloat16*>(dst), N, K, KB);
    return cudaGetLastError();
}

bool pdl_enabled() {
    static int v = -1;
    if (v < 0) {
        const char* e = getenv("ODB_PDL");
        v = (e && e[0] == '0') ? 0 : 1;
    }
    return v != 0;
}

static int target_ctas() {
    static int v = 0;
    if (!v) {
        const char* e = getenv("ODB_GEMM_TARGET_CTAS");
        v = e ? atoi(e) : 2 * 148;
        if (v < 1) v = 2 * 148;
    }
    return v;
}

int gemm_whole_splits(int splits, int nkb) {
    if (splits < 1) splits = 1;
    while (splits > 1 && ((nkb + splits - 1) / splits) * (splits - 1) >= nkb) --splits;
    return splits;
}

int gemm_pick_splits(int M, int N, int K) {
    const int n_tiles = (N + kBM - 1) / kBM;
    const int bn = use_pair(M, n_tiles) ? 2 * kBM : pick_bn(M);
    const int tiles = n_tiles * ((M + bn - 1) / bn);
    const int nkb = (K + kBK - 1) / kBK;
    if (M > 128) {
        // many rows (refresh): compute bound, and every K split costs M x N fp32 partials written and
        // read back, so split only when the tiles alone cannot occupy the SMs: 296 tiles are one wave of single CTAs (two per
        // SM), and two waves of CTA pairs (74, two weight tiles each)
        static int big_target = 0;
        if (!big_target) {
            const char* e = getenv("ODB_GEMM_BIG_TARGET_CTAS");
            big_target = e ? atoi(e) : 296;
        }
        int sp = tiles >= big_target ? 1 : big_target / tiles;
        // at least 12 k-blocks (5 us of main loop) per split: below that its epilogue and the partials' way through memory
        // cost more than the idle pairs once there are many rows.  Refresh of two layers, us with 8 / with 12: d 1024 at 160 rows
        // 159 / 166, 350 rows 183 / 189, 1118 rows 262 / 242, 1224 rows 249 / 224; d 2048 at 160 rows 203 / 190, 350 rows
        // 262 / 271, 1118 rows 376 / 375.  A choice between the two by waves and partials was never more than 1 % from the better,
        // but any other split of a sum flips greedy tokens that tie (1.2 % of them at d 2048, 1020 rows).
        if (sp > nkb / 12) sp = nkb / 12;
        if (sp > kMaxKSplits) sp = kMaxKSplits;
        return gemm_whole_splits(sp, nkb);
    }
    // all work units must be resident at once (two CTA slots per SM) and equal in size: a
    // second, partly filled wave would double the kernel's time
    int splits = target_ctas() / tiles;
    if (splits > nkb / 4) splits = nkb / 4;
    if (splits > kMaxKSplits) splits = kMaxKSplits;
    return gemm_whole_splits(splits, nkb);
}

cudaError_t launch_gemm(const GemmArgs& a, cudaStream_t st) {
    const bool swiglu = a.act_out != nullptr;
    const int n_tiles = swiglu ? (a.N + 63) / 64 : (a.N + kBM - 1) / kBM;
    if ((swiglu || a.conf.part || a.qkv || a.add_to || a.norm.h) && a.splits != 1) return cudaErrorInvalidValue;
    if (a.norm.h && (a.M > 32 || a.N > kNormOutCols || swiglu || a.conf.part || a.row_scale.ssq || a.peers.n)) return cudaErrorInvalidValue;
    if (use_pair(a.plan_rows > a.M ? a.plan_rows : a.M, n_tiles)) return launch_gemm_rows(a, n_tiles, st);
    if (a.qkv || a.add_to) return cudaErrorInvalidValue;   // epilogues of the many-row kernel only
    if (swiglu) return launch_epi<EPI_SWIGLU>(a, st);
    return a.conf.part ? launch_epi<EPI_CONF>(a, st) : launch_epi<EPI_PARTIAL>(a, st);
}

cudaError_t launch_reduce_partials(const float* partial, int splits, size_t stride, float* out, size_t n,
                                   cudaStream_t st) {
    reduce_partials_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(partial, splits, stride, out, n);
    return cudaGetLastError();
}

}  // namespace odb
