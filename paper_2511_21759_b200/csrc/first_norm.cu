// The first kernel of a forward: the row and tile tables of a refresh or a block step, and its first norm, whose residual
// stream is the embedding of each row's token.
//
// The tables were a kernel of their own, one block per sequence, with the norm behind it.  What bounds both is the chain of
// dependent reads (state, tokens, embedding row), not any amount of work, and what the first projection waits for is the
// launch of three kernels in a row: at 2 to 2.5 us each on the host its weights were first asked for 4.4 us after the step began.
// So blocks 0 .. batch - 1 write the tables, and every other block finds the tokens of its rows from the sequences' states
// itself.
#include "norm_common.cuh"

namespace odb {

namespace {

// ------------------------------------------------------------------------------------------------ tables

// Rows of a refresh: every position of every active sequence, in sequence order.
__device__ void write_refresh_tables(const ControlBuffers& c, int seq, const int32_t* block_index, int block_len) {
    SeqState* st = c.state + seq;
    if (!st->active || block_index[seq] < 0) {
        if (threadIdx.x == 0) st->in_fwd = 0;
        return;
    }
    // what the sequences in front take: one thread per sequence (serially, sixteen sequences were 9 us of dependent loads)
    __shared__ int row0, lm0, tile0, big0;
    if (threadIdx.x == 0) row0 = lm0 = tile0 = big0 = 0;
    __syncthreads();
    if (threadIdx.x < seq) {
        const SeqState* o = c.state + threadIdx.x;
        if (o->active && block_index[threadIdx.x] >= 0) {
            atomicAdd(&row0, o->T);
            atomicAdd(&lm0, o->T - (o->P + block_index[threadIdx.x] * block_len));
            atomicAdd(&tile0, (o->T + 63) / 64);
            atomicAdd(&big0, (o->T + 127) / 128);
        }
    }
    __syncthreads();
    const int T = st->T;
    const int s = st->P + block_index[seq] * block_len;
    if (threadIdx.x == 0) {
        st->in_fwd = 1;
        st->block_idx = block_index[seq];
        st->s = s;
        st->e = min(s + block_len, T);
        st->row0 = row0;
        st->n_rows = T;
        st->lm_row0 = lm0;
        st->lm_s = s;
        st->lm_n = T - s;
        st->n_ranks = 0;
        st->n_copies = 1;
        st->copy_mask[0] = 0;
        st->stage2 = 0;
    }
    const int32_t* x = c.x + static_cast<size_t>(seq) * c.max_seq;
    for (int p = threadIdx.x; p < T; p += blockDim.x) {
        const int row = row0 + p;
        c.row_tok[row] = x[p];
        c.row_pos[row] = p;
        c.row_seq[row] = seq;
        c.row_copy[row] = 0;
        c.row_flags[row] = 0;
        if (p >= s) c.lm_rows[lm0 + (p - s)] = row;
    }
    for (int j = threadIdx.x; j < (T + 63) / 64; j += blockDim.x) {
        QTile q;
        q.q_row0 = row0 + 64 * j;
        q.nq = min(64, T - 64 * j);
        q.seq = seq;
        q.cA = 0; q.cB0 = 0; q.cB1 = 0;
        q.f0 = row0; q.n0 = T;
        q.f1 = 0; q.n1 = 0;
        c.tiles[tile0 + j] = q;
    }
    for (int j = threadIdx.x; j < (T + 127) / 128; j += blockDim.x) {
        QTile q;
        q.q_row0 = row0 + 128 * j;
        q.nq = min(128, T - 128 * j);
        q.seq = seq;
        q.cA = 0; q.cB0 = 0; q.cB1 = 0;
        q.f0 = row0; q.n0 = T;
        q.f1 = 0; q.n1 = 0;
        c.big_tiles[big0 + j] = q;
    }
}

// Rows of a block step (Section 4.2; decoded-share layout: Section 4.2.2, caption of Fig. 8):
// copy 0 holds the whole block; a speculative copy holds the whole block (stage 1) or only the
// positions still masked in the committed state (stage 2).  Position ids are the true positions.
__device__ int step_rows_of(const SeqState* st) {
    const int B = st->e - st->s;
    return st->stage2 ? B + (st->n_copies - 1) * st->n_masked : st->n_copies * B;
}

__device__ int step_tiles_of(const SeqState* st) {
    const int B = st->e - st->s;
    return step_tiles_of_counts(st->n_copies, B, st->stage2 ? st->n_masked : B);
}

// One block of at least 64 threads per sequence.  The state is worked on in shared memory, the sequences in front are counted by
// one thread each and the attention work items filled in by one thread per slab: written as one thread's walk over global
// memory this was 6 us at batch 1 and 22 us at batch 16, and with the items alone walked by one thread 3.9 us with four copies
// and 5.9 with eight (one copy: 1.5).
__device__ void write_step_tables(const ControlBuffers& c, int seq, int mask_id) {
    const int tid = threadIdx.x, n_threads = blockDim.x;
    __shared__ SeqState sst;
    __shared__ int xs[kMaxBlock];      // the block's committed tokens
    __shared__ unsigned masked_w[2];   // bit i: position i of the block is masked
    __shared__ int row_base, tile_base, stile_base;
    {
        const int* gs = reinterpret_cast<const int*>(c.state + seq);
        for (int i = tid; i < static_cast<int>(sizeof(SeqState) / 4); i += n_threads) reinterpret_cast<int*>(&sst)[i] = gs[i];
        if (tid == 0) row_base = tile_base = stile_base = 0;
    }
    __syncthreads();
    SeqState* st = &sst;
    if (!st->active || st->n_masked <= 0) {
        if (tid == 0) c.state[seq].in_fwd = 0;
        return;
    }
    const int32_t* x = c.x + static_cast<size_t>(seq) * c.max_seq;
    const int s = st->s, e = st->e, B = e - s;   // B <= kMaxBlock
    if (tid < kMaxBlock) {
        const int my_tok = tid < B ? x[s + tid] : 0;
        if (tid < seq) {
            const SeqState* o = c.state + tid;
            if (o->active && o->n_masked > 0) {
                atomicAdd(&row_base, step_rows_of(o));
                atomicAdd(&tile_base, o->n_copies);
                atomicAdd(&stile_base, step_tiles_of(o));
            }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, tid < B && my_tok == mask_id);
        if ((tid & 31) == 0) masked_w[tid >> 5] = bal;
        xs[tid] = my_tok;
    }
    __syncthreads();
    const unsigned long long masked = static_cast<unsigned long long>(masked_w[1]) << 32 | masked_w[0];
    const int nm = __popcll(masked), n_copies = st->n_copies, row0 = row_base;
    // copy 0 holds the whole block; a speculative copy the whole block or, in the decoded-share layout, the positions still masked
    const int n_other = st->stage2 ? nm : B;
    auto rows_of = [&](int cp) { return cp == 0 ? B : n_other; };
    auto row0_of = [&](int cp) { return cp == 0 ? row0 : row0 + B + (cp - 1) * n_other; };
    // one thread per (copy, position): the rows of the copies, copy after copy
    for (int it = tid; it < n_copies * B; it += n_threads) {
        const int cp = it / B, i = it % B;
        const bool decoded = !((masked >> i) & 1ull);
        const bool shared = st->stage2 && cp > 0;
        if (shared && decoded) continue;
        const int row = row0_of(cp) + (shared ? __popcll(masked & ((1ull << i) - 1ull)) : i);
        int tok = xs[i];
        for (int r = 0; r < st->n_ranks; ++r)
            if (((st->copy_mask[cp] >> r) & 1) && st->rank_off[r] == i) tok = st->rank_tok[r];
        c.row_tok[row] = tok;
        c.row_pos[row] = s + i;
        c.row_seq[row] = seq;
        c.row_copy[row] = cp;
        c.row_flags[row] = decoded ? kRowDecoded : 0;
        c.lm_rows[row] = row;
    }
    if (tid < n_copies) {
        const int cp = tid;
        QTile q;
        q.q_row0 = row0_of(cp);
        q.nq = rows_of(cp);
        q.seq = seq;
        q.cA = s; q.cB0 = e; q.cB1 = st->T;
        q.f0 = q.q_row0; q.n0 = q.nq;
        const bool shared = st->stage2 && cp > 0;
        q.f1 = shared ? row0 : 0;
        q.n1 = shared ? B : 0;
        c.tiles[tile_base + cp] = q;
    }
    // attention work items that share the cached K/V among copies: copies are packed, in order, into items of at most 8 slabs of
    // 16 rows (the host counts them with the same rule, step_tiles_of).  Thread (copy, slab) of the first two warps; entries of
    // an item beyond its counts are never read.
    if (tid < kMaxBlock && (tid >> 3) < n_copies) {
        const int cp = tid >> 3, k = tid & 7, n = rows_of(cp), slabs = (n + 15) / 16;
        int item = 0, first = 0, have = 0;   // this copy's item, the item's first copy, slabs in the item in front of this copy
        for (int j = 0; j <= cp; ++j) {
            const int need = (rows_of(j) + 15) / 16;
            if (have && have + need > 8) { ++item; first = j; have = 0; }
            if (j < cp) have += need;
        }
        StepTile* t = c.step_tiles + stile_base + item;
        if (k < slabs) {
            t->slab_copy[have + k] = cp;
            t->slab_row0[have + k] = row0_of(cp) + 16 * k;
            t->slab_n[have + k] = min(16, n - 16 * k);
        }
        if (k == 0) {
            t->src_copy[cp - first] = cp;
            t->src_row0[cp - first] = row0_of(cp);
            t->src_n[cp - first] = n;
            if (cp == first) {
                int last = cp, n_slabs = slabs;
                while (last + 1 < n_copies && n_slabs + (rows_of(last + 1) + 15) / 16 <= 8) n_slabs += (rows_of(++last) + 15) / 16;
                int n_src = last - first + 1;
                if (st->stage2 && first > 0) {   // copy 0's decoded rows are visible to every speculative copy
                    t->src_copy[n_src] = 0;
                    t->src_row0[n_src] = row0;
                    t->src_n[n_src] = B;
                    ++n_src;
                }
                t->seq = seq; t->cA = s; t->cB0 = e; t->cB1 = st->T;
                t->n_slabs = n_slabs; t->n_src = n_src; t->stage2 = st->stage2;
            }
        }
    }
    // the placement back to the device state; other blocks read active, s, e, n_masked, n_copies, stage2 and the candidates only,
    // which stay
    SeqState* gst = c.state + seq;
    if (tid == 0) {
        gst->in_fwd = 1;
        gst->row0 = row0; gst->n_rows = B + (n_copies - 1) * n_other; gst->lm_row0 = row0;
    }
    if (tid < n_copies) {
        gst->copy_row0[tid] = row0_of(tid);
        gst->copy_nrows[tid] = rows_of(tid);
    }
}

// ------------------------------------------------------------------------------------------------ tokens of a block's rows

// first row of every sequence, base[batch] = all rows; by the first warp, behind it a block barrier
__device__ void count_rows(const FirstRows& f, int* base) {
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int n[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int t = 2 * lane + u;
            n[u] = 0;
            if (t < f.batch) {
                const SeqState* st = f.cb.state + t;
                if (f.step) {
                    if (st->active && st->n_masked > 0) n[u] = step_rows_of(st);
                } else if (st->active && f.block_index[t] >= 0) {
                    n[u] = st->T;
                }
            }
        }
        int sum = n[0] + n[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += up;
        }
        if (2 * lane <= f.batch) base[2 * lane] = sum - n[0] - n[1];
        if (2 * lane + 1 <= f.batch) base[2 * lane + 1] = sum - n[1];
        if (lane == 31 && f.batch == 64) base[64] = sum;
    }
    __syncthreads();
}

// the token of row `row`: one whole warp, same result in every lane
__device__ int token_of_row(const FirstRows& f, const int* base, int row) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = f.batch;                   // the last sequence with base <= row (those without rows share their successor's)
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (base[mid] <= row) lo = mid; else hi = mid;
    }
    const int r = row - base[lo];
    const SeqState* st = f.cb.state + lo;
    const int32_t* x = f.cb.x + static_cast<size_t>(lo) * f.cb.max_seq;
    if (!f.step) return x[r];
    const int s = st->s, B = st->e - s, stage2 = st->stage2, n_ranks = st->n_ranks;
    int off[ODB_MAX_RANKS], tok[ODB_MAX_RANKS];
#pragma unroll
    for (int k = 0; k < ODB_MAX_RANKS; ++k) { off[k] = st->rank_off[k]; tok[k] = st->rank_tok[k]; }
    const int x0 = lane < B ? x[s + lane] : 0, x1 = lane + 32 < B ? x[s + 32 + lane] : 0;
    int cp = r / B, i = r - cp * B;
    if (stage2 && r >= B) {                     // row j of a speculative copy: the j-th masked position
        const unsigned m0 = __ballot_sync(0xffffffffu, lane < B && x0 == f.mask_id);
        const unsigned m1 = __ballot_sync(0xffffffffu, lane + 32 < B && x1 == f.mask_id);
        const int n0 = __popc(m0), nm = n0 + __popc(m1);
        cp = 1 + (r - B) / nm;
        const int j = (r - B) % nm;
        const unsigned below = (1u << lane) - 1u;
        const unsigned a0 = __ballot_sync(0xffffffffu, ((m0 >> lane) & 1u) && __popc(m0 & below) == j);
        const unsigned a1 = __ballot_sync(0xffffffffu, ((m1 >> lane) & 1u) && n0 + __popc(m1 & below) == j);
        i = a0 ? __ffs(a0) - 1 : 31 + __ffs(a1);
    }
    int t = __shfl_sync(0xffffffffu, i < 32 ? x0 : x1, i & 31);
    const int fills = st->copy_mask[cp];
#pragma unroll
    for (int k = 0; k < ODB_MAX_RANKS; ++k)
        if (k < n_ranks && ((fills >> k) & 1) && off[k] == i) t = tok[k];
    return t;
}

// float4 i of the embedding row of a token
__device__ __forceinline__ float4 embed_load4(const FirstRows& f, int token, int i, int d) {
    const __nv_bfloat16* row = f.table + static_cast<size_t>(token) * d;
    uint2 x;
    if (f.halves) {
        x.x = reinterpret_cast<const uint32_t*>(row)[2 * i];
        x.y = reinterpret_cast<const uint32_t*>(row)[2 * i + 1];
    } else {
        x = reinterpret_cast<const uint2*>(row)[i];
    }
    return make_float4(__uint_as_float(x.x << 16), __uint_as_float(x.x & 0xffff0000u), __uint_as_float(x.y << 16),
                       __uint_as_float(x.y & 0xffff0000u));
}

// Blocks 0 .. batch - 1: the tables of a sequence each.  The others: ROWS rows x a slice of kNormSliceCols columns each, one
// float4 per thread and row: h = the embedding, out = bf16(h * gain), ssq = the slice's sum of squares (the other norms of the
// forward: elementwise.cu; SECOND_FIRST as theirs).
//
// Programmatic dependent launch: the blocks with tables let the successor start when their tables are visible device-wide, the
// others at once, so no later kernel of the chain starts before the tables are complete.  That is what allows the attention
// kernels to read their work items, and a step's K/V cache, before their own griddepcontrol.wait.
template <int ROWS>
__global__ void __launch_bounds__(kNormSliceCols / 4) first_norm_kernel(float* __restrict__ h, const float* __restrict__ gain,
                                                                        __nv_bfloat16* __restrict__ out, float* __restrict__ ssq, int M,
                                                                        int d, const __grid_constant__ FirstRows f, L2Prefetch pf) {
    if (static_cast<int>(blockIdx.x) < f.batch) {
        if (f.step) write_step_tables(f.cb, blockIdx.x, f.mask_id);
        else write_refresh_tables(f.cb, blockIdx.x, f.block_index, f.block_len);
        __threadfence();
        __syncthreads();
        pdl_launch_dependents();
        return;
    }
    pdl_launch_dependents();
    __shared__ float red[ROWS][32];
    __shared__ int base[65], tok[ROWS];
    const int slices = (d + kNormSliceCols - 1) / kNormSliceCols;
    const int b = static_cast<int>(blockIdx.x) - f.batch, slice = b % slices, row0 = b / slices * ROWS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    l2_prefetch_slice(pf, b, gridDim.x - f.batch);
    const int i = slice * (kNormSliceCols / 4) + threadIdx.x;   // float4 index within the row
    const bool in = i < (d >> 2);
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
    if (in) g = reinterpret_cast<const float4*>(gain)[i];
    count_rows(f, base);
    if (warp < ROWS && row0 + warp < M) {
        const int t = token_of_row(f, base, row0 + warp);
        if (lane == 0) tok[warp] = t;
    }
    __syncthreads();
    float4 v[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
        if (in && row0 + r < M) v[r] = embed_load4(f, tok[r], i, d);
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        float ss = 0.f;
        if (in && row0 + r < M) {
            const size_t row = static_cast<size_t>(row0 + r) * d;
            reinterpret_cast<float4*>(h + row)[i] = v[r];
            ss = squares4<ROWS == 1>(v[r]);
            reinterpret_cast<uint2*>(out + row)[i] = pack4_bf16(v[r].x * g.x, v[r].y * g.y, v[r].z * g.z, v[r].w * g.w);
        }
        ss = warp_sum(ss);
        if (lane == 0) red[r][warp] = ss;
    }
    __syncthreads();
    if (threadIdx.x < ROWS && row0 + threadIdx.x < M) {
        float total = 0.f;
        for (int w = 0; w < nw; ++w) total += red[threadIdx.x][w];
        ssq[static_cast<size_t>(row0 + threadIdx.x) * slices + slice] = total;
    }
}

__global__ void __launch_bounds__(64) build_step_rows_kernel(ControlBuffers c, int mask_id) { write_step_tables(c, blockIdx.x, mask_id); }

template <int ROWS>
cudaError_t launch_rows(float* h, const float* gain, __nv_bfloat16* out, float* ssq, int M, int d, const FirstRows& f, L2Prefetch pf,
                        cudaStream_t st) {
    const unsigned blocks = static_cast<unsigned>((M + ROWS - 1) / ROWS) * ((d + kNormSliceCols - 1) / kNormSliceCols);
    first_norm_kernel<ROWS><<<f.batch + blocks, kNormSliceCols / 4, 0, st>>>(h, gain, out, ssq, M, d, f, pf);
    return cudaGetLastError();
}

}  // namespace

// Launched without programmatic stream serialization: it starts when everything enqueued before it (the previous accept) has
// completed.  Four rows per block from 256 rows up, as the other norms.
cudaError_t launch_first_norm(float* h, const float* gain, __nv_bfloat16* out, float* ssq, int M, int d, const FirstRows& f, L2Prefetch pf,
                              cudaStream_t st) {
    return M >= 256 ? launch_rows<4>(h, gain, out, ssq, M, d, f, L2Prefetch{nullptr, 0}, st) : launch_rows<1>(h, gain, out, ssq, M, d, f, pf, st);
}

cudaError_t launch_build_step_rows(const ControlBuffers& c, int batch, int mask_id, cudaStream_t st) {
    build_step_rows_kernel<<<batch, 64, 0, st>>>(c, mask_id);
    return cudaGetLastError();
}

}  // namespace odb
