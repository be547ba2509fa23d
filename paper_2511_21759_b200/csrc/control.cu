// Control kernels: the unmask/accept kernel (threshold accept rule, accept-jump walk over the block copies, adaptive
// length prediction, choice of the next speculative candidates).  A few hundred scalars per sequence: one small
// block per sequence, the sequential parts on thread 0.  (The row tables: first_norm.cu.)
#include "odb_internal.cuh"

namespace odb {

namespace {

typedef unsigned long long Mask;   // bit i: position i of the block (blocks have at most 64 positions)

// Accept rule (Section 3, Observation 3): every masked position whose confidence exceeds tau
// (strict); if none, the single most confident one (lowest position on a tie).
__device__ Mask accept_set(const float* conf, Mask masked, float tau) {
    Mask acc = 0;
    int best = -1;
    float best_conf = 0.f;
    for (Mask left = masked; left; left &= left - 1) {
        const int i = __ffsll(left) - 1;
        const float ci = conf[i];
        if (ci > tau) acc |= 1ull << i;
        if (best < 0 || ci > best_conf) { best = i; best_conf = ci; }
    }
    if (acc == 0 && best >= 0) acc = 1ull << best;
    return acc;
}

// Stochastic reverse step (Section 2.1, Eq. 1) at iteration k of the n_steps a block is decoded in: a masked
// position stays masked with probability s / t = (n_steps - k - 1) / (n_steps - k), decided by its uniform
// deviate u (unmask iff u >= s / t, in fp32); the last iteration unmasks everything left.
__device__ Mask sample_set(const float* u, Mask masked, int k, int n_steps) {
    if (k >= n_steps - 1) return masked;
    const float stay = static_cast<float>(n_steps - k - 1) / static_cast<float>(n_steps - k);
    Mask acc = 0;
    for (Mask left = masked; left; left &= left - 1) {
        const int i = __ffsll(left) - 1;
        if (u[i] >= stay) acc |= 1ull << i;
    }
    return acc;
}

// rank set i of the copies of a step, one byte each: {}, {1}, {2}, {1,2}, {3}, {1,2,3}, {4}, {1,2,3,4}
__device__ __forceinline__ int copy_set(int i) { return static_cast<int>(0x0f08070403020100ull >> (8 * i)) & 0xff; }

// Block of 64 threads.  st / res: the block's shared-memory copies of the sequence's state and result (the decisions are one
// thread's serial walk: every field it touches would otherwise be a dependent global load).  wait_forward() returns when the
// forward's confidences and tokens are there; what stands in front of it needs the states and tokens alone.
template <class Wait>
__device__ void accept_body(const ControlBuffers& c, const odb_decode_params& p, int after_refresh, int mask_id, int eos_id,
                            int dry, SeqState* st, odb_result* res, Wait wait_forward) {
    const int seq = blockIdx.x;
    if (!st->active || !st->in_fwd) {
        if (threadIdx.x == 0) {
            res->masks_left = st->active ? st->n_masked : 0;
            res->n_accepted = 0;
            res->chain_len = 0;
            res->gen_len = st->T - st->P;
            res->block_start = st->s;
            res->block_end = st->e;
        }
        return;
    }
    __shared__ float conf[ODB_MAX_COPIES][kMaxBlock];
    __shared__ int tok[ODB_MAX_COPIES][kMaxBlock];
    __shared__ unsigned masked_w[2];       // bit i: position i of the block is masked
    __shared__ int first_eos;
    int32_t* x = c.x + static_cast<size_t>(seq) * c.max_seq;
    const int s = st->s;
    const int n_copies = after_refresh || dry ? 1 : st->n_copies;
    {   // up to the block's end before a length prediction, which can only move it forward
        const int i = threadIdx.x;
        const bool masked = s + i < (after_refresh ? min(s + p.block_len, st->T) : st->e) && __ldcg(x + s + i) == mask_id;
        const unsigned w = __ballot_sync(0xffffffffu, masked);
        if ((i & 31) == 0) masked_w[i >> 5] = w;
    }
    if (!dry) wait_forward();
    // The whole block gathers what the decisions need - the [EOS] scan of a refresh, the copies' confidences and tokens,
    // the block's tokens; the decisions below are taken by thread 0 alone, in the order the method states them.  (One
    // thread scanning and gathering a 256-token response: 42 us; the block: 12 us.)
    if (after_refresh) {
        // adaptive length prediction (Section 4.1): first [EOS] of the whole predicted response
        // whose confidence exceeds the truncate threshold cuts the response there (slot kept)
        const bool alp = p.alp && !dry;
        if (threadIdx.x == 0) first_eos = 0x7fffffff;
        __syncthreads();
        if (alp)
            for (int q = s + threadIdx.x; q < st->T; q += blockDim.x) {
                const int r = st->lm_row0 + (q - st->lm_s);
                if (c.tok[r] == eos_id && c.conf[r] > p.truncate_threshold) { atomicMin(&first_eos, q); break; }
            }
        __syncthreads();
        if (threadIdx.x == 0) {
            if (first_eos != 0x7fffffff) st->T = first_eos + 1;
            st->e = min(s + p.block_len, st->T);
        }
        __syncthreads();
    }
    // A row whose logits are all NaN has no greedy token (0x7fffffff, with confidence 1 / 0), and one of a forward whose waits ran out
    // whatever was there: committed or filled in, they would be rows far behind the embedding.  They count as [EOS] with confidence 0 (as another
    // id where that is [MASK], which committed would stay masked).
    const int none = eos_id != mask_id ? eos_id : mask_id == 0 ? 1 : 0;
    auto gather = [&](int cp, int i, int r) {
        const int t = c.tok[r];
        const bool known = t >= 0 && t < c.vocab;
        conf[cp][i] = known ? c.conf[r] : 0.f;
        tok[cp][i] = known ? t : none;
    };
    if (!dry && after_refresh) {
        for (int i = threadIdx.x; i < st->e - s; i += blockDim.x) gather(0, i, st->lm_row0 + (s + i - st->lm_s));
    } else if (!dry) {
        for (int i = threadIdx.x; i < n_copies * kMaxBlock; i += blockDim.x) {
            conf[i / kMaxBlock][i % kMaxBlock] = -1.f;
            tok[i / kMaxBlock][i % kMaxBlock] = -1;
        }
        __syncthreads();
        for (int cp = 0; cp < n_copies; ++cp) {
            const int r0 = st->copy_row0[cp], r1 = r0 + st->copy_nrows[cp];
            for (int r = r0 + threadIdx.x; r < r1; r += blockDim.x) gather(cp, c.row_pos[r] - s, r);
        }
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const int B = st->e - s;
    const Mask masked0 = (static_cast<Mask>(masked_w[1]) << 32 | masked_w[0]) & (B >= 64 ? ~0ull : (1ull << B) - 1ull);

    if (dry) {
        // model without LM head (layer microbenchmark): there is nothing to decide on, so commit
        // nothing and lay out the next step as if no position had been accepted; the speculative
        // fills are the first masked positions with token id 0
        int n_ranks = 0;
        const int k_ranks = p.n_copies >= 8 ? 4 : p.n_copies >= 4 ? 2 : 0;
        for (Mask left = masked0; left && n_ranks < k_ranks; left &= left - 1) {
            st->rank_off[n_ranks] = __ffsll(left) - 1;
            st->rank_tok[n_ranks] = 0;
            ++n_ranks;
        }
        const int n_masked = __popcll(masked0);
        st->n_ranks = n_ranks;
        st->n_masked = n_masked;
        const int thr = p.stage2_min_decoded >= 0 ? p.stage2_min_decoded : (4 * B + 6) / 7;
        const int stage2 = (p.n_copies >= 8 && (B - n_masked) >= thr) ? 1 : 0;
        const int want = p.n_copies >= 8 ? (stage2 ? 8 : 4) : p.n_copies >= 4 ? 4 : 1;
        int nc = 0;
        for (int i = 0; i < want; ++i)
            if ((copy_set(i) >> n_ranks) == 0) st->copy_mask[nc++] = copy_set(i);
        st->n_copies = nc;
        st->stage2 = stage2;
        res->masks_left = n_masked;
        res->n_accepted = 0;
        res->chain_len = 1;
        res->chain[0] = 0;
        res->gen_len = st->T - st->P;
        res->block_start = s;
        res->block_end = st->e;
        return;
    }
    if (after_refresh) st->block_iter = 0;
    const int k_iter = st->block_iter < kMaxLoopIters ? st->block_iter : kMaxLoopIters - 1;
    const float* noise = c.noise + (static_cast<size_t>(seq) * kMaxLoopIters + k_iter) * kMaxBlock;
    ++st->block_iter;
    Mask taken = 0;

    // accept-jump walk (Section 4.2.1): start in the main block; a candidate is hit if its
    // position was accepted with the token it had been filled with; jump to the largest copy
    // whose extra candidates are all hit; the accepted sets along the chain are committed,
    // an earlier link winning at a shared position
    int cur = 0, chain_len = 0, n_acc = 0;
    const bool pick = p.pick_best && !after_refresh;
    auto commit = [&](int i, int t) {
        taken |= 1ull << i;
        x[s + i] = t;
        if (n_acc < 64) { res->accepted_pos[n_acc] = s + i; res->accepted_tok[n_acc] = t; }
        ++n_acc;
    };
    auto commit_all = [&](Mask m) {   // the block's positions in m that no earlier link has taken
        for (Mask left = m & ~taken; left; left &= left - 1) {
            const int i = __ffsll(left) - 1;
            commit(i, tok[cur][i]);
        }
    };
    if (pick) {
        // the compared speculation (Fig. 7(a), Section 5.3): candidates verified in the main block only; the copy
        // filling the largest set of hits is adopted, and its fills and own accept set are the whole result
        Mask acc = accept_set(conf[0], masked0, p.accept_threshold);
        int hit = 0;
        for (int r = 0; r < st->n_ranks; ++r) {
            const int o = st->rank_off[r];
            if (((acc >> o) & 1) && tok[0][o] == st->rank_tok[r]) hit |= 1 << r;
        }
        for (int cp = 1; cp < n_copies; ++cp) {
            const int Y = st->copy_mask[cp];
            if (Y & ~hit) continue;
            if (cur == 0 || __popc(Y) > __popc(st->copy_mask[cur]) ||
                (__popc(Y) == __popc(st->copy_mask[cur]) && Y < st->copy_mask[cur]))
                cur = cp;
        }
        if (cur != 0) {
            const int Y = st->copy_mask[cur];
            Mask masked = masked0;
            for (int r = 0; r < st->n_ranks; ++r)
                if ((Y >> r) & 1) { masked &= ~(1ull << st->rank_off[r]); commit(st->rank_off[r], st->rank_tok[r]); }
            acc = masked ? accept_set(conf[cur], masked, p.accept_threshold) : 0;
        }
        commit_all(acc);
        res->chain[0] = cur;
        chain_len = 1;
    }
    while (!pick) {
        res->chain[chain_len < ODB_MAX_CHAIN ? chain_len : ODB_MAX_CHAIN - 1] = cur;
        ++chain_len;
        const int X = after_refresh ? 0 : st->copy_mask[cur];
        Mask masked = masked0;
        for (int r = 0; r < st->n_ranks; ++r)
            if ((X >> r) & 1) masked &= ~(1ull << st->rank_off[r]);
        if (!masked) break;
        const Mask acc = p.sampling ? sample_set(noise, masked, k_iter, p.sample_steps) : accept_set(conf[cur], masked, p.accept_threshold);
        commit_all(acc);
        if (after_refresh) break;
        int hit = 0;
        for (int r = 0; r < st->n_ranks; ++r) {
            const int o = st->rank_off[r];
            if (!((X >> r) & 1) && ((acc >> o) & 1) && tok[cur][o] == st->rank_tok[r]) hit |= 1 << r;
        }
        int best = -1;
        for (int cp = 0; cp < n_copies; ++cp) {
            const int Y = st->copy_mask[cp];
            if ((Y & X) != X || Y == X || ((Y & ~X) & ~hit)) continue;
            if (best < 0 || __popc(Y) > __popc(st->copy_mask[best]) ||
                (__popc(Y) == __popc(st->copy_mask[best]) && Y < st->copy_mask[best]))
                best = cp;
        }
        if (best < 0) break;
        cur = best;
    }

    // state after the walk; next candidates: the most confident still-masked positions of the
    // adopted copy (Section 4.2), ties to the lower position
    Mask open = masked0 & ~taken;
    const int n_masked = __popcll(open);
    const int k_ranks = p.n_copies >= 8 ? 4 : p.n_copies >= 4 ? 2 : 0;
    int n_ranks = 0;
    for (int r = 0; r < k_ranks; ++r) {
        int best = -1;
        for (Mask left = open; left; left &= left - 1) {
            const int i = __ffsll(left) - 1;
            if (best < 0 || conf[cur][i] > conf[cur][best]) best = i;
        }
        if (best < 0) break;
        open &= ~(1ull << best);
        st->rank_off[n_ranks] = best;
        st->rank_tok[n_ranks] = tok[cur][best];
        ++n_ranks;
    }
    st->n_ranks = n_ranks;
    st->n_masked = n_masked;
    // stage switch (Section 4.2.2 gives no number): decoded-share once eight copies fit the row
    // budget of four full copies, B + 7 (B - n_dec) <= 4 B
    const int thr = p.stage2_min_decoded >= 0 ? p.stage2_min_decoded : (4 * B + 6) / 7;
    const int stage2 = (p.n_copies >= 8 && (B - n_masked) >= thr) ? 1 : 0;
    const int want = p.n_copies >= 8 ? (stage2 ? 8 : 4) : p.n_copies >= 4 ? 4 : 1;
    int nc = 0;
    for (int i = 0; i < want; ++i)
        if ((copy_set(i) >> n_ranks) == 0) st->copy_mask[nc++] = copy_set(i);
    st->n_copies = nc;
    st->stage2 = stage2;

    res->masks_left = n_masked;
    res->n_accepted = n_acc;
    res->chain_len = chain_len;
    res->gen_len = st->T - st->P;
    res->block_start = s;
    res->block_end = st->e;
}

// One block per sequence.  After the decisions, the block writes the sequence's state and result (and block 0
// the status word) straight into pinned host memory.
struct AcceptShared {
    SeqState st;
    odb_result res;
};
// from L2: in front of the wait nothing else orders these reads behind an L1 line of an earlier kernel
__device__ __forceinline__ void accept_load(const ControlBuffers& c, AcceptShared* sh) {
    const int seq = blockIdx.x;
    const int* gs = reinterpret_cast<const int*>(c.state + seq);
    const int* gr = reinterpret_cast<const int*>(c.results + seq);
    for (int i = threadIdx.x; i < static_cast<int>(sizeof(SeqState) / 4); i += blockDim.x) reinterpret_cast<int*>(&sh->st)[i] = __ldcg(gs + i);
    for (int i = threadIdx.x; i < static_cast<int>(sizeof(odb_result) / 4); i += blockDim.x) reinterpret_cast<int*>(&sh->res)[i] = __ldcg(gr + i);
    __syncthreads();
}
// state and result back to the device copies and out to pinned host memory (host_res: where this call's results go)
__device__ __forceinline__ void accept_store(const ControlBuffers& c, const AcceptShared* sh, odb_result* host_res) {
    const int seq = blockIdx.x;
    const int* ss = reinterpret_cast<const int*>(&sh->st);
    const int* sr = reinterpret_cast<const int*>(&sh->res);
    int* gs = reinterpret_cast<int*>(c.state + seq);
    int* hs = reinterpret_cast<int*>(c.host_state + seq);
    for (int i = threadIdx.x; i < static_cast<int>(sizeof(SeqState) / 4); i += blockDim.x) { gs[i] = ss[i]; hs[i] = ss[i]; }
    int* gr = reinterpret_cast<int*>(c.results + seq);
    int* hr = reinterpret_cast<int*>(host_res);
    for (int i = threadIdx.x; i < static_cast<int>(sizeof(odb_result) / 4); i += blockDim.x) { gr[i] = sr[i]; hr[i] = sr[i]; }
}

// Launched under the last kernel of the forward, and it starts when the forward's first kernel has written the tables and the
// states (first_norm.cu): it reads states and tokens, which nothing behind that kernel writes, before it waits for the forward.
// Without an LM head that is all it decides on.  Behind the wait are stores alone: us in an 8B layer step with one copy / four,
// 3.7 / 5.0 when it waited first and one thread walked over the block's tokens.
__global__ void __launch_bounds__(kMaxBlock) accept_kernel(ControlBuffers c, odb_decode_params p, int after_refresh, int mask_id, int eos_id, int dry) {
    __shared__ AcceptShared sh;
    accept_load(c, &sh);
    accept_body(c, p, after_refresh, mask_id, eos_id, dry, &sh.st, &sh.res, []() { pdl_wait(); });
    pdl_wait();
    __syncthreads();
    accept_store(c, &sh, c.host_results + blockIdx.x);
    if (blockIdx.x == 0 && threadIdx.x == 0) *c.host_status = *c.status;
    // no fence: the host reads after synchronising the stream, and the kernel's end makes its stores visible
}

// The accept of the device-resident loop: the same decisions, then the hand-over to the next iteration.
__global__ void __launch_bounds__(kMaxBlock) accept_loop_kernel(ControlBuffers c, odb_decode_params p, int mask_id, int eos_id, int dry, LoopControl lc) {
    __shared__ AcceptShared sh;
    accept_load(c, &sh);
    accept_body(c, p, 0, mask_id, eos_id, dry, &sh.st, &sh.res, []() { pdl_wait(); });
    pdl_wait();
    __syncthreads();
    const int seq = blockIdx.x, batch = gridDim.x;
    const int it = *lc.iter;      // stable until every block has arrived below
    accept_store(c, &sh, lc.host_log + static_cast<size_t>(it) * batch + seq);
    __threadfence();              // the state, for the last block; the host log is read after the stream has been synchronised
    __syncthreads();
    if (threadIdx.x != 0) return;
    // fail-safe: the loop ends unless the last block below asks for another pass (block 0 writes this before it
    // arrives, the last block writes after every arrival, so the last block's word stands)
    if (seq == 0) {
        cudaGraphSetConditional(lc.handle, 0u);
        __threadfence();
    }
    if (atomicAdd(lc.arrivals, 1) != batch - 1) return;
    // last block of the iteration: every sequence's state is final
    __threadfence();
    StepShape next{0, 0, 0, 0};
    for (int i = 0; i < batch; ++i) {
        const volatile SeqState* vs = c.state + i;
        SeqState st{};
        st.active = vs->active; st.n_masked = vs->n_masked; st.s = vs->s; st.e = vs->e;
        st.n_copies = vs->n_copies; st.stage2 = vs->stage2;
        step_shape_add(next, st);
    }
    const int err = *reinterpret_cast<const volatile int*>(c.status);
    const bool same = next.rows == lc.shape.rows && next.tiles == lc.shape.tiles &&
                      next.step_tiles == lc.shape.step_tiles && next.multi == lc.shape.multi;
    const int limit = min(*lc.max_iters, kMaxLoopIters);
    const bool again = it + 1 < limit && err == 0 && next.rows > 0 && same;
    *lc.arrivals = 0;
    *lc.iter = it + 1;
    *lc.host_iters = it + 1;
    *c.host_status = err;
    cudaGraphSetConditional(lc.handle, again ? 1u : 0u);
}

// A wait that runs out by design: the barrier is initialised for one arrival that never comes.
__global__ void expire_wait_kernel(long long limit_cycles, int* status) {
    __shared__ uint64_t bar;
    __shared__ int abort_word;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(&bar))));
        abort_word = 0;
    }
    __syncthreads();
    mbar_wait_bounded(&bar, 0, &abort_word, status, limit_cycles);
}

}  // namespace

cudaError_t launch_expire_wait(long long limit_cycles, int* status, cudaStream_t st) {
    expire_wait_kernel<<<1, 32, 0, st>>>(limit_cycles, status);
    return cudaGetLastError();
}

cudaError_t launch_accept_loop(const ControlBuffers& c, int batch, const odb_decode_params& p, int mask_id, int eos_id,
                               int dry, const LoopControl& lc, cudaStream_t st) {
    return launch_kernel(accept_loop_kernel, dim3(batch), dim3(kMaxBlock), 0, st, c, p, mask_id, eos_id, dry, lc);
}

cudaError_t launch_accept(const ControlBuffers& c, int batch, const odb_decode_params& p, int after_refresh,
                          int mask_id, int eos_id, int dry, cudaStream_t st) {
    return launch_kernel(accept_kernel, dim3(batch), dim3(kMaxBlock), 0, st, c, p, after_refresh, mask_id, eos_id, dry);
}

}  // namespace odb
