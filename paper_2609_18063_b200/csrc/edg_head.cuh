// Publication of head logits and of the routing made of them (a1, a2), shared by the two forms of the batch-1 layer-step.
#pragma once

#include "edg_ptx.cuh"

namespace edg {

constexpr int kTraceMarks = 32;

template <typename P>
__device__ __forceinline__ void trace_stamp(const P& p, int m) {
    if (p.trace != nullptr) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        p.trace[(size_t)blockIdx.x * kTraceMarks + m] = t;
    }
}

static __device__ __noinline__ void topk_any(float* work, int E, int K, int lane, int32_t* inds, float* gates) {
    warp_softmax_topk(work, E, K, lane, inds, gates);
}

// The usual case of warp_softmax_topk_reg, E <= 256: a logit for every choice and no two of the chosen equal.  False: it is
// not this case, nothing useful has been written.  A round takes the largest key of the warp and strikes it from the lane that
// held it -- no sorted lists, nothing to shuffle in between.
__device__ __forceinline__ bool topk_distinct(const float* work, int E, int K, int lane, int32_t* inds, float* gates) {
    const unsigned full = 0xFFFFFFFFu;
    uint32_t key[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int e = u * 32 + lane;
        const float v = e < E ? work[e] : __int_as_float(0x7fffffff);
        key[u] = (v == v) ? float_key(v) : 0u;
    }
    float myv = 0.f;
    bool fine = true;
#pragma unroll 1
    for (int j = 0; j < K; ++j) {
        const uint32_t best = __reduce_max_sync(full, max(max(max(key[0], key[1]), max(key[2], key[3])), max(max(key[4], key[5]), max(key[6], key[7]))));
        int hits = 0, at = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (key[u] == best) { ++hits; at = u; key[u] = 0u; }
        const unsigned who = __ballot_sync(full, hits > 0);
        fine = fine && best != 0u && hits <= 1 && (who & (who - 1)) == 0u;
        if (hits) inds[j] = at * 32 + lane;
        if (lane == j) myv = key_float(best);
    }
    if (!__all_sync(full, fine)) return false;
    __syncwarp();
    const int myi = lane < K ? inds[lane] : 0x7FFFFFFF;
    const float m = __shfl_sync(full, myv, 0);
    const float ex = lane < K ? expf(myv - m) : 0.f;
    const float sum = warp_sum(ex);
    int rank = 0;
#pragma unroll 8
    for (int i = 0; i < K; ++i) rank += __shfl_sync(full, myi, i) < myi ? 1 : 0;
    __syncwarp();
    if (lane < K) { inds[rank] = myi; gates[rank] = ex / sum; }
    return true;
}

// The top-k of the logits in `work` by one warp, into the caller's inds_next / gates_next and, first, as one (expert, gate) word per
// choice into `pair` (this lane's word of the ring slot, or null), where a chained next step picks them up.  FENCE: what the
// publishers of the logits had observed travels on with them.  `work`: E floats and 256 bytes for the winners.
template <bool FENCE, typename P>
__device__ __forceinline__ void emit_routing(const P& p, float* work, int lane, unsigned long long* pair) {
    __syncwarp();
    int32_t* s_i = reinterpret_cast<int32_t*>(work) + p.E;        // [K] winners, then [K] gates
    float* s_g = reinterpret_cast<float*>(s_i + 32);
    if (p.E > 256 || !topk_distinct(work, p.E, p.K, lane, s_i, s_g)) topk_any(work, p.E, p.K, lane, s_i, s_g);
    __syncwarp();
    if (lane == 0) trace_stamp(p, 25);
    if (lane < p.K) {
        // the step that takes the pairs resets the slot only after all of its CTAs have read them, i.e.
        // after this warp has long finished with the logits
        if (pair != nullptr) {
            if (FENCE) __threadfence();
            if (lane == 0) trace_stamp(p, 26);
            st_relaxed_gpu_u64(pair, ((unsigned long long)__float_as_uint(s_g[lane]) << 32) | (uint32_t)s_i[lane]);
        }
        p.inds_next[lane] = s_i[lane];
        p.gates_next[lane] = s_g[lane];
        // (each entry is final by itself: the host polls the mirror until all K are >= 0)
        if (p.inds_mirror != nullptr)
            asm volatile("st.relaxed.sys.global.s32 [%0], %1;" ::"l"(p.inds_mirror + lane), "r"(s_i[lane]) : "memory");
    }
}

// One warp publishes head logits -- lane l owns logit `e` with value `v` when `own` is set -- into the
// ring slot the next layer-step reads, and if they were the last ones of the head, computes the
// top-k: the (expert, gate) pairs go behind the logits of the ring slot, where a chained next step
// picks them up, and into the caller's inds_next / gates_next.  `state` is the lane's entry of
// the ring slot as it was when the kernel started: a slot is written again only after the step
// that read it has ended and has reset it.  `work`: shared memory for the E logits and the winners, E * 4 + 256 bytes.
template <typename P>
__device__ __noinline__ void publish_logits(const P& p, float* work, float v, int e, bool own, int lane, uint32_t state) {
    int mine = 0;
    const int ring = p.flag_out >= 0 ? p.flag_out : 0;
    float* logits_ws = p.logits_ws + (size_t)ring * (p.E + kPairWords);
    int32_t* pre_counter = p.pre_counter + ring;
    if (own) {
        if (p.flag_out >= 0) {
            uint32_t it = 0;
            while (state != kNotYet && ++it < kSpinLimit) state = ld_relaxed_gpu_u32(&logits_ws[e]);
            if (state != kNotYet) atomicExch(p.status, EDG_E_TIMEOUT);
            // "the step that last read this slot is over" travels on to the reader of this logit
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
        }
        st_relaxed_gpu_u32(&logits_ws[e], __float_as_uint(v));
        mine = 1;
    }
    const int n_mine = __popc(__ballot_sync(0xFFFFFFFFu, mine));
    __syncwarp();
    int last = 0;
    // the counting atomic releases this warp's logits and acquires everyone else's
    if (lane == 0) last = (atom_add_acq_rel_gpu(pre_counter, n_mine) + n_mine == p.E) ? 1 : 0;
    last = __shfl_sync(0xFFFFFFFFu, last, 0);
    if (!last) return;
    if (lane == 0) {
        atomicSub(pre_counter, p.E);      // commutes with the arrivals of the head that uses this slot next
        trace_stamp(p, 16);
    }
#pragma unroll 1
    for (int i0 = 0; i0 < p.E; i0 += 256) {                     // 8 independent loads per lane and pass
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * 32 + lane;
            v[u] = i < p.E ? __ldcg(&logits_ws[i]) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * 32 + lane;
            if (i < p.E) {
                work[i] = v[u];
                if (p.logits_next != nullptr) p.logits_next[i] = v[u];
            }
        }
    }
    __syncwarp();
    if (lane == 0) trace_stamp(p, 17);
    emit_routing<true>(p, work, lane, p.flag_out >= 0 ? reinterpret_cast<unsigned long long*>(logits_ws + p.E) + lane : nullptr);
    if (lane == 0) trace_stamp(p, 15);
}

}  // namespace edg
