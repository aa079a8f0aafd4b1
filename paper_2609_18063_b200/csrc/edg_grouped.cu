// a4'-a6' grouped form (T tokens, each with its own top-K routing): the choice between the two engines, and the grouping
// and reduce of the tcgen05 engine.
//
// (token, choice) pairs are grouped per slot; each group is a small GEMM with the expert's int4 weights, dequantised on
// the fly.  Few pairs per slot (batched decode, chunks of a prompt) go through the streaming kernel of
// edg_grouped_ffn.cu, many (prefill) through the 128-token tcgen05 tiles of edg_grouped_umma.cu.  Every pair's
// gate-weighted output goes to a [T*K][H] scratch and is reduced per token in the order of its K choices, so y does not
// depend on how the groups were scheduled.
#include "edg_grouped.cuh"
#include "edg_ptx.cuh"

namespace edg {

// The slot of every (token, choice) pair.
__global__ void __launch_bounds__(256) umma_prepare_kernel(GroupedParams p) {
    pdl_launch_dependents();
    pdl_wait_prior_grid();
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i == 0) *p.n_tiles = 0;
    if (i < (size_t)p.T * p.K) {
        int s = p.slots[i];
        const int e = p.table != nullptr ? s : (p.experts != nullptr ? p.experts[i] : 0);
        if (p.table != nullptr) s = (s >= 0 && s < p.E) ? p.table[s] : -1;
        if (s < 0 || s >= p.n_slots || (p.rank > 0 && p.n_adapters != 1 && (e < 0 || e >= p.E))) { s = -1; atomicExch(p.status, EDG_E_RANGE); }
        p.pair_slot[i] = s;
    }
}

// One CTA per slot: the slot's pairs in ascending pair index (deterministic, no atomics), behind those of the slots before it, and the
// slot's tiles.  Each warp owns a contiguous range of pairs; a first pass counts, a second pass writes at the offsets.  (Which number
// a tile gets is decided by a counter: nothing that is computed depends on it.)
constexpr int kListWarps = 32;
__global__ void __launch_bounds__(kListWarps * 32) build_lists_kernel(GroupedParams p) {
    const int s = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ int s_cnt[kListWarps], s_less[kListWarps], s_first, s_tile0;
    pdl_launch_dependents();
    pdl_wait_prior_grid();
    const int P = p.T * p.K;
    const int per = ((P + kListWarps - 1) / kListWarps + 127) / 128 * 128;   // pairs per warp, a multiple of 128: four per lane at a time
    const int lo = min(P, warp * per), hi = min(P, lo + per);
    auto four = [&](int base) {                                          // (pair_slot is 256-byte aligned, base a multiple of 128)
        const int i = base + 4 * lane;
        if (i + 3 < hi) return __ldcg(reinterpret_cast<const int4*>(p.pair_slot + i));
        return make_int4(i < hi ? p.pair_slot[i] : -1, i + 1 < hi ? p.pair_slot[i + 1] : -1, i + 2 < hi ? p.pair_slot[i + 2] : -1, -1);
    };
    int cnt = 0, less = 0;
#pragma unroll 4
    for (int base = lo; base < hi; base += 128) {
        const int4 v = four(base);
        cnt += (v.x == s) + (v.y == s) + (v.z == s) + (v.w == s);
        less += ((unsigned)v.x < (unsigned)s) + ((unsigned)v.y < (unsigned)s) + ((unsigned)v.z < (unsigned)s) + ((unsigned)v.w < (unsigned)s);
    }
    cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
    less = __reduce_add_sync(0xFFFFFFFFu, less);
    if (lane == 0) { s_cnt[warp] = cnt; s_less[warp] = less; }
    __syncthreads();
    int off = 0, total = s_cnt[lane], start = s_less[lane];
    off = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? total : 0);
    total = __reduce_add_sync(0xFFFFFFFFu, total);
    start = __reduce_add_sync(0xFFFFFFFFu, start);
    if (total == 0) return;
    const int n_tiles = (total + kUmmaTokens - 1) / kUmmaTokens;
    if (threadIdx.x == 0) s_tile0 = atomicAdd(p.n_tiles, n_tiles);
    if (cnt > 0) {
        off += start;
#pragma unroll 4
        for (int base = lo; base < hi; base += 128) {
            const int4 v = four(base);
            const int mine = (v.x == s) + (v.y == s) + (v.z == s) + (v.w == s);
            if (!__any_sync(0xFFFFFFFFu, mine)) continue;
            int at = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xFFFFFFFFu, at, o);
                if (lane >= o) at += x;
            }
            const int all = __shfl_sync(0xFFFFFFFFu, at, 31);
            at += off - mine;
            const int i = base + 4 * lane;
            if (mine > 0 && at == start) s_first = v.x == s ? i : (v.y == s ? i + 1 : (v.z == s ? i + 2 : i + 3));
            if (v.x == s) p.order[at++] = i;
            if (v.y == s) p.order[at++] = i + 1;
            if (v.z == s) p.order[at++] = i + 2;
            if (v.w == s) p.order[at++] = i + 3;
            off += all;
        }
    }
    __syncthreads();
    int ad = 0;
    if (p.rank > 0 && p.n_adapters != 1) ad = p.table != nullptr ? p.slots[s_first] : p.experts[s_first];
    for (int t = threadIdx.x; t < n_tiles; t += kListWarps * 32)
        p.tiles[s_tile0 + t] = make_int4(s, start + t * kUmmaTokens, min(kUmmaTokens, total - t * kUmmaTokens), ad);
}

// ---------------------------------------------------------------- host

bool grouped_use_umma(const edg_layer_desc& d, int T) {
    return (int64_t)T * d.K > grouped_streaming_pairs(d) && umma_grouped_supported(d);
}
int64_t grouped_streaming_pairs(const edg_layer_desc& d) {
    return (int64_t)(d.group >= 64 && d.n_slots <= kUmmaSlots ? kUmmaPairsPerSlot : kUmmaPairsPerSlot32) * d.n_slots;
}

int32_t run_grouped(const edg_layer_desc* d, const void* slot_pool, int32_t T, const int32_t* slots, const int32_t* table,
                    const int32_t* experts, const float* gates, const void* x, const edg_lora* lora, void* y,
                    void* workspace, cudaStream_t st) {
    if (d->I % 128 != 0 || d->H % 256 != 0 || d->group > 128) return EDG_E_SHAPE;
    const bool has_lora = lora != nullptr && d->rank > 0;
    const WorkspaceLayout W = workspace_layout(*d, T);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    GroupedParams p{};
    p.pool = static_cast<const uint8_t*>(slot_pool);
    p.slots = slots; p.table = table; p.experts = experts; p.gates = gates;
    p.x = static_cast<const uint16_t*>(x);
    if (has_lora) p.lora = *lora;
    p.y = y;
    p.status = reinterpret_cast<int32_t*>(ws + W.ctrl);
    p.u_gu = reinterpret_cast<__half*>(ws + W.u_gu);
    p.u_d = reinterpret_cast<__half*>(ws + W.u_d);
    p.o = reinterpret_cast<float*>(ws + W.o);
    p.pair_slot = reinterpret_cast<int32_t*>(ws + W.pair_slot);
    p.T = T; p.H = d->H; p.I = d->I; p.E = d->E; p.K = d->K; p.group = d->group;
    while ((1 << p.gshift) < d->group) ++p.gshift;
    p.rank = has_lora ? d->rank : 0;
    p.n_adapters = d->n_adapters; p.n_slots = d->n_slots; p.out_dtype = d->out_dtype;
    p.sigma = d->lora_scale;
    p.L = record_layout(d->H, d->I, d->group);
    if (!grouped_use_umma(*d, T)) return run_grouped_ffn(d, p, W, ws, st);

    p.n_tiles = reinterpret_cast<int32_t*>(ws + W.n_tiles);
    p.tiles = reinterpret_cast<int4*>(ws + W.tiles);
    p.order = reinterpret_cast<int32_t*>(ws + W.order);
    p.hq = ws + W.hq;
    p.hf = has_lora && grouped_wide_h(*d) ? reinterpret_cast<float*>(ws + W.hf) : nullptr;
    p.xq = ws + W.xq;
    const size_t P = (size_t)T * d->K;
    const int max_tiles = (int)umma_max_tiles(*d, T);
    EDG_CUDA_TRY(launch_pdl(umma_prepare_kernel, dim3((unsigned)((P + 255) / 256)), 256, 0, st, p));
    EDG_CUDA_TRY(launch_pdl(build_lists_kernel, dim3(d->n_slots), kListWarps * 32, 0, st, p));
    if (has_lora) EDG_CUDA_TRY(launch_lora_ax(p, max_tiles, st));
    EDG_CUDA_TRY(launch_umma(p, false, max_tiles, st));
    if (has_lora) EDG_CUDA_TRY(launch_lora_adh(p, max_tiles, st));
    EDG_CUDA_TRY(launch_umma(p, true, max_tiles, st));
    EDG_CUDA_TRY(launch_sum_choices(p, st));
    return EDG_OK;
}

}  // namespace edg
