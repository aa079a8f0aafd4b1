// a4'-a6' grouped form (T tokens, each with its own top-K routing): the choice between the two engines, and the grouping
// and reduce of the tcgen05 engine.
//
// (token, choice) pairs are grouped per slot; each group is a small GEMM with the expert's int4 weights, dequantised on
// the fly.  Few pairs per slot (batched decode, chunks of a prompt) go through the streaming kernel of
// edg_grouped_ffn.cu, many (prefill) through the 128-token tcgen05 tiles of edg_grouped_umma.cu.  Every pair's
// gate-weighted output goes to a [T*K][H] scratch and is reduced per token in the order of its K choices, so y does not
// depend on how the groups were scheduled.
#include "edg_grouped.cuh"

namespace edg {

__global__ void resolve_pairs_kernel(GroupedParams p) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.T * p.K) return;
    int s = p.slots[i];
    const int e = p.table != nullptr ? s : (p.experts != nullptr ? p.experts[i] : 0);
    if (p.table != nullptr) s = (s >= 0 && s < p.E) ? p.table[s] : -1;
    int ad = 0;
    if (p.rank > 0 && p.n_adapters != 1) ad = (e >= 0 && e < p.E) ? e : -1;
    if (s < 0 || s >= p.n_slots || ad < 0) { s = -1; atomicExch(p.status, EDG_E_RANGE); }
    p.pair_slot[i] = s;
    p.pair_ad[i] = ad;
}

// One CTA per slot: the slot's pairs in ascending pair index (deterministic, no atomics).  Each
// warp owns a contiguous range of pairs; a first pass counts, a second pass writes at the offsets.
constexpr int kListWarps = 16;
__global__ void __launch_bounds__(kListWarps * 32) build_lists_kernel(GroupedParams p) {
    const int s = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ int s_cnt[kListWarps];
    const int P = p.T * p.K;
    const int per = ((P + kListWarps - 1) / kListWarps + 31) / 32 * 32;      // pairs per warp, a multiple of 32
    const int lo = warp * per, hi = min(P, lo + per);
    int cnt = 0;
    for (int base = lo; base < hi; base += 32) {
        const int i = base + lane;
        cnt += __popc(__ballot_sync(0xFFFFFFFFu, i < hi && p.pair_slot[i] == s));
    }
    if (lane == 0) s_cnt[warp] = cnt;
    __syncthreads();
    int off = 0, total = 0;
    for (int w = 0; w < kListWarps; ++w) { if (w < warp) off += s_cnt[w]; total += s_cnt[w]; }
    for (int base = lo; base < hi; base += 32) {
        const int i = base + lane;
        const bool m = i < hi && p.pair_slot[i] == s;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, m);
        if (m) p.lists[(size_t)s * p.T + off + __popc(bal & ((1u << lane) - 1))] = i;
        off += __popc(bal);
    }
    if (threadIdx.x == 0) p.counts[s] = total;
}

// Tile table: slot s contributes ceil(count / ntok) tiles; an exclusive scan over the slots gives
// each its first tile.  One CTA, slots strided over the threads, scan through shared memory.
__global__ void __launch_bounds__(1024) build_tiles_kernel(GroupedParams p) {
    __shared__ int s_n[1024];
    const int tid = threadIdx.x;
    // n_slots can exceed the block: each thread owns a contiguous run of slots
    const int per = (p.n_slots + 1023) / 1024;
    const int s0 = tid * per, s1 = min(p.n_slots, s0 + per);
    int mine = 0;
    for (int s = s0; s < s1; ++s) mine += (p.counts[s] + p.ntok - 1) / p.ntok;
    s_n[tid] = mine;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {          // inclusive scan
        const int v = tid >= o ? s_n[tid - o] : 0;
        __syncthreads();
        s_n[tid] += v;
        __syncthreads();
    }
    int n = s_n[tid] - mine;                       // exclusive prefix
    for (int s = s0; s < s1; ++s)
        for (int first = 0; first < p.counts[s]; first += p.ntok) { p.tiles[2 * n] = s; p.tiles[2 * n + 1] = first; ++n; }
    if (tid == 1023) *p.n_tiles = s_n[1023];
}

// ---------------------------------------------------------------- host

void launch_lora_a(const edg_layer_desc* d, const void* slots, const void* table, const void* experts, const void* x,
                   const edg_lora* lora, float* u_gu, float* h, float* u_d, int32_t* status, int T, int phase, cudaStream_t st);

bool grouped_use_umma(const edg_layer_desc& d, int T) {
    return (int64_t)T * d.K > (int64_t)kUmmaPairsPerSlot * d.n_slots && umma_grouped_supported(d);
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
    p.u_gu = reinterpret_cast<float*>(ws + W.u_gu);
    p.h = reinterpret_cast<float*>(ws + W.h);
    p.u_d = reinterpret_cast<float*>(ws + W.u_d);
    p.o = reinterpret_cast<float*>(ws + W.o);
    p.pair_slot = reinterpret_cast<int32_t*>(ws + W.pair_slot);
    p.T = T; p.H = d->H; p.I = d->I; p.E = d->E; p.K = d->K; p.group = d->group;
    p.rank = has_lora ? d->rank : 0;
    p.n_adapters = d->n_adapters; p.n_slots = d->n_slots; p.out_dtype = d->out_dtype;
    p.sigma = d->lora_scale;
    p.L = record_layout(d->H, d->I, d->group);
    if (!grouped_use_umma(*d, T)) return run_grouped_ffn(d, p, W, ws, st);

    p.pair_ad = reinterpret_cast<int32_t*>(ws + W.pair_ad);
    p.counts = reinterpret_cast<int32_t*>(ws + W.counts);
    p.n_tiles = reinterpret_cast<int32_t*>(ws + W.n_tiles);
    p.tiles = reinterpret_cast<int32_t*>(ws + W.tiles);
    p.lists = reinterpret_cast<int32_t*>(ws + W.lists);
    p.hq = ws + W.hq;
    p.xq = ws + W.xq;
    p.ntok = kUmmaTokens;
    const int P = T * d->K, max_tiles = (P + p.ntok - 1) / p.ntok + d->n_slots;
    resolve_pairs_kernel<<<(P + 255) / 256, 256, 0, st>>>(p);
    build_lists_kernel<<<d->n_slots, kListWarps * 32, 0, st>>>(p);
    build_tiles_kernel<<<1, 1024, 0, st>>>(p);
    if (has_lora && !launch_lora_ax_tokens(d, x, lora, p.u_gu, T, st))
        launch_lora_a(d, slots, table, experts, x, lora, p.u_gu, p.h, p.u_d, p.status, T, 0, st);
    EDG_CUDA_TRY(launch_umma_gate_up(p, max_tiles, st));
    if (has_lora && !launch_lora_adh_pairs(d, lora, p.h, p.u_d, P, st))
        launch_lora_a(d, slots, table, experts, x, lora, p.u_gu, p.h, p.u_d, p.status, T, 1, st);
    EDG_CUDA_TRY(launch_umma_down(p, max_tiles, st));
    EDG_CUDA_TRY(launch_sum_choices(p, st));
    return EDG_OK;
}

}  // namespace edg
