// A batch-1 layer-step that runs alone -- launched by itself on a stream, or as the next link of a chain of dependent steps --
// as ONE kernel over all SMs, built for latency (a1-a2 for the next step, a3 take, a4-a6 for this one).
//
// What bounds it is not the 15 MB it streams (2.4 us) but the chain of trips -- routing -> table -> weights -> h -> other
// CTAs -> y -- and the instructions between them.  So everything that does not depend on a trip is under way before it: a CTA
// issues all its gate/up weights at once (72 KB in eight bulk copies, by the warp that learns the routing; as 16-byte copies of
// all warps the issue alone took 2 us), announces its down weights to the L2, and loads its adapter rows; sixteen warps share
// the arithmetic.
//   * Gate/up: expert CTA 16 k + 4 c + j computes rows c I/4 + j I/16 .. of gate and up of routed expert k over all of
//     K = H.  Warp w multiplies H/512 chunks (32 codes each) of every row tile on mma.sync fragments.
//   * h, and the partial A_down h, go to all CTAs through global memory, in band: a word that does not hold the
//     "not yet" pattern (a NaN no arithmetic produces) is valid by itself, so the exchange costs one store and
//     one load on the way, and no barrier.  Four copies: 128 readers of the same lines queue at their slice of the L2.  The
//     rank-r projections A x are shared by all CTAs of the grid in the same way, those without expert work first; so are the
//     head's logits, which one warp turns into the next routing (a counter of arrivals with its fences took 10 us from x to
//     the routing, most of a step; now 7 us).
//   * Down: CTA d computes output rows 16 d .. 16 d + 15 over the h of ALL experts, so y needs no second pass over partials
//     (the throughput form writes 32 partial rows per output, counts arrivals and lets four CTAs sum them).
//   * Head rows have CTAs of their own, among those that the experts leave of one per SM.
//   * A dependent chain hands x + y on, unnormalised, in band as well: every CTA of the next step, resident and
//     with its weights in shared memory by then, polls it, forms the norm and its bf16 state by itself.  Eight copies: 148
//     pollers of the same lines held the writes up by 2-4 us.  A CTA without expert work writes the caller's x_next meanwhile.
// Two launches of this form fit an SM side by side (64 registers x 512 threads, under 113 KB of shared memory).  So do two steps that need
// nothing of one another (the layers of a token whose inputs are all given): such a run waits for what came before it once, in its first
// step; the others start beside their predecessor and leave after it.
//
// Measured (H 2048, I 512, E 256, K 8, groups of 64, rank 16; the four-CTA clusters per expert quarter it replaces first): a link of
// a chain 20.4 -> 12.1 us, a step alone 24 -> 14.1 us (12 layers of K = 4 through the resident stack, host loop included: 295 -> 154 us).
// Of the 12.1 us the two exchanges take 5.5 (a store, a poll under way, a poll that sees it, the slowest of 128), the
// arithmetic of gate/up 1.7, of down 1.6.
//
// Waiting is safe without a cooperative launch: a CTA reads the words of others only when all CTAs of its grid have
// started and cleared what they will publish (a counter in the control block says so).  One that finds its grid not fully resident for a while -- other grids hold the
// SMs -- leaves its down rows to the CTA that starts last.
// Nothing in the exchange buffers is taken over from a launch before: ahead of counting itself in, a CTA sets the words that it
// will publish to "not yet", a store or two per lane while the routing is on its way.  So it does not matter what the workspace
// held -- a prompt's scratch, the buffers of another layer shape, zeros --; the control block is all that has to last.
//
// The order of every sum is that of the throughput form of the layer kernel with four clusters per expert: per row four
// chains over K, per (expert, quarter of I) one partial with its adapter delta, partials summed in order.  A chain of
// dependent steps (EX = false: biased codes, edg_mma.cuh) therefore reproduces the results of earlier versions bit for bit.
#include <type_traits>

#include "edg_mma.cuh"
#include "edg_head.cuh"

namespace edg {
namespace {

constexpr int TW = 16;                        // warps
constexpr int TThreads = TW * 32;
constexpr int kStepMaxK = 16;
constexpr int kStepMaxRank = 64;
constexpr uint32_t kEpochStarts = 8192;       // what one grid adds to the start counter in total
constexpr uint32_t kWaitStarted = 256;        // polls before a CTA whose grid is not fully resident gives its rows away
constexpr int kStateCopies = 8, kHCopies = 4;

// byte offsets in shared memory; h .. udi lie inside the union, used once the gate/up weights are
struct StepSmem {
    uint32_t un, sz, sz_tile, xb, x, xsum, xbias, bgu, ad, bd, u4, uf, hl, sel, red, bar, total;
    uint32_t h, hb, hsum, hbias, part, udi;
};

struct StepParams {
    const uint8_t* pool;
    const int32_t *slots, *table, *experts;   // slots, or expert ids when table != null; experts: for the adapters otherwise
    const float* gates;
    const uint16_t* x;
    edg_lora lora, shared_lora;
    const uint8_t* shared_rec;
    void* y;
    int32_t* status;
    int32_t* done;                            // readers of a ring slot, in the control block
    float* logits_ws;                         // [ring][E + kPairWords]
    const void* W_pre;
    int32_t* inds_next;
    float *gates_next, *logits_next;
    int32_t* inds_mirror;
    uint16_t* x_next;
    uint32_t *starts, *ready;                 // CTAs that have started; that have cleared their words
    float* hx;                                // this link's exchange buffer: kHCopies of (h; the A_down h partials of every expert CTA); the A x partials; head logits
    float *vx, *vx_in;                        // [kStateCopies][H]: x + y of a dependent chain, of this link and of the one before it
    uint32_t* defer;                          // [kStepDeferWords]: units left to the CTA that starts last, a bit each
    uint32_t hc_words, ud_off, ux_off, lx_off;
    int I, E, K, Kt, group, gshift, rank, rank_shared, rmax, n_adapters, n_slots, pre_dtype, out_dtype;
    int cta_route, cta_state;                 // CTAs that compute the routing for the next step and the caller's x_next, or -1
    int n_gu, n_dn, n_exp, n_head, n_headc;   // CTAs with gate/up, with down work, the larger of both; tiles of the head, CTAs for them
    int head_tile;                            // rows of a tile of the head
    int flag_in, flag_out, dep;               // dep: x arrives in band from the step before
    int run;                                  // of independent steps: 1 begins one, 2 goes on with it
    float sigma, eps;
    RecordLayout L;
    StepSmem S;
};

__device__ __forceinline__ void trace_stamp(const StepParams&, int) {}                   // (this form is not traced)
__device__ __forceinline__ void cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ uint4 ld_relaxed16(const void* p) {
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed16(void* p, uint4 v) {
    asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ bool there(uint4 v) { return v.x != kNotYet && v.y != kNotYet && v.z != kNotYet && v.w != kNotYet; }
__device__ __forceinline__ float round_as(float v, int out_dtype) {      // a value as it reads back from the output type
    if (out_dtype == EDG_F32) return v;
    if (out_dtype == EDG_F16) return __half2float(__float2half_rn(v));
    uint32_t u = __float_as_uint(v);
    u += 0x7FFFu + ((u >> 16) & 1u);
    return __uint_as_float(u & 0xFFFF0000u);
}
// v + sum of eight bf16 products, in order
__device__ __forceinline__ float fma8(uint4 a, uint4 x, float v) {
    v = fmaf(bf16_lo(a.x), bf16_lo(x.x), v); v = fmaf(bf16_hi(a.x), bf16_hi(x.x), v);
    v = fmaf(bf16_lo(a.y), bf16_lo(x.y), v); v = fmaf(bf16_hi(a.y), bf16_hi(x.y), v);
    v = fmaf(bf16_lo(a.z), bf16_lo(x.z), v); v = fmaf(bf16_hi(a.z), bf16_hi(x.z), v);
    v = fmaf(bf16_lo(a.w), bf16_lo(x.w), v); v = fmaf(bf16_hi(a.w), bf16_hi(x.w), v);
    return v;
}
// sum_j B[j] u[j] over a bf16 row in shared memory, r a multiple of 8
__device__ __forceinline__ float b_dot(const uint16_t* B, const float* u, int r) {
    float d = 0.f;
    for (int j = 0; j < r; j += 8) {
        const uint4 b = *reinterpret_cast<const uint4*>(B + j);
        d = fmaf(bf16_lo(b.x), u[j + 0], d); d = fmaf(bf16_hi(b.x), u[j + 1], d);
        d = fmaf(bf16_lo(b.y), u[j + 2], d); d = fmaf(bf16_hi(b.y), u[j + 3], d);
        d = fmaf(bf16_lo(b.z), u[j + 4], d); d = fmaf(bf16_hi(b.z), u[j + 5], d);
        d = fmaf(bf16_lo(b.w), u[j + 6], d); d = fmaf(bf16_hi(b.w), u[j + 7], d);
    }
    return d;
}

// 1 / rms of the state x + y held four values a thread (thread t: 4 t ..), summed as the throughput form's four reducers do; every
// thread gets it.  s_red: 16 floats.
__device__ __forceinline__ float inv_rms(float* s_red, float4 v, bool on, int H, float eps) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float ss = 0.f;
    if (on) { ss = fmaf(v.x, v.x, ss); ss = fmaf(v.y, v.y, ss); ss = fmaf(v.z, v.z, ss); ss = fmaf(v.w, v.w, ss); }
    ss = warp_sum(ss);
    if (lane == 0) s_red[warp] = ss;
    __syncthreads();
    const int per = H / 512;                                     // warps per quarter of the rows
    float all = 0.f;
    for (int c = 0; c < 4; ++c) {
        float tot = 0.f;
        for (int w = 0; w < per; ++w) tot += s_red[c * per + w];
        all += tot;
    }
    return rsqrtf(all / (float)H + eps);
}

// 16 head rows (in shared memory, row by row with 16 bytes of padding) as the M of the MMA, the state as column 0, a quarter of K
// per warp of four; part [16] receives this warp's sums.
template <int H>
__device__ __forceinline__ void head_rows(const uint8_t* rows, const uint16_t* x, float* part, int warp, int lane) {
    const int g8 = lane >> 2, t4 = lane & 3;
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    const uint8_t* wr = rows + g8 * (H * 2 + 16) + warp * (H / 2) + t4 * 16;
#pragma unroll 8
    for (int j = 0; j < H / 128; ++j) {
        const uint4 a = *reinterpret_cast<const uint4*>(wr + j * 64), b = *reinterpret_cast<const uint4*>(wr + 8 * (H * 2 + 16) + j * 64);
        uint4 xb = make_uint4(0, 0, 0, 0);
        if (g8 == 0) {
            const uint4 v = *reinterpret_cast<const uint4*>(x + warp * (H / 4) + j * 32 + t4 * 8);
            xb = make_uint4(h2_as_u32(__floats2half2_rn(bf16_lo(v.x), bf16_hi(v.x))), h2_as_u32(__floats2half2_rn(bf16_lo(v.y), bf16_hi(v.y))),
                            h2_as_u32(__floats2half2_rn(bf16_lo(v.z), bf16_hi(v.z))), h2_as_u32(__floats2half2_rn(bf16_lo(v.w), bf16_hi(v.w))));
        }
        mma16816(c, a.x, b.x, a.y, b.y, xb.x, xb.y);
        mma16816(c, a.z, b.z, a.w, b.w, xb.z, xb.w);
    }
    if (t4 == 0) { part[g8] = c[0]; part[8 + g8] = c[2]; }
}

// NCK = H / 512: chunks of 32 codes per warp; DCH = I / 128: chunks of a quarter of I; CPB: chunks per scaled block; EX: code arithmetic.
template <int NCK, int DCH, int CPB, bool EX>
__global__ void __launch_bounds__(TThreads, 2) step_kernel(const __grid_constant__ StepParams p) {
    constexpr int H = NCK * 512, TG = DCH / 2, RG = 16 * TG, NT = 2 * TG, NBW = NCK / CPB, sw = 32 * DCH, NBQ = DCH / CPB;
    extern __shared__ __align__(128) uint8_t smem[];
    const StepSmem& S = p.S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g8 = lane >> 2, t4 = lane & 3;
    const int cta = blockIdx.x, crank = cta % 4;
    const bool has_gu = cta < p.n_gu, has_dn = cta < p.n_dn, has_head = cta >= p.n_exp && cta - p.n_exp < p.n_headc;
    const int kpos = cta / 16, n0 = ((cta % 16) / 4) * sw + crank * RG;  // this CTA's expert, and its first row of h
    const bool is_shared = kpos >= p.K;
    const edg_lora& lo = is_shared ? p.shared_lora : p.lora;
    const int r = has_gu ? (is_shared ? p.rank_shared : p.rank) : 0;

    uint8_t* un = smem + S.un;
    uint4* s_xb = reinterpret_cast<uint4*>(smem + S.xb);
    uint16_t* s_x = reinterpret_cast<uint16_t*>(smem + S.x);
    float* s_xsum = reinterpret_cast<float*>(smem + S.xsum);
    float* s_xbias = reinterpret_cast<float*>(smem + S.xbias);
    float* s_u4 = reinterpret_cast<float*>(smem + S.u4);                 // [4][2][kStepMaxRank]
    float* s_uf = reinterpret_cast<float*>(smem + S.uf);                 // [2][kStepMaxRank]
    float* s_hl = reinterpret_cast<float*>(smem + S.hl);                 // [RG]
    int* s_slot = reinterpret_cast<int*>(smem + S.sel);                  // [20] slot or -1, [20] gates, [20] adapters
    float* s_gate = reinterpret_cast<float*>(s_slot + 20);
    int* s_ad = s_slot + 40;
    int* s_misc = s_slot + 60;                                           // [0] epoch, [1] this CTA started last, [2], [3] scratch
    float* s_red = reinterpret_cast<float*>(smem + S.red);               // [64]
    uint64_t* bar_w = reinterpret_cast<uint64_t*>(smem + S.bar);         // gate/up weights
    constexpr int MP = CPB == 2 ? 2 : 1, VP = MP;                        // row tiles, and items of the down projection, at once
    constexpr int CT = NCK * TW * 256;                                   // bytes of a row tile's codes

    if (tid == 0) {
        mbar_init(bar_w, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // rows of A_gate, A_up of every set: four tasks (the four warps of the throughput form) per row, all CTAs share them, those without
    // expert work first, then the last warps of the others
    const int sets = p.n_adapters == 1 ? 1 : p.K;
    const int set_tasks = 8 * p.rank, n_task = sets * set_tasks + 8 * p.rank_shared, spare = (int)gridDim.x - p.n_exp;
    auto task_set = [&](int task) { return task >= sets * set_tasks ? sets : (sets == 1 ? 0 : task / set_tasks); };
    auto first_task = [&](int w) { return cta >= p.n_exp ? (TW - 1 - w) * spare + cta - p.n_exp : TW * spare + (TW - 1 - w) * p.n_exp + cta; };
    float* hx = p.hx;
    auto ux_word = [&](int task) {
        const int set = task_set(task), q = task - set * set_tasks;
        return hx + p.ux_off + (size_t)set * 8 * p.rmax + (q & 3) * 2 * p.rmax + (q >> 2);
    };
    // ---- start (warp 1): count this CTA in, let the next kernel come; "not yet" into every word this CTA will publish, and say so
    const bool links = p.flag_in >= 0 || p.flag_out >= 0 || p.run != 0;  // the next kernel may be one that does not wait for this one's end
    if (tid == 32) {
        uint32_t old;
        asm volatile("atom.relaxed.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(p.starts) : "memory");
        const bool last = old % kEpochStarts == gridDim.x - 1;
        if (last) {                                                      // (returns before the next kernel, which counts on, may come)
            uint32_t sum;
            asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(sum) : "l"(p.starts), "r"(kEpochStarts - gridDim.x) : "memory");
            s_misc[2] = (int)sum;
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
        }
        s_misc[0] = (int)(old / kEpochStarts);
        s_misc[1] = last ? 1 : 0;
        if (!links) pdl_launch_dependents();
    }
    // a step on its own: everything queued before it has happened (of a run of independent steps the first has seen to that)
    if (p.flag_in < 0 && p.run != 2) pdl_wait_prior_grid();
    if (warp == 1) {
        const uint4 none = make_uint4(kNotYet, kNotYet, kNotYet, kNotYet);
        if (has_gu) {
            for (int i = lane; i < kHCopies * RG / 4; i += 32)
                st_relaxed16(hx + (size_t)(i / (RG / 4)) * p.hc_words + (size_t)kpos * p.I + n0 + i % (RG / 4) * 4, none);
            for (int i = lane; i < r; i += 32)
                for (int c = 0; c < kHCopies; ++c) st_relaxed_gpu_u32(hx + (size_t)c * p.hc_words + p.ud_off + (size_t)cta * p.rmax + i, kNotYet);
        }
        if (lane < TW)
            for (int task = first_task(lane); task < n_task; task += TW * gridDim.x) st_relaxed_gpu_u32(ux_word(task), kNotYet);
        if (has_head && lane < p.head_tile)
            for (int e = (cta - p.n_exp) * p.head_tile + lane; e < p.E; e += p.n_headc * p.head_tile) st_relaxed_gpu_u32(hx + p.lx_off + e, kNotYet);
        if (has_dn && p.x_next != nullptr)
            for (int i = lane; i < kStateCopies * 4; i += 32) st_relaxed16(p.vx + (size_t)(i / 4) * H + cta * 16 + i % 4 * 4, none);
        if (p.flag_in < 0 && p.flag_out >= 0)                            // a chain starts: so does its hand-off ring
            for (int i = cta * 32 + lane; i < kHandoffRing * (p.E + kPairWords) / 4; i += gridDim.x * 32) st_relaxed16(p.logits_ws + (size_t)i * 4, none);
        __syncwarp();
        if (lane == 0) {
            // every grid adds kEpochStarts in total
            asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p.ready), "r"(cta == 0 ? kEpochStarts - gridDim.x + 1 : 1u) : "memory");
            if (links) {                                                 // (a link finds its words and its predecessor's cleared)
                __threadfence();
                pdl_launch_dependents();
            }
        }
    }
    // eight values of the state (value i of them): the B words of the MMAs, the block sums
    auto take_x = [&](int i, uint4 v) {
        const float f[8] = {bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y), bf16_lo(v.z), bf16_hi(v.z), bf16_lo(v.w), bf16_hi(v.w)};
        float scale = 1.f;
        if (EX) {                                                        // the largest magnitude of the state, over the warps that hold it
            uint32_t* s_max = reinterpret_cast<uint32_t*>(s_red) + 32;
            const uint32_t m = __reduce_max_sync(0xFFFFFFFFu, abs_max8(f));
            if (lane == 0) s_max[i / 32] = m;
            asm volatile("bar.sync 2, %0;" ::"n"(H / 8) : "memory");
            uint32_t all = 0;
#pragma unroll
            for (int w = 0; w < H / 256; ++w) all = max(all, s_max[w]);
            scale = vector_scale(all);
            if (i == 0) s_xbias[0] = kUnscaleS * vector_unscale(scale);
        }
        s_xb[i] = EX ? permute8_s(f, scale) : permute8(f);
        float sum = 0.f, sodd = 0.f;
#pragma unroll
        for (int e = 0; e < 8; e += 2) {                                 // of what the MMA sees
            sum += EX ? f[e] : __half2float(__float2half_rn(f[e]));
            sodd += EX ? f[e + 1] : __half2float(__float2half_rn(f[e + 1]));
        }
        sum = group_sum<4 * CPB>(sum);
        sodd = group_sum<4 * CPB>(sodd);
        if (i % (4 * CPB) == 0) {
            s_xsum[i / (4 * CPB)] = EX ? (sum + sodd) * (kScaleS * scale) : sum + sodd;
            if (!EX) s_xbias[i / (4 * CPB)] = fmaf(1024.f, sum, 64.f * sodd);
        }
    };
    if (!p.dep && tid >= TThreads - H / 8) {                             // (by the last warps: the first is after the routing)
        const int i = tid - (TThreads - H / 8);
        const uint4 v = __ldcg(reinterpret_cast<const uint4*>(p.x + i * 8));
        *reinterpret_cast<uint4*>(s_x + i * 8) = v;
        take_x(i, v);
    }
    const bool head_mma = p.pre_dtype == EDG_F16 && p.E % 16 == 0;
    auto load_head = [&](int tile, int threads) {                        // row by row, padded by 16 bytes against bank conflicts
        const uint8_t* src = static_cast<const uint8_t*>(p.W_pre) + (size_t)tile * 16 * H * 2;
#pragma unroll 4
        for (int i = tid; i < 16 * (H / 8); i += threads) cp16(un + (i / (H / 8)) * (H * 2 + 16) + (i % (H / 8)) * 16, src + (size_t)i * 16);
    };
    if (has_head && head_mma) load_head(cta - p.n_exp, TThreads);

    // ---- the routing (warp 0): from memory, or from the hand-off ring for a link of a chain
    if (warp == 0) {
        int vi = -1;
        float vg = 0.f;
        bool from_memory = p.flag_in < 0;
        if (p.flag_in >= 0) {
            const unsigned long long* pr = reinterpret_cast<const unsigned long long*>(p.logits_ws + (size_t)p.flag_in * (p.E + kPairWords) + p.E);
            unsigned long long w = 0;
            bool got = false;
            for (uint32_t it = 0; !got && it < kSpinLimit; ++it) {
                if (lane < p.K) w = ld_relaxed_gpu_u64(pr + lane);
                got = __all_sync(0xFFFFFFFFu, (uint32_t)w != kNotYet);
            }
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            if (got) { vi = (int)(uint32_t)w; vg = __uint_as_float((uint32_t)(w >> 32)); }
            else {                                                       // never seen: the previous kernel's end is always sufficient
                if (lane == 0) { atomicExch(p.status, EDG_E_TIMEOUT); pdl_wait_prior_grid(); }
                __syncwarp();
                from_memory = true;
            }
        }
        if (from_memory && lane < p.K) { vi = __ldcg(&p.slots[lane]); vg = __ldcg(&p.gates[lane]); }
        int slot = -1, ad = 0;
        if (lane < p.K) {
            const int expert = p.table != nullptr ? vi : (p.experts != nullptr ? __ldcg(&p.experts[lane]) : 0);
            slot = p.table != nullptr ? ((vi >= 0 && vi < p.E) ? __ldcg(&p.table[vi]) : -1) : vi;
            if (p.rank > 0 && p.n_adapters != 1) ad = (expert >= 0 && expert < p.E) ? expert : -1;
            if (slot < 0 || slot >= p.n_slots || ad < 0) { slot = -1; ad = 0; if (cta == 0) atomicExch(p.status, EDG_E_RANGE); }
        }
        if (lane == p.K && p.Kt > p.K) { slot = 0; vg = 1.f; }           // the shared expert: always on, weight 1
        if (lane < p.Kt) { s_slot[lane] = slot; s_gate[lane] = vg; s_ad[lane] = ad; }
        // all of this CTA's gate/up weights: a row tile's codes and its (scale, zero) pairs are one run each
        const int mine = __shfl_sync(0xFFFFFFFFu, slot, has_gu ? kpos : 0);
        if (has_gu && mine >= 0) {
            if (lane == 0) mbar_expect_tx(bar_w, NT * (CT + S.sz_tile));
            __syncwarp();
            const uint8_t* rec = is_shared ? p.shared_rec : p.pool + (size_t)mine * p.L.bytes;
            const int mt = lane % NT, n = n0 + 16 * (mt % TG);
            if (lane < NT) bulk_g2s(un + mt * CT, rec + (mt / TG ? p.L.codes_up : p.L.codes_gate) + code_off(H, n, 0), CT, bar_w);
            else if (lane < 2 * NT) bulk_g2s(smem + S.sz + mt * S.sz_tile, rec + (mt / TG ? p.L.sz_up : p.L.sz_gate) + sz_off(H, p.group, n, 0), S.sz_tile, bar_w);
        }
    }
    __syncthreads();
    const uint32_t epoch = (uint32_t)s_misc[0];
    auto record = [&](int k) { return k >= p.K ? p.shared_rec : p.pool + (size_t)s_slot[k] * p.L.bytes; };
    const bool valid = has_gu && s_slot[kpos] >= 0;
    const int gsh = p.gshift, ad_k = has_gu ? s_ad[kpos] : 0;

    // ---- the adapter's slices: this CTA's rows of B_gate and B_up, its columns of A_down, B_down rows of its output rows
    if (valid && r > 0) {
        const int per = RG * r / 8;                                      // 16-byte pieces of one matrix's rows
        for (int i = tid; i < 2 * per; i += TThreads) {
            const uint16_t* B = static_cast<const uint16_t*>(i >= per ? lo.B_up : lo.B_gate) + ((size_t)ad_k * p.I + n0) * r;
            cp16(smem + S.bgu + i * 16, B + (i % per) * 8);
        }
        constexpr int cpr = RG / 8;
        for (int i = tid; i < r * cpr; i += TThreads)
            cp16(smem + S.ad + i * 16, static_cast<const uint16_t*>(lo.A_down) + ((size_t)ad_k * r + i / cpr) * p.I + n0 + (i % cpr) * 8);
    }
    auto load_bd = [&](int d) {                                          // [set][16][rank]: one set, or one per expert; the shared expert's behind them
        for (int s = warp; s <= sets; s += TW) {
            const int rk = s == sets ? p.rank_shared : p.rank;
            const void* B = s == sets ? p.shared_lora.B_down : p.lora.B_down;
            const size_t row = (size_t)(s == sets || p.n_adapters == 1 ? 0 : s_ad[s]) * H + d * 16;
            for (int i = lane; i < 2 * rk; i += 32)
                cp16(smem + S.bd + (size_t)s * 32 * p.rmax + i * 16, static_cast<const uint16_t*>(B) + row * rk + i * 8);
        }
    };
    if (has_dn) load_bd(cta);
    cp_commit();
    // ---- its down weights are announced to the L2, an (expert, quarter of I) per lane
    if (has_dn && warp == 1)
        for (int i = lane; i < p.Kt * 4; i += 32)
            if (s_slot[i >> 2] >= 0) {
                const uint8_t* rec = record(i >> 2);
                bulk_prefetch_l2(rec + p.L.codes_down + (size_t)(i & 3) * ((size_t)H * sw / 2) + code_off(sw, cta * 16, 0), DCH * 256);
                bulk_prefetch_l2(rec + p.L.sz_down + down_sz_off(H, p.I, p.group, cta * 16, (i & 3) * (sw >> gsh)), (sw >> gsh) * 64);
            }
    auto a_row = [&](int set, int q) {                                   // lane's first values of task q of a set
        const edg_lora& l = set == sets ? p.shared_lora : p.lora;
        const int rk = set == sets ? p.rank_shared : p.rank, up = (q >> 2) >= rk ? 1 : 0;
        const size_t row = (size_t)(set == sets || p.n_adapters == 1 ? 0 : s_ad[set]) * rk + ((q >> 2) - up * rk);
        return static_cast<const uint16_t*>(up ? l.A_up : l.A_gate) + row * H + ((q & 3) * 32 + lane) * 8;
    };
    const int task0 = first_task(warp);
    uint4 pa[NCK / 2];
    if (task0 < n_task) {
        const int set = task_set(task0);
        const uint16_t* a = a_row(set, task0 - set * set_tasks);
#pragma unroll
        for (int sweep = 0; sweep < NCK / 2; ++sweep) pa[sweep] = ld_keep16(a + sweep * 1024);
    }
    // Have all CTAs of this grid started, and cleared their words?  (Asked by the warps that read A x, by one at least, while they wait
    // for something else; ahead of the products it would hold them up.)
    auto all_ready = [&]() {
        uint32_t c;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(p.ready) : "memory");
        return c / kEpochStarts != epoch;
    };
    const bool asks = warp >= 8 && (warp == 8 || tid - 256 < 2 * r);
    bool open = asks && all_ready();
    // A_down h partials this thread adds up (tid -> (expert and quarter, rank))
    const int udq = p.rmax > 0 ? tid / p.rmax : 0, udj = tid - udq * p.rmax, udn = p.rmax > 0 ? TThreads / p.rmax : TThreads;   // (none: no rounds beyond those of h)
    // ---- the hidden state
    if (p.dep) {
        const bool on = tid * 4 < H;
        const float* src = p.vx_in + (size_t)(cta % kStateCopies) * H + 4 * tid;
        uint4 w = make_uint4(0, 0, 0, 0);
        bool got = !on;
        for (uint32_t it = 0; !got && it < kSpinLimit; ++it) {
            w = ld_relaxed16(src);
            got = there(w);
            if (!got) __nanosleep(32);
        }
        const float4 v = make_float4(__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w));
        const int fail = __syncthreads_or(!got);
        const float inv = inv_rms(s_red, v, on, H, p.eps);
        if (on) {
            bf16_t* xs = reinterpret_cast<bf16_t*>(s_x) + 4 * tid;
            store_out<bf16_t>(xs, 0, v.x * inv); store_out<bf16_t>(xs, 1, v.y * inv);
            store_out<bf16_t>(xs, 2, v.z * inv); store_out<bf16_t>(xs, 3, v.w * inv);
        }
        if (fail) {                                                      // it did not come: the previous kernel's end is always sufficient
            if (tid == 0) { atomicExch(p.status, EDG_E_TIMEOUT); pdl_wait_prior_grid(); }
            __syncthreads();
            if (on) *reinterpret_cast<uint2*>(s_x + 4 * tid) = __ldcg(reinterpret_cast<const uint2*>(p.x + 4 * tid));
        }
        __syncthreads();
    }
    if (p.dep && tid < H / 8) take_x(tid, *reinterpret_cast<const uint4*>(s_x + tid * 8));
    if (has_head) cp_wait<0>();
    if (p.dep || has_head) __syncthreads();
    // a word of another CTA that does not come: the result is flagged at the very end
    auto late = [&](uint32_t it) {
        if (it < kSpinLimit) return false;
        atomicExch(p.status, EDG_E_TIMEOUT);
        return true;
    };
    // ---- the head's rows.  Four warps take tiles of 16 through the tensor cores; any other head goes in tiles of four, a row in four tasks
    if (has_head && head_mma && warp < 4) {
#pragma unroll 1
        for (int tile = cta - p.n_exp; tile < p.n_head; tile += p.n_headc) {
            if (tile >= p.n_headc) {                                     // (the first tile has been on its way since the start)
                load_head(tile, 128);
                cp_commit();
                cp_wait<0>();
                asm volatile("bar.sync 1, 128;" ::: "memory");
            }
            head_rows<H>(un, s_x, s_red + warp * 16, warp, lane);
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (tid < 16) {
                float lg = s_red[tid];
                for (int w = 1; w < 4; ++w) lg += s_red[w * 16 + tid];   // fixed order
                st_relaxed_gpu_u32(hx + p.lx_off + tile * 16 + tid, __float_as_uint(lg));
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");
        }
    } else if (has_head && !head_mma) {
#pragma unroll 1
        for (int tile = cta - p.n_exp; tile < p.n_head; tile += p.n_headc) {
            const int e = tile * 4 + (warp >> 2), part = (warp & 3) * 32 + lane;
            float acc = 0.f;
            if (e < p.E && p.pre_dtype == EDG_F16) {
                const __half* wr = static_cast<const __half*>(p.W_pre) + (size_t)e * H;
                for (int c = part * 8; c < H; c += 1024) {
                    const uint4 w = ld_keep16(wr + c);
                    const uint4 xv = *reinterpret_cast<const uint4*>(s_x + c);
                    const float2 a = __half22float2(u32_as_h2(w.x)), b = __half22float2(u32_as_h2(w.y));
                    const float2 d = __half22float2(u32_as_h2(w.z)), f = __half22float2(u32_as_h2(w.w));
                    acc = fmaf(a.x, bf16_lo(xv.x), acc); acc = fmaf(a.y, bf16_hi(xv.x), acc);
                    acc = fmaf(b.x, bf16_lo(xv.y), acc); acc = fmaf(b.y, bf16_hi(xv.y), acc);
                    acc = fmaf(d.x, bf16_lo(xv.z), acc); acc = fmaf(d.y, bf16_hi(xv.z), acc);
                    acc = fmaf(f.x, bf16_lo(xv.w), acc); acc = fmaf(f.y, bf16_hi(xv.w), acc);
                }
            } else if (e < p.E) {
                const float* wr = static_cast<const float*>(p.W_pre) + (size_t)e * H + part * 4;
                uint4 w[NCK];
#pragma unroll
                for (int j = 0; j < NCK; ++j) w[j] = ld_keep16(wr + j * 512);
#pragma unroll
                for (int j = 0; j < NCK; ++j) {
                    const uint2 xv = *reinterpret_cast<const uint2*>(s_x + part * 4 + j * 512);
                    acc = fmaf(__uint_as_float(w[j].x), bf16_lo(xv.x), acc); acc = fmaf(__uint_as_float(w[j].y), bf16_hi(xv.x), acc);
                    acc = fmaf(__uint_as_float(w[j].z), bf16_lo(xv.y), acc); acc = fmaf(__uint_as_float(w[j].w), bf16_hi(xv.y), acc);
                }
            }
            acc = warp_sum(acc);
            __syncthreads();                                             // (the sums of the tile before have been read)
            if (lane == 0) s_red[warp] = acc;
            __syncthreads();
            if (tid < 4 && tile * 4 + tid < p.E) {
                float lg = 0.f;
                for (int w = 0; w < 4; ++w) lg += s_red[tid * 4 + w];
                st_relaxed_gpu_u32(hx + p.lx_off + tile * 4 + tid, __float_as_uint(lg));
            }
        }
    }
    // ---- this warp's share of A x
    auto a_dot = [&](int set, int q, bool first) {
        float v = 0.f;
        const uint16_t* a = a_row(set, q);
#pragma unroll
        for (int sweep = 0; sweep < NCK / 2; ++sweep)
            v = fma8(first ? pa[sweep] : ld_keep16(a + sweep * 1024), *reinterpret_cast<const uint4*>(s_x + sweep * 1024 + ((q & 3) * 32 + lane) * 8), v);
        return warp_sum(v);
    };
#pragma unroll 1
    for (int task = task0; task < n_task; task += TW * gridDim.x) {
        const int set = task_set(task), q = task - set * set_tasks;
        const float v = a_dot(set, q, task == task0);
        if (lane == 0) st_relaxed_gpu_u32(ux_word(task), __float_as_uint(v));
    }
    if (valid) {
        // ---- gate/up on the tensor cores, a gate tile and its up tile at once where the registers allow it; per (row, scaled block)
        // the scale and what it multiplies stay in the region the codes came in
        mbar_wait(bar_w, 0, p.status);
        const uint4* xbp = s_xb + warp * NCK * 4 + t4;
#pragma unroll 1
        for (int t = 0; t < NT / MP; ++t) {
            float c[MP][NBW][4];
#pragma unroll
            for (int u = 0; u < CPB; ++u)
#pragma unroll
                for (int b = 0; b < NBW; ++b) {
                    const int i = b * CPB + u;
                    uint4 xb = make_uint4(0, 0, 0, 0);
                    if (g8 == 0) xb = xbp[i * 4];
#pragma unroll
                    for (int m = 0; m < MP; ++m) {
                        const uint8_t* cb = un + (m * TG + t) * CT + (warp * NCK + i) * 256 + g8 * 16 + t4 * 4;
                        uint32_t alo[4], ahi[4];
                        dequant_code_word<EX>(*reinterpret_cast<const uint32_t*>(cb), alo);
                        dequant_code_word<EX>(*reinterpret_cast<const uint32_t*>(cb + 128), ahi);
                        if (u == 0) mma16816_zero(c[m][b], alo[0], ahi[0], alo[1], ahi[1], xb.x, xb.y);
                        else mma16816(c[m][b], alo[0], ahi[0], alo[1], ahi[1], xb.x, xb.y);
                        mma16816(c[m][b], alo[2], ahi[2], alo[3], ahi[3], xb.z, xb.w);
                    }
                }
            __syncwarp();                                                // every lane is done with these tiles' codes
            if (t4 == 0) {
                const int at = (g8 + 4 * (warp >> 1)) & 15;              // rotated against bank conflicts
#pragma unroll
                for (int b = 0; b < NBW; ++b) {
                    const int blk = warp * NBW + b;
                    const float xs = s_xsum[blk], xbias = EX ? 0.f : s_xbias[blk];
#pragma unroll
                    for (int m = 0; m < MP; ++m) {
                        const uint8_t* zb = smem + S.sz + (m * TG + t) * S.sz_tile + ((blk * CPB * 32) >> gsh) * 64 + g8 * 4;
                        const __half2 z0 = u32_as_h2(*reinterpret_cast<const uint32_t*>(zb)), z1 = u32_as_h2(*reinterpret_cast<const uint32_t*>(zb + 32));
                        float2* ts = reinterpret_cast<float2*>(un + (m * TG + t) * CT + warp * NCK * 256) + b * 16;      // [16 rows] (scale, term)
                        ts[at] = make_float2(__low2float(z0), fmaf(-__high2float(z0), xs, EX ? c[m][b][0] : c[m][b][0] - xbias));
                        ts[at ^ 8] = make_float2(__low2float(z1), fmaf(-__high2float(z1), xs, EX ? c[m][b][2] : c[m][b][2] - xbias));
                    }
                }
            }
        }
    }
    // A x of this expert: the four tasks of a row, from whoever has computed them
    if (asks)
        for (uint32_t it = 0; !open && (it < kWaitStarted || (s_misc[1] && it < kSpinLimit)); ++it) open = all_ready();
    if (open && valid && tid - 256 < 2 * r) {
        const float* ux = hx + p.ux_off + (size_t)(is_shared ? sets : (p.n_adapters == 1 ? 0 : kpos)) * 8 * p.rmax + (tid - 256);
        uint32_t u[4];
        bool got = false;
        for (uint32_t it = 0; !got; ++it) {
#pragma unroll
            for (int w = 0; w < 4; ++w) u[w] = ld_relaxed_gpu_u32(ux + w * 2 * p.rmax);
            got = (u[0] != kNotYet && u[1] != kNotYet && u[2] != kNotYet && u[3] != kNotYet) || late(it);
        }
        s_uf[tid - 256] = ((__uint_as_float(u[0]) + __uint_as_float(u[1])) + __uint_as_float(u[2])) + __uint_as_float(u[3]);
    }
    cp_wait<0>();
    open = !__syncthreads_or(asks && !open);
    if (!open) {                                                         // not all of this grid is resident: all of them here
        const int set = is_shared ? sets : (p.n_adapters == 1 ? 0 : kpos);
#pragma unroll 1
        for (int q = warp; q < 8 * r; q += TW) {
            const float u = a_dot(set, q, false);
            if (lane == 0) s_u4[(q & 3) * 2 * kStepMaxRank + (q >> 2)] = u;
        }
        __syncthreads();
        if (tid < 2 * r) {
            float u = 0.f;
            for (int w = 0; w < 4; ++w) u += s_u4[w * 2 * kStepMaxRank + tid];
            s_uf[tid] = u;
        }
        __syncthreads();
    }

    // ---- finish gate/up: four chains per row (as the four warps of the throughput form), adapter, SiLU, product
    if (has_gu) {
        if (tid < 2 * RG * 4) {
            float v = 0.f;
            const int slot = tid >> 2, w = tid & 3, m = slot & 1, i = slot >> 1, mt = m * TG + (i >> 4), row = i & 15;
            if (valid) {
                constexpr int NB = 2 * NBW;                              // blocks of one half of a chain
#pragma unroll
                for (int half = 0; half < 2; ++half)
#pragma unroll
                    for (int j = 0; j < NB; ++j) {
                        const int blk = (w + 4 * half) * NB + j;         // block of the row; NBW of them per warp here
                        const float2 st = reinterpret_cast<const float2*>(un + mt * CT + (blk / NBW) * NCK * 256)[(blk % NBW) * 16 + ((row + 4 * w) & 15)];
                        v = fmaf(st.x, st.y, v);
                    }
                if (EX) v *= s_xbias[0];
            }
            const float p1 = __shfl_down_sync(0xFFFFFFFFu, v, 1), p2 = __shfl_down_sync(0xFFFFFFFFu, v, 2), p3 = __shfl_down_sync(0xFFFFFFFFu, v, 3);
            v = ((v + p1) + p2) + p3;
            if (valid && r > 0 && w == 0)
                v = fmaf(p.sigma, b_dot(reinterpret_cast<const uint16_t*>(smem + S.bgu) + (m * RG + i) * r, s_uf + m * r, r), v);
            const float up = __shfl_down_sync(0xFFFFFFFFu, v, 4);
            if ((tid & 7) == 0) {
                s_hl[i] = valid ? silu_f(v) * up : 0.f;
            }
        }
        __syncthreads();
        if (warp == TW - 1)                                              // h goes out, 16 bytes and a copy per lane
            for (int i = lane; i < kHCopies * RG / 4; i += 32)
                st_relaxed16(hx + (size_t)(i / (RG / 4)) * p.hc_words + (size_t)kpos * p.I + n0 + i % (RG / 4) * 4, reinterpret_cast<const uint4*>(s_hl)[i % (RG / 4)]);
        if (r > 0 && warp * 8 < r) {                                     // partial of A_down h over this CTA's rows, four lanes per rank
            const uint16_t* A = reinterpret_cast<const uint16_t*>(smem + S.ad);
            const int j = tid >> 2, part = tid & 3;                      // (TThreads / 4 ranks in one go: kStepMaxRank and more)
            float u = 0.f;
            if (j < r && valid)
                for (int n = part; n < RG; n += 4) u = fmaf(bf16_bits_to_float(A[j * RG + n]), s_hl[n], u);
            u = group_sum<4>(u);
            static_assert(kHCopies == 4, "a copy per lane of the group");
            if (j < r) st_relaxed_gpu_u32(hx + (size_t)part * p.hc_words + p.ud_off + (size_t)cta * p.rmax + j, __float_as_uint(u));
        }
    }

    // ---- the down weights of this CTA's output rows: the first two items of every warp are on their way from here on
    constexpr int kPre = 2;
    uint32_t dw[kPre][DCH][2], dz[kPre][NBQ][2];
    const int n_items = p.Kt * 4;                                        // (expert, quarter of I)
    auto load_item = [&](int d, int item, uint32_t (&w)[DCH][2], uint32_t (&z)[NBQ][2]) {
        const int k = min(item >> 2, p.Kt - 1), c = item & 3;
        const bool ok = item < n_items && s_slot[k] >= 0;
        const uint8_t* rec = ok ? record(k) : p.pool;
        const uint8_t* cw = rec + p.L.codes_down + (size_t)c * ((size_t)H * sw / 2) + code_off(sw, d * 16, 0) + g8 * 16 + t4 * 4;
        const uint8_t* cz = rec + p.L.sz_down + down_sz_off(H, p.I, p.group, d * 16, c * (sw >> gsh)) + g8 * 4;
#pragma unroll
        for (int i = 0; i < DCH; ++i) { w[i][0] = ok ? ld_stream4(cw + i * 256) : 0u; w[i][1] = ok ? ld_stream4(cw + i * 256 + 128) : 0u; }
#pragma unroll
        for (int b = 0; b < NBQ; ++b) {
            const int gi = (b * CPB * 32) >> gsh;
            z[b][0] = ok ? ld_stream4(cz + gi * 64) : 0u; z[b][1] = ok ? ld_stream4(cz + gi * 64 + 32) : 0u;
        }
    };
    if (has_dn) {
#pragma unroll
        for (int u = 0; u < kPre; ++u) load_item(cta, warp + u * TW, dw[u], dz[u]);
    }

    constexpr int kHPad = 32 * CPB + 4;                                  // (a block of h, padded against bank conflicts)

    // ---- down: output rows 16 d .. 16 d + 15 over the h of all experts
    float* s_h = reinterpret_cast<float*>(un + S.h);
    uint4* s_hb = reinterpret_cast<uint4*>(un + S.hb);
    float* s_hsum = reinterpret_cast<float*>(un + S.hsum);
    float* s_hbias = reinterpret_cast<float*>(un + S.hbias);
    float* s_part = reinterpret_cast<float*>(un + S.part);               // [items][17]
    float* s_udi = reinterpret_cast<float*>(un + S.udi);                 // [items][rmax + 1]
    auto down_unit = [&](int d, auto is_own) {
        constexpr bool own = decltype(is_own)::value;
        const int n8 = p.Kt * p.I / 8;
        const float* hr = hx + (size_t)(cta % kHCopies) * p.hc_words;
#pragma unroll 1
        for (int i0 = 0, m = 0; i0 < n8 || m * udn < n_items; i0 += TThreads, ++m) {
            const int i = i0 + tid, item = m * udn + udq;
            const bool on = i < n8, ud = udq < udn && item < n_items && p.rmax > 0 && (item >= 4 * p.K ? p.rank_shared : p.rank) > 0;
            uint4 a = make_uint4(0, 0, 0, 0), b = a, u = a;
            const float* up = hr + p.ud_off + (size_t)item * 4 * p.rmax + udj;
            bool got = !on && !ud;
            for (uint32_t it = 0; !got; ++it) {
                if (on) { a = ld_relaxed16(hr + i * 8); b = ld_relaxed16(hr + i * 8 + 4); }
                if (ud) {
                    u.x = ld_relaxed_gpu_u32(up); u.y = ld_relaxed_gpu_u32(up + p.rmax);
                    u.z = ld_relaxed_gpu_u32(up + 2 * p.rmax); u.w = ld_relaxed_gpu_u32(up + 3 * p.rmax);
                }
                got = (there(a) && there(b) && there(u)) || late(it);
            }
            if (ud)                                                      // A_down h of an (expert, quarter): its four CTAs in order
                s_udi[item * (p.rmax + 1) + udj] = ((__uint_as_float(u.x) + __uint_as_float(u.y)) + __uint_as_float(u.z)) + __uint_as_float(u.w);
            const float f[8] = {__uint_as_float(a.x), __uint_as_float(a.y), __uint_as_float(a.z), __uint_as_float(a.w),
                                __uint_as_float(b.x), __uint_as_float(b.y), __uint_as_float(b.z), __uint_as_float(b.w)};
            const float scale = EX ? vector_scale(group_max<4 * DCH>(abs_max8(f))) : 1.f;      // of an (expert, quarter)
            if (on) {                                                    // [chunk][value, residual][4]
                s_hb[(i >> 2) * 8 + (i & 3)] = EX ? permute8_s(f, scale) : permute8(f);
                s_hb[(i >> 2) * 8 + 4 + (i & 3)] = EX ? permute8_lo_s(f, scale) : permute8_lo(f);
            }
            if (EX) {
                float s = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7]));
                s = group_sum<4 * CPB>(s);
                if (on && i % (4 * CPB) == 0) s_hsum[i / (4 * CPB)] = s * (kScaleS * scale);
                if (on && i % (4 * DCH) == 0) s_hbias[i / (4 * DCH)] = kUnscaleS * vector_unscale(scale);
            } else if (on) {
                float* q = s_h + (i / (4 * CPB)) * kHPad + (i % (4 * CPB)) * 8;
                *reinterpret_cast<uint4*>(q) = a;
                *reinterpret_cast<uint4*>(q + 4) = b;
            }
        }
        if constexpr (!own) { load_bd(d); cp_commit(); cp_wait<0>(); }
        __syncthreads();
        if (!EX) {                                                       // block sums in the order of the throughput form
            for (int blk = tid; blk < p.Kt * p.I / (32 * CPB); blk += TThreads) {
                const float4* hq = reinterpret_cast<const float4*>(s_h + blk * kHPad);
                float v = 0.f, vo = 0.f;
#pragma unroll
                for (int e = 0; e < 8 * CPB; ++e) {
                    const float4 q = hq[e];
                    v += q.x; vo += q.y; v += q.z; vo += q.w;
                }
                s_hsum[blk] = v + vo;
                s_hbias[blk] = fmaf(1024.f, v, 64.f * vo);
            }
            __syncthreads();
        }
        auto delta = [&](int item) {                                     // adapter delta of row `warp` for an (expert, quarter)
            const int k = item >> 2, rk = k >= p.K ? p.rank_shared : p.rank, set = k >= p.K ? sets : (p.n_adapters == 1 ? 0 : k);
            return b_dot(reinterpret_cast<const uint16_t*>(smem + S.bd) + (size_t)set * 16 * p.rmax + warp * rk, s_udi + item * (p.rmax + 1), rk);
        };
        const float dl0 = p.rmax > 0 && lane < n_items ? delta(lane) : 0.f;
#pragma unroll 1
        for (int i0 = warp; i0 < n_items; i0 += kPre * TW) {
            if (!own || i0 != warp) {
#pragma unroll
                for (int v = 0; v < kPre; ++v) load_item(d, i0 + v * TW, dw[v], dz[v]);
            }
#pragma unroll
            for (int v0 = 0; v0 < kPre; v0 += VP) {
                float c[VP][NBQ][4];
#pragma unroll
                for (int u = 0; u < CPB; ++u)
#pragma unroll
                    for (int b = 0; b < NBQ; ++b)
#pragma unroll
                        for (int v = 0; v < VP; ++v) {
                            const int i = b * CPB + u, item = min(i0 + (v0 + v) * TW, n_items - 1);
                            uint4 hb = make_uint4(0, 0, 0, 0);
                            if (g8 < 2) hb = s_hb[((item * DCH + i) * 2 + g8) * 4 + t4];
                            uint32_t alo[4], ahi[4];
                            dequant_code_word<EX>(dw[v0 + v][i][0], alo);
                            dequant_code_word<EX>(dw[v0 + v][i][1], ahi);
                            if (u == 0) mma16816_zero(c[v][b], alo[0], ahi[0], alo[1], ahi[1], hb.x, hb.y);
                            else mma16816(c[v][b], alo[0], ahi[0], alo[1], ahi[1], hb.x, hb.y);
                            mma16816(c[v][b], alo[2], ahi[2], alo[3], ahi[3], hb.z, hb.w);
                        }
#pragma unroll
                for (int v = 0; v < VP; ++v) {
                    const int item = i0 + (v0 + v) * TW;
                    if (t4 == 0 && item < n_items) {
                        float acc_lo = 0.f, acc_hi = 0.f;
#pragma unroll
                        for (int b = 0; b < NBQ; ++b) {
                            const __half2 z0 = u32_as_h2(dz[v0 + v][b][0]), z1 = u32_as_h2(dz[v0 + v][b][1]);
                            const float hs = s_hsum[item * NBQ + b], hbias = EX ? 0.f : s_hbias[item * NBQ + b];
                            acc_lo = fmaf(__low2float(z0), fmaf(-__high2float(z0), hs, EX ? c[v][b][0] + c[v][b][1] : c[v][b][0] + c[v][b][1] - hbias), acc_lo);
                            acc_hi = fmaf(__low2float(z1), fmaf(-__high2float(z1), hs, EX ? c[v][b][2] + c[v][b][3] : c[v][b][2] + c[v][b][3] - hbias), acc_hi);
                        }
                        s_part[item * 17 + g8] = EX ? acc_lo * s_hbias[item] : acc_lo;
                        s_part[item * 17 + 8 + g8] = EX ? acc_hi * s_hbias[item] : acc_hi;
                    }
                }
            }
        }
        __syncthreads();
        // warp w: row w; lane: (expert, quarter).  Adapter delta, gate weight, then the sum in order.
        float yv = 0.f;
        for (int b0 = 0; b0 < n_items; b0 += 32) {
            const int item = b0 + lane;
            float o = 0.f;
            if (item < n_items && s_slot[item >> 2] >= 0) o = s_gate[item >> 2] * fmaf(p.sigma, b0 == 0 ? dl0 : delta(item), s_part[item * 17 + warp]);
            const int n = min(32, n_items - b0);
#pragma unroll 8
            for (int i = 0; i < n; ++i) yv += __shfl_sync(0xFFFFFFFFu, o, i);
        }
        if (lane == 0) {
            s_red[warp] = yv;
            s_red[16 + warp] = bf16_bits_to_float(s_x[d * 16 + warp]) + round_as(yv, p.out_dtype);
        }
        __syncthreads();
        static_assert(kStateCopies == 8, "a copy per four lanes");
        if (warp == 0) {
            if (p.x_next != nullptr)
                st_relaxed16(p.vx + (size_t)(lane / 4) * H + d * 16 + lane % 4 * 4, reinterpret_cast<const uint4*>(s_red + 16)[lane % 4]);
        } else if (warp == 1 && lane < 16) {
            const float v = s_red[lane];
            const int row = d * 16 + lane;
            if (p.out_dtype == EDG_F32) store_out<float>(static_cast<float*>(p.y), row, v);
            else if (p.out_dtype == EDG_F16) store_out<__half>(static_cast<__half*>(p.y), row, v);
            else store_out<bf16_t>(static_cast<bf16_t*>(p.y), row, v);
        }
        __syncthreads();
    };
    // the caller's x_next (one CTA without expert work; the next link of the chain does not wait for it)
    auto finish_state = [&]() {
        const bool on = tid * 4 < H;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        bool got = !on;
        for (uint32_t it = 0; !got; ++it) {
            const uint4 w = ld_relaxed16(p.vx + (size_t)(cta % kStateCopies) * H + 4 * tid);
            got = there(w) || late(it);
            v = make_float4(__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w));
            if (!got) __nanosleep(32);
        }
        __syncthreads();
        const float inv = inv_rms(s_red, v, on, H, p.eps);
        if (on) {
            bf16_t* xn = reinterpret_cast<bf16_t*>(p.x_next) + 4 * tid;
            store_out<bf16_t>(xn, 0, v.x * inv); store_out<bf16_t>(xn, 1, v.y * inv);
            store_out<bf16_t>(xn, 2, v.z * inv); store_out<bf16_t>(xn, 3, v.w * inv);
        }
        __syncthreads();
    };
    // the routing of the next step, by one warp, as soon as all logits are there
    auto route = [&]() {
        if (warp == 0) {
            float* work = reinterpret_cast<float*>(un);                  // [E], and 256 bytes for the winners
            float* kept = work + p.E + 64;                               // [E] (selecting may overwrite the others)
            float* slot = p.logits_ws + (size_t)max(p.flag_out, 0) * (p.E + kPairWords);
            unsigned long long* pr = reinterpret_cast<unsigned long long*>(slot + p.E) + lane;
            unsigned long long was = ~0ull;
            if (p.flag_out >= 0 && lane < p.K) was = ld_relaxed_gpu_u64(pr);
#pragma unroll 1
            for (int i0 = 0; i0 < p.E; i0 += 256) {          // 8 independent loads per lane and pass
                uint32_t v[8];
                bool got = false;
                for (uint32_t it = 0; !got; ++it) {
                    bool all = true;
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int i = i0 + u * 32 + lane;
                        v[u] = i < p.E ? ld_relaxed_gpu_u32(hx + p.lx_off + i) : 0u;
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) all = all && v[u] != kNotYet;
                    got = __all_sync(0xFFFFFFFFu, all) || late(it);
                }
                // the step that last read this slot of the ring has reset it
                for (uint32_t it = 0; was != ~0ull && it < kSpinLimit; ++it) was = ld_relaxed_gpu_u64(pr);
                if (was != ~0ull) atomicExch(p.status, EDG_E_TIMEOUT);
                __syncwarp();
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (i0 + u * 32 + lane < p.E) work[i0 + u * 32 + lane] = kept[i0 + u * 32 + lane] = __uint_as_float(v[u]);
            }
            emit_routing<false>(p, work, lane, p.flag_out >= 0 ? pr : nullptr);
            // The logits move on into the ring slot and to the caller.  The next step may be under way with that routing by now: it
            // resets the slot only when this kernel has ended.
#pragma unroll 4
            for (int i = lane; i < p.E; i += 32) {
                if (p.flag_out >= 0) st_relaxed_gpu_u32(slot + i, __float_as_uint(kept[i]));
                st_relaxed_gpu_u32(hx + p.lx_off + i, kNotYet);
                if (p.logits_next != nullptr) p.logits_next[i] = kept[i];
            }
        }
        __syncthreads();
    };
    // A CTA's own units (its rows, or the routing: n_dn + 1, and the caller's x_next: n_dn); then, if it is the one that started last,
    // what others have left to it.  A bit is claimed by an atomic: by the last starter, or by the one that left it, if it finds
    // afterwards that the last one has started -- then nothing stands in the way of waiting any more.
    int unit = has_dn ? cta : (cta == p.cta_route ? p.n_dn + 1 : (cta == p.cta_state ? p.n_dn : -1));
    int then = cta == p.cta_route && cta == p.cta_state ? p.n_dn : -1;
    if (has_dn && open) {                                                // (by far the usual case; the loop is code that is hardly ever fetched)
        down_unit(cta, std::true_type{});
        unit = -1;
    }
#pragma unroll 1
    for (;;) {
        if (unit >= 0 && !open) {
            if (tid == 0) {
                const uint32_t bit = 1u << (unit & 31);
                atomicOr(p.defer + (unit >> 5), bit);
                __threadfence();
                s_misc[3] = all_ready() ? 1 : 0;
                s_misc[2] = s_misc[3] && (atomicAnd(p.defer + (unit >> 5), ~bit) & bit) ? 1 : 0;
            }
            __syncthreads();
            if (!s_misc[2]) unit = -1;
            open = s_misc[3] != 0;
            __syncthreads();
        }
        if (unit >= 0) {
            if (unit < p.n_dn) down_unit(unit, std::false_type{});
            else if (unit == p.n_dn) finish_state();
            else route();
        }
        if (then >= 0) { unit = then; then = -1; continue; }
        if (!s_misc[1]) break;                                           // (uniform: written before the first barrier)
        if (warp == 0) {                                                 // the words at once: a trip each would hold the end of the step up
            __threadfence();
            int next = -1;
            for (;;) {
                const uint32_t left = lane < kStepDeferWords ? ld_relaxed_gpu_u32(p.defer + lane) : 0u;
                const unsigned any = __ballot_sync(0xFFFFFFFFu, left != 0);
                if (any == 0) break;
                const uint32_t bit = left & (0u - left);
                if (lane == __ffs(any) - 1 && (atomicAnd(p.defer + lane, ~bit) & bit)) next = lane * 32 + __ffs(bit) - 1;
                next = __shfl_sync(0xFFFFFFFFu, next, __ffs(any) - 1);
                if (next >= 0) break;
            }
            if (lane == 0) s_misc[2] = next;
        }
        __syncthreads();
        unit = s_misc[2];
        __syncthreads();
        if (unit < 0) break;
    }
    // ---- independent steps complete in order, too, and for the reason given below: none meets the step four before it in their buffer
    if (p.run == 2) pdl_wait_prior_grid();
    // ---- a link of a chain: the last CTA to have read the routing resets its ring slot; kernels of a chain complete in order
    if (p.flag_in >= 0) {
        // No CTA leaves before the kernel before this one has: the CTAs of the next one but one take over from that kernel, one on
        // every SM, before an SM can offer them two places.  What that kernel still had to write into the slot is there, too.
        pdl_wait_prior_grid();
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            s_misc[2] = (atomicAdd(&p.done[p.flag_in], 1) == (int)gridDim.x - 1) ? 1 : 0;
        }
        __syncthreads();
        if (s_misc[2]) {
            if (tid == 0) p.done[p.flag_in] = 0;
            float* slot = p.logits_ws + (size_t)p.flag_in * (p.E + kPairWords);
            // (the routing pairs behind the logits first: whoever finds a logit reset finds them reset too)
            for (int i = tid; i < kPairWords; i += TThreads) st_relaxed_gpu_u32(slot + p.E + i, kNotYet);
            __threadfence();
            __syncthreads();
            for (int i = tid; i < p.E; i += TThreads) st_relaxed_gpu_u32(slot + i, kNotYet);
        }
    }
}

StepSmem step_smem(const edg_layer_desc& d, int Kt, int rmax) {
    StepSmem S;
    const uint32_t NCK = d.H / 512, TG = d.I / 256, NT = 2 * TG, RG = 16 * TG, sets = (d.n_adapters == 1 ? 1 : d.K) + 1;
    const uint32_t hw = Kt * d.I, items = Kt * 4;
    auto up16 = [](uint32_t v) { return (v + 15) / 16 * 16; };
    S.h = 0;
    S.hb = up16(hw / 32 * 36 * 4);                                       // (blocks of 32 or more values, four words of padding each)
    S.hsum = S.hb + hw * 4;
    S.hbias = up16(S.hsum + hw / 32 * 4);
    S.part = up16(S.hbias + hw / 32 * 4);
    S.udi = up16(S.part + items * 17 * 4);
    uint32_t un = up16(S.udi + items * (rmax + 1) * 4);
    auto at_least = [&](uint32_t v) { if (un < v) un = up16(v); };
    at_least(NT * NCK * TW * 256);
    if (d.pre_dtype == EDG_F16) at_least(16u * (d.H * 2 + 16));          // a tile of the head
    at_least((uint32_t)d.E * 8 + 256);                                   // the logits, for the routing
    S.un = 0;
    uint32_t o = un;
    S.sz_tile = d.H / d.group * 64;
    S.sz = o;        o += NT * S.sz_tile;
    S.xb = o;        o += d.H * 2;
    S.x = o;         o += d.H * 2;
    S.xsum = o;      o += d.H / 32 * 4;
    S.xbias = o;     o += d.H / 32 * 4;
    S.bgu = o;       o += 2 * RG * rmax * 2;
    S.ad = o;        o += rmax * RG * 2;
    S.bd = o;        o += sets * 16 * rmax * 2;
    S.u4 = o;        o += 4 * 2 * kStepMaxRank * 4;
    S.uf = o;        o += 2 * kStepMaxRank * 4;
    S.hl = o;        o += 32 * 4;
    S.sel = o;       o += 64 * 4;
    S.red = o;       o += 64 * 4;
    S.bar = o;       o += 16;
    S.total = o;
    return S;
}

constexpr size_t kStepSmemLimit = 112 * 1024, kStepSmemLone = 120 * 1024;      // two CTAs per SM, one

template <int NCK, int DCH, int CPB, bool EX>
cudaError_t launch_step(const StepParams& p, int grid, cudaStream_t st) {
    auto kern = step_kernel<NCK, DCH, CPB, EX>;
    static OncePerDevice once;
    const cudaError_t e = once([&] {
        const cudaError_t s = allow_smem(kStepSmemLone, kern);
        return s != cudaSuccess ? s : cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(TThreads, 1, 1);
    // A step that does not start a chain asks for more than half an SM: with two such launches in flight, the CTAs of one that find an
    // SM free twice would share it (30 SMs of 148 did, once started so: 17.4 us a step instead of 14.4; without the
    // programmatic launch, 17.3).
    cfg.dynamicSmemBytes = p.flag_in < 0 && p.x_next == nullptr && p.run == 0 && grid <= sm_count() ? max(p.S.total, (uint32_t)kStepSmemLone) : p.S.total;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p);
}

template <int NCK, int DCH>
cudaError_t launch_shape(const StepParams& p, int grid, cudaStream_t st) {
    const bool exact = p.x_next == nullptr;
    if (p.group >= 64) return exact ? launch_step<NCK, DCH, 2, true>(p, grid, st) : launch_step<NCK, DCH, 2, false>(p, grid, st);
    return exact ? launch_step<NCK, DCH, 1, true>(p, grid, st) : launch_step<NCK, DCH, 1, false>(p, grid, st);
}

}  // namespace

bool step_supported(const edg_layer_desc& d, bool shared) {
    if (!fused_supported(d) || d.K > kStepMaxK || d.rank > kStepMaxRank) return false;
    return step_smem(d, d.K + (shared ? 1 : 0), d.rank).total <= kStepSmemLimit;
}

static size_t step_copy_words(const edg_layer_desc& d) { return ((size_t)(d.K + 1) * d.I + (size_t)16 * (d.K + 1) * d.rank + 63) / 64 * 64; }
size_t step_exchange_words(const edg_layer_desc& d) {
    const size_t sets = (d.n_adapters == 1 ? 1 : d.K) + 1;               // h, A_down h, A x, logits
    return kHCopies * step_copy_words(d) + (sets * 8 * d.rank + d.E + 63) / 64 * 64;
}
size_t step_region_words(const edg_layer_desc& d) { return kStepBufs * (step_exchange_words(d) + (size_t)kStateCopies * d.H); }

int32_t run_step(const edg_layer_desc* d, const void* slot_pool, const int32_t* slots, const int32_t* table, const int32_t* experts,
                 const float* gates, const void* x, const edg_lora* lora, void* y, const void* W_pre, int32_t* inds_next, float* gates_next,
                 float* logits_next, void* workspace, int flag_in, int flag_out, int pos, cudaStream_t st, const FusedExtras& ex) {
    StepParams p{};
    p.pool = static_cast<const uint8_t*>(slot_pool);
    p.slots = slots; p.table = table; p.experts = experts; p.gates = gates;
    p.x = static_cast<const uint16_t*>(x);
    const bool has_lora = lora != nullptr && d->rank > 0;
    if (has_lora) p.lora = *lora;
    p.rank = has_lora ? d->rank : 0;
    p.K = d->K; p.Kt = d->K;
    if (ex.shared_rec != nullptr) {
        p.shared_rec = static_cast<const uint8_t*>(ex.shared_rec);
        p.Kt = d->K + 1;
        if (ex.shared_lora != nullptr && d->rank > 0) { p.shared_lora = *ex.shared_lora; p.rank_shared = d->rank; }
    }
    p.rmax = p.rank > p.rank_shared ? p.rank : p.rank_shared;
    p.y = y;
    const WorkspaceLayout W = workspace_layout(*d, 1);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    p.status = reinterpret_cast<int32_t*>(ws + W.ctrl);
    p.done = reinterpret_cast<int32_t*>(ws + W.ctrl + kCtrlDone);
    p.logits_ws = reinterpret_cast<float*>(ws + W.logits);
    p.W_pre = W_pre; p.inds_next = inds_next; p.gates_next = gates_next; p.logits_next = logits_next; p.inds_mirror = ex.inds_mirror;
    p.x_next = static_cast<uint16_t*>(ex.x_next);
    p.eps = ex.eps;
    const int buf = pos % kStepBufs, before = (pos + kStepBufs - 1) % kStepBufs;
    const size_t hx_words = step_exchange_words(*d);
    p.starts = reinterpret_cast<uint32_t*>(ws + W.ctrl + kCtrlStarts);
    p.ready = p.starts + 16;
    p.defer = reinterpret_cast<uint32_t*>(ws + W.ctrl + kCtrlDefer) + buf * kStepDeferWords;
    float* region = reinterpret_cast<float*>(ws + W.step_x);
    p.hx = region + buf * hx_words;
    p.vx = region + kStepBufs * hx_words + (size_t)buf * kStateCopies * d->H;
    p.vx_in = region + kStepBufs * hx_words + (size_t)before * kStateCopies * d->H;
    p.ud_off = (uint32_t)(d->K + 1) * d->I;
    p.hc_words = (uint32_t)step_copy_words(*d);
    p.ux_off = kHCopies * p.hc_words;
    p.lx_off = p.ux_off + ((d->n_adapters == 1 ? 1u : (uint32_t)d->K) + 1u) * 8u * d->rank;
    p.I = d->I; p.E = d->E; p.group = d->group;
    while ((1 << p.gshift) < d->group) ++p.gshift;
    p.n_adapters = d->n_adapters; p.n_slots = d->n_slots; p.pre_dtype = d->pre_dtype; p.out_dtype = d->out_dtype;
    p.sigma = d->lora_scale;
    p.L = record_layout(d->H, d->I, d->group);
    p.n_gu = 16 * p.Kt; p.n_dn = d->H / 16;
    p.n_exp = p.n_gu > p.n_dn ? p.n_gu : p.n_dn;
    p.head_tile = d->pre_dtype == EDG_F16 && d->E % 16 == 0 ? 16 : 4;
    p.n_head = W_pre != nullptr ? (d->E + p.head_tile - 1) / p.head_tile : 0;
    // One CTA per SM when they suffice: two launches of a chain then sit side by side on every SM, and no SM has two CTAs of the
    // same launch (which held a step up by 5 us of 15).  The head's tiles share the CTAs that the experts leave.
    const int n_sm = sm_count(), spare = n_sm - p.n_exp;
    p.n_headc = min(p.n_head, spare > 2 ? spare - 2 : 16);               // (two more for the routing and the caller's x_next)
    const int extra = max(p.n_headc, p.x_next != nullptr ? 1 : 0);       // (somebody has to write x_next)
    const int grid = max(n_sm, p.n_exp + extra), idle = p.n_exp + p.n_headc;
    p.cta_route = W_pre == nullptr ? -1 : (idle < grid ? idle : idle - 1);
    p.cta_state = p.x_next == nullptr ? -1 : (W_pre == nullptr ? p.n_exp : (idle + 1 < grid ? idle + 1 : p.n_exp));
    p.flag_in = flag_in; p.flag_out = W_pre != nullptr ? flag_out : -1;
    p.run = flag_in < 0 && ex.x_next == nullptr ? ex.run : 0;
    p.dep = flag_in >= 0 && ex.dep_wait >= 0;
    p.S = step_smem(*d, p.Kt, p.rmax);
    const cudaError_t e = d->H == 2048 ? (d->I == 512 ? launch_shape<4, 4>(p, grid, st) : launch_shape<4, 2>(p, grid, st))
                                       : (d->I == 512 ? launch_shape<2, 4>(p, grid, st) : launch_shape<2, 2>(p, grid, st));
    EDG_CUDA_TRY(e);
    return EDG_OK;
}

}  // namespace edg
