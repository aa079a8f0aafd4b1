// a1 + a2: prerouter head logits, softmax, top-k and renormalised gate weights
// (Sec. 3.2 "Head" linear path; Appendix A softmax-topk).
//
// One thread-block cluster per head: the E rows of the head are split over the CTAs of the
// cluster, every CTA writes its logits straight into the leader CTA's shared memory
// (distributed shared memory; a first arrival says that they all run), and after one cluster barrier a single warp of the leader does
// softmax + top-k with warp shuffles.  No global scratch, no atomics, one launch.
//
// All kernels of this file are launched as programmatic dependents: a call's launch is under way while the kernel before it
// ends (4096 rows of sigmoid-group routing, call after call, 8.2 -> 5.8 us; 40 full heads 39.0 -> 37.2).  Every thread waits before it
// reads or writes global memory.  None lets the kernel behind it come before it has ended itself: a link of a chain does not wait for
// what was queued before it, and may write what these kernels read or write (let go at once, the two took 6.3 and 37.1 us).
#include <cooperative_groups.h>
#include <math_constants.h>

#include "edg_common.cuh"
#include "edg_mma.cuh"
#include "edg_head.cuh"

namespace cg = cooperative_groups;

namespace edg {

constexpr int kPreCluster = 8;      // CTAs per head (portable cluster size)
constexpr int kPreWarps = 8;

struct PreParams {
    const void* W;          // [n_heads][E][H]
    const uint16_t* s;      // [n_heads][H] bf16
    int32_t* inds;          // [n_heads][K]
    float* gates;           // [n_heads][K]
    float* logits;          // [n_heads][E] or null
    int H, E, K;
    int shared_head;        // 1: every state uses head 0 (batched tokens of one layer)
    int32_t* mirror;        // [n_heads][K] in mapped pinned host memory, or null
};

template <typename WT> struct RowDot;

// fp16 head: 8 weights (16 bytes) per lane per step
template <> struct RowDot<__half> {
    static __device__ __forceinline__ float partial(const void* W, size_t row, const float* sx, int H, int lane) {
        const uint4* wp = reinterpret_cast<const uint4*>(static_cast<const __half*>(W) + row * H);
        float acc = 0.f;
#pragma unroll 8
        for (int c = lane; c < H / 8; c += 32) {
            const uint4 w = ld_stream16(wp + c);
            const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&w.x));
            const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&w.y));
            const float2 d = __half22float2(*reinterpret_cast<const __half2*>(&w.z));
            const float2 e = __half22float2(*reinterpret_cast<const __half2*>(&w.w));
            const float* x = sx + c * 8;
            acc = fmaf(a.x, x[0], acc); acc = fmaf(a.y, x[1], acc);
            acc = fmaf(b.x, x[2], acc); acc = fmaf(b.y, x[3], acc);
            acc = fmaf(d.x, x[4], acc); acc = fmaf(d.y, x[5], acc);
            acc = fmaf(e.x, x[6], acc); acc = fmaf(e.y, x[7], acc);
        }
        return acc;
    }
    static __device__ __forceinline__ float run(const void* W, size_t row, const float* sx, int H, int lane) {
        return warp_sum(partial(W, row, sx, H, lane));
    }
};

// fp32 head: 4 weights (16 bytes) per lane per step
template <> struct RowDot<float> {
    static __device__ __forceinline__ float partial(const void* W, size_t row, const float* sx, int H, int lane) {
        const uint4* wp = reinterpret_cast<const uint4*>(static_cast<const float*>(W) + row * H);
        float acc = 0.f;
#pragma unroll 4
        for (int c = lane; c < H / 4; c += 32) {
            const uint4 w = ld_stream16(wp + c);
            const float* x = sx + c * 4;
            acc = fmaf(__uint_as_float(w.x), x[0], acc); acc = fmaf(__uint_as_float(w.y), x[1], acc);
            acc = fmaf(__uint_as_float(w.z), x[2], acc); acc = fmaf(__uint_as_float(w.w), x[3], acc);
        }
        return acc;
    }
    static __device__ __forceinline__ float run(const void* W, size_t row, const float* sx, int H, int lane) {
        return warp_sum(partial(W, row, sx, H, lane));
    }
};

template <typename WT>
__global__ void __launch_bounds__(kPreWarps * 32) prerouter_kernel(PreParams p) {
    cluster_arrive_relaxed();
    cg::cluster_group cluster = cg::this_cluster();
    const int crank = (int)cluster.block_rank();
    const int csize = (int)cluster.num_blocks();
    const int head = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    extern __shared__ float smem[];
    float* s_logits = smem;             // [E]   (the leader's copy collects every CTA's rows)
    float* s_x = smem + p.E;            // [H]   hidden state widened to fp32

    pdl_wait_prior_grid();
    const uint16_t* sv = p.s + (size_t)head * p.H;
    for (int i = threadIdx.x; i < p.H; i += blockDim.x) s_x[i] = bf16_bits_to_float(sv[i]);
    __syncthreads();
    cluster_wait();                     // every CTA of the cluster runs: the leader's shared memory may be written

    float* leader = cluster.map_shared_rank(s_logits, 0);
    const int per = (p.E + csize - 1) / csize;
    const int e0 = crank * per, e1 = min(p.E, e0 + per);
    const size_t wbase = p.shared_head ? 0 : (size_t)head * p.E;
    for (int e = e0 + warp; e < e1; e += kPreWarps) {
        const float l = RowDot<WT>::run(p.W, wbase + e, s_x, p.H, lane);
        if (lane == 0) leader[e] = l;
    }
    cluster.sync();                     // every CTA's logits have landed in the leader
    if (crank != 0) return;

    if (p.logits != nullptr)
        for (int e = threadIdx.x; e < p.E; e += blockDim.x) p.logits[(size_t)head * p.E + e] = s_logits[e];
    __syncthreads();
    if (warp == 0) {
        warp_softmax_topk(s_logits, p.E, p.K, lane, p.inds + (size_t)head * p.K, p.gates + (size_t)head * p.K);
        mirror_inds(p.mirror != nullptr ? p.mirror + (size_t)head * p.K : nullptr, p.inds + (size_t)head * p.K, p.K, lane);
    }
}

// One head, T hidden states (batched decode of one layer): a cluster handles kTokBlock tokens, so
// a row of the head is read once per token block instead of once per token.  CTA c of the cluster
// computes its share of the E rows for all tokens of the block (one warp per row, the tokens' states
// in shared memory as fp32), writes the logits into the leader's shared memory, and after the cluster
// barrier warp w of the leader does softmax + top-k for token w of the block.
constexpr int kTokBlock = 8;

template <typename WT>
__global__ void __launch_bounds__(kPreWarps * 32) prerouter_tokens_kernel(PreParams p, int T) {
    cluster_arrive_relaxed();
    cg::cluster_group cluster = cg::this_cluster();
    const int crank = (int)cluster.block_rank();
    const int csize = (int)cluster.num_blocks();
    const int t0 = blockIdx.y * kTokBlock;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    extern __shared__ float smem[];
    float* s_logits = smem;                         // [kTokBlock][E]  (the leader's copy collects every CTA's rows)
    float* s_x = smem + kTokBlock * p.E;            // [kTokBlock][H]  hidden states widened to fp32
    pdl_wait_prior_grid();
    for (int tt = 0; tt < kTokBlock; ++tt) {
        const int t = t0 + tt;
        for (int i = threadIdx.x; i < p.H; i += blockDim.x)
            s_x[tt * p.H + i] = t < T ? bf16_bits_to_float(p.s[(size_t)t * p.H + i]) : 0.f;
    }
    __syncthreads();
    cluster_wait();                     // every CTA of the cluster runs: the leader's shared memory may be written

    float* leader = cluster.map_shared_rank(s_logits, 0);
    const int per = (p.E + csize - 1) / csize;
    const int e0 = crank * per, e1 = min(p.E, e0 + per);
    constexpr int VPL = 16 / (int)sizeof(WT);       // weights per 16-byte load
    const int n16 = p.H / VPL;                      // 16-byte pieces of a row
    for (int e = e0 + warp; e < e1; e += kPreWarps) {
        const uint4* wp = reinterpret_cast<const uint4*>(static_cast<const WT*>(p.W) + (size_t)e * p.H);
        float acc[kTokBlock];
#pragma unroll
        for (int t = 0; t < kTokBlock; ++t) acc[t] = 0.f;
        for (int c0 = 0; c0 < n16; c0 += 8 * 32) {   // 8 independent loads per lane in flight, then the arithmetic
            uint4 wr[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = c0 + j * 32 + lane;
                wr[j] = c < n16 ? ld_stream16(wp + c) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = c0 + j * 32 + lane;
                if (c >= n16) continue;
                const uint4 w = wr[j];
                float wf[8];
                if (VPL == 8) {
                    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&w.x));
                    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&w.y));
                    const float2 d = __half22float2(*reinterpret_cast<const __half2*>(&w.z));
                    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w.w));
                    wf[0] = a.x; wf[1] = a.y; wf[2] = b.x; wf[3] = b.y; wf[4] = d.x; wf[5] = d.y; wf[6] = f.x; wf[7] = f.y;
                } else {
                    wf[0] = __uint_as_float(w.x); wf[1] = __uint_as_float(w.y); wf[2] = __uint_as_float(w.z); wf[3] = __uint_as_float(w.w);
                    wf[4] = wf[5] = wf[6] = wf[7] = 0.f;
                }
#pragma unroll
                for (int t = 0; t < kTokBlock; ++t) {
                    const float* x = s_x + t * p.H + c * VPL;
                    const float4 x0 = *reinterpret_cast<const float4*>(x);
                    float a = acc[t];
                    a = fmaf(wf[0], x0.x, a); a = fmaf(wf[1], x0.y, a); a = fmaf(wf[2], x0.z, a); a = fmaf(wf[3], x0.w, a);
                    if (VPL == 8) {
                        const float4 x1 = *reinterpret_cast<const float4*>(x + 4);
                        a = fmaf(wf[4], x1.x, a); a = fmaf(wf[5], x1.y, a); a = fmaf(wf[6], x1.z, a); a = fmaf(wf[7], x1.w, a);
                    }
                    acc[t] = a;
                }
            }
        }
#pragma unroll
        for (int t = 0; t < kTokBlock; ++t) {
            const float l = warp_sum(acc[t]);
            if (lane == 0) leader[t * p.E + e] = l;
        }
    }
    cluster.sync();                     // every CTA's logits have landed in the leader
    if (crank != 0) return;

    const int t = t0 + warp;            // kPreWarps == kTokBlock: warp w finishes token w of the block
    if (warp < kTokBlock && t < T) {
        float* row = s_logits + warp * p.E;
        if (p.logits != nullptr)
            for (int e = lane; e < p.E; e += 32) p.logits[(size_t)t * p.E + e] = row[e];
        __syncwarp();
        warp_softmax_topk(row, p.E, p.K, lane, p.inds + (size_t)t * p.K, p.gates + (size_t)t * p.K);
    }
}

// The same for an fp16 head on the tensor cores: the block's 8 tokens are the 8 columns of an
// m16n8k16 tile, 16 rows of the head its rows.  A CTA takes its share of the rows two tiles at a
// time; warp w multiplies K slice w of both.  Operands are fetched 16 bytes at a time: lane (g, t4)
// reads k = 8 t4 .. 8 t4 + 7 of every 32-k block, of head rows g and g + 8 (straight from memory) and
// of token g (fp16 in shared memory, rows padded by 64 bytes against bank conflicts), and feeds words
// 0, 1 of each to one MMA and words 2, 3 to a second one -- a permutation of k that A and B share, so
// the dot products are unchanged.  All loads of a warp's slice are issued before the first MMA (one
// trip to memory); the slices are summed through shared memory, and the logits go to the leader as
// above.  fp16 of a bf16 state is exact in the normal range; products are exact in fp32 and summed
// in fp32.
constexpr int kMmaHeadKs = 256;        // k per warp and pass: 8 blocks of 32
__global__ void __launch_bounds__(kPreWarps * 32) prerouter_tokens_mma_kernel(PreParams p, int T) {
    cluster_arrive_relaxed();
    cg::cluster_group cluster = cg::this_cluster();
    const int crank = (int)cluster.block_rank();
    const int csize = (int)cluster.num_blocks();
    const int t0 = blockIdx.y * kTokBlock;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t4 = lane & 3;
    extern __shared__ float smem[];
    float* s_logits = smem;                                             // [kTokBlock][E]
    float* s_red = smem + kTokBlock * p.E;                              // [kPreWarps][2 x 16 x 8] partial tiles
    const int xs = p.H * 2 + 64;                                        // bytes per token row
    uint8_t* s_xh = reinterpret_cast<uint8_t*>(s_red + kPreWarps * 256);    // [kTokBlock][H + 32] fp16
    const __half* W = static_cast<const __half*>(p.W);
    const int per = p.E / csize;                                        // rows of this CTA: a multiple of 16
    const int ksl = p.H / kPreWarps;                                    // k per warp: a multiple of 32

    // the head rows of the first pass are on their way while the tokens' states are converted
    uint4 a[2][kMmaHeadKs / 32][2];
    auto load_a = [&](int r0, int k0, bool two) {
#pragma unroll
        for (int tile = 0; tile < 2; ++tile) {
            const __half* w = W + (size_t)(r0 + (two ? 16 * tile : 0) + g) * p.H + warp * ksl + k0 + 8 * t4;
#pragma unroll
            for (int j = 0; j < kMmaHeadKs / 32; ++j) {
                const bool on = k0 + 32 * j < ksl;
                a[tile][j][0] = on ? ld_stream16(w + 32 * j) : make_uint4(0, 0, 0, 0);
                a[tile][j][1] = on ? ld_stream16(w + (size_t)8 * p.H + 32 * j) : make_uint4(0, 0, 0, 0);
            }
        }
    };
    pdl_wait_prior_grid();
    const int r_first = crank * per;
    load_a(r_first, 0, r_first + 16 < (crank + 1) * per);
    for (int i = threadIdx.x; i < kTokBlock * (p.H / 8); i += blockDim.x) {
        const int tt = i / (p.H / 8), c = i % (p.H / 8), t = t0 + tt;
        uint4 o = make_uint4(0, 0, 0, 0);
        if (t < T) {
            const uint4 v = *reinterpret_cast<const uint4*>(p.s + (size_t)t * p.H + c * 8);
            o.x = h2_as_u32(__floats2half2_rn(bf16_lo(v.x), bf16_hi(v.x)));
            o.y = h2_as_u32(__floats2half2_rn(bf16_lo(v.y), bf16_hi(v.y)));
            o.z = h2_as_u32(__floats2half2_rn(bf16_lo(v.z), bf16_hi(v.z)));
            o.w = h2_as_u32(__floats2half2_rn(bf16_lo(v.w), bf16_hi(v.w)));
        }
        *reinterpret_cast<uint4*>(s_xh + tt * xs + c * 16) = o;
    }
    __syncthreads();
    cluster_wait();                     // every CTA of the cluster runs: the leader's shared memory may be written

    float* leader = cluster.map_shared_rank(s_logits, 0);
    for (int r0 = r_first; r0 < (crank + 1) * per; r0 += 32) {
        const bool two = r0 + 16 < (crank + 1) * per;
        const uint8_t* xb = s_xh + g * xs + (warp * ksl + 8 * t4) * 2;
        float c[4] = {0.f, 0.f, 0.f, 0.f}, d[4] = {0.f, 0.f, 0.f, 0.f};
        for (int k0 = 0; k0 < ksl; k0 += kMmaHeadKs) {
            if (k0 > 0 || r0 > r_first) load_a(r0, k0, two);
#pragma unroll
            for (int j = 0; j < kMmaHeadKs / 32; ++j) {
                if (k0 + 32 * j < ksl) {
                    const uint4 b = *reinterpret_cast<const uint4*>(xb + (k0 + 32 * j) * 2);
                    mma16816(c, a[0][j][0].x, a[0][j][1].x, a[0][j][0].y, a[0][j][1].y, b.x, b.y);
                    mma16816(c, a[0][j][0].z, a[0][j][1].z, a[0][j][0].w, a[0][j][1].w, b.z, b.w);
                    mma16816(d, a[1][j][0].x, a[1][j][1].x, a[1][j][0].y, a[1][j][1].y, b.x, b.y);
                    mma16816(d, a[1][j][0].z, a[1][j][1].z, a[1][j][0].w, a[1][j][1].w, b.z, b.w);
                }
            }
        }
        // rows g / g + 8, tokens 2 t4 / 2 t4 + 1 of this warp's K slice, for both tiles
        float* mine = s_red + warp * 256;
        mine[g * 8 + 2 * t4] = c[0]; mine[g * 8 + 2 * t4 + 1] = c[1];
        mine[(g + 8) * 8 + 2 * t4] = c[2]; mine[(g + 8) * 8 + 2 * t4 + 1] = c[3];
        mine[128 + g * 8 + 2 * t4] = d[0]; mine[128 + g * 8 + 2 * t4 + 1] = d[1];
        mine[128 + (g + 8) * 8 + 2 * t4] = d[2]; mine[128 + (g + 8) * 8 + 2 * t4 + 1] = d[3];
        __syncthreads();
        if (threadIdx.x < 128 || two) {
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < kPreWarps; ++w) v += s_red[w * 256 + threadIdx.x];
            const int row = threadIdx.x >> 3, tok = threadIdx.x & 7;      // row 0..31 over the two tiles
            leader[tok * p.E + r0 + row] = v;
        }
        __syncthreads();
    }
    cluster.sync();                     // every CTA's logits have landed in the leader
    if (crank != 0) return;

    const int t = t0 + warp;            // kPreWarps == kTokBlock: warp w finishes token w of the block
    if (warp < kTokBlock && t < T) {
        float* row = s_logits + warp * p.E;
        if (p.logits != nullptr)
            for (int e = lane; e < p.E; e += 32) p.logits[(size_t)t * p.E + e] = row[e];
        __syncwarp();
        warp_softmax_topk(row, p.E, p.K, lane, p.inds + (size_t)t * p.K, p.gates + (size_t)t * p.K);
    }
}

// Many tokens of a head that the kernel above does not take (fp32, or rows that do not split into eight whole tiles): a CTA computes all rows
// for 16 tokens on the tensor cores, K split over its warps, and does their softmax and top-k; no cluster.  Products are exact: the
// states are bf16 as they are, an fp32 weight is the sum of three bf16 (8 of its 24 bits each), an fp16 one of two.  Every 32 k start a
// fresh accumulator, the large parts apart from the small ones, and are added in fp32.
__device__ __forceinline__ void load8(const float* w, float (&f)[8]) {
    const uint4 a = ld_stream16(w), b = ld_stream16(w + 4);
    f[0] = __uint_as_float(a.x); f[1] = __uint_as_float(a.y); f[2] = __uint_as_float(a.z); f[3] = __uint_as_float(a.w);
    f[4] = __uint_as_float(b.x); f[5] = __uint_as_float(b.y); f[6] = __uint_as_float(b.z); f[7] = __uint_as_float(b.w);
}
__device__ __forceinline__ void load8(const __half* w, float (&f)[8]) {
    const uint4 a = ld_stream16(w);
    const float2 x = __half22float2(u32_as_h2(a.x)), y = __half22float2(u32_as_h2(a.y)), z = __half22float2(u32_as_h2(a.z)), v = __half22float2(u32_as_h2(a.w));
    f[0] = x.x; f[1] = x.y; f[2] = y.x; f[3] = y.y; f[4] = z.x; f[5] = z.y; f[6] = v.x; f[7] = v.y;
}
constexpr int kRowTok = 16;
// Whether T tokens are ahead here of the clusters of FMA warps.  Both times (us a call, those : this) are flat until a form's CTAs fill the GPU a second
// time: here beyond 2368 tokens, there the sooner the longer the state is (128 tokens at H 4096, 256 at 2048, 384 at 1024); until
// then a block of 16 rows costs more here (0.6 + 1.26 H / 1024, fp16 0.5 + 0.95) and the start less.  So few rows come here
// from the start, the more of them the longer the state; others where the clusters begin their second or third round, more
// rows later.  Fitted to 2240 points (H 256 to 4096, 16 to 1008 rows, 2 to 1024 tokens), of which four are more than 2 % slower than the other form,
// by 0.3 us at most.  H 2048, fp32: 48 rows 2 tokens 11.1 : 13.6, 8 18.2 : 14.3; 64 rows 96 tokens 19.5 : 19.9, 128 21.3 : 20.1; 256 rows 320
// tokens 49 : 58, 512 86 : 59; 4096 tokens, 64 rows 218 : 30.  H 256: 64 rows 64 tokens 6.8 : 9.7, 512 12.9 : 10.
// Its error against 64 bits is below theirs (8.3e-8 and 1.4e-7 rms, 256 rows).
inline bool rows_mma_ahead(const edg_layer_desc& d, int T) {
    const bool half = d.pre_dtype == EDG_F16;
    const int n = d.E / 16, parts = n * (half ? 2 : 3);                  // blocks of 16 rows, bf16 parts of them
    int lg = 0;                                                          // log2(H / 256)
    while ((512 << lg) <= d.H) ++lg;
    if (half ? 2 * n <= 5 * lg : n <= lg) return T >= (parts <= 6 ? 2 : (parts <= 10 ? 4 : 8));
    if (T <= 8) return T >= 6 && (half ? 2 * n <= 5 * lg + 3 : n <= lg + 1);     // (one column of tokens instead of two)
    if (half) {
        if (lg == 0) return T >= (n == 1 ? 96 : (n <= 12 ? 256 : 320));
        return T >= (lg == 4 || n <= (5 << lg) / 2 + 4 ? 128 : 256);
    }
    if (lg == 4) return T >= (n <= 16 ? 128 : (n <= 24 ? 256 : (n <= 32 ? 384 : 768)));
    const int over = lg == 0 ? n + 3 : n - lg;
    return T >= (over <= 1 ? 128 : (over == 2 ? 256 : (over <= 4 ? 320 : (over <= 11 ? 384 : (over <= 20 || lg >= 2 ? 512 : 768)))));
}
inline size_t rows_mma_smem(int E, int H) { return (size_t)kRowTok * E * 4 + kPreWarps * 256 * 4 + (size_t)kRowTok * (H * 2 + 64); }

template <typename WT>
__global__ void __launch_bounds__(kPreWarps * 32) prerouter_rows_mma_kernel(PreParams p, int T) {
    constexpr int PARTS = sizeof(WT) == 4 ? 3 : 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t4 = lane & 3, t0 = blockIdx.x * kRowTok;
    extern __shared__ float smem[];
    float* s_logits = smem;                                             // [kRowTok][E]
    float* s_red = smem + kRowTok * p.E;                                // [kPreWarps][16 rows][16 tokens]
    const int xs = p.H * 2 + 64;                                        // bytes per token row (padded against bank conflicts)
    uint8_t* s_x = reinterpret_cast<uint8_t*>(s_red + kPreWarps * 256);
    pdl_wait_prior_grid();
    for (int i = threadIdx.x; i < kRowTok * (p.H / 8); i += kPreWarps * 32) {
        const int tt = i / (p.H / 8), c = i % (p.H / 8), t = t0 + tt;
        *reinterpret_cast<uint4*>(s_x + tt * xs + c * 16) = t < T ? *reinterpret_cast<const uint4*>(p.s + (size_t)t * p.H + c * 8) : make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
    const int ksl = p.H / kPreWarps;                                    // k per warp: a multiple of 32
    const uint8_t* xb = s_x + g * xs + (warp * ksl + 8 * t4) * 2;
    for (int r0 = 0; r0 < p.E; r0 += 16) {
        const WT* w = static_cast<const WT*>(p.W) + (size_t)(r0 + g) * p.H + warp * ksl + 8 * t4;
        float sum[2][4] = {};
#pragma unroll 2
        for (int k = 0; k < ksl; k += 32) {
            float lo[8], hi[8];
            load8(w + k, lo);
            load8(w + (size_t)8 * p.H + k, hi);
            uint32_t a[PARTS][4], b[PARTS][4];
            bf16_parts<PARTS>(lo, a);
            bf16_parts<PARTS>(hi, b);
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                const uint4 v = *reinterpret_cast<const uint4*>(xb + n * 8 * xs + k * 2);
                float c[2][4] = {};
#pragma unroll
                for (int q = PARTS - 1; q >= 0; --q) {
                    mma16816_bf16(c[q > 0], a[q][0], b[q][0], a[q][1], b[q][1], v.x, v.y);
                    mma16816_bf16(c[q > 0], a[q][2], b[q][2], a[q][3], b[q][3], v.z, v.w);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) sum[n][e] += c[0][e] + c[1][e];
            }
        }
        float* mine = s_red + warp * 256;                               // rows g / g + 8, tokens 8 n + 2 t4, + 1
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            mine[g * 16 + n * 8 + 2 * t4] = sum[n][0]; mine[g * 16 + n * 8 + 2 * t4 + 1] = sum[n][1];
            mine[(g + 8) * 16 + n * 8 + 2 * t4] = sum[n][2]; mine[(g + 8) * 16 + n * 8 + 2 * t4 + 1] = sum[n][3];
        }
        __syncthreads();
        double v = 0.0;
#pragma unroll
        for (int q = 0; q < kPreWarps; ++q) v += s_red[q * 256 + threadIdx.x];
        float l = (float)v;
        // The parts of an infinity, or zero parts times one, are not numbers: the warp forms such a logit from what is given, and leaves those
        // of a state that is not a number as they are.  (By one thread each, 1024 tokens of which 64 are padding that is not a number, 160
        // rows: 361 us instead of 39.)
        for (unsigned odd = __ballot_sync(0xFFFFFFFFu, !(fabsf(l) <= 3.4e38f)); odd != 0; odd &= odd - 1) {
            const int src = __ffs(odd) - 1;
            const WT* row = static_cast<const WT*>(p.W) + (size_t)(r0 + warp * 2 + (src >> 4)) * p.H;
            const uint8_t* x = s_x + (src & 15) * xs;
            bool nan = false;
            for (int k = lane * 8; k < p.H; k += 256) {
                const uint4 u = *reinterpret_cast<const uint4*>(x + k * 2);
                const uint32_t most = __vmaxu2(__vmaxu2(u.x & 0x7FFF7FFFu, u.y & 0x7FFF7FFFu), __vmaxu2(u.z & 0x7FFF7FFFu, u.w & 0x7FFF7FFFu));
                nan |= (most & 0xFFFFu) > 0x7F80u || (most >> 16) > 0x7F80u;
            }
            if (__any_sync(0xFFFFFFFFu, nan)) continue;
            float a = 0.f;
            for (int k = lane * 8; k < p.H; k += 256) {
                float f[8];
                load8(row + k, f);
                const uint4 u = *reinterpret_cast<const uint4*>(x + k * 2);
                const uint32_t xw[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) a = fmaf(f[2 * i + 1], bf16_hi(xw[i]), fmaf(f[2 * i], bf16_lo(xw[i]), a));
            }
            a = warp_sum(a);
            if (lane == src) l = a;
        }
        s_logits[(threadIdx.x & 15) * p.E + r0 + (threadIdx.x >> 4)] = l;
        __syncthreads();
    }
    for (int tt = warp; tt < kRowTok; tt += kPreWarps) {
        const int t = t0 + tt;
        if (t >= T) break;
        float* row = s_logits + tt * p.E;
        if (p.logits != nullptr)
            for (int e = lane; e < p.E; e += 32) p.logits[(size_t)t * p.E + e] = row[e];
        __syncwarp();
        warp_softmax_topk(row, p.E, p.K, lane, p.inds + (size_t)t * p.K, p.gates + (size_t)t * p.K);
    }
}

// a2 alone: one warp per row of given logits.
__global__ void __launch_bounds__(128) softmax_topk_rows_kernel(const float* logits, int T, int E, int K,
                                                                int32_t* inds, float* gates) {
    extern __shared__ float smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_wait_prior_grid();
    const int t = blockIdx.x * 4 + warp;
    if (t >= T) return;
    float* work = smem + warp * E;
    for (int e = lane; e < E; e += 32) work[e] = logits[(size_t)t * E + e];
    __syncwarp();
    warp_softmax_topk(work, E, K, lane, inds + (size_t)t * K, gates + (size_t)t * K);
}

// ---------------------------------------------------------------- the full head (Sec. 3.2 "Head")
// fc1 -> erf-gelu -> fc2 plus the linear residual path, one cluster per head.  The feature is the
// hidden state followed by two K-hot vectors (this layer's experts at this token and at the previous
// one), so fc1 is a dot product over the hidden state plus a gather of 2K columns.  Phase 1: the D
// rows of fc1 are dealt to the CTAs of the cluster, a warp per row; every activation is written
// into the shared memory of all CTAs; then the E residual rows over the hidden state, whose sums stay with the
// lanes.  Phase 2: the E rows of fc2; the logits land in the leader, which does softmax + top-k.
struct MlpParams {
    const __half* W1;       // [n_heads][D][H + 2E]
    const __half* b1;       // [n_heads][D] or null
    const __half* W2;       // [n_heads][E][D]
    const __half* b2;       // [n_heads][E] or null
    const void* Wres;       // [n_heads][E][H] (fp16 or fp32) or null
    const uint16_t* s;      // [n_heads][H] bf16
    const int32_t* cur;     // [n_heads][K]
    const int32_t* prev;    // [n_heads][K]
    int32_t* inds;          // [n_heads][K]
    float* gates;           // [n_heads][K]
    float* logits;          // [n_heads][E] or null
    int H, E, K, D;
    int32_t* mirror;        // [n_heads][K] in mapped pinned host memory, or null
};

#ifndef EDG_MLP_RING_POLLS
#define EDG_MLP_RING_POLLS kSpinLimit
#endif
static __device__ __forceinline__ bool ring_wait(uint64_t* bar, uint32_t parity, uint32_t polls) {
    for (uint32_t i = 0; i < polls; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// piece c of a row of weights times v, whose values 0-3 of every eight are in v0 and 4-7 in v1: eight fp16 weights, or four fp32
static __device__ __forceinline__ float mul_halves(const uint4& w, const float* v0, const float* v1, int c, float acc) {
    const float4 x0 = *reinterpret_cast<const float4*>(v0 + c * 4), x1 = *reinterpret_cast<const float4*>(v1 + c * 4);
    const float2 a = __half22float2(u32_as_h2(w.x)), b = __half22float2(u32_as_h2(w.y)), d = __half22float2(u32_as_h2(w.z)), e = __half22float2(u32_as_h2(w.w));
    acc = fmaf(a.x, x0.x, acc); acc = fmaf(a.y, x0.y, acc); acc = fmaf(b.x, x0.z, acc); acc = fmaf(b.y, x0.w, acc);
    acc = fmaf(d.x, x1.x, acc); acc = fmaf(d.y, x1.y, acc); acc = fmaf(e.x, x1.z, acc); acc = fmaf(e.y, x1.w, acc);
    return acc;
}
static __device__ __forceinline__ float mul_floats(const uint4& w, const float* v0, const float* v1, int c, float acc) {
    const float4 x = *reinterpret_cast<const float4*>((c & 1 ? v1 : v0) + (c >> 1) * 4);
    acc = fmaf(__uint_as_float(w.x), x.x, acc); acc = fmaf(__uint_as_float(w.y), x.y, acc);
    acc = fmaf(__uint_as_float(w.z), x.z, acc); acc = fmaf(__uint_as_float(w.w), x.w, acc);
    return acc;
}
// fc1 with its gathered columns and bias, gelu
static __device__ __forceinline__ float gelu_row(float z, __half gc, __half gq, bool biased, float bias) {
    z = warp_sum(z + __half2float(gc) + __half2float(gq));
    if (biased) z += bias;
    return 0.5f * z * (1.f + erff(z * 0.70710678118654752f));
}

constexpr int kMlpWarps = 8;            // warps per CTA of the full head
constexpr int kMlpPieces = 128;          // 16-byte pieces of a row in one slot of a warp's ring
constexpr int kMlpSlots = 3;

// What bounds the full head is its 3.9 MB of weights (H 2048, D 512, E 256): 40 heads take 24 us to stream.  Loads into registers
// left the memory idle between a warp's rows (reduction, gelu), across the cluster barrier and in front of the residual path: 64.6 us
// (2.3 TB/s).  Here every warp streams all its rows -- W1, then the residual rows, which need no activations, then W2 -- through a
// ring of three 2 KB slots of its own, refilled by bulk copies as soon as a slot is read, so the barrier finds the W2 rows in
// place; three CTAs fit an SM (100 KB in flight): 39.3 us.
// Per lane the products are summed in the order of the pieces (lane, lane + 32, ..), then over the lanes: results do not depend
// on the slots.
// There is no status word to raise when a copy does not come.  A warp that has polled for one in vain (EDG_MLP_RING_POLLS times) issues no
// more of them, and in the end the leader evaluates the head once more by itself, with plain loads in the same order.
template <typename WT>
static __device__ __noinline__ void head_with_plain_loads(const MlpParams& p, int head, const float* s_x0, const float* s_x1, float* s_a0, float* s_a1,
                                                          float* s_logits) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int hc = lane < p.K ? p.cur[(size_t)head * p.K + lane] : -1, hq = lane < p.K ? p.prev[(size_t)head * p.K + lane] : -1;
    if (hc >= p.E) hc = -1;
    if (hq >= p.E) hq = -1;
    for (int r = warp; r < p.D; r += kMlpWarps) {
        const __half* row = p.W1 + ((size_t)head * p.D + r) * (p.H + 2 * p.E);
        const __half gc = hc >= 0 ? row[p.H + hc] : __float2half(0.f), gq = hq >= 0 ? row[p.H + p.E + hq] : __float2half(0.f);
        float z = 0.f;
        for (int c = lane; c < p.H / 8; c += 32) z = mul_halves(reinterpret_cast<const uint4*>(row)[c], s_x0, s_x1, c, z);
        z = gelu_row(z, gc, gq, p.b1 != nullptr, p.b1 != nullptr ? __half2float(p.b1[(size_t)head * p.D + r]) : 0.f);
        if (lane == 0) ((r & 4) ? s_a1 : s_a0)[(r >> 3) * 4 + (r & 3)] = z;
    }
    __syncthreads();
    for (int e = warp; e < p.E; e += kMlpWarps) {
        float l = 0.f, v = 0.f;
        const uint4* row = reinterpret_cast<const uint4*>(p.W2 + ((size_t)head * p.E + e) * p.D);
        for (int c = lane; c < p.D / 8; c += 32) l = mul_halves(row[c], s_a0, s_a1, c, l);
        if (p.Wres != nullptr) {
            row = reinterpret_cast<const uint4*>(static_cast<const WT*>(p.Wres) + ((size_t)head * p.E + e) * p.H);
            for (int c = lane; c < p.H * (int)sizeof(WT) / 16; c += 32)
                v = sizeof(WT) == 2 ? mul_halves(row[c], s_x0, s_x1, c, v) : mul_floats(row[c], s_x0, s_x1, c, v);
            l += v;
        }
        l = warp_sum(l);
        if (p.b2 != nullptr) l += __half2float(p.b2[(size_t)head * p.E + e]);
        if (lane == 0) s_logits[e] = l;
    }
    __syncthreads();
}

template <typename WT>
__global__ void __launch_bounds__(kMlpWarps * 32) prerouter_mlp_kernel(const __grid_constant__ MlpParams p) {
    cluster_arrive_relaxed();
    cg::cluster_group cluster = cg::this_cluster();
    const int crank = (int)cluster.block_rank();
    const int csize = (int)cluster.num_blocks();
    const int head = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kSlotBytes = kMlpPieces * 16;
    extern __shared__ __align__(128) uint8_t smem8[];
    uint8_t* ring = smem8 + warp * kMlpSlots * kSlotBytes;                              // this warp's slots
    float* s_x0 = reinterpret_cast<float*>(smem8 + kMlpWarps * kMlpSlots * kSlotBytes); // [H/2] values 0-3 of every eight of the state,
    float* s_x1 = s_x0 + p.H / 2 + 16;  // [H/2] and values 4-7 (in other banks: fp32 rows read both at once)
    float* s_a0 = s_x1 + p.H / 2;       // [D/2] gelu(fc1) in the same way, complete in every CTA after the first cluster barrier
    float* s_a1 = s_a0 + p.D / 2;       // [D/2]
    const int perD = (p.D + csize - 1) / csize, perE = (p.E + csize - 1) / csize;
    float* s_part = s_a1 + p.D / 2;     // [perE][32] lanes' sums of the residual path
    float* s_logits = s_part + perE * 32;   // [E]   (the leader's copy collects every CTA's rows)
    float* s_win = s_logits + p.E;      // 64 words for the winners
    __shared__ __align__(8) uint64_t bars[kMlpWarps][kMlpSlots];
    __shared__ int s_lost[kMlpWarps + 1];   // per warp the first item whose copy did not come, or -1; whether there is one at all (the leader's)

    if (lane == 0) {
        s_lost[warp] = -1;
        s_lost[kMlpWarps] = 0;
        for (int i = 0; i < kMlpSlots; ++i) mbar_init(&bars[warp][i], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    // this warp's items: rows of W1, rows of the residual path, rows of W2, each in pieces of up to a slot
    const int F = p.H + 2 * p.E;
    const int r0 = crank * perD + warp, rend = min(p.D, (crank + 1) * perD), e0 = crank * perE + warp, eend = min(p.E, (crank + 1) * perE);
    const int n1 = r0 < rend ? (rend - r0 + kMlpWarps - 1) / kMlpWarps : 0, n2 = e0 < eend ? (eend - e0 + kMlpWarps - 1) / kMlpWarps : 0;
    const int p1 = p.H / 8, pr = p.Wres != nullptr ? p.H * (int)sizeof(WT) / 16 : 0, p2 = p.D / 8;       // 16-byte pieces of a row
    const int c1 = (p1 + kMlpPieces - 1) / kMlpPieces, cr = (pr + kMlpPieces - 1) / kMlpPieces, c2 = (p2 + kMlpPieces - 1) / kMlpPieces;
    int total = n1 * c1 + n2 * (cr + c2);
    uint32_t polls = EDG_MLP_RING_POLLS;                                 // 0 once a copy has not come
    // the slot after next: which row and piece the next copy fetches
    int f_kind = n1 > 0 ? 0 : (cr > 0 ? 1 : 2), f_row = 0, f_chunk = 0, fetched = 0;
    auto fetch = [&]() {                                                 // lane 0
        const uint8_t* src;
        int pieces, chunks, rows;
        if (f_kind == 0) {
            src = reinterpret_cast<const uint8_t*>(p.W1 + ((size_t)head * p.D + r0 + f_row * kMlpWarps) * F);
            pieces = p1; chunks = c1; rows = n1;
        } else if (f_kind == 1) {
            src = static_cast<const uint8_t*>(p.Wres) + ((size_t)head * p.E + e0 + f_row * kMlpWarps) * p.H * sizeof(WT);
            pieces = pr; chunks = cr; rows = n2;
        } else {
            src = reinterpret_cast<const uint8_t*>(p.W2 + ((size_t)head * p.E + e0 + f_row * kMlpWarps) * p.D);
            pieces = p2; chunks = c2; rows = n2;
        }
        const int slot = fetched % kMlpSlots, n = min(kMlpPieces, pieces - f_chunk * kMlpPieces);
        mbar_expect_tx(&bars[warp][slot], n * 16);
        bulk_g2s(ring + slot * kSlotBytes, src + (size_t)f_chunk * kSlotBytes, n * 16, &bars[warp][slot]);
        ++fetched;
        if (++f_chunk == chunks) {
            f_chunk = 0;
            if (++f_row == rows) { f_row = 0; f_kind = f_kind == 0 && cr > 0 ? 1 : 2; }
        }
    };
    pdl_wait_prior_grid();
    if (lane == 0)
        for (int i = 0; i < min(total, kMlpSlots); ++i) fetch();

    const uint16_t* sv = p.s + (size_t)head * p.H;
    for (int i = threadIdx.x; i < p.H / 8; i += blockDim.x) {
        const uint4 v = *reinterpret_cast<const uint4*>(sv + i * 8);
        *reinterpret_cast<float4*>(s_x0 + i * 4) = make_float4(bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y));
        *reinterpret_cast<float4*>(s_x1 + i * 4) = make_float4(bf16_lo(v.z), bf16_hi(v.z), bf16_lo(v.w), bf16_hi(v.w));
    }
    __syncthreads();
    cluster_wait();                     // every CTA of the cluster runs: its shared memory may be written

    int used = 0;
    // acc + this lane's share of a row (n pieces, in c chunks) times v; the row's slots go back to the ring
    auto row_dot = [&](int n, int chunks, auto piece) {
        float acc = 0.f;
        for (int ch = 0; ch < chunks; ++ch, ++used) {
            const int slot = used % kMlpSlots;
            if (!ring_wait(&bars[warp][slot], (used / kMlpSlots) & 1, polls)) {
                if (lane == 0 && s_lost[warp] < 0) { s_lost[warp] = used; total = fetched; }
                polls = 0;
            }
            const uint4* src = reinterpret_cast<const uint4*>(ring + slot * kSlotBytes);
            uint4 w[kMlpPieces / 32];
#pragma unroll
            for (int j = 0; j < kMlpPieces / 32; ++j)
                w[j] = ch * kMlpPieces + j * 32 + lane < n ? src[j * 32 + lane] : make_uint4(0, 0, 0, 0);
            __syncwarp();
            if (lane == 0 && fetched < total) fetch();
#pragma unroll
            for (int j = 0; j < kMlpPieces / 32; ++j)
                if (ch * kMlpPieces + j * 32 + lane < n) acc = piece(w[j], ch * kMlpPieces + j * 32 + lane, acc);
        }
        return acc;
    };
    auto by_state = [&](const uint4& w, int c, float acc) { return mul_halves(w, s_x0, s_x1, c, acc); };
    auto by_state32 = [&](const uint4& w, int c, float acc) { return mul_floats(w, s_x0, s_x1, c, acc); };
    auto by_gelu = [&](const uint4& w, int c, float acc) { return mul_halves(w, s_a0, s_a1, c, acc); };
    // the K-hot parts of the feature pick columns: lane k < K holds the k-th expert of either list
    int hc = -1, hq = -1;
    if (lane < p.K) {
        hc = p.cur[(size_t)head * p.K + lane];
        hq = p.prev[(size_t)head * p.K + lane];
        if (hc < 0 || hc >= p.E) hc = -1;
        if (hq < 0 || hq >= p.E) hq = -1;
    }
    for (int i = 0; i < n1; ++i) {
        const int r = r0 + i * kMlpWarps;
        // (the gathered columns are fetched while the row is on its way)
        const __half* row = p.W1 + ((size_t)head * p.D + r) * F;
        const __half gc = hc >= 0 ? row[p.H + hc] : __float2half(0.f), gq = hq >= 0 ? row[p.H + p.E + hq] : __float2half(0.f);
        const float bias = p.b1 != nullptr ? __half2float(p.b1[(size_t)head * p.D + r]) : 0.f;
        const float a = gelu_row(row_dot(p1, c1, by_state), gc, gq, p.b1 != nullptr, bias);
        if (lane < csize) *cluster.map_shared_rank(((r & 4) ? s_a1 : s_a0) + (r >> 3) * 4 + (r & 3), lane) = a;
    }
    if (cr > 0)
        for (int i = 0; i < n2; ++i) {
            float v;
            if constexpr (sizeof(WT) == 2) v = row_dot(pr, cr, by_state);
            else v = row_dot(pr, cr, by_state32);
            s_part[(warp + i * kMlpWarps) * 32 + lane] = v;
        }
    cluster.sync();                     // every CTA holds all D activations

    float* leader = cluster.map_shared_rank(s_logits, 0);
    for (int i = 0; i < n2; ++i) {
        const int e = e0 + i * kMlpWarps;
        const float bias = p.b2 != nullptr ? __half2float(p.b2[(size_t)head * p.E + e]) : 0.f;
        float l = row_dot(p2, c2, by_gelu);
        if (cr > 0) l += s_part[(warp + i * kMlpWarps) * 32 + lane];
        l = warp_sum(l);
        if (p.b2 != nullptr) l += bias;
        if (lane == 0) leader[e] = l;
    }
    if (polls == 0) *cluster.map_shared_rank(s_lost + kMlpWarps, 0) = 1;
    if (lane == 0 && s_lost[warp] >= 0) // (copies still on their way land before this CTA ends)
        for (int i = s_lost[warp]; i < fetched; ++i) ring_wait(&bars[warp][i % kMlpSlots], (i / kMlpSlots) & 1, kSpinLimit);
    cluster.sync();                     // every CTA's logits have landed in the leader
    if (crank != 0) return;
    if (s_lost[kMlpWarps] != 0) head_with_plain_loads<WT>(p, head, s_x0, s_x1, s_a0, s_a1, s_logits);

    if (warp == 0) {
        int32_t* s_i = reinterpret_cast<int32_t*>(s_win);
        int32_t* inds = p.inds + (size_t)head * p.K;
        float* gates = p.gates + (size_t)head * p.K;
        if (p.E <= 256 && topk_distinct(s_logits, p.E, p.K, lane, s_i, s_win + 32)) {
            __syncwarp();
            if (lane < p.K) { inds[lane] = s_i[lane]; gates[lane] = s_win[32 + lane]; }
            if (p.mirror != nullptr && lane < p.K)
                asm volatile("st.relaxed.sys.global.s32 [%0], %1;" ::"l"(p.mirror + (size_t)head * p.K + lane), "r"(s_i[lane]) : "memory");
        } else {
            if (p.logits != nullptr)                                     // (the general form may overwrite them)
                for (int e = lane; e < p.E; e += 32) p.logits[(size_t)head * p.E + e] = s_logits[e];
            __syncwarp();
            warp_softmax_topk(s_logits, p.E, p.K, lane, inds, gates);
            mirror_inds(p.mirror != nullptr ? p.mirror + (size_t)head * p.K : nullptr, inds, p.K, lane);
        }
    } else if (p.logits != nullptr && p.E <= 256)
        for (int e = threadIdx.x - 32; e < p.E; e += blockDim.x - 32) p.logits[(size_t)head * p.E + e] = s_logits[e];
}

// Appendix A, sigmoid-group routing when the groups divide the warp and the experts are 32 times one of the V below (the 8B tier: 128
// experts in 8 groups; the other multiples of 32 up to 1024 have no instantiation and take the form over shared memory):
// lane l holds the V = E / 32 consecutive entries from l V on, so a group is a run of lanes and everything stays in registers;
// order by (lane, entry) is order by index, so the first lane that holds a round's best key has the winner, ties included.
// The form over shared memory below spends its time on instructions too, three times as many: a call on 4096 rows of 128, one after
// the other, 11.1 us, here 8.2 with ordinary launches and 5.8 as programmatic dependents (the host's share is about as long).
// Same values in the same order as that form.
template <int V>
__global__ void __launch_bounds__(256) sigmoid_group_topk_lanes_kernel(const float* logits, const float* bias, int T, int K, int n, int keep,
                                                                       float scale, int32_t* inds, float* gates) {
    constexpr int E = 32 * V;
    const unsigned full = 0xFFFFFFFFu;
    __shared__ int s_i[8][32];
    __shared__ float s_g[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_wait_prior_grid();
    const int t = blockIdx.x * 8 + warp;
    if (t >= T) return;
    float sg[V], sel[V];
    constexpr int W = V % 4 == 0 ? 4 : (V % 2 == 0 ? 2 : 1);
    const float* src = logits + (size_t)t * E + lane * V;
#pragma unroll
    for (int u = 0; u < V; u += W) {
        if constexpr (W == 4) {
            const float4 v = *reinterpret_cast<const float4*>(src + u);
            sg[u] = v.x; sg[u + 1] = v.y; sg[u + 2] = v.z; sg[u + 3] = v.w;
        } else if constexpr (W == 2) {
            const float2 v = *reinterpret_cast<const float2*>(src + u);
            sg[u] = v.x; sg[u + 1] = v.y;
        } else sg[u] = src[u];
    }
    float m1 = -CUDART_INF_F, m2 = -CUDART_INF_F;
#pragma unroll
    for (int u = 0; u < V; ++u) {
        sg[u] = 1.f / (1.f + expf(-sg[u]));
        sel[u] = bias != nullptr ? sg[u] + bias[lane * V + u] : sg[u];
        if (sel[u] > m1) { m2 = m1; m1 = sel[u]; } else if (sel[u] > m2) m2 = sel[u];
    }
    // group scores, merged over the 32 / n lanes of a group, and the group's rank
    const int lpg = 32 / n, grp = lane / lpg;
    for (int o = 1; o < lpg; o <<= 1) {
        const float o1 = __shfl_xor_sync(full, m1, o), o2 = __shfl_xor_sync(full, m2, o);
        const float hi = fmaxf(m1, o1), lo = fminf(m1, o1);
        m2 = fmaxf(lo, fmaxf(m2, o2));
        m1 = hi;
    }
    const float gs = m1 + m2;
    int rank = 0;
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
        const float gj = __shfl_sync(full, gs, j * lpg);
        rank += (gj > gs || (gj == gs && j < grp)) ? 1 : 0;
    }
    uint32_t key[V];
    uint32_t top = 0u;
#pragma unroll
    for (int u = 0; u < V; ++u) {
        key[u] = rank < keep && sel[u] == sel[u] ? float_key(sel[u]) : 0u;
        top = max(top, key[u]);
    }
    int got = 0;
    for (; got < K; ++got) {
        const uint32_t best = __reduce_max_sync(full, top);
        if (best == 0u) break;                                   // fewer than K survivors
        const unsigned who = __ballot_sync(full, top == best);
        if (lane == __ffs(who) - 1) {
            int at = 0;
            float g = 0.f;
#pragma unroll
            for (int u = V - 1; u >= 0; --u)
                if (key[u] == best) { at = u; g = sg[u]; }
            top = 0u;
#pragma unroll
            for (int u = 0; u < V; ++u) {
                if (u == at) key[u] = 0u;
                top = max(top, key[u]);
            }
            s_i[warp][got] = lane * V + at;
            s_g[warp][got] = g;
        }
    }
    __syncwarp();
    const int myi = lane < got ? s_i[warp][lane] : 0x7FFFFFFF;
    const float myv = lane < got ? s_g[warp][lane] : 0.f;
    const float sum = warp_sum(myv);
    int pos = 0;
#pragma unroll 4
    for (int i = 0; i < K; ++i) pos += __shfl_sync(full, myi, i) < myi ? 1 : 0;
    if (lane < got) {
        inds[(size_t)t * K + pos] = myi;
        gates[(size_t)t * K + pos] = scale * myv / (sum + 1e-20f);
    }
}

// Appendix A, sigmoid-group routing, one warp per row of given logits: sigma = sigmoid(l); a group's
// score is the sum of its two largest selection scores (sigma, plus a bias when one is given); the
// best `keep` of the `n` groups survive (ties to the lower group); top-K among the survivors by
// selection score (ties to the lower index); w = scale * sigma[inds] / (sum sigma[inds] + 1e-20):
// the weights use the raw sigmoid.  Winners are written in ascending index.
__global__ void __launch_bounds__(128) sigmoid_group_topk_rows_kernel(const float* logits, const float* bias, int T, int E, int K,
                                                                      int n, int keep, float scale, int32_t* inds, float* gates) {
    extern __shared__ float smem[];
    const unsigned full = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_wait_prior_grid();
    const int t = blockIdx.x * 4 + warp;
    if (t >= T) return;
    float* sig = smem + warp * 2 * E;          // [E] raw sigmoid
    float* sel = sig + E;                      // [E] selection score; NaN = not a candidate (any more)
    for (int e = lane; e < E; e += 32) {
        const float sg = 1.f / (1.f + expf(-logits[(size_t)t * E + e]));
        sig[e] = sg;
        sel[e] = bias != nullptr ? sg + bias[e] : sg;
    }
    __syncwarp();
    // group scores.  When the groups divide the warp, 32 / n lanes share a group: each scans its part,
    // the (largest, second largest) pairs are merged by a butterfly, and every lane of the group
    // ends up with the group's score; otherwise lane g scans group g alone.
    const int per = E / n;
    float gs = -CUDART_INF_F;
    const int lpg = 32 / n;                    // lanes per group (when n divides 32)
    const bool split = (32 % n) == 0 && (per % lpg) == 0;
    if (split || lane < n) {
        const int grp = split ? lane / lpg : lane, part = split ? lane % lpg : 0, cnt = split ? per / lpg : per;
        float m1 = -CUDART_INF_F, m2 = -CUDART_INF_F;
        for (int i = 0; i < cnt; ++i) {
            const float v = sel[grp * per + part * cnt + i];
            if (v > m1) { m2 = m1; m1 = v; } else if (v > m2) m2 = v;
        }
        if (split) {
            for (int o = 1; o < lpg; o <<= 1) {
                const float o1 = __shfl_xor_sync(full, m1, o), o2 = __shfl_xor_sync(full, m2, o);
                const float hi = fmaxf(m1, o1), lo = fminf(m1, o1);
                m2 = fmaxf(lo, fmaxf(m2, o2));
                m1 = hi;
            }
        }
        gs = m1 + m2;
    }
    int rank = 0;
    const int mygrp = split ? lane / lpg : lane;
    for (int j = 0; j < n; ++j) {
        const float gj = __shfl_sync(full, gs, split ? j * lpg : j);
        rank += (gj > gs || (gj == gs && j < mygrp)) ? 1 : 0;
    }
    const unsigned alive_l = __ballot_sync(full, (split || lane < n) && rank < keep);
    // (one bit per group)
    unsigned alive = 0u;
    for (int j = 0; j < n; ++j) alive |= ((alive_l >> (split ? j * lpg : j)) & 1u) << j;
    for (int e = lane; e < E; e += 32)
        if (!((alive >> (e / per)) & 1u)) sel[e] = __int_as_float(0x7fffffff);
    __syncwarp();
    // top-K among the survivors, ties to the lower index
    float myv = 0.f;
    int myi = 0x7FFFFFFF;
    if (E <= 256) {
        warp_topk_reg<8>(sel, E, K, lane, myv, myi);
        if (lane < K && myi != 0x7FFFFFFF) myv = sig[myi];
    } else {
        // every lane keeps its best remaining candidate, the owner of a round's winner rescans
        uint32_t key;
        int idx;
        lane_best(sel, E, lane, key, idx);
        for (int j = 0; j < K; ++j) {
            const uint32_t best = __reduce_max_sync(full, idx == 0x7FFFFFFF ? 0u : key);
            const int cand = (idx != 0x7FFFFFFF && key == best) ? idx : 0x7FFFFFFF;
            const int win = (int)__reduce_min_sync(full, (unsigned)cand);
            if (win == 0x7FFFFFFF) break;                   // fewer than K survivors
            if (lane == j) { myv = sig[win]; myi = win; }
            __syncwarp();
            if (idx == win) {
                sel[win] = __int_as_float(0x7fffffff);
                lane_best(sel, E, lane, key, idx);
            }
            __syncwarp();
        }
    }
    const float sum = warp_sum((lane < K && myi != 0x7FFFFFFF) ? myv : 0.f);
    int pos = 0;
    for (int i = 0; i < K; ++i) {
        const int oi = __shfl_sync(full, myi, i);
        pos += (oi < myi) ? 1 : 0;
    }
    if (lane < K && myi != 0x7FFFFFFF) {
        inds[(size_t)t * K + pos] = myi;
        gates[(size_t)t * K + pos] = scale * myv / (sum + 1e-20f);
    }
}

int32_t run_prerouter(const edg_layer_desc* d, const void* W_pre, const void* s, int32_t n_heads,
                      int32_t* inds, float* gates, float* logits_opt, cudaStream_t st, int shared_head,
                      int32_t* mirror) {
    int32_t rc = check_desc(d);
    if (rc != EDG_OK) return rc;
    if (!W_pre || !s || !inds || !gates || n_heads < 1 || n_heads > 65535) return EDG_E_INVAL;
    if (!aligned(W_pre, 16) || !aligned(s, 16)) return EDG_E_INVAL;
    PreParams p{W_pre, static_cast<const uint16_t*>(s), inds, gates, logits_opt, d->H, d->E, d->K, shared_head, mirror};

    const bool batched = shared_head != 0 && n_heads > 1;     // one head, several tokens: a cluster per block of tokens
    const dim3 grid(kPreCluster, batched ? (n_heads + kTokBlock - 1) / kTokBlock : n_heads, 1);
    const size_t smem = (size_t)(d->E + d->H) * sizeof(float) * (batched ? kTokBlock : 1);
    auto launch = [&](auto kern, size_t bytes, auto... args) { return launch_pdl_cluster(kPreCluster, kern, grid, kPreWarps * 32, bytes, st, args...); };
    if (batched) {
        static OncePerDevice once;
        EDG_CUDA_TRY(once([] {
            return allow_smem(200 * 1024, prerouter_tokens_kernel<__half>, prerouter_tokens_kernel<float>, prerouter_tokens_mma_kernel,
                              prerouter_rows_mma_kernel<__half>, prerouter_rows_mma_kernel<float>);
        }));
        if (smem > 200 * 1024) return EDG_E_SHAPE;
        // an fp16 head whose rows and columns split into whole MMA tiles goes to the tensor cores
        if (d->pre_dtype == EDG_F16 && d->E % (16 * kPreCluster) == 0 && d->H % (32 * kPreWarps) == 0) {
            const size_t bytes = (size_t)kTokBlock * d->E * 4 + kPreWarps * 256 * 4 + (size_t)kTokBlock * (d->H * 2 + 64);
            EDG_CUDA_TRY(launch(prerouter_tokens_mma_kernel, bytes, p, (int)n_heads));
            return EDG_OK;
        }
        const size_t rows_smem = rows_mma_smem(d->E, d->H);
        if (d->E % 16 == 0 && d->H % (32 * kPreWarps) == 0 && rows_mma_ahead(*d, n_heads) && rows_smem <= 200 * 1024) {
            EDG_CUDA_TRY(launch_pdl(d->pre_dtype == EDG_F16 ? prerouter_rows_mma_kernel<__half> : prerouter_rows_mma_kernel<float>,
                                    dim3((unsigned)(n_heads + kRowTok - 1) / kRowTok), kPreWarps * 32, rows_smem, st, p, (int)n_heads));
            return EDG_OK;
        }
        if (d->pre_dtype == EDG_F16) EDG_CUDA_TRY(launch(prerouter_tokens_kernel<__half>, smem, p, (int)n_heads));
        else EDG_CUDA_TRY(launch(prerouter_tokens_kernel<float>, smem, p, (int)n_heads));
        return EDG_OK;
    }
    if (d->pre_dtype == EDG_F16) EDG_CUDA_TRY(launch(prerouter_kernel<__half>, smem, p));
    else EDG_CUDA_TRY(launch(prerouter_kernel<float>, smem, p));
    return EDG_OK;
}

}  // namespace edg

extern "C" int32_t prerouter_topk(const edg_layer_desc* desc, const void* W_pre, const void* s, int32_t n_heads,
                                  int32_t* inds, float* gates, float* logits_opt, int32_t* inds_host_mirror_opt,
                                  void* stream) {
    return edg::run_prerouter(desc, W_pre, s, n_heads, inds, gates, logits_opt, static_cast<cudaStream_t>(stream), 0,
                              inds_host_mirror_opt);
}

extern "C" int32_t prerouter_topk_tokens(const edg_layer_desc* desc, const void* W_pre, const void* s, int32_t T,
                                         int32_t* inds, float* gates, float* logits_opt, void* stream) {
    return edg::run_prerouter(desc, W_pre, s, T, inds, gates, logits_opt, static_cast<cudaStream_t>(stream), 1);
}

extern "C" int32_t softmax_topk_rows(const edg_layer_desc* desc, const float* logits, int32_t T,
                                     int32_t* inds, float* gates, void* stream) {
    int32_t rc = edg::check_desc(desc);
    if (rc != EDG_OK) return rc;
    if (!logits || !inds || !gates || T < 1) return EDG_E_INVAL;
    const size_t sm = 4 * (size_t)desc->E * sizeof(float);
    EDG_CUDA_TRY(edg::launch_pdl(edg::softmax_topk_rows_kernel, dim3((unsigned)((T + 3) / 4)), 128, sm, static_cast<cudaStream_t>(stream),
                                 logits, (int)T, desc->E, desc->K, inds, gates));
    return EDG_OK;
}

extern "C" int32_t sigmoid_group_topk_rows(const float* logits, int32_t T, int32_t E, int32_t K, int32_t n_groups,
                                           int32_t keep_groups, float scale, const float* bias_opt,
                                           int32_t* inds, float* gates, void* stream) {
    if (!logits || !inds || !gates || T < 1) return EDG_E_INVAL;
    if (E < 2 || E > 1024 || n_groups < 1 || n_groups > 32 || E % n_groups != 0 || E / n_groups < 2) return EDG_E_SHAPE;
    if (keep_groups < 1 || keep_groups > n_groups || K < 1 || K > 32 || K > keep_groups * (E / n_groups)) return EDG_E_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (32 % n_groups == 0 && E % 32 == 0 && edg::aligned(logits, 16)) {       // (E / n_groups is then a multiple of E / 32)
        void (*k)(const float*, const float*, int, int, int, int, float, int32_t*, float*) = nullptr;
        switch (E / 32) {
            case 1: k = edg::sigmoid_group_topk_lanes_kernel<1>; break;
            case 2: k = edg::sigmoid_group_topk_lanes_kernel<2>; break;
            case 3: k = edg::sigmoid_group_topk_lanes_kernel<3>; break;
            case 4: k = edg::sigmoid_group_topk_lanes_kernel<4>; break;
            case 5: k = edg::sigmoid_group_topk_lanes_kernel<5>; break;
            case 6: k = edg::sigmoid_group_topk_lanes_kernel<6>; break;
            case 8: k = edg::sigmoid_group_topk_lanes_kernel<8>; break;
            case 12: k = edg::sigmoid_group_topk_lanes_kernel<12>; break;
            case 16: k = edg::sigmoid_group_topk_lanes_kernel<16>; break;
        }
        if (k != nullptr) {
            EDG_CUDA_TRY(edg::launch_pdl(k, dim3((unsigned)((T + 7) / 8)), 256, 0, st, logits, bias_opt, (int)T, (int)K, (int)n_groups, (int)keep_groups,
                                         scale, inds, gates));
            return EDG_OK;
        }
    }
    const size_t sm = 4 * 2 * (size_t)E * sizeof(float);
    EDG_CUDA_TRY(edg::launch_pdl(edg::sigmoid_group_topk_rows_kernel, dim3((unsigned)((T + 3) / 4)), 128, sm, st, logits, bias_opt, (int)T, (int)E, (int)K,
                                 (int)n_groups, (int)keep_groups, scale, inds, gates));
    return EDG_OK;
}

extern "C" int32_t prerouter_mlp_topk(const edg_layer_desc* desc, const edg_mlp_head* head, const void* s,
                                      const int32_t* cur_inds, const int32_t* prev_inds, int32_t n_heads,
                                      int32_t* inds, float* gates, float* logits_opt, void* stream) {
    return edg::run_prerouter_mlp(desc, head, s, cur_inds, prev_inds, n_heads, inds, gates, logits_opt,
                                  static_cast<cudaStream_t>(stream), nullptr);
}

int32_t edg::run_prerouter_mlp(const edg_layer_desc* desc, const edg_mlp_head* head, const void* s,
                               const int32_t* cur_inds, const int32_t* prev_inds, int32_t n_heads,
                               int32_t* inds, float* gates, float* logits_opt, cudaStream_t stream, int32_t* mirror) {
    int32_t rc = edg::check_desc(desc);
    if (rc != EDG_OK) return rc;
    if (!head || !head->W1 || !head->W2 || !s || !cur_inds || !prev_inds || !inds || !gates || n_heads < 1 || n_heads > 65535)
        return EDG_E_INVAL;
    const int D = head->width;
    if (D < 8 || D > 4096 || D % 8 != 0 || desc->H % 8 != 0 || (desc->H + 2 * desc->E) % 8 != 0) return EDG_E_SHAPE;
    if (!edg::aligned(head->W1, 16) || !edg::aligned(head->W2, 16) || !edg::aligned(s, 16) ||
        (head->W_res && !edg::aligned(head->W_res, 16)))
        return EDG_E_INVAL;
    edg::MlpParams p{static_cast<const __half*>(head->W1), static_cast<const __half*>(head->b1),
                     static_cast<const __half*>(head->W2), static_cast<const __half*>(head->b2), head->W_res,
                     static_cast<const uint16_t*>(s), cur_inds, prev_inds, inds, gates, logits_opt,
                     desc->H, desc->E, desc->K, D, mirror};
    if ((size_t)(desc->E + desc->H + D) * sizeof(float) > 48 * 1024) return EDG_E_SHAPE;
    const int perE = (desc->E + edg::kPreCluster - 1) / edg::kPreCluster;
    const size_t smem = edg::kMlpWarps * edg::kMlpSlots * edg::kMlpPieces * 16 + (size_t)(desc->E + desc->H + 16 + D + perE * 32 + 64) * sizeof(float);
    static edg::OncePerDevice once;
    EDG_CUDA_TRY(once([] { return edg::allow_smem(200 * 1024, edg::prerouter_mlp_kernel<__half>, edg::prerouter_mlp_kernel<float>); }));
    auto launch = [&](auto kern) { return edg::launch_pdl_cluster(edg::kPreCluster, kern, dim3(edg::kPreCluster, n_heads, 1), edg::kMlpWarps * 32, smem, stream, p); };
    EDG_CUDA_TRY(desc->pre_dtype == EDG_F16 ? launch(edg::prerouter_mlp_kernel<__half>) : launch(edg::prerouter_mlp_kernel<float>));
    return EDG_OK;
}
