// a4'-a6' for several tokens (batched decode, chunks of a prompt): grouping of the (token, choice) pairs, their
// operand tiles, and ONE persistent kernel that streams the int4 weights of every routed expert once per tile and
// multiplies them with the tokens of the tile on mma.sync fragments.
//
// A call is four kernels, launched as programmatic dependents of one another:
//   group_pairs_kernel    one CTA: resolves every pair's slot, sorts the pairs by slot (stable, so a second run is
//                         bit-identical) and cuts each slot's run into tiles of up to `cap` pairs; up to 128 pairs the next
//                         kernel's CTAs do that, each for its tile
//   tile_operands_kernel  per tile: the tokens' states as fp16 B words in the order the ring stages read them, and the
//                         adapter projections sigma A_gate x, sigma A_up x (bf16 MMA, fp32 sums)
//   grouped_ffn_kernel    see below
//   sum_choices_kernel    y[t] = sum of the token's K gate-weighted rows, in the order of its choices
//
// grouped_ffn_kernel.  Bound by HBM on the union of the routed experts' records while tiles are small and by the rate
// of mma.sync when they are full.  One CTA per SM with two independent groups of eight consumer warps; each group
// has a ring of stages of its own, a producer lane that feeds it and a warp for the rank-r projections of h.  Work
// units come from a ticket counter (all gate/up units of all tiles, then all down units), so ragged tiles balance
// themselves and the weights of the first down units are on their way while the last gate/up units are computed:
//   gate/up unit: 8 row tiles (16 rows each) of gate and of up, one per warp, over all of K = H (with few tiles: 4, a warp for each
//                 of gate and of up);
//   down unit:    16 row tiles of the output, two per warp, over all of K = I.
// A stage is 128 k for every warp of a group: its codes are ONE tensor copy of 16 KB (the record's tile-major sections seen
// as an array of runs, row tiles, matrices or column slices, and slots), the (scale, zero) pairs one more (2 KB at groups
// of 64), the tokens' words one bulk copy (2 or 4 KB per 8 tokens): three issues per 20 to 34 KB, because arming a barrier or
// issuing a copy holds its lane for 50 to 100 ns whatever its size.
// No CTA-wide barrier after the start: a warp owns whole rows, so nothing is exchanged between warps but h, which
// goes through global memory in operand order; a counter per tile says when all of a tile's rows are there.  Units are handed
// out in order, so whoever waits waits for units that are already running; every wait is bounded all the same.
//
// Measured (B200, H 2048, I 512, 256 experts, top 8, groups of 64, rank 16; the whole call with its routing), against the
// kernels before it (clusters of 4 CTAs x 4 warps with sixteen copies per 36 KB, five barriers an item and
// eight launches; above 8 pairs per slot the tcgen05 path):
//   5 tokens  80 -> 62 us a layer, 64 tokens 195 -> 134 us (3.6 TB/s in the kernel), 333 tokens 580 -> 250 us;
// then, with narrow units and without the kernel that sorts where there are few pairs, 5 tokens 59 -> 46, 2 tokens 53 -> 41.
// With the arithmetic left out the 64-token kernel takes 80 of its 109 us, with the copies left out 100: what bounds it now
// is the issue rate of sixteen warps (nine instructions per eight codes) next to the memory system.  Three groups of
// eight warps (72 registers) lose more to spills than they gain (113 us).
#include <cuda.h>

#include <cmath>

#include "edg_grouped.cuh"
#include "edg_ptx.cuh"

namespace edg {
namespace {

constexpr int GGroups = 2;                     // consumer groups of a CTA
constexpr int GW = 8;                          // warps of a consumer group
constexpr int GThreads = (GGroups * GW + 2 * GGroups) * 32;
constexpr int GStageK = 128;                   // k of a stage
constexpr uint32_t GCodeBytes = 2 * GW * 1024; // codes of a stage: two 16-row runs of 128 k per warp
constexpr int GMaxStages = 6;
constexpr int GQueue = 4;                      // down units the producer may be ahead of the projection warp
constexpr uint32_t GSmemLimit = 227 * 1024;

// byte offsets in shared memory, from the start of a group's part
struct GffnSmem {
    uint32_t stage_bytes, sz0, sz_bytes, act0, h, ud, pr, info, queue, bars, group_bytes;
    int stages;
};

struct GffnParams {
    const int4* tiles;            // {slot, first position in order, pairs, adapter}
    const int32_t* n_tiles;
    const int32_t* order;         // [P] pairs sorted by slot
    const float* gates;
    int32_t* ticket;
    int32_t* done;                // [tiles] finished row tiles of h
    int32_t* status;
    const uint8_t* xq;            // [tile][cap * H * 2]
    uint8_t* hq;                  // [tile][cap * I * 4]
    const __half* u;              // [tile][2][cap][r16]
    float* o;                     // [P][H]
    edg_lora lora;
    int H, I, rank, r16, cap, gshift;
    int n1, n2, ns1, ns2;         // units per tile, stages per unit
    int sp, cps, csh;             // down: slices per stage, 32-code chunks of a stage in one slice, log2 of that
    float sigma;
    int evict_first;
    int rows1;                    // row tiles of gate and of up in a unit: 8, or 4
    GffnSmem S;
};

__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4, uint64_t* bar, uint64_t pol) {
    asm volatile("cp.async.bulk.tensor.5d.shared::cta.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3,%4,%5,%6,%7}], [%2], %8;"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "l"(pol) : "memory");
}
__device__ __forceinline__ uint64_t policy_evict_normal() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
// bounded wait, inlined: a call would spill the accumulators around it
__device__ __forceinline__ void ring_wait(uint64_t* bar, uint32_t parity, int32_t* status) {
    uint32_t i = 0;
    while (!mbar_try_wait(bar, parity))
        if (++i >= kSpinLimit) { atomicExch(status, EDG_E_TIMEOUT); break; }
}

// where a warp finds its two runs (matrices of gate/up, neighbouring row tiles of down) inside a stage
struct WarpRuns {
    uint32_t code[2], sz[2];      // first byte of each run
    uint32_t code_part, sz_part;  // from one slice of a down stage to the next
    int csh;                      // log2 of the chunks of a run in one slice (2: the whole stage)
};

// one stage: acc[m][nt] += W_m[16 rows x 128 k] . act[128 k x 8 tokens]; LO: act carries values and residuals
template <int NT, int CPB, bool LO, int NM>
__device__ __forceinline__ void mma_stage(float (&acc)[NM][NT][4], const uint8_t* st, const WarpRuns& R, const uint8_t* act, int gshift) {
    const int lane = threadIdx.x & 31, g8 = lane >> 2, t4 = lane & 3;
    const uint32_t lane_c = g8 * 16 + t4 * 4, lane_b = g8 * 64 + t4 * 16;
    constexpr int kTok = 8 * NT * 64;              // bytes of one chunk of token words
#pragma unroll NT == 1 ? 4 / CPB : 1
    for (int b = 0; b < 4 / CPB; ++b) {
        float sf[NM][2];
        __half2 mz[NM][2];
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const int i = b * CPB, part = i >> R.csh, gi = ((i - (part << R.csh)) * 32) >> gshift;
            const uint8_t* z = st + R.sz[m] + part * R.sz_part + gi * 64 + g8 * 4;
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const __half2 v = u32_as_h2(*reinterpret_cast<const uint32_t*>(z + hh * 32));
                sf[m][hh] = __low2float(v);
                mz[m][hh] = neg_zero_x(v);
            }
        }
        uint32_t a[CPB][NM][2][4];
#pragma unroll
        for (int u = 0; u < CPB; ++u) {
            const int i = b * CPB + u, part = i >> R.csh;
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                const uint8_t* w = st + R.code[m] + part * R.code_part + (i - (part << R.csh)) * 256 + lane_c;
                dequant_word_x(*reinterpret_cast<const uint32_t*>(w), mz[m][0], a[u][m][0]);
                dequant_word_x(*reinterpret_cast<const uint32_t*>(w + 128), mz[m][1], a[u][m][1]);
            }
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            float c[NM][4];
#pragma unroll
            for (int u = 0; u < CPB; ++u) {
                const uint8_t* bp = act + (LO ? 2 : 1) * (b * CPB + u) * kTok + nt * 512 + lane_b;
#pragma unroll
                for (int lo = 0; lo < (LO ? 2 : 1); ++lo) {
                    const uint4 v = *reinterpret_cast<const uint4*>(bp + lo * kTok);
#pragma unroll
                    for (int m = 0; m < NM; ++m) {
                        if (u == 0 && lo == 0) mma16816_zero(c[m], a[u][m][0][0], a[u][m][1][0], a[u][m][0][1], a[u][m][1][1], v.x, v.y);
                        else mma16816(c[m], a[u][m][0][0], a[u][m][1][0], a[u][m][0][1], a[u][m][1][1], v.x, v.y);
                    }
#pragma unroll
                    for (int m = 0; m < NM; ++m) mma16816(c[m], a[u][m][0][2], a[u][m][1][2], a[u][m][0][3], a[u][m][1][3], v.z, v.w);
                }
            }
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                fma2(acc[m][nt][0], acc[m][nt][1], sf[m][0], c[m][0], c[m][1]);
                fma2(acc[m][nt][2], acc[m][nt][3], sf[m][1], c[m][2], c[m][3]);
            }
        }
    }
}

// two neighbouring bf16 of an adapter row as an fp16 pair; entries at or beyond n are zero
__device__ __forceinline__ uint32_t bf16_pair(const uint16_t* row, int k, int n) {
    if (k + 1 < n && (n & 1) == 0) {
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(row + k));
        return h2_as_u32(__floats2half2_rn(bf16_lo(w), bf16_hi(w)));
    }
    const float a = k < n ? bf16_bits_to_float(row[k]) : 0.f, b = k + 1 < n ? bf16_bits_to_float(row[k + 1]) : 0.f;
    return h2_as_u32(__floats2half2_rn(a, b));
}
struct RingPos {
    int st;
    uint32_t phase;
    __device__ __forceinline__ void next(int stages) { if (++st == stages) { st = 0; phase ^= 1u; } }
};

struct Gffn {
    const GffnParams& p;
    uint8_t* smem;
    uint64_t *full, *empty, *q_full, *q_empty, *ud_full, *ud_empty;
    int lane, warp, g8, t4;                // warp: inside the group

    __device__ __forceinline__ uint8_t* stage(int s) const { return smem + (size_t)s * p.S.stage_bytes; }
    __device__ __forceinline__ void release(const RingPos& rp) const {
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[rp.st]);
    }
    template <int NT, int NM>
    static __device__ __forceinline__ void clear(float (&acc)[NM][NT][4]) {
#pragma unroll
        for (int m = 0; m < NM; ++m)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[m][nt][q] = 0.f;
    }
    // the MMA has seen (q - z) * 2^-9
    template <int NT, int NM>
    static __device__ __forceinline__ void unscale(float (&acc)[NM][NT][4]) {
#pragma unroll
        for (int m = 0; m < NM; ++m)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[m][nt][q] *= kUnscaleX;
    }
    // the adapter's B rows of 16 ranks as an A fragment: row g8 of the tile (at `B`) and the one eight below
    __device__ __forceinline__ void lora_rows(const uint16_t* B, int kr, uint32_t (&a)[4]) const {
        const int k0 = kr + 2 * t4, k1 = k0 + 8;
        a[0] = bf16_pair(B, k0, p.rank); a[1] = bf16_pair(B + (size_t)8 * p.rank, k0, p.rank);
        a[2] = bf16_pair(B, k1, p.rank); a[3] = bf16_pair(B + (size_t)8 * p.rank, k1, p.rank);
    }

    // ---- gate/up: this warp's row tile of both matrices; h = silu(gate) up to global in operand order
    template <int NT, int CPB>
    __device__ __forceinline__ void gate_up(int tile, int sub, int ad, RingPos& rp) {
        const int row0 = (sub * GW + warp) * 16;
        float acc[2][NT][4];
        clear(acc);
        // the adapter's operands (first 16 ranks) are asked for now and used behind the main loop, where registers allow it
        const bool lora = p.rank > 0 && row0 < p.I;
        constexpr bool ahead = NT <= 2;
        uint32_t lb[2][4], lu[2][NT][2];
        const __half* uq = p.u + (size_t)tile * 2 * p.cap * p.r16 + (size_t)g8 * p.r16 + 2 * t4;
        auto b_rows = [&](int m) { return static_cast<const uint16_t*>(m ? p.lora.B_up : p.lora.B_gate) + ((size_t)ad * p.I + row0 + g8) * p.rank; };
        auto lora_load = [&]() {
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                lora_rows(b_rows(m), 0, lb[m]);
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        lu[m][nt][q] = __ldg(reinterpret_cast<const uint32_t*>(uq + (size_t)(m * p.cap + nt * 8) * p.r16 + 8 * q));
            }
        };
        if (ahead && lora) lora_load();
        WarpRuns R;
        const uint32_t szrun = (uint32_t)(GStageK >> p.gshift) * 64;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            R.code[m] = (uint32_t)(m * GW + warp) * 1024;
            R.sz[m] = p.S.sz0 + (uint32_t)(m * GW + warp) * szrun;
        }
        R.code_part = R.sz_part = 0; R.csh = 2;
#pragma unroll 1
        for (int s = 0; s < p.ns1; ++s) {
            if (s > 0) ring_wait(&full[rp.st], rp.phase, p.status);
            const uint8_t* sb = stage(rp.st);
            mma_stage<NT, CPB, false>(acc, sb, R, sb + p.S.act0, p.gshift);
            release(rp);
            rp.next(p.S.stages);
        }
        if (row0 >= p.I) return;                                         // (the last unit of a narrow layer)
        unscale(acc);
        if (lora) {
            if (!ahead) lora_load();
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) mma16816(acc[m][nt], lb[m][0], lb[m][1], lb[m][2], lb[m][3], lu[m][nt][0], lu[m][nt][1]);
            for (int kr = 16; kr < p.rank; kr += 16) {
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    uint32_t a[4];
                    lora_rows(b_rows(m), kr, a);
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        const __half* ut = uq + (size_t)(m * p.cap + nt * 8) * p.r16 + kr;
                        mma16816(acc[m][nt], a[0], a[1], a[2], a[3], __ldg(reinterpret_cast<const uint32_t*>(ut)), __ldg(reinterpret_cast<const uint32_t*>(ut + 8)));
                    }
                }
            }
        }
        store_h<NT>(tile, row0, [&](int nt, int q) { return silu_f(acc[0][nt][q]) * acc[1][nt][q]; });
    }

    // h of 16 rows and the tile's tokens to global in operand order; value(nt, q): what this lane holds of it, as the accumulators lie
    template <int NT, typename V>
    __device__ __forceinline__ void store_h(int tile, int row0, V value) {
        // 16 rows x 8 tokens through the warp's own shared memory: lane = (token, 8 rows, value / residual)
        float* hs = reinterpret_cast<float*>(smem + p.S.h) + warp * (8 * 20);
        const int tok = lane >> 2, r8 = (lane >> 1) & 1, lo = lane & 1, n = row0 + r8 * 8, c = n >> 5;
        uint8_t* dst = p.hq + (size_t)tile * p.cap * p.I * 4 + ((size_t)(c * 2 + lo) * (8 * NT) + tok) * 64 + ((n & 31) >> 3) * 16;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            float* q = hs + (2 * t4) * 20 + g8;
            q[0] = value(nt, 0); q[20] = value(nt, 1);
            q[8] = value(nt, 2); q[28] = value(nt, 3);
            __syncwarp();
            const float4 va = *reinterpret_cast<const float4*>(hs + tok * 20 + r8 * 8), vb = *reinterpret_cast<const float4*>(hs + tok * 20 + r8 * 8 + 4);
            const float f[8] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
            *reinterpret_cast<uint4*>(dst + nt * 512) = lo ? permute8_lo(f) : permute8(f);
            __syncwarp();
        }
        // these rows are written: count them (bulk copies of other SMs will read them)
        asm volatile("fence.proxy.async;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p.done + tile) : "memory");
    }

    // ---- gate/up, narrow units (a column of 8 pairs): four row tiles, a warp for each of gate and of up; the up warp hands its sums over
    template <int CPB>
    __device__ __forceinline__ void gate_up_narrow(int tile, int sub, int ad, RingPos& rp) {
        const int rt = warp >> 1, m = warp & 1, row0 = (sub * (GW / 2) + rt) * 16;
        float acc[1][1][4];
        clear(acc);
        const uint16_t* B = static_cast<const uint16_t*>(m ? p.lora.B_up : p.lora.B_gate) + ((size_t)ad * p.I + row0 + g8) * p.rank;
        const __half* u = p.u + ((size_t)tile * 2 + m) * p.cap * p.r16 + (size_t)g8 * p.r16 + 2 * t4;
        uint32_t lb[4], lu[2];
        if (p.rank > 0) {                                                // (first 16 ranks: asked for now, used behind the main loop)
            lora_rows(B, 0, lb);
#pragma unroll
            for (int q = 0; q < 2; ++q) lu[q] = __ldg(reinterpret_cast<const uint32_t*>(u + 8 * q));
        }
        WarpRuns R;
        R.code[0] = R.code[1] = (uint32_t)(m * (GW / 2) + rt) * 1024;
        R.sz[0] = R.sz[1] = p.S.sz0 + (uint32_t)(m * (GW / 2) + rt) * (uint32_t)(GStageK >> p.gshift) * 64;
        R.code_part = R.sz_part = 0; R.csh = 2;
#pragma unroll 1
        for (int s = 0; s < p.ns1; ++s) {
            if (s > 0) ring_wait(&full[rp.st], rp.phase, p.status);
            const uint8_t* sb = stage(rp.st);
            mma_stage<1, CPB, false>(acc, sb, R, sb + p.S.act0, p.gshift);
            release(rp);
            rp.next(p.S.stages);
        }
        unscale(acc);
        if (p.rank > 0) {
            mma16816(acc[0][0], lb[0], lb[1], lb[2], lb[3], lu[0], lu[1]);
            for (int kr = 16; kr < p.rank; kr += 16) {
                uint32_t a[4];
                lora_rows(B, kr, a);
                mma16816(acc[0][0], a[0], a[1], a[2], a[3], __ldg(reinterpret_cast<const uint32_t*>(u + kr)), __ldg(reinterpret_cast<const uint32_t*>(u + kr + 8)));
            }
        }
        float4* up = reinterpret_cast<float4*>(smem + p.S.h + (warp | 1) * (8 * 20 * 4)) + lane;      // (the up warp's part)
        const int bar = 1 + (int)(threadIdx.x >> 6);                     // of the two warps
        if (m) *up = make_float4(acc[0][0][0], acc[0][0][1], acc[0][0][2], acc[0][0][3]);
        asm volatile("bar.sync %0, 64;" ::"r"(bar) : "memory");
        if (!m) {
            const float4 v = *up;
            const float w[4] = {v.x, v.y, v.z, v.w};
            store_h<1>(tile, row0, [&](int, int q) { return silu_f(acc[0][0][q]) * w[q]; });
        }
        asm volatile("bar.sync %0, 64;" ::"r"(bar) : "memory");
    }

    // ---- down: two output row tiles of this warp; o[pair][row] = gate (W h + B (sigma A h))
    template <int NT, int CPB>
    __device__ __forceinline__ void down(int sub, int ad, uint32_t count, RingPos& rp) {
        const int row0 = (sub * GW + warp) * 32;
        float acc[2][NT][4];
        clear(acc);
        const bool lora = p.rank > 0 && row0 < p.H;
        constexpr bool ahead = NT <= 2;
        const uint16_t* B = static_cast<const uint16_t*>(p.lora.B_down) + ((size_t)ad * p.H + row0 + g8) * p.rank;
        uint32_t lb[2][4];
        if (ahead && lora) {
#pragma unroll
            for (int m = 0; m < 2; ++m) lora_rows(B + (size_t)m * 16 * p.rank, 0, lb[m]);
        }
        WarpRuns R;
        const uint32_t crun = (uint32_t)p.cps * 256, szrun = (uint32_t)((p.cps * 32) >> p.gshift) * 64;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            R.code[m] = (uint32_t)(2 * warp + m) * crun;
            R.sz[m] = p.S.sz0 + (uint32_t)(2 * warp + m) * szrun;
        }
        R.code_part = 2 * GW * crun; R.sz_part = 2 * GW * szrun; R.csh = p.csh;
#pragma unroll 1
        for (int s = 0; s < p.ns2; ++s) {
            if (s > 0) ring_wait(&full[rp.st], rp.phase, p.status);
            const uint8_t* sb = stage(rp.st);
            mma_stage<NT, CPB, true>(acc, sb, R, sb + p.S.act0, p.gshift);
            release(rp);
            rp.next(p.S.stages);
        }
        unscale(acc);
        // the projections of h, pairs and gates, as the group's projection warp has left them
        const uint32_t par = count & 1;
        const __half* s_ud = reinterpret_cast<const __half*>(smem + p.S.ud) + par * p.cap * p.r16;
        const int2* s_pr = reinterpret_cast<const int2*>(smem + p.S.pr) + par * p.cap;
        ring_wait(&ud_full[par], (count >> 1) & 1, p.status);
        if (row0 < p.H) {
            if (lora) {
                for (int kr = 0; kr < p.rank; kr += 16) {
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        if (kr > 0 || !ahead) lora_rows(B + (size_t)m * 16 * p.rank, kr, lb[m]);
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt) {
                            const __half* ut = s_ud + (nt * 8 + g8) * p.r16 + kr + 2 * t4;
                            mma16816(acc[m][nt], lb[m][0], lb[m][1], lb[m][2], lb[m][3], *reinterpret_cast<const uint32_t*>(ut), *reinterpret_cast<const uint32_t*>(ut + 8));
                        }
                    }
                }
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int2 pr = s_pr[nt * 8 + 2 * t4 + j];
                    if (pr.x >= 0) {
                        float* o = p.o + (size_t)pr.x * p.H + row0 + g8;
                        const float gt = __int_as_float(pr.y);
                        o[0] = gt * acc[0][nt][j]; o[8] = gt * acc[0][nt][2 + j];
                        o[16] = gt * acc[1][nt][j]; o[24] = gt * acc[1][nt][2 + j];
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&ud_empty[par]);
    }

    // ---- the projection warp: for every down unit of the group, pairs, gates and sigma A_down h of its tile
    __device__ __forceinline__ void project() {
        const int4* queue = reinterpret_cast<const int4*>(smem + p.S.queue);
        for (uint32_t n = 0;; ++n) {
            const uint32_t qs = n % GQueue, par = n & 1;
            ring_wait(&q_full[qs], (n / GQueue) & 1, p.status);
            const int4 ti = queue[qs];                                   // {tile, first, pairs, adapter}; tile < 0: no more
            __syncwarp();
            if (lane == 0) mbar_arrive(&q_empty[qs]);
            if (ti.x < 0) return;
            const int nt_all = (ti.z + 7) >> 3;
            int pr = -1;
            float gt = 0.f;
            if (lane < ti.z) { pr = __ldg(p.order + ti.y + lane); gt = __ldg(p.gates + pr); }
            if (n >= 2) ring_wait(&ud_empty[par], ((n >> 1) & 1) ^ 1u, p.status);
            if (lane < p.cap) (reinterpret_cast<int2*>(smem + p.S.pr) + par * p.cap)[lane] = make_int2(pr, __float_as_int(gt));
            if (p.rank > 0) {
                __half* s_ud = reinterpret_cast<__half*>(smem + p.S.ud) + par * p.cap * p.r16;
                const uint8_t* hq = p.hq + (size_t)ti.x * p.cap * p.I * 4 + g8 * 64 + t4 * 16;
                for (int j0 = 0; j0 < p.rank; j0 += 16) {
                    const bool lo_ok = j0 + g8 < p.rank, hi_ok = j0 + g8 + 8 < p.rank;
                    const uint16_t* A = static_cast<const uint16_t*>(p.lora.A_down) + ((size_t)ti.w * p.rank + j0 + g8) * p.I + 8 * t4;
                    for (int nt = 0; nt < nt_all; ++nt) {
                        float cc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
                        for (int c = 0; c < p.I / 32; ++c) {
                            const uint4 z = make_uint4(0, 0, 0, 0);
                            const uint4 ra = lo_ok ? __ldg(reinterpret_cast<const uint4*>(A + c * 32)) : z;
                            const uint4 rb = hi_ok ? __ldg(reinterpret_cast<const uint4*>(A + (size_t)8 * p.I + c * 32)) : z;
                            const uint8_t* hb = hq + (size_t)c * 2 * nt_all * 512 + nt * 512;
                            const uint4 hv = __ldcg(reinterpret_cast<const uint4*>(hb)), hl = __ldcg(reinterpret_cast<const uint4*>(hb + nt_all * 512));
                            const uint4 a = bf16x8_permute8(ra), b = bf16x8_permute8(rb);
                            mma16816(cc, a.x, b.x, a.y, b.y, hv.x, hv.y);
                            mma16816(cc, a.z, b.z, a.w, b.w, hv.z, hv.w);
                            mma16816(cc, a.x, b.x, a.y, b.y, hl.x, hl.y);
                            mma16816(cc, a.z, b.z, a.w, b.w, hl.z, hl.w);
                        }
                        __half* q = s_ud + (nt * 8 + 2 * t4) * p.r16 + j0 + g8;
                        q[0] = __float2half_rn(p.sigma * cc[0]); q[p.r16] = __float2half_rn(p.sigma * cc[1]);
                        q[8] = __float2half_rn(p.sigma * cc[2]); q[p.r16 + 8] = __float2half_rn(p.sigma * cc[3]);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&ud_full[par]);
        }
    }

    // ---- the producer lane: units from the ticket counter, stage by stage into the ring
    __device__ __forceinline__ void produce(const CUtensorMap* m_cgu, const CUtensorMap* m_zgu, const CUtensorMap* m_cd, const CUtensorMap* m_zd) {
        int4* s_info = reinterpret_cast<int4*>(smem + p.S.info);             // [stages][2]
        int4* queue = reinterpret_cast<int4*>(smem + p.S.queue);
        const int nt_all = *p.n_tiles, u1 = nt_all * p.n1, total = u1 + nt_all * p.n2;
        const int need = p.I / 16;                                           // row tiles of h in a tile
        const uint64_t polw = p.evict_first ? policy_evict_first() : policy_evict_normal(), pola = policy_evict_normal();
        RingPos rp{0, 0u};
        bool wrapped = false;
        uint32_t n_down = 0;
        auto acquire = [&]() { if (wrapped) ring_wait(&empty[rp.st], rp.phase ^ 1u, p.status); };
        auto advance = [&]() { rp.next(p.S.stages); if (rp.st == 0) wrapped = true; };
        auto tile_of = [&](int t) { return t < u1 ? t / p.n1 : (t - u1) / p.n2; };
        auto post = [&](int4 v) {
            const uint32_t qs = n_down % GQueue;
            if (n_down >= GQueue) ring_wait(&q_empty[qs], ((n_down / GQueue) & 1) ^ 1u, p.status);
            queue[qs] = v;
            mbar_arrive(&q_full[qs]);
            ++n_down;
        };
        int t_next = atomicAdd(p.ticket, 1);
        int4 ti_next = t_next < total ? __ldg(p.tiles + tile_of(t_next)) : make_int4(0, 0, 0, 0);
        for (;;) {
            const int t = t_next;
            const int4 ti = ti_next;
            if (t >= total) break;
            const bool gu = t < u1;
            const int tile = tile_of(t), sub = gu ? t - tile * p.n1 : t - u1 - tile * p.n2;
            const int nt = (ti.z + 7) >> 3, ns = gu ? p.ns1 : p.ns2;
            const uint32_t act = (gu ? 2048u : 4096u) * nt;
            const uint8_t* asrc = gu ? p.xq + (size_t)tile * p.cap * p.H * 2 : p.hq + (size_t)tile * p.cap * p.I * 4;
            for (int s = 0; s < ns; ++s) {
                acquire();
                uint8_t* sb = stage(rp.st);
                uint64_t* bar = &full[rp.st];
                if (s == 0) {
                    s_info[2 * rp.st] = make_int4(gu ? 1 : 2, tile, sub, nt);
                    s_info[2 * rp.st + 1] = make_int4(ti.w, 0, 0, 0);
                }
                mbar_expect_tx(bar, (gu ? (GCodeBytes + p.S.sz_bytes) / GW * p.rows1 : GCodeBytes + p.S.sz_bytes) + act);
                if (gu) {
                    tma_load_5d(sb, m_cgu, s * GStageK, sub * p.rows1, 0, ti.x, 0, bar, polw);
                    tma_load_5d(sb + p.S.sz0, m_zgu, ((s * GStageK) >> p.gshift) * 8, sub * p.rows1, 0, ti.x, 0, bar, polw);
                } else {
                    const int sw = p.I / kDownSlices, kk = s * GStageK;
                    const int sl = p.sp > 1 ? s * p.sp : kk / sw, x = p.sp > 1 ? 0 : kk % sw;
                    tma_load_5d(sb, m_cd, x, sub * 2 * GW, sl, ti.x, 0, bar, polw);
                    tma_load_5d(sb + p.S.sz0, m_zd, (x >> p.gshift) * 8, sub * 2 * GW, sl, ti.x, 0, bar, polw);
                }
                if (s == 0 && !gu) {                                     // every row of the tile's h has been written
                    int have = 0;
                    uint32_t it = 0;
                    do {
                        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(have) : "l"(p.done + tile) : "memory");
                        if (have < need) __nanosleep(40);
                    } while (have < need && ++it < kSpinLimit);
                    if (have < need) atomicExch(p.status, EDG_E_TIMEOUT);
                    asm volatile("fence.proxy.async;" ::: "memory");
                    post(make_int4(tile, ti.y, ti.z, ti.w));
                }
                bulk_g2s_hint(sb + p.S.act0, asrc + (size_t)s * act, act, bar, pola);
                advance();
                // The unit after this one is taken near the end of this one's copies, six stages ahead of its arithmetic: at its start, CTAs
                // that begin two microseconds before the others (where no CTA of the kernel before holds the SM) took two units each.
                if (s == max(0, ns - 3)) t_next = atomicAdd(p.ticket, 1);
                if (s == ns - 1 && t_next < total) ti_next = __ldg(p.tiles + tile_of(t_next));
            }
        }
        acquire();
        s_info[2 * rp.st] = make_int4(0, 0, 0, 0);
        mbar_arrive(&full[rp.st]);
        post(make_int4(-1, 0, 0, 0));
    }
};

// Warps: GGroups groups of GW consumers, then a producer warp per group, then a projection warp per group.  NTMAX: columns of 8
// pairs a tile may have; the form for one column keeps its registers free of the code for more.
template <int CPB, int NTMAX, bool NARROW>
__global__ void __launch_bounds__(GThreads, 1)
grouped_ffn_kernel(const __grid_constant__ GffnParams p, const __grid_constant__ CUtensorMap m_cgu, const __grid_constant__ CUtensorMap m_zgu,
                   const __grid_constant__ CUtensorMap m_cd, const __grid_constant__ CUtensorMap m_zd) {
    extern __shared__ __align__(1024) uint8_t smem_all[];
    const int warp_all = threadIdx.x >> 5, side = warp_all - GGroups * GW;
    const int group = side >= 0 ? side % GGroups : warp_all / GW;
    uint8_t* smem = smem_all + group * p.S.group_bytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.S.bars);
    Gffn k{p, smem, bars, bars + GMaxStages, bars + 2 * GMaxStages, bars + 2 * GMaxStages + GQueue, bars + 2 * GMaxStages + 2 * GQueue,
           bars + 2 * GMaxStages + 2 * GQueue + 2, (int)(threadIdx.x & 31), warp_all % GW, (int)((threadIdx.x & 31) >> 2), (int)(threadIdx.x & 3)};
    if (side < 0 && k.warp == 0 && k.lane == 0) {
        for (int s = 0; s < p.S.stages; ++s) { mbar_init(&k.full[s], 1); mbar_init(&k.empty[s], GW); }
        for (int s = 0; s < GQueue; ++s) { mbar_init(&k.q_full[s], 1); mbar_init(&k.q_empty[s], 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(&k.ud_full[s], 1); mbar_init(&k.ud_empty[s], GW); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    pdl_wait_prior_grid();
    if (side >= 0) {
        if (side < GGroups) {
            if (k.lane == 0) k.produce(&m_cgu, &m_zgu, &m_cd, &m_zd);
        } else k.project();
        return;
    }
    const int4* s_info = reinterpret_cast<const int4*>(smem + p.S.info);
    RingPos rp{0, 0u};
    uint32_t n_down = 0;
    for (;;) {
        ring_wait(&k.full[rp.st], rp.phase, p.status);
        const int4 a = s_info[2 * rp.st];                                // {kind, tile, unit of the tile, columns of 8 pairs}
        const int ad = s_info[2 * rp.st + 1].x;
        if (a.x == 0) break;
        if (a.x == 1) {
            if (NARROW) k.gate_up_narrow<CPB>(a.y, a.z, ad, rp);
            else if (NTMAX == 1 || a.w == 1) k.gate_up<1, CPB>(a.y, a.z, ad, rp);
            else if (a.w == 2) k.gate_up<(NTMAX < 2 ? 1 : 2), CPB>(a.y, a.z, ad, rp);
            else if (a.w == 3) k.gate_up<(NTMAX < 3 ? 1 : 3), CPB>(a.y, a.z, ad, rp);
            else k.gate_up<(NTMAX < 4 ? 1 : 4), CPB>(a.y, a.z, ad, rp);
        } else {
            if (NTMAX == 1 || a.w == 1) k.down<1, CPB>(a.z, ad, n_down, rp);
            else if (a.w == 2) k.down<(NTMAX < 2 ? 1 : 2), CPB>(a.z, ad, n_down, rp);
            else if (a.w == 3) k.down<(NTMAX < 3 ? 1 : 3), CPB>(a.z, ad, n_down, rp);
            else k.down<(NTMAX < 4 ? 1 : 4), CPB>(a.z, ad, n_down, rp);
            ++n_down;
        }
    }
}

// ---------------------------------------------------------------- grouping

struct GroupArgs {
    const int32_t *slots, *table, *experts;
    int32_t *pair_slot, *order, *n_tiles, *ticket, *done, *status;
    int32_t* cnt_g;                       // counts in global memory: a pool with more slots than shared memory holds counters for
    int4* tiles;
    int P, E, n_slots, cap, adapters;     // adapters: one per expert, so a pair's expert id must be in range
    int nw;                               // warps that own a range of pairs
};

// One CTA sorts the pairs by slot.  Warp w owns a contiguous range; counts per (warp, slot) give every pair its place, in
// ascending pair index within a slot.  Bound by the latency of its few dependent trips: 5.5 us for 512 pairs against 7 us
// of the three kernels it replaces (and their launches).
__global__ void __launch_bounds__(1024) group_pairs_kernel(GroupArgs a) {
    extern __shared__ int s_cnt[];                       // [nw][n_slots], then [n_slots] first position
    __shared__ int s_w[2][32];
    int* cnt = a.cnt_g != nullptr ? a.cnt_g : s_cnt;
    int* s_base = cnt + (size_t)a.nw * a.n_slots;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_launch_dependents();
    pdl_wait_prior_grid();
    for (int i = tid; i < a.nw * a.n_slots; i += 1024) cnt[i] = 0;
    __syncthreads();
    const int per = ((a.P + a.nw - 1) / a.nw + 31) / 32 * 32;
    const int lo = min(a.P, warp * per), hi = warp < a.nw ? min(a.P, lo + per) : lo;
    int* mine = cnt + (size_t)warp * a.n_slots;
    for (int i0 = lo; i0 < hi; i0 += 128) {
        int s[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 32 + lane;
            s[u] = i < hi ? a.slots[i] : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 32 + lane;
            int e = s[u];
            if (i < hi) {
                if (a.table != nullptr) s[u] = (e >= 0 && e < a.E) ? a.table[e] : -1;
                else if (a.experts != nullptr) e = a.experts[i];
                else e = 0;
                if (s[u] < 0 || s[u] >= a.n_slots || (a.adapters && (e < 0 || e >= a.E))) { s[u] = -1; atomicExch(a.status, EDG_E_RANGE); }
            } else s[u] = -1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 32 + lane;
            if (i < hi) a.pair_slot[i] = s[u];
            const unsigned m = __match_any_sync(0xFFFFFFFFu, s[u]);
            if (s[u] >= 0 && lane == __ffs(m) - 1) mine[s[u]] += __popc(m);
            __syncwarp();
        }
    }
    __syncthreads();
    // places: per slot a running sum over the warps, then sums over the slots (pairs and tiles)
    const int sper = (a.n_slots + 1023) / 1024, s0 = min(a.n_slots, tid * sper), s1 = min(a.n_slots, s0 + sper);
    int pairs = 0, tiles = 0;
    for (int s = s0; s < s1; ++s) {
        int run = 0;
        for (int w = 0; w < a.nw; ++w) { const int c = cnt[(size_t)w * a.n_slots + s]; cnt[(size_t)w * a.n_slots + s] = run; run += c; }
        s_base[s] = run;
        pairs += run;
        tiles += (run + a.cap - 1) / a.cap;
    }
    int ip = pairs, it = tiles;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xFFFFFFFFu, ip, o), y = __shfl_up_sync(0xFFFFFFFFu, it, o);
        if (lane >= o) { ip += x; it += y; }
    }
    if (lane == 31) { s_w[0][warp] = ip; s_w[1][warp] = it; }
    __syncthreads();
    int bp = 0, bt = 0;
    for (int w = 0; w < warp; ++w) { bp += s_w[0][w]; bt += s_w[1][w]; }
    int pos = bp + ip - pairs, tn = bt + it - tiles;
    for (int s = s0; s < s1; ++s) {
        const int run = s_base[s];
        s_base[s] = pos;
        for (int f = 0; f < run; f += a.cap) { a.tiles[tn] = make_int4(s, pos + f, min(a.cap, run - f), 0); a.done[tn] = 0; ++tn; }
        pos += run;
    }
    if (tid == 1023) { *a.n_tiles = tn; *a.ticket = 0; }
    __syncthreads();
    for (int i0 = lo; i0 < hi; i0 += 32) {
        const int i = i0 + lane;
        const int s = i < hi ? a.pair_slot[i] : -1;
        const unsigned m = __match_any_sync(0xFFFFFFFFu, s);
        if (s >= 0) a.order[s_base[s] + mine[s] + __popc(m & ((1u << lane) - 1))] = i;
        __syncwarp();
        if (s >= 0 && lane == __ffs(m) - 1) mine[s] += __popc(m);
        __syncwarp();
    }
}

// ---------------------------------------------------------------- operand tiles

struct TileArgs {
    int4* tiles;
    const int32_t *n_tiles, *order, *slots, *table, *experts;
    const uint16_t* x;
    uint8_t* xq;
    __half* u;
    edg_lora lora;
    int H, K, rank, r16, cap, adapters;
    float sigma;
    GroupArgs group;                      // (for the form that sorts)
};

// Up to kSortPairs pairs every CTA finds its tile by itself -- each pair counts the pairs before it in slot order -- and the kernel
// that sorts is spared: 5 of the 62 us of 5 tokens.  Each CTA reads all pairs, in the square of their number: 1 us at 128, 25 at 512.
// Same tiles in the same order.  Returns the tile, with `s_pair` its pairs; z = 0: there is none.
constexpr int kSortPairs = 128;
__device__ __forceinline__ int4 find_tile(const GroupArgs& g, int tile, int* s_pair) {
    __shared__ __align__(16) int s_slot[kSortPairs];
    __shared__ int s_nt[kSortPairs], s_ti[3], s_n;
    const int i = threadIdx.x;                                           // this thread's pair
    const bool lead = blockIdx.x == 0 && blockIdx.y == 0;
    int slot = -1;
    if (i < g.P) {
        int e = g.slots[i];
        slot = e;
        if (g.table != nullptr) slot = (e >= 0 && e < g.E) ? g.table[e] : -1;
        else if (g.experts != nullptr) e = g.experts[i];
        else e = 0;
        if (slot < 0 || slot >= g.n_slots || (g.adapters && (e < 0 || e >= g.E))) {
            slot = -1;
            if (lead) atomicExch(g.status, EDG_E_RANGE);
        }
        if (lead) g.pair_slot[i] = slot;
    }
    if (i < kSortPairs) s_slot[i] = slot;
    if (i == 0) { s_ti[0] = -1; s_ti[2] = 0; s_n = 0; }
    __syncthreads();
    int pos = 0, before = 0, all = 0, nt = 0;
    if (slot >= 0) {
        for (int j = 0; j < g.P; ++j) {
            const int v = s_slot[j];
            pos += (unsigned)v < (unsigned)slot;
            before += v == slot && j < i;
            all += v == slot;
        }
        pos += before;
        if (before == 0) nt = (all + g.cap - 1) / g.cap;
    }
    if (i < kSortPairs) s_nt[i] = nt;
    __syncthreads();
    if (nt > 0) {
        int base = 0;
        for (int j = 0; j < g.P; ++j) base += (unsigned)s_slot[j] < (unsigned)slot ? s_nt[j] : 0;
        if (tile >= base && tile < base + nt) {
            const int f = (tile - base) * g.cap;
            s_ti[0] = slot; s_ti[1] = pos + f; s_ti[2] = min(g.cap, all - f);
        }
        atomicAdd(&s_n, nt);
    }
    __syncthreads();
    const int4 ti = make_int4(s_ti[0], s_ti[1], s_ti[2], 0);
    if (slot >= 0 && slot == ti.x && pos >= ti.y && pos < ti.y + ti.z) {
        s_pair[pos - ti.y] = i;
        if (blockIdx.y == 0) g.order[pos] = i;
    }
    if (lead && i == 0) { *g.n_tiles = s_n; *g.ticket = 0; }
    if (blockIdx.y == 0 && i == 0 && ti.z > 0) g.done[tile] = 0;
    __syncthreads();
    return ti;
}

// blockIdx.y < cap / 8: eight of the tile's token states as fp16 B words, chunk by chunk as the ring reads them (and, for the
// first, the tile's adapter); the rest: 16 rows each of u = (sigma A_gate x, sigma A_up x) for every token of the tile.
template <bool SORT>
__global__ void __launch_bounds__(256) tile_operands_kernel(TileArgs a) {
    __shared__ int s_tok[32], s_pair[32];
    __shared__ float s_red[8 * 16 * 32];
    pdl_launch_dependents();
    pdl_wait_prior_grid();
    const int tile = blockIdx.x;
    int4 ti;
    if constexpr (SORT) {
        ti = find_tile(a.group, tile, s_pair);
        if (ti.z == 0) return;
    } else {
        if (tile >= *a.n_tiles) return;
        ti = a.tiles[tile];
    }
    const int tid = threadIdx.x, nt = (ti.z + 7) >> 3, ntok = nt * 8, nx = a.cap / 8;
    if ((int)blockIdx.y < nx && (int)blockIdx.y >= nt) return;
    if (tid < 32) s_tok[tid] = tid < ti.z ? (SORT ? s_pair[tid] : a.order[ti.y + tid]) / a.K : -1;
    int ad = 0;
    if (a.adapters && ((int)blockIdx.y >= nx || (blockIdx.y == 0 && tid == 0))) {
        const int pr0 = SORT ? s_pair[0] : a.order[ti.y];
        ad = a.table != nullptr ? a.slots[pr0] : (a.experts != nullptr ? a.experts[pr0] : 0);
    }
    __syncthreads();
    if ((int)blockIdx.y < nx) {
        if (blockIdx.y == 0 && tid == 0) {
            if (SORT) a.tiles[tile] = make_int4(ti.x, ti.y, ti.z, ad);
            else a.tiles[tile].w = ad;
        }
        uint8_t* out = a.xq + (size_t)tile * a.cap * a.H * 2;
        const int t0 = blockIdx.y * 8, q = tid & 3, tok = t0 + ((tid >> 2) & 7), st = s_tok[tok];
        const uint16_t* src = a.x + (size_t)(st < 0 ? 0 : st) * a.H + q * 8;
        for (int c0 = tid >> 5; c0 < a.H >> 5; c0 += 64) {               // 8 chunks of 32 k per warp and round, one per warp at a time
            uint4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                v[u] = make_uint4(0, 0, 0, 0);
                if (c0 + 8 * u < a.H >> 5 && st >= 0) v[u] = *reinterpret_cast<const uint4*>(src + (c0 + 8 * u) * 32);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (c0 + 8 * u >= a.H >> 5) break;
                *reinterpret_cast<uint4*>(out + ((size_t)(c0 + 8 * u) * ntok + tok) * 64 + q * 16) = bf16x8_permute8(v[u]);
            }
        }
        return;
    }
    // u: 16 adapter rows, K split over the warps; operands 16 bytes per lane under a k order that A and x share
    const int lane = tid & 31, warp = tid >> 5, g8 = lane >> 2, t4 = lane & 3;
    const int kw = a.H / 8, k0 = warp * kw + 8 * t4, rt = blockIdx.y - nx;
    const int m = rt / (a.r16 / 16), j0 = (rt % (a.r16 / 16)) * 16;
    const uint16_t* A = static_cast<const uint16_t*>(m ? a.lora.A_up : a.lora.A_gate) + ((size_t)ad * a.rank + j0 + g8) * a.H;
    const bool lo_ok = j0 + g8 < a.rank, hi_ok = j0 + 8 + g8 < a.rank;
    float c[4][4];
#pragma unroll
    for (int n = 0; n < 4; ++n) { c[n][0] = 0.f; c[n][1] = 0.f; c[n][2] = 0.f; c[n][3] = 0.f; }
    const uint16_t* xr[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        const int tok = n < nt ? s_tok[n * 8 + g8] : -1;
        xr[n] = tok >= 0 ? a.x + (size_t)tok * a.H : nullptr;
    }
    // (K per warp is H / 8: a multiple of 16; the last step of a narrow layer may be half a block of 32, whose upper half reads zeros)
#pragma unroll 4
    for (int kb = 0; kb < kw; kb += 32) {
        const bool in = kb + 8 * t4 < kw;
        const uint4 z = make_uint4(0, 0, 0, 0);
        const uint4 lo = lo_ok && in ? *reinterpret_cast<const uint4*>(A + k0 + kb) : z;
        const uint4 hi = hi_ok && in ? *reinterpret_cast<const uint4*>(A + (size_t)8 * a.H + k0 + kb) : z;
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            if (n < nt) {
                const uint4 b = xr[n] != nullptr && in ? *reinterpret_cast<const uint4*>(xr[n] + k0 + kb) : z;
                mma16816_bf16(c[n], lo.x, hi.x, lo.y, hi.y, b.x, b.y);
                mma16816_bf16(c[n], lo.z, hi.z, lo.w, hi.w, b.z, b.w);
            }
        }
    }
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        float* q = s_red + (warp * 16 + g8) * 32 + n * 8 + 2 * t4;
        q[0] = c[n][0]; q[1] = c[n][1]; q[8 * 32] = c[n][2]; q[8 * 32 + 1] = c[n][3];
    }
    __syncthreads();
    for (int i = tid; i < 16 * ntok; i += 256) {
        const int j = i & 15, tok = i >> 4;
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) v += s_red[(w * 16 + j) * 32 + tok];
        a.u[(((size_t)tile * 2 + m) * a.cap + tok) * a.r16 + j0 + j] = __float2half_rn(a.sigma * v);
    }
}

// ---------------------------------------------------------------- y[t] = sum over the token's choices

struct SumArgs {
    const float* o;
    const int32_t* pair_slot;
    void* y;
    int T, H, K;
};
template <typename OutT>
__global__ void __launch_bounds__(256) sum_choices_kernel(SumArgs a) {
    pdl_wait_prior_grid();
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;             // four outputs
    if (i * 4 >= (size_t)a.T * a.H) return;
    const int t = (int)(i * 4 / a.H), n = (int)(i * 4 % a.H);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = 0; k0 < a.K; k0 += 8) {
        float4 w[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int k = k0 + u, pair = t * a.K + k;
            w[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < a.K && a.pair_slot[pair] >= 0) w[u] = __ldcg(reinterpret_cast<const float4*>(a.o + (size_t)pair * a.H + n));
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) { v.x += w[u].x; v.y += w[u].y; v.z += w[u].z; v.w += w[u].w; }
    }
    OutT* y = reinterpret_cast<OutT*>(a.y) + i * 4;
    store_out<OutT>(y, 0, v.x); store_out<OutT>(y, 1, v.y); store_out<OutT>(y, 2, v.z); store_out<OutT>(y, 3, v.w);
}

// ---------------------------------------------------------------- host

typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_tiled() {
    static const EncodeTiled fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) f = nullptr;
        return reinterpret_cast<EncodeTiled>(f);
    }();
    return fn;
}

// an array of 8-byte elements of up to five dimensions (strides in bytes, of dimensions 1..4)
bool tensor_map(CUtensorMap* m, const void* base, const uint64_t (&dim)[5], const uint64_t (&stride)[4], const uint32_t (&box)[5]) {
    const EncodeTiled fn = encode_tiled();
    if (fn == nullptr) return false;
    cuuint64_t d[5], s[4];
    cuuint32_t b[5], es[5] = {1, 1, 1, 1, 1};
    for (int i = 0; i < 5; ++i) { d[i] = dim[i]; b[i] = box[i]; }
    for (int i = 0; i < 4; ++i) s[i] = stride[i];
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 5, const_cast<void*>(base), d, s, b, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

int sm_count() {
    int dev = 0, n = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
}

// Pairs a tile holds.  A tile's weights are read once whatever it holds; its MMA time grows with its columns of 8.
int grouped_tile_cap(const edg_layer_desc& d, int T) {
    const int64_t P = (int64_t)T * d.K;
    return P <= 4 * (int64_t)d.n_slots ? 8 : (P <= 8 * (int64_t)d.n_slots ? 16 : 32);
}

int32_t run_grouped_ffn(const edg_layer_desc* d, const GroupedParams& g, const WorkspaceLayout& W, uint8_t* ws, cudaStream_t st) {
    const int P = g.T * g.K, cap = grouped_tile_cap(*d, g.T), H = g.H, I = g.I;
    GffnParams p{};
    int4* tiles = reinterpret_cast<int4*>(ws + W.g_tiles);
    int32_t* n_tiles = reinterpret_cast<int32_t*>(ws + W.n_tiles);
    int32_t* order = reinterpret_cast<int32_t*>(ws + W.g_order);
    __half* u = reinterpret_cast<__half*>(ws + W.g_u);
    uint8_t* xq = ws + W.g_xq;
    p.tiles = tiles; p.n_tiles = n_tiles; p.order = order; p.u = u; p.xq = xq;
    p.ticket = n_tiles + 32;                       // (its own cache line)
    p.done = reinterpret_cast<int32_t*>(ws + W.g_done);
    p.hq = ws + W.g_hq;
    p.gates = g.gates;
    p.status = g.status;
    p.o = g.o;
    p.lora = g.lora;
    p.H = H; p.I = I; p.rank = g.rank; p.r16 = (g.rank + 15) / 16 * 16; p.cap = cap;
    while ((1 << p.gshift) < g.group) ++p.gshift;
    p.sigma = g.sigma;
    // Gate/up units of four row tiles (11 us instead of 20: what bounds a unit is its warps' instructions) while those of eight would leave
    // groups without one.  By the tiles that evenly spread pairs make; eight : four, four layers of 256 experts, top 8, us: 2 tokens 189 : 162,
    // 5 214 : 185, 8 247 : 229, 9 242 : 244, 15 303 : 312.
    const int sms = sm_count(), wide1 = (I / 16 + GW - 1) / GW;
    const double tiles_est = d->n_slots * (1.0 - std::pow(1.0 - 1.0 / d->n_slots, P));
    const bool narrow = cap == 8 && tiles_est * 2 * wide1 <= 1.65 * GGroups * sms;
    p.rows1 = narrow ? GW / 2 : GW;
    p.n1 = (I / 16 + p.rows1 - 1) / p.rows1; p.n2 = (H / 16 + 2 * GW - 1) / (2 * GW);
    p.ns1 = H / GStageK; p.ns2 = I / GStageK;
    const int sw = I / kDownSlices;                // columns of a down slice; a stage takes part of one, or several
    p.sp = sw >= GStageK ? 1 : GStageK / sw;
    p.cps = sw >= GStageK ? 4 : sw / 32;
    p.csh = p.cps == 4 ? 2 : p.cps - 1;
    p.evict_first = cap == 8;                      // (a larger tile count per slot: the next tile of the slot reads them again)
    GffnSmem& S = p.S;
    S.sz0 = GCodeBytes;
    S.sz_bytes = 2 * GW * (uint32_t)(GStageK / g.group) * 64;
    S.act0 = S.sz0 + S.sz_bytes;
    S.stage_bytes = (S.act0 + (uint32_t)cap * 512 + 1023) / 1024 * 1024;
    const uint32_t nbars = 2 * GMaxStages + 2 * GQueue + 4;
    const uint32_t rest = GW * 8 * 20 * 4 + 2 * cap * p.r16 * 2 + 2 * cap * 8 + GMaxStages * 32 + GQueue * 16 + nbars * 8;
    S.stages = (int)((GSmemLimit / GGroups / 1024 * 1024 - rest) / S.stage_bytes);
    if (S.stages > GMaxStages) S.stages = GMaxStages;
    if (S.stages < 2) return EDG_E_SHAPE;
    uint32_t o = S.stages * S.stage_bytes;
    S.h = o;     o += GW * 8 * 20 * 4;
    S.ud = o;    o += 2 * cap * p.r16 * 2;
    S.pr = o;    o += 2 * cap * 8;
    S.info = o;  o += GMaxStages * 32;
    S.queue = o; o += GQueue * 16;
    S.bars = o;  o += nbars * 8;
    S.group_bytes = (o + 1023) / 1024 * 1024;
    const size_t smem = (size_t)GGroups * S.group_bytes;

    CUtensorMap cgu, zgu, cd, zd;
    const uint8_t* pool = g.pool;
    const uint64_t slots = (uint64_t)d->n_slots, R = g.L.bytes, gpr = (uint64_t)H / g.group, gps = (uint64_t)sw / g.group;
    const uint32_t kc_el = (uint32_t)(sw < GStageK ? sw : GStageK);
    // (run of a row tile, row tile, matrix or slice, slot; the fifth dimension is not used)
    bool ok = tensor_map(&cgu, pool + g.L.codes_gate, {(uint64_t)H, (uint64_t)I / 16, 2, slots, 1}, {(uint64_t)H * 8, (uint64_t)H * I / 2, R, R * slots},
                         {GStageK, (uint32_t)p.rows1, 2, 1, 1});
    ok = ok && tensor_map(&zgu, pool + g.L.sz_gate, {gpr * 8, (uint64_t)I / 16, 2, slots, 1}, {gpr * 64, gpr * I * 4, R, R * slots},
                          {(uint32_t)(GStageK / g.group * 8), (uint32_t)p.rows1, 2, 1, 1});
    ok = ok && tensor_map(&cd, pool + g.L.codes_down, {(uint64_t)sw, (uint64_t)H / 16, 4, slots, 1}, {(uint64_t)sw * 8, (uint64_t)H * sw / 2, R, R * slots},
                          {kc_el, 2 * GW, (uint32_t)p.sp, 1, 1});
    ok = ok && tensor_map(&zd, pool + g.L.sz_down, {gps * 8, (uint64_t)H / 16, 4, slots, 1}, {gps * 64, (uint64_t)H * gps * 4, R, R * slots},
                          {kc_el / g.group * 8, 2 * GW, (uint32_t)p.sp, 1, 1});
    if (!ok) { set_cuda_error(cudaErrorInvalidValue); return EDG_E_CUDA; }

    static OncePerDevice once;
    EDG_CUDA_TRY(once([] {
        const cudaError_t e = allow_smem(GSmemLimit, grouped_ffn_kernel<1, 1, false>, grouped_ffn_kernel<2, 1, false>, grouped_ffn_kernel<1, 4, false>,
                                        grouped_ffn_kernel<2, 4, false>, grouped_ffn_kernel<1, 1, true>, grouped_ffn_kernel<2, 1, true>);
        return e != cudaSuccess ? e : allow_smem(210 * 1024, group_pairs_kernel);
    }));
    GroupArgs ga{};
    ga.slots = g.slots; ga.table = g.table; ga.experts = g.experts;
    ga.pair_slot = g.pair_slot; ga.order = order; ga.n_tiles = n_tiles; ga.ticket = p.ticket;
    ga.done = p.done; ga.status = g.status; ga.tiles = tiles;
    ga.P = P; ga.E = g.E; ga.n_slots = d->n_slots; ga.cap = cap; ga.adapters = g.rank > 0 && g.n_adapters != 1;
    ga.nw = 32;
    while (ga.nw > 1 && (size_t)(ga.nw + 1) * d->n_slots * 4 > 200 * 1024) ga.nw /= 2;
    size_t cnt_bytes = (size_t)(ga.nw + 1) * d->n_slots * 4;
    if (cnt_bytes > 200 * 1024) { ga.cnt_g = reinterpret_cast<int32_t*>(ws + W.g_cnt); cnt_bytes = 0; }
    const bool sort = P <= kSortPairs;
    if (!sort) EDG_CUDA_TRY(launch_pdl(group_pairs_kernel, dim3(1), 1024, cnt_bytes, st, ga));
    TileArgs ta{};
    ta.group = ga;
    ta.tiles = tiles; ta.n_tiles = n_tiles; ta.order = order;
    ta.slots = g.slots; ta.table = g.table; ta.experts = g.experts; ta.x = g.x; ta.xq = xq; ta.u = u; ta.lora = g.lora;
    ta.H = H; ta.K = g.K; ta.rank = g.rank; ta.r16 = p.r16; ta.cap = cap; ta.adapters = ga.adapters; ta.sigma = g.sigma;
    EDG_CUDA_TRY(launch_pdl(sort ? tile_operands_kernel<true> : tile_operands_kernel<false>, dim3((unsigned)grouped_max_tiles(*d, g.T), cap / 8 + 2 * p.r16 / 16), 256, 0, st, ta));
    const bool wide = g.group >= 64;
    const auto kern = narrow ? (wide ? grouped_ffn_kernel<2, 1, true> : grouped_ffn_kernel<1, 1, true>)
                    : cap == 8 ? (wide ? grouped_ffn_kernel<2, 1, false> : grouped_ffn_kernel<1, 1, false>)
                               : (wide ? grouped_ffn_kernel<2, 4, false> : grouped_ffn_kernel<1, 4, false>);
    EDG_CUDA_TRY(launch_pdl(kern, dim3(sms), GThreads, smem, st, p, cgu, zgu, cd, zd));
    EDG_CUDA_TRY(launch_sum_choices(g, st));
    return EDG_OK;
}

cudaError_t launch_sum_choices(const GroupedParams& g, cudaStream_t st) {
    SumArgs sa{g.o, g.pair_slot, g.y, g.T, g.H, g.K};
    const dim3 grid((unsigned)(((size_t)g.T * g.H / 4 + 255) / 256));
    if (g.out_dtype == EDG_F32) return launch_pdl(sum_choices_kernel<float>, grid, 256, 0, st, sa);
    if (g.out_dtype == EDG_F16) return launch_pdl(sum_choices_kernel<__half>, grid, 256, 0, st, sa);
    return launch_pdl(sum_choices_kernel<bf16_t>, grid, 256, 0, st, sa);
}

}  // namespace edg
