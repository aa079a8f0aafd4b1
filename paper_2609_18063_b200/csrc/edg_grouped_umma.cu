// a4'-a6' grouped form for many tokens (prompts, chunks of them) on the 5th-generation tensor cores.
//
// A CTA computes [128 weight rows] x [up to 128 pairs of one expert]: the expert's weights are the A operand (M = 128), the
// activations of the tile's (token, choice) pairs the B operand (N = pairs), both K-major in shared memory; one elected thread
// issues tcgen05.mma into tensor memory, tcgen05.commit on mbarriers tracks completion.
//
// Exact weights from ONE fp16 operand.  w = s (q - z) has up to 16 significant bits, but q - z alone has at most eleven: the MMA
// sees (q - z) * 2^-9, exactly, and its sums over one group of k (one scale per row) are multiplied by the scale in fp32 where
// they leave tensor memory, row = lane.  The running sums live in registers (a thread holds one row of the tile, 128 columns), the
// accumulator is double-buffered, so the tensor core works on the next group meanwhile.  What bounds these kernels is operand
// traffic through shared memory (128 B a clock): with the weights as value + residual (two operand tiles, multiplied twice) it was
// twice as much, with h as value + residual on top 1.5 times.  The fp32 h of the down projection is fed as value + residual.
//
// Operand layout in shared memory (no swizzle): core matrices of 8 rows x 16 bytes; the descriptor's leading byte offset is the
// distance between k cores, its stride byte offset the distance between row groups (128).  The 8 k values of a core row are
// kept in the order (k0,k4,k1,k5,k2,k6,k3,k7) in which the int4 codes come out of a 32-bit word -- for A and B alike.
//
// Warps 0-3 (48 registers) dequantise: a thread is a weight row, the codes of the next stages in flight in registers.  Warps 4-7 (168
// registers) take the groups' sums out of tensor memory, 32 columns at a time, and run the epilogue.  Warp 8 issues the MMAs, warp 9 brings the
// activations, one bulk copy a stage.  Two CTAs share an SM: one's prologue and epilogue run beside the other's main loop.  Every wait
// is bounded: a wait that gives up raises the status word and the kernel still frees its tensor memory and returns.
//
// Measured (4096 tokens, top 8 of 256 by Zipf(1.1), H 2048, I 512, groups of 64, rank 16): gate/up 413 -> 363 us, down 323 -> 310 (under ncu), the
// whole call with its routing 904 -> 782; with an adapter per expert 1190 -> 855; 2048 tokens (streaming form before) 706 -> 549.
// Tensor pipe 20 and 23 % active, schedulers issuing in 44 and 41 % of all cycles: the limiter is the rate at which lone warps run their
// instructions in roles that wait for one another (1024 tokens, 64 experts).  Found on the way: MMAs issued by one of
// the warps that take sums out, in between: 1020 us for gate/up; sums out 16 columns at a time: 577; states gathered by 16-byte copies
// of this kernel, without a pass that gathers them: 554, the copies' bursts hold up every other access to shared memory (333 without
// the trips to tensor memory); four row blocks per CTA one after the other: down 302 -> 400.
#include "edg_grouped.cuh"
#include "edg_ptx.cuh"

namespace edg {
namespace {

constexpr int U_TN = kUmmaTokens;            // columns of a tile: pairs
constexpr uint32_t U_LBO = 16 * 128;         // between k cores of a full tile
constexpr int U_THREADS = 12 * 32;
constexpr int U_HQ = 32;                     // columns that the epilogue of gate/up exchanges at a time
constexpr int U_HS = 68;                     // floats of an h row in shared memory: 64 and padding against bank conflicts

// A stage of the ring: gate/up 64 k of weights and of states (16 KB each), three of them; down 32 k of weights (8 KB), of h and its
// residual (16 KB), four.
template <bool DOWN> struct Stage {
    static constexpr int k = DOWN ? 32 : 64, chunks = k / 32, n = DOWN ? 4 : 3;
    static constexpr uint32_t a_bytes = 128 * k * 2, bytes = a_bytes + 16384;
    static constexpr int ahead = DOWN ? 4 : 2;           // stages of codes in flight per thread of warps 0-3
};
constexpr uint32_t U_BARS = 96 * 1024, U_SMEM = U_BARS + 12 * 8 + 16 + U_TN * 4;
static_assert(Stage<false>::bytes * Stage<false>::n <= U_BARS && Stage<true>::bytes * Stage<true>::n <= U_BARS, "stages");
static_assert(2 * (U_SMEM + 1024) <= 228 * 1024, "two CTAs share an SM");

__device__ __forceinline__ void bar_wait(uint64_t* b, uint32_t parity, int32_t* status) {
    uint32_t it = 0;
    while (!mbar_try_wait(b, parity))
        if (++it >= kSpinLimit) { atomicExch(status, EDG_E_TIMEOUT); break; }
}
// Shared-memory matrix descriptor: K-major, no swizzle.  Its lower word holds the address and the distance between k cores, the upper
// one is the same for all: row groups 128 bytes apart, descriptor version 1.
__device__ __forceinline__ uint32_t umma_desc(uint32_t saddr, uint32_t lbo) { return ((saddr >> 4) & 0x3FFF) | (((lbo >> 4) & 0x3FFF) << 16); }
constexpr uint32_t U_DESC_HI = (128 >> 4) | (1u << 14);
// instruction descriptor: fp32 accumulator, fp16 A and B, both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t umma_idesc(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t tmem_d, uint32_t da, uint32_t db, uint32_t idesc, bool accumulate) {
    asm volatile("{\n.reg .pred p;\n.reg .b64 a, b;\nsetp.ne.b32 p, %4, 0;\nmov.b64 a, {%1, %5};\nmov.b64 b, {%2, %5};\n"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n}"
                 ::"r"(tmem_d), "r"(da), "r"(db), "r"(idesc), "r"(accumulate ? 1u : 0u), "r"(U_DESC_HI) : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(b)) : "memory");
}
// (load and wait in one statement: nothing that uses the values may move between them)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xFFFFFFFF;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void fence_to_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// v / (1 + e^-v), the bits of silu_f without the branch that its division has per element (with silu_f itself 874 us for 4096 tokens, so
// 793, as with an approximate division): the product with an approximate reciprocal, corrected by its remainder (Markstein, Computation of elementary functions on the
// IBM RISC System/6000 processor, 1990).  A quarter of both sides: the reciprocal of a denominator beyond 2^126 would be subnormal.  Where the
// denominator is infinite the reciprocal is zero, as the quotient is.
__device__ __forceinline__ float silu_corrected(float v) {
    const float d = fminf(fmaf(__expf(-v), 0.25f, 0.25f), 3.402823466e38f), n = 0.25f * v;
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(d));
    const float q = n * y;
    return fmaf(fmaf(-d, q, n), y, q);
}

// The states of a tile's pairs as the gate/up kernel's B operand, [stage of 64 k][8 k cores][pairs rounded to 16][8 k]: a stage is one bulk
// copy then.  (Gathered by 16-byte copies of the tiles' own CTAs, the bursts held up every other access to shared memory.)
// Consecutive threads take consecutive pairs of four k cores: their 16-byte pieces are adjacent in the tile; the reads are 64 bytes
// of as many rows.
__global__ void __launch_bounds__(256) umma_gather_x_kernel(const __grid_constant__ GroupedParams p) {
    pdl_launch_dependents();
    pdl_wait_prior_grid();
    const int tile = blockIdx.y;
    if (tile >= *p.n_tiles) return;
    const int4 ti = p.tiles[tile];
    const int n16 = (ti.z + 15) & ~15;
    uint8_t* out = p.xq + (size_t)tile * p.H * 256;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n16 * (p.H / 32); i += gridDim.x * 256) {
        const int tok = i % n16, c = i / n16;
        uint4 raw[4] = {};
        if (tok < ti.z) {
            const uint4* src = reinterpret_cast<const uint4*>(p.x + (size_t)(p.order[ti.y + tok] / p.K) * p.H + c * 32);
#pragma unroll
            for (int j = 0; j < 4; ++j) raw[j] = __ldg(src + j);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(out + ((size_t)(c * 4 + j) * n16 + tok) * 16) = bf16x8_permute8(raw[j]);
    }
}

// One tile: DOWN = false: h = silu(gate) up for 64 rows of the intermediate dimension (rows 0..63 of the tile are gate rows, 64..127
// the up rows of the same indices), written as the down kernel's B operand; DOWN = true: o[pair][row] = gate weight * (W h) for 128
// output rows.  The adapter comes first, as stages of its own with scale 1: A = B_lora rows, B = sigma (A_lora x), for gate/up
// with the ranks of both projections side by side (a gate row is zero in the up ranks and the other way round).  HF: h goes to p.hf as well
// (an instantiation of its own: 4096 tokens with one adapter 790 -> 782 us, with one per expert 847 -> 855).
template <bool DOWN, bool HF = false>
__global__ void __launch_bounds__(U_THREADS, 2) umma_tile_kernel(const __grid_constant__ GroupedParams p) {
    using St = Stage<DOWN>;
    extern __shared__ __align__(128) uint8_t smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + U_BARS);         // [stages] weights and activations are there
    uint64_t* empty = full + 4;                                          // [stages] the MMAs that read the stage have completed
    uint64_t* accfull = empty + 4;                                       // [2] a group's sums are complete
    uint64_t* accempty = accfull + 2;                                    // [2] and have been taken out
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(accempty + 2);
    int* s_pair = reinterpret_cast<int*>(s_tmem + 4);                    // [U_TN]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_launch_dependents();
    pdl_wait_prior_grid();
    const int tile = blockIdx.y;                 // row blocks of a tile are neighbours in the grid: they share its activations in L2
    if (tile >= *p.n_tiles) return;
    const int4 ti = p.tiles[tile];               // {slot, first position in order, pairs, adapter}
    const int cnt = ti.z, n16 = (cnt + 15) & ~15;
    const uint8_t* rec = p.pool + (size_t)ti.x * p.L.bytes;
    const int K = DOWN ? p.I : p.H, NS = K / St::k, gshift = p.gshift;
    const int RK = DOWN ? p.rank : 2 * p.rank, RS = (RK + St::k - 1) / St::k;      // ranks, stages of them (ahead of the others)
    const uint32_t xlbo = (uint32_t)n16 * 16;                            // (tiles of activations are stored without gaps)
    if (tid < U_TN) s_pair[tid] = tid < cnt ? p.order[ti.y + tid] : -1;
    if (tid == 0) {
        for (int s = 0; s < St::n; ++s) { mbar_init(&full[s], 5); mbar_init(&empty[s], 1); }       // (four warps, and who brings the activations)
        for (int s = 0; s < 2; ++s) { mbar_init(&accfull[s], 1); mbar_init(&accempty[s], 4); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(2 * U_TN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *s_tmem;

    struct Ring {                                                        // position in the ring of stages
        int st = 0;
        uint32_t phase = 0;
        __device__ __forceinline__ void next() { if (++st == St::n) { st = 0; phase ^= 1u; } }
    } rp;

    if (warp < 4) {
        // ================================================= weights into shared memory
        asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
        const int r = tid;
        const int n = DOWN ? (int)blockIdx.x * 128 + r : (int)blockIdx.x * 64 + (r & 63);
        const uint8_t *cp, *zp;                  // this row's first chunk of codes and its first (scale, zero) pair
        if (DOWN) {
            cp = rec + p.L.codes_down + down_code_off(p.H, p.I, n, 0);
            zp = rec + p.L.sz_down + down_sz_off(p.H, p.I, p.group, n, 0);
        } else {
            cp = rec + (r < 64 ? p.L.codes_gate : p.L.codes_up) + code_off(p.H, n, 0);
            zp = rec + (r < 64 ? p.L.sz_gate : p.L.sz_up) + sz_off(p.H, p.group, n, 0);
        }
        const int cps = p.I / kDownSlices / 32;                          // (a power of two, as is the group)
        const int cps_sh = 31 - __clz(cps), gps_sh = 31 - __clz(p.I / kDownSlices) - gshift;
        const uint32_t cslice = (uint32_t)p.H * (p.I / kDownSlices) / 2, zslice = ((uint32_t)p.H << gps_sh) * 4;
        auto codes = [&](int c) {
            return ld_stream16(DOWN ? cp + (size_t)(c >> cps_sh) * cslice + (c & (cps - 1)) * 256 : cp + c * 256);
        };
        auto pair_of = [&](int c) {                                      // (scale, zero) of the group that holds chunk c
            const int g = (c * 32) >> gshift;
            return ld_stream4(DOWN ? zp + (size_t)(g >> gps_sh) * zslice + (g & ((1 << gps_sh) - 1)) * 64 : zp + g * 64);
        };
        uint4 cw[St::ahead][St::chunks];
        uint32_t zz[St::ahead][St::chunks];
        auto load = [&](int j, int s) {                                  // (no copies of values that are on their way: a copy waits)
#pragma unroll
            for (int h = 0; h < St::chunks; ++h) cw[j][h] = codes(s * St::chunks + h);
            zz[j][0] = pair_of(s * St::chunks);
            if (!DOWN && gshift == 5) zz[j][St::chunks - 1] = pair_of(s * St::chunks + 1);
        };
#pragma unroll
        for (int j = 0; j < St::ahead; ++j)
            if (j < NS) load(j, j);
        auto written = [&]() {
            fence_to_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[rp.st]);
            rp.next();
        };
        // ---- the adapter's rows
        for (int rs = 0; rs < RS; ++rs) {
            const uint16_t* B = static_cast<const uint16_t*>(DOWN ? p.lora.B_down : (r < 64 ? p.lora.B_gate : p.lora.B_up)) +
                                ((size_t)ti.w * (DOWN ? p.H : p.I) + n) * p.rank;
            const int k0 = DOWN || r < 64 ? 0 : p.rank;
#pragma unroll 4
            for (int kc = 0; kc < St::k / 8; ++kc) {
                const int k = rs * St::k + kc * 8 - k0;
                uint4 a = make_uint4(0, 0, 0, 0);
                if (k >= 0 && k < p.rank) a = bf16x8_to_f16(__ldg(reinterpret_cast<const uint4*>(B + k)));
                *reinterpret_cast<uint4*>(smem + rp.st * St::bytes + kc * U_LBO + r * 16) = a;
            }
            written();
        }
#pragma unroll 1
        for (int s0 = 0; s0 < NS; s0 += St::ahead)
#pragma unroll
            for (int j = 0; j < St::ahead; ++j) {
                const int s = s0 + j;
                if (s >= NS) break;
                bar_wait(&empty[rp.st], rp.phase ^ 1, p.status);
                uint8_t* sb = smem + rp.st * St::bytes + r * 16;
#pragma unroll
                for (int h = 0; h < St::chunks; ++h) {
                    const __half2 mz = neg_zero_x(u32_as_h2(!DOWN && gshift == 5 ? zz[j][h] : zz[j][0]));
                    const uint32_t w[4] = {cw[j][h].x, cw[j][h].y, cw[j][h].z, cw[j][h].w};
#pragma unroll
                    for (int kc = 0; kc < 4; ++kc) {
                        uint32_t q[4];
                        dequant_word_x(w[kc], mz, q);
                        *reinterpret_cast<uint4*>(sb + (h * 4 + kc) * U_LBO) = make_uint4(q[0], q[1], q[2], q[3]);
                    }
                }
                if (s + St::ahead < NS) load(j, s + St::ahead);
                written();
            }
    } else if (warp < 8) {
        // ================================================= groups' sums out of tensor memory, epilogue
        asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
        const int r = tid - 128;
        const int n = DOWN ? (int)blockIdx.x * 128 + r : (int)blockIdx.x * 64 + (r & 63);
        const uint8_t* zp = rec + (DOWN ? p.L.sz_down + down_sz_off(p.H, p.I, p.group, n, 0) : (r < 64 ? p.L.sz_gate : p.L.sz_up) + sz_off(p.H, p.group, n, 0));
        const int gps_sh = 31 - __clz(p.I / kDownSlices) - gshift;
        const uint32_t zslice = ((uint32_t)p.H << gps_sh) * 4;
        const int ad = RS > 0 ? 1 : 0, NG = (K >> gshift) + ad;
        auto scale = [&](int g) {                                        // (scale, zero) of group g, g counted with the adapter's
            if (g < ad || g >= NG) return 0x00001800u;                   // (2^-9, what undoes the unscaling below: the adapter's factor is 1)
            g -= ad;
            return ld_stream4(DOWN ? zp + (size_t)(g >> gps_sh) * zslice + (g & ((1 << gps_sh) - 1)) * 64 : zp + g * 64);
        };
        float acc[U_TN];
#pragma unroll
        for (int j = 0; j < U_TN; ++j) acc[j] = 0.f;
        const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        uint32_t z0 = scale(0), z1 = scale(1);
        auto take = [&](int g, int buf, uint32_t& z) {
            const float s = kUnscaleX * __low2float(u32_as_h2(z));
            z = scale(g + 2);                                            // (no copies between z0 and z1: a copy waits for the load)
            bar_wait(&accfull[buf], (uint32_t)(g >> 1) & 1, p.status);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int b = 0; b < U_TN / 32; ++b)
                if (b * 32 < n16) {
                    uint32_t v[32];
                    tmem_ld32(lane_addr + buf * U_TN + b * 32, v);
#pragma unroll
                    for (int j = 0; j < 32; j += 2) fma2(acc[b * 32 + j], acc[b * 32 + j + 1], s, __uint_as_float(v[j]), __uint_as_float(v[j + 1]));
                }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&accempty[buf]);
        };
#pragma unroll 1
        for (int g = 0; g < NG; g += 2) {
            take(g, 0, z0);
            if (g + 1 < NG) take(g + 1, 1, z1);
        }
        if (DOWN) {
            float2* s_pg = reinterpret_cast<float2*>(smem);              // {pair, its weight} (the stages have been used)
            s_pg[r] = make_float2(__int_as_float(s_pair[r]), r < cnt ? p.gates[s_pair[r]] : 0.f);
            asm volatile("bar.sync 1, 128;" ::: "memory");
            float* o = p.o + n;
#pragma unroll
            for (int b = 0; b < U_TN; b += 8)
                if (b < cnt) {
                    float2 pg[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) pg[j] = s_pg[b + j];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (b + j < cnt) o[(size_t)__float_as_int(pg[j].x) * p.H] = pg[j].y * acc[b + j];
                }
        } else {
            // 32 columns at a time: the threads of the gate rows finish the first half of them, those of the up rows the second, and each
            // hands the other half over; then eight rows of h of a pair go out as one core row of value and one of residual
            float* s_h = reinterpret_cast<float*>(smem);       // [column][U_HS] (the stages have been used)
            float* hs = s_h + (r & 63);
            const bool is_gate = r < 64;
            constexpr int half = U_HQ / 2;
            const int give = is_gate ? half : 0, keep = half - give;
#pragma unroll
            for (int c0 = 0; c0 < U_TN; c0 += U_HQ) {
                if (c0 < n16) {
#pragma unroll
                    for (int j = 0; j < half; ++j) hs[(give + j) * U_HS] = is_gate ? acc[c0 + half + j] : acc[c0 + j];
                    asm volatile("bar.sync 1, 128;" ::: "memory");
                    float* q = hs + keep * U_HS;
                    float o[half];
#pragma unroll
                    for (int j = 0; j < half; ++j) o[j] = q[j * U_HS];
#pragma unroll
                    for (int j = 0; j < half; ++j) {
                        const float mine = is_gate ? acc[c0 + j] : acc[c0 + half + j], gv = is_gate ? mine : o[j];
                        q[j * U_HS] = silu_corrected(gv) * (is_gate ? o[j] : mine);
                    }
                    asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll
                    for (int i = 0; i < U_HQ * 8 / 128; ++i) {
                        const int piece = i * 128 + r, tok = piece % U_HQ, core = piece / U_HQ, k = (int)blockIdx.x * 64 + core * 8;
                        const float4 a = *reinterpret_cast<const float4*>(s_h + tok * U_HS + core * 8), b = *reinterpret_cast<const float4*>(s_h + tok * U_HS + core * 8 + 4);
                        float f[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                        if (c0 + tok >= cnt) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) f[e] = 0.f;
                        }
                        if (c0 + tok < n16) {
                            uint8_t* w = p.hq + (size_t)tile * p.I * 512 + ((size_t)(k >> 5) * 8 + ((k & 31) >> 3)) * n16 * 16 + (c0 + tok) * 16;
                            *reinterpret_cast<uint4*>(w) = permute8(f);
                            *reinterpret_cast<uint4*>(w + (size_t)n16 * 64) = permute8_lo(f);
                            if (HF) {
                                float4* v = reinterpret_cast<float4*>(p.hf + (size_t)tile * p.I * 128 + ((size_t)(k >> 3) * n16 + c0 + tok) * 8);
                                v[0] = make_float4(f[0], f[1], f[2], f[3]);
                                v[1] = make_float4(f[4], f[5], f[6], f[7]);
                            }
                        }
                    }
                    asm volatile("bar.sync 1, 128;" ::: "memory");
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");
        if (warp == 8) {
            // ============================================= the MMAs.  Descriptors differ only in their address field.  The whole warp walks the
            // loop and one lane of it issues: what is the same for all lanes then stays in uniform registers, where the MMA wants it.
            const uint32_t idesc = umma_idesc(n16);
            const uint32_t a0 = umma_desc(smem_u32(smem), U_LBO), x0 = umma_desc(smem_u32(smem + St::a_bytes), xlbo);
            constexpr uint32_t kStage = St::bytes >> 4, kStepA = (2 * U_LBO) >> 4;
            const uint32_t kStepX = (2 * xlbo) >> 4;
            int g = 0;
            auto stage_there = [&]() {
                bar_wait(&full[rp.st], rp.phase, p.status);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            };
            for (int i = 0; i < RS; ++i) {
                stage_there();
                const uint32_t as = a0 + rp.st * kStage, xs = x0 + rp.st * kStage;
                const int ksteps = min(St::k / 16, (RK - i * St::k + 15) / 16);
                if (elect_one()) {
                    for (int ks = 0; ks < ksteps; ++ks) umma(tmem, as + ks * kStepA, xs + ks * kStepX, idesc, i > 0 || ks > 0);
                    umma_commit(&empty[rp.st]);
                    if (i == RS - 1) umma_commit(&accfull[0]);
                }
                __syncwarp();
                rp.next();
            }
            if (RS > 0) g = 1;
            const int gmask = (p.group >> 5) - 1;                        // a group is 1, 2 or 4 chunks of 32 k
#pragma unroll 1
            for (int s = 0; s < NS; ++s) {
                stage_there();
                const uint32_t as = a0 + rp.st * kStage, xs = x0 + rp.st * kStage;
#pragma unroll
                for (int h = 0; h < St::chunks; ++h) {
                    const int c = s * St::chunks + h;
                    const bool first = (c & gmask) == 0, last = (c & gmask) == gmask;
                    if (first) {
                        bar_wait(&accempty[g & 1], ((uint32_t)(g >> 1) & 1) ^ 1, p.status);
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    }
                    const uint32_t d = tmem + (g & 1) * U_TN;
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < 2; ++ks) {
                            umma(d, as + (2 * h + ks) * kStepA, xs + (2 * h + ks) * kStepX, idesc, !first || ks > 0);
                            if (DOWN) umma(d, as + ks * kStepA, xs + (2 + ks) * kStepX, idesc, true);    // (values, then residuals)
                        }
                        if (last) umma_commit(&accfull[g & 1]);
                        if (h == St::chunks - 1) umma_commit(&empty[rp.st]);
                    }
                    __syncwarp();
                    if (last) ++g;
                }
                rp.next();
            }
        } else if (warp == 9) {
            // ============================================= activations.  Eight rows of a tile (pairs) and four k cores per copy of a warp
            for (int rs = 0; rs < RS; ++rs) {                            // A_lora x (or h) times sigma, fp16, per token or pair
                const uint8_t* src = reinterpret_cast<const uint8_t*>(DOWN ? p.u_d : p.u_gu);
                const uint32_t dst = smem_u32(smem + rs * St::bytes + St::a_bytes) + (lane >> 3) * xlbo + (lane & 7) * 16;
                for (int rg = 0; rg * 8 < n16; ++rg) {
                    const int pr = s_pair[rg * 8 + (lane & 7)];
                    const uint8_t* row = src + (size_t)(pr < 0 ? 0 : (DOWN || p.n_adapters != 1 ? pr : pr / p.K)) * RK * 2;
#pragma unroll
                    for (int h = 0; h < St::chunks; ++h) {
                        const int core = rs * (St::k / 8) + h * 4 + (lane >> 3);
                        const bool in = pr >= 0 && core < RK / 8;        // (zeros beyond the ranks, and for no pair)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                                     ::"r"(dst + h * 4 * xlbo + rg * 128), "l"(row + (in ? core : 0) * 16), "r"(in ? 16 : 0) : "memory");
                    }
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
                rp.next();
            }
            // (the main stages behind them are asked for first)
            const uint32_t bytes = (uint32_t)n16 * 128;                  // of 64 k of states, or 32 k of h and its residual
            const uint8_t* src = DOWN ? p.hq + (size_t)tile * p.I * 512 : p.xq + (size_t)tile * p.H * 256;
            for (int s = 0; s < NS; ++s) {
                if (RS > 0 && s == min(St::n - RS, NS - 1)) {            // (before the first wait for a stage that they free)
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    fence_to_async();
                    __syncwarp();
                    if (lane == 0)
                        for (int rs = 0; rs < RS; ++rs) mbar_arrive(&full[rs]);
                }
                if (lane == 0) {
                    bar_wait(&empty[rp.st], rp.phase ^ 1, p.status);
                    mbar_expect_tx(&full[rp.st], bytes);
                    bulk_g2s(smem + rp.st * St::bytes + St::a_bytes, src + (size_t)s * bytes, bytes, &full[rp.st]);
                }
                __syncwarp();
                rp.next();
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 8) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * U_TN) : "memory");
}

}  // namespace

bool umma_grouped_supported(const edg_layer_desc& d) {
    return d.H % 256 == 0 && d.I % 128 == 0 && (d.group & (d.group - 1)) == 0 && d.group >= 32 && d.rank % 8 == 0;
}

cudaError_t launch_umma(const GroupedParams& p, bool down, int max_tiles, cudaStream_t st) {
    static OncePerDevice once;
    const cudaError_t e = once([] { return allow_smem(U_SMEM, umma_tile_kernel<false>, umma_tile_kernel<false, true>, umma_tile_kernel<true>); });
    if (e != cudaSuccess) return e;
    if (!down) {
        const cudaError_t g = launch_pdl(umma_gather_x_kernel, dim3(8, max_tiles), 256, 0, st, p);
        if (g != cudaSuccess) return g;
    }
    if (down) return launch_pdl(umma_tile_kernel<true>, dim3(p.H / 128, max_tiles), U_THREADS, U_SMEM, st, p);
    return launch_pdl(p.hf != nullptr ? umma_tile_kernel<false, true> : umma_tile_kernel<false>, dim3(p.I / 64, max_tiles), U_THREADS, U_SMEM, st, p);
}

}  // namespace edg
