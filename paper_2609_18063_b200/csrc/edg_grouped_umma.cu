// a4'-a6' grouped form for large token groups (prefill) on the 5th-generation tensor cores.
//
// A CTA computes a tile [128 weight rows] x [up to 128 tokens of one expert]: the expert's weights are
// the A operand (M = 128), the gathered token states the B operand (N = tokens), both K-major in shared
// memory; tcgen05.mma accumulates in tensor memory (fp32), one elected thread issues, completion is
// tracked by tcgen05.commit on mbarriers, and the epilogue reads the accumulators with tcgen05.ld.
//
// Exact weights from fp16 operands.  w = s * (q - z) has up to 16 significant bits (11 of the fp16
// scale, 5 of the integer), one fp16 cannot hold it, and rounding it costs more than the parity bar
// allows.  So every weight is fed as two fp16 values: hi = fp16(s (q - z)) and the residual
// lo = s (q - z) - hi, which is exact (an fma computes it without rounding); the tile is multiplied
// twice into the same accumulator.  The bf16 activations convert to fp16 exactly; the fp32 h of the
// down projection is fed as an fp16 value plus an fp16 residual (hi.hi + lo.hi + hi.lo).
//
// Operand layout in shared memory (no swizzle): core matrices of 8 rows x 16 bytes, a [128 x 32] fp16
// tile being [k core 0..3][row group 0..15][8 rows][16 B]; the descriptor's leading byte offset is the
// distance between k cores (2048), its stride byte offset the distance between row groups (128).
// The 8 k values of a core row are kept in the order (k0,k4,k1,k5,k2,k6,k3,k7) in which the int4 codes
// come out of a 32-bit word -- for A and B alike, so the dot product is unchanged.
//
// Warps 0-7 dequantise the weights into a ring of two stages, with the codes of the next four chunks in flight in registers, and
// later run the epilogue (each warp its 32 lanes of tensor memory, half of the token columns); warp 8 allocates the tensor memory
// and its lane 0 issues the MMAs; lane 0 of warp 9 fetches the activations into a ring of their own.
// Every wait is bounded: a wait that gives up raises the status word and the kernel still frees its
// tensor memory and returns.
#include "edg_grouped.cuh"

namespace edg {
namespace {

constexpr int U_TN = kUmmaTokens;            // token columns per tile
constexpr int U_KC = 32;                     // k per stage
constexpr int U_STAGES = 2;                  // of weights: four operand tiles each
constexpr int U_ACT_MAX = 4;                 // slots of activations
constexpr int U_AHEAD = 4;                   // chunks of codes in flight per thread
constexpr uint32_t U_TILE = 128 * U_KC * 2;  // bytes of a [128 x 32] fp16 operand tile
constexpr uint32_t U_LBO = 16 * 128;         // between k cores
constexpr uint32_t U_SBO = 128;              // between row groups
constexpr uint32_t U_SPIN = 1u << 22;
constexpr int U_PROD_WARPS = 8;
constexpr int U_THREADS = (U_PROD_WARPS + 2) * 32;

__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s32(b)) : "memory");
}
__device__ __forceinline__ void bar_wait(uint64_t* b, uint32_t parity, int32_t* status) {
    uint32_t ok = 0, it = 0;
    while (!ok && ++it < U_SPIN)
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                     : "=r"(ok) : "r"(s32(b)), "r"(parity) : "memory");
    if (!ok) atomicExch(status, EDG_E_TIMEOUT);
}
// shared-memory matrix descriptor: K-major, no swizzle
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((U_LBO >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((U_SBO >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
// instruction descriptor: fp32 accumulator, fp16 A and B, both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t umma_idesc(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, bool accumulate) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate ? 1u : 0u) : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s32(b)) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                   "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                   "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(taddr));
}

// offset of (row r, k core kc) inside an operand tile
__device__ __forceinline__ uint32_t core_off(int r, int kc) { return (uint32_t)(((kc * 16 + (r >> 3)) * 8 + (r & 7)) * 16); }

// One 32-bit word = 8 codes of a row -> the core row of s (q - z): fp16 value and exact fp16 residual.
__device__ __forceinline__ void dequant_hi_lo(uint32_t w, __half2 s2, __half2 z2, uint4& hi, uint4& lo) {
    uint32_t q[4];
    dequant_word(w, z2, q);                              // (q - z): (k0,k4) (k1,k5) (k2,k6) (k3,k7)
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __half2 qz = u32_as_h2(q[i]);
        const __half2 a = __hmul2(s2, qz);
        h[i] = h2_as_u32(a);
        l[i] = h2_as_u32(__hfma2(s2, qz, __hneg2(a)));
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// 8 bf16 -> 8 fp16 in natural order (adapter matrices)
__device__ __forceinline__ uint4 bf16x8_to_f16(uint4 v) {
    uint4 o;
    o.x = h2_as_u32(__floats2half2_rn(bf16_lo(v.x), bf16_hi(v.x)));
    o.y = h2_as_u32(__floats2half2_rn(bf16_lo(v.y), bf16_hi(v.y)));
    o.z = h2_as_u32(__floats2half2_rn(bf16_lo(v.z), bf16_hi(v.z)));
    o.w = h2_as_u32(__floats2half2_rn(bf16_lo(v.w), bf16_hi(v.w)));
    return o;
}
// 8 fp32 * sigma -> 8 fp16 in natural order; missing entries (j >= n) are zero
__device__ __forceinline__ uint4 f32x8_to_f16(const float* src, int n, float sigma) {
    float f[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) f[j] = (src != nullptr && j < n) ? sigma * src[j] : 0.f;
    uint4 o;
    o.x = h2_as_u32(__floats2half2_rn(f[0], f[1]));
    o.y = h2_as_u32(__floats2half2_rn(f[2], f[3]));
    o.z = h2_as_u32(__floats2half2_rn(f[4], f[5]));
    o.w = h2_as_u32(__floats2half2_rn(f[6], f[7]));
    return o;
}

struct UmmaSmem {
    uint8_t* stage;     // [U_STAGES][4 tiles]
    uint8_t* act;       // [slots of activations]
    uint64_t* full;     // [stages] weights written (one arrival per producer warp)
    uint64_t* empty;    // [stages] MMAs that read the stage have completed
    uint64_t* afull;    // [slots] activations arrived
    uint64_t* aempty;   // [slots] MMAs that read the slot have completed
    uint64_t* done;     // all MMAs of the tile have completed
    uint32_t* tptr;
    int* pair;          // [U_TN]
};
__device__ __forceinline__ UmmaSmem carve(uint8_t* smem, uint32_t act_bytes) {
    UmmaSmem S;
    S.stage = smem;
    S.act = smem + U_STAGES * 4 * U_TILE;
    S.full = reinterpret_cast<uint64_t*>(S.act + act_bytes);
    S.empty = S.full + U_STAGES;
    S.afull = S.empty + U_STAGES;
    S.aempty = S.afull + U_ACT_MAX;
    S.done = S.aempty + U_ACT_MAX;
    S.tptr = reinterpret_cast<uint32_t*>(S.done + 1);
    S.pair = reinterpret_cast<int*>(S.tptr + 2);
    return S;
}
// gate/up: x, 8 KB a chunk, four slots; down: h and its residual, 16 KB a chunk, three slots.  Two CTAs fit an SM either way.
constexpr int U_ACT_GU = 4, U_ACT_D = 3;
constexpr uint32_t U_ACT_GU_BYTES = U_ACT_GU * U_TILE, U_ACT_D_BYTES = U_ACT_D * 2 * U_TILE;
constexpr size_t umma_smem_bytes(uint32_t act_bytes) { return (size_t)U_STAGES * 4 * U_TILE + act_bytes + 128 + U_TN * 4; }

// common prologue: pair list, barriers, tensor memory
__device__ __forceinline__ uint32_t umma_begin(const GroupedParams& p, const UmmaSmem& S, int slot, int first, int cnt, int cols) {
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid < U_TN) S.pair[tid] = tid < cnt ? p.lists[(size_t)slot * p.T + first + tid] : -1;
    if (tid == 0) {
        for (int s = 0; s < U_STAGES; ++s) { bar_init(&S.full[s], U_PROD_WARPS); bar_init(&S.empty[s], 1); }
        for (int s = 0; s < U_ACT_MAX; ++s) { bar_init(&S.afull[s], 1); bar_init(&S.aempty[s], 1); }
        bar_init(S.done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == U_PROD_WARPS) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(S.tptr)), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return *S.tptr;
}
__device__ __forceinline__ void umma_end(uint32_t tmem, int cols) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if ((threadIdx.x >> 5) == U_PROD_WARPS)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}
// lane 0 of the copy warp: the activations of every chunk, as slots become free
__device__ __forceinline__ void fetch_activations(const UmmaSmem& S, const uint8_t* src, int n_chunks, int slots, uint32_t bytes, int32_t* status) {
    for (int c = 0; c < n_chunks; ++c) {
        const int sl = c % slots;
        bar_wait(&S.aempty[sl], ((uint32_t)(c / slots) & 1) ^ 1, status);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s32(&S.afull[sl])), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(s32(S.act + sl * bytes)), "l"(src + (size_t)c * bytes), "r"(bytes), "r"(s32(&S.afull[sl])) : "memory");
    }
}
// a producer warp has written its part of a stage
__device__ __forceinline__ void stage_written(uint64_t* full) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // generic-proxy writes -> visible to the tensor core
    __syncwarp();
    if ((threadIdx.x & 31) == 0) bar_arrive(full);
}

// A producer thread: row r of the two operand tiles at `tile` of every stage, from 32 codes a chunk.  The loads run four chunks
// ahead: with one, a chunk took as long as a load from memory.
template <typename LC, typename LZ>
__device__ __forceinline__ void produce(const UmmaSmem& S, int n_chunks, int gshift, int tile, int r, LC codes, LZ sz, int32_t* status) {
    uint4 cw[U_AHEAD];
    uint32_t nz[U_AHEAD];
    auto starts = [&](int c) { return ((c * U_KC) & ((1 << gshift) - 1)) == 0; };      // a group of k begins with chunk c
#pragma unroll
    for (int j = 0; j < U_AHEAD; ++j) {                                  // (the chunks are a multiple of four)
        cw[j] = codes(j);
        nz[j] = starts(j) ? sz((j * U_KC) >> gshift) : 0u;
    }
    __half2 sc = __float2half2_rn(0.f), zr = sc;
    for (int c0 = 0; c0 < n_chunks; c0 += U_AHEAD)
#pragma unroll
        for (int j = 0; j < U_AHEAD; ++j) {
            const int c = c0 + j, st = c % U_STAGES;
            const uint32_t w[4] = {cw[j].x, cw[j].y, cw[j].z, cw[j].w};
            if (starts(c)) {
                const __half2 a = u32_as_h2(nz[j]);
                sc = __low2half2(a); zr = __high2half2(a);
            }
            if (c + U_AHEAD < n_chunks) {
                cw[j] = codes(c + U_AHEAD);
                if (starts(c + U_AHEAD)) nz[j] = sz(((c + U_AHEAD) * U_KC) >> gshift);
            }
            bar_wait(&S.empty[st], ((uint32_t)(c / U_STAGES) & 1) ^ 1, status);        // the MMAs that read this stage are done
            uint8_t* sb = S.stage + (st * 4 + tile) * U_TILE;
#pragma unroll
            for (int kc = 0; kc < 4; ++kc) {
                uint4 hi, lo;
                dequant_hi_lo(w[kc], sc, zr, hi, lo);
                *reinterpret_cast<uint4*>(sb + core_off(r, kc)) = hi;
                *reinterpret_cast<uint4*>(sb + U_TILE + core_off(r, kc)) = lo;
            }
            stage_written(&S.full[st]);
        }
}

// ---------------------------------------------------------------- token states as operand tiles
// xq[tile][chunk of 32 k][128 tokens x 32 k]: thread = (token of the tile, k core); the four row blocks
// of a tile then fetch every chunk with one bulk copy instead of gathering it again.
__global__ void __launch_bounds__(256) umma_gather_x_kernel(GroupedParams p) {
    const int tile = blockIdx.y;
    if (tile >= *p.n_tiles) return;
    const int slot = p.tiles[2 * tile], first = p.tiles[2 * tile + 1];
    const int cnt = min(U_TN, p.counts[slot] - first);
    const int cores = p.H / 8;                                   // 16-byte pieces per token
    uint8_t* out = p.xq + (size_t)tile * (p.H / 32) * U_TILE;
    // consecutive threads take consecutive tokens of four k cores: their 16-byte pieces are adjacent in the operand tile (coalesced
    // writes); the reads are 64 bytes from 128 different rows (one k core at a time, half of every 32-byte sector came in vain:
    // 64 us for 4096 tokens of 8 choices, now 55)
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < U_TN * (cores / 4); i += gridDim.x * blockDim.x) {
        const int tok = i % U_TN, c = i / U_TN;
        uint4 raw[4] = {};
        if (tok < cnt) {
            const int pair = p.lists[(size_t)slot * p.T + first + tok];
            const uint4* src = reinterpret_cast<const uint4*>(p.x + (size_t)(pair / p.K) * p.H + c * 32);
#pragma unroll
            for (int j = 0; j < 4; ++j) raw[j] = src[j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float f[8] = {bf16_lo(raw[j].x), bf16_hi(raw[j].x), bf16_lo(raw[j].y), bf16_hi(raw[j].y),
                                bf16_lo(raw[j].z), bf16_hi(raw[j].z), bf16_lo(raw[j].w), bf16_hi(raw[j].w)};
            *reinterpret_cast<uint4*>(out + (size_t)c * U_TILE + core_off(tok, j)) = permute8(f);
        }
    }
}

// ---------------------------------------------------------------- gate/up
// stage = [gate hi][gate lo][up hi][up lo], x in slots of its own (one bulk copy per chunk); tensor memory: gate in
// columns 0..127, up in 128..255.  Thread t dequantises row t % 128 of gate (t < 128) or up.
__global__ void __launch_bounds__(U_THREADS, 2) umma_gate_up_kernel(GroupedParams p) {
    const int tile = blockIdx.y;             // row blocks of a tile are neighbours in the grid: they share its activations in L2
    if (tile >= *p.n_tiles) return;
    extern __shared__ __align__(128) uint8_t smem[];
    const UmmaSmem S = carve(smem, U_ACT_GU_BYTES);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int slot = p.tiles[2 * tile], first = p.tiles[2 * tile + 1];
    const int cnt = min(U_TN, p.counts[slot] - first);
    const int row0 = blockIdx.x * 128;
    const uint8_t* rec = p.pool + (size_t)slot * p.L.bytes;
    const uint32_t tmem = umma_begin(p, S, slot, first, cnt, 2 * U_TN);
    const int n_chunks = p.H / U_KC;
    const int r_chunks = p.rank > 0 ? (p.rank + 31) / 32 : 0;          // adapter: chunks of up to 32 ranks
    const int gshift = 31 - __clz(p.group);

    if (warp < U_PROD_WARPS) {
        const int r = tid & 127, half = tid >> 7;                    // weight row; matrix (0 gate, 1 up) and, in the epilogue, half of the columns
        const int pair = S.pair[r];
        const uint8_t* cp = rec + (half ? p.L.codes_up : p.L.codes_gate);
        const uint8_t* zp = rec + (half ? p.L.sz_up : p.L.sz_gate);
        produce(S, n_chunks, gshift, 2 * half, r, [&](int c) { return ld_stream16(cp + code_off(p.H, row0 + r, c)); },
                [&](int g) { return ld_stream4(zp + sz_off(p.H, p.group, row0 + r, g)); }, p.status);
        // the adapter as extra k: A = B_gate / B_up rows (fp16 of bf16), B = sigma * (A_gate x) / sigma * (A_up x);
        // the threads of matrix m write its A rows and its B rows (gate's B in tile 3, up's in tile 1)
        if (r_chunks > 0) {
            const int first_pair = S.pair[0];
            const int ad = first_pair >= 0 ? p.pair_ad[first_pair] : 0;
            const int n_sets = p.n_adapters == 1 ? 1 : p.K;
            const float* um = nullptr;
            if (pair >= 0) um = p.u_gu + (((size_t)(pair / p.K) * n_sets + (p.n_adapters == 1 ? 0 : pair % p.K)) * 2 + half) * p.rank;
            const uint16_t* Bm = reinterpret_cast<const uint16_t*>(half ? p.lora.B_up : p.lora.B_gate) + ((size_t)ad * p.I + row0 + r) * p.rank;
            for (int rc = 0; rc < r_chunks; ++rc) {
                const int c = n_chunks + rc, st = c % U_STAGES;
                const uint32_t use = (uint32_t)(c / U_STAGES);
                bar_wait(&S.empty[st], (use & 1) ^ 1, p.status);
                uint8_t* sb = S.stage + st * 4 * U_TILE;
#pragma unroll
                for (int kc = 0; kc < 4; ++kc) {
                    const int j0 = rc * 32 + kc * 8, n = p.rank - j0;          // rank is a multiple of 8
                    uint4 a = make_uint4(0, 0, 0, 0);
                    if (n > 0) a = bf16x8_to_f16(*reinterpret_cast<const uint4*>(Bm + j0));
                    *reinterpret_cast<uint4*>(sb + (2 * half) * U_TILE + core_off(r, kc)) = a;
                    *reinterpret_cast<uint4*>(sb + (half ? 1 : 3) * U_TILE + core_off(r, kc)) = f32x8_to_f16(um != nullptr ? um + j0 : nullptr, n, p.sigma);
                }
                stage_written(&S.full[st]);
            }
        }
        // ---- epilogue: h = silu(gate) * up, thread = weight row, 32 token columns at a time
        bar_wait(S.done, 0, p.status);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        for (int c0 = half * (U_TN / 2); c0 < min(cnt, (half + 1) * (U_TN / 2)); c0 += 32) {
            uint32_t g[32], u[32];
            tmem_ld32(lane_addr + c0, g);
            tmem_ld32(lane_addr + U_TN + c0, u);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            // h goes out twice: fp32 per pair (for the down adapter's projection), and as the down
            // kernel's B operand: fp16 value and fp16 residual in operand-tile order, this row being k
            // index i = row0 + r of the tile's chunk i / 32 (k core (i % 32) / 8, slot of i % 8 in the
            // (k0,k4,k1,k5,k2,k6,k3,k7) order)
            const int i = row0 + r, e = i & 7;
            uint8_t* hq = p.hq + ((size_t)tile * (p.I / 32) + (i >> 5)) * 2 * U_TILE + (size_t)((e < 4 ? 2 * e : 2 * (e - 4) + 1) * 2);
            const int kc = (i & 31) >> 3;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const int pr = (c0 + j) < cnt ? S.pair[c0 + j] : -1;
                if (pr >= 0) {
                    const float hv = silu_f(__uint_as_float(g[j])) * __uint_as_float(u[j]);
                    p.h[(size_t)pr * p.I + i] = hv;
                    const __half hh = __float2half_rn(hv);
                    const __half hl = __float2half_rn(hv - __half2float(hh));
                    *reinterpret_cast<__half*>(hq + core_off(c0 + j, kc)) = hh;
                    *reinterpret_cast<__half*>(hq + U_TILE + core_off(c0 + j, kc)) = hl;
                }
            }
        }
    } else if (warp == U_PROD_WARPS + 1) {
        if (lane == 0) fetch_activations(S, p.xq + (size_t)tile * (p.H / 32) * U_TILE, n_chunks, U_ACT_GU, U_TILE, p.status);
    } else if (lane == 0) {
        // ---- the MMA issuer.  Descriptors differ only in their address field: base + offset >> 4.
        const uint32_t idesc = umma_idesc((cnt + 15) & ~15);
        const uint64_t d0 = umma_desc(s32(S.stage)), a0 = umma_desc(s32(S.act));
        constexpr uint64_t kTile = U_TILE >> 4, kStep = (2 * U_LBO) >> 4, kStage = (4 * U_TILE) >> 4;
        const uint32_t tg = tmem, tu = tmem + U_TN;
        for (int c = 0; c < n_chunks; ++c) {
            const int st = c % U_STAGES, sl = c % U_ACT_GU;
            bar_wait(&S.full[st], (uint32_t)(c / U_STAGES) & 1, p.status);
            bar_wait(&S.afull[sl], (uint32_t)(c / U_ACT_GU) & 1, p.status);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t ds = d0 + st * kStage, as = a0 + sl * kTile;
#pragma unroll
            for (int ks = 0; ks < U_KC / 16; ++ks) {
                const uint64_t dk = ds + ks * kStep, db = as + ks * kStep;
                umma(tg, dk, db, idesc, c > 0 || ks > 0);
                umma(tg, dk + kTile, db, idesc, true);
                umma(tu, dk + 2 * kTile, db, idesc, c > 0 || ks > 0);
                umma(tu, dk + 3 * kTile, db, idesc, true);
            }
            umma_commit(&S.empty[st]);
            umma_commit(&S.aempty[sl]);
        }
        for (int rc = 0; rc < r_chunks; ++rc) {
            const int c = n_chunks + rc, st = c % U_STAGES;
            bar_wait(&S.full[st], (uint32_t)(c / U_STAGES) & 1, p.status);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t ds = d0 + st * kStage;
            const int ksteps = min(2, (p.rank - rc * 32 + 15) / 16);
            for (int ks = 0; ks < ksteps; ++ks) {
                const uint64_t dk = ds + ks * kStep;
                umma(tg, dk, dk + 3 * kTile, idesc, true);
                umma(tu, dk + 2 * kTile, dk + kTile, idesc, true);
            }
            umma_commit(&S.empty[st]);
        }
        umma_commit(S.done);
    }
    umma_end(tmem, 2 * U_TN);
}

// ---------------------------------------------------------------- down
// A CTA covers 256 output rows (two accumulators of 128 columns in tensor memory) for the tile's tokens:
// stage = [W0 hi][W0 lo][W1 hi][W1 lo], thread t dequantising row t of the 256; [h hi][h lo] in slots of their own, one bulk copy
// per chunk (written in operand order by the gate/up kernel).
// o = gate weight * (W h + sigma B (A h))
__global__ void __launch_bounds__(U_THREADS, 2) umma_down_kernel(GroupedParams p) {
    const int tile = blockIdx.y;             // row blocks of a tile are neighbours in the grid: they share its activations in L2
    if (tile >= *p.n_tiles) return;
    extern __shared__ __align__(128) uint8_t smem[];
    const UmmaSmem S = carve(smem, U_ACT_D_BYTES);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int slot = p.tiles[2 * tile], first = p.tiles[2 * tile + 1];
    const int cnt = min(U_TN, p.counts[slot] - first);
    const int row0 = blockIdx.x * 256;
    const uint8_t* rec = p.pool + (size_t)slot * p.L.bytes;
    const uint32_t tmem = umma_begin(p, S, slot, first, cnt, 2 * U_TN);
    const int n_chunks = p.I / U_KC;
    const int r_chunks = p.rank > 0 ? (p.rank + 31) / 32 : 0;
    const int gshift = 31 - __clz(p.group);

    if (warp < U_PROD_WARPS) {
        const int r = tid & 127, m = tid >> 7;                       // row r of half m: output row row0 + tid
        const uint8_t* cdp = rec + p.L.codes_down;
        const float my_gate = m == 0 && S.pair[r] >= 0 ? p.gates[S.pair[r]] : 0.f;
        produce(S, n_chunks, gshift, 2 * m, r, [&](int c) { return ld_stream16(cdp + down_code_off(p.H, p.I, row0 + tid, c)); },
                [&](int g) { return ld_stream4(rec + p.L.sz_down + down_sz_off(p.H, p.I, p.group, row0 + tid, g)); }, p.status);
        if (r_chunks > 0) {
            const int first_pair = S.pair[0];
            const int ad = first_pair >= 0 ? p.pair_ad[first_pair] : 0;
            const int pair = S.pair[r];
            const float* ud = (m == 0 && pair >= 0) ? p.u_d + (size_t)pair * p.rank : nullptr;
            const uint16_t* Bd = reinterpret_cast<const uint16_t*>(p.lora.B_down) + ((size_t)ad * p.H + row0 + tid) * p.rank;
            for (int rc = 0; rc < r_chunks; ++rc) {
                const int c = n_chunks + rc, st = c % U_STAGES;
                const uint32_t use = (uint32_t)(c / U_STAGES);
                bar_wait(&S.empty[st], (use & 1) ^ 1, p.status);
                uint8_t* sb = S.stage + st * 4 * U_TILE;
#pragma unroll
                for (int kc = 0; kc < 4; ++kc) {
                    const int j0 = rc * 32 + kc * 8, n = p.rank - j0;
                    uint4 a = make_uint4(0, 0, 0, 0);
                    if (n > 0) a = bf16x8_to_f16(*reinterpret_cast<const uint4*>(Bd + j0));
                    *reinterpret_cast<uint4*>(sb + (2 * m) * U_TILE + core_off(r, kc)) = a;
                    if (m == 0) *reinterpret_cast<uint4*>(sb + U_TILE + core_off(r, kc)) = f32x8_to_f16(ud != nullptr ? ud + j0 : nullptr, n, p.sigma);
                }
                stage_written(&S.full[st]);
            }
        }
        // ---- epilogue: o[pair][row] = gate weight * acc; thread t = row t, accumulator t / 128
        bar_wait(S.done, 0, p.status);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float* gate = reinterpret_cast<float*>(S.act);               // (the activations have been used)
        if (m == 0) gate[r] = my_gate;
        asm volatile("bar.sync 1, %0;" ::"n"(U_PROD_WARPS * 32) : "memory");
        const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + m * U_TN;
        for (int c0 = 0; c0 < cnt; c0 += 32) {
            uint32_t v[32];
            tmem_ld32(lane_addr + c0, v);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const int pr = (c0 + j) < cnt ? S.pair[c0 + j] : -1;
                if (pr >= 0) p.o[(size_t)pr * p.H + row0 + tid] = gate[c0 + j] * __uint_as_float(v[j]);
            }
        }
    } else if (warp == U_PROD_WARPS + 1) {
        if (lane == 0) fetch_activations(S, p.hq + (size_t)tile * (p.I / 32) * 2 * U_TILE, n_chunks, U_ACT_D, 2 * U_TILE, p.status);
    } else if (lane == 0) {
        const uint32_t idesc = umma_idesc((cnt + 15) & ~15);
        const uint64_t d0 = umma_desc(s32(S.stage)), a0 = umma_desc(s32(S.act));
        constexpr uint64_t kTile = U_TILE >> 4, kStep = (2 * U_LBO) >> 4, kStage = (4 * U_TILE) >> 4;
        for (int c = 0; c < n_chunks; ++c) {
            const int st = c % U_STAGES, sl = c % U_ACT_D;
            bar_wait(&S.full[st], (uint32_t)(c / U_STAGES) & 1, p.status);
            bar_wait(&S.afull[sl], (uint32_t)(c / U_ACT_D) & 1, p.status);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t ds = d0 + st * kStage, as = a0 + sl * 2 * kTile;
#pragma unroll
            for (int ks = 0; ks < U_KC / 16; ++ks) {
                const uint64_t w0 = ds + ks * kStep, hhi = as + ks * kStep;
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const uint64_t whi = w0 + 2 * m * kTile;
                    umma(tmem + m * U_TN, whi, hhi, idesc, c > 0 || ks > 0);
                    umma(tmem + m * U_TN, whi + kTile, hhi, idesc, true);
                    umma(tmem + m * U_TN, whi, hhi + kTile, idesc, true);
                }
            }
            umma_commit(&S.empty[st]);
            umma_commit(&S.aempty[sl]);
        }
        for (int rc = 0; rc < r_chunks; ++rc) {
            const int c = n_chunks + rc, st = c % U_STAGES;
            bar_wait(&S.full[st], (uint32_t)(c / U_STAGES) & 1, p.status);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t ds = d0 + st * kStage;
            const int ksteps = min(2, (p.rank - rc * 32 + 15) / 16);
            for (int ks = 0; ks < ksteps; ++ks) {
                const uint64_t w0 = ds + ks * kStep;
                umma(tmem, w0, w0 + kTile, idesc, true);
                umma(tmem + U_TN, w0 + 2 * kTile, w0 + kTile, idesc, true);
            }
            umma_commit(&S.empty[st]);
        }
        umma_commit(S.done);
    }
    umma_end(tmem, 2 * U_TN);
}

}  // namespace

bool umma_grouped_supported(const edg_layer_desc& d) {
    return d.H % 256 == 0 && d.I % 128 == 0 && (d.group & (d.group - 1)) == 0 && d.group >= 32 && d.rank % 8 == 0;
}

cudaError_t launch_umma_gate_up(const GroupedParams& p, int max_tiles, cudaStream_t st) {
    static OncePerDevice once;
    const cudaError_t e = once([] { return allow_smem(umma_smem_bytes(U_ACT_GU_BYTES), umma_gate_up_kernel); });
    if (e != cudaSuccess) return e;
    umma_gather_x_kernel<<<dim3(8, max_tiles), 256, 0, st>>>(p);
    umma_gate_up_kernel<<<dim3(p.I / 128, max_tiles), U_THREADS, umma_smem_bytes(U_ACT_GU_BYTES), st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_umma_down(const GroupedParams& p, int max_tiles, cudaStream_t st) {
    static OncePerDevice once;
    const cudaError_t e = once([] { return allow_smem(umma_smem_bytes(U_ACT_D_BYTES), umma_down_kernel); });
    if (e != cudaSuccess) return e;
    umma_down_kernel<<<dim3(p.H / 256, max_tiles), U_THREADS, umma_smem_bytes(U_ACT_D_BYTES), st>>>(p);
    return cudaGetLastError();
}

}  // namespace edg
