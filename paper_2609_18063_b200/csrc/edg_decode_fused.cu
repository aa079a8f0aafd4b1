// The batch-1 layer-step as ONE kernel (a1-a2 for the next step, a3 take, a4-a6 for this step).
//
// Work split.  CTAs of 128 threads in thread-block clusters of kC = 4, four CTAs to an SM.  A cluster
// owns `qpc` quarters of the intermediate dimension of one routed expert (of two, one after the
// other, when the experts share one adapter) and walks them in sequence: for a quarter its CTAs
// compute their gate/up rows (over all of K), exchange h = silu(gate) * up inside the cluster, and
// add the quarter's columns to the H/4 output rows each CTA owns, so no exchange ever crosses a
// cluster.  A step chained to its predecessor uses one cluster per expert or pair of experts
// (qpc = 4: few, long-lived CTAs, dozens of steps share the GPU); a step launched alone uses four
// clusters per expert (qpc = 1: all SMs at once).
//   * Weights stream through two stage buffers by bulk asynchronous copies (cp.async.bulk, completion
//     on mbarriers), one 36 KB load in flight per CTA at any time: the first half of the K range of
//     the quarter's gate/up rows (a K quarter per stage), the second half, then the quarter's down
//     block across both stages.  The exchange of h runs while the down block is on its way.  What
//     keeps the memory system busy is the number of such pipelines: four per SM.
//   * Issuing a bulk copy costs its lane some 50 ns and the lanes of a warp take turns, so the 16
//     copies of a load are dealt to the four warps behind a CTA barrier, and the score of small
//     copies for the adapter slices is issued while the quarter's weights are still in flight.
//   * Both projections run on mma.sync.m16n8k16 fragments: the codes masked straight into fp16 --
//     subnormal, or biased in dependent chains (edg_mma.cuh), five instructions a word -- the activations
//     as column 0 of the B tile; zero point and scale are applied in fp32 per 64-code block.  The loops over K
//     blocks are rolled and the operands live in shared memory on purpose: a CTA runs most of this
//     code once, and instruction fetch competes with the weight stream.
//   * The rank-r LoRA projections A.x are split over the CTAs of a cluster and exchanged through
//     distributed shared memory, as are h and the partials of A_down.h (summed over the quarters,
//     B_down applied once at the end, its rows read straight from memory).  The exchanges are
//     remote stores that count their bytes on an mbarrier of the receiving CTA (st.async); the only
//     cluster barrier is a handshake at start-up, because a cluster-scope barrier also waits for
//     every bulk copy in flight into the SM.
//   * The rows of the prerouter head are dealt to the first CTAs of the grid, two rows per warp at
//     a time; every warp publishes its logits into a ring slot of the workspace by itself, and the
//     warp that delivers the last one selects the experts: it leaves the (expert, gate) pairs
//     behind the logits in the ring slot and writes the caller's inds_next / gates_next.
// The reduce y = sum_k w_k o_k goes through an fp32 scratch (one set per ring slot): each CTA writes
// its gate-weighted partial, and the last CTA to arrive for a block of rows (one atomic counter per
// block) sums the partials in a fixed order, so the result does not depend on arrival order.
// Consecutive layer-steps are chained by programmatic dependent launch: every CTA releases the next
// step's kernel as soon as it runs, so steps queue up on the device as far as its CTA slots go; a
// step evaluates its head first, then takes its routing from the ring slot of the step before it
// and streams its weights while earlier steps are still computing.  It never waits for the
// previous kernel to end.  Every wait on another CTA or kernel is bounded and falls back to a safe
// path (or flags the result) when it gives up.
#include <cooperative_groups.h>

#include "edg_mma.cuh"
#include "edg_head.cuh"

namespace cg = cooperative_groups;

namespace edg {

constexpr int kC = 4;             // CTAs per cluster
constexpr int kE16 = kC * kDownSlices;   // CTAs per expert
constexpr int kFW = 4;            // warps per CTA
constexpr int kStages = 2;        // copy stages per CTA: a quarter of the gate/up K range each, or half of the down block
constexpr int kMaxRank = 64;
constexpr int kMaxEpc = 4;         // experts a cluster may take, one after the other
constexpr int kRing = kHandoffRing;   // chained layer-steps in flight: hand-off slots for logits, reduce scratch, counters

// ---------------------------------------------------------------- shared-memory carve-up
// Byte offsets, identical on host and device.  The two stages (a quarter of the gate/up K range
// each) come first; the down block later takes both (it is exactly two stages large).  A CTA stays
// under a quarter of an SM's shared memory, so four CTAs -- of this launch or of later ones -- share
// an SM.
struct FusedSmem {
    uint32_t stage0, stage_bytes;                      // stage s (a quarter of the K range) at stage0 + s * stage_bytes
    uint32_t mat_codes, mat_sz;                        // bytes of one (matrix, row tile) run of codes / sz inside a stage
    uint32_t sz0;                                      // offset of the sz runs inside a stage
    uint32_t d_codes, d_sz;                            // down block, from stage0
    uint32_t lora0, lora_bytes;                        // two buffers of per-quarter adapter slices: B_gate rows, B_up rows, A_down columns
    uint32_t bars, s_u, s_h, s_ud_part, s_ud, s_gu, s_o, s_red, s_hloc, s_topk, s_part, s_table, s_xb, s_xsum, s_xbias, s_hb, s_hsum, s_hbias, flag, s_ex, total;
};
__host__ __device__ inline FusedSmem fused_smem(int H, int I, int E, int group, int rank) {
    FusedSmem S;
    const uint32_t rows_gu = I / kE16, rows_d = H / kC, sw = I / kDownSlices, tg = rows_gu / 16;
    // a stage holds, for gate and up and each of their tg row tiles, H/128 chunks (H/4 codes per row)
    S.mat_codes = (uint32_t)(H / 128) * 256;
    S.mat_sz = (uint32_t)((H / 4) / group) * 64;
    S.sz0 = 2 * tg * S.mat_codes;
    S.stage_bytes = 2 * tg * (S.mat_codes + S.mat_sz);
    uint32_t o = 0;
    S.stage0 = o;     o += kStages * S.stage_bytes;
    S.d_codes = S.stage0;
    S.d_sz = S.stage0 + rows_d * sw / 2;               // rows_d * (sw/2 + sw/group*4) == 2 * stage_bytes
    S.lora_bytes = 3 * rows_gu * (uint32_t)rank * 2;   // B_gate[rows_gu][rank], B_up[rows_gu][rank], A_down[rank][rows_gu]
    S.lora0 = o;      o += 2 * S.lora_bytes;
    o = (o + 15) / 16 * 16;
    S.bars = o;       o += 8 * 12;
    o = (o + 15) / 16 * 16;
    S.s_u = o;        o += 2 * kMaxRank * 4;
    S.s_h = o;        o += 2 * sw * 4;                // the quarter's h, double-buffered
    S.s_ud_part = o;  o += 2 * kC * kMaxRank * 4;
    S.s_ud = o;       o += kMaxRank * 4;
    S.s_gu = o;       o += 2 * rows_gu * 4;
    S.s_o = o;        o += rows_d * 4;
    S.s_red = o;      o += 40 * kFW * 4;              // per-warp partials: up to 32 adapter rows + 8 head rows per CTA
    S.s_hloc = o;     o += 32 * 4;
    // logits gathered by the warp that finishes the head, then its K winners: in s_o when that is
    // large enough (s_o is first written by the down phase of the first quarter, barriers later)
    if (rows_d * 4 >= (uint32_t)E * 4 + 256) S.s_topk = S.s_o;
    else { S.s_topk = o; o += (uint32_t)E * 4 + 256; }
    S.s_part = o;     o += kFW * 2 * rows_gu * 4;     // per-warp (k-slice) partial sums of the gate/up rows
    // this layer's slot table, fetched before the routing is known and used up before the first
    // quarter starts: in s_part when that is large enough
    if (kFW * 2 * rows_gu * 4 >= (uint32_t)E * 4) S.s_table = S.s_part;
    else { S.s_table = o; o += (uint32_t)E * 4; }
    o = (o + 15) / 16 * 16;
    S.s_xb = o;       o += (uint32_t)H * 2;           // x as fp16 B-fragment words, k-slot order
    S.s_xsum = o;     o += (uint32_t)(H / 32) * 4;    // sums of x per scaled block
    S.s_xbias = o;    o += (uint32_t)(H / 32) * 4;    // what the biased codes add per scaled block: 1024 * (even positions) + 64 * (odd positions)
    S.s_hb = o;       o += (sw / 32) * 2 * 64;        // the quarter's h as (hi, lo) B-fragment words
    S.s_hsum = o;     o += (sw / 32) * 4;
    S.s_hbias = o;    o += (sw / 32) * 4;
    S.flag = o;       o += 16;
    S.s_ex = o;       o += 96;                        // the cluster's experts: raw routing, then what the take made of it
    S.total = (o + 15) / 16 * 16;
    return S;
}

struct FusedParams {
    const uint8_t* pool;
    const int32_t* slots;         // [K] slots, or expert ids when table != null
    const int32_t* table;         // [E] or null
    const int32_t* experts;       // [K] or null
    const float* gates;           // [K]
    const uint16_t* x;            // [H] bf16
    edg_lora lora;
    void* y;                      // [H]
    int32_t* status;
    int32_t* counters;            // [kRing][kC] one per ring slot and block of output rows, zero between uses
    int32_t* pre_counter;         // [kRing] rows of the head delivered so far, back to zero after every head
    float* partial;               // [kRing][K][H]
    float* logits_ws;             // [kRing][E] logits of the next step's head; all-ones words = not yet written
    const void* W_pre;            // [E][H] or null
    int32_t* inds_next;
    float* gates_next;
    float* logits_next;
    int H, I, E, K, group, rank, n_adapters, n_slots, pre_dtype, out_dtype;
    float sigma;
    RecordLayout L;
    unsigned long long* trace;    // optional [grid CTAs][kTraceMarks] globaltimer stamps, or null
    int32_t* done;                // [kRing] reducers of the step that has read each routing slot and are finished
    int ring;                     // ring slot of this step's reduce scratch
    int flag_in;                  // -1: the routing is already in memory; else the ring slot to take it from
    int flag_out;                 // -1 or the ring slot that receives inds_next / gates_next
    int gshift;                   // log2(group)
    int qpc;                      // quarters of the intermediate dimension per cluster: 4 (one cluster per expert), 2 or 1
    int epc;                      // experts per cluster, one after the other: 1, or 2 or 4 (only with qpc = 4)
    int32_t* inds_mirror;         // [K] copy of inds_next in mapped pinned host memory, or null
    uint16_t* x_next;             // [H] bf16 or null: bf16(rmsnorm(x + y)), the next layer-step's hidden state in a dependent chain
    float* dep_ws;                // [kRing][kDepWords]: per ring slot, kC partial sums of squares, (words 4..7) the reducers' "my rows of x_next are written" flags
    int32_t* norm_cnt;            // [kRing] reducers that have delivered their sum of squares
    float eps;
    int head_extra;               // CTAs behind those of the experts that evaluate the head and nothing else (0: the first CTAs of the grid do)
    int dep_wait;                 // -1, or the ring slot whose flag says that this step's x has been written
    int slot_until_end;           // the step before may write to this step's ring slot until it ends
    const uint8_t* shared_rec;    // record of the layer's always-on shared expert (one more expert with gate 1), or null
    edg_lora shared_lora;         // its own adapter, leading dimension 1 (null pointers with rank_shared == 0)
    int n_shared;                 // 0 or 1
    int rank_shared;
    FusedSmem S;                  // shared-memory carve-up
};


__device__ __forceinline__ void trace_mark(const FusedParams& p, int m) {
    if (p.trace != nullptr && threadIdx.x == 0) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        p.trace[(size_t)blockIdx.x * kTraceMarks + m] = t;
    }
}

// four consecutive outputs (i a multiple of 4)
__device__ __forceinline__ void store_y4(void* y, int out_dtype, size_t i, float4 v) {
    if (out_dtype == EDG_F32) {
        *reinterpret_cast<float4*>(static_cast<float*>(y) + i) = v;
    } else if (out_dtype == EDG_F16) {
        __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
        *reinterpret_cast<uint2*>(static_cast<__half*>(y) + i) = make_uint2(h2_as_u32(a), h2_as_u32(b));
    } else {
        bf16_t* o = static_cast<bf16_t*>(y) + i;
        store_out<bf16_t>(o, 0, v.x); store_out<bf16_t>(o, 1, v.y); store_out<bf16_t>(o, 2, v.z); store_out<bf16_t>(o, 3, v.w);
    }
}

__device__ __forceinline__ void store_y(void* y, int out_dtype, size_t i, float v) {
    if (out_dtype == EDG_F32) store_out<float>(static_cast<float*>(y), i, v);
    else if (out_dtype == EDG_F16) store_out<__half>(static_cast<__half*>(y), i, v);
    else store_out<bf16_t>(static_cast<bf16_t*>(y), i, v);
}

// four consecutive stored outputs (i a multiple of 4) as floats, read past the L1 (another CTA wrote them)
__device__ __forceinline__ float4 load_y4_cg(const void* y, int out_dtype, size_t i) {
    if (out_dtype == EDG_F32) return __ldcg(reinterpret_cast<const float4*>(static_cast<const float*>(y) + i));
    const uint2 w = __ldcg(reinterpret_cast<const uint2*>(static_cast<const unsigned short*>(y) + i));
    if (out_dtype == EDG_F16) {
        const float2 a = __half22float2(u32_as_h2(w.x)), b = __half22float2(u32_as_h2(w.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    return make_float4(bf16_lo(w.x), bf16_hi(w.x), bf16_lo(w.y), bf16_hi(w.y));
}
// a value as it reads back after being stored in the output type
__device__ __forceinline__ float round_out(float v, int out_dtype) {
    if (out_dtype == EDG_F32) return v;
    if (out_dtype == EDG_F16) return __half2float(__float2half_rn(v));
    uint32_t u = __float_as_uint(v);
    u += 0x7FFFu + ((u >> 16) & 1u);
    return __uint_as_float(u & 0xFFFF0000u);
}

// the same over a bf16 row in global memory (read-only path)
__device__ __forceinline__ float gmem_b_dot(const uint16_t* B, const float* u, int r) {
    float d = 0.f;
    for (int j = 0; j < r; j += 8) {
        const uint4 b = __ldg(reinterpret_cast<const uint4*>(B + j));
        d = fmaf(bf16_lo(b.x), u[j + 0], d); d = fmaf(bf16_hi(b.x), u[j + 1], d);
        d = fmaf(bf16_lo(b.y), u[j + 2], d); d = fmaf(bf16_hi(b.y), u[j + 3], d);
        d = fmaf(bf16_lo(b.z), u[j + 4], d); d = fmaf(bf16_hi(b.z), u[j + 5], d);
        d = fmaf(bf16_lo(b.w), u[j + 6], d); d = fmaf(bf16_hi(b.w), u[j + 7], d);
    }
    return d;
}

// sum_j B[j] * u[j] over a bf16 row in shared memory, r a multiple of 8
__device__ __forceinline__ float smem_b_dot(const uint16_t* B, const float* u, int r) {
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

// mbarriers: one per stage (two arrivals: the two warps that issue its copies), then the down
// block, the adapter slices (two buffers), the adapter projections, h (two buffers)
enum { BAR_DOWN = 2, BAR_LORA = 3, BAR_U = 5, BAR_H = 6, kNumBars = 8 };

// ---------------------------------------------------------------- head rows (a1) and top-k (a2)
// The E rows of the head are dealt round-robin to the first CTAs of the grid; a row is split over
// all threads of its CTA, so it costs one trip to memory.  The warp that delivers the last logits
// (an atomic counter) gathers all E and does softmax + top-k.

// Partial dot of head row e with the hidden state over this thread's elements, any dtype and H.
__device__ __noinline__ float head_row_partial(const void* W_pre, int pre_dtype, const uint16_t* x, int H, int e, int tid) {
    float acc = 0.f;
    if (pre_dtype == EDG_F16) {
        const __half* wr = static_cast<const __half*>(W_pre) + (size_t)e * H;
        for (int c = tid * 8; c < H; c += kFW * 32 * 8) {
            const uint4 w = ld_keep16(wr + c);
            const uint4 xv = ld_keep16(x + c);
            const float2 a = __half22float2(u32_as_h2(w.x)), b = __half22float2(u32_as_h2(w.y));
            const float2 d = __half22float2(u32_as_h2(w.z)), f = __half22float2(u32_as_h2(w.w));
            acc = fmaf(a.x, bf16_lo(xv.x), acc); acc = fmaf(a.y, bf16_hi(xv.x), acc);
            acc = fmaf(b.x, bf16_lo(xv.y), acc); acc = fmaf(b.y, bf16_hi(xv.y), acc);
            acc = fmaf(d.x, bf16_lo(xv.z), acc); acc = fmaf(d.y, bf16_hi(xv.z), acc);
            acc = fmaf(f.x, bf16_lo(xv.w), acc); acc = fmaf(f.y, bf16_hi(xv.w), acc);
        }
    } else {
        const float* wr = static_cast<const float*>(W_pre) + (size_t)e * H;
        for (int c = tid * 4; c < H; c += kFW * 32 * 4) {
            const uint4 w = ld_keep16(wr + c);
            const uint2 xv = *reinterpret_cast<const uint2*>(x + c);
            acc = fmaf(__uint_as_float(w.x), bf16_lo(xv.x), acc); acc = fmaf(__uint_as_float(w.y), bf16_hi(xv.x), acc);
            acc = fmaf(__uint_as_float(w.z), bf16_lo(xv.y), acc); acc = fmaf(__uint_as_float(w.w), bf16_hi(xv.y), acc);
        }
    }
    return acc;
}

// ---------------------------------------------------------------- the fused kernel
// NCW = H / 256 = chunks (of 32 codes) per warp in gate/up; DCH = I / 128 = chunks of a down row-slice;
// TG = I / 256 = row tiles per matrix and CTA in gate/up; TD = H / 512 = row tiles per warp in down;
// CPB = chunks per scaled block (2 for groups of 64 or 128 codes, 1 for groups of 32).
// Most of the kernel is straight-line code that a CTA runs once or four times, so its size is kept
// small on purpose (loops over K blocks are not unrolled, operands come from shared memory):
// instruction fetches compete with the weight stream for the same memory system.

constexpr int kPreRed = 32;       // s_red rows 0..31: adapter projections, 32..39: head rows
constexpr int kMaxPre = 8 * kFW;  // head rows per head CTA (up to four batches of two per warp)

template <int NCW, int DCH, int TG, int TD, int CPB, bool EX>
__global__ void __launch_bounds__(kFW * 32, 4) fused_layer_kernel(const __grid_constant__ FusedParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int cl = blockIdx.x / kC;                // cluster: an expert, or some quarters of it
    const int nq = kDownSlices / p.qpc;            // clusters per expert
    // the clusters behind those of the routed experts take the shared expert: an expert like the
    // others, always on (gate 1), with a record and an adapter of its own, partial number K
    const int n_routed_cl = (p.K / p.epc) * nq;
    const bool is_shared = cl >= n_routed_cl;
    const int epc_l = is_shared ? 1 : p.epc;       // experts this cluster takes, one after the other
    const int k = is_shared ? p.K : (cl / nq) * p.epc;   // position of the cluster's (first) expert in the routing
    const int cq = is_shared ? cl - n_routed_cl : cl % nq;   // which of the expert's clusters this is
    const edg_lora& lo = is_shared ? p.shared_lora : p.lora;
    const int c0 = cq * p.qpc;                     // first quarter of the intermediate dimension of this cluster
    const int crank = blockIdx.x % kC;             // rank inside the cluster
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
    const int g8 = lane >> 2, t4 = lane & 3;       // fragment coordinates: row slot, quad lane

    const FusedSmem& S = p.S;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S.bars);
    float* s_u = reinterpret_cast<float*>(smem + S.s_u);            // [2][kMaxRank]
    float* s_h = reinterpret_cast<float*>(smem + S.s_h);            // [2][I/4]   (double-buffered over quarters)
    float* s_ud_part = reinterpret_cast<float*>(smem + S.s_ud_part);// [2][kC][kMaxRank]
    float* s_ud = reinterpret_cast<float*>(smem + S.s_ud);          // [kMaxRank]
    float* s_gu = reinterpret_cast<float*>(smem + S.s_gu);          // [2][rows_gu]
    float* s_o = reinterpret_cast<float*>(smem + S.s_o);            // [rows_d]
    float* s_red = reinterpret_cast<float*>(smem + S.s_red);        // [40][kFW]
    float* s_hloc = reinterpret_cast<float*>(smem + S.s_hloc);      // [rows_gu]
    float* s_part = reinterpret_cast<float*>(smem + S.s_part);      // [kFW][2 * rows_gu]
    int* s_flag = reinterpret_cast<int*>(smem + S.flag);
    int* s_table = reinterpret_cast<int*>(smem + S.s_table);        // [E]
    uint4* s_xb = reinterpret_cast<uint4*>(smem + S.s_xb);          // [H/8]  x as B-fragment words
    float* s_xsum = reinterpret_cast<float*>(smem + S.s_xsum);      // [H/(32 CPB)] block sums of x
    float* s_xbias = reinterpret_cast<float*>(smem + S.s_xbias);    // [H/(32 CPB)] bias carried by the codes of a block
    uint4* s_hb = reinterpret_cast<uint4*>(smem + S.s_hb);          // [DCH][2][4] h (hi, lo) as B-fragment words
    float* s_hsum = reinterpret_cast<float*>(smem + S.s_hsum);      // [DCH/CPB]
    float* s_hbias = reinterpret_cast<float*>(smem + S.s_hbias);    // [DCH/CPB]

    constexpr int rows_gu = 16 * TG, rows_d = 128 * TD, sw = 32 * DCH;
    const int n0_d = crank * rows_d;               // first down (= output) row of this CTA
    const int r = is_shared ? p.rank_shared : p.rank;
    // reduce scratch of this step's ring slot: a chained step never waits for the previous kernel to
    // end, so steps in flight must not share it
    const int np = (p.K + p.n_shared) * nq;        // partial outputs per output row
    float* partial = p.partial + (size_t)p.ring * kDownSlices * (p.K + 1) * p.H;
    int32_t* counters = p.counters + p.ring * kC;
    trace_mark(p, 0);
    // A step that produces the next hidden state clears its "written" flag before it releases the
    // next kernel, which may start polling it at once.
    if (p.x_next != nullptr && blockIdx.x == 0 && tid == 0) {
        for (int c = 0; c < kC; ++c) st_relaxed_gpu_u32(p.dep_ws + p.ring * kDepWords + 4 + c, 0u);
        __threadfence();
    }
    if (tid == 0) pdl_launch_dependents();

    // ---- a1 for the next step, first of all: the loads of the head rows depend on nothing but x,
    //      and the routing they lead to is what the next layer-step waits for.  The rows are dealt
    //      round-robin to the first CTAs of the grid; a row is split over all threads of its CTA
    //      (8 elements each).
    const int max_pre = (p.pre_dtype == EDG_F16 && p.H <= 2048) ? kMaxPre : kFW;     // two rows per warp only on the fast path below
    // An fp16 head whose rows split into 16-row tiles goes to the tensor cores, the hidden state as
    // column 0 of the B operand -- an eighth of the instructions of the FMA form below.  A chained step
    // (few CTAs) gives a head CTA two tiles, each over half of K per warp; a step that runs alone one
    // tile over a quarter of K per warp, and there the head has CTAs of its own behind those of the
    // experts (p.head_extra of them, on SMs the experts leave idle), so that no expert waits for it.
    const int n_expert_ctas = (int)gridDim.x - p.head_extra;
    const bool head_only = (int)blockIdx.x >= n_expert_ctas;
    const int head_idx = p.head_extra > 0 ? (int)blockIdx.x - n_expert_ctas : (int)blockIdx.x;
    const int tpc = p.qpc == kDownSlices ? 2 : 1;                 // tiles per head CTA
    const int ksplit = kFW / tpc;                                 // warps sharing the K range of a tile
    const bool pre_mma = p.W_pre != nullptr && p.pre_dtype == EDG_F16 && (p.E % (16 * tpc)) == 0 && (p.H % (256 * ksplit)) == 0 &&
                         p.E / (16 * tpc) <= (p.head_extra > 0 ? p.head_extra : (int)gridDim.x);
    const int n_head_ctas = p.W_pre == nullptr ? 0 : pre_mma ? p.E / (16 * tpc) : min((int)gridDim.x, max(32, (p.E + max_pre - 1) / max_pre));
    const bool head_cta = head_idx >= 0 && head_idx < n_head_ctas;
    const int n_pre = (head_cta && !pre_mma) ? min(max_pre, (p.E - (int)blockIdx.x + n_head_ctas - 1) / n_head_ctas) : 0;
    const bool mma_head = pre_mma && head_cta;
    const int mrow0 = (head_idx * tpc + warp % tpc) * 16;         // first row of this warp's tile
    const int mk0 = (warp / tpc) * (p.H / ksplit);                // first k of this warp's share of K
    // Usual case (fp16 head, H <= 2048): warp w evaluates row w of this CTA's rows by itself, each
    // lane covering 8 runs of 8 elements, and publishes it without waiting for any other warp.
    const bool pre_fast = n_pre > 0 && p.pre_dtype == EDG_F16 && p.H <= 2048;
    // Its rows beyond the first two follow in further batches of two.
    int my_e = (int)blockIdx.x + warp * n_head_ctas;             // fast path: this warp's row, and its second row
    int my_e2 = (int)blockIdx.x + (warp + kFW) * n_head_ctas;
    bool my_row = pre_fast && warp < n_pre && my_e < p.E;
    bool my_row2 = pre_fast && warp + kFW < n_pre && my_e2 < p.E;
    uint4 lw[8], lw2[8];
    // (tensor-core form: rows g and g + 8 of the tile, 8 k per lane and chunk of 32 k; the first 8 chunks now)
    const __half* mwa = static_cast<const __half*>(p.W_pre) + (size_t)(mrow0 + g8) * p.H + mk0 + t4 * 8;
    if (mma_head) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            lw[j] = ld_keep16(mwa + j * 32);
            lw2[j] = ld_keep16(mwa + (size_t)8 * p.H + j * 32);
        }
    }
    if (my_row) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = (j * 32 + lane) * 8;
            lw[j] = i < p.H ? ld_keep16(static_cast<const __half*>(p.W_pre) + (size_t)my_e * p.H + i) : make_uint4(0, 0, 0, 0);
        }
    }
    if (my_row2) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = (j * 32 + lane) * 8;
            lw2[j] = i < p.H ? ld_keep16(static_cast<const __half*>(p.W_pre) + (size_t)my_e2 * p.H + i) : make_uint4(0, 0, 0, 0);
        }
    }
    const bool pre_lane = tid * 8 < p.H;
    uint32_t pre_state = kNotYet, pre_state2 = kNotYet;   // the ring-slot entries this lane will publish into, as the kernel finds them
    if (p.flag_out >= 0) {
        if (mma_head && warp < tpc && lane < 16)
            pre_state = ld_relaxed_gpu_u32(&p.logits_ws[(size_t)p.flag_out * (p.E + kPairWords) + mrow0 + lane]);
        if (my_row && lane == 0) pre_state = ld_relaxed_gpu_u32(&p.logits_ws[(size_t)p.flag_out * (p.E + kPairWords) + my_e]);
        if (my_row2 && lane == 0) pre_state2 = ld_relaxed_gpu_u32(&p.logits_ws[(size_t)p.flag_out * (p.E + kPairWords) + my_e2]);
        if (n_pre > 0 && !pre_fast && warp == kFW - 1 && lane < n_pre) {
            const int e = (int)blockIdx.x + lane * n_head_ctas;
            if (e < p.E) pre_state = ld_relaxed_gpu_u32(&p.logits_ws[(size_t)p.flag_out * (p.E + kPairWords) + e]);
        }
    }

    // ---- thread 0: the barriers (peers will count bytes on BAR_U / BAR_H of this CTA, so they must
    //      exist, and every CTA of the cluster must be running, before anyone sends)
    if (tid == 0) {
        for (int s = 0; s < kNumBars; ++s)
            mbar_init(&bars[s], s < kStages ? 2 : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        // bytes this CTA will receive: 2r adapter projections once; per quarter, that quarter of h
        // and kC partials of A_down.h (the barriers of quarters 2 and 3 are re-armed below)
        if (r > 0) mbar_expect_tx(&bars[BAR_U], 2u * r * 4u);
        mbar_expect_tx(&bars[BAR_H], (uint32_t)(sw + kC * r) * 4u);
        if (p.qpc * epc_l > 1) mbar_expect_tx(&bars[BAR_H + 1], (uint32_t)(sw + kC * r) * 4u);
    }
    // The cluster handshake starts here (thread 0 after its barrier set-up) and is completed
    // before the first remote store: the arriving side of a cluster-scope barrier waits for every
    // bulk copy in flight into the SM, those of a neighbouring CTA included, and that wait is
    // hidden behind the loads below.
    cluster_arrive();

    // ---- everyone: the slot table of this layer (one coalesced read now saves a dependent trip to
    //      memory once the routing is known) and the hidden state as the MMA's B operand, kept in
    //      shared memory.  Thread t converts activations 8t .. 8t+7 (word t%4 of chunk t/4) into
    //      the k-slot order of the fragments; s_xsum[j] = sum of the activations of scaled block j
    //      (for the zero points).
    if (p.table != nullptr && warp == 0)      // (warp 0 alone: it resolves the routing before the CTA's first barrier)
        for (int i = lane; i < p.E; i += 32) s_table[i] = __ldcg(&p.table[i]);
    auto convert_x = [&]() {
    constexpr int kRounds = NCW / 4;                              // eight activations a thread and round
    uint4 v[kRounds];
    uint32_t m = 0;
#pragma unroll
    for (int q = 0; q < kRounds; ++q) {
        v[q] = *reinterpret_cast<const uint4*>(p.x + (q * kFW * 32 + tid) * 8);
        const uint32_t w = max(max(max(v[q].x & 0x7FFFu, v[q].y & 0x7FFFu), max(v[q].z & 0x7FFFu, v[q].w & 0x7FFFu)) << 16,
                               max(max(v[q].x & 0x7FFF0000u, v[q].y & 0x7FFF0000u), max(v[q].z & 0x7FFF0000u, v[q].w & 0x7FFF0000u)));
        m = max(m, w);
    }
    float scale = 1.f;
    if (EX) {                                                     // the largest magnitude of the state
        m = __reduce_max_sync(0xFFFFFFFFu, m);
        if (lane == 0) s_flag[warp] = (int)m;
        __syncthreads();
        scale = vector_scale(max(max((uint32_t)s_flag[0], (uint32_t)s_flag[1]), max((uint32_t)s_flag[2], (uint32_t)s_flag[3])));
        if (tid == 0) s_xbias[0] = kUnscaleS * vector_unscale(scale);
    }
#pragma unroll
    for (int q = 0; q < kRounds; ++q) {
        const int t = q * kFW * 32 + tid;
        float sum = 0.f, sodd = 0.f;
        const float f[8] = {bf16_lo(v[q].x), bf16_hi(v[q].x), bf16_lo(v[q].y), bf16_hi(v[q].y),
                            bf16_lo(v[q].z), bf16_hi(v[q].z), bf16_lo(v[q].w), bf16_hi(v[q].w)};
        s_xb[t] = EX ? permute8_s(f, scale) : permute8(f);
#pragma unroll
        for (int e = 0; e < 8; e += 2) {          // of what the MMA will see (without a scale fp16 is exact in its normal range only)
            sum += EX ? f[e] : __half2float(__float2half_rn(f[e]));
            sodd += EX ? f[e + 1] : __half2float(__float2half_rn(f[e + 1]));
        }
        sum = group_sum<4 * CPB>(sum);
        sodd = group_sum<4 * CPB>(sodd);
        if ((t % (4 * CPB)) == 0) {
            s_xsum[t / (4 * CPB)] = EX ? (sum + sodd) * (kScaleS * scale) : sum + sodd;
            if (!EX) s_xbias[t / (4 * CPB)] = fmaf(1024.f, sum, 64.f * sodd);
        }
    }
    };
    static_assert(kFW == 4, "a word of s_flag per warp");
    if (p.dep_wait < 0) convert_x();          // (a step that waits for its hidden state converts it once it is there)
    if (tid < kMaxRank) s_ud[tid] = 0.f;

    // ---- a3: take, for the experts of this cluster (up to kMaxEpc, one after the other), as a
    //      function of the routing warp 0 has put into s_ex.  The decision is the same in every CTA
    //      of the cluster.  An expert that is out of range is skipped (and flagged).  Lane 0 of warp
    //      0 resolves -- before the CTA's first barrier, for the copies warp 0 issues -- and leaves
    //      the result in shared memory: s_ex[0..7] raw (expert or slot, gate) pairs, [8] number of
    //      valid experts, [9] adapter, [10] mask of valid experts, [12..15] the valid experts in
    //      order, [16..19] their slots, [20..23] their gates.
    int* s_ex = reinterpret_cast<int*>(smem + S.s_ex);
    auto take = [&]() {               // warp 0
        if (lane == 0) {
            int nv = 0, okm = 0, adv = 0;
            for (int e = 0; e < epc_l; ++e) {
                int slot = s_ex[2 * e];
                const int expert = is_shared ? 0 : (p.table != nullptr ? slot : (p.experts != nullptr ? p.experts[k + e] : 0));
                if (p.table != nullptr && !is_shared) slot = (slot >= 0 && slot < p.E) ? s_table[slot] : -1;
                int a_e = 0;          // several experts per cluster only with one shared adapter: 0 for all
                if (r > 0 && p.n_adapters != 1) a_e = (expert >= 0 && expert < p.E) ? expert : -1;
                if (is_shared) { slot = 0; a_e = 0; }
                const bool ok = slot >= 0 && slot < p.n_slots && a_e >= 0;
                if (ok) { s_ex[12 + nv] = e; s_ex[16 + e] = slot; okm |= 1 << e; ++nv; if (e == 0) adv = a_e; }
                s_ex[20 + e] = s_ex[2 * e + 1];
            }
            s_ex[8] = nv; s_ex[9] = adv; s_ex[10] = okm;
        }
        __syncwarp();
    };
    int ad = 0, n_items = 0;          // set from s_ex: by warp 0 right after its take, by everyone after the barrier
    bool valid = false;
    auto read_take = [&]() { n_items = s_ex[8] * p.qpc; ad = s_ex[9]; valid = n_items > 0; };
    // the items of this cluster's stream: the quarters of its valid experts, one expert after the other
    auto item_expert = [&](int w) { return s_ex[12 + w / p.qpc]; };
    auto item_rec = [&](int w) { return is_shared ? p.shared_rec : p.pool + (size_t)s_ex[16 + item_expert(w)] * p.L.bytes; };
    const int cps = p.H / 128;            // chunks of a row per stage
    const int gpst = (p.H / 4) >> p.gshift;   // groups of a row per stage
    const int gps = sw >> p.gshift;       // groups of a down row-slice

    // K quarters 2 pair and 2 pair + 1 of the gate/up rows of item w (a quarter of one of the
    // cluster's experts) go into stages 0 and 1 as 16 copies, one run each (codes or sz of a
    // (matrix, row tile)); issuing a copy costs its lane some 50 ns and the lanes of a warp take
    // turns, so the copies are dealt to the four warps: warp v issues runs 4 (v & 1) .. + 3 of
    // stage v / 2 from its lanes 0..3, after lane 0 has armed the stage's barrier with their bytes
    // (one arrival per issuing warp).  The calling warp plays warps v0 .. v1 - 1.
    auto issue_gu = [&](int w, int pair, int v0, int v1) {
        const int c = c0 + w % p.qpc;
        const uint8_t* rec = item_rec(w);
        const uint64_t pol = policy_evict_first();       // weights stream through L2 once
        for (int v = v0; v < v1; ++v) {
            const int s = v >> 1, run = (v & 1) * 4 + lane, kq = pair * 2 + s;
            const int n_runs = min(4, max(0, 4 * TG - (v & 1) * 4));
            if (lane == 0) mbar_expect_tx(&bars[s], (uint32_t)(n_runs / 2) * (S.mat_codes + S.mat_sz));
            __syncwarp();
            if (lane < n_runs) {
                uint8_t* st = smem + S.stage0 + s * S.stage_bytes;
                const int mt = run >> 1, is_sz = run & 1, m = mt / TG, ti = mt % TG;
                const int n = c * sw + crank * rows_gu + 16 * ti;
                if (!is_sz) bulk_g2s_hint(st + mt * S.mat_codes, rec + (m ? p.L.codes_up : p.L.codes_gate) + code_off(p.H, n, kq * cps),
                                          S.mat_codes, &bars[s], pol);
                else bulk_g2s_hint(st + S.sz0 + mt * S.mat_sz, rec + (m ? p.L.sz_up : p.L.sz_gate) + sz_off(p.H, p.group, n, kq * gpst),
                                   S.mat_sz, &bars[s], pol);
            }
        }
    };
    // A step that waits for its hidden state has time to spare: it asks the L2 for the rest of its
    // first item (second half of K, down block), so that those loads later come from the L2.
    auto prefetch_rest = [&](int w) {
        const int c = c0 + w % p.qpc;
        const uint8_t* rec = item_rec(w);
        if (lane < 4 * TG) {
            const int mt = lane >> 1, is_sz = lane & 1, m = mt / TG, ti = mt % TG;
            const int n = c * sw + crank * rows_gu + 16 * ti;
            // (K quarters 2 and 3 of a (matrix, row tile) follow each other in memory: one run of twice the size)
            if (!is_sz) bulk_prefetch_l2(rec + (m ? p.L.codes_up : p.L.codes_gate) + code_off(p.H, n, 2 * cps), 2 * S.mat_codes);
            else bulk_prefetch_l2(rec + (m ? p.L.sz_up : p.L.sz_gate) + sz_off(p.H, p.group, n, 2 * gpst), 2 * S.mat_sz);
        } else if (lane == 4 * TG) {
            bulk_prefetch_l2(rec + p.L.codes_down + down_code_off(p.H, p.I, n0_d, c * (sw / 32)), (uint32_t)rows_d * sw / 2);
        } else if (lane == 4 * TG + 1) {
            bulk_prefetch_l2(rec + p.L.sz_down + down_sz_off(p.H, p.I, p.group, n0_d, c * gps), (uint32_t)rows_d * gps * 4);
        }
    };
    // One warp issues the adapter slices of item w into buffer w & 1: this CTA's rows of B_gate and
    // B_up for the item's quarter, and its columns of A_down (one 16-byte-multiple run per rank index).
    auto issue_lora = [&](int w) {
        const int c = c0 + w % p.qpc, it = w;
        const uint32_t bgu = rows_gu * r * 2, ad_row = rows_gu * 2;
        uint8_t* buf = smem + S.lora0 + (it & 1) * S.lora_bytes;
        const int n0 = c * sw + crank * rows_gu;
        if (lane == 0) mbar_expect_tx(&bars[BAR_LORA + (it & 1)], 2 * bgu + r * ad_row);
        __syncwarp();
        const size_t bo = ((size_t)ad * p.I + n0) * r * 2;
        if (lane == 0) bulk_g2s(buf, static_cast<const uint8_t*>(lo.B_gate) + bo, bgu, &bars[BAR_LORA + (it & 1)]);
        if (lane == 1) bulk_g2s(buf + bgu, static_cast<const uint8_t*>(lo.B_up) + bo, bgu, &bars[BAR_LORA + (it & 1)]);
        for (int j = lane; j < r; j += 32)
            bulk_g2s(buf + 2 * bgu + j * ad_row, static_cast<const uint8_t*>(lo.A_down) + (((size_t)ad * r + j) * p.I + n0) * 2,
                     ad_row, &bars[BAR_LORA + (it & 1)]);
    };

    // ---- the routing and the first copies (warp 0), around the head rows (every warp).  A chained
    //      step takes its routing from the hand-off ring: the (expert, gate) pairs that the head of
    //      the step before it has left behind its logits, long before that kernel ends.  Its own
    //      head rows come first (pass 0) -- nothing this kernel owes to a later step is ever held
    //      back by a wait -- then warp 0 waits for the pairs (pass 1) and takes; the copies of the
    //      first quarter are issued by all warps right behind the CTA's first barrier.  A step that
    //      is not chained has its routing in memory: warp 0 issues before its head rows.  Bounded wait; on a
    //      time-out fall back to waiting for the whole previous kernel and to the routing it has
    //      written, which is always sufficient.
    // A step whose hidden state is still being produced (dependent chain) routes first as well: its
    // routing is known long before its x, and the first quarter's weights stream in meanwhile.
    const bool early_route = p.flag_in < 0 || p.dep_wait >= 0;
    bool routed = false;                  // warp 0: routing taken, first copies issued
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        if (warp == 0 && !routed && !head_only && (pass || early_route)) {
            int vi[kMaxEpc], vg[kMaxEpc];
#pragma unroll
            for (int e = 0; e < kMaxEpc; ++e) { vi[e] = -1; vg[e] = 0; }
            bool got = false;
            if (p.flag_in >= 0) {
                const unsigned long long* pr = reinterpret_cast<const unsigned long long*>(p.logits_ws + (size_t)p.flag_in * (p.E + kPairWords) + p.E);
                uint32_t it = 0;
                unsigned long long w = 0;
                do {
                    if (lane < p.K) w = ld_relaxed_gpu_u64(pr + lane);
                    got = __all_sync(0xFFFFFFFFu, (uint32_t)w != kNotYet);
                } while (!got && ++it < kSpinLimit);
                if (got) {
                    // everything the writers of this routing had observed (the reduce scratch of this
                    // ring slot being free again, above all) is ordered before what this CTA does next
                    asm volatile("fence.acq_rel.gpu;" ::: "memory");
#pragma unroll
                    for (int e = 0; e < kMaxEpc; ++e) {
                        const unsigned long long we = __shfl_sync(0xFFFFFFFFu, w, (k + e) & 31);
                        if (e < epc_l) { vi[e] = (int)(uint32_t)we; vg[e] = (int)(uint32_t)(we >> 32); }
                    }
                    trace_mark(p, 19);
                } else if (pass) {
                    if (lane == 0) {
                        atomicExch(p.status, EDG_E_TIMEOUT);
                        pdl_wait_prior_grid();
                    }
                    __syncwarp();
                }
            }
            if (p.flag_in < 0 || (!got && pass)) {
#pragma unroll
                for (int e = 0; e < kMaxEpc; ++e)
                    if (e < epc_l && !is_shared) { vi[e] = __ldcg(&p.slots[k + e]); vg[e] = __float_as_int(__ldcg(&p.gates[k + e])); }
                got = true;
            }
            if (is_shared) { vi[0] = 0; vg[0] = __float_as_int(1.f); }      // not routed: always on, weight 1
            if (got) {
                if (lane == 0) {
#pragma unroll
                    for (int e = 0; e < kMaxEpc; ++e) { s_ex[2 * e] = vi[e]; s_ex[2 * e + 1] = vg[e]; }
                }
                __syncwarp();
                trace_mark(p, 14);
                take();
                read_take();
                // A step on its own issues the copies of the first quarter here, ahead of its head
                // rows; in a chained step the other warps are already waiting at the barrier below,
                // and all four issue their share right behind it, which is quicker.
                if (valid && early_route) {
                    issue_gu(0, 0, 0, kFW);
                    if (r > 0) issue_lora(0);
                    if (p.dep_wait >= 0) prefetch_rest(0);
                }
                trace_mark(p, 1);
                routed = true;
            }
        }
        if (pass) break;
        // ---- a dependent step: everything that does not need the hidden state is on its way; now
        //      wait (bounded) until the step before this one has written it
        if (p.dep_wait >= 0) {
            if (warp == 0) {
                // one flag per reducer of the step before (its rows of the state are written): lane c polls flag c
                const float* flag = p.dep_ws + p.dep_wait * kDepWords + 4 + (lane < kC ? lane : 0);
                uint32_t it = 0, v = 0;
                bool all = false;
                do {
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
                    all = __all_sync(0xFFFFFFFFu, v != 0u);
                    if (!all) __nanosleep(40);
                } while (!all && ++it < kSpinLimit);
                if (!all && lane == 0) {               // never seen: the previous kernel's end is always sufficient
                    atomicExch(p.status, EDG_E_TIMEOUT);
                    pdl_wait_prior_grid();
                }
                __syncwarp();
                if (lane == 0) trace_mark(p, 20);
            }
            __syncthreads();
            convert_x();
        }
        // ---- the head on the tensor cores: 16 rows x this warp's K half, the hidden state as column 0
        //      of B (from s_xb, whose words hold (x0,x4) (x1,x5) (x2,x6) (x3,x7): the natural pairs
        //      the fp16 rows need are byte permutations of them)
        if (pre_mma) {
            __syncthreads();                               // s_xb is complete (every CTA passes here: the condition is grid-uniform)
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            if (mma_head) {
                const int nb = p.H / ksplit / 256;         // batches of 8 chunks in this warp's share of K
#pragma unroll 1
                for (int b = 0; b < nb; ++b) {
                    const uint4* xbp = s_xb + (mk0 + b * 256) / 8 + t4;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        uint4 xb = make_uint4(0, 0, 0, 0);
                        if (g8 == 0) {
                            if (EX) {                          // (s_xb holds scaled blocks)
                                const uint4 v = *reinterpret_cast<const uint4*>(p.x + mk0 + b * 256 + j * 32 + t4 * 8);
                                const float f[8] = {bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y), bf16_lo(v.z), bf16_hi(v.z), bf16_lo(v.w), bf16_hi(v.w)};
                                xb = permute8(f);
                            } else xb = xbp[j * 4];
                        }
                        mma16816(c, lw[j].x, lw2[j].x, lw[j].y, lw2[j].y, __byte_perm(xb.x, xb.y, 0x5410), __byte_perm(xb.z, xb.w, 0x5410));
                        mma16816(c, lw[j].z, lw2[j].z, lw[j].w, lw2[j].w, __byte_perm(xb.x, xb.y, 0x7632), __byte_perm(xb.z, xb.w, 0x7632));
                    }
                    if (b + 1 < nb) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            lw[j] = ld_keep16(mwa + (b + 1) * 256 + j * 32);
                            lw2[j] = ld_keep16(mwa + (size_t)8 * p.H + (b + 1) * 256 + j * 32);
                        }
                    }
                }
                // the warps of the upper K shares hand their 16 sums to the warp of the lowest one
                // (s_red is free until the adapter projections, behind the next barriers)
                if (warp >= tpc && t4 == 0) {
                    s_red[(warp / tpc - 1) * 32 + (warp % tpc) * 16 + g8] = c[0];
                    s_red[(warp / tpc - 1) * 32 + (warp % tpc) * 16 + 8 + g8] = c[2];
                }
            }
            __syncthreads();
            if (mma_head && warp < tpc) {
                // rows g and g + 8 sit in the lanes with t4 == 0; lane L < 16 publishes row L of the tile
                float lo_ = c[0], hi_ = c[2];
                for (int q = 0; q + 1 < ksplit; ++q) {       // fixed order
                    lo_ += s_red[q * 32 + warp * 16 + g8];
                    hi_ += s_red[q * 32 + warp * 16 + 8 + g8];
                }
                const float v_lo = __shfl_sync(0xFFFFFFFFu, lo_, (lane & 7) * 4);
                const float v_hi = __shfl_sync(0xFFFFFFFFu, hi_, (lane & 7) * 4);
                if (warp == 0) trace_mark(p, 12);
                publish_logits(p, reinterpret_cast<float*>(smem + p.S.s_topk), lane < 8 ? v_lo : v_hi, mrow0 + lane, lane < 16, lane, pre_state);
                if (warp == 0) trace_mark(p, 13);
            }
        }
        // ---- the head rows (the loads of the first two have been in flight since the kernel started),
        //      published by their warp as soon as they are summed
#pragma unroll 1
        for (int b = 0; pre_fast && b * 2 * kFW < n_pre; ++b) {
            if (!my_row) break;           // (a warp's rows are valid in ascending order)
            float v = 0.f, v2 = 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int i = (j * 32 + lane) * 8;
                if (i < p.H) {
                    const uint4 xv = *reinterpret_cast<const uint4*>(p.x + i);
                    const float x0 = bf16_lo(xv.x), x1 = bf16_hi(xv.x), x2 = bf16_lo(xv.y), x3 = bf16_hi(xv.y);
                    const float x4 = bf16_lo(xv.z), x5 = bf16_hi(xv.z), x6 = bf16_lo(xv.w), x7 = bf16_hi(xv.w);
                    {
                        const uint4 w = lw[j];
                        const float2 a = __half22float2(u32_as_h2(w.x)), b = __half22float2(u32_as_h2(w.y));
                        const float2 d = __half22float2(u32_as_h2(w.z)), f = __half22float2(u32_as_h2(w.w));
                        v = fmaf(a.x, x0, v); v = fmaf(a.y, x1, v); v = fmaf(b.x, x2, v); v = fmaf(b.y, x3, v);
                        v = fmaf(d.x, x4, v); v = fmaf(d.y, x5, v); v = fmaf(f.x, x6, v); v = fmaf(f.y, x7, v);
                    }
                    if (my_row2) {
                        const uint4 w = lw2[j];
                        const float2 a = __half22float2(u32_as_h2(w.x)), b = __half22float2(u32_as_h2(w.y));
                        const float2 d = __half22float2(u32_as_h2(w.z)), f = __half22float2(u32_as_h2(w.w));
                        v2 = fmaf(a.x, x0, v2); v2 = fmaf(a.y, x1, v2); v2 = fmaf(b.x, x2, v2); v2 = fmaf(b.y, x3, v2);
                        v2 = fmaf(d.x, x4, v2); v2 = fmaf(d.y, x5, v2); v2 = fmaf(f.x, x6, v2); v2 = fmaf(f.y, x7, v2);
                    }
                }
            }
            v = warp_sum(v);
            v2 = warp_sum(v2);
            if (warp == 0) trace_mark(p, 12);
            // the next two rows of this warp, if any: on their way while these are published
            const int pe = my_e, pe2 = my_e2;
            const bool prow2 = my_row2;
            const uint32_t ps = pre_state, ps2 = pre_state2;
            {
                const int r1 = warp + kFW * 2 * (b + 1);
                my_e = (int)blockIdx.x + r1 * n_head_ctas;
                my_e2 = (int)blockIdx.x + (r1 + kFW) * n_head_ctas;
                my_row = r1 < n_pre && my_e < p.E;
                my_row2 = r1 + kFW < n_pre && my_e2 < p.E;
                pre_state = kNotYet; pre_state2 = kNotYet;
                if (my_row) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int i = (j * 32 + lane) * 8;
                        lw[j] = i < p.H ? ld_keep16(static_cast<const __half*>(p.W_pre) + (size_t)my_e * p.H + i) : make_uint4(0, 0, 0, 0);
                        if (my_row2) lw2[j] = i < p.H ? ld_keep16(static_cast<const __half*>(p.W_pre) + (size_t)my_e2 * p.H + i) : make_uint4(0, 0, 0, 0);
                    }
                    if (p.flag_out >= 0 && lane == 0) {
                        pre_state = ld_relaxed_gpu_u32(&p.logits_ws[(size_t)p.flag_out * (p.E + kPairWords) + my_e]);
                        if (my_row2) pre_state2 = ld_relaxed_gpu_u32(&p.logits_ws[(size_t)p.flag_out * (p.E + kPairWords) + my_e2]);
                    }
                }
            }
            // both rows in one go: lane 0 publishes the first, lane 1 the second
            const uint32_t st2 = __shfl_sync(0xFFFFFFFFu, ps2, 0);
            publish_logits(p, reinterpret_cast<float*>(smem + p.S.s_topk), lane == 1 ? v2 : v, lane == 1 ? pe2 : pe, lane == 0 || (lane == 1 && prow2), lane,
                         lane == 1 ? st2 : ps);
            if (warp == 0) trace_mark(p, 13);
        }
    }

    // a CTA that is there for the head alone is done (its cluster's handshake completed first)
    if (head_only) {
        cluster_wait();
        trace_mark(p, 9);
        return;
    }

    // ---- any other head (fp32 weights, wider rows): every row is split over all threads of the CTA
    //      and published by one warp after the barrier below
    if (n_pre > 0 && !pre_fast) {
#pragma unroll 1
        for (int ri = 0; ri < n_pre; ++ri) {
            float v = head_row_partial(p.W_pre, p.pre_dtype, p.x, p.H, (int)blockIdx.x + ri * n_head_ctas, tid);
            v = warp_sum(v);
            if (lane == 0) s_red[(kPreRed + ri) * kFW + warp] = v;
        }
    }
    __syncthreads();                      // routing, slot table and x fragments are in shared memory
    if (n_pre > 0 && !pre_fast && warp == kFW - 1) {
        const int e = (int)blockIdx.x + lane * n_head_ctas;
        const bool own = lane < n_pre && e < p.E;
        float v = 0.f;
        if (own)
            for (int w = 0; w < kFW; ++w) v += s_red[(kPreRed + lane) * kFW + w];
        publish_logits(p, reinterpret_cast<float*>(smem + p.S.s_topk), v, e, own, lane, pre_state);
    }

    read_take();
    if (valid && !early_route) {
        issue_gu(0, 0, warp, warp + 1);
        if (warp == kFW - 1 && r > 0) issue_lora(0);
    }
    trace_mark(p, 10);
    cluster_wait();

    if (valid) {
        // ---- with the weights on their way: this CTA's share of the 2r rows of A_gate / A_up, per-warp
        //      partial dot products into s_red.  All threads take part, each covering 8 elements of a
        //      row per sweep; the loads of up to 8 rows are in flight together, so the share costs one
        //      trip to memory.
        const int per = (2 * r + kC - 1) / kC;
        // (a step that has waited for its hidden state finds its first weights landed: it starts on
        // them at once and computes these projections while the second half of K is on its way)
        const bool late_ax = p.dep_wait >= 0;
        auto lora_ax = [&]() {
        if (r > 0) {
#pragma unroll 1
            for (int q0 = 0; q0 < per; q0 += 8) {
                float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
                for (int cc = tid * 8; cc < p.H; cc += kFW * 32 * 8) {
                    const uint4 ux = ld_keep16(p.x + cc);
                    uint4 ua[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int q = min(crank * per + min(q0 + u, per - 1), 2 * r - 1);
                        const int up = q >= r ? 1 : 0;
                        const uint16_t* A = reinterpret_cast<const uint16_t*>(up ? lo.A_up : lo.A_gate) +
                                            ((size_t)ad * r + (q - up * r)) * p.H;
                        ua[u] = ld_keep16(A + cc);
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        v[u] = fmaf(bf16_lo(ua[u].x), bf16_lo(ux.x), v[u]); v[u] = fmaf(bf16_hi(ua[u].x), bf16_hi(ux.x), v[u]);
                        v[u] = fmaf(bf16_lo(ua[u].y), bf16_lo(ux.y), v[u]); v[u] = fmaf(bf16_hi(ua[u].y), bf16_hi(ux.y), v[u]);
                        v[u] = fmaf(bf16_lo(ua[u].z), bf16_lo(ux.z), v[u]); v[u] = fmaf(bf16_hi(ua[u].z), bf16_hi(ux.z), v[u]);
                        v[u] = fmaf(bf16_lo(ua[u].w), bf16_lo(ux.w), v[u]); v[u] = fmaf(bf16_hi(ua[u].w), bf16_hi(ux.w), v[u]);
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float t_ = warp_sum(v[u]);
                    if (lane == 0 && q0 + u < per) s_red[(q0 + u) * kFW + warp] = t_;
                }
            }
        }
        __syncthreads();                  // s_red complete
        // every CTA of the cluster gets this CTA's adapter projections, counted on its BAR_U
        for (int i = tid; i < per * kC; i += kFW * 32) {
            const int qi = i / kC, dst = i % kC, q = crank * per + qi;
            if (q < 2 * r) {
                float v = 0.f;
                for (int w = 0; w < kFW; ++w) v += s_red[qi * kFW + w];
                const int up = q >= r ? 1 : 0;
                st_async_f32(map_to_cta(&s_u[up * kMaxRank + (q - up * r)], dst), v, map_to_cta(&bars[BAR_U], dst));
            }
        }
        trace_mark(p, 2);
        };
        if (!late_ax) lora_ax();

        // ---- the four quarters of the intermediate dimension, one after the other.  For quarter c
        //      this CTA computes its rows_gu gate/up rows (over all of K), the cluster exchanges
        //      h = silu(gate) * up, and the CTA adds the quarter's columns to its rows_d output rows.
        //      The weights stream through the two stage buffers, one load at a time: the first half
        //      of the K range of the gate/up rows (a K quarter per stage), the second half, the
        //      quarter's down block, then the next quarter's first half.
#pragma unroll 1
        for (int w = 0; w < n_items; ++w) {
            const int it = w % p.qpc, c = c0 + it, e = item_expert(w);
            const uint8_t* rec = item_rec(w);
            const uint32_t par = w & 1, par2 = (w >> 1) & 1;
            // the adapter slices of the next quarter go into the buffer the previous quarter used:
            // a score of small copies, issued while this quarter's weights are still on their way
            if (warp == kFW - 1 && r > 0 && w + 1 < n_items) issue_lora(w + 1);
            // ---- gate/up on the tensor cores.  Warp w owns the K range of its NCW chunks (inside
            //      stage w / 2) for every row tile of gate and up; the 16 x 32 codes of a (tile,
            //      chunk) are 256 contiguous bytes of shared memory, lane (g, t) reading word t of
            //      rows g and g+8.  The activations are column 0 of the 8-column B tile: the lanes
            //      of quad 0 read their words from s_xb, every other lane holds zeros.  Partial sums
            //      of a scaled block are exact integer-code dot products in fp32; scale and zero
            //      point are applied per block: acc += s * (c - z * sum(x)).
            {
                const int s = warp / 2;
                const uint8_t* st = smem + S.stage0 + s * S.stage_bytes;
                const int ch0 = (warp & 1) * NCW;                        // first chunk of this warp inside the stage
                constexpr int NT = 2 * TG;                               // (matrix, row tile) pairs, all independent: interleaved
                float a_lo[NT], a_hi[NT];                                // rows g and g+8, column 0
#pragma unroll
                for (int mt = 0; mt < NT; ++mt) { a_lo[mt] = 0.f; a_hi[mt] = 0.f; }
                const uint8_t* cbase = st + ch0 * 256 + g8 * 16 + t4 * 4;
                // the K range in two halves: K quarters 0 and 1 fill the two stages first, quarters 2
                // and 3 follow into the same stages as soon as their two warps are done with them
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    const int vw = warp + kFW * half;                    // this warp's K slice: chunks vw NCW .. vw NCW + NCW - 1 of a row
                    mbar_wait(&bars[s], half, p.status);
                    if (w == 0 && half == 0) trace_mark(p, 3);
                    const uint4* xbp = s_xb + (vw * NCW) * 4 + t4;
#pragma unroll 1
                    for (int ib = 0; ib < NCW / CPB; ++ib) {             // scaled blocks of this warp's K range
                        float cfr[NT][4];
#pragma unroll
                        for (int u = 0; u < CPB; ++u) {
                            const int i = ib * CPB + u;
                            uint4 xb = make_uint4(0, 0, 0, 0);
                            if (g8 == 0) xb = xbp[i * 4];
#pragma unroll
                            for (int mt = 0; mt < NT; ++mt) {
                                const uint8_t* cw = cbase + mt * S.mat_codes + i * 256;
                                uint32_t alo[4], ahi[4];
                                dequant_code_word<EX>(*reinterpret_cast<const uint32_t*>(cw), alo);
                                dequant_code_word<EX>(*reinterpret_cast<const uint32_t*>(cw + 128), ahi);
                                if (u == 0) mma16816_zero(cfr[mt], alo[0], ahi[0], alo[1], ahi[1], xb.x, xb.y);
                                else mma16816(cfr[mt], alo[0], ahi[0], alo[1], ahi[1], xb.x, xb.y);
                                mma16816(cfr[mt], alo[2], ahi[2], alo[3], ahi[3], xb.z, xb.w);
                            }
                        }
                        const int gi = ((ch0 + ib * CPB) * 32) >> p.gshift;
                        const float xs = s_xsum[(vw * NCW) / CPB + ib], xbias = EX ? 0.f : s_xbias[(vw * NCW) / CPB + ib];
#pragma unroll
                        for (int mt = 0; mt < NT; ++mt) {
                            const uint8_t* zw = st + S.sz0 + mt * S.mat_sz + gi * 64 + g8 * 4;
                            const __half2 z0 = u32_as_h2(*reinterpret_cast<const uint32_t*>(zw));
                            const __half2 z1 = u32_as_h2(*reinterpret_cast<const uint32_t*>(zw + 32));
                            a_lo[mt] = fmaf(__low2float(z0), fmaf(-__high2float(z0), xs, EX ? cfr[mt][0] : cfr[mt][0] - xbias), a_lo[mt]);
                            a_hi[mt] = fmaf(__low2float(z1), fmaf(-__high2float(z1), xs, EX ? cfr[mt][2] : cfr[mt][2] - xbias), a_hi[mt]);
                        }
                    }
                    // the second half of the K range follows into the same stages as soon as all
                    // four warps are done with the first
                    if (half == 0) {
                        __syncthreads();
                        issue_gu(w, 1, warp, warp + 1);
                        if (late_ax && w == 0) lora_ax();
                    }
                }
                if (t4 == 0) {
                    const float un = EX ? s_xbias[0] : 1.f;
#pragma unroll
                    for (int mt = 0; mt < NT; ++mt) {
                        s_part[warp * 2 * rows_gu + mt * 16 + g8] = EX ? a_lo[mt] * un : a_lo[mt];
                        s_part[warp * 2 * rows_gu + mt * 16 + 8 + g8] = EX ? a_hi[mt] * un : a_hi[mt];
                    }
                }
            }
            __syncthreads();
            // both stages are free: the quarter's down block follows (a warp that has no part in the sums below issues it)
            if (warp == kFW - 2 && lane < 2) {
                const uint64_t pol = policy_evict_first();
                const uint32_t dcb = (uint32_t)rows_d * sw / 2, dzb = (uint32_t)rows_d * gps * 4;
                if (lane == 0) mbar_expect_tx(&bars[BAR_DOWN], dcb + dzb);
                __syncwarp(0x3u);
                if (lane == 0) bulk_g2s_hint(smem + S.d_codes, rec + p.L.codes_down + down_code_off(p.H, p.I, n0_d, c * (sw / 32)), dcb, &bars[BAR_DOWN], pol);
                else bulk_g2s_hint(smem + S.d_sz, rec + p.L.sz_down + down_sz_off(p.H, p.I, p.group, n0_d, c * gps), dzb, &bars[BAR_DOWN], pol);
            }
            // sum the kFW k-slices: row mt*16 + j of (matrix, tile) order == s_gu[proj * rows_gu + row]
            if (tid < 2 * rows_gu) {
                float v = 0.f;
#pragma unroll
                for (int w = 0; w < kFW; ++w) v += s_part[w * 2 * rows_gu + tid];
                s_gu[tid] = v;
            }
            __syncthreads();
            if (w == 0) {
                trace_mark(p, 4);
                if (r > 0) mbar_wait(&bars[BAR_U], 0, p.status);        // every CTA's A.x has landed in s_u
                trace_mark(p, 5);
            }

            // ---- finish gate/up: LoRA B (one thread per (projection, row)), SiLU, product
            const uint8_t* lbuf = smem + S.lora0 + par * S.lora_bytes;
            if (r > 0 && tid < 2 * rows_gu) {
                mbar_wait(&bars[BAR_LORA + par], par2, p.status);
                const int proj = tid / rows_gu, row = tid % rows_gu;
                const uint16_t* Bm = reinterpret_cast<const uint16_t*>(lbuf) + (proj * rows_gu + row) * r;
                const float d = smem_b_dot(Bm, s_u + proj * kMaxRank, r);
                s_gu[proj * rows_gu + row] = fmaf(p.sigma, d, s_gu[proj * rows_gu + row]);
            }
            __syncthreads();
            if (tid < rows_gu) s_hloc[tid] = silu_f(s_gu[tid]) * s_gu[rows_gu + tid];
            __syncthreads();
            // all-gather h inside the cluster: this CTA's rows_gu values go to every CTA, 16 bytes at a time
            float* hq = s_h + par * sw;
            {
                constexpr int vecs = rows_gu / 4;
                for (int i = tid; i < vecs * kC; i += kFW * 32) {
                    const int v = i % vecs, dst = i / vecs;
                    st_async_f32x4(map_to_cta(&hq[crank * rows_gu + 4 * v], dst), *reinterpret_cast<const float4*>(&s_hloc[4 * v]),
                                   map_to_cta(&bars[BAR_H + par], dst));
                }
            }
            // partial of A_down . h over this CTA's rows of h (kC lanes per rank index), sent to every CTA of the cluster
            float* udp = s_ud_part + par * kC * kMaxRank;
            for (int j = tid / kC; j < r; j += kFW * 32 / kC) {
                const int part = tid % kC;
                const uint16_t* Ad = reinterpret_cast<const uint16_t*>(lbuf + 2 * rows_gu * r * 2) + j * rows_gu;
                float v = 0.f;
                for (int n = part; n < rows_gu; n += kC) v = fmaf(bf16_bits_to_float(Ad[n]), s_hloc[n], v);
                v = group_sum<kC>(v);
                st_async_f32(map_to_cta(&udp[crank * kMaxRank + j], part), v, map_to_cta(&bars[BAR_H + par], part));
            }
            if (w == 0) trace_mark(p, 6);
            mbar_wait(&bars[BAR_H + par], par2, p.status);              // the quarter's h and A_down.h partials
            if (w == 0) trace_mark(p, 7);

            // ---- down on the tensor cores: this quarter's columns for this CTA's H/4 output rows.  h is
            //      fp32: column 0 of the B tile carries its fp16 value, column 1 the fp16 residual
            //      (lanes of quads 0 and 1 read their words from s_hb), and the two result columns
            //      are added.
            if (tid < r) {
                float v = s_ud[tid];
                for (int cc = 0; cc < kC; ++cc) v += udp[cc * kMaxRank + tid];
                s_ud[tid] = v;
            }
            if (tid < DCH * 8) {
                const int i = tid >> 3, lo = (tid >> 2) & 1, q = tid & 3;
                const float4 a = *reinterpret_cast<const float4*>(hq + i * 32 + q * 8);
                const float4 b = *reinterpret_cast<const float4*>(hq + i * 32 + q * 8 + 4);
                const float f[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                if (EX) {
                    constexpr unsigned mask = DCH * 8 == 32 ? 0xFFFFFFFFu : (1u << (DCH * 8)) - 1;
                    const float scale = vector_scale(__reduce_max_sync(mask, abs_max8(f)));
                    s_hb[tid] = lo ? permute8_lo_s(f, scale) : permute8_s(f, scale);
                    if (tid == 0) s_hbias[0] = scale;
                } else s_hb[tid] = lo ? permute8_lo(f) : permute8(f);
            } else if (tid >= 64 && tid < 64 + DCH / CPB) {
                const int j = tid - 64;
                float v = 0.f, vo = 0.f;
                for (int e = 0; e < 32 * CPB; e += 2) {                         // hi + lo == h up to 2^-22: sum h itself
                    v += hq[j * 32 * CPB + e];
                    vo += hq[j * 32 * CPB + e + 1];
                }
                s_hsum[j] = EX ? (v + vo) * kScaleS : v + vo;                  // (EX: without the quarter's power of two)
                if (!EX) s_hbias[j] = fmaf(1024.f, v, 64.f * vo);
            }
            __syncthreads();
            // this buffer's barrier is used again two quarters on: arm it before anyone can send
            if (tid == 0 && w + 2 < n_items) mbar_expect_tx(&bars[BAR_H + par], (uint32_t)(sw + kC * r) * 4u);
            mbar_wait(&bars[BAR_DOWN], par, p.status);
            {
                const uint8_t* dbase = smem + S.d_codes + g8 * 16 + t4 * 4;
                const uint8_t* dsz = smem + S.d_sz;
                const float hscale = EX ? s_hbias[0] : 1.f, hun = EX ? kUnscaleS * vector_unscale(hscale) : 1.f;
                // a warp's row tiles in two passes of TD tiles (the registers of one pass); the sums
                // over the quarters of an expert are kept in s_o, every row by the lane that owns it
#pragma unroll 1
                for (int ps = 0; ps < 2; ++ps) {
                    float acc_lo[TD], acc_hi[TD];                        // rows g and g+8 of TD row tiles
#pragma unroll
                    for (int tt = 0; tt < TD; ++tt) { acc_lo[tt] = 0.f; acc_hi[tt] = 0.f; }
#pragma unroll 1
                    for (int ib = 0; ib < DCH / CPB; ++ib) {
                        float cfr[TD][4];
#pragma unroll
                        for (int u = 0; u < CPB; ++u) {
                            const int i = ib * CPB + u;
                            uint4 hb = make_uint4(0, 0, 0, 0);
                            if (g8 < 2) hb = s_hb[(i * 2 + g8) * 4 + t4];
#pragma unroll
                            for (int tt = 0; tt < TD; ++tt) {
                                const int ti = warp + kFW * (ps * TD + tt);
                                const uint8_t* cw = dbase + (ti * DCH + i) * 256;
                                uint32_t alo[4], ahi[4];
                                dequant_code_word<EX>(*reinterpret_cast<const uint32_t*>(cw), alo);
                                dequant_code_word<EX>(*reinterpret_cast<const uint32_t*>(cw + 128), ahi);
                                if (u == 0) mma16816_zero(cfr[tt], alo[0], ahi[0], alo[1], ahi[1], hb.x, hb.y);
                                else mma16816(cfr[tt], alo[0], ahi[0], alo[1], ahi[1], hb.x, hb.y);
                                mma16816(cfr[tt], alo[2], ahi[2], alo[3], ahi[3], hb.z, hb.w);
                            }
                        }
                        const int gi = (ib * CPB * 32) >> p.gshift;
                        const float hs = EX ? s_hsum[ib] * hscale : s_hsum[ib], hbias = EX ? 0.f : s_hbias[ib];
#pragma unroll
                        for (int tt = 0; tt < TD; ++tt) {
                            const int ti = warp + kFW * (ps * TD + tt);
                            const uint8_t* zw = dsz + (ti * gps + gi) * 64 + g8 * 4;
                            const __half2 z0 = u32_as_h2(*reinterpret_cast<const uint32_t*>(zw));
                            const __half2 z1 = u32_as_h2(*reinterpret_cast<const uint32_t*>(zw + 32));
                            acc_lo[tt] = fmaf(__low2float(z0), fmaf(-__high2float(z0), hs, EX ? cfr[tt][0] + cfr[tt][1] : cfr[tt][0] + cfr[tt][1] - hbias), acc_lo[tt]);
                            acc_hi[tt] = fmaf(__low2float(z1), fmaf(-__high2float(z1), hs, EX ? cfr[tt][2] + cfr[tt][3] : cfr[tt][2] + cfr[tt][3] - hbias), acc_hi[tt]);
                        }
                    }
                    if (t4 == 0) {
#pragma unroll
                        for (int tt = 0; tt < TD; ++tt) {
                            const int ti = warp + kFW * (ps * TD + tt);
                            // (the first quarter of an expert starts the sums)
                            const float vl = EX ? acc_lo[tt] * hun : acc_lo[tt], vh = EX ? acc_hi[tt] * hun : acc_hi[tt];
                            s_o[ti * 16 + g8] = it ? s_o[ti * 16 + g8] + vl : vl;
                            s_o[ti * 16 + 8 + g8] = it ? s_o[ti * 16 + 8 + g8] + vh : vh;
                        }
                    }
                }
            }
            // the next quarter's K quarters 0-1 go into the stages once every warp is done with the down block
            if (w + 1 < n_items) {
                __syncthreads();
                issue_gu(w + 1, 0, warp, warp + 1);
            }
            if (w == 0) trace_mark(p, 24);

            // ---- the last quarter of an expert: its gate-weighted output rows go to the reduce scratch
            if (it == p.qpc - 1) {
                __syncthreads();          // s_o and s_ud complete
                // LoRA B for down (A_down.h summed over the quarters; the rows of B_down come
                // straight from memory, 2r bytes each) and the gate weight: one thread per output row
                const float gate_k = __int_as_float(s_ex[20 + e]);
                float* prow = partial + ((size_t)(k + e) * nq + cq) * p.H + n0_d;
                const uint16_t* Bd = static_cast<const uint16_t*>(lo.B_down) + ((size_t)ad * p.H + n0_d) * r;
                constexpr int kRowsPerThread = rows_d / (kFW * 32);
                float dl[kRowsPerThread];
#pragma unroll
                for (int q = 0; q < kRowsPerThread; ++q) {
                    dl[q] = 0.f;
                    if (r > 0) dl[q] = gmem_b_dot(Bd + (size_t)(tid + q * kFW * 32) * r, s_ud, r);
                }
#pragma unroll
                for (int q = 0; q < kRowsPerThread; ++q) {
                    const int lr = tid + q * kFW * 32;
                    prow[lr] = gate_k * fmaf(p.sigma, dl[q], s_o[lr]);
                }
                if (w + 1 < n_items) {   // another expert follows: its A_down.h starts from zero
                    __syncthreads();
                    if (tid < kMaxRank) s_ud[tid] = 0.f;
                }
            }
        }
        trace_mark(p, 8);
    }
    // a skipped expert contributes nothing
    if (s_ex[8] != epc_l) {
        if (tid == 0) atomicExch(p.status, EDG_E_RANGE);
        for (int e = 0; e < epc_l; ++e)
            if (!((s_ex[10] >> e) & 1))
                for (int i = tid; i < rows_d; i += kFW * 32) partial[((size_t)(k + e) * nq + cq) * p.H + n0_d + i] = 0.f;
    }

    // ---- a6: this partial is published; the last arriver for the block of rows sums all partials.
    //      The counting atomic of thread 0, behind the CTA's barrier, releases the partial rows of all its
    //      threads and, in the last arriver, acquires everyone else's (read past the L1 below).
    __syncthreads();
    if (tid == 0) s_flag[0] = (atom_add_acq_rel_gpu(&counters[crank], 1) == n_expert_ctas / kC - 1) ? 1 : 0;   // one arrival per cluster of experts
    __syncthreads();
    if (s_flag[0]) {
        // (sixteen partials in flight per thread and round: this sum is on the critical path of a step that runs alone;
        //  a thread owns one group of four rows: rows_d / 4 <= 128)
        const int i = tid;
        const bool on = i < rows_d / 4;
        uint2 xr = make_uint2(0u, 0u);
        float4 yv = make_float4(0.f, 0.f, 0.f, 0.f);
        float ss = 0.f;
        if (on) {
            if (p.x_next != nullptr) xr = *reinterpret_cast<const uint2*>(p.x + n0_d + 4 * i);
#pragma unroll 1
            for (int k0 = 0; k0 < np; k0 += 16) {
                float4 t[16];
#pragma unroll
                for (int u = 0; u < 16; ++u)
                    t[u] = k0 + u < np ? __ldcg(reinterpret_cast<const float4*>(&partial[(size_t)(k0 + u) * p.H + n0_d + 4 * i]))
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int u = 0; u < 16; ++u) { yv.x += t[u].x; yv.y += t[u].y; yv.z += t[u].z; yv.w += t[u].w; }
            }
            store_y4(p.y, p.out_dtype, (size_t)n0_d + 4 * i, yv);
            if (p.x_next != nullptr) {           // x + y with y as stored (rounded to the output type), and its squares
                yv.x = bf16_lo(xr.x) + round_out(yv.x, p.out_dtype); yv.y = bf16_hi(xr.x) + round_out(yv.y, p.out_dtype);
                yv.z = bf16_lo(xr.y) + round_out(yv.z, p.out_dtype); yv.w = bf16_hi(xr.y) + round_out(yv.w, p.out_dtype);
                ss = fmaf(yv.x, yv.x, ss); ss = fmaf(yv.y, yv.y, ss); ss = fmaf(yv.z, yv.z, ss); ss = fmaf(yv.w, yv.w, ss);
            }
        }
        if (tid == 0) counters[crank] = 0;
        if (p.x_next != nullptr) {
            // ---- the next hidden state of a dependent chain, x_next = bf16(rmsnorm(x + y)).  Each of the kC
            //      reducers sums the squares of its rows, publishes the sum, waits (bounded) until all kC
            //      sums are there -- the reducers are running CTAs that publish before they wait --, adds
            //      them in a fixed order and normalises the rows it still holds in registers.  The last one
            //      to have written its rows raises the flag the next step waits for.
            ss = warp_sum(ss);
            if (lane == 0) s_red[warp] = ss;
            __syncthreads();
            if (tid == 0) {
                float tot = 0.f;
                for (int w = 0; w < kFW; ++w) tot += s_red[w];
                st_relaxed_gpu_u32(p.dep_ws + p.ring * kDepWords + crank, __float_as_uint(tot));
                int seen = atom_add_acq_rel_gpu(&p.norm_cnt[p.ring], 1) + 1;
                uint32_t it = 0;
                while ((seen & 0xFF) < kC && ++it < kSpinLimit) {
                    __nanosleep(20);
                    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(p.norm_cnt + p.ring) : "memory");
                }
                if ((seen & 0xFF) < kC) atomicExch(p.status, EDG_E_TIMEOUT);
                float all = 0.f;
                for (int c = 0; c < kC; ++c) all += __uint_as_float(ld_relaxed_gpu_u32(p.dep_ws + p.ring * kDepWords + c));
                s_red[kFW] = rsqrtf(all / (float)p.H + p.eps);
            }
            __syncthreads();
            if (on) {
                const float inv = s_red[kFW];
                bf16_t* xn = reinterpret_cast<bf16_t*>(p.x_next) + n0_d + 4 * i;
                store_out<bf16_t>(xn, 0, yv.x * inv);
                store_out<bf16_t>(xn, 1, yv.y * inv);
                store_out<bf16_t>(xn, 2, yv.z * inv);
                store_out<bf16_t>(xn, 3, yv.w * inv);
            }
            __syncthreads();                      // this CTA's rows of the next state are written
            if (tid == 0) {
                // (the release covers the rows every thread of this CTA wrote before the barrier)
                asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p.dep_ws + p.ring * kDepWords + 4 + crank), "r"(1u) : "memory");
                trace_stamp(p, 21);
                // off the critical path: the last reducer past the exchange of sums resets the counter (arrivals in its low byte,
                // reducers past the exchange above it)
                if (atom_add_acq_rel_gpu(&p.norm_cnt[p.ring], 256) >> 8 == kC - 1) st_relaxed_gpu(p.norm_cnt + p.ring, 0);
            }
        }
        if (p.flag_in >= 0) {
            // The last of the kC reducers resets the ring slot this step has taken its logits from.
            // By then every CTA has read them and the reduce scratch of this ring slot is free
            // again; the step that reuses either gets its own routing only after this.
            if (p.slot_until_end) pdl_wait_prior_grid();
            __threadfence();
            __syncthreads();
            if (tid == 0) s_flag[3] = (atomicAdd(&p.done[p.flag_in], 1) == kC - 1) ? 1 : 0;
            __syncthreads();
            if (s_flag[3]) {
                if (tid == 0) p.done[p.flag_in] = 0;
                // (the routing pairs behind the logits first: whoever finds a logit reset finds them reset too)
                for (int i = tid; i < kPairWords; i += kFW * 32)
                    st_relaxed_gpu_u32(&p.logits_ws[(size_t)p.flag_in * (p.E + kPairWords) + p.E + i], kNotYet);
                __threadfence();
                __syncthreads();
                for (int i = tid; i < p.E; i += kFW * 32)
                    st_relaxed_gpu_u32(&p.logits_ws[(size_t)p.flag_in * (p.E + kPairWords) + i], kNotYet);
            }
        }
    }
    // Kernels of a chain complete in order: one CTA of every grid waits for the grid before it, so
    // work queued after the last kernel of a chain finds all of them finished.
    if (p.flag_in >= 0 && blockIdx.x == 0) pdl_wait_prior_grid();
    trace_mark(p, 9);
}

// ---------------------------------------------------------------- host side

static unsigned long long* g_trace = nullptr;     // set by edg_set_trace_buffer
unsigned long long* trace_buffer() { return g_trace; }

constexpr size_t kFusedSmemLimit = 56 * 1024;     // four CTAs per SM

bool fused_supported(const edg_layer_desc& d) {
    if (!((d.H == 1024 || d.H == 2048) && (d.I == 256 || d.I == 512))) return false;
    if ((d.I / kE16) % 16 != 0 || d.I / kE16 > 32) return false;   // whole 16-row tiles per CTA
    // the head rows are dealt to the first CTAs of the grid, at most kMaxPre each
    const int max_pre = (d.pre_dtype == EDG_F16 && d.H <= 2048) ? kMaxPre : kFW;
    const int need = (d.E + max_pre - 1) / max_pre;
    const int grid = d.K * kC, head_ctas = grid < 32 ? grid : (grid < need ? grid : (need > 32 ? need : 32));
    if (head_ctas * max_pre < d.E) return false;
    if (d.group > 128 || (d.group & (d.group - 1)) != 0) return false;
    if (d.rank % 8 != 0) return false;            // adapter slices are staged by 16-byte bulk copies
    return fused_smem(d.H, d.I, d.E, d.group, d.rank).total <= kFusedSmemLimit;
}

template <int NCW, int DCH, int TG, int TD, int CPB, bool EX>
static cudaError_t launch_form(const FusedParams& p, size_t smem, bool pdl, cudaStream_t st) {
    auto kern = fused_layer_kernel<NCW, DCH, TG, TD, CPB, EX>;
    static OncePerDevice once;
    const cudaError_t e = once([&] {
        const cudaError_t s = allow_smem(kFusedSmemLimit, kern);
        // four CTAs per SM: more clusters resident at once
        return s != cudaSuccess ? s : cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((p.K / p.epc + p.n_shared) * (kDownSlices / p.qpc) * kC + p.head_extra, 1, 1);
    cfg.blockDim = dim3(kFW * 32, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kC;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, p);
}

// Steps of a dependent chain (they write the next hidden state) keep the biased code arithmetic, all others take the subnormal
// form (edg_mma.cuh): the 1280-step burst of the 35B-class layer 4.42 -> 4.25 ms, two subtractions per scaled block fewer.
template <int NCW, int DCH, int TG, int TD, int CPB>
static cudaError_t launch_fused(const FusedParams& p, size_t smem, bool pdl, cudaStream_t st) {
    return p.x_next == nullptr ? launch_form<NCW, DCH, TG, TD, CPB, true>(p, smem, pdl, st)
                               : launch_form<NCW, DCH, TG, TD, CPB, false>(p, smem, pdl, st);
}

// One fused launch for a batch-1 layer-step.  W_pre may be null (no prediction).
int32_t run_fused_layer(const edg_layer_desc* d, const void* slot_pool, const int32_t* slots, const int32_t* table,
                        const int32_t* experts, const float* gates, const void* x, const edg_lora* lora, void* y,
                        const void* W_pre, int32_t* inds_next, float* gates_next, float* logits_next,
                        void* workspace, int flag_in, int flag_out, int ring, cudaStream_t st,
                        const FusedExtras* extras) {
    const bool has_lora = lora != nullptr && d->rank > 0;
    FusedParams p{};
    p.pool = static_cast<const uint8_t*>(slot_pool);
    p.slots = slots; p.table = table; p.experts = experts; p.gates = gates;
    p.x = static_cast<const uint16_t*>(x);
    if (has_lora) p.lora = *lora;
    p.y = y;
    const WorkspaceLayout W = workspace_layout(*d, 1);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    p.status = reinterpret_cast<int32_t*>(ws + W.ctrl);
    p.counters = reinterpret_cast<int32_t*>(ws + W.ctrl + kCtrlCounters);
    p.pre_counter = reinterpret_cast<int32_t*>(ws + W.ctrl + kCtrlHead);
    p.partial = reinterpret_cast<float*>(ws + W.partial);
    p.logits_ws = reinterpret_cast<float*>(ws + W.logits);
    p.W_pre = W_pre; p.inds_next = inds_next; p.gates_next = gates_next; p.logits_next = logits_next;
    p.H = d->H; p.I = d->I; p.E = d->E; p.K = d->K; p.group = d->group;
    p.rank = has_lora ? d->rank : 0;
    if (extras != nullptr && extras->shared_rec != nullptr) {
        p.shared_rec = static_cast<const uint8_t*>(extras->shared_rec);
        p.n_shared = 1;
        if (extras->shared_lora != nullptr && d->rank > 0) { p.shared_lora = *extras->shared_lora; p.rank_shared = d->rank; }
    }
    p.n_adapters = d->n_adapters; p.n_slots = d->n_slots;
    p.pre_dtype = d->pre_dtype; p.out_dtype = d->out_dtype;
    p.sigma = d->lora_scale;
    p.L = record_layout(d->H, d->I, d->group);
    p.S = fused_smem(d->H, d->I, d->E, d->group, p.rank > p.rank_shared ? p.rank : p.rank_shared);
    p.gshift = 0;
    while ((1 << p.gshift) < d->group) ++p.gshift;
    p.trace = g_trace;
    p.done = reinterpret_cast<int32_t*>(ws + W.ctrl + kCtrlDone);
    p.ring = ring;
    p.dep_wait = -1;
    if (extras != nullptr) {
        p.inds_mirror = extras->inds_mirror;
        p.x_next = static_cast<uint16_t*>(extras->x_next);
        p.eps = extras->eps;
        p.dep_wait = flag_in >= 0 ? extras->dep_wait : -1;
        p.slot_until_end = extras->slot_until_end ? 1 : 0;
    }
    p.dep_ws = reinterpret_cast<float*>(ws + W.dep);
    p.norm_cnt = reinterpret_cast<int32_t*>(ws + W.ctrl + kCtrlNorm);
    // a chained step shares the GPU with its neighbours: few, long-lived CTAs; a lone step wants all SMs at once
    // (a step of a dependent chain runs one after the other however it is launched: all SMs at once too)
    p.qpc = (flag_in >= 0 && p.dep_wait < 0) ? kDownSlices : 1;
    // ... and when the experts share one adapter a cluster takes two or four experts, one after the other:
    // fewer CTAs per step, each amortising its start-up over more bytes
    const bool fast_head = W_pre == nullptr || (d->pre_dtype == EDG_F16 && d->H <= 2048);   // up to 8 kFW head rows per CTA
    p.epc = 1;
    for (int c = 2; c <= kMaxEpc; c *= 2)
        if (flag_in >= 0 && p.qpc == kDownSlices && d->K % c == 0 && (p.rank == 0 || d->n_adapters == 1) && fast_head && (W_pre == nullptr || (d->K / c) * kC * kMaxPre >= d->E))
            p.epc = c;
    p.flag_in = flag_in;
    p.flag_out = W_pre != nullptr ? flag_out : -1;
    // a step that runs alone gives an fp16 head CTAs of its own: one 16-row MMA tile each, whole clusters
    p.head_extra = 0;
    if (p.qpc == 1 && W_pre != nullptr && d->pre_dtype == EDG_F16 && d->E % 16 == 0 && d->H % 1024 == 0)
        p.head_extra = (d->E / 16 + kC - 1) / kC * kC;
    const bool pdl = flag_in >= 0;
    const size_t smem = p.S.total;
    cudaError_t e;
    const bool wide = d->group >= 64;         // scaled blocks of 64 codes (groups of 64 or 128) or of 32
    if (d->H == 2048 && d->I == 512) e = wide ? launch_fused<8, 4, 2, 4, 2>(p, smem, pdl, st) : launch_fused<8, 4, 2, 4, 1>(p, smem, pdl, st);
    else if (d->H == 2048 && d->I == 256) e = wide ? launch_fused<8, 2, 1, 4, 2>(p, smem, pdl, st) : launch_fused<8, 2, 1, 4, 1>(p, smem, pdl, st);
    else if (d->H == 1024 && d->I == 512) e = wide ? launch_fused<4, 4, 2, 2, 2>(p, smem, pdl, st) : launch_fused<4, 4, 2, 2, 1>(p, smem, pdl, st);
    else if (d->H == 1024 && d->I == 256) e = wide ? launch_fused<4, 2, 1, 2, 2>(p, smem, pdl, st) : launch_fused<4, 2, 1, 2, 1>(p, smem, pdl, st);
    else return EDG_E_SHAPE;
    EDG_CUDA_TRY(e);
    return EDG_OK;
}

}  // namespace edg

// Tracing hook: with a device buffer of (CTAs in the grid) x kTraceMarks uint64, every CTA of the
// fused layer kernel stamps %globaltimer (ns) at its phase boundaries (the header lists the slots).
// NULL switches tracing off.
extern "C" int32_t edg_set_trace_buffer(void* dev_buffer) {
    edg::g_trace = static_cast<unsigned long long*>(dev_buffer);
    return EDG_OK;
}
