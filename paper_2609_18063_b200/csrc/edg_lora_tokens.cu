// The rank-r projections of the unmerged adapter (Sec. 3.3: delta = sigma * B (A v)) for the tcgen05 tiles of many tokens:
// u = sigma A_gate x and sigma A_up x before gate/up, u_d = sigma A_down h before down, fp16 as the tiles' operands take them.  Adapter
// rows are the rows of m16n8k16 tiles, tokens (16 for A x) or pairs (32 for A_down h) their columns, so an A row is read once per 16 or 32;
// K is split over the warps and summed through shared memory, in fixed order.  With one adapter per layer A x is computed per token, with one per expert per
// pair, tile by tile (all pairs of a tile have one expert).  x and its adapter rows are bf16 as they are.  h of one adapter of
// up to 32 ranks (I 256 or 512) is the tiles' fp16 value and residual (two MMAs), the adapter rows are fp16 (exact in the normal range);
// otherwise h is fp32, the exact sum of three bf16 (three MMAs), the rows are bf16 as they are, and any magnitude keeps its bits.
// Accumulation is fp32.
#include "edg_grouped.cuh"
#include "edg_ptx.cuh"

namespace edg {
namespace {

constexpr int L_WARPS = 8;

// X: u_gu[token or pair][2 rank] = sigma A x, rows 0 .. r-1 from A_gate, r .. 2r-1 from A_up.  Otherwise u_d[pair][rank] = sigma A_down h.
// blockIdx.x: 8 N tokens, or that part of a tile; blockIdx.y: 16 M rows.  WIDE: h from p.hf.
template <bool X, int M, int N, bool WIDE>
__global__ void __launch_bounds__(L_WARPS * 32, M == 1 && !WIDE ? 3 : 2) lora_rows_kernel(const __grid_constant__ GroupedParams p) {
    constexpr int L_ROWS = 16 * M, L_TOK = 8 * N, SUBS = kUmmaTokens / L_TOK;
    __shared__ float s_red[L_WARPS * L_ROWS * (L_TOK + 1)];
    __shared__ int s_id[L_TOK];                                          // where a column's results go: a token or a pair, or -1
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g8 = lane >> 2, t4 = lane & 3;
    pdl_launch_dependents();
    pdl_wait_prior_grid();
    const bool by_token = X && p.n_adapters == 1;
    const int tile = blockIdx.x / SUBS, sub = blockIdx.x % SUBS;
    int ad = 0, cnt, n16 = 0, first = 0;
    if (by_token) {
        cnt = min(L_TOK, p.T - (int)blockIdx.x * L_TOK);
    } else {
        if (tile >= *p.n_tiles) return;
        const int4 ti = p.tiles[tile];
        cnt = min(L_TOK, ti.z - sub * L_TOK);
        if (cnt <= 0) return;
        n16 = (ti.z + 15) & ~15;
        first = ti.y + sub * L_TOK;
        ad = ti.w;
    }
    if (tid < L_TOK) s_id[tid] = tid >= cnt ? -1 : (by_token ? (int)blockIdx.x * L_TOK + tid : p.order[first + tid]);
    __syncthreads();
    const int rows = X ? 2 * p.rank : p.rank, row0 = blockIdx.y * L_ROWS, nt = (cnt + 7) >> 3, K = X ? p.H : p.I;
    const uint16_t* A[M][2];
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int row = row0 + m * 16 + hh * 8 + g8;
            const uint16_t* base = static_cast<const uint16_t*>(X ? (row < p.rank ? p.lora.A_gate : p.lora.A_up) : p.lora.A_down);
            A[m][hh] = row < rows ? base + ((size_t)ad * p.rank + (X && row >= p.rank ? row - p.rank : row)) * K + 8 * t4 : nullptr;
        }
    float c[M][N][4];
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
        for (int n = 0; n < N; ++n)
#pragma unroll
            for (int q = 0; q < 4; ++q) c[m][n][q] = 0.f;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    const uint16_t* xr[N];
    if (X)
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const int id = s_id[n * 8 + g8];
            xr[n] = id < 0 ? nullptr : p.x + (size_t)(by_token ? id : id / p.K) * p.H + 8 * t4;
        }
    const uint8_t* hq = p.hq + (size_t)tile * p.I * 512 + (size_t)t4 * n16 * 16 + (sub * L_TOK + g8) * 16;
    const float* hf = WIDE ? p.hf + (size_t)tile * p.I * 128 + ((size_t)t4 * n16 + sub * L_TOK + g8) * 8 : nullptr;
    // X: the warp's eighth of K, 32 k at a time; h: every eighth chunk of 32
#pragma unroll X ? 4 : 2
    for (int kb = X ? warp * (K / L_WARPS) : warp * 32; kb < (X ? (warp + 1) * (K / L_WARPS) : K); kb += X ? 32 : L_WARPS * 32) {
        uint4 a[M][2], b[N], bl[N];                                      // (WIDE: b, bl are the bits of the eight floats)
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) a[m][hh] = A[m][hh] != nullptr ? __ldg(reinterpret_cast<const uint4*>(A[m][hh] + kb)) : zero;
#pragma unroll
        for (int n = 0; n < N; ++n) {
            b[n] = zero; bl[n] = zero;
            if (X) {
                if (xr[n] != nullptr) b[n] = __ldg(reinterpret_cast<const uint4*>(xr[n] + kb));
            } else if (WIDE && sub * L_TOK + n * 8 < n16) {
                const uint4* q = reinterpret_cast<const uint4*>(hf + (size_t)(kb >> 3) * n16 * 8 + n * 64);
                b[n] = __ldcg(q);
                bl[n] = __ldcg(q + 1);
            } else if (sub * L_TOK + n * 8 < n16) {
                const uint8_t* q = hq + (size_t)(kb >> 5) * n16 * 128 + n * 128;
                b[n] = __ldcg(reinterpret_cast<const uint4*>(q));
                bl[n] = __ldcg(reinterpret_cast<const uint4*>(q + (size_t)n16 * 64));
            }
        }
#pragma unroll
        for (int m = 0; m < M; ++m) {
            if (!X && !WIDE) { a[m][0] = bf16x8_permute8(a[m][0]); a[m][1] = bf16x8_permute8(a[m][1]); }
#pragma unroll
            for (int n = 0; n < N; ++n) {
                if (n >= nt) continue;
                if (X) {
                    mma16816_bf16(c[m][n], a[m][0].x, a[m][1].x, a[m][0].y, a[m][1].y, b[n].x, b[n].y);
                    mma16816_bf16(c[m][n], a[m][0].z, a[m][1].z, a[m][0].w, a[m][1].w, b[n].z, b[n].w);
                } else if (WIDE) {
                    const float4 v = *reinterpret_cast<const float4*>(&b[n]), w = *reinterpret_cast<const float4*>(&bl[n]);
                    const float f[8] = {v.x, v.y, v.z, v.w, w.x, w.y, w.z, w.w};
                    uint32_t part[3][4];
                    bf16_parts(f, part);
#pragma unroll
                    for (int q = 2; q >= 0; --q) {
                        mma16816_bf16(c[m][n], a[m][0].x, a[m][1].x, a[m][0].y, a[m][1].y, part[q][0], part[q][1]);
                        mma16816_bf16(c[m][n], a[m][0].z, a[m][1].z, a[m][0].w, a[m][1].w, part[q][2], part[q][3]);
                    }
                } else {
                    mma16816(c[m][n], a[m][0].x, a[m][1].x, a[m][0].y, a[m][1].y, b[n].x, b[n].y);
                    mma16816(c[m][n], a[m][0].z, a[m][1].z, a[m][0].w, a[m][1].w, b[n].z, b[n].w);
                    mma16816(c[m][n], a[m][0].x, a[m][1].x, a[m][0].y, a[m][1].y, bl[n].x, bl[n].y);
                    mma16816(c[m][n], a[m][0].z, a[m][1].z, a[m][0].w, a[m][1].w, bl[n].z, bl[n].w);
                }
            }
        }
    }
#pragma unroll
    for (int m = 0; m < M; ++m)
#pragma unroll
        for (int n = 0; n < N; ++n) {
            float* q = s_red + (warp * L_ROWS + m * 16 + g8) * (L_TOK + 1) + n * 8 + 2 * t4;
            q[0] = c[m][n][0]; q[1] = c[m][n][1];
            q[8 * (L_TOK + 1)] = c[m][n][2]; q[8 * (L_TOK + 1) + 1] = c[m][n][3];
        }
    __syncthreads();
    __half* out = X ? p.u_gu : p.u_d;
    for (int i = tid; i < L_ROWS * L_TOK; i += L_WARPS * 32) {
        const int row = i % L_ROWS, tok = i / L_ROWS;
        if (tok >= cnt || row0 + row >= rows) continue;
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < L_WARPS; ++w) v += s_red[(w * L_ROWS + row) * (L_TOK + 1) + tok];
        out[(size_t)s_id[tok] * rows + row0 + row] = __float2half_rn(p.sigma * v);
    }
}

}  // namespace

// 4096 tokens of 8 choices, rank 16: 9 and 23 us.  (Not kept: 32 tokens or pairs and 32 rows a CTA in both, one CTA an SM for its registers: 27 and 77.)
cudaError_t launch_lora_ax(const GroupedParams& p, int max_tiles, cudaStream_t st) {
    if (p.n_adapters == 1) return launch_pdl(lora_rows_kernel<true, 2, 2, false>, dim3((unsigned)(p.T + 15) / 16, (2 * p.rank + 31) / 32), L_WARPS * 32, 0, st, p);
    return launch_pdl(lora_rows_kernel<true, 2, 2, false>, dim3(8u * max_tiles, (2 * p.rank + 31) / 32), L_WARPS * 32, 0, st, p);
}
cudaError_t launch_lora_adh(const GroupedParams& p, int max_tiles, cudaStream_t st) {
    return launch_pdl(p.hf != nullptr ? lora_rows_kernel<false, 1, 4, true> : lora_rows_kernel<false, 1, 4, false>, dim3(4u * max_tiles, (p.rank + 15) / 16), L_WARPS * 32, 0, st, p);
}

}  // namespace edg
