// Parameters shared by the grouped (T > 1) kernels: the streaming form for small groups and the
// tcgen05 tiles for large ones.
#pragma once

#include "edg_mma.cuh"

namespace edg {

struct GroupedParams {
    const uint8_t* pool;
    const int32_t* slots;     // [T][K] slots, or expert ids when table != null
    const int32_t* table;
    const int32_t* experts;
    const float* gates;       // [T][K]
    const uint16_t* x;        // [T][H] bf16
    edg_lora lora;
    void* y;
    int32_t* status;
    __half* u_gu;             // [T, or T*K with an adapter per expert][2][rank]  sigma (A_gate x), sigma (A_up x)
    __half* u_d;              // [T*K][rank]                                      sigma (A_down h)
    float* o;                 // [T*K][H]
    int32_t* pair_slot;       // [T*K]
    int32_t* order;           // [T*K] pairs sorted by slot
    int4* tiles;              // {slot, first position in order, pairs, adapter} of every tile of 128 pairs
    int32_t* n_tiles;
    uint8_t* hq;              // h of every tile as fp16 operand tiles, value and residual
    float* hf;                // h as it is, [tile][8 rows of h][pair][8], or null
    uint8_t* xq;              // the gathered token states of every tile as fp16 operand tiles
    int T, H, I, E, K, group, gshift, rank, n_adapters, n_slots, out_dtype;
    float sigma;
    RecordLayout L;
};

// tcgen05 path for large groups (prefill): tiles of 128 tokens
constexpr int kUmmaTokens = 128;
// Where the 128-token tiles overtake the streaming form, in pairs per slot (us, streaming : tcgen05; H 2048, I 512, groups of 64 where
// nothing else is said).  256 experts, top 8: 32 422 : 452, 64 701 : 454; 64 experts: 41 156 : 132, 64 200 : 149; 2 experts: 42 79 : 54;
// groups of 128: 21 185 : 220, 40 263 : 249; H 1024, I 256, 16 experts: 41 54.5 : 44.7, 64 56 : 48.  The average says enough of steeper and
// sparser routing, where the tiles gain less and more: Zipf(2.0) over 256 experts 41 483 : 443, 64 698 : 538, over 64 of H 512, I 256 64
// 45.7 : 45.3; 32 of 256 slots in use 41 422 : 240.  With groups of 32 the sums leave tensor memory twice as often: 64 214 : 230, 128 322 : 296.
// Beyond 1024 slots (no table names more) the line stays where it was: what is counted per slot of the pool says nothing about the slots
// in use then, each slot has a CTA that reads all pairs, and with 65,535 tokens of 32 choices the tiles would not fit a grid.
constexpr int kUmmaPairsPerSlot = 40, kUmmaPairsPerSlot32 = 96, kUmmaSlots = 1024;
bool umma_grouped_supported(const edg_layer_desc& d);
cudaError_t launch_umma(const GroupedParams& p, bool down, int max_tiles, cudaStream_t st);

// streaming form for small and middling groups (edg_grouped_ffn.cu)
int32_t run_grouped_ffn(const edg_layer_desc* d, const GroupedParams& p, const WorkspaceLayout& W, uint8_t* ws, cudaStream_t st);
cudaError_t launch_sum_choices(const GroupedParams& p, cudaStream_t st);

// adapter projections of the tcgen05 path (edg_lora_tokens.cu): A_gate x and A_up x; A_down h from the tiles' h
cudaError_t launch_lora_ax(const GroupedParams& p, int max_tiles, cudaStream_t st);
cudaError_t launch_lora_adh(const GroupedParams& p, int max_tiles, cudaStream_t st);

}  // namespace edg
