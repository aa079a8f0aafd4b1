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
    float* u_gu;              // [T][n_sets][2][rank]
    float* h;                 // [T*K][I]
    float* u_d;               // [T*K][rank]
    float* o;                 // [T*K][H]
    int32_t* pair_slot;       // [T*K]
    int32_t* pair_ad;         // [T*K]
    int32_t* counts;          // [n_slots]
    int32_t* lists;           // [n_slots][T]
    int32_t* tiles;           // [max tiles][2] = (slot, first position in the slot's list)
    int32_t* n_tiles;
    uint8_t* hq;              // h of every 128-token tile as fp16 operand tiles (tcgen05 path)
    uint8_t* xq;              // the gathered token states of every tile as fp16 operand tiles (tcgen05 path)
    int T, H, I, E, K, group, rank, n_adapters, n_slots, out_dtype;
    int ntok;                 // tokens per tile of the tcgen05 engine (128)
    float sigma;
    RecordLayout L;
};

// tcgen05 path for large groups (prefill): tiles of 128 tokens
constexpr int kUmmaTokens = 128;
// Where the 128-token tiles overtake the streaming form, by the layer of 256 experts (us, streaming against tcgen05): 87 pairs per slot
// 920 : 947, 128 1297 : 1166.  Smaller layers would cross later, and lose what lies between: 64 experts, 62 361 : 384, 125 667 : 675,
// 256 1286 : 1203; H 1024, I 256, 250 85 : 131, 1024 243 : 218.  (A line by the layer's size and the units per SM is not worked out.)
constexpr int kUmmaPairsPerSlot = 96;
bool umma_grouped_supported(const edg_layer_desc& d);
cudaError_t launch_umma_gate_up(const GroupedParams& p, int max_tiles, cudaStream_t st);
cudaError_t launch_umma_down(const GroupedParams& p, int max_tiles, cudaStream_t st);

// streaming form for small and middling groups (edg_grouped_ffn.cu)
int32_t run_grouped_ffn(const edg_layer_desc* d, const GroupedParams& p, const WorkspaceLayout& W, uint8_t* ws, cudaStream_t st);
cudaError_t launch_sum_choices(const GroupedParams& p, cudaStream_t st);

// adapter projections for many tokens / pairs on the tensor cores (one shared adapter); false = shape not covered
bool launch_lora_ax_tokens(const edg_layer_desc* d, const void* x, const edg_lora* lora, float* u_gu, int T, cudaStream_t st);
bool launch_lora_adh_pairs(const edg_layer_desc* d, const edg_lora* lora, const float* h, float* u_d, int P, cudaStream_t st);

}  // namespace edg
