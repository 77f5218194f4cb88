// Interface of the one-launch decoder forward (forward.cu).
#pragma once

#include "tc_gemm.cuh"

namespace mtad {

constexpr int FW_SLOT = 32 * 1024;        // bytes of one ring slot: one step of a projection, or 128 keys of K or V
constexpr int FW_KEYS = 128;              // keys of an attention tile
constexpr int FW_MAX_ROWS = 60;           // rows of a call
constexpr int FW_MAX_QROWS = 16;          // query rows of one KV head and sequence

// Tile geometry of one projection.  A unit is what one box (two for gate / up) of the weight map brings: h feature rows
// (QKV: h rotary pairs of a head; gate / up: h gate rows and the h matching up rows), in `slots` rows of shared memory.
// h depends on the matrix and the SM count alone, so the weight maps are encoded once per model; how many units make a
// tile, how many k-blocks a step and whether the step's k-blocks lie side by side in the MMA's M dimension (S > 1)
// depends on the call's row count.
struct FwPhase {
    int h, slots, n_units, u;             // u: units per head (QKV)
    int upt, n_tiles, rows;               // units per tile, tiles, shared-memory rows of a tile's weights
    int S, kp, steps;                     // k-blocks side by side, k-blocks one after the other in a step, steps of a tile
    int a_bytes, b_off;                   // weights of one k-block, offset of the operand rows in the slot
    int box_bytes;                        // bytes that one unit brings per k-block
    int k_blocks;
};
enum { FW_QKV = 0, FW_ATTN = 1, FW_O = 2, FW_GATEUP = 3, FW_DOWN = 4, FW_LM = 5 };

struct alignas(64) FwLayer {              // device table, one entry per layer
    CUtensorMap wq, wk, wv, wo, gate, up, down;
    const __nv_bfloat16 *gain_ffn, *gain_next;
};

struct FwArgs {
    CUtensorMap xd, xa, xf, lm, kv;
    FwPhase ph[6];                        // by kind; the entry of the attention is unused
    const FwLayer* layers;
    int n_layers, n_cta, slots;           // slots: ring depth
    int T, terms, cols, B, R, d, F, V, Hq, Hkv, hd, max_batch, lm_plain;
    int pieces;                           // stride of the attention partials: pieces per (row, head)
    int parts0;                           // statistics of the prepared rows: parts of sumsq_a
    long long cap;
    float inv_dim, eps;
    int32_t *sync, *acnt;                 // phase counters, arrival counters of the attention's (sequence, KV head) pairs
    float *sumsq_a, *sumsq_b, *hidden;
    __nv_bfloat16 *x_d, *x_a, *x_f, *q_hi, *q_lo, *cache;
    const float* rope;
    RowMeta rm;
    float* part;
    const float* uniforms;
    float4* lm_part;
    float *logits, *node_z;
    uint32_t* status;
    unsigned int wait_limit;
    int debug_no_operands;
};

// Host side.  fw_geometry fills h, slots, n_units, u of every projection; fw_plan the rest for a call of B x R rows and
// returns false where the one-launch forward does not apply.  fw_parts_max: units of the LM head (lm) or of O / down,
// i.e. the most partial results that a row of a call has.
void fw_geometry(FwPhase ph[6], const mtad_model_desc& d, int n_cta);
bool fw_plan(FwArgs& a, const mtad_model_desc& d, int B, int R, int n_cta);
size_t fw_parts_max(const mtad_model_desc& d, int n_cta, bool lm);
// words of the phase and arrival counters (zeroed by the row preparation of every call)
inline size_t fw_sync_words(int layers, int max_batch, int Hkv) { return (size_t)5 * layers + 1 + (size_t)max_batch * Hkv; }
cudaError_t launch_forward(const FwArgs& a, cudaStream_t st);

}  // namespace mtad
