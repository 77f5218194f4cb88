// Interface of the one-launch decoder forward (forward.cu).
#pragma once

#include "tc_gemm.cuh"

namespace mtad {

constexpr int FW_RING = 192 * 1024;       // the copy ring: four slots, or three where the operand rows are many; a slot
                                          // holds one step of a projection, or 128 keys of K or V
constexpr int FW_KEYS = 128;              // keys of an attention tile
// Rows of a call.  Gate / up ends them: two boxes of 2 x 80 accumulator columns and the rows' sums put by between the parts
// of a tile's k-range (2 x 80 more) are 480 of the 512 columns of tensor memory.  Speed does not: eight layers of the 7B shape
// on 1024 keys, chain of launches -> one launch, 65 / 73 / 77 rows 1500 -> 1197, 1610 -> 1272, 1626 -> 1285 us, and in a trial
// without the sums put by (less exact than the chain) 101 rows 1997 -> 1444; 13B, 77 rows 1978 -> 1746.
constexpr int FW_MAX_ROWS = 80;
constexpr int FW_MAX_COLS = 160;          // operand rows (terms x rows) of a call
constexpr int FW_QROWS = 16;              // query rows of one KV head and sequence that an attention item takes at most,
constexpr int FW_QROWS_WIDE = 40;         // or in the wide variant: more are cut into blocks of equal size

// Tile geometry of one projection.  A step brings nbox boxes of hr weight rows x kb k-blocks (one copy each) and one box of
// operand rows.  nbox = 1: the rows of h features (QKV: of h rotary pairs of a head, hr = 2 h); nbox = 2: h gate rows and
// the h matching up rows, or 2 h rows of the LM head.  The geometry depends on the matrix, the SM count and the class of
// the call's operand rows, so that the weight maps are encoded once per model and class (seven sets, 49 maps and 6.3 KB a layer):
// kb is the most that a ring slot holds.
// Big boxes matter twice: a thread issues a copy about every quarter of a microsecond whatever its size, and rows of 256
// bytes and more pass at 70 GB/s per SM where rows of 128 bytes pass at 43.
// Three larger slots from 80 operand rows on, where a slot of a quarter of the ring holds one k-block only: 13B, 56 rows 8.64 ms
// with three, 8.75 with four; 7B, 33 rows 3.50 and 3.62.  At up to 64 four are as good (7B, 18 rows 3.98 and 3.96).
// Beyond 128 operand rows the split QKV's step, two boxes of 128 rows, does not fit a quarter of the ring at all.
constexpr int FW_CLASSES = 7;
struct FwClass { int cols, slots; };      // operand rows up to, ring slots
constexpr FwClass FW_CLASS[FW_CLASSES] = {{16, 4}, {32, 4}, {64, 4}, {80, 3}, {112, 3}, {144, 3}, {FW_MAX_COLS, 3}};
struct FwPhase {
    int h, hr, nbox, n_tiles, u;          // u: tiles per head (QKV)
    int c;                                // blocks that share a tile's k-range (their partial sums meet in global memory): O, down,
                                          // and QKV, where a tile then is two heads
    int kb, flat, S, steps;               // k-blocks of a box, its map's view, k-blocks side by side in the MMA, steps of all k-blocks
    int box_bytes, b_off;                 // bytes of one weight box, offset of the operand rows in the slot
    int k_blocks, K;
    int na, segs;                         // accumulators of a box, which take the MMAs along k in turn; parts of a tile's k-range
                                          // after which the accumulators are put by and begun afresh
    int both, stash, blk;                 // a tile takes both accumulator buffers; tensor-memory column where the parts are put
                                          // by; rows that the epilogue takes at a time
};
enum { FW_QKV = 0, FW_ATTN = 1, FW_O = 2, FW_GATEUP = 3, FW_DOWN = 4, FW_LM = 5 };

struct alignas(64) FwLayer {              // device table, one entry per layer
    CUtensorMap w[FW_CLASSES][7];         // wq, wk, wv, wo, gate, up, down
    const __nv_bfloat16 *gain_ffn, *gain_next;
};

struct FwArgs {
    CUtensorMap x[6], lm, kv;             // operand rows by kind
    int cls, slots;                       // class of the operand rows, ring slots
    FwPhase ph[6];                        // by kind; the entry of the attention is unused
    const FwLayer* layers;
    int n_layers, n_cta;
    int p_lo, p_hi;                       // phases of this launch: all, or one attention
    int T, terms, cols, B, R, d, F, V, Hq, Hkv, hd, max_batch, lm_plain;
    int nqb, qrows;                       // wide attention: blocks that a sequence's query rows of a KV head are cut into, rows of a block
    int pieces;                           // stride of the attention partials: pieces per (row, head)
    int parts0;                           // statistics of the prepared rows: parts of sumsq_a
    long long cap;
    float inv_dim, eps;
    int32_t *sync, *acnt;                 // phase counters, arrival counters of the attention's (sequence, KV head, query block)s
    int32_t* kcnt;                        // arrivals at the split tiles of O, of down, of QKV
    float* kpart;                         // their partial sums [block][row][feature]
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
    int debug_no_operands;                // test hook: 1 no operand rows, 2 no K and V tiles are copied, so the waits on them run out
};

// Host side.  fw_geometry fills the geometry of class cls; fw_plan the rest for a call of B x R rows and returns false
// where the one-launch forward does not apply.  fw_parts_max: most tiles of the LM head (lm) or of O / down, i.e. the
// partial results that a row of a call has.
void fw_geometry(FwPhase ph[6], const mtad_model_desc& d, int n_cta, int cls);
bool fw_plan(FwArgs& a, const mtad_model_desc& d, int B, int R, int n_cta);
// The attention alone, wide variant, for a call whose projections run as launches of their own; run for one layer with
// launch_forward_attention.
bool fw_attn_plan(FwArgs& a, const mtad_model_desc& d, int B, int R, int n_cta);
// Whether the one-launch forward of a call of B x R rows, of up to `total` keys a sequence, is the faster one; the same of the
// wide attention as a launch of its own.
bool fw_pays(const mtad_model_desc& d, int B, int R, long long total);
bool fw_attn_pays(const mtad_model_desc& d, int B, int R, long long total);
size_t fw_parts_max(const mtad_model_desc& d, int n_cta, bool lm);
// (sequence, KV head, query block)s of a call at most: B * ceil(G R / rows) with B R <= TC_MAX_ROWS
inline size_t fw_pairs(const mtad_model_desc& d, int max_batch) {
    const int G = d.n_q_heads / d.n_kv_heads;
    return (size_t)d.n_kv_heads * ((G * TC_MAX_ROWS + FW_QROWS_WIDE - 1) / FW_QROWS_WIDE + max_batch);
}
// words of the phase and arrival counters (zeroed by the row preparation of every call)
inline size_t fw_sync_words(const mtad_model_desc& d, int max_batch, int n_cta) {
    return (size_t)5 * d.layers + 1 + fw_pairs(d, max_batch) + 3 * (size_t)n_cta;
}
// partial sums of the split projections of calls of up to max_batch x max_rows rows
size_t fw_part_floats(const mtad_model_desc& d, int n_cta, int max_batch, int max_rows);
// Its blocks wait on one another: whether the current device holds n_cta of them at once.  A launch that does not fit returns
// cudaErrorCooperativeLaunchTooLarge and does nothing (`refuse`, for tests: ask for more blocks than any device holds).
bool forward_fits(int n_cta);
cudaError_t launch_forward(const FwArgs& a, cudaStream_t st, bool refuse = false);
cudaError_t launch_forward_attention(FwArgs& a, int layer, cudaStream_t st, bool refuse = false);

}  // namespace mtad
