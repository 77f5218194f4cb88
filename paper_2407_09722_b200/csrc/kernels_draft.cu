// Beam-sampling draft with the auxiliary model (Sec. 2.1 of the paper, the p_beam equation; every intermediate
// beam becomes a node of the candidate tree, Sec. 3.3): row bookkeeping of each draft step, the Gumbel-top-b
// selection over (beam, token) pairs, and the roll-forward of the auxiliary KV cache after a verification.
//
// Virtual rows of one draft: the P pending tokens (not yet in the auxiliary cache, the last one is the root) are
// rows 0 .. P-1, node n is row P + n; row v lives in cache slot aux_len + v.
#include <math_constants.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace mtad {

namespace {

__device__ __forceinline__ float wsum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

struct Cand {
    float y;      // perturbed joint score
    int flat;     // beam * V + token
};
__device__ __forceinline__ bool before(const Cand& a, const Cand& b) {     // a ranks ahead of b
    return a.y > b.y || (a.y == b.y && a.flat < b.flat);
}

// The best candidate of a block of 256 threads, returned to every thread: butterfly inside each warp, then the eight
// warp winners through shared memory (two barriers a call; s_w is free again on return).
__device__ __forceinline__ Cand block_best(Cand c, Cand* s_w, int tid) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const Cand c2{__shfl_xor_sync(0xffffffffu, c.y, o), __shfl_xor_sync(0xffffffffu, c.flat, o)};
        if (before(c2, c)) c = c2;
    }
    if ((tid & 31) == 0) s_w[tid >> 5] = c;
    __syncthreads();
    Cand best = s_w[0];
#pragma unroll
    for (int w = 1; w < 8; ++w)
        if (before(s_w[w], best)) best = s_w[w];
    __syncthreads();
    return best;
}

}  // namespace

// ---------------------------------------------------------------------------------------------------------------
// rows of one draft step: step 0 runs the pending tokens as a causal chain, step s >= 1 the nodes of layer s
// ---------------------------------------------------------------------------------------------------------------

// What the rows of a draft step are made from and where they go.
struct DraftRows {
    const __nv_bfloat16* embed;
    int d, vocab, hd;
    RopeInv rinv;
    long long cap;
    SeqState s;
    RowMeta rm;
    float *hidden, *rope;
    const __nv_bfloat16* gain0;
    __nv_bfloat16* x;           // operand rows of the tensor-core path, or null
    int terms;
    float* sumsq;
    int32_t* sync;              // the one-launch forward's counters
    int sync_words;
    int32_t* arrive;
};
static DraftRows draft_rows(const ModelView& m, const SeqState& s, const RowMeta& rm, const Scratch& sc, int T, bool tc) {
    return DraftRows{static_cast<const __nv_bfloat16*>(m.d.embed), m.d.d_model, m.d.vocab, m.d.head_dim,
                     rope_inv((double)m.d.rope_base, m.d.head_dim), (long long)m.d.kv_capacity, s, rm, sc.hidden, sc.rope,
                     tc ? m.w(0, 0) : (const __nv_bfloat16*)nullptr, tc ? sc.xd : (__nv_bfloat16*)nullptr, tc_terms(T), sc.sumsq_a,
                     sc.fw_sync, sc.fw_sync_words, sc.arrive};
}

struct RowInfo {
    int tok, pos;
    bool ok;
    int hole;                   // a cache row to clear, or -1
};
// Row r of sequence bi in a step goes to the call's row data.  nbp: beams kept by the step before.
__device__ __forceinline__ RowInfo write_row(const DraftRows& a, int bi, int seq, int R, int r, int step, int beam, int L, int P, int tok,
                                             int pos, int vrow, bool active, int hole, const uint32_t* mask, int nbp) {
    const RowMeta& rm = a.rm;
    const int t = bi * R + r;
    if (tok < 0 || tok >= a.vocab) tok = 0;
    rm.tok[t] = tok;
    rm.depth[t] = step;
    rm.pos[t] = pos;
    if (L < 0 || P < 1 || P > MTAD_MAX_DEPTH + 1 || (long long)L + vrow >= a.cap) active = false;
    rm.slot[t] = active ? L + vrow : -1;
    rm.seq[t] = seq;
    rm.prow[t] = -1;
    // the mask is indexed by cache slot minus L: virtual rows
#pragma unroll
    for (int i = 0; i < MTAD_MASK_WORDS; ++i) rm.mask[(size_t)t * MTAD_MASK_WORDS + i] = mask[i];
    if (r == 0) {
        const bool state_ok = L >= 0 && P >= 1 && P <= MTAD_MAX_DEPTH + 1 && P <= (step == 0 ? R : MTAD_MAX_DEPTH + 1) &&
                              (long long)L + P + (long long)step * beam <= a.cap;
        rm.n_rows[bi] = !state_ok ? 0 : (step == 0 ? P : nbp);
        rm.n_spec[bi] = !state_ok ? 0 : (step == 0 ? P : P + step * beam);
        rm.kv_base[bi] = L;
        rm.call_seq[bi] = seq;
    }
    return RowInfo{tok, pos, active, (hole >= 0 && L >= 0 && (long long)hole < a.cap) ? hole : -1};
}

// Its token, position, slot and mask from the state.
__device__ __forceinline__ RowInfo draft_row(const DraftRows& a, const DraftState& ds, int bi, int seq, int R, int r, int step, int beam,
                                             bool holes) {
    const SeqState& s = a.s;
    const int L = step == 0 ? s.aux_len[seq] : ds.base_len[seq];
    const int P = step == 0 ? s.aux_npend[seq] : ds.npend[seq];
    if (step == 0 && r == 0) { ds.base_len[seq] = L; ds.npend[seq] = P; ds.status[bi] = 0; a.arrive[bi] = 0; }
    uint32_t mask[MTAD_MASK_WORDS];
#pragma unroll
    for (int i = 0; i < MTAD_MASK_WORDS; ++i) mask[i] = 0;
    int tok = 0, pos = L, vrow = 0, hole = -1;
    bool active;
    if (step == 0) {
        active = r < P;
        if (active) {
            tok = s.aux_pend[seq * (MTAD_MAX_DEPTH + 1) + r];
            vrow = r;
            pos = L + r;
            for (int i = 0; i <= r; ++i) mask[i >> 5] |= 1u << (i & 31);        // causal over the pending rows
        }
    } else {
        // the beams the step before kept: the beam width, or fewer on warped rows
        const int nbp = min(max(ds.nb[seq * MTAD_MAX_DEPTH + step - 1], 0), beam);
        active = r < nbp;
        // A beam slot of the layer before that no beam took is a cache row nobody wrote.  This step's rows never
        // look at it (their masks name ancestors only), but a masked key still meets its value row with weight 0, and
        // 0 x (whatever the memory held) must stay 0: the row is cleared (holes: only then can slots be empty).
        hole = (holes && !active && r < beam) ? L + P + (step - 1) * beam + r : -1;
        if (active) {
            const int n = (step - 1) * beam + r;
            tok = ds.node_tok[seq * MTAD_DRAFT_NODES + n];
            vrow = P + n;
            pos = L + P - 1 + step;
#pragma unroll
            for (int i = 0; i < MTAD_MASK_WORDS; ++i)
                mask[i] = ds.node_mask[((size_t)seq * MTAD_DRAFT_NODES + n) * MTAD_MASK_WORDS + i];
        }
    }
    const int nbp = step == 0 ? 0 : min(max(ds.nb[seq * MTAD_MAX_DEPTH + step - 1], 0), beam);
    return write_row(a, bi, seq, R, r, step, beam, L, P, tok, pos, vrow, active, hole, mask, nbp);
}

__global__ void draft_prepare_kernel(DraftRows a, DraftState ds, SeqList seqs, int R, int step, int beam,
                                     __nv_bfloat16* __restrict__ cache, int layers, int max_batch, int Hkv) {
    const int t = blockIdx.x, bi = t / R, r = t % R;
    const int seq = seqs.v[bi];
    __shared__ RowInfo row;
    pdl_wait();               // the sequence and draft state, and every buffer written here, belong to earlier kernels
    pdl_trigger();
    for (int i = t * blockDim.x + threadIdx.x; i < a.sync_words; i += gridDim.x * blockDim.x) a.sync[i] = 0;
    if (threadIdx.x == 0) row = draft_row(a, ds, bi, seq, R, r, step, beam, cache != nullptr);
    __syncthreads();
    const int d = a.d, hd = a.hd;
    if (row.hole >= 0) {
        for (int i = threadIdx.x; i < layers * 2 * Hkv * hd; i += blockDim.x) {
            const int j = i % hd, head = (i / hd) % Hkv, kv = (i / (hd * Hkv)) & 1, layer = i / (2 * hd * Hkv);
            cache[idx_cache(layer, max_batch, seq, kv, Hkv, head, a.cap, row.hole, hd) + j] = __float2bfloat16_rn(0.f);
        }
    }
    float share[1];
    embed_row(a.embed + (size_t)row.tok * d, row.ok, d, a.hidden + (size_t)t * d, a.gain0, a.x ? a.x + (size_t)t * a.terms * d : nullptr,
              a.terms, threadIdx.x, blockDim.x, share);
    if (a.x) {
        __shared__ float red[32];
        const float ss = wsum(share[0]);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
        __syncthreads();
        if (threadIdx.x == 0) {
            float v = 0.f;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w];
            a.sumsq[t] = v;
        }
    }
    for (int i = threadIdx.x; i < hd / 2; i += blockDim.x) {
        float cs, sn;
        rope_cs((double)row.pos, a.rinv.v[i], cs, sn);
        a.rope[((size_t)t * (hd / 2) + i) * 2 + 0] = cs;
        a.rope[((size_t)t * (hd / 2) + i) * 2 + 1] = sn;
    }
}

cudaError_t launch_draft_prepare(const ModelView& m, const SeqState& s, const DraftState& ds, const RowMeta& rm,
                                 const Scratch& sc, const SeqList& seqs, int B, int R, int step, int beam, bool tc,
                                 bool warped, bool pdl, cudaStream_t st) {
    return launch_pdl(draft_prepare_kernel, dim3(B * R), dim3(128), 0, st, pdl, draft_rows(m, s, rm, sc, B * R, tc), ds, seqs, R,
                      step, beam, warped ? static_cast<__nv_bfloat16*>(m.d.kv_cache) : (__nv_bfloat16*)nullptr, m.d.layers,
                      m.max_batch, m.d.n_kv_heads);
}

// ---------------------------------------------------------------------------------------------------------------
// selection: the `beam` largest of log q(beam) + log q(token | beam) + Gumbel noise over all (beam, token) pairs
//
// One launch, a block per (chunk of the vocabulary, beam row, sequence).  First (draft_scan) the chunk's share of
// the row's log-sum-exp (running maximum and sum) and its `beam` largest perturbed logits t = z - log(-log u).  The
// joint score of a pair is t + (log q(beam) - lse(row)), a per-row constant added in fp32 (monotone), so a pair
// among the overall `beam` largest is among the `beam` largest of its chunk.  Then the block of a sequence that finishes last
// (draft_pick) merges the chunks of every row in chunk order, scores the surviving pairs and takes the `beam` largest
// (ties to the lower flat index beam * V + token), writes the new layer of the tree, and of a narrow model (draft_rows_ahead)
// makes the next step's rows from it.  As three launches - scan, pick, rows - a step of the 7B pair spent 21 us between two forwards.
// ---------------------------------------------------------------------------------------------------------------

__device__ __forceinline__ Cand warp_best(Cand c) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const Cand c2{__shfl_xor_sync(0xffffffffu, c.y, o), __shfl_xor_sync(0xffffffffu, c.flat, o)};
        if (before(c2, c)) c = c2;
    }
    return c;
}
// The k best of up to 32 lists, each sorted, by a warp: lane i walks list i (n_i entries `stride` apart).  Entry r of the result
// goes to (y, flat)[r]; past the end flat is 0x7fffffff.
__device__ __forceinline__ void merge_lists(const float* ly, const int* lf, int n, int stride, int k, float* y, int* flat, int lane) {
    int at = 0;
    Cand c{-CUDART_INF_F, 0x7fffffff};
    if (at < n) c = Cand{ly[0], lf[0]};
    for (int r = 0; r < k; ++r) {
        const Cand win = warp_best(c);
        if (lane == 0) { y[r] = win.y; flat[r] = win.flat; }
        if (c.flat == win.flat && win.flat != 0x7fffffff) {              // (flat indices are unique)
            ++at;
            c = at < n ? Cand{ly[at * stride], lf[at * stride]} : Cand{-CUDART_INF_F, 0x7fffffff};
        }
    }
}

struct ScanShared {
    float m[8], s[8];
    float y[8][MTAD_MAX_CAND];
    int v[8][MTAD_MAX_CAND];
};
// kpb: perturbed logits of this chunk to hand on (the beam width, or with all candidates kept the candidates
// recorded per beam: beam * beam of the single beam of step 0, beam afterwards).  Every warp finds its own kpb best by shuffles, then
// the first warp merges the eight lists.  (Rounds of the whole block, two barriers each, over sorted lists that every thread kept by
// insertion: the selection of eight sequences took 40 us between two forwards.)
__device__ __forceinline__ void draft_scan(const float* __restrict__ logits, int V, int R, int step, int gamma, int beam, int kpb,
                                           const float* __restrict__ uni, int P, DraftPart* __restrict__ part, int nch, ScanShared& sh) {
    const int c = blockIdx.x, j = blockIdx.y, bi = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row = step == 0 ? P - 1 : j;
    const float* z = logits + (size_t)(bi * R + row) * V;
    const float* ub = uni + (((size_t)bi * gamma + step) * beam + j) * V;
    const int len = (V + nch - 1) / nch, v0 = c * len, v1 = min(V, v0 + len);
    // A list of NL tokens a thread.  A longer chunk (vocabulary above 65536) takes more passes, in which the warp's kpb best so far
    // take the lists' first places.
    constexpr int NL = MTAD_MAX_BEAM, HELD = MTAD_MAX_CAND / 32;
    static_assert(HELD < NL, "room for tokens beside the best so far");
    float m = -CUDART_INF_F, sum = 0.f;
    auto pass = [&](int at, auto held_places) {
        constexpr int held = decltype(held_places)::value;
        // all of a thread's tokens at once
        float zv[NL], uv[NL];
        Cand loc[NL];
#pragma unroll
        for (int k = held; k < NL; ++k) {
            const int v = at + tid + 256 * (k - held);
            zv[k] = v < v1 ? z[v] : -CUDART_INF_F;
            uv[k] = v < v1 ? ub[v] : 0.5f;
        }
        const float before_max = m;
#pragma unroll
        for (int k = held; k < NL; ++k) m = fmaxf(m, zv[k]);
        if (held && m != before_max) sum = before_max == -CUDART_INF_F ? 0.f : sum * expf(before_max - m);
#pragma unroll
        for (int k = held; k < NL; ++k) {
            const int v = at + tid + 256 * (k - held);
            loc[k] = Cand{-CUDART_INF_F, 0x7fffffff};
            if (256 * k < len && v < v1) {
                sum += m == -CUDART_INF_F ? 0.f : (zv[k] == m ? 1.f : expf(zv[k] - m));
                const float y = zv[k] - logf(-logf(uv[k]));
                if (y == y) loc[k] = Cand{y, v};             // (NaN is no candidate)
            }
        }
#pragma unroll
        for (int k = 0; k < held; ++k) {
            const int r = lane + 32 * k;
            loc[k] = r < kpb ? Cand{sh.y[warp][r], sh.v[warp][r]} : Cand{-CUDART_INF_F, 0x7fffffff};
        }
        __syncwarp();
        // the warp's kpb best
        Cand top = loc[0];
#pragma unroll
        for (int q = 1; q < NL; ++q)
            if (before(loc[q], top)) top = loc[q];
        for (int k = 0; k < kpb; ++k) {
            const Cand win = warp_best(top);
            if (lane == 0) { sh.y[warp][k] = win.y; sh.v[warp][k] = win.flat; }
            if (top.flat == win.flat && win.flat != 0x7fffffff) {        // the owner takes it off its list (tokens are unique)
                top = Cand{-CUDART_INF_F, 0x7fffffff};
#pragma unroll
                for (int q = 0; q < NL; ++q) {
                    if (loc[q].flat == win.flat) loc[q] = Cand{-CUDART_INF_F, 0x7fffffff};
                    if (before(loc[q], top)) top = loc[q];
                }
            }
        }
        __syncwarp();
    };
    pass(v0, std::integral_constant<int, 0>{});
#pragma unroll 1
    for (int at = v0 + 256 * NL; at < v1; at += 256 * (NL - HELD)) pass(at, std::integral_constant<int, HELD>{});
    // the chunk's maximum and sum of exponentials (fixed combination order: butterfly, then warps in order)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, o), s2 = __shfl_xor_sync(0xffffffffu, sum, o);
        const float M = fmaxf(m, m2);
        sum = (M == -CUDART_INF_F) ? 0.f : sum * expf(m - M) + s2 * expf(m2 - M);
        m = M;
    }
    if (lane == 0) { sh.m[warp] = m; sh.s[warp] = sum; }
    __syncthreads();
    if (warp) return;
    DraftPart* dst = part + ((size_t)(bi * MTAD_MAX_BEAM + j)) * nch + c;
    merge_lists(sh.y[lane & 7], sh.v[lane & 7], lane < 8 ? kpb : 0, 1, kpb, dst->t, dst->v, lane);
    if (lane == 0) {
        float M = -CUDART_INF_F;
        for (int w = 0; w < 8; ++w) M = fmaxf(M, sh.m[w]);
        float a = 0.f;
        for (int w = 0; w < 8; ++w) a += (sh.m[w] == -CUDART_INF_F) ? 0.f : sh.s[w] * expf(sh.m[w] - M);
        dst->m = M;
        dst->s = a;
    }
}

struct PickShared {
    float y[MTAD_MAX_BEAM * MTAD_DRAFT_CHUNKS * MTAD_MAX_BEAM];    // the chunks' lists, [beam][chunk][kpb]
    int flat[MTAD_MAX_BEAM * MTAD_DRAFT_CHUNKS * MTAD_MAX_BEAM];
    float lse[MTAD_MAX_BEAM], lq[MTAD_MAX_BEAM];
    int slot[MTAD_MAX_BEAM], tree[MTAD_MAX_BEAM];                  // the current beams: beam slot and tree id (-1: the context)
    uint32_t mask[MTAD_MAX_BEAM][MTAD_MASK_WORDS];
    float by[MTAD_MAX_CAND], bz[MTAD_MAX_CAND];                    // every beam's kpb best pairs: perturbed score, log-likelihood,
    int bflat[MTAD_MAX_CAND];                                      // flat pair
    float ky[MTAD_MAX_BEAM];                                       // the beams kept for the next step
    int kflat[MTAD_MAX_BEAM];
    int ktok[MTAD_MAX_BEAM];
    uint32_t kmask[MTAD_MAX_BEAM][MTAD_MASK_WORDS];
};
// (L2 loads of the parts: other blocks of this launch wrote them)
__device__ __forceinline__ void draft_pick(const float* __restrict__ logits, int V, int R, int step, int gamma, int beam,
                                           int keep_all, int kpb, const DraftState& ds, int bi, int seq, int P, const DraftPart* part,
                                           int nch, const DraftOut& out, PickShared& sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_beams = step == 0 ? 1 : beam;
    const int per_layer = keep_all ? beam * beam : beam;          // nodes of a layer of the caller's tree
    const int N = gamma * per_layer;
    const DraftPart* pp = part + (size_t)bi * MTAD_MAX_BEAM * nch;
    static_assert(MTAD_DRAFT_CHUNKS <= 32 && MTAD_MAX_BEAM <= 8, "a lane per chunk, a warp per beam");
    // a warp per beam row: log-sum-exp (a lane per chunk, combined in a fixed order), scores of the chunks' candidates, their kpb best
    if (warp < n_beams) {
        const int j = warp, slot = step == 0 ? -1 : (step - 1) * beam + j;
        const DraftPart* pj = pp + (size_t)j * nch;
        const float mc = lane < nch ? __ldcg(&pj[lane].m) : -CUDART_INF_F, sc = lane < nch ? __ldcg(&pj[lane].s) : 0.f;
        const int tree = slot < 0 ? -1 : ds.tree_id[seq * MTAD_DRAFT_NODES + slot];
        const float lq = slot < 0 ? 0.f : ds.node_logq[seq * MTAD_DRAFT_NODES + slot];
        if (slot >= 0 && lane < MTAD_MASK_WORDS)
            sh.mask[j][lane] = ds.node_mask[((size_t)seq * MTAD_DRAFT_NODES + slot) * MTAD_MASK_WORDS + lane];
        float* ly = sh.y + (j * nch) * kpb;
        int* lf = sh.flat + (j * nch) * kpb;
        for (int i = lane; i < nch * kpb; i += 32) {
            const int c = i / kpb, k = i - c * kpb, v = __ldcg(&pj[c].v[k]);
            ly[i] = __ldcg(&pj[c].t[k]);
            lf[i] = v == 0x7fffffff ? v : j * V + v;
        }
        float M = mc;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        float a = mc == -CUDART_INF_F ? 0.f : sc * expf(mc - M);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        const float lse = M + logf(a);
        if (lane == 0) { sh.lse[j] = lse; sh.slot[j] = slot; sh.tree[j] = tree; sh.lq[j] = lq; }
        __syncwarp();
        // lane c scores its chunk's list; the constant may make equals of what it rounds: those go by flat index
        if (lane < nch) {
            float* y = ly + lane * kpb;
            int* f = lf + lane * kpb;
            const float off = lq - lse;
            for (int k = 0; k < kpb; ++k) {
                Cand cd{y[k] + off, f[k]};
                if (f[k] == 0x7fffffff || cd.y != cd.y) cd = Cand{-CUDART_INF_F, 0x7fffffff};
                int at = k;
                for (; at > 0 && before(cd, Cand{y[at - 1], f[at - 1]}); --at) { y[at] = y[at - 1]; f[at] = f[at - 1]; }
                y[at] = cd.y;
                f[at] = cd.flat;
            }
        }
        __syncwarp();
        merge_lists(ly + lane * kpb, lf + lane * kpb, lane < nch ? kpb : 0, 1, kpb, sh.by + j * kpb, sh.bflat + j * kpb, lane);
        __syncwarp();
        const int row = step == 0 ? P - 1 : j;
        for (int k = lane; k < kpb; k += 32) {
            const int f = sh.bflat[j * kpb + k];
            sh.bz[j * kpb + k] = lq + logits[(size_t)(bi * R + row) * V + (f == 0x7fffffff ? 0 : f - j * V)] - lse;
        }
    }
    __syncthreads();
    // The beams kept for the next step: the best pairs of all, in order (the plain tree's layer is those).
    if (warp == 0)
        merge_lists(sh.by + lane * kpb, sh.bflat + lane * kpb, lane < n_beams ? kpb : 0, 1, beam, sh.ky, sh.kflat, lane);
    __syncthreads();
    // every node of the layer, one thread each: the caller's tree, and for a kept node the beam state of the next step
    for (int m = tid; m < per_layer; m += 256) {
        const int f = keep_all ? sh.bflat[m] : sh.kflat[m];
        const bool valid = f != 0x7fffffff;                // a vocabulary of at least per_layer tokens always fills the layer
        const int j = valid ? f / V : 0, v = valid ? f % V : 0;
        const int n = step * per_layer + m;
        int k = keep_all ? -1 : m, b = keep_all ? m : -1;  // its rank among the kept beams, its place among the beams' best
        if (keep_all) {
            // Fewer pairs than beams (scores of NaN): the ranks that no pair took go to the first nodes without one, so that every
            // beam of the next step has a token and a mask, as in the plain tree.
            int free = 0;
            if (!valid)
                for (int q = 0; q < m; ++q) free += sh.bflat[q] == 0x7fffffff;
            for (int q = 0; q < beam; ++q)
                if (sh.kflat[q] == f && (valid || free-- == 0)) k = q;
        } else {
            for (int q = 0; q < kpb; ++q)
                if (sh.bflat[j * kpb + q] == f) b = j * kpb + q;
        }
        const float lq = sh.bz[max(b, 0)];
        out.tok[bi * N + n] = v;
        out.parent[bi * N + n] = sh.tree[j];
        out.depth[bi * N + n] = step + 1;
        out.node_logq[bi * N + n] = lq;
        if (n < MTAD_DRAFT_NODES) ds.tree2slot[seq * MTAD_DRAFT_NODES + n] = k >= 0 ? step * beam + k : -1;
        if (k >= 0) {
            const int slot = step * beam + k, parent = sh.slot[j];
            sh.ktok[k] = v;
            ds.node_tok[seq * MTAD_DRAFT_NODES + slot] = v;
            ds.node_parent[seq * MTAD_DRAFT_NODES + slot] = parent;
            ds.node_logq[seq * MTAD_DRAFT_NODES + slot] = lq;
            ds.tree_id[seq * MTAD_DRAFT_NODES + slot] = n;
            uint32_t* mk = ds.node_mask + ((size_t)seq * MTAD_DRAFT_NODES + slot) * MTAD_MASK_WORDS;
#pragma unroll
            for (int i = 0; i < MTAD_MASK_WORDS; ++i) {
                uint32_t w;
                if (parent >= 0) w = sh.mask[j][i];
                else {                                        // child of the root: sees all pending rows
                    const int lo = i * 32;
                    w = P >= lo + 32 ? 0xffffffffu : (P > lo ? (1u << (P - lo)) - 1u : 0u);
                }
                if (((P + slot) >> 5) == i) w |= 1u << ((P + slot) & 31);
                mk[i] = w;
                sh.kmask[k][i] = w;
            }
        }
    }
    __syncthreads();
    if (tid == 0) ds.nb[seq * MTAD_MAX_DEPTH + step] = beam;      // every beam slot of the layer is taken
    if (step == gamma - 1 && tid == 0) {
        // x**: the final beam with the highest draft likelihood (lowest tree id on ties), and its prefix likelihoods
        __threadfence_block();
        int best = (gamma - 1) * beam;
        for (int k = 1; k < beam; ++k) {
            const int sl = (gamma - 1) * beam + k;
            const float a = ds.node_logq[seq * MTAD_DRAFT_NODES + sl], b0 = ds.node_logq[seq * MTAD_DRAFT_NODES + best];
            if (a > b0 || (a == b0 && ds.tree_id[seq * MTAD_DRAFT_NODES + sl] < ds.tree_id[seq * MTAD_DRAFT_NODES + best]))
                best = sl;
        }
        int cur = best;
        for (int i = gamma - 1; i >= 0 && cur >= 0; --i) {
            out.best_path[bi * gamma + i] = ds.tree_id[seq * MTAD_DRAFT_NODES + cur];
            out.logq_ref[bi * gamma + i] = ds.node_logq[seq * MTAD_DRAFT_NODES + cur];
            ds.best_path[seq * MTAD_MAX_DEPTH + i] = cur;
            cur = ds.node_parent[seq * MTAD_DRAFT_NODES + cur];
        }
        ds.gamma[seq] = gamma;
        ds.beam[seq] = beam;
        if (out.n_nodes) out.n_nodes[bi] = N;
    }
}

__global__ void __launch_bounds__(256, 4) draft_select_kernel(const float* __restrict__ logits, int V, int R, int step, int gamma,
                                                           int beam, int keep_all, int kpb, const float* __restrict__ uni,
                                                           DraftState ds, SeqList seqs, DraftPart* part, int nch, DraftOut out,
                                                           DraftRows rows, bool next) {
    const int bi = blockIdx.z, seq = seqs.v[bi], tid = threadIdx.x;
    __shared__ union { ScanShared scan; PickShared pick; } sh;
    __shared__ bool last;
    pdl_wait();               // the logits come from the kernel before
    pdl_trigger();
    if (next)                 // (the forward that used the counters has ended)
        for (int i = ((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * 256 + tid; i < rows.sync_words;
             i += gridDim.x * gridDim.y * gridDim.z * 256)
            rows.sync[i] = 0;
    const int L = ds.base_len[seq], npend = ds.npend[seq];
    const int P = min(max(npend, 1), step == 0 ? R : MTAD_MAX_DEPTH + 1);          // in range whatever the state holds
    draft_scan(logits, V, R, step, gamma, beam, kpb, uni, P, part, nch, sh.scan);
    if (tid == 0) {           // (the thread that wrote the block's part)
        __threadfence();
        last = atomicAdd(rows.arrive + bi, 1) == (int)(gridDim.x * gridDim.y) - 1;
        if (last) rows.arrive[bi] = 0;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    draft_pick(logits, V, R, step, gamma, beam, keep_all, kpb, ds, bi, seq, P, part, nch, out, sh.pick);
    if (!next) return;
    // the next step's rows, a warp per row
    const int lane = tid & 31, warp = tid >> 5, hd = rows.hd, d = rows.d;
    __shared__ RowInfo row[MTAD_MAX_BEAM];
    if (warp < beam) {
        if (lane == 0)
            row[warp] = write_row(rows, bi, seq, beam, warp, step + 1, beam, L, npend, sh.pick.ktok[warp], L + npend + step,
                                  npend + step * beam + warp, true, -1, sh.pick.kmask[warp], beam);
        __syncwarp();
        const int t = bi * beam + warp;
        float share[4], ss = 0.f;
        embed_row(rows.embed + (size_t)row[warp].tok * d, row[warp].ok, d, rows.hidden + (size_t)t * d, rows.gain0,
                  rows.x ? rows.x + (size_t)t * rows.terms * d : nullptr, rows.terms, lane, 32, share);
#pragma unroll
        for (int k = 0; k < 4; ++k) ss += wsum(share[k]);
        if (rows.x && lane == 0) rows.sumsq[t] = ss;
    }
    __syncthreads();
    for (int i = tid; i < beam * (hd / 2); i += 256) {
        const int r = i / (hd / 2), j = i - r * (hd / 2);
        float cs, sn;
        rope_cs((double)row[r].pos, rows.rinv.v[j], cs, sn);
        reinterpret_cast<float2*>(rows.rope)[(size_t)bi * beam * (hd / 2) + i] = make_float2(cs, sn);
    }
}

// ---------------------------------------------------------------------------------------------------------------
// selection on warped rows (App. F): every beam row has been cut to its kept tokens (warp_scan / warp_merge: at most
// MTAD_MAX_TOPK tokens with renormalised log-probabilities), so the candidates of a step are the at most
// beam * MTAD_MAX_TOPK (beam, kept token) pairs and one block per sequence ranks them all.  A step may find fewer
// pairs than beams: it keeps what there is, the layer holds fewer nodes, node ids stay consecutive.
// ---------------------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) draft_pick_warped_kernel(const WarpRow* __restrict__ rows, int V, int R, int step,
                                                                int gamma, int beam, int keep_all,
                                                                const float* __restrict__ uni, DraftState ds,
                                                                SeqList seqs, DraftOut out) {
    const int bi = blockIdx.x, seq = seqs.v[bi];
    const int tid = threadIdx.x;
    const int P = min(max(ds.npend[seq], 1), step == 0 ? R : MTAD_MAX_DEPTH + 1);
    const int n_beams = step == 0 ? 1 : min(max(ds.nb[seq * MTAD_MAX_DEPTH + step - 1], 0), beam);
    const int kpb = (keep_all && step == 0) ? beam * beam : beam;       // nodes a beam may contribute with all kept
    const int N = gamma * (keep_all ? beam * beam : beam);              // capacity of the caller's arrays
    constexpr int NC = MTAD_MAX_BEAM * MTAD_MAX_TOPK;
    __shared__ float s_lq[MTAD_MAX_BEAM];
    __shared__ int s_slot[MTAD_MAX_BEAM], s_tree[MTAD_MAX_BEAM];
    __shared__ float s_y[NC], s_lp[NC];
    __shared__ int s_flat[NC];
    __shared__ Cand s_w[8];
    __shared__ float l_y[MTAD_MAX_CAND], l_lp[MTAD_MAX_CAND];
    __shared__ int l_flat[MTAD_MAX_CAND], l_rank[MTAD_MAX_CAND], l_id[MTAD_MAX_CAND];
    __shared__ int s_count[2];                       // nodes of the layer, beams kept
    if (tid < n_beams) {
        const int slot = step == 0 ? -1 : (step - 1) * beam + tid;
        s_slot[tid] = slot;
        s_tree[tid] = slot < 0 ? -1 : ds.tree_id[seq * MTAD_DRAFT_NODES + slot];
        s_lq[tid] = slot < 0 ? 0.f : ds.node_logq[seq * MTAD_DRAFT_NODES + slot];
    }
    __syncthreads();
    if (tid < NC) {
        const int j = tid / MTAD_MAX_TOPK, i = tid % MTAD_MAX_TOPK;
        bool ok = j < n_beams;
        float y = -CUDART_INF_F, lp = 0.f;
        int flat = 0x7fffffff;
        if (ok) {
            const WarpRow& row = rows[bi * R + (step == 0 ? P - 1 : j)];
            ok = i < min(row.n, MTAD_MAX_TOPK);
            if (ok) {
                const int v = row.idx[i];
                ok = v >= 0 && v < V;
                if (ok) {
                    lp = row.lp[i];
                    y = (s_lq[j] + lp) - logf(-logf(uni[(((size_t)bi * gamma + step) * beam + j) * V + v]));
                    flat = j * V + v;
                }
            }
        }
        s_y[tid] = y; s_lp[tid] = lp; s_flat[tid] = flat;
    }
    __syncthreads();
    // the layer's nodes: the `beam` best pairs of all, or with every candidate kept each beam's kpb best, best first
    const int n_groups = keep_all ? n_beams : 1, rounds = keep_all ? min(kpb, MTAD_MAX_TOPK) : beam;
    for (int gidx = 0; gidx < n_groups; ++gidx) {
        const int lo = keep_all ? gidx * MTAD_MAX_TOPK : 0, hi = keep_all ? lo + MTAD_MAX_TOPK : NC;
        for (int k = 0; k < rounds; ++k) {
            Cand best{-CUDART_INF_F, 0x7fffffff};
            const int i = lo + tid;
            if (i < hi && s_flat[i] != 0x7fffffff) best = Cand{s_y[i], s_flat[i]};
            const Cand win = block_best(best, s_w, tid);
            const bool found = win.flat != 0x7fffffff;
            if (tid == 0) {
                const int m = gidx * rounds + k;
                if (m < MTAD_MAX_CAND) { l_y[m] = found ? win.y : -CUDART_INF_F; l_flat[m] = win.flat; l_rank[m] = -1; }
            }
            if (found && best.flat == win.flat) {                     // the owner (pairs are unique) strikes the winner out
                const int m = gidx * rounds + k;
                if (m < MTAD_MAX_CAND) l_lp[m] = s_lp[i];
                s_flat[i] = 0x7fffffff;
            }
            __syncthreads();
        }
    }
    const int per_layer = min(n_groups * rounds, MTAD_MAX_CAND);
    if (tid == 0) {
        // consecutive node ids for the pairs that exist; the beams kept: the `beam` best of them
        const int base_id = step == 0 ? 0 : max(ds.n_tree[seq], 0);
        int cnt = 0;
        for (int m = 0; m < per_layer; ++m) l_id[m] = l_flat[m] != 0x7fffffff ? base_id + cnt++ : -1;
        int kept = 0;
        for (int k = 0; k < beam; ++k) {
            int bm = -1;
            for (int m = 0; m < per_layer; ++m)
                if (l_rank[m] < 0 && l_flat[m] != 0x7fffffff &&
                    (bm < 0 || before(Cand{l_y[m], l_flat[m]}, Cand{l_y[bm], l_flat[bm]})))
                    bm = m;
            if (bm < 0) break;
            l_rank[bm] = k;
            ++kept;
        }
        s_count[0] = cnt;
        s_count[1] = kept;
        ds.nb[seq * MTAD_MAX_DEPTH + step] = kept;
        ds.n_tree[seq] = base_id + cnt;
    }
    __syncthreads();
    for (int m = tid; m < per_layer; m += 256) {
        const int n = l_id[m];
        if (n < 0 || n >= N || n >= MTAD_DRAFT_NODES) continue;
        const int j = l_flat[m] / V, v = l_flat[m] % V;
        const float lq = s_lq[j] + l_lp[m];
        out.tok[bi * N + n] = v;
        out.parent[bi * N + n] = s_tree[j];
        out.depth[bi * N + n] = step + 1;
        out.node_logq[bi * N + n] = lq;
        const int k = l_rank[m];
        ds.tree2slot[seq * MTAD_DRAFT_NODES + n] = k >= 0 ? step * beam + k : -1;
        if (k >= 0) {
            const int slot = step * beam + k, parent = s_slot[j];
            ds.node_tok[seq * MTAD_DRAFT_NODES + slot] = v;
            ds.node_parent[seq * MTAD_DRAFT_NODES + slot] = parent;
            ds.node_logq[seq * MTAD_DRAFT_NODES + slot] = lq;
            ds.tree_id[seq * MTAD_DRAFT_NODES + slot] = n;
            uint32_t* mk = ds.node_mask + ((size_t)seq * MTAD_DRAFT_NODES + slot) * MTAD_MASK_WORDS;
            for (int i = 0; i < MTAD_MASK_WORDS; ++i) {
                uint32_t w;
                if (parent >= 0) w = ds.node_mask[((size_t)seq * MTAD_DRAFT_NODES + parent) * MTAD_MASK_WORDS + i];
                else {                                        // child of the root: sees all pending rows
                    const int lo = i * 32;
                    w = P >= lo + 32 ? 0xffffffffu : (P > lo ? (1u << (P - lo)) - 1u : 0u);
                }
                if (((P + slot) >> 5) == i) w |= 1u << ((P + slot) & 31);
                mk[i] = w;
            }
        }
    }
    __syncthreads();
    if (step == gamma - 1 && tid == 0) {
        // x**: the final beam with the highest draft likelihood (lowest node id on ties), and its prefix likelihoods
        __threadfence_block();
        const int kept = s_count[1];
        int best = -1;
        for (int k = 0; k < kept; ++k) {
            const int sl = (gamma - 1) * beam + k;
            if (best < 0) { best = sl; continue; }
            const float a = ds.node_logq[seq * MTAD_DRAFT_NODES + sl], b0 = ds.node_logq[seq * MTAD_DRAFT_NODES + best];
            if (a > b0 || (a == b0 && ds.tree_id[seq * MTAD_DRAFT_NODES + sl] < ds.tree_id[seq * MTAD_DRAFT_NODES + best]))
                best = sl;
        }
        int cur = best;
        for (int i = gamma - 1; i >= 0 && cur >= 0; --i) {
            out.best_path[bi * gamma + i] = ds.tree_id[seq * MTAD_DRAFT_NODES + cur];
            out.logq_ref[bi * gamma + i] = ds.node_logq[seq * MTAD_DRAFT_NODES + cur];
            ds.best_path[seq * MTAD_MAX_DEPTH + i] = cur;
            cur = ds.node_parent[seq * MTAD_DRAFT_NODES + cur];
        }
        ds.gamma[seq] = gamma;
        ds.beam[seq] = beam;
        if (out.n_nodes) out.n_nodes[bi] = ds.n_tree[seq];
    }
}

cudaError_t launch_draft_select_warped(const ModelView& m, const DraftState& ds, const Scratch& sc, const SeqList& seqs,
                                       int B, int R, int step, int gamma, int beam, int keep_all, const float* uniforms,
                                       const DraftOut& out, cudaStream_t st) {
    draft_pick_warped_kernel<<<B, 256, 0, st>>>(sc.warp_row, m.d.vocab, R, step, gamma, beam, keep_all, uniforms, ds, seqs,
                                                out);
    return cudaGetLastError();
}

// A sequence's rows of the next step are made by one block at the end of the selection, a warp a row, which saves a launch; as a launch of
// their own they have a block each.  Drafts of four steps, us, one way and the other: width 512, 4 beams 228 / 232; 768, 1 / 4 / 8 beams
// 209 / 214, 233 / 235, 265 / 267, eight sequences of four 310 / 313; 1024, 4 beams 238 / 239, eight sequences of eight 383 / 381; 1536, 4 and 8
// beams 241 / 240, 281 / 277; 2048 256 / 254, 299 / 291; 4096 306 / 299, 366 / 345; 8192 412 / 393, 481 / 436.
bool draft_rows_ahead(const mtad_model_desc& d) { return d.d_model <= 1024; }

// next: the next step's rows too; tc: as operand rows of the tensor-core path.
cudaError_t launch_draft_select(const ModelView& m, const DraftState& ds, const Scratch& sc, const SeqList& seqs, int B,
                                int R, int step, int gamma, int beam, int keep_all, const float* uniforms,
                                const DraftOut& out, const SeqState& s, const RowMeta& rm, bool next, bool tc, bool pdl,
                                cudaStream_t st) {
    const int V = m.d.vocab;
    int nch = (V + 1023) / 1024;
    nch = nch < 1 ? 1 : (nch > MTAD_DRAFT_CHUNKS ? MTAD_DRAFT_CHUNKS : nch);
    const int n_beams = step == 0 ? 1 : beam;
    const int kpb = (keep_all && step == 0) ? beam * beam : beam;
    return launch_pdl(draft_select_kernel, dim3(nch, n_beams, B), dim3(256), 0, st, pdl, (const float*)sc.logits, V, R, step, gamma,
                      beam, keep_all, kpb, uniforms, ds, seqs, sc.draft_part, nch, out, draft_rows(m, s, rm, sc, B * beam, tc), next);
}

// ---------------------------------------------------------------------------------------------------------------
// Roll-forward after a verification: the accepted rows of both caches move to their positions (commit_kernel), then the states
// of the sequences (advance_kernel).
// ---------------------------------------------------------------------------------------------------------------

// Beam slot of accepted node r of a verified draft.  mode 0: the verified chain was the draft's output sequence (chain
// node i = beam slot best_path[i]); mode 1: the verified tree was the draft's tree (node ids of that tree; a node that
// was recorded as a candidate only has no slot).  -1: no slot, -2: the path entry itself is out of range.
__device__ __forceinline__ int aux_slot_of(const DraftState& ds, const mtad_result& res, int bi, int seq, int D, int mode,
                                           int r) {
    const int pn = res.path[bi * D + r];
    if (pn < 0 || pn >= (mode == 0 ? MTAD_MAX_DEPTH : MTAD_DRAFT_NODES)) return -2;
    const int slot = mode == 0 ? ds.best_path[seq * MTAD_MAX_DEPTH + pn] : ds.tree2slot[seq * MTAD_DRAFT_NODES + pn];
    return slot >= MTAD_DRAFT_NODES ? -2 : (slot < 0 ? -1 : slot);
}

// Accepted nodes whose keys and values the draft left in the auxiliary cache: the leading ones that were beams of a
// layer before the last (the last layer, and candidates that were not kept, never ran).  At most one accepted token
// can follow them (such a node is a leaf of the tree).  Returns -1 when the path, the state or a cache row that the
// roll-forward would touch is out of range: accepted node r (r < kept) is read from slot base + beam slot and written
// to slot base + r, all inside [0, cap).
__device__ __forceinline__ int aux_kept_rows(const DraftState& ds, const mtad_result& res, int bi, int seq, int D, int mode,
                                             int eta, int base, long long cap) {
    const int gamma = ds.gamma[seq], beam = ds.beam[seq];
    if (gamma < 1 || gamma > MTAD_MAX_DEPTH || beam < 1 || beam > MTAD_MAX_BEAM || eta > D || base < 0) return -1;
    int kept = 0;
    for (; kept < eta; ++kept) {
        const int slot = aux_slot_of(ds, res, bi, seq, D, mode, kept);
        if (slot == -2) return -1;
        if (slot < 0 || slot >= (gamma - 1) * beam) break;
        if ((long long)base + slot >= cap) return -1;
    }
    if (eta - kept > 1 || kept > MTAD_MAX_DEPTH || (long long)base + kept > cap) return -1;
    return kept;
}

// What keeps the auxiliary model from following the accepted tokens of a sequence (0: nothing): then its target does not either.
// mode 2: no draft produced the verified rows.
__device__ __forceinline__ uint32_t aux_obstacle(const SeqState& s, const DraftState& ds, const mtad_result& res, int bi, int seq, int D,
                                                 int mode, int max_batch, long long cap, int& kept) {
    const int eta = res.eta[bi];
    kept = 0;
    if ((unsigned)seq >= (unsigned)max_batch || eta < 0 || eta > D) return MTAD_ST_RANGE;
    if (mode == 2) return s.aux_npend[seq] + eta + 1 > MTAD_MAX_DEPTH + 1 ? MTAD_ST_AUX_PENDING : 0u;
    kept = aux_kept_rows(ds, res, bi, seq, D, mode, eta, ds.base_len[seq] + ds.npend[seq], cap);
    return kept < 0 ? MTAD_ST_RANGE : 0u;
}

struct CommitCache {
    __nv_bfloat16* cache;       // null: no auxiliary model
    int planes, Hkv, hd;        // planes: layers x K|V x KV heads
    long long cap;
};

// Node path[i] (cache slot L + 1 + path[i], of the auxiliary model base + beam slot) moves to position L + 1 + i (base + i).  Blocks
// 0 .. nt - 1 of a sequence share out the target's rows, the others the auxiliary model's, in columns of 16 bytes (what every attention
// kernel reads at a time) of a (layer, K|V, KV head): a thread reads its column of all rows before it writes any (a destination may
// be a later move's source), so the loads of the rows are in flight together and no thread waits for another.  Rows that stay
// where they are (an accepted chain) are left alone.
__global__ void __launch_bounds__(128) commit_kernel(CommitCache tg, CommitCache ax, SeqState s, DraftState ds,
                                                     const int32_t* __restrict__ call_seq, mtad_result res, int D, int mode,
                                                     int max_batch, int nt) {
    __shared__ int src[MTAD_MAX_DEPTH];
    __shared__ int n_rows, dst, moved, stop;
    const int bi = blockIdx.y, tid = threadIdx.x;
    const bool target = (int)blockIdx.x < nt;
    pdl_wait();
    pdl_trigger();
    if (res.status[bi] != 0) return;
    const int eta = res.eta[bi], seq = call_seq[bi];
    if (eta <= 0 || eta > D || eta > MTAD_MAX_DEPTH || (unsigned)seq >= (unsigned)max_batch) return;
    if (tid == 0) {
        int kept = 0, n = eta, to;
        const uint32_t no = ax.cache ? aux_obstacle(s, ds, res, bi, seq, D, mode, max_batch, ax.cap, kept) : 0u;
        if (target) {
            // every source and destination row inside the cache, or nothing moves (advance_kernel flags the sequence)
            to = s.kv_len[seq] + 1;
            if (no || to < 1 || (long long)to + eta > tg.cap) n = 0;
        } else {
            n = no || mode == 2 ? 0 : kept;
            to = mode == 2 ? 0 : ds.base_len[seq] + ds.npend[seq];
        }
        n_rows = n;
        dst = to;
        moved = stop = 0;
    }
    __syncthreads();
    const int n = n_rows;
    if (n == 0) return;
    if (tid < n) {
        const int from = target ? res.path[bi * D + tid] : aux_slot_of(ds, res, bi, seq, D, mode, tid);
        src[tid] = from;
        if (from != tid) moved = 1;
        if (target && (from < 0 || (long long)dst + from >= tg.cap)) stop = 1;
    }
    __syncthreads();
    if (stop || !moved) return;
    const CommitCache& c = target ? tg : ax;
    const int cols = c.hd / 8, items = c.planes * cols, step = (target ? nt : (int)gridDim.x - nt) * 128;
    for (int i = (target ? blockIdx.x : blockIdx.x - nt) * 128 + tid; i < items; i += step) {
        const int pl = i / cols, head = pl % c.Hkv, kv = (pl / c.Hkv) & 1, layer = pl / (2 * c.Hkv);
        uint4* b = reinterpret_cast<uint4*>(c.cache + idx_cache(layer, max_batch, seq, kv, c.Hkv, head, c.cap, dst, c.hd)) + i % cols;
        constexpr int NV = 8;
        if (n <= NV) {
            uint4 v[NV];
#pragma unroll
            for (int r = 0; r < NV; ++r)
                if (r < n) v[r] = b[(size_t)src[r] * cols];
#pragma unroll
            for (int r = 0; r < NV; ++r)
                if (r < n) b[(size_t)r * cols] = v[r];
        } else {
            uint4 v[MTAD_MAX_DEPTH];
            for (int r = 0; r < n; ++r) v[r] = b[(size_t)src[r] * cols];
            for (int r = 0; r < n; ++r) b[(size_t)r * cols] = v[r];
        }
    }
}

// New states.  Auxiliary, mode 0 / 1: after a draft (see above); mode 2: the accepted tokens and the new root simply join the pending
// list (to be replayed by the next draft).
__global__ void advance_kernel(SeqState s, DraftState ds, const int32_t* __restrict__ call_seq, mtad_result res, int D, int mode,
                               int B, int max_batch, bool has_aux, long long aux_cap, long long cap) {
    const int bi = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    pdl_trigger();
    if (bi >= B || res.status[bi] != 0) return;
    const int seq = call_seq[bi], eta = res.eta[bi];
    if (has_aux) {
        int kept;
        const uint32_t no = aux_obstacle(s, ds, res, bi, seq, D, mode, max_batch, aux_cap, kept);
        if (no) { atomicOr(&res.status[bi], no); return; }
        int32_t* pend = s.aux_pend + seq * (MTAD_MAX_DEPTH + 1);
        if (mode == 2) {
            const int np = s.aux_npend[seq];
            for (int i = 0; i <= eta; ++i) pend[np + i] = res.out_tok[bi * (D + 1) + i];
            s.aux_npend[seq] = np + eta + 1;
        } else {
            s.aux_len[seq] = ds.base_len[seq] + ds.npend[seq] + kept;
            int np = 0;
            if (eta > kept) pend[np++] = res.out_tok[bi * (D + 1) + eta - 1];   // accepted, but never run by the auxiliary model
            pend[np++] = res.out_tok[bi * (D + 1) + eta];
            s.aux_npend[seq] = np;
        }
    }
    bool ok = (unsigned)seq < (unsigned)max_batch && eta >= 0 && eta <= D;
    if (ok) {
        const long long L = s.kv_len[seq];
        ok = L >= 0 && L + 1 + eta <= cap;
        for (int r = 0; r < eta && ok; ++r) {
            const int pn = res.path[bi * D + r];
            ok = pn >= 0 && L + 1 + pn < cap;
        }
    }
    if (!ok) { atomicOr(&res.status[bi], MTAD_ST_RANGE); return; }
    s.kv_len[seq] += eta + 1;
    s.root_tok[seq] = res.out_tok[bi * (D + 1) + eta];
}

cudaError_t launch_commit(const ModelView& m, const ModelView* aux, const SeqState& s, const DraftState& ds, int B,
                          const int32_t* call_seq_dev, const mtad_result& res, int max_depth, int mode, bool pdl, cudaStream_t st) {
    auto cache_of = [](const ModelView& v) {
        return CommitCache{static_cast<__nv_bfloat16*>(v.d.kv_cache), v.d.layers * 2 * v.d.n_kv_heads, v.d.n_kv_heads, v.d.head_dim,
                           (long long)v.d.kv_capacity};
    };
    const CommitCache tg = cache_of(m), ax = aux ? cache_of(*aux) : CommitCache{};
    // A thread per 16-byte column while a wave (8 blocks an SM) holds that many, then several a thread.  What bounds it is the moved rows'
    // traffic where there is some, and otherwise its chain of a few dependent loads and two launches.  us with the launch after it: 40
    // layers of 40 heads, 8 sequences, 6 rows of 128 moved each 24, 20 rows 83 (a block per plane, elements of two bytes through shared
    // memory: 91 and 239; 592 blocks that took the planes in turn: 169 and 509); 32 x 32 heads, 4 rows, 1 / 64 sequences 11 / 56 (15 / 297,
    // 19 / 360); nothing to move 9 (17..89 with a block per plane).
    auto blocks = [&](const CommitCache& c) { return std::min((c.planes * (c.hd / 8) + 127) / 128, std::max(16, 8 * 148 / B)); };
    const int nt = blocks(tg), na = aux && mode != 2 ? blocks(ax) : 0;
    cudaError_t e = launch_pdl(commit_kernel, dim3(nt + na, B), dim3(128), 0, st, pdl, tg, ax, s, ds, call_seq_dev, res, max_depth,
                               mode, m.max_batch, nt);
    if (e != cudaSuccess) return e;
    return launch_pdl(advance_kernel, dim3(1), dim3(64), 0, st, pdl, s, ds, call_seq_dev, res, max_depth, mode, B, m.max_batch,
                      aux != nullptr, ax.cap, tg.cap);
}

}  // namespace mtad
