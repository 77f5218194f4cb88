// The rule of vanilla speculative decoding (Sec. 2.2 of the paper) as a second accept mode on the same verify
// forward: draft token i is accepted iff u_i < min(1, p_i(x_i) / q_i(x_i)); the first rejection ends the scan and
// its position is resampled from norm(max(0, p_i - q_i)); with every token accepted one more is drawn from the
// target's next row.  Works on the plain logits [rows, V] of the forward and the auxiliary model's normalised
// log-distributions at the draft positions (the caller's), a block per row and chunk.
#include <math_constants.h>

#include "common.cuh"

namespace mtad {

namespace {

struct Pick {
    float y;
    int v;
};
__device__ __forceinline__ bool ahead(const Pick& a, const Pick& b) { return a.y > b.y || (a.y == b.y && a.v < b.v); }

}  // namespace

// Three launches.  One block per sequence for everything walked 2 R + 1 vocabulary rows one after the other, bound by the
// latency of its loads and the instructions of one SM (117 us for three sequences of six rows and 32000 tokens); now a block per
// row forms the log-sum-exp, a block per chunk of the vocabulary the best candidate of the last token, and a warp per
// sequence picks among the chunks (together 26 us).
constexpr int SPD_CHUNKS = 16;
static_assert(SPD_CHUNKS <= MTAD_DRAFT_CHUNKS && sizeof(Pick) <= sizeof(WarpPart), "the chunks' picks lie in warp_part");

__device__ __forceinline__ bool spd_skip(const RowMeta& rm, const mtad_result& out, int bi) {
    return out.status[bi] != 0 || rm.n_rows[bi] == 0;
}

// log-sum-exp of every row (fixed combination order)
__global__ void __launch_bounds__(1024) spd_lse_kernel(const float* __restrict__ logits, int V, RowMeta rm, int R,
                                                       float* __restrict__ row_lse, mtad_result out) {
    const int bi = blockIdx.y, t = bi * R + blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ float s_red[32];
    pdl_wait();
    pdl_trigger();
    if (spd_skip(rm, out, bi)) return;
    const float* z = logits + (size_t)t * V;
    float m = -CUDART_INF_F;
#pragma unroll 8
    for (int v = tid; v < V; v += 1024) m = fmaxf(m, z[v]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) s_red[warp] = m;
    __syncthreads();
    m = s_red[0];
    for (int w = 1; w < 32; ++w) m = fmaxf(m, s_red[w]);
    __syncthreads();
    float sum = 0.f;
#pragma unroll 8
    for (int v = tid; v < V; v += 1024) sum += expf(z[v] - m);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s_red[warp] = sum;
    __syncthreads();
    if (tid == 0) {
        float acc = 0.f;
        for (int w = 0; w < 32; ++w) acc += s_red[w];
        row_lse[t] = m + logf(acc);
    }
}

// The accept scan (every block for itself, the first one of a sequence writes it), and the chunk's best candidate of the
// last token: from the target's row after the chain, or from the positive part of p - q at the rejection.
__global__ void __launch_bounds__(256) spd_scan_kernel(const float* __restrict__ logits, int V, RowMeta rm, SpdArgs a,
                                                       const float* __restrict__ row_lse, WarpPart* __restrict__ parts,
                                                       mtad_result out) {
    const int bi = blockIdx.y, ch = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int R = a.R, g = R - 1, D = a.max_depth;
    __shared__ int s_eta;
    __shared__ Pick s_p[8];
    pdl_wait();
    pdl_trigger();
    // (what a sequence with nothing to do reports, the last launch writes: these blocks read the status)
    if (spd_skip(rm, out, bi)) return;
    const float* z0 = logits + (size_t)bi * R * V;
    const float* lse0 = row_lse + (size_t)bi * R;
    if (warp == 0) {
        bool finite = true;
        for (int r = lane; r < R; r += 32) finite = finite && isfinite(lse0[r]);
        finite = __all_sync(0xffffffffu, finite);
        // a lane per draft token; accepted up to the first rejection
        int eta = 0;
        float margin = CUDART_INF_F;
        for (int i0 = 0; i0 < g && finite && eta == i0; i0 += 32) {
            const int i = i0 + lane;
            bool ok = false;
            float lp = 0.f, gap = CUDART_INF_F;
            int x = 0;
            if (i < g) {
                x = a.tok[bi * g + i];
                lp = z0[(size_t)i * V + x] - lse0[i];
                const float ratio = fminf(0.f, lp - a.logq_rows[((size_t)bi * g + i) * V + x]);
                const float lu = logf(a.accept_uniform[bi * g + i]);
                gap = fabsf(lu - ratio);
                ok = lu < ratio;
            }
            const uint32_t no = __ballot_sync(0xffffffffu, !ok);
            const int n = min(no ? __ffs(no) - 1 : 32, g - i0);
            eta = i0 + n;
            if (lane > n) gap = CUDART_INF_F;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) gap = fminf(gap, __shfl_xor_sync(0xffffffffu, gap, o));
            margin = fminf(margin, gap);
            if (ch == 0 && lane < n) {
                out.path[bi * D + i] = i;
                out.out_tok[bi * (D + 1) + i] = x;
                out.out_lp[bi * (D + 1) + i] = lp;
            }
        }
        if (lane == 0) {
            s_eta = finite ? eta : -1;
            if (ch == 0 && finite) {
                out.eta[bi] = eta;
                out.winner[bi] = eta - 1;
                out.n_out[bi] = eta + 1;
                if (out.margin) { out.margin[bi * 2] = margin; out.margin[bi * 2 + 1] = CUDART_INF_F; }
            }
        }
    }
    __syncthreads();
    const int eta = s_eta;
    if (eta < 0) return;
    const float* z = z0 + (size_t)eta * V;
    const float lse = lse0[eta];
    const float* lq = eta < g ? a.logq_rows + ((size_t)bi * g + eta) * V : nullptr;
    const float* u = a.resample_uniform + (size_t)bi * V;
    const int per = (V + SPD_CHUNKS - 1) / SPD_CHUNKS, v1 = min(V, (ch + 1) * per);
    Pick best{-CUDART_INF_F, 0x7fffffff};
#pragma unroll 4
    for (int v = ch * per + tid; v < v1; v += 256) {
        float s;
        if (lq) {
            const float w = expf(z[v] - lse) - expf(lq[v]);
            s = w > 0.f ? logf(w) : -CUDART_INF_F;
        } else {
            s = z[v] - lse;
        }
        if (s == -CUDART_INF_F) continue;
        const Pick c{s - logf(-logf(u[v])), v};
        if (ahead(c, best)) best = c;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const Pick c{__shfl_xor_sync(0xffffffffu, best.y, o), __shfl_xor_sync(0xffffffffu, best.v, o)};
        if (ahead(c, best)) best = c;
    }
    if (lane == 0) s_p[warp] = best;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < 8; ++w)
            if (ahead(s_p[w], best)) best = s_p[w];
        *reinterpret_cast<Pick*>(parts + (size_t)bi * MTAD_DRAFT_CHUNKS + ch) = best;
    }
}

__global__ void __launch_bounds__(32) spd_pick_kernel(const float* __restrict__ logits, int V, RowMeta rm, SpdArgs a,
                                                      const float* __restrict__ row_lse, const WarpPart* __restrict__ parts,
                                                      mtad_result out) {
    const int bi = blockIdx.x, lane = threadIdx.x, R = a.R, g = R - 1, D = a.max_depth;
    pdl_wait();
    pdl_trigger();
    const float* lse0 = row_lse + (size_t)bi * R;
    bool finite = true;
    const bool skip = spd_skip(rm, out, bi);
    if (!skip)
        for (int r = lane; r < R; r += 32) finite = finite && isfinite(lse0[r]);
    finite = __all_sync(0xffffffffu, finite);
    if (skip || !finite) {
        // rows of NaN logits: flag the sequence and accept nothing, as the other modes do
        if (lane == 0) {
            if (!finite) atomicOr(&out.status[bi], MTAD_ST_NONFINITE);
            out.eta[bi] = 0; out.winner[bi] = -1; out.n_out[bi] = 0;
        }
        return;
    }
    const int eta = out.eta[bi], nrows = rm.n_rows[bi];
    Pick best{-CUDART_INF_F, 0x7fffffff};
    if (lane < SPD_CHUNKS) best = *reinterpret_cast<const Pick*>(parts + (size_t)bi * MTAD_DRAFT_CHUNKS + lane);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const Pick c{__shfl_xor_sync(0xffffffffu, best.y, o), __shfl_xor_sync(0xffffffffu, best.v, o)};
        if (ahead(c, best)) best = c;
    }
    const float* z0 = logits + (size_t)bi * R * V;
    if (lane == 0) {
        // (p == q everywhere leaves no residual mass; the ratio test cannot reject then, so a row is always found)
        const int t = best.v == 0x7fffffff ? 0 : best.v;
        out.out_tok[bi * (D + 1) + eta] = t;
        out.out_lp[bi * (D + 1) + eta] = z0[(size_t)eta * V + t] - lse0[eta];
    }
    // optional per-row outputs of the result struct
    if (out.row_lse) for (int r = lane; r < R; r += 32) out.row_lse[bi * R + r] = r < nrows ? lse0[r] : 0.f;
    if (out.node_lp) for (int n = lane; n < g; n += 32)
        out.node_lp[bi * g + n] = z0[(size_t)n * V + a.tok[bi * g + n]] - lse0[n];
}

cudaError_t launch_spd_accept(const ModelView& m, const RowMeta& rm, const Scratch& sc, const SpdArgs& a,
                              const mtad_result& out, bool pdl, cudaStream_t st) {
    const float* logits = sc.logits;
    const int V = m.d.vocab;
    cudaError_t e = launch_pdl(spd_lse_kernel, dim3(a.R, a.B), dim3(1024), 0, st, pdl, logits, V, rm, a.R, sc.row_lse, out);
    if (e == cudaSuccess)
        e = launch_pdl(spd_scan_kernel, dim3(SPD_CHUNKS, a.B), dim3(256), 0, st, pdl, logits, V, rm, a,
                       (const float*)sc.row_lse, sc.warp_part, out);
    if (e == cudaSuccess)
        e = launch_pdl(spd_pick_kernel, dim3(a.B), dim3(32), 0, st, pdl, logits, V, rm, a, (const float*)sc.row_lse,
                       (const WarpPart*)sc.warp_part, out);
    return e;
}

}  // namespace mtad
