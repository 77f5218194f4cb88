// The decoder forward of a few draft rows as one cooperative launch: one block per SM walks every layer's phases
//   QKV (+ rotary, KV append)  |  attention  |  O (+ residual)  |  gate / up (+ SwiGLU)  |  down (+ residual)
// and the LM head, with a grid barrier between phases.
//
// What bounds it: the weights (and K / V) pass once through every SM's copy ring, so the floor is HBM bandwidth.  As a
// chain of launches this work lost 7..8 us at every projection - drain, split-K exchange, epilogue, the launch boundary,
// and a copy ring that starts empty.  Here the weight producer does not know phases: as the last k-blocks of a projection
// leave the ring, the first ones of the next (or the committed K / V tiles of the attention) take their place, so HBM
// stays busy across the barrier for as long as the ring is deep.  Two more things keep the boundary short: every block
// owns whole output features (the features are cut into one tile per SM, not into 128-row tiles), so no partial sum leaves
// an SM while rows are few; and only the call's terms x rows operand rows are multiplied (16 columns for five rows).
// Measured (chain of launches -> one launch, both ways in turn on one GPU, a whole verification step): 7B, 5 rows 3.36 ->
// 2.94 ms (weights and K / V in 2.2 ms at copy speed), 33 rows 4.30 -> 3.53, 65 rows 6.03 -> 4.56; 13B, 8 x 7 rows 9.98 -> 8.58;
// two-layer auxiliary model of width 768, four draft steps 506 -> 380 us.  A phase of a large model costs its bytes plus about
// 3 us (barrier 1.1, first operand rows 0.6, last MMA to last store 1.2 and up); the phases of the auxiliary model, which move next to
// nothing, take about 6, and the attention of a chain 7 more than its bytes.  Part of that is waiting for instructions: what an
// epilogue executes runs once a phase, and a layer's worth of it does not fit an SM's instruction cache (four layers of 7B, 5 rows:
// 6.3k misses of 23.8k lookups an SM; 8.1k of 26.6k, and 0.3 us more a phase, before the code of few rows was made smaller).  Code here
// should be short before it is clever: unrolled groups of loads that saved round trips made a step slower.
//
// Contraction.  Weights are the 128-row MMA operand A, the operand rows (two or three bf16 terms per activation, see
// store_terms) operand B.  Where a block owns at most 64 features, the MMA takes S k-blocks at once: their weights lie
// side by side in A, their operand rows side by side in B, and of the S x S blocks of the product the diagonal ones are
// the k-blocks' contributions, summed by the epilogue.  One MMA of 128 x 64 costs what one of 128 x 16 does, so this is S
// times fewer MMAs (an MMA takes 65 cycles whatever N <= 128 is: 32 rows at a time would cap an SM at 30 GB/s).
//
// Attention: keys as the M dimension.  The (sequence, KV head, 128-key tile) items are dealt out in pieces of one (sequence, KV head)
// each, or evenly, in order.
//   S^T = K Q^T   A = K tile as it lies in the cache, B = query rows (bf16 hi rows, then lo rows)
//   P = exp2(S - m), a thread per key and half of the query rows, written to shared memory as three bf16 terms
//   O^T += V^T P  A = V tile (MN-major), B = P; a thread per head dimension and half of the rows adds it to its registers
// Pieces of a (sequence, KV head) held by several blocks meet in global memory; the block that arrives last merges them.
// An item takes up to 8 or 16 query rows of a KV head, or 40 in the wide variant (an instantiation each: the softmax's time
// goes with the rows, padding included; beyond 40 a thread's 20 rows would leave its registers), and more are cut into
// blocks of equal size.  Per tile 0.75 us at 8 rows, 1.6 at 40, against 1.3 us that K and V take at copy speed (before the
// third term of P).  7B, 65 rows on 2048 keys: 39 -> 35 us a layer against `mma.sync` warps; 64 heads on 8 KV heads, 129 rows,
// 1024 keys: a layer of the whole step 960 -> 846.
//
// Warps: 0 weight and K / V producer (TMA), 1 operand-row producer (TMA; waits for the phase before), 2 and 3 MMA issuers
// (3 owns the tensor memory), 4..11 epilogue and softmax.
// Every wait is bounded by a number of polls (WAIT_LIMIT); a block that gives up raises MTAD_ST_TIMEOUT for every sequence of
// the call and leaves, and the others run into their own limits at the grid barrier.
#include <math_constants.h>

#include <cstddef>

#include <algorithm>
#include <type_traits>

#include "forward.cuh"
#include "tc_device.cuh"

namespace mtad {
using namespace tcdev;

namespace {

constexpr int FW_THREADS = 32 * 12;
constexpr int FW_EPI_WARP0 = 4;
constexpr int FW_EPI = 256;
constexpr int FW_UNION = 32 * 1024;       // epilogue tile Y, or the attention's query and probability tiles
constexpr int FW_ACC = 240;               // accumulator columns of a tile, of 256 (the drain reads up to 16 columns further),
constexpr int FW_ACC_ONE = 496;           // or of 512 where a tile takes both buffers
static_assert(FW_ACC + 16 <= 256 && FW_ACC_ONE + 16 <= 512, "columns that a drain reads");
static_assert(2 * FW_MAX_COLS + 2 * FW_MAX_ROWS <= 512 && FW_MAX_ROWS % 16 == 0, "gate / up with the sums put by");
constexpr float FW_LAZY = 64.f;           // log2 of how far a score may exceed its row's reference value
constexpr float FW_UNSEEN = -1e30f;       // the reference value of a row that has seen no key

__device__ __forceinline__ bool grid_wait(const int* c, int want, volatile int* abort_flag) {
    const uint32_t limit = (uint32_t)abort_flag[1];
    for (uint32_t it = 0; it < limit; ++it) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(c) : "memory");
        if (v >= want) return true;
        if ((it & 31u) == 31u && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
// The layer table's tensor maps lie in global memory, where the host wrote them: an SM's descriptor cache may still hold
// what an earlier table had at the same address (a context that is gone), so each is acquired before its first use.
__device__ __forceinline__ void map_acquire(const CUtensorMap* m) {
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// before TMA reads what other SMs wrote to global memory (after the acquire that saw it); the form for all state spaces, which also
// waits for this thread's shared memory, takes 0.3 us longer a phase
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ uint2 pack4(float x, float y, float z, float w) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(x, y), q = __floats2bfloat162_rn(z, w);
    return make_uint2(*reinterpret_cast<const uint32_t*>(&p), *reinterpret_cast<const uint32_t*>(&q));
}
__device__ __forceinline__ void store_bf4(const float* v, __nv_bfloat16* d) {
    *reinterpret_cast<uint2*>(d) = pack4(v[0], v[1], v[2], v[3]);
}
// four values times `scale` as bf16 hi and lo parts
__device__ __forceinline__ void split_store4(const float* v, float scale, __nv_bfloat16* hi, __nv_bfloat16* lo) {
    const float x = v[0] * scale, y = v[1] * scale, z = v[2] * scale, w = v[3] * scale;
    const uint2 h = pack4(x, y, z, w);
    *reinterpret_cast<uint2*>(hi) = h;
    *reinterpret_cast<uint2*>(lo) = pack4(x - __uint_as_float(h.x << 16), y - __uint_as_float(h.x & 0xffff0000u),
                                          z - __uint_as_float(h.y << 16), w - __uint_as_float(h.y & 0xffff0000u));
}
// barrier and consensus of `n` threads
__device__ __forceinline__ bool all_of(int id, int n, bool ok) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.red.and.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(ok ? 1u : 0u), "r"(id), "r"(n)
        : "memory");
    return r != 0;
}
// one lane of the warp waits
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, bool ok, int lane) {
    if (lane == 0 && ok) ok = mbar_wait(bar, parity, abort_flag);
    return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}
__device__ __forceinline__ void bar_n(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z, int u,
                                            uint64_t hint) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4, %5, %6}], [%2], %7;" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(u), "l"(hint)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z,
                                            uint64_t hint) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4, %5}], [%2], %6;" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z), "l"(hint)
        : "memory");
}
// MN-major, 128-byte swizzle: a k row (one key) is 64 elements = 128 bytes, 8 keys are 1024 bytes, the next 64 elements
// of the M dimension lie 128 keys further
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((FW_KEYS * 128) >> 4) << 16) | (64ull << 32) | (1ull << 46) |
           (2ull << 61);
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
    const int n = valid ? 16 : 0;                      // src-size 0: the 16 bytes are zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// 16 columns of a box's `na` accumulators (up to four), `stride` columns apart, added up
__device__ __forceinline__ void acc_ld16(uint32_t at, int stride, int na, float* v) {
    if (na == 1) {
        tc_ld16(at, v);
        return;
    }
    tc_ld16_sum(at, at + stride, v);
    if (na > 2) {
        float w[16];
        if (na > 3) tc_ld16_sum(at + 2 * stride, at + 3 * stride, w);
        else tc_ld16(at + 2 * stride, w);
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] += w[j];
    }
}

// What a call's sequence looks like to the attention
struct SeqMeta {
    int nrows, L, nkeys, seq;
};

// The attention items of a call: sequences in order, KV heads in order, 128-key tiles in order.  Either block c takes
// [c * per, (c + 1) * per), or (`cut`) every (sequence, KV head) is cut into pieces of `per` tiles, a block each.
struct AttnPos {
    int bi, g, tile, nt;                  // nt: tiles of the sequence
    int f0;                               // first item of the (sequence, KV head)
};
__device__ __forceinline__ int attn_tiles(const SeqMeta& m) { return m.nrows > 0 ? (m.nkeys + FW_KEYS - 1) / FW_KEYS : 0; }
__device__ __forceinline__ AttnPos attn_find(const SeqMeta* meta, int B, int Hkv, int x) {
    AttnPos it{};
    int base = 0;
    for (int b = 0; b < B; ++b) {
        const int nt = attn_tiles(meta[b]);
        if (x < base + nt * Hkv) {
            it.bi = b;
            it.nt = nt;
            it.g = (x - base) / nt;
            it.tile = x - base - it.g * nt;
            it.f0 = x - it.tile;
            break;
        }
        base += nt * Hkv;
    }
    return it;
}
__device__ __forceinline__ void attn_next(AttnPos& it, const SeqMeta* meta, int B, int Hkv) {
    if (++it.tile < it.nt) return;
    it.f0 += it.nt;
    it.tile = 0;
    if (++it.g < Hkv) return;
    it.g = 0;
    do ++it.bi; while (it.bi < B && attn_tiles(meta[it.bi]) == 0);
    if (it.bi < B) it.nt = attn_tiles(meta[it.bi]);
}

// Pieces of a (sequence, KV head), and which of them is that of block `cta`, which holds the tile `q`.
__device__ __forceinline__ int attn_pieces(const AttnPos& q, int per, bool cut) {
    return cut ? (q.nt + per - 1) / per : (q.f0 + q.nt - 1) / per - q.f0 / per + 1;
}
__device__ __forceinline__ int attn_piece(const AttnPos& q, int per, bool cut, int cta) { return cut ? q.tile / per : cta - q.f0 / per; }
// First item and number of items of block `cta` when the (sequence, KV head)s are cut into pieces of `per` tiles; returns
// how many blocks that takes in all.
__device__ __forceinline__ int attn_cut(const SeqMeta* meta, int B, int heads, int per, int cta, int& lo, int& n) {
    int blocks = 0, items = 0;
    lo = n = 0;
    for (int b = 0; b < B; ++b) {
        const int nt = attn_tiles(meta[b]), np = (nt + per - 1) / per;
        if (cta >= blocks && cta < blocks + np * heads) {
            const int g = (cta - blocks) / np, x = (cta - blocks - g * np) * per;
            lo = items + g * nt + x;
            n = min(per, nt - x);
        }
        blocks += np * heads;
        items += nt * heads;
    }
    return blocks;
}

// Where a tile's weights lie: map and row coordinate of its boxes (QKV: pair and half-head coordinates).
struct TileSrc {
    const CUtensorMap *m, *m2;
    int row, row2, half, half2;
};
__device__ __forceinline__ TileSrc tile_src(const FwArgs& a, int kind, int layer, int tile) {
    const FwPhase& f = a.ph[kind];
    const CUtensorMap* w = a.layers[layer].w[a.cls];           // (not read for the LM head)
    TileSrc t{w, w, tile * f.nbox * f.h, 0, 0, 0};
    auto of_head = [&](int hg, const CUtensorMap*& map, int& pos) {
        pos = 2 * (hg < a.Hq ? hg : (hg < a.Hq + a.Hkv ? hg - a.Hq : hg - a.Hq - a.Hkv));
        map = w + (hg < a.Hq ? 0 : (hg < a.Hq + a.Hkv ? 1 : 2));
    };
    if (kind == FW_QKV && f.nbox == 2) {                       // a tile of two heads
        const int hg = tile / f.c * 2;
        t.row = 0;
        of_head(hg, t.m, t.half);
        of_head(min(hg + 1, a.Hq + 2 * a.Hkv - 1), t.m2, t.half2);
    } else if (kind == FW_QKV) {
        const int hg = tile / f.u;
        t.row = (tile - hg * f.u) * f.h;
        of_head(hg, t.m, t.half);
    } else if (kind == FW_GATEUP) {
        t.m = w + 4;
        t.m2 = w + 5;
        t.row = t.row2 = tile * f.h;
    } else if (kind == FW_LM) {
        t.m = t.m2 = &a.lm;
        t.row2 = t.row + f.h;
    } else {
        t.m = kind == FW_O ? w + 3 : w + 6;
        if (f.c > 1) t.row = tile / f.c * f.h;
    }
    if (kind != FW_LM) {
        map_acquire(t.m);
        if (f.nbox == 2) map_acquire(t.m2);
    }
    return t;
}
// one step of a tile's weights to the ring slot at `base`
__device__ __forceinline__ void copy_step(const FwArgs& a, int kind, const TileSrc& t, int step, uint32_t base, uint32_t bar) {
    const FwPhase& f = a.ph[kind];
    const int kx = f.flat ? step * TC_TILE_K : 0, kz = f.flat ? 0 : step * f.kb;
    mbar_expect_tx(bar, (uint32_t)(f.nbox * f.box_bytes + f.kb * a.cols * 128));
    if (kind == FW_QKV) {
        tma_load_4d(base, t.m, bar, kx, t.row, t.half, kz, HINT_STREAM);
        if (f.nbox == 2) tma_load_4d(base + f.box_bytes, t.m2, bar, kx, t.row, t.half2, kz, HINT_STREAM);
    } else {
        tma_load_3d(base, t.m, bar, kx, t.row, kz, HINT_STREAM);
        if (f.nbox == 2) tma_load_3d(base + f.box_bytes, t.m2, bar, kx, t.row2, kz, HINT_STREAM);
    }
}
// steps [k_first, k_end) of a tile are its block's: all of them, or its share
__device__ __forceinline__ int k_first(const FwPhase& f, int tile) { return f.c > 1 ? (tile % f.c) * f.steps / f.c : 0; }
__device__ __forceinline__ int k_end(const FwPhase& f, int tile) { return f.c > 1 ? (tile % f.c + 1) * f.steps / f.c : f.steps; }

// What the attention's epilogue warps tell one another, for NR rows in each half of them
template <int NR>
struct alignas(16) FwAttn {
    float smx[2][NR][4];                  // row maxima of the four warps
    float sl[2][2][NR][4];                // row sums of the four warps, two segments
    float sm[2][NR];                      // reference values
};
struct FwTail {
    SeqMeta meta[MTAD_MAX_BATCH];
    float rstd[FW_MAX_ROWS];
    int slot[FW_MAX_ROWS];                // cache slot of a row, -1: inactive
    uint8_t rowb[FW_MAX_ROWS];            // its sequence within the call
    FwAttn<FW_QROWS / 2> attn;            // (the wide attention's lies behind its query tile)
    uint64_t full[4], empty[4];
    uint64_t tfull[2], tempty[2], sfull[2], pfull[2], ofull[2], qfull[2];
    uint32_t tmem_ptr;
    int abort_flag[2];
    int last[2];
    AttnPos apos[3];                      // attention items of this block: the lowest, the highest, the one it takes first
    int arange[3];                        // how many; tiles of a block or piece, whether they are pieces
};
static_assert(offsetof(FwTail, attn) % 16 == 0 && offsetof(FwTail, full) % 8 == 0, "alignment of the tail");
static_assert(FW_RING + FW_UNION + sizeof(FwTail) <= 227 * 1024, "shared memory of the forward");

// O or down where c blocks share the k-range of a tile: each leaves its accumulators in global memory as they lie in tensor
// memory (a row's features, the S slices side by side), the blocks wait for one another, and each finishes a share of the
// rows, a warp per row, adding the parts in order (deterministic).
__device__ __forceinline__ bool split_residual(const FwArgs& a, FwTail& s, const FwPhase& f, bool is_o, int layer, int tcount, int e,
                                               uint32_t tmem_lane, int tile) {
    volatile int* abort_flag = s.abort_flag;
    const int lane = e & 31, w = e >> 5, quad = w & 3, half = w >> 2;
    const int T = a.T, terms = a.terms, cols = a.cols, S = f.S, hr = f.hr, yb = S * hr, c = f.c;
    const int tl = quad * 32 + lane, my = tl / hr, s0 = quad * 32 / hr, s1 = min(S - 1, (quad * 32 + 31) / hr);
    const int per = terms == 3 ? 5 : 8, buf = tcount & 1;
    const int kp = tile % c, ra = T * kp / c, rn = T * (kp + 1) / c, n = tile / c * hr + 4 * lane;
    const bool in = 4 * lane < hr && n < a.d;
    constexpr int RW = 3;                                  // rows of a warp whose loads are in flight together
    float4 hid[RW];
    auto load_hid = [&](int t0) {
#pragma unroll
        for (int x = 0; x < RW; ++x)
            hid[x] = in && t0 + 8 * x < rn ? __ldcg(reinterpret_cast<const float4*>(a.hidden + (size_t)(t0 + 8 * x) * a.d + n))
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    load_hid(ra + w);
    float g[4];
    const __nv_bfloat16* gain = is_o ? a.layers[layer].gain_ffn : a.layers[layer].gain_next;
#pragma unroll
    for (int x = 0; x < 4; ++x) g[x] = in ? __bfloat162float(gain[n + x]) : 0.f;
    bool ok = true;
    if (e == 0) ok = mbar_wait(smem_u32(&s.tfull[buf]), (uint32_t)(tcount >> 1) & 1u, abort_flag);
    ok = all_of(1, FW_EPI, ok);
    if (!ok) return false;
    tc_fence_after();
    const uint32_t t_acc = tmem_lane + (f.both ? 0 : buf * 256);
    float* mine = a.kpart + (size_t)tile * T * yb + tl;
    for (int rb = half * per; rb < T; rb += 2 * per)
        for (int sl = s0; sl <= s1; ++sl) {
            float v[16];
            acc_ld16(t_acc + sl * cols + rb * terms, S * cols, f.na, v);
            if (my == sl && tl < yb) {
                float* y = mine + (size_t)rb * yb;
                if (terms == 3) {
#pragma unroll
                    for (int j = 0; j < 5; ++j, y += yb)
                        if (rb + j < T) __stcg(y, v[3 * j] + (v[3 * j + 1] + v[3 * j + 2]));
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j, y += yb)
                        if (rb + j < T) __stcg(y, v[2 * j] + v[2 * j + 1]);
                }
            }
            __syncwarp();
        }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&s.tempty[buf]));
    bar_n(1, FW_EPI);
    if (e == 0) {
        int32_t* cnt = a.kcnt + (is_o ? 0 : a.n_cta) + tile / c;
        asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(cnt) : "memory");
        ok = grid_wait(cnt, c * (layer + 1), abort_flag);
    }
    ok = all_of(1, FW_EPI, ok);
    if (!ok) return false;
    const float* parts = a.kpart + (size_t)(tile / c * c) * T * yb + 4 * lane;
    for (int t0 = ra + w; t0 < rn; t0 += 8 * RW) {
        if (t0 != ra + w) load_hid(t0);
        float4 q[RW];
#pragma unroll
        for (int x = 0; x < RW; ++x) q[x] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in) {
            const float* p = parts + (size_t)t0 * yb;
            int sl = 0;
#pragma unroll 4
            for (int k = 0; k < c * S; ++k) {
#pragma unroll
                for (int x = 0; x < RW; ++x) {
                    if (t0 + 8 * x >= rn) continue;
                    const float4 z = __ldcg(reinterpret_cast<const float4*>(p + (size_t)(8 * x) * yb));
                    q[x].x += z.x; q[x].y += z.y; q[x].z += z.z; q[x].w += z.w;
                }
                if (++sl == S) { sl = 0; p += (size_t)T * yb - (S - 1) * hr; }
                else p += hr;
            }
        }
#pragma unroll
        for (int x = 0; x < RW; ++x) {
            const int t = t0 + 8 * x;
            if (t >= rn) continue;                         // (the whole warp)
            float ss = 0.f;
            if (in) {
                const float4 y = make_float4(q[x].x + hid[x].x, q[x].y + hid[x].y, q[x].z + hid[x].z, q[x].w + hid[x].w);
                *reinterpret_cast<float4*>(a.hidden + (size_t)t * a.d + n) = y;
                store_terms4(make_float4(y.x * g[0], y.y * g[1], y.z * g[2], y.w * g[3]), a.x_d + (size_t)t * terms * a.d + n, a.d, terms);
                ss = (y.x * y.x + y.y * y.y) + (y.z * y.z + y.w * y.w);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            if (lane == 0) (is_o ? a.sumsq_b : a.sumsq_a)[(size_t)(tile / c) * TC_X_ROWS + t] = ss;
        }
    }
    return true;
}

// QKV where c blocks share the k-range of a tile of two heads (128 rows each): the same exchange, then a warp per row, four
// rotary pairs of a head a lane.
template <int HD>
__device__ __forceinline__ bool split_qkv(const FwArgs& a, FwTail& s, const FwPhase& f, int layer, int tcount, int e,
                                          uint32_t tmem_lane, int tile) {
    volatile int* abort_flag = s.abort_flag;
    constexpr int hp = HD / 2;
    const int lane = e & 31, w = e >> 5, quad = w & 3, half = w >> 2;
    const int T = a.T, terms = a.terms, cols = a.cols, c = f.c, buf = tcount & 1, per = terms == 3 ? 5 : 8;
    const int kp = tile % c, ra = T * kp / c, rn = T * (kp + 1) / c;
    bool ok = true;
    if (e == 0) ok = mbar_wait(smem_u32(&s.tfull[buf]), (uint32_t)(tcount >> 1) & 1u, abort_flag);
    ok = all_of(1, FW_EPI, ok);
    if (!ok) return false;
    tc_fence_after();
    const uint32_t t_acc = tmem_lane + (f.both ? 0 : buf * 256) + half * cols;     // the two warps of a quadrant: a head each
    float* y = a.kpart + (size_t)tile * T * 256 + half * 128 + quad * 32 + lane;
    for (int rb = 0; rb < T; rb += per) {
        float v[16];
        acc_ld16(t_acc + rb * terms, 2 * cols, f.na, v);
        if (terms == 3) {
#pragma unroll
            for (int j = 0; j < 5; ++j, y += 256)
                if (rb + j < T) __stcg(y, v[3 * j] + (v[3 * j + 1] + v[3 * j + 2]));
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j, y += 256)
                if (rb + j < T) __stcg(y, v[2 * j] + v[2 * j + 1]);
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&s.tempty[buf]));
    bar_n(1, FW_EPI);
    if (e == 0) {
        int32_t* cnt = a.kcnt + 2 * a.n_cta + tile / c;
        asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(cnt) : "memory");
        ok = grid_wait(cnt, c * (layer + 1), abort_flag);
    }
    ok = all_of(1, FW_EPI, ok);
    if (!ok) return false;
    const int box = lane >> 4, j = (lane & 15) * 4, hg = tile / c * 2 + box, heads = a.Hq + 2 * a.Hkv;
    const bool rot = hg < a.Hq + a.Hkv;
    const float scale = rsqrtf((float)HD) * 1.4426950408889634f;
    const float* parts = a.kpart + (size_t)(tile / c * c) * T * 256 + box * 128 + j;
#pragma unroll 2
    for (int t = ra + w; t < rn; t += 8) {
        const int sl = s.slot[t];
        if (j >= hp || hg >= heads || sl < 0) continue;
        float va[4] = {0.f, 0.f, 0.f, 0.f}, vb[4] = {0.f, 0.f, 0.f, 0.f}, cs[8];
        const float* rp = a.rope + ((size_t)t * hp + j) * 2;
        *reinterpret_cast<float4*>(cs) = *reinterpret_cast<const float4*>(rp);
        *reinterpret_cast<float4*>(cs + 4) = *reinterpret_cast<const float4*>(rp + 4);
#pragma unroll 4
        for (int k = 0; k < c; ++k) {
            const float* p = parts + ((size_t)k * T + t) * 256;
            const float4 x = __ldcg(reinterpret_cast<const float4*>(p)), z = __ldcg(reinterpret_cast<const float4*>(p + hp));
            va[0] += x.x; va[1] += x.y; va[2] += x.z; va[3] += x.w;
            vb[0] += z.x; vb[1] += z.y; vb[2] += z.z; vb[3] += z.w;
        }
        const float rs = s.rstd[t];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const float ya = va[x] * rs, yb = vb[x] * rs;
            va[x] = rot ? ya * cs[2 * x] - yb * cs[2 * x + 1] : ya;
            vb[x] = rot ? yb * cs[2 * x] + ya * cs[2 * x + 1] : yb;
        }
        if (hg < a.Hq) {
            const size_t o = ((size_t)t * a.Hq + hg) * HD + j;
            split_store4(va, scale, a.q_hi + o, a.q_lo + o);
            split_store4(vb, scale, a.q_hi + o + hp, a.q_lo + o + hp);
        } else {
            const int sq = s.meta[s.rowb[t]].seq, kv = rot ? 0 : 1;
            if (sl < a.cap && (unsigned)sq < (unsigned)a.max_batch) {                  // never past the cache
                __nv_bfloat16* d = a.cache + idx_cache(layer, a.max_batch, sq, kv, a.Hkv, hg - a.Hq - kv * a.Hkv, a.cap, sl, HD) + j;
                store_bf4(va, d);
                store_bf4(vb, d + hp);
            }
        }
    }
    return true;
}

__device__ __forceinline__ int up16(int x) { return (x + 15) & ~15; }

// End of a part of a tile's k-range other than the last (two boxes, a warp of a quadrant each; one slice): the rows' sums so
// far go to the tensor-memory columns from f.stash on, and the accumulators are free.
__device__ __forceinline__ bool put_by(const FwArgs& a, FwTail& s, const FwPhase& f, int part, int tcount, int e, uint32_t tmem_lane) {
    const int lane = e & 31, half = e >> 7, T = a.T, cols = a.cols, buf = tcount & 1;
    bool ok = true;
    if (e == 0) ok = mbar_wait(smem_u32(&s.tfull[buf]), (uint32_t)(tcount >> 1) & 1u, s.abort_flag);
    ok = all_of(1, FW_EPI, ok);
    if (!ok) return false;
    tc_fence_after();
    const uint32_t at = tmem_lane + (f.both ? 0 : buf * 256) + half * cols, st = tmem_lane + f.stash + half * up16(T);
    for (int rb = 0; rb < T; rb += 16) {
        float r[16];
        if (a.terms == 3) {
            float v[48];
#pragma unroll
            for (int h = 0; h < 3; ++h) acc_ld16(at + rb * 3 + 16 * h, 2 * cols, f.na, v + 16 * h);
#pragma unroll
            for (int j = 0; j < 16; ++j) r[j] = v[3 * j] + (v[3 * j + 1] + v[3 * j + 2]);
        } else {
            float v[32];
#pragma unroll
            for (int h = 0; h < 2; ++h) acc_ld16(at + rb * 2 + 16 * h, 2 * cols, f.na, v + 16 * h);
#pragma unroll
            for (int j = 0; j < 16; ++j) r[j] = v[2 * j] + v[2 * j + 1];
        }
        if (part > 0) {
            float o[16];
            tc_ld16(st + rb, o);
#pragma unroll
            for (int j = 0; j < 16; ++j) r[j] += o[j];
        }
        tc_st16(st + rb, r);
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&s.tempty[buf]));
    return true;
}

// The epilogue group's part of one projection: row statistics, then per tile the accumulators -> Y in shared memory ->
// the fused epilogue.  KIND is a template parameter so that the phase's geometry is read straight from the launch
// parameters; index arithmetic and global loads stand ahead of the wait for the accumulator, because everything after it
// is a chain of latencies between the last weight and the next phase's first.  FEW (up to eight rows): an element per
// thread, as little code as possible (with a warp or two per scheduler, and code that runs once a phase, time goes by the
// instruction); otherwise four neighbouring features per thread.
template <int KIND, int HD, bool FEW>
__device__ __forceinline__ bool epi_phase(const FwArgs& a, FwTail& s, float* Y, int p, int layer, int& tcount, int e,
                                          uint32_t tmem_lane, int cta, int kind) {
    const FwPhase& f = a.ph[KIND == FW_O ? kind : KIND];               // (O and down are one instance)
    const bool is_o = kind == FW_O;
    if (cta >= f.n_tiles) return true;
    volatile int* abort_flag = s.abort_flag;
    constexpr int V = FEW ? 1 : 4;                         // features per item
    const int lane = e & 31, w = e >> 5, quad = w & 3, half = w >> 2;
    const int T = a.T, terms = FEW ? 3 : a.terms, cols = a.cols, n_cta = a.n_cta;
    const int hr = f.hr, S = f.S, nbox = f.nbox, na = f.na, acc_stride = nbox * S * cols;
    const int yb = S * hr, ys = nbox * yb + 4;             // columns of Y that a box takes, row stride of Y
    const int nf = KIND == FW_LM ? nbox * f.h : f.h;       // features (pairs) of a tile
    const int nv = nf / V;                                 // items of a row
    const int per = terms == 3 ? 5 : (!FEW && KIND == FW_GATEUP && f.S == 1 ? 8 : 16), blk = FEW ? 8 : f.blk;      // rows of a drain load, rows that Y holds at a time
    // a lane's slice of the S k-blocks that the MMA takes side by side is tl / hr; a warp's lanes may lie in several
    const int tl = quad * 32 + lane, my = tl / hr;
    const int s0 = S > 1 ? quad * 32 / hr : 0, s1 = S > 1 ? min(S - 1, (quad * 32 + 31) / hr) : 0;
    const int it0 = e / nv, ij0 = (e - it0 * nv) * V, dt = FW_EPI / nv, dj = (FW_EPI - dt * nv) * V;    // items (row, feature)
    bool ok = true;
    if (KIND == FW_QKV || KIND == FW_GATEUP || KIND == FW_LM) {
        // scale of the deferred RMSNorm: the rows' sums of squares come from every block
        if (p > 0) {
            if (e == 0) ok = grid_wait(a.sync + p - 1, n_cta, abort_flag);
            ok = all_of(1, FW_EPI, ok);
            if (!ok) return false;
        }
        const float* sq = KIND == FW_GATEUP ? a.sumsq_b : a.sumsq_a;
        const FwPhase& from = a.ph[KIND == FW_GATEUP ? FW_O : FW_DOWN];
        const int parts = KIND != FW_GATEUP && p == 0 ? a.parts0 : (FEW ? from.n_tiles : from.n_tiles / from.c);
        if (FEW) {
            for (int r = w; r < T; r += 8) {
                float v = 0.f;
#pragma unroll 5
                for (int q = lane; q < parts; q += 32) v += __ldcg(sq + (size_t)q * TC_X_ROWS + r);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) s.rstd[r] = rsqrtf(v * a.inv_dim + a.eps);
            }
        } else {
            // A lane per row and every eighth part a warp, so that a load is whole lines and the parts' loads are in flight together.
            // (A warp per row, a lane per part, took 1 us a row: with 32 rows of a small model this ended 3 us after the
            // accumulators, twice a layer.)  Added in the order of 32 lanes and a butterfly, which is also that of few rows: no chain is
            // longer than five parts (one sum a warp lost up to 1e-6 of a row's, tests/test_gpu_row_sums.py).
            constexpr int NX = (FW_MAX_ROWS + 31) / 32, NQ = 20;             // (NQ x 8 parts: those of 148 blocks)
#pragma unroll 1
            for (int r = lane; r - lane < T; r += 32) {
                float v[4] = {0.f, 0.f, 0.f, 0.f};
                for (int q0 = w; q0 < parts; q0 += 8 * NQ) {
                    float x[NQ];
#pragma unroll
                    for (int k = 0; k < NQ; ++k) x[k] = q0 + 8 * k < parts && r < T ? __ldcg(sq + (size_t)(q0 + 8 * k) * TC_X_ROWS + r) : 0.f;
#pragma unroll
                    for (int k = 0; k < NQ; ++k) v[k % 4] += x[k];
                }
                Y[w * (32 * NX) + r] = (v[0] + v[2]) + (v[1] + v[3]);
            }
            bar_n(1, FW_EPI);
            if (e < T) {
                constexpr int q = 32 * NX;
                const float* y = Y + e;
                const float t = ((y[0] + y[4 * q]) + (y[2 * q] + y[6 * q])) + ((y[q] + y[5 * q]) + (y[3 * q] + y[7 * q]));
                s.rstd[e] = rsqrtf(t * a.inv_dim + a.eps);
            }
        }
    }
    if (!FEW && (KIND == FW_O)) {
        // the residual stream comes from other blocks where O and down are cut differently
        if (e == 0) ok = grid_wait(a.sync + p - 1, n_cta, abort_flag);
        ok = all_of(1, FW_EPI, ok);
        if (!ok) return false;
    }
    const __nv_bfloat16* gain = nullptr;
    if (KIND == FW_O) gain = is_o ? a.layers[layer].gain_ffn : a.layers[layer].gain_next;
    if (!FEW && (KIND == FW_O) && f.c > 1) {
        ok = split_residual(a, s, f, is_o, layer, tcount, e, tmem_lane, cta);
        ++tcount;
        return ok;
    }
    if constexpr (!FEW && KIND == FW_QKV && HD == 128)
        if (f.c > 1) {
            ok = split_qkv<HD>(a, s, f, layer, tcount, e, tmem_lane, cta);
            ++tcount;
            return ok;
        }
    for (int tile = cta; tile < f.n_tiles; tile += n_cta, ++tcount) {
        const int f0 = tile * nf;                          // first feature (O, down, gate / up, LM head)
        // ---- what the first items need besides the accumulator
        const int hg = KIND == FW_QKV ? tile / f.u : 0, j0 = KIND == FW_QKV ? (tile - hg * f.u) * f.h : 0;
        float cs[2 * V];                                   // QKV: cosines and sines of an item's pairs
        auto rope_load = [&](int t, int j) {
            if (t < T && j0 + j < HD / 2) {
                const float* src = a.rope + ((size_t)t * (HD / 2) + j0 + j) * 2;
                if (V == 4) {
#pragma unroll
                    for (int x = 0; x < V / 2; ++x)
                        *reinterpret_cast<float4*>(&cs[4 * x]) = *reinterpret_cast<const float4*>(src + 4 * x);
                } else {
                    *reinterpret_cast<float2*>(&cs[0]) = *reinterpret_cast<const float2*>(src);
                }
            }
        };
        float hid = 0.f, gain0 = 0.f;                      // O, down with few rows: the residual element of (row w, feature lane)
        float gum[8];                                      // LM head: the Gumbel noise of the warp's tokens, one draw per sequence
        int gum_seq = -1;
        auto lm_load = [&](int t) {
            const int sq = t / a.R;
            if (t >= T || sq == gum_seq) return;
            gum_seq = sq;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int jl = lane + 32 * i, n = f0 + jl;
                gum[i] = (jl < nf && n < a.V) ? a.uniforms[(size_t)sq * a.V + n] : 0.5f;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) gum[i] = logf(-logf(gum[i]));
        };
        if (KIND == FW_QKV) rope_load(it0, ij0);
        if (FEW && (KIND == FW_O) && lane < nf && f0 + lane < a.d) {
            gain0 = __bfloat162float(gain[f0 + lane]);
            if (w < T) hid = __ldcg(a.hidden + (size_t)w * a.d + f0 + lane);
        }
        if (KIND == FW_LM && !a.lm_plain) lm_load(w);
        if (!FEW && KIND == FW_GATEUP)
            for (int sg = 0; sg + 1 < f.segs; ++sg, ++tcount)
                if (!put_by(a, s, f, sg, tcount, e, tmem_lane)) return false;
        const int buf = tcount & 1;
        // (one thread polls: 256 of them would take the shared-memory pipe away from the copies' barriers)
        if (e == 0) ok = mbar_wait(smem_u32(&s.tfull[buf]), (uint32_t)(tcount >> 1) & 1u, abort_flag);
        ok = all_of(1, FW_EPI, ok);
        if (!ok) return false;
        tc_fence_after();
        const uint32_t t_acc = tmem_lane + (f.both ? 0 : buf * 256);
        if constexpr (!FEW && KIND == FW_GATEUP)
            if (f.S == 1) {
                // A thread has a feature's gate and up sums of every row in its tensor-memory lane: no way through shared memory, the
                // two warps of a quadrant take the rows in turn, eight at a time (terms three: five).
                const int n = f0 + tl;
                const bool in = tl < f.h && n < a.F;
                if (quad * 32 < f.h)
                    for (int rb = half * per; rb < T; rb += 2 * per) {
                        float v[2][16];
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            acc_ld16(t_acc + q * cols + rb * terms, acc_stride, na, v[q]);
                            if (terms == 3) {
#pragma unroll
                                for (int j = 0; j < 5; ++j) v[q][j] = v[q][3 * j] + (v[q][3 * j + 1] + v[q][3 * j + 2]);
                            } else {
#pragma unroll
                                for (int j = 0; j < 8; ++j) v[q][j] = v[q][2 * j] + v[q][2 * j + 1];
                            }
                            if (f.segs > 1) {
                                float o[8];
                                tc_ld8(tmem_lane + f.stash + q * up16(T) + rb, o);
#pragma unroll
                                for (int j = 0; j < 8; ++j) v[q][j] += o[j];
                            }
                        }
                        __nv_bfloat16* o = a.x_f + (size_t)rb * terms * a.F + n;
#pragma unroll
                        for (int j = 0; j < 8; ++j, o += (size_t)terms * a.F) {
                            if (j >= per || rb + j >= T) break;
                            const float rs = s.rstd[rb + j], gx = v[0][j] * rs;
                            if (in) store_terms(gx / (1.f + expf(-gx)) * (v[1][j] * rs), o, a.F, terms);
                        }
                        __syncwarp();
                    }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s.tempty[buf]));
                continue;
            }
        for (int r0 = 0; r0 < T; r0 += blk) {
            const int r1 = min(T, r0 + blk), nr = r1 - r0;
            // ---- accumulators -> Y[row][box][lane], the terms of a row added up
            int b = 0, rb = r0 + (nbox == 1 ? half * per : 0);
            if (nbox == 2) b = half;                       // the two warps of a quadrant share out the boxes, or the row groups
            for (; rb < r1; rb += nbox == 1 ? 2 * per : per)
                for (int sl = s0; sl <= s1; ++sl) {
                    float* y = Y + (rb - r0) * ys + b * yb + tl;
                    const bool here = my == sl && tl < yb;
                    if (FEW && s1 > s0 && na == 1) {
                        // narrow slices, several in a warp's lanes: up to four at a time, and a lane keeps its own
                        const uint32_t at = t_acc + b * S * cols + rb * 3;
                        float v[4][16];
                        for (int q0 = s0; q0 <= s1; q0 += 4) {
                            auto col = [&](int q) { return at + min(q0 + q, s1) * cols; };
                            tc_ld16x4(col(0), col(1), col(2), col(3), v);
                            const int q = my - q0;
                            if (q >= 0 && q < 4 && tl < yb)
#pragma unroll
                                for (int j = 0; j < 5; ++j) {
                                    float o = 0.f;
#pragma unroll
                                    for (int i = 0; i < 4; ++i)
                                        if (i == q) o = v[i][3 * j] + (v[i][3 * j + 1] + v[i][3 * j + 2]);
                                    if (rb + j < r1) y[j * ys] = o;
                                }
                        }
                        break;
                    }
                    if (FEW || terms == 3) {
                        float v[16];
                        acc_ld16(t_acc + (b * S + sl) * cols + rb * 3, acc_stride, na, v);
#pragma unroll
                        for (int j = 0; j < 5; ++j) v[j] = v[3 * j] + (v[3 * j + 1] + v[3 * j + 2]);
                        if (here)
#pragma unroll
                            for (int j = 0; j < 5; ++j)
                                if (rb + j < r1) y[j * ys] = v[j];
                    } else {
                        float v[32];
                        const uint32_t at = t_acc + (b * S + sl) * cols + rb * 2;
                        if (na == 1) {
                            tc_ld32(at, v);
                        } else {
                            acc_ld16(at, acc_stride, na, v);
                            acc_ld16(at + 16, acc_stride, na, v + 16);
                        }
#pragma unroll
                        for (int j = 0; j < 16; ++j) v[j] = v[2 * j] + v[2 * j + 1];
                        if (here)
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                if (rb + j < r1) y[j * ys] = v[j];
                    }
                    __syncwarp();
                }
            if (r1 == T) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s.tempty[buf]));
            }
            bar_n(1, FW_EPI);
            // values of (row of the block, box, weight rows `row` ..): the S slices lie side by side
            auto yv1 = [&](int t, int q, int row) -> float {
                const float* y = Y + t * ys + q * yb + row;
                float v = y[0];
                if (S == 4) return (v + y[hr]) + (y[2 * hr] + y[3 * hr]);
#pragma unroll 1
                for (int sl = 1; sl < S; ++sl) v += y[sl * hr];
                return v;
            };
            auto yv = [&](int t, int q, int row, float* o) {
                if (V == 1) { o[0] = yv1(t, q, row); return; }
                const float* y = Y + t * ys + q * yb + row;
                float4 v = *reinterpret_cast<const float4*>(y);
                for (int sl = 1; sl < S; ++sl) {
                    const float4 x = *reinterpret_cast<const float4*>(y + sl * hr);
                    v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
                }
                o[0] = v.x; o[V - 3 > 0 ? 1 : 0] = v.y; o[V - 2 > 0 ? 2 % V : 0] = v.z; o[V - 1] = v.w;
            };
            if (KIND == FW_QKV) {
                constexpr int hp = HD / 2;
                const float scale = rsqrtf((float)HD) * 1.4426950408889634f;      // (the attention's softmax runs on exp2)
                int t = it0, j = ij0;
                for (int i = e; i < nr * nv; i += FW_EPI) {
                    if (FEW ? i != e : r0 > 0 && i == e) rope_load(r0 + t, j);
                    const int jj = j0 + j, tt = r0 + t;
                    int tn = t + dt, jn = j + dj;                     // the next item
                    if (jn >= nf) { jn -= nf; ++tn; }
                    float c[2 * V];
#pragma unroll
                    for (int x = 0; x < 2 * V; ++x) c[x] = cs[x];
                    if (!FEW && i + FW_EPI < nr * nv) rope_load(r0 + tn, jn);        // ahead by one round
                    const int sl = s.slot[tt];
                    if (jj < hp && sl >= 0) {                         // (no slot: an inactive row has no query and no keys)
                        const float rs = s.rstd[tt];
                        float va[V], vb[V];
                        yv(t, 0, j, va);
                        yv(t, 0, f.h + j, vb);
                        const bool rot = hg < a.Hq + a.Hkv;
#pragma unroll
                        for (int x = 0; x < V; ++x) {
                            const float ya = va[x] * rs, yb2 = vb[x] * rs;
                            va[x] = rot ? ya * c[2 * x] - yb2 * c[2 * x + 1] : ya;
                            vb[x] = rot ? yb2 * c[2 * x] + ya * c[2 * x + 1] : yb2;
                        }
                        if (hg < a.Hq) {
                            // attention operands: q * log2(e) / sqrt(hd) as bf16 hi + lo
                            const size_t o = ((size_t)tt * a.Hq + hg) * HD + jj;
                            if (V == 1) {
                                split_store(va[0] * scale, a.q_hi + o, a.q_lo + o);
                                split_store(vb[0] * scale, a.q_hi + o + hp, a.q_lo + o + hp);
                            } else {
                                split_store4(va, scale, a.q_hi + o, a.q_lo + o);
                                split_store4(vb, scale, a.q_hi + o + hp, a.q_lo + o + hp);
                            }
                        } else {
                            const int sq = s.meta[s.rowb[tt]].seq, kv = rot ? 0 : 1;
                            if (sl < a.cap && (unsigned)sq < (unsigned)a.max_batch) {   // never past the cache
                                __nv_bfloat16* d = a.cache + idx_cache(layer, a.max_batch, sq, kv, a.Hkv, hg - a.Hq - kv * a.Hkv,
                                                                       a.cap, sl, HD) + jj;
                                if (V == 1) {
                                    d[0] = __float2bfloat16_rn(va[0]);
                                    d[hp] = __float2bfloat16_rn(vb[0]);
                                } else {
                                    store_bf4(va, d);
                                    store_bf4(vb, d + hp);
                                }
                            }
                        }
                    }
                    t = tn; j = jn;
                }
            } else if (KIND == FW_GATEUP) {
                int t = it0, j = ij0;
#pragma unroll(FEW ? 1 : 2)
                for (int i = e; i < nr * nv; i += FW_EPI) {
                    const int n = f0 + j;
                    if (n < a.F) {
                        const float rs = s.rstd[r0 + t];
                        float g[V], u[V];
                        yv(t, 0, j, g);
                        yv(t, 1, j, u);
#pragma unroll
                        for (int x = 0; x < V; ++x) {
                            const float gx = g[x] * rs;
                            g[x] = gx / (1.f + expf(-gx)) * (u[x] * rs);
                        }
                        __nv_bfloat16* o = a.x_f + (size_t)(r0 + t) * terms * a.F + n;
                        if (V == 1) store_terms(g[0], o, a.F, terms);
                        else store_terms4(make_float4(g[0], g[1 % V], g[2 % V], g[3 % V]), o, a.F, terms);
                    }
                    t += dt; j += dj;
                    if (j >= nf) { j -= nf; ++t; }
                }
            } else if (KIND == FW_LM) {
                if (a.lm_plain) {
                    int t = it0, j = ij0;
#pragma unroll(FEW ? 1 : 2)
                    for (int i = e; i < nr * nv; i += FW_EPI) {
                        const int q = j >= f.h ? 1 : 0, n = f0 + j;
                        float z[V];
                        yv(t, q, j - q * f.h, z);
                        const float rs = s.rstd[r0 + t];
                        float* o = a.logits + (size_t)(r0 + t) * a.V + n;
                        if (V == 4 && (a.V & 3) == 0) {
                            if (n < a.V) *reinterpret_cast<float4*>(o) = make_float4(z[0] * rs, z[1 % V] * rs, z[2 % V] * rs, z[3 % V] * rs);
                        } else {
#pragma unroll
                            for (int x = 0; x < V; ++x)
                                if (n + x < a.V) o[x] = z[x] * rs;
                        }
                        t += dt; j += dj;
                        if (j >= nf) { j -= nf; ++t; }
                    }
                } else {
                    // a warp per row: maximum, sum of exponentials, arg-max of the perturbed logits over the tile
                    for (int t = r0 + w; t < r1; t += 8) {
                        float z[8], m = -CUDART_INF_F, bv = -CUDART_INF_F, sum = 0.f;
                        int bi = 0x7fffffff;
                        const float rs = s.rstd[t];
                        if (t != w) lm_load(t);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int jl = lane + 32 * i, n = f0 + jl, q = jl >= f.h ? 1 : 0;
                            const bool in = jl < nf && n < a.V;
                            z[i] = in ? yv1(t - r0, q, jl - q * f.h) * rs : -CUDART_INF_F;
                            m = fmaxf(m, z[i]);
                            const float pz = in ? z[i] - gum[i] : -CUDART_INF_F;
                            if (in && (pz > bv || (pz == bv && n < bi))) { bv = pz; bi = n; }
                        }
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) {
                            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                            const float v2 = __shfl_xor_sync(0xffffffffu, bv, o);
                            const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
                            if (v2 > bv || (v2 == bv && i2 < bi)) { bv = v2; bi = i2; }
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i) sum += z[i] == -CUDART_INF_F ? 0.f : expf(z[i] - m);
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                        if (lane == 0) a.lm_part[idx_lm_part(t, f.n_tiles, tile)] = make_float4(m, sum, bv, __int_as_float(bi));
                    }
                    // logit of each node's token under its parent row, where it falls into this tile
                    for (int t = e; t < T; t += FW_EPI) {
                        const int pr = a.rm.prow[t];
                        if (pr < r0 || pr >= r1) continue;
                        const int tk = a.rm.tok[t] - f0, q = tk >= f.h ? 1 : 0;
                        if (tk >= 0 && tk < nf) a.node_z[t] = yv1(pr - r0, q, tk - q * f.h) * s.rstd[pr];
                    }
                }
            } else if (FEW) {
                // residual, a warp per row: emits the next operand rows and the row's share of its sum of squares
                if (w < T) {
                    float ss = 0.f;
                    for (int jl = lane; jl < nf && f0 + jl < a.d; jl += 32) {
                        const int n = f0 + jl;
                        if (jl != lane) { hid = __ldcg(a.hidden + (size_t)w * a.d + n); gain0 = __bfloat162float(gain[n]); }
                        const float y = yv1(w, 0, jl) + hid;
                        a.hidden[(size_t)w * a.d + n] = y;
                        store_terms(y * gain0, a.x_d + (size_t)w * 3 * a.d + n, a.d, 3);
                        ss += y * y;
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                    if (lane == 0) (is_o ? a.sumsq_b : a.sumsq_a)[(size_t)tile * TC_X_ROWS + w] = ss;
                }
            } else {
                // residual, four features per item; the items' sums of squares meet in Y (each over its own first element)
                int t = it0, j = ij0;
#pragma unroll 2
                for (int i = e; i < nr * nv; i += FW_EPI) {
                    const int n = f0 + j;
                    float ss = 0.f;
                    if (n < a.d) {
                        float4* hp = reinterpret_cast<float4*>(a.hidden + (size_t)(r0 + t) * a.d + n);
                        float4 y = __ldcg(hp);
                        float g[4], v[V];
#pragma unroll
                        for (int x = 0; x < 4; ++x) g[x] = __bfloat162float(gain[n + x]);
                        yv(t, 0, j, v);
                        y.x += v[0]; y.y += v[1 % V]; y.z += v[2 % V]; y.w += v[3 % V];
                        *hp = y;
                        store_terms4(make_float4(y.x * g[0], y.y * g[1], y.z * g[2], y.w * g[3]),
                                     a.x_d + (size_t)(r0 + t) * terms * a.d + n, a.d, terms);
                        ss = (y.x * y.x + y.y * y.y) + (y.z * y.z + y.w * y.w);
                    }
                    Y[t * ys + j] = ss;
                    t += dt; j += dj;
                    if (j >= nf) { j -= nf; ++t; }
                }
                bar_n(1, FW_EPI);
                for (int tr = w; tr < nr; tr += 8) {
                    float ss = lane < nv ? Y[tr * ys + lane * V] : 0.f;       // (nv <= 32: at most 128 features)
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                    if (lane == 0) (is_o ? a.sumsq_b : a.sumsq_a)[(size_t)tile * TC_X_ROWS + r0 + tr] = ss;
                }
            }
            if (r1 < T || tile + n_cta < f.n_tiles) bar_n(1, FW_EPI);       // Y is rewritten by the next rows or tile
        }
    }
    return true;
}

__device__ __forceinline__ float exp2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Sums over the 32 lanes of N values in about 2 N instructions instead of 10 N: at each step a lane passes on half of its
// values and keeps the other half.  Leaves one sum in v[0] and returns which (N: none; several lanes may hold the same).
template <int N>
__device__ __forceinline__ int lane_sums(float* v, int lane) {
    int n = N, idx = 0, have = N;
#pragma unroll
    for (int bit = 16; bit > 0; bit >>= 1) {
        if (n > 1) {
            const int h = (n + 1) / 2;                     // the lanes with this bit keep the upper half of the values
            const bool up = lane & bit;
#pragma unroll
            for (int k = 0; k < (N + 1) / 2; ++k)
                if (k < h) {
                    const float hiv = h + k < n ? v[h + k] : 0.f;
                    const float mine = up ? hiv : v[k], other = up ? v[k] : hiv;
                    v[k] = mine + __shfl_xor_sync(0xffffffffu, other, bit);
                }
            idx += up ? h : 0;
            have = up ? have - h : min(have, h);
            n = h;
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], bit);
        }
    }
    return have > 0 ? idx : N;
}

// Merge of rows [ra, rn) of a (sequence, KV head, query block)'s pieces by the epilogue threads: four output elements of NI rows
// a thread, the pieces in order (deterministic) and NP at a time, so that their loads are in flight together.
template <int HD, int NQP, int NP, int NI>
__device__ __forceinline__ void merge_rows(const FwArgs& a, const FwTail& s, const AttnPos& q, int n_piece, int G, int e, int kp) {
    const int nqb = NQP > FW_QROWS ? a.nqb : 1, g = q.g / nqb, r0 = (q.g - g * nqb) * a.qrows;
    const int nrows = s.meta[q.bi].nrows, n_q = max(0, min(G * nrows - r0, a.qrows));
    const int ra = kp < 0 ? 0 : n_q * kp / n_piece, rn = kp < 0 ? n_q : n_q * (kp + 1) / n_piece;
    constexpr int DR = FW_EPI / (HD / 4);              // rows that the group takes at a time
    const int c4 = e % (HD / 4);
    for (int rr = ra + e / (HD / 4); rr < rn; rr += DR * NI) {
        const size_t o = ((size_t)(q.bi * a.Hkv + g) * G * a.R + r0) * a.pieces;
        const float2* ml = reinterpret_cast<const float2*>(a.part + (size_t)a.T * a.Hq * a.pieces * HD) + o;
        const float4* po = reinterpret_cast<const float4*>(a.part + o * HD) + c4;
        float M[NI], ls[NI];
        float4 o4[NI];
#pragma unroll
        for (int x = 0; x < NI; ++x) { M[x] = -CUDART_INF_F; ls[x] = 0.f; o4[x] = make_float4(0.f, 0.f, 0.f, 0.f); }
        for (int k0 = 0; k0 < n_piece; k0 += NP) {
            float2 v[NI][NP];
            float4 y[NI][NP];
#pragma unroll
            for (int x = 0; x < NI; ++x)
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                    const int i = min(rr + DR * x, rn - 1) * a.pieces + min(k0 + k, n_piece - 1);
                    v[x][k] = __ldcg(ml + i);
                    y[x][k] = __ldcg(po + (size_t)i * (HD / 4));
                    if (k0 + k >= n_piece) v[x][k].x = -CUDART_INF_F;
                }
#pragma unroll
            for (int x = 0; x < NI; ++x) {
                float mn = M[x];
#pragma unroll
                for (int k = 0; k < NP; ++k) mn = fmaxf(mn, v[x][k].x);
                const float mz = mn == -CUDART_INF_F ? 0.f : mn;
                const float fo = exp2f(M[x] - mz);
                ls[x] *= fo;
                o4[x].x *= fo; o4[x].y *= fo; o4[x].z *= fo; o4[x].w *= fo;
                M[x] = mn;
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                    const float wg = exp2f(v[x][k].x - mz);
                    if (wg != 0.f) {                   // (a piece without a visible key wrote no sum worth multiplying)
                        ls[x] += wg * v[x][k].y;
                        o4[x].x += wg * y[x][k].x; o4[x].y += wg * y[x][k].y; o4[x].z += wg * y[x][k].z; o4[x].w += wg * y[x][k].w;
                    }
                }
            }
        }
#pragma unroll
        for (int x = 0; x < NI; ++x) {
            if (rr + DR * x >= rn) continue;
            const int r = r0 + rr + DR * x, hq = G == 1 ? 0 : r / nrows, t = q.bi * a.R + r - hq * nrows, h = g * G + hq;
            const float f = 1.f / ls[x];
            store_terms4(make_float4(o4[x].x * f, o4[x].y * f, o4[x].z * f, o4[x].w * f),
                         a.x_a + (size_t)t * a.terms * a.Hq * HD + (size_t)h * HD + c4 * 4, (size_t)a.Hq * HD, a.terms);
        }
    }
}
// Wide items have many rows in few pieces: of two, a thread's rows are fetched side by side.  Pieces six at a time -> two of three rows,
// us of eight layers: two pieces 675 -> 669, 852 -> 833, 742 -> 732, 937 -> 925 (7B, 65 rows 4755 -> 4705); four to eight pieces 451 -> 459,
// 505 -> 516, 701 -> 714.
template <int HD, int NQP>
__device__ __forceinline__ void merge_pieces(const FwArgs& a, const FwTail& s, const AttnPos& q, int n_piece, int G, int e, int kp) {
    if (NQP > FW_QROWS && n_piece <= 2) merge_rows<HD, NQP, 2, 3>(a, s, q, n_piece, G, e, kp);
    else merge_rows<HD, NQP, 6, 1>(a, s, q, n_piece, G, e, kp);
}

template <int HD, int NQP, bool FEW, int NS>
__global__ void __launch_bounds__(FW_THREADS, 1) forward_kernel(const __grid_constant__ FwArgs a) {
    constexpr int NCH = HD / 64;                       // 64-element chunks of a head row
    constexpr int NQ2 = 2 * NQP;                       // query rows as hi and lo parts
    constexpr uint32_t KV_BYTES = FW_KEYS * HD * 2;
    constexpr int Q_BYTES = NQ2 * HD * 2;              // one query tile
    // Probabilities as three terms, exactly.  Two leave 2^-18 of each, and with one reference value for all keys of a tile even
    // the largest is not exact (mma.sync warps had a maximum for every 16 or 64 keys, whose probability is 1): 400 keys of a
    // 64-wide head 2.85e-6 of the output off, 2.45 with mma.sync, 1.40 with three terms.  Costs about 3 us a layer of 65 rows at 7B width (the step
    // 4830 -> 4930 us), below 1 % of a step of five.
    constexpr int NP3 = 3 * NQP;
    constexpr int P_N = (NP3 + 15) / 16 * 16;          // N of the output MMA: may read up to eight rows past the tile
    constexpr int P_BYTES = NP3 * FW_KEYS * 2;         // one probability tile
    constexpr int FW_SLOT = FW_RING / NS;
    // From nine query rows on the tiles outgrow the union, and the probabilities lie in the ring, behind the K and V tiles, which
    // do not fill their slots: behind V; wide (up to 40 query rows; one query tile instead of two) and with four slots the second
    // 64 keys behind K.  That space is a tile's own: an item that fills its slot (a step of a projection) came before the
    // attention, or comes after the output has been formed (PBK: so the last two K tiles are released only then).
    constexpr bool PRING = NQP > 8, WIDE = NQP > FW_QROWS, PBK = WIDE && NS == 4;
    static_assert(!PRING || (int)KV_BYTES + P_BYTES / (PBK ? 2 : 1) + (P_N - NP3) * 128 <= FW_SLOT, "probabilities in the ring");
    static_assert((WIDE ? Q_BYTES + (int)sizeof(FwAttn<NQP / 2>) : 2 * Q_BYTES + (PRING ? 0 : 2 * P_BYTES + (P_N - NP3) * 128)) <= FW_UNION,
                  "query rows and probabilities");
    constexpr int TM = WIDE ? 128 : 64;                // attention: tensor-memory columns 0 / TM scores, 2 TM / 3 TM outputs
    static_assert(P_N <= TM, "output columns");
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* uni = smem + FW_RING;
    FwTail& s = *reinterpret_cast<FwTail*>(uni + FW_UNION);
    float* Y = reinterpret_cast<float*>(uni);
    uint8_t* Qs = uni;                                 // [2][Q_BYTES], wide: [Q_BYTES]
    uint8_t* Ps = uni + 2 * Q_BYTES;                   // [2][P_BYTES]
    const int nqb = WIDE ? a.nqb : 1, heads = a.Hkv * nqb;           // attention: (KV head, query block)s of a sequence
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int cta = (int)blockIdx.x, n_cta = a.n_cta;
    const int T = a.T, cols = a.cols, terms = FEW ? 3 : a.terms;
    const int n_phases = 5 * a.n_layers + 1;
    auto slot_ptr = [&](int pos) { return smem_u32(smem) + (uint32_t)(pos % NS) * FW_SLOT; };
    auto full_bar = [&](int pos) { return smem_u32(&s.full[pos % NS]); };
    auto empty_bar = [&](int pos) { return smem_u32(&s.empty[pos % NS]); };
    auto ring_par = [&](int pos) { return (uint32_t)(pos / NS) & 1u; };
    int n_pre = 0;                                     // (thread 0)
    if (threadIdx.x == 0) {
        for (int i = 0; i < NS; ++i) {
            mbar_init(smem_u32(&s.full[i]), 1);
            mbar_init(smem_u32(&s.empty[i]), 2);       // both MMA warps
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&s.tfull[i]), 2);
            mbar_init(smem_u32(&s.tempty[i]), 8);
            mbar_init(smem_u32(&s.sfull[i]), 1);
            mbar_init(smem_u32(&s.pfull[i]), 8);
            mbar_init(smem_u32(&s.ofull[i]), 1);
            mbar_init(smem_u32(&s.qfull[i]), 8);
        }
        s.abort_flag[0] = 0;
        s.abort_flag[1] = (int)(a.wait_limit ? a.wait_limit : WAIT_LIMIT);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        // The first projection's weights wait for nothing: as many steps as the ring holds are asked for before the rest of the
        // block's set-up, which takes 2 us.
        if (a.p_lo % 5 == FW_QKV && a.p_lo < 5 * a.n_layers && cta < a.ph[FW_QKV].n_tiles) {
            const FwPhase& f = a.ph[FW_QKV];
            const TileSrc src = tile_src(a, FW_QKV, a.p_lo / 5, cta);
            const int k0 = k_first(f, cta);
            n_pre = min(NS, k_end(f, cta) - k0);
            for (int i = 0; i < n_pre; ++i) copy_step(a, FW_QKV, src, k0 + i, slot_ptr(i), full_bar(i));
        }
    }
    for (int b = (int)threadIdx.x - 32; b >= 0 && b < a.B; b += FW_THREADS - 32) {         // (not the warp that issues copies)
        SeqMeta m;
        m.nrows = __ldcg(a.rm.n_rows + b);
        m.L = __ldcg(a.rm.kv_base + b);
        m.nkeys = min(m.L + __ldcg(a.rm.n_spec + b), a.pieces * FW_KEYS);
        m.seq = __ldcg(a.rm.call_seq + b);
        s.meta[b] = m;
    }
    for (int t = (int)threadIdx.x - 32; t >= 0 && t < min(T, FW_MAX_ROWS); t += FW_THREADS - 32) {     // (more rows: the attention alone)
        s.slot[t] = __ldcg(a.rm.slot + t);
        s.rowb[t] = (uint8_t)(t / a.R);
    }
    if (warp == 3) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s.tmem_ptr)), "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s.tmem_ptr;
    volatile int* abort_flag = s.abort_flag;
    int a_tot = 0;
    for (int b = 0; b < a.B; ++b) a_tot += attn_tiles(s.meta[b]) * heads;
    // This block's items in the order it takes them: if its range holds more than one segment (run of tiles of one sequence
    // and KV head), the first segment comes last, because it ends with the tile that holds the call's own rows and cannot
    // be requested before the phase has been released.  a_wrap: where the order returns to the front of the range.
    const AttnPos &a_zero = s.apos[0], &a_last = s.apos[1], &a_first = s.apos[2];
    if (warp == 1) {
        // Dealt out evenly, a block's tiles may be of two (sequence, KV head)s or more, and the end of each (sums over the keys,
        // output to global memory, the next one's first scores) costs as much as a few tiles: pieces that keep to one are
        // taken where they are at most two tiles longer, a lane per length tried.  7B chain, 32 heads of 17 tiles, one tile longer:
        // a step 2954 -> 2894 us; 65-row tree 4794 -> 4705.  Eight layers of width 1024, runs -> pieces one tile longer: heads of 64
        // 315 -> 304 us, wide items 526 -> 505, heads of 128 442 -> 433, wide 762 -> 732; two longer 485 -> 484, 854 -> 833, 557 -> 558,
        // 953 -> 925; four longer (with a bound of five) 560 -> 570, 994 -> 1003, 659 -> 669, 1103 -> 1117.
        int per = max(1, (a_tot + n_cta - 1) / n_cta), lo = min(cta * per, a_tot), n = min(lo + per, a_tot) - lo, lo2 = 0, n2 = 0;
        const bool fits = lane < 3 && a_tot > 0 && attn_cut(s.meta, a.B, heads, per + lane, cta, lo2, n2) <= n_cta;
        const uint32_t can = __ballot_sync(0xffffffffu, fits);
        if (can) {
            const int t = __ffs(can) - 1;
            per += t;
            lo = __shfl_sync(0xffffffffu, lo2, t);
            n = __shfl_sync(0xffffffffu, n2, t);
        }
        if (lane == 0) { s.arange[0] = n; s.arange[1] = per; s.arange[2] = can != 0; }
        if (lane < 2) s.apos[lane] = attn_find(s.meta, a.B, heads, lane == 0 ? lo : max(lo, lo + n - 1));
        __syncwarp();
        if (lane == 0) {
            const int rest = s.apos[0].nt - s.apos[0].tile;
            s.apos[2] = rest < n ? attn_find(s.meta, a.B, heads, lo + rest) : s.apos[0];
        }
    }
    __syncthreads();
    const int a_n = s.arange[0], a_per = s.arange[1];
    const bool a_cut = s.arange[2] != 0;
    const int a_rot = a_zero.nt - a_zero.tile < a_n ? a_zero.nt - a_zero.tile : 0, a_wrap = a_n - a_rot;
    auto attn_step = [&](AttnPos& it, int next) {          // item `next` of the order, from the one before
        if (next == a_wrap) it = a_zero;
        else attn_next(it, s.meta, a.B, heads);
    };
    // kind of phase p
    auto kind_of = [&](int p) { return p == n_phases - 1 ? (int)FW_LM : p % 5; };

    if (warp == 0) {
        // ---------------- weight and K / V producer: walks all phases; only the K / V tiles that hold this call's own
        // rows wait for the phase that writes them
        if (lane == 0) {
            int pos = 0;
            bool ok = true;
            for (int p = a.p_lo; p < a.p_hi && ok; ++p) {
                const int kind = kind_of(p), layer = p / 5;
                if (kind == FW_ATTN) {
                    bool waited = p == a.p_lo;
                    AttnPos it = a_first;
                    for (int i = 0; i < a_n && ok; attn_step(it, ++i)) {
                        const SeqMeta sm = s.meta[it.bi];
                        const int plane = ((layer * a.max_batch + sm.seq) * 2) * a.Hkv + it.g / nqb;
                        if (!waited && (it.tile + 1) * FW_KEYS > sm.L) {
                            ok = grid_wait(a.sync + p - 1, n_cta, abort_flag);
                            proxy_fence();
                            waited = true;
                        }
                        for (int kv = 0; kv < 2 && ok; ++kv, ++pos) {
                            ok = mbar_wait(empty_bar(pos), ring_par(pos) ^ 1u, abort_flag);
                            if (!ok) break;
                            const uint32_t bar = full_bar(pos), dst = slot_ptr(pos);
                            mbar_expect_tx(bar, KV_BYTES);
                            if (a.debug_no_operands == 2) continue;
#pragma unroll
                            for (int c = 0; c < NCH; ++c)
#pragma unroll
                                for (int k = 0; k < FW_KEYS / 64; ++k)
                                    tma_load_3d(dst + c * (FW_KEYS * 128) + k * 8192, &a.kv, bar, c * 64,
                                                it.tile * FW_KEYS + k * 64, plane + kv * a.Hkv, HINT_STREAM);
                        }
                    }
                    continue;
                }
                const FwPhase& f = a.ph[kind];
                for (int tile = cta; tile < f.n_tiles && ok; tile += n_cta) {
                    const TileSrc src = tile_src(a, kind, layer, tile);
                    const int k1 = k_end(f, tile);
                    for (int step = k_first(f, tile); step < k1; ++step, ++pos) {
                        if (pos < n_pre) continue;
                        ok = mbar_wait(empty_bar(pos), ring_par(pos) ^ 1u, abort_flag);
                        if (!ok) break;
                        copy_step(a, kind, src, step, slot_ptr(pos), full_bar(pos));
                    }
                }
            }
            if (!ok)       // give the copies in flight a bounded chance to land before the block exits
                for (int j = max(0, pos - NS); j < pos; ++j)
                    for (uint32_t it = 0; it < (1u << 12) && !mbar_test(full_bar(j), ring_par(j)); ++it) __nanosleep(64);
        }
    } else if (warp == 1) {
        // ---------------- operand-row producer: the rows of a phase exist once every block has finished the one before
        if (lane == 0) {
            int pos = 0;
            bool ok = true;
            for (int p = a.p_lo; p < a.p_hi && ok; ++p) {
                const int kind = kind_of(p);
                if (kind == FW_ATTN) { pos += 2 * a_n; continue; }
                const FwPhase& f = a.ph[kind];
                const CUtensorMap* m = &a.x[kind];
                if (p > a.p_lo) {
                    ok = grid_wait(a.sync + p - 1, n_cta, abort_flag);
                    proxy_fence();
                }
                for (int tile = cta; tile < f.n_tiles && ok; tile += n_cta) {
                    const int k1 = k_end(f, tile);
                    for (int step = k_first(f, tile); step < k1; ++step, ++pos) {
                        ok = mbar_wait(empty_bar(pos), ring_par(pos) ^ 1u, abort_flag);
                        if (!ok) break;
                        const uint32_t bar = full_bar(pos), base = slot_ptr(pos) + f.b_off;
                        if (a.debug_no_operands != 1)
                            tma_load_3d(base, m, bar, f.flat ? step * TC_TILE_K : 0, 0, f.flat ? 0 : step * f.kb, HINT_KEEP);
                    }
                }
            }
        }
    } else if (warp < FW_EPI_WARP0) {
        // ---------------- MMA issuers, warps 2 and 3 (the whole warp runs the loop, see tc_mma_one).  In a projection they
        // share out the boxes, or (one box, room for two accumulators) the MMAs along k; in the attention warp 2 forms the
        // scores and warp 3 the outputs.  Every slot of the ring is released by both, or twice by the one that used it.
        constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);      // bf16 x bf16 -> fp32, M = 128
        const uint32_t one = elect_one();
        const int me = warp - 2;
        int pos = 0, tcount = 0, at = 0, as = 0;       // ring position, projection tiles, attention tiles, segments so far
        bool ok = true;
        for (int p = a.p_lo; p < a.p_hi && ok; ++p) {
            const int kind = kind_of(p);
            if (kind == FW_ATTN) {
                if (me == 0) {
                    constexpr uint32_t idesc_s = IDESC | ((uint32_t)(NQ2 >> 3) << 17);
                    AttnPos it = a_first;
                    for (int i = 0; i < a_n; attn_step(it, ++i)) {
                        const bool fresh = i == 0 || i == a_wrap || it.tile == 0;
                        if (fresh && i > 0) ++as;
                        const int kpos = pos + 2 * i, b = (at + i) & 1;
                        // Query rows of the segment, the score buffer (read by the softmax two tiles ago), and the K tile.  With an
                        // odd ring the K tile's slot held the V tile of two tiles ago, whose arrival this warp has not followed:
                        // the slot's barrier may be a phase behind, and the parity would then name the phase before the one
                        // meant.  The output of that tile being complete says that the V tile has come and gone.
                        const uint32_t before = ((uint32_t)((at + i) >> 1) & 1u) ^ 1u;
                        ok = (!fresh || mbar_wait_warp(smem_u32(&s.qfull[as & 1]), (uint32_t)(as >> 1) & 1u, abort_flag)) &&
                             mbar_wait_warp(smem_u32(NS % 2 ? &s.ofull[b] : &s.pfull[b]), before, abort_flag) &&
                             mbar_wait_warp(full_bar(kpos), ring_par(kpos), abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        const uint64_t ka = smem_desc(slot_ptr(kpos)), qa = smem_desc(smem_u32(Qs) + (WIDE ? 0 : as & 1) * Q_BYTES);
#pragma unroll
                        for (int ks = 0; ks < HD / 16; ++ks)
                            tc_mma_one(one, tmem + b * TM, ka + (ks >> 2) * (FW_KEYS * 8) + (ks & 3) * 2,
                                       qa + (ks >> 2) * (NQ2 * 8) + (ks & 3) * 2, idesc_s, ks > 0 ? 1u : 0u);
                        tc_commit_one(one, smem_u32(&s.sfull[b]));
                        if (!PBK || i < a_n - 2) {
                            tc_commit_one(one, empty_bar(kpos));
                            tc_commit_one(one, empty_bar(kpos));
                        }
                    }
                    if (a_n > 0) ++as;
                    if (NS % 2 && a_n > 1 && ok) {     // (the next phase's first slot held the last V tile but one)
                        const int n = at + a_n - 2;
                        ok = mbar_wait_warp(smem_u32(&s.ofull[n & 1]), (uint32_t)(n >> 1) & 1u, abort_flag);
                    }
                } else {
                    constexpr uint32_t idesc_o = IDESC | (1u << 15) | ((uint32_t)(P_N >> 3) << 17);
                    for (int i = 0; i < a_n; ++i) {
                        const int vpos = pos + 2 * i + 1, b = (at + i) & 1;
                        const uint32_t par = (uint32_t)((at + i) >> 1) & 1u;
                        // (the probabilities' arrival also says that every epilogue warp has read the output two tiles ago)
                        ok = mbar_wait_warp(smem_u32(&s.pfull[b]), par, abort_flag) &&
                             mbar_wait_warp(full_bar(vpos), ring_par(vpos), abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        const uint64_t va = smem_desc_mn(slot_ptr(vpos)), pa = smem_desc(PRING ? slot_ptr(vpos) + KV_BYTES : smem_u32(Ps) + b * P_BYTES);
                        const uint64_t pb = PBK ? smem_desc(slot_ptr(vpos - 1) + KV_BYTES) : pa + NP3 * 8;       // keys 64 ..
#pragma unroll
                        for (int ks = 0; ks < FW_KEYS / 16; ++ks)
                            tc_mma_one(one, tmem + (2 + b) * TM, va + ks * 128, (ks < 4 ? pa : pb) + (ks & 3) * 2,
                                       idesc_o, ks > 0 ? 1u : 0u);
                        tc_commit_one(one, smem_u32(&s.ofull[b]));
                        tc_commit_one(one, empty_bar(vpos));
                        tc_commit_one(one, empty_bar(vpos));
                        if (PBK && i >= a_n - 2) {
                            tc_commit_one(one, empty_bar(vpos - 1));
                            tc_commit_one(one, empty_bar(vpos - 1));
                        }
                    }
                }
                at += a_n;
                pos += 2 * a_n;
                continue;
            }
            const FwPhase& f = a.ph[kind];
            const int groups = f.kb / f.S, sc = f.S * cols, nbox = f.nbox;      // MMAs along k, accumulator columns of a box
            const int na = f.na;
            const uint32_t idesc = IDESC | ((uint32_t)(sc >> 3) << 17);
            const uint32_t a_step = f.S * f.hr * 8, b_step = sc * 8;            // 16-byte units
            for (int tile = cta; tile < f.n_tiles && ok; tile += n_cta) {
                const int k0 = k_first(f, tile), k1 = k_end(f, tile);
                for (int sg = 0; sg < f.segs && ok; ++sg, ++tcount) {
                    const int buf = tcount & 1;
                    ok = mbar_wait_warp(smem_u32(&s.tempty[buf]), ((uint32_t)(tcount >> 1) & 1u) ^ 1u, abort_flag);
                    if (f.both && tcount > 0)          // (its accumulators take the columns of the tile before as well)
                        ok = ok && mbar_wait_warp(smem_u32(&s.tempty[buf ^ 1]), (uint32_t)((tcount - 1) >> 1) & 1u, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d0 = tmem + (f.both ? 0 : buf * 256) + (nbox == 2 ? me * sc : 0);
                    int turn = 0;                      // accumulator of the next MMA along k; one box: warp `me` forms every other one
                    uint32_t acc = 0;                  // (the first round over the accumulators begins them)
                    const int end = k0 + (k1 - k0) * (sg + 1) / f.segs;
                    for (int step = k0 + (k1 - k0) * sg / f.segs; step < end; ++step, ++pos) {
                        ok = mbar_wait_warp(full_bar(pos), ring_par(pos), abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t base = slot_ptr(pos);
                        uint64_t ad = smem_desc(base), bd = smem_desc(base + f.b_off);
                        if (nbox == 2) ad += (uint32_t)(me * f.box_bytes) >> 4;
                        for (int gr = 0; gr < groups; ++gr, ad += a_step, bd += b_step) {
                            if (nbox == 2 || (turn & 1) == me) {
                                const uint32_t d = d0 + turn * nbox * sc;
#pragma unroll
                                for (int k4 = 0; k4 < TC_TILE_K / 16; ++k4)
                                    tc_mma_one(one, d, ad + k4 * 2, bd + k4 * 2, idesc, k4 > 0 ? 1u : acc);
                            }
                            if (++turn == na) { turn = 0; acc = 1u; }
                        }
                        tc_commit_one(one, empty_bar(pos));
                    }
                    if (ok) tc_commit_one(one, smem_u32(&s.tfull[buf]));
                }
            }
        }
        if (!ok)               // gave up: the MMAs in flight end before the block frees its tensor memory and leaves
            for (int i = 0; i < 64; ++i) __nanosleep(1000);
    } else {
        // ---------------- epilogue warps
        const int e = threadIdx.x - 32 * FW_EPI_WARP0;   // 0..255
        const int quad = warp & 3, half = (warp - FW_EPI_WARP0) >> 2;     // TMEM lane quadrant; which of its two warps
        const uint32_t t_lane = tmem + ((uint32_t)(quad * 32) << 16);
        int tcount = 0, at = 0, as = 0, pos = 0;
        bool ok = true;
        auto steps_of = [&](const FwPhase& f) {
            if (cta >= f.n_tiles) return 0;
            return f.c > 1 ? k_end(f, cta) - k_first(f, cta) : ((f.n_tiles - 1 - cta) / n_cta + 1) * f.steps;
        };
        const int ring_other = steps_of(a.ph[FW_O]) + steps_of(a.ph[FW_GATEUP]) + steps_of(a.ph[FW_DOWN]);
        const int ring_qkv = steps_of(a.ph[FW_QKV]);
        for (int p = a.p_lo; p < a.p_hi && ok; ++p) {
            const int kind = kind_of(p), layer = p / 5;
            if (kind == FW_ATTN) {
                if (e == 0 && p > a.p_lo) ok = grid_wait(a.sync + p - 1, n_cta, abort_flag);
                ok = all_of(1, FW_EPI, ok);
                if (!ok) break;
                if (p > a.p_lo) pos += ring_qkv;
                const int G = a.Hq / a.Hkv, kl = quad * 32 + lane;    // this thread's key of a tile, later its head dimension
                constexpr int NR = NQP / 2;                           // this thread's query rows: half, half + 2, ...; wide:
                auto row_of = [&](int x) { return WIDE ? half * NR + x : 2 * x + half; };        // NR neighbouring ones
                auto& sa = *reinterpret_cast<FwAttn<WIDE ? NR : FW_QROWS / 2>*>(WIDE ? Qs + Q_BYTES : reinterpret_cast<uint8_t*>(&s.attn));
                // scores at column `col`: this thread's rows, hi and lo parts added up
                auto tm_rows = [&](int col, float* v) {
                    if constexpr (WIDE) {
                        tc_ld20_sum(t_lane + col + half * NR, t_lane + col + NQP + half * NR, v);
                    } else {
                        float c[NQ2];
                        if constexpr (NQ2 == 16) tc_ld16(t_lane + col, c);
                        else tc_ld32(t_lane + col, c);
#pragma unroll
                        for (int x = 0; x < NR; ++x) v[x] = half == 0 ? c[2 * x] + c[NQP + 2 * x] : c[2 * x + 1] + c[NQP + 2 * x + 1];
                    }
                };
                // the same for outputs, which have three parts
                auto tm_out = [&](int col, float* v) {
                    if constexpr (WIDE) {
                        float c[NR];
                        tc_ld20_sum(t_lane + col + NQP + half * NR, t_lane + col + 2 * NQP + half * NR, v);
                        tc_ld20(t_lane + col + half * NR, c);
#pragma unroll
                        for (int x = 0; x < NR; ++x) v[x] += c[x];
                    } else {
                        float c[NP3 > 32 ? 48 : 32];
                        if constexpr (NP3 > 32) tc_ld48(t_lane + col, c);
                        else tc_ld32(t_lane + col, c);
#pragma unroll
                        for (int x = 0; x < NR; ++x)
                            v[x] = half == 0 ? c[2 * x] + (c[NQP + 2 * x] + c[2 * NQP + 2 * x])
                                             : c[2 * x + 1] + (c[NQP + 2 * x + 1] + c[2 * NQP + 2 * x + 1]);
                    }
                };
                // query rows of a segment: KV head, first row, how many
                auto q_head = [&](const AttnPos& q) { return WIDE ? q.g / nqb : q.g; };
                auto q_base = [&](const AttnPos& q) { return WIDE ? q.g % nqb * a.qrows : 0; };
                auto q_count = [&](const AttnPos& q) { return min(G * s.meta[q.bi].nrows - q_base(q), a.qrows); };
                // query rows of (sequence, KV head) -> buffer `qb`, hi rows then lo rows, K-major
                auto load_q = [&](const AttnPos& q, int qb) {
                    const int nrows = s.meta[q.bi].nrows, n_q = q_count(q), rb = q_base(q);
                    uint8_t* dst = Qs + (WIDE ? 0 : qb) * Q_BYTES;
#pragma unroll
                    for (int idx = e; idx < NQ2 * (HD / 8); idx += FW_EPI) {
                        const int row = idx / (HD / 8), c = idx % (HD / 8), r = row >= NQP ? row - NQP : row;
                        const bool valid = r < n_q;
                        const int rr = valid ? rb + r : 0, hq = G == 1 ? 0 : rr / nrows;
                        const __nv_bfloat16* src = (row >= NQP ? a.q_lo : a.q_hi) +
                            ((size_t)(q.bi * a.R + rr - hq * nrows) * a.Hq + q_head(q) * G + hq) * HD + c * 8;
                        cp_async16(smem_u32(dst + (c >> 3) * (NQ2 * 128) + row * 128 + (((c & 7) ^ (row & 7)) << 4)), src, valid);
                    }
                    asm volatile("cp.async.commit_group;" ::: "memory");
                };
                auto q_ready = [&](int qb) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&s.qfull[qb]));
                };
                // the first two segments' query rows go out at once, a later segment's when the one two before it has ended (wide:
                // the first one's, and a later one's when the scores of the one before it have been formed)
                AttnPos ahead = a_first;
                int ahead_i = 0;
                bool more = a_n > 0;
                auto next_seg = [&]() {
                    const int n = min(ahead.nt - ahead.tile, (ahead_i < a_wrap ? a_wrap : a_n) - ahead_i);
                    ahead.tile += n - 1;
                    ahead_i += n;
                    more = ahead_i < a_n;
                    if (more) attn_step(ahead, ahead_i);
                };
                if (more) {
                    load_q(ahead, as & 1);
                    next_seg();
                    if (!WIDE && more) {
                        load_q(ahead, (as + 1) & 1);
                        asm volatile("cp.async.wait_group 1;" ::: "memory");
                        q_ready(as & 1);
                        asm volatile("cp.async.wait_group 0;" ::: "memory");
                        q_ready((as + 1) & 1);
                    } else {
                        asm volatile("cp.async.wait_group 0;" ::: "memory");
                        q_ready(as & 1);
                    }
                }
                AttnPos it = a_first;
                // (The reference values lie in shared memory too: wide, they would not fit the registers beside the rest.)
                float m[NR], l[NR], acc[NR];
                // output of the tile before: this thread's head dimension of its rows, out of tensor memory
                auto output = [&](int tile_no) {
                    const int b = tile_no & 1;
                    ok = warp_wait(smem_u32(&s.ofull[b]), (uint32_t)(tile_no >> 1) & 1u, abort_flag, ok, lane);
                    tc_fence_after();
                    float c[NR];
                    tm_out((2 + b) * TM, c);
#pragma unroll
                    for (int x = 0; x < NR; ++x) acc[x] += c[x];
                };
                // end of a segment: the rows' sums over the lanes, then the rows leave - final, or as a piece
                auto finish = [&](const AttnPos& q) {
                    const int sb = as & 1;
                    const int which = lane_sums<NR>(l, lane);
                    if (which < NR) sa.sl[sb][half][which][quad] = l[0];
                    ok = all_of(2 + half, 128, ok);
                    const int nrows = s.meta[q.bi].nrows, n_q = q_count(q), rb = q_base(q), g = q_head(q);
                    const int n_piece = attn_pieces(q, a_per, a_cut), piece = attn_piece(q, a_per, a_cut, cta);
                    auto row_sum = [&](int x) {
                        const float4 l4 = *reinterpret_cast<const float4*>(sa.sl[sb][half][x]);
                        return (l4.x + l4.y) + (l4.z + l4.w);
                    };
                    // (code that runs once a phase costs its instructions' way from L2: keep the loops over rows short)
                    if (ok && n_piece > 1) {
                        const size_t o = ((size_t)(q.bi * a.Hkv + g) * G * a.R + rb + row_of(0)) * a.pieces + piece;
                        constexpr int DR = WIDE ? 1 : 2;
                        float* po = a.part + o * HD + kl;
                        const int left = n_q - row_of(0);
                        if (HD == 128 || kl < HD)
#pragma unroll
                            for (int x = 0; x < NR; ++x, po += DR * a.pieces * HD)
                                if (DR * x < left) *po = acc[x];
                        float2* ml = reinterpret_cast<float2*>(a.part + (size_t)T * a.Hq * a.pieces * HD) + o;
                        if (WIDE) {
                            if (kl < NR && kl < left) ml[kl * a.pieces] = make_float2(sa.sm[half][kl], row_sum(kl));
                        } else if (kl == 0) {
#pragma unroll
                            for (int x = 0; x < NR; ++x)
                                if (DR * x < left) ml[DR * x * a.pieces] = make_float2(m[x], row_sum(x));
                        }
                    } else if (ok && (HD == 128 || kl < HD)) {
#pragma unroll
                        for (int x = 0; x < NR; ++x) {
                            const int r = row_of(x);
                            if (r < n_q) {
                                const int hq = G == 1 ? 0 : (rb + r) / nrows, t = q.bi * a.R + rb + r - hq * nrows, h = g * G + hq;
                                store_terms(acc[x] / row_sum(x), a.x_a + (size_t)t * terms * a.Hq * HD + (size_t)h * HD + kl,
                                            (size_t)a.Hq * HD, terms);
                            }
                        }
                    }
                    if (!WIDE && more) next_seg();
                    if (!WIDE && more) {                                  // (the scores of this segment are formed, its query buffer is free)
                        load_q(ahead, sb);
                        asm volatile("cp.async.wait_group 0;" ::: "memory");
                        q_ready(sb);
                    }
                    ++as;
                };
                int L = 0, nkeys = 0;
                for (int i = 0; a_n > 0; ++i) {
                    const bool fresh = i == 0 || i == a_wrap || i == a_n || it.tile + 1 == it.nt;     // (it: the item before)
                    if (fresh && i > 0) {
                        output(at - 1);
                        finish(it);
                    }
                    if (i == a_n) break;
                    if (i > 0) attn_step(it, i);
                    if (fresh) {
#pragma unroll
                        for (int x = 0; x < NR; ++x) { m[x] = FW_UNSEEN; l[x] = 0.f; acc[x] = 0.f; }
                    }
                    if (fresh) { L = s.meta[it.bi].L; nkeys = s.meta[it.bi].nkeys; }
                    const bool turn = WIDE && i + 1 < a_n && (i + 1 == a_wrap || it.tile + 1 == it.nt);     // the segment's last
                    const int b = at & 1;
                    const uint32_t par = (uint32_t)(at >> 1) & 1u;
                    const int j = it.tile * FW_KEYS + kl;
                    // which of this thread's rows see its key: all of a committed one; of a draft row those that have it among
                    // their ancestors and themselves; none past the last key
                    uint32_t vis = 0xffffffffu;
                    if ((it.tile + 1) * FW_KEYS > L) {
                        const int sr = j - L, nrows = s.meta[it.bi].nrows, n_q = q_count(it), rb = q_base(it);
                        const int t0 = it.bi * a.R;                   // query row r: row t0 + r % nrows, head g * G + r / nrows
                        vis = j < nkeys ? 0xffffffffu : 0u;
                        if (WIDE && sr >= 0 && vis) {
                            const uint32_t* words = a.rm.mask + (size_t)t0 * MTAD_MASK_WORDS + (sr >> 5);
                            int r = row_of(0), rr = (rb + min(r, n_q - 1)) % nrows;
                            vis = 0;
#pragma unroll
                            for (int x = 0; x < NR; ++x) {
                                vis |= ((words[rr * MTAD_MASK_WORDS] >> (sr & 31)) & 1u) << x;
                                if (++r < n_q && ++rr == nrows) rr = 0;
                            }
                        } else if (sr >= 0 && vis) {
                            vis = 0;
#pragma unroll
                            for (int x = 0; x < NR; ++x) {
                                const int r = row_of(x), rr = r < n_q ? (G == 1 ? rb + r : (rb + r) % nrows) : 0;
                                vis |= ((a.rm.mask[(size_t)(t0 + rr) * MTAD_MASK_WORDS + (sr >> 5)] >> (sr & 31)) & 1u) << x;
                            }
                        }
                    }
                    ok = warp_wait(smem_u32(&s.sfull[b]), par, abort_flag, ok, lane);
                    tc_fence_after();
                    float v[NR];
                    tm_rows(b * TM, v);
                    if (__any_sync(0xffffffffu, vis != 0xffffffffu))
#pragma unroll
                        for (int x = 0; x < NR; ++x) v[x] = ((vis >> x) & 1u) ? v[x] : -CUDART_INF_F;
                    if (turn) load_q(ahead, 0);                       // (this segment's scores are formed, the query tile is free)
                    // The reference value m of a row need not be its maximum: numerators and sums have the exponent range that
                    // fp32 and bf16 share, and a common factor costs no precision.  A segment starts with the score of its first
                    // key, and m moves to the maximum only when a score exceeds it by more than 2^64 (or no key was seen yet).
                    if (fresh) {
                        if (kl == 0)
#pragma unroll
                            for (int x = 0; x < NR; ++x) sa.sm[half][x] = fmaxf(v[x], FW_UNSEEN);
                        bar_n(2 + half, 128);
                    }
                    if (WIDE || fresh)
#pragma unroll
                        for (int x = 0; x < NR; ++x) m[x] = sa.sm[half][x];
                    float most = -CUDART_INF_F;
#pragma unroll
                    for (int x = 0; x < NR; ++x) { v[x] -= m[x]; most = fmaxf(most, v[x]); }
                    const bool quiet = all_of(2 + half, 128, most <= FW_LAZY);
                    if (!quiet) {
                        if (!fresh) output(at - 1);                   // (before the reference moves)
                        float wm[NR];
                        tm_rows(b * TM, v);
#pragma unroll
                        for (int x = 0; x < NR; ++x) wm[x] = v[x] = ((vis >> x) & 1u) ? v[x] : -CUDART_INF_F;
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                            for (int x = 0; x < NR; ++x) wm[x] = fmaxf(wm[x], __shfl_xor_sync(0xffffffffu, wm[x], o));
#pragma unroll
                        for (int x = 0; x < NR; ++x)
                            if (lane == x) sa.smx[half][x][quad] = wm[x];
                        bar_n(2 + half, 128);
#pragma unroll
                        for (int x = 0; x < NR; ++x) {
                            const float4 q4 = *reinterpret_cast<const float4*>(sa.smx[half][x]);
                            const float mn = fmaxf(m[x], fmaxf(fmaxf(q4.x, q4.y), fmaxf(q4.z, q4.w)));
                            const float f = exp2f(m[x] - mn);
                            m[x] = mn;
                            v[x] -= mn;
                            l[x] *= f;
                            acc[x] *= f;
                        }
                        if (WIDE && kl == 0)
#pragma unroll
                            for (int x = 0; x < NR; ++x) sa.sm[half][x] = m[x];
                        bar_n(2 + half, 128);                         // (smx is free again)
                    }
                    uint8_t* pt = (PRING ? smem + (size_t)((pos + 2 * i + (PBK && kl >= 64 ? 0 : 1)) % NS) * FW_SLOT + KV_BYTES : Ps + b * P_BYTES) +
                                  (PBK ? 0 : kl >> 6) * (NP3 * 128) + (kl & 7) * 2 + row_of(0) * 128;
                    constexpr int RS = WIDE ? 128 : 256;              // bytes between this thread's rows
                    const int pc = (kl & 63) >> 3;
#pragma unroll
                    for (int x = 0; x < NR; ++x) {
                        // (exp2(-inf) = 0; results below 2^-126 of a sum of at least 1, the reference being a key's score, go to 0)
                        const float pv = exp2_ftz(v[x]);
                        l[x] += pv;
                        const __nv_bfloat16 hi = __float2bfloat16_rn(pv);
                        uint8_t* d = pt + ((pc ^ (row_of(x) & 7)) << 4) + x * RS;
                        *reinterpret_cast<__nv_bfloat16*>(d) = hi;
                        const float rest = pv - __bfloat162float(hi);
                        const __nv_bfloat16 lo = __float2bfloat16_rn(rest);
                        *reinterpret_cast<__nv_bfloat16*>(d + NQP * 128) = lo;
                        *reinterpret_cast<__nv_bfloat16*>(d + 2 * NQP * 128) = __float2bfloat16_rn(rest - __bfloat162float(lo));
                    }
                    if ((it.tile + 1) * FW_KEYS > nkeys) {
                        // rows of V past the last key: their probabilities are 0, but 0 x (stale value) must not make a NaN
                        const int vpos = pos + 2 * i + 1;
                        ok = warp_wait(full_bar(vpos), ring_par(vpos), abort_flag, ok, lane);
                        if (ok && j >= nkeys) {
                            uint8_t* vs = smem + (size_t)(vpos % NS) * FW_SLOT + kl * 128 + half * 64;
#pragma unroll
                            for (int c = 0; c < NCH * 4; ++c)
                                *reinterpret_cast<uint4*>(vs + (c >> 2) * (FW_KEYS * 128) + (c & 3) * 16) = make_uint4(0u, 0u, 0u, 0u);
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    if (quiet && !fresh) output(at - 1);              // (tile i - 1 of the same segment, while this one's output is formed)
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&s.pfull[b]));
                    if (turn) {
                        asm volatile("cp.async.wait_group 0;" ::: "memory");
                        q_ready((as + 1) & 1);
                        next_seg();
                    }
                    ++at;
                }
                pos += 2 * a_n + ring_other;
                ok = all_of(1, FW_EPI, ok);
                if (!ok) break;
                // pieces shared with other blocks (at most the first and the last of this block's range): who arrives last merges
                // them; with many rows the blocks wait for one another and take a share of the rows each
                if (a_n > 0) {
                    if (e < 2) {
                        const AttnPos q = e == 0 ? a_zero : a_last;
                        const int n_piece = attn_pieces(q, a_per, a_cut);
                        int last = 0;
                        if (n_piece > 1 && (e == 0 || a_last.f0 != a_zero.f0)) {
                            int old;
                            asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;"
                                         : "=r"(old) : "l"(a.acnt + q.bi * heads + q.g) : "memory");
                            last = WIDE || old + 1 == n_piece * (layer + 1) ? n_piece : 0;
                        }
                        s.last[e] = last;
                        __syncwarp(3u);
                        if (WIDE && last) ok = grid_wait(a.acnt + q.bi * heads + q.g, n_piece * (layer + 1), abort_flag);
                    }
                    ok = all_of(1, FW_EPI, ok);
                    if (!ok) break;
                    for (int x = 0; x < 2; ++x)
                        if (s.last[x]) {
                            const AttnPos q = x == 0 ? a_zero : a_last;
                            merge_pieces<HD, NQP>(a, s, q, s.last[x], G, e, WIDE ? attn_piece(q, a_per, a_cut, cta) : -1);
                        }
                }
            } else if (kind == FW_QKV) {
                ok = epi_phase<FW_QKV, HD, FEW>(a, s, Y, p, layer, tcount, e, t_lane, cta, kind);
            } else if (kind == FW_O || kind == FW_DOWN) {
                ok = epi_phase<FW_O, HD, FEW>(a, s, Y, p, layer, tcount, e, t_lane, cta, kind);
            } else if (kind == FW_GATEUP) {
                ok = epi_phase<FW_GATEUP, HD, FEW>(a, s, Y, p, layer, tcount, e, t_lane, cta, kind);
            } else {
                ok = epi_phase<FW_LM, HD, FEW>(a, s, Y, p, layer, tcount, e, t_lane, cta, kind);
            }
            if (kind != FW_LM && ok) {
                // phase barrier: the release covers the whole group's stores (the readers' proxy fence follows their acquire)
                bar_n(1, FW_EPI);
                if (e == 0) {
                    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(a.sync + p) : "memory");
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 3) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
    if (threadIdx.x == 0 && *abort_flag && a.status)
        for (int b = 0; b < a.B; ++b) atomicOr(a.status + b, MTAD_ST_TIMEOUT);
}

int up_div(int x, int y) { return (x + y - 1) / y; }
int up8(int x) { return (x + 7) / 8 * 8; }

}  // namespace

// Ring slots: those of the class, or four where steps are few (auxiliary model of width 1024, eight sequences of four beams:
// six draft steps 1147 us with three, 1120 with four) and a step of two boxes of 128 rows fits.
static int fw_slots(const mtad_model_desc& d, int cls) {
    return d.d_model <= 2048 && (256 + FW_CLASS[cls].cols) * 128 <= FW_RING / 4 ? 4 : FW_CLASS[cls].slots;
}

// Up to eight rows the lean epilogues (an element per thread, a warp per row: beyond, a row would wait for its turn), which know
// no split projections.
static bool fw_few(int T, int query_rows) { return T <= 8 && query_rows <= FW_QROWS; }

void fw_geometry(FwPhase ph[6], const mtad_model_desc& d, int n_cta, int cls) {
    const int qd = d.n_q_heads * d.head_dim, hp = d.head_dim / 2, heads = d.n_q_heads + 2 * d.n_kv_heads;
    const int cols = FW_CLASS[cls].cols, slot = FW_RING / fw_slots(d, cls);
    for (int k = 0; k < 6; ++k) ph[k].c = ph[k].u = 1;
    // rows of a matrix: one tile per SM, in whole groups of eight rows (swizzle atoms)
    auto rows = [&](FwPhase& f, int N, int K, int nbox, int cut) {
        f.K = K;
        f.k_blocks = up_div(K, TC_TILE_K);
        f.nbox = nbox;
        f.h = f.hr = std::min(128, std::max(8, up8(up_div(N, n_cta * cut))));
        f.n_tiles = up_div(N, f.h * cut);
    };
    rows(ph[FW_O], d.d_model, qd, 1, 1);
    rows(ph[FW_DOWN], d.d_model, d.d_ffn, 1, 1);
    rows(ph[FW_GATEUP], d.d_ffn, d.d_model, 2, 1);
    const int lm_boxes = up_div(d.vocab, n_cta) > 64 ? 2 : 1;
    rows(ph[FW_LM], d.vocab, d.d_model, lm_boxes, lm_boxes);
    // O and down: a tile's k-range over c blocks where that pays.  With many operand rows the SMs' intake bounds a narrow
    // tile (every block reads all operand rows of its k-blocks, about 100 GB/s an SM from L2); c blocks on a tile c times as
    // wide read them a c-th as often, and pay about 3.5 us to exchange their partial sums.  13B, 56 rows: O and down 24 and
    // 48 us a layer unsplit, 17 and 32.5 over three blocks each.  The rates and what an exchange costs are fitted to the phases'
    // times at 7B and 13B width and 33, 56 and 65 rows; they only rank the splits.
    for (int k : {FW_O, FW_DOWN}) {
        FwPhase& f = ph[k];
        double best = 1e30;
        for (int c = 1; c <= 4; ++c) {
            const int h = std::max(8, up8(up_div(d.d_model, n_cta / c)));
            if (c > 1 && (h > 128 || f.k_blocks < 8 * c || cls < 2)) break;
            const double intake = (double)(h + cols) * 128.0 * up_div(f.k_blocks, c) / 100e3;
            const double floor_us = 2.0 * d.d_model * f.K / 6.5e6;
            const double us = std::max(intake, floor_us) + (c > 1 ? 3.5 : 0.0);
            if (us < best) {
                best = us;
                f.c = c;
                f.h = f.hr = std::min(128, h);
                f.n_tiles = up_div(d.d_model, f.h) * c;
            }
        }
    }
    // QKV: the rotary pairs of a head in u tiles, as many as the SMs allow
    FwPhase& q = ph[FW_QKV];
    q.u = std::max(1, std::min(n_cta / heads, hp / 4));
    q.h = up_div(up_div(hp, q.u), 4) * 4;
    q.u = up_div(hp, q.h);
    q.hr = 2 * q.h;
    q.nbox = 1;
    q.n_tiles = heads * q.u;
    q.K = d.d_model;
    q.k_blocks = up_div(q.K, TC_TILE_K);
    // The same split for QKV, two heads of 128 on a tile: it meets the operand rows half as often and spreads over all SMs
    // (7B, 32 heads: 96 tiles of one head leave a third of them idle), at about 4.5 us for the exchange.  7B, 65 rows: 35 ->
    // 26 us a layer; at 33 rows both ways take 24, and the unsplit one, which needs no exchange buffer, is taken unless the split
    // is estimated 2 us faster (the 2.0).  The lower rate is that of the wider boxes: 256 weight rows beside the operand rows.
    if (d.head_dim == 128 && q.u == 1 && cls >= 2) {
        const double floor_us = 2.0 * heads * 128 * q.K / 6.5e6;
        double best = std::max((128.0 + cols) * 128.0 * q.k_blocks / 85e3, floor_us) - 2.0;
        for (int c = 2; c <= 4; ++c) {
            const int tiles = up_div(heads, 2) * c;
            if (tiles > n_cta || q.k_blocks < 8 * c || (256 + cols) * 128 > slot) break;
            const double us = std::max((256.0 + cols) * 128.0 * up_div(q.k_blocks, c) / 85e3, floor_us) + 4.5;
            if (us < best) {
                best = us;
                q.c = c;
                q.nbox = 2;
                q.n_tiles = tiles;
            }
        }
    }
    for (int k = 0; k < 6; ++k) {
        if (k == FW_ATTN) continue;
        FwPhase& f = ph[k];
        int kb = slot / ((f.nbox * f.hr + cols) * 128);
        kb = std::min(std::min(kb, f.k_blocks), 16);
        // a multiple of the k-blocks that the MMA can take side by side
        const int S = std::min(TC_TILE_N / f.hr, FW_ACC / (cols * f.nbox));
        if (S > 1 && kb > S) kb -= kb % S;
        f.kb = (f.K % TC_TILE_K || kb < 1) ? 1 : kb;
        f.flat = tc_kb_flat(f.K, f.kb) ? 1 : 0;
        f.steps = up_div(f.k_blocks, f.kb);
        f.box_bytes = f.hr * 128 * f.kb;
        f.b_off = f.nbox * f.box_bytes;
    }
}

bool fw_plan(FwArgs& a, const mtad_model_desc& d, int B, int R, int n_cta) {
    const int T = B * R, G = d.n_q_heads / d.n_kv_heads;
    if (d.head_dim != 64 && d.head_dim != 128) return false;
    if (T > FW_MAX_ROWS || B > MTAD_MAX_BATCH) return false;
    if (d.d_model >= 8192 && T > 32) return false;          // the accurate K / V projection has launches of its own
    a.T = T; a.B = B; a.R = R; a.terms = tc_terms(T);
    a.cols = (a.terms * T + 15) / 16 * 16;
    if (a.cols > FW_MAX_COLS) return false;
    const bool wide = G * R > FW_QROWS;
    a.nqb = wide ? up_div(G * R, FW_QROWS_WIDE) : 1;
    a.qrows = up_div(G * R, a.nqb);
    a.cls = fw_few(T, G * R) ? 0 : 2;
    while (FW_CLASS[a.cls].cols < a.cols) ++a.cls;
    a.slots = fw_slots(d, a.cls);
    fw_geometry(a.ph, d, n_cta, a.cls);
    a.n_cta = n_cta; a.n_layers = d.layers;
    a.p_lo = 0; a.p_hi = 5 * d.layers + 1;
    a.d = d.d_model; a.F = d.d_ffn; a.V = d.vocab; a.Hq = d.n_q_heads; a.Hkv = d.n_kv_heads; a.hd = d.head_dim;
    for (int k = 0; k < 6; ++k) {
        if (k == FW_ATTN) continue;
        FwPhase& f = a.ph[k];
        f.S = 1;
        for (int S = 2; S <= f.kb; ++S)
            if (f.kb % S == 0 && S * f.hr <= TC_TILE_N && S * a.cols * f.nbox <= FW_ACC) f.S = S;
        if (f.b_off + f.kb * a.cols * 128 > FW_RING / a.slots || f.nbox * f.S * a.cols > FW_ACC_ONE) return false;
        if ((k == FW_O || k == FW_DOWN || f.c > 1) && (f.n_tiles > n_cta || f.steps < f.c)) return false;
        // Accumulators.  At every addition into an accumulator the tensor core cuts off what fp32 does not hold, toward zero,
        // so a sum's error goes with the k-blocks that one accumulator takes (6.9e-8 each).  A box has as many accumulators as
        // keep them below `cap`, which take the k-blocks in turn and are added by the epilogue (one box: at least two where the
        // tile keeps to its buffer, so that both issuing warps have one).  The caps are about what the chain of launches,
        // whose blocks share a tile's k-range, leaves to an accumulator; its error against 64 bits is the measure.  7B, 4096 ->
        // 11008 -> 4096: gate / up 7.5e-6 there, 11.2e-6 with one accumulator, 8.0e-6 with two; down of 65 rows 2.2, 3.2 and
        // 1.7e-6.  It costs 1 % of a step of five rows, 2 % of one of 65.
        const int cap = std::max(4, k == FW_QKV ? std::min(f.k_blocks / 2, 43) : (k == FW_O ? f.k_blocks / 4 : (k == FW_GATEUP ?
                                f.k_blocks / 2 : (k == FW_DOWN ? f.k_blocks / 6 : f.k_blocks))));
        const int base = f.nbox * f.S * a.cols, most = f.n_tiles <= n_cta ? FW_ACC_ONE : FW_ACC;
        const int fewest = f.steps / f.c * (f.kb / f.S);          // MMAs along k of a block, at least and at most
        const int longest = up_div(f.steps, f.c) * (f.kb / f.S);
        const int room = std::max(1, std::min(std::min(4, fewest), most / base));
        f.na = f.nbox == 1 && 2 * base <= FW_ACC ? std::min(2, room) : 1;
        while (f.na < room && up_div(longest, f.na) > cap) ++f.na;
        f.both = f.na * base > FW_ACC ? 1 : 0;
        // Gate / up of many rows: two boxes leave room for one or two accumulators each, and the k-range of a tile is taken
        // in parts instead, after each of which the sums move to other columns of the tensor memory.
        f.segs = 1;
        f.stash = 0;
        if (k == FW_GATEUP && a.cls >= 2 && f.S == 1 && up_div(longest, f.na) > cap) {
            const int put = 2 * ((a.T + 15) / 16 * 16);
            for (int n = f.na; n >= 1; --n) {
                const int segs = up_div(up_div(longest, n), cap), used = n * base;
                const bool one = used <= FW_ACC && used + put <= 256;
                if ((!one && (f.n_tiles > n_cta || used + put > 512)) || f.steps / segs * f.kb < n) continue;
                f.na = n;
                f.segs = segs;
                f.both = one ? 0 : 1;
                f.stash = used;
                break;
            }
        }
        const int per = a.terms == 3 ? 5 : 16;             // rows of one drain load (gate / up with one slice has no use for blk)
        const int fit = FW_UNION / (per * (f.nbox * f.S * f.hr + 4) * 4);
        if (fit < 1) return false;
        f.blk = std::min(up_div(T, per), fit) * per;
    }
    return true;
}

// A (sequence, KV head) costs the attention of the one launch about 2 us beside its tiles, and a tile takes as long with one
// query row as with eight.  With heads of 128 its tiles are bound by their bytes all the same (64 sequences of one row, 7B
// width: 0.96..1.01 of the chain); with heads of 64 the mma.sync warps, which spread over more blocks, are faster from some
// number of sequences on.  Measured, chain -> one launch, us of a step (eight layers of width 2048, 32 heads of 64): 64 x 1
// rows, 64 / 512 / 2048 / 4096 keys 1111 -> 1196, 1343 -> 1498, 2050 -> 2616, 3011 -> 4045; 40 x 1, 2048 keys 1520 -> 1667;
// 32 x 1, 2048 keys 1383 -> 1454; 28 x 2, 4096 keys 1958 -> 1909; 24 x 1 1646 -> 1628; 18 x 4, 2048 and 4096 keys 1306 ->
// 1286, 1618 -> 1712; 8 x 8, 8192 and 16384 keys 1430 -> 1455, 2076 -> 2201.  A draft of the 13B pair (16 heads), 64 x 1, 2048
// keys 1404 -> 1643; 32 x 2 1127 -> 1159; 32 x 1 1023 -> 1002.
bool fw_pays(const mtad_model_desc& d, int B, int R, long long total) {
    if (d.head_dim != 64) return true;
    const long long heads = (long long)B * d.n_kv_heads, tiles = heads * ((total + FW_KEYS - 1) / FW_KEYS);
    return B <= 32 && heads < 1000 && (B * R < 64 || (B < 32 && tiles < 80 * 148));
}

// The launch of its own costs 7..10 us more a layer than attn_mma_kernel's two, which overlap their neighbours; it gains by
// its tiles: with more than 96 query rows per KV head, six tiles of 16, that kernel takes them in rounds, and with heads of
// 128 it is slower by the key from 17 rows on.  Measured a step of eight layers, attn_mma_kernel -> here, us: 64 heads of 128
// on 8 KV heads, 129 rows, 1024 keys 7682 -> 6770, 6 x 18 rows 5317 -> 5359, 2048 keys 5704 -> 5441; 32 heads of 128 on as
// many, 81 rows, 16 / 1024 / 4096 keys 1588 -> 1644, 1770 -> 1719, 2119 -> 1964; 129 rows 2780 -> 2695, 3028 -> 2833, 3944 ->
// 3140; 6 x 18 rows, 1024 and 4096 keys 2089 -> 2136, 2681 -> 2586; 32 heads of 64 on as many, 81 rows 945 -> 996, 996 ->
// 1076, 1133 -> 1308; 97 rows, 64 and 2048 keys 1013 -> 1050, 1293 -> 1195; 32 heads of 64 on 8, 4 x 30 rows, 256 and 2048
// keys 1052 -> 1074, 1298 -> 1220; 81 rows 1049 -> 978, 1209 -> 1101.
bool fw_attn_pays(const mtad_model_desc& d, int B, int R, long long total) {
    const int tiles = (d.n_q_heads / d.n_kv_heads * R + 15) / 16;
    if (total >= 2048) return tiles > 6 || (d.head_dim == 128 && B <= 8);
    return B <= 4 && tiles > (d.head_dim == 128 ? 6 : 9);
}

bool fw_attn_plan(FwArgs& a, const mtad_model_desc& d, int B, int R, int n_cta) {
    const int G = d.n_q_heads / d.n_kv_heads;
    if ((d.head_dim != 64 && d.head_dim != 128) || G * R <= FW_QROWS || B * R > TC_MAX_ROWS || B > MTAD_MAX_BATCH) return false;
    a.T = B * R; a.B = B; a.R = R; a.terms = tc_terms(a.T); a.cls = FW_CLASSES - 1; a.slots = 4;
    a.nqb = up_div(G * R, FW_QROWS_WIDE);
    a.qrows = up_div(G * R, a.nqb);
    a.n_cta = n_cta; a.n_layers = d.layers;
    a.Hq = d.n_q_heads; a.Hkv = d.n_kv_heads; a.hd = d.head_dim;
    return true;
}

cudaError_t launch_forward_attention(FwArgs& a, int layer, cudaStream_t st, bool refuse) {
    a.p_lo = 5 * layer + FW_ATTN;
    a.p_hi = a.p_lo + 1;
    return launch_forward(a, st, refuse);
}

size_t fw_parts_max(const mtad_model_desc& d, int n_cta, bool lm) {
    size_t most = 0;
    for (int c = 0; c < FW_CLASSES; ++c) {
        FwPhase ph[6];
        fw_geometry(ph, d, n_cta, c);
        for (int k : {FW_O, FW_DOWN, FW_LM})
            if ((k == FW_LM) == lm) most = std::max(most, (size_t)(ph[k].n_tiles / ph[k].c));
    }
    return most;
}

size_t fw_part_floats(const mtad_model_desc& d, int n_cta, int max_batch, int max_rows) {
    const int T = max_batch * max_rows;
    if (fw_few(T, d.n_q_heads / d.n_kv_heads * max_rows)) return 0;
    size_t most = 0;
    for (int c = 2; c < FW_CLASSES; ++c) {
        FwPhase ph[6];
        fw_geometry(ph, d, n_cta, c);
        for (int k : {FW_QKV, FW_O, FW_DOWN})               // (a box's k-blocks side by side are 128 rows at most)
            if (ph[k].c > 1) most = std::max(most, (size_t)ph[k].n_tiles * ph[k].nbox * TC_TILE_N);
    }
    return most * std::min(T, FW_MAX_ROWS);
}

bool forward_fits(int n_cta) {
    int dev = 0, sms = 0, coop = 0, smem = 0;
    // (a block per SM: each asks for nearly all of an SM's shared memory)
    return cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
           sms >= n_cta && coop && smem >= 227 * 1024;
}

cudaError_t launch_forward(const FwArgs& a, cudaStream_t st, bool refuse) {
    const size_t smem = (size_t)FW_RING + FW_UNION + sizeof(FwTail);
    auto go = [&](auto kernel) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(refuse ? 1 << 20 : a.n_cta);
        cfg.blockDim = dim3(FW_THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeCooperative;         // the blocks wait on one another: all of them resident, or an error
        at[0].val.cooperative = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kernel, a);
    };
    // instantiations: head size, query rows of an attention item, few rows in all, ring slots
    auto pick = [&](auto hd) -> cudaError_t {
        constexpr int HD = decltype(hd)::value;
        const int n_q = (a.Hq / a.Hkv) * a.R;
        auto rows = [&](auto few, auto slots) -> cudaError_t {
            constexpr bool FEW = decltype(few)::value;
            constexpr int NS = decltype(slots)::value;
            if (n_q <= 8) return go(forward_kernel<HD, 8, FEW, NS>);
            if (FEW || n_q <= FW_QROWS) return go(forward_kernel<HD, FW_QROWS, FEW, NS>);
            return go(forward_kernel<HD, FEW ? FW_QROWS : FW_QROWS_WIDE, FEW, NS>);
        };
        using std::integral_constant;
        if (a.cls < 2) return rows(std::true_type{}, integral_constant<int, 4>{});
        return a.slots == 3 ? rows(std::false_type{}, integral_constant<int, 3>{}) : rows(std::false_type{}, integral_constant<int, 4>{});
    };
    return a.hd == 128 ? pick(std::integral_constant<int, 128>{}) : pick(std::integral_constant<int, 64>{});
}

}  // namespace mtad
