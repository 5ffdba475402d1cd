// cs_blend.cu -- front-to-back alpha compositing of a CrowdSplat frame.
//
// The 3DGS rasteriser CrowdSplat renders with (cited in Sec. 1 and Sec. 2)
// composites, for every pixel, the depth-sorted splats of its 16x16 tile:
//   q = -(A dx^2 + C dy^2)/2 - B dx dy;  skip q > 0;
//   alpha = min(0.99, o e^q);  skip alpha < 1/255;
//   T' = T (1 - alpha);  stop (without this splat) once T' < 1e-4;
//   C += c alpha T;  T = T'.
// A splat also contributes only where the pixel centre lies in its square
// support box (|dx|, |dy| <= r), which makes the image independent of the
// tile size.
//
// Pass 1 of a plain frame (k_blend_pp) composites each 8x4 pixel block of
// a tile with a long list with eight warps that split the block's
// depth-ordered pairs into sub-ranges and chain their partial composites,
// and every tile with a short list with one CTA, one warp per block
// (described at the kernel).
//
// Statistics and training frames take k_blend_walk: a CTA per tile, a warp
// per 8x4 block of it, one pixel per lane, each warp walking its block's
// pairs on its own.  So do the split passes of long lists: a list is split
// in depth order (the compositing operator is associative); the first
// `budget` pairs of every tile are composited as above (kBudget in plain
// frames, kTrainBudget in training), tiles with unsaturated pixels left hand
// the rest to k_blend_chunks, which composites chunks of kChunk pairs in
// parallel, each from T = 1 and only for pixels still open; the warp that
// finishes a block's last chunk then combines, per pixel, C += T C_k,
// T *= T_k in order, up to the chunk (if any) inside which the pixel meets
// the stop rule (T T_k < 1e-4);
// k_blend_fix composites each such chunk again, in parallel over chunks, for
// its stopping pixels from their true T, so the stop rule holds exactly as in
// the definition.
//
// Rounding of T.  The stop rule compares T with a constant, so an ulp of T
// can decide whether a pixel takes one more splat (up to 1e-3 in colour).  T
// is therefore always the product over the same groups of pairs: in training
// frames over chunks of kChunk pairs whether they are composited in turn
// (the walk, settle_group) or in parallel.
#include <algorithm>

#include "crowdsplat.h"
#include "cs_internal.cuh"

namespace cs {

constexpr int kBlendThreads = kTile * kTile;
constexpr int kBlockW = kBlendBlockW, kBlockH = kBlendBlockH;  // pixels per warp
constexpr float kLog2e = 1.4426950408889634f;
constexpr uint32_t kBudget = kBlendBudget;  // pairs of pass 1 per tile in plain frames
constexpr uint32_t kChunk = kBlendChunk;    // pairs per pass-2 chunk
constexpr size_t kChunkGrid = 8192;         // CTAs of the chunk and fix-up grids at most
constexpr int kBlocks = kTile * kTile / 32;  // 8x4 blocks per tile
constexpr int kWalkCtas = 5;                // resident CTAs per SM of the walking kernels (48 registers)
constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kClosed = 2.0f;             // alpha threshold of a pixel that takes no more splats
constexpr float kStopped = 3.0f;            // the same, stopped inside the current group of pairs
static_assert(kBwdChunk == kChunk && kTrainBudget % kBwdChunk == 0, "backward chunk boundaries fall on group starts");

// e^q evaluated as 2^(q log2 e) on the hardware ex2 unit
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Two FP32 values in one 64-bit register: the packed instructions round each
// half exactly as the scalar ones do, at half the issue slots.
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo2(f2 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(f2 v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// The splats of 32 consecutive pairs that meet a block, compacted in depth
// order, two neighbours side by side so that one 16-byte load feeds two
// packed operands.  p = q log2 e = a' dx^2 + b' dx dy + c' dy^2.
struct __align__(16) HitStage {
    ulonglong2 uv[16];  // -u, -v
    ulonglong2 ab[16];  // a', b'
    ulonglong2 cl[16];  // c', log2 o
    ulonglong2 rr[16];  // radius, r
    ulonglong2 gb[16];  // g, b
    uint32_t id[32];    // splat id (statistics) or one past the pair's index (training)
};

__device__ __forceinline__ void put2(ulonglong2 *dst, int pos, float first, float second) {
    float *f = reinterpret_cast<float *>(dst) + (pos >> 1) * 4 + (pos & 1);
    f[0] = first;
    f[2] = second;
}

__device__ __forceinline__ void stage_hit(HitStage &st, int pos, const float4 &q, const float4 &a, const float4 &c) {
    put2(st.uv, pos, -a.x, -a.y);
    put2(st.ab, pos, -0.5f * kLog2e * a.z, -kLog2e * a.w);
    put2(st.cl, pos, -0.5f * kLog2e * q.w, q.z);
    put2(st.rr, pos, c.w, c.x);
    put2(st.gb, pos, c.y, c.z);
}

// A splat that contributes nowhere: fills the last pair of an odd count.
__device__ __forceinline__ void stage_pad(HitStage &st, int pos) {
    put2(st.uv, pos, 0.0f, 0.0f);
    put2(st.ab, pos, 0.0f, 0.0f);
    put2(st.cl, pos, 0.0f, 0.0f);
    put2(st.rr, pos, -1.0f, 0.0f);
    put2(st.gb, pos, 0.0f, 0.0f);
    st.id[pos] = 0u;
}

struct Pixel {
    f2 x, y;         // pixel centre, in both halves
    float T, thr;    // transmittance; smallest alpha that counts (above 1: the pixel takes no more splats)
    float T0, P;     // T before the current group of pairs; product of 1 - alpha over the group so far
    f2 r, g, b;      // colour sums of the even and the odd hits
    uint32_t last;   // one past the last composited pair (training)
};

__device__ __forceinline__ Pixel make_pixel(float x, float y, bool open, const float4 &s, uint32_t last) {
    return Pixel{pack2(x, x), pack2(y, y), s.w, open ? kAlphaMin : kClosed, s.w, 1.0f, pack2(s.x, 0.0f),
                 pack2(s.y, 0.0f), pack2(s.z, 0.0f), last};
}
__device__ __forceinline__ bool closed(const Pixel &p) { return p.thr > 1.0f; }
// r, g, b and w
__device__ __forceinline__ float4 pixel_state(const Pixel &p, float w) {
    return make_float4(lo2(p.r) + hi2(p.r), lo2(p.g) + hi2(p.g), lo2(p.b) + hi2(p.b), w);
}

__device__ __forceinline__ float keep_alpha(float dx, float dy, float radius, float p, float e, float thr) {
    const float alpha = fminf(0.99f, ex2_approx(e));
    return fmaxf(fabsf(dx), fabsf(dy)) > radius || p > 0.0f || alpha < thr ? 0.0f : alpha;
}

// alpha of hits 2k and 2k + 1 at the pixel, 0 where a splat does not
// contribute (outside its support box, q > 0, alpha below the threshold):
// compositing alpha = 0 leaves T and C unchanged exactly, so no test follows.
__device__ __forceinline__ void pair_alpha(const HitStage &st, int k, const Pixel &px, float &a0, float &a1) {
    const ulonglong2 uv = st.uv[k], ab = st.ab[k], cl = st.cl[k];
    const f2 rad = st.rr[k].x;
    const f2 dx = add2(px.x, uv.x), dy = add2(px.y, uv.y);
    const f2 p = fma2(mul2(cl.x, dy), dy, mul2(dx, fma2(ab.y, dy, mul2(ab.x, dx))));
    const f2 e = add2(p, cl.y);
    a0 = keep_alpha(lo2(dx), lo2(dy), lo2(rad), lo2(p), lo2(e), px.thr);
    a1 = keep_alpha(hi2(dx), hi2(dy), hi2(rad), hi2(p), hi2(e), px.thr);
}

// The same for one splat.
__device__ __forceinline__ float splat_alpha(float dx, float dy, float a, float b, float c, float lo, float radius) {
    const float p = __fmaf_rn(__fmul_rn(c, dy), dy, __fmul_rn(dx, __fmaf_rn(b, dy, __fmul_rn(a, dx))));
    return keep_alpha(dx, dy, radius, p, __fadd_rn(p, lo), kAlphaMin);
}

// The colour of a splat with weight zero must not count: zero times an
// infinite colour is NaN.  kWild: some of the staged colours are not finite.
template <bool kWild>
__device__ __forceinline__ void add_colour(const HitStage &st, int k, Pixel &px, f2 w) {
    const ulonglong2 gb = st.gb[k];
    const auto used = [w](f2 c) {
        return kWild ? pack2(lo2(w) > 0.0f ? lo2(c) : 0.0f, hi2(w) > 0.0f ? hi2(c) : 0.0f) : c;
    };
    px.r = fma2(used(st.rr[k].y), w, px.r);
    px.g = fma2(used(gb.x), w, px.g);
    px.b = fma2(used(gb.y), w, px.b);
}

// kMode 0: colour only; 1 (statistics): also add every composited weight
// alpha T, summed over the warp's pixels, to contrib[splat]; 2 (training):
// also track the last composited pair.
enum { kPlain = 0, kStats = 1, kTraining = 2 };

// The staged hits composited in order, with the stop rule.  Every lane of
// the warp calls it.
template <int kMode, bool kWild>
__device__ __forceinline__ void walk_hits(const HitStage &st, int cnt, Pixel &px, float *__restrict__ contrib) {
#pragma unroll 1
    for (int k = 0; 2 * k < cnt; ++k) {
        float a0, a1;
        pair_alpha(st, k, px, a0, a1);
        const float o0 = 1.0f - a0, o1 = 1.0f - a1, P1 = px.P * o0;
        float T1 = px.T * o0, T2 = T1 * o1;
        if (kMode == kTraining) px.P = P1 * o1;
        if (__any_sync(0xffffffffu, T2 < 1e-4f)) {
            // some pixel stops at one of the two (closed ones keep their T)
            if (T1 < 1e-4f) {
                a0 = a1 = 0.0f;
                T1 = T2 = px.T;
                if (kMode == kTraining) px.P = P1;
                px.thr = kStopped;
            } else if (T2 < 1e-4f) {
                a1 = 0.0f;
                T2 = T1;
                px.thr = kStopped;
            }
        }
        const float w0 = a0 * px.T, w1 = a1 * T1;
        add_colour<kWild>(st, k, px, pack2(w0, w1));
        px.T = T2;
        if (kMode == kTraining) {
            if (a0 > 0.0f) px.last = st.id[2 * k];
            if (a1 > 0.0f) px.last = st.id[2 * k + 1];
        }
        if (kMode == kStats && __any_sync(0xffffffffu, w0 + w1 > 0.0f)) {
            // both sums in five exchanges: each half warp takes one splat
            const bool up = (threadIdx.x & 16) != 0;
            float v = (up ? w1 : w0) + __shfl_xor_sync(0xffffffffu, up ? w0 : w1, 16);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if ((threadIdx.x & 15) == 0 && v > 0.0f) atomicAdd(contrib + st.id[2 * k + (up ? 1 : 0)], v);
        }
    }
}

// Lane's pair as loaded ahead: its splat and first record word.
__device__ __forceinline__ bool meets_block(const float4 &q, int bx0, int by0) {
    const uint32_t rx = __float_as_uint(q.x), ry = __float_as_uint(q.y);
    return (int)(rx & 0xFFFFu) <= bx0 + kBlockW - 1 && (int)(rx >> 16) >= bx0 &&
           (int)(ry & 0xFFFFu) <= by0 + kBlockH - 1 && (int)(ry >> 16) >= by0;
}

// Stage the lanes' pairs whose reach box meets the block; returns how many,
// and in `wild` whether a colour among them is not finite (their sum is not).
// Only those load the other 32 bytes of their record.
template <int kMode>
__device__ __forceinline__ int stage_hits(HitStage &st, bool have, uint32_t s, const float4 &q, uint32_t pair,
                                          const float4 *__restrict__ rec, int bx0, int by0, bool &wild) {
    const int lane = threadIdx.x & 31;
    const bool mine = have && meets_block(q, bx0, by0);
    const uint32_t m = __ballot_sync(0xffffffffu, mine);
    const int cnt = __popc(m);
    bool odd = false;
    if (mine) {
        const float4 *p = rec + (size_t)s * kRecVec;
        const float4 a = __ldg(p + 1), c = __ldg(p + 2);
        const int pos = __popc(m & ((1u << lane) - 1u));
        stage_hit(st, pos, q, a, c);
        odd = !(c.x + c.y + c.z < INFINITY);
        if (kMode != kPlain) st.id[pos] = kMode == kStats ? s : pair + 1u;
    }
    if (lane == 0 && (cnt & 1)) stage_pad(st, cnt);
    wild = __any_sync(0xffffffffu, odd);
    return cnt;
}

// Training: what a pixel keeps for the backward, its final state and one
// past its last composited pair.
__device__ __forceinline__ void store_final(const BlendWork &work, size_t pix, uint32_t last, const float4 &s) {
    work.px_end[pix] = last;
    work.px_fin[pix] = s;
}

// Training: an open pixel's state before pair `base` of the tile's list, at
// every kBwdChunk-th pair (p: the pixel's number in its tile).
__device__ __forceinline__ void store_boundary(const BlendWork &work, uint32_t start, uint32_t base, int p,
                                               const float4 &s) {
    if (base > start && (base - start) % kBwdChunk == 0)
        work.px_bnd[(size_t)(base / kBwdChunk) * kBlendThreads + p] = s;
}

// The pixel stopped inside the group by its pair-by-pair T, but not by T0 P
// (one rounding apart).  The group's whole product decides: below the
// threshold, the pixel stays stopped where it is; otherwise it takes the
// pairs from the stopping one to the group's end as well.  Lanes that come
// here (one pixel in millions) read the group's pairs [g0, g1) again.
__device__ __noinline__ void settle_stop(Pixel &px, uint32_t g0, uint32_t g1, const uint32_t *__restrict__ pval,
                                         const float4 *__restrict__ rec) {
    float P = 1.0f, T = px.T0, Ts = 0.0f, r = 0.0f, g = 0.0f, b = 0.0f;
    uint32_t last = px.last;
    bool past = false;
    for (uint32_t i = g0; i < g1; ++i) {
        const uint32_t s = __ldg(pval + i);
        const float4 *p = rec + (size_t)s * kRecVec;
        const float4 q = __ldg(p), a = __ldg(p + 1), c = __ldg(p + 2);
        const float alpha = splat_alpha(lo2(px.x) - a.x, lo2(px.y) - a.y, -0.5f * kLog2e * a.z, -kLog2e * a.w,
                                        -0.5f * kLog2e * q.w, q.z, c.w);
        P *= 1.0f - alpha;
        const float Tn = T * (1.0f - alpha);
        if (!past && Tn < 1e-4f) {
            past = true;
            Ts = T;
        }
        if (past && alpha > 0.0f) {
            const float w = alpha * T;
            r += c.x * w;
            g += c.y * w;
            b += c.z * w;
            last = i + 1u;
        }
        T = Tn;
    }
    const float Tq = px.T0 * P;
    if (Tq < 1e-4f) {
        px.T = Ts;
        px.thr = kClosed;
        return;
    }
    px.T = Tq;
    px.thr = kAlphaMin;
    px.last = last;
    px.r = add2(px.r, pack2(r, 0.0f));
    px.g = add2(px.g, pack2(g, 0.0f));
    px.b = add2(px.b, pack2(b, 0.0f));
}

// End of the group of pairs [g0, g1): T is T0 times the group's product
// where that stays above the stop threshold, the pair-by-pair T (and where it
// stopped) otherwise.  A pixel that is below the threshold by the product
// alone stays open, but takes no more: its T is within 1,024 roundings (6e-5)
// of the threshold, and every splat that counts takes at least 1/255 of it.
// The chunks close such a pixel: the same image and list end.
__device__ __forceinline__ void settle_group(Pixel &px, uint32_t g0, uint32_t g1, const uint32_t *__restrict__ pval,
                                             const float4 *__restrict__ rec) {
    const float Tq = px.T0 * px.P;
    const bool stopped = px.thr == kStopped;
    if (Tq >= 1e-4f) {
        if (stopped) {
            Pixel t = px;  // a copy: the pixel itself stays in registers
            settle_stop(t, g0, g1, pval, rec);
            px = t;
        } else if (!closed(px)) {
            px.T = Tq;
        }
    } else if (stopped) {
        px.thr = kClosed;
    }
    px.T0 = px.T;
    px.P = 1.0f;
}

// The warp's block composited over pairs [start, end), 32 at a time; the
// splat ids are loaded two batches ahead and the reach boxes one, so that
// only the hits' records are waited for.  With `groups` (training),
// T is settled every kChunk pairs from start and each open pixel's state
// kept where they begin; without, T is the pair-by-pair product.
template <int kMode>
__device__ __forceinline__ void warp_walk(HitStage &st, uint32_t start, uint32_t end, const uint32_t *__restrict__ pval,
                                          const float4 *__restrict__ rec, int bx0, int by0, Pixel &px,
                                          const BlendWork &work, bool groups) {
    const int lane = threadIdx.x & 31;
    if (start >= end || __all_sync(0xffffffffu, closed(px))) return;
    uint32_t i = start + (uint32_t)lane;
    uint32_t s = i < end ? __ldg(pval + i) : 0u;
    uint32_t s1 = i + 32u < end ? __ldg(pval + i + 32) : 0u;
    float4 q = i < end ? __ldg(rec + (size_t)s * kRecVec) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (uint32_t base = start; base < end; base += 32u, i += 32u) {
        if (kMode == kTraining && groups && !closed(px))
            store_boundary(work, start, base, (int)threadIdx.x, pixel_state(px, px.T));
        bool wild;
        const int cnt = stage_hits<kMode>(st, i < end, s, q, i, rec, bx0, by0, wild);
        s = s1;
        if (i + 32u < end) q = __ldg(rec + (size_t)s * kRecVec);
        if (i + 64u < end) s1 = __ldg(pval + i + 64);
        __syncwarp();
        if (wild) walk_hits<kMode, true>(st, cnt, px, work.contrib);
        else walk_hits<kMode, false>(st, cnt, px, work.contrib);
        __syncwarp();  // the staging buffer is refilled by the next batch
        const uint32_t next = base + 32u;
        bool settled = true;
        if (kMode == kTraining && groups) {
            if (next >= end || (next - start) % kChunk == 0u)
                settle_group(px, next - 1u - (next - 1u - start) % kChunk, min(next, end), pval, rec);
            settled = px.thr != kStopped || px.T0 * px.P < 1e-4f;
        }
        if (__all_sync(0xffffffffu, closed(px) && settled)) break;
    }
}

struct BlockGeom {
    int bx0, by0, px, py;
    bool inside;
    float fpx, fpy;
};

// Block blk of a tile (column blk % 2, row blk / 2) and the lane's pixel.
__device__ __forceinline__ BlockGeom block_geom(int tile, int blk, int tiles_x, int W, int H, int ox, int oy) {
    BlockGeom g;
    const int tyi = tile / tiles_x, txi = tile - tyi * tiles_x, lane = threadIdx.x & 31;
    g.bx0 = txi * kTile + (blk & 1) * kBlockW;
    g.by0 = tyi * kTile + (blk >> 1) * kBlockH;
    g.px = g.bx0 + (lane & (kBlockW - 1));
    g.py = g.by0 + lane / kBlockW;
    g.inside = g.px < W && g.py < H;
    g.fpx = (float)(g.px + ox) + 0.5f;
    g.fpy = (float)(g.py + oy) + 0.5f;
    return g;
}

// The pixel's state at the start of the split passes (T negated when closed).
__device__ __forceinline__ void keep_state(const BlendWork &work, int slot, const Pixel &px, bool open) {
    const size_t sp = (size_t)slot * kBlendThreads + threadIdx.x;
    work.state[sp] = pixel_state(px, open ? px.T : -px.T);
    work.slast[sp] = px.last;
    if (open) work.cand_done[slot] = 0u;  // any of them: the plan set it to 1
}

// Statistics frames (every list to its end) and the first kTrainBudget pairs
// of training frames: a CTA per tile, tiles in decreasing list length class,
// a warp per block.  The warps share nothing but the cache lines of the
// tile's records: no CTA barrier, so a warp whose block saturates early waits
// for nobody, and only pairs in front of the saturating one are evaluated.
// Bound by instruction issue (68% of the slots at 52% of the warps).  Against
// a CTA of eight warps in step over batches of 256 pairs (stalled 13 of 22
// cycles at its barriers, one atomic per pixel and splat): statistics frame
// of 100 full-detail characters at 3840x2160 2.63 -> 2.05 ms (this kernel
// 1.91 -> 1.18).  Against chunks of kChunk pairs composited in parallel from
// T = 1, which evaluates the hidden ones too: training frame of 64
// characters at 512x512 1.52 -> 0.69 ms of compositing.  48 registers and 40
// warps per SM are faster than 40 and 48 (spills) or 32 and 64.
template <int kMode>
__global__ void __launch_bounds__(kBlendThreads, kWalkCtas) k_blend_walk(int tiles_x, int W, int H,
                                                                         const uint2 *__restrict__ ranges,
                                                                         const uint32_t *__restrict__ pval,
                                                                         const float4 *__restrict__ rec,
                                                                         float4 *__restrict__ out, BlendWork work) {
    __shared__ HitStage st[kBlocks];
    const int tile = work.pp_tile[blockIdx.x], warp = threadIdx.x >> 5;
    if (!in_bounds(tile < tiles_x * ((H + kTile - 1) / kTile), kChkTile)) return;
    const BlockGeom g = block_geom(tile, warp, tiles_x, W, H, work.ox, work.oy);
    const size_t pix = (size_t)g.py * W + g.px;
    uint2 rg = ranges[tile];
    if (!in_bounds(rg.x <= rg.y && rg.y <= work.n_pairs, kChkPair)) rg.y = rg.x;
    const uint32_t n = rg.y - rg.x, end = rg.x + (kMode == kStats ? n : min(n, work.budget));
    Pixel px = make_pixel(g.fpx, g.fpy, g.inside, make_float4(0.f, 0.f, 0.f, 1.f), n ? rg.x : 0u);
    warp_walk<kMode>(st[warp], rg.x, end, pval, rec, g.bx0, g.by0, px, work, kMode == kTraining);
    if (kMode == kTraining && end < rg.y && in_bounds(work.cand_slot[tile] >= 0, kChkSlot)) {
        // the merge reads the whole tile's states
        const bool open = !closed(px), any = __any_sync(0xffffffffu, open);
        keep_state(work, work.cand_slot[tile], px, open);
        if (any) return;
    }
    if (g.inside) {
        out[pix] = pixel_state(px, 1.0f - px.T);
        if (kMode == kTraining) store_final(work, pix, px.last, pixel_state(px, px.T));
    }
}

// ---------------------------------------------------------------------------
// Pass 1 of plain frames, pair-parallel.  A CTA of kPpWarps warps
// composites one 8x4 pixel block of a tile, one pixel per lane, in rounds
// of kPpRound pairs: warp k composites pairs
// [32 k, 32 k + 32) of the round for the block's pixels from T = 1 (a
// partial (C_k, T_k), no stop rule); warp 0 then chains the partials in
// depth order, C += T C_k, T *= T_k, and where T T_k would fall below the
// stop threshold it composites sub-range k again from the true T with the
// stop rule, so the stop rule holds exactly as in the sequential definition
// (only it needs the true T; the rest of the operator is associative).  A
// block's dependency chain is one round per kPpRound pairs, split over
// eight warps, instead of every pair in turn: a long list of large splats
// no longer leaves the GPU waiting on a single CTA.
//
// In frames with many busy tiles (blend_key), a tile whose list is shorter
// (below 2^(kPpTileClass - 1) pairs) is one item of its own instead: the CTA stages each batch of kPpRound pairs once
// for the whole tile, with the blocks each reach box meets as one bit mask
// per block, and warp w composites block w's pairs in depth order, as the
// definition reads.  Eight block items would stage every pair eight times
// and pay eight rounds of barriers and chaining; where lists are mid-length
// and many (a 4K frame of a large crowd) the pass is bound by instruction
// issue, and the tile items issue about a fifth fewer instructions there.
//
// Persistent CTAs take items in decreasing schedule key (blend_key: the
// list length class, raised for tile items), so the longest dependency
// chains start first; empty tiles (background) come last.
// ---------------------------------------------------------------------------
constexpr int kPpWarps = 8;
constexpr int kPpThreads = 32 * kPpWarps;
constexpr uint32_t kPpRound = 32 * kPpWarps;
constexpr int kPpBlocks = kTile * kTile / 32;  // 8x4 blocks per tile
constexpr int kPpTileClass = 14;               // lists of fewer than 8,192 pairs: tile items
static_assert((1u << (kPpTileClass - 1)) <= kBlendBudget, "a tile item composites its whole list");

struct PpShared {
    float4 s0[kPpWarps][32];  // u, v, a', b' with p = q log2 e = a' dx^2 + b' dx dy + c' dy^2
    float4 s1[kPpWarps][32];  // c', log2 o, radius, -
    float4 s2[kPpWarps][32];  // r, g, b, -
    float4 part[kPpWarps][32];
    uint32_t wm[kPpBlocks][kPpWarps];  // tile items: bit l of wm[b][k]: pair 32 k + l meets block b
    uint32_t m[kPpWarps];  // pairs of each sub-range whose reach box meets the block
    uint32_t done;         // pixels of the block that are done
    int tile, kind, blk;   // the current item: kind 0 empty tile, 1 tile item, 2 block item
    int seg_item[kBlendKeys + 1], seg_tile[kBlendKeys + 1];  // first item and tile of each key, decreasing key
};

// List length class of a tile: 0 empty, else 1 + floor(log2 n) (capped).
__device__ __forceinline__ int blend_class(uint32_t n) {
    return n == 0u ? 0 : 1 + min(kBlendClasses - 2, 31 - __clz((int)n));
}

// Schedule key of a tile in pass 1 (larger first), from its class c: 2c + 1
// for block items; for a tile item 2 (c + kPpTileShift), moved up because
// one warp composites each block's pairs in turn (a far longer dependency
// chain than a block item's for the same n, and a CTA held for the whole
// tile); 0 for an empty tile.  Longest chains first keeps the tail of the
// persistent grid short.  Tile items are used only in frames with at least
// kPpTileItemsPerCta busy tiles per persistent CTA: with fewer, block items
// keep more of the GPU busy and the frame is bound by its longest chains,
// not by instruction issue.  The shift, the threshold class and the busy
// tile count were chosen by timing the 1080p 3,500-instance frame (long
// lists), the 4K 10,000-instance frame (mostly mid-length lists) and
// 1280x720 frames of 1 to 5,000 characters.
constexpr int kPpTileShift = 4;
constexpr int kPpTileItemsPerCta = 8;
static_assert(2 * (kBlendClasses - 1) + 1 < kBlendKeys && 2 * (kPpTileClass - 1 + kPpTileShift) < kBlendKeys,
              "schedule keys");
__device__ __forceinline__ int blend_key(int c, bool tiles) {
    return c == 0 ? 0 : (tiles && c < kPpTileClass ? 2 * (c + kPpTileShift) : 2 * c + 1);
}

// Class of the tiles of schedule key k, or -1 when no class maps to it.
__device__ __forceinline__ int key_class(int k, bool tiles) {
    if (k == 0) return 0;
    if (k & 1) {
        const int c = (k - 1) >> 1;
        return c >= 1 && c < kBlendClasses && (!tiles || c >= kPpTileClass) ? c : -1;
    }
    const int c = (k >> 1) - kPpTileShift;
    return tiles && c >= 1 && c < kPpTileClass ? c : -1;
}

// Segments of the schedule in decreasing key, scanned by one warp (two keys
// per lane): segment s = key kBlendKeys - 1 - s starts at tile seg_tile[s]
// of pp_tile and at item seg_item[s] (kPpBlocks items per tile for odd keys,
// block items; one otherwise); entry kBlendKeys holds the totals.  Returns
// whether the frame uses tile items (the same answer in every CTA; forced
// by `items` unless CS_BLEND_ITEMS_AUTO).
static_assert(kBlendKeys == 64 && kBlendClasses <= 32, "one warp: two schedule keys, one class per lane");
__device__ __forceinline__ bool key_segments(const int32_t *__restrict__ meta, int ctas, int items, int *seg_item,
                                             int *seg_tile) {
    const int lane = threadIdx.x & 31, s0 = 2 * lane, k0 = kBlendKeys - 1 - s0, k1 = k0 - 1;
    int busy = lane >= 1 && lane < kBlendClasses ? meta[kBlendCountAt + lane] : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) busy += __shfl_xor_sync(0xffffffffu, busy, o);
    const bool tiles = items == CS_BLEND_ITEMS_TILES || (items == CS_BLEND_ITEMS_AUTO && busy >= kPpTileItemsPerCta * ctas);
    const int q0 = key_class(k0, tiles), q1 = key_class(k1, tiles);
    const int c0 = q0 >= 0 ? meta[kBlendCountAt + q0] : 0, c1 = q1 >= 0 ? meta[kBlendCountAt + q1] : 0;
    const int i0 = (k0 & 1) ? c0 * kPpBlocks : c0, i1 = (k1 & 1) ? c1 * kPpBlocks : c1;
    const int ii = (int)warp_inclusive_scan((uint32_t)(i0 + i1));
    const int it = (int)warp_inclusive_scan((uint32_t)(c0 + c1));
    if (seg_item) {
        seg_item[s0] = ii - i0 - i1;
        seg_item[s0 + 1] = ii - i1;
        if (lane == 31) seg_item[kBlendKeys] = ii;
    }
    seg_tile[s0] = it - c0 - c1;
    seg_tile[s0 + 1] = it - c1;
    if (lane == 31) seg_tile[kBlendKeys] = it;
    __syncwarp();
    return tiles;
}

// alpha of a staged splat at a pixel centre; 0 when the splat does not
// contribute there (outside its support box, q > 0, alpha < 1/255).  kBranchFree evaluates every test
// without branches: a splat that does not contribute then leaves T and C
// unchanged when composited with alpha = 0 (T (1 - 0) = T exactly), so the
// caller needs no test either.  That pays where the pairs of a sub-range
// are composited by many warps at once (no divergence); one warp walking a
// block's pairs in turn is faster skipping early.
template <bool kBranchFree>
__device__ __forceinline__ float staged_alpha(const float4 &a, const float4 &b, float fpx, float fpy) {
    const float dx = fpx - a.x, dy = fpy - a.y;
    if (kBranchFree) {
        const float p = dx * (a.z * dx + a.w * dy) + b.x * dy * dy;
        const float alpha = fminf(0.99f, ex2_approx(p + b.y));
        const bool skip = fmaxf(fabsf(dx), fabsf(dy)) > b.z || p > 0.0f || alpha < (1.0f / 255.0f);
        return skip ? 0.0f : alpha;
    }
    if (fmaxf(fabsf(dx), fabsf(dy)) > b.z) return 0.0f;
    const float p = dx * (a.z * dx + a.w * dy) + b.x * dy * dy;
    if (p > 0.0f) return 0.0f;
    const float alpha = fminf(0.99f, ex2_approx(p + b.y));
    return alpha < (1.0f / 255.0f) ? 0.0f : alpha;
}

__global__ void __launch_bounds__(kPpThreads, 8) k_blend_pp(int tiles_x, int W, int H, const uint2 *__restrict__ ranges,
                                                         const uint32_t *__restrict__ pval,
                                                         const float4 *__restrict__ rec, float4 *__restrict__ out,
                                                         BlendWork work) {
    __shared__ PpShared sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // items in decreasing schedule key
    if (warp == 0) key_segments(work.meta, gridDim.x, work.items, sh.seg_item, sh.seg_tile);
    for (;;) {
        if (threadIdx.x == 0) {
            const int item = (int)atomicAdd(reinterpret_cast<unsigned *>(work.meta + 3), 1u);
            int seg = 0;
            while (seg < kBlendKeys && item >= sh.seg_item[seg + 1]) ++seg;
            int tile = -1, kind = 0, blk = 0;
            if (seg < kBlendKeys) {
                const int key = kBlendKeys - 1 - seg, off = item - sh.seg_item[seg];
                const int per = (key & 1) ? kPpBlocks : 1;
                tile = work.pp_tile[sh.seg_tile[seg] + off / per];
                blk = off % per;
                kind = key == 0 ? 0 : ((key & 1) ? 2 : 1);
            }
            sh.tile = tile;
            sh.kind = kind;
            sh.blk = blk;
        }
        __syncthreads();
        const int tile = sh.tile, kind = sh.kind;
        if (tile < 0) return;
        if (!in_bounds(tile < tiles_x * ((H + kTile - 1) / kTile), kChkTile)) {
            __syncthreads();  // the item fields are rewritten for the next item
            continue;
        }
        if (kind != 2) {
            const int tyi = tile / tiles_x, txi = tile - tyi * tiles_x;
            const int tx0 = txi * kTile, ty0 = tyi * kTile;
            if (kind == 0) {
                // a tile without pairs: background (C = 0, T = 1)
                for (int q = threadIdx.x; q < kTile * kTile; q += kPpThreads) {
                    const int x = tx0 + (q & (kTile - 1)), y = ty0 + q / kTile;
                    if (x < W && y < H) out[(size_t)y * W + x] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                }
                __syncthreads();  // the item fields are rewritten for the next item
                continue;
            }
            // a short list: the whole tile, warp w compositing block w
            const int px = tx0 + (warp & 1) * kBlockW + (lane & (kBlockW - 1));
            const int py = ty0 + (warp >> 1) * kBlockH + lane / kBlockW;
            const bool inside = px < W && py < H;
            const float fpx = (float)(px + work.ox) + 0.5f, fpy = (float)(py + work.oy) + 0.5f;
            uint2 rg = ranges[tile];
            if (!in_bounds(rg.x <= rg.y && rg.y <= work.n_pairs, kChkPair)) rg.y = rg.x;
            float T = 1.0f, cr = 0.0f, cg = 0.0f, cb = 0.0f;
            bool done = !inside;
            float4 *const f0 = &sh.s0[0][0], *const f1 = &sh.s1[0][0], *const f2 = &sh.s2[0][0];
            for (uint32_t base = rg.x; base < rg.y; base += kPpRound) {
                // stage pair base + tid with the blocks its reach box meets
                const uint32_t i = base + threadIdx.x;
                uint32_t bm = 0;
                if (i < rg.y) {
                    const uint32_t s = __ldg(pval + i);
                    const float4 *p = rec + (size_t)s * kRecVec;
                    const float4 rq = __ldg(p);  // reach x, reach y, log2 o, C
                    const uint32_t rx = __float_as_uint(rq.x), ry = __float_as_uint(rq.y);
                    const int x0 = (int)(rx & 0xFFFFu) - tx0, x1 = (int)(rx >> 16) - tx0;
                    const int y0 = (int)(ry & 0xFFFFu) - ty0, y1 = (int)(ry >> 16) - ty0;
#pragma unroll
                    for (int b = 0; b < kPpBlocks; ++b) {
                        const int bx = (b & 1) * kBlockW, by = (b >> 1) * kBlockH;
                        if (x0 <= bx + kBlockW - 1 && x1 >= bx && y0 <= by + kBlockH - 1 && y1 >= by) bm |= 1u << b;
                    }
                    if (bm) {
                        const float4 ra = __ldg(p + 1), rc = __ldg(p + 2);
                        f0[threadIdx.x] = make_float4(ra.x, ra.y, -0.5f * kLog2e * ra.z, -kLog2e * ra.w);
                        f1[threadIdx.x] = make_float4(-0.5f * kLog2e * rq.w, rq.z, rc.w, 0.0f);
                        f2[threadIdx.x] = rc;
                    }
                }
#pragma unroll
                for (int b = 0; b < kPpBlocks; ++b) {
                    const uint32_t word = __ballot_sync(0xffffffffu, (bm >> b) & 1u);
                    if (lane == 0) sh.wm[b][warp] = word;
                }
                __syncthreads();
                for (int k = 0; k < kPpWarps && !done; ++k) {
                    uint32_t m = sh.wm[warp][k];
                    while (m) {
                        const int j = 32 * k + __ffs(m) - 1;
                        m &= m - 1;
                        const float alpha = staged_alpha<false>(f0[j], f1[j], fpx, fpy);
                        if (alpha == 0.0f) continue;
                        const float Tn = T * (1.0f - alpha);
                        if (Tn < 1e-4f) {
                            done = true;
                            break;
                        }
                        const float4 col = f2[j];
                        const float wgt = alpha * T;
                        cr += col.x * wgt;
                        cg += col.y * wgt;
                        cb += col.z * wgt;
                        T = Tn;
                    }
                }
                // the staging buffers are refilled by the next batch
                if (__syncthreads_count(done) == kPpThreads) break;
            }
            if (inside) out[(size_t)py * W + px] = make_float4(cr, cg, cb, 1.0f - T);
            continue;  // the loop's barriers keep the item fields until every thread has read them
        }
        const int blk = sh.blk;
        const int tyi = tile / tiles_x, txi = tile - tyi * tiles_x;
        const int bx0 = txi * kTile + (blk & 1) * kBlockW, by0 = tyi * kTile + (blk >> 1) * kBlockH;
        const int px = bx0 + (lane & (kBlockW - 1)), py = by0 + lane / kBlockW;
        const bool inside = px < W && py < H;
        const float fpx = (float)(px + work.ox) + 0.5f, fpy = (float)(py + work.oy) + 0.5f;
        uint2 rg = ranges[tile];
        if (!in_bounds(rg.x <= rg.y && rg.y <= work.n_pairs, kChkPair)) rg.y = rg.x;
        const uint32_t end1 = rg.y - rg.x > kBudget ? rg.x + kBudget : rg.y;
        // the block's chained state (warp 0)
        float T = 1.0f, cr = 0.0f, cg = 0.0f, cb = 0.0f;
        bool done = !inside;
        if (warp == 0) {
            const uint32_t dm = __ballot_sync(0xffffffffu, done);
            if (lane == 0) sh.done = dm;
        }
        __syncthreads();
        for (uint32_t base = rg.x; base < end1; base += kPpRound) {
            const uint32_t dmask = sh.done;
            if (dmask == 0xffffffffu) break;
            // stage this warp's sub-range
            const uint32_t i = base + (uint32_t)warp * 32u + (uint32_t)lane;
            bool mine = false;
            if (i < end1) {
                const uint32_t s = __ldg(pval + i);
                const float4 *p = rec + (size_t)s * kRecVec;
                // the reach box first: the rest of the record only for
                // splats whose reach box meets this block
                const float4 rq = __ldg(p);  // reach x, reach y, log2 o, C
                const uint32_t rx = __float_as_uint(rq.x), ry = __float_as_uint(rq.y);
                mine = (int)(rx & 0xFFFFu) <= bx0 + kBlockW - 1 && (int)(rx >> 16) >= bx0 &&
                       (int)(ry & 0xFFFFu) <= by0 + kBlockH - 1 && (int)(ry >> 16) >= by0;
                if (mine) {
                    const float4 ra = __ldg(p + 1), rc = __ldg(p + 2);
                    sh.s0[warp][lane] = make_float4(ra.x, ra.y, -0.5f * kLog2e * ra.z, -kLog2e * ra.w);
                    sh.s1[warp][lane] = make_float4(-0.5f * kLog2e * rq.w, rq.z, rc.w, 0.0f);
                    sh.s2[warp][lane] = rc;
                }
            }
            uint32_t m = __ballot_sync(0xffffffffu, mine);
            if (lane == 0) sh.m[warp] = m;
            __syncwarp();
            // the sub-range's partial composite from T = 1
            float Tk = 1.0f, kr = 0.0f, kg = 0.0f, kb = 0.0f;
            while (m) {
                const int j = __ffs(m) - 1;
                m &= m - 1;
                // a done pixel's partial is computed and left unused
                const float alpha = staged_alpha<true>(sh.s0[warp][j], sh.s1[warp][j], fpx, fpy);
                const float4 col = sh.s2[warp][j];
                const float wgt = alpha * Tk;
                kr += col.x * wgt;
                kg += col.y * wgt;
                kb += col.z * wgt;
                Tk *= 1.0f - alpha;
            }
            sh.part[warp][lane] = make_float4(kr, kg, kb, Tk);
            __syncthreads();
            // chain the partials in depth order
            if (warp == 0) {
                for (int k = 0; k < kPpWarps && !done;) {
                    // the first sub-range from k in which the stop rule can
                    // fall (its transmittances read at once), then the ones
                    // before it applied as wholes, in order
                    float Tq[kPpWarps];
#pragma unroll
                    for (int i = 0; i < kPpWarps; ++i) Tq[i] = i >= k ? sh.part[i][lane].w : 1.0f;
                    int ks = kPpWarps;
                    float Tb = T;
#pragma unroll
                    for (int i = 0; i < kPpWarps; ++i) {
                        if (i < k || ks < kPpWarps) continue;
                        if (Tb * Tq[i] < 1e-4f) ks = i;
                        else Tb *= Tq[i];
                    }
#pragma unroll
                    for (int i = 0; i < kPpWarps; ++i) {
                        if (i < k || i >= ks) continue;
                        // no splat of the sub-range meets the stop rule from this T
                        const float4 q = sh.part[i][lane];
                        cr += T * q.x;
                        cg += T * q.y;
                        cb += T * q.z;
                        T *= q.w;
                    }
                    if (ks == kPpWarps) break;
                    k = ks + 1;
                    // the stop falls inside sub-range ks: composite it from the true T
                    uint32_t mk = sh.m[ks];
                    while (mk) {
                        const int j = __ffs(mk) - 1;
                        mk &= mk - 1;
                        const float alpha = staged_alpha<true>(sh.s0[ks][j], sh.s1[ks][j], fpx, fpy);
                        const float Tn = T * (1.0f - alpha);
                        if (Tn < 1e-4f) {
                            done = true;
                            break;
                        }
                        const float4 col = sh.s2[ks][j];
                        const float wgt = alpha * T;
                        cr += col.x * wgt;
                        cg += col.y * wgt;
                        cb += col.z * wgt;
                        T = Tn;
                    }
                }
                const uint32_t dm = __ballot_sync(0xffffffffu, done);
                if (lane == 0) sh.done = dm;
            }
            __syncthreads();
        }
        if (warp == 0) {
            bool final_out = true;
            const int slot = end1 < rg.y ? work.cand_slot[tile] : -1;
            if (end1 < rg.y && in_bounds(slot >= 0, kChkSlot)) {
                // pairs remain: the state for pass 2 and the merge, as pass 1 records it
                const bool all = __all_sync(0xffffffffu, done);
                if (lane == 0 && !all) atomicAnd(work.cand_done + slot, 0u);
                work.state[(size_t)slot * kBlendThreads + blk * 32 + lane] = make_float4(cr, cg, cb, done ? -T : T);
                final_out = all;
            }
            if (final_out && inside) out[(size_t)py * W + px] = make_float4(cr, cg, cb, 1.0f - T);
        }
        __syncthreads();  // the item fields and the staging buffers are reused by the next item
    }
}

// Merge of one 8x4 block: the state at the budget, then the chunks in depth
// order, per pixel, up to the chunk in which the pixel meets the stop rule:
// such pixels keep their state before that chunk (in work.state) and its
// index (work.stop) for the fix-up pass; the others are final.  The partials
// are read past L1: other CTAs wrote them.
template <bool kTrain>
__device__ __forceinline__ void merge_block(const BlockGeom &g, size_t pix, const uint2 rg, uint32_t c0, uint32_t c1, int W,
                                            float4 *__restrict__ out, const BlendWork &work) {
    const float4 s1 = work.state[pix];
    float T = fabsf(s1.w), r = s1.x, gg = s1.y, b = s1.z;
    bool done = !g.inside || s1.w < 0.0f;
    uint32_t last = kTrain ? work.slast[pix] : 0u;
    int32_t stop = -1;
    // four chunks' partials loaded at a time (independent loads), applied in order
    for (uint32_t w0 = c0; w0 < c1 && !done; w0 += 4) {
        float4 pk[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            pk[i] = w0 + i < c1 ? __ldcg(work.part + (size_t)(w0 + i) * kBlendThreads + threadIdx.x)
                                : make_float4(0.f, 0.f, 0.f, 1.f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (done || w0 + i >= c1) break;
            if (kTrain) store_boundary(work, rg.x, rg.x + work.budget + (w0 + i - c0) * kChunk, (int)threadIdx.x, make_float4(r, gg, b, T));
            const float Tk = fabsf(pk[i].w);
            if (T * Tk >= 1e-4f) {
                // no splat of the chunk reaches the stop rule from this T: the
                // chunk's composite applies as a whole
                r += T * pk[i].x;
                gg += T * pk[i].y;
                b += T * pk[i].z;
                T *= Tk;
                if (kTrain) {
                    const uint32_t lk = __ldcg(work.last + (size_t)(w0 + i) * kBlendThreads + threadIdx.x);
                    if (lk) last = lk;
                }
                done = pk[i].w < 0.0f;
            } else {
                stop = (int32_t)(w0 + i);
                done = true;
            }
        }
    }
    work.stop[pix] = stop;
    if (stop >= 0) {
        work.state[pix] = make_float4(r, gg, b, T);
        if (kTrain) work.slast[pix] = last;
    } else if (g.inside) {
        out[(size_t)g.py * W + g.px] = make_float4(r, gg, b, 1.0f - T);
        if (kTrain) store_final(work, (size_t)g.py * W + g.px, last, make_float4(r, gg, b, T));
    }
}

// Chunk c of a tile's pairs past the budget, from T = 1, for the pixels still
// open; a warp per block.  Writes (r, g, b, T) with T negated when the chunk
// met the stop rule.  The warp that finishes a block's last chunk (a ticket
// per block, counted in the first word of its work.stop, which the plan
// cleared) merges the block: as a kernel of its own the merge started when
// the last chunk of the frame was done.  One avatar of 202,738 Gaussians at
// 720p 338 -> 334 us a frame, 5,000 characters 2,139 -> 2,124 us, training
// 64 x 65,536 at 512x512 1,882 -> 1,868 us.
template <bool kTrain>
__global__ void __launch_bounds__(kBlendThreads, kWalkCtas) k_blend_chunks(int tiles_x, int W, int H,
                                                                           const uint2 *__restrict__ ranges,
                                                                           const uint32_t *__restrict__ pval,
                                                                           const float4 *__restrict__ rec,
                                                                           float4 *__restrict__ out, BlendWork work) {
    __shared__ HitStage st[kBlocks];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // chunk w of the frame, grid-stride (the grid is capped, not sized for
    // the worst case)
    for (uint32_t w = blockIdx.x; w < (uint32_t)work.meta[1]; w += gridDim.x) {
        const int slot = work.chunk_slot[w];
        if (work.cand_done[slot]) continue;
        const int tile = work.cand_tile[slot];
        const BlockGeom g = block_geom(tile, warp, tiles_x, W, H, work.ox, work.oy);
        const uint2 rg = ranges[tile];
        if (!in_bounds(rg.y <= work.n_pairs, kChkPair)) continue;
        const uint32_t c0 = work.cand_chunk0[slot], start = rg.x + work.budget + (w - c0) * kChunk;
        const size_t pix = (size_t)slot * kBlendThreads + threadIdx.x;
        const bool open = g.inside && work.state[pix].w >= 0.0f;
        Pixel px = make_pixel(g.fpx, g.fpy, open, make_float4(0.f, 0.f, 0.f, 1.f), 0u);
        warp_walk<kTrain ? kTraining : kPlain>(st[warp], start, min(rg.y, start + kChunk), pval, rec, g.bx0, g.by0, px,
                                               work, false);
        work.part[(size_t)w * kBlendThreads + threadIdx.x] = pixel_state(px, open && closed(px) ? -px.T : px.T);
        if (kTrain) work.last[(size_t)w * kBlendThreads + threadIdx.x] = px.last;
        __threadfence();  // the partials before the ticket
        __syncwarp();     // (also: the staging buffer is reused by the next chunk)
        const uint32_t chunks = (rg.y - rg.x - work.budget + kChunk - 1) / kChunk;
        uint32_t ticket = 0;
        if (lane == 0) ticket = atomicAdd(reinterpret_cast<unsigned *>(work.stop + pix), 1u);
        if (__shfl_sync(0xffffffffu, ticket, 0) == chunks - 1u) {
            __threadfence();
            merge_block<kTrain>(g, pix, rg, c0, c0 + chunks, W, out, work);
        }
    }
}

// Fix-up: chunk w composited again, from their true transmittance, for the
// pixels that meet the stop rule inside it.
template <bool kTrain>
__global__ void __launch_bounds__(kBlendThreads, kWalkCtas) k_blend_fix(int tiles_x, int W, int H,
                                                                        const uint2 *__restrict__ ranges,
                                                                        const uint32_t *__restrict__ pval,
                                                                        const float4 *__restrict__ rec,
                                                                        float4 *__restrict__ out, BlendWork work) {
    __shared__ HitStage st[kBlocks];
    const int warp = threadIdx.x >> 5;
    for (uint32_t w = blockIdx.x; w < (uint32_t)work.meta[1]; w += gridDim.x) {
        const int slot = work.chunk_slot[w];
        if (work.cand_done[slot]) continue;
        const size_t sp = (size_t)slot * kBlendThreads + threadIdx.x;
        const bool mine = work.stop[sp] == (int32_t)w;
        if (!__any_sync(0xffffffffu, mine)) continue;
        const int tile = work.cand_tile[slot];
        const BlockGeom g = block_geom(tile, warp, tiles_x, W, H, work.ox, work.oy);
        const uint2 rg = ranges[tile];
        if (!in_bounds(rg.y <= work.n_pairs, kChkPair)) continue;
        Pixel px = make_pixel(g.fpx, g.fpy, mine, mine ? work.state[sp] : make_float4(0.f, 0.f, 0.f, 1.f),
                              kTrain && mine ? work.slast[sp] : 0u);
        const uint32_t start = rg.x + work.budget + (w - work.cand_chunk0[slot]) * kChunk;
        warp_walk<kTrain ? kTraining : kPlain>(st[warp], start, min(rg.y, start + kChunk), pval, rec, g.bx0, g.by0, px,
                                               work, false);
        if (mine && g.inside) {
            const size_t pix = (size_t)g.py * W + g.px;
            out[pix] = pixel_state(px, 1.0f - px.T);
            if (kTrain) store_final(work, pix, px.last, pixel_state(px, px.T));
        }
        __syncwarp();  // the staging buffer is reused by the next chunk
    }
}

// Plan, part 1 (one thread per tile; meta zeroed before): tiles per list
// length class (warp-aggregated atomics), and a slot plus
// ceil((n - budget) / kChunk) consecutive chunks for every tile with more
// than budget pairs.  Slot and chunk numbers depend on the order of the
// atomics; no result does (a tile's chunks are consecutive and merged in
// order).
__global__ void __launch_bounds__(256) k_blend_count(int n_tiles, const uint2 *__restrict__ ranges, BlendWork work) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const uint32_t n = t < n_tiles ? ranges[t].y - ranges[t].x : 0u;
    const int cls = t < n_tiles ? blend_class(n) : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, cls);
    if (cls >= 0 && lane == __ffs(peers) - 1) atomicAdd(work.meta + kBlendCountAt + cls, __popc(peers));
    if (t >= n_tiles) return;
    int slot = -1;
    if (n > work.budget) {
        const uint32_t nk = (n - work.budget + kChunk - 1) / kChunk;
        slot = atomicAdd(work.meta + 0, 1);
        const uint32_t c0 = atomicAdd(reinterpret_cast<unsigned *>(work.meta + 1), nk);
        if (in_bounds((uint32_t)slot < work.max_slots && c0 + nk <= work.max_chunks, kChkSlot)) {
            work.cand_tile[slot] = t;
            work.cand_chunk0[slot] = c0;
            work.cand_done[slot] = 1u;  // cleared unless every pixel is closed
            // the blocks' chunk tickets
            for (int b = 0; b < kBlocks; ++b) work.stop[(size_t)slot * kBlendThreads + 32 * b] = 0;
            for (uint32_t c = 0; c < nk; ++c) work.chunk_slot[c0 + c] = slot;
        } else {
            slot = -1;
        }
    }
    work.cand_slot[t] = slot;
}

// Plan, part 2: pp_tile in decreasing schedule key (the order inside a key
// is that of the atomics and affects no result).
__global__ void __launch_bounds__(256) k_blend_order(int n_tiles, const uint2 *__restrict__ ranges, int pp_ctas,
                                                     BlendWork work) {
    __shared__ int seg_tile[kBlendKeys + 1];  // first tile of key kBlendKeys - 1 - s
    __shared__ bool tiles;
    if (threadIdx.x < 32) {
        const bool t_ = key_segments(work.meta, pp_ctas, work.items, nullptr, seg_tile);
        if (threadIdx.x == 0) tiles = t_;
    }
    __syncthreads();
    const int t = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const int cls = t < n_tiles ? blend_class(ranges[t].y - ranges[t].x) : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, cls);
    const int leader = __ffs(peers) - 1;
    int pos = 0;
    if (cls >= 0 && lane == leader) pos = atomicAdd(work.meta + kBlendCursorAt + cls, __popc(peers));
    pos = __shfl_sync(0xffffffffu, pos, leader) + __popc(peers & ((1u << lane) - 1u));
    if (cls >= 0) work.pp_tile[seg_tile[kBlendKeys - 1 - blend_key(cls, tiles)] + pos] = t;
}

// Persistent grid of the pair-parallel pass: as many CTAs as fit on the
// device at once.
static unsigned pp_grid() {
    static int cached_device = -1;
    static unsigned grid = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != cached_device) {
        int sms = 0, per_sm = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_blend_pp, kPpThreads, 0);
        grid = (unsigned)std::max(1, sms * std::max(1, per_sm));
        cached_device = dev;
    }
    return grid;
}

// The plan's kernels: tile classes, slots and chunks, then the tile order.
static int launch_plan(int n, const uint2 *ranges, const BlendWork &work, cudaStream_t st) {
    const unsigned tb = (unsigned)((n + 255) / 256);
    k_blend_count<<<tb, 256, 0, st>>>(n, ranges, work);
    k_blend_order<<<tb, 256, 0, st>>>(n, ranges, (int)pp_grid(), work);
    return 2;
}

// The split passes (nothing when no list is longer than the budget).
template <bool kTrain>
static int launch_split(int tiles_x, int W, int H, const uint2 *ranges, const uint32_t *pval, const float4 *rec,
                        float4 *out, const BlendWork &work, cudaStream_t st) {
    if (work.n_pairs <= work.budget) return 0;
    // chunk grids capped at kChunkGrid CTAs (grid-stride over the frame's
    // chunks): a frame whose lists all end within the budget does not pay for
    // a worst-case grid of CTAs that return at once
    const unsigned chunk_grid = (unsigned)std::min<size_t>(work.max_chunks, kChunkGrid);
    k_blend_chunks<kTrain><<<chunk_grid, kBlendThreads, 0, st>>>(tiles_x, W, H, ranges, pval, rec, out, work);
    k_blend_fix<kTrain><<<chunk_grid, kBlendThreads, 0, st>>>(tiles_x, W, H, ranges, pval, rec, out, work);
    return 2;
}

int launch_blend(int tiles_x, int tiles_y, int W, int H, const uint2 *ranges, const uint32_t *pval,
                 const float4 *rec, float4 *out, const BlendWork &work, cudaStream_t st) {
    const int n = tiles_x * tiles_y;
    if (n <= 0) return 0;
    BlendWork w = work;
    if (work.contrib || work.px_end) w.items = CS_BLEND_ITEMS_BLOCKS;  // tiles by decreasing list length class
    int launched = launch_plan(n, ranges, w, st);
    if (work.contrib) {
        // statistics: every list walked to its end
        k_blend_walk<kStats><<<n, kBlendThreads, 0, st>>>(tiles_x, W, H, ranges, pval, rec, out, w);
        return launched + 1;
    }
    if (work.px_end) {
        k_blend_walk<kTraining><<<n, kBlendThreads, 0, st>>>(tiles_x, W, H, ranges, pval, rec, out, w);
        return launched + 1 + launch_split<true>(tiles_x, W, H, ranges, pval, rec, out, w, st);
    }
    // pass 1 of every tile: persistent CTAs, longest chains first
    k_blend_pp<<<pp_grid(), kPpThreads, 0, st>>>(tiles_x, W, H, ranges, pval, rec, out, w);
    return launched + 1 + launch_split<false>(tiles_x, W, H, ranges, pval, rec, out, w, st);
}

CS_DEFINE_CHECK_READER(check_word_blend)

}  // namespace cs
