// Gradients of a rendered frame: reverse-mode through compositing, EWA
// projection, SH colour, linear blend skinning and forward kinematics.
//
// The loss enters as dL/d(pixel RGBA).  Kernels, in order:
//   k_blend_backward     one CTA per chunk of kBwdChunk pairs of a 16x16
//                        tile's list: each pixel walks its contributors in
//                        the chunk back to front (recomputing alpha, and the
//                        transmittance from the state the forward kept at the
//                        chunk's end, or from its final state), producing
//                        per splat the moments that give dL/d(u, v, conic,
//                        opacity) and dL/d(rgb), summed over each warp's
//                        pixels before the atomic adds; the chunks of one
//                        list run in parallel
//   k_project_backward   one CTA per (instance, 256 Gaussians), like the
//                        forward projection: recompute, then the chain rule to
//                        the template mean, canonical covariance, opacity and
//                        SH coefficients (summed over instances) and to the
//                        instance's 24 skinning transforms (summed in shared
//                        memory per CTA)
//   k_fk_backward        one warp per instance: skinning transforms to the
//                        24 axis-angle joint rotations
//   k_cov_backward       one thread per template Gaussian: its summed
//                        gradients to the caller's arrays, canonical
//                        covariance to scales and quaternion
// Every step differentiates the forward as written (3DGS conventions, the
// readings of the forward kernels); clamps (alpha at 0.99, the EWA x/z and
// y/z limits, colour at 0) pass no gradient where active, and the discrete
// decisions (support box, alpha >= 1/255, the stop rule, the radius) are held
// fixed.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "cs_internal.cuh"

namespace cs {

namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr int kBwdThreads = 256;
constexpr int kBlockW = kBlendBlockW, kBlockH = kBlendBlockH;  // the forward's pixels per warp

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---------------------------------------------------------------------------
// compositing backward
// ---------------------------------------------------------------------------

// Backward chunks of each tile's list: ceil(n / kBwdChunk).
__global__ void __launch_bounds__(256) k_bwd_chunk_counts(int n_tiles, const uint2 *__restrict__ ranges,
                                                          uint32_t *__restrict__ cnt) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_tiles) cnt[t] = (ranges[t].y - ranges[t].x + kBwdChunk - 1) / kBwdChunk;
}

// The last t in [0, n) with first[t] <= w (first ascends from 0), 32 probes
// at a time by the whole warp.
__device__ __forceinline__ int last_at_most(const uint32_t *__restrict__ first, int n, uint32_t w) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) / 32, i = lo + lane * step;
        const int below = __popc(__ballot_sync(0xffffffffu, i < hi && first[i] <= w));
        lo += (below - 1) * step;
        hi = min(hi, lo + step);
    }
    return lo;
}

constexpr int kBwdHits = 3;   // hits whose gradients are summed together
constexpr int kBwdGrads = 9;  // sums per splat (see dsplat)
constexpr int kBwdRows = kBwdHits * kBwdGrads, kBwdLd = 36;
static_assert(kBwdRows <= 32, "one lane per row");

// One warp's splats of 32 pairs and the rows it sums over its 32 pixels.
// Rows are 36 floats apart: eight lanes' 16-byte loads of eight rows fall in
// different banks.
struct BwdWarp {
    float4 s0[32];  // u, v, a', b' (the forward's scaled conic)
    float4 s1[32];  // c', log2 o, radius, splat id (bits)
    float4 s2[32];  // r, g, b, pair index (bits)
    float rows[kBwdRows][kBwdLd];
};

// Adds the sums of the first n rows to dsplat; row l, taken by lane l, is sum
// l % kBwdGrads of the splat the lane names.  (The address needs 64 bits: a
// frame may hold more than 2^32 / 12 splats.)
__device__ __forceinline__ void flush_rows(const BwdWarp &sh, int n, uint32_t splat, float *__restrict__ dsplat) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < n) {
        const float4 *r = reinterpret_cast<const float4 *>(sh.rows[lane]);
        float4 t = r[0];
#pragma unroll
        for (int i = 1; i < 8; ++i) {
            const float4 v = r[i];
            t.x += v.x;
            t.y += v.y;
            t.z += v.z;
            t.w += v.w;
        }
        const float x = (t.x + t.y) + (t.z + t.w);
        if (x != 0.0f) atomicAdd(dsplat + (size_t)splat * 12u + lane % kBwdGrads, x);
    }
    __syncwarp();
}

// A CTA per chunk of kBwdChunk pairs, a warp per 8x4 block of the tile; the
// warps share nothing, so none waits at a CTA barrier.  A warp walks its
// block's pairs back to front, 32 at a time (only those whose reach box
// meets the block are staged), recomputing alpha with the forward's
// expressions.  Each pixel gives a splat nine terms: with G = dL/dalpha alpha
// (0 where alpha is clamped) the moments G, G dx, G dy, G dx^2, G dx dy,
// G dy^2, from which the projection backward takes the gradients of opacity,
// mean and conic, and dL/d(r, g, b).
// The rows of three splats are summed through shared memory (27 stores, 8
// loads and 32 adds per lane), a third of the instructions of a butterfly of
// shuffles per splat.  Bound by instruction issue; 65,536 Gaussians x 64
// instances, 512x512: 1.08 -> 0.44 ms against CTAs of eight warps in step with
// butterflies and shared-memory atomics.
__global__ void __launch_bounds__(kBwdThreads, 5) k_blend_backward(
    int tiles_x, int W, int H, const uint2 *__restrict__ ranges, const uint32_t *__restrict__ pval,
    const float4 *__restrict__ rec, const uint32_t *__restrict__ px_end, const float4 *__restrict__ px_fin,
    const float4 *__restrict__ px_bnd, const uint32_t *__restrict__ chunk0, int n_tiles,
    const float4 *__restrict__ dl_drgba, float *__restrict__ dsplat) {
    __shared__ BwdWarp shared[kBwdThreads / 32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    BwdWarp &sh = shared[warp];
    // chunk w of the frame: the tile whose chunks [chunk0[t], chunk0[t + 1]) hold it
    const uint32_t w = blockIdx.x;
    if (w >= chunk0[n_tiles]) return;
    const int tile = last_at_most(chunk0, n_tiles, w);
    // pixel layout of the forward: warp w covers an 8x4 block
    const int bx0 = (tile % tiles_x) * kTile + (warp & 1) * kBlockW, by0 = (tile / tiles_x) * kTile + (warp >> 1) * kBlockH;
    const int px = bx0 + (lane % kBlockW), py = by0 + (lane / kBlockW);
    const float fpx = (float)px + 0.5f, fpy = (float)py + 0.5f;
    const uint2 rg = ranges[tile];
    // this chunk: pairs [lo, hi) of the tile's list
    const uint32_t lo = rg.x + (w - chunk0[tile]) * kBwdChunk, hi = min(rg.y, lo + kBwdChunk);
    uint32_t end = lo;
    float Tf = 1.0f;
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
    float T = 1.0f;                      // transmittance behind the current splat
    float Sr = 0.f, Sg = 0.f, Sb = 0.f;  // colour composited behind it
    if (px < W && py < H) {
        const size_t p = (size_t)py * W + px;
        const uint32_t e = px_end[p];
        end = min(e, hi);
        if (end > lo) {
            const float4 fin = px_fin[p];
            Tf = fin.w;
            g = dl_drgba[p];
            if (e <= hi) {
                // the pixel's list ends in this chunk: the walk starts from its final state
                T = Tf;
            } else {
                // it goes on past the chunk: the state the forward kept at hi, and
                // the colour composited behind it (final minus in front of it)
                const float4 st = px_bnd[(size_t)(hi / kBwdChunk) * kBwdThreads + tid];
                T = st.w;
                Sr = fin.x - st.x;
                Sg = fin.y - st.y;
                Sb = fin.z - st.z;
            }
        }
    }
    const uint32_t top = __reduce_max_sync(0xffffffffu, end);
    int n_rows = 0;
    uint32_t splat = 0u;  // of the lane's row
    uint32_t base = lo + ((top - 1u - lo) & ~31u);
    uint32_t i = base + (uint32_t)lane;
    if (top <= lo) return;
    uint32_t s = i < top ? __ldg(pval + i) : 0u;
    for (;;) {
        const bool more = base > lo;
        const uint32_t s_next = more ? __ldg(pval + i - 32) : 0u;  // the batch before, while this one is walked
        bool mine = false;
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < top) {
            q = __ldg(rec + (size_t)s * kRecVec);
            const uint32_t rx = __float_as_uint(q.x), ry = __float_as_uint(q.y);
            mine = (int)(rx & 0xFFFFu) <= bx0 + kBlockW - 1 && (int)(rx >> 16) >= bx0 &&
                   (int)(ry & 0xFFFFu) <= by0 + kBlockH - 1 && (int)(ry >> 16) >= by0;
        }
        const uint32_t m = __ballot_sync(0xffffffffu, mine);
        if (mine) {
            const float4 a = __ldg(rec + (size_t)s * kRecVec + 1), c = __ldg(rec + (size_t)s * kRecVec + 2);
            const int pos = __popc(m & ((1u << lane) - 1u));
            sh.s0[pos] = make_float4(a.x, a.y, -0.5f * kLog2e * a.z, -kLog2e * a.w);
            sh.s1[pos] = make_float4(-0.5f * kLog2e * q.w, q.z, c.w, __uint_as_float(s));
            sh.s2[pos] = make_float4(c.x, c.y, c.z, __uint_as_float(i));
        }
        __syncwarp();
#pragma unroll 1
        for (int k = __popc(m) - 1; k >= 0; --k) {
            const float4 a = sh.s0[k], b = sh.s1[k], c = sh.s2[k];
            // the forward's tests, evaluated the same way
            const float dx = fpx - a.x, dy = fpy - a.y;
            const float p = __fmaf_rn(__fmul_rn(b.x, dy), dy, __fmul_rn(dx, __fmaf_rn(a.w, dy, __fmul_rn(a.z, dx))));
            const float araw = ex2_approx(p + b.y), alpha = fminf(0.99f, araw);
            const bool takes = __float_as_uint(c.w) < end && fmaxf(fabsf(dx), fabsf(dy)) <= b.z && p <= 0.0f &&
                               alpha >= (1.0f / 255.0f);
            if (!__any_sync(0xffffffffu, takes)) continue;
            float G = 0.f, gr = 0.f, gg = 0.f, gb = 0.f;
            if (takes) {
                // one reciprocal of 1 - alpha for the five quotients (off by
                // an ulp from dividing each): the walk back divides T by it
                // at every splat, so the chain waits on a multiply only
                const float iom = 1.0f / (1.0f - alpha);
                const float Tb = T * iom;  // transmittance in front of this splat
                const float wgt = alpha * Tb;
                gr = wgt * g.x;
                gg = wgt * g.y;
                gb = wgt * g.z;
                // d pixel / d alpha: own colour minus what it hides, and the alpha channel
                const float galpha = g.x * (c.x * Tb - Sr * iom) + g.y * (c.y * Tb - Sg * iom) +
                                     g.z * (c.z * Tb - Sb * iom) + g.w * (Tf * iom);
                Sr += c.x * wgt;
                Sg += c.y * wgt;
                Sb += c.z * wgt;
                T = Tb;
                if (araw < 0.99f) G = galpha * araw;
            }
            const float Gx = G * dx, Gy = G * dy;
            const float v[kBwdGrads] = {G, Gx, Gy, Gx * dx, Gx * dy, Gy * dy, gr, gg, gb};
#pragma unroll
            for (int e = 0; e < kBwdGrads; ++e) sh.rows[n_rows + e][lane] = v[e];
            if ((uint32_t)(lane - n_rows) < (uint32_t)kBwdGrads) splat = __float_as_uint(b.w);
            n_rows += kBwdGrads;
            if (n_rows == kBwdRows) {
                flush_rows(sh, kBwdRows, splat, dsplat);
                n_rows = 0;
            }
        }
        if (!more) break;
        __syncwarp();  // the staging buffer is refilled by the next batch
        base -= 32u;
        i -= 32u;
        s = s_next;
    }
    flush_rows(sh, n_rows, splat, dsplat);
}

// ---------------------------------------------------------------------------
// projection backward
// ---------------------------------------------------------------------------

// Real SH basis to degree 3 (3DGS signs) and its gradient with respect to
// the (unnormalised) direction components, from the polynomials.
template <int deg>
__device__ __forceinline__ void sh_basis_grad(float x, float y, float z, float Y[16], float dY[16][3]) {
    const float C0 = 0.28209479177387814f, C1 = 0.4886025119029199f;
    const float A2 = 1.0925484305920792f, B2 = 0.31539156525252005f, E2 = 0.5462742152960396f;
    const float K0 = 0.5900435899266435f, K1 = 2.890611442640554f, K2 = 0.4570457994644658f;
    const float K3 = 0.3731763325901154f, K5 = 1.445305721320277f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        Y[k] = 0.f;
        dY[k][0] = dY[k][1] = dY[k][2] = 0.f;
    }
    Y[0] = C0;
    if (deg < 1) return;
    Y[1] = -C1 * y; dY[1][1] = -C1;
    Y[2] = C1 * z;  dY[2][2] = C1;
    Y[3] = -C1 * x; dY[3][0] = -C1;
    if (deg < 2) return;
    const float xx = x * x, yy = y * y, zz = z * z;
    Y[4] = A2 * x * y;  dY[4][0] = A2 * y; dY[4][1] = A2 * x;
    Y[5] = -A2 * y * z; dY[5][1] = -A2 * z; dY[5][2] = -A2 * y;
    Y[6] = B2 * (2.f * zz - xx - yy); dY[6][0] = -2.f * B2 * x; dY[6][1] = -2.f * B2 * y; dY[6][2] = 4.f * B2 * z;
    Y[7] = -A2 * x * z; dY[7][0] = -A2 * z; dY[7][2] = -A2 * x;
    Y[8] = E2 * (xx - yy); dY[8][0] = 2.f * E2 * x; dY[8][1] = -2.f * E2 * y;
    if (deg < 3) return;
    Y[9] = -K0 * y * (3.f * xx - yy);
    dY[9][0] = -6.f * K0 * x * y; dY[9][1] = -3.f * K0 * (xx - yy);
    Y[10] = K1 * x * y * z;
    dY[10][0] = K1 * y * z; dY[10][1] = K1 * x * z; dY[10][2] = K1 * x * y;
    Y[11] = -K2 * y * (4.f * zz - xx - yy);
    dY[11][0] = 2.f * K2 * x * y; dY[11][1] = -K2 * (4.f * zz - xx - 3.f * yy); dY[11][2] = -8.f * K2 * y * z;
    Y[12] = K3 * z * (2.f * zz - 3.f * xx - 3.f * yy);
    dY[12][0] = -6.f * K3 * x * z; dY[12][1] = -6.f * K3 * y * z; dY[12][2] = K3 * (6.f * zz - 3.f * xx - 3.f * yy);
    Y[13] = -K2 * x * (4.f * zz - xx - yy);
    dY[13][0] = -K2 * (4.f * zz - 3.f * xx - yy); dY[13][1] = 2.f * K2 * x * y; dY[13][2] = -8.f * K2 * x * z;
    Y[14] = K5 * z * (xx - yy);
    dY[14][0] = 2.f * K5 * x * z; dY[14][1] = -2.f * K5 * y * z; dY[14][2] = K5 * (xx - yy);
    Y[15] = -K0 * x * (xx - 3.f * yy);
    dY[15][0] = -3.f * K0 * (xx - yy); dY[15][1] = 6.f * K0 * x * y;
}

// One 16-byte global reduction (no value returned).
__device__ __forceinline__ void red4(float *p, float x, float y, float z, float w) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

// Colour of Gaussian gsrc seen along the unit direction d: adds dL/d(SH) to
// gsh and returns dL/dd.  The coefficient planes are read twice (the second
// time from L1): keeping all 48 would cost a third of the CTAs in registers.
template <int DEG>
__device__ __forceinline__ void sh_backward(const float4 *__restrict__ sh, int n, const float d[3], const float c[3],
                                            float *__restrict__ gsh, bool vec, float gd[3]) {
    constexpr int K = (DEG + 1) * (DEG + 1), P = (K * 3 + 3) / 4;
    float Y[16], dY[16][3];
    sh_basis_grad<DEG>(d[0], d[1], d[2], Y, dY);
    float pre[3] = {0.5f, 0.5f, 0.5f};
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const float4 v = __ldg(sh + (int64_t)p * n);
        const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (4 * p + q < 3 * K) pre[(4 * p + q) % 3] += Y[(4 * p + q) / 3] * e[q];
    }
    // colour clamp at 0 passes no gradient
    const float gc[3] = {pre[0] > 0.f ? c[0] : 0.f, pre[1] > 0.f ? c[1] : 0.f, pre[2] > 0.f ? c[2] : 0.f};
    gd[0] = gd[1] = gd[2] = 0.f;
    if (gc[0] == 0.f && gc[1] == 0.f && gc[2] == 0.f) return;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const float4 v = __ldg(sh + (int64_t)p * n);
        const float e[4] = {v.x, v.y, v.z, v.w};
        float g[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int f = 4 * p + q;
            if (f >= 3 * K) continue;
            g[q] = Y[f / 3] * gc[f % 3];
            // (a channel without gradient adds nothing, whatever its coefficients)
            const float cf = gc[f % 3] != 0.f ? e[q] * gc[f % 3] : 0.f;
            gd[0] += cf * dY[f / 3][0];
            gd[1] += cf * dY[f / 3][1];
            gd[2] += cf * dY[f / 3][2];
        }
        if (vec) {
            red4(gsh + 4 * p, g[0], g[1], g[2], g[3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (4 * p + q < 3 * K) atomicAdd(gsh + 4 * p + q, g[q]);
        }
    }
}

constexpr int kBwdAcc = 12;  // per Gaussian: mean (3), opacity, canonical covariance (6), two unused
constexpr int kWLd = 25;     // skinning weights of a splat, dense over the joints (odd row: conflict free)
struct ProjBwdShared {
    float4 B[kJoints * 3];
    float W[kBwdThreads][kWLd];
    float4 M[kBwdThreads][3];  // dL/d(blended transform)
    uint16_t active[kBwdThreads];
    int n;
};

// A CTA per (visible instance, 256 Gaussians of its level).  Most of a
// crowd's splats are hidden and have no gradient: the CTA lists the ones
// that do and its first threads take them, so that the chain rule runs in
// full warps.  Template gradients go out as 16-byte reductions; the sums
// over the CTA's splats of w_j dM, dense in the 24 joints, are a small
// matrix product in shared memory, one 16-byte reduction per result.
// Bound by the latency of the chain rule in the few warps with work.  65,536
// Gaussians x 64 instances, 512x512: 1.18 -> 0.25 ms against one thread per
// splat (7 of 32 lanes active), 58 scalar global atomics per splat and 48
// contended shared-memory atomics per splat.
__global__ void __launch_bounds__(kBwdThreads, 3) k_project_backward(
    const Group *__restrict__ groups, int n_groups, const int32_t *__restrict__ vis, const float *__restrict__ Bm,
    const float *__restrict__ Vm, const float *__restrict__ Cloc, const float *__restrict__ root, TemplateArrays ta,
    const TemplateInfo *__restrict__ tpls, CamParams cam, LodParams lod, int skin_mode, int sh_frame,
    const float4 *__restrict__ rec, const float4 *__restrict__ dsplat, float *__restrict__ g_acc,
    float *__restrict__ g_sh, bool vec_sh, float *__restrict__ g_B) {
    extern __shared__ __align__(16) unsigned char proj_bwd_dyn[];
    ProjBwdShared &sh = *reinterpret_cast<ProjBwdShared *>(proj_bwd_dyn);
    __shared__ int s_group;
    const int t = threadIdx.x;
    if (t == 0) {
        int lo = 0, hi = n_groups - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (groups[mid].block0 <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
        }
        s_group = lo;
        sh.n = 0;
    }
    __syncthreads();
    const Group G = groups[s_group];
    const int per_inst = (G.ng + kBwdThreads - 1) / kBwdThreads;
    const int rb = (int)blockIdx.x - G.block0;
    const int islot = rb / per_inst;
    const int g0 = (rb - islot * per_inst) * kBwdThreads;
    const int inst = vis[G.slot0 + islot];
    const size_t s0 = (size_t)G.splat0 + (size_t)islot * G.ng + g0;  // first splat of the CTA
    {
        bool any = false;
        if (g0 + t < G.ng) {
            const float4 *d = dsplat + (s0 + t) * 3;
            const float4 a = d[0], b = d[1];
            any = a.x != 0.f || a.y != 0.f || a.z != 0.f || a.w != 0.f || b.x != 0.f || b.y != 0.f || b.z != 0.f ||
                  b.w != 0.f || d[2].x != 0.f;
        }
        const unsigned m = __ballot_sync(0xffffffffu, any);
        int first = 0;
        if ((t & 31) == 0 && m) first = atomicAdd(&sh.n, __popc(m));
        first = __shfl_sync(0xffffffffu, first, 0);
        if (any) sh.active[first + __popc(m & ((1u << (t & 31)) - 1u))] = (uint16_t)t;
        const float4 *Bi = reinterpret_cast<const float4 *>(Bm + (size_t)inst * kJoints * 12);
        for (int k = t; k < kJoints * 3; k += kBwdThreads) sh.B[k] = __ldg(Bi + k);
    }
    __syncthreads();
    const int n = sh.n;
    if (n == 0) return;
    if (t < n) {
        const int gg = g0 + sh.active[t];
        const size_t s = s0 + sh.active[t];
        const float4 m0 = dsplat[s * 3], m1 = dsplat[s * 3 + 1];  // G, G dx, G dy, G dx^2 | G dx dy, G dy^2, dr, dg
        const float db = dsplat[s * 3 + 2].x;
        const float4 rq = __ldg(rec + s * kRecVec), ra = __ldg(rec + s * kRecVec + 1);
        // from the moments: opacity (alpha = o e^q), mean and conic
        const float go = m0.x * exp2f(-rq.z);
        const float gu = ra.z * m0.y + ra.w * m0.z, gv = ra.w * m0.y + rq.w * m0.z;
        const TemplateInfo &T = tpls[G.tpl];
        const int sub = T.lod_idx_off[G.lvl];
        const int gsrc = sub >= 0 ? (int)__ldg(ta.lod_idx + sub + gg) : gg;
        const int gi = T.g_off + gsrc;
        // ---- recompute the forward ---------------------------------------
        const float4 w = __ldg(ta.skin_w + gi);
        const uint32_t packed = __ldg(ta.skin_i + gi);
        const float wk[4] = {w.x, w.y, w.z, w.w};
        int jk[4];
        float M[12];
#pragma unroll
        for (int e = 0; e < 12; ++e) M[e] = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            jk[k] = (packed >> (8 * k)) & 0xFF;
            const float4 b0 = sh.B[jk[k] * 3 + 0], b1 = sh.B[jk[k] * 3 + 1], b2 = sh.B[jk[k] * 3 + 2];
            M[0] += wk[k] * b0.x; M[1] += wk[k] * b0.y; M[2] += wk[k] * b0.z; M[3] += wk[k] * b0.w;
            M[4] += wk[k] * b1.x; M[5] += wk[k] * b1.y; M[6] += wk[k] * b1.z; M[7] += wk[k] * b1.w;
            M[8] += wk[k] * b2.x; M[9] += wk[k] * b2.y; M[10] += wk[k] * b2.z; M[11] += wk[k] * b2.w;
        }
        const float4 mo = __ldg(ta.mean_op + gi);
        const float mu[3] = {mo.x, mo.y, mo.z};
        float pl[3];  // posed mean, instance local
#pragma unroll
        for (int r = 0; r < 3; ++r) pl[r] = M[r * 4] * mu[0] + M[r * 4 + 1] * mu[1] + M[r * 4 + 2] * mu[2] + M[r * 4 + 3];
        const float4 *Vi = reinterpret_cast<const float4 *>(Vm + (size_t)inst * 12);
        const float4 v0 = __ldg(Vi), v1 = __ldg(Vi + 1), v2 = __ldg(Vi + 2);
        const float VR[9] = {v0.x, v0.y, v0.z, v1.x, v1.y, v1.z, v2.x, v2.y, v2.z};
        const float tx = v0.x * pl[0] + v0.y * pl[1] + v0.z * pl[2] + v0.w;
        const float ty = v1.x * pl[0] + v1.y * pl[1] + v1.z * pl[2] + v1.w;
        const float tz = v2.x * pl[0] + v2.y * pl[1] + v2.z * pl[2] + v2.w;
        float Wm[9];  // V_R A (full skinning) or V_R (means only)
        if (skin_mode == 0) {
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    Wm[r * 3 + c] = VR[r * 3] * M[c] + VR[r * 3 + 1] * M[4 + c] + VR[r * 3 + 2] * M[8 + c];
        } else {
#pragma unroll
            for (int e = 0; e < 9; ++e) Wm[e] = VR[e];
        }
        const float4 ca = __ldg(ta.cov_a + gi);
        const float2 cb = __ldg(ta.cov_b + gi);
        const float m = lod.mult[G.lvl], m2 = m * m;
        const float Sg[9] = {ca.x * m2, ca.y * m2, ca.z * m2, ca.y * m2, ca.w * m2, cb.x * m2,
                             ca.z * m2, cb.x * m2, cb.y * m2};
        const float iz = __fdividef(1.0f, tz);
        const float rx = tx * iz, ry = ty * iz;
        const bool clx = rx < -cam.limx || rx > cam.limx, cly = ry < -cam.limy || ry > cam.limy;
        const float txz = fminf(fmaxf(rx, -cam.limx), cam.limx);
        const float tyz = fminf(fmaxf(ry, -cam.limy), cam.limy);
        const float J[6] = {cam.fx * iz, 0.f, -cam.fx * txz * iz, 0.f, cam.fy * iz, -cam.fy * tyz * iz};
        float Tm[6];  // J W
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) Tm[r * 3 + c] = J[r * 3] * Wm[c] + J[r * 3 + 1] * Wm[3 + c] + J[r * 3 + 2] * Wm[6 + c];
        float TS[6];  // T Sigma
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) TS[r * 3 + c] = Tm[r * 3] * Sg[c] + Tm[r * 3 + 1] * Sg[3 + c] + Tm[r * 3 + 2] * Sg[6 + c];
        const float a = TS[0] * Tm[0] + TS[1] * Tm[1] + TS[2] * Tm[2] + 0.3f;
        const float b = TS[0] * Tm[3] + TS[1] * Tm[4] + TS[2] * Tm[5];
        const float c = TS[3] * Tm[3] + TS[4] * Tm[4] + TS[5] * Tm[5] + 0.3f;
        const float idet = 1.0f / (a * c - b * b);
        const float QA = c * idet, QB = -b * idet, QC = a * idet;
        // ---- conic -> 2D covariance: gK = -Q gQ Q ------------------------
        const float gQA = -0.5f * m0.w, gQB = -0.5f * m1.x, gQC = -0.5f * m1.y;  // symmetric matrix of dL/dQ
        // P = gQ Q
        const float P00 = gQA * QA + gQB * QB, P01 = gQA * QB + gQB * QC;
        const float P10 = gQB * QA + gQC * QB, P11 = gQB * QB + gQC * QC;
        const float gK00 = -(QA * P00 + QB * P10), gK01 = -(QA * P01 + QB * P11);
        const float gK11 = -(QB * P01 + QC * P11);
        // G2 = dL/dK as a symmetric matrix (K = T S T^T + 0.3 I)
        const float G00 = gK00, G01 = gK01, G11 = gK11;
        // gT = 2 G2 T S  (2x3)
        float gT[6];
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) {
            gT[cc] = 2.f * (G00 * TS[cc] + G01 * TS[3 + cc]);
            gT[3 + cc] = 2.f * (G01 * TS[cc] + G11 * TS[3 + cc]);
        }
        // gS = T^T G2 T (3x3)
        float gS[9];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float u0 = G00 * Tm[i] + G01 * Tm[3 + i], u1 = G01 * Tm[i] + G11 * Tm[3 + i];
#pragma unroll
            for (int j = 0; j < 3; ++j) gS[i * 3 + j] = u0 * Tm[j] + u1 * Tm[3 + j];
        }
        // T = J W: gJ = gT W^T, gW = J^T gT
        float gJ[6], gW[9];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k = 0; k < 3; ++k) gJ[r * 3 + k] = gT[r * 3] * Wm[k * 3] + gT[r * 3 + 1] * Wm[k * 3 + 1] + gT[r * 3 + 2] * Wm[k * 3 + 2];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int cc = 0; cc < 3; ++cc) gW[k * 3 + cc] = J[k] * gT[cc] + J[3 + k] * gT[3 + cc];
        // camera-space mean: the projection u, v and the Jacobian entries
        float gtx = gu * cam.fx * iz, gty = gv * cam.fy * iz;
        float gtz = -gu * cam.fx * tx * iz * iz - gv * cam.fy * ty * iz * iz;
        gtz += -gJ[0] * cam.fx * iz * iz - gJ[4] * cam.fy * iz * iz;
        if (!clx) {
            gtx += -gJ[2] * cam.fx * iz * iz;
            gtz += gJ[2] * 2.f * cam.fx * tx * iz * iz * iz;
        } else {
            gtz += gJ[2] * cam.fx * txz * iz * iz;
        }
        if (!cly) {
            gty += -gJ[5] * cam.fy * iz * iz;
            gtz += gJ[5] * 2.f * cam.fy * ty * iz * iz * iz;
        } else {
            gtz += gJ[5] * cam.fy * tyz * iz * iz;
        }
        // t = V_R p + V_t
        float gp[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) gp[i] = VR[i] * gtx + VR[3 + i] * gty + VR[6 + i] * gtz;
        // ---- colour: SH at the viewing direction --------------------------
        {
            const float4 cl = __ldg(reinterpret_cast<const float4 *>(Cloc) + inst);
            float e[3] = {pl[0] - cl.x, pl[1] - cl.y, pl[2] - cl.z};
            float Rf[9] = {1.f, 0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f, 1.f};
            if (sh_frame == 1) {
                const float *rt = root + (size_t)inst * 12;
                Rf[0] = rt[0]; Rf[1] = rt[1]; Rf[2] = rt[2];
                Rf[3] = rt[4]; Rf[4] = rt[5]; Rf[5] = rt[6];
                Rf[6] = rt[8]; Rf[7] = rt[9]; Rf[8] = rt[10];
            }
            float ew[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) ew[i] = Rf[i * 3] * e[0] + Rf[i * 3 + 1] * e[1] + Rf[i * 3 + 2] * e[2];
            const float inv = rsqrtf(ew[0] * ew[0] + ew[1] * ew[1] + ew[2] * ew[2]);
            const float dd[3] = {ew[0] * inv, ew[1] * inv, ew[2] * inv}, drgb[3] = {m1.z, m1.w, db};
            const float4 *shp = ta.sh + T.sh_off + gsrc;
            float *gsh = g_sh + (size_t)gi * 48;
            float gd[3];
            switch (T.sh_deg) {
                case 0: sh_backward<0>(shp, T.n, dd, drgb, gsh, vec_sh, gd); break;
                case 1: sh_backward<1>(shp, T.n, dd, drgb, gsh, vec_sh, gd); break;
                case 2: sh_backward<2>(shp, T.n, dd, drgb, gsh, vec_sh, gd); break;
                default: sh_backward<3>(shp, T.n, dd, drgb, gsh, vec_sh, gd); break;
            }
            // d = ew / |ew|: gew = (gd - d (d . gd)) / |ew|, e = Rf^T ew
            const float dg = dd[0] * gd[0] + dd[1] * gd[1] + dd[2] * gd[2];
            float gew[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) gew[i] = (gd[i] - dd[i] * dg) * inv;
#pragma unroll
            for (int i = 0; i < 3; ++i) gp[i] += Rf[i] * gew[0] + Rf[3 + i] * gew[1] + Rf[6 + i] * gew[2];
        }
        // ---- LBS: p = M [mu; 1], W = V_R A --------------------------------
        float gM[12];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            gM[r * 4 + 0] = gp[r] * mu[0];
            gM[r * 4 + 1] = gp[r] * mu[1];
            gM[r * 4 + 2] = gp[r] * mu[2];
            gM[r * 4 + 3] = gp[r];
        }
        if (skin_mode == 0) {
            // gA = V_R^T gW
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int cc = 0; cc < 3; ++cc)
                    gM[r * 4 + cc] += VR[r] * gW[cc] + VR[3 + r] * gW[3 + cc] + VR[6 + r] * gW[6 + cc];
        }
        float gmu[3];
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) gmu[cc] = M[cc] * gp[0] + M[4 + cc] * gp[1] + M[8 + cc] * gp[2];
        float *acc = g_acc + (size_t)gi * kBwdAcc;
        red4(acc, gmu[0], gmu[1], gmu[2], go);
        // canonical covariance (6 stored entries; off-diagonals count twice)
        red4(acc + 4, m2 * gS[0], m2 * (gS[1] + gS[3]), m2 * (gS[2] + gS[6]), m2 * gS[4]);
        red4(acc + 8, m2 * (gS[5] + gS[7]), m2 * gS[8], 0.f, 0.f);
        // skinning transforms of the instance: dB_j += w_j dM
        float *row = sh.W[t];
#pragma unroll
        for (int j = 0; j < kJoints; ++j) row[j] = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) row[jk[k]] += wk[k];  // a repeated joint adds up
#pragma unroll
        for (int r = 0; r < 3; ++r) sh.M[t][r] = make_float4(gM[r * 4], gM[r * 4 + 1], gM[r * 4 + 2], gM[r * 4 + 3]);
    }
    __syncthreads();
    // row r of dB_j = sum over the active splats of w_j times row r of dM
    constexpr int kSlices = kBwdThreads / (kJoints * 3);
    const int slice = t / (kJoints * 3), j = (t % (kJoints * 3)) / 3, r = t % 3;
    if (slice < kSlices) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int i = slice; i < n; i += kSlices) {
            const float w = sh.W[i][j];
            if (w == 0.f) continue;  // (most; and a gradient that is not finite stays with its joints)
            const float4 v = sh.M[i][r];
            a.x += w * v.x;
            a.y += w * v.y;
            a.z += w * v.z;
            a.w += w * v.w;
        }
        if (a.x != 0.f || a.y != 0.f || a.z != 0.f || a.w != 0.f)
            red4(g_B + ((size_t)inst * kJoints + j) * 12 + 4 * r, a.x, a.y, a.z, a.w);
    }
}

// ---------------------------------------------------------------------------
// forward kinematics backward
// ---------------------------------------------------------------------------

// R(v) by Rodrigues' formula, and dR/dv_i from the compact formula of
// Gallego and Yezzi, "A compact formula for the derivative of a 3-D rotation
// in exponential coordinates", J. Math. Imaging Vis. 51 (2015):
// dR/dv_i = (v_i [v]x + [v x ((I - R) e_i)]x) R / |v|^2, and the series
// [e_i]x + ([e_i]x [v]x + [v]x [e_i]x) / 2 for small |v|.
__device__ void rodrigues_grad(const float v[3], float R[9], float dR[3][9]) {
    const float th2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    const float K[9] = {0.f, -v[2], v[1], v[2], 0.f, -v[0], -v[1], v[0], 0.f};
    float K2[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) K2[i * 3 + j] = K[i * 3] * K[j] + K[i * 3 + 1] * K[3 + j] + K[i * 3 + 2] * K[6 + j];
    float a, b;
    if (th2 < 1e-12f) {
        a = 1.f;
        b = 0.5f;
    } else {
        const float th = sqrtf(th2);
        a = sinf(th) / th;
        const float h = sinf(0.5f * th) / th;
        b = 2.f * h * h;
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) R[e] = (e % 4 == 0 ? 1.f : 0.f) + a * K[e] + b * K2[e];
    for (int i = 0; i < 3; ++i) {
        float E[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // [e_i]x
        if (i == 0) { E[5] = -1.f; E[7] = 1.f; }
        if (i == 1) { E[2] = 1.f; E[6] = -1.f; }
        if (i == 2) { E[1] = -1.f; E[3] = 1.f; }
        if (th2 < 1e-6f) {
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    float ek = 0.f, ke = 0.f;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        ek += E[r * 3 + k] * K[k * 3 + c];
                        ke += K[r * 3 + k] * E[k * 3 + c];
                    }
                    dR[i][r * 3 + c] = E[r * 3 + c] + 0.5f * (ek + ke);
                }
        } else {
            // w = v x ((I - R) e_i)
            const float col[3] = {(i == 0 ? 1.f : 0.f) - R[0 * 3 + i], (i == 1 ? 1.f : 0.f) - R[1 * 3 + i],
                                  (i == 2 ? 1.f : 0.f) - R[2 * 3 + i]};
            const float w[3] = {v[1] * col[2] - v[2] * col[1], v[2] * col[0] - v[0] * col[2], v[0] * col[1] - v[1] * col[0]};
            const float S[9] = {0.f, -(v[i] * v[2] + w[2]), v[i] * v[1] + w[1], v[i] * v[2] + w[2], 0.f,
                                -(v[i] * v[0] + w[0]), -(v[i] * v[1] + w[1]), v[i] * v[0] + w[0], 0.f};
            const float inv = 1.f / th2;
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    dR[i][r * 3 + c] = (S[r * 3] * R[c] + S[r * 3 + 1] * R[3 + c] + S[r * 3 + 2] * R[6 + c]) * inv;
        }
    }
}

// One warp per instance, lane j = joint j: rotations down the tree level by
// level (shuffles from the parent's lane), gradients back up it (a level's
// joints add to their parents in shared memory).
constexpr int kFkBwdWarps = 8;
__global__ void __launch_bounds__(32 * kFkBwdWarps) k_fk_backward(int n_inst, int n_tpl, const int32_t *__restrict__ tid,
                                                                  const float *__restrict__ pose,
                                                                  const TemplateInfo *__restrict__ tpls, int max_depth,
                                                                  const float *__restrict__ g_B,
                                                                  float *__restrict__ g_pose) {
    __shared__ float sg[kFkBwdWarps][kJoints][13];  // dL/d(global rotation, translation); odd rows: conflict free
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int inst = blockIdx.x * kFkBwdWarps + warp;
    if (inst >= n_inst) return;  // uniform per warp
    const int t = tid[inst];
    if (t < 0 || t >= n_tpl) return;
    const TemplateInfo &T = tpls[t];
    const bool on = lane < kJoints;
    const int j = on ? lane : kJoints - 1;
    const int p = T.parent[j], src = p >= 0 ? p : j, dep = on ? (int)T.depth[j] : 1 << 20;
    const float *pv = pose + (size_t)inst * kJoints * 3 + j * 3;
    const float v[3] = {pv[0], pv[1], pv[2]};
    float R[9], dR[3][9];
    rodrigues_grad(v, R, dR);
    const float J[3] = {T.rest[j * 3], T.rest[j * 3 + 1], T.rest[j * 3 + 2]};
    const float o[3] = {J[0] - T.rest[src * 3], J[1] - T.rest[src * 3 + 1], J[2] - T.rest[src * 3 + 2]};
    // forward: G_j = G_parent R_j (rotations; the translations are not needed)
    float GR[9], PR[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) GR[e] = R[e];
    for (int level = 1; level <= max_depth; ++level) {
#pragma unroll
        for (int e = 0; e < 9; ++e) PR[e] = __shfl_sync(0xffffffffu, GR[e], src);
        if (dep == level) {
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    GR[r * 3 + c] = PR[r * 3] * R[c] + PR[r * 3 + 1] * R[3 + c] + PR[r * 3 + 2] * R[6 + c];
        }
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) PR[e] = __shfl_sync(0xffffffffu, GR[e], src);
    // B_j = [G_R | G_t - G_R J_j]: dG_R = dB_R - dB_t J_j^T, dG_t = dB_t
    float *own = sg[warp][j];
    if (on) {
        const float *gb = g_B + ((size_t)inst * kJoints + j) * 12;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float gt = gb[r * 4 + 3];
#pragma unroll
            for (int c = 0; c < 3; ++c) own[r * 3 + c] = gb[r * 4 + c] - gt * J[c];
            own[9 + r] = gt;
        }
    }
    __syncwarp();
    // children before parents: G_R = G_pR R_j, G_t = G_pR o + G_pt
    for (int level = max_depth; level >= 1; --level) {
        if (dep == level && p >= 0) {
            float *up = sg[warp][p];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const float gt = own[9 + r];
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    atomicAdd(up + r * 3 + c, own[r * 3] * R[c * 3] + own[r * 3 + 1] * R[c * 3 + 1] +
                                                  own[r * 3 + 2] * R[c * 3 + 2] + gt * o[c]);
                atomicAdd(up + 9 + r, gt);
            }
        }
        __syncwarp();
    }
    if (!on) return;
    // dL/dR_j = G_pR^T dG_R (the root has no parent), then through the axis-angle
    float gR[9];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            gR[r * 3 + c] = p < 0 ? own[r * 3 + c] : PR[r] * own[c] + PR[3 + r] * own[3 + c] + PR[6 + r] * own[6 + c];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        float acc = 0.f;
#pragma unroll
        for (int e = 0; e < 9; ++e) acc += gR[e] * dR[i][e];
        g_pose[(size_t)inst * kJoints * 3 + j * 3 + i] += acc;
    }
}

// ---------------------------------------------------------------------------
// canonical covariance -> scales and quaternion
// ---------------------------------------------------------------------------

// Adds a Gaussian's summed gradients (kBwdAcc) to the caller's arrays.
__global__ void k_cov_backward(int n, const float4 *__restrict__ scale, const float4 *__restrict__ quat,
                               const float *__restrict__ g_acc, float *__restrict__ g_mean,
                               float *__restrict__ g_opacity, float *__restrict__ g_scale, float *__restrict__ g_quat) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    const float *acc = g_acc + (size_t)g * kBwdAcc, *gc = acc + 4;
    for (int k = 0; k < 3; ++k) g_mean[(size_t)g * 3 + k] += acc[k];
    g_opacity[g] += acc[3];
    // dL/dSigma as a symmetric matrix (off-diagonal stored entries count twice)
    const float Gm[9] = {gc[0], 0.5f * gc[1], 0.5f * gc[2], 0.5f * gc[1], gc[3], 0.5f * gc[4],
                         0.5f * gc[2], 0.5f * gc[4], gc[5]};
    const float4 s4 = scale[g], q4 = quat[g];
    const float s[3] = {s4.x, s4.y, s4.z};
    const float qn = sqrtf(q4.x * q4.x + q4.y * q4.y + q4.z * q4.z + q4.w * q4.w);
    const float w = q4.x / qn, x = q4.y / qn, y = q4.z / qn, z = q4.w / qn;
    const float R[9] = {1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)};
    // Sigma = R diag(s^2) R^T: ds_k = 2 s_k (R^T G R)_kk, dR = 2 G R diag(s^2)
    float GR[9];
    for (int i = 0; i < 3; ++i)
        for (int k = 0; k < 3; ++k) GR[i * 3 + k] = Gm[i * 3] * R[k] + Gm[i * 3 + 1] * R[3 + k] + Gm[i * 3 + 2] * R[6 + k];
    for (int k = 0; k < 3; ++k) {
        const float d = R[k] * GR[k] + R[3 + k] * GR[3 + k] + R[6 + k] * GR[6 + k];
        g_scale[(size_t)g * 3 + k] += 2.f * s[k] * d;
    }
    float gR[9];
    for (int i = 0; i < 3; ++i)
        for (int k = 0; k < 3; ++k) gR[i * 3 + k] = 2.f * GR[i * 3 + k] * s[k] * s[k];
    // R(w, x, y, z) of the normalised quaternion
    const float gw = 2.f * (-z * gR[1] + y * gR[2] + z * gR[3] - x * gR[5] - y * gR[6] + x * gR[7]);
    const float gx = 2.f * (y * gR[1] + z * gR[2] + y * gR[3] - 2.f * x * gR[4] - w * gR[5] + z * gR[6] + w * gR[7] -
                            2.f * x * gR[8]);
    const float gy = 2.f * (-2.f * y * gR[0] + x * gR[1] + w * gR[2] + x * gR[3] + z * gR[5] - w * gR[6] + z * gR[7] -
                            2.f * y * gR[8]);
    const float gz = 2.f * (-2.f * z * gR[0] - w * gR[1] + x * gR[2] + w * gR[3] - 2.f * z * gR[4] + y * gR[5] +
                            x * gR[6] + y * gR[7]);
    // through the normalisation q / |q|
    const float dot = w * gw + x * gx + y * gy + z * gz;
    g_quat[(size_t)g * 4 + 0] += (gw - w * dot) / qn;
    g_quat[(size_t)g * 4 + 1] += (gx - x * dot) / qn;
    g_quat[(size_t)g * 4 + 2] += (gy - y * dot) / qn;
    g_quat[(size_t)g * 4 + 3] += (gz - z * dot) / qn;
}

}  // namespace

int launch_backward(const BackwardArgs &a, cudaStream_t st) {
    int launched = 0;
    const int T = a.tiles_x * a.tiles_y;
    if (T > 0 && a.n_pairs > 0) {
        // chunks of kBwdChunk pairs per tile, numbered tile by tile; one CTA
        // per chunk walks it back to front from the state the forward kept
        k_bwd_chunk_counts<<<(T + 255) / 256, 256, 0, st>>>(T, a.ranges, a.chunk_cnt);
        launched += 1 + exclusive_scan(a.chunk_cnt, nullptr, a.chunk0, (uint32_t)T, a.scan_scratch, st);
        const unsigned grid = a.n_pairs / kBwdChunk + (unsigned)T;  // at least the chunks of the frame
        k_blend_backward<<<grid, kBwdThreads, 0, st>>>(a.tiles_x, a.W, a.H, a.ranges, a.pval, a.rec, a.px_end,
                                                        a.px_fin, a.px_bnd, a.chunk0, T, a.dl_drgba,
                                                        reinterpret_cast<float *>(a.dsplat));
        ++launched;
    }
    if (a.proj_blocks > 0) {
        static int configured_device = -1;
        int dev = 0;
        cudaGetDevice(&dev);
        if (configured_device != dev) {
            cudaFuncSetAttribute(k_project_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ProjBwdShared));
            configured_device = dev;
        }
        // the caller's SH array may start on any float
        const bool vec_sh = (reinterpret_cast<uintptr_t>(a.g_sh) & 15u) == 0;
        k_project_backward<<<a.proj_blocks, kBwdThreads, sizeof(ProjBwdShared), st>>>(
            a.groups, a.n_groups, a.vis, a.B, a.V, a.Cloc, a.root, a.ta, a.tpls, a.cam, a.lod, a.skin_mode,
            a.sh_frame, a.rec, a.dsplat, a.g_acc, a.g_sh, vec_sh, a.g_B);
        ++launched;
    }
    if (a.n_inst > 0) {
        k_fk_backward<<<(a.n_inst + kFkBwdWarps - 1) / kFkBwdWarps, 32 * kFkBwdWarps, 0, st>>>(
            a.n_inst, a.n_tpl, a.tid, a.pose, a.tpls, a.max_depth, a.g_B, a.g_pose);
        ++launched;
    }
    if (a.n_gauss > 0) {
        k_cov_backward<<<(a.n_gauss + 255) / 256, 256, 0, st>>>(a.n_gauss, a.scale, a.quat, a.g_acc, a.g_mean,
                                                                 a.g_opacity, a.g_scale, a.g_quat);
        ++launched;
    }
    return launched;
}

}  // namespace cs
