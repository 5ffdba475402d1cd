// The LoD ranking MLP: 48 -> 64 -> 64 -> 1 with ReLU, BF16 tensor-core
// matrix products with FP32 accumulation, FP32 master weights and Adam.
// k_mlp is the forward pass (mma m16n8k16); k_mlp_train a training step's
// forward and backward pass with per-CTA weight-gradient partials (tcgen05);
// a third kernel reduces the partials in a fixed order and applies Adam.
//
// Forward pass, warp-level fragments of mma.m16n8k16 (bf16 in, f32 accumulate), lane =
// 4 * g + q (g = lane / 4, q = lane % 4):
//   A 16x16 row-major, 4 registers of two bf16 each (low half = lower column):
//     a0 = A[g][2q, 2q+1]  a1 = A[g+8][2q, 2q+1]  a2 = A[g][2q+8, 2q+9]  a3 = A[g+8][2q+8, 2q+9]
//   B 16x8, two registers:  b0 = B[2q, 2q+1][g]  b1 = B[2q+8, 2q+9][g]
//   C 16x8 f32:  c0, c1 = C[g][2q, 2q+1]   c2, c3 = C[g+8][2q, 2q+1]
// Two neighbouring C tiles of a 16-row block therefore hold exactly the A
// fragment of the next layer's 16-wide k step, so activations stay in
// registers between layers.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/crowdsplat.h"
#include "../../include/crowdsplat_lod.h"

namespace {

constexpr int kIn = CS_MLP_IN;      // 48
constexpr int kH = CS_MLP_HIDDEN;   // 64
constexpr int kFeat = CS_LOD_FEATURES;
constexpr int kP = CS_MLP_PARAMS;   // 7361
constexpr int oW1 = 0, oB1 = oW1 + kIn * kH, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH, oB3 = oW3 + kH;
static_assert(oB3 + 1 == kP, "parameter layout");

// forward pass: 8 warps, 16 rows of the CTA's tile each
constexpr int kWarps = 8, kThreads = 32 * kWarps, kTile = 16 * kWarps;
// leading dimensions of the weight copies (bf16 elements): 28 and 36 words, so
// that the eight 16-byte rows of an ldmatrix fall in different banks
constexpr int kLdW1 = 56;   // W1^T  [64 hidden][48 in]
constexpr int kLdW2 = 72;   // W2^T and W2 [64][64]

constexpr size_t kW1Elems = (size_t)kH * kLdW1, kW2Elems = (size_t)kH * kLdW2;
constexpr size_t kSmemWeights = (kW1Elems + kW2Elems) * 2 + (3 * kH + 4) * 4;

struct Weights {
    const __nv_bfloat16 *w1t;  // [64][kLdW1]: w1t[n][k] = bf16(W1[k][n])
    const __nv_bfloat16 *w2t;  // [64][kLdW2]: w2t[n][k] = bf16(W2[k][n])
    const __nv_bfloat16 *w2n;  // [64][kLdW2]: w2n[k][n] = bf16(W2[k][n])
    const float *master;       // FP32 parameters
};

__device__ __forceinline__ void mma16816(float d[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t bits16(__nv_bfloat16 v) { return (uint32_t)__bfloat16_as_ushort(v); }
__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 lo, __nv_bfloat16 hi) { return bits16(lo) | (bits16(hi) << 16); }

// Four 8x8 bf16 matrices (rows of 16 bytes at the lanes' addresses, lanes 8 i
// to 8 i + 7 giving matrix i).
__device__ __forceinline__ void ldsm4(uint32_t r[4], const __nv_bfloat16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p))
                 : "memory");
}

constexpr int kChains = 2;  // independent products in flight: column tiles computed at a time

// d[i] += a (16 rows x 64) times column tile i of a weight matrix in shared
// memory; wp: row mr of the first tile, column 8 mi.
__device__ __forceinline__ void mma_chains(float (&d)[kChains][4], const uint32_t (&a)[4][4], const __nv_bfloat16 *wp) {
#pragma unroll
    for (int kk = 0; kk < 4; kk += 2) {
        uint32_t b[kChains][4];
#pragma unroll
        for (int i = 0; i < kChains; ++i) ldsm4(b[i], wp + 8 * i * kLdW2 + 16 * kk);
#pragma unroll
        for (int i = 0; i < kChains; ++i) mma16816(d[i], a[kk], b[i][0], b[i][1]);
#pragma unroll
        for (int i = 0; i < kChains; ++i) mma16816(d[i], a[kk + 1], b[i][2], b[i][3]);
    }
}

// What a lane reads of its rows g and g + 8: features 8 i + 2 q and the next
// (i = 0 to 3) and the band (-1: none, an all-zero one-hot).
struct RowInputs {
    float2 x[2][4];
    int band[2];
};

__device__ __forceinline__ void load_rows(RowInputs &in, int64_t row, int64_t n, int q, const float *__restrict__ feat,
                                          const int32_t *__restrict__ band) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t r = row + 8 * h;
        const bool v = r < n;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            in.x[h][i] = v ? __ldg(reinterpret_cast<const float2 *>(feat + r * kFeat + 8 * i + 2 * q)) : make_float2(0.f, 0.f);
        in.band[h] = v ? __ldg(band + r) : -1;
    }
}

// The forward pass: a warp per 16 rows, weights as fragments from shared
// memory (four 8x8 matrices per ldmatrix), activations in registers from
// layer to layer, a tile's inputs loaded during the tile before.
__global__ void __launch_bounds__(kThreads, 2)
    k_mlp(int64_t n, int n_tiles, const float *__restrict__ feat, const int32_t *__restrict__ band, Weights W,
          float *__restrict__ score) {
    extern __shared__ __align__(16) unsigned char smem[];
    __nv_bfloat16 *sW1t = reinterpret_cast<__nv_bfloat16 *>(smem);
    __nv_bfloat16 *sW2t = sW1t + kW1Elems;
    float *sb1 = reinterpret_cast<float *>(sW2t + kW2Elems);
    float *sb2 = sb1 + kH, *sw3 = sb2 + kH, *sb3 = sw3 + kH;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
    const int mi = lane >> 3, mr = lane & 7;  // the matrix and row whose address the lane gives an ldmatrix
    {
        const uint4 *s1 = reinterpret_cast<const uint4 *>(W.w1t);
        const uint4 *s2 = reinterpret_cast<const uint4 *>(W.w2t);
        uint4 *d1 = reinterpret_cast<uint4 *>(sW1t), *d2 = reinterpret_cast<uint4 *>(sW2t);
        for (int i = tid; i < (int)(kW1Elems / 8); i += kThreads) d1[i] = s1[i];
        for (int i = tid; i < (int)(kW2Elems / 8); i += kThreads) d2[i] = s2[i];
        for (int i = tid; i < kH; i += kThreads) {
            sb1[i] = W.master[oB1 + i];
            sb2[i] = W.master[oB2 + i];
            sw3[i] = W.master[oW3 + i];
        }
        if (tid == 0) sb3[0] = W.master[oB3];
    }
    __syncthreads();

    RowInputs in;
    load_rows(in, (int64_t)blockIdx.x * kTile + warp * 16 + g, n, q, feat, band);
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int64_t r0 = (int64_t)tile * kTile + warp * 16;
        const int64_t ra = r0 + g, rb = r0 + g + 8;
        const bool va = ra < n, vb = rb < n;

        // ---- layer 1: z1 = x W1 + b1 -------------------------------------
        uint32_t a1[3][4];
#pragma unroll
        for (int kk = 0; kk < 3; ++kk) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int c = 16 * kk + 8 * half + 2 * q;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // columns 32 to 35: one-hot band; 36 to 47: zero
                    const int b = c - kFeat;
                    const float2 x = kk < 2 ? in.x[h][2 * kk + half]
                                            : make_float2(b < 4 && b == in.band[h] ? 1.f : 0.f,
                                                          b < 4 && b + 1 == in.band[h] ? 1.f : 0.f);
                    a1[kk][2 * half + h] = pack2(__float2bfloat16_rn(x.x), __float2bfloat16_rn(x.y));
                }
            }
        }
        uint32_t a2[4][4];  // bf16 h1 as layer-2 A fragments
#pragma unroll
        for (int n0 = 0; n0 < 8; n0 += kChains) {
            float d[kChains][4];
            uint32_t b[kChains][4], bx[kChains / 2][4];  // k steps 0 and 1; the third of two column tiles
#pragma unroll
            for (int i = 0; i < kChains; ++i) {
                const float2 bias = *reinterpret_cast<const float2 *>(sb1 + 8 * (n0 + i) + 2 * q);
                d[i][0] = d[i][2] = bias.x;
                d[i][1] = d[i][3] = bias.y;
                ldsm4(b[i], sW1t + (8 * (n0 + i) + mr) * kLdW1 + 8 * mi);
                if (!(i & 1)) ldsm4(bx[i / 2], sW1t + (8 * (n0 + i + (mi >> 1)) + mr) * kLdW1 + 32 + 8 * (mi & 1));
            }
#pragma unroll
            for (int i = 0; i < kChains; ++i) mma16816(d[i], a1[0], b[i][0], b[i][1]);
#pragma unroll
            for (int i = 0; i < kChains; ++i) mma16816(d[i], a1[1], b[i][2], b[i][3]);
#pragma unroll
            for (int i = 0; i < kChains; ++i) mma16816(d[i], a1[2], bx[i / 2][2 * (i & 1)], bx[i / 2][2 * (i & 1) + 1]);
#pragma unroll
            for (int i = 0; i < kChains; ++i) {
                const int nt = n0 + i;
                __nv_bfloat16 h[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) h[e] = __float2bfloat16_rn(fmaxf(d[i][e], 0.f));
                a2[nt >> 1][(nt & 1) * 2] = pack2(h[0], h[1]);
                a2[nt >> 1][(nt & 1) * 2 + 1] = pack2(h[2], h[3]);
            }
        }
        // ---- layer 2: z2 = h1 W2 + b2; output y = relu(z2) w3 + b3 --------
        float pa = 0.f, pb = 0.f;
#pragma unroll
        for (int n0 = 0; n0 < 8; n0 += kChains) {
            float d[kChains][4];
#pragma unroll
            for (int i = 0; i < kChains; ++i) {
                const float2 bias = *reinterpret_cast<const float2 *>(sb2 + 8 * (n0 + i) + 2 * q);
                d[i][0] = d[i][2] = bias.x;
                d[i][1] = d[i][3] = bias.y;
            }
            mma_chains(d, a2, sW2t + (8 * n0 + mr) * kLdW2 + 8 * mi);
#pragma unroll
            for (int i = 0; i < kChains; ++i) {
                const float2 w3 = *reinterpret_cast<const float2 *>(sw3 + 8 * (n0 + i) + 2 * q);
                pa += fmaxf(d[i][0], 0.f) * w3.x + fmaxf(d[i][1], 0.f) * w3.y;
                pb += fmaxf(d[i][2], 0.f) * w3.x + fmaxf(d[i][3], 0.f) * w3.y;
            }
        }
        pa += __shfl_xor_sync(0xffffffffu, pa, 1);
        pa += __shfl_xor_sync(0xffffffffu, pa, 2);
        pb += __shfl_xor_sync(0xffffffffu, pb, 1);
        pb += __shfl_xor_sync(0xffffffffu, pb, 2);
        const float ya = pa + sb3[0], yb = pb + sb3[0];
        if (q == 0) {
            if (va) score[ra] = ya;
            if (vb) score[rb] = yb;
        }
        load_rows(in, ra + (int64_t)gridDim.x * kTile, n, q, feat, band);
    }
}

// ---------------------------------------------------------------------------
// training: forward, backward and weight gradients on the fifth-generation
// tensor cores (tcgen05, accumulators in TMEM)
//
// A CTA is two groups of eight warps; a group works through tiles of 128 rows
// by itself, two threads per row (the TMEM lane of the accumulators), one for
// each half of the 64 hidden units:
//   Z1 = X W1        M 128, N 64, K 48     then h1 = relu(Z1 + b1)
//   Z2 = H1 W2       M 128, N 64, K 64     then y, dy, dz2 = dy w3 [z2 > 0]
//   dH1 = dZ2 W2^T   M 128, N 64, K 64     then dz1 = dH1 [h1 > 0]
//   G += [H1 | X]^T [dZ2 | dZ1]   M 128, N 128, K 128 (the rows)
// The last product holds dW2 in its first 64 rows and columns and dW1 in its
// last; the other two quarters are not read.  It stays in TMEM over all the
// group's tiles.  The column sums (dw3, db2, db1) stay in registers: 96 per
// thread, since a thread sees 32 columns of every tile.
//
// Activations lie in shared memory row by row, 128 bytes a row, in the
// 128-byte swizzle (16-byte chunk c of row r at chunk c ^ (r & 7)).  The same
// bytes serve as a K-major operand (rows are M or N, 8-row groups 1,024 bytes
// apart) and as an MN-major one (rows are K; the next 64 columns of M or N
// are in the next buffer), so nothing is transposed.  X has two buffers: the
// next tile's features arrive by one bulk copy and are converted while a
// product of this tile runs, and its first product is issued right after this
// tile's last.  One thread of a group issues all its products, which complete in
// order, so the wait for one also covers those before it.
//
// Bound by latency (issue slots 45%, shared-memory and TMEM data path 47%,
// tensor pipe 17%): a group's three waits per tile and its loads from TMEM,
// with two groups an SM: a thread's 128 registers (96 of them column sums)
// leave no room for a third, nor do 100 KB of shared memory and 192 TMEM
// columns each.  A training step of 2,752,512 rows: 541 us with mma.sync
// (weights, activations and gradients as fragments from shared memory, 503 us
// of it this kernel) -> 412 us (372).  One thread per row instead of two 429;
// the features by 8-byte cp.async 432; FP32 operations one by one and BF16
// conversions one by one 466.
//
// Steps of a few thousand rows pay for what a CTA does once: one tile per CTA
// while there are SMs for that, the first features under way before the
// weights are read, column sums in 31 shuffles a warp instead of 160 per 32
// columns, the gradient through shared memory to consecutive addresses, the
// loss written to the host's memory by the update.  A step and its loss at
// 3,000 rows 52 -> 36 us, 19,456 rows 52 -> 37, without the loss 39 -> 29 and
// 41 -> 30; 300,000 rows 76.9 -> 65.1, 2,752,512 rows 390 -> 372.  (128-row
// tiles with mma.sync, one tile per SM: 41, 44; 30, 34; 104, 690.)
// ---------------------------------------------------------------------------

constexpr int kTcGroups = 2, kTcGroupThreads = 256, kTcThreads = kTcGroupThreads * kTcGroups, kTcRows = 128;
constexpr uint32_t kTcBuf = kTcRows * 128;            // a buffer of 128 rows
constexpr uint32_t kTcGroupBytes = 5 * kTcBuf;        // H1, X (two), dZ2, dZ1
constexpr uint32_t kTcWBuf = kH * 128;                // a weight matrix of 64 rows
constexpr uint32_t kTcStage = kTcRows * (kFeat + 2) * 4;  // a tile's FP32 features; shares of y
constexpr uint32_t kTcOffW = kTcGroups * kTcGroupBytes;
constexpr uint32_t kTcOffStage = kTcOffW + 3 * kTcWBuf;
static_assert(kTcStage % 128 == 0, "alignment of what follows");
constexpr uint32_t kTcOffVec = kTcOffStage + kTcGroups * kTcStage;  // b1, b2, w3, b3
constexpr uint32_t kTcOffBar = kTcOffVec + (3 * kH + 4) * 4;        // mbarriers, TMEM address
constexpr size_t kSmemTc = kTcOffBar + 64 + 1024;                   // (1,024: alignment)
static_assert(kSmemTc <= 227 * 1024, "shared memory of the training kernel");
constexpr uint32_t kTcCols = 512;  // TMEM columns: 64 per group for Z, 128 per group for G (from 128 on)
// a wait gives up after about a second, and not before it has polled some more
// (the clock also runs while the context is switched out)
constexpr long long kTcWaitClocks = 2000000000ll;
constexpr int kTcLatePolls = 256;

// matrix descriptor (128-byte swizzle): start address, stride between the
// 64-column halves of an MN-major operand, 1,024 bytes between 8-row groups
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t half_stride) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(half_stride >> 4) << 16) | ((uint64_t)(1024u >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}
// instruction descriptor: BF16 operands, FP32 accumulator
__host__ __device__ constexpr uint32_t tc_idesc(bool mn_major, int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((mn_major ? 3u : 0u) << 15) | ((uint32_t)(n / 8) << 17) |
           ((uint32_t)(m / 16) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate)
        : "memory");
}
// the mbarrier arrives when all products issued so far by this thread are done
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void group_sync(int group) { asm volatile("bar.sync %0, 256;" ::"r"(group + 1) : "memory"); }
// The same barrier; whether a thread of the group came with `failed` (the same
// answer in all of them).
__device__ __forceinline__ bool group_failed(int group, uint32_t failed) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %2, 0;\n\tbar.red.or.pred q, %1, 256, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(group + 1), "r"(failed)
        : "memory");
    return r != 0u;
}

// Waits for phase `parity` of the mbarrier; false after kTcWaitClocks.
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    for (int late = 0;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > kTcWaitClocks && ++late > kTcLatePolls) return false;
    }
}

// pairs of FP32 values, one instruction for both
using f2 = unsigned long long;
__device__ __forceinline__ f2 make2(float lo, float hi) {
    return (f2)__float_as_uint(lo) | ((f2)__float_as_uint(hi) << 32);
}
__device__ __forceinline__ float lo2(f2 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(f2 v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 relu2(f2 v) { return make2(fmaxf(lo2(v), 0.f), fmaxf(hi2(v), 0.f)); }

// sixteen columns of the thread's TMEM lane, in pairs
__device__ __forceinline__ void tc_load16(f2 (&z)[8], uint32_t addr) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) z[i] = (f2)r[2 * i] | ((f2)r[2 * i + 1] << 32);
}

__device__ __forceinline__ uint32_t cvt2(f2 v) {  // to two BF16, the lower in the lower half
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo2(v), hi2(v));
    return *reinterpret_cast<const uint32_t *>(&h);
}
// 16-byte chunk c of row r of a swizzled buffer
__device__ __forceinline__ uint4 *tc_chunk(unsigned char *buf, int r, int c) {
    return reinterpret_cast<uint4 *>(buf + r * 128 + ((c ^ (r & 7)) << 4));
}

// The tile's FP32 features to the staging buffer: one bulk copy, whose
// arrival the mbarrier counts, or (an array at an odd multiple of 8 bytes)
// loads and stores by the group's threads.  t: thread of the group.
__device__ __forceinline__ void tc_stage(unsigned char *stage, uint32_t bar, bool bulk, int64_t row0, int64_t n, int t,
                                         const float *__restrict__ feat) {
    const int rows = (int)min((int64_t)kTcRows, n - row0);
    const float *src = feat + row0 * kFeat;
    if (!bulk) {
        for (int i = t; i < rows * kFeat / 2; i += kTcGroupThreads)
            reinterpret_cast<float2 *>(stage)[i] = __ldg(reinterpret_cast<const float2 *>(src) + i);
    } else if (t == 32) {
        const uint32_t bytes = (uint32_t)rows * kFeat * 4;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(stage)),
                     "l"(src), "r"(bytes), "r"(bar)
                     : "memory");
    }
}

// The staged features to X as BF16, and by the first half's threads their
// row's one-hot band (columns 40 to 63 stay zero); rows past n are zero.
__device__ __forceinline__ void tc_input(unsigned char *x, const unsigned char *stage, int64_t row0, int64_t n, int t,
                                         int band) {
    const int r0 = t >> 3, p = t & 7;  // 16-byte piece p of rows r0 + 32 i
    unsigned char *to = x + r0 * 128 + (((p >> 1) ^ (r0 & 7)) << 4) + 8 * (p & 1);
#pragma unroll
    for (int i = 0; i < kTcRows / 32; ++i) {
        float4 a = reinterpret_cast<const float4 *>(stage)[t + kTcGroupThreads * i];
        if (row0 + r0 + 32 * i >= n) a = make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<uint2 *>(to + 4096 * i) = make_uint2(cvt2(make2(a.x, a.y)), cvt2(make2(a.z, a.w)));
    }
    if (t < kTcRows) {
        const uint32_t one = 0x3F80u;  // 1.0
        *tc_chunk(x, t, 4) = make_uint4((band == 0 ? one : 0u) | (band == 1 ? one << 16 : 0u),
                                        (band == 2 ? one : 0u) | (band == 3 ? one << 16 : 0u), 0u, 0u);
    }
}

// Lane l's result: the sum over the warp's lanes of value l of their 32 (half of
// what is left is sent and received at each step: 31 shuffles in place of 160).
__device__ __forceinline__ float lane_column_sum(const f2 (&v)[16]) {
    const int lane = threadIdx.x & 31;
    float x[32];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        x[2 * i] = lo2(v[i]);
        x[2 * i + 1] = hi2(v[i]);
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const bool upper = (lane & s) != 0;
#pragma unroll
        for (int i = 0; i < s; ++i) {
            const float got = __shfl_xor_sync(0xffffffffu, upper ? x[i] : x[i + s], s);
            x[i] = (upper ? x[i + s] : x[i]) + got;
        }
    }
    return x[0];
}

__global__ void __launch_bounds__(kTcThreads, 1)
    k_mlp_train(int64_t n, int n_tiles, const float *__restrict__ feat, const int32_t *__restrict__ band,
                const float *__restrict__ target, Weights W, float inv_n, bool bulk, bool lose, float *__restrict__ partial,
                uint32_t *__restrict__ err, volatile uint32_t *host_err) {
    extern __shared__ unsigned char tc_raw[];
    unsigned char *smem = tc_raw + ((1024u - ((uint32_t)__cvta_generic_to_shared(tc_raw) & 1023u)) & 1023u);
    // t: thread of the group; r: its row of the tile, half: its half of the hidden units
    const int tid = threadIdx.x, group = tid >> 8, t = tid & 255, half = t >> 7, r = t & 127, warp = tid >> 5, lane = tid & 31;
    unsigned char *sH1 = smem + group * kTcGroupBytes, *sX = sH1 + kTcBuf, *sD2 = sX + 2 * kTcBuf, *sD1 = sD2 + kTcBuf;
    unsigned char *sW = smem + kTcOffW;  // W1^T, W2^T, W2
    unsigned char *stage = smem + kTcOffStage + group * kTcStage;
    float *s_y = reinterpret_cast<float *>(stage) + kTcRows * kFeat;  // shares of y, by half
    float *sb1 = reinterpret_cast<float *>(smem + kTcOffVec), *sb2 = sb1 + kH, *sw3 = sb2 + kH, *sb3 = sw3 + kH;
    const ulonglong2 *vb1 = reinterpret_cast<const ulonglong2 *>(sb1), *vb2 = reinterpret_cast<const ulonglong2 *>(sb2),
                     *vw3 = reinterpret_cast<const ulonglong2 *>(sw3);  // four values each
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kTcOffBar);
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(bars + 2 * kTcGroups);
    // of a group: its products, its staged features
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(bars + group), stage_bar = bar + 8 * kTcGroups;

    // the group's first features start before the weights are read
    const int first = (int)blockIdx.x + group * (int)gridDim.x, step = (int)gridDim.x * kTcGroups;
    const int64_t first0 = (int64_t)first * kTcRows;
    if (t == 32) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(stage_bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tc_fence_smem();
    }
    int nband = -1;
    float ntarget = 0.f;
    auto next_row = [&](int64_t row) {  // band and target of the thread's row of a coming tile
        nband = row < n ? __ldg(band + row) : -1;
        ntarget = row < n ? __ldg(target + row) : 0.f;
    };
    if (first < n_tiles) {
        tc_stage(stage, stage_bar, bulk, first0, n, t, feat);
        next_row(first0 + r);
    }
    // weights into the swizzled layout (columns past a row's length zero), one
    // 16-byte chunk of each matrix a thread
    {
        static_assert(kTcThreads == kH * 8, "a chunk per thread");
        const int wr = tid >> 3, c = tid & 7;
        uint4 v1 = make_uint4(0u, 0u, 0u, 0u);
        if (c < kIn / 8) v1 = *reinterpret_cast<const uint4 *>(W.w1t + wr * kLdW1 + 8 * c);
        const uint4 v2 = *reinterpret_cast<const uint4 *>(W.w2t + wr * kLdW2 + 8 * c);
        const uint4 v3 = *reinterpret_cast<const uint4 *>(W.w2n + wr * kLdW2 + 8 * c);
        if (tid < 3 * kH) sb1[tid] = W.master[(tid < kH ? oB1 : tid < 2 * kH ? oB2 - kH : oW3 - 2 * kH) + tid];
        if (tid == 3 * kH) sb3[0] = W.master[oB3];
        *tc_chunk(sW, wr, c) = v1;
        *tc_chunk(sW + kTcWBuf, wr, c) = v2;
        *tc_chunk(sW + 2 * kTcWBuf, wr, c) = v3;
    }
    for (int c = 5; c < 8; ++c) *tc_chunk(sX + half * kTcBuf, r, c) = make_uint4(0u, 0u, 0u, 0u);
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(s_tmem)),
                     "r"(kTcCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    const uint32_t z_cols = tmem + 64u * group, g_cols = tmem + 128u + 128u * group;
    const uint32_t my_lanes = (uint32_t)(warp & 3) << 21;  // lane 32 (warp % 4) in bits 16 and up
    constexpr int kMine = kH / 2;                          // the thread's columns, from `mine` on
    const int mine = kMine * half;
    const bool issuer = t == 0;
    const uint32_t aH1 = (uint32_t)__cvta_generic_to_shared(sH1), aX = (uint32_t)__cvta_generic_to_shared(sX),
                   aD2 = (uint32_t)__cvta_generic_to_shared(sD2), aW = (uint32_t)__cvta_generic_to_shared(sW);
    constexpr uint32_t kFwd = tc_idesc(false, 128, 64), kGrad = tc_idesc(true, 128, 128);

    f2 s_w3[kMine / 2], s_b2[kMine / 2], s_b1[kMine / 2];  // column sums over the thread's rows
#pragma unroll
    for (int i = 0; i < kMine / 2; ++i) s_w3[i] = s_b2[i] = s_b1[i] = 0ull;
    float acc_loss = 0.f, acc_b3 = 0.f;
    bool any = false;  // a tile has been added to G

    // the first tile's inputs and first product
    // A wait that gives up leaves its phase as it is and is noted in the flags;
    // the group's next barrier tells all its threads, which then leave.
    // One register of flags: the phases to wait for, a copy that may be in
    // flight, what was given up, and that the group has left.
    constexpr uint32_t kPhase = 1u, kStagePhase = 2u, kStaging = 4u, kLostProduct = 8u, kLostStage = 16u, kLeft = 32u;
    constexpr uint32_t kLost = kLostProduct | kLostStage;
    uint32_t flags = first < n_tiles ? kStaging : 0u;
    auto staged = [&] {  // the staged features are there
        if (!bulk) {
            group_sync(group);
            flags &= ~kStaging;
        } else if (tc_wait(stage_bar, (flags / kStagePhase) & 1u)) {
            flags = (flags ^ kStagePhase) & ~kStaging;
        } else {
            flags |= kLostStage;
        }
        __syncwarp();
    };
    auto product = [&] {  // the last committed product is there
        flags = tc_wait(bar, flags & kPhase) ? flags ^ kPhase : flags | kLostProduct;
        __syncwarp();
        tc_fence_after();
    };
    if (first < n_tiles) {
        staged();
        tc_input(sX, stage, first0, n, t, nband);
        tc_fence_smem();
        tc_fence_before();
        if (group_failed(group, flags & kLost)) {
            flags |= kLeft;
        } else if (first + step < n_tiles) {
            flags |= kStaging;
            tc_stage(stage, stage_bar, bulk, (int64_t)(first + step) * kTcRows, n, t, feat);
        }
        if (issuer && !(flags & kLeft)) {
            tc_fence_after();
#pragma unroll
            for (int k = 0; k < kIn / 16; ++k) tc_mma(z_cols, tc_desc(aX + 32 * k, 0), tc_desc(aW + 32 * k, 0), kFwd, k > 0);
            if (!(lose && tid == 0 && blockIdx.x == 0)) tc_commit(bar);
        }
    }
    int xbuf = 0;
    for (int tile = first; tile < n_tiles && !(flags & kLeft); tile += step, xbuf ^= 1) {
        const bool valid = (int64_t)tile * kTcRows + r < n, more = tile + step < n_tiles;
        const int64_t next0 = (int64_t)(tile + step) * kTcRows;
        const float y_target = ntarget;
        if (more) next_row(next0 + r);
        // ---- h1 = relu(Z1 + b1) ------------------------------------------
        product();
#pragma unroll
        for (int c0 = 0; c0 < kMine; c0 += 16) {
            f2 z[8];
            tc_load16(z, z_cols + my_lanes + mine + c0);
            uint32_t h[8];
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                const ulonglong2 b = vb1[(mine + c0) / 4 + i / 2];
                h[i] = cvt2(relu2(add2(z[i], b.x)));
                h[i + 1] = cvt2(relu2(add2(z[i + 1], b.y)));
            }
            *tc_chunk(sH1, r, (mine + c0) / 8) = make_uint4(h[0], h[1], h[2], h[3]);
            *tc_chunk(sH1, r, (mine + c0) / 8 + 1) = make_uint4(h[4], h[5], h[6], h[7]);
        }
        tc_fence_smem();
        tc_fence_before();
        if (group_failed(group, flags & kLost)) {
            flags |= kLeft;
            break;
        }
        if (issuer) {
            tc_fence_after();
#pragma unroll
            for (int k = 0; k < kH / 16; ++k)
                tc_mma(z_cols, tc_desc(aH1 + 32 * k, 0), tc_desc(aW + kTcWBuf + 32 * k, 0), kFwd, k > 0);
            tc_commit(bar);
        }
        // the next tile's inputs, while Z2 is computed
        if (more) {
            staged();
            tc_input(sX + (xbuf ^ 1) * kTcBuf, stage, next0, n, t, nband);
        }
        // ---- y, dy, dz2 = dy w3 [z2 > 0] ---------------------------------
        product();
        f2 y2 = 0ull;
#pragma unroll
        for (int c0 = 0; c0 < kMine; c0 += 16) {
            f2 z[8];
            tc_load16(z, z_cols + my_lanes + mine + c0);
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                const ulonglong2 b = vb2[(mine + c0) / 4 + i / 2], w = vw3[(mine + c0) / 4 + i / 2];
                y2 = fma2(relu2(add2(z[i], b.x)), w.x, y2);
                y2 = fma2(relu2(add2(z[i + 1], b.y)), w.y, y2);
            }
        }
        // the halves' shares of y meet in shared memory
        s_y[t] = lo2(y2) + hi2(y2);
        group_sync(group);
        const float y = s_y[r] + s_y[r + 128];
        const float e = valid ? y + sb3[0] - y_target : 0.f;
        const float dy = 2.f * e * inv_n;
        const f2 dy2 = make2(dy, dy);
        if (half == 0) {
            acc_loss += e * e;
            acc_b3 += dy;
        }
#pragma unroll
        for (int c0 = 0; c0 < kMine; c0 += 16) {
            f2 z[8];
            tc_load16(z, z_cols + my_lanes + mine + c0);
            uint32_t h[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const ulonglong2 b4 = vb2[(mine + c0) / 4 + i / 2], w4 = vw3[(mine + c0) / 4 + i / 2];
                const f2 zb = add2(z[i], i & 1 ? b4.y : b4.x), p = mul2(dy2, i & 1 ? w4.y : w4.x);
                const f2 d = make2(lo2(zb) > 0.f ? lo2(p) : 0.f, hi2(zb) > 0.f ? hi2(p) : 0.f);
                s_w3[c0 / 2 + i] = fma2(dy2, relu2(zb), s_w3[c0 / 2 + i]);
                s_b2[c0 / 2 + i] = add2(s_b2[c0 / 2 + i], d);
                h[i] = cvt2(d);
            }
            *tc_chunk(sD2, r, (mine + c0) / 8) = make_uint4(h[0], h[1], h[2], h[3]);
            *tc_chunk(sD2, r, (mine + c0) / 8 + 1) = make_uint4(h[4], h[5], h[6], h[7]);
        }
        tc_fence_smem();
        tc_fence_before();
        if (group_failed(group, flags & kLost)) {
            flags |= kLeft;
            break;
        }
        if (tile + 2 * step < n_tiles) {
            flags |= kStaging;
            tc_stage(stage, stage_bar, bulk, (int64_t)(tile + 2 * step) * kTcRows, n, t, feat);
        }
        if (issuer) {
            tc_fence_after();
#pragma unroll
            for (int k = 0; k < kH / 16; ++k)
                tc_mma(z_cols, tc_desc(aD2 + 32 * k, 0), tc_desc(aW + 2 * kTcWBuf + 32 * k, 0), kFwd, k > 0);
            tc_commit(bar);
        }
        // ---- dz1 = dH1 [h1 > 0] ------------------------------------------
        product();
#pragma unroll
        for (int c0 = 0; c0 < kMine; c0 += 16) {
            f2 z[8];
            tc_load16(z, z_cols + my_lanes + mine + c0);
            const uint4 ha = *tc_chunk(sH1, r, (mine + c0) / 8), hb = *tc_chunk(sH1, r, (mine + c0) / 8 + 1);
            const uint32_t hw[8] = {ha.x, ha.y, ha.z, ha.w, hb.x, hb.y, hb.z, hb.w};
            uint32_t h[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const f2 d = make2(hw[i] & 0xFFFFu ? lo2(z[i]) : 0.f, hw[i] > 0xFFFFu ? hi2(z[i]) : 0.f);
                s_b1[c0 / 2 + i] = add2(s_b1[c0 / 2 + i], d);
                h[i] = cvt2(d);
            }
            *tc_chunk(sD1, r, (mine + c0) / 8) = make_uint4(h[0], h[1], h[2], h[3]);
            *tc_chunk(sD1, r, (mine + c0) / 8 + 1) = make_uint4(h[4], h[5], h[6], h[7]);
        }
        tc_fence_smem();
        tc_fence_before();
        if (group_failed(group, flags & kLost)) {
            flags |= kLeft;
            break;
        }
        if (issuer) {
            tc_fence_after();
            // G, sixteen rows a product: [H1 | X] and [dZ2 | dZ1]
            const uint32_t to_x = kTcBuf * (1 + xbuf);
#pragma unroll
            for (int k = 0; k < kTcRows / 16; ++k)
                tc_mma(g_cols, tc_desc(aH1 + 2048 * k, to_x), tc_desc(aD2 + 2048 * k, kTcBuf), kGrad, any || k > 0);
            if (more) {
                const uint32_t x = aX + (xbuf ^ 1) * kTcBuf;
#pragma unroll
                for (int k = 0; k < kIn / 16; ++k) tc_mma(z_cols, tc_desc(x + 32 * k, 0), tc_desc(aW + 32 * k, 0), kFwd, k > 0);
            }
            tc_commit(bar);
        }
        any = true;
    }
    if (any && !(flags & kLeft)) product();
    // after a wait that gave up: what is still in flight reads or writes
    // shared memory and TMEM (a second wait, with the same limit)
    if (flags & kLostProduct) tc_wait(bar, flags & kPhase);
    if (bulk && (flags & kStaging)) tc_wait(stage_bar, (flags / kStagePhase) & 1u);
    tc_fence_before();
    const bool bad = __syncthreads_or((int)(flags & kLost));
    tc_fence_after();
    if (bad) {
        // no gradient: the host is told, the parameters stay
        if (tid == 0) {
            atomicOr(err, 1u);
            *host_err = 1u;
        }
        __syncwarp();
        if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols) : "memory");
        return;
    }

    // ---- per-CTA partial gradient, written in a fixed order --------------
    // Over the activations: each group's quarters of G (a row's two threads
    // read half of its columns each) and its warps' column sums; then
    // consecutive threads write consecutive values.  A group without a tile
    // has neither.
    float *out = partial + (size_t)blockIdx.x * (kP + 1);
    constexpr int kLdG = kH + 1, kGFloats = 2 * kH * kLdG;
    float *sG = reinterpret_cast<float *>(smem);            // [groups][128][kLdG]
    float *sRed = sG + kTcGroups * kGFloats;                // [8 warp rows][3 kH + 2]
    constexpr int kLdR = 3 * kH + 2;
    const bool both = (int)(blockIdx.x + gridDim.x) < n_tiles;  // the second group had a tile
    if (any) {
        // (warps 0, 1, 4 and 5 of a group hold dW2's rows, the others dW1's)
        const uint32_t my_g = g_cols + my_lanes + (r < kH ? 0 : kH) + mine;  // dW2's columns, dW1's
        float *row = sG + group * kGFloats + r * kLdG + mine;
#pragma unroll
        for (int c0 = 0; c0 < kMine; c0 += 16) {
            f2 z[8];
            tc_load16(z, my_g + c0);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                row[c0 + 2 * i] = lo2(z[i]);
                row[c0 + 2 * i + 1] = hi2(z[i]);
            }
        }
        float *red = sRed + (4 * group + (warp & 3)) * kLdR;  // 32 rows of the tiles, both halves' columns
        red[mine + lane] = lane_column_sum(s_w3);
        red[kH + mine + lane] = lane_column_sum(s_b2);
        red[2 * kH + mine + lane] = lane_column_sum(s_b1);
        float l = acc_loss, b3 = acc_b3;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            l += __shfl_xor_sync(0xffffffffu, l, s);
            b3 += __shfl_xor_sync(0xffffffffu, b3, s);
        }
        if (lane == 0 && half == 0) {
            red[3 * kH] = b3;
            red[3 * kH + 1] = l;
        }
    }
    __syncthreads();
    // row r of dW2, row r - 64 of dW1 (its rows past kIn are padding)
    for (int i = tid; i < (kH + kIn) * kH; i += kTcThreads) {
        const float *g = sG + (i / kH) * kLdG + i % kH;
        out[i < kH * kH ? oW2 + i : oW1 + i - kH * kH] = both ? g[0] + g[kGFloats] : g[0];
    }
    if (tid < kLdR) {
        float a = 0.f;
        for (int w = 0; w < (both ? 8 : 4); ++w) a += sRed[w * kLdR + tid];
        const int o = tid < kH ? oW3 + tid : tid < 2 * kH ? oB2 + tid - kH : tid < 3 * kH ? oB1 + tid - 2 * kH
                                                                          : tid == 3 * kH ? oB3 : kP;
        out[o] = a;  // (kP: the sum of squared errors)
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols) : "memory");
    }
}

// Sum the per-CTA partials, then Adam on the FP32 master weights and refresh
// the BF16 copies.  A block takes 32 parameters, a warp a run of the
// partials; the eight warps' sums are added in order.  Parameter kP is the
// sum of the squared errors, which goes to the host's memory (pinned).  After a training kernel that gave up waiting
// (*err) the parameters stay as they are.  One thread per parameter over all
// 152 partials took 16 us (a chain of loads).
constexpr int kAdamWarps = 8;

__global__ void __launch_bounds__(32 * kAdamWarps)
    k_mlp_adam(int n_part, const float *__restrict__ partial, float *__restrict__ master, float *__restrict__ m1,
               float *__restrict__ m2, float *__restrict__ grad, __nv_bfloat16 *__restrict__ w1t,
               __nv_bfloat16 *__restrict__ w2t, __nv_bfloat16 *__restrict__ w2n, float lr, float bc1, float bc2,
               float *__restrict__ sse, const uint32_t *__restrict__ err) {
    __shared__ float sums[kAdamWarps][32];
    const int warp = threadIdx.x >> 5, p = blockIdx.x * 32 + (threadIdx.x & 31);
    const int run = (n_part + kAdamWarps - 1) / kAdamWarps, c1 = min(n_part, (warp + 1) * run);
    // (what the update reads is loaded with the partials, not after them)
    const bool mine = warp == 0 && p < kP;
    const float m0 = mine ? m1[p] : 0.f, v0 = mine ? m2[p] : 0.f, th0 = mine ? master[p] : 0.f;
    const bool failed = *err != 0u;
    float s = 0.f;
    if (p <= kP) {
#pragma unroll 8
        for (int c = warp * run; c < c1; ++c) s += partial[(size_t)c * (kP + 1) + p];
    }
    sums[warp][threadIdx.x & 31] = s;
    __syncthreads();
    if (warp > 0 || p > kP || failed) return;
    s = 0.f;
    for (int w = 0; w < kAdamWarps; ++w) s += sums[w][threadIdx.x];
    if (p == kP) {
        *sse = s;
        return;
    }
    grad[p] = s;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float m = b1 * m0 + (1.f - b1) * s;
    const float v = b2 * v0 + (1.f - b2) * s * s;
    m1[p] = m;
    m2[p] = v;
    const float th = th0 - lr * (m / bc1) / (sqrtf(v / bc2) + eps);
    master[p] = th;
    if (p < oB1) {
        const int k = p / kH, n = p % kH;
        w1t[n * kLdW1 + k] = __float2bfloat16_rn(th);
    } else if (p >= oW2 && p < oB2) {
        const int k = (p - oW2) / kH, n = (p - oW2) % kH;
        w2t[n * kLdW2 + k] = __float2bfloat16_rn(th);
        w2n[k * kLdW2 + n] = __float2bfloat16_rn(th);
    }
}

// BF16 copies of W1 and W2 from the master weights (after set_params).
__global__ void k_mlp_copies(const float *__restrict__ master, __nv_bfloat16 *__restrict__ w1t,
                             __nv_bfloat16 *__restrict__ w2t, __nv_bfloat16 *__restrict__ w2n) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < oB1) {
        const int k = p / kH, n = p % kH;
        w1t[n * kLdW1 + k] = __float2bfloat16_rn(master[p]);
    } else if (p >= oW2 && p < oB2) {
        const int k = (p - oW2) / kH, n = (p - oW2) % kH;
        w2t[n * kLdW2 + k] = __float2bfloat16_rn(master[p]);
        w2n[k * kLdW2 + n] = __float2bfloat16_rn(master[p]);
    }
}

// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014) of a counter.
uint64_t splitmix64(uint64_t x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

}  // namespace

struct cs_mlp {
    int device = 0;
    cudaStream_t stream = nullptr;
    int n_sm = 0;
    std::string err;
    float *master = nullptr, *m1 = nullptr, *m2 = nullptr, *grad = nullptr, *h_sse = nullptr;
    uint32_t *failed = nullptr;  // set by a training kernel that gave up waiting: no update
    __nv_bfloat16 *w1t = nullptr, *w2t = nullptr, *w2n = nullptr;
    float *partial = nullptr;
    int n_part_cap = 0;
    int64_t steps = 0;
    bool lose_product = false;  // cs_debug_mlp_lose_product
    // the same for the host (pinned, behind the sum of the squared errors)
    volatile uint32_t *gave_up() const { return reinterpret_cast<volatile uint32_t *>(h_sse + 2); }
};

namespace {

int mfail(cs_mlp *m, int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    m->err = buf;
    return code;
}

int failed_step(cs_mlp *m) {
    return mfail(m, CS_ERR_CUDA, "a training step gave up waiting for its tensor-core products or inputs: the parameters "
                 "are those before it (cs_mlp_set_params to go on)");
}

#define MLP_CUDA(m, call)                                                                         \
    do {                                                                                          \
        cudaError_t e_ = (call);                                                                  \
        if (e_ != cudaSuccess) {                                                                  \
            cudaGetLastError();                                                                   \
            return mfail(m, e_ == cudaErrorMemoryAllocation ? CS_ERR_OOM : CS_ERR_CUDA, "%s: %s", \
                         #call, cudaGetErrorString(e_));                                          \
        }                                                                                         \
    } while (0)

bool aligned(const void *p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

int grid_for(const cs_mlp *m, int64_t n, int rows, int per_sm) {
    return (int)std::min<int64_t>((n + rows - 1) / rows, (int64_t)per_sm * m->n_sm);
}

int refresh_copies(cs_mlp *m) {
    MLP_CUDA(m, cudaMemsetAsync(m->w1t, 0, kW1Elems * 2, m->stream));
    MLP_CUDA(m, cudaMemsetAsync(m->w2t, 0, kW2Elems * 2, m->stream));
    MLP_CUDA(m, cudaMemsetAsync(m->w2n, 0, kW2Elems * 2, m->stream));
    k_mlp_copies<<<(kP + 255) / 256, 256, 0, m->stream>>>(m->master, m->w1t, m->w2t, m->w2n);
    MLP_CUDA(m, cudaGetLastError());
    return CS_OK;
}

}  // namespace

extern "C" {

int cs_mlp_create(cs_mlp **out, int32_t device, void *stream, uint64_t seed) {
    if (!out) return CS_ERR_ARG;
    *out = nullptr;
    cs_mlp *m = new cs_mlp();
    m->device = device;
    m->stream = reinterpret_cast<cudaStream_t>(stream);
    auto bail = [&](int code) {
        cs_mlp_destroy(m);
        return code;
    };
    if (cudaSetDevice(device) != cudaSuccess) return bail(CS_ERR_CUDA);
    if (cudaDeviceGetAttribute(&m->n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return bail(CS_ERR_CUDA);
    if (cudaMalloc(&m->master, kP * 4) != cudaSuccess || cudaMalloc(&m->m1, kP * 4) != cudaSuccess ||
        cudaMalloc(&m->m2, kP * 4) != cudaSuccess || cudaMalloc(&m->grad, kP * 4) != cudaSuccess ||
        cudaMalloc(&m->failed, sizeof(uint32_t)) != cudaSuccess || cudaMalloc(&m->w1t, kW1Elems * 2) != cudaSuccess ||
        cudaMalloc(&m->w2t, kW2Elems * 2) != cudaSuccess || cudaMalloc(&m->w2n, kW2Elems * 2) != cudaSuccess ||
        cudaMallocHost(&m->h_sse, 16) != cudaSuccess) {
        cudaGetLastError();
        return bail(CS_ERR_OOM);
    }
    if (cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemTc) != cudaSuccess)
        return bail(CS_ERR_CUDA);
    // initial weights from the counter-based generator
    std::vector<float> p(kP, 0.0f);
    auto uni = [&](uint64_t i) {  // uniform in [-1, 1)
        return (float)((double)(splitmix64(seed * 0x100000001B3ull + i) >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0);
    };
    const float s1 = std::sqrt(6.0f / 36.0f), s2 = std::sqrt(6.0f / 64.0f), s3 = std::sqrt(3.0f / 64.0f);
    for (int k = 0; k < 36; ++k)
        for (int n = 0; n < kH; ++n) p[oW1 + k * kH + n] = s1 * uni(oW1 + k * kH + n);
    for (int i = 0; i < kH * kH; ++i) p[oW2 + i] = s2 * uni(oW2 + i);
    for (int i = 0; i < kH; ++i) p[oW3 + i] = s3 * uni(oW3 + i);
    int rc = cs_mlp_set_params(m, p.data());
    if (rc != CS_OK) return bail(rc);
    *out = m;
    return CS_OK;
}

void cs_mlp_destroy(cs_mlp *m) {
    if (!m) return;
    cudaSetDevice(m->device);
    if (m->stream) cudaStreamSynchronize(m->stream);
    cudaFree(m->master);
    cudaFree(m->m1);
    cudaFree(m->m2);
    cudaFree(m->grad);
    cudaFree(m->failed);
    cudaFree(m->w1t);
    cudaFree(m->w2t);
    cudaFree(m->w2n);
    cudaFree(m->partial);
    cudaFreeHost(m->h_sse);
    delete m;
}

const char *cs_mlp_last_error(const cs_mlp *m) { return m ? m->err.c_str() : "null MLP"; }

int cs_mlp_get_params(cs_mlp *m, float *host_out) {
    if (!m) return CS_ERR_ARG;
    if (!host_out) return mfail(m, CS_ERR_ARG, "NULL output");
    MLP_CUDA(m, cudaSetDevice(m->device));
    MLP_CUDA(m, cudaMemcpyAsync(host_out, m->master, kP * 4, cudaMemcpyDeviceToHost, m->stream));
    MLP_CUDA(m, cudaStreamSynchronize(m->stream));
    return *m->gave_up() ? failed_step(m) : CS_OK;
}

int cs_mlp_set_params(cs_mlp *m, const float *host_in) {
    if (!m) return CS_ERR_ARG;
    if (!host_in) return mfail(m, CS_ERR_ARG, "NULL parameters");
    for (int i = 0; i < kP; ++i)
        if (!std::isfinite(host_in[i])) return mfail(m, CS_ERR_ARG, "parameter %d is not finite", i);
    MLP_CUDA(m, cudaSetDevice(m->device));
    MLP_CUDA(m, cudaMemcpyAsync(m->master, host_in, kP * 4, cudaMemcpyHostToDevice, m->stream));
    MLP_CUDA(m, cudaMemsetAsync(m->m1, 0, kP * 4, m->stream));
    MLP_CUDA(m, cudaMemsetAsync(m->m2, 0, kP * 4, m->stream));
    MLP_CUDA(m, cudaMemsetAsync(m->failed, 0, sizeof(uint32_t), m->stream));
    int rc = refresh_copies(m);
    if (rc != CS_OK) return rc;
    MLP_CUDA(m, cudaStreamSynchronize(m->stream));
    *m->gave_up() = 0u;
    m->steps = 0;
    return CS_OK;
}

int cs_mlp_forward(cs_mlp *m, int64_t n, const float *feat, const int32_t *band, float *score_out) {
    if (!m) return CS_ERR_ARG;
    if (n < 0) return mfail(m, CS_ERR_ARG, "n must be >= 0");
    if (n == 0) return CS_OK;
    if (n > (int64_t)INT32_MAX) return mfail(m, CS_ERR_CAPACITY, "n exceeds 2^31 - 1");
    if (!feat || !band || !score_out || !aligned(feat, 8) || !aligned(band, 4) || !aligned(score_out, 4))
        return mfail(m, CS_ERR_ARG, "NULL or misaligned array");
    MLP_CUDA(m, cudaSetDevice(m->device));
    const int tiles = (int)((n + kTile - 1) / kTile);
    Weights W{m->w1t, m->w2t, m->w2n, m->master};
    k_mlp<<<grid_for(m, n, kTile, 2), kThreads, kSmemWeights, m->stream>>>(n, tiles, feat, band, W, score_out);
    MLP_CUDA(m, cudaGetLastError());
    return CS_OK;
}

int cs_mlp_train_step(cs_mlp *m, int64_t n, const float *feat, const int32_t *band, const float *target, float lr,
                      float *loss_out) {
    if (!m) return CS_ERR_ARG;
    if (n < 1) return mfail(m, CS_ERR_ARG, "n must be >= 1");
    if (n > (int64_t)INT32_MAX) return mfail(m, CS_ERR_CAPACITY, "n exceeds 2^31 - 1");
    if (!(lr > 0.0f) || !std::isfinite(lr)) return mfail(m, CS_ERR_ARG, "lr must be > 0");
    if (!feat || !band || !target || !aligned(feat, 8) || !aligned(band, 4) || !aligned(target, 4))
        return mfail(m, CS_ERR_ARG, "NULL or misaligned array");
    if (*m->gave_up()) return failed_step(m);
    MLP_CUDA(m, cudaSetDevice(m->device));
    const int grid = grid_for(m, n, kTcRows, 1);
    if (grid > m->n_part_cap) {
        MLP_CUDA(m, cudaStreamSynchronize(m->stream));
        cudaFree(m->partial);
        m->partial = nullptr;
        m->n_part_cap = 0;
        MLP_CUDA(m, cudaMalloc(&m->partial, (size_t)grid * (kP + 1) * 4));
        m->n_part_cap = grid;
    }
    const int tiles = (int)((n + kTcRows - 1) / kTcRows);
    Weights W{m->w1t, m->w2t, m->w2n, m->master};
    k_mlp_train<<<grid, kTcThreads, kSmemTc, m->stream>>>(n, tiles, feat, band, target, W, (float)(1.0 / (double)n),
                                                          aligned(feat, 16), m->lose_product, m->partial, m->failed,
                                                          m->gave_up());
    MLP_CUDA(m, cudaGetLastError());
    const int64_t t = m->steps + 1;
    const float bc1 = (float)(1.0 - std::pow(0.9, (double)t)), bc2 = (float)(1.0 - std::pow(0.999, (double)t));
    k_mlp_adam<<<(kP + 1 + 31) / 32, 32 * kAdamWarps, 0, m->stream>>>(grid, m->partial, m->master, m->m1, m->m2, m->grad,
                                                              m->w1t, m->w2t, m->w2n, lr, bc1, bc2, m->h_sse, m->failed);
    MLP_CUDA(m, cudaGetLastError());
    m->steps = t;
    if (loss_out) {
        MLP_CUDA(m, cudaStreamSynchronize(m->stream));
        if (*m->gave_up()) {
            m->steps = t - 1;
            return failed_step(m);
        }
        *loss_out = (float)((double)*static_cast<volatile float *>(m->h_sse) / (double)n);
    }
    return CS_OK;
}

int cs_mlp_get_grad(cs_mlp *m, float *host_out) {
    if (!m) return CS_ERR_ARG;
    if (!host_out) return mfail(m, CS_ERR_ARG, "NULL output");
    if (m->steps == 0 && !*m->gave_up()) return mfail(m, CS_ERR_STATE, "no training step yet");
    MLP_CUDA(m, cudaSetDevice(m->device));
    MLP_CUDA(m, cudaMemcpyAsync(host_out, m->grad, kP * 4, cudaMemcpyDeviceToHost, m->stream));
    MLP_CUDA(m, cudaStreamSynchronize(m->stream));
    return *m->gave_up() ? failed_step(m) : CS_OK;
}

int cs_debug_mlp_lose_product(cs_mlp *m, int32_t on) {
    if (!m) return CS_ERR_ARG;
    m->lose_product = on != 0;
    return CS_OK;
}

}  // extern "C"
