// cs_sort.cu -- tile binning and the (tile, depth) sort of a CrowdSplat frame.
//
// The 3DGS rasteriser the paper renders with (CrowdSplat Sec. 1 and Sec. 2
// cite Kerbl et al. 2023) duplicates each splat into every 16x16 tile its
// support box touches and sorts the (tile, depth) keys so that each tile
// can composite its splats front to back.  Here the order is reached in two
// stable stages instead of one 64-bit sort:
//   1. a stable LSD radix sort of the splats by depth key (as many bits as
//      the frame's depth range needs, digits of at most 9 bits);
//   2. pairs are emitted in that depth order (prefix sum of tile counts),
//      then a stable LSD radix sort by tile index (16-bit keys, 13 bits at
//      1080p as 7 + 6) leaves every tile's pairs in (depth, splat id) order.
// Each radix pass is reduce-then-scan (histogram of each digit per block,
// one CTA per digit scanning its row of block counts, scatter): no
// inter-block waits, and the order is deterministic.  Sorts of up to eight
// blocks run in one launch of a thread-block cluster.
#include <cooperative_groups.h>

#include <algorithm>

#include "cs_internal.cuh"

namespace cs {

namespace cg = cooperative_groups;

// ---------------------------------------------------------------------------
// exclusive scan of uint32 (three kernels: tile sums, spine, down-sweep)
// ---------------------------------------------------------------------------

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *total) {
    return block_exclusive_scan(v, total);
}

// element i of a scan input: plain value (MODE 0) or pair count of a bin
// word (MODE 1)
template <int MODE>
__device__ __forceinline__ uint32_t scan_load(const uint32_t *in, uint32_t i) {
    return MODE == 1 ? bin_count(in[i]) : in[i];
}

template <int MODE>
__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const uint32_t *__restrict__ in,
                                                              uint32_t n, uint32_t *__restrict__ sums) {
    __shared__ uint32_t total;
    const uint32_t base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    uint32_t v = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
        if (base + k < n) v += scan_load<MODE>(in, base + k);
    block_excl_scan(v, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// Exclusive scan of the block sums in place by one block of kThreads threads,
// total at sums[nb] and, when set, at host[0] in pinned host memory, then seq
// at host[2] (read past L1: other CTAs may have written them in this launch).
template <int kThreads>
__device__ __forceinline__ void scan_sums(uint32_t *sums, uint32_t nb, uint32_t *total, uint32_t *host, uint32_t seq) {
    constexpr int kPer = kScanTile / kThreads;
    uint32_t carry = 0;
    for (uint32_t base = 0; base < nb; base += kScanTile) {
        const uint32_t i0 = base + threadIdx.x * kPer;
        uint32_t v[kPer], sum = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            v[k] = i0 + k < nb ? __ldcg(sums + i0 + k) : 0u;
            sum += v[k];
        }
        uint32_t ex = block_excl_scan(sum, total) + carry;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            if (i0 + k < nb) sums[i0 + k] = ex;
            ex += v[k];
        }
        carry += *total;
    }
    if (threadIdx.x == 0) {
        sums[nb] = carry;
        if (host) {
            host[0] = carry;
            __threadfence_system();
            *reinterpret_cast<volatile uint32_t *>(host + 2) = seq;
        }
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_spine(uint32_t *sums, uint32_t nb, uint32_t *host, uint32_t seq) {
    __shared__ uint32_t total;
    scan_sums<kScanThreads>(sums, nb, &total, host, seq);
}

template <int MODE>
__global__ void __launch_bounds__(kScanThreads) k_scan_down(const uint32_t *__restrict__ in, uint32_t n,
                                                            const uint32_t *__restrict__ sums,
                                                            uint32_t nb, uint32_t *__restrict__ out) {
    __shared__ uint32_t total;
    const uint32_t base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = base + k < n ? scan_load<MODE>(in, base + k) : 0u;
        s += v[k];
    }
    uint32_t ex = block_excl_scan(s, &total) + sums[blockIdx.x];
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < n) out[base + k] = ex;
        ex += v[k];
    }
    if (blockIdx.x == nb - 1 && threadIdx.x == 0) out[n] = sums[nb];
}

size_t scan_scratch_words(size_t n) { return (n + kScanTile - 1) / kScanTile + 1; }

template <int MODE>
static int scan_impl(const uint32_t *in, uint32_t *out, uint32_t n, uint32_t *scratch, cudaStream_t st) {
    if (n == 0) {
        cudaMemsetAsync(out, 0, sizeof(uint32_t), st);
        return 0;
    }
    const uint32_t nb = (n + kScanTile - 1) / kScanTile;
    k_scan_reduce<MODE><<<nb, kScanThreads, 0, st>>>(in, n, scratch);
    k_scan_spine<<<1, kScanThreads, 0, st>>>(scratch, nb, nullptr, 0u);
    k_scan_down<MODE><<<nb, kScanThreads, 0, st>>>(in, n, scratch, nb, out);
    return 3;
}

int exclusive_scan(const uint32_t *in, const uint32_t *, uint32_t *out, uint32_t n, uint32_t *scratch,
                   cudaStream_t st) {
    return scan_impl<0>(in, out, n, scratch, st);
}

int exclusive_scan_bins(const uint32_t *bins, uint32_t *out, uint32_t n, uint32_t *scratch, cudaStream_t st) {
    return scan_impl<1>(bins, out, n, scratch, st);
}

// ---------------------------------------------------------------------------
// stable LSD radix sort, digits of up to 9 bits, reduce-then-scan per pass
//
// A sort of b-bit keys takes ceil(b / 9) passes of near-equal digit width
// (13-bit tile keys: 7 + 6 bits; 26-bit depth keys: 9 + 9 + 8; 32-bit keys:
// 4 x 8): a narrower digit needs fewer ballots to rank and smaller count
// tables, a wider one may save a pass.  A block owns
// 4,096 consecutive elements; warp w owns 512 of them, read in 16 rounds of
// 32 consecutive elements (coalesced, all loads issued before any
// shared-memory update).  Histogram pass: per-warp digit counts (shared
// atomics), one row per digit in the global count matrix (digit-major),
// which an exclusive scan turns into each block's global digit offsets.
// Scatter pass: stable ranks from per-warp running counts, the lanes that
// share a digit found with one ballot per digit bit, then a block-local
// sort in shared memory, then each digit's run is written out with
// consecutive threads on consecutive addresses.
// ---------------------------------------------------------------------------

constexpr int kRadixThreads = 256;
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kRadixItems = 16;                              // per lane
constexpr int kRadixTile = kRadixThreads * kRadixItems;      // per block (4,096)
constexpr int kRadixWarpTile = 32 * kRadixItems;             // per warp (512)
constexpr int kRadixMaxBits = 9;
constexpr int kRadixDigits = 1 << kRadixMaxBits;             // largest digit range

template <typename K, int kBits>
__global__ void __launch_bounds__(kRadixThreads) k_radix_hist(const K *__restrict__ keys, uint32_t n,
                                                              int shift, uint32_t *__restrict__ hist,
                                                              uint32_t nblocks) {
    constexpr uint32_t kDigits = 1u << kBits;
    __shared__ uint32_t h[kRadixWarps][kDigits];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int d = threadIdx.x; d < kRadixWarps * (int)kDigits; d += kRadixThreads) (&h[0][0])[d] = 0;
    const uint32_t base = blockIdx.x * kRadixTile + warp * kRadixWarpTile;
    uint32_t dig[kRadixItems];
    const K *block = keys + (size_t)blockIdx.x * kRadixTile;
    if (blockIdx.x < n / kRadixTile && (reinterpret_cast<uintptr_t>(block) & 15u) == 0u) {
        // a full block: 16-byte loads (the counts don't depend on the order)
        constexpr int kVec = 16 / (int)sizeof(K);
#pragma unroll
        for (int r = 0; r < kRadixItems; r += kVec) {
            const uint4 u = __ldg(reinterpret_cast<const uint4 *>(block) + (r / kVec) * kRadixThreads + threadIdx.x);
            const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int j = 0; j < kVec; ++j)
                dig[r + j] = (w[j * (int)sizeof(K) / 4] >> (8 * (j * (int)sizeof(K) % 4) + shift)) & (kDigits - 1);
        }
    } else {
#pragma unroll
        for (int r = 0; r < kRadixItems; ++r) {
            const uint32_t i = base + r * 32 + lane;
            dig[r] = i < n ? (uint32_t)((keys[i] >> shift) & (kDigits - 1)) : kDigits;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRadixItems; ++r)
        if (dig[r] < kDigits) atomicAdd(&h[warp][dig[r]], 1u);
    __syncthreads();
    for (int d = threadIdx.x; d < (int)kDigits; d += kRadixThreads) {
        uint32_t s = 0;
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) s += h[w][d];
        hist[(size_t)d * nblocks + blockIdx.x] = s;
    }
}

// Exclusive scan of each digit's row of the (digit, block) count matrix
// (digit-major), one CTA per digit: offs[d][b] = counts of digit d in blocks
// before b; tot[d] = the digit's total.  The scatter adds the digit's base
// (an exclusive scan of tot it computes itself).
__global__ void __launch_bounds__(kScanThreads) k_radix_rowscan(const uint32_t *__restrict__ hist, uint32_t nb,
                                                                uint32_t *__restrict__ offs,
                                                                uint32_t *__restrict__ tot) {
    __shared__ uint32_t total;
    const uint32_t *row = hist + (size_t)blockIdx.x * nb;
    uint32_t *orow = offs + (size_t)blockIdx.x * nb;
    uint32_t carry = 0;
    for (uint32_t base = 0; base < nb; base += kScanTile) {
        const uint32_t i0 = base + threadIdx.x * kScanItems;
        uint32_t v[kScanItems], sum = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            v[k] = i0 + k < nb ? row[i0 + k] : 0u;
            sum += v[k];
        }
        uint32_t ex = block_excl_scan(sum, &total) + carry;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            if (i0 + k < nb) orow[i0 + k] = ex;
            ex += v[k];
        }
        carry += total;
    }
    if (threadIdx.x == 0) tot[blockIdx.x] = carry;
}

// One block of the scatter; kFull: all kRadixTile elements are there, no
// index is compared with n.
template <typename K, int kBits, bool kFull>
__device__ __forceinline__ void radix_scatter_block(uint32_t (*wcnt)[1 << kBits], uint32_t *delta, uint32_t *total,
                                                    K *skey, uint32_t *sval, const K *__restrict__ kin,
                                                    const uint32_t *__restrict__ vin, K *__restrict__ kout,
                                                    uint32_t *__restrict__ vout, uint32_t n, int shift,
                                                    const uint32_t *__restrict__ offs,
                                                    const uint32_t *__restrict__ dtot_g, uint32_t nblocks,
                                                    const uint32_t *__restrict__ gsrc, uint32_t *__restrict__ gdst) {
    constexpr uint32_t kDigits = 1u << kBits;
    constexpr int kPer = kDigits > (uint32_t)kRadixThreads ? (int)kDigits / kRadixThreads : 1;  // digits per thread
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t blk0 = blockIdx.x * kRadixTile;
    const uint32_t base = blk0 + warp * kRadixWarpTile + lane;
    const uint32_t mine = kFull ? kRadixTile : n - blk0;  // elements of the block
    K k[kRadixItems];
    uint32_t v[kRadixItems], dr[kRadixItems];  // digit | rank << 16
#pragma unroll
    for (int r = 0; r < kRadixItems; ++r) {
        const uint32_t i = base + r * 32;
        const bool ok = kFull || i < n;
        k[r] = ok ? kin[i] : (K)0;
        v[r] = ok ? (vin ? vin[i] : i) : 0u;
    }
    __syncthreads();
    // stable rank within the warp's 512 elements
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < kRadixItems; ++r) {
        const bool ok = kFull || base + r * 32 < n;
        const uint32_t d = (uint32_t)(k[r] >> shift) & (kDigits - 1);
        // lanes holding the same digit: agree on all kBits bits, among valid lanes
        unsigned peers = kFull ? 0xffffffffu : __ballot_sync(0xffffffffu, ok);
#pragma unroll
        for (int b = 0; b < kBits; ++b) {
            const bool bit = (d >> b) & 1u;
            const unsigned m = __ballot_sync(0xffffffffu, bit);
            peers &= m ^ (bit ? 0u : 0xffffffffu);
        }
        const uint32_t before = wcnt[warp][d], below = __popc(peers & lt);
        __syncwarp();
        if (ok && below == 0u) wcnt[warp][d] = before + __popc(peers);
        __syncwarp();
        dr[r] = d | ((before + below) << 16);
    }
    __syncthreads();
    // per digit (thread t: digits t kPer .. t kPer + kPer - 1): the digit's
    // block total from the warps' counts, and its global total for the digit
    // bases
    uint32_t tot = 0, dtot[kPer], gtot = 0, gt[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int d = threadIdx.x * kPer + j;
        dtot[j] = 0;
        gt[j] = 0;
        if (d < (int)kDigits) {
#pragma unroll
            for (int w = 0; w < kRadixWarps; ++w) dtot[j] += wcnt[w][d];
            tot += dtot[j];
            gt[j] = dtot_g[d];
            gtot += gt[j];
        }
    }
    // block-local digit starts
    uint32_t ex = block_excl_scan(tot, total);
    // global digit bases: exclusive scan of the digit totals
    uint32_t gex = block_excl_scan(gtot, total);
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int d = threadIdx.x * kPer + j;
        if (d < (int)kDigits) {
            // a block-local position p of digit d goes to delta[d] + p
            delta[d] = gex + offs[(size_t)d * nblocks + blockIdx.x] - ex;
            uint32_t run = ex;
#pragma unroll
            for (int w = 0; w < kRadixWarps; ++w) {
                const uint32_t c = wcnt[w][d];
                wcnt[w][d] = run;
                run += c;
            }
        }
        ex += dtot[j];
        gex += gt[j];
    }
    __syncthreads();
    // block-local sort in shared memory
#pragma unroll
    for (int r = 0; r < kRadixItems; ++r) {
        if (kFull || base + r * 32 < n) {
            const uint32_t lp = wcnt[warp][dr[r] & 0xFFFFu] + (dr[r] >> 16);
            skey[lp] = k[r];
            sval[lp] = v[r];
        }
    }
    __syncthreads();
    // runs of equal digits go to consecutive global addresses
#pragma unroll 4
    for (int r = 0; r < kRadixItems; ++r) {
        const uint32_t p = threadIdx.x + r * kRadixThreads;
        if (!kFull && p >= mine) break;
        const K key = skey[p];
        const uint32_t g = delta[(uint32_t)(key >> shift) & (kDigits - 1)] + p;
        const uint32_t val = sval[p];
        if (!in_bounds(g < n, kChkSort)) continue;
        kout[g] = key;
        vout[g] = val;
        if (gdst && in_bounds(val < n, kChkSort)) gdst[g] = gsrc[val];
    }
}

// Bound by the latency of the block's phases and by instruction issue (48% of
// the slots, 114 instructions per 32 elements with 9-bit digits).  14.5 M
// depth keys, 9 bits: 103 -> 94 us, 20.5 M pairs, 6 bits: 98 -> 79 us against
// index comparisons in full blocks, digit starts kept apart from the warps'
// offsets and a base and a start read per element written; the histograms
// 22 -> 20 and 15 -> 12 us with 16-byte loads.
template <typename K, int kBits>
__global__ void __launch_bounds__(kRadixThreads, 3) k_radix_scatter(
    const K *__restrict__ kin, const uint32_t *__restrict__ vin, K *__restrict__ kout,
    uint32_t *__restrict__ vout, uint32_t n, int shift, const uint32_t *__restrict__ offs,
    const uint32_t *__restrict__ dtot_g, uint32_t nblocks, const uint32_t *__restrict__ gsrc,
    uint32_t *__restrict__ gdst) {
    constexpr uint32_t kDigits = 1u << kBits;
    __shared__ uint32_t wcnt[kRadixWarps][kDigits];  // running counts, then block-local positions
    __shared__ uint32_t delta[kDigits];              // global less block-local start of each digit
    __shared__ uint32_t total;
    // block-local sort buffers (dynamic: with 9-bit digits the CTA needs
    // more than the 48 KB of static shared memory)
    extern __shared__ __align__(16) unsigned char radix_dyn[];
    uint32_t *sval = reinterpret_cast<uint32_t *>(radix_dyn);
    K *skey = reinterpret_cast<K *>(radix_dyn + kRadixTile * sizeof(uint32_t));
    for (int d = threadIdx.x; d < kRadixWarps * (int)kDigits; d += kRadixThreads) (&wcnt[0][0])[d] = 0;
    if (blockIdx.x < n / kRadixTile)
        radix_scatter_block<K, kBits, true>(wcnt, delta, &total, skey, sval, kin, vin, kout, vout, n, shift, offs,
                                            dtot_g, nblocks, gsrc, gdst);
    else
        radix_scatter_block<K, kBits, false>(wcnt, delta, &total, skey, sval, kin, vin, kout, vout, n, shift, offs,
                                             dtot_g, nblocks, gsrc, gdst);
}

// The whole sort of up to kClusterBlocks blocks in one launch: a cluster of
// CTAs, one per 4,096 elements, runs every pass, reading the other CTAs'
// digit counts from their shared memory and handing the elements on through
// global memory (L2), with two cluster barriers a pass.  Such sorts are
// bound by launches: three kernels a pass, each shorter than the gap to the
// next.  Same digits, same order.  A 256x256 frame of 16,384 splats: 194 ->
// 162 us; a training frame of 12,291 splats: 424 -> 394 us.
constexpr int kClusterBlocks = 8;  // the portable cluster size
// Twice the threads of the pass-by-pass kernels, half the elements each: one
// block's latency is all there is (158 -> 154 us for the 256x256 frame; large
// sorts lose from it, 2,197 -> 2,285 us for 5,000 characters).  Elements handed
// on by stores to the other CTAs' shared memory instead: 165 us.
constexpr int kClusterThreads = 512, kClusterWarps = kClusterThreads / 32;
constexpr int kClusterItems = kRadixTile / kClusterThreads, kClusterWarpTile = 32 * kClusterItems;

// Digit width of pass p of `passes` over `bits` bits, from bit `shift` on.
__host__ __device__ inline int radix_width(int bits, int shift, int passes, int p) {
    const int w = (bits - shift + (passes - p) - 1) / (passes - p);
    return w < 4 ? 4 : w;
}

template <typename K>
__global__ void __launch_bounds__(kClusterThreads) k_radix_cluster(K *k0, uint32_t *v0, K *k1, uint32_t *v1, uint32_t n,
                                                                 int bits, int passes, bool iota,
                                                                 const uint32_t *__restrict__ gsrc,
                                                                 uint32_t *__restrict__ gdst) {
    __shared__ uint32_t wcnt[kClusterWarps][kRadixDigits];  // running counts, then warp offsets
    __shared__ uint32_t dcnt[kRadixDigits];               // this block's digit counts, read by the cluster
    __shared__ uint32_t dstart[kRadixDigits], gbase[kRadixDigits];
    __shared__ uint32_t total;
    extern __shared__ __align__(16) unsigned char cluster_dyn[];
    uint32_t *sval = reinterpret_cast<uint32_t *>(cluster_dyn);
    K *skey = reinterpret_cast<K *>(cluster_dyn + kRadixTile * sizeof(uint32_t));
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), blocks = (int)cluster.num_blocks();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t blk0 = (uint32_t)rank * kRadixTile, base = blk0 + warp * kClusterWarpTile;
    constexpr int kPer = kRadixDigits / kClusterThreads;  // digits per thread
    for (int p = 0, shift = 0; p < passes; ++p) {
        const int width = radix_width(bits, shift, passes, p);
        const uint32_t mask = (1u << width) - 1u;
        const K *ki = p & 1 ? k1 : k0;
        const uint32_t *vi = p & 1 ? v1 : v0;
        K *ko = p & 1 ? k0 : k1;
        uint32_t *vo = p & 1 ? v0 : v1;
        for (int d = threadIdx.x; d < kClusterWarps * kRadixDigits; d += kClusterThreads) (&wcnt[0][0])[d] = 0;
        K k[kClusterItems];
        uint32_t v[kClusterItems], dr[kClusterItems];
#pragma unroll
        for (int r = 0; r < kClusterItems; ++r) {
            // past L1: another CTA of the cluster wrote them in the pass before
            const uint32_t i = base + r * 32 + lane;
            k[r] = i < n ? __ldcg(ki + i) : (K)0;
            v[r] = i >= n ? 0u : (p == 0 && iota ? i : __ldcg(vi + i));
        }
        __syncthreads();
        // stable rank within the warp's elements, as k_radix_scatter
#pragma unroll
        for (int r = 0; r < kClusterItems; ++r) {
            const bool ok = base + r * 32 + lane < n;
            const uint32_t d = ok ? (uint32_t)(k[r] >> shift) & mask : (uint32_t)kRadixDigits;
            unsigned peers = __ballot_sync(0xffffffffu, ok);
            for (int b = 0; b < width; ++b) {
                const unsigned m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
                peers &= ((d >> b) & 1u) ? m : ~m;
            }
            const uint32_t before = ok ? wcnt[warp][d] : 0u;
            __syncwarp();
            if (ok && (peers & lt) == 0u) wcnt[warp][d] = before + __popc(peers);
            __syncwarp();
            dr[r] = d | ((before + __popc(peers & lt)) << 16);
        }
        __syncthreads();
        uint32_t mine[kPer], tot = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int d = threadIdx.x * kPer + j;
            uint32_t run = 0;
#pragma unroll
            for (int w = 0; w < kClusterWarps; ++w) {
                const uint32_t c = wcnt[w][d];
                wcnt[w][d] = run;
                run += c;
            }
            dcnt[d] = mine[j] = run;
            tot += run;
        }
        cluster.sync();  // every block's digit counts are there
        uint32_t pre[kPer], all[kPer], gtot = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) pre[j] = all[j] = 0;
        for (int b = 0; b < blocks; ++b) {
            const uint32_t *other = cluster.map_shared_rank(dcnt, b);
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const uint32_t c = other[threadIdx.x * kPer + j];
                if (b < rank) pre[j] += c;
                all[j] += c;
            }
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) gtot += all[j];
        uint32_t ex = block_excl_scan(tot, &total), gex = block_excl_scan(gtot, &total);
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int d = threadIdx.x * kPer + j;
            dstart[d] = ex;
            gbase[d] = gex + pre[j];
            ex += mine[j];
            gex += all[j];
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kClusterItems; ++r) {
            const uint32_t d = dr[r] & 0xFFFFu;
            if (d < (uint32_t)kRadixDigits) {
                const uint32_t lp = dstart[d] + wcnt[warp][d] + (dr[r] >> 16);
                skey[lp] = k[r];
                sval[lp] = v[r];
            }
        }
        __syncthreads();
        const uint32_t cnt = n > blk0 ? min((uint32_t)kRadixTile, n - blk0) : 0u;
        const bool last = p == passes - 1;
        for (uint32_t q = threadIdx.x; q < cnt; q += kClusterThreads) {
            const K key = skey[q];
            const uint32_t d = (uint32_t)(key >> shift) & mask;
            const uint32_t g = gbase[d] + (q - dstart[d]);
            const uint32_t val = sval[q];
            if (!in_bounds(g < n, kChkSort)) continue;
            ko[g] = key;
            vo[g] = val;
            if (last && gdst && in_bounds(val < n, kChkSort)) gdst[g] = gsrc[val];
        }
        shift += width;
        cluster.sync();  // the pass is written, and nobody reads these counts any more
    }
}

template <typename K>
static int radix_cluster(K *k0, uint32_t *v0, K *k1, uint32_t *v1, uint32_t n, uint32_t nb, int bits, int passes,
                         bool iota, const uint32_t *gsrc, uint32_t *gdst, cudaStream_t st) {
    constexpr int kDyn = kRadixTile * (int)(sizeof(uint32_t) + sizeof(K));
    static int configured_device = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_device != dev) {
        cudaFuncSetAttribute(k_radix_cluster<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDyn);
        configured_device = dev;
    }
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = nb;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = nb;
    cfg.blockDim = kClusterThreads;
    cfg.dynamicSmemBytes = kDyn;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_radix_cluster<K>, k0, v0, k1, v1, n, bits, passes, iota, gsrc, gdst);
    return 1;
}

size_t radix_scratch_words(size_t n) {
    size_t nb = (n + kRadixTile - 1) / kRadixTile;
    if (nb == 0) nb = 1;
    size_t hist = (size_t)kRadixDigits * nb;
    return 2 * hist + kRadixDigits;
}

// one pass over digit bits [shift, shift + kBits)
template <typename K, int kBits>
static int radix_pass(const K *ki, const uint32_t *vi, K *ko, uint32_t *vo, uint32_t n, int shift, uint32_t nb,
                      uint32_t *scratch, const uint32_t *gsrc, uint32_t *gdst, cudaStream_t st) {
    const uint32_t hn = (1u << kBits) * nb;
    uint32_t *hist = scratch;
    uint32_t *offs = scratch + hn;
    uint32_t *dtot = scratch + 2 * hn;
    constexpr int kDyn = kRadixTile * (int)(sizeof(uint32_t) + sizeof(K));
    static int configured_device = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_device != dev) {
        cudaFuncSetAttribute(k_radix_scatter<K, kBits>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDyn);
        configured_device = dev;
    }
    k_radix_hist<K, kBits><<<nb, kRadixThreads, 0, st>>>(ki, n, shift, hist, nb);
    k_radix_rowscan<<<1u << kBits, kScanThreads, 0, st>>>(hist, nb, offs, dtot);
    k_radix_scatter<K, kBits><<<nb, kRadixThreads, kDyn, st>>>(ki, vi, ko, vo, n, shift, offs, dtot, nb, gsrc,
                                                              gdst);
    return 3;
}

template <typename K>
static int radix_sort(K *k0, uint32_t *v0, K *k1, uint32_t *v1, uint32_t n, int bits,
                      uint32_t *scratch, cudaStream_t st, int *in_second, const uint32_t *gsrc,
                      uint32_t *gdst, bool iota_values) {
    *in_second = 0;
    if (n == 0 || bits <= 0) return 0;
    int launched = 0;
    const uint32_t nb = (n + kRadixTile - 1) / kRadixTile;
    // fewest passes of at most 9 bits, near-equal widths (4 bits at least)
    const int passes = (bits + kRadixMaxBits - 1) / kRadixMaxBits;
    if (nb <= (uint32_t)kClusterBlocks) {
        *in_second = passes & 1;
        return radix_cluster<K>(k0, v0, k1, v1, n, nb, bits, passes, iota_values, gsrc, gdst, st);
    }
    int cur = 0;
    for (int p = 0, shift = 0; p < passes; ++p) {
        const K *ki = cur ? k1 : k0;
        const uint32_t *vi = p == 0 && iota_values ? nullptr : (cur ? v1 : v0);
        K *ko = cur ? k0 : k1;
        uint32_t *vo = cur ? v0 : v1;
        const int width = radix_width(bits, shift, passes, p);
        const bool last = p == passes - 1;
        const uint32_t *gs = last ? gsrc : nullptr;
        uint32_t *gd = last ? gdst : nullptr;
        switch (width) {
            case 4: launched += radix_pass<K, 4>(ki, vi, ko, vo, n, shift, nb, scratch, gs, gd, st); break;
            case 5: launched += radix_pass<K, 5>(ki, vi, ko, vo, n, shift, nb, scratch, gs, gd, st); break;
            case 6: launched += radix_pass<K, 6>(ki, vi, ko, vo, n, shift, nb, scratch, gs, gd, st); break;
            case 7: launched += radix_pass<K, 7>(ki, vi, ko, vo, n, shift, nb, scratch, gs, gd, st); break;
            case 8: launched += radix_pass<K, 8>(ki, vi, ko, vo, n, shift, nb, scratch, gs, gd, st); break;
            default: launched += radix_pass<K, 9>(ki, vi, ko, vo, n, shift, nb, scratch, gs, gd, st); break;
        }
        shift += width;
        cur ^= 1;
    }
    *in_second = cur;
    return launched;
}

int radix_sort_u32(uint32_t *k0, uint32_t *v0, uint32_t *k1, uint32_t *v1, uint32_t n, int bits,
                   uint32_t *scratch, cudaStream_t st, int *in_second, const uint32_t *gather_src,
                   uint32_t *gather_dst, bool iota_values) {
    return radix_sort<uint32_t>(k0, v0, k1, v1, n, bits, scratch, st, in_second, gather_src, gather_dst,
                                iota_values);
}

int radix_sort_u16(uint16_t *k0, uint32_t *v0, uint16_t *k1, uint32_t *v1, uint32_t n, int bits,
                   uint32_t *scratch, cudaStream_t st, int *in_second) {
    return radix_sort<uint16_t>(k0, v0, k1, v1, n, bits, scratch, st, in_second, nullptr, nullptr, false);
}

// ---------------------------------------------------------------------------
// pair emission in depth order, tile ranges, live count
// ---------------------------------------------------------------------------

// Pairs of one splat: every tile its reach box meets, written to
// ptile / pval from position o (at most e - o of them).  Small splats carry
// those tiles as a 3x3 mask in their bin word (gathered into depth order by
// the depth sort); larger ones take the reach box from the record.
__device__ __forceinline__ void emit_splat_pairs(uint32_t b, uint32_t s, uint32_t o, uint32_t e,
                                                 const float4 *__restrict__ rec, int tiles_x,
                                                 uint16_t *__restrict__ ptile, uint32_t *__restrict__ pval,
                                                 uint32_t n_tiles, uint32_t n_pairs) {
    if (o >= e || !in_bounds(e <= n_pairs, kChkPair)) return;
    if (!(b & kBinLarge)) {
        const uint32_t x0 = b & 0xFFu, y0 = (b >> 8) & 0xFFu;
        uint32_t m = (b >> 16) & 0x1FFu;
        while (m && o < e) {
            const uint32_t k = __ffs(m) - 1;
            m &= m - 1;
            const uint32_t tile = (y0 + k / 3) * (uint32_t)tiles_x + x0 + k % 3;
            if (in_bounds(tile < n_tiles, kChkTile)) {
                ptile[o] = (uint16_t)tile;
                pval[o] = s;
            }
            ++o;
        }
        return;
    }
    const float4 r3 = rec[(size_t)s * kRecVec];  // reach x, reach y, log2 o, C
    const uint32_t rx = __float_as_uint(r3.x), ry = __float_as_uint(r3.y);
    const int ax0 = (int)(rx & 0xFFFFu), ax1 = (int)(rx >> 16);
    const int ay0 = (int)(ry & 0xFFFFu), ay1 = (int)(ry >> 16);
    for (int yy = ay0 >> 4; yy <= (ay1 >> 4); ++yy) {
        for (int xx = ax0 >> 4; xx <= (ax1 >> 4); ++xx) {
            if (o >= e) return;
            if (in_bounds((uint32_t)(yy * tiles_x + xx) < n_tiles, kChkTile)) {
                ptile[o] = (uint16_t)(yy * tiles_x + xx);
                pval[o] = s;
            }
            ++o;
        }
    }
}

// Thread per sorted splat, offsets from a scan of the sorted bin words.
__global__ void __launch_bounds__(256) k_emit_pairs(uint32_t n, const uint32_t *__restrict__ order,
                                                    const uint32_t *__restrict__ bins,
                                                    const uint32_t *__restrict__ pair_off,
                                                    const float4 *__restrict__ rec, int tiles_x, uint32_t n_tiles,
                                                    uint16_t *__restrict__ ptile,
                                                    uint32_t *__restrict__ pval) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t s = order[i];
    if (!in_bounds(s < n, kChkSplat)) return;
    emit_splat_pairs(bins[i], s, pair_off[i], pair_off[i + 1], rec, tiles_x, ptile, pval, n_tiles, pair_off[n]);
}

// Pair emission fused with the down-sweep of the pair-count scan.  A block
// takes 256 kRounds splats in depth order, warp w the 32 kRounds from
// w 32 kRounds on; the warp's offset is the scanned block sum plus the
// totals of the warps before it, so there is one barrier and no per-splat
// offset array.  Each step of 64 splats, two a lane, is scanned in the warp
// and its pairs are written 32 at a time, one per lane: the splats with pairs
// are left compacted in shared memory, a bit per splat start in the window of
// 32 pairs (one reduction) tells each lane its splat, and the pair's rank
// among the splat's tiles its tile (row-major; a 3x3 mask by a table of the
// positions of its set bits).  Exactly the pairs emit_splat_pairs writes, in
// their order.
// Bound by instruction issue (about 400 per 64 splats and their 90 pairs).
// 42.5 M pairs of 22.7 M splats: 228 us with 1,024-thread blocks, three
// barriers a round, small splats written by their own threads and larger ones
// queued; 178 with warps of 32 splats a step; 162 with 64 (fewer scans and
// fuller windows).  The sums before it 27 -> 18 us (16-byte loads).
constexpr int kEmitThreads = 256;
constexpr int kEmitWarps = kEmitThreads / 32;
// Blocks of 4,096 splats leave SMs idle below a few million splats (202,738
// splats are 50 blocks: 21 us, 13 with blocks of 1,024, 8 with
// blocks of 256); larger frames would only lengthen the one-block scan of the
// sums with smaller blocks.
constexpr int kEmitRounds = 16, kEmitFewRounds = 4, kEmitOneRound = 1;
constexpr size_t kEmitFewSplats = (size_t)1 << 22, kEmitOneSplats = (size_t)1 << 18;

// Pair counts of the blocks.  With the smallest blocks (few splats) the CTA
// that finishes last (a ticket taken after a memory fence) scans them, which
// as a launch of its own costs such a frame 4 us (16,384 splats 153 -> 148 us,
// 202,738 splats 334 -> 328 us a frame with the smaller blocks); with
// thousands of CTAs the fences cost more than the launch (22.7 M splats 2,664
// -> 2,680 us).
template <int kRounds>
__global__ void __launch_bounds__(kEmitThreads) k_bin_sums(const uint32_t *__restrict__ bins, uint32_t n,
                                                           uint32_t *sums, uint32_t *ticket, uint32_t *host,
                                                           uint32_t seq) {
    __shared__ uint32_t wsum[kEmitWarps], total;
    __shared__ bool last;
    const uint32_t base = blockIdx.x * (kEmitThreads * kRounds);
    uint32_t v = 0;
    if (kRounds == 1) {
        if (base + threadIdx.x < n) v = bin_count(bins[base + threadIdx.x]);
    } else {
#pragma unroll
        for (int j = 0; j < kRounds / 4; ++j) {
            const uint32_t i = base + (j * kEmitThreads + threadIdx.x) * 4u;
            if (i + 4u <= n) {
                const uint4 w = __ldg(reinterpret_cast<const uint4 *>(bins + i));  // (the words start 16-byte aligned)
                v += bin_count(w.x) + bin_count(w.y) + bin_count(w.z) + bin_count(w.w);
            } else {
                for (uint32_t k = i; k < n; ++k) v += bin_count(bins[k]);
            }
        }
    }
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < kEmitWarps; ++w) t += wsum[w];
        sums[blockIdx.x] = t;
        if (kRounds == kEmitOneRound) {
            __threadfence();
            last = atomicAdd(ticket, 1u) == gridDim.x - 1u;
        }
    }
    if (kRounds == kEmitOneRound) {
        __syncthreads();
        if (!last) return;
        __threadfence();
        scan_sums<kEmitThreads>(sums, gridDim.x, &total, host, seq);
    }
}

// Words i and i + 1 (i even, the array 8-byte aligned); zero from `end` on.
__device__ __forceinline__ uint2 load_two(const uint32_t *__restrict__ p, uint32_t i, uint32_t end) {
    if (i + 1u < end) return __ldg(reinterpret_cast<const uint2 *>(p + i));
    return make_uint2(i < end ? p[i] : 0u, 0u);
}

// A splat with pairs as its warp's lanes read it: splat id, first pair, tile
// x0 | y0 << 16, mask or kBinLarge | tiles per row.
__device__ __forceinline__ uint4 staged_splat(uint32_t b, uint32_t s, uint32_t first, const float4 *__restrict__ rec,
                                              uint32_t n) {
    uint4 e = make_uint4(s, first, (b & 0xFFu) | ((b & 0xFF00u) << 8), (b >> 16) & 0x1FFu);
    if ((b & kBinLarge) && in_bounds(s < n, kChkSplat)) {
        const float4 q = rec[(size_t)s * kRecVec];  // reach x, reach y, log2 o, C
        const uint32_t rx = __float_as_uint(q.x), ry = __float_as_uint(q.y);
        const uint32_t x0 = (rx & 0xFFFFu) >> 4, y0 = (ry & 0xFFFFu) >> 4;
        e.z = x0 | (y0 << 16);
        e.w = kBinLarge | (((rx >> 16) >> 4) - x0 + 1u);
    }
    return e;
}

template <int kRounds>
__global__ void __launch_bounds__(kEmitThreads, 8)
    k_emit_pairs_scan(uint32_t n, const uint32_t *__restrict__ order, const uint32_t *__restrict__ bins,
                      const uint32_t *__restrict__ sums, const float4 *__restrict__ rec, int tiles_x,
                      uint32_t n_tiles, uint16_t *__restrict__ ptile, uint32_t *__restrict__ pval,
                      uint2 *__restrict__ ranges, int32_t *__restrict__ blend_meta) {
    __shared__ uint4 stage[kEmitWarps][64];
    __shared__ uint32_t nth[512];            // positions of a mask's first eight set bits, four bits each
    __shared__ uint32_t wsum[kEmitWarps];
    for (uint32_t k = blockIdx.x * kEmitThreads + threadIdx.x; k < n_tiles; k += gridDim.x * kEmitThreads)
        ranges[k] = make_uint2(0u, 0u);
    if (blockIdx.x == 0 && threadIdx.x < kBlendMetaWords) blend_meta[threadIdx.x] = 0;
    const uint32_t n_pairs = CS_CHECKS ? sums[gridDim.x] : 0xFFFFFFFFu;  // the scan's total
    for (uint32_t m = threadIdx.x; m < 512u; m += kEmitThreads) {
        uint32_t x = 0, k = 0;
        for (uint32_t j = 0; j < 9u; ++j)
            if ((m >> j) & 1u) {
                if (k < 8u) x |= j << (4u * k);
                ++k;
            }
        nth[m] = x;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t base = (blockIdx.x * kEmitWarps + warp) * (32u * kRounds);
    const uint32_t end = min(n, base + 32u * kRounds);
    constexpr int kSteps = (kRounds + 1) / 2;  // of 64 splats, two consecutive ones a lane
    uint32_t i = base + 2 * lane, mine = 0;
#pragma unroll
    for (int r = 0; r < kSteps; ++r) {
        const uint2 b = load_two(bins, i + 64 * r, end);
        mine += bin_count(b.x) + bin_count(b.y);
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) wsum[warp] = mine;
    __syncthreads();
    if (mine == 0u) return;
    uint32_t o0 = sums[blockIdx.x];
    for (int w = 0; w < warp; ++w) o0 += wsum[w];
    // bin words are read two steps ahead, splat ids one
    uint2 b = load_two(bins, i, end), b1 = load_two(bins, i + 64u, end);
    uint2 s = bin_count(b.x) + bin_count(b.y) ? load_two(order, i, end) : make_uint2(0u, 0u);
#pragma unroll 1
    for (int r = 0; r < kSteps; ++r, i += 64) {
        const uint2 b2 = load_two(bins, i + 128u, end);
        const uint2 s1 = bin_count(b1.x) + bin_count(b1.y) ? load_two(order, i + 64u, end) : make_uint2(0u, 0u);
        const uint32_t c0 = bin_count(b.x), c1 = bin_count(b.y);
        const uint32_t incl = warp_inclusive_scan(c0 + c1), first0 = incl - c0 - c1, first1 = incl - c1;
        const uint32_t pairs = __shfl_sync(0xffffffffu, incl, 31);
        const unsigned have0 = __ballot_sync(0xffffffffu, c0 != 0u), have1 = __ballot_sync(0xffffffffu, c1 != 0u);
        const uint32_t at = __popc(have0 & lt) + __popc(have1 & lt);
        if (c0) stage[warp][at] = staged_splat(b.x, s.x, first0, rec, n);
        if (c1) stage[warp][at + (c0 != 0u)] = staged_splat(b.y, s.y, first1, rec, n);
        __syncwarp();
        uint32_t started = 0;
        for (uint32_t w0 = 0; w0 < pairs; w0 += 32u) {
            const unsigned starts = __reduce_or_sync(0xffffffffu, (c0 && first0 - w0 < 32u ? 1u << (first0 - w0) : 0u) |
                                                                      (c1 && first1 - w0 < 32u ? 1u << (first1 - w0) : 0u));
            const uint32_t p = w0 + lane;
            const uint32_t owner = started + __popc(starts & (lt | (1u << lane))) - 1u;
            started += __popc(starts);
            if (p >= pairs) continue;
            const uint4 e = stage[warp][owner];
            const uint32_t k = p - e.y;  // rank among the splat's tiles
            uint32_t row, col;
            if (e.w & kBinLarge) {
                // k / width: exact for k < 2^16 (the quotient is at least half
                // a width's inverse away from an integer, the reciprocal's
                // error a few ulp)
                const uint32_t width = e.w & ~kBinLarge;
                row = (uint32_t)(((float)k + 0.5f) * __fdividef(1.0f, (float)width));
                col = k - row * width;
            } else {
                const uint32_t at = k < 8u ? (nth[e.w] >> (4u * k)) & 15u : 8u;
                row = at / 3u;
                col = at - 3u * row;
            }
            const uint32_t tile = ((e.z >> 16) + row) * (uint32_t)tiles_x + (e.z & 0xFFFFu) + col;
            const uint32_t o = o0 + p;
            if (in_bounds(o < n_pairs, kChkPair) && in_bounds(e.x < n, kChkSplat) && in_bounds(tile < n_tiles, kChkTile)) {
                ptile[o] = (uint16_t)tile;
                pval[o] = e.x;
            }
        }
        __syncwarp();  // the staged splats are replaced by the next round's
        o0 += pairs;
        b = b1;
        b1 = b2;
        s = s1;
    }
}

// rounds of a block of the two kernels above
static int emit_rounds(size_t n) {
    return n <= kEmitOneSplats ? kEmitOneRound : n <= kEmitFewSplats ? kEmitFewRounds : kEmitRounds;
}

size_t bin_scan_blocks(size_t n) {
    const size_t tile = (size_t)kEmitThreads * emit_rounds(n);
    return (n + tile - 1) / tile;
}

int bin_scan_sums(const uint32_t *bins, uint32_t n, uint32_t *sums, uint32_t *ticket, uint32_t *host, uint32_t seq,
                  cudaStream_t st) {
    if (n == 0) return 0;
    const uint32_t nb = (uint32_t)bin_scan_blocks(n);
    switch (emit_rounds(n)) {
        case kEmitOneRound: k_bin_sums<kEmitOneRound><<<nb, kEmitThreads, 0, st>>>(bins, n, sums, ticket, host, seq); return 1;
        case kEmitFewRounds: k_bin_sums<kEmitFewRounds><<<nb, kEmitThreads, 0, st>>>(bins, n, sums, nullptr, nullptr, 0u); break;
        default: k_bin_sums<kEmitRounds><<<nb, kEmitThreads, 0, st>>>(bins, n, sums, nullptr, nullptr, 0u); break;
    }
    k_scan_spine<<<1, kScanThreads, 0, st>>>(sums, nb, host, seq);
    return 2;
}

int launch_emit_pairs_scan(uint32_t n_splats, const uint32_t *order, const uint32_t *bins_sorted,
                           const uint32_t *sums, const float4 *rec, int tiles_x, uint32_t n_tiles, uint16_t *ptile,
                           uint32_t *pval, uint2 *ranges, int32_t *blend_meta, cudaStream_t st) {
    if (n_splats == 0) return 0;
    const uint32_t nb = (uint32_t)bin_scan_blocks(n_splats);
    switch (emit_rounds(n_splats)) {
        case kEmitOneRound:
            k_emit_pairs_scan<kEmitOneRound><<<nb, kEmitThreads, 0, st>>>(n_splats, order, bins_sorted, sums, rec, tiles_x,
                                                                         n_tiles, ptile, pval, ranges, blend_meta);
            break;
        case kEmitFewRounds:
            k_emit_pairs_scan<kEmitFewRounds><<<nb, kEmitThreads, 0, st>>>(n_splats, order, bins_sorted, sums, rec, tiles_x,
                                                                          n_tiles, ptile, pval, ranges, blend_meta);
            break;
        default:
            k_emit_pairs_scan<kEmitRounds><<<nb, kEmitThreads, 0, st>>>(n_splats, order, bins_sorted, sums, rec, tiles_x,
                                                                       n_tiles, ptile, pval, ranges, blend_meta);
            break;
    }
    return 1;
}

int launch_emit_pairs(uint32_t n_splats, const uint32_t *order, const uint32_t *bins_sorted,
                      const uint32_t *pair_off, const float4 *rec, int tiles_x, uint32_t n_tiles, uint16_t *ptile,
                      uint32_t *pval, cudaStream_t st) {
    if (n_splats == 0) return 0;
    k_emit_pairs<<<(n_splats + 255) / 256, 256, 0, st>>>(n_splats, order, bins_sorted, pair_off, rec,
                                                          tiles_x, n_tiles, ptile, pval);
    return 1;
}

// Tile boundaries of the sorted pair list: each thread reads 8 tile keys
// with one 16-byte load (the list starts 16-byte aligned) plus its two
// neighbours, and writes the start / end of every tile that begins / ends
// among its keys.
__global__ void __launch_bounds__(256) k_tile_ranges(uint32_t n, const uint16_t *__restrict__ ptile,
                                                     uint2 *__restrict__ ranges, uint32_t n_tiles) {
    const uint32_t base = (blockIdx.x * blockDim.x + threadIdx.x) * 8u;
    if (base >= n) return;
    uint32_t v[8];
    if (base + 8u <= n) {
        const uint4 w = __ldg(reinterpret_cast<const uint4 *>(ptile + base));
        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[2 * k] = ww[k] & 0xFFFFu;
            v[2 * k + 1] = ww[k] >> 16;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = base + k < n ? (uint32_t)__ldg(ptile + base + k) : 0x10000u;
    }
    uint32_t prev = base > 0 ? (uint32_t)__ldg(ptile + base - 1) : 0x10000u;
    const uint32_t next = base + 8u < n ? (uint32_t)__ldg(ptile + base + 8) : 0x10000u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t t = v[k];
        if (t > 0xFFFFu) break;  // past the end
        const uint32_t after = k < 7 ? v[k + 1] : next;
        if (in_bounds(t < n_tiles, kChkTile)) {
            if (t != prev) ranges[t].x = base + k;
            if (t != after) ranges[t].y = base + k + 1;
        }
        prev = t;
    }
}

int launch_tile_ranges(uint32_t n_pairs, const uint16_t *ptile, uint2 *ranges, uint32_t n_tiles, cudaStream_t st) {
    if (n_pairs == 0) return 0;
    const uint32_t threads = (n_pairs + 7) / 8;
    k_tile_ranges<<<(threads + 255) / 256, 256, 0, st>>>(n_pairs, ptile, ranges, n_tiles);
    return 1;
}

__global__ void __launch_bounds__(256) k_count_live(uint32_t n, const uint32_t *__restrict__ keys,
                                                    int32_t *__restrict__ out) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const bool live = keys[i] != 0xFFFFFFFFu;
    const bool next_live = i + 1 < n && keys[i + 1] != 0xFFFFFFFFu;
    if (i == 0 && !live) *out = 0;
    if (live && !next_live) *out = (int32_t)(i + 1);
}

int launch_count_live(uint32_t n, const uint32_t *sorted_keys, int32_t *out, cudaStream_t st) {
    cudaMemsetAsync(out, 0, sizeof(int32_t), st);
    if (n == 0) return 0;
    k_count_live<<<(n + 255) / 256, 256, 0, st>>>(n, sorted_keys, out);
    return 1;
}

CS_DEFINE_CHECK_READER(check_word_sort)

}  // namespace cs
