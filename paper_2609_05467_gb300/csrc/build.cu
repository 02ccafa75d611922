// build.cu -- device construction of the part's acceleration structure and
// the per-face data of Section 3.1 (normal, area, centroid), plus sampling.
//
// Pipeline (one stream):
//   face_prep   : FP64 normal / area / centroid per face, fp32 face boxes,
//                 mesh validation, scene bounds (atomics)
//   morton      : 48-bit Morton code of each face-box centre (16 bits per axis)
//   radix sort  : 6 passes of 8-bit LSD (histogram / scan / stable scatter)
//   karras      : binary radix tree over the sorted codes (Karras, HPG 2012)
//   refit       : triangle records (48 B), boxes bottom-up and BVH2 nodes
//                 holding both child boxes (64 B, leaves of up to kLeafMax
//                 consecutive triangles) in one launch: within a block in
//                 shared memory, across blocks by arrival counters
//   wide        : top-down collapse into 4-wide nodes (128 B): six levels in
//                 one block, further ones a launch each, the subtrees below
//                 depth-first
//   area cdf    : 2^32-quantised face areas, inclusive int64 prefix
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "rc_internal.cuh"

namespace rc {

// device scratch of a build step, freed in stream order when the scope ends
// (on every path, error returns included)
struct BuildScratch {
    cudaStream_t s;
    void* p[3] = {nullptr, nullptr, nullptr};
    ~BuildScratch()
    {
        for (void* q : p)
            if (q) cudaFreeAsync(q, s);
    }
};


// ---------------------------------------------------------------------------
// face preparation and validation
// ---------------------------------------------------------------------------
// fl32(c / len) from the FP64 product q = c * inv, where inv is within 2^-44 of
// 1 / len (0: unknown): the same fp32 value unless q lies within 2^-43 of a
// midpoint of two fp32 values (2^-42 taken; 4 in 10^6), or outside the range
// of normal fp32 values.  No FP64 division where three were.
__device__ __forceinline__ float quotient32(double c, double len, double inv)
{
    if ((__double_as_longlong(c) << 1) == 0) return __int_as_float(__double2hiint(c) & 0x80000000);
    const double q = __dmul_rn(c, inv);
    const unsigned e = ((unsigned)__double2hiint(q) >> 20) & 0x7FFu;
    const int low = (__double2loint(q) & 0x1FFFFFFF) - 0x10000000;
    if (e < 1023u - 120u || e > 1023u + 120u || abs(low) <= 2048) return __double2float_rn(__ddiv_rn(c, len));
    return narrow(q);
}

// Bound by FP64, which issues at 1/64 of the fp32 rate (85% of its cycles):
// no face divides in FP64, conversions, comparisons and the halving go by
// integers, and the largest area is reduced as an integer.  Blocks stay for
// many faces and reduce in shared memory before their atomics.  1.93M faces:
// 345 -> 179 us.
constexpr int kPrepThreads = 256;

__global__ void __launch_bounds__(kPrepThreads)
k_face_prep(const float* __restrict__ V, int64_t nV, const int32_t* __restrict__ F,
            int64_t T, float* fnorm, double* farea, float* tbox, DevScalars* sc)
{
    // contributions to the scene bounds; neutral when absent
    float cmin[3] = {INFINITY, INFINITY, INFINITY}, cmax[3] = {-INFINITY, -INFINITY, -INFINITY};
    float mabs = 0.0f;
    unsigned long long amax = 0;       // bits of the area (>= 0, so they order as integers)
    for (int64_t f = blockIdx.x * (int64_t)kPrepThreads + threadIdx.x; f < T; f += (int64_t)gridDim.x * kPrepThreads) {
        int32_t id[3];
        bool bad = false;
        for (int k = 0; k < 3; ++k) {
            id[k] = F[3 * f + k];
            if (id[k] < 0 || id[k] >= nV) bad = true;
        }
        if (bad) {
            atomicMin(&sc->err_index, (int)f);
            for (int k = 0; k < 6; ++k) tbox[6 * f + k] = 0.0f;
        } else {
            float v[3][3];
            for (int a = 0; a < 3; ++a) {
                for (int k = 0; k < 3; ++k) {
                    v[a][k] = V[3 * (int64_t)id[a] + k];
                    if (!isfinite(v[a][k])) {
                        atomicMin(&sc->err_vertex, id[a]);
                        v[a][k] = 0.0f;
                    }
                    mabs = fmaxf(mabs, fabsf(v[a][k]));
                }
            }
            // c = (B - A) x (C - A) in FP64, each operation rounded separately
            double e1[3], e2[3];
            for (int k = 0; k < 3; ++k) {
                const double o = widen(v[0][k]);
                e1[k] = __dsub_rn(widen(v[1][k]), o);
                e2[k] = __dsub_rn(widen(v[2][k]), o);
            }
            const double c0 = __dsub_rn(__dmul_rn(e1[1], e2[2]), __dmul_rn(e1[2], e2[1]));
            const double c1 = __dsub_rn(__dmul_rn(e1[2], e2[0]), __dmul_rn(e1[0], e2[2]));
            const double c2 = __dsub_rn(__dmul_rn(e1[0], e2[1]), __dmul_rn(e1[1], e2[0]));
            const double len =
                __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(c0, c0), __dmul_rn(c1, c1)), __dmul_rn(c2, c2)));
            // len is zero or far inside the normal range (products of
            // differences of fp32 values): halving lowers its exponent
            const long long lb = __double_as_longlong(len);
            const long long ab = lb > 0 ? lb - (1LL << 52) : 0;
            farea[f] = __longlong_as_double(ab);
            amax = max(amax, (unsigned long long)ab);
            float n0 = 0.0f, n1 = 0.0f, n2 = 0.0f;
            if (lb > 0) {
                // one Newton step from the fp32 reciprocal of len cut to fp32
                // (0: outside fp32's range)
                double inv = 0.0;
                const unsigned e = (unsigned)(lb >> 52);
                if (e > 1023u - 100u && e < 1023u + 100u) {
                    const double y = widen(__frcp_rn(__uint_as_float(((unsigned)(lb >> 32) - 0x38000000u) << 3 | (unsigned)lb >> 29)));
                    inv = __fma_rn(y, __fma_rn(-len, y, 1.0), y);
                }
                n0 = quotient32(c0, len, inv);
                n1 = quotient32(c1, len, inv);
                n2 = quotient32(c2, len, inv);
            }
            fnorm[3 * f + 0] = n0;
            fnorm[3 * f + 1] = n1;
            fnorm[3 * f + 2] = n2;
            for (int k = 0; k < 3; ++k) {
                const float lo = fminf(v[0][k], fminf(v[1][k], v[2][k]));
                const float hi = fmaxf(v[0][k], fmaxf(v[1][k], v[2][k]));
                tbox[6 * f + k] = lo;
                tbox[6 * f + 3 + k] = hi;
                const float c = 0.5f * (lo + hi);
                cmin[k] = fminf(cmin[k], c);
                cmax[k] = fmaxf(cmax[k], c);
            }
        }
    }
    constexpr int W = kPrepThreads / 32;
    __shared__ float s_f[7][W];
    __shared__ unsigned long long s_a[W];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k = 0; k < 3; ++k) {
        cmin[k] = warp_min(cmin[k]);
        cmax[k] = warp_max(cmax[k]);
    }
    mabs = warp_max(mabs);
    const unsigned hi = __reduce_max_sync(0xFFFFFFFFu, (unsigned)(amax >> 32));
    const unsigned lo = __reduce_max_sync(0xFFFFFFFFu, (unsigned)(amax >> 32) == hi ? (unsigned)amax : 0u);
    if (lane == 0) {
        for (int k = 0; k < 3; ++k) {
            s_f[k][warp] = cmin[k];
            s_f[3 + k][warp] = cmax[k];
        }
        s_f[6][warp] = mabs;
        s_a[warp] = ((unsigned long long)hi << 32) | lo;
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        const int k = threadIdx.x;
        if (k < 7) {
            float v = s_f[k][0];
            for (int w = 1; w < W; ++w) v = k < 3 ? fminf(v, s_f[k][w]) : fmaxf(v, s_f[k][w]);
            if (k < 3 && v < INFINITY) atomicMin(&sc->cmin[k], float_to_ordered(v));
            else if (k >= 3 && k < 6 && v > -INFINITY) atomicMax(&sc->cmax[k - 3], float_to_ordered(v));
            else if (k == 6) atomicMax(&sc->vmaxabs, float_to_ordered(v));
        } else {
            unsigned long long v = s_a[0];
            for (int w = 1; w < W; ++w) v = max(v, s_a[w]);
            atomicMax(&sc->amax_bits, v);
        }
    }
}

// ---------------------------------------------------------------------------
// Morton codes
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long spread21(unsigned long long x)
{
    x &= 0x1FFFFFULL;
    x = (x | (x << 32)) & 0x1F00000000FFFFULL;
    x = (x | (x << 16)) & 0x1F0000FF0000FFULL;
    x = (x | (x << 8)) & 0x100F00F00F00F00FULL;
    x = (x | (x << 4)) & 0x10C30C30C30C30C3ULL;
    x = (x | (x << 2)) & 0x1249249249249249ULL;
    return x;
}

// Morton code of each face-box centre, kMortonBits per axis (interleaved
// x, y, z from the top); the radix sort then needs kMortonPasses byte passes
#ifndef RC_MORTON_BITS
#define RC_MORTON_BITS 16
#endif
constexpr int kMortonBits = RC_MORTON_BITS;
constexpr int kMortonPasses = (3 * kMortonBits + 7) / 8;
static_assert(kMortonBits >= 8 && kMortonBits <= 21, "Morton bits per axis out of range");
static_assert(kMortonPasses % 2 == 0, "an even number of sort passes leaves the result in place");

__global__ void k_morton(const float* __restrict__ tbox, int64_t T, const DevScalars* sc,
                         unsigned long long* keys, int32_t* vals)
{
    int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (f >= T) return;
    unsigned long long code = 0;
    for (int k = 0; k < 3; ++k) {
        float lo = ordered_to_float(sc->cmin[k]);
        float hi = ordered_to_float(sc->cmax[k]);
        float c = 0.5f * (tbox[6 * f + k] + tbox[6 * f + 3 + k]);
        float ext = hi - lo;
        float u = ext > 0.0f ? (c - lo) / ext : 0.0f;
        u = fminf(fmaxf(u, 0.0f), 1.0f);
        const float cells = (float)(1 << kMortonBits);
        unsigned long long q = (unsigned long long)fminf(u * cells, cells - 1.0f);
        code |= spread21(q) << (2 - k);
    }
    keys[f] = code;
    vals[f] = (int32_t)f;
}

// ---------------------------------------------------------------------------
// LSD radix sort of (uint64 key, int32 value), 8-bit digits, stable
// ---------------------------------------------------------------------------
constexpr int kMaxWalk = 4096;   // bound on leaf-to-root walks
constexpr int kSortThreads = 256;

__global__ void k_sort_hist(const unsigned long long* __restrict__ keys, int64_t T, int shift, int tile,
                            int nblk, unsigned int* __restrict__ counts)
{
    __shared__ unsigned int h[256];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) h[i] = 0;
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * tile;
    int64_t end = min64(T, base + tile);
    for (int64_t i = base + threadIdx.x; i < end; i += blockDim.x)
        atomicAdd(&h[(keys[i] >> shift) & 255], 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += blockDim.x) counts[(int64_t)i * nblk + blockIdx.x] = h[i];
}

__device__ __forceinline__ unsigned int warp_incl_scan(unsigned int v, int lane)
{
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned int u = __shfl_up_sync(0xFFFFFFFFu, v, off);
        if (lane >= off) v += u;
    }
    return v;
}

// per digit, the exclusive prefix of its counts over the blocks (in place,
// digit-major layout counts[d * nblk + b]) and the digit's total; one warp
// per digit, a lane per run of consecutive counts, so that the loads do not
// wait for one another
constexpr int kScanRun = 32;       // counts per lane and round: one round for up to 1,024 blocks

__global__ void __launch_bounds__(256) k_sort_scan(unsigned int* __restrict__ counts, int nblk,
                                                   unsigned int* __restrict__ totals)
{
    const int lane = threadIdx.x & 31;
    const int d = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (d >= 256) return;
    unsigned int* c = counts + (int64_t)d * nblk;
    unsigned int carry = 0;
    for (int b0 = 0; b0 < nblk; b0 += 32 * kScanRun) {
        const int m = min(32 * kScanRun, nblk - b0), run = (m + 31) / 32;
        const int i0 = b0 + lane * run, i1 = min(i0 + run, b0 + m);
        unsigned int v[kScanRun], sum = 0;
#pragma unroll
        for (int k = 0; k < kScanRun; ++k) v[k] = k < run && i0 + k < i1 ? c[i0 + k] : 0u;
#pragma unroll
        for (int k = 0; k < kScanRun; ++k) sum += v[k];
        const unsigned int inc = warp_incl_scan(sum, lane);
        unsigned int at = carry + inc - sum;
#pragma unroll
        for (int k = 0; k < kScanRun; ++k) {
            if (k < run && i0 + k < i1) c[i0 + k] = at;
            at += v[k];
        }
        carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    if (lane == 0) totals[d] = carry;
}

// the lanes with the same digit (eight votes; the match instruction on 32
// mostly different digits takes several times as long)
__device__ __forceinline__ unsigned int same_digit(unsigned int dig, bool ok)
{
    unsigned int peers = __ballot_sync(0xFFFFFFFFu, ok);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool set = (dig >> b) & 1u;
        const unsigned int m = __ballot_sync(0xFFFFFFFFu, set);
        peers &= set ? m : ~m;
    }
    return peers;
}

// A block ranks its tile's keys once: warp w holds keys [w, w + 1) * 32 * kItems
// of the tile in registers, kItems rounds of 32; within a round equal digits
// find each other by votes, and the warp's digit counters carry from round to
// round.  The tile is then put in order in shared memory and written out from
// there, so that a warp writes a few runs instead of 32 places.  Six block
// barriers per tile, where one pass per 256 keys took 64.  1.93M keys: 37 ->
// 18 us per pass.
template <int kItems>
__global__ void __launch_bounds__(kSortThreads)
k_sort_scatter(const unsigned long long* __restrict__ kin, const int32_t* __restrict__ vin,
               int64_t T, int shift, int nblk, const unsigned int* __restrict__ offs,
               const unsigned int* __restrict__ totals, unsigned long long* __restrict__ kout,
               int32_t* __restrict__ vout, unsigned int* err)
{
    constexpr int W = kSortThreads / 32, kTile = kItems * kSortThreads;
    static_assert(kSortThreads == 256, "one thread per digit");
    __shared__ unsigned long long s_key[kTile];
    __shared__ int32_t s_val[kTile];
    __shared__ unsigned short wcnt[W][256];     // then the warps' first places in the ordered tile
    __shared__ int to[256];                     // global place of a digit's first key, less its place in the tile
    __shared__ unsigned int wsum[2][W];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < W * 128; i += kSortThreads) ((unsigned int*)&wcnt[0][0])[i] = 0;
    // the digit's start = the totals of the smaller digits (a block scan of
    // the 256 totals) + this digit's count in the blocks before this one
    const unsigned int t = totals[threadIdx.x], mine = offs[(int64_t)threadIdx.x * nblk + blockIdx.x];
    const unsigned int inc = warp_incl_scan(t, lane);
    if (lane == 31) wsum[0][warp] = inc;
    const int64_t tile0 = (int64_t)blockIdx.x * kTile, first = tile0 + warp * (32 * kItems) + lane;
    const int m = (int)min64(kTile, T - tile0);
    unsigned long long key[kItems];
    int32_t val[kItems];
    unsigned short rank[kItems];
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        const int64_t i = first + 32 * r;
        key[r] = i < T ? kin[i] : 0ULL;
        val[r] = i < T ? vin[i] : 0;
    }
    __syncthreads();
    unsigned int before = 0;
    for (int w = 0; w < warp; ++w) before += wsum[0][w];
    const unsigned int start = before + inc - t + mine;
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        const bool ok = first + 32 * r < T;
        const unsigned int dig = (unsigned int)((key[r] >> shift) & 255);
        const unsigned int peers = same_digit(dig, ok);
        const unsigned int at = __popc(peers & ((1u << lane) - 1u));
        const unsigned int had = ok ? wcnt[warp][dig] : 0u;
        __syncwarp();
        if (ok && at == 0) wcnt[warp][dig] = (unsigned short)(had + __popc(peers));
        __syncwarp();
        rank[r] = (unsigned short)(had + at);
    }
    __syncthreads();
    // this thread's digit: its keys in the tile, their first place there, and
    // the warps' places
    unsigned int total = 0;
    for (int w = 0; w < W; ++w) total += wcnt[w][threadIdx.x];
    const unsigned int inc2 = warp_incl_scan(total, lane);
    if (lane == 31) wsum[1][warp] = inc2;
    __syncthreads();
    unsigned int run = inc2 - total;
    for (int w = 0; w < warp; ++w) run += wsum[1][w];
    to[threadIdx.x] = (int)(start - run);
    for (int w = 0; w < W; ++w) {
        const unsigned int c = wcnt[w][threadIdx.x];
        wcnt[w][threadIdx.x] = (unsigned short)run;
        run += c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        if (first + 32 * r >= T) continue;
        const unsigned int at = wcnt[warp][(key[r] >> shift) & 255] + rank[r];
        s_key[at & (kTile - 1)] = key[r];
        s_val[at & (kTile - 1)] = val[r];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += kSortThreads) {
        const unsigned long long k = s_key[i];
        const int64_t pos = (int64_t)to[(k >> shift) & 255] + i;
        if (pos >= 0 && pos < T) {
            kout[pos] = k;
            vout[pos] = s_val[i];
        } else {
            atomicAdd(err, 1u);
        }
    }
}

// All passes of a small sort by one block, keys and values in shared memory:
// a part of a few thousand triangles or points is bound by launches (three
// per pass), not by work.  1,472 keys, six passes: 18 launches of 4 us -> one
// of 16 us.
constexpr int kSmallItems = 4, kSmallThreads = 1024;
constexpr int kSmallSort = kSmallItems * kSmallThreads;
struct SmallSort {
    unsigned long long key[kSmallSort];
    int32_t val[kSmallSort];
    unsigned short cnt[kSmallThreads / 32][256];
    unsigned int base[256], wsum[8];
};

__global__ void __launch_bounds__(kSmallThreads)
k_sort_small(unsigned long long* __restrict__ keys, int32_t* __restrict__ vals, int n, int passes, unsigned int* err)
{
    extern __shared__ __align__(16) unsigned char s_sort[];
    SmallSort& sm = *(SmallSort*)s_sort;
    constexpr int W = kSmallThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int first = warp * 32 * kSmallItems + lane;
    unsigned long long key[kSmallItems];
    int32_t val[kSmallItems];
#pragma unroll
    for (int r = 0; r < kSmallItems; ++r) {
        const int i = first + 32 * r;
        key[r] = i < n ? keys[i] : 0ULL;
        val[r] = i < n ? vals[i] : 0;
    }
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = 8 * pass;
        for (int i = threadIdx.x; i < W * 256; i += kSmallThreads) (&sm.cnt[0][0])[i] = 0;
        __syncthreads();
        unsigned int rank[kSmallItems];
#pragma unroll
        for (int r = 0; r < kSmallItems; ++r) {
            const bool ok = first + 32 * r < n;
            const unsigned int dig = (unsigned int)((key[r] >> shift) & 255);
            const unsigned int peers = same_digit(dig, ok);
            const unsigned int at = __popc(peers & ((1u << lane) - 1u));
            const unsigned int had = ok ? sm.cnt[warp][dig] : 0u;
            __syncwarp();
            if (ok && at == 0) sm.cnt[warp][dig] = (unsigned short)(had + __popc(peers));
            __syncwarp();
            rank[r] = had + at;
        }
        __syncthreads();
        // per digit the prefix over the warps, then over the digits
        unsigned int total = 0, inc = 0;
        if (threadIdx.x < 256) {
            for (int w = 0; w < W; ++w) {
                const unsigned int c = sm.cnt[w][threadIdx.x];
                sm.cnt[w][threadIdx.x] = (unsigned short)total;
                total += c;
            }
            inc = warp_incl_scan(total, lane);
            if (lane == 31) sm.wsum[warp] = inc;
        }
        __syncthreads();
        if (threadIdx.x < 256) {
            unsigned int before = 0;
            for (int w = 0; w < warp; ++w) before += sm.wsum[w];
            sm.base[threadIdx.x] = before + inc - total;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSmallItems; ++r) {
            if (first + 32 * r >= n) continue;
            const unsigned int dig = (unsigned int)((key[r] >> shift) & 255);
            const unsigned int pos = sm.base[dig] + sm.cnt[warp][dig] + rank[r];
            if (pos < (unsigned int)n) {
                sm.key[pos] = key[r];
                sm.val[pos] = val[r];
            } else {
                atomicAdd(err, 1u);
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kSmallItems; ++r) {
            const int i = first + 32 * r;
            if (i < n) {
                key[r] = sm.key[i];
                val[r] = sm.val[i];
            }
        }
    }
#pragma unroll
    for (int r = 0; r < kSmallItems; ++r) {
        const int i = first + 32 * r;
        if (i < n) {
            keys[i] = key[r];
            vals[i] = val[r];
        }
    }
}

// ---------------------------------------------------------------------------
// Karras binary radix tree
// ---------------------------------------------------------------------------
__device__ __forceinline__ int kdelta(const unsigned long long* keys, int64_t T, int64_t i, int64_t j)
{
    if (j < 0 || j >= T) return -1;
    unsigned long long a = keys[i], b = keys[j];
    if (a == b) return 64 + __clz((unsigned int)(i ^ j));
    return __clzll(a ^ b);
}

__global__ void k_karras(const unsigned long long* __restrict__ keys, int64_t T, int32_t* child,
                         int32_t* range, int32_t* parent)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t n_int = T - 1;
    if (i >= n_int) return;
    const int d = (kdelta(keys, T, i, i + 1) - kdelta(keys, T, i, i - 1)) >= 0 ? 1 : -1;
    const int dmin = kdelta(keys, T, i, i - d);
    int64_t lmax = 2;
    while (kdelta(keys, T, i, i + lmax * d) > dmin) lmax <<= 1;
    int64_t l = 0;
    for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
        if (kdelta(keys, T, i, i + (l + t) * d) > dmin) l += t;
    const int64_t j = i + l * d;
    const int dnode = kdelta(keys, T, i, j);
    int64_t s = 0, t = l;
    do {
        t = (t + 1) >> 1;
        if (kdelta(keys, T, i, i + (s + t) * d) > dnode) s += t;
    } while (t > 1);
    const int64_t gamma = i + s * d + (d < 0 ? -1 : 0);
    const int64_t lo = i < j ? i : j, hi = i < j ? j : i;
    const int32_t left = (int32_t)(lo == gamma ? n_int + gamma : gamma);
    const int32_t right = (int32_t)(hi == gamma + 1 ? n_int + gamma + 1 : gamma + 1);
    child[2 * i] = left;
    child[2 * i + 1] = right;
    range[2 * i] = (int32_t)lo;
    range[2 * i + 1] = (int32_t)hi;
    parent[left] = (int32_t)i;
    parent[right] = (int32_t)i;
    if (i == 0) parent[0] = -1;
}

// ---------------------------------------------------------------------------
// PLOC (Meister and Bittner, "Parallel Locally-Ordered Clustering for
// Bounding Volume Hierarchy Construction", IEEE TVCG 2018): clusters start as
// the Morton-ordered leaves; each round every cluster finds, within kPlocR
// positions, the cluster whose merged box has the smallest surface area;
// mutual nearest neighbours merge into a new interior node (at the lower
// position) and the array is compacted in order.  Raw interior ids come from
// an atomic counter; the tree is then renumbered in depth-first order (root
// 0, each subtree's leaves contiguous) so that packing, the 4-wide collapse
// and refit work on it as on the Karras tree.
// ---------------------------------------------------------------------------
constexpr int kPlocR = 16;
constexpr int kPlocThreads = 256;

__device__ __forceinline__ float merged_area(const float* a, const float* b)
{
    const float dx = fmaxf(a[3], b[3]) - fminf(a[0], b[0]);
    const float dy = fmaxf(a[4], b[4]) - fminf(a[1], b[1]);
    const float dz = fmaxf(a[5], b[5]) - fminf(a[2], b[2]);
    return dx * dy + dy * dz + dz * dx;
}

__global__ void k_ploc_init(const float* __restrict__ tbox, const int32_t* __restrict__ order, int64_t T,
                            int64_t n_int, int32_t* cl, float* cb, int* n_ptr)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k == 0) *n_ptr = (int)T;
    if (k >= T) return;
    cl[k] = (int32_t)(n_int + k);
    const int32_t f = order[k];
    for (int c = 0; c < 6; ++c) cb[6 * k + c] = tbox[6 * (int64_t)f + c];
}

__global__ void __launch_bounds__(kPlocThreads)
k_ploc_nn(const int* __restrict__ n_ptr, const float* __restrict__ cb, int32_t* __restrict__ nn)
{
    __shared__ float sb[kPlocThreads + 2 * kPlocR][6];
    const int n = *n_ptr;
    const int base = blockIdx.x * kPlocThreads;
    if (base >= n) return;
    for (int t = threadIdx.x; t < kPlocThreads + 2 * kPlocR; t += blockDim.x) {
        const int j = base - kPlocR + t;
        if (j >= 0 && j < n)
            for (int c = 0; c < 6; ++c) sb[t][c] = cb[6 * (int64_t)j + c];
    }
    __syncthreads();
    const int i = base + threadIdx.x;
    if (i >= n) return;
    const float* bi = sb[threadIdx.x + kPlocR];
    int best = -1;
    float ba = INFINITY;
    const int j0 = max(0, i - kPlocR), j1 = min(n - 1, i + kPlocR);
    for (int j = j0; j <= j1; ++j) {
        if (j == i) continue;
        const float a = merged_area(bi, sb[j - base + kPlocR]);
        if (a < ba) { ba = a; best = j; }          // ascending j: ties go to the lower position
    }
    nn[i] = best;
}

__global__ void k_ploc_merge(const int* __restrict__ n_ptr, const int32_t* __restrict__ nn,
                             const int32_t* __restrict__ cl, const float* __restrict__ cb, int32_t* cl_tmp,
                             float* cb_tmp, int* keep, int32_t* child_raw, int32_t* parent_raw, int* counter,
                             int64_t n_int)
{
    const int n = *n_ptr;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int j = nn[i];
    if (j >= 0 && nn[j] == i) {
        if (i > j) { keep[i] = 0; return; }        // merged into its partner
        const int id = atomicAdd(counter, 1);
        if (id >= n_int) { keep[i] = 0; return; }  // cannot happen for a valid cluster array
        const int32_t a = cl[i], b = cl[j];
        child_raw[2 * id] = a;
        child_raw[2 * id + 1] = b;
        parent_raw[a] = id;
        parent_raw[b] = id;
        for (int c = 0; c < 3; ++c) {
            cb_tmp[6 * (int64_t)i + c] = fminf(cb[6 * (int64_t)i + c], cb[6 * (int64_t)j + c]);
            cb_tmp[6 * (int64_t)i + 3 + c] = fmaxf(cb[6 * (int64_t)i + 3 + c], cb[6 * (int64_t)j + 3 + c]);
        }
        cl_tmp[i] = id;
    } else {
        cl_tmp[i] = cl[i];
        for (int c = 0; c < 6; ++c) cb_tmp[6 * (int64_t)i + c] = cb[6 * (int64_t)i + c];
    }
    keep[i] = 1;
}

// order-preserving compaction of the kept clusters: per-block counts, one
// block scanning them (it also writes the new count), then the scatter
constexpr int kCompact = 1024;

__global__ void k_ploc_count(const int* __restrict__ n_ptr, const int* __restrict__ keep, int* bsum)
{
    __shared__ int warp_tot[kCompact / 32];
    const int n = *n_ptr;
    const int i = blockIdx.x * kCompact + threadIdx.x;
    const int v = i < n ? keep[i] : 0;
    const int c = __popc(__ballot_sync(0xFFFFFFFFu, v));
    if ((threadIdx.x & 31) == 0) warp_tot[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kCompact / 32; ++w) t += warp_tot[w];
        bsum[blockIdx.x] = t;
    }
}

__global__ void k_ploc_scan(int* bsum, int nb, const int* __restrict__ n_ptr, int* n_next)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int n = *n_ptr;
    const int used = (n + kCompact - 1) / kCompact;
    int run = 0;
    for (int b = 0; b < nb && b < used; ++b) {
        const int v = bsum[b];
        bsum[b] = run;
        run += v;
    }
    *n_next = run;
}

__global__ void k_ploc_scatter(const int* __restrict__ n_ptr, const int* __restrict__ keep,
                               const int* __restrict__ bsum, const int32_t* __restrict__ cl_tmp,
                               const float* __restrict__ cb_tmp, int32_t* cl_out, float* cb_out)
{
    __shared__ int warp_pre[kCompact / 32];
    const int n = *n_ptr;
    const int i = blockIdx.x * kCompact + threadIdx.x;
    const int v = i < n ? keep[i] : 0;
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, v);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) warp_pre[w] = __popc(bal);
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        for (int k = 0; k < kCompact / 32; ++k) {
            const int c = warp_pre[k];
            warp_pre[k] = run;
            run += c;
        }
    }
    __syncthreads();
    if (!v) return;
    const int pos = bsum[blockIdx.x] + warp_pre[w] + __popc(bal & ((1u << lane) - 1u));
    cl_out[pos] = cl_tmp[i];
    for (int c = 0; c < 6; ++c) cb_out[6 * (int64_t)pos + c] = cb_tmp[6 * (int64_t)i + c];
}

// An arrival: what the thread wrote before is seen by the one that arrives
// second, and that one's reads come after.  (With a fence on either side of a
// plain exchange a refit of 1.93M triangles took 630 us, so 603.)
__device__ __forceinline__ int exchange_acq_rel(int32_t* p, int v)
{
    int old;
    asm volatile("atom.acq_rel.gpu.global.exch.b32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// subtree sizes (leaves, interior nodes) bottom-up with arrival counters;
// sizes of raw interior id p at sz_leaf[p], sz_int[p]
__global__ void k_ploc_sizes(int64_t T, int64_t n_int, const int32_t* __restrict__ parent_raw,
                             const int32_t* __restrict__ child_raw, int32_t* sz_leaf, int32_t* sz_int, int32_t* visits,
                             int* err)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= T) return;
    int32_t p = parent_raw[n_int + k];
    for (int steps = 0; p >= 0; ++steps) {
        if (steps > kMaxWalk) { atomicExch(err, 1); return; }
        if (exchange_acq_rel(&visits[p], 1) == 0) return;
        const int32_t a = child_raw[2 * p], b = child_raw[2 * p + 1];
        const int la = a >= n_int ? 1 : __ldcg(&sz_leaf[a]), lb = b >= n_int ? 1 : __ldcg(&sz_leaf[b]);
        const int ia = a >= n_int ? 0 : __ldcg(&sz_int[a]), ib = b >= n_int ? 0 : __ldcg(&sz_int[b]);
        __stcg(&sz_leaf[p], la + lb);
        __stcg(&sz_int[p], ia + ib + 1);
        p = parent_raw[p];
    }
}

// depth-first numbering: every node walks to the root adding, for each
// ancestor whose right subtree it is in, the sizes of the left sibling
// subtree.  Interior raw id p -> preorder index newid[p]; leaf k -> leaf
// position pos[k] (a subtree's leaves are contiguous in that order).
__global__ void k_ploc_number(int64_t T, int64_t n_int, const int32_t* __restrict__ parent_raw,
                              const int32_t* __restrict__ child_raw, const int32_t* __restrict__ sz_leaf,
                              const int32_t* __restrict__ sz_int, int32_t* newid, int32_t* leafstart,
                              int32_t* pos, int* err)
{
    const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x >= n_int + T) return;
    int pre = x < n_int ? 0 : 0, lstart = 0;
    int32_t cur = (int32_t)x;
    int steps = 0;
    for (int32_t p = parent_raw[cur]; p >= 0; cur = p, p = parent_raw[p]) {
        if (++steps > kMaxWalk) { atomicExch(err, 1); return; }
        const int32_t left = child_raw[2 * p];
        pre += 1;                                   // the parent comes first
        if (cur != left) {
            pre += left >= n_int ? 0 : sz_int[left];
            lstart += left >= n_int ? 1 : sz_leaf[left];
        }
    }
    if (x < n_int) {
        newid[x] = pre;
        leafstart[x] = lstart;
    } else {
        pos[x - n_int] = lstart;
    }
}

// the renumbered tree: child / parent in combined indexing (interior
// preorder ids, leaf n_int + position), ranges, and the leaf order
__global__ void k_ploc_emit(int64_t T, int64_t n_int, const int32_t* __restrict__ parent_raw,
                            const int32_t* __restrict__ child_raw, const int32_t* __restrict__ newid,
                            const int32_t* __restrict__ leafstart, const int32_t* __restrict__ sz_leaf,
                            const int32_t* __restrict__ pos, const int32_t* __restrict__ order_in, int32_t* child,
                            int32_t* range, int32_t* parent, int32_t* order_out)
{
    const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x >= n_int + T) return;
    auto map = [&](int32_t c) -> int32_t { return c >= n_int ? (int32_t)(n_int + pos[c - n_int]) : newid[c]; };
    const int32_t p = parent_raw[x];
    const int32_t me = map((int32_t)x);
    parent[me] = p >= 0 ? newid[p] : -1;
    if (x < n_int) {
        child[2 * me] = map(child_raw[2 * x]);
        child[2 * me + 1] = map(child_raw[2 * x + 1]);
        range[2 * me] = leafstart[x];
        range[2 * me + 1] = leafstart[x] + sz_leaf[x] - 1;
    } else {
        order_out[pos[x - n_int]] = order_in[x - n_int];
    }
}

// ---------------------------------------------------------------------------
// bottom-up refit and packing into the traversal layout
// ---------------------------------------------------------------------------
// The corners of sorted slot k's triangle; false for a face or vertex index
// out of range (a bad mesh, reported by the build, must not be gathered).
__device__ __forceinline__ bool gather_tri(const float* __restrict__ V, int64_t nV, const int32_t* __restrict__ F, int64_t T,
                                           int32_t f, float v[3][3])
{
    bool ok = f >= 0 && f < T;
    for (int a = 0; a < 3; ++a) {
        const int64_t vi = ok ? F[3 * (int64_t)f + a] : -1;
        const bool in = vi >= 0 && vi < nV;
        for (int c = 0; c < 3; ++c) v[a][c] = in ? V[3 * vi + c] : 0.0f;
        ok &= in;
    }
    return ok;
}

// From a leaf up: the second thread to arrive at a node has its box, the
// first one's box and both heights, and goes on.  A node whose leaves all
// belong to one block (255 of 256 do) meets in shared memory, at the place of
// its split (the last leaf of its left subtree, which no other node has).
// The others meet in global memory: an exchange that orders both sides and a
// read back, a microsecond or two per level; that chain bounds a small tree,
// and the boxes' traffic a large one.  kPack: the packed binary nodes are
// written on the way (both children's boxes are at hand), and `sc` receives the
// tree's depth and box at the root; otherwise every node's box goes to nbox.
// The arrival word of a node holds 1 + the first arrival's height, so depth
// needs no walk of its own.
constexpr int kClimb = 256;        // leaves (threads) per block
struct ClimbShared {
    float box[2][6][kClimb];       // of the left and the right child, by split
    int height[2][kClimb];
    int arrived[kClimb];
};

__device__ __forceinline__ void put_box(float* nbox, int64_t node, const float lo[3], const float hi[3])
{
    for (int c = 0; c < 3; ++c) {
        __stcg(&nbox[6 * node + c], lo[c]);
        __stcg(&nbox[6 * node + 3 + c], hi[c]);
    }
}

// the whole block calls it (threads past the last leaf with leaf = false)
template <bool kPack>
__device__ __forceinline__ void climb(ClimbShared& sm, bool leaf, int64_t T, int64_t n_int, const int32_t* __restrict__ parent,
                                      const int32_t* __restrict__ child, const int32_t* __restrict__ range, float* nbox,
                                      float4* nodes, int32_t* visits, DevScalars* sc, int64_t k, float lo[3], float hi[3])
{
    sm.arrived[threadIdx.x] = 0;
    __syncthreads();
    if (!leaf) return;
    const int64_t b0 = blockIdx.x * (int64_t)kClimb, b1 = min64(b0 + kClimb, T) - 1;
    int32_t cur = (int32_t)(n_int + k);
    int32_t first = (int32_t)k, last = (int32_t)k;      // leaves below cur
    int height = 0;
    if (!kPack) put_box(nbox, cur, lo, hi);
    // every chain ends at the root; the cap only guards against a malformed
    // tree (the depth recorded is then one that the build rejects)
    int32_t p = parent[cur];
    for (int steps = 0; p >= 0 && steps <= kMaxWalk; ++steps) {
        const int32_t a = child[2 * p], b = child[2 * p + 1], r0 = range[2 * p], r1 = range[2 * p + 1];
        const bool left = a == cur;
        const int32_t split = left ? last : first - 1;  // last leaf of the left child
        float slo[3], shi[3];
        if (r0 >= b0 && r1 <= b1 && split >= b0 && split < b1) {
            const int at = (int)(split - b0), me = left ? 0 : 1;
            for (int c = 0; c < 3; ++c) {
                sm.box[me][c][at] = lo[c];
                sm.box[me][3 + c][at] = hi[c];
            }
            sm.height[me][at] = height;
            __threadfence_block();
            if (atomicExch(&sm.arrived[at], 1) == 0) return;     // first arrival stops
            __threadfence_block();
            volatile float* bx = &sm.box[1 - me][0][at];
            for (int c = 0; c < 3; ++c) {
                slo[c] = bx[c * kClimb];
                shi[c] = bx[(3 + c) * kClimb];
            }
            height = max(height, *(volatile int*)&sm.height[1 - me][at]) + 1;
        } else {
            if (kPack) put_box(nbox, cur, lo, hi);      // (else it is there)
            // the box above is written before the arrival, the sibling's read after its own
            const int other = exchange_acq_rel(&visits[p], height + 1);
            if (other == 0) return;
            const int64_t sib = left ? b : a;
            for (int c = 0; c < 3; ++c) {
                slo[c] = __ldcg(&nbox[6 * sib + c]);
                shi[c] = __ldcg(&nbox[6 * sib + 3 + c]);
            }
            height = max(height, other - 1) + 1;
        }
        if (kPack) {
            // a child of at most kLeafMax triangles becomes a leaf
            const int nl = split - r0 + 1, nr = r1 - split;
            const int ca = nl <= kLeafMax ? leaf_code(r0, nl) : a, cb = nr <= kLeafMax ? leaf_code(split + 1, nr) : b;
            const float* Al = left ? lo : slo;
            const float* Ah = left ? hi : shi;
            const float* Bl = left ? slo : lo;
            const float* Bh = left ? shi : hi;
            float4* nd = nodes + 4 * (int64_t)p;
            nd[0] = make_float4(Al[0], Ah[0], Al[1], Ah[1]);
            nd[1] = make_float4(Bl[0], Bh[0], Bl[1], Bh[1]);
            nd[2] = make_float4(Al[2], Ah[2], Bl[2], Bh[2]);
            nd[3] = make_float4(__int_as_float(ca), __int_as_float(cb), 0.0f, 0.0f);
        }
        for (int c = 0; c < 3; ++c) {
            lo[c] = fminf(lo[c], slo[c]);
            hi[c] = fmaxf(hi[c], shi[c]);
        }
        if (!kPack) put_box(nbox, p, lo, hi);
        cur = p;
        first = r0;
        last = r1;
        p = parent[p];
    }
    if (kPack) {
        sc->max_depth = p < 0 ? height : kMaxWalk;
        for (int c = 0; c < 3; ++c) {
            sc->lo[c] = lo[c];
            sc->hi[c] = hi[c];
        }
    }
}

// Triangle records, leaf boxes, all boxes above them and the packed binary
// nodes in one launch: the corners are gathered once.  1.93M triangles: the
// four kernels this replaces took 331 us, this one 200 us.
__global__ void __launch_bounds__(kClimb)
k_refit(const float* __restrict__ V, int64_t nV, const int32_t* __restrict__ F, const int32_t* __restrict__ order, int64_t T,
        int64_t n_int, const int32_t* __restrict__ parent, const int32_t* __restrict__ child,
        const int32_t* __restrict__ range, float* nbox, float4* nodes, float4* tris, int32_t* visits, DevScalars* sc)
{
    __shared__ ClimbShared sm;
    const int64_t k = blockIdx.x * (int64_t)kClimb + threadIdx.x;
    float lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
    if (k < T) {
        const int32_t f = order[k];
        float v[3][3];
        gather_tri(V, nV, F, T, f, v);
        float le = 0.0f;
        for (int c = 0; c < 3; ++c) {
            le = fmaxf(le, fabsf(v[1][c] - v[0][c]));
            le = fmaxf(le, fabsf(v[2][c] - v[1][c]));
            le = fmaxf(le, fabsf(v[0][c] - v[2][c]));
        }
        tris[3 * k + 0] = make_float4(v[0][0], v[0][1], v[0][2], le);
        tris[3 * k + 1] = make_float4(v[1][0], v[1][1], v[1][2], __int_as_float(f));
        tris[3 * k + 2] = make_float4(v[2][0], v[2][1], v[2][2], 0.0f);
        for (int c = 0; c < 3; ++c) {
            lo[c] = fminf(v[0][c], fminf(v[1][c], v[2][c]));
            hi[c] = fmaxf(v[0][c], fmaxf(v[1][c], v[2][c]));
        }
    }
    if (parent) climb<true>(sm, k < T, T, n_int, parent, child, range, nbox, nodes, visits, sc, k, lo, hi);
}

// ---------------------------------------------------------------------------
// 4-wide tree: top-down collapse of the binary tree, one level per launch.
// A wide node starts from a binary interior node's two children and keeps
// replacing its interior child of largest box surface area by that child's
// two children until it has four children or only leaves.  Wide node layout
// (8 float4, 128 B): lo.x, hi.x, lo.y, hi.y, lo.z, hi.z of the four
// children, then the four child indices (>= 0 wide node, < 0 leaf as in the
// binary layout), then padding.  Empty slots have an empty box.
// ---------------------------------------------------------------------------
// the children of a wide node: boxes (lo, hi), codes (a binary interior node
// >= 0, or a leaf), and how many
struct WideKids {
    float lo[4][3], hi[4][3];
    int32_t code[4];
    int n;
};

// The children of the wide node made from binary interior node b: b's two
// children, the interior one of largest box surface area replaced by its own
// two until there are four or only leaves.  Reads one packed 64-byte node per
// replacement (boxes and codes together; child, range and box arrays took
// four dependent gathers each).
__device__ __forceinline__ WideKids wide_kids(int32_t b, const float4* __restrict__ nodes)
{
    WideKids w;
    w.n = 0;
    int at = 0;
    for (;;) {
        const float4* nd = nodes + 4 * (int64_t)b;
        const float4 n0 = nd[0], n1 = nd[1], n2 = nd[2], n3 = nd[3];
        const int other = w.n == 0 ? 1 : w.n;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k == at) {
                w.lo[k][0] = n0.x; w.hi[k][0] = n0.y; w.lo[k][1] = n0.z; w.hi[k][1] = n0.w;
                w.lo[k][2] = n2.x; w.hi[k][2] = n2.y;
                w.code[k] = __float_as_int(n3.x);
            }
            if (k == other) {
                w.lo[k][0] = n1.x; w.hi[k][0] = n1.y; w.lo[k][1] = n1.z; w.hi[k][1] = n1.w;
                w.lo[k][2] = n2.z; w.hi[k][2] = n2.w;
                w.code[k] = __float_as_int(n3.y);
            }
        }
        w.n = other + 1;
        if (w.n == 4) return w;
        at = -1;
        float most = -1.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k >= w.n || w.code[k] < 0) continue;
            const float dx = w.hi[k][0] - w.lo[k][0], dy = w.hi[k][1] - w.lo[k][1], dz = w.hi[k][2] - w.lo[k][2];
            const float a = dx * dy + dy * dz + dz * dx;
            if (a > most) {
                most = a;
                at = k;
                b = w.code[k];
            }
        }
        if (at < 0) return w;
    }
}

// write wide node w: its children's boxes and their indices idx (wide node
// >= 0, leaf < 0); empty slots get an empty box and index -1
__device__ __forceinline__ void wide_write(float4* wnodes, int32_t w, const WideKids& kids, const int32_t idx[4])
{
    float lo[3][4], hi[3][4];
    int32_t ix[4], id[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool on = k < kids.n;
        for (int a = 0; a < 3; ++a) {
            lo[a][k] = on ? kids.lo[k][a] : INFINITY;
            hi[a][k] = on ? kids.hi[k][a] : -INFINITY;
        }
        ix[k] = on ? idx[k] : -1;
        // the binary node the child was made from, for the boxes of the same
        // tree in another coordinate frame (-1: empty slot)
        id[k] = on ? (kids.code[k] >= 0 ? kids.code[k] : kLeafChild) : -1;
    }
    wnodes[wide_at(w, 0)] = make_float4(lo[0][0], lo[0][1], lo[0][2], lo[0][3]);
    wnodes[wide_at(w, 1)] = make_float4(hi[0][0], hi[0][1], hi[0][2], hi[0][3]);
    wnodes[wide_at(w, 2)] = make_float4(lo[1][0], lo[1][1], lo[1][2], lo[1][3]);
    wnodes[wide_at(w, 3)] = make_float4(hi[1][0], hi[1][1], hi[1][2], hi[1][3]);
    wnodes[wide_at(w, 4)] = make_float4(lo[2][0], lo[2][1], lo[2][2], lo[2][3]);
    wnodes[wide_at(w, 5)] = make_float4(hi[2][0], hi[2][1], hi[2][2], hi[2][3]);
    wnodes[wide_at(w, 6)] = make_float4(__int_as_float(ix[0]), __int_as_float(ix[1]), __int_as_float(ix[2]), __int_as_float(ix[3]));
    wnodes[wide_at(w, 7)] = make_float4(__int_as_float(id[0]), __int_as_float(id[1]), __int_as_float(id[2]), __int_as_float(id[3]));
}

// The first of n (0..4) consecutive numbers from a counter, for every active
// lane: one atomic per warp (a lane each, on one address, took most of the
// collapse's time).
__device__ __forceinline__ int take_numbers(int* counter, int n)
{
    const unsigned active = __activemask(), lane = threadIdx.x & 31, below = active & ((1u << lane) - 1u);
    const unsigned b0 = __ballot_sync(active, n & 1), b1 = __ballot_sync(active, n & 2), b2 = __ballot_sync(active, n & 4);
    const int before = __popc(b0 & below) + 2 * __popc(b1 & below) + 4 * __popc(b2 & below);
    const int total = __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2);
    const int leader = __ffs(active) - 1;
    int first = 0;
    if ((int)lane == leader && total) first = atomicAdd(counter, total);
    return __shfl_sync(active, first, leader) + before;
}

// A queue of (binary node, wide node) pairs: one node and its place.
// Expands one queued binary node into its wide node; interior children get
// consecutive wide numbers and go to the next queue.
__device__ __forceinline__ void wide_expand(const float4* __restrict__ nodes, int2 q, int2* qout, int* qout_count,
                                            int* wide_count, float4* wnodes)
{
    const WideKids kids = wide_kids(q.x, nodes);
    int ni = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) ni += k < kids.n && kids.code[k] >= 0;
    int nw = take_numbers(wide_count, ni), at = take_numbers(qout_count, ni);
    int32_t idx[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        idx[k] = -1;
        if (k >= kids.n) continue;
        idx[k] = kids.code[k];
        if (kids.code[k] >= 0) {
            qout[at++] = make_int2(kids.code[k], nw);
            idx[k] = nw++;
        }
    }
    wide_write(wnodes, q.y, kids, idx);
}

// The top levels of the tree in one block: level by level until a queue may
// outgrow it (level l holds at most 4^l nodes), a launch each otherwise: at
// 10 us and more a level, the top six had cost as much as the rest.
constexpr int kWideTop = 6, kWideTopThreads = 1024;   // 4^5 nodes on the sixth level

__global__ void __launch_bounds__(kWideTopThreads)
k_wide_top(const float4* __restrict__ nodes, int2* qa, int2* qb, int* counts /*[2]: sizes of qa and qb*/, int* wide_count,
           float4* wnodes, DevScalars* sc, int levels)
{
    __shared__ int s_count[2];
    if (threadIdx.x == 0) {
        qa[0] = make_int2(0, 0);
        s_count[0] = 1;
        s_count[1] = 0;
        *wide_count = 1;
    }
    __syncthreads();
    int depth = 0;
    for (int l = 0; l < levels; ++l) {
        const int n = s_count[l & 1];
        int2* in = l & 1 ? qb : qa;
        int2* out = l & 1 ? qa : qb;
        if (n > 0) depth = l + 1;
        for (int t = threadIdx.x; t < n; t += kWideTopThreads)
            wide_expand(nodes, in[t], out, &s_count[1 - (l & 1)], wide_count, wnodes);
        __syncthreads();
        if (threadIdx.x == 0) s_count[l & 1] = 0;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        counts[0] = s_count[0];
        counts[1] = s_count[1];
        sc->wide_depth = depth;
    }
}

// one further level, a launch each
__global__ void __launch_bounds__(256)
k_wide_level(const float4* __restrict__ nodes, const int2* __restrict__ qin, int* qin_count, int2* qout, int* qout_count,
             int* wide_count, float4* wnodes, DevScalars* sc, int level)
{
    const int n = *qin_count;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    if (t == 0) atomicMax(&sc->wide_depth, level + 1);
    wide_expand(nodes, qin[t], qout, qout_count, wide_count, wnodes);
}

// the rest of the tree: each thread finishes the subtree below one queued
// binary node depth-first, so a subtree's wide nodes are made by one thread
// (numbered with the siblings of a node consecutive).  A subtree deeper than
// the stack reports a wide depth that the host rejects.
constexpr int kWideDfs = 96;
#ifndef RC_WIDE_SUBTREE
#define RC_WIDE_SUBTREE 4.0      // binary nodes per subtree thread (0: one launch per level throughout)
#endif

__global__ void k_wide_subtrees(const float4* __restrict__ nodes, const int2* __restrict__ qin,
                                const int* __restrict__ qin_count, int* wide_count, float4* wnodes, DevScalars* sc, int level)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= *qin_count) return;
    int2 st[kWideDfs];
    uint8_t sd[kWideDfs];
    st[0] = qin[t];
    sd[0] = 0;
    int sp = 1, maxd = 0;
    while (sp > 0) {
        --sp;
        const int32_t w = st[sp].y;
        const int d = sd[sp];
        const WideKids kids = wide_kids(st[sp].x, nodes);
        int ni = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) ni += k < kids.n && kids.code[k] >= 0;
        if (sp + ni > kWideDfs || d + 1 > 250) {
            atomicMax(&sc->wide_depth, kStack4);
            return;
        }
        const int base = take_numbers(wide_count, ni);
        int32_t idx[4];
        int nw = base;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            idx[k] = -1;
            if (k < kids.n) idx[k] = kids.code[k] >= 0 ? nw++ : kids.code[k];
        }
        wide_write(wnodes, w, kids, idx);
        maxd = max(maxd, d + 1);
#pragma unroll
        for (int k = 3; k >= 0; --k) {           // the first child is taken next
            if (k >= kids.n || kids.code[k] < 0) continue;
            st[sp] = make_int2(kids.code[k], idx[k]);
            sd[sp] = (uint8_t)(d + 1);
            ++sp;
        }
    }
    atomicMax(&sc->wide_depth, level + maxd);
}

// wide root for parts with at most kLeafMax triangles: one leaf child
__global__ void k_wide_small(int64_t T, const float* __restrict__ tbox, float4* wnodes, DevScalars* sc)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t f = 0; f < T; ++f)
        for (int c = 0; c < 3; ++c) {
            lo[c] = fminf(lo[c], tbox[6 * f + c]);
            hi[c] = fmaxf(hi[c], tbox[6 * f + 3 + c]);
        }
    const float I = INFINITY;
    wnodes[0] = make_float4(lo[0], I, I, I);
    wnodes[1] = make_float4(hi[0], -I, -I, -I);
    wnodes[2] = make_float4(lo[1], I, I, I);
    wnodes[3] = make_float4(hi[1], -I, -I, -I);
    wnodes[4] = make_float4(lo[2], I, I, I);
    wnodes[5] = make_float4(hi[2], -I, -I, -I);
    wnodes[6] = make_float4(__int_as_float(leaf_code(0, (int)T)), __int_as_float(-1), __int_as_float(-1),
                            __int_as_float(-1));
    wnodes[7] = make_float4(__int_as_float(kAllTris), __int_as_float(-1), __int_as_float(-1), __int_as_float(-1));
    sc->wide_depth = 1;
    sc->wide_nodes = 1;
}

// single-leaf root for parts with at most kLeafMax triangles
__global__ void k_pack_small(int64_t T, const float* __restrict__ tbox, float4* nodes, DevScalars* sc)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t f = 0; f < T; ++f)
        for (int c = 0; c < 3; ++c) {
            lo[c] = fminf(lo[c], tbox[6 * f + c]);
            hi[c] = fmaxf(hi[c], tbox[6 * f + 3 + c]);
        }
    for (int c = 0; c < 3; ++c) {
        sc->lo[c] = lo[c];
        sc->hi[c] = hi[c];
    }
    nodes[0] = make_float4(lo[0], hi[0], lo[1], hi[1]);
    nodes[1] = make_float4(INFINITY, -INFINITY, INFINITY, -INFINITY);
    nodes[2] = make_float4(lo[2], hi[2], INFINITY, -INFINITY);
    nodes[3] = make_float4(__int_as_float(leaf_code(0, (int)T)), __int_as_float(-1), 0.0f, 0.0f);
}

// ---------------------------------------------------------------------------
// area CDF (2^32-quantised areas, inclusive prefix in int64)
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 1024, kScanItems = 4;
constexpr int kScanBlock = kScanThreads * kScanItems;

// llround(area / amax * 2^32) from the product with scale = 2^32 / amax, within
// 2^-18 of the quotient's value; taken as it is unless that close to a
// half-integer (2^-17 taken: 1 in 65,536), where the division decides.
__device__ __forceinline__ long long quantise_area(double area, double amax, double scale)
{
    const double C = 6755399441055744.0;           // 1.5 * 2^52: adding it leaves the integer in the low bits
    const double q = __dmul_rn(area, scale), t = __dadd_rn(q, C);
    const double off = __dsub_rn(q, __dsub_rn(t, C));          // |off| < 0.5 - 2^-17, compared by its high word
    if ((__double2hiint(off) & 0x7FFFFFFF) >= 0x3FDFFFE0) return llround(__dmul_rn(__ddiv_rn(area, amax), 4294967296.0));
    return __double_as_longlong(t) - __double_as_longlong(C);
}

// block-wise inclusive scan, writing per-block totals; with farea the scanned
// values are the quantised areas, formed here (FP64 divisions in a kernel of
// their own had taken 45 us for 1.93M faces, the scan of 1,024-value blocks
// with a barrier per doubling 25; together now 51)
__global__ void __launch_bounds__(kScanThreads)
k_scan_block(long long* x, int64_t n, const double* __restrict__ farea, const DevScalars* sc, long long* bsum, long long* total)
{
    __shared__ long long wsum[32];
    __shared__ double s_scale;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double amax = farea ? __longlong_as_double((long long)sc->amax_bits) : 0.0;
    if (farea) {
        if (threadIdx.x == 0) s_scale = amax > 0.0 ? __ddiv_rn(4294967296.0, amax) : 0.0;
        __syncthreads();
    }
    const int64_t i0 = blockIdx.x * (int64_t)kScanBlock + (int64_t)threadIdx.x * kScanItems;
    long long v[kScanItems], sum = 0;
    static_assert(kScanItems == 4, "two 16-byte loads");
    if (i0 + 4 <= n) {
        const longlong2* src = (const longlong2*)(farea ? (const long long*)farea : x) + i0 / 2;
        const longlong2 a = src[0], b = src[1];
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    } else {
        for (int k = 0; k < 4; ++k) v[k] = i0 + k < n ? (farea ? __double_as_longlong(farea[i0 + k]) : x[i0 + k]) : 0;
    }
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (farea) v[k] = amax > 0.0 && i0 + k < n ? quantise_area(__longlong_as_double(v[k]), amax, s_scale) : 0LL;
        sum += v[k];
    }
    long long inc = sum;
    for (int off = 1; off < 32; off <<= 1) {
        const long long u = __shfl_up_sync(0xFFFFFFFFu, inc, off);
        if (lane >= off) inc += u;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        long long t = wsum[lane];
        for (int off = 1; off < 32; off <<= 1) {
            const long long u = __shfl_up_sync(0xFFFFFFFFu, t, off);
            if (lane >= off) t += u;
        }
        wsum[lane] = t;
    }
    __syncthreads();
    long long run = inc - sum + (warp ? wsum[warp - 1] : 0);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        run += v[k];
        if (i0 + k < n) x[i0 + k] = run;
    }
    if (threadIdx.x == kScanThreads - 1) {
        bsum[blockIdx.x] = run;
        if (gridDim.x == 1) *total = run;          // the last level: one block holds the sum of everything
    }
}

__global__ void __launch_bounds__(kScanThreads)
k_scan_add(long long* x, int64_t n, const long long* bsum_incl)
{
    if (blockIdx.x == 0) return;
    const long long add = bsum_incl[blockIdx.x - 1];
    const int64_t i0 = blockIdx.x * (int64_t)kScanBlock;
    for (int k = threadIdx.x; k < kScanBlock; k += kScanThreads)
        if (i0 + k < n) x[i0 + k] += add;
}

// inclusive scan of x, or of the quantised areas into x; *total (device) = the sum
static rc_status scan_inclusive(long long* x, int64_t n, const double* farea, const DevScalars* sc, long long* total, cudaStream_t s)
{
    if (n <= 0) return RC_OK;
    const int64_t nb = (n + kScanBlock - 1) / kScanBlock;
    long long* bs = nullptr;
    BuildScratch g{s};
    RC_CUDA(cudaMallocAsync(&bs, sizeof(long long) * nb, s));
    g.p[0] = bs;
    k_scan_block<<<(unsigned)nb, kScanThreads, 0, s>>>(x, n, farea, sc, bs, total);
    RC_LAUNCHED();
    if (nb > 1) {
        rc_status st = scan_inclusive(bs, nb, nullptr, nullptr, total, s);
        if (st != RC_OK) return st;
        k_scan_add<<<(unsigned)nb, kScanThreads, 0, s>>>(x, n, bs);
        RC_LAUNCHED();
    }
    return RC_OK;
}

// ---------------------------------------------------------------------------
// sampling (Section 3.1)
// ---------------------------------------------------------------------------
__device__ __forceinline__ double uniform01(unsigned long long seed, long long i, int k)
{
    const unsigned long long ctr = (unsigned long long)(3 * i + k) * 0x9E3779B97F4A7C15ULL;
    const unsigned long long r = splitmix64(seed ^ ctr);
    return __dmul_rn(__ull2double_rn(r >> 11), 1.0 / 9007199254740992.0);
}

// total = cdf[T - 1], which the build has read back: the search need not wait
// for it.  kMany: conversions by integers, which spare the FP64 pipe but are a
// longer chain; they pay from about 128 points an SM on (203k triangles: 37
// points 6.5 us without and 7.4 with, 20,000 8.6 and 8.0, a million 93 and 76).
template <bool kMany>
__global__ void k_sample_area(const float* __restrict__ V, const int32_t* __restrict__ F, int64_t T,
                              const long long* __restrict__ cdf, long long total, const float* __restrict__ fnorm, int64_t n, unsigned long long seed,
                              float* P, float* Nout, int32_t* face, double* weight)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double u0 = uniform01(seed, i, 0), u1 = uniform01(seed, i, 1), u2 = uniform01(seed, i, 2);
    const long long target = (long long)floor(__dmul_rn(u0, __ll2double_rn(total)));
    int64_t lo = 0, hi = T - 1;
    while (lo < hi) {
        const int64_t mid = lo + (hi - lo) / 2;
        if (cdf[mid] > target) hi = mid; else lo = mid + 1;
    }
    const int64_t f = lo;
    const double s = __dsqrt_rn(u1);
    const double wa = __dsub_rn(1.0, s);
    const double wb = __dmul_rn(s, __dsub_rn(1.0, u2));
    const double wc = __dmul_rn(s, u2);
    for (int k = 0; k < 3; ++k) {
        const float a = V[3 * (int64_t)F[3 * f + 0] + k], b = V[3 * (int64_t)F[3 * f + 1] + k], c = V[3 * (int64_t)F[3 * f + 2] + k];
        const double A = kMany ? widen(a) : (double)a, B = kMany ? widen(b) : (double)b, C = kMany ? widen(c) : (double)c;
        double p = __dadd_rn(__dmul_rn(wa, A), __dmul_rn(wb, B));
        p = __dadd_rn(p, __dmul_rn(wc, C));
        P[3 * i + k] = kMany ? narrow(p) : __double2float_rn(p);
        Nout[3 * i + k] = fnorm[3 * f + k];
    }
    face[i] = (int32_t)f;
    if (weight) weight[i] = 1.0;
}

__global__ void k_sample_centroid(const float* __restrict__ V, const int32_t* __restrict__ F,
                                  const float* __restrict__ fnorm,
                                  const double* __restrict__ farea, int64_t T, float* P, float* Nout,
                                  int32_t* face, double* weight)
{
    int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (f >= T) return;
    for (int k = 0; k < 3; ++k) {
        P[3 * f + k] = face_centroid(V, F, f, k);
        Nout[3 * f + k] = fnorm[3 * f + k];
    }
    face[f] = (int32_t)f;
    if (weight) weight[f] = farea[f];
}

// Morton code (10 bits per axis) of each point inside the box [lo, hi]
__global__ void k_point_morton(const float* __restrict__ P, int64_t n, float lx, float ly, float lz, float sx,
                               float sy, float sz, unsigned long long* keys, int32_t* vals)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float lo[3] = {lx, ly, lz}, sc[3] = {sx, sy, sz};
    unsigned long long code = 0;
    for (int k = 0; k < 3; ++k) {
        float u = (P[3 * i + k] - lo[k]) * sc[k];
        u = fminf(fmaxf(u, 0.0f), 1023.0f);
        unsigned long long q = (unsigned long long)u;
        q = (q | (q << 16)) & 0x030000FFULL;
        q = (q | (q << 8)) & 0x0300F00FULL;
        q = (q | (q << 4)) & 0x030C30C3ULL;
        q = (q | (q << 2)) & 0x09249249ULL;
        code |= q << (2 - k);
    }
    keys[i] = code;
    vals[i] = (int32_t)i;
}

// ---------------------------------------------------------------------------
// host drivers
// ---------------------------------------------------------------------------
static inline unsigned nblocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

int device_sms()
{
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
    return sms;
}

// Stable LSD sort of (key, value) pairs by the low `passes` bytes of the key;
// the result is back in (keys, vals) when `passes` is even.
static rc_status sort_pairs(unsigned long long* keys, int32_t* vals, int64_t n, int passes, unsigned int* err,
                            cudaStream_t s)
{
    if (n <= 1) return RC_OK;
    if (n <= kSmallSort) {
        RC_CUDA(cudaFuncSetAttribute(k_sort_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSort)));
        k_sort_small<<<1, kSmallThreads, sizeof(SmallSort), s>>>(keys, vals, (int)n, passes, err);
        RC_LAUNCHED();
        return RC_OK;
    }
    unsigned long long* k1 = nullptr;
    int32_t* v1 = nullptr;
    unsigned int* counts = nullptr;
    // tiles of 512 to 2,048 keys, at least two per SM: small sorts spread over
    // the GPU, large ones keep the count table short (2,048 keys leave room
    // for five blocks per SM)
    const int sms = device_sms();
    const int items = n <= (int64_t)2 * sms * 512 ? 2 : n <= (int64_t)2 * sms * 1024 ? 4 : 8;
    const int64_t tile = (int64_t)items * kSortThreads;
    const int nblk = (int)((n + tile - 1) / tile);
    BuildScratch g{s};
    RC_CUDA(cudaMallocAsync(&k1, sizeof(unsigned long long) * n, s));
    g.p[0] = k1;
    RC_CUDA(cudaMallocAsync(&v1, sizeof(int32_t) * n, s));
    g.p[1] = v1;
    RC_CUDA(cudaMallocAsync(&counts, sizeof(unsigned int) * (256 * (size_t)nblk + 256), s));   // counts, then digit totals
    g.p[2] = counts;
    unsigned long long *kin = keys, *kout = k1;
    int32_t *vin = vals, *vout = v1;
    const auto scatter = items == 2 ? k_sort_scatter<2> : items == 4 ? k_sort_scatter<4> : k_sort_scatter<8>;
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = 8 * pass;
        k_sort_hist<<<nblk, kSortThreads, 0, s>>>(kin, n, shift, (int)tile, nblk, counts);
        RC_LAUNCHED();
        k_sort_scan<<<32, 256, 0, s>>>(counts, nblk, counts + (int64_t)256 * nblk);
        RC_LAUNCHED();
        scatter<<<nblk, kSortThreads, 0, s>>>(kin, vin, n, shift, nblk, counts, counts + (int64_t)256 * nblk, kout, vout,
                                              err);
        RC_LAUNCHED();
        std::swap(kin, kout);
        std::swap(vin, vout);
    }
    return RC_OK;
}

// Processing order of sample points: indices sorted by the Morton code of
// the point within the part's bounding box (written to `order`).
rc_status point_order(rc_bvh h, const float* P, int64_t n, int32_t* order, cudaStream_t s)
{
    unsigned long long* keys = nullptr;
    BuildScratch g{s};
    RC_CUDA(cudaMallocAsync(&keys, sizeof(unsigned long long) * n, s));
    g.p[0] = keys;
    float sc[3];
    for (int k = 0; k < 3; ++k) {
        const float ext = h->hi[k] - h->lo[k];
        sc[k] = ext > 0.0f ? 1024.0f / ext : 0.0f;
    }
    k_point_morton<<<nblocks(n, 256), 256, 0, s>>>(P, n, h->lo[0], h->lo[1], h->lo[2], sc[0], sc[1], sc[2], keys,
                                                   order);
    RC_LAUNCHED();
    return sort_pairs(keys, order, n, 4, (unsigned int*)&h->sc->pad, s);
}

__global__ void k_init_scalars(DevScalars* sc)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    sc->amax_bits = 0;
    for (int k = 0; k < 3; ++k) { sc->cmin[k] = 0x7FFFFFFF; sc->cmax[k] = (int)0x80000000; }
    sc->vmaxabs = 0;
    sc->err_index = 0x7FFFFFFF;
    sc->err_vertex = 0x7FFFFFFF;
    sc->max_depth = 0;
    sc->pad = 0;
    sc->wide_depth = 0;
    sc->wide_nodes = 0;
}

static rc_status init_scalars(DevScalars* sc, cudaStream_t s)
{
    k_init_scalars<<<1, 32, 0, s>>>(sc);
    RC_LAUNCHED();
    return RC_OK;
}

static rc_status face_data(rc_bvh h, float* tbox, cudaStream_t s)
{
    rc_status st = init_scalars(h->sc, s);
    if (st != RC_OK) return st;
    k_face_prep<<<(unsigned)std::min<int64_t>(nblocks(h->T, kPrepThreads), 8 * (int64_t)device_sms()), kPrepThreads, 0, s>>>(
        h->V, h->nV, h->F, h->T, h->fnorm, h->farea, tbox, h->sc);
    RC_LAUNCHED();
    return scan_inclusive(h->cdf, h->T, h->farea, h->sc, &h->sc->total, s);
}

// mesh validity and scene bounds from the scalars already read back
static rc_status checked_scalars(rc_bvh h)
{
    const DevScalars& d = h->host_sc;
    if (d.err_index != 0x7FFFFFFF)
        return set_error(RC_E_ARG, "face " + std::to_string(d.err_index) + " has a vertex index outside [0, nV)");
    if (d.err_vertex != 0x7FFFFFFF)
        return set_error(RC_E_ARG, "vertex " + std::to_string(d.err_vertex) + " is not finite");
    h->scene_maxabs = std::max(1.0f, ordered_to_float(d.vmaxabs));
    // the tree depth is set by the build once the tree exists (a refit keeps
    // the topology and hence the depth)
    return RC_OK;
}

// PLOC build of the binary tree over the Morton-sorted leaves (h->order);
// writes h->child, h->range, h->parent in the Karras layout and replaces
// h->order by the depth-first leaf order.
static rc_status build_ploc(rc_bvh h, const float* tbox, cudaStream_t s)
{
    const int64_t T = h->T, n_int = h->n_int;
    if (T > 0x7FFFFFFF / 2) return set_error(RC_E_UNSUPPORTED, "too many triangles for the PLOC build");
    const int64_t nb_max = (T + kCompact - 1) / kCompact;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
    const size_t o_cla = take(4 * T), o_clt = take(4 * T), o_cba = take(24 * T), o_cbt = take(24 * T);
    const size_t o_nn = take(4 * T), o_keep = take(4 * T), o_bsum = take(4 * nb_max), o_n = take(16);
    const size_t o_craw = take(8 * n_int), o_praw = take(4 * (n_int + T)), o_szl = take(4 * n_int);
    const size_t o_szi = take(4 * n_int), o_nid = take(4 * n_int), o_ls = take(4 * n_int), o_pos = take(4 * T);
    const size_t o_ord = take(4 * T);
    char* base = nullptr;
    BuildScratch g{s};
    RC_CUDA(cudaMallocAsync((void**)&base, off, s));
    g.p[0] = base;
    int32_t* cl_a = (int32_t*)(base + o_cla);
    int32_t* cl_t = (int32_t*)(base + o_clt);
    float* cb_a = (float*)(base + o_cba);
    float* cb_t = (float*)(base + o_cbt);
    int32_t* nn = (int32_t*)(base + o_nn);
    int* keep = (int*)(base + o_keep);
    int* bsum = (int*)(base + o_bsum);
    int* dn = (int*)(base + o_n);          // [0], [1]: cluster counts (ping-pong), [2]: node counter, [3]: error
    int32_t* child_raw = (int32_t*)(base + o_craw);
    int32_t* parent_raw = (int32_t*)(base + o_praw);
    int32_t* sz_leaf = (int32_t*)(base + o_szl);
    int32_t* sz_int = (int32_t*)(base + o_szi);
    int32_t* newid = (int32_t*)(base + o_nid);
    int32_t* lstart = (int32_t*)(base + o_ls);
    int32_t* pos = (int32_t*)(base + o_pos);
    int32_t* order_out = (int32_t*)(base + o_ord);
    RC_CUDA(cudaMemsetAsync(dn, 0, 16, s));
    RC_CUDA(cudaMemsetAsync(parent_raw, 0xFF, 4 * (n_int + T), s));
    k_ploc_init<<<nblocks(T, 256), 256, 0, s>>>(tbox, h->order, T, n_int, cl_a, cb_a, dn);
    RC_LAUNCHED();
    int cur = 0;
    int64_t n_host = T;
    const int kRoundsPerCheck = 8;
    int rounds = 0;
    while (n_host > 1) {
        if (rounds > 64 + 8 * 64) return set_error(RC_E_DEVICE, "PLOC build did not converge");
        const unsigned g_nn = (unsigned)((n_host + kPlocThreads - 1) / kPlocThreads);
        const unsigned g_c = (unsigned)((n_host + kCompact - 1) / kCompact);
        for (int r = 0; r < kRoundsPerCheck; ++r, ++rounds) {
            k_ploc_nn<<<g_nn, kPlocThreads, 0, s>>>(dn + cur, cb_a, nn);
            RC_LAUNCHED();
            k_ploc_merge<<<g_nn, kPlocThreads, 0, s>>>(dn + cur, nn, cl_a, cb_a, cl_t, cb_t, keep, child_raw,
                                                       parent_raw, dn + 2, n_int);
            RC_LAUNCHED();
            k_ploc_count<<<g_c, kCompact, 0, s>>>(dn + cur, keep, bsum);
            RC_LAUNCHED();
            k_ploc_scan<<<1, 32, 0, s>>>(bsum, (int)g_c, dn + cur, dn + 1 - cur);
            RC_LAUNCHED();
            k_ploc_scatter<<<g_c, kCompact, 0, s>>>(dn + cur, keep, bsum, cl_t, cb_t, cl_a, cb_a);
            RC_LAUNCHED();
            cur = 1 - cur;
        }
        int hn[3];
        RC_CUDA(cudaMemcpyAsync(hn, dn, sizeof hn, cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaStreamSynchronize(s));
        n_host = hn[cur];
        if (n_host == 1 && hn[2] != n_int)
            return set_error(RC_E_DEVICE, "PLOC build made a wrong number of interior nodes");
    }
    // depth-first renumbering into the Karras layout
    RC_CUDA(cudaMemsetAsync(h->visits, 0, sizeof(int32_t) * n_int, s));
    k_ploc_sizes<<<nblocks(T, 256), 256, 0, s>>>(T, n_int, parent_raw, child_raw, sz_leaf, sz_int, h->visits,
                                                 dn + 3);
    RC_LAUNCHED();
    k_ploc_number<<<nblocks(n_int + T, 256), 256, 0, s>>>(T, n_int, parent_raw, child_raw, sz_leaf, sz_int, newid,
                                                          lstart, pos, dn + 3);
    RC_LAUNCHED();
    k_ploc_emit<<<nblocks(n_int + T, 256), 256, 0, s>>>(T, n_int, parent_raw, child_raw, newid, lstart, sz_leaf, pos,
                                                        h->order, h->child, h->range, h->parent, order_out);
    RC_LAUNCHED();
    RC_CUDA(cudaMemcpyAsync(h->order, order_out, sizeof(int32_t) * T, cudaMemcpyDeviceToDevice, s));
    int herr = 0;
    RC_CUDA(cudaMemcpyAsync(&herr, dn + 3, sizeof herr, cudaMemcpyDeviceToHost, s));
    RC_CUDA(cudaStreamSynchronize(s));
    if (herr) return set_error(RC_E_DEVICE, "PLOC tree walk exceeded its bound");
    return RC_OK;
}

// Collapse the binary tree into the 4-wide layout (wnodes), or make the
// one-leaf wide root for tiny parts.  Needs the binary tree and its boxes.
static rc_status build_wide(rc_bvh h, const float* tbox, cudaStream_t s)
{
    const int64_t T = h->T;
    if (!h->wnodes) RC_CUDA(cudaMallocAsync(&h->wnodes, sizeof(float4) * 8 * h->n_int, s));
    if (T <= kLeafMax) {
        k_wide_small<<<1, 32, 0, s>>>(T, tbox, h->wnodes, h->sc);
        RC_LAUNCHED();
        return RC_OK;
    }
    const int64_t n_int = h->n_int;
    int2* q = nullptr;
    BuildScratch g{s};
    RC_CUDA(cudaMallocAsync(&q, sizeof(int2) * (2 * n_int + 1), s));   // two queues, then their sizes
    g.p[0] = q;
    int2 *qa = q, *qb = q + n_int;
    int *ca = (int*)(q + 2 * n_int), *cb = ca + 1;
    int* wide_count = &h->sc->wide_nodes;
    // The top `split` levels go level by level (a level's queue is at most
    // 4^level long); then one launch finishes every queued subtree, a thread
    // each, once the queue holds about n_int / RC_WIDE_SUBTREE nodes.  Levels
    // past the bottom of a shallow tree find an empty queue.
    int split = 0;
    while (split < 30 && std::pow(4.0, (double)split) * RC_WIDE_SUBTREE < (double)n_int) ++split;
    if (RC_WIDE_SUBTREE <= 0) split = kStack;      // a deeper tree is rejected anyway
    int level = std::min(split, kWideTop);
    k_wide_top<<<1, kWideTopThreads, 0, s>>>(h->nodes, qa, qb, ca, wide_count, h->wnodes, h->sc, level);
    RC_LAUNCHED();
    if (level & 1) {
        std::swap(qa, qb);
        std::swap(ca, cb);
    }
    for (; level < split; ++level) {
        const double cap = std::min((double)n_int, std::pow(4.0, (double)std::min(level, 30)));
        const unsigned grid = (unsigned)std::max(1.0, std::ceil(cap / 256.0));
        RC_CUDA(cudaMemsetAsync(cb, 0, sizeof(int), s));
        k_wide_level<<<grid, 256, 0, s>>>(h->nodes, qa, ca, qb, cb, wide_count, h->wnodes, h->sc, level);
        RC_LAUNCHED();
        std::swap(qa, qb);
        std::swap(ca, cb);
    }
    {
        const double cap = std::min((double)n_int, std::pow(4.0, (double)std::min(level, 30)));
        const unsigned grid = (unsigned)std::max(1.0, std::ceil(cap / 256.0));
        k_wide_subtrees<<<grid, 256, 0, s>>>(h->nodes, qa, ca, wide_count, h->wnodes, h->sc, level);
        RC_LAUNCHED();
    }
    return RC_OK;
}

// ---------------------------------------------------------------------------
// The 4-wide tree with its child boxes in the coordinates of a machining
// frame (rows of M = the frame's columns): the same nodes, codes and
// triangles; each box is the bounding box of the frame coordinates of its
// triangles' vertices, evaluated in two-term fp32 sums and rounded outward.  The
// axis walk of the orthogonal cast tests these boxes (its rays run along a
// frame axis) and still tests triangles in world coordinates.
// ---------------------------------------------------------------------------
// q (two-term, exact to 1e-13 of sum |x_i f_i|) of a vertex along one frame
// axis, rounded outward; the roundings of frame coordinates in FP64 are covered
__device__ __forceinline__ void frame_bounds(float x, float y, float z, float a, float b, float c, float& lo, float& hi)
{
    float h, l;
    dot2(x, a, y, b, z, c, h, l);
    const float e = 2e-13f * (fabsf(x * a) + fabsf(y * b) + fabsf(z * c)) + 1e-36f;
    const bool in = fabsf(h) < INFINITY;           // else beyond fp32's range: no bound
    lo = fminf(lo, in ? __fadd_rd(h, __fsub_rd(l, e)) : -INFINITY);
    hi = fmaxf(hi, in ? __fadd_ru(h, __fadd_ru(l, e)) : INFINITY);
}

// leaf boxes in frame coordinates and all boxes above them.  The bounds are
// formed in two-term fp32 sums: in FP64 (1/64 of the fp32 rate) the leaf boxes
// alone took 50 us for 203k triangles and the climb 49, together now 43.
__global__ void __launch_bounds__(kClimb)
k_frame_refit(const float* __restrict__ V, int64_t nV, const int32_t* __restrict__ F, const int32_t* __restrict__ order,
              int64_t T, int64_t n_int, FrameArgs fa, const int32_t* __restrict__ parent,
              const int32_t* __restrict__ child, const int32_t* __restrict__ range, float* nbox_f, int32_t* visits)
{
    __shared__ ClimbShared sm;
    const int64_t k = blockIdx.x * (int64_t)kClimb + threadIdx.x;
    float v[3][3];
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    if (k < T && gather_tri(V, nV, F, T, order[k], v))
        for (int a = 0; a < 3; ++a)
            for (int j = 0; j < 3; ++j)            // frame coordinate j: column j of the row-major frame
                frame_bounds(v[a][0], v[a][1], v[a][2], fa.f[0][j], fa.f[0][3 + j], fa.f[0][6 + j], lo[j], hi[j]);
    if (parent) climb<false>(sm, k < T, T, n_int, parent, child, range, nbox_f, nullptr, visits, nullptr, k, lo, hi);
    else if (k < T) put_box(nbox_f, n_int + k, lo, hi);
}

__global__ void k_frame_pack(const float4* __restrict__ wnodes, int64_t n_int, int64_t T,
                             const DevScalars* __restrict__ sc, const float* __restrict__ nbox_f,
                             const float* __restrict__ all_box, float4* __restrict__ ftree)
{
    const int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (w >= sc->wide_nodes || w >= n_int) return;
    const float4 idv = wnodes[wide_at(w, 7)];
    const int32_t ids[4] = {__float_as_int(idv.x), __float_as_int(idv.y), __float_as_int(idv.z), __float_as_int(idv.w)};
    float lo[3][4], hi[3][4];
    const float4 cv = wnodes[wide_at(w, 6)];
    const int32_t codes[4] = {__float_as_int(cv.x), __float_as_int(cv.y), __float_as_int(cv.z), __float_as_int(cv.w)};
    for (int k = 0; k < 4; ++k) {
        const float* b = nullptr;
        int n = 1;
        if (ids[k] == kAllTris) b = all_box;
        else if (ids[k] >= 0 && ids[k] < n_int) b = nbox_f + 6 * (int64_t)ids[k];
        else if (ids[k] == kLeafChild && leaf_first(codes[k]) + leaf_count(codes[k]) <= T) {
            b = nbox_f + 6 * (n_int + leaf_first(codes[k]));
            n = leaf_count(codes[k]);
        }
        for (int a = 0; a < 3; ++a) {
            lo[a][k] = INFINITY;
            hi[a][k] = -INFINITY;
            for (int t = 0; b && t < n; ++t) {
                lo[a][k] = fminf(lo[a][k], b[6 * t + a]);
                hi[a][k] = fmaxf(hi[a][k], b[6 * t + 3 + a]);
            }
        }
    }
    for (int a = 0; a < 3; ++a) {
        ftree[wide_at(w, 2 * a)] = make_float4(lo[a][0], lo[a][1], lo[a][2], lo[a][3]);
        ftree[wide_at(w, 2 * a + 1)] = make_float4(hi[a][0], hi[a][1], hi[a][2], hi[a][3]);
    }
    ftree[wide_at(w, 6)] = wnodes[wide_at(w, 6)];
    ftree[wide_at(w, 7)] = idv;
}

// box of all leaf slots [0, T) of nbox_f (tiny parts: the one-leaf root)
__global__ void k_frame_all_box(const float* __restrict__ nbox_f, int64_t n_int, int64_t T, float* out)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t k = 0; k < T; ++k)
        for (int a = 0; a < 3; ++a) {
            lo[a] = fminf(lo[a], nbox_f[6 * (n_int + k) + a]);
            hi[a] = fmaxf(hi[a], nbox_f[6 * (n_int + k) + 3 + a]);
        }
    for (int a = 0; a < 3; ++a) { out[a] = lo[a]; out[3 + a] = hi[a]; }
}

rc_status frame_tree(rc_bvh h, const float f9[9], float4* ftree, cudaStream_t s)
{
    const int64_t T = h->T, n_int = h->n_int;
    FrameArgs fa = {};
    for (int k = 0; k < 9; ++k) fa.f[0][k] = f9[k];
    float* nbox_f = nullptr;
    int32_t* visits = nullptr;
    BuildScratch g{s};
    RC_CUDA(cudaMallocAsync(&nbox_f, sizeof(float) * 6 * (n_int + T + 1), s));
    g.p[0] = nbox_f;
    float* all_box = nbox_f + 6 * (n_int + T);
    const unsigned grid = nblocks(T, kClimb);
    if (T > kLeafMax) {
        RC_CUDA(cudaMallocAsync(&visits, sizeof(int32_t) * n_int, s));
        g.p[1] = visits;
        RC_CUDA(cudaMemsetAsync(visits, 0, sizeof(int32_t) * n_int, s));
        k_frame_refit<<<grid, kClimb, 0, s>>>(h->V, h->nV, h->F, h->order, T, n_int, fa, h->parent, h->child, h->range,
                                              nbox_f, visits);
        RC_LAUNCHED();
    } else {
        k_frame_refit<<<grid, kClimb, 0, s>>>(h->V, h->nV, h->F, h->order, T, n_int, fa, nullptr, nullptr, nullptr, nbox_f,
                                              nullptr);
        RC_LAUNCHED();
        k_frame_all_box<<<1, 32, 0, s>>>(nbox_f, n_int, T, all_box);
        RC_LAUNCHED();
    }
    k_frame_pack<<<(unsigned)((n_int + 255) / 256), 256, 0, s>>>(h->wnodes, n_int, T, h->sc, nbox_f, all_box, ftree);
    RC_LAUNCHED();
    return RC_OK;
}

// triangle records, boxes and packed binary nodes of the tree in h (tiny
// parts: records only)
static rc_status refit_tree(rc_bvh h, cudaStream_t s)
{
    const bool tree = h->T > kLeafMax;
    if (tree) RC_CUDA(cudaMemsetAsync(h->visits, 0, sizeof(int32_t) * h->n_int, s));
    k_refit<<<nblocks(h->T, kClimb), kClimb, 0, s>>>(h->V, h->nV, h->F, h->order, h->T, h->n_int, tree ? h->parent : nullptr,
                                               h->child, h->range, h->nbox, h->nodes, h->tris, h->visits, h->sc);
    RC_LAUNCHED();
    return RC_OK;
}

rc_status build_bvh(rc_bvh h, cudaStream_t s)
{
    const int64_t T = h->T;
    float* tbox = nullptr;
    BuildScratch g{s};
    RC_CUDA(cudaMallocAsync(&tbox, sizeof(float) * 6 * T, s));
    g.p[0] = tbox;
    // No host synchronisation until the end: a bad mesh is reported from the
    // one final readback (every kernel in between guards its gathers).
    rc_status st = face_data(h, tbox, s);
    if (st != RC_OK) return st;

    h->n_int = T > kLeafMax ? T - 1 : 1;
    RC_CUDA(cudaMallocAsync(&h->nodes, sizeof(float4) * 4 * h->n_int, s));
    RC_CUDA(cudaMallocAsync(&h->tris, sizeof(float4) * 3 * T, s));
    RC_CUDA(cudaMallocAsync(&h->order, sizeof(int32_t) * T, s));

    if (T <= kLeafMax) {
        int32_t ord[kLeafMax];
        for (int i = 0; i < kLeafMax; ++i) ord[i] = i;
        RC_CUDA(cudaMemcpyAsync(h->order, ord, sizeof(int32_t) * T, cudaMemcpyHostToDevice, s));
        k_pack_small<<<1, 32, 0, s>>>(T, tbox, h->nodes, h->sc);
        RC_LAUNCHED();
        h->max_depth = 1;
    } else {
        unsigned long long* k0 = nullptr;
        RC_CUDA(cudaMallocAsync(&k0, sizeof(unsigned long long) * T, s));
        g.p[1] = k0;
        k_morton<<<nblocks(T, 256), 256, 0, s>>>(tbox, T, h->sc, k0, h->order);
        RC_LAUNCHED();
        rc_status sst = sort_pairs(k0, h->order, T, kMortonPasses, (unsigned int*)&h->sc->pad, s);
        if (sst != RC_OK) return sst;
        // after an even number of passes the sorted data is back in (k0, h->order)
        const int64_t n_int = h->n_int;
        RC_CUDA(cudaMallocAsync(&h->parent, sizeof(int32_t) * (n_int + T), s));
        RC_CUDA(cudaMallocAsync(&h->child, sizeof(int32_t) * 2 * n_int, s));
        RC_CUDA(cudaMallocAsync(&h->range, sizeof(int32_t) * 2 * n_int, s));
        RC_CUDA(cudaMallocAsync(&h->nbox, sizeof(float) * 6 * (n_int + T), s));
        RC_CUDA(cudaMallocAsync(&h->visits, sizeof(int32_t) * n_int, s));
        if (h->builder == RC_BUILDER_PLOC) {
            rc_status pst = build_ploc(h, tbox, s);
            if (pst != RC_OK) return pst;
        } else {
            k_karras<<<nblocks(n_int, 256), 256, 0, s>>>(k0, T, h->child, h->range, h->parent);
            RC_LAUNCHED();
        }
    }
    if ((st = refit_tree(h, s)) != RC_OK) return st;
    st = build_wide(h, tbox, s);
    if (st != RC_OK) return st;
    RC_CUDA(cudaMemcpyAsync(&h->host_sc, h->sc, sizeof(DevScalars), cudaMemcpyDeviceToHost, s));
    RC_CUDA(cudaStreamSynchronize(s));
    if ((st = checked_scalars(h)) != RC_OK) return st;
    if (h->host_sc.pad != 0) return set_error(RC_E_DEVICE, "radix sort produced an out-of-range position");
    if (T > kLeafMax) h->max_depth = h->host_sc.max_depth;
    h->wide_depth = h->host_sc.wide_depth;
    for (int k = 0; k < 3; ++k) { h->lo[k] = h->host_sc.lo[k]; h->hi[k] = h->host_sc.hi[k]; }
    if (h->max_depth >= kStack)
        return set_error(RC_E_UNSUPPORTED, "BVH depth " + std::to_string(h->max_depth) +
                                               " exceeds the traversal stack");
    if (3 * h->wide_depth + 1 >= kStack4)
        return set_error(RC_E_UNSUPPORTED, "4-wide BVH depth " + std::to_string(h->wide_depth) +
                                               " exceeds the traversal stack");
    return RC_OK;
}

rc_status refit_bvh(rc_bvh h, cudaStream_t s)
{
    const int64_t T = h->T;
    float* tbox = nullptr;
    BuildScratch g{s};
    RC_CUDA(cudaMallocAsync(&tbox, sizeof(float) * 6 * T, s));
    g.p[0] = tbox;
    rc_status st = face_data(h, tbox, s);
    if (st != RC_OK) return st;
    if (T <= kLeafMax) {
        k_pack_small<<<1, 32, 0, s>>>(T, tbox, h->nodes, h->sc);
        RC_LAUNCHED();
    }
    if ((st = refit_tree(h, s)) != RC_OK) return st;
    st = build_wide(h, tbox, s);
    if (st != RC_OK) return st;
    // one synchronisation, as in the build: a bad vertex is reported from the
    // final readback
    RC_CUDA(cudaMemcpyAsync(&h->host_sc, h->sc, sizeof(DevScalars), cudaMemcpyDeviceToHost, s));
    RC_CUDA(cudaStreamSynchronize(s));
    if ((st = checked_scalars(h)) != RC_OK) return st;
    for (int k = 0; k < 3; ++k) { h->lo[k] = h->host_sc.lo[k]; h->hi[k] = h->host_sc.hi[k]; }
    h->wide_depth = h->host_sc.wide_depth;
    if (3 * h->wide_depth + 1 >= kStack4)
        return set_error(RC_E_UNSUPPORTED, "4-wide BVH depth exceeds the traversal stack after refit");
    return RC_OK;
}

rc_status sample_points(rc_bvh h, int64_t n, const rc_params* p, float* P, float* N, int32_t* face,
                        double* weight, cudaStream_t s)
{
    if (p->sample_mode == RC_SAMPLE_FACE_CENTROID) {
        k_sample_centroid<<<nblocks(h->T, 256), 256, 0, s>>>(h->V, h->F, h->fnorm, h->farea, h->T, P, N, face,
                                                             weight);
        RC_LAUNCHED();
        return RC_OK;
    }
    const auto kernel = n > 128 && n > 128 * (int64_t)device_sms() ? k_sample_area<true> : k_sample_area<false>;
    kernel<<<nblocks(n, 256), 256, 0, s>>>(h->V, h->F, h->T, h->cdf, h->host_sc.total, h->fnorm, n, p->seed, P, N, face,
                                           weight);
    RC_LAUNCHED();
    return RC_OK;
}

}  // namespace rc
