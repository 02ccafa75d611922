// reduce.cu -- Section 3.3 reductions: directional variability of the
// visible directions (dominant axis, axis concentration, part sums), the
// per-direction visible-area histogram, fixture faces and face classes with
// the 64-bin histogram of reachable-axis masks for the setup cover.
//
// The counts, shares and concentrations are int64 sums of fixed-point
// values, and the area-weighted sums are FP64 sums in a fixed order (per
// warp, per block, then over the blocks by one warp), so the summary does
// not depend on the order in which blocks finish.
#include <math.h>
#include <string.h>

#include <algorithm>

#include "rc_internal.cuh"

namespace rc {

enum { S_COUNTED = 0, S_DOM = 1, S_COUNT = 4, S_CONC = 5, S_N = 6 };
static_assert(S_N <= kVarSums, "integer sums of the variability scratch");

// round(x * 2^40) to nearest, ties to even, for an fp32 x with |x| < 8, in
// fp32 arithmetic: x * 2^40 = hi * 2^22 + lo with hi = rint(x * 2^18) and
// lo = rint((x * 2^18 - hi) * 2^22).  x * 2^18 and its remainder are exact;
// each rint adds 1.5 * 2^23, whose ulp is 1, and reads the integer from the
// bits.  hi * 2^22 is even, so rounding the remainder alone makes the same
// tie decisions as rounding the whole (equal to llrint((double)x * 2^40)).
__device__ __forceinline__ void fixed40_split(float x, int& hi, int& lo)
{
    const float C = 12582912.0f;
    const float t = __fmul_rn(x, 262144.0f);
    const float a = __fadd_rn(t, C);
    hi = __float_as_int(a) - __float_as_int(C);
    const float r = __fsub_rn(t, __fsub_rn(a, C));
    lo = __float_as_int(__fmaf_rn(r, 4194304.0f, C)) - __float_as_int(C);
}

// Two fp32 values per register pair: one instruction issues both operations,
// each rounded as the scalar one.
using f2 = unsigned long long;
__device__ __forceinline__ f2 pack2(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// The rounded product: a fused multiply-add of minus zero, whose value the
// compiler must not know.  It joins mul.rn.f32x2 and add.rn.f32x2 into a fused
// multiply-add (for scalars it does not), which moved the largest component of
// a direction in 30 of 10^6 points x 2048 directions.
__device__ __forceinline__ f2 mul2(f2 a, f2 b, f2 minus_zero)
{
    return fma2(a, b, minus_zero);
}

// The exact direction sums of one point, by one warp: M_k = sum over visible
// j of llrint(d_jk * 2^40), the same in every lane.  The bit row is read 32
// words at a time by the whole warp (one coalesced load) and each word is
// handed to the lanes by a shuffle.
struct DirSums { long long M[3]; };

__device__ __noinline__ DirSums exact_sums(const uint32_t* __restrict__ bits, float nx, float ny, float nz, int64_t i, int W,
                                           const float4* __restrict__ dirs)
{
    const int lane = threadIdx.x & 31;
    const Onb b = make_onb(nx, ny, nz);
    long long M0 = 0, M1 = 0, M2 = 0;
    for (int w0 = 0; w0 < W; w0 += 32) {
        const int wn = min(32, W - w0);
        const uint32_t mine = lane < wn ? __ldg(&bits[i * W + w0 + lane]) : 0u;
        // per 32 words a lane adds at most 32 terms: |sum hi| < 2^24,
        // |sum lo| < 2^27, so int32 partial sums are exact
        int h0 = 0, h1 = 0, h2 = 0, l0 = 0, l1 = 0, l2 = 0;
        for (int dw = 0; dw < wn; ++dw) {
            const uint32_t word = __shfl_sync(0xFFFFFFFFu, mine, dw);
            if (!((word >> lane) & 1u)) continue;
            const float4 h = __ldg(&dirs[32 * (w0 + dw) + lane]);
            float dx, dy, dz;
            local_to_world(b, nx, ny, nz, h.x, h.y, h.z, dx, dy, dz);
            int qh, ql;
            fixed40_split(dx, qh, ql);
            h0 += qh;
            l0 += ql;
            fixed40_split(dy, qh, ql);
            h1 += qh;
            l1 += ql;
            fixed40_split(dz, qh, ql);
            h2 += qh;
            l2 += ql;
        }
        M0 += (long long)h0 * 4194304LL + l0;
        M1 += (long long)h1 * 4194304LL + l1;
        M2 += (long long)h2 * 4194304LL + l2;
    }
    for (int off = 16; off; off >>= 1) {
        M0 += __shfl_xor_sync(0xFFFFFFFFu, M0, off);
        M1 += __shfl_xor_sync(0xFFFFFFFFu, M1, off);
        M2 += __shfl_xor_sync(0xFFFFFFFFu, M2, off);
    }
    return DirSums{{M0, M1, M2}};
}

// Per point: visible rays, the axis of the largest |M_k|, and the visible
// rays whose largest |component| is that axis.  A warp takes the points in
// groups of G (a power of two up to 32): it goes through a point's directions
// lane by lane, lane q keeps the results of the group's point q, and the
// group's quotients are then formed by all its lanes at once.  What it was
// bound by: FP64, which issues at 1/64 of the fp32 rate -- one lane formed
// each point's quotients -- and then the three fixed-point conversions per
// visible direction.  Now:
//   - Only the axis of the largest sum is needed (conc_mode 0), so the sums
//     are taken in fp32 and the exact ones only where the two largest lie
//     within their error bound u B count (W / 2 + 8), |d_k| <= B: a lane adds
//     at most W / 2 terms per half, then the halves and five shuffles.
//   - Two directions per instruction (f32x2), from a table in shared memory
//     whose entries are the pairs of words 2 p and 2 p + 1.
// 300k points x 1000 directions, 70% visible: 729 -> 467 us.
// conc_mode 1 (kSums) needs the exact sums themselves and no counts by axis: it
// takes them in the one pass, two directions per instruction as well (300k
// points x 1000 directions 532 us, 20k x 8192, whose table is read from L1,
// 374; the fp32 pass and then exact_sums 1151 and 705).
constexpr int kVarThreads = 256, kVarBlocks = 4;   // 3, 5 and 6 blocks per SM measured 6 to 9% slower
constexpr int kVarTableWords = 96;     // most words of the shared table (36 KB); beyond, the table is read from L1

// fixed40_split of the two values of x where they are visible, added to the
// sums hi and lo, each with the bits of C on top (kFixedC a value, modulo
// 2^32: taken off once per sum)
constexpr unsigned kFixedC = 0x4B400000u;
__device__ __forceinline__ void add_fixed40(f2 x, bool v0, bool v1, unsigned& hi, unsigned& lo)
{
    const float C = 12582912.0f;                             // the float of bits kFixedC
    const f2 k18 = pack2(262144.0f, 262144.0f), k22 = pack2(4194304.0f, 4194304.0f), c = pack2(C, C), neg = pack2(-1.0f, -1.0f);
    float x0, x1;
    unpack2(x, x0, x1);
    const f2 y = pack2(v0 ? x0 : 0.0f, v1 ? x1 : 0.0f);      // zero adds zero to both
    const f2 a = fma2(y, k18, c), r = fma2(y, k18, fma2(a, neg, c)), l = fma2(r, k22, c);
    float a0, a1, l0, l1;
    unpack2(a, a0, a1);
    unpack2(l, l0, l1);
    hi += __float_as_uint(a0) + __float_as_uint(a1);
    lo += __float_as_uint(l0) + __float_as_uint(l1);
}

template <bool kTable, bool kSums>
__global__ void __launch_bounds__(kVarThreads, kVarBlocks)
k_variability(const uint32_t* __restrict__ bits, const float* __restrict__ Nrm,
              const double* __restrict__ weight, int64_t n,
              const float4* __restrict__ dirs, int n_dirs, int G, float* acc, int8_t* dom,
              float* conc, unsigned long long* sums, double* wpart)
{
    constexpr unsigned kAll = 0xFFFFFFFFu;
    extern __shared__ float2 s_dirs[];     // [3][pairs of words][32]
    __shared__ long long blk[S_N];
    __shared__ double wsh[2][kVarThreads / 32];
    const int lane = threadIdx.x & 31;
    const int W = (n_dirs + 31) >> 5, np = (W + 1) >> 1;
    const float nzero = __int_as_float((int)(0x80000000u | (unsigned)(n >> 63)));   // n >= 0: -0.0f
    const f2 mz = pack2(nzero, nzero);
    if (threadIdx.x < S_N) blk[threadIdx.x] = 0;
    if (kTable)
        for (int k = threadIdx.x; k < 32 * np; k += kVarThreads) {
            const int p = k >> 5, l = k & 31;
            const float4 h0 = __ldg(&dirs[64 * p + l]);
            const float4 h1 = 2 * p + 1 < W ? __ldg(&dirs[64 * p + 32 + l]) : h0;
            s_dirs[k] = make_float2(h0.x, h1.x);
            s_dirs[32 * np + k] = make_float2(h0.y, h1.y);
            s_dirs[64 * np + k] = make_float2(h0.z, h1.z);
        }
    __syncthreads();
    long long loc[S_N] = {0, 0, 0, 0, 0, 0};
    double lwc = 0.0, lw = 0.0;            // this lane's points: sum w_i count_i and sum w_i, in order
    const int64_t nw = (int64_t)gridDim.x * (kVarThreads >> 5);
    for (int64_t g = (int64_t)blockIdx.x * (kVarThreads >> 5) + (threadIdx.x >> 5); g * G < n; g += nw) {
        const int m = (int)min64(G, n - g * G);
        int my_cnt = 0, my_axis = 0, my_dm = -1;   // point `lane` of the group: visible rays, those along dm, dm
        long long my_M = 0;                        // |M_dm| (kSums)
        for (int q = 0; q < m; ++q) {
            const int64_t i = g * G + q;
            const float nx = Nrm[3 * i], ny = Nrm[3 * i + 1], nz = Nrm[3 * i + 2];
            const Onb b = make_onb(nx, ny, nz);
            const f2 ax = pack2(b.t1x, b.t1x), ay = pack2(b.t1y, b.t1y), az = pack2(b.t1z, b.t1z);
            const f2 bx = pack2(b.t2x, b.t2x), by = pack2(b.t2y, b.t2y), bz = pack2(b.t2z, b.t2z);
            const f2 cx = pack2(nx, nx), cy = pack2(ny, ny), cz = pack2(nz, nz);
            f2 sx = 0, sy = 0, sz = 0;
            long long M0 = 0, M1 = 0, M2 = 0;
            int a1 = 0, a2 = 0, cnt = 0;
            for (int w0 = 0; w0 < W; w0 += 32) {
                const int wn = min(32, W - w0);
                const uint32_t mine = lane < wn ? __ldg(&bits[i * W + w0 + lane]) : 0u;
                cnt += __popc(mine);
                unsigned h0 = 0, h1 = 0, h2 = 0, l0 = 0, l1 = 0, l2 = 0;   // as in exact_sums
                unsigned off = 0;
                for (int dw = 0; dw < wn; dw += 2) {
                    const uint32_t u0 = __shfl_sync(kAll, mine, dw), u1 = __shfl_sync(kAll, mine, dw + 1);
                    if ((u0 | u1) == 0u) continue;
                    if (kSums) off -= 2 * kFixedC;
                    f2 hx, hy, hz;
                    if (kTable) {
                        const float2* t = s_dirs + 16 * (w0 + dw) + lane;
                        hx = *(const f2*)t;
                        hy = *(const f2*)(t + 32 * np);
                        hz = *(const f2*)(t + 64 * np);
                    } else {
                        const float4 h0 = __ldg(&dirs[32 * (w0 + dw) + lane]);
                        const float4 h1 = dw + 1 < wn ? __ldg(&dirs[32 * (w0 + dw + 1) + lane]) : h0;
                        hx = pack2(h0.x, h1.x);
                        hy = pack2(h0.y, h1.y);
                        hz = pack2(h0.z, h1.z);
                    }
                    // local_to_world for both
                    const f2 dx = add2(add2(mul2(ax, hx, mz), mul2(bx, hy, mz)), mul2(cx, hz, mz));
                    const f2 dy = add2(add2(mul2(ay, hx, mz), mul2(by, hy, mz)), mul2(cy, hz, mz));
                    const f2 dz = add2(add2(mul2(az, hx, mz), mul2(bz, hy, mz)), mul2(cz, hz, mz));
                    const bool v0 = (u0 >> lane) & 1u, v1 = (u1 >> lane) & 1u;
                    if (kSums) {
                        add_fixed40(dx, v0, v1, h0, l0);
                        add_fixed40(dy, v0, v1, h1, l1);
                        add_fixed40(dz, v0, v1, h2, l2);
                        continue;
                    }
                    const f2 on = pack2(v0 ? 1.0f : 0.0f, v1 ? 1.0f : 0.0f);
                    sx = fma2(on, dx, sx);
                    sy = fma2(on, dy, sy);
                    sz = fma2(on, dz, sz);
                    float x0, x1, y0, y1, z0, z1;
                    unpack2(dx, x0, x1);
                    unpack2(dy, y0, y1);
                    unpack2(dz, z0, z1);
                    const bool z0m = fabsf(z0) > fmaxf(fabsf(x0), fabsf(y0)), z1m = fabsf(z1) > fmaxf(fabsf(x1), fabsf(y1));
                    a2 += v0 && z0m;
                    a2 += v1 && z1m;
                    a1 += v0 && !z0m && fabsf(y0) > fabsf(x0);
                    a1 += v1 && !z1m && fabsf(y1) > fabsf(x1);
                }
                if (kSums) {
                    M0 += (long long)(int)(h0 + off) * 4194304LL + (int)(l0 + off);
                    M1 += (long long)(int)(h1 + off) * 4194304LL + (int)(l1 + off);
                    M2 += (long long)(int)(h2 + off) * 4194304LL + (int)(l2 + off);
                }
            }
            cnt = __reduce_add_sync(kAll, cnt);
            if (cnt == 0) continue;                // the lane's initial values
            int dm = 0;
            bool clear = false;
            if (!kSums) {
                a1 = __reduce_add_sync(kAll, a1);
                a2 = __reduce_add_sync(kAll, a2);
                float S[3], t;
                unpack2(sx, S[0], t);
                S[0] += t;
                unpack2(sy, S[1], t);
                S[1] += t;
                unpack2(sz, S[2], t);
                S[2] += t;
                for (int off = 16; off; off >>= 1) {
                    S[0] += __shfl_xor_sync(kAll, S[0], off);
                    S[1] += __shfl_xor_sync(kAll, S[1], off);
                    S[2] += __shfl_xor_sync(kAll, S[2], off);
                }
                const float B = fmaxf(fabsf(b.t1x) + fabsf(b.t2x) + fabsf(nx),
                                      fmaxf(fabsf(b.t1y) + fabsf(b.t2y) + fabsf(ny), fabsf(b.t1z) + fabsf(b.t2z) + fabsf(nz)));
                const float err = 6.3e-8f * B * (float)cnt * (float)(W / 2 + 8);
                const float A0 = fabsf(S[0]), A1 = fabsf(S[1]), A2 = fabsf(S[2]);
                dm = A1 > A0 ? 1 : 0;
                if (A2 > fmaxf(A0, A1)) dm = 2;
                const float first = fmaxf(A0, fmaxf(A1, A2)), second = fmaxf(fminf(A0, A1), fminf(fmaxf(A0, A1), A2));
                clear = first - second > 2.0f * err;
            }
            long long M = 0;
            if (!clear) {
                DirSums e;
                if (kSums) {
                    for (int off = 16; off; off >>= 1) {
                        M0 += __shfl_xor_sync(kAll, M0, off);
                        M1 += __shfl_xor_sync(kAll, M1, off);
                        M2 += __shfl_xor_sync(kAll, M2, off);
                    }
                    e = DirSums{{M0, M1, M2}};
                } else {
                    e = exact_sums(bits, nx, ny, nz, i, W, dirs);
                }
                M0 = e.M[0] < 0 ? -e.M[0] : e.M[0];
                M1 = e.M[1] < 0 ? -e.M[1] : e.M[1];
                M2 = e.M[2] < 0 ? -e.M[2] : e.M[2];
                dm = M1 > M0 ? 1 : 0;
                M = M1 > M0 ? M1 : M0;
                if (M2 > M) {
                    dm = 2;
                    M = M2;
                }
            }
            if (lane == q) {
                my_cnt = cnt;
                my_dm = dm;
                my_axis = dm == 0 ? cnt - a1 - a2 : dm == 1 ? a1 : a2;
                my_M = M;
            }
        }
        if (lane < m) {
            const int64_t i = g * G + lane;
            double cc = 0.0;
            if (my_cnt > 0) {
                if (!kSums)
                    cc = __ddiv_rn((double)my_axis, (double)my_cnt);
                else
                    cc = __ddiv_rn(__ll2double_rn(my_M), __dmul_rn(1099511627776.0, (double)my_cnt));
                loc[S_COUNTED] += 1;
                loc[S_DOM] += my_dm == 0;
                loc[S_DOM + 1] += my_dm == 1;
                loc[S_DOM + 2] += my_dm == 2;
                loc[S_CONC] += llrint(__dmul_rn(cc, 1099511627776.0));
            }
            loc[S_COUNT] += my_cnt;
            if (weight) {
                const double wi = weight[i];
                lwc = __dadd_rn(lwc, __dmul_rn(wi, (double)my_cnt));
                lw = __dadd_rn(lw, wi);
            }
            if (acc) acc[i] = __double2float_rn(__ddiv_rn((double)my_cnt, (double)n_dirs));
            if (dom) dom[i] = (int8_t)my_dm;
            if (conc) conc[i] = __double2float_rn(cc);
        }
    }
    for (int off = 16; off; off >>= 1)
        for (int k = 0; k < S_N; ++k) loc[k] += __shfl_xor_sync(kAll, loc[k], off);
    if (lane == 0)
        for (int k = 0; k < S_N; ++k)
            if (loc[k]) atomicAdd((unsigned long long*)&blk[k], (unsigned long long)loc[k]);
    if (weight) {
        // the lanes' weighted sums in a fixed order
        for (int off = 16; off; off >>= 1) {
            lwc = __dadd_rn(lwc, __shfl_xor_sync(kAll, lwc, off));
            lw = __dadd_rn(lw, __shfl_xor_sync(kAll, lw, off));
        }
        if (lane == 0) {
            wsh[0][threadIdx.x >> 5] = lwc;
            wsh[1][threadIdx.x >> 5] = lw;
        }
    }
    __syncthreads();
    if (threadIdx.x < S_N && blk[threadIdx.x])
        atomicAdd(&sums[threadIdx.x], (unsigned long long)blk[threadIdx.x]);
    if (weight && threadIdx.x == 0) {
        // the block's weighted sums, its warps in order; every block writes
        // its slot (zero when it had no point)
        double a = 0.0, b = 0.0;
        for (int k = 0; k < kVarThreads / 32; ++k) {
            a = __dadd_rn(a, wsh[0][k]);
            b = __dadd_rn(b, wsh[1][k]);
        }
        wpart[blockIdx.x] = a;
        wpart[kVarMaxBlocks + blockIdx.x] = b;
    }
}

// Sum of the blocks' weighted partials in a fixed order: lane l adds blocks
// l, l + 32, ... in turn, then a fixed butterfly over the lanes.  One warp.
__global__ void k_wsum_finish(const double* __restrict__ wpart, int nblocks, double* out /*[2]*/)
{
    const int lane = threadIdx.x;
    double a = 0.0, b = 0.0;
    for (int k = lane; k < nblocks; k += 32) {
        a = __dadd_rn(a, wpart[k]);
        b = __dadd_rn(b, wpart[kVarMaxBlocks + k]);
    }
    for (int off = 16; off; off >>= 1) {
        a = __dadd_rn(a, __shfl_xor_sync(0xFFFFFFFFu, a, off));
        b = __dadd_rn(b, __shfl_xor_sync(0xFFFFFFFFu, b, off));
    }
    if (lane == 0) {
        out[0] = a;
        out[1] = b;
    }
}

// Per-direction visible weight: sum over points where direction j is
// visible of w_i (1 for unit weights).  A block takes a chunk of points, a
// warp a word of the rows at a time, lane = bit.  It was bound by one FP64
// addition per row and word (FP64 issues at 1/64 of the fp32 rate), so the
// points go in fours: their 16 possible sums are formed once per block, and a
// lane looks the sum of its four bits up and adds that (16 doubles, one per
// two banks, so no lookup conflicts).  In a chunk whose weights are all equal
// the lanes count instead, and count times weight is added.  With unit
// weights every sum is an integer below 2^53, so the result is exact in any
// order; with real weights the order of the additions is not fixed (relative
// differences of order 1e-16 between runs).  300k points x 1000 directions,
// with k_variability: 1.41 -> 0.59 ms with equal weights, 0.71 ms with others
// (sums of eight bits, 256 entries: 0.73; 32 words a block, which share the
// table: 0.67 and 0.74).
constexpr int kDirChunk = 512, kDirWords = 8;

__global__ void __launch_bounds__(256)
k_dir_hist(const uint32_t* __restrict__ bits, int64_t n, int W, int n_dirs, const double* __restrict__ weight,
           double* dir_area)
{
    __shared__ double sum4[kDirChunk / 4][16];
    const int64_t i0 = (int64_t)blockIdx.x * kDirChunk;
    const int m = (int)min64(kDirChunk, n - i0), quads = (m + 3) / 4;
    const double first = weight ? weight[i0] : 1.0;
    bool same = true;
    if (weight)
        for (int k = threadIdx.x; k < m; k += blockDim.x) same &= weight[i0 + k] == first;
    const bool equal = __syncthreads_and(same);
    if (!equal) {
        for (int k = threadIdx.x; k < quads * 16; k += blockDim.x) {
            double v = 0.0;
            for (int b = 0; b < 4; ++b) {
                const int at = 4 * (k >> 4) + b;
                if (((k >> b) & 1) && at < m) v = __dadd_rn(v, weight[i0 + at]);
            }
            sum4[k >> 4][k & 15] = v;
        }
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int w = blockIdx.y * kDirWords + (threadIdx.x >> 5);
    if (w < W) {
        const uint32_t* row = bits + i0 * W + w;
        double s = 0.0;
        int cnt = 0;
        if (equal) {
#pragma unroll 8
            for (int q = 0; q < m; ++q) cnt += (__ldg(row + (int64_t)q * W) >> lane) & 1u;
            if (cnt) s = __dmul_rn((double)cnt, first);      // (an infinite weight times no point is no weight)
        } else {
            int q = 0;
#pragma unroll 4
            for (; q < m / 4; ++q) {
                const uint32_t* r = row + (int64_t)4 * q * W;
                const uint32_t a = __ldg(r), b = __ldg(r + W), c = __ldg(r + 2 * (int64_t)W), d = __ldg(r + 3 * (int64_t)W);
                const unsigned k = ((a >> lane) & 1u) | (((b >> lane) & 1u) << 1) | (((c >> lane) & 1u) << 2) |
                                   (((d >> lane) & 1u) << 3);
                s = __dadd_rn(s, sum4[q][k]);
            }
            if (q < quads) {
                unsigned k = 0;
                for (int b = 0; 4 * q + b < m; ++b) k |= ((__ldg(row + (int64_t)(4 * q + b) * W) >> lane) & 1u) << b;
                s = __dadd_rn(s, sum4[q][k]);
            }
        }
        const int j = 32 * w + lane;
        if (s != 0.0 && j < n_dirs) atomicAdd(&dir_area[j], s);
    }
}

// Fixture faces: all three vertices within tol of one frame bounding-box
// plane and the normal pointing out through it to within 1e-6.
__global__ void k_fixture(const float* __restrict__ V, const int32_t* __restrict__ F,
                          const float* __restrict__ fnorm, int64_t T, const double* __restrict__ frame,
                          const double* __restrict__ fbox, uint8_t* fixture)
{
    // the frame's constants once per block: formed by every thread, their
    // FP64 took 16 us for 203k faces where the rest takes 8
    __shared__ double s_tol;
    __shared__ float s_f[9], s_b[6];
    if (threadIdx.x < 9) s_f[threadIdx.x] = (float)frame[threadIdx.x];
    if (threadIdx.x < 6) s_b[threadIdx.x] = (float)fbox[threadIdx.x];
    if (threadIdx.x == 0) {
        const double d0 = __dsub_rn(fbox[3], fbox[0]), d1 = __dsub_rn(fbox[4], fbox[1]), d2 = __dsub_rn(fbox[5], fbox[2]);
        const double diag = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d1, d1)), __dmul_rn(d2, d2)));
        s_tol = __dmul_rn(1e-6, diag);
    }
    __syncthreads();
    const int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (f >= T) return;
    const double tol = s_tol;
    const double lim = 1.0 - 1e-6;
    // fp32 pre-check.  The frame entries are fp32 values, so the fp32 frame
    // coordinate q of a vertex (three rounded operations) is within 3 u s of
    // the exact one, s = sum |V_i f_i|, and the fp32 plane within u |plane|
    // of the FP64 one; a vertex farther than tol + 4 u (s + |plane|) from a
    // plane in fp32 is farther than tol in FP64 (whose own error is far
    // smaller), and the FP64 test of that plane is skipped
    const float u4 = 4.0f * 5.9604644775390625e-8f;
    const float tolf = (float)tol;
    bool fx = false;
    for (int k = 0; k < 3; ++k) {
        const float f0 = s_f[k], f1 = s_f[3 + k], f2 = s_f[6 + k];
        const float blo = s_b[k], bhi = s_b[3 + k];
        bool near_lo = true, near_hi = true;
        for (int a = 0; a < 3; ++a) {
            const int64_t v = F[3 * f + a];
            const float x = V[3 * v], y = V[3 * v + 1], z = V[3 * v + 2];
            const float q = fmaf(x, f0, fmaf(y, f1, z * f2));
            const float sv = (fabsf(x * f0) + fabsf(y * f1) + fabsf(z * f2)) * 1.01f;
            near_lo &= fabsf(q - blo) <= tolf + u4 * (sv + fabsf(blo));
            near_hi &= fabsf(q - bhi) <= tolf + u4 * (sv + fabsf(bhi));
        }
        if (!near_lo && !near_hi) continue;
        bool hi_all = true, lo_all = true;
        for (int a = 0; a < 3; ++a) {
            const int64_t v = F[3 * f + a];
            double q = __dadd_rn(__dmul_rn((double)V[3 * v], frame[k]), __dmul_rn((double)V[3 * v + 1], frame[3 + k]));
            q = __dadd_rn(q, __dmul_rn((double)V[3 * v + 2], frame[6 + k]));
            hi_all &= fabs(__dsub_rn(q, fbox[3 + k])) <= tol;
            lo_all &= fabs(__dsub_rn(q, fbox[k])) <= tol;
        }
        double nq = __dadd_rn(__dmul_rn((double)fnorm[3 * f], frame[k]), __dmul_rn((double)fnorm[3 * f + 1], frame[3 + k]));
        nq = __dadd_rn(nq, __dmul_rn((double)fnorm[3 * f + 2], frame[6 + k]));
        fx |= (hi_all && nq >= lim) || (lo_all && nq <= -lim);
    }
    fixture[f] = fx ? 1 : 0;
}

// Face classes and the 64-bin histogram of viable reachable masks.
__global__ void k_classes(const uint8_t* __restrict__ mask, const float* __restrict__ travel,
                          const int32_t* __restrict__ face, const uint8_t* __restrict__ fixture, int64_t T, int64_t n,
                          float tool_length, uint8_t* cls_out, unsigned long long* hist /*64 + 4*/)
{
    __shared__ unsigned int h[68];
    for (int k = threadIdx.x; k < 68; k += blockDim.x) h[k] = 0;
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const unsigned m = mask[i];
        unsigned reach = 0;
        for (int a = 0; a < 6; ++a)
            if (((m >> a) & 1u) && travel[6 * i + a] <= tool_length) reach |= 1u << a;
        unsigned c = reach ? 0u : (m ? 1u : 2u);
        const int32_t fi = face[i];
        if (fi >= 0 && fi < T && fixture[fi]) c = 3u;
        if (cls_out) cls_out[i] = (uint8_t)c;
        atomicAdd(&h[64 + c], 1u);
        if (c == 0u) atomicAdd(&h[reach], 1u);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < 68; k += blockDim.x)
        if (h[k]) atomicAdd(&hist[k], (unsigned long long)h[k]);
}

// ---------------------------------------------------------------------------
// host drivers
// ---------------------------------------------------------------------------
rc_status launch_variability(const uint32_t* bits, const float* N, const double* weight, int64_t n,
                             const float4* dirs, const rc_params* p, float* acc, int8_t* dom, float* conc,
                             double* dir_area, void* scratch, cudaStream_t s)
{
    const int nd = p->n_dirs;
    unsigned long long* sums = (unsigned long long*)scratch;
    double* wsum = (double*)((char*)scratch + kVarWsumOffset);
    double* wpart = (double*)((char*)scratch + kVarPartOffset);
    RC_CUDA(cudaMemsetAsync(scratch, 0, kVarWsumOffset + 2 * sizeof(double), s));
    if (n > 0) {
        int sm = 0, dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev);
        // points per group: as many as leave every resident warp a group
        // (32 lanes share the quotients' FP64; a small part needs the warps)
        const int W = (nd + 31) / 32;
        const int64_t warps = (int64_t)sm * kVarBlocks * (kVarThreads / 32);
        int G = 1;
        while (G < 32 && (int64_t)2 * G * warps <= n) G *= 2;
        const int64_t groups = (n + G - 1) / G;
        int64_t blocks = std::min<int64_t>((groups + kVarThreads / 32 - 1) / (kVarThreads / 32), (int64_t)sm * kVarBlocks);
        if (blocks > kVarMaxBlocks) blocks = kVarMaxBlocks;
        const bool table = W <= kVarTableWords;
        const auto kernel = p->conc_mode == 0 ? (table ? k_variability<true, false> : k_variability<false, false>)
                                              : (table ? k_variability<true, true> : k_variability<false, true>);
        kernel<<<(unsigned)blocks, kVarThreads, table ? (size_t)((W + 1) / 2) * 32 * 3 * sizeof(float2) : 0, s>>>(
            bits, N, weight, n, dirs, nd, G, acc, dom, conc, sums, wpart);
        RC_LAUNCHED();
        if (weight) {
            k_wsum_finish<<<1, 32, 0, s>>>(wpart, (int)blocks, wsum);
            RC_LAUNCHED();
        }
    }
    if (dir_area) {
        RC_CUDA(cudaMemsetAsync(dir_area, 0, sizeof(double) * (size_t)nd, s));
        const int W = (nd + 31) / 32;
        const int64_t chunks = (n + kDirChunk - 1) / kDirChunk;
        if (chunks > 0) {
            const dim3 grid((unsigned)chunks, (unsigned)((W + kDirWords - 1) / kDirWords));
            k_dir_hist<<<grid, 32 * kDirWords, 0, s>>>(bits, n, W, nd, weight, dir_area);
            RC_LAUNCHED();
        }
    }
    return RC_OK;
}

void fill_summary(const long long* sums, const double* wsum, int64_t n, int32_t n_dirs, bool weighted,
                  rc_summary* out)
{
    rc_summary& o = *out;
    memset(&o, 0, sizeof o);
    const long long counted = sums[S_COUNTED];
    o.n_points = n;
    o.n_counted = counted;
    o.n_zero_visible = n - counted;
    for (int k = 0; k < 3; ++k) {
        o.dom_count[k] = sums[S_DOM + k];
        o.axis_share[k] = counted ? (double)sums[S_DOM + k] / (double)counted : 0.0;
    }
    o.count_sum = sums[S_COUNT];
    o.conc_sum_q = sums[S_CONC];
    if (weighted) {
        o.weighted_count = wsum[0];
        o.weight_sum = wsum[1];
    } else {
        o.weighted_count = (double)sums[S_COUNT];
        o.weight_sum = (double)n;
    }
    const double den = o.weight_sum * (double)n_dirs;
    o.overall_access = den > 0.0 ? o.weighted_count / den : 0.0;
    o.overall_access_unweighted = n ? (double)sums[S_COUNT] / ((double)n * (double)n_dirs) : 0.0;
    o.mean_conc = counted ? (double)sums[S_CONC] / (1099511627776.0 * (double)counted) : 0.0;
}

rc_status launch_classes(rc_bvh h, const uint8_t* mask, const float* travel, const int32_t* face, int64_t n,
                         const rc_params* p, uint8_t* cls, const double* frame_d, const double* fbox_d,
                         uint8_t* fixture, unsigned long long* hist, cudaStream_t s)
{
    k_fixture<<<(unsigned)((h->T + 255) / 256), 256, 0, s>>>(h->V, h->F, h->fnorm, h->T, frame_d, fbox_d, fixture);
    RC_LAUNCHED();
    if (n > 0) {
        int64_t blocks = (n + 255) / 256;
        if (blocks > 1024) blocks = 1024;
        k_classes<<<(unsigned)blocks, 256, 0, s>>>(mask, travel, face, fixture, h->T, n, p->tool_length, cls, hist);
        RC_LAUNCHED();
    }
    return RC_OK;
}

}  // namespace rc
