// cast.cu -- any-hit occlusion traversal (Section 3.1 hemispherical cast,
// Section 3.2 orthogonal cast).
//
// Each ray/triangle pair is first decided in FP32: by signed volumes in the
// pooled hemispherical walk (tri_test_mt), elsewhere with the watertight test
// of Woop, Benthin and Wald (JCGT 2013), together with a forward error bound
// on its edge functions U, V, W, on det = U+V+W and on the unscaled
// plane-crossing value T' = U*az + V*bz + W*cz (see tri_test32).  The FP32
// outcome is accepted only when it is certain -- a clear hit outside the
// 1e-9 relative ambiguity band, or certainly no hit -- otherwise the pair is
// re-decided in FP64 (retest64), which evaluates the occlusion predicate
// directly (signed volumes against each edge, plane crossing N.a / N.d) and
// reports whether the pair lies inside the ambiguity band.  Box tests are
// conservative, so no triangle that can be hit at t > 0 is skipped: the
// 4-wide walk computes each slab distance with one FMA and widens it by a
// proven absolute margin (make_slab_ray), the binary walk scales the far
// distance by 1 + 2*gamma_3 (Ize, JCGT 2013).
//
// Kernels: k_hemisphere (the default cast: persistent warps, one point per
// warp, its rays' walks pooled in shared memory, the last points in parts),
// k_hemisphere_update (re-cast after an edit), k_batch (many parts in one
// launch), k_orthogonal_axis (one frame axis for 32 points per work item),
// k_tool_cast_axis (the sampled ball-end tool), and the frame set-up
// kernels (k_frame_init, k_frame_box).
#include <math.h>

#include <algorithm>

#include "rc_internal.cuh"

namespace rc {

enum { kMiss = 0, kHit = 1, kUnsure = 2 };

struct Ray {
    float ox, oy, oz;
    float dx, dy, dz;
    float ix, iy, iz;   // 1/d (IEEE, +-inf for zero components)
    float Sx, Sy;       // watertight shear
    int kx, ky, kz;     // watertight permutation
    float rs;           // bound on max(1, |o|inf, |vertex|inf)
    float dkz;          // d[kz]
    float ef;           // sheared-coordinate error per unit of max |translated coordinate|
};

__device__ __forceinline__ float sel3(float a, float b, float c, int k)
{
    return k == 0 ? a : (k == 1 ? b : c);
}

__device__ __forceinline__ void setup_ray(Ray& r, float ox, float oy, float oz, float dx, float dy,
                                          float dz, float scene_maxabs)
{
    r.ox = ox; r.oy = oy; r.oz = oz;
    r.dx = dx; r.dy = dy; r.dz = dz;
    // reciprocals; a zero (or tiny) component gets +-2^100 instead of
    // +-inf, so slab products stay finite (no inf * 0 = NaN) and, 2^100
    // being a power of two, exact: such a slab is decided by the sign of
    // b - o alone.  That holds for coordinates up to 2.6e8; beyond, o times
    // 2^100 overflows and the 4-wide walk may miss boxes of such a ray
    r.ix = __frcp_rn(dx);
    r.iy = __frcp_rn(dy);
    r.iz = __frcp_rn(dz);
    if (!(fabsf(r.ix) <= 0x1p100f)) r.ix = copysignf(0x1p100f, dx);
    if (!(fabsf(r.iy) <= 0x1p100f)) r.iy = copysignf(0x1p100f, dy);
    if (!(fabsf(r.iz) <= 0x1p100f)) r.iz = copysignf(0x1p100f, dz);
    const float ax = fabsf(dx), ay = fabsf(dy), az = fabsf(dz);
    int kz = ax >= ay ? (ax >= az ? 0 : 2) : (ay >= az ? 1 : 2);
    int kx = kz == 2 ? 0 : kz + 1;
    int ky = kx == 2 ? 0 : kx + 1;
    const float dk = sel3(dx, dy, dz, kz);
    if (dk < 0.0f) { int t = kx; kx = ky; ky = t; }
    r.kx = kx; r.ky = ky; r.kz = kz;
    r.dkz = dk;
    const float rk = __frcp_rn(dk);
    r.Sx = __fmul_rn(sel3(dx, dy, dz, kx), rk);
    r.Sy = __fmul_rn(sel3(dx, dy, dz, ky), rk);
    // translation rounds once (u|a|); a non-zero shear adds the rounding of
    // S (2u|S||a_z|: reciprocal and product), of a_z (u|S||a_z|) and of the
    // fused subtraction (u|A|); a zero shear leaves the subtraction exact
    const float sm = fmaxf(fabsf(r.Sx), fabsf(r.Sy));
    const float u = 5.9604644775390625e-8f;
    r.ef = sm == 0.0f ? 1.01f * u : (2.0f + 4.0f * sm) * 1.01f * u;
    r.rs = fmaxf(fmaxf(1.0f, scene_maxabs), fmaxf(fabsf(ox), fmaxf(fabsf(oy), fabsf(oz))));
}

// The decision of the watertight test from its edge functions, their error
// bound eU and the vertices' distances along the permuted axis (error model
// below; `extent` is the triangle's largest edge component).  kBand: eU has the
// ambiguity band on top, and a crossing behind the origin must lie beyond its
// band too, so that no pair of the band is called a miss.
template <bool kBand>
__device__ __forceinline__ int tri_decide(const Ray& r, float extent, float U, float V, float W, float eU, float az,
                                          float bz, float cz)
{
    const float u = 5.9604644775390625e-8f;
    const bool uc = fabsf(U) > eU, vc = fabsf(V) > eU, wc = fabsf(W) > eU;
    const bool pos = (uc && U > 0.0f) || (vc && V > 0.0f) || (wc && W > 0.0f);
    const bool neg = (uc && U < 0.0f) || (vc && V < 0.0f) || (wc && W < 0.0f);
    if (pos && neg) return kMiss;

    const float S = fabsf(U) + fabsf(V) + fabsf(W);
    const float det = U + V + W;
    const float Tp = fmaf(U, az, fmaf(V, bz, W * cz));
    const float Zs = fabsf(az) + fabsf(bz) + fabsf(cz);
    const float Zm = fmaxf(fabsf(az), fmaxf(fabsf(bz), fabsf(cz)));
    const float eD = (3.0f * eU + 2.01f * u * S) * 1.0625f;
    const float eT = (eU * Zs + 4.01f * u * S * Zm) * 1.0625f;
    const bool det_ok = fabsf(det) > eD;
    const bool tp_ok = fabsf(Tp) > eT;
    // sign of t = sign(T') * sign(det) * sign(d[kz])
    const bool ahead = ((Tp > 0.0f) == (det > 0.0f)) == (r.dkz > 0.0f);
    // plane crossed behind the origin
    if (det_ok && tp_ok && !ahead && (!kBand || fabsf(Tp) > eT + 1e-9f * r.rs * (fabsf(det) + eD) * 1.01f)) return kMiss;

    // clear hit: every edge function beyond its error and the tau band, and
    // the crossing ahead and beyond tau*R along the ray
    const float tau_edge = 3.0f * 1e-9f * r.rs * extent * 1.01f;
    const float thr = eU + tau_edge;
    if (fabsf(U) > thr && fabsf(V) > thr && fabsf(W) > thr && tp_ok && ahead) {
        const float need = eT + 1e-9f * r.rs * (fabsf(det) + eD) * 1.01f;
        if (fabsf(Tp) > need) return kHit;
    }
    return kUnsure;
}

// FP32 watertight test with a forward error bound.  Returns kHit only when
// the pair is certainly a clear hit (both outside the ambiguity band and
// certain in sign), kMiss only when it is certainly not a hit, else kUnsure.
//
// Error model (u = 2^-24, all translated coordinates |.| <= M, all sheared
// coordinates |.| <= P, S = max(|Sx|,|Sy|) <= 1 because kz is the largest |d|):
//   sheared coordinate error        E  <= (2 + 4 S) u M, and u M when S = 0
//                                        (the fused subtraction is then exact)
//   edge function error             eU <= 4 P E + 6 E^2 + 3 u P^2
//   det error                       eD <= 3 eU + 2.01 u S        (S = sum |U|)
//   plane-crossing error            eT <= eU Zs + 4.01 u S Zm    (Zs = sum |z|, Zm = max |z|)
// each scaled by 1.0625 for the rounding of the bound itself.
__device__ __forceinline__ int tri_test32(const Ray& r, const float4 v0, const float4 v1,
                                          const float4 v2)
{
    const float u = 5.9604644775390625e-8f;
    const float a0 = v0.x - r.ox, a1 = v0.y - r.oy, a2 = v0.z - r.oz;
    const float b0 = v1.x - r.ox, b1 = v1.y - r.oy, b2 = v1.z - r.oz;
    const float c0 = v2.x - r.ox, c1 = v2.y - r.oy, c2 = v2.z - r.oz;
    const float ax = sel3(a0, a1, a2, r.kx), ay = sel3(a0, a1, a2, r.ky), az = sel3(a0, a1, a2, r.kz);
    const float bx = sel3(b0, b1, b2, r.kx), by = sel3(b0, b1, b2, r.ky), bz = sel3(b0, b1, b2, r.kz);
    const float cx = sel3(c0, c1, c2, r.kx), cy = sel3(c0, c1, c2, r.ky), cz = sel3(c0, c1, c2, r.kz);
    const float Ax = fmaf(-r.Sx, az, ax), Ay = fmaf(-r.Sy, az, ay);
    const float Bx = fmaf(-r.Sx, bz, bx), By = fmaf(-r.Sy, bz, by);
    const float Cx = fmaf(-r.Sx, cz, cx), Cy = fmaf(-r.Sy, cz, cy);
    const float U = fmaf(Cx, By, -(Cy * Bx));
    const float V = fmaf(Ax, Cy, -(Ay * Cx));
    const float W = fmaf(Bx, Ay, -(By * Ax));

    const float M = fmaxf(fmaxf(fmaxf(fabsf(a0), fabsf(a1)), fmaxf(fabsf(a2), fabsf(b0))),
                          fmaxf(fmaxf(fabsf(b1), fabsf(b2)), fmaxf(fmaxf(fabsf(c0), fabsf(c1)), fabsf(c2))));
    const float P = fmaxf(fmaxf(fmaxf(fabsf(Ax), fabsf(Ay)), fmaxf(fabsf(Bx), fabsf(By))),
                          fmaxf(fabsf(Cx), fabsf(Cy)));
    const float E = r.ef * M;
    const float eU = (4.0f * E * P + 6.0f * E * E + 3.0f * u * P * P) * 1.0625f;
    return tri_decide<false>(r, v0.w, U, V, W, eU, az, bz, cz);
}

// The same test for a pair that tri_test32 leaves open because the triangle is
// close to the ray but far from its origin: there E is a few u M with M the
// distance to the origin.  Here one vertex is translated and sheared in
// two-term arithmetic (hi + lo; the shear ratio too) and the others follow by
// the sheared edges, so that E scales with the triangle and its distance from
// the ray: E <= 3 u P + (2 + 3 S) u e + 1e-11 M, e the largest edge
// component.  E can be smaller than the ambiguity band here, which is added to
// the bound.  About 150 fp32 operations in place of 75 to 250 in FP64, which
// issue at 1/64 of the rate: the axis rays of a frame search on the turned
// prismatic part left 0.53 pairs per ray open, now 0.002.  With the bands and
// the eligibility test in fp32 too its axis cast went from 2955 to 1310 us,
// and the six axes and the tool in one turned frame from 748 + 1079 to
// 678 + 618 us (100k points).
__device__ __noinline__ int tri_test_close(const Ray& r, const float4 v0, const float4 v1, const float4 v2)
{
    const float u = 5.9604644775390625e-8f;
    const float rk = __frcp_rn(r.dkz);
    const float px = sel3(r.dx, r.dy, r.dz, r.kx), py = sel3(r.dx, r.dy, r.dz, r.ky);
    const float sx = __fmul_rn(px, rk), sy = __fmul_rn(py, rk);
    const float tx = __fmul_rn(__fmaf_rn(-sx, r.dkz, px), rk), ty = __fmul_rn(__fmaf_rn(-sy, r.dkz, py), rk);
    const float ox = sel3(r.ox, r.oy, r.oz, r.kx), oy = sel3(r.ox, r.oy, r.oz, r.ky), oz = sel3(r.ox, r.oy, r.oz, r.kz);
    const float vx = sel3(v0.x, v0.y, v0.z, r.kx), vy = sel3(v0.x, v0.y, v0.z, r.ky), vz = sel3(v0.x, v0.y, v0.z, r.kz);
    // a - b = hi + lo exactly (Knuth)
    const auto diff2 = [](float a, float b, float& hi, float& lo) {
        hi = __fsub_rn(a, b);
        const float t = __fsub_rn(hi, a);
        lo = __fsub_rn(__fsub_rn(a, __fsub_rn(hi, t)), __fadd_rn(b, t));
    };
    float xh, xl, yh, yl, zh, zl;
    diff2(vx, ox, xh, xl);
    diff2(vy, oy, yh, yl);
    diff2(vz, oz, zh, zl);
    // (x - s z) for the two-term x, s, z
    const auto shear2 = [&](float h, float l, float s, float t) {
        const float p = __fmul_rn(s, zh), q = __fadd_rn(__fmaf_rn(s, zh, -p), __fmaf_rn(s, zl, __fmul_rn(t, zh)));
        float dh, dl;
        diff2(h, p, dh, dl);
        return __fadd_rn(dh, __fadd_rn(dl, __fsub_rn(l, q)));
    };
    const float Ax = shear2(xh, xl, sx, tx), Ay = shear2(yh, yl, sy, ty);
    const float bx = sel3(v1.x, v1.y, v1.z, r.kx), by = sel3(v1.x, v1.y, v1.z, r.ky), bz = sel3(v1.x, v1.y, v1.z, r.kz);
    const float cx = sel3(v2.x, v2.y, v2.z, r.kx), cy = sel3(v2.x, v2.y, v2.z, r.ky), cz = sel3(v2.x, v2.y, v2.z, r.kz);
    const float ez = bz - vz, fz = cz - vz;
    const float Bx = Ax + fmaf(-sx, ez, bx - vx), By = Ay + fmaf(-sy, ez, by - vy);
    const float Cx = Ax + fmaf(-sx, fz, cx - vx), Cy = Ay + fmaf(-sy, fz, cy - vy);
    const float U = fmaf(Cx, By, -(Cy * Bx));
    const float V = fmaf(Ax, Cy, -(Ay * Cx));
    const float W = fmaf(Bx, Ay, -(By * Ax));
    const float P = fmaxf(fmaxf(fmaxf(fabsf(Ax), fabsf(Ay)), fmaxf(fabsf(Bx), fabsf(By))), fmaxf(fabsf(Cx), fabsf(Cy)));
    const float S = fmaxf(fabsf(sx), fabsf(sy)), M = fmaxf(fabsf(xh), fmaxf(fabsf(yh), fabsf(zh)));
    const float E = 3.0f * u * P + (2.1f + 3.1f * S) * u * v0.w + 1e-11f * M;
    const float eU = (4.0f * E * P + 6.0f * E * E + 3.0f * u * P * P) * 1.0625f + 3.0f * 1e-9f * r.rs * v0.w * 1.01f + 1e-36f;
    return tri_decide<true>(r, v0.w, U, V, W, eU, zh, bz - oz, cz - oz);
}

// FP64 decision of one pair, written from the definition: the ray's line
// meets the closed triangle iff the signed volumes of the ray direction with
// each edge (relative to the origin) do not take both signs; the plane is
// crossed at t = (N.a)/(N.d).  `state` is kMiss / kHit / kUnsure (= the
// pair lies in the 1e-9 relative ambiguity band); `hit64` is the plain FP64
// sign decision (used for rays that only ambiguous pairs decide).
struct Pair64 { int state; bool hit64; };

// kQuick ends early, after a third of the work, for most pairs; the casts of
// hemisphere rays, which call it 5 times in 10,000, take the form that costs
// their kernels fewer registers (2% of the impeller's time).
template <bool kQuick>
__device__ __forceinline__ Pair64 retest64_of(float ox, float oy, float oz, float dx, float dy, float dz, const float4 v0,
                                        const float4 v1, const float4 v2)
{
    const double o[3] = {ox, oy, oz}, d[3] = {dx, dy, dz};
    const double A[3] = {v0.x, v0.y, v0.z}, B[3] = {v1.x, v1.y, v1.z}, C[3] = {v2.x, v2.y, v2.z};
    double a[3], b[3], c[3], eab[3], ebc[3], eca[3];
    for (int k = 0; k < 3; ++k) {
        a[k] = A[k] - o[k];
        b[k] = B[k] - o[k];
        c[k] = C[k] - o[k];
        eab[k] = B[k] - A[k];
        ebc[k] = C[k] - B[k];
        eca[k] = A[k] - C[k];
    }
    const float Rf = fmaxf(fmaxf(fmaxf(1.0f, fmaxf(fabsf(ox), fmaxf(fabsf(oy), fabsf(oz)))),
                                 fmaxf(fabsf(v0.x), fmaxf(fabsf(v0.y), fabsf(v0.z)))),
                           fmaxf(fmaxf(fabsf(v1.x), fmaxf(fabsf(v1.y), fabsf(v1.z))),
                                 fmaxf(fabsf(v2.x), fmaxf(fabsf(v2.y), fabsf(v2.z)))));
    const double band = kTau * (double)Rf;
    // signed volume of (p, e, d) and |e x d| for the three edges
    const double* P3[3] = {b, c, a};
    const double* E3[3] = {ebc, eca, eab};
    double Ev[3], Lv[3] = {0.0, 0.0, 0.0};
    // (quick: a bound above the band on the volume, band |e x d| <= band
    // |e|_1 |d|_1, in fp32 with 1% to spare; beyond it |e x d| is not needed)
    bool clear[3] = {false, false, false}, posc = false, negc = false;
    if (kQuick) {
        const float l1[3] = {fabsf(v2.x - v1.x) + fabsf(v2.y - v1.y) + fabsf(v2.z - v1.z),
                             fabsf(v0.x - v2.x) + fabsf(v0.y - v2.y) + fabsf(v0.z - v2.z),
                             fabsf(v1.x - v0.x) + fabsf(v1.y - v0.y) + fabsf(v1.z - v0.z)};
        const float wide = 1.01e-9f * Rf * (fabsf(dx) + fabsf(dy) + fabsf(dz));
        for (int k = 0; k < 3; ++k) {
            const double* p = P3[k];
            const double* e = E3[k];
            const double w0 = p[1] * e[2] - p[2] * e[1];
            const double w1 = p[2] * e[0] - p[0] * e[2];
            const double w2 = p[0] * e[1] - p[1] * e[0];
            Ev[k] = w0 * d[0] + w1 * d[1] + w2 * d[2];
            const float f = __double2float_rn(Ev[k]);
            clear[k] = fabsf(f) > wide * l1[k] + 1e-36f;
            posc |= clear[k] && f > 0.0f;
            negc |= clear[k] && f < 0.0f;
        }
        if (posc && negc) return Pair64{kMiss, false};
    }
    for (int k = 0; k < 3; ++k) {
        const double* e = E3[k];
        if (!kQuick) {
            const double* p = P3[k];
            const double w0 = p[1] * e[2] - p[2] * e[1];
            const double w1 = p[2] * e[0] - p[0] * e[2];
            const double w2 = p[0] * e[1] - p[1] * e[0];
            Ev[k] = w0 * d[0] + w1 * d[1] + w2 * d[2];
        }
        if (clear[k]) continue;
        const double x0 = e[1] * d[2] - e[2] * d[1];
        const double x1 = e[2] * d[0] - e[0] * d[2];
        const double x2 = e[0] * d[1] - e[1] * d[0];
        Lv[k] = sqrt(x0 * x0 + x1 * x1 + x2 * x2);
    }
    Pair64 res;
    const bool spos = Ev[0] > 0.0 || Ev[1] > 0.0 || Ev[2] > 0.0;
    const bool sneg = Ev[0] < 0.0 || Ev[1] < 0.0 || Ev[2] < 0.0;
    // N = (B-A) x (C-A) = eab x (-eca)
    const double N0 = -(eab[1] * eca[2] - eab[2] * eca[1]);
    const double N1 = -(eab[2] * eca[0] - eab[0] * eca[2]);
    const double N2 = -(eab[0] * eca[1] - eab[1] * eca[0]);
    const double nd = N0 * d[0] + N1 * d[1] + N2 * d[2];
    const double na = N0 * a[0] + N1 * a[1] + N2 * a[2];
    res.hit64 = !(spos && sneg) && nd != 0.0 && na != 0.0 && ((na > 0.0) == (nd > 0.0));

    bool pos = posc, neg = negc, small = false;
    for (int k = 0; k < 3; ++k) {
        if (clear[k]) continue;
        if (fabs(Ev[k]) <= band * Lv[k]) { small = true; continue; }
        if (Ev[k] > 0.0) pos = true; else neg = true;
    }
    if (pos && neg) { res.state = kMiss; return res; }
    if (nd == 0.0) { res.state = small ? kUnsure : kMiss; return res; }
    const double dn = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    if (fabs(na) * dn <= band * fabs(nd)) { res.state = kUnsure; return res; }
    if ((na > 0.0) != (nd > 0.0)) { res.state = kMiss; return res; }
    res.state = small ? kUnsure : kHit;
    return res;
}

template <bool kQuick>
__device__ __noinline__ Pair64 retest64(float ox, float oy, float oz, float dx, float dy, float dz, const float4 v0,
                                        const float4 v1, const float4 v2)
{
    return retest64_of<kQuick>(ox, oy, oz, dx, dy, dz, v0, v1, v2);
}

// of a ray by itself in its lane: passed by reference (its six values in
// registers cost the walk around the call more spills: binary walk, housing,
// 20k points x 1024 directions, 2.45 ms, 2.70 by value and quick)
__device__ __noinline__ Pair64 retest64(const Ray& r, const float4 v0, const float4 v1, const float4 v2)
{
    return retest64_of<false>(r.ox, r.oy, r.oz, r.dx, r.dy, r.dz, v0, v1, v2);
}

// Conservative slab test of both children of a packed node.
__device__ __forceinline__ void box2(const Ray& r, const float4 n0, const float4 n1, const float4 n2,
                                     bool& h0, bool& h1, float& t0, float& t1)
{
    const float rob = 1.0f + 2.0f * 1.7881394e-7f;   // 1 + 2*gamma_3, gamma_3 = 3u/(1-3u)
    const bool sx = signbit(r.ix), sy = signbit(r.iy), sz = signbit(r.iz);
    // child 0: (n0.x lo_x, n0.y hi_x, n0.z lo_y, n0.w hi_y, n2.x lo_z, n2.y hi_z)
    float nx = ((sx ? n0.y : n0.x) - r.ox) * r.ix, fx = ((sx ? n0.x : n0.y) - r.ox) * r.ix;
    float ny = ((sy ? n0.w : n0.z) - r.oy) * r.iy, fy = ((sy ? n0.z : n0.w) - r.oy) * r.iy;
    float nz = ((sz ? n2.y : n2.x) - r.oz) * r.iz, fz = ((sz ? n2.x : n2.y) - r.oz) * r.iz;
    float tn = fmaxf(fmaxf(nx, ny), fmaxf(nz, 0.0f));
    float tf = fminf(fminf(fx, fy), fz) * rob;
    h0 = tn <= tf;
    t0 = tn;
    // child 1: (n1.x lo_x, n1.y hi_x, n1.z lo_y, n1.w hi_y, n2.z lo_z, n2.w hi_z)
    nx = ((sx ? n1.y : n1.x) - r.ox) * r.ix; fx = ((sx ? n1.x : n1.y) - r.ox) * r.ix;
    ny = ((sy ? n1.w : n1.z) - r.oy) * r.iy; fy = ((sy ? n1.z : n1.w) - r.oy) * r.iy;
    nz = ((sz ? n2.w : n2.z) - r.oz) * r.iz; fz = ((sz ? n2.z : n2.w) - r.oz) * r.iz;
    tn = fmaxf(fmaxf(nx, ny), fmaxf(nz, 0.0f));
    tf = fminf(fminf(fx, fy), fz) * rob;
    h1 = tn <= tf;
    t1 = tn;
}

// Per-warp-lane counters of a cast.
struct CastAccFwd {
    int amb = 0, retests = 0, overflow = 0;
    long long rays = 0, nvis = 0, ntri = 0, nbox = 0;
};

// Result bits of trace(): bit 0 blocked, bit 1 decided by ambiguous pairs.
// With kStats the walk also counts interior-node fetches and triangle tests
// (the instrumented build used to measure algorithmic bytes per ray).
struct TraceOut { int flags; int retests; int overflow; int nodes; int tris; };

template <bool kStats>
__device__ __forceinline__ TraceOut trace(const float4* __restrict__ nodes, const float4* __restrict__ tris,
                                          const Ray& r, int max_steps)
{
    TraceOut out = {0, 0, 0, 0, 0};
    int stack[kStack];
    int sp = 0;
    int cur = 0;
    bool amb = false, ambhit = false;
    // a well-formed tree visits each node at most once, so max_steps (the
    // node count) is never reached; the cap only bounds a malformed tree
    for (int steps = 0;; ++steps) {
        if (steps > max_steps) { out.overflow = 1; out.flags = 1; return out; }
        if (cur >= 0) {
            if (kStats) ++out.nodes;
            const float4 n0 = __ldg(&nodes[4 * cur + 0]);
            const float4 n1 = __ldg(&nodes[4 * cur + 1]);
            const float4 n2 = __ldg(&nodes[4 * cur + 2]);
            const float4 n3 = __ldg(&nodes[4 * cur + 3]);
            bool h0, h1;
            float t0, t1;
            box2(r, n0, n1, n2, h0, h1, t0, t1);
            const int c0 = __float_as_int(n3.x), c1 = __float_as_int(n3.y);
            if (h0 && h1) {
                const bool first0 = t0 <= t1;
                if (sp >= kStack) { out.overflow = 1; out.flags = 1; return out; }
                stack[sp++] = first0 ? c1 : c0;
                cur = first0 ? c0 : c1;
                continue;
            }
            if (h0) { cur = c0; continue; }
            if (h1) { cur = c1; continue; }
        } else {
            const int first = leaf_first(cur), cnt = leaf_count(cur);
            for (int k = 0; k < cnt; ++k) {
                const float4* t = tris + 3 * (first + k);
                const float4 v0 = __ldg(t), v1 = __ldg(t + 1), v2 = __ldg(t + 2);
                if (kStats) ++out.tris;
                const int s = tri_test32(r, v0, v1, v2);
                if (s == kHit) { out.flags = 1; return out; }
                if (s == kUnsure) {
                    ++out.retests;
                    const Pair64 p = retest64(r, v0, v1, v2);
                    if (p.state == kHit) { out.flags = 1; return out; }
                    if (p.state == kUnsure) { amb = true; ambhit |= p.hit64; }
                }
            }
        }
        if (sp == 0) break;
        cur = stack[--sp];
    }
    out.flags = (ambhit ? 1 : 0) | (amb ? 2 : 0);
    return out;
}

// Per-ray constants of the 4-wide slab test.  A slab distance is one FMA,
// t = b * i - o * i, with the near / far bound of each axis picked by the
// load address (the node stores lo and hi of an axis in adjacent float4s).
// Conservative: with u = 2^-24, i = fl(1/d), M >= |every box coordinate|,
// the computed b*i - fl(o*i) differs from (b - o)/d by at most
// 2u|t| + 2u|o i| (+ lower-order terms) <= 4.01 u (M + |o|) |i|; every near
// distance is lowered and every far distance raised by E = 5 u (M + |o|) |i|
// (folded into the subtracted constant, its rounding included), so a box
// the exact ray enters is never rejected.  An axis with i = +-2^100 (the
// direction has no component along it) needs no margin: see setup_ray.
struct SlabRay {
    float ix, iy, iz;
    float nox, noy, noz;    // o * i + E  (subtracted for near distances)
    float fox, foy, foz;    // o * i - E  (subtracted for far distances)
    int offx, offy, offz;   // 1 when the axis runs backwards: near = hi
};

__device__ __forceinline__ SlabRay make_slab_ray(const Ray& r, float M)
{
    const float u = 5.9604644775390625e-8f;
    SlabRay s;
    s.ix = r.ix; s.iy = r.iy; s.iz = r.iz;
    // a +-2^100 reciprocal (axis parallel to the slab) makes b*i and o*i
    // exact, so only the sign-preserving final rounding remains: no margin
    const float ex = fabsf(r.ix) == 0x1p100f ? 0.0f : 5.0f * u * ((M + fabsf(r.ox)) * fabsf(r.ix));
    const float ey = fabsf(r.iy) == 0x1p100f ? 0.0f : 5.0f * u * ((M + fabsf(r.oy)) * fabsf(r.iy));
    const float ez = fabsf(r.iz) == 0x1p100f ? 0.0f : 5.0f * u * ((M + fabsf(r.oz)) * fabsf(r.iz));
    const float oix = r.ox * r.ix, oiy = r.oy * r.iy, oiz = r.oz * r.iz;
    s.nox = oix + ex; s.noy = oiy + ey; s.noz = oiz + ez;
    s.fox = oix - ex; s.foy = oiy - ey; s.foz = oiz - ez;
    s.offx = signbit(r.ix) ? 1 : 0;
    s.offy = signbit(r.iy) ? 1 : 0;
    s.offz = signbit(r.iz) ? 1 : 0;
    return s;
}

// Where wide node w's float4s start to be read, and float4 c of it: trees are
// allocated on 256-byte boundaries, so wide_at is one exclusive or on the
// address.
__device__ __forceinline__ const float4* wide_ptr(const float4* __restrict__ tree, int w)
{
    return (const float4*)((const char*)tree + (((size_t)(unsigned)w << 7) | (((unsigned)w & 7u) << 4)));
}
__device__ __forceinline__ float4 wide_ld(const float4* nd, int c)
{
    return __ldg((const float4*)((uintptr_t)nd ^ (uintptr_t)(c << 4)));
}

// Slab test of the four children of wide node w: d[k] = entry distance of a
// hit child (else +inf), c[k] = child index; returns the number of hits.
__device__ __forceinline__ int slab4(const float4* __restrict__ wnodes, int w, const SlabRay& s, float d[4], int c[4])
{
    const float4* nd = wide_ptr(wnodes, w);
    const float4 nxv = wide_ld(nd, s.offx), fxv = wide_ld(nd, 1 - s.offx);
    const float4 nyv = wide_ld(nd, 2 + s.offy), fyv = wide_ld(nd, 3 - s.offy);
    const float4 nzv = wide_ld(nd, 4 + s.offz), fzv = wide_ld(nd, 5 - s.offz);
    const float4 ci = wide_ld(nd, 6);
    const float nx[4] = {nxv.x, nxv.y, nxv.z, nxv.w}, fx[4] = {fxv.x, fxv.y, fxv.z, fxv.w};
    const float ny[4] = {nyv.x, nyv.y, nyv.z, nyv.w}, fy[4] = {fyv.x, fyv.y, fyv.z, fyv.w};
    const float nz[4] = {nzv.x, nzv.y, nzv.z, nzv.w}, fz[4] = {fzv.x, fzv.y, fzv.z, fzv.w};
    const int cc[4] = {__float_as_int(ci.x), __float_as_int(ci.y), __float_as_int(ci.z), __float_as_int(ci.w)};
    int nh = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float tn = fmaxf(fmaxf(fmaf(nx[k], s.ix, -s.nox), fmaf(ny[k], s.iy, -s.noy)),
                               fmaxf(fmaf(nz[k], s.iz, -s.noz), 0.0f));
        const float tf = fminf(fminf(fmaf(fx[k], s.ix, -s.fox), fmaf(fy[k], s.iy, -s.foy)),
                               fmaf(fz[k], s.iz, -s.foz));
        const bool hit = tn <= tf;
        d[k] = hit ? tn : INFINITY;
        c[k] = cc[k];
        nh += hit;
    }
    return nh;
}

// ---------------------------------------------------------------------------
// Per-point frontier of the 4-wide walk.  All hemisphere rays of a point
// start at the same origin o, and a box that contains o is entered by every
// one of them: its near slab distances are <= 0 and its far ones >= 0, and
// the conservative margin only lowers the near and raises the far ones.  So
// every ray's walk from the root visits the same nodes whose boxes contain o
// (the origin set: the root and every child box containing o below it).
// The warp finds that set once per point and keeps in shared memory what
// each ray must still decide for itself: the triangles of the leaves whose
// boxes contain o (local triangles), and the children of origin-set nodes
// whose boxes do not contain o (the frontier).  A ray tests the local
// triangles, tests the frontier boxes with its own slab test and walks the
// subtrees it enters: the triangles its walk from the root would test, so
// the same decisions.  A local triangle wholly below the point's tangent
// plane is dropped, because a hemisphere ray leaves that plane (d.n > 0 for
// every direction of the set, N <= 65536, when n is of unit length to within
// the rounding of an fp32 normal) and meets no point of it at t > 0; that
// test runs once per point, in fp32 where its sign is clear and in FP64
// otherwise.  For the same reason a frontier box
// wholly below the plane is dropped, and so is a frontier leaf whose
// triangles all lie below it (conservative fp32 tests).  Large boxes then
// make way for their children's while there is room (see build_frontier),
// and the boxes are sorted by distance.  What finds no room stays whole, as
// a frontier box that every ray enters.
// ---------------------------------------------------------------------------
// 64 boxes: of the impeller's points 1 in 800 has more.  96 and 128 measured
// within 2% of 64 (fewer walk steps, less L1 left beside the shared memory).
constexpr int kFrontEntries = 64;                // frontier boxes kept per point
constexpr int kFrontTris = 8;                    // local triangles kept per point
constexpr int kFrontRounds = 8;                  // most rounds of growth, eight boxes each
constexpr int kFrontWords = kFrontEntries / 32;  // boxes per lane
static_assert(kFrontEntries % 32 == 0 && kFrontEntries <= 128, "a lane looks at whole words of boxes; a list of bytes");

struct Frontier {
    float4 box[2 * kFrontEntries]; // per entry: lo xyz and its code, hi xyz
    float4 tri[kFrontTris * 3];    // local triangle records
    int nboxes, ntris, nvis;
};

// n . (v - o) < 0 for the three vertices, in FP64: the differences of fp32
// values are exact there and the products and sums round far below the
// margin taken (4e-15 of the sum of the terms' magnitudes)
__device__ __noinline__ bool below_tangent64(float x, float y, float z, float ox, float oy, float oz, float nx, float ny, float nz)
{
    const double a = (double)x - ox, b = (double)y - oy, c = (double)z - oz;
    const double s = __dadd_rn(__dadd_rn(__dmul_rn((double)nx, a), __dmul_rn((double)ny, b)), __dmul_rn((double)nz, c));
    const double m = fabs((double)nx * a) + fabs((double)ny * b) + fabs((double)nz * c);
    return s < -4e-15 * m;
}

// the same, decided in fp32 where the sign is clear (each difference, product
// and sum rounds once: under 4u of the sum of the terms' magnitudes, 8u taken)
__device__ __forceinline__ bool below_tangent(float4 v, float ox, float oy, float oz, float nx, float ny, float nz)
{
    const float a = (v.x - ox) * nx, b = (v.y - oy) * ny, c = (v.z - oz) * nz;
    const float s = a + b + c, e = 8.0f * 5.9604644775390625e-8f * (fabsf(a) + fabsf(b) + fabsf(c)) + 1e-36f;
    if (fabsf(s) > e && e < 1e30f) return s < 0.0f;
    return below_tangent64(v.x, v.y, v.z, ox, oy, oz, nx, ny, nz);
}

// Shortcuts that skip what lies below a point's tangent plane need every
// direction of the set above it.  With |n|^2 = 1 + delta the basis tilts by
// about |delta|, so d.n >= z_min - 3 |delta| - 1e-6 with z_min = 1/(2N) >=
// 1/(64 W) (W = ceil(N/32)); a normal further from unit length takes none.
// In fp32 where the comparison is clear by 1e-6 (rounding: 3u nn and less).
__device__ __noinline__ bool tangent_shortcuts_ok64(float nx, float ny, float nz, int W)
{
    const double nn = (double)nx * nx + (double)ny * ny + (double)nz * nz;
    return fabs(nn - 1.0) <= 0.25 * (1.0 / (64.0 * W) - 2e-6);
}

__device__ __forceinline__ bool tangent_shortcuts_ok(float nx, float ny, float nz, int W)
{
    const float off = fabsf(nx * nx + ny * ny + nz * nz - 1.0f) - (__fdividef(0.25f, 64.0f * (float)W) - 5e-7f);
    if (fabsf(off) > 1e-6f && off < 1.0f) return off < 0.0f;
    return tangent_shortcuts_ok64(nx, ny, nz, W);
}

// A box wholly below the tangent plane through o: the largest n.(x - o) over
// its corners, sum over the axes of max(n_k (lo_k - o_k), n_k (hi_k - o_k)),
// is negative beyond the rounding of its fp32 evaluation (each difference,
// product and sum rounds once: under 4u of the sum of the terms' magnitudes,
// 8u taken).  Every triangle inside such a box is wholly below the plane too.
__device__ __forceinline__ bool box_below_tangent(float lx, float hx, float ly, float hy, float lz, float hz,
                                                  float ox, float oy, float oz, float nx, float ny, float nz)
{
    const float mx = fmaxf(nx * (lx - ox), nx * (hx - ox));
    const float my = fmaxf(ny * (ly - oy), ny * (hy - oy));
    const float mz = fmaxf(nz * (lz - oz), nz * (hz - oz));
    const float u = 5.9604644775390625e-8f;
    return (mx + my) + mz < -8.0f * u * (fabsf(mx) + fabsf(my) + fabsf(mz));
}

// Component c (0..5: lo.x, hi.x, lo.y, hi.y, lo.z, hi.z; 6: code) of child k
// of a wide node.
__device__ __forceinline__ float child_ld(const float4* __restrict__ wnodes, int w, int c, int k)
{
    return __ldg((const float*)(wnodes + wide_at(w, c)) + k);
}

// The warp builds the point's frontier: the origin set of o (the nodes whose
// boxes contain o) is walked level by level, up to eight nodes at a time, a
// lane per child; `queue` (shared, kFrontQueue ints) holds the nodes visited
// and to be visited.  A node or leaf for which there is no room stays whole:
// a frontier box that every ray enters.
constexpr int kFrontQueue = 256;

__device__ __noinline__ void build_frontier(const float4* __restrict__ wnodes, const float4* __restrict__ tris,
                                            float ox, float oy, float oz, float nx, float ny, float nz, bool drop,
                                            float theta2, int rounds, Frontier* f, int* queue)
{
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    int head = 0, tail = 1, ne = 0, nt = 0;
    if (lane == 0) queue[0] = 0;
    __syncwarp();
    while (head < tail && tail + 32 <= kFrontQueue) {
        const int m = min(8, tail - head), k = lane & 3;
        const bool on = (lane >> 2) < m;
        const int nd = queue[on ? head + (lane >> 2) : head];
        const float lx = child_ld(wnodes, nd, 0, k), hx = child_ld(wnodes, nd, 1, k), ly = child_ld(wnodes, nd, 2, k);
        const float hy = child_ld(wnodes, nd, 3, k), lz = child_ld(wnodes, nd, 4, k), hz = child_ld(wnodes, nd, 5, k);
        const int code = __float_as_int(child_ld(wnodes, nd, 6, k));
        head += m;
        const bool box = on && lx <= hx;   // an empty slot has an empty box (its code -1 is also a leaf's)
        const bool in = box && lx <= ox && ox <= hx && ly <= oy && oy <= hy && lz <= oz && oz <= hz;
        bool out = box && !in;
        // a box below the tangent plane holds no hit of any ray of the point
        if (out && drop && box_below_tangent(lx, hx, ly, hy, lz, hz, ox, oy, oz, nx, ny, nz)) out = false;
        // leaves: a triangle of one that contains o becomes a local triangle
        // unless it lies below the plane; one that does not is dropped
        // when all its triangles do (fp32)
        const int first = leaf_first(code), cnt = box && code < 0 && (in || (out && drop)) ? leaf_count(code) : 0;
        bool above = !(out && drop && code < 0);
        const int nt0 = nt;
        for (int q = 0; __any_sync(kAll, q < cnt); ++q) {
            bool keep = false;
            float4 v0, v1, v2;
            if (q < cnt) {
                const float4* tp = tris + 3 * (int64_t)(first + q);
                v0 = __ldg(tp);
                v1 = __ldg(tp + 1);
                v2 = __ldg(tp + 2);
                if (in)
                    keep = !(drop && below_tangent(v0, ox, oy, oz, nx, ny, nz) &&
                             below_tangent(v1, ox, oy, oz, nx, ny, nz) && below_tangent(v2, ox, oy, oz, nx, ny, nz));
                else
                    above |= !(box_below_tangent(v0.x, v0.x, v0.y, v0.y, v0.z, v0.z, ox, oy, oz, nx, ny, nz) &&
                               box_below_tangent(v1.x, v1.x, v1.y, v1.y, v1.z, v1.z, ox, oy, oz, nx, ny, nz) &&
                               box_below_tangent(v2.x, v2.x, v2.y, v2.y, v2.z, v2.z, ox, oy, oz, nx, ny, nz));
            }
            const unsigned mt = __ballot_sync(kAll, keep);
            if (keep && nt + __popc(mt & below) < kFrontTris) {
                const int at = 3 * (nt + __popc(mt & below));
                f->tri[at] = v0;
                f->tri[at + 1] = v1;
                f->tri[at + 2] = v2;
            }
            nt += __popc(mt);
        }
        // no room for their triangles: these leaves stay whole, as boxes
        // that every ray enters
        const bool whole_leaf = nt > kFrontTris && in && code < 0;
        if (nt > kFrontTris) nt = nt0;
        const unsigned mq = __ballot_sync(kAll, in && code >= 0);
        const bool entry = (out && above) || whole_leaf;
        const unsigned me = __ballot_sync(kAll, entry);
        if (ne + __popc(me) + (tail - head) + __popc(mq) > kFrontEntries) {
            // no room: these nodes stay whole, and so do those still queued
            nt = nt0;
            head -= m;
            break;
        }
        if (in && code >= 0) queue[tail + __popc(mq & below)] = code;
        tail += __popc(mq);
        if (entry) {
            const int at = 2 * (ne + __popc(me & below));
            f->box[at] = make_float4(lx, ly, lz, __int_as_float(code));
            f->box[at + 1] = make_float4(hx, hy, hz, 0.0f);
        }
        ne += __popc(me);
        __syncwarp();
    }
    const int visited = head;
    for (; head < tail; head += 32) {
        if (lane < tail - head) {
            const int at = 2 * (ne + lane);
            f->box[at] = make_float4(-INFINITY, -INFINITY, -INFINITY, __int_as_float(queue[head + lane]));
            f->box[at + 1] = make_float4(INFINITY, INFINITY, INFINITY, 0.0f);
        }
        ne += min(32, tail - head);
    }
    __syncwarp();
    // Boxes that look large from o make way for their children's while there
    // is room.  Testing a tile's rays against a box costs about as much as
    // three (ray, node) pairs of the walk, and a tile first drops the boxes
    // it cannot meet, so a box is worth it down to the angle at which each of
    // its children is met by a few rays (theta2 = 20 / N steradian; the room
    // runs out first nearly always).  A round costs a point about what a
    // tenth of a tile does, hence the fewer rounds the fewer tiles.  Measured
    // (100k points): impeller 35.4 -> 32.4 ms, housing 6.72 -> 6.11 ms at
    // 2048 and 1024 directions; with 8 rounds at 150 directions 2.91 -> 3.31.
    int grown = 0;
    for (int round = 0; round < rounds && kFrontEntries - ne >= 3; ++round) {
        float r[kFrontWords], most = 0.0f;
#pragma unroll
        for (int q = 0; q < kFrontWords; ++q) {
            const int e = 32 * q + lane;
            r[q] = 0.0f;
            if (e < ne) {
                const float4 lo = f->box[2 * e], hi = f->box[2 * e + 1];
                const float dx = fmaxf(fmaxf(lo.x - ox, ox - hi.x), 0.0f), dy = fmaxf(fmaxf(lo.y - oy, oy - hi.y), 0.0f),
                            dz = fmaxf(fmaxf(lo.z - oz, oz - hi.z), 0.0f);
                const float ext = fmaxf(hi.x - lo.x, fmaxf(hi.y - lo.y, hi.z - lo.z));
                if (__float_as_int(lo.w) >= 0 && ext > 0.0f && ext < INFINITY)
                    r[q] = ext * ext / (dx * dx + dy * dy + dz * dz + 1e-30f);
            }
            most = fmaxf(most, r[q]);
        }
        most = warp_max(most);
        const float least = fmaxf(theta2, 0.25f * most);
        const int room = min(8, (kFrontEntries - ne) / 3);
        int m = 0;
#pragma unroll
        for (int q = 0; q < kFrontWords; ++q) {
            const unsigned b = __ballot_sync(kAll, r[q] > least);
            const int at = m + __popc(b & below);
            if (r[q] > least && at < room) queue[at] = 32 * q + lane;
            m += __popc(b);
        }
        m = min(m, room);
        if (m == 0) break;
        __syncwarp();
        const int k = lane & 3;
        const bool on = (lane >> 2) < m;
        const int nd = __float_as_int(f->box[2 * queue[on ? lane >> 2 : 0]].w);
        const float lx = child_ld(wnodes, nd, 0, k), hx = child_ld(wnodes, nd, 1, k), ly = child_ld(wnodes, nd, 2, k);
        const float hy = child_ld(wnodes, nd, 3, k), lz = child_ld(wnodes, nd, 4, k), hz = child_ld(wnodes, nd, 5, k);
        const int code = __float_as_int(child_ld(wnodes, nd, 6, k));
        const bool keep = on && lx <= hx &&
                          !(drop && box_below_tangent(lx, hx, ly, hy, lz, hz, ox, oy, oz, nx, ny, nz));
        const unsigned mk = __ballot_sync(kAll, keep);
        __syncwarp();
        // the children take their parents' places, then new ones; a place
        // left over holds a box that no ray meets
        const int rank = __popc(mk & below), at = rank < m ? queue[rank] : ne + rank - m;
        const int spare = lane >= __popc(mk) && lane < m ? queue[lane] : -1;
        __syncwarp();
        if (keep) {
            f->box[2 * at] = make_float4(lx, ly, lz, __int_as_float(code));
            f->box[2 * at + 1] = make_float4(hx, hy, hz, 0.0f);
        }
        if (spare >= 0) {
            f->box[2 * spare] = make_float4(1e30f, 1e30f, 1e30f, __int_as_float(-1));
            f->box[2 * spare + 1] = make_float4(-1e30f, -1e30f, -1e30f, 0.0f);
        }
        ne += max(0, __popc(mk) - m);
        grown += m;
        __syncwarp();
    }
    if (grown) {
        // nearest last: the boxes are tested from the end (in the order of
        // growth the impeller took 40.1 ms instead of 32.4, farthest first 59)
        float* key = (float*)queue;
        float4 lo[kFrontWords], hi[kFrontWords];
        float d[kFrontWords];
        int at[kFrontWords];
#pragma unroll
        for (int q = 0; q < kFrontWords; ++q) {
            const int e = 32 * q + lane;
            at[q] = 0;
            d[q] = 0.0f;
            if (e < ne) {
                lo[q] = f->box[2 * e];
                hi[q] = f->box[2 * e + 1];
                const float dx = fmaxf(fmaxf(lo[q].x - ox, ox - hi[q].x), 0.0f),
                            dy = fmaxf(fmaxf(lo[q].y - oy, oy - hi[q].y), 0.0f),
                            dz = fmaxf(fmaxf(lo[q].z - oz, oz - hi[q].z), 0.0f);
                d[q] = dx * dx + dy * dy + dz * dz;
                key[e] = d[q];
            }
        }
        __syncwarp();
        for (int e = 0; e < ne; ++e) {
            const float k = key[e];
#pragma unroll
            for (int q = 0; q < kFrontWords; ++q) at[q] += k > d[q] || (k == d[q] && e < 32 * q + lane);
        }
#pragma unroll
        for (int q = 0; q < kFrontWords; ++q)
            if (32 * q + lane < ne) {
                f->box[2 * at[q]] = lo[q];
                f->box[2 * at[q] + 1] = hi[q];
            }
        __syncwarp();
    }
    if (lane == 0) {
        f->nboxes = ne;
        f->ntris = nt;
        f->nvis = visited + grown;
    }
    __syncwarp();
}

// Any-hit walk of the 4-wide tree by one lane, with its stack in local memory:
// the same ray, box and triangle decisions as trace(); per node the four child
// boxes are tested together, the nearest hit child is visited next and the
// others are pushed partly ordered.
template <bool kStats>
__device__ __forceinline__ TraceOut trace4(const float4* __restrict__ wnodes, const float4* __restrict__ tris,
                                           const Ray& r, int max_steps)
{
    TraceOut out = {0, 0, 0, 0, 0};
    int stack[kStack4];
    int sp = 0;
    int cur = 0;
    bool amb = false, ambhit = false;
    const SlabRay sr = make_slab_ray(r, r.rs);
    for (int steps = 0;; ++steps) {
        if (steps > max_steps) { out.overflow = 1; out.flags = 1; return out; }
        if (cur >= 0) {
            if (kStats) ++out.nodes;
            float d[4];
            int c[4];
            const int nh = slab4(wnodes, cur, sr, d, c);
            if (nh == 0) {
                if (sp == 0) break;
                cur = stack[--sp];
                continue;
            }
#define RC_CSWAP(a, b)                                              \
    if (d[b] < d[a]) {                                              \
        const float td = d[a]; d[a] = d[b]; d[b] = td;              \
        const int tc = c[a]; c[a] = c[b]; c[b] = tc;                \
    }
            // three of the five exchanges of the sorting network: the nearest
            // child reaches slot 0 and the others stay partly ordered (faster
            // than the full network, and no more nodes visited)
            RC_CSWAP(0, 1) RC_CSWAP(2, 3) RC_CSWAP(0, 2)
#undef RC_CSWAP
            if (sp + nh - 1 > kStack4) { out.overflow = 1; out.flags = 1; return out; }
            if (d[3] != INFINITY) stack[sp++] = c[3];
            if (d[2] != INFINITY) stack[sp++] = c[2];
            if (d[1] != INFINITY) stack[sp++] = c[1];
            cur = c[0];
            continue;
        } else {
            const int first = leaf_first(cur), cnt = leaf_count(cur);
            for (int k = 0; k < cnt; ++k) {
                const float4* t = tris + 3 * (first + k);
                const float4 v0 = __ldg(t), v1 = __ldg(t + 1), v2 = __ldg(t + 2);
                if (kStats) ++out.tris;
                const int s = tri_test32(r, v0, v1, v2);
                if (s == kHit) { out.flags = 1; return out; }
                if (s == kUnsure) {
                    ++out.retests;
                    const Pair64 p = retest64(r, v0, v1, v2);
                    if (p.state == kHit) { out.flags = 1; return out; }
                    if (p.state == kUnsure) { amb = true; ambhit |= p.hit64; }
                }
            }
        }
        if (sp == 0) break;
        cur = stack[--sp];
    }
    out.flags = (ambhit ? 1 : 0) | (amb ? 2 : 0);
    return out;
}

template <bool kStats, bool kWide>
__device__ __forceinline__ TraceOut trace_any(const float4* __restrict__ nodes, const float4* __restrict__ tris,
                                              const Ray& r, int max_steps)
{
    if (kWide) return trace4<kStats>(nodes, tris, r, max_steps);
    return trace<kStats>(nodes, tris, r, max_steps);
}

// ---------------------------------------------------------------------------
// Axis rays (Section 3.2: rays along the six principal directions of the
// machining frame).  Their walk tests the child boxes of the frame's own tree
// (the same nodes with boxes in frame coordinates, FrameDev::tree) and the
// triangles in world coordinates, exactly as the hemispherical walk does.
// A ray o + t d, d = +-column k of the fp32 frame F, has frame coordinates
// q(o) + t F^T d = q(o) +- t G[:, k] (G = F^T F): along k they grow (shrink)
// with t, and across k they drift by at most t |G[j][k]|, a few ulps times
// t for an fp32 frame.  Every hit lies in the part's box, so t is at most
// (|o - c| + r) / |d| (c, r: the box's centre and half diagonal).  The ray
// can therefore only meet triangles whose frame boxes overlap the band
// [q_j(o) - tol_j, q_j(o) + tol_j] across k and lie on its side of q_k(o)
// along k, where tol_j covers that drift, the 1e-9 R ambiguity band and the
// FP64 rounding of q and of the boxes; the band is rounded outward to fp32.
// For the identity frame the drift is zero and the tree is the world tree.
// A ray along a wall 1e-4 mm above it, which the world boxes of a turned
// part's wall triangles all admit, lies outside their frame boxes.
// ---------------------------------------------------------------------------
struct AxisRay {
    float lo[3], hi[3];   // frame-coordinate band the ray can reach (+-inf on its far side along k)
};

// The band of an axis ray (see above).  Its bounds are sums hi + lo -+ tol
// rounded outward; everything in tol is rounded up by its spare factors.  A
// coordinate beyond fp32's range has no band, and a length whose square is
// beyond it is bounded by the sum of its components.
__device__ __forceinline__ AxisRay make_axis_ray(const FrameDev& fd, int a, float ox, float oy, float oz, float rs)
{
    AxisRay ar;
    const int k = a >> 1;
    const bool pos = (a & 1) == 0;
    const float ex = ox - fd.c32[0], ey = oy - fd.c32[1], ez = oz - fd.c32[2];
    const float ee = ex * ex + ey * ey + ez * ez;
    const float len = ee < INFINITY ? sqrtf(ee) : fabsf(ex) + fabsf(ey) + fabsf(ez);
    const float reach = (len + fd.r32 + 1e-6f * rs) * fd.rlen[k] + 1e-6f;
    for (int j = 0; j < 3; ++j) {
        const float f0 = fd.axes[6 * j], f1 = fd.axes[6 * j + 1], f2 = fd.axes[6 * j + 2];   // column j
        float hi, lo;
        dot2(ox, f0, oy, f1, oz, f2, hi, lo);
        const float qs = fabsf(ox * f0) + fabsf(oy * f1) + fabsf(oz * f2);
        float tol = 1.01e-9f * rs + 2e-13f * (qs + 4.0f * rs + 1.0f);
        if (j != k) tol += reach * fd.gram_up[3 * j + k];
        tol *= 1.001f;
        const bool in = fabsf(hi) < INFINITY;
        ar.lo[j] = in ? __fadd_rd(hi, __fsub_rd(lo, tol)) : -INFINITY;
        ar.hi[j] = in ? __fadd_ru(hi, __fadd_ru(lo, tol)) : INFINITY;
        if (j == k) {
            if (pos) ar.hi[j] = INFINITY;
            else ar.lo[j] = -INFINITY;
        }
    }
    return ar;
}

__device__ __forceinline__ void warp_add_counters(unsigned long long* counters, long long rays,
                                                  int amb, int retests, int overflow, long long nvis = 0,
                                                  long long ntri = 0)
{
    const unsigned full = 0xFFFFFFFFu;
    for (int off = 16; off; off >>= 1) {
        rays += __shfl_xor_sync(full, rays, off);
        amb += __shfl_xor_sync(full, amb, off);
        retests += __shfl_xor_sync(full, retests, off);
        overflow += __shfl_xor_sync(full, overflow, off);
        nvis += __shfl_xor_sync(full, nvis, off);
        ntri += __shfl_xor_sync(full, ntri, off);
    }
    if ((threadIdx.x & 31) == 0 && counters) {
        if (rays) atomicAdd(&counters[0], (unsigned long long)rays);
        if (amb) atomicAdd(&counters[1], (unsigned long long)amb);
        if (retests) atomicAdd(&counters[2], (unsigned long long)retests);
        if (overflow) atomicAdd(&counters[3], (unsigned long long)overflow);
        if (nvis) atomicAdd(&counters[4], (unsigned long long)nvis);
        if (ntri) atomicAdd(&counters[5], (unsigned long long)ntri);
    }
}

// n.a >= -par_tol, as decided in FP64 (x, y, z order): in fp32 where its
// error, under 4 u of the terms' magnitudes, cannot matter
__device__ __forceinline__ bool eligible(float nx, float ny, float nz, float dx, float dy, float dz, double par_tol)
{
    const float s = fmaf(nx, dx, fmaf(ny, dy, nz * dz)), t = (float)par_tol;
    const float m = 5e-7f * (fabsf(nx * dx) + fabsf(ny * dy) + fabsf(nz * dz) + t) + 1e-36f;
    if (s + t > m) return true;
    if (s + t < -m) return false;
    double nd = __dadd_rn(__dmul_rn((double)nx, (double)dx), __dmul_rn((double)ny, (double)dy));
    nd = __dadd_rn(nd, __dmul_rn((double)nz, (double)dz));
    return nd >= -par_tol;
}

// ---------------------------------------------------------------------------
// Section 3.1: hemispherical cast.  One warp per point (dynamic work
// counter).  The warp casts the point's N directions in N/32 tiles of 32
// spatially close directions (the table is stored in tile order, each entry
// carrying its canonical index j), so that the rays of a warp walk nearly
// the same part of the tree.  Direction j is bit j & 31 of word j >> 5 of the
// warp's shared-memory row, which is written out in canonical order once the
// point is done.
// ---------------------------------------------------------------------------
// 5 blocks of 4 warps of the pooled walk: 96 registers with some 100 bytes of
// spills, and the 25 KB of pools and 12 bytes per warp and word of directions
// that a block keeps in shared memory leave L1 85 KB at 2,048 directions.  4
// and 6 blocks measured 30.1 and 31.3 ms against 27.0 on the impeller (100k
// points x 2048).  Five fit an SM up to 13,300 directions, three up to 34,112,
// and beyond that a point is cast in segments (kSegTiles), five again.
#ifndef RC_HEMI_MIN_BLOCKS
#define RC_HEMI_MIN_BLOCKS 5
#endif
#ifndef RC_UPDATE_MIN_BLOCKS
#define RC_UPDATE_MIN_BLOCKS 7
#endif
#ifndef RC_AXIS_MIN_BLOCKS
#define RC_AXIS_MIN_BLOCKS 5
#endif
#ifndef RC_BATCH_MIN_BLOCKS
#define RC_BATCH_MIN_BLOCKS 5
#endif
#ifndef RC_TAIL_SPLITS
#define RC_TAIL_SPLITS 4
#endif
#ifndef RC_TAIL_POINTS
#define RC_TAIL_POINTS 2        // points cast in parts, per resident warp
#endif

using CastAcc = CastAccFwd;

// ---------------------------------------------------------------------------
// Pooled walk of one point's rays by one warp (4-wide tree).  A tile of 32
// walks, one per lane, keeps a warp at about 11 active lanes: walk lengths
// are heavy-tailed, and lanes at a node wait for lanes at a leaf.  Here the
// unit of work is a pair (ray, node) or (ray, leaf).  The warp keeps a stack
// of such pairs in shared memory and takes up to 32 from its top at a time, a
// pair per lane, whichever rays they belong to, so every box test and every
// triangle test runs on (nearly) full warps.
//   - Rays enter in tiles: a ray's direction and reciprocals live in a slot
//     in shared memory; slots 32..63 hold the tile that entered last and
//     slots 0..31 the rays of the pairs left over from earlier tiles (moved
//     there when the next tile enters).
//   - A tile first finds the frontier boxes it can meet at all (interval
//     slab test on its directions, a lane per box: 5 of 25 on the impeller).
//     Those are tested for its rays, nearest first, while fewer than 32 pairs
//     wait, and the next tile enters when they are used up.  So the warp does
//     not run dry before the point's last tile, and a tile whose rays are all
//     blocked leaves its remaining boxes untested.  Testing boxes ahead (48
//     or 64 pairs) fills the lanes better and still measured 11% and 22%
//     slower: more pairs of rays that a nearer box would have blocked.
//   - Pairs of a blocked ray are dropped when they are taken.  The triangles
//     of a leaf wait, each for itself, in a queue of their own for a full step
//     of tests (a lane per leaf left the second test a third empty: impeller
//     28.4 -> 27.2 ms per 100k points); those of at most 32 pairs left over
//     move on to the next tile with the nodes (29.2 -> 28.4 ms).
//   - Entered children are pushed as they lie in the node, one of every lane
//     on top, so the walk stays depth-first; steps of 22 lanes and more are
//     taken as they come (27.0 ms; refilled to 28: 27.2, to 30: 27.5).
// Every ray meets the same boxes and triangles as in a walk of its own, less
// those that a hit found earlier makes unnecessary, so the bits are the same.
// What bounds it: the latency of dependent instructions and loads at 20 warps
// per SM (a warp issues every 7.7 cycles, 63% of the issue slots at 28 active
// lanes); more warps would need fewer registers than the walk has, and their
// pools would take the L1 they live from (6 blocks per SM: 31.3 ms, 4: 30.1).
// Steps at nodes take 55% of the time, at triangles 25%.
// ---------------------------------------------------------------------------
constexpr int kPoolPairs = 320;        // pairs (ray, node or leaf) on the stack
constexpr int kPoolLeaves = 128;       // pairs (ray, triangle) that wait for a full step
constexpr int kPoolFill = 22;          // lanes that are enough for a step
// Room on the stack: a step takes n <= 32 pairs and adds up to 4 n.  Before a
// step that may find no room the lowest kPoolMove pairs move to the lanes'
// local memory; they come back when fewer than 32 wait (axis rays: none).
// Taking fewer pairs a step instead, down to one, starved parts whose boxes
// overlap: 16,384 diagonal needles, 1,024 points x 256 directions 259 ms, now
// 62 (a ray per lane: 150), their 3,072 axis rays 54.8 ms, now 10.0 (18.2).
// All pairs together: what a step adds lies on top, and what lies above a pair
// that waits descends from pairs added with it.  So at most one step's pairs
// wait per level of the tree, 128 for each of (kStack4 - 1) / 3 levels, on top
// of a box's rays and what was left before them.
constexpr int kPoolFull = kPoolPairs - 96;
constexpr int kPoolMove = 128;         // four a lane
constexpr int kPoolStore = 128;        // pairs a lane can keep aside
static_assert(kPoolFull >= 64 && kPoolMove <= kPoolFull, "a box's rays on top of what waits");
static_assert(32 * kPoolStore >= 63 + 128 * ((kStack4 - 1) / 3), "every pair of a walk has a place");

// A pair: a code (node >= 0, leaf < 0) and the slot of its ray.  32 bits hold
// codes of 26 bits, that is 2^25 nodes and 2^24 triangles; parts beyond that
// use 64 (0.3 ms of 31 slower on the impeller, and half the stack more of L1).
template <bool kBig>
struct PairOf {
    int v;
    static __device__ __forceinline__ PairOf make(int code, int slot) { return {(code << 6) | slot}; }
    __device__ __forceinline__ int code() const { return v >> 6; }
    __device__ __forceinline__ int slot() const { return v & 63; }
};
template <>
struct PairOf<true> {
    int c, s;
    static __device__ __forceinline__ PairOf make(int code, int slot) { return {code, slot}; }
    __device__ __forceinline__ int code() const { return c; }
    __device__ __forceinline__ int slot() const { return s; }
};
constexpr int64_t kPairTris = 1 << 24;     // most triangles of 32-bit pairs (leaves of 2, nodes fewer)
static_assert(kLeafMax == 2, "a leaf code of 2^24 triangles has 26 bits with its sign; a leaf adds two pairs at most");

template <bool kBig>
struct __align__(16) PoolOf {
    Frontier front;
    float4 onb[3];                 // basis t1, t2 and the normal: components x, y, z
    float4 inv[64];                // reciprocals of the ray's direction, canonical index
    float4 dir[64];                // direction, its largest |component|
    PairOf<kBig> pair[kPoolPairs];
    PairOf<kBig> leaf[kPoolLeaves];
    uint8_t met[kFrontEntries];    // the frontier boxes that the current tile can meet
};
static_assert(kPoolPairs >= kFrontQueue, "the stack also serves as the frontier's queue");

// The lowest kPoolMove of the stack's sp pairs go to the lanes' stores (each
// place is read and written by one lane: no barrier in between), and back.
// The warp calls both; a barrier before and after.
template <class Pair>
__device__ __forceinline__ void pool_aside(Pair* pair, int& sp, Pair* store, int& stored)
{
    const int lane = threadIdx.x & 31;
    for (int k = 0; k < kPoolMove / 32; ++k) store[stored + k] = pair[32 * k + lane];
    stored += kPoolMove / 32;
    for (int q = kPoolMove + lane; q < sp; q += 32) pair[q - kPoolMove] = pair[q];
    sp -= kPoolMove;
    __syncwarp();
}
template <class Pair>
__device__ __forceinline__ void pool_back(Pair* pair, int& sp, Pair* store, int& stored)
{
    const int lane = threadIdx.x & 31;
    stored -= kPoolMove / 32;
    if (lane < sp) pair[kPoolMove + lane] = pair[lane];
    for (int k = 0; k < kPoolMove / 32; ++k) pair[32 * k + lane] = store[stored + k];
    sp += kPoolMove;
    __syncwarp();
}

// bit rows of a warp: visible so far, met an ambiguous pair, met an ambiguous
// pair that FP64 calls a hit, and (instrumented cast) re-tested in FP64
__host__ __device__ __forceinline__ constexpr int pool_rows(bool stats) { return stats ? 4 : 3; }

// A point of more than kWholeWords words of directions is cast in segments of
// kSegTiles tiles, whose rows hold the words that the segment's tiles reach:
// a band of the tile order has as many tiles as words, the same ones, and at
// most kMaxBand.  Up to kWholeWords three blocks with whole rows fit an SM;
// with 65,536 directions it was one (6,000 points of the housing 51.4 ms, now
// 21.1; 49,152 directions, 500 points, 3.07 and 2.67).  Segments from the
// words on at which five blocks fit no more would gain nothing: their kernel
// spills more (10,000 x 32,768: 19.6 ms whole, 20.2; 20,000 x 16,384: 15.3 and
// 15.8), and so would one kernel for both (4,096 directions 10% slower).
constexpr int kSegTiles = 256, kSegWords = kSegTiles + 2 * kMaxBand, kWholeWords = 1066;

// FP32 decision of one pair by signed volumes (Moeller and Trumbore 1997),
// with a forward error bound; kHit and kMiss only when certain, as
// tri_test32.  With s = A - o, e1 = B - A, e2 = C - A, p = d x e2 and
// q = s x e1 the hit point is A + (U/D) e1 + (V/D) e2 at t = T/D, where
// U = s.p, V = d.q, D = -(e1.p), T = e2.q; the third edge is W = D - U - V.
// Unlike the sheared form it needs no permutation of the coordinates by the
// ray's largest component, and the bound needs only the largest |s_k| (S),
// the triangle's largest edge component (e, stored in its record) and the
// ray's largest |d_k| (m):
//   inputs     s and e round once (u relative; e is a computed value)
//   |p| <= 2me, error 5 u m e        |q| <= 2Se, error 7 u S e
//   U: 15 (p) + 6 (s) + 12 (sum) = 33 u S m e;   V: 21 + 12 = 33 u S m e
//   D: 15 + 6 + 12 = 33 u m e^2;     T: 21 + 6 + 12 = 39 u S e^2
//   W: U + V + D and two roundings = u m e (84 S + 45 e)
// each scaled by 1.0625 for second-order terms and the bound's own rounding;
// 1e-36 covers products that leave the normal range.
__device__ __forceinline__ int tri_test_mt(float ox, float oy, float oz, float dx, float dy, float dz, float m,
                                           float rs, const float4 v0, const float4 v1, const float4 v2)
{
    const float u = 5.9604644775390625e-8f;
    const float s0 = v0.x - ox, s1 = v0.y - oy, s2 = v0.z - oz;
    const float a0 = v1.x - v0.x, a1 = v1.y - v0.y, a2 = v1.z - v0.z;
    const float b0 = v2.x - v0.x, b1 = v2.y - v0.y, b2 = v2.z - v0.z;
    const float p0 = fmaf(dy, b2, -(dz * b1)), p1 = fmaf(dz, b0, -(dx * b2)), p2 = fmaf(dx, b1, -(dy * b0));
    const float q0 = fmaf(s1, a2, -(s2 * a1)), q1 = fmaf(s2, a0, -(s0 * a2)), q2 = fmaf(s0, a1, -(s1 * a0));
    const float U = fmaf(s0, p0, fmaf(s1, p1, s2 * p2));
    const float V = fmaf(dx, q0, fmaf(dy, q1, dz * q2));
    const float D = -fmaf(a0, p0, fmaf(a1, p1, a2 * p2));
    const float W = (D - U) - V;
    const float S = fmaxf(fabsf(s0), fmaxf(fabsf(s1), fabsf(s2)));
    const float e = v0.w;
    const float ume = u * m * e;
    const float eU = fmaf(35.1f * ume, S, 1e-36f);
    const float eW = fmaf(89.3f * ume, S, fmaf(47.9f * ume, e, 1e-36f));
    const bool pos = fmaxf(U, V) > eU || W > eW, neg = fminf(U, V) < -eU || W < -eW;
    if (pos && neg) return kMiss;

    const float T = fmaf(b0, q0, fmaf(b1, q1, b2 * q2));
    const float eD = fmaf(35.1f * ume, e, 1e-36f);
    const float eT = fmaf(41.5f * u * S, e * e, 1e-36f);
    const bool tp_ok = fabsf(T) > eT;
    if (fabsf(D) > eD && tp_ok && (T > 0.0f) != (D > 0.0f)) return kMiss;   // plane crossed behind the origin
    // clear hit: every edge beyond its error and the tau band (|edge x d| <=
    // 3 m e), hence all of one sign, which is D's; the crossing ahead and
    // beyond tau R along the ray
    const float tau_edge = 3.0f * 1e-9f * 1.01f * rs * m * e;
    if (fminf(fabsf(U), fabsf(V)) > eU + tau_edge && fabsf(W) > eW + tau_edge && tp_ok &&
        (T > 0.0f) == (U > 0.0f) && (fabsf(T) - eT) * m > 1.01e-9f * rs * (fabsf(D) + eD))
        return kHit;
    return kUnsure;
}

// One axis of the slab test on a tile's directions: their components span
// [dl, dh], and a box spans [l, h] relative to the shared origin.  Some ray of
// the tile can be inside the slab at t >= 0 only for t in [tn, tf]:
// l <= t d with d <= dh gives t >= l / dh, and so on; a component that spans
// zero (or nearly) bounds t from below only.  Roundings are covered by the
// box's margin (ex, ey, ez) and the 1e-5 by which the caller widens tf.
struct TileAxis {
    float a, b, c, d, far;
    __device__ __forceinline__ void clip(float l, float h, float& tn, float& tf) const
    {
        tn = fmaxf(tn, fmaxf(l * a, h * b));
        tf = fminf(tf, fmaf(h, c, fmaf(l, d, far)));
    }
};

__device__ __forceinline__ float rcp_approx(float x)   // within 2^-23 relative
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// a lane's share of a ray's reciprocals: one unit in the last place off at
// most, zero components as in setup_ray
__device__ __forceinline__ float ray_rcp(float d)
{
    const float i = rcp_approx(d);
    return fabsf(i) <= 0x1p100f ? i : copysignf(0x1p100f, d);
}

__device__ __forceinline__ TileAxis tile_axis(float x)
{
    const float lo = warp_min(x), hi = warp_max(x);
    constexpr float kSmall = 1e-4f;
    TileAxis t;
    const float rl = rcp_approx(lo), rh = rcp_approx(hi);
    t.a = hi >= kSmall ? rh : (hi > 0.0f ? 1.0f / kSmall : 0.0f);
    t.b = lo <= -kSmall ? rl : (lo < 0.0f ? -1.0f / kSmall : 0.0f);
    t.c = lo >= kSmall ? rl : 0.0f;
    t.d = hi <= -kSmall ? rh : 0.0f;
    t.far = lo >= kSmall || hi <= -kSmall ? 0.0f : INFINITY;
    return t;
}

// FP64 decision of the lanes' pairs (ray j in direction d, triangle record
// tp) that FP32 left open; true for a clear hit.  Not inlined: it is rare.
template <bool kStats>
__device__ __noinline__ bool pool_retest(float ox, float oy, float oz, const float4 d, int j, const float4* tp,
                                         uint32_t* rows, int R, int64_t i, long long* relist, long long relist_cap,
                                         unsigned long long* relist_ctr)
{
    const Pair64 q = retest64<false>(ox, oy, oz, d.x, d.y, d.z, tp[0], tp[1], tp[2]);
    const uint32_t b = 1u << (j & 31);
    if (kStats && relist && !(atomicOr(&rows[3 * R + (j >> 5)], b) & b)) {
        const unsigned long long at = atomicAdd(relist_ctr, 1ULL);
        if (at < (unsigned long long)relist_cap) relist[at] = (long long)i * 65536 + j;
    }
    if (q.state == kUnsure) {
        atomicOr(&rows[R + (j >> 5)], b);
        if (q.hit64) atomicOr(&rows[2 * R + (j >> 5)], b);
    }
    return q.state == kHit;
}

// cast_point on the 4-wide tree (same arguments; pool and rows: the warp's
// shared memory)
template <bool kStats, bool kBig, bool kSeg>
__device__ __forceinline__ void cast_point_pooled(const float4* __restrict__ wnodes, const float4* __restrict__ tris,
                                                  int max_steps, float scene_maxabs, const float* __restrict__ P,
                                                  const float* __restrict__ Nrm, int64_t i,
                                                  const float4* __restrict__ tdirs, int W, double eps,
                                                  PoolOf<kBig>* pool, uint32_t* rows, uint32_t* __restrict__ bits,
                                                  int32_t* __restrict__ count, CastAcc& acc, int t0, int t1,
                                                  bool whole, long long* relist, long long relist_cap,
                                                  unsigned long long* relist_ctr)
{
    using Pair = PairOf<kBig>;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    // the rows hold words [w0, w1), R words apart, and start at word w0
    const int R = kSeg ? kSegWords : W, w0 = kSeg ? max(0, t0 - kMaxBand) : 0, w1 = kSeg ? min(W, t1 + kMaxBand) : W;
    for (int w = lane; w < pool_rows(kStats) * R; w += 32) rows[w] = 0u;
    rows -= w0;
    uint32_t* vis = rows;
    Frontier* f = &pool->front;
    float ox, oy, oz;
    {
        const float nx = Nrm[3 * i], ny = Nrm[3 * i + 1], nz = Nrm[3 * i + 2];
        ox = offset_coord(P[3 * i], nx, eps);
        oy = offset_coord(P[3 * i + 1], ny, eps);
        oz = offset_coord(P[3 * i + 2], nz, eps);
        build_frontier(wnodes, tris, ox, oy, oz, nx, ny, nz, tangent_shortcuts_ok(nx, ny, nz, W),
                       20.0f / (32.0f * W), min(kFrontRounds, W / 4), f, (int*)pool->pair);
        if (lane == 0) {
            const Onb b = make_onb(nx, ny, nz);
            pool->onb[0] = make_float4(b.t1x, b.t2x, nx, 0.0f);
            pool->onb[1] = make_float4(b.t1y, b.t2y, ny, 0.0f);
            pool->onb[2] = make_float4(b.t1z, b.t2z, nz, 0.0f);
        }
        __syncwarp();
    }
    if (kStats && lane == 0) acc.nvis += f->nvis;
    // M >= every coordinate, and the margin of a slab distance per unit of
    // |reciprocal| (see SlabRay), here 6 u (M + |o|) <= 12 u M: a reciprocal
    // off by 2 u, the products and sums of the constants 2 u, the final FMA u
    const float rs = fmaxf(fmaxf(1.0f, scene_maxabs), fmaxf(fabsf(ox), fmaxf(fabsf(oy), fabsf(oz))));
    const float em = 12.0f * 5.9604644775390625e-8f * rs;
    int sp = 0, lsp = 0;                   // pairs on the stack, leaves that wait
    unsigned live0 = 0, live1 = 0;         // slots 0..31 and 32..63 whose rays are not known to be blocked
    int t = t0;                            // next tile
    int boxes = 0;                         // of pool->met still to be tested
    Pair store[kPoolStore];                // pairs set aside (pool_aside)
    int stored = 0;                        // of store, the same in every lane
    // On a well-formed tree a ray meets each node and leaf at most once, and a
    // step takes at least one pair: at most 64 rays have pairs between two
    // entries of tiles.  The cap only bounds a malformed tree.
    const int most = (int)min64(0x7FFFFFFF, 64 * (int64_t)max_steps);
    int steps = most;
    for (;;) {
        if (lsp < 32 && sp < 32 && (boxes > 0 || stored > 0)) {
            if (stored > 0) {
                pool_back(pool->pair, sp, store, stored);
                continue;
            }
            // the tile's rays against its frontier boxes, nearest first (the
            // deepest), until a step's worth of pairs waits
            if (live1 == 0) {
                boxes = 0;
                continue;
            }
            const bool on = (live1 >> lane) & 1u;
            const float4 v = pool->inv[32 + lane];
            const float x = ox * v.x, y = oy * v.y, z = oz * v.z;
            const float mx = em * fabsf(v.x), my = em * fabsf(v.y), mz = em * fabsf(v.z);
            const bool bx = signbit(v.x), by = signbit(v.y), bz = signbit(v.z);
            do {
                const int e = pool->met[--boxes];
                const float4 lo = f->box[2 * e], hi = f->box[2 * e + 1];
                const float tn = fmaxf(fmaxf(fmaf(bx ? hi.x : lo.x, v.x, -(x + mx)), fmaf(by ? hi.y : lo.y, v.y, -(y + my))),
                                       fmaxf(fmaf(bz ? hi.z : lo.z, v.z, -(z + mz)), 0.0f));
                const float tf = fminf(fminf(fmaf(bx ? lo.x : hi.x, v.x, mx - x), fmaf(by ? lo.y : hi.y, v.y, my - y)),
                                       fmaf(bz ? lo.z : hi.z, v.z, mz - z));
                const bool in = on && tn <= tf;
                if (kStats) acc.nbox += on;
                const unsigned m = __ballot_sync(kAll, in);
                if (in) pool->pair[sp + __popc(m & below)] = Pair::make(__float_as_int(lo.w), 32 + lane);
                sp += __popc(m);
            } while (boxes > 0 && sp < 32);
            __syncwarp();
            continue;
        }
        if (lsp < 32 && (sp >= 32 || (sp > 0 && t >= t1))) {
            // up to 32 live pairs with a node from the top of the stack, one
            // per lane; pairs with a leaf move to the leaf queue, pairs of
            // blocked rays are dropped, and lanes left without look again
            if (--steps < 0) break;
            if (sp > kPoolFull) pool_aside(pool->pair, sp, store, stored);
            bool have = false;
            int code = 0, slot = 0;
            for (;;) {
                const unsigned want = __ballot_sync(kAll, !have);
                const int at = sp - 1 - __popc(want & below);
                bool leaf = false;
                if (!have && at >= 0) {
                    const Pair q = pool->pair[at];
                    slot = q.slot();
                    code = q.code();
                    const bool live = ((slot & 32 ? live1 : live0) >> (slot & 31)) & 1u;
                    have = live && code >= 0;
                    leaf = live && code < 0;
                }
                const bool two = leaf && leaf_count(code) == 2;
                const unsigned ml = __ballot_sync(kAll, leaf), m2 = __ballot_sync(kAll, two);
                if (leaf) pool->leaf[lsp + __popc(ml & below)] = Pair::make(leaf_code(leaf_first(code), 1), slot);
                lsp += __popc(ml);
                if (two) pool->leaf[lsp + __popc(m2 & below)] = Pair::make(leaf_code(leaf_first(code) + 1, 1), slot);
                lsp += __popc(m2);
                sp = max(0, sp - __popc(want));
                if (sp == 0 || lsp > kPoolLeaves - 64 || __popc(__ballot_sync(kAll, have)) >= kPoolFill) break;
            }
            bool i0 = false, i1 = false, i2 = false, i3 = false;
            float4 ci = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (have) {
                if (kStats) acc.nvis += 1;
                const float4 v = pool->inv[slot];
                const float x = ox * v.x, y = oy * v.y, z = oz * v.z;
                const float mx = em * fabsf(v.x), my = em * fabsf(v.y), mz = em * fabsf(v.z);
                // near and far planes by the sign of the direction (wide_at:
                // float4 c lies at c ^ (node & 7))
                const unsigned at = ((unsigned)code & 7u) << 4;
                const unsigned qx = at ^ ((__float_as_uint(v.x) >> 27) & 16u),
                               qy = at ^ ((__float_as_uint(v.y) >> 27) & 16u) ^ 32u,
                               qz = at ^ ((__float_as_uint(v.z) >> 27) & 16u) ^ 64u;
                const auto ld = [&](unsigned q) {
                    if (kBig) return __ldg((const float4*)((const char*)wnodes + ((size_t)code << 7) + q));
                    return __ldg((const float4*)((const char*)wnodes + (((unsigned)code << 7) | q)));
                };
                const float4 nx = ld(qx), fx = ld(qx ^ 16u), ny = ld(qy), fy = ld(qy ^ 16u), nz = ld(qz), fz = ld(qz ^ 16u);
                ci = ld(at ^ 96u);
                const auto entry = [&](float nxk, float nyk, float nzk, float fxk, float fyk, float fzk) {
                    const float tn = fmaxf(fmaxf(fmaf(nxk, v.x, -(x + mx)), fmaf(nyk, v.y, -(y + my))),
                                           fmaxf(fmaf(nzk, v.z, -(z + mz)), 0.0f));
                    const float tf = fminf(fminf(fmaf(fxk, v.x, mx - x), fmaf(fyk, v.y, my - y)),
                                           fmaf(fzk, v.z, mz - z));
                    return tn <= tf;
                };
                i0 = entry(nx.x, ny.x, nz.x, fx.x, fy.x, fz.x);
                i1 = entry(nx.y, ny.y, nz.y, fx.y, fy.y, fz.y);
                i2 = entry(nx.z, ny.z, nz.z, fx.z, fy.z, fz.z);
                i3 = entry(nx.w, ny.w, nz.w, fx.w, fy.w, fz.w);
            }
            __syncwarp();
            // push the entered children: the last three first (a lane's side
            // by side, its count 0..3 summed over the lower lanes bit by bit),
            // then the first of every lane.  Nothing is gained by sorting
            // them by distance: an any-hit ray ends as soon in either order
            // (impeller 29.3 ms per 100k points sorted, 29.2 as they lie)
            const unsigned b0 = __ballot_sync(kAll, i1 ^ i2 ^ i3), b1 = __ballot_sync(kAll, (i1 & i2) | (i3 & (i1 | i2))),
                           bn = __ballot_sync(kAll, i0);
            int at = sp + __popc(b0 & below) + 2 * __popc(b1 & below);
            if (i3) pool->pair[at++] = Pair::make(__float_as_int(ci.w), slot);
            if (i2) pool->pair[at++] = Pair::make(__float_as_int(ci.z), slot);
            if (i1) pool->pair[at] = Pair::make(__float_as_int(ci.y), slot);
            sp += __popc(b0) + 2 * __popc(b1);
            if (i0) pool->pair[sp + __popc(bn & below)] = Pair::make(__float_as_int(ci.x), slot);
            sp += __popc(bn);
            __syncwarp();
            continue;
        }
        if (lsp >= 32 || (lsp > 0 && (t >= t1 || sp + lsp > 32))) {
            // up to 32 pairs with a triangle, one per lane
            const int at = lsp - 1 - lane;
            lsp = max(0, lsp - 32);
            int slot = 0;
            bool hit = false;
            if (at >= 0) {
                const Pair q = pool->leaf[at];
                slot = q.slot();
                if (((slot & 32 ? live1 : live0) >> (slot & 31)) & 1u) {
                    const float4 rd = pool->dir[slot];
                    const float4* tp = tris + 3 * (int64_t)leaf_first(q.code());
                    if (kStats) acc.ntri += 1;
                    int st = tri_test_mt(ox, oy, oz, rd.x, rd.y, rd.z, rd.w, rs, __ldg(tp), __ldg(tp + 1), __ldg(tp + 2));
                    if (st == kUnsure) {
                        acc.retests += 1;
                        if (pool_retest<kStats>(ox, oy, oz, rd, __float_as_int(pool->inv[slot].w), tp, rows, R, i, relist,
                                                relist_cap, relist_ctr))
                            st = kHit;
                    }
                    hit = st == kHit;
                }
            }
            if (hit) {
                const int j = __float_as_int(pool->inv[slot].w);
                atomicAnd(&vis[j >> 5], ~(1u << (j & 31)));
            }
            const unsigned bit = hit ? 1u << (slot & 31) : 0u;
            live0 &= ~__reduce_or_sync(kAll, slot & 32 ? 0u : bit);
            live1 &= ~__reduce_or_sync(kAll, slot & 32 ? bit : 0u);
            __syncwarp();
            continue;
        }
        if (t >= t1) break;
        steps = most;
        // the next tile enters; the rays of the pairs left over move down
        // (one slot per ray, the lowest pair's)
        if (sp + lsp > 0) {
            const bool mine = lane < sp + lsp;
            Pair* const at = lane < sp ? &pool->pair[lane] : &pool->leaf[lane - sp];
            Pair q = Pair::make(0, 0);
            if (mine) q = *at;
            const int from = q.slot();
            const float4 li = pool->inv[from], ld = pool->dir[from];
            const bool live = mine && (((from & 32 ? live1 : live0) >> (from & 31)) & 1u);
            const int to = __ffs(__match_any_sync(kAll, live ? __float_as_int(li.w) : -1 - lane)) - 1;
            live0 = __ballot_sync(kAll, live && to == lane);
            __syncwarp();                  // every slot is read before one is written
            if (live && to == lane) {
                pool->inv[lane] = li;
                pool->dir[lane] = ld;
            }
            if (mine) *at = Pair::make(q.code(), to);    // a pair of a blocked ray: its own slot, not live
            __syncwarp();
        }
        const float4 h = __ldg(&tdirs[32 * t + lane]);
        const float4 cx = pool->onb[0], cy = pool->onb[1], cz = pool->onb[2];
        const int jt = __float_as_int(h.w);    // -1: padding of the last tile
        const Onb b = {cx.x, cy.x, cz.x, cx.y, cy.y, cz.y};
        float4 rd;
        local_to_world(b, cx.z, cy.z, cz.z, h.x, h.y, h.z, rd.x, rd.y, rd.z);
        rd.w = fmaxf(fabsf(rd.x), fmaxf(fabsf(rd.y), fabsf(rd.z)));
        pool->inv[32 + lane] = make_float4(ray_rcp(rd.x), ray_rcp(rd.y), ray_rcp(rd.z), h.w);
        pool->dir[32 + lane] = rd;
        ++t;
        // the point's local triangles
        bool open = jt >= 0;
        for (int k = 0; k < f->ntris; ++k) {
            if (!open) continue;
            if (kStats) acc.ntri += 1;
            int st = tri_test_mt(ox, oy, oz, rd.x, rd.y, rd.z, rd.w, rs, f->tri[3 * k], f->tri[3 * k + 1],
                                 f->tri[3 * k + 2]);
            if (st == kUnsure) {
                acc.retests += 1;
                if (pool_retest<kStats>(ox, oy, oz, rd, jt, &f->tri[3 * k], rows, R, i, relist, relist_cap, relist_ctr))
                    st = kHit;
            }
            open = st != kHit;
        }
        if (open) atomicOr(&vis[jt >> 5], 1u << (jt & 31));
        live1 = __ballot_sync(kAll, open);
        // the frontier boxes that the tile can meet: the slab test on the
        // intervals that its directions span, a lane per box
        const int src = __ffs(__ballot_sync(kAll, jt >= 0)) - 1;
        const float sx = __shfl_sync(kAll, rd.x, src), sy = __shfl_sync(kAll, rd.y, src),
                    sz = __shfl_sync(kAll, rd.z, src);
        const TileAxis ax = tile_axis(jt >= 0 ? rd.x : sx), ay = tile_axis(jt >= 0 ? rd.y : sy),
                       az = tile_axis(jt >= 0 ? rd.z : sz);
        for (int q = 0; q < f->nboxes; q += 32) {
            const int k = q + lane;
            bool in = k < f->nboxes;
            if (in) {
                const float4 lo = f->box[2 * k], hi = f->box[2 * k + 1];
                float tn = 0.0f, tf = INFINITY;
                ax.clip(lo.x - ox - em, hi.x - ox + em, tn, tf);
                ay.clip(lo.y - oy - em, hi.y - oy + em, tn, tf);
                az.clip(lo.z - oz - em, hi.z - oz + em, tn, tf);
                in = tn <= tf * 1.00001f;
            }
            const unsigned m = __ballot_sync(kAll, in);
            if (in) pool->met[boxes + __popc(m & below)] = (uint8_t)k;
            boxes += __popc(m);
        }
        __syncwarp();
    }
    if (steps < 0) {
        // rays that are not decided count as blocked (those of later tiles have no bit yet)
        acc.overflow += lane == 0;
        for (int q = 0; q < 2; ++q)
            if (((q ? live1 : live0) >> lane) & 1u) {
                const int j = __float_as_int(pool->inv[32 * q + lane].w);
                atomicAnd(&vis[j >> 5], ~(1u << (j & 31)));
            }
        __syncwarp();
    }
    // visible, less the rays that only an FP64-ambiguous pair blocks
    int cnt = 0;
    for (int w = w0 + lane; w < w1; w += 32) {
        const uint32_t v = vis[w];
        acc.amb += __popc(v & rows[R + w]);
        const uint32_t r = v & ~rows[2 * R + w];
        cnt += __popc(r);
        if (whole)
            bits[i * W + w] = r;
        else if (r)
            atomicOr(&bits[i * W + w], r);
    }
    for (int off = 16; off; off >>= 1) cnt += __shfl_xor_sync(kAll, cnt, off);
    if (lane == 0) {
        if (whole)
            count[i] = cnt;
        else
            atomicAdd(&count[i], cnt);
    }
    __syncwarp();
    acc.rays += (t1 - t0) - (t1 == W && __float_as_int(__ldg(&tdirs[32 * (W - 1) + lane]).w) < 0 ? 1 : 0);
}

// ---------------------------------------------------------------------------
// Pooled walk of 32 parallel axis rays by one warp (frame tree).  As the
// hemispherical walk above: pairs (ray, node or leaf) on a stack in shared
// memory, 32 taken at a time.  Here one long walk matters most: a ray that
// runs along a fillet or a bore 1e-4 mm above it enters hundreds of boxes,
// and alone in its lane it set the time of the launch; pooled, its pairs
// fill the warp.  The rays of a warp share direction and axis, so a slot
// holds an origin and a band only.  A queue of 32 triangles is tested at once,
// fewer when no nodes are left (testing fewer earlier measured the same).
// Prismatic part turned off its axes, 100k points: six axes, covers and a
// ball-end tool 3.86 -> 2.61 ms, choice of a frame 5.84 -> 4.01 ms.  Children
// pushed as they lie and triangles queued one by one: 1.45 -> 1.30 and 2.0 ->
// 1.85 ms of what later changes had left.
// ---------------------------------------------------------------------------
template <bool kBig>
struct __align__(16) AxisPoolOf {
    float4 lo[32], hi[32];         // band (AxisRay) and the origin's x, y
    float oz[32];
    PairOf<kBig> pair[kPoolPairs];
    PairOf<kBig> leaf[kPoolLeaves];
};

struct AxisAcc { int amb = 0, retests = 0, overflow = 0; long long rays = 0, nvis = 0, ntri = 0; };

// All lanes call it; `cast` lanes have a ray (r, ar; the same axis and
// direction in every lane, cast or not).  True where the lane's ray is
// blocked.
template <bool kStats, bool kBig>
__device__ __forceinline__ bool trace_axis(const float4* __restrict__ ftree, const float4* __restrict__ tris, const Ray& r,
                                           const AxisRay& ar, bool cast, float scene_maxabs, int max_steps,
                                           AxisPoolOf<kBig>* pool, AxisAcc& acc)
{
    using Pair = PairOf<kBig>;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    unsigned live = __ballot_sync(kAll, cast);
    if (live == 0) return false;
    unsigned amb = 0, hit64 = 0;           // rays with an ambiguous pair; one that FP64 calls a hit
    __syncwarp();
    if (cast) {
        pool->lo[lane] = make_float4(ar.lo[0], ar.lo[1], ar.lo[2], r.ox);
        pool->hi[lane] = make_float4(ar.hi[0], ar.hi[1], ar.hi[2], r.oy);
        pool->oz[lane] = r.oz;
        pool->pair[__popc(live & below)] = Pair::make(0, lane);
        acc.rays += 1;
    }
    int sp = __popc(live), lsp = 0;
    Pair store[kPoolStore];                // pairs set aside (pool_aside)
    int stored = 0;
    __syncwarp();
    // on a well-formed tree each of 32 rays meets a node or leaf at most once,
    // and a step takes at least one pair; the cap only bounds a malformed tree
    int steps = (int)min64(0x7FFFFFFF, 32 * (int64_t)max_steps);
    for (;;) {
        if (lsp < 32 && sp > 0) {
            if (--steps < 0) break;
            if (sp > kPoolFull) pool_aside(pool->pair, sp, store, stored);
            bool have = false;
            int code = 0, slot = 0;
            for (;;) {
                const unsigned want = __ballot_sync(kAll, !have);
                const int at = sp - 1 - __popc(want & below);
                bool leaf = false;
                if (!have && at >= 0) {
                    const Pair q = pool->pair[at];
                    slot = q.slot();
                    code = q.code();
                    const bool on = (live >> slot) & 1u;
                    have = on && code >= 0;
                    leaf = on && code < 0;
                }
                const bool two = leaf && leaf_count(code) == 2;
                const unsigned ml = __ballot_sync(kAll, leaf), m2 = __ballot_sync(kAll, two);
                if (leaf) pool->leaf[lsp + __popc(ml & below)] = Pair::make(leaf_code(leaf_first(code), 1), slot);
                lsp += __popc(ml);
                if (two) pool->leaf[lsp + __popc(m2 & below)] = Pair::make(leaf_code(leaf_first(code) + 1, 1), slot);
                lsp += __popc(m2);
                sp = max(0, sp - __popc(want));
                if (sp == 0 || lsp > kPoolLeaves - 64 || __popc(__ballot_sync(kAll, have)) >= kPoolFill) break;
            }
            bool i0 = false, i1 = false, i2 = false, i3 = false;
            float4 ci = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (have) {
                if (kStats) acc.nvis += 1;
                const float4* nd = wide_ptr(ftree, code);
                const float4 lx = wide_ld(nd, 0), hx = wide_ld(nd, 1), ly = wide_ld(nd, 2), hy = wide_ld(nd, 3);
                const float4 lz = wide_ld(nd, 4), hz = wide_ld(nd, 5);
                ci = wide_ld(nd, 6);
                const float4 l = pool->lo[slot], h = pool->hi[slot];
                const auto entry = [&](float lxk, float hxk, float lyk, float hyk, float lzk, float hzk) {
                    return lxk <= h.x && hxk >= l.x && lyk <= h.y && hyk >= l.y && lzk <= h.z && hzk >= l.z;
                };
                i0 = entry(lx.x, hx.x, ly.x, hy.x, lz.x, hz.x);
                i1 = entry(lx.y, hx.y, ly.y, hy.y, lz.y, hz.y);
                i2 = entry(lx.z, hx.z, ly.z, hy.z, lz.z, hz.z);
                i3 = entry(lx.w, hx.w, ly.w, hy.w, lz.w, hz.w);
            }
            __syncwarp();
            const unsigned b0 = __ballot_sync(kAll, i1 ^ i2 ^ i3), b1 = __ballot_sync(kAll, (i1 & i2) | (i3 & (i1 | i2))),
                           bn = __ballot_sync(kAll, i0);
            int at = sp + __popc(b0 & below) + 2 * __popc(b1 & below);
            if (i3) pool->pair[at++] = Pair::make(__float_as_int(ci.w), slot);
            if (i2) pool->pair[at++] = Pair::make(__float_as_int(ci.z), slot);
            if (i1) pool->pair[at] = Pair::make(__float_as_int(ci.y), slot);
            sp += __popc(b0) + 2 * __popc(b1);
            if (i0) pool->pair[sp + __popc(bn & below)] = Pair::make(__float_as_int(ci.x), slot);
            sp += __popc(bn);
            __syncwarp();
            continue;
        }
        if (lsp < 32 && stored > 0) {
            pool_back(pool->pair, sp, store, stored);
            continue;
        }
        if (lsp == 0) break;
        const int at = lsp - 1 - lane;
        lsp = max(0, lsp - 32);
        int slot = 0;
        bool hit = false, ua = false, uh = false;
        if (at >= 0) {
            const Pair pr = pool->leaf[at];
            slot = pr.slot();
            if ((live >> slot) & 1u) {
                Ray q = r;
                q.ox = pool->lo[slot].w;
                q.oy = pool->hi[slot].w;
                q.oz = pool->oz[slot];
                q.rs = fmaxf(fmaxf(1.0f, scene_maxabs), fmaxf(fabsf(q.ox), fmaxf(fabsf(q.oy), fabsf(q.oz))));
                const float4* tp = tris + 3 * (int64_t)leaf_first(pr.code());
                if (kStats) acc.ntri += 1;
                const float4 v0 = __ldg(tp), v1 = __ldg(tp + 1), v2 = __ldg(tp + 2);
                int st = tri_test32(q, v0, v1, v2);
                if (st == kUnsure) st = tri_test_close(q, v0, v1, v2);
                if (st == kUnsure) {
                    ++acc.retests;
                    const Pair64 w = retest64<true>(q.ox, q.oy, q.oz, q.dx, q.dy, q.dz, v0, v1, v2);
                    st = w.state;
                    ua = st == kUnsure;
                    uh = ua && w.hit64;
                }
                hit = st == kHit;
            }
        }
        if (__any_sync(kAll, ua)) {
            amb |= __reduce_or_sync(kAll, ua ? 1u << slot : 0u);
            hit64 |= __reduce_or_sync(kAll, uh ? 1u << slot : 0u);
        }
        live &= ~__reduce_or_sync(kAll, hit ? 1u << slot : 0u);
        __syncwarp();
    }
    if (steps < 0) {
        acc.overflow += lane == 0;
        live = 0;                              // rays that are not decided count as blocked
    }
    const bool open = (live >> lane) & 1u;
    if (open && ((amb >> lane) & 1u)) ++acc.amb;
    return cast && !(open && !((hit64 >> lane) & 1u));
}

// The hemispherical cast of one point by one warp on the binary tree (see
// above), a ray per lane.  `tdirs` is the tile-ordered table, `row` the
// warp's shared-memory row of W words.  Tiles [t0, t1) are cast; a whole
// point (0, W) writes its bit row and count, a part of a point ORs its bits
// into the (zeroed) row in memory and adds its count.
template <bool kStats>
__device__ __forceinline__ void cast_point_binary(const float4* __restrict__ nodes, const float4* __restrict__ tris,
                                                  int max_steps, float scene_maxabs, const float* __restrict__ P,
                                                  const float* __restrict__ Nrm, int64_t i,
                                                  const float4* __restrict__ tdirs, int W, double eps, uint32_t* row,
                                                  uint32_t* __restrict__ bits, int32_t* __restrict__ count,
                                                  CastAcc& acc, int t0, int t1, long long* relist,
                                                  long long relist_cap, unsigned long long* relist_ctr)
{
    const int lane = threadIdx.x & 31;
    const bool whole = t1 < 0;
    if (whole) t1 = W;
    for (int w = lane; w < W; w += 32) row[w] = 0u;
    const float px = P[3 * i], py = P[3 * i + 1], pz = P[3 * i + 2];
    const float nx = Nrm[3 * i], ny = Nrm[3 * i + 1], nz = Nrm[3 * i + 2];
    const float ox = offset_coord(px, nx, eps), oy = offset_coord(py, ny, eps), oz = offset_coord(pz, nz, eps);
    __syncwarp();
    const Onb b = make_onb(nx, ny, nz);
    int cnt = 0;
    for (int t = t0; t < t1; ++t) {
        // canonical index j; when 32 does not divide N the last tile is
        // padded with entries j = -1 that carry a real direction: they are
        // cast like the others (no branch in the loop) and then discarded
        const float4 h = __ldg(&tdirs[32 * t + lane]);
        const int j = __float_as_int(h.w);
        float dx, dy, dz;
        local_to_world(b, nx, ny, nz, h.x, h.y, h.z, dx, dy, dz);
        Ray r;
        setup_ray(r, ox, oy, oz, dx, dy, dz, scene_maxabs);
        const TraceOut tr = trace<kStats>(nodes, tris, r, max_steps);
        acc.retests += tr.retests;
        acc.overflow += tr.overflow;
        acc.amb += (j >= 0) & ((tr.flags >> 1) & 1);
        if (kStats) {
            acc.nvis += tr.nodes;
            acc.ntri += tr.tris;
            // the instrumented cast can list the rays an FP64 re-test took part in
            if (relist && tr.retests > 0 && j >= 0) {
                const unsigned long long k = atomicAdd(relist_ctr, 1ULL);
                if (k < (unsigned long long)relist_cap) relist[k] = (long long)i * 65536 + j;
            }
        }
        const bool visible = (tr.flags & 1) == 0 && j >= 0;
        if (visible) atomicOr(&row[j >> 5], 1u << (j & 31));
        cnt += __popc(__ballot_sync(0xFFFFFFFFu, visible));
    }
    __syncwarp();
    if (whole) {
        for (int w = lane; w < W; w += 32) bits[i * W + w] = row[w];
        if (lane == 0) count[i] = cnt;
    } else {
        for (int w = lane; w < W; w += 32)
            if (row[w]) atomicOr(&bits[i * W + w], row[w]);
        if (lane == 0) atomicAdd(&count[i], cnt);
    }
    __syncwarp();
    // rays per lane: the tiles cast, less the pad of the last tile if this
    // lane has one
    acc.rays += (t1 - t0) - (t1 == W && __float_as_int(__ldg(&tdirs[32 * (W - 1) + lane]).w) < 0 ? 1 : 0);
}

// One point by one warp, by the tree's kind: a ray per lane on the binary
// tree, pooled on the 4-wide one (with 64-bit pairs on the largest parts).
enum { kBinary = 0, kWide4 = 1, kWide4Big = 2, kWide4Seg = 3, kWide4BigSeg = 4 };   // Seg: in segments (point casts)
__host__ __device__ constexpr bool is_big(int kind) { return kind == kWide4Big || kind == kWide4BigSeg; }
__host__ __device__ constexpr bool is_seg(int kind) { return kind >= kWide4Seg; }

// Resident blocks per SM of the hemispherical cast.  The binary walk keeps no
// pool, and what it waits for are loads of its own, one ray a lane: more warps
// hide them (housing, 20k points x 1024 directions: 2.45 ms with 7, 2.50 and
// 2.66 with 6 and 5, 2.60 with 8).
constexpr int hemi_blocks(int kind) { return kind == kBinary ? 7 : RC_HEMI_MIN_BLOCKS; }

// dynamic shared memory of the axis casts (four warps)
__host__ __device__ __forceinline__ constexpr size_t axis_smem(int kind)
{
    return kind == kBinary ? 0 : 4 * (kind == kWide4 ? sizeof(AxisPoolOf<false>) : sizeof(AxisPoolOf<true>));
}

// Dynamic shared memory of the point casts: each warp's pool (4-wide tree),
// then each warp's bit rows of W words (of a segment's: kSegWords).
__host__ __device__ __forceinline__ constexpr int cast_words(int kind, int W, bool stats)
{
    return kind == kBinary ? W : pool_rows(stats) * (is_seg(kind) ? kSegWords : W);
}
__host__ __device__ __forceinline__ constexpr size_t pool_bytes(int kind)
{
    return kind == kBinary ? 0 : is_big(kind) ? sizeof(PoolOf<true>) : sizeof(PoolOf<false>);
}
__host__ __device__ __forceinline__ size_t cast_smem(int warps, int W, int kind, bool stats)
{
    return warps * (pool_bytes(kind) + cast_words(kind, W, stats) * sizeof(uint32_t));
}

// Let a kernel have the shared memory of the most directions.  The limit
// belongs to the kernel, not to a launch, and casts of other threads may have
// other direction counts: it is always set to the same value.
template <class Kernel>
static cudaError_t allow_cast_smem(Kernel kernel, int warps, int kind, bool stats)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)cast_smem(warps, kind == kWide4 || kind == kWide4Big ? kWholeWords : kMaxDirs / 32, kind, stats));
}

template <bool kStats, int kKind>
__device__ __forceinline__ void cast_point(const float4* __restrict__ nodes, const float4* __restrict__ tris,
                                           int max_steps, float scene_maxabs, const float* __restrict__ P,
                                           const float* __restrict__ Nrm, int64_t i,
                                           const float4* __restrict__ tdirs, int W, double eps, unsigned char* smem,
                                           uint32_t* __restrict__ bits, int32_t* __restrict__ count, CastAcc& acc,
                                           int t0 = 0, int t1 = -1, long long* relist = nullptr,
                                           long long relist_cap = 0, unsigned long long* relist_ctr = nullptr)
{
    const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    uint32_t* rows = (uint32_t*)(smem + warps * pool_bytes(kKind)) + warp * cast_words(kKind, W, kStats);
    if (kKind == kBinary) {
        cast_point_binary<kStats>(nodes, tris, max_steps, scene_maxabs, P, Nrm, i, tdirs, W, eps, rows, bits, count,
                                  acc, t0, t1, relist, relist_cap, relist_ctr);
        return;
    }
    const bool whole = t1 < 0;
    if (whole) t1 = W;
    auto* pool = (PoolOf<is_big(kKind)>*)smem + warp;
    static_assert(4 * sizeof(PoolOf<is_big(kKind)>) >= kMaxDirs / 32 * sizeof(uint32_t),
                  "the rows' place less a segment's first word lies in the block's shared memory still");
    if (!is_seg(kKind)) {
        cast_point_pooled<kStats, is_big(kKind), false>(nodes, tris, max_steps, scene_maxabs, P, Nrm, i, tdirs, W, eps, pool,
                                                        rows, bits, count, acc, t0, t1, whole, relist, relist_cap, relist_ctr);
        return;
    }
    if (whole) {                           // the segments add to the point's row and count
        for (int w = threadIdx.x & 31; w < W; w += 32) bits[i * W + w] = 0u;
        if ((threadIdx.x & 31) == 0) count[i] = 0;
        __syncwarp();
    }
    for (; t0 < t1; t0 += kSegTiles)
        cast_point_pooled<kStats, is_big(kKind), true>(nodes, tris, max_steps, scene_maxabs, P, Nrm, i, tdirs, W, eps, pool,
                                                       rows, bits, count, acc, t0, min(t1, t0 + kSegTiles), false, relist,
                                                       relist_cap, relist_ctr);
}

template <bool kStats, int kKind>
__global__ void __launch_bounds__(128, hemi_blocks(kKind))
k_hemisphere(const float4* __restrict__ nodes, const float4* __restrict__ tris, int max_steps, float scene_maxabs,
             const float* __restrict__ P, const float* __restrict__ Nrm, int64_t n,
             const int32_t* __restrict__ order, const float4* __restrict__ tdirs, int n_dirs, double eps,
             uint32_t* __restrict__ bits, int32_t* __restrict__ count, unsigned long long* counters,
             unsigned long long* work, int64_t n_whole, int splits, long long* relist, long long relist_cap)
{
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const int lane = threadIdx.x & 31;
    const int W = (n_dirs + 31) >> 5;
    CastAcc acc;
    // With a work counter the warps take work until none is left: the first
    // n_whole points of the processing order whole, then the last n - n_whole
    // points in `splits` parts each, so that the launch ends on short items
    // instead of whole points.  Without a counter (grid sized to the work)
    // each warp casts exactly its own point, so blocks are short-lived and
    // kernels of concurrent requests interleave.
    const unsigned long long own = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const unsigned long long items = (unsigned long long)n_whole + (unsigned long long)(n - n_whole) * splits;
    const int tw = (W + splits - 1) / splits;
    for (bool first = true;; first = false) {
        unsigned long long k = items;
        if (work) {
            if (lane == 0) k = atomicAdd(work, 1ULL);
            k = __shfl_sync(0xFFFFFFFFu, k, 0);
        } else if (first) {
            k = own;
        }
        if (k >= items) break;
        // item k: a whole point (tiles 0..W, t1 = -1) or a part of one
        int64_t r = (int64_t)k;
        int t0 = 0, t1 = -1;
        if (k >= (unsigned long long)n_whole) {
            const unsigned long long q = k - (unsigned long long)n_whole;
            r = n_whole + (int64_t)(q / splits);
            t0 = (int)(q % splits) * tw;
            t1 = min(W, t0 + tw);
            if (t0 >= t1) continue;
        }
        const int64_t i = order ? (int64_t)__ldg(&order[r]) : r;
        cast_point<kStats, kKind>(nodes, tris, max_steps, scene_maxabs, P, Nrm, i, tdirs, W, eps, s_dyn, bits, count, acc,
                                  t0, t1, relist, relist_cap, counters ? counters + 6 : nullptr);
    }
    warp_add_counters(counters, acc.rays, acc.amb, acc.retests, acc.overflow, acc.nvis + (acc.nbox + 3) / 4, acc.ntri);
}

// zero the bit rows and counts of the points cast in parts (positions
// [n_whole, n) of the processing order)
__global__ void k_zero_split(const int32_t* __restrict__ order, int64_t n_whole, int64_t n, int W,
                             uint32_t* __restrict__ bits, int32_t* __restrict__ count)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t r = n_whole + t / W;
    if (r >= n) return;
    const int64_t i = order ? (int64_t)order[r] : r;
    const int w = (int)(t % W);
    bits[i * W + w] = 0u;
    if (w == 0) count[i] = 0;
}

// ---------------------------------------------------------------------------
// Re-analysis after an edit that keeps the triangle list (reading: every
// sample point stays on its face).  The result of a ray depends only on the
// triangles it can meet; the edited triangles lie in the box [blo, bhi] in
// both the old and the new part, so a ray from an unmoved point that cannot
// enter that box (the conservative slab test of the traversal, monotone in
// the box) keeps its old bit.  Points on moved faces are cast in full; an
// unmoved point whose tangent plane has the whole box behind it (every
// hemisphere direction has d.n > 0 when its normal is of unit length, see
// tangent_shortcuts_ok) is skipped outright.  Rays whose old
// and new decisions are both made only by FP64-ambiguous pairs may differ
// from a full re-cast; they are counted as ambiguous like any other.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool ray_enters_box(const Ray& r, const float4 lo, const float4 hi)
{
    const float rob = 1.0f + 2.0f * 1.7881394e-7f;
    const bool sx = signbit(r.ix), sy = signbit(r.iy), sz = signbit(r.iz);
    const float nx = ((sx ? hi.x : lo.x) - r.ox) * r.ix, fx = ((sx ? lo.x : hi.x) - r.ox) * r.ix;
    const float ny = ((sy ? hi.y : lo.y) - r.oy) * r.iy, fy = ((sy ? lo.y : hi.y) - r.oy) * r.iy;
    const float nz = ((sz ? hi.z : lo.z) - r.oz) * r.iz, fz = ((sz ? lo.z : hi.z) - r.oz) * r.iz;
    const float tn = fmaxf(fmaxf(nx, ny), fmaxf(nz, 0.0f));
    const float tf = fminf(fminf(fx, fy), fz) * rob;
    return tn <= tf;
}

// max over the box corners of (c - o).n in FP64, with its rounding bound; in
// fp32 where the sign is clear by 50 times the rounding of the terms
__device__ __forceinline__ bool box_in_front(const float4 lo, const float4 hi, float ox, float oy, float oz, float nx,
                                             float ny, float nz)
{
    const float ax = (lo.x - ox) * nx, bx = (hi.x - ox) * nx, ay = (lo.y - oy) * ny, by = (hi.y - oy) * ny,
                az = (lo.z - oz) * nz, bz = (hi.z - oz) * nz;
    const float s = fmaxf(ax, bx) + fmaxf(ay, by) + fmaxf(az, bz);
    const float m = fmaxf(fabsf(ax), fabsf(bx)) + fmaxf(fabsf(ay), fabsf(by)) + fmaxf(fabsf(az), fabsf(bz));
    if (m < 1e30f && fabsf(s) > 1e-5f * m + 1e-30f) return s > 0.0f;
    double best = -INFINITY, mag = 0.0;
    for (int c = 0; c < 8; ++c) {
        const double x = __dsub_rn((double)((c & 1) ? hi.x : lo.x), (double)ox);
        const double y = __dsub_rn((double)((c & 2) ? hi.y : lo.y), (double)oy);
        const double z = __dsub_rn((double)((c & 4) ? hi.z : lo.z), (double)oz);
        const double a = __dmul_rn(x, (double)nx), b = __dmul_rn(y, (double)ny), e = __dmul_rn(z, (double)nz);
        best = fmax(best, __dadd_rn(__dadd_rn(a, b), e));
        mag = fmax(mag, __dadd_rn(__dadd_rn(fabs(a), fabs(b)), fabs(e)));
    }
    return best > -1e-12 * mag;
}

struct UpdateCtl {
    unsigned long long far, near, work;     // points of either kind in the list, next item
};

// list entries: the point above two bits
constexpr int kUpdMoved = 1, kUpdLevel = 2;   // on a moved face; tangent_shortcuts_ok

// The points to look at, a lane per point: from the front of `list` those
// that see the edit's box far off, from its back those on moved faces (their
// rows zeroed) and those within 2.5 half diagonals of the box's centre, many
// of whose rays are cast again.  A warp per point had every lane form the same
// FP64 sums (1/64 of the fp32 rate), 0.9 ms for 200k points; now 17 us.
__global__ void __launch_bounds__(256)
k_update_pick(const float* __restrict__ P, const float* __restrict__ Nrm, int64_t n, const int32_t* __restrict__ order,
              const int32_t* __restrict__ face, const uint8_t* __restrict__ changed, float4 blo, float4 bhi, int W,
              double eps, uint32_t* __restrict__ bits, int64_t* __restrict__ list, UpdateCtl* ctl)
{
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    bool moved = false, far = false, near = false;
    int64_t i = 0, e = 0;
    if (k < n) {
        i = order ? (int64_t)__ldg(&order[k]) : k;
        const float nx = Nrm[3 * i], ny = Nrm[3 * i + 1], nz = Nrm[3 * i + 2];
        const float px = P[3 * i], py = P[3 * i + 1], pz = P[3 * i + 2];
        moved = changed[face[i]] != 0;
        const bool level = tangent_shortcuts_ok(nx, ny, nz, W);
        const bool look = moved || !level || box_in_front(blo, bhi, offset_coord(px, nx, eps), offset_coord(py, ny, eps),
                                                          offset_coord(pz, nz, eps), nx, ny, nz);
        const float x = 0.5f * (blo.x + bhi.x) - px, y = 0.5f * (blo.y + bhi.y) - py, z = 0.5f * (blo.z + bhi.z) - pz;
        const float hx = bhi.x - blo.x, hy = bhi.y - blo.y, hz = bhi.z - blo.z;
        near = look && (moved || x * x + y * y + z * z < 1.5625f * (hx * hx + hy * hy + hz * hz));
        far = look && !near;
        e = i * 4 + (moved ? kUpdMoved : 0) + (level ? kUpdLevel : 0);
    }
    const unsigned mf = __ballot_sync(kAll, far), mn = __ballot_sync(kAll, near), below = (1u << lane) - 1u;
    unsigned long long at = 0;
    if (lane == 0 && mf) at = atomicAdd(&ctl->far, (unsigned long long)__popc(mf));
    if (lane == 1 && mn) at = atomicAdd(&ctl->near, (unsigned long long)__popc(mn));
    const long long af = (long long)__shfl_sync(kAll, at, 0), an = (long long)__shfl_sync(kAll, at, 1);
    if (far) list[af + __popc(mf & below)] = e;
    if (near) list[n - 1 - (an + __popc(mn & below))] = e;
    for (unsigned m = __ballot_sync(kAll, moved); m; m &= m - 1) {
        const int64_t r = __shfl_sync(kAll, i, __ffs(m) - 1);
        for (int w = lane; w < W; w += 32) bits[r * W + w] = 0u;
    }
}

constexpr int kUpdateRun = 4;          // tiles of a near point per item (1, 2 and 8: within 4%)
constexpr int kUpdateQueue = 64;       // rays that wait, per warp

// The rays to decide again, gathered from tiles and points until a walk has
// 32 of them.  An edit is small and seen from few tiles of a point: a lane
// compares a tile's cone (axis and cosine of the half angle, made once per
// block in shared memory) with the cone of the edit's box, and of the tiles
// left the slab test of the rays decides as before; a tile alone filled 5 to
// 10 lanes of a walk.  Near points are handed out a few tiles at a time, and
// first: whole, with a thousand rays each, they were a tail of half the time.
// A tile of a point on a moved face is 32 rays already and walks as it is
// (everything moved, 20k points x 512 directions: 1.53 ms, by way of the queue
// 1.58).  The margin of the cones covers the slab test's rounding (4e-7 of a
// distance) and normals off unit length (tilt 3 delta, delta <= 0.004 / W).
// Bound by the walks.  Edit of one blade, 1.93M triangles, 200k points x 1024
// directions: 1776 -> 730 us with the two kernels beside it.
template <bool kWide>
__global__ void __launch_bounds__(128, RC_UPDATE_MIN_BLOCKS)
k_hemisphere_update(const float4* __restrict__ nodes, const float4* __restrict__ tris, int max_steps,
                    float scene_maxabs, const float* __restrict__ P, const float* __restrict__ Nrm, int64_t n,
                    const int64_t* __restrict__ list, float4 blo, float4 bhi, const float4* __restrict__ tdirs,
                    int W, double eps, uint32_t* __restrict__ bits, unsigned long long* counters, UpdateCtl* ctl)
{
    constexpr unsigned kAll = 0xFFFFFFFFu;
    extern __shared__ float4 s_cone[];     // [W]
    __shared__ float4 s_ray[4][2][kUpdateQueue], s_onb[4][3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int t = warp; t < W; t += 4) {
        const float4 h = __ldg(&tdirs[32 * t + lane]);
        const bool on = __float_as_int(h.w) >= 0;
        float x = on ? h.x : 0.0f, y = on ? h.y : 0.0f, z = on ? h.z : 0.0f;
        for (int off = 16; off; off >>= 1) {
            x += __shfl_xor_sync(kAll, x, off);
            y += __shfl_xor_sync(kAll, y, off);
            z += __shfl_xor_sync(kAll, z, off);
        }
        const float s = rsqrtf(fmaxf(x * x + y * y + z * z, 1e-20f));
        x *= s, y *= s, z *= s;
        const float c = warp_min(on ? h.x * x + h.y * y + h.z * z : 1.0f);
        if (lane == 0) s_cone[t] = make_float4(x, y, z, fminf(c, 1.0f));
    }
    __syncthreads();
    float4* const ray_o = s_ray[warp][0];
    float4* const ray_d = s_ray[warp][1];
    float4* const onb = s_onb[warp];
    const unsigned below = (1u << lane) - 1u;
    const long long near = (long long)ctl->near, parts = (W + kUpdateRun - 1) / kUpdateRun;
    const long long items = near * parts + (long long)ctl->far;
    const float margin = 1e-4f + 0.02f / (float)W;
    CastAcc acc;
    int64_t i = 0;
    bool full = false, cull = false, more = true;
    int t0 = 0, t1 = 0, qn = 0;            // tiles [t0, t1) are still to be compared
    unsigned todo = 0;                     // of tiles [t0 - 32, t0): those left
    float bx = 0.0f, by = 0.0f, bz = 0.0f, ca = 0.0f, sa = 0.0f;   // the box's cone in the point's basis
    for (;;) {
        float4 o, d;                       // the ray to walk: from the queue, or of a tile that is cast in full
        bool walk = false;
        if (qn >= 32 || (qn > 0 && !more)) {
            const int m = min(32, qn);
            qn -= m;
            walk = lane < m;
            if (walk) {
                o = ray_o[qn + lane];
                d = ray_d[qn + lane];
            }
        } else if (!more) {
            break;
        } else if (todo == 0) {
            if (t0 >= t1) {
                // the next item
                unsigned long long k = 0;
                if (lane == 0) k = atomicAdd(&ctl->work, 1ULL);
                k = __shfl_sync(kAll, k, 0);
                if ((long long)k >= items) {
                    more = false;
                    continue;
                }
                const bool run = (long long)k < near * parts;
                const int64_t e = __ldg(&list[run ? n - 1 - (long long)k / parts : (long long)k - near * parts]);
                i = e >> 2;
                full = (e & kUpdMoved) != 0;
                t0 = run ? (int)((long long)k % parts) * kUpdateRun : 0;
                t1 = run ? min(W, t0 + kUpdateRun) : W;
                const float nx = Nrm[3 * i], ny = Nrm[3 * i + 1], nz = Nrm[3 * i + 2];
                const float ox = offset_coord(P[3 * i], nx, eps), oy = offset_coord(P[3 * i + 1], ny, eps),
                            oz = offset_coord(P[3 * i + 2], nz, eps);
                const Onb b = make_onb(nx, ny, nz);
                if (lane == 0) {
                    onb[0] = make_float4(b.t1x, b.t2x, nx, ox);
                    onb[1] = make_float4(b.t1y, b.t2y, ny, oy);
                    onb[2] = make_float4(b.t1z, b.t2z, nz, oz);
                }
                __syncwarp();
                // the box's cone: towards its centre, as wide as its corners;
                // none (no tile is left out) when a corner lies 87 degrees
                // off or more, or anything is not finite
                float mx = 0.5f * (blo.x + bhi.x) - ox, my = 0.5f * (blo.y + bhi.y) - oy, mz = 0.5f * (blo.z + bhi.z) - oz;
                const float s = rsqrtf(mx * mx + my * my + mz * mz);
                mx *= s, my *= s, mz *= s;
                const float cx = (lane & 1 ? bhi.x : blo.x) - ox, cy = (lane & 2 ? bhi.y : blo.y) - oy,
                            cz = (lane & 4 ? bhi.z : blo.z) - oz;
                const float q = (cx * mx + cy * my + cz * mz) * rsqrtf(cx * cx + cy * cy + cz * cz);
                ca = warp_min(fminf(q, 1.0f));
                cull = !full && (e & kUpdLevel) && ca > 0.05f && __all_sync(kAll, q > 0.05f);
                sa = sqrtf(fmaxf(0.0f, 1.0f - ca * ca));
                bx = b.t1x * mx + b.t1y * my + b.t1z * mz;
                by = b.t2x * mx + b.t2y * my + b.t2z * mz;
                bz = nx * mx + ny * my + nz * mz;
                continue;
            }
            bool in = t0 + lane < t1;
            if (in && cull) {
                // apart by more than the two half angles
                const float4 c = s_cone[t0 + lane];
                const float sb = sqrtf(fmaxf(0.0f, 1.0f - c.w * c.w));
                const float dot = c.x * bx + c.y * by + c.z * bz;
                in = !(dot < ca * c.w - sa * sb - margin && sa * c.w + ca * sb > 0.0f && c.w > 0.0f);
            }
            todo = __ballot_sync(kAll, in);
            t0 += 32;
            continue;
        } else {
            const int t = t0 - 32 + __ffs(todo) - 1;
            todo &= todo - 1;
            const float4 h = __ldg(&tdirs[32 * t + lane]);
            const float4 cx = onb[0], cy = onb[1], cz = onb[2];
            const Onb b = {cx.x, cy.x, cz.x, cx.y, cy.y, cz.y};
            float dx, dy, dz;
            local_to_world(b, cx.z, cy.z, cz.z, h.x, h.y, h.z, dx, dy, dz);
            bool on = __float_as_int(h.w) >= 0;
            if (!full && on) {
                Ray r;
                setup_ray(r, cx.w, cy.w, cz.w, dx, dy, dz, scene_maxabs);
                on = ray_enters_box(r, blo, bhi);       // otherwise it keeps its old bit
            }
            o = make_float4(cx.w, cy.w, cz.w, __uint_as_float((unsigned)i));
            d = make_float4(dx, dy, dz, __int_as_float(__float_as_int(h.w) | (int)(i >> 32) << 16));   // j < 65536
            if (!full) {
                const unsigned m = __ballot_sync(kAll, on);
                if (on) {
                    const int at = qn + __popc(m & below);
                    ray_o[at] = o;
                    ray_d[at] = d;
                }
                qn += __popc(m);
                __syncwarp();
                continue;
            }
            walk = on;
        }
        if (walk) {
            const int j = __float_as_int(d.w) & 0xFFFF;
            Ray r;
            setup_ray(r, o.x, o.y, o.z, d.x, d.y, d.z, scene_maxabs);
            const TraceOut tr = trace_any<false, kWide>(nodes, tris, r, max_steps);
            acc.retests += tr.retests;
            acc.overflow += tr.overflow;
            acc.amb += (tr.flags >> 1) & 1;
            acc.rays += 1;
            const int64_t at = (int64_t)__float_as_uint(o.w) | (int64_t)(__float_as_uint(d.w) >> 16) << 32;
            uint32_t* row = bits + at * W + (j >> 5);
            if ((tr.flags & 1) == 0) atomicOr(row, 1u << (j & 31));
            else atomicAnd(row, ~(1u << (j & 31)));
        }
        __syncwarp();
    }
    warp_add_counters(counters, acc.rays, acc.amb, acc.retests, acc.overflow);
}

// the counts of the listed points, 2^shift lanes per point
__global__ void __launch_bounds__(256)
k_update_count(const int64_t* __restrict__ list, int64_t n, const UpdateCtl* ctl, int W, int shift,
               const uint32_t* __restrict__ bits, int32_t* __restrict__ count)
{
    const int64_t far = (int64_t)ctl->far, all = far + (int64_t)ctl->near;
    const int sub = threadIdx.x & ((1 << shift) - 1);
    const int64_t step = ((int64_t)gridDim.x * blockDim.x) >> shift;
    for (int64_t k0 = (blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31)) >> shift; k0 < all; k0 += step) {
        const int64_t k = k0 + ((threadIdx.x & 31) >> shift);
        int cnt = 0;
        int64_t i = 0;
        if (k < all) {
            i = __ldg(&list[k < far ? k : n - 1 - (k - far)]) >> 2;
            for (int w = sub; w < W; w += 1 << shift) cnt += __popc(bits[i * W + w]);
        }
        for (int off = 1 << shift >> 1; off; off >>= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, off);
        if (k < all && sub == 0) count[i] = cnt;
    }
}

// ---------------------------------------------------------------------------
// Batched hemispherical cast: one persistent launch over the points of many
// parts.  Work items are runs of `ppi` consecutive points (in each part's
// processing order) of one part; a warp takes items from one global counter,
// finds the part by binary search over the parts' first item, and casts the
// points as k_hemisphere does.  Counters are kept per part.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void flush_part_counters(unsigned long long* c, CastAcc& a)
{
    warp_add_counters(c, a.rays, a.amb, a.retests, a.overflow);
    a = CastAcc();
}

template <bool kStats, int kKind>
__global__ void __launch_bounds__(128, RC_BATCH_MIN_BLOCKS)
k_batch(const BatchPart* __restrict__ parts, int n_parts, long long n_items, int ppi,
        const float4* __restrict__ tdirs, int n_dirs, double eps, unsigned long long* work)
{
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const int lane = threadIdx.x & 31;
    const int W = (n_dirs + 31) >> 5;
    CastAcc acc;
    int cur = -1;
    for (;;) {
        unsigned long long k = 0;
        if (lane == 0) k = atomicAdd(work, 1ULL);
        k = __shfl_sync(0xFFFFFFFFu, k, 0);
        if (k >= (unsigned long long)n_items) break;
        int lo = 0, hi = n_parts - 1;            // last part with first_item <= k
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((unsigned long long)parts[mid].first_item <= k) lo = mid; else hi = mid - 1;
        }
        const BatchPart& bp = parts[lo];
        if (lo != cur) {
            if (cur >= 0) flush_part_counters(parts[cur].counters, acc);
            cur = lo;
        }
        const long long q0 = ((long long)k - bp.first_item) * ppi;
        const long long q1 = q0 + ppi < bp.n ? q0 + ppi : bp.n;
        for (long long q = q0; q < q1; ++q) {
            const int64_t i = bp.order ? (int64_t)__ldg(&bp.order[q]) : (int64_t)q;
            cast_point<kStats, kKind>(bp.nodes, bp.tris, bp.max_steps, bp.scene_maxabs, bp.P, bp.N, i, tdirs, W, eps,
                                      s_dyn, bp.bits, bp.count, acc);
        }
    }
    if (cur >= 0) flush_part_counters(parts[cur].counters, acc);
}

// ---------------------------------------------------------------------------
// Section 3.2: orthogonal cast along the six frame axes (+X', -X', +Y', -Y',
// +Z', -Z').  A work item (frame f, axis a, group g) is 32 consecutive points
// of the Morton processing order cast along one axis, one ray per lane --
// parallel rays from neighbouring origins.  Warps take items one at a time
// from a counter, because a few rays that graze a surface parallel to an axis
// (along a fillet or a bore) take far longer than the rest.  Travel to the
// frame bounding box is FP64.  Frame f writes travel[f n + i][6]; reachable
// bits gather in mbits[f n + i] (zeroed by the caller) and are packed into
// mask[f n + i] afterwards.
// ---------------------------------------------------------------------------
template <bool kStats, int kKind>
__global__ void __launch_bounds__(128, RC_AXIS_MIN_BLOCKS)
k_orthogonal_axis(const float4* __restrict__ nodes, const float4* __restrict__ tris, int max_steps,
                  float scene_maxabs, const float* __restrict__ P, const float* __restrict__ Nrm, int64_t n,
                  const int32_t* __restrict__ order, const FrameDev* __restrict__ fds, int nf, double eps,
                  double par_tol, uint32_t* __restrict__ mbits, float* __restrict__ travel,
                  unsigned long long* counters, unsigned long long* work)
{
    extern __shared__ __align__(16) unsigned char s_axis[];
    auto* pool = (AxisPoolOf<kKind == kWide4Big>*)s_axis + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    AxisAcc acc;
    const int64_t G = (n + 31) >> 5;
    const int64_t items = (int64_t)nf * 6 * G;
    // without a work counter (grid sized to the work) each warp casts only
    // its own item, so blocks stay short and concurrent requests interleave
    const unsigned long long own = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    for (bool first = true;; first = false) {
        unsigned long long w = (unsigned long long)items;
        if (work) {
            if (lane == 0) w = atomicAdd(work, 1ULL);
            w = __shfl_sync(0xFFFFFFFFu, w, 0);
        } else if (first) {
            w = own;
        }
        const int64_t it = (int64_t)w;
        if (it >= items) break;
        const int fa = (int)(it / G);
        const int64_t g = it - (int64_t)fa * G;
        const int f = fa / 6, a = fa - 6 * f;
        const int64_t k = g * 32 + lane;
        const bool on = k < n;
        bool cast = false;
        int64_t row = 0;
        float ox = 0.0f, oy = 0.0f, oz = 0.0f;
        const float* axes = fds[f].axes;
        const float dx = axes[3 * a], dy = axes[3 * a + 1], dz = axes[3 * a + 2];
        if (on) {
            const int64_t i = order ? (int64_t)__ldg(&order[k]) : k;
            const float px = P[3 * i], py = P[3 * i + 1], pz = P[3 * i + 2];
            const float nx = Nrm[3 * i], ny = Nrm[3 * i + 1], nz = Nrm[3 * i + 2];
            const double* frame = fds[f].frame;
            const double* fbox = fds[f].fbox;
            row = (int64_t)f * n + i;
            const int kk = a >> 1;
            double q = __dadd_rn(__dmul_rn((double)px, frame[kk]), __dmul_rn((double)py, frame[3 + kk]));
            q = __dadd_rn(q, __dmul_rn((double)pz, frame[6 + kk]));
            const double tv = (a & 1) ? __dsub_rn(q, fbox[kk]) : __dsub_rn(fbox[3 + kk], q);
            travel[6 * row + a] = __double2float_rn(tv);
            cast = eligible(nx, ny, nz, dx, dy, dz, par_tol);
            ox = offset_coord(px, nx, eps);
            oy = offset_coord(py, ny, eps);
            oz = offset_coord(pz, nz, eps);
        }
        // every lane: the pooled walk tests other lanes' rays of this direction
        Ray r;
        setup_ray(r, ox, oy, oz, dx, dy, dz, scene_maxabs);
        AxisRay ar = {};
        if (kKind != kBinary && cast) ar = make_axis_ray(fds[f], a, ox, oy, oz, r.rs);
        bool blocked = false;
        if (kKind == kBinary) {
            if (cast) {
                const TraceOut t = trace<kStats>(nodes, tris, r, max_steps);
                acc.retests += t.retests;
                acc.overflow += t.overflow;
                acc.amb += (t.flags >> 1) & 1;
                acc.rays += 1;
                if (kStats) { acc.nvis += t.nodes; acc.ntri += t.tris; }
                blocked = t.flags & 1;
            }
        } else {
            blocked = trace_axis<kStats>(fds[f].tree, tris, r, ar, cast, scene_maxabs, max_steps, pool, acc);
        }
        if (cast && !blocked) atomicOr(&mbits[row], 1u << a);
    }
    warp_add_counters(counters, acc.rays, acc.amb, acc.retests, acc.overflow, acc.nvis, acc.ntri);
}

__global__ void k_mask_pack(const uint32_t* __restrict__ mbits, int64_t m, uint8_t* __restrict__ mask)
{
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r < m) mask[r] = (uint8_t)mbits[r];
}

// ---------------------------------------------------------------------------
// Tool-aware accessibility (a reading of the accessibility cones of the prior
// art the paper cites; the paper itself casts thin rays).  A ball-end tool of
// radius r touches the point: centre c = p + (r + eps) n (FP64).  Along axis
// a its shank is sampled by the ray from c and K rays from the ring
// c + r (cos t_k u + sin t_k v), (u, v) the branchless orthonormal basis of
// a (Duff et al. 2017) in FP64; origins are rounded to fp32, every ray goes
// along a.  The axis is tool-accessible iff it is eligible (n.a >=
// -parallel_tol) and none of the 1 + K rays is obstructed.  Work items are
// (axis, 32 consecutive points) as in the orthogonal cast; accessible bits
// gather in mbits[i] (zeroed by the caller).
// ---------------------------------------------------------------------------
template <int kKind>
__global__ void __launch_bounds__(128, RC_AXIS_MIN_BLOCKS)
k_tool_cast_axis(const float4* __restrict__ nodes, const float4* __restrict__ tris, int max_steps,
                 float scene_maxabs, const float* __restrict__ P, const float* __restrict__ Nrm, int64_t n,
                 const int32_t* __restrict__ order, const FrameDev* __restrict__ fd, double eps, double par_tol,
                 double radius, const double2* __restrict__ ring /*cos, sin*/, int K, uint32_t* __restrict__ mbits,
                 unsigned long long* counters, unsigned long long* work)
{
    extern __shared__ __align__(16) unsigned char s_axis[];
    auto* pool = (AxisPoolOf<kKind == kWide4Big>*)s_axis + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    AxisAcc acc;
    const int64_t G = (n + 31) >> 5;
    const int64_t items = 6 * G;
    for (;;) {
        unsigned long long w = 0;
        if (lane == 0) w = atomicAdd(work, 1ULL);
        const int64_t it = (int64_t)__shfl_sync(0xFFFFFFFFu, w, 0);
        if (it >= items) break;
        const int a = (int)(it / G);
        const int64_t k = (it - (int64_t)a * G) * 32 + lane;
        const float dx = fd->axes[3 * a], dy = fd->axes[3 * a + 1], dz = fd->axes[3 * a + 2];
        bool open = k < n;
        int64_t i = 0;
        double cx = 0.0, cy = 0.0, cz = 0.0;
        if (open) {
            i = order ? (int64_t)__ldg(&order[k]) : k;
            const double px = P[3 * i], py = P[3 * i + 1], pz = P[3 * i + 2];
            const double nx = Nrm[3 * i], ny = Nrm[3 * i + 1], nz = Nrm[3 * i + 2];
            open = eligible(Nrm[3 * i], Nrm[3 * i + 1], Nrm[3 * i + 2], dx, dy, dz, par_tol);
            const double h = __dadd_rn(radius, eps);
            cx = __dadd_rn(px, __dmul_rn(h, nx));
            cy = __dadd_rn(py, __dmul_rn(h, ny));
            cz = __dadd_rn(pz, __dmul_rn(h, nz));
        }
        // orthonormal basis (u, v) of the axis, FP64
        const double ax = dx, ay = dy, az = dz;
        const double sg = az >= 0.0 ? 1.0 : -1.0;
        const double q = __ddiv_rn(-1.0, __dadd_rn(sg, az));
        const double bb = __dmul_rn(__dmul_rn(ax, ay), q);
        const double ux = __dadd_rn(1.0, __dmul_rn(__dmul_rn(__dmul_rn(sg, ax), ax), q));
        const double uy = __dmul_rn(sg, bb), uz = __dmul_rn(-sg, ax);
        const double vx = bb, vy = __dadd_rn(sg, __dmul_rn(__dmul_rn(ay, ay), q)), vz = -ay;
        // the warp's rays of one ring position at a time, for the points still open
        for (int r = -1; r < K && __any_sync(0xFFFFFFFFu, open); ++r) {
            float ox = 0.0f, oy = 0.0f, oz = 0.0f;
            if (open) {
                if (r < 0) {
                    ox = __double2float_rn(cx);
                    oy = __double2float_rn(cy);
                    oz = __double2float_rn(cz);
                } else {
                    const double rc = __dmul_rn(radius, ring[r].x), rs = __dmul_rn(radius, ring[r].y);
                    ox = __double2float_rn(__dadd_rn(__dadd_rn(cx, __dmul_rn(rc, ux)), __dmul_rn(rs, vx)));
                    oy = __double2float_rn(__dadd_rn(__dadd_rn(cy, __dmul_rn(rc, uy)), __dmul_rn(rs, vy)));
                    oz = __double2float_rn(__dadd_rn(__dadd_rn(cz, __dmul_rn(rc, uz)), __dmul_rn(rs, vz)));
                }
            }
            Ray ray;
            setup_ray(ray, ox, oy, oz, dx, dy, dz, scene_maxabs);
            AxisRay ar = {};
            if (kKind != kBinary && open) ar = make_axis_ray(*fd, a, ox, oy, oz, ray.rs);
            if (kKind == kBinary) {
                if (open) {
                    const TraceOut t = trace<false>(nodes, tris, ray, max_steps);
                    acc.retests += t.retests;
                    acc.overflow += t.overflow;
                    acc.amb += (t.flags >> 1) & 1;
                    acc.rays += 1;
                    open = (t.flags & 1) == 0;
                }
            } else {
                // called by every lane: the walk is the whole warp's
                const bool blocked = trace_axis<false>(fd->tree, tris, ray, ar, open, scene_maxabs, max_steps, pool, acc);
                open = open && !blocked;
            }
        }
        if (open) atomicOr(&mbits[i], 1u << a);
    }
    warp_add_counters(counters, acc.rays, acc.amb, acc.retests, acc.overflow);
}

// Vertex bounding boxes in the frames' coordinates (FP64, exact; the frames
// are fp32 matrices): block (x, f) takes vertices for frame f.  A warp takes
// 256 vertices at a time: in fp32 their extremes, then FP64 (1/64 of the fp32
// rate) only for those within 2^-19 S of one, S >= sum |x_i f_i| of every
// vertex of the 256.  The fp32 coordinate is within 4.1 u S of the FP64 one,
// so the FP64 extreme lies within 8.2 u S = 2^-20.9 S of the fp32 one.  The
// last block converts the sums.  101k vertices: 22 us and 8 us for two
// kernels beside it per frame -> 20 us for five frames.
__global__ void __launch_bounds__(256)
k_frame_box(const float* __restrict__ V, int64_t nV, FrameDev* __restrict__ frames)
{
    __shared__ long long s_box[6];
    __shared__ bool s_last;
    FrameDev* const d = frames + blockIdx.y;
    if (threadIdx.x < 6) s_box[threadIdx.x] = threadIdx.x < 3 ? 0x7FFFFFFFFFFFFFFFLL : (long long)0x8000000000000000ULL;
    __syncthreads();
    float g[9];
    for (int k = 0; k < 3; ++k)
        for (int c = 0; c < 3; ++c) g[3 * c + k] = d->axes[6 * k + c];
    const int lane = threadIdx.x & 31;
    long long lo[3], hi[3];
    for (int k = 0; k < 3; ++k) {
        lo[k] = 0x7FFFFFFFFFFFFFFFLL;
        hi[k] = (long long)0x8000000000000000ULL;
    }
    const int64_t step = (int64_t)gridDim.x * 8 * 256;
    for (int64_t v0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * 256; v0 < nV; v0 += step) {
        float x[8], y[8], z[8], ax = 0.0f, ay = 0.0f, az = 0.0f;
        for (int r = 0; r < 8; ++r) {
            const int64_t v = min64(v0 + 32 * r + lane, nV - 1);
            x[r] = V[3 * v], y[r] = V[3 * v + 1], z[r] = V[3 * v + 2];
            ax = fmaxf(ax, fabsf(x[r])), ay = fmaxf(ay, fabsf(y[r])), az = fmaxf(az, fabsf(z[r]));
        }
        ax = warp_max(ax), ay = warp_max(ay), az = warp_max(az);
        for (int k = 0; k < 3; ++k) {
            float q[8], mn = INFINITY, mx = -INFINITY;
            for (int r = 0; r < 8; ++r) {
                q[r] = fmaf(x[r], g[k], fmaf(y[r], g[3 + k], z[r] * g[6 + k]));
                mn = fminf(mn, q[r]), mx = fmaxf(mx, q[r]);
            }
            const float w = 1.9073486328125e-06f * (ax * fabsf(g[k]) + ay * fabsf(g[3 + k]) + az * fabsf(g[6 + k]));
            mn = warp_min(mn) + w, mx = warp_max(mx) - w;
            for (int r = 0; r < 8; ++r)
                if (!(q[r] > mn && q[r] < mx)) {
                    double t = __dadd_rn(__dmul_rn(widen(x[r]), (double)g[k]), __dmul_rn(widen(y[r]), (double)g[3 + k]));
                    t = __dadd_rn(t, __dmul_rn(widen(z[r]), (double)g[6 + k]));
                    const long long o = double_to_ordered(t);
                    lo[k] = min(lo[k], o), hi[k] = max(hi[k], o);
                }
        }
    }
    for (int k = 0; k < 3; ++k)
        if (lo[k] <= hi[k]) {
            atomicMin(&s_box[k], lo[k]);
            atomicMax(&s_box[3 + k], hi[k]);
        }
    __syncthreads();
    if (threadIdx.x < 3) atomicMin(&d->box[threadIdx.x], s_box[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(&d->box[threadIdx.x], s_box[threadIdx.x]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&d->done, 1u) + 1 == gridDim.x;
    __syncthreads();
    if (s_last && threadIdx.x < 6) {
        __threadfence();
        d->fbox[threadIdx.x] = ordered_to_double(*(volatile long long*)&d->box[threadIdx.x]);
    }
}

// ---------------------------------------------------------------------------
// host drivers
// ---------------------------------------------------------------------------
static int max_steps(rc_bvh h) { return (int)(2 * (h->n_int + h->T) + 64); }

// the 4-wide tree is the default; tree_width 2 selects the binary tree
bool use_wide(const rc_params* p) { return p->tree_width != 2; }

// the point casts' walk: 32-bit pairs wherever a code fits (see PairOf)
static int cast_kind(const rc_params* p, int64_t max_tris)
{
    return !use_wide(p) ? kBinary : max_tris <= kPairTris ? kWide4 : kWide4Big;
}

// and, with more directions than a point's rows should hold, in segments
static int point_kind(const rc_params* p, int64_t max_tris)
{
    const int kind = cast_kind(p, max_tris);
    return kind == kBinary || (p->n_dirs + 31) / 32 <= kWholeWords ? kind : kind == kWide4 ? kWide4Seg : kWide4BigSeg;
}

static int g_sm_count = 0;

static int sm_count()
{
    if (g_sm_count == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sm_count, cudaDevAttrMultiProcessorCount, dev);
        if (g_sm_count <= 0) g_sm_count = 1;
    }
    return g_sm_count;
}

rc_status point_order(rc_bvh h, const float* P, int64_t n, int32_t* order, cudaStream_t s);

// device scratch of a launch, freed in stream order when the scope ends
struct LaunchScratch {
    cudaStream_t s;
    void* p[3] = {nullptr, nullptr, nullptr};
    ~LaunchScratch()
    {
        for (void* q : p)
            if (q) cudaFreeAsync(q, s);
    }
};

rc_status launch_hemisphere(rc_bvh h, const float* P, const float* N, int64_t n, const float4* tdirs, const rc_params* p,
                            uint32_t* bits, int32_t* count, unsigned long long* counters, bool stats,
                            cudaStream_t s, long long* relist, long long relist_cap)
{
    LaunchScratch ls{s};
    unsigned long long* work = nullptr;
    if (p->launch_mode == 0) {
        RC_CUDA(cudaMallocAsync(&work, sizeof(unsigned long long), s));
        ls.p[0] = work;
        RC_CUDA(cudaMemsetAsync(work, 0, sizeof(unsigned long long), s));
    }
    int32_t* order = nullptr;
    if (p->point_order == 0 && n > 1) {
        RC_CUDA(cudaMallocAsync(&order, sizeof(int32_t) * n, s));
        ls.p[1] = order;
        rc_status st = point_order(h, P, n, order, s);
        if (st != RC_OK) return st;
    }
    const int threads = 128;
    const int kind = point_kind(p, h->T);
    const int per_sm = p->blocks_per_sm > 0 ? p->blocks_per_sm : hemi_blocks(kind);
    int64_t blocks = (int64_t)sm_count() * per_sm;
    if (p->launch_mode == 1) work = nullptr;
    const bool wide = use_wide(p);
    const size_t smem = cast_smem(threads / 32, (p->n_dirs + 31) / 32, kind, stats);
    const float4* tree = wide ? h->wnodes : h->nodes;
    {
        // the last points (RC_TAIL_POINTS per resident warp) are cast in parts;
        // with a grid sized to the work (one item per warp) the parts are the
        // highest blocks, which the block scheduler starts last.  Few points
        // go out in more parts, down to a tile each, until there are two per
        // resident warp, although each part finds its frontier anew (37
        // points x 2048 directions in 4, 16, 32 and 64 parts: 365, 187, 137
        // and 117 us; 200 points in 4, 15, 30: 367, 207, 192; 1,000 x 1024
        // in 4, 6: 275, 268; from 1,500 points on four parts fill the
        // chip).  Not for a grid sized to the work, which shares the GPU.
        const int W = (p->n_dirs + 31) / 32;
        const int64_t resident_warps = (int64_t)sm_count() * per_sm * (threads / 32);
        int splits = std::min(RC_TAIL_SPLITS, W);
        if (work && n > 0) splits = (int)std::max<int64_t>(splits, std::min<int64_t>(2 * resident_warps / n, W));
        int64_t n_split = splits > 1 ? std::min<int64_t>(n, RC_TAIL_POINTS * resident_warps) : 0;
        if (n_split == 0) splits = 1;
        const int64_t need = std::max<int64_t>(1, (((n - n_split) + n_split * splits) * 32 + threads - 1) / threads);
        if (!work && need > 0x7FFFFFFF) return set_error(RC_E_UNSUPPORTED, "too many points for one launch");
        if (!work || blocks > need) blocks = need;
        if (n_split > 0) {
            k_zero_split<<<(unsigned)((n_split * W + 255) / 256), 256, 0, s>>>(order, n - n_split, n, W, bits, count);
            RC_LAUNCHED();
        }
        const auto run = [&](auto kernel) -> rc_status {
            if (smem > 48 * 1024) RC_CUDA(allow_cast_smem(kernel, threads / 32, kind, stats));
            kernel<<<(unsigned)blocks, threads, smem, s>>>(tree, h->tris, max_steps(h), h->scene_maxabs, P, N, n, order,
                                                           tdirs, p->n_dirs, p->origin_offset, bits, count, counters,
                                                           work, n - n_split, splits, relist, relist_cap);
            return RC_OK;
        };
        const auto pick = [&](auto with, auto without) { return run(stats ? with : without); };
        rc_status st = RC_OK;
        if (kind == kWide4) st = pick(k_hemisphere<true, kWide4>, k_hemisphere<false, kWide4>);
        else if (kind == kBinary) st = pick(k_hemisphere<true, kBinary>, k_hemisphere<false, kBinary>);
        else if (kind == kWide4Big) st = pick(k_hemisphere<true, kWide4Big>, k_hemisphere<false, kWide4Big>);
        else if (kind == kWide4Seg) st = pick(k_hemisphere<true, kWide4Seg>, k_hemisphere<false, kWide4Seg>);
        else st = pick(k_hemisphere<true, kWide4BigSeg>, k_hemisphere<false, kWide4BigSeg>);
        if (st != RC_OK) return st;
    }
    RC_LAUNCHED();
    return RC_OK;
}

// Re-analysis of the points after an edit (see k_hemisphere_update); bits
// and count hold the old results on entry.
rc_status launch_hemisphere_update(rc_bvh h, const float* P, const float* N, int64_t n, const int32_t* face,
                                   const uint8_t* changed, const float box[6], const float4* tdirs,
                                   const rc_params* p, uint32_t* bits, int32_t* count, unsigned long long* counters,
                                   cudaStream_t s)
{
    LaunchScratch ls{s};
    UpdateCtl* ctl = nullptr;              // and the list of points behind it
    RC_CUDA(cudaMallocAsync(&ctl, sizeof(UpdateCtl) + sizeof(int64_t) * n, s));
    ls.p[0] = ctl;
    int64_t* list = (int64_t*)(ctl + 1);
    RC_CUDA(cudaMemsetAsync(ctl, 0, sizeof(UpdateCtl), s));
    int32_t* order = nullptr;
    if (p->point_order == 0 && n > 1) {
        RC_CUDA(cudaMallocAsync(&order, sizeof(int32_t) * n, s));
        ls.p[1] = order;
        rc_status st = point_order(h, P, n, order, s);
        if (st != RC_OK) return st;
    }
    const int threads = 128;
    const int per_sm = p->blocks_per_sm > 0 ? p->blocks_per_sm : RC_UPDATE_MIN_BLOCKS;
    int64_t blocks = (int64_t)sm_count() * per_sm;
    const int W = (p->n_dirs + 31) / 32;
    const int64_t need = (n * ((W + kUpdateRun - 1) / kUpdateRun) * 32 + threads - 1) / threads;   // every point moved
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    const size_t smem = sizeof(float4) * W;                    // 32 KB at most
    const float4 lo = make_float4(box[0], box[1], box[2], 0.0f), hi = make_float4(box[3], box[4], box[5], 0.0f);
    k_update_pick<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(P, N, n, order, face, changed, lo, hi, W, p->origin_offset,
                                                             bits, list, ctl);
    RC_LAUNCHED();
    if (use_wide(p))
        k_hemisphere_update<true><<<(unsigned)blocks, threads, smem, s>>>(h->wnodes, h->tris, max_steps(h),
                                                                         h->scene_maxabs, P, N, n, list, lo, hi, tdirs,
                                                                         W, p->origin_offset, bits, counters, ctl);
    else
        k_hemisphere_update<false><<<(unsigned)blocks, threads, smem, s>>>(h->nodes, h->tris, max_steps(h),
                                                                          h->scene_maxabs, P, N, n, list, lo, hi, tdirs,
                                                                          W, p->origin_offset, bits, counters, ctl);
    RC_LAUNCHED();
    int shift = 0;
    while (shift < 5 && (1 << shift) < W) ++shift;
    const int64_t cblocks = std::min<int64_t>(((n << shift) + 255) / 256, 8 * (int64_t)sm_count());
    k_update_count<<<(unsigned)cblocks, 256, 0, s>>>(list, n, ctl, W, shift, bits, count);
    RC_LAUNCHED();
    return RC_OK;
}

// block f: frame f, an entry per lane
__global__ void k_frame_init(const __grid_constant__ FrameArgs a, FrameDev* frames)
{
    const int t = threadIdx.x, j = t / 3, k = t % 3;
    const float* f = a.f[blockIdx.x];
    FrameDev* d = frames + blockIdx.x;
    if (t < 9) {
        const auto product = [&](int a, int b) {
            return __dadd_rn(__dadd_rn(__dmul_rn((double)f[a], (double)f[b]), __dmul_rn((double)f[3 + a], (double)f[3 + b])),
                             __dmul_rn((double)f[6 + a], (double)f[6 + b]));
        };
        const double gram = product(j, k);
        d->frame[t] = (double)f[t];
        // its rounding, 1e-15 of the columns' lengths at most, is on top
        d->gram_up[t] = __double2float_ru(fabs(gram) + 1e-15 * sqrt(product(j, j)) * sqrt(product(k, k)));
        if (j == k) d->rlen[j] = __double2float_ru(1.01 / sqrt(gram));
    }
    if (t < 18) d->axes[t] = (t / 3) & 1 ? -f[3 * k + t / 6] : f[3 * k + t / 6];
    if (t < 6) d->box[t] = t < 3 ? 0x7FFFFFFFFFFFFFFFLL : (long long)0x8000000000000000ULL;
    if (t < 3) {
        d->c32[t] = __double2float_rn(a.sc_c[t]);
    }
    if (t == 0) {
        d->tree = a.tree[blockIdx.x];
        d->r32 = __double2float_ru(a.sc_r);
        d->done = 0;
    }
}

// Frame axes, frame matrices (FP64) and the vertices' frame bounding boxes,
// all on the device; the frames travel as kernel arguments (no host copy).
rc_status frame_setups(rc_bvh h, const float (*f9)[9], const float4* const* trees, int nf, FrameDev* d, cudaStream_t s)
{
    FrameArgs a = {};
    for (int f = 0; f < nf; ++f) {
        for (int k = 0; k < 9; ++k) a.f[f][k] = f9[f][k];
        a.tree[f] = trees && trees[f] ? trees[f] : h->wnodes;
    }
    double r2 = 0.0;
    for (int j = 0; j < 3; ++j) {
        a.sc_c[j] = 0.5 * ((double)h->lo[j] + (double)h->hi[j]);
        r2 += ((double)h->hi[j] - (double)h->lo[j]) * ((double)h->hi[j] - (double)h->lo[j]);
    }
    a.sc_r = 0.5 * sqrt(r2);
    k_frame_init<<<nf, 32, 0, s>>>(a, d);
    RC_LAUNCHED();
    const int64_t fb = std::min<int64_t>((h->nV + 2047) / 2048, (int64_t)sm_count() * 4);
    k_frame_box<<<dim3((unsigned)std::max<int64_t>(fb, 1), nf), 256, 0, s>>>(h->V, h->nV, d);
    RC_LAUNCHED();
    return RC_OK;
}

rc_status frame_setup_f(rc_bvh h, const float* f9, FrameDev* d, cudaStream_t s, const float4* tree)
{
    return frame_setups(h, (const float(*)[9])f9, &tree, 1, d, s);
}

rc_status frame_setup(rc_bvh h, const rc_params* p, FrameDev* d, cudaStream_t s, const float4* tree)
{
    return frame_setup_f(h, p->frame, d, s, tree);
}

bool is_identity_frame(const float f9[9])
{
    for (int k = 0; k < 9; ++k)
        if (f9[k] != ((k % 4) == 0 ? 1.0f : 0.0f)) return false;
    return true;
}

rc_status make_frame_tree(rc_bvh h, const float f9[9], const rc_params* p, float4** ftree, cudaStream_t s)
{
    *ftree = nullptr;
    if (!use_wide(p) || is_identity_frame(f9)) return RC_OK;
    const int64_t nodes = h->host_sc.wide_nodes > 0 ? h->host_sc.wide_nodes : h->n_int;
    RC_CUDA(cudaMallocAsync(ftree, sizeof(float4) * 8 * nodes, s));
    const rc_status st = frame_tree(h, f9, *ftree, s);
    if (st != RC_OK) {
        cudaFreeAsync(*ftree, s);
        *ftree = nullptr;
    }
    return st;
}

// Orthogonal cast of n points in nf frames (fds: device array of nf set-up
// frames); mask [nf][n], travel [nf][n][6].
// Orthogonal cast into caller-provided scratch: order (n points in their
// processing order, or null for index order; filled by the caller) and
// mbits (ortho_scratch_words(nf, n) words, cleared here).  Allocates nothing,
// so it can be captured in a graph.
int64_t ortho_scratch_words(int nf, int64_t n) { return ((((int64_t)nf * n) + 1) & ~(int64_t)1) + 2; }

rc_status launch_orthogonal_frames_into(rc_bvh h, const float* P, const float* N, int64_t n, const rc_params* p,
                                        const FrameDev* fds, int nf, uint8_t* mask, float* travel,
                                        unsigned long long* counters, const int32_t* order, uint32_t* mbits,
                                        cudaStream_t s)
{
    if (n == 0) return RC_OK;
    const int64_t m = (int64_t)nf * n;
    const int64_t mw = (m + 1) & ~(int64_t)1;   // m words, then the item counter
    RC_CUDA(cudaMemsetAsync(mbits, 0, sizeof(uint32_t) * (mw + 2), s));
    unsigned long long* work = (unsigned long long*)(mbits + mw);
    const int64_t items = (int64_t)nf * 6 * ((n + 31) / 32);
    const int kind = cast_kind(p, h->T);
    const int64_t cap = (int64_t)sm_count() * RC_AXIS_MIN_BLOCKS;
    int64_t blocks = (items + 3) / 4;
    if (blocks > cap && p->launch_mode == 0) blocks = cap;
    if (p->launch_mode == 1) work = nullptr;
    const float4* tree = use_wide(p) ? h->wnodes : h->nodes;
    const auto run = [&](auto kernel) {
        kernel<<<(unsigned)blocks, 128, axis_smem(kind), s>>>(tree, h->tris, max_steps(h), h->scene_maxabs, P, N, n, order,
                                                             fds, nf, p->origin_offset, p->parallel_tol, mbits, travel,
                                                             counters, work);
    };
    const bool stats = p->collect_stats != 0;
    if (kind == kWide4) stats ? run(k_orthogonal_axis<true, kWide4>) : run(k_orthogonal_axis<false, kWide4>);
    else if (kind == kBinary) stats ? run(k_orthogonal_axis<true, kBinary>) : run(k_orthogonal_axis<false, kBinary>);
    else stats ? run(k_orthogonal_axis<true, kWide4Big>) : run(k_orthogonal_axis<false, kWide4Big>);
    RC_LAUNCHED();
    k_mask_pack<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(mbits, m, mask);
    RC_LAUNCHED();
    return RC_OK;
}

rc_status launch_orthogonal_frames(rc_bvh h, const float* P, const float* N, int64_t n, const rc_params* p,
                                   const FrameDev* fds, int nf, uint8_t* mask, float* travel,
                                   unsigned long long* counters, cudaStream_t s)
{
    if (n == 0) return RC_OK;
    LaunchScratch ls{s};
    int32_t* order = nullptr;
    if (p->point_order == 0 && n > 1) {
        RC_CUDA(cudaMallocAsync(&order, sizeof(int32_t) * n, s));
        ls.p[0] = order;
        rc_status pst = point_order(h, P, n, order, s);
        if (pst != RC_OK) return pst;
    }
    uint32_t* mbits = nullptr;
    RC_CUDA(cudaMallocAsync(&mbits, sizeof(uint32_t) * ortho_scratch_words(nf, n), s));
    ls.p[1] = mbits;
    return launch_orthogonal_frames_into(h, P, N, n, p, fds, nf, mask, travel, counters, order, mbits, s);
}

rc_status launch_orthogonal(rc_bvh h, const float* P, const float* N, int64_t n, const rc_params* p,
                            uint8_t* mask, float* travel, unsigned long long* counters, cudaStream_t s)
{
    FrameDev* fd = nullptr;
    float4* ftree = nullptr;
    RC_CUDA(cudaMallocAsync(&fd, sizeof(FrameDev), s));
    rc_status st = n > 0 ? make_frame_tree(h, p->frame, p, &ftree, s) : RC_OK;
    if (st == RC_OK) st = frame_setup(h, p, fd, s, ftree);
    if (st == RC_OK) st = launch_orthogonal_frames(h, P, N, n, p, fd, 1, mask, travel, counters, s);
    if (ftree) cudaFreeAsync(ftree, s);
    cudaFreeAsync(fd, s);
    return st;
}

// RC_LAUNCHED without the early return
static rc_status launch_status()
{
    count_launch();
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? RC_OK : cuda_error(e, "kernel launch");
}

rc_status launch_tool_cast(rc_bvh h, const float* P, const float* N, int64_t n, const rc_params* p, double radius,
                          const double2* ring, int K, uint8_t* mask, unsigned long long* counters, cudaStream_t s)
{
    if (n == 0) return RC_OK;
    FrameDev* fd = nullptr;
    int32_t* order = nullptr;
    uint32_t* mbits = nullptr;                     // n words, then the item counter
    const int64_t mw = (n + 1) & ~(int64_t)1;
    cudaError_t e = cudaMallocAsync(&fd, sizeof(FrameDev), s);
    if (e == cudaSuccess && p->point_order == 0 && n > 1) e = cudaMallocAsync(&order, sizeof(int32_t) * n, s);
    if (e == cudaSuccess) e = cudaMallocAsync(&mbits, sizeof(uint32_t) * (mw + 2), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(mbits, 0, sizeof(uint32_t) * (mw + 2), s);
    rc_status st = e == cudaSuccess ? RC_OK : cuda_error(e, "tool cast scratch");
    float4* ftree = nullptr;
    if (st == RC_OK) st = make_frame_tree(h, p->frame, p, &ftree, s);
    if (st == RC_OK) st = frame_setup(h, p, fd, s, ftree);
    if (st == RC_OK && order) st = point_order(h, P, n, order, s);
    if (st == RC_OK) {
        int64_t blocks = (6 * ((n + 31) / 32) + 3) / 4;
        const int kind = cast_kind(p, h->T);
        const int64_t cap = (int64_t)sm_count() * RC_AXIS_MIN_BLOCKS;
        if (blocks > cap) blocks = cap;
        unsigned long long* work = (unsigned long long*)(mbits + mw);
        const auto kernel = kind == kWide4 ? k_tool_cast_axis<kWide4> : kind == kBinary ? k_tool_cast_axis<kBinary>
                                                                                      : k_tool_cast_axis<kWide4Big>;
        kernel<<<(unsigned)blocks, 128, axis_smem(kind), s>>>(use_wide(p) ? h->wnodes : h->nodes, h->tris, max_steps(h),
                                                             h->scene_maxabs, P, N, n, order, fd, p->origin_offset,
                                                             p->parallel_tol, radius, ring, K, mbits, counters, work);
        st = launch_status();
    }
    if (st == RC_OK) {
        k_mask_pack<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(mbits, n, mask);
        st = launch_status();
    }
    if (mbits) cudaFreeAsync(mbits, s);
    if (order) cudaFreeAsync(order, s);
    if (ftree) cudaFreeAsync(ftree, s);
    if (fd) cudaFreeAsync(fd, s);
    return st;
}

rc_status launch_batch(const BatchPart* d_parts, int n_parts, long long n_items, int ppi, const float4* tdirs,
                       const rc_params* p, int64_t max_tris, unsigned long long* work, cudaStream_t s)
{
    const int threads = 128;
    const int kind = point_kind(p, max_tris);
    const size_t smem = cast_smem(threads / 32, (p->n_dirs + 31) / 32, kind, false);
    const int per_sm = p->blocks_per_sm > 0 ? p->blocks_per_sm : RC_BATCH_MIN_BLOCKS;
    int64_t blocks = (int64_t)sm_count() * per_sm;
    const int64_t need = (n_items * 32 + threads - 1) / threads;
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    const auto kernel = kind == kWide4      ? k_batch<false, kWide4>
                        : kind == kBinary   ? k_batch<false, kBinary>
                        : kind == kWide4Big ? k_batch<false, kWide4Big>
                        : kind == kWide4Seg ? k_batch<false, kWide4Seg>
                                            : k_batch<false, kWide4BigSeg>;
    kernel<<<(unsigned)blocks, threads, smem, s>>>(d_parts, n_parts, n_items, ppi, tdirs, p->n_dirs, p->origin_offset,
                                                   work);
    RC_LAUNCHED();
    return RC_OK;
}

rc_status prepare_batch_kernel()
{
    RC_CUDA(allow_cast_smem(k_batch<false, kBinary>, 4, kBinary, false));
    RC_CUDA(allow_cast_smem(k_batch<false, kWide4>, 4, kWide4, false));
    RC_CUDA(allow_cast_smem(k_batch<false, kWide4Big>, 4, kWide4Big, false));
    RC_CUDA(allow_cast_smem(k_batch<false, kWide4Seg>, 4, kWide4Seg, false));
    RC_CUDA(allow_cast_smem(k_batch<false, kWide4BigSeg>, 4, kWide4BigSeg, false));
    return RC_OK;
}

}  // namespace rc
