// Closed-form 3-point Kabsch (Sec. 3.5), shared by the clique search (which
// solves each pivot's cliques as soon as it has chosen them) and by the
// clique-Kabsch entry point.
//
// Closed-form 3-point Kabsch.  With a_k = x_k - mean(x), b_k = y_k - mean(y)
// the cross-covariance H = sum_k a_k b_k^T has rank <= 2 (three points are
// coplanar).  Write a_k = E P_k, b_k = F Q_k with E = [e1 e2], F = [f1 f2]
// orthonormal in-plane frames and n_x = e1 x e2, n_y = f1 x f2.  Then
// H = E M F^T with the 2x2 M = sum_k P_k Q_k^T, and every proper rotation
// maximising tr(R H) has the form R = F X E^T + det(X) n_y n_x^T with X in
// O(2) maximising tr(X M):
//   rotation   X = [[c,-s],[s,c]] : tr = c(m11+m22) + s(m12-m21)
//   reflection X = [[c,s],[s,-c]] : tr = c(m11-m22) + s(m12+m21)
// The larger of the two vector norms is sigma1 + sigma2, the smaller
// |sigma1 - sigma2| (singular values of M, hence of H), and (c, s) is the
// normalised winning vector.  No iteration, no atan2.
//
// Precision: FP32.  For a thin triangle (kappa = sigma1/sigma2 large) all of
// the closed form's rounding error enters through the triangle normal, a
// cross product of two nearly parallel edges (relative error ~ u kappa); the
// frames, projections and the 2x2 step are well conditioned.  So when kappa
// exceeds the bound (default 100) or the FP32 frames are undefined, the two
// normals are recomputed in FP64 from exact FP64 differences of the FP32
// inputs, rounded to FP32, and the rest is redone in FP32: checked against the
// FP64 SVD, the rotation then stays within ~4e-7 of it up to kappa ~ 1e5,
// where the all-FP32 form is off by ~4e-3.  The clique search computes these
// FP64 components with six lanes per clique (one per triangle and component),
// so a warp issues a dozen FP64 instructions instead of a hundred.  A clique
// with sigma2 <= 1e-12 sigma1 (collinear or repeated points) is invalid.
//
// Every product and sum names its rounding (__fmaf_rn, __fmul_rn, __fadd_rn), so
// that a clique's R, t and kappa are the same bits in every kernel that solves
// it: one problem's search, a batch's solve kernel, the clique-Kabsch entry.  Left
// to the compiler, which products it contracts changed with the kernel's shape
// and register budget.  (The order of the operations is the one the search's
// kernels had been given: the results are the earlier ones.)
#pragma once

#include "tr_common.cuh"
#include "tr_problem.h"

namespace tr {

namespace {

__device__ __forceinline__ float inv_sqrt(float x) { return 1.0f / sqrtf(x); }

struct KabschOut {
    float R[9];
    float t[3];
    float kappa;
    bool ok;    // frames defined and sigma1 > 0
    float s1, s2;
};

// a b - c d
__device__ __forceinline__ float diff_prod(float a, float b, float c, float d)
{
    return __fmaf_rn(a, b, -__fmul_rn(c, d));
}

__device__ __forceinline__ void cross3(const float a[3], const float b[3], float c[3])
{
    c[0] = diff_prod(a[1], b[2], a[2], b[1]);
    c[1] = diff_prod(a[2], b[0], a[0], b[2]);
    c[2] = diff_prod(a[0], b[1], a[1], b[0]);
}

__device__ __forceinline__ float dot3(const float a[3], const float b[3])
{
    return __fmaf_rn(a[2], b[2], __fmaf_rn(a[0], b[0], __fmul_rn(a[1], b[1])));
}

// Component c of the normal (p1 - p0) x (p2 - p0) in FP64 from exact FP64
// differences of the FP32 coordinates, rounded to FP32.
__device__ __forceinline__ float exact_normal_comp(const float (&p)[3][3], int c)
{
    const int c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1;
    const double a1 = static_cast<double>(p[1][c1]) - static_cast<double>(p[0][c1]);
    const double a2 = static_cast<double>(p[1][c2]) - static_cast<double>(p[0][c2]);
    const double b1 = static_cast<double>(p[2][c1]) - static_cast<double>(p[0][c1]);
    const double b2 = static_cast<double>(p[2][c2]) - static_cast<double>(p[0][c2]);
    return static_cast<float>(__fma_rn(a1, b2, -__dmul_rn(a2, b1)));
}

// In-plane orthonormal frame of a triangle: e1 along its longest edge,
// n = unit normal of (p1 - p0) x (p2 - p0), e2 = n x e1.  ng: the normal's
// components given by the caller (FP64 cross product rounded to FP32), and
// then *nlen receives their length |(p1 - p0) x (p2 - p0)| (twice the area).
template <bool kGiven>
__device__ __forceinline__ bool frame3(const float p[3][3], float e1[3], float e2[3], float nrm[3], const float* ng,
                                       float* nlen)
{
    float d01[3], d02[3], d12[3];
    for (int c = 0; c < 3; ++c) {
        d01[c] = __fsub_rn(p[1][c], p[0][c]);
        d02[c] = __fsub_rn(p[2][c], p[0][c]);
        d12[c] = __fsub_rn(p[2][c], p[1][c]);
    }
    float nn;
    if (kGiven) {
        nrm[0] = ng[0]; nrm[1] = ng[1]; nrm[2] = ng[2];
        nn = __fmaf_rn(nrm[2], nrm[2], __fmaf_rn(nrm[1], nrm[1], __fmul_rn(nrm[0], nrm[0])));
        *nlen = sqrtf(nn);
    } else {
        cross3(d01, d02, nrm);
        nn = dot3(nrm, nrm);
    }
    const float l01 = dot3(d01, d01), l02 = dot3(d02, d02), l12 = dot3(d12, d12);
    int sel = 0;   // longest edge, selected by value (no pointer into local arrays)
    float le = l01;
    if (l02 > le) { sel = 1; le = l02; }
    if (l12 > le) { sel = 2; le = l12; }
    if (!(nn > 0.f) || !(le > 0.f)) return false;
    const float in = inv_sqrt(nn), ie = inv_sqrt(le);
    for (int c = 0; c < 3; ++c) {
        nrm[c] = __fmul_rn(nrm[c], in);
        e1[c] = __fmul_rn(sel == 0 ? d01[c] : sel == 1 ? d02[c] : d12[c], ie);
    }
    cross3(nrm, e1, e2);
    return true;
}

// kGiven: the two triangles' normals nxg, nyg are given by the caller (the
// FP64 path); otherwise they are the FP32 cross products.
template <bool kGiven = false>
__device__ __forceinline__ void kabsch3(const float p[3][3], const float q[3][3], KabschOut& o,
                                        const float* nxg = nullptr, const float* nyg = nullptr)
{
    constexpr float kThird = static_cast<float>(1.0 / 3.0);
    float cx[3], sy[3];   // mean of the p, sum of the q
    for (int c = 0; c < 3; ++c) {
        cx[c] = __fmul_rn(__fadd_rn(__fadd_rn(p[0][c], p[1][c]), p[2][c]), kThird);
        sy[c] = __fadd_rn(__fadd_rn(q[0][c], q[1][c]), q[2][c]);
    }
    float e1[3], e2[3], nx[3], f1[3], f2[3], ny[3];
    float lx = 0.f, ly = 0.f;
    o.ok = frame3<kGiven>(p, e1, e2, nx, nxg, &lx) && frame3<kGiven>(q, f1, f2, ny, nyg, &ly);
    if (!o.ok) {
        o.kappa = INFINITY;
        o.s1 = o.s2 = 0.f;
        return;
    }
    float m11 = 0.f, m12 = 0.f, m21 = 0.f, m22 = 0.f;
    for (int k = 0; k < 3; ++k) {
        float a[3], b[3];
        for (int c = 0; c < 3; ++c) {
            a[c] = __fsub_rn(p[k][c], cx[c]);
            b[c] = __fmaf_rn(-sy[c], kThird, q[k][c]);
        }
        const float P1 = dot3(a, e1), P2 = dot3(a, e2);
        const float Q1 = dot3(b, f1), Q2 = dot3(b, f2);
        m11 = __fmaf_rn(P1, Q1, m11); m12 = __fmaf_rn(P1, Q2, m12);
        m21 = __fmaf_rn(P2, Q1, m21); m22 = __fmaf_rn(P2, Q2, m22);
    }
    const float rx = __fadd_rn(m11, m22), ry = __fsub_rn(m12, m21);   // rotation candidate
    const float fx = __fsub_rn(m11, m22), fy = __fadd_rn(m12, m21);   // reflection candidate
    const float r2 = __fmaf_rn(ry, ry, __fmul_rn(rx, rx)), q2 = __fmaf_rn(fy, fy, __fmul_rn(fx, fx));
    if (!(r2 > 0.f || q2 > 0.f)) {
        o.ok = false;
        o.kappa = INFINITY;
        o.s1 = o.s2 = 0.f;
        return;
    }
    const bool rot = r2 >= q2;
    const float hi2 = rot ? r2 : q2, lo2 = rot ? q2 : r2;
    const float ih = inv_sqrt(hi2);                     // 1 / (sigma1 + sigma2)
    const float lo = lo2 > 0.f ? __fmul_rn(lo2, inv_sqrt(lo2)) : 0.f;
    o.s1 = __fmul_rn(__fmaf_rn(hi2, ih, lo), 0.5f);
    o.s2 = __fmul_rn(__fmaf_rn(hi2, ih, -lo), 0.5f);
    if (kGiven && o.s1 > 0.f) {
        // sigma2 of a thin clique from sigma1 sigma2 = |det M| = |n_x| |n_y| / 3
        // (Cauchy-Binet over three centred points), with the lengths of the
        // accurate normals, instead of the cancelling difference (hi - lo) / 2
        o.s2 = __fmul_rn(lx, ly) / __fmul_rn(3.f, o.s1);
    }
    o.kappa = o.s2 > 0.f ? o.s1 / o.s2 : INFINITY;
    float X00, X01, X10, X11, sg;
    if (rot) {
        const float c = __fmul_rn(rx, ih), s = __fmul_rn(ry, ih);
        X00 = c; X01 = -s; X10 = s; X11 = c; sg = 1.f;
    } else {
        const float c = __fmul_rn(fx, ih), s = __fmul_rn(fy, ih);
        X00 = c; X01 = s; X10 = s; X11 = -c; sg = -1.f;
    }
    for (int r = 0; r < 3; ++r) {
        const float xa = __fmul_rn(X00, f1[r]), xb = __fmul_rn(X01, f1[r]);
        const float xc = __fmul_rn(X10, f2[r]), xd = __fmul_rn(X11, f2[r]), xe = __fmul_rn(sg, ny[r]);
        for (int c = 0; c < 3; ++c) {
            float v = __fmaf_rn(xa, e1[c], __fmul_rn(xb, e2[c]));
            v = __fmaf_rn(xc, e1[c], v);
            v = __fmaf_rn(xd, e2[c], v);
            o.R[r * 3 + c] = __fmaf_rn(xe, nx[c], v);
        }
    }
    for (int r = 0; r < 3; ++r) o.t[r] = __fmaf_rn(sy[r], kThird, -dot3(&o.R[r * 3], cx));
}

__device__ __forceinline__ void load_clique(const ProbView& v, const int4 cl, float p[3][3], float q[3][3])
{
    const int idx[3] = {cl.x, cl.y, cl.z};
    for (int a = 0; a < 3; ++a) {
        const float4* r = reinterpret_cast<const float4*>(v.pts8 + (size_t)idx[a] * 8);
        const float4 u = r[0], w = r[1];
        p[a][0] = u.x; p[a][1] = u.y; p[a][2] = u.z;
        q[a][0] = u.w; q[a][1] = w.x; q[a][2] = w.y;
    }
}

// Writes hypothesis h: R, t and kappa of a solved clique (flags: 1 valid,
// 2 the FP64 normals were used), zero for an empty slot; the inlier count
// and score are cleared.
__device__ __forceinline__ void store_hypothesis(const ProbView& v, int h, bool present, const KabschOut& o,
                                                 uint32_t flags)
{
    v.inl[h] = 0;
    v.score[h] = 0ull;
    float o16[13];
#pragma unroll
    for (int r = 0; r < 13; ++r) o16[r] = 0.f;
    if (present) {
        if (o.ok && o.s1 > 0.f && o.s2 > 1e-12f * o.s1) {
#pragma unroll
            for (int r = 0; r < 9; ++r) o16[r] = o.R[r];
#pragma unroll
            for (int r = 0; r < 3; ++r) o16[9 + r] = o.t[r];
            flags |= 1u;
        }
        o16[12] = o.kappa;
    } else {
        flags = 0u;
    }
    float4* o4 = reinterpret_cast<float4*>(v.rt + (size_t)h * 16);
    o4[0] = make_float4(o16[0], o16[1], o16[2], o16[3]);
    o4[1] = make_float4(o16[4], o16[5], o16[6], o16[7]);
    o4[2] = make_float4(o16[8], o16[9], o16[10], o16[11]);
    o4[3] = make_float4(o16[12], __int_as_float(static_cast<int>(flags)), 0.f, 0.f);
}

// Closed form of hypothesis h with clique cl by one thread (the FP64 normals,
// when needed, computed by the same thread).
__device__ __forceinline__ void kabsch_hypothesis(const ProbView& v, int h, int4 cl)
{
    KabschOut o;
    uint32_t flags = 0;
    if (cl.w) {
        float p[3][3], q[3][3];
        load_clique(v, cl, p, q);
        kabsch3(p, q, o);
        if (!(o.ok && o.kappa <= v.kappa_fp64)) {   // ill-conditioned: FP64 normals
            float nx[3], ny[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                nx[c] = exact_normal_comp(p, c);
                ny[c] = exact_normal_comp(q, c);
            }
            kabsch3<true>(p, q, o, nx, ny);
            flags = 2u;
        }
    }
    store_hypothesis(v, h, cl.w != 0, o, flags);
}

}  // namespace

}  // namespace tr
