// element.cuh -- per-element arithmetic of the integration step (Eqs. 7-9) for
// the 8-node trilinear brick (2x2x2 Gauss) and the 4-node linear tetrahedron
// (exact 1-point rule), in FP32 or FP64.
//
// Formulation.  With J_q the Jacobian at Gauss point q (rows d x / d xi_i) and
// B_q = J_q^{-1} dN_q (Section 3), the element matrix of Eq. 9 is
//     k_ab = c * sum_q  dN_q,a^T  M_q  dN_q,b,
//     M_q  = w_q |det J_q| J_q^{-T} J_q^{-1} = w_q cof(J_q) cof(J_q)^T / |det J_q|,
// where the rows of cof(J) are cross products of the rows of J.  Nothing is
// dropped or approximated: this is Eq. 9 with the inverse written as
// adj(J) / det J.  For the brick the natural derivatives are tensor products of
// the 1D hat functions, so the map from the 8 x 6 values of M_q to the 36
// packed entries factorises along the three axes (sum factorisation): about
// 1 kflop per element instead of about 3.8 kflop for forming B and B^T B
// point by point.  J_q itself is a bilinear interpolation of the 4 element edges
// along each axis, formed from coordinate differences so that FP32 keeps its
// accuracy relative to the element size.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "pair.cuh"

namespace fem {

// ----------------------------------------------------------------- brick layout
// Node a of the brick has axis bits (a1, a2, a3) in {0,1}^3 (xi = 2*bit - 1):
// nodes 0-3 on t = -1 counter-clockwise from (-1,-1,-1), nodes 4-7 on t = +1.
__host__ __device__ constexpr int hb1(int a) { return (a == 1 || a == 2 || a == 5 || a == 6) ? 1 : 0; }
__host__ __device__ constexpr int hb2(int a) { return (a == 2 || a == 3 || a == 6 || a == 7) ? 1 : 0; }
__host__ __device__ constexpr int hb3(int a) { return a >= 4 ? 1 : 0; }
__host__ __device__ constexpr int hnode(int b1, int b2, int b3) {
    return b3 * 4 + (b2 ? (b1 ? 2 : 3) : (b1 ? 1 : 0));
}
// class of a pair of bits: 0 = (0,0), 1 = (1,1), 2 = mixed
__host__ __device__ constexpr int hcls(int x, int y) { return x == y ? x : 2; }
__host__ __device__ constexpr int hsig(int x) { return x ? 1 : -1; }

// 1D two-point Gauss rule on [-1, 1]: points -g, +g (g = 1/sqrt(3)), weights 1.
// phi_i(x_j) of the linear hats phi_0 = (1 - x)/2, phi_1 = (1 + x)/2 is GP if
// i == j else GQ.  Products: GP^2 = 1/3 + g/2, GQ^2 = 1/3 - g/2, GP GQ = 1/6.
#define FEM_GP 0.78867513459481288225
#define FEM_GQ 0.21132486540518711775
#define FEM_GPP 0.62200846792814621559
#define FEM_GQQ 0.04465819873852045108
#define FEM_GPQ 0.16666666666666666667

template <typename T>
struct Vec3 {
    T x, y, z;
};
template <typename T>
__device__ __forceinline__ Vec3<T> cross3(const Vec3<T> &a, const Vec3<T> &b) {
    return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
template <typename T>
__device__ __forceinline__ T dot3(const Vec3<T> &a, const Vec3<T> &b) {
    return a.x * b.x + a.y * b.y + a.z * b.z;
}
// Reciprocals.  FP32: the hardware approximation (rcp.approx) refined by one
// Newton-Raphson step r' = r + r (1 - x r), about 1 ulp, FP32 pipe only.  (The
// correctly rounded FP32 reciprocal and any conversion to double use the FP64
// pipe, which on this part runs at 1/64 of the FP32 rate.)  FP64: the correctly
// rounded double reciprocal.
__device__ __forceinline__ float rcp_rn(float x) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    const float e = fmaf(-x, r, 1.0f);
    return fmaf(r, e, r);
}
__device__ __forceinline__ double rcp_rn(double x) { return __drcp_rn(x); }

// a*b - c*d with a single rounding error (Kahan's FMA-based 2x2 determinant):
// w = c*d is rounded, its rounding error is recovered exactly by an FMA.
__device__ __forceinline__ float det2(float a, float b, float c, float d) {
    const float w = __fmul_rn(c, d);
    const float err = __fmaf_rn(-c, d, w);
    const float f = __fmaf_rn(a, b, -w);
    return __fadd_rn(f, err);
}
__device__ __forceinline__ Vec3<float> cross3_accurate(const Vec3<float> &a, const Vec3<float> &b) {
    return {det2(a.y, b.z, a.z, b.y), det2(a.z, b.x, a.x, b.z), det2(a.x, b.y, a.y, b.x)};
}

// Error-free transformations: Knuth's TwoSum (a + b = s + e exactly) and the FMA
// form of Dekker's product (a * b = p + e exactly).  Written with the _rn
// intrinsics, which the compiler never contracts into FMAs: a contraction of
// p = a * b into a later sum would break the exactness, and could differ between
// kernels that inline the same code.
__device__ __forceinline__ void two_sum_f(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void two_prod_f(float a, float b, float &p, float &e) {
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}

// x - y split into a float pair (h, l) with h + l == x - y: exactly for float
// inputs (TwoSum), to ~2^-48 relative for double inputs.
__device__ __forceinline__ void diff_ds(float x, float y, float &h, float &l) { two_sum_f(x, -y, h, l); }
__device__ __forceinline__ void diff_ds(double x, double y, float &h, float &l) {
    const double d = x - y;
    h = (float)d;
    l = (float)(d - (double)h);
}

// Jacobian determinant of a tetrahedron, det [x1 - x0; x2 - x0; x3 - x0], in
// double-single arithmetic: the edge vectors are formed exactly as float pairs,
// each product of pairs is split exactly (the FMA form of Dekker's product) with
// its cross terms added, each 2x2 minor and the final dot product are summed with
// TwoSum.  The result, rounded once to float, is accurate to a few units of
// 2^-46 times the sum of the magnitudes of the determinant's terms: what an FP64
// evaluation from the same coordinates gives a float result, in FP32 arithmetic.
template <typename S>
__device__ __forceinline__ float det3_ds(const S (*xc)[3]) {
    float h[3][3], l[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) diff_ds(xc[i + 1][k], xc[0][k], h[i][k], l[i][k]);
    // product of pairs (ah + al)(bh + bl) as (p, e), dropping al * bl
    auto mul = [](float ah, float al, float bh, float bl, float &p, float &e) {
        two_prod_f(ah, bh, p, e);
        e = fmaf(ah, bl, fmaf(al, bh, e));
    };
    // minors of rows 1, 2 (the cofactors of row 0) as unevaluated pairs (s, t)
    float s[3], t[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int u = (k + 1) % 3, v = (k + 2) % 3;
        float p, ep, q, eq, es;
        mul(h[1][u], l[1][u], h[2][v], l[2][v], p, ep);
        mul(h[1][v], l[1][v], h[2][u], l[2][u], q, eq);
        two_sum_f(p, -q, s[k], es);
        t[k] = es + (ep - eq);
    }
    float P[3], E[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        two_prod_f(h[0][k], s[k], P[k], E[k]);
        E[k] = fmaf(h[0][k], t[k], fmaf(l[0][k], s[k], E[k]));
    }
    float a, e1, b, e2;
    two_sum_f(P[0], P[1], a, e1);
    two_sum_f(a, P[2], b, e2);
    return b + ((e1 + e2) + (E[0] + E[1] + E[2]));
}

template <typename T>
__device__ __forceinline__ Vec3<T> lerp2(T wa, const Vec3<T> &a, T wb, const Vec3<T> &b) {
    return {wa * a.x + wb * b.x, wa * a.y + wb * b.y, wa * a.z + wb * b.z};
}

// The two Gauss-point values (P a + Q b, Q a + P b) of the linear hats through
// a and b.  P + Q = 1, so they are b + P (a - b) and a - P (a - b): one
// subtraction and two explicit FMAs instead of two products and two FMAs.
template <typename T>
__device__ __forceinline__ void hat_pair(T a, T b, T &o0, T &o1) {
    const T d = a - b;
    o0 = fma(T(FEM_GP), d, b);
    o1 = fma(-T(FEM_GP), d, a);
}
template <typename T>
__device__ __forceinline__ void hat_pair(const Vec3<T> &a, const Vec3<T> &b, Vec3<T> &o0, Vec3<T> &o1) {
    hat_pair(a.x, b.x, o0.x, o1.x);
    hat_pair(a.y, b.y, o0.y, o1.y);
    hat_pair(a.z, b.z, o0.z, o1.z);
}

// Edge vectors of a brick along each axis, e[axis][i][j], the two other axes'
// bits (i, j) in increasing axis order.  xc[a] = coordinates of node a (input
// precision S); the differences are formed in S and rounded once to T.
template <typename T, typename S>
__device__ __forceinline__ void brick_edges(const S (*xc)[3], Vec3<T> (&e)[3][2][2]) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r0 = hnode(0, i, j), r1 = hnode(1, i, j);
            const int s0 = hnode(i, 0, j), s1 = hnode(i, 1, j);
            const int t0 = hnode(i, j, 0), t1 = hnode(i, j, 1);
            e[0][i][j] = {T(xc[r1][0] - xc[r0][0]), T(xc[r1][1] - xc[r0][1]), T(xc[r1][2] - xc[r0][2])};
            e[1][i][j] = {T(xc[s1][0] - xc[s0][0]), T(xc[s1][1] - xc[s0][1]), T(xc[s1][2] - xc[s0][2])};
            e[2][i][j] = {T(xc[t1][0] - xc[t0][0]), T(xc[t1][1] - xc[t0][1]), T(xc[t1][2] - xc[t0][2])};
        }
}

// Jacobian rows (times 2) at the Gauss points: row[axis][u][v] with (u, v) the
// Gauss indices of the two other axes.  row = sum_ij phi_i(u) phi_j(v) e[i][j].
template <typename T>
__device__ __forceinline__ void brick_jrows(const Vec3<T> (&e)[3][2][2], Vec3<T> (&row)[3][2][2]) {
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        Vec3<T> m[2][2];  // m[i][v] = interpolation along the last axis
#pragma unroll
        for (int i = 0; i < 2; ++i) hat_pair(e[ax][i][0], e[ax][i][1], m[i][0], m[i][1]);
#pragma unroll
        for (int v = 0; v < 2; ++v) hat_pair(m[0][v], m[1][v], row[ax][0][v], row[ax][1][v]);
    }
}

// ------------------------------------------------------ brick stiffness, in pairs
// The brick's arithmetic runs on pairs (pair.cuh): every quantity that depends on
// the Gauss point index q1 is held for q1 = 0 and 1 together, so FP32 needs one
// packed instruction for two points.  Only the 1D operators along axis 1 itself
// work inside a pair, in scalars.  The build kernels are bound by latency at 16
// warps an SM, so an element's shorter instruction stream pays less than its count:
// 1M bricks 236 -> 228 us mixed (512 meshes in one launch 3.30 -> 3.17 ms), with
// the FP32 result's error against 64 bits 1.1e-7 -> 0.7e-7; FP64, whose pipe is
// busy throughout, 2.41 -> 2.26 ms from the shared sums alone.

// Rows of 2 J_q at the Gauss points: R (axis 1) does not depend on q1, S (axis 2)
// and U (axis 3) hold q1 = 0 and 1 as pairs: R[q2][q3], S[q3], U[q2].
template <typename T>
struct BrickRows {
    Vec3<T> R[2][2];
    Vec3<Pair<T>> S[2], U[2];
};

// Edges (differences formed in S, rounded once to T): r[i][j] along axis 1 at bits
// (i, j) of axes 2 and 3; s[j], u[j] along axes 2 and 3 as pairs over the bit of
// axis 1, at bit j of axis 3 and 2.
template <typename T, typename S>
__device__ __forceinline__ void brick_edge_pairs(const S (*xc)[3], int k, T (&r)[2][2], Pair<T> (&s)[2],
                                                 Pair<T> (&u)[2]) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) r[i][j] = T(xc[hnode(1, i, j)][k] - xc[hnode(0, i, j)][k]);
    if constexpr (sizeof(S) == sizeof(T)) {
        Pair<T> x[2][2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) x[i][j] = pair(xc[hnode(0, i, j)][k], xc[hnode(1, i, j)][k]);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            s[j] = x[1][j] - x[0][j];
            u[j] = x[j][1] - x[j][0];
        }
    } else {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            s[j] = pair(T(xc[hnode(0, 1, j)][k] - xc[hnode(0, 0, j)][k]),
                        T(xc[hnode(1, 1, j)][k] - xc[hnode(1, 0, j)][k]));
            u[j] = pair(T(xc[hnode(0, j, 1)][k] - xc[hnode(0, j, 0)][k]),
                        T(xc[hnode(1, j, 1)][k] - xc[hnode(1, j, 0)][k]));
        }
    }
}

// hat_pair elementwise, and along axis 1 inside a pair.
template <typename T>
__device__ __forceinline__ void hat_pair(Pair<T> a, Pair<T> b, Pair<T> &o0, Pair<T> &o1) {
    const Pair<T> d = a - b;
    o0 = pfma(pair(T(FEM_GP), T(FEM_GP)), d, b);
    o1 = pfma(pair(-T(FEM_GP), -T(FEM_GP)), d, a);
}
template <typename T>
__device__ __forceinline__ Pair<T> hat_in_pair(Pair<T> p) {
    T o0, o1;
    hat_pair(pair_lo(p), pair_hi(p), o0, o1);
    return pair(o0, o1);
}

template <typename T>
__device__ __forceinline__ void brick_rows_k(const T (&r)[2][2], const Pair<T> (&s)[2], const Pair<T> (&u)[2],
                                             T (&R)[2][2], Pair<T> (&So)[2], Pair<T> (&Uo)[2]) {
    T m[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i) hat_pair(r[i][0], r[i][1], m[i][0], m[i][1]);
#pragma unroll
    for (int v = 0; v < 2; ++v) hat_pair(m[0][v], m[1][v], R[0][v], R[1][v]);
    Pair<T> a, b;
    hat_pair(s[0], s[1], a, b);
    So[0] = hat_in_pair(a), So[1] = hat_in_pair(b);
    hat_pair(u[0], u[1], a, b);
    Uo[0] = hat_in_pair(a), Uo[1] = hat_in_pair(b);
}

template <typename T, typename S>
__device__ __forceinline__ void brick_rows(const S (*xc)[3], BrickRows<T> &o) {
    T r[2][2], R[2][2];
    Pair<T> s[2], u[2], So[2], Uo[2];
#define FEM_BRICK_ROWS(k, c)                          \
    brick_edge_pairs<T, S>(xc, k, r, s, u);           \
    brick_rows_k(r, s, u, R, So, Uo);                 \
    o.R[0][0].c = R[0][0], o.R[0][1].c = R[0][1], o.R[1][0].c = R[1][0], o.R[1][1].c = R[1][1]; \
    o.S[0].c = So[0], o.S[1].c = So[1], o.U[0].c = Uo[0], o.U[1].c = Uo[1];
    FEM_BRICK_ROWS(0, x)
    FEM_BRICK_ROWS(1, y)
    FEM_BRICK_ROWS(2, z)
#undef FEM_BRICK_ROWS
}

// a x b of pairs, given na = -a (packed instructions have no free negation).
template <typename T>
__device__ __forceinline__ Vec3<Pair<T>> cross3(const Vec3<Pair<T>> &a, const Vec3<Pair<T>> &na,
                                                const Vec3<Pair<T>> &b) {
    return {pfma(a.y, b.z, na.z * b.y), pfma(a.z, b.x, na.x * b.z), pfma(a.x, b.y, na.y * b.x)};
}
template <typename T>
__device__ __forceinline__ Pair<T> dot3(const Vec3<Pair<T>> &a, const Vec3<Pair<T>> &b) {
    return pfma(a.z, b.z, pfma(a.y, b.y, a.x * b.x));
}
template <typename T>
__device__ __forceinline__ Vec3<Pair<T>> neg3(const Vec3<Pair<T>> &a) {
    return {-a.x, -a.y, -a.z};
}
template <typename T>
__device__ __forceinline__ Vec3<Pair<T>> both3(const Vec3<T> &a) {
    return {pair(a.x, a.x), pair(a.y, a.y), pair(a.z, a.z)};
}

// 1 / |d| of both halves, as rcp_rn.  The FP32 form iterates on -1/|d|, whose sign
// makes the residual 1 - |d| r a plain packed FMA, and returns -1/|d|.
__device__ __forceinline__ Pair<float> neg_rcp_abs(Pair<float> d) {
    const float x0 = fabsf(pair_lo(d)), x1 = fabsf(pair_hi(d));
    float n0, n1;
    asm("rcp.approx.f32 %0, %1;" : "=f"(n0) : "f"(-x0));
    asm("rcp.approx.f32 %0, %1;" : "=f"(n1) : "f"(-x1));
    const Pair<float> n = pair(n0, n1);
    return pfma(n, pfma(pair(x0, x1), n, pair(1.f, 1.f)), n);
}
__device__ __forceinline__ Pair<double> neg_rcp_abs(Pair<double> d) {
    return {-rcp_rn(fabs(d.x)), -rcp_rn(fabs(d.y))};
}

// The hat products along one axis are taken six times over: 6 F_0 = (2 + g3, 2 - g3),
// 6 F_1 = (2 - g3, 2 + g3), 6 F_2 = (1, 1) with g3 = sqrt(3), so that a contraction
// is 2 (a + b) +- g3 (a - b) and a + b, five operations instead of six.  The
// diagonal terms pass two such contractions and the cross terms one: their M_q are
// scaled by 1/36 and 1/6.
#define FEM_G3 1.7320508075688772935
template <typename T>
__device__ __forceinline__ void prod6(T a, T b, T &o0, T &o1, T &o2) {
    o2 = a + b;
    const T t = T(FEM_G3) * (a - b);
    o0 = fma(T(2), o2, t);
    o1 = fma(T(2), o2, -t);
}
template <typename T>
__device__ __forceinline__ void prod6(Pair<T> a, Pair<T> b, Pair<T> (&o)[3]) {
    const Pair<T> d = a - b;
    o[2] = a + b;
    const Pair<T> s = o[2] + o[2];
    o[0] = pfma(pair(T(FEM_G3), T(FEM_G3)), d, s);
    o[1] = pfma(pair(-T(FEM_G3), -T(FEM_G3)), d, s);
}

// M~_q = cof(2J_q) cof(2J_q)^T / |det 2J_q| (k_e = c/8 sum_q dN~_a^T M~_q dN~_b with
// dN~ = 2 dN = +-1 times hats) as pairs over q1: M[q2][q3] holds (rr, ss, tt)
// scaled by s/36 and (rs, rt, st) scaled by s/6; det = det(2 J_q).
template <typename T>
__device__ __forceinline__ void brick_M(const BrickRows<T> &row, T s, Pair<T> (&M)[2][2][6], Pair<T> (&det)[2][2]) {
    const T sd = s * T(-1.0 / 36.0), sc = s * T(-1.0 / 6.0);
    const Pair<T> wd = pair(sd, sd), wc = pair(sc, sc);
    Vec3<Pair<T>> nU[2];
#pragma unroll
    for (int q2 = 0; q2 < 2; ++q2) nU[q2] = neg3(row.U[q2]);
#pragma unroll
    for (int q3 = 0; q3 < 2; ++q3) {
        const Vec3<Pair<T>> &S = row.S[q3];
        const Vec3<Pair<T>> nS = neg3(S);
#pragma unroll
        for (int q2 = 0; q2 < 2; ++q2) {
            const Vec3<Pair<T>> R = both3(row.R[q2][q3]);
            const Vec3<Pair<T>> &U = row.U[q2];
            const Vec3<Pair<T>> C0 = cross3(S, nS, U), C1 = cross3(U, nU[q2], R);
            // R x S = -(S x R) = (-S) x R
            const Vec3<Pair<T>> C2 = cross3(nS, S, R);
            det[q2][q3] = dot3(R, C0);
            const Pair<T> inv = neg_rcp_abs(det[q2][q3]);
            const Pair<T> id = inv * wd, ic = inv * wc;
            Pair<T>(&m)[6] = M[q2][q3];
            m[0] = dot3(C0, C0) * id;
            m[1] = dot3(C1, C1) * id;
            m[2] = dot3(C2, C2) * id;
            m[3] = dot3(C0, C1) * ic;
            m[4] = dot3(C0, C2) * ic;
            m[5] = dot3(C1, C2) * ic;
        }
    }
}

// T[c][d] = sum_{u,v} A[u][v] 6F_c(u) 6F_d(v); A[v] and the rows c = 0, 1 are pairs
// over u and c: To[d] = (T[0][d], T[1][d]), T2[d] = T[2][d].
template <typename T>
__device__ __forceinline__ void contract_FF(Pair<T> A0, Pair<T> A1, Pair<T> (&To)[3], T (&T2)[3]) {
    Pair<T> W[3];
    prod6(A0, A1, W);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        T o0, o1;
        prod6(pair_lo(W[d]), pair_hi(W[d]), o0, o1, T2[d]);
        To[d] = pair(o0, o1);
    }
}

// Packed lower k_e (36 entries, p = a(a+1)/2 + b) from brick_M's M.  k_ab is a sum
// of nine contracted terms:
//   s1 Trr[c2][c3] + s2 Tss[c1][c3] + s3 Ttt[c1][c2]
//   + the cross terms in (r,s), (r,t), (s,t),
// c_i the class of the pair's bits on axis i (0, 1, or 2 = mixed) and s_i = -1 for
// mixed bits.  Pairs of nodes with equal bits on axis 1 come two at a time (bit 0
// and 1), the 16 with mixed bits one by one; sums that several entries share are
// formed once.
template <typename T>
__device__ __forceinline__ void brick_contract(const Pair<T> (&M)[2][2][6], T (&k)[36]) {
    // (c1 = 0, 1) as pairs, c1 = 2 as scalars
    Pair<T> Tss[3], Ttt[3];  // [c3], [c2]
    T Tss2[3], Ttt2[3], Trr[3][3];
    {
        T a[2][2];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int v = 0; v < 2; ++v) a[u][v] = pair_lo(M[u][v][0]) + pair_hi(M[u][v][0]);  // sum over q1
        Pair<T> o[3];
        T o2[3];
        contract_FF(pair(a[0][0], a[1][0]), pair(a[0][1], a[1][1]), o, o2);
#pragma unroll
        for (int d = 0; d < 3; ++d) Trr[0][d] = pair_lo(o[d]), Trr[1][d] = pair_hi(o[d]), Trr[2][d] = o2[d];
    }
    contract_FF(M[0][0][1] + M[1][0][1], M[0][1][1] + M[1][1][1], Tss, Tss2);  // sum over q2
    contract_FF(M[0][0][2] + M[0][1][2], M[1][0][2] + M[1][1][2], Ttt, Ttt2);  // sum over q3
    // cross terms: Vrs[x][y][c3], Vrt[x][c2][z] (pairs over x), Vst[c1][y][z]
    Pair<T> Vrs[2][3], Vrt[3][2], Vst[2][2];
    T Vst2[2][2];
    {
        Pair<T> W[2][3];
#pragma unroll
        for (int b = 0; b < 2; ++b) prod6(M[b][0][3], M[b][1][3], W[b]);
#pragma unroll
        for (int c3 = 0; c3 < 3; ++c3) {
            Pair<T> y0, y1;
            hat_pair(W[0][c3], W[1][c3], y0, y1);
            Vrs[0][c3] = hat_in_pair(y0);
            Vrs[1][c3] = hat_in_pair(y1);
        }
    }
    {
        Pair<T> W[2][2];
#pragma unroll
        for (int b = 0; b < 2; ++b) hat_pair(M[b][0][4], M[b][1][4], W[b][0], W[b][1]);
#pragma unroll
        for (int z = 0; z < 2; ++z) {
            Pair<T> o[3];
            prod6(W[0][z], W[1][z], o);
#pragma unroll
            for (int c2 = 0; c2 < 3; ++c2) Vrt[c2][z] = hat_in_pair(o[c2]);
        }
    }
    {
        Pair<T> W[2][2];
#pragma unroll
        for (int b = 0; b < 2; ++b) hat_pair(M[b][0][5], M[b][1][5], W[b][0], W[b][1]);
#pragma unroll
        for (int z = 0; z < 2; ++z) {
            Pair<T> y[2];
            hat_pair(W[0][z], W[1][z], y[0], y[1]);
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                T o0, o1;
                prod6(pair_lo(y[b]), pair_hi(y[b]), o0, o1, Vst2[b][z]);
                Vst[b][z] = pair(o0, o1);
            }
        }
    }
    // pairs with equal bits on axis 1 (value x): the (r,s) term is
    // sig(x) (sig(b2) V[x][a2][c3] + sig(a2) V[x][b2][c3]) = sig(x) times 2 sig(a2) V[a2]
    // for equal bits on axis 2 and V[0] - V[1] for mixed ones; the (r,t) term alike
    const Pair<T> sig = pair(T(-1), T(1)), sig2 = pair(T(-2), T(2)), msig2 = pair(T(2), T(-2));
    const Pair<T> two = pair(T(2), T(2)), mtwo = pair(T(-2), T(-2));
    Pair<T> base[3][3];  // [c2][c3]: all but the (s,t) term
#pragma unroll
    for (int c2 = 0; c2 < 3; ++c2)
#pragma unroll
        for (int c3 = 0; c3 < 3; ++c3) {
            Pair<T> v = pair(Trr[c2][c3], Trr[c2][c3]);
            v = c2 == 2 ? v - Tss[c3] : v + Tss[c3];
            v = c3 == 2 ? v - Ttt[c2] : v + Ttt[c2];
            v = c2 == 2 ? pfma(sig, Vrs[0][c3] - Vrs[1][c3], v) : pfma(c2 ? sig2 : msig2, Vrs[c2][c3], v);
            v = c3 == 2 ? pfma(sig, Vrt[c2][0] - Vrt[c2][1], v) : pfma(c3 ? sig2 : msig2, Vrt[c2][c3], v);
            base[c2][c3] = v;
        }
    auto put = [&](int a, int b, T v) { k[a > b ? a * (a + 1) / 2 + b : b * (b + 1) / 2 + a] = v; };
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q <= p; ++q) {
            const int a2 = p >> 1, a3 = p & 1, b2 = q >> 1, b3 = q & 1;
            const int c2 = hcls(a2, b2), c3 = hcls(a3, b3);
            Pair<T> v = base[c2][c3];
            if (c2 != 2 && c3 != 2) v = pfma(a2 == a3 ? two : mtwo, Vst[a2][a3], v);
            else if (c3 != 2) v = a3 ? v + (Vst[0][a3] - Vst[1][a3]) : v - (Vst[0][a3] - Vst[1][a3]);
            else if (c2 != 2) v = a2 ? v + (Vst[a2][0] - Vst[a2][1]) : v - (Vst[a2][0] - Vst[a2][1]);
            else if (a2 == a3) v = v - (Vst[0][1] + Vst[1][0]);
            else v = v + (Vst[0][0] + Vst[1][1]);
            put(hnode(0, a2, a3), hnode(0, b2, b3), pair_lo(v));
            put(hnode(1, a2, a3), hnode(1, b2, b3), pair_hi(v));
        }
    // pairs with mixed bits on axis 1: node (1, a2, a3) against (0, b2, b3)
    T rs[2][2][3], rt[3][2][2], st[4][4], base2[3][3];
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                // sig(b2) V[0][a2] - sig(a2) V[1][b2], (x, y) = (a2, b2); alike in (r,t)
                const T u = pair_lo(Vrs[x][c]), w = pair_hi(Vrs[y][c]);
                rs[x][y][c] = y ? (x ? u - w : u + w) : (x ? -u - w : w - u);
                const T ut = pair_lo(Vrt[c][x]), wt = pair_hi(Vrt[c][y]);
                rt[c][x][y] = y ? (x ? ut - wt : ut + wt) : (x ? -ut - wt : wt - ut);
            }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q <= p; ++q) {
            const int a2 = p >> 1, a3 = p & 1, b2 = q >> 1, b3 = q & 1;
            const T u = Vst2[b2][a3], w = Vst2[a2][b3];
            // sig(a2) sig(b3) V[b2][a3] + sig(a3) sig(b2) V[a2][b3]
            st[p][q] = st[q][p] = (a2 == b3 ? u : -u) + (a3 == b2 ? w : -w);
        }
#pragma unroll
    for (int c2 = 0; c2 < 3; ++c2)
#pragma unroll
        for (int c3 = 0; c3 < 3; ++c3)
            base2[c2][c3] = (c2 == 2 ? -Tss2[c3] : Tss2[c3]) + (c3 == 2 ? -Ttt2[c2] : Ttt2[c2]) - Trr[c2][c3];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int a2 = p >> 1, a3 = p & 1, b2 = q >> 1, b3 = q & 1;
            const int c2 = hcls(a2, b2), c3 = hcls(a3, b3);
            put(hnode(1, a2, a3), hnode(0, b2, b3), base2[c2][c3] + rs[a2][b2][c3] + rt[c2][a3][b3] + st[p][q]);
        }
}

// Full brick element: packed k_e in precision T from node coordinates in S.
template <typename T, typename S>
__device__ __forceinline__ void brick_ke(const S (*xc)[3], T c, T (&k)[36]) {
    BrickRows<T> row;
    brick_rows<T, S>(xc, row);
    Pair<T> M[2][2][6], det[2][2];
    brick_M(row, c * T(0.125), M, det);
    brick_contract(M, k);
}

// Whether an element is distorted: max_q det J > thr min_q det J, or a det J <= 0.
template <typename T>
__device__ __forceinline__ bool brick_distorted(const Pair<T> (&det)[2][2], float thr) {
    T lo = pair_lo(det[0][0]), hi = lo;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const T a = pair_lo(det[q >> 1][q & 1]), b = pair_hi(det[q >> 1][q & 1]);
        lo = fmin(lo, fmin(a, b));
        hi = fmax(hi, fmax(a, b));
    }
    return !(lo > T(0)) || hi > T(thr) * lo;
}

// Distorted bricks (mixed precision): a brick whose max_q det J / min_q det J exceeds
// the threshold (or with a det J <= 0) takes its M_q, or determinants, from FP64.

// Gauss point q = 4 q1 + 2 q2 + q3 of a brick in FP64 from its node coordinates (edge
// differences formed in S): M[0..5] as brick_M scales it (s = c / 8), rounded to
// floats; M[6] = det 2J_q.  One copy of the code, so that every kernel gets the same
// bits; a few elements in a million come here.
template <typename S>
__device__ __noinline__ void brick_point(const S (*x)[3], int q, double s, float *M) {
    const int g[3] = {q >> 2, (q >> 1) & 1, q & 1};
    double w[3][2];  // the hats of each axis at the point
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        w[ax][0] = g[ax] ? FEM_GQ : FEM_GP;
        w[ax][1] = g[ax] ? FEM_GP : FEM_GQ;
    }
    double row[3][3];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            double v = 0.0;
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int n0 = ax == 0 ? hnode(0, i, j) : ax == 1 ? hnode(i, 0, j) : hnode(i, j, 0);
                    const int n1 = ax == 0 ? hnode(1, i, j) : ax == 1 ? hnode(i, 1, j) : hnode(i, j, 1);
                    v = fma(w[ax == 0 ? 1 : 0][i] * w[ax == 2 ? 1 : 2][j], (double)(x[n1][d] - x[n0][d]), v);
                }
            row[ax][d] = v;
        }
    const Vec3<double> R = {row[0][0], row[0][1], row[0][2]}, Sv = {row[1][0], row[1][1], row[1][2]},
                       U = {row[2][0], row[2][1], row[2][2]};
    const Vec3<double> C0 = cross3(Sv, U), C1 = cross3(U, R), C2 = cross3(R, Sv);
    const double d = dot3(R, C0), inv = rcp_rn(fabs(d)) * s;
    M[0] = (float)(dot3(C0, C0) * inv * (1.0 / 36.0));
    M[1] = (float)(dot3(C1, C1) * inv * (1.0 / 36.0));
    M[2] = (float)(dot3(C2, C2) * inv * (1.0 / 36.0));
    M[3] = (float)(dot3(C0, C1) * inv * (1.0 / 6.0));
    M[4] = (float)(dot3(C0, C2) * inv * (1.0 / 6.0));
    M[5] = (float)(dot3(C1, C2) * inv * (1.0 / 6.0));
    M[6] = (float)d;
}

// All eight points by the calling lane.
template <typename S>
__device__ __noinline__ void brick_points(const S (*x)[3], float c, float (*M)[7]) {
    for (int q = 0; q < 8; ++q) brick_point<S>(x, q, (double)c * 0.125, M[q]);
}

// All eight points of one element by eight consecutive lanes (q = lane & 7), the
// results to all of them.  One lane alone runs some 900 FP64 instructions of about 60
// cycles each, 20 us, for which its whole block waits at the next barrier: the one such
// block among a few hundred decided the kernel's time.
template <typename S>
__device__ __forceinline__ void brick_points_shared(const S (*x)[3], float c, float (&M)[8][7]) {
    float m[7];
    brick_point<S>(x, threadIdx.x & 7, (double)c * 0.125, m);
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int i = 0; i < 7; ++i) M[q][i] = __shfl_sync(0xffffffffu, m[i], q, 8);
}

__device__ __forceinline__ void pairs_of_points(const float (&P)[8][7], Pair<float> (&M)[2][2][6]) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < 6; ++i) M[q >> 1][q & 1][i] = pair(P[q][i], P[4 + q][i]);
}
__device__ __forceinline__ void pairs_of_dets(const float (&P)[8][7], Pair<float> (&det)[2][2]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) det[q >> 1][q & 1] = pair(P[q][6], P[4 + q][6]);
}

// Brick in FP32; returns whether it is distorted (then k is not its final matrix).
template <typename S>
__device__ __forceinline__ bool brick_ke_fp32(const S (*xc)[3], float c, float thr, float (&k)[36]) {
    BrickRows<float> row;
    brick_rows<float, S>(xc, row);
    Pair<float> M[2][2][6], det[2][2];
    brick_M(row, c * 0.125f, M, det);
    brick_contract(M, k);
    return brick_distorted(det, thr);
}

// Mixed precision brick: FP32 throughout, except for the FP64 M_q of a distorted
// element.  Returns true when the FP64 path was taken.
template <typename S>
__device__ __forceinline__ bool brick_ke_mixed(const S (*xc)[3], float c, float thr, float (&k)[36]) {
    BrickRows<float> row;
    brick_rows<float, S>(xc, row);
    Pair<float> M[2][2][6], det[2][2];
    brick_M(row, c * 0.125f, M, det);
    const bool flagged = brick_distorted(det, thr);
    if (flagged) {
        S x[8][3];  // copies: only these live in local memory
        float P[8][7];
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int d = 0; d < 3; ++d) x[a][d] = xc[a][d];
        brick_points<S>(x, c, P);
        pairs_of_points(P, M);
    }
    brick_contract(M, k);
    return flagged;
}

// ----------------------------------------------------------- brick mass matrix
// M_ab = c integral N_a N_b (the mass operator of Section 5's generalisation) by
// the same 2x2x2 rule: M_ab = c sum_q |det J_q| N_a(q) N_b(q).  N_a(q) is a product
// of 1D hats, so the sum factorises like the stiffness matrix: with
// D[q1][q2][q3] = |det J_q| and V = D contracted with the hat products F_c on every
// axis, M_ab = c V[cls(a1,b1)][cls(a2,b2)][cls(a3,b3)].  det(2 J_q) = 8 det J_q.
template <typename T>
__device__ __forceinline__ void brick_dets(const BrickRows<T> &row, Pair<T> (&det)[2][2]) {
#pragma unroll
    for (int q3 = 0; q3 < 2; ++q3) {
        const Vec3<Pair<T>> nS = neg3(row.S[q3]);
#pragma unroll
        for (int q2 = 0; q2 < 2; ++q2)
            det[q2][q3] = dot3(both3(row.R[q2][q3]), cross3(row.S[q3], nS, row.U[q2]));
    }
}

template <typename T>
__device__ __forceinline__ Pair<T> pair_abs(Pair<T> p) {
    const T a = pair_lo(p), b = pair_hi(p);
    return pair(a < T(0) ? -a : a, b < T(0) ? -b : b);
}

// Packed mass matrix from det(2 J_q): the determinants contracted with the hat
// products (times 6, see prod6) on every axis, as pairs over the classes 0 and 1 of
// axis 1.
template <typename T>
__device__ __forceinline__ void brick_mass_from_dets(const Pair<T> (&det)[2][2], T c, T (&m)[36]) {
    Pair<T> W[2][3], Y[3][3];
#pragma unroll
    for (int q2 = 0; q2 < 2; ++q2) prod6(pair_abs(det[q2][0]), pair_abs(det[q2][1]), W[q2]);
#pragma unroll
    for (int c3 = 0; c3 < 3; ++c3) {
        Pair<T> o[3];
        prod6(W[0][c3], W[1][c3], o);
#pragma unroll
        for (int c2 = 0; c2 < 3; ++c2) Y[c2][c3] = o[c2];
    }
    const T s = c * T(0.125 / 216.0);
    T V[3][3][3];
#pragma unroll
    for (int c2 = 0; c2 < 3; ++c2)
#pragma unroll
        for (int c3 = 0; c3 < 3; ++c3) {
            T o0, o1, o2;
            prod6(pair_lo(Y[c2][c3]), pair_hi(Y[c2][c3]), o0, o1, o2);
            V[0][c2][c3] = s * o0, V[1][c2][c3] = s * o1, V[2][c2][c3] = s * o2;
        }
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b)
            m[a * (a + 1) / 2 + b] = V[hcls(hb1(a), hb1(b))][hcls(hb2(a), hb2(b))][hcls(hb3(a), hb3(b))];
}

template <typename T, typename S>
__device__ __forceinline__ void brick_me(const S (*xc)[3], T c, T (&m)[36]) {
    BrickRows<T> row;
    brick_rows<T, S>(xc, row);
    Pair<T> det[2][2];
    brick_dets(row, det);
    brick_mass_from_dets(det, c, m);
}

// Brick determinants det(2 J_q) at the 8 Gauss points in precision T; with
// `mixed`, FP32 unless max_q det J / min_q det J exceeds thr (or some det J <= 0),
// then from FP64.  Returns true when FP64 was used.
template <typename T, typename S>
__device__ __forceinline__ bool brick_gauss_dets(const S (*xc)[3], float thr, bool mixed, Pair<T> (&det)[2][2]) {
    BrickRows<T> row;
    brick_rows<T, S>(xc, row);
    brick_dets(row, det);
    bool flagged = false;
    if constexpr (sizeof(T) == 4) {
        flagged = mixed && brick_distorted(det, thr);
        if (flagged) {
            S x[8][3];
            float P[8][7];
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int d = 0; d < 3; ++d) x[a][d] = xc[a][d];
            brick_points<S>(x, 0.f, P);
            pairs_of_dets(P, det);
        }
    }
    return flagged;
}

// Brick load vector f_a = s integral N_a = (s / 8) sum_q |det(2 J_q)| N_a(q): the
// determinants contracted with the single hats on every axis.
template <typename T>
__device__ __forceinline__ void brick_load_from_dets(const Pair<T> (&det)[2][2], T s, T (&f)[8]) {
    Pair<T> W[2][2];
#pragma unroll
    for (int q2 = 0; q2 < 2; ++q2) hat_pair(pair_abs(det[q2][0]), pair_abs(det[q2][1]), W[q2][0], W[q2][1]);
#pragma unroll
    for (int z = 0; z < 2; ++z) {
        Pair<T> y[2];
        hat_pair(W[0][z], W[1][z], y[0], y[1]);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const Pair<T> v = hat_in_pair(y[b]);
            f[hnode(0, b, z)] = s * T(0.125) * pair_lo(v);
            f[hnode(1, b, z)] = s * T(0.125) * pair_hi(v);
        }
    }
}

// Mixed precision: FP32, except for the FP64 determinants of a distorted element.
template <typename S>
__device__ __forceinline__ bool brick_me_mixed(const S (*xc)[3], float c, float thr, float (&m)[36]) {
    Pair<float> det[2][2];
    const bool flagged = brick_gauss_dets<float, S>(xc, thr, true, det);
    brick_mass_from_dets(det, c, m);
    return flagged;
}
template <typename S>
__device__ __forceinline__ bool brick_me_fp32(const S (*xc)[3], float c, float thr, float (&m)[36]) {
    BrickRows<float> row;
    brick_rows<float, S>(xc, row);
    Pair<float> det[2][2];
    brick_dets(row, det);
    brick_mass_from_dets(det, c, m);
    return brick_distorted(det, thr);
}

// The final matrix (mass or stiffness) of a distorted element, by eight consecutive
// lanes of a full warp; all of them get it.
template <typename S>
__device__ __forceinline__ void brick_distorted_shared(const S (*xc)[3], float c, bool mass, float (&k)[36]) {
    float P[8][7];
    brick_points_shared<S>(xc, c, P);
    if (mass) {
        Pair<float> det[2][2];
        pairs_of_dets(P, det);
        brick_mass_from_dets(det, c, k);
    } else {
        Pair<float> M[2][2][6];
        pairs_of_points(P, M);
        brick_contract(M, k);
    }
}

// ---------------------------------------------------------------- tetrahedron
// Rows of J are the edge vectors x_i - x_0 (i = 1..3).  The gradient of the
// barycentric function lambda_a is F_a / det J, where F_a is twice the area
// vector of the face opposite node a: F_1, F_2, F_3 are the cofactor rows
// (R1 x R2, R2 x R0, R0 x R1) and F_0 = (x3 - x1) x (x2 - x1) = -(F_1 + F_2 + F_3).
// Hence k_ab = c |det J|/6 grad(lambda_a).grad(lambda_b) = c F_a.F_b / (6 |det J|).
// F_0 is formed from its own coordinate differences rather than as -(F_1+F_2+F_3),
// so no entry is a cancelling sum (the FP32 error stays relative to the element).
template <typename T>
struct TetGeom {
    Vec3<T> R0, R1, R2, D1, D2;  // x1-x0, x2-x0, x3-x0, x2-x1, x3-x1
};

template <typename T, typename S>
__device__ __forceinline__ void tet_geom(const S (*xc)[3], TetGeom<T> &g) {
    auto d = [&](int i, int j) {
        return Vec3<T>{T(xc[i][0] - xc[j][0]), T(xc[i][1] - xc[j][1]), T(xc[i][2] - xc[j][2])};
    };
    g.R0 = d(1, 0);
    g.R1 = d(2, 0);
    g.R2 = d(3, 0);
    g.D1 = d(2, 1);
    g.D2 = d(3, 1);
}

template <typename T>
__device__ __forceinline__ void tet_faces(const TetGeom<T> &g, Vec3<T> (&F)[4], T &det) {
    F[1] = cross3(g.R1, g.R2);
    F[2] = cross3(g.R2, g.R0);
    F[3] = cross3(g.R0, g.R1);
    F[0] = cross3(g.D2, g.D1);
    det = dot3(g.R0, F[1]);
}

template <typename T>
__device__ __forceinline__ void tet_from_faces(const Vec3<T> (&F)[4], T det, T c, T (&k)[10]) {
    const T s = c * rcp_rn(T(6) * (det < T(0) ? -det : det));
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) k[a * (a + 1) / 2 + b] = dot3(F[a], F[b]) * s;
}

template <typename T, typename S>
__device__ __forceinline__ void tet_ke(const S (*xc)[3], T c, T (&k)[10]) {
    TetGeom<T> g;
    tet_geom<T, S>(xc, g);
    Vec3<T> F[4];
    T det;
    tet_faces(g, F, det);
    tet_from_faces(F, det, c, k);
}

// Mixed precision tetrahedron: the aspect ratio (longest edge over shortest
// altitude = L_max |F|_max / |det J|) is evaluated in FP32; above `thr` the
// face vectors are recomputed with one rounding each and the determinant to
// FP64 accuracy -- in double-single FP32 arithmetic (det3_ds) by default, or in
// FP64 arithmetic when fp64_det is set -- and rounded once.  Returns true when
// the accurate path was taken.
template <typename S>
__device__ __forceinline__ bool tet_geometry_mixed(const S (*xc)[3], float thr, bool fp64_det, Vec3<float> (&F)[4],
                                                   float &det) {
    TetGeom<float> g;
    tet_geom<float, S>(xc, g);
    tet_faces(g, F, det);
    const Vec3<float> E5 = {g.R2.x - g.R1.x, g.R2.y - g.R1.y, g.R2.z - g.R1.z};
    const float L2 = fmaxf(fmaxf(fmaxf(dot3(g.R0, g.R0), dot3(g.R1, g.R1)), fmaxf(dot3(g.R2, g.R2), dot3(g.D1, g.D1))),
                           fmaxf(dot3(g.D2, g.D2), dot3(E5, E5)));
    const float A2 = fmaxf(fmaxf(dot3(F[0], F[0]), dot3(F[1], F[1])), fmaxf(dot3(F[2], F[2]), dot3(F[3], F[3])));
    const bool flagged = !(L2 * A2 <= thr * thr * det * det);
    if (flagged) {
        // Distorted: cofactors (face vectors) with one rounding each, and the
        // Jacobian determinant to FP64 accuracy.  The double-single form keeps
        // the work off the FP64 pipe (1/64 of the FP32 rate on this part), where
        // a warp with one distorted lane would otherwise stall all 32.
        F[1] = cross3_accurate(g.R1, g.R2);
        F[2] = cross3_accurate(g.R2, g.R0);
        F[3] = cross3_accurate(g.R0, g.R1);
        F[0] = cross3_accurate(g.D2, g.D1);
        if (fp64_det) {
            // FP64 from the coordinates: the edge vectors are exact in double
            // (differences of floats), the products of two of them too
            double r[3][3];
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int k = 0; k < 3; ++k) r[i][k] = (double)xc[i + 1][k] - (double)xc[0][k];
            const double m0 = fma(r[1][1], r[2][2], -(r[1][2] * r[2][1]));
            const double m1 = fma(r[1][2], r[2][0], -(r[1][0] * r[2][2]));
            const double m2 = fma(r[1][0], r[2][1], -(r[1][1] * r[2][0]));
            det = (float)fma(r[0][0], m0, fma(r[0][1], m1, r[0][2] * m2));
        } else {
            det = det3_ds<S>(xc);
        }
    }
    return flagged;
}

template <typename S>
__device__ __forceinline__ bool tet_ke_mixed(const S (*xc)[3], float c, float thr, bool fp64_det, float (&k)[10]) {
    Vec3<float> F[4];
    float det;
    const bool flagged = tet_geometry_mixed<S>(xc, thr, fp64_det, F, det);
    tet_from_faces(F, det, c, k);
    return flagged;
}

// ------------------------------------------------------------ tet mass matrix
// M_ab = c integral lambda_a lambda_b = c |T| (1 + delta_ab) / 20, |T| = |det J| / 6.
template <typename T>
__device__ __forceinline__ void tet_mass_from_det(T det, T c, T (&m)[10]) {
    const T s = c * (det < T(0) ? -det : det) * T(1.0 / 120.0);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) m[a * (a + 1) / 2 + b] = a == b ? s + s : s;
}

template <typename T, typename S>
__device__ __forceinline__ void tet_me(const S (*xc)[3], T c, T (&m)[10]) {
    TetGeom<T> g;
    tet_geom<T, S>(xc, g);
    Vec3<T> F[4];
    T det;
    tet_faces(g, F, det);
    tet_mass_from_det(det, c, m);
}

// Mixed precision: the same indicator and FP64-accurate determinant as k_e.
template <typename S>
__device__ __forceinline__ bool tet_me_mixed(const S (*xc)[3], float c, float thr, bool fp64_det, float (&m)[10]) {
    Vec3<float> F[4];
    float det;
    const bool flagged = tet_geometry_mixed<S>(xc, thr, fp64_det, F, det);
    tet_mass_from_det(det, c, m);
    return flagged;
}

}  // namespace fem
