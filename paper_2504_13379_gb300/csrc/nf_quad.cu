// nf_quad.cu -- RBF quadrature weights (§3.2 Eq. (3.5), §3.3 Eq. (3.6)) on the GPU, in FP64.
//
// Per element: the local frame (flat: centroid; surface: projection point from three cutting
// planes, central projection of the stencil to the element plane and the Jacobian of the map),
// the saddle system of Eq. (3.4) with r^3 and monomials up to deg, analytic right-hand side, LU
// with partial pivoting in shared memory, element weights; then a deterministic gather
// q_i = sum of the element weights of every stencil entry naming node i, in a fixed order (32
// strands of the (element, position) ranks and a butterfly over them).
//
// Bound: the FP64 pipe, two lanes per clock and SM -- a warp instruction costs 16 clocks however
// few of its lanes are active.  The elimination of a k = 48, degree-4 system (N = 63) is 2,700
// such instructions; everything around it is laid out to keep lanes full: what is the same for a
// whole element (frame, moments, edges) is computed by one thread per element in a kernel of
// its own, pivots are compared as integers, one reciprocal per column replaces the divisions.
#include "nf_internal.cuh"

#include <algorithm>
#include <cmath>
namespace nfi {

constexpr int QW_THREADS = 128;
constexpr int QW_KMAX = 64;
constexpr int QW_DEGMAX = 4;
constexpr double QW_PIVOT_TOL = 1e-14;
constexpr double QW_PROJ_COND_MAX = 1e10;

// ---------------------------------------------------------------- adjacency
constexpr unsigned long long EMPTY_KEY = 0xffffffffffffffffull;

__device__ __forceinline__ unsigned long long edge_key(int32_t a, int32_t b) {
    const unsigned lo = (unsigned)min(a, b), hi = (unsigned)max(a, b);
    return ((unsigned long long)lo << 32) | hi;
}
__device__ __forceinline__ unsigned long long mix64(unsigned long long x) {
    x ^= x >> 33;
    x *= 0xff51afd7ed558ccdull;
    x ^= x >> 33;
    x *= 0xc4ceb9fe1a85ec53ull;
    x ^= x >> 33;
    return x;
}

__global__ void edge_insert_kernel(const int32_t *tris, int64_t m, unsigned long long *keys, long long *v0,
                                   long long *v1, int64_t cap, int *flag) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 3 * m) return;
    const int64_t e = t / 3;
    const int kk = (int)(t % 3);
    const unsigned long long key = edge_key(tris[3 * e + kk], tris[3 * e + (kk + 1) % 3]);
    int64_t h = (int64_t)(mix64(key) & (unsigned long long)(cap - 1));
    for (int64_t probe = 0; probe < cap; ++probe) {
        const unsigned long long prev = atomicCAS(&keys[h], EMPTY_KEY, key);
        if (prev == EMPTY_KEY || prev == key) {
            if (atomicCAS((unsigned long long *)&v0[h], (unsigned long long)-1ll, (unsigned long long)t) !=
                (unsigned long long)-1ll) {
                if (atomicCAS((unsigned long long *)&v1[h], (unsigned long long)-1ll, (unsigned long long)t) !=
                    (unsigned long long)-1ll)
                    atomicExch(flag, 1);  // edge shared by more than two elements
            }
            return;
        }
        h = (h + 1) & (cap - 1);
    }
    atomicExch(flag, 2);
}

__global__ void edge_lookup_kernel(const int32_t *tris, int64_t m, const unsigned long long *keys,
                                   const long long *v0, const long long *v1, int64_t cap, const int *flag,
                                   int64_t *nbr) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 3 * m) return;
    const int64_t e = t / 3;
    const int kk = (int)(t % 3);
    const unsigned long long key = edge_key(tris[3 * e + kk], tris[3 * e + (kk + 1) % 3]);
    int64_t h = (int64_t)(mix64(key) & (unsigned long long)(cap - 1));
    nbr[t] = -1;
    if (*flag) return;  // non-manifold: every element falls back to parallel projection
    for (int64_t probe = 0; probe < cap; ++probe) {
        if (keys[h] == key) {
            const long long a = v0[h], b = v1[h];
            const long long other = (a == t) ? b : a;
            nbr[t] = (other >= 0) ? other / 3 : -1;
            return;
        }
        if (keys[h] == EMPTY_KEY) return;
        h = (h + 1) & (cap - 1);
    }
}

// ---------------------------------------------------------------- small geometry
struct V3 {
    double x, y, z;
};
__device__ __forceinline__ V3 v3(const double *p) { return {p[0], p[1], p[2]}; }
__device__ __forceinline__ V3 sub(V3 a, V3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ V3 add(V3 a, V3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ V3 scl(V3 a, double s) { return {a.x * s, a.y * s, a.z * s}; }
__device__ __forceinline__ double dot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ V3 cross(V3 a, V3 b) {
    return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
__device__ __forceinline__ double nrm(V3 a) { return sqrt(dot(a, a)); }

__device__ V3 element_normal(const double *X, const double *NS, const int32_t *tri) {
    const V3 a = v3(X + 3 * (int64_t)tri[0]), b = v3(X + 3 * (int64_t)tri[1]), c = v3(X + 3 * (int64_t)tri[2]);
    V3 nE = cross(sub(b, a), sub(c, a));
    nE = scl(nE, 1.0 / nrm(nE));
    const V3 ref = add(add(v3(NS + 3 * (int64_t)tri[0]), v3(NS + 3 * (int64_t)tri[1])), v3(NS + 3 * (int64_t)tri[2]));
    if (dot(nE, ref) < 0.0) nE = scl(nE, -1.0);
    return nE;
}

// Solve A p = b (3x3) via the Gauss-Jordan inverse; returns ||A||_inf ||A^-1||_inf.
__device__ double solve3x3(const double A[9], const double b[3], double p[3]) {
    double W[3][6];
    double anorm = 0.0;
    for (int r = 0; r < 3; ++r) {
        anorm = fmax(anorm, fabs(A[3 * r]) + fabs(A[3 * r + 1]) + fabs(A[3 * r + 2]));
        for (int c = 0; c < 6; ++c) W[r][c] = (c < 3) ? A[3 * r + c] : (c - 3 == r ? 1.0 : 0.0);
    }
    for (int c = 0; c < 3; ++c) {
        int piv = c;
        for (int r = c + 1; r < 3; ++r)
            if (fabs(W[r][c]) > fabs(W[piv][c])) piv = r;
        if (W[piv][c] == 0.0) return INFINITY;
        if (piv != c)
            for (int cc = 0; cc < 6; ++cc) {
                const double t = W[c][cc];
                W[c][cc] = W[piv][cc];
                W[piv][cc] = t;
            }
        const double pv = W[c][c];
        for (int cc = 0; cc < 6; ++cc) W[c][cc] /= pv;
        for (int r = 0; r < 3; ++r) {
            if (r == c) continue;
            const double l = W[r][c];
            for (int cc = 0; cc < 6; ++cc) W[r][cc] -= l * W[c][cc];
        }
    }
    double inorm = 0.0;
    for (int r = 0; r < 3; ++r) inorm = fmax(inorm, fabs(W[r][3]) + fabs(W[r][4]) + fabs(W[r][5]));
    for (int r = 0; r < 3; ++r) p[r] = W[r][3] * b[0] + W[r][4] * b[1] + W[r][5] * b[2];
    return anorm * inorm;
}

// ---------------------------------------------------------------- per-element frame
// What a whole element shares, one thread per element.
constexpr int QF_C = 0, QF_E1 = 3, QF_E2 = 6, QF_N = 9, QF_P = 12, QF_CENTRAL = 15;
constexpr int QF_TV = 16;     // local vertices x0, y0, x1, y1, x2, y2
constexpr int QF_EDGE = 22;   // per edge: unit tangent tx, ty, length
constexpr int QF_SIGN = 31;   // +-1: orientation of the local triangle
constexpr int QF_MOM = 32;    // moments int_T x^a y^b in the order of the monomials
constexpr int QF_SIZE = 48;   // doubles per element

struct QwArgs {
    const double *X;
    const double *NS;   // null when flat
    int dim;
    const int32_t *tris;
    int64_t m;
    const int32_t *sten;
    int k;
    int deg;
    const int64_t *nbr;  // 3 per element (surfaces)
    double *frame;       // m x QF_SIZE
    double *elem_w;      // m x k
    unsigned long long *first_bad;
};

// Moments of the triangle: with u_i = x_i s + y_i t for its vertices,
//   int_T (x s + y t)^d = 2 |T| d! / (d + 2)! h_d(u_0, u_1, u_2),
// h_d the complete homogeneous symmetric polynomial, so int_T x^a y^b is
// 2 |T| a! b! / (a + b + 2)! times the s^a t^b coefficient of h_d.  The h_d follow from
// h_d(u_0..u_i) = h_d(u_0..u_{i-1}) + u_i h_{d-1}(u_0..u_i): about 70 operations for degree 4.
__device__ void triangle_moments(int deg, const double *v, double *mom) {
    double H[QW_DEGMAX + 1][QW_DEGMAX + 1];  // H[d][b]: coefficient of s^(d - b) t^b
#pragma unroll
    for (int d = 0; d <= QW_DEGMAX; ++d)
#pragma unroll
        for (int b = 0; b <= QW_DEGMAX; ++b) H[d][b] = (d == 0 && b == 0) ? 1.0 : 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int d = 1; d <= QW_DEGMAX; ++d)
            if (d <= deg)
#pragma unroll
                for (int b = 0; b <= QW_DEGMAX; ++b)
                    if (b <= d) {
                        if (b < d) H[d][b] = fma(v[2 * i], H[d - 1][b], H[d][b]);
                        if (b > 0) H[d][b] = fma(v[2 * i + 1], H[d - 1][b - 1], H[d][b]);
                    }
    const double area2 = fabs((v[2] - v[0]) * (v[5] - v[1]) - (v[3] - v[1]) * (v[4] - v[0]));
    const double f[QW_DEGMAX + 3] = {1.0, 1.0, 2.0, 6.0, 24.0, 120.0, 720.0};
    int c = 0;
#pragma unroll
    for (int d = 0; d <= QW_DEGMAX; ++d)
#pragma unroll
        for (int b = 0; b <= QW_DEGMAX; ++b)  // x^(d - b) y^b: descending power of x
            if (b <= d) {
                if (d <= deg) mom[c] = area2 * (f[d - b] * f[b] / f[d + 2]) * H[d][b];
                ++c;
            }
}

__global__ void quad_frame_kernel(QwArgs a) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= a.m) return;
    const int32_t *tri = a.tris + 3 * e;
    double *f = a.frame + e * QF_SIZE;
    double tv[6];
    if (a.dim == 2) {
        double c[2];
        for (int d = 0; d < 2; ++d) {
            c[d] = ((a.X[2 * (int64_t)tri[0] + d] + a.X[2 * (int64_t)tri[1] + d]) + a.X[2 * (int64_t)tri[2] + d]) / 3.0;
            f[QF_C + d] = c[d];
        }
        for (int i = 0; i < 3; ++i)
            for (int d = 0; d < 2; ++d) tv[2 * i + d] = a.X[2 * (int64_t)tri[i] + d] - c[d];
    } else {
        const V3 A = v3(a.X + 3 * (int64_t)tri[0]), B = v3(a.X + 3 * (int64_t)tri[1]), C = v3(a.X + 3 * (int64_t)tri[2]);
        const V3 cE = {((A.x + B.x) + C.x) / 3.0, ((A.y + B.y) + C.y) / 3.0, ((A.z + B.z) + C.z) / 3.0};
        const V3 nE = element_normal(a.X, a.NS, tri);
        V3 e1 = sub(B, A);
        e1 = scl(e1, 1.0 / nrm(e1));
        const V3 e2 = cross(nE, e1);
        double Am[9], rhs[3], p[3] = {0, 0, 0};
        bool central = true;
        for (int kk = 0; kk < 3; ++kk) {
            const int64_t nb = a.nbr[3 * e + kk];
            if (nb < 0) {
                central = false;
                break;
            }
            const V3 dn = sub(nE, element_normal(a.X, a.NS, a.tris + 3 * nb));
            Am[3 * kk] = dn.x;
            Am[3 * kk + 1] = dn.y;
            Am[3 * kk + 2] = dn.z;
            rhs[kk] = dot(dn, v3(a.X + 3 * (int64_t)tri[kk]));
        }
        if (central) {
            const double cond = solve3x3(Am, rhs, p);
            central = isfinite(cond) && cond < QW_PROJ_COND_MAX;
        }
        const V3 put[4] = {cE, e1, e2, nE};
        for (int i = 0; i < 4; ++i) f[3 * i] = put[i].x, f[3 * i + 1] = put[i].y, f[3 * i + 2] = put[i].z;
        for (int i = 0; i < 3; ++i) f[QF_P + i] = p[i];
        f[QF_CENTRAL] = central ? 1.0 : 0.0;
        const V3 vs[3] = {A, B, C};
        for (int i = 0; i < 3; ++i) {
            const V3 v = sub(vs[i], cE);
            tv[2 * i] = dot(v, e1);
            tv[2 * i + 1] = dot(v, e2);
        }
    }
    for (int i = 0; i < 6; ++i) f[QF_TV + i] = tv[i];
    for (int i = 0; i < 3; ++i) {
        const int j = (i + 1) % 3;
        const double ex = tv[2 * j] - tv[2 * i], ey = tv[2 * j + 1] - tv[2 * i + 1];
        const double L = sqrt(ex * ex + ey * ey);
        f[QF_EDGE + 3 * i] = ex / L;
        f[QF_EDGE + 3 * i + 1] = ey / L;
        f[QF_EDGE + 3 * i + 2] = L;
    }
    f[QF_SIGN] = (tv[2] - tv[0]) * (tv[5] - tv[1]) - (tv[3] - tv[1]) * (tv[4] - tv[0]) > 0.0 ? 1.0 : -1.0;
    triangle_moments(a.deg, tv, f + QF_MOM);
}

// ---------------------------------------------------------------- analytic integrals
// int_T |x - p|^3 dx in the frame f: a signed fan of three wedges.  A wedge over an edge at
// distance d from p, whose ends lie at a_A, a_B along it (r_A, r_B from p), is
//   d^5 [G(a_B / d) - G(a_A / d)] / 5, G the antiderivative of sec^5:
//   d (a r^3) / 4 + 3 d^3 (a r) / 8 + 3 d^5 asinh(a / d) / 8 between the ends, and
//   asinh(a_B / d) - asinh(a_A / d) = log((r_A + r_B + L) / (r_A + r_B - L)),
// one logarithm per edge instead of two asinh.  As p approaches the edge the logarithm grows
// while d^5 vanishes; below r_A + r_B - L = 1e-13 (r_A + r_B) the term is under 1e-30.
__device__ double tri_r3_integral(double px, double py, const double *f) {
    double r[3], dx[3], dy[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        dx[i] = f[QF_TV + 2 * i] - px;
        dy[i] = f[QF_TV + 2 * i + 1] - py;
        r[i] = sqrt(dx[i] * dx[i] + dy[i] * dy[i]);
    }
    double total = 0.0;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int j = (e + 1) % 3;
        const double tx = f[QF_EDGE + 3 * e], ty = f[QF_EDGE + 3 * e + 1], L = f[QF_EDGE + 3 * e + 2];
        const double cr = dx[e] * ty - dy[e] * tx, d = fabs(cr);
        if (d == 0.0) continue;
        const double aA = dx[e] * tx + dy[e] * ty, aB = aA + L;
        const double d2 = d * d, s = r[e] + r[j], t = s - L;
        // differences between the ends from r_B - r_A = L (a_A + a_B) / (r_A + r_B), without the
        // cancellation of a_B r_B - a_A r_A for far points (a third less error)
        const double rA2 = r[e] * r[e], rB2 = r[j] * r[j], ad = aA * (L * (aA + aB) / s);
        const double d1 = L * r[j] + ad, d3 = L * (r[j] * rB2) + ad * (rA2 + r[e] * r[j] + rB2);
        double part = 0.25 * d3 + 0.375 * d2 * d1;
        if (t > 1e-13 * s) part += 0.375 * (d2 * d2) * log((s + L) / t);
        total += cr * part;
    }
    return f[QF_SIGN] * (total / 5.0);
}

// ---------------------------------------------------------------- per-element solve
// |v| as an ordered integer key; a NaN never wins a comparison.
__device__ __forceinline__ unsigned long long abs_key(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    return b > 0x7ff0000000000000ull ? 0ull : b + 1ull;
}

// sqrt(q) for q in FP32 range: reciprocal square root of FP32, one Goldschmidt iteration for the
// root and half its reciprocal, and a final residual correction (Markstein, "IA-64 and Elementary
// Functions", 2000): seven FP64 operations, half of the library call's.  Within one unit in
// the last place of sqrt (a run of its own over 6.5e7 random arguments found no difference; the tests
// check the weights, not this function).  0 and values outside FP32's normal range take the library's.
__device__ __forceinline__ double root(double q) {
    const float qf = (float)q;
    if (!(qf > 1e-30f && qf < 1e30f)) return sqrt(q);
    const double y = (double)rsqrtf(qf);
    double g = q * y, h = 0.5 * y;
    const double r = fma(-g, h, 0.5);
    g = fma(g, r, g);
    h = fma(h, r, h);
    return fma(fma(-g, g, q), h, g);
}

// One block per element.  After the frame's node-parallel part, column c of the elimination is
// three phases with two barriers: (1) the row swap and the multipliers l_r = M_rc / pivot;
// (2) warp 0 updates column c + 1, finds its pivot (first maximal entry) and the pivot's
// reciprocal while the other warps update the remaining columns, entries dealt out evenly.
// The leading dimension is odd, so columns are read without bank conflicts.
__global__ void __launch_bounds__(QW_THREADS) quad_element_kernel(QwArgs a) {
    extern __shared__ __align__(16) double qsm[];
    const int k = a.k;
    const int P = (a.deg + 1) * (a.deg + 2) / 2;
    const int N = k + P, ld = N | 1;
    double *M = qsm;                  // N x ld
    double *z = M + (size_t)N * ld;   // N + 1
    double *lc = z + N + 1;           // N: multipliers of the current column
    double *invd = lc + N;            // N: reciprocals of the pivots
    double *xi = invd + N;            // 2k scaled local coordinates
    double *jac = xi + 2 * k;         // k
    double *f = jac + k;              // QF_SIZE: the element's frame
    __shared__ double s_red[QW_THREADS / 32], s_inv, s_old;
    __shared__ unsigned long long s_best;
    __shared__ int s_piv;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t e = blockIdx.x;

    for (int i = tid; i < QF_SIZE; i += QW_THREADS) f[i] = a.frame[e * QF_SIZE + i];
    __syncthreads();
    // node r of the stencil (k <= 64: warps 0 and 1): projection, Jacobian, r^3 integral
    double x = 0.0, y = 0.0, zr = 0.0, jr = 1.0, r2 = 0.0;
    if (tid < k) {
        const int64_t j = a.sten[e * k + tid];
        if (a.dim == 2) {
            x = a.X[2 * j] - f[QF_C];
            y = a.X[2 * j + 1] - f[QF_C + 1];
        } else {
            const V3 X = v3(a.X + 3 * j), ns = v3(a.NS + 3 * j);
            const V3 cE = v3(f + QF_C), e1 = v3(f + QF_E1), e2 = v3(f + QF_E2), nE = v3(f + QF_N), p = v3(f + QF_P);
            V3 q;
            if (f[QF_CENTRAL] != 0.0) {
                const V3 xp = sub(X, p);
                const double t = dot(sub(cE, p), nE) / dot(xp, nE);
                q = add(p, scl(xp, t));
                // |n_E . u| / |n_S . u| with u = (x - p) / |x - p|: the length cancels
                jr = (1.0 / (t * t)) * (fabs(dot(nE, xp)) / fabs(dot(ns, xp)));
            } else {
                const double sd = dot(sub(X, cE), nE);
                q = sub(X, scl(nE, sd));
                jr = 1.0 / fabs(dot(ns, nE));
            }
            const V3 v = sub(q, cE);
            x = dot(v, e1);
            y = dot(v, e2);
        }
        r2 = x * x + y * y;
        zr = tri_r3_integral(x, y, f);
        jac[tid] = jr;
    }
    {
        unsigned long long key = (unsigned long long)__double_as_longlong(r2);  // r2 >= 0: ordered as integers
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ok = __shfl_xor_sync(0xffffffffu, key, o);
            key = ok > key ? ok : key;
        }
        if (lane == 0) s_red[warp] = __longlong_as_double((long long)key);
    }
    __syncthreads();
    // the stencil's radius rho scales the coordinates; the unscaled integrals follow by powers
    if (tid < N) {
        const unsigned long long k0 = (unsigned long long)__double_as_longlong(s_red[0]),
                                 k1 = (unsigned long long)__double_as_longlong(s_red[1]);
        const double rho = sqrt(__longlong_as_double((long long)(k0 > k1 ? k0 : k1)));
        const double ir = 1.0 / rho, ir2 = ir * ir;
        if (tid == 0) s_old = rho;
        if (tid < k) {
            x = x / rho;
            y = y / rho;
            xi[2 * tid] = x;
            xi[2 * tid + 1] = y;
            z[tid] = zr * (ir2 * ir2 * ir);
            M[tid * ld + tid] = 0.0;
            double px = 1.0;
            for (int ax = 0; ax <= a.deg; ++ax) {  // x^ax y^b at column of degree ax + b
                double v = px;
                for (int b = 0; ax + b <= a.deg; ++b) {
                    const int d = ax + b, c = k + d * (d + 1) / 2 + b;
                    M[tid * ld + c] = v;
                    M[c * ld + tid] = v;
                    v *= y;
                }
                px *= x;
            }
        } else {
            const int c = tid - k;
            int d = 0;
            while ((d + 1) * (d + 2) / 2 <= c) ++d;
            double sc = ir2;
            for (int i = 0; i < d; ++i) sc *= ir;
            z[tid] = f[QF_MOM + c] * sc;
            for (int cc = k; cc < N; ++cc) M[tid * ld + cc] = 0.0;
        }
    }
    __syncthreads();
    const double rho = s_old;
    // r^3 for every pair of stencil nodes once (the matrix is symmetric)
    for (int t = tid; t < k * (k - 1) / 2; t += QW_THREADS) {
        int c = (int)((1.f + sqrtf(1.f + 8.f * (float)t)) * 0.5f);
        while (c * (c - 1) / 2 > t) --c;
        while ((c + 1) * c / 2 <= t) ++c;
        const int r = t - c * (c - 1) / 2;
        const double dx = xi[2 * r] - xi[2 * c], dy = xi[2 * r + 1] - xi[2 * c + 1];
        const double rr = root(dx * dx + dy * dy), v = rr * rr * rr;
        M[r * ld + c] = v;
        M[c * ld + r] = v;
    }
    __syncthreads();
    // infinity norm, and the pivot of column 0
    {
        double s = 0.0;
        if (tid < N)
            for (int c = 0; c < N; ++c) s += fabs(M[tid * ld + c]);
        unsigned long long key = (unsigned long long)__double_as_longlong(s);
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ok = __shfl_xor_sync(0xffffffffu, key, o);
            key = ok > key ? ok : key;
        }
        if (lane == 0) s_red[warp] = __longlong_as_double((long long)key);
    }
    // warp 0: pivot among the entries v[i] of rows c + lane + 32 i of column c
    auto find_pivot = [&](int c, const double (&v)[3]) {
        unsigned long long best = 0ull;
        int piv = N;
        double pv = 0.0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int r = c + lane + 32 * i;
            const unsigned long long key = r < N ? abs_key(v[i]) : 0ull;
            if (key > best) best = key, piv = r, pv = v[i];
        }
        const unsigned hi = (unsigned)(best >> 32), mhi = __reduce_max_sync(0xffffffffu, hi);
        const unsigned lo = hi == mhi ? (unsigned)best : 0u, mlo = __reduce_max_sync(0xffffffffu, lo);
        const bool top = hi == mhi && (unsigned)best == mlo;
        const unsigned first = __reduce_min_sync(0xffffffffu, top ? (unsigned)piv : 0xffffffffu);
        if (lane == 0) s_old = v[0];
        if (top && (unsigned)piv == first) {  // one lane: rows are distinct
            s_piv = piv;
            s_best = best;
            const double inv = 1.0 / pv;
            s_inv = inv;
            invd[c] = inv;
        }
    };
    if (warp == 0) {
        double v[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) v[i] = lane + 32 * i < N ? M[(lane + 32 * i) * ld] : 0.0;
        find_pivot(0, v);
    }
    __syncthreads();
    double anorm = 0.0;
    for (int w = 0; w < (N + 31) / 32; ++w) anorm = s_red[w] > anorm ? s_red[w] : anorm;
    const unsigned long long tol = isnan(anorm) ? ~0ull : abs_key(QW_PIVOT_TOL * anorm);

    for (int c = 0; c < N; ++c) {
        const int piv = s_piv;
        const double inv = s_inv;
        if (!(s_best > tol)) {
            if (tid == 0) atomicMin(a.first_bad, (unsigned long long)e);
            return;  // uniform across the block
        }
        const int m = N - c - 1;  // rows below the pivot
        if (piv != c) {
            for (int cc = c + tid; cc < N; cc += QW_THREADS) {
                const double t = M[c * ld + cc];
                M[c * ld + cc] = M[piv * ld + cc];
                M[piv * ld + cc] = t;
            }
            if (tid == QW_THREADS - 1) {
                const double t = z[c];
                z[c] = z[piv];
                z[piv] = t;
            }
        }
        // multipliers (the last warps; row piv holds the displaced row c)
        const int lr = c + QW_THREADS - tid;  // c + 1 .. c + 128
        if (lr < N) lc[lr] = (lr == piv ? s_old : M[lr * ld + c]) * inv;
        __syncthreads();
        if (warp == 0 && m > 0) {
            const double u = M[c * ld + c + 1];
            double v[3] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int r = c + 1 + lane + 32 * i;
                if (r < N) {
                    v[i] = fma(-lc[r], u, M[r * ld + c + 1]);
                    M[r * ld + c + 1] = v[i];
                }
            }
            find_pivot(c + 1, v);
        }
        // columns c + 2 .. N - 1 and the right-hand side: m entries per row, dealt out evenly
        if (m > 0) {
            int r = tid / m, cc = tid - r * m;
            const int dr = QW_THREADS / m, dc = QW_THREADS - dr * m;
            while (r < m) {
                const double l = lc[c + 1 + r];
                if (cc + 1 < m) {
                    double *p = M + (c + 1 + r) * ld + c + 2 + cc;
                    *p = fma(-l, M[c * ld + c + 2 + cc], *p);
                } else {
                    z[c + 1 + r] = fma(-l, z[c], z[c + 1 + r]);
                }
                r += dr;
                cc += dc;
                if (cc >= m) cc -= m, ++r;
            }
        }
        __syncthreads();
    }
    // back substitution, column by column: lane holds the rows lane + 32 i
    if (warp == 0) {
        double v[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) v[i] = lane + 32 * i < N ? z[lane + 32 * i] : 0.0;
        for (int r = N - 1; r >= 0; --r) {
            const int own = r >> 5;
            double s = own == 0 ? v[0] : (own == 1 ? v[1] : v[2]);
            s = __shfl_sync(0xffffffffu, s, r & 31) * invd[r];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int row = lane + 32 * i;
                if (i <= own && row < r) v[i] = fma(-M[row * ld + r], s, v[i]);
                if (row == r) v[i] = s;
            }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
            if (lane + 32 * i < k) z[lane + 32 * i] = v[i];
    }
    __syncthreads();
    if (tid < k) a.elem_w[e * k + tid] = z[tid] * rho * rho * jac[tid];
}

// ---------------------------------------------------------------- deterministic gather
__global__ void count_refs_kernel(const int32_t *sten, int64_t mk, int32_t *cnt) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < mk) atomicAdd(&cnt[sten[t]], 1);
}
__global__ void fill_refs_kernel(const int32_t *sten, int64_t mk, const int32_t *start, int32_t *fill,
                                 int64_t *refs) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= mk) return;
    const int32_t i = sten[t];
    refs[start[i] + atomicAdd(&fill[i], 1)] = t;
}
// q_i = sum over its references, sorted by flat (element * k + position): one warp per node.  A
// reference's rank is the number of smaller ones (they are distinct); lane l adds the entries of
// ranks l, l + 32, ... in ascending order, then a butterfly adds the lanes: a fixed order.
// Nodes with more than GW_CAP references are sorted in place by one lane first.
constexpr int GW_CAP = 256, GW_WARPS = 4;
__global__ void __launch_bounds__(32 * GW_WARPS)
gather_weights_kernel(int64_t n, const int32_t *start, int64_t *refs, const double *elem_w, double *q) {
    __shared__ int64_t ref[GW_WARPS][GW_CAP];
    __shared__ double val[GW_WARPS][GW_CAP];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * GW_WARPS + warp;
    if (i >= n) return;
    const int32_t b = start[i], e = start[i + 1], cnt = e - b;
    double acc = 0.0;
    if (cnt <= GW_CAP) {
        for (int p = lane; p < cnt; p += 32) ref[warp][p] = refs[b + p];
        __syncwarp();
        for (int p = lane; p < cnt; p += 32) {
            const int64_t mine = ref[warp][p];
            int rank = 0;
            for (int j = 0; j < cnt; ++j) rank += ref[warp][j] < mine ? 1 : 0;
            val[warp][rank] = elem_w[mine];
        }
        __syncwarp();
        for (int p = lane; p < cnt; p += 32) acc += val[warp][p];
    } else {
        if (lane == 0)
            for (int32_t p = b + 1; p < e; ++p) {
                const int64_t v = refs[p];
                int32_t s = p;
                while (s > b && refs[s - 1] > v) {
                    refs[s] = refs[s - 1];
                    --s;
                }
                refs[s] = v;
            }
        __syncwarp();
        for (int p = lane; p < cnt; p += 32) acc += elem_w[refs[b + p]];
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) q[i] = acc;
}

}  // namespace nfi

using namespace nfi;

extern "C" nf_status nf_quad_weights(const double *nodes, const double *normals, int64_t n, int dim,
                                     const int32_t *tris, int64_t m, const int32_t *stencils, int k, int deg,
                                     double *q, int64_t *bad_element, void *stream) {
    clear_error();
    if (bad_element) *bad_element = -1;
    NF_ARG(nodes && tris && stencils && q, "nodes, tris, stencils and q must be non-NULL");
    NF_ARG(dim == 2 || dim == 3, "dim must be 2 or 3");
    NF_ARG((dim == 3) == (normals != nullptr), "normals are required for dim 3 and must be NULL for dim 2");
    NF_ARG(n >= 3 && n < ((int64_t)1 << 31) && m >= 1 && m < ((int64_t)1 << 31), "n or m out of range");
    NF_ARG(deg >= 0 && deg <= QW_DEGMAX, "deg must be in 0..%d", QW_DEGMAX);
    const int P = (deg + 1) * (deg + 2) / 2;
    NF_ARG(k >= P, "k = %d is below the %d polynomial terms of degree %d (unisolvency)", k, P, deg);
    NF_ARG(k <= QW_KMAX && k <= n, "k = %d must be <= min(n, %d)", k, QW_KMAX);
    cudaStream_t s = as_stream(stream);
    const int N = k + P;
    const size_t smem = sizeof(double) * ((size_t)N * (N | 1) + 3 * N + 1 + 3 * (size_t)k + QF_SIZE);
    // per call: the attribute belongs to the current device, and a call costs microseconds
    NF_CUDA_TRY(cudaFuncSetAttribute(quad_element_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int64_t *nbr = nullptr;
    unsigned long long *keys = nullptr;
    long long *v0 = nullptr, *v1 = nullptr;
    int *flag = nullptr;
    unsigned long long *first_bad = nullptr;
    double *elem_w = nullptr, *frame = nullptr;
    NF_CUDA_TRY(cudaMallocAsync(&first_bad, 64, s));
    flag = reinterpret_cast<int *>(reinterpret_cast<char *>(first_bad) + 16);
    NF_CUDA_TRY(cudaMemsetAsync(first_bad, 0xff, 8, s));
    NF_CUDA_TRY(cudaMemsetAsync(flag, 0, 4, s));
    {
        launch_validate_indices(tris, 3 * m, n, flag, s);
        launch_validate_indices(stencils, m * k, n, flag, s);
        int hflag = 0;
        NF_CUDA_TRY(cudaMemcpyAsync(&hflag, flag, sizeof(int), cudaMemcpyDeviceToHost, s));
        NF_CUDA_TRY(cudaStreamSynchronize(s));
        if (hflag) {
            cudaFreeAsync(first_bad, s);
            return fail(NF_ERR_ARG, "tris or stencils hold a node index outside [0, n)");
        }
    }
    NF_CUDA_TRY(cudaMallocAsync(&elem_w, sizeof(double) * m * k, s));
    NF_CUDA_TRY(cudaMallocAsync(&frame, sizeof(double) * m * QF_SIZE, s));
    if (dim == 3) {
        int64_t cap = 1;
        while (cap < 4 * 3 * m) cap <<= 1;
        NF_CUDA_TRY(cudaMallocAsync(&nbr, sizeof(int64_t) * 3 * m, s));
        NF_CUDA_TRY(cudaMallocAsync(&keys, sizeof(unsigned long long) * cap, s));
        NF_CUDA_TRY(cudaMallocAsync(&v0, sizeof(long long) * cap, s));
        NF_CUDA_TRY(cudaMallocAsync(&v1, sizeof(long long) * cap, s));
        NF_CUDA_TRY(cudaMemsetAsync(keys, 0xff, sizeof(unsigned long long) * cap, s));
        NF_CUDA_TRY(cudaMemsetAsync(v0, 0xff, sizeof(long long) * cap, s));
        NF_CUDA_TRY(cudaMemsetAsync(v1, 0xff, sizeof(long long) * cap, s));
        edge_insert_kernel<<<(unsigned)ceil_div(3 * m, 256), 256, 0, s>>>(tris, m, keys, v0, v1, cap, flag);
        edge_lookup_kernel<<<(unsigned)ceil_div(3 * m, 256), 256, 0, s>>>(tris, m, keys, v0, v1, cap, flag, nbr);
        NF_CUDA_TRY(cudaGetLastError());
    }
    QwArgs qa{nodes, normals, dim, tris, m, stencils, k, deg, nbr, frame, elem_w, first_bad};
    quad_frame_kernel<<<(unsigned)ceil_div(m, 128), 128, 0, s>>>(qa);
    NF_CUDA_TRY(cudaGetLastError());
    quad_element_kernel<<<(unsigned)m, QW_THREADS, smem, s>>>(qa);
    NF_CUDA_TRY(cudaGetLastError());
    int32_t *cnt = nullptr, *start = nullptr;
    int64_t *refs = nullptr;
    NF_CUDA_TRY(cudaMallocAsync(&cnt, sizeof(int32_t) * n, s));
    NF_CUDA_TRY(cudaMallocAsync(&start, sizeof(int32_t) * (n + 1), s));
    NF_CUDA_TRY(cudaMallocAsync(&refs, sizeof(int64_t) * m * k, s));
    NF_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * n, s));
    count_refs_kernel<<<(unsigned)ceil_div(m * k, 256), 256, 0, s>>>(stencils, m * k, cnt);
    launch_exclusive_scan(cnt, n, start, s);
    NF_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * n, s));
    fill_refs_kernel<<<(unsigned)ceil_div(m * k, 256), 256, 0, s>>>(stencils, m * k, start, cnt, refs);
    gather_weights_kernel<<<(unsigned)ceil_div(n, GW_WARPS), 32 * GW_WARPS, 0, s>>>(n, start, refs, elem_w, q);
    NF_CUDA_TRY(cudaGetLastError());
    unsigned long long hbad = ~0ull;
    NF_CUDA_TRY(cudaMemcpyAsync(&hbad, first_bad, 8, cudaMemcpyDeviceToHost, s));
    NF_CUDA_TRY(cudaStreamSynchronize(s));
    cudaFreeAsync(cnt, s);
    cudaFreeAsync(start, s);
    cudaFreeAsync(refs, s);
    cudaFreeAsync(elem_w, s);
    cudaFreeAsync(frame, s);
    cudaFreeAsync(first_bad, s);
    if (nbr) cudaFreeAsync(nbr, s);
    if (keys) cudaFreeAsync(keys, s);
    if (v0) cudaFreeAsync(v0, s);
    if (v1) cudaFreeAsync(v1, s);
    NF_CUDA_TRY(cudaStreamSynchronize(s));
    if (hbad != ~0ull) {
        if (bad_element) *bad_element = (int64_t)hbad;
        return fail(NF_ERR_SINGULAR, "singular interpolation system at element %lld", (long long)hbad);
    }
    return NF_OK;
}

extern "C" nf_status nf_quad_weights_opts(const double *nodes, const double *normals, int64_t n, const int32_t *tris,
                                          int64_t m, const int32_t *stencils, int k, const nf_quad_opts *o, double *q,
                                          int64_t *bad_element, void *stream) {
    clear_error();
    NF_ARG(o, "options must be non-NULL");
    NF_ARG(o->dim == 2 || o->dim == 3, "dim must be 2 or 3 (got %d)", o->dim);
    NF_ARG(o->curved == (o->dim == 3 ? 1 : 0), "curved must be 1 for dim 3 (surfaces) and 0 for dim 2");
    if (o->phs_order != 3)
        return fail(NF_ERR_UNSUPPORTED, "phs_order %d: the polyharmonic spline r^3 is implemented", o->phs_order);
    return nf_quad_weights(nodes, o->curved ? normals : nullptr, n, o->dim, tris, m, stencils, k, o->poly_deg, q,
                           bad_element, stream);
}
