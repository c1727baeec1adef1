// nf_mf.cu -- matrix-free nonlocal sum (§2.2, Eq. (2.9)) and the fused RK4 stage
// kernel.
//
// Pair kernel.  I[b, i] = sum_j w(|x_i - x_j|) g[b, j], g = q o f(U) (FP32), with the
// Mexican-hat kernel w(r) = A1 exp(-r^2/s1^2) - A2 exp(-r^2/s2^2).  Work is split
// into items (row block, column split): each warp owns R rows (coordinates in
// registers); its lanes stride over the columns of the split; column tiles are staged
// into shared memory by the TMA bulk-copy unit, double buffered on mbarriers.  The scalar
// kernel below serves the allocation-free call (NB = 1), whose nodes are in the caller's order,
// and groups of exactly 16 trajectories (NB = 16), where the packed kernel of nf_multi.cu spills
// its 64 accumulators (n = 20,000: 544 against 584 us per sum).  Per pair 3 FADD + FMUL + 2 FFMA
// (r^2), 2 FMUL (exponent scaling), 2 MUFU.EX2, and 2 FFMA (NB = 1: separate e1 and e2
// accumulators) or FMUL + FFMA + NB FFMA.
// Each warp reduces its rows with shuffles and writes one partial sum per
// (split, trajectory, row); the stage kernel (or the reduce kernel) adds the
// splits in a fixed order, so results are deterministic.
#include "nf_pairs.cuh"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

namespace nfi {

constexpr int MF_THREADS = 256;
constexpr int MF_WARPS = MF_THREADS / 32;
constexpr int MF_TJ = 512;  // columns per shared-memory tile; divides kNodePad
static_assert(kNodePad % MF_TJ == 0, "tile must divide the node padding");

template <int NB>
struct MfSmem {
    float4 xs[2][MF_TJ];
    float gs[2][NB][MF_TJ];
    uint64_t bar[2];
};

template <int NB, int R>
__global__ void __launch_bounds__(MF_THREADS)
mf_pair_kernel(const float4 *__restrict__ x4, const float *__restrict__ g, int64_t n_pad, int B, int b_base,
               int64_t jchunk, float c1, float c2, float A1, float A2, float per, float *__restrict__ partial,
               int *__restrict__ err) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const float iper = per > 0.f ? 1.f / per : 0.f;
    MfSmem<NB> &sm = *reinterpret_cast<MfSmem<NB> *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int split = blockIdx.y;
    const int b0 = b_base + blockIdx.z * NB;
    const int64_t j0 = (int64_t)split * jchunk;
    const int64_t j1 = min(n_pad, j0 + jchunk);
    const int ntiles = (int)((j1 - j0) / MF_TJ);
    const int64_t row0 = ((int64_t)blockIdx.x * MF_WARPS + warp) * R;
    constexpr uint32_t kTileBytes = MF_TJ * 16 + NB * MF_TJ * 4;

    if (tid == 0) {
        mbar_init(&sm.bar[0], 1);
        mbar_init(&sm.bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();

    auto issue = [&](int t) {
        const int buf = t & 1;
        const int64_t jt = j0 + (int64_t)t * MF_TJ;
        mbar_arrive_expect_tx(&sm.bar[buf], kTileBytes);
        bulk_g2s(sm.xs[buf], x4 + jt, MF_TJ * 16, &sm.bar[buf]);
#pragma unroll
        for (int b = 0; b < NB; ++b) bulk_g2s(sm.gs[buf][b], g + (int64_t)(b0 + b) * n_pad + jt, MF_TJ * 4, &sm.bar[buf]);
    };
    if (tid == 0) {
        if (ntiles > 0) issue(0);
        if (ntiles > 1) issue(1);
    }

    float xi[R], yi[R], zi[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float4 p = x4[row0 + r];
        xi[r] = p.x;
        yi[r] = p.y;
        zi[r] = p.z;
    }
    constexpr int NA = (NB == 1) ? 2 : NB;  // NB == 1: separate e1 / e2 accumulators
    float acc[R][NA];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int a = 0; a < NA; ++a) acc[r][a] = 0.f;

    bool timed_out = false;
    for (int t = 0; t < ntiles; ++t) {
        const int buf = t & 1;
        const bool ok = mbar_wait_bounded(&sm.bar[buf], (uint32_t)((t >> 1) & 1));
        // Uniform decision; this barrier also certifies that every warp has finished
        // tile t-1, whose buffer the next issue overwrites.
        if (__syncthreads_or(!ok)) {
            timed_out = true;
            break;
        }
        if (tid == 0 && t >= 1 && t + 1 < ntiles) issue(t + 1);
        const float4 *xs = sm.xs[buf];
        auto sweep = [&](auto tag) {
            constexpr bool P = decltype(tag)::value;
#pragma unroll 4
        for (int jj = lane; jj < MF_TJ; jj += 32) {
            const float4 xj = xs[jj];
            float gb[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) gb[b] = sm.gs[buf][b][jj];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float dx = xi[r] - xj.x, dy = yi[r] - xj.y;
                const float dz = zi[r] - xj.z;
                if constexpr (P) {
                    dx = wrap1(dx, per, iper);
                    dy = wrap1(dy, per, iper);
                }
                const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                const float e1 = ex2_sfu(r2 * c1);
                const float e2 = ex2_sfu(r2 * c2);
                if constexpr (NB == 1) {
                    acc[r][0] = fmaf(e1, gb[0], acc[r][0]);
                    acc[r][1] = fmaf(e2, gb[0], acc[r][1]);
                } else {
                    const float w = fmaf(A1, e1, -A2 * e2);
#pragma unroll
                    for (int b = 0; b < NB; ++b) acc[r][b] = fmaf(w, gb[b], acc[r][b]);
                }
            }
        }
        };
        if (per > 0.f)
            sweep(PerTag<true>{});
        else
            sweep(PerTag<false>{});
    }
    if (timed_out) {
        if (tid == 0) set_dev_error(err, DEV_TIMEOUT);
        // let any copy still in flight land before the block's shared memory is released
        if (tid == 0)
            for (int b = 0; b < 2; ++b) (void)mbar_wait_bounded(&sm.bar[b], 0), (void)mbar_wait_bounded(&sm.bar[b], 1);
        return;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            float v = (NB == 1) ? (A1 * acc[r][0] - A2 * acc[r][1]) : acc[r][b];
            v = warp_sum(v);
            if (lane == 0) partial[((int64_t)split * B + (b0 + b)) * n_pad + row0 + r] = v;
        }
    }
}

// ----------------------------------------------------------------------------
// RK4 stage of one node, shared by the stage kernel and the fused small-set kernel.
__device__ __forceinline__ float firing_rate(float u, float beta, float theta) {
    return 1.0f / (1.0f + expf(-beta * (u - theta)));
}

// Constants of the flat manufactured forcing (host side of forcing_value): per Gaussian of the
// kernel with amplitude A and width w, p = 1 / w^2.
struct FlatTerm {
    double amp;        // +-A / (2 pi sigma^2)
    double rs, prs;    // r / (p + r), -p r / (p + r)
    double k;          // sqrt(p + r)
    double half_root;  // sqrt(pi / (p + r)) / 2
};
struct FlatConst {
    double L, iL, r, norm;  // period, 1 / (2 sigma^2), 1 / (2 pi sigma^2)
    double c0;              // the convolution's constant part
    FlatTerm t[2];
    int terms;
};

// Fused RK4 stage: I = sum of splits; k_s = -U_s + I + gamma(t_s); RK4 bookkeeping;
// next stage input and its g.  On the last stage the last block advances the
// device step counter, so one captured step can be replayed.
struct StageKArgs {
    const float *partial;
    int splits;
    int64_t n, n_pad;
    int B;
    float *u;           // caller's state, written by stage 4 (null: kept inside only)
    float *us;          // the state in the operator's order: u itself without perm
    float *U, *ks, *g;
    const float *q;     // matrix-free: g = q f; dense: g = f (q lives in W)
    const float *rs;    // BF16X2 row scale, or null
    const float *beta, *theta;
    nf_forcing F;
    FlatConst fc;       // flat manufactured forcing
    const float4 *x4;   // node coordinates (manufactured forcings)
    const double *t0;
    double dt;
    int stage;
    long long *step_ctr;
    unsigned *done_ctr;
    float *ckpt;
    int C;
    const int *perm;    // caller's node of each position (u, ckpt, Y1, Y2), or null
    float *stage_out;   // next stage's input, kept by the adjoint's recomputation, or null
    int *err;           // operator's device flag: DEV_NONFINITE on a non-finite new state
};

// Flat manufactured forcing (NF_FORCE_MMS_FLAT).  One factor of the convolution term:
//   J(a) = int_{-L/2}^{L/2} exp(-p d^2) exp(-e(d)^2 / (2 sigma^2)) dd,  e(d) = nearest image of a - d,
// a = nearest image of x - x0 in one coordinate.  e(d) = a - d except past the point where
// a - d leaves [-L/2, L/2] (d < a - L/2 for a >= 0, d > a + L/2 for a < 0), where it is
// a - d -+ L.  Each piece is a Gaussian product integrated in closed form:
//   int_{d0}^{d1} exp(-p d^2 - r (d - a')^2) dd
//     = exp(-p r a'^2 / (p + r)) (1/2) sqrt(pi / (p + r)) [erf(k (d1 - m)) - erf(k (d0 - m))],
// r = 1 / (2 sigma^2), m = r a' / (p + r), k = sqrt(p + r).
// The forcing is FP64 arithmetic on a chip whose FP64 pipe gives two lanes per clock per SM, so
// what does not depend on the node is taken out: constants come from the host, cos t and sin t
// from one thread per block, an erf is evaluated only where it is not +-1 to the last bit, and a
// piece whose two erf agree is 0 without its exponential (all pieces but one, away from the
// kink lines).
constexpr double kPi = 3.14159265358979323846;
__device__ __forceinline__ double erf_sat(double z) { return z >= 6.0 ? 1.0 : (z <= -6.0 ? -1.0 : erf(z)); }
__device__ __forceinline__ double gauss_piece(const FlatTerm &g, double a, double d0, double d1) {
    const double m = g.rs * a, diff = erf_sat(g.k * (d1 - m)) - erf_sat(g.k * (d0 - m));
    return diff == 0.0 ? 0.0 : exp(g.prs * a * a) * g.half_root * diff;
}
__device__ __forceinline__ double flat_factor(const FlatTerm &g, double a, double L) {
    const double h = 0.5 * L;
    if (a >= 0.0) return gauss_piece(g, a - L, -h, a - h) + gauss_piece(g, a, a - h, h);
    return gauss_piece(g, a, -h, a + h) + gauss_piece(g, a + L, a + h, h);
}

// i: position in the operator's order (x4); node: the caller's index (Y1, Y2); ct, sn = cos t, sin t
__device__ __forceinline__ double forcing_value(const nf_forcing &F, const FlatConst &fc, const float4 *x4, int64_t i,
                                                int64_t node, double ct, double sn, float beta, float theta) {
    if (F.kind == NF_FORCE_MMS_FLAT) {
        // z = G(x, x0(t); sigma) + c on the periodic square; gamma = du*/dt + u* - scale C,
        // C = int_cell w(dist(x, y)) z(y) dy: the constant part integrates w over the
        // displacement square, the Gaussian part is separable (flat_factor per coordinate)
        const double x0 = F.radius * ct, y0 = F.radius * sn;
        const float4 xi = x4[i];
        double ax = (double)xi.x - x0, ay = (double)xi.y - y0;
        ax -= fc.L * rint(ax * fc.iL);
        ay -= fc.L * rint(ay * fc.iL);
        const double G = exp(-(ax * ax + ay * ay) * fc.r) * fc.norm;
        const double z = G + F.c;
        const double dz = G * (ay * x0 - ax * y0) * (2.0 * fc.r);
        const double us = (double)theta + log(z / (1.0 - z)) / (double)beta;
        const double dus = dz / ((double)beta * z * (1.0 - z));
        double C = fc.c0;
        for (int h = 0; h < fc.terms; ++h)
            C += fc.t[h].amp * (flat_factor(fc.t[h], ax, fc.L) * flat_factor(fc.t[h], ay, fc.L));
        return dus + us - F.scale * C;
    }
    double Y1, Y2;
    if (F.kind == NF_FORCE_MMS_SPHERE) {  // Y1 = z / 2 (degree 1), Y2 = x y (degree 2) at the node
        const float4 xi = x4[i];
        Y1 = 0.5 * (double)xi.z;
        Y2 = (double)xi.x * (double)xi.y;
    } else {
        Y1 = F.Y1[node];
        Y2 = F.Y2[node];
    }
    const double Y = Y1 + Y2;
    const double a = F.a0 * ct, da = -F.a0 * sn;
    const double z = F.c + a * Y;
    const double us = (double)theta + log(z / (1.0 - z)) / (double)beta;
    const double dus = da * Y / ((double)beta * z * (1.0 - z));
    return dus + us - (F.lam0 * F.c + a * (F.lam1 * Y1 + F.lam2 * Y2));
}

// The tableau update of one node from its sum I: k_s = -U_s + I + gamma, the RK4 bookkeeping, the
// next stage's input and its g (g_out: where the next sum reads it).
struct StageNode {
    float Uv, uv, ksv, bb, th, qv;  // U_s, u, slope accumulator, beta, theta, q
    int64_t node;                   // the caller's index
};
__device__ __forceinline__ StageNode stage_load(const StageKArgs &a, int b, int64_t i, int64_t idx) {
    return StageNode{ld_l2(a.U + idx), ld_l2(a.us + idx), a.stage > 1 ? ld_l2(a.ks + idx) : 0.f, a.beta[b], a.theta[b],
                     a.q ? a.q[i] : 1.f, a.perm ? (int64_t)a.perm[i] : i};
}
__device__ __forceinline__ void stage_update(const StageKArgs &a, const StageNode &s, long long step, int b, int64_t i,
                                             int64_t idx, float I, float gam, float *g_out) {
    const float k = (-s.Uv + I) + gam;
    const float dt = (float)a.dt;
    float Un;
    if (a.stage == 1) {
        a.ks[idx] = k;
        Un = fmaf(0.5f * dt, k, s.uv);
    } else if (a.stage == 2) {
        a.ks[idx] = fmaf(2.f, k, s.ksv);
        Un = fmaf(0.5f * dt, k, s.uv);
    } else if (a.stage == 3) {
        a.ks[idx] = fmaf(2.f, k, s.ksv);
        Un = fmaf(dt, k, s.uv);
    } else {
        const float unew = fmaf(dt / 6.f, s.ksv + k, s.uv);
        a.us[idx] = unew;
        const int64_t cidx = (int64_t)b * a.n + s.node;
        if (a.perm && a.u) a.u[cidx] = unew;
        Un = unew;
        if (!isfinite(unew) && *a.err == DEV_OK) atomicCAS(a.err, DEV_OK, DEV_NONFINITE);
        if (a.ckpt && ((step + 1) % a.C) == 0) a.ckpt[(int64_t)((step + 1) / a.C) * a.B * a.n + cidx] = unew;
    }
    a.U[idx] = Un;
    if (a.stage_out) a.stage_out[idx] = Un;
    const float f = firing_rate(Un, s.bb, s.th);
    g_out[(int64_t)b * a.n_pad + i] = a.q ? s.qv * f : f;
}

// End of a step (stage 4): the last of `blocks` blocks advances the device step counter.
__device__ __forceinline__ void step_done(const StageKArgs &a, unsigned blocks) {
    if (a.stage != 4) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(a.done_ctr, 1u);
        if (prev == blocks - 1) {
            *a.done_ctr = 0u;
            atomicAdd(reinterpret_cast<unsigned long long *>(a.step_ctr), 1ull);
            __threadfence();
        }
    }
}

// ----------------------------------------------------------------------------
// Single-trajectory variant on packed FP32 pairs (f32x2: one instruction, two lanes of
// the FMA pipe).  Column tiles are staged as structure-of-arrays (x, y, z, g), so a
// lane reads two adjacent columns with one 8-byte load; each row's coordinates are held
// duplicated in a 64-bit register pair.  Difference form, per two pairs: 3 SUB2, MUL2 +
// 2 FMA2 (r^2), MUL2 (exponent), MUL2 (second exponent), 4 MUFU.EX2, 2 FMA2 -- the rounding of the
// scalar kernel.  Expanded form (below): 3 FMA2, MUL2, 4 MUFU.EX2, 2 FMA2, plus 6 per column pair
// shared by the warp's rows, which leaves the SFU (2 exponentials per pair) as the bound.
template <int TJ>
struct MfPackedSmem {
    float xs[2][TJ], ys[2][TJ], zs[2][TJ], gs[2][TJ];
    uint64_t bar[2];
};

// The nodes are in Hilbert order, so the R rows of a warp usually lie close together.  Such a warp expands the squared distance
// about the centre c of its rows' bounding box:
//   r^2 = |x_i - c|^2 + |x_j - c|^2 - 2 (x_i - c).(x_j - c) = n_i + s_ij,
//   s_ij = n_j - 2 (x_i - c).(x_j - c),
// and accumulates 2^(-s_ij) and 2^(-k2 s_ij); the row factors 2^(-n_i), 2^(-k2 n_i) are
// applied once at the end.  Per column pair the centred coordinates and n_j cost 6 lane
// operations shared by the warp's R rows; per pair the exponent argument is then a chain
// of 3 FMAs instead of 3 SUB + 2 MUL + 2 FMA.  FP32 rounding of s_ij is relative to
// n_i + n_j + 2 |x_i - c||x_j - c|, so the form is used only when every row of the warp has
// n_i <= kMfLocalSpread as an exponent of the narrower Gaussian evaluated (|x_i - c| <= s / 2.4, s its
// width).  Warps whose rows are spread out use the difference form.  The choice is warp-uniform
// and fixed per launch shape, so results stay deterministic.  The threshold trades rounding for
// time at 2,000 to 3,000 nodes: over 56 kernels and node sets of 500 to 3,001 nodes the relative L2 error
// against FP64 has a geometric mean of 0.78e-7 with 0.25 as with 0.5, and at worst 2.6e-7 against 3.5e-7
// (a lattice on which the two Gaussians nearly cancel); 0.0625 takes 5 to 8 % longer.  Coordinates
// rounded to exponent units and exp2f's row factors gave 1.32e-7, at worst 7.4e-7.
//
// Integer width ratio.  When m = s2^2 / s1^2 is a small integer (M = 2, 3, 4; the paper's
// lateral-inhibition kernels have sigma_i = 2 sigma_e, i.e. m = 4), the expanded form takes
// e2 = 2^(-s_ij), in units of s2, from the SFU and e1 = e2^M by squaring on the FMA pipe: one
// exponential per pair instead of two.  The relative error of e1 grows to about M times that of
// ex2.approx (a few 1e-7).  M = 0 is the general form.
constexpr float kMfLocalSpread = 0.25f;

// xyz: the exact set's coordinates (times a power of two; the exponent of a pair is uu r^2) as
// structure of arrays [x(n_pad) | y(n_pad) | z(n_pad)];
// g_all: B x n_pad firing rates (times q); both in Hilbert order, like the partial sums.
//
// MODE 0 writes partial sums.  Small node sets (MODE 1, 2: one column split, so a warp holds the
// whole sums of its rows) finish in the same launch: MODE 1 performs the RK4 stage of its rows,
// MODE 2 writes them to the caller's I.  At 1,500 nodes a sum is 1 us of arithmetic; what
// counts is launches and their dependent loads, so the static tiles are staged before
// pdl_wait(), the rows' state is read while the tiles are swept, and g alternates between two
// buffers (other blocks still read this stage's while the first rows of the next are written).
struct FusedOut {
    StageKArgs st;  // MODE 1
    float *g_next;  // MODE 1: the other g buffer
    float *I;       // MODE 2, caller's order
    const int *perm;
    int64_t n;
};
template <int R, int TJ, int M, int MODE>
__global__ void __launch_bounds__(MF_THREADS, R >= 8 ? 2 : 4)
mf_pair_packed_kernel(const float *__restrict__ xyz, const float *g_all, int64_t n_pad, int B, int b_base,
                      int64_t jchunk, float uu, float k2, float A1, float A2, float per, float *__restrict__ partial,
                      int *__restrict__ err, const __grid_constant__ FusedOut fo) {
    static_assert(M >= 0 && M <= 4, "form M: 0 general, 1 one Gaussian, 2-4 width ratio");
    __shared__ __align__(128) MfPackedSmem<TJ> sm;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int split = blockIdx.y;
    const int64_t j0 = (int64_t)split * jchunk;
    const int64_t j1 = min(n_pad, j0 + jchunk);
    const int ntiles = (int)((j1 - j0) / TJ);
    const int64_t slot0 = ((int64_t)blockIdx.x * MF_WARPS + warp) * R;
    constexpr uint32_t kTileBytes = 4 * TJ * 4;
    const float *X = xyz, *Y = xyz + n_pad, *Z = xyz + 2 * n_pad;
    const int b = b_base + blockIdx.z;
    const float *g = g_all + (int64_t)b * n_pad;
    if (tid == 0) {
        mbar_init(&sm.bar[0], 1);
        mbar_init(&sm.bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    auto issue_xyz = [&](int t) {
        const int buf = t & 1;
        const int64_t jt = j0 + (int64_t)t * TJ;
        mbar_arrive_expect_tx(&sm.bar[buf], kTileBytes);
        bulk_g2s(sm.xs[buf], X + jt, TJ * 4, &sm.bar[buf]);
        bulk_g2s(sm.ys[buf], Y + jt, TJ * 4, &sm.bar[buf]);
        bulk_g2s(sm.zs[buf], Z + jt, TJ * 4, &sm.bar[buf]);
    };
    auto issue_g = [&](int t) { bulk_g2s(sm.gs[t & 1], g + j0 + (int64_t)t * TJ, TJ * 4, &sm.bar[t & 1]); };
    if (tid == 0) {
        if (ntiles > 0) issue_xyz(0);
        if (ntiles > 1) issue_xyz(1);
    }
    // the warp's rows (all lanes hold the same values) and the centre of their bounding box
    float xr[R], yr[R], zr[R];
    float lox = 3.4e38f, loy = 3.4e38f, loz = 3.4e38f, hix = -3.4e38f, hiy = -3.4e38f, hiz = -3.4e38f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        xr[r] = X[slot0 + r];
        yr[r] = Y[slot0 + r];
        zr[r] = Z[slot0 + r];
        lox = fminf(lox, xr[r]), hix = fmaxf(hix, xr[r]);
        loy = fminf(loy, yr[r]), hiy = fmaxf(hiy, yr[r]);
        loz = fminf(loz, zr[r]), hiz = fmaxf(hiz, zr[r]);
    }
    const float cx = 0.5f * (lox + hix), cy = 0.5f * (loy + hiy), cz = 0.5f * (loz + hiz);
    // Expanded form: coordinates centred and scaled in one FMA, w x - w c with w = sqrt(uu): the same one
    // rounding of the difference as in x - c, and no multiplication by uu left in the loop.
    const float w = sqrtf(uu), ncx = -(w * cx), ncy = -(w * cy), ncz = -(w * cz);
    float spread = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float dx = fmaf(w, xr[r], ncx), dy = fmaf(w, yr[r], ncy), dz = fmaf(w, zr[r], ncz);
        spread = fmaxf(spread, dx * dx + dy * dy + dz * dz);
    }
    // warp-uniform, the threshold as an exponent, for the narrower Gaussian evaluated; periodic
    // distances take the difference form (nearest images per pair)
    const float most = M >= 2 ? kMfLocalSpread * k2 : (M == 0 ? kMfLocalSpread / fmaxf(1.f, k2) : kMfLocalSpread);
    const bool local = spread <= most && !(per > 0.f);
    // local: xi, yi, zi hold -2 w (x_i - c); otherwise x_i itself (both halves of the pair).
    // M >= 2: one pair weight e2 + c_i e1, c_i = -(A1 f1) / (A2 f2) with the row factors, and one sum: the
    // difference of the two Gaussians' sums magnifies the rounding of either (see nf_sym.cu)
    constexpr bool CW = M >= 2;
    u64 xi[R], yi[R], zi[R], h1[CW ? R : 1], a1[R], a2[CW ? 1 : R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float x = local ? -2.f * fmaf(w, xr[r], ncx) : xr[r];
        const float y = local ? -2.f * fmaf(w, yr[r], ncy) : yr[r];
        const float z = local ? -2.f * fmaf(w, zr[r], ncz) : zr[r];
        xi[r] = f2_pack(x, x);
        yi[r] = f2_pack(y, y);
        zi[r] = f2_pack(z, z);
        a1[r] = 0ull;
        if constexpr (CW) {
            const float ni = local ? 0.25f * (x * x + y * y + z * z) : 0.f;
            h1[r] = f2_dup(scale_pow2(-(A1 / A2), -(float)(M - 1) * ni, local ? kEx2Low : 0.f));
        } else {
            a2[r] = 0ull;
        }
    }
    // with a = uu r^2 the exponent of a pair: M < 2: e1 = 2^(-a), e2 = 2^(-k2 a) with
    // k2 = s1^2 / s2^2; M >= 2: e2 = 2^(-a), e1 = 2^(-M a)
    const u64 uup = f2_dup(uu);
    const u64 nk2 = M >= 2 ? f2_dup(-(float)M) : f2_dup(-k2);
    const u64 wp = f2_dup(w), cxp = f2_dup(ncx), cyp = f2_dup(ncy), czp = f2_dup(ncz);
    const float iper = per > 0.f ? 1.f / per : 0.f;
    const u64 ipp = f2_pack(iper, iper), npp = f2_pack(-per, -per), mgp = f2_pack(kRintMagic, kRintMagic);
    // MODE 1: lane r < R carries row r's state
    long long step = 0;
    StageNode sn{};
    const int64_t own = slot0 + lane;
    const bool mine = MODE != 0 && lane < R && own < fo.n;
    pdl_wait();  // the kernel before wrote g and the rows' state
    pdl_trigger();
    if constexpr (MODE == 1) {
        step = *fo.st.step_ctr;
        if (mine) sn = stage_load(fo.st, b, own, (int64_t)b * fo.n + own);
    }
    if (tid == 0) {
        if (ntiles > 0) issue_g(0);
        if (ntiles > 1) issue_g(1);
    }
    bool timed_out = false;
    for (int t = 0; t < ntiles; ++t) {
        const int buf = t & 1;
        const bool ok = mbar_wait_bounded(&sm.bar[buf], (uint32_t)((t >> 1) & 1));
        if (__syncthreads_or(!ok)) {
            timed_out = true;
            break;
        }
        if (tid == 0 && t >= 1 && t + 1 < ntiles) {
            issue_xyz(t + 1);
            issue_g(t + 1);
        }
        const u64 *xs = reinterpret_cast<const u64 *>(sm.xs[buf]);
        const u64 *ys = reinterpret_cast<const u64 *>(sm.ys[buf]);
        const u64 *zs = reinterpret_cast<const u64 *>(sm.zs[buf]);
        const u64 *gs = reinterpret_cast<const u64 *>(sm.gs[buf]);
        if (local) {
#pragma unroll 2
            for (int jp = lane; jp < TJ / 2; jp += 32) {
                const u64 xt = f2_fma(xs[jp], wp, cxp), yt = f2_fma(ys[jp], wp, cyp), zt = f2_fma(zs[jp], wp, czp);
                const u64 nj = f2_fma(zt, zt, f2_fma(yt, yt, f2_mul(xt, xt)));
                const u64 gj = gs[jp];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const u64 sij = f2_fma(xi[r], xt, f2_fma(yi[r], yt, f2_fma(zi[r], zt, nj)));
                    float s0, s1v;
                    f2_unpack(sij, s0, s1v);
                    const u64 e = f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v));
                    if constexpr (CW) {
                        const u64 sq = f2_mul(e, e);
                        a1[r] = f2_fma(f2_fma(M == 2 ? sq : (M == 3 ? f2_mul(sq, e) : f2_mul(sq, sq)), h1[r], e), gj, a1[r]);
                    } else {
                        a1[r] = f2_fma(e, gj, a1[r]);
                        if constexpr (M == 0) a2[r] = f2_fma(f2_ex2(f2_mul(sij, nk2)), gj, a2[r]);
                    }
                }
            }
        } else {
            auto sweep = [&](auto tag) {
                constexpr bool P = decltype(tag)::value;
#pragma unroll 2
            for (int jp = lane; jp < TJ / 2; jp += 32) {
                const u64 xj = xs[jp], yj = ys[jp], zj = zs[jp], gj = gs[jp];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    u64 dx = f2_sub(xi[r], xj), dy = f2_sub(yi[r], yj);
                    const u64 dz = f2_sub(zi[r], zj);
                    if constexpr (P) {
                        dx = f2_wrap(dx, ipp, npp, mgp);
                        dy = f2_wrap(dy, ipp, npp, mgp);
                    }
                    const u64 r2s = f2_mul(f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx))), uup);
                    float s0, s1v;
                    f2_unpack(r2s, s0, s1v);
                    // 2^(-r2s): the narrow Gaussian, or for M >= 2 the wide one
                    const u64 e = f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v));
                    if constexpr (CW) {
                        a1[r] = f2_fma(f2_fma(f2_ex2(f2_mul(r2s, nk2)), h1[r], e), gj, a1[r]);
                    } else {
                        a1[r] = f2_fma(e, gj, a1[r]);
                        if constexpr (M == 0) a2[r] = f2_fma(f2_ex2(f2_mul(r2s, nk2)), gj, a2[r]);
                    }
                }
            }
            };
            if (per > 0.f)
                sweep(PerTag<true>{});
            else
                sweep(PerTag<false>{});
        }
    }
    if (timed_out) {
        if (tid == 0) {
            set_dev_error(err, DEV_TIMEOUT);
            for (int b = 0; b < 2; ++b) (void)mbar_wait_bounded(&sm.bar[b], 0), (void)mbar_wait_bounded(&sm.bar[b], 1);
        }
        if constexpr (MODE == 1) step_done(fo.st, gridDim.x * gridDim.z);  // uncounted, it would shift later steps' count
        return;
    }
    float total = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        // first sum, with the factor of its Gaussian (M >= 2: of the wide one), then the second
        float s1f = (CW ? -A2 : A1) * f2_fold(a1[r]), s2f = 0.f;
        if constexpr (M == 0) s2f = A2 * f2_fold(a2[r]);
        if (local) {  // n_i from the same rounded centred coordinates the loop used
            float mx, my, mz, unused;
            f2_unpack(xi[r], mx, unused);
            f2_unpack(yi[r], my, unused);
            f2_unpack(zi[r], mz, unused);
            const float ni = 0.25f * (mx * mx + my * my + mz * mz);  // in units of s2 when M >= 2
            s1f = scale_pow2(s1f, -ni, kEx2Low);
            if constexpr (M == 0) s2f = scale_pow2(s2f, -k2 * ni, kEx2Low);
        }
        const float v = warp_sum(s1f - s2f);
        if constexpr (MODE == 0) {
            if (lane == 0) partial[((int64_t)split * B + b) * n_pad + slot0 + r] = v;
        } else {
            if (lane == r) total = v;
        }
    }
    if constexpr (MODE == 1) {
        if (mine) stage_update(fo.st, sn, step, b, own, (int64_t)b * fo.n + own, total, 0.f, fo.g_next);
        step_done(fo.st, gridDim.x * gridDim.z);
    } else if constexpr (MODE == 2) {
        if (mine) fo.I[(int64_t)b * fo.n + fo.perm[own]] = total;
    }
}

// ----------------------------------------------------------------------------
// split planner: (row blocks x column splits) items of equal cost; pick the number
// of splits (at most max_splits) that best fills whole waves of resident blocks.
SplitPlan plan_splits(int64_t n_pad, int rows_per_block, int tile_cols, int resident_blocks_per_sm, int max_splits) {
    SplitPlan p{};
    p.rows_per_block = rows_per_block;
    p.row_blocks = n_pad / rows_per_block;
    const int64_t tiles = n_pad / tile_cols;
    const int64_t slots = (int64_t)num_sms() * std::max(1, resident_blocks_per_sm);
    double best = -1.0;
    int best_s = 1;
    const int64_t smax = std::min<int64_t>(tiles, std::max(1, max_splits));
    for (int64_t s = 1; s <= smax; ++s) {
        const int64_t per = ceil_div(tiles, s);
        const int64_t s_eff = ceil_div(tiles, per);
        if (s_eff != s) continue;
        const int64_t items = p.row_blocks * s_eff;
        const int64_t waves = ceil_div(items, slots);
        double eff = (double)items / (double)(waves * slots);
        // each extra split costs a little (prologue, partial traffic): prefer fewer
        eff -= 0.002 * (double)s;
        if (eff > best + 1e-9) {
            best = eff;
            best_s = (int)s;
        }
        if (items >= 16 * slots) break;  // enough waves that the tail is negligible
    }
    p.splits = best_s;
    p.jchunk = ceil_div(tiles, best_s) * tile_cols;
    return p;
}

template <int NB, int R>
static cudaError_t set_mf_attr() {
    return cudaFuncSetAttribute(mf_pair_kernel<NB, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(MfSmem<NB>));
}

// The attributes belong to the device's context: set once per device (under a lock, so that
// concurrent first calls on one device do not race), with that device current.
static nf_status mf_init_attrs_device();

nf_status mf_init_attrs() {
    static std::mutex mu;
    static bool done[64] = {false};
    const int d = device_id();
    if (d < 0 || d >= 64) return mf_init_attrs_device();
    std::lock_guard<std::mutex> lock(mu);
    if (done[d]) return NF_OK;
    NF_TRY(mf_init_attrs_device());
    done[d] = true;
    return NF_OK;
}

static nf_status mf_init_attrs_device() {
    NF_TRY(dense_init_attrs());
    NF_TRY(sym_init_attrs());
    NF_TRY(adj_init_attrs());
    NF_TRY(multi_init_attrs());
    NF_CUDA_TRY((set_mf_attr<1, 2>()));
    NF_CUDA_TRY((set_mf_attr<1, 4>()));
    NF_CUDA_TRY((set_mf_attr<8, 4>()));
    NF_CUDA_TRY((set_mf_attr<16, 2>()));
    NF_CUDA_TRY((set_mf_attr<16, 4>()));
    return NF_OK;
}

template <int NB, int R>
static nf_status launch_mf_group(nf_operator *op, int B, int b_base, int groups, const SplitPlan &pl,
                                 cudaStream_t s) {
    const size_t smem = sizeof(MfSmem<NB>);
    const float L2E = 1.4426950408889634f;
    const nf_kernel &k = op->kp;
    const float c1 = -L2E / (k.s1 * k.s1), c2 = -L2E / (k.s2 * k.s2);
    dim3 grid((unsigned)pl.row_blocks, (unsigned)pl.splits, (unsigned)groups);
    mf_pair_kernel<NB, R><<<grid, MF_THREADS, smem, s>>>(op->x4, op->g, op->n_pad, B, b_base, pl.jchunk, c1, c2,
                                                         k.A1, k.A2, k.period, op->partial, op->err);
    NF_CUDA_TRY(cudaGetLastError());
    return NF_OK;
}

template <int NB, int R>
static int mf_resident() {
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, mf_pair_kernel<NB, R>, MF_THREADS, sizeof(MfSmem<NB>));
    return std::max(nb, 1);
}

// Launch shapes of the packed kernel the autotuner chooses from: rows per warp, tile width.
struct MfVariant {
    int R, TJ;
};
constexpr MfVariant kMfVariants[] = {{2, 512}, {4, 512}, {4, 1024}, {8, 1024}};

template <int R, int TJ>
static int packed_resident() {
    int nb0 = 0, nb4 = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb0, mf_pair_packed_kernel<R, TJ, 0, 0>, MF_THREADS, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb4, mf_pair_packed_kernel<R, TJ, 4, 0>, MF_THREADS, 0);
    return std::max(std::min(nb0, nb4), 1);
}

static int variant_resident(int v) {
    switch (v) {
        case 0: return packed_resident<2, 512>();
        case 1: return packed_resident<4, 512>();
        case 2: return packed_resident<4, 1024>();
        default: return packed_resident<8, 1024>();
    }
}

template <int R, int TJ>
static void launch_packed(nf_operator *op, int B, int b_base, int groups, const SplitPlan &pl, cudaStream_t s) {
    const nf_kernel &k = op->kp;
    const ExactUnits &eu = op->eu;
    dim3 grid((unsigned)pl.row_blocks, (unsigned)pl.splits, (unsigned)groups);
#define NF_PACKED_ARGS \
    op->xyz2, op->g, op->n_pad, B, b_base, pl.jchunk, eu.uu, eu.k2, k.A1, k.A2, eu.per, op->partial, op->err, FusedOut{}
    switch (op->form) {
        case 1: mf_pair_packed_kernel<R, TJ, 1, 0><<<grid, MF_THREADS, 0, s>>>(NF_PACKED_ARGS); break;
        case 2: mf_pair_packed_kernel<R, TJ, 2, 0><<<grid, MF_THREADS, 0, s>>>(NF_PACKED_ARGS); break;
        case 3: mf_pair_packed_kernel<R, TJ, 3, 0><<<grid, MF_THREADS, 0, s>>>(NF_PACKED_ARGS); break;
        case 4: mf_pair_packed_kernel<R, TJ, 4, 0><<<grid, MF_THREADS, 0, s>>>(NF_PACKED_ARGS); break;
        default: mf_pair_packed_kernel<R, TJ, 0, 0><<<grid, MF_THREADS, 0, s>>>(NF_PACKED_ARGS); break;
    }
#undef NF_PACKED_ARGS
}

static nf_status launch_mf_packed(nf_operator *op, int B, int b_base, int groups, const SplitPlan &pl,
                                  cudaStream_t s) {
    switch (op->mf_variant) {
        case 0: launch_packed<2, 512>(op, B, b_base, groups, pl, s); break;
        case 1: launch_packed<4, 512>(op, B, b_base, groups, pl, s); break;
        case 2: launch_packed<4, 1024>(op, B, b_base, groups, pl, s); break;
        default: launch_packed<8, 1024>(op, B, b_base, groups, pl, s); break;
    }
    NF_CUDA_TRY(cudaGetLastError());
    return NF_OK;
}

// Up to kSymMaxB trajectories take the symmetric kernel, one launch with a grid z per
// trajectory: each trajectory's pairs are evaluated once, which beats the multi-trajectory
// kernels (ordered pairs, exponentials shared across trajectories) until about four
// trajectories (n = 100,000: 1.10 ms per symmetric trajectory, B = 4 in 4.0 ms there; n = 20,000:
// B = 3 symmetric in 0.193 ms, B = 4 there in 0.202).
constexpr int kSymMaxB = 3;

// Small node sets on the automatic schedule take one launch per sum: 2 rows per warp, columns in
// tiles of 1,024 (one or two at most sizes here; 512-node tiles, 1 or 4 rows per warp measured
// slower at most sizes).  Per RK4 stage on GB300, against the packed pair kernel and the stage
// kernel with and without overlapped launches: n = 1,000 4.2 us (4.8, 5.9), 2,000 5.7 to 6.1 (6.4,
// 8.4), 3,000 9.4 (9.4, 11.0); at 4,000 nodes 11.5, where the symmetric kernel on 256-node blocks
// takes 9.6 (15.1 before), hence the line.
constexpr int64_t kFusedMaxN = 3072;
constexpr int kFusedRows = 2, kFusedTile = 1024;
bool fused_fits(const nf_operator *op, int B) {
    return op->path == NF_MATRIX_FREE && op->mf_sched == NF_MF_AUTO && !op->mf_cull && op->n <= kFusedMaxN &&
           B <= kSymMaxB;
}

template <int MODE>
static cudaError_t launch_fused(nf_operator *op, int B, const float *g, const FusedOut &fo, bool overlap, cudaStream_t s) {
    constexpr int R = kFusedRows, TJ = kFusedTile;
    const nf_kernel &k = op->kp;
    const ExactUnits &eu = op->eu;
    // row blocks with a real node only; every column tile
    const dim3 grid((unsigned)ceil_div(op->n, MF_WARPS * R), 1, (unsigned)B);
    auto go = [&](auto kernel) {
        return launch_dependent(kernel, grid, MF_THREADS, 0, s, overlap, op->xyz2, g, op->n_pad, B, 0, op->n_pad,
                                eu.uu, eu.k2, k.A1, k.A2, eu.per, (float *)nullptr, op->err, fo);
    };
    switch (op->form) {
        case 1: return go(mf_pair_packed_kernel<R, TJ, 1, MODE>);
        case 2: return go(mf_pair_packed_kernel<R, TJ, 2, MODE>);
        case 3: return go(mf_pair_packed_kernel<R, TJ, 3, MODE>);
        case 4: return go(mf_pair_packed_kernel<R, TJ, 4, MODE>);
        default: return go(mf_pair_packed_kernel<R, TJ, 0, MODE>);
    }
}

// Launch shape of the packed kernel (single trajectories inside a multi-trajectory call):
// small node sets want more, smaller blocks.
static int default_variant(int64_t n_pad) { return n_pad >= 16384 ? 3 : 0; }

// Block pairs of 1,024 nodes, and slots of the symmetric kernel at the operator's block size.
static int64_t sym_pairs_1024(const nf_operator *op) {
    const int64_t nb = op->n_pad / 1024;
    return nb * (nb + 1) / 2;
}
int sym_slots(const nf_operator *op) { return (int)(op->n_pad / op->sym_blk); }

// Up to kSymMaxB trajectories take the symmetric kernel beyond kFusedMaxN nodes, on blocks of
//   256 nodes  while 1,024-node block pairs are fewer than 2/3 of the SMs (n below ~13,300): the
//              packed row-block x column-split kernel that served these sizes before evaluates
//              ordered pairs (per RK4 stage, packed before / 256 / 512: n = 5,500 23.9 / 12.9 /
//              20.8 us, 8,000 40.4 / 20.6 / 20.8, 13,000 82 / 41 / 43);
//   512, 1,024 above, by timing (mf_autotune).
// The automatic schedule also keeps the symmetric partial sums (one slot of n_pad floats per
// node block, growing as n^2) within an eighth of the device memory: beyond that (n
// above about 3 million on a GB300) the packed kernel, whose layout grows with its column
// splits only, takes over.
static bool sym_layout_fits(const nf_operator *op) {
    static std::atomic<size_t> budget[64];  // per device, an eighth of its memory
    const int d = device_id();
    size_t b = (d >= 0 && d < 64) ? budget[d].load() : 0;
    if (!b) {
        size_t freeb = 0, total = 0;
        b = (cudaMemGetInfo(&freeb, &total) == cudaSuccess && total > 0) ? total / 8 : ((size_t)8 << 30);
        if (d >= 0 && d < 64) budget[d].store(b);
    }
    return (double)(op->n_pad / 1024) * (double)op->n_pad * sizeof(float) <= (double)b;
}

static bool use_sym(const nf_operator *op) {
    if (op->mf_sched == NF_MF_SYMMETRIC) return true;
    if (op->mf_sched == NF_MF_PACKED) return false;
    return op->n > kFusedMaxN && sym_layout_fits(op);
}

int mf_splits(nf_operator *op, int B) {
    if (B <= kSymMaxB && use_sym(op)) return sym_slots(op);
    return B == 1 ? mf_plan(op).splits : multi_plan(op).splits;
}

static SplitPlan variant_plan(int64_t n_pad, int v) {
    return plan_splits(n_pad, MF_WARPS * kMfVariants[v].R, kMfVariants[v].TJ, variant_resident(v));
}

SplitPlan mf_plan(nf_operator *op) {
    if (op->mf_variant < 0) op->mf_variant = default_variant(op->n_pad);
    return variant_plan(op->n_pad, op->mf_variant);
}

// Shape of the single-trajectory (symmetric) launch: rows per warp, block width, slots.
void mf_launch_shape(nf_operator *op, int *R, int *TJ, int *splits) {
    if (fused_fits(op, 1)) {
        *R = kFusedRows;
        *TJ = kFusedTile;
        *splits = 1;
        return;
    }
    if (!use_sym(op)) {
        const SplitPlan pl = mf_plan(op);
        *R = kMfVariants[op->mf_variant].R;
        *TJ = kMfVariants[op->mf_variant].TJ;
        *splits = pl.splits;
        return;
    }
    *R = kPassRows;
    *TJ = op->sym_blk;
    *splits = sym_slots(op);
}

// Rows per warp of the scalar kernel (2 or 4 are instantiated).
static int mf_rows_per_warp(int64_t n_pad) { return n_pad >= 16384 ? 4 : 2; }

// Time the symmetric kernel's node blocks (1,024, or 512 where those give too few CTAs) once on
// this operator's nodes and keep the faster (cached per device, padded size, form and tune_class).  Runs
// outside any stream capture.
nf_status mf_autotune(nf_operator *op, cudaStream_t s) {
    static std::mutex mu;
    static std::map<std::tuple<int, int64_t, int, int>, int> cache;
    op->mf_variant = default_variant(op->n_pad);
    if (!sym_layout_fits(op)) return NF_OK;  // packed by default
    if (3 * sym_pairs_1024(op) < 2 * (int64_t)num_sms()) {
        op->sym_blk = op->auto_blk = op->n > kFusedMaxN ? 256 : 128;  // 128: only when the schedule asks for symmetric
        return NF_OK;
    }
    // 512-node blocks only where 1,024-node pairs fill fewer than four waves of two CTAs per
    // SM (n below ~49,000): four times the CTAs even out the last wave there
    if (sym_pairs_1024(op) >= 8 * (int64_t)num_sms()) return NF_OK;
    const auto key = std::make_tuple(op->device, op->n_pad, op->form, op->tune_class);
    {
        std::lock_guard<std::mutex> lock(mu);
        auto it = cache.find(key);
        if (it != cache.end()) {
            op->sym_blk = it->second;
            return NF_OK;
        }
    }
    cudaEvent_t e0, e1;
    NF_CUDA_TRY(cudaEventCreate(&e0));
    NF_CUDA_TRY(cudaEventCreate(&e1));
    float best = 1e30f;
    int best_blk = 1024;
    NF_TRY(ensure_workspace(op, 1, (int)(op->n_pad / 512), s));
    NF_CUDA_TRY(cudaMemsetAsync(op->g, 0, sizeof(float) * op->n_pad, s));
    for (const int blk : {1024, 512}) {
        op->sym_blk = blk;
        NF_TRY(launch_sym(op, 1, 0, s));  // warm-up
        // each launch between its own events, the fastest of three: host-side gaps between
        // launches (a profiler attached to the process, a busy host) then do not enter
        float ms = 1e30f;
        for (int rep = 0; rep < 3; ++rep) {
            NF_CUDA_TRY(cudaEventRecord(e0, s));
            NF_TRY(launch_sym(op, 1, 0, s));
            NF_CUDA_TRY(cudaEventRecord(e1, s));
            NF_CUDA_TRY(cudaEventSynchronize(e1));
            float t = 0.f;
            NF_CUDA_TRY(cudaEventElapsedTime(&t, e0, e1));
            ms = std::min(ms, t);
        }
        if (ms < best) {
            best = ms;
            best_blk = blk;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    op->sym_blk = best_blk;
    std::lock_guard<std::mutex> lock(mu);
    cache[key] = best_blk;
    return NF_OK;
}

// ---- block-pair culling (opt-in).  A block pair whose bounding boxes are so far apart that
// the wider Gaussian's exponent exceeds 160 (log2 units) for every pair in it contributes
// exactly zero in FP32: ex2 flushes results below 2^-126 to 0, e1 = e2^m then is 0 too, and
// adding those zeros leaves every row and column sum unchanged.  Culling skips such pairs:
// the symmetric kernel runs over the live pairs only, and each node then adds the slots of
// its block's live pairs, in ascending slot order, into slot 0 -- the same nonzero terms in
// the same order as the full sum, so results are bit-identical to it.
__global__ void cull_reduce_kernel(float *__restrict__ partial, int64_t n_pad, int B, int b0, int blk,
                                   const int *__restrict__ ptr, const int *__restrict__ slots) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int b = b0 + blockIdx.y;  // trajectory
    if (i >= n_pad) return;
    const int K = (int)(i / blk);
    float acc = 0.f;
    for (int p = ptr[K]; p < ptr[K + 1]; ++p) acc += partial[((int64_t)slots[p] * B + b) * n_pad + i];
    partial[(int64_t)b * n_pad + i] = acc;
}

// The adjoint pass over culled pairs: each node adds its 1,024-node block's live W nu slots
// of trajectory b into slot 0 (the epilogue then reads one slot).
nf_status launch_adj_cull_reduce(nf_operator *op, float *wpart, int B, int b, cudaStream_t s) {
    cull_reduce_kernel<<<dim3((unsigned)ceil_div(op->n_pad, 256), 1), 256, 0, s>>>(
        wpart, op->n_pad, B, b, 1024, op->adj_ptr, op->adj_slots);
    NF_CUDA_TRY(cudaGetLastError());
    return NF_OK;
}

// Live block pairs of the node blocks of size blk, in the stored coordinate units, for a kernel
// whose wider exponential has exponent wide * r^2 there; per: the period in these units (0:
// none).  Also each block's live slots (CSR).
struct CullLists {
    std::vector<int> pairs, ptr, slots;
};

static void build_cull_lists(const std::vector<float> &xyz, int64_t n, int64_t n_pad, int64_t blk, double wide,
                             double per, CullLists &L) {
    const int64_t nb = n_pad / blk, npairs = nb * (nb + 1) / 2;
    std::vector<double> lo((size_t)3 * nb, 1e300), hi((size_t)3 * nb, -1e300);
    std::vector<char> empty((size_t)nb, 1);
    for (int64_t p = 0; p < n; ++p) {
        const int64_t K = p / blk;
        empty[(size_t)K] = 0;
        for (int d = 0; d < 3; ++d) {
            const double v = (double)xyz[(size_t)(d * n_pad + p)];
            lo[(size_t)(3 * K + d)] = std::min(lo[(size_t)(3 * K + d)], v);
            hi[(size_t)(3 * K + d)] = std::max(hi[(size_t)(3 * K + d)], v);
        }
    }
    auto live = [&](int64_t I, int64_t J) {
        if (I == J) return true;
        if (empty[(size_t)I] || empty[(size_t)J]) return false;  // no real node: all g are 0
        double d2 = 0.0;
        for (int d = 0; d < 3; ++d) {
            const double cI = 0.5 * (lo[(size_t)(3 * I + d)] + hi[(size_t)(3 * I + d)]);
            const double cJ = 0.5 * (lo[(size_t)(3 * J + d)] + hi[(size_t)(3 * J + d)]);
            const double H = 0.5 * (hi[(size_t)(3 * I + d)] - lo[(size_t)(3 * I + d)]) +
                             0.5 * (hi[(size_t)(3 * J + d)] - lo[(size_t)(3 * J + d)]);
            double D = cJ - cI;
            if (per > 0.0 && d < 2) D -= per * std::nearbyint(D / per);  // nearest image
            const double gap = std::max(0.0, std::fabs(D) - H);
            d2 += gap * gap;
        }
        return wide * d2 < 160.0 * (1.0 + 1e-4);
    };
    std::vector<char> lv((size_t)npairs);
    L.pairs.clear();
    for (int64_t J = 0; J < nb; ++J)
        for (int64_t I = 0; I <= J; ++I) {
            const int64_t t = J * (J + 1) / 2 + I;
            lv[(size_t)t] = live(I, J) ? 1 : 0;
            if (lv[(size_t)t]) L.pairs.push_back((int)t);
        }
    L.ptr.assign((size_t)nb + 1, 0);
    L.slots.clear();
    for (int64_t K = 0; K < nb; ++K) {
        for (int64_t S = 0; S < nb; ++S) {
            const int64_t a = std::min(K, S), b = std::max(K, S);
            if (lv[(size_t)(b * (b + 1) / 2 + a)]) L.slots.push_back((int)S);
        }
        L.ptr[(size_t)K + 1] = (int)L.slots.size();
    }
}

static nf_status upload_int(const std::vector<int> &v, int **dst, cudaStream_t s) {
    cudaFree(*dst);
    *dst = nullptr;
    NF_CUDA_TRY(cudaMalloc(dst, sizeof(int) * std::max<size_t>(1, v.size())));
    NF_CUDA_TRY(cudaMemcpyAsync(*dst, v.data(), sizeof(int) * v.size(), cudaMemcpyHostToDevice, s));
    return NF_OK;
}

nf_status mf_set_cull(nf_operator *op, int enable, int64_t *live_out, int64_t *total_out, cudaStream_t s) {
    const int64_t n = op->n, n_pad = op->n_pad, blk = op->sym_blk, nb = n_pad / blk, npairs = nb * (nb + 1) / 2;
    if (total_out) *total_out = npairs;
    if (live_out) *live_out = npairs;
    if (op->mf_cull) destroy_graphs(op);
    op->mf_cull = 0;
    if (!enable) return NF_OK;
    // boxes of the node blocks over their real nodes, in the kernels' coordinate units
    std::vector<float> xyz((size_t)3 * n_pad);
    NF_CUDA_TRY(cudaMemcpyAsync(xyz.data(), op->xyz, sizeof(float) * 3 * n_pad, cudaMemcpyDeviceToHost, s));
    NF_CUDA_TRY(cudaStreamSynchronize(s));
    const nf_kernel &k = op->kp;
    const double k2 = ((double)k.s1 * k.s1) / ((double)k.s2 * k.s2);
    const double per = (double)mf_period(op);
    // forward: the wider exponential evaluated (the second Gaussian is not when A2 = 0);
    // adjoint: 1,024-node blocks, and both Gaussians always (the parameter sums of A2 and s2
    // need e2 even when A2 = 0)
    CullLists fw, ad;
    build_cull_lists(xyz, n, n_pad, blk, op->form > 0 ? 1.0 : std::min(1.0, k2), per, fw);
    build_cull_lists(xyz, n, n_pad, 1024, op->form >= 2 ? 1.0 : std::min(1.0, k2), per, ad);
    NF_TRY(upload_int(fw.pairs, &op->cull_pairs, s));
    NF_TRY(upload_int(fw.ptr, &op->cull_ptr, s));
    NF_TRY(upload_int(fw.slots, &op->cull_slots, s));
    NF_TRY(upload_int(ad.pairs, &op->adj_pairs, s));
    NF_TRY(upload_int(ad.ptr, &op->adj_ptr, s));
    NF_TRY(upload_int(ad.slots, &op->adj_slots, s));
    NF_CUDA_TRY(cudaStreamSynchronize(s));
    op->cull_live = (int64_t)fw.pairs.size();
    op->adj_live = (int64_t)ad.pairs.size();
    op->mf_cull = 1;
    if (live_out) *live_out = op->cull_live;
    return NF_OK;
}

// The same column splits for a kernel of R rows per warp.
static SplitPlan rows_of(SplitPlan pl, int64_t n_pad, int R) {
    pl.rows_per_block = MF_WARPS * R;
    pl.row_blocks = n_pad / pl.rows_per_block;
    return pl;
}

// Groups of exactly 8 take the scalar kernel, too, in the general form where few tiles are far enough to be
// skipped (the wider Gaussian reaches over 0.7 of the nodes' bounding box's diagonal): two
// exponentials per pair are then needed nearly everywhere, and the packed kernel's operands keep its
// FMA pipe at half rate.  Per sum, packed / scalar, (1.2, 0.08, 0.6, 0.25) on an ellipsoid of diameter 2: n = 20,000
// 342 / 333 us, 30,000 748 / 716, 50,000 1,997 / 1,854; (1.2, 0.13, 0.6, 0.04), which skips: 323 / 334,
// 677 / 715, 1,742 / 1,853.
static bool scalar_8(const nf_operator *op) {
    if (op->form != 0 || op->n_pad < 16384 || op->kp.period > 0.f) return false;
    float tail, skip;
    class_limits(op, &tail, &skip);
    return op->span2 <= 2.f * skip;
}

nf_status launch_mf_pair(nf_operator *op, int B, cudaStream_t s, int *splits_out) {
    if (B <= kSymMaxB && use_sym(op)) {  // symmetric kernel, one partial slot per node block
        NF_TRY(launch_sym(op, B, 0, s));
        *splits_out = sym_slots(op);
        if (op->mf_cull) {  // only live pairs ran: add each node's live slots into slot 0
            cull_reduce_kernel<<<dim3((unsigned)ceil_div(op->n_pad, 256), (unsigned)B), 256, 0, s>>>(
                op->partial, op->n_pad, B, 0, op->sym_blk, op->cull_ptr, op->cull_slots);
            NF_CUDA_TRY(cudaGetLastError());
            *splits_out = 1;
        }
        return NF_OK;
    }
    if (B == 1) {  // the packed kernel over (row block, column split) items
        const SplitPlan pl = mf_plan(op);
        NF_TRY(launch_mf_packed(op, 1, 0, 1, pl, s));
        *splits_out = pl.splits;
        return NF_OK;
    }
    // several: groups of exactly 16 on the scalar kernel, the rest on the packed one, over the same
    // column splits
    const SplitPlan pl = multi_plan(op);
    *splits_out = pl.splits;
    const int full = B / 16, R = mf_rows_per_warp(op->n_pad);
    if (full > 0) {
        const SplitPlan sixteen = rows_of(pl, op->n_pad, R);
        if (R == 4)
            NF_TRY((launch_mf_group<16, 4>(op, B, 0, full, sixteen, s)));
        else
            NF_TRY((launch_mf_group<16, 2>(op, B, 0, full, sixteen, s)));
    }
    const int left = B - 16 * full;
    if (left == 1) {
        // One more trajectory: the packed kernel, over the same splits, instead of a group of four.  Per sum of
        // 17 trajectories (ratio-4 kernel), four / one: n = 8,000 166 / 163 us, 15,000 464 / 450, 30,000
        // 1,545 / 1,429; eight rows and 1,024-column tiles measured the same.
        if (R == 4)
            launch_packed<4, 512>(op, B, 16 * full, 1, rows_of(pl, op->n_pad, 4), s);
        else
            launch_packed<2, 512>(op, B, 16 * full, 1, rows_of(pl, op->n_pad, 2), s);
        NF_CUDA_TRY(cudaGetLastError());
        return NF_OK;
    }
    if (left == 8 && scalar_8(op))
        return launch_mf_group<8, 4>(op, B, 16 * full, 1, rows_of(pl, op->n_pad, 4), s);
    return left > 0 ? launch_multi(op, B, 16 * full, s) : NF_OK;
}

// Launch plan of launch_mf_pair_single: at most max_splits column splits.
SplitPlan plan_mf_pair_single(int64_t n_pad, int max_splits) {
    const int R = mf_rows_per_warp(n_pad);
    return plan_splits(n_pad, MF_WARPS * R, MF_TJ, R == 4 ? mf_resident<1, 4>() : mf_resident<1, 2>(), max_splits);
}

// Single-trajectory pair sums into caller-provided buffers (x4, g padded to n_pad,
// partial [splits][n_pad]); the planner considers at most max_splits column splits.
nf_status launch_mf_pair_single(const float4 *x4, const float *g, int64_t n_pad, const nf_kernel &k, int max_splits,
                                float *partial, int *err, cudaStream_t s, int *splits_out) {
    const int R = mf_rows_per_warp(n_pad);
    const SplitPlan pl = plan_mf_pair_single(n_pad, max_splits);
    const float L2E = 1.4426950408889634f;
    const float c1 = -L2E / (k.s1 * k.s1), c2 = -L2E / (k.s2 * k.s2);
    dim3 grid((unsigned)pl.row_blocks, (unsigned)pl.splits, 1);
    if (R == 4)
        mf_pair_kernel<1, 4><<<grid, MF_THREADS, sizeof(MfSmem<1>), s>>>(x4, g, n_pad, 1, 0, pl.jchunk, c1, c2, k.A1,
                                                                      k.A2, k.period, partial, err);
    else
        mf_pair_kernel<1, 2><<<grid, MF_THREADS, sizeof(MfSmem<1>), s>>>(x4, g, n_pad, 1, 0, pl.jchunk, c1, c2, k.A1,
                                                                      k.A2, k.period, partial, err);
    NF_CUDA_TRY(cudaGetLastError());
    *splits_out = pl.splits;
    return NF_OK;
}

// ----------------------------------------------------------------------------
// Elementwise kernels.

// The elementwise kernels run over the operator's positions (thread idx = b n + p) and touch
// the caller's arrays at node perm[p] (perm == nullptr: the same order).

// g[b, p] = q_p f_b(u[b, perm[p]]) (q == nullptr: f alone);  optionally U[b, p] = us[b, p] = u.
__global__ void prep_g_kernel(const float *__restrict__ u, const int *__restrict__ perm, int64_t n, int64_t n_pad,
                              int B, const float *__restrict__ q, const float *__restrict__ beta,
                              const float *__restrict__ theta, float *__restrict__ g, float *__restrict__ U,
                              float *__restrict__ us) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)B * n) return;
    const int b = (int)(idx / n);
    const int64_t j = idx - (int64_t)b * n;
    const float uv = u[perm ? (int64_t)b * n + perm[j] : idx];
    const float f = firing_rate(uv, beta[b], theta[b]);
    g[(int64_t)b * n_pad + j] = q ? q[j] * f : f;
    if (U) U[idx] = uv;
    if (us) us[idx] = uv;
}

nf_status launch_prep_g(nf_operator *op, const float *u, int B, const float *beta, const float *theta,
                        bool copy_to_U, cudaStream_t s) {
    const int64_t tot = (int64_t)B * op->n;
    const int T = 256;
    const bool mf = q_on_vector(op);
    prep_g_kernel<<<(unsigned)ceil_div(tot, T), T, 0, s>>>(u, op->perm, op->n, op->n_pad, B, mf ? op->q : nullptr,
                                                          beta, theta, op->g, copy_to_U ? op->U : nullptr,
                                                          copy_to_U ? op->us : nullptr);
    NF_CUDA_TRY(cudaGetLastError());
    return NF_OK;
}

__global__ void reduce_I_kernel(const float *partial, int splits, int64_t n, int64_t n_pad, int B,
                                const float *__restrict__ rs, const int *__restrict__ perm, float *__restrict__ I) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (idx >= (int64_t)B * n) return;
    const int b = (int)(idx / n);
    const int64_t i = idx - (int64_t)b * n;
    const float acc = sum_slots(partial + (int64_t)b * n_pad + i, (int64_t)B * n_pad, splits);
    I[perm ? (int64_t)b * n + perm[i] : idx] = rs ? acc * rs[i] : acc;
}

nf_status launch_reduce_I(nf_operator *op, int B, int splits, float *I, cudaStream_t s) {
    const int64_t tot = (int64_t)B * op->n;
    const int T = 256;
    const float *rs = (op->path == NF_DENSE_BF16X2) ? op->rs : nullptr;
    NF_CUDA_TRY(launch_dependent(reduce_I_kernel, dim3((unsigned)ceil_div(tot, T)), T, 0, s, true, op->partial, splits,
                                 op->n, op->n_pad, B, rs, op->perm, I));
    return NF_OK;
}

// ----------------------------------------------------------------------------
__global__ void rk4_stage_kernel(StageKArgs a) {
    // What earlier stage kernels wrote is complete (pdl_trigger of the pair kernel in between), so
    // the state is read while the pair kernel still runs; only the partial sums wait for it.
    const long long step = ld_l2(a.step_ctr);
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = idx < (int64_t)a.B * a.n;
    const int b = in ? (int)(idx / a.n) : 0;
    const int64_t i = in ? idx - (int64_t)b * a.n : 0;
    const StageNode sn = stage_load(a, b, i, in ? idx : 0);
    const float rsv = a.rs ? a.rs[i] : 1.f;
    float gam = 0.f;
    if (a.F.kind != NF_FORCE_NONE) {
        __shared__ double time_cs[2];  // cos t, sin t of the stage
        if (threadIdx.x == 0) {
            const double cs = (a.stage == 1) ? 0.0 : (a.stage == 4 ? 1.0 : 0.5);
            const double t0 = __longlong_as_double(ld_l2(reinterpret_cast<const long long *>(a.t0)));
            const double ts = t0 + (double)step * a.dt + cs * a.dt;
            sincos(ts, &time_cs[1], &time_cs[0]);
        }
        __syncthreads();
        if (in) gam = (float)forcing_value(a.F, a.fc, a.x4, i, sn.node, time_cs[0], time_cs[1], sn.bb, sn.th);
    }
    pdl_wait();
    pdl_trigger();
    if (in) {
        float I = sum_slots(a.partial + (int64_t)b * a.n_pad + i, (int64_t)a.B * a.n_pad, a.splits);
        if (a.rs) I *= rsv;
        stage_update(a, sn, step, b, i, idx, I, gam, a.g);
    }
    step_done(a, gridDim.x);
}

// Start a new nf_rk4_advance call: clock t0, step counter 0, no block of a step counted yet.
__global__ void set_clock_kernel(double *t0_dev, long long *step_ctr, unsigned *done_ctr, double t0) {
    *t0_dev = t0;
    *step_ctr = 0;
    *done_ctr = 0u;
}

nf_status launch_set_clock(nf_operator *op, double t0, cudaStream_t s) {
    set_clock_kernel<<<1, 1, 0, s>>>(op->t0_dev, op->step_ctr, op->done_ctr, t0);
    NF_CUDA_TRY(cudaGetLastError());
    return NF_OK;
}

static FlatConst flat_const(const nf_forcing &F, const nf_kernel &kp) {
    FlatConst c{};
    const double sg2 = F.sigma * F.sigma;
    c.L = kp.period;
    c.iL = 1.0 / c.L;
    c.r = 1.0 / (2.0 * sg2);
    c.norm = 1.0 / (2.0 * kPi * sg2);
    const double amp[2] = {(double)kp.A1, -(double)kp.A2}, wid[2] = {(double)kp.s1, (double)kp.s2};
    for (int h = 0; h < 2; ++h) {
        if (amp[h] == 0.0) continue;
        const double p = 1.0 / (wid[h] * wid[h]), s = p + c.r;
        const double e = std::sqrt(kPi) * wid[h] * std::erf(0.5 * c.L / wid[h]);
        c.c0 += amp[h] * F.c * e * e;
        c.t[c.terms++] = FlatTerm{amp[h] * c.norm, c.r / s, -p * c.r / s, std::sqrt(s), 0.5 * std::sqrt(kPi / s)};
    }
    return c;
}

static StageKArgs stage_args(nf_operator *op, int B, const StageParams &p) {
    StageKArgs a{};
    a.partial = op->partial;
    a.splits = p.splits;
    a.n = op->n;
    a.n_pad = op->n_pad;
    a.B = B;
    a.u = p.u;
    a.us = op->perm ? op->us : p.u;
    a.U = op->U;
    a.ks = op->ks;
    a.g = op->g;
    a.q = q_on_vector(op) ? op->q : nullptr;
    a.rs = (op->path == NF_DENSE_BF16X2) ? op->rs : nullptr;
    a.beta = p.beta;
    a.theta = p.theta;
    a.F = p.forcing;
    if (a.F.kind == NF_FORCE_MMS_FLAT) a.fc = flat_const(a.F, op->kp);
    a.x4 = op->x4;
    a.t0 = op->t0_dev;
    a.dt = p.dt;
    a.stage = p.stage;
    a.step_ctr = op->step_ctr;
    a.done_ctr = op->done_ctr;
    a.ckpt = p.ckpt;
    a.C = p.C;
    a.err = op->err;
    a.perm = op->perm;
    a.stage_out = p.stage_out;
    return a;
}

nf_status launch_stage(nf_operator *op, int B, const StageParams &p, cudaStream_t s) {
    const StageKArgs a = stage_args(op, B, p);
    const int64_t tot = (int64_t)B * op->n;
    const int T = 256;
    NF_CUDA_TRY(launch_dependent(rk4_stage_kernel, dim3((unsigned)ceil_div(tot, T)), T, 0, s, p.overlap, a));
    return NF_OK;
}

nf_status fused_stage(nf_operator *op, int B, const StageParams &p, cudaStream_t s) {
    const int64_t half = (int64_t)B * op->n_pad;
    float *const g_in = op->g + ((p.stage - 1) & 1) * half;
    const FusedOut fo{stage_args(op, B, p), op->g + (p.stage & 1) * half, nullptr, op->perm, op->n};
    NF_CUDA_TRY(launch_fused<1>(op, B, g_in, fo, p.overlap, s));
    return NF_OK;
}

nf_status fused_apply(nf_operator *op, int B, float *I, cudaStream_t s) {
    FusedOut fo{};
    fo.I = I;
    fo.perm = op->perm;
    fo.n = op->n;
    NF_CUDA_TRY(launch_fused<2>(op, B, op->g, fo, true, s));
    return NF_OK;
}

}  // namespace nfi
