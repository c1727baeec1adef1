// nf_adj_sym.cu -- symmetric pair kernel of the discrete adjoint (one trajectory b).
//
// W is symmetric, so each unordered pair of nodes is evaluated once, as in the forward
// symmetric kernel (nf_sym.cu): one CTA per pair of node blocks in Hilbert order (I <= J), rows of
// block I swept R at a time against block J in shared memory, expanded about the pass's centre
// when its rows are close.  Per pair it
//   * adds e1, e2 times nu to the row sums (W nu)_i and, per warp in shared memory, to the
//     column sums (W nu)_j: row sums go to slot J, column sums to slot I of wpart, the
//     stage epilogue adds the slots in a fixed order;
//   * adds the pair's share of the kernel-parameter sums
//         P1 = sum nu_i g_j e1, Q1 = sum nu_i g_j r^2 e1, P2 = sum nu_i g_j e2, Q2 = ... r^2 e2
//     over ordered pairs: off the diagonal an unordered pair carries the weight
//     nu_i g_j + nu_j g_i, on a diagonal block pair every ordered pair is swept with
//     nu_i g_j.  Each CTA writes its four sums (r^2 in exponent units: of s2 when M > 0, else
//     of s1) to gpart; a fixed-order FP64 reduction adds them.
//
// Tile classes as in nf_sym.cu, with the limits of these sums: skip where both exponentials are
// exactly 0, tail where the narrow one is (e1 = e2^M rounds to 0 below 2^-150), so that its four
// sums gain nothing: 10 FMA-pipe operations per pair instead of 16.  Swept tiles give the full
// form's sums bit for bit; blocks with a non-finite nu or g sweep every tile in full.  Bound: the FP32
// FMA pipe (63 % busy, three-operand packed FMAs); torus n = 40,000 617 -> 478 us per pass.
#include "nf_pairs.cuh"

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>

namespace nfi {

constexpr int AS_THREADS = 256;
constexpr int AS_WARPS = AS_THREADS / 32;
// shared memory (4-byte words): columns x, y, z, nu, g (5 BLK); rows: operands, factors, nu, g
// (8 BLK); pass centres and half extents (BLK); tile boxes (BLK / 16); column sums per warp
constexpr size_t as_smem_bytes(int blk) {
    return sizeof(float) * ((5 + 8 + 1 + AS_WARPS) * (size_t)blk + blk / 16);
}

// R = 4: two CTAs per SM (128 registers); R = 8: one CTA per SM with the whole register
// file.  BLK: node block of 1,024 or 512 (four times the CTAs, for node sets whose 1,024-node
// block pairs leave the last wave of CTAs partly empty).
template <int R, int M, int BLK>
__global__ void __launch_bounds__(AS_THREADS, R >= 8 ? 1 : 2)
adj_sym_kernel(SymNodes nd, const float *nu_all, const float *g_all, int B, int b, float k2,
               float A1, float A2, float per, float lim_tail, float lim_skip, float *__restrict__ wpart,
               float *__restrict__ gpart, const int *__restrict__ pairs) {
    static_assert(M == 0 || (M >= 2 && M <= 4), "width ratio M must be 0 (general), 2, 3 or 4");
    static_assert(R == 4 || R == 8, "rows per warp");
    static_assert(BLK == 512 || BLK == 1024, "block size");
    constexpr int NPASS = BLK / R, NT = BLK / kTileCols;
    // CW (integer width ratios, A2 != 0): per pair the W nu sums take the combined weight
    // u = e2 + c_i e1 (c_i = -A1 f1 / (A2 f2), as in mf_sym_kernel), and the parameter sums
    // the symmetric pair weight p_ij = nu_i g_j + g_i nu_j, formed once per pair: per row
    // the lane keeps U = sum u nu_j (the W nu row sum), sum e1 p, sum e2 p, sum arg e1 p and
    // sum arg e2 p -- 16 FMA-pipe instructions per row and column pair instead of 17, and
    // five accumulators per row instead of eight.
    constexpr bool CW = M >= 2;
    extern __shared__ __align__(16) float as_smem[];
    float *xs = as_smem, *ys = xs + BLK, *zs = ys + BLK, *vs = zs + BLK, *gsm = vs + BLK;
    float4 *rg = reinterpret_cast<float4 *>(gsm + BLK);
    float2 *rw = reinterpret_cast<float2 *>(rg + BLK);
    float *rnu = reinterpret_cast<float *>(rw + BLK), *rgv = rnu + BLK;
    float4 *pc = reinterpret_cast<float4 *>(rgv + BLK), *pe = pc + BLK / kPassRows;
    float4 *tcs = pe + BLK / kPassRows, *tes = tcs + NT;
    float *colacc = reinterpret_cast<float *>(tes + NT);  // [AS_WARPS][BLK]
    __shared__ float gred[AS_WARPS][4];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t n_pad = nd.n_pad;
    int I, J;
    sym_pair(pairs ? (int64_t)__ldg(pairs + blockIdx.x) : (int64_t)blockIdx.x, I, J);  // pairs: live list
    const bool diag = I == J;
    const float *nu = nu_all + (int64_t)b * n_pad, *g = g_all + (int64_t)b * n_pad;
    const int64_t cbase = (int64_t)J * BLK, rbase = (int64_t)I * BLK;
    const float iper = per > 0.f ? 1.f / per : 0.f;
    float *out_rows = wpart + ((int64_t)J * B + b) * n_pad + rbase;
    float *out_cols = wpart + ((int64_t)I * B + b) * n_pad + cbase;
    float *out_g = gpart + ((int64_t)b * gridDim.x + blockIdx.x) * 4;

    bool bad = false, live = false;
    for (int k = tid; k < BLK / 4; k += AS_THREADS) {
        cp_async16(xs + 4 * k, nd.xyz + cbase + 4 * k);
        cp_async16(ys + 4 * k, nd.xyz + n_pad + cbase + 4 * k);
        cp_async16(zs + 4 * k, nd.xyz + 2 * n_pad + cbase + 4 * k);
    }
    for (int k = tid; k < BLK; k += AS_THREADS) cp_async16(rg + k, nd.rg + rbase + k);
    for (int k = tid; k < BLK / 2; k += AS_THREADS) cp_async16(rw + 2 * k, nd.rw + rbase + 2 * k);
    for (int k = tid; k < BLK / kPassRows; k += AS_THREADS) {
        cp_async16(pc + k, nd.pc + rbase / kPassRows + k);
        cp_async16(pe + k, nd.pe + rbase / kPassRows + k);
    }
    if (tid < NT) {
        cp_async16(tcs + tid, nd.tc + cbase / kTileCols + tid);
        cp_async16(tes + tid, nd.te + cbase / kTileCols + tid);
    }
    if (!diag)
        for (int k = tid; k < AS_WARPS * BLK / 4; k += AS_THREADS)
            reinterpret_cast<float4 *>(colacc)[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    // everything above depends on the operator alone; nu and g are written by the kernel before
    pdl_wait();
    pdl_trigger();
    for (int k = tid; k < BLK / 4; k += AS_THREADS) {
        const float4 v[4] = {
            reinterpret_cast<const float4 *>(nu + cbase)[k], reinterpret_cast<const float4 *>(g + cbase)[k],
            reinterpret_cast<const float4 *>(nu + rbase)[k], reinterpret_cast<const float4 *>(g + rbase)[k]};
        reinterpret_cast<float4 *>(vs)[k] = v[0];
        reinterpret_cast<float4 *>(gsm)[k] = v[1];
        reinterpret_cast<float4 *>(rnu)[k] = v[2];
        reinterpret_cast<float4 *>(rgv)[k] = v[3];
#pragma unroll
        for (int t = 0; t < 4; ++t)  // 0 * v is NaN for a non-finite v
            bad |= !(0.f * v[t].x + 0.f * v[t].y + 0.f * v[t].z + 0.f * v[t].w == 0.f);
    }
    if (tid < NT * NT) {
        const int64_t ti = rbase / kTileCols + tid / NT, tj = cbase / kTileCols + tid % NT;
        live = box_d2(__ldg(nd.tc + ti), __ldg(nd.te + ti), __ldg(nd.tc + tj), __ldg(nd.te + tj), per, iper) <= lim_skip;
    }
    if (__syncthreads_or(bad)) lim_tail = lim_skip = __int_as_float(0x7f800000), live = true;
    if (!__syncthreads_or(live)) {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = tid; k < BLK / 4; k += AS_THREADS) {
            reinterpret_cast<float4 *>(out_rows)[k] = zero;
            reinterpret_cast<float4 *>(out_cols)[k] = zero;
        }
        if (tid < 4) out_g[tid] = 0.f;
        cp_async_wait_all();
        return;
    }
    cp_async_wait_all();
    __syncthreads();

    const u64 nk2 = f2_dup(-k2);
    const u64 ipp = f2_dup(iper), npp = f2_dup(-per), mgp = f2_dup(kRintMagic);
    const u64 *xs2 = reinterpret_cast<const u64 *>(xs), *ys2 = reinterpret_cast<const u64 *>(ys);
    const u64 *zs2 = reinterpret_cast<const u64 *>(zs), *vs2 = reinterpret_cast<const u64 *>(vs);
    const u64 *gs2 = reinterpret_cast<const u64 *>(gsm);
    u64 *cw2 = reinterpret_cast<u64 *>(colacc + warp * BLK);
    const int ntile = (int)min((int64_t)NT, (nd.n - cbase + kTileCols - 1) / kTileCols);  // tiles with real nodes
    float P1 = 0.f, Q1 = 0.f, P2 = 0.f, Q2 = 0.f;  // per lane, over all its pairs
    for (int ps = warp; ps < NPASS; ps += AS_WARPS) {
        const int r0 = ps * R, grp = r0 / kPassRows;
        if (rbase + r0 >= nd.n) break;  // padding: no row to write, nu = g = 0 in every other sum
        const float4 c = pc[grp], e = pe[grp];
        float d2 = 3.4e38f;
        if (lane < ntile) d2 = box_d2(c, e, tcs[lane], tes[lane], per, iper);
        const unsigned live_t = __ballot_sync(0xffffffffu, lane < ntile && d2 <= lim_skip);
        // periodic distances take plain differences, reduced pair by pair; so do rows that the forward
        // sums expand for the first Gaussian alone (A2 = 0) but that lie too far apart for the second
        const bool local = c.w == 1.f && !(per > 0.f) && (M > 0 || k2 * e.w <= kSymLocalSpread);  // warp-uniform
        const unsigned full_t = local ? live_t & __ballot_sync(0xffffffffu, d2 <= lim_tail) : live_t;
        const unsigned tail_t = live_t & ~full_t;
        // per row, over the lane's columns j (e1, e2 without the row factors):
        //   a = sum e nu_j, b = sum e g_j, c = sum arg e g_j, d = sum arg e nu_j
        // CW: a1 = U, b1, b2 = sum e p, c1, c2 = sum arg e p; pn, pg = nu_i, g_i; h1 = c_i
        u64 xi[R], yi[R], zi[R], h1[R], h2[R], a1[R], a2[R], b1[R], b2[R], c1[R], c2[R], d1[R], d2s[R];
        u64 pn[R], pg[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float4 p = rg[r0 + r];
            float2 w = rw[r0 + r];
            const float nui = rnu[r0 + r], gi = diag ? 0.f : rgv[r0 + r];
            if (!local) {
                p.x = __ldg(nd.xyz + rbase + r0 + r);
                p.y = __ldg(nd.xyz + n_pad + rbase + r0 + r);
                p.z = __ldg(nd.xyz + 2 * n_pad + rbase + r0 + r);
                w = make_float2(CW ? -(A1 / A2) : A1, -A2);
            }
            xi[r] = f2_dup(p.x);
            yi[r] = f2_dup(p.y);
            zi[r] = f2_dup(p.z);
            h1[r] = f2_dup(CW ? w.x : w.x * nui);
            h2[r] = f2_dup(w.y * nui);
            if constexpr (CW) {
                pn[r] = f2_dup(nui);
                pg[r] = f2_dup(gi);
                a1[r] = b1[r] = b2[r] = c1[r] = c2[r] = 0ull;
            } else {
                a1[r] = a2[r] = b1[r] = b2[r] = c1[r] = c2[r] = d1[r] = d2s[r] = 0ull;
            }
        }
        const u64 cxp = f2_dup(c.x), cyp = f2_dup(c.y), czp = f2_dup(c.z);
        // per (row, column pair): e1, e2 from the exponent argument arg (r^2 - n_i in the
        // expanded form, r^2 otherwise), then the W nu and row-sum updates; TAIL: e1 = 0
        auto pair = [&](auto tail, int r, u64 arg, u64 vj, u64 gj, u64 &cacc) {
            constexpr bool TAIL = decltype(tail)::value;
            float s0, s1v;
            f2_unpack(arg, s0, s1v);
            if constexpr (CW) {
                const u64 e2 = f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v));
                const u64 s2e = f2_mul(arg, e2);
                const u64 pw = f2_fma(pn[r], gj, f2_mul(pg[r], vj));
                u64 u = e2;
                if constexpr (!TAIL) {
                    const u64 sq = f2_mul(e2, e2);
                    const u64 e1 = M == 2 ? sq : (M == 3 ? f2_mul(sq, e2) : f2_mul(sq, sq));
                    const u64 s1e = f2_mul(arg, e1);
                    u = f2_fma(e1, h1[r], e2);
                    b1[r] = f2_fma(e1, pw, b1[r]);
                    c1[r] = f2_fma(s1e, pw, c1[r]);
                }
                a1[r] = f2_fma(u, vj, a1[r]);
                cacc = f2_fma(u, h2[r], cacc);
                b2[r] = f2_fma(e2, pw, b2[r]);
                c2[r] = f2_fma(s2e, pw, c2[r]);
            } else {
                const u64 e2 = f2_ex2(f2_mul(arg, nk2));
                const u64 s2e = f2_mul(arg, e2);
                cacc = f2_fma(e2, h2[r], cacc);
                if constexpr (!TAIL) {
                    const u64 e1 = f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v));
                    const u64 s1e = f2_mul(arg, e1);
                    cacc = f2_fma(e1, h1[r], cacc);
                    a1[r] = f2_fma(e1, vj, a1[r]);
                    b1[r] = f2_fma(e1, gj, b1[r]);
                    c1[r] = f2_fma(s1e, gj, c1[r]);
                    d1[r] = f2_fma(s1e, vj, d1[r]);
                }
                a2[r] = f2_fma(e2, vj, a2[r]);
                b2[r] = f2_fma(e2, gj, b2[r]);
                c2[r] = f2_fma(s2e, gj, c2[r]);
                d2s[r] = f2_fma(s2e, vj, d2s[r]);
            }
        };
        // a tile is two steps of 64 columns, two consecutive ones per lane
        auto sweep_local = [&](auto tail, unsigned tiles) {
#pragma unroll 1
            for (; tiles; tiles &= tiles - 1) {
                const int t0 = (__ffs(tiles) - 1) * (kTileCols / 2) + lane;
#pragma unroll 1
                for (int jp = t0; jp < t0 + kTileCols / 2; jp += 32) {
                    const u64 xt = f2_sub(xs2[jp], cxp), yt = f2_sub(ys2[jp], cyp), zt = f2_sub(zs2[jp], czp);
                    const u64 nj = f2_fma(zt, zt, f2_fma(yt, yt, f2_mul(xt, xt)));
                    const u64 vj = vs2[jp], gj = gs2[jp];
                    u64 cacc = 0ull;
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        pair(tail, r, f2_fma(xi[r], xt, f2_fma(yi[r], yt, f2_fma(zi[r], zt, nj))), vj, gj, cacc);
                    if (!diag) cw2[jp] = f2_add(cw2[jp], cacc);
                }
            }
        };
        auto sweep_diff = [&](auto tag, unsigned tiles) {
            constexpr bool P = decltype(tag)::value;
#pragma unroll 1
            for (; tiles; tiles &= tiles - 1) {
                const int t0 = (__ffs(tiles) - 1) * (kTileCols / 2) + lane;
#pragma unroll 1
                for (int jp = t0; jp < t0 + kTileCols / 2; jp += 32) {
                    const u64 xj = xs2[jp], yj = ys2[jp], zj = zs2[jp], vj = vs2[jp], gj = gs2[jp];
                    u64 cacc = 0ull;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        u64 dx = f2_sub(xi[r], xj), dy = f2_sub(yi[r], yj);
                        const u64 dz = f2_sub(zi[r], zj);
                        if constexpr (P) {
                            dx = f2_wrap(dx, ipp, npp, mgp);
                            dy = f2_wrap(dy, ipp, npp, mgp);
                        }
                        pair(PerTag<false>{}, r, f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx))), vj, gj, cacc);
                    }
                    if (!diag) cw2[jp] = f2_add(cw2[jp], cacc);
                }
            }
        };
        if (local) {
            sweep_local(PerTag<true>{}, tail_t);
            sweep_local(PerTag<false>{}, full_t);
        } else if (per > 0.f) {
            sweep_diff(PerTag<true>{}, full_t);
        } else {
            sweep_diff(PerTag<false>{}, full_t);
        }
        float v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            // the row factors 2^(-n_i) of e1 and e2 (n_i = 0 outside the expanded form)
            const float ni = local ? rg[r0 + r].w : 0.f;
            const float f1 = exp2f(M > 0 ? -(float)M * ni : -ni), f2 = exp2f(M > 0 ? -ni : -k2 * ni);
            if constexpr (CW) {
                const float P1s = f2_fold(b1[r]), P2s = f2_fold(b2[r]);
                v[r] = (-A2 * f2) * f2_fold(a1[r]);
                P1 += f1 * P1s;
                Q1 += f1 * (f2_fold(c1[r]) + ni * P1s);
                P2 += f2 * P2s;
                Q2 += f2 * (f2_fold(c2[r]) + ni * P2s);
            } else {
                const float A1s = f2_fold(a1[r]), A2s = f2_fold(a2[r]), B1s = f2_fold(b1[r]), B2s = f2_fold(b2[r]);
                const float nui = rnu[r0 + r], gi = diag ? 0.f : rgv[r0 + r];
                v[r] = (A1 * f1) * A1s + (-A2 * f2) * A2s;
                // pair weight e (nu_i g_j + g_i nu_j) with the row factors, g_i = 0 on diagonal
                // block pairs; r^2 = arg + n_i
                P1 += f1 * nui * B1s + f1 * gi * A1s;
                Q1 += f1 * nui * (f2_fold(c1[r]) + ni * B1s) + f1 * gi * (f2_fold(d1[r]) + ni * A1s);
                P2 += f2 * nui * B2s + f2 * gi * A2s;
                Q2 += f2 * nui * (f2_fold(c2[r]) + ni * B2s) + f2 * gi * (f2_fold(d2s[r]) + ni * A2s);
            }
        }
        int row;
        const float tot = warp_reduce_rows<R>(v, lane, row);
        if ((lane & (32 / R - 1)) == 0) out_rows[r0 + row] = tot;
    }
    // the CTA's parameter sums: lanes, then warps, in a fixed order
    float gs4[4] = {P1, Q1, P2, Q2};
#pragma unroll
    for (int k = 0; k < 4; ++k) gs4[k] = warp_sum(gs4[k]);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < 4; ++k) gred[warp][k] = gs4[k];
    __syncthreads();
    if (tid < 4) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < AS_WARPS; ++w) s += gred[w][tid];
        out_g[tid] = s;
    }
    if (diag) return;
    for (int k = tid; k < BLK; k += AS_THREADS) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < AS_WARPS; ++w) s += colacc[w * BLK + k];
        out_cols[k] = s;
    }
}

// ------------------------------------------------------------------ launch
template <int R, int BLK>
static cudaError_t adj_attrs() {
    const int smem = (int)as_smem_bytes(BLK);
    cudaError_t e = cudaFuncSetAttribute(adj_sym_kernel<R, 0, BLK>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(adj_sym_kernel<R, 2, BLK>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(adj_sym_kernel<R, 3, BLK>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(adj_sym_kernel<R, 4, BLK>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e;
}
nf_status adj_init_attrs() {
    NF_CUDA_TRY((adj_attrs<4, 1024>()));
    NF_CUDA_TRY((adj_attrs<8, 1024>()));
    NF_CUDA_TRY((adj_attrs<4, 512>()));
    NF_CUDA_TRY((adj_attrs<8, 512>()));
    return NF_OK;
}

// The adjoint kernel's node block: the tuned one, or 1,024 when culling (its live-pair lists
// are built over 1,024-node blocks).
static int adj_block(const nf_operator *op) {
    return (op->mf_cull && op->adj_pairs) || op->adj_blk == 0 ? 1024 : op->adj_blk;
}
int64_t adj_pair_count(const nf_operator *op) {
    const int64_t nb = op->n_pad / adj_block(op);
    return nb * (nb + 1) / 2;
}
int adj_slots(const nf_operator *op) { return (int)(op->n_pad / adj_block(op)); }
int64_t adj_pair_capacity(const nf_operator *op) {
    const int64_t nb = op->n_pad / 512;
    return nb * (nb + 1) / 2;
}
int adj_slot_capacity(const nf_operator *op) { return (int)(op->n_pad / 512); }

// Squared distances (stored units) beyond which a tile takes the tail form (e1 exactly 0 in
// every pair) and beyond which it adds nothing; see class_limits of the forward kernel.  The
// second Gaussian is evaluated even when A2 = 0 (the A2 and s2 gradients need it).
static void adj_limits(const nf_operator *op, float *tail, float *skip) {
    const nf_kernel &k = op->kp;
    const double k2 = ((double)k.s1 * k.s1) / ((double)k.s2 * k.s2), none = 126.0 + 4.0 + 1.0;
    double t, s;
    if (op->form >= 2) {
        s = none;
        t = (150.0 + 4.0 + 1.0) / op->form;  // M n_i <= 4 in these units
    } else {
        s = none / std::min(1.0, k2);
        t = k2 <= 1.0 ? none : s;
    }
    *skip = (float)std::min(s, 3.0e38);
    *tail = (float)std::min(t, (double)*skip);
}

// Adjoint pair sums of trajectory b over all node-block pairs: W nu slots into wpart
// [slots][B][n_pad], parameter sums into gpart [B][pairs][4] with r^2 in exponent units;
// *r2_phys receives the factor to physical r^2.
nf_status launch_adj_sym(nf_operator *op, const float *nu, const float *g, int B, int b, float *wpart, float *gpart,
                         float *r2_phys, cudaStream_t s) {
    const nf_kernel &k = op->kp;
    const float k2 = (k.s1 * k.s1) / (k.s2 * k.s2);
    const int m = op->form >= 2 ? op->form : 0;
    const double L2E = 1.4426950408889634;
    *r2_phys = (float)((m > 0 ? (double)k.s2 * k.s2 : (double)k.s1 * k.s1) / L2E);
    const bool cull = op->mf_cull && op->adj_pairs;
    const int blk = adj_block(op);
    const unsigned grid = (unsigned)(cull ? op->adj_live : adj_pair_count(op));
    const size_t smem = as_smem_bytes(blk);
    const SymNodes nd = sym_nodes(op);
    const int *pairs = cull ? op->adj_pairs : nullptr;
    const float per = mf_period(op);
    float tail, skip;
    adj_limits(op, &tail, &skip);
    auto go = [&](auto kernel) {
        return launch_dependent(kernel, dim3(grid), AS_THREADS, smem, s, true, nd, nu, g, B, b, k2, k.A1, k.A2, per, tail,
                                skip, wpart, gpart, pairs);
    };
    auto form = [&](auto r_tag, auto blk_tag) {
        constexpr int R = decltype(r_tag)::value, BLK = decltype(blk_tag)::value;
        switch (m) {
            case 2: return go(adj_sym_kernel<R, 2, BLK>);
            case 3: return go(adj_sym_kernel<R, 3, BLK>);
            case 4: return go(adj_sym_kernel<R, 4, BLK>);
            default: return go(adj_sym_kernel<R, 0, BLK>);
        }
    };
    if (blk == 512)
        NF_CUDA_TRY(op->adj_r == 8 ? form(CInt<8>{}, CInt<512>{}) : form(CInt<4>{}, CInt<512>{}));
    else
        NF_CUDA_TRY(op->adj_r == 8 ? form(CInt<8>{}, CInt<1024>{}) : form(CInt<4>{}, CInt<1024>{}));
    return NF_OK;
}

// Shape of the adjoint pair kernel -- rows per warp (4: two CTAs per SM; 8: one CTA per SM)
// and node block (1,024, or 512 where the 1,024-node block pairs fill fewer than eight waves
// of CTAs) -- chosen by timing the candidates on the operator's own node set: three launches
// each, each between its own events; the fastest of the last two counts.  The launches write
// the call's scratch buffers only (sized for 512-node blocks), before the call's own passes
// overwrite them.
nf_status adj_autotune(nf_operator *op, const float *nu, const float *g, int B, float *wpart, float *gpart,
                       cudaStream_t s) {
    if (op->adj_r) return NF_OK;
    // 512-node blocks only on the automatic schedule without culling: an explicit symmetric
    // schedule pins the block size, and the culled pass's live-pair lists use 1,024-node
    // blocks.  The choice is cached per (device, node count, kernel form, tune_class, whether 512 is
    // allowed), so operators on the same node set run the same shape (culled and unculled
    // gradients then agree bit for bit).
    static std::mutex mu;
    static std::map<std::tuple<int, int64_t, int, int, bool>, std::pair<int, int>> cache;
    const bool cull = op->mf_cull && op->adj_pairs;
    const int64_t nb1024 = op->n_pad / 1024, pairs1024 = nb1024 * (nb1024 + 1) / 2;
    const bool try512 = !cull && op->mf_sched == NF_MF_AUTO && pairs1024 < 8 * (int64_t)num_sms();
    const auto key = std::make_tuple(op->device, op->n_pad, op->form, op->tune_class, try512);
    {
        std::lock_guard<std::mutex> lock(mu);
        auto it = cache.find(key);
        if (it != cache.end()) {
            op->adj_r = it->second.first;
            op->adj_blk = it->second.second;
            return NF_OK;
        }
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    NF_CUDA_TRY(cudaEventCreate(&e0));
    cudaError_t ce = cudaEventCreate(&e1);
    if (ce != cudaSuccess) {
        cudaEventDestroy(e0);
        return cuda_fail(ce, "cudaEventCreate", __FILE__, __LINE__);
    }
    const int cand_r[4] = {4, 8, 4, 8}, cand_b[4] = {1024, 1024, 512, 512};
    float best = 3.4e38f;
    int best_r = 4, best_b = 1024;
    nf_status st = NF_OK;
    float r2 = 1.f;
    for (int c = 0; c < (try512 ? 4 : 2) && st == NF_OK; ++c) {
        op->adj_r = cand_r[c];
        op->adj_blk = cand_b[c];
        for (int rep = 0; rep < 3 && st == NF_OK; ++rep) {
            ce = cudaEventRecord(e0, s);
            if (ce == cudaSuccess) st = launch_adj_sym(op, nu, g, B, 0, wpart, gpart, &r2, s);
            if (st == NF_OK && ce == cudaSuccess) ce = cudaEventRecord(e1, s);
            if (st == NF_OK && ce == cudaSuccess) ce = cudaEventSynchronize(e1);
            float ms = 0.f;
            if (st == NF_OK && ce == cudaSuccess) ce = cudaEventElapsedTime(&ms, e0, e1);
            if (ce != cudaSuccess && st == NF_OK) st = cuda_fail(ce, "adjoint autotune", __FILE__, __LINE__);
            if (st == NF_OK && rep >= 1 && ms < best) {  // the first launch warms up
                best = ms;
                best_r = cand_r[c];
                best_b = cand_b[c];
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    op->adj_r = st == NF_OK ? best_r : 0;
    op->adj_blk = st == NF_OK ? best_b : 0;
    if (st == NF_OK) {
        std::lock_guard<std::mutex> lock(mu);
        cache[key] = {best_r, best_b};
    }
    return st;
}

}  // namespace nfi
