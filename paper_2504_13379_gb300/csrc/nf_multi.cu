// nf_multi.cu -- matrix-free nonlocal sums of several trajectories (§2.2, Eq. (2.9)).
//
// Each pair's weight is formed once for up to 16 trajectories.  A CTA takes 32 rows (4 per warp)
// against one column split: tiles of 512 columns are staged in shared memory, the trajectories'
// g transposed so that a column's NB values are contiguous; a lane takes two columns per step,
// forms the weights of its 8 pairs on packed FP32 pairs as in nf_sym.cu (expanded form, tile
// classes: skip and tail), and adds w g_b to 4 NB accumulators held as pairs of trajectories, so
// that the weight is the operand that consecutive packed FMAs share.  Row sums go to the split's
// partial slot; the stage kernel adds the splits in a fixed order.
//
// Bound: the FP32 FMA pipe, NB + 3 to 8 lane operations per ordered pair (NB + 10 with two
// exponentials per pair in the scalar kernel that served every width before, in groups of 16, 8,
// 4, 2, 1).  Per sum before / now, n = 15,000: 4 trajectories 159 / 119 us, 6 285 / 172, 8 210 /
// 172, 12 365 / 248; groups of exactly 16 stay on the scalar kernel.  Scalar accumulators in
// place of the pairs measured the same.
#include "nf_pairs.cuh"

#include <algorithm>

namespace nfi {

constexpr int MM_THREADS = 256, MM_WARPS = MM_THREADS / 32, MM_R = 4, MM_TJ = 512;
constexpr int MM_ROWS = MM_WARPS * MM_R;
// Threshold of the expanded form, half of the symmetric kernels'.  Geometric mean over 32 kernels and node
// sets (n = 500 to 15,000) of the relative L2 error against FP64: 0.78e-7 (0.80e-7 with their threshold,
// which is up to 4 % faster at 8,000 nodes; 0.77e-7 with half of this one, up to 4 % slower).  The
// scalar kernel that served every width before, on plain differences of the caller's
// coordinates, has 0.76e-7; with coordinates rounded to exponent units and exp2f's row factors
// this kernel had 1.20e-7.
constexpr float kMultiSpread = 2.0f;
// floats per column of the transposed g tile: strides of 4, 12 and 20 words spread eight adjacent
// columns' 16-byte reads over all banks
constexpr int mm_stride(int nb) { return nb == 8 ? 12 : (nb == 16 ? 20 : nb); }
constexpr size_t mm_smem_bytes(int nb) { return sizeof(float) * MM_TJ * (3 + (size_t)mm_stride(nb)); }

template <int NB, int M>
__global__ void __launch_bounds__(MM_THREADS, 2)
mf_multi_kernel(SymNodes nd, const float *g, int B, int b0, int64_t jchunk, float uu, float k2, float A1, float A2,
                float spread_max, float per, float lim_tail, float lim_skip, float *__restrict__ partial) {
    static_assert(NB % 4 == 0 && NB <= 16 && M >= 0 && M <= 4, "trajectories per group, form");
    constexpr int GS = mm_stride(NB), NT = MM_TJ / kTileCols;
    constexpr bool CW = M >= 2, HAS_TAIL = M != 1;
    extern __shared__ __align__(16) float mm_smem[];
    float *xs = mm_smem, *ys = xs + MM_TJ, *zs = ys + MM_TJ, *gs = zs + MM_TJ;  // gs: [MM_TJ][GS]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t n_pad = nd.n_pad;
    const int nv = min(NB, B - b0);  // trajectories b0 .. b0 + nv - 1 of the B
    const int64_t row0 = ((int64_t)blockIdx.x * MM_WARPS + warp) * MM_R;
    const int64_t j0 = (int64_t)blockIdx.y * jchunk, j1 = min(n_pad, j0 + jchunk);
    const float iper = per > 0.f ? 1.f / per : 0.f;
    const float4 c = __ldg(nd.pc + row0 / kPassRows), e = __ldg(nd.pe + row0 / kPassRows);
    const bool local = c.w == 1.f && e.w <= spread_max && !(per > 0.f);  // else differences, periodic ones per pair
    u64 xi[MM_R], yi[MM_R], zi[MM_R], h1[MM_R], h2[MM_R];
#pragma unroll
    for (int r = 0; r < MM_R; ++r) {
        float4 p = __ldg(nd.rg + row0 + r);
        float2 w = __ldg(nd.rw + row0 + r);
        if (!local) {
            p.x = __ldg(nd.xyz + row0 + r);
            p.y = __ldg(nd.xyz + n_pad + row0 + r);
            p.z = __ldg(nd.xyz + 2 * n_pad + row0 + r);
            w = make_float2(CW ? -(A1 / A2) : A1, -A2);
        }
        xi[r] = f2_dup(p.x);
        yi[r] = f2_dup(p.y);
        zi[r] = f2_dup(p.z);
        h1[r] = f2_dup(w.x);
        h2[r] = f2_dup(w.y);
    }
    const u64 uup = f2_dup(uu), nk2 = f2_dup(-k2), cxp = f2_dup(c.x), cyp = f2_dup(c.y), czp = f2_dup(c.z);
    const u64 ipp = f2_dup(iper), npp = f2_dup(-per), mgp = f2_dup(kRintMagic);
    u64 acc[MM_R][NB / 2];
#pragma unroll
    for (int r = 0; r < MM_R; ++r)
#pragma unroll
        for (int p = 0; p < NB / 2; ++p) acc[r][p] = 0ull;

    // pair weights from the exponent argument; CW: without the factor -A2 f2, M = 1: without A1 f1
    auto weight = [&](auto tail, int r, u64 arg) -> u64 {
        float s0, s1v;
        f2_unpack(arg, s0, s1v);
        if constexpr (M == 1) {
            return f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v));
        } else if constexpr (CW) {
            const u64 e2 = f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v));
            if constexpr (decltype(tail)::value) return e2;
            const u64 sq = f2_mul(e2, e2);
            const u64 e1 = M == 2 ? sq : (M == 3 ? f2_mul(sq, e2) : f2_mul(sq, sq));
            return f2_fma(e1, h1[r], e2);
        } else {
            const u64 w2 = f2_mul(f2_ex2(f2_mul(arg, nk2)), h2[r]);
            if constexpr (decltype(tail)::value) return w2;
            return f2_fma(f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v)), h1[r], w2);
        }
    };
    // w[r]: weights of the lane's columns q and q + 32 (adjacent lanes on adjacent columns, so that
    // their 16-byte reads of g hit all banks)
    auto add = [&](const u64 (&w)[MM_R], int q) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            u64 gp[NB / 2];
            const float4 *src = reinterpret_cast<const float4 *>(gs + (q + 32 * h) * GS);
#pragma unroll
            for (int p = 0; p < NB / 4; ++p) {
                const float4 v = src[p];
                gp[2 * p] = f2_lo(v);
                gp[2 * p + 1] = f2_hi(v);
            }
#pragma unroll
            for (int r = 0; r < MM_R; ++r) {
                float lo, hi;
                f2_unpack(w[r], lo, hi);
                const u64 wd = f2_dup(h ? hi : lo);
#pragma unroll
                for (int p = 0; p < NB / 2; ++p) acc[r][p] = f2_fma(wd, gp[p], acc[r][p]);
            }
        }
    };
    auto sweep_local = [&](auto tail, unsigned tiles) {
#pragma unroll 1
        for (; tiles; tiles &= tiles - 1) {
            const int t0 = (__ffs(tiles) - 1) * kTileCols + lane;
#pragma unroll
            for (int qq = 0; qq < kTileCols; qq += 64) {
                const int q = t0 + qq;
                const u64 xt = f2_sub(f2_pack(xs[q], xs[q + 32]), cxp), yt = f2_sub(f2_pack(ys[q], ys[q + 32]), cyp),
                          zt = f2_sub(f2_pack(zs[q], zs[q + 32]), czp);
                const u64 nj = f2_mul(f2_fma(zt, zt, f2_fma(yt, yt, f2_mul(xt, xt))), uup);
                u64 w[MM_R];
#pragma unroll
                for (int r = 0; r < MM_R; ++r)
                    w[r] = weight(tail, r, f2_fma(xi[r], xt, f2_fma(yi[r], yt, f2_fma(zi[r], zt, nj))));
                add(w, q);
            }
        }
    };
    auto sweep_diff = [&](auto wrap, unsigned tiles) {
#pragma unroll 1
        for (; tiles; tiles &= tiles - 1) {
            const int t0 = (__ffs(tiles) - 1) * kTileCols + lane;
#pragma unroll 1
            for (int q = t0; q < t0 + kTileCols; q += 64) {
                const u64 xj = f2_pack(xs[q], xs[q + 32]), yj = f2_pack(ys[q], ys[q + 32]), zj = f2_pack(zs[q], zs[q + 32]);
                u64 w[MM_R];
#pragma unroll
                for (int r = 0; r < MM_R; ++r) {
                    u64 dx = f2_sub(xi[r], xj), dy = f2_sub(yi[r], yj);
                    const u64 dz = f2_sub(zi[r], zj);
                    if constexpr (decltype(wrap)::value) {
                        dx = f2_wrap(dx, ipp, npp, mgp);
                        dy = f2_wrap(dy, ipp, npp, mgp);
                    }
                    w[r] = weight(PerTag<false>{}, r, f2_mul(f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx))), uup));
                }
                add(w, q);
            }
        }
    };

    pdl_wait();
    pdl_trigger();
    for (int64_t jt = j0; jt < j1; jt += MM_TJ) {
        if (jt > j0) __syncthreads();  // the previous tile is still being read
        bool bad = false;
#pragma unroll
        for (int t = 0; t < MM_TJ / MM_THREADS; ++t) {
            const int k = tid + t * MM_THREADS;
            const int64_t j = jt + k;
            const bool in = j < j1;
            // The rates' loads first, and as ld_written: with plain loads, or the coordinates first, the sweeps
            // below came out slower (n = 15,000: 8 trajectories 186 us, plain loads first 184, ld_written
            // second 176, both 172; 12 trajectories 254, 248, 254, 248).
            float v[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) v[b] = in && b < nv ? ld_written(g + (int64_t)(b0 + b) * n_pad + j) : 0.f;
            xs[k] = in ? __ldg(nd.xyz + j) : 0.f;
            ys[k] = in ? __ldg(nd.xyz + n_pad + j) : 0.f;
            zs[k] = in ? __ldg(nd.xyz + 2 * n_pad + j) : 0.f;
#pragma unroll
            for (int b = 0; b < NB; ++b) bad |= !(0.f * v[b] == 0.f);  // non-finite
#pragma unroll
            for (int b = 0; b < NB; b += 4)
                *reinterpret_cast<float4 *>(gs + k * GS + b) = make_float4(v[b], v[b + 1], v[b + 2], v[b + 3]);
        }
        bad = __syncthreads_or(bad);
        // classes of the tiles with real nodes, one lane per tile; a non-finite g sweeps all in full
        float d2 = 3.4e38f;
        const int64_t tj = jt / kTileCols + lane;
        const bool real = lane < NT && tj * kTileCols < nd.n && jt + lane * kTileCols < j1;
        if (real) d2 = bad ? 0.f : box_d2(c, e, __ldg(nd.tc + tj), __ldg(nd.te + tj), per, iper);
        const unsigned live_t = __ballot_sync(0xffffffffu, real && d2 <= lim_skip);
        const unsigned full_t = HAS_TAIL && local ? live_t & __ballot_sync(0xffffffffu, d2 <= lim_tail) : live_t;
        if (local) {
            if constexpr (HAS_TAIL) sweep_local(PerTag<true>{}, live_t & ~full_t);
            sweep_local(PerTag<false>{}, full_t);
        } else if (per > 0.f) {
            sweep_diff(PerTag<true>{}, full_t);
        } else {
            sweep_diff(PerTag<false>{}, full_t);
        }
    }
    constexpr int NR = NB <= 4 ? 4 : (NB <= 8 ? 8 : 16);  // a power of two for the butterfly
#pragma unroll
    for (int r = 0; r < MM_R; ++r) {
        float v[NR];
#pragma unroll
        for (int p = 0; p < NR / 2; ++p) {
            if (p < NB / 2) {
                f2_unpack(acc[r][p < NB / 2 ? p : 0], v[2 * p], v[2 * p + 1]);
            } else {
                v[2 * p] = v[2 * p + 1] = 0.f;
            }
        }
        int b;
        float tot = warp_reduce_rows<NR>(v, lane, b);
        if constexpr (M > 0) {  // the row factor left out of the weights
            const float2 w = __ldg(nd.rw + row0 + r);
            tot *= CW ? (local ? w.y : -A2) : (local ? w.x : A1);
        }
        if ((lane & (32 / NR - 1)) == 0 && b < nv)
            partial[((int64_t)blockIdx.y * B + b0 + b) * n_pad + row0 + r] = tot;
    }
}

template <int NB>
static cudaError_t multi_attrs() {
    const int smem = (int)mm_smem_bytes(NB);
    cudaError_t e = cudaFuncSetAttribute(mf_multi_kernel<NB, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mf_multi_kernel<NB, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mf_multi_kernel<NB, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mf_multi_kernel<NB, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mf_multi_kernel<NB, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e;
}
nf_status multi_init_attrs() {
    NF_CUDA_TRY(multi_attrs<4>());
    NF_CUDA_TRY(multi_attrs<8>());
    NF_CUDA_TRY(multi_attrs<12>());
    NF_CUDA_TRY(multi_attrs<16>());
    return NF_OK;
}

SplitPlan multi_plan(const nf_operator *op) { return plan_splits(op->n_pad, MM_ROWS, MM_TJ, 2); }

// Trajectories b0 .. B - 1 (at most 16), the width rounded up to 4, 8, 12 or 16.
nf_status launch_multi(nf_operator *op, int B, int b0, cudaStream_t s) {
    const nf_kernel &k = op->kp;
    const ExactUnits &eu = op->eu;
    const SplitPlan pl = multi_plan(op);
    const int group = B - b0;
    // rows within n_i of kMultiSpread, in units of the narrower Gaussian evaluated
    const float spread = kMultiSpread * (op->form >= 2 ? eu.k2 : (op->form == 0 ? 1.f / std::max(1.f, eu.k2) : 1.f));
    float tail, skip;
    class_limits(op, &tail, &skip);
    tail /= eu.uu;  // boxes are in stored units
    skip /= eu.uu;
    const dim3 grid((unsigned)ceil_div(op->n, MM_ROWS), (unsigned)pl.splits, 1);
    auto form = [&](auto nb_tag) {
        constexpr int NB = decltype(nb_tag)::value;
        auto go = [&](auto kernel) {
            return launch_dependent(kernel, grid, MM_THREADS, mm_smem_bytes(NB), s, !op->profile, exact_nodes(op),
                                    (const float *)op->g, B, b0, pl.jchunk, eu.uu, eu.k2, k.A1, k.A2, spread, eu.per,
                                    tail, skip, op->partial);
        };
        switch (op->form) {
            case 1: return go(mf_multi_kernel<NB, 1>);
            case 2: return go(mf_multi_kernel<NB, 2>);
            case 3: return go(mf_multi_kernel<NB, 3>);
            case 4: return go(mf_multi_kernel<NB, 4>);
            default: return go(mf_multi_kernel<NB, 0>);
        }
    };
    if (group <= 4)
        NF_CUDA_TRY(form(std::integral_constant<int, 4>{}));
    else if (group <= 8)
        NF_CUDA_TRY(form(std::integral_constant<int, 8>{}));
    else if (group <= 12)
        NF_CUDA_TRY(form(std::integral_constant<int, 12>{}));
    else
        NF_CUDA_TRY(form(std::integral_constant<int, 16>{}));
    return NF_OK;
}

}  // namespace nfi
