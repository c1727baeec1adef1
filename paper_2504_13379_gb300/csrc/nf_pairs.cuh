// nf_pairs.cuh -- what the matrix-free pair kernels share: packed FP32 arithmetic, block-pair
// enumeration, warp reductions, and the operator's node data in Hilbert order.
#pragma once

#include "nf_internal.cuh"

namespace nfi {

// ------------------------------------------------------------------ packed FP32 pairs
typedef unsigned long long u64;
__device__ __forceinline__ u64 f2_sub(u64 a, u64 b) {
    u64 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 f2_add(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 f2_mul(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 f2_fma(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 f2_pack(float lo, float hi) {
    u64 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ void f2_unpack(u64 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ u64 f2_ex2(u64 a) {
    float lo, hi;
    f2_unpack(a, lo, hi);
    return f2_pack(ex2_sfu(lo), ex2_sfu(hi));
}
__device__ __forceinline__ float f2_fold(u64 x) {
    float lo, hi;
    f2_unpack(x, lo, hi);
    return lo + hi;
}
// The SFU's ex2 is low by 3e-8 on average over the exponents of a planar Gaussian (measured over 2^20
// arguments; rms 5.5e-8), its powers e2^M by about twice that.
constexpr float kEx2Low = 3.1e-8f;

// s 2^x (1 + up) for -100 < x <= 0, rounded about once: 2^r - 1 for the fraction r of x, |r| <= 1/2, by its
// Taylor series in r ln 2 to degree 8 (remainder below 4e-10), added to s in one FMA.  For the
// row factors of the expanded forms: their error is common to a row's whole sum, and the
// difference of the two Gaussians' sums magnifies it.  exp2f (two units in the last place) and the
// products around it made up most of the 1e-7 that sums of several trajectories were off.
__device__ __forceinline__ float scale_pow2(float s, float x, float up) {
    const float k = rintf(x), r = x - k;
    float p = 1.3215487e-6f;              // (ln 2)^8 / 8!
    p = fmaf(p, r, 1.5252734e-5f);        // (ln 2)^7 / 7!
    p = fmaf(p, r, 1.5403530e-4f);        // ...
    p = fmaf(p, r, 1.3333558e-3f);
    p = fmaf(p, r, 9.6181291e-3f);
    p = fmaf(p, r, 5.5504109e-2f);
    p = fmaf(p, r, 2.4022651e-1f);
    p = fmaf(p, r, 6.9314718e-1f);        // ln 2
    return fmaf(s, fmaf(p, r, up), s) * __int_as_float((127 + (int)k) << 23);
}
__device__ __forceinline__ u64 f2_dup(float v) { return f2_pack(v, v); }
__device__ __forceinline__ u64 f2_lo(float4 v) { return f2_pack(v.x, v.y); }
__device__ __forceinline__ u64 f2_hi(float4 v) { return f2_pack(v.z, v.w); }

// Nearest image of a packed pair of coordinate differences (see wrap1): ip = 1/p, np = -p,
// mg = the rounding constant, each in both halves.
__device__ __forceinline__ u64 f2_wrap(u64 d, u64 ip, u64 np, u64 mg) {
    return f2_fma(f2_sub(f2_fma(d, ip, mg), mg), np, d);
}

// 16-byte asynchronous copy global -> shared (both addresses 16-byte aligned).
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ------------------------------------------------------------------ thread-block clusters
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// This CTA's shared variable `p` as cluster CTA `rank` holds it.
__device__ __forceinline__ float ld_cluster(const float *p, uint32_t rank) {
    float v;
    asm volatile("{\n\t.reg .u32 a;\n\tmapa.shared::cluster.u32 a, %1, %2;\n\tld.shared::cluster.f32 %0, [a];\n\t}"
                 : "=f"(v)
                 : "r"(smem_u32(p)), "r"(rank)
                 : "memory");
    return v;
}

// Block pair of CTA t over node blocks, enumerated as (0,0), (0,1), (1,1), (0,2), ...  An FP32
// root, then integer corrections: the FP64 root this replaces cost every CTA 1.6 us of the SM's
// FP64 pipe (two lanes per clock), 5 % of a sum at n = 100,000 and 12 % at 20,000.
__device__ __forceinline__ void sym_pair(int64_t t, int &I, int &J) {
    int64_t j = (int64_t)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    while (j * (j + 1) / 2 > t) --j;
    while ((j + 1) * (j + 2) / 2 <= t) ++j;
    J = (int)j;
    I = (int)(t - j * (j + 1) / 2);
}

// Sum R per-lane values over the warp.  Transposed butterfly: at each of the first log2(R)
// steps a lane keeps half of its rows and adds its partner's copy of them (R - 1 shuffles
// in total), then plain xor steps finish.  Every lane returns the total of row `row`.
template <int R>
__device__ __forceinline__ float warp_reduce_rows(float (&v)[R], int lane, int &row) {
    int base = 0;
    int cnt = R;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        if (cnt > 1) {
            const int h = cnt >> 1;
            const bool upper = (lane & off) != 0;
#pragma unroll
            for (int k = 0; k < R / 2; ++k) {
                if (k < h) {
                    const float send = upper ? v[k] : v[k + h];
                    const float keep = upper ? v[k + h] : v[k];
                    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                }
            }
            if (upper) base += h;
            cnt = h;
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
        }
    }
    row = base;
    return v[0];
}

// ------------------------------------------------------------------ node data
// A matrix-free operator keeps its nodes in Hilbert order (nf_operator::perm), in the units of
// its kernel's exponents.  Node groups: passes of kPassRows consecutive nodes (the rows a warp
// holds in registers) and tiles of kTileCols (the columns it sweeps in one step); each has the
// box of its nodes (centre and half extents), from which a warp bounds the distance between
// a pass and a tile.  SymNodes points at the data that depend on the nodes and the kernel only.
constexpr int kPassRows = 8;
constexpr int kTileCols = 128;

// The expanded form's threshold: rows within 2 s / sqrt(log2 e) of their centre, s the smaller width
// of the Gaussians evaluated.  The rounding of r^2 = n_i + s_ij for the pairs that carry weight
// stays of order eps * n_i (below 3e-7 relative in the exponential at n_i = 4), and 2^(-s_ij) and
// the row factor 2^(-n_i) stay in range in either Gaussian: with s1 = 10 s2 a threshold in units of s1
// alone let n_i reach 400 in units of s2, infinity times zero.  The expanded form saves three of the
// difference form's six exponent operations per pair.  Measured on GB300 against a threshold
// of 1: the same error against the FP64 oracle (1.4e-7 relative L2 on the precision torus,
// 9.3e-7 on the periodic square), 2.37 vs 2.63 ms on the periodic square at n = 131,072,
// 0.157 vs 0.175 ms on the 20,000-node sphere.
constexpr float kSymLocalSpread = 4.0f;

struct SymNodes {
    const float *xyz;    // 3 x n_pad, exponent units; padding repeats the last node
    const float4 *rg;    // n_pad: row operands mx, my, mz and n_i (see sym_static_kernel)
    const float2 *rw;    // n_pad: row factors
    const float4 *pc;    // n_pad / kPassRows: pass centre, form
    const float4 *pe;    // n_pad / kPassRows: half extents of the pass's box; w: its largest n_i
    const float4 *tc;    // n_pad / kTileCols: tile box centre
    const float4 *te;    // n_pad / kTileCols: tile box half extents
    int64_t n, n_pad;
};
inline SymNodes sym_nodes(const nf_operator *op) {
    return SymNodes{op->xyz, op->rg, op->rw, op->pc, op->pe, op->tc, op->te, op->n, op->n_pad};
}

// The exact set (nf_operator::xyz2): coordinates times a power of two, so differences of the caller's
// coordinates are rounded once; the exponent of a squared distance r2 is uu r2 (ExactUnits), one
// multiplication per column of a pass, or per pair in the difference forms.
inline SymNodes exact_nodes(const nf_operator *op) {
    return SymNodes{op->xyz2, op->rg2, op->rw2, op->pc2, op->pe2, op->tc2, op->te2, op->n, op->n_pad};
}
// Lower bound of the squared distance between the nodes of two boxes (centre c, half extents
// h); per > 0: nearest images in x and y.  A box with a non-finite node has infinite half
// extents, which gives 0.
__device__ __forceinline__ float box_d2(float4 ca, float4 ha, float4 cb, float4 hb, float per, float iper) {
    float dx = ca.x - cb.x, dy = ca.y - cb.y;
    const float dz = ca.z - cb.z;
    if (per > 0.f) {
        dx -= per * rintf(dx * iper);
        dy -= per * rintf(dy * iper);
    }
    const float gx = fmaxf(0.f, fabsf(dx) - (ha.x + hb.x)), gy = fmaxf(0.f, fabsf(dy) - (ha.y + hb.y)),
                gz = fmaxf(0.f, fabsf(dz) - (ha.z + hb.z));
    return gx * gx + gy * gy + gz * gz;
}

}  // namespace nfi
