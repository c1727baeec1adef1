// nf_sym.cu -- node data in Hilbert order and the symmetric single-trajectory pair kernel of the
// matrix-free nonlocal sum (§2.2, Eq. (2.9)).
//
// w(x_i, x_j) = w(x_j, x_i), so every unordered pair is evaluated once and feeds both sums:
// I_i += w_ij g_j and I_j += w_ij g_i.  Nodes are kept in Hilbert order and cut into blocks of
// BLK nodes (1,024, or 512 where the operator's autotuner measured the smaller blocks faster);
// one CTA takes a block pair (I <= J): it stages block J's coordinates and g and block I's row
// operands in shared memory, its warps sweep block I eight rows at a time against tiles of 128
// columns, accumulate the row sums in registers and the column sums per warp in shared memory.
// Row sums of pair (I, J) go to partial slot J, column sums to slot I; a diagonal pair (I = I)
// sweeps all ordered pairs of the block and writes rows only.  Every (slot, node) entry is
// written exactly once, and the stage kernel adds the n_pad / BLK slots in a fixed order, so
// results are deterministic.
//
// Tile classes.  Before it sweeps a pass of eight rows, a warp bounds the distance from the
// rows' box to each tile's box (one lane per tile) and sorts the tiles into three classes:
//   skip   the exponentials of every pair flush to exactly 0 in FP32 (ex2.approx.ftz below
//          2^-126): nothing is added to any sum;
//   tail   (width ratio M >= 2) the narrow Gaussian is below half an ulp of the wide one in
//          every pair: |c_i| e1 < 2^-26 e2, so the FP32 sum e2 + c_i e1 is e2 itself; (general
//          form, s1 <= s2) e1 is exactly 0.  One exponential and five FMA-pipe operations per
//          pair instead of eight;
//   full   everything else.
// The classes change which operations run, not what they would have added: a swept tile gives
// bit for bit the sums of the full form.  Blocks that hold a non-finite g sweep every tile in
// full, so NaN and infinity spread as in the plain sum.
//
// Bound: the FP32 FMA pipe at the rate it reaches with three different 64-bit operands (88 of its
// 128 lanes per clock and SM).  A loop of full tiles alone runs 11.0 unordered pairs per clock
// and SM, of tail tiles alone 14.4; scalar FMAs, pairs of rows instead of columns, and 4 or 16
// rows per pass all measured slower.  On GB300, RK4 step before and after the classes: torus
// n = 100,000 5.98 -> 4.49 ms (1.48 -> 1.12 ms per sum), periodic square n = 131,072 with
// Gauss(1/40) 9.3 -> 0.82 ms (97 % of the tile visits are skipped; half of the rest is forcing).
#include "nf_pairs.cuh"

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>

namespace nfi {

constexpr int MS_THREADS = 256;
constexpr int MS_WARPS = MS_THREADS / 32;
// shared memory (4-byte words): columns x, y, z, g (4 BLK); row operands, factors and weights
// (7 BLK); pass centres and half extents (BLK); tile boxes (BLK / 16); per-warp column sums
// (MS_WARPS BLK)
constexpr size_t ms_smem_bytes(int blk) {
    return sizeof(float) * ((4 + 7 + 1 + MS_WARPS) * (size_t)blk + blk / 16);
}

// ------------------------------------------------------------------ kernel forms
// Integer width ratio m = s2^2 / s1^2 in {2, 3, 4} (to FP32 rounding of the k2 the kernel
// receives), else 0: selects the one-exponential form.
static int width_ratio(const nf_kernel &k) {
    const float k2 = (k.s1 * k.s1) / (k.s2 * k.s2);
    for (int m = 2; m <= 4; ++m)
        if (std::fabs((double)m * (double)k2 - 1.0) <= 4.0 * (double)FLT_EPSILON) return m;
    return 0;
}

// Pair form of a kernel: 1 for a single Gaussian (A2 = 0); the width ratio 2-4, whose kernels
// combine the two Gaussians through the ratio -A1 f1 / (A2 f2) per row, which stays finite
// while |A1 / A2| <= 2^100; else 0, the general form.
int mf_form(const nf_kernel &k) {
    if (k.A2 == 0.f) return 1;
    const int m = width_ratio(k);
    if (m >= 2 && !(std::fabs((double)k.A1) <= 0x1p100 * std::fabs((double)k.A2))) return 0;
    return m;
}

// Coordinates are stored times sqrt(log2 e) / s1, so that squared distances are exponents of 2
// of the narrow Gaussian; with a width ratio M >= 2 in units of s2 (times s1 / s2), the exponents
// of the wide Gaussian, from which the narrow one follows by powers.
float mf_unit(const nf_operator *op) {
    const nf_kernel &k = op->kp;
    const float u = std::sqrt(1.4426950408889634f) / k.s1;
    return op->form >= 2 ? u * std::sqrt((k.s1 * k.s1) / (k.s2 * k.s2)) : u;
}

// The kernel's period in the units of the stored coordinates; 0 for the Euclidean distance.
float mf_period(const nf_operator *op) { return op->kp.period > 0.f ? op->kp.period * mf_unit(op) : 0.f; }

// The exact set's units.  uu and k2 are rounded once each, k2 so that the product uu k2 is the second
// Gaussian's exponent to rounding.
static ExactUnits exact_units(const nf_operator *op) {
    const nf_kernel &k = op->kp;
    const double L2E = 1.4426950408889634074, s1 = k.s1, s2 = k.s2;
    const double e1 = L2E / (s1 * s1), e2 = L2E / (s2 * s2), e = op->form >= 2 ? e2 : e1;
    const double p = std::min(126.0, std::max(-126.0, std::round(0.5 * std::log2(e))));
    ExactUnits u;
    u.unit = (float)std::exp2(p);
    u.uu = (float)(e * std::exp2(-2.0 * p));
    u.k2 = (float)(e2 * std::exp2(-2.0 * p) / (double)u.uu);
    if (op->form >= 2) u.k2 = (float)((s1 * s1) / (s2 * s2));
    u.per = k.period > 0.f ? k.period * u.unit : 0.f;
    return u;
}

// Squared distances (exponents) beyond which a pair of nodes takes the tail form, and beyond
// which it contributes exactly 0.
//   skip: the wider exponential evaluated has exponent > 126 with the expanded form's row part
//         n_i <= 4 already taken out of it; one more unit for the rounding of the box bound.
//   tail: M >= 2: |c_i| e1 / e2 = |A1 / A2| 2^(-(M - 1) r^2) < 2^-26 (c_i carries the row
//         factors), half a unit for rounding; general form with s1 <= s2: e1 flushes as above;
//         one Gaussian: no tail.
void class_limits(const nf_operator *op, float *tail, float *skip) {
    const nf_kernel &k = op->kp;
    const double k2 = ((double)k.s1 * k.s1) / ((double)k.s2 * k.s2);
    const double none = 126.0 + 4.0 + 1.0;
    const double inf = 3.0e38;
    double t = inf, s = none;
    if (op->form >= 2) {
        const double lr = k.A1 != 0.f ? std::log2(std::fabs((double)k.A1 / (double)k.A2)) : -26.0;
        t = std::max(0.0, (26.0 + lr) / (op->form - 1)) + 0.5;
    } else if (op->form == 0) {
        if (k2 <= 1.0) t = none;
        s = none / std::min(1.0, k2);
    }
    *skip = (float)std::min(s, inf);
    *tail = (float)std::min(t, (double)*skip);
}

// ------------------------------------------------------------------ node data
// Box of one group of consecutive nodes, over its real ones: centre and half extents.  The
// half extents are rounded up; a non-finite coordinate makes them infinite (see box_d2).
struct Box {
    float lo[3], hi[3];
    bool bad;
    __device__ __forceinline__ Box() : bad(false) {
#pragma unroll
        for (int d = 0; d < 3; ++d) lo[d] = 3.4e38f, hi[d] = -3.4e38f;
    }
    __device__ __forceinline__ void add(const float *x, int64_t n_pad, int64_t p) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float v = x[d * n_pad + p];
            bad |= !isfinite(v);
            lo[d] = fminf(lo[d], v);
            hi[d] = fmaxf(hi[d], v);
        }
    }
    __device__ __forceinline__ float4 centre() const {
        return make_float4(0.5f * (lo[0] + hi[0]), 0.5f * (lo[1] + hi[1]), 0.5f * (lo[2] + hi[2]), 0.f);
    }
    __device__ __forceinline__ float4 half(float4 c) const {
        const float up = 1.f + 1e-6f, inf = __int_as_float(0x7f800000);
        if (bad) return make_float4(inf, inf, inf, 0.f);
        return make_float4(fmaxf(hi[0] - c.x, c.x - lo[0]) * up, fmaxf(hi[1] - c.y, c.y - lo[1]) * up,
                           fmaxf(hi[2] - c.z, c.z - lo[2]) * up, 0.f);
    }
};

// One thread per pass of kPassRows nodes: centre of the pass, its form and box, and the row
// operands.  uu: exponent per squared stored unit (1: the scaled set, else ExactUnits).  Forms: 1
// expanded about the centre c, uu r^2 = n_i + s_ij, s_ij = n_j - 2 uu (x_i - c).(x_j - c) (rows hold
// -2 uu (x_i - c)), for rows within spread_max of c; 0 differences (rows
// x_i); periodic kernels: 2 differences of centred coordinates (rows x_i - c), and in forms 1
// and 2 the columns taken at their nearest image of c.  That image is the pair's nearest image
// unless the column lies within e (the rows' distance from c) of c's antipodal lines; such a
// pair is at least L/2 - e apart in both images, and when the wider Gaussian's exponent there
// exceeds 160 (log2 units) both images give exactly 0 (ex2 flushes below 2^-126).  Otherwise
// form 3: centred differences reduced to their nearest image pair by pair.  f1, f2 are the row
// factors 2^(-n_i) of e1 and e2 (1 outside form 1); rw holds (c_i, -A2 f2) for width ratios
// M >= 2, with c_i = -(A1 f1) / (A2 f2), else (A1 f1, -A2 f2).
struct NodeSet {  // one of the operator's two sets (blockIdx.y)
    const float *xyz;
    float uu, k2, per, spread_max;
    float4 *rg;
    float2 *rw;
    float4 *pc, *pe, *tc, *te;
};
struct NodeSets {
    NodeSet s[2];
};
__global__ void sym_static_kernel(const __grid_constant__ NodeSets sets, int64_t n_pad, int M, float A1, float A2,
                                  int *__restrict__ count) {
    const NodeSet &ns = sets.s[blockIdx.y];
    const float *xyz = ns.xyz;
    const float uu = ns.uu, k2 = ns.k2, per = ns.per, spread_max = ns.spread_max;
    float4 *rg = ns.rg, *pc = ns.pc, *pe = ns.pe;
    float2 *rw = ns.rw;
    const int64_t ps = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (ps >= n_pad / kPassRows) return;
    const int64_t r0 = ps * kPassRows;
    Box bx;
    for (int r = 0; r < kPassRows; ++r) bx.add(xyz, n_pad, r0 + r);
    const float4 c = bx.centre();
    float spread = 0.f;
    for (int r = 0; r < kPassRows; ++r) {
        const float dx = xyz[r0 + r] - c.x, dy = xyz[n_pad + r0 + r] - c.y, dz = xyz[2 * n_pad + r0 + r] - c.z;
        spread = fmaxf(spread, dx * dx + dy * dy + dz * dz);
    }
    const float far = sqrtf(spread);  // the rows' largest distance from the centre
    spread *= uu;                     // as an exponent
    bool local = spread <= spread_max;
    int form = local ? 1 : 0;
    if (per > 0.f) {
        const float wide = M > 0 ? 1.f : fminf(1.f, k2);  // exponent of the wider Gaussian per unit of r^2
        const float m = 0.5f * per - far;
        if (m > 0.f && wide * uu * m * m >= 160.f) {
            form = local ? 1 : 2;
        } else {
            form = 3;
            local = false;
        }
    }
    if (blockIdx.y == 0) {  // expanded passes of the scaled set
        const unsigned act = __activemask(), loc = __ballot_sync(act, form == 1);
        if ((int)(threadIdx.x & 31) == __ffs(act) - 1) atomicAdd(count, __popc(loc));
    }
    pc[ps] = make_float4(c.x, c.y, c.z, (float)form);
    float4 he = bx.half(c);
    he.w = spread;
    pe[ps] = he;
    const bool centred = form >= 2;
    for (int r = 0; r < kPassRows; ++r) {
        const int64_t k = r0 + r;
        const float px = xyz[k], py = xyz[n_pad + k], pz = xyz[2 * n_pad + k];
        const float m2 = -2.f * uu;
        const float x = local ? m2 * (px - c.x) : (centred ? px - c.x : px);
        const float y = local ? m2 * (py - c.y) : (centred ? py - c.y : py);
        const float z = local ? m2 * (pz - c.z) : pz;  // z never wraps
        const float ni = local ? 0.25f / uu * (x * x + y * y + z * z) : 0.f;
        rg[k] = make_float4(x, y, z, ni);
        rw[k] = make_float2(M >= 2 ? scale_pow2(-(A1 / A2), -(float)(M - 1) * ni, kEx2Low) : scale_pow2(A1, -ni, kEx2Low),
                            scale_pow2(-A2, M > 0 ? -ni : -k2 * ni, kEx2Low));
    }
}

// One warp per tile of kTileCols nodes: its box.
__global__ void sym_tiles_kernel(const __grid_constant__ NodeSets sets, int64_t n_pad) {
    const float *xyz = sets.s[blockIdx.y].xyz;
    float4 *tc = sets.s[blockIdx.y].tc, *te = sets.s[blockIdx.y].te;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (t >= n_pad / kTileCols) return;
    Box bx;
    for (int k = lane; k < kTileCols; k += 32) bx.add(xyz, n_pad, t * kTileCols + k);
    bx.bad = __any_sync(0xffffffffu, bx.bad);
    for (int o = 16; o > 0; o >>= 1)
        for (int d = 0; d < 3; ++d) {
            bx.lo[d] = fminf(bx.lo[d], __shfl_xor_sync(0xffffffffu, bx.lo[d], o));
            bx.hi[d] = fmaxf(bx.hi[d], __shfl_xor_sync(0xffffffffu, bx.hi[d], o));
        }
    if (lane == 0) {
        const float4 c = bx.centre();
        tc[t] = c;
        te[t] = bx.half(c);
    }
}

// Node order: position along a Hilbert curve through the 1024^3 cubic cells of the bounding box,
// ties by index, so that consecutive nodes are near each other; without the jumps of a Z-order
// curve the boxes of 128-node tiles are smaller (torus, n = 100,000: 12 % of the tile visits in
// the full class and 15 % skipped, against 15 % and 11 % in Z-order).  Keys (code << 32 |
// index) are unique; a bitonic network over the next power of two sorts them.  Padding keeps
// its place.

// Bounding box of the n nodes (one block): box = {lo x, lo y, lo z, hi x, hi y, hi z}.
__global__ void row_bbox_kernel(const float *__restrict__ x, int64_t n, float *__restrict__ box, int *__restrict__ count) {
    if (threadIdx.x == 0) *count = 0;
    __shared__ float red[6][32];
    float v[6] = {3.4e38f, 3.4e38f, 3.4e38f, -3.4e38f, -3.4e38f, -3.4e38f};
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x)
        for (int d = 0; d < 3; ++d) {
            const float c = x[3 * j + d];
            v[d] = fminf(v[d], c);
            v[3 + d] = fmaxf(v[3 + d], c);
        }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1)
        for (int d = 0; d < 3; ++d) {
            v[d] = fminf(v[d], __shfl_xor_sync(0xffffffffu, v[d], o));
            v[3 + d] = fmaxf(v[3 + d], __shfl_xor_sync(0xffffffffu, v[3 + d], o));
        }
    if (lane == 0)
        for (int d = 0; d < 6; ++d) red[d][warp] = v[d];
    __syncthreads();
    if (threadIdx.x < 6) {
        const int d = threadIdx.x;
        float a = red[d][0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) a = d < 3 ? fminf(a, red[d][w]) : fmaxf(a, red[d][w]);
        box[d] = a;
    }
}

// Hilbert code of a cell (10 bits per axis) by Skilling's transform ("Programming the Hilbert
// curve", 2004): axes to the transposed index, whose bits are then interleaved.
__device__ __forceinline__ uint32_t hilbert_code(uint32_t x, uint32_t y, uint32_t z) {
    uint32_t v[3] = {x, y, z};
    for (uint32_t q = 512; q > 1; q >>= 1) {
        const uint32_t p = q - 1;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            if (v[i] & q) {
                v[0] ^= p;
            } else {
                const uint32_t t = (v[0] ^ v[i]) & p;
                v[0] ^= t;
                v[i] ^= t;
            }
        }
    }
    v[1] ^= v[0];
    v[2] ^= v[1];
    uint32_t t = 0;
    for (uint32_t q = 512; q > 1; q >>= 1)
        if (v[2] & q) t ^= q - 1;
    uint32_t code = 0;
    for (int b = 9; b >= 0; --b)
#pragma unroll
        for (int i = 0; i < 3; ++i) code = (code << 1) | (((v[i] ^ t) >> b) & 1u);
    return code;
}

__global__ void row_key_kernel(const float *__restrict__ x, int64_t n, int64_t m, const float *__restrict__ box,
                               unsigned long long *__restrict__ keys) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    if (j >= n) {
        keys[j] = ~0ull;
        return;
    }
    const float ext = fmaxf(box[3] - box[0], fmaxf(box[4] - box[1], box[5] - box[2]));
    uint32_t c[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float t = ext > 0.f ? (x[3 * j + d] - box[d]) / ext : 0.f;
        c[d] = (uint32_t)fminf(fmaxf(t * 1024.f, 0.f), 1023.f);
    }
    keys[j] = ((unsigned long long)hilbert_code(c[0], c[1], c[2]) << 32) | (unsigned long long)j;
}

// One compare-exchange step of the bitonic network (block size kk, partner distance jj).
__global__ void row_bitonic_kernel(unsigned long long *__restrict__ keys, int64_t m, int64_t jj, int64_t kk) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const int64_t l = i ^ jj;
    if (l <= i) return;
    const unsigned long long a = keys[i], b = keys[l];
    const bool ascending = (i & kk) == 0;
    if ((a > b) == ascending) {
        keys[i] = b;
        keys[l] = a;
    }
}

// All steps of the network that stay within blocks of SORT_BLK keys, in shared memory: block
// sizes kk0 .. kk1, partner distances below SORT_BLK (a sort of 131,072 keys takes 28 launches
// instead of 153).
constexpr int SORT_BLK = 2048;
__global__ void __launch_bounds__(SORT_BLK / 2)
row_bitonic_local_kernel(unsigned long long *__restrict__ keys, int blk, int64_t kk0, int64_t kk1) {
    __shared__ unsigned long long k[SORT_BLK];
    const int64_t base = (int64_t)blockIdx.x * blk;
    for (int i = threadIdx.x; i < blk; i += blockDim.x) k[i] = keys[base + i];
    __syncthreads();
    for (int64_t kk = kk0; kk <= kk1; kk <<= 1)
        for (int jj = (int)min(kk, (int64_t)blk) >> 1; jj > 0; jj >>= 1) {
            for (int t = threadIdx.x; t < blk / 2; t += blockDim.x) {
                const int i = (t / jj) * 2 * jj + t % jj, l = i + jj;
                const unsigned long long a = k[i], b = k[l];
                if ((a > b) == (((base + i) & kk) == 0)) {
                    k[i] = b;
                    k[l] = a;
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < blk; i += blockDim.x) keys[base + i] = k[i];
}

// Node arrays in Hilbert order.  Padding repeats the last node (so that it widens no box) with
// q = 0 (so that it contributes nothing).
__global__ void pack_sorted_kernel(const float *__restrict__ x, const float *__restrict__ q,
                                   const unsigned long long *__restrict__ keys, int64_t n, int64_t n_pad, float unit,
                                   float unit2, float4 *__restrict__ x4, float *__restrict__ xyz,
                                   float *__restrict__ xyz2, float *__restrict__ qp, int *__restrict__ perm) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_pad) return;
    const int64_t j = (int64_t)(keys[min(p, n - 1)] & 0xffffffffull);
    const float a = x[3 * j], b = x[3 * j + 1], c = x[3 * j + 2];
    perm[p] = (int)(p < n ? j : p);
    x4[p] = make_float4(a, b, c, 0.f);
    xyz[p] = a * unit;
    xyz[n_pad + p] = b * unit;
    xyz[2 * n_pad + p] = c * unit;
    xyz2[p] = a * unit2;
    xyz2[n_pad + p] = b * unit2;
    xyz2[2 * n_pad + p] = c * unit2;
    qp[p] = p < n ? q[j] : 0.f;
}

// What the best node block of the symmetric kernels depends on besides the node count and the form: how far
// the tail and skip classes reach against the nodes' extent (in steps of two of the squared
// distance), the share of expanded passes (in quarters), and the planar and periodic variants.  Sum
// on 512-node blocks over sum on 1,024: from 0.41 (narrow kernel, 20,000 nodes in a periodic square)
// to 1.5 (wide general kernel, 20,000 in a cube) at one node count and form.
static int tune_class(const nf_operator *op, double expanded) {
    float tail, skip;
    class_limits(op, &tail, &skip);
    auto reach = [&](float lim) {
        const double r = (double)lim / std::max((double)op->span2, 1e-30);
        return std::min(31, std::max(0, 24 + (int)std::floor(std::log2(std::max(r, 1e-30)))));
    };
    const int share = std::min(3, (int)(4.0 * expanded));
    return (((share * 32 + reach(tail)) * 32 + reach(skip)) * 2 + op->planar) * 2 + (op->kp.period > 0.f ? 1 : 0);
}

nf_status mf_build_nodes(nf_operator *op, const float *x, const float *q, cudaStream_t s) {
    const int64_t n = op->n, n_pad = op->n_pad;
    const nf_kernel &k = op->kp;
    op->form = mf_form(k);
    int64_t m = 1;
    while (m < n_pad) m <<= 1;
    // One allocation for all node arrays, 16-byte types first, and the bounding box.  The sort's keys
    // (m < 2 n_pad of 8 bytes) take rg's place until sym_static_kernel writes it.
    const int64_t np = n_pad / kPassRows, nt = n_pad / kTileCols;
    unsigned char *mem = nullptr;
    NF_CUDA_TRY(cudaMalloc(&mem, sizeof(float4) * (3 * n_pad + 4 * np + 4 * nt) + 2 * sizeof(float2) * n_pad +
                                     (7 * sizeof(float) + sizeof(int)) * n_pad + 64));
    op->rg = reinterpret_cast<float4 *>(mem);
    op->x4 = op->rg + n_pad;
    op->pc = op->x4 + n_pad;
    op->pe = op->pc + np;
    op->tc = op->pe + np;
    op->te = op->tc + nt;
    op->rg2 = op->te + nt;
    op->pc2 = op->rg2 + n_pad;
    op->pe2 = op->pc2 + np;
    op->tc2 = op->pe2 + np;
    op->te2 = op->tc2 + nt;
    op->xyz = reinterpret_cast<float *>(op->te2 + nt);  // n_pad is a multiple of 1024: each array stays aligned
    op->xyz2 = op->xyz + 3 * n_pad;
    op->q = op->xyz2 + 3 * n_pad;
    op->rw = reinterpret_cast<float2 *>(op->q + n_pad);
    op->rw2 = op->rw + n_pad;
    op->perm = reinterpret_cast<int *>(op->rw2 + n_pad);
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(op->rg);
    float *box = reinterpret_cast<float *>(op->perm + n_pad);
    int *count = reinterpret_cast<int *>(box + 6);
    row_bbox_kernel<<<1, 1024, 0, s>>>(x, n, box, count);
    row_key_kernel<<<(unsigned)ceil_div(m, 256), 256, 0, s>>>(x, n, m, box, keys);
    const int blk = (int)std::min<int64_t>(m, SORT_BLK);
    row_bitonic_local_kernel<<<(unsigned)(m / blk), SORT_BLK / 2, 0, s>>>(keys, blk, 2, blk);
    for (int64_t kk = 2 * blk; kk <= m; kk <<= 1) {
        for (int64_t jj = kk >> 1; jj >= blk; jj >>= 1)
            row_bitonic_kernel<<<(unsigned)ceil_div(m, 256), 256, 0, s>>>(keys, m, jj, kk);
        row_bitonic_local_kernel<<<(unsigned)(m / blk), SORT_BLK / 2, 0, s>>>(keys, blk, kk, kk);
    }
    const ExactUnits eu = op->eu = exact_units(op);
    pack_sorted_kernel<<<(unsigned)ceil_div(n_pad, 256), 256, 0, s>>>(x, q, keys, n, n_pad, mf_unit(op), eu.unit, op->x4,
                                                                     op->xyz, op->xyz2, op->q, op->perm);
    // the threshold of the expanded form as an exponent, for the narrower of the Gaussians that the
    // forward sums evaluate
    const float k2 = (k.s1 * k.s1) / (k.s2 * k.s2);
    const float narrow = op->form >= 2 ? k2 : (op->form == 0 ? 1.f / std::max(1.f, k2) : 1.f);
    const float most = kSymLocalSpread * narrow;
    const NodeSets sets{{{op->xyz, 1.f, k2, mf_period(op), most, op->rg, op->rw, op->pc, op->pe, op->tc, op->te},
                         {op->xyz2, eu.uu, eu.k2, eu.per, most, op->rg2, op->rw2, op->pc2, op->pe2, op->tc2, op->te2}}};
    sym_static_kernel<<<dim3((unsigned)ceil_div(np, 128), 2), 128, 0, s>>>(sets, n_pad, op->form, k.A1, k.A2, count);
    sym_tiles_kernel<<<dim3((unsigned)ceil_div(32 * nt, 128), 2), 128, 0, s>>>(sets, n_pad);
    float hbox[7] = {0, 0, 0, 0, 0, 0, 0};  // with the count behind the box
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(hbox, box, sizeof(hbox), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    op->planar = (e == cudaSuccess && hbox[2] == hbox[5]) ? 1 : 0;  // one z for every node
    if (e != cudaSuccess) return cuda_fail(e, "node order", __FILE__, __LINE__);
    for (int d = 0; d < 3; ++d) {
        const float w = (hbox[3 + d] - hbox[d]) * mf_unit(op);
        op->span2 += w * w;
    }
    int expanded = 0;
    std::memcpy(&expanded, &hbox[6], sizeof(int));
    op->tune_class = tune_class(op, (double)expanded / (double)np);
    return NF_OK;
}

// ------------------------------------------------------------------ the pair kernel
// Per unordered pair (expanded form, M >= 2): 3 FMA exponent, 2 MUL e1 = e2^M, 1 FMA pair weight,
// 1 FMA row sum, 1 FMA column sum in the full class; 3 FMA, row and column FMA in the tail class.
// D2: every node has the same z (flat domains), so the z terms of the distance vanish
// identically and are left out (bit-identical sums, one FMA fewer per pair).
// Blocks of 256 and 128 nodes (sets below ~13,300 nodes) work on the exact set: with coordinates
// rounded to exponent units two and three trajectories were 1.2 to 2 times as far from FP64 as with
// the kernel that formed their differences before (0.8e-7 -> 1.1e-7 relative L2).  The larger
// blocks keep the scaled set, whose columns need one multiplication less (1.5 to 2 % of a sum).
constexpr bool sym_exact(int blk) { return blk <= 256; }

template <int M, int BLK, bool D2>
__global__ void __launch_bounds__(MS_THREADS, 2)
mf_sym_kernel(SymNodes nd, const float *g_all, int B, int b_base, float uu, float k2, float per, float lim_tail,
              float lim_skip, float *__restrict__ partial, const int *__restrict__ pairs) {
    static_assert(M >= 0 && M <= 4, "form M: 0 general, 1 one Gaussian (A2 = 0), 2-4 width ratio");
    static_assert(BLK >= 128 && BLK <= 1024 && (BLK & (BLK - 1)) == 0, "block size");
    constexpr int R = kPassRows, NPASS = BLK / R, NT = BLK / kTileCols;
    static_assert(NT <= 32 && NT * NT <= MS_THREADS, "one lane per tile, one thread per tile pair");
    // Integer width ratios combine the two Gaussians per pair: with the row factors f1, f2,
    //   w_ij = A1 f1 e1 - A2 f2 e2 = (-A2 f2) (e2 + c_i e1),  c_i = -(A1 f1) / (A2 f2),
    // so one FMA forms the pair weight u = e2 + c_i e1 and one FMA each adds u g_j to the
    // row sum and u (-A2 f2 g_i) to the column sum: 8 FMA-pipe lane operations per
    // unordered pair instead of 9 (separate e1 and e2 row sums, two column FMAs).
    constexpr bool CW = M >= 2;
    constexpr bool HAS_TAIL = M != 1;
    constexpr bool EXACT = sym_exact(BLK);  // nd is the exact set, uu its exponent per squared unit
    extern __shared__ __align__(16) float ms_smem[];
    float *xs = ms_smem, *ys = xs + BLK, *zs = ys + BLK, *gs = zs + BLK;
    // per row: operands and first weight (mx, my, mz, c_i; M < 2: A1 f1 g_i), factors, and the
    // weight -A2 f2 g_i of the row's terms in the column sums
    float4 *rg = reinterpret_cast<float4 *>(gs + BLK);
    float2 *rw = reinterpret_cast<float2 *>(rg + BLK);
    float *rh = reinterpret_cast<float *>(rw + BLK);
    float4 *pc = reinterpret_cast<float4 *>(rh + BLK), *pe = pc + NPASS;
    float4 *tcs = pe + NPASS, *tes = tcs + NT;
    float *colacc = reinterpret_cast<float *>(tes + NT);  // [MS_WARPS][BLK]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t n_pad = nd.n_pad;
    int I, J;
    sym_pair(pairs ? (int64_t)__ldg(pairs + blockIdx.x) : (int64_t)blockIdx.x, I, J);  // pairs: live list
    const bool diag = I == J;
    const int b = b_base + blockIdx.z;
    const float *g = g_all + (int64_t)b * n_pad;
    const int64_t cbase = (int64_t)J * BLK, rbase = (int64_t)I * BLK;
    const float iper = per > 0.f ? 1.f / per : 0.f;
    float *out_rows = partial + ((int64_t)J * B + b) * n_pad + rbase;
    float *out_cols = partial + ((int64_t)I * B + b) * n_pad + cbase;

    // The column block's coordinates and the passes' and tiles' boxes are copied while g decides:
    // a non-finite value switches the classes off, a block pair without a live tile pair writes
    // its zero sums and leaves.
    for (int k = tid; k < BLK / 4; k += MS_THREADS) {
        cp_async16(xs + 4 * k, nd.xyz + cbase + 4 * k);
        cp_async16(ys + 4 * k, nd.xyz + n_pad + cbase + 4 * k);
        cp_async16(zs + 4 * k, nd.xyz + 2 * n_pad + cbase + 4 * k);
    }
    for (int k = tid; k < NPASS; k += MS_THREADS) {
        cp_async16(pc + k, nd.pc + rbase / R + k);
        cp_async16(pe + k, nd.pe + rbase / R + k);
    }
    if (tid < NT) {
        cp_async16(tcs + tid, nd.tc + cbase / kTileCols + tid);
        cp_async16(tes + tid, nd.te + cbase / kTileCols + tid);
    }
    constexpr int KT = (BLK + MS_THREADS - 1) / MS_THREADS;  // nodes per thread
    float4 p[KT];
    float2 w[KT];
#pragma unroll
    for (int t = 0; t < KT; ++t) {
        const int k = min(tid + t * MS_THREADS, BLK - 1);
        p[t] = __ldg(nd.rg + rbase + k);
        w[t] = __ldg(nd.rw + rbase + k);
    }
    bool bad = false, live = false;
    if (tid < NT * NT) {
        const int64_t ti = rbase / kTileCols + tid / NT, tj = cbase / kTileCols + tid % NT;
        live = box_d2(__ldg(nd.tc + ti), __ldg(nd.te + ti), __ldg(nd.tc + tj), __ldg(nd.te + tj), per, iper) <= lim_skip;
    }
    if (!diag)
        for (int k = tid; k < MS_WARPS * BLK / 4; k += MS_THREADS)
            reinterpret_cast<float4 *>(colacc)[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    // everything above depends on the operator alone; g is written by the kernel before
    pdl_wait();
    pdl_trigger();
#pragma unroll
    for (int t = 0; t < KT; ++t) {
        const int k = tid + t * MS_THREADS;
        if (k < BLK) {
            const float gc = g[cbase + k], gr = g[rbase + k];
            gs[k] = gc;
            rg[k] = make_float4(p[t].x, p[t].y, p[t].z, CW ? w[t].x : w[t].x * gr);
            rw[k] = w[t];
            rh[k] = w[t].y * gr;
            bad |= !(0.f * gc + 0.f * gr == 0.f);  // 0 * v is NaN for a non-finite v
        }
    }
    if (!__syncthreads_or(bad || live)) {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = tid; k < BLK / 4; k += MS_THREADS) {
            reinterpret_cast<float4 *>(out_rows)[k] = zero;
            reinterpret_cast<float4 *>(out_cols)[k] = zero;
        }
        cp_async_wait_all();
        return;
    }
    if (__syncthreads_or(bad)) lim_tail = lim_skip = __int_as_float(0x7f800000);
    cp_async_wait_all();
    __syncthreads();

    const u64 nk2 = f2_dup(-k2), uup = f2_dup(uu);
    const u64 ipp = f2_dup(iper), npp = f2_dup(-per), mgp = f2_dup(kRintMagic);
    const float4 *xs4 = reinterpret_cast<const float4 *>(xs), *ys4 = reinterpret_cast<const float4 *>(ys);
    const float4 *zs4 = reinterpret_cast<const float4 *>(zs), *gs4 = reinterpret_cast<const float4 *>(gs);
    float4 *cw4 = reinterpret_cast<float4 *>(colacc + warp * BLK);
    const int ntile = (int)min((int64_t)NT, (nd.n - cbase + kTileCols - 1) / kTileCols);  // tiles with real nodes

    for (int ps = warp; ps < NPASS; ps += MS_WARPS) {
        const int r0 = ps * R;
        if (rbase + r0 >= nd.n) break;  // padding: no row to write, and g = 0 in every column sum
        const float4 c = pc[ps];
        // tile classes of this pass, one lane per tile
        float d2 = 3.4e38f;
        if (lane < ntile) d2 = box_d2(c, pe[ps], tcs[lane], tes[lane], per, iper);
        const unsigned live_t = __ballot_sync(0xffffffffu, lane < ntile && d2 <= lim_skip);
        const int form = (int)c.w;  // warp-uniform
        // the tail class is taken in the expanded form only
        const unsigned full_t = HAS_TAIL && form == 1 ? live_t & __ballot_sync(0xffffffffu, d2 <= lim_tail) : live_t;
        const unsigned tail_t = live_t & ~full_t;
        u64 xi[R], yi[R], zi[R], h1[R], h2[R], a1[R], a2[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 p = rg[r0 + r];
            xi[r] = f2_dup(p.x);
            yi[r] = f2_dup(p.y);
            zi[r] = f2_dup(p.z);
            h1[r] = f2_dup(p.w);
            h2[r] = f2_dup(rh[r0 + r]);
            a1[r] = 0ull;
            a2[r] = 0ull;
        }
        // e1, e2 of two pairs from the exponent argument (expanded s_ij or r^2).  e1 = e2^M by
        // squaring on the FMA pipe; taking it from the SFU instead (ex2 of -M s) measured slower.
        auto exps = [&](u64 arg, u64 &e1, u64 &e2) {
            float s0, s1v;
            f2_unpack(arg, s0, s1v);
            if constexpr (M == 1) {
                e1 = f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v));
                e2 = 0ull;
            } else if constexpr (M > 0) {
                e2 = f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v));
                const u64 sq = f2_mul(e2, e2);
                e1 = M == 2 ? sq : (M == 3 ? f2_mul(sq, e2) : f2_mul(sq, sq));
            } else {
                e1 = f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v));
                e2 = f2_ex2(f2_mul(arg, nk2));
            }
        };
        // one pair's contribution to row r's sums and to the column sum cacc
        auto accum = [&](int r, u64 arg, u64 gj, u64 &cacc) {
            u64 e1, e2;
            exps(arg, e1, e2);
            if constexpr (M == 1) {
                a1[r] = f2_fma(e1, gj, a1[r]);
                cacc = f2_fma(e1, h1[r], cacc);
            } else if constexpr (CW) {
                const u64 u = f2_fma(e1, h1[r], e2);
                a1[r] = f2_fma(u, gj, a1[r]);
                cacc = f2_fma(u, h2[r], cacc);
            } else {
                a1[r] = f2_fma(e1, gj, a1[r]);
                a2[r] = f2_fma(e2, gj, a2[r]);
                cacc = f2_fma(e1, h1[r], f2_fma(e2, h2[r], cacc));
            }
        };
        // the same in the tail class: e2 alone
        auto accum_tail = [&](int r, u64 arg, u64 gj, u64 &cacc) {
            u64 e2;
            if constexpr (CW) {
                float s0, s1v;
                f2_unpack(arg, s0, s1v);
                e2 = f2_pack(ex2_sfu(-s0), ex2_sfu(-s1v));
                a1[r] = f2_fma(e2, gj, a1[r]);
            } else {
                e2 = f2_ex2(f2_mul(arg, nk2));
                a2[r] = f2_fma(e2, gj, a2[r]);
            }
            cacc = f2_fma(e2, h2[r], cacc);
        };
        const u64 cxp = f2_dup(c.x), cyp = f2_dup(c.y), czp = f2_dup(c.z);
        auto add_cols = [&](int q, const u64 (&cacc)[2]) {
            if (!diag) {
                float4 cv = cw4[q];
                u64 c0 = f2_add(f2_lo(cv), cacc[0]), c1 = f2_add(f2_hi(cv), cacc[1]);
                f2_unpack(c0, cv.x, cv.y);
                f2_unpack(c1, cv.z, cv.w);
                cw4[q] = cv;
            }
        };
        // each lane takes 4 consecutive columns (two f32x2 pairs) of every tile.
        // form 1: expanded about c; P: columns at their nearest image of c; TAIL: the tail class
        auto sweep_local = [&](auto tag, auto tail, unsigned tiles) {
            constexpr bool P = decltype(tag)::value, TAIL = decltype(tail)::value;
#pragma unroll 1
            for (; tiles; tiles &= tiles - 1) {
                const int q = (__ffs(tiles) - 1) * (kTileCols / 4) + lane;
                const float4 x4 = xs4[q], y4 = ys4[q], g4 = gs4[q];
                const float4 z4 = D2 ? make_float4(0.f, 0.f, 0.f, 0.f) : zs4[q];
                u64 xt[2] = {f2_sub(f2_lo(x4), cxp), f2_sub(f2_hi(x4), cxp)};
                u64 yt[2] = {f2_sub(f2_lo(y4), cyp), f2_sub(f2_hi(y4), cyp)};
                const u64 zt[2] = {f2_sub(f2_lo(z4), czp), f2_sub(f2_hi(z4), czp)};
                if constexpr (P) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        xt[h] = f2_wrap(xt[h], ipp, npp, mgp);
                        yt[h] = f2_wrap(yt[h], ipp, npp, mgp);
                    }
                }
                const u64 gj[2] = {f2_lo(g4), f2_hi(g4)};
                u64 nj[2], cacc[2] = {0ull, 0ull};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    nj[h] = f2_fma(yt[h], yt[h], f2_mul(xt[h], xt[h]));
                    if constexpr (!D2) nj[h] = f2_fma(zt[h], zt[h], nj[h]);
                    if constexpr (EXACT) nj[h] = f2_mul(nj[h], uup);
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const u64 zz = D2 ? nj[h] : f2_fma(zi[r], zt[h], nj[h]);
                        const u64 sij = f2_fma(xi[r], xt[h], f2_fma(yi[r], yt[h], zz));
                        if constexpr (TAIL)
                            accum_tail(r, sij, gj[h], cacc[h]);
                        else
                            accum(r, sij, gj[h], cacc[h]);
                    }
                }
                add_cols(q, cacc);
            }
        };
        // forms 0, 2, 3: coordinate differences; CEN: rows centred on c and columns' x, y at
        // their nearest image of c (forms 2, 3); PW: each pair's x, y differences reduced to
        // their nearest image (form 3)
        auto sweep_diff = [&](auto tag_c, auto tag_w, unsigned tiles) {
            constexpr bool CEN = decltype(tag_c)::value, PW = decltype(tag_w)::value;
#pragma unroll 1
            for (; tiles; tiles &= tiles - 1) {
                const int q = (__ffs(tiles) - 1) * (kTileCols / 4) + lane;
                const float4 x4 = xs4[q], y4 = ys4[q], g4 = gs4[q];
                const float4 z4 = D2 ? make_float4(0.f, 0.f, 0.f, 0.f) : zs4[q];
                u64 xj[2] = {f2_lo(x4), f2_hi(x4)}, yj[2] = {f2_lo(y4), f2_hi(y4)};
                const u64 zj[2] = {f2_lo(z4), f2_hi(z4)};
                if constexpr (CEN) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        xj[h] = f2_wrap(f2_sub(xj[h], cxp), ipp, npp, mgp);
                        yj[h] = f2_wrap(f2_sub(yj[h], cyp), ipp, npp, mgp);
                    }
                }
                const u64 gj[2] = {f2_lo(g4), f2_hi(g4)};
                u64 cacc[2] = {0ull, 0ull};
#pragma unroll
                for (int r = 0; r < R; ++r) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        u64 dx = f2_sub(xi[r], xj[h]), dy = f2_sub(yi[r], yj[h]);
                        const u64 dz = f2_sub(zi[r], zj[h]);
                        if constexpr (PW) {
                            dx = f2_wrap(dx, ipp, npp, mgp);
                            dy = f2_wrap(dy, ipp, npp, mgp);
                        }
                        u64 r2 = f2_fma(dy, dy, f2_mul(dx, dx));
                        if constexpr (!D2) r2 = f2_fma(dz, dz, r2);
                        if constexpr (EXACT) r2 = f2_mul(r2, uup);
                        accum(r, r2, gj[h], cacc[h]);
                    }
                }
                add_cols(q, cacc);
            }
        };
        if (form == 1) {
            if (per > 0.f) {
                if constexpr (HAS_TAIL) sweep_local(PerTag<true>{}, PerTag<true>{}, tail_t);
                sweep_local(PerTag<true>{}, PerTag<false>{}, full_t);
            } else {
                if constexpr (HAS_TAIL) sweep_local(PerTag<false>{}, PerTag<true>{}, tail_t);
                sweep_local(PerTag<false>{}, PerTag<false>{}, full_t);
            }
        } else if (form == 0) {
            sweep_diff(PerTag<false>{}, PerTag<false>{}, full_t);
        } else if (form == 2) {
            sweep_diff(PerTag<true>{}, PerTag<false>{}, full_t);
        } else {
            sweep_diff(PerTag<true>{}, PerTag<true>{}, full_t);
        }
        float v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            v[r] = f2_fold(a1[r]);
            if constexpr (M == 0) v[r] = rw[r0 + r].x * v[r] + rw[r0 + r].y * f2_fold(a2[r]);
        }
        int row;
        float tot = warp_reduce_rows<R>(v, lane, row);
        if constexpr (M > 0) tot *= CW ? rw[r0 + row].y : rw[r0 + row].x;
        if ((lane & (32 / R - 1)) == 0) out_rows[r0 + row] = tot;
    }
    if (diag) return;
    __syncthreads();
    for (int k = tid; k < BLK; k += MS_THREADS) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < MS_WARPS; ++w) v += colacc[w * BLK + k];
        out_cols[k] = v;
    }
}

// ------------------------------------------------------------------ launch
template <int M, int BLK, bool D2>
static cudaError_t sym_attr() {
    return cudaFuncSetAttribute(mf_sym_kernel<M, BLK, D2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)ms_smem_bytes(BLK));
}
template <int M>
static cudaError_t sym_attrs() {
    cudaError_t e = sym_attr<M, 1024, false>();
    if (e == cudaSuccess) e = sym_attr<M, 1024, true>();
    if (e == cudaSuccess) e = sym_attr<M, 512, false>();
    if (e == cudaSuccess) e = sym_attr<M, 512, true>();
    if (e == cudaSuccess) e = sym_attr<M, 256, false>();
    if (e == cudaSuccess) e = sym_attr<M, 128, false>();
    return e;
}
nf_status sym_init_attrs() {
    NF_CUDA_TRY(sym_attrs<0>());
    NF_CUDA_TRY(sym_attrs<1>());
    NF_CUDA_TRY(sym_attrs<2>());
    NF_CUDA_TRY(sym_attrs<3>());
    NF_CUDA_TRY(sym_attrs<4>());
    return NF_OK;
}

template <int BLK, bool D2>
static cudaError_t launch_sym_blk(nf_operator *op, int B, int b_base, cudaStream_t s) {
    const nf_kernel &k = op->kp;
    constexpr bool EXACT = sym_exact(BLK);
    const ExactUnits &eu = op->eu;
    const float uu = EXACT ? eu.uu : 1.f, k2 = EXACT ? eu.k2 : (k.s1 * k.s1) / (k.s2 * k.s2);
    const int64_t nb = op->n_pad / BLK;
    // blockIdx.z: trajectory b_base + z of the B in the partial-sum layout
    dim3 grid((unsigned)(op->mf_cull ? op->cull_live : nb * (nb + 1) / 2), 1, (unsigned)(B - b_base));
    const size_t smem = ms_smem_bytes(BLK);
    const SymNodes nd = EXACT ? exact_nodes(op) : sym_nodes(op);
    const int *pairs = op->mf_cull ? op->cull_pairs : nullptr;
    const float per = EXACT ? eu.per : mf_period(op);
    float tail, skip;
    class_limits(op, &tail, &skip);
    tail /= uu;  // boxes are in stored units
    skip /= uu;
    const float *g = op->g;
    float *partial = op->partial;
    auto go = [&](auto kernel) {
        return launch_dependent(kernel, grid, MS_THREADS, smem, s, !op->profile, nd, g, B, b_base, uu, k2, per, tail,
                                skip, partial, pairs);
    };
    switch (op->form) {
        case 1: return go(mf_sym_kernel<1, BLK, D2>);
        case 2: return go(mf_sym_kernel<2, BLK, D2>);
        case 3: return go(mf_sym_kernel<3, BLK, D2>);
        case 4: return go(mf_sym_kernel<4, BLK, D2>);
        default: return go(mf_sym_kernel<0, BLK, D2>);
    }
}

nf_status launch_sym(nf_operator *op, int B, int b_base, cudaStream_t s) {
    switch (op->sym_blk) {
        case 128: NF_CUDA_TRY((launch_sym_blk<128, false>(op, B, b_base, s))); break;
        case 256: NF_CUDA_TRY((launch_sym_blk<256, false>(op, B, b_base, s))); break;
        case 512:
            if (op->planar)
                NF_CUDA_TRY((launch_sym_blk<512, true>(op, B, b_base, s)));
            else
                NF_CUDA_TRY((launch_sym_blk<512, false>(op, B, b_base, s)));
            break;
        default:
            if (op->planar)
                NF_CUDA_TRY((launch_sym_blk<1024, true>(op, B, b_base, s)));
            else
                NF_CUDA_TRY((launch_sym_blk<1024, false>(op, B, b_base, s)));
    }
    return NF_OK;
}

}  // namespace nfi
