// nf_dense.cu -- precomputed operator W diag(q) of Eq. (2.9) and its streaming
// matrix-vector product.
//
// Build (once per operator): WQ[i, j] = w(|x_i - x_j|) q_j, row-major, leading
// dimension n_pad (padded columns are zero because q is zero there).
//   NF_DENSE_FP32:   FP32 plane.
//   NF_DENSE_BF16X2: s_i = 2^ceil(log2 max_j |WQ_ij|) (a power of two, so dividing by
//                    it is exact); hi = bf16_rn(WQ/s_i), lo = bf16_rn(WQ/s_i - hi).
//                    hi + lo carries ~16 significant bits; I_i = s_i sum_j (hi+lo) F_j.
//                    The two planes use the blocked layout (128 x 64 blocks of 16 KB), the
//                    tile the batched tensor-core GEMM reads with one sequential copy.
// Apply (every stage): HBM-bound stream of 4 bytes per entry for either plane type.
//   NF_DENSE_SYM_FP32: the kernel matrix K_ij = w(|x_i - x_j|) itself (q moves to the vector
//                    side, g = q o f), symmetric, so only its upper-triangle 1024 x 1024
//                    blocks are stored (n_pad^2 / 2 + n_pad * 512 entries).  One CTA streams
//                    a block (I <= J) once and produces both its row sums (K_IJ g_J, to
//                    partial slot J) and its column sums (K_IJ^T g_I, to slot I): half the
//                    HBM bytes of the full matrix per stage.
//   NF_DENSE_SYM_BF16X2: the same blocks as bf16 hi + lo planes with symmetric power-of-two
//                    scaling s_i s_j (the vector is scaled on the way in, each output by its
//                    own s_i): the precision form of the symmetric operator.
// Several trajectories share one stream of the matrix (passes of up to 8 on the full planes, up to
// 4 on the symmetric ones).  Work items (32-row block, column split) write partial sums like the
// matrix-free kernel, so the same stage kernel finishes the RK4 step.
#include "nf_pairs.cuh"

#include <algorithm>

namespace nfi {

// ---------------------------------------------------------------- build
__device__ __forceinline__ float mexhat(float r2, float A1, float is1, float A2, float is2) {
    return A1 * expf(-r2 * is1) - A2 * expf(-r2 * is2);
}

// Squared distance; per > 0: x and y differences reduced to their nearest images (§4,
// Eq. (dist)), ip = 1 / per.
__device__ __forceinline__ float pair_r2(float4 a, float4 b, float per, float ip) {
    float dx = a.x - b.x, dy = a.y - b.y;
    const float dz = a.z - b.z;
    if (per > 0.f) {
        dx = wrap1(dx, per, ip);
        dy = wrap1(dy, per, ip);
    }
    return dx * dx + dy * dy + dz * dz;
}

// one block per row i; FP32 plane
__global__ void dense_build_fp32_kernel(const float4 *__restrict__ x4, const float *__restrict__ q, int64_t n,
                                        int64_t n_pad, float A1, float is1, float A2, float is2, float per,
                                        float ip, float *__restrict__ W) {
    const int64_t i = blockIdx.x;
    const float4 xi = x4[i];
    float *row = W + i * n_pad;
    for (int64_t j = threadIdx.x; j < n_pad; j += blockDim.x) {
        const float4 xj = x4[j];
        const float r2 = pair_r2(xi, xj, per, ip);
        row[j] = mexhat(r2, A1, is1, A2, is2) * q[j];
    }
}

// one block per row: row scale s_i (power of two), then hi / lo planes
__global__ void dense_build_bf16x2_kernel(const float4 *__restrict__ x4, const float *__restrict__ q, int64_t n,
                                          int64_t n_pad, float A1, float is1, float A2, float is2, float per,
                                          float ip, uint16_t *__restrict__ Whi, uint16_t *__restrict__ Wlo,
                                          float *__restrict__ rs) {
    __shared__ float red[32];
    const int64_t i = blockIdx.x;
    const float4 xi = x4[i];
    float mx = 0.f;
    for (int64_t j = threadIdx.x; j < n_pad; j += blockDim.x) {
        const float4 xj = x4[j];
        const float r2 = pair_r2(xi, xj, per, ip);
        mx = fmaxf(mx, fabsf(mexhat(r2, A1, is1, A2, is2) * q[j]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x < 32) {
        float v = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (threadIdx.x == 0) red[0] = v;
    }
    __syncthreads();
    mx = red[0];
    // s = 2^e with mx <= s (frexp: mx = m 2^e, m in [0.5, 1))
    int e = 0;
    float s = 1.f;
    if (mx > 0.f) {
        (void)frexpf(mx, &e);
        s = ldexpf(1.f, e);
    }
    const float inv = 1.f / s;  // exact: power of two
    if (threadIdx.x == 0) rs[i] = s;
    for (int64_t j = threadIdx.x; j < n_pad; j += blockDim.x) {
        const float4 xj = x4[j];
        const float r2 = pair_r2(xi, xj, per, ip);
        const float v = mexhat(r2, A1, is1, A2, is2) * q[j] * inv;
        const __nv_bfloat16 hi = __float2bfloat16_rn(v);
        const __nv_bfloat16 lo = __float2bfloat16_rn(v - __bfloat162float(hi));
        const int64_t o = blocked_offset(i, j, n_pad);
        Whi[o] = __bfloat16_as_ushort(hi);
        Wlo[o] = __bfloat16_as_ushort(lo);
    }
}

// ---- symmetric blocks: block pair t = J (J + 1) / 2 + I (I <= J) holds K over rows of node
// block I and columns of node block J, row-major, SB x SB
constexpr int SB = 1024;
constexpr int SYM_THREADS = 256;
constexpr int SYM_WARPS = SYM_THREADS / 32;

// grid (pairs, SB / 16): each block writes 16 rows of one block pair
__global__ void dense_build_sym_kernel(const float4 *__restrict__ x4, float A1, float is1, float A2, float is2,
                                       float per, float ip, float *__restrict__ K) {
    int I, J;
    sym_pair(blockIdx.x, I, J);
    float *blk = K + (int64_t)blockIdx.x * SB * SB;
    for (int rr = 0; rr < 16; ++rr) {
        const int r = blockIdx.y * 16 + rr;
        const float4 xi = x4[(int64_t)I * SB + r];
        for (int c = threadIdx.x; c < SB; c += blockDim.x) {
            const float4 xj = x4[(int64_t)J * SB + c];
            const float r2 = pair_r2(xi, xj, per, ip);
            blk[(int64_t)r * SB + c] = mexhat(r2, A1, is1, A2, is2);
        }
    }
}

// ---- symmetric bf16 hi + lo blocks (NF_DENSE_SYM_BF16X2).  K_ij = s_i s_j (hi_ij + lo_ij)
// with s_i = 2^round(log2 sqrt(max_j |K_ij|)) over the real nodes: a power of two, so the
// division by s_i s_j is exact, and the scaled matrix stays symmetric.  hi = bf16_rn(K / s s),
// lo = bf16_rn(K / s s - hi): 16 significant bits, |K / s s - hi - lo| <= 2^-18 |K / s s|.
// Block pair t (I <= J) holds rows of node block I x columns of node block J; a row is 128
// chunks of 8 columns, each chunk 16 bytes of hi followed by 16 bytes of lo (one 32-byte
// piece per lane and chunk).  Entries of padded rows or columns are zero.
constexpr int SBC = SB / 8;  // chunks per block row

__global__ void sym_rowscale_kernel(const float4 *__restrict__ x4, int64_t n, float A1, float is1, float A2,
                                    float is2, float per, float ip, float *__restrict__ sc) {
    __shared__ float red[32];
    const int64_t i = blockIdx.x;
    if (i >= n) {  // padded row: any power of two
        if (threadIdx.x == 0) sc[i] = 1.f;
        return;
    }
    const float4 xi = x4[i];
    float mx = 0.f;
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) mx = fmaxf(mx, fabsf(mexhat(pair_r2(xi, x4[j], per, ip), A1, is1, A2, is2)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        float v = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v = fmaxf(v, red[w]);
        int e = 0;
        if (v > 0.f) {
            (void)frexpf(v, &e);  // v = m 2^e, m in [0.5, 1)
        }
        sc[i] = v > 0.f ? ldexpf(1.f, e / 2) : 1.f;  // ~ sqrt(v), a power of two
    }
}

// grid (pairs, SB / 16): each block writes 16 rows of one block pair
__global__ void dense_build_sym_bf16x2_kernel(const float4 *__restrict__ x4, const float *__restrict__ sc, int64_t n,
                                              float A1, float is1, float A2, float is2, float per, float ip,
                                              uint4 *__restrict__ K) {
    int I, J;
    sym_pair(blockIdx.x, I, J);
    uint4 *blk = K + (int64_t)blockIdx.x * SB * SBC * 2;
    for (int rr = 0; rr < 16; ++rr) {
        const int r = blockIdx.y * 16 + rr;
        const int64_t i = (int64_t)I * SB + r;
        const float4 xi = x4[i];
        const float si = sc[i];
        for (int c = threadIdx.x; c < SBC; c += blockDim.x) {
            uint32_t h[4], l[4];
#pragma unroll
            for (int e = 0; e < 8; e += 2) {
                float v[2];
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int64_t j = (int64_t)J * SB + 8 * c + e + t;
                    v[t] = (i < n && j < n) ? mexhat(pair_r2(xi, x4[j], per, ip), A1, is1, A2, is2) / (si * sc[j]) : 0.f;
                }
                const __nv_bfloat16 h0 = __float2bfloat16_rn(v[0]), h1 = __float2bfloat16_rn(v[1]);
                const __nv_bfloat16 l0 = __float2bfloat16_rn(v[0] - __bfloat162float(h0));
                const __nv_bfloat16 l1 = __float2bfloat16_rn(v[1] - __bfloat162float(h1));
                h[e / 2] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                l[e / 2] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
            }
            blk[((int64_t)r * SBC + c) * 2] = make_uint4(h[0], h[1], h[2], h[3]);
            blk[((int64_t)r * SBC + c) * 2 + 1] = make_uint4(l[0], l[1], l[2], l[3]);
        }
    }
}

nf_status launch_dense_build(nf_operator *op, cudaStream_t s) {
    const nf_kernel &k = op->kp;
    const float is1 = 1.f / (k.s1 * k.s1), is2 = 1.f / (k.s2 * k.s2);
    const float per = k.period > 0.f ? k.period : 0.f, ip = per > 0.f ? 1.f / per : 0.f;
    if (op->path == NF_DENSE_SYM_FP32) {
        const int64_t nb = op->n_pad / SB;
        dense_build_sym_kernel<<<dim3((unsigned)(nb * (nb + 1) / 2), SB / 16), 256, 0, s>>>(op->x4, k.A1, is1, k.A2,
                                                                                       is2, per, ip, op->W32);
    } else if (op->path == NF_DENSE_SYM_BF16X2) {
        const int64_t nb = op->n_pad / SB;
        sym_rowscale_kernel<<<(unsigned)op->n_pad, 256, 0, s>>>(op->x4, op->n, k.A1, is1, k.A2, is2, per, ip, op->rs);
        NF_CUDA_TRY(cudaGetLastError());
        dense_build_sym_bf16x2_kernel<<<dim3((unsigned)(nb * (nb + 1) / 2), SB / 16), 128, 0, s>>>(
            op->x4, op->rs, op->n, k.A1, is1, k.A2, is2, per, ip, reinterpret_cast<uint4 *>(op->Whi));
    } else if (op->path == NF_DENSE_FP32) {
        dense_build_fp32_kernel<<<(unsigned)op->n_pad, 256, 0, s>>>(op->x4, op->q, op->n, op->n_pad, k.A1, is1, k.A2,
                                                               is2, per, ip, op->W32);
    } else {
        dense_build_bf16x2_kernel<<<(unsigned)op->n_pad, 256, 0, s>>>(op->x4, op->q, op->n, op->n_pad, k.A1, is1,
                                                                 k.A2, is2, per, ip, op->Whi, op->Wlo, op->rs);
    }
    NF_CUDA_TRY(cudaGetLastError());
    return NF_OK;
}

// ---------------------------------------------------------------- GEMV
constexpr int DG_THREADS = 256;
constexpr int DG_WARPS = DG_THREADS / 32;
constexpr int DG_R = 4;                        // rows per warp
constexpr int DG_ROWS = DG_WARPS * DG_R;       // rows per block
constexpr int DG_TILE = 1024;                  // columns per inner tile
static_assert(kNodePad % DG_TILE == 0, "tile must divide the node padding");

__device__ __forceinline__ float4 ld_stream_f4(const float *p) {
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 ld_stream_u4(const void *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// Sums of NB trajectories over the full plane: W is streamed once for all of them (it was once per
// trajectory).  A warp takes 4 rows; every W value it loads meets NB vector values from L1.  HL:
// bf16 hi + lo planes in the blocked layout, lane l on columns tile + 8 l + 256 u; else the FP32
// plane, columns tile + 4 l + 128 u.  Bound: HBM, 4 bytes per entry whatever NB: per RK4 stage at
// n = 30,000 on the bf16 planes 1, 2, 3, 4, 8 trajectories in 506, 529, 526, 552, 638 us (559,
// 1,112, 1,667, 2,219, 4,450 with one stream each).  Two CTAs per SM at 128 registers beat one
// with more (3 trajectories 526 against 689 us); one trajectory on the bf16 planes takes three (four, at 64
// registers, spill: 588 us).
template <int NB, bool HL>
__global__ void __launch_bounds__(DG_THREADS, NB == 1 && HL ? 3 : 2)
gemv_kernel(const void *__restrict__ W0, const uint16_t *__restrict__ Wlo, const float *F, int64_t n_pad,
            int B, int b0, int64_t jchunk, float *__restrict__ partial) {
    constexpr int C = HL ? 8 : 4;                 // columns per load
    constexpr int UB = (HL ? 2 : 4) / (NB > 4 ? 2 : 1);  // loads per row in flight: 16 (8) x 16 bytes a lane
    constexpr int NU = DG_TILE / (32 * C);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int split = blockIdx.y;
    const int64_t row0 = ((int64_t)blockIdx.x * DG_WARPS + warp) * DG_R;
    const int64_t j0 = (int64_t)split * jchunk, j1 = min(n_pad, j0 + jchunk);
    const float *Fb = F + (int64_t)b0 * n_pad;
    const float *W32 = static_cast<const float *>(W0);
    const uint16_t *Whi = static_cast<const uint16_t *>(W0);
    float acc[DG_R][NB];
#pragma unroll
    for (int r = 0; r < DG_R; ++r)
#pragma unroll
        for (int v = 0; v < NB; ++v) acc[r][v] = 0.f;
    pdl_wait();
    pdl_trigger();
    for (int64_t t = j0; t < j1; t += DG_TILE) {
#pragma unroll
        for (int uh = 0; uh < NU; uh += UB) {
            uint4 h[DG_R][UB], l[DG_R][HL ? UB : 1];
#pragma unroll
            for (int r = 0; r < DG_R; ++r)
#pragma unroll
                for (int u = 0; u < UB; ++u) {
                    const int64_t col = t + 32 * C * (uh + u) + C * lane;
                    if constexpr (HL) {
                        const int64_t off = blocked_offset(row0 + r, col, n_pad);
                        h[r][u] = ld_stream_u4(Whi + off);
                        l[r][u] = ld_stream_u4(Wlo + off);
                    } else {
                        h[r][u] = ld_stream_u4(W32 + (row0 + r) * n_pad + col);
                    }
                }
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const float *fp = Fb + t + 32 * C * (uh + u) + C * lane;
                float fv[NB][C];
#pragma unroll
                for (int v = 0; v < NB; ++v)
#pragma unroll
                    for (int c = 0; c < C; c += 4) {
                        // (plain loads spill 232 bytes a thread on the bf16 planes with 8 trajectories: n = 30,000
                        // 919 us against 638; on the FP32 plane they are the better ones: 643 against 667)
                        const float *src = fp + (int64_t)v * n_pad + c;
                        const float4 f = HL ? ld_written4(src) : *reinterpret_cast<const float4 *>(src);
                        fv[v][c] = f.x, fv[v][c + 1] = f.y, fv[v][c + 2] = f.z, fv[v][c + 3] = f.w;
                    }
#pragma unroll
                for (int r = 0; r < DG_R; ++r) {
                    float w[C];
                    const uint32_t hw[4] = {h[r][u].x, h[r][u].y, h[r][u].z, h[r][u].w};
                    if constexpr (HL) {
                        const uint32_t lw[4] = {l[r][u].x, l[r][u].y, l[r][u].z, l[r][u].w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            w[2 * q] = __uint_as_float(hw[q] << 16) + __uint_as_float(lw[q] << 16);
                            w[2 * q + 1] = __uint_as_float(hw[q] & 0xffff0000u) + __uint_as_float(lw[q] & 0xffff0000u);
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < 4; ++q) w[q] = __uint_as_float(hw[q]);
                    }
#pragma unroll
                    for (int v = 0; v < NB; ++v)
#pragma unroll
                        for (int c = 0; c < C; ++c) acc[r][v] = fmaf(w[c], fv[v][c], acc[r][v]);
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < DG_R; ++r)
#pragma unroll
        for (int v = 0; v < NB; ++v) {
            const float s = warp_sum(acc[r][v]);
            if (lane == 0) partial[((int64_t)split * B + b0 + v) * n_pad + row0 + r] = s;
        }
}

// Symmetric blocks, up to NB trajectories per stream of the matrix.  A cluster of S CTAs takes one
// stored block pair (I <= J), 1024 / S rows each (S > 1 where the pairs alone would leave most of
// the GPU idle: 36 pairs at n = 8,000).  The columns are swept in NB parts of 1024 / NB, so that a
// lane's share of the vectors and of the column sums stays in 32 registers each whatever NB:
// warp w takes rows w, w + 8, ...; per row and part a lane loads 32 / NB columns with 16-byte
// streaming loads; the row's dot products with g_J are reduced 8 rows at a time across the warp
// by a transposed butterfly and added over the parts in shared memory; the column sums with
// g_I are added over the warps, then over the cluster's CTAs through distributed shared memory,
// each in a fixed order.  Row sums go to partial slot J, column sums to slot I; diagonal blocks
// write their row sums only.
//   HL: bf16 hi + lo blocks with symmetric scales: the vector is scaled on the way in
// (g'_j = s_j g_j) and each output by its own s_i.
template <int NB>
constexpr size_t sym_smem_floats(int rows) {
    return (size_t)2 * NB * rows + (size_t)SYM_WARPS * SB + (size_t)NB * SB;
}
template <int NB, bool HL>
__global__ void __launch_bounds__(SYM_THREADS, 2)
gemv_sym_kernel(const void *__restrict__ K, const float *g_all, const float *__restrict__ sc,
                int64_t n_pad, int B, int b0, int rows, float *__restrict__ partial) {
    constexpr int COLS = SB / NB;    // columns per part
    constexpr int CL = 32 / NB;      // columns per lane and part
    constexpr int RB = NB;           // rows in flight: 8 16-byte loads per lane
    extern __shared__ __align__(16) float gs_smem[];
    float *gI = gs_smem;                      // [NB][rows]
    float *rowacc = gI + NB * rows;           // [NB][rows]
    float *colred = rowacc + NB * rows;       // [SYM_WARPS][NB][COLS]
    float *colsum = colred + SYM_WARPS * SB;  // [NB][SB]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int I, J;
    sym_pair(blockIdx.x, I, J);
    const bool diag = I == J;
    const int slice = blockIdx.y, row_off = slice * rows, nv = min(NB, B - b0);
    // lane's column c of a part: FP32 4 lane + 128 u + (c & 3), u = c / 4; HL 8 lane + 256 u + (c & 7)
    auto col_of = [&](int c) { return HL ? 8 * lane + 256 * (c >> 3) + (c & 7) : 4 * lane + 128 * (c >> 2) + (c & 3); };
    pdl_wait();
    pdl_trigger();
    for (int k = tid; k < NB * rows; k += SYM_THREADS) {
        const int v = k / rows, r = k - v * rows;
        const int64_t node = (int64_t)I * SB + row_off + r;
        float x = v < nv ? g_all[(int64_t)(b0 + v) * n_pad + node] : 0.f;
        if constexpr (HL) x *= sc[node];
        gI[k] = x;
    }
    __syncthreads();
    const float *blk32 = static_cast<const float *>(K) + (int64_t)blockIdx.x * SB * SB;
    const uint4 *blkhl = static_cast<const uint4 *>(K) + (int64_t)blockIdx.x * SB * SBC * 2;
    for (int part = 0; part < NB; ++part) {
        float gj[NB][CL], col[NB][CL];
#pragma unroll
        for (int c = 0; c < CL; c += 4) {
            const int64_t node = (int64_t)J * SB + part * COLS + col_of(c);
            float4 s4 = make_float4(1.f, 1.f, 1.f, 1.f);
            if constexpr (HL) s4 = __ldg(reinterpret_cast<const float4 *>(sc + node));
#pragma unroll
            for (int v = 0; v < NB; ++v) {
                float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
                if (v < nv) f = *reinterpret_cast<const float4 *>(g_all + (int64_t)(b0 + v) * n_pad + node);
                gj[v][c] = f.x * s4.x, gj[v][c + 1] = f.y * s4.y, gj[v][c + 2] = f.z * s4.z, gj[v][c + 3] = f.w * s4.w;
                col[v][c] = col[v][c + 1] = col[v][c + 2] = col[v][c + 3] = 0.f;
            }
        }
        for (int r0 = warp; r0 < rows; r0 += 8 * SYM_WARPS) {  // 8 rows per group: r0, r0 + 8, ..., r0 + 56
            float dot[NB][8];
#pragma unroll
            for (int kk = 0; kk < 8; kk += RB) {
                float w[RB][CL];
#pragma unroll
                for (int q = 0; q < RB; ++q) {
                    const int64_t r = row_off + r0 + 8 * (kk + q);
                    if constexpr (HL) {
#pragma unroll
                        for (int u = 0; u < CL / 8; ++u) {
                            const uint4 *p = blkhl + (r * SBC + part * (COLS / 8) + lane + 32 * u) * 2;
                            const uint4 hv = ld_stream_u4(p), lv = ld_stream_u4(p + 1);
                            const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w}, lw[4] = {lv.x, lv.y, lv.z, lv.w};
#pragma unroll
                            for (int t = 0; t < 4; ++t) {
                                w[q][8 * u + 2 * t] = __uint_as_float(hw[t] << 16) + __uint_as_float(lw[t] << 16);
                                w[q][8 * u + 2 * t + 1] =
                                    __uint_as_float(hw[t] & 0xffff0000u) + __uint_as_float(lw[t] & 0xffff0000u);
                            }
                        }
                    } else {
#pragma unroll
                        for (int u = 0; u < CL / 4; ++u) {
                            const float4 f = ld_stream_f4(blk32 + r * SB + part * COLS + 4 * lane + 128 * u);
                            w[q][4 * u] = f.x, w[q][4 * u + 1] = f.y, w[q][4 * u + 2] = f.z, w[q][4 * u + 3] = f.w;
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < RB; ++q)
#pragma unroll
                    for (int v = 0; v < NB; ++v) {
                        const float gi = gI[v * rows + r0 + 8 * (kk + q)];
                        float d = 0.f;
#pragma unroll
                        for (int c = 0; c < CL; ++c) {
                            d = fmaf(w[q][c], gj[v][c], d);
                            col[v][c] = fmaf(w[q][c], gi, col[v][c]);
                        }
                        dot[v][kk + q] = d;
                    }
            }
#pragma unroll
            for (int v = 0; v < NB; ++v) {
                int row;
                const float tot = warp_reduce_rows<8>(dot[v], lane, row);
                float *dst = rowacc + v * rows + r0 + 8 * row;
                if ((lane & 3) == 0) *dst = part == 0 ? tot : *dst + tot;
            }
        }
        if (!diag) {
#pragma unroll
            for (int v = 0; v < NB; ++v)
#pragma unroll
                for (int c = 0; c < CL; c += 4)
                    *reinterpret_cast<float4 *>(colred + (warp * NB + v) * COLS + col_of(c)) =
                        make_float4(col[v][c], col[v][c + 1], col[v][c + 2], col[v][c + 3]);
            __syncthreads();
            for (int k = tid; k < SB; k += SYM_THREADS) {
                const int v = k / COLS, c = k - v * COLS;
                float s = 0.f;
#pragma unroll
                for (int w = 0; w < SYM_WARPS; ++w) s += colred[(w * NB + v) * COLS + c];
                colsum[v * SB + part * COLS + c] = s;
            }
            __syncthreads();
        }
    }
    __syncthreads();
    for (int k = tid; k < nv * rows; k += SYM_THREADS) {
        const int v = k / rows, r = k - v * rows;
        const int64_t node = (int64_t)I * SB + row_off + r;
        partial[((int64_t)J * B + b0 + v) * n_pad + node] = HL ? sc[node] * rowacc[k] : rowacc[k];
    }
    if (diag) return;  // uniform over the cluster
    const int S = SB / rows;
    if (S > 1) cluster_barrier();
    for (int k = tid; k < nv * rows; k += SYM_THREADS) {  // this CTA's share of the columns
        const int v = k / rows, c = row_off + (k - v * rows);
        float s = 0.f;
        if (S == 1) {
            s = colsum[v * SB + c];
        } else {
            for (int q = 0; q < S; ++q) s += ld_cluster(colsum + v * SB + c, (uint32_t)q);
        }
        const int64_t node = (int64_t)J * SB + c;
        partial[((int64_t)I * B + b0 + v) * n_pad + node] = HL ? sc[node] * s : s;
    }
    if (S > 1) cluster_barrier();  // no CTA leaves while another may read its sums
}

// ---------------------------------------------------------------- GEMM (several trajectories)
// I[b, i] = sum_j WQ[i, j] F[b, j] for B >= kGemmMinB trajectories on the FP32 plane: a
// register-tiled SIMT GEMM on the FP32 FMA pipe (the plain-FP32 counterpart of the batched
// tensor-core path), so that W is streamed once per 128 or 64 trajectories instead of once
// per trajectory.  CTA tile 128 rows (i) x GB_BN trajectories (b) x 16 columns (j) per
// step, 256 threads; thread (tm, tn) = (tid & 15, tid >> 4) owns the row pairs
// (2 tm + 32 r, 2 tm + 32 r + 1), r = 0..3, and the trajectories tn * 4 + c (plus
// 64 + tn * 4 + c when GB_BN = 128).  Accumulators are FP32 pairs along i, updated by
// fma.rn.f32x2 with the trajectory operand stored twice in shared memory (f, f): per k a
// warp reads its 32 rows' W values as one 128-byte row of pairs and its two trajectories'
// F values by broadcast.  Tiles are staged through registers into double-buffered shared
// memory (transposed: k-major).  Small node sets split K (grid z) into partial-sum slots
// that the stage kernel adds in a fixed order.
constexpr int GB_BM = 128, GB_BK = 16, GB_THREADS = 256;
constexpr int kGemmMinB = 33;  // below, passes of gemv_kernel over 8 trajectories: n = 30,000 8 in 0.65 ms, 32 in
                               // 2.6; one tile of 64 takes 3.1 ms however few of it are used

// Row strides are padded (130 floats, GB_BN + 2 pairs) so that the transposing stores of a
// warp (8 rows or trajectories x 4 k-quads) fall into distinct banks, while every row stays
// 8-byte (a) and 16-byte (b) aligned for the compute loop's vector loads.
constexpr int GB_AS = GB_BM + 2;
template <int GB_BN>
struct GemmSmem {
    float a[2][GB_BK][GB_AS];                       // W tile, k-major
    unsigned long long b[2][GB_BK][GB_BN + 2];      // (f, f) pairs, k-major
};

template <int GB_BN>
__global__ void __launch_bounds__(GB_THREADS, 2)
gemm_fp32_kernel(const float *__restrict__ W, const float *__restrict__ F, int64_t n_pad, int B, int64_t kchunk,
                 float *__restrict__ partial) {
    constexpr int NC = GB_BN / 16;                   // trajectories per thread (8 or 4)
    constexpr int BLD = GB_BN * 4 / GB_THREADS;      // float4 loads of the F tile per thread (2 or 1)
    extern __shared__ __align__(16) unsigned char gm_raw[];
    GemmSmem<GB_BN> &sm = *reinterpret_cast<GemmSmem<GB_BN> *>(gm_raw);
    const int tid = threadIdx.x, tm = tid & 15, tn = tid >> 4;
    const int64_t m0 = (int64_t)blockIdx.x * GB_BM;
    const int n0 = blockIdx.y * GB_BN;
    const int64_t k0 = (int64_t)blockIdx.z * kchunk, k1 = min(n_pad, k0 + kchunk);
    const int nkt = (int)((k1 - k0) / GB_BK);
    float4 ra[2], rb[BLD];
    auto load = [&](int kt) {
        const int64_t kb = k0 + (int64_t)kt * GB_BK;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int idx = tid + GB_THREADS * p, r = idx >> 2, kq = idx & 3;
            ra[p] = __ldg(reinterpret_cast<const float4 *>(W + (m0 + r) * n_pad + kb + 4 * kq));
        }
#pragma unroll
        for (int p = 0; p < BLD; ++p) {
            const int idx = tid + GB_THREADS * p, c = idx >> 2, kq = idx & 3;
            const int b = n0 + c;
            rb[p] = b < B ? __ldg(reinterpret_cast<const float4 *>(F + (int64_t)b * n_pad + kb + 4 * kq))
                          : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int idx = tid + GB_THREADS * p, r = idx >> 2, kq = idx & 3;
            sm.a[buf][4 * kq + 0][r] = ra[p].x;
            sm.a[buf][4 * kq + 1][r] = ra[p].y;
            sm.a[buf][4 * kq + 2][r] = ra[p].z;
            sm.a[buf][4 * kq + 3][r] = ra[p].w;
        }
#pragma unroll
        for (int p = 0; p < BLD; ++p) {
            const int idx = tid + GB_THREADS * p, c = idx >> 2, kq = idx & 3;
            sm.b[buf][4 * kq + 0][c] = f2_dup(rb[p].x);
            sm.b[buf][4 * kq + 1][c] = f2_dup(rb[p].y);
            sm.b[buf][4 * kq + 2][c] = f2_dup(rb[p].z);
            sm.b[buf][4 * kq + 3][c] = f2_dup(rb[p].w);
        }
    };
    u64 acc[4][NC];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[r][c] = 0ull;
    if (nkt > 0) {
        load(0);
        store(0);
    }
    __syncthreads();
    for (int kt = 0; kt < nkt; ++kt) {
        const int buf = kt & 1;
        if (kt + 1 < nkt) load(kt + 1);  // global loads in flight during the compute below
#pragma unroll 4
        for (int k = 0; k < GB_BK; ++k) {
            u64 bd[NC];
#pragma unroll
            for (int c2 = 0; c2 < NC; c2 += 2) {
                const int col = (c2 < 4 ? tn * 4 : 64 + tn * 4) + (c2 & 3);
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&sm.b[buf][k][col]);
                bd[c2] = v.x;
                bd[c2 + 1] = v.y;
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const u64 a = *reinterpret_cast<const u64 *>(&sm.a[buf][k][2 * tm + 32 * r]);
#pragma unroll
                for (int c = 0; c < NC; ++c) acc[r][c] = f2_fma(a, bd[c], acc[r][c]);
            }
        }
        if (kt + 1 < nkt) store(buf ^ 1);
        __syncthreads();
    }
    float *out = partial + (int64_t)blockIdx.z * B * n_pad;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int b = n0 + (c < 4 ? tn * 4 : 64 + tn * 4) + (c & 3);
        if (b >= B) continue;
#pragma unroll
        for (int r = 0; r < 4; ++r)
            *reinterpret_cast<u64 *>(out + (int64_t)b * n_pad + m0 + 2 * tm + 32 * r) = acc[r][c];
    }
}

// (K splits, K columns per split) of the GEMM: the split count (at most 16, each split at
// least 64 K steps) whose CTAs best fill whole waves of two CTAs per SM; each extra split
// costs one more B x n partial-sum slot, a small penalty.
static SplitPlan gemm_plan(const nf_operator *op, int B) {
    SplitPlan p{};
    const int bn = B > 64 ? 128 : 64;
    const int64_t tiles = (op->n_pad / GB_BM) * ((B + bn - 1) / bn);
    const int64_t ktiles = op->n_pad / GB_BK;
    const int64_t slots = 2 * (int64_t)num_sms();
    int s = 1;
    double best = -1.0;
    for (int c = 1; c <= 16 && (c == 1 || ktiles / c >= 64); ++c) {
        const int64_t per_c = ceil_div(ktiles, c);
        if (ceil_div(ktiles, per_c) != c) continue;
        const int64_t items = tiles * c;
        const double eff = (double)items / (double)(ceil_div(items, slots) * slots) - 0.005 * c;
        if (eff > best + 1e-9) {
            best = eff;
            s = c;
        }
    }
    const int64_t per = ceil_div(ktiles, s);
    p.rows_per_block = GB_BM;
    p.row_blocks = op->n_pad / GB_BM;
    p.splits = (int)ceil_div(ktiles, per);
    p.jchunk = per * GB_BK;
    return p;
}

// Planes of up to 2,048 padded nodes give the GEMM few tiles: 94 to 140 us per sum for any number of
// trajectories, while a pass of 8 over the plane, which stays in L2, takes 6.  Per sum at
// n = 2,000, passes / GEMM: 64 trajectories 55 / 96 us, 128 105 / 136, 192 154 / 137, 256 203 / 138,
// 512 394 / 142 (n = 700: 52 / 96, 98 / 136, 146 / 136, 192 / 136, 377 / 136).
constexpr int kGemmMinBSmall = 169;
static bool use_gemm(const nf_operator *op, int B) {
    return op->path == NF_DENSE_FP32 && B >= (op->n_pad > 2048 ? kGemmMinB : kGemmMinBSmall);
}

template <int NB>
static cudaError_t sym_gemv_attrs() {
    const int smem = (int)(sym_smem_floats<NB>(SB) * sizeof(float));
    cudaError_t e = cudaFuncSetAttribute(gemv_sym_kernel<NB, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(gemv_sym_kernel<NB, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e;
}

nf_status dense_init_attrs() {
    NF_CUDA_TRY(sym_gemv_attrs<1>());
    NF_CUDA_TRY(sym_gemv_attrs<2>());
    NF_CUDA_TRY(sym_gemv_attrs<4>());
    NF_CUDA_TRY(cudaFuncSetAttribute(gemm_fp32_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(GemmSmem<128>)));
    NF_CUDA_TRY(cudaFuncSetAttribute(gemm_fp32_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(GemmSmem<64>)));
    return NF_OK;
}

// The columns' splits fill whole waves of resident CTAs: two per SM on the FP32 plane, on the bf16 planes four,
// which is two waves of two for several trajectories.  One trajectory there runs three and takes the
// splits that fill these where they are more (n = 8,000: 43 us against 49), but never fewer: the
// chains of FP32 adds would grow (n = 100,000: relative L2 error 5.3e-7 instead of 2.8e-7).
SplitPlan dense_plan(nf_operator *op, int B) {
    const bool fp32 = op->path == NF_DENSE_FP32;
    const SplitPlan p = plan_splits(op->n_pad, DG_ROWS, DG_TILE, fp32 ? 2 : 4);
    if (fp32 || B > 1) return p;
    const SplitPlan three = plan_splits(op->n_pad, DG_ROWS, DG_TILE, 3);
    return three.splits > p.splits ? three : p;
}

int dense_splits(nf_operator *op, int B) {
    if (use_gemm(op, B)) return gemm_plan(op, B).splits;
    const bool sym = op->path == NF_DENSE_SYM_FP32 || op->path == NF_DENSE_SYM_BF16X2;
    return sym ? (int)(op->n_pad / SB) : dense_plan(op, B).splits;
}

size_t dense_sym_entries(int64_t n_pad) {
    const int64_t nb = n_pad / SB;
    return (size_t)(nb * (nb + 1) / 2) * SB * SB;
}

// CTAs per block pair of the symmetric GEMV: enough for one and a half waves of two CTAs per SM, at
// most 8 (a portable cluster).  Per RK4 stage, one CTA per pair before / now: n = 4,000 38.9 /
// 11.0 us, 8,000 81.8 / 27.1, 16,000 104.7 / 97.6; from about 465 pairs (n = 30,000) one CTA per
// pair streams at the HBM limit and the exchange only costs (292.8 us with one, 302.1 with four).
static int sym_slices(int64_t pairs) {
    int S = 1;
    while (S < 8 && pairs * S < 3 * (int64_t)num_sms()) S *= 2;
    return S;
}

template <int NB, bool HL>
static cudaError_t launch_sym_gemv(nf_operator *op, int B, int b0, cudaStream_t s) {
    const int64_t nb = op->n_pad / SB, pairs = nb * (nb + 1) / 2;
    const int S = sym_slices(pairs), rows = SB / S;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)pairs, (unsigned)S, 1);
    cfg.blockDim = dim3(SYM_THREADS, 1, 1);
    cfg.dynamicSmemBytes = sym_smem_floats<NB>(rows) * sizeof(float);
    cfg.stream = s;
    cudaLaunchAttribute attr[2]{};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = (unsigned)S;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = op->profile ? 1 : 2;
    return cudaLaunchKernelEx(&cfg, gemv_sym_kernel<NB, HL>,
                              HL ? static_cast<const void *>(op->Whi) : static_cast<const void *>(op->W32),
                              (const float *)op->g, (const float *)op->rs, op->n_pad, B, b0, rows, op->partial);
}

template <bool HL>
static nf_status launch_sym_gemvs(nf_operator *op, int B, cudaStream_t s) {
    for (int b = 0; b < B;) {  // 3 or 4 trajectories as 4, then 2, then 1
        const int left = B - b;
        if (left >= 3) {
            NF_CUDA_TRY((launch_sym_gemv<4, HL>(op, B, b, s)));
            b += 4;
        } else if (left == 2) {
            NF_CUDA_TRY((launch_sym_gemv<2, HL>(op, B, b, s)));
            b += 2;
        } else {
            NF_CUDA_TRY((launch_sym_gemv<1, HL>(op, B, b, s)));
            b += 1;
        }
    }
    return NF_OK;
}

template <bool HL>
static nf_status launch_gemvs(nf_operator *op, int B, const SplitPlan &pl, cudaStream_t s) {
    const dim3 grid((unsigned)pl.row_blocks, (unsigned)pl.splits);
    const void *W0 = HL ? static_cast<const void *>(op->Whi) : static_cast<const void *>(op->W32);
    auto go = [&](auto kernel, int b) {
        return launch_dependent(kernel, grid, DG_THREADS, 0, s, !op->profile, W0, (const uint16_t *)op->Wlo,
                                (const float *)op->g, op->n_pad, B, b, pl.jchunk, op->partial);
    };
    for (int b = 0; b < B;) {
        const int left = B - b;
        if (left >= 8) {
            NF_CUDA_TRY(go(gemv_kernel<8, HL>, b));
            b += 8;
        } else if (left >= 4) {
            NF_CUDA_TRY(go(gemv_kernel<4, HL>, b));
            b += 4;
        } else if (left == 3) {
            NF_CUDA_TRY(go(gemv_kernel<3, HL>, b));
            b += 3;
        } else if (left == 2) {
            NF_CUDA_TRY(go(gemv_kernel<2, HL>, b));
            b += 2;
        } else {
            NF_CUDA_TRY(go(gemv_kernel<1, HL>, b));
            b += 1;
        }
    }
    return NF_OK;
}

nf_status launch_dense_gemv(nf_operator *op, int B, cudaStream_t s, int *splits_out) {
    if (op->path == NF_DENSE_SYM_FP32 || op->path == NF_DENSE_SYM_BF16X2) {
        if (op->path == NF_DENSE_SYM_FP32)
            NF_TRY(launch_sym_gemvs<false>(op, B, s));
        else
            NF_TRY(launch_sym_gemvs<true>(op, B, s));
        *splits_out = (int)(op->n_pad / SB);
        return NF_OK;
    }
    if (use_gemm(op, B)) {
        const SplitPlan gp = gemm_plan(op, B);
        if (B > 64) {
            dim3 grid((unsigned)gp.row_blocks, (unsigned)((B + 127) / 128), (unsigned)gp.splits);
            gemm_fp32_kernel<128><<<grid, GB_THREADS, sizeof(GemmSmem<128>), s>>>(op->W32, op->g, op->n_pad, B,
                                                                                gp.jchunk, op->partial);
        } else {
            dim3 grid((unsigned)gp.row_blocks, (unsigned)((B + 63) / 64), (unsigned)gp.splits);
            gemm_fp32_kernel<64><<<grid, GB_THREADS, sizeof(GemmSmem<64>), s>>>(op->W32, op->g, op->n_pad, B,
                                                                              gp.jchunk, op->partial);
        }
        NF_CUDA_TRY(cudaGetLastError());
        *splits_out = gp.splits;
        return NF_OK;
    }
    const SplitPlan pl = dense_plan(op, B);
    if (op->path == NF_DENSE_FP32)
        NF_TRY(launch_gemvs<false>(op, B, pl, s));
    else
        NF_TRY(launch_gemvs<true>(op, B, pl, s));
    *splits_out = pl.splits;
    return NF_OK;
}

}  // namespace nfi
