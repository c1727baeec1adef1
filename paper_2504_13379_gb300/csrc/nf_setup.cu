// nf_setup.cu -- stencils (§3.1) on the GPU, in FP64.
//
// Stencils: nodes are binned into a uniform grid; each query point (an element's centroid, or a
// given centre) gathers the nodes of the cells around it until its k nearest, by (distance^2,
// index), cannot lie outside.  All distances that decide use explicitly rounded FP64
// operations (no contraction) in a fixed order, so the selection equals a brute-force FP64
// selection bit for bit.
#include "nf_internal.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace nfi {

constexpr int KNN_KMAX = 128;

// ------------------------------------------------------------------ helpers
__device__ __forceinline__ double dsq(double t) { return __dmul_rn(t, t); }

__device__ __forceinline__ void centroid_of(const double *nodes, int dim, const int32_t *tri, double *c) {
    for (int d = 0; d < dim; ++d) {
        double s = __dadd_rn(nodes[(int64_t)tri[0] * dim + d], nodes[(int64_t)tri[1] * dim + d]);
        s = __dadd_rn(s, nodes[(int64_t)tri[2] * dim + d]);
        c[d] = __ddiv_rn(s, 3.0);
    }
}

__device__ __forceinline__ double exact_d2(const double *x, const double *c, int dim) {
    double s = dsq(__dsub_rn(x[0], c[0]));
    s = __dadd_rn(s, dsq(__dsub_rn(x[1], c[1])));
    if (dim == 3) s = __dadd_rn(s, dsq(__dsub_rn(x[2], c[2])));
    return s;
}

// ------------------------------------------------------------------ input validation
// flag <- 1 if any of the cnt indices is outside [0, n)
__global__ void validate_indices_kernel(const int32_t *idx, int64_t cnt, int64_t n, int *flag) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < cnt && (idx[t] < 0 || idx[t] >= n)) atomicExch(flag, 1);
}

// ------------------------------------------------------------------ grid build
struct Grid {
    double lo[3];
    double h;
    int G[3];
    int64_t ncell;
};

__global__ void bbox_partial_kernel(const double *nodes, int64_t n, int dim, double *out) {
    __shared__ double smin[3][256], smax[3][256];
    double mn[3] = {1e300, 1e300, 1e300}, mx[3] = {-1e300, -1e300, -1e300};
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
        for (int d = 0; d < dim; ++d) {
            const double v = nodes[j * dim + d];
            mn[d] = fmin(mn[d], v);
            mx[d] = fmax(mx[d], v);
        }
    for (int d = 0; d < 3; ++d) {
        smin[d][threadIdx.x] = mn[d];
        smax[d][threadIdx.x] = mx[d];
    }
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if ((int)threadIdx.x < st)
            for (int d = 0; d < 3; ++d) {
                smin[d][threadIdx.x] = fmin(smin[d][threadIdx.x], smin[d][threadIdx.x + st]);
                smax[d][threadIdx.x] = fmax(smax[d][threadIdx.x], smax[d][threadIdx.x + st]);
            }
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int d = 0; d < 3; ++d) {
            out[blockIdx.x * 6 + d] = smin[d][0];
            out[blockIdx.x * 6 + 3 + d] = smax[d][0];
        }
}

__device__ __forceinline__ int cell_coord(double v, double lo, double h, int G) {
    int c = (int)floor((v - lo) / h);
    return c < 0 ? 0 : (c >= G ? G - 1 : c);
}

__global__ void cell_count_kernel(const double *nodes, int64_t n, int dim, Grid gr, int32_t *cell_of,
                                  int32_t *counts) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    int c[3] = {0, 0, 0};
    for (int d = 0; d < dim; ++d) c[d] = cell_coord(nodes[j * dim + d], gr.lo[d], gr.h, gr.G[d]);
    const int32_t id = (int32_t)(((int64_t)c[2] * gr.G[1] + c[1]) * gr.G[0] + c[0]);
    cell_of[j] = id;
    atomicAdd(&counts[id], 1);
}

// Single-block exclusive scan (a few million entries at most): sequential chunks per thread, the
// chunk sums scanned by warps.
__global__ void __launch_bounds__(1024) exclusive_scan_kernel(const int32_t *in, int64_t len, int32_t *out) {
    __shared__ int32_t wsum[32];
    const int T = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t per = (len + T - 1) / T;
    const int64_t b = min(len, threadIdx.x * per), e = min(len, b + per);
    int32_t s = 0;
    for (int64_t i = b; i < e; ++i) s += in[i];
    int32_t inc = s;  // inclusive over the warp, then over the block
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int32_t w = wsum[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t v = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += v;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    int32_t run = inc - s + (warp ? wsum[warp - 1] : 0);
    for (int64_t i = b; i < e; ++i) {
        const int32_t v = in[i];
        out[i] = run;
        run += v;
    }
    if (threadIdx.x == T - 1) out[len] = run;
}

void launch_validate_indices(const int32_t *idx, int64_t cnt, int64_t n, int *flag, cudaStream_t s) {
    validate_indices_kernel<<<(unsigned)ceil_div(cnt, 256), 256, 0, s>>>(idx, cnt, n, flag);
}
void launch_exclusive_scan(const int32_t *in, int64_t len, int32_t *out, cudaStream_t s) {
    exclusive_scan_kernel<<<1, 1024, 0, s>>>(in, len, out);
}

// Nodes by cell, with their FP32 offsets from the grid's corner (for the first rejection).
__global__ void cell_fill_kernel(const double *nodes, int64_t n, int dim, Grid gr, const int32_t *cell_of,
                                 const int32_t *start, int32_t *fill, int32_t *sorted, float4 *sx) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int32_t c = cell_of[j];
    const int32_t pos = start[c] + atomicAdd(&fill[c], 1);
    sorted[pos] = (int32_t)j;
    const double *x = nodes + j * dim;
    sx[pos] = make_float4((float)(x[0] - gr.lo[0]), (float)(x[1] - gr.lo[1]), dim == 3 ? (float)(x[2] - gr.lo[2]) : 0.f, 0.f);
}

// Query points and their cells: the centroids of the triangles, or the given centres.
__global__ void query_kernel(const double *__restrict__ nodes, int dim, const int32_t *__restrict__ tris,
                             const double *__restrict__ centers, int64_t m, Grid gr, double *__restrict__ qc,
                             int4 *__restrict__ qcell) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m) return;
    double c[3] = {0, 0, 0};
    if (centers) {
        for (int d = 0; d < dim; ++d) c[d] = centers[e * dim + d];
    } else {
        centroid_of(nodes, dim, tris + 3 * e, c);
    }
    int cc[3] = {0, 0, 0};
    for (int d = 0; d < dim; ++d) cc[d] = cell_coord(c[d], gr.lo[d], gr.h, gr.G[d]);
    for (int d = 0; d < 3; ++d) qc[3 * e + d] = c[d];
    qcell[e] = make_int4(cc[0], cc[1], cc[2], 0);
}

// One warp per query point.  The cube of cells within rho of the query's cell holds every node
// closer than rho h, so once k nodes lie strictly within that radius they contain the answer;
// until then rho grows.  A cube is swept as runs of x-adjacent cells, which lie next to each
// other in `sorted`: FP32 offsets reject most nodes (with a margin for their rounding), the rest
// get the exact FP64 distance and, if inside the radius, are ranked against each other by
// (distance^2, index), each lane counting the entries before its own.  Against one thread per
// query with its sorted list in local memory: 13 -> 2 ms for 200,000 queries of k = 48.
// Where the radius holds more than KNN_CAP nodes (a refined part of the set: cells are sized for
// the whole) it shrinks, over the cells it still meets, until it holds between k and KNN_CAP:
// any radius up to rho h serves (100,000 planar queries of k = 24, four fifths of the nodes in 1 % of
// the width: 16 ms; one thread per query 337, a warp that gives up first 351).  Queries for
// which there is none (many nodes at one place) are left to knn_query_kernel (their row's first
// entry is -1).
constexpr int KNN_CAP = 512, KNN_WARPS = 4, KNN_SHRINK = 40;
__global__ void __launch_bounds__(32 * KNN_WARPS)
knn_warp_kernel(const double *__restrict__ nodes, int dim, int64_t m, int k, Grid gr, int rho0, double slack,
                const int32_t *__restrict__ start, const int32_t *__restrict__ sorted, const float4 *__restrict__ sx,
                const double *__restrict__ qc, const int4 *__restrict__ qcell, int32_t *__restrict__ stencils,
                int *__restrict__ left) {
    __shared__ unsigned long long keys[KNN_WARPS][KNN_CAP];
    __shared__ int32_t ids[KNN_WARPS][KNN_CAP];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t e = (int64_t)blockIdx.x * KNN_WARPS + warp;
    if (e >= m) return;
    unsigned long long *key = keys[warp];
    int32_t *id = ids[warp];
    const double c[3] = {qc[3 * e], qc[3 * e + 1], qc[3 * e + 2]};
    const int4 cell = qcell[e];
    const float fx = (float)(c[0] - gr.lo[0]), fy = (float)(c[1] - gr.lo[1]), fz = dim == 3 ? (float)(c[2] - gr.lo[2]) : 0.f;
    const int gmax = max(gr.G[0], max(gr.G[1], gr.G[2]));
    constexpr unsigned long long kNone = ~0ull;
    int cnt = 0, valid = 0, rho = rho0;
    bool fits = false;
    double few = 0.0, many = 0.0;  // radii: too few nodes; too many (0: not met yet)
    for (int shrunk = 0; shrunk < KNN_SHRINK;) {
        const bool grow = many == 0.0;
        const bool whole = grow && rho >= gmax;  // the cube covers the grid: every node counts
        const double rad = grow ? (double)rho * gr.h : (few > 0.0 ? sqrt(few * many) : 0.5 * many);
        const double lim2 = whole ? INFINITY : rad * rad * (1.0 - 1e-9);
        const float lim2f = whole ? INFINITY : (float)((rad + slack) * (rad + slack)) * (1.f + 1e-5f);
        int c0[3] = {max(0, cell.x - rho), max(0, cell.y - rho), dim == 3 ? max(0, cell.z - rho) : 0};
        int c1[3] = {min(gr.G[0] - 1, cell.x + rho), min(gr.G[1] - 1, cell.y + rho), dim == 3 ? min(gr.G[2] - 1, cell.z + rho) : 0};
        if (!grow) {
            ++shrunk;
#pragma unroll
            for (int d = 0; d < 3; ++d)
                if (d < dim) {
                    c0[d] = cell_coord(c[d] - rad, gr.lo[d], gr.h, gr.G[d]);
                    c1[d] = cell_coord(c[d] + rad, gr.lo[d], gr.h, gr.G[d]);
                }
        }
        const int x0 = c0[0], x1 = c1[0], y0 = c0[1], z0 = c0[2];
        const int ny = c1[1] - y0 + 1, runs = ny * (c1[2] - z0 + 1);
        cnt = 0;
        for (int rb = 0; rb < runs && cnt <= KNN_CAP; rb += 32) {
            // each lane one run's bounds, then the runs one after another
            int32_t p0 = 0, p1 = 0;
            if (rb + lane < runs) {
                const int z = z0 + (rb + lane) / ny, y = y0 + (rb + lane) % ny;
                const int64_t row = ((int64_t)z * gr.G[1] + y) * gr.G[0];
                p0 = start[row + x0];
                p1 = start[row + x1 + 1];
            }
            unsigned some = __ballot_sync(0xffffffffu, p1 > p0);
            for (; some && cnt <= KNN_CAP; some &= some - 1) {
                const int src = __ffs(some) - 1;
                const int32_t b0 = __shfl_sync(0xffffffffu, p0, src), b1 = __shfl_sync(0xffffffffu, p1, src);
                for (int32_t b = b0; b < b1; b += 32) {
                    bool in = false;
                    if (b + lane < b1) {
                        const float4 s = __ldg(sx + b + lane);
                        const float dx = s.x - fx, dy = s.y - fy, dz = s.z - fz;
                        in = dx * dx + dy * dy + dz * dz <= lim2f;
                    }
                    const unsigned got = __ballot_sync(0xffffffffu, in);
                    const int at = cnt + __popc(got & ((1u << lane) - 1u));
                    if (in && at < KNN_CAP) id[at] = sorted[b + lane];
                    cnt += __popc(got);
                    if (cnt > KNN_CAP) break;
                }
            }
        }
        if (cnt > KNN_CAP) {
            many = rad;
            continue;
        }
        __syncwarp();
        valid = 0;
        for (int i0 = 0; i0 < cnt; i0 += 32) {
            bool ok = false;
            if (i0 + lane < cnt) {
                const double d2 = exact_d2(nodes + (int64_t)id[i0 + lane] * dim, c, dim);
                ok = d2 < lim2;
                key[i0 + lane] = ok ? (unsigned long long)__double_as_longlong(d2) : kNone;  // d2 >= 0: ordered bits
            }
            valid += __popc(__ballot_sync(0xffffffffu, ok));
        }
        __syncwarp();
        fits = valid >= k;
        if (fits || whole) break;
        few = rad;
        if (grow) ++rho;
    }
    if (!fits) {
        if (lane == 0) {
            stencils[e * k] = -1;
            *left = 1;
        }
        return;
    }
    for (int i0 = 0; i0 < cnt; i0 += 128) {  // four entries per lane
        unsigned long long mk[4];
        int32_t mi[4];
        int rank[4] = {0, 0, 0, 0};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int i = i0 + 32 * t + lane;
            mk[t] = i < cnt ? key[i] : kNone;
            mi[t] = i < cnt ? id[i] : 0x7fffffff;
        }
        for (int j = 0; j < cnt; ++j) {
            const unsigned long long kj = key[j];
            const int32_t ij = id[j];
#pragma unroll
            for (int t = 0; t < 4; ++t) rank[t] += (kj < mk[t] || (kj == mk[t] && ij < mi[t])) ? 1 : 0;
        }
#pragma unroll
        for (int t = 0; t < 4; ++t)
            if (mk[t] != kNone && rank[t] < k) stencils[e * k + rank[t]] = mi[t];
    }
}

// The queries that knn_warp_kernel left over, one thread each with an insertion-sorted list.
__global__ void knn_query_kernel(const double *__restrict__ nodes, int64_t n, int dim, int64_t m, int k, Grid gr,
                                 const int32_t *__restrict__ start, const int32_t *__restrict__ sorted,
                                 const double *__restrict__ qc, const int4 *__restrict__ qcell,
                                 int32_t *__restrict__ stencils, const int *__restrict__ left) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m || !*left || stencils[e * k] >= 0) return;
    const double c[3] = {qc[3 * e], qc[3 * e + 1], qc[3 * e + 2]};
    const int4 cell = qcell[e];
    const int cc[3] = {cell.x, cell.y, cell.z};
    double bd[KNN_KMAX];
    int32_t bi[KNN_KMAX];
    int cnt = 0;
    const int gmax = max(gr.G[0], max(gr.G[1], gr.G[2]));
    for (int rho = 0; rho <= gmax; ++rho) {
        const int zr = (dim == 3) ? rho : 0;
        for (int dz = -zr; dz <= zr; ++dz) {
            const int z = cc[2] + dz;
            if (z < 0 || z >= gr.G[2]) continue;
            for (int dy = -rho; dy <= rho; ++dy) {
                const int y = cc[1] + dy;
                if (y < 0 || y >= gr.G[1]) continue;
                for (int dx = -rho; dx <= rho; ++dx) {
                    if (max(abs(dx), max(abs(dy), abs(dz))) != rho) continue;  // shell only
                    const int x = cc[0] + dx;
                    if (x < 0 || x >= gr.G[0]) continue;
                    const int64_t id = ((int64_t)z * gr.G[1] + y) * gr.G[0] + x;
                    for (int32_t p = start[id]; p < start[id + 1]; ++p) {
                        const int32_t j = sorted[p];
                        const double d2 = exact_d2(nodes + (int64_t)j * dim, c, dim);
                        if (cnt == k && !(d2 < bd[k - 1] || (d2 == bd[k - 1] && j < bi[k - 1]))) continue;
                        int pos = (cnt < k) ? cnt : k - 1;
                        while (pos > 0 && (d2 < bd[pos - 1] || (d2 == bd[pos - 1] && j < bi[pos - 1]))) {
                            bd[pos] = bd[pos - 1];
                            bi[pos] = bi[pos - 1];
                            --pos;
                        }
                        bd[pos] = d2;
                        bi[pos] = j;
                        if (cnt < k) ++cnt;
                    }
                }
            }
        }
        // every unvisited node is at least rho * h away from the centroid
        if (cnt == k) {
            const double lim = (double)rho * gr.h;
            if (bd[k - 1] < lim * lim * (1.0 - 1e-9)) break;
        }
    }
    for (int r = 0; r < k; ++r) stencils[e * k + r] = bi[r];
}

}  // namespace nfi

using namespace nfi;

// k nearest nodes to each query point: triangle centroids (tris) or given centres (centers).
// The search grid covers the nodes and, with centres, the centres as well, so that its
// shell-by-shell stopping rule holds for query points outside the nodes' bounding box.
static nf_status build_stencils(const double *nodes, int64_t n, int dim, const int32_t *tris, const double *centers,
                                int64_t m, int k, int32_t *stencils, cudaStream_t s) {
    NF_ARG(dim == 2 || dim == 3, "dim must be 2 or 3 (got %d)", dim);
    NF_ARG(n >= 1 && n < ((int64_t)1 << 31), "n out of range");
    NF_ARG(m >= 1 && m < ((int64_t)1 << 31), "m out of range");
    NF_ARG(k >= 1 && k <= KNN_KMAX && k <= n, "k = %d must satisfy 1 <= k <= min(n, %d)", k, KNN_KMAX);
    // bounding box of the nodes (first nb partials) and of the centres (next nbc)
    const int nb = (int)std::min<int64_t>(256, ceil_div(n, 256));
    const int nbc = centers ? (int)std::min<int64_t>(256, ceil_div(m, 256)) : 0;
    double *dbox = nullptr;
    NF_CUDA_TRY(cudaMallocAsync(&dbox, sizeof(double) * 6 * (nb + nbc) + 16, s));  // box, index flag, left-over flag
    int *dflag = reinterpret_cast<int *>(dbox + 6 * (nb + nbc));
    NF_CUDA_TRY(cudaMemsetAsync(dflag, 0, sizeof(int), s));
    if (tris) launch_validate_indices(tris, 3 * m, n, dflag, s);
    bbox_partial_kernel<<<nb, 256, 0, s>>>(nodes, n, dim, dbox);
    if (centers) bbox_partial_kernel<<<nbc, 256, 0, s>>>(centers, m, dim, dbox + 6 * nb);
    NF_CUDA_TRY(cudaGetLastError());
    std::vector<double> hbox(6 * (nb + nbc));
    int hflag = 0;
    NF_CUDA_TRY(cudaMemcpyAsync(hbox.data(), dbox, sizeof(double) * 6 * (nb + nbc), cudaMemcpyDeviceToHost, s));
    NF_CUDA_TRY(cudaMemcpyAsync(&hflag, dflag, sizeof(int), cudaMemcpyDeviceToHost, s));
    NF_CUDA_TRY(cudaStreamSynchronize(s));
    if (hflag) {
        cudaFreeAsync(dbox, s);
        return fail(NF_ERR_ARG, "tris holds a node index outside [0, n)");
    }
    double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
    for (int b = 0; b < nb + nbc; ++b)
        for (int d = 0; d < 3; ++d) {
            lo[d] = std::min(lo[d], hbox[6 * b + d]);
            hi[d] = std::max(hi[d], hbox[6 * b + 3 + d]);
        }
    for (int d = 0; d < dim; ++d)
        if (!std::isfinite(lo[d]) || !std::isfinite(hi[d])) {
            cudaFreeAsync(dbox, s);
            return fail(NF_ERR_ARG, "non-finite node or centre coordinates");
        }
    Grid gr{};
    double ext = 0.0;
    for (int d = 0; d < dim; ++d) ext = std::max(ext, hi[d] - lo[d]);
    if (!(ext > 0.0)) ext = 1.0;
    const double per = (dim == 3) ? std::cbrt((double)n / 2.0) : std::sqrt((double)n / 4.0);
    gr.h = ext / std::max(1.0, std::floor(per));
    for (int d = 0; d < 3; ++d) {
        gr.lo[d] = (d < dim) ? lo[d] : 0.0;
        gr.G[d] = (d < dim) ? std::max(1, (int)std::ceil((hi[d] - lo[d]) / gr.h) + 1) : 1;
    }
    gr.ncell = (int64_t)gr.G[0] * gr.G[1] * gr.G[2];
    NF_ARG(gr.ncell < ((int64_t)1 << 30), "degenerate node bounding box");
    int32_t *cell_of = nullptr, *counts = nullptr, *start = nullptr, *sorted = nullptr;
    float4 *sx = nullptr;
    double *qc = nullptr;
    int4 *qcell = nullptr;
    NF_CUDA_TRY(cudaMallocAsync(&cell_of, sizeof(int32_t) * n, s));
    NF_CUDA_TRY(cudaMallocAsync(&counts, sizeof(int32_t) * gr.ncell, s));
    NF_CUDA_TRY(cudaMallocAsync(&start, sizeof(int32_t) * (gr.ncell + 1), s));
    NF_CUDA_TRY(cudaMallocAsync(&sorted, sizeof(int32_t) * n, s));
    NF_CUDA_TRY(cudaMallocAsync(&sx, sizeof(float4) * n, s));
    NF_CUDA_TRY(cudaMallocAsync(&qc, sizeof(double) * 3 * m, s));
    NF_CUDA_TRY(cudaMallocAsync(&qcell, sizeof(int4) * m, s));
    int *const left = dflag + 1;
    NF_CUDA_TRY(cudaMemsetAsync(left, 0, sizeof(int), s));
    NF_CUDA_TRY(cudaMemsetAsync(counts, 0, sizeof(int32_t) * gr.ncell, s));
    cell_count_kernel<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(nodes, n, dim, gr, cell_of, counts);
    launch_exclusive_scan(counts, gr.ncell, start, s);
    NF_CUDA_TRY(cudaMemsetAsync(counts, 0, sizeof(int32_t) * gr.ncell, s));
    cell_fill_kernel<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(nodes, n, dim, gr, cell_of, start, counts, sorted, sx);
    query_kernel<<<(unsigned)ceil_div(m, 256), 256, 0, s>>>(nodes, dim, tris, centers, m, gr, qc, qcell);
    // the first radius tried: on flat domains the one that holds about 1.3 k nodes of an even
    // distribution over the bounding box; on surfaces one cell, which holds some 120 nodes
    int rho0 = 1;
    if (dim == 2) {
        const double cells = (hi[0] - lo[0]) * (hi[1] - lo[1]) / (gr.h * gr.h);
        const double r2 = 1.3 * k * cells / (3.14159265358979 * (double)n);
        if (r2 > 1.0) rho0 = (int)std::min(64.0, std::ceil(std::sqrt(r2)));
    }
    // FP32 offsets are off by up to 2^-24 of the grid's extent each, per coordinate and node
    const double rel = 4.0 * 5.97e-8 * (double)std::max(gr.G[0], std::max(gr.G[1], gr.G[2]));
    // Coordinates so large or small that squared FP32 offsets leave FP32's normal range: the rejection
    // would decide wrongly, so every query goes to the thread kernel, which works in FP64 alone.
    if (gr.h > 1e-12 && ext < 1e18) {
        knn_warp_kernel<<<(unsigned)ceil_div(m, KNN_WARPS), 32 * KNN_WARPS, 0, s>>>(
            nodes, dim, m, k, gr, rho0, rel * gr.h, start, sorted, sx, qc, qcell, stencils, left);
    } else {
        NF_CUDA_TRY(cudaMemsetAsync(stencils, 0xff, sizeof(int32_t) * m * k, s));
        NF_CUDA_TRY(cudaMemsetAsync(left, 1, sizeof(int), s));
    }
    knn_query_kernel<<<(unsigned)ceil_div(m, 128), 128, 0, s>>>(nodes, n, dim, m, k, gr, start, sorted, qc, qcell,
                                                                stencils, left);
    NF_CUDA_TRY(cudaGetLastError());
    cudaFreeAsync(cell_of, s);
    cudaFreeAsync(counts, s);
    cudaFreeAsync(start, s);
    cudaFreeAsync(sorted, s);
    cudaFreeAsync(sx, s);
    cudaFreeAsync(qc, s);
    cudaFreeAsync(qcell, s);
    cudaFreeAsync(dbox, s);
    return NF_OK;
}

extern "C" nf_status nf_build_stencils(const double *nodes, int64_t n, int dim, const int32_t *tris, int64_t m,
                                       int k, int32_t *stencils, void *stream) {
    clear_error();
    NF_ARG(nodes && tris && stencils, "nodes, tris and stencils must be non-NULL");
    return build_stencils(nodes, n, dim, tris, nullptr, m, k, stencils, as_stream(stream));
}

extern "C" nf_status nf_build_stencils_at(const double *nodes, int64_t n, int dim, const double *centers, int64_t m,
                                          int k, int32_t *stencils, void *stream) {
    clear_error();
    NF_ARG(nodes && centers && stencils, "nodes, centers and stencils must be non-NULL");
    return build_stencils(nodes, n, dim, nullptr, centers, m, k, stencils, as_stream(stream));
}
