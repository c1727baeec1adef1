// nf_adjoint.cu -- discrete adjoint of the RK4 map of nf_rk4_advance (matrix-free).
//
// One RK4 step (b = (1, 2, 2, 1) / 6, c = (1/2, 1/2, 1) for U_{s+1} = u + c_s dt k_s)
// is reversed stage by stage:
//     nu_4 = dt b_4 lam,                mu_s = J(U_s)^T nu_s = -nu_s + q o f'(U_s) o (W nu_s),
//     nu_s = dt b_s lam + c_s dt mu_{s+1}  (s = 3, 2, 1),
//     lam <- lam + mu_1 + mu_2 + mu_3 + mu_4,
// with W symmetric because the kernel is radial.  Kernel-parameter gradients add
//     <nu_s, (d_theta W) (q o f(U_s))>,  d w / dA1 = e1, d w / ds1 = 2 A1 r^2 e1 / s1^3,
//     d w / dA2 = -e2,  d w / ds2 = -2 A2 r^2 e2 / s2^3.
// The adjoint pair kernel (adj_sym_kernel, with the forward symmetric kernel's block-pair
// schedule: each unordered pair evaluated once) computes W nu as partial-slot sums and the
// four parameter sums sum_ij nu_i g_j (e1, r^2 e1, e2, r^2 e2) as per-CTA partials.  The
// epilogue adds the slots, applies the recurrences and prepares (nu, g) of the next stage;
// a fixed-order FP64 reduction accumulates the parameter gradients.  Stage inputs are
// recomputed segment by segment from checkpoints, on a second stream: while segment k is
// reversed on the caller's stream, segment k - 1 is recomputed into the other of two stage
// buffers, so each launch's last, partly filled wave and the small elementwise kernels of
// one stream overlap the other's pair kernels.  The results do not depend on the overlap
// (every kernel's summation order is fixed).
#include "nf_internal.cuh"

#include <algorithm>

namespace nfi {

__device__ __forceinline__ float sigmoid_rate(float u, float beta, float theta) {
    return 1.0f / (1.0f + expf(-beta * (u - theta)));
}

// The adjoint state (lam, acc, nu, the stage inputs) lives in the operator's node order; only
// lambda_T, the checkpoints and grad_u0 are in the caller's.
__global__ void adj_gather_kernel(const float *__restrict__ src, const int *__restrict__ perm, int64_t n, int B,
                                  float *__restrict__ dst) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)B * n) return;
    const int64_t b = idx / n;
    dst[idx] = src[b * n + perm[idx - b * n]];
}

// nu[b, i] = dt b4 lam_i, g[b, i] = q_i f(U_i)  -- entering the last stage of a step
__global__ void adj_prep_kernel(const float *__restrict__ lam, const float *__restrict__ U, const float *__restrict__ q,
                                const float *__restrict__ beta, const float *__restrict__ theta, int64_t n,
                                int64_t n_pad, int B, float dtb4, float *__restrict__ nu, float *__restrict__ g) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)B * n) return;
    const int b = (int)(idx / n);
    const int64_t i = idx - (int64_t)b * n;
    nu[(int64_t)b * n_pad + i] = dtb4 * lam[idx];
    g[(int64_t)b * n_pad + i] = q[i] * sigmoid_rate(U[idx], beta[b], theta[b]);
}

struct AdjEpiArgs {
    const float *wpart;      // [slots][B][n_pad]: partial sums of W nu
    int slots;
    int64_t n, n_pad;
    int B;
    int stg;                 // 0..3 (stage s = stg + 1)
    const float *Ucur;       // U_s
    const float *Uprev;      // U_{s-1} (stg > 0), U_4 of the previous step (stg == 0), or null
    float *lam, *acc;
    float *nu, *g;           // B x n_pad each
    const float *q, *beta, *theta;
    const int *perm;         // caller's node of each position
    float *out;              // dL/du_0 in the caller's order (the last stage of all), or null
    float dt;
};

// gk[b][k] += scale[k] * sum_c gpart[b][c][k] over the CTAs c of the stage's pair launch, in a fixed
// order.  scale = (1, 2 A1 / s1^3 * r2phys, -1, -2 A2 / s2^3 * r2phys): d w / dA1 = e1,
// d w / ds1 = 2 A1 r^2 e1 / s1^3, d w / dA2 = -e2, d w / ds2 = -2 A2 r^2 e2 / s2^3, with r^2
// converted from exponent units.
struct AdjScale {
    double k[4];
};

// Epilogue of a stage (blocks 0 .. eblocks - 1: one node per thread) and the parameter sums (blocks
// eblocks + 4 b + k), in one launch: the sums are a chain of FP64 adds that the epilogue hides.
__global__ void __launch_bounds__(256)
adj_epilogue_kernel(AdjEpiArgs a, int eblocks, const float *gpart, int64_t ncta, AdjScale sc, double *gk) {
    if ((int)blockIdx.x >= eblocks) {
        __shared__ double red[256];
        const int out = (int)blockIdx.x - eblocks, b = out >> 2, k = out & 3;
        const float *c = gpart + (int64_t)b * ncta * 4 + k;
        pdl_wait();
        double s = 0.0;
        for (int64_t i = threadIdx.x; i < ncta; i += blockDim.x) s += (double)c[i * 4];
        red[threadIdx.x] = s;
        __syncthreads();
        for (int st = blockDim.x / 2; st > 0; st >>= 1) {
            if ((int)threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
            __syncthreads();
        }
        if (threadIdx.x == 0) gk[out] += sc.k[k] * red[0];
        return;
    }
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = idx < (int64_t)a.B * a.n;
    const int b = in ? (int)(idx / a.n) : 0;
    const int64_t i = in ? idx - (int64_t)b * a.n : 0;
    const int64_t vi = (int64_t)b * a.n_pad + i;
    pdl_wait();
    pdl_trigger();
    if (!in) return;
    const float Wnu = sum_slots(a.wpart + (int64_t)b * a.n_pad + i, (int64_t)a.B * a.n_pad, a.slots);
    const float nu = a.nu[vi];
    const float bb = a.beta[b], th = a.theta[b];
    const float f = sigmoid_rate(a.Ucur[idx], bb, th);
    const float fp = a.q[i] * bb * f * (1.f - f);
    const float mu = -nu + fp * Wnu;
    const float bw[4] = {1.f / 6.f, 2.f / 6.f, 2.f / 6.f, 1.f / 6.f};
    const float cprev[4] = {0.f, 0.5f, 0.5f, 1.f};
    if (a.stg > 0) {
        const float accv = (a.stg == 3) ? mu : a.acc[idx] + mu;
        a.acc[idx] = accv;
        const float nun = a.dt * bw[a.stg - 1] * a.lam[idx] + cprev[a.stg] * a.dt * mu;
        a.nu[vi] = nun;
        a.g[vi] = a.q[i] * sigmoid_rate(a.Uprev[idx], bb, th);
    } else {
        const float lamn = a.lam[idx] + (a.acc[idx] + mu);
        a.lam[idx] = lamn;
        if (a.out) a.out[(int64_t)b * a.n + a.perm[i]] = lamn;
        if (a.Uprev) {
            a.nu[vi] = a.dt * bw[3] * lamn;
            a.g[vi] = a.q[i] * sigmoid_rate(a.Uprev[idx], bb, th);
        }
    }
}

__global__ void adj_finish_kernel(const double *__restrict__ gk, int cnt, float *__restrict__ out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < cnt) out[t] = (float)gk[t];
}

// Stream-ordered scratch buffers of one call, released on every return path (an early
// return after a failed launch or allocation frees what was allocated before it).
struct StreamScratch {
    cudaStream_t s;
    void *p[8] = {};
    int count = 0;
    explicit StreamScratch(cudaStream_t st) : s(st) {}
    StreamScratch(const StreamScratch &) = delete;
    StreamScratch &operator=(const StreamScratch &) = delete;
    template <typename T>
    cudaError_t alloc(T **out, size_t bytes) {
        *out = nullptr;
        if (count == 8) return cudaErrorInvalidValue;
        void *q = nullptr;
        const cudaError_t e = cudaMallocAsync(&q, bytes, s);
        if (e != cudaSuccess) return e;
        p[count++] = q;
        *out = static_cast<T *>(q);
        return cudaSuccess;
    }
    ~StreamScratch() {
        for (int i = 0; i < count; ++i) cudaFreeAsync(p[i], s);
    }
};

// A second stream forked from the caller's, on which checkpoint segments are recomputed
// while the previous segment is reversed on the caller's stream.  Events: fork, join, and per
// stage buffer "recomputed" and "reversed".  The destructor joins the side stream back into
// the caller's stream (on every return path, before the scratch buffers are released), so
// the call stays stream-ordered on the caller's stream as a whole.
struct SideStream {
    cudaStream_t main, side = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr, rec[2] = {}, rev[2] = {};
    bool forked = false;
    explicit SideStream(cudaStream_t m) : main(m) {}
    SideStream(const SideStream &) = delete;
    SideStream &operator=(const SideStream &) = delete;
    cudaError_t start() {
        cudaError_t e = cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking);
        cudaEvent_t *evs[6] = {&fork, &join, &rec[0], &rec[1], &rev[0], &rev[1]};
        for (int i = 0; i < 6 && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(evs[i], cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventRecord(fork, main);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(side, fork, 0);
        forked = e == cudaSuccess;
        return e;
    }
    ~SideStream() {
        if (forked && cudaEventRecord(join, side) == cudaSuccess) cudaStreamWaitEvent(main, join, 0);
        cudaEvent_t evs[6] = {fork, join, rec[0], rec[1], rev[0], rev[1]};
        for (cudaEvent_t ev : evs)
            if (ev) cudaEventDestroy(ev);
        if (side) cudaStreamDestroy(side);
    }
};

}  // namespace nfi

using namespace nfi;

extern "C" nf_status nf_adjoint(nf_operator *op, const float *ckpt, int C, int B, double t0, double dt, int nsteps,
                                const float *beta, const float *theta, const nf_forcing *g, const float *lambda_T,
                                float *grad_u0, float *grad_kernel, void *stream) {
    clear_error();
    NF_ARG(op, "op is NULL");
    NF_ARG(ckpt && beta && theta && lambda_T && grad_u0 && grad_kernel, "array arguments must be non-NULL");
    NF_ARG(B >= 1 && B <= 65535 && C >= 1 && nsteps >= 0, "B, C or nsteps out of range");
    if (op->path != NF_MATRIX_FREE)
        return fail(NF_ERR_UNSUPPORTED, "nf_adjoint needs a matrix-free operator (W^T is applied on the fly)");
    if (g && (g->kind == NF_FORCE_MMS_FLAT || g->kind == NF_FORCE_MMS_SPHERE))
        return fail(NF_ERR_UNSUPPORTED, "this manufactured forcing depends on the kernel parameters; nf_adjoint "
                                        "treats forcing as data and does not differentiate it");
    if (g && g->kind != NF_FORCE_NONE && g->kind != NF_FORCE_MMS_EIGEN) return fail(NF_ERR_ARG, "unknown forcing");
    if (g && g->kind == NF_FORCE_MMS_EIGEN) NF_ARG(g->Y1 && g->Y2, "forcing: Y1 and Y2 are required");
    cudaStream_t s = as_stream(stream);
    const int64_t n = op->n, n_pad = op->n_pad;
    const size_t BN = (size_t)B * n;
    NF_TRY(ensure_workspace(op, B, mf_splits(op, B), s));
    // block-pair culling (nf_operator_mf_cull): the adjoint kernel runs over its own live
    // pairs, and each node's live W nu slots are added into slot 0 before the epilogue
    const bool cull = op->mf_cull && op->adj_pairs;
    const int Cseg = std::min(C, std::max(nsteps, 1));
    float *stages = nullptr, *lam = nullptr, *acc = nullptr, *wpart = nullptr, *gpart = nullptr;
    float *nu = nullptr;
    double *gk = nullptr;
    StreamScratch scratch(s);  // freed (stream-ordered) on every return below
    // two stage buffers: segment k - 1 is recomputed into one while segment k is reversed
    // from the other
    const size_t seg_elems = BN * 4 * (size_t)Cseg;
    NF_CUDA_TRY(scratch.alloc(&stages, sizeof(float) * 2 * seg_elems));
    NF_CUDA_TRY(scratch.alloc(&lam, sizeof(float) * BN));
    NF_CUDA_TRY(scratch.alloc(&acc, sizeof(float) * BN));
    // W nu slots and parameter partials for the smallest node block the kernel may take
    NF_CUDA_TRY(scratch.alloc(&wpart, sizeof(float) * (size_t)adj_slot_capacity(op) * B * n_pad));
    NF_CUDA_TRY(scratch.alloc(&gpart, sizeof(float) * 4 * (size_t)B * adj_pair_capacity(op)));
    const size_t BP = (size_t)B * n_pad;
    NF_CUDA_TRY(scratch.alloc(&nu, sizeof(float) * 2 * BP));
    float *const gv = nu + BP;
    NF_CUDA_TRY(scratch.alloc(&gk, sizeof(double) * 4 * B));
    NF_CUDA_TRY(cudaMemsetAsync(nu, 0, sizeof(float) * 2 * BP, s));  // padded columns stay zero
    NF_TRY(adj_autotune(op, nu, gv, B, wpart, gpart, s));  // first call on this operator only
    const int slots = adj_slots(op);  // one W nu slot per node block of the chosen shape
    const int64_t ncta = adj_pair_count(op);
    const int64_t ncta_run = cull ? op->adj_live : ncta;
    NF_CUDA_TRY(cudaMemsetAsync(gk, 0, sizeof(double) * 4 * B, s));
    static const nf_forcing none{NF_FORCE_NONE, nullptr, nullptr, 0, 0, 0, 0, 0, 0, 0, 0};
    const nf_forcing F = g ? *g : none;
    const nf_kernel &kp = op->kp;
    const int T = 256;
    const unsigned eg = (unsigned)ceil_div((int64_t)BN, T);
    adj_gather_kernel<<<eg, T, 0, s>>>(lambda_T, op->perm, n, B, lam);
    NF_CUDA_TRY(cudaGetLastError());
    const int nseg = (nsteps + C - 1) / C;
    // ---- recompute segment seg forward into st, keeping every stage input (stream ss)
    auto recompute = [&](int seg, float *st, cudaStream_t ss) -> nf_status {
        const int s0 = seg * C;
        const int cnt = std::min(C, nsteps - s0);
        NF_TRY(launch_prep_g(op, ckpt + (size_t)seg * BN, B, beta, theta, true, ss));
        NF_TRY(launch_set_clock(op, t0 + (double)s0 * dt, ss));
        // the first stage input is the state itself; every stage kernel leaves the next one
        NF_CUDA_TRY(cudaMemcpyAsync(st, op->U, sizeof(float) * BN, cudaMemcpyDeviceToDevice, ss));
        for (int j = 0; j < cnt; ++j) {
            for (int stage = 1; stage <= 4; ++stage) {
                StageParams p{};
                p.u = nullptr;  // the state advances inside the operator only
                p.beta = beta;
                p.theta = theta;
                p.forcing = F;
                p.dt = dt;
                p.stage = stage;
                p.ckpt = nullptr;
                p.C = 1;
                p.overlap = true;
                // the segment's last state is the next checkpoint: computed for its check alone
                if (stage < 4 || j + 1 < cnt) p.stage_out = st + ((size_t)j * 4 + stage) * BN;
                // the forward run's kernels: the stage inputs are its own to the last bit
                if (fused_fits(op, B) && F.kind == NF_FORCE_NONE) {
                    NF_TRY(fused_stage(op, B, p, ss));
                    continue;
                }
                NF_TRY(launch_mf_pair(op, B, ss, &p.splits));
                NF_TRY(launch_stage(op, B, p, ss));
            }
        }
        return NF_OK;
    };
    SideStream side(s);  // joined into s before the scratch buffers are released
    if (nseg > 0) {
        NF_CUDA_TRY(side.start());
        NF_TRY(recompute(nseg - 1, stages + (size_t)((nseg - 1) & 1) * seg_elems, side.side));
        NF_CUDA_TRY(cudaEventRecord(side.rec[(nseg - 1) & 1], side.side));
    }
    for (int seg = nseg - 1; seg >= 0; --seg) {
        const int cnt = std::min(C, nsteps - seg * C);
        const int bufi = seg & 1;
        // the next segment back is recomputed on the side stream while this one is reversed;
        // its buffer was last read by the reverse pass of segment seg + 1
        if (seg >= 1) {
            if (seg + 1 < nseg) NF_CUDA_TRY(cudaStreamWaitEvent(side.side, side.rev[(seg + 1) & 1], 0));
            NF_TRY(recompute(seg - 1, stages + (size_t)((seg - 1) & 1) * seg_elems, side.side));
            NF_CUDA_TRY(cudaEventRecord(side.rec[(seg - 1) & 1], side.side));
        }
        NF_CUDA_TRY(cudaStreamWaitEvent(s, side.rec[bufi], 0));
        float *const segst = stages + (size_t)bufi * seg_elems;
        // ---- reverse through the segment
        adj_prep_kernel<<<eg, T, 0, s>>>(lam, segst + ((size_t)(cnt - 1) * 4 + 3) * BN, op->q, beta, theta, n,
                                         n_pad, B, (float)(dt / 6.0), nu, gv);
        NF_CUDA_TRY(cudaGetLastError());
        for (int j = cnt - 1; j >= 0; --j) {
            for (int stg = 3; stg >= 0; --stg) {
                float r2phys = 1.f;
                for (int b = 0; b < B; ++b) {
                    NF_TRY(launch_adj_sym(op, nu, gv, B, b, wpart, gpart, &r2phys, s));
                    if (cull) NF_TRY(launch_adj_cull_reduce(op, wpart, B, b, s));
                }
                AdjEpiArgs ea{};
                ea.wpart = wpart;
                ea.slots = cull ? 1 : slots;
                ea.n = n;
                ea.n_pad = n_pad;
                ea.B = B;
                ea.stg = stg;
                ea.Ucur = segst + ((size_t)j * 4 + stg) * BN;
                ea.Uprev = (stg > 0) ? segst + ((size_t)j * 4 + stg - 1) * BN
                                     : (j > 0 ? segst + ((size_t)(j - 1) * 4 + 3) * BN : nullptr);
                ea.lam = lam;
                ea.acc = acc;
                ea.nu = nu;
                ea.g = gv;
                ea.perm = op->perm;
                ea.out = (seg == 0 && j == 0 && stg == 0) ? grad_u0 : nullptr;
                ea.q = op->q;
                ea.beta = beta;
                ea.theta = theta;
                ea.dt = (float)dt;
                AdjScale sc{{1.0, 2.0 * kp.A1 / ((double)kp.s1 * kp.s1 * kp.s1) * r2phys, -1.0,
                             -2.0 * kp.A2 / ((double)kp.s2 * kp.s2 * kp.s2) * r2phys}};
                NF_CUDA_TRY(launch_dependent(adj_epilogue_kernel, dim3(eg + 4 * (unsigned)B), T, 0, s, true, ea, (int)eg,
                                             (const float *)gpart, ncta_run, sc, gk));
            }
        }
        NF_CUDA_TRY(cudaEventRecord(side.rev[bufi], s));  // segst may now be overwritten
    }
    if (nsteps == 0) NF_CUDA_TRY(cudaMemcpyAsync(grad_u0, lambda_T, sizeof(float) * BN, cudaMemcpyDeviceToDevice, s));
    adj_finish_kernel<<<(unsigned)ceil_div(4 * B, 256), 256, 0, s>>>(gk, 4 * B, grad_kernel);
    NF_CUDA_TRY(cudaGetLastError());
    return NF_OK;
}
