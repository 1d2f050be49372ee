// PC-LSQR on the device: preconditioner, LSQR vector updates with the
// scalar recurrences kept on the GPU, and the CUDA graph of one whole solve.
//
// Mathematics (Paige & Saunders 1982, "Algorithm LSQR", damp = 0) on the
// column-scaled matrix Ap = A diag(p) of the paper's PC-LSQR (§2, §3):
//   beta_1 u_1 = b, alpha_1 v_1 = Ap^T u_1, w_1 = v_1, z_0 = 0,
//   phibar_1 = beta_1, rhobar_1 = alpha_1; per iteration i:
//   beta_{i+1} u_{i+1} = Ap v_i - alpha_i u_i
//   alpha_{i+1} v_{i+1} = Ap^T u_{i+1} - beta_{i+1} v_i
//   rho = sqrt(rhobar^2 + beta^2), c = rhobar/rho, s = beta/rho,
//   theta = s alpha_{i+1}, rhobar = -c alpha_{i+1}, phi = c phibar,
//   phibar = s phibar, z += (phi/rho) w, var += (w/rho)^2,
//   w = v_{i+1} - (theta/rho) w.
// The matrix values are never rescaled: Ap v = A (p o v) and
// Ap^T u = p o (A^T u), so the row kernels gather vp = p o v and the vector
// kernel applies p to A^T u.
//
// Neither u nor v is normalised in memory; scalars carry the scales.  The
// stored vectors are U_{i+1} = alpha_i beta_{i+1} u_{i+1} and
// V_i = alpha_i v_i (alpha_0 = 1), so
//   U_{i+1} = A (p o V_i) + cy U_i,    cy = -alpha_i^2 / (alpha_{i-1} beta_i),
//   beta_{i+1} = ||U_{i+1}|| / alpha_i,
//   V_{i+1} = (p o A^T U_{i+1}) / (alpha_i beta_{i+1}) - (beta_{i+1}/alpha_i) V_i,
//   alpha_{i+1} = ||V_{i+1}||,  w_i = V_i / alpha_i - (theta_i/rho_{i-1}) w_{i-1}.
// One vector pass per iteration therefore does what the normalisation and
// the w update would otherwise need a second pass for.
//
// One iteration = aprod 1 (+ ||U||^2; its last block derives beta, 1/beta,
// 1/rho, phi/rho), aprod 2 (single launch + combine), and the vector pass
// (w_i, z, var, V_{i+1}, p o V_{i+1}, three norms; its last block advances
// the recurrences and applies the stopping rules).  The loop is a
// conditional WHILE graph node whose flag that last block clears when LSQR
// stops.
#include <cuda_runtime.h>
#include <math.h>

#include "gsr_internal.cuh"
#include "gsr_lsqr.cuh"
#include "gsr_reduce.cuh"
#include "gsr_split.cuh"

namespace gsr {


__device__ __forceinline__ int64_t gtid() { return blockIdx.x * (int64_t)blockDim.x + threadIdx.x; }
__device__ __forceinline__ int64_t gstride() { return (int64_t)gridDim.x * blockDim.x; }

// p_j = 1/sqrt(sum of squares), 1 for an empty column (in place)
__global__ void k_precond_finish(double *p, int64_t n)
{
    for (int64_t j = gtid(); j < n; j += gstride()) {
        const double s = p[j];
        p[j] = (s > 0.0) ? 1.0 / sqrt(s) : 1.0;
    }
}

__global__ void k_zero(double *a, int64_t n)
{
    for (int64_t j = gtid(); j < n; j += gstride())
        a[j] = 0.0;
}

// u~ = b, beta_1 = ||b||; state reset
__global__ void __launch_bounds__(kThreads)
k_init_u(const SolveArgs *args, double *u, int64_t m, SolveState *st, double *partial,
         unsigned *counter)
{
    const double *b = args->b;
    double acc[1] = {0.0};
    for (int64_t i = gtid(); i < m; i += gstride()) {
        const double bi = b[i];
        u[i] = bi;
        acc[0] = fma(bi, bi, acc[0]);
    }
    if (grid_reduce<1>(acc, partial, counter) && threadIdx.x == 0) {
        SolveState s = {};
        s.beta = sqrt(acc[0]);
        s.bnorm = s.beta;
        s.rnorm = s.beta;
        s.nonfinite = !isfinite(s.beta);
        s.ib = (s.beta > 0.0) ? 1.0 / s.beta : 0.0;
        s.bnext = s.beta;
        s.ia = 1.0;  // alpha_0 = 1: U_1 = b
        *st = s;
    }
}

// Start of the recurrences once alpha_1 = ||V_1|| is known: rhobar_1 =
// alpha_1, phibar_1 = beta_1; istop = 0 when alpha_1 beta_1 = 0 (x = 0 is
// exact).  Thread 0 of the last block of the first vector pass.
__device__ void init_scalars(SolveState *st, const SolveArgs *args, double vnorm2,
                             cudaGraphConditionalHandle loop, int in_graph)
{
    const double beta = st->beta;
    const double alpha = sqrt(vnorm2);
    st->alpha = alpha;
    st->rhobar = alpha;
    st->phibar = beta;
    st->arnorm = alpha * beta;
    st->t = beta * args->isdof;
    st->cy = -alpha * alpha * st->ib;  // -alpha_1^2 / (alpha_0 beta_1)
    st->ia = (alpha > 0.0) ? 1.0 / alpha : 1.0;
    st->theta = 0.0;  // W_0 = 0: the first W update takes no old W
    if (!isfinite(alpha) || st->nonfinite) {
        st->nonfinite = 1;
        st->istop = kIstopNonfinite;
        st->done = 1;
    } else if (alpha * beta == 0.0) {
        st->istop = 0;
        st->done = 1;
    }
    if (st->done && in_graph)
        cudaGraphSetConditional(loop, 0u);
}

// The vector pass of iteration i (first: the start, V_1 = p o A^T b / beta_1
// with w, z, var cleared).  The stored w is W_i = w_i / rho_i of the paper's
// recurrence, which takes the division by rho out of three updates:
//   W_i = V_i / (alpha_i rho_i) - (theta_i / rho_i) W_{i-1},
//   var += W_i^2,  z_i = z_{i-1} + phi_i W_i,
// then V_{i+1} (in place), vp = p o V_{i+1}, and the reductions
// ||V_{i+1}||^2, sum W_i^2, ||z_i||^2.  When beta_{i+1} = 0 V is kept (alpha
// unchanged).  The three sums of squares accumulate on the binary32 pipes
// from exact splits (acc3_sqr: within about 2^-60 of the exact sum; values
// outside the split window in binary64), so an element costs 8 FP64
// operations, the ones that produce stored values.
// INL: q holds only the astrometric part of A^T U (single-launch aprod 2);
// the other columns come from its partial sums, and the global column from
// one fixed slice of the per-unit partials per block, added by the last
// block, which also updates V at the global column.  Otherwise q is complete
// and its non-astrometric part is cleared for the next aprod 2.
template <bool INL>
__global__ void __launch_bounds__(kThreads)
k_vec(const SysView A, const double *__restrict__ p, double *__restrict__ q, double *__restrict__ v,
      double *__restrict__ vp, double *__restrict__ w, double *__restrict__ z,
      double *__restrict__ var, SolveState *st, const SolveArgs *args, double *partial,
      unsigned *counter, cudaGraphConditionalHandle loop, int in_graph, int first, A2Parts P,
      const int *kerr)
{
    const int64_t n = A.n, att0 = A.att0, glb0 = A.glb0;
    const bool late = threadIdx.x == 0 && wait_expired(kerr);
    const VecCoef k = vec_coef(st, first);
    const VecPass X = {p, v, vp, w, z, var};
    VecSums S;
    double gacc = 0.0;
    // an instrument with many window totals is summed by a warp, which then
    // updates its column
    const bool warp_instr = INL && P.isplit > kThreadParts;
    if (warp_instr) {
        for (int64_t f = gtid() >> 5; f < A.I; f += gstride() >> 5) {
            double t = 0.0;
            for (int qq = threadIdx.x & 31; qq < P.isplit; qq += 32)
                t += P.ipart[(int64_t)qq * A.I + f];
            t = warp_sum(t);
            if ((threadIdx.x & 31) == 0)
                vec_column(X, k, S, A.ins0 + f, false, [&] { return t; });
        }
    }
#pragma unroll 2
    for (int64_t j = gtid(); j < n; j += gstride()) {
        if (INL) {
            if (warp_instr && j >= A.ins0 && j < glb0)
                continue;
            vec_column(X, k, S, j, j == glb0, [&] {
                return (j < att0) ? q[j] : (j < glb0 ? q_from_parts(A, P, j) : 0.0);
            });
        } else {
            vec_column(X, k, S, j, false, [&] {
                const double qj = q[j];
                if (j >= att0)
                    q[j] = 0.0;
                return qj;
            });
        }
    }
    if (INL) {  // this block's fixed slice of the global-column partials
        const uint32_t per = ((uint32_t)P.ngpart + gridDim.x - 1) / gridDim.x;
        const uint32_t b0 = blockIdx.x * per;
        const uint32_t b1 = min((uint32_t)P.ngpart, b0 + per);
        for (uint32_t b = b0 + threadIdx.x; b < b1; b += blockDim.x)
            gacc += P.gpart[b];
    }
    double acc[4];
#pragma unroll
    for (int i = 0; i < 3; i++)
        acc[i] = S.total(i);
    acc[3] = gacc;
    if (grid_reduce<4>(acc, partial, counter)) {
        __shared__ double vn2;
        if (threadIdx.x == 0) {
            vn2 = acc[0];
            if (INL) {
                const double vo = first ? 0.0 : v[glb0];
                const double pj = p[glb0];
                const double vn = k.upd ? fma(pj * acc[3], k.k1, k.k2 * vo) : vo;
                v[glb0] = vn;
                vp[glb0] = pj * vn;
                vn2 = fma(vn, vn, vn2);
                *P.ctr = 0ull;  // work counter of the single-launch aprod 2
            }
        }
        __syncthreads();
        if (first) {
            if (threadIdx.x == 0)
                init_scalars(st, args, vn2, loop, in_graph);
        } else {
            lsqr_scalars(st, args, vn2, acc[1], acc[2], late, loop, in_graph);
        }
    }
}

// blocks of the LSQR vector pass: two per SM (measured on the medium
// workload, in the solve: 32.9 us against 33.4 us with three and 37.2 us
// with one; more blocks add per-block reductions), no more than the vector
// needs
int lsqr_vec_grid(const gsr_handle_t *h)
{
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_vec<true>, kThreads, 0) != cudaSuccess ||
        occ < 1)
        return -1;
    if (occ > 2)
        occ = 2;
    int64_t g = (int64_t)h->nsm * occ;
    const int64_t need = (h->sys.n + kThreads - 1) / kThreads;
    if (g > need) g = need;
    if (g > kMaxPartials) g = kMaxPartials;
    return (int)(g < 1 ? 1 : g);
}

// x = p o z, se = p o sqrt(var) * rnorm / sqrt(dof)
__global__ void k_finalize(const double *__restrict__ p, const double *__restrict__ z,
                           const double *__restrict__ var, int64_t n, int64_t m,
                           const SolveState *st, const SolveArgs *args)
{
    double *x = args->x;
    double *se = args->se;
    const double t = st->t;
    for (int64_t j = gtid(); j < n; j += gstride()) {
        x[j] = p[j] * z[j];
        if (se)
            se[j] = p[j] * t * sqrt(var[j]);
    }
}

cudaError_t launch_precond_finish(const gsr_handle_t *h, double *p, cudaStream_t st)
{
    k_precond_finish<<<h->grid_vec, kThreads, 0, st>>>(p, h->sys.n);
    return cudaGetLastError();
}

// column sums of squares -> p (the non-astrometric part must start at zero)
static cudaError_t enqueue_precond(const gsr_handle_t *h, double *p, cudaStream_t st)
{
    const int64_t n = h->sys.n, att0 = h->sys.att0;
    k_zero<<<h->grid_vec, kThreads, 0, st>>>(p + att0, n - att0);
    cudaError_t e = launch_aprod2(h, nullptr, p, kA2Squares, st);
    if (e != cudaSuccess)
        return e;
    return launch_precond_finish(h, p, st);
}

cudaError_t enqueue_precondition(const gsr_handle_t *h, double *p, cudaStream_t st)
{
    return enqueue_precond(h, p, st);
}

cudaError_t find_graph_leaf(cudaGraph_t g, cudaGraphNode_t *leaf)
{
    size_t nn = 0;
    cudaError_t e = cudaGraphGetNodes(g, nullptr, &nn);
    if (e != cudaSuccess || nn == 0)
        return e != cudaSuccess ? e : cudaErrorInvalidValue;
    cudaGraphNode_t *nodes = new cudaGraphNode_t[nn];
    e = cudaGraphGetNodes(g, nodes, &nn);
    int found = 0;
    for (size_t i = 0; e == cudaSuccess && i < nn; i++) {
        size_t nd = 0;
        e = cudaGraphNodeGetDependentNodes(nodes[i], nullptr, nullptr, &nd);
        if (e == cudaSuccess && nd == 0) {
            *leaf = nodes[i];
            found++;
        }
    }
    delete[] nodes;
    if (e == cudaSuccess && found != 1)
        e = cudaErrorInvalidValue;
    return e;
}

#define GSR_TRY(x)                      \
    do {                                \
        cudaError_t e_ = (x);           \
        if (e_ != cudaSuccess) {        \
            err = e_;                   \
            goto fail;                  \
        }                               \
    } while (0)

// q = A^T U (overwrite) and the vector pass; with the single-launch aprod 2
// the vector pass combines its partial sums itself
[[nodiscard]] static cudaError_t a2_and_vec(const gsr_handle_t *h, cudaStream_t s,
                                            cudaGraphConditionalHandle loop, int in_graph, int first,
                                            cudaEvent_t mid = nullptr)
{
    double *part = h->d_partial + kRedV * kPartialsPerKind;
    unsigned *cnt = h->d_counter + kRedV;
    A2Parts P = {};
    const bool inl = aprod2_partials(h, h->d_u, h->d_q, &P.S, &P.ipart, &P.isplit, &P.gpart,
                                     &P.ngpart, &P.ctr, s);
    if (!inl) {
        cudaError_t e = launch_aprod2(h, h->d_u, h->d_q, kA2Overwrite, s);
        if (e != cudaSuccess)
            return e;
        if (mid && (e = cudaEventRecord(mid, s)) != cudaSuccess)
            return e;
        k_vec<false><<<h->grid_lsqr_vec, kThreads, 0, s>>>(h->sys, h->d_p, h->d_q, h->d_v, h->d_vp, h->d_w,
                                                      h->d_z, h->d_var, h->d_state, h->d_args, part,
                                                      cnt, loop, in_graph, first, P,
                                                      h->d_kerr);
    } else {
        if (mid) {
            cudaError_t e = cudaEventRecord(mid, s);
            if (e != cudaSuccess)
                return e;
        }
        k_vec<true><<<h->grid_lsqr_vec, kThreads, 0, s>>>(h->sys, h->d_p, h->d_q, h->d_v, h->d_vp, h->d_w,
                                                     h->d_z, h->d_var, h->d_state, h->d_args, part,
                                                     cnt, loop, in_graph, first, P,
                                                     h->d_kerr);
    }
    return cudaGetLastError();
}

// The three parts of one solve.  `in_graph` says whether the kernels run
// inside the solve graph (and may clear its loop flag).
cudaError_t enqueue_prologue(const gsr_handle_t *h, cudaStream_t s,
                             cudaGraphConditionalHandle loop, int in_graph)
{
    const SysView &A = h->sys;
    double *part = h->d_partial;
    unsigned *cnt = h->d_counter;
    cudaError_t e = enqueue_precond(h, h->d_p, s);
    if (e != cudaSuccess)
        return e;
    k_init_u<<<h->grid_vec, kThreads, 0, s>>>(h->d_args, h->d_u, A.m, h->d_state,
                                               part + kRedBnorm * kPartialsPerKind, cnt + kRedBnorm);
    k_zero<<<h->grid_vec, kThreads, 0, s>>>(h->d_q + A.att0, A.n - A.att0);
    return a2_and_vec(h, s, loop, in_graph, 1);
}

cudaError_t enqueue_iteration(const gsr_handle_t *h, cudaStream_t s,
                              cudaGraphConditionalHandle loop, int in_graph)
{
    cudaError_t e = launch_aprod1(h, h->d_vp, h->d_u, 1, s);
    if (e != cudaSuccess)
        return e;
    return a2_and_vec(h, s, loop, in_graph, 0);
}

// One iteration launched from the host with events between its launches:
// ev[0] before aprod 1, ev[1] after it, ev[2] after aprod 2, ev[3] after the
// vector pass (ev[0] may be the previous iteration's ev[3]).
cudaError_t enqueue_iteration_timed(const gsr_handle_t *h, cudaStream_t s, const cudaEvent_t *ev)
{
    cudaError_t e = launch_aprod1(h, h->d_vp, h->d_u, 1, s);
    if (e == cudaSuccess)
        e = cudaEventRecord(ev[1], s);
    if (e == cudaSuccess)
        e = a2_and_vec(h, s, 0, 0, 0, ev[2]);
    if (e == cudaSuccess)
        e = cudaEventRecord(ev[3], s);
    return e;
}

cudaError_t enqueue_epilogue(const gsr_handle_t *h, cudaStream_t s)
{
    const SysView &A = h->sys;
    k_finalize<<<h->grid_vec, kThreads, 0, s>>>(h->d_p, h->d_z, h->d_var, A.n, A.m, h->d_state,
                                                 h->d_args);
    return cudaGetLastError();
}

// an unfinished capture on s and the graph g are given up
static void drop_capture(cudaStream_t s, cudaGraph_t g)
{
    cudaStreamCaptureStatus cs;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
        cudaGraph_t junk = nullptr;
        cudaStreamEndCapture(s, &junk);
        if (junk && junk != g)
            cudaGraphDestroy(junk);
    }
    if (g)
        cudaGraphDestroy(g);
    cudaGetLastError();
}

// Build and instantiate the graph of one whole solve:
//   [precondition, U_1 = b, q = A^T U_1, V_1]  ->  WHILE(flag) { iteration }
//   ->  [x = p o z, se]
cudaError_t build_launch_graph(gsr_handle_t *h, cudaGraphExec_t *exec)
{
    cudaError_t err = cudaSuccess;
    cudaGraph_t g = nullptr;
    cudaGraphConditionalHandle loop;
    cudaGraphNode_t pre_leaf, wnode;
    cudaGraphNodeParams cp = {};
    cudaGraph_t body;
    cudaStream_t s = h->cap_stream;

    GSR_TRY(cudaGraphCreate(&g, 0));
    GSR_TRY(cudaGraphConditionalHandleCreate(&loop, g, 1u, cudaGraphCondAssignDefault));

    GSR_TRY(cudaStreamBeginCaptureToGraph(s, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    GSR_TRY(enqueue_prologue(h, s, loop, 1));
    GSR_TRY(cudaStreamEndCapture(s, &g));
    GSR_TRY(find_graph_leaf(g, &pre_leaf));

    // WHILE node: one LSQR iteration per trip
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = loop;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    GSR_TRY(cudaGraphAddNode(&wnode, g, &pre_leaf, nullptr, 1, &cp));
    body = cp.conditional.phGraph_out[0];
    GSR_TRY(cudaStreamBeginCaptureToGraph(s, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    GSR_TRY(enqueue_iteration(h, s, loop, 1));
    GSR_TRY(cudaStreamEndCapture(s, &body));

    GSR_TRY(cudaStreamBeginCaptureToGraph(s, g, &wnode, nullptr, 1, cudaStreamCaptureModeThreadLocal));
    GSR_TRY(enqueue_epilogue(h, s));
    GSR_TRY(cudaStreamEndCapture(s, &g));

    GSR_TRY(cudaGraphInstantiate(exec, g, 0));
    cudaGraphDestroy(g);
    return cudaSuccess;
fail:
    drop_capture(s, g);
    return err;
}

// ... or, for a small system, with one launch for all iterations in place of
// the loop (k_lsqr_loop)
cudaError_t build_solve_graph(gsr_handle_t *h)
{
    if (!lsqr_loop_fits(h))
        return build_launch_graph(h, &h->solve_exec);
    cudaError_t err = cudaSuccess;
    cudaGraph_t g = nullptr;
    cudaStream_t s = h->cap_stream;
    GSR_TRY(cudaGraphCreate(&g, 0));
    GSR_TRY(cudaStreamBeginCaptureToGraph(s, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    GSR_TRY(enqueue_prologue(h, s, 0, 0));
    GSR_TRY(launch_lsqr_loop(h, s));
    GSR_TRY(enqueue_epilogue(h, s));
    GSR_TRY(cudaStreamEndCapture(s, &g));
    GSR_TRY(cudaGraphInstantiate(&h->solve_exec, g, 0));
    cudaGraphDestroy(g);
    return cudaSuccess;
fail:
    drop_capture(s, g);
    return err;
}

}  // namespace gsr
