// Pieces of an LSQR iteration shared by the vector pass and the one-launch
// loop of small systems: the scalar recurrences with the stopping rules, and
// the update of the columns.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "gsr_internal.cuh"
#include "gsr_reduce.cuh"
#include "gsr_split.cuh"

namespace gsr {

constexpr int kIstopNonfinite = 8;
constexpr int kThreadParts = 8;  // window totals of an instrument that one thread adds

// A bounded wait of a kernel before this one has expired: the results are
// undefined, and each further iteration could wait as long.  Read at the start
// of a kernel, beside its other loads, by the threads that form the scalars.
__device__ __forceinline__ bool wait_expired(const int *kerr)
{
    return *(const volatile int *)kerr != 0;
}

// Square roots and the reciprocal that the scalar recurrences of an iteration
// start from: alpha_{i+1}, ||z||, ||A||, sqrt(ddnorm), 1/alpha_{i+1}, rho_i
struct LsqrRoots {
    double alpha, xnorm, anorm, ddroot, ia, rho;
};

// Scalar recurrences of one LSQR iteration by one thread, with products by
// reciprocals already known (1/rho from the aprod 1 pass) instead of
// divisions: FP64 divisions and square roots take a third of a microsecond
// each on this part and every dependent operation 65 clocks.  The tests of
// the machine-precision rules are multiplied out: 1 + a / b <= 1 exactly when
// a <= 2^-53 b (up to the rounding of a / b).  late: a wait has expired, the
// iterations end.
__device__ __forceinline__ void lsqr_finish(SolveState *st, const SolveArgs *args, const LsqrRoots &R,
                                            double anorm2, double ddnorm, bool late,
                                            cudaGraphConditionalHandle loop, int in_graph)
{
    constexpr double kHalfEps = 1.0 / 9007199254740992.0;  // 2^-53
    const double beta = st->bnext;
    SolveState s = *st;
    const double alpha = R.alpha;
    const double irho = s.irho;
    const double rho = R.rho;
    const double c = s.rhobar * irho;
    const double sn = beta * irho;
    const double phi = c * s.phibar;
    s.anorm2 = anorm2;
    s.theta = sn * alpha;
    s.rhobar = -c * alpha;
    s.phibar = sn * s.phibar;
    const double tau = sn * phi;
    s.rho = rho;
    s.cs = c;
    s.sn = sn;
    s.phi = phi;
    s.alpha = alpha;
    s.beta = beta;
    s.cy = -alpha * alpha * s.ia * s.ib;  // -alpha_{i+1}^2 / (alpha_i beta_{i+1})
    s.ddnorm = ddnorm;
    s.xnorm = R.xnorm;
    s.anorm = R.anorm;
    s.acond = s.anorm * R.ddroot;
    s.ia = R.ia;
    s.rnorm = s.phibar;
    s.arnorm = alpha * fabs(tau);
    s.itn += 1;
    s.t = s.rnorm * args->isdof;

    // stopping rules (P&S 1982 §6) in multiplied form; a later rule wins
    const double anx = s.anorm * s.xnorm;
    const double rtol_b = args->btol * s.bnorm + args->atol * anx;  // rtol * bnorm
    const double anr = s.anorm * s.rnorm;
    int istop = 0;
    if (s.itn >= args->itmax) istop = 7;
    if (s.acond * kHalfEps >= 1.0) istop = 6;
    if (anr != 0.0 && s.arnorm <= kHalfEps * anr) istop = 5;
    if (s.bnorm + anx > 0.0 && s.rnorm <= kHalfEps * (s.bnorm + anx)) istop = 4;
    if (args->ctol * s.acond >= 1.0 && args->ctol > 0.0) istop = 3;
    if (anr != 0.0 && s.arnorm <= args->atol * anr) istop = 2;
    if (s.rnorm <= rtol_b) istop = 1;
    const bool bad = !isfinite(rho) || !isfinite(alpha) || !isfinite(s.phibar) ||
                     !isfinite(s.xnorm) || !isfinite(s.ddnorm) || rho == 0.0;
    if (bad) {
        s.nonfinite = 1;
        istop = kIstopNonfinite;
    }
    if (args->force_itmax && !bad && s.itn < args->itmax)
        istop = 0;
    s.istop = istop;
    if (istop != 0 || late) {
        s.done = 1;
        if (in_graph)
            cudaGraphSetConditional(loop, 0u);
    }
    *st = s;
}

// ... by the whole last block of the vector pass: the independent roots go to
// different warps
__device__ __forceinline__ void lsqr_scalars(SolveState *st, const SolveArgs *args, double vnorm2,
                                             double dd, double zz, bool late,
                                             cudaGraphConditionalHandle loop, int in_graph)
{
    __shared__ LsqrRoots sq;
    const double beta = st->bnext;
    const bool upd = beta > 0.0;
    const double anorm2 = upd ? st->anorm2 + st->alpha * st->alpha + beta * beta : st->anorm2;
    const double ddnorm = st->ddnorm + dd;
    if (threadIdx.x == 0)
        sq.alpha = upd ? sqrt(vnorm2) : st->alpha;
    if (threadIdx.x == 32)
        sq.xnorm = sqrt(zz);
    if (threadIdx.x == 64)
        sq.anorm = sqrt(anorm2);
    if (threadIdx.x == 96)
        sq.ddroot = sqrt(ddnorm);
    if (threadIdx.x == 128) {
        const double a = upd ? sqrt(vnorm2) : st->alpha;
        sq.ia = (a > 0.0) ? 1.0 / a : 1.0;
    }
    if (threadIdx.x == 160)
        sq.rho = sqrt(st->rhobar * st->rhobar + beta * beta);
    __syncthreads();
    if (threadIdx.x == 0)
        lsqr_finish(st, args, sq, anorm2, ddnorm, late, loop, in_graph);
}

// ... by one warp: the roots in different lanes
__device__ __forceinline__ void lsqr_scalars_warp(SolveState *st, const SolveArgs *args,
                                                  double vnorm2, double dd, double zz)
{
    const int lane = threadIdx.x & 31;
    const double beta = st->bnext, alpha0 = st->alpha, rhobar = st->rhobar;
    const bool upd = beta > 0.0;
    const double anorm2 = upd ? st->anorm2 + alpha0 * alpha0 + beta * beta : st->anorm2;
    const double ddnorm = st->ddnorm + dd;
    double r = sqrt(lane == 0 ? vnorm2 : lane == 1 ? zz : lane == 2 ? anorm2
                    : lane == 3 ? ddnorm : rhobar * rhobar + beta * beta);
    if (lane == 0 && !upd)
        r = alpha0;
    LsqrRoots R;
    R.alpha = __shfl_sync(0xffffffffu, r, 0);
    R.xnorm = __shfl_sync(0xffffffffu, r, 1);
    R.anorm = __shfl_sync(0xffffffffu, r, 2);
    R.ddroot = __shfl_sync(0xffffffffu, r, 3);
    R.rho = __shfl_sync(0xffffffffu, r, 4);
    R.ia = (R.alpha > 0.0) ? 1.0 / R.alpha : 1.0;
    __syncwarp();  // every lane has read the state
    if (lane == 0)
        lsqr_finish(st, args, R, anorm2, ddnorm, false, 0, 0);
}

// Coefficients of the column updates of iteration i (W = w / rho, see k_vec)
struct VecCoef {
    double c1, c2, phi, k1, k2;
    bool upd, first;
};

__device__ __forceinline__ VecCoef vec_coef(const SolveState *st, int first)
{
    VecCoef k;
    const double ia = st->ia;                          // 1/alpha_i
    const double ib = st->ib;                          // 1/beta_{i+1}
    const double bn = st->bnext;                       // beta_{i+1}
    const double irho = first ? 0.0 : st->irho;        // 1/rho_i
    k.first = first != 0;
    k.c1 = ia * irho;                                  // 1/(alpha_i rho_i)
    k.c2 = first ? 0.0 : -st->theta * irho;
    k.phi = first ? 0.0 : st->t1;                      // phi_i
    k.upd = bn > 0.0;
    k.k1 = ia * ib;
    k.k2 = -bn * ia;
    return k;
}

// Vectors of the pass and its three sums of squares (||V||^2, sum W^2, ||z||^2:
// on the binary32 pipes from exact splits, fb for values outside the window)
struct VecPass {
    const double *p;
    double *v, *vp, *w, *z, *var;
};
struct VecSums {
    Acc3 c[3] = {Acc3{0.f, 0.f, 0.f}, Acc3{0.f, 0.f, 0.f}, Acc3{0.f, 0.f, 0.f}};
    double fb[3] = {0.0, 0.0, 0.0};
    __device__ __forceinline__ double total(int k) const { return acc3_to_double(c[k]) + fb[k]; }
};

// Column j with q_j = qf(): the loads of the vectors come first, so that they
// are in flight together with those of the partial sums.  no_v: W, z and var
// only (the global column of k_vec, whose V its last block updates).
template <typename QF>
__device__ __forceinline__ void vec_column(const VecPass &X, const VecCoef &k, VecSums &S, int64_t j,
                                           bool no_v, QF qf)
{
    const double pj = X.p[j];
    double vo = 0.0, wo = 0.0, zo = 0.0, ro = 0.0;
    if (!k.first) {
        vo = X.v[j];
        wo = X.w[j];
        zo = X.z[j];
        ro = X.var[j];
    }
    const double qj = qf();
    double wj = 0.0, zj = 0.0, vr = 0.0;
    if (!k.first) {
        wj = fma(k.c2, wo, vo * k.c1);
        vr = fma(wj, wj, ro);
        zj = fma(k.phi, wj, zo);
        acc3_sqr_or(S.c[1], S.fb[1], wj);
        acc3_sqr_or(S.c[2], S.fb[2], zj);
    }
    X.w[j] = wj;
    X.z[j] = zj;
    X.var[j] = vr;
    if (no_v)
        return;
    const double vn = k.upd ? fma(pj * qj, k.k1, k.k2 * vo) : vo;
    X.v[j] = vn;
    X.vp[j] = pj * vn;
    acc3_sqr_or(S.c[0], S.fb[0], vn);
}

}  // namespace gsr
