// Mixed-precision PC solve: binary32 storage of A for the inner iterations,
// FP64 refinement of the normal-equation residual.
//
// Inner operator (the products of aprod 1 / aprod 2 of Alg. 1 / Alg. 2 on
// the binary32 copy A32 of A): every product of a binary32 value with a
// binary32 vector entry is formed in binary32, and the products are
// accumulated as double-float pairs (hi + lo, Knuth's error-free TwoSum) on
// the FP32 pipes, which is as accurate as FP64 accumulation for these sums.
// GB300 runs FP64 at 2 FMA per clock per SM and FP32 at 128, so the inner
// passes stay on the FP32 pipes and read half the bytes of the FP64 form.
//
// Outer loop (host driven, FP64): with p the column-norm preconditioner,
//   r = b - A x,  c = p o (A^T r)         (FP64 kernels of gsr_kernels.cu)
//   stop when ||c|| <= atol ||A diag(p)||_F ||r||   (P&S rule S2, exact terms)
//   solve (diag(p) A32^T A32 diag(p)) z = c approximately by CG
//   x += p o z
// The fixed point is A^T (b - A x) = 0, the FP64 least-squares solution.
//
// CG on the normal equations (Hestenes-Stiefel) with s_0 = c, d_0 = s_0:
//   q = A32 (p o d), alpha = |s|^2 / |q|^2, z += alpha d,
//   s -= alpha p o (A32^T q), beta = |s_new|^2 / |s|^2, d = s + beta d.
// One inner iteration = 4 launches (the main pass with both products of the
// attitude and global part, the star and instrument passes in one launch, two
// vector passes) in a CUDA graph with a conditional WHILE node, like the LSQR
// loop.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "gsr_internal.cuh"
#include "gsr_lsqr.cuh"
#include "gsr_reduce.cuh"
#include "gsr_df.cuh"
#include "gsr_att32.cuh"
#include "gsr_ell.cuh"

namespace gsr {


__device__ __forceinline__ int64_t gtid32() { return blockIdx.x * (int64_t)blockDim.x + threadIdx.x; }
__device__ __forceinline__ int64_t gstride32() { return (int64_t)gridDim.x * blockDim.x; }

// the passes of the main kernel
constexpr int kF32A1 = 1;  // q = A32 x
constexpr int kF32A2 = 2;  // attitude and global part of A32^T q

// ---------------------------------------------------------------------------
// Main pass of the inner operator over the offset-ordered values, one row per
// lane (binary32 products, double-float sums).
// A1 and A2 (CG): q32[row] = fl32(A32 x32) with |q|^2 (alpha = gamma / |q|^2
// by the last block), the attitude sums of A32^T q into S[place of the unit][4a + j] and
// its global column into *glb.  A1 alone: y[row] += A32 x32 in FP64.  A2
// alone: q is read from q32, *glb += its global column.
// One reading of the values (96 B a row) serves both products, the row's q is
// scattered to row order (28 MB at 7.0e6 rows: it stays in L2); the
// astrometric x of a random star is one 32-byte sector of x8.
// At 7.0e6 rows 186 us, against 124 us for its 120 B a row at the copy rate:
// 490 instructions a visit keep 55 % of the issue slots busy, the rest is
// latency with 16 warps an SM; without the scatter of q 173 us, without the
// gather of x 174.  The product A32 x alone took 156 us in row order.
// ---------------------------------------------------------------------------
constexpr int kMainWarps = 16;  // one block per SM
constexpr int kMainThreads = 32 * kMainWarps;

// Where the instrumental x is (six random reads a row): in shared memory
// beside three stages a warp up to 12,288 instruments, beside two up to
// 27,648; beyond, in global memory, with two stages so that more of it stays
// in L1.  20,000 instruments, 7.0e7 rows: 3.97 ms from global memory beside
// three stages, 3.85 from shared memory beside two (3.23 with the units in the
// order of their rows, which keeps the scatter of q in L2).
enum MainX { kXGlobal = 0, kXThree = 1, kXTwo = 2 };
constexpr int64_t kXThreeMax = 12288, kXTwoMax = 27648;
__host__ __device__ constexpr int main_stages(int where) { return where == kXThree ? 3 : 2; }

// [stages][x of the attitude taps: 16 floats a warp][barriers][instrument x]
__host__ __device__ constexpr size_t main_smem(int where)
{
    return kMainWarps * (main_stages(where) * (kAttTileBytes + sizeof(uint64_t)) +
                         16 * sizeof(float));
}

template <int MODE, int X>
__global__ void __launch_bounds__(kMainThreads, 1)
k_f32_main(SysView A, Att32 U, const float *__restrict__ x32, const float *__restrict__ x8,
           float *__restrict__ q32, double *__restrict__ y, double *__restrict__ S,
           double *__restrict__ glb, CgState *cg, double *partial, unsigned *counter, int *kerr)
{
    constexpr bool A1 = (MODE & kF32A1) != 0, A2 = (MODE & kF32A2) != 0, SMEMX = X != kXGlobal;
    constexpr int NS = main_stages(X);
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char *stages = smem + wib * NS * kAttTileBytes;
    float *s_xa = reinterpret_cast<float *>(smem + kMainWarps * NS * kAttTileBytes) + 16 * wib;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kMainWarps * (NS * kAttTileBytes +
                                                                       16 * sizeof(float))) +
                     NS * wib;
    float *s_x32 = reinterpret_cast<float *>(smem + main_smem(X));
    // units are dealt to the warps of all blocks round-robin, blocks first, so
    // that a small system spreads over the SMs
    AttWalk<NS> walk(U, stages, bars, blockIdx.x + (int64_t)gridDim.x * wib,
                     (int64_t)gridDim.x * kMainWarps);
    if (A1 && SMEMX) {
        for (int64_t f = threadIdx.x; f < A.I; f += blockDim.x)
            s_x32[f] = x32[A.ins0 + f];
        __syncthreads();
    }
    const float xg = A1 ? __ldg(x32 + A.glb0) : 0.f;
    const float *xk = x32 + A.att0 + (lane >> 2) * A.D + (lane & 3);  // lane k < 12: tap k
    float nh = 0.f, nl = 0.f;  // |q|^2 of this thread (double-float)
    float gh = 0.f, gl = 0.f;  // its global sum
    f32x2 sh[kNAtt / 2], sl[kNAtt / 2];  // attitude sums, taps k and k + 1 packed
    // astrometric x of the row (one sector), or its q, one visit ahead
    f32x2 s01 = 0ull, s23 = 0ull;
    float s4 = 0.f, xt = 0.f;
    auto prefetch = [&](int j, f32x2 &a, f32x2 &b, float &c, float &x) {
        if (A1) {
            asm("{ .reg .b32 a, b, c, d, f, g, h, i;\n"
                "ld.global.nc.v8.b32 {a, b, c, d, f, g, h, i}, [%3];\n"
                "mov.b64 %0, {a, b}; mov.b64 %1, {c, d}; mov.b32 %2, f; }"
                : "=l"(a), "=l"(b), "=f"(c) : "l"(x8 + 8 * (int64_t)walk.rec(j).x));
            x = (lane < kNAtt && walk.d[j].first()) ? __ldg(xk + walk.d[j].un.x) : 0.f;
        } else {
            c = __ldg(q32 + walk.row(j));
        }
    };
    bool ok = walk.d[0].ok && walk.arrived(0, kerr);
    if (ok)
        prefetch(0, s01, s23, s4, xt);
    while (ok) {
        f32x2 n01 = 0ull, n23 = 0ull;
        float n4 = 0.f, nt = 0.f;
        const bool more = walk.d[1].ok;
        if (more) {
            ok = walk.arrived(1, kerr);
            if (ok)
                prefetch(1, n01, n23, n4, nt);
        }
        const Visit v = walk.d[0];
        if (v.first()) {
            if (A1) {
                if (lane < kNAtt)
                    s_xa[lane] = xt;
                __syncwarp();
            }
#pragma unroll
            for (int k = 0; k < kNAtt / 2; k++)
                sh[k] = sl[k] = 0ull;
        }
        const uint32_t e = (v.t << 5) + lane;
        if (e >= v.un.y && e < v.un.z) {
            const float *vk = walk.val() + lane;  // plane k at vk[32 k]
            const uint32_t r = walk.row();
            float q;
            if constexpr (A1) {
                const uint4 rc = walk.rec(0);
                float xi[kNInstr];
#pragma unroll
                for (int j = 0; j < kNInstr; j++) {
                    const uint32_t f = instr_at32(rc, j);
                    xi[j] = SMEMX ? s_x32[f] : __ldg(x32 + A.ins0 + f);
                }
                // the 24 products as 12 pairs: two chains of sums, packed
                f32x2 h = 0ull, l = 0ull;
#pragma unroll
                for (int k = 0; k < kNAtt; k += 2)
                    df_acc_v(h, l, v_mul(pack2(vk[32 * (5 + k)], vk[32 * (6 + k)]),
                                         *reinterpret_cast<const f32x2 *>(s_xa + k)));
                df_acc_v(h, l, v_mul(pack2(vk[0], vk[32]), s01));
                df_acc_v(h, l, v_mul(pack2(vk[64], vk[96]), s23));
                df_acc_v(h, l, v_mul(pack2(vk[128], vk[32 * 23]), pack2(s4, xg)));
#pragma unroll
                for (int j = 0; j < kNInstr; j += 2)
                    df_acc_v(h, l, v_mul(pack2(vk[32 * (17 + j)], vk[32 * (18 + j)]),
                                         pack2(xi[j], xi[j + 1])));
                float h0, h1, l0, l1;
                unpack2(h, h0, h1);
                unpack2(l, l0, l1);
                df_acc(h0, l0, h1);
                l0 = __fadd_rn(l0, l1);
                if constexpr (A2) {
                    q = __fadd_rn(h0, l0);
                    q32[r] = q;
                    // q^2 = pq + eq exactly (product error by FMA), accumulated
                    // in double-float on the FP32 pipe
                    const float pq = __fmul_rn(q, q);
                    df_acc(nh, nl, pq);
                    nl = __fadd_rn(nl, __fmaf_rn(q, q, -pq));
                } else {
                    q = 0.f;
                    y[r] += df_to_d(h0, l0);
                }
            } else {
                q = s4;
            }
            if constexpr (A2) {
                const f32x2 qq = pack2(q, q);
#pragma unroll
                for (int k = 0; k < kNAtt; k += 2)
                    df_acc_v(sh[k / 2], sl[k / 2],
                             v_mul(pack2(vk[32 * (5 + k)], vk[32 * (6 + k)]), qq));
                df_acc(gh, gl, __fmul_rn(vk[32 * 23], q));
            }
        }
        if (v.last()) {
            if constexpr (A2) {
                // reduce-scatter over the warp in double-float (FP32 pipe):
                // after the butterfly, lane pair (2k, 2k+1) holds sum k
                __syncwarp();
                float rh[16], rl[16];
#pragma unroll
                for (int k = 0; k < 16; k += 2) {
                    rh[k] = rh[k + 1] = rl[k] = rl[k + 1] = 0.f;
                    if (k < kNAtt) {
                        unpack2(sh[k / 2], rh[k], rh[k + 1]);
                        unpack2(sl[k / 2], rl[k], rl[k + 1]);
                    }
                }
                df_reduce_scatter<16, 32>(rh, rl, lane);
                const int kk = lane >> 1;
                if ((lane & 1) == 0 && kk < kNAtt)
                    S[(int64_t)v.un.w * kNAtt + kk] = df_to_d(rh[0], rl[0]);
            }
        }
        if (!more || !ok)
            break;
        walk.advance();
        s01 = n01;
        s23 = n23;
        s4 = n4;
        xt = nt;
    }
    if constexpr (A2) {
        double v2[2] = {df_to_d(nh, nl), df_to_d(gh, gl)};
        if (grid_reduce<2, kMainThreads>(v2, partial, counter) && threadIdx.x == 0) {
            if (A1) {
                cg->xi = v2[0];
                cg->alpha = (v2[0] > 0.0) ? cg->gamma / v2[0] : 0.0;
                *glb = v2[1];
            } else {
                *glb += v2[1];
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Astrometric part of the inner aprod 2, one star group of the rest kernel:
// G lanes per star over the row-ordered q.  MODE kA2Accumulate: out += ,
// kA2Overwrite: written.
// ---------------------------------------------------------------------------
template <int G, int MODE>
__device__ __forceinline__ void stars_body_f32(const SysView &A, const float *__restrict__ sv,
                                               const float *__restrict__ y32,
                                               double *__restrict__ out, int64_t grp)
{
    static_assert(G >= kNAstro, "a star group needs a lane per astrometric sum");
    constexpr int GPW = 32 / G;
    const int lane = threadIdx.x & (G - 1);
    const int gw = (threadIdx.x & 31) / G;
    const int64_t s0 = grp * GPW;
    // the GPW stars of a warp have similar row counts (stars taken in
    // decreasing row count), so its lane groups finish together
    const int64_t s = (s0 + gw < A.S) ? (int64_t)A.sorder[s0 + gw] : A.S;
    uint32_t r0 = 0, r1 = 0;
    if (s < A.S) {
        r0 = A.star_ptr[s];
        r1 = A.star_ptr[s + 1];
    }
    float ah[kNAstro], al[kNAstro];
#pragma unroll
    for (int k = 0; k < kNAstro; k++)
        ah[k] = al[k] = 0.f;
#pragma unroll 2
    for (uint32_t r = r0 + lane; r < r1; r += G) {
        const float *v = sv + tidx<kNAstro>(0, r);
        const float yi = __ldg(y32 + r);
#pragma unroll
        for (int k = 0; k < kNAstro; k++)
            df_acc(ah[k], al[k], __fmul_rn(__ldcs(v + 32 * k), yi));
    }
    // the star's five sums over its G lanes, in double-float
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) {
#pragma unroll
        for (int k = 0; k < kNAstro; k++) {
            const float oh = __shfl_xor_sync(0xffffffffu, ah[k], off);
            const float ol = __shfl_xor_sync(0xffffffffu, al[k], off);
            df_add(ah[k], al[k], oh, ol);
        }
    }
    if (lane < kNAstro && s < A.S) {
        // lane k writes sum k (all lanes of the group hold all five)
        float kh = ah[0], kl = al[0];
#pragma unroll
        for (int k = 1; k < kNAstro; k++)
            if (lane == k) {
                kh = ah[k];
                kl = al[k];
            }
        double *xs = out + kNAstro * s + lane;
        if (MODE == kA2Accumulate)
            *xs += df_to_d(kh, kl);
        else
            *xs = df_to_d(kh, kl);
    }
}

// inner aprod 2, instrumental part over the instrument-sorted binary32 copy,
// four gathers in flight per lane, double-float sums.  One row window: unit
// w is piece k = w % npieces of instrument f = w / npieces (pieces by count
// over iseg), total to part[k I + f].  (This plain form measured 10% faster
// than the windowed decode of instr_body_f32_win with one window.)
__device__ __forceinline__ void instr_body_f32_one(const SysView &A, const uint32_t *__restrict__ iseg,
                                               const uint32_t *__restrict__ irow,
                                               const float *__restrict__ ival32,
                                               const float *__restrict__ y32,
                                               double *__restrict__ part, int nsplit, int64_t warp,
                                               int64_t nwarps)
{
    const int lane = threadIdx.x & 31;
    for (int64_t w = warp; w < A.I * nsplit; w += nwarps) {
        const int64_t f = w / nsplit;
        const int q = (int)(w - f * nsplit);
        const uint32_t s0 = iseg[f];
        const uint64_t len = iseg[f + 1] - s0;
        const uint32_t e1 = s0 + (uint32_t)(len * (q + 1) / nsplit);
        uint32_t e = s0 + (uint32_t)(len * q / nsplit) + lane;
        float h[4] = {0.f, 0.f, 0.f, 0.f}, l[4] = {0.f, 0.f, 0.f, 0.f};
        for (; e + 96 < e1; e += 128) {
            uint32_t r[4];
            float v[4], yv[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                r[u] = __ldcs(irow + e + 32 * u);
                v[u] = __ldcs(ival32 + e + 32 * u);
            }
#pragma unroll
            for (int u = 0; u < 4; u++)
                yv[u] = __ldg(y32 + r[u]);
#pragma unroll
            for (int u = 0; u < 4; u++)
                df_acc(h[u], l[u], __fmul_rn(v[u], yv[u]));
        }
        for (int u = 0; e < e1; e += 32, u++)
            df_acc(h[u & 3], l[u & 3], __fmul_rn(__ldcs(ival32 + e), __ldg(y32 + __ldcs(irow + e))));
        df_add(h[0], l[0], h[1], l[1]);
        df_add(h[2], l[2], h[3], l[3]);
        df_add(h[0], l[0], h[2], l[2]);
        df_warp_sum(h[0], l[0]);
        if (lane == 0)
            part[(int64_t)q * A.I + f] = df_to_d(h[0], l[0]);
    }
}

// Several row windows: piece k of instrument f in row window q (unit
// w = (q I + f) ks + k), total to part[(q ks + k) I + f].
__device__ __forceinline__ void instr_body_f32_win(const SysView &A, const uint32_t *__restrict__ seg,
                                               const uint32_t *__restrict__ irow,
                                               const float *__restrict__ ival32,
                                               const float *__restrict__ y32,
                                               double *__restrict__ part, int nwin, int ks,
                                               int64_t warp, int64_t nwarps)
{
    const int lane = threadIdx.x & 31;
    const int64_t per = A.I * ks;  // units per window
    for (int64_t w = warp; w < per * nwin; w += nwarps) {
        // unit w: piece k of instrument f in row window q (window-major,
        // then instrument-major); seg is the window table (d_cseg32)
        const int64_t q = w / per;
        const int64_t r = w - q * per;
        const int64_t f = r / ks;
        const int k = (int)(r - f * ks);
        const uint32_t s0 = seg[q * A.I + f];
        const uint64_t len = seg[(q + 1) * A.I + f] - s0;
        const uint32_t e1 = s0 + (uint32_t)(len * (k + 1) / ks);
        uint32_t e = s0 + (uint32_t)(len * k / ks) + lane;
        float h[4] = {0.f, 0.f, 0.f, 0.f}, l[4] = {0.f, 0.f, 0.f, 0.f};
        for (; e + 96 < e1; e += 128) {
            uint32_t r[4];
            float v[4], yv[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                r[u] = __ldcs(irow + e + 32 * u);
                v[u] = __ldcs(ival32 + e + 32 * u);
            }
#pragma unroll
            for (int u = 0; u < 4; u++)
                yv[u] = __ldg(y32 + r[u]);
#pragma unroll
            for (int u = 0; u < 4; u++)
                df_acc(h[u], l[u], __fmul_rn(v[u], yv[u]));
        }
        for (int u = 0; e < e1; e += 32, u++)
            df_acc(h[u & 3], l[u & 3], __fmul_rn(__ldcs(ival32 + e), __ldg(y32 + __ldcs(irow + e))));
        df_add(h[0], l[0], h[1], l[1]);
        df_add(h[2], l[2], h[3], l[3]);
        df_add(h[0], l[0], h[2], l[2]);
        df_warp_sum(h[0], l[0]);
        if (lane == 0)
            part[(q * ks + k) * A.I + f] = df_to_d(h[0], l[0]);
    }
}

// Rest of the inner aprod 2 in one launch: star units and instrument units
// from one work queue (as k_aprod2_fused, without attitude units)
template <int G, int MODE, bool WIN>
__global__ void __launch_bounds__(kThreads)
k_f32_rest(SysView A, Att32 U, const float *__restrict__ y32, double *__restrict__ out,
           const uint32_t *__restrict__ cseg, const uint32_t *__restrict__ irow,
           const float *__restrict__ ival32, double *__restrict__ part, int nwin, int ks, A2Queue q)
{
    const int lane = threadIdx.x & 31;
    const int L = q.ns + q.ni;
    for (;;) {
        unsigned long long u = 0;
        if (lane == 0)
            u = atomicAdd(q.ctr, 1ull);
        u = __shfl_sync(0xffffffffu, u, 0);
        if ((int64_t)u >= q.total)
            break;
        // 32-bit unit decode below 2^32 units (a 64-bit division is a long
        // instruction sequence, partly on the FP64 pipe)
        int64_t c;
        int slot;
        if (q.total <= (int64_t)0xffffffffll) {
            c = (uint32_t)u / (uint32_t)L;
            slot = (int)((uint32_t)u - (uint32_t)c * (uint32_t)L);
        } else {
            c = (int64_t)u / L;
            slot = (int)((int64_t)u - c * L);
        }
        if (slot < q.ns) {
            const int64_t i = c * q.ns + slot;
            if (i < q.nstar_units) {
                for (int k = 0; k < q.star_k; k++) {
                    const int64_t grp = i * q.star_k + k;
                    if (grp < q.nstar_groups)
                        stars_body_f32<G, MODE>(A, U.sv, y32, out, grp);
                }
            }
        } else {
            const int64_t i = c * q.ni + (slot - q.ns);
            if (i < q.ninstr_units)
                if (WIN)
                    instr_body_f32_win(A, cseg, irow, ival32, y32, part, nwin, ks, i,
                                       q.ninstr_units);
                else  // one window: pieces by count over iseg
                    instr_body_f32_one(A, cseg, irow, ival32, y32, part, ks, i, q.ninstr_units);
        }
    }
}

// The rest of the inner aprod 2 with the instruments in row windows: 16 warps
// of a block sum its windows, the others take star units, and the first 16
// join them
constexpr int kRestThreads = 768;

template <int G, int MODE>
__global__ void __launch_bounds__(kRestThreads, 1)
k_f32_rest_win(SysView A, Att32 U, Ell E, const float *__restrict__ y32, double *__restrict__ out,
               A2Queue q, int *kerr)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ EllShared sh;
    const uint32_t nfix = gridDim.x * (kRestThreads / 32 - kEllWarps);
    uint32_t u = 0xffffffffu;
    if (threadIdx.x < kEllThreads)
        ell32_part(E, y32, A.m, smem, &sh, kerr, A.I);
    else
        u = blockIdx.x + gridDim.x * ((threadIdx.x - kEllThreads) >> 5);
    for (;;) {
        if (u != 0xffffffffu && (int64_t)u < q.nstar_units)
            for (int k = 0; k < q.star_k; k++) {
                const int64_t grp = (int64_t)u * q.star_k + k;
                if (grp < q.nstar_groups)
                    stars_body_f32<G, MODE>(A, U.sv, y32, out, grp);
            }
        if ((int64_t)nfix >= q.nstar_units)
            break;
        if ((threadIdx.x & 31) == 0)
            u = nfix + (uint32_t)atomicAdd(q.ctr, 1ull);
        u = __shfl_sync(0xffffffffu, u, 0);
        if ((int64_t)u >= q.nstar_units)
            break;
    }
}

// attitude or instrument column j of A32^T q from the units' sums and the
// instrument totals (fixed order)
__device__ __forceinline__ double q_from_units(const SysView &A, const uint32_t *__restrict__ useg,
                                               const double *__restrict__ S,
                                               const double *__restrict__ ipart, int npart,
                                               int64_t j)
{
    double t = 0.0;
    if (j < A.ins0) {
        const int64_t c = j - A.att0;
        const int64_t a = (c >= A.D) + (c >= 2 * A.D), k = c - a * A.D;
#pragma unroll
        for (int jj = 0; jj < 4; jj++) {
            const int64_t o = k - jj;
            if (o >= 0 && o < A.nseg) {
                const uint32_t u0 = __ldg(useg + o), u1 = __ldg(useg + o + 1);
#pragma unroll 4
                for (uint32_t u = u0; u < u1; u++)
                    t += S[(int64_t)u * kNAtt + 4 * a + jj];
            }
        }
    } else {
        const int64_t f = j - A.ins0;
        for (int q = 0; q < npart; q++)
            t += ipart[(int64_t)q * A.I + f];
    }
    return t;
}

// out += the attitude and instrument columns of A32^T q; resets the counter
__global__ void __launch_bounds__(kThreads)
k_f32_combine(SysView A, const uint32_t *__restrict__ useg, const double *__restrict__ S,
              const double *__restrict__ ipart, int npart, double *__restrict__ out,
              unsigned long long *ctr, Ell E)
{
    if (blockIdx.x == 0 && threadIdx.x == 0)
        *ctr = 0ull;
    if (npart == 0)  // the instruments' partials of the row windows
        for (int64_t f = gtid32() >> 5; f < A.I; f += gstride32() >> 5) {
            const double t = ell_total(E, f, A.I);
            if ((threadIdx.x & 31) == 0)
                out[A.ins0 + f] += t;
        }
    const int64_t end = npart ? A.glb0 : A.ins0;
    for (int64_t j = A.att0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < end;
         j += (int64_t)gridDim.x * blockDim.x)
        out[j] += q_from_units(A, useg, S, ipart, npart, j);
}

// ---------------------------------------------------------------------------
// vector kernels (FP64)
// ---------------------------------------------------------------------------

__global__ void k_to_f32(const double *__restrict__ a, float *__restrict__ b, int64_t n)
{
    for (int64_t j = gtid32(); j < n; j += gstride32())
        b[j] = __double2float_rn(a[j]);
}

// Entry j of a binary32 x: the astrometric part as 8 floats (one sector) per
// star, the rest in place
__device__ __forceinline__ void store_x32(float *__restrict__ x32, float *__restrict__ x8,
                                          int64_t att0, int64_t j, float v)
{
    if (j < att0) {
        const int64_t s = j / kNAstro;
        x8[8 * s + (j - kNAstro * s)] = v;
    } else {
        x32[j] = v;
    }
}
__device__ __forceinline__ void store_x32(double *__restrict__ xp, float *, int64_t, int64_t j,
                                          double v)
{
    xp[j] = v;
}

// API form: x32 = fl32(x)
__global__ void k_x_to_f32(const double *__restrict__ x, float *__restrict__ x32,
                           float *__restrict__ x8, int64_t n, int64_t att0)
{
    for (int64_t j = gtid32(); j < n; j += gstride32())
        store_x32(x32, x8, att0, j, __double2float_rn(x[j]));
}

// s = p o c, d = s, z = 0, xp32 = fl32(p o d), gamma = |s|^2; clears the
// instrumental/global part of t for the first inner aprod 2
template <typename XT>
__global__ void __launch_bounds__(kThreads)
k_cg_init(const double *__restrict__ p, const double *__restrict__ c, double *__restrict__ s,
          double *__restrict__ d, double *__restrict__ z, XT *__restrict__ xp32,
          double *__restrict__ t, int64_t n, int64_t ins0, CgState *cg, const CgArgs *args,
          double *partial, unsigned *counter, cudaGraphConditionalHandle loop, int in_graph,
          float *__restrict__ x8, int64_t att0)
{
    double acc[1] = {0.0};
    for (int64_t j = gtid32(); j < n; j += gstride32()) {
        const double sj = p[j] * c[j];
        s[j] = sj;
        d[j] = sj;
        z[j] = 0.0;
        store_x32(xp32, x8, att0, j, (XT)(p[j] * sj));
        if (j >= ins0)
            t[j] = 0.0;
        acc[0] = fma(sj, sj, acc[0]);
    }
    if (grid_reduce<1>(acc, partial, counter) && threadIdx.x == 0) {
        CgState g = {};
        g.gamma = acc[0];
        g.gamma0 = acc[0];
        g.stop2 = args->tol * args->tol * acc[0];
        if (!(acc[0] > 0.0) || args->max_inner < 1) {
            g.done = 1;
            if (in_graph)
                cudaGraphSetConditional(loop, 0u);
        }
        *cg = g;
    }
}

// Where the column sums of aprod 2 are when k_cg_vec1 reads them
enum CgSums {
    kSumsDone = 0,   // all in t
    kSumsUnits = 1,  // binary32 form: units of Att32 and the instruments' partials
    kSumsParts = 2   // FP64 single-launch aprod 2: its partial sums
};

// s -= alpha p o t, z += alpha d, gamma' = |s|^2; the last block forms beta
// and applies the inner stopping rule.  SUMS: t holds the astrometric part
// (and the global column but for kSumsParts), the other columns are added up
// here (no combine launch); with kSumsParts the global column comes from one
// fixed slice of the star units' partials per block, added by the last block.
// The last block resets the work counter.
template <int SUMS>
__global__ void __launch_bounds__(kThreads)
k_cg_vec1(const SysView A, const double *__restrict__ p, const double *__restrict__ t,
          double *__restrict__ s, const double *__restrict__ d, double *__restrict__ z, CgState *cg,
          const CgArgs *args, double *partial, unsigned *counter,
          cudaGraphConditionalHandle loop, int in_graph, const uint32_t *__restrict__ useg, A2Parts P,
          const int *kerr)
{
    const int64_t n = A.n;
    const double alpha = cg->alpha;
    const bool late = threadIdx.x == 0 && wait_expired(kerr);
    double acc[SUMS == kSumsParts ? 2 : 1] = {};
    // column j with t_j = tf(): the loads of the vectors come first
    auto update = [&](int64_t j, auto tf) {
        const double dj = d[j], zo = z[j], pj = p[j], so = s[j];
        const double sj = fma(-alpha, pj * tf(), so);
        z[j] = fma(alpha, dj, zo);
        s[j] = sj;
        acc[0] = fma(sj, sj, acc[0]);
    };
    // instruments in row windows, or with many window totals: a warp each
    const bool win = SUMS == kSumsUnits && P.isplit == 0;
    const bool warp_instr = win || (SUMS == kSumsParts && P.isplit > kThreadParts);
    if (warp_instr) {
        for (int64_t f = gtid32() >> 5; f < A.I; f += gstride32() >> 5) {
            double v = 0.0;
            if (win) {
                v = ell_total(P.ell, f, A.I);
            } else {
                for (int qq = threadIdx.x & 31; qq < P.isplit; qq += 32)
                    v += P.ipart[(int64_t)qq * A.I + f];
                v = warp_sum(v);
            }
            if ((threadIdx.x & 31) == 0)
                update(A.ins0 + f, [&] { return v; });
        }
    }
    for (int64_t j = gtid32(); j < n; j += gstride32()) {
        if (warp_instr && j >= A.ins0 && j < A.glb0)
            continue;
        if (SUMS == kSumsParts && j == A.glb0)
            continue;  // the last block
        update(j, [&] {
            if (SUMS == kSumsDone || j < A.att0 || j >= A.glb0)
                return t[j];
            return SUMS == kSumsUnits ? q_from_units(A, useg, P.S, P.ipart, P.isplit, j)
                                      : q_from_parts(A, P, j);
        });
    }
    if constexpr (SUMS == kSumsParts) {
        const uint32_t per = ((uint32_t)P.ngpart + gridDim.x - 1) / gridDim.x;
        const uint32_t b0 = blockIdx.x * per, b1 = min((uint32_t)P.ngpart, b0 + per);
        for (uint32_t b = b0 + threadIdx.x; b < b1; b += blockDim.x)
            acc[1] += P.gpart[b];
    }
    if (grid_reduce(acc, partial, counter) && threadIdx.x == 0) {
        CgState g = *cg;
        double gnew = acc[0];
        if constexpr (SUMS == kSumsParts) {
            const int64_t j = A.glb0;
            const double sj = fma(-alpha, p[j] * acc[1], s[j]);
            z[j] = fma(alpha, d[j], z[j]);
            s[j] = sj;
            gnew = fma(sj, sj, gnew);
        }
        if (SUMS != kSumsDone)
            *P.ctr = 0ull;
        g.beta = gnew / g.gamma;
        g.gamma = gnew;
        g.it += 1;
        const bool bad = !isfinite(gnew) || !isfinite(g.alpha);
        if (bad)
            g.nonfinite = 1;
        g.late = late;
        if (bad || late || g.it >= args->max_inner || gnew <= g.stop2 || g.xi <= 0.0) {
            g.done = 1;
            if (in_graph)
                cudaGraphSetConditional(loop, 0u);
        }
        *cg = g;
    }
}

// d = s + beta d, xp32 = fl32(p o d); clears the instrumental/global part of t
// (the FP64 form: the binary32 products write theirs)
template <typename XT>
__global__ void k_cg_vec2(const double *__restrict__ p, const double *__restrict__ s,
                          double *__restrict__ d, XT *__restrict__ xp32, double *__restrict__ t,
                          int64_t n, int64_t ins0, const CgState *cg, float *__restrict__ x8,
                          int64_t att0)
{
    const double beta = cg->beta;
    for (int64_t j = gtid32(); j < n; j += gstride32()) {
        const double dj = fma(beta, d[j], s[j]);
        d[j] = dj;
        store_x32(xp32, x8, att0, j, (XT)(p[j] * dj));
        if (j >= ins0)
            t[j] = 0.0;
    }
}

// x += p o z
__global__ void k_axpy_p(const double *__restrict__ p, const double *__restrict__ z,
                         double *__restrict__ x, int64_t n)
{
    for (int64_t j = gtid32(); j < n; j += gstride32())
        x[j] = fma(p[j], z[j], x[j]);
}

// y = b - y_neg_source ... (r = b; r -= A x is done as r = b, aprod1 with -x)
__global__ void k_neg(const double *__restrict__ a, double *__restrict__ b, int64_t n)
{
    for (int64_t j = gtid32(); j < n; j += gstride32())
        b[j] = -a[j];
}

// |p o c|^2 and |r|^2 for the outer stopping rule
__global__ void __launch_bounds__(kThreads)
k_outer_norms(const double *__restrict__ p, const double *__restrict__ c, int64_t n,
              const double *__restrict__ r, int64_t m, double *out2, double *partial,
              unsigned *counter)
{
    double acc[2] = {0.0, 0.0};
    for (int64_t j = gtid32(); j < n; j += gstride32()) {
        const double v = p[j] * c[j];
        acc[0] = fma(v, v, acc[0]);
    }
    for (int64_t i = gtid32(); i < m; i += gstride32())
        acc[1] = fma(r[i], r[i], acc[1]);
    if (grid_reduce<2>(acc, partial, counter) && threadIdx.x == 0) {
        out2[0] = acc[0];
        out2[1] = acc[1];
    }
}

// number of nonempty columns from the column sums of squares
__global__ void k_count_pos(const double *__restrict__ a, int64_t n, double *partial,
                            unsigned *counter, double *out)
{
    double acc[1] = {0.0};
    for (int64_t j = gtid32(); j < n; j += gstride32())
        acc[0] += (a[j] > 0.0) ? 1.0 : 0.0;
    if (grid_reduce<1>(acc, partial, counter) && threadIdx.x == 0)
        *out = acc[0];
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static A2Queue rest_queue(const gsr_handle_t *h)
{
    return a2_queue(h, 8, (int64_t)h->sys.I * h->nq32 * h->ks32, 0);
}

template <int MODE, int X>
static cudaError_t main_launch(const gsr_handle_t *h, double *y, double *glb, cudaStream_t st)
{
    const size_t smem = main_smem(X) + (X == kXGlobal ? 0 : (size_t)h->sys.I * sizeof(float));
    k_f32_main<MODE, X><<<h->grid_main32, kMainThreads, smem, st>>>(
        h->sys, h->att32, h->d_x32, h->d_x8, h->d_q32, y, h->d_attS32, glb, h->d_cg,
        h->d_partial + kRedU * kPartialsPerKind, h->d_counter + kRedU, h->d_kerr);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t f32_main(const gsr_handle_t *h, double *y, double *glb, cudaStream_t st)
{
    if (h->sys.I <= kXThreeMax)
        return main_launch<MODE, kXThree>(h, y, glb, st);
    if (h->sys.I <= kXTwoMax)
        return main_launch<MODE, kXTwo>(h, y, glb, st);
    return main_launch<MODE, kXGlobal>(h, y, glb, st);
}

// the rest of aprod 2 over the row-ordered q32: stars and instruments; *P:
// where the attitude and instrument sums are (isplit 0: in the row windows'
// partials)
template <int MODE, int G>
static cudaError_t rest_win(const gsr_handle_t *h, double *out, cudaStream_t st)
{
    // at most two star groups a unit: the 8 warps that start with stars end
    // nearer to the 16 of the windows (113 -> 106 us at m = 7.0e6)
    A2Queue q = a2_queue(h, G, 0, 0);
    if (q.star_k > 2) {
        q.star_k = 2;
        q.nstar_units = (q.nstar_groups + 1) / 2;
    }
    k_f32_rest_win<G, MODE><<<h->nsm, kRestThreads, kEllSmem32 + h->ell.nacc * sizeof(double), st>>>(
        h->sys, h->att32, h->ell, h->d_q32, out, q, h->d_kerr);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t f32_rest(const gsr_handle_t *h, double *out, A2Parts *P, cudaStream_t st)
{
    *P = {h->d_attS32, h->d_ipart, h->ell_on ? 0 : h->nq32 * h->ks32, nullptr, 0, h->d_a2ctr, h->ell};
    if (h->ell_on) {
        // a lane takes about as many rows of long stars with more lanes
        const int64_t mean = h->sys.m / h->sys.S;
        return mean >= 256 ? rest_win<MODE, 32>(h, out, st)
                           : (mean >= 128 ? rest_win<MODE, 16>(h, out, st)
                                          : rest_win<MODE, 8>(h, out, st));
    }
    const A2Queue q = rest_queue(h);
    if (h->nq32 > 1)
        k_f32_rest<8, MODE, true><<<h->grid_rest32, kThreads, 0, st>>>(
            h->sys, h->att32, h->d_q32, out, h->d_cseg32, h->d_irow, h->d_ival32, h->d_ipart,
            h->nq32, h->ks32, q);
    else
        k_f32_rest<8, MODE, false><<<h->grid_rest32, kThreads, 0, st>>>(
            h->sys, h->att32, h->d_q32, out, h->d_iseg, h->d_irow, h->d_ival32, h->d_ipart, 1,
            h->ks32, q);
    return cudaGetLastError();
}

// API forms (FP64 vectors in and out)
cudaError_t launch_aprod1_f32_api(const gsr_handle_t *h, const double *x, double *y, cudaStream_t st)
{
    k_x_to_f32<<<h->grid_vec, kThreads, 0, st>>>(x, h->d_x32, h->d_x8, h->sys.n, h->sys.att0);
    return f32_main<kF32A1>(h, y, nullptr, st);
}

cudaError_t launch_aprod2_f32_api(const gsr_handle_t *h, const double *y, double *x, cudaStream_t st)
{
    k_to_f32<<<h->grid_vec, kThreads, 0, st>>>(y, h->d_q32, h->sys.m);
    cudaError_t e = f32_main<kF32A2>(h, nullptr, x + h->sys.glb0, st);
    A2Parts P;
    if (e == cudaSuccess)
        e = f32_rest<kA2Accumulate>(h, x, &P, st);
    if (e != cudaSuccess)
        return e;
    k_f32_combine<<<h->nsm * 2, kThreads, 0, st>>>(h->sys, h->d_useg, P.S, P.ipart, P.isplit, x,
                                                   P.ctr, P.ell);
    return cudaGetLastError();
}

[[nodiscard]] static cudaError_t cg_prologue(const gsr_handle_t *h, cudaStream_t s,
                                             cudaGraphConditionalHandle loop, int in_graph)
{
    const SysView &A = h->sys;
    k_cg_init<float><<<h->grid_vec, kThreads, 0, s>>>(h->d_p, h->d_c, h->d_s, h->d_d, h->d_zc, h->d_x32,
                                                h->d_t, A.n, A.ins0, h->d_cg, h->d_cgargs,
                                                h->d_partial + kRedBnorm * kPartialsPerKind,
                                                h->d_counter + kRedBnorm, loop, in_graph,
                                                h->d_x8, A.att0);
    return cudaGetLastError();
}

[[nodiscard]] static cudaError_t cg_iteration(const gsr_handle_t *h, cudaStream_t s,
                                              cudaGraphConditionalHandle loop, int in_graph)
{
    const SysView &A = h->sys;
    A2Parts P;
    cudaError_t e = f32_main<kF32A1 | kF32A2>(h, nullptr, h->d_t + A.glb0, s);
    if (e == cudaSuccess)
        e = f32_rest<kA2Overwrite>(h, h->d_t, &P, s);
    if (e != cudaSuccess)
        return e;
    k_cg_vec1<kSumsUnits><<<h->grid_vec, kThreads, 0, s>>>(A, h->d_p, h->d_t, h->d_s, h->d_d,
                                                           h->d_zc, h->d_cg, h->d_cgargs,
                                                           h->d_partial + kRedV * kPartialsPerKind,
                                                           h->d_counter + kRedV, loop, in_graph,
                                                           h->d_useg, P, h->d_kerr);
    k_cg_vec2<float><<<h->grid_vec, kThreads, 0, s>>>(h->d_p, h->d_s, h->d_d, h->d_x32, h->d_t, A.n, A.n,
                                                h->d_cg, h->d_x8, A.att0);
    return cudaGetLastError();
}

#define CG_TRY(x)                       \
    do {                                \
        cudaError_t e_ = (x);           \
        if (e_ != cudaSuccess) {        \
            err = e_;                   \
            goto fail;                  \
        }                               \
    } while (0)

cudaError_t find_graph_leaf(cudaGraph_t g, cudaGraphNode_t *leaf);

// graph: [CG init] -> WHILE(flag) { CG iteration } -> [x += p o z]
cudaError_t build_cg_graph(gsr_handle_t *h)
{
    cudaError_t err = cudaSuccess;
    cudaGraph_t g = nullptr;
    cudaGraphConditionalHandle loop;
    cudaGraphNode_t pre_leaf, wnode;
    cudaGraphNodeParams cp = {};
    cudaGraph_t body;
    cudaStream_t s = h->cap_stream;
    CG_TRY(cudaGraphCreate(&g, 0));
    CG_TRY(cudaGraphConditionalHandleCreate(&loop, g, 1u, cudaGraphCondAssignDefault));
    CG_TRY(cudaStreamBeginCaptureToGraph(s, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    CG_TRY(cg_prologue(h, s, loop, 1));
    CG_TRY(cudaStreamEndCapture(s, &g));
    CG_TRY(find_graph_leaf(g, &pre_leaf));
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = loop;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    CG_TRY(cudaGraphAddNode(&wnode, g, &pre_leaf, nullptr, 1, &cp));
    body = cp.conditional.phGraph_out[0];
    CG_TRY(cudaStreamBeginCaptureToGraph(s, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    CG_TRY(cg_iteration(h, s, loop, 1));
    CG_TRY(cudaStreamEndCapture(s, &body));
    CG_TRY(cudaStreamBeginCaptureToGraph(s, g, &wnode, nullptr, 1, cudaStreamCaptureModeThreadLocal));
    k_axpy_p<<<h->grid_vec, kThreads, 0, s>>>(h->d_p, h->d_zc, h->d_xm, h->sys.n);
    CG_TRY(cudaGetLastError());
    CG_TRY(cudaStreamEndCapture(s, &g));
    CG_TRY(cudaGraphInstantiate(&h->cg_exec, g, 0));
    cudaGraphDestroy(g);
    return cudaSuccess;
fail:
    {
        cudaStreamCaptureStatus cs;
        if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
            cudaGraph_t junk = nullptr;
            cudaStreamEndCapture(s, &junk);
            if (junk && junk != g)
                cudaGraphDestroy(junk);
        }
    }
    if (g)
        cudaGraphDestroy(g);
    cudaGetLastError();
    return err;
}

// one inner solve: graph, or host-driven launches in eager mode
cudaError_t run_cg(gsr_handle_t *h, cudaStream_t st, int max_inner)
{
    if (!h->cfg.eager)
        return cudaGraphLaunch(h->cg_exec, st);
    cudaError_t e = cg_prologue(h, st, 0, 0);
    for (int it = 0; e == cudaSuccess && it < max_inner; it++) {
        e = cudaMemcpyAsync(h->h_cg, h->d_cg, sizeof(CgState), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(st);
        if (e != cudaSuccess || h->h_cg->done)
            break;
        e = cg_iteration(h, st, 0, 0);
    }
    if (e == cudaSuccess) {
        k_axpy_p<<<h->grid_vec, kThreads, 0, st>>>(h->d_p, h->d_zc, h->d_xm, h->sys.n);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t launch_outer_norms(const gsr_handle_t *h, const double *r, cudaStream_t st)
{
    k_outer_norms<<<h->grid_vec, kThreads, 0, st>>>(h->d_p, h->d_c, h->sys.n, r, h->sys.m,
                                                     h->d_onorm, h->d_partial + kRedU * kPartialsPerKind,
                                                     h->d_counter + kRedU);
    return cudaGetLastError();
}

cudaError_t launch_norms2(const gsr_handle_t *h, const double *c, const double *r, double *out2,
                          cudaStream_t st)
{
    k_outer_norms<<<h->grid_vec, kThreads, 0, st>>>(h->d_p, c, h->sys.n, r, h->sys.m, out2,
                                                     h->d_partial + kRedU * kPartialsPerKind,
                                                     h->d_counter + kRedU);
    return cudaGetLastError();
}

cudaError_t launch_neg(const gsr_handle_t *h, const double *a, double *b, int64_t n, cudaStream_t st)
{
    k_neg<<<h->grid_vec, kThreads, 0, st>>>(a, b, n);
    return cudaGetLastError();
}

cudaError_t launch_count_pos(const gsr_handle_t *h, const double *a, double *out, cudaStream_t st)
{
    k_count_pos<<<h->grid_vec, kThreads, 0, st>>>(a, h->sys.n, h->d_partial + kRedU * kPartialsPerKind,
                                                   h->d_counter + kRedU, out);
    return cudaGetLastError();
}

cudaError_t launch_to_f32(const gsr_handle_t *h, const double *a, float *b, int64_t n, cudaStream_t st)
{
    k_to_f32<<<h->nsm * 8, kThreads, 0, st>>>(a, b, n);
    return cudaGetLastError();
}

// one block per SM, no more than the units need
int f32_main_grid(const gsr_handle_t *h)
{
    // the most that any handle of this process asks for: the attribute is
    // shared by all of them
    const struct {
        const void *f;
        size_t smem;
    } fns[9] = {
#define GSR_MAIN(X, MAX)                                                    \
    {(const void *)k_f32_main<1, X>, main_smem(X) + (MAX) * sizeof(float)}, \
    {(const void *)k_f32_main<2, X>, main_smem(X) + (MAX) * sizeof(float)}, \
    {(const void *)k_f32_main<3, X>, main_smem(X) + (MAX) * sizeof(float)}
        GSR_MAIN(kXGlobal, 0), GSR_MAIN(kXThree, kXThreeMax), GSR_MAIN(kXTwo, kXTwoMax)
#undef GSR_MAIN
    };
    for (const auto &k : fns)
        if (cudaFuncSetAttribute(k.f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem) !=
            cudaSuccess)
            return -1;
    const int64_t nu = h->att32.nunits;
    return (int)(nu < h->nsm ? nu : h->nsm);
}

int f32_rest_grid(const gsr_handle_t *h)
{
    // the most that any handle of the process may ask for
    const void *fns[6] = {
        (const void *)k_f32_rest_win<8, kA2Accumulate>,  (const void *)k_f32_rest_win<8, kA2Overwrite>,
        (const void *)k_f32_rest_win<16, kA2Accumulate>, (const void *)k_f32_rest_win<16, kA2Overwrite>,
        (const void *)k_f32_rest_win<32, kA2Accumulate>, (const void *)k_f32_rest_win<32, kA2Overwrite>};
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 6 && e == cudaSuccess; i++)
        e = cudaFuncSetAttribute(fns[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(kEllSmem32 + kEllAccMax * sizeof(double)));
    if (e != cudaSuccess)
        return -1;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &occ, k_f32_rest<8, kA2Overwrite, true>, kThreads, 0);
    if (e != cudaSuccess || occ <= 0)
        return -1;
    const A2Queue q = rest_queue(h);
    const int64_t need = (q.total + kThreads / 32 - 1) / (kThreads / 32);
    const int64_t g = (int64_t)h->nsm * occ;
    return (int)(g < need ? g : need);
}

// the binary32 copies from the FP64 values: the offset-ordered tiles, the
// astrometric planes in row order; one plane when k1 >= 0
__global__ void k_atile(SysView A, unsigned char *__restrict__ tile, int k1)
{
    for (int64_t e = gtid32(); e < A.m; e += gstride32()) {
        const int64_t r = A.perm[e];
        const int l = (int)(e & 31);
        unsigned char *tp = tile + (e >> 5) * kAttTileBytes;
        float *v = reinterpret_cast<float *>(tp) + l;
        if (k1 >= 0) {
            v[32 * k1] = (float)A.val[tidx<kNPar>(k1, r)];
            continue;
        }
#pragma unroll
        for (int k = 0; k < kNPar; k++)
            v[32 * k] = (float)A.val[tidx<kNPar>(k, r)];
        uint4 rc = A.rec[r];
        rc.x = star_of_row(A, r >> 5, r);
        reinterpret_cast<uint4 *>(tp + kAttRecAt)[l] = rc;
        reinterpret_cast<uint32_t *>(tp + kAttRowAt)[l] = (uint32_t)r;
    }
}

__global__ void k_sv32(SysView A, float *__restrict__ sv, int k1)
{
    for (int64_t r = gtid32(); r < A.m; r += gstride32()) {
#pragma unroll
        for (int k = 0; k < kNAstro; k++)
            if (k1 < 0 || k == k1)
                sv[tidx<kNAstro>(k, r)] = (float)A.val[tidx<kNPar>(k, r)];
    }
}

cudaError_t build_att32(gsr_handle_t *h, cudaStream_t st)
{
    k_atile<<<h->nsm * 8, kThreads, 0, st>>>(h->sys, h->d_atile, -1);
    k_sv32<<<h->nsm * 8, kThreads, 0, st>>>(h->sys, h->d_sv32, -1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP64 conjugate gradients on the preconditioned normal equations
// (diag(p) A^T A diag(p)) z = diag(p) c, q = p o z: the same recurrences as
// the inner solve above with the FP64 products of gsr_kernels.cu (used for
// the adjoint of the least-squares solution)
// ---------------------------------------------------------------------------
[[nodiscard]] static cudaError_t cg64_prologue(const gsr_handle_t *h, cudaStream_t s,
                                               cudaGraphConditionalHandle loop, int in_graph)
{
    const SysView &A = h->sys;
    k_cg_init<double><<<h->grid_vec, kThreads, 0, s>>>(h->d_p, h->d_c, h->d_s, h->d_d, h->d_zc,
                                                        h->d_xp64, h->d_t, A.n, A.ins0, h->d_cg,
                                                        h->d_cgargs,
                                                        h->d_partial + kRedBnorm * kPartialsPerKind,
                                                        h->d_counter + kRedBnorm, loop, in_graph,
                                                        nullptr, 0);
    return cudaGetLastError();
}

[[nodiscard]] static cudaError_t cg64_iteration(const gsr_handle_t *h, cudaStream_t s,
                                                cudaGraphConditionalHandle loop, int in_graph)
{
    const SysView &A = h->sys;
    cudaError_t e = launch_aprod1_cg(h, h->d_xp64, h->d_q64, s);
    if (e != cudaSuccess)
        return e;
    double *part = h->d_partial + kRedV * kPartialsPerKind;
    unsigned *cnt = h->d_counter + kRedV;
    A2Parts P = {};
    if (aprod2_partials(h, h->d_q64, h->d_t, &P.S, &P.ipart, &P.isplit, &P.gpart, &P.ngpart, &P.ctr,
                        s)) {
        k_cg_vec1<kSumsParts><<<h->grid_vec, kThreads, 0, s>>>(A, h->d_p, h->d_t, h->d_s, h->d_d,
                                                               h->d_zc, h->d_cg, h->d_cgargs, part,
                                                               cnt, loop, in_graph, nullptr, P, h->d_kerr);
    } else {
        e = launch_aprod2(h, h->d_q64, h->d_t, kA2Overwrite, s);
        if (e != cudaSuccess)
            return e;
        k_cg_vec1<kSumsDone><<<h->grid_vec, kThreads, 0, s>>>(A, h->d_p, h->d_t, h->d_s, h->d_d,
                                                              h->d_zc, h->d_cg, h->d_cgargs, part,
                                                              cnt, loop, in_graph, nullptr, P, h->d_kerr);
    }
    k_cg_vec2<double><<<h->grid_vec, kThreads, 0, s>>>(h->d_p, h->d_s, h->d_d, h->d_xp64, h->d_t,
                                                        A.n, A.ins0, h->d_cg, nullptr, 0);
    return cudaGetLastError();
}

cudaError_t build_cg64_graph(gsr_handle_t *h)
{
    cudaError_t err = cudaSuccess;
    cudaGraph_t g = nullptr;
    cudaGraphConditionalHandle loop;
    cudaGraphNode_t pre_leaf, wnode;
    cudaGraphNodeParams cp = {};
    cudaGraph_t body;
    cudaStream_t s = h->cap_stream;
    CG_TRY(cudaGraphCreate(&g, 0));
    CG_TRY(cudaGraphConditionalHandleCreate(&loop, g, 1u, cudaGraphCondAssignDefault));
    CG_TRY(cudaStreamBeginCaptureToGraph(s, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    CG_TRY(cg64_prologue(h, s, loop, 1));
    CG_TRY(cudaStreamEndCapture(s, &g));
    CG_TRY(find_graph_leaf(g, &pre_leaf));
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = loop;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    CG_TRY(cudaGraphAddNode(&wnode, g, &pre_leaf, nullptr, 1, &cp));
    body = cp.conditional.phGraph_out[0];
    CG_TRY(cudaStreamBeginCaptureToGraph(s, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    CG_TRY(cg64_iteration(h, s, loop, 1));
    CG_TRY(cudaStreamEndCapture(s, &body));
    CG_TRY(cudaStreamBeginCaptureToGraph(s, g, &wnode, nullptr, 1, cudaStreamCaptureModeThreadLocal));
    k_axpy_p<<<h->grid_vec, kThreads, 0, s>>>(h->d_p, h->d_zc, h->d_xm, h->sys.n);
    CG_TRY(cudaGetLastError());
    CG_TRY(cudaStreamEndCapture(s, &g));
    CG_TRY(cudaGraphInstantiate(&h->cg64_exec, g, 0));
    cudaGraphDestroy(g);
    return cudaSuccess;
fail:
    {
        cudaStreamCaptureStatus cs;
        if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
            cudaGraph_t junk = nullptr;
            cudaStreamEndCapture(s, &junk);
            if (junk && junk != g)
                cudaGraphDestroy(junk);
        }
    }
    if (g)
        cudaGraphDestroy(g);
    cudaGetLastError();
    return err;
}

cudaError_t run_cg64(gsr_handle_t *h, cudaStream_t st, int max_iter)
{
    if (!h->cfg.eager)
        return cudaGraphLaunch(h->cg64_exec, st);
    cudaError_t e = cg64_prologue(h, st, 0, 0);
    for (int it = 0; e == cudaSuccess && it < max_iter; it++) {
        e = cudaMemcpyAsync(h->h_cg, h->d_cg, sizeof(CgState), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(st);
        if (e != cudaSuccess || h->h_cg->done)
            break;
        e = cg64_iteration(h, st, 0, 0);
    }
    if (e == cudaSuccess) {
        k_axpy_p<<<h->grid_vec, kThreads, 0, st>>>(h->d_p, h->d_zc, h->d_xm, h->sys.n);
        e = cudaGetLastError();
    }
    return e;
}

// binary32 copies of plane k after it changed
cudaError_t launch_f32_plane(const gsr_handle_t *h, int k, cudaStream_t st)
{
    k_atile<<<h->nsm * 8, kThreads, 0, st>>>(h->sys, h->d_atile, k);
    if (k < kNAstro)
        k_sv32<<<h->nsm * 8, kThreads, 0, st>>>(h->sys, h->d_sv32, k);
    return cudaGetLastError();
}

}  // namespace gsr
