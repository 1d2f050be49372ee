// Batched k right-hand-side solve: the mixed-precision refinement of
// gsr_mixed.cu for k right-hand sides at once.  The inner products become
// skinny sparse-times-dense products: every row's binary32 values are read
// once per column tile and applied to KT columns (KT = 1, 2, 4 or 8), so the
// matrix traffic of k solves is paid ceil(k/KT) times instead of k times.
//
// Dense blocks of the inner solve are stored in panels of 8 columns: entry
// (j, c) of a block with `rows` rows is at ((c / 8) rows + j) 8 + c % 8
// (pidx).  A column tile of KT <= 8 columns lies in one panel, so the gather
// of unknown j fetches KT consecutive values (one 32-byte sector for KT = 8
// binary32) and a tile's gathers touch only its own rows x 8 panel, whatever
// the number of columns (with one row-major block of leading dimension k, 32
// columns spread a tile's sectors over four times the address range and its
// products ran 1.7x slower than at 8 columns).
//
// Column sections (Att32 layout, gsr_internal.cuh):
//   A X with the attitude and global part of A^T Q: one pass over the
//            offset-ordered values (k_b_main);
//   astrometric: star-parallel, G lanes per star, in row order;
//   instrumental: instrument-sorted copy, pieces of one instrument per warp.
// Every sum has a fixed order: no atomics on values.
// CG: k independent Hestenes-Stiefel recurrences with per-column scalars.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "gsr_att32.cuh"
#include "gsr_df.cuh"
#include "gsr_internal.cuh"
#include "gsr_lsqr.cuh"
#include "gsr_reduce.cuh"

namespace gsr {

// A stream and the events that fork it from another one and join it again
// while the inner loop is captured; released with the object, the graph keeps
// the branch.
struct Branch {
    cudaStream_t s = nullptr;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    cudaError_t make()
    {
        cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
        for (int i = 0; i < 2 && e == cudaSuccess; i++)
            e = cudaEventCreateWithFlags(&ev[i], cudaEventDisableTiming);
        return e;
    }
    cudaError_t fork(cudaStream_t from)
    {
        const cudaError_t e = cudaEventRecord(ev[0], from);
        return e == cudaSuccess ? cudaStreamWaitEvent(s, ev[0], 0) : e;
    }
    cudaError_t join(cudaStream_t to)
    {
        const cudaError_t e = cudaEventRecord(ev[1], s);
        return e == cudaSuccess ? cudaStreamWaitEvent(to, ev[1], 0) : e;
    }
    ~Branch()
    {
        for (cudaEvent_t e : ev)
            if (e)
                cudaEventDestroy(e);
        if (s)
            cudaStreamDestroy(s);
    }
};

// The branches of an iteration: the second run of tiles beside the first, in
// each run the instrument pass beside the star pass
struct BatchSide {
    Branch run, instr[2];
    cudaError_t make()
    {
        cudaError_t e = run.make();
        for (int i = 0; i < 2 && e == cudaSuccess; i++)
            e = instr[i].make();
        return e;
    }
};

constexpr int kPanel = 8;  // columns per panel of the dense blocks

// offset of entry (r, c) in a panelled block of `rows` rows
__host__ __device__ __forceinline__ int64_t pidx(int64_t r, int64_t rows, int c)
{
    return ((int64_t)(c / kPanel) * rows + r) * kPanel + (c % kPanel);
}

// KT consecutive columns of one row as packed pairs (one scalar for KT = 1)
template <int KT>
struct Cols {
    typedef f32x2 V;
    static constexpr int N = KT / 2;
};
template <>
struct Cols<1> {
    typedef float V;
    static constexpr int N = 1;
};

__device__ __forceinline__ void v_bcast(float &d, float a) { d = a; }
__device__ __forceinline__ void v_bcast(f32x2 &d, float a) { d = pack2(a, a); }

// The KT = 8 row is one aligned 32-byte sector, fetched by one 256-bit load:
// random rows arrive at 0.93 per clock and SM from L2 (1.6 from L1) against
// 0.56 with two 128-bit loads.
template <int KT>
__device__ __forceinline__ void load_cols(const float *__restrict__ p,
                                          typename Cols<KT>::V (&v)[Cols<KT>::N])
{
    if constexpr (KT == 8) {
        asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];"
            : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p));
    } else if constexpr (KT == 4) {
        asm("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(v[0]), "=l"(v[1]) : "l"(p));
    } else if constexpr (KT == 2) {
        asm("ld.global.nc.b64 %0, [%1];" : "=l"(v[0]) : "l"(p));
    } else {
        v[0] = __ldg(p);
    }
}

template <int KT>
__device__ __forceinline__ void store_cols(float *p, const typename Cols<KT>::V (&v)[Cols<KT>::N])
{
    if constexpr (KT == 1) {
        *p = v[0];
    } else if constexpr (KT == 2) {
        *reinterpret_cast<f32x2 *>(p) = v[0];
    } else {
        ulonglong2 *d = reinterpret_cast<ulonglong2 *>(p);
#pragma unroll
        for (int i = 0; i < Cols<KT>::N / 2; i++)
            d[i] = make_ulonglong2(v[2 * i], v[2 * i + 1]);
    }
}

// column c (compile time) of a packed row
template <int KT>
__device__ __forceinline__ float col_of(const typename Cols<KT>::V (&v)[Cols<KT>::N], int c)
{
    if constexpr (KT == 1) {
        return v[0];
    } else {
        float a, b;
        unpack2(v[c / 2], a, b);
        return (c & 1) ? b : a;
    }
}

// Tiles of KT columns: every kernel below takes the tiles of one launch from
// blockIdx.y (tile y: columns c_first + y KT ...).  Tiles are independent, so
// one launch covers all of them: on a system too small to fill the chip with
// one tile they run side by side, on a large one the blocks of a tile are
// dispatched before those of the next and keep its panel in L2.

// the products of one launch of the main kernel
constexpr int kBA1 = 1;  // Q = A32 X
constexpr int kBA2 = 2;  // attitude and global part of A32^T Q

// ---------------------------------------------------------------------------
// Main pass over the offset-ordered values on KT columns, units as in
// k_f32_main.  A1: Q32[row, c0+c] = fl32(A32 X32[:, c0+c]) with |Q[:, c]|^2
// and alpha_c = gamma_c / |Q[:, c]|^2 (0 for a finished column); A2: the
// attitude sums of A32^T Q into S[unit][4a + j][c] of the tile's block and
// T[global], on the Q just formed (or on Q itself without A1).
// The row sums take one row per lane.  The attitude sums take one output per
// lane (tap 4a + j, column c), 12 KT of them in NI rounds: their accumulators
// are a few registers instead of 24 KT, and a unit needs no reduction over
// the warp.  They read the values from the tile's stage and the rows of Q
// through shared memory, two rows per packed operation (even and odd rows are
// two chains); the lanes of different taps start 8 rows apart, so that they
// read different banks.  A chain ends with its tile, after 16 terms, and the
// tiles of a unit are added in three words: a lane per row had chains of a
// thirty-second of the offset's rows and a tree over the lanes (rms error in
// units of the sum of |terms|, 50 / 200 / 350 / 1,000 rows an offset: 3.9 / 4.9
// / 5.5 / 8.6e-18; now 2.7 / 2.5 / 1.9 / 0.7e-18; one chain over the unit had
// 9.8 / 43 / 26 / 23e-18).
// Bound by the FP32 pipe: 8 lane operations per product, 37 products a row
// and column (0.47 ms at 7.0e6 rows and 8 columns with all lanes busy; 0.73
// measured, against 0.76 + 0.39 ms for the two products as passes in row order
// and in offset order; 0.69 with one chain over the unit).
// ---------------------------------------------------------------------------
constexpr int kBWarps = 16;  // one block per SM
constexpr int kBThreads = 32 * kBWarps;
constexpr int kBStages = 2;
constexpr int kBRow = 34;  // row stride of Q in shared memory: distinct banks, 8-byte aligned pairs

// one warp's shared memory
template <int KT>
struct alignas(128) BWarp {
    unsigned char stage[kBStages * kAttTileBytes];
    float x[kNAtt][KT];  // attitude rows of X of the unit
    float q[KT][kBRow];  // Q of the tile's rows
    uint64_t bar[kBStages];
};

// this lane's attitude sums over the rows of a tile; rows outside lo .. hi-1
// (a tile shared with another offset) are skipped
template <int KT, int NI, bool FULL>
__device__ __forceinline__ void b_att_tile(const float *__restrict__ val, const BWarp<KT> &W,
                                           int lane, int lo, int hi, f32x2 (&sh)[NI], f32x2 (&sl)[NI])
{
    const int g = lane / KT;
#pragma unroll 4
    for (int i2 = 0; i2 < 32; i2 += 2) {
        const int rr = (i2 + 8 * g) & 31;
        f32x2 qv = *reinterpret_cast<const f32x2 *>(&W.q[lane % KT][rr]);
#pragma unroll
        for (int i = 0; i < NI; i++) {
            const int k = g + i * (32 / KT);
            f32x2 av = *reinterpret_cast<const f32x2 *>(val + 32 * (kNAstro + (k < kNAtt ? k : 0)) + rr);
            if (!FULL) {
                float a0, a1;
                unpack2(av, a0, a1);
                av = pack2(rr >= lo && rr < hi ? a0 : 0.f, rr + 1 >= lo && rr + 1 < hi ? a1 : 0.f);
            }
            df_acc_v(sh[i], sl[i], v_mul(av, qv));
        }
    }
}

template <int KT, int MODE>
__global__ void __launch_bounds__(kBThreads, 1)
k_b_main(SysView A, Att32 U, const float *__restrict__ X, float *__restrict__ Q,
         double *__restrict__ Sall, double *__restrict__ T, int c_first, BatchState *bs,
         double *partial, unsigned *counter, int *kerr)
{
    typedef typename Cols<KT>::V V;
    constexpr int N = Cols<KT>::N;
    constexpr bool A1 = (MODE & kBA1) != 0, A2 = (MODE & kBA2) != 0;
    constexpr int NOUT = kNAtt * KT, NI = (NOUT + 31) / 32;
    extern __shared__ __align__(128) unsigned char smem[];
    const int c0 = c_first + blockIdx.y * KT;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    BWarp<KT> &W = reinterpret_cast<BWarp<KT> *>(smem)[wib];
    const float *Xp = X + pidx(0, A.n, c0);  // row j of the panel at Xp + 8 j
    float *Qp = Q + pidx(0, A.m, c0);
    double *S = Sall + (int64_t)c0 * U.nunits * kNAtt;
    AttWalk<kBStages> walk(U, W.stage, W.bar, blockIdx.x + (int64_t)gridDim.x * wib,
                           (int64_t)gridDim.x * kBWarps);
    V nh[N], nl[N], gh[N], gl[N];  // |Q[:, c]|^2 and the global sums of this thread
#pragma unroll
    for (int c = 0; c < N; c++)
        nh[c] = nl[c] = gh[c] = gl[c] = V(0);
    Df3<f32x2> su[NI];  // this lane's attitude sums of the unit, even and odd rows
    bool ok = walk.d[0].ok && walk.arrived(0, kerr);
    while (ok) {
        const Visit v = walk.d[0];
        if (v.first()) {
            if (A1) {
                for (int i = lane; i < NOUT; i += 32) {
                    const int k = i / KT, c = i % KT;
                    W.x[k][c] =
                        __ldg(Xp + kPanel * (A.att0 + (k >> 2) * A.D + v.un.x + (k & 3)) + c);
                }
                __syncwarp();
            }
#pragma unroll
            for (int i = 0; i < NI; i++)
                su[i].hi = su[i].lo = su[i].c = 0ull;
        }
        const uint32_t e = (v.t << 5) + lane;
        const float *val = walk.val();  // plane k of the tile at val + 32 k
        V h[N], l[N];
#pragma unroll
        for (int c = 0; c < N; c++)
            h[c] = l[c] = V(0);
        if (e >= v.un.y && e < v.un.z) {
            const float *vk = val + lane;
            const uint32_t r = walk.row();
            V ag;
            v_bcast(ag, vk[32 * (kNPar - 1)]);
            if constexpr (A1) {
                // the rows of X of the star are on their way while the
                // attitude products are formed, those of the instruments
                // while the astrometric ones are
                const uint4 rc = walk.rec(0);
                const float *xs = Xp + (int64_t)kPanel * kNAstro * rc.x;
                V xv[kNAstro][N], xi[kNInstr][N], xg[N];
#pragma unroll
                for (int k = 0; k < kNAstro; k++)
                    load_cols<KT>(xs + kPanel * k, xv[k]);
#pragma unroll
                for (int k = 0; k < kNAtt; k++) {
                    V a;
                    v_bcast(a, vk[32 * (kNAstro + k)]);
#pragma unroll
                    for (int c = 0; c < N; c++)
                        df_acc_v(h[c], l[c], v_mul(a, reinterpret_cast<const V *>(W.x[k])[c]));
                }
#pragma unroll
                for (int j = 0; j < kNInstr; j++)
                    load_cols<KT>(Xp + kPanel * (A.ins0 + instr_at32(rc, j)), xi[j]);
#pragma unroll
                for (int k = 0; k < kNAstro; k++) {
                    V a;
                    v_bcast(a, vk[32 * k]);
#pragma unroll
                    for (int c = 0; c < N; c++)
                        df_acc_v(h[c], l[c], v_mul(a, xv[k][c]));
                }
                load_cols<KT>(Xp + kPanel * A.glb0, xg);
#pragma unroll
                for (int j = 0; j < kNInstr; j++) {
                    V a;
                    v_bcast(a, vk[32 * (17 + j)]);
#pragma unroll
                    for (int c = 0; c < N; c++)
                        df_acc_v(h[c], l[c], v_mul(a, xi[j][c]));
                }
#pragma unroll
                for (int c = 0; c < N; c++)
                    df_acc_v(h[c], l[c], v_mul(ag, xg[c]));
#pragma unroll
                for (int c = 0; c < N; c++) {
                    h[c] = v_add(h[c], l[c]);        // the row's q
                    const V pq = v_mul(h[c], h[c]);  // q^2 = pq + fma(q, q, -pq) exactly
                    df_acc_v(nh[c], nl[c], pq);
                    nl[c] = v_add(nl[c], v_fma(h[c], h[c], v_neg(pq)));
                }
                store_cols<KT>(Qp + (int64_t)kPanel * r, h);
            } else {
                load_cols<KT>(Qp + (int64_t)kPanel * r, h);
            }
            if constexpr (A2) {
#pragma unroll
                for (int c = 0; c < N; c++)
                    df_acc_v(gh[c], gl[c], v_mul(ag, h[c]));
            }
        }
        if constexpr (A2) {
#pragma unroll
            for (int c = 0; c < KT; c++)
                W.q[c][lane] = col_of<KT>(h, c);
            __syncwarp();
            f32x2 sh[NI], sl[NI];  // of the tile
#pragma unroll
            for (int i = 0; i < NI; i++)
                sh[i] = sl[i] = 0ull;
            const uint32_t b = v.t << 5;
            if (v.un.y <= b && v.un.z >= b + 32)
                b_att_tile<KT, NI, true>(val, W, lane, 0, 32, sh, sl);
            else
                b_att_tile<KT, NI, false>(val, W, lane, (int)(max(v.un.y, b) - b),
                                          (int)(min(v.un.z, b + 32) - b), sh, sl);
#pragma unroll
            for (int i = 0; i < NI; i++)
                su[i].add(sh[i], sl[i]);
            if (v.last()) {
#pragma unroll
                for (int i = 0; i < NI; i++) {
                    float h0, h1, l0, l1, c0, c1;
                    unpack2(su[i].hi, h0, h1);
                    unpack2(su[i].lo, l0, l1);
                    unpack2(su[i].c, c0, c1);
                    if (lane + 32 * i < NOUT)
                        S[(int64_t)v.un.w * NOUT + lane + 32 * i] =
                            df_to_d(h0, h1) + (df_to_d(l0, l1) + df_to_d(c0, c1));
                }
            }
        }
        if (!walk.d[1].ok)
            break;
        walk.advance();
        ok = walk.arrived(0, kerr);
    }
    double v[KT];
    if constexpr (A1) {
#pragma unroll
        for (int c = 0; c < KT; c++)
            v[c] = df_to_d(col_of<KT>(nh, c), col_of<KT>(nl, c));
        if (grid_reduce<KT, kBThreads>(v, partial + (int64_t)c0 * kMaxPartials, counter + c0) &&
            threadIdx.x == 0) {
#pragma unroll
            for (int c = 0; c < KT; c++) {
                const int cc = c0 + c;
                bs->xi[cc] = v[c];
                bs->alpha[cc] = (!bs->done[cc] && v[c] > 0.0) ? bs->gamma[cc] / v[c] : 0.0;
            }
        }
    }
    if constexpr (A2) {
#pragma unroll
        for (int c = 0; c < KT; c++)
            v[c] = df_to_d(col_of<KT>(gh, c), col_of<KT>(gl, c));
        if (grid_reduce<KT, kBThreads>(v, partial + (int64_t)(kMaxBatch + c0) * kMaxPartials,
                                       counter + kMaxBatch + c0) && threadIdx.x == 0) {
#pragma unroll
            for (int c = 0; c < KT; c++)
                T[pidx(A.glb0, A.n, c0) + c] = v[c];
        }
    }
}

// ---------------------------------------------------------------------------
// aprod 2, astrometric nonzeros on KT columns (star-parallel): T[astro rows].
// G lanes own a star: KT / 2 lanes take a pair of columns each of one row, G
// over that many rows at a time.  A lane holds five packed sums, so that
// enough warps and rows are in flight (with a whole row of 8 columns per lane:
// 144 registers, 8 warps per SM, 276 us at 7.0e6 rows).  The chain of a lane
// is KT / 2 times as long as with a row per lane; its low word is renormalised
// at each addition (df_acc_norm), which keeps the error of the shorter chains
// (rms in units of the sum of |terms|, 8 columns on 16 lanes, 70 / 200 / 400
// rows a star: 3.6 / 5.7 / 6.4e-18, a row per lane 3.7 / 5.7 / 7.1e-18, without
// it 6.2 / 15 / 29e-18).
// ---------------------------------------------------------------------------
template <int KT, int G>
__global__ void __launch_bounds__(kThreads, 4)
k_b_stars(SysView A, const float *__restrict__ sv, const float *__restrict__ Y,
          double *__restrict__ T, int c_first)
{
    constexpr int KP = KT > 1 ? 2 : 1;  // columns per lane
    typedef typename Cols<KP>::V V;
    constexpr int CL = KT / KP;  // lanes per row
    constexpr int RS = G / CL;   // rows at a time
    constexpr int GPW = 32 / G;
    const int c0 = c_first + blockIdx.y * KT;
    const int lane = threadIdx.x & (G - 1);
    const int gw = (threadIdx.x & 31) / G;
    const int cl = lane % CL, slot = lane / CL;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const float *Yp = Y + pidx(0, A.m, c0) + KP * cl;
    for (int64_t s0 = warp * GPW; s0 < A.S; s0 += nwarps * GPW) {
        const int64_t s = s0 + gw;
        uint32_t r0 = 0, r1 = 0;
        if (s < A.S) {
            r0 = A.star_ptr[s];
            r1 = A.star_ptr[s + 1];
        }
        V h[kNAstro], l[kNAstro];
#pragma unroll
        for (int k = 0; k < kNAstro; k++)
            h[k] = l[k] = V(0);
#pragma unroll 2
        for (uint32_t r = r0 + slot; r < r1; r += RS) {
            const float *v = sv + tidx<kNAstro>(0, r);
            V yv[Cols<KP>::N];
            load_cols<KP>(Yp + (int64_t)kPanel * r, yv);
#pragma unroll
            for (int k = 0; k < kNAstro; k++) {
                V a;
                v_bcast(a, __ldcs(v + 32 * k));
                if constexpr (CL > 1)
                    df_acc_norm(h[k], l[k], v_mul(a, yv[0]));
                else
                    df_acc_v(h[k], l[k], v_mul(a, yv[0]));
            }
        }
        // over the RS rows in double-float; slot q writes sums q, q + RS, ...
        float rh[kNAstro][KP], rl[kNAstro][KP];
#pragma unroll
        for (int k = 0; k < kNAstro; k++)
#pragma unroll
            for (int c = 0; c < KP; c++) {
                const V hv[1] = {h[k]}, lv[1] = {l[k]};
                rh[k][c] = col_of<KP>(hv, c);
                rl[k][c] = col_of<KP>(lv, c);
#pragma unroll
                for (int off = CL; off < G; off <<= 1) {
                    const float oh = __shfl_xor_sync(0xffffffffu, rh[k][c], off);
                    const float ol = __shfl_xor_sync(0xffffffffu, rl[k][c], off);
                    df_add(rh[k][c], rl[k][c], oh, ol);
                }
            }
        if (s < A.S) {
#pragma unroll
            for (int k = 0; k < kNAstro; k++)
                if (k % RS == slot) {
                    double *t = T + pidx((int64_t)kNAstro * s + k, A.n, c0) + KP * cl;
#pragma unroll
                    for (int c = 0; c < KP; c++)
                        t[c] = df_to_d(rh[k][c], rl[k][c]);
                }
        }
    }
}

// attitude column colrow = a D + k of T, column c of the tile whose sums are S
template <int KT>
__device__ __forceinline__ double att_total(const SysView &A, const uint32_t *__restrict__ useg,
                                            const double *__restrict__ S, int64_t colrow, int c)
{
    const int64_t a = (colrow >= A.D) + (colrow >= 2 * A.D), k = colrow - a * A.D;
    double t = 0.0;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const int64_t o = k - j;
        if (o >= 0 && o < A.nseg) {
            const uint32_t u0 = __ldg(useg + o), u1 = __ldg(useg + o + 1);
#pragma unroll 4
            for (uint32_t u = u0; u < u1; u++)
                t += S[((int64_t)u * kNAtt + 4 * a + j) * KT + c];
        }
    }
    return t;
}

// attitude columns of T (products alone; the CG pass combines them itself)
template <int KT>
__global__ void k_b_att_combine(SysView A, Att32 U, const double *__restrict__ Sall,
                                double *__restrict__ T, int c_first)
{
    const int c0 = c_first + blockIdx.y * KT;
    const double *S = Sall + (int64_t)c0 * U.nunits * kNAtt;
    const int64_t total = 3 * A.D * KT;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % KT);
        const int64_t colrow = i / KT;  // a * D + k
        T[pidx(A.att0 + colrow, A.n, c0) + c] = att_total<KT>(A, U.useg, S, colrow, c);
    }
}

// ---------------------------------------------------------------------------
// aprod 2, instrumental nonzeros on KT columns: one warp per piece q of
// instrument f's entries (row irow[e], value ival[e]) in the
// instrument-sorted copy of the whole matrix; the warp that finishes an
// instrument's last piece (ticket) adds its np pieces in order into T
// ---------------------------------------------------------------------------
template <int KT>
__global__ void __launch_bounds__(kThreads)
k_b_instr(SysView A, const uint32_t *__restrict__ iseg, const uint32_t *__restrict__ irow,
          const float *__restrict__ ival, const float *__restrict__ Y, double *__restrict__ part_all,
          unsigned *__restrict__ ticket_all, double *__restrict__ T, int c_first, int np)
{
    typedef typename Cols<KT>::V V;
    constexpr int N = Cols<KT>::N;
    const int c0 = c_first + blockIdx.y * KT;
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const float *Yp = Y + pidx(0, A.m, c0);
    double *part = part_all + (int64_t)c0 * A.I * np;
    unsigned *ticket = ticket_all + (int64_t)c0 * A.I;
    for (uint32_t wi = (uint32_t)warp; wi < (uint32_t)A.I * np; wi += (uint32_t)nwarps) {
        // piece-major: at any time the warps take one quantile of every
        // instrument's rows, so their gathers stay within about 1/np of Y
        // (which need not fit in L2: 224 MB at 7.0e6 rows and 8 columns)
        const uint32_t q = wi / (uint32_t)A.I;
        const uint32_t f = wi - q * (uint32_t)A.I;
        const uint32_t s0 = iseg[f];
        const uint64_t len = iseg[f + 1] - s0;
        const uint32_t e0 = s0 + (uint32_t)(len * q / np);
        const uint32_t e1 = s0 + (uint32_t)(len * (q + 1) / np);
        V h[N], l[N];
#pragma unroll
        for (int c = 0; c < N; c++)
            h[c] = l[c] = V(0);
        uint32_t e = e0 + lane;
        // four entries per lane in flight (the gathers of Y depend on the row
        // indices); the sums take the entries in order
        for (; e + 96 < e1; e += 128) {
            uint32_t r4[4];
            float v4[4];
            V y4[4][N];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                r4[u] = __ldcs(irow + e + 32 * u);
                v4[u] = __ldcs(ival + e + 32 * u);
            }
#pragma unroll
            for (int u = 0; u < 4; u++)
                load_cols<KT>(Yp + (int64_t)kPanel * r4[u], y4[u]);
#pragma unroll
            for (int u = 0; u < 4; u++) {
                V a;
                v_bcast(a, v4[u]);
#pragma unroll
                for (int c = 0; c < N; c++)
                    df_acc_v(h[c], l[c], v_mul(a, y4[u][c]));
            }
        }
        for (; e < e1; e += 32) {
            V yv[N], a;
            load_cols<KT>(Yp + (int64_t)kPanel * __ldcs(irow + e), yv);
            v_bcast(a, __ldcs(ival + e));
#pragma unroll
            for (int c = 0; c < N; c++)
                df_acc_v(h[c], l[c], v_mul(a, yv[c]));
        }
        float rh[KT], rl[KT];
#pragma unroll
        for (int c = 0; c < KT; c++) {
            rh[c] = col_of<KT>(h, c);
            rl[c] = col_of<KT>(l, c);
        }
        // lane groups of 32 / KT lanes end with the total of one column
        df_reduce_scatter<KT, 32>(rh, rl, lane);
        constexpr int REST = 32 / KT;
        const int c = lane / REST;
        if ((lane % REST) == 0)
            part[((int64_t)f * np + q) * KT + c] = df_to_d(rh[0], rl[0]);
        __threadfence();
        __syncwarp();
        unsigned last = 0;
        if (lane == 0)
            last = atomicAdd(ticket + f, 1u) == (unsigned)np - 1;
        if (!__shfl_sync(0xffffffffu, last, 0))
            continue;
        __threadfence();
        // fixed order: lane (c, i) adds pieces i, i + REST, ..., then the lanes
        double t = 0.0;
        for (int k = lane % REST; k < np; k += REST)
            t += __ldcg(part + ((int64_t)f * np + k) * KT + c);
#pragma unroll
        for (int off = REST / 2; off > 0; off >>= 1)
            t += __shfl_xor_sync(0xffffffffu, t, off);
        if ((lane % REST) == 0)
            T[pidx(A.ins0 + f, A.n, c0) + c] = t;
        if (lane == 0)
            ticket[f] = 0u;
    }
}

// ---------------------------------------------------------------------------
// batched CG vector kernels: n x k panelled FP64 blocks, per-column scalars.
// Thread i takes entry (row i / KT, column i % KT) of its tile, so a warp
// reads consecutive doubles and a thread keeps one column (one thread per row
// and all its columns read 8-byte words 64 bytes apart and reduced 8 sums:
// 88 against 58 us at n = 562,001 and 8 columns).
// ---------------------------------------------------------------------------
// sum over the grid of one value per thread, by column (thread t holds column
// t % KT); true in the last block, whose threads 0 .. KT-1 hold the totals
template <int KT>
__device__ __forceinline__ bool grid_reduce_col(double &v, double *partial, unsigned *counter)
{
    constexpr int NW = kThreads / 32;
    __shared__ double sh[NW][KT];
    __shared__ bool am_last;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 16; off >= KT; off >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, off);
    if (lane < KT)
        sh[threadIdx.x >> 5][lane] = v;
    __syncthreads();
    if (threadIdx.x < KT) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < NW; w++)
            t += sh[w][threadIdx.x];
        partial[(int64_t)threadIdx.x * kMaxPartials + blockIdx.x] = t;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        am_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!am_last)
        return false;
    __threadfence();
    double t = 0.0;  // thread t: column t % KT, blocks t / KT, + kThreads / KT, ...
    for (unsigned b = threadIdx.x / KT; b < gridDim.x; b += kThreads / KT)
        t += __ldcg(partial + (int64_t)(threadIdx.x % KT) * kMaxPartials + b);
#pragma unroll
    for (int off = 16; off >= KT; off >>= 1)
        t += __shfl_xor_sync(0xffffffffu, t, off);
    if (lane < KT)
        sh[threadIdx.x >> 5][lane] = t;
    __syncthreads();
    if (threadIdx.x < KT) {
        v = 0.0;
#pragma unroll
        for (int w = 0; w < NW; w++)
            v += sh[w][threadIdx.x];
    }
    if (threadIdx.x == 0)
        *counter = 0u;
    return true;
}

// S = p o C, Dd = S, Z = 0, X32 = fl32(p o Dd), gamma_c = |S_c|^2
template <int KT>
__global__ void __launch_bounds__(kThreads)
k_b_init(const double *__restrict__ p, const double *__restrict__ C, double *__restrict__ Sv,
         double *__restrict__ Dd, double *__restrict__ Z, float *__restrict__ X32, int64_t n,
         int c_first, BatchState *bs, const BatchArgs *args, double *partial, unsigned *counter)
{
    const int c0 = c_first + blockIdx.y * KT;
    const int64_t base = pidx(0, n, c0);
    double acc = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n * KT;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = i / KT, e = base + j * kPanel + (i % KT);
        const double pj = p[j];
        const double sj = pj * C[e];
        Sv[e] = sj;
        Dd[e] = sj;
        Z[e] = 0.0;
        X32[e] = (float)(pj * sj);
        acc = fma(sj, sj, acc);
    }
    if (grid_reduce_col<KT>(acc, partial + (int64_t)c0 * kMaxPartials, counter + c0)) {
        if (c0 == 0 && threadIdx.x == 0) {
            bs->nonfinite = 0;
            bs->late = 0;
            bs->all_done = 0;
        }
        if (threadIdx.x < KT) {
            const int cc = c0 + threadIdx.x;
            bs->gamma[cc] = acc;
            bs->gamma0[cc] = acc;
            bs->beta[cc] = 0.0;
            bs->done[cc] = (acc > 0.0) ? 0 : 1;
            bs->it[cc] = 0;
        }
    }
}

// S_c -= alpha_c p o T_c, Z_c += alpha_c Dd_c, gamma'_c = |S_c|^2; the
// attitude columns of T come from the segment sums Sall
template <int KT>
__global__ void __launch_bounds__(kThreads)
k_b_vec1(SysView A, Att32 U, const double *__restrict__ p, const double *__restrict__ T,
         const double *__restrict__ Sall, double *__restrict__ Sv,
         const double *__restrict__ Dd, double *__restrict__ Z, int c_first, BatchState *bs,
         const BatchArgs *args, double *partial, unsigned *counter, const int *kerr)
{
    const int c0 = c_first + blockIdx.y * KT;
    const int c = threadIdx.x % KT;
    const int64_t base = pidx(0, A.n, c0);
    const double *S = Sall + (int64_t)c0 * U.nunits * kNAtt;
    const double al = bs->alpha[c0 + c];
    const bool late = threadIdx.x < KT && wait_expired(kerr);
    double acc = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < A.n * KT;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = i / KT, e = base + j * kPanel + c;
        const double tj = (j < A.att0 || j >= A.ins0) ? T[e] : att_total<KT>(A, U.useg, S, j - A.att0, c);
        const double sj = fma(-al, p[j] * tj, Sv[e]);
        Sv[e] = sj;
        Z[e] = fma(al, Dd[e], Z[e]);
        acc = fma(sj, sj, acc);
    }
    if (grid_reduce_col<KT>(acc, partial + (int64_t)c0 * kMaxPartials, counter + c0) &&
        threadIdx.x < KT) {
        const int cc = c0 + threadIdx.x;
        if (bs->done[cc]) {
            bs->beta[cc] = 0.0;
        } else {
            const double gnew = acc;
            bs->beta[cc] = gnew / bs->gamma[cc];
            bs->gamma[cc] = gnew;
            bs->it[cc] += 1;
            if (!isfinite(gnew))
                bs->nonfinite = 1;
            if (late)
                bs->late = 1;
            if (!isfinite(gnew) || late || gnew <= args->tol * args->tol * bs->gamma0[cc] ||
                bs->it[cc] >= args->max_inner)
                bs->done[cc] = 1;
        }
    }
}

// Dd = S + beta_c Dd, X32 = fl32(p o Dd); with last set (every tile's vec1 of
// the iteration has run) one thread clears the loop flag when every one of
// the k columns is done
template <int KT>
__global__ void k_b_vec2(const double *__restrict__ p, const double *__restrict__ Sv,
                         double *__restrict__ Dd, float *__restrict__ X32, int64_t n, int c_first,
                         BatchState *bs, int k, cudaGraphConditionalHandle loop, int in_graph,
                         int last)
{
    const int c0 = c_first + blockIdx.y * KT;
    const int c = threadIdx.x % KT;
    const int64_t base = pidx(0, n, c0);
    const double be = bs->beta[c0 + c];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n * KT;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = i / KT, e = base + j * kPanel + c;
        const double dj = fma(be, Dd[e], Sv[e]);
        Dd[e] = dj;
        X32[e] = (float)(p[j] * dj);
    }
    if (last && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        int all = 1;
        for (int q = 0; q < k; q++)
            all &= bs->done[q];
        bs->all_done = all;
        if (all && in_graph)
            cudaGraphSetConditional(loop, 0u);
    }
}

// loop flag before the first iteration: clear when every column is done
__global__ void k_b_flag(BatchState *bs, int k, cudaGraphConditionalHandle loop, int in_graph)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        int all = 1;
        for (int c = 0; c < k; c++)
            all &= bs->done[c];
        bs->all_done = all;
        if (all && in_graph)
            cudaGraphSetConditional(loop, 0u);
    }
}

// generic layout change with optional binary32 output: to_rm = 1 maps a
// column-major (rows x k) block to the panelled layout, 0 the reverse
__global__ void k_b_layout(int to_rm, const double *__restrict__ src, double *__restrict__ dst64,
                           float *__restrict__ dst32, int64_t rows, int k)
{
    const int64_t total = rows * k;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t c = i / rows;
        const int64_t r = i - c * rows;
        const int64_t rm = pidx(r, rows, (int)c), cm = i;
        const double v = to_rm ? src[cm] : src[rm];
        const int64_t to = to_rm ? rm : cm;
        if (dst32)
            dst32[to] = (float)v;
        else
            dst64[to] = v;
    }
}

// panelled binary32 (rows x k) -> column-major FP64 (rows x k)
__global__ void k_b_rm32_to_cm(const float *__restrict__ src, double *__restrict__ dst, int64_t rows,
                               int k)
{
    const int64_t total = rows * k;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t c = i / rows;
        const int64_t r = i - c * rows;
        dst[i] = (double)src[pidx(r, rows, (int)c)];
    }
}

// dst_f32: 0 FP64 out, 1 binary32 out, 2 binary32 panelled source -> FP64
// column-major out (to_rm = 1: column-major in, panelled out).
cudaError_t launch_b_layout(const gsr_handle_t *h, int to_rm, const double *src, void *dst,
                            int dst_f32, int64_t rows, int k, cudaStream_t st)
{
    if (dst_f32 == 2)
        k_b_rm32_to_cm<<<h->nsm * 8, kThreads, 0, st>>>((const float *)src, (double *)dst, rows, k);
    else
        k_b_layout<<<h->nsm * 8, kThreads, 0, st>>>(to_rm, src, dst_f32 ? nullptr : (double *)dst,
                                                     dst_f32 ? (float *)dst : nullptr, rows, k);
    return cudaGetLastError();
}

// X[:, c] += p o Z[:, c] (X column-major n x k, Z panelled)
__global__ void k_b_update_x(const double *__restrict__ p, const double *__restrict__ Z,
                             double *__restrict__ X, int64_t n, int k)
{
    const int64_t total = n * k;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i / n);
        const int64_t j = i - c * n;
        X[i] = fma(p[j], Z[pidx(j, n, c)], X[i]);
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// blocks for `warps` warps of work, at most the resident ones
static int b_blocks(const gsr_handle_t *h, int occ, int64_t warps)
{
    const int64_t need = (warps + kThreads / 32 - 1) / (kThreads / 32);
    int64_t g = (int64_t)h->nsm * (occ < 1 ? 1 : occ);
    if (g > need)
        g = need;
    if (g > kMaxPartials)
        g = kMaxPartials;
    return (int)(g < 1 ? 1 : g);
}

template <typename F>
static int b_occ(F f)
{
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, f, kThreads, 0) != cudaSuccess)
        occ = 1;
    return occ;
}

// pieces per instrument: about 2048 entries each, four at least (an instrument
// that many rows use gives four warps work, and the chains of sums stay short)
int batched_instr_pieces(const gsr_handle_t *h)
{
    const int64_t mean = kNInstr * h->sys.m / h->sys.I;
    const int64_t np = (mean + 2047) / 2048;
    return (int)(np < 4 ? 4 : (np > 256 ? 256 : np));
}

template <int KT, int MODE>
static cudaError_t b_main(const gsr_handle_t *h, const float *X, float *Q, double *T, int c0, int ny,
                          cudaStream_t st)
{
    constexpr size_t smem = kBWarps * sizeof(BWarp<KT>);
    const cudaError_t e = cudaFuncSetAttribute(
        k_b_main<KT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    const int gx = (int)(h->att32.nunits < h->nsm ? h->att32.nunits : h->nsm);
    k_b_main<KT, MODE><<<dim3(gx, ny), kBThreads, smem, st>>>(h->sys, h->att32, X, Q, h->d_bS, T, c0,
                                                              h->d_bs, h->d_bpartial,
                                                              h->d_bcounter, h->d_kerr);
    return cudaGetLastError();
}

template <int KT, int G>
static void b_stars(const gsr_handle_t *h, const float *Y, double *T, int c0, int ny,
                    cudaStream_t st)
{
    const int occ = b_occ(k_b_stars<KT, G>);
    const int gx = b_blocks(h, occ, (h->sys.S + 32 / G - 1) / (32 / G));
    k_b_stars<KT, G><<<dim3(gx, ny), kThreads, 0, st>>>(h->sys, h->att32.sv, Y, T, c0);
}

// The star and instrument passes write different sums and run side by side
// when a branch is given (graph capture): one bound by its gathers shares the
// SMs with one bound by the FP32 pipe.
template <int KT>
static cudaError_t b_rest(const gsr_handle_t *h, const float *Y, double *T, int c0, int ny,
                          cudaStream_t st, Branch *br)
{
    cudaError_t e = br ? br->fork(st) : cudaSuccess;
    if (e != cudaSuccess)
        return e;
    const cudaStream_t si = br ? br->s : st;
    const int occ_i = b_occ(k_b_instr<KT>);
    const int npi = batched_instr_pieces(h);
    k_b_instr<KT><<<dim3(b_blocks(h, 2 * occ_i, h->sys.I * npi), ny), kThreads, 0, si>>>(
        h->sys, h->d_iseg, h->d_irow, h->d_ival32, Y, h->d_bipart, h->d_bticket, T, c0, npi);
    switch (h->b_lanes) {
    case 8: b_stars<KT, 8>(h, Y, T, c0, ny, st); break;
    case 32: b_stars<KT, 32>(h, Y, T, c0, ny, st); break;
    default: b_stars<KT, 16>(h, Y, T, c0, ny, st); break;
    }
    e = cudaGetLastError();
    return br && e == cudaSuccess ? br->join(st) : e;
}

template <int KT>
static int vec_blocks(const gsr_handle_t *h)
{
    const int64_t need = (h->sys.n * KT + kThreads - 1) / kThreads;
    const int64_t g = (int64_t)h->nsm * 4;
    return (int)(g < need ? g : need);
}

template <int KT>
static cudaError_t b_prologue_tiles(const gsr_handle_t *h, int c0, int ny, cudaStream_t s)
{
    k_b_init<KT><<<dim3(vec_blocks<KT>(h), ny), kThreads, 0, s>>>(
        h->d_p, h->d_bC, h->d_bS_, h->d_bD, h->d_bZ, h->d_bX32, h->sys.n, c0, h->d_bs, h->d_bargs,
        h->d_bpartial, h->d_bcounter);
    return cudaGetLastError();
}

template <int KT>
static cudaError_t b_products_tiles(const gsr_handle_t *h, const float *X, float *Q, float *Y,
                                    double *T, int c0, int ny, cudaStream_t s)
{
    cudaError_t e = b_main<KT, kBA1>(h, X, Q, T, c0, ny, s);
    if (e == cudaSuccess)
        e = b_main<KT, kBA2>(h, nullptr, Y, T, c0, ny, s);
    if (e == cudaSuccess)
        e = b_rest<KT>(h, Y, T, c0, ny, s, nullptr);
    if (e == cudaSuccess) {
        k_b_att_combine<KT><<<dim3(h->nsm, ny), kThreads, 0, s>>>(h->sys, h->att32, h->d_bS, T, c0);
        e = cudaGetLastError();
    }
    return e;
}

template <int KT>
static cudaError_t b_iteration_tiles(const gsr_handle_t *h, int c0, int ny, cudaStream_t s, int k,
                                     cudaGraphConditionalHandle loop, int in_graph, int last,
                                     Branch *br)
{
    cudaError_t e = b_main<KT, kBA1 | kBA2>(h, h->d_bX32, h->d_bQ32, h->d_bT, c0, ny, s);
    if (e == cudaSuccess)
        e = b_rest<KT>(h, h->d_bQ32, h->d_bT, c0, ny, s, br);
    if (e != cudaSuccess)
        return e;
    const dim3 g(vec_blocks<KT>(h), ny);
    k_b_vec1<KT><<<g, kThreads, 0, s>>>(h->sys, h->att32, h->d_p, h->d_bT, h->d_bS, h->d_bS_,
                                        h->d_bD, h->d_bZ, c0, h->d_bs, h->d_bargs, h->d_bpartial,
                                        h->d_bcounter, h->d_kerr);
    k_b_vec2<KT><<<g, kThreads, 0, s>>>(h->d_p, h->d_bS_, h->d_bD, h->d_bX32, h->sys.n, c0, h->d_bs,
                                        k, loop, in_graph, last);
    return cudaGetLastError();
}

// The k columns as runs of equal tiles: whole tiles of the chosen width, then
// the rest in one tile of the least width that holds it (its further columns
// are zero: 19 columns at width 8 are two tiles of 8 and one of 4).
// f(kt, c0, ny) per run; the last run is told.
template <typename F>
static cudaError_t for_runs(const gsr_handle_t *h, int k, F f)
{
    const int whole = k / h->b_kt;
    if (whole > 0) {
        const cudaError_t e = f(h->b_kt, 0, whole, whole * h->b_kt == k);
        if (e != cudaSuccess)
            return e;
    }
    const int rest = k - whole * h->b_kt;
    if (rest == 0)
        return cudaSuccess;
    int kt = 1;
    while (kt < rest)
        kt *= 2;
    return f(kt, whole * h->b_kt, 1, true);
}

// the inner solve of the k columns: prologue, then iterations until every
// column is done (graph with a conditional loop, or host-driven in eager mode)
static cudaError_t b_prologue(const gsr_handle_t *h, int k, cudaStream_t s,
                              cudaGraphConditionalHandle loop, int in_graph)
{
    cudaError_t e = for_runs(h, k, [&](int kt, int c0, int ny, bool) {
        switch (kt) {
        case 1: return b_prologue_tiles<1>(h, c0, ny, s);
        case 2: return b_prologue_tiles<2>(h, c0, ny, s);
        case 4: return b_prologue_tiles<4>(h, c0, ny, s);
        default: return b_prologue_tiles<8>(h, c0, ny, s);
        }
    });
    if (e != cudaSuccess)
        return e;
    k_b_flag<<<1, 32, 0, s>>>(h->d_bs, k, loop, in_graph);
    return cudaGetLastError();
}

// With branches the runs are independent chains and the loop flag follows
// their join; otherwise the last run's vector pass sets it.
static cudaError_t b_iteration(const gsr_handle_t *h, int k, cudaStream_t s,
                               cudaGraphConditionalHandle loop, int in_graph, BatchSide *side)
{
    const bool two = side && k > h->b_kt && k % h->b_kt != 0;
    cudaError_t e = two ? side->run.fork(s) : cudaSuccess;
    if (e != cudaSuccess)
        return e;
    e = for_runs(h, k, [&](int kt, int c0, int ny, bool last) {
        const int i = c0 > 0;
        const cudaStream_t st = two && i ? side->run.s : s;
        Branch *br = side ? &side->instr[i] : nullptr;
        const int flag = last && !two;
        switch (kt) {
        case 1: return b_iteration_tiles<1>(h, c0, ny, st, k, loop, in_graph, flag, br);
        case 2: return b_iteration_tiles<2>(h, c0, ny, st, k, loop, in_graph, flag, br);
        case 4: return b_iteration_tiles<4>(h, c0, ny, st, k, loop, in_graph, flag, br);
        default: return b_iteration_tiles<8>(h, c0, ny, st, k, loop, in_graph, flag, br);
        }
    });
    if (e != cudaSuccess || !two)
        return e;
    e = side->run.join(s);
    if (e != cudaSuccess)
        return e;
    k_b_flag<<<1, 32, 0, s>>>(h->d_bs, k, loop, in_graph);
    return cudaGetLastError();
}

#define B_TRY(x)                        \
    do {                                \
        cudaError_t e_ = (x);           \
        if (e_ != cudaSuccess) {        \
            err = e_;                   \
            goto fail;                  \
        }                               \
    } while (0)

cudaError_t find_graph_leaf(cudaGraph_t g, cudaGraphNode_t *leaf);

cudaError_t build_batched_graph(gsr_handle_t *h, int k)
{
    cudaError_t err = cudaSuccess;
    cudaGraph_t g = nullptr;
    cudaGraphConditionalHandle loop;
    cudaGraphNode_t pre_leaf, wnode;
    cudaGraphNodeParams cp = {};
    cudaGraph_t body;
    cudaStream_t s = h->cap_stream;
    BatchSide side;
    B_TRY(side.make());
    B_TRY(cudaGraphCreate(&g, 0));
    B_TRY(cudaGraphConditionalHandleCreate(&loop, g, 1u, cudaGraphCondAssignDefault));
    B_TRY(cudaStreamBeginCaptureToGraph(s, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    B_TRY(b_prologue(h, k, s, loop, 1));
    B_TRY(cudaStreamEndCapture(s, &g));
    B_TRY(find_graph_leaf(g, &pre_leaf));
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = loop;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    B_TRY(cudaGraphAddNode(&wnode, g, &pre_leaf, nullptr, 1, &cp));
    body = cp.conditional.phGraph_out[0];
    B_TRY(cudaStreamBeginCaptureToGraph(s, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    B_TRY(b_iteration(h, k, s, loop, 1, &side));
    B_TRY(cudaStreamEndCapture(s, &body));
    B_TRY(cudaGraphInstantiate(&h->b_exec[k], g, 0));
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

cudaError_t run_batched_inner(gsr_handle_t *h, int k, int max_inner, cudaStream_t st)
{
    if (!h->cfg.eager)
        return cudaGraphLaunch(h->b_exec[k], st);
    cudaError_t e = b_prologue(h, k, st, 0, 0);
    for (int it = 0; e == cudaSuccess && it < max_inner + 1; it++) {
        e = cudaMemcpyAsync(h->h_bs, h->d_bs, sizeof(BatchState), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(st);
        if (e != cudaSuccess || h->h_bs->all_done)
            break;
        e = b_iteration(h, k, st, 0, 0, nullptr);
    }
    return e;
}

cudaError_t launch_b_update_x(const gsr_handle_t *h, double *X, int k, cudaStream_t st)
{
    k_b_update_x<<<h->nsm * 8, kThreads, 0, st>>>(h->d_p, h->d_bZ, X, h->sys.n, k);
    return cudaGetLastError();
}

// single products on the binary32 copy for k columns (panelled blocks),
// for the parity tests and the tuner: Q = A32 X and T = A32^T Y
cudaError_t launch_b_products(const gsr_handle_t *h, int k, const float *X, float *Q, float *Y,
                              double *T, cudaStream_t st)
{
    return for_runs(h, k, [&](int kt, int c0, int ny, bool) {
        switch (kt) {
        case 1: return b_products_tiles<1>(h, X, Q, Y, T, c0, ny, st);
        case 2: return b_products_tiles<2>(h, X, Q, Y, T, c0, ny, st);
        case 4: return b_products_tiles<4>(h, X, Q, Y, T, c0, ny, st);
        default: return b_products_tiles<8>(h, X, Q, Y, T, c0, ny, st);
        }
    });
}

}  // namespace gsr
