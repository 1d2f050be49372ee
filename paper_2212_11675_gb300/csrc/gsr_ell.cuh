// Instrumental part of the binary32 aprod 2 (Alg. 2: column f receives sum
// value * y_row over the nonzeros of instrument f) over row windows held in
// shared memory.
//
// The rows are cut into windows of W <= 8160 rows.  Inside a window the
// nonzeros of one instrument, in row order, form one or more columns of at
// most kEllLen entries, one lane each; 32 columns of like length are one slice
// (sliced ELL: entries 2 i and 2 i + 1 of the 32 lanes are contiguous), so a warp reads values
// and row numbers in whole segments and needs no reduction across lanes.  A
// block stages the window of y in shared memory and gathers it from there; the
// columns' sums of all its windows are added in shared memory too (added in
// global memory they cost 50 of 128 us) and leave it as one partial per
// instrument and block.  Every sum has a fixed order.
//
// Why: gathered from L2 (one instrument's rows spread over all of y) the 6 m
// gathers alone take 0.145 ms at m = 7.0e6 (random 32-byte sectors arrive at
// 0.93 per clock and SM), next to 48 B a row of values and row numbers; here
// they are shared-memory reads next to 36 B a row (6 B an entry).  With I
// instruments a column holds about 6 W / I entries, which bounds the form to
// I <= 6144 (kEllInstrMax: eight entries at least).  Beyond that the
// instrument-sorted copy with its gathers stays; so it does for FP64, where
// the FP64 pipe is the limit and the windows gained nothing (356 against
// 340 us for the whole aprod 2 at m = 7.0e6).
//
// kEllWarps warps of a block run the pass (the others, and these once they
// have finished, take the star units).  The next window of y is copied by the
// bulk-copy engine while the current one is summed, and every warp has its next
// sixteen entries (of this slice or the next) on their way while it sums
// eight: with eight on their way the pass took 128 us of HBM latency for its
// 300 MB.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gsr_df.cuh"
#include "gsr_internal.cuh"
#include "gsr_reduce.cuh"
#include "gsr_tma.cuh"

namespace gsr {

constexpr int kEllWarps = 16;
constexpr int kEllThreads = 32 * kEllWarps;
constexpr int kEllRows = 8192;  // shared rows: W <= 8160, the last one is the padding's zero
constexpr size_t kEllSmem32 = 2 * kEllRows * sizeof(float);

// barrier of the kEllThreads threads of the pass
__device__ __forceinline__ void ell_sync()
{
    asm volatile("bar.sync 1, %0;" ::"n"(kEllThreads) : "memory");
}

// kEllStep entries of each lane's column, and with the last ones of a slice
// where their sum goes (pos; kEllMore: the column goes on)
struct EllRun {
    float2 v[kEllStep / 2];
    uint32_t r[kEllStep / 2];  // two window rows
    uint32_t pos;
};
constexpr uint32_t kEllMore = 0xfffffffeu;

// The slices sl, sl + kEllWarps, ... of one window as a sequence of runs, their
// descriptions one slice ahead
struct EllCursor {
    const Ell &E;
    uint32_t sl, sl1, i = 0;
    uint2 s, sn;
    uint32_t pos, pn;
    int lane;

    __device__ __forceinline__ EllCursor(const Ell &E_, uint32_t sl_, uint32_t sl1_)
        : E(E_), sl(sl_), sl1(sl1_), lane(threadIdx.x & 31)
    {
        if (sl < sl1) {
            s = __ldg(E.slice + sl);
            pos = __ldcs(E.pos + (int64_t)sl * 32 + lane);
            describe();
        }
    }
    __device__ __forceinline__ void describe()
    {
        sn = s;
        pn = pos;
        if (sl + kEllWarps < sl1) {
            sn = __ldg(E.slice + sl + kEllWarps);
            pn = __ldcs(E.pos + (int64_t)(sl + kEllWarps) * 32 + lane);
        }
    }
    __device__ __forceinline__ bool fetch(EllRun &a)
    {
        if (sl >= sl1)
            return false;
        // the lane's first pair; its pairs are 32 pairs apart
        const int64_t p = ((int64_t)s.x + i) * 32 + 2 * lane;
#pragma unroll
        for (int k = 0; k < kEllStep / 2; k++) {
            a.v[k] = __ldcs(reinterpret_cast<const float2 *>(E.val32 + p + 64 * k));
            a.r[k] = __ldcs(reinterpret_cast<const uint32_t *>(E.idx + p + 64 * k));
        }
        i += kEllStep;
        a.pos = kEllMore;
        if (i >= s.y) {
            a.pos = pos;
            sl += kEllWarps;
            s = sn;
            pos = pn;
            i = 0;
            describe();
        }
        return true;
    }
};

struct EllShared {
    uint64_t bar[2];
    volatile int fail;
};

// Two shared-memory buffers of a window of y (16-byte aligned, W a multiple of
// 32): the next window is copied while the current one is used.
struct EllWindows {
    float *buf;  // 2 kEllRows
    EllShared *sh;
    uint32_t bar;
    const float *y;
    int64_t m, W;
    uint32_t phase = 0;

    __device__ __forceinline__ int rows(int64_t w) const
    {
        return (int)(m - w * W < W ? m - w * W : W);
    }
    __device__ __forceinline__ void init(float *b, EllShared *sh_, const float *y_, int64_t m_,
                                         int64_t W_, bool late)
    {
        buf = b;
        sh = sh_;
        bar = smem_addr(sh->bar);
        y = y_;
        m = m_;
        W = W_;
        if (threadIdx.x == 0) {
            buf[kEllPad] = buf[kEllRows + kEllPad] = 0.f;
            sh->fail = 0;
            mbar_init(bar, late);
            mbar_init(bar + 8, late);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        ell_sync();
    }
    // start the copy of window w into buffer b (the tail of a ragged window
    // that no 16 bytes cover is stored by the threads)
    __device__ __forceinline__ void fetch(int64_t w, int b)
    {
        const int nr = rows(w), whole = nr / 4 * 4;
        float *d = buf + b * kEllRows;
        const float *src = y + w * W;
        if (threadIdx.x == 0 && whole) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect(bar + 8 * b, whole * sizeof(float));
            bulk_copy(smem_addr(d), src, whole * sizeof(float), bar + 8 * b);
        }
        for (int i = whole + threadIdx.x; i < nr; i += kEllThreads)
            d[i] = __ldg(src + i);
    }
    // window w in buffer b is complete, for every thread; false on a timeout
    __device__ __forceinline__ bool wait(int64_t w, int b, int *kerr)
    {
        if (rows(w) >= 4) {
            if (!mbar_wait(bar + 8 * b, (phase >> b) & 1u))
                sh->fail = 1;
            phase ^= 1u << b;
        }
        ell_sync();
        if (sh->fail == 0)
            return true;
        if (threadIdx.x == 0)
            atomicExch(kerr, 1);
        return false;
    }
};

// the windows of this block (w = blockIdx.x, + E.nblk, ...): use(w, window of
// y) for each; called by the first kEllThreads threads
template <typename Use>
__device__ __forceinline__ void ell_windows(const Ell &E, const float *y, int64_t m, float *buf,
                                            EllShared *sh, int *kerr, Use use)
{
    EllWindows win;
    int64_t w = blockIdx.x;
    win.init(buf, sh, y, m, E.W, w == E.late);
    int b = 0;
    win.fetch(w, 0);
    for (; w < E.nwin; w += E.nblk, b ^= 1) {
        // the other buffer was last read before the barrier that ended the
        // previous window's use
        const int64_t wn = w + E.nblk;
        if (wn < E.nwin)
            win.fetch(wn, b ^ 1);
        if (!win.wait(w, b, kerr)) {
            if (wn < E.nwin)
                win.wait(wn, b ^ 1, kerr);  // let the copy in flight land
            return;
        }
        use(w, buf + b * kEllRows);
        ell_sync();
    }
}

// binary32 values and y: binary32 products, double-float sums (two entries per
// packed operation), FP64 partials
__device__ __forceinline__ void ell32_part(const Ell &E, const float *y, int64_t m,
                                           unsigned char *smem, EllShared *sh, int *kerr, int64_t I)
{
    double *acc = reinterpret_cast<double *>(smem + kEllSmem32);  // [nacc]
    if (blockIdx.x >= E.nblk)
        return;
    for (int i = threadIdx.x; i < E.nacc; i += kEllThreads)
        acc[i] = 0.0;
    ell_windows(E, y, m, reinterpret_cast<float *>(smem), sh, kerr, [&](int64_t w, const float *yw) {
        EllCursor cur(E, __ldg(E.win + w) + (threadIdx.x >> 5), __ldg(E.win + w + 1));
        f32x2 h[2] = {0ull, 0ull}, l[2] = {0ull, 0ull};
        EllRun a, b, c;
        bool ok = cur.fetch(a), okb = cur.fetch(b);
        while (ok) {
            const bool okc = cur.fetch(c);
#pragma unroll
            for (int k = 0; k < kEllStep / 2; k++)
                df_acc_v(h[k & 1], l[k & 1],
                         v_mul(pack2(a.v[k].x, a.v[k].y),
                               pack2(yw[a.r[k] & kEllRowMask], yw[(a.r[k] >> 16) & kEllRowMask])));
            if (a.pos != kEllMore) {
                float th[4], tl[4];
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    unpack2(h[k], th[2 * k], th[2 * k + 1]);
                    unpack2(l[k], tl[2 * k], tl[2 * k + 1]);
                    h[k] = l[k] = 0ull;
                }
                df_add(th[0], tl[0], th[1], tl[1]);
                df_add(th[2], tl[2], th[3], tl[3]);
                df_add(th[0], tl[0], th[2], tl[2]);
                const double t = df_to_d(th[0], tl[0]);
                if (a.pos != kEllNone)  // one column of the window has this sum
                    acc[a.pos] += t;
            }
            a = b;
            b = c;
            ok = okb;
            okb = okc;
        }
    });
    // the pieces of an instrument in order
    const uint32_t *start = E.start + (int64_t)blockIdx.x * (I + 1);
    for (int64_t f = threadIdx.x; f < I; f += kEllThreads) {
        double t = 0.0;
        for (uint32_t i = __ldg(start + f); i < __ldg(start + f + 1); i++)
            t += acc[i];
        E.part[(int64_t)blockIdx.x * I + f] = t;
    }
}

// total of instrument f, by one warp (every lane has it), in a fixed order
__device__ __forceinline__ double ell_total(const Ell &E, int64_t f, int64_t I)
{
    double t = 0.0;
#pragma unroll 5
    for (int64_t b = threadIdx.x & 31; b < E.nblk; b += 32)
        t += __ldcg(E.part + b * I + f);
    __syncwarp();
    return warp_sum(t);
}

}  // namespace gsr
