// Instrumental part of the binary32 aprod 2 (Alg. 2: column f receives sum
// value * y_row over the nonzeros of instrument f) over row windows held in
// shared memory.
//
// The rows are cut into windows of W <= 8160 rows.  Inside a window the
// nonzeros of one instrument, in row order, form one or more columns of at
// most kEllLen entries, one lane each; 32 columns of like length are one slice
// (sliced ELL: entry i of the 32 lanes is contiguous), so a warp reads values
// and row numbers in whole segments and needs no reduction across lanes.  A
// block stages the window of y in shared memory and gathers it from there;
// every column keeps one partial sum per block, so an instrument has about as
// many partials as there are SMs.  Every sum has a fixed order.
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
// bulk-copy engine while the current one is summed, and every warp loads its
// next eight entries (of this slice or the next) before it sums the current
// eight.
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

// kEllStep entries of a column: values, window rows
template <typename T>
struct EllRun {
    T v[kEllStep];
    uint32_t r[kEllStep];
};

template <typename T>
__device__ __forceinline__ void ell_load(EllRun<T> &a, const T *__restrict__ val,
                                         const uint16_t *__restrict__ idx, int64_t p)
{
#pragma unroll
    for (int k = 0; k < kEllStep; k++) {
        a.v[k] = __ldcs(val + p + 32 * k);
        a.r[k] = (uint32_t)__ldcs(idx + p + 32 * k) & kEllRowMask;
    }
}

// The slices of one window, dealt to the kEllWarps warps; body(a) sums
// kEllStep entries, done() ends a column and returns its sum, which is added to
// the column's partial (stored where the block has not written it yet).  A
// slice's description and partials are loaded a slice ahead.
template <typename T, typename Body, typename Done>
__device__ __forceinline__ void ell_slices(const Ell &E, const T *__restrict__ val, uint32_t sl,
                                           uint32_t sl1, Body body, Done done)
{
    const int lane = threadIdx.x & 31;
    sl += threadIdx.x >> 5;
    if (sl >= sl1)
        return;
    uint2 s = __ldg(E.slice + sl);
    uint32_t pos = __ldcs(E.pos + (int64_t)sl * 32 + lane);
    EllRun<T> a;
    ell_load(a, val, E.idx, (int64_t)s.x * 32 + lane);
    for (;;) {
        const bool more = sl + kEllWarps < sl1;
        uint2 sn = s;
        uint32_t pn = kEllNone;
        if (more) {
            sn = __ldg(E.slice + sl + kEllWarps);
            pn = __ldcs(E.pos + (int64_t)(sl + kEllWarps) * 32 + lane);
        }
        double *part = E.part + (pos & ~kEllFirst);
        const double old = (pos & kEllFirst) ? 0.0 : *part;  // none: flagged too
        const int64_t p0 = (int64_t)s.x * 32 + lane;
        for (uint32_t i = kEllStep; i < s.y; i += kEllStep) {
            EllRun<T> b;
            ell_load(b, val, E.idx, p0 + 32 * (int64_t)i);
            body(a);
            a = b;
        }
        EllRun<T> b;
        ell_load(b, val, E.idx, (int64_t)sn.x * 32 + lane);
        body(a);
        const double t = done();
        if (pos != kEllNone)
            *part = (pos & kEllFirst) ? t : old + t;
        if (!more)
            return;
        a = b;
        s = sn;
        pos = pn;
        sl += kEllWarps;
    }
}

struct EllShared {
    uint64_t bar[2];
    volatile int fail;
};

// Two shared-memory buffers of a window of y: the window after next is copied
// while the next is used.  One bulk copy per window where y is 16-byte
// aligned, plain loads otherwise.
template <typename T>
struct EllWindows {
    T *buf;  // 2 kEllRows
    EllShared *sh;
    uint32_t bar;
    const T *y;
    int64_t m, W;
    bool bulk;
    uint32_t phase = 0;

    __device__ __forceinline__ int rows(int64_t w) const
    {
        return (int)(m - w * W < W ? m - w * W : W);
    }
    __device__ __forceinline__ void init(T *b, EllShared *sh_, const T *y_, int64_t m_, int64_t W_)
    {
        buf = b;
        sh = sh_;
        bar = smem_addr(sh->bar);
        y = y_;
        m = m_;
        W = W_;
        bulk = ((uintptr_t)y & 15u) == 0;
        if (threadIdx.x == 0) {
            buf[kEllPad] = buf[kEllRows + kEllPad] = T(0);
            sh->fail = 0;
            mbar_init(bar);
            mbar_init(bar + 8);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        ell_sync();
    }
    // start the copy of window w into buffer b (the tail of a ragged window
    // that no 16 bytes cover is stored by the thread itself)
    __device__ __forceinline__ void fetch(int64_t w, int b)
    {
        const int nr = rows(w);
        T *d = buf + b * kEllRows;
        const T *src = y + w * W;
        constexpr int Q = 16 / sizeof(T);
        const int whole = bulk ? nr / Q * Q : 0;
        if (threadIdx.x == 0 && whole) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect(bar + 8 * b, whole * sizeof(T));
            bulk_copy(smem_addr(d), src, whole * sizeof(T), bar + 8 * b);
        }
        for (int i = whole + threadIdx.x; i < nr; i += kEllThreads)
            d[i] = __ldg(src + i);
    }
    // window w in buffer b is complete, for every thread; false on a timeout
    __device__ __forceinline__ bool wait(int64_t w, int b, int *kerr)
    {
        if (bulk && rows(w) * sizeof(T) >= 16) {
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
template <typename T, typename Use>
__device__ __forceinline__ void ell_windows(const Ell &E, const T *y, int64_t m, T *buf,
                                            EllShared *sh, int *kerr, Use use)
{
    EllWindows<T> win;
    int64_t w = blockIdx.x;
    if (w >= E.nblk)
        return;
    win.init(buf, sh, y, m, E.W);
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
                                           unsigned char *smem, EllShared *sh, int *kerr)
{
    ell_windows<float>(E, y, m, reinterpret_cast<float *>(smem), sh, kerr,
                       [&](int64_t w, const float *yw) {
        f32x2 h[2] = {0ull, 0ull}, l[2] = {0ull, 0ull};
        ell_slices<float>(E, E.val32, __ldg(E.win + w), __ldg(E.win + w + 1),
                          [&](const EllRun<float> &a) {
#pragma unroll
            for (int k = 0; k < kEllStep; k += 2)
                df_acc_v(h[(k / 2) & 1], l[(k / 2) & 1],
                         v_mul(pack2(a.v[k], a.v[k + 1]), pack2(yw[a.r[k]], yw[a.r[k + 1]])));
        }, [&] {
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
            return df_to_d(th[0], tl[0]);
        });
    });
}

// total of instrument f, by one warp (every lane has it), in a fixed order
__device__ __forceinline__ double ell_total(const Ell &E, int64_t f)
{
    const uint32_t a = __ldg(E.ptr + f), b = __ldg(E.ptr + f + 1);
    double t = 0.0;
#pragma unroll 4
    for (uint32_t p = a + (threadIdx.x & 31); p < b; p += 32)
        t += __ldcg(E.part + p);
    __syncwarp();
    return warp_sum(t);
}

}  // namespace gsr
