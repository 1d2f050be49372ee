// Construction of the row windows of the binary32 instrument pass
// (gsr_ell.cuh) and of the instrument-sorted copy from them.
#include "gsr_ell.cuh"

namespace gsr {

// values and window rows from the entry codes (6 row + slot; kEllNone pads)
__global__ void k_ell_fill(SysView A, int64_t W, const uint32_t *__restrict__ code, int64_t total,
                           uint16_t *__restrict__ idx, float *__restrict__ val32)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < total;
         p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t c = code[p];
        float v = 1.f;  // the padding: 1 times the zero row
        uint32_t i = kEllPad;
        if (c != kEllNone) {
            const uint32_t row = c / kNInstr, slot = c - row * kNInstr;
            v = (float)A.val[tidx<kNPar>(kNAstro + kNAtt + slot, row)];
            i = (row % (uint32_t)W) | (slot << kEllRowBits);
        }
        idx[p] = (uint16_t)i;
        val32[p] = v;
    }
}

// the values of instrument slot `slot` again, after its plane changed
__global__ void k_ell_plane(SysView A, Ell E, int slot, float *__restrict__ val32)
{
    for (int64_t w = blockIdx.x; w < E.nwin; w += gridDim.x) {
        const uint32_t a = E.win[w], b = E.win[w + 1];
        if (a == b)
            continue;
        const uint2 e = E.slice[b - 1];
        const int64_t p1 = ((int64_t)e.x + e.y) * 32;
        for (int64_t p = (int64_t)E.slice[a].x * 32 + threadIdx.x; p < p1; p += blockDim.x) {
            const uint32_t i = E.idx[p], r = i & kEllRowMask;
            if (r != kEllPad && (int)(i >> kEllRowBits) == slot)
                val32[p] = (float)A.val[tidx<kNPar>(kNAstro + kNAtt + slot, w * E.W + r)];
        }
    }
}

// the instrument-sorted copy (rows, FP64 and binary32 values) from the
// columns: the column in lane l of slice s starts at sorted entry
// start[32 s + l]
__global__ void k_ell_sorted(SysView A, Ell E, const uint32_t *__restrict__ start,
                             uint32_t *__restrict__ irow, double *__restrict__ ival,
                             float *__restrict__ ival32)
{
    const int lane = threadIdx.x & 31;
    for (int64_t w = blockIdx.x; w < E.nwin; w += gridDim.x) {
        for (uint32_t sl = E.win[w] + (threadIdx.x >> 5); sl < E.win[w + 1]; sl += blockDim.x >> 5) {
            const uint2 s = E.slice[sl];
            uint32_t d = start[(int64_t)sl * 32 + lane];
            if (d == kEllNone)
                continue;
            for (uint32_t i = 0; i < s.y; i++, d++) {
                const int64_t p = (int64_t)s.x * 32 + (i >> 1) * 64 + 2 * lane + (i & 1);
                const uint32_t c = E.idx[p], r = c & kEllRowMask;
                if (r == kEllPad)
                    break;
                const int64_t row = w * E.W + r;
                const double v = A.val[tidx<kNPar>(kNAstro + kNAtt + (int)(c >> kEllRowBits), row)];
                irow[d] = (uint32_t)row;
                ival[d] = v;
                ival32[d] = (float)v;
            }
        }
    }
}

cudaError_t launch_ell_fill(const gsr_handle_t *h, const uint32_t *code, int64_t total, cudaStream_t st)
{
    k_ell_fill<<<h->nsm * 8, kThreads, 0, st>>>(h->sys, h->ell.W, code, total, h->d_eidx, h->d_eval32);
    return cudaGetLastError();
}

cudaError_t launch_ell_plane(const gsr_handle_t *h, int slot, cudaStream_t st)
{
    k_ell_plane<<<h->nsm * 4, kThreads, 0, st>>>(h->sys, h->ell, slot, h->d_eval32);
    return cudaGetLastError();
}

cudaError_t launch_ell_sorted(const gsr_handle_t *h, const uint32_t *start, cudaStream_t st)
{
    k_ell_sorted<<<h->nsm * 8, kThreads, 0, st>>>(h->sys, h->ell, start, h->d_irow, h->d_ival,
                                                   h->d_ival32);
    return cudaGetLastError();
}

}  // namespace gsr
