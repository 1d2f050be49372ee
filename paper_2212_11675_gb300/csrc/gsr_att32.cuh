// A warp's walk over the units of the offset-ordered binary32 layout (Att32),
// its tiles staged in shared memory by the bulk-copy engine.
//
// A visit is one 32-entry tile of one unit (a tile shared by two offsets is
// visited once for each), staged by one bulk copy: the values, records and
// rows of a tile are one block.  NS stages per warp: with three, tile i + 1
// has arrived while tile i is computed, so gathers of x that depend on its
// records can be issued a visit ahead; with two, tile i + 1 is on its way.
#pragma once

#include "gsr_internal.cuh"
#include "gsr_tma.cuh"

namespace gsr {

struct Visit {
    uint4 un;    // offset, first entry, end of the unit, where its sums go
    uint32_t t;  // tile
    bool ok;
    __device__ __forceinline__ bool first() const { return t == (un.y >> 5); }
    __device__ __forceinline__ bool last() const { return t == ((un.z - 1) >> 5); }
};

// One warp's visits: units u0, u0 + stride, ...
template <int NS>
struct AttWalk {
    const Att32 &U;
    const unsigned char *sp;  // this warp's stages
    uint32_t sbase, bar;      // their address and their barriers'
    int64_t u, stride;        // unit of the newest descriptor
    Visit d[NS];              // compute, (prefetch,) copy
    uint32_t phase = 0;       // bit s: parity of the phase that stage s completes next
    int s = 0;                // stage of d[0]
    int lane;

    __device__ __forceinline__ AttWalk(const Att32 &U_, unsigned char *stages, uint64_t *bars,
                                       int64_t u0, int64_t stride_)
        : U(U_), sp(stages), sbase(smem_addr(stages)), bar(smem_addr(bars)), u(u0),
          stride(stride_), lane(threadIdx.x & 31)
    {
        if (lane == 0) {
            for (int j = 0; j < NS; j++)
                mbar_init(bar + 8 * j, u0 == U.late);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        d[0].ok = u < U.nunits;
        if (d[0].ok) {
            d[0].un = __ldg(U.unit + u);
            d[0].t = d[0].un.y >> 5;
        }
        copy(d[0], 0);
#pragma unroll
        for (int j = 1; j < NS; j++) {
            d[j] = next(d[j - 1]);
            copy(d[j], j);
        }
    }

    __device__ __forceinline__ Visit next(const Visit &v)
    {
        Visit n = v;
        if (!v.ok)
            return n;
        if (!v.last()) {
            n.t++;
            return n;
        }
        u += stride;
        n.ok = u < U.nunits;
        if (n.ok) {
            n.un = __ldg(U.unit + u);
            n.t = n.un.y >> 5;
        }
        return n;
    }

    __device__ __forceinline__ void copy(const Visit &v, int st)
    {
        if (lane != 0 || !v.ok)
            return;
        mbar_expect(bar + 8 * st, kAttTileBytes);
        bulk_copy(sbase + st * kAttTileBytes, U.tile + (int64_t)v.t * kAttTileBytes, kAttTileBytes,
                  bar + 8 * st);
    }

    // stage of d[j] has arrived; false (after the other copies in flight have
    // landed, and with *kerr set) when the wait ran out
    __device__ __forceinline__ bool arrived(int j, int *kerr)
    {
        const int st = (s + j) % NS;
        const uint32_t bit = 1u << st;
        if (__all_sync(0xffffffffu, mbar_wait(bar + 8 * st, (phase & bit) ? 1u : 0u))) {
            phase ^= bit;
            return true;
        }
        if (lane == 0)
            atomicExch(kerr, 1);
        for (int i = j + 1; i < NS; i++) {
            const int si = (s + i) % NS;
            if (d[i].ok)
                mbar_wait(bar + 8 * si, (phase >> si) & 1u);
        }
        return false;
    }

    __device__ __forceinline__ const unsigned char *stage(int j) const
    {
        return sp + ((s + j) % NS) * kAttTileBytes;
    }
    __device__ __forceinline__ const float *val(int j = 0) const
    {
        return reinterpret_cast<const float *>(stage(j));
    }
    __device__ __forceinline__ uint4 rec(int j) const
    {
        return reinterpret_cast<const uint4 *>(stage(j) + kAttRecAt)[lane];
    }
    __device__ __forceinline__ uint32_t row(int j = 0) const
    {
        return reinterpret_cast<const uint32_t *>(stage(j) + kAttRowAt)[lane];
    }

    // the warp has read stage d[0]: refill it and move on
    __device__ __forceinline__ void advance()
    {
        __syncwarp();
        const Visit n = next(d[NS - 1]);
        if (lane == 0 && n.ok)
            // the warp's reads of the stage come before the engine's writes
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        copy(n, s);
#pragma unroll
        for (int j = 0; j + 1 < NS; j++)
            d[j] = d[j + 1];
        d[NS - 1] = n;
        s = (s + 1) % NS;
    }
};

}  // namespace gsr
