// What the resident marches (res2d.cu, rescyl.cu) share: cluster and mbarrier primitives, the exchange
// flags, and the projection's sums.
#pragma once
#include <cuda_runtime.h>

#include "kernels.h"

namespace cas {

namespace {

template <bool B>
struct ResFlag {
    static constexpr bool value = B;
};

template <typename R>
struct Vec16 {
    static constexpr int N = 16 / sizeof(R);
    alignas(16) R c[N];
};

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size()
{
    unsigned r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// full barrier of the cluster's threads (start and end of a launch; the steps use the mbarriers below)
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared::cluster address of this CTA's shared address `a` in the CTA of rank `r`
__device__ __forceinline__ unsigned map_rank(unsigned a, unsigned r)
{
    unsigned o;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(a), "r"(r));
    return o;
}
// 16 bytes to another CTA of the cluster, counted on that CTA's mbarrier when they have landed
__device__ __forceinline__ void st_async(unsigned a, unsigned mb, const Vec16<float> &v)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a),
                 "r"(__float_as_uint(v.c[0])), "r"(__float_as_uint(v.c[1])), "r"(__float_as_uint(v.c[2])), "r"(__float_as_uint(v.c[3])), "r"(mb)
                 : "memory");
}
__device__ __forceinline__ void st_async(unsigned a, unsigned mb, const Vec16<double> &v)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(a),
                 "l"(__double_as_longlong(v.c[0])), "l"(__double_as_longlong(v.c[1])), "r"(mb)
                 : "memory");
}
__device__ __forceinline__ void mb_init(unsigned mb, unsigned count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mb), "r"(count) : "memory"); }
__device__ __forceinline__ void mb_expect(unsigned mb, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mb_try(unsigned mb, unsigned parity)
{
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, 0x4000;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(mb), "r"(parity)
                 : "memory");
    return ok;
}
// Tries of a wait before it gives up, so that the kernel always ends.  A try that finds the phase unfinished
// takes 3.8 us (the hardware's limit on its suspension), all of them half a second of the kernel's own time,
// which no correct run comes near; no clock is read, so time the context is switched away does not count.
#ifndef RES_WAIT_TRIES
#define RES_WAIT_TRIES (1 << 17)
#endif
__device__ __noinline__ bool mb_wait_long(unsigned mb, unsigned parity)
{
    for (int i = 64; i < RES_WAIT_TRIES; ++i)
        if (mb_try(mb, parity)) return true;
    return false;
}
// Waits for the phase of the given parity; false: it gave up.
__device__ __forceinline__ bool mb_wait(unsigned mb, unsigned parity)
{
    for (int i = 0; i < (RES_WAIT_TRIES < 64 ? RES_WAIT_TRIES : 64); ++i)
        if (mb_try(mb, parity)) return true;
    return mb_wait_long(mb, parity);
}

// The end of a thread whose wait ran out: its CTA's shared memory stays a while (about a millisecond; a copy
// takes microseconds) for rows its neighbours sent that may still be in flight.
__device__ __noinline__ void linger()
{
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
}

// bits of the packed per-thread state
constexpr unsigned F_ACTIVE = 1u, F_SHORT = 2u, F_FARU = 4u, F_FARD = 8u, F_NEEDU = 16u, F_NEEDD = 32u, F_LEADU = 64u, F_LEADD = 128u,
                   F_LATE = 256u, F_STAGE = 512u, F_MINE = 1024u, F_DEAD = 2048u, F_FIRST = 4096u, F_STAGEW = 8192u;
constexpr unsigned F_PLAIN = 1u << 23;
// What a thread whose wait ran out (F_DEAD) takes no further part in: it waits no more, arms no mbarrier (another
// arrival on an unfinished phase would be undefined) and sends no row (no neighbour may count more bytes than it
// waits for); its rows go to its own CTA's slots, where nothing reads a failed run's values.
constexpr unsigned F_EXCHANGE = F_FARU | F_FARD | F_NEEDU | F_NEEDD | F_LEADU | F_LEADD;
constexpr int RES_WIN = 16;              // steps of a window of the projection
constexpr int F_W = 14;                  // valid columns less one (2 bits)
constexpr int F_ROWS = 16;               // staged rows of the block (7 bits)
constexpr int F_CU = 24, F_CD = 28;      // CTAs of the bands above and below

// (double)v; a float's without the FP64 pipe, which takes 64 clocks for a warp's conversions
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v)
{
    const unsigned b = __float_as_uint(v), m = b & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u || m == 0u)   // normal, or zero
        return __hiloint2double((int)((b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)), (int)(b << 29));
    return (double)v;
}

// The projection's sums of one CTA (indices into its dynamic shared memory, in doubles; the history in elements)
template <typename R>
struct ResSums {
    double *dd;             // dynamic shared memory
    double *terms;          // this launch's terms by piece and step, in global memory
    const short *slot, *piece;
    int n_lo, n_tail;       // first step of the launch, first step of the tail's sums
    int np, rounded, nem;   // pieces of the CTA, whether products are rounded, entries of a CTA at most
    int gw_i, we_i, ps_i, at_i, hist_i;

    // behind the staged rows at 16-byte word `w`: the launch's weights, the entries' weights, partial sums, rank 0's
    // terms by tile and launch index, the history
    __device__ __forceinline__ void layout(int w, const DevRes &D)
    {
        nem = D.ne_max;
        gw_i = 2 * w;
        we_i = gw_i + RES_LAUNCH_STEPS;
        ps_i = we_i + nem;
        at_i = ps_i + D.np_max * 16 * RES_WIN;
        hist_i = (at_i + 2 * D.ntile_max * RES_LAUNCH_INDICES) * (int)(8 / sizeof(R));
    }
    // Sums of the steps of window k that lie in [n_lo, last]: 32 partial sums a piece, added as a warp's shuffles
    // add its lanes (on horizontal faces an entry's partial sum is its place in its row and the products are
    // rounded, as in the other 2D kernels).  A half warp takes one partial sum, a lane of it one step; with
    // entries in the first 16 alone, the halves take neighbouring ones.
    __device__ __forceinline__ void part_sums(int k, int last) const
    {
        const int ln = (int)threadIdx.x & 31, half = ln / RES_WIN, st = ln & (RES_WIN - 1), n = k * RES_WIN + st;
        const R *const hs = reinterpret_cast<const R *>(dd) + hist_i + (n & (2 * RES_WIN - 1)) * nem;
        for (int pc = 0; pc < np; ++pc) {
            const short *const sl = slot + 32 * pc;
            const bool low = sl[16] == sl[32];
            for (int q = (int)threadIdx.x >> 5; q < (low ? 8 : 16); q += (int)blockDim.x >> 5) {
                double p = 0.0;
                const int g = low ? 2 * q + half : q + 16 * half;
                int e = sl[g];
                const int e1 = sl[g + 1];
                if (e < e1 && n >= n_lo && n <= last) {
                    p = dd[we_i + e] * widen(hs[e]);
                    if (rounded)
                        for (++e; e < e1; ++e) p = __dadd_rn(p, __dmul_rn(dd[we_i + e], widen(hs[e])));
                    else
                        for (++e; e < e1; ++e) p = fma(dd[we_i + e], widen(hs[e]), p);
                }
                if (!low) p += __shfl_down_sync(0xffffffffu, p, RES_WIN);
                if (low || half == 0) dd[ps_i + (pc * 16 + (g & 15)) * RES_WIN + st] = p;
            }
        }
    }
    __device__ __forceinline__ void add_window(int k, int last) const   // by the last warps, after the barrier that follows part_sums
    {
        const int nw = (int)blockDim.x >> 5;
        for (int pc = nw - 1 - ((int)threadIdx.x >> 5); pc < np; pc += nw) {
            const int ln = (int)threadIdx.x & 31, half = ln / RES_WIN, st = ln & (RES_WIN - 1), n = k * RES_WIN + st;
            const double *const ps = dd + ps_i + (pc * 16 + half) * RES_WIN + st;   // groups half, half + 2, ...
            const double a0 = ps[0] + ps[8 * RES_WIN], a2 = ps[2 * RES_WIN] + ps[10 * RES_WIN];
            const double a4 = ps[4 * RES_WIN] + ps[12 * RES_WIN], a6 = ps[6 * RES_WIN] + ps[14 * RES_WIN];
            double s = (a0 + a4) + (a2 + a6);
            s += __shfl_down_sync(0xffffffffu, s, RES_WIN);
            if (half == 0 && n >= n_lo && n <= last)
                terms[piece[pc] * RES_LAUNCH_STEPS + (n - n_lo)] = dd[gw_i + n - n_lo] * s;
        }
    }
    // Thread e of the CTA moves the value of entry e of the launch's step i, staged before the last barrier,
    // into the history; a window whose last step joined it before that barrier is summed, and its terms are
    // formed a step later (the same for every warp of the CTA).
    __device__ __forceinline__ void consume(int i, bool mine, const R *staged, int off) const
    {
        const int n = n_lo + i;
        if (mine) reinterpret_cast<R *>(dd)[hist_i + (n & (2 * RES_WIN - 1)) * nem + (int)threadIdx.x] = staged[off];
        if (nem > 0 && (n & (RES_WIN - 2)) == 0) {
            if ((n & 1) == 0 && i > 0) part_sums((n - 1) / RES_WIN, n - 1);
            if ((n & 1) == 1 && i > 1) add_window((n - 2) / RES_WIN, n - 2);
        }
    }
    // The end of a launch (cnt steps): the windows not summed yet, then rank 0 adds the terms to the
    // simulation's sums, by tile and launch index (k steps).
    __device__ __forceinline__ void finish(const DevRes &D, int cnt, double *acc, double *tail) const
    {
        const int n_hi = n_lo + cnt - 1, t2 = (int)threadIdx.x;
        __syncthreads();
        if (cnt > 1 && (n_hi & (RES_WIN - 1)) == 0) add_window((n_hi - 1) / RES_WIN, n_hi - 1);
        __syncthreads();
        part_sums(n_hi / RES_WIN, n_hi);
        __syncthreads();
        add_window(n_hi / RES_WIN, n_hi);
        if (cluster_size() > 1) {
            __syncwarp();
            cluster_sync();
        } else {
            __syncthreads();
        }
        if (cluster_rank() != 0) return;
        const int K = D.k, nt = D.ntile, total = (cnt + K - 1) / K * nt;
        const short *const tp = D.tile_pieces;
        for (int x = t2; x < total; x += (int)blockDim.x) {
            const int l = x / nt, tl = x - l * nt;
            double c = 0.0, ct = 0.0;
            for (int i = l * K; i < min(cnt, l * K + K); ++i) {
                double cq = 0.0;
                for (int p = tp[tl]; p < tp[tl + 1]; ++p) cq += *const_cast<volatile const double *>(terms + p * RES_LAUNCH_STEPS + i);
                c += cq;
                if (n_lo + i >= n_tail) ct += cq;
            }
            dd[at_i + x] = c;
            dd[at_i + D.ntile_max * RES_LAUNCH_INDICES + x] = ct;
        }
        __syncthreads();
        if (t2 == 0) {
            double a = *acc;
#pragma unroll 8
            for (int x = 0; x < total; ++x) a += dd[at_i + x];
            *acc = a;
        }
        if (t2 == (int)blockDim.x - 1 && n_hi >= n_tail) {
            double a = *tail;
#pragma unroll 8
            for (int x = 0; x < total; ++x) a += dd[at_i + D.ntile_max * RES_LAUNCH_INDICES + x];
            *tail = a;
        }
    }
};

}  // namespace

}  // namespace cas
