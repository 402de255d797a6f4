// dpo_device.cuh -- device helpers shared by the kernels of the delayed step:
// packet I/O (fp32 packets as one 256-bit access, bf16 packets as one
// 128-bit access, streaming cache hints) and the per-thread tensor cursor of
// the grid-stride walk over the virtual concatenation of the tensors.
#pragma once

#include "dpo_internal.h"

#include <cuda_bf16.h>
#include <math.h>

namespace dpo {
namespace {

// ------------------------------------------------------ launch overlap ----
// The step's kernels are launched with programmatic serialization
// (launch_pdl): a kernel is set up, and its CTAs start, as the last CTAs of
// the one before it exit, without waiting for that grid to be retired. Every
// thread of every such kernel calls pdl_wait before it touches memory that
// another kernel writes, or writes memory that another reads; only the
// kernel's parameters and the tables uploaded at init are read before it. It
// returns once all earlier work of the stream is complete and visible (the
// kernel before completed only after its own wait, and so on).
// So a kernel is live while the one before it still writes, and what that one
// writes is not read-only for the kernel's lifetime: the non-coherent path
// (ld_table; ld.global.nc) is for the tables of init alone. Everything else is
// read by an ordinary load: a plain one, which the wait's memory clobber keeps
// behind it, or a volatile asm, which keeps its place among volatile asms.
// No kernel asks for its successor earlier than that
// (griddepcontrol.launch_dependents at its start): CTAs that arrive while
// others still run are spread unevenly over the SMs, and the persistent
// kernels lose more than the launch costs. GB300, with against without it: the
// GPT-2 AdamW step 768 / 741 us, the clipped 1B step 8006 / 7876, GPT-2's
// Newton-Schulz step 1679 / 1565; only a clipped step on 74 thousand elements
// gained (9.5 / 10.0).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Entry of a table uploaded at init, which no kernel writes.
template <class I> __device__ __forceinline__ I ld_table(const I *p) { return __ldg(p); }

// ---------------------------------------------------------------- I/O ----
// fp32 packet: one 32-byte (256-bit) load or store per thread.

__device__ __forceinline__ void ld8(const float *p, float (&r)[8])
{
    asm volatile("ld.global.cs.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]),
                   "=f"(r[6]), "=f"(r[7])
                 : "l"(p));
}

__device__ __forceinline__ void st8(float *p, const float (&r)[8])
{
    asm volatile("st.global.cs.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 :: "l"(p), "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]),
                    "f"(r[6]), "f"(r[7])
                 : "memory");
}

// bf16 packet: one 16-byte load or store; values widen exactly to fp32.
__device__ __forceinline__ uint4 ld_packet(const __nv_bfloat16 *p)
{
    uint4 q;
    asm volatile("ld.global.cs.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w)
                 : "l"(p));
    return q;
}

__device__ __forceinline__ void ld8(const __nv_bfloat16 *p, float (&r)[8])
{
    const uint4 q = ld_packet(p);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        r[2 * j] = __uint_as_float(w[j] << 16);
        r[2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
    }
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);   // round to nearest even
    return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ void st8(__nv_bfloat16 *p, const float (&r)[8])
{
    const uint4 q = make_uint4(pack_bf16x2(r[0], r[1]), pack_bf16x2(r[2], r[3]),
                               pack_bf16x2(r[4], r[5]), pack_bf16x2(r[6], r[7]));
    __stcs(reinterpret_cast<uint4 *>(p), q);
}

__device__ __forceinline__ float ld1(const float *p)
{
    float x;
    asm volatile("ld.global.cs.f32 %0, [%1];" : "=f"(x) : "l"(p));
    return x;
}
__device__ __forceinline__ float ld1(const __nv_bfloat16 *p)
{
    uint16_t x;
    asm volatile("ld.global.b16 %0, [%1];" : "=h"(x) : "l"(p));
    return __uint_as_float((uint32_t)x << 16);
}
// A partial sum that another CTA wrote, from L2.
__device__ __forceinline__ double ld_partial(const double *p)
{
    double x;
    asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(x) : "l"(p) : "memory");
    return x;
}
__device__ __forceinline__ void st1(float *p, float x) { __stcs(p, x); }
__device__ __forceinline__ void st1(__nv_bfloat16 *p, float x) { *p = __float2bfloat16_rn(x); }

template <bool BF16> struct Elem { using T = float; };
template <> struct Elem<true> { using T = __nv_bfloat16; };

template <int SK> struct StashT { using T = float; };
template <> struct StashT<kStashBF16> { using T = __nv_bfloat16; };

// --------------------------------------------------------------- clip ----

// Norm and clip coefficient min(1, max_norm / (norm + 1e-6)) from a sum of
// squares; a NaN norm stays NaN and reaches every element.
__device__ __forceinline__ float clip_coefficient(double total, double max_norm, double &norm)
{
    norm = sqrt(total);
    const double coef = max_norm / (norm + 1e-6);
    return (float)(coef > 1.0 ? 1.0 : coef);
}

__device__ __forceinline__ void finish_clip(double total, double max_norm, NormScalars *out)
{
    double norm;
    out->clip = clip_coefficient(total, max_norm, norm);
    out->norm = norm;
    if (!isfinite(total))
        out->flags |= 1u;
}

// ------------------------------------------------------------- cursor ----

// Last i with begin[i] <= p in a sorted table (begin[0] <= p), for a p that all
// 32 lanes of the warp share. Each round the lanes probe 32 evenly spaced
// entries at once: one load latency up to 32 entries, two up to 1024, where a
// bisection takes one per halving, before a CTA's first load. GB300, against
// bisection: a clipped step on 6M elements in 60 tensors 50.0 -> 48.5 us, on 1M
// in 120 22.2 -> 21.1; five tensors and the large sets are unchanged.
template <class I>
__device__ __forceinline__ int warp_find(const I *begin, int n, I p)
{
    const int lane = threadIdx.x & 31;
    int lo = 0, len = n;   // answer in [lo, lo + len)
    while (len > 1) {
        const int step = (len + 31) / 32;
        const int i = lane * step;
        const unsigned below =
            __ballot_sync(0xFFFFFFFFu, i < len && ld_table(begin + lo + i) <= p);
        const int k = __popc(below) - 1;   // lane 0's entry is <= p
        lo += k * step;
        len = min(step, len - k * step);
    }
    return lo;
}

// The tensor holding a thread's current packet. Packet indices only grow, so
// the cursor moves forward, skipping whole tensors (empty ones included).
struct Cursor {
    int t;
    int64_t tb, te;   // packet range [tb, te) of tensor t

    // Every lane of the warp calls this, with growing packets p by lane: the
    // cursor is left on the tensor of lane 0's packet, and advance() takes it
    // on to the lane's own.
    __device__ __forceinline__ void seek(const int64_t *pkt_begin, int n, int64_t p, int64_t total)
    {
        t = warp_find(pkt_begin, n, min(__shfl_sync(0xFFFFFFFFu, p, 0), total - 1));
        tb = ld_table(pkt_begin + t);
        te = ld_table(pkt_begin + t + 1);
    }
    // true when the packet moved to another tensor (p < total)
    __device__ __forceinline__ bool advance(const int64_t *pkt_begin, int64_t p)
    {
        if (p < te)
            return false;
        do {
            ++t;
            tb = te;
            te = ld_table(pkt_begin + t + 1);
        } while (p >= te);
        return true;
    }
};

}  // namespace
}  // namespace dpo
