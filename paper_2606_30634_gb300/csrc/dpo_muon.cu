// dpo_muon.cu -- one-step-delayed Muon (Alg. 2 of arXiv 2606.30634) on the
// sm_103a tensor cores: kernels, Newton-Schulz driver and the C ABI of
// dpo_muon.h.
//
// Per step, in stream order:
//   grad_sqnorm_kernel      global ||G||^2 for clipping (shared with the
//                           elementwise path), when clipping is on
//   muon_momentum_kernel    M <- mu M + (1 - mu) G^, per-chunk partial sums of
//                           M^2 (fixed chunks: deterministic) and, by the last
//                           CTA of each matrix, 1 / (||M||_F + eps)
//   muon_normalize_kernel   X_0 = bf16(M / (||M||_F + eps)) into the padded
//                           workspace, in the wide orientation
//   ns_gemm_kernel x 3 per Newton-Schulz step and matrix shape, batched over
//                           every matrix of that shape (dpo_gemm.cuh):
//                             A = X X^T;  B = c A A + b A;  X <- B X + a X
//                           (the third reads X MN-major; at the last step it
//                           writes X^T, their output, for the tall matrices)
//   muon_apply_kernel       U = lr (r O + wd X_t) and the delayed or EF
//                           update, stash, history and bf16 weights
// With the SAPipe-WP updated-state prediction (App. B.1) the step then runs
// the pipeline once more for the prediction update: the momentum kernel
// forms M' = mu M + (1 - mu) G^ into the history buffer, M' is normalised and
// put through a second Newton-Schulz chain, and muon_predict_kernel writes
// U' = lr (r O' + wd X_{t+1}) into the history.
#include "dpo_muon.h"

#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <tuple>
#include <vector>

#include "dpo_device.cuh"
#include "dpo_gemm.cuh"
#include "dpo_reduce.cuh"

namespace dpo {
namespace muon {

constexpr int kThreads = 256;
constexpr int64_t kRound = (int64_t)kThreads * kPacket;   // elements of one CTA round (2048)
constexpr int64_t kMaxChunk = 16 * kRound;                // elements per CTA, at most
constexpr int kPad = 256;                                       // workspace padding

struct DevMat {
    void *param;
    float *master, *mom;
    void *stash;
    float *ef;
    const void *grad;
    int64_t rows, cols;
    const __nv_bfloat16 *o;   // Newton-Schulz output (workspace), row-major, pitch o_ld
    int64_t o_ld;
    __nv_bfloat16 *x, *xt;    // workspace: X_0 (R x W) and X^T (W x R)
    int64_t R, W;             // padded r <= w of the wide orientation
    float wd_lr_scale;        // 1 with DPO_WD_ON, else 0
    float r_scale;            // rms_scale sqrt(max(rows, cols)), or 1
    int sync;                 // DPO_SYNC: trained synchronously (no stash, no history)
};

// The momentum, update and prediction passes are flat over all matrices:
// matrix i owns chunks [begin[i], begin[i + 1]) of `elems` elements each, one
// CTA per chunk. One CTA row per matrix, as wide as the largest matrix, left
// a set of small matrices on a dozen CTAs (two 256 x 768 matrices: 7.9 us of
// momentum, 11.7 us of update) and launched mostly empty CTAs where sizes
// differ.
//
// The normalisation reads the momentum that was just written, and the update
// the Newton-Schulz output that was: where a pass's data outgrows L2 (129 MB),
// the next one goes through it from the end, whose lines are still there.
// Smaller sets go forward, largest matrices first in most models: five odd
// shapes (32 MB of momentum) lost 1 % backward. GB300, whole step: four
// 768-wide layers 593 -> 585 us, GPT-2 1781 -> 1773.
constexpr int64_t kBackwardBytes = 64 << 20;   // fp32 momentum of the set

struct Chunks {
    const int *begin;         // n + 1 prefix offsets
    int n;
    int elems;                // elements per chunk, a multiple of kRound
};

// Row and column of element e of a matrix with `cols` columns, by the cheaper
// 32-bit division where the matrix allows it (`small`), as most do.
__device__ __forceinline__ void row_col(int64_t e, int64_t cols, bool small, int64_t &i, int64_t &j)
{
    i = small ? (int64_t)((uint32_t)e / (uint32_t)cols) : e / cols;
    j = e - i * cols;
}

// Eight consecutive elements e.. of the Newton-Schulz output (row-major, pitch
// o_ld): one 16-byte load where rows are whole packets, else element by
// element, passing to the next row where a row ends inside the packet.
__device__ __forceinline__ void load_o8(const DevMat &d, int64_t e, bool small, float (&o)[8])
{
    int64_t i, j;
    row_col(e, d.cols, small, i, j);
    if (d.cols % kPacket == 0) {
        ld8(d.o + i * d.o_ld + j, o);
        return;
    }
    const __nv_bfloat16 *row = d.o + i * d.o_ld;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        o[k] = __bfloat162float(row[j]);
        if (++j == d.cols) {   // the packet ends inside the matrix, so a next row exists
            j = 0;             // whenever an element of it is read
            row += d.o_ld;
        }
    }
}

struct MomArgs {
    const DevMat *mats;
    Chunks ch;
    const float *clip;        // device clip coefficient, or nullptr
    float mu, omm;
    double *partials;         // one per chunk
    unsigned int *tickets;    // per matrix: chunks done, 0 between launches
    float eps;
    float *inv_norm;          // per matrix: 1 / (||M||_F + eps)
    int predict;              // M' = mu M + (1 - mu) G^ into the history buffer of each
                              // delayed matrix; M keeps its value
};

template <class GT>
__global__ void __launch_bounds__(kThreads) muon_momentum_kernel(const MomArgs a)
{
    __shared__ double red[kThreads / 32];
    __shared__ bool last;
    const int mi = warp_find(a.ch.begin, a.ch.n, (int)blockIdx.x);
    const int c0 = ld_table(a.ch.begin + mi), c1 = ld_table(a.ch.begin + mi + 1);
    const DevMat &d = a.mats[mi];
    pdl_wait();
    // the prediction pass leaves a synchronous matrix (and its history) alone
    const bool skip = a.predict && (d.sync || d.ef == nullptr);
    const int64_t n = skip ? 0 : d.rows * d.cols;
    float *out = a.predict ? d.ef : d.mom;
    const int64_t lo = (int64_t)((int)blockIdx.x - c0) * a.ch.elems;
    float sum = 0.0f, comp = 0.0f;
    if (lo < n) {
        const float clip = a.clip != nullptr ? *a.clip : 1.0f;
        const int64_t hi = lo + a.ch.elems < n ? lo + a.ch.elems : n;
        const GT *grad = static_cast<const GT *>(d.grad);
        for (int64_t e = lo + (int64_t)threadIdx.x * kPacket; e < hi; e += (int64_t)kThreads * kPacket) {
            if (e + kPacket <= hi) {
                float m[8], g[8];
                ld8(d.mom + e, m);
                ld8(grad + e, g);
                float s = 0.0f;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float gc = g[j] * clip;
                    const float p = a.omm * gc;
                    m[j] = fmaf(a.mu, m[j], p) + fmaf(a.omm, gc, -p);
                    s = fmaf(m[j], m[j], s);
                }
                st8(out + e, m);
                const float y = s - comp, t = sum + y;   // Kahan
                comp = (t - sum) - y;
                sum = t;
            } else {
                for (int64_t i = e; i < hi; ++i) {
                    const float gc = ld1(grad + i) * clip;
                    const float p = a.omm * gc;
                    const float m = fmaf(a.mu, d.mom[i], p) + fmaf(a.omm, gc, -p);
                    out[i] = m;
                    const float y = m * m - comp, t = sum + y;
                    comp = (t - sum) - y;
                    sum = t;
                }
            }
        }
    }
    // The last CTA of the matrix to arrive adds its chunks' partials in a fixed
    // order (strided over the threads, then the block's fixed tree), so the norm
    // does not depend on arrival order. A kernel of its own for this took 2.5 us
    // (two small matrices) to 9.5 us (a 7B layer's 1376 partials per matrix on
    // one warp each) and a launch.
    const double cta = block_sum<kThreads>((double)sum - (double)comp, red);
    if (threadIdx.x == 0) {
        a.partials[blockIdx.x] = cta;
        __threadfence();
        last = atomicAdd(&a.tickets[mi], 1u) == (unsigned)(c1 - c0 - 1);
    }
    __syncthreads();
    if (!last)
        return;
    __threadfence();
    double acc = 0.0;
    for (int c = c0 + (int)threadIdx.x; c < c1; c += kThreads)
        acc += ld_partial(a.partials + c);
    const double total = block_sum<kThreads>(acc, red);
    if (threadIdx.x == 0) {
        a.inv_norm[mi] = (float)(1.0 / (sqrt(total) + (double)a.eps));
        a.tickets[mi] = 0u;   // ready for the next launch
    }
}

// The normalisation works on tiles of kTile elements of X, one CTA each, over
// all matrices in one launch (matrix i owns tiles [begin[i], begin[i + 1])):
// kTileI x kTileJ of them where M is transposed, else kTile in a row.
constexpr int kTileI = 64, kTileJ = 128, kTile = kTileI * kTileJ;

struct NormalizeArgs {
    const DevMat *mats;
    const int *tile_begin;    // n + 1 prefix offsets
    int n;
    const float *inv_norm;
    int backward;             // last tiles first (see kBackwardBytes)
    int write_xt;             // no Newton-Schulz steps: X_0^T is the output of tall matrices
    int predict;              // read M' from the history buffer (zeros for a
                              // synchronous matrix) instead of M
};

// Element (i, j) of the shared tile: rows of kTileJ floats whose 16-byte
// groups are permuted by the row, so that 4 consecutive j at 8 rows i that are
// 8 apart (a warp's transposing store) and 32 groups of one row (its load)
// each take all 32 banks once.
__device__ __forceinline__ int tile_at(int i, int j)
{
    return i * kTileJ + (((j >> 2) ^ ((i ^ (i >> 3)) & 7)) << 2) + (j & 3);
}

// X_0 = bf16(M / (||M||_F + eps)) in the wide orientation, zero outside r x w.
// HBM-bound: 4 bytes in, 2 out per element. A wide matrix of whole packets has
// X's rows where M has them and is streamed through registers, four packets
// in flight per thread; a tall one is transposed through shared memory, and so
// are widths of no whole packets, whose rows start at any 4-byte address: they
// are loaded element by element, consecutive lanes on consecutive elements.
// GB300, against 64 x 64 tiles through padded shared memory for every matrix
// and one launch per shape: a 7B layer 227 -> 205 us (5.9 TB/s), GPT-2's set
// 97 -> 89 us, four 1B layers 258 -> 250 us, odd shapes 23 -> 20 us and four
// launches fewer.
__global__ void __launch_bounds__(kThreads) muon_normalize_kernel(const NormalizeArgs a)
{
    __shared__ __align__(16) float tile[kTile];
    const int block = (int)(a.backward ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
    const int mi = warp_find(a.tile_begin, a.n, block);
    const DevMat &d = a.mats[mi];
    const int t = block - ld_table(a.tile_begin + mi);
    const bool tall = d.rows > d.cols, packets = d.cols % kPacket == 0;
    pdl_wait();
    const float s = a.inv_norm[mi];
    const float *src = a.predict ? (d.sync ? nullptr : d.ef) : d.mom;
    constexpr int kVec = kTile / kPacket / kThreads;   // packets per thread
    if (!tall && packets) {
        const int64_t at = (int64_t)t * kTile;
        const int64_t ib = at / d.W;
        const uint32_t jb = (uint32_t)(at - ib * d.W), W = (uint32_t)d.W;
        float x[kVec][8];
#pragma unroll
        for (int h = 0; h < kVec; ++h) {
            const uint32_t q = jb + (threadIdx.x + h * kThreads) * kPacket;
            const int64_t i = ib + q / W, j = q % W;
            if (src != nullptr && i < d.rows && j < d.cols) {
                ld8(src + i * d.cols + j, x[h]);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    x[h][e] = 0.0f;
            }
        }
#pragma unroll
        for (int h = 0; h < kVec; ++h) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                x[h][e] *= s;
            st8(d.x + at + (threadIdx.x + h * kThreads) * kPacket, x[h]);
        }
        return;
    }
    const int tiles_j = (int)(d.W / kTileJ);
    const int64_t i0 = (int64_t)(t / tiles_j) * kTileI, j0 = (int64_t)(t % tiles_j) * kTileJ;
    // the tile of M: rows mr0.., columns mc0..
    const int64_t mr0 = tall ? j0 : i0, mc0 = tall ? i0 : j0;
    if (packets) {   // tall: 8 packets per row of M
        static_assert(kTileI / kPacket == 8, "packets per row of M");
#pragma unroll
        for (int h = 0; h < kVec; ++h) {
            const int v = (int)threadIdx.x + h * kThreads;
            const int row = v >> 3, c8 = (v & 7) * kPacket;
            float x[8];
            if (src != nullptr && mr0 + row < d.rows && mc0 + c8 < d.cols) {
                ld8(src + (mr0 + row) * d.cols + mc0 + c8, x);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    x[e] = 0.0f;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e)
                tile[tile_at(c8 + e, row)] = x[e] * s;   // X row = M column
        }
    } else {
        const int width = tall ? kTileI : kTileJ;
#pragma unroll 8
        for (int h = 0; h < kTile / kThreads; ++h) {
            const int q = (int)threadIdx.x + h * kThreads;
            const int row = q / width, col = q % width;
            const float x = src != nullptr && mr0 + row < d.rows && mc0 + col < d.cols
                                ? ld1(src + (mr0 + row) * d.cols + mc0 + col)
                                : 0.0f;
            tile[tall ? tile_at(col, row) : tile_at(row, col)] = x * s;
        }
    }
    __syncthreads();
    // one row of the tile per warp: 4 consecutive elements per lane
    static_assert(kTileJ == 32 * 4, "one row of the tile per warp");
    const int lane = (int)threadIdx.x & 31;
#pragma unroll
    for (int row = (int)threadIdx.x >> 5; row < kTileI; row += kThreads / 32) {
        const float4 o = *reinterpret_cast<const float4 *>(tile + tile_at(row, lane * 4));
        __stcs(reinterpret_cast<uint2 *>(d.x + (i0 + row) * d.W + j0 + lane * 4),
               make_uint2(pack_bf16x2(o.x, o.y), pack_bf16x2(o.z, o.w)));
    }
    if (a.write_xt && tall) {
#pragma unroll
        for (int h = 0; h < kVec; ++h) {
            const int v = (int)threadIdx.x + h * kThreads;
            const int row = v >> 3, c8 = (v & 7) * kPacket;   // row of X^T, its columns
            float o[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                o[e] = tile[tile_at(c8 + e, row)];
            st8(d.xt + (j0 + row) * d.R + i0 + c8, o);
        }
    }
}

// The update's per-call scalars (host-formed, or device-formed for a
// capturable context by muon_scalars_kernel).
struct ApplyScalars {
    float lr, lr_wd;
    int ef_now;
};

// Device-resident counters of a capturable context.
struct MuonCounters {
    int64_t k, phase_k0;
};

struct ApplyArgs {
    const DevMat *mats;
    Chunks ch;
    int backward;             // last chunks first (see kBackwardBytes)
    float lr, lr_wd, lam;
    int ef_now, hist, delayed;
    int sapipe;               // SAPipe-WP: stash := x_t - U_prev, standard rule
    int keep_hist;            // SAPipe-WP updated state: the history receives the
                              // prediction update later (muon_predict_kernel)
    const ApplyScalars *dev;  // capturable context: lr, lr_wd, ef_now of this call
};

// One thread: the next call's lr (from *lr_src when set), lr wd and whether
// EF applies (Alg. 1: from t = 2 of the delayed phase); advances k.
__global__ void muon_scalars_kernel(MuonCounters *cnt, const float *lr_src, float lr_host,
                                    double weight_decay, int ef_possible, ApplyScalars *out)
{
    pdl_wait();
    const int64_t k = cnt->k + 1;
    const int64_t t = k - cnt->phase_k0;
    const float lr = lr_src != nullptr ? *lr_src : lr_host;
    ApplyScalars sc;
    sc.lr = lr;
    sc.lr_wd = (float)((double)lr * weight_decay);
    sc.ef_now = ef_possible && t >= 2;
    *out = sc;
    cnt->k = k;
}

template <int SK>
__global__ void __launch_bounds__(kThreads) muon_apply_kernel(const ApplyArgs a)
{
    using ST = typename StashT<SK>::T;
    const int block = (int)(a.backward ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
    const int mi = warp_find(a.ch.begin, a.ch.n, block);
    const DevMat &d = a.mats[mi];
    const int64_t n = d.rows * d.cols;
    const int64_t lo = (int64_t)(block - ld_table(a.ch.begin + mi)) * a.ch.elems;
    const int64_t hi = lo + a.ch.elems < n ? lo + a.ch.elems : n;
    pdl_wait();
    const ApplyScalars sc = a.dev != nullptr ? *a.dev : ApplyScalars{a.lr, a.lr_wd, a.ef_now};
    const float lr_r = sc.lr * d.r_scale, lr_wd = sc.lr_wd * d.wd_lr_scale;
    ST *stash = static_cast<ST *>(d.stash);
    __nv_bfloat16 *param = static_cast<__nv_bfloat16 *>(d.param);
    const bool small = n <= (int64_t)UINT32_MAX;
    // a DPO_SYNC matrix takes the standard update with no stash and no history
    const bool dly = a.delayed && !d.sync;
    const bool hist = a.hist && dly, ef_now = sc.ef_now && dly;
    const bool sapipe = a.sapipe && hist;
    const bool write_hist = hist && !a.keep_hist;
    for (int64_t e = lo + (int64_t)threadIdx.x * kPacket; e < hi; e += (int64_t)kThreads * kPacket) {
        if (e + kPacket <= hi) {
            float x[8], o[8], up[8], u[8];
            ld8(d.master + e, x);
            load_o8(d, e, small, o);
            if (ef_now || sapipe)
                ld8(d.ef + e, up);
            if (SK != kStashNone && dly) {
                if (sapipe) {   // the prediction point x_t - U_prev
                    float xp[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        xp[k] = x[k] - up[k];
                    st8(stash + e, xp);
                } else {
                    st8(stash + e, x);
                }
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                u[k] = fmaf(lr_r, o[k], lr_wd * x[k]);
                x[k] -= ef_now ? fmaf(a.lam, u[k] - up[k], u[k]) : u[k];
            }
            st8(d.master + e, x);
            if (write_hist)
                st8(d.ef + e, u);
            if (param != nullptr)
                st8(param + e, x);
        } else {
            for (int64_t q = e; q < hi; ++q) {   // the matrix's last, partial packet
                const int64_t i = q / d.cols, j = q - i * d.cols;
                float x = d.master[q];
                const float o = __bfloat162float(d.o[i * d.o_ld + j]);
                if (SK != kStashNone && dly)
                    st1(stash + q, sapipe ? x - d.ef[q] : x);
                const float u = fmaf(lr_r, o, lr_wd * x);
                x -= ef_now ? fmaf(a.lam, u - d.ef[q], u) : u;
                d.master[q] = x;
                if (write_hist)
                    d.ef[q] = u;
                if (param != nullptr)
                    st1(param + q, x);
            }
        }
    }
}

// SAPipe-WP updated state (App. B.1): the prediction update
// U' = lr (r O' + wd X_{t+1}) of each delayed matrix into its history, O' the
// Newton-Schulz output of M' and X_{t+1} the master the real update left.
__global__ void __launch_bounds__(kThreads) muon_predict_kernel(const ApplyArgs a)
{
    const int mi = warp_find(a.ch.begin, a.ch.n, (int)blockIdx.x);
    const DevMat &d = a.mats[mi];
    pdl_wait();
    if (d.sync || d.ef == nullptr)
        return;
    const int64_t n = d.rows * d.cols;
    const int64_t lo = (int64_t)((int)blockIdx.x - ld_table(a.ch.begin + mi)) * a.ch.elems;
    const int64_t hi = lo + a.ch.elems < n ? lo + a.ch.elems : n;
    const ApplyScalars sc = a.dev != nullptr ? *a.dev : ApplyScalars{a.lr, a.lr_wd, a.ef_now};
    const float lr_r = sc.lr * d.r_scale, lr_wd = sc.lr_wd * d.wd_lr_scale;
    const bool small = n <= (int64_t)UINT32_MAX;
    for (int64_t e = lo + (int64_t)threadIdx.x * kPacket; e < hi; e += (int64_t)kThreads * kPacket) {
        if (e + kPacket <= hi) {
            float x[8], o[8], u[8];
            ld8(d.master + e, x);
            load_o8(d, e, small, o);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                u[k] = fmaf(lr_r, o[k], lr_wd * x[k]);
            st8(d.ef + e, u);
        } else {
            for (int64_t q = e; q < hi; ++q) {
                const int64_t i = q / d.cols, j = q - i * d.cols;
                d.ef[q] = fmaf(lr_r, __bfloat162float(d.o[i * d.o_ld + j]), lr_wd * d.master[q]);
            }
        }
    }
}

// Start state (zero_mom, zero_ef: mom = 0, ef = 0) or the restart of Alg. 1
// on entering delayed training (zero_ef only): stash := master for matrices
// trained delayed, param := master.
template <int SK>
__global__ void __launch_bounds__(kThreads) muon_init_kernel(const DevMat *mats, int zero_mom,
                                                             int zero_ef)
{
    using ST = typename StashT<SK>::T;
    const DevMat &d = mats[blockIdx.y];
    const int64_t n = d.rows * d.cols;
    ST *stash = static_cast<ST *>(d.stash);
    __nv_bfloat16 *param = static_cast<__nv_bfloat16 *>(d.param);
    for (int64_t q = (int64_t)blockIdx.x * kThreads + threadIdx.x; q < n;
         q += (int64_t)gridDim.x * kThreads) {
        const float x = d.master[q];
        if (zero_mom)
            d.mom[q] = 0.0f;
        if (zero_ef && d.ef != nullptr)
            d.ef[q] = 0.0f;
        if (SK != kStashNone && stash != nullptr && !d.sync)
            st1(stash + q, x);
        if (param != nullptr)
            st1(param + q, x);
    }
}

}  // namespace muon
}  // namespace dpo

// ------------------------------------------------------------------ host ----

namespace {

using dpo::muon::DevMat;
using dpo::muon::kPad;
using dpo::muon::kThreads;

thread_local std::string g_muon_init_err;

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                 const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                 const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_fn()
{
    static EncodeTiled fn = nullptr;
    if (fn == nullptr) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
    }
    return fn;
}

// 3-D map over nb row-major bf16 matrices of rows x cols (pitch cols),
// consecutive in memory: boxes of 64 columns x box_rows rows, 128-byte swizzle.
bool make_map(CUtensorMap *m, void *base, int64_t rows, int64_t cols, int64_t nb, int box_rows)
{
    EncodeTiled enc = encode_fn();
    if (enc == nullptr)
        return false;
    const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)nb};
    const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)(rows * cols) * 2};
    const cuuint32_t box[3] = {(cuuint32_t)dpo::gemm::kBoxK, (cuuint32_t)box_rows, 1};
    const cuuint32_t es[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same over rows x cols with 32 x 32 boxes and the 64-byte swizzle: the
// epilogue's TMA stores.
bool make_store_map(CUtensorMap *m, void *base, int64_t rows, int64_t cols, int64_t nb)
{
    EncodeTiled enc = encode_fn();
    if (enc == nullptr)
        return false;
    const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)nb};
    const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)(rows * cols) * 2};
    const cuuint32_t box[3] = {32, 32, 1};
    const cuuint32_t es[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
               CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

using GemmFn = void (*)(dpo::gemm::GemmLaunch);

// By CTAs per tile and epilogue warps (single CTAs always have eight).
GemmFn gemm_kernel(bool b_mn, int cg, int ew)
{
    using dpo::gemm::ns_gemm_kernel;
    if (cg == 1)
        return b_mn ? ns_gemm_kernel<true, 1, 8> : ns_gemm_kernel<false, 1, 8>;
    if (ew == 4)
        return b_mn ? ns_gemm_kernel<true, 2, 4> : ns_gemm_kernel<false, 2, 4>;
    return b_mn ? ns_gemm_kernel<true, 2, 8> : ns_gemm_kernel<false, 2, 8>;
}

// Estimated clocks of a launch over tiles with these K blocks, dealt round-robin
// to `slots` CTAs (cg 1) or pairs (cg 2): a slot's mainloops run back to back,
// each hiding the epilogue of the tile before it, and the last epilogue shows.
// Each product of a launch set takes the form with the smaller estimate. The
// single CTA's tile needs as many bytes per K block as its half of a pair's
// and does half of the multiplications, so it loses once every SM has several
// tiles; with few it spreads a product over more SMs, computes less past the
// diagonal and has half the epilogue. GB300, whole step, all products by pairs
// / by single CTAs / by this rule: two 256x768 matrices 133 / 99 / 99 us, one
// 768-wide layer 289 / 243 / 243, three of them 466 / 480 / 464, two
// 1024-wide layers 627 / 604 / 604, a 1536-wide one 809 / 861 / 808, an
// 1100-wide one 405 / 410 / 409. The clocks per K block and per epilogue are
// the set, of nine tried, that came closest to the better form on 15 sets.
int64_t launch_clocks(const std::vector<int> &k_blocks, int slots, int cg)
{
    const int64_t block = cg == 1 ? 700 : 1100, epilogue = cg == 1 ? 2600 : 5000;
    int64_t worst = 0;
    for (int s = 0; s < slots && s < (int)k_blocks.size(); ++s) {
        int64_t t = 0;
        for (size_t i = s; i < k_blocks.size(); i += slots)
            t += std::max(k_blocks[i] * block, i == (size_t)s ? (int64_t)0 : epilogue);
        worst = std::max(worst, t + epilogue);
    }
    return worst;
}

// A pair launch of more than kLongRounds rounds of tiles, each of at least
// kLongBlocks K blocks, is drained by four epilogue warps instead of eight: the
// next tile's mainloop hides either, and at the power cap the eight cost clocks.
// GB300, eight against four warps, whole step: the 7B set 332.0 -> 323.8 ms (327.6
// before the eight came in), a 7B layer 10370 -> 10180 us, six 2048-wide layers
// 8107 -> 8063 us, each pair from one call (runs of the single layers on another box
// were 4 % apart: the choice rests on the 7B set). Shorter K needs
// the eight (kEpiWarps), and so does a launch whose last tile is much of it.
constexpr int kLongBlocks = 16;
constexpr int64_t kLongRounds = 4;

// Rounds of single-CTA tiles above which a launch goes to the pairs unweighed.
constexpr int64_t kFewRounds = 4;

int64_t pad_up(int64_t v) { return (v + kPad - 1) / kPad * kPad; }

// One Newton-Schulz launch set: up to kMaxGroups shape groups that share each
// product's launch, and per product (X X^T, c A A + b A, B X + a X) the order
// of its groups and its part of the tile table.
struct LaunchSet {
    int n = 0;
    int group[dpo::gemm::kMaxGroups];
    struct {
        int order[dpo::gemm::kMaxGroups];   // positions in group[]
        int64_t first = 0;                  // first entry of the tile table
        int tiles = 0;
        int cg = 2;                         // CTAs per tile: 256 x 256 pairs, or 128 x 128
        int ew = 8;                         // epilogue warps of a CTA
    } prod[3];
};

struct Group {
    int64_t r, w, R, W;
    std::vector<int> mats;
    bool has_tall = false;
    // X ping-pongs between x[0] and x[1]: every tile of X <- B X + a X reads
    // all of the old X, so the new one goes to the other buffer.
    __nv_bfloat16 *x[2] = {nullptr, nullptr}, *xt = nullptr, *a = nullptr, *b = nullptr;
    CUtensorMap x128[2], a128, b128;   // 128-row K-major boxes: one CTA's half of a pair tile
    CUtensorMap x_mn[2];               // 64 x 64 boxes of X read MN-major (B of B X)
    CUtensorMap st_x[2], st_xt, st_a, st_b;   // 32 x 32 store boxes of X, X^T, A, B
};

// The matrices by their wide orientation r x w (r <= w); empty ones in no group.
std::vector<Group> group_shapes(const dpo_matrix *mats, int n)
{
    std::vector<Group> groups;
    std::map<std::pair<int64_t, int64_t>, int> gidx;
    for (int i = 0; i < n; ++i) {
        const dpo_matrix &m = mats[i];
        if (m.rows * m.cols == 0)
            continue;
        const int64_t r = std::min(m.rows, m.cols), w = std::max(m.rows, m.cols);
        auto key = std::make_pair(r, w);
        if (!gidx.count(key)) {
            gidx[key] = (int)groups.size();
            Group g;
            g.r = r;
            g.w = w;
            g.R = pad_up(r);
            g.W = pad_up(w);
            groups.push_back(g);
        }
        Group &g = groups[gidx[key]];
        g.mats.push_back(i);
        g.has_tall = g.has_tall || m.rows > m.cols;
    }
    return groups;
}

// CTA pairs and single CTAs the GEMM kernels keep resident at once.
cudaError_t gemm_residency(int sms, int *pairs, int *ctas)
{
    *pairs = *ctas = 1 << 30;
    cudaError_t e = cudaSuccess;
    for (int form = 0; form < 6 && e == cudaSuccess; ++form) {
        const int cg = form < 2 ? 1 : 2, ew = form < 4 ? 8 : 4;
        const void *fn = (const void *)gemm_kernel(form & 1, cg, ew);
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 dpo::gemm::kSmemBytes);
        int n_res = 0;
        if (e == cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(2 * std::max(1, sms / 2));
            cfg.blockDim = dim3(dpo::gemm::gemm_threads(ew));
            cfg.dynamicSmemBytes = dpo::gemm::kSmemBytes;
            e = cudaOccupancyMaxActiveClusters(&n_res, fn, &cfg);
        }
        int &have = cg == 2 ? *pairs : *ctas;
        have = std::min(have, n_res);
    }
    return e;
}

// Tiles of the three products, all by CTA pairs.
int64_t pair_tiles(const std::vector<Group> &groups)
{
    int64_t tiles = 0;
    for (const Group &g : groups) {
        const int64_t m = g.R / dpo::gemm::TM, n = g.W / dpo::gemm::TN;
        tiles += (int64_t)g.mats.size() * (m * (m + 1) + m * n);
    }
    return tiles;
}

// The GEMM launches of a Newton-Schulz step: launch sets and their tiles.
struct GemmPlan {
    bool grouped = false;
    std::vector<LaunchSet> sets;
    std::vector<int4> tiles;
};

GemmPlan plan_gemms(const dpo_matrix *mats, const std::vector<Group> &groups, int pairs, int ctas)
{
    GemmPlan plan;
    // When some shape group's launches are short (at most 16 rounds of tiles
    // over the CTA pairs), each product of a Newton-Schulz step covers all
    // shape groups in one launch: one group's tiles fill the pairs another
    // leaves idle, and a step takes 3 launches instead of 3 per group (GPT-2:
    // every group short; the Llama-1B set's 512 x 2048 group: 20.08 -> 19.80
    // ms of GEMMs per step on GB300). Sets whose groups are all long keep one
    // group per launch and run the groups' chains one after another (7B set:
    // 0.3% slower grouped; two chains at once on two streams mixed their
    // operands in L2, 336 -> 410 ms per step).
    int64_t min_tiles = INT64_MAX;
    for (const Group &g : groups)
        min_tiles = std::min<int64_t>(min_tiles, (int64_t)g.mats.size() *
                                                     (g.R / dpo::gemm::TM) * (g.W / dpo::gemm::TN));
    plan.grouped = groups.size() > 1 && min_tiles <= 16 * (int64_t)std::max(1, pairs);
    // Launch sets and their tile tables. A launch takes its groups with more K
    // blocks first: the pairs take tiles round-robin, so the longest tiles go
    // out first and the short ones fill the last round.
    std::vector<int4> &tiles = plan.tiles;
    const int per_set = plan.grouped ? dpo::gemm::kMaxGroups : 1;
    for (int g0 = 0; g0 < (int)groups.size(); g0 += per_set) {
        LaunchSet ls;
        ls.n = std::min(per_set, (int)groups.size() - g0);
        for (int q = 0; q < ls.n; ++q)
            ls.group[q] = g0 + q;
        for (int prod = 0; prod < 3; ++prod) {
            auto &p = ls.prod[prod];
            auto k_of = [&](int q) {
                const Group &g = groups[ls.group[q]];
                return prod == 0 ? g.w : g.r;
            };
            for (int q = 0; q < ls.n; ++q)
                p.order[q] = q;
            std::stable_sort(p.order, p.order + ls.n, [&](int x, int y) { return k_of(x) > k_of(y); });
            std::vector<int4> list[2];   // by single CTAs, by pairs
            std::vector<int> k_blocks[2];
            for (int cg = 1; cg <= 2; ++cg) {
                const int side = dpo::gemm::kTile(cg);
                for (int q = 0; q < ls.n; ++q) {
                    const Group &g = groups[ls.group[p.order[q]]];
                    const int64_t rows = g.r, cols = prod == 2 ? g.w : g.r;
                    const dpo::gemm::TileGrid tg{(int)((rows + side - 1) / side),
                                                 (int)((cols + side - 1) / side),
                                                 (int)g.mats.size(), prod != 2, side};
                    if (cg == 1 && tg.count() + (int64_t)list[0].size() > kFewRounds * ctas) {
                        list[0].clear();
                        break;
                    }
                    const int kb = (int)((k_of(p.order[q]) + dpo::gemm::BK - 1) / dpo::gemm::BK);
                    tg.walk([&](int b, int m0, int n0) {
                        int flags = 0;
                        if (cg == 2)
                            flags = (rows <= m0 + side / 2 ? dpo::gemm::kTileHalfM : 0) |
                                    (cols <= n0 + side / 2 ? dpo::gemm::kTileHalfN : 0);
                        const dpo_matrix &m = mats[g.mats[(size_t)b]];
                        if (m.rows > m.cols)
                            flags |= dpo::gemm::kTileTall;
                        list[cg - 1].push_back(make_int4(q | flags, b, m0, n0));
                        k_blocks[cg - 1].push_back(kb);
                    });
                }
            }
            p.cg = !list[0].empty() && launch_clocks(k_blocks[0], ctas, 1) <
                                           launch_clocks(k_blocks[1], pairs, 2)
                       ? 1
                       : 2;
            p.first = (int64_t)tiles.size();
            p.tiles = (int)list[p.cg - 1].size();
            if (p.cg == 2 && p.tiles > kLongRounds * pairs &&
                *std::min_element(k_blocks[1].begin(), k_blocks[1].end()) >= kLongBlocks)
                p.ew = 4;
            tiles.insert(tiles.end(), list[p.cg - 1].begin(), list[p.cg - 1].end());
        }
        plan.sets.push_back(ls);
    }
    return plan;
}

}  // namespace

struct dpo_muon_ctx {
    int device = 0;
    int n = 0;
    dpo_dtype stash_dt = DPO_F32, grad_dt = DPO_F32;
    dpo_muon_hparams hp{};
    bool ef = false;
    bool has_stash = false;   // some matrix has a stash buffer
    bool can_delay = true;    // every matrix without DPO_SYNC has one
    // step counters; a capturable context keeps the authoritative copy on
    // the device (d_cnt) and refreshes these from it when the host needs them
    mutable int64_t k = 0;
    mutable int64_t phase_k0 = 0;     // k when the current delayed phase began
    bool capturable = false;          // dpo_muon_set_capturable
    const float *lr_src = nullptr;    // capturable: device learning rate, or nullptr
    dpo::muon::MuonCounters *d_cnt = nullptr;
    dpo::muon::ApplyScalars *d_asc = nullptr;
    int sms = 0;
    int gemm_pairs = 0;   // clusters of 2 the GEMM kernel keeps resident at once
    int gemm_ctas = 0;    // CTAs of its single-CTA form
    int stall_launches = 0;   // dpo_muon_test_stall: GEMM launches left to stall
    std::vector<dpo_matrix> mats;
    std::vector<DevMat> host_mats;
    std::vector<Group> groups;
    std::vector<LaunchSet> sets;
    int4 *d_tiles = nullptr;          // tile table of every set and product
    int n_chunks = 0;         // CTAs of the momentum, update and prediction passes
    int chunk_elems = 0;
    int n_tiles = 0;          // CTAs of the normalisation
    int64_t total_elems = 0;
    bool backward = false;    // normalisation and update from the end (kBackwardBytes)
    int64_t ws_bytes = 0;
    double flops = 0.0;
    // device memory: one block for tables and scratch, one for the workspace
    void *dev_block = nullptr;
    void *ws = nullptr;
    DevMat *d_mats = nullptr;
    int *d_chunk_begin = nullptr;
    int *d_tile_begin = nullptr;
    double *d_partials = nullptr;
    unsigned int *d_tickets = nullptr;
    float *d_inv_norm = nullptr;
    unsigned int *d_err = nullptr;
    // gradient norm for clipping (the elementwise path's kernel and table)
    dpo::DevTensor *d_norm_table = nullptr;
    int64_t *d_pkt_begin = nullptr;
    double *d_norm_partials = nullptr;
    dpo::NormScalars *d_norm_scalars = nullptr;
    const double *clip_src = nullptr;   // external sum of squares (dpo_muon_set_clip_source)
    int64_t total_pkts = 0;
    int norm_grid = 0;
    int norm_per_thread = 1;   // packets a thread of the norm pass takes per round
    // GEMM timing (dpo_muon_set_timing): event pairs recorded since the last read
    bool timing = false;
    std::vector<cudaEvent_t> ev_pool;
    size_t ev_used = 0;
    // short GEMM launches: one launch per product covers every shape group
    bool grouped = false;
    int64_t gemm_launches = 0;
    std::string err;
};

namespace {

int mfail(dpo_muon_ctx *c, int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (c != nullptr)
        c->err = buf;
    else
        g_muon_init_err = buf;
    return code;
}

int mcuda(dpo_muon_ctx *c, cudaError_t e, const char *what)
{
    return mfail(c, DPO_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

bool aligned32(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 31u) == 0; }

void free_ctx(dpo_muon_ctx *c)
{
    if (c == nullptr)
        return;
    for (cudaEvent_t e : c->ev_pool)
        cudaEventDestroy(e);
    if (c->ws != nullptr)
        cudaFree(c->ws);
    if (c->dev_block != nullptr)
        cudaFree(c->dev_block);
    delete c;
}

int launch_init(dpo_muon_ctx *c, cudaStream_t s, int zero_mom, int zero_ef)
{
    int64_t max_n = 0;
    for (const dpo_matrix &m : c->mats)
        max_n = std::max<int64_t>(max_n, m.rows * m.cols);
    if (max_n == 0 || c->n == 0)
        return DPO_OK;
    const dim3 grid((unsigned)std::min<int64_t>((max_n + kThreads - 1) / kThreads, 4096),
                    (unsigned)c->n);
    const DevMat *m = c->d_mats;
    if (!c->has_stash)
        dpo::muon::muon_init_kernel<dpo::kStashNone><<<grid, kThreads, 0, s>>>(m, zero_mom, zero_ef);
    else if (c->stash_dt == DPO_BF16)
        dpo::muon::muon_init_kernel<dpo::kStashBF16><<<grid, kThreads, 0, s>>>(m, zero_mom, zero_ef);
    else
        dpo::muon::muon_init_kernel<dpo::kStashF32><<<grid, kThreads, 0, s>>>(m, zero_mom, zero_ef);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? DPO_OK : mcuda(c, e, "muon init launch");
}

}  // namespace

extern "C" const char *dpo_muon_last_error(const dpo_muon_ctx *c)
{
    if (c == nullptr)
        return g_muon_init_err.c_str();
    return c->err.c_str();
}

extern "C" int dpo_muon_init(dpo_muon_ctx **out, const dpo_matrix *mats, int n,
                             dpo_dtype stash_dtype, dpo_dtype grad_dtype,
                             const dpo_muon_hparams *hp, int init_mode, void *stream)
{
    if (out == nullptr)
        return mfail(nullptr, DPO_EINVAL, "out is NULL");
    *out = nullptr;
    if (hp == nullptr || n < 0 || (n > 0 && mats == nullptr))
        return mfail(nullptr, DPO_EINVAL, "NULL arguments or negative count");
    if ((stash_dtype != DPO_F32 && stash_dtype != DPO_BF16) ||
        (grad_dtype != DPO_F32 && grad_dtype != DPO_BF16))
        return mfail(nullptr, DPO_EDTYPE, "stash and grad dtypes must be F32 or BF16");
    if (!(hp->momentum >= 0.0f && hp->momentum < 1.0f) || !(hp->weight_decay >= 0.0f) ||
        !std::isfinite(hp->ef_lambda) || hp->ns_steps < 0 || hp->ns_steps > 16 ||
        !(hp->ns_eps >= 0.0f) || !(hp->rms_scale >= 0.0f) || (hp->delay != 0 && hp->delay != 1) ||
        !std::isfinite(hp->ns_a) || !std::isfinite(hp->ns_b) || !std::isfinite(hp->ns_c))
        return mfail(nullptr, DPO_EINVAL, "hyperparameter out of range");
    if (hp->correction != DPO_CORR_EF && hp->correction != DPO_CORR_SAPIPE_SAME &&
        hp->correction != DPO_CORR_SAPIPE_UPDATED)
        return mfail(nullptr, DPO_EINVAL, "correction must be one of DPO_CORR_*");
    if (init_mode != DPO_INIT_FRESH && init_mode != DPO_INIT_RESUME)
        return mfail(nullptr, DPO_EINVAL, "bad init_mode");
    const bool ef = n > 0 && mats[0].ef != nullptr;
    for (int i = 0; i < n; ++i) {
        const dpo_matrix &m = mats[i];
        if (m.rows < 0 || m.cols < 0)
            return mfail(nullptr, DPO_EINVAL, "matrix %d: negative shape", i);
        if (m.rows * m.cols == 0)
            continue;
        if (m.master == nullptr || m.mom == nullptr || m.grad == nullptr)
            return mfail(nullptr, DPO_EINVAL, "matrix %d: master, mom and grad are required", i);
        if ((m.flags & ~(DPO_WD_ON | DPO_SYNC)) != 0)
            return mfail(nullptr, DPO_EINVAL, "matrix %d: unknown flags", i);
        if (hp->delay == 1 && m.stash == nullptr && !(m.flags & DPO_SYNC))
            return mfail(nullptr, DPO_EINVAL, "matrix %d: delay 1 needs a stash", i);
        if ((m.ef != nullptr) != ef)
            return mfail(nullptr, DPO_EINVAL, "ef buffers must be given for all matrices or none");
        const void *ps[6] = {m.param, m.master, m.mom, m.stash, m.ef, m.grad};
        for (const void *p : ps)
            if (p != nullptr && !aligned32(p))
                return mfail(nullptr, DPO_EALIGN, "matrix %d: buffer not 32-byte aligned", i);
    }

    dpo_muon_ctx *c = new dpo_muon_ctx();
    c->n = n;
    c->stash_dt = stash_dtype;
    c->grad_dt = grad_dtype;
    c->hp = *hp;
    c->ef = ef;
    c->mats.assign(mats, mats + n);
    for (int i = 0; i < n; ++i) {
        if (mats[i].rows * mats[i].cols == 0)
            continue;
        c->has_stash = c->has_stash || mats[i].stash != nullptr;
        c->can_delay = c->can_delay && (mats[i].stash != nullptr || (mats[i].flags & DPO_SYNC));
    }
    cudaGetDevice(&c->device);
    cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, c->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);

    c->groups = group_shapes(mats, n);
    for (int i = 0; i < n; ++i) {
        const int64_t r = std::min(mats[i].rows, mats[i].cols);
        const int64_t w = std::max(mats[i].rows, mats[i].cols);
        c->total_elems += r * w;
        // unique entries of the symmetric products X X^T (r (r + 1) / 2, each
        // w multiply-adds) and A A (r (r + 1) / 2, r each), all of B X
        c->flops += (double)hp->ns_steps * ((double)r * (r + 1) * w + (double)r * (r + 1) * r +
                                            2.0 * (double)r * r * w);
    }
    // Chunks of the flat passes: about 16 CTAs per SM, so a set of a few
    // million elements still covers the SMs several times over, and at most
    // kMaxChunk elements each, where a CTA's fixed cost no longer shows.
    const int64_t want = c->total_elems / (16 * (int64_t)std::max(1, c->sms));
    int64_t ce = std::max<int64_t>(
        dpo::muon::kRound,
        std::min<int64_t>(dpo::muon::kMaxChunk,
                          (want + dpo::muon::kRound - 1) / dpo::muon::kRound * dpo::muon::kRound));
    std::vector<int> chunk_begin(n + 1, 0), tile_begin(n + 1, 0);
    int64_t n_chunks = 0, n_tiles = 0;   // below 2^31 for any set that fits the device
    for (int i = 0; i < n; ++i) {
        const int64_t ne = mats[i].rows * mats[i].cols;
        n_chunks += (ne + ce - 1) / ce;
        chunk_begin[i + 1] = (int)n_chunks;
        if (ne > 0)
            n_tiles += pad_up(mats[i].rows) * pad_up(mats[i].cols) / dpo::muon::kTile;
        tile_begin[i + 1] = (int)n_tiles;
    }
    c->n_chunks = (int)n_chunks;
    c->backward = 4 * c->total_elems > dpo::muon::kBackwardBytes;
    c->chunk_elems = (int)ce;
    c->n_tiles = (int)n_tiles;

    // Workspace: per group X twice, X^T (the output of tall matrices), A, B (bf16).
    int64_t ws = 0;
    for (const Group &g : c->groups) {
        const int64_t nb = (int64_t)g.mats.size();
        ws += nb * (g.R * g.W * 3 + g.R * g.R * 2) * 2;
    }
    c->ws_bytes = ws;
    // (a failure is reported after the allocations, where the launches it stops
    // would come)
    const cudaError_t e_gemm = gemm_residency(c->sms, &c->gemm_pairs, &c->gemm_ctas);
    // Room for the GEMM tile table, at most: a launch goes to single CTAs with up
    // to kFewRounds rounds of them, four in the place of a pair's. The table is
    // made once the workspace is there: that of a set far past the device would
    // take the host's memory before the allocation could fail.
    const int64_t by_pairs = pair_tiles(c->groups);
    const int64_t max_tiles =
        by_pairs + 3 * std::min<int64_t>(by_pairs, (int64_t)c->groups.size() * kFewRounds *
                                                       (e_gemm == cudaSuccess ? c->gemm_ctas : 0));
    // Norm-pass table (the elementwise path's gradient-norm kernel).
    int64_t total_pkts = 0;
    std::vector<int64_t> pkt_begin(n + 1, 0);
    for (int i = 0; i < n; ++i) {
        pkt_begin[i] = total_pkts;
        total_pkts += (mats[i].rows * mats[i].cols + dpo::kPacket - 1) / dpo::kPacket;
    }
    pkt_begin[n] = total_pkts;
    c->total_pkts = total_pkts;
    int per_sm_norm = 0;
    dpo::norm_ctas_per_sm(grad_dtype == DPO_BF16, &per_sm_norm);
    c->norm_per_thread = dpo::norm_per_thread(grad_dtype == DPO_BF16, total_pkts);
    const int64_t norm_groups =
        (total_pkts + (int64_t)dpo::kNormThreads * c->norm_per_thread - 1) /
        ((int64_t)dpo::kNormThreads * c->norm_per_thread);
    c->norm_grid = (int)std::max<int64_t>(
        1, std::min<int64_t>(norm_groups, (int64_t)std::max(1, c->sms) * std::max(1, per_sm_norm)));

    // Device block: mats | partials | chunk and tile prefixes | tickets |
    // inv_norm | err | norm table | pkt_begin | norm partials | norm scalars |
    // capturable counters and scalars | GEMM tile table.
    auto al = [](int64_t v) { return (v + 255) / 256 * 256; };
    int64_t off = 0;
    const int64_t o_mats = off;
    off += al((int64_t)sizeof(DevMat) * std::max(1, n));
    const int64_t o_part = off;
    off += al((int64_t)sizeof(double) * std::max(1, c->n_chunks));
    const int64_t o_cbeg = off;
    off += al((int64_t)sizeof(int) * (n + 1));
    const int64_t o_tbeg = off;
    off += al((int64_t)sizeof(int) * (n + 1));
    const int64_t o_tick = off;
    off += al((int64_t)sizeof(unsigned int) * std::max(1, n));
    const int64_t o_inv = off;
    off += al((int64_t)sizeof(float) * std::max(1, n));
    const int64_t o_err = off;
    off += al(sizeof(unsigned int));
    const int64_t o_ntab = off;
    off += al((int64_t)sizeof(dpo::DevTensor) * std::max(1, n));
    const int64_t o_pkt = off;
    off += al((int64_t)sizeof(int64_t) * (n + 1));
    const int64_t o_npart = off;
    off += al((int64_t)sizeof(double) * c->norm_grid);
    const int64_t o_nsc = off;
    off += al(sizeof(dpo::NormScalars));
    const int64_t o_cnt = off;
    off += al(sizeof(dpo::muon::MuonCounters));
    const int64_t o_asc = off;
    off += al(sizeof(dpo::muon::ApplyScalars));
    const int64_t o_tiles = off;
    off += al((int64_t)sizeof(int4) * std::max<int64_t>(1, max_tiles));

    cudaError_t e = dpo::device_alloc(&c->dev_block, (size_t)off);
    if (e != cudaSuccess) {
        free_ctx(c);
        return mfail(nullptr, DPO_ENOMEM, "device table allocation failed");
    }
    if (ws > 0) {
        e = dpo::device_alloc(&c->ws, (size_t)ws);
        if (e != cudaSuccess) {
            free_ctx(c);
            return mfail(nullptr, DPO_ENOMEM, "Newton-Schulz workspace (%lld bytes) allocation failed",
                         (long long)ws);
        }
    }
    if (e_gemm != cudaSuccess || c->gemm_pairs < 1 || c->gemm_ctas < 1) {
        free_ctx(c);
        return e_gemm != cudaSuccess ? mcuda(nullptr, e_gemm, "GEMM launch configuration")
                                     : mfail(nullptr, DPO_ECUDA, "GEMM kernel cannot be resident");
    }
    const GemmPlan plan = plan_gemms(mats, c->groups, c->gemm_pairs, c->gemm_ctas);
    if ((int64_t)plan.tiles.size() > max_tiles) {
        free_ctx(c);
        return mfail(nullptr, DPO_ECUDA, "GEMM tile table larger than its room");
    }
    c->grouped = plan.grouped;
    c->sets = plan.sets;
    char *blk = static_cast<char *>(c->dev_block);
    c->d_mats = reinterpret_cast<DevMat *>(blk + o_mats);
    c->d_partials = reinterpret_cast<double *>(blk + o_part);
    c->d_chunk_begin = reinterpret_cast<int *>(blk + o_cbeg);
    c->d_tile_begin = reinterpret_cast<int *>(blk + o_tbeg);
    c->d_tickets = reinterpret_cast<unsigned int *>(blk + o_tick);
    c->d_inv_norm = reinterpret_cast<float *>(blk + o_inv);
    c->d_err = reinterpret_cast<unsigned int *>(blk + o_err);
    c->d_norm_table = reinterpret_cast<dpo::DevTensor *>(blk + o_ntab);
    c->d_pkt_begin = reinterpret_cast<int64_t *>(blk + o_pkt);
    c->d_norm_partials = reinterpret_cast<double *>(blk + o_npart);
    c->d_norm_scalars = reinterpret_cast<dpo::NormScalars *>(blk + o_nsc);
    c->d_cnt = reinterpret_cast<dpo::muon::MuonCounters *>(blk + o_cnt);
    c->d_asc = reinterpret_cast<dpo::muon::ApplyScalars *>(blk + o_asc);
    c->d_tiles = reinterpret_cast<int4 *>(blk + o_tiles);

    // Carve the workspace and build the tensor maps.
    char *wp = static_cast<char *>(c->ws);
    c->host_mats.resize(n);
    for (int i = 0; i < n; ++i) {
        const dpo_matrix &m = mats[i];
        DevMat &d = c->host_mats[i];
        d.param = m.param;
        d.master = m.master;
        d.mom = m.mom;
        d.stash = m.stash;
        d.ef = m.ef;
        d.grad = m.grad;
        d.rows = m.rows;
        d.cols = m.cols;
        d.o = nullptr;
        d.o_ld = 0;
        d.x = d.xt = nullptr;
        d.R = d.W = 0;
        d.wd_lr_scale = (m.flags & DPO_WD_ON) ? 1.0f : 0.0f;
        d.r_scale = hp->rms_scale > 0.0f
                        ? (float)(hp->rms_scale * std::sqrt((double)std::max(m.rows, m.cols)))
                        : 1.0f;
        d.sync = (m.flags & DPO_SYNC) ? 1 : 0;
    }
    for (Group &g : c->groups) {
        const int64_t nb = (int64_t)g.mats.size();
        for (int q = 0; q < 2; ++q) {
            g.x[q] = reinterpret_cast<__nv_bfloat16 *>(wp);
            wp += nb * g.R * g.W * 2;
        }
        g.xt = reinterpret_cast<__nv_bfloat16 *>(wp);
        wp += nb * g.W * g.R * 2;
        g.a = reinterpret_cast<__nv_bfloat16 *>(wp);
        wp += nb * g.R * g.R * 2;
        g.b = reinterpret_cast<__nv_bfloat16 *>(wp);
        wp += nb * g.R * g.R * 2;
        const bool ok = make_map(&g.x128[0], g.x[0], g.R, g.W, nb, dpo::gemm::BM) &&
                        make_map(&g.x128[1], g.x[1], g.R, g.W, nb, dpo::gemm::BM) &&
                        make_map(&g.a128, g.a, g.R, g.R, nb, dpo::gemm::BM) &&
                        make_map(&g.b128, g.b, g.R, g.R, nb, dpo::gemm::BM) &&
                        make_map(&g.x_mn[0], g.x[0], g.R, g.W, nb, 64) &&
                        make_map(&g.x_mn[1], g.x[1], g.R, g.W, nb, 64) &&
                        make_store_map(&g.st_x[0], g.x[0], g.R, g.W, nb) &&
                        make_store_map(&g.st_x[1], g.x[1], g.R, g.W, nb) &&
                        make_store_map(&g.st_xt, g.xt, g.W, g.R, nb) &&
                        make_store_map(&g.st_a, g.a, g.R, g.R, nb) &&
                        make_store_map(&g.st_b, g.b, g.R, g.R, nb);
        if (!ok) {
            free_ctx(c);
            return mfail(nullptr, DPO_ECUDA, "tensor map encoding failed");
        }
        // Newton-Schulz output: X (wide matrices) or X^T (tall ones, whose
        // rows are the original matrix's rows; written by the normalisation
        // when there are no steps, else by the last step).
        for (size_t bi = 0; bi < g.mats.size(); ++bi) {
            DevMat &d = c->host_mats[g.mats[bi]];
            d.x = g.x[0] + (int64_t)bi * g.R * g.W;
            d.xt = g.xt + (int64_t)bi * g.W * g.R;
            d.R = g.R;
            d.W = g.W;
            if (d.rows > d.cols) {
                d.o = g.xt + (int64_t)bi * g.W * g.R;
                d.o_ld = g.R;
            } else {   // the buffer the last step wrote
                d.o = g.x[hp->ns_steps % 2] + (int64_t)bi * g.R * g.W;
                d.o_ld = g.W;
            }
        }
    }
    std::vector<dpo::DevTensor> ntab(n);
    for (int i = 0; i < n; ++i) {
        dpo::DevTensor t{};
        t.grad = mats[i].grad;
        t.numel = mats[i].rows * mats[i].cols;
        ntab[i] = t;
    }

#define MUON_COPY(dst, src, bytes)                                                      \
    do {                                                                                \
        if ((bytes) > 0) {                                                              \
            e = cudaMemcpyAsync((dst), (src), (size_t)(bytes), cudaMemcpyHostToDevice, s); \
            if (e != cudaSuccess) {                                                     \
                free_ctx(c);                                                            \
                return mcuda(nullptr, e, "table upload");                               \
            }                                                                           \
        }                                                                               \
    } while (0)
    MUON_COPY(c->d_mats, c->host_mats.data(), sizeof(DevMat) * n);
    MUON_COPY(c->d_norm_table, ntab.data(), sizeof(dpo::DevTensor) * n);
    MUON_COPY(c->d_pkt_begin, pkt_begin.data(), sizeof(int64_t) * (n + 1));
    MUON_COPY(c->d_chunk_begin, chunk_begin.data(), sizeof(int) * (n + 1));
    MUON_COPY(c->d_tiles, plan.tiles.data(), sizeof(int4) * plan.tiles.size());
    MUON_COPY(c->d_tile_begin, tile_begin.data(), sizeof(int) * (n + 1));
#undef MUON_COPY
    e = cudaMemsetAsync(c->d_err, 0, sizeof(unsigned int), s);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(c->d_norm_scalars, 0, sizeof(dpo::NormScalars), s);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(c->d_tickets, 0, sizeof(unsigned int) * std::max(1, n), s);
    if (e == cudaSuccess && ws > 0)
        e = cudaMemsetAsync(c->ws, 0, (size_t)ws, s);   // zero padding stays zero
    if (e != cudaSuccess) {
        free_ctx(c);
        return mcuda(nullptr, e, "workspace clear");
    }
    if (init_mode == DPO_INIT_FRESH) {
        const int rc = launch_init(c, s, 1, 1);
        if (rc != DPO_OK) {
            g_muon_init_err = c->err;
            free_ctx(c);
            return rc;
        }
    }
    *out = c;
    return DPO_OK;
}

namespace {

// One product of a Newton-Schulz step for one shape group.
struct GemmJob {
    const CUtensorMap *ta, *tb, *td, *tdt;
    dpo::gemm::Params p;
};

// One launch over the jobs of one product of a launch set (all read B K-major,
// or all MN-major), in the order of its tile table.
int launch_gemm(dpo_muon_ctx *c, const LaunchSet &ls, int prod, const GemmJob *jobs, cudaStream_t s)
{
    const auto &pr = ls.prod[prod];
    dpo::gemm::GemmLaunch L;
    std::memset(&L, 0, sizeof L);
    for (int q = 0; q < ls.n; ++q) {
        const GemmJob &j = jobs[pr.order[q]];
        dpo::gemm::GemmGroup &G = L.g[q];
        G.a = *j.ta;
        G.b = *j.tb;
        G.d = *j.td;
        G.dt = *j.tdt;
        G.p = j.p;
    }
    L.tiles = c->d_tiles + pr.first;
    L.n_groups = ls.n;
    L.n_tiles = pr.tiles;
    // one CTA pair per co-resident cluster slot, or one CTA per SM (the tile
    // walk assumes that all of them run at once)
    const int grid = pr.cg * std::min(pr.tiles, pr.cg == 2 ? c->gemm_pairs : c->gemm_ctas);
    const cudaError_t e =
        dpo::launch_pdl(gemm_kernel(prod == 2, pr.cg, pr.ew), dim3(grid),
                        dpo::gemm::gemm_threads(pr.ew), dpo::gemm::kSmemBytes, s, L);
    if (c->timing)
        ++c->gemm_launches;
    return e == cudaSuccess ? DPO_OK : mcuda(c, e, "Newton-Schulz GEMM launch");
}

}  // namespace

namespace {

// Momentum (M <- mu M + (1 - mu) G^, or with `predict` M' into the history
// buffers), its Frobenius norms, the normalisation into the workspace and the
// Newton-Schulz chains of every shape group: the Newton-Schulz output of each
// matrix is then in the workspace (DevMat::o).
int orthogonalize(dpo_muon_ctx *c, cudaStream_t s, bool predict)
{
    // momentum and its Frobenius norms
    dpo::muon::MomArgs ma{};
    ma.mats = c->d_mats;
    ma.ch = dpo::muon::Chunks{c->d_chunk_begin, c->n, c->chunk_elems};
    ma.clip = c->hp.max_grad_norm > 0.0f ? &c->d_norm_scalars->clip : nullptr;
    ma.mu = c->hp.momentum;
    ma.omm = (float)(1.0 - (double)c->hp.momentum);
    ma.partials = c->d_partials;
    ma.tickets = c->d_tickets;
    ma.eps = c->hp.ns_eps;
    ma.inv_norm = c->d_inv_norm;
    ma.predict = predict ? 1 : 0;
    const dim3 mgrid((unsigned)c->n_chunks);
    cudaError_t e = dpo::launch_pdl(c->grad_dt == DPO_BF16
                                        ? dpo::muon::muon_momentum_kernel<__nv_bfloat16>
                                        : dpo::muon::muon_momentum_kernel<float>,
                                    mgrid, kThreads, 0, s, ma);
    if (e != cudaSuccess)
        return mcuda(c, e, "momentum launch");
    const dpo::muon::NormalizeArgs na{c->d_mats, c->d_tile_begin, c->n, c->d_inv_norm,
                                      c->backward ? 1 : 0,
                                      c->hp.ns_steps == 0 ? 1 : 0, predict ? 1 : 0};
    e = dpo::launch_pdl(dpo::muon::muon_normalize_kernel, dim3((unsigned)c->n_tiles), kThreads, 0,
                        s, na);
    if (e != cudaSuccess)
        return mcuda(c, e, "normalize launch");
    cudaEvent_t ev_end = nullptr;
    if (c->timing && c->hp.ns_steps > 0) {
        if (c->ev_used + 2 > c->ev_pool.size()) {
            for (int q = 0; q < 2; ++q) {
                cudaEvent_t ev;
                if ((e = cudaEventCreate(&ev)) != cudaSuccess)
                    return mcuda(c, e, "timing event");
                c->ev_pool.push_back(ev);
            }
        }
        if ((e = cudaEventRecord(c->ev_pool[c->ev_used], s)) != cudaSuccess)
            return mcuda(c, e, "timing event record");
        ev_end = c->ev_pool[c->ev_used + 1];
        c->ev_used += 2;
    }
    // Newton-Schulz, per step: A = X X^T, B = c A A + b A, X <- B X + a X.
    // Short launches (c->grouped) take the same product of up to kMaxGroups
    // shape groups in one launch, step by step; long ones run one group's
    // chain after another, one launch per product.
    auto stall_next = [c]() {
        if (c->stall_launches <= 0)
            return 0;
        --c->stall_launches;
        return 1;
    };
    for (const LaunchSet &ls : c->sets) {
        for (int it = 0; it < c->hp.ns_steps; ++it) {
            const bool last = it + 1 == c->hp.ns_steps;
            const int cur = it % 2, nxt = cur ^ 1;
            GemmJob xx[dpo::gemm::kMaxGroups], aa[dpo::gemm::kMaxGroups],
                bx[dpo::gemm::kMaxGroups];
            const int st_xx = stall_next(), st_aa = stall_next(), st_bx = stall_next();
            for (int q = 0; q < ls.n; ++q) {
                Group &g = c->groups[ls.group[q]];
                dpo::gemm::Params p{};
                p.err = c->d_err;
                // A = X X^T
                p.alpha = 1.0f;
                p.k_blocks = (int)((g.w + dpo::gemm::BK - 1) / dpo::gemm::BK);
                p.sym = 1;
                p.stall = st_xx;
                xx[q] = GemmJob{&g.x128[cur], &g.x128[cur], &g.st_a, &g.st_a, p};
                // B = c A A + b A
                p.c = g.a;
                p.ldc = g.R;
                p.c_bstride = g.R * g.R;
                p.alpha = c->hp.ns_c;
                p.beta = c->hp.ns_b;
                p.k_blocks = (int)((g.r + dpo::gemm::BK - 1) / dpo::gemm::BK);
                p.stall = st_aa;
                aa[q] = GemmJob{&g.a128, &g.a128, &g.st_b, &g.st_b, p};
                // X <- B X + a X (X read MN-major in place of X^T), and at the
                // last step X^T, the output, in place of X for the tall matrices
                p.sym = 0;
                p.trans = last && g.has_tall ? 1 : 0;
                p.c = g.x[cur];
                p.ldc = g.W;
                p.c_bstride = g.R * g.W;
                p.alpha = 1.0f;
                p.beta = c->hp.ns_a;
                p.k_blocks = (int)((g.r + dpo::gemm::BK - 1) / dpo::gemm::BK);
                p.stall = st_bx;
                bx[q] = GemmJob{&g.b128, &g.x_mn[cur], &g.st_x[nxt], &g.st_xt, p};
            }
            int rc = launch_gemm(c, ls, 0, xx, s);
            if (rc == DPO_OK)
                rc = launch_gemm(c, ls, 1, aa, s);
            if (rc == DPO_OK)
                rc = launch_gemm(c, ls, 2, bx, s);
            if (rc != DPO_OK)
                return rc;
        }
    }
    if (ev_end != nullptr && (e = cudaEventRecord(ev_end, s)) != cudaSuccess)
        return mcuda(c, e, "timing event record");

    return DPO_OK;
}

}  // namespace

namespace {

// ||G||^2 over all matrices: into *accum when it is given, else to the norm and
// clip coefficient of the context.
cudaError_t launch_grad_norm(dpo_muon_ctx *c, double *accum, cudaStream_t s)
{
    const dpo::NormArgs na{c->d_norm_table, c->d_pkt_begin, c->n, c->total_pkts,
                           c->norm_per_thread, c->d_norm_partials};
    const cudaError_t e = dpo::launch_norm(c->grad_dt == DPO_BF16, c->norm_grid, na, s);
    if (e != cudaSuccess)
        return e;
    return dpo::launch_norm_finish(c->d_norm_partials, c->norm_grid, c->hp.max_grad_norm, accum,
                                   c->d_norm_scalars, s);
}

}  // namespace

extern "C" int dpo_muon_step(dpo_muon_ctx *c, float lr, void *stream)
{
    if (c == nullptr)
        return DPO_EINVAL;
    if (!(lr > 0.0f) || !std::isfinite(lr))
        return mfail(c, DPO_EINVAL, "lr must be positive and finite");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int64_t k = c->k + 1;
    if (c->n == 0 || c->total_elems == 0) {
        if (c->capturable) {   // keep the device counter in step
            const cudaError_t e = dpo::launch_pdl(dpo::muon::muon_scalars_kernel, dim3(1), 1, 0, s,
                                                  c->d_cnt, c->lr_src, lr, 0.0, 0, c->d_asc);
            return e == cudaSuccess ? DPO_OK : mcuda(c, e, "scalars launch");
        }
        c->k = k;
        return DPO_OK;
    }
    const bool clip = c->hp.max_grad_norm > 0.0f;
    if (clip && c->clip_src != nullptr) {
        const cudaError_t e = dpo::launch_clip_from_sumsq(c->clip_src, c->hp.max_grad_norm,
                                                          c->d_norm_scalars, s);
        if (e != cudaSuccess)
            return mcuda(c, e, "clip-coefficient launch");
    } else if (clip) {
        const cudaError_t e = launch_grad_norm(c, nullptr, s);
        if (e != cudaSuccess)
            return mcuda(c, e, "norm launch");
    }
    int rc = orthogonalize(c, s, false);
    if (rc != DPO_OK)
        return rc;
    cudaError_t e;
    const dim3 mgrid((unsigned)c->n_chunks);

    // update, stash, history, weights
    const int64_t t = k - c->phase_k0;   // Alg. 1 iteration within the delayed phase
    dpo::muon::ApplyArgs aa{};
    aa.mats = c->d_mats;
    aa.ch = dpo::muon::Chunks{c->d_chunk_begin, c->n, c->chunk_elems};
    aa.backward = c->backward ? 1 : 0;
    aa.lr = lr;
    aa.lr_wd = (float)((double)lr * (double)c->hp.weight_decay);
    aa.delayed = c->hp.delay == 1;
    aa.hist = c->ef && c->hp.delay == 1;
    const bool updated = c->hp.correction == DPO_CORR_SAPIPE_UPDATED;
    aa.sapipe = c->hp.correction == DPO_CORR_SAPIPE_SAME || updated;
    aa.keep_hist = updated;
    aa.ef_now = aa.hist && !aa.sapipe && t >= 2 && c->hp.ef_lambda != 0.0f;
    aa.lam = c->hp.ef_lambda;
    if (c->capturable) {   // lr and EF's start from the device counters
        e = dpo::launch_pdl(dpo::muon::muon_scalars_kernel, dim3(1), 1, 0, s, c->d_cnt, c->lr_src,
                            lr, (double)c->hp.weight_decay,
                            aa.hist && !aa.sapipe && c->hp.ef_lambda != 0.0f ? 1 : 0, c->d_asc);
        if (e != cudaSuccess)
            return mcuda(c, e, "scalars launch");
        aa.dev = c->d_asc;
    }
    const bool st = c->hp.delay == 1;
    e = dpo::launch_pdl(!st ? dpo::muon::muon_apply_kernel<dpo::kStashNone>
                        : c->stash_dt == DPO_BF16 ? dpo::muon::muon_apply_kernel<dpo::kStashBF16>
                                                  : dpo::muon::muon_apply_kernel<dpo::kStashF32>,
                        mgrid, kThreads, 0, s, aa);
    if (e != cudaSuccess)
        return mcuda(c, e, "apply launch");
    if (updated && aa.hist) {
        // SAPipe-WP updated state: the step once more on the same gradient
        // from the momentum just stored, decaying X_{t+1}, into the history
        if ((rc = orthogonalize(c, s, true)) != DPO_OK)
            return rc;
        if ((e = dpo::launch_pdl(dpo::muon::muon_predict_kernel, mgrid, kThreads, 0, s, aa)) !=
            cudaSuccess)
            return mcuda(c, e, "prediction launch");
    }
    if (!c->capturable)
        c->k = k;
    return DPO_OK;
}

namespace {

// A capturable context's counters live on the device: refresh the host copy
// (after all work so far), or write the host copy back.
int mpull(const dpo_muon_ctx *c)
{
    if (!c->capturable)
        return DPO_OK;
    dpo::muon::MuonCounters h{};
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess)
        e = cudaMemcpy(&h, c->d_cnt, sizeof h, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess)
        return DPO_ECUDA;
    c->k = h.k;
    c->phase_k0 = h.phase_k0;
    return DPO_OK;
}

int mpush(const dpo_muon_ctx *c, cudaStream_t s)
{
    const dpo::muon::MuonCounters h{c->k, c->phase_k0};
    // pageable source: the call returns once the bytes are staged
    return cudaMemcpyAsync(c->d_cnt, &h, sizeof h, cudaMemcpyHostToDevice, s) == cudaSuccess
               ? DPO_OK
               : DPO_ECUDA;
}

}  // namespace

extern "C" int dpo_muon_set_capturable(dpo_muon_ctx *c, int on, const float *lr_source,
                                       void *stream)
{
    if (c == nullptr)
        return DPO_EINVAL;
    if (lr_source != nullptr && reinterpret_cast<uintptr_t>(lr_source) % alignof(float) != 0)
        return mfail(c, DPO_EINVAL, "lr_source must be 4-byte aligned");
    if (on) {
        if (!c->capturable && mpush(c, static_cast<cudaStream_t>(stream)) != DPO_OK)
            return mfail(c, DPO_ECUDA, "writing the device step counters failed");
        c->capturable = true;
        c->lr_src = lr_source;
    } else {
        if (c->capturable && mpull(c) != DPO_OK)
            return mfail(c, DPO_ECUDA, "reading the device step counters failed");
        c->capturable = false;
        c->lr_src = nullptr;
    }
    return DPO_OK;
}

extern "C" int dpo_muon_set_delay(dpo_muon_ctx *c, int delay, void *stream)
{
    if (c == nullptr)
        return DPO_EINVAL;
    if (delay != 0 && delay != 1)
        return mfail(c, DPO_EINVAL, "delay must be 0 or 1");
    if (delay == c->hp.delay)
        return DPO_OK;
    if (delay == 1) {
        if (!c->can_delay)
            return mfail(c, DPO_ESTATE,
                         "delayed training needs a stash for every matrix without DPO_SYNC");
        // stash := the current weights, update history := 0: Alg. 1 restarts
        const int rc = launch_init(c, static_cast<cudaStream_t>(stream), 0, 1);
        if (rc != DPO_OK)
            return rc;
        if (mpull(c) != DPO_OK)
            return mfail(c, DPO_ECUDA, "reading the device step counters failed");
        c->phase_k0 = c->k;
        if (c->capturable && mpush(c, static_cast<cudaStream_t>(stream)) != DPO_OK)
            return mfail(c, DPO_ECUDA, "writing the device step counters failed");
    }
    c->hp.delay = delay;
    return DPO_OK;
}

extern "C" int dpo_muon_last_update(const dpo_muon_ctx *c, int i, const void **ptr, int64_t *ld)
{
    if (c == nullptr || ptr == nullptr || ld == nullptr || i < 0 || i >= c->n)
        return DPO_EINVAL;
    *ptr = c->host_mats[i].o;
    *ld = c->host_mats[i].o_ld;
    return DPO_OK;
}

extern "C" int dpo_muon_copy_update(const dpo_muon_ctx *c, int i, void *dst, void *stream)
{
    if (c == nullptr || dst == nullptr || i < 0 || i >= c->n)
        return DPO_EINVAL;
    const DevMat &d = c->host_mats[i];
    if (d.rows * d.cols == 0)
        return DPO_OK;
    const cudaError_t e = cudaMemcpy2DAsync(dst, (size_t)d.cols * 2, d.o, (size_t)d.o_ld * 2,
                                            (size_t)d.cols * 2, (size_t)d.rows,
                                            cudaMemcpyDeviceToDevice,
                                            static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? DPO_OK : DPO_ECUDA;
}

extern "C" int dpo_muon_get_status(dpo_muon_ctx *c, uint32_t *bits)
{
    if (c == nullptr || bits == nullptr)
        return DPO_EINVAL;
    unsigned int v = 0;
    const cudaError_t e = cudaMemcpy(&v, c->d_err, sizeof v, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess)
        return mcuda(c, e, "status read");
    *bits = v;
    return DPO_OK;
}

extern "C" int dpo_muon_clear_status(dpo_muon_ctx *c, void *stream)
{
    if (c == nullptr)
        return DPO_EINVAL;
    const cudaError_t e = cudaMemsetAsync(c->d_err, 0, sizeof(unsigned int),
                                          static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? DPO_OK : mcuda(c, e, "status reset");
}

extern "C" int dpo_muon_test_stall(dpo_muon_ctx *c, int launches)
{
    if (c == nullptr)
        return DPO_EINVAL;
    if (launches < 0)
        return mfail(c, DPO_EINVAL, "launches must be >= 0");
    c->stall_launches = launches;
    return DPO_OK;
}

extern "C" int dpo_muon_test_tiles(const dpo_matrix *mats, int n, int pairs, int ctas, int product,
                                   int64_t *counts)
{
    if (n < 0 || (n > 0 && mats == nullptr) || pairs < 0 || ctas < 0 || (pairs > 0) != (ctas > 0) ||
        product < 0 || product > 2 || counts == nullptr)
        return DPO_EINVAL;
    for (int i = 0; i < n; ++i)
        if (mats[i].rows < 0 || mats[i].cols < 0)
            return DPO_EINVAL;
    if (pairs == 0) {
        int device = 0, sms = 0;
        if (cudaGetDevice(&device) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
            gemm_residency(sms, &pairs, &ctas) != cudaSuccess || pairs < 1 || ctas < 1)
            return DPO_ECUDA;
    }
    const std::vector<Group> groups = group_shapes(mats, n);
    if (pair_tiles(groups) > DPO_MUON_TEST_MAX_TILES)
        return DPO_EINVAL;
    const GemmPlan plan = plan_gemms(mats, groups, pairs, ctas);
    std::fill(counts, counts + 4, 0);
    for (const LaunchSet &ls : plan.sets) {
        const auto &p = ls.prod[product];
        counts[p.cg - 1] += p.tiles;
        counts[3] += p.ew == 4 ? p.tiles : 0;
        for (int64_t t = p.first; t < p.first + p.tiles; ++t)
            counts[2] += (plan.tiles[t].x & (dpo::gemm::kTileHalfM | dpo::gemm::kTileHalfN)) != 0;
    }
    return DPO_OK;
}

extern "C" int dpo_muon_grad_sqnorm(dpo_muon_ctx *c, double *d_sumsq, void *stream)
{
    if (c == nullptr)
        return mfail(nullptr, DPO_EINVAL, "ctx is NULL");
    if (d_sumsq == nullptr || reinterpret_cast<uintptr_t>(d_sumsq) % alignof(double) != 0)
        return mfail(c, DPO_EINVAL, "d_sumsq must be an 8-byte aligned device pointer");
    if (c->total_pkts == 0)
        return DPO_OK;
    const cudaError_t e = launch_grad_norm(c, d_sumsq, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess)
        return mcuda(c, e, "norm launch");
    return DPO_OK;
}

extern "C" int dpo_muon_set_clip_source(dpo_muon_ctx *c, const double *d_sumsq)
{
    if (c == nullptr)
        return mfail(nullptr, DPO_EINVAL, "ctx is NULL");
    if (d_sumsq != nullptr && reinterpret_cast<uintptr_t>(d_sumsq) % alignof(double) != 0)
        return mfail(c, DPO_EINVAL, "d_sumsq must be 8-byte aligned");
    if (d_sumsq != nullptr && !(c->hp.max_grad_norm > 0.0f))
        return mfail(c, DPO_ESTATE, "a clip source needs max_grad_norm > 0");
    c->clip_src = d_sumsq;
    return DPO_OK;
}

extern "C" int dpo_muon_get_phase_start(const dpo_muon_ctx *c, int64_t *k0)
{
    if (c == nullptr || k0 == nullptr)
        return DPO_EINVAL;
    if (mpull(c) != DPO_OK)
        return DPO_ECUDA;
    *k0 = c->phase_k0;
    return DPO_OK;
}

extern "C" int dpo_muon_set_phase_start(dpo_muon_ctx *c, int64_t k0)
{
    if (c == nullptr)
        return DPO_EINVAL;
    if (mpull(c) != DPO_OK)
        return mfail(c, DPO_ECUDA, "reading the device step counters failed");
    if (k0 < 0 || k0 > c->k)
        return mfail(c, DPO_EINVAL, "phase start must lie in [0, k]");
    c->phase_k0 = k0;
    if (c->capturable && (mpush(c, nullptr) != DPO_OK || cudaDeviceSynchronize() != cudaSuccess))
        return mfail(c, DPO_ECUDA, "writing the device step counters failed");
    return DPO_OK;
}

extern "C" int dpo_muon_get_step(const dpo_muon_ctx *c, int64_t *k)
{
    if (c == nullptr || k == nullptr)
        return DPO_EINVAL;
    if (mpull(c) != DPO_OK)
        return DPO_ECUDA;
    *k = c->k;
    return DPO_OK;
}

extern "C" int dpo_muon_set_step(dpo_muon_ctx *c, int64_t k)
{
    if (c == nullptr || k < 0)
        return DPO_EINVAL;
    if (mpull(c) != DPO_OK)
        return mfail(c, DPO_ECUDA, "reading the device step counters failed");
    c->k = k;
    if (c->phase_k0 > k)
        c->phase_k0 = k;
    if (c->capturable && (mpush(c, nullptr) != DPO_OK || cudaDeviceSynchronize() != cudaSuccess))
        return mfail(c, DPO_ECUDA, "writing the device step counters failed");
    return DPO_OK;
}

extern "C" int dpo_muon_flops(const dpo_muon_ctx *c, double *flops)
{
    if (c == nullptr || flops == nullptr)
        return DPO_EINVAL;
    // the updated-state prediction runs the Newton-Schulz chains a second
    // time (delayed training with history buffers)
    const bool twice = c->hp.correction == DPO_CORR_SAPIPE_UPDATED && c->ef && c->hp.delay == 1;
    *flops = twice ? 2.0 * c->flops : c->flops;
    return DPO_OK;
}

extern "C" int dpo_muon_set_timing(dpo_muon_ctx *c, int on)
{
    if (c == nullptr)
        return DPO_EINVAL;
    c->timing = on != 0;
    return DPO_OK;
}

extern "C" int dpo_muon_get_gemm_time(dpo_muon_ctx *c, double *ms, int64_t *launches)
{
    if (c == nullptr || ms == nullptr || launches == nullptr)
        return DPO_EINVAL;
    double total = 0.0;
    for (size_t q = 0; q + 1 < c->ev_used; q += 2) {
        cudaError_t e = cudaEventSynchronize(c->ev_pool[q + 1]);
        float t = 0.0f;
        if (e == cudaSuccess)
            e = cudaEventElapsedTime(&t, c->ev_pool[q], c->ev_pool[q + 1]);
        if (e != cudaSuccess)
            return mcuda(c, e, "timing event read");
        total += t;
    }
    *ms = total;
    *launches = c->gemm_launches;
    c->ev_used = 0;
    c->gemm_launches = 0;
    return DPO_OK;
}

extern "C" int dpo_muon_workspace_bytes(const dpo_muon_ctx *c, int64_t *bytes)
{
    if (c == nullptr || bytes == nullptr)
        return DPO_EINVAL;
    *bytes = c->ws_bytes;
    return DPO_OK;
}

extern "C" void dpo_muon_destroy(dpo_muon_ctx *c)
{
    free_ctx(c);
}
