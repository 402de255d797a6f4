// dpo_gemm.cuh -- batched bf16 GEMM on the sm_103a tensor cores (tcgen05,
// TMA, TMEM) with the epilogues of the Newton-Schulz iteration.
//
//   D[b] = alpha * A[b] B[b]^T + beta * C[b]      (optionally also D[b]^T)
//
// A[b] (M x K) and B[b] (N x K) are row-major bf16 ("K-major" operands), the
// product accumulates in fp32 in tensor memory, and the epilogue rounds once
// to bf16. The Newton-Schulz scratch is padded with zeros to multiples of 256,
// so every tile is whole; K is taken up to the next multiple of 128, and a
// tile whose lower or right half is padding skips that half's work.
//
// A persistent grid of CTA pairs (clusters of 2, one CTA per SM) walks the
// 256 x 256 output tiles with the 2-SM MMA; launches of few tiles take the
// same kernel by single CTAs instead (128 x 128 tiles, the 1-SM MMA, no
// cluster; CG = 1), where "both CTAs" below is the one. In each CTA:
//   warp 0      TMA producer: this CTA's 128 x 128 half of the A block and
//               128 x 128 half of the B block (bf16, 128-byte swizzle, two
//               boxes each) into a 3-stage ring, completing on the leader
//               CTA's mbarrier;
//   warp 1      allocates 512 TMEM columns (two accumulators) together with
//               the peer; in the leader, one lane issues
//               tcgen05.mma.cta_group::2.kind::f16 (M 256, N 256, K 16) eight
//               times per stage, reading both CTAs' halves, and commits each
//               stage and each finished tile to both CTAs;
//   the others  eight warps, or four (EW): epilogue of this CTA's 128 rows:
//               tcgen05.ld 32 lanes x 32 columns at a time, scale, add the
//               addend, round to bf16, stage the 32 x 32 chunk (or its
//               transpose, or both) in shared memory and write it with a
//               TMA store.
// Per CTA a stage is 64 KiB for 8.4 MFLOP, a third less than one SM holding
// a whole 128 x 256 operand pair, so three stages fit and keep the tensor
// pipe fed across the L2 / DRAM round trip.
// Symmetric products (Params::sym; X X^T and c A A + b A): only tiles on or
// above the diagonal block (n0 >= m0) are computed; each of their
// elements (i, j) is also stored at (j, i) when the tile holding (j, i) is
// not computed. Every element is then written exactly once, by one thread,
// and the result does not depend on scheduling.
// Every wait on an mbarrier gives up after kWaitNs, records an error code and
// lets the CTA finish (draining its own TMA loads first), so a fault in the
// pipeline surfaces as a status instead of a hang.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cstdint>

#include "dpo_device.cuh"

namespace dpo {
namespace gemm {

// A CTA pair (a cluster of 2) computes one TM x TN output tile with the
// 2-SM MMA: each CTA holds BM = TM / 2 rows of A and BH = TN / 2 rows of B
// per stage, and its TMEM holds its BM rows of the accumulator. A stage
// spans BK = 128 of K as two TMA boxes of kBoxK = 64 (the 128-byte swizzle
// span); eight MMAs per stage halve the barrier hand-offs per MMA against
// 64-wide stages, which are slower on GB300 at equal ring size (six of them:
// a 7B layer's step 10.1 -> 10.7 ms, four 1B layers 6.5 -> 6.8), and so is a
// barrier for each half of a stage (6.44 -> 6.51).
// kTile(2) is that tile. kTile(1) is the tile of a single CTA (128 x 128, the
// 1-SM MMA, the same stages), for launches of few tiles.
__host__ __device__ constexpr int kTile(int cg) { return 128 * cg; }
constexpr int TM = kTile(2), TN = kTile(2);
constexpr int BM = 128, BH = 128, BK = 128, kBoxK = 64, kStages = 3;
// Epilogue warps, at most: two per TMEM lane quarter, each taking half of the
// tile's columns: a tile's epilogue is a serial chain per warp (TMEM read,
// addend, staging, store), which the 6 k-blocks of a K = 768 tile do not hide at
// four warps. GB300, four against eight warps, whole step: GPT-2 1816 -> 1777 us,
// twelve 768-wide layers 1525 -> 1486, two 256x768 matrices 145 -> 133. Long
// launches with long K run four (kLongBlocks in dpo_muon.cu).
constexpr int kEpiWarps = 8;
__host__ __device__ constexpr int gemm_threads(int ew) { return 64 + 32 * ew; }
constexpr int kABytes = BM * BK * 2;                 // 32 KiB
constexpr int kBBytes = BH * BK * 2;                 // 32 KiB
constexpr int kStageBytes = kABytes + kBBytes;       // 64 KiB per CTA
// Epilogue staging behind the ring: per epilogue warp two buffers of 2 KiB, in
// the 64-byte-swizzled layout the TMA store reads: two 32 x 32 chunks of D in
// turn, or one chunk of D and its transpose.
constexpr int kChunkBytes = 32 * 32 * 2;
constexpr int kEpiBytes = kEpiWarps * 2 * kChunkBytes;      // 32 KiB
// ring + 1024-byte alignment slack + staging
constexpr int kSmemBytes = kStages * kStageBytes + 1024 + kEpiBytes;
constexpr unsigned long long kWaitNs = 1000000000ull;  // 1 s per wait

// Error codes OR-ed into Params::err (kErrWaitDone: an accumulator hand-off).
constexpr unsigned int kErrWaitFull = 1u, kErrWaitEmpty = 2u, kErrWaitDone = 4u,
                       kErrDrain = 8u;

// D is written through the group's store map d (boxes of 32 x 32, 64-byte
// swizzle), D^T through dt.
struct Params {
    const __nv_bfloat16 *c;       // M x N addend, or nullptr
    int64_t ldc, c_bstride;
    float alpha, beta;
    int k_blocks;                 // K / BK
    int sym;                      // D is symmetric (M == N): see ns_gemm_kernel
    int trans;                    // tiles of tall matrices (kTileTall) write D^T (N x M)
                                  // through the map dt: see the epilogue
    int stall;                    // test hook: the MMA lane's first accumulator wait
                                  // targets a phase no arrival completes, so it gives up
    unsigned int *err;
};

__device__ __forceinline__ unsigned long long globaltimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase with the given parity to complete, for at most kWaitNs.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    if (mbar_try(bar, parity))
        return true;
    const unsigned long long t0 = globaltimer();
    while (!mbar_try(bar, parity))
        if (globaltimer() - t0 > kWaitNs)
            return false;
    return true;
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

// TMA tile load into this CTA's shared memory; with CG == 2 the mbarrier (a
// shared::cluster address) may belong to either CTA of the pair.
template <int CG>
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int x, int y,
                                            int z, uint32_t bar_cluster)
{
    if (CG == 2)
        asm volatile(
            "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
            " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
            "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar_cluster)
            : "memory");
    else
        asm volatile(
            "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
            " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
            "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar_cluster)
            : "memory");
}

// TMA store of a 32 x 32 bf16 box from this CTA's shared memory to global
// coordinates (x = column, y = row, z = batch entry), in this thread's bulk
// async-group.
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *map, uint32_t src, int x, int y,
                                             int z)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(x), "r"(y), "r"(z)
                 : "memory");
}

// Byte offset of 16-byte granule g of row r in a tile of 64-byte rows with
// the 64-byte swizzle (granule index XOR bits 1-2 of the row).
__device__ __forceinline__ uint32_t swz64(int r, int g)
{
    return (uint32_t)(r * 64 + ((g ^ ((r >> 1) & 3)) << 4));
}

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// shared::cluster address of the same shared::cta offset in CTA `rank`
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

// One arrival on the leader's mbarrier at this shared::cta offset.
template <int CG> __device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    if (CG == 2)
        asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                         map_to_rank(bar, 0))
                     : "memory");
    else
        asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// All threads of the CTA, or of the pair.
template <int CG> __device__ __forceinline__ void group_sync()
{
    if (CG == 2) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
        __syncthreads();
    }
}

// Shared-memory matrix descriptor of a K-major operand tile stored as rows of
// 64 bf16 (128 bytes) with the 128-byte swizzle, 8-row groups 1024 bytes
// apart (the layout the TMA box above produces): start address, leading
// byte offset 16 (unused by swizzled K-major layouts), stride byte offset
// 1024, descriptor version 1, swizzle mode 2 (128-byte).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(16 >> 4) << 16) |
           ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// Shared-memory descriptor of an MN-major operand tile: rows of 64 bf16
// (128 bytes) along N with the 128-byte swizzle, one row per K index, 8-row
// K groups 1024 bytes apart (stride byte offset), and the second 64-column
// N chunk 8192 bytes further (leading byte offset: one 64-row TMA box).
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(8192 >> 4) << 16) |
           ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// Instruction descriptor of kind::f16: fp32 accumulator, bf16 A and B, A
// K-major, N = M = kTile(cg) (cg 2: the pair's 2-SM shape); B K-major, or
// MN-major with bit 16 (B read as stored row-major along N).
__host__ __device__ constexpr uint32_t idesc_of(int cg, bool bmn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTile(cg) >> 3) << 17) |
           ((uint32_t)(kTile(cg) >> 4) << 24) | (bmn ? 1u << 16 : 0u);
}
// XOR-ed in for N = TN / 2 (a tile whose right half is padding): each CTA of the
// pair then supplies 64 rows of B.
constexpr uint32_t kIdescHalfN = ((uint32_t)(TN >> 3) << 17) ^ ((uint32_t)(TN >> 4) << 17);

// One 16-deep step of a tile, issued by the leader CTA; CG == 2: A rows from
// both CTAs' shared memory at the descriptor's offset, B likewise, the
// accumulator rows in each CTA's TMEM.
template <int CG>
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a_desc, uint64_t b_desc,
                                         uint32_t idesc, uint32_t accumulate)
{
    if (CG == 2)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
            "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate));
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
            "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate));
}

// Arrive on the mbarrier at this shared::cta offset, in both CTAs of a pair,
// once the leader's MMAs issued so far have completed.
template <int CG> __device__ __forceinline__ void mma_commit(uint32_t bar)
{
    if (CG == 2)
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
            " [%0], %1;" ::"r"(bar), "h"((uint16_t)0x3)
            : "memory");
    else
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                     ::"r"(bar) : "memory");
}

// TMEM columns of both accumulators, allocated and freed by one warp (of both
// CTAs of a pair).
template <int CG> __device__ __forceinline__ void tmem_alloc(uint32_t slot)
{
    if (CG == 2) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot),
                     "r"(2 * kTile(CG))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot),
                     "r"(2 * kTile(CG))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
}

template <int CG> __device__ __forceinline__ void tmem_free(uint32_t tmem)
{
    if (CG == 2)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(2 * kTile(CG))
                     : "memory");
    else
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(2 * kTile(CG))
                     : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// The order in which a launch's tiles of one product go out. A full product
// walks bands of kBandRows block rows (all of them, up to 4096 rows), each
// band column by column, so the tiles in flight at once (one per CTA pair)
// share the band's A row blocks and a few B column blocks in L2, and each B
// column block comes from DRAM about once per band. On a 4096 x 11008 operand,
// walking whole block rows instead had the pairs stream all 43 B column blocks
// every round. A symmetric product (sym, m_tiles == n_tiles) enumerates only
// the tiles on or above the diagonal, column by column (column n holds n + 1
// of them), so the pairs' shares of its work differ by at most one tile, and
// the tiles in flight at once read the first block rows of the operand before
// the pairs move on to the last ones.
constexpr int kBandRows = 16;   // block rows per band of a full product's walk (256-row tiles)

struct TileGrid {
    int m_tiles, n_tiles, nb, sym, tile;
    int per_batch() const { return sym ? m_tiles * (m_tiles + 1) / 2 : m_tiles * n_tiles; }
    int count() const { return per_batch() * nb; }
    // fn(batch entry, first row, first column) for every tile in order
    template <class F>
    void walk(F &&fn) const
    {
        for (int b = 0; b < nb; ++b) {
            if (sym) {
                for (int n = 0; n < n_tiles; ++n)
                    for (int m = 0; m <= n; ++m)
                        fn(b, m * tile, n * tile);
            } else {
                for (int first = 0; first < m_tiles; first += kBandRows)
                    for (int n = 0; n < n_tiles; ++n)
                        for (int m = first; m < m_tiles && m < first + kBandRows; ++m)
                            fn(b, m * tile, n * tile);
            }
        }
    }
};

// One launch computes the same product for up to kMaxGroups batches of
// different shapes (the shape groups of a Newton-Schulz step): each group
// has its own operand and output maps and epilogue, and its tiles follow the
// previous group's in the launch's order. Small sets then fill the CTA pairs
// with one launch per product instead of one per shape: five odd shapes take
// 303 us a step on GB300 in one set of launches, 485 us in two (four groups and
// one). Eight groups are 4.8 KB of launch parameters, of the 32 KB there may
// be; against four they cost a launch of one group 15 ns.
constexpr int kMaxGroups = 8;

struct GemmGroup {
    CUtensorMap a, b, d, dt;   // A, B (operands), D and D^T (stores)
    Params p;
};

// The tiles come from a table made at init: x the group and flags, y the batch
// entry, z and w the tile's first row and column. kTileHalfM and kTileHalfN
// mark tiles whose lower or right half lies in the padding of a matrix whose
// size, rounded up to 128, is an odd multiple of 128: their MMAs take half of
// the columns, and the CTA of the pair that holds padding rows loads no A and
// stores nothing. With K rounded up to 128 too, nothing reads what they leave
// unwritten: it stays the zeros of init, which a computed tile would write.
// GB300, without against with the halves and the rounded K, whole step: four
// 384-wide layers 231 -> 207 us, three 640-wide ones 343 -> 329, two 1100-wide
// ones 735 -> 702; where no tile has a padded half it costs up to 1 % (two
// 256x768 matrices 132.0 -> 133.4, GPT-2 1789 -> 1793).
// Each role of the kernel reads its next entry while it works on the current
// one. Deriving them from t in the kernel (a search over the groups, four
// divisions) read the launch's parameters through dependent loads and took every
// role, the MMA lane among them, some 3,900 cycles per tile: a third of a
// K = 768 tile's time.
constexpr int kTileGroup = 0xff, kTileHalfM = 0x100, kTileHalfN = 0x200, kTileTall = 0x400;

struct GemmLaunch {
    GemmGroup g[kMaxGroups];
    const int4 *tiles;
    int n_groups;
    int n_tiles;               // over all groups
};

// 16 bytes of the addend, pinned where it is written, before the wait for the
// accumulator. Through L1, which keeps the other half of each line for the next
// chunk's load: with L1::no_allocate GPT-2's step takes 1766 us against 1750, two
// 256 x 768 matrices 100.9 against 99.9.
__device__ __forceinline__ uint4 load_c(const __nv_bfloat16 *p)
{
    uint4 q;
    asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w)
                 : "l"(p));
    return q;
}

// Entry t of the tile table (made at init), pinned where it is written (a plain
// load may be moved down to its first use, a tile later).
__device__ __forceinline__ int4 load_tile(const int4 *p)
{
    int4 q;
    asm volatile("ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w)
                 : "l"(p));
    return q;
}

// Persistent: the CTA pairs (clusters of 2; with CG = 1, the CTAs) take tiles
// c, c + pairs, ...
// Within a pair, rank 0 (the leader) issues the MMAs; both ranks load their
// halves of A and B and drain their own accumulator rows. Two accumulators
// in TMEM, a tile's width of columns each, let the MMA fill one while the
// epilogues drain the other.
//   full[s]      (leader) both ranks' TMA bytes of stage s have landed
//   empty[s]     (each)   the leader's MMAs have finished reading stage s
//   acc_full[a]  (each)   accumulator a holds a finished tile
//   acc_empty[a] (leader) all epilogue warps of the pair have read it
// EW: epilogue warps, 8 or 4; with 4 each takes both halves of the columns.
// BMN: the B operand is stored N-contiguous (a row-major K x N matrix) and
// loaded as two 64 x 64 boxes per stage, read MN-major by the MMA.
template <bool BMN, int CG, int EW>
__global__ void __cluster_dims__(CG, 1, 1) __launch_bounds__(gemm_threads(EW), 1)
    ns_gemm_kernel(const __grid_constant__ GemmLaunch L)
{
    constexpr int T = kTile(CG);                   // tile side, TMEM columns of an accumulator
    constexpr int kEpiCols = T / 2;                // columns an epilogue warp drains at a time
    unsigned int *const err = L.g[0].p.err;   // err and stall are the launch's
    const int stall = L.g[0].p.stall;
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bars[2 * kStages + 4];
    __shared__ uint32_t tmem_slot;
    __shared__ int aborted;
    __shared__ Params params[kMaxGroups];   // read per tile, by every role

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = CG == 2 ? cluster_rank() : 0u;
    const bool leader = rank == 0;
    const int pair = blockIdx.x / CG, n_pairs = gridDim.x / CG;
    const uint32_t raw = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;   // the swizzle atoms repeat every 1024 B
    const uint32_t sa = ring, sb = ring + kStages * kABytes;
    const uint32_t bar0 = (uint32_t)__cvta_generic_to_shared(bars);
    auto full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
    auto empty = [&](int s) { return bar0 + 8u * (uint32_t)(kStages + s); };
    auto acc_full = [&](int a) { return bar0 + 8u * (uint32_t)(2 * kStages + a); };
    auto acc_empty = [&](int a) { return bar0 + 8u * (uint32_t)(2 * kStages + 2 + a); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(acc_full(a), 1);
            mbar_init(acc_empty(a), CG * EW);   // one arrival per epilogue warp of the pair
        }
        aborted = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if ((int)threadIdx.x >= 64 && (int)threadIdx.x < 64 + L.n_groups)
        params[threadIdx.x - 64] = L.g[threadIdx.x - 64].p;
    if (warp == 1)   // both CTAs of a pair allocate together
        tmem_alloc<CG>((uint32_t)__cvta_generic_to_shared(&tmem_slot));
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    group_sync<CG>();   // barriers of both CTAs initialised before any remote use
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const int n_tiles = L.n_tiles;
    const int4 *const tiles = L.tiles;
    int4 next = {0, 0, 0, 0};   // this pair's next tile (constant table: read before the wait)
    if (pair < n_tiles)
        next = load_tile(tiles + pair);
    pdl_wait();

    if (warp == 0) {
        if (lane == 0) {
            for (int gi = 0; gi < L.n_groups; ++gi) {
                asm volatile("prefetch.tensormap [%0];"
                             ::"l"(reinterpret_cast<uint64_t>(&L.g[gi].a)) : "memory");
                asm volatile("prefetch.tensormap [%0];"
                             ::"l"(reinterpret_cast<uint64_t>(&L.g[gi].b)) : "memory");
            }
            int it = 0;   // k-blocks issued by this CTA
            for (int t = pair; t < n_tiles && !*(volatile int *)&aborted; t += n_pairs) {
                const int gi = next.x & kTileGroup, b = next.y, m0 = next.z, n0 = next.w;
                const bool half_m = CG == 2 && (next.x & kTileHalfM);
                const bool half_n = CG == 2 && (next.x & kTileHalfN);
                if (t + n_pairs < n_tiles)
                    next = load_tile(tiles + t + n_pairs);
                // both CTAs' bytes of a stage: A of the rows that are not all
                // padding; of a half-wide MN-major B one box of 64 columns, of
                // a K-major one the box of 128 rows of which 64 are used
                const uint32_t bytes =
                    CG == 1 ? (uint32_t)kStageBytes
                            : (uint32_t)((half_m ? 1 : 2) * kABytes +
                                         (BMN && half_n ? 1 : 2) * kBBytes);
                const bool load_a = leader || !half_m;
                const CUtensorMap *tma_a = &L.g[gi].a, *tma_b = &L.g[gi].b;
                const int kb_n = params[gi].k_blocks;
                const int ma = m0 + (int)rank * BM, nb_ = n0 + (int)rank * (half_n ? BH / 2 : BH);
                for (int kb = 0; kb < kb_n; ++kb, ++it) {
                    const int s = it % kStages;
                    const uint32_t ph = (uint32_t)(it / kStages) & 1u;
                    if (!mbar_wait(empty(s), ph ^ 1u) || *(volatile int *)&aborted) {
                        atomicOr(err, kErrWaitEmpty);
                        aborted = 1;
                        break;
                    }
                    const uint32_t fbar = CG == 2 ? map_to_rank(full(s), 0) : full(s);
                    if (leader)   // the leader's barrier counts both CTAs' bytes
                        mbar_arrive_expect_tx(full(s), bytes);
#pragma unroll
                    for (int h = 0; h < BK / kBoxK; ++h) {   // the two 64-wide K halves
                        const int k0 = kb * BK + h * kBoxK;
                        const uint32_t ah = sa + (uint32_t)(s * kABytes + h * (kABytes / 2));
                        const uint32_t bh = sb + (uint32_t)(s * kBBytes + h * (kBBytes / 2));
                        if (load_a)
                            tma_load_3d<CG>(ah, tma_a, k0, ma, b, fbar);
                        if (BMN) {   // two 64 x 64 boxes: N columns nb_.. and nb_ + 64..
                            tma_load_3d<CG>(bh, tma_b, nb_, k0, b, fbar);
                            if (!half_n)
                                tma_load_3d<CG>(bh + (uint32_t)(kBBytes / 4), tma_b, nb_ + 64, k0,
                                                b, fbar);
                        } else {
                            tma_load_3d<CG>(bh, tma_b, k0, nb_, b, fbar);
                        }
                    }
                }
            }
            // Drain (leader): every stage issued by either CTA has landed
            // before the pair leaves (the peer waits at the final cluster
            // barrier for this).
            if (leader)
                for (int q = it - kStages < 0 ? 0 : it - kStages; q < it; ++q)
                    if (!mbar_wait(full(q % kStages), (uint32_t)(q / kStages) & 1u))
                        atomicOr(err, kErrDrain);
        }
    } else if (warp == 1) {
        if (lane == 0 && leader) {
            int it = 0, lt = 0;   // k-blocks consumed, tiles accumulated
            for (int t = pair; t < n_tiles && !*(volatile int *)&aborted; t += n_pairs) {
                const int kb_n = params[next.x & kTileGroup].k_blocks;
                const uint32_t idesc =
                    idesc_of(CG, BMN) ^ (CG == 2 && (next.x & kTileHalfN) ? kIdescHalfN : 0u);
                if (t + n_pairs < n_tiles)
                    next = load_tile(tiles + t + n_pairs);
                const int a = lt & 1;
                const uint32_t aph = (uint32_t)(lt >> 1) & 1u;
                if (!mbar_wait(acc_empty(a), stall && lt == 0 ? aph : aph ^ 1u)) {
                    atomicOr(err, kErrWaitDone);
                    aborted = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d = tmem + (uint32_t)(a * T);
                bool ok = true;
                for (int kb = 0; kb < kb_n; ++kb, ++it) {
                    const int s = it % kStages;
                    const uint32_t ph = (uint32_t)(it / kStages) & 1u;
                    if (!mbar_wait(full(s), ph) || *(volatile int *)&aborted) {
                        atomicOr(err, kErrWaitFull);
                        aborted = 1;
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        const int h = k / (kBoxK / 16), kk = k % (kBoxK / 16);
                        const uint32_t ah = sa + (uint32_t)(s * kABytes + h * (kABytes / 2));
                        const uint32_t bh = sb + (uint32_t)(s * kBBytes + h * (kBBytes / 2));
                        const uint64_t ad = smem_desc(ah + (uint32_t)(kk * 32));
                        const uint64_t bd = BMN ? smem_desc_mn(bh + (uint32_t)(kk * 16 * 128))
                                                : smem_desc(bh + (uint32_t)(kk * 32));
                        mma_bf16<CG>(d, ad, bd, idesc, (kb | k) != 0 ? 1u : 0u);
                    }
                    mma_commit<CG>(empty(s));
                }
                mma_commit<CG>(acc_full(a));   // when this tile's MMAs have completed
                ++lt;
                if (!ok) {
                    // the MMAs issued for this tile finish before the pair
                    // leaves and its TMEM is released
                    if (!mbar_wait(acc_full(a), aph))
                        atomicOr(err, kErrDrain);
                    break;
                }
            }
        }
    } else {
        // Epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31 = this CTA's
        // tile rows m0 + BM rank + 32 (w % 4) + lane, and the half of the tile's
        // columns that (w - 2) / 4 names (of four warps: both halves in turn).
        // Each 32 x 32 chunk is staged in
        // shared memory (and its transpose, for a mirrored or a transposed
        // output) and written by one TMA store per box from lane 0; direct
        // stores from 32 rows at a time cost the MMAs a fifth of their rate
        // on GB300. Lane 0 waits until the buffers it is about to rewrite have
        // been read.
        const int q = warp & 3, half0 = (warp - 2) >> 2;
        const uint32_t wbuf =
            ring + (uint32_t)(kStages * kStageBytes + (warp - 2) * 2 * kChunkBytes);
        // The addend C (c A A + b A, B X + a X) of all the warp's chunks is
        // read before the accumulator is ready, coalesced: lane l loads
        // granule l % 4 (8 columns) of rows l / 4 + 8 i of the warp's 32 x 32
        // chunk, 8 rows of 64 bytes per instruction; the chunk is then turned
        // through its staging buffer so that each lane holds its own row. C is
        // never the launch's output.
        constexpr int kChunks = kEpiCols / 32;
        const int crs = lane >> 2, cg = lane & 3;   // coalesced load: sub-row, granule
        int lt = 0;
        for (int t = pair; t < n_tiles; t += n_pairs) {
            const int flags = next.x, gi = flags & kTileGroup, b = next.y, m0 = next.z;
            const int tile_n0 = next.w;
            if (t + n_pairs < n_tiles)
                next = load_tile(tiles + t + n_pairs);
            const GemmGroup &G = L.g[gi];
            const Params p = params[gi];   // in registers: the asm statements below clobber memory
            // D^T instead of D: half the stores of the last product, GPT-2's
            // step 1769 -> 1748 us.  Single CTAs run the few-tile launches, whose
            // time is the epilogue's length and not its bytes; there the test
            // costs more than the stores (two 256 x 512 matrices 97.2 -> 98.3 us),
            // and every tile writes both.
            const bool only_t = CG == 2 && p.trans != 0 && (flags & kTileTall);
            const bool both = p.trans != 0 && CG == 1;
            const int a = lt & 1;
            const int row0 = m0 + (int)rank * BM + q * 32;
            bool seen = true;
#pragma unroll
            for (int h = 0; h < kEpiWarps / EW; ++h) {
                const int half = half0 + h, n0 = tile_n0 + half * kEpiCols;
                // these rows or columns are all padding: the warp only passes
                // the accumulator on
                const bool idle = CG == 2 && ((flags & kTileHalfM && !leader) ||
                                              (flags & kTileHalfN && half));
                uint4 cpre[kChunks][4];
                if (p.c != nullptr && !idle) {
                    // C at (row0 + crs, n0 + 8 cg); rows 8 i further for i = 0..3
                    const __nv_bfloat16 *crow = p.c + (int64_t)b * p.c_bstride +
                                                (int64_t)(row0 + crs) * p.ldc + n0 + cg * 8;
#pragma unroll
                    for (int c = 0; c < kChunks; ++c)
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            cpre[c][i] = load_c(crow + 8 * i * p.ldc + c * 32);
                }
                if (h == 0) {
                    seen = mbar_wait(acc_full(a), (uint32_t)(lt >> 1) & 1u);
                    if (!seen)
                        atomicOr(err, kErrWaitDone);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    // tcgen05.ld is warp-collective: the whole warp goes on, or
                    // none of it.
                    seen = __all_sync(0xFFFFFFFFu, seen && !*(volatile int *)&aborted);
                }
                if (!seen)
                    break;
                const uint32_t acc =
                    tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * T + half * kEpiCols);
                if (!idle)
#pragma unroll
                for (int ch = 0; ch < kChunks; ++ch) {
                    uint32_t r[32];
                    tmem_ld32(acc + (uint32_t)(ch * 32), r);
                    float v[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        v[j] = p.alpha * __uint_as_float(r[j]);
                    const int col0 = n0 + ch * 32;
                    // Mirror of a symmetric product: (col, row) lies in the tile
                    // (col / T, row / T), not computed when row / T < col / T.
                    // Uniform over the warp (its rows share row / T) and the chunk
                    // (its columns share col / T).
                    const bool mirror = p.sym && row0 / T < col0 / T;
                    const bool trans = mirror || only_t || both;
                    // Without transposes the two buffers alternate, and only the
                    // chunk before the last one must have been read; a tile's
                    // first chunk may follow one with a transpose.
                    const uint32_t rb = wbuf + (trans ? 0u : (uint32_t)((ch & 1) * kChunkBytes));
                    const uint32_t tb = wbuf + (uint32_t)kChunkBytes;
                    if (lane == 0) {
                        if (trans || ch == 0)
                            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        else
                            asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    }
                    __syncwarp();
                    if (p.c != nullptr) {
                        // the coalesced chunk of C into rb, then this lane's row out
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint4 cv = cpre[ch][i];
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                                         ::"r"(rb + swz64(crs + 8 * i, cg)), "r"(cv.x), "r"(cv.y),
                                           "r"(cv.z), "r"(cv.w)
                                         : "memory");
                        }
                        __syncwarp();
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            uint4 cv;
                            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                         : "=r"(cv.x), "=r"(cv.y), "=r"(cv.z), "=r"(cv.w)
                                         : "r"(rb + swz64(lane, g))
                                         : "memory");
                            const __nv_bfloat162 *c2 = reinterpret_cast<const __nv_bfloat162 *>(&cv);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float2 f = __bfloat1622float2(c2[e]);
                                v[g * 8 + 2 * e] = fmaf(p.beta, f.x, v[g * 8 + 2 * e]);
                                v[g * 8 + 2 * e + 1] = fmaf(p.beta, f.y, v[g * 8 + 2 * e + 1]);
                            }
                        }
                        // each lane rewrites only the row it has read
                    }
                    if (!only_t) {
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            const uint32_t w0 = pack_bf16(v[g * 8 + 0], v[g * 8 + 1]);
                            const uint32_t w1 = pack_bf16(v[g * 8 + 2], v[g * 8 + 3]);
                            const uint32_t w2 = pack_bf16(v[g * 8 + 4], v[g * 8 + 5]);
                            const uint32_t w3 = pack_bf16(v[g * 8 + 6], v[g * 8 + 7]);
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                                         ::"r"(rb + swz64(lane, g)), "r"(w0), "r"(w1), "r"(w2), "r"(w3)
                                         : "memory");
                        }
                    }
                    if (trans) {   // element (row, col0 + j) at row j, column lane of the transpose
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const __nv_bfloat16 h = __float2bfloat16_rn(v[j]);
                            asm volatile("st.shared.b16 [%0], %1;" ::"r"(tb + swz64(j, lane >> 3) +
                                                                          (uint32_t)((lane & 7) * 2)),
                                         "h"(*reinterpret_cast<const uint16_t *>(&h))
                                         : "memory");
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        if (!only_t)
                            tma_store_3d(&G.d, rb, col0, row0, b);
                        if (trans)
                            tma_store_3d(mirror ? &G.d : &G.dt, tb, row0, col0, b);
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
            }
            if (!seen)
                break;
            // this warp's rows of the accumulator are read: release them to
            // the leader's MMA lane
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0)
                mbar_arrive<CG>(acc_empty(a));
            ++lt;
        }
        if (lane == 0)   // every store has been written before the CTA ends
            asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    __syncthreads();
    if (CG == 2)
        group_sync<CG>();   // no CTA leaves while its peer may still read its shared memory
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_free<CG>(tmem);
    }
}

}  // namespace gemm
}  // namespace dpo
