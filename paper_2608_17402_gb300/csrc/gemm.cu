// gemm.cu -- persistent grouped GEMM on tcgen05 / TMEM with 2-SM MMAs, for the
// MoE-ViE layer (App. B, Algorithm 1, Kernels 1 and 2; also the router logits),
// sm_103a.
//
// One launch computes, for every group g (an expert) and every row r of its
// segment:   D[r, :] = A[row(r), :] . B[g]   (bf16 inputs, fp32 accumulation)
// and hands each tile to a fused epilogue:
//   EPI_GELU_BF16   hidden = bf16(GELU(D))                      (Kernel 1, GELU)
//   EPI_STORE_BF16  out    = bf16(D)
//   EPI_ADD_F32     y[tok(r)] += gate(r) * D   (Kernel 2: routing weight + scatter-add)
//   EPI_STORE_F32   y[tok(r)]  = scale * D     (first writer of y; router logits)
//
// CTA pairs.  The grid is made of clusters of two CTAs on neighbouring SMs.  A
// pair computes a 256 x BN tile with tcgen05.mma.cta_group::2 (M = 256): CTA r
// holds rows 128 r .. 128 r + 127 of A and columns r BN/2 .. (r+1) BN/2 - 1 of B
// in its shared memory, and receives rows 128 r .. of D in its TMEM.  Per SM this
// halves the B traffic of a 128 x BN tile, so shared memory bandwidth (the MMA
// reads what TMA writes) no longer caps the tensor pipe.  CTA 0 of the pair (the
// leader) issues every MMA; its commits arrive on the barriers of both CTAs.
//
// Work items are (256-row m-tile, n-tile) pairs in group-major order with the
// n-tile fastest; a persistent pair walks them with a static stride.  The m-tiles
// come from a device tile table {group, first row, rows <= 256} written by the
// permute step (no host read of segment sizes), or, for one dense group, from
// arithmetic.
//
// Warp roles (608 threads per CTA, one CTA per SM):
//   warps 0-7   epilogue: tcgen05.ld of the CTA's 128 accumulator rows (warp w: TMEM lanes
//               32 (w%4)..+31, every other 32-column chunk), fused math, and stores or
//               reductions of whole sectors through a buffer per warp.  (The transposed
//               product, epilogue_addt: with warps 10-17, straight from registers.)
//   warp 8      TMEM allocation (both CTAs, jointly); the leader's issues the MMAs (the
//               issuing roles run as whole warps, one elected lane issues)
//   warp 9      TMA loads of the B half and, for contiguous A rows, of A; the leader
//               posts the byte count of both CTAs on its full barrier.  With contiguous A
//               warp 18 takes turns with it, stage by stage
//   warps 10-17 token gather: 16-byte cp.async of A rows straight into the 128-byte
//               swizzled K-major layout; each thread hands the completion of its
//               copies to the stage's local afull barrier and moves on
//   warp 18     waits for afull, fences the stage to the async proxy and
//               publishes it on the leader's full barrier (from the peer: a 16-byte
//               bulk copy that completes transaction bytes there)
// Shared memory: 6 stages and an epilogue buffer (5 for the activation-derivative
// epilogue) x (A 128x64 + B 64x128) bf16; TMEM: two fp32 accumulators
// of 256 columns, so the epilogue of one tile overlaps the main loop of the next.
//
// Operand layouts (tcgen05 shared-memory descriptors, 128-byte swizzle):
//   A  K-major : row r of the 128x64 tile at byte r*128, 16-byte chunk c stored
//                at chunk c ^ (r % 8); 8-row groups 1024 B apart (SBO = 1024).
//                The k-th 16-wide K slice starts 32*k bytes into the tile.
//   B  MN-major: TMA box {64 (N), 64 (K)}: K row j at byte j*128 (swizzled), the
//                next 64 columns of N 8192 B further (LBO = 8192), 8-row K groups
//                1024 B apart (SBO = 1024).  The k-th K slice starts 2048*k bytes in.
#include <cudaTypedefs.h>
#include <math.h>

#include "internal.h"

namespace mv {

namespace {


// ------------------------------------------------------------ pair helpers

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Address of the same shared-memory object in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                     : "memory");
}
// 16-byte async-proxy copy from this CTA's shared memory to `dst_cluster` (shared
// memory of a CTA of the cluster) that completes 16 transaction bytes on the
// barrier `bar_cluster` of that CTA.
__device__ __forceinline__ void bulk_signal_remote(uint32_t dst_cluster, uint32_t src,
                                                   uint32_t bar_cluster) {
    asm volatile(
        "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], 16, [%2];" ::
            "r"(dst_cluster), "r"(src), "r"(bar_cluster)
        : "memory");
}
// Arrival on a barrier of another CTA of the cluster, with the default (CTA-scope)
// release: used where the arriving thread has nothing to publish but completed
// tcgen05.ld reads (ordered by tcgen05 fences around the barrier), so no
// cluster-wide release of its earlier stores is needed.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar_cluster) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}
// TMA loads into this CTA's shared memory that complete on a barrier of either CTA
// of the pair.
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* tm,
                                                 uint32_t bar_cluster, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(tm), "r"(c0), "r"(c1), "r"(c2), "r"(bar_cluster)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm,
                                                 uint32_t bar_cluster, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(tm), "r"(c0), "r"(c1), "r"(bar_cluster)
        : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                                 uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive once on the barrier at shared offset `bar` of both CTAs when all prior
// tcgen05 operations of this thread have completed.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
        " [%0], %1;" ::"r"(bar),
        "h"((uint16_t)3)
        : "memory");
}

// ------------------------------------------------------------------ tiles

struct Tile {
    int g, row0, nrows, n0;
    int kb0, kb1;   // k-blocks [kb0, kb1) of this item's split of K
    int ks;         // split index
    int m0;         // weight-gradient items: first row of the output tile within its group
    int store;      // weight-gradient items: the only item of its output tile (store, not add)
};

// A work item's table entry, loaded but not yet checked.  The roles that walk the
// items load the entry of an item one item ahead (tile_load) and check it when the
// item starts (tile_finish), so that no role waits on that load at an item boundary.
struct TileLd {
    int4 d;   // table entry (unused for one dense group)
    int ks;   // split of K
    int q;    // item index without the split: table entry (item table) or m-tile x n-tile
};

// Work-item counts stay far below 2^31 (m-tiles x n-tiles x K splits), so item indices
// are split with 32-bit arithmetic, each division done once.
__device__ __forceinline__ TileLd tile_load(const GemmArgs& p, int64_t w64) {
    TileLd l;
    const int w = (int)w64;
    l.q = w;
    l.ks = 0;
    if (p.ksplit > 1) {   // split of K fastest
        l.q = w / p.ksplit;
        l.ks = w - l.q * p.ksplit;
    }
    if (p.item_table) l.d = __ldg(p.tiles + l.q);
    else if (p.tiles) l.d = __ldg(p.tiles + l.q / p.n_ntiles);
    else l.d = make_int4(0, 0, 0, 0);
    return l;
}

// k-blocks [kb0, kb1) of split ks of K.
__device__ __forceinline__ void tile_kb(const GemmArgs& p, int ks, int& kb0, int& kb1) {
    kb0 = (int)((int64_t)ks * p.num_kb / p.ksplit);
    kb1 = (int)((int64_t)(ks + 1) * p.num_kb / p.ksplit);
}

__device__ __forceinline__ Tile tile_finish(const GemmArgs& p, const TileLd& l) {
    Tile t;
    t.ks = l.ks;
    t.m0 = 0;
    t.store = 0;
    if (p.item_table == 2) {   // a weight-gradient item {g, m0 | n0 << 16, kb0, kb1 (| store bit)}
        t.g = l.d.x;
        t.m0 = l.d.y & 0xffff;
        t.n0 = (int)((uint32_t)l.d.y >> 16);
        t.kb0 = l.d.z;
        t.kb1 = l.d.w & (BWD_STORE_BIT - 1);
        t.store = (l.d.w & BWD_STORE_BIT) ? 1 : 0;
        t.row0 = t.g * p.wg_M + t.m0;
        t.nrows = min(GM_BM, p.wg_M - t.m0);
        if (t.g < 0 || t.g >= p.G || t.m0 >= p.wg_M || t.n0 >= p.N || t.kb0 < 0 || t.kb1 <= t.kb0 ||
            (int64_t)t.row0 + t.nrows > p.m_total) {
            report(p.status, MOEVIE_ERR_DEVICE, SITE_GEMM_TILES, t.g, t.kb0);
            t.nrows = 0;
            t.g = 0;
            t.n0 = 0;
            t.kb1 = t.kb0 = 0;
        }
        return t;
    }
    tile_kb(p, l.ks, t.kb0, t.kb1);
    if (p.item_table) {   // an explicit (m-tile, n-tile) item
        t.g = l.d.x;
        t.row0 = l.d.y;
        t.nrows = l.d.z;
        t.n0 = l.d.w;
        if (t.nrows < 0 || t.nrows > GM_BM || t.g < 0 || t.g >= p.G || t.n0 < 0 || t.n0 >= p.N ||
            (int64_t)t.row0 + t.nrows > p.m_total) {
            report(p.status, MOEVIE_ERR_DEVICE, SITE_GEMM_TILES, t.row0, t.nrows);
            t.nrows = 0;
            t.g = 0;
            t.n0 = 0;
        }
        return t;
    }
    const int mt = l.q / p.n_ntiles;
    const int nt = l.q - mt * p.n_ntiles;
    if (p.tiles) {
        t.g = l.d.x;
        t.row0 = l.d.y;
        t.nrows = l.d.z;
    } else {   // one dense group of m_total rows
        t.g = 0;
        t.row0 = mt * GM_BM;
        const int64_t left = p.m_total - t.row0;
        t.nrows = (int)(left < GM_BM ? left : GM_BM);
    }
    if (t.nrows < 0 || t.nrows > GM_BM || t.g < 0 || t.g >= p.G ||
        (int64_t)t.row0 + t.nrows > p.m_total) {
        report(p.status, MOEVIE_ERR_DEVICE, SITE_GEMM_TILES, t.row0, t.nrows);
        t.nrows = 0;
        t.g = 0;
    }
    t.n0 = nt * p.n_step;
    return t;
}

__device__ __forceinline__ Tile decode_tile(const GemmArgs& p, int64_t w) {
    return tile_finish(p, tile_load(p, w));
}

// GELU(u) = u/2 (1 + erf(u / sqrt 2)) = max(u, 0) - |u|/2 erfc(|u| / sqrt 2), the
// second form free of the cancellation of 1 + erf for u < 0.  erfc from Abramowitz &
// Stegun 7.1.28: erfc(z) = (1 + a1 z + a2 z^2 + ... + a6 z^6)^-16 for z >= 0, with
// |error| <= 3e-7 (one reciprocal and no exponential; the sixteenth power by four
// squarings, which overflow to +inf, and so to erfc = 0, only where erfc is far
// below fp32 resolution).  Evaluated in fp32 the GELU error stays below 1e-6 in
// absolute value; the hidden activation is then rounded to bf16 (2^-9 relative).
// Two values at a time with the packed fp32x2 instructions.
__device__ __forceinline__ void erfc_as2(float a0, float a1, float& q0, float& q1) {   // a0, a1 >= 0
    const uint64_t z = f2_mul(f2_pack(a0, a1), f2_pack(0.70710678118654752f, 0.70710678118654752f));
    uint64_t P = f2_fma(z, f2_pack(0.0000430638f, 0.0000430638f), f2_pack(0.0002765672f, 0.0002765672f));
    P = f2_fma(P, z, f2_pack(0.0001520143f, 0.0001520143f));
    P = f2_fma(P, z, f2_pack(0.0092705272f, 0.0092705272f));
    P = f2_fma(P, z, f2_pack(0.0422820123f, 0.0422820123f));
    P = f2_fma(P, z, f2_pack(0.0705230784f, 0.0705230784f));
    P = f2_fma(P, z, f2_pack(1.0f, 1.0f));
    P = f2_mul(P, P);
    P = f2_mul(P, P);
    P = f2_mul(P, P);
    P = f2_mul(P, P);
    float p0, p1;
    f2_unpack(P, p0, p1);
    q0 = rcp_approx(p0);
    q1 = rcp_approx(p1);
}

__device__ __forceinline__ void gelu_erf2(float& u0, float& u1) {
    float q0, q1;
    erfc_as2(fabsf(u0), fabsf(u1), q0, q1);
    const uint64_t r = f2_fma(f2_mul(f2_pack(fabsf(u0), fabsf(u1)), f2_pack(-0.5f, -0.5f)), f2_pack(q0, q1),
                              f2_pack(fmaxf(u0, 0.0f), fmaxf(u1, 0.0f)));
    f2_unpack(r, u0, u1);
}

// GELU'(u) = Phi(u) + u phi(u) (the derivative of the erf form) of two values, for the
// training path: Phi(u) = erfc(-u / sqrt 2) / 2 from the erfc above (1 - q / 2 for
// u >= 0, q / 2 below), phi(u) = exp(-u^2 / 2) / sqrt(2 pi) with CUDA's __expf.
// Absolute error below 1e-6.
__device__ __forceinline__ void gelu_grad2(float& u0, float& u1) {
    float q0, q1;
    erfc_as2(fabsf(u0), fabsf(u1), q0, q1);
    const float c0 = u0 >= 0.0f ? 1.0f - 0.5f * q0 : 0.5f * q0;
    const float c1 = u1 >= 0.0f ? 1.0f - 0.5f * q1 : 0.5f * q1;
    u0 = fmaf(u0, 0.3989422804014327f * __expf(-0.5f * u0 * u0), c0);
    u1 = fmaf(u1, 0.3989422804014327f * __expf(-0.5f * u1 * u1), c1);
}

struct Smem {
    uint32_t a0, b0;          // shared addresses of stage 0
    uint32_t full, empty;     // barrier arrays (8 bytes apart)
    uint32_t afull;           // peer CTA: its gather warps' copies of a stage have landed
    uint32_t tfull, tempty;
    uint32_t drain;
    uint32_t sink;            // 16 bytes: target / source of the peer's stage signals
    int nstages;              // operand ring depth of this launch
    float* stg;               // the epilogue's buffers (gm_stg_bytes)
    uint32_t rank;            // rank of this CTA in its pair
    int64_t pair, npairs;     // pair index and count
};

__device__ __forceinline__ void set_abort(volatile int* flag, DevStatus* st, int site, int a,
                                          int b) {
    *flag = 1;
    report(st, MOEVIE_ERR_TIMEOUT, site, a, b);
}

// Rows of tile t held by this CTA: 128 rank .. 128 rank + rows_half(t) - 1.
__device__ __forceinline__ int rows_half(const Tile& t, uint32_t rank) {
    const int r = t.nrows - (int)rank * GM_HALF;
    return r < 0 ? 0 : (r > GM_HALF ? GM_HALF : r);
}

// N of a transposed tile's MMAs: its rows rounded up to 64 (32 per CTA's half of B).
__device__ __forceinline__ int trans_n(const Tile& t) { return t.nrows > 64 ? (t.nrows + 63) / 64 * 64 : 64; }

// --------------------------------------------------------------- producers

// TMA producers (all lanes of a warp in step, one elected lane issues): the CTA's half of
// B, and A when its rows are contiguous.  `np` warps take the stages in turn, warp `pid`
// every np-th one.  The byte-count arrival, the copies and the wait of one stage are a chain
// of about 725 cycles in one warp (clock sums in the kernel), longer than the 512 cycles of
// the stage's MMAs: two producers took the down-projection at T = 8192, d = 1280, h = 854
// from 141 to 137 us.  With gathered A a second producer slowed small launches; the one there
// issues two stages at once when both are free (up-projection of that layer 203 -> 199 us).
// The leader posts the byte count of both CTAs on its full barrier.
template <bool GATHER, bool TRAIN, bool ONE, bool TRANS, int NP>
__device__ void producer_tma(const GemmArgs& p, const Smem& sm, int64_t n_work, int pid,
                             volatile int* abort_flag) {
    tma_prefetch_desc(&p.tmB);
    if (p.g_split < p.G || p.swiglu) tma_prefetch_desc(&p.tmB2);
    if (p.g_split < p.G && p.swiglu) {
        tma_prefetch_desc(&p.tmB3);
        tma_prefetch_desc(&p.tmB4);
    }
    if (!GATHER) tma_prefetch_desc(&p.tmA);
    if (TRANS) tma_prefetch_desc(&p.tmA2);
    const uint32_t half_n = (uint32_t)p.BN / 2;
    const uint32_t nboxh = (half_n + 63) / 64;
    // B per CTA and stage: nboxh boxes of 64 columns x 64 K rows (N-major), or half_n rows
    // of 64 K values (K-major)
    const uint32_t b_bytes = (TRAIN && p.b_kmajor) ? half_n * 128u : nboxh * GM_BK * 128;
    const uint32_t cta_bytes = b_bytes + (GATHER ? 0u : (uint32_t)GM_A_BYTES);
    // gathering: plus the 16-byte signal with which the peer publishes its A half
    const uint32_t stage_tx = 2 * cta_bytes + (GATHER ? 16u : 0u);
    const uint32_t full_leader = peer_addr(sm.full, 0);
    int s = 0, turn = 0;
    uint32_t ph = 0;
    bool ready = false;
    int64_t w = sm.pair;
    if (w >= n_work) return;
    Tile t = decode_tile(p, w);
    for (; w < n_work; w += sm.npairs) {
        const int64_t wn = w + sm.npairs;
        // checked after this item's loads (loaded whether there is a next item or not: a
        // conditional load would be waited for here, where its two values merge)
        const TileLd nl = tile_load(p, wn < n_work ? wn : w);
        // B of this group: groups >= g_split from their own map; with swiglu the second
        // CTA of the pair loads the up projection (W3) beside the gate's (W1) columns
        const bool tail = t.g >= p.g_split;
        const CUtensorMap* tmb = tail ? &p.tmB2 : &p.tmB;
        if (p.swiglu)
            tmb = sm.rank == 1 ? (tail ? &p.tmB4 : &p.tmB2) : (tail ? &p.tmB3 : &p.tmB);
        const int gb = (TRAIN && p.item_table == 2) ? 0 : (tail ? t.g - p.g_split : t.g);
        const int ncol0 = p.swiglu ? t.n0 : t.n0 + (int)(sm.rank * (TRANS ? (uint32_t)GM_HALF : half_n));
        const int rhalf = TRANS ? trans_n(t) / 2 : 0;   // rows of the CTA's half of the transposed B
        const int row = t.row0 + (int)sm.rank * (TRANS ? rhalf : GM_HALF);
        auto issue = [&](int st, int kb) {   // one lane: the byte count and the copies of k-block kb into stage st
            const uint32_t bar = full_leader + 8 * st;
            const uint32_t a_dst = sm.a0 + st * GM_A_BYTES, b_dst = sm.b0 + st * GM_B_BYTES;
            const int kk = kb * GM_BK;
            if (TRANS) {
                if (sm.rank == 0)
                    mbar_arrive_expect_tx(sm.full + 8 * st, 2u * (uint32_t)(GM_A_BYTES + rhalf * 128));
                if (TRAIN && p.b_kmajor) {   // 128 output columns' rows of 64 K values
                    tma_load_3d_pair(a_dst, tmb, bar, kk, ncol0, gb);
                } else {                     // two boxes of 64 columns x 64 K rows
                    tma_load_3d_pair(a_dst, tmb, bar, ncol0, kk, gb);
                    tma_load_3d_pair(a_dst + GM_BK * 128, tmb, bar, ncol0 + 64, kk, gb);
                }
                if (rhalf == GM_HALF) {
                    tma_load_2d_pair(b_dst, &p.tmA2, bar, kk, row);
                } else {
                    for (int j = 0; j < rhalf; j += GM_ROW_BOX)
                        tma_load_2d_pair(b_dst + j * 128, &p.tmA, bar, kk, row + j);
                }
                return;
            }
            if (sm.rank == 0) mbar_arrive_expect_tx(sm.full + 8 * st, stage_tx);
            if (TRAIN && p.b_kmajor) {   // half_n rows of the CTA's columns, 64 K values each
                tma_load_3d_pair(b_dst, tmb, bar, kk, ncol0, gb);
            } else {
                for (uint32_t j = 0; j < nboxh; ++j)
                    tma_load_3d_pair(b_dst + j * (GM_BK * 128), tmb, bar, ncol0 + (int)(64 * j), kk, gb);
            }
            if (GATHER) return;
            if (TRAIN && p.a_mn) {   // two 64-row halves of the CTA's 128 output rows, 64 K rows each
                const int m = t.m0 + (int)sm.rank * GM_HALF;
                tma_load_3d_pair(a_dst, &p.tmA, bar, m, kk, 0);
                tma_load_3d_pair(a_dst + GM_BK * 128, &p.tmA, bar, m + 64, kk, 0);
            } else {
                const int col = p.a_kperiod ? kk % p.a_kperiod : kk;
                tma_load_2d_pair(a_dst, &p.tmA, bar, col, row);
            }
        };
        for (int kb = t.kb0; kb < t.kb1; ++kb) {
            if (NP == 1 || turn == pid) {
                if (!mbar_wait_warp<ONE>(sm.empty + 8 * s, ph ^ 1u, p.limit_ns, abort_flag, ready)) {
                    set_abort(abort_flag, p.status, SITE_GEMM_WAIT_EMPTY, (int)sm.pair, 1);
                    return;
                }
                // the next stage with this one when it is free already
                const int s2 = s + 1 == sm.nstages ? 0 : s + 1;
                const bool two = NP == 1 && !ONE && kb + 1 < t.kb1 &&
                                 __all_sync(0xffffffffu, mbar_test(sm.empty + 8 * s2, (s2 ? ph : ph ^ 1u) ^ 1u));
                if (elect_one()) {
                    issue(s, kb);
                    if (two) issue(s2, kb + 1);
                }
                __syncwarp();
                if (two) {
                    s = s2;
                    if (s == 0) ph ^= 1u;
                    ++kb;
                }
            }
            if (++turn == NP) turn = 0;
            if (++s == sm.nstages) {
                s = 0;
                ph ^= 1u;
            }
            ready = !ONE && (NP == 1 || turn == pid) && mbar_test(sm.empty + 8 * s, ph ^ 1u);
        }
        if (wn < n_work) t = tile_finish(p, nl);
    }
}

// Table rows of this thread's GM_GATHER_ROWS rows of tile t (r = rb + GM_GATHER_RSTEP j of
// the CTA's half; past the tile row 0's, unused), loaded one item ahead of their use.
__device__ __forceinline__ void gather_rows_load(const GemmArgs& p, const Tile& t, uint32_t rank,
                                                 int rb, int (&raw)[GM_GATHER_ROWS]) {
    const int nh = rows_half(t, rank);
#pragma unroll
    for (int j = 0; j < GM_GATHER_ROWS; ++j) {
        const int r = rb + GM_GATHER_RSTEP * j;
        const int gr = t.row0 + (int)rank * GM_HALF + r;
        raw[j] = p.a_ident ? gr : __ldg(p.a_rows + (r < nh ? gr : 0));
    }
}

// A row pointers from the loaded table rows (nullptr past the tile; an A row outside
// [0, a_nrows) is a device error and is not read).  This runs between two items, on the path
// that paces the launch: the division by a_div is a multiplication (four divisions a thread here
// cost the stage calls' up-projection 2 %: T = 8192, d = 512, E = 16, k = 2 19.5 -> 19.0 us).
__device__ __forceinline__ void gather_rows_finish(const GemmArgs& p, const Tile& t, uint32_t rank,
                                                   int rb, const int (&raw)[GM_GATHER_ROWS],
                                                   const __nv_bfloat16* (&src)[GM_GATHER_ROWS]) {
    const int nh = rows_half(t, rank);
#pragma unroll
    for (int j = 0; j < GM_GATHER_ROWS; ++j) {
        const int r = rb + GM_GATHER_RSTEP * j;
        const int idx = raw[j] < 0 ? -1 : (int)((uint64_t)(uint32_t)raw[j] * p.a_div_mul >> p.a_div_shift);
        if (r < nh && idx >= 0 && idx < p.a_nrows) {
            src[j] = p.A + (int64_t)idx * p.lda;
        } else {
            if (r < nh && !(p.a_neg_zero && raw[j] < 0))   // padding rows read as zeros
                report(p.status, MOEVIE_ERR_DEVICE, SITE_GEMM_A_ROW, t.row0 + (int)rank * GM_HALF + r,
                       idx);
            src[j] = nullptr;
        }
    }
}

// Token gather (GM_GATHER_WARPS warps): each thread copies one 16-byte chunk of
// GM_GATHER_ROWS rows per stage straight into the 128-byte swizzled K-major layout,
// then hands the completion of its copies to the stage's afull barrier
// (cp.async.mbarrier.arrive.noinc) and moves on without waiting; gather_forwarder
// publishes the stage once every gather thread's copies have landed.
__device__ void producer_gather(const GemmArgs& p, const Smem& sm, int64_t n_work,
                                volatile int* abort_flag) {
    const int pt = threadIdx.x - GM_WARP_GATHER * 32;   // 0 .. GM_GATHER_WARPS * 32 - 1
    const int c = pt & 7, rb = pt >> 3;                  // 16-byte chunk, first row
    // gathered rows are re-read by every expert of their tokens: keep them in L2
    const uint64_t keep_pol = l2_policy_evict_last();
    int s = 0;
    uint32_t ph = 0;
    bool ready = false;
    int64_t w = sm.pair;
    // The per-item set-up is pipelined so that no load is waited on at an item start:
    // item w's row pointers are ready when it starts; the next item's table rows were
    // loaded one item earlier, after its tile entry (loaded earlier still) was checked.
    // Past the last item the last one is loaded again (unused): conditional loads would be
    // waited for where their values merge, several thousand cycles an item.
    if (w >= n_work) return;
    const __nv_bfloat16* src[GM_GATHER_ROWS];
    int nraw[GM_GATHER_ROWS];
    const int64_t w1 = w + sm.npairs < n_work ? w + sm.npairs : w;
    const TileLd l0 = tile_load(p, w), l1 = tile_load(p, w1);
    TileLd nnl = tile_load(p, w1 + sm.npairs < n_work ? w1 + sm.npairs : w1);
    Tile t = tile_finish(p, l0), tn = tile_finish(p, l1);
    {
        int raw[GM_GATHER_ROWS];
        gather_rows_load(p, t, sm.rank, rb, raw);
        gather_rows_load(p, tn, sm.rank, rb, nraw);
        gather_rows_finish(p, t, sm.rank, rb, raw, src);
    }
    const uint32_t dst_t = sm.a0 + rb * 128 + ((c ^ (rb & 7)) << 4);
    static_assert(GM_GATHER_RSTEP % 8 == 0, "the swizzle phase is the same for all rows of a thread");
    for (; w < n_work; w += sm.npairs) {
        for (int kb = t.kb0; kb < t.kb1; ++kb) {
            if (!mbar_wait_warp(sm.empty + 8 * s, ph ^ 1u, p.limit_ns, abort_flag, ready)) {
                set_abort(abort_flag, p.status, SITE_GEMM_WAIT_EMPTY, (int)sm.pair, 0);
                cp_async_wait_all();
                return;
            }
            const uint32_t dst0 = dst_t + s * GM_A_BYTES;
            const int kk = kb * GM_BK + c * 8;
            const bool col_ok = kk < p.K;
#pragma unroll
            for (int j = 0; j < GM_GATHER_ROWS; ++j) {
                const bool v = col_ok && src[j] != nullptr;
                cp_async16_hint(dst0 + j * (GM_GATHER_RSTEP * 128), v ? (const void*)(src[j] + kk) : (const void*)p.A,
                                v ? 16u : 0u, keep_pol);
            }
            cp_async_arrive_noinc(sm.afull + 8 * s);
            if (++s == sm.nstages) {
                s = 0;
                ph ^= 1u;
            }
            ready = mbar_test(sm.empty + 8 * s, ph ^ 1u);
        }
        // advance: the next item's pointers, the table rows of the one after, a further entry
        gather_rows_finish(p, tn, sm.rank, rb, nraw, src);
        t = tn;
        tn = tile_finish(p, nnl);
        gather_rows_load(p, tn, sm.rank, rb, nraw);
        const int64_t w3 = w + 3 * sm.npairs;
        nnl = tile_load(p, w3 < n_work ? w3 : w);
    }
    cp_async_wait_all();
}

// Warp GM_WARP_FWD (one elected lane), in both CTAs: once all of this CTA's gather threads'
// copies of a stage have landed (its afull barrier), make them visible to the async
// proxy that tcgen05.mma reads shared memory through, and publish the stage on the
// leader's full barrier: a local arrival in the leader; from the peer, a 16-byte
// async-proxy copy into the leader that completes 16 transaction bytes on that
// barrier (the leader's expect_tx counts them).  Being ordered after the proxy
// fence, the copy's completion implies the gathered rows are visible to the MMA,
// without the cost of a cluster-scope release by this thread.
__device__ void gather_forwarder(const GemmArgs& p, const Smem& sm, int64_t n_work,
                                 volatile int* abort_flag) {
    const uint32_t full_leader = peer_addr(sm.full, 0);
    const uint32_t sink_leader = peer_addr(sm.sink, 0);
    int s = 0;
    uint32_t ph = 0;
    bool ready = false;
    for (int64_t w = sm.pair; w < n_work; w += sm.npairs) {
        int kb0, kb1;   // the item's stages; its table entry is not needed here
        tile_kb(p, (int)(w % p.ksplit), kb0, kb1);
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!mbar_wait_warp(sm.afull + 8 * s, ph, p.limit_ns, abort_flag, ready)) {
                set_abort(abort_flag, p.status, SITE_GEMM_WAIT_FULL, (int)sm.pair, -1 - kb);
                return;
            }
            if (elect_one()) {
                fence_proxy_async_smem();
                if (sm.rank == 0) mbar_arrive(sm.full + 8 * s);
                else bulk_signal_remote(sink_leader, sm.sink, full_leader + 8 * s);
            }
            __syncwarp();
            if (++s == sm.nstages) {
                s = 0;
                ph ^= 1u;
            }
            ready = mbar_test(sm.afull + 8 * s, ph);
        }
    }
}

// ------------------------------------------------------------------- MMA

// Leader CTA, warp 8, all lanes in step; one elected lane issues.
template <bool TRAIN, bool ONE, bool TRANS>
__device__ void mma_issuer(const GemmArgs& p, const Smem& sm, uint32_t tmem, int64_t n_work,
                           volatile int* abort_flag) {
    // K-major operands: k-slice +32 B; MN-major operands: next 64-element atom LBO 8192,
    // k-slice +2048 B (16 K rows of 128 bytes).  The forward's A is K-major, its B MN-major;
    // transposed, the weights are the MMA's A and the rows its K-major B.
    const bool a_mn = TRANS ? !(TRAIN && p.b_kmajor) : TRAIN && p.a_mn;
    const bool b_km = TRANS || (TRAIN && p.b_kmajor);
    uint32_t idesc = idesc_bf16_f32(2 * GM_HALF, p.BN, a_mn, !b_km);
    const uint64_t adesc0 = a_mn ? smem_desc_sw128(sm.a0, 8192, 1024) : smem_desc_sw128(sm.a0, 16, 1024);
    const uint64_t bdesc0 = b_km ? smem_desc_sw128(sm.b0, 16, 1024) : smem_desc_sw128(sm.b0, 8192, 1024);
    const uint32_t a_step = a_mn ? (2048 >> 4) : (32 >> 4);
    const uint32_t b_step = b_km ? (32 >> 4) : (2048 >> 4);
    static_assert(GM_BK == 64, "four k-slices of 16 per stage");
    int s = 0;
    uint32_t ph = 0;
    int it = 0;
    bool issued = false, ready = false;
    if (sm.pair >= n_work) return;
    TileLd nl = tile_load(p, sm.pair);   // loaded one item ahead, checked when the item starts
    for (int64_t w = sm.pair; w < n_work; w += sm.npairs, ++it) {
        const Tile t = tile_finish(p, nl);
        nl = tile_load(p, w + sm.npairs < n_work ? w + sm.npairs : w);
        const int acc = it & 1;
        const uint32_t aph = (uint32_t)(it >> 1) & 1u;
        if (!mbar_wait_warp<ONE>(sm.tempty + 8 * acc, aph ^ 1u, p.limit_ns, abort_flag)) {
            set_abort(abort_flag, p.status, SITE_GEMM_WAIT_TEMPTY, (int)sm.pair, it);
            break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem + (uint32_t)acc * GM_MAXBN;
        if (TRANS) idesc = idesc_bf16_f32(2 * GM_HALF, trans_n(t), a_mn, false);
        bool ok = true;
        for (int kb = t.kb0; kb < t.kb1; ++kb) {
            // Operands in shared memory are ordered by the barrier alone (TMA bytes, or
            // gathered rows fenced to the async proxy before they were published); the
            // tcgen05 thread-sync fence is needed only where TMEM changes hands.
            if (!mbar_wait_warp<ONE>(sm.full + 8 * s, ph, p.limit_ns, abort_flag, ready)) {
                set_abort(abort_flag, p.status, SITE_GEMM_WAIT_FULL, (int)sm.pair, kb);
                ok = false;
                break;
            }
            // Descriptors differ from the stage-0 ones only in the start-address field
            // (bits 0-13, address >> 4; shared addresses stay below 256 KB, no carry).
            const uint64_t ad = adesc0 + (uint64_t)((s * GM_A_BYTES) >> 4);
            const uint64_t bd = bdesc0 + (uint64_t)((s * GM_B_BYTES) >> 4);
            if (elect_one()) {
                tc_mma_bf16_pair(d_tmem, ad, bd, idesc, kb != t.kb0 ? 1u : 0u);
                tc_mma_bf16_pair(d_tmem, ad + a_step, bd + b_step, idesc, 1u);
                tc_mma_bf16_pair(d_tmem, ad + 2 * a_step, bd + 2 * b_step, idesc, 1u);
                tc_mma_bf16_pair(d_tmem, ad + 3 * a_step, bd + 3 * b_step, idesc, 1u);
                tc_commit_pair(sm.empty + 8 * s);
            }
            __syncwarp();
            issued = true;
            if (++s == sm.nstages) {
                s = 0;
                ph ^= 1u;
            }
            ready = mbar_test(sm.full + 8 * s, ph);
        }
        if (!ok) break;
        if (elect_one()) tc_commit_pair(sm.tfull + 8 * acc);
        __syncwarp();
    }
    // Every tcgen05.mma must be complete before TMEM is released.
    if (issued) {
        if (elect_one()) tc_commit_pair(sm.drain);
        __syncwarp();
        if (!mbar_wait_warp<ONE>(sm.drain, 0, p.limit_ns, nullptr))
            report(p.status, MOEVIE_ERR_TIMEOUT, SITE_GEMM_DRAIN, (int)sm.pair, 0);
    }
}

// -------------------------------------------------------------- epilogue

// Epilogue of the transposed product (EPI_ADD_F32 of rows): the accumulator holds D^T, so
// TMEM lane l of the CTA is output column n0 + 128 rank + l and TMEM column j is row j of
// the tile.  A warp takes 32 columns and every fourth chunk of 32 rows; register i of all
// its lanes is row i, so one scalar reduction instruction covers 128 contiguous bytes of one
// token's row of y: whole L2 lines straight from registers.  (The product the other way
// round holds a row per lane: its reductions needed a transposition through shared memory.)
// Scalar 128-byte reductions run at 6.6 TB/s into an L2-resident buffer, as fast as 16-byte
// vector ones.  The reductions bound the tile (1024 per CTA and full tile, 6 cycles each at
// that rate, against 4096 cycles of MMAs at K = 512), so the gather warps, idle here, join
// the eight epilogue warps: while some load their tables and accumulators the others keep
// the reductions going.  The rows' tokens and scales are loaded one tile ahead and reach all
// lanes through 256 bytes of shared memory per warp (two rows per 16-byte broadcast).
template <bool TRAIN>
__device__ void epilogue_addt(const GemmArgs& p, const Smem& sm, uint32_t tmem, int64_t n_work, int warp,
                              volatile int* abort_flag) {
    const int lane = threadIdx.x & 31;
    const int quad = warp & 3;   // the TMEM lanes a warp may read
    const int part = warp < GM_EPI_WARPS ? warp >> 2 : 2 + ((warp - GM_WARP_GATHER) >> 2);
    constexpr int NCH = GM_BM / 32 / GM_ADDT_PARTS;   // chunks of a warp in a full tile
    const uint32_t tempty_leader = peer_addr(sm.tempty, 0);
    int2* info = reinterpret_cast<int2*>(sm.stg) + (part * 4 + quad) * 32;
    const int4* info2 = reinterpret_cast<const int4*>(info);
    if (sm.pair >= n_work) return;
    // token and scale of this lane's row of each of the warp's chunks (past the tile row 0's,
    // unused); the forward has both tables
    auto rows_load = [&](const Tile& t, int (&tok)[NCH], float (&sc)[NCH]) {
#pragma unroll
        for (int i = 0; i < NCH; ++i) {
            const int r = (part + GM_ADDT_PARTS * i) * 32 + lane;
            const int gr = r < t.nrows ? t.row0 + r : 0;
            tok[i] = !TRAIN || p.o_rows ? __ldg(p.o_rows + gr) : gr;
            sc[i] = !TRAIN ? __ldg(p.row_scale + gr) : p.scale;
        }
    };
    int64_t w = sm.pair;
    const int64_t w1 = w + sm.npairs < n_work ? w + sm.npairs : w;
    const TileLd l0 = tile_load(p, w);
    TileLd nl = tile_load(p, w1);
    Tile t = tile_finish(p, l0);
    int tok[NCH], ntok[NCH];
    float sc[NCH], nsc[NCH];
    rows_load(t, tok, sc);
    const int ld = (int)p.ldy;
    int it = 0;
    for (; w < n_work; w += sm.npairs, ++it) {
        // the next tile's entry (loaded a tile ago) and rows, the entry after it
        const Tile tn = tile_finish(p, nl);
        rows_load(tn, ntok, nsc);
        const int64_t w2 = w + 2 * sm.npairs;
        nl = tile_load(p, w2 < n_work ? w2 : w);
        const int acc = it & 1;
        const int nch = trans_n(t) / 32;
        const int col = t.n0 + (int)sm.rank * GM_HALF + quad * 32 + lane;
        const bool col_ok = col < p.N;
        float* yb = p.yacc + col;
        if (!mbar_wait(sm.tfull + 8 * acc, (uint32_t)(it >> 1) & 1u, p.limit_ns, abort_flag)) {
            set_abort(abort_flag, p.status, SITE_GEMM_WAIT_TFULL, (int)sm.pair, it);
            return;
        }
        tc_fence_after();
        const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)acc * GM_MAXBN;
        if (part >= nch) {   // no rows for this warp in this tile
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(tempty_leader + 8 * acc);
        }
#pragma unroll
        for (int i = 0; i < NCH; ++i) {
            const int ch = part + GM_ADDT_PARTS * i;
            if (ch >= nch) break;
            uint32_t v[32];
            tmem_ld_32x32b_x32(tbase + ch * 32, v);
            int tk = tok[i];
            if (ch * 32 + lane >= t.nrows) tk = -1;
            else if (tk < 0 || tk >= p.o_nrows) {
                if (!(p.o_neg_skip && tk < 0))   // a padding row writes nothing
                    report(p.status, MOEVIE_ERR_DEVICE, SITE_GEMM_OUT_ROW, t.row0 + ch * 32 + lane, tk);
                tk = -1;
            }
            info[lane] = make_int2(tk, __float_as_int(sc[i]));
            __syncwarp();
            tmem_wait_ld();
            if (ch + GM_ADDT_PARTS >= nch) {   // this warp's last read of the accumulator
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_remote(tempty_leader + 8 * acc);
            }
            if (col_ok) {
#pragma unroll
                for (int r0 = 0; r0 < 32; r0 += 8) {
                    int4 q[4];   // four broadcasts in flight before the eight reductions
#pragma unroll
                    for (int j = 0; j < 4; ++j) q[j] = info2[r0 / 2 + j];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int r = r0 + 2 * j;
                        red_add_f32_if(yb + (int64_t)q[j].x * ld, __int_as_float(q[j].y) * __uint_as_float(v[r]), q[j].x);
                        red_add_f32_if(yb + (int64_t)q[j].z * ld, __int_as_float(q[j].w) * __uint_as_float(v[r + 1]),
                                       q[j].z);
                    }
                }
            }
            __syncwarp();
        }
        t = tn;
#pragma unroll
        for (int i = 0; i < NCH; ++i) {
            tok[i] = ntok[i];
            sc[i] = nsc[i];
        }
    }
}

// One 32-column chunk of the fp32 outputs of one warp: each lane holds its row's 32 values
// (scaled by sc; tok < 0: no row).  The 32 rows pass the warp's 4 KB buffer (16-byte piece q of
// row r at r * 128 + 16 (q ^ (r & 7)): no bank conflicts either way), so that eight lanes store
// or reduce the 128 contiguous bytes of a row, whole L2 lines.  Stored by each lane from its own
// registers the pieces of 32 different lines an instruction held the router GEMM up:
// moevie_route at T = 65536, E = 256 235 -> 219 us, at T = 32768, E = 128 92.0 -> 86.7.  Reduced 16
// rows at a time through rows of 36 floats (half the lanes idle, bank conflicts) the band-ordered
// down-projection took 397 us at T = 32768, E = 128, this way 373.
__device__ __forceinline__ void out_chunk(const GemmArgs& p, uint8_t* buf, int lane, const float (&f)[32], float sc,
                                          int tok, int64_t base, int col0, int ncols, bool add, bool banded, uint64_t keep) {
#pragma unroll
    for (int q = 0; q < 8; ++q)
        *reinterpret_cast<float4*>(buf + lane * 128 + 16 * (q ^ (lane & 7))) =
            make_float4(sc * f[4 * q], sc * f[4 * q + 1], sc * f[4 * q + 2], sc * f[4 * q + 3]);
    __syncwarp();
    const int q = lane & 7;
    const bool col_ok = col0 + 4 * q < ncols;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3);
        const int tk = __shfl_sync(0xffffffffu, tok, r);
        const float4 v = *reinterpret_cast<const float4*>(buf + r * 128 + 16 * (q ^ (r & 7)));
        if (tk >= 0 && col_ok) {
            float4* dst = reinterpret_cast<float4*>(p.yacc + base + (int64_t)tk * p.ldy + col0 + 4 * q);
            if (add && banded) red_add_v4_hint(dst, v, keep);
            else if (add) atomicAdd(dst, v);
            else *dst = v;
        }
    }
    __syncwarp();
}

// Epilogue of the fp32 outputs.  Warp w reads TMEM lanes 32 (w % 4) .. +31 (its rows) and
// the 32-column chunks c = w / 4, w / 4 + 2, ... of each tile (out_chunk).  When a warp
// has read its last chunk of the accumulator it arrives (once) on the leader's tempty barrier.
template <int ECLS, bool TRAIN>
__device__ void epilogue(const GemmArgs& p, const Smem& sm, uint32_t tmem, int64_t n_work,
                         volatile int* abort_flag) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int quad = warp & 3, half = warp >> 2;
    const int nchunk = p.BN / 32;
    uint8_t* buf = reinterpret_cast<uint8_t*>(sm.stg) + warp * 4096;   // 32 rows x 128 bytes
    const uint32_t tempty_leader = peer_addr(sm.tempty, 0);
    // Band-ordered reductions keep the accumulator's lines in L2 (evict-last) beside the streamed
    // weights and rows: down-projection at T = 65536, d = 1664, E = 256 with loads after Zipf's
    // law 1048 -> 926-950 us, the conversion that reads the accumulator next 96 -> 90; at T = 32768,
    // d = 1536, E = 128 369-380 -> 365-387 (no difference beyond the runs'), conversion 43 -> 39.
    // (Operand rows evict-first instead: 903 -> 1113 on a skewed T = 65536 layer.)
    const bool banded = ECLS == ECLS_ADD && p.item_table == 1;
    const uint64_t keep = banded ? l2_policy_evict_last() : 0;
    int it = 0;
    if (sm.pair >= n_work) return;
    TileLd nl = tile_load(p, sm.pair);   // one item ahead
    for (int64_t w = sm.pair; w < n_work; w += sm.npairs, ++it) {
        const Tile t = tile_finish(p, nl);
        nl = tile_load(p, w + sm.npairs < n_work ? w + sm.npairs : w);
        const int acc = it & 1;
        const uint32_t aph = (uint32_t)(it >> 1) & 1u;
        const int myrow = quad * 32 + lane;
        const int gr = t.row0 + (int)sm.rank * GM_HALF + myrow;
        int64_t tok = gr;
        float sc = p.scale;
        bool ok_row = myrow < rows_half(t, sm.rank);
        if (ok_row) {
            if (p.o_rows) tok = __ldg(p.o_rows + gr) / p.o_div;
            if (p.row_scale) sc = __ldg(p.row_scale + gr);
            if (tok < 0 || tok >= p.o_nrows) {
                if (!(p.o_neg_skip && tok < 0))   // a padding row writes nothing
                    report(p.status, MOEVIE_ERR_DEVICE, SITE_GEMM_OUT_ROW, gr, (int)tok);
                ok_row = false;
            }
        }
        if (!mbar_wait(sm.tfull + 8 * acc, aph, p.limit_ns, abort_flag)) {
            set_abort(abort_flag, p.status, SITE_GEMM_WAIT_TFULL, (int)sm.pair, it);
            return;
        }
        tc_fence_after();
        const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)acc * GM_MAXBN;
        if (ECLS == ECLS_F32 && p.epi == EPI_SUM2_F32) {
            // two column groups of N / 2 (one n-tile): chunk ch of the output is the sum of
            // accumulator chunks ch and ch + nc2
            const int nc2 = nchunk / 2;
            if (half >= nc2) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_remote(tempty_leader + 8 * acc);
            }
            for (int ch = half; ch < nc2; ch += 2) {
                uint32_t v[32];
                float s2[32];
                tmem_ld_32x32b_x32(tbase + ch * 32, v);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) s2[i] = __uint_as_float(v[i]);
                tmem_ld_32x32b_x32(tbase + (ch + nc2) * 32, v);
                tmem_wait_ld();
                if (ch + 2 >= nc2) {   // this warp's last read of the accumulator
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_remote(tempty_leader + 8 * acc);
                }
#pragma unroll
                for (int i = 0; i < 32; ++i) s2[i] += __uint_as_float(v[i]);
                out_chunk(p, buf, lane, s2, sc, ok_row ? (int)tok : -1, t.ks * p.y_split_stride, ch * 32, p.N / 2, false, false, 0);
            }
            continue;
        }
        if (half >= nchunk) {   // no columns for this warp in this tile
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(tempty_leader + 8 * acc);
        }
        for (int ch = half; ch < nchunk; ch += 2) {
            const int c0 = ch * 32;
            uint32_t v[32];
            tmem_ld_32x32b_x32(tbase + c0, v);
            tmem_wait_ld();
            if (ch + 2 >= nchunk) {   // this warp's last read of the accumulator
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_remote(tempty_leader + 8 * acc);
            }
            float f[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) f[i] = __uint_as_float(v[i]);
            // weight-gradient items that are their tile's only one store instead of adding
            out_chunk(p, buf, lane, f, sc, ok_row ? (int)tok : -1, t.ks * p.y_split_stride, t.n0 + c0, p.N,
                      ECLS == ECLS_ADD && !(TRAIN && t.store), banded, keep);
        }
    }
}

// Epilogue of the bf16 outputs (gathered rows: GELU or SwiGLU; dense rows: GELU or plain; the
// training path's also keep the pre-activations).  Warp w reads TMEM lanes 32 (w % 4) .. +31 (its
// rows); each thread forms 32 (training path 16) columns of its own row at a time, and the warp's 32
// rows pass a buffer in shared memory, from which whole sectors are stored, 64 (training path 32)
// bytes of a row by neighbouring lanes.  (Stored by each thread straight from its registers they
// leave as 16-byte pieces of 32 different lines an instruction: up-projection T = 65536, d =
// 1664, E = 256 612 us against 593, T = 32768, E = 128 287 against 268.)  Below about 1024 columns of K
// the instructions of this epilogue bound the launch, 256 columns a tile against K / 64 stages, so
// what does not change is formed once a tile or a launch: the copies' addresses, and whether
// there is an activation (a template parameter).  Up-projection, addresses formed and the
// activation looked up at every piece -> this form, T = 8192: d = 512, E = 8, k = 2, h = 1000
// 33.1 -> 29.1 us (straight from registers 29.0), d = 512, E = 64, h = 256 33.7 -> 29.0, d = 768 36.6 -> 34.9,
// d = 1024, E = 64, h = 512 66.2 -> 61.9 (70.5); T = 1024, d = 1536 41.7 -> 40.0 (42.8).
template <bool TRAIN, bool GATHER, bool GELU>
__device__ void epilogue_bf16(const GemmArgs& p, const Smem& sm, uint32_t tmem, int64_t n_work,
                              volatile int* abort_flag) {
    constexpr int COLS = TRAIN ? 16 : 32, NP = COLS / 8;   // columns a step, 16-byte pieces of a row
    constexpr int ARR = 32 * COLS * 2;                     // bytes of one array's step
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int quad = warp & 3, half = warp >> 2;
    const bool swiglu = GATHER && p.swiglu;
    const int nchunk = swiglu ? p.BN / 64 : p.BN / 32;   // 32-column chunks of the output
    const int up0 = swiglu ? p.BN / 2 : 0;               // SwiGLU: first accumulator column of the up projection
    // bf16 results are written once and read back later: let them leave L2 first
    const uint64_t stream_pol = l2_policy_evict_first();
    const uint32_t tempty_leader = peer_addr(sm.tempty, 0);
    uint8_t* buf = reinterpret_cast<uint8_t*>(sm.stg) + warp * gm_bf16_warp_bytes(TRAIN);
    // piece q of row r at r * 2 COLS + 16 (q ^ swizzle(r)): eight consecutive rows' pieces (the
    // threads' writes) and eight consecutive pieces (the copies out) hit all banks
    auto place = [](int r, int q) { return r * (2 * COLS) + 16 * (q ^ (NP == 4 ? (r >> 1) & 3 : (r >> 2) & 1)); };
    // copied out: piece q0 of rows r0, r0 + RS, ... (RS rows on the swizzle is the same)
    constexpr int RS = 32 / NP, STEP = RS * 2 * COLS;
    const int r0 = lane / NP, q0 = lane % NP;
    const uint8_t* from = buf + place(r0, q0);
    if (sm.pair >= n_work) return;
    TileLd nl = tile_load(p, sm.pair);   // one item ahead
    int it = 0;
    for (int64_t w = sm.pair; w < n_work; w += sm.npairs, ++it) {
        const Tile t = tile_finish(p, nl);
        nl = tile_load(p, w + sm.npairs < n_work ? w + sm.npairs : w);
        const int acc = it & 1;
        const int nrow = rows_half(t, sm.rank) - quad * 32;   // rows of this warp (may be < 1 or > 32)
        const int64_t row0 = t.row0 + (int64_t)sm.rank * GM_HALF + quad * 32;
        if (!mbar_wait(sm.tfull + 8 * acc, (uint32_t)(it >> 1) & 1u, p.limit_ns, abort_flag)) {
            set_abort(abort_flag, p.status, SITE_GEMM_WAIT_TFULL, (int)sm.pair, it);
            return;
        }
        tc_fence_after();
        const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)acc * GM_MAXBN;
        if (half >= nchunk) {   // no columns for this warp in this tile
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(tempty_leader + 8 * acc);
        }
        const int64_t off0 = (row0 + r0) * p.ldo + t.n0 + 8 * q0;
        auto put = [&](int arr, int at, const float (&o)[8]) {
            uint4 u;
            u.x = pack_bf16x2(o[0], o[1]);
            u.y = pack_bf16x2(o[2], o[3]);
            u.z = pack_bf16x2(o[4], o[5]);
            u.w = pack_bf16x2(o[6], o[7]);
            *reinterpret_cast<uint4*>(buf + arr * ARR + at) = u;
        };
        // eight accumulator columns x (SwiGLU: the gate's, y the up projection's) into piece q of the lane's row
        auto act8 = [&](const uint32_t* x, const uint32_t* y, int q) {
            float f[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) f[i] = __uint_as_float(x[i]);
            const int at = place(lane, q);
            if (TRAIN && p.out2) put(1, at, f);   // the pre-activation (SwiGLU: the gate's) as well
            if (swiglu) {
                float g[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) g[i] = __uint_as_float(y[i]);
                if (TRAIN && p.out2) put(2, at, g);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    // SiLU(u) v = u v / (1 + e^-u); e^-u = inf for u far below 0 gives 0
                    f[i] = __fdividef(f[i], 1.0f + __expf(-f[i])) * g[i];
            } else if (GELU) {
#pragma unroll
                for (int i = 0; i < 8; i += 2) gelu_erf2(f[i], f[i + 1]);
            }
            put(0, at, f);
        };
        auto release = [&]() {   // this warp's last read of the accumulator
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(tempty_leader + 8 * acc);
        };
        auto copy_out = [&](int c) {   // the step's rows, written by all lanes, to columns t.n0 + c ..
            __syncwarp();
            const bool ok = t.n0 + c + 8 * q0 < p.N;
            // SwiGLU: a chunk's stores apart, each address formed before its store (at T = 8192, d = 1280,
            // h = 854 196 us; back to back as below 200)
            if (!TRAIN && swiglu) {
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    const int row = (lane + 32 * i) / NP, q = (lane + 32 * i) % NP;
                    if (row < nrow && t.n0 + c + 8 * q < p.N)
                        st_global_v4_hint(p.out + (row0 + row) * p.ldo + t.n0 + c + 8 * q,
                                          *reinterpret_cast<const uint4*>(buf + place(row, q)), stream_pol);
                }
                __syncwarp();   // copied out before the next step overwrites it
                return;
            }
            uint4 m[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                m[i] = *reinterpret_cast<const uint4*>(from + i * STEP);
                if (TRAIN && p.out2 && ok && r0 + RS * i < nrow) {
                    const int64_t off = off0 + c + i * (RS * p.ldo);
                    *reinterpret_cast<uint4*>(p.out2 + off) = *reinterpret_cast<const uint4*>(from + i * STEP + ARR);
                    if (swiglu)
                        *reinterpret_cast<uint4*>(p.out3 + off) = *reinterpret_cast<const uint4*>(from + i * STEP + 2 * ARR);
                }
            }
            __syncwarp();   // read before the next step overwrites it
#pragma unroll
            for (int i = 0; i < NP; ++i)
                if (ok && r0 + RS * i < nrow) st_global_v4_hint(p.out + off0 + c + i * (RS * p.ldo), m[i], stream_pol);
        };
        for (int ch = half; ch < nchunk; ch += 2) {
            if (!TRAIN && !swiglu) {
                uint32_t v[32];
                tmem_ld_32x32b_x32(tbase + ch * 32, v);
                tmem_wait_ld();
                if (ch + 2 >= nchunk) release();
#pragma unroll
                for (int q = 0; q < 4; ++q) act8(v + 8 * q, v + 8 * q, q);
                copy_out(ch * 32);
            } else {
#pragma unroll
                for (int c0 = 0; c0 < 32; c0 += COLS) {
                    const int c = ch * 32 + c0;
#pragma unroll
                    for (int s0 = 0; s0 < COLS; s0 += 16) {
                        uint32_t x[16], y[16];
                        tmem_ld_32x32b_x16(tbase + c + s0, x);
                        if (swiglu) tmem_ld_32x32b_x16(tbase + up0 + c + s0, y);
                        tmem_wait_ld();
                        if (ch + 2 >= nchunk && c0 + s0 + 16 == 32) release();
#pragma unroll
                        for (int q = 0; q < 2; ++q) act8(x + 8 * q, y + 8 * q, s0 / 8 + q);
                    }
                    copy_out(c);
                }
            }
        }
    }
}

// Epilogue of the activation derivatives (EPI_DGELU_BF16, EPI_DSWIGLU_BF16): each thread takes
// its own row, 16 columns at a time: du = scale acc GELU'(u) (SwiGLU: du = scale acc v
// SiLU'(u), dv = scale acc SiLU(u)) and the row dot acc . a.  What bounds it is the latency of
// the u, v and a rows (64 KB a tile each), so they come through a double buffer in shared
// memory, whole 32-byte sectors by cp.async one 16-column step ahead, also across tiles.
// At T = 8192, d = 1024, E = 31, k = 3, h = 684 (SwiGLU) the launch took 236 us with each
// thread loading its row's 16-byte pieces as it needed them, 156 us with the pieces one step
// ahead in registers (which spilled), and 75 us this way.
template <bool SWIGLU>
__device__ void epilogue_dact(const GemmArgs& p, const Smem& sm, uint32_t tmem, int64_t n_work,
                              volatile int* abort_flag) {
    constexpr int NARR = SWIGLU ? 3 : 2;   // u, a (, v)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int quad = warp & 3, half = warp >> 2;
    const int nchunk = p.BN / 32;
    const int nsub = half < nchunk ? (nchunk - half + 1) / 2 * 2 : 0;   // 16-column steps of this warp
    const uint32_t tempty_leader = peer_addr(sm.tempty, 0);
    // this warp's buffer: 2 slots x NARR arrays x 32 rows x 32 bytes; 16-byte piece q of row r
    // at r * 32 + 16 (q ^ (r / 4 & 1)), so that eight consecutive rows' pieces hit all banks
    uint8_t* buf = reinterpret_cast<uint8_t*>(sm.stg) + warp * (2 * NARR * 1024);
    const uint32_t buf_a = smem_u32(buf);
    if (sm.pair >= n_work) return;
    auto col_of = [&](int k) { return (half + 2 * (k >> 1)) * 32 + (k & 1) * 16; };
    // step k of tile tt into slot `slot`: lane l copies piece l & 1 of rows l / 2 and l / 2 + 16
    auto fetch = [&](const Tile& tt, int k, int slot) {
        const int q = lane & 1;
        const int n = tt.n0 + col_of(k) + 8 * q;
        const int nh = rows_half(tt, sm.rank);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = (lane >> 1) + 16 * i;
            const bool ok = quad * 32 + r < nh && n < p.N;
            const int64_t off = ok ? (int64_t)(tt.row0 + (int)sm.rank * GM_HALF + quad * 32 + r) * p.ldo + n : 0;
            const uint32_t dst = buf_a + slot * (NARR * 1024) + r * 32 + 16 * (q ^ ((r >> 2) & 1));
            cp_async16(dst, p.epi_u + off, ok ? 16u : 0u);
            cp_async16(dst + 1024, p.epi_a + off, ok ? 16u : 0u);
            if (SWIGLU) cp_async16(dst + 2048, p.epi_v + off, ok ? 16u : 0u);
        }
    };
    const TileLd l0 = tile_load(p, sm.pair);
    TileLd nl = tile_load(p, sm.pair + sm.npairs < n_work ? sm.pair + sm.npairs : sm.pair);
    Tile t = tile_finish(p, l0);
    if (nsub > 0) fetch(t, 0, 0);
    cp_async_commit();
    int it = 0;
    for (int64_t w = sm.pair; w < n_work; w += sm.npairs, ++it) {
        const Tile tn = tile_finish(p, nl);   // (past the last item: the last one again)
        const int64_t w2 = w + 2 * sm.npairs;
        nl = tile_load(p, w2 < n_work ? w2 : w);
        const int acc = it & 1;
        const int myrow = quad * 32 + lane;
        const int gr = t.row0 + (int)sm.rank * GM_HALF + myrow;
        const bool ok_row = myrow < rows_half(t, sm.rank);
        const float sc = p.row_scale ? __ldg(p.row_scale + (ok_row ? gr : 0)) : p.scale;
        const int64_t row = (int64_t)(ok_row ? gr : 0) * p.ldo;
        if (!mbar_wait(sm.tfull + 8 * acc, (uint32_t)(it >> 1) & 1u, p.limit_ns, abort_flag)) {
            set_abort(abort_flag, p.status, SITE_GEMM_WAIT_TFULL, (int)sm.pair, it);
            cp_async_wait_all();
            return;
        }
        tc_fence_after();
        const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)acc * GM_MAXBN;
        if (nsub == 0) {   // no columns for this warp in this tile
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(tempty_leader + 8 * acc);
        }
        float dg_acc = 0.f;   // this thread's share of its row's dot
        for (int k = 0; k < nsub; ++k) {   // nsub is even: step k of every tile uses slot k & 1
            __syncwarp();   // every lane has read the slot that is filled next
            if (k + 1 < nsub) fetch(t, k + 1, (k + 1) & 1);
            else fetch(tn, 0, 0);
            cp_async_commit();
            uint32_t x[16];
            tmem_ld_32x32b_x16(tbase + col_of(k), x);
            cp_async_wait<1>();
            tmem_wait_ld();
            __syncwarp();   // step k's pieces, copied by all lanes
            if (k + 1 == nsub) {   // this warp's last read of the accumulator
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_remote(tempty_leader + 8 * acc);
            }
            if (!ok_row) continue;
            const int n = t.n0 + col_of(k);
            const uint8_t* in = buf + (k & 1) * (NARR * 1024) + lane * 32;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (n + 8 * q >= p.N) break;
                const uint8_t* piece = in + 16 * (q ^ ((lane >> 2) & 1));
                float uf[8], af[8], fu[8];
                unpack_bf16x8(*reinterpret_cast<const uint4*>(piece), uf);
                unpack_bf16x8(*reinterpret_cast<const uint4*>(piece + 1024), af);
                if constexpr (SWIGLU) {
                    float vf[8], fv[8];
                    unpack_bf16x8(*reinterpret_cast<const uint4*>(piece + 2048), vf);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float a = __uint_as_float(x[8 * q + i]);
                        const bool ok = n + 8 * q + i < p.N;   // columns past N: padding
                        dg_acc += ok ? a * af[i] : 0.f;
                        const float sg = __fdividef(1.0f, 1.0f + __expf(-uf[i]));   // SiLU(u) = u sg
                        fu[i] = ok ? sc * a * vf[i] * sg * (1.0f + uf[i] * (1.0f - sg)) : 0.f;
                        fv[i] = ok ? sc * a * uf[i] * sg : 0.f;
                    }
                    uint4 o;
                    o.x = pack_bf16x2(fv[0], fv[1]);
                    o.y = pack_bf16x2(fv[2], fv[3]);
                    o.z = pack_bf16x2(fv[4], fv[5]);
                    o.w = pack_bf16x2(fv[6], fv[7]);
                    *reinterpret_cast<uint4*>(p.out2 + row + n + 8 * q) = o;
                } else {
#pragma unroll
                    for (int i = 0; i < 8; i += 2) gelu_grad2(uf[i], uf[i + 1]);   // GELU'(u)
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float a = __uint_as_float(x[8 * q + i]);
                        const bool ok = n + 8 * q + i < p.N;   // columns past N: padding
                        dg_acc += ok ? a * af[i] : 0.f;
                        fu[i] = ok ? sc * a * uf[i] : 0.f;
                    }
                }
                uint4 o;
                o.x = pack_bf16x2(fu[0], fu[1]);
                o.y = pack_bf16x2(fu[2], fu[3]);
                o.z = pack_bf16x2(fu[4], fu[5]);
                o.w = pack_bf16x2(fu[6], fu[7]);
                *reinterpret_cast<uint4*>(p.out + row + n + 8 * q) = o;
            }
        }
        if (ok_row && p.dg_part)   // row dot (the gates' gradient; none for the shared expert)
            p.dg_part[(int64_t)(2 * (t.n0 / p.n_step) + half) * p.m_total + gr] = dg_acc;
        t = tn;
    }
    cp_async_wait_all();
}

template <bool GATHER, int ECLS, bool TRAIN>
__global__ void __launch_bounds__(GM_THREADS, 1) grouped_gemm_kernel(const __grid_constant__ GemmArgs p) {
    extern __shared__ uint8_t gm_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(gm_smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint8_t* sA = smem;
    constexpr int nst = gm_stages(ECLS);
    uint8_t* sB = smem + nst * GM_A_BYTES;
    uint8_t* sStg = sB + nst * GM_B_BYTES;                       // epilogue staging
    uint64_t* bars = reinterpret_cast<uint64_t*>(sStg + gm_stg_bytes(ECLS, TRAIN));
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 3 * GM_STAGES_MAX + 5);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    uint8_t* sink = reinterpret_cast<uint8_t*>(bars) + 256;   // 16-byte aligned, after the barriers

    Smem sm;
    sm.a0 = smem_u32(sA);
    sm.b0 = smem_u32(sB);
    sm.full = smem_u32(bars);
    sm.empty = sm.full + 8 * GM_STAGES_MAX;
    sm.afull = sm.empty + 8 * GM_STAGES_MAX;
    sm.tfull = sm.afull + 8 * GM_STAGES_MAX;
    sm.tempty = sm.tfull + 16;
    sm.drain = sm.tempty + 16;
    sm.nstages = nst;
    sm.stg = reinterpret_cast<float*>(sStg);
    sm.sink = smem_u32(sink);
    sm.rank = cluster_rank();
    sm.pair = blockIdx.x >> 1;
    sm.npairs = gridDim.x >> 1;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);   // warp-uniform
    constexpr bool gather = GATHER;   // A rows gathered by the gather warps (else TMA)
    // TMA producer warps: with contiguous A the forwarder, idle there, joins GM_WARP_LOAD (not
    // beside the router GEMM's side jobs, where it cost 5 %)
    constexpr int NPROD = GATHER || ECLS == ECLS_F32 ? 1 : 2;
    const int prod_id = warp == GM_WARP_LOAD ? 0 : NPROD > 1 && warp == GM_WARP_FWD ? 1 : -1;
    if (threadIdx.x == 0) {
        for (int s = 0; s < nst; ++s) {
            // leader's expect_tx arrival (+ the leader's forwarder; the peer's signals
            // are transaction bytes)
            mbar_init(sm.full + 8 * s, 1 + (gather ? 1 : 0));
            mbar_init(sm.empty + 8 * s, 1);         // multicast tcgen05.commit
            mbar_init(sm.afull + 8 * s, GM_GATHER_WARPS * 32);   // gather threads (async arrivals)
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(sm.tfull + 8 * a, 1);         // multicast tcgen05.commit
            // every epilogue warp of the pair
            mbar_init(sm.tempty + 8 * a, 2 * (ECLS == ECLS_ADDT ? 4 * GM_ADDT_PARTS : GM_EPI_WARPS));
        }
        mbar_init(sm.drain, 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == GM_WARP_MMA) {
        tmem_alloc_pair(smem_u32(tmem_slot), 2 * GM_MAXBN);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // barriers of both CTAs initialised before any remote arrival
    tc_fence_after();
    pdl_wait();       // the previous kernel's outputs (tile tables, A, row maps) are ready
    const uint32_t tmem = *tmem_slot;
    int64_t n_mtiles;
    if (p.tiles) {
        n_mtiles = __ldg(p.n_tiles_dev);
        if (n_mtiles < 0 || n_mtiles > p.max_mtiles) {   // inconsistent offsets: no work
            if (threadIdx.x == 0) report(p.status, MOEVIE_ERR_DEVICE, SITE_GEMM_TILES, (int)n_mtiles, -1);
            n_mtiles = 0;
        }
    } else {
        n_mtiles = (p.m_total + GM_BM - 1) / GM_BM;
    }
    const int64_t n_work = p.item_table ? n_mtiles * p.ksplit : n_mtiles * p.n_ntiles * p.ksplit;

    if (warp < GM_EPI_WARPS || (ECLS == ECLS_ADDT && warp >= GM_WARP_GATHER && warp < GM_WARP_FWD)) {
        if constexpr (ECLS == ECLS_ADDT) epilogue_addt<TRAIN>(p, sm, tmem, n_work, warp, abort_flag);
        else if constexpr (ECLS == ECLS_DGELU) epilogue_dact<false>(p, sm, tmem, n_work, abort_flag);
        else if constexpr (ECLS == ECLS_DSWIGLU) epilogue_dact<true>(p, sm, tmem, n_work, abort_flag);
        else if constexpr (ECLS == ECLS_BF16) {
            if (GATHER || p.epi == EPI_GELU_BF16) epilogue_bf16<TRAIN, GATHER, true>(p, sm, tmem, n_work, abort_flag);
            else epilogue_bf16<TRAIN, GATHER, false>(p, sm, tmem, n_work, abort_flag);
        }
        else epilogue<ECLS, TRAIN>(p, sm, tmem, n_work, abort_flag);
    } else if (warp == GM_WARP_MMA) {
        if (sm.rank == 0) mma_issuer<TRAIN, ECLS == ECLS_F32, ECLS == ECLS_ADDT>(p, sm, tmem, n_work, abort_flag);
    } else if (prod_id >= 0) {
        producer_tma<GATHER, TRAIN, ECLS == ECLS_F32, ECLS == ECLS_ADDT, NPROD>(p, sm, n_work, prod_id, abort_flag);
    } else if (GATHER && warp == GM_WARP_FWD) {
        if constexpr (GATHER) gather_forwarder(p, sm, n_work, abort_flag);
    } else if (GATHER && warp >= GM_WARP_GATHER && warp < GM_WARP_FWD) {
        if constexpr (GATHER) producer_gather(p, sm, n_work, abort_flag);
    } else if (!GATHER && ECLS == ECLS_F32 && (p.zero || p.nrm_out || p.wn_out) &&
               warp >= GM_WARP_GATHER && warp < GM_WARP_FWD) {
        // Side jobs for the gather warps of a dense-A GEMM, while the MMAs run.
        // 1. Row norms of the A rows of this CTA's items (the router's |x_t|, read while
        //    the TMA brings the same rows in): one warp per row, lanes over 16-byte chunks;
        //    the K splits of an m-tile share its rows.
        if (p.nrm_out) {
            const int q = warp - GM_WARP_GATHER, lane = threadIdx.x & 31;
            for (int64_t w = sm.pair; w < n_work; w += sm.npairs) {
                const Tile t = decode_tile(p, w);
                if (t.n0 != 0) continue;
                const int nh = rows_half(t, sm.rank);
                // the K splits of an m-tile share its rows: split ks takes rows ks mod ksplit
                for (int r = t.ks + q * p.ksplit; r < nh; r += GM_GATHER_WARPS * p.ksplit) {
                    const int64_t row = t.row0 + (int64_t)sm.rank * GM_HALF + r;
                    const uint4* v = reinterpret_cast<const uint4*>(p.nrm_x + row * p.nrm_ld);
                    float acc = 0.f;
                    for (int c = lane; c < p.nrm_cols / 8; c += 32) {
                        const uint4 u = v[c];
                        float f[8];
                        unpack_bf16x8(u, f);
#pragma unroll
                        for (int i = 0; i < 8; ++i) acc = fmaf(f[i], f[i], acc);
                    }
#pragma unroll
                    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                    if (lane == 0) p.nrm_out[row] = sqrtf(acc);
                }
            }
        }
        // 2. Column norms from per-CTA partial sums of squares (wn_sets sets of wn_nparts
        //    parts): one warp per column, lanes over the parts, then a fixed shuffle tree
        //    (deterministic).
        if (p.wn_out) {
            const int q = warp - GM_WARP_GATHER, lane = threadIdx.x & 31;
            for (int j = blockIdx.x * GM_GATHER_WARPS + q; j < p.wn_sets * p.wn_E;
                 j += gridDim.x * GM_GATHER_WARPS) {
                const int set = j / p.wn_E, e = j - set * p.wn_E;
                const float* part = p.wn_part + (int64_t)set * p.wn_nparts * p.wn_Ep;
                float v = 0.f;
                for (int pp = lane; pp < p.wn_nparts; pp += 32) v += part[(int64_t)pp * p.wn_Ep + e];
#pragma unroll
                for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) p.wn_out[j] = sqrtf(v);
            }
        }
        // 3. Clear another buffer (the y accumulator) with 16-byte stores, grid-strided
        //    (evict-first: the zeros must not push the GEMM's re-read operands out of L2).
        if (p.zero) {
            const uint4 z = make_uint4(0u, 0u, 0u, 0u);
            const uint64_t pol = l2_policy_evict_first();
            const int64_t per = (int64_t)GM_GATHER_WARPS * 32;
            for (int64_t i = (int64_t)blockIdx.x * per + (threadIdx.x - GM_WARP_GATHER * 32);
                 i < p.zero_n; i += (int64_t)gridDim.x * per)
                st_global_v4_hint(p.zero + i, z, pol);
        }
    }

    tc_fence_before();
    __syncthreads();
    cluster_sync();   // the leader's MMAs have drained; both CTAs are done with TMEM
    if (warp == GM_WARP_MMA) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, 2 * GM_MAXBN);
    }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    }
    return fn;
}

}  // namespace

bool make_weight_tmap_strided(CUtensorMap* tm, const void* base, int64_t N, int64_t K, int64_t G,
                              int64_t k_ld, int64_t g_ld) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)N, (cuuint64_t)K, (cuuint64_t)G};
    cuuint64_t strides[2] = {(cuuint64_t)k_ld * 2, (cuuint64_t)g_ld * 2};
    cuuint32_t box[3] = {64, GM_BK, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims,
                     strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

bool make_weight_tmap(CUtensorMap* tm, const void* base, int64_t N, int64_t K, int64_t G) {
    return make_weight_tmap_strided(tm, base, N, K, G, N, N * K);
}

bool make_kmajor_tmap(CUtensorMap* tm, const void* base, int64_t K, int64_t N, int64_t G, int64_t k_ld,
                      int64_t g_ld, int box_n) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode_fn();
    if (!enc || box_n < 8 || box_n > 256) return false;
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)N, (cuuint64_t)G};
    cuuint64_t strides[2] = {(cuuint64_t)k_ld * 2, (cuuint64_t)g_ld * 2};
    cuuint32_t box[3] = {GM_BK, (cuuint32_t)box_n, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
                     estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

bool make_rows_tmap(CUtensorMap* tm, const void* base, int64_t cols, int64_t rows, int64_t ld,
                    int box_rows) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode_fn();
    if (!enc || box_rows < 8 || box_rows > 256) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                     box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

void choose_bn(int N, int* BN, int* n_ntiles) {
    const int nt = (N + GM_MAXBN - 1) / GM_MAXBN;
    int bn = (N + nt - 1) / nt;
    bn = (bn + 31) / 32 * 32;   // each CTA of a pair holds BN / 2 columns, a multiple of 16
    *BN = bn;
    *n_ntiles = (N + bn - 1) / bn;
}

cudaError_t launch_grouped_gemm(const GemmArgs& a, int grid, cudaStream_t s) {
    // one instance per (A path, epilogue class, training-path layouts): each holds only the
    // code its launches run (constant trip counts, no other epilogue or operand layout to
    // crowd its registers)
    using Kern = void (*)(GemmArgs);
    struct Inst {
        Kern kern;
        int ecls;
        bool train = false;
    };
    static const Inst insts[10] = {
        {grouped_gemm_kernel<false, ECLS_ADDT, false>, ECLS_ADDT},
        {grouped_gemm_kernel<false, ECLS_F32, false>, ECLS_F32},
        {grouped_gemm_kernel<false, ECLS_BF16, false>, ECLS_BF16},
        {grouped_gemm_kernel<true, ECLS_BF16, false>, ECLS_BF16},
        // the training path: K-major weights, M-major A, weight-gradient items, backward epilogues
        {grouped_gemm_kernel<true, ECLS_BF16, true>, ECLS_BF16, true},
        {grouped_gemm_kernel<false, ECLS_ADDT, true>, ECLS_ADDT, true},
        {grouped_gemm_kernel<false, ECLS_ADD, true>, ECLS_ADD, true},
        {grouped_gemm_kernel<false, ECLS_ADD, false>, ECLS_ADD},
        {grouped_gemm_kernel<true, ECLS_DGELU, true>, ECLS_DGELU, true},
        {grouped_gemm_kernel<true, ECLS_DSWIGLU, true>, ECLS_DSWIGLU, true}};
    const bool gathered = a.a_rows || a.a_ident;   // A rows through the gather warps
    const bool train = a.b_kmajor || a.a_mn || a.item_table == 2 || a.epi == EPI_GELU2_BF16 ||
                       a.epi == EPI_DGELU_BF16 || a.epi == EPI_DSWIGLU_BF16 || a.out2 != nullptr;
    const bool bf16_out = a.epi == EPI_GELU_BF16 || a.epi == EPI_STORE_BF16 || a.epi == EPI_SWIGLU_BF16 ||
                          a.epi == EPI_GELU2_BF16 || a.epi == EPI_DGELU_BF16 || a.epi == EPI_DSWIGLU_BF16;
    if (gathered && (!bf16_out || a.epi == EPI_STORE_BF16)) return cudaErrorInvalidValue;
    if (!gathered && a.epi == EPI_SWIGLU_BF16) return cudaErrorInvalidValue;
    if (a.trans && (a.epi != EPI_ADD_F32 || a.item_table)) return cudaErrorInvalidValue;
    int which;
    if (a.trans) which = train ? 5 : 0;
    else if (train && gathered) which = a.epi == EPI_DGELU_BF16 ? 8 : a.epi == EPI_DSWIGLU_BF16 ? 9 : 4;
    else if (a.epi == EPI_ADD_F32) which = train ? 6 : 7;
    else if (train) return cudaErrorInvalidValue;
    else if (gathered) which = 3;
    else which = a.epi == EPI_STORE_F32 || a.epi == EPI_SUM2_F32 ? 1 : 2;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        for (const Inst& k : insts) {
            cudaError_t e = cudaFuncSetAttribute(k.kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 gm_smem_bytes(k.ecls, k.train));
            if (e != cudaSuccess) return e;
        }
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((grid + 1) & ~1));   // whole pairs
    cfg.blockDim = dim3(GM_THREADS);
    cfg.dynamicSmemBytes = gm_smem_bytes(insts[which].ecls, insts[which].train);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see launch_pdl
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, insts[which].kern, a);
    count_launches(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace mv
