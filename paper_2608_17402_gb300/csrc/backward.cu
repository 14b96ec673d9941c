// backward.cu -- the training path of the MoE-ViE layer (App. B: grouped GEMMs with the
// activation as a separate step; gradients of sum_t dy_t . y_t with the top-k selection
// held fixed, through the renormalised gates of Eqs. 4-5 into W_r and x), sm_103a.
//
// The grouped GEMMs run on grouped_gemm_kernel (gemm.cu); this file holds the steps
// around them, all memory- or latency-bound:
//   bwd_gates_kernel   per token, the fp32 logits of its k selected experts (W_r's
//                      transposed copy), sigma, their sum S and the gates g = sigma / S
//   bwd_plan_kernel    expert segments padded to multiples of 64 rows (the K blocks of
//                      the weight-gradient GEMMs never straddle two experts), their m-tiles,
//                      and every weight-gradient item table, a CTA per table
//   bwd_rows_kernel    per padded row its token (-1 for padding) and gate (0), and per
//                      routing slot its padded row
//   bwd_zero_kernel    clears dx, ds and, of every weight gradient, what its items will add
//                      into or not write: groups with no rows or several chunks, pad columns
//   bwd_gather_kernel  the padded rows of x and of g dy (bf16; zero rows for padding)
//   bwd_router_kernel  per token: dg_j = dy . E_j(x) from the partial row dots, the gate
//                      derivative ds (Eqs. 4-5), dx += ds W_r^T, and ds into a dense
//                      [T][E_pad] bf16 matrix for dW_r = x^T ds
#include <math.h>

#include <algorithm>

#include "internal.h"

namespace mv {

namespace {

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// One warp per token: s_j = x_t . W_r[:, e_j] for its k experts (fp32, lanes over d; KB dot
// products advance together, U steps' loads ahead of their sums; KB = k up to 8, then passes of
// 8 with MORE), sigma_j = 1 / (1 + e^-s_j), S = sum_j sigma_j, g_j = sigma_j / S.  The selected
// rows of W_r come from L2; what bounds it is how many of their loads are in flight, so the
// loads are unconditional and the registers leave room for four CTAs on an SM.  At T =
// 8192, d = 1024, E = 64, in us:                   k = 1     4     8     9    16    32
//   this form                                        6.4  11.6  17.7  28.1  31.8  57.3
//   KB = 4, 8 or 32 >= k, U = 4, 4, 1 (116 to 204
//   registers from KB = 8 on)                       16.6  17.7  30.4   158   184   268
//   loads skipped where j >= k, U = 1               16.9  21.8  23.3   107   123   159
template <int KB, bool MORE, int U, int CTAS>
__global__ void __launch_bounds__(256, CTAS) bwd_gates_kernel(const __nv_bfloat16* __restrict__ x,
                                                              const float* __restrict__ wrt, int dp,
                                                              const int32_t* __restrict__ idx, int64_t T,
                                                              int d, int E, int k, float* __restrict__ sig,
                                                              float* __restrict__ gate, DevStatus* st) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= T) return;
    const __nv_bfloat16* xr = x + t * d;
    const int n = MORE ? k : KB;
    float ssum = 0.f, mine = 0.f;   // lane j keeps sigma_j
    for (int j0 = 0; j0 < n; j0 += KB) {
        int w[KB];   // offsets of the rows (E dp < 2^31: E <= 1024, d < 2^16); bad ids and past k: row 0, unused
        float acc[KB];
        uint32_t okm = 0;
#pragma unroll
        for (int j = 0; j < KB; ++j) {
            acc[j] = 0.f;
            const int e = !MORE || j0 + j < k ? idx[t * k + j0 + j] : 0;
            const bool ok = e >= 0 && e < E;
            if (!ok && lane == 0) report(st, MOEVIE_ERR_DEVICE, SITE_PERMUTE_ID, (int)(t * k + j0 + j), e);
            if (ok) okm |= 1u << j;
            w[j] = (ok ? e : 0) * dp;
        }
        int i = lane;
        for (; i + 32 * (U - 1) < d; i += 32 * U) {
            float xi[U], wv[U][KB];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                xi[u] = __bfloat162float(xr[i + 32 * u]);
#pragma unroll
                for (int j = 0; j < KB; ++j) wv[u][j] = __ldg(wrt + w[j] + i + 32 * u);
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int j = 0; j < KB; ++j) acc[j] = fmaf(xi[u], wv[u][j], acc[j]);
        }
        for (; i < d; i += 32) {
            const float xi = __bfloat162float(xr[i]);
#pragma unroll
            for (int j = 0; j < KB; ++j) acc[j] = fmaf(xi, __ldg(wrt + w[j] + i), acc[j]);
        }
#pragma unroll
        for (int j = 0; j < KB; ++j) {
            if (MORE && j0 + j >= k) break;
            const float sgm = 1.0f / (1.0f + expf(-warp_sum_f((okm >> j) & 1u ? acc[j] : 0.f)));
            if (lane == j0 + j) mine = sgm;
            ssum += sgm;
        }
    }
    if (lane < k) {
        sig[t * k + lane] = mine;
        gate[t * k + lane] = mine / ssum;
    }
}

// Exclusive scan of one int per thread over a CTA of 1024; *total = the sum (s_w: 33 ints).
__device__ __forceinline__ int block_scan_1024(int v, int* s_w, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int w = s_w[lane];
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += u;
        }
        s_w[lane] = wi - w;
        if (lane == 31) s_w[32] = wi;
    }
    __syncthreads();
    const int ex = s_w[warp] + inc - v;
    *total = s_w[32];
    __syncthreads();   // s_w may be reused
    return ex;
}

// The plan of the backward in one launch, CTAs of 1024 threads, one thread per expert (E <=
// 1024): every CTA forms the padded offsets (counts rounded up to 64 rows) itself.  CTA 0
// writes poff[E + 1] and the m-tile table of the padded rows; CTA q > 0 the item table of set
// q - 1 (BwdItemSet): group g (an expert, or the one dense group) has the k-blocks of its
// padded rows, cut into chunks of at most BWD_KCH; its items are every (m-tile of 256 of M
// rows, n-tile of BN of N columns, chunk).  items[i] = {g, m0 | n0 << 16, kb0, kb1}; *n_items =
// their number (at most max_items; more is a device error and none are listed).  A group
// of one chunk writes each of its gradient's elements once: its items carry BWD_STORE_BIT in
// kb1 (the GEMM stores instead of adding) and gclear[g] = 0; a group with no rows or several
// chunks has gclear[g] = 1 (its gradient is cleared first).  (One launch for all the
// tables: of one CTA each they take 3 - 4 us apiece, seven to nine of them.)
__global__ void __launch_bounds__(1024) bwd_plan_kernel(const __grid_constant__ BwdPlan p) {
    pdl_wait();
    __shared__ int s_w[33];
    const int e = threadIdx.x;
    int total;
    const int v = e < p.E ? (p.counts[e] + 63) / 64 * 64 : 0;
    const int off = block_scan_1024(v, s_w, &total);
    if (blockIdx.x == 0) {
        if (e < p.E) p.poff[e] = off;
        if (e == 0) p.poff[p.E] = total;
        const int nt = (v + GM_BM - 1) / GM_BM;
        int ntiles;
        const int toff = block_scan_1024(nt, s_w, &ntiles);
        for (int m = 0; m < nt; ++m) p.tiles[toff + m] = make_int4(e, off + m * GM_BM, min(GM_BM, v - m * GM_BM), 0);
        if (e == 0) *p.n_tiles = ntiles;
        return;
    }
    const BwdItemSet& q = p.sets[blockIdx.x - 1];
    const int G = q.dense_rows > 0 ? 1 : p.E;
    const int mt = (q.M + GM_BM - 1) / GM_BM, nt = (q.N + q.BN - 1) / q.BN;
    int kb0 = 0, kb1 = 0;
    if (e < G) {
        kb0 = q.dense_rows > 0 ? 0 : off / GM_BK;
        kb1 = q.dense_rows > 0 ? (int)((q.dense_rows + GM_BK - 1) / GM_BK) : (off + v) / GM_BK;
    }
    const int chunks = (kb1 - kb0 + (int)BWD_KCH - 1) / (int)BWD_KCH;
    int n;
    int pos = block_scan_1024(chunks * mt * nt, s_w, &n);
    if (n > q.max_items) {
        if (e == 0) {
            report(p.st, MOEVIE_ERR_DEVICE, SITE_GEMM_TILES, n, q.max_items);
            *q.n_items = 0;
        }
        return;
    }
    const int store = chunks == 1 ? BWD_STORE_BIT : 0;
    for (int c = 0; c < chunks; ++c) {
        const int a = kb0 + c * (int)BWD_KCH, b = min(kb1, a + (int)BWD_KCH);
        for (int m = 0; m < mt; ++m)
            for (int j = 0; j < nt; ++j)
                q.items[pos++] = make_int4(e, (m * GM_BM) | ((j * q.BN) << 16), a, b | store);
    }
    if (e < G) q.gclear[e] = chunks == 1 ? 0 : 1;
    if (e == 0) *q.n_items = n;
}

// Threads over routing slots (t, j) and over (expert, padding row < 64): the padded row of
// slot t k + j is poff[e] + (its expert-major row - offsets[e]); padding rows of expert e
// (poff[e] + counts[e] .. poff[e + 1] - 1) get token -1 and gate 0.
__global__ void bwd_rows_kernel(const int32_t* __restrict__ idx, const int32_t* __restrict__ inv,
                                const int32_t* __restrict__ counts, const int32_t* __restrict__ offsets,
                                const int32_t* __restrict__ poff, const float* __restrict__ gate,
                                int64_t n_slots, int k, int E, int32_t* __restrict__ ptok,
                                float* __restrict__ pgate, int32_t* __restrict__ slot_prow) {
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_slots) {
        const int e = idx[i];
        const int r = inv[i];
        if (e >= 0 && e < E && r >= 0) {
            const int pr = poff[e] + (r - offsets[e]);
            ptok[pr] = (int32_t)(i / k);
            pgate[pr] = gate[i];
            slot_prow[i] = pr;
        } else {
            slot_prow[i] = -1;
        }
    }
    if (i < (int64_t)E * 64) {
        const int e = (int)(i >> 6), j = (int)(i & 63);
        const int pr = poff[e] + counts[e] + j;
        if (pr < poff[e + 1]) {
            ptok[pr] = -1;
            pgate[pr] = 0.f;
        }
    }
}

// Clears in one launch, blockIdx.y the buffer: of out [G][M][ld] (fp32) every row of a group
// with gclear[g] set (or all rows, gclear == nullptr), and the pad columns [N, ld) of the
// other groups' rows (what a weight gradient's items will not write).  One warp per row,
// grid-strided; ld % 4 == 0.
__global__ void __launch_bounds__(256) bwd_zero_kernel(const __grid_constant__ BwdZero z) {
    pdl_wait();
    const BwdZeroJob& j = z.jobs[blockIdx.y];
    const int lane = threadIdx.x & 31;
    const int64_t rows = (int64_t)j.G * j.M;
    for (int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < rows;
         q += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        float* row = j.out + q * j.ld;
        if (!j.gclear || j.gclear[q / j.M]) {
            float4* r4 = reinterpret_cast<float4*>(row);
            for (int64_t c = lane; c < j.ld / 4; c += 32) r4[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            for (int64_t c = j.N + lane; c < j.ld; c += 32) row[c] = 0.f;
        }
    }
}

// Padded rows r (threads over r and 8-column groups): xp[r] = x[ptok[r]], gdy[r] =
// pgate[r] dy[ptok[r]] (bf16), zero rows where ptok[r] < 0.
__global__ void bwd_gather_kernel(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ dy,
                                  const int32_t* __restrict__ ptok, const float* __restrict__ pgate,
                                  const int32_t* __restrict__ poff, int E, int d,
                                  __nv_bfloat16* __restrict__ xp, __nv_bfloat16* __restrict__ gdy) {
    pdl_wait();
    const int64_t rows = poff[E];
    const int cpr = d / 8;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rows * cpr;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / cpr;
        const int c = (int)(i - r * cpr) * 8;
        const int t = ptok[r];
        uint4 xv = make_uint4(0u, 0u, 0u, 0u), gv = xv;
        if (t >= 0) {
            xv = *reinterpret_cast<const uint4*>(x + (int64_t)t * d + c);
            float f[8];
            unpack_bf16x8(*reinterpret_cast<const uint4*>(dy + (int64_t)t * d + c), f);
            const float g = pgate[r];
            gv.x = pack_bf16x2(g * f[0], g * f[1]);
            gv.y = pack_bf16x2(g * f[2], g * f[3]);
            gv.z = pack_bf16x2(g * f[4], g * f[5]);
            gv.w = pack_bf16x2(g * f[6], g * f[7]);
        }
        *reinterpret_cast<uint4*>(xp + r * d + c) = xv;
        *reinterpret_cast<uint4*>(gdy + r * d + c) = gv;
    }
}

// One warp per token (Eqs. 4-5 backward): dg_j = sum of the nparts partial row dots of
// its padded row, gdg = sum_j g_j dg_j, ds_j = sigma_j (1 - sigma_j) (dg_j - gdg) / S;
// dx_t += sum_j ds_j W_r[:, e_j] (after the grouped dx GEMM, same stream; four columns a
// lane and the k experts' loads together, 16 bytes each: with scalar loads the chain of
// d / 32 latencies took 42 us at T = 8192, d = 1024), and ds_j into ds[t][e_j] (bf16, the rest
// of the row already zero).
template <int KB>
__global__ void __launch_bounds__(256) bwd_router_kernel(
    const int32_t* __restrict__ idx, const float* __restrict__ sig, const float* __restrict__ gate,
    const int32_t* __restrict__ slot_prow, const float* __restrict__ dg_part, int nparts,
    int64_t part_stride, const float* __restrict__ wrt, int dp, int64_t T, int d, int E, int k,
    int Ep, float* __restrict__ dx, __nv_bfloat16* __restrict__ ds_out) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= T) return;
    // lanes j < k hold slot j: its dg, sigma and gate
    float dg = 0.f, sg = 0.f, g = 0.f;
    int e = -1;
    if (lane < k) {
        const int pr = slot_prow[t * k + lane];
        e = idx[t * k + lane];
        sg = sig[t * k + lane];
        g = gate[t * k + lane];
        if (pr >= 0)
            for (int q = 0; q < nparts; ++q) dg += dg_part[(int64_t)q * part_stride + pr];
    }
    const float S = warp_sum_f(sg);
    const float gdg = warp_sum_f(g * dg);
    const float ds = lane < k ? sg * (1.f - sg) * (dg - gdg) / S : 0.f;
    if (lane < k && e >= 0 && e < E) ds_out[t * Ep + e] = __float2bfloat16_rn(ds);
    const float* w[KB];   // past k and for bad ids: any row, with factor 0 and not added
    float dsj[KB];
    uint32_t okm = 0;
#pragma unroll
    for (int j = 0; j < KB; ++j) {
        dsj[j] = __shfl_sync(0xffffffffu, ds, j);
        const int ej = __shfl_sync(0xffffffffu, e, j);
        const bool ok = j < k && ej >= 0 && ej < E;
        if (ok) okm |= 1u << j;
        w[j] = wrt + (int64_t)(ok ? ej : 0) * dp;
    }
    float4* dxr = reinterpret_cast<float4*>(dx + t * d);   // d % 8 == 0, rows 16-byte aligned
    for (int i = lane; i < d / 4; i += 32) {
        float4 a = dxr[i];
        float4 v[KB];
#pragma unroll
        for (int j = 0; j < KB; ++j) v[j] = __ldg(reinterpret_cast<const float4*>(w[j]) + i);
#pragma unroll
        for (int j = 0; j < KB; ++j)
            if ((okm >> j) & 1u) {
                a.x = fmaf(dsj[j], v[j].x, a.x);
                a.y = fmaf(dsj[j], v[j].y, a.y);
                a.z = fmaf(dsj[j], v[j].z, a.z);
                a.w = fmaf(dsj[j], v[j].w, a.w);
            }
        dxr[i] = a;
    }
}

// dst[r][c] = src[r][c] for c < cols (src rows ld_src apart).
__global__ void bwd_copy_kernel(const float* __restrict__ src, int64_t ld_src, float* __restrict__ dst,
                                int64_t rows, int64_t cols) {
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rows * cols;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / cols, c = i - r * cols;
        dst[i] = src[r * ld_src + c];
    }
}

int grid_of(int64_t n, int threads) {
    int64_t g = (n + threads - 1) / threads;
    if (g > 152 * 16) g = 152 * 16;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace

cudaError_t launch_bwd_gates(const __nv_bfloat16* x, const float* wrt, int dp, const int32_t* idx, int64_t T,
                             int d, int E, int k, float* sig, float* gate, DevStatus* st, cudaStream_t s) {
    const dim3 grid((unsigned)((T * 32 + 255) / 256));
    cudaError_t e;
    using Kern = decltype(&bwd_gates_kernel<1, false, 4, 4>);
    static const Kern kerns[9] = {
        bwd_gates_kernel<8, true, 2, 4>,
        bwd_gates_kernel<1, false, 8, 4>, bwd_gates_kernel<2, false, 4, 4>, bwd_gates_kernel<3, false, 4, 4>,
        bwd_gates_kernel<4, false, 4, 4>, bwd_gates_kernel<5, false, 2, 4>, bwd_gates_kernel<6, false, 2, 4>,
        bwd_gates_kernel<7, false, 2, 4>, bwd_gates_kernel<8, false, 2, 4>};
    if (k < 1 || k > 32) return cudaErrorInvalidValue;
    const Kern kern = kerns[k <= 8 ? k : 0];
    e = launch_pdl(kern, grid, dim3(256), 0, s, x, wrt, dp, idx, T, d, E, k, sig, gate, st);
    count_launches(1);
    return e;
}

cudaError_t launch_bwd_plan(const BwdPlan& p, cudaStream_t s) {
    if (p.E > 1024 || p.nsets < 0 || p.nsets > BWD_MAX_SETS) return cudaErrorInvalidValue;
    const cudaError_t e = launch_pdl(bwd_plan_kernel, dim3(1 + p.nsets), dim3(1024), 0, s, p);
    count_launches(1);
    return e;
}

cudaError_t launch_bwd_rows(const int32_t* idx, const int32_t* inv, const int32_t* counts,
                            const int32_t* offsets, const int32_t* poff, const float* gate, int64_t n_slots,
                            int k, int E, int32_t* ptok, float* pgate, int32_t* slot_prow, cudaStream_t s) {
    const int64_t n = n_slots > (int64_t)E * 64 ? n_slots : (int64_t)E * 64;
    const cudaError_t e = launch_pdl(bwd_rows_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, s, idx,
                                     inv, counts, offsets, poff, gate, n_slots, k, E, ptok, pgate, slot_prow);
    count_launches(1);
    return e;
}

int64_t bwd_max_items(int64_t rows, int G, int M, int N, int BN) {
    const int64_t mt = (M + GM_BM - 1) / GM_BM, nt = (N + BN - 1) / BN;
    return ((rows + GM_BK * BWD_KCH - 1) / (GM_BK * BWD_KCH) + G) * mt * nt;
}

cudaError_t launch_bwd_zero(const BwdZero& z, int num_sms, cudaStream_t s) {
    int64_t rows = 1;
    for (int j = 0; j < z.njobs; ++j) {
        if (z.jobs[j].ld % 4 != 0 || z.jobs[j].N > z.jobs[j].ld) return cudaErrorInvalidValue;
        rows = std::max<int64_t>(rows, (int64_t)z.jobs[j].G * z.jobs[j].M);
    }
    if (z.njobs < 1 || z.njobs > BWD_MAX_ZERO) return cudaErrorInvalidValue;
    const int64_t blocks = std::min<int64_t>((rows + 7) / 8, (int64_t)num_sms * 8);
    const cudaError_t e = launch_pdl(bwd_zero_kernel, dim3((unsigned)blocks, (unsigned)z.njobs), dim3(256), 0, s, z);
    count_launches(1);
    return e;
}

cudaError_t launch_bwd_gather(const __nv_bfloat16* x, const __nv_bfloat16* dy, const int32_t* ptok,
                              const float* pgate, const int32_t* poff, int E, int d, int64_t max_rows,
                              __nv_bfloat16* xp, __nv_bfloat16* gdy, cudaStream_t s) {
    const cudaError_t e = launch_pdl(bwd_gather_kernel, dim3(grid_of(max_rows * (d / 8), 256)), dim3(256), 0, s,
                                     x, dy, ptok, pgate, poff, E, d, xp, gdy);
    count_launches(1);
    return e;
}

cudaError_t launch_bwd_router(const int32_t* idx, const float* sig, const float* gate, const int32_t* slot_prow,
                              const float* dg_part, int nparts, int64_t part_stride, const float* wrt, int dp,
                              int64_t T, int d, int E, int k, int Ep, float* dx, __nv_bfloat16* ds,
                              cudaStream_t s) {
    const dim3 grid((unsigned)((T * 32 + 255) / 256));
    cudaError_t e;
    if (k <= 4)
        e = launch_pdl(bwd_router_kernel<4>, grid, dim3(256), 0, s, idx, sig, gate, slot_prow, dg_part, nparts,
                       part_stride, wrt, dp, T, d, E, k, Ep, dx, ds);
    else if (k <= 8)
        e = launch_pdl(bwd_router_kernel<8>, grid, dim3(256), 0, s, idx, sig, gate, slot_prow, dg_part, nparts,
                       part_stride, wrt, dp, T, d, E, k, Ep, dx, ds);
    else if (k <= 32)
        e = launch_pdl(bwd_router_kernel<32>, grid, dim3(256), 0, s, idx, sig, gate, slot_prow, dg_part, nparts,
                       part_stride, wrt, dp, T, d, E, k, Ep, dx, ds);
    else
        return cudaErrorInvalidValue;
    count_launches(1);
    return e;
}

cudaError_t launch_bwd_copy(const float* src, int64_t ld_src, float* dst, int64_t rows, int64_t cols,
                            cudaStream_t s) {
    const cudaError_t e = launch_pdl(bwd_copy_kernel, dim3(grid_of(rows * cols, 256)), dim3(256), 0, s, src,
                                     ld_src, dst, rows, cols);
    count_launches(1);
    return e;
}

}  // namespace mv
