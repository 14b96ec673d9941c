// route.cu -- router of the MoE-ViE layer (Eqs. 1, 7, 4-5), sm_103a.
//
// The logits s = x . W_r run on the tensor cores (grouped_gemm_kernel, one dense
// group): W_r is split exactly into bf16 pieces, W_r = hi + mid + lo, and the GEMM
// accumulates the fast logits x . (hi + mid) in fp32 (each piece padded to a multiple of
// 64 rows with zeros; for E <= 128 the two pieces sit side by side along N and the
// epilogue adds them, otherwise one after another along K).  Every product of a bf16 x
// and a bf16 piece is exact in fp32, so the error is the fp32 accumulation plus the
// left-out x . lo, which Cauchy-Schwarz bounds by |x_t| |lo_e| (lo holds the last 8 of
// w's 24 significand bits).  When there are few tokens, K is split over several CTA
// pairs (route_ksplit) and each split writes its own fp32 partial logits; they are summed
// in a fixed order.  This file holds the steps around that GEMM:
//
//  1. route_split_kernel: the two pieces, an fp32 copy of W_r transposed to
//     [E][d_pad] (read by the exact re-decision), and per-CTA partial sums of squares
//     of W_r's columns and of lo's (the router GEMM's idle warps finish |W_r[:, e]| and
//     |lo_e| from them).
//  2. route_topk_kernel: one warp per token; the partial logits summed, keys
//     sigmoid(s) + b, k rounds of warp arg-max (ties to the lower id), and a
//     certificate.  Every expert's key lies in
//     [key_e - tau_e, key_e + tau_e]; tau_e is the logit error bound (logit_tau) times
//     the largest sigmoid slope inside the logit interval, plus fp32 evaluation slack.
//     The selection is certain when the lowest selected lower end is above the highest
//     unselected upper end (tried first with the slope bound 1/4, then with the exact
//     slope).  Certified tokens write ascending ids and gates sigmoid(s) / sum (the bias
//     only selects).
//  3. route_fallback_kernel: one CTA per uncertified token.  An expert is surely in
//     when its lower end is above the k-th largest upper end of the others, surely
//     out when its upper end is below the k-th largest lower end; the rest get exact
//     logits (each product of a bf16 and an fp32 value is an integer of at most 32 bits
//     times a power of two; the CTA sums them in 128-bit fixed-point accumulators on
//     the integer pipes, see long_acc_term), and the remaining places are filled from
//     their keys (fp64), ties to the lower id.
//
// Small problems take one launch instead (route_small_kernel, launch_route_small): fp32 logits
// on the FMA pipes, the same certified selection and the same exact re-decision.
#include <math.h>

#include <algorithm>

#include "internal.h"

namespace mv {

namespace {

constexpr int SPLIT_TILE = 32;    // W_r rows (and experts) per CTA of the split kernel

// CTA (bx, by): experts 32 bx .. +31 and rows 32 by .. +31 of W_r (rows past d are
// zero); 32 x 8 threads.  Writes the two bf16 pieces hi, mid, the transposed fp32 copy
// and the CTA's partial sums of w^2 and of lo^2 per expert (lo = w - hi - mid, the
// piece the fast logits leave out).
__global__ void __launch_bounds__(256) route_split_kernel(const float* __restrict__ Wr, int d,
                                                          int dp, int E, int Ep,
                                                          __nv_bfloat16* __restrict__ Wsplit,
                                                          float* __restrict__ wrt,
                                                          float* __restrict__ wpart, int parts,
                                                          int32_t* __restrict__ wexp,
                                                          DevStatus* st, int concat) {
    pdl_wait();
    if (st && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) st->fb_count = 0;
    __shared__ float tile[SPLIT_TILE][SPLIT_TILE + 1];
    __shared__ float red[2][8][32];
    __shared__ int redx[8][32];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int e = blockIdx.x * SPLIT_TILE + tx;
    const int i0 = blockIdx.y * SPLIT_TILE;
    // piece p of element (i, e): [p][dp][Ep] (along K), or [dp][2 Ep] (side by side along N)
    const size_t piece = concat ? (size_t)Ep : (size_t)dp * Ep;
    const size_t row = concat ? (size_t)2 * Ep : (size_t)Ep;
    float sq = 0.f, sql = 0.f;
    int ex = 1;   // largest exponent field (subnormals and zero count as 1)
#pragma unroll
    for (int r = ty; r < SPLIT_TILE; r += 8) {
        const int i = i0 + r;
        const float w = (e < E && i < d) ? Wr[(int64_t)i * E + e] : 0.f;
        ex = max(ex, (int)((__float_as_uint(w) >> 23) & 0xffu));
        const __nv_bfloat16 hi = __float2bfloat16_rn(w);
        const float r1 = w - __bfloat162float(hi);                 // exact
        const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
        const float lo = r1 - __bfloat162float(mid);               // exact
        if (e < Ep) {
            const size_t o = (size_t)i * row + e;
            Wsplit[o] = hi;
            Wsplit[piece + o] = mid;
        }
        tile[r][tx] = w;
        sq = fmaf(w, w, sq);
        sql = fmaf(lo, lo, sql);
    }
    red[0][ty][tx] = sq;
    red[1][ty][tx] = sql;
    redx[ty][tx] = ex;
    __syncthreads();
    if (ty < 2 && e < Ep) {
        float v = 0.f;
        for (int q = 0; q < 8; ++q) v += red[ty][q][tx];
        wpart[((int64_t)ty * parts + blockIdx.y) * Ep + e] = v;
    } else if (ty == 2 && e < Ep) {
        int m = 1;
        for (int q = 0; q < 8; ++q) m = max(m, redx[q][tx]);
        wexp[(int64_t)blockIdx.y * Ep + e] = m;
    }
#pragma unroll
    for (int r = ty; r < SPLIT_TILE; r += 8) {
        const int ee = blockIdx.x * SPLIT_TILE + r;
        if (ee < E) wrt[(int64_t)ee * dp + i0 + tx] = tile[tx][r];
    }
}

// Fast sigmoid: __expf (ex2.approx) and __fdividef.  For the keys compared below
// its absolute error stays under 1e-6, inside ROUTE_KEY_SLACK (2e-6): the relative
// error of e^{-v} is at most |v| log2(e) 2^-24 + 2^-22 and enters the sigmoid
// multiplied by s(1 - s) <= 1/4 (and by e^{-|v|} for large |v|); the division adds
// two ulp.
__device__ __forceinline__ float sigmoid_fast(float v) {
    return __fdividef(1.0f, 1.0f + __expf(-v));
}

// Logit error bound of expert e for a token (internal.h): the accumulation error
// ROUTE_TAU_C 2^-24 |x_t| (|W_r[:, e]| + |lo_e|) plus the left-out piece |x_t| |lo_e|,
// rounded up by the factor 1.001: the norms are fp32 sums of squares along chains far
// shorter than 2^14 terms, so their relative error (and that of the few operations
// here) stays below 2^-10.
__device__ __forceinline__ float logit_tau(float xn, float wn, float wl) {
    return (ROUTE_TAU_C * 5.9604645e-8f * (wn + wl) + wl) * xn * 1.001f;
}

// Key half-width with the largest sigmoid slope inside [s - tau_s, s + tau_s]
// (the slope s(1 - s) falls with |s|).
__device__ __forceinline__ float key_tau_exact_slope(float s, float tau_s) {
    const float z = fmaxf(fabsf(s) - tau_s, 0.f);
    const float sz = sigmoid_fast(z);
    return tau_s * (sz * (1.f - sz)) + ROUTE_KEY_SLACK;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Order-preserving code of a float (larger float, larger code; an arithmetic NaN above all).
__device__ __forceinline__ uint32_t ord_f32(float f) {
    const uint32_t u = __float_as_uint(f);
    return u ^ ((u & 0x80000000u) ? 0xffffffffu : 0x80000000u);
}

__device__ __forceinline__ float from_ord_f32(uint32_t c) {
    return __uint_as_float(c ^ ((c & 0x80000000u) ? 0x80000000u : 0xffffffffu));
}

// k-th and (k+1)-th largest of v over the warp, counting equal values separately
// (k or k + 1 rounds: warp maximum of the order codes by redux.sync, then one holder
// of that maximum leaves; k <= E).
template <int NPL>
__device__ __forceinline__ void warp_kth_values(const float (&v)[NPL], int E, int k, int lane,
                                                float& kth, float& kth1) {
    uint32_t code[NPL];
#pragma unroll
    for (int i = 0; i < NPL; ++i) code[i] = (lane + 32 * i < E) ? ord_f32(v[i]) : 0u;
    uint32_t used = 0;
    kth = -INFINITY;
    kth1 = -INFINITY;
    const int rounds = k < E ? k + 1 : k;
    for (int j = 0; j < rounds; ++j) {
        uint32_t best = 0;
#pragma unroll
        for (int i = 0; i < NPL; ++i) {
            const uint32_t c = ((used >> i) & 1u) ? 0u : code[i];
            best = c > best ? c : best;
        }
        best = __reduce_max_sync(0xffffffffu, best);
#pragma unroll
        for (int i = 0; i < NPL; ++i) {
            const uint32_t m = __ballot_sync(0xffffffffu, !((used >> i) & 1u) && code[i] == best);
            if (m) {
                if (lane == __ffs(m) - 1) used |= 1u << i;
                break;
            }
        }
        const float bv = from_ord_f32(best);
        if (j == k - 1) kth = bv;
        if (j == k) kth1 = bv;
    }
}

// Exact logits by a long fixed-point accumulator (the exact dot product of Kulisch
// and Miranker, with a window fitted to the operands).  A bf16 x_i is mx 2^(ex - 134)
// and an fp32 w_i is mw 2^(ew - 150) (mx < 2^8, mw < 2^24 integers; ex, ew the biased
// exponents, 1 for subnormals), so x_i w_i = P 2^(q - 284) with the integer P = mx mw
// < 2^32 and q = ex + ew.  With a window Q >= every q, the term is P 2^(64 - (Q - q))
// units of 2^(Q - 348): a left shift (exact) when Q - q <= 64, else a right shift that
// drops less than one unit.  The units of d terms sum in a 128-bit integer (|sum| <
// 2^120 for d < 2^24), exactly and in any order; the logit is that sum times
// 2^(Q - 348), within d 2^(Q - 348) + 2^-51 |s| of the exact value.  Everything but the
// final conversion runs on the integer pipes.
__device__ __forceinline__ int bf16_exp_field(uint32_t hx) { return (int)((hx >> 7) & 0xffu); }
__device__ __forceinline__ int f32_exp_field(uint32_t uw) { return (int)((uw >> 23) & 0xffu); }

// x as its signed mantissa and its exponent (1 at least), w the same way.
__device__ __forceinline__ void long_acc_x(uint32_t hx, int& mx, int& ex) {
    const int e = bf16_exp_field(hx), m = (int)((hx & 0x7fu) | (e ? 0x80u : 0u));
    mx = hx & 0x8000u ? -m : m;
    ex = max(e, 1);
}
__device__ __forceinline__ void long_acc_w(uint32_t uw, int& mw, int& ew) {
    const int e = f32_exp_field(uw), m = (int)((uw & 0x7fffffu) | (e ? 0x800000u : 0u));
    mw = (int)uw < 0 ? -m : m;
    ew = max(e, 1);
}
// acc += mx mw 2^sh (sh <= 64; below 0 the magnitude's dropped bits are less than one unit).  The
// product (33 bits with its sign) and its two shifts are 64-bit; PTX clamps a shift by 64 or more.
__device__ __forceinline__ void long_acc_add(int mx, int mw, int sh, unsigned __int128& acc) {
    int64_t p = (int64_t)mx * mw;
    if (sh < 0) {   // rare: a term 2^64 times smaller than the largest it might have been
        const int64_t m = (p < 0 ? -p : p) >> min(-sh, 63);
        p = p < 0 ? -m : m;
        sh = 0;
    }
    uint64_t lo, hi;
    asm("shl.b64 %0, %1, %2;" : "=l"(lo) : "l"(p), "r"(sh));
    asm("shr.s64 %0, %1, %2;" : "=l"(hi) : "l"(p), "r"(64 - sh));
    acc += ((unsigned __int128)hi << 64) | lo;
}
// acc += x w in units of 2^(Q - 348) (hx: bf16 bits of x, uw: fp32 bits of w).
__device__ __forceinline__ void long_acc_term(uint32_t hx, uint32_t uw, int Q, unsigned __int128& acc) {
    int mx, ex, mw, ew;
    long_acc_x(hx, mx, ex);
    long_acc_w(uw, mw, ew);
    long_acc_add(mx, mw, 64 - Q + ex + ew, acc);
}

__device__ __forceinline__ unsigned __int128 warp_sum_u128(unsigned __int128 v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const uint64_t lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)(uint64_t)v, o);
        const uint64_t hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(uint64_t)(v >> 64), o);
        v += ((unsigned __int128)hi << 64) | lo;
    }
    return v;
}

// The signed 128-bit sum `u` (two's complement) times 2^(Q - 348), in double: the
// magnitude's two 64-bit words are rounded and added (relative error below 3 2^-53).
__device__ __forceinline__ double long_acc_value(unsigned __int128 u, int Q) {
    const bool neg = (long long)(uint64_t)(u >> 64) < 0;
    const unsigned __int128 m = neg ? (unsigned __int128)0 - u : u;
    const double hi = (double)(unsigned long long)(uint64_t)(m >> 64);
    const double lo = (double)(unsigned long long)(uint64_t)m;
    const double v = fma(hi, 18446744073709551616.0, lo);   // hi 2^64 + lo
    // 2^(Q - 348) with 2 <= Q <= 508: a normal double, so the product is exact
    const double r = v * __longlong_as_double((long long)((uint64_t)(Q - 348 + 1023) << 52));
    return neg ? -r : r;
}

// The k experts of largest key sigmoid(s) + b of one token (a warp; expert e sits in lane
// e % 32, slot e / 32), ties to the lower id, and whether the logit error bounds ts certify
// them.  Each of the k selection rounds takes the warp maximum of the keys' order codes
// (redux.sync) and then the lowest id holding it (ballots in slot order).
template <int NPL>
__device__ __forceinline__ bool select_certified(const float (&sv)[NPL], const float (&ts)[NPL],
                                                 const float* __restrict__ b, int E, int k, int lane,
                                                 float (&sg)[NPL], uint32_t& taken) {
    float key[NPL];
    uint32_t code[NPL];
#pragma unroll
    for (int i = 0; i < NPL; ++i) {
        const int e = lane + 32 * i;
        if (e < E) {
            sg[i] = sigmoid_fast(sv[i]);
            key[i] = sg[i] + b[e];
            code[i] = ord_f32(key[i]);
        } else {
            sg[i] = 0.f;
            key[i] = -INFINITY;
            code[i] = 0;
        }
    }
    taken = 0;
    for (int j = 0; j < k; ++j) {
        uint32_t best = 0;
#pragma unroll
        for (int i = 0; i < NPL; ++i) {
            const uint32_t c = ((taken >> i) & 1u) ? 0u : code[i];
            best = c > best ? c : best;
        }
        best = __reduce_max_sync(0xffffffffu, best);
#pragma unroll
        for (int i = 0; i < NPL; ++i) {
            const uint32_t m = __ballot_sync(0xffffffffu, !((taken >> i) & 1u) && code[i] == best);
            if (m) {
                if (lane == __ffs(m) - 1) taken |= 1u << i;
                break;
            }
        }
    }
    bool certain = k >= E;
    for (int pass = 0; pass < 2 && !certain; ++pass) {
        float lo_in = INFINITY, hi_out = -INFINITY;
#pragma unroll
        for (int i = 0; i < NPL; ++i) {
            const int e = lane + 32 * i;
            if (e >= E) continue;
            const float tk = pass == 0 ? 0.25f * ts[i] + ROUTE_KEY_SLACK
                                       : key_tau_exact_slope(sv[i], ts[i]);
            if ((taken >> i) & 1u) lo_in = fminf(lo_in, key[i] - tk);
            else hi_out = fmaxf(hi_out, key[i] + tk);
        }
        certain = __reduce_min_sync(0xffffffffu, ord_f32(lo_in)) >
                  __reduce_max_sync(0xffffffffu, ord_f32(hi_out));
    }
    return certain;
}

// Ascending ids of the selected experts and their gates sigmoid(s) / sum.
template <int NPL>
__device__ __forceinline__ void write_selection(uint32_t taken, const float (&sg)[NPL], int64_t t, int k, int lane,
                                                int32_t* __restrict__ idx, float* __restrict__ gate) {
    float ssum = 0.f;
#pragma unroll
    for (int i = 0; i < NPL; ++i) ssum += ((taken >> i) & 1u) ? sg[i] : 0.f;
    ssum = warp_sum(ssum);
    const uint32_t lt = (1u << lane) - 1u;
    int base = 0;
#pragma unroll
    for (int i = 0; i < NPL; ++i) {
        const uint32_t m = __ballot_sync(0xffffffffu, (taken >> i) & 1u);
        const int pos = base + __popc(m & lt);
        if (((taken >> i) & 1u) && pos < k) {   // (there are k)
            idx[t * k + pos] = lane + 32 * i;
            gate[t * k + pos] = __fdividef(sg[i], ssum);
        }
        base += __popc(m);
    }
}

// One warp per token.  NPL = experts per lane (expert e sits in lane e % 32, slot e / 32).
// s holds nparts partial logit arrays, part p at s + p * part_stride.
// A token the certificate cannot settle is listed for route_fallback_kernel.
template <int NPL>
__global__ void __launch_bounds__(256) route_topk_kernel(
    const __nv_bfloat16* __restrict__ x, float* __restrict__ s, int ld, int nparts,
    int64_t part_stride, const float* __restrict__ b, const float* __restrict__ wnorm, int T,
    int d, int E, int k, int32_t* __restrict__ idx, float* __restrict__ gate,
    const float* __restrict__ xnorm, int32_t* __restrict__ fb_tokens, DevStatus* st,
    float4* __restrict__ zero, int64_t zero_n4) {
    pdl_wait();
    // Side job: clear another buffer (the layer's fp32 y accumulator) with 16-byte
    // evict-first stores, grid-strided; this kernel leaves HBM mostly idle.
    if (zero) {
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        const uint64_t pol = l2_policy_evict_first();
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < zero_n4;
             i += (int64_t)gridDim.x * blockDim.x)
            st_global_v4_hint(zero + i, z, pol);
    }
    const int lane = threadIdx.x & 31;
    const int t = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (t >= T) return;
    float* srow = s + (int64_t)t * ld;
    float sv[NPL];
#pragma unroll
    for (int i = 0; i < NPL; ++i) {
        const int e = lane + 32 * i;
        sv[i] = e < E ? srow[e] : 0.f;
    }
    for (int q = 1; q < nparts; ++q) {
#pragma unroll
        for (int i = 0; i < NPL; ++i) {
            const int e = lane + 32 * i;
            if (e < E) sv[i] += srow[q * part_stride + e];
        }
    }
    const float xn = xnorm[t];   // |x_t|, written by the router GEMM
    float sg[NPL], ts[NPL];
#pragma unroll
    for (int i = 0; i < NPL; ++i) {
        const int e = lane + 32 * i;
        ts[i] = e < E ? logit_tau(xn, wnorm[e], wnorm[E + e]) : 0.f;
    }
    uint32_t taken;
    const bool certain = select_certified<NPL>(sv, ts, b, E, k, lane, sg, taken);
    if (!certain) {
        if (nparts > 1) {   // the re-decision reads the summed logits from part 0
#pragma unroll
            for (int i = 0; i < NPL; ++i) {
                const int e = lane + 32 * i;
                if (e < E) srow[e] = sv[i];
            }
        }
        if (lane == 0) {
            const int p = atomicAdd(&st->fb_count, 1);
            fb_tokens[p] = t;
        }
        return;
    }
    write_selection<NPL>(taken, sg, t, k, lane, idx, gate);
}


// The two warp steps of an exact re-decision.  First, from the fast logits sv and their error
// bounds ts (slots past E get anything): the experts that are surely in, and the candidates for
// the remaining places.
template <int NPL>
__device__ __forceinline__ void bound_candidates(const float (&sv)[NPL], const float (&ts)[NPL],
                                                 const float* __restrict__ b, int E, int k, int lane,
                                                 uint32_t& sure_in, uint32_t& cand) {
    float up[NPL], lo[NPL];
#pragma unroll
    for (int i = 0; i < NPL; ++i) {
        const int e = lane + 32 * i;
        if (e < E) {
            const float key = sigmoid_fast(sv[i]) + b[e];
            const float tk = key_tau_exact_slope(sv[i], ts[i]);
            up[i] = key + tk;
            lo[i] = key - tk;
        } else {
            up[i] = lo[i] = -INFINITY;
        }
    }
    // k-th / (k+1)-th largest upper ends and k-th largest lower end
    float u_k, u_k1, l_k, l_k1;
    warp_kth_values<NPL>(up, E, k, lane, u_k, u_k1);
    warp_kth_values<NPL>(lo, E, k, lane, l_k, l_k1);
    sure_in = cand = 0;
#pragma unroll
    for (int i = 0; i < NPL; ++i) {
        const int e = lane + 32 * i;
        if (e >= E) continue;
        // k-th largest upper end among the others (u_k when e may sit at rank k: conservative)
        const float thr = up[i] > u_k ? u_k1 : u_k;
        if (k >= E || lo[i] > thr) sure_in |= 1u << i;
        else if (!(up[i] < l_k)) cand |= 1u << i;
    }
}
// Order code of a key in 64 bits (larger key, larger code, above 0); NaN above all, as in ord_f32:
// the order has to be total, or the lanes would disagree on the choice.
__device__ __forceinline__ uint64_t ord_f64(double v) {
    const uint64_t u = (uint64_t)__double_as_longlong(v);
    return v != v ? ~0ull : u ^ (u >> 63 ? ~0ull : 1ull << 63);
}
// Then, with the candidates' exact keys: `need` of them (no more than there are) by key, ties to
// the lower id; exactly one a round, whatever the keys are.
template <int NPL>
__device__ __forceinline__ uint32_t choose_exact(const double (&exk)[NPL], uint32_t sure_in, uint32_t cand, int need,
                                                 int lane) {
    uint32_t chosen = sure_in;
    for (int r = 0; r < need; ++r) {
        uint64_t bv = 0;
        int bi = 0x7fffffff;
#pragma unroll
        for (int i = 0; i < NPL; ++i) {
            const uint64_t v = ((cand & ~chosen) >> i) & 1u ? ord_f64(exk[i]) : 0;
            if (v > bv) {
                bv = v;
                bi = lane + 32 * i;
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const uint64_t ov = __shfl_xor_sync(0xffffffffu, (unsigned long long)bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ov > bv || (ov == bv && oi < bi)) {
                bv = ov;
                bi = oi;
            }
        }
        if ((bi & 31) == lane && bv) chosen |= 1u << (bi >> 5);
    }
    return chosen;
}

// Exact re-decision of the uncertified tokens, a CTA of 8 warps per token.  The CTA stages
// the token's x row in shared memory (16-byte loads) and finds its largest exponent
// field; warp 0 bounds the keys and lists the candidates; then the candidates' exact
// logits are formed FB_BATCH at a time by all 256 threads (threads over the d terms,
// one long accumulator per candidate and thread, then a warp sum and a sum over the 8
// warps, all exact), their keys in fp64; finally warp 0 fills the remaining places from
// the exact keys, ties to the lower id, and writes ids and gates.
//
// The window of candidate e is Q = qx + qw(e), qx the largest exponent field of x_t and
// qw(e) that of W_r[:, e] (both at least 1: subnormals and zeros count as exponent 1), so
// every term's q is at most Q and one pass over the terms suffices; the logit is within
// d 2^(Q - 348) + 2^-51 |s| of the exact value, and d 2^(Q - 348) <= d 2^-64
// |x_t|_inf |W_r[:, e]|_inf.  A non-finite x_t or column (exponent field 255) gives a
// NaN logit.
constexpr int FB_BATCH = 4;       // candidates per pass over the terms
constexpr int FB_X_SMEM = 16384;  // largest d whose x row is staged in shared memory
// CTAs per SM the re-decision keeps resident for E <= 256 (its registers allow five), so
// that up to five tokens per SM are re-decided at once
constexpr int FB_CTAS_PER_SM = 5;

// Largest exponent field of the eight bf16 values in v.
__device__ __forceinline__ int bf16x8_exp_max(const uint4& v) {
    const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
    int m = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) m = max(m, max((int)((w4[j] >> 7) & 0xffu), (int)((w4[j] >> 23) & 0xffu)));
    return m;
}

template <int NPL>
__global__ void __launch_bounds__(256, (NPL <= 8 ? FB_CTAS_PER_SM : 1)) route_fallback_kernel(
    const __nv_bfloat16* __restrict__ x, const float* __restrict__ wrt, int dp,
    const int32_t* __restrict__ wexp, int wexp_parts, int Ep,
    const float* __restrict__ b, const float* __restrict__ s, int ld,
    const float* __restrict__ xnorm, const float* __restrict__ wnorm, int d, int E, int k,
    int32_t* __restrict__ idx, float* __restrict__ gate, const int32_t* __restrict__ fb_tokens,
    DevStatus* st) {
    pdl_wait();
    extern __shared__ __align__(16) uint16_t fb_x[];   // the token's x row when d <= FB_X_SMEM
    __shared__ int s_cand[32 * NPL];
    __shared__ double s_key[32 * NPL];
    __shared__ unsigned long long s_acc[8][FB_BATCH][2];
    __shared__ int s_q[FB_BATCH];
    __shared__ int s_ncand, s_qx;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const int nfb = st->fb_count;
    const bool staged = d <= FB_X_SMEM;
    for (int f = blockIdx.x; f < nfb; f += gridDim.x) {
        const int t = fb_tokens[f];
        const uint16_t* xg = reinterpret_cast<const uint16_t*>(x) + (int64_t)t * d;
        if (threadIdx.x == 0) s_qx = 1;
        __syncthreads();
        if (warp > 0 || !staged) {   // warps 1-7 stage x_t while warp 0 bounds the keys
            int m = 1;
            const int nthr = staged ? (int)blockDim.x - 32 : (int)blockDim.x;
            const int tid = staged ? (int)threadIdx.x - 32 : (int)threadIdx.x;
            for (int i = tid; i < d / 8; i += nthr) {   // d % 8 == 0, rows 16-byte aligned
                const uint4 v = reinterpret_cast<const uint4*>(xg)[i];
                if (staged) reinterpret_cast<uint4*>(fb_x)[i] = v;
                m = max(m, bf16x8_exp_max(v));
            }
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) atomicMax(&s_qx, m);
        }
        float sv[NPL];
        uint32_t sure_in = 0, cand = 0;
        int need = 0;
        if (warp == 0) {
            float ts[NPL];
            const float xn = xnorm[t];
#pragma unroll
            for (int i = 0; i < NPL; ++i) {
                const int e = lane + 32 * i;
                sv[i] = e < E ? s[(int64_t)t * ld + e] : 0.f;
                ts[i] = e < E ? logit_tau(xn, wnorm[e], wnorm[E + e]) : 0.f;
            }
            bound_candidates<NPL>(sv, ts, b, E, k, lane, sure_in, cand);
            int n_in = 0, n_cand = 0;
#pragma unroll
            for (int i = 0; i < NPL; ++i) {
                n_in += __popc(__ballot_sync(0xffffffffu, (sure_in >> i) & 1u));
                const uint32_t m = __ballot_sync(0xffffffffu, (cand >> i) & 1u);
                if ((cand >> i) & 1u) s_cand[n_cand + __popc(m & lt)] = lane + 32 * i;
                n_cand += __popc(m);
            }
            need = k - n_in;
            const bool bad = need < 0 || need > n_cand;
            if (lane == 0) {
                if (bad) report(st, MOEVIE_ERR_DEVICE, SITE_ROUTE_FALLBACK, t, need);
                s_ncand = bad ? -1 : (need == 0 ? 0 : n_cand);
            }
        }
        __syncthreads();
        const int nc = s_ncand;
        const int qx = s_qx;
        const uint16_t* xs = staged ? fb_x : xg;
        for (int c0 = 0; c0 < nc; c0 += FB_BATCH) {
            const int cn = min(FB_BATCH, nc - c0);
            if (warp < cn) {   // warp c: the window of candidate c0 + c
                const int e = s_cand[c0 + warp];
                int qw = 1;
                for (int pp = lane; pp < wexp_parts; pp += 32) qw = max(qw, __ldg(wexp + (int64_t)pp * Ep + e));
                qw = __reduce_max_sync(0xffffffffu, qw);
                if (lane == 0) s_q[warp] = (qx == 255 || qw == 255) ? -1 : qx + qw;   // -1: NaN
            }
            __syncthreads();
            unsigned __int128 acc[FB_BATCH];
            int Q[FB_BATCH];
            int ec[FB_BATCH];
#pragma unroll
            for (int c = 0; c < FB_BATCH; ++c) {
                acc[c] = 0;
                Q[c] = c < cn ? s_q[c] : -1;
                ec[c] = s_cand[c0 + (c < cn ? c : 0)];
            }
            for (int i = threadIdx.x; i < d; i += blockDim.x) {
                const uint32_t hx = xs[i];
                uint32_t uw[FB_BATCH];
#pragma unroll
                for (int c = 0; c < FB_BATCH; ++c) uw[c] = Q[c] > 0 ? __float_as_uint(__ldg(wrt + (int64_t)ec[c] * dp + i)) : 0u;
#pragma unroll
                for (int c = 0; c < FB_BATCH; ++c)
                    if (Q[c] > 0) long_acc_term(hx, uw[c], Q[c], acc[c]);
            }
#pragma unroll
            for (int c = 0; c < FB_BATCH; ++c) {
                if (Q[c] <= 0) continue;   // uniform over the CTA
                const unsigned __int128 a = warp_sum_u128(acc[c]);
                if (lane == 0) {
                    s_acc[warp][c][0] = (unsigned long long)(uint64_t)a;
                    s_acc[warp][c][1] = (unsigned long long)(uint64_t)(a >> 64);
                }
            }
            __syncthreads();
            if (warp == 0 && lane < cn) {   // candidate c0 + lane: the sum over the 8 warps
                const int q = s_q[lane];
                double v = __longlong_as_double(0x7ff8000000000000ll);
                if (q > 0) {
                    unsigned __int128 u = 0;
#pragma unroll
                    for (int ww = 0; ww < 8; ++ww)
                        u += ((unsigned __int128)s_acc[ww][lane][1] << 64) | s_acc[ww][lane][0];
                    v = long_acc_value(u, q);
                }
                s_key[c0 + lane] = 1.0 / (1.0 + exp(-v)) + (double)b[s_cand[c0 + lane]];
            }
            __syncthreads();
        }
        if (warp == 0 && nc >= 0) {
            double exk[NPL];
            int base = 0;
#pragma unroll
            for (int i = 0; i < NPL; ++i) {
                const uint32_t m = __ballot_sync(0xffffffffu, (cand >> i) & 1u);
                exk[i] = ((cand >> i) & 1u && nc > 0) ? s_key[base + __popc(m & lt)] : -INFINITY;
                base += __popc(m);
            }
            const uint32_t chosen = choose_exact<NPL>(exk, sure_in, cand, need, lane);
            float sg[NPL];
#pragma unroll
            for (int i = 0; i < NPL; ++i) sg[i] = ((chosen >> i) & 1u) ? sigmoid_fast(sv[i]) : 0.f;
            write_selection<NPL>(chosen, sg, t, k, lane, idx, gate);
        }
        __syncthreads();   // the shared arrays are reused by the next token
    }
}

// The whole router of a layer with few tokens x experts x d in one launch: fp32 logits on the
// FMA pipes straight from W_r, the certified top-k, and the exact re-decision.  The
// tensor-core route (split of W_r, GEMM, top-k, re-decision) is four dependent launches, 17.5
// us at T = 512, d = 768, E = 16 and 18.0 at T = 256, E = 31 (back to back calls); this kernel
// takes 10.5 (the rate of the calls) and 12.8.  A CTA of 8 warps takes up to 8 tokens, each warp an
// eighth of d: chunks of CH rows of W_r and columns of x go through registers (one chunk
// ahead) into the warp's shared memory as fp32, and each lane forms one token x 8 NE experts
// with packed FMAs (lane = 4 token + expert group).  What bounds it is the L2 latency of the
// chunks, about half a microsecond each: the rule that chooses it is route_small.  A product
// of a bf16 and an fp32 value is rounded once with its sum (fma), `per` terms a warp, the
// warps' sums added in order, so
//   |s_fast - s| <= (per + 8) 2^-24 |x_t| |W_r[:, e]|
// to first order (one more unit covers the rest): rigorous.  The loading lanes also form
// |W_r[:, e]|, the columns' largest exponent fields and |x_t|.
constexpr int RS_TB = 8, RS_NW = 8;   // tokens and warps per CTA
constexpr int ROUTE_SMALL_ED = 32768;   // largest 32 ceil(E / 32) d (route_small)
template <int NE>
constexpr int RS_G = 4 / NE;            // tokens whose exact logits are formed together
template <int NE>
constexpr size_t route_small_sums = 16 * RS_NW * 32 * NE * RS_G<NE>;
template <int NE>
constexpr size_t route_small_smem() {
    constexpr size_t EP = 32 * NE, CH = 16 / NE;
    constexpr size_t logits = 4 * RS_NW * (CH * (RS_TB + EP) > RS_TB * EP ? CH * (RS_TB + EP) : RS_TB * EP);
    constexpr size_t exact = route_small_sums<NE> + 4 * RS_G<NE> * (ROUTE_SMALL_ED / EP);   // route_small_exact's sums and xp
    return logits > exact ? logits : exact;
}
// Exact keys of the uncertified tokens `list` of a CTA of route_small_kernel (x rows from xg on, ldx
// apart, RS_NW warps): key[tt][e] for the candidates cand[tt], from the same long accumulators as
// route_fallback_kernel's and with the same windows (wmax: the columns' largest exponent fields).
// The tokens with at most FB_BATCH candidates go all at once, the eight warps shared among them, lanes
// over the d terms: a call with one such token takes 4 us longer than one with none, mostly to
// fetch this code (four terms unrolled: 0.3 us more).  Tokens with more candidates go RS_G together,
// lanes over the experts: the weights are read as whole rows of W_r and taken apart once for those
// tokens, the warps (with E <= 16 also the parts of a warp) share the terms, and a pass costs
// the same however many of the experts tie; the integer instructions bound it (about 20 a term).
// The whole router on tokens that tie in every key (W_r = 0, b = 0): 36 us at T = 64, d = 1024, E =
// 32, 93 at T = 1216, d = 512, E = 64, against 57 and 186 of the tensor-core route; on 1216 tokens
// with two candidates each (d = 1024, E = 32) 27 against 31.  One token after another through all of
// its steps, the threads over the terms for any number of candidates: 330, 470 and 57.
// sums: the warps' sums, [RS_NW][FB_BATCH] and the candidates' ids, or [RS_G][RS_NW][EP]; xp: the
// tokens' x as (mantissa << 16 | exponent), [RS_G][d].
template <int NE>
__device__ __forceinline__ void route_small_exact(uint32_t list, const __nv_bfloat16* __restrict__ xg, int64_t ldx,
                                                  const float* __restrict__ Wr, int d, int E,
                                                  const uint32_t (*cand)[NE], const int* qx, const uint32_t* wmax,
                                                  const float* __restrict__ b, ulonglong2* sums, int* xp,
                                                  double (*key)[32 * NE]) {
    constexpr int EP = 32 * NE, NW = RS_NW, G = RS_G<NE>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto window = [&](int tt, int e) { return qx[tt] == 255 || wmax[e] == 255u ? -1 : qx[tt] + (int)wmax[e]; };   // -1: NaN
    auto put = [&](int at, const unsigned __int128& a) {
        sums[at] = make_ulonglong2((unsigned long long)(uint64_t)a, (unsigned long long)(uint64_t)(a >> 64));
    };
    // the key of token tt, expert e from its n parts sums[at], sums[at + by], ...
    auto finish = [&](int tt, int e, int at, int by, int n) {
        const int Q = window(tt, e);
        double v = __longlong_as_double(0x7ff8000000000000ll);
        if (Q > 0) {
            unsigned __int128 u = 0;
            for (int q = 0; q < n; ++q) {
                const ulonglong2 a = sums[at + q * by];
                u += ((unsigned __int128)a.y << 64) | a.x;
            }
            v = long_acc_value(u, Q);
        }
        key[tt][e] = 1.0 / (1.0 + exp(-v)) + (double)b[e];
    };
    // (the same for the whole CTA, as all that branches on them)
    uint32_t few = 0, wide = 0;   // tokens with at most FB_BATCH candidates; with more
    for (; list; list &= list - 1u) {
        const int tt = __ffs(list) - 1;
        int n = 0;
#pragma unroll
        for (int i = 0; i < NE; ++i) n += __popc(cand[tt][i]);
        if (n > FB_BATCH) wide |= 1u << tt;
        else if (n > 0) few |= 1u << tt;
    }
    if (few) {
        const int n = __popc(few), P = n > 4 ? 8 : n > 2 ? 4 : n;   // P tokens at once, NW / P warps each
        static_assert(RS_TB == 8 && NW == 8, "a warp a token at least");
        int* ids = reinterpret_cast<int*>(sums + NW * FB_BATCH);    // [NW][FB_BATCH] the candidates, -1: none
        auto token = [&](int j) {   // the j-th of them
            uint32_t m = few;
            for (; j > 0; --j) m &= m - 1u;
            return __ffs(m) - 1;
        };
        if (warp % P < n) {
            const int tt = token(warp % P);
            const uint16_t* xr = reinterpret_cast<const uint16_t*>(xg) + tt * ldx;
            uint32_t cm[NE];
#pragma unroll
            for (int i = 0; i < NE; ++i) cm[i] = cand[tt][i];
            const int step = 32 * (NW / P);
#pragma unroll 1
            for (int c = 0; c < FB_BATCH; c += 2) {   // mostly there are two; one copy of the code, which is fetched cold
                int e[2], Q[2];
                unsigned __int128 acc[2];
#pragma unroll
                for (int v = 0; v < 2; ++v) {   // the lowest id left
                    e[v] = -1;
#pragma unroll
                    for (int i = 0; i < NE; ++i)
                        if (e[v] < 0 && cm[i]) {
                            e[v] = 32 * i + __ffs(cm[i]) - 1;
                            cm[i] &= cm[i] - 1u;
                        }
                    if (lane == 0) ids[warp * FB_BATCH + c + v] = e[v];
                    Q[v] = e[v] >= 0 ? window(tt, e[v]) : -1;
                    acc[v] = 0;
                }
                if (Q[0] <= 0 && Q[1] <= 0) continue;
#pragma unroll 1
                for (int i = warp / P * 32 + lane; i < d; i += step) {
                    const uint32_t hx = xr[i];
                    uint32_t uw[2];
#pragma unroll
                    for (int v = 0; v < 2; ++v) uw[v] = Q[v] > 0 ? __float_as_uint(__ldg(Wr + (int64_t)i * E + e[v])) : 0u;
#pragma unroll
                    for (int v = 0; v < 2; ++v) long_acc_term(hx, uw[v], Q[v], acc[v]);   // (Q < 0: not used)
                }
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    acc[v] = warp_sum_u128(acc[v]);
                    if (lane == 0) put(warp * FB_BATCH + c + v, acc[v]);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x < n * FB_BATCH) {
            const int j = threadIdx.x / FB_BATCH, c = threadIdx.x % FB_BATCH, e = ids[j * FB_BATCH + c];
            if (e >= 0) finish(token(j), e, j * FB_BATCH + c, P * FB_BATCH, NW / P);
        }
    }
    const int W = NE > 1 || E > 16 ? 32 : E > 8 ? 16 : 8;   // lanes over the experts; 32 / W parts of a warp
    const int sub = lane / W, le = lane % W, step = NW * (32 / W);
    while (wide) {
        int tok[G];   // -1: none left
        unsigned __int128 acc[G][NE];
        int base[G][NE];   // 64 - Q; 128: not a candidate, or its logit is NaN
#pragma unroll
        for (int u = 0; u < G; ++u) {
            tok[u] = __ffs(wide) - 1;
            wide &= wide - 1u;
#pragma unroll
            for (int i = 0; i < NE; ++i) {
                acc[u][i] = 0;
                base[u][i] = 128;
                if (tok[u] >= 0 && ((cand[tok[u]][i] >> le) & 1u)) {
                    const int Q = window(tok[u], le + 32 * i);
                    if (Q > 0) base[u][i] = 64 - Q;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < G; ++u)
            if (tok[u] >= 0)
                for (int g = threadIdx.x; g < d / 8; g += 32 * NW) {
                    const uint4 v = reinterpret_cast<const uint4*>(xg + tok[u] * ldx)[g];
                    const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
                    int o[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        int mx, ex;
                        long_acc_x(w4[j / 2] >> (16 * (j & 1)), mx, ex);
                        o[j] = mx * 65536 + ex;
                    }
                    int4* to = reinterpret_cast<int4*>(xp + u * d + 8 * g);
                    to[0] = make_int4(o[0], o[1], o[2], o[3]);
                    to[1] = make_int4(o[4], o[5], o[6], o[7]);
                }
        // four terms a step, the next step's weights loaded ahead of them
        uint32_t un[4][NE];
        auto load = [&](int g) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < NE; ++i)
                    un[j][i] = g < d / 4 && le + 32 * i < E ? __float_as_uint(__ldg(Wr + (int64_t)(4 * g + j) * E + le + 32 * i)) : 0u;
        };
        load(warp * (32 / W) + sub);
        __syncthreads();   // xp; and the sums of the tokens before have been taken
        for (int g = warp * (32 / W) + sub; g < d / 4; g += step) {
            int mw[4][NE], ew[4][NE];
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < NE; ++i) long_acc_w(un[j][i], mw[j][i], ew[j][i]);
            load(g + step);
#pragma unroll
            for (int u = 0; u < G; ++u) {
                if (tok[u] < 0) break;
                const int4 x4 = *reinterpret_cast<const int4*>(xp + u * d + 4 * g);
                const int xq[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int i = 0; i < NE; ++i)
                        if (base[u][i] < 128)
                            long_acc_add(xq[j] >> 16, mw[j][i], base[u][i] + (xq[j] & 0xffff) + ew[j][i], acc[u][i]);
            }
        }
#pragma unroll
        for (int u = 0; u < G; ++u)
#pragma unroll
            for (int i = 0; i < NE; ++i) {
                for (int o = W; o < 32; o <<= 1) {
                    const uint64_t lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)(uint64_t)acc[u][i], o);
                    const uint64_t hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(uint64_t)(acc[u][i] >> 64), o);
                    acc[u][i] += ((unsigned __int128)hi << 64) | lo;
                }
                if (sub == 0 && base[u][i] < 128) put((u * NW + warp) * EP + le + 32 * i, acc[u][i]);
            }
        __syncthreads();
        if (threadIdx.x < G * EP) {
            const int u = threadIdx.x / EP;
            int tt = -1;
#pragma unroll
            for (int v = 0; v < G; ++v) tt = u == v ? tok[v] : tt;
            const int e = threadIdx.x % EP;
            if (tt >= 0 && ((cand[tt][e / 32] >> (e & 31)) & 1u)) finish(tt, e, u * NW * EP + e, EP, NW);
        }
    }
}

// Units of 2^-24 |x_t| |W_r[:, e]| certified at least: twice the sum's own bound at d = 192.
constexpr int ROUTE_SMALL_TAU_MIN = 64;
template <int NE>
__global__ void __launch_bounds__(256, 1) route_small_kernel(
    const __nv_bfloat16* __restrict__ x, const float* __restrict__ Wr, const float* __restrict__ b, int T, int d,
    int E, int k, int32_t* __restrict__ idx, float* __restrict__ gate, DevStatus* st, float4* __restrict__ zero,
    int64_t zero_n4) {
    pdl_wait();
    if (zero) {   // side job: clear another buffer (the layer's fp32 y accumulator)
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        const uint64_t pol = l2_policy_evict_first();
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < zero_n4;
             i += (int64_t)gridDim.x * blockDim.x)
            st_global_v4_hint(zero + i, z, pol);
    }
    constexpr int TB = RS_TB, EP = 32 * NE, NW = RS_NW, CH = 16 / NE;
    constexpr int XPC = TB * CH / 8;          // 16-byte pieces of x a chunk: piece q of token tt is q * TB + tt
    static_assert(XPC <= 32, "at most one piece of x a lane");
    // per warp: x [CH][TB] and w [CH][EP]; afterwards the partial logits [NW][TB][EP]
    constexpr int WBUF = CH * (TB + EP);
    extern __shared__ __align__(16) float buf[];   // route_small_smem<NE>()
    __shared__ float s_w2[NW][EP];      // partial sums of squares of W_r's columns, then |W_r[:, e]|
    __shared__ uint32_t s_wmax[NW][EP]; // largest |w| bits, then exponent fields
    __shared__ float s_x2[NW][TB];
    __shared__ uint32_t s_cand[TB][NE];    // uncertified tokens: candidates of each 32-expert slot
    __shared__ int s_qx[TB];               //   largest exponent field of x_t
    __shared__ uint32_t s_again;           //   which of the CTA's tokens they are
    __shared__ double s_key[TB][EP];       //   the candidates' exact keys
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // this CTA's tokens: blockIdx.x + tt gridDim.x, so that neighbours that are alike fall to different CTAs
    const int nt = ((int)T - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
    auto token = [&](int tt) { return (int64_t)blockIdx.x + tt * (int64_t)gridDim.x; };
    if (threadIdx.x == 0) s_again = 0u;
    float* xs = buf + warp * WBUF;
    float* ws = xs + CH * TB;
    const int per = (d / 8 + NW - 1) / NW * 8;   // d % 8 == 0: slices of whole groups of 8
    const int kbeg = warp * per, kend = min(d, kbeg + per);
    const int xt = lane % TB, xk = 8 * (lane / TB);   // this lane's piece of x: its token, its first column
    const __nv_bfloat16* xp = x + token(xt) * d + xk;   // (xt past nt: not read)
    uint4 xr;
    float wv[CH][NE];
    auto load = [&](int k0) {   // chunk k0 .. k0 + CH - 1 into registers (zeros past kend, nt and E)
        const bool ok = lane < XPC && k0 + xk < kend && xt < nt;
        xr = ok ? *reinterpret_cast<const uint4*>(xp + k0) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < CH; ++u)
#pragma unroll
            for (int i = 0; i < NE; ++i) {
                const int e = lane + 32 * i;
                wv[u][i] = k0 + u < kend && e < E ? __ldg(Wr + (int64_t)(k0 + u) * E + e) : 0.f;
            }
    };
    uint64_t acc[4 * NE];   // token lane / 4, expert pairs 32 (p / 4) + 8 (lane % 4) + 2 (p % 4)
#pragma unroll
    for (int p = 0; p < 4 * NE; ++p) acc[p] = 0ull;
    float w2[NE], x2 = 0.f;
    uint32_t wm[NE];
#pragma unroll
    for (int i = 0; i < NE; ++i) {
        w2[i] = 0.f;
        wm[i] = 0u;
    }
    const int tg = lane >> 2, eg = lane & 3;
    if (kbeg < kend) load(kbeg);
    for (int k0 = kbeg; k0 < kend; k0 += CH) {
        __syncwarp();   // the previous chunk has been read
        if (lane < XPC) {
            float f[8];
            unpack_bf16x8(xr, f);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                xs[(xk + i) * TB + xt] = f[i];
                x2 = fmaf(f[i], f[i], x2);
            }
        }
#pragma unroll
        for (int u = 0; u < CH; ++u)
#pragma unroll
            for (int i = 0; i < NE; ++i) {
                ws[u * EP + lane + 32 * i] = wv[u][i];
                w2[i] = fmaf(wv[u][i], wv[u][i], w2[i]);
                wm[i] = max(wm[i], __float_as_uint(wv[u][i]) & 0x7fffffffu);
            }
        __syncwarp();
        if (k0 + CH < kend) load(k0 + CH);
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            uint64_t w[4 * NE];
#pragma unroll
            for (int i = 0; i < NE; ++i)
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(ws + u * EP + 32 * i + 8 * eg + 4 * p);
                    w[4 * i + 2 * p] = v.x;
                    w[4 * i + 2 * p + 1] = v.y;
                }
            const float xv = xs[u * TB + tg];
            const uint64_t xx = f2_pack(xv, xv);
#pragma unroll
            for (int p = 0; p < 4 * NE; ++p) acc[p] = f2_fma(xx, w[p], acc[p]);
        }
    }
    __syncthreads();   // the chunks are done with
#pragma unroll
    for (int p = 0; p < 4 * NE; ++p) {
        float a0, a1;
        f2_unpack(acc[p], a0, a1);
        *reinterpret_cast<float2*>(buf + (warp * TB + tg) * EP + 32 * (p / 4) + 8 * eg + 2 * (p % 4)) =
            make_float2(a0, a1);
    }
#pragma unroll
    for (int i = 0; i < NE; ++i) {
        s_w2[warp][lane + 32 * i] = w2[i];
        s_wmax[warp][lane + 32 * i] = wm[i];
    }
#pragma unroll
    for (int o = TB; o < 32; o <<= 1) x2 += __shfl_xor_sync(0xffffffffu, x2, o);   // a token's pieces: lanes TB apart
    if (lane < TB) s_x2[warp][lane] = x2;
    __syncthreads();
    for (int e = threadIdx.x; e < EP; e += blockDim.x) {
        float v = 0.f;
        uint32_t m = 0u;
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            v += s_w2[q][e];
            m = max(m, s_wmax[q][e]);
        }
        s_w2[0][e] = sqrtf(v);
        s_wmax[0][e] = max(1u, m >> 23);   // exponent field (subnormals and zero count as 1)
    }
    __syncthreads();
    const float tau = (float)max(per + NW + 1, ROUTE_SMALL_TAU_MIN) * 5.9604645e-8f * 1.001f;
    static_assert(TB == NW, "a warp per token");
    const int64_t t = token(warp);
    float sv[NE];
    uint32_t sure_in = 0, cand = 0;
    int need = 0;
    bool again = false;   // this warp's token is re-decided
    uint32_t cm[NE];      // its candidates, bit e of slot i (none: certified, or no exact keys needed)
#pragma unroll
    for (int i = 0; i < NE; ++i) cm[i] = 0u;
    if (warp < nt) {
        float ts[NE], sg[NE];
        float q2 = 0.f;
#pragma unroll
        for (int q = 0; q < NW; ++q) q2 += s_x2[q][warp];
        const float xn = sqrtf(q2);
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            float v = 0.f;
#pragma unroll
            for (int q = 0; q < NW; ++q) v += buf[(q * TB + warp) * EP + lane + 32 * i];
            sv[i] = v;
            ts[i] = tau * s_w2[0][lane + 32 * i] * xn;
        }
        uint32_t taken;
        if (select_certified<NE>(sv, ts, b, E, k, lane, sg, taken)) {
            write_selection<NE>(taken, sg, t, k, lane, idx, gate);
        } else {
            again = true;
            uint4 xv[4];   // the token's x row (d <= 1024), on its way while the keys are bounded
            static_assert(ROUTE_SMALL_ED <= 32 * 4 * 32 * 8, "four pieces a lane");
#pragma unroll
            for (int i = 0; i < 4; ++i)
                xv[i] = lane + 32 * i < d / 8 ? reinterpret_cast<const uint4*>(x + t * d)[lane + 32 * i] : make_uint4(0u, 0u, 0u, 0u);
            bound_candidates<NE>(sv, ts, b, E, k, lane, sure_in, cand);
            int n_in = 0, n_cand = 0;
#pragma unroll
            for (int i = 0; i < NE; ++i) {
                n_in += __popc(__ballot_sync(0xffffffffu, (sure_in >> i) & 1u));
                cm[i] = __ballot_sync(0xffffffffu, (cand >> i) & 1u);
                n_cand += __popc(cm[i]);
            }
            need = k - n_in;
            if (need < 0 || need > n_cand) {
                if (lane == 0) report(st, MOEVIE_ERR_DEVICE, SITE_ROUTE_FALLBACK, (int)t, need);
                need = -1;
            }
            if (need <= 0) {
#pragma unroll
                for (int i = 0; i < NE; ++i) cm[i] = 0u;
            }
            int m = 1;
#pragma unroll
            for (int i = 0; i < 4; ++i) m = max(m, bf16x8_exp_max(xv[i]));
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) {
                atomicOr(&s_again, 1u << warp);
                s_qx[warp] = m;
            }
        }
    }
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < NE; ++i) s_cand[warp][i] = cm[i];
    }
    __syncthreads();   // the fast logits in buf are done with, too
    const uint32_t list = s_again;
    if (list) {
        route_small_exact<NE>(list, x + token(0) * d, (int64_t)gridDim.x * d, Wr, d, E, s_cand, s_qx, s_wmax[0], b,
                              reinterpret_cast<ulonglong2*>(buf),
                              reinterpret_cast<int*>(buf) + route_small_sums<NE> / 4, s_key);
        __syncthreads();
        if (again && need >= 0) {
            double exk[NE];
            float sg[NE];
#pragma unroll
            for (int i = 0; i < NE; ++i) {
                const int e = lane + 32 * i;
                exk[i] = (cm[i] >> lane) & 1u ? s_key[warp][e] : -INFINITY;
            }
            const uint32_t chosen = choose_exact<NE>(exk, sure_in, cand, need, lane);
#pragma unroll
            for (int i = 0; i < NE; ++i) sg[i] = ((chosen >> i) & 1u) ? sigmoid_fast(sv[i]) : 0.f;
            write_selection<NE>(chosen, sg, t, k, lane, idx, gate);
        }
    }
    // tokens re-decided in this call: the last CTA publishes the sum and clears the counters
    if (threadIdx.x == 0) {
        if (list) atomicAdd(&st->route_sum, __popc(list));
        __threadfence();
        if (atomicAdd(&st->route_ticket, 1) == (int)gridDim.x - 1) {
            __threadfence();
            st->fb_count = atomicExch(&st->route_sum, 0);
            st->route_ticket = 0;
        }
    }
}

// out[t, e] = sum of the nparts partial logits, in order (used for inspection).
__global__ void route_sum_parts_kernel(const float* __restrict__ s, int64_t part_stride,
                                       int nparts, int64_t n, float* __restrict__ out) {
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float v = s[i];
    for (int q = 1; q < nparts; ++q) v += s[q * part_stride + i];
    out[i] = v;
}

}  // namespace

int route_split_parts(int d) { return route_dpad(d) / SPLIT_TILE; }

int route_ksplit(int64_t T, int d, int E) {
    int BN = 0, n_ntiles = 0;
    const bool cc = route_concat(E);
    choose_bn(cc ? 2 * route_epad(E) : E, &BN, &n_ntiles);
    const int64_t items = (T + GM_BM - 1) / GM_BM * n_ntiles;
    const int nkb = (cc ? 1 : 2) * route_dpad(d) / GM_BK;
    // work items to aim for: with the pieces side by side (K = d_pad) fewer, longer
    // splits pay (measured: c1 64 items 4.8 us faster than 160)
    const int64_t target = cc ? ROUTE_SPLIT_TARGET_CONCAT : ROUTE_SPLIT_TARGET;
    int64_t p = items > 0 ? (target + items - 1) / items : 1;
    if (p > nkb / 3) p = nkb / 3;   // at least three K blocks per split
    if (p > ROUTE_MAX_KSPLIT) p = ROUTE_MAX_KSPLIT;
    return p < 1 ? 1 : (int)p;
}

int64_t route_logits_rows(int64_t T, int d, int E) {
    (void)d;
    int BN = 0, n_ntiles = 0;
    choose_bn(E, &BN, &n_ntiles);
    const int64_t a = (int64_t)ROUTE_MAX_KSPLIT * T;
    const int64_t b = (ROUTE_SPLIT_TARGET + (T + GM_BM - 1) / GM_BM * n_ntiles) * GM_BM;
    return a < b ? a : b;
}

cudaError_t launch_route_split(const float* Wr, int d, int E, __nv_bfloat16* Wsplit, float* wrt,
                               float* wpart, int32_t* wexp, DevStatus* st, cudaStream_t s) {
    const int Ep = route_epad(E);
    const int parts = route_split_parts(d);
    cudaError_t e = launch_pdl(route_split_kernel, dim3((Ep + SPLIT_TILE - 1) / SPLIT_TILE, parts),
                               dim3(256), 0, s, Wr, d, route_dpad(d), E, Ep, Wsplit, wrt, wpart, parts,
                               wexp, st, route_concat(E) ? 1 : 0);
    count_launches(1);
    return e;
}

cudaError_t launch_route_sum_parts(const float* logits, int64_t part_stride, int nparts, int64_t n,
                                   float* out, cudaStream_t s) {
    const cudaError_t e = launch_pdl(route_sum_parts_kernel, dim3((unsigned)((n + 255) / 256)),
                                     dim3(256), 0, s, logits, part_stride, nparts, n, out);
    count_launches(1);
    return e;
}

// The one-launch router takes up to eight tokens for each SM (one wave of CTAs) and chunks
// few enough: 32 ceil(E / 32) d <= ROUTE_SMALL_ED, so at most eight chunks a warp.  Measured against the
// tensor-core route, back to back calls: T = 512, d = 768, E = 16 10.5 against 17.5 us, T = 256,
// E = 31 12.8 against 18.0; past the line, T = 1024, d = 1536, E = 64 (24 chunks) 31 against 24.
constexpr int ROUTE_SMALL_SMS = 152;
bool route_small(int64_t T, int d, int E) {
    return T >= 1 && T <= RS_TB * ROUTE_SMALL_SMS && E <= 64 && (int64_t)(E + 31) / 32 * 32 * d <= ROUTE_SMALL_ED;
}

cudaError_t launch_route_small(const __nv_bfloat16* x, const float* Wr, const float* b, int T, int d, int E, int k,
                               int32_t* idx, float* gate, DevStatus* st, cudaStream_t s, float* zero,
                               int64_t zero_n) {
    if (!route_small(T, d, E)) return cudaErrorInvalidValue;
    static_assert(route_small_smem<1>() <= 38 * 1024 && route_small_smem<2>() <= 38 * 1024,
                  "no opt-in needed beside the static arrays (9 KB)");
    // as few tokens a CTA as one wave of the SMs allows (a CTA takes as long with two as with eight),
    // so that tokens that need the exact keys are spread over the SMs: T = 16, d = 512, E = 64, all
    // tied, 34 us with two tokens a CTA, 53 with four (one: 27, but 10.7 instead of 10.2 untied)
    const int tb = std::max(2, (T + ROUTE_SMALL_SMS - 1) / ROUTE_SMALL_SMS);
    const auto kern = E <= 32 ? route_small_kernel<1> : route_small_kernel<2>;
    const cudaError_t e = launch_pdl(kern, dim3((unsigned)((T + tb - 1) / tb)), dim3(256),
                                     E <= 32 ? route_small_smem<1>() : route_small_smem<2>(), s, x, Wr, b, T, d, E,
                                     k, idx, gate, st, reinterpret_cast<float4*>(zero), zero ? zero_n / 4 : (int64_t)0);
    count_launches(1);
    return e;
}

cudaError_t launch_route_select(const __nv_bfloat16* x, const float* wrt, const float* b,
                                float* logits, int ld, int nparts, int64_t part_stride,
                                const float* wnorm, const int32_t* wexp, int T, int d, int E, int k,
                                int32_t* idx, float* gate, int32_t* fb_tokens, float* xnorm,
                                DevStatus* st, int num_sms, cudaStream_t s, float* zero,
                                int64_t zero_n) {
    const int blocks = (int)(((int64_t)T * 32 + 255) / 256);
    const int fb_per_sm = (E + 31) / 32 <= 8 ? FB_CTAS_PER_SM : 3;
    const int fb_blocks = T < fb_per_sm * num_sms ? T : fb_per_sm * num_sms;   // one resident wave
    const size_t fb_smem = d <= FB_X_SMEM ? (size_t)2 * d : 0;
    const int npl = (E + 31) / 32;
    const int dp = route_dpad(d);
    const int parts = route_split_parts(d), Ep = route_epad(E);
    cudaError_t e = cudaSuccess;
#define MV_ROUTE(N)                                                                                \
    do {                                                                                           \
        e = launch_pdl(route_topk_kernel<N>, dim3(blocks), dim3(256), 0, s, x, logits, ld, nparts,  \
                       part_stride, b, wnorm, T, d, E, k, idx, gate, (const float*)xnorm,           \
                       fb_tokens, st, reinterpret_cast<float4*>(zero), zero ? zero_n / 4 : 0);      \
        if (e == cudaSuccess)                                                                      \
            e = launch_pdl(route_fallback_kernel<N>, dim3(fb_blocks), dim3(256), fb_smem, s, x,    \
                           wrt, dp, wexp, parts, Ep, b, (const float*)logits, ld,                  \
                           (const float*)xnorm, wnorm, d, E, k, idx, gate,                          \
                           (const int32_t*)fb_tokens, st);                                         \
    } while (0)
    if (npl <= 1) MV_ROUTE(1);
    else if (npl <= 2) MV_ROUTE(2);
    else if (npl <= 4) MV_ROUTE(4);
    else if (npl <= 8) MV_ROUTE(8);
    else if (npl <= 16) MV_ROUTE(16);
    else MV_ROUTE(32);
#undef MV_ROUTE
    count_launches(2);
    return e;
}

}  // namespace mv
