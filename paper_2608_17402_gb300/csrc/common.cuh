// common.cuh -- device helpers shared by the MoE-ViE layer kernels (sm_103a).
//
// Device errors never trap: a kernel that finds a bad index, or whose pipeline
// wait runs past its time limit, records the first such event in the status
// block at the start of the caller's workspace and returns.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "moevie.h"

namespace mv {

// ------------------------------------------------------------------ status

// Lives at byte 0 of every workspace (256 bytes, zeroed by moevie_workspace_init).
struct DevStatus {
    int code;        // first device error (MOEVIE_ERR_*), 0 when none
    int site;        // which check (Site)
    int a, b;        // two values describing it
    int fb_count;    // router: tokens re-decided with exact logits in the last call
    int bar_count;   // grid barrier of a cooperative launch: arrivals so far (0 between barriers)
    int bar_gen;     //   and the barrier's generation (bumped by the last arrival)
    int route_sum;    // one-launch router: tokens re-decided so far in the running call,
    int route_ticket; //   and its CTAs done (both 0 between calls)
    int pad[55];
};
static_assert(sizeof(DevStatus) == 256, "status block is 256 bytes");

enum Site : int {
    SITE_GEMM_WAIT_FULL = 1,
    SITE_GEMM_WAIT_EMPTY = 2,
    SITE_GEMM_WAIT_TFULL = 3,
    SITE_GEMM_WAIT_TEMPTY = 4,
    SITE_GEMM_DRAIN = 5,
    SITE_GEMM_A_ROW = 6,
    SITE_GEMM_TILES = 7,
    SITE_GEMM_OUT_ROW = 8,
    SITE_PERMUTE_ID = 10,
    SITE_ROUTE_FALLBACK = 20,
    SITE_BIAS_COUNTS = 21,
    SITE_TIMEOUT_PROBE = 30,
    SITE_PERMUTE_BARRIER = 31,
};

__device__ __forceinline__ void report(DevStatus* st, int code, int site, int a, int b) {
    if (atomicCAS(&st->code, 0, code) == 0) {
        st->site = site;
        st->a = a;
        st->b = b;
    }
}

// Grid-wide barrier of a cooperative launch (all nblocks CTAs co-resident) with a time
// limit: the last CTA to arrive resets the count and bumps the generation; the others
// wait for the bump for at most limit_ns.  Returns false (after recording
// MOEVIE_ERR_TIMEOUT at `site`) when the wait ran out; the caller then stops.  The count
// starts at 0 (a zeroed status block) and returns to 0 after every barrier.
__device__ __forceinline__ bool grid_barrier(DevStatus* st, unsigned nblocks, uint64_t limit_ns, int site) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int* genp = &st->bar_gen;
        const int gen = *genp;
        __threadfence();   // this CTA's writes before its arrival
        int ok = 1;
        if (atomicAdd(&st->bar_count, 1) == (int)nblocks - 1) {
            st->bar_count = 0;
            __threadfence();
            atomicAdd(&st->bar_gen, 1);
        } else {
            uint64_t t0;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
            for (uint32_t i = 1; *genp == gen; ++i) {
                if ((i & 63u) == 0u) {
                    uint64_t t1;
                    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
                    if (t1 - t0 > limit_ns) {
                        ok = 0;
                        report(st, MOEVIE_ERR_TIMEOUT, site, (int)blockIdx.x, gen);
                        break;
                    }
                }
            }
        }
        __threadfence();   // the other CTAs' writes after the barrier
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialization may start while its predecessor finishes; it waits here (at the
// top, before touching anything the predecessor writes) until that predecessor has
// completed and its memory is visible.  A no-op for ordinary launches.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---------------------------------------------------------------- basics

__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// --------------------------------------------------------------- mbarrier

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
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

// Wait for the phase of `parity` to complete.  Gives up (returns false) once
// `limit_ns` of device time has passed, or as soon as *abort_flag is set by
// another role of the same CTA.  Every pipeline wait in this library goes here.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint64_t limit_ns,
                                          const volatile int* abort_flag) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t i = 1;; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 127u) == 0u) {
            if (abort_flag && *abort_flag) return false;
            if (globaltimer_ns() - t0 > limit_ns) return false;
        }
    }
}

// The same wait by a whole converged warp: every lane polls, the vote keeps the warp
// converged (as elect.sync and the issue of tcgen05 / TMA instructions behind it need)
// and makes the outcome warp-uniform.  `ready`: an earlier mbar_try_wait on the same
// phase, polled while the previous stage's instructions were in flight, so that a phase
// already complete costs no wait here.  ONE: only lane 0 polls (beside warps that keep the
// load pipes busy, the router GEMM's norm jobs, whole-warp polling cost that GEMM 30 %).
template <bool ONE = false>
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, uint64_t limit_ns,
                                               const volatile int* abort_flag, bool ready = false) {
    if (ONE) {
        int ok = 1;
        if ((threadIdx.x & 31) == 0) ok = ready || mbar_wait(bar, parity, limit_ns, abort_flag);
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();   // orders what lane 0 has seen before what the elected lane issues (the shuffle orders no memory)
        return ok != 0;
    }
    if (__all_sync(0xffffffffu, ready || mbar_try_wait(bar, parity))) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t i = 1;; ++i) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if ((i & 127u) == 0u) {
            const bool stop = (abort_flag && *abort_flag) || globaltimer_ns() - t0 > limit_ns;
            if (__any_sync(0xffffffffu, stop)) return false;
        }
    }
}
// One poll that does not suspend the thread.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// True in one lane of a converged warp, always the same one.  Code that one lane runs
// behind this predicate is known to ptxas to run in a single lane, so the instructions
// with warp-uniform operands (tcgen05.mma and commit, TMA and bulk copies) need no loop
// over the active lanes, which they do behind a condition on threadIdx.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

// ------------------------------------------------------------- cp.async

// 16-byte global->shared copy; src_bytes < 16 zero-fills the rest (0: all zeros,
// nothing read).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
                 "r"(src_bytes)
                 : "memory");
}
// L2 cache policies (createpolicy): keep lines (evict_last) or let them go first.
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
// cp_async16 with an L2 cache policy for the global read.
__device__ __forceinline__ void cp_async16_hint(uint32_t dst, const void* src, uint32_t src_bytes,
                                                uint64_t pol) {
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2, %3;" ::"r"(dst),
                 "l"(src), "r"(src_bytes), "l"(pol)
                 : "memory");
}
// 16-byte global store with an L2 cache policy.
__device__ __forceinline__ void st_global_v4_hint(void* p, const uint4& v, uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.v4.b32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "r"(v.x),
                 "r"(v.y), "r"(v.z), "r"(v.w), "l"(pol)
                 : "memory");
}
// *p += v (16 bytes, relaxed) with an L2 cache policy.  p: 16-byte aligned global memory.
__device__ __forceinline__ void red_add_v4_hint(float4* p, const float4& v, uint64_t pol) {
    asm volatile("red.relaxed.gpu.global.add.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p),
                 "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "l"(pol)
                 : "memory");
}
// *p += v as a relaxed reduction when sel >= 0 (predicated, no branch).  No memory clobber:
// loads may move across it (nothing in the kernels that use it reads what it adds to).
__device__ __forceinline__ void red_add_f32_if(float* p, float v, int sel) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ge.s32 q, %2, 0;\n\t"
        "@q red.relaxed.gpu.global.add.f32 [%0], %1;\n\t}" ::"l"(p),
        "f"(v), "r"(sel));
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// Arrive on `bar` once all cp.async copies issued so far by this thread have landed
// (the barrier's expected count includes this arrival).
__device__ __forceinline__ void cp_async_arrive_noinc(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_all;" ::: "memory");
}
// Orders this thread's generic-proxy shared-memory writes before later
// async-proxy reads (tcgen05.mma operands, TMA stores).
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ------------------------------------------------------------------- TMA

__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* tm) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(tm) : "memory");
}

// --------------------------------------------------------------- tcgen05

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp gets lane
// (base lane + i), columns [col, col + 32).
__device__ __forceinline__ void tmem_ld_32x32b_x32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
// 32 lanes x 16 consecutive 32-bit columns (thread i: lane base + i, columns col..col+15).
__device__ __forceinline__ void tmem_ld_32x32b_x16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Shared-memory matrix descriptor (tcgen05), 128-byte swizzle.
//   bits  0-13 start address >> 4      bits 16-29 leading byte offset >> 4
//   bits 32-45 stride byte offset >> 4 bits 46-47 descriptor version (1)
//   bits 49-51 base offset (0: atoms 1024-byte aligned)   bits 61-63 layout (2 = SW128)
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
    d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
    d |= static_cast<uint64_t>(1) << 46;
    d |= static_cast<uint64_t>(2) << 61;
    return d;
}

// Instruction descriptor of kind::f16 with bf16 A/B and fp32 D.
//   bits 4-5 D format (1 = f32)   bits 7-9 A format (1 = bf16)  bits 10-12 B format (1 = bf16)
//   bit 15 A major (0 = K)        bit 16 B major (1 = MN)       bits 17-22 N >> 3
//   bits 24-28 M >> 4
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N, bool a_mn_major,
                                                     bool b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(a_mn_major) << 15) |
           (static_cast<uint32_t>(b_mn_major) << 16) | ((static_cast<uint32_t>(N) >> 3) << 17) |
           ((static_cast<uint32_t>(M) >> 4) << 24);
}

// -------------------------------------------------------------- bf16 pack

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
// Packed pairs of fp32 values (one 64-bit register pair) and the sm_100-family
// two-wide fp32 arithmetic on them: one instruction does the work of two.
__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t r, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ void unpack_bf16x8(const uint4& u, float (&v)[8]) {
    const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float2 f = __bfloat1622float2(p[i]);
        v[2 * i] = f.x;
        v[2 * i + 1] = f.y;
    }
}

}  // namespace mv
