// Inline-PTX wrappers for the sm_103a tensor-core passes: mbarriers, bulk and
// tensor (TMA) copies, tcgen05 MMA / commit / tensor-memory loads, and the
// shared-memory and instruction descriptors they take.
#pragma once
#include <cstdint>

#include <cuda_bf16.h>

#include "bm_device.cuh"

namespace bm {
namespace tc {

__device__ __forceinline__ unsigned s_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* b, unsigned cnt) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s_addr(b)), "r"(cnt) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void expect_tx(unsigned long long* b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s_addr(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void arrive(unsigned long long* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s_addr(b)) : "memory");
}
__device__ __forceinline__ bool try_wait(unsigned long long* b, unsigned parity) {
    unsigned ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok)
                 : "r"(s_addr(b)), "r"(parity)
                 : "memory");
    return ok != 0;
}
// try_wait that may suspend the thread for up to `ns` nanoseconds while the
// phase is incomplete (it returns as soon as the phase completes).
__device__ __forceinline__ bool try_wait_sleep(unsigned long long* b, unsigned parity, unsigned ns) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(s_addr(b)), "r"(parity), "r"(ns)
        : "memory");
    return ok != 0;
}
// Limits of the bounded waits: `polls` polls, each suspending the thread for
// at most `ns` nanoseconds (0: a plain poll).  The default, 2^18 polls of at
// most 20 us, ends a wait after about 5 s; bm_debug_set_wait_limit sets
// smaller values for a test that makes a wait run out.
struct WaitLimit { unsigned polls, ns; };
constexpr WaitLimit kDefaultWait = {1u << 18, 20000u};

// Bounded wait.  Gives up when `abort` is raised by another role of the CTA,
// or once the limit is spent (then it raises `abort` and the timeout flag),
// so that no role of a CTA can wait forever on another.
__device__ __forceinline__ bool wait(unsigned long long* b, unsigned parity, volatile int* abort, Globals* g,
                                     WaitLimit lim) {
    for (unsigned i = 0; i < lim.polls; ++i) {
        if (lim.ns ? try_wait_sleep(b, parity, lim.ns) : try_wait(b, parity)) return true;
        if (*abort) return false;
    }
    *abort = 1;
    atomicOr(&g->err, kErrTimeout);
    return false;
}

// The same wait by every lane of a warp (no lane has to pass the outcome on);
// true for all lanes or for none.
__device__ __forceinline__ bool wait_warp(unsigned long long* b, unsigned parity, volatile int* abort, Globals* g,
                                          WaitLimit lim) {
    bool ok = try_wait(b, parity);
    if (!ok) ok = wait(b, parity, abort, g, lim);
    return __all_sync(0xffffffffu, ok);
}

// 1-D bulk copy global -> shared (addresses and size multiples of 16 bytes).
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* b) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     s_addr(dst)),
                 "l"(src), "r"(bytes), "r"(s_addr(b))
                 : "memory");
}
// 2-D tiled tensor copy global -> shared through a tensor map; (x, y) is the
// box origin in elements (x * element size must be a multiple of 16 bytes).
__device__ __forceinline__ void tma_load_2d(void* dst, const void* tmap, int x, int y, unsigned long long* b) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(s_addr(dst)),
        "l"(tmap), "r"(x), "r"(y), "r"(s_addr(b))
        : "memory");
}

// 64-bit shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row
// groups 1024 bytes apart, descriptor version 1.
__device__ __forceinline__ unsigned long long desc_sw128(unsigned addr) {
    unsigned long long d = 0;
    d |= (unsigned long long)((addr >> 4) & 0x3FFFu);          // start address
    d |= (unsigned long long)1u << 16;                          // leading byte offset (unused here)
    d |= (unsigned long long)(1024u >> 4) << 32;                // stride byte offset
    d |= (unsigned long long)1u << 46;                          // version
    d |= (unsigned long long)2u << 61;                          // 128-byte swizzle
    return d;
}
// Instruction descriptors: FP32 accumulate, A and B K-major, M x N.
// kind::f16 with BF16 operands (format 1).
__host__ __device__ constexpr unsigned idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(unsigned tmem_d, unsigned long long adesc, unsigned long long bdesc,
                                         unsigned idesc, unsigned accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive on `b` once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void commit(unsigned long long* b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s_addr(b))
                 : "memory");
}
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
// Generic-proxy writes to shared memory made visible to the async proxy.
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Tensor-memory allocation (whole warp); the address lands in *slot.
__device__ __forceinline__ void tmem_alloc(unsigned* slot, unsigned cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_addr(slot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(unsigned taddr, unsigned cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

// 32 lanes x 16 columns of 32-bit tensor-memory cells -> 16 registers per
// thread (no wait; pair with wait_ld16).
__device__ __forceinline__ void ld16(unsigned taddr, unsigned (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// ---------------------------------------------- epilogue helpers (g top-2)
// The BF16 pass reads, per row, g_j = fl(ccb_j - 2 acc_j) from the
// accumulator columns in chunks of 16 and keep the two least g (pass 1),
// then a bit mask of the columns with g <= lim, i.e. below next_up(lim) (pass 2).

// 16 tensor-memory columns in flight into r: the wait for them takes r as
// operands, so that no use of r can be scheduled before the wait.
__device__ __forceinline__ void wait_ld16(unsigned (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15])
                 :
                 : "memory");
}

// g of the columns c0 + 4 q .. c0 + 4 q + 3 from 16 accumulator cells:
// fl(ccb - 2 acc).
__device__ __forceinline__ void g_quad(float (&e)[4], const unsigned (&va)[16], const float* ccb, int c0, int q) {
    const float4 cq = *reinterpret_cast<const float4*>(ccb + c0 + 4 * q);
    const float2 e01 = __ffma2_rn(make_float2(-2.f, -2.f),
                                  make_float2(__uint_as_float(va[4 * q]), __uint_as_float(va[4 * q + 1])),
                                  make_float2(cq.x, cq.y));
    const float2 e23 = __ffma2_rn(make_float2(-2.f, -2.f),
                                  make_float2(__uint_as_float(va[4 * q + 2]), __uint_as_float(va[4 * q + 3])),
                                  make_float2(cq.z, cq.w));
    e[0] = e01.x;
    e[1] = e01.y;
    e[2] = e23.x;
    e[3] = e23.y;
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
// Pass 1 over the columns c0 .. c0 + 15 (the first `nv` of them when PART):
// four chains of the least and second least g.  Each pair of columns is
// sorted (lo, hi) and merged: t2 = min(t2, hi, max(t1, lo)), t1 = min(t1, lo).
template <bool PART>
__device__ __forceinline__ void min2_chunk(float (&t1)[4], float (&t2)[4], const unsigned (&va)[16], const float* ccb,
                                           int c0, int nv) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (PART && 4 * q >= nv) break;
        float e[4];
        g_quad(e, va, ccb, c0, q);
        if (PART)                                   // columns past k: +inf
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = (4 * q + i < nv) ? e[i] : __int_as_float(0x7f800000);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int c = (2 * q + p) & 3;
            const float lo = fminf(e[2 * p], e[2 * p + 1]), hi = fmaxf(e[2 * p], e[2 * p + 1]);
            t2[c] = min3f(t2[c], hi, fmaxf(t1[c], lo));
            t1[c] = fminf(t1[c], lo);
        }
    }
}
// Pass 2 over the columns c0 .. c0 + 15 (the first `nv` when PART): mk moves
// 16 bits up and takes, first column in the highest of them, whether g is
// below L: the sign of g - L (exact in sign) by a funnel shift, which costs
// one ALU operation per column instead of a compare and a predicated or
// (10^7 x 64, k = 100, tau = 1e-3, the whole call with 64-bit distance sums and
// waits by whole warps: 680 -> 643 us).
template <bool PART>
__device__ __forceinline__ unsigned below_mask16(unsigned mk, const unsigned (&va)[16], const float* ccb, int c0,
                                                 float L, int nv) {
    const float2 mL = make_float2(-L, -L);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (PART && 4 * q >= nv) { mk <<= 4; continue; }
        float e[4];
        g_quad(e, va, ccb, c0, q);
        const float2 d0 = __fadd2_rn(make_float2(e[0], e[1]), mL), d1 = __fadd2_rn(make_float2(e[2], e[3]), mL);
        mk = __funnelshift_l(__float_as_uint(d0.x), mk, 1);
        mk = __funnelshift_l(__float_as_uint(d0.y), mk, 1);
        mk = __funnelshift_l(__float_as_uint(d1.x), mk, 1);
        mk = __funnelshift_l(__float_as_uint(d1.y), mk, 1);
    }
    return PART ? mk & ~((1u << (16 - nv)) - 1u) : mk;
}
// The float above v (v < next_up(w) exactly when v <= w); NaN for +inf and NaN.
__device__ __forceinline__ float next_up(float v) {
    const int b = __float_as_int(v);
    return v == 0.f ? 0x1p-149f : __int_as_float(b < 0 ? b - 1 : b + 1);
}

// 32 lanes x 32 columns of 32-bit tensor-memory cells -> 32 registers per
// thread, waited for (the wait takes the registers as operands, so that no use
// of them can be scheduled before it).
__device__ __forceinline__ void wait_ld32(unsigned (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                   "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}
__device__ __forceinline__ void ld32(unsigned taddr, unsigned (&r)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                   "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    wait_ld32(r);
}
// The same, with the least of the 32 values (as FP32) taken on the way.
__device__ __forceinline__ void ld32_min(unsigned taddr, unsigned (&r)[32], float& mn) {
    unsigned u;
    asm volatile("tcgen05.ld.red.sync.aligned.32x32b.x32.min.f32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, %32, [%33];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                   "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(u)
                 : "r"(taddr));
    wait_ld32(r);
    asm volatile("" : "+r"(u));                    // not before the wait either
    mn = __uint_as_float(u);
}
// 32 floats of shared memory (16-byte aligned) into 32 columns of every lane
// of the warp (pair with wait_st).
__device__ __forceinline__ void st32_shared(unsigned taddr, const float* p) {
    unsigned r[32];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const uint4 v = *reinterpret_cast<const uint4*>(p + 4 * q);
        r[4 * q] = v.x; r[4 * q + 1] = v.y; r[4 * q + 2] = v.z; r[4 * q + 3] = v.w;
    }
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};" ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
                 "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]),
                 "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
                 "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]), "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Bit 31 - i set where the i-th of 32 values is below L: v - L is exact in
// sign (gradual underflow), and a funnel shift moves the sign bit in.
__device__ __forceinline__ unsigned below_mask32(const unsigned (&va)[32], float L) {
    unsigned mk = 0;
    const float2 mL = make_float2(-L, -L);
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
        const float2 d = __fadd2_rn(make_float2(__uint_as_float(va[i]), __uint_as_float(va[i + 1])), mL);
        mk = __funnelshift_l(__float_as_uint(d.x), mk, 1);
        mk = __funnelshift_l(__float_as_uint(d.y), mk, 1);
    }
    return mk;
}

// Eight values as BF16 pairs h = bf16(v) and l = bf16(v - h) (v - h is exact).
__device__ __forceinline__ void split_bf16(const float (&v)[8], uint4& h, uint4& l) {
    unsigned hw[4], lw[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        hw[i] = *reinterpret_cast<const unsigned*>(&a);
        const float2 f = make_float2(__uint_as_float(hw[i] << 16), __uint_as_float(hw[i] & 0xffff0000u));
        const float2 r = __ffma2_rn(make_float2(-1.f, -1.f), f, make_float2(v[2 * i], v[2 * i + 1]));
        const __nv_bfloat162 b = __floats2bfloat162_rn(r.x, r.y);
        lw[i] = *reinterpret_cast<const unsigned*>(&b);
    }
    h = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    l = make_uint4(lw[0], lw[1], lw[2], lw[3]);
}

}  // namespace tc
}  // namespace bm
