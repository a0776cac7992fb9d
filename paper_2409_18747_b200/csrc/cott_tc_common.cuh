// Helpers shared by the warp-specialised tensor-core kernels of cott_tc_bwd.cu and
// cott_tc_bidir.cu: the bounded mbarrier wait with its abort protocol, and a few small device
// functions.  Every kernel that uses them lays out its control block the same way: mbarriers in
// the first 448 bytes, then the tensor-memory slot (offset 448), the abort flag (452) and, three
// words behind it, the wait limit in units of 1024 SM cycles.
#pragma once
#include "cott_sm100.cuh"

namespace cott {
namespace tc {

using namespace sm100;

constexpr int kCtlTmemSlot = 448, kCtlAbort = 452;
constexpr uint32_t kDescHi = smem_desc_hi(1024);
#ifndef COTT_WAIT_HINT_NS
#define COTT_WAIT_HINT_NS 1000
#endif
constexpr uint32_t kWaitHintNs = COTT_WAIT_HINT_NS;   // a waiting thread may be parked this long per try

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Bounded wait that also gives up as soon as any thread of the CTA has given up.  The thread
// that gives up first leaves a record of where: bit 31 set, warp index in bits 16-20, byte
// offset of the barrier inside the barrier block in bits 4-13, parity in bit 0.
// (The loop is a function of its own, not inlined: these kernels have dozens of waits, and
// their code must stay small enough for the instruction caches -- several roles run different
// code on one SM at the same time.)
static __device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    const long long t0 = clock64();
    for (uint32_t it = 1;; ++it) {
        if (kWaitHintNs ? mbar_try_wait_hint(bar, parity, kWaitHintNs) : mbar_try_wait(bar, parity)) return true;
        if ((it & 15u) == 1) {
            if (*abort_flag) return false;
            if (clock64() - t0 > ((long long)abort_flag[3] << 10)) {
                const uint32_t bars = (uint32_t)__cvta_generic_to_shared((const void*)abort_flag) - (uint32_t)kCtlAbort;
                const uint32_t where = 0x80000000u | ((threadIdx.x >> 5) << 16) | (((bar - bars) & 0x3FFu) << 4) | (parity & 1u);
                atomicCAS(const_cast<int*>(abort_flag), 0, (int)where);
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    if (mbar_try_wait(bar, parity)) return true;
    return wait_slow(bar, parity, abort_flag);
}

// The same with the limit checked between a test and a (suspending) try: for a kernel whose only wait is
// shorter than one suspension, so that its bound is a bound there too.  (Inlined: a call would first wait
// for every load its caller has in flight.)
// (wait_expired: one poll of such a wait that began at t0.)
__device__ __forceinline__ bool wait_expired(uint32_t bar, uint32_t parity, long long t0, volatile int* abort_flag) {
    if (mbar_test_wait(bar, parity) || clock64() - t0 <= ((long long)abort_flag[3] << 10)) return false;
    const uint32_t bars = (uint32_t)__cvta_generic_to_shared((const void*)abort_flag) - (uint32_t)kCtlAbort;
    const uint32_t where = 0x80000000u | ((threadIdx.x >> 5) << 16) | (((bar - bars) & 0x3FFu) << 4) | (parity & 1u);
    atomicCAS(const_cast<int*>(abort_flag), 0, (int)where);
    return true;
}
__device__ __forceinline__ bool wait_polling(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    const long long t0 = clock64();
    for (;;) {
        if (mbar_test_wait(bar, parity)) return true;
        if (*abort_flag || wait_expired(bar, parity, t0, abort_flag)) return false;
        if (mbar_try_wait(bar, parity)) return true;
    }
}

__device__ __forceinline__ uint4 pack8(const uint32_t* r) {
    uint4 w;
    w.x = pack_bf16(__uint_as_float(r[0]), __uint_as_float(r[1]));
    w.y = pack_bf16(__uint_as_float(r[2]), __uint_as_float(r[3]));
    w.z = pack_bf16(__uint_as_float(r[4]), __uint_as_float(r[5]));
    w.w = pack_bf16(__uint_as_float(r[6]), __uint_as_float(r[7]));
    return w;
}

// x * rn in fp32, rounded to bf16 once.
__device__ __forceinline__ __nv_bfloat162 scale_round(__nv_bfloat162 x, float rn) {
    const float2 f = __fmul2_rn(__bfloat1622float2(x), make_float2(rn, rn));
    return __floats2bfloat162_rn(f.x, f.y);
}

// x * rn in packed bf16 arithmetic with the scale split in two bf16 terms (rn = hi + lo to 2^-17):
// round(x hi + round(x lo)) is x rn rounded once, up to a second rounding of the small term.
struct RowScale {
    __nv_bfloat162 hi2, lo2;
    __device__ __forceinline__ explicit RowScale(float rn) {
        const __nv_bfloat16 hi = __float2bfloat16_rn(rn);
        const __nv_bfloat16 lo = __float2bfloat16_rn(rn - __bfloat162float(hi));
        hi2 = __halves2bfloat162(hi, hi); lo2 = __halves2bfloat162(lo, lo);
    }
    __device__ __forceinline__ __nv_bfloat162 operator()(__nv_bfloat162 x) const { return __hfma2(x, hi2, __hmul2(x, lo2)); }
};

// Sum of squares of 64 bf16 values held in w[8] (eight 16-byte chunks), packed fp32 arithmetic.
__device__ __forceinline__ float sumsq_row64(const uint4 (&w)[8]) {
    float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
        const float2 f0 = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w)[j]);
        const float2 f1 = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w)[j + 1]);
        s0 = __ffma2_rn(f0, f0, s0); s1 = __ffma2_rn(f1, f1, s1);
    }
    return (s0.x + s0.y) + (s1.x + s1.y);
}

// x / max(||x||, eps) on one row of 64 bf16 values held in w[8].  Returns the norm; *rn_out = 1 / max(norm, eps).
__device__ __forceinline__ float normalise_row64(uint4 (&w)[8], float eps, float* rn_out) {
    const float nrm = sqrtf(sumsq_row64(w));
    const float rn = 1.0f / fmaxf(nrm, eps);
    const RowScale rs(rn);
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        __nv_bfloat162& e = reinterpret_cast<__nv_bfloat162*>(w)[j];
        e = rs(e);
    }
    *rn_out = rn;
    return nrm;
}

}  // namespace tc
}  // namespace cott
