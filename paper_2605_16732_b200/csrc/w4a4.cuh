// What the two second kernels of the grouped INT4 formats share (w4a4_gemm.cu, w4a4_narrow.cu): tile constants, parameters,
// wait accounting, packed fp32 arithmetic, code expansion.
#pragma once
#include "common.h"
#include "ptx.cuh"

#include <cuda_bf16.h>

namespace dirotq {
namespace {

constexpr int BM = 128;
constexpr int BKC = 128;  // one-byte codes per k-block (128-byte rows)
constexpr int A_BYTES = BM * BKC;          // 16 KB  activation codes / bf16 x~_h chunk
constexpr uint32_t kSignMag = 0x87878787u;  // sign and 3-bit magnitude of four one-byte codes
constexpr float kAccUnit = kI8Path ? 1.0f : kWScaleFold;  // integer group sum = accumulator value x this

struct GemmKernelParams {
    int M, N, n_g, num_kb, lr_chunks;
    const float* bias;
    uint16_t* y;
    int32_t* partials;
    int* status;
    int early_weights;  // see GemmArgs
    int x_rows;         // rows of the activation tiles' boxes (box_rows)
};

// Compile-time loop: f(Int<0>{}), ..., f(Int<N - 1>{}).
template <int V>
struct Int { static constexpr int value = V; };
template <int N, int I = 0, class F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (I < N) {
        f(Int<I>{});
        static_for<N, I + 1>(f);
    }
}

// Wait accounting (diagnostics): cycles a role spends blocked on each kind of barrier are summed into
// 64-bit counters that follow the status word in the workspace (8-byte slots 1..8, see WaitSlot; nothing waits for scales by themselves, slot 6 stays 0).
// What try_wait's own suspension of the thread covers (most waits of a call) is counted in the diagnostic build only: a test and two clock reads for
// every such wait are 1 % of a call (4608 x 3072 -> 9216 233.9 -> 235.9 us; 18432 rows, groups of 128 562 -> 574).
enum WaitSlot : int { WS_PROD_EMPTY = 1, WS_MMA_OPERANDS = 2, WS_MMA_TEMPTY = 3, WS_UNPACK_FULL = 4, WS_EPI_TFULL = 5,
                      WS_EPI_TOTAL = 7, WS_KERNEL = 8 };

__device__ __forceinline__ bool timed_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, int code,
                                           long long& acc) {
    if (kTraceBuild ? mbar_test_wait(bar, parity) : mbar_try_wait(bar, parity)) return true;  // the common case costs no clock reads
    const long long t0 = clock64();
    const bool ok = mbar_wait(bar, parity, abort_flag, status, code);
    acc += clock64() - t0;
    return ok;
}

__device__ __forceinline__ void flush_wait(int* status, int slot, long long cycles) {
    atomicAdd(reinterpret_cast<unsigned long long*>(status) + slot, static_cast<unsigned long long>(cycles));
}

// Two fp32 values in one 64-bit register pair (sm_100 has packed fp32 arithmetic on such pairs).
__device__ __forceinline__ uint64_t pack_u32x2(uint32_t lo, uint32_t hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) { return pack_u32x2(__float_as_uint(lo), __float_as_uint(hi)); }
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& lo, float& hi) {
    uint32_t a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(v));
    lo = __uint_as_float(a);
    hi = __uint_as_float(b);
}
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {  // round to nearest even, per element
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Four weight codes as the bytes the MMA reads: the sign-magnitude bytes themselves (E4M3 path) or, in the integer-path
// build, their two's complement (per byte: (m ^ s) - s with s = 0xFF where the sign bit is set).
__device__ __forceinline__ uint32_t code_bytes(uint32_t v) {
    if constexpr (!kI8Path) {
        return v;
    } else {
        const uint32_t sg = ((v >> 7) & 0x01010101u) * 0xFFu;
        return __vsub4((v & 0x07070707u) ^ sg, sg);
    }
}

__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {  // round to nearest even, per element
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

}  // namespace
}  // namespace dirotq
