// tile_common.cuh -- device helpers shared by the attention kernels on tcgen05:
// exact e4m3 widening, q narrowing with its range check, bounded waits of a
// warp, partial-row stores.
#pragma once

#include "device_common.cuh"
#include "internal.h"

namespace parason {
namespace {

__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint32_t two_bytes) {
    uint32_t out;
    asm("{\n\t.reg .b16 lo, hi;\n\t"
        "mov.b32 {lo, hi}, %1;\n\t"
        "cvt.rn.f16x2.e4m3x2 %0, lo;\n\t}"
        : "=r"(out)
        : "r"(two_bytes));
    return out;
}

// Four e4m3 values (one word) widened exactly to two f16 pairs: bytes 0-1
// to `lo`, bytes 2-3 to `hi`.
__device__ __forceinline__ void e4m3x4_to_f16x2x2(uint32_t four_bytes, uint32_t &lo, uint32_t &hi) {
    asm("{\n\t.reg .b16 l, h;\n\t"
        "mov.b32 {l, h}, %2;\n\t"
        "cvt.rn.f16x2.e4m3x2 %0, l;\n\t"
        "cvt.rn.f16x2.e4m3x2 %1, h;\n\t}"
        : "=r"(lo), "=r"(hi)
        : "r"(four_bytes));
}

// A bf16 pair of q narrowed to an f16 pair for the e4m3 MMAs.  The f16
// values are exact for |q| < 65504 (tiny values lose low bits); an element
// of magnitude 65520 or more (including inf) would round to inf, so `big` is
// set and the caller reports PARASON_ERANGE rather than returning a silently
// wrong result.  NaN is passed through and not flagged.
__device__ __forceinline__ uint32_t q_pair_to_f16(uint32_t two, bool &big) {
    const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162 *>(&two);
    const float lo = __low2float(b), hi = __high2float(b);
    big |= fmaxf(fabsf(lo), fabsf(hi)) >= 65520.f;
    return dev::pack_f16(lo, hi);
}

// Record PARASON_ERANGE once per warp if any lane saw an out-of-range q.
__device__ __forceinline__ void report_q_range(const AttnArgs &a, bool big, int lane) {
    if (__any_sync(0xffffffffu, big) && lane == 0) dev::record_error(a.err, PARASON_ERANGE, kSiteQRange);
}

__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(addr));
    return v;
}

// x = -inf when q >= seen (a score's bits, or its value).  Volatile, so that
// the few blocks with hidden keys branch to a run of these: as plain C++ they
// were folded into selects that every block ran.
__device__ __forceinline__ void hide_from(uint32_t &x, int q, int seen) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ge.s32 p, %1, %2;\n\t"
        "selp.b32 %0, 0xff800000, %0, p;\n\t}"
        : "+r"(x)
        : "r"(q), "r"(seen));
}

__device__ __forceinline__ void hide_from(float &x, int q, int seen) {
    uint32_t u = __float_as_uint(x);
    hide_from(u, q, seen);
    x = __uint_as_float(u);
}

// 32 consecutive fp32 values of one partial row (128 bytes, 32-byte
// aligned), scaled, as four 32-byte stores: every store fills whole sectors
// (16-byte stores from the 32 rows of a warp left each sector to be filled
// by two instructions).
__device__ __forceinline__ void store_row32(float *dst, const uint32_t (&v)[32], float scale) {
#pragma unroll
    for (int q = 0; q < 32; q += 8)
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + q),
                     "f"(__uint_as_float(v[q]) * scale), "f"(__uint_as_float(v[q + 1]) * scale),
                     "f"(__uint_as_float(v[q + 2]) * scale), "f"(__uint_as_float(v[q + 3]) * scale),
                     "f"(__uint_as_float(v[q + 4]) * scale), "f"(__uint_as_float(v[q + 5]) * scale),
                     "f"(__uint_as_float(v[q + 6]) * scale), "f"(__uint_as_float(v[q + 7]) * scale)
                     : "memory");
}

__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity, long long limit,
                                        volatile int *abort) {
    return dev::mbar_wait_bounded(bar, parity, limit, abort);
}

// one warp: lane 0 waits, the warp agrees on the outcome
__device__ __forceinline__ bool tc_warp_wait(uint32_t bar, uint32_t parity, long long limit,
                                             volatile int *abort, int lane) {
    int ok = 1;
    if (lane == 0) ok = tc_wait(bar, parity, limit, abort) ? 1 : 0;
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

__device__ __forceinline__ void tc_fail(const AttnArgs &a, volatile int *abort, int site) {
    if (!*abort) {
        *abort = 1;
        dev::record_error(a.err, PARASON_ETIMEOUT, site);
    }
}

}  // namespace
}  // namespace parason
