// Device-side building blocks: counter hash, set hash, row loads, the row-wise
// min-max quantizer with nearest-even or stochastic rounding (Section 3
// "Precision"/"Rounding", Algorithm 1).  Every FP32 operation that feeds a stored
// code is spelled with an explicit rounding intrinsic so that the compiler can
// neither contract nor reorder it.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace mpe {

constexpr uint32_t DOMAIN_INIT = 1, DOMAIN_SR = 2, DOMAIN_FLUSH = 3;
constexpr int LOC_MISS = -1;      // unique row not cache resident
constexpr int LOC_INVALID = -2;   // pseudo row collecting out-of-range indices

__host__ __device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x ^= x >> 16; x *= 0x7feb352dU; x ^= x >> 15; x *= 0x846ca68bU; x ^= x >> 16;
    return x;
}
__host__ __device__ __forceinline__ uint32_t absorb(uint32_t h, uint32_t w) { return mix32((h ^ w) + 0x9E3779B9U); }

// per-(row, step) key of the counter-based generator; one mixing round per column follows
__host__ __device__ __forceinline__ uint32_t rowkey(uint64_t seed, uint32_t domain, uint32_t table, uint32_t row, uint64_t step) {
    uint32_t h = 0x243F6A88U;
    h = absorb(h, (uint32_t)seed); h = absorb(h, (uint32_t)(seed >> 32));
    h = absorb(h, domain); h = absorb(h, table); h = absorb(h, row);
    h = absorb(h, (uint32_t)step); h = absorb(h, (uint32_t)(step >> 32));
    return h;
}
__device__ __forceinline__ float uniform01(uint32_t key, uint32_t column) {
    uint32_t bits = mix32(key ^ (column * 0x9E3779B9U + 0x7F4A7C15U));
    return __uint2float_rn(bits >> 8) * 0x1p-24f;   // exact
}
__host__ __device__ __forceinline__ uint32_t table_salt(uint64_t seed, uint32_t table) {
    uint32_t h = 0x13198A2EU;
    h = absorb(h, (uint32_t)seed); h = absorb(h, (uint32_t)(seed >> 32)); h = absorb(h, table);
    return h;
}
// h : row -> set (Section 3 "Cache Structure")
__device__ __forceinline__ int set_of(uint32_t row, uint32_t salt, int n_sets) {
    return (int)(((uint64_t)mix32(row ^ salt) * (uint64_t)(uint32_t)n_sets) >> 32);
}

// A row of `dim` values is handled by dim/4 consecutive lanes, four columns per lane.
__device__ __forceinline__ uint32_t group_mask(int lanes_per_row) {
    const int lane = threadIdx.x & 31;
    return lanes_per_row == 32 ? 0xffffffffU : (((1U << lanes_per_row) - 1U) << (lane & ~(lanes_per_row - 1)));
}

// The four stored values of one lane (columns 4*sub .. 4*sub+3) are BITS*4 adjacent bits of the row: one byte (INT2),
// one u16 (INT4), one u32 (INT8) or two u32 (FP16 table, BITS = 16); the lowest column sits in the lowest bits.
// Loads of memory that the running kernel does not write, so that the compiler may move them past its stores.  Not through the
// non-coherent path (ld.global.nc, __ldg): that one is for memory nobody writes while the kernel is resident, and a kernel launched by
// LAUNCH_NEXT is resident while the one before it still writes.  ld_once_*: data that is used once (a low-precision row on its way
// to FP32), without taking a line of L1, which is better spent on the FP32 rows that many bags share.
__device__ __forceinline__ float4 ld_f32x4(const void* p) {
    float4 v; asm("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p)); return v;
}
__device__ __forceinline__ int32_t ld_i32(const int32_t* p) { int32_t v; asm("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p)); return v; }
__device__ __forceinline__ uint32_t ld_once_u8(const void* p) { uint32_t v; asm("ld.global.L1::no_allocate.u8 %0, [%1];" : "=r"(v) : "l"(p)); return v; }
__device__ __forceinline__ uint32_t ld_once_u16(const void* p) { unsigned short v; asm("ld.global.L1::no_allocate.u16 %0, [%1];" : "=h"(v) : "l"(p)); return v; }
__device__ __forceinline__ uint32_t ld_once_u32(const void* p) { uint32_t v; asm("ld.global.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p)); return v; }
__device__ __forceinline__ uint2 ld_once_u32x2(const void* p) { uint2 v; asm("ld.global.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p)); return v; }
__device__ __forceinline__ float2 ld_once_f32x2(const void* p) { float2 v; asm("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p)); return v; }

// First statement of every kernel that is launched by LAUNCH_NEXT: lets the kernel behind it in the stream be set up from now on,
// and waits until the one before it has finished and its writes are visible.  Nothing of memory that another kernel writes may be
// touched before.  Returns the thread's number, which the compiler takes for a result of the wait: addresses formed from it, and what
// is loaded from there, cannot be moved in front of it, not even loads that may be moved past stores.
__device__ __forceinline__ uint32_t after_previous_kernel() {
    uint32_t thread = threadIdx.x;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" : "+r"(thread) :: "memory");
    return thread;
}

// Where the low-precision rows are: codes and (scale, bias) of row r at codes + r * code_stride and sb + r * sb_stride.  On the GPU
// both usually are parts of one record per row (see mpe_create_placed).
struct LowRows {
    uint8_t *codes, *sb;
    uint32_t code_stride, sb_stride;
    __host__ __device__ uint8_t* codes_of(int64_t r) const { return codes + r * (int64_t)code_stride; }
    __host__ __device__ float2* sb_of(int64_t r) const { return reinterpret_cast<float2*>(sb + r * (int64_t)sb_stride); }
};

template <int BITS, bool RO>
__device__ __forceinline__ uint2 load_codes4(const LowRows& low, int64_t grow, int sub) {
    const uint8_t* row = low.codes_of(grow);
    if (BITS == 16) return RO ? ld_once_u32x2(reinterpret_cast<const uint2*>(row) + sub) : reinterpret_cast<const uint2*>(row)[sub];
    uint32_t q;
    if (BITS == 8) q = RO ? ld_once_u32(reinterpret_cast<const uint32_t*>(row) + sub) : reinterpret_cast<const uint32_t*>(row)[sub];
    else if (BITS == 4) q = RO ? ld_once_u16(reinterpret_cast<const uint16_t*>(row) + sub) : reinterpret_cast<const uint16_t*>(row)[sub];
    else q = RO ? ld_once_u8(row + sub) : row[sub];
    return make_uint2(q, 0u);
}
template <int BITS>
__device__ __forceinline__ void store_packed4(const LowRows& low, int64_t grow, int sub, uint32_t q) {
    uint8_t* row = low.codes_of(grow);
    if (BITS == 8) reinterpret_cast<uint32_t*>(row)[sub] = q;
    else if (BITS == 4) reinterpret_cast<uint16_t*>(row)[sub] = (uint16_t)q;
    else row[sub] = (uint8_t)q;
}

// element-wise IEEE additions / fused multiply-adds
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z), __fadd_rn(a.w, b.w));
}
__device__ __forceinline__ float4 fma4(float m, float4 g, float4 x) {       // m * g + x, fused, per component
    return make_float4(__fmaf_rn(m, g.x, x.x), __fmaf_rn(m, g.y, x.y), __fmaf_rn(m, g.z, x.z), __fmaf_rn(m, g.w, x.w));
}
// minimum / maximum over the lanes of `mask` in one instruction (floating-point warp reduction of sm_100a)
__device__ __forceinline__ float group_min(float v, uint32_t mask) {
    float r; asm volatile("redux.sync.min.f32 %0, %1, %2;" : "=f"(r) : "f"(v), "r"(mask)); return r;
}
__device__ __forceinline__ float group_max(float v, uint32_t mask) {
    float r; asm volatile("redux.sync.max.f32 %0, %1, %2;" : "=f"(r) : "f"(v), "r"(mask)); return r;
}

// four stored values -> FP32: q*scale + bias for integer codes (Algorithm 1, up-conversion), exact for FP16
template <int BITS>
__device__ __forceinline__ float4 decode4(uint2 qq, float2 p) {
    float4 x;
    if (BITS == 16) {
        x.x = __half2float(__ushort_as_half((unsigned short)(qq.x & 0xffffu)));
        x.y = __half2float(__ushort_as_half((unsigned short)(qq.x >> 16)));
        x.z = __half2float(__ushort_as_half((unsigned short)(qq.y & 0xffffu)));
        x.w = __half2float(__ushort_as_half((unsigned short)(qq.y >> 16)));
        return x;
    }
    constexpr uint32_t M = (1u << (BITS & 15)) - 1u;
    const uint32_t q = qq.x;
    x.x = __uint2float_rn(q & M);
    x.y = __uint2float_rn((q >> (BITS & 15)) & M);
    x.z = __uint2float_rn((q >> ((2 * BITS) & 31)) & M);
    x.w = __uint2float_rn((q >> ((3 * BITS) & 31)) & M);
    return fma4(p.x, x, make_float4(p.y, p.y, p.y, p.y));      // q * s + b
}

// RO = the table is not written by the running kernel
template <int BITS, bool RO>
__device__ __forceinline__ float4 dequant4(const LowRows& low, int64_t grow, int sub) {
    float2 p = make_float2(1.0f, 0.0f);
    if (BITS != 16) p = RO ? ld_once_f32x2(low.sb_of(grow)) : *low.sb_of(grow);
    return decode4<BITS>(load_codes4<BITS, RO>(low, grow, sub), p);
}

// Four values -> their codes, packed with the first in the lowest bits; `stochastic` picks the rounding of Section 3 "Rounding" (it
// is the same for a whole kernel).  The integer part of y comes out of the mantissa of y + 2^23, rounded down (or to the nearest,
// ties to even): two full-rate additions where a rounding and a conversion instruction run at a quarter of the rate.  The 2^23 that
// stays in each term is taken off once, from the packed sum.  Scalar on purpose: with packed f32x2 arithmetic the moves that pair
// and unpair registers outnumbered the instructions it saved.
template <int BITS>
__device__ __forceinline__ uint32_t quant_pack(float4 x, float mn, float inv, uint32_t key, uint32_t column, bool stochastic) {
    constexpr float qmax = (float)((1 << BITS) - 1);
    constexpr uint32_t BASE = 0x4B000000u;                                      // 2^23 as FP32
    uint32_t packed = 0u - (BASE + (BASE << BITS) + (BASE << (2 * BITS)) + (BASE << (3 * BITS)));
    const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        // (x - b)/s as (x - b) * (1/s)
        const float y = fminf(fmaxf(__fmul_rn(__fsub_rn(v[i], mn), inv), 0.0f), qmax);
        float t;
        bool up = false;
        if (stochastic) {
            t = __fadd_rd(y, 8388608.0f);
            const float p = __fsub_rn(y, __fsub_rn(t, 8388608.0f));             // y - floor(y), exact
            up = uniform01(key, column + (uint32_t)i) < p;                      // x+ with probability p: expectation y
        } else t = __fadd_rn(y, 8388608.0f);
        packed += (__float_as_uint(t) + (up ? 1u : 0u)) << (BITS * i);
    }
    return packed;
}

// one value -> FP16 bits: the nearer neighbour, or one of the two neighbours x- <= x <= x+ (one unit in the last
// place apart) with P(x+) = (x - x-)/(x+ - x-)   (Section 3 "Rounding")
__device__ __forceinline__ uint32_t half1(float x, uint32_t key, uint32_t column, bool stochastic) {
    const float v = fminf(fmaxf(x, -65504.0f), 65504.0f);                    // stay inside the finite FP16 range
    if (!stochastic) return __half_as_ushort(__float2half_rn(v));
    const __half lo = __float2half_rd(v), hi = __float2half_ru(v);
    const unsigned short blo = __half_as_ushort(lo), bhi = __half_as_ushort(hi);
    if (blo == bhi) return blo;
    const float flo = __half2float(lo), fhi = __half2float(hi);
    const float p = __fdiv_rn(__fsub_rn(v, flo), __fsub_rn(fhi, flo));        // exact
    return uniform01(key, column) < p ? bhi : blo;
}

// Down-convert one FP32 row (four columns per lane) into the low-precision table.
template <int BITS>
__device__ __forceinline__ void quantize_store(float4 x, const LowRows& low, int64_t grow, int sub, int lanes_per_row, uint32_t key, bool stochastic) {
    if (BITS == 16) {       // FP16 table: element-wise, no scale or bias
        const uint32_t c = 4u * (uint32_t)sub;
        reinterpret_cast<uint2*>(low.codes_of(grow))[sub] =
            make_uint2(half1(x.x, key, c, stochastic) | (half1(x.y, key, c + 1, stochastic) << 16),
                       half1(x.z, key, c + 2, stochastic) | (half1(x.w, key, c + 3, stochastic) << 16));
        return;
    }
    const uint32_t mask = group_mask(lanes_per_row);
    float mn = fminf(fminf(x.x, x.y), fminf(x.z, x.w));
    float mx = fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w));
    if (lanes_per_row > 1) {                               // which zero a tie between -0 and +0 yields does not matter below
        mn = group_min(mn, mask);
        mx = group_max(mx, mask);
    }
    mn = __fadd_rn(mn, 0.0f);                              // -0 -> +0
    const float qmax = (float)((1 << (BITS & 15)) - 1);
    float s = __fdiv_rn(__fsub_rn(mx, mn), qmax);          // s = (max - min)/(2^N - 1)
    float inv = 0.0f;
    if (s >= 1.17549435e-38f) inv = __fdiv_rn(1.0f, s);
    if (inv == 0.0f) s = 0.0f;
    const uint32_t c = 4u * (uint32_t)sub;
    store_packed4<BITS>(low, grow, sub, quant_pack<BITS & 15>(x, mn, inv, key, c, stochastic));
    if (sub == 0) *low.sb_of(grow) = make_float2(s, mn);
}

}  // namespace mpe
