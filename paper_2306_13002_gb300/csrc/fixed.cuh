// Block-scaled 64-bit fixed point: sums of FP64 values on the integer pipes.
//
// GB300 issues 2 FP64 operations per clock and SM but 64 to 128 integer ones, so a kernel that
// mostly adds neighbours runs 5 to 8 times longer on the FP64 pipe than it takes to add the same
// numbers as 64-bit integers (two 32-bit instructions per sum of three terms). The marches that use
// this header convert every input once, when its plane is staged, to
//     q = floor(v / d) + bias,   d = 2^(E0 - 1023 - 59),
// with one exponent E0 per block and segment (the largest exponent staged), |v / d| < 2^60. Integer
// sums are exact, so the only errors are the conversion's (less than d per input, 2^-59 of the
// segment's largest value) and the final rounding. FP64 rounds every partial sum to 53 bits.
//
// Values far below the block's largest lose their low bits in this form. The star march tests each point for
// it and evaluates those that fail in FP64; the RHS march takes only planes whose values keep ranges that
// leave its errors below FP64's. Both leave the form when an input exceeds E0 or is not finite. What a
// block leaves runs in a staged FP64 march at its end.
#pragma once

#include "device_ops.cuh"

namespace acs {

typedef unsigned long long u64;
typedef unsigned int u32;

// Exponents a segment may be scaled to: results and intermediate scales stay normal numbers.
constexpr int kFixMinExp = 520, kFixMaxExp = 1600;

// The thread's coordinates, read anew at every call: what is reckoned from them is then not carried in
// registers across the loops over segments and units of work.
__device__ __forceinline__ int tid_x() {
    int t;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    return t;
}
__device__ __forceinline__ int tid_y() {
    int t;
    asm volatile("mov.u32 %0, %%tid.y;" : "=r"(t));
    return t;
}

// Planes a block leaves for the FP64 march.
constexpr int kBlockLeft = 16;
struct BlockLeft {
    int i0, j0, from, to;
};

// PTX shifts clamp amounts of 64 and more (the result is then 0).
__device__ __forceinline__ u64 shr64(u64 v, int s) {
    u64 r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}

// 16-byte shared-memory accesses by 32-bit address (the compiler loses the address space of a
// rounded-up base and would use generic ones).
struct U64x2 {
    u64 x, y;
};
__device__ __forceinline__ U64x2 lds2(u32 addr) {
    U64x2 r;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(r.x), "=l"(r.y) : "r"(addr) : "memory");
    return r;
}
__device__ __forceinline__ void sts1(u32 addr, u64 v) {
    asm volatile("st.shared.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ u64 lds1(u32 addr) {
    u64 r;
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(r) : "r"(addr) : "memory");
    return r;
}

__device__ __forceinline__ int lds_int(u32 addr) {
    int r;
    asm volatile("ld.shared.s32 %0, [%1];" : "=r"(r) : "r"(addr) : "memory");
    return r;
}
__device__ __forceinline__ int4 lds_int4(u32 addr) {
    int4 r;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(addr) : "memory");
    return r;
}

__device__ __forceinline__ u64 pack64(u32 hi, u32 lo) { return ((u64)hi << 32) | lo; }
__device__ __forceinline__ u32 hi32(u64 v) { return (u32)(v >> 32); }
__device__ __forceinline__ u32 lo32(u64 v) { return (u32)v; }

// The bits v of a double as fixed point: floor(v / d) + (bias_hi << 32), its leading bit at 59 for the
// exponent E0 (an exact negative multiple of d comes out one lower). s: the bits between v's exponent
// and E0, negative if it exceeds E0 (infinities and NaN do). Zeros and values too small for the scale
// give 0 or -1. E0 >= kFixMinExp.
__device__ __forceinline__ u64 to_fixed_by(u64 v, int E0, u32 bias_hi, int& s) {
    const u32 hi = hi32(v), lo = lo32(v);
    s = E0 - (int)((hi << 1) >> 21);
    const u32 mh = (__funnelshift_l(lo, hi, 7) & 0x07ffffffu) | 0x08000000u;
    const u64 m = shr64(pack64(mh, lo << 7), s);
    const u32 sg = (u32)((int)hi >> 31);
    return pack64((hi32(m) ^ sg) + bias_hi, lo32(m) ^ sg);
}
// The same; `bad` turns negative if v's exponent exceeds E0.
__device__ __forceinline__ u64 to_fixed(u64 v, int E0, u32 bias_hi, int& bad) {
    int s;
    const u64 r = to_fixed_by(v, E0, bias_hi, s);
    bad |= s;
    return r;
}

// Constants that turn a 64-bit integer t into the double t * 2^e2 (times -1 if `neg`): the two
// halves of t as mantissas of doubles with fixed exponents, and the sum of those exponents' values.
struct FixOut {
    u32 hi, lo;
    double off;
};
__device__ __forceinline__ FixOut fix_out(int e2, bool neg) {
    const u32 add = ((u32)e2 << 20) ^ (neg ? 0x80000000u : 0u);
    // 2^84 + 2^63 + 2^52, negated and scaled
    return FixOut{0x45300000u + add, 0x43300000u + add,
                  __hiloint2double((int)((0x45300000u + add) ^ 0x80000000u), (int)0x80100000u)};
}
// Two FP64 additions, the first exact: t * 2^e2 rounded once, to nearest.
__device__ __forceinline__ double from_fixed(i64 t, const FixOut& c) {
    const double h = __hiloint2double((int)c.hi, (int)(hi32((u64)t) ^ 0x80000000u));
    const double l = __hiloint2double((int)c.lo, (int)lo32((u64)t));
    return (h + c.off) + l;
}

// Weighted sums of 64-bit words. A weight W is held as Wh 2^LB + Wl; the products' four partial
// sums are kept apart (each fits 64 bits, but for hh, which only needs to be right modulo 2^64)
// and joined once per point. A negative Wh is multiplied as Wh + 2^32: fix_neg takes the excess out.
struct FixAcc {
    u64 hh, hl, lh, ll;
};
// One multiply-add instruction each (written out: the compiler splits the C form in two).
__device__ __forceinline__ void mad_wide(u64& acc, u32 x, u32 y) {
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(acc) : "r"(x), "r"(y));
}
__device__ __forceinline__ void fix_mac(FixAcc& a, u64 v, u32 wh, u32 wl) {
    mad_wide(a.hh, hi32(v), wh);
    mad_wide(a.hl, hi32(v), wl);
    mad_wide(a.lh, lo32(v), wh);
    mad_wide(a.ll, lo32(v), wl);
}
__device__ __forceinline__ void fix_neg(FixAcc& a, u32 sum_hi, u32 sum_lo) {
    a.hh = pack64(hi32(a.hh) - sum_hi, lo32(a.hh));
    a.lh = pack64(hi32(a.lh) - sum_lo, lo32(a.lh));
}

}  // namespace acs
