// 64-bit modular arithmetic for primes of at most 60 bits (device).
//
//  * Shoup multiplication by a fixed operand w with w' = floor(w 2^64 / q):
//    x w - floor(x w' / 2^64) q lies in [0, 2q) for any 64-bit x.
//  * Single-word Barrett reduction of a 128-bit value x < 2^(63 + bitlen(q)):
//    with s = bitlen(q) - 1 and mu = floor(2^(64+s) / q), the estimate
//    floor((x >> s) mu / 2^64) is at most 3 below floor(x / q), so the
//    remainder is in [0, 3q) before two conditional subtractions.  Sums of up
//    to 8 products of residues (each below 2^60 and below the target prime)
//    stay inside that bound.
#pragma once
#include <stdint.h>

#include "pft_internal.h"

namespace pft {

// Programmatic dependent launch.  A kernel started by launch_pdl becomes resident as the CTAs of the
// kernel before it on the stream run out; pdl_wait returns when everything before this kernel has
// completed and is visible.  Before pdl_wait a kernel reads only its parameters and the context's
// constant tables.  Operands are read after it, with plain loads through plain pointers: __ldg
// (ld.global.nc) is for data that nothing writes during the kernel's whole life, which begins here
// before the previous kernel's words are visible, and neither it nor a __restrict__ pointer's load
// is ordered by the wait.  (Letting the next kernel in earlier, with griddepcontrol.launch_dependents
// at the start, measured slower: its waiting CTAs hold the slots.  One rotation at level 30: 481 us
// with ordinary launches, 486 with the early trigger, 453 without.)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ u64 mulhi(u64 a, u64 b) { return __umul64hi(a, b); }

// x * w mod q in [0, 2q)
__device__ __forceinline__ u64 mul_shoup_lazy(u64 x, u64 w, u64 wp, u64 q) {
    u64 hq = mulhi(x, wp);
    return x * w - hq * q;
}
__device__ __forceinline__ u64 mul_shoup(u64 x, u64 w, u64 wp, u64 q) {
    u64 r = mul_shoup_lazy(x, w, wp, q);
    return r >= q ? r - q : r;
}

struct U128 {
    u64 lo, hi;
};
__device__ __forceinline__ U128 mul_wide(u64 a, u64 b) {
    U128 r;
    r.lo = a * b;
    r.hi = mulhi(a, b);
    return r;
}
__device__ __forceinline__ void mac_wide(U128& acc, u64 a, u64 b) {
    u64 lo = a * b, hi = mulhi(a, b);
    acc.lo += lo;
    acc.hi += hi + (acc.lo < lo ? 1 : 0);
}

// Sums of up to 8 products of values below 2^60 in three 64-bit partial sums: with
// a = a1 2^30 + a0 and b = b1 2^30 + b0 (all halves below 2^30),
//   sum a b = S00 + 2^30 S01 + 2^60 S11,  S00 = sum a0 b0 < 2^63,
//   S01 = sum (a0 b1 + a1 b0) < 2^64,  S11 = sum a1 b1 < 2^63,
// so every term is one 32x32+64 multiply-add and no carry is handled per term.
struct Acc3 {
    u64 s00, s01, s11;
};
__device__ __forceinline__ void split30(u64 a, u32& lo, u32& hi) {
    lo = (u32)a & 0x3fffffffu;
    hi = (u32)(a >> 30);
}
// acc + a b as one widening multiply-add (32 x 32 + 64 -> 64)
__device__ __forceinline__ u64 mad_wide(u32 a, u32 b, u64 acc) {
    u64 r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(acc));
    return r;
}
__device__ __forceinline__ void acc3_mac(Acc3& A, u32 a0, u32 a1, u32 b0, u32 b1) {
    A.s00 = mad_wide(a0, b0, A.s00);
    A.s01 = mad_wide(a0, b1, A.s01);
    A.s01 = mad_wide(a1, b0, A.s01);
    A.s11 = mad_wide(a1, b1, A.s11);
}
// Karatsuba form: S00 = sum a0 b0, S11 = sum a1 b1 and SM = sum (a0 + a1)(b0 + b1) (each
// factor below 2^31); the middle sum is SM - S00 - S11.  Three products per term instead of
// four.  SM is kept modulo 2^64: up to 4 terms it does not wrap; up to 8 terms it may, but the
// middle sum itself is below 2^64 (8 terms of a0 b1 + a1 b0 < 2^61), so SM - S00 - S11 taken
// modulo 2^64 is still exactly the middle sum.
struct Acc3K {
    u64 s00, sm, s11;
};
__device__ __forceinline__ void acc3k_mac(Acc3K& A, u32 a0, u32 a1, u32 a01, u32 b0, u32 b1, u32 b01) {
    A.s00 = mad_wide(a0, b0, A.s00);
    A.s11 = mad_wide(a1, b1, A.s11);
    A.sm = mad_wide(a01, b01, A.sm);
}
__device__ __forceinline__ Acc3 acc3k_fold(const Acc3K& A) { return Acc3{A.s00, A.sm - A.s00 - A.s11, A.s11}; }
// the 128-bit value S00 + 2^30 S01 + 2^60 S11
__device__ __forceinline__ U128 acc3_value(const Acc3& A) {
    U128 r;
    r.lo = A.s00;
    r.hi = 0;
    const u64 t1 = A.s01 << 30;
    r.lo += t1;
    r.hi += (A.s01 >> 34) + (r.lo < t1 ? 1 : 0);
    const u64 t2 = A.s11 << 60;
    r.lo += t2;
    r.hi += (A.s11 >> 4) + (r.lo < t2 ? 1 : 0);
    return r;
}

// Montgomery reduction of the partial sums with R = 2^60, in two steps of 30 bits on the sums as they
// are: V = S00 + 2^30 S01 + 2^60 S11 -> V 2^-60 mod p, below V / 2^60 + p.  Each step adds a multiple of p
// that clears 30 bits: m = (low 30 bits) (-p^-1) mod 2^30, p = p1 2^30 + p0.  S00 and S11 hold up to 12
// products (12 2^60 + 2^60 < 2^64); S01 takes m0 p1 and a carry besides: with NORM its own high part goes
// to S11 first (sums of more than 4 terms of 60-bit factors), without it S01 < 2^63.  Against forming
// the 128-bit value and one 64-bit Montgomery step this is 4 widening and 2 low-word multiplies and
// about 20 instructions instead of 5 and 2 and about 50.
struct Mont30 {
    u32 p0, p1, np;
};
__device__ __forceinline__ Mont30 mont30(u64 p, u64 mneg) {
    return Mont30{(u32)p & 0x3fffffffu, (u32)(p >> 30), (u32)mneg & 0x3fffffffu};
}
template <bool NORM>
__device__ __forceinline__ u64 mont60(const Acc3& A, const Mont30& M) {
    u64 s01 = A.s01, s11 = A.s11;
    if (NORM) {
        s11 += s01 >> 30;
        s01 = (u32)s01 & 0x3fffffffu;
    }
    const u32 m0 = ((u32)A.s00 * M.np) & 0x3fffffffu;
    s01 = mad_wide(m0, M.p1, s01 + (mad_wide(m0, M.p0, A.s00) >> 30));
    const u32 m1 = ((u32)s01 * M.np) & 0x3fffffffu;
    return mad_wide(m1, M.p1, s11 + (mad_wide(m1, M.p0, s01) >> 30));
}

// x mod q for x = hi 2^64 + lo < 2^(64 + s)
__device__ __forceinline__ u64 barrett_reduce(u64 hi, u64 lo, const DPrime& P) {
    u64 x1 = (hi << (64 - P.s)) | (lo >> P.s);
    u64 qt = mulhi(x1, P.mu);
    u64 r = lo - qt * P.q;
    if (r >= 2 * P.q) r -= 2 * P.q;
    if (r >= P.q) r -= P.q;
    return r;
}
__device__ __forceinline__ u64 mulmod(u64 a, u64 b, const DPrime& P) {
    U128 x = mul_wide(a, b);
    return barrett_reduce(x.hi, x.lo, P);
}
__device__ __forceinline__ u64 reduce64(u64 a, const DPrime& P) { return barrett_reduce(0, a, P); }

__device__ __forceinline__ u64 addmod(u64 a, u64 b, u64 q) {
    u64 s = a + b;
    return s >= q ? s - q : s;
}
__device__ __forceinline__ u64 submod(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }

__device__ __forceinline__ DPrime load_prime(const DPrime* tab, int i) {
    DPrime p;
    p.q = __ldg(&tab[i].q);
    p.mu = __ldg(&tab[i].mu);
    p.r64 = __ldg(&tab[i].r64);
    p.mneg = __ldg(&tab[i].mneg);
    p.r60 = __ldg(&tab[i].r60);
    p.s = __ldg(&tab[i].s);
    return p;
}

// Galois automorphism X -> X^g in the evaluation layout, as a source index.
// Entry i holds a(psi^(2 brv(i) + 1)); a(X^g) there equals a(psi^((2 brv(i) + 1) g)),
// i.e. entry brv(((2 brv(i) + 1) g mod 2N - 1) / 2) of the input.
__device__ __forceinline__ u32 automorph_src(u32 i, int logn, u64 g) {
    const u32 mask2n = (2u << logn) - 1;
    const u32 bi = __brev(i) >> (32 - logn);
    const u32 e = (u32)(((u64)(2 * bi + 1) * g) & mask2n);
    return __brev((e - 1) >> 1) >> (32 - logn);
}
// The top bits of a source index depend only on the top bits of its destination, so every aligned
// block of 2^b destinations reads one aligned block of 2^b sources.

}  // namespace pft
