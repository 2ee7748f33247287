// lb_f64.cuh -- FP64 arithmetic of the plain step, arranged for a chip whose
// FP64 pipe is its narrowest part.
//
// A GB300 SM starts one FP64 warp instruction every 16 to 19 clocks (2 lanes)
// against 4 instructions of every other kind per clock, so the plain FP64 step
// is bound by the number of its FP64 instructions and nothing else.  What is
// measured on the device (clocks an SM spends per warp instruction):
//   fma with three register operands                       16.0
//   add, multiply, fma with a constant operand              19.0
//   product by the integer routine below, alone             16.1
//   add + multiply 40.1, add + integer product              22.8
// The step therefore keeps only sums on the FP64 pipe, each written as an fma
// with the factor 1 in a register (exact: one rounding, as the add), and forms
// its products in integer instructions, which run beside them.  Every result
// has the bits of the IEEE operation it stands for, so the step still rounds
// as a plain evaluation of the equations, operation by operation.  With the
// products shared between neighbours (Stage64) a node of the one-pass step
// costs 369 FP64 instructions instead of 641; a 1024^2 step 0.67 ms instead
// of 1.30, its FP64 pipe 86 % busy.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbk {

// A factor of an integer product: sign and exponent bits, the 53-bit mantissa
// as (21, 32) bits, and whether it is zero.
struct Factor {
    uint32_t se, m1, m0;
    bool zero;
};

__device__ __forceinline__ Factor factor(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    Factor f;
    f.zero = ((hi & 0x7fffffffu) | lo) == 0u;
    f.se = hi & 0xfff00000u;
    f.m1 = (hi & 0x000fffffu) | 0x00100000u;
    f.m0 = lo;
    return f;
}

// The IEEE product (round to nearest even) of two factors that are zero or
// normal, where the product is zero or normal too.  The second mantissa is
// aligned to the top of 64 bits, so the upper half H of the 117-bit product
// has 52 or 53 bits; one conditional shift normalises it, the lower half
// decides the rounding, and a carry out of the mantissa runs into the
// exponent by itself.  Signs add up in the top bit.
__device__ __forceinline__ double factor_mul(const Factor &a, const Factor &b)
{
    const uint32_t b1 = (b.m1 << 11) | (b.m0 >> 21), b0 = b.m0 << 11;
    const uint64_t p00 = (uint64_t)a.m0 * b0;
    const uint64_t t = (uint64_t)a.m0 * b1 + (p00 >> 32);
    const uint64_t v = (uint64_t)a.m1 * b0 + (uint32_t)t;
    const uint64_t H = (uint64_t)a.m1 * b1 + (t >> 32) + (v >> 32);
    uint32_t hh = (uint32_t)(H >> 32), hl = (uint32_t)H, lh = (uint32_t)v;
    const uint32_t lost = (uint32_t)p00;
    const uint32_t short_bit = ~hh & 0x00100000u, n = short_bit >> 20;   // 1: H has 52 bits
    hh = __funnelshift_l(hl, hh, n);
    hl = __funnelshift_l(lh, hl, n);
    lh = __funnelshift_l(lost, lh, n);
    const uint32_t top = hh + (a.se + b.se - 0x3ff00000u - short_bit);
    uint32_t rl, rh;
    // up where the discarded part lh:lost is above one half, or one half and
    // H odd: the carry of lh + 0x7fffffff + (1 if H is odd or lost is not 0)
    asm("{\n\t.reg .u32 t;\n\t"
        "add.cc.u32 t, %2, 0xffffffff;\n\t"
        "addc.cc.u32 t, %3, 0x7fffffff;\n\t"
        "addc.cc.u32 %0, %4, 0;\n\t"
        "addc.u32 %1, %5, 0;\n\t}"
        : "=r"(rl), "=r"(rh)
        : "r"(lost | (hl & 1u)), "r"(lh), "r"(hl), "r"(top));
    const bool z = a.zero || b.zero;
    return __hiloint2double((int)(z ? (a.se ^ b.se) & 0x80000000u : rh), (int)(z ? 0u : rl));
}

// Where the node's products are formed, every factor and every product is
// zero or normal, provided that
//   the populations, densities and psi it reads are zero or in
//     [2^-179, 2^77) (base_outside() is 0),
//   the couplings, relaxation rates and body forces are zero or in
//     [2^-58, 2^64) (checked on the host: Lat::products), so that times a weight
//     of at least 1/36 they are above 2^-64, and
//   the velocity's components are zero or in [2^-255, 2^256)
//     (velocity_outside() is 0).
// A nonzero sum is at least 2^-53 times its smallest term, so stencil sums
// are above 2^-250, forces above 2^-550, the Guo vectors above 2^-310, their
// products with the force above 2^-920 and with (1 - omega/2) w above
// 2^-980; the largest magnitudes stay below 2^700.
__device__ __forceinline__ uint32_t base_outside(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    // exponent fields 0x34c .. 0x44b, moved down, leave the top three bits clear
    return (((hi & 0x7fffffffu) | lo) == 0u) ? 0u : (hi - 0x34c00000u) & 0x70000000u;
}
__device__ __forceinline__ uint32_t velocity_outside(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    // exponent fields 0x300 .. 0x4ff, moved up by 0x100, have top bits 10
    return (((hi & 0x7fffffffu) | lo) == 0u) ? 0u : ((hi + 0x10000000u) ^ 0x40000000u) & 0x60000000u;
}

// 1.0 in a register, for kernels without a lattice descriptor in memory.
__device__ __forceinline__ double opaque_one()
{
    double v;
    asm volatile("mov.f64 %0, 0d3FF0000000000000;" : "=d"(v));
    return v;
}

// Arithmetic of a node: sums as register fmas, products by factor_mul (kInt)
// or the FP64 pipe (the same bits).
template <bool kInt>
struct Arith64 {
    double one;   // 1.0, in a register the compiler knows nothing about
    __device__ __forceinline__ explicit Arith64(double one_) : one(one_) {}
    __device__ __forceinline__ double add(double a, double b) const { return __fma_rn(a, one, b); }
    __device__ __forceinline__ double sub(double a, double b) const { return __fma_rn(-b, one, a); }
    __device__ __forceinline__ double mul(double a, double b) const
    {
        if constexpr (kInt) return factor_mul(factor(a), factor(b));
        else return __dmul_rn(a, b);
    }
};

// ---- exp and the two divisions of a node -----------------------------------------

// exp(-r) by table (P. T. P. Tang, "Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15, 1989):
// with j the nearest integer to 512 r and t = r - j/512 (exact),
//   exp(-r) = T_j exp(-t) = T_j + T_j p,   p = -t + t^2 (1/2 - t/6 + t^2/24 - t^3/120)
// to 2^-69 for |t| <= 2^-10, T_j as a double and its remainder.  10 FP64
// instructions, where exp() takes 15 (1024^2 one-pass step 704 -> 674 us, 333 x 97
// 34.1 -> 33.0, 64^2 11.4 -> 10.9).  Largest error seen on 2e7 arguments 0.5015 ulp.  Outside the
// table (densities below 0 or from 2 on) exp().
constexpr int kExpSteps = 512, kExpSize = 2 * kExpSteps + 1;

__device__ __forceinline__ double exp_minus(double r, double one, const double2 *__restrict__ table)
{
    if (!(r >= 0.0 && r < 2.0)) return exp(-r);
    constexpr double kRound = 0x1.8p43;   // 1.5 2^52 / 512: the sum's last bits count in 1/512
    const double m = __fma_rn(r, one, kRound);
    const double2 T = __ldg(&table[__double2loint(m)]);
    const double t = __fma_rn(__fma_rn(-kRound, one, m), -one, r);
    double q = __fma_rn(t, -1.0 / 120.0, 1.0 / 24.0);
    q = __fma_rn(q, t, -1.0 / 6.0);
    q = __fma_rn(q, t, 0.5);
    const double p = __fma_rn(t * q, t, -t);
    return __fma_rn(T.x, one, __fma_rn(T.x, p, T.y));
}

// psi = 1 - exp(-rho) (Sec. II B)
__device__ __forceinline__ double psi64(double r, double one, const double2 *__restrict__ table)
{
    return __fma_rn(-exp_minus(r, one, table), one, 1.0);
}

// x / d, rounded to nearest, from y = 1 / d rounded to nearest (__drcp_rn), for
// several x by one d.  P. Markstein ("Computation of elementary functions on the
// IBM RISC System/6000 processor", IBM J. Res. Dev. 34, 1990): where y is the
// rounded reciprocal and q one of the two doubles next to x / d, the residual
// x - q d is exact and q + (x - q d) y rounds to the rounded quotient.  x y
// itself may be off by 3/2 ulp (half a unit of its own rounding, up to one from
// y's), so a first correction brings it next to x / d: its residual is within
// 2^-52 of itself, so the sum is x / d within 2^-50 ulp before it is rounded.
// Holds where nothing leaves the normal range; d = 0 and the like give NaN, for
// the caller to find.  The tile kernels share one reciprocal: with a plain
// division per component the collide kernel of the two-pass step takes 12 % more
// (1024^2 719 us a step against 643; k_small64 forms one quotient a warp and
// divides).
__device__ __forceinline__ double quotient64(double x, double d, double y)
{
    double q = x * y;
    q = __fma_rn(__fma_rn(-q, d, x), y, q);
    return __fma_rn(__fma_rn(-q, d, x), y, q);
}

}  // namespace lbk
