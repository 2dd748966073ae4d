// push64.cuh -- the per-particle arithmetic of the float64 mode, shared by the
// push kernel (push.cu) and the many-step launch (steps64.cu).
//
// GB300 issues float64 at 2 lanes per clock per SM, so a float64 instruction
// of a warp takes the pipe for 16 clocks, the time of some 40 integer
// instructions.  The kernel keeps five per particle -- gather, kick, v v', sum
// v', drift -- and does the rest in integers:
//   locate    u = x NG/L as the high 64 bits of the product of the two
//             mantissas, shifted to F = 62 - floor(log2(NG)) bits after the binary
//             point (float64 keeps 52 - log2(u)); plus 1/2, its integer part is
//             the tile index and the rest the fraction;
//   gather    E_l + f (E_r - E_l) = fma(1 + f, dE, E_l - dE): 1 + f is the
//             fraction's bits under the exponent of 1, dE and E_l - dE are
//             kept as pairs in shared memory;
//   deposit   the weights are integers of 2^-53, f truncated to F bits and those
//             (the fraction of a float64 u + 1/2 >= 1/2 is a multiple of 2^-53
//             at best, and of NG 2^-53 at the far end of the box), summed exactly: runs of equal cell in registers (two open runs
//             of a thread's 4 particles, as PAIR), then in a tile of three
//             32-bit words per node.  Native 32-bit shared adds take the place
//             of float64 compare-and-swap loops, and the density no longer
//             depends on the order of the adds.
// The tile goes to global memory as two 64-bit sums per node, of the low 40
// bits and of the rest: at most 4096 blocks of less than 2^40 each, so neither
// needs a carry.
// Measured (2^24 particles, 1024 cells, sorted every 20 steps): 178 us a push,
// 145 us of it the five float64 instructions at the pipe's rate; 353 us with
// the two s = x NG/L + 1/2 as float64 FMAs and the wrap predicated (9.3 float64
// instructions), 1509 us with float64 floors, a segmented shuffle sum of the
// weights and float64 shared adds.
#pragma once

#include "particle_ops.cuh"

namespace pic {

constexpr u64 kOne53 = 1ull << 53;

struct Loc64 {
    unsigned j;                   // tile index (left node + 1)
    unsigned fh, fl;              // fraction in 2^-64
    bool ok;
};

struct Push64 {
    const double2 *pair;          // (E_l - dE, dE) of tile index j
    u64 lbits;                    // bits of L
    u64 wide;                     // mantissa of NG/L, its top bit set
    int frac_bits;                // F
    int shift;                    // u = high(mantissa(x) wide) >> (shift - exponent bits of x)
};

__device__ __forceinline__ Push64 push64_consts(const PushArgs64 &a, const double2 *pair) {
    Push64 c;
    c.pair = pair;
    c.lbits = (u64)__double_as_longlong(a.length);
    const u64 w = (u64)__double_as_longlong(a.inv_dx);
    c.wide = ((w & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 11;
    // U = u 2^F must hold NG + 1/2 in 64 bits: F = 63 - (bits of NG)
    c.frac_bits = 31 + __clz(a.ng);
    // x = M 2^(ex - 63), NG/L = W 2^(k - 63): u 2^F = high64(M W) 2^(ex + k - 62 + F)
    const int k = (int)(w >> 52) - 1023;
    c.shift = 62 - c.frac_bits - k + 1023;
    return c;
}

__device__ __forceinline__ Loc64 locate64(double x, double inv_dx, int ng, const Push64 &c) {
    const u64 b = (u64)__double_as_longlong(x);
    Loc64 l;
    u64 U;
    if (b < c.lbits) {                               // 0 <= x < L
        const u64 m = ((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 11;
        const unsigned r = (unsigned)(c.shift - (int)(b >> 52));
        U = r < 64u ? __umul64hi(m, c.wide) >> r : 0ull;   // u < 2^-F: 0
        U += 1ull << (c.frac_bits - 1);
        l.ok = true;
    } else {
        // outside the box: what lies within half a cell of it (left of node 0 or
        // right of node NG - 1) still has two nodes
        const double s = fma(x, inv_dx, 0.5);
        l.ok = s >= 0.0 && s < (double)(ng + 1);
        U = l.ok ? __double2ull_rz(scalbn(s, c.frac_bits)) : 0ull;
    }
    l.j = (unsigned)(U >> c.frac_bits);
    const u64 f = U << (64 - c.frac_bits);
    l.fh = (unsigned)(f >> 32);
    l.fl = (unsigned)f;
    return l;
}

__device__ __forceinline__ void push_particle64(double &x, double &v, const PushArgs64 &a,
                                                const Push64 &c, double &ke, double &mom) {
    const Loc64 l = locate64(x, a.inv_dx, a.ng, c);
    const double g = __hiloint2double((int)(0x3FF00000u | (l.fh >> 12)),
                                      (int)__funnelshift_l(l.fl, l.fh, 20));
    const double2 p = c.pair[l.j];
    const double ep = l.ok ? fma(g, p.y, p.x) : 0.0;
    const double vn = fma(a.qmdt, ep, v);
    ke = fma(v, vn, ke);
    mom += vn;
    double xn = fma(vn, a.dt, x);
    // x < 0, x >= L and NaN all have bits of at least those of L (the vote
    // keeps it a branch: as predicated instructions the three comparisons and
    // two adds took the float64 pipe for every particle)
    const bool out = (u64)__double_as_longlong(xn) >= c.lbits;
    if (__any_sync(__activemask(), out) && out) {
        if (xn < 0.0) xn += a.length;
        else if (xn >= a.length) xn -= a.length;
        if (xn >= a.length) xn = 0.0;
    }
    x = xn;
    v = vn;
}

}  // namespace pic
