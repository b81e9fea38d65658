// Row q of block row i of A times x, FP64: the SpMV's inner product, shared by
// the product kernel and the residual kernels so that every FP64 product of A
// runs the same operations.  The first four blocks' loads are issued before
// any arithmetic, so each thread keeps up to 8 independent 16-byte loads in
// flight.  Blocks in order, within a block x_j[0..3]; the third and fourth
// blocks' eight products are summed with integer instructions (fx_dot8).
#pragma once
#include "common.cuh"

namespace abilu {

// sum_k a[k] x[k], k < 8, in integer arithmetic, rounded once to FP64.
//
// Why: this GPU executes two FP64 FMA per SM and clock, so a row's 16 FMAs
// take longer (53 us per product of 2.1 M blocks at 100% of that pipe) than its
// 528 bytes take to arrive (47 us), while the integer lanes idle: 64 issue
// slots pass per warp-wide FP64 FMA, and an integer product-and-add below is
// about 25 instructions.  With half of a row's products here that pipe is 52%
// busy and the integer pipe 43% (all FMA: 86% and little), and a row's chain of
// dependent FMAs is half as long.  512x512 (us): product 65.7 -> 60.8, fused
// product and dots of one to five vectors 76-95 -> 73-91, residual 78 -> 71;
// 2.6 M rows, batch: fused 358 -> 330.  One block of four in integers gained
// nothing (75 us: its chain is as long, its share of the pipe small).
//
// Precision: each product of two 53-bit significands, aligned to the largest
// product's exponent, is kept to 2^-58 of the largest product (off by at most
// three such units) and added exactly in 64 bits; the sum is rounded once.
// Eight FP64 FMAs round eight times, to 2^-53 of the running sum.  On random
// products its error was half of theirs (rms 6.5e-17 against 1.4e-16 of the
// largest product, largest 5.8e-16 against 1.4e-15), and a whole product of the
// 512x512 grid is 1.1e-16 from the exact one where FMAs gave 1.5e-16.  Sums of
// integers below 2^26 stay exact.
//
// Range: taken when every operand is below 2^478 in magnitude and the largest
// product is at least 2^-446: then a zero's or subnormal's product (exponent
// field 0, read as if normal) is shifted out entirely, which is its value to
// far below the rounding.  Otherwise (also Inf and NaN) FP64 FMAs.
__device__ __forceinline__ double fx_dot8(const double (&a)[8], const double (&x)[8]) {
    constexpr unsigned EXP = 0x7FF00000u;   // the exponent field of an operand's high word
    unsigned e[8], top = 0u, emax = 0u;     // e: the two exponents' sum, in place
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const unsigned ea = (unsigned)__double2hiint(a[k]) & EXP, ex = (unsigned)__double2hiint(x[k]) & EXP;
        e[k] = ea + ex;
        top = max(top, max(ea, ex));
        emax = max(emax, e[k]);
    }
    if (top > (1500u << 20) || emax < (1600u << 20)) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < 8; k++) s = fma(a[k], x[k], s);
        return s;
    }
    long long acc = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const int ah = __double2hiint(a[k]), xh = __double2hiint(x[k]);
        const unsigned al = (unsigned)__double2loint(a[k]), xl = (unsigned)__double2loint(x[k]);
        // significands shifted up by 9 (62 bits)
        const unsigned ahi = __funnelshift_l(al, (unsigned)(ah & 0xFFFFF) | 0x100000u, 9), alo = al << 9;
        const unsigned xhi = __funnelshift_l(xl, (unsigned)(xh & 0xFFFFF) | 0x100000u, 9), xlo = xl << 9;
        const unsigned long long m = (unsigned long long)alo * xhi + (unsigned long long)ahi * xlo;
        unsigned long long r = (unsigned long long)ahi * xhi + (m >> 32);   // 2^58 .. 2^60
        r >>= min((emax - e[k]) >> 20, 63u);
        const int sg = (ah ^ xh) >> 31;   // 0 or -1
        acc += ((long long)r ^ (long long)sg) + (long long)(sg & 1);
    }
    // |acc| < 2^63, to FP64
    if (acc == 0) return 0.0;
    const unsigned sgn = (unsigned)((unsigned long long)acc >> 32) & 0x80000000u;
    unsigned long long u = (unsigned long long)(acc < 0 ? -acc : acc);
    const int z = __clzll((long long)u);
    u <<= z;                                   // bit 63 set
    unsigned long long f = (u >> 11) + ((u >> 10) & 1ull);   // 53 bits, rounded (may carry to 2^53)
    // the significands carry 2^1075 each and r 2^-46: value = u 2^(emax - 2104 - z)
    const int ef = (int)(emax >> 20) - 1018 - z;            // exponent field of bit 63
    f += ((unsigned long long)(unsigned)(ef - 1)) << 52;     // adds the hidden bit's one
    return __hiloint2double((int)((unsigned)(f >> 32) | sgn), (int)(unsigned)f);
}

__device__ __forceinline__ double row_dot_blocks(const PatternView &P, const double *__restrict__ A,
                                                 const double *__restrict__ x, int i, int q) {
    const int p0 = P.rowptr[i], p1 = P.rowptr[i + 1];
    double2 a0[4], a1[4];
    int jj[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int p = p0 + k;
        if (p < p1) {
            jj[k] = __ldg(P.colind + p);
            const double2 *ap = reinterpret_cast<const double2 *>(A + (size_t)p * BB + q * BS);
            a0[k] = __ldg(ap);
            a1[k] = __ldg(ap + 1);
        } else {
            jj[k] = -1;
        }
    }
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        if (jj[k] >= 0) {
            const double2 *xp = reinterpret_cast<const double2 *>(x + (size_t)jj[k] * BS);
            double2 x0 = __ldg(xp), x1 = __ldg(xp + 1);
            s = fma(a0[k].x, x0.x, s);
            s = fma(a0[k].y, x0.y, s);
            s = fma(a1[k].x, x1.x, s);
            s = fma(a1[k].y, x1.y, s);
        }
    }
    if (jj[2] >= 0) {
        double av[8], xv[8];
#pragma unroll
        for (int k = 2; k < 4; k++) {
            double2 x0 = make_double2(0.0, 0.0), x1 = x0;
            if (jj[k] >= 0) {
                const double2 *xp = reinterpret_cast<const double2 *>(x + (size_t)jj[k] * BS);
                x0 = __ldg(xp);
                x1 = __ldg(xp + 1);
            } else {
                a0[k] = a1[k] = x0;
            }
            double *ak = av + 4 * (k - 2), *xk = xv + 4 * (k - 2);
            ak[0] = a0[k].x; ak[1] = a0[k].y; ak[2] = a1[k].x; ak[3] = a1[k].y;
            xk[0] = x0.x; xk[1] = x0.y; xk[2] = x1.x; xk[3] = x1.y;
        }
        s += fx_dot8(av, xv);
    }
    for (int p = p0 + 4; p < p1; p++) {  // rows longer than four blocks
        const int j = __ldg(P.colind + p);
        const double2 *ap = reinterpret_cast<const double2 *>(A + (size_t)p * BB + q * BS);
        const double2 *xp = reinterpret_cast<const double2 *>(x + (size_t)j * BS);
        double2 b0 = __ldg(ap), b1 = __ldg(ap + 1), x0 = __ldg(xp), x1 = __ldg(xp + 1);
        s = fma(b0.x, x0.x, s);
        s = fma(b0.y, x0.y, s);
        s = fma(b1.x, x1.x, s);
        s = fma(b1.y, x1.y, s);
    }
    return s;
}

}  // namespace abilu
