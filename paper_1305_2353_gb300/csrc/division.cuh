// division.cuh -- the pivot search's division by a divisor whose rounded reciprocal is
// known; compiles for the device and, for its test, for the host.
#pragma once

#ifdef __CUDACC__
#define CTP_DIV_FN __device__ __forceinline__
#define CTP_DIV_MUL __dmul_rn
#define CTP_DIV_FMA __fma_rn
#define CTP_DIV_DIV __ddiv_rn
#else  // plain operators, not to be contracted
#include <math.h>
#include <string.h>
#define CTP_DIV_FN static inline
#define CTP_DIV_MUL(a, b) ((a) * (b))
#define CTP_DIV_FMA(a, b, c) fma(a, b, c)
#define CTP_DIV_DIV(a, b) ((a) / (b))
#endif

// x / d correctly rounded, given y = RN(1/d): two steps of Markstein's division
// ("Computation of elementary functions on the IBM RISC System/6000 processor",
// IBM J. Res. Dev. 34, 1990: with y the correctly rounded reciprocal, q within
// one unit of x/d and the residual r = x - q d exact, RN(q + r y) is x/d
// correctly rounded); the first step brings q within a unit.  Where exponents leave
// no room, the division.  (With the rows of earlier pivots skipped as well, the search
// at p = 256, all pivots accepted, went from 1789 to 1653 us.)
CTP_DIV_FN double div_by(double x, double d, double y) {
#ifdef __CUDACC__
    const unsigned long long bx = (unsigned long long)__double_as_longlong(x), bd = (unsigned long long)__double_as_longlong(d);
#else
    unsigned long long bx, bd;
    memcpy(&bx, &x, 8);
    memcpy(&bd, &d, 8);
#endif
    const unsigned ex = (unsigned)(bx >> 52) & 0x7FFu, ed = (unsigned)(bd >> 52) & 0x7FFu;
    const bool zero = bx << 1 == 0ull;
    if ((ex - 400u > 1246u && !zero) || ed - 723u > 600u) return CTP_DIV_DIV(x, d);
    const double q0 = CTP_DIV_MUL(x, y);
    const double q1 = CTP_DIV_FMA(CTP_DIV_FMA(-q0, d, x), y, q0);
    const double q2 = CTP_DIV_FMA(CTP_DIV_FMA(-q1, d, x), y, q1);
    return zero ? q0 : q2;
}
