// FP64 quotients by a divisor that many values are divided by (the pivot of a factorization).
#pragma once

namespace hec {

// a / b for a pivot b whose reciprocal y = RN(1 / b) is kept with its row: Markstein's corrected quotient
// (P. Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", 1990; IA-64
// and Elementary Functions, 2000).  q1 = q0 + y (a - b q0) is within one ulp of a / b, and with y correctly
// rounded q1 + y (a - b q1) rounds to RN(a / b), as long as no step leaves the normal range: the
// exponents are checked, and anything else takes the division.  Five FP64 instructions.
__device__ __forceinline__ double div_by(double a, double b, double y) {
    const int ea = (int)(((unsigned long long)__double_as_longlong(a) >> 52) & 0x7ff);
    const int eb = (int)(((unsigned long long)__double_as_longlong(b) >> 52) & 0x7ff);
    const int eq = ea - eb + 1023;
    // a, b, 1 / b and the quotient well inside the normal range, and the residuals (about a / 2^53) too
    if (ea < 120 || ea > 1900 || eb < 120 || eb > 1900 || eq < 120 || eq > 1900) return __ddiv_rn(a, b);
    const double q0 = __dmul_rn(a, y);
    const double q1 = __fma_rn(__fma_rn(-b, q0, a), y, q0);
    return __fma_rn(__fma_rn(-b, q1, a), y, q1);
}

}  // namespace hec
