// Correctly rounded binary64 division in 32-bit integer arithmetic.
//
// GB300 executes every binary64 instruction of a warp in 64 cycles of its
// scheduler's one FP64 pipe, whatever the number of active lanes, and a
// division takes 565 cycles (1 096 for two warps of one scheduler).  The panel kernels divide once per row and column on their critical
// path.  The schoolbook division below needs about 70 integer instructions
// and no FP64 pipe.
//
// With b = mb 2^x, 2^52 <= mb < 2^53, rec is a 32-bit lower bound of
// 2^84 / mb: a 23-bit reciprocal from the FP32 unit, one Newton step in
// integers (error below 2^-42 relative, then rounding to 32 bits), and 8
// units taken off, so that rec <= 2^84 / mb <= rec + 16.  The quotient of
// a = ma 2^y, scaled so that mb <= ma < 2 mb, comes digit by digit, each
// digit a lower bound and each remainder exact modulo 2^64:
//   q1 = floor(rec * floor(ma 2^10 / 2^32) / 2^32)   ma/mb 2^30, short by < 21
//   r1 = ma 2^30 - q1 mb                              0 <= r1 < 21 mb < 2^58
//   q2 = floor(rec * floor(r1 / 2^26) / 2^32)         r1/mb 2^26, short by < 16
//   r2 = r1 2^26 - q2 mb                              0 <= r2 < 16 mb < 2^58
//   q3 = floor(rec * floor(r2 / 2^26) / 2^58)         floor(r2/mb), or one less
//   r3 = r2 - q3 mb, then one conditional subtraction: 0 <= r3 < mb
// so q = q1 2^26 + q2 + q3 (+ 1) = floor(ma/mb 2^56) with its remainder: 53
// bits, 4 more and a sticky bit decide round-to-nearest-even.  A zero
// dividend gives a zero of the quotient's sign; other operands that are zero,
// subnormal, infinite or NaN, and quotients outside the normal range, take
// the hardware division (the whole warp waits for it).
#pragma once
#include <cuda_runtime.h>

namespace lu {

#ifdef __CUDACC__                                  // (a host build brings its own)
__device__ __forceinline__ float approx_rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float approx_rsqrt(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// volatile: not computed ahead of the branch that needs them
__device__ __forceinline__ double hardware_div(double a, double b) {
    double r;
    asm volatile("div.rn.f64 %0, %1, %2;" : "=d"(r) : "d"(a), "d"(b));
    return r;
}
__device__ __forceinline__ double hardware_sqrt(double x) {
    double r;
    asm volatile("sqrt.rn.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}
#endif

// An approximation of a value in [1/2, 1] as an integer in units of 2^-32.
// (Approximations may come out below 1/2 or above 1.)
__device__ __forceinline__ unsigned approx_bits(float y) {
    const unsigned b = __float_as_uint(y);
    return b >= 0x3f800000u ? 0xffffffffu : b < 0x3f000000u ? 0x80000000u : (0x80000000u | (b << 8));
}

// rec for the divisor b; 0 where b takes the hardware division.
__device__ __forceinline__ unsigned div_rec(double b) {
    const unsigned hi = static_cast<unsigned>(__double2hiint(b)), lo = static_cast<unsigned>(__double2loint(b));
    const unsigned e = (hi >> 20) & 0x7ffu;
    const unsigned bt = 0x80000000u | (hi << 11) | (lo >> 21);          // mb / 2^21, rounded down
    const unsigned rec0 = approx_bits(approx_rcp(__uint_as_float(0x3f800000u | ((bt >> 8) & 0x7fffffu))));
    const long long t = static_cast<long long>(0x8000000000000000ull - static_cast<unsigned long long>(bt) * rec0);
    const int corr = __mulhi(static_cast<int>(t >> 10), static_cast<int>(rec0 >> 1)) >> 20;
    // (rec0 + corr may pass 2^32 when mb is near 2^52)
    const long long s = static_cast<long long>(rec0) + corr - 8;
    const unsigned rec = s > 0xffffffffll ? 0xffffffffu : static_cast<unsigned>(s);
    return (e - 1u < 2046u) ? rec : 0u;
}

// a / b, rounded to nearest even; rec = div_rec(b).
__device__ __forceinline__ double div_by(double a, double b, unsigned rec) {
    const unsigned ahi = static_cast<unsigned>(__double2hiint(a)), alo = static_cast<unsigned>(__double2loint(a));
    const unsigned bhi = static_cast<unsigned>(__double2hiint(b)), blo = static_cast<unsigned>(__double2loint(b));
    const int ea = static_cast<int>((ahi >> 20) & 0x7ffu), eb = static_cast<int>((bhi >> 20) & 0x7ffu);
    unsigned long long ma = (static_cast<unsigned long long>((ahi & 0xfffffu) | 0x100000u) << 32) | alo;
    const unsigned mbh = (bhi & 0xfffffu) | 0x100000u;
    const unsigned long long mb = (static_cast<unsigned long long>(mbh) << 32) | blo;
    const bool less = ma < mb;
    const int e = ea - eb + 1023 - (less ? 1 : 0);
    ma <<= (less ? 1 : 0);
    const unsigned q1 = __umulhi(static_cast<unsigned>(ma >> 22), rec);
    const unsigned long long r1 = (ma << 30) - static_cast<unsigned long long>(q1) * mb;
    const unsigned q2 = __umulhi(static_cast<unsigned>(r1 >> 26), rec);
    const unsigned long long r2 = (r1 << 26) - static_cast<unsigned long long>(q2) * mb;
    const unsigned q3 = __umulhi(static_cast<unsigned>(r2 >> 26), rec) >> 26;
    unsigned long long r3 = r2 - static_cast<unsigned long long>(q3) * mb;
    unsigned long long q = (static_cast<unsigned long long>(q1) << 26) + q2 + q3;
    const unsigned long long one = r3 >= mb ? 1ull : 0ull;
    r3 -= mb & (0ull - one);
    q += one;
    // 2^56 <= q < 2^57: keep 53 bits; the half is bit 3, the rest sticky
    const unsigned low = (static_cast<unsigned>(q) & 31u) | (r3 != 0 ? 1u : 0u);   // bit 4: the kept last bit
    // round up when the half bit is set and (the last bit or anything below the
    // half) is: adding 7 or 8 to the five low bits carries out of bit 3 then
    const unsigned up = ((low & 15u) + 7u + (low >> 4)) >> 4;
    const unsigned long long m = (q >> 4) + up;                    // 2^52 <= m <= 2^53 (the carry moves the exponent)
    const unsigned long long sign = static_cast<unsigned long long>((ahi ^ bhi) & 0x80000000u) << 32;
    const unsigned long long bits =
        sign + (static_cast<unsigned long long>(static_cast<unsigned>(e - 1)) << 52) + m;
    const bool zero = ((ahi << 1) | alo) == 0u;
    double r = __longlong_as_double(static_cast<long long>(zero ? sign : bits));
    // (with e >= 2046 a rounding carry could reach the infinity's exponent)
    if (rec == 0u || (!zero && (static_cast<unsigned>(ea - 1) >= 2046u || static_cast<unsigned>(e - 1) >= 2045u)))
        r = hardware_div(a, b);
    return r;
}

// sqrt(d), rounded to nearest even, the same way (the hardware's is 599
// cycles of the FP64 pipe): d = M 2^x with x even, 2^52 <= M < 2^54, so the
// root is S 2^(x/2 - 26) with S = floor(sqrt(M 2^52)) a 53-bit integer.  Y1, a
// lower bound of 2^32 / sqrt(M / 2^52) by at most 16 (FP32 reciprocal root,
// one Newton step in integers), gives 31 bits of S (s1, short by at most 18),
// then 22 more from the exact remainder M 2^8 - s1^2; S is then off by -3 to
// +1 and the exact remainder M 2^52 - S^2 (modulo 2^64) puts it right.  It
// rounds up when that remainder passes S; a tie cannot occur.  Anything but a
// positive normal number takes the hardware's.
__device__ __forceinline__ double sqrt_int(double d) {
    const unsigned hi = static_cast<unsigned>(__double2hiint(d)), lo = static_cast<unsigned>(__double2loint(d));
    const unsigned ex = hi >> 20, even = (ex & 1u) ^ 1u;
    const unsigned long long M =
        ((static_cast<unsigned long long>((hi & 0xfffffu) | 0x100000u) << 32) | lo) << even;
    const unsigned Mt = static_cast<unsigned>(M >> 22);
    const unsigned Y0 = approx_bits(
        approx_rsqrt(__uint_as_float(((127u + even) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29))));
    const long long err = static_cast<long long>(0x4000000000000000ull -
                                                 static_cast<unsigned long long>(Mt) * __umulhi(Y0, Y0));
    const int corr = __mulhi(static_cast<int>(err >> 11), static_cast<int>(Y0 >> 1)) >> 19;
    const long long Ys = static_cast<long long>(Y0) + corr - 8;
    const unsigned Y1 = Ys > 0xffffffffll ? 0xffffffffu : static_cast<unsigned>(Ys);
    const unsigned s1 = __umulhi(Mt, Y1);
    const unsigned long long R1 = (M << 8) - static_cast<unsigned long long>(s1) * s1;
    const unsigned s2 = __umulhi(static_cast<unsigned>(R1 >> 5), Y1) >> 4;
    long long S = static_cast<long long>((static_cast<unsigned long long>(s1) << 22) + s2);
    long long rem = static_cast<long long>((M << 52) - static_cast<unsigned long long>(S) * S);
    const long long c = __mulhi(static_cast<int>(rem >> 26), static_cast<int>(Y1 >> 1)) >> 26;
    rem -= c * (2 * S + c);
    S += c;
    const long long dn = rem < 0 ? 1 : 0;
    S -= dn;
    rem += dn * (2 * S + 1);
    const long long up = rem > 2 * S ? 1 : 0;
    rem -= up * (2 * S + 1);
    S += up;
    S += rem > S ? 1 : 0;
    double r = __longlong_as_double(
        static_cast<long long>(static_cast<unsigned long long>((ex - even + 1023u) / 2u - 1u) << 52) + S);
    if (ex - 1u >= 2046u) r = hardware_sqrt(d);
    return r;
}

}  // namespace lu
