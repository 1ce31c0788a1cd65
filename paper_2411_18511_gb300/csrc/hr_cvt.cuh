// hr_cvt.cuh -- binary64 <-> pair of floats and float -> binary64 in integer
// arithmetic (plain C++ as well as CUDA, HR_HD, so that the host can check it).
//
// GB300's FP64 pipe converts and adds 1.7 to 2 numbers a clock and SM, so packing
// and unpacking a field, which only move its numbers between canonical doubles
// and the packed layouts, ran at a third of the memory rate on six (split) and
// three (join) such operations a real.  About 20 integer operations give the
// same bits.  Each function returns false outside its range (stated there), and
// the caller then converts with the FP64 pipe.
#pragma once

#include "hr_fix.cuh"

namespace hr {

// h = RN(x), l = RN(x - h) for 2^-63 <= |x| < 2^120, and for zero
HR_HD inline bool cvt_split(double x, float &h, float &l)
{
    const unsigned long long u = fx_dbits(x);
    const unsigned hi = (unsigned)(u >> 32), lo = (unsigned)u;
    const int e = (int)(hi >> 20) & 0x7ff, sg = (int)hi >> 31;
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    const unsigned m24 = (unsigned)((m + 0x0fffffffu + ((lo >> 29) & 1u)) >> 29); // ties to even; 2^24 carries
    const int d = (int)(lo - (m24 << 29));                                       // m - m24 2^29, |d| <= 2^28
    h = fx_float((hi & 0x80000000u) | (((unsigned)(e - 897) << 23) + m24));
    l = fx_mul((float)((d ^ sg) - sg), fx_float((unsigned)(e - 948) << 23));
    if (((hi << 1) | lo) == 0u) {
        h = fx_float(hi);
        l = 0.f;
        return true;
    }
    return e >= 960 && e <= 1142;
}

// RN(h + l) for h normal and l zero or normal, between 2^-39 and 2^-24 of h in exponent,
// unless h is a power of two and l of the other sign; and for two zeros
HR_HD inline bool cvt_join(float h, float l, double &x)
{
    const unsigned uh = fx_bits(h), ul = fx_bits(l);
    const int eh = (int)(uh >> 23) & 0xff, el = (int)(ul >> 23) & 0xff, d = eh - el;
    const bool l0 = (ul << 1) == 0u;
    const unsigned ml = l0 ? 0u : (ul & 0x7fffffu) | 0x800000u;
    const unsigned long long b = ((unsigned long long)(ml << 7) << 32) >> (d & 63);
    const unsigned long long n = (unsigned long long)(long long)((int)(uh ^ ul) >> 31);
    // h at bits 39 .. 62, l added or subtracted below
    const unsigned long long s = ((unsigned long long)(((uh & 0x7fffffu) | 0x800000u) << 7) << 32) + ((b ^ n) - n);
    const unsigned long long r = (s + 0x1ffu + ((s >> 10) & 1u)) >> 10; // ties to even; 2^53 carries
    x = fx_double((((unsigned long long)(unsigned)(eh + 895) << 52) + r) |
                  ((unsigned long long)(uh & 0x80000000u) << 32));
    if (((uh | ul) << 1) == 0u) {
        x = fx_double((unsigned long long)(uh & ul) << 32);
        return true;
    }
    return eh >= 1 && eh <= 254 && (l0 || (el >= 1 && d >= 24 && d <= 39)) && (unsigned)(s >> 62) == 1u;
}

// f as a double, for f normal or zero
HR_HD inline bool cvt_widen(float f, double &x)
{
    const unsigned u = fx_bits(f), e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
    const bool zero = (u << 1) == 0u;
    const unsigned hi = (u & 0x80000000u) | (zero ? 0u : ((e + 896u) << 20) | (m >> 3));
    x = fx_double(((unsigned long long)hi << 32) | (m << 29));
    return zero || (e >= 1 && e <= 254);
}

} // namespace hr
