// Natural logarithm in double for the kernels that take many of them.
#pragma once

namespace {

// log a for positive normal a, table-driven (P. T. P. Tang, ACM TOMS 16, 1990): with
// a = 2^e m, c the tabulated 1/m to 7 bits, r = c m - 1, |r| <= 2^-8,
//   log a = e log 2 + log(1/c) + (r - r^2/2 + r^3/3 - ... + r^7/7),
// the remainder below 2^-66: 12 double instructions.  The table: c_j = 128/(128 + j) rounded
// to float (c m - 1 has one rounding, relative to r), formed by each thread block.
struct LogTab {
    double c[129], l[129];
};

__device__ __forceinline__ double log_tab(double a, const LogTab &t)
{
    const int hi = __double2hiint(a);
    int e = (hi >> 20) - 1023;
    const int j = ((hi & 0xfffff) + (1 << 12)) >> 13;  // m to the nearest 1/128, 0..128
    const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(a));
    const double r = fma(m, t.c[j], -1.0);
    // e as a double from the integer's bits (2^52 + 2^31 + e less 2^52 + 2^31)
    const double ed = __hiloint2double(0x43300000, e ^ 0x80000000) - 4503601774854144.0;
    double q = 1.0 / 7.0;
    q = fma(q, r, -1.0 / 6.0);
    q = fma(q, r, 1.0 / 5.0);
    q = fma(q, r, -1.0 / 4.0);
    q = fma(q, r, 1.0 / 3.0);
    q = fma(q, r, -0.5);
    const double r2 = r * r;
    return fma(ed, 0.69314718055994530942, t.l[j]) + fma(q, r2, r);
}

// the table, by the threads of a block (a barrier follows)
__device__ __forceinline__ void log_table(LogTab &t)
{
    for (int k = threadIdx.x; k < 129; k += blockDim.x) {
        const double c = (double)(float)(128.0 / (128.0 + k));
        t.c[k] = c;
        t.l[k] = -log(c);
    }
}

// log a for any a (zero, subnormal, infinite and NaN arguments by the library)
__device__ __forceinline__ double log_any(double a, const LogTab &t)
{
    return a > 0x1p-1000 && a < 0x1p1000 ? log_tab(a, t) : log(a);
}

}  // namespace
