// Expansions as integers: the reals of an expansion in units of 2^(e - 54), e an exponent of
// the box, each real scaled by a power of two of its own (its order over two) so that they
// are of like size.  Used by the tensor-core M2L (lbf_m2l.cu) and the integer shifts
// (lbf_passes.cu).
#pragma once

namespace {

constexpr int kBadExp = 1 << 20;   // exponent of a box with an infinity or NaN
constexpr int kZeroExp = -5118;    // exponent of a box of zeros

__host__ __device__ inline int real_pitch(int P) { return (2 * P + 7) / 8 * 8; }

// v as an integer in units of 2^(e - 54), rounded, |v| < 2^e: its double bits with the
// exponent lowered by `drop`; top: the largest lowered exponent field of the set (> 0)
__device__ __forceinline__ long long fixed54(long long bits, int drop, int top)
{
    const int E = (int)((bits >> 52) & 0x7ff);
    if (E == 0) return 0;  // zero (a subnormal is far below any unit here)
    const int d = top - (E - drop);
    if (d > 60) return 0;
    unsigned long long m = ((unsigned long long)bits & 0xfffffffffffffull) | 0x10000000000000ull;
    m <<= 1;
    if (d > 0) m = (m + (1ull << (d - 1))) >> d;
    return bits < 0 ? -(long long)m : (long long)m;
}

// w 2^E (|w| < 2^63) as a double, rounded half up, without the double pipe
__device__ __forceinline__ double pack_double(long long w, int E)
{
    unsigned long long m = w < 0 ? (unsigned long long)-w : (unsigned long long)w;
    if (m == 0) return 0.0;
    const int lz = __clzll((long long)m);
    m <<= lz;
    const int ef = 1023 + 63 - lz + E;
    const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);  // hidden bit at 52, may carry
    unsigned long long bits;
    if (ef <= 0) bits = 0;
    else if (ef >= 2047) bits = 0x7ff0000000000000ull;
    else bits = ((unsigned long long)(ef - 1) << 52) + r;
    return __longlong_as_double((long long)(bits | (w < 0 ? 0x8000000000000000ull : 0ull)));
}

}  // namespace
