// Expansions as integers: the reals of an expansion in units of 2^(e - 54), e an exponent of
// the box, each real scaled by a power of two of its own (its order over two) so that they
// are of like size.  Used by the tensor-core M2L (lbf_m2l.cu) and the integer shifts
// (lbf_passes.cu).
#pragma once

namespace {

constexpr int kBadExp = 1 << 20;   // exponent of a box with an infinity or NaN
constexpr int kZeroExp = -5118;    // exponent of a box of zeros

__host__ __device__ inline int real_pitch(int P) { return (2 * P + 7) / 8 * 8; }

// Words of an expansion as its readers find them: the integer in 56 bits (the exponent in 24)
// under a tag of 8 bits, the application's number.  A reader of the same launch waits on the
// words themselves until they carry the tag, so a box is handed on with one store and one
// load where a flag costs a fence and two trips to L2 more.  The tags go round 1 .. 255 (0:
// words that no launch of that kind wrote) and every launch rewrites all words, so an old word
// never carries the tag waited for.
__device__ __forceinline__ long long tag_word(long long x, unsigned tag)
{
    return (long long)(((unsigned long long)x & 0xffffffffffffffull) | ((unsigned long long)tag << 56));
}
__device__ __forceinline__ long long untag(long long w) { return (long long)((unsigned long long)w << 8) >> 8; }
__device__ __forceinline__ bool has_tag(long long w, unsigned tag) { return (unsigned)((unsigned long long)w >> 56) == tag; }
__device__ __forceinline__ int tag_exp(int e, unsigned tag) { return (int)(((unsigned)e & 0xffffffu) | (tag << 24)); }
__device__ __forceinline__ int untag_exp(int w) { return (int)((unsigned)w << 8) >> 8; }
__device__ __forceinline__ bool exp_has_tag(int w, unsigned tag) { return (unsigned)w >> 24 == tag; }

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
