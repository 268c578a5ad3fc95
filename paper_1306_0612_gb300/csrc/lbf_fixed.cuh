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
// words that no launch wrote) and every launch writes all words of the boxes it hands on, zeros
// past its own order (launches of several orders share the words and the count of launches), so
// an old word never carries the tag waited for.
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

// Dot products on the integer pipes.  A 32 x 32 -> 64 bit multiply-add leaves a scheduler every
// 4 cycles, a double one every 64; an integer x of 54 bits (|x| <= 2^53) goes as two words,
// x = hi 2^27 + lo, |hi| <= 2^26, |lo| <= 2^26, and a product as the three of them that reach the
// leading 54 of its 106 bits (measured 2.16e12 such products a second, 0.49e12 double).
__device__ __forceinline__ int2 split27(long long x)
{
    const int lo = (int)((unsigned)x << 5) >> 5;
    return make_int2(lo, (int)((x - lo) >> 27));
}
struct Dot {  // sum = h 2^54 + m 2^27, of 768 products at most
    long long h, m;
};
__device__ __forceinline__ void dot_add(Dot &d, int2 e, int2 x)
{
    d.h += (long long)e.y * x.y;
    d.m += (long long)e.y * x.x;
    d.m += (long long)e.x * x.y;
}
// asks for the tiles at p (a multiple of 256 bytes) to be brought to L2, by one lane
__device__ __forceinline__ void prefetch_tiles(const double *p, int tiles, int lane)
{
    if (lane == 0 && tiles > 0)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(tiles * 256) : "memory");
}
__device__ __forceinline__ int2 shfl_word(int2 v, int src)
{
    return make_int2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ long long shfl_xor_ll(long long v, int mask)
{
    return (long long)__shfl_xor_sync(0xffffffffu, (unsigned long long)v, mask);
}
// a lane keeps one of two sums (the second: `second`) and adds its partner's part of it
__device__ __forceinline__ Dot dot_meet(const Dot &x, const Dot &y, bool second, int bit)
{
    const Dot keep = second ? y : x, send = second ? x : y;
    return Dot{keep.h + shfl_xor_ll(send.h, bit), keep.m + shfl_xor_ll(send.m, bit)};
}
// d 2^E as a double
__device__ __forceinline__ double dot_double(Dot d, int E)
{
    const long long t = d.h + (d.m >> 27);
    const int f = (int)(d.m & 0x7ffffff);
    const int sh = min(27, __clzll(t < 0 ? ~t : t) - 2);  // room left of t's bits
    return pack_double((long long)((unsigned long long)t << sh) + (f >> (27 - sh)), E + 54 - sh);
}
// the words of v, its exponent field raised by `up`, in a sum whose largest raised field is top
__device__ __forceinline__ int2 dot_word(double v, int up, int top)
{
    return split27(fixed54(__double_as_longlong(v), -up, top + 1));
}
__device__ __forceinline__ int exp_field(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7ff); }

// f<NG>() for the number of row groups of a block, 1 to 8: the loops over tiles have a copy
// each, and nothing else does (with whole kernels copied the warps waited for instructions)
#define LBF_GROUPS(ng, CALL)    \
    switch (ng) {               \
    case 1: CALL(1); break;     \
    case 2: CALL(2); break;     \
    case 3: CALL(3); break;     \
    case 4: CALL(4); break;     \
    case 5: CALL(5); break;     \
    case 6: CALL(6); break;     \
    case 7: CALL(7); break;     \
    default: CALL(8); break;    \
    }

}  // namespace
