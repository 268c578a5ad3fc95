// The upward and downward passes of a double application on a plan whose leaf rows
// (lbf_rows.cu) and translations (lbf_m2l.cu) are stored, P <= 32:
//
//   k_up        P2M from the rows' local columns (the powers u_i^l of the leaf's nodes are
//               there already) and M2M;
//   k_p2l_big   P2L of the few boxes whose X lists are not near columns;
//   k_l2l       each box's translations added up and its parent's expansion shifted to it,
//               in one launch; also the chain of the multiplier potential's expansions.
//
// P2M: with the stored powers a node and coefficient take two multiply-adds a real where
// the recurrence took six double instructions and left the lanes past a leaf's last node
// idle (26 of 32 at 16.8 million nodes).
//
// Shifts on the integer pipes.  A shift is a triangle of binomials between powers of
// 2d = +-1 +- i,
//   M2M  a_l  = d^l     sum_{k <= l} C(l, k) (2d)^-k a'_k,
//   L2L  b'_l = (2d)^-l sum_{k >= l} C(k, l) d^k b_k,
// and this GPU issues a double multiply-add every 64 cycles per scheduler, a 32 x 32 -> 64 bit
// integer one every few.  The expansions are integers of 54 bits below the box's largest
// (lbf_fixed.cuh, the form the translations take too), the powers of 1 + i are additions,
// swaps and shifts, C(l, k) and 2^(31-k) C(k, l) are below 2^31, and a sum of at most 32
// products of a 56-bit integer is exact in two 64-bit accumulators (28 low bits, the rest):
// one rounding a coefficient and level, 2^-54 of the box's largest.
//
// Both passes are one launch each whose warps wait on the expansions themselves: every word
// carries the launch's tag (lbf_fixed.cuh), so a level costs one trip through L2 and no fence.
// Measured, microseconds at 8192 nodes and at 16.8 million: up 50 and 3300 (double shifts
// and P2M 8000 at the latter; integer shifts with arrival counters 91 and 6100, P2M still
// double), a chain 27 and, at the latter, the density's 1710, the potential's 4330 (5400 in the mean;
// with flags 70 and 3600).  What is left is bound by the
// dependent loads of a box (a third fewer instructions for its sums changed nothing) and by
// the depth of the tree.
#include <algorithm>

#include "lbf_fixed.cuh"
#include "lbf_fmm_tpl.cuh"

using fmm::BoxGeo;
using fmm::cx;
using fmm::mk;

namespace {

constexpr int kP2lSmem = 4 * 32 * 33 * 16;
constexpr int kGroups = 8;  // row groups of a block at most (lbf_rows.cu)

// re[h], im[h] += the tiles of chunk h (of n, at most 4) times the rows' values
template <int NG>
__device__ __forceinline__ void p2m_chunks(const double *__restrict__ t, const int2 *cr, const int2 *ci,
                                           int n, Dot *re, Dot *im)
{
#pragma unroll
    for (int h = 0; h < 4; h++) {
        const double *th = t + 32 * NG * min(h, n - 1);  // (beyond n: a sum nobody takes)
#pragma unroll
        for (int g = 0; g < NG; g++) {
            const int2 e = *(const int2 *)&th[32 * g];
            dot_add(re[h], e, cr[g]);
            dot_add(im[h], e, ci[g]);
        }
    }
}

// P2M of leaf t by a warp: a_l = sum_i q_i u_i^l, the reals left in a[2 P].  Column 2 l of a row holds -(1/pi) Im u^l, column 2 l + 1 -(1/pi) Re u^l,
// both times 2^-(l/2): an even lane adds their parts of both reals of coefficient l, an odd lane
// likewise, and one exchange leaves the real part on the even lane, the imaginary part on the
// odd one.  The charges are integers in units of the leaf's largest (up bits more for a leaf
// of many nodes); sum: room for the 2 P sums of a leaf of several row blocks.
__device__ __forceinline__ void leaf_p2m(int64_t t, int P, int lchunks,
                                         const int32_t *__restrict__ block0,
                                         const RowItem *__restrict__ items,
                                         const double *__restrict__ rows,
                                         const double2 *__restrict__ q, double *a, Dot *sum, int lane)
{
    const int k0 = block0[t], k1 = block0[t + 1];
    const bool odd = (lane & 1) != 0, u = (lane & 16) != 0, w = (lane & 8) != 0;
    int top = 0, n = 0;
    bool bad = false;
    for (int k = k0; k < k1; k++) {
        const RowItem it = items[k];
        const int row0 = it.row0, nrow = it.nrow, ng = (nrow + 3) / 4;  // 32 rows at most
        prefetch_tiles(rows + ((int64_t)it.tile + (int64_t)it.nchunk * ng) * 32, lchunks * ng, lane);
        const double2 qq = lane < nrow ? q[row0 + lane] : make_double2(0.0, 0.0);
        const int E = max(exp_field(qq.x), exp_field(qq.y));
        bad |= E == 0x7ff;
        top = max(top, E);
        n += nrow;
    }
    top = __reduce_max_sync(0xffffffffu, top);
    bad = __any_sync(0xffffffffu, bad);
    const int up = n > 128 ? 25 - __clz(n) : 0;  // n 2^-up <= 128
    for (int k = k0; k < k1; k++) {
        const RowItem it = items[k];
        const int ng = (it.nrow + 3) / 4;
        // a charge a lane, then the rows of each lane's sums: (im, -re) of q for the columns of
        // Im u^l, (-re, -im) for those of Re u^l
        const double2 qq = lane < it.nrow ? q[it.row0 + lane] : make_double2(0.0, 0.0);
        const int2 qx = dot_word(-qq.x, 0, top + up), qy = dot_word(qq.y, 0, top + up);
        int2 cr[kGroups], ci[kGroups];
#pragma unroll
        for (int g = 0; g < kGroups; g++) {
            const int2 x = shfl_word(qx, 4 * g + (lane >> 3)), y = shfl_word(qy, 4 * g + (lane >> 3));
            cr[g] = odd ? x : y;
            ci[g] = odd ? make_int2(-y.x, -y.y) : x;
        }
        const double *tl = rows + ((int64_t)it.tile + (int64_t)it.nchunk * ng) * 32 + lane;
        for (int c = 0; c < lchunks; c += 4, tl += 128 * ng) {
            Dot re[4], im[4];
#pragma unroll
            for (int h = 0; h < 4; h++) re[h] = im[h] = Dot{0, 0};
#define LBF_DOT(NG) p2m_chunks<NG>(tl, cr, ci, lchunks - c, re, im)
            LBF_GROUPS(ng, LBF_DOT)
#undef LBF_DOT
            Dot s[4];
#pragma unroll
            for (int h = 0; h < 4; h++) s[h] = dot_meet(re[h], im[h], odd, 1);
            Dot v = dot_meet(dot_meet(s[0], s[2], u, 16), dot_meet(s[1], s[3], u, 16), w, 8);
            const int h = (u ? 2 : 0) + (w ? 1 : 0), m = 8 * (c + h) + (lane & 7);
            if (c + h < lchunks && m < 2 * P) {
                if (k > k0) {
                    v.h += sum[m].h;
                    v.m += sum[m].m;
                }
                if (k + 1 < k1) sum[m] = v;
                else a[m] = bad ? __longlong_as_double(0x7ff8000000000000ll)
                                : dot_double(v, top + up - 1129 + (m >> 2)) * LBF_PI;
            }
        }
    }
}

// boxes with X lists that are not near columns (plan time)
__global__ void k_bigx_list(int64_t nbox, int thr, const int32_t *__restrict__ bg,
                            const int32_t *__restrict__ en, const int32_t *__restrict__ nx,
                            int32_t *__restrict__ count, int32_t *__restrict__ list, int cap)
{
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b >= nbox || nx[b] == 0 || en[b] - bg[b] <= thr) return;
    const int k = atomicAdd(count, 1);
    if (k < cap) list[k] = (int32_t)b;
}

// their P2L: b_l = (1/r) (-1)^l sum_j q_j tau_j^(l+1), tau_j = r/(c - xi_j), a thread block of
// four warps per box, the X nodes' chunks of 32 dealt to the warps in turn
__global__ void __launch_bounds__(128)
k_p2l_big(int n, const int32_t *__restrict__ list, const int32_t *__restrict__ level,
          const int32_t *__restrict__ ix, const int32_t *__restrict__ iy,
          const int32_t *__restrict__ bg, const int32_t *__restrict__ en,
          const int32_t *__restrict__ xlist, const int32_t *__restrict__ nx, BoxGeo g, int P,
          const double2 *__restrict__ xi, const double2 *__restrict__ q, cx<double> *__restrict__ loc,
          const int *gate, int64_t slab)
{
    lbf_rhs(slab, q, loc, gate);
    if (fmm::gate_closed(gate)) return;
    extern __shared__ __align__(16) unsigned char p2l_sm[];  // per warp 32 x 33 terms
    __shared__ cx<double> part[4][32];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cx<double> *T = (cx<double> *)p2l_sm + wid * 32 * 33;
    const int b = list[blockIdx.x];
    double cxd, cyd, ir;
    box_centre_ir(g, level[b], ix[b], iy[b], cxd, cyd, ir);
    cx<double> s = mk<double>(0, 0);
    int turn = 0;
    for (int xq = 0; xq < nx[b]; xq++) {
        const int c = xlist[b * 16 + xq];
        for (int base = bg[c]; base < en[c]; base += 32, turn++) {
            if ((turn & 3) != wid) continue;
            const int j = base + lane;
            cx<double> tau = mk<double>(0, 0), term = mk<double>(0, 0);
            if (j < en[c]) {
                const double2 z = xi[j], qq = q[j];
                tau = fmm::crcp(mk<double>((cxd - z.x) * ir, (cyd - z.y) * ir));
                term = fmm::cmul(mk<double>(qq.x, qq.y), tau);
            }
            for (int l = 0; l < P; l++) {
                T[l * 33 + lane] = (l & 1) ? mk<double>(-term.x, -term.y) : term;
                term = fmm::cmul(term, tau);
            }
            __syncwarp();
            const int nin = min(32, en[c] - base);
            if (lane < P)
                for (int m = 0; m < nin; m++) {
                    s.x += T[lane * 33 + m].x;
                    s.y += T[lane * 33 + m].y;
                }
            __syncwarp();
        }
    }
    part[wid][lane] = s;
    __syncthreads();
    if (wid != 0 || lane >= P) return;
    for (int w = 1; w < 4; w++) {
        s.x += part[w][lane].x;
        s.y += part[w][lane].y;
    }
    loc[(int64_t)b * P + lane] = mk<double>(s.x * ir, s.y * ir);
}

// What a box's expansion takes beside its parent's: of the density block its translations and
// its P2L part where it has one (in loc already); of the multiplier potential (lbf_border.cu)
// the stored expansions of its centres times their strengths y.
struct Own {
    const int32_t *ptr;        // first translation, or first (box, centre) pair, of each box
    const cx<double> *part;    // P coefficients each
    const int32_t *src;        // the pairs' centres (null: translations, with weight 1 / r)
    const double *y;
    const int32_t *bg, *en, *nx;
    int thr;
    double *sums;              // pairs: [0] = sum y, [1] = sum of y lam over the finite centres
    const int32_t *kind;
    const double *lam;
    int M;
};

__device__ __forceinline__ cx<double> own_part(const Own &w, int64_t b, int P, int lane, double ir,
                                               const cx<double> *loc)
{
    cx<double> o = mk<double>(0, 0);
    if (lane >= P) return o;
    const int v1 = w.ptr[b + 1];
    if (w.src) {
#pragma unroll 4
        for (int v = w.ptr[b]; v < v1; v++) {
            const cx<double> a = w.part[(int64_t)v * P + lane];
            const double y = w.y[w.src[v]];
            o.x = fma(y, a.x, o.x);
            o.y = fma(y, a.y, o.y);
        }
        return o;
    }
#pragma unroll 4
    for (int v = w.ptr[b]; v < v1; v++) {
        const cx<double> a = w.part[(int64_t)v * P + lane];
        o.x += a.x;
        o.y += a.y;
    }
    o.x *= ir;
    o.y *= ir;
    if (w.nx[b] && w.en[b] - w.bg[b] > w.thr) {
        const cx<double> x = fmm::ldcg_cx(&loc[b * P + lane]);
        o.x += x.x;
        o.y += x.y;
    }
    return o;
}

// the sums of the strengths, by the warp that has box 0
__device__ __forceinline__ void strength_sums(const Own &w, int lane)
{
    double Y = 0.0, Lam = 0.0;
    for (int m = lane; m < w.M; m += 32) {
        Y += w.y[m];
        if (w.kind[m]) Lam = fma(w.y[m], w.lam[m], Lam);
    }
    Y = fmm::wsum(Y);
    Lam = fmm::wsum(Lam);
    if (lane == 0) {
        w.sums[0] = Y;
        w.sums[1] = Lam;
    }
}

// ---- shifts of integer expansions ------------------------------------------------------

// (x + iy) times (2d)^k up to the power of two 2^(k/2) (k even) or 2^((k-1)/2) (k odd), for
// n = k (2h + 1) mod 8, 2d = sqrt 2 e^(i (2h + 1) pi/4): i^(n/2), times 1 + i when n is odd
__device__ __forceinline__ void mul_pow(long long &x, long long &y, int n)
{
    if (n & 1) {
        const long long t = x - y;
        y = x + y;
        x = t;
    }
    if (n & 2) {
        const long long t = x;
        x = -y;
        y = t;
    }
    if (n & 4) {
        x = -x;
        y = -y;
    }
}

// 2h + 1 of the child at (ix, iy)
__device__ __forceinline__ int quadrant(int ix, int iy)
{
    return (iy & 1) ? ((ix & 1) ? 1 : 3) : ((ix & 1) ? 7 : 5);
}

// v 2^-s, rounded (s >= 0)
__device__ __forceinline__ long long shift_down(long long v, int s)
{
    return s == 0 ? v : s > 62 ? 0ll : (v + (1ll << (s - 1))) >> s;
}

// the two words of a 57-bit integer: 28 low bits and the rest
__device__ __forceinline__ int4 words(long long x, long long y)
{
    return make_int4((int)(x & 0xfffffff), (int)(x >> 28), (int)(y & 0xfffffff), (int)(y >> 28));
}

struct Sum {  // sums of weight times word, of the real and the imaginary part
    unsigned long long xl, yl;
    long long xh, yh;
};
__device__ __forceinline__ void add_term(Sum &s, unsigned c, int4 z)
{
    s.xl += (unsigned long long)c * (unsigned)z.x;
    s.xh += (long long)(int)c * z.y;
    s.yl += (unsigned long long)c * (unsigned)z.z;
    s.yh += (long long)(int)c * z.w;
}
// a row's sum: the other half-warp's part of it added
__device__ __forceinline__ Sum meet(const Sum &mine, const Sum &other)
{
    Sum r;
    r.xl = mine.xl + __shfl_xor_sync(0xffffffffu, other.xl, 16);
    r.xh = mine.xh + __shfl_xor_sync(0xffffffffu, other.xh, 16);
    r.yl = mine.yl + __shfl_xor_sync(0xffffffffu, other.yl, 16);
    r.yh = mine.yh + __shfl_xor_sync(0xffffffffu, other.yh, 16);
    return r;
}
// (hi 2^28 + lo) 2^-s, rounded, s in 1 .. 33
__device__ __forceinline__ long long scale_sum(long long hi, unsigned long long lo, int s)
{
    const long long t = hi + (long long)(lo >> 28);
    const unsigned f = (unsigned)lo & 0xfffffffu;
    if (s <= 28) return (t << (28 - s)) + ((f + (1u << (s - 1))) >> s);
    return (t + (1ll << (s - 29))) >> (s - 28);
}
__device__ __forceinline__ int bits_of(long long x, long long y)
{
    const unsigned long long m = (unsigned long long)(x < 0 ? -x : x) | (unsigned long long)(y < 0 ? -y : y);
    return 64 - __clzll((long long)m);
}
// x in the unit 2^sh times larger (sh < 0: smaller)
__device__ __forceinline__ long long rescale(long long x, int sh)
{
    return sh > 0 ? shift_down(x, sh) : x << -sh;
}

// words read and written by warps of one launch, each word on its own
__device__ __forceinline__ longlong2 ld_words(const long long *p)
{
    longlong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_word(const int32_t *p)
{
    int v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_words(long long *p, long long x, long long y)
{
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(x), "l"(y) : "memory");
}
__device__ __forceinline__ void st_word(int32_t *p, int v)
{
    asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// the words of lanes < n of an expansion and its exponent once they carry the tag (bounded)
__device__ __forceinline__ longlong2 wait_words(const long long *x, const int32_t *ex, int n, int lane,
                                                unsigned tag, unsigned lim, int *status, int &e)
{
    longlong2 v = make_longlong2(0, 0);
    for (unsigned spins = 0;; spins++) {
        bool ok = true;
        if (lane < n) {
            v = ld_words(x + 2 * lane);
            ok = has_tag(v.x, tag) && has_tag(v.y, tag);
        }
        const int w = ld_word(ex);
        e = untag_exp(w);
        if (__all_sync(0xffffffffu, ok && exp_has_tag(w, tag))) break;
        if (spins > lim) {
            if (lane == 0) atomicOr(status, LBF_DEV_TIMEOUT);
            break;
        }
    }
    v.x = untag(v.x);
    v.y = untag(v.y);
    return v;
}

constexpr unsigned kPassSpins = 1u << 22;

// P2M per leaf and M2M per box with children: warps take the leaves and then the boxes, the
// deepest first, from a counter, and a box waits (bounded) for the words of its children, which
// running warps took earlier.  Each box's multipole
// is written as doubles (evaluation, the rows' M2P columns) and as integers: X_k = a_k
// 2^-(k/2) in units of 2^(e - 54).  With conj(2d)^k taken exactly, 2 (2d)^-k a'_k is X_k
// rotated (times 2, k even, or 1 +- i, k odd), and the sum over k times 2^-(l+1), rotated by
// (2d)^l, is the parent's X_l.  Lane j of a half-warp has the rows j and P - 1 - j of the
// triangle, P + 1 terms, a half of them each half.
__global__ void __launch_bounds__(128, 4)
k_up(int64_t nleaf, int64_t nbox, const int32_t *__restrict__ leaves, const int32_t *__restrict__ ix,
     const int32_t *__restrict__ iy, const int32_t *__restrict__ child0,
     const int32_t *__restrict__ nchild, int P, int lchunks, const int32_t *__restrict__ block0,
     const RowItem *__restrict__ items, const double *__restrict__ rows,
     const double *__restrict__ binom, const double2 *__restrict__ q, cx<double> *mp, long long *X,
     int32_t *ex, unsigned *words_, int run, int *status, const int *gate, int64_t slab)
{
    lbf_rhs(slab, q, mp, X, ex, words_, gate);
    if (fmm::gate_closed(gate)) return;
    __shared__ unsigned Cl[32 * 32];
    __shared__ int4 Zs[4][32];
    __shared__ double vs[4][64];
    __shared__ Dot sums[4][64];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < P * P; e += blockDim.x) {
        const int k = e / P, l = e % P;
        Cl[k * 32 + l] = k <= l ? (unsigned)binom[l * LBF_MAX_TERMS + k] : 0u;  // C(l, k)
    }
    __syncthreads();
    const int pitch = real_pitch(P);
    const unsigned epoch = *(volatile unsigned *)&words_[2], tag = 1u + epoch % 255u;
    const unsigned lim = wait_limit(status, kPassSpins);
    const int hf = lane >> 4, j = lane & 15, nr = (P + 1) / 2;
    const int r1 = j < nr ? j : 0, r2 = P - 1 - r1, n1 = r1 + 1, mid = (P + 2) / 2;
    const int i0 = hf ? mid : 0, i1 = hf ? P + 1 : mid, row = hf ? r2 : r1;
    const bool on = j < nr && (hf == 0 || r2 != r1);
    for (;;) {
        unsigned ti = 0;
        if (lane == 0) ti = atomicAdd(&words_[0], (unsigned)run);
        const int64_t t0 = (int64_t)__shfl_sync(0xffffffffu, ti, 0);
        if (t0 >= nleaf + nbox) break;
        for (int64_t t = t0; t < min(t0 + run, nleaf + nbox); t++) {
            if (t < nleaf) {
                const int b = leaves[t];
                leaf_p2m(t, P, lchunks, block0, items, rows, q, vs[wid], sums[wid], lane);
                __syncwarp();
                double v[2];
                int top = -4096;
                bool bad = false;
#pragma unroll
                for (int h = 0; h < 2; h++) {  // lane: coefficient
                    const int m = 2 * lane + h;
                    v[h] = m < 2 * P ? vs[wid][m] : 0.0;
                    const int E = (int)((__double_as_longlong(v[h]) >> 52) & 0x7ff);
                    bad |= E == 0x7ff;
                    if (E) top = max(top, E - (lane >> 1));
                }
                top = __reduce_max_sync(0xffffffffu, top);
                bad = __any_sync(0xffffffffu, bad);
                if (2 * lane < pitch)
                    st_words(&X[(int64_t)b * pitch + 2 * lane],
                             tag_word(fixed54(__double_as_longlong(v[0]), lane >> 1, top), tag),
                             tag_word(fixed54(__double_as_longlong(v[1]), lane >> 1, top), tag));
                if (lane == 0) st_word(&ex[b], tag_exp(bad ? kBadExp : top - 1022, tag));
                if (lane < P) mp[(int64_t)b * P + lane] = mk<double>(v[0], v[1]);
                __syncwarp();
                continue;
            }
            const int64_t p = nbox - 1 - (t - nleaf);
            const int nc = nchild[p], c0 = child0[p];
            if (nc == 0) continue;
            long long sx = 0, sy = 0;
            int emax = -(1 << 22);
            for (int c = 0; c < nc; c++) {
                const int h2 = quadrant(ix[c0 + c], iy[c0 + c]);
                int ec;
                longlong2 v = wait_words(X + (int64_t)(c0 + c) * pitch, ex + c0 + c, P, lane, tag, lim, status, ec);
                mul_pow(v.x, v.y, (-lane * h2) & 7);
                Zs[wid][lane] = (lane & 1) ? words(v.x, v.y) : words(2 * v.x, 2 * v.y);
                __syncwarp();
                Sum acc{0, 0, 0, 0}, first{0, 0, 0, 0};
#pragma unroll 4
                for (int it = i0; it < i1; it++) {
                    if (it == n1) {
                        first = acc;
                        acc = Sum{0, 0, 0, 0};
                    }
                    const int k = it < n1 ? it : it - n1;
                    add_term(acc, Cl[k * 32 + (it < n1 ? r1 : r2)], Zs[wid][k]);
                }
                if (i1 <= n1) {
                    first = acc;
                    acc = Sum{0, 0, 0, 0};
                }
                const Sum s = meet(hf ? acc : first, hf ? first : acc);
                long long x = scale_sum(s.xh, s.xl, row + 1), y = scale_sum(s.yh, s.yl, row + 1);
                mul_pow(x, y, (row * h2) & 7);
                // to the larger unit of the children so far and this one
                const int em = max(emax, ec);
                sx = shift_down(sx, em - emax) + shift_down(x, em - ec);
                sy = shift_down(sy, em - emax) + shift_down(y, em - ec);
                emax = em;
                __syncwarp();
            }
            const bool bad = emax >= kBadExp;
            const int nb = __reduce_max_sync(0xffffffffu, on ? bits_of(sx, sy) : 0), sh = nb - 54;
            if (on)
                st_words(&X[p * pitch + 2 * row], tag_word(rescale(sx, sh), tag), tag_word(rescale(sy, sh), tag));
            if (lane == 0) st_word(&ex[p], tag_exp(bad ? kBadExp : nb == 0 ? kZeroExp : emax + sh, tag));
            for (int m = 2 * P + lane; m < pitch; m += 32) X[p * pitch + m] = tag_word(0, tag);
            if (on) {
                const double nan = __longlong_as_double(0x7ff8000000000000ll);
                const int E = emax - 54 + (row >> 1);
                mp[p * P + row] = bad ? mk<double>(nan, nan) : mk<double>(pack_double(sx, E), pack_double(sy, E));
            }
        }
    }
    // the last warp to finish readies the counters for the next application
    if (lane == 0) {
        const unsigned total = gridDim.x * 4u;
        if (atomicAdd(&words_[1], 1u) == total - 1u) {
            words_[0] = 0u;
            words_[1] = 0u;
            __threadfence();
            atomicExch(&words_[2], epoch + 1u);
        }
    }
}

// Every box's local expansion: its own part, and from level 3 on its parent's expansion
// shifted down.  A box with children is left as integers (LX, pitch reals a box), X_k = b_k
// 2^(k/2) in units of 2^(e - 54): then d^k b_k is X_k rotated (times 1 +- i, k odd) times 2^-k, the
// weights 2^(31-k) C(k, l) are integers below 2^31 (but for k = 0, added on its own), and the
// sum, rotated by conj(2d)^l (and halved, l odd), is the child's X_l.  A leaf is left as
// doubles in loc.  Warps take the boxes in index order from pull[3] and wait for their
// parent's words; pull[1] counts the finished warps, word the applications.
__global__ void __launch_bounds__(256, 3)
k_l2l(int64_t nbox, int P, const int32_t *__restrict__ level, const int32_t *__restrict__ ix,
      const int32_t *__restrict__ iy, const int32_t *__restrict__ parent,
      const int32_t *__restrict__ nchild, Own w, BoxGeo g, const double *__restrict__ binom,
      cx<double> *loc, long long *LX, int pitch, int32_t *ex, unsigned *pull, unsigned *word, int *status,
      const int *gate, int64_t slab)
{
    lbf_rhs(slab, loc, LX, ex, pull, word, gate, w.y, w.sums);
    if (!w.src) lbf_rhs(slab, w.part);
    if (fmm::gate_closed(gate)) return;
    __shared__ unsigned Wd[32 * 32];
    __shared__ int4 Zs[8][32];
    const int nw = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < P * P; e += blockDim.x) {
        const int k = e / P, l = e % P;
        Wd[k * 32 + l] = k >= l && k > 0 ? (unsigned)binom[k * LBF_MAX_TERMS + l] << (31 - k) : 0u;
    }
    __syncthreads();
    const unsigned epoch = *(volatile unsigned *)word, tag = 1u + epoch % 255u;
    const unsigned lim = wait_limit(status, kPassSpins);
    // lane j of a half has the rows r1 = j and r2 = P - 1 - j of the triangle, P + 1 terms
    // (n1 = P - r1 of them row r1's); half hf sums the terms i0 .. i1 - 1
    const int hf = lane >> 4, j = lane & 15, nr = (P + 1) / 2;
    const int r1 = j < nr ? j : 0, r2 = P - 1 - r1, n1 = P - r1, mid = (P + 2) / 2;
    const int i0 = hf ? mid : 0, i1 = hf ? P + 1 : mid, row = hf ? r2 : r1;
    const bool on = j < nr && (hf == 0 || r2 != r1);
    for (;;) {
        unsigned bi = 0;
        if (lane == 0) bi = atomicAdd(&pull[3], 1u);
        const int64_t b = (int64_t)__shfl_sync(0xffffffffu, bi, 0);
        if (b >= nbox) break;
        const int lv = level[b], p = parent[b], h2 = quadrant(ix[b], iy[b]);
        const bool leaf = nchild[b] == 0;
        if (w.sums && b == 0) strength_sums(w, lane);
        const cx<double> own = own_part(w, b, P, lane, g.invL * fmm::pow2<double>(lv + 1), loc);
        // its exponent, and the row of this lane
        const int Ex = (int)((__double_as_longlong(own.x) >> 52) & 0x7ff);
        const int Ey = (int)((__double_as_longlong(own.y) >> 52) & 0x7ff);
        const int Em = max(Ex, Ey);
        bool bad = __any_sync(0xffffffffu, Em == 0x7ff);
        int e = __reduce_max_sync(0xffffffffu, Em ? Em + (lane >> 1) : -4096) - 1022;
        const long long ox = __shfl_sync(0xffffffffu, __double_as_longlong(own.x), row);
        const long long oy = __shfl_sync(0xffffffffu, __double_as_longlong(own.y), row);
        long long sx = 0, sy = 0;
        if (lv >= 3) {
            int ep;
            longlong2 v = wait_words(LX + (int64_t)p * pitch, ex + p, P, lane, tag, lim, status, ep);
            mul_pow(v.x, v.y, (lane * h2) & 7);
            Zs[wid][lane] = words(v.x, v.y);
            __syncwarp();
            Sum acc{0, 0, 0, 0}, first{0, 0, 0, 0};
#pragma unroll 4
            for (int it = i0; it < i1; it++) {
                if (it == n1) {
                    first = acc;
                    acc = Sum{0, 0, 0, 0};
                }
                const int l = it < n1 ? r1 : r2, k = it < n1 ? r1 + it : r2 + (it - n1);
                add_term(acc, Wd[k * 32 + l], Zs[wid][k]);
            }
            if (i1 <= n1) {
                first = acc;
                acc = Sum{0, 0, 0, 0};
            }
            Sum s = meet(hf ? acc : first, hf ? first : acc);
            if (row == 0) {  // k = 0, weight 2^31
                const int4 z = Zs[wid][0];
                s.xl += (unsigned long long)(unsigned)z.x << 31;
                s.xh += (long long)z.y << 31;
                s.yl += (unsigned long long)(unsigned)z.z << 31;
                s.yh += (long long)z.w << 31;
            }
            sx = scale_sum(s.xh, s.xl, 31 + (row & 1));
            sy = scale_sum(s.yh, s.yl, 31 + (row & 1));
            mul_pow(sx, sy, (-row * h2) & 7);
            bad |= ep >= kBadExp;
            const int eb = max(e, ep);
            sx = shift_down(sx, eb - ep);
            sy = shift_down(sy, eb - ep);
            e = eb;
            __syncwarp();
        }
        sx += fixed54(ox, -(row >> 1), e + 1022);
        sy += fixed54(oy, -(row >> 1), e + 1022);
        if (leaf) {
            const double nan = __longlong_as_double(0x7ff8000000000000ll);
            const int E = e - 54 - (row >> 1);
            if (on)
                loc[b * P + row] = bad ? mk<double>(nan, nan)
                                       : mk<double>(pack_double(sx, E), pack_double(sy, E));
        } else {
            const int nb = __reduce_max_sync(0xffffffffu, on ? bits_of(sx, sy) : 0), sh = nb - 54;
            if (on)
                st_words(&LX[b * pitch + 2 * row], tag_word(rescale(sx, sh), tag),
                         tag_word(rescale(sy, sh), tag));
            if (lane == 0) st_word(&ex[b], tag_exp(bad ? kBadExp : nb == 0 ? kZeroExp : e + sh, tag));
            // the rows past P too: the two chains have orders of their own, and rows left with an
            // earlier launch's tag would pass for this kind's 255 launches on
            for (int r = P + lane; 2 * r < pitch; r += 32)
                st_words(&LX[b * pitch + 2 * r], tag_word(0, tag), tag_word(0, tag));
        }
    }
    if (lane == 0) {
        const unsigned total = gridDim.x * (unsigned)nw;
        if (atomicAdd(&pull[1], 1u) == total - 1u) {
            pull[1] = 0u;
            pull[3] = 0u;
            __threadfence();
            atomicExch(word, epoch + 1u);
        }
    }
}

BoxGeo geo_of(const Tree &T)
{
    return BoxGeo{T.xmin, T.ymin, T.L, (float)(1.0 / T.L), df64(1.0 / T.L), 1.0 / T.L};
}

}  // namespace

static unsigned *pass_words(const lbf_plan *pl) { return (unsigned *)(pl->loc_e + pl->xcap); }

static int l2l(lbf_plan *pl, int P, const Own &w, cx<double> *loc, int kid, const int *gate,
               cudaStream_t s)
{
    const Tree &T = pl->tree;
    const int64_t grid = std::min<int64_t>(lbf_cdiv(T.nbox, 8), 3 * (int64_t)std::max(pl->nsm, 1));
    LBF_LAUNCH_P(kid, k_l2l, lbf_grid(pl, grid), 256, 0, s, T.nbox, P, T.level, T.ix, T.iy, T.parent,
                 T.nchild, w, geo_of(T), pl->tab_binom, loc, pl->loc_X, pl->lx_pitch, pl->loc_e, pl->pull,
                 pass_words(pl) + 3, pl->dev_status, gate, pl->slab);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

// whether the plan's double applications take these passes
bool lbf_passes_ready(const lbf_plan *pl) { return pl->rows && pl->m2l_cap && pl->loc_X && pl->nbigx >= 0; }

int lbf_passes_build(lbf_plan *pl, cudaStream_t s, int32_t *scratch)
{
    pl->nbigx = -1;
    if (!pl->rows || !pl->m2l_cap) return LBF_OK;
    Tree &T = pl->tree;
    int32_t n = 0;
    const int cap = (int)std::min<int64_t>(pl->bigx_cap, INT32_MAX);
    LBF_CUDA(cudaMemsetAsync(scratch, 0, sizeof(int32_t), s));
    LBF_LAUNCH(k_bigx_list, lbf_cdiv(T.nbox, 256), 256, 0, s, T.nbox, pl->rows_thr, T.begin, T.end, T.nx,
               scratch, pl->bigx, cap);
    LBF_CHECK_LAUNCH();
    LBF_CUDA(cudaMemcpyAsync(&n, scratch, sizeof(n), cudaMemcpyDeviceToHost, s));
    LBF_CUDA(cudaStreamSynchronize(s));
    if (n <= cap) pl->nbigx = n;
    return LBF_OK;
}

// leaves and boxes a warp of k_up takes at a time, of n in all: several where every warp has
// many turns (16.8 million nodes, 8: 3.3 ms, 1: 3.6), one where the chain of a small tree
// counts.  (Boxes of k_l2l one by one: their parents are near in the order, and eight at a time
// held a level up, 29 ms against 3.)
static int run_of(int64_t n, int64_t warps) { return (int)std::max<int64_t>(1, std::min<int64_t>(8, n / (8 * warps))); }

// multipoles of the charges pl->q
int lbf_passes_up(lbf_plan *pl, const int *gate, cudaStream_t s)
{
    const Tree &T = pl->tree;
    const int P = pl->P, lch = (2 * P + 7) / 8;
    const int64_t grid = std::min<int64_t>(lbf_cdiv(T.nleaf + T.nbox, 4), 8 * (int64_t)std::max(pl->nsm, 1));
    LBF_LAUNCH_P(LBF_KERNEL_UP, k_up, lbf_grid(pl, grid), 128, 0, s, T.nleaf, T.nbox, T.leaves, T.ix, T.iy,
                 T.child0, T.nchild, P, lch, pl->rows_block0, pl->rows_items, pl->rows, pl->tab_binom,
                 pl->q, (cx<double> *)pl->mpole, pl->m2l_X, pl->m2l_e, pass_words(pl),
                 run_of(T.nleaf + T.nbox, 4 * grid), pl->dev_status, gate, pl->slab);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

// multipoles and full local expansions of the charges pl->q
int lbf_passes_apply(lbf_plan *pl, const int *gate, cudaStream_t s)
{
    const Tree &T = pl->tree;
    const int P = pl->P;
    int rc = lbf_passes_up(pl, gate, s);
    if (rc) return rc;
    rc = lbf_m2l_apply(pl, gate, s, true);
    if (rc) return rc;
    if (pl->nbigx > 0)
        LBF_LAUNCH_P(LBF_KERNEL_DOWN, k_p2l_big, lbf_grid(pl, pl->nbigx), 128, kP2lSmem, s,
                     (int)pl->nbigx, pl->bigx, T.level, T.ix, T.iy, T.begin, T.end, T.xlist, T.nx,
                     geo_of(T), P, pl->xi, pl->q, (cx<double> *)pl->local, gate, pl->slab);
    Own w{};
    w.ptr = pl->m2l_vptr;
    w.part = (const cx<double> *)pl->m2l_out;
    w.bg = T.begin;
    w.en = T.end;
    w.nx = T.nx;
    w.thr = pl->rows_thr;
    return l2l(pl, P, w, (cx<double> *)pl->local, LBF_KERNEL_DOWN, gate, s);
}

// Full local expansions of the multiplier potential E y (P = 32 terms, lbf_border.cu) and its
// sums of the strengths, from the stored expansions of the (box, centre) pairs: the P2L formed
// every pair's powers and logarithm again in each application, 7.1 ms for 5.3 million pairs
// where the stored coefficients are 0.4 ms of HBM, then wrote and read every expansion once
// more for the chain.
int lbf_mp_chain_apply(lbf_plan *pl, const double *y, const int *gate, cudaStream_t s)
{
    const Border &B = pl->bd;
    Own w{};
    w.ptr = B.p2l_ptr;
    w.part = (const cx<double> *)B.p2l_exp;
    w.src = B.p2l_src;
    w.y = y;
    w.sums = B.sums;
    w.kind = B.kind;
    w.lam = B.lam;
    w.M = pl->M;
    return l2l(pl, B.Pe, w, (cx<double> *)B.loc, LBF_KERNEL_ESUM, gate, s);
}

int lbf_passes_init_attrs()
{
    LBF_CUDA(cudaFuncSetAttribute(k_p2l_big, cudaFuncAttributeMaxDynamicSharedMemorySize, kP2lSmem));
    return LBF_OK;
}
