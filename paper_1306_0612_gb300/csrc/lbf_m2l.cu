// Multipole-to-local translations of the double FMM on the tensor cores.
//
// A same-level translation takes the 2 P reals of a source box's scaled multipole through
// one of 40 constant matrices,
//   out_l = sum_k T_o(l, k) a_k,   T_o(l, k) = (-1)^l C(k+l, l) t^(k+l+1),
//   t = 1/(2 (dx + i dy)), o = (dx, dy) the offset of the target box from the source,
// 2 P^2 double multiply-adds and 14 P more: at 16.8 million nodes 6.4 million translations
// took 17 ms of the double pipe (1/64 of the float rate).  Sorted by offset they are 40
// matrix products of up to half a million rows, and the tensor cores form them exactly from
// integer slices (Ozaki's scheme, as in the LU's trailing update, lbf_schur_lu.cu):
//
//   * each box's reals, scaled by 2^-(k/2) (|u| <= sqrt 2: the k-th power of a multipole may
//     grow like 2^(k/2)), are rounded once to integers of 54 bits below the box's largest
//     (k_m2l_fix); each row of T_o (an output) likewise below its largest entry;
//   * an integer is seven balanced base-256 digits, each exact in bf16; a product of two
//     digits is at most 2^14, a sum of 64 of them over at most seven digit pairs stays below
//     2^23: exact in the float accumulators of tcgen05.mma;
//   * the digit pairs with s + t <= 7 (34 of 49) go into eight TMEM accumulators, one per
//     s + t.  A dropped pair is at most 2^-62 of 2^108, all of them over 64 columns below 2^-53
//     of the product of the two maxima, 2^-59 as digits fall.  (Without s + t = 7, up to
//     2^-45 and 2^-51.4: measured on translations of forty charges over all offsets, in units of
//     2^-53 of their absolute sum, 0.63, with it 0.13, as a double evaluation, which rounds each
//     of its terms, 0.40);
//   * the accumulators are combined as integers and packed into doubles without an
//     instruction on the double pipe.
//
// Work: 34 products of 128 x N x K a tile of 128 translations (N, K = 2 P rounded up to 16).
// The matrix's digits stand one after another along N, so digit s of the rows meets digits
// 0 .. 7 - s of the matrix in one or two MMAs of up to 256 columns, twelve a K step of 16 (one
// digit pair an MMA re-read the 4 KB of rows for every 64 columns).  k_m2l_tc is persistent,
// one CTA an SM: eight warps expand the gathered rows' digits into shared memory (112 KB; the
// next tile's integers are fetched before the wait for the MMAs) and one of their threads
// issues the MMAs, eight warps read the accumulators back and write each translation's local
// expansion; the expansion of one tile's digits overlaps the readout of the one before: 2.9 ms for
// the 6.6 million translations at 16.8 million nodes (2.65 without the products of place 7).  The
// target's warp in k_down then adds its translations in list order (two additions a
// coefficient).
//
// Chosen for P <= 32 (K = 64: one accumulator set fills TMEM's 512 columns); longer
// expansions keep the double loop in k_down.
#include <algorithm>

#include "lbf_fixed.cuh"
#include "lbf_fmm_tpl.cuh"
#include "lbf_tc.cuh"

using fmm::cx;

namespace {

constexpr int kSl = 7;                  // digits of an operand
constexpr int kAcc = 8;                 // sums of digit products, by the digits' places
constexpr int kRowsT = 128;             // translations a tile
constexpr int kABytes = kRowsT * 64 * 2;  // one digit of a tile's rows
constexpr int kBBytes = 64 * 64 * 2;      // room for one digit of a translation matrix
constexpr int kM2lSmem = kSl * (kABytes + kBBytes);
constexpr int kM2lThreads = 512;
constexpr int kNoffs = 49;              // offsets (dx + 3) 7 + dy + 3
constexpr unsigned kM2lSpins = 1u << 24;

__host__ __device__ inline int tile_cols(int P) { return (2 * P + 15) / 16 * 16; }

// the seven base-256 digits of x (|x| <= 2^54), most significant first, each plus 128
__device__ __forceinline__ unsigned long long digits(long long x)
{
    return (unsigned long long)(x + 0x0080808080808080ll);
}
// digit s (0 the most significant) as a float
__device__ __forceinline__ float digit_f(unsigned lo, unsigned hi, int s)
{
    const int byte = 6 - s;
    const unsigned w = byte < 4 ? lo : hi;
    return __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7440u | (unsigned)(byte & 3))) - 8388736.0f;
}

// every box's multipole as integers (pitch reals a box), and its exponent, a warp per box
__global__ void k_m2l_fix(int64_t nbox, int P, const cx<double> *__restrict__ mp,
                          long long *__restrict__ X, int32_t *__restrict__ ex, const int *gate,
                          int64_t slab)
{
    lbf_rhs(slab, mp, X, ex, gate);
    if (fmm::gate_closed(gate)) return;
    const int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (b >= nbox) return;
    const long long *a = (const long long *)(mp + b * P);
    long long v[2];
    int top = -4096;
    bool bad = false;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int m = lane + 32 * h;
        v[h] = m < 2 * P ? a[m] : 0;
        const int E = (int)((v[h] >> 52) & 0x7ff);
        bad |= E == 0x7ff;
        if (E) top = max(top, E - (m >> 2));
    }
    top = __reduce_max_sync(0xffffffffu, top);
    bad = __any_sync(0xffffffffu, bad);
    const int pitch = real_pitch(P);
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int m = lane + 32 * h;
        if (m < pitch) X[b * pitch + m] = tag_word(fixed54(v[h], m >> 2, top), 0);
    }
    if (lane == 0) ex[b] = tag_exp(bad ? kBadExp : top - 1022, 0);
}

// digit images (the rows of the digits one after another) and row exponents of the
// translation matrices, a block per offset
__global__ void k_m2l_matrices(int P, const double *__restrict__ binom,
                               const cx<double> *__restrict__ tpow, uint4 *__restrict__ img,
                               int32_t *__restrict__ fx)
{
    const int o = blockIdx.x, dx = o / 7 - 3, dy = o % 7 - 3;
    if (abs(dx) <= 1 && abs(dy) <= 1) return;
    __shared__ int top[64];
    const cx<double> *tp = tpow + (size_t)o * (LBF_MAX_TERMS + 1);
    const int N = tile_cols(P);
    unsigned short *out = (unsigned short *)(img + (size_t)o * kSl * kBBytes / 16);
    for (int n = threadIdx.x; n < 64; n += blockDim.x) top[n] = -4096;
    __syncthreads();
    // row n = 2 l + (0: Re, 1: Im), column k' = 2 k + (0: Re, 1: Im): the real form of T_o
    auto entry = [&](int n, int kk) {
        const int l = n >> 1, k = kk >> 1;
        if (l >= P || k >= P) return 0.0;
        const cx<double> t = fmm::cmul(tp[k], tp[l + 1]);
        const double c = binom[(k + l) * LBF_MAX_TERMS + l];
        double v = (n & 1) == (kk & 1) ? t.x : ((n & 1) ? t.y : -t.y);
        if (l & 1) v = -v;
        return v * c * fmm::pow2<double>(k >> 1);
    };
    for (int e = threadIdx.x; e < N * 64; e += blockDim.x) {
        const double v = entry(e >> 6, e & 63);
        const int E = (int)((__double_as_longlong(v) >> 52) & 0x7ff);
        if (E) atomicMax(&top[e >> 6], E);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < N * 64; e += blockDim.x) {
        const int n = e >> 6, kk = e & 63;
        const unsigned long long d = digits(fixed54(__double_as_longlong(entry(n, kk)), 0, top[n]));
        for (int s = 0; s < kSl; s++)
            out[core_off(s * N + n, kk)] =
                (unsigned short)(__float_as_uint(digit_f((unsigned)d, (unsigned)(d >> 32), s)) >> 16);
    }
    for (int n = threadIdx.x; n < 64; n += blockDim.x) fx[o * 64 + n] = top[n] - 1022;
}

// ---- the translations sorted by offset (plan time) ----------------------------------

__device__ __forceinline__ int offset_of(int bx, int by, int sx, int sy)
{
    return (bx - sx + 3) * 7 + (by - sy + 3);
}

__global__ void k_m2l_count(int64_t nbox, const int32_t *__restrict__ nv, int32_t *__restrict__ cnt)
{
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b <= nbox) cnt[b] = b < nbox ? nv[b] : 0;
}

__global__ void k_m2l_hist(int64_t nbox, const int32_t *__restrict__ ix, const int32_t *__restrict__ iy,
                           const int32_t *__restrict__ vlist, const int32_t *__restrict__ nv,
                           int32_t *__restrict__ hist)
{
    __shared__ int sh[kNoffs];
    for (int k = threadIdx.x; k < kNoffs; k += blockDim.x) sh[k] = 0;
    __syncthreads();
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b < nbox)
        for (int q = 0; q < nv[b]; q++) {
            const int s = vlist[b * 27 + q];
            atomicAdd(&sh[offset_of(ix[b], iy[b], ix[s], iy[s])], 1);
        }
    __syncthreads();
    for (int k = threadIdx.x; k < kNoffs; k += blockDim.x)
        if (sh[k]) atomicAdd(&hist[k], sh[k]);
}

// tile0[o]: first tile of offset o (each offset's last tile filled up with empty rows);
// the histogram becomes the offsets' write positions
__global__ void k_m2l_tiles(int32_t *hist, int32_t *tile0)
{
    if (threadIdx.x || blockIdx.x) return;
    int t = 0;
    for (int o = 0; o < kNoffs; o++) {
        const int n = hist[o];
        tile0[o] = t;
        hist[o] = t * kRowsT;
        t += (n + kRowsT - 1) / kRowsT;
    }
    tile0[kNoffs] = t;
}

// (source box, row of the result) of every translation; the order within an offset is that
// of the atomics, and no result depends on it
__global__ void k_m2l_place(int64_t nbox, const int32_t *__restrict__ ix, const int32_t *__restrict__ iy,
                            const int32_t *__restrict__ vlist, const int32_t *__restrict__ nv,
                            const int32_t *__restrict__ vptr, int32_t *__restrict__ cursor,
                            int2 *__restrict__ pairs)
{
    __shared__ int sh[kNoffs], at[kNoffs];
    for (int k = threadIdx.x; k < kNoffs; k += blockDim.x) sh[k] = 0;
    __syncthreads();
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int n = b < nbox ? nv[b] : 0;
    for (int q = 0; q < n; q++) {
        const int s = vlist[b * 27 + q];
        atomicAdd(&sh[offset_of(ix[b], iy[b], ix[s], iy[s])], 1);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kNoffs; k += blockDim.x) {
        at[k] = sh[k] ? atomicAdd(&cursor[k], sh[k]) : 0;
        sh[k] = 0;
    }
    __syncthreads();
    for (int q = 0; q < n; q++) {
        const int s = vlist[b * 27 + q], o = offset_of(ix[b], iy[b], ix[s], iy[s]);
        pairs[at[o] + atomicAdd(&sh[o], 1)] = make_int2(s, vptr[b] + q);
    }
}

// ---- per application -----------------------------------------------------------------

__global__ void __launch_bounds__(kM2lThreads, 1)
k_m2l_tc(int P, const int32_t *__restrict__ tile0, const int2 *__restrict__ pairs,
         const long long *__restrict__ X, const int32_t *__restrict__ ex,
         const uint4 *__restrict__ img, const int32_t *__restrict__ fx, double *__restrict__ out,
         const int *gate, int *status, int64_t slab)
{
    lbf_rhs(slab, X, ex, out, gate);
    if (fmm::gate_closed(gate)) return;
    extern __shared__ __align__(128) uint4 sm[];
    __shared__ uint32_t tmem_base;
    __shared__ __align__(8) unsigned long long bar_b, bar_mma, bar_free;
    __shared__ int s_tile0[kNoffs + 1];
    constexpr int kHalf = kM2lThreads / 2;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint4 *sA = sm, *sB = sm + kSl * kABytes / 16;
    const uint32_t mb = smem_u32(&bar_b), mm = smem_u32(&bar_mma), mf = smem_u32(&bar_free);
    for (int k = tid; k <= kNoffs; k += blockDim.x) s_tile0[k] = tile0[k];
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&tmem_base)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(mb), "r"(1) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(mm), "r"(1) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(mf), "r"(kHalf / 32) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int N = tile_cols(P), nk = N / 16, pitch = real_pitch(P), nc = pitch / 8;
    // columns past the reals stay zero
    for (int k = tid; k < kSl * kRowsT * (8 - nc); k += blockDim.x) {
        const int c = nc + k % (8 - nc), r = k / (8 - nc) % kRowsT, d = k / (8 - nc) / kRowsT;
        sA[(d * kABytes + 2 * core_off(r, 8 * c)) / 16] = make_uint4(0, 0, 0, 0);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    // every wait is bounded; after one has given up the others of its thread poll once, so
    // the loop (the same for all threads) still ends and the status word says why
    unsigned lim = wait_limit(status, kM2lSpins);
    auto wait = [&](uint32_t bar, uint32_t parity) {
        if (!mbar_wait(bar, parity, lim)) {
            atomicOr(status, LBF_DEV_TIMEOUT);
            lim = 1;
        }
    };
    const int ntile = s_tile0[kNoffs];
    const int t0 = (int)((long long)ntile * blockIdx.x / gridDim.x);
    const int t1 = (int)((long long)ntile * (blockIdx.x + 1) / gridDim.x);
    if (tid >= kHalf) {
        // ---- digits into shared memory, MMAs: two threads a row, alternate chunks of 8 ----
        const int r = tid & (kRowsT - 1), c0 = (tid - kHalf) / kRowsT;
        const uint64_t dA = tc_desc(smem_u32(sA)), dB = tc_desc(smem_u32(sB));
        longlong2 x[4][4];
        auto fetch = [&](int t) {
            const int src = t < t1 ? pairs[(int64_t)t * kRowsT + r].x : -1;
            const longlong2 *xr = (const longlong2 *)(X + (int64_t)max(src, 0) * pitch);
#pragma unroll
            for (int h = 0; h < 4; h++)
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const int c = c0 + 2 * h;
                    x[h][i] = src >= 0 && c < nc ? xr[4 * c + i] : make_longlong2(0, 0);
                }
        };
        int o = -1;
        unsigned nb = 0;
        fetch(t0);
        for (int t = t0; t < t1; t++) {
            const unsigned n = (unsigned)(t - t0);
            if (n > 0) wait(mm, (n - 1) & 1);  // the operands are free
            bool load = false;
            while (o < 0 || t >= s_tile0[o + 1]) {
                o++;
                load = true;
            }
            if (load && tid == kHalf) {
                const int bytes = kSl * N * 128;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                             :: "r"(mb), "r"(bytes) : "memory");
                bulk_g2s(smem_u32(sB), (const char *)img + (size_t)o * kSl * kBBytes, bytes, mb);
            }
#pragma unroll
            for (int h = 0; h < 4; h++) {
                const int c = c0 + 2 * h;
                if (c >= nc) break;
                unsigned lo[8], hi[8];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const unsigned long long a = digits(untag(x[h][i].x)), b = digits(untag(x[h][i].y));
                    lo[2 * i] = (unsigned)a;
                    hi[2 * i] = (unsigned)(a >> 32);
                    lo[2 * i + 1] = (unsigned)b;
                    hi[2 * i + 1] = (unsigned)(b >> 32);
                }
#pragma unroll
                for (int s = 0; s < kSl; s++) {
                    unsigned w[4];
#pragma unroll
                    for (int i = 0; i < 4; i++)  // two exact bf16 are the upper halves of two floats
                        w[i] = __byte_perm(__float_as_uint(digit_f(lo[2 * i], hi[2 * i], s)),
                                           __float_as_uint(digit_f(lo[2 * i + 1], hi[2 * i + 1], s)), 0x7632);
                    sA[(s * kABytes + 2 * core_off(r, 8 * c)) / 16] = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("bar.sync 1, %0;" :: "r"(kHalf) : "memory");
            if (tid == kHalf) {
                if (load) wait(mb, nb++ & 1);
                if (n > 0) wait(mf, (n - 1) & 1);  // the accumulators have been read
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // digit s of the rows by digits 0 .. 7 - s of the matrix into sums s .. 7 (sum 7
                // begins with s = 1, the others with s = 0)
                auto mul = [&](int s, int c, int w, bool first) {
                    const uint32_t idesc = tc_idesc(kRowsT, w);
                    for (int k = 0; k < nk; k++)
                        tc_mma(tmem + (uint32_t)(s * N + c), dA + (uint64_t)((s * kABytes + k * 256) >> 4),
                               dB + (uint64_t)((c * 128 + k * 256) >> 4), idesc, !first || k > 0 ? 1u : 0u);
                };
                for (int s = 0; s < kSl; s++) {
                    const int cols = (s == 0 ? kSl : s == 1 ? kSl - 1 : kAcc - s) * N;
                    for (int c = 0; c < cols; c += 256) mul(s, c, min(256, cols - c), s == 0);
                    if (s == 1) mul(1, cols, N, true);
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             :: "r"(mm) : "memory");
            }
            fetch(t + 1);
        }
        if (t1 > t0) wait(mm, (unsigned)(t1 - t0 - 1) & 1);
    } else {
        // ---- accumulators into local expansions: two threads a translation, half of the
        //      columns each ----
        const int quarter = warp & 3, h0 = (warp >> 2) * (N / 2);
        const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
        int o = 0;
        for (int t = t0; t < t1; t++) {
            const unsigned n = (unsigned)(t - t0);
            while (t >= s_tile0[o + 1]) o++;
            const int2 pr = pairs[(int64_t)t * kRowsT + quarter * 32 + lane];
            const int e = pr.x >= 0 ? untag_exp(ex[pr.x]) : 0;
            const int32_t *f = fx + o * 64;
            double *dst = out + (int64_t)pr.y * 2 * P;
            wait(mm, n & 1);
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int c = h0; c < h0 + N / 2; c += 8) {
                float a[kAcc][8];
#pragma unroll
                for (int g = 0; g < kAcc; g++) tc_ld8(trow + (uint32_t)(g * N + c), a[g]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int g = 0; g < kAcc; g++)
#pragma unroll
                    for (int i = 0; i < 8; i++) asm volatile("" : "+f"(a[g][i]));  // not before the wait
                if (c + 8 >= h0 + N / 2) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0)
                        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(mf) : "memory");
                }
                if (pr.x >= 0) {
                    double v[8];
#pragma unroll
                    for (int i = 0; i < 8; i++) {
                        int d[kAcc];
#pragma unroll
                        for (int g = 0; g < kAcc; g++) d[g] = __float2int_rn(a[g][i]);
                        // sum_g d_g 256^(6 - g) in units of 16
                        const long long w = (long long)(d[0] * 256 + d[1]) * (1ll << 36) +
                                            (long long)(d[2] * 256 + d[3]) * (1ll << 20) +
                                            (long long)(d[4] * 256 + d[5]) * 16ll +
                                            ((d[6] + ((d[7] + 128) >> 8) + 8) >> 4);
                        v[i] = pack_double(w, e + f[c + i] - 56);
                    }
                    if (e == kBadExp)  // an infinity or NaN in the multipole
#pragma unroll
                        for (int i = 0; i < 8; i++) v[i] = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
                    for (int i = 0; i < 8; i += 2)
                        if (c + i < 2 * P) *(double2 *)(dst + c + i) = make_double2(v[i], v[i + 1]);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(512) : "memory");
}

}  // namespace

// Room for the translations: 4 a reserved box (measured 2.3), in a small system, whose reserve is
// mostly for depth, 6 a box of 8 N / leaf_size (measured 3 to 4.4), dropped when the workspace
// has none.  The buffers an application writes are a right-hand side's own (layout of views too).
void lbf_m2l_layout_rhs(const lbf_plan *pl, lbf_plan *v, Arena &A)
{
    const bool on = pl->m2l_cap > 0;
    v->m2l_X = on ? A.get<long long>(pl->xcap * real_pitch(pl->P)) : nullptr;
    v->m2l_e = on ? A.get<int32_t>(pl->xcap) : nullptr;
    v->m2l_out = on ? A.get<double>(pl->m2l_cap * 2 * pl->P) : nullptr;
}

void lbf_m2l_layout(lbf_plan *pl, const lbf_options &o, int64_t cap)
{
    pl->m2l_cap = 0;
    if (o.matvec != LBF_MATVEC_FMM || o.p + 1 > 32 || !(pl->parts & LBF_PART_M2L)) return;
    Arena &A = pl->arena;
    const size_t off = A.off;
    const bool full = A.overflow;
    pl->P = o.p + 1;
    pl->m2l_cap = std::min<int64_t>(4 * cap, 6 * pl->xcap);
    pl->m2l_pairs = A.get<int2>(pl->m2l_cap + kNoffs * kRowsT);
    pl->m2l_vptr = A.get<int32_t>(cap + 1);
    pl->m2l_tile0 = A.get<int32_t>(2 * (kNoffs + 1));
    pl->m2l_img = A.get<uint4>((int64_t)kNoffs * kSl * kBBytes / 16);
    pl->m2l_f = A.get<int32_t>(kNoffs * 64);
    lbf_m2l_layout_rhs(pl, pl, A);
    if (A.overflow && !full) {
        A.off = off;
        A.overflow = false;
        pl->m2l_cap = 0;
    }
}

int lbf_m2l_init_attrs()
{
    LBF_CUDA(cudaFuncSetAttribute(k_m2l_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kM2lSmem));
    return LBF_OK;
}

int lbf_m2l_build(lbf_plan *pl, cudaStream_t s, int32_t *scratch, int64_t scratch_len)
{
    if (!pl->m2l_cap) return LBF_OK;
    Tree &T = pl->tree;
    const int64_t nb = T.nbox;
    int32_t *hist = pl->m2l_tile0 + kNoffs + 1;
    LBF_CUDA(cudaMemsetAsync(hist, 0, sizeof(int32_t) * kNoffs, s));
    LBF_LAUNCH(k_m2l_matrices, kNoffs, 256, 0, s, pl->P, pl->tab_binom,
               (const cx<double> *)pl->tab_tpow, (uint4 *)pl->m2l_img, pl->m2l_f);
    LBF_LAUNCH(k_m2l_count, lbf_cdiv(nb + 1, 256), 256, 0, s, nb, T.nv, pl->m2l_vptr);
    LBF_LAUNCH(k_m2l_hist, lbf_cdiv(nb, 256), 256, 0, s, nb, T.ix, T.iy, T.vlist, T.nv, hist);
    LBF_LAUNCH(k_m2l_tiles, 1, 32, 0, s, hist, pl->m2l_tile0);
    LBF_CHECK_LAUNCH();
    const int rc = lbf_scan_i32(pl->m2l_vptr, pl->m2l_vptr, nb + 1, scratch, scratch_len, s);
    if (rc) return rc;
    int32_t n = 0, tiles = 0;
    LBF_CUDA(cudaMemcpyAsync(&n, pl->m2l_vptr + nb, sizeof(n), cudaMemcpyDeviceToHost, s));
    LBF_CUDA(cudaMemcpyAsync(&tiles, pl->m2l_tile0 + kNoffs, sizeof(tiles), cudaMemcpyDeviceToHost, s));
    LBF_CUDA(cudaStreamSynchronize(s));
    if (n > pl->m2l_cap || nb > pl->xcap) {
        pl->m2l_cap = 0;
        return LBF_OK;
    }
    pl->m2l_tiles = tiles;
    LBF_CUDA(cudaMemsetAsync(pl->m2l_pairs, 0xff, sizeof(int2) * (size_t)tiles * kRowsT, s));
    LBF_LAUNCH(k_m2l_place, lbf_cdiv(nb, 256), 256, 0, s, nb, T.ix, T.iy, T.vlist, T.nv, pl->m2l_vptr,
               hist, pl->m2l_pairs);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

// m2l_out from the plan's (or view's) multipoles, of which m2l_X and m2l_e hold the integers
// already where `fixed` is set (lbf_passes.cu)
int lbf_m2l_apply(lbf_plan *pl, const int *gate, cudaStream_t s, bool fixed)
{
    if (!pl->m2l_tiles) return LBF_OK;
    const Tree &T = pl->tree;
    if (!fixed)
        LBF_LAUNCH_P(LBF_KERNEL_DOWN, k_m2l_fix, lbf_grid(pl, lbf_cdiv(T.nbox, 8)), 256, 0, s, T.nbox, pl->P,
                     (const cx<double> *)pl->mpole, pl->m2l_X, pl->m2l_e, gate, pl->slab);
    const int64_t grid = std::min<int64_t>(pl->m2l_tiles, std::max(pl->nsm, 1));
    LBF_LAUNCH_P(LBF_KERNEL_DOWN, k_m2l_tc, lbf_grid(pl, grid), kM2lThreads, kM2lSmem, s, pl->P, pl->m2l_tile0,
                 pl->m2l_pairs, pl->m2l_X, pl->m2l_e, (const uint4 *)pl->m2l_img, pl->m2l_f, pl->m2l_out,
                 gate, pl->dev_status, pl->slab);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}
