// Stored leaf rows: the part of the density block's forward rows (Sec. 5, Eq. disc_sphere)
// that depends on the geometry alone, kept per plan as dense tiles and applied as a
// matrix-vector product.
//
// For a node i of leaf b the accurate forward row is
//   v_i = sum_j G_ij sigma_j + sum_k M_ik mp_s[k] + sum_l L_il loc_b[l] + 2 beta.sigma,
//   G_ij = (1/pi) Im(w_j / (xi_j - xi_i)),  G_ii = 2 dself_i,
//   L_i  = the L2P of the leaf's local expansion, -(1/pi) Im(b_l u_i^l), u_i = (xi_i - c)/r,
//   M_i  = the M2P of the other boxes s of W(b), -(1/pi) Im(a_k rho^(k+1))/r_s,
//          rho = r_s/(xi_i - c_s),
// with j over the near nodes of b: U(b), the small boxes of W(b), and the small boxes' X
// lists (below).  A GMRES solve applies the same rows tens of times.
//
// Why stored: this GPU issues double at 1/64 of float, and a near pair formed on the fly
// takes ten double instructions (difference, squared distance, reciprocal, product) of
// which one, the multiply-add with sigma_j, depends on the density.  At 16.8 million nodes
// (2.1e9 pairs) that is 33 ms of the double pipe per application; 8 bytes a pair from HBM
// are 2.5 ms and the multiply-adds 3.3 ms.
//
// Small W and X boxes enter as pairs: for c a leaf, s in W(c) with n_s nodes, the M2P at
// c's nodes and the P2L of c's nodes into s cost about 10 P double instructions per node
// of c, the pairs in both directions 2 n_s multiply-adds, so s is taken as pairs when
// n_s <= 4 P (and exactly, without a truncated expansion); k_down then leaves out X(s).
// The others' M2P rows are columns too (2 P reals of the multipole a box): 0.06 to 0.08
// such boxes a leaf, but up to 22, and a chain of P dependent steps for each, run by the
// leaf's warp, held the launch at 181,783 nodes to 250 us.
//
// On the integer pipes: a double multiply-add leaves a scheduler every 64 cycles, the three
// 32 x 32 -> 64 bit products that stand for one every 17 (lbf_fixed.cuh).  An entry is an integer
// of 54 bits below its row's largest near entry (rexp), the density below the largest of the run
// of up to 512 columns it is summed with, the local columns and the expansion below fixed sizes
// (|u_i^l| 2^-(l/2) < 3/2); the sums are exact but for the products' last 52 bits.  Errors of whole
// applications against 64 bits are what they were with double entries, to three digits, at orders
// 22 to 31; of single rows, relative to the sums of their terms' sizes, they are a few 2^-53 or less,
// also where densities of 1 and 1e-12 meet, and blocks whose entries differ too much stay double
// (kWideTop).  The multipole columns, few and in units of their own, stay double.
//
// Layout: a leaf's rows are cut into blocks of at most kGroups groups of four rows, its
// columns into chunks of eight; a tile is one group x one chunk, 32 doubles, row-major,
// so lane = 8 (row mod 4) + (column mod 8) and a warp's load is 256 contiguous bytes.  A
// block's tiles are stored chunk by chunk: the near nodes, the W multipoles' reals, then
// the 2 P reals of the local expansion.  Each lane holds one sum per group; eight lanes share a
// row, and a butterfly that halves the groups at each step adds them in 7 additions for 8 groups (lanes on
// rows alone would leave 19 % of the lanes idle at 26 nodes a leaf, lanes on columns
// alone would add 31 shuffled sums to 4 x 26 multiply-adds).
//
// Measured, rows of one application at 16.8 million nodes, 416,768 and 8192: 6.6 ms, 128 us
// and 16 us (double entries 7.4 ms, 201 us, 22 us); transposed, 131,072 nodes, 93 and 97 us
// (147 and 137).  Bound by memory at the large end, 36.4 GB (25.6 of entries, the rest the padding of
// rows to four and columns to eight) at 5.55 of 6.68 TB/s, by the latency of the tiles' loads below:
// the next eight chunks are asked for ahead, four are read at once; more warps with fewer loads
// each were slower (6.9 ms with two chunks at once, 8.8 with 24 warps an SM).
//
// The transposed rows (K^T tau)_i read the same tiles: near pairs are symmetric (b's columns
// hold leaf t's nodes exactly when t's hold b's), so each leaf forms z = G_b^T tau_b over its
// columns (k_rows_t) and a node adds its entry of every z it is a column of, in a fixed
// order (k_rows_t_out), from a list per leaf of where its nodes begin in the others' columns.
// The far field is Im(w_i Phi(xi_i)): the same local and M2P columns with two sums a row.
#include <algorithm>

#include "lbf_fixed.cuh"
#include "lbf_fmm_tpl.cuh"

using fmm::BoxGeo;
using fmm::cx;

namespace {

// kGroups row groups a warp where there are leaves enough to fill the chip; in a smaller
// system a leaf is shared by several thread blocks of four warps (kGroupsSmall row groups a
// block, a quarter of the columns a warp): 326 leaves of 8192 nodes would fill half a wave
constexpr int kGroups = 8, kGroupsSmall = 2;
// (8192 nodes: 458 us an application with whole leaves a warp, 408 shared; at 7130 leaves
// the two are within 1 %, at 16,150 sharing costs 4 % of a solve)
constexpr int64_t kSmallLeaves = 4864;
// (several right-hand sides in lockstep share no columns once their blocks make this many warps
// an SM, four times what is resident; their sums are those of a separate solve all the same:
// 16 of 64,000 nodes 1003 us shared, 850 not)
constexpr int64_t kFullWarps = 64;
constexpr int kLocalTop = 1021;  // exponent field of the local columns' largest: [1/4, 1/2)
constexpr int kRowBlocks = 4;    // thread blocks an SM
constexpr int kRun = 4;          // chunks read at a time (2 or 4)
constexpr int kAhead = 8;        // chunks asked for before they are read
// A block with a near entry of 1/2 or more, or one that is not finite, keeps its near entries as
// doubles.  Entries above 1/pi are curves closer than their node spacing; the integers would
// take from the row's other entries what such an entry needs, and in transposed sums, which have
// one unit for a block's rows, from all of the block's columns (median error of transposed rows
// beside two islands that touch, in units of 2^-53 of their terms: 0.9 with entries up to 0.3, 48
// with 32, 409 with 3200; 18 to 20 with pairs formed on the fly, 1 to 2 as doubles).
constexpr int kWideTop = 1021;  // largest exponent field of an integer block's entries
constexpr int kDotChunks = 64;   // chunks a Dot takes at most between two conversions (a multiple of 4)
static_assert(kDotChunks % 4 == 0, "xs is filled by four chunks");

// the column ranges of leaf b, in order: U(b), the small boxes of W(b), the X lists of
// b and its ancestors that are small.  f(first node, end)
struct TreeLists {
    const int32_t *level, *ix, *iy, *parent, *begin, *end, *uptr, *uidx, *wptr, *widx, *xlist, *nx;
};
// (f(first node, end) in a fixed order)
template <class F> __device__ __forceinline__ void for_ranges(const TreeLists &T, int b, int thr, F f)
{
    for (int q = T.uptr[b]; q < T.uptr[b + 1]; q++) f(T.begin[T.uidx[q]], T.end[T.uidx[q]]);
    for (int q = T.wptr[b]; q < T.wptr[b + 1]; q++) {
        const int s = T.widx[q];
        if (T.end[s] - T.begin[s] <= thr) f(T.begin[s], T.end[s]);
    }
    for (int a = b; a >= 0 && T.end[a] - T.begin[a] <= thr; a = T.parent[a])
        for (int q = 0; q < T.nx[a]; q++) {
            const int c = T.xlist[a * 16 + q];
            f(T.begin[c], T.end[c]);
        }
}

__device__ __forceinline__ long long near_nodes(const TreeLists &T, int b, int thr)
{
    long long n = 0;
    for_ranges(T, b, thr, [&](int s, int e) { n += e - s; });
    return n;
}
// the boxes of W(b) that enter by M2P
__device__ __forceinline__ int big_boxes(const TreeLists &T, int b, int thr)
{
    int n = 0;
    for (int q = T.wptr[b]; q < T.wptr[b + 1]; q++)
        n += T.end[T.widx[q]] - T.begin[T.widx[q]] > thr ? 1 : 0;
    return n;
}

// per leaf: its near chunks and row blocks; total[0] += tiles, total[1] += chunks
__global__ void k_rows_count(int64_t nleaf, const int32_t *__restrict__ leaves, TreeLists T,
                             int thr, int P, int lchunks, int groups, int32_t *__restrict__ chunks,
                             int32_t *__restrict__ blocks, int32_t *__restrict__ tiles,
                             unsigned long long *__restrict__ total)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    unsigned long long nt = 0, nc = 0;
    if (t < nleaf) {
        const int b = leaves[t];
        const long long ch = (near_nodes(T, b, thr) + 7) / 8 + (2ll * P * big_boxes(T, b, thr) + 7) / 8, g = (T.end[b] - T.begin[b] + 3) / 4;
        nc = (unsigned long long)ch;
        nt = (unsigned long long)(g * (ch + lchunks));
        chunks[t] = (int32_t)ch;
        blocks[t] = (int32_t)((g + groups - 1) / groups);
        tiles[t] = nt < (1ull << 30) ? (int32_t)nt : (1 << 30);
    }
    for (int o = 16; o > 0; o >>= 1) {
        nt += __shfl_xor_sync(0xffffffffu, nt, o);
        nc += __shfl_xor_sync(0xffffffffu, nc, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&total[0], nt);
        atomicAdd(&total[1], nc);
    }
}

// the row blocks of each leaf, a thread per leaf (groups spread evenly over its blocks)
__global__ void k_rows_items(int64_t nleaf, const int32_t *__restrict__ leaves, TreeLists T,
                             int thr, int lchunks, int groups, const int32_t *__restrict__ chunk0,
                             const int32_t *__restrict__ block0, const int32_t *__restrict__ tile0,
                             RowItem *__restrict__ items, int32_t *__restrict__ leaf)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= nleaf) return;
    const int b = leaves[t];
    const int n = T.end[b] - T.begin[b], g = (n + 3) / 4, nb = (g + groups - 1) / groups;
    const int ch = chunk0[t + 1] - chunk0[t];
    for (int i = T.begin[b]; i < T.end[b]; i++) leaf[i] = (int32_t)t;
    for (int k = 0; k < nb; k++) {
        const int g0 = (int)((long long)g * k / nb), g1 = (int)((long long)g * (k + 1) / nb);
        RowItem it;
        it.box = b;
        it.row0 = T.begin[b] + 4 * g0;
        it.nrow = min(n, 4 * g1) - 4 * g0;
        it.tile = tile0[t] + g0 * (ch + lchunks);
        it.chunk = chunk0[t];
        it.nchunk = ch;
        it.ncol = (int)near_nodes(T, b, thr);
        it.leaf = (int32_t)t;
        items[block0[t] + k] = it;
    }
}

// each leaf's columns, a warp per leaf: the near nodes, then from the next chunk on -1 - m for
// the real m of the multipoles; both are filled up to a chunk with the leaf's first node (zero
// entries)
__global__ void k_rows_cols(int64_t nleaf, const int32_t *__restrict__ leaves, TreeLists T, int thr,
                            int P,
                            const int32_t *__restrict__ chunk0, int32_t *__restrict__ cols)
{
    const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (t >= nleaf) return;
    const int b = leaves[t];
    int32_t *c = cols + (int64_t)chunk0[t] * 8;
    int m = 0;
    for_ranges(T, b, thr, [&](int s, int e) {
        for (int j = s + lane; j < e; j += 32) c[m + j - s] = j;
        m += e - s;
    });
    if (m + lane < (m + 7) / 8 * 8) c[m + lane] = T.begin[b];
    m = (m + 7) / 8 * 8;
    for (int q = T.wptr[b]; q < T.wptr[b + 1]; q++) {
        const int s = T.widx[q];
        if (T.end[s] - T.begin[s] <= thr) continue;
        for (int e = lane; e < 2 * P; e += 32) c[m + e] = -1 - (s * 2 * P + e);
        m += 2 * P;
    }
    if (m + lane < (m + 7) / 8 * 8) c[m + lane] = T.begin[b];
}

// Per leaf, where its first node stands in the columns of the leaves that hold its nodes: a
// thread per holding leaf goes through its own columns and appends to the lists of the leaves
// it finds (base null: counts them), and k_rows_rev_sort puts each list in ascending order, so
// that the sums over it do not depend on the atomics.
__global__ void k_rows_rev(int64_t nleaf, const int32_t *__restrict__ leaves, TreeLists T, int thr,
                           const int32_t *__restrict__ chunk0, const int32_t *__restrict__ leaf,
                           int32_t *__restrict__ count, const int32_t *__restrict__ ptr,
                           int32_t *__restrict__ base)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= nleaf) return;
    int at = chunk0[t] * 8;
    for_ranges(T, leaves[t], thr, [&](int s, int e) {
        for (int j = s; j < e;) {
            const int h = leaf[j], k = atomicAdd(&count[h], 1), next = T.end[leaves[h]];
            if (base) base[ptr[h] + k] = at + (j - s);
            j = next;
        }
        at += e - s;
    });
}

__global__ void k_rows_rev_sort(int64_t nleaf, const int32_t *__restrict__ ptr, int32_t *__restrict__ base)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= nleaf) return;
    for (int i = ptr[t] + 1; i < ptr[t + 1]; i++) {
        const int32_t v = base[i];
        int k = i - 1;
        for (; k >= ptr[t] && base[k] > v; k--) base[k + 1] = base[k];
        base[k + 1] = v;
    }
}

// the entries, a warp per row block: the near ones as doubles first, turned into integers in
// the unit of their row's largest once that is known (unless one is too large for that, or not
// finite: the self term 0/0 of a node where the parametrisation stops)
__global__ void k_rows_fill(int64_t nitem, RowItem *__restrict__ items, TreeLists T, int thr,
                            BoxGeo g, int P, int lchunks, const int32_t *__restrict__ cols,
                            const double2 *__restrict__ xi, const double2 *__restrict__ w,
                            const double *__restrict__ dself, double *__restrict__ rows,
                            int32_t *__restrict__ rexp)
{
    const int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (k >= nitem) return;
    const RowItem it = items[k];
    const int ng = (it.nrow + 3) / 4;
    const int ncol = it.ncol, nn = (ncol + 7) / 8;
    const int nend = 8 * nn + 2 * P * big_boxes(T, it.box, thr);
    double *t = rows + (int64_t)it.tile * 32 + lane;
    int top[kGroups];
#pragma unroll
    for (int q = 0; q < kGroups; q++) top[q] = 0;
    for (int c = 0; c < nn; c++, t += 32 * ng) {
        const int m = 8 * c + (lane & 7);
        const bool node = m < ncol;
        const int j = node ? cols[(int64_t)it.chunk * 8 + m] : it.row0;
        const double2 zj = xi[j], w1 = w[j], wj = make_double2(w1.x * (1.0 / LBF_PI), w1.y * (1.0 / LBF_PI));
#pragma unroll
        for (int q = 0; q < kGroups; q++) {
            if (q >= ng) break;
            const int r = 4 * q + (lane >> 3), i = it.row0 + r;
            double e = 0.0;
            if (r < it.nrow && node) {
                if (i == j) {
                    e = 2.0 * dself[i];
                } else {
                    const double2 zi = xi[i];
                    const double dr = zj.x - zi.x, di = zj.y - zi.y;
                    const double d2 = fma(dr, dr, di * di);
                    // coincident nodes add nothing; outside rcp_near's range, a division
                    const double id = abs(exp_field(d2) - 1023) < 120 ? fmm::rcp_near(d2)
                                      : d2 > 0.0                      ? 1.0 / d2
                                                                      : 0.0;
                    e = fma(wj.y, dr, -wj.x * di) * id;
                }
            }
            t[32 * q] = e;
            top[q] = max(top[q], exp_field(e));
        }
    }
    int most = 0;
#pragma unroll
    for (int q = 0; q < kGroups; q++) most = max(most, top[q]);
    const bool wide = __any_sync(0xffffffffu, most > kWideTop);
#pragma unroll
    for (int q = 0; q < kGroups; q++) {
        if (q >= ng) break;
        for (int o = 4; o > 0; o >>= 1) top[q] = max(top[q], __shfl_xor_sync(0xffffffffu, top[q], o));
        const int r = 4 * q + (lane >> 3);
        if ((lane & 7) == 0 && r < it.nrow) rexp[it.row0 + r] = top[q];
    }
    if (wide && lane == 0) items[k].leaf = ~it.leaf;
    t = rows + (int64_t)it.tile * 32 + lane;
    for (int c = 0; c < nn; c++, t += 32 * ng)
#pragma unroll
        for (int q = 0; q < kGroups; q++)
            if (q < ng && !wide) *(int2 *)&t[32 * q] = dot_word(t[32 * q], 0, top[q]);
    for (int c = nn; c < it.nchunk; c++, t += 32 * ng)
        for (int q = 0; q < ng; q++)
            if (8 * c + (lane & 7) >= nend || 4 * q + (lane >> 3) >= it.nrow) t[32 * q] = 0.0;
    const int b = it.box;
    // the M2P columns: powers of rho_i, a lane per row
    if (lane < it.nrow && nend > 8 * nn) {
        const double2 zi = xi[it.row0 + lane];
        int m = 8 * nn;
        for (int q = T.wptr[b]; q < T.wptr[b + 1]; q++) {
            const int s = T.widx[q];
            if (T.end[s] - T.begin[s] <= thr) continue;
            double sx, sy, sir;
            box_centre_ir(g, T.level[s], T.ix[s], T.iy[s], sx, sy, sir);
            const cx<double> rho = fmm::crcp(fmm::mk<double>((zi.x - sx) * sir, (zi.y - sy) * sir));
            const double f = sir * (-1.0 / LBF_PI);
            cx<double> p{rho.x * f, rho.y * f};
            for (int l = 0; l < P; l++, m += 2) {
                double *e = rows + ((int64_t)it.tile + (int64_t)(lane >> 2)) * 32 + (lane & 3) * 8;
                e[(int64_t)(m >> 3) * ng * 32 + (m & 7)] = p.y;
                e[(int64_t)((m + 1) >> 3) * ng * 32 + ((m + 1) & 7)] = p.x;
                p = cmul(p, rho);
            }
        }
    }
    // the local expansion's columns: powers of u_i, times 2^-(l/2) below 1/2, a lane per row
    double cxd, cyd, r;
    box_centre(g, T.level[b], T.ix[b], T.iy[b], cxd, cyd, r);
    const double ir = 1.0 / r;
    const bool on = lane < it.nrow;
    double2 z = xi[on ? it.row0 + lane : it.row0];
    const cx<double> u{(z.x - cxd) * ir, (z.y - cyd) * ir};
    cx<double> p{on ? -1.0 / LBF_PI : 0.0, 0.0};
    double *base = rows + ((int64_t)it.tile + (int64_t)it.nchunk * ng) * 32;
    if (lane < 4 * ng)
        for (int l = 0; l < 4 * lchunks; l++) {
            // times (b_l.x, b_l.y)
            const int2 ey = dot_word(p.y, -(l >> 1), kLocalTop), ex = dot_word(p.x, -(l >> 1), kLocalTop);
            *(int4 *)(base + ((int64_t)(l >> 2) * ng + (lane >> 2)) * 32 + (lane & 3) * 8 + 2 * (l & 3)) =
                make_int4(ey.x, ey.y, ex.x, ex.y);
            p = cmul(p, u);
        }
}

// ---- per application -----------------------------------------------------------------

__device__ __forceinline__ double local_real(const cx<double> *loc, int64_t at)
{
    return ((const double *)loc)[at];
}
__device__ __forceinline__ double local_real(const cx<df64> *loc, int64_t at)
{
    const float2 v = ((const float2 *)loc)[at];
    return (double)v.x + (double)v.y;
}

// Add the eight lanes of a row over G groups: at each step a lane keeps one half of its groups
// and sends the other half to its partner; once one is left, plain sums.  Returns the lane's
// group (G: another lane has this row).
template <int G, class F> __device__ __forceinline__ int fold_rows(int lane, F add)
{
    int grp = 0;
#pragma unroll
    for (int bit = 4, h = G / 2; bit > 0; bit >>= 1, h >>= 1) {
        const bool up = (lane & bit) != 0;
        if (h >= 1) {
#pragma unroll
            for (int q = 0; q < (h >= 1 ? h : 1); q++) add(q, q + h, up, bit);
            grp += up ? h : 0;
        } else {
            add(0, 0, up, bit);
            if (up) grp = G;
        }
    }
    return grp;
}
// the largest exponent field of a leaf's b_l 2^(l/2); bad: one is not finite
template <typename R>
__device__ __forceinline__ int local_top(const cx<R> *loc, int64_t lb, int P, int lane, bool &bad)
{
    int top = 0;
    bad = false;
    for (int m = lane; m < 2 * P; m += 32) {
        const int E = exp_field(local_real(loc, lb + m));
        bad |= E == 0x7ff;
        if (E) top = max(top, E + (m >> 2));
    }
    bad = __any_sync(0xffffffffu, bad);
    return __reduce_max_sync(0xffffffffu, top);
}

// acc += the n chunks of x (eight columns each, zeros up to a multiple of four) times their
// tiles of NG row groups; the tiles of kRun chunks are all asked for before the first is used
template <int NG>
__device__ __forceinline__ void dot_chunks(const double *__restrict__ t, const int2 *x, int n, int lane,
                                           Dot *acc)
{
    for (int k = 0; k < n; k += kRun, x += 8 * kRun) {
        prefetch_tiles(t - lane + 32 * NG * (k + kAhead), NG * min(kRun, n - k - kAhead), lane);
        int2 e[kRun * NG];
#pragma unroll
        for (int h = 0; h < kRun; h++) {
            const double *th = t + 32 * NG * min(k + h, n - 1);
#pragma unroll
            for (int q = 0; q < NG; q++) e[h * NG + q] = *(const int2 *)&th[32 * q];
        }
#pragma unroll
        for (int h = 0; h < kRun; h++) {
            const int2 xk = x[8 * h];
#pragma unroll
            for (int q = 0; q < NG; q++) dot_add(acc[q], e[h * NG + q], xk);
        }
    }
}

// The sum of a lane's row over the chunks w, w + step, .. of n of double entries whose columns are
// nodes.  Not inlined: few blocks have any, and beside the integer loops its sums cost them
// registers (rows of 407 ragged islands 143 us inlined, 133 so; the multipoles' loop, which many
// blocks enter, 152 and 133 the other way round).
template <int G>
__device__ __noinline__ double wide_rows(const double *__restrict__ t, const int32_t *__restrict__ cl,
                                         int ncol, int w, int step, int n, int ng,
                                         const double *__restrict__ sigma, int lane)
{
    double d[G];
#pragma unroll
    for (int q = 0; q < G; q++) d[q] = 0.0;
    t += (int64_t)32 * ng * w;
    for (int k = w; k < n; k += step, t += 32 * step * ng) {
        const int m = 8 * k + (lane & 7);
        const double x = m < ncol ? sigma[cl[m]] : 0.0;
#pragma unroll
        for (int q = 0; q < G; q++)
            if (q < ng) d[q] = fma(t[32 * q], x, d[q]);
    }
    fold_rows<G>(lane, [&](int a, int b, bool up, int bit) {
        const double keep = up ? d[b] : d[a], send = up ? d[a] : d[b];
        d[a] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
    });
    return d[0];
}

// The values of n column chunks from chunk k on (near nodes, or far: the local expansion's) in xs,
// zeros up to a multiple of four chunks, as they are (each lane's its own); the lane's largest
// exponent field, kBadExp where one is not finite
template <typename R>
__device__ __forceinline__ int run_values(const RowItem &it, const int32_t *__restrict__ cl,
                                          const double *__restrict__ sigma, const cx<R> *__restrict__ loc,
                                          int P, bool far, int k, int n, int2 *xs, int lane)
{
    const int64_t lb = (int64_t)it.box * 2 * P;
    const int off = 8 * (far ? it.nchunk : 0), end = min(far ? off + 2 * P : it.ncol, 8 * (k + n));
    const int m1 = 8 * (k + (n + 3) / 4 * 4);
    int top = 0;
#pragma unroll 2
    for (int m = 8 * k + lane; m < m1; m += 32) {
        double v = 0.0;
        if (m < end) v = far ? local_real(loc, lb + m - off) : sigma[cl[m]];
        const int E = exp_field(v);
        if (E) top = max(top, E == 0x7ff ? kBadExp : E + (far ? (m - off) >> 2 : 0));
        xs[m - 8 * k] = make_int2(__double2loint(v), __double2hiint(v));
    }
    return top;
}
// and the values as words in the unit of top (of the local expansion from its chunk k on)
__device__ __forceinline__ void run_words(bool far, int k, int n, int top, int2 *xs, int lane)
{
#pragma unroll 2
    for (int m = lane; m < 8 * ((n + 3) / 4 * 4); m += 32) {
        const int2 b = xs[m];
        xs[m] = dot_word(__hiloint2double(b.y, b.x), far ? (8 * k + m) >> 2 : 0, top);
    }
}
// the lane's row's sum over n integer chunks at t
template <int G>
__device__ __forceinline__ Dot run_dot(const double *__restrict__ t, const int2 *xs, int n, int ng, int lane)
{
    Dot acc[G];
#pragma unroll
    for (int q = 0; q < G; q++) acc[q] = Dot{0, 0};
#define LBF_DOT(NG) dot_chunks<(NG <= G ? NG : G)>(t, xs + (lane & 7), n, lane, acc)
    if (G <= 2) {
        if (ng == 1) LBF_DOT(1);
        else LBF_DOT(2);
    } else {
        LBF_GROUPS(ng, LBF_DOT)
    }
#undef LBF_DOT
    fold_rows<G>(lane, [&](int a, int b, bool up, int bit) { acc[a] = dot_meet(acc[a], acc[b], up, bit); });
    return acc[0];
}
// its sum over the multipole chunks w, w + step, .. of W boxes (few, and in units of their own), t at
// the first
template <int G, typename R>
__device__ __forceinline__ double far_chunks(const double *__restrict__ t, const RowItem &it,
                                             const int32_t *__restrict__ cl, const cx<R> *__restrict__ mp,
                                             int w, int step, int ng, int lane)
{
    double d[G];
#pragma unroll
    for (int q = 0; q < G; q++) d[q] = 0.0;
    t += (int64_t)32 * ng * w;
    for (int c = (it.ncol + 7) / 8 + w; c < it.nchunk; c += step, t += 32 * step * ng) {
        const int j = cl[8 * c + (lane & 7)];
        const double x = j < 0 ? local_real(mp, -1 - j) : 0.0;
#pragma unroll
        for (int q = 0; q < G; q++)
            if (q < ng) d[q] = fma(t[32 * q], x, d[q]);
    }
    fold_rows<G>(lane, [&](int a, int b, bool up, int bit) {
        const double keep = up ? d[b] : d[a], send = up ? d[a] : d[b];
        d[a] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
    });
    return d[0];
}
__device__ __forceinline__ double run_double(const Dot &d, int top, int unit)
{
    return top >= kBadExp ? __longlong_as_double(0x7ff8000000000000ll) : dot_double(d, top + unit);
}

// The sum of a lane's row of a block of at most G row groups over its columns, by one warp: near
// chunks, multipole chunks, then the local expansion's.  Near nodes are taken in runs of up to
// kDotChunks chunks, in units of the run's largest density and the row's largest entry, the local
// expansion in that of its largest b_l 2^(l/2).  (Blocks that may be shared add four sums of
// double chunks, as shared_rows does.)
template <int G, typename R>
__device__ __forceinline__ double block_rows(const RowItem &it, const double *__restrict__ rows,
                                             const int32_t *__restrict__ rexp,
                                             const int32_t *__restrict__ cols,
                                             const double *__restrict__ sigma,
                                             const cx<R> *__restrict__ loc,
                                             const cx<R> *__restrict__ mp, int P, int lchunks,
                                             int2 *xs, int lane, int row)
{
    constexpr int kStep = G == kGroupsSmall ? 4 : 1;
    const int ng = (it.nrow + 3) / 4;
    const double *t = rows + (int64_t)it.tile * 32 + lane;
    const int32_t *cl = cols + (int64_t)it.chunk * 8;
    const int nn = (it.ncol + 7) / 8, nk = it.nchunk + lchunks;
    prefetch_tiles(t - lane, ng * min(nk, kAhead), lane);
    double s = 0.0;
    int k = 0;
    if (it.leaf < 0) {  // near entries kept as doubles
        s = wide_rows<G>(t, cl, it.ncol, 0, kStep, nn, ng, sigma, lane);
#pragma unroll 1
        for (int w = 1; w < kStep; w++) s += wide_rows<G>(t, cl, it.ncol, w, kStep, nn, ng, sigma, lane);
        t += (int64_t)32 * nn * ng;
        k = nn;
    }
    while (k < nk) {
        if (k >= nn && k < it.nchunk) {
            double m = far_chunks<G>(t, it, cl, mp, 0, kStep, ng, lane);
#pragma unroll 1
            for (int w = 1; w < kStep; w++) m += far_chunks<G>(t, it, cl, mp, w, kStep, ng, lane);
            s += m;
            t += (int64_t)32 * (it.nchunk - k) * ng;
            k = it.nchunk;
            continue;
        }
        const bool far = k >= nn;
        const int n = min((far ? nk : nn) - k, kDotChunks);
        if (k > 0) prefetch_tiles(t - lane, ng * min(n, kAhead), lane);
        __syncwarp();
        const int top = __reduce_max_sync(0xffffffffu, run_values(it, cl, sigma, loc, P, far, k, n, xs, lane));
        run_words(far, k - it.nchunk, n, top, xs, lane);
        __syncwarp();
        const Dot d = run_dot<G>(t, xs, n, ng, lane);
        k += n;
        t += (int64_t)32 * n * ng;
        if (row < it.nrow) s += run_double(d, top, far ? -1129 : rexp[it.row0 + row] - 2150);
    }
    return s;
}

// What four warps share of a block
struct Shared {
    int top[2][4];
    Dot dot[2][4][32];
    double part[4][32];
};

// The same sums by the four warps of a thread block, the first warp's valid, and the same bits: the
// warps take quarters of every run, find its unit together and add their integer sums exactly
// before one is turned into a double; double chunks are four sums, of every fourth chunk, added in
// order.  The last run of near nodes and the local expansion go together (two barriers for most
// blocks).
template <typename R>
__device__ __forceinline__ double shared_rows(const RowItem &it, const double *__restrict__ rows,
                                              const int32_t *__restrict__ rexp,
                                              const int32_t *__restrict__ cols,
                                              const double *__restrict__ sigma,
                                              const cx<R> *__restrict__ loc,
                                              const cx<R> *__restrict__ mp, int P, int lchunks,
                                              int2 *xs, Shared &sh, int wid, int lane, int row)
{
    constexpr int G = kGroupsSmall;
    const int ng = (it.nrow + 3) / 4;
    const double *tiles = rows + (int64_t)it.tile * 32 + lane;
    const int32_t *cl = cols + (int64_t)it.chunk * 8;
    const int nn = (it.ncol + 7) / 8;
    auto add_parts = [&](double mine) {
        sh.part[wid][lane] = mine;
        __syncthreads();
        const double s = ((sh.part[0][lane] + sh.part[1][lane]) + sh.part[2][lane]) + sh.part[3][lane];
        __syncthreads();
        return s;
    };
    auto add_dots = [&](int i) {
        Dot d = sh.dot[i][0][lane];
#pragma unroll
        for (int w = 1; w < 4; w++) {
            d.h += sh.dot[i][w][lane].h;
            d.m += sh.dot[i][w][lane].m;
        }
        return d;
    };
    const int re = row < it.nrow ? rexp[it.row0 + row] : 0;  // (not at the end, where nothing hides the load)
    double s = 0.0, local = 0.0;
    int k = 0;
    if (it.leaf < 0) {
        s = add_parts(wide_rows<G>(tiles, cl, it.ncol, wid, 4, nn, ng, sigma, lane));
        k = nn;
    }
    const int l0 = it.nchunk + lchunks * wid / 4, ln = it.nchunk + lchunks * (wid + 1) / 4 - l0;
    const double *tl = tiles + (int64_t)32 * ng * l0;
    prefetch_tiles(tl - lane, ng * ln, lane);
    for (bool last = false; !last;) {
        const int n = min(nn - k, kDotChunks);
        const int c0 = k + n * wid / 4, cn = k + n * (wid + 1) / 4 - c0;
        const double *t = tiles + (int64_t)32 * ng * c0;
        int2 *xl = xs + 8 * ((cn + 3) / 4 * 4);
        k += n;
        last = k >= nn;
        prefetch_tiles(t - lane, ng * min(cn, kAhead), lane);
        __syncwarp();
        int top = __reduce_max_sync(0xffffffffu, run_values(it, cl, sigma, loc, P, false, c0, cn, xs, lane));
        int topl = last ? __reduce_max_sync(0xffffffffu, run_values(it, cl, sigma, loc, P, true, l0, ln, xl, lane)) : 0;
        if (lane == 0) {
            sh.top[0][wid] = top;
            sh.top[1][wid] = topl;
        }
        __syncthreads();
        top = max(max(sh.top[0][0], sh.top[0][1]), max(sh.top[0][2], sh.top[0][3]));
        topl = max(max(sh.top[1][0], sh.top[1][1]), max(sh.top[1][2], sh.top[1][3]));
        run_words(false, 0, cn, top, xs, lane);
        if (last) run_words(true, l0 - it.nchunk, ln, topl, xl, lane);
        __syncwarp();
        sh.dot[0][wid][lane] = run_dot<G>(t, xs, cn, ng, lane);
        if (last) sh.dot[1][wid][lane] = run_dot<G>(tl, xl, ln, ng, lane);
        __syncthreads();
        if (wid == 0 && row < it.nrow) {
            if (n > 0) s += run_double(add_dots(0), top, re - 2150);
            if (last) local = run_double(add_dots(1), topl, -1129);
        }
    }
    if (nn < it.nchunk)
        s += add_parts(far_chunks<G>(tiles + (int64_t)32 * ng * nn, it, cl, mp, wid, 4, ng, lane));
    return s + local;
}

// v of a block's rows: a warp per block of at most G row groups, or (SPLIT) the four warps of a
// thread block
template <typename R, int G, bool SPLIT>
__global__ void __launch_bounds__(128, kRowBlocks)
k_rows_apply(int64_t nitem, const RowItem *__restrict__ items, const double *__restrict__ rows,
             const int32_t *__restrict__ rexp, const int32_t *__restrict__ cols,
             const double *__restrict__ sigma,
             const cx<R> *__restrict__ loc, const cx<R> *__restrict__ mp, int P, int lchunks,
             const double *__restrict__ bsig, double *__restrict__ v, const int *gate, int64_t slab)
{
    lbf_rhs(slab, sigma, loc, mp, bsig, v, gate);
    if (fmm::gate_closed(gate)) return;
    __shared__ int2 xs[4][8 * (SPLIT ? kDotChunks / 4 + 16 : kDotChunks)];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t k = SPLIT ? (int64_t)blockIdx.x : blockIdx.x * (int64_t)(blockDim.x >> 5) + wid;
    if (k >= nitem) return;
    const int4 i0 = ((const int4 *)items)[2 * k], i1 = ((const int4 *)items)[2 * k + 1];
    const RowItem it{i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
    const int grp = fold_rows<G>(lane, [](int, int, bool, int) {});
    const int row = 4 * grp + (lane >> 3) < it.nrow ? 4 * grp + (lane >> 3) : it.nrow;
    const double beta = SPLIT ? *bsig : 0.0;
    double s;
    if constexpr (SPLIT) {
        __shared__ Shared sh;
        s = shared_rows(it, rows, rexp, cols, sigma, loc, mp, P, lchunks, xs[wid], sh, wid, lane, row);
    } else {
        s = block_rows<G>(it, rows, rexp, cols, sigma, loc, mp, P, lchunks, xs[wid], lane, row);
    }
    if ((!SPLIT || wid == 0) && row < it.nrow) v[it.row0 + row] = s + 2.0 * (SPLIT ? beta : *bsig);
}

// a[h] += the tiles of chunk h (of n, at most 4) times the rows' values
template <int NG>
__device__ __forceinline__ void dot_rows(const double *__restrict__ t, const int2 *x, int n, Dot *a)
{
#pragma unroll
    for (int h = 0; h < 4; h++) {
        const double *th = t + 32 * NG * min(h, n - 1);  // (beyond n: a sum nobody takes)
#pragma unroll
        for (int q = 0; q < NG; q++) dot_add(a[h], *(const int2 *)&th[32 * q], x[q]);
    }
}

// z = G^T tau over each leaf's columns, thread blocks of four warps per leaf, a part of the
// columns a warp (no sums between warps; a warp per leaf left the leaf with the most
// columns, 1500 of a mean of 200, running alone: 582 us at 131,072 nodes).  Four chunks at a
// time: a lane sums its rows' parts of a column of each, and the four lanes of a column are
// added in 3 additions.
__global__ void __launch_bounds__(128)
k_rows_t(const int32_t *__restrict__ block0, const RowItem *__restrict__ items,
         const double *__restrict__ rows, const int32_t *__restrict__ rexp,
         const double *__restrict__ tau, double *__restrict__ z, const int *gate)
{
    if (fmm::gate_closed(gate)) return;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t t = blockIdx.x;
    const int b0 = block0[t], b1 = block0[t + 1];
    const bool u = (lane & 16) != 0, w = (lane & 8) != 0;
    for (int k = b0; k < b1; k++) {
        const RowItem it = items[k];
        const int ng = (it.nrow + 3) / 4, nk = (it.ncol + 7) / 8;
        const int nw = 4 * gridDim.y, iw = 4 * blockIdx.y + wid;
        const int k0 = (int)((int64_t)nk * iw / nw), k1 = (int)((int64_t)nk * (iw + 1) / nw);
        if (k0 == k1) continue;
        // tau_r in the unit of its row's entries, as an integer in that of the block's largest,
        // a lane a row; then the rows of each lane's sums
        const double tr = lane < it.nrow ? tau[it.row0 + lane] : 0.0;
        if (it.leaf < 0) {  // near entries kept as doubles
            const double *tl = rows + ((int64_t)it.tile + (int64_t)k0 * ng) * 32 + lane;
            for (int c = k0; c < k1; c++, tl += 32 * ng) {
                double s = 0.0;
                for (int q = 0; q < ng; q++)
                    s = fma(tl[32 * q], __shfl_sync(0xffffffffu, tr, 4 * q + (lane >> 3)), s);
                s += __shfl_xor_sync(0xffffffffu, s, 8);
                s += __shfl_xor_sync(0xffffffffu, s, 16);
                double *o = z + ((int64_t)it.chunk + c) * 8 + lane;
                if (lane < 8) *o = k == b0 ? s : *o + s;
            }
            __syncwarp();  // (another lane may add to these columns in the next block)
            continue;
        }
        const int re = lane < it.nrow ? rexp[it.row0 + lane] : 0, E = exp_field(tr);
        const bool bad = __any_sync(0xffffffffu, E == 0x7ff);
        const int top = __reduce_max_sync(0xffffffffu, E ? E + re : 0);
        const int2 x = dot_word(tr, re, top);
        int2 tv[kGroups];
#pragma unroll
        for (int q = 0; q < kGroups; q++) tv[q] = shfl_word(x, 4 * q + (lane >> 3));
        const double *tl = rows + ((int64_t)it.tile + (int64_t)k0 * ng) * 32 + lane;
        prefetch_tiles(tl - lane, ng * min(k1 - k0, 2 * kAhead), lane);
        for (int c = k0; c < k1; c += 4, tl += 128 * ng) {
            prefetch_tiles(tl - lane + (int64_t)64 * kAhead * ng, ng * min(4, k1 - c - 2 * kAhead), lane);
            Dot a[4];
#pragma unroll
            for (int h = 0; h < 4; h++) a[h] = Dot{0, 0};
#define LBF_DOT(NG) dot_rows<NG>(tl, tv, k1 - c, a)
            LBF_GROUPS(ng, LBF_DOT)
#undef LBF_DOT
            const Dot d = dot_meet(dot_meet(a[0], a[2], u, 16), dot_meet(a[1], a[3], u, 16), w, 8);
            const int h = (u ? 2 : 0) + (w ? 1 : 0);  // the chunk this lane's sum belongs to
            if (c + h < k1) {
                double *o = z + ((int64_t)it.chunk + c + h) * 8 + (lane & 7);
                const double s = bad ? __longlong_as_double(0x7ff8000000000000ll) : dot_double(d, top - 2150);
                *o = k == b0 ? s : *o + s;
            }
        }
        __syncwarp();
    }
}

// v_i = Im(w_i Phi_far)/pi + 2 beta_i sum tau + the node's entries of the z vectors, a warp
// per row block
template <typename R>
__global__ void __launch_bounds__(128)
k_rows_t_out(int64_t nitem, const RowItem *__restrict__ items, const double *__restrict__ rows,
             const int32_t *__restrict__ cols, const double *__restrict__ z,
             const int32_t *__restrict__ rptr, const int32_t *__restrict__ rbase,
             const int32_t *__restrict__ begin, const cx<R> *__restrict__ loc,
             const cx<R> *__restrict__ mp, int P, int lchunks, const double2 *__restrict__ w,
             const double *__restrict__ beta, const double *__restrict__ bsig,
             double *__restrict__ v, const int *gate)
{
    if (fmm::gate_closed(gate)) return;
    const int64_t k = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (k >= nitem) return;
    const RowItem it = items[k];
    const int ng = (it.nrow + 3) / 4;
    // columns 2 l and 2 l + 1 hold -(1/pi) (Im, Re) of a power, to be met by (x, y) of the
    // coefficient for the imaginary part of the sum and by (-y, x) for the real part
    const int nn = (it.ncol + 7) / 8, par = lane & 1;
    const double *t = rows + ((int64_t)it.tile + (int64_t)nn * ng) * 32 + lane;
    const int64_t lb = (int64_t)it.box * 2 * P;
    double fi = 0.0, fr = 0.0;
    if (nn < it.nchunk) {
        double ai[kGroups], ar[kGroups];
#pragma unroll
        for (int q = 0; q < kGroups; q++) ai[q] = ar[q] = 0.0;
        for (int c = nn; c < it.nchunk; c++, t += 32 * ng) {
            const int j = cols[(int64_t)it.chunk * 8 + 8 * c + (lane & 7)];
            double si = 0.0, sr = 0.0;
            if (j < 0) {
                const int e = -1 - j;
                si = local_real(mp, e);
                sr = (e & 1) ? local_real(mp, e - 1) : -local_real(mp, e + 1);
            }
#pragma unroll
            for (int q = 0; q < kGroups; q++)
                if (q < ng) {
                    const double e = t[32 * q];
                    ai[q] = fma(e, si, ai[q]);
                    ar[q] = fma(e, sr, ar[q]);
                }
        }
        fold_rows<kGroups>(lane, [&](int a, int b, bool up, int bit) {
            const double ki = up ? ai[b] : ai[a], sdi = up ? ai[a] : ai[b];
            const double kr = up ? ar[b] : ar[a], sdr = up ? ar[a] : ar[b];
            ai[a] = ki + __shfl_xor_sync(0xffffffffu, sdi, bit);
            ar[a] = kr + __shfl_xor_sync(0xffffffffu, sdr, bit);
        });
        fi = ai[0];
        fr = ar[0];
    }
    // the local expansion, in units of its largest b_l 2^(l/2)
    bool bad;
    const int top = local_top(loc, lb, P, lane, bad);
    Dot di[kGroups], dr[kGroups];
#pragma unroll
    for (int q = 0; q < kGroups; q++) di[q] = dr[q] = Dot{0, 0};
    for (int c = 0; c < lchunks; c++, t += 32 * ng) {
        const int m = 8 * c + (lane & 7);
        const int2 xi = m < 2 * P ? dot_word(local_real(loc, lb + m), m >> 2, top) : make_int2(0, 0);
        int2 xr = make_int2(__shfl_xor_sync(0xffffffffu, xi.x, 1), __shfl_xor_sync(0xffffffffu, xi.y, 1));
        if (!par) xr = make_int2(-xr.x, -xr.y);
#pragma unroll
        for (int q = 0; q < kGroups; q++)
            if (q < ng) {
                const int2 e = *(const int2 *)&t[32 * q];
                dot_add(di[q], e, xi);
                dot_add(dr[q], e, xr);
            }
    }
    const int grp = fold_rows<kGroups>(lane, [&](int a, int b, bool up, int bit) {
        di[a] = dot_meet(di[a], di[b], up, bit);
        dr[a] = dot_meet(dr[a], dr[b], up, bit);
    });
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    fi += bad ? nan : dot_double(di[0], top - 1129);
    fr += bad ? nan : dot_double(dr[0], top - 1129);
    const int row = 4 * grp + (lane >> 3);
    if (row >= it.nrow) return;
    const int i = it.row0 + row, at = i - begin[it.box], leaf = it.leaf < 0 ? ~it.leaf : it.leaf;
    double s = 0.0;
    for (int e = rptr[leaf]; e < rptr[leaf + 1]; e++) s += z[(int64_t)rbase[e] + at];
    const double2 ww = w[i];
    v[i] = s - fma(ww.x, fi, ww.y * fr) + 2.0 * (beta[i] * *bsig);
}

// out_i = x_i + v_i + s (E y)_i (v nullable): the multiplier potential's local expansions loc
// (P terms) through the stored columns, a warp per row block, Re(b_l u^l) as -pi times column
// 2 l against -Im b_l and column 2 l + 1 against Re b_l; then the node's direct centres
// (partial), the centres summed directly everywhere and the constants.
// Bound by the columns' bytes: 1.9 ms at 16.8 million nodes (10.2 GB at 5.3 TB/s), 4.2 as a Horner chain a node
// (four double multiply-adds a term).
__global__ void __launch_bounds__(128, 4)
k_rows_mp(int64_t nitem, const RowItem *__restrict__ items, const double *__restrict__ rows, int P,
          const cx<double> *__restrict__ loc, const double2 *__restrict__ xi,
          const int32_t *__restrict__ glob, int nglob, const double2 *__restrict__ xc,
          const double *__restrict__ y, const double *__restrict__ ell, const double *__restrict__ sums,
          const double *__restrict__ x, const double *__restrict__ v, double sc, double *__restrict__ out,
          const int *gate, const int32_t *__restrict__ nodebase, const double *__restrict__ partial,
          int64_t slab)
{
    lbf_rhs(slab, loc, y, sums, x, v, out, gate, partial);
    if (fmm::gate_closed(gate)) return;
    __shared__ int2 xs[4][64];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t k = blockIdx.x * (int64_t)(blockDim.x >> 5) + wid;
    if (k >= nitem) return;
    const RowItem it = items[k];
    const int ng = (it.nrow + 3) / 4, n = (2 * P + 7) / 8;
    const double *t = rows + ((int64_t)it.tile + (int64_t)it.nchunk * ng) * 32 + lane;
    prefetch_tiles(t - lane, ng * n, lane);
    const int64_t lb = (int64_t)it.box * 2 * P;
    bool bad;
    const int top = local_top(loc, lb, P, lane, bad);
    for (int m = lane; m < 64; m += 32) {
        double b = 0.0;
        if (m < 2 * P) b = (m & 1) ? local_real(loc, lb + m - 1) : -local_real(loc, lb + m + 1);
        xs[wid][m] = dot_word(b, m >> 2, top);
    }
    __syncwarp();
    Dot acc[kGroups];
#pragma unroll
    for (int q = 0; q < kGroups; q++) acc[q] = Dot{0, 0};
#define LBF_DOT(NG) dot_chunks<NG>(t, xs[wid] + (lane & 7), n, lane, acc)
    LBF_GROUPS(ng, LBF_DOT)
#undef LBF_DOT
    const int grp = fold_rows<kGroups>(lane, [&](int a, int b, bool up, int bit) { acc[a] = dot_meet(acc[a], acc[b], up, bit); });
    const int row = 4 * grp + (lane >> 3);
    if (row >= it.nrow) return;
    const int i = it.row0 + row;
    double lsum = bad ? __longlong_as_double(0x7ff8000000000000ll) : -LBF_PI * dot_double(acc[0], top - 1129);
    for (int q = nodebase[i]; q < nodebase[i + 1]; q++) lsum += partial[q];
    if (nglob) {
        const double2 zi = xi[i];
        for (int q = 0; q < nglob; q++) {
            const int m = glob[q];
            const double ex = zi.x - xc[m].x, ey = zi.y - xc[m].y;
            lsum += y[m] * 0.5 * log(ex * ex + ey * ey);
        }
    }
    const double phi = ((ell[i] - LBF_LN2) * sums[0] + sums[1] - 2.0 * lsum) * (1.0 / (2.0 * LBF_PI));
    out[i] = x[i] + (v ? v[i] : 0.0) + sc * phi;
}

TreeLists lists_of(const Tree &T)
{
    return TreeLists{T.level, T.ix,    T.iy,    T.parent, T.begin, T.end,
                     T.u_ptr, T.u_idx, T.w_ptr, T.w_idx,  T.xlist, T.nx};
}

BoxGeo geo_of(const Tree &T)
{
    return BoxGeo{T.xmin, T.ymin, T.L, (float)(1.0 / T.L), df64(1.0 / T.L), 1.0 / T.L};
}

int local_chunks(int P) { return (2 * P + 7) / 8; }

}  // namespace

// Room for the rows after everything else in the workspace: about 4 leaf_size near columns
// a node (measured 125 + 56 at leaf 48 on star caps), the local columns and the padding (more in a small system, whose larger W boxes are pairs),
// while that is at most 64 GB (about 25 million nodes at the default order and leaf
// size); a plan without room for them, or whose tree needs more, forms the pairs on the fly.
void lbf_rows_layout(lbf_plan *pl, int64_t N, const lbf_options &o, int64_t cap)
{
    pl->rows = nullptr;
    if (o.matvec != LBF_MATVEC_FMM || !(pl->parts & LBF_PART_ROWS)) return;
    // local columns for the density's expansions and, where E y is one, the multipliers'
    const int Pl = std::max(o.p + 1, pl->bd.p2l_exp_cap ? pl->bd.Pe : 0);
    pl->rows_lch = local_chunks(Pl);
    const int64_t cols = (N <= 1 << 18 ? 10 : 4) * (int64_t)o.leaf_size + 2 * Pl + 48;
    // a chunk of columns serves every row group of its leaf (leaves hold about half of leaf_size)
    const int64_t tiles = (N * cols) / 32 + 4096;
    const int64_t chunks = tiles / std::max(1, o.leaf_size / 10) + 4096;
    if (tiles > (int64_t)250000000) return;
    Arena &A = pl->arena;
    const size_t off = A.off;
    const bool full = A.overflow, had_loc = pl->use_loc;
    if (!had_loc && pl->m2l_cap) {  // the passes over the stored parts
        lbf_loc_layout(pl, pl, A);
        pl->use_loc = true;
    }
    pl->rows_tiles = tiles;
    pl->rows_chunks = chunks;
    pl->rows_items_cap = N / 4 + cap;
    pl->rows_rev_cap = 12 * cap;
    pl->rows_items = A.get<RowItem>(pl->rows_items_cap);
    pl->rows_cols = A.get<int32_t>(8 * chunks);
    pl->rows_block0 = A.get<int32_t>(cap + 1);
    pl->rows_rptr = A.get<int32_t>(cap + 1);
    pl->rows_rbase = A.get<int32_t>(pl->rows_rev_cap);
    pl->rows_z = A.get<double>(8 * chunks);
    pl->rows_e = A.get<int32_t>(N);
    pl->bigx_cap = cap / 8 + 16;
    pl->bigx = A.get<int32_t>(pl->bigx_cap);
    pl->rows = A.get<double>(32 * tiles);
    if (A.overflow && !full) {  // a workspace of the size without rows
        A.off = off;
        A.overflow = false;
        pl->rows = nullptr;
        if (!had_loc) {
            pl->use_loc = false;
            pl->loc_X = nullptr;
            pl->loc_e = nullptr;
        }
    }
}

// leaf: room for the leaf of each node (plan time)
int lbf_rows_build(lbf_plan *pl, cudaStream_t s, int32_t *scratch, int64_t scratch_len,
                   int32_t *leaf)
{
    if (!pl->rows) return LBF_OK;
    Tree &T = pl->tree;
    const int64_t nl = T.nleaf;
    const int P = pl->P, lch = pl->rows_lch;
        // (in a small system W and X boxes of up to 512 nodes are pairs while there is room: their
    // few P2L and M2P are dependent steps that the whole application waits for; with boxes of up
    // to 2048 the longest rows hold it up instead, 85 against 22 us for the rows of 8192 nodes)
    const bool small = nl < kSmallLeaves;
    pl->rows_split = small ? 1 : 0;
    const int groups = small ? kGroupsSmall : kGroups;
    const TreeLists tl = lists_of(T);
    int32_t *chunks = scratch + 8, *tiles = chunks + nl + 1, *blocks = pl->rows_block0;
    int32_t *sc = tiles + nl + 1;
    const int64_t sc_len = scratch_len - 8 - 2 * (nl + 1);
    unsigned long long *total = (unsigned long long *)scratch;
    if (sc_len < nl / 1024 + 64 || T.nbox * 2 * P >= INT32_MAX) {
        pl->rows = nullptr;
        return LBF_OK;
    }
    int rc;
    int32_t nitem = 0;
    for (int large = small;; large = 0) {
        pl->rows_thr = large ? std::max(512, 4 * P) : 4 * P;
        LBF_CUDA(cudaMemsetAsync(scratch, 0, sizeof(int32_t) * (8 + 2 * (nl + 1)), s));
        LBF_CUDA(cudaMemsetAsync(blocks, 0, sizeof(int32_t) * (nl + 1), s));
        LBF_LAUNCH(k_rows_count, lbf_cdiv(nl, 128), 128, 0, s, nl, T.leaves, tl, pl->rows_thr, P, lch,
                   groups, chunks, blocks, tiles, total);
        LBF_CHECK_LAUNCH();
        if ((rc = lbf_scan_i32(blocks, blocks, nl + 1, sc, sc_len, s))) return rc;
        unsigned long long h[2];
        LBF_CUDA(cudaMemcpyAsync(h, total, sizeof(h), cudaMemcpyDeviceToHost, s));
        LBF_CUDA(cudaMemcpyAsync(&nitem, blocks + nl, sizeof(nitem), cudaMemcpyDeviceToHost, s));
        LBF_CUDA(cudaStreamSynchronize(s));
        if (h[0] <= (unsigned long long)pl->rows_tiles && h[1] <= (unsigned long long)pl->rows_chunks &&
            nitem <= pl->rows_items_cap)
            break;
        if (!large) {
            pl->rows = nullptr;
            return LBF_OK;
        }
    }
    LBF_CUDA(cudaMemsetAsync(pl->rows_rptr, 0, sizeof(int32_t) * (nl + 1), s));
    if ((rc = lbf_scan_i32(chunks, chunks, nl + 1, sc, sc_len, s))) return rc;
    if ((rc = lbf_scan_i32(tiles, tiles, nl + 1, sc, sc_len, s))) return rc;
    pl->rows_nitem = nitem;
    LBF_LAUNCH(k_rows_items, lbf_cdiv(nl, 128), 128, 0, s, nl, T.leaves, tl, pl->rows_thr, lch,
               groups, chunks, blocks, tiles, pl->rows_items, leaf);
    LBF_LAUNCH(k_rows_cols, lbf_cdiv(nl, 4), 128, 0, s, nl, T.leaves, tl, pl->rows_thr, P, chunks,
               pl->rows_cols);
    LBF_LAUNCH(k_rows_fill, lbf_cdiv((int64_t)nitem, 4), 128, 0, s, (int64_t)nitem, pl->rows_items, tl,
               pl->rows_thr, geo_of(T), P, lch, pl->rows_cols, pl->xi, pl->w, pl->dself, pl->rows, pl->rows_e);
    // the transposed rows' lists
    LBF_LAUNCH(k_rows_rev, lbf_cdiv(nl, 128), 128, 0, s, nl, T.leaves, tl, pl->rows_thr, chunks, leaf,
               pl->rows_rptr, (const int32_t *)nullptr, (int32_t *)nullptr);
    LBF_CHECK_LAUNCH();
    if ((rc = lbf_scan_i32(pl->rows_rptr, pl->rows_rptr, nl + 1, sc, sc_len, s))) return rc;
    int32_t nrev = 0;
    LBF_CUDA(cudaMemcpyAsync(&nrev, pl->rows_rptr + nl, sizeof(nrev), cudaMemcpyDeviceToHost, s));
    LBF_CUDA(cudaStreamSynchronize(s));
    if (nrev > pl->rows_rev_cap) {
        pl->rows_rptr = nullptr;  // transposed applications form their rows on the fly
        return LBF_OK;
    }
    LBF_CUDA(cudaMemsetAsync(tiles, 0, sizeof(int32_t) * nl, s));  // the lists' write positions
    LBF_LAUNCH(k_rows_rev, lbf_cdiv(nl, 128), 128, 0, s, nl, T.leaves, tl, pl->rows_thr, chunks, leaf,
               tiles, (const int32_t *)pl->rows_rptr, pl->rows_rbase);
    LBF_LAUNCH(k_rows_rev_sort, lbf_cdiv(nl, 128), 128, 0, s, nl, pl->rows_rptr, pl->rows_rbase);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

int lbf_rows_apply(lbf_plan *pl, const double *sigma, double *v, const int *gate, cudaStream_t s,
                   bool df)
{
    const int64_t n = pl->rows_nitem;
    const bool small = pl->rows_split != 0;
    const bool split = small && (pl->nrhs == 1 || n * pl->nrhs < kFullWarps * (int64_t)std::max(pl->nsm, 1));
    const dim3 grid = lbf_grid(pl, split ? n : lbf_cdiv(n, 4));
#define LBF_ROWS(R, G, SPLIT)                                                                      \
    LBF_LAUNCH_P(LBF_KERNEL_LEAF, (k_rows_apply<R, G, SPLIT>), grid, 128, 0, s, n, pl->rows_items, pl->rows, \
                 pl->rows_e, pl->rows_cols, sigma, (const cx<R> *)pl->local,                       \
                 (const cx<R> *)pl->mpole, pl->P, local_chunks(pl->P), pl->bsig, v, gate, pl->slab)
#define LBF_ROWS_OF(R)                                  \
    if (split) LBF_ROWS(R, kGroupsSmall, true);         \
    else if (small) LBF_ROWS(R, kGroupsSmall, false);   \
    else LBF_ROWS(R, kGroups, false)
    if (df) {
        LBF_ROWS_OF(df64);
    } else {
        LBF_ROWS_OF(double);
    }
#undef LBF_ROWS_OF
#undef LBF_ROWS
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

// out = x + v + sc E y from the multiplier potential's local expansions (B.loc, Pe terms)
int lbf_rows_mp(lbf_plan *pl, const double *y, const double *x, const double *v, double sc, double *out,
                const int *gate, cudaStream_t s)
{
    const Border &B = pl->bd;
    const int64_t n = pl->rows_nitem;
    LBF_LAUNCH_P(LBF_KERNEL_ESUM, k_rows_mp, lbf_grid(pl, lbf_cdiv(n, 4)), 128, 0, s, n, pl->rows_items,
                 pl->rows, B.Pe, (const cx<double> *)B.loc, pl->xi, B.glob, B.nglob_h, B.xc, y, B.ell,
                 B.sums, x, v, sc, out, gate, B.nodebase, B.partial, pl->slab);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

int lbf_rows_apply_t(lbf_plan *pl, const double *tau, double *v, const int *gate, cudaStream_t s,
                     bool df)
{
    const Tree &T = pl->tree;
    const int64_t n = pl->rows_nitem;
    LBF_LAUNCH_P(LBF_KERNEL_LEAF, k_rows_t, dim3((unsigned)T.nleaf, pl->rows_split ? 4 : 1), 128, 0, s, pl->rows_block0, pl->rows_items,
                 pl->rows, pl->rows_e, tau, pl->rows_z, gate);
    const int lch = local_chunks(pl->P);
    if (df)
        LBF_LAUNCH_P(LBF_KERNEL_LEAF, k_rows_t_out<df64>, lbf_cdiv(n, 4), 128, 0, s, n, pl->rows_items,
                     pl->rows, pl->rows_cols, pl->rows_z, pl->rows_rptr, pl->rows_rbase, T.begin,
                     (const cx<df64> *)pl->local, (const cx<df64> *)pl->mpole, pl->P, lch, pl->w,
                     pl->beta, pl->bsig, v, gate);
    else
        LBF_LAUNCH_P(LBF_KERNEL_LEAF, k_rows_t_out<double>, lbf_cdiv(n, 4), 128, 0, s, n,
                     pl->rows_items, pl->rows, pl->rows_cols, pl->rows_z, pl->rows_rptr,
                     pl->rows_rbase, T.begin, (const cx<double> *)pl->local,
                     (const cx<double> *)pl->mpole, pl->P, lch, pl->w, pl->beta, pl->bsig, v, gate);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}
