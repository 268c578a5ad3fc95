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
// Layout: a leaf's rows are cut into blocks of at most kGroups groups of four rows, its
// columns into chunks of eight; a tile is one group x one chunk, 32 doubles, row-major,
// so lane = 8 (row mod 4) + (column mod 8) and a warp's load is 256 contiguous bytes.  A
// block's tiles are stored chunk by chunk: the near nodes and the W multipoles' reals, then
// the 2 P reals of the local expansion.  Each lane holds one sum per group; eight lanes share a row, and a butterfly
// that halves the groups at each step adds them in 7 additions for 8 groups (lanes on
// rows alone would leave 19 % of the lanes idle at 26 nodes a leaf, lanes on columns
// alone would add 31 shuffled sums to 4 x 26 multiply-adds).
#include <algorithm>

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

// the column ranges of leaf b, in order: U(b), the small boxes of W(b), the X lists of
// b and its ancestors that are small.  f(first node, end)
struct TreeLists {
    const int32_t *level, *ix, *iy, *parent, *begin, *end, *uptr, *uidx, *wptr, *widx, *xlist, *nx;
};
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
        const long long cols = near_nodes(T, b, thr) + 2ll * P * big_boxes(T, b, thr);
        const long long ch = (cols + 7) / 8, g = (T.end[b] - T.begin[b] + 3) / 4;
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
                             int lchunks, int groups, const int32_t *__restrict__ chunk0,
                             const int32_t *__restrict__ block0, const int32_t *__restrict__ tile0,
                             RowItem *__restrict__ items)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= nleaf) return;
    const int b = leaves[t];
    const int n = T.end[b] - T.begin[b], g = (n + 3) / 4, nb = (g + groups - 1) / groups;
    const int ch = chunk0[t + 1] - chunk0[t];
    for (int k = 0; k < nb; k++) {
        const int g0 = (int)((long long)g * k / nb), g1 = (int)((long long)g * (k + 1) / nb);
        RowItem it;
        it.box = b;
        it.row0 = T.begin[b] + 4 * g0;
        it.nrow = min(n, 4 * g1) - 4 * g0;
        it.tile = tile0[t] + g0 * (ch + lchunks);
        it.chunk = chunk0[t];
        it.nchunk = ch;
        it.pad[0] = it.pad[1] = 0;
        items[block0[t] + k] = it;
    }
}

// each leaf's columns, a warp per leaf: node j, or -1 - m for the real m of the multipoles;
// the last chunk is filled up with the leaf's first node (zero entries)
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
    for (int q = T.wptr[b]; q < T.wptr[b + 1]; q++) {
        const int s = T.widx[q];
        if (T.end[s] - T.begin[s] <= thr) continue;
        for (int e = lane; e < 2 * P; e += 32) c[m + e] = -1 - (s * 2 * P + e);
        m += 2 * P;
    }
    if (m + lane < (m + 7) / 8 * 8) c[m + lane] = T.begin[b];
}

// the entries, a warp per row block
__global__ void k_rows_fill(int64_t nitem, const RowItem *__restrict__ items, TreeLists T, int thr,
                            BoxGeo g, int P, int lchunks, const int32_t *__restrict__ cols,
                            const double2 *__restrict__ xi, const double2 *__restrict__ w,
                            const double *__restrict__ dself, double *__restrict__ rows)
{
    const int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (k >= nitem) return;
    const RowItem it = items[k];
    const int ng = (it.nrow + 3) / 4;
    const int ncol = (int)near_nodes(T, it.box, thr);
    const int nend = ncol + 2 * P * big_boxes(T, it.box, thr);
    double *t = rows + (int64_t)it.tile * 32 + lane;
    for (int c = 0; c < it.nchunk; c++) {
        const int m = 8 * c + (lane & 7);
        const bool node = m < ncol;
        const int j = node ? cols[(int64_t)it.chunk * 8 + m] : it.row0;
        const double2 zj = xi[j], wj = w[j];
        for (int q = 0; q < ng; q++, t += 32) {
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
                    const double id = d2 > 0x1p-120 && d2 < 0x1p120 ? fmm::rcp_near(d2)
                                      : d2 > 0.0                    ? 1.0 / d2
                                                                    : 0.0;
                    e = fma(wj.y, dr, -wj.x * di) * id * (1.0 / LBF_PI);
                }
            }
            if (node || m >= nend || r >= it.nrow) *t = e;
        }
    }
    const int b = it.box;
    // the M2P columns: powers of rho_i, a lane per row
    if (lane < it.nrow && nend > ncol) {
        const double2 zi = xi[it.row0 + lane];
        int m = ncol;
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
    // the local expansion's columns: powers of u_i, a lane per row
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
            double2 e = make_double2(0.0, 0.0);
            if (l < P) e = make_double2(p.y, p.x);  // times (b_l.x, b_l.y)
            *(double2 *)(base + ((int64_t)(l >> 2) * ng + (lane >> 2)) * 32 + (lane & 3) * 8 +
                         2 * (l & 3)) = e;
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

// The sums of a block of NG row groups over its column chunks k0 .. k1 - 1 (near chunks,
// then the local expansion's); lane's result (after the butterfly) and its row.  The
// columns' values are fetched 32 at a time, a column a lane, one step ahead of their tiles,
// and handed to the row lanes by shuffles: the chain index -> density -> multiply-add is
// then two loads per 4 NG tiles (a fetch per chunk left a small system waiting on it).
template <int NG, typename R>
__device__ __forceinline__ double block_rows(const RowItem &it, const double *__restrict__ rows,
                                             const int32_t *__restrict__ cols,
                                             const double *__restrict__ sigma,
                                             const cx<R> *__restrict__ loc,
                                             const cx<R> *__restrict__ mp, int P, int k0, int k1,
                                             int lane, int &row)
{
    constexpr int NP = NG <= 1 ? 1 : NG <= 2 ? 2 : NG <= 4 ? 4 : 8;  // power of two >= NG
    double acc[NP];
#pragma unroll
    for (int q = 0; q < NP; q++) acc[q] = 0.0;
    const double *t = rows + ((int64_t)it.tile + (int64_t)k0 * NG) * 32 + lane;
    const int near = 8 * it.nchunk, end = 8 * k1;
    const int32_t *c = cols + (int64_t)it.chunk * 8;
    const int64_t lb = (int64_t)it.box * 2 * P;
    auto index = [&](int m) { return m < near && m < end ? c[m] : 0; };
    auto value = [&](int m, int j) {
        if (m < near) return j >= 0 ? sigma[j] : local_real(mp, -1 - j);
        return m < near + 2 * P ? local_real(loc, lb + m - near) : 0.0;
    };
    int m = 8 * k0 + lane;
    double s = m < end ? value(m, index(m)) : 0.0;
    int jn = index(m + 32);
    for (int k = k0; k < k1; k += 4) {
        const double sc = s;
        m += 32;
        s = m < end ? value(m, jn) : 0.0;
        jn = index(m + 32);
#pragma unroll
        for (int h = 0; h < 4; h++) {
            if (k + h < k1) {
                double e[NG];
#pragma unroll
                for (int q = 0; q < NG; q++) e[q] = t[32 * (h * NG + q)];
                const double sh = __shfl_sync(0xffffffffu, sc, 8 * h + (lane & 7));
#pragma unroll
                for (int q = 0; q < NG; q++) acc[q] = fma(e[q], sh, acc[q]);
            }
        }
        t += 32 * 4 * NG;
    }
    // add the eight lanes of a row: at each step a lane keeps one half of its groups and
    // sends the other half to its partner; once one is left, plain sums
    int grp = 0;
#pragma unroll
    for (int bit = 4, h = NP / 2; bit > 0; bit >>= 1, h >>= 1) {
        const bool up = (lane & bit) != 0;
        if (h >= 1) {
#pragma unroll
            for (int q = 0; q < (h >= 1 ? h : 1); q++) {
                const double keep = up ? acc[q + h] : acc[q], send = up ? acc[q] : acc[q + h];
                acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
            }
            grp += up ? h : 0;
        } else {
            acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], bit);
            if (up) grp = NG;  // another lane writes this row
        }
    }
    row = grp < NG ? 4 * grp + (lane >> 3) : it.nrow;
    return acc[0];
}

// v of a block's rows: a warp per block, or (split) the four warps of a thread block, each
// over a quarter of the columns, the quarters added in order.
template <typename R>
__global__ void __launch_bounds__(128)
k_rows_apply(int64_t nitem, const RowItem *__restrict__ items, const double *__restrict__ rows,
             const int32_t *__restrict__ cols, const double *__restrict__ sigma,
             const cx<R> *__restrict__ loc, const cx<R> *__restrict__ mp, int P, int lchunks,
             const double *__restrict__ bsig, double *__restrict__ v, const int *gate, int split,
             int64_t slab)
{
    lbf_rhs(slab, sigma, loc, mp, bsig, v, gate);
    if (fmm::gate_closed(gate)) return;
    __shared__ double part[4][32];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t k = split ? (int64_t)blockIdx.x : blockIdx.x * (int64_t)(blockDim.x >> 5) + wid;
    if (k >= nitem) return;
    const int4 i0 = ((const int4 *)items)[2 * k], i1 = ((const int4 *)items)[2 * k + 1];
    const RowItem it{i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, {0, 0}};
    const int nk = it.nchunk + lchunks;
    const int k0 = split ? nk * wid / 4 : 0, k1 = split ? nk * (wid + 1) / 4 : nk;
    int row;
    double s;
    switch ((it.nrow + 3) / 4) {
#define LBF_ROWS(NG) \
    case NG: s = block_rows<NG>(it, rows, cols, sigma, loc, mp, P, k0, k1, lane, row); break
        LBF_ROWS(1);
        LBF_ROWS(2);
        LBF_ROWS(3);
        LBF_ROWS(4);
        LBF_ROWS(5);
        LBF_ROWS(6);
        LBF_ROWS(7);
    default: s = block_rows<8>(it, rows, cols, sigma, loc, mp, P, k0, k1, lane, row); break;
#undef LBF_ROWS
    }
    if (split) {
        part[wid][lane] = s;
        __syncthreads();
        if (wid != 0) return;
        s = part[0][lane] + part[1][lane] + part[2][lane] + part[3][lane];
    }
    if (row < it.nrow) v[it.row0 + row] = s + 2.0 * *bsig;
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
    if (o.matvec != LBF_MATVEC_FMM) return;
    const int64_t cols = (N <= 1 << 18 ? 10 : 4) * (int64_t)o.leaf_size + 2 * (o.p + 1) + 48;
    // a chunk of columns serves every row group of its leaf (leaves hold about half of leaf_size)
    const int64_t tiles = (N * cols) / 32 + 4096;
    const int64_t chunks = tiles / std::max(1, o.leaf_size / 16) + 4096;
    if (tiles > (int64_t)250000000) return;
    Arena &A = pl->arena;
    const size_t off = A.off;
    const bool full = A.overflow;
    pl->rows_tiles = tiles;
    pl->rows_chunks = chunks;
    pl->rows_items_cap = N / 4 + cap;
    pl->rows_items = A.get<RowItem>(pl->rows_items_cap);
    pl->rows_cols = A.get<int32_t>(8 * chunks);
    pl->rows = A.get<double>(32 * tiles);
    if (A.overflow && !full) {  // a workspace of the size without rows
        A.off = off;
        A.overflow = false;
        pl->rows = nullptr;
    }
}

int lbf_rows_build(lbf_plan *pl, cudaStream_t s, int32_t *scratch, int64_t scratch_len)
{
    if (!pl->rows) return LBF_OK;
    Tree &T = pl->tree;
    const int64_t nl = T.nleaf;
    const int P = pl->P, lch = local_chunks(P);
        // (in a small system the few larger W boxes are pairs too: an M2P there is a chain of
    // P dependent steps that the whole launch waits for)
    const bool small = nl < kSmallLeaves;
    pl->rows_thr = small ? std::max(512, 4 * P) : 4 * P;
    pl->rows_split = small ? 1 : 0;
    const int groups = small ? kGroupsSmall : kGroups;
    const TreeLists tl = lists_of(T);
    int32_t *chunks = scratch + 8, *blocks = chunks + nl + 1, *tiles = blocks + nl + 1;
    int32_t *sc = tiles + nl + 1;
    const int64_t sc_len = scratch_len - 8 - 3 * (nl + 1);
    unsigned long long *total = (unsigned long long *)scratch;
    if (sc_len < nl / 1024 + 64 || T.nbox * 2 * P >= INT32_MAX) {
        pl->rows = nullptr;
        return LBF_OK;
    }
    LBF_CUDA(cudaMemsetAsync(scratch, 0, sizeof(int32_t) * (8 + 3 * (nl + 1)), s));
    LBF_LAUNCH(k_rows_count, lbf_cdiv(nl, 128), 128, 0, s, nl, T.leaves, tl, pl->rows_thr, P,
               lch, groups, chunks, blocks, tiles, total);
    LBF_CHECK_LAUNCH();
    int rc;
    if ((rc = lbf_scan_i32(blocks, blocks, nl + 1, sc, sc_len, s))) return rc;
    unsigned long long h[2];
    int32_t nitem = 0;
    LBF_CUDA(cudaMemcpyAsync(h, total, sizeof(h), cudaMemcpyDeviceToHost, s));
    LBF_CUDA(cudaMemcpyAsync(&nitem, blocks + nl, sizeof(nitem), cudaMemcpyDeviceToHost, s));
    LBF_CUDA(cudaStreamSynchronize(s));
    if (h[0] > (unsigned long long)pl->rows_tiles || h[1] > (unsigned long long)pl->rows_chunks ||
        nitem > pl->rows_items_cap) {
        pl->rows = nullptr;
        return LBF_OK;
    }
    if ((rc = lbf_scan_i32(chunks, chunks, nl + 1, sc, sc_len, s))) return rc;
    if ((rc = lbf_scan_i32(tiles, tiles, nl + 1, sc, sc_len, s))) return rc;
    pl->rows_nitem = nitem;
    LBF_LAUNCH(k_rows_items, lbf_cdiv(nl, 128), 128, 0, s, nl, T.leaves, tl, lch, groups, chunks,
               blocks, tiles, pl->rows_items);
    LBF_LAUNCH(k_rows_cols, lbf_cdiv(nl, 4), 128, 0, s, nl, T.leaves, tl, pl->rows_thr, P, chunks,
               pl->rows_cols);
    LBF_LAUNCH(k_rows_fill, lbf_cdiv((int64_t)nitem, 4), 128, 0, s, (int64_t)nitem, pl->rows_items, tl,
               pl->rows_thr, geo_of(T), P, lch, pl->rows_cols, pl->xi, pl->w, pl->dself, pl->rows);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

int lbf_rows_apply(lbf_plan *pl, const double *sigma, double *v, const int *gate, cudaStream_t s)
{
    const int64_t n = pl->rows_nitem;
    const dim3 grid = lbf_grid(pl, pl->rows_split ? n : lbf_cdiv(n, 4));
    if (pl->qdf)
        LBF_LAUNCH_P(LBF_KERNEL_LEAF, k_rows_apply<df64>, grid, 128, 0, s, n, pl->rows_items, pl->rows,
                     pl->rows_cols, sigma, (const cx<df64> *)pl->local, (const cx<df64> *)pl->mpole,
                     pl->P, local_chunks(pl->P), pl->bsig, v, gate, pl->rows_split, pl->slab);
    else
        LBF_LAUNCH_P(LBF_KERNEL_LEAF, k_rows_apply<double>, grid, 128, 0, s, n, pl->rows_items,
                     pl->rows, pl->rows_cols, sigma, (const cx<double> *)pl->local,
                     (const cx<double> *)pl->mpole, pl->P, local_chunks(pl->P), pl->bsig, v, gate, pl->rows_split, pl->slab);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}
