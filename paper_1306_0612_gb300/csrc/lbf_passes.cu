// The upward and downward passes of a double application on a plan whose leaf rows
// (lbf_rows.cu) and translations (lbf_m2l.cu) are stored, P <= 32:
//
//   k_up_rows   P2M from the rows' local columns (the powers u_i^l of the leaf's nodes are
//               there already), then M2M by the warp that completes a box's last child;
//   k_p2l_big   P2L of the few boxes whose X lists are not near columns;
//   k_l2l       each box's translations added up and its parent's expansion shifted to it,
//               in one launch: warps take the boxes in index order and wait (bounded) for
//               the parent, which a running warp took earlier; also the chain of the
//               multiplier potential's expansions.
//
// P2M: with the stored powers a node and coefficient take two multiply-adds a real where
// the recurrence took six double instructions and left the lanes past a leaf's last node
// idle (26 of 32 at 16.8 million nodes).  L2L: a warp a box, the two halves of a warp
// sharing each coefficient's sum, so a box's shift is (P + 1)/2 dependent steps where the
// half-warp form of k_down takes P + 1; and no shared-memory staging but the shift matrix
// and one expansion a warp, so an SM holds 64 warps.
//
// A small system is a chain of some ten to seventeen levels that nothing hides, and a warp
// issues a double instruction every 64 cycles: there a thread block of four warps, on the
// SM's four schedulers, takes a leaf or a box (k_up_small, k_l2l_small).  Four warps a box
// lower a level's shift from P + 1 dependent steps to 4.  Up and down at 8192 nodes 122 to
// 63 us and 75 to 46 us; at 7130 leaves an application 907 to 863 us, at 16,150 the two forms
// are equal, at 647,307 the block form takes 10.4 + 10.9 ms where the warp form takes
// 8.0 + 8.6 (of 10.5 + 28.7 with the passes of lbf_fmm_tpl.cuh).
#include <algorithm>

#include "lbf_fmm_tpl.cuh"

using fmm::BoxGeo;
using fmm::cx;
using fmm::mk;

namespace {

constexpr int64_t kSmallLeaves = 12000;
constexpr int kP2lSmem = 4 * 32 * 33 * 16;
constexpr int kGroups = 8;  // row groups of a block at most (lbf_rows.cu)

// P2M of leaf t by a warp, the chunks cbeg .. cend - 1 of eight reals: sum_i q_i u_i^l over the
// leaf's row blocks, four chunks at a time.  Column 2 l of a row holds -(1/pi) Im u^l, column 2 l + 1 -(1/pi) Re u^l:
// an even lane adds their parts of both reals of coefficient l, an odd lane likewise, and
// one exchange leaves the real part on the even lane, the imaginary part on the odd one.
__device__ __forceinline__ void leaf_p2m(int64_t t, int b, int P,
                                         const int32_t *__restrict__ block0,
                                         const RowItem *__restrict__ items,
                                         const double *__restrict__ rows,
                                         const double2 *__restrict__ q, double *__restrict__ a,
                                         int lane, int cbeg, int cend)
{
    const int k0 = block0[t], k1 = block0[t + 1];
    const bool odd = (lane & 1) != 0, u = (lane & 16) != 0, w = (lane & 8) != 0;
    for (int c = cbeg; c < cend; c += 4) {
        double re[4] = {0.0, 0.0, 0.0, 0.0}, im[4] = {0.0, 0.0, 0.0, 0.0};
        for (int k = k0; k < k1; k++) {
            const RowItem it = items[k];
            const int ng = (it.nrow + 3) / 4;
            const double *tl = rows + ((int64_t)it.tile + (int64_t)(it.nchunk + c) * ng) * 32 + lane;
#pragma unroll
            for (int g = 0; g < kGroups; g++)
                if (g < ng) {
                    const int r = 4 * g + (lane >> 3);
                    const double2 qq = r < it.nrow ? q[it.row0 + r] : make_double2(0.0, 0.0);
                    const double cr = odd ? -qq.x : qq.y, ci = odd ? -qq.y : -qq.x;
#pragma unroll
                    for (int h = 0; h < 4; h++)
                        if (c + h < cend) {
                            const double e = tl[32 * (h * ng + g)];
                            re[h] = fma(e, cr, re[h]);
                            im[h] = fma(e, ci, im[h]);
                        }
                }
        }
        double s[4];
#pragma unroll
        for (int h = 0; h < 4; h++)
            s[h] = (odd ? im[h] : re[h]) + __shfl_xor_sync(0xffffffffu, odd ? re[h] : im[h], 1);
        const double b0 = (u ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, u ? s[0] : s[2], 16);
        const double b1 = (u ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, u ? s[1] : s[3], 16);
        const double v = (w ? b1 : b0) + __shfl_xor_sync(0xffffffffu, w ? b0 : b1, 8);
        const int h = (u ? 2 : 0) + (w ? 1 : 0), m = 8 * (c + h) + (lane & 7);
        if (c + h < cend && m < 2 * P) a[(int64_t)b * 2 * P + m] = v * LBF_PI;
    }
}

// P2M per leaf, then M2M by the warp that completes a box's last child
// (a_l = d^l sum_{k <= l} C(l, k) (2d)^-k a'_k, two children at a time, one a half-warp:
// lane j of a half sums the rows l = j and P - 1 - j of the triangle in one loop)
__global__ void __launch_bounds__(128)
k_up_rows(int64_t nleaf, const int32_t *__restrict__ leaves, const int32_t *__restrict__ ix,
          const int32_t *__restrict__ iy, const int32_t *__restrict__ parent,
          const int32_t *__restrict__ child0, const int32_t *__restrict__ nchild, int P, int lchunks,
          const int32_t *__restrict__ block0, const RowItem *__restrict__ items,
          const double *__restrict__ rows, const double *__restrict__ binom,
          const cx<double> *__restrict__ dtab, const double2 *__restrict__ q, cx<double> *mp,
          int *cnt, const int *gate, int64_t slab)
{
    lbf_rhs(slab, q, mp, cnt, gate);
    if (fmm::gate_closed(gate)) return;
    __shared__ double Cl[32 * 32];
    __shared__ cx<double> As[4][2][32];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < P * P; e += blockDim.x) {
        const int k = e / P, l = e % P;
        Cl[e] = k <= l ? binom[l * LBF_MAX_TERMS + k] : 0.0;  // C(l, k)
    }
    __syncthreads();
    const int64_t t = blockIdx.x * 4ll + wid;
    if (t >= nleaf) return;
    const int b = leaves[t];
    leaf_p2m(t, b, P, block0, items, rows, q, (double *)mp, lane, 0, lchunks);
    const int hf = lane >> 4, j = lane & 15;
    const unsigned hmask = hf ? 0xffff0000u : 0x0000ffffu;
    const int nr = (P + 1) / 2, r1 = j < nr ? j : 0, r2 = P - 1 - r1, n1 = r1 + 1;
    cx<double> *Ah = As[wid][hf];
    for (int cur = b;;) {
        const int p = parent[cur];
        if (p < 0) break;
        __threadfence();
        __syncwarp();
        int last = 0;
        if (lane == 0) {
            last = atomicAdd(&cnt[p], 1) == nchild[p] - 1;
            if (last) cnt[p] = 0;  // ready for the next application
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        if (!last) break;
        __threadfence();
        cx<double> a1 = mk<double>(0, 0), a2 = mk<double>(0, 0);
        const int cend = child0[p] + nchild[p];
        for (int c0 = child0[p]; c0 < cend; c0 += 2) {
            const int c = c0 + hf;
            if (c < cend) {
                const int d = (ix[c] & 1) + 2 * (iy[c] & 1);
                const cx<double> *inv = fmm::d2inv(dtab, d);
                for (int k = j; k < P; k += 16)
                    Ah[k] = fmm::cmul(fmm::ldcg_cx(&mp[(int64_t)c * P + k]), inv[k]);
                __syncwarp(hmask);
                cx<double> acc = mk<double>(0, 0), s1 = mk<double>(0, 0);
                for (int it = 0; it <= P; it++) {
                    const bool first = it < n1;
                    if (it == n1) {
                        s1 = acc;
                        acc = mk<double>(0, 0);
                    }
                    const int k = first ? it : it - n1, l = first ? r1 : r2;
                    const cx<double> a = Ah[k];
                    const double cc = Cl[k * P + l];
                    acc.x = fma(cc, a.x, acc.x);
                    acc.y = fma(cc, a.y, acc.y);
                }
                const cx<double> *dp = fmm::dpow(dtab, d);
                a1 = fmm::cfma(dp[r1], s1, a1);
                a2 = fmm::cfma(dp[r2], acc, a2);
                __syncwarp(hmask);
            }
        }
        a1.x += __shfl_xor_sync(0xffffffffu, a1.x, 16);
        a1.y += __shfl_xor_sync(0xffffffffu, a1.y, 16);
        a2.x += __shfl_xor_sync(0xffffffffu, a2.x, 16);
        a2.y += __shfl_xor_sync(0xffffffffu, a2.y, 16);
        if (j < nr) {
            if (hf == 0) mp[(int64_t)p * P + r1] = a1;
            else if (r2 != r1) mp[(int64_t)p * P + r2] = a2;
        }
        cur = p;
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

constexpr unsigned kL2lSpins = 1u << 24;

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

__device__ __forceinline__ cx<double> own_part(const Own &w, int64_t b, int P, int lane, int v0, int dv,
                                               double ir, const cx<double> *loc)
{
    cx<double> o = mk<double>(0, 0);
    if (lane >= P) return o;
    const int v1 = w.ptr[b + 1];
    if (w.src) {
#pragma unroll 4
        for (int v = w.ptr[b] + v0; v < v1; v += dv) {
            const cx<double> a = w.part[(int64_t)v * P + lane];
            const double y = w.y[w.src[v]];
            o.x = fma(y, a.x, o.x);
            o.y = fma(y, a.y, o.y);
        }
        return o;
    }
#pragma unroll 4
    for (int v = w.ptr[b] + v0; v < v1; v += dv) {
        const cx<double> a = w.part[(int64_t)v * P + lane];
        o.x += a.x;
        o.y += a.y;
    }
    o.x *= ir;
    o.y *= ir;
    if (v0 == 0 && w.nx[b] && w.en[b] - w.bg[b] > w.thr) {
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

// Every box's local expansion: its own part, and from level 3 on its parent's expansion
// shifted down,
//   b'_l = (2d)^-l sum_{k >= l} C(k, l) d^k b_k.
// pull: the words of k_down's chain ([1] finished warps, [2] epoch, [3] box counter, then
// nbox words unused here and nbox epochs in which a box was finished).
__global__ void __launch_bounds__(256)
k_l2l(int64_t nbox, int P, const int32_t *__restrict__ level, const int32_t *__restrict__ ix,
      const int32_t *__restrict__ iy, const int32_t *__restrict__ parent, Own w, BoxGeo g,
      const double *__restrict__ binom, const cx<double> *__restrict__ dtab, cx<double> *loc,
      unsigned *pull, int *status, const int *gate, int64_t slab)
{
    lbf_rhs(slab, loc, pull, gate, w.y, w.sums);
    if (!w.src) lbf_rhs(slab, w.part);
    if (fmm::gate_closed(gate)) return;
    __shared__ double Cd[32 * 32];
    __shared__ cx<double> As[8][32];
    const int nw = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < P * P; e += blockDim.x) {
        const int k = e / P, l = e % P;
        Cd[e] = k >= l ? binom[k * LBF_MAX_TERMS + l] : 0.0;
    }
    __syncthreads();
    unsigned *done = pull + 4 + nbox;
    unsigned epoch = 0;
    if (lane == 0) epoch = *(volatile unsigned *)&pull[2];
    epoch = __shfl_sync(0xffffffffu, epoch, 0);
    cx<double> *A = As[wid];
    // lane j of a half has the rows r1 = j and r2 = P - 1 - j of the triangle, P + 1 terms
    // (n1 = P - r1 of them row r1's); half hf sums the terms [hf mid, hf ? P + 1 : mid)
    const int hf = lane >> 4, j = lane & 15, nr = (P + 1) / 2;
    const int r1 = j < nr ? j : 0, r2 = P - 1 - r1, n1 = P - r1, mid = (P + 2) / 2;
    const int i0 = hf ? mid : 0, i1 = hf ? P + 1 : mid;
    for (;;) {
        unsigned bi = 0;
        if (lane == 0) bi = atomicAdd(&pull[3], 1u);
        const int64_t b = (int64_t)__shfl_sync(0xffffffffu, bi, 0);
        if (b >= nbox) break;
        const int lv = level[b], p = parent[b];
        if (w.sums && b == 0) strength_sums(w, lane);
        const cx<double> own = own_part(w, b, P, lane, 0, 1, g.invL * fmm::pow2<double>(lv + 1), loc);
        if (lv >= 3) {
            const int d = (ix[b] & 1) + 2 * (iy[b] & 1);
            const cx<double> *dp = fmm::dpow(dtab, d), *inv = fmm::d2inv(dtab, d);
            const cx<double> dk = dp[lane], iv = inv[hf ? r2 : r1];
            if (lane == 0) {
                unsigned spins = 0;
                const unsigned lim = wait_limit(status, kL2lSpins);
                while (*(volatile unsigned *)&done[p] != epoch + 1u)
                    if (++spins > lim) {
                        atomicOr(status, LBF_DEV_TIMEOUT);
                        break;
                    }
                __threadfence();
            }
            __syncwarp();
            if (lane < P) A[lane] = fmm::cmul(fmm::ldcg_cx(&loc[(int64_t)p * P + lane]), dk);
            __syncwarp();
            cx<double> acc = mk<double>(0, 0), first = mk<double>(0, 0);
            for (int it = i0; it < i1; it++) {
                if (it == n1) {
                    first = acc;
                    acc = mk<double>(0, 0);
                }
                const int k = it < n1 ? r1 + it : r2 + (it - n1), l = it < n1 ? r1 : r2;
                const cx<double> a = A[k];
                const double c = Cd[k * P + l];
                acc.x = fma(c, a.x, acc.x);
                acc.y = fma(c, a.y, acc.y);
            }
            if (i1 <= n1) {  // the half's terms were all row r1's
                first = acc;
                acc = mk<double>(0, 0);
            }
            // the first half of the warp finishes the rows r1, the second the rows r2
            const cx<double> mine = hf ? acc : first, other = hf ? first : acc;
            cx<double> s = mk<double>(mine.x + __shfl_xor_sync(0xffffffffu, other.x, 16),
                                      mine.y + __shfl_xor_sync(0xffffffffu, other.y, 16));
            const int row = hf ? r2 : r1;
            const cx<double> o = mk<double>(__shfl_sync(0xffffffffu, own.x, row),
                                            __shfl_sync(0xffffffffu, own.y, row));
            s = fmm::cfma(iv, s, o);
            if (j < nr && (hf == 0 || r2 != r1)) loc[b * P + row] = s;
        } else if (lane < P) {
            loc[b * P + lane] = own;
        }
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicExch(&done[b], epoch + 1u);
    }
    if (lane == 0) {
        const unsigned total = gridDim.x * (unsigned)nw;
        if (atomicAdd(&pull[1], 1u) == total - 1u) {
            pull[1] = 0u;
            pull[3] = 0u;
            __threadfence();
            atomicExch(&pull[2], epoch + 1u);
        }
    }
}

// The two passes of a small system, a thread block of four warps a leaf or box.
//
// Up: two chunks of a leaf's reals a warp; then the block that completes a box's last child
// forms the box, a child a warp, the halves of a warp sharing each row's sum as in k_l2l.
__global__ void __launch_bounds__(128)
k_up_small(const int32_t *__restrict__ leaves, const int32_t *__restrict__ ix,
           const int32_t *__restrict__ iy, const int32_t *__restrict__ parent,
           const int32_t *__restrict__ child0, const int32_t *__restrict__ nchild, int P, int lchunks,
           const int32_t *__restrict__ block0, const RowItem *__restrict__ items,
           const double *__restrict__ rows, const double *__restrict__ binom,
           const cx<double> *__restrict__ dtab, const double2 *__restrict__ q, cx<double> *mp,
           int *cnt, const int *gate, int64_t slab)
{
    lbf_rhs(slab, q, mp, cnt, gate);
    if (fmm::gate_closed(gate)) return;
    __shared__ double Cl[32 * 32];
    __shared__ cx<double> As[4][32], part[4][32];
    __shared__ int s_last;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < P * P; e += blockDim.x) {
        const int k = e / P, l = e % P;
        Cl[e] = k <= l ? binom[l * LBF_MAX_TERMS + k] : 0.0;  // C(l, k)
    }
    const int64_t t = blockIdx.x;
    const int b = leaves[t];
    leaf_p2m(t, b, P, block0, items, rows, q, (double *)mp, lane, min(lchunks, 2 * wid),
             min(lchunks, 2 * wid + 2));
    const int hf = lane >> 4, j = lane & 15, nr = (P + 1) / 2;
    const int r1 = j < nr ? j : 0, r2 = P - 1 - r1, n1 = r1 + 1, mid = (P + 2) / 2;
    const int i0 = hf ? mid : 0, i1 = hf ? P + 1 : mid, row = hf ? r2 : r1;
    for (int cur = b;;) {
        const int p = parent[cur];
        if (p < 0) break;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            const int last = atomicAdd(&cnt[p], 1) == nchild[p] - 1;
            if (last) cnt[p] = 0;  // ready for the next application
            __threadfence();
            s_last = last;
        }
        __syncthreads();
        if (!s_last) break;
        const int nc = nchild[p], c = child0[p] + wid;
        if (wid < nc) {
            const int d = (ix[c] & 1) + 2 * (iy[c] & 1);
            if (lane < P)
                As[wid][lane] = fmm::cmul(fmm::ldcg_cx(&mp[(int64_t)c * P + lane]), fmm::d2inv(dtab, d)[lane]);
            const cx<double> dr = fmm::dpow(dtab, d)[row];
            __syncwarp();
            cx<double> acc = mk<double>(0, 0), first = mk<double>(0, 0);
            for (int it = i0; it < i1; it++) {
                if (it == n1) {
                    first = acc;
                    acc = mk<double>(0, 0);
                }
                const int k = it < n1 ? it : it - n1, l = it < n1 ? r1 : r2;
                const cx<double> a = As[wid][k];
                const double cc = Cl[k * P + l];
                acc.x = fma(cc, a.x, acc.x);
                acc.y = fma(cc, a.y, acc.y);
            }
            if (i1 <= n1) {
                first = acc;
                acc = mk<double>(0, 0);
            }
            const cx<double> mine = hf ? acc : first, other = hf ? first : acc;
            const cx<double> s = mk<double>(mine.x + __shfl_xor_sync(0xffffffffu, other.x, 16),
                                            mine.y + __shfl_xor_sync(0xffffffffu, other.y, 16));
            if (j < nr && (hf == 0 || r2 != r1)) part[wid][row] = fmm::cmul(dr, s);
        }
        __syncthreads();
        if (wid == 0 && lane < P) {
            cx<double> a = part[0][lane];
            for (int w = 1; w < nc; w++) {
                a.x += part[w][lane].x;
                a.y += part[w][lane].y;
            }
            mp[(int64_t)p * P + lane] = a;
        }
        cur = p;
    }
}

// Down: as k_l2l, a box a thread block: the warps add every fourth translation, wait for the
// parent together, and take a quarter of the shift's terms each (a half-warp an eighth).
__global__ void __launch_bounds__(128)
k_l2l_small(int64_t nbox, int P, const int32_t *__restrict__ level, const int32_t *__restrict__ ix,
            const int32_t *__restrict__ iy, const int32_t *__restrict__ parent, Own w, BoxGeo g,
            const double *__restrict__ binom, const cx<double> *__restrict__ dtab, cx<double> *loc,
            unsigned *pull, int *status, const int *gate, int64_t slab)
{
    lbf_rhs(slab, loc, pull, gate, w.y, w.sums);
    if (!w.src) lbf_rhs(slab, w.part);
    if (fmm::gate_closed(gate)) return;
    __shared__ double Cd[32 * 32];
    __shared__ cx<double> As[4][32], part[4][32], own[4][32];
    __shared__ unsigned s_ticket, s_epoch;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < P * P; e += blockDim.x) {
        const int k = e / P, l = e % P;
        Cd[e] = k >= l ? binom[k * LBF_MAX_TERMS + l] : 0.0;
    }
    if (threadIdx.x == 0) s_epoch = *(volatile unsigned *)&pull[2];
    unsigned *done = pull + 4 + nbox;
    const int hf = lane >> 4, j = lane & 15, nr = (P + 1) / 2, eighth = 2 * wid + hf;
    const int r1 = j < nr ? j : 0, r2 = P - 1 - r1, n1 = P - r1;
    const int i0 = (P + 1) * eighth / 8, i1 = (P + 1) * (eighth + 1) / 8;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_ticket = atomicAdd(&pull[3], 1u);
        __syncthreads();
        const int64_t b = (int64_t)s_ticket;
        const unsigned epoch = s_epoch;
        if (b >= nbox) break;
        const int lv = level[b], p = parent[b];
        const int d = (ix[b] & 1) + 2 * (iy[b] & 1);
        const cx<double> dk = fmm::dpow(dtab, d)[lane], iv = fmm::d2inv(dtab, d)[lane];
        if (w.sums && b == 0 && wid == 3) strength_sums(w, lane);
        own[wid][lane] = own_part(w, b, P, lane, wid, 4, g.invL * fmm::pow2<double>(lv + 1), loc);
        if (lv >= 3) {
            if (threadIdx.x == 0) {
                unsigned spins = 0;
                const unsigned lim = wait_limit(status, kL2lSpins);
                while (*(volatile unsigned *)&done[p] != epoch + 1u)
                    if (++spins > lim) {
                        atomicOr(status, LBF_DEV_TIMEOUT);
                        break;
                    }
                __threadfence();
            }
            __syncthreads();
            if (lane < P) As[wid][lane] = fmm::cmul(fmm::ldcg_cx(&loc[(int64_t)p * P + lane]), dk);
            __syncwarp();
            cx<double> acc = mk<double>(0, 0), first = mk<double>(0, 0);
            for (int it = i0; it < i1; it++) {
                if (it == n1) {
                    first = acc;
                    acc = mk<double>(0, 0);
                }
                const int k = it < n1 ? r1 + it : r2 + (it - n1), l = it < n1 ? r1 : r2;
                const cx<double> a = As[wid][k];
                const double c = Cd[k * P + l];
                acc.x = fma(c, a.x, acc.x);
                acc.y = fma(c, a.y, acc.y);
            }
            if (i1 <= n1) {
                first = acc;
                acc = mk<double>(0, 0);
            }
            const cx<double> mine = hf ? acc : first, other = hf ? first : acc;
            const cx<double> s = mk<double>(mine.x + __shfl_xor_sync(0xffffffffu, other.x, 16),
                                            mine.y + __shfl_xor_sync(0xffffffffu, other.y, 16));
            if (j < nr && (hf == 0 || r2 != r1)) part[wid][hf ? r2 : r1] = s;
        }
        __syncthreads();
        if (wid == 0) {
            if (lane < P) {
                cx<double> o = own[0][lane];
                for (int w = 1; w < 4; w++) {
                    o.x += own[w][lane].x;
                    o.y += own[w][lane].y;
                }
                if (lv >= 3) {
                    cx<double> s = part[0][lane];
                    for (int w = 1; w < 4; w++) {
                        s.x += part[w][lane].x;
                        s.y += part[w][lane].y;
                    }
                    o = fmm::cfma(iv, s, o);
                }
                loc[b * P + lane] = o;
            }
            __threadfence();
            __syncwarp();
            if (lane == 0) atomicExch(&done[b], epoch + 1u);
        }
    }
    if (threadIdx.x == 0 && atomicAdd(&pull[1], 1u) == gridDim.x - 1u) {
        pull[1] = 0u;
        pull[3] = 0u;
        __threadfence();
        atomicExch(&pull[2], s_epoch + 1u);
    }
}

BoxGeo geo_of(const Tree &T)
{
    return BoxGeo{T.xmin, T.ymin, T.L, (float)(1.0 / T.L), df64(1.0 / T.L), 1.0 / T.L};
}

}  // namespace

static int l2l(lbf_plan *pl, int P, const Own &w, cx<double> *loc, int kid, const int *gate,
               cudaStream_t s)
{
    const Tree &T = pl->tree;
    const int64_t nsm = std::max(pl->nsm, 1);
    if (T.nleaf < kSmallLeaves)
        LBF_LAUNCH_P(kid, k_l2l_small, lbf_grid(pl, std::min<int64_t>(T.nbox, 8 * nsm)), 128, 0, s, T.nbox,
                     P, T.level, T.ix, T.iy, T.parent, w, geo_of(T), pl->tab_binom,
                     (const cx<double> *)pl->tab_dshift, loc, pl->pull, pl->dev_status, gate, pl->slab);
    else
        LBF_LAUNCH_P(kid, k_l2l, lbf_grid(pl, std::min<int64_t>(lbf_cdiv(T.nbox, 8), 4 * nsm)), 256, 0, s,
                     T.nbox, P, T.level, T.ix, T.iy, T.parent, w, geo_of(T), pl->tab_binom,
                     (const cx<double> *)pl->tab_dshift, loc, pl->pull, pl->dev_status, gate, pl->slab);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

// whether the plan's double applications take these passes
bool lbf_passes_ready(const lbf_plan *pl) { return pl->rows && pl->m2l_cap && pl->nbigx >= 0; }

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

// multipoles of the charges pl->q
int lbf_passes_up(lbf_plan *pl, const int *gate, cudaStream_t s)
{
    const Tree &T = pl->tree;
    const int P = pl->P, lch = (2 * P + 7) / 8;
    const bool small = T.nleaf < kSmallLeaves;
    if (small)
        LBF_LAUNCH_P(LBF_KERNEL_UP, k_up_small, lbf_grid(pl, T.nleaf), 128, 0, s, T.leaves, T.ix, T.iy,
                     T.parent, T.child0, T.nchild, P, lch, pl->rows_block0, pl->rows_items, pl->rows,
                     pl->tab_binom, (const cx<double> *)pl->tab_dshift, pl->q, (cx<double> *)pl->mpole,
                     pl->upcnt, gate, pl->slab);
    else
        LBF_LAUNCH_P(LBF_KERNEL_UP, k_up_rows, lbf_grid(pl, lbf_cdiv(T.nleaf, 4)), 128, 0, s, T.nleaf,
                     T.leaves, T.ix, T.iy, T.parent, T.child0, T.nchild, P, lch, pl->rows_block0,
                     pl->rows_items, pl->rows, pl->tab_binom, (const cx<double> *)pl->tab_dshift, pl->q,
                     (cx<double> *)pl->mpole, pl->upcnt, gate, pl->slab);
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
    rc = lbf_m2l_apply(pl, gate, s);
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
