// Adjoint of the solve-and-evaluate map (Sec. 4.1, Eq. u_multi; Sec. 5, Eq. disc_sphere):
// the transposed evaluation at off-curve targets and the gradient of a target
// functional with respect to the planar node positions xi_j (xi'_j, xi''_j fixed).
//
// With A z = b (z = [sigma; a], b = [2 g; 0]) and u = C z at the targets, a scalar
// L(u) with ubar = dL/du has dL/dg = 2 lam_sigma where A^T lam = C^T ubar, and
//   dL/dxi_j = d/dxi_j (ubar^T C z) - lam^T (dA/dxi_j) z.
// Every term is a Cauchy-type sum (the derivative FMM), a node-target sum, or the
// gradient of the multiplier potential; they are combined per node below.
#include <algorithm>

#include "lbf_fmm_tpl.cuh"

using fmm::BoxGeo;
using fmm::cx;
using fmm::mk;

namespace {

__device__ __forceinline__ double wsum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

struct Rot3 {
    double r[9];
    int on;
};

// target t on the sphere -> the plan's frame; xi_t, or w <= 0 at the pole
__device__ __forceinline__ void target_plane(const double *t, int64_t k, const Rot3 &R, double p[3],
                                             double &zx, double &zy, bool &finite)
{
    p[0] = t[3 * k];
    p[1] = t[3 * k + 1];
    p[2] = t[3 * k + 2];
    if (R.on) {
        double a = R.r[0] * p[0] + R.r[1] * p[1] + R.r[2] * p[2];
        double b = R.r[3] * p[0] + R.r[4] * p[1] + R.r[5] * p[2];
        double c = R.r[6] * p[0] + R.r[7] * p[1] + R.r[8] * p[2];
        p[0] = a; p[1] = b; p[2] = c;
    }
    double w = 1.0 - p[2];
    finite = w > 0.0;
    zx = finite ? p[0] / w : 0.0;
    zy = finite ? p[1] / w : 0.0;
}

// Per node (sorted order) the target sums, Power 1: S = sum_t ubar_t/(xi - xi_t), Power 2:
// S = sum_t ubar_t/(xi - xi_t)^2.
//
// Few pairs (N T <= kDirectPairs): all of them (k_node_target, targets tiled through shared
// memory and projected by each block).  More: the targets as sources of the FMM's downward
// pass.  They are sorted by their Morton key on the nodes' quadtree, so that the targets of any
// cell are one run of the sorted list, found by binary search; a box takes the targets of the
// cells that are separated from it but whose parents touch its parent's (P2L, at most 27
// cells), the expansions are shifted down, and a leaf adds the targets of the 3 x 3 cells around
// it directly.  Nothing of it goes through the host, so the call stays asynchronous.  A
// target is at least 3 half-widths from a box's centre, its nodes at most sqrt 2: kTerms = 48
// terms leave (sqrt 2/3)^48 = 2e-16.  At 131,072 nodes and 4096 targets 21.3 ms of pairs (both
// powers, with a division) a call to 1.9 ms, 0.7 of it P2L, 0.4 the shifts.
constexpr int64_t kDirectPairs = 1 << 24;
constexpr int kTerms = 48;

template <int Power>
__device__ __forceinline__ void target_term(double2 z, double2 t, double ub, double2 &s)
{
    const double dr = z.x - t.x, di = z.y - t.y;
    const double d2 = fma(dr, dr, di * di);
    const double id = d2 > 0x1p-120 && d2 < 0x1p120 ? fmm::rcp_near(d2) : 1.0 / d2;
    // 1/d = conj(d)/|d|^2, 1/d^2 = conj(d)^2/|d|^4
    const double er = dr * id, ei = -di * id;
    if (Power == 1) {
        s.x = fma(ub, er, s.x);
        s.y = fma(ub, ei, s.y);
    } else {
        const double ur = ub * er;
        s.x = fma(ur, er, fma(-ub * ei, ei, s.x));
        s.y = fma(ur + ur, ei, s.y);
    }
}

template <int Power>
__global__ void k_node_target(int64_t N, const double2 *__restrict__ xi, int64_t T,
                              const double *__restrict__ t, Rot3 R, const double *__restrict__ ub,
                              double2 *__restrict__ S)
{
    __shared__ double2 tz[256];
    __shared__ double tu[256];
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const double2 z = i < N ? xi[i] : make_double2(0, 0);
    double2 s = make_double2(0.0, 0.0);
    for (int64_t base = 0; base < T; base += 256) {
        __syncthreads();
        int64_t k = base + threadIdx.x;
        if (k < T) {
            double p[3], zx, zy;
            bool fin;
            target_plane(t, k, R, p, zx, zy, fin);
            tz[threadIdx.x] = make_double2(zx, zy);
            tu[threadIdx.x] = fin ? ub[k] : 0.0;  // a target at the pole has no Cauchy term
        }
        __syncthreads();
        int n = (int)(T - base < 256 ? T - base : 256);
        for (int m = 0; m < n; m++) target_term<Power>(z, tz[m], tu[m], s);
    }
    if (i < N) S[i] = s;
}

__device__ __forceinline__ uint64_t spread32(uint64_t v)
{
    v &= 0xffffffffull;
    v = (v | (v << 16)) & 0x0000ffff0000ffffull;
    v = (v | (v << 8)) & 0x00ff00ff00ff00ffull;
    v = (v | (v << 4)) & 0x0f0f0f0f0f0f0f0full;
    v = (v | (v << 2)) & 0x3333333333333333ull;
    v = (v | (v << 1)) & 0x5555555555555555ull;
    return v;
}

// key of each target's cell at depth D of the nodes' square, or past every cell's outside it
__global__ void k_target_keys(int64_t T, const double *__restrict__ t, Rot3 R, BoxGeo g, int D,
                              uint64_t *__restrict__ key, int32_t *__restrict__ idx)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= T) return;
    double p[3], zx, zy;
    bool fin;
    target_plane(t, k, R, p, zx, zy, fin);
    const double sc = g.invL * fmm::pow2<double>(D), top = fmm::pow2<double>(D);
    const double fx = (zx - g.xmin) * sc, fy = (zy - g.ymin) * sc;
    const bool in = fin && fx >= 0.0 && fy >= 0.0 && fx < top && fy < top;
    key[k] = in ? spread32((uint64_t)fx) | (spread32((uint64_t)fy) << 1) : 1ull << (2 * D);
    idx[k] = (int32_t)k;
}

// positions and weights in the sorted order
__global__ void k_target_gather(int64_t T, const double *__restrict__ t, Rot3 R,
                                const double *__restrict__ ub, const int32_t *__restrict__ idx,
                                double2 *__restrict__ tz, double *__restrict__ tu)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= T) return;
    const int64_t j = idx[k];
    double p[3], zx, zy;
    bool fin;
    target_plane(t, j, R, p, zx, zy, fin);
    tz[k] = make_double2(zx, zy);
    tu[k] = fin ? ub[j] : 0.0;
}

// first sorted target with a key >= v
__device__ __forceinline__ int lower_key(const uint64_t *__restrict__ key, int T, uint64_t v)
{
    int lo = 0, hi = T;
    while (lo < hi) {
        const int m = (lo + hi) >> 1;
        if (key[m] < v) lo = m + 1;
        else hi = m;
    }
    return lo;
}
// the targets of cell (x, y) of level l (none outside the square)
__device__ __forceinline__ int2 cell_run(const uint64_t *__restrict__ key, int T, int D, int l, int x,
                                         int y)
{
    if (x < 0 || y < 0 || x >= (1 << l) || y >= (1 << l)) return make_int2(0, 0);
    const uint64_t k0 = (spread32((uint64_t)x) | (spread32((uint64_t)y) << 1)) << (2 * (D - l));
    const int a = lower_key(key, T, k0);
    return make_int2(a, lower_key(key, T, k0 + (1ull << (2 * (D - l)))));
}

// P2L of the separated cells' targets into each box, a thread block of four warps per box, the
// targets' chunks of 32 dealt to the warps in turn:
// b_l = (1/r) (-1)^l sum_t ubar_t tau_t^(l+1), tau_t = r/(c - xi_t)
__global__ void __launch_bounds__(128)
k_target_p2l(const int32_t *__restrict__ level, const int32_t *__restrict__ ix,
             const int32_t *__restrict__ iy, BoxGeo g, int D, int T, const uint64_t *__restrict__ key,
             const double2 *__restrict__ tz, const double *__restrict__ tu, cx<double> *__restrict__ loc)
{
    extern __shared__ __align__(16) unsigned char tp_sm[];
    __shared__ int s_run[36], s_end[36], s_total;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cx<double> *term_s = (cx<double> *)tp_sm + wid * kTerms * 33;
    const int64_t b = blockIdx.x;
    const int l = level[b], bx = ix[b], by = iy[b];
    if (wid == 0) {
        int total = 0;
        for (int q0 = 0; q0 < 36; q0 += 32) {
            const int q = q0 + lane;
            int2 r = make_int2(0, 0);
            if (l >= 2 && q < 36) {
                const int x = 2 * ((bx >> 1) - 1) + q % 6, y = 2 * ((by >> 1) - 1) + q / 6;
                if (abs(x - bx) > 1 || abs(y - by) > 1) r = cell_run(key, T, D, l, x, y);
            }
            int inc = r.y - r.x;
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += v;
            }
            if (q < 36) {
                s_end[q] = total + inc;
                s_run[q] = r.x - (total + inc - (r.y - r.x));  // target = run + position
            }
            total += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) s_total = total;
    }
    __syncthreads();
    const int total = s_total;
    double cxd, cyd, ir;
    box_centre_ir(g, l, bx, by, cxd, cyd, ir);
    cx<double> s0 = mk<double>(0, 0), s1 = mk<double>(0, 0);
    for (int base = 32 * wid; base < total; base += 128) {
        const int at = base + lane;
        cx<double> tau = mk<double>(0, 0), term = mk<double>(0, 0);
        if (at < total) {
            int q = 0;
            while (at >= s_end[q]) q++;
            const int k = s_run[q] + at;
            const double2 z = tz[k];
            tau = fmm::crcp(mk<double>((cxd - z.x) * ir, (cyd - z.y) * ir));
            term = mk<double>(tu[k] * tau.x, tu[k] * tau.y);
        }
        for (int m = 0; m < kTerms; m++) {
            term_s[m * 33 + lane] = (m & 1) ? mk<double>(-term.x, -term.y) : term;
            term = fmm::cmul(term, tau);
        }
        __syncwarp();
        const int n = min(32, total - base);
        for (int m = 0; m < n; m++) {
            s0.x += term_s[lane * 33 + m].x;
            s0.y += term_s[lane * 33 + m].y;
        }
        if (lane + 32 < kTerms)
            for (int m = 0; m < n; m++) {
                s1.x += term_s[(lane + 32) * 33 + m].x;
                s1.y += term_s[(lane + 32) * 33 + m].y;
            }
        __syncwarp();
    }
    // the warps' sums, through the terms' memory
    term_s[lane] = s0;
    if (lane + 32 < kTerms) term_s[lane + 32] = s1;
    __syncthreads();
    if (threadIdx.x < kTerms) {
        const cx<double> *p = (const cx<double> *)tp_sm + threadIdx.x;
        cx<double> s = p[0];
        for (int w = 1; w < 4; w++) {
            s.x += p[w * kTerms * 33].x;
            s.y += p[w * kTerms * 33].y;
        }
        loc[b * kTerms + threadIdx.x] = mk<double>(s.x * ir, s.y * ir);
    }
}

// S at the nodes of a leaf, a thread block of four warps per leaf: the targets of the cells
// around it and those outside the square (a large leaf between large empty cells has
// thousands), and the local expansion (phi = sum ubar/(z - xi_t), S2 = -phi').  A chunk of 32
// nodes at a time: TP >= n lanes on the nodes, 128 / TP groups of lanes on every so many of the
// targets, their sums added in order.
template <int Power>
__global__ void __launch_bounds__(128)
k_target_nodes(const int32_t *__restrict__ leaves, const int32_t *__restrict__ level,
               const int32_t *__restrict__ ix, const int32_t *__restrict__ iy,
               const int32_t *__restrict__ bg, const int32_t *__restrict__ en, BoxGeo g, int D, int T,
               const uint64_t *__restrict__ key, const double2 *__restrict__ tz,
               const double *__restrict__ tu, const cx<double> *__restrict__ loc,
               const double2 *__restrict__ xi, double2 *__restrict__ S)
{
    __shared__ int2 run[10];
    __shared__ double2 part[128];
    const int b = leaves[blockIdx.x], l = level[b], bx = ix[b], by = iy[b], tid = threadIdx.x;
    // runs of the nine cells, and of the targets outside the square
    if (tid < 9) run[tid] = cell_run(key, T, D, l, bx + tid % 3 - 1, by + tid / 3 - 1);
    if (tid == 9) run[9] = make_int2(lower_key(key, T, 1ull << (2 * D)), T);
    __syncthreads();
    double cxd, cyd, ir;
    box_centre_ir(g, l, bx, by, cxd, cyd, ir);
    const cx<double> *lb = loc + (int64_t)b * kTerms;
    for (int i0 = bg[b]; i0 < en[b]; i0 += 32) {
        const int n = min(32, en[b] - i0);
        const int TP = n <= 1 ? 1 : 1 << (32 - __clz(n - 1)), G = 128 / TP;
        const int r = tid & (TP - 1), grp = tid / TP;
        const double2 z = xi[i0 + min(r, n - 1)];
        double2 s = make_double2(0.0, 0.0);
        for (int c = 0; c < 10; c++)
            for (int k = run[c].x + grp; k < run[c].y; k += G) target_term<Power>(z, tz[k], tu[k], s);
        part[tid] = s;
        __syncthreads();
        if (tid < n) {
            for (int w = 1; w < G; w++) {
                s.x += part[w * TP + tid].x;
                s.y += part[w * TP + tid].y;
            }
            if (l >= 2) {
                const cx<double> u = mk<double>((z.x - cxd) * ir, (z.y - cyd) * ir);
                cx<double> h = lb[kTerms - 1];
                if (Power == 2) h = mk<double>((kTerms - 1) * h.x, (kTerms - 1) * h.y);
#pragma unroll 4
                for (int m = kTerms - 2; m >= (Power == 2 ? 1 : 0); m--) {
                    const cx<double> c = lb[m];
                    h = fmm::cfma(h, u, Power == 2 ? mk<double>(m * c.x, m * c.y) : c);
                }
                s = Power == 2 ? make_double2(s.x - h.x * ir, s.y - h.y * ir)
                               : make_double2(s.x + h.x, s.y + h.y);
            }
            S[i0 + tid] = s;
        }
        __syncthreads();
    }
}

// s[0] = sum ubar, s[1] = sum lam_sigma (lam nullable), s[2] = sum a (a nullable); one block
__global__ void k_sums3(int64_t T, const double *__restrict__ ub, int64_t N,
                        const double *__restrict__ lam, int M, const double *__restrict__ a,
                        double *__restrict__ s)
{
    __shared__ double sh[3][32];
    double v[3] = {0.0, 0.0, 0.0};
    for (int64_t k = threadIdx.x; k < T; k += blockDim.x) v[0] += ub[k];
    if (lam)
        for (int64_t k = threadIdx.x; k < N; k += blockDim.x) v[1] += lam[k];
    if (a)
        for (int64_t k = threadIdx.x; k < M; k += blockDim.x) v[2] += a[k];
    for (int c = 0; c < 3; c++) {
        double x = wsum(v[c]);
        if ((threadIdx.x & 31) == 0) sh[c][threadIdx.x >> 5] = x;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double x = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) x += sh[threadIdx.x][w];
        s[threadIdx.x] = x;
    }
}

// sbar_i = (1/2pi) Im(w_i S1_i) + beta_i sum ubar  (sorted i -> caller perm[i])
__global__ void k_sbar(int64_t N, const int32_t *__restrict__ perm, const double2 *__restrict__ w,
                       const double *__restrict__ beta, const double2 *__restrict__ S1,
                       const double *__restrict__ s, double *__restrict__ out)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double2 ww = w[i], a = S1[i];
    out[perm[i]] = (ww.x * a.y + ww.y * a.x) * (1.0 / (2.0 * LBF_PI)) + beta[i] * s[0];
}

// abar_m = sum_t ubar_t G(t, c_m), G = (1/4pi) log(2 / |t - c|^2) (Eq. greens_func); warp per centre
__global__ void k_abar(int M, const double *__restrict__ c, int64_t T, const double *__restrict__ t,
                       Rot3 R, const double *__restrict__ ub, double *__restrict__ out)
{
    int m = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (m >= M) return;
    double acc = 0.0;
    for (int64_t k = lane; k < T; k += 32) {
        double p[3], zx, zy;
        bool fin;
        target_plane(t, k, R, p, zx, zy, fin);
        double d0 = p[0] - c[3 * m], d1 = p[1] - c[3 * m + 1], d2 = p[2] - c[3 * m + 2];
        acc += ub[k] * (1.0 / (4.0 * LBF_PI)) * log(2.0 / (d0 * d0 + d1 * d1 + d2 * d2));
    }
    acc = wsum(acc);
    if (lane == 0) out[m] = acc;
}

// gradient of beta_i = -(1/2pi) (X w_y - Y w_x) / (1 + X^2 + Y^2) in (X, Y) = xi_i
__device__ __forceinline__ double2 grad_beta(double2 z, double2 w)
{
    const double num = z.x * w.y - z.y * w.x, den = 1.0 + z.x * z.x + z.y * z.y;
    const double k = -1.0 / (2.0 * LBF_PI * den * den);
    return make_double2(k * (w.y * den - 2.0 * z.x * num), k * (-w.x * den - 2.0 * z.y * num));
}

// dL/dxi_i, sorted i -> caller perm[i] (N x 2):
//   (a)  Im/Re of  -(w_i sigma_i/2pi) S2_i        + U sigma_i grad beta_i        (evaluation)
//   (b1) -2 Im/Re of (w_i sigma_i/2pi) Dlam_i                                     (i as a source)
//   (b2) +2 lam_i Im/Re of (1/2pi) Dq_i                                           (i as a target)
//   (b3) -2 Lam sigma_i grad beta_i                                               (sphere correction)
//   (b4) -lam_i grad (E a)_i                                                      (multiplier potential)
// with Dlam = Phi'_lam, Dq = Phi'_(w sigma), U = sum ubar, Lam = sum lam_sigma.
__global__ void k_grad(int64_t N, const int32_t *__restrict__ perm, const double2 *__restrict__ xi,
                       const double2 *__restrict__ w, const double *__restrict__ sig,
                       const double *__restrict__ lam, const double2 *__restrict__ S2,
                       const double2 *__restrict__ Dl, const double2 *__restrict__ Dq,
                       const double2 *__restrict__ Eg, const double *__restrict__ s,
                       double *__restrict__ out)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double k = 1.0 / (2.0 * LBF_PI);
    const double2 ww = w[i], z = xi[i];
    const double sg = sig[i], lm = lam[i];
    // c = w_i sigma_i / 2pi
    const double cr = ww.x * sg * k, ci = ww.y * sg * k;
    auto cm = [](double ar, double ai, double br, double bi, double &rr, double &ri) {
        rr = ar * br - ai * bi;
        ri = ar * bi + ai * br;
    };
    double gr, gi;  // (Im F', Re F') convention: d/dX = Im F', d/dY = Re F'
    double gx = 0.0, gy = 0.0;
    cm(cr, ci, S2[i].x, S2[i].y, gr, gi);  // (a): F' = -c S2
    gx += -gi;
    gy += -gr;
    cm(cr, ci, Dl[i].x, Dl[i].y, gr, gi);  // (b1): H = c Dlam, contributes -2 (Im H, Re H)
    gx -= 2.0 * gi;
    gy -= 2.0 * gr;
    // (b2): Q = -(1/2pi) Dq, contributes -2 lam (Im Q, Re Q)
    gx += 2.0 * lm * k * Dq[i].y;
    gy += 2.0 * lm * k * Dq[i].x;
    const double2 gb = grad_beta(z, ww);
    const double fb = (s[0] - 2.0 * s[1]) * sg;  // (a) beta term and (b3)
    gx += fb * gb.x;
    gy += fb * gb.y;
    gx -= lm * Eg[i].x;  // (b4)
    gy -= lm * Eg[i].y;
    const int32_t j = perm[i];
    out[2 * j] = gx;
    out[2 * j + 1] = gy;
}

Rot3 plan_rot(const lbf_plan *pl)
{
    Rot3 R;
    R.on = pl->has_rot;
    for (int i = 0; i < 9; i++) R.r[i] = pl->rot[i];
    return R;
}

// dL/dg_j = 2 lam_j: the Dirichlet data enter the bordered system only through its
// doubled right-hand side [2 g; 0] (Eq. disc_sphere), so the adjoint of b -> z carries
// the factor 2 onto the node part of lam (caller order in and out)
__global__ void k_grad_data(int64_t N, const double *__restrict__ lam, double *__restrict__ gg)
{
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j < N) gg[j] = 2.0 * lam[j];
}

}  // namespace

// S of one power into S (N), scratch: the rest of the region from `free` on
template <int Power>
static int target_sums(lbf_plan *pl, int64_t T, const double *t, const double *ub, double2 *S,
                       char *free, cudaStream_t s)
{
    const int64_t N = pl->N;
    const Rot3 R = plan_rot(pl);
    const Tree &Tr = pl->tree;
    const int D = pl->opt.max_depth;
    char *end = pl->region + pl->region_bytes;
    auto take = [&](size_t bytes) {
        char *p = (char *)(((uintptr_t)free + 255) & ~(uintptr_t)255);
        free = p + bytes;
        return p;
    };
    const int64_t scratch_len = 256 * lbf_cdiv(T, 1024) + T / 4 + 8192;
    uint64_t *key = (uint64_t *)take(sizeof(uint64_t) * T), *key2 = (uint64_t *)take(sizeof(uint64_t) * T);
    int32_t *idx = (int32_t *)take(sizeof(int32_t) * T), *idx2 = (int32_t *)take(sizeof(int32_t) * T);
    double2 *tz = (double2 *)take(sizeof(double2) * T);
    double *tu = (double *)take(sizeof(double) * T);
    int32_t *scratch = (int32_t *)take(sizeof(int32_t) * scratch_len);
    cx<double> *loc = (cx<double> *)take(sizeof(cx<double>) * Tr.nbox * kTerms);
    if (pl->opt.matvec != LBF_MATVEC_FMM || T <= kDirectPairs / N || T > INT32_MAX / 2 || free > end ||
        !pl->pull) {
        LBF_LAUNCH(k_node_target<Power>, lbf_cdiv(N, 256), 256, 0, s, N, pl->xi, T, t, R, ub, S);
        LBF_CHECK_LAUNCH();
        return LBF_OK;
    }
    const BoxGeo g{Tr.xmin, Tr.ymin, Tr.L, (float)(1.0 / Tr.L), df64(1.0 / Tr.L), 1.0 / Tr.L};
    LBF_LAUNCH(k_target_keys, lbf_cdiv(T, 256), 256, 0, s, T, t, R, g, D, key, idx);
    LBF_CHECK_LAUNCH();
    int rc = lbf_radix_sort(key, key2, idx, idx2, T, 2 * D + 1, scratch, scratch_len, s);
    if (rc) return rc;
    constexpr int smem = 4 * kTerms * 33 * (int)sizeof(cx<double>);
    LBF_CUDA(cudaFuncSetAttribute(k_target_p2l, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    LBF_LAUNCH(k_target_gather, lbf_cdiv(T, 256), 256, 0, s, T, t, R, ub, idx, tz, tu);
    LBF_LAUNCH(k_target_p2l, Tr.nbox, 128, smem, s, Tr.level, Tr.ix, Tr.iy, g, D, (int)T, key, tz, tu, loc);
    LBF_CHECK_LAUNCH();
    if ((rc = lbf_mp_shift_down(pl, kTerms, (double2 *)loc, s))) return rc;
    LBF_LAUNCH(k_target_nodes<Power>, Tr.nleaf, 128, 0, s, Tr.leaves, Tr.level, Tr.ix, Tr.iy,
                Tr.begin, Tr.end, g, D, (int)T, key, tz, tu, loc, pl->xi, S);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

int lbf_gradient_data_impl(lbf_plan *pl, const double *lam, double *grad_g, cudaStream_t s)
{
    if (pl->N > 0) LBF_LAUNCH(k_grad_data, lbf_cdiv(pl->N, 256), 256, 0, s, pl->N, lam, grad_g);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

int lbf_evaluate_transpose_impl(lbf_plan *pl, int64_t T, const double *t, const double *ub,
                                double *sbar, double *abar, cudaStream_t s)
{
    int64_t N = pl->N;
    int M = pl->M;
    // scratch: the GMRES basis region (unused outside a solve)
    double2 *S1 = (double2 *)pl->region;
    double *sums = (double *)(S1 + N);
    Rot3 R = plan_rot(pl);
    LBF_LAUNCH(k_sums3, 1, 1024, 0, s, T, ub, N, (const double *)nullptr, M,
               (const double *)nullptr, sums);
    const int rc = target_sums<1>(pl, T, t, ub, S1, (char *)(sums + 8), s);
    if (rc) return rc;
    LBF_LAUNCH(k_sbar, lbf_cdiv(N, 256), 256, 0, s, N, pl->perm, pl->w, pl->beta, S1, sums, sbar);
    if (abar) LBF_LAUNCH(k_abar, lbf_cdiv((int64_t)M * 32, 256), 256, 0, s, M, pl->centres, T, t, R, ub, abar);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

int lbf_gradient_nodes_impl(lbf_plan *pl, const double *sigma, const double *a, const double *lam,
                            int64_t T, const double *t, const double *ub, double *grad,
                            cudaStream_t s)
{
    int64_t N = pl->N;
    int M = pl->M;
    double2 *S2 = (double2 *)pl->region, *Dl = S2 + N, *Dq = Dl + N, *Eg = Dq + N;
    double *sg = (double *)(Eg + N), *lm = sg + N, *sums = lm + N;
    int rc;
    if ((rc = lbf_permute_in(pl, sigma, sg, 0, s)) || (rc = lbf_permute_in(pl, lam, lm, 0, s)))
        return rc;
    LBF_LAUNCH(k_sums3, 1, 1024, 0, s, T, ub, N, lm, M, a, sums);
    LBF_CHECK_LAUNCH();
    if ((rc = target_sums<2>(pl, T, t, ub, S2, (char *)(sums + 8), s))) return rc;
    if ((rc = lbf_cauchy_deriv(pl, lm, false, Dl, s))) return rc;
    if ((rc = lbf_cauchy_deriv(pl, sg, true, Dq, s))) return rc;
    if ((rc = lbf_mp_gradient(pl, a, Eg, s))) return rc;
    LBF_LAUNCH(k_grad, lbf_cdiv(N, 256), 256, 0, s, N, pl->perm, pl->xi, pl->w, sg, lm, S2, Dl, Dq,
               Eg, sums, grad);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}
