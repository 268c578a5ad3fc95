// The representation formula at off-curve targets (Eq. u_multi, planar form of the double
// layer, Eq. dlpC):
//   u(t) = (1/2pi) Im sum_j q_j/(xi_j - xi_t) + beta.sigma + sum_m a_m G(t, c_m).
//
// Few pairs (T N <= kDirectPairs): the sum over all nodes, a warp per target and run of
// nodes, then a warp per target over its partial sums: two launches of some ten
// microseconds where the upward pass and the walk of one target down the tree take 200
// (16 targets and 14,000 nodes, the batched workload: 345 -> 25 us).  More: multipoles of the
// boxes well separated from the target, a warp per target (k_eval_walk).
//
// The walk pops up to 32 boxes at a time from a stack in shared memory, a box a lane.  A box
// to be taken as a multipole waits in a list until there are 32, so that the Horner sums run
// with every lane at work, and a leaf to be summed directly is summed by the whole warp:
// a lane that did its box's series or its leaf's nodes alone left the double pipe, which
// charges an instruction in full whatever its active lanes, to a few lanes (40,000 targets
// and 65,536 nodes: 6.0 ms).
#include <algorithm>

#include "lbf_fmm_tpl.cuh"
#include "lbf_log.cuh"

using fmm::BoxGeo;
using fmm::cx;
using fmm::mk;

namespace {

constexpr int64_t kDirectPairs = 1 << 24;
// boxes at least kEvalSep half-widths away enter through their multipole (every node of the
// box is within sqrt(2) r of its centre, so the series ratio is at most 1/3 and the
// truncation after P terms is below 3^-P relative)
constexpr double kEvalSep = 4.25;
// A step pops 32 boxes and pushes at most 128; below a popped box's level the stack grows by
// at most 96 a level, so 30 levels need at most 3,008 entries.
constexpr int kStack = 3072;
constexpr int kEvalWarps = 4;
constexpr int kEvalSmem = kEvalWarps * (kStack + 64) * (int)sizeof(int32_t);

struct Target {
    double p[3];  // on the sphere, in the plan's frame
    double zx, zy;
    bool finite;  // a target at the pole sees no Cauchy term (xi = infinity)
};

__device__ __forceinline__ Target target_of(const double *__restrict__ t, int64_t k, int rot_on,
                                            const double *__restrict__ rot)
{
    Target r;
    const double a = t[3 * k], b = t[3 * k + 1], c = t[3 * k + 2];
    if (rot_on) {
        r.p[0] = rot[0] * a + rot[1] * b + rot[2] * c;
        r.p[1] = rot[3] * a + rot[4] * b + rot[5] * c;
        r.p[2] = rot[6] * a + rot[7] * b + rot[8] * c;
    } else {
        r.p[0] = a;
        r.p[1] = b;
        r.p[2] = c;
    }
    const double w = 1.0 - r.p[2];
    r.finite = w > 0.0;
    r.zx = r.finite ? r.p[0] / w : 0.0;
    r.zy = r.finite ? r.p[1] / w : 0.0;
    return r;
}

// Im q/(xi - t)
__device__ __forceinline__ double pair_im(double2 z, double2 q, double zx, double zy, double acc)
{
    const double dr = z.x - zx, di = z.y - zy;
    const double d2 = fma(dr, dr, di * di);
    const double id = d2 > 0x1p-120 && d2 < 0x1p120 ? fmm::rcp_near(d2) : 1.0 / d2;
    return fma(fma(q.y, dr, -q.x * di), id, acc);
}

// sum_m a_m G(t, c_m), lanes over the centres (not yet added over the lanes)
__device__ __forceinline__ double centres_part(const Target &t, int M, const double *__restrict__ a,
                                               const double *__restrict__ c, const LogTab &tab,
                                               int lane)
{
    double s = 0.0;
    for (int m = lane; m < M; m += 32) {
        const double d0 = t.p[0] - c[3 * m], d1 = t.p[1] - c[3 * m + 1], d2 = t.p[2] - c[3 * m + 2];
        s = fma(a[m], LBF_LN2 - log_any(fma(d0, d0, fma(d1, d1, d2 * d2)), tab), s);
    }
    return s * (1.0 / (4.0 * LBF_PI));
}

// part[target][run]: the pair sums over a run of nodes, a warp each
__global__ void __launch_bounds__(128)
k_eval_pairs(int64_t N, const double2 *__restrict__ xi, const double2 *__restrict__ q, int64_t T,
             const double *__restrict__ t, int rot_on, const double *__restrict__ rot, int nrun,
             double *__restrict__ part)
{
    const int64_t w = blockIdx.x * 4ll + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (w >= T * nrun) return;
    const int64_t k = w / nrun, r = w % nrun;
    const Target tg = target_of(t, k, rot_on, rot);
    double acc = 0.0;
    if (tg.finite) {
        const int64_t e = N * (r + 1) / nrun;
#pragma unroll 2
        for (int64_t j = N * r / nrun + lane; j < e; j += 32)
            acc = pair_im(xi[j], q[j], tg.zx, tg.zy, acc);
    }
    acc = fmm::wsum(acc);
    if (lane == 0) part[w] = acc;
}

__global__ void __launch_bounds__(128)
k_eval_sum(int M, const double *__restrict__ part, int nrun, const double *__restrict__ bsig,
           const double *__restrict__ a, const double *__restrict__ c, int64_t T,
           const double *__restrict__ t, int rot_on, const double *__restrict__ rot,
           double *__restrict__ u)
{
    __shared__ LogTab tab;
    if (a) log_table(tab);
    __syncthreads();
    const int64_t k = blockIdx.x * 4ll + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (k >= T) return;
    double s = 0.0;
    for (int r = lane; r < nrun; r += 32) s += part[k * nrun + r];
    s *= 1.0 / (2.0 * LBF_PI);
    if (a) s += centres_part(target_of(t, k, rot_on, rot), M, a, c, tab, lane);
    s = fmm::wsum(s);
    if (lane == 0) u[k] = s + *bsig;
}

__global__ void __launch_bounds__(32 * kEvalWarps)
k_eval_walk(int M, const double2 *__restrict__ xi, const double2 *__restrict__ q,
            const cx<double> *__restrict__ mp, int P, const int32_t *__restrict__ level,
            const int32_t *__restrict__ ix, const int32_t *__restrict__ iy,
            const int32_t *__restrict__ child0, const int32_t *__restrict__ nchild,
            const int32_t *__restrict__ bg, const int32_t *__restrict__ en, BoxGeo g,
            const double *__restrict__ bsig, const double *__restrict__ a,
            const double *__restrict__ c, int64_t T, const double *__restrict__ t, int rot_on,
            const double *__restrict__ rot, double *__restrict__ u, int *__restrict__ status)
{
    extern __shared__ int32_t eval_sm[];
    __shared__ LogTab tab;
    if (a) log_table(tab);
    __syncthreads();
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t k = blockIdx.x * (int64_t)kEvalWarps + wid;
    if (k >= T) return;
    int32_t *stack = eval_sm + wid * (kStack + 64), *far = stack + kStack;
    const Target tg = target_of(t, k, rot_on, rot);
    double acc = 0.0, fac = 0.0;  // Im of the pairs, and of the multipoles' Phi
    const unsigned below = (1u << lane) - 1u;
    auto box_offset = [&](int b, double &dx, double &dy, double &ir) {
        double cx_, cy_;
        box_centre_ir(g, level[b], ix[b], iy[b], cx_, cy_, ir);
        dx = tg.zx - cx_;
        dy = tg.zy - cy_;
    };
    // M2P of the first n listed boxes, a box a lane: Phi(t) = (1/r) sum_k a_k rho^(k+1),
    // rho = r/(t - c); q/(xi - t) = -Phi
    auto take = [&](int n) {
        __syncwarp();
        if (lane < n) {
            const int b = far[lane];
            double dx, dy, ir;
            box_offset(b, dx, dy, ir);
            dx *= ir;
            dy *= ir;
            // |t - c|/r is above 4; targets beyond rcp_near's range are at infinity for the box
            const double d2 = fma(dx, dx, dy * dy);
            const double id = d2 < 0x1p120 ? fmm::rcp_near(d2) : 1.0 / d2;
            const cx<double> rho = mk<double>(dx * id, -dy * id);
            const cx<double> *ak = mp + (int64_t)b * P;
            cx<double> ps = ak[P - 1];
#pragma unroll 4
            for (int l = P - 2; l >= 0; l--) ps = fmm::cfma(ps, rho, ak[l]);
            fac = fma(fma(ps.x, rho.y, ps.y * rho.x), ir, fac);
        }
        __syncwarp();
    };
    if (tg.finite) {
        int top = 1, nfar = 0;
        if (lane == 0) stack[0] = 0;
        __syncwarp();
        while (top > 0) {
            const int n = min(top, 32);
            top -= n;
            int b = -1, kids = 0;
            bool multi = false, leaf = false;
            if (lane < n) {
                b = stack[top + lane];
                double dx, dy, ir;
                box_offset(b, dx, dy, ir);
                dx *= ir;
                dy *= ir;
                multi = b != 0 && fma(dx, dx, dy * dy) >= kEvalSep * kEvalSep;
                kids = multi ? 0 : nchild[b];
                leaf = !multi && kids == 0;
            }
            __syncwarp();
            // far boxes to the list (at most 31 + 32 entries)
            const unsigned fm = __ballot_sync(0xffffffffu, multi);
            if (multi) far[nfar + __popc(fm & below)] = b;
            nfar += __popc(fm);
            if (nfar >= 32) {
                take(32);
                const int rest = nfar - 32;
                const int32_t v = lane < rest ? far[32 + lane] : 0;
                __syncwarp();
                if (lane < rest) far[lane] = v;
                nfar = rest;
            }
            // leaves: the whole warp over the nodes of each
            for (unsigned lm = __ballot_sync(0xffffffffu, leaf); lm; lm &= lm - 1) {
                const int lb = __shfl_sync(0xffffffffu, b, __ffs(lm) - 1);
                const int e = en[lb];
                for (int j = bg[lb] + lane; j < e; j += 32) acc = pair_im(xi[j], q[j], tg.zx, tg.zy, acc);
            }
            // the children, in lane order
            int incl = kids;
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            if (top + total > kStack) {
                if (lane == 0) atomicOr(status, 8);
                break;
            }
            for (int i = 0; i < kids; i++) stack[top + incl - kids + i] = child0[b] + i;
            top += total;
            __syncwarp();
        }
        take(nfar);
    }
    double s = (acc - fac) * (1.0 / (2.0 * LBF_PI));
    if (a) s += centres_part(tg, M, a, c, tab, lane);
    s = fmm::wsum(s);
    if (lane == 0) u[k] = s + *bsig;
}

}  // namespace

int lbf_evaluate_init_attrs()
{
    LBF_CUDA(cudaFuncSetAttribute(k_eval_walk, cudaFuncAttributeMaxDynamicSharedMemorySize, kEvalSmem));
    return LBF_OK;
}

int lbf_evaluate_impl(lbf_plan *pl, const double *sigma_sorted, const double *a, int64_t T,
                      const double *t, double *u, cudaStream_t s)
{
    const int64_t N = pl->N;
    if (T <= 0) return lbf_eval_charges(pl, sigma_sorted, s);
    int rc;
    // direct: plans without an FMM, and few pairs; the partial sums stand in the region of
    // the GMRES basis (unused outside a solve)
    const int64_t warps = 16 * 4 * (int64_t)std::max(pl->nsm, 1);
    int nrun = (int)std::max<int64_t>(1, std::min<int64_t>(lbf_cdiv(warps, T), lbf_cdiv(N, 128)));
    nrun = (int)std::min<int64_t>(nrun, std::max<int64_t>(1, (int64_t)(pl->region_bytes / sizeof(double)) / T));
    const bool room = (size_t)T * nrun * sizeof(double) <= pl->region_bytes;
    if (pl->opt.matvec != LBF_MATVEC_FMM || (T <= kDirectPairs / N && room)) {
        if ((rc = lbf_eval_charges(pl, sigma_sorted, s))) return rc;
        const int64_t batch = room ? T : std::max<int64_t>(1, (int64_t)(pl->region_bytes / sizeof(double)));
        for (int64_t k = 0; k < T; k += batch) {
            const int64_t n = std::min(batch, T - k);
            double *part = (double *)pl->region;
            LBF_LAUNCH(k_eval_pairs, lbf_cdiv(n * nrun, 4), 128, 0, s, N, pl->xi, pl->q, n, t + 3 * k,
                       pl->has_rot, pl->rot_d, nrun, part);
            LBF_LAUNCH(k_eval_sum, lbf_cdiv(n, 4), 128, 0, s, pl->M, part, nrun, pl->bsig, a, pl->centres,
                       n, t + 3 * k, pl->has_rot, pl->rot_d, u + k);
        }
        LBF_CHECK_LAUNCH();
        return LBF_OK;
    }
    if ((rc = lbf_eval_multipoles(pl, sigma_sorted, s))) return rc;
    const Tree &Tr = pl->tree;
    const BoxGeo g{Tr.xmin, Tr.ymin, Tr.L, (float)(1.0 / Tr.L), df64(1.0 / Tr.L), 1.0 / Tr.L};
    LBF_LAUNCH(k_eval_walk, lbf_cdiv(T, kEvalWarps), 32 * kEvalWarps, kEvalSmem, s, pl->M, pl->xi, pl->q,
               (const cx<double> *)pl->mpole, pl->P, Tr.level, Tr.ix, Tr.iy, Tr.child0, Tr.nchild,
               Tr.begin, Tr.end, g, pl->bsig, a, pl->centres, T, t, pl->has_rot, pl->rot_d, u,
               pl->dev_status);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}
