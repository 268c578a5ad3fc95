// The multiplier block E (Eq. u_multi, matrix_eqns) stored for a few hundred islands:
// E_im = 2 G(x_i, c_m) at every node and centre, applied as a dense product.
//
// The tree form of E y (lbf_border.cu) costs four launches, one of them a serial chain down
// the tree, and about 128 double multiply-adds a node; its transpose needs an upward pass
// of 36 terms and a walk per centre.  With M <= 512 and N M <= 1e8 the stored block is one
// multiply-add and 8 bytes an entry in either direction, in one launch (two transposed): at
// 131,072 nodes and 256 islands E y 460 -> 70 us and E^T tau 960 -> 75 us, at 9,808 nodes
// and 24 islands E y with 16 right-hand sides 440 -> 25 us.  Above, the logarithms of the
// set-up (about 16 double instructions an entry) cost more than the applications of one solve
// save: 1e8 entries are 3 ms.
//
// Layout: nodes in blocks of 32 (Morton order, the last filled up with zero rows), centres in
// chunks of 8 (filled up with zero columns); a tile is 4 nodes x 8 centres, 32 doubles
// (lane = 8 (node mod 4) + centre mod 8), the 8 tiles of a block and chunk together.
#include <algorithm>

#include "lbf_fmm_tpl.cuh"
#include "lbf_log.cuh"

namespace {

constexpr int kEmatIslands = 512;
constexpr int64_t kEmatEntries = 100000000;

// E, a warp per (node block, chunk) in turn
__global__ void k_emat_fill(int64_t N, int M, int nch, const double2 *__restrict__ xi,
                            const double *__restrict__ ell, const double2 *__restrict__ xc,
                            const double *__restrict__ lam, const int32_t *__restrict__ live,
                            double *__restrict__ E)
{
    __shared__ LogTab tab;
    log_table(tab);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t nb = (N + 31) / 32, nw = gridDim.x * (int64_t)(blockDim.x >> 5);
    for (int64_t w = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); w < nb * nch; w += nw) {
    const int64_t b = w / nch;
    const int m = 8 * (int)(w % nch) + (lane & 7);
    const bool on = m < M;
    const double2 c = on ? xc[m] : make_double2(0.0, 0.0);
    const bool lv = on && live[m] != 0;
    const double lm = lv ? lam[m] - LBF_LN2 : -LBF_LN2;
    double *t = E + w * 256 + lane;
    for (int q = 0; q < 8; q++) {
        const int64_t i = 32 * b + 4 * q + (lane >> 3);
        double e = 0.0;
        if (i < N && on) {
            e = ell[i] + lm;
            if (lv) {
                const double2 z = xi[i];
                const double dx = z.x - c.x, dy = z.y - c.y;
                const double d2 = fma(dx, dx, dy * dy);
                e -= log_any(d2, tab);
            }
            e *= 1.0 / (2.0 * LBF_PI);
        }
        t[32 * q] = e;
    }
    }
}

// out_i = x_i + v_i + s sum_m E_im y_m (v nullable), a warp per node block
__global__ void __launch_bounds__(128)
k_emat_apply(int64_t N, int M, int nch, const double *__restrict__ E, const double *__restrict__ y,
             const double *x, const double *v, double s, double *out, const int *gate, int64_t slab)
{
    lbf_rhs(slab, y, x, v, out, gate);
    if (fmm::gate_closed(gate)) return;
    const int64_t b = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= (N + 31) / 32) return;
    const double *t = E + b * nch * 256 + lane;
    double acc[8];
#pragma unroll
    for (int q = 0; q < 8; q++) acc[q] = 0.0;
    double yn = lane < M ? y[lane] : 0.0;
    for (int c = 0; c < nch; c += 4) {
        const double yc = yn;
        const int m = 8 * c + 32 + lane;
        yn = m < M ? y[m] : 0.0;
#pragma unroll
        for (int h = 0; h < 4; h++) {
            if (c + h < nch) {
                double e[8];
#pragma unroll
                for (int q = 0; q < 8; q++) e[q] = t[32 * (8 * h + q)];
                const double ym = __shfl_sync(0xffffffffu, yc, 8 * h + (lane & 7));
#pragma unroll
                for (int q = 0; q < 8; q++) acc[q] = fma(e[q], ym, acc[q]);
            }
        }
        t += 1024;
    }
    // add the eight lanes of a node, halving the groups a lane holds at each step
    int q0 = 0;
#pragma unroll
    for (int bit = 4; bit > 0; bit >>= 1) {
        const bool up = (lane & bit) != 0;
#pragma unroll
        for (int q = 0; q < bit; q++) {
            const double keep = up ? acc[q + bit] : acc[q], send = up ? acc[q] : acc[q + bit];
            acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
        }
        q0 += up ? bit : 0;
    }
    const int64_t i = 32 * b + 4 * q0 + (lane >> 3);
    if (i < N) out[i] = x[i] + (v ? v[i] : 0.0) + s * acc[0];
}

// part[strip][m] = sum of E_im tau_i over the strip's node blocks, a warp per (strip, chunk)
__global__ void k_emat_t(int64_t N, int M, int nch, int nstrip, const double *__restrict__ E,
                         const double *__restrict__ tau, double *__restrict__ part, const int *gate)
{
    if (fmm::gate_closed(gate)) return;
    const int64_t w = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (w >= (int64_t)nstrip * nch) return;
    const int strip = (int)(w / nch), c = (int)(w % nch);
    const int64_t nb = (N + 31) / 32, b0 = nb * strip / nstrip, b1 = nb * (strip + 1) / nstrip;
    double a0 = 0.0, a1 = 0.0;
    double tn = b0 < b1 && 32 * b0 + lane < N ? tau[32 * b0 + lane] : 0.0;
    for (int64_t b = b0; b < b1; b++) {
        const double tc = tn;
        const int64_t i = 32 * (b + 1) + lane;
        tn = b + 1 < b1 && i < N ? tau[i] : 0.0;
        const double *t = E + (b * nch + c) * 256 + lane;
        double e[8];
#pragma unroll
        for (int q = 0; q < 8; q++) e[q] = t[32 * q];
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
            a0 = fma(e[q], __shfl_sync(0xffffffffu, tc, 4 * q + (lane >> 3)), a0);
            a1 = fma(e[q + 1], __shfl_sync(0xffffffffu, tc, 4 * q + 4 + (lane >> 3)), a1);
        }
    }
    double s = a0 + a1;
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    if (lane < 8) part[((int64_t)strip * nch + c) * 8 + lane] = s;
}

// out_m = add_m + s sum over the strips, in order (a warp per centre)
__global__ void k_emat_tsum(int M, int nch, int nstrip, const double *__restrict__ part, double s,
                            const double *add, double *out, const int *gate)
{
    if (fmm::gate_closed(gate)) return;
    const int m = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (m >= M) return;
    double a = 0.0;
    for (int k = lane; k < nstrip; k += 32) a += part[(int64_t)k * nch * 8 + m];
    a = fmm::wsum(a);
    if (lane == 0) out[m] = (add ? add[m] : 0.0) + s * a;
}

}  // namespace

// Room for E (null: E y by the tree), dropped when the workspace has none.
void lbf_emat_layout(lbf_plan *pl, int64_t N, int M, const lbf_options &o)
{
    Border &B = pl->bd;
    B.E = nullptr;
    B.use_E = false;
    B.nch = (M + 7) / 8;
    if (!o.border || M > kEmatIslands || N * (int64_t)M > kEmatEntries || !(pl->parts & LBF_PART_E)) return;
    Arena &A = pl->arena;
    const size_t off = A.off;
    const bool full = A.overflow;
    B.E = A.get<double>(lbf_cdiv(N, 32) * B.nch * 256);
    if (A.overflow && !full) {
        A.off = off;
        A.overflow = false;
        B.E = nullptr;
    } else {
        B.use_E = true;
    }
}

int lbf_emat_build(lbf_plan *pl, cudaStream_t s)
{
    Border &B = pl->bd;
    if (!B.E) return LBF_OK;
    const int64_t grid = std::min<int64_t>(lbf_cdiv(lbf_cdiv(pl->N, 32) * B.nch, 8), 8 * (int64_t)std::max(pl->nsm, 1));
    LBF_LAUNCH(k_emat_fill, grid, 256, 0, s, pl->N, pl->M, B.nch, pl->xi, B.ell, B.xc, B.lam, B.live,
               B.E);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

// out = x + v + sc E y (v nullable)
int lbf_emat_apply(lbf_plan *pl, const double *y, const double *x, const double *v, double sc,
                   double *out, const int *gate, cudaStream_t s)
{
    const Border &B = pl->bd;
    LBF_LAUNCH_P(LBF_KERNEL_ESUM, k_emat_apply, lbf_grid(pl, lbf_cdiv(lbf_cdiv(pl->N, 32), 4)), 128, 0,
                 s, pl->N, pl->M, B.nch, B.E, y, x, v, sc, out, gate, pl->slab);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}

// out = add + sc E^T tau (add nullable)
int lbf_emat_apply_transpose(lbf_plan *pl, const double *tau, double sc, const double *add,
                             double *out, const int *gate, cudaStream_t s)
{
    const Border &B = pl->bd;
    // about 16 warps a scheduler, bounded by the partial sums' room
    const int64_t most = std::min<int64_t>(4 * 16 * (int64_t)std::max(pl->nsm, 1) / B.nch,
                                           B.partial_cap / (8 * (int64_t)B.nch));
    const int nstrip = (int)std::max<int64_t>(1, std::min<int64_t>(lbf_cdiv(pl->N, 32), most));
    LBF_LAUNCH(k_emat_t, lbf_cdiv((int64_t)nstrip * B.nch, 4), 128, 0, s, pl->N, pl->M, B.nch, nstrip,
               B.E, tau, B.partial, gate);
    LBF_LAUNCH(k_emat_tsum, lbf_cdiv(pl->M, 4), 128, 0, s, pl->M, B.nch, nstrip, B.partial, sc, add, out,
               gate);
    LBF_CHECK_LAUNCH();
    return LBF_OK;
}
