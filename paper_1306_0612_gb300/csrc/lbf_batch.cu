// Batched solves of independent geometries (many instances of the system of Sec. 5,
// each with several right-hand sides).  A host-side scheduler: worker threads, each
// with its own CUDA stream, take whole instances largest-first (plan, every
// right-hand side's solve and evaluation, plan destroyed) so that the small,
// latency-bound solves of different instances overlap on the GPU.
#include <algorithm>
#include <atomic>
#include <thread>
#include <vector>

#include "lbf_internal.cuh"

namespace {

constexpr size_t kRoundUp = 65536;  // what a caller may round a workspace's size up by

int run_item(lbf_batch_item &it, const lbf_options &opt_all, cudaStream_t s)
{
    lbf_plan *pl = nullptr;
    int64_t need = 0;
    lbf_options opt = opt_all;
    opt.box_capacity = it.box_capacity;
    // the right-hand sides in lockstep when the item's workspace holds their buffers after the
    // plan's: with as many stored parts as leave room for them (lbf_workspace_sizes); one after
    // another in a workspace of a plan's own size, whole
    size_t pbytes = it.bytes;
    bool lock = false, plans = false;
    for (int r = 0; r < LBF_WORKSPACE_SIZES && it.nrhs > 1; r++) {
        size_t pb = 0, ib = 0;
        if (lbf_rung_size(it.M, it.island_ptr, opt, it.nrhs, r, &pb, &ib) != LBF_OK || ib == pb) break;
        plans = plans || (it.bytes >= pb && it.bytes < pb + kRoundUp);
        if (!lock && ib <= it.bytes) {
            lock = true;
            pbytes = (pb + 255) & ~size_t(255);
        }
    }
    if (plans) {
        lock = false;
        pbytes = it.bytes;
    }
    int rc = lbf_plan_create(&pl, it.M, it.island_ptr, it.x, it.dx, it.d2x, it.centres, nullptr,
                             &opt, it.workspace, pbytes, &need, (lbf_stream_t)s);
    if (rc) {
        it.box_capacity_needed = need;
        return rc;
    }
    const int64_t N = pl->N;
    int worst = LBF_OK;
    size_t mbytes = 0;
    lock = lock && lbf_gmres_workspace_many(pl, it.nrhs, &mbytes) == LBF_OK && mbytes > 0 &&
           it.bytes >= pbytes + mbytes;
    if (lock) {
        std::vector<int> its(it.nrhs, 0);
        std::vector<double> rr(it.nrhs, 0.0);
        rc = lbf_gmres_solve_many(pl, it.nrhs, it.g, it.sigma, it.a, its.data(), rr.data(),
                                  (char *)it.workspace + pbytes, it.bytes - pbytes, (lbf_stream_t)s);
        if (rc < 0) {
            worst = rc;
        } else {
            if (rc == LBF_NOCONV) worst = LBF_NOCONV;
            for (int r = 0; r < it.nrhs; r++) {
                it.iters += its[r];
                it.max_rel_res = std::max(it.max_rel_res, rr[r]);
            }
            int64_t st[4];
            lbf_solve_stats(pl, st);
            it.fp64_applies += st[1];
            it.fp32_applies += st[2];
            for (int r = 0; r < it.nrhs && it.T > 0 && it.u && worst >= 0; r++) {
                rc = lbf_evaluate(pl, it.sigma + r * N, it.a ? it.a + (int64_t)r * it.M : nullptr,
                                  it.T, it.targets, it.u + r * it.T, (lbf_stream_t)s);
                if (rc) worst = rc;
            }
        }
    }
    for (int r = 0; r < it.nrhs && worst >= 0 && !lock; r++) {
        int its = 0;
        double rr = 0.0;
        rc = lbf_gmres_solve(pl, it.g + r * N, it.sigma + r * N, it.a ? it.a + (int64_t)r * it.M : nullptr,
                             nullptr, &its, &rr, (lbf_stream_t)s);
        if (rc < 0) {
            worst = rc;
            break;
        }
        if (rc == LBF_NOCONV) worst = LBF_NOCONV;
        it.iters += its;
        it.max_rel_res = std::max(it.max_rel_res, rr);
        int64_t st[4];
        lbf_solve_stats(pl, st);
        it.fp64_applies += st[1];
        it.fp32_applies += st[2];
        if (it.T > 0 && it.u) {
            rc = lbf_evaluate(pl, it.sigma + r * N, it.a ? it.a + (int64_t)r * it.M : nullptr, it.T,
                              it.targets, it.u + r * it.T, (lbf_stream_t)s);
            if (rc) worst = rc;
        }
    }
    // every path: the item's kernels finish before its plan (and the caller's view of
    // its workspace) is released
    if (cudaStreamSynchronize(s) != cudaSuccess && worst >= 0) worst = LBF_ECUDA;
    lbf_plan_destroy(pl);
    return worst;
}

// largest first: nodes times right-hand sides
std::vector<int> order_of(int nitems, const lbf_batch_item *items)
{
    std::vector<int> order(nitems);
    for (int q = 0; q < nitems; q++) order[q] = q;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
        const int64_t wx = items[x].island_ptr[items[x].M] * std::max(items[x].nrhs, 1);
        const int64_t wy = items[y].island_ptr[items[y].M] * std::max(items[y].nrhs, 1);
        return wx > wy;
    });
    return order;
}

// Offsets of the workers' slices of a shared workspace, and its end: worker w begins with the
// w-th item of the order and later takes some behind the nw-th
std::vector<size_t> slices_of(const std::vector<int> &order, const lbf_batch_item *items, int nw)
{
    size_t later = 0;
    for (size_t k = nw; k < order.size(); k++) later = std::max(later, items[order[k]].bytes);
    std::vector<size_t> at(nw + 1, 0);
    for (int w = 0; w < nw; w++) {
        const size_t first = (size_t)w < order.size() ? items[order[w]].bytes : 0;
        at[w + 1] = at[w] + ((std::max(first, later) + 255) & ~size_t(255));
    }
    return at;
}

int workers_of(int nitems, int nworkers) { return std::max(1, std::min(nworkers, std::max(nitems, 1))); }

bool valid_items(int nitems, const lbf_batch_item *items, bool shared)
{
    for (int q = 0; q < nitems; q++) {
        const lbf_batch_item &it = items[q];
        if (it.nrhs < 0 || it.M < 1 || !it.island_ptr || (!shared && !it.workspace) ||
            (it.nrhs > 0 && (!it.g || !it.sigma)) || it.T < 0 || (it.T > 0 && it.u && !it.targets))
            return false;
    }
    return true;
}

// pool: the shared workspace, or null (every item has its own)
int run(int nitems, lbf_batch_item *items, const lbf_options *opt, int nworkers, char *pool,
        const std::vector<int> &order, const std::vector<size_t> &slice)
{
    for (int q = 0; q < nitems; q++) {
        lbf_batch_item &it = items[q];
        it.status = LBF_OK;
        it.iters = 0;
        it.fp64_applies = it.fp32_applies = 0;
        it.max_rel_res = 0.0;
        it.box_capacity_needed = 0;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LBF_ECUDA;
    const int nw = workers_of(nitems, nworkers);
    std::atomic<int> next{nw};  // worker w begins with item w
    std::atomic<int> fail{0};
    auto worker = [&](int w) {
        if (cudaSetDevice(dev) != cudaSuccess) {
            fail.store(1);
            return;
        }
        cudaStream_t s;
        if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) {
            fail.store(1);
            return;
        }
        for (int k = w; k < nitems; k = next.fetch_add(1)) {
            lbf_batch_item &it = items[order[k]];
            if (pool) it.workspace = pool + slice[w];
            it.status = run_item(it, *opt, s);
        }
        cudaStreamSynchronize(s);
        cudaStreamDestroy(s);
    };
    std::vector<std::thread> threads;
    threads.reserve(nw);
    for (int w = 0; w < nw; w++) threads.emplace_back(worker, w);
    for (auto &t : threads) t.join();
    return fail.load() ? LBF_ECUDA : LBF_OK;
}

}  // namespace

extern "C" int lbf_batch_run(int nitems, lbf_batch_item *items, const lbf_options *opt,
                             int nworkers)
{
    if (nitems < 0 || (nitems > 0 && !items) || !opt || nworkers < 1) return LBF_EINVAL;
    if (!valid_items(nitems, items, false)) return LBF_EINVAL;
    return run(nitems, items, opt, nworkers, nullptr, order_of(nitems, items), {});
}

extern "C" int lbf_batch_shared_size(int nitems, const lbf_batch_item *items, int nworkers, size_t *bytes)
{
    if (nitems < 0 || (nitems > 0 && !items) || nworkers < 1 || !bytes) return LBF_EINVAL;
    if (!valid_items(nitems, items, true)) return LBF_EINVAL;
    *bytes = slices_of(order_of(nitems, items), items, workers_of(nitems, nworkers)).back() + 256;
    return LBF_OK;
}

extern "C" int lbf_batch_run_shared(int nitems, lbf_batch_item *items, const lbf_options *opt,
                                    int nworkers, void *workspace, size_t bytes)
{
    if (nitems < 0 || (nitems > 0 && !items) || !opt || nworkers < 1 || !workspace) return LBF_EINVAL;
    if (!valid_items(nitems, items, true)) return LBF_EINVAL;
    const std::vector<int> order = order_of(nitems, items);
    const std::vector<size_t> slice = slices_of(order, items, workers_of(nitems, nworkers));
    char *base = (char *)(((uintptr_t)workspace + 255) & ~(uintptr_t)255);
    if ((size_t)(base - (char *)workspace) + slice.back() > bytes) return LBF_EWORKSPACE;
    return run(nitems, items, opt, nworkers, base, order, slice);
}
