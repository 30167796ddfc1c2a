// batch.cu -- many independent IM queries solved together (im_solve_batch).
//
// Queries may differ in graph, model, k and theta.  The batch runs in a fixed
// number of launches whatever the number of queries:
//   1. one sampling launch per model over the flattened samples of all its
//      queries (each sample finds its query and that query's graph, see
//      run_sampling in sample.cu);
//   2. one scan and one segmented sort over all sets;
//   3. members are moved into one vertex space (query q's vertex u becomes
//      vbase[q] + u) so that one radix sort builds the covering subsets of every
//      query at once;
//   4. one launch of the standard greedy for all plain queries, each on a group
//      of blocks by its share of the members (greedy_many in cover.cu).
// Each query's result equals what it gets alone (the random stream of a
// sample depends only on the query's seed and the sample id).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <new>
#include <numeric>
#include <tuple>
#include <vector>

#include "internal.cuh"

struct im_batch {
    int device = 0;
    void *arena = nullptr;
    size_t arena_bytes = 0;
    void *sscratch = nullptr;  // sampling scratch
    size_t sscratch_bytes = 0;
    // members per set to reserve, per graph and model: twice the most seen in
    // earlier batches (64 before any), four times more after a capacity miss
    std::map<std::pair<const im_graph *, int32_t>, int64_t> entry_hint;
    // RandGreedi queries: a pool view per graph (its partition and RandGreedi
    // buffers are owned, the index is the batch's), and the partition count
    // picked for each (graph, model, power-of-two theta)
    std::map<const im_graph *, im_pool *> views;
    std::map<std::tuple<const im_graph *, int32_t, int32_t>, int32_t> rg_parts;
};

namespace im {
namespace {

// Vertices of a query's graph at most.  No kernel of the batch needs the limit (one
// that kept its bounds in shared memory did); callers that meet it have the
// one-query path, and it is known before any work is done.
constexpr int64_t kBatchMaxN = 200 * 1024 / 8 * 1024;

struct BatchQuery {
    int64_t vbase;     // first vertex of the query in the batch vertex space
    int64_t n;
    int64_t sbase;     // first set of the query in the batch
    int64_t theta;
    int64_t cbase;     // first word of the query's covered bitmap
    int64_t out;       // row of the query in the seeds output (original index)
    int32_t k;
};

// First member position of every query's sets: out[i] = set_off[qset[i]].
__global__ void k_query_bounds(const int64_t *set_off, const int64_t *qset, int32_t nq,
                               int64_t *out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= nq; i += gridDim.x * blockDim.x)
        out[i] = set_off[qset[i]];
}

// A RandGreedi query reads its covering subsets with its own set ids: the
// batch ids of its entries [vtx_off[0], vtx_off[n]) lose the query's first set.
__global__ void k_localize(int32_t *set_ids, const int64_t *vtx_off, int64_t n, int64_t sbase) {
    const int64_t b = vtx_off[0], e = vtx_off[n];
    for (int64_t t = b + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < e;
         t += (int64_t)gridDim.x * blockDim.x)
        set_ids[t] -= (int32_t)sbase;
}

// Moves the members into the batch's vertex space: those of query q, positions
// [bounds[q], bounds[q + 1]), gain vbase[q].  A warp takes kGlobalRun positions.
constexpr int kGlobalRun = 1024;

__global__ void __launch_bounds__(256) k_globalize(int32_t *members, int64_t T, const int64_t *bounds,
                                                   const int64_t *vbase, int32_t nq) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t t0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kGlobalRun; t0 < T;
         t0 += warps * kGlobalRun) {
        int lo = 0, hi = nq - 1;                 // the query of the run's first position
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(bounds + mid) <= t0) lo = mid;
            else hi = mid - 1;
        }
        int64_t end = __ldg(bounds + lo + 1);
        int32_t vb = (int32_t)__ldg(vbase + lo);
#pragma unroll 8
        for (int i = 0; i < kGlobalRun; i += 32) {
            const int64_t t = t0 + i + lane;
            if (t >= T) break;
            while (t >= end) {
                ++lo;
                end = __ldg(bounds + lo + 1);
                vb = (int32_t)__ldg(vbase + lo);
            }
            members[t] += vb;
        }
    }
}

// Stage offsets of the second sampling launch, relative to its part of the
// stage, become relative to the stage (kept apart from the flag in their top bits
// by being far below it).
__global__ void k_shift(const int64_t *in, int64_t count, int64_t by, int64_t *out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = in[i] + by;
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

im_status grow(void **p, size_t *have, size_t need) {
    if (need <= *have) return IM_OK;
    if (*p) {
        IM_CUDA(cudaDeviceSynchronize());
        cudaFree(*p);
        *p = nullptr;
        *have = 0;
    }
    const size_t want = need + need / 4 + 4096;
    if (cudaMalloc(p, want) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        set_error("im_solve_batch: device memory exhausted");
        return IM_ERR_OOM;
    }
    *have = want;
    return IM_OK;
}

// A pool that borrows a batch's covering subsets for one query at a time:
// theta, vtx_off and set_ids are set per query; the partition, RandGreedi and
// scratch buffers are its own, kept between queries on the same graph.
im_pool *make_pool_view(const im_graph *g, int device) {
    im_pool *v = new (std::nothrow) im_pool();
    if (!v) return nullptr;
    std::memset(v, 0, sizeof(*v));
    v->g = g;
    v->device = device;
    return v;
}

void release_pool_view(im_pool *v) {
    if (!v) return;
    for (void *b : {(void *)v->vtx_cursor, (void *)v->part, (void *)v->part_off,
                    (void *)v->part_vtx, (void *)v->part_loc, (void *)v->rg_block, v->scratch,
                    v->res})
        dev_free(b);
    delete v;
}

// The partition counts a RandGreedi query may use: powers of two from 16 and
// the SM count, each part small enough for one producer block.
std::vector<int32_t> partition_candidates(int64_t n) {
    std::vector<int32_t> c;
    for (int32_t P = 16; P < num_sms(); P *= 2) c.push_back(P);
    c.push_back(num_sms());
    std::vector<int32_t> ok;
    for (int32_t P : c)
        if (P <= n && (n + P - 1) / P <= 16384) ok.push_back(P);
    if (ok.empty()) ok.push_back((int32_t)std::min<int64_t>(n, std::max<int64_t>(1, (n + 16383) / 16384)));
    return ok;
}

}  // namespace
}  // namespace im

using namespace im;

extern "C" {

im_status im_batch_create(im_batch **out) {
    if (!out) return IM_ERR_INVALID_ARG;
    im_batch *b = new (std::nothrow) im_batch();
    if (!b) return IM_ERR_OOM;
    cudaGetDevice(&b->device);
    *out = b;
    return IM_OK;
}

im_status im_batch_destroy(im_batch *b) {
    if (!b) return IM_ERR_INVALID_ARG;
    cudaDeviceSynchronize();
    for (auto &kv : b->views) release_pool_view(kv.second);
    cudaFree(b->arena);
    cudaFree(b->sscratch);
    delete b;
    return IM_OK;
}

im_status im_solve_batch(im_batch *b, const im_query *qs, int32_t nq, int32_t kmax, int32_t *seeds,
                         int64_t *gains, im_result *res, void *stream) {
    if (!b || !qs || nq < 1 || kmax < 1 || !seeds || !res) {
        set_error("im_solve_batch: bad arguments");
        return IM_ERR_INVALID_ARG;
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // validate; LT queries need their graph's LT index
    int64_t n_total = 0, sets_total = 0, n_max = 1;
    for (int32_t q = 0; q < nq; ++q) {
        const im_query &Q = qs[q];
        if (!Q.graph || (Q.model != IM_IC && Q.model != IM_LT) || Q.k < 1 || Q.k > kmax ||
            Q.k > Q.graph->n || Q.theta < 0 || Q.theta >= ((int64_t)1 << 31) ||
            Q.graph->device != b->device) {
            set_error("im_solve_batch: query out of range");
            return IM_ERR_INVALID_ARG;
        }
        const im_cover_opts &o = Q.cover;
        if (o.algo == IM_RANDGREEDI) {
            if (o.partitions < 0 || o.partitions > 4096 || o.partitions > Q.graph->n ||
                o.alpha_num < 1 || o.alpha_den < 1 || o.alpha_num > o.alpha_den ||
                !(o.delta > 0.0 && o.delta < 0.5) ||
                (o.aggregator != IM_AGG_STREAM && o.aggregator != IM_AGG_GREEDY)) {
                set_error("im_solve_batch: RandGreedi options out of range");
                return IM_ERR_INVALID_ARG;
            }
        } else if (o.algo != IM_GREEDY_PLAIN && o.algo != IM_GREEDY_LAZY) {
            set_error("im_solve_batch: unknown algorithm");
            return IM_ERR_INVALID_ARG;
        }
        if (Q.model == IM_LT) {
            im_status s = build_lt_index(const_cast<im_graph *>(Q.graph), st);
            if (s != IM_OK) return s;
            if (!Q.graph->lt_valid) {
                set_error("im_solve_batch: LT query on a graph whose in-weights exceed 1");
                return IM_ERR_INVALID_ARG;
            }
        } else {
            IM_TRY(build_ic_index(const_cast<im_graph *>(Q.graph), st));
        }
        n_total += Q.graph->n;
        sets_total += Q.theta;
        n_max = std::max<int64_t>(n_max, Q.graph->n);
    }
    if (n_total >= ((int64_t)1 << 31)) {
        set_error("im_solve_batch: the batch's vertices exceed 2^31");
        return IM_ERR_CAPACITY;
    }
    if (n_max > kBatchMaxN) {
        set_error("im_solve_batch: a query graph is too large for the batched greedy");
        return IM_ERR_UNSUPPORTED;
    }
    // batch order: IC queries, then LT queries (one sampling launch each)
    std::vector<int32_t> order(nq);
    std::iota(order.begin(), order.end(), 0);
    std::stable_partition(order.begin(), order.end(), [&](int32_t q) { return qs[q].model == IM_IC; });
    std::vector<BatchQuery> bq(nq);
    std::vector<int64_t> qset(nq + 1, 0), vbase(nq, 0);
    int64_t vb = 0, sb = 0, cb = 0;
    for (int32_t i = 0; i < nq; ++i) {
        const im_query &Q = qs[order[i]];
        bq[i].vbase = vb;
        bq[i].n = Q.graph->n;
        bq[i].sbase = sb;
        bq[i].theta = Q.theta;
        bq[i].cbase = cb;
        bq[i].out = order[i];
        bq[i].k = Q.k;
        vbase[i] = vb;
        qset[i] = sb;
        vb += Q.graph->n;
        sb += Q.theta;
        cb += (Q.theta + 31) / 32;
    }
    qset[nq] = sb;
    const int64_t cov_words = std::max<int64_t>(cb, 1);
    std::vector<int64_t> greedy_n;                   // vertices of the queries of greedy_many
    for (int32_t q = 0; q < nq; ++q)
        if (qs[q].cover.algo != IM_RANDGREEDI) greedy_n.push_back(qs[q].graph->n);

    for (int attempt = 0; attempt < 8; ++attempt) {
        int64_t cap = 1024;
        for (int32_t q = 0; q < nq; ++q) {
            auto it = b->entry_hint.find({qs[q].graph, qs[q].model});
            cap += qs[q].theta * (it == b->entry_hint.end() ? 64 : it->second);
        }
        // arena layout
        size_t off = 0;
        auto take = [&](size_t bytes) {
            size_t at = off;
            off += up256(bytes);
            return at;
        };
        const size_t o_stage = take((size_t)cap * 4), o_mem = take((size_t)cap * 4),
                     o_sids = take((size_t)cap * 4), o_soff = take((size_t)(sets_total + 1) * 8),
                     o_sizes = take((size_t)std::max<int64_t>(sets_total, 1) * 4),
                     o_stoff = take((size_t)std::max<int64_t>(sets_total, 1) * 8),
                     o_voff = take((size_t)(n_total + 1) * 8), o_cur = take((size_t)n_total * 4),
                     o_key = take((size_t)n_total * 4), o_stamp = take((size_t)n_total * 4),
                     o_cov = take((size_t)cov_words * 4),
                     o_qset = take((size_t)(nq + 1) * 8), o_vbase = take((size_t)nq * 8),
                     o_tmp = take(std::max(scan_tmp_bytes(std::max(sets_total, n_total)),
                                           (size_t)(2 + 2 * std::max<int64_t>(sets_total, 1)) * 8)),
                     o_out = take(up256((size_t)nq * kmax * 4) + up256((size_t)nq * kmax * 8) +
                                  up256((size_t)nq * 4) + up256((size_t)nq * 8)),
                     o_bounds = take((size_t)(nq + 1) * 8),
                     o_many = take(greedy_many_scratch(greedy_n, cap)), o_gbar = take(256);
        im_status s = grow(&b->arena, &b->arena_bytes, off);
        if (s != IM_OK) return s;
        char *A = (char *)b->arena;
        int32_t *stage = (int32_t *)(A + o_stage);
        int64_t *set_off = (int64_t *)(A + o_soff);
        int32_t *sizes = (int32_t *)(A + o_sizes);
        int64_t *stage_off = (int64_t *)(A + o_stoff);

        // 1. sampling: one launch per model
        int64_t added = 0, examined = 0;
        bool capacity = false;
        unsigned long long long_sets = 0;
        int64_t done_sets = 0;
        for (int mi = 0; mi < 2 && !capacity; ++mi) {
            const im_model model = mi == 0 ? IM_IC : IM_LT;
            SamplingJob job;
            job.model = model;
            job.n_max = 1;
            for (int32_t i = 0; i < nq; ++i) {
                const im_query &Q = qs[order[i]];
                if (Q.model != model) continue;
                job.views.push_back(query_view(Q.graph, Q.seed, 0));
                job.counts.push_back(Q.theta);
                job.n_max = std::max<int64_t>(job.n_max, Q.graph->n);
            }
            if (job.views.empty()) continue;
            int64_t nsets = 0;
            for (int64_t c : job.counts) nsets += c;
            job.stage = stage + added;
            job.stage_cap = cap - added;
            SamplingResult r;
            s = run_sampling(job,
                             [&](size_t bytes, void **p) {
                                 im_status g2 = grow(&b->sscratch, &b->sscratch_bytes, bytes);
                                 *p = b->sscratch;
                                 return g2;
                             },
                             st, &r);
            if (s == IM_ERR_CAPACITY) {
                capacity = true;
                break;
            }
            if (s != IM_OK) return s;
            // gather sizes and stage offsets (relative to `stage`) in batch order
            IM_CUDA(cudaMemcpyAsync(sizes + done_sets, r.sizes, (size_t)nsets * 4,
                                    cudaMemcpyDeviceToDevice, st));
            {
                KernelTimer kt(st, "batch_shift");
                k_shift<<<num_sms() * 4, 256, 0, st>>>(r.stage_off, nsets, added, stage_off + done_sets);
            }
            IM_CUDA(cudaGetLastError());
            done_sets += nsets;
            added += r.added;
            long_sets += r.long_sets;
            examined += r.examined;
        }
        if (capacity) {
            std::map<std::pair<const im_graph *, int32_t>, bool> seen;
            for (int32_t q = 0; q < nq; ++q) {
                const auto key = std::make_pair(qs[q].graph, (int32_t)qs[q].model);
                if (seen[key]) continue;                 // once per graph and model
                seen[key] = true;
                auto &h = b->entry_hint[key];
                h = std::max<int64_t>(h, 64) * 4;
            }
            continue;
        }
        IM_CUDA(cudaStreamSynchronize(st));


        // 2. set offsets and sorted members
        void *tmp = A + o_tmp;
        s = exclusive_scan_i32_to_i64(sizes, set_off, sets_total, nullptr, tmp,
                                      scan_tmp_bytes(sets_total), st);
        if (s != IM_OK) return s;
        int32_t *members = (int32_t *)(A + o_mem);
        s = segmented_sort_sets(members, set_off, sets_total, stage, stage_off, tmp, n_max,
                                long_sets, st);
        if (s != IM_OK) return s;
        // 3. one vertex space, one index
        IM_CUDA(cudaMemcpyAsync(A + o_qset, qset.data(), (size_t)(nq + 1) * 8, cudaMemcpyHostToDevice, st));
        IM_CUDA(cudaMemcpyAsync(A + o_vbase, vbase.data(), (size_t)nq * 8, cudaMemcpyHostToDevice, st));
        int64_t *d_bounds = (int64_t *)(A + o_bounds);
        {
            KernelTimer kt(st, "batch_bounds");
            k_query_bounds<<<std::max(1, std::min(num_sms(), (nq + 256) / 256)), 256, 0, st>>>(
                set_off, (const int64_t *)(A + o_qset), nq, d_bounds);
        }
        if (added > 0) {
            KernelTimer kt(st, "batch_globalize");
            k_globalize<<<num_sms() * 8, 256, 0, st>>>(members, added, d_bounds,
                                                       (const int64_t *)(A + o_vbase), nq);
        }
        IM_CUDA(cudaGetLastError());
        int64_t *vtx_off = (int64_t *)(A + o_voff);
        int32_t *set_ids = (int32_t *)(A + o_sids);
        // the radix build where its buffers fit (the sampling scratch is free by
        // now; 12 bytes a member), else the counting build
        s = tune_value(IM_TUNE_INDEX_REPLICAS) == 0
                ? grow(&b->sscratch, &b->sscratch_bytes, radix_index_bytes(added, n_total))
                : IM_ERR_UNSUPPORTED;
        if (s == IM_OK)
            s = build_index_radix(set_off, members, sets_total, added, n_total, vtx_off, set_ids,
                                  (int32_t *)(A + o_cur), b->sscratch, st);
        else
            s = build_index_raw(set_off, members, sets_total, added, n_total, vtx_off, set_ids,
                                (int32_t *)(A + o_cur), 1, tmp, st);
        if (s != IM_OK) return s;
        // 4. seed selection: the plain queries in one launch, on groups of blocks
        int32_t *d_seeds = (int32_t *)(A + o_out);
        int64_t *d_gains = (int64_t *)(A + o_out + up256((size_t)nq * kmax * 4));
        int32_t *d_ns = (int32_t *)((char *)d_gains + up256((size_t)nq * kmax * 8));
        int64_t *d_cov = (int64_t *)((char *)d_ns + up256((size_t)nq * 4));
        std::vector<int64_t> hb(nq + 1);
        IM_CUDA(cudaMemcpyAsync(hb.data(), d_bounds, (size_t)(nq + 1) * 8, cudaMemcpyDeviceToHost, st));
        IM_CUDA(cudaStreamSynchronize(st));
        int *d_gstatus = (int *)(A + o_gbar);
        IM_CUDA(cudaMemsetAsync(d_gstatus, 0, sizeof(int), st));
        std::vector<GreedyQuery> gq;
        for (int32_t i = 0; i < nq; ++i) {
            if (qs[order[i]].cover.algo == IM_RANDGREEDI) continue;
            const BatchQuery &Q = bq[i];
            GreedyQuery g;
            g.n = Q.n;
            g.theta = Q.theta;
            g.members = hb[i + 1] - hb[i];
            g.vtx_off = vtx_off + Q.vbase;
            g.sshift = Q.sbase;
            g.vshift = Q.vbase;
            g.k = Q.k;
            g.counts = (int32_t *)(A + o_key) + Q.vbase;
            g.ranks = (int32_t *)(A + o_stamp) + Q.vbase;
            g.cands = (int32_t *)(A + o_cur) + Q.vbase;
            g.covered = (uint32_t *)(A + o_cov) + Q.cbase;
            g.seeds = d_seeds + Q.out * kmax;
            g.gains = d_gains + Q.out * kmax;
            g.nseeds = d_ns + Q.out;
            g.coverage = d_cov + Q.out;
            gq.push_back(g);
        }
        s = greedy_many(gq, set_off, members, set_ids, A + o_many, d_gstatus, st);
        if (s != IM_OK) return s;
        // RandGreedi queries: each on a view of the batch's index, with its own
        // set ids; the partition count picked by timing when the query leaves it open
        std::vector<int32_t> parts_used(nq, 0);
        for (int32_t i = 0; i < nq; ++i) {
            const BatchQuery &Q = bq[i];
            const im_query &q = qs[order[i]];
            if (q.cover.algo != IM_RANDGREEDI) continue;
            {
                KernelTimer kt(st, "batch_localize");
                k_localize<<<num_sms() * 4, 256, 0, st>>>(set_ids, vtx_off + Q.vbase, Q.n, Q.sbase);
            }
            IM_CUDA(cudaGetLastError());
            im_pool *&view = b->views[q.graph];
            if (!view) view = make_pool_view(q.graph, b->device);
            if (!view) return IM_ERR_OOM;
            view->theta = Q.theta;
            view->total = hb[i + 1] - hb[i];
            view->vtx_off = vtx_off + Q.vbase;
            view->set_ids = set_ids;
            view->index_valid = true;
            im_cover_opts o = q.cover;
            o.fused = 0;
            if (o.partitions == 0) {
                int32_t lg = 0;
                while (((int64_t)1 << (lg + 1)) <= Q.theta) ++lg;
                const auto key = std::make_tuple(q.graph, (int32_t)q.model, lg);
                auto it = b->rg_parts.find(key);
                if (it == b->rg_parts.end()) {
                    // time every candidate count (second of two runs) and keep the fastest
                    cudaEvent_t e0, e1;
                    IM_CUDA(cudaEventCreate(&e0));
                    IM_CUDA(cudaEventCreate(&e1));
                    float best = 0.f;
                    int32_t bestP = 0;
                    for (int32_t P : partition_candidates(Q.n)) {
                        o.partitions = P;
                        float ms = 0.f;
                        for (int rep = 0; rep < 2 && s == IM_OK; ++rep) {
                            cudaEventRecord(e0, st);
                            s = randgreedi(view, Q.k, &o, d_seeds + Q.out * kmax,
                                           d_gains + Q.out * kmax, d_ns + Q.out, d_cov + Q.out, st,
                                           d_gstatus);
                            cudaEventRecord(e1, st);
                            cudaEventSynchronize(e1);
                            cudaEventElapsedTime(&ms, e0, e1);
                        }
                        if (s != IM_OK) break;
                        if (bestP == 0 || ms < best) {
                            best = ms;
                            bestP = P;
                        }
                    }
                    cudaEventDestroy(e0);
                    cudaEventDestroy(e1);
                    if (s != IM_OK) return s;
                    it = b->rg_parts.emplace(key, bestP).first;
                }
                o.partitions = it->second;
            }
            s = randgreedi(view, Q.k, &o, d_seeds + Q.out * kmax, d_gains + Q.out * kmax,
                           d_ns + Q.out, d_cov + Q.out, st, d_gstatus);
            if (s != IM_OK) return s;
            parts_used[i] = o.partitions;
        }
        // 5. results
        std::vector<int32_t> hns(nq);
        std::vector<int64_t> hcov(nq);
        IM_CUDA(cudaMemcpyAsync(seeds, d_seeds, (size_t)nq * kmax * 4, cudaMemcpyDefault, st));
        if (gains) IM_CUDA(cudaMemcpyAsync(gains, d_gains, (size_t)nq * kmax * 8, cudaMemcpyDefault, st));
        IM_CUDA(cudaMemcpyAsync(hns.data(), d_ns, (size_t)nq * 4, cudaMemcpyDeviceToHost, st));
        IM_CUDA(cudaMemcpyAsync(hcov.data(), d_cov, (size_t)nq * 8, cudaMemcpyDeviceToHost, st));
        int gstatus = 0;
        IM_CUDA(cudaMemcpyAsync(&gstatus, d_gstatus, sizeof(int), cudaMemcpyDeviceToHost, st));
        IM_CUDA(cudaStreamSynchronize(st));
        if (gstatus != 0) return map_dev_status(gstatus, "im_solve_batch greedy");
        for (int32_t i = 0; i < nq; ++i) {
            const int32_t q = order[i];
            res[q].num_seeds = hns[q];
            res[q].status = IM_OK;
            res[q].coverage = hcov[q];
            res[q].entries = hb[i + 1] - hb[i];
            res[q].partitions = parts_used[i];
            res[q].reserved = 0;
            // the hint for the next batches with this graph and model
            const int64_t per = qs[q].theta ? (2 * (hb[i + 1] - hb[i]) + qs[q].theta - 1) / qs[q].theta : 1;
            auto &h = b->entry_hint[{qs[q].graph, qs[q].model}];
            h = std::max<int64_t>({h, per, 1});
        }
        (void)examined;
        return IM_OK;
    }
    set_error("im_solve_batch: RRR sets did not fit after growing the arena");
    return IM_ERR_CAPACITY;
}

}  // extern "C"
