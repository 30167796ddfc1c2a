// spread.cu -- forward simulation of the diffusion from a seed set (im_spread).
//
// The influence spread sigma(S) (Sec. 2) is the expected number of vertices
// the seeds activate; the paper judges the selected seeds by it (Sec. 4.1).
// Run r simulates the live-edge world of RRR sample r -- the same IC coins
// and LT picks the sampler uses -- forward from S by a BFS
// over out-edges (one block per run, level by level, each warp expanding 32
// queued vertices at a time).  Under LT a run stops where it would pass n / 8
// out-edges, and goes on from there or, where that is cheaper (pull_pays), is
// redone by k_spread_pull, which draws every vertex's pick once instead of once
// per in-edge from an activated vertex.
//   IC: in-edge e is live iff lane (e & 3) of Philox(r, e >> 2, e >> 34, coin
//       tag) is below w[e];
//   LT: in-edge e into v is live iff v's pick draw x = Philox(r, v, 0, pick
//       tag).x falls in [sum(e) - w[e], sum(e)), sum(e) being the running
//       in-weight sum of v up to and including e (the LT index's leaves), i.e.
//       iff e is the first in-edge whose running sum exceeds x.
// Because run r and RRR sample r share their world, the run's root is
// activated exactly when S meets RRR set r (the RIS identity).
#include <algorithm>
#include <mutex>

#include "internal.cuh"

namespace im {

namespace {

constexpr int kSpreadThreads = 512;

// Out-edge index: for every source u, one 16-byte record per out-edge
// {head v, in-CSR id e, w[e], lo(e)} where lo(e) is v's running in-weight sum
// before e (mod 2^32).  An LT draw x of v picks e iff (x - lo(e)) mod 2^32 <
// w[e]: with valid LT weights lo(e) + w[e] <= 2^32, so the difference wraps to
// at least 2^32 - lo(e) >= w[e] whenever x < lo(e).
__global__ void k_out_hist(const int32_t *in_src, int64_t m, int32_t *cnt) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&cnt[in_src[e]], 1);
}

__global__ void k_out_fill(const int64_t *in_off, const int32_t *in_src, const uint32_t *w,
                           int64_t n, const int64_t *out_off, int32_t *cursor, uint4 *out_rec) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t v = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); v < n;
         v += nw) {
        const int64_t b = in_off[v], e1 = in_off[v + 1];
        unsigned long long carry = 0;
        for (int64_t base = b; base < e1; base += 32) {
            const int64_t e = base + lane;
            const uint32_t we = e < e1 ? w[e] : 0u;
            const unsigned long long incl = warp_incl_scan<unsigned long long>(we, lane);
            if (e < e1) {
                const int32_t u = in_src[e];
                const int64_t pos = out_off[u] + atomicAdd(&cursor[u], 1);
                out_rec[pos] = make_uint4((uint32_t)v, (uint32_t)e, we,
                                          (uint32_t)(carry + incl - we));
            }
            carry += __shfl_sync(kFull, incl, 31);
        }
    }
}

// A run that k_spread stopped before a level: the first `tail` vertices it activated
// are in its row of the lot, the first `head` of them expanded, at the price of
// `done` out-edges.
struct Stopped {
    unsigned long long run, head, tail, done;
};

struct SpreadArgs {
    int64_t n;
    uint64_t seed;
    uint64_t first;
    int64_t runs;
    const int32_t *seeds;
    int32_t k;
    const int64_t *out_off;
    const uint4 *out_rec;
    uint32_t *vis;                    // [blocks][words]
    int64_t words;
    int32_t *queues;                  // [blocks][qcap]
    int64_t qcap;
    unsigned long long *work;
    unsigned long long *total;
    int64_t *activated;               // [runs] or null
    uint8_t *root_hit;                // [runs] or null
    int *status;
    int64_t first_new;                // work item w is stopped run again + w, and, past them
    unsigned long long again, nagain; // all (nagain), run first_new + w - nagain
    // LT: a run that would pass `budget` out-edges with its next level stops before it
    unsigned long long budget;
    Stopped *list;                    // [list_cap]
    unsigned long long list_cap;
    unsigned long long *nlist;        // how many (or more, where runs found no place)
    int32_t *lot;                     // [list_cap][lot_row], null: a stopped run is not gone on with
    int64_t lot_row;
    unsigned long long *pace;         // [2] out-edges of whole levels, and the blocks' ns for them (with a lot)
    unsigned long long from, to;      // k_spread_pull: the places it finishes
    unsigned long long *rest;         // ... and the out-edges they had left, or null
    QueryView view;                   // LT: the graph's pick tables
    int32_t *next;                    // [groups][n] k_spread_pull
    GridBarrier *bars;                // [groups]
    unsigned long long *left;         // [groups][4] per-round and result counters
    int32_t groups;
};

// One run per block: a level-synchronous BFS whose warps take 32 vertices
// of the current level at a time and append the vertices they activate to
// the block's queue (one atomic per warp and step).  LT: a run stops between two
// levels, when those so far and the next have more than a.budget out-edges.
template <bool LT>
__global__ void __launch_bounds__(kSpreadThreads) k_spread(const __grid_constant__ SpreadArgs a) {
    __shared__ unsigned long long s_run;
    __shared__ unsigned long long s_tail, s_cursor, s_edges, s_at;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *vis = a.vis + (int64_t)blockIdx.x * a.words;
    int32_t *q = a.queues + (int64_t)blockIdx.x * a.qcap;
    const uint32_t k0 = seed_lo(a.seed), k1 = seed_hi(a.seed);
    unsigned long long my_total = 0, my_edges = 0, my_ns = 0;
    for (;;) {
        if (threadIdx.x == 0) {
            s_run = atomicAdd(a.work, 1ull);
            s_tail = 0;
            s_edges = 0;
        }
        __syncthreads();
        unsigned long long i = s_run;
        long long head = 0;
        const bool again = LT && i < a.nagain;   // (block-uniform)
        if (again) {                         // go on with a stopped run
            const Stopped r = a.list[a.again + i];
            const int32_t *row = a.lot + (int64_t)(a.again + i) * a.lot_row;
            for (int64_t x = threadIdx.x; x < (int64_t)r.tail; x += kSpreadThreads) {
                const int32_t u = row[x];
                q[x] = u;
                atomicOr(&vis[u >> 5], 1u << (u & 31));
            }
            i = r.run;
            head = (long long)r.head;
            if (threadIdx.x == 0) s_tail = r.tail;
        } else {
            i = (unsigned long long)a.first_new + (i - a.nagain);
            if (i >= (unsigned long long)a.runs) break;
        }
        const uint32_t s = (uint32_t)(a.first + i);
        const uint64_t t_begin = LT && a.lot ? global_ns() : 0;
        // the seeds, each once
        if (warp == 0 && !again) {
            for (int32_t b = 0; b < a.k; b += 32) {
                bool fresh = false;
                int32_t u = -1;
                if (b + lane < a.k) {
                    u = a.seeds[b + lane];
                    if (u < 0 || u >= a.n) {
                        raise_status(a.status, kDevBadInput);
                        u = -1;
                    } else {
                        const uint32_t bit = 1u << (u & 31);
                        fresh = !(atomicOr(&vis[u >> 5], bit) & bit);
                    }
                }
                const unsigned fm = __ballot_sync(kFull, fresh);
                if (fresh) q[s_tail + __popc(fm & ((1u << lane) - 1u))] = u;
                __syncwarp();
                if (lane == 0) s_tail += __popc(fm);
                __syncwarp();
            }
        }
        __syncthreads();
        unsigned long long done = 0;         // out-edges of the levels before this one
        unsigned long long budget = LT ? a.budget : ~0ull;
        bool stop = false;                   // (block-uniform)
        for (;;) {
            const long long lvl_end = (long long)s_tail;
            if (head >= lvl_end) break;
            __syncthreads();                 // everyone has read s_tail
            if (threadIdx.x == 0) s_cursor = (unsigned long long)head;
            if (LT && budget != ~0ull) {           // the level's out-edges (the expansion finds what this reads in L1)
                unsigned long long e = 0;
                for (long long x = head + threadIdx.x; x < lvl_end; x += kSpreadThreads) {
                    const int32_t u = q[x];
                    e += (unsigned long long)(a.out_off[u + 1] - a.out_off[u]);
                }
                if (__any_sync(kFull, e != 0ull)) {
                    e = warp_sum<unsigned long long>(e);
                    if (lane == 0) atomicAdd(&s_edges, e);
                }
            }
            __syncthreads();
            if (LT && budget != ~0ull) {
                if (s_edges > budget) {      // (the levels' sum so far)
                    if (threadIdx.x == 0) {
                        s_at = atomicAdd(a.nlist, 1ull);
                    }
                    __syncthreads();
                    stop = s_at < a.list_cap;
                    if (stop) break;
                    budget = ~0ull;          // no place in the list
                }
                done = s_edges;
            }
            for (;;) {
                long long base = 0;
                if (lane == 0) base = (long long)atomicAdd(&s_cursor, 32ull);
                base = __shfl_sync(kFull, base, 0);
                if (base >= lvl_end) break;
                const int nb = (int)(lvl_end - base < 32 ? lvl_end - base : 32);
                int64_t ob = 0, oe = 0;
                if (lane < nb) {
                    const int32_t u = q[base + lane];
                    ob = a.out_off[u];
                    oe = a.out_off[u + 1];
                }
                const int64_t len = oe - ob;
                const int64_t incl = warp_incl_scan<int64_t>(len, lane);
                const int64_t total = __shfl_sync(kFull, incl, 31);
                for (int64_t eb = 0; eb < total; eb += 32) {
                    const int64_t t = eb + lane;
                    int owner = 0;   // first lane whose inclusive count exceeds t
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1) {
                        const int64_t c = __shfl_sync(kFull, incl, owner + step - 1);
                        if (c <= t) owner += step;
                    }
                    const int64_t o_incl = __shfl_sync(kFull, incl, owner);
                    const int64_t o_len = __shfl_sync(kFull, len, owner);
                    const int64_t o_ob = __shfl_sync(kFull, ob, owner);
                    bool fresh = false;
                    uint32_t v = 0;
                    if (t < total) {
                        const uint4 r = __ldg(a.out_rec + o_ob + (t - (o_incl - o_len)));
                        v = r.x;
                        if (!((__ldcg(vis + (v >> 5)) >> (v & 31)) & 1u)) {
                            bool live;
                            if (!LT) {
                                const uint32_t e = r.y;   // in-CSR id (< 2^31)
                                const uint4 c = philox4x32_10(
                                    make_uint4(s, e >> 2, 0u, kStreamCoin), k0, k1);
                                const int ln = (int)(e & 3);
                                const uint32_t coin =
                                    ln == 0 ? c.x : ln == 1 ? c.y : ln == 2 ? c.z : c.w;
                                live = coin < r.z;
                            } else {
                                const uint32_t x =
                                    philox4x32_10(make_uint4(s, v, 0u, kStreamPick), k0, k1).x;
                                live = x - r.w < r.z;
                            }
                            if (live) {
                                const uint32_t bit = 1u << (v & 31);
                                fresh = !(atomicOr(&vis[v >> 5], bit) & bit);
                            }
                        }
                    }
                    const unsigned fm = __ballot_sync(kFull, fresh);
                    if (fm) {
                        long long at = 0;
                        if (lane == 0) at = (long long)atomicAdd(&s_tail, (unsigned long long)__popc(fm));
                        at = __shfl_sync(kFull, at, 0);
                        if (fresh) q[at + __popc(fm & ((1u << lane) - 1u))] = (int32_t)v;
                    }
                }
            }
            __syncthreads();
            head = lvl_end;
        }
        const long long tail = (long long)s_tail;
        if (LT && a.lot) {
            my_edges += stop ? done : s_edges;
            my_ns += global_ns() - t_begin;
        }
        if (LT && stop) {
            if (threadIdx.x == 0)
                a.list[s_at] = Stopped{i, (unsigned long long)head, (unsigned long long)tail, done};
            if (a.lot) {
                int32_t *row = a.lot + (int64_t)s_at * a.lot_row;
                for (int64_t x = threadIdx.x; x < tail; x += kSpreadThreads) row[x] = q[x];
            }
        }
        if (!stop && threadIdx.x == 0) {
            const uint32_t root = rrr_root(a.seed, s, (uint32_t)a.n);
            const bool hit = (vis[root >> 5] >> (root & 31)) & 1u;
            if (a.activated) a.activated[i] = tail;
            if (a.root_hit) a.root_hit[i] = hit ? 1 : 0;
            my_total += (unsigned long long)tail;
        }
        __syncthreads();
        // clear this run's visited bits
        if (tail > a.words) {
            for (int64_t x = threadIdx.x; x < a.words; x += blockDim.x) vis[x] = 0u;
        } else {
            for (int64_t x = threadIdx.x; x < tail; x += blockDim.x) vis[q[x] >> 5] = 0u;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && my_total) atomicAdd(a.total, my_total);
    if (LT && threadIdx.x == 0 && my_edges) {
        atomicAdd(a.pace, my_edges);
        atomicAdd(a.pace + 1, my_ns);
    }
}

// The source that vertex v picks in sample s (draw x), or -1: the rules of the LT
// sampler over its tables (equal in-weights by the record's reciprocal, else the
// cut point and, past it, a search of doubling stride in the running sums).
__device__ __forceinline__ int32_t lt_pick_source(const QueryView &V, uint32_t v, uint32_t x) {
    const uint4 vr = __ldg(V.lt_vrec + v);
    const uint32_t d = vr.y;
    if (vr.w != 0u) {
        uint32_t e = __umulhi(x, vr.z), rem = x - e * vr.w;
        if (rem >= vr.w) { ++e; rem -= vr.w; }
        if (rem >= vr.w) ++e;
        return e < d ? __ldg(V.in_src + vr.x + e) : -1;
    }
    if (d == 0u) return -1;
    const uint4 gv = __ldg(V.lt_guide + vr.x + __umulhi(x, d));
    if ((unsigned long long)x < (((unsigned long long)gv.y << 32) | gv.x)) return (int32_t)gv.z;
    const unsigned long long *leaf = V.lt_leaf + vr.x;
    uint32_t lo = gv.w + 1, hi = d, stride = 1;
    unsigned long long at = 0;
    while (lo < hi) {
        const uint32_t p = hi < d ? (lo + hi) >> 1 : min(lo + stride - 1u, d - 1u);
        const unsigned long long r = __ldg(leaf + p);
        if ((unsigned long long)x < (r >> 31)) {
            hi = p;
            at = r;
        } else {
            lo = p + 1;
        }
        stride <<= 1;
    }
    return hi < d ? (int32_t)(at & 0x7fffffffull) : -1;
}

// LT runs that activate a large part of the graph.  In an LT world every vertex
// keeps at most one in-edge, so the world is one pointer a vertex, and v is
// activated iff its chain of pointers reaches a seed.  A group of blocks draws
// the n pointers of a run (next[v]: the pick; -1: a seed; -2: nothing picked),
// then lets every pointer jump to where its target points until no more chain
// ends at a seed or at nothing; what is still unresolved runs into a cycle.  (A
// round with an unresolved chain that ends always resolves one: the unresolved
// vertex nearest its end points at a resolved one.)  Concurrent jumps only ever
// shorten chains, so rounds work in place.
// n draws and about ten rounds of n gathers in L2 instead of a draw per out-edge
// of an activated vertex (1.5 x 10^7 of 1.7 x 10^7 at scale 20 from 100 of the
// largest vertices): a call of 256 runs 76 -> 4.6 ms.  The groups' pointers together
// stay below kPullBytes, so that the gathers hit L2.
constexpr int kPullThreads = 1024;
constexpr int64_t kPullBytes = 64ll << 20;
constexpr int kPullU = 4;                    // gathers in flight per thread

__global__ void __launch_bounds__(kPullThreads) k_spread_pull(const __grid_constant__ SpreadArgs a) {
    __shared__ unsigned long long s_cnt[kPullThreads / 32];
    const int group = blockIdx.x % a.groups;             // blocks of a group on different SMs
    const uint32_t rank = blockIdx.x / a.groups, nb = (gridDim.x - group + a.groups - 1) / a.groups;
    int32_t *next = a.next + (int64_t)group * a.n;
    GridBarrier *bar = a.bars + group;
    unsigned long long *left = a.left + 4 * group;       // [0], [1] resolved in a round, [2] activated, [3] their out-edges
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tid = (int64_t)rank * kPullThreads + threadIdx.x, stride = (int64_t)nb * kPullThreads;
    const uint32_t k0 = seed_lo(a.seed), k1 = seed_hi(a.seed);
    // adds the block's counts to *to
    auto block_add = [&](unsigned int mine, unsigned long long *to) {
        mine = __reduce_add_sync(kFull, mine);
        if (lane == 0) s_cnt[warp] = mine;
        __syncthreads();
        if (warp == 0) {
            const unsigned long long t = warp_sum<unsigned long long>(s_cnt[lane]);
            if (lane == 0 && t) atomicAdd(to, t);
        }
        __syncthreads();
    };
    for (unsigned long long i = a.from + group; i < a.to; i += a.groups) {
        const unsigned long long run = a.list[i].run;
        const uint32_t s = (uint32_t)(a.first + run);
        for (int64_t v = tid; v < a.n; v += stride) {
            const int32_t u = lt_pick_source(
                a.view, (uint32_t)v, philox4x32_10(make_uint4(s, (uint32_t)v, 0u, kStreamPick), k0, k1).x);
            next[v] = u >= 0 ? u : -2;
        }
        if (tid == 0) left[0] = left[1] = left[2] = left[3] = 0ull;
        if (!grid_sync(bar, nb, a.status)) return;
        for (int64_t b = tid; b < a.k; b += stride) next[a.seeds[b]] = -1;
        if (!grid_sync(bar, nb, a.status)) return;
        for (int round = 0;; ++round) {
            unsigned int resolved = 0;
            for (int64_t v0 = tid; v0 < a.n; v0 += stride * kPullU) {
                int32_t p[kPullU], q[kPullU];
#pragma unroll
                for (int u = 0; u < kPullU; ++u) {
                    const int64_t v = v0 + u * stride;
                    p[u] = v < a.n ? __ldcg(next + v) : -1;
                }
#pragma unroll
                for (int u = 0; u < kPullU; ++u) q[u] = p[u] >= 0 ? __ldcg(next + p[u]) : 0;
#pragma unroll
                for (int u = 0; u < kPullU; ++u)
                    if (p[u] >= 0) {
                        next[v0 + u * stride] = q[u];
                        resolved += q[u] < 0;
                    }
            }
            block_add(resolved, left + (round & 1));
            if (!grid_sync(bar, nb, a.status)) return;
            const unsigned long long any = *(volatile unsigned long long *)(left + (round & 1));
            // (the other counter's last readers passed the barrier above)
            if (tid == 0) left[(round + 1) & 1] = 0ull;
            if (any == 0ull) break;
            if (!grid_sync(bar, nb, a.status)) return;
        }
        unsigned int act = 0;
        unsigned long long edges = 0;
        for (int64_t v = tid; v < a.n; v += stride)
            if (__ldcg(next + v) == -1) {
                ++act;
                if (a.rest) edges += (unsigned long long)(a.out_off[v + 1] - a.out_off[v]);
            }
        block_add(act, left + 2);
        if (a.rest) {
            edges = warp_sum<unsigned long long>(edges);
            if (lane == 0 && edges) atomicAdd(left + 3, edges);
        }
        if (!grid_sync(bar, nb, a.status)) return;
        if (tid == 0) {
            const unsigned long long t = *(volatile unsigned long long *)(left + 2);
            const uint32_t root = rrr_root(a.seed, s, (uint32_t)a.n);
            if (a.activated) a.activated[run] = (int64_t)t;
            if (a.root_hit) a.root_hit[run] = __ldcg(next + root) == -1 ? 1 : 0;
            atomicAdd(a.total, t);
            if (a.rest) a.rest[i] = *(volatile unsigned long long *)(left + 3) - a.list[i].done;
        }
        if (!grid_sync(bar, nb, a.status)) return;       // before next and left are rewritten
    }
}

constexpr int64_t kPullList = 1 << 20;        // runs listed to be pulled at most

// Whether `count` stopped runs cost less to pull than to push to their end, from the
// out-edges `rest` that the first of them turned out to have left (the runs of a call
// differ in their random worlds alone) and the pace (out-edges, ns) of the blocks.
// Neither n, m nor a run's past tells: stopped before 131,072 out-edges at scale 20,
// runs from 100 of the largest vertices have 1.4 x 10^7 left at 16 out-edges a vertex,
// and 2.5 x 10^5 at 2 and U[0, 0.1] weights, where pulling all of 3,000 runs took 60
// ms and pushing them takes 34.
//   pulling  1 us + 16 ps a vertex of the whole GPU a run (17 us at scale 20; pointers
//            beyond the L2 cache are gathered from DRAM, at a sixteenth of the rate),
//            and 100 us for the launch;
//   pushing  at the blocks' pace, at most 6 x 10^10 out-edges a second together, and
//            the longest run at a block's.  That lies between a warp's, 2.4 x 10^7 (it
//            expands a hub, and any 32 vertices, alone), and 3 x 10^8.  Where nothing was
//            measured, every run having stopped at its first level, it is that of the
//            warps which that level (run `one`) keeps busy.  The longest run slows
//            down by half as it comes to the hubs.
bool pull_pays(const std::vector<unsigned long long> &rest, double count, int64_t n,
               const unsigned long long *pace, const Stopped &one, int64_t blocks) {
    double sum = 0.0, most = 0.0;
    for (const unsigned long long r : rest) {
        sum += (double)r;
        most = std::max(most, (double)r);
    }
    const double block = pace[1] ? (double)pace[0] * 1e9 / (double)pace[1]         // out-edges a second
                                 : std::min(3e8, 2.4e7 * (double)((one.tail - one.head + 31) / 32));
    const double push = std::max(count * sum / (double)rest.size() / std::min(6e10, block * (double)blocks),
                                 1.5 * most / block);
    const double pull = 1e-4 + count * (1e-6 + 16e-12 * (double)n * (n * 4 <= kPullBytes ? 1.0 : 16.0));
    return pull < push;
}

std::mutex g_out_index_mu;   // graphs are shared between threads

im_status build_out_index(im_graph *g, cudaStream_t st) {
    std::lock_guard<std::mutex> lk(g_out_index_mu);
    if (g->out_off) return IM_OK;   // set only once the whole index is built
    const int64_t n = g->n, m = g->m;
    // the index: handed to g once complete, freed on any failure
    struct Parts {
        int64_t *off = nullptr;
        uint4 *rec = nullptr;
        ~Parts() {
            if (off || rec) {
                cudaDeviceSynchronize();
                cudaFree(off);
                cudaFree(rec);
            }
        }
    } t;
    CallBuf cnt_buf(st), scan_buf(st);
    IM_TRY(cnt_buf.alloc((size_t)n * 4));
    IM_TRY(scan_buf.alloc(scan_tmp_bytes(n)));
    int32_t *cnt = cnt_buf.as<int32_t>();
    IM_CUDA(cudaMalloc(&t.off, (size_t)(n + 1) * 8));
    IM_CUDA(cudaMalloc(&t.rec, (size_t)std::max<int64_t>(m, 1) * sizeof(uint4)));
    IM_CUDA(cudaMemsetAsync(cnt, 0, (size_t)n * 4, st));
    {
        KernelTimer kt(st, "out_index");
        if (m > 0) k_out_hist<<<num_sms() * 4, 256, 0, st>>>(g->in_src, m, cnt);
    }
    IM_CUDA(cudaGetLastError());
    IM_TRY(exclusive_scan_i32_to_i64(cnt, t.off, n, nullptr, scan_buf.as<void>(), scan_tmp_bytes(n), st));
    IM_CUDA(cudaMemsetAsync(cnt, 0, (size_t)n * 4, st));
    {
        KernelTimer kt(st, "out_index");
        if (m > 0)
            k_out_fill<<<num_sms() * 8, 256, 0, st>>>(g->in_off, g->in_src, g->w, n, t.off,
                                                      cnt, t.rec);
    }
    IM_CUDA(cudaGetLastError());
    IM_CUDA(cudaStreamSynchronize(st));
    g->out_rec = t.rec;
    g->out_off = t.off;
    t.off = nullptr;
    t.rec = nullptr;
    return IM_OK;
}

}  // namespace

}  // namespace im

using namespace im;

extern "C" im_status im_spread(const im_graph *gc, im_model model, const int32_t *seeds, int32_t k,
                               uint64_t seed, uint64_t first_run, uint64_t runs, int64_t *activated,
                               uint8_t *root_hit, int64_t *total, void *stream) {
    if (!gc || k < 0 || (k > 0 && !seeds) || (model != IM_IC && model != IM_LT) ||
        first_run + runs > (1ull << 32) || runs > (1ull << 32)) {
        set_error("im_spread: bad arguments");
        return IM_ERR_INVALID_ARG;
    }
    im_graph *g = const_cast<im_graph *>(gc);
    DeviceGuard dg(g->device);
    cudaStream_t st = as_stream(stream);
    if (model == IM_LT) {
        IM_TRY(build_lt_index(g, st));
        if (!g->lt_valid) {
            set_error("im_spread: LT needs every vertex's in-weights to sum to at most 2^32");
            return IM_ERR_INVALID_ARG;
        }
    }
    IM_TRY(build_out_index(g, st));
    if (total) *total = 0;
    if (runs == 0) return IM_OK;
    const int64_t n = g->n, words = (n + 31) / 32;
    // blocks (one run each at a time): occupancy-sized, and the per-block
    // queue (n entries) and bitmap within about 2 GB
    int per_sm = 0;
    const void *kern = model == IM_LT ? (const void *)k_spread<true> : (const void *)k_spread<false>;
    IM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSpreadThreads, 0));
    // LT: runs stop here before they pass this many out-edges (see pull_pays)
    const int64_t budget = std::max<int64_t>(n / 8, 1 << 16);
    bool pull = model == IM_LT && g->m > budget;
    int pull_grid = 0;
    if (pull) {
        int per = 0;
        IM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_spread_pull, kPullThreads, 0));
        pull_grid = per * num_sms();
        pull = per > 0;
    }
    const int64_t per_block = n * 4 + words * 4;
    int64_t blocks = std::max(1, per_sm) * (int64_t)num_sms();
    blocks = std::min<int64_t>(blocks, std::max<int64_t>(1, (2ll << 30) / per_block));
    blocks = std::min<int64_t>(blocks, (int64_t)runs);
    const int64_t groups = std::max<int64_t>(
        1, std::min<int64_t>({blocks, (int64_t)pull_grid / 4, kPullBytes / (n * 4)}));
    // LT: the runs that find room in a lot of 1 GB if they stop, which tell how to go on
    // with the others; what a run activates before it stops is bounded by the budget
    const int64_t lot_row = std::min<int64_t>(n, budget + k);
    int64_t head_runs = std::min<int64_t>((int64_t)runs, std::max<int64_t>(1, (1ll << 30) / (lot_row * 4)));
    CallBuf lot(st);
    if (pull && lot.alloc((size_t)head_runs * lot_row * 4) != IM_OK) pull = false;
    if (!pull) head_runs = (int64_t)runs;
    const int64_t list = pull ? std::max(head_runs, std::min<int64_t>((int64_t)runs - head_runs, kPullList)) : 0;
    const int64_t qcap = pull ? lot_row : n;
    const bool host_act = activated && !is_device_ptr(activated);
    const bool host_hit = root_hit && !is_device_ptr(root_hit);
    const bool host_seeds = k > 0 && !is_device_ptr(seeds);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t at = off;
        off += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t o_ctr = take(6 * 8), o_seeds = take((size_t)std::max(k, 1) * 4),
                 o_vis = take((size_t)blocks * words * 4), o_q = take((size_t)blocks * qcap * 4),
                 o_act = take(host_act ? (size_t)runs * 8 : 0),
                 o_hit = take(host_hit ? (size_t)runs : 0),
                 o_list = take((size_t)list * sizeof(Stopped)),
                 o_rest = take(pull ? (size_t)groups * 8 : 0),
                 o_bars = take(pull ? (size_t)groups * sizeof(GridBarrier) : 0),
                 o_left = take(pull ? (size_t)groups * 4 * 8 : 0);
    CallBuf buf(st), next(st), queues(st);
    IM_TRY(buf.alloc(off));
    char *B = buf.as<char>();
    IM_CUDA(cudaMemsetAsync(B + o_ctr, 0, 6 * 8, st));
    IM_CUDA(cudaMemsetAsync(B + o_vis, 0, (size_t)blocks * words * 4, st));
    if (k > 0) IM_CUDA(cudaMemcpyAsync(B + o_seeds, seeds, (size_t)k * 4, cudaMemcpyDefault, st));
    SpreadArgs a;
    a.n = n;
    a.seed = seed;
    a.first = first_run;
    a.runs = head_runs;
    a.seeds = (const int32_t *)(B + o_seeds);
    a.k = k;
    a.out_off = g->out_off;
    a.out_rec = g->out_rec;
    a.vis = (uint32_t *)(B + o_vis);
    a.words = words;
    a.queues = (int32_t *)(B + o_q);
    a.qcap = qcap;
    unsigned long long *ctr = (unsigned long long *)(B + o_ctr);
    a.work = ctr;
    a.total = ctr + 1;
    a.status = (int *)(ctr + 2);
    a.nlist = ctr + 3;
    a.pace = ctr + 4;
    a.first_new = 0;
    a.again = a.nagain = 0;
    a.budget = pull ? (unsigned long long)budget : ~0ull;
    a.list = (Stopped *)(B + o_list);
    a.list_cap = (unsigned long long)head_runs;
    a.lot = pull ? lot.as<int32_t>() : nullptr;
    a.lot_row = lot_row;
    a.from = a.to = 0;
    a.rest = nullptr;
    a.view = query_view(g, seed, first_run);
    a.next = nullptr;
    a.bars = (GridBarrier *)(B + o_bars);
    a.left = (unsigned long long *)(B + o_left);
    a.groups = 0;
    a.activated = host_act ? (int64_t *)(B + o_act) : activated;
    a.root_hit = host_hit ? (uint8_t *)(B + o_hit) : root_hit;
    unsigned long long hc[6] = {0, 0, 0, 0, 0, 0};
    auto pull_runs = [&](unsigned long long from, unsigned long long to, unsigned long long *rest) -> im_status {
        a.from = from;
        a.to = to;
        a.rest = rest;
        a.groups = (int32_t)std::min<unsigned long long>(groups, to - from);
        IM_CUDA(cudaMemsetAsync(B + o_bars, 0, (size_t)groups * sizeof(GridBarrier), st));
        void *args[] = {&a};
        KernelTimer kt(st, "spread_lt");
        IM_CUDA(cudaLaunchCooperativeKernel((const void *)k_spread_pull, dim3(pull_grid),
                                            dim3(kPullThreads), args, 0, st));
        return IM_OK;
    };
    auto push_runs = [&]() -> im_status {
        KernelTimer kt(st, model == IM_LT ? "spread_lt" : "spread_ic");
        if (model == IM_LT) k_spread<true><<<(unsigned)blocks, kSpreadThreads, 0, st>>>(a);
        else k_spread<false><<<(unsigned)blocks, kSpreadThreads, 0, st>>>(a);
        IM_CUDA(cudaGetLastError());
        return IM_OK;
    };
    auto read_counters = [&]() -> im_status {
        IM_CUDA(cudaMemcpyAsync(hc, ctr, sizeof(hc), cudaMemcpyDeviceToHost, st));
        IM_CUDA(cudaStreamSynchronize(st));
        return IM_OK;
    };
    auto dev_ok = [&] { return (int)(hc[2] & 0xffffffffu) == kDevOk; };
    IM_TRY(push_runs());
    if (pull) {
        IM_TRY(read_counters());
        const unsigned long long stopped = hc[3];        // (every one has its place in the list)
        const int64_t later = (int64_t)runs - head_runs;
        if (dev_ok() && (stopped > 0 || later > 0)) {
            // the first of them are pulled in any case (no room for their pointers: none is)
            unsigned long long pulled = 0;
            bool push = next.alloc((size_t)groups * n * 4) != IM_OK;
            a.next = next.as<int32_t>();
            if (stopped > 0 && !push) {
                pulled = std::min<unsigned long long>(stopped, groups);
                IM_TRY(pull_runs(0, pulled, (unsigned long long *)(B + o_rest)));
                if (later > 0 || stopped > 2 * pulled) {
                    std::vector<unsigned long long> rest(pulled);
                    IM_CUDA(cudaMemcpyAsync(rest.data(), B + o_rest, pulled * 8, cudaMemcpyDeviceToHost, st));
                    Stopped one;
                    IM_CUDA(cudaMemcpyAsync(&one, a.list, sizeof(one), cudaMemcpyDeviceToHost, st));
                    IM_CUDA(cudaStreamSynchronize(st));
                    const double count = (double)(stopped - pulled) + (double)stopped * later / head_runs;
                    push = !pull_pays(rest, count, n, hc + 4, one, blocks);
                }
                if (!push && stopped > pulled) {
                    IM_TRY(pull_runs(pulled, stopped, nullptr));
                    pulled = stopped;
                }
            }
            if (pulled < stopped || later > 0) {
                // push on the runs that still wait, then the later ones: to their end,
                // or until they stop (for good, to be pulled)
                IM_CUDA(cudaMemsetAsync(a.work, 0, 8, st));
                IM_CUDA(cudaMemsetAsync(a.nlist, 0, 8, st));
                a.again = pulled;
                a.nagain = stopped - pulled;
                a.first_new = head_runs;
                a.runs = (int64_t)runs;
                if (push) a.budget = ~0ull;
                else a.lot = nullptr;
                a.list_cap = (unsigned long long)list;
                if (push || later > list) {              // runs that do not stop
                    while (queues.alloc((size_t)blocks * n * 4) != IM_OK) {
                        if (blocks == 1) return IM_ERR_OOM;
                        blocks /= 2;
                    }
                    a.queues = queues.as<int32_t>();
                    a.qcap = n;
                }
                IM_TRY(push_runs());
                if (!push) {
                    IM_TRY(read_counters());
                    if (hc[3] > 0 && dev_ok()) IM_TRY(pull_runs(0, std::min(hc[3], a.list_cap), nullptr));
                }
            }
        }
    }
    IM_CUDA(cudaMemcpyAsync(hc, ctr, sizeof(hc), cudaMemcpyDeviceToHost, st));
    if (host_act) IM_CUDA(cudaMemcpyAsync(activated, B + o_act, (size_t)runs * 8, cudaMemcpyDeviceToHost, st));
    if (host_hit) IM_CUDA(cudaMemcpyAsync(root_hit, B + o_hit, (size_t)runs, cudaMemcpyDeviceToHost, st));
    IM_CUDA(cudaStreamSynchronize(st));
    (void)host_seeds;
    const int dev_status = (int)(hc[2] & 0xffffffffu);
    if (dev_status != kDevOk) {
        if (dev_status == kDevBadInput) {
            set_error("im_spread: a seed id is outside [0, n)");
            return IM_ERR_INVALID_ARG;
        }
        return map_dev_status(dev_status, "im_spread");
    }
    if (total) *total = (int64_t)hc[1];
    return IM_OK;
}
