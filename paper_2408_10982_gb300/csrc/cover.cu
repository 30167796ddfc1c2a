// cover.cu -- max-k-cover over the pool: standard greedy (Sec. 3.2) and
// RandGreedi with streaming aggregation and truncation (Alg. 4, Alg. 5,
// Sec. 3.3.2).
//
// Standard greedy: one cooperative persistent kernel runs all k steps.  A step
// is a grid-wide argmax over the marginal gains counts[v] (packed as
// gain << 32 | ~v so that ties go to the smallest id), a grid barrier, the
// cover of S(v*) (atomicOr on a theta-bit bitmap; every newly covered set
// decrements the gains of its members), and a second barrier (a third after
// sets that were cut into pieces).  Barriers wait
// at most kWaitLimitNs and then report IM_ERR_TIMEOUT.
//
// RandGreedi: the paper's m sender machines are m "producer" blocks, each
// running the lazy local greedy of one vertex part V_p (Alg. 2) with its
// gains in shared memory and its own theta-bit covered bitmap.  A producer
// publishes its j-th seed (j < ceil(alpha k)) in slot (j, p) of a device array
// and raises a release flag; the buckets consume the slots in (j, p) order, so
// they see the same stream order in every run.  The receiver's B bucketing
// threads become, after the producers finish, k_rg_stream_small (a block per
// bucket: short streams, or more than 64 buckets) or k_rg_stream_masks: one
// 64-bit mask per RRR set holds the buckets covering it, so one pass over a
// streamed subset counts its gain for every bucket.  Alternatives (tuning
// knob values): one "consumer" block or thread-block cluster per bucket, and
// a fused mode where producers and consumers are one cooperative launch and
// the consumers read the slots with acquire loads as they are published, the
// paper's streaming overlap.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "internal.cuh"

namespace cg = cooperative_groups;

namespace im {

namespace {

constexpr int kGreedyThreads = 512;
constexpr int kRGThreads = 512;
constexpr int kProdThreads = 1024;           // producer blocks of the two-launch mode, at most
constexpr int kProdMinThreads = 512;         // ... and at least (64 a candidate, see scan_ids)
constexpr size_t kProdSmemCap = 200 * 1024;  // their keys, and what fits beside them
constexpr size_t kProdInfoCap = 56 * 1024;   // keys and subsets beside a bitmap in global memory
constexpr int kBatch = 256;                  // stream slots a consumer reads at once
constexpr int kUnroll = 8;                   // independent loads in flight per lane in scans
constexpr int kSpec = 32;                    // largest speculative group of stream elements
constexpr size_t kClusterSmemCap = 200 * 1024;  // bucket bitmap slice per block
constexpr int kMaskG = 64;                   // largest group of stream slots (mask stage)
constexpr int kMaskWindow = 512;             // ... slots read ahead (mask stage)
constexpr int kMaskStrips = 16;              // entries per lane in one warp work item
constexpr int kMaskItem = 32 * kMaskStrips;  // entries per warp work item

// The largest of a warp's values, by 32-bit reductions.
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long v) {
    const uint32_t hi = __reduce_max_sync(kFull, (uint32_t)(v >> 32));
    const uint32_t lo = __reduce_max_sync(kFull, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
    return (unsigned long long)hi << 32 | lo;
}

__device__ __forceinline__ unsigned long long block_max_u64(unsigned long long v,
                                                            unsigned long long *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_max_u64(v);
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    if (warp == 0) {
        unsigned long long x = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0ull;
        x = warp_max_u64(x);
        if (lane == 0) sh[32] = x;
    }
    __syncthreads();
    const unsigned long long r = sh[32];
    __syncthreads();
    return r;
}

// Calls f(id) for every entry of ids[off, off + len) with 16-byte vector
// loads for the aligned body (each thread keeps U of them in flight) and
// scalar loads for the unaligned head and tail; f gets -1 for padding.
// Every thread of the calling group (tid < nth, nth >= 64) must call it.
template <int U, typename F>
__device__ __forceinline__ void scan_ids(const int32_t *__restrict__ ids, int64_t off, int64_t len,
                                         int tid, int nth, F &&f) {
    const int64_t end = off + len;
    int64_t a4 = (off + 3) & ~(int64_t)3;
    if (a4 > end) a4 = end;
    const int64_t b4 = a4 + ((end - a4) & ~(int64_t)3);
    if (tid < a4 - off) f(__ldg(ids + off + tid));
    else if (tid >= 32 && tid - 32 < end - b4) f(__ldg(ids + b4 + (tid - 32)));
    const int4 *v = reinterpret_cast<const int4 *>(ids + a4);
    const int64_t n4 = (b4 - a4) >> 2;
    for (int64_t i = tid; i < n4; i += (int64_t)nth * U) {
        int4 w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t k = i + (int64_t)u * nth;
            w[u] = k < n4 ? __ldg(v + k) : make_int4(-1, -1, -1, -1);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            f(w[u].x);
            f(w[u].y);
            f(w[u].z);
            f(w[u].w);
        }
    }
}

// ---------------------------------------------------------------------------
// standard greedy
// ---------------------------------------------------------------------------
struct GreedyArgs {
    int64_t n, theta;
    const int64_t *set_off;
    const int32_t *members;
    const int64_t *vtx_off;
    const int32_t *set_ids;
    int32_t k;
    int32_t *counts;                    // [n], or [32 ceil(n/32)] with spread
    uint32_t *covered;                  // [ceil(theta/32)]
    unsigned long long *gmax;           // [3] best key of a round
    GridBarrier *bar;
    int32_t *seeds;
    int64_t *gains;
    int32_t *nseeds;
    int64_t *coverage;
    int *status;
    // a query inside a batch: set ids in set_ids and vertex ids in members are
    // offset by sshift and vshift (the query's first set and first vertex)
    int64_t sshift, vshift;
    // ---- optional (NULL / 0: off), used by the pool's own greedy --------------
    // counts spread over 32 ceil(n / 32) slots: vertex v at (v mod 32) L + v / 32
    int32_t spread;
    // hubs, |S(v)| >= max |S(v)| >> hub_shift (at most hub_cap): each keeps its
    // gain as kHubRep partial counts, decremented by set id mod kHubRep
    int32_t *hub_rank;                  // [n] row of a hub, or -1
    int32_t *hub_cnt;                   // [hub_cap][kHubRep]
    int32_t *hub_list;                  // [hub_cap] the vertex of each row
    int32_t *cand;                      // [n] the other vertices with |S(v)| >= tau
    int32_t *ctl;                       // [4] hub rows, candidates, max |S(v)|, 0
    int32_t hub_cap, hub_shift, cand_shift;
    unsigned long long *work;           // [2] per-step chunk counters
    // pieces of long newly covered sets: first member << 16 | members << 5 | set
    // id mod 32, and how many this step has
    unsigned long long *piece;          // [2 T / kGreedyPiece + 1]
    unsigned long long *npiece;         // [1]
};

constexpr int kHubRep = 32;             // partial counts of a hub (one per set id mod 32)
// Entries of S(v*) a warp takes at a time: its share of the list, at least one
// (a newly covered set can hold hundreds of members, and the step waits for the
// slowest warp) and at most kGreedyChunk, beyond which lists are claimed from a
// counter.  Always claiming 16: 4,096 sets of 200 members (scale 10) .266 against
// .190 ms, IMM's greedy calls 19.3 against 14.7, 4.2 M LT walks 3.62 against
// 3.50; claiming half or an eighth of a share at a time: the claims, atomics on
// one word, cost .7 and 2.7 ms on the LT walks.
constexpr int kGreedyChunk = 16;
constexpr int64_t kGreedyTake = 1 << 26;  // members of a set walked at a time
// A newly covered set longer than this is put aside in pieces of this many
// members, which the whole grid shares after the claims of the step: the
// percolating sets of equal-probability IC hold 10^4 to 10^6 members each, and
// the ~100 warps that claim S(v*) would walk them alone (4,096 sets of U[0, 0.1]
// at scale 20, 1.1 x 10^8 members: 42.1 -> 1.9 ms; no change where sets are
// short).
constexpr int kGreedyPiece = 1024;
constexpr int kHubCap = 4096;           // hub rows at most
constexpr int kHubShift = 6;            // hubs: |S(v)| >= max |S(v)| / 64

// Standard greedy (Sec. 3.2), all k steps in one cooperative launch: a step
// takes the argmax of the gains (packed gain << 32 | ~v: ties to the smallest
// id), covers S(v*) on the theta-bit bitmap and decrements the gain of every
// member of every newly covered set; two grid barriers per step, three where it
// put pieces of long sets aside.
//
// On graphs with hubs most decrements land on a few vertices, and atomics on
// one address serialise in its L2 slice: with hub rows, a hub's gain is the
// sum of kHubRep partial counts, each taking the decrements of the sets whose
// id is that value mod kHubRep, and the spread layout puts the other
// high-degree vertices -- low ids on a degree-ordered graph -- in different
// cache lines.  The argmax reads only the hub rows and the candidate list
// (|S(v)| >= tau) while the best gain is at least tau, since every other
// gain is below |S(v)| < tau; those vertices are frozen -- not decremented,
// keeping |S(v)| as a stale bound -- which skips most decrements (low-degree
// vertices are most members).  Once the best gain falls below tau, one pass
// makes the frozen gains exact and every step reads all.
// A warp's first chunk of S(v*) goes by its number, consecutive chunks to
// different SMs, the others by a per-step counter.  The argmax meets in one word
// (an atomic per block, no second pass over block results).  Every wait is
// bounded (grid_sync).  A step is its barriers and the dependent loads between
// them and the decrements.
struct GreedyShared {
    unsigned long long best[2][32];
};

// Run by block `rank` of `nb`; false: a wait ran out.
__device__ __forceinline__ bool greedy_steps(const GreedyArgs &a, uint32_t rank, uint32_t nb,
                                             GreedyShared &sh) {
    int par = 0;                             // the buffer of the next block maximum
    auto block_max = [&](unsigned long long v) {
        const int l = threadIdx.x & 31;
        v = warp_max_key(v);
        if (l == 0) sh.best[par][threadIdx.x >> 5] = v;
        __syncthreads();
        const unsigned long long r = warp_max_key(l < (int)(blockDim.x >> 5) ? sh.best[par][l] : 0ull);
        par ^= 1;                            // (its readers pass a barrier before it is written again)
        return r;
    };
    const int64_t tid = (int64_t)rank * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)nb * blockDim.x;
    const int lane = threadIdx.x & 31;
    const int64_t gwarp = tid >> 5, nwarps = stride >> 5;
    const int64_t words = (a.theta + 31) / 32;
    const int64_t vwords = (a.n + 31) / 32;
    const int64_t nslots = a.spread ? 32 * vwords : a.n;
    auto slot = [&](int64_t v) { return a.spread ? (v & 31) * vwords + (v >> 5) : v; };
    auto vert = [&](int64_t i) { return a.spread ? (i % vwords) * 32 + i / vwords : i; };
    unsigned long long lmax = 0;
    for (int64_t i = tid; i < nslots; i += stride) {
        const int64_t v = vert(i);
        const int32_t d = v < a.n ? (int32_t)(a.vtx_off[v + 1] - a.vtx_off[v]) : 0;
        a.counts[i] = d;
        lmax = (unsigned long long)d > lmax ? (unsigned long long)d : lmax;
    }
    for (int64_t x = tid; x < words; x += stride) a.covered[x] = 0u;
    if (tid == 0) a.gmax[0] = a.gmax[1] = a.gmax[2] = 0ull;
    if (a.hub_rank) {
        lmax = block_max(lmax);
        if (threadIdx.x == 0 && lmax) atomicMax(a.ctl + 2, (int32_t)lmax);
    }
    if (!grid_sync(a.bar, nb, a.status)) return false;
    uint32_t tau = 0;                        // > 0: the argmax reads hubs + candidates
    int32_t nhub = 0, ncand = 0;
    if (a.hub_rank) {
        const uint32_t l = (uint32_t)__ldcg(a.ctl + 2);
        const uint32_t th = l >> a.hub_shift > 0 ? l >> a.hub_shift : 1;
        tau = a.cand_shift > 0 ? (l >> a.cand_shift > 0 ? l >> a.cand_shift : 1) : 0;
        for (int64_t v = tid; v < a.n; v += stride) {
            const uint32_t d = (uint32_t)(a.vtx_off[v + 1] - a.vtx_off[v]);
            int32_t r = -1;
            if (d >= th) {
                r = atomicAdd(a.ctl + 0, 1);
                if (r < a.hub_cap) {
                    a.hub_list[r] = (int32_t)v;
                    a.hub_cnt[(int64_t)r * kHubRep] = (int32_t)d;
                    for (int q = 1; q < kHubRep; ++q) a.hub_cnt[(int64_t)r * kHubRep + q] = 0;
                    a.counts[slot(v)] = 0;   // the row holds the gain
                } else {
                    r = -1;
                }
            }
            // below tau a vertex is frozen (-2): its gain stays |S(v)| < tau, a
            // stale bound, until the best gain drops below tau
            if (r < 0 && tau > 0) r = d >= tau ? -1 : -2;
            a.hub_rank[v] = r;
            if (r == -1 && tau > 0) a.cand[atomicAdd(a.ctl + 1, 1)] = (int32_t)v;
        }
        if (!grid_sync(a.bar, nb, a.status)) return false;
        nhub = min(__ldcg(a.ctl + 0), a.hub_cap);
        ncand = __ldcg(a.ctl + 1);
    }
    // a newly covered set of id = rep (mod 32) holds batch vertex mv
    auto decrement = [&](int32_t mv, int rep) {
        const int64_t u = mv - a.vshift;
        const int32_t hr = a.hub_rank ? __ldcg(a.hub_rank + u) : -1;
        if (hr >= 0) red_add_s32(a.hub_cnt + (int64_t)hr * kHubRep + rep, -1);
        else if (hr == -1) red_add_s32(a.counts + slot(u), -1);   // -2: frozen
    };
    int64_t cov = 0;
    int32_t j = 0;
    const int64_t claim = (int64_t)(threadIdx.x >> 5) * nb + rank;   // neighbours on different SMs
    for (int round = 0; j < a.k; ++round) {
        unsigned long long best = 0;
        auto consider = [&](int32_t c, uint32_t v) {
            if (c > 0) {
                const unsigned long long key =
                    ((unsigned long long)(uint32_t)c << 32) | (0xffffffffu - v);
                best = key > best ? key : best;
            }
        };
        if (tau > 0) {
            for (int64_t q = tid; q < ncand; q += stride) {
                const uint32_t v = (uint32_t)__ldcg(a.cand + q);
                consider(__ldcg(a.counts + slot(v)), v);
            }
        } else {
            for (int64_t i = tid; i < nslots; i += stride)
                consider(__ldcg(a.counts + i), (uint32_t)vert(i));
        }
        for (int64_t h = gwarp; h < nhub; h += nwarps) {      // a hub's gain: its row's sum
            const int32_t c = warp_sum<int32_t>(__ldcg(a.hub_cnt + h * kHubRep + lane));
            consider(c, (uint32_t)__ldcg(a.hub_list + h));
        }
        // the grid's maximum by one atomic a block on the round's word; of the
        // three words, the one of the round before is cleared for the round after
        // the next (every block has read it: it passed this round's barrier)
        best = block_max(best);
        if (threadIdx.x == 0 && best) atomicMax(a.gmax + round % 3, best);
        if (!grid_sync(a.bar, nb, a.status)) return false;
        const unsigned long long gbest = __ldcg(a.gmax + round % 3);
        if (tid == 0) a.gmax[(round + 2) % 3] = 0ull;
        if (tau > 0 && (uint32_t)(gbest >> 32) < tau) {
            // the best gain fell below tau: the frozen vertices may now win.
            // Make their gains exact against the sets covered so far, thaw
            // them, and read every gain from here on
            for (int64_t v = gwarp; v < a.n; v += nwarps) {
                if (__ldcg(a.hub_rank + v) != -2) continue;
                const int64_t sb = a.vtx_off[v], se = a.vtx_off[v + 1];
                int miss = 0;
                for (int64_t t = sb + lane; t < se; t += 32) {
                    const int64_t il = __ldg(a.set_ids + t) - a.sshift;
                    miss += !((__ldcg(a.covered + (il >> 5)) >> (il & 31)) & 1u);
                }
                miss = warp_sum<int>(miss);
                if (lane == 0) {
                    a.counts[slot(v)] = miss;
                    a.hub_rank[v] = -1;
                }
            }
            tau = 0;
            if (!grid_sync(a.bar, nb, a.status)) return false;
            continue;
        }
        if (gbest == 0) break;                       // every remaining gain is zero
        const int32_t vs = (int32_t)(0xffffffffu - (uint32_t)(gbest & 0xffffffffu));
        const int64_t gain = (int64_t)(gbest >> 32);
        if (rank == 0 && threadIdx.x == 0) {
            a.seeds[j] = vs;
            a.gains[j] = gain;
        }
        cov += gain;
        const int64_t sb = a.vtx_off[vs], se = a.vtx_off[vs + 1];
        // chunks of S(v*): the first by the warp's number, the others from this
        // step's counter (every warp's first one is taken when it starts); the other
        // step's counter is cleared meanwhile (its last use ended at the previous
        // step's closing barrier)
        const int64_t share = (se - sb + nwarps - 1) / nwarps;
        const int chunk = (int)(share < 1 ? 1 : share < kGreedyChunk ? share : kGreedyChunk);
        unsigned long long *work = a.work && se - sb > nwarps * chunk ? a.work + (j & 1) : nullptr;
        if (a.work && tid == 0) a.work[(j + 1) & 1] = 0ull;
        for (int64_t base = sb + claim * chunk;;) {
            if (base >= se) break;
            const int64_t t = base + lane;
            int32_t i = -1;
            if (lane < chunk && t < se) i = a.set_ids[t];
            const bool fresh = warp_bitmap_set(a.covered, i >= 0 ? i - a.sshift : -1, lane);
            if (__any_sync(kFull, fresh)) {
                // decrement the gains of every member of the lane's newly
                // covered set: the warp walks the concatenation of those
                // member lists 32 entries at a time, U loads in flight per lane
                int64_t mo = 0, ml = 0;
                if (fresh) {
                    mo = a.set_off[i];
                    ml = a.set_off[i + 1] - mo;
                }
                if (a.piece && ml > kGreedyPiece) {
                    const int64_t np = (ml + kGreedyPiece - 1) / kGreedyPiece;
                    unsigned long long *to = a.piece + atomicAdd(a.npiece, (unsigned long long)np);
                    for (int64_t q = 0; q < np; ++q) {
                        const int64_t left = ml - q * kGreedyPiece;
                        to[q] = (unsigned long long)(mo + q * kGreedyPiece) << 16 |
                                (unsigned long long)(left < kGreedyPiece ? left : kGreedyPiece) << 5 |
                                (unsigned long long)(i & (kHubRep - 1));
                    }
                    ml = 0;
                }
                // (kGreedyTake members of each at a time, so that positions stay
                // below 2^31 where sets of any length are not cut into pieces)
                do {
                    const int32_t mt = (int32_t)(ml < kGreedyTake ? ml : kGreedyTake);
                    const int32_t incl = warp_incl_scan<int32_t>(mt, lane);
                    const int32_t tot = __shfl_sync(kFull, incl, 31);
                    const int64_t from = mo + mt - incl;   // the lane's member for position 0
                    constexpr int U = 4;
                    for (int32_t p0 = 0; p0 < tot; p0 += 32 * U) {
                        int32_t mv[U], ms[U];
#pragma unroll
                        for (int uu = 0; uu < U; ++uu) {
                            const int32_t q = p0 + uu * 32 + lane;
                            int owner = 0;           // first lane whose inclusive count exceeds q
#pragma unroll
                            for (int step = 16; step > 0; step >>= 1)
                                if (__shfl_sync(kFull, incl, owner + step - 1) <= q) owner += step;
                            const int64_t o_from = __shfl_sync(kFull, from, owner);
                            ms[uu] = __shfl_sync(kFull, i, owner);
                            mv[uu] = q < tot ? __ldg(a.members + o_from + q) : -1;
                        }
#pragma unroll
                        for (int uu = 0; uu < U; ++uu)
                            if (mv[uu] >= 0) decrement(mv[uu], ms[uu] & (kHubRep - 1));
                    }
                    mo += mt;
                    ml -= mt;
                } while (__any_sync(kFull, ml > 0));
            }
            if (work) {
                unsigned long long c = 0;
                if (lane == 0) c = atomicAdd(work, (unsigned long long)chunk);
                base = sb + nwarps * chunk + (int64_t)__shfl_sync(kFull, c, 0);
            } else {
                base += nwarps * chunk;
            }
        }
        if (!grid_sync(a.bar, nb, a.status)) return false;
        const int64_t np = a.piece ? (int64_t)__ldcg(a.npiece) : 0;
        if (np > 0) {                                // (grid-uniform)
            for (int64_t p = gwarp; p < np; p += nwarps) {
                const unsigned long long pc = __ldcg(a.piece + p);
                const int32_t *mem = a.members + (pc >> 16);
                const int len = (int)(pc >> 5 & 2047), rep = (int)(pc & (kHubRep - 1));
                constexpr int U = 8;
                for (int x0 = lane; x0 < len; x0 += 32 * U) {
                    int32_t mv[U];
#pragma unroll
                    for (int uu = 0; uu < U; ++uu)
                        mv[uu] = x0 + uu * 32 < len ? __ldg(mem + x0 + uu * 32) : -1;
#pragma unroll
                    for (int uu = 0; uu < U; ++uu)
                        if (mv[uu] >= 0) decrement(mv[uu], rep);
                }
            }
            if (!grid_sync(a.bar, nb, a.status)) return false;
            // (the next pieces are put aside after the next barrier)
            if (rank == 0 && threadIdx.x == 0) *a.npiece = 0ull;
        }
        ++j;
    }
    if (rank == 0 && threadIdx.x == 0) {
        *a.nseeds = j;
        *a.coverage = cov;
    }
    return true;
}

__global__ void __launch_bounds__(kGreedyThreads, 2) k_greedy(GreedyArgs a) {
    __shared__ GreedyShared sh;
    greedy_steps(a, blockIdx.x, gridDim.x, sh);
}

// Many queries at once: group g of the launch, blocks [first[g], first[g + 1]),
// runs queries g, g + groups, ... of the table, each with its own barrier.  A
// query of a batch is a chain of short steps that a few SMs feed, and its
// barriers cost less among a few blocks; one launch after the other over the
// whole grid took 19 us a step whatever the query's size.
__global__ void __launch_bounds__(kGreedyThreads, 2) k_greedy_many(const GreedyArgs *tab, int32_t nq,
                                                                   const int32_t *first,
                                                                   int32_t groups) {
    __shared__ GreedyShared sh;
    __shared__ GreedyArgs s_a;
    __shared__ int32_t s_g;
    for (int g = threadIdx.x; g < groups; g += blockDim.x)
        if (first[g] <= (int32_t)blockIdx.x && (int32_t)blockIdx.x < first[g + 1]) s_g = g;
    __syncthreads();
    const int32_t g = s_g;
    const uint32_t rank = blockIdx.x - first[g], nb = first[g + 1] - first[g];
    for (int32_t q = g; q < nq; q += groups) {
        __syncthreads();
        for (int i = threadIdx.x; i < (int)(sizeof(GreedyArgs) / 4); i += blockDim.x)
            reinterpret_cast<uint32_t *>(&s_a)[i] = reinterpret_cast<const uint32_t *>(tab + q)[i];
        __syncthreads();
        if (!greedy_steps(s_a, rank, nb, sh)) return;
    }
}
static_assert(sizeof(GreedyArgs) % 4 == 0, "copied by words");

// ---------------------------------------------------------------------------
// RandGreedi
// ---------------------------------------------------------------------------
struct RGArgs {
    int64_t n, theta, words;
    int32_t k, P, trunc, B;
    const int64_t *vtx_off;
    const int32_t *set_ids;
    const int32_t *part_off;
    const int32_t *part_vtx;
    uint4 *cinfo;             // [n] by part position: first entry (64 bits), length and vertex of S(v),
    int32_t cinfo_smem;       // unless the producers keep it in shared memory
    uint32_t *covered;        // [P][words] producer bitmaps (unless in shared memory)
    uint32_t *bcovered;       // [B][words] bucket bitmaps
    int32_t *local_seeds;
    int64_t *local_gains;
    int32_t *local_n;
    int64_t *local_cov;
    const int64_t *thr;
    int64_t *bucket_cov;
    int32_t *bucket_n;
    int32_t *bucket_seeds;
    int64_t *bucket_gains;
    uint32_t *flags;          // [trunc][P]: 0 empty, 1 seed ready, 2 no seed
    int32_t *elems;           // [trunc][P]
    int32_t nprod, ncons;     // block roles in this launch
    int32_t first_role;       // 0: blocks start with producers; 1: consumers only
    int32_t max_np;           // largest part: key[] and stamp[] are max_np each
    int32_t evals;            // local greedy: candidates re-evaluated per round (<= kProdW)
    long long *stats;         // [P + B][6] diagnostics (see im_randgreedi_stats)
    int *status;
    // bucket-mask stage (k_rg_stream_masks)
    unsigned long long *mask; // [theta]: bit b set once bucket b covers the set
    uint32_t *gbuf;           // [2][kMaskG][64] per-slot, per-bucket gains
    GridBarrier *bar;
    int32_t *slot_x;          // [trunc * P] element of each stream slot, -1 if none
    int64_t *slot_beg, *slot_len;   // its covering subset in set_ids
};

// Local greedy of part p (Alg. 4, one sender), run as the lazy greedy of
// Alg. 2: key[l] holds a gain of candidate l that is exact when stamp[l]
// equals the current round and an upper bound otherwise (gains only shrink,
// by submodularity).  The largest key (ties: smallest id) is taken when it is
// exact, which picks exactly the standard greedy's sequence.
//
// cmax[c] is the largest packed key (gain << 32 | ~l) of the 32 candidates of
// chunk c.  A round takes the best candidate of each of the W chunks with the
// largest cmax and re-evaluates the stale ones at once (blockDim / W threads
// each) against the part's covered bitmap; then, if the overall largest key is
// exact, it is taken.  Evaluating more candidates than the sequential rule
// would only replaces upper bounds by exact values, so the sequence of picks is
// unchanged while a pick takes one or two rounds instead of one round per stale
// candidate.
//
// A round is a chain: select, read the candidates' subsets, probe the bitmap,
// add up.  Warp 0 does all that is serial (keys, chunk maxima, the selection of
// the next round, by 32-bit reductions) while the others wait at one barrier or,
// after a pick, cover its subset meanwhile; a candidate's subset comes in one
// read.  With few sets the bitmap lies in shared memory (SB), where 32
// probes take a few cycles; in global memory they take one L1 line each, and at
// 4 x 10^6 sets that is what bounds the part (2.7 x 10^6 probes and 0.6 x 10^6
// marks a part, 0.63 of them a cycle).  148 parts of R-MAT scale 20, k = 100, 4.2 x
// 10^6 LT sets: 3.13 -> 2.82 ms; 512 parts, 2.1 x 10^6 weighted-cascade sets (two
// blocks an SM): 3.58 -> 1.74 ms; 64 parts, 2 x 10^5 sets: 0.40 -> 0.30 ms.
constexpr int kProdW = 8;

__device__ __forceinline__ unsigned long long prod_key(int32_t g, int32_t l) {
    return g > 0 ? ((unsigned long long)(uint32_t)g << 32) | (0xffffffffu - (uint32_t)l) : 0ull;
}

// cmax of chunk c, by one warp
__device__ __forceinline__ void prod_chunk_max(const int32_t *key, unsigned long long *cmax,
                                               int32_t np, int32_t c, int lane) {
    const int32_t l = c * 32 + lane;
    const unsigned long long v = warp_max_key(l < np ? prod_key(key[l], l) : 0ull);
    if (lane == 0) cmax[c] = v;
}

template <bool SB>
__device__ void produce(const RGArgs &a, int p, int32_t *key) {
    __shared__ int32_t s_cand[kProdW];           // the round's candidates, -1: none
    __shared__ int32_t s_stale[kProdW];          // ... 1: to be evaluated
    __shared__ int32_t s_cnt[kProdW];            // ... their gains
    __shared__ int64_t s_beg[kProdW];            // ... their subsets
    __shared__ int32_t s_len[kProdW];
    __shared__ int s_act;                        // 0 done, 1 evaluate, 2 take candidate 0
    const int32_t vb = a.part_off[p], np = a.part_off[p + 1] - vb;
    int32_t *stamp = key + a.max_np;
    unsigned long long *cmax = reinterpret_cast<unsigned long long *>(key + 2 * a.max_np);
    const int32_t nch = (np + 31) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    unsigned char *rest = reinterpret_cast<unsigned char *>(cmax + ((a.max_np + 63) / 64) * 2);
    uint4 *cinfo = a.cinfo_smem ? reinterpret_cast<uint4 *>(rest) : a.cinfo + vb;
    if (a.cinfo_smem) rest += (size_t)a.max_np * sizeof(uint4);
    uint32_t *cov = SB ? reinterpret_cast<uint32_t *>(rest) : a.covered + (size_t)p * (size_t)a.words;
    for (int64_t x = threadIdx.x; x < a.words; x += blockDim.x) cov[x] = 0u;
    for (int32_t l = threadIdx.x; l < np; l += blockDim.x) {
        const int32_t v = a.part_vtx[vb + l];
        const int64_t b = a.vtx_off[v], n = a.vtx_off[v + 1] - b;
        cinfo[l] = make_uint4((uint32_t)b, (uint32_t)((uint64_t)b >> 32), (uint32_t)n, (uint32_t)v);
        key[l] = (int32_t)n;
        stamp[l] = 0;                                   // exact: nothing is covered yet
    }
    __syncthreads();
    for (int32_t c = warp; c < nch; c += nwarp) prod_chunk_max(key, cmax, np, c, lane);
    __syncthreads();
    const uint64_t t_begin = global_ns();
    long long n_rounds = 0, n_evals = 0, eval_entries = 0, cover_entries = 0;   // (warp 0's)
    int64_t total = 0;
    int32_t j = 0;
    const int W = a.evals;
    const int gsz = blockDim.x / W, grp = threadIdx.x / gsz, gt = threadIdx.x % gsz;
    // warp 0: the candidates of the next round, and what to do with them
    auto select = [&]() {
        unsigned long long taken = ~0ull;        // the last one chosen; keys are distinct
        int32_t mine = -1;                       // candidate of lane w
        unsigned long long top = 0ull;
        for (int w = 0; w < W; ++w) {
            unsigned long long best = 0ull;
            for (int32_t c = lane; c < nch; c += 32) {
                const unsigned long long v = cmax[c];
                if (v > best && v < taken) best = v;
            }
            const unsigned long long m = warp_max_key(best);
            if (m == 0ull) break;
            if (w == 0) top = m;
            if (lane == w) mine = (int32_t)(0xffffffffu - (uint32_t)m);
            taken = m;
            // an exact top is taken: no need of the others
            if (w == 0 && stamp[0xffffffffu - (uint32_t)m] == j) break;
        }
        bool stale = false;
        if (mine >= 0) {
            stale = stamp[mine] != j;
            const uint4 ci = cinfo[mine];
            s_beg[lane] = (int64_t)((uint64_t)ci.y << 32 | ci.x);
            s_len[lane] = (int32_t)ci.z;
        }
        if (lane < W) {
            s_cand[lane] = mine;
            s_stale[lane] = stale;
            s_cnt[lane] = 0;
        }
        const bool top_stale = __shfl_sync(kFull, stale, 0);
        if (lane == 0) s_act = top == 0ull ? 0 : top_stale ? 1 : 2;
        __syncwarp();
    };
    if (warp == 0) select();
    __syncthreads();
    while (s_act != 0) {
        if (s_act == 1) {
            // ---- re-evaluate every stale candidate of the round at once
            ++n_rounds;
            if (s_stale[grp]) {
                int miss = 0;
                // global bitmap: L1-cached probes.  It is written only by this block
                // (atomics, ordered before these loads by the block barriers), and
                // S(v) is scanned in ascending set order when the index comes from
                // the radix build, so neighbouring ids share cached lines
                scan_ids<4>(a.set_ids, s_beg[grp], s_len[grp], gt, gsz, [&](int32_t i) {
                    if (i >= 0)
                        miss += !(((SB ? cov[i >> 5] : __ldca(cov + (i >> 5))) >> (i & 31)) & 1u);
                });
                miss = __reduce_add_sync(kFull, miss);
                if (lane == 0 && miss) atomicAdd(&s_cnt[grp], miss);
            }
            __syncthreads();
            if (warp == 0) {
                for (int w = 0; w < W; ++w) {
                    if (!s_stale[w]) continue;
                    const int32_t l = s_cand[w];
                    if (lane == 0) {
                        key[l] = s_cnt[w];
                        stamp[l] = j;
                    }
                    ++n_evals;
                    eval_entries += s_len[w];
                    __syncwarp();
                    prod_chunk_max(key, cmax, np, l >> 5, lane);
                    __syncwarp();
                }
                select();
            }
        } else {
            // ---- take candidate 0; the next round's are selected meanwhile
            const int32_t l = s_cand[0];
            const int64_t sb = s_beg[0];
            const int32_t n = s_len[0];
            __syncthreads();                     // everyone has read the candidate
            if (warp == 0) {
                const int32_t gain = key[l];
                __syncwarp();                    // every lane has read it
                if (lane == 0) {
                    const int32_t v = (int32_t)cinfo[l].w;
                    a.local_seeds[(int64_t)p * a.k + j] = v;
                    a.local_gains[(int64_t)p * a.k + j] = gain;
                    if (j < a.trunc) {
                        a.elems[(int64_t)j * a.P + p] = v;
                        st_release_u32(&a.flags[(int64_t)j * a.P + p], 1u);
                    }
                    key[l] = 0;
                }
                total += gain;
                cover_entries += n;
                __syncwarp();
                prod_chunk_max(key, cmax, np, l >> 5, lane);
                __syncwarp();
            }
            ++j;
            if (j < a.k) {
                if (warp == 0) select();
                else
                    scan_ids<4>(a.set_ids, sb, n, (int)threadIdx.x - 32, (int)blockDim.x - 32, [&](int32_t i) {
                        if (i >= 0) atomicOr(&cov[i >> 5], 1u << (i & 31));
                    });
            } else if (threadIdx.x == 0) {
                s_act = 0;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        a.local_n[p] = j;
        a.local_cov[p] = total;
        for (int32_t jj = j; jj < a.trunc; ++jj) st_release_u32(&a.flags[(int64_t)jj * a.P + p], 2u);
        if (a.stats) {
            long long *st = a.stats + 6 * (int64_t)p;
            st[0] = (long long)t_begin;
            st[1] = (long long)global_ns();
            st[2] = n_rounds + j;
            st[3] = n_evals;
            st[4] = eval_entries;
            st[5] = cover_entries;
        }
    }
    __syncthreads();
}

// Streaming bucket b (Alg. 5): consume the stream in (j, p) order.
//
// Elements are evaluated speculatively in groups of W against the bucket as
// it stands: the first element of the group whose gain reaches the threshold
// is the next one the sequential rule accepts (every element before it saw
// the same bucket and fell short), so it is accepted and evaluation resumes
// right after it; later elements of the group are evaluated again.  W doubles
// after a group without an accept and halves after one, which bounds the
// repeated work by the number of accepts times W.
__device__ void consume(const RGArgs &a, int b, long long *shs) {
    __shared__ int32_t s_x[kBatch];
    __shared__ int64_t s_off[kBatch];
    __shared__ int64_t s_len[kBatch];
    __shared__ int s_cand[kSpec];
    __shared__ unsigned long long s_miss[kSpec];
    __shared__ int s_ncand, s_end, s_acc, s_timeout;
    uint32_t *C = a.bcovered + (size_t)b * (size_t)a.words;
    for (int64_t x = threadIdx.x; x < a.words; x += blockDim.x) C[x] = 0u;
    if (threadIdx.x == 0) s_timeout = 0;
    __syncthreads();
    const int64_t T = a.thr[b];
    const int64_t E = (int64_t)a.trunc * a.P;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const uint64_t t_begin = global_ns();
    long long n_eval = 0, scanned = 0, wait_ns = 0;
    int32_t bn = 0;
    int64_t bcov = 0;
    int W = 1;
    for (int64_t base = 0; base < E && bn < a.k; base += kBatch) {
        const int cntb = (int)min((int64_t)kBatch, E - base);
        const uint64_t tw0 = global_ns();
        if (threadIdx.x < cntb) {
            const int64_t slot = base + threadIdx.x;
            uint32_t f = ld_acquire_u32(a.flags + slot);
            if (f == 0) {
                const uint64_t t0 = global_ns();
                while ((f = ld_acquire_u32(a.flags + slot)) == 0) {
                    if (global_ns() - t0 > kWaitLimitNs) {
                        raise_status(a.status, kDevTimeout);
                        s_timeout = 1;
                        break;
                    }
                    __nanosleep(128);
                }
            }
            int32_t x = -1;
            int64_t off = 0, len = 0;
            if (f == 1) {
                x = __ldcg(a.elems + slot);
                off = a.vtx_off[x];
                len = a.vtx_off[x + 1] - off;
            }
            s_x[threadIdx.x] = x;
            s_off[threadIdx.x] = off;
            s_len[threadIdx.x] = len;
        }
        __syncthreads();
        wait_ns += (long long)(global_ns() - tw0);
        if (s_timeout) break;
        int q = 0;
        while (q < cntb && bn < a.k) {
            if (threadIdx.x == 0) {
                // next W candidates; |S(x)| < threshold rejects x without a scan
                int n = 0, r = q;
                while (r < cntb && n < W) {
                    if (s_x[r] >= 0 && s_len[r] >= T) s_cand[n++] = r;
                    ++r;
                }
                s_ncand = n;
                s_end = r;
            }
            if (threadIdx.x < kSpec) s_miss[threadIdx.x] = 0;
            __syncthreads();
            const int n = s_ncand;
            if (n == 0) {
                q = s_end;
                __syncthreads();
                continue;
            }
            // |S(x) \ C_b| for every candidate, all warps in flight at once
            for (int c = 0; c < n; ++c) {
                const int r = s_cand[c];
                const int64_t off = s_off[r], len = s_len[r];
                unsigned m = 0;
                for (int64_t c0 = (int64_t)warp * 32 * kUnroll; c0 < len;
                     c0 += (int64_t)nwarps * 32 * kUnroll) {
                    int32_t ids[kUnroll];
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u) {
                        const int64_t t = c0 + u * 32 + lane;
                        ids[u] = t < len ? __ldg(a.set_ids + off + t) : -1;
                    }
                    unsigned words[kUnroll];
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u)
                        words[u] = ids[u] >= 0 ? __ldcg(C + (ids[u] >> 5)) : ~0u;
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u)
                        m += __popc(__ballot_sync(kFull, !((words[u] >> (ids[u] & 31)) & 1u)));
                }
                if (lane == 0 && m) atomicAdd(&s_miss[c], (unsigned long long)m);
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                int acc = -1;
                for (int c = 0; c < n; ++c)
                    if ((int64_t)s_miss[c] >= T) {
                        acc = c;
                        break;
                    }
                s_acc = acc;
            }
            __syncthreads();
            const int acc = s_acc;
            n_eval += acc < 0 ? n : acc + 1;
            for (int c = 0; c < n; ++c) scanned += s_len[s_cand[c]];
            if (acc < 0) {
                q = s_end;
                W = min(kSpec, 2 * W);
            } else {
                const int r = s_cand[acc];
                const int64_t off = s_off[r], len = s_len[r];
                for (int64_t t = threadIdx.x; t < len; t += blockDim.x) {
                    const int32_t i = __ldg(a.set_ids + off + t);
                    atomicOr(&C[i >> 5], 1u << (i & 31));
                }
                const int64_t gain = (int64_t)s_miss[acc];
                if (threadIdx.x == 0) {
                    a.bucket_seeds[(int64_t)b * a.k + bn] = s_x[r];
                    a.bucket_gains[(int64_t)b * a.k + bn] = gain;
                }
                ++bn;
                bcov += gain;
                q = r + 1;
                W = max(1, W / 2);
            }
            __syncthreads();
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        a.bucket_n[b] = bn;
        a.bucket_cov[b] = bcov;
        if (a.stats) {
            long long *st = a.stats + 6 * ((int64_t)a.P + b);
            st[0] = (long long)t_begin;
            st[1] = (long long)global_ns();
            st[2] = n_eval;
            st[3] = bn;
            st[4] = scanned;
            st[5] = wait_ns;
        }
    }
    __syncthreads();
}

// The producers alone (two-launch mode): one block per part.
template <bool SB>
__global__ void __launch_bounds__(kProdThreads) k_rg_local(RGArgs a) {
    extern __shared__ __align__(16) int32_t key[];   // (produce() reads 16 bytes at a time)
    for (int p = blockIdx.x; p < a.P; p += gridDim.x) produce<SB>(a, p, key);
}

__global__ void __launch_bounds__(kRGThreads) k_randgreedi(RGArgs a) {
    extern __shared__ __align__(16) int32_t key[];
    __shared__ long long shs[33];
    const int r = blockIdx.x;
    if (a.first_role == 0 && r < a.nprod) {
        for (int p = r; p < a.P; p += a.nprod) produce<false>(a, p, key);
    } else {
        const int c = a.first_role == 0 ? r - a.nprod : r;
        for (int b = c; b < a.B; b += a.ncons) consume(a, b, shs);
    }
}

// Streaming buckets with the bucket bitmap in shared memory (Alg. 5, run after
// the local greedy has finished).  A cluster of CS blocks serves one bucket
// at a time (buckets are taken from a global counter): block r keeps the bits
// of set ids [r * R, (r + 1) * R) in its shared memory, scans every entry of
// S(x) and tests only the ids in its own range.  The per-candidate counts of
// the CS blocks are added over distributed shared memory after a cluster
// barrier, and every block takes the same accept decision.  Candidates go in
// the same speculative groups as in consume(); partial-count arrays alternate
// between two buffers so one barrier per group suffices.
__global__ void __launch_bounds__(kRGThreads) k_rg_stream_cluster(RGArgs a, int64_t R,
                                                                  unsigned *bucket_counter) {
    extern __shared__ uint32_t bits[];               // R bits, then 2 x kSpec partial counts
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned CS = cluster.num_blocks();
    const unsigned rank = cluster.block_rank();
    const int64_t words = R / 32;
    unsigned *part = bits + words;                   // [2][kSpec]
    __shared__ int32_t w_x[kBatch];                  // stream window: element, offset, length
    __shared__ int64_t w_off[kBatch], w_len[kBatch];
    __shared__ int s_cand[kSpec];
    __shared__ unsigned long long s_tot[kSpec];
    __shared__ int s_n, s_bucket, s_end, s_acc;
    const int64_t lo = (int64_t)rank * R;
    const int lane = threadIdx.x & 31;
    const int64_t E = (int64_t)a.trunc * a.P;
    for (;;) {
        if (rank == 0 && threadIdx.x == 0) s_bucket = (int)atomicAdd(bucket_counter, 1u);
        cluster.sync();
        if (threadIdx.x == 0) s_bucket = *cluster.map_shared_rank(&s_bucket, 0);
        cluster.sync();
        const int b = s_bucket;
        if (b >= a.B) break;
        for (int64_t x = threadIdx.x; x < words; x += blockDim.x) bits[x] = 0u;
        const int64_t T = a.thr[b];
        const uint64_t t_begin = global_ns();
        long long n_eval = 0, scanned = 0;
        int32_t bn = 0;
        int64_t bcov = 0;
        int W = 1, phase = 0;
        cluster.sync();
        for (int64_t base = 0; base < E && bn < a.k; base += kBatch) {
            // the producers have finished: every slot is final (1 seed, 2 none)
            const int cntb = (int)min((int64_t)kBatch, E - base);
            if (threadIdx.x < cntb) {
                const int64_t slot = base + threadIdx.x;
                int32_t x = -1;
                int64_t off = 0, len = 0;
                if (ld_acquire_u32(a.flags + slot) == 1u) {
                    x = __ldcg(a.elems + slot);
                    off = a.vtx_off[x];
                    len = a.vtx_off[x + 1] - off;
                }
                w_x[threadIdx.x] = x;
                w_off[threadIdx.x] = off;
                w_len[threadIdx.x] = len;
            }
            __syncthreads();
            int qq = 0;
            while (qq < cntb && bn < a.k) {
                if (threadIdx.x == 0) {
                    // next W candidates; |S(x)| < threshold rejects x without a scan
                    int n = 0, r = qq;
                    while (r < cntb && n < W) {
                        if (w_x[r] >= 0 && w_len[r] >= T) s_cand[n++] = r;
                        ++r;
                    }
                    s_n = n;
                    s_end = r;
                }
                unsigned *mine = part + phase * kSpec;
                if (threadIdx.x < kSpec) mine[threadIdx.x] = 0u;
                __syncthreads();
                const int n = s_n;
                if (n == 0) {
                    qq = s_end;
                    __syncthreads();
                    continue;
                }
                for (int c = 0; c < n; ++c) {
                    const int r = s_cand[c];
                    unsigned m = 0;
                    scan_ids<4>(a.set_ids, w_off[r], w_len[r], threadIdx.x, blockDim.x,
                                [&](int32_t id) {
                                    const int64_t rel = (int64_t)id - lo;
                                    if (id >= 0 && rel >= 0 && rel < R)
                                        m += !((bits[rel >> 5] >> (rel & 31)) & 1u);
                                });
                    m = warp_sum<unsigned>(m);
                    if (lane == 0 && m) atomicAdd(&mine[c], m);
                }
                cluster.sync();
                // candidate c's total over the cluster, summed by thread c
                if (threadIdx.x < n) {
                    unsigned long long tot = 0;
                    for (unsigned r2 = 0; r2 < CS; ++r2)
                        tot += cluster.map_shared_rank(mine, r2)[threadIdx.x];
                    s_tot[threadIdx.x] = tot;
                }
                __syncthreads();
                if (threadIdx.x < 32) {
                    const bool ok = lane < n && (int64_t)s_tot[lane] >= T;
                    const unsigned bal = __ballot_sync(kFull, ok);
                    if (lane == 0) s_acc = bal ? __ffs(bal) - 1 : -1;
                }
                __syncthreads();
                const int acc = s_acc;
                n_eval += acc < 0 ? n : acc + 1;
                for (int c = 0; c < n; ++c) scanned += w_len[s_cand[c]];
                if (acc < 0) {
                    qq = s_end;
                    W = min(kSpec, 2 * W);
                } else {
                    const int r = s_cand[acc];
                    scan_ids<4>(a.set_ids, w_off[r], w_len[r], threadIdx.x, blockDim.x,
                                [&](int32_t id) {
                                    const int64_t rel = (int64_t)id - lo;
                                    if (id >= 0 && rel >= 0 && rel < R)
                                        atomicOr(&bits[rel >> 5], 1u << (rel & 31));
                                });
                    const int64_t gain = (int64_t)s_tot[acc];
                    if (rank == 0 && threadIdx.x == 0) {
                        a.bucket_seeds[(int64_t)b * a.k + bn] = w_x[r];
                        a.bucket_gains[(int64_t)b * a.k + bn] = gain;
                    }
                    ++bn;
                    bcov += gain;
                    qq = r + 1;
                    W = max(1, W / 2);
                }
                phase ^= 1;
                __syncthreads();
            }
            __syncthreads();
        }
        if (rank == 0 && threadIdx.x == 0) {
            a.bucket_n[b] = bn;
            a.bucket_cov[b] = bcov;
            if (a.stats) {
                long long *st = a.stats + 6 * ((int64_t)a.P + b);
                st[0] = (long long)t_begin;
                st[1] = (long long)global_ns();
                st[2] = n_eval;
                st[3] = bn;
                st[4] = scanned;
                st[5] = 0;
            }
        }
        cluster.sync();
    }
}

// Streaming buckets over per-set bucket masks (Alg. 5, run after the local
// greedy has finished; B <= 64).  mask[i] holds one bit per bucket: bit b is
// set once bucket b covers RRR set i.  A single pass over S(x) therefore
// yields the marginal gain of x for every bucket at once -- the count of
// entries whose bit b is clear -- instead of one pass per bucket.
//
// The stream is consumed in (j, p) slot order in speculative groups of up to
// kMaskG slots.  Every warp of the grid takes work items of kMaskItem entries
// of the group's subsets and adds its per-bucket counts to gbuf; after a grid
// barrier every block replays the same sequential decision for each bucket
// from those counts.  A count taken against the bucket as it stood at the
// start of the group is exact until the bucket accepts something in the
// group, and an upper bound after that (coverage only grows), so a later slot
// below the threshold is still rejected exactly; a later slot at or above it
// needs a fresh count, and the group is cut there for all buckets.  The
// accepted subsets are then or-ed into the masks and the next group starts at
// the cut.  Group sizes double after a group without a cut and halve after a
// cut.
// The slot whose work items hold item c: the largest u < gn with s_off[u] <= c.
__device__ __forceinline__ int mask_slot_of(const int64_t *s_off, int gn, int64_t c) {
    int lo = 0, hi = gn - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_off[mid] <= c) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Exclusive prefix of the work items of slots [0, gn) (items[u] from f(u)),
// written to s_off[0..gn]; gn <= 64, run by warp 0.
template <typename F>
__device__ __forceinline__ void mask_item_prefix(int64_t *s_off, int gn, F &&f) {
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    const int u0 = 2 * lane, u1 = 2 * lane + 1;
    const int64_t a0 = u0 < gn ? f(u0) : 0, a1 = u1 < gn ? f(u1) : 0;
    const int64_t incl = warp_incl_scan<int64_t>(a0 + a1, lane);
    const int64_t excl = incl - a0 - a1;
    if (u0 < gn) s_off[u0] = excl;
    if (u1 < gn) s_off[u1] = excl + a0;
    if (lane == 31) s_off[gn] = incl;
}

__global__ void __launch_bounds__(kRGThreads) k_rg_stream_masks(RGArgs a) {
    // a window of the stream's slots, read ahead of the groups
    __shared__ int32_t s_wx[kMaskWindow];
    __shared__ int64_t s_wbeg[kMaskWindow], s_wlen[kMaskWindow];
    __shared__ int32_t s_cnt0[kMaskG + 1];           // block 0: elements in the group's first u slots
    __shared__ int64_t s_len0[kMaskG + 1];           // ... and the entries of their subsets
    __shared__ uint32_t s_g[kMaskG * 64];            // the group's gains, staged once
    __shared__ unsigned long long s_pass[64];        // slots reaching each bucket's threshold
    __shared__ int64_t s_thr[64];
    __shared__ int64_t s_off[kMaskG + 1];            // work-item prefix over the group's slots
    __shared__ unsigned long long s_acc[kMaskG];     // buckets accepting each slot
    __shared__ int32_t s_n[64];
    __shared__ int64_t s_cov[64];
    __shared__ long long s_eval[64], s_scan[64];
    __shared__ int s_cut;
    const int lane = threadIdx.x & 31;
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gstride = (int64_t)gridDim.x * blockDim.x;
    // warps numbered block-minor, so the few work items of a small group land
    // on different SMs
    const int64_t gwarp = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const int64_t nwarps = gstride >> 5;
    const int64_t nslots = (int64_t)a.trunc * a.P;
    const uint64_t t_begin = global_ns();
    for (int64_t i = gtid; i < a.theta; i += gstride) a.mask[i] = 0ull;
    for (int64_t i = gtid; i < 2 * kMaskG * 64; i += gstride) a.gbuf[i] = 0u;
    // slot table: element (or -1) and its covering-subset range, read once
    for (int64_t t = gtid; t < nslots; t += gstride) {
        const int32_t x = ld_acquire_u32(a.flags + t) == 1u ? __ldcg(a.elems + t) : -1;
        const int64_t b = x >= 0 ? a.vtx_off[x] : 0;
        a.slot_x[t] = x;
        a.slot_beg[t] = b;
        a.slot_len[t] = x >= 0 ? a.vtx_off[x + 1] - b : 0;
    }
    if (threadIdx.x < 64) {
        s_thr[threadIdx.x] = threadIdx.x < a.B ? a.thr[threadIdx.x] : 0;
        s_n[threadIdx.x] = 0;
        s_cov[threadIdx.x] = 0;
        s_eval[threadIdx.x] = 0;
        s_scan[threadIdx.x] = 0;
    }
    if (!grid_sync(a.bar, gridDim.x, a.status)) return;
    int64_t g0 = 0, w0 = -1;                         // the window holds slots [w0, w0 + kMaskWindow)
    int G = 8, buf = 0;
    while (g0 < nslots) {
        const int gn = (int)(nslots - g0 < G ? nslots - g0 : G);
        if (w0 < 0 || g0 + kMaskG > w0 + kMaskWindow) {
            w0 = g0;
            for (int i = threadIdx.x; i < kMaskWindow && w0 + i < nslots; i += blockDim.x) {
                s_wx[i] = __ldcg(a.slot_x + w0 + i);
                s_wbeg[i] = __ldcg(a.slot_beg + w0 + i);
                s_wlen[i] = __ldcg(a.slot_len + w0 + i);
            }
        }
        const int32_t *s_x = s_wx + (g0 - w0);       // the group's slots
        const int64_t *s_beg = s_wbeg + (g0 - w0), *s_len = s_wlen + (g0 - w0);
        if (threadIdx.x < kMaskG) s_acc[threadIdx.x] = 0ull;
        if (threadIdx.x == 0) s_cut = gn;
        __syncthreads();
        mask_item_prefix(s_off, gn, [&](int u) { return (s_len[u] + kMaskItem - 1) / kMaskItem; });
        if (blockIdx.x == 0 && threadIdx.x >= 32 && threadIdx.x < 64) {
            const int u0 = 2 * lane, u1 = u0 + 1;
            const int32_t c0 = u0 < gn && s_x[u0] >= 0, c1 = u1 < gn && s_x[u1] >= 0;
            const int64_t l0 = c0 ? s_len[u0] : 0, l1 = c1 ? s_len[u1] : 0;
            const int32_t ci = warp_incl_scan<int32_t>(c0 + c1, lane);
            const int64_t li = warp_incl_scan<int64_t>(l0 + l1, lane);
            s_cnt0[u0] = ci - c0 - c1;
            s_cnt0[u1] = ci - c1;
            s_len0[u0] = li - l0 - l1;
            s_len0[u1] = li - l1;
            if (lane == 31) {
                s_cnt0[kMaskG] = ci;
                s_len0[kMaskG] = li;
            }
        }
        __syncthreads();
        uint32_t *gb = a.gbuf + (size_t)buf * kMaskG * 64;
        // ---- counts of every slot of the group against the current masks
        for (int64_t c = gwarp; c < s_off[gn]; c += nwarps) {
            const int u = mask_slot_of(s_off, gn, c);
            const int64_t e0 = (c - s_off[u]) * kMaskItem;
            const int64_t len = s_len[u];
            const int32_t *ids = a.set_ids + s_beg[u];
            // all ids first, then all masks: two memory round trips per item
            int32_t id[kMaskStrips];
#pragma unroll
            for (int st = 0; st < kMaskStrips; ++st) {
                const int64_t e = e0 + st * 32 + lane;
                id[st] = e < len ? __ldg(ids + e) : -1;
            }
            unsigned long long mk[kMaskStrips];
#pragma unroll
            for (int st = 0; st < kMaskStrips; ++st)
                mk[st] = id[st] >= 0 ? ~__ldcg(a.mask + id[st]) : 0ull;
            // 5-bit vertical counters, one bit-plane per 64-bit word
            unsigned long long c0 = 0, c1 = 0, c2 = 0, c3 = 0, c4 = 0;
#pragma unroll
            for (int st = 0; st < kMaskStrips; ++st) {
                unsigned long long m = mk[st];
                unsigned long long t = c0 & m;
                c0 ^= m;
                m = t;
                t = c1 & m;
                c1 ^= m;
                m = t;
                t = c2 & m;
                c2 ^= m;
                m = t;
                t = c3 & m;
                c3 ^= m;
                m = t;
                c4 |= m;
            }
            // add the 32 lanes' counters bit-serially in a butterfly: after
            // round r every lane holds the sum over its 2^(r+1)-lane group
            unsigned long long pl[10] = {c0, c1, c2, c3, c4, 0, 0, 0, 0, 0};
#pragma unroll
            for (int r = 0; r < 5; ++r) {
                unsigned long long carry = 0;
#pragma unroll
                for (int q = 0; q < 5 + r; ++q) {
                    const unsigned long long x = pl[q];
                    const unsigned long long y = __shfl_xor_sync(kFull, x, 1 << r);
                    pl[q] = x ^ y ^ carry;
                    carry = (x & y) | (carry & (x ^ y));
                }
                pl[5 + r] = carry;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int b = lane + 32 * h;
                uint32_t v = 0;
#pragma unroll
                for (int q = 0; q < 10; ++q) v |= (uint32_t)((pl[q] >> b) & 1ull) << q;
                if (b < a.B && v) atomicAdd(gb + u * 64 + b, v);
            }
        }
        if (!grid_sync(a.bar, gridDim.x, a.status)) return;
        // ---- the sequential rule of every bucket, replayed in every block.
        // Within a group a bucket takes at most its first passing slot: a
        // second one (while the bucket still has room) needs a fresh count,
        // so the group is cut there.
        if (threadIdx.x < 64) s_pass[threadIdx.x] = 0ull;
        __syncthreads();
        for (int i = threadIdx.x; i < gn * 64; i += blockDim.x) {
            const uint32_t g = __ldcg(gb + i);
            s_g[i] = g;
            const int u = i >> 6, b = i & 63;
            if (b < a.B && s_x[u] >= 0 && (int64_t)g >= s_thr[b]) atomicOr(&s_pass[b], 1ull << u);
        }
        __syncthreads();
        const int b = threadIdx.x;
        const bool own = b < a.B && s_n[b] < a.k;
        int first = kMaskG;
        if (own && s_pass[b]) {
            const unsigned long long pm = s_pass[b];
            first = __ffsll((long long)pm) - 1;
            const unsigned long long rest = pm & (pm - 1);
            if (rest && s_n[b] + 1 < a.k) atomicMin(&s_cut, __ffsll((long long)rest) - 1);
        }
        __syncthreads();
        const int cut = s_cut;
        if (own) {
            if (first < cut) {
                const int64_t g = (int64_t)s_g[first * 64 + b];
                atomicOr(&s_acc[first], 1ull << b);
                if (blockIdx.x == 0) {
                    a.bucket_seeds[(int64_t)b * a.k + s_n[b]] = s_x[first];
                    a.bucket_gains[(int64_t)b * a.k + s_n[b]] = g;
                }
                ++s_n[b];
                s_cov[b] += g;
            }
            // diagnostics: slots this bucket considered (up to the cut, or to
            // its accept when that filled it)
            if (blockIdx.x == 0) {
                const int last = (first < cut && s_n[b] == a.k) ? first + 1 : cut;
                s_eval[b] += s_cnt0[last];
                s_scan[b] += s_len0[last];
            }
        }
        __syncthreads();
        // ---- or the accepted subsets into the masks; clear the other buffer
        mask_item_prefix(s_off, cut, [&](int u) {
            return s_acc[u] ? (s_len[u] + kMaskItem - 1) / kMaskItem : (int64_t)0;
        });
        __syncthreads();
        for (int64_t c = gwarp; c < s_off[cut]; c += nwarps) {
            const int u = mask_slot_of(s_off, cut, c);   // slots without items are skipped
            const unsigned long long acc = s_acc[u];
            const int64_t e0 = (c - s_off[u]) * kMaskItem;
            const int64_t len = s_len[u];
            const int32_t *ids = a.set_ids + s_beg[u];
            int32_t id[kMaskStrips];
#pragma unroll
            for (int st = 0; st < kMaskStrips; ++st) {
                const int64_t e = e0 + st * 32 + lane;
                id[st] = e < len ? __ldg(ids + e) : -1;
            }
#pragma unroll
            for (int st = 0; st < kMaskStrips; ++st)
                if (id[st] >= 0) atomicOr(a.mask + id[st], acc);
        }
        uint32_t *other = a.gbuf + (size_t)(buf ^ 1) * kMaskG * 64;
        for (int64_t i = gtid; i < kMaskG * 64; i += gstride) other[i] = 0u;
        if (!grid_sync(a.bar, gridDim.x, a.status)) return;
        g0 += cut;
        buf ^= 1;
        G = cut < gn ? (G > 1 ? G / 2 : 1) : (G < kMaskG ? G * 2 : kMaskG);
    }
    if (blockIdx.x == 0 && threadIdx.x < a.B) {
        const int b = threadIdx.x;
        a.bucket_n[b] = s_n[b];
        a.bucket_cov[b] = s_cov[b];
        if (a.stats) {
            long long *st = a.stats + 6 * ((int64_t)a.P + b);
            st[0] = (long long)t_begin;
            st[1] = (long long)global_ns();
            st[2] = s_eval[b];
            st[3] = s_n[b];
            st[4] = s_scan[b];
            st[5] = 0;
        }
    }
}

// Streaming buckets, one block each, over a bitmap in shared memory (Alg. 5, run
// after the local greedy has finished; theta <= kSmallBits).  For short
// streams and many buckets: the stage is then a chain of decisions, not a
// scan, and the chain of one bucket lives within one SM -- block barriers where
// k_rg_stream_masks has grid barriers, and no bucket waits for another's cut.
//
// The block takes kSmallThreads stream slots at a time, keeps those whose
// subset reaches the bucket's threshold at all, and counts the gains of 32 of
// them against the bucket as it stands, in pieces of kSmallPiece entries over
// all warps.  The first that reaches the threshold is accepted (the slots
// before it saw the same bucket); the slots behind it that fell short still
// do, since gains only shrink, so only those that passed are counted again.
// Hence a group costs one count and one short recount per accepted seed.
// Bound by that chain (a few hundred cycles a link), not by memory.  OPIM at
// k = 1,000 (94 buckets, 37,000 slots, 10,780 sets): 36.6 -> 2.07 ms against a
// cluster per bucket counting one candidate at a time.
// The line to the masks: with B <= 64 the masks read every subset once for all
// buckets, a block here reads it for its own.  At 2.7 x 10^6 members the masks
// take 0.56 ms, the blocks 0.69; over the 24 RandGreedi queries of the batched
// mix 12.5 ms with the line at 2^20 members, 13.4 without the blocks, 40.4 with
// it at 2^24.  With B > 64 the other choice is the cluster kernel, which reads
// as much and one candidate at a time.
constexpr int kSmallThreads = 512;
constexpr int kSmallPiece = 256;             // entries of a subset a warp counts at once
constexpr int64_t kSmallBits = 1600 * 1024;  // sets whose bitmap fits (200 KB)
constexpr int64_t kSmallTotal = 1 << 20;     // pool members from which a stream counts as long

// The stream's slots as {element or -1, |S(x)|} and the subset's first entry.
__global__ void k_rg_slots(RGArgs a) {
    const int64_t nslots = (int64_t)a.trunc * a.P;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nslots;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t x = a.flags[t] == 1u ? a.elems[t] : -1;
        const int64_t b = x >= 0 ? a.vtx_off[x] : 0;
        a.slot_x[t] = x;
        a.slot_beg[t] = b;
        a.slot_len[t] = x >= 0 ? a.vtx_off[x + 1] - b : 0;
    }
}

__global__ void __launch_bounds__(kSmallThreads) k_rg_stream_small(RGArgs a) {
    extern __shared__ uint32_t bits[];       // [ceil(theta / 32)]
    constexpr int kWarpsS = kSmallThreads / 32;
    __shared__ int32_t s_x[kSmallThreads], s_len[kSmallThreads];
    __shared__ int64_t s_beg[kSmallThreads];
    __shared__ int32_t s_gain[32], s_off[33];
    __shared__ int32_t s_wcnt[kWarpsS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t nslots = (int64_t)a.trunc * a.P;
    for (int b = blockIdx.x; b < a.B; b += gridDim.x) {
        for (int64_t x = threadIdx.x; x < a.words; x += blockDim.x) bits[x] = 0u;
        const int64_t T = a.thr[b];
        const uint64_t t_begin = global_ns();
        long long n_eval = 0, scanned = 0;
        int32_t bn = 0;
        int64_t bcov = 0;
        for (int64_t base = 0; base < nslots && bn < a.k; base += kSmallThreads) {
            // ---- the window's slots that can pass, in stream order
            __syncthreads();                 // the last group has been read; bits are cleared
            const int64_t t = base + threadIdx.x;
            const int32_t x = t < nslots ? __ldg(a.slot_x + t) : -1;
            const int64_t len = t < nslots ? __ldg(a.slot_len + t) : 0;
            const bool keep = x >= 0 && len >= T;
            const unsigned km = __ballot_sync(kFull, keep);
            if (lane == 0) s_wcnt[warp] = __popc(km);
            __syncthreads();
            int before = 0, nc = 0;
            for (int w = 0; w < kWarpsS; ++w) {
                if (w < warp) before += s_wcnt[w];
                nc += s_wcnt[w];
            }
            if (keep) {
                const int at = before + __popc(km & lt);
                s_x[at] = x;
                s_len[at] = (int32_t)len;    // |S(x)| <= theta <= kSmallBits
                s_beg[at] = __ldg(a.slot_beg + t);
            }
            __syncthreads();
            for (int c0 = 0; c0 < nc && bn < a.k; c0 += 32) {
                // lane u of every warp stands for slot c0 + u
                const int32_t my_len = c0 + lane < nc ? s_len[c0 + lane] : 0;
                unsigned todo = nc - c0 < 32 ? (1u << (nc - c0)) - 1u : kFull;
                n_eval += __popc(todo);
                for (;;) {
                    if (warp == 0) {
                        const int32_t pieces = todo >> lane & 1u ? (my_len + kSmallPiece - 1) / kSmallPiece : 0;
                        const int32_t incl = warp_incl_scan<int32_t>(pieces, lane);
                        s_off[lane] = incl - pieces;
                        if (lane == 31) s_off[32] = incl;
                        s_gain[lane] = 0;
                    }
                    __syncthreads();         // also: the accepted subset is in the bitmap
                    const int32_t my_off = s_off[lane], total = s_off[32];
                    for (int32_t c = warp; c < total; c += kWarpsS) {
                        // the last slot of todo that starts at or before piece c
                        const unsigned at = __ballot_sync(kFull, (todo >> lane & 1u) && my_off <= c);
                        const int u = 31 - __clz(at);
                        const int32_t e0 = (c - __shfl_sync(kFull, my_off, u)) * kSmallPiece;
                        const int32_t n = s_len[c0 + u];
                        const int32_t *ids = a.set_ids + s_beg[c0 + u];
                        int32_t id[kSmallPiece / 32];
#pragma unroll
                        for (int q = 0; q < kSmallPiece / 32; ++q) {
                            const int32_t i = e0 + q * 32 + lane;
                            id[q] = i < n ? __ldg(ids + i) : -1;
                        }
                        int miss = 0;
#pragma unroll
                        for (int q = 0; q < kSmallPiece / 32; ++q)
                            if (id[q] >= 0) miss += !((bits[id[q] >> 5] >> (id[q] & 31)) & 1u);
                        miss = __reduce_add_sync(kFull, miss);
                        if (lane == 0 && miss) atomicAdd(&s_gain[u], miss);
                    }
                    __syncthreads();
                    const int32_t g = s_gain[lane];
                    const unsigned pass = __ballot_sync(kFull, (todo >> lane & 1u) && (int64_t)g >= T);
                    scanned += (long long)__reduce_add_sync(kFull, todo >> lane & 1u ? my_len : 0);
                    if (!pass) break;
                    const int u = __ffs(pass) - 1;
                    const int32_t gain = __shfl_sync(kFull, g, u);
                    if (threadIdx.x == 0) {
                        a.bucket_seeds[(int64_t)b * a.k + bn] = s_x[c0 + u];
                        a.bucket_gains[(int64_t)b * a.k + bn] = gain;
                    }
                    ++bn;
                    bcov += gain;
                    if (bn == a.k) break;
                    const int32_t n = s_len[c0 + u];
                    const int32_t *ids = a.set_ids + s_beg[c0 + u];
                    for (int32_t i = threadIdx.x; i < n; i += kSmallThreads) {
                        const int32_t id = __ldg(ids + i);
                        atomicOr(&bits[id >> 5], 1u << (id & 31));
                    }
                    todo = pass & ~((2u << u) - 1u);
                    if (!todo) break;
                    __syncthreads();         // s_gain and s_off have been read by every warp
                }
                __syncthreads();             // likewise, and the bitmap is complete
            }
        }
        if (threadIdx.x == 0) {
            a.bucket_n[b] = bn;
            a.bucket_cov[b] = bcov;
            if (a.stats) {
                long long *st = a.stats + 6 * ((int64_t)a.P + b);
                st[0] = (long long)t_begin;
                st[1] = (long long)global_ns();
                st[2] = n_eval;
                st[3] = bn;
                st[4] = scanned;
                st[5] = 0;
            }
        }
        __syncthreads();
    }
}

// Alg. 4's final compare: best bucket (ties: smallest b) against the best
// local solution (ties: smallest p); the bucket wins ties.  One block: maxima by
// block reductions, the winner's seeds copied by all threads (one thread
// walking both lists took 85 us at P = 148, k = 1,000).
constexpr int kFinalThreads = 256;

// The largest of cov[0 .. n) and its smallest index, by the whole block.
__device__ __forceinline__ int64_t best_coverage(const int64_t *cov, int n, int *at,
                                                 unsigned long long *shm) {
    unsigned long long m = 0;                // coverage + 1
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const unsigned long long c = (unsigned long long)cov[i] + 1ull;
        m = c > m ? c : m;
    }
    m = block_max_u64(m, shm);
    unsigned long long k = 0;                // 2^32 - index
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        if ((unsigned long long)cov[i] + 1ull == m && (1ull << 32) - i > k) k = (1ull << 32) - i;
    *at = (int)((1ull << 32) - block_max_u64(k, shm));
    return (int64_t)m - 1;
}

__global__ void __launch_bounds__(kFinalThreads) k_rg_final(RGArgs a, int32_t *seeds, int64_t *gains,
                                                            int32_t *nseeds, int64_t *coverage,
                                                            int32_t *chosen) {
    __shared__ unsigned long long shm[33];
    int b, p;
    const int64_t bcov = best_coverage(a.bucket_cov, a.B, &b, shm);
    const int64_t pcov = best_coverage(a.local_cov, a.P, &p, shm);
    const bool bucket = bcov >= pcov;
    const int32_t m = bucket ? a.bucket_n[b] : a.local_n[p];
    const int32_t *s = bucket ? a.bucket_seeds + (int64_t)b * a.k : a.local_seeds + (int64_t)p * a.k;
    const int64_t *g = bucket ? a.bucket_gains + (int64_t)b * a.k : a.local_gains + (int64_t)p * a.k;
    for (int32_t j = threadIdx.x; j < m; j += kFinalThreads) {
        seeds[j] = s[j];
        gains[j] = g[j];
    }
    if (threadIdx.x == 0) {
        *chosen = bucket ? -1 : p;
        *nseeds = m;
        *coverage = bucket ? bcov : pcov;
    }
}

}  // namespace

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

int32_t num_buckets(int32_t k, double delta) {
    double x = 1.0;
    int32_t b = 0;
    while (x < (double)k) {
        x *= 1.0 + delta;
        ++b;
    }
    return b < 1 ? 1 : b;
}

im_status greedy_plain(im_pool *p, int32_t k, int32_t *d_seeds, int64_t *d_gains,
                       int32_t *d_nseeds, int64_t *d_cov, cudaStream_t st, int *d_status) {
    const int64_t n = p->g->n, theta = p->theta;
    int per_sm = 0;
    IM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_greedy, kGreedyThreads, 0));
    if (per_sm < 1) return IM_ERR_UNSUPPORTED;
    const int grid = per_sm * num_sms();
    const int64_t words = (theta + 31) / 32;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t at = off;
        off += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const int32_t cand_shift = (int32_t)tune_value(IM_TUNE_GREEDY_HOT);
    const int64_t vwords = (n + 31) / 32;
    const size_t o_cnt = take((size_t)vwords * 32 * 4),
                 o_cov = take((size_t)std::max<int64_t>(words, 1) * 4),
                 o_best = take(3 * 8), o_bar = take(sizeof(GridBarrier)),
                 o_work = take(16), o_hrank = take((size_t)n * 4),
                 o_hcnt = take((size_t)kHubCap * kHubRep * 4), o_hlist = take((size_t)kHubCap * 4),
                 o_cand = take((size_t)n * 4), o_ctl = take(32),
                 o_piece = take((size_t)(2 * p->total / kGreedyPiece + 1) * 8);
    void *base = nullptr;
    im_status s = pool_scratch(p, off, &base);
    if (s != IM_OK) return s;
    char *B = (char *)base;
    IM_CUDA(cudaMemsetAsync(B + o_bar, 0, sizeof(GridBarrier), st));
    IM_CUDA(cudaMemsetAsync(B + o_work, 0, 16, st));
    IM_CUDA(cudaMemsetAsync(B + o_ctl, 0, 32, st));
    IM_CUDA(cudaMemsetAsync(d_nseeds, 0, sizeof(int32_t), st));
    IM_CUDA(cudaMemsetAsync(d_cov, 0, sizeof(int64_t), st));
    GreedyArgs a;
    std::memset(&a, 0, sizeof(a));
    a.n = n;
    a.theta = theta;
    a.set_off = p->set_off;
    a.members = p->members;
    a.vtx_off = p->vtx_off;
    a.set_ids = p->set_ids;
    a.k = k;
    a.counts = (int32_t *)(B + o_cnt);
    a.covered = (uint32_t *)(B + o_cov);
    a.gmax = (unsigned long long *)(B + o_best);
    a.bar = (GridBarrier *)(B + o_bar);
    a.seeds = d_seeds;
    a.gains = d_gains;
    a.nseeds = d_nseeds;
    a.coverage = d_cov;
    a.status = d_status;
    a.spread = 1;
    a.hub_rank = (int32_t *)(B + o_hrank);
    a.hub_cnt = (int32_t *)(B + o_hcnt);
    a.hub_list = (int32_t *)(B + o_hlist);
    a.cand = (int32_t *)(B + o_cand);
    a.ctl = (int32_t *)(B + o_ctl);
    a.hub_cap = kHubCap;
    a.hub_shift = kHubShift;
    a.cand_shift = cand_shift;
    a.work = (unsigned long long *)(B + o_work);
    a.piece = (unsigned long long *)(B + o_piece);
    a.npiece = (unsigned long long *)(B + o_ctl + 16);
    void *args[] = {&a};
    KernelTimer kt(st, "greedy");
    IM_CUDA(cudaLaunchCooperativeKernel((const void *)k_greedy, dim3(grid), dim3(kGreedyThreads),
                                        args, 0, st));
    return IM_OK;
}

// Launches the standard greedy kernel on caller-provided scratch (used by the
// allocation-free entry point in noalloc.cu).
im_status greedy_launch(int64_t n, int64_t theta, const int64_t *set_off, const int32_t *members,
                        const int64_t *vtx_off, const int32_t *set_ids, int32_t k, int32_t *counts,
                        uint32_t *covered, unsigned long long *block_best, int max_grid,
                        void *barrier, int32_t *seeds, int64_t *gains, int32_t *nseeds,
                        int64_t *coverage, int *status, cudaStream_t st) {
    int per_sm = 0;
    IM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_greedy, kGreedyThreads, 0));
    if (per_sm < 1) return IM_ERR_UNSUPPORTED;
    const int grid = std::min(per_sm * num_sms(), max_grid);
    GreedyArgs a;
    std::memset(&a, 0, sizeof(a));
    a.n = n;
    a.theta = theta;
    a.set_off = set_off;
    a.members = members;
    a.vtx_off = vtx_off;
    a.set_ids = set_ids;
    a.k = k;
    a.counts = counts;
    a.covered = covered;
    a.gmax = block_best;
    a.bar = (GridBarrier *)barrier;
    a.seeds = seeds;
    a.gains = gains;
    a.nseeds = nseeds;
    a.coverage = coverage;
    a.status = status;
    void *args[] = {&a};
    KernelTimer kt(st, "greedy");
    IM_CUDA(cudaLaunchCooperativeKernel((const void *)k_greedy, dim3(grid), dim3(kGreedyThreads),
                                        args, 0, st));
    return IM_OK;
}

// Queries of a batch: scratch of greedy_many for queries of n[] vertices and
// `members` members in all (its own arrays; counts, ranks and candidates come with
// the queries).
constexpr int32_t kManyHubs = 1024;     // hub rows of a query at most

namespace {
struct ManyState {                      // zeroed before the launch
    GridBarrier bar;
    unsigned long long work[2], npiece, gmax[3];
    int32_t ctl[4];
};
size_t many_pieces(int64_t members) { return (size_t)(2 * members / kGreedyPiece + 1); }
}  // namespace

int64_t greedy_hub_rows(int64_t n) { return std::min<int64_t>(n, kManyHubs); }

size_t greedy_query_bytes(int64_t n) {
    return sizeof(GreedyArgs) + 4 + sizeof(ManyState) + (size_t)greedy_hub_rows(n) * (kHubRep + 1) * 4 + 8;
}

size_t greedy_many_scratch(const std::vector<int64_t> &n, int64_t members) {
    size_t rows = 0;
    for (const int64_t x : n) rows += (size_t)greedy_hub_rows(x);
    const size_t nq = n.size();
    return align256(nq * sizeof(GreedyArgs)) + align256((nq + 1) * 4) + align256(nq * sizeof(ManyState)) +
           align256(rows * kHubRep * 4) + align256(rows * 4) + align256((many_pieces(members) + nq) * 8);
}

im_status greedy_many(const std::vector<GreedyQuery> &qs, const int64_t *set_off,
                      const int32_t *members, const int32_t *set_ids, void *scratch, int *status,
                      cudaStream_t st) {
    const int32_t nq = (int32_t)qs.size();
    if (nq == 0) return IM_OK;
    int per_sm = 0;
    IM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_greedy_many, kGreedyThreads, 0));
    if (per_sm < 1) return IM_ERR_UNSUPPORTED;
    const int grid = std::min(per_sm, 2) * num_sms();
    int64_t total = 0;
    size_t rows = 0;
    for (const GreedyQuery &q : qs) {
        total += q.members;
        rows += (size_t)greedy_hub_rows(q.n);
    }
    char *B = (char *)scratch;
    auto take = [&](size_t bytes) {
        char *r = B;
        B += align256(bytes);
        return r;
    };
    GreedyArgs *tab = (GreedyArgs *)take((size_t)nq * sizeof(GreedyArgs));
    int32_t *first = (int32_t *)take((size_t)(nq + 1) * 4);
    ManyState *state = (ManyState *)take((size_t)nq * sizeof(ManyState));
    int32_t *hub_cnt = (int32_t *)take(rows * kHubRep * 4);
    int32_t *hub_list = (int32_t *)take(rows * 4);
    unsigned long long *piece = (unsigned long long *)take((many_pieces(total) + (size_t)nq) * 8);

    // largest first; blocks by weight: the members a query may decrement, and a
    // floor for its steps
    std::vector<int32_t> order(nq);
    for (int32_t i = 0; i < nq; ++i) order[i] = i;
    auto weight = [&](int32_t i) { return (double)qs[i].members + 2e4 * (double)qs[i].k; };
    std::stable_sort(order.begin(), order.end(),
                     [&](int32_t x, int32_t y) { return weight(x) > weight(y); });
    const int32_t groups = std::min<int32_t>(nq, grid);
    double sum = 0.0;
    for (int32_t g = 0; g < groups; ++g) sum += weight(order[g]);
    std::vector<int32_t> hfirst(groups + 1, 0), blocks(groups, 1);
    int32_t left = grid - groups;
    for (int32_t g = 0; g < groups; ++g) {
        const int32_t more = std::min<int32_t>(
            left, std::max<int32_t>(0, (int32_t)((double)grid * weight(order[g]) / sum) - 1));
        blocks[g] += more;
        left -= more;
    }
    for (int32_t g = 0; left > 0; g = (g + 1) % groups, --left) ++blocks[g];
    for (int32_t g = 0; g < groups; ++g) hfirst[g + 1] = hfirst[g] + blocks[g];

    const int32_t cand_shift = (int32_t)tune_value(IM_TUNE_GREEDY_HOT);
    std::vector<GreedyArgs> h(nq);
    size_t at = 0, row = 0;
    for (int32_t r = 0; r < nq; ++r) {
        const GreedyQuery &q = qs[order[r]];
        GreedyArgs &a = h[r];
        std::memset(&a, 0, sizeof(a));
        a.n = q.n;
        a.theta = q.theta;
        a.set_off = set_off;
        a.members = members;
        a.vtx_off = q.vtx_off;
        a.set_ids = set_ids;
        a.k = q.k;
        a.counts = q.counts;
        a.covered = q.covered;
        a.gmax = state[r].gmax;
        a.bar = &state[r].bar;
        a.seeds = q.seeds;
        a.gains = q.gains;
        a.nseeds = q.nseeds;
        a.coverage = q.coverage;
        a.status = status;
        a.sshift = q.sshift;
        a.vshift = q.vshift;
        a.hub_rank = q.ranks;
        a.hub_cnt = hub_cnt + row * kHubRep;
        a.hub_list = hub_list + row;
        a.cand = q.cands;
        a.ctl = state[r].ctl;
        a.hub_cap = (int32_t)greedy_hub_rows(q.n);
        row += (size_t)a.hub_cap;
        a.hub_shift = kHubShift;
        a.cand_shift = cand_shift;
        a.work = state[r].work;
        a.piece = piece + at;
        a.npiece = &state[r].npiece;
        at += many_pieces(q.members);
    }
    IM_CUDA(cudaMemcpyAsync(tab, h.data(), (size_t)nq * sizeof(GreedyArgs), cudaMemcpyHostToDevice, st));
    IM_CUDA(cudaMemcpyAsync(first, hfirst.data(), (size_t)(groups + 1) * 4, cudaMemcpyHostToDevice, st));
    IM_CUDA(cudaMemsetAsync(state, 0, (size_t)nq * sizeof(ManyState), st));
    const GreedyArgs *ctab = tab;
    const int32_t *cfirst = first;
    int32_t cnq = nq, cgroups = groups;
    void *args[] = {&ctab, &cnq, &cfirst, &cgroups};
    KernelTimer kt(st, "greedy_many");
    IM_CUDA(cudaLaunchCooperativeKernel((const void *)k_greedy_many, dim3(grid),
                                        dim3(kGreedyThreads), args, 0, st));
    return IM_OK;
}

im_status randgreedi(im_pool *p, int32_t k, const im_cover_opts *o, int32_t *d_seeds,
                     int64_t *d_gains, int32_t *d_nseeds, int64_t *d_cov, cudaStream_t st,
                     int *d_status) {
    const int32_t P = o->partitions;
    const int64_t n = p->g->n, theta = p->theta;
    const int64_t words = std::max<int64_t>(1, (theta + 31) / 32);
    // IM_AGG_GREEDY: Alg. 4's global step as written -- a greedy (the lazy one
    // of Alg. 2) over the union of the gathered local seeds -- reported as a
    // single "bucket" 0 without a threshold
    const bool naive = o->aggregator == IM_AGG_GREEDY;
    const int32_t B = naive ? 1 : num_buckets(k, o->delta);
    int64_t tr = ((int64_t)k * o->alpha_num + o->alpha_den - 1) / o->alpha_den;
    const int32_t trunc = (int32_t)std::max<int64_t>(1, std::min<int64_t>(k, tr));

    im_status s = build_partition(p, P, o->partition_seed, st);
    if (s != IM_OK) return s;
    // the largest part sizes the producers' shared memory
    std::vector<int32_t> hoff(P + 1);
    IM_CUDA(cudaMemcpyAsync(hoff.data(), p->part_off, (P + 1) * 4, cudaMemcpyDeviceToHost, st));
    IM_CUDA(cudaStreamSynchronize(st));
    int32_t max_np = 0;
    for (int q = 0; q < P; ++q) max_np = std::max(max_np, hoff[q + 1] - hoff[q]);
    max_np = std::max((max_np + 1) & ~1, 2);             // (16-byte steps in shared memory)
    // key + stamp (4 bytes each per candidate) + one 8-byte maximum per 32
    size_t prod_smem = (size_t)max_np * 8 + (size_t)((max_np + 63) / 64) * 16;
    if (prod_smem > kProdSmemCap) {
        set_error("RandGreedi: a vertex part is too large for shared memory; use more partitions");
        return IM_ERR_UNSUPPORTED;
    }

    // result buffers kept in the pool for im_randgreedi_details
    const size_t need = align256((size_t)P * k * 4) + align256((size_t)P * k * 8) +
                        align256((size_t)P * 4) + align256((size_t)P * 8) +
                        align256((size_t)B * 8) * 2 + align256((size_t)B * 4) +
                        align256((size_t)B * k * 4) + align256((size_t)B * k * 8) +
                        align256((size_t)(P + B) * 6 * 8);
    if (p->rg_cap_bytes < need) {
        dev_free(p->rg_block);
        p->rg_block = nullptr;
        p->rg_cap_bytes = 0;
        IM_TRY(dev_alloc(&p->rg_block, need));
        p->rg_cap_bytes = need;
    }
    {
        char *R = (char *)p->rg_block;
        size_t at = 0;
        auto grab = [&](size_t bytes) {
            char *q = R + at;
            at += align256(bytes);
            return q;
        };
        p->rg_local_seeds = (int32_t *)grab((size_t)P * k * 4);
        p->rg_local_gains = (int64_t *)grab((size_t)P * k * 8);
        p->rg_local_n = (int32_t *)grab((size_t)P * 4);
        p->rg_local_cov = (int64_t *)grab((size_t)P * 8);
        p->rg_thr = (int64_t *)grab((size_t)B * 8);
        p->rg_bucket_cov = (int64_t *)grab((size_t)B * 8);
        p->rg_bucket_n = (int32_t *)grab((size_t)B * 4);
        p->rg_bucket_seeds = (int32_t *)grab((size_t)B * k * 4);
        p->rg_bucket_gains = (int64_t *)grab((size_t)B * k * 8);
        p->rg_stats = (long long *)grab((size_t)(P + B) * 6 * 8);
    }
    p->rg_P = P;
    p->rg_B = B;
    p->rg_k = k;

    // scratch: producer + bucket bitmaps, stream slots, flags, l
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t at = off;
        off += align256(bytes);
        return at;
    };
    // two-launch mode: the candidates' subsets, and the producers' bitmaps, in
    // shared memory where they fit beside the keys.  A bitmap in global memory
    // wants the L1 cache, which is what shared memory leaves of an SM's 256 KB:
    // beside one, the subsets go there only below kProdInfoCap (at 7,100
    // candidates and 4 x 10^6 sets, 177 KB: 3.49 ms against 2.82; at 2,050 and 2 x
    // 10^6, 49 KB: 1.74 against 1.94).
    const bool two = naive || o->fused == 0;
    const size_t info_bytes = (size_t)max_np * sizeof(uint4), bits_bytes = (size_t)words * 4;
    const bool smem_info = two && (prod_smem + info_bytes + bits_bytes <= kProdSmemCap ||
                                   prod_smem + info_bytes <= kProdInfoCap);
    if (smem_info) prod_smem += info_bytes;
    const size_t bits_smem = prod_smem + bits_bytes;
    const bool smem_bits = two && bits_smem <= kProdSmemCap;
    const size_t o_cov = take(smem_bits ? 0 : (size_t)P * words * 4);
    const size_t o_cinfo = take(smem_info ? 0 : (size_t)n * sizeof(uint4));
    const size_t o_flags = take((size_t)trunc * P * 4);
    const size_t o_elems = take((size_t)trunc * P * 4);
    const size_t o_l = take(64);
    // two-launch mode, automatic layout: a block per bucket where the bitmaps fit
    // and the stream is short (kSmallTotal) or has more buckets than a mask has
    // bits; else the bucket-mask stage (B <= 64)
    const bool automatic = !naive && o->fused == 0 && tune_value(IM_TUNE_RG_CLUSTER) == 0;
    const bool use_small = automatic && theta <= kSmallBits && (p->total <= kSmallTotal || B > 64);
    const bool use_masks = automatic && !use_small && B <= 64;
    const size_t o_mask = use_masks ? take((size_t)std::max<int64_t>(theta, 1) * 8) : 0;
    const size_t o_gbuf = use_masks ? take((size_t)2 * kMaskG * 64 * 4) : 0;
    const size_t o_bar = use_masks ? take(sizeof(GridBarrier)) : 0;
    const size_t o_bcov = take(use_masks || use_small || naive ? 0 : (size_t)B * words * 4);
    const bool slots = use_masks || use_small;
    const size_t o_sx = slots ? take((size_t)trunc * P * 4) : 0;
    const size_t o_sb = slots ? take((size_t)trunc * P * 8) : 0;
    const size_t o_sl = slots ? take((size_t)trunc * P * 8) : 0;
    const size_t o_lazy = naive ? take(lazy_greedy_scratch(n, theta)) : 0;
    void *base = nullptr;
    s = pool_scratch(p, off, &base);
    if (s != IM_OK) return s;
    char *Bs = (char *)base;
    IM_CUDA(cudaMemsetAsync(Bs + o_flags, 0, (size_t)trunc * P * 4, st));
    // l = max_v |S(v)|: a lower bound on the optimum of the stream, u = k l
    int64_t l = 0;
    if (!naive) {
        s = max_segment_length(p->vtx_off, n, (int64_t *)(Bs + o_l), st);
        if (s != IM_OK) return s;
        IM_CUDA(cudaMemcpyAsync(&l, Bs + o_l, 8, cudaMemcpyDeviceToHost, st));
        IM_CUDA(cudaStreamSynchronize(st));
    }
    std::vector<int64_t> thr(B, 0);
    if (!naive) {
        double guess = (double)l;
        for (int32_t b = 0; b < B; ++b) {
            thr[b] = (int64_t)std::ceil(guess / (2.0 * (double)k));
            guess *= 1.0 + o->delta;
        }
    }
    IM_CUDA(cudaMemcpyAsync(p->rg_thr, thr.data(), (size_t)B * 8, cudaMemcpyHostToDevice, st));

    RGArgs a;
    a.n = n;
    a.theta = theta;
    a.words = words;
    a.k = k;
    a.P = P;
    a.trunc = trunc;
    a.B = B;
    a.vtx_off = p->vtx_off;
    a.set_ids = p->set_ids;
    a.part_off = p->part_off;
    a.part_vtx = p->part_vtx;
    a.covered = (uint32_t *)(Bs + o_cov);
    a.cinfo = (uint4 *)(Bs + o_cinfo);
    a.cinfo_smem = smem_info;
    a.bcovered = (uint32_t *)(Bs + o_bcov);
    a.local_seeds = p->rg_local_seeds;
    a.local_gains = p->rg_local_gains;
    a.local_n = p->rg_local_n;
    a.local_cov = p->rg_local_cov;
    a.thr = p->rg_thr;
    a.bucket_cov = p->rg_bucket_cov;
    a.bucket_n = p->rg_bucket_n;
    a.bucket_seeds = p->rg_bucket_seeds;
    a.bucket_gains = p->rg_bucket_gains;
    a.flags = (uint32_t *)(Bs + o_flags);
    a.elems = (int32_t *)(Bs + o_elems);
    a.status = d_status;
    a.max_np = max_np;
    a.evals = (int32_t)std::min<int64_t>(kProdW, std::max<int64_t>(1, tune_value(IM_TUNE_RG_EVALS)));
    a.stats = p->rg_stats;
    a.mask = use_masks ? (unsigned long long *)(Bs + o_mask) : nullptr;
    a.gbuf = use_masks ? (uint32_t *)(Bs + o_gbuf) : nullptr;
    a.bar = use_masks ? (GridBarrier *)(Bs + o_bar) : nullptr;
    a.slot_x = slots ? (int32_t *)(Bs + o_sx) : nullptr;
    a.slot_beg = slots ? (int64_t *)(Bs + o_sb) : nullptr;
    a.slot_len = slots ? (int64_t *)(Bs + o_sl) : nullptr;
    if (use_masks) IM_CUDA(cudaMemsetAsync(Bs + o_bar, 0, sizeof(GridBarrier), st));

    IM_TRY(raise_dyn_smem((const void *)k_randgreedi, prod_smem));
    int per_sm = 0;
    IM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_randgreedi, kRGThreads,
                                                          prod_smem));
    if (per_sm < 1) return IM_ERR_UNSUPPORTED;
    const int resident = per_sm * num_sms();
    bool fused = !naive && o->fused != 0 && resident >= 2;
    if (fused) {
        a.ncons = std::min<int32_t>(B, resident / 2);
        a.nprod = std::min<int32_t>(P, resident - a.ncons);
        a.first_role = 0;
        void *args[] = {&a};
        KernelTimer kt(st, "randgreedi_fused");
        IM_CUDA(cudaLaunchCooperativeKernel((const void *)k_randgreedi,
                                            dim3(a.nprod + a.ncons), dim3(kRGThreads), args,
                                            prod_smem, st));
    } else {
        // producers alone, then consumers alone (the stream is complete by then)
        const size_t local_smem = smem_bits ? bits_smem : prod_smem;
        const void *local = smem_bits ? (const void *)k_rg_local<true> : (const void *)k_rg_local<false>;
        IM_TRY(raise_dyn_smem(local, local_smem));
        // more parts than SMs: smaller blocks, so that two parts share one
        int threads = kProdThreads;
        int per_l = 0;
        for (;; threads /= 2) {
            IM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_l, local, threads, local_smem));
            if (per_l * num_sms() >= P || threads <= kProdMinThreads) break;
        }
        if (per_l < 1) return IM_ERR_UNSUPPORTED;
        a.nprod = std::min<int32_t>(P, per_l * num_sms());
        a.ncons = 0;
        a.first_role = 0;
        {
            KernelTimer kt(st, "randgreedi_local");
            if (smem_bits) k_rg_local<true><<<a.nprod, threads, local_smem, st>>>(a);
            else k_rg_local<false><<<a.nprod, threads, local_smem, st>>>(a);
        }
        IM_CUDA(cudaGetLastError());
        const int64_t want = tune_value(IM_TUNE_RG_CLUSTER);   // 0 auto, -1 off, 1..8
        if (naive) {
            // the global greedy over the first `trunc` seeds of every part
            int32_t W = (int32_t)tune_value(IM_TUNE_GREEDY_EVALS);
            if (W <= 0) W = 16;
            IM_CUDA(cudaMemsetAsync(p->rg_bucket_n, 0, sizeof(int32_t), st));
            IM_CUDA(cudaMemsetAsync(p->rg_bucket_cov, 0, sizeof(int64_t), st));
            IM_CUDA(cudaMemsetAsync(p->rg_stats + (size_t)P * 6, 0, 6 * 8, st));
            s = greedy_lazy_launch(n, theta, p->vtx_off, p->set_ids, k, W, Bs + o_lazy,
                                   p->rg_bucket_seeds, p->rg_bucket_gains, p->rg_bucket_n,
                                   p->rg_bucket_cov, p->lz_stats, d_status, st,
                                   p->rg_local_seeds, p->rg_local_n, P, trunc, k);
            if (s != IM_OK) return s;
        } else if (use_small) {
            const size_t smem = (size_t)words * 4;
            IM_TRY(raise_dyn_smem((const void *)k_rg_stream_small, smem));
            KernelTimer kt(st, "randgreedi_stream");
            k_rg_slots<<<num_sms(), 256, 0, st>>>(a);
            k_rg_stream_small<<<B, kSmallThreads, smem, st>>>(a);
            IM_CUDA(cudaGetLastError());
        } else if (use_masks) {
            // buckets: one pass over each streamed subset serves all buckets
            int per = 0;
            IM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_rg_stream_masks,
                                                                  kRGThreads, 0));
            if (per < 1) return IM_ERR_UNSUPPORTED;
            // one block an SM: 128 registers a thread fit no second (at 64, two
            // blocks measured 2.07 ms against 2.03)
            const int grid = num_sms();
            void *args[] = {&a};
            KernelTimer kt(st, "randgreedi_stream");
            IM_CUDA(cudaLaunchCooperativeKernel((const void *)k_rg_stream_masks, dim3(grid),
                                                dim3(kRGThreads), args, 0, st));
        }
        // buckets: shared-memory bitmaps split over a cluster when theta fits
        int CS = want > 0 ? (int)want : 1;
        int64_t R = 0;
        size_t csmem = 0;
        for (; CS <= 8; CS *= 2) {
            R = (theta + (int64_t)CS * 32 - 1) / ((int64_t)CS * 32) * 32;
            csmem = (size_t)(R / 8) + 2 * kSpec * sizeof(unsigned);
            if (csmem <= kClusterSmemCap) break;
        }
        if (want < 0) CS = 16;   // global-memory bitmaps requested
        if (naive || use_masks || use_small) {
            // done above
        } else if (CS <= 8) {
            unsigned *counter = (unsigned *)(Bs + o_l) + 2;
            IM_CUDA(cudaMemsetAsync(counter, 0, sizeof(unsigned), st));
            IM_TRY(raise_dyn_smem((const void *)k_rg_stream_cluster, csmem));
            const int nclusters = std::max(1, std::min<int>(B, num_sms() / CS));
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(nclusters * CS);
            cfg.blockDim = dim3(kRGThreads);
            cfg.dynamicSmemBytes = csmem;
            cfg.stream = st;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = CS;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            KernelTimer kt(st, "randgreedi_stream");
            IM_CUDA(cudaLaunchKernelEx(&cfg, k_rg_stream_cluster, a, R, counter));
        } else {
            a.ncons = std::min<int32_t>(B, resident);
            a.first_role = 1;
            {
                KernelTimer kt(st, "randgreedi_stream");
                k_randgreedi<<<a.ncons, kRGThreads, prod_smem, st>>>(a);
            }
            IM_CUDA(cudaGetLastError());
        }
    }
    int32_t *d_chosen = (int32_t *)(Bs + o_l);   // l is no longer needed
    {
        KernelTimer kt(st, "randgreedi_final");
        k_rg_final<<<1, kFinalThreads, 0, st>>>(a, d_seeds, d_gains, d_nseeds, d_cov, d_chosen);
    }
    IM_CUDA(cudaGetLastError());
    int32_t chosen = 0;
    IM_CUDA(cudaMemcpyAsync(&chosen, d_chosen, 4, cudaMemcpyDeviceToHost, st));
    IM_CUDA(cudaStreamSynchronize(st));
    p->rg_chosen = chosen;
    return IM_OK;
}

}  // namespace im
