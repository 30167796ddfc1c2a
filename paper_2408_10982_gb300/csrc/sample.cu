// sample.cu -- RRR sampling (IC reverse BFS, LT backward walk), compaction into
// the pool's CSR, and the segmented sorts that put every set in ascending order.
//
// Every sampler is a persistent kernel that takes the next sample id from a
// global counter (dynamic balancing: set sizes are heavy tailed on R-MAT).
// IC (Def. 3 under the IC live-edge world): one warp per sample expands up to
// 32 queued vertices at once, four coins to a Philox call; live edges are
// listed and followed 32 at a time.  Sets that percolate, or outgrow the warp's
// queue, are finished by k_sample_ic_big, one block per sample.  LT:
// k_sample_lt1 (default) runs one walk per thread; the picked in-edge (first
// edge whose running weight sum exceeds the draw) comes from one division when
// the vertex's in-edges weigh the same, else from a cut-point table in O(1)
// expected loads, and revisits are tested through a per-walk Bloom filter
// (flagged walks are checked exactly, two at a time).  k_sample_lt<G> runs a
// walk per group of G lanes, picking by the same division or over a fanout-32
// search tree (a tuning-knob alternative, and the second pass for walks longer
// than the thread kernel's queue).  The LT index they read (vertex records;
// running sums, tree and cut points only when some vertex's in-edges weigh
// differently) is built once per graph by build_lt_index: in-lists of up to 32
// edges get their running sums from one thread each, up to 1024 from a warp,
// longer ones from a block.
#include <algorithm>
#include <mutex>

#include "internal.cuh"

namespace im {

namespace {

constexpr int kSampleThreads = 256;          // 8 warps per block
constexpr int kWarps = kSampleThreads / 32;
constexpr int64_t kSmemVisBits = 1 << 15;    // IC visited bitmap in shared memory when n <= this
constexpr int kPathSmem = 256;               // LT path entries mirrored in smem (warp walks)
constexpr int kPathSmemGroup = 64;           // ... per walk when a warp runs several walks
constexpr int64_t kQueueCapIC = 1 << 14;     // per-warp queue entries (first pass)
constexpr int64_t kQueueCapLT = 1 << 11;
constexpr int kWarpSortKeys = 1024;          // sets up to this length are sorted by one warp
// set in stage_off of a set that lies in the stage in ascending order already
constexpr int64_t kStageAscending = (int64_t)1 << 62;
constexpr int kBlockSortCap = 16384;         // ... by one block in shared memory (int32)

// An IC sample that a warp handed over: its members so far are hand[off .. off +
// tail), of which the first `head` are expanded (examined in-edges so far).  tail is
// at least kICWarpFront, so that off / kICWarpFront is a place of its own in the
// table, and the table is as long as the buffer of members allows, whatever the
// number of samples.  The entry in ovf_list is the sample's index, with that
// place + 1 in the bits from kHandedShift on; 0 there: start again from the root.
struct Handed {
    int64_t off;
    unsigned long long examined;
    int32_t head, tail;
};
constexpr int kHandedShift = 44;

struct SampleArgs {
    const QueryView *qv;      // [nq] graphs and streams of the queries of this launch
    const int64_t *qstart;    // [nq + 1] first flattened sample index of each query
    int32_t nq;
    int64_t count;            // work items
    const int64_t *list;      // if non-null: work item i is sample index list[i]
    int32_t *stage;
    int64_t stage_cap;
    unsigned long long *stage_cursor;
    int64_t *stage_off;       // [count of the call]
    int32_t *sizes;           // [count of the call]; -1 marks a queue overflow
    int32_t *queues;
    int64_t qcap;
    uint32_t *gvis;
    int64_t vis_words;
    unsigned long long *examined;
    unsigned long long *alg_bytes;
    unsigned long long *work;
    int64_t *ovf_list;
    unsigned long long *ovf_count;
    int *status;
    struct Handed *handed;    // [hand_cap / kICWarpFront + 1] state of handed-over samples (IC)
    int32_t *hand;            // their members
    int64_t hand_cap;
    unsigned long long *hand_cursor;
    uint2 *recs;              // LT walks: {sample, first entry} of finished walks, [warp][k][lane]
    unsigned long long *nlong;    // sets longer than kWarpSortKeys, plus 2^32 for every
                                  // unsorted one longer than kBlockSortCap
    uint32_t rk[20];          // Philox round keys of the launch's query, when it has only one
};

// The query that flattened sample index j belongs to (largest q, qstart[q] <= j).
__device__ __forceinline__ int find_query(const SampleArgs &a, int64_t j) {
    int lo = 0, hi = a.nq - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(a.qstart + mid) <= j) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}


// ---------------------------------------------------------------------------
// IC: stochastic reverse BFS.  Edge e of sample s is live iff lane (e & 3) of
// Philox(s, e >> 2 (low word), e >> 34, coin tag) is below w[e].
//
// The bound is the coins: every in-edge of every member takes one, four to a
// Philox call, so the kernels are built around an inner loop that is little
// more than the ten rounds.  Three things keep it that small.
//   - m < 2^31, so the counter's third word is 0 and the first word is the
//     sample id: of the first three rounds only two products depend on the
//     edge (CoinStream), the rest is computed once a sample.
//   - A vertex whose in-edges all weigh the same (weighted cascade, uniform p)
//     takes its threshold from its record (im_graph.ic_rec): no weights are
//     read at all.  Sources are read only for live edges.
//   - Live edges are rare (a few per hundred, or per ten thousand under
//     weighted cascade).  The loop only lists them, in shared memory; when a
//     warp has 32, its lanes take one each: source, visited test, append.
//     So the long-latency part (source load, bitmap atomic) runs with 32
//     lanes busy and once per 32 live edges, not inside the coin loop.
// A warp expands up to 32 queued vertices together: those with at least
// kICWide edge groups one after another on all lanes (no search for an edge's
// owner), the short lists packed.
// Measured against one lane loop that loaded weights and sources with every
// group and claimed live sources where it found them: weighted cascade on the
// LiveJournal shape (IMM, 1.6 x 10^11 coins) 597 -> 130 ms, U[0, 0.1] at scale
// 20 (9.8 x 10^9 coins) 55 -> 24.5 ms, trivalency on the LiveJournal shape
// (6.3 x 10^9) 45 -> 20.7 ms.  ncu, weighted cascade at scale 15: 126
// instructions per 128 coins, issue 64 % and ALU and FMA-heavy pipes 59 % busy
// while DRAM is idle, so what is left is the instructions of the coins.  Tried
// and not kept: one call site for all kinds of lists (a state machine; fewer
// instruction-fetch stalls, more instructions: 31.5 against 23.5 ms at scale
// 20); lists from 12 groups on for the whole warp (26.1 against 23.5 ms).
// ---------------------------------------------------------------------------
constexpr int kICWide = 64;                  // edge groups from which a vertex gets the whole warp
constexpr int kCandCap = 32 + 128;           // listed live edges of a warp: < 32 left over + 128 new
constexpr int kICQueueSmem = 384;            // queue entries of a warp in shared memory
constexpr int kICHash = 1024;                // visited-set slots of a warp (n > kSmemVisBits)
constexpr int kICHashMax = kICQueueSmem;              // members from which the visited set spills to a bitmap
// A warp leaves a sample to the second pass when it has expanded this many
// in-edges and this many members wait to be expanded.
constexpr uint32_t kICWideEdges = 1u << 16;
constexpr int32_t kICWarpFront = 1024;
constexpr int64_t kICHandCap = 1 << 23;      // members handed over to the second pass (32 MB)

// One sample's draws of one kind (TAG: coins of edge group g, or the LT pick of
// vertex g): Philox4x32-10 of counter (s, g, 0, TAG), with what does not depend
// on g computed by begin().  KEYS: the round keys come from rk (kernel
// parameters, so constant-bank operands); else they are kept in registers (HELD)
// or derived from k0, k1 as the rounds go.
template <uint32_t TAG, bool KEYS, bool HELD = false>
struct DrawStream {
    uint32_t k0, k1;
    uint32_t gx, c1, ca, cb, cc;
    uint32_t held[HELD ? 13 : 1];            // K0(3 .. 9), K1(4 .. 9)
    __device__ __forceinline__ uint32_t K0(const uint32_t *rk, int r) const {
        return KEYS ? rk[2 * r] : HELD && r >= 3 ? held[r - 3] : k0 + (uint32_t)r * 0x9E3779B9u;
    }
    __device__ __forceinline__ uint32_t K1(const uint32_t *rk, int r) const {
        return KEYS ? rk[2 * r + 1] : HELD && r >= 4 ? held[r + 3] : k1 + (uint32_t)r * 0xBB67AE85u;
    }
    __device__ __forceinline__ void begin(const uint32_t *rk, uint32_t s, uint32_t key0,
                                          uint32_t key1) {
        k0 = key0;
        k1 = key1;
        if (HELD) {
#pragma unroll
            for (int r = 3; r < 10; ++r) {
                held[r - 3] = k0 + (uint32_t)r * 0x9E3779B9u;
                if (r >= 4) held[r + 3] = k1 + (uint32_t)r * 0xBB67AE85u;
            }
            // (kept as values: not to be derived again in the coin loop)
#pragma unroll
            for (int i = 0; i < 13; ++i) asm volatile("" : "+r"(held[i]));
        }
        gx = K0(rk, 0);                                           // round 0: x = g ^ gx
        const uint32_t z1 = __umulhi(0xD2511F53u, s) ^ TAG ^ K1(rk, 0);
        c1 = (0xD2511F53u * s) ^ K1(rk, 1);                       // round 1: z = hi(a) ^ c1
        const uint32_t x2 = __umulhi(0xCD9E8D57u, z1) ^ K0(rk, 1);
        ca = (0xCD9E8D57u * z1) ^ K0(rk, 2);                      // round 2: x = hi(b) ^ ca
        cb = __umulhi(0xD2511F53u, x2) ^ K1(rk, 2);               //          z = lo(a) ^ cb
        cc = (0xD2511F53u * x2) ^ K1(rk, 3);                      // round 3: z = hi(a) ^ cc
    }
    __device__ __forceinline__ uint4 operator()(const uint32_t *rk, uint32_t g) const {
        auto wide = [](uint32_t m, uint32_t x, uint32_t &lo, uint32_t &hi) {
            const unsigned long long p = (unsigned long long)m * x;
            lo = (uint32_t)p;
            hi = (uint32_t)(p >> 32);
        };
        uint32_t al, ah, bl, bh, dl, dh, el, eh;
        wide(0xD2511F53u, g ^ gx, al, ah);
        wide(0xCD9E8D57u, ah ^ c1, bl, bh);
        wide(0xD2511F53u, bh ^ ca, dl, dh);
        wide(0xCD9E8D57u, al ^ cb, el, eh);
        uint4 x = make_uint4(eh ^ bl ^ K0(rk, 3), el, dh ^ cc, dl);
#pragma unroll
        for (int r = 4; r < 10; ++r) {
            wide(0xD2511F53u, x.x, al, ah);
            wide(0xCD9E8D57u, x.z, bl, bh);
            x = make_uint4(bh ^ x.y ^ K0(rk, r), bl, ah ^ x.w ^ K1(rk, r), al);
        }
        return x;
    }
};

template <bool KEYS, bool HELD = false>
using CoinStream = DrawStream<kStreamCoin, KEYS, HELD>;
template <bool KEYS>
using PickStream = DrawStream<kStreamPick, KEYS>;

// What a warp expands: the in-edge lists of up to 32 vertices, one per lane.
struct ICItem {
    uint32_t eb, ee;     // in-edges [eb, ee)
    uint32_t w;          // their common threshold, when equal
    uint32_t equal;      // 1: all in-edges weigh w
};

__device__ __forceinline__ ICItem ic_item(const uint4 *rec, uint32_t v) {
    const uint4 r = __ldg(rec + v);
    return ICItem{r.x, r.x + r.y, r.z, r.w};
}

// Edge groups (of four, aligned) of an item; 0 when no in-edge can be live.
__device__ __forceinline__ uint32_t ic_groups(const ICItem &it) {
    if (it.ee == it.eb || (it.equal && it.w == 0u)) return 0u;
    return ((it.ee - 1u) >> 2) - (it.eb >> 2) + 1u;
}

// Live edges of group g within [eb, ee), as four bits, from its coins c and
// thresholds wv.
__device__ __forceinline__ uint32_t ic_live(const uint4 c, const uint4 wv, uint32_t g, uint32_t eb,
                                            uint32_t ee) {
    uint32_t m = (c.x < wv.x ? 1u : 0u) | (c.y < wv.y ? 2u : 0u) | (c.z < wv.z ? 4u : 0u) |
                 (c.w < wv.w ? 8u : 0u);
    const uint32_t e0 = g << 2;
    if (e0 < eb) m &= 15u << (eb - e0);                // first group
    if (e0 + 4u > ee) m &= 15u >> (e0 + 4u - ee);      // last group
    return m;
}

// Lists the live edges of the warp's groups (bits m of the group starting at
// edge e0) after the ncand listed before.
__device__ __forceinline__ void ic_list(uint32_t m, uint32_t e0, uint32_t *cand, int &ncand,
                                        int lane) {
    // the lane's place: the live edges of the lanes below it, from ballots of the
    // bits of their counts (one ballot per edge instead: 4 to 7 % slower)
    const unsigned lt = (1u << lane) - 1u;
    const int k = __popc(m);
    const unsigned b0 = __ballot_sync(kFull, k & 1), b1 = __ballot_sync(kFull, k & 2);
    int at = ncand + __popc(b0 & lt) + 2 * __popc(b1 & lt);
    ncand += __popc(b0) + 2 * __popc(b1);
    const unsigned b2 = __ballot_sync(kFull, k & 4);
    if (b2) {
        at += 4 * __popc(b2 & lt);
        ncand += 4 * __popc(b2);
    }
    while (m) {
        cand[at++] = e0 + (uint32_t)(__ffs(m) - 1);
        m &= m - 1u;
    }
}

// Calls visit(m, e0) for the groups with a live edge among groups [t0, n) of
// one in-list.  Equal weights: pairs of groups per lane, and the smallest coin
// of the warp's 64 groups decides whether any edge is live; the bits, and what
// lies outside the list in its first and last group, are looked at only then.
// Unequal weights: the next groups' are loaded while these are tested.
template <typename CS, typename F>
__device__ __forceinline__ void ic_expand_wide(const CS &cs, const uint32_t *rk,
                                               const uint32_t *wgt, const ICItem &o, uint32_t t0,
                                               uint32_t n, int lane, F &&visit) {
    const uint32_t g0 = o.eb >> 2;
    if (o.equal) {
        while (n - t0 >= 64u) {
            const uint32_t g = g0 + t0 + lane;
            const uint4 c0 = cs(rk, g), c1 = cs(rk, g + 32u);
            t0 += 64u;
            const uint32_t least = min(min(min(c0.x, c0.y), min(c0.z, c0.w)),
                                       min(min(c1.x, c1.y), min(c1.z, c1.w)));
            if (__any_sync(kFull, least < o.w)) {
                const uint4 wv = make_uint4(o.w, o.w, o.w, o.w);
                uint32_t m = ic_live(c0, wv, g, o.eb, o.ee), e0 = g << 2;
                uint32_t m1 = ic_live(c1, wv, g + 32u, o.eb, o.ee);
#pragma unroll 1
                for (int u = 0; u < 2; ++u) {
                    if (__any_sync(kFull, m)) visit(m, e0);
                    m = m1;
                    e0 += 128u;
                }
            }
        }
    }
    if (t0 >= n) return;
    uint4 wv = make_uint4(o.w, o.w, o.w, o.w);
    const uint4 *wp = reinterpret_cast<const uint4 *>(wgt) + g0 + lane;
    if (!o.equal && t0 + lane < n) wv = __ldg(wp + t0);
#pragma unroll 1
    for (; t0 < n; t0 += 32u) {
        const uint32_t g = g0 + t0 + lane;
        uint4 wn = wv;
        if (!o.equal && t0 + 32u + lane < n) wn = __ldg(wp + t0 + 32u);
        const uint4 c = cs(rk, g);
        uint32_t m = 0;
        if (t0 + lane < n) m = ic_live(c, wv, g, o.eb, o.ee);
        if (__any_sync(kFull, m)) visit(m, g << 2);
        wv = wn;
    }
}

// The same for the lists of a warp's lanes (ng groups in this lane's): those of
// at least kICWide groups one after another on all lanes, the others packed.
template <typename CS, typename F>
__device__ __forceinline__ void ic_expand(const CS &cs, const uint32_t *rk,
                                          const uint32_t *wgt, const ICItem &it, uint32_t ng,
                                          int lane, F &&visit) {
    unsigned wide = __ballot_sync(kFull, ng >= (uint32_t)kICWide);
    while (wide) {
        const int l = __ffs(wide) - 1;
        wide &= wide - 1u;
        const ICItem o{__shfl_sync(kFull, it.eb, l), __shfl_sync(kFull, it.ee, l),
                       __shfl_sync(kFull, it.w, l), __shfl_sync(kFull, it.equal, l)};
        ic_expand_wide(cs, rk, wgt, o, 0u, __shfl_sync(kFull, ng, l), lane, visit);
    }
    const uint32_t ns = ng >= (uint32_t)kICWide ? 0u : ng;
    const uint32_t incl = warp_incl_scan<uint32_t>(ns, lane);
    const uint32_t total = __shfl_sync(kFull, incl, 31);
#pragma unroll 1
    for (uint32_t t0 = 0; t0 < total; t0 += 32) {
        const uint32_t t = t0 + lane;
        int owner = 0;                       // first lane whose inclusive count exceeds t
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
            if (__shfl_sync(kFull, incl, owner + step - 1) <= t) owner += step;
        const uint32_t before = __shfl_sync(kFull, incl - ns, owner);
        const uint32_t eb = __shfl_sync(kFull, it.eb, owner);
        const uint32_t ee = __shfl_sync(kFull, it.ee, owner);
        const uint32_t w = __shfl_sync(kFull, it.w, owner);
        const bool equal = __shfl_sync(kFull, it.equal, owner) != 0u;
        const uint32_t g = (eb >> 2) + (t - before);
        uint4 wv = make_uint4(w, w, w, w);
        if (!equal && t < total) wv = __ldg(reinterpret_cast<const uint4 *>(wgt) + g);
        const uint4 c = cs(rk, g);
        uint32_t m = 0;
        if (t < total) m = ic_live(c, wv, g, eb, ee);
        if (__any_sync(kFull, m)) visit(m, g << 2);
    }
}

__device__ __forceinline__ uint32_t ic_hash(uint32_t u) {
    return (u * 0x9E3779B1u) >> (32 - 10);
}
static_assert(kICHash == 1 << 10, "ic_hash gives a slot of kICHash");

// One warp per sample.  BITS: the visited set is an n-bit bitmap in shared
// memory (n <= kSmemVisBits).  Otherwise it is a hash set of kICHash slots in
// shared memory -- an RRR set of a large graph is mostly a few dozen members,
// and a bitmap of its own in global memory would cost a DRAM access per probe
// -- which moves to the warp's bitmap in global memory (cleared by the warp on
// its first use, and kept clear) when the set passes kICHashMax members.
// Shared memory of a warp: visited words, kICQueueSmem queue entries (later
// entries in global memory), kCandCap listed edges.  Three blocks an SM, 80
// registers: four blocks at 64 measured 4 % slower, and without KEYS the round
// keys fit as well (held; deriving them in the loop: batched mix 66.9 against
// 62.5 ms).
template <bool BITS, bool KEYS>
__global__ void __launch_bounds__(kSampleThreads, 3) k_sample_ic(const __grid_constant__ SampleArgs a) {
    extern __shared__ uint32_t ic_smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t gw = (int64_t)blockIdx.x * kWarps + wib;
    const int svis = BITS ? (int)((a.vis_words + 3) & ~(int64_t)3) : kICHash;
    uint32_t *vis = ic_smem + (size_t)wib * (svis + kICQueueSmem + kCandCap);
    int32_t *sq = reinterpret_cast<int32_t *>(vis + svis);
    uint32_t *cand = reinterpret_cast<uint32_t *>(sq + kICQueueSmem);
    uint32_t *gvis = BITS ? nullptr : a.gvis + (size_t)gw * (size_t)a.vis_words;
    int32_t *q = a.queues + (size_t)gw * (size_t)a.qcap;
    constexpr uint32_t kClear = BITS ? 0u : 0xffffffffu;
    for (int i = lane; i < svis; i += 32) vis[i] = kClear;
    __syncwarp();
    bool gclear = false;                     // the global bitmap has been cleared
    unsigned long long exam = 0, abytes = 0;
    // the next sample index is taken while this one's set is built
    unsigned long long jn = 0;
    if (lane == 0) jn = atomicAdd(a.work, 1ull);
    for (;;) {
        const unsigned long long jw = __shfl_sync(kFull, jn, 0);
        if (jw >= (unsigned long long)a.count) break;
        if (lane == 0) jn = atomicAdd(a.work, 1ull);
        const int64_t j = a.list ? a.list[jw] : (int64_t)jw;
        const int qi = a.nq == 1 ? 0 : find_query(a, j);
        const QueryView &V = a.qv[qi];
        const uint4 *rec = V.ic_rec;
        const int32_t *in_src = V.in_src;
        const uint32_t *wgt = V.w;
        const uint64_t seed = V.seed;
        const uint32_t s = V.first + (uint32_t)(j - __ldg(a.qstart + qi));
        const uint32_t root = rrr_root(seed, s, V.n);
        CoinStream<KEYS, !KEYS> cs;
        cs.begin(a.rk, s, seed_lo(seed), seed_hi(seed));
        int32_t head = 0, tail = 1;
        int ncand = 0;
        bool spilled = false, lost = false;
        uint32_t work = 0;                   // in-edges of the expanded members (saturating)
        unsigned long long sexam = 0;
        if (lane == 0) {
            if (BITS) vis[root >> 5] |= 1u << (root & 31);
            else vis[ic_hash(root)] = root;
            sq[0] = (int32_t)root;
        }
        __syncwarp();
        // the last min(32, ncand) listed edges: source, visited test, append
        auto flush = [&]() {
            const int take = ncand < 32 ? ncand : 32;
            ncand -= take;
            __syncwarp();
            uint32_t u = 0;
            bool fresh = false;
            if (lane < take) u = (uint32_t)__ldg(in_src + cand[ncand + lane]);
            if (!BITS && !spilled && tail + 32 > kICHashMax) {
                // the hash set moves to the warp's bitmap in global memory
                if (!gclear) {
                    for (int64_t i = lane; i < a.vis_words; i += 32) gvis[i] = 0u;
                    gclear = true;
                    __syncwarp();
                }
                for (int32_t i = lane; i < tail; i += 32) {
                    const uint32_t x = (uint32_t)sq[i];
                    atomicOr(&gvis[x >> 5], 1u << (x & 31));
                }
                spilled = true;
                __syncwarp();
            }
            if (lane < take) {
                const uint32_t bit = 1u << (u & 31);
                if (BITS) {
                    fresh = !(atomicOr(&vis[u >> 5], bit) & bit);
                } else if (spilled) {
                    fresh = !(atomicOr(&gvis[u >> 5], bit) & bit);
                } else {
                    uint32_t h = ic_hash(u);
                    for (;;) {           // at most kICHashMax of kICHash slots are taken
                        const uint32_t old = atomicCAS(&vis[h], 0xffffffffu, u);
                        if (old == 0xffffffffu) fresh = true;
                        if (old == 0xffffffffu || old == u) break;
                        h = (h + 1) & (kICHash - 1);
                    }
                }
            }
            const unsigned fm = __ballot_sync(kFull, fresh);
            const int nf = __popc(fm);
            if ((int64_t)tail + nf > a.qcap) {
                // a queue overflow: the sample starts again in the second pass;
                // un-mark what was just marked (bitmaps only: the hash set
                // holds at most kICHashMax <= qcap)
                if (fresh) atomicAnd(BITS ? &vis[u >> 5] : &gvis[u >> 5], ~(1u << (u & 31)));
                lost = true;
                ncand = 0;
                __syncwarp();
                return;
            }
            if (fresh) {
                const int32_t at = tail + __popc(fm & lt);
                if (at < kICQueueSmem) sq[at] = (int32_t)u;
                else q[at] = (int32_t)u;
            }
            tail += nf;
            __syncwarp();
        };
        bool leave = false;
        while (!lost) {
            if (head == tail || leave) {
                if (ncand == 0) break;
                flush();
                continue;
            }
            // a set that percolates: its frontier feeds a whole block.  (A long
            // set with a narrow frontier -- weighted cascade grows them thin and
            // deep -- stays: the block's levels would leave most warps idle, 152
            // against 139 ms of IMM on the LiveJournal shape.)
            leave = work >= kICWideEdges && tail - head >= kICWarpFront;
            if (leave) continue;
            const int nb = tail - head < 32 ? tail - head : 32;
            ICItem it{0u, 0u, 0u, 1u};
            if (lane < nb) {
                const int32_t x = head + lane;
                it = ic_item(rec, (uint32_t)(x < kICQueueSmem ? sq[x] : q[x]));
            }
            const uint32_t deg = it.ee - it.eb;
            work = min(work + __reduce_add_sync(kFull, deg < (1u << 25) ? deg : 1u << 25),
                       kICWideEdges);
            sexam += (unsigned long long)deg;
            head += nb;
            ic_expand(cs, a.rk, wgt, it, ic_groups(it), lane, [&](uint32_t m, uint32_t e0) {
                if (lost) return;
                ic_list(m, e0, cand, ncand, lane);
                while (ncand >= 32) flush();
            });
        }
        const bool overflow = lost || head < tail;
        __syncwarp();
        if (overflow) {
            // second pass: the state goes along if there is room for it
            const unsigned long long ex = warp_sum<unsigned long long>(sexam);
            unsigned long long off = ~0ull;
            if (lane == 0 && !lost) {
                off = atomicAdd(a.hand_cursor, (unsigned long long)tail);
                if ((int64_t)off + tail > a.hand_cap) off = ~0ull;
            }
            off = __shfl_sync(kFull, off, 0);
            if (off != ~0ull)
                for (int32_t i = lane; i < tail; i += 32)
                    a.hand[off + i] = i < kICQueueSmem ? sq[i] : q[i];
            if (lane == 0) {
                a.sizes[j] = -1;
                a.stage_off[j] = 0;
                const unsigned long long at = atomicAdd(a.ovf_count, 1ull);
                if (off != ~0ull) {
                    const int64_t place = (int64_t)off / kICWarpFront;
                    a.handed[place] = Handed{(int64_t)off, ex, head, tail};
                    a.ovf_list[at] = j | (place + 1) << kHandedShift;
                } else {
                    a.ovf_list[at] = j;
                }
            }
        } else {
            unsigned long long pos = 0;
            if (lane == 0) pos = atomicAdd(a.stage_cursor, (unsigned long long)tail);
            pos = __shfl_sync(kFull, pos, 0);
            if ((int64_t)pos + tail > a.stage_cap) {
                if (lane == 0) {
                    raise_status(a.status, kDevStageOverflow);
                    a.sizes[j] = 0;
                    a.stage_off[j] = 0;
                }
            } else {
                for (int32_t i = lane; i < tail; i += 32)
                    a.stage[pos + i] = i < kICQueueSmem ? sq[i] : q[i];
                if (lane == 0) {
                    a.stage_off[j] = (int64_t)pos;
                    a.sizes[j] = tail;
                    if (tail > kWarpSortKeys) atomicAdd(a.nlong, 1ull);
                }
            }
            exam += sexam;
            // 16 B record + 4 B write per member, 8 B per examined edge, 8 B per set
            abytes += 8ull * sexam + (lane == 0 ? 20ull * (unsigned long long)tail + 8ull : 0ull);
        }
        // reset the visited set
        if (BITS && tail <= svis) {
            for (int32_t i = lane; i < tail; i += 32)
                vis[(uint32_t)(i < kICQueueSmem ? sq[i] : q[i]) >> 5] = 0u;
        } else {
            for (int i = lane; i < svis; i += 32) vis[i] = kClear;
        }
        if (spilled) {
            if (tail > a.vis_words) {
                for (int64_t i = lane; i < a.vis_words; i += 32) gvis[i] = 0u;
            } else {
                for (int32_t i = lane; i < tail; i += 32)
                    gvis[(uint32_t)(i < kICQueueSmem ? sq[i] : q[i]) >> 5] = 0u;
            }
        }
        __syncwarp();
    }
    exam = warp_sum<unsigned long long>(exam);
    abytes = warp_sum<unsigned long long>(abytes);
    if (lane == 0 && exam) atomicAdd(a.examined, exam);
    if (lane == 0 && abytes) atomicAdd(a.alg_bytes, abytes);
}

// IC, one block per sample: the second pass for the sets longer than a warp's
// queue.  The giant sets of hub-heavy graphs (hundreds of thousands of
// members, tens of millions of examined in-edges) are a level-synchronous
// BFS: the 32 warps take 32 queued vertices of the level at a time and expand
// them as k_sample_ic does; in-lists of at least kICHubGroups groups are put
// aside and shared out over the whole block at the end of the level, so that
// no warp is left alone with a hub.  The queue and visited bitmap (n entries /
// n bits per block) live in global memory; a warp appends what 32 listed live
// edges reach with one block-level atomic.  The set is copied to the stage by
// the block.
constexpr int kICBigThreads = 1024;
constexpr uint32_t kICHubGroups = 512;       // edge groups from which a list is shared by the block
constexpr int kICHubCap = 256;               // shared lists a level holds (others stay with their warp)

template <bool KEYS>
__global__ void __launch_bounds__(kICBigThreads) k_sample_ic_big(const __grid_constant__ SampleArgs a) {
    __shared__ unsigned long long s_item, s_pos;
    __shared__ unsigned int s_tail, s_cursor, s_nhub;
    __shared__ ICItem s_hub[kICHubCap];
    __shared__ uint32_t s_cand[kICBigThreads / 32][kCandCap];
    __shared__ unsigned long long s_red[kICBigThreads / 32];

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    int32_t *q = a.queues + (size_t)blockIdx.x * (size_t)a.qcap;
    uint32_t *vis = a.gvis + (size_t)blockIdx.x * (size_t)a.vis_words;
    uint32_t *cand = s_cand[warp];
    for (;;) {
        if (threadIdx.x == 0) {
            s_item = atomicAdd(a.work, 1ull);
            s_nhub = 0;
        }
        __syncthreads();
        const unsigned long long jw = s_item;
        if (jw >= (unsigned long long)a.count) break;
        const int64_t entry = a.list[jw];
        const int64_t j = entry & (((int64_t)1 << kHandedShift) - 1), place = (entry >> kHandedShift) - 1;
        const int qi = find_query(a, j);
        const QueryView &V = a.qv[qi];
        const uint4 *rec = V.ic_rec;
        const int32_t *in_src = V.in_src;
        const uint32_t *wgt = V.w;
        const uint32_t s = V.first + (uint32_t)(j - __ldg(a.qstart + qi));
        CoinStream<KEYS> cs;
        cs.begin(a.rk, s, seed_lo(V.seed), seed_hi(V.seed));
        unsigned long long sexam = 0;
        unsigned int head = 0;
        if (place >= 0) {                    // go on where the warp stopped
            const Handed hd = a.handed[place];
            for (int32_t x = threadIdx.x; x < hd.tail; x += kICBigThreads) {
                const int32_t u = a.hand[hd.off + x];
                q[x] = u;
                atomicOr(&vis[u >> 5], 1u << (u & 31));
            }
            head = (unsigned)hd.head;
            if (threadIdx.x == 0) {
                s_tail = (unsigned)hd.tail;
                sexam = hd.examined;
            }
        } else if (threadIdx.x == 0) {
            const uint32_t root = rrr_root(V.seed, s, V.n);
            atomicOr(&vis[root >> 5], 1u << (root & 31));
            q[0] = (int32_t)root;
            s_tail = 1;
        }
        __syncthreads();
        int ncand = 0;
        // the last min(32, ncand) listed edges: source, visited test, append
        // (the queue holds n entries, so it cannot overflow)
        auto flush = [&]() {
            const int take = ncand < 32 ? ncand : 32;
            ncand -= take;
            __syncwarp();
            uint32_t u = 0;
            bool fresh = false;
            if (lane < take) {
                u = (uint32_t)__ldg(in_src + cand[ncand + lane]);
                const uint32_t bit = 1u << (u & 31);
                // most live edges of a giant set reach a member: a load answers
                // those, an atomic the rest
                if (!(__ldcg(vis + (u >> 5)) & bit))
                    fresh = !(atomicOr(&vis[u >> 5], bit) & bit);
            }
            const unsigned fm = __ballot_sync(kFull, fresh);
            if (fm) {
                unsigned int at = 0;
                if (lane == 0) at = atomicAdd(&s_tail, (unsigned int)__popc(fm));
                at = __shfl_sync(kFull, at, 0);
                if (fresh) q[at + __popc(fm & lt)] = (int32_t)u;
            }
            __syncwarp();
        };
        auto visit = [&](uint32_t m, uint32_t e0) {
            ic_list(m, e0, cand, ncand, lane);
            while (ncand >= 32) flush();
        };
        for (;;) {
            const unsigned int lvl_end = s_tail;
            if (head >= lvl_end) break;
            __syncthreads();                 // everyone has read s_tail
            if (threadIdx.x == 0) s_cursor = head;
            __syncthreads();
            for (;;) {
                unsigned int base = 0;
                if (lane == 0) base = atomicAdd(&s_cursor, 32u);
                base = __shfl_sync(kFull, base, 0);
                if (base >= lvl_end) break;
                ICItem it{0u, 0u, 0u, 1u};
                if (base + lane < lvl_end) {
                    it = ic_item(rec, (uint32_t)q[base + lane]);
                    sexam += (unsigned long long)(it.ee - it.eb);
                }
                uint32_t ng = ic_groups(it);
                if (ng >= kICHubGroups) {    // shared by the block below
                    const unsigned int h = atomicAdd(&s_nhub, 1u);
                    if (h < (unsigned)kICHubCap) {
                        s_hub[h] = it;
                        ng = 0;
                    }
                }
                __syncwarp();
                ic_expand(cs, a.rk, wgt, it, ng, lane, visit);
            }
            __syncthreads();
            const int nhub = (int)(s_nhub < (unsigned)kICHubCap ? s_nhub : (unsigned)kICHubCap);
            for (int h = 0; h < nhub; ++h) {  // this warp's slice of every shared list
                const ICItem it = s_hub[h];
                const uint32_t n = ic_groups(it);
                const uint32_t per =
                    ((n + kICBigThreads / 32 - 1) / (kICBigThreads / 32) + 31u) & ~31u;
                const uint32_t t = min(n, warp * per);
                ic_expand_wide(cs, a.rk, wgt, it, t, min(n, t + per), lane, visit);
            }
            while (ncand > 0) flush();
            __syncthreads();
            if (threadIdx.x == 0) s_nhub = 0;
            head = lvl_end;
        }
        // emit: reserve the stage range, write the set, record size and offset.
        // A long set is read off its bitmap, in ascending order (so that it
        // needs no sorting: 0.9 ms a set when the sort marked and read a bitmap
        // of its own), which also clears it; a short one is copied from the
        // queue.
        const long long len = (long long)s_tail;
        const bool ascending = len > kBlockSortCap || (len > kWarpSortKeys && a.vis_words <= 64 * len);
        const unsigned long long ex = warp_sum<unsigned long long>(sexam);
        if (lane == 0) s_red[warp] = ex;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long tot = 0;
            for (int w2 = 0; w2 < kICBigThreads / 32; ++w2) tot += s_red[w2];
            s_pos = atomicAdd(a.stage_cursor, (unsigned long long)len);
            if ((long long)s_pos + len > a.stage_cap) {
                raise_status(a.status, kDevStageOverflow);
                a.sizes[j] = 0;
                a.stage_off[j] = 0;
                s_pos = ~0ull;
            } else {
                a.stage_off[j] = (int64_t)s_pos | (ascending ? kStageAscending : 0);
                a.sizes[j] = (int32_t)len;
                if (len > kWarpSortKeys) atomicAdd(a.nlong, 1ull);
                atomicAdd(a.examined, tot);
                // 16 B record + 4 B write per member, 8 B per examined edge, 8 B per set
                atomicAdd(a.alg_bytes, 8ull * tot + 20ull * (unsigned long long)len + 8ull);
            }
        }
        __syncthreads();
        if (ascending && s_pos != ~0ull) {
            // each warp a run of words: the members before it, then its own
            const int64_t run = ((a.vis_words + kICBigThreads - 1) / kICBigThreads) * 32;
            const int64_t w0 = min(a.vis_words, warp * run), w1 = min(a.vis_words, w0 + run);
            int cnt = 0;
#pragma unroll 4
            for (int64_t x = w0 + lane; x < w1; x += 32) cnt += __popc(__ldcg(vis + x));
            cnt = __reduce_add_sync(kFull, cnt);
            if (lane == 0) s_red[warp] = (unsigned long long)cnt;
            __syncthreads();
            const int incl = warp_incl_scan<int>((int)s_red[lane], lane);
            int64_t at = (int64_t)s_pos + (warp ? __shfl_sync(kFull, incl, warp - 1) : 0);
            uint32_t next = w0 + lane < w1 ? __ldcg(vis + w0 + lane) : 0u;
            for (int64_t x0 = w0; x0 < w1; x0 += 32) {
                const int64_t x = x0 + lane;
                uint32_t bitset = next;
                next = x + 32 < w1 ? __ldcg(vis + x + 32) : 0u;
                if (bitset) vis[x] = 0u;
                const int mine = __popc(bitset);
                const int upto = warp_incl_scan<int>(mine, lane);
                int64_t p = at + upto - mine;
                while (bitset) {
                    const int c = __ffs(bitset) - 1;
                    bitset &= bitset - 1u;
                    a.stage[p++] = (int32_t)(x * 32 + c);
                }
                at += __shfl_sync(kFull, upto, 31);
            }
        } else {
            if (s_pos != ~0ull)
                for (long long x = threadIdx.x; x < len; x += blockDim.x) a.stage[s_pos + x] = q[x];
            // clear this sample's visited bits
            if (len > a.vis_words) {
                for (int64_t x = threadIdx.x; x < a.vis_words; x += blockDim.x) vis[x] = 0u;
            } else {
                for (long long x = threadIdx.x; x < len; x += blockDim.x) vis[q[x] >> 5] = 0u;
            }
        }
        __syncthreads();
    }
}

// In-edge records of the IC kernels: {first in-edge, in-degree, common weight,
// 1 if all in-edges have it}.  A lane looks at up to kICRecLane in-edges of
// its own vertex -- with unequal weights that settles nearly every list -- and
// the warp scans the rest of the undecided lists together, until the first
// difference.
constexpr int kICRecLane = 4;

__global__ void __launch_bounds__(256) k_ic_records(const int64_t *in_off, const uint32_t *w,
                                                    int64_t n, uint4 *rec) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t v0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; v0 < n;
         v0 += warps * 32) {
        const int64_t v = v0 + lane;
        int64_t b = 0, e = 0;
        if (v < n) {
            b = in_off[v];
            e = in_off[v + 1];
        }
        const uint32_t w0 = e > b ? __ldg(w + b) : 0u;
        bool same = true;
#pragma unroll
        for (int i = 1; i < kICRecLane; ++i)
            if (b + i < e) same &= __ldg(w + b + i) == w0;
        unsigned open = __ballot_sync(kFull, same && e - b > kICRecLane);
        while (open) {
            const int l = __ffs(open) - 1;
            open &= open - 1u;
            const int64_t lb = __shfl_sync(kFull, b, l), le = __shfl_sync(kFull, e, l);
            const uint32_t lw = __shfl_sync(kFull, w0, l);
            bool ok = true;
            for (int64_t i0 = lb + kICRecLane; i0 < le && ok; i0 += 256) {
                bool mine = true;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int64_t i = i0 + u * 32 + lane;
                    if (i < le) mine &= __ldg(w + i) == lw;
                }
                ok = __all_sync(kFull, mine);
            }
            if (lane == l) same = ok;
        }
        if (v < n)
            rec[v] = make_uint4((uint32_t)b, (uint32_t)(e - b), w0, same ? 1u : 0u);
    }
}

// ---------------------------------------------------------------------------
// LT: backward walk of the LT live-edge world.  Vertex v picks the first
// in-edge whose running weight sum exceeds Philox(s, v, 0, pick tag).x; the
// walk stops when nothing is picked or the picked source is already on it.
//
// The pick is found in a fanout-32 search tree over v's running sums (built
// by k_lt_index): every level is read as one contiguous window of at most 32
// values, one per lane, and a ballot selects the child -- so a step costs
// ceil(log32 d) + 1 coalesced loads instead of scattered probes, and the leaf
// that matches also carries the source id.
// ---------------------------------------------------------------------------
// Group-wide helpers: a group is G consecutive lanes of a warp running one walk.
template <int G>
__device__ __forceinline__ unsigned group_mask(int lane) {
    return G == 32 ? kFull : (((1u << G) - 1u) << ((lane / G) * G));
}

// One walk per group of G lanes; a warp runs 32 / G walks in lockstep.  The
// loop is warp-uniform: every iteration each group advances its own walk by
// one step (groups without a walk idle through predication, so the warp never
// splits and the Philox draw, the search and the revisit test of all its
// walks share one instruction stream); a group whose walk ended emits it and
// takes the next sample at the top of the next iteration.  Every level of the
// search tree is a window of up to 32 values; lane l of a group holds values
// [l * 32/G, (l + 1) * 32/G) of it.
template <int G>
__global__ void __launch_bounds__(kSampleThreads, G == 32 ? 8 : 5) k_sample_lt(SampleArgs a) {
    constexpr int NG = 32 / G;                       // walks per warp
    constexpr int NV = 32 / G;                       // window values per lane
    constexpr int PS = G == 32 ? kPathSmem : kPathSmemGroup;
    constexpr unsigned GBITS = G == 32 ? kFull : ((1u << G) - 1u);
    __shared__ int32_t spath[kWarps * NG][PS];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int grp = lane / G, gl = lane % G, gbase = grp * G;
    const unsigned gmask = group_mask<G>(lane);
    const int64_t slot = ((int64_t)blockIdx.x * kWarps + wib) * NG + grp;
    int32_t *q = a.queues + (size_t)slot * (size_t)a.qcap;
    int32_t *sp = spath[wib * NG + grp];
    unsigned long long exam = 0, abytes = 0;
    bool active = false, exhausted = false;
    int64_t j = 0;
    uint32_t s = 0, cur = 0, k0 = 0, k1 = 0;
    const uint4 *vrec = nullptr;
    const unsigned long long *leaf_arr = nullptr, *tree = nullptr;
    const int32_t *srcs = nullptr;
    int32_t len = 0;
    unsigned long long sexam = 0;
    uint32_t sbytes = 0;   // flushed into abytes before it can wrap
    for (;;) {
        if (!active && !exhausted) {                 // group-uniform
            unsigned long long jw = 0;
            if (gl == 0) jw = atomicAdd(a.work, 1ull);
            jw = __shfl_sync(gmask, jw, 0, G);
            if (jw < (unsigned long long)a.count) {
                j = a.list ? a.list[jw] : (int64_t)jw;
                const int qi = find_query(a, j);
                const QueryView &V = a.qv[qi];
                vrec = V.lt_vrec;
                leaf_arr = V.lt_leaf;
                tree = V.lt_tree;
                srcs = V.in_src;
                k0 = seed_lo(V.seed);
                k1 = seed_hi(V.seed);
                s = V.first + (uint32_t)(j - __ldg(a.qstart + qi));
                cur = rrr_root(V.seed, s, V.n);
                if (gl == 0) {
                    q[0] = (int32_t)cur;
                    sp[0] = (int32_t)cur;
                }
                len = 1;
                sexam = 0;
                sbytes = 8;
                active = true;
            } else {
                exhausted = true;
            }
        }
        __syncwarp();
        if (!__any_sync(kFull, active)) break;

        // ---- one step of every active walk ----
        const uint32_t x = philox4x32_10(make_uint4(s, cur, 0u, kStreamPick), k0, k1).x;
        const unsigned long long xs = (unsigned long long)x;
        const uint4 vr = active ? __ldg(vrec + cur) : make_uint4(0u, 0u, 0u, 0u);
        const int32_t d = (int32_t)vr.y;
        // in-edges of equal weight u: the pick is edge floor(x / u), no search
        // (the running sums and tree exist only when some vertex needs them)
        const bool eqw = vr.w != 0u;
        bool live = active && d > 0 && !eqw;         // group-uniform
        const uint32_t nlev = vr.z >> 28;
        const int lmax = (int)__reduce_max_sync(kFull, live ? nlev : 0u);
        const unsigned long long *lvl = tree + (vr.z & 0x0fffffffu);   // levels stored top-down
        int32_t blk = 0;
        for (int l = lmax; l >= 1; --l) {
            const bool here = live && l <= (int)nlev;
            const int32_t sz = here ? (int32_t)(((int64_t)d + (1ll << (5 * l)) - 1) >> (5 * l)) : 0;
            int lf = NV;
#pragma unroll
            for (int v = NV - 1; v >= 0; --v) {
                const int32_t idx = blk * 32 + gl * NV + v;
                if (idx < sz && xs < __ldg(lvl + idx)) lf = v;
            }
            const unsigned bal = (__ballot_sync(kFull, lf < NV) >> gbase) & GBITS;
            const int f = bal ? __ffs(bal) - 1 : 0;
            const int lfv = __shfl_sync(kFull, lf, gbase + f);
            if (here) {
                if (!bal) live = false;
                else {
                    blk = blk * 32 + f * NV + lfv;
                    lvl += sz;
                }
            }
        }
        int32_t pick = -1;
        unsigned long long leaf = 0;
        {
            int lf = NV;
            unsigned long long hit = 0;
#pragma unroll
            for (int v = NV - 1; v >= 0; --v) {
                const int32_t idx = blk * 32 + gl * NV + v;
                if (live && idx < d) {
                    const unsigned long long r = __ldg(leaf_arr + vr.x + idx);
                    if (xs < (r >> 31)) {
                        lf = v;
                        hit = r;
                    }
                }
            }
            const unsigned bal = (__ballot_sync(kFull, lf < NV) >> gbase) & GBITS;
            const int f = bal ? __ffs(bal) - 1 : 0;
            const int lfv = __shfl_sync(kFull, lf, gbase + f);
            const unsigned long long hv = __shfl_sync(kFull, hit, gbase + f);
            if (live && bal) {
                pick = blk * 32 + f * NV + lfv;
                leaf = hv;
            }
        }
        if (active && eqw) {
            const uint32_t ei = x / vr.w;
            if (ei < (uint32_t)d) {
                pick = (int32_t)ei;
                leaf = (unsigned long long)(uint32_t)__ldg(srcs + vr.x + ei);   // its source
            }
        }
        if (active && gl == 0) {
            sexam += (unsigned long long)(pick >= 0 ? pick + 1 : d);
            // vertex record, binary search of d cumulative weights (none for equal
            // weights), source, member write
            sbytes += 16u + (d > 0 && !eqw ? 8u * (uint32_t)(32 - __clz((uint32_t)d)) : 0u) +
                      (pick >= 0 ? 4u : 0u) + 4u;
            if (sbytes > (1u << 30)) {   // only long walks of the second pass get here
                abytes += sbytes;
                sbytes = 0;
            }
        }
        // revisit test of the picked source against the walk so far
        const bool picked = active && pick >= 0;
        const int32_t u = (int32_t)(leaf & 0x7fffffffull);
        const int lenmax = (int)__reduce_max_sync(kFull, picked ? (unsigned)len : 0u);
        bool seen = false;
        for (int32_t i = gl; i < lenmax; i += G)
            if (picked && i < len) seen |= (i < PS ? sp[i] : q[i]) == u;
        const bool seen_g = ((__ballot_sync(kFull, seen) >> gbase) & GBITS) != 0;
        const bool grow = picked && !seen_g && len < a.qcap;
        const bool ovf = picked && !seen_g && len >= a.qcap;
        if (grow) {
            if (gl == 0) {
                q[len] = u;
                if (len < PS) sp[len] = u;
            }
            ++len;
            cur = (uint32_t)u;
        }
        __syncwarp();
        if (active && !grow) {                       // the walk ended: emit it
            if (ovf) {
                if (gl == 0) {
                    a.sizes[j] = -1;
                    a.stage_off[j] = 0;
                    a.ovf_list[atomicAdd(a.ovf_count, 1ull)] = j;
                }
            } else {
                unsigned long long pos = 0;
                if (gl == 0) pos = atomicAdd(a.stage_cursor, (unsigned long long)len);
                pos = __shfl_sync(gmask, pos, 0, G);
                if ((int64_t)pos + len > a.stage_cap) {
                    if (gl == 0) {
                        raise_status(a.status, kDevStageOverflow);
                        a.sizes[j] = 0;
                        a.stage_off[j] = 0;
                    }
                } else {
                    for (int32_t i = gl; i < len; i += G) a.stage[pos + i] = i < PS ? sp[i] : q[i];
                    if (gl == 0) {
                        a.stage_off[j] = (int64_t)pos;
                        a.sizes[j] = len;
                        if (len > kWarpSortKeys)
                            atomicAdd(a.nlong, 1ull + (len > kBlockSortCap ? 1ull << 32 : 0ull));
                    }
                }
                exam += sexam;
                if (gl == 0) abytes += sbytes;
            }
            active = false;
        }
        __syncwarp();
    }
    exam = warp_sum<unsigned long long>(exam);
    abytes = warp_sum<unsigned long long>(abytes);
    if (lane == 0 && exam) atomicAdd(a.examined, exam);
    if (lane == 0 && abytes) atomicAdd(a.alg_bytes, abytes);
}

// LT, one walk per thread.  A step is one Philox draw, the vertex record and
// one dependent load: the source of in-edge floor(x / u) when all in-edges of
// the vertex weigh u (1/in-degree weights, for one), else one guide entry (see
// k_lt_guide), with a binary search over the running sums only when the draw
// lies past the guide's edge.
//
// The two dependent loads are what a step cannot do without; a warp hides them
// behind the other 31 of its SM.  Everything else a walk needs -- its start, the
// check for a revisit, its way to the stage -- happens once in tens of steps of
// a lane, but with 32 lanes nearly every iteration has some lane at one of them,
// and each costs a warp a round trip to L2.  So each is put off until it serves
// many lanes or many walks:
//   - A warp takes sample indices kLT1Chunk at a time; its lanes draw the roots
//     and look at their records together, write the sets of roots without
//     in-edges (half of an R-MAT graph) at once, and keep the others in a ring in
//     shared memory.  Lanes without a walk wait until kLT1Refill of them do.
//   - A revisit is noticed by a 1024-bit Bloom filter of the walk in shared
//     memory (two hashes).  The walk goes on: after a true revisit it repeats
//     its cycle (a vertex's pick is the same in the whole sample), so the next
//     source is in the filter too, and a source that is not proves the hit before
//     it false.  Only after two hits in a row is the first one checked, exactly,
//     by the whole warp over the walk's path, two walks at a time.
//   - Finished walks stay in the lane's buffer, one behind the other, and are
//     moved to the stage when some lane has kLT1Flush members of them: one
//     reservation and one coalesced copy of all the lanes' finished walks.
// Waiting changes no draw: a walk's steps are the same whenever they run.
//
// Measured at 4,194,304 sets on R-MAT scale 20 with 1/in-degree weights (1.7 x
// 10^8 steps): 4.14 + 0.98 -> 3.7 ms, the 0.98 a second pass for walks longer
// than the 512 entries a lane had; U[0, 0.1] weights (1.6 x 10^7 members) 1.51 ->
// 0.80 ms.  What is left is the two random reads: ncu shows 12.8 instructions a
// step (19.2), issue 41 % busy, half of the reads missing L2, and 24 warps an SM
// only 4 % slower than 32.  Not kept: 16-byte in-edge records (source and its
// vertex record) for one read a step: 4.76 ms, every one of them from DRAM (268
// MB against 84 MB of records and sources); five blocks an SM (spills) 5.4 ms;
// streaming stores to the stage, kLT1Flush 64 to 384, kLT1Refill 2 to 5,
// kLT1Check 1 to 3: within 2 %.
constexpr int kLT1Threads = 256;
constexpr int kLT1Warps = kLT1Threads / 32;
constexpr int kBloomWords = 32;              // 1024 bits per walk
constexpr int64_t kQueueCapLT1 = 1024;       // entries of a lane's buffer at most
constexpr unsigned kLT1Chunk = 32;           // sample indices a warp takes at once (one per lane)
constexpr int kLT1Refill = 3;                // lanes without a walk that start new ones
constexpr int kLT1Check = 2;                 // walks waiting for an exact check that start it
constexpr int kLT1Group = 2;                 // paths scanned together
constexpr int kLT1Flush = 192;               // finished members of a lane that start a flush
constexpr int kLT1Recs = 32;                 // finished walks a lane keeps at most
constexpr int kLT1Blocks = 4;                // blocks an SM
// The work items of one launch stay below this count, so that the warp's chunk
// bounds fit 32 bits (a larger job takes the grouped kernel).
constexpr int64_t kLT1MaxCount = (1ll << 32) - (1ll << 28);

__device__ __forceinline__ uint32_t bloom_h1(uint32_t u) { return (u * 0x9E3779B1u) >> 22; }
__device__ __forceinline__ uint32_t bloom_h2(uint32_t u) {
    return ((u ^ (u >> 16)) * 0x85EBCA6Bu) >> 22;
}

// bl points at this thread's column: word w of its filter is bl[w * kLT1Threads]
// (a warp touching any words hits 32 distinct banks)
__device__ __forceinline__ void bloom_add(uint32_t *bl, uint32_t u) {
    const uint32_t h1 = bloom_h1(u), h2 = bloom_h2(u);
    bl[(h1 >> 5) * kLT1Threads] |= 1u << (h1 & 31);
    bl[(h2 >> 5) * kLT1Threads] |= 1u << (h2 & 31);
}

__device__ __forceinline__ bool bloom_has(const uint32_t *bl, uint32_t u) {
    const uint32_t h1 = bloom_h1(u), h2 = bloom_h2(u);
    return ((bl[(h1 >> 5) * kLT1Threads] >> (h1 & 31)) & (bl[(h2 >> 5) * kLT1Threads] >> (h2 & 31)) &
            1u) != 0;
}

// 16-byte read-only load with an L2 eviction-priority policy (createpolicy).
__device__ __forceinline__ uint4 ldg_policy(const uint4 *p, uint64_t pol) {
    uint4 r;
    asm("ld.global.nc.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
        : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
        : "l"(p), "l"(pol));
    return r;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// CP (IM_TUNE_LT_CACHE): 0 plain loads; 1 the vertex records (n x 16 B, read
// at every step) are kept in L2 ahead of other lines (evict_last); 2 as 1, and
// the cut points (m x 16 B, mostly single-use) leave L2 first (evict_first).
// KEYS: the launch has one query, whose round keys are in the arguments.
// Launched with a.count <= kLT1MaxCount.
// A lane's buffer (a.qcap entries): finished walks in [fb, wb), the current one
// in [wb, wb + len); its finished walks' {sample, first entry} in a.recs.
template <int CP, bool KEYS>
__global__ void __launch_bounds__(kLT1Threads, kLT1Blocks) k_sample_lt1(const __grid_constant__ SampleArgs a) {
    extern __shared__ uint32_t bloom[];          // [kBloomWords][kLT1Threads]
    // drawn roots with in-edges, their sample ids, indices and queries
    constexpr uint32_t kRing = 2 * kLT1Chunk;
    __shared__ uint32_t ring_root[kLT1Warps][kRing], ring_s[kLT1Warps][kRing], ring_j[kLT1Warps][kRing];
    __shared__ int32_t ring_q[kLT1Warps][kRing];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t *bl = bloom + threadIdx.x;
    const int32_t cap = (int32_t)a.qcap;
    const int64_t warp_id = (int64_t)blockIdx.x * kLT1Warps + wib;
    int32_t *q = a.queues + (warp_id * 32 + lane) * a.qcap;
    uint2 *recs = a.recs + warp_id * 32 * kLT1Recs + lane;
    const uint4 *vrec = a.qv[0].lt_vrec;
    const int32_t *srcs = a.qv[0].in_src;
    PickStream<KEYS> ps;
    bool active = false, pend = false, exhausted = false;
    uint32_t j = 0, cur = 0;
    int32_t qi = 0, len = 0, fb = 0, wb = 0, nrec = 0;
    // hits: filter hits in a row at the end of the path (0 to 2); the first of
    // them is path entry `hit`.  What the steps from there on examined and moved
    // counts only once the hit is known to be false (pexam, pbytes).
    int32_t hits = 0, hit = 0;
    unsigned long long sexam = 0, pexam = 0, tot_exam = 0, tot_bytes = 0;
    uint32_t sbytes = 0, pbytes = 0;
    uint32_t rhead = 0, rcnt = 0;                // the ring (warp-uniform)
    for (;;) {
        // ---- lanes without a walk take the next drawn roots
        const unsigned idle = __ballot_sync(kFull, !active);
        if (idle == kFull && exhausted && rcnt == 0) break;
        if ((__popc(idle) >= kLT1Refill || idle == kFull) && (rcnt > 0 || !exhausted)) {
            if (rcnt < (uint32_t)__popc(idle) && !exhausted) {
                unsigned long long nb = 0;
                if (lane == 0) nb = atomicAdd(a.work, (unsigned long long)kLT1Chunk);
                nb = __shfl_sync(kFull, nb, 0);
                if (nb >= (unsigned long long)a.count) {
                    exhausted = true;
                } else {
                    const int64_t jc = (int64_t)nb + lane;
                    const bool have = jc < a.count;
                    uint32_t root = 0, sc = 0, d = 0;
                    int qc = 0;
                    if (have) {
                        qc = KEYS ? 0 : find_query(a, jc);
                        const QueryView &V = a.qv[qc];
                        sc = V.first + (uint32_t)(jc - __ldg(a.qstart + qc));
                        root = rrr_root(V.seed, sc, V.n);
                        d = __ldg(reinterpret_cast<const uint32_t *>(V.lt_vrec + root) + 1);
                    }
                    // roots without in-edges are sets of their own
                    const unsigned sm = __ballot_sync(kFull, have && d == 0u);
                    if (sm) {
                        unsigned long long pos = 0;
                        if (lane == 0) pos = atomicAdd(a.stage_cursor, (unsigned long long)__popc(sm));
                        pos = __shfl_sync(kFull, pos, 0);
                        if (have && d == 0u) {
                            const int64_t at = (int64_t)pos + __popc(sm & lt);
                            if (at < a.stage_cap) {
                                a.stage[at] = (int32_t)root;
                                a.stage_off[jc] = at;
                                a.sizes[jc] = 1;
                                tot_bytes += 8u + 4u + 16u;   // set offset, root write, record
                            } else {
                                raise_status(a.status, kDevStageOverflow);
                            }
                        }
                    }
                    const unsigned wm = __ballot_sync(kFull, have && d != 0u);
                    if (have && d != 0u) {
                        const uint32_t e = (rhead + rcnt + (uint32_t)__popc(wm & lt)) & (kRing - 1);
                        ring_root[wib][e] = root;
                        ring_s[wib][e] = sc;
                        ring_j[wib][e] = (uint32_t)jc;
                        if (!KEYS) ring_q[wib][e] = qc;
                    }
                    rcnt += (uint32_t)__popc(wm);
                    __syncwarp();
                }
            }
            const uint32_t rank = (uint32_t)__popc(idle & lt);
            if (!active && rank < rcnt) {
                const uint32_t e = (rhead + rank) & (kRing - 1);
                cur = ring_root[wib][e];
                j = ring_j[wib][e];
                if (KEYS) {
                    ps.begin(a.rk, ring_s[wib][e], 0u, 0u);
                } else {
                    qi = ring_q[wib][e];
                    const QueryView &V = a.qv[qi];
                    vrec = V.lt_vrec;
                    srcs = V.in_src;
                    ps.begin(a.rk, ring_s[wib][e], seed_lo(V.seed), seed_hi(V.seed));
                }
                if (fb == wb) fb = wb = 0;           // nothing finished is left in the buffer
                q[wb] = (int32_t)cur;
#pragma unroll
                for (int w = 0; w < kBloomWords; ++w) bl[w * kLT1Threads] = 0u;
                bloom_add(bl, cur);
                len = 1;
                hits = 0;
                sexam = pexam = 0;
                pbytes = 0;
                sbytes = 8u + 4u;                    // set offset, root write
                active = true;
            }
            const uint32_t took = min(rcnt, (uint32_t)__popc(idle));
            rhead += took;
            rcnt -= took;
            __syncwarp();
        }

        // ---- one step of every walk that is not waiting for its exact check
        bool ending = false;
        if (active && !pend) {
            const uint32_t x = ps(a.rk, cur).x;
            uint32_t u = 0, e = 0xffffffffu;         // the pick: source and index
            uint32_t stepb = 16u;                    // vertex record
            // (the L2 policies are made where they are used: one instruction,
            // and no registers held across the loop)
            const uint4 vr =
                CP >= 1 ? ldg_policy(vrec + cur, l2_policy_evict_last()) : __ldg(vrec + cur);
            const uint32_t d = vr.y;
            if (vr.w != 0u) {
                // equal in-weights: edge floor(x / weight), from the reciprocal in
                // the record, at most 2 too small
                uint32_t ei = __umulhi(x, vr.z), rem = x - ei * vr.w;
                if (rem >= vr.w) { ++ei; rem -= vr.w; }
                if (rem >= vr.w) ++ei;
                if (ei < d) {
                    e = ei;
                    u = (uint32_t)__ldg(srcs + vr.x + ei);
                    stepb += 4u;                     // source of the pick
                }
            } else if (d > 0) {
                const QueryView &V = a.qv[qi];
                const uint4 *gp = V.lt_guide + vr.x + __umulhi(x, d);
                const uint4 gv = CP >= 2 ? ldg_policy(gp, l2_policy_evict_first()) : __ldg(gp);
                const unsigned long long cum = ((unsigned long long)gv.y << 32) | gv.x;
                stepb += 16u;                        // cut point
                if ((unsigned long long)x < cum) {
                    e = gv.w;
                    u = gv.z;
                } else {
                    // the first edge past the guide's with x < sum: with unequal
                    // weights that is about every second draw, and mostly the next
                    // edge, so the search doubles its stride from there (halving
                    // all that is left of the list read log2 d scattered sums)
                    const unsigned long long *leaf = V.lt_leaf + vr.x;
                    uint32_t lo = gv.w + 1, hi = d, stride = 1;
                    unsigned long long at = 0;       // the sum and source of edge hi < d
                    while (lo < hi) {
                        const uint32_t p = hi < d ? (lo + hi) >> 1 : min(lo + stride - 1u, d - 1u);
                        const unsigned long long r = __ldg(leaf + p);
                        stepb += 8u;                 // search probe
                        if ((unsigned long long)x < (r >> 31)) {
                            hi = p;
                            at = r;
                        } else {
                            lo = p + 1;
                        }
                        stride <<= 1;
                    }
                    if (hi < d) {
                        e = hi;
                        u = (uint32_t)(at & 0x7fffffffull);
                        stepb += 8u;                 // picked leaf
                    }
                }
            }
            if (e == 0xffffffffu) {                  // no in-edge picked: the walk stops, and
                sexam += pexam + d;                  // hits before this were false
                sbytes += pbytes + stepb;
                ending = true;
            } else {
                const unsigned long long stepx = (unsigned long long)e + 1ull;
                if (!bloom_has(bl, u)) {             // a new vertex, so earlier hits were false
                    sexam += pexam + stepx;
                    sbytes += pbytes + stepb + 4u;   // ... and a member write
                    pexam = 0;
                    pbytes = 0;
                    hits = 0;
                    bloom_add(bl, u);
                } else if (hits == 0) {              // maybe a revisit, which this step found
                    sexam += stepx;
                    sbytes += stepb;
                    pbytes = 4u;
                    hits = 1;
                    hit = len;
                } else {                             // again: check the first
                    pexam = stepx;
                    pbytes += stepb + 4u;
                    pend = true;
                }
                q[wb + len] = (int32_t)u;            // (room: see the end of the loop)
                ++len;
                cur = u;
            }
        }
        // ---- exact checks of the walks that wait for one, once kLT1Check do (or
        // every active walk does): is path entry `hit` among those before it?
        const unsigned pm = __ballot_sync(kFull, pend);
        if (pm && (__popc(pm) >= kLT1Check || pm == __ballot_sync(kFull, active && !ending))) {
            __syncwarp();                            // the paths are read across lanes
            bool seen = false;
            unsigned rest = pm;
            do {
                int l[kLT1Group];
#pragma unroll
                for (int g = 0; g < kLT1Group; ++g) {   // lanes of the group; repeats when fewer
                    l[g] = rest ? __ffs(rest) - 1 : l[0];
                    rest &= rest - 1u;
                }
                int32_t lg[kLT1Group], at[kLT1Group], ug[kLT1Group];
                int32_t lmax = 0;
#pragma unroll
                for (int g = 0; g < kLT1Group; ++g) {
                    lg[g] = __shfl_sync(kFull, hit, l[g]);
                    at[g] = __shfl_sync(kFull, wb, l[g]);
                    ug[g] = __ldcg(q + (int64_t)(l[g] - lane) * a.qcap + at[g] + lg[g]);
                    lmax = max(lmax, lg[g]);
                }
                bool f[kLT1Group];
#pragma unroll
                for (int g = 0; g < kLT1Group; ++g) f[g] = false;
                for (int32_t i = lane; i < lmax; i += 32) {
                    int32_t v[kLT1Group];
#pragma unroll
                    for (int g = 0; g < kLT1Group; ++g)      // lane l[g]'s path entry i
                        v[g] = i < lg[g] ? __ldcg(q + (int64_t)(l[g] - lane) * a.qcap + at[g] + i) : -1;
#pragma unroll
                    for (int g = 0; g < kLT1Group; ++g) f[g] |= v[g] == ug[g];
                }
#pragma unroll
                for (int g = 0; g < kLT1Group; ++g) {
                    const bool any = __any_sync(kFull, f[g]);
                    if (lane == l[g]) seen = any;
                }
            } while (rest);
            if (pend) {
                pend = false;
                if (seen) {                          // a revisit: the walk stopped before it
                    len = hit;
                    ending = true;
                } else {                             // a new vertex; the hit after it is now the first
                    sexam += pexam;
                    sbytes += pbytes - 4u;
                    pexam = 0;
                    pbytes = 4u;
                    ++hit;
                }
            }
        }
        if (ending) {                                // stays in the buffer
            a.sizes[j] = len;
            recs[nrec * 32] = make_uint2(j, (uint32_t)wb);
            ++nrec;
            wb += len;
            tot_exam += sexam;
            tot_bytes += sbytes;
            active = false;
            len = 0;
        }
        // ---- the finished walks of all lanes go to the stage when one lane has many
        // of them, or has no room for its next member (without a walk: for a root
        // and the member after it)
        const bool tight = wb + len + (active ? 0 : 1) >= cap;
        if (__any_sync(kFull, wb - fb >= kLT1Flush || nrec == kLT1Recs || tight)) {
            __syncwarp();                            // the buffers are read across lanes
            const int32_t mine = wb - fb;
            const int32_t upto = warp_incl_scan<int32_t>(mine, lane), excl = upto - mine;
            const int32_t tot = __shfl_sync(kFull, upto, 31);
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(a.stage_cursor, (unsigned long long)tot);
            base = __shfl_sync(kFull, base, 0);
            if ((int64_t)base + tot <= a.stage_cap) {
                const int32_t most = __reduce_max_sync(kFull, nrec);
#pragma unroll 4
                for (int32_t k = 0; k < most; ++k)
                    if (k < nrec) {
                        const uint2 r = __ldcg(recs + k * 32);
                        a.stage_off[r.x] = (int64_t)base + excl + ((int32_t)r.y - fb);
                    }
                const int64_t from = fb - excl;      // the lane's entry for position 0
                constexpr int U = 4;
                for (int32_t t0 = 0; t0 < tot; t0 += 32 * U) {
                    int32_t v[U];
#pragma unroll
                    for (int uu = 0; uu < U; ++uu) {
                        const int32_t t = t0 + uu * 32 + lane;
                        int owner = 0;               // first lane whose inclusive count exceeds t
#pragma unroll
                        for (int step = 16; step > 0; step >>= 1)
                            if (__shfl_sync(kFull, upto, owner + step - 1) <= t) owner += step;
                        const int64_t o_from = __shfl_sync(kFull, from, owner);
                        v[uu] = t < tot ? __ldcg(q + (int64_t)(owner - lane) * a.qcap + o_from + t) : 0;
                    }
#pragma unroll
                    for (int uu = 0; uu < U; ++uu) {
                        const int32_t t = t0 + uu * 32 + lane;
                        if (t < tot) a.stage[(int64_t)base + t] = v[uu];
                    }
                }
            } else if (lane == 0) {
                raise_status(a.status, kDevStageOverflow);
            }
            fb = wb;
            nrec = 0;
            // lanes without room: the current walk moves to the front of the
            // buffer, or is longer than it (second pass)
            unsigned full = __ballot_sync(kFull, tight && active);
            while (full) {
                const int l = __ffs(full) - 1;
                full &= full - 1u;
                const int32_t lw = __shfl_sync(kFull, wb, l), ln = __shfl_sync(kFull, len, l);
                if (lw == 0) {
                    if (lane == l) {
                        a.sizes[j] = -1;
                        a.stage_off[j] = 0;
                        a.ovf_list[atomicAdd(a.ovf_count, 1ull)] = (int64_t)j;
                        active = pend = false;
                        len = 0;
                    }
                    continue;
                }
                int32_t *b = q + (int64_t)(l - lane) * a.qcap;
                for (int32_t i0 = 0; i0 < ln; i0 += 32) {   // (read before it is overwritten)
                    const int32_t i = i0 + lane;
                    const int32_t v = i < ln ? __ldcg(b + lw + i) : 0;
                    __syncwarp();
                    if (i < ln) b[i] = v;
                    __syncwarp();
                }
                if (lane == l) fb = wb = 0;
            }
            if (!active) fb = wb = 0;                // nothing is left in the buffer
        }
        __syncwarp();
    }
    // what the lanes still hold
    {
        const int32_t mine = wb - fb;
        const int32_t upto = warp_incl_scan<int32_t>(mine, lane), excl = upto - mine;
        const int32_t tot = __shfl_sync(kFull, upto, 31);
        unsigned long long base = 0;
        if (lane == 0 && tot) base = atomicAdd(a.stage_cursor, (unsigned long long)tot);
        base = __shfl_sync(kFull, base, 0);
        if ((int64_t)base + tot <= a.stage_cap) {
            for (int32_t k = 0; k < nrec; ++k) {
                const uint2 r = __ldcg(recs + k * 32);
                a.stage_off[r.x] = (int64_t)base + excl + ((int32_t)r.y - fb);
            }
            for (int l = 0; l < 32; ++l) {
                const int32_t n = __shfl_sync(kFull, mine, l), o = __shfl_sync(kFull, excl, l);
                const int32_t f = __shfl_sync(kFull, fb, l);
                for (int32_t i = lane; i < n; i += 32)
                    a.stage[(int64_t)base + o + i] = __ldcg(q + (int64_t)(l - lane) * a.qcap + f + i);
            }
        } else if (lane == 0) {
            raise_status(a.status, kDevStageOverflow);
        }
    }
    tot_exam = warp_sum<unsigned long long>(tot_exam);
    tot_bytes = warp_sum<unsigned long long>(tot_bytes);
    if (lane == 0 && tot_exam) atomicAdd(a.examined, tot_exam);
    if (lane == 0 && tot_bytes) atomicAdd(a.alg_bytes, tot_bytes);
}

// LT search index.  vrec[v] = {eb, d, z, u} with u the common weight of v's
// in-edges when they all carry the same nonzero weight (0 otherwise).  For such
// a vertex the pick needs no table: the running sum of edge i is (i + 1) u, so a
// draw x picks edge floor(x / u) when that is below d and nothing otherwise; z is
// then floor((2^32 - 1) / u), which gives the quotient as the high word of x z,
// at most 2 too small (x / u - x z / 2^32 < 1 + x / 2^32).  Otherwise z is the
// tree offset | L << 28 with L the number of upper tree levels (tree offsets stay
// below 2^28 since m < 2^31).
// For vertex v with in-edges [eb, eb + d):
//   leaf[e] = (sum of w over v's in-edges up to and including e) << 31 | src(e)
// (the running sum is at most 2^32 for valid LT weights -- 33 bits -- and
// source ids stay below 2^31, so the pair packs into 64 bits), and for
// d > 32 the upper levels l = L .. 1 of a fanout-32 tree, stored top-down at
// tree[tree_off(v) ..]: level l has ceil(d / 32^l) entries, entry i being the
// running sum at the last leaf of its 32^l-leaf block.
__device__ __forceinline__ int64_t lt_tree_size(int64_t d) {
    int64_t total = 0;
    while (d > 32) {
        d = (d + 31) >> 5;
        total += d;
    }
    return total;
}

__device__ __forceinline__ uint4 lt_record(int64_t b, int64_t d, uint32_t tree, uint32_t w) {
    return make_uint4((uint32_t)b, (uint32_t)d, w ? 0xffffffffu / w : tree, w);
}

// In-degree above which one block, not one warp, builds a vertex's running
// sums (a warp on R-MAT's largest in-list, ~7 x 10^4 edges, is the whole build's
// critical path).  At most m / (kLtBlockDeg + 1) vertices qualify.
constexpr int64_t kLtBlockDeg = 1024;

// Tree size of every vertex; lists the vertices of k_lt_index_block in big
// (in no particular order; nbig counts them).
__global__ void k_lt_tree_sizes(const int64_t *in_off, int64_t n, int32_t *sizes, int32_t *big,
                                int *nbig) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t d = in_off[v + 1] - in_off[v];
        sizes[v] = (int32_t)lt_tree_size(d);
        if (d > kLtBlockDeg) big[atomicAdd(nbig, 1)] = (int32_t)v;
    }
}

// Vertices with at most 32 in-edges (no upper tree levels): one thread each.
// The three index kernels write the vertex records and the flags always, and
// the running sums (leaf) and tree levels only when leaf is non-null.
__global__ void k_lt_index_small(const int64_t *in_off, const int32_t *in_src, const uint32_t *w,
                                 const int64_t *tree_off, unsigned long long *leaf, uint4 *vrec,
                                 int64_t n, int *invalid) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = in_off[v], e = in_off[v + 1], d = e - b;
        if (d > 32) continue;   // k_lt_index
        unsigned long long c = 0;
        const uint32_t w0 = d > 0 ? w[b] : 0u;
        bool same = true;
        for (int64_t i = b; i < e; ++i) {
            const uint32_t wi = w[i];
            same &= wi == w0;
            c += (unsigned long long)wi;
            if (leaf) leaf[i] = (c << 31) | (unsigned long long)(uint32_t)in_src[i];
        }
        if (c > (1ull << 32)) atomicExch(invalid, 1);
        if (d > 0 && !(same && w0 != 0u)) invalid[2] = 1;   // the cut points are needed
        vrec[v] = lt_record(b, d, (uint32_t)tree_off[v], same ? w0 : 0u);
    }
}

// Vertices with more than 32 in-edges: one warp each, running sums by warp
// scans, then the upper levels of the fanout-32 tree.
__global__ void k_lt_index(const int64_t *in_off, const int32_t *in_src, const uint32_t *w,
                           const int64_t *tree_off, unsigned long long *leaf,
                           unsigned long long *tree, uint4 *vrec, int64_t n, int *invalid) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t v = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); v < n;
         v += nw) {
        const int64_t b = in_off[v], e = in_off[v + 1], d = e - b;
        if (d <= 32 || d > kLtBlockDeg) continue;   // k_lt_index_small, k_lt_index_block
        unsigned long long carry = 0;
        const uint32_t w0 = w[b];
        bool same = true;
        for (int64_t base = b; base < e; base += 32) {
            const int64_t i = base + lane;
            const uint32_t wi = i < e ? w[i] : w0;
            same &= wi == w0;
            const unsigned long long x = i < e ? (unsigned long long)wi : 0ull;
            const unsigned long long incl = warp_incl_scan<unsigned long long>(x, lane);
            if (leaf && i < e)
                leaf[i] = ((carry + incl) << 31) | (unsigned long long)(uint32_t)in_src[i];
            carry += __shfl_sync(kFull, incl, 31);
        }
        same = __all_sync(kFull, same);
        if (lane == 0 && carry > (1ull << 32)) atomicExch(invalid, 1);
        if (lane == 0 && !(same && w0 != 0u)) invalid[2] = 1;
        int L = 0;
        for (int64_t t = d; t > 32; t = (t + 31) >> 5) ++L;
        if (lane == 0)
            vrec[v] = lt_record(b, d, (uint32_t)tree_off[v] | ((uint32_t)L << 28), same ? w0 : 0u);
        __syncwarp();
        if (!leaf) continue;
        // upper levels, top-down
        unsigned long long *lvl = tree + tree_off[v];
        for (int l = L; l >= 1; --l) {
            const int64_t sz = (d + (1ll << (5 * l)) - 1) >> (5 * l);
            for (int64_t i = lane; i < sz; i += 32) {
                const int64_t last = min((i + 1) << (5 * l), d) - 1;
                lvl[i] = leaf[b + last] >> 31;
            }
            lvl += sz;
        }
    }
}

// Vertices with more than kLtBlockDeg in-edges: one block of 256 threads each,
// 2048 edges per pass (8 consecutive ones per thread: sequential sums, then a
// block scan of the thread totals), then the upper tree levels as above.
__global__ void __launch_bounds__(256) k_lt_index_block(
    const int64_t *in_off, const int32_t *in_src, const uint32_t *w, const int64_t *tree_off,
    const int32_t *big, int nbig, unsigned long long *leaf, unsigned long long *tree, uint4 *vrec,
    int *invalid) {
    __shared__ unsigned long long wsum[8];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int j = blockIdx.x; j < nbig; j += gridDim.x) {
        const int64_t v = big[j];
        const int64_t b = in_off[v], e = in_off[v + 1], d = e - b;
        const uint32_t w0 = w[b];
        bool same = true;
        unsigned long long carry = 0;
        for (int64_t base = b; base < e; base += 2048) {
            const int64_t i0 = base + (int64_t)tid * 8;
            unsigned long long s[8], run = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t wi = i0 + q < e ? w[i0 + q] : w0;
                same &= wi == w0;
                run += i0 + q < e ? (unsigned long long)wi : 0ull;
                s[q] = run;
            }
            const unsigned long long incl = warp_incl_scan<unsigned long long>(run, lane);
            if (lane == 31) wsum[wid] = incl;
            __syncthreads();
            unsigned long long before = 0, tot = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const unsigned long long x = wsum[q];
                before += q < wid ? x : 0ull;
                tot += x;
            }
            const unsigned long long off = carry + before + (incl - run);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (leaf && i0 + q < e)
                    leaf[i0 + q] = ((off + s[q]) << 31) | (unsigned long long)(uint32_t)in_src[i0 + q];
            carry += tot;
            __syncthreads();   // wsum is rewritten by the next pass
        }
        same = __syncthreads_and(same) != 0;
        if (tid == 0 && carry > (1ull << 32)) atomicExch(invalid, 1);
        if (tid == 0 && !(same && w0 != 0u)) invalid[2] = 1;
        int L = 0;
        for (int64_t t = d; t > 32; t = (t + 31) >> 5) ++L;
        if (tid == 0)
            vrec[v] = lt_record(b, d, (uint32_t)tree_off[v] | ((uint32_t)L << 28), same ? w0 : 0u);
        __syncthreads();   // every leaf of v written by the block is visible to it
        if (!leaf) continue;   // (block-uniform)
        unsigned long long *lvl = tree + tree_off[v];
        for (int l = L; l >= 1; --l) {
            const int64_t sz = (d + (1ll << (5 * l)) - 1) >> (5 * l);
            for (int64_t i = tid; i < sz; i += blockDim.x) {
                const int64_t last = min((i + 1) << (5 * l), d) - 1;
                lvl[i] = leaf[b + last] >> 31;
            }
            lvl += sz;
        }
    }
}

// Cut points of the inverse-CDF pick, exact for any weights.  A draw x of
// vertex v (in-edges [eb, eb + d)) falls in bucket b = floor(x d / 2^32); the
// smallest draw of bucket b is lo_b = ceil(b 2^32 / d).  guide[eb + b]
// describes the first in-edge e whose running sum exceeds lo_b, or the last
// in-edge when none does: {running sum low word, high word, source, e}.
// Every edge before e has a running sum <= lo_b <= x, so x picks e exactly
// when x < running sum(e); otherwise the pick lies after e (or there is none).
__global__ void k_lt_guide(const int64_t *in_off, const unsigned long long *leaf,
                           const uint4 *vrec, int64_t n, int64_t m, uint4 *guide) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m;
         t += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = n - 1;                  // vertex owning position t
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (in_off[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        if (vrec[lo].w != 0u) continue;              // equal weights: no table needed
        const int64_t eb = in_off[lo], d = in_off[lo + 1] - eb, b = t - eb;
        const unsigned long long lob =
            (((unsigned long long)b << 32) + (unsigned long long)d - 1ull) / (unsigned long long)d;
        int64_t l2 = 0, h2 = d;                      // first e with lo_b < running sum(e)
        while (l2 < h2) {
            const int64_t mid = (l2 + h2) >> 1;
            if (lob < (leaf[eb + mid] >> 31)) h2 = mid;
            else l2 = mid + 1;
        }
        const int64_t e = l2 < d ? l2 : d - 1;
        const unsigned long long r = leaf[eb + e];
        const unsigned long long cum = r >> 31;
        guide[t] = make_uint4((uint32_t)cum, (uint32_t)(cum >> 32), (uint32_t)(r & 0x7fffffffull),
                              (uint32_t)e);
    }
}

// ---------------------------------------------------------------------------
// segmented sort: every segment [seg_off[i], seg_off[i+1]) ascending
// ---------------------------------------------------------------------------
template <typename Key>
__device__ __forceinline__ Key key_max();
template <>
__device__ __forceinline__ int32_t key_max<int32_t>() { return 0x7fffffff; }

template <typename Key>
__device__ __forceinline__ void order_pair(Key &x, Key &y) {
    const Key lo = min(x, y), hi = max(x, y);
    x = lo;
    y = hi;
}

// N keys of one thread ascending (N a power of two, fully unrolled): Batcher's
// odd-even merge sort, 63 comparators for 16 keys where a bitonic network has 80.
template <typename Key, int N>
__device__ __forceinline__ void thread_sort(Key (&v)[N]) {
#pragma unroll
    for (int p = 1; p < N; p <<= 1) {
#pragma unroll
        for (int d = p; d > 0; d >>= 1) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int x = i - d % p;             // i heads a pair of this pass?
                if (x >= 0 && i + d < N && x % (2 * d) < d && i / (2 * p) == (i + d) / (2 * p))
                    order_pair(v[i], v[i + d]);
            }
        }
    }
}

// 32 E keys of a warp ascending, the lane's E keys consecutive in that order:
// bitonic merges whose first pass pairs a block's halves mirrored, so that every
// pass keeps the smaller key at the lower place.  Whatever E, 15 passes cross
// lanes (a shuffle and a selected minimum per key); the others are a minimum and
// a maximum in registers.
template <typename Key, int E>
__device__ __forceinline__ void warp_sort_regs(Key (&v)[E], int lane) {
    thread_sort<Key, E>(v);
#pragma unroll
    for (int q = 2; q <= 32; q <<= 1) {              // blocks of q lanes
        const bool low = (lane & (q >> 1)) == 0;
#pragma unroll
        for (int r = 0; r < (E + 1) / 2; ++r) {
            const Key a = __shfl_xor_sync(kFull, v[r], q - 1);
            if (r != E - 1 - r) {
                const Key b = __shfl_xor_sync(kFull, v[E - 1 - r], q - 1);
                v[r] = low ? min(v[r], b) : max(v[r], b);
            }
            v[E - 1 - r] = low ? min(v[E - 1 - r], a) : max(v[E - 1 - r], a);
        }
#pragma unroll
        for (int j = q >> 2; j > 0; j >>= 1) {
            const bool lo = (lane & j) == 0;
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const Key o = __shfl_xor_sync(kFull, v[r], j);
                v[r] = lo ? min(v[r], o) : max(v[r], o);
            }
        }
#pragma unroll
        for (int j = E >> 1; j > 0; j >>= 1) {
#pragma unroll
            for (int r = 0; r < E; ++r)
                if (!(r & j)) order_pair(v[r], v[r | j]);
        }
    }
}

// At most 32 E keys of src, sorted, to buf: key i at word i + i / 32 (the
// padding keeps either side free of bank conflicts).
template <typename Key, int E>
__device__ __forceinline__ void warp_sort_to(Key *buf, const Key *src, int len, int lane) {
    Key v[E];
#pragma unroll
    for (int r = 0; r < E; ++r) v[r] = r * 32 + lane < len ? src[r * 32 + lane] : key_max<Key>();
    warp_sort_regs<Key, E>(v, lane);
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const int i = lane * E + r;
        buf[i + (i >> 5)] = v[r];
    }
    __syncwarp();
}

template <typename Key, int E>
__device__ __forceinline__ void warp_sort_copy(Key *out, const Key *src, int len, Key *buf,
                                               int lane) {
    warp_sort_to<Key, E>(buf, src, len, lane);
#pragma unroll
    for (int r = 0; r < E; ++r)
        if (r * 32 + lane < len) out[r * 32 + lane] = buf[r * 33 + lane];
}

// 513 to 1,024 distinct keys: two sorted runs of 512 at most, then every key to
// its place in its run plus the number of smaller keys of the other run.
// (1,024 keys in registers would leave 16 warps an SM.)
constexpr int kSortRun = 512, kSortRunWords = kSortRun + kSortRun / 32;
template <typename Key>
__device__ __forceinline__ void warp_sort_two(Key *out, const Key *src, int len, Key *buf,
                                              int lane) {
#pragma unroll 1
    for (int h = 0; h < 2; ++h)
        warp_sort_to<Key, kSortRun / 32>(buf + h * kSortRunWords, src + h * kSortRun,
                                         h ? len - kSortRun : kSortRun, lane);
    for (int t = lane; t < len; t += 32) {
        const int h = t >= kSortRun, i = t - h * kSortRun;
        const Key x = buf[h * kSortRunWords + i + (i >> 5)];
        const Key *o = buf + (1 - h) * kSortRunWords;
        int lo = 0, hi = h ? kSortRun : len - kSortRun;
        while (lo < hi) {
            const int m = (lo + hi) >> 1;
            if (o[m + (m >> 5)] < x) lo = m + 1;
            else hi = m;
        }
        out[i + lo] = x;
    }
}

constexpr int kSortBuf = 2 * kSortRunWords;  // words of a warp's buffer
static_assert(kWarpSortKeys == 2 * kSortRun, "two runs");

// One segment sorted by the whole warp in registers (len > kLaneSort), or listed
// in `big` for k_sort_block.  Instructions bound it.  Against bitonic passes over
// keys a lane-stride apart (where most passes are shuffles) and, beyond 512 keys,
// over shared memory: the 5.9 M weighted-cascade sets of an IMM run 3.68 ->
// 1.02 ms, 4.2 M LT walks of 41 members 1.25 -> .93, 200 k sets at scale 15 .148
// -> .040.  Five blocks an SM: three cost 5 to 20 % more.
template <typename Key>
__device__ __forceinline__ void warp_sort_segment(Key *out, const Key *src, int64_t len, int64_t i,
                                                  Key *buf, int64_t *big, unsigned long long *nbig,
                                                  int lane) {
    if (len <= 32) {
        Key v[1] = {lane < len ? src[lane] : key_max<Key>()};
        warp_sort_regs<Key, 1>(v, lane);
        if (lane < len) out[lane] = v[0];
    } else if (len <= 64) warp_sort_copy<Key, 2>(out, src, (int)len, buf, lane);
    else if (len <= 128) warp_sort_copy<Key, 4>(out, src, (int)len, buf, lane);
    else if (len <= 256) warp_sort_copy<Key, 8>(out, src, (int)len, buf, lane);
    else if (len <= 512) warp_sort_copy<Key, 16>(out, src, (int)len, buf, lane);
    else if (len <= kWarpSortKeys) warp_sort_two<Key>(out, src, (int)len, buf, lane);
    else if (lane == 0) big[atomicAdd(nbig, 1ull)] = i;
    __syncwarp();
}

// Copies stage segments into place and sorts the short ones.  A warp takes 32 consecutive segments at once (their offsets in
// one coalesced load each): segments of at most kLaneSort keys -- most RRR
// sets -- are sorted by their own lane in registers; the longer ones are
// listed in `mid` for k_sort_mid, one warp each.
constexpr int kLaneSort = 16;

template <typename Key>
__global__ void __launch_bounds__(256, 5) k_sort_small(Key *dst, const int64_t *seg_off, int64_t nseg,
                                                    const Key *stage, const int64_t *stage_off,
                                                    int64_t *mid, unsigned long long *nmid,
                                                    bool inline_long, int64_t *big,
                                                    unsigned long long *nbig) {
    __shared__ Key sbuf[8][kSortBuf];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t nw = (int64_t)gridDim.x * 8;
    for (int64_t i0 = ((int64_t)blockIdx.x * 8 + wib) * 32; i0 < nseg; i0 += nw * 32) {
        const int64_t i = i0 + lane;
        int64_t o = 0, len = 0;
        const Key *src = nullptr;
        if (i < nseg) {
            o = seg_off[i];
            len = seg_off[i + 1] - o;
            src = stage + (stage_off[i] & ~kStageAscending);
        }
        Key *out = dst + o;
        if (len == 1) {
            out[0] = src[0];
        } else if (len > 1 && len <= kLaneSort) {
            Key v[kLaneSort];
#pragma unroll
            for (int r = 0; r < kLaneSort; ++r) v[r] = r < len ? src[r] : key_max<Key>();
            thread_sort<Key, kLaneSort>(v);
#pragma unroll
            for (int r = 0; r < kLaneSort; ++r)
                if (r < len) out[r] = v[r];
        }
        unsigned longer = __ballot_sync(kFull, len > kLaneSort);
        if (longer && inline_long) {   // many segments per warp: the warp sorts them itself
            while (longer) {
                const int l = __ffs(longer) - 1;
                longer &= longer - 1;
                const int64_t ol = __shfl_sync(kFull, o, l);
                const int64_t ll = __shfl_sync(kFull, len, l);
                const Key *sl = (const Key *)__shfl_sync(kFull, (unsigned long long)src, l);
                warp_sort_segment<Key>(dst + ol, sl, ll, i0 + l, sbuf[wib], big, nbig, lane);
            }
        } else if (longer) {
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(nmid, (unsigned long long)__popc(longer));
            base = __shfl_sync(kFull, base, 0);
            if (len > kLaneSort) mid[base + __popc(longer & ((1u << lane) - 1u))] = i;
        }
    }
}

// One warp per listed segment longer than kLaneSort keys (grid-stride over
// the list): sorted in registers or in the warp's shared buffer; segments
// longer than that buffer are listed in `big`.
template <typename Key>
__global__ void __launch_bounds__(256, 5) k_sort_mid(Key *dst, const int64_t *seg_off,
                                                  const Key *stage, const int64_t *stage_off,
                                                  const int64_t *mid,
                                                  const unsigned long long *nmid, int64_t *big,
                                                  unsigned long long *nbig) {
    __shared__ Key sbuf[8][kSortBuf];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t nw = (int64_t)gridDim.x * 8;
    const int64_t cnt = (int64_t)*nmid;
    for (int64_t x = (int64_t)blockIdx.x * 8 + wib; x < cnt; x += nw) {
        const int64_t i = mid[x];
        const int64_t o = seg_off[i];
        const int64_t len = seg_off[i + 1] - o;
        warp_sort_segment<Key>(dst + o, stage + (stage_off[i] & ~kStageAscending), len, i,
                               sbuf[wib], big, nbig, lane);
    }
}

// A block sorts up to kBlockKeys keys a thread; sets up to kMidSortCap go to
// blocks of 256, of which an SM holds four, the others to blocks of 1,024.
constexpr int kBlockKeys = 16;
constexpr int kMidSortCap = 256 * kBlockKeys;
static_assert(kBlockSortCap == 1024 * kBlockKeys, "the larger blocks");

// One block of T threads per listed segment of its class: copied from the stage
// when it is ascending there, or listed in `giant` for k_sort_giant when it has
// more than kBlockSortCap keys, else sorted: runs of kSortRun keys by the warps,
// then merged pairwise.  A key's place after a merge is its place in its run plus
// the number of smaller keys in the other (keys are distinct), found by a binary
// search; the keys wait in registers while the buffer is rewritten.
// Against a bitonic network over shared memory (66 to 105 passes of it): the long
// sets of an IMM run, weighted cascade on the LiveJournal shape, 4.1 -> 1.2 ms.
template <typename Key, int T>
__global__ void __launch_bounds__(T, 1024 / T) k_sort_block(Key *dst, const int64_t *seg_off,
                                                            const Key *stage,
                                                            const int64_t *stage_off,
                                                            const int64_t *big,
                                                            const unsigned long long *nbig,
                                                            int64_t *giant,
                                                            unsigned long long *ngiant) {
    extern __shared__ __align__(16) unsigned char sraw[];
    Key *buf = reinterpret_cast<Key *>(sraw);
    const int64_t nb = (int64_t)*nbig;
    const int tid = threadIdx.x, lane = tid & 31;
    for (int64_t b = blockIdx.x; b < nb; b += gridDim.x) {
        const int64_t i = big[b];
        const int64_t o = seg_off[i];
        const int64_t seg = seg_off[i + 1] - o;
        if ((T == 256) != (seg <= kMidSortCap)) continue;
        const int64_t so = stage_off[i];
        const Key *src = stage + (so & ~kStageAscending);
        if (so & kStageAscending) {
            constexpr int U = 8;
            for (int64_t t0 = tid; t0 < seg; t0 += (int64_t)U * T) {
                Key v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t t = t0 + (int64_t)u * T;
                    if (t < seg) v[u] = src[t];
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t t = t0 + (int64_t)u * T;
                    if (t < seg) dst[o + t] = v[u];
                }
            }
            continue;
        }
        if (seg > kBlockSortCap) {
            if (tid == 0) giant[atomicAdd(ngiant, 1ull)] = i;
            continue;
        }
        const int len = (int)seg;
        for (int r = tid >> 5; r * kSortRun < len; r += T / 32)
            warp_sort_to<Key, kSortRun / 32>(buf + r * kSortRunWords, src + r * kSortRun,
                                             len - r * kSortRun, lane);
        __syncthreads();
        for (int w = kSortRun; w < len; w <<= 1) {
            const bool last = 2 * w >= len;
            Key x[kBlockKeys];
            int at[kBlockKeys];
#pragma unroll
            for (int u = 0; u < kBlockKeys; ++u) {
                const int t = tid + u * T;
                if (t < len) {
                    x[u] = buf[t + (t >> 5)];
                    const int first = t & ~(2 * w - 1);          // of the pair of runs
                    const int from = t & w ? first : min(first + w, len);
                    int lo = from, hi = t & w ? first + w : min(first + 2 * w, len);
                    while (lo < hi) {
                        const int m = (lo + hi) >> 1;
                        if (buf[m + (m >> 5)] < x[u]) lo = m + 1;
                        else hi = m;
                    }
                    at[u] = first + (t & (w - 1)) + lo - from;
                    if (last) dst[o + at[u]] = x[u];
                }
            }
            __syncthreads();
            if (last) break;
#pragma unroll
            for (int u = 0; u < kBlockKeys; ++u)
                if (tid + u * T < len) buf[at[u] + (at[u] >> 5)] = x[u];
            __syncthreads();
        }
    }
}

// Unsorted segments longer than kBlockSortCap (LT walks) of distinct vertex
// ids: mark them in an n-bit bitmap (one per block) and read the bitmap back in
// order.
__global__ void __launch_bounds__(1024) k_sort_giant(int32_t *dst, const int64_t *seg_off,
                                                     const int32_t *stage,
                                                     const int64_t *stage_off,
                                                     const int64_t *giant,
                                                     const unsigned long long *ngiant,
                                                     uint32_t *bitmaps, int64_t words) {
    __shared__ int64_t sh[33];
    uint32_t *bm = bitmaps + (size_t)blockIdx.x * (size_t)words;
    const int64_t ng = (int64_t)*ngiant;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t b = blockIdx.x; b < ng; b += gridDim.x) {
        const int64_t i = giant[b];
        const int64_t o = seg_off[i];
        const int64_t len = seg_off[i + 1] - o;
        const int64_t so = stage_off[i];
        for (int64_t t = threadIdx.x; t < len; t += blockDim.x) {
            const uint32_t u = (uint32_t)stage[so + t];
            atomicOr(&bm[u >> 5], 1u << (u & 31));
        }
        __syncthreads();
        const int64_t per = (words + blockDim.x - 1) / blockDim.x;
        const int64_t w0 = (int64_t)threadIdx.x * per;
        const int64_t w1 = min(words, w0 + per);
        int64_t cnt = 0;
        for (int64_t x = w0; x < w1; ++x) cnt += __popc(bm[x]);
        // block exclusive scan of cnt
        int64_t incl = warp_incl_scan<int64_t>(cnt, lane);
        if (lane == 31) sh[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            int64_t v = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0;
            int64_t vi = warp_incl_scan<int64_t>(v, lane);
            if (lane < (int)(blockDim.x >> 5)) sh[lane] = vi - v;
        }
        __syncthreads();
        int64_t at = o + sh[warp] + incl - cnt;
        __syncthreads();
        for (int64_t x = w0; x < w1; ++x) {
            uint32_t bits = bm[x];
            while (bits) {
                const int bpos = __ffs(bits) - 1;
                bits &= bits - 1;
                dst[at++] = (int32_t)(x * 32 + bpos);
            }
        }
        __syncthreads();
        for (int64_t x = w0; x < w1; ++x) bm[x] = 0;
        __syncthreads();
    }
}

int blocks_for(const void *kernel, int threads, size_t smem) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    if (per_sm < 1) per_sm = 1;
    return per_sm * num_sms();
}

}  // namespace

static std::mutex g_lt_index_mu;   // graphs are shared by serving workers (LT and IC records)

im_status build_lt_index(im_graph *g, cudaStream_t st) {
    std::lock_guard<std::mutex> lk(g_lt_index_mu);
    if (g->lt_vrec) return IM_OK;   // set only once the whole index is built
    const int64_t n = g->n, m = g->m;
    CallBuf sizes_buf(st), big_buf(st), toff_buf(st), flags_buf(st);
    // the index itself: handed to g once complete, freed on any failure
    struct Index {
        unsigned long long *leaf = nullptr, *tree = nullptr;
        uint4 *vrec = nullptr, *guide = nullptr;
        ~Index() {
            if (leaf || tree || vrec || guide) {
                cudaDeviceSynchronize();
                for (void *p : {(void *)leaf, (void *)tree, (void *)vrec, (void *)guide})
                    cudaFree(p);
            }
        }
    } x;
    const int64_t big_cap = m / (kLtBlockDeg + 1) + 1;
    IM_TRY(sizes_buf.alloc((size_t)n * 4));
    IM_TRY(big_buf.alloc((size_t)big_cap * 4));
    IM_TRY(toff_buf.alloc((size_t)(n + 1) * 8 + scan_tmp_bytes(n) + 256));
    IM_TRY(flags_buf.alloc(3 * sizeof(int)));
    struct {
        int32_t *sizes, *big;
        int64_t *toff;
        int *flags;             // [0] weights of some vertex sum above 2^32, [1] listed
                                // vertices, [2] some vertex needs the cut points
    } t = {sizes_buf.as<int32_t>(), big_buf.as<int32_t>(), toff_buf.as<int64_t>(), flags_buf.as<int>()};
    IM_CUDA(cudaMemsetAsync(t.flags, 0, 3 * sizeof(int), st));
    {
        KernelTimer kt(st, "lt_index");
        k_lt_tree_sizes<<<num_sms() * 4, 256, 0, st>>>(g->in_off, n, t.sizes, t.big, t.flags + 1);
    }
    void *scan_tmp = (char *)t.toff + (((size_t)(n + 1) * 8 + 255) & ~(size_t)255);
    IM_TRY(exclusive_scan_i32_to_i64(t.sizes, t.toff, n, nullptr, scan_tmp, scan_tmp_bytes(n), st));
    int64_t tree_total = 0;
    int nbig = 0;
    IM_CUDA(cudaMemcpyAsync(&tree_total, t.toff + n, 8, cudaMemcpyDeviceToHost, st));
    IM_CUDA(cudaMemcpyAsync(&nbig, t.flags + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
    IM_CUDA(cudaStreamSynchronize(st));
    if (nbig < 0 || nbig > big_cap) {
        set_error("LT index: vertex list out of range");
        return IM_ERR_CUDA;
    }
    IM_CUDA(cudaMalloc(&x.vrec, (size_t)n * sizeof(uint4)));
    // vertex records and flags; running sums and tree when leaf is set
    auto index_pass = [&]() -> im_status {
        KernelTimer kt(st, "lt_index");
        k_lt_index_small<<<num_sms() * 8, 256, 0, st>>>(g->in_off, g->in_src, g->w, t.toff,
                                                        x.leaf, x.vrec, n, t.flags);
        k_lt_index<<<num_sms() * 8, 256, 0, st>>>(g->in_off, g->in_src, g->w, t.toff, x.leaf,
                                                  x.tree, x.vrec, n, t.flags);
        if (nbig > 0)
            k_lt_index_block<<<std::min(nbig, num_sms() * 8), 256, 0, st>>>(
                g->in_off, g->in_src, g->w, t.toff, t.big, nbig, x.leaf, x.tree, x.vrec,
                t.flags);
        IM_CUDA(cudaGetLastError());
        return IM_OK;
    };
    // first the vertex records alone: when every vertex's in-edges weigh the
    // same (1/in-degree weights, for one) the walks pick by division and need
    // neither running sums, tree nor cut points
    IM_TRY(index_pass());
    int hflags[3] = {0, 0, 0};
    IM_CUDA(cudaMemcpyAsync(hflags, t.flags, sizeof(hflags), cudaMemcpyDeviceToHost, st));
    IM_CUDA(cudaStreamSynchronize(st));
    if (hflags[2] && m > 0) {
        // some vertex's in-edges weigh differently (or all zero): the full
        // index (the records are rewritten with the same values), then the cut
        // points, which serve only such vertices
        IM_CUDA(cudaMalloc(&x.leaf, (size_t)m * 8));
        IM_CUDA(cudaMalloc(&x.tree, (size_t)std::max<int64_t>(tree_total, 1) * 8));
        IM_TRY(index_pass());
        IM_CUDA(cudaMalloc(&x.guide, (size_t)m * sizeof(uint4)));
        {
            KernelTimer kt(st, "lt_index");
            k_lt_guide<<<num_sms() * 8, 256, 0, st>>>(g->in_off, x.leaf, x.vrec, n, m, x.guide);
        }
        IM_CUDA(cudaGetLastError());
        IM_CUDA(cudaStreamSynchronize(st));
    }
    g->lt_valid = hflags[0] ? 0 : 1;
    g->lt_tree = x.tree;
    g->lt_vrec = x.vrec;
    g->lt_guide = x.guide;
    g->lt_leaf = x.leaf;
    x.leaf = x.tree = nullptr;
    x.vrec = x.guide = nullptr;
    return IM_OK;
}

// In-edge records of the IC samplers (k_ic_records), built on the first IC use
// of a graph and kept with it.
im_status build_ic_index(im_graph *g, cudaStream_t st) {
    std::lock_guard<std::mutex> lk(g_lt_index_mu);
    if (g->ic_rec) return IM_OK;   // set only once the records are complete
    uint4 *rec = nullptr;
    IM_CUDA(cudaMalloc((void **)&rec, (size_t)g->n * sizeof(uint4)));
    cudaError_t e;
    {
        KernelTimer kt(st, "ic_index");
        k_ic_records<<<num_sms() * 8, 256, 0, st>>>(g->in_off, g->w, g->n, rec);
    }
    if ((e = cudaGetLastError()) != cudaSuccess || (e = cudaStreamSynchronize(st)) != cudaSuccess) {
        cudaFree(rec);
        return cuda_fail(e, "IC index");
    }
    g->ic_rec = rec;
    return IM_OK;
}

QueryView query_view(const im_graph *g, uint64_t seed, uint64_t first) {
    QueryView v;
    v.in_off = g->in_off;
    v.in_src = g->in_src;
    v.w = g->w;
    v.ic_rec = g->ic_rec;
    v.lt_vrec = g->lt_vrec;
    v.lt_leaf = g->lt_leaf;
    v.lt_tree = g->lt_tree;
    v.lt_guide = g->lt_guide;
    v.seed = seed;
    v.n = (uint32_t)g->n;
    v.first = (uint32_t)first;
    return v;
}

static void (*lt1_kernel(int cache, bool one_key))(const SampleArgs) {
    if (cache == 0) return one_key ? k_sample_lt1<0, true> : k_sample_lt1<0, false>;
    if (cache == 1) return one_key ? k_sample_lt1<1, true> : k_sample_lt1<1, false>;
    return one_key ? k_sample_lt1<2, true> : k_sample_lt1<2, false>;
}

// ---------------------------------------------------------------------------
// One sampling launch over a table of queries (see SamplingJob).
// ---------------------------------------------------------------------------
im_status run_sampling(const SamplingJob &job, const std::function<im_status(size_t, void **)> &alloc,
                       cudaStream_t st, SamplingResult *res) {
    const im_model model = job.model;
    const int32_t nq = (int32_t)job.views.size();
    std::vector<int64_t> qstart(nq + 1, 0);
    for (int32_t q = 0; q < nq; ++q) qstart[q + 1] = qstart[q] + job.counts[q];
    const int64_t cnt = qstart[nq];
    const int64_t n = job.n_max;
    const bool smem_vis = model == IM_IC && n <= kSmemVisBits;
    const bool one_key = nq == 1;                    // the round keys go in the launch's arguments
    const int64_t vis_words = (n + 31) / 32;

    // launch shape: persistent, occupancy-sized
    int G = model == IM_LT ? (int)tune_value(IM_TUNE_LT_GROUP) : 32;
    if (G == 1 && cnt > kLT1MaxCount) G = 32;        // chunk bounds of k_sample_lt1 are 32-bit
    const int lt_cache = (int)tune_value(IM_TUNE_LT_CACHE);
    const bool lt1 = model == IM_LT && G == 1;      // one walk per thread
    const void *kern = model == IM_LT
                           ? (G == 1    ? (const void *)lt1_kernel(lt_cache, one_key)
                              : G == 8  ? (const void *)k_sample_lt<8>
                              : G == 16 ? (const void *)k_sample_lt<16>
                                        : (const void *)k_sample_lt<32>)
                       : smem_vis ? (one_key ? (const void *)k_sample_ic<true, true>
                                             : (const void *)k_sample_ic<true, false>)
                                  : (one_key ? (const void *)k_sample_ic<false, true>
                                             : (const void *)k_sample_ic<false, false>);
    const int threads = lt1 ? kLT1Threads : kSampleThreads;
    const size_t ic_words = (smem_vis ? (vis_words + 3) & ~(int64_t)3 : kICHash) + kICQueueSmem +
                            kCandCap;                // a warp's shared memory
    const size_t dyn_smem = model == IM_IC ? (size_t)kWarps * ic_words * 4
                            : lt1          ? (size_t)kBloomWords * kLT1Threads * 4
                                           : 0;
    if (dyn_smem > 48 * 1024)
        IM_TRY(raise_dyn_smem(kern, dyn_smem));
    int blocks = blocks_for(kern, threads, dyn_smem);
    // global visited bitmaps are n bits per warp: keep them within ~4 GB
    if (model == IM_IC && !smem_vis) {
        int64_t cap_blocks = std::max<int64_t>(
            num_sms(), (int64_t)(4ll << 30) / ((int64_t)kWarps * vis_words * 4));
        blocks = (int)std::min<int64_t>(blocks, cap_blocks);
    }
    const int64_t warps = (int64_t)blocks * (threads / 32);
    const int64_t slots = warps * (32 / G);           // one queue per walk in flight
    // (a walk of one thread goes up to two entries past its end)
    const int64_t qcap =
        lt1 ? std::min<int64_t>((n + 3 + 3) & ~(int64_t)3, kQueueCapLT1)
            : std::min<int64_t>(n, model == IM_LT ? kQueueCapLT : kQueueCapIC);

    // scratch layout
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t at = off;
        off += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t o_ctr = take(8 * sizeof(unsigned long long));
    const size_t o_views = take((size_t)nq * sizeof(QueryView));
    const size_t o_qstart = take((size_t)(nq + 1) * 8);
    const size_t o_soff = take((size_t)cnt * 8);
    const size_t o_sizes = take((size_t)cnt * 4);
    const size_t o_ovf = take((size_t)cnt * 8);
    const size_t o_scan = take(scan_tmp_bytes(cnt));
    const size_t o_sort = take((size_t)(2 + 2 * cnt) * 8);
    const int64_t hand_cap = model == IM_IC ? std::min<int64_t>(kICHandCap, cnt * qcap) : 0;
    const size_t o_handed = take(model == IM_IC ? (size_t)(hand_cap / kICWarpFront + 1) * sizeof(Handed) : 0);
    const size_t o_hand = take((size_t)hand_cap * 4);
    const size_t o_recs = take(lt1 ? (size_t)slots * kLT1Recs * sizeof(uint2) : 0);
    const size_t o_q = take((size_t)slots * qcap * 4);
    const size_t o_vis = take(model == IM_IC && !smem_vis ? (size_t)warps * vis_words * 4 : 0);
    void *base = nullptr;
    im_status rs = alloc(off, &base);
    if (rs != IM_OK) return rs;
    char *B = (char *)base;
    unsigned long long *ctr = (unsigned long long *)(B + o_ctr);
    // ctr: 0 work, 1 stage cursor, 2 examined, 3 overflow count, 4 status (int),
    //      5 algorithmic bytes, 6 handed-over members, 7 long sets (SampleArgs::nlong)
    IM_CUDA(cudaMemsetAsync(ctr, 0, 8 * sizeof(unsigned long long), st));
    IM_CUDA(cudaMemcpyAsync(B + o_views, job.views.data(), (size_t)nq * sizeof(QueryView),
                            cudaMemcpyHostToDevice, st));
    IM_CUDA(cudaMemcpyAsync(B + o_qstart, qstart.data(), (size_t)(nq + 1) * 8,
                            cudaMemcpyHostToDevice, st));

    SampleArgs a;
    a.qv = (const QueryView *)(B + o_views);
    a.qstart = (const int64_t *)(B + o_qstart);
    a.nq = nq;
    a.count = cnt;
    a.list = nullptr;
    a.stage = job.stage;
    a.stage_cap = job.stage_cap;
    a.stage_cursor = ctr + 1;
    a.stage_off = (int64_t *)(B + o_soff);
    a.sizes = (int32_t *)(B + o_sizes);
    a.queues = (int32_t *)(B + o_q);
    a.qcap = qcap;
    a.gvis = (uint32_t *)(B + o_vis);
    a.vis_words = vis_words;
    a.examined = ctr + 2;
    a.alg_bytes = ctr + 5;
    a.work = ctr;
    a.ovf_list = (int64_t *)(B + o_ovf);
    a.ovf_count = ctr + 3;
    a.status = (int *)(ctr + 4);
    a.handed = (Handed *)(B + o_handed);
    a.hand = (int32_t *)(B + o_hand);
    a.hand_cap = hand_cap;
    a.hand_cursor = ctr + 6;
    a.recs = (uint2 *)(B + o_recs);
    a.nlong = ctr + 7;
    for (int r = 0; r < 10; ++r) {
        a.rk[2 * r] = one_key ? (uint32_t)job.views[0].seed + (uint32_t)r * 0x9E3779B9u : 0u;
        a.rk[2 * r + 1] =
            one_key ? (uint32_t)(job.views[0].seed >> 32) + (uint32_t)r * 0xBB67AE85u : 0u;
    }

    auto launch = [&](int nblocks, int group) {
        KernelTimer kt(st, model == IM_LT ? "sample_lt" : "sample_ic");
        if (model == IM_LT) {
            if (group == 1) lt1_kernel(lt_cache, one_key)<<<nblocks, kLT1Threads, dyn_smem, st>>>(a);
            else if (group == 8) k_sample_lt<8><<<nblocks, kSampleThreads, 0, st>>>(a);
            else if (group == 16) k_sample_lt<16><<<nblocks, kSampleThreads, 0, st>>>(a);
            else k_sample_lt<32><<<nblocks, kSampleThreads, 0, st>>>(a);
        } else if (smem_vis) {
            if (one_key) k_sample_ic<true, true><<<nblocks, kSampleThreads, dyn_smem, st>>>(a);
            else k_sample_ic<true, false><<<nblocks, kSampleThreads, dyn_smem, st>>>(a);
        } else {
            if (one_key) k_sample_ic<false, true><<<nblocks, kSampleThreads, dyn_smem, st>>>(a);
            else k_sample_ic<false, false><<<nblocks, kSampleThreads, dyn_smem, st>>>(a);
        }
    };
    launch(blocks, G);
    IM_CUDA(cudaGetLastError());

    unsigned long long hc[8];
    IM_CUDA(cudaMemcpyAsync(hc, ctr, sizeof(hc), cudaMemcpyDeviceToHost, st));
    IM_CUDA(cudaStreamSynchronize(st));
    int dev_status = (int)(hc[4] & 0xffffffffu);
    if (dev_status == kDevOk && hc[3] > 0) {
        // second pass for the sets the first gave up (LT: longer than the
        // per-walk queue; IC: longer than that, or of too many in-edges for one
        // warp), with queues of n entries
        const int64_t novf = (int64_t)hc[3];
        const bool ic_big = model == IM_IC;
        // IC: one block per sample; LT: one walk per warp
        const int64_t per_unit = (int64_t)n * 4 + (ic_big ? vis_words * 4 : 0);
        int64_t units = ic_big ? std::min<int64_t>(novf, (int64_t)num_sms())
                               : std::min<int64_t>((novf + kWarps - 1) / kWarps, num_sms()) * kWarps;
        if (ic_big) units = std::max<int64_t>(1, std::min<int64_t>(units, (4ll << 30) / per_unit));
        const int nb2 = (int)(ic_big ? units : std::max<int64_t>(1, units / kWarps));
        const size_t need2 = (size_t)units * (size_t)per_unit;
        // the first pass's queues and bitmaps are free by now, and mostly enough
        // (mapping fresh memory took 2 to 5 ms a call)
        const bool own = need2 > off - o_q;
        CallBuf q2_buf(st);
        if (own) IM_TRY(q2_buf.alloc(need2));
        int32_t *q2 = own ? q2_buf.as<int32_t>() : (int32_t *)(B + o_q);
        uint32_t *vis2 = (uint32_t *)((char *)q2 + (size_t)units * (size_t)n * 4);
        if (ic_big) IM_CUDA(cudaMemsetAsync(vis2, 0, (size_t)units * vis_words * 4, st));
        IM_CUDA(cudaMemsetAsync(ctr, 0, sizeof(unsigned long long), st));
        SampleArgs a2 = a;
        a2.list = a.ovf_list;
        a2.count = novf;
        a2.queues = q2;
        a2.qcap = n;
        a2.gvis = vis2;
        a2.vis_words = vis_words;
        a2.ovf_list = a.ovf_list + cnt;   // never written: qcap = n cannot overflow
        a = a2;
        if (ic_big) {
            KernelTimer kt(st, "sample_ic_big");
            if (one_key) k_sample_ic_big<true><<<nb2, kICBigThreads, 0, st>>>(a);
            else k_sample_ic_big<false><<<nb2, kICBigThreads, 0, st>>>(a);
        } else {
            launch(nb2, 32);   // one walk per warp: queues of n entries for the longest walks
        }
        IM_CUDA(cudaGetLastError());
        IM_CUDA(cudaMemcpyAsync(hc, ctr, sizeof(hc), cudaMemcpyDeviceToHost, st));
        IM_CUDA(cudaStreamSynchronize(st));
        dev_status = (int)(hc[4] & 0xffffffffu);
    }
    if (dev_status != kDevOk) {
        if (dev_status == kDevStageOverflow) {
            set_error("RRR set capacity exceeded while sampling");
            return IM_ERR_CAPACITY;
        }
        return map_dev_status(dev_status, "sampling");
    }
    res->stage_off = (int64_t *)(B + o_soff);
    res->sizes = (int32_t *)(B + o_sizes);
    res->scan_tmp = B + o_scan;
    res->sort_tmp = B + o_sort;
    res->total = cnt;
    res->added = (int64_t)hc[1];
    res->examined = (int64_t)hc[2];
    res->alg_bytes = (int64_t)hc[5];
    res->long_sets = hc[7];
    return IM_OK;
}

// Copies every set from the stage into dst at seg_off and sorts it ascending.
// long_sets: what the sampling counted (SamplingResult::long_sets), so that the
// passes for long sets are launched only when there are any.  tmp: (2 + 2 nseg)
// * 8 bytes.
im_status segmented_sort_sets(int32_t *dst, const int64_t *seg_off, int64_t nseg, const int32_t *stage,
                              const int64_t *stage_off, void *tmp, int64_t n_max,
                              unsigned long long long_sets, cudaStream_t st) {
    // tmp layout: [2 counters][list for k_sort_block, nseg][list for k_sort_mid, nseg]
    unsigned long long *ctr = (unsigned long long *)tmp;
    int64_t *big = (int64_t *)tmp + 2;
    int64_t *mid = big + nseg;
    if (nseg == 0) return IM_OK;
    IM_CUDA(cudaMemsetAsync(ctr, 0, 2 * sizeof(unsigned long long), st));
    const int gs = blocks_for((const void *)k_sort_small<int32_t>, 256, 0);
    // with at least four groups of 32 segments per warp the longer segments
    // spread over the warps anyway: each warp sorts its own; with fewer, they
    // are listed and k_sort_mid gives each its own warp
    const bool inline_long = nseg >= (int64_t)gs * 8 * 32 * 4;
    {
        KernelTimer kt(st, "sort_sets_warp");
        k_sort_small<int32_t><<<gs, 256, 0, st>>>(dst, seg_off, nseg, stage, stage_off, mid,
                                                   ctr + 1, inline_long, big, ctr);
        if (!inline_long) {
            const int gm = blocks_for((const void *)k_sort_mid<int32_t>, 256, 0);
            k_sort_mid<int32_t><<<gm, 256, 0, st>>>(dst, seg_off, stage, stage_off, mid, ctr + 1,
                                                     big, ctr);
        }
    }
    IM_CUDA(cudaGetLastError());
    if (long_sets == 0) return IM_OK;
    const size_t mid_smem = kMidSortCap / kSortRun * kSortRunWords * sizeof(int32_t);
    const size_t smem = kBlockSortCap / kSortRun * kSortRunWords * sizeof(int32_t);
    IM_TRY(raise_dyn_smem((const void *)k_sort_block<int32_t, 1024>, smem));
    IM_CUDA(cudaMemsetAsync(ctr + 1, 0, sizeof(unsigned long long), st));
    {
        KernelTimer kt(st, "sort_sets_block");
        k_sort_block<int32_t, 1024><<<num_sms(), 1024, smem, st>>>(dst, seg_off, stage, stage_off,
                                                                   big, ctr, mid, ctr + 1);
        k_sort_block<int32_t, 256><<<num_sms() * 4, 256, mid_smem, st>>>(
            dst, seg_off, stage, stage_off, big, ctr, mid, ctr + 1);
    }
    IM_CUDA(cudaGetLastError());
    const int64_t ngiant = (int64_t)(long_sets >> 32);
    if (ngiant > 0) {
        // an n-bit bitmap per block
        const int64_t gwords = (n_max + 31) / 32;
        const int blocks3 = (int)std::min<int64_t>(ngiant, num_sms());
        CallBuf gbm_buf(st);
        IM_TRY(gbm_buf.alloc((size_t)blocks3 * gwords * 4));
        uint32_t *gbm = gbm_buf.as<uint32_t>();
        IM_CUDA(cudaMemsetAsync(gbm, 0, (size_t)blocks3 * gwords * 4, st));
        {
            KernelTimer kt(st, "sort_sets_bitmap");
            k_sort_giant<<<blocks3, 1024, 0, st>>>(dst, seg_off, stage, stage_off, mid, ctr + 1,
                                                   gbm, gwords);
        }
        IM_CUDA(cudaGetLastError());
    }
    return IM_OK;
}

// ---------------------------------------------------------------------------
// Sample(G, count): append sample ids first .. first+count-1 to the pool.
// ---------------------------------------------------------------------------
im_status sample_append(const im_graph *gc, im_model model, uint64_t seed, uint64_t first,
                        uint64_t count, im_pool *pool, cudaStream_t st) {
    im_graph *g = const_cast<im_graph *>(gc);
    if (model == IM_LT) {
        im_status s = build_lt_index(g, st);
        if (s != IM_OK) return s;
        if (!g->lt_valid) {
            set_error("LT sampling needs every vertex's in-weights to sum to at most 2^32");
            return IM_ERR_INVALID_ARG;
        }
    } else {
        IM_TRY(build_ic_index(g, st));
    }
    if (count == 0) return IM_OK;
    if (pool->theta + (int64_t)count > pool->max_sets) {
        set_error("pool max_sets exceeded");
        return IM_ERR_CAPACITY;
    }
    const int64_t cnt = (int64_t)count;
    SamplingJob job;
    job.model = model;
    job.views.push_back(query_view(g, seed, first));
    job.counts.push_back(cnt);
    job.n_max = g->n;
    job.stage = pool->set_ids;                      // the index buffer doubles as the stage
    job.stage_cap = pool->max_entries - pool->total;
    pool->index_valid = false;
    SamplingResult r;
    im_status rs = run_sampling(job, [&](size_t b, void **p) { return pool_scratch(pool, b, p); },
                                st, &r);
    if (rs != IM_OK) {
        if (rs == IM_ERR_CAPACITY) set_error("pool max_entries exceeded while sampling");
        return rs;
    }
    // set_off[theta .. theta+cnt] = set_off[theta] + exclusive scan of sizes
    int64_t *so = pool->set_off + pool->theta;
    rs = exclusive_scan_i32_to_i64(r.sizes, so, cnt, so, r.scan_tmp, scan_tmp_bytes(cnt), st);
    if (rs != IM_OK) return rs;
    // copy stage -> members and sort each set ascending
    rs = segmented_sort_sets(pool->members, so, cnt, job.stage, r.stage_off, r.sort_tmp, g->n,
                             r.long_sets, st);
    if (rs != IM_OK) return rs;
    pool->theta += cnt;
    pool->total += r.added;
    pool->examined += r.examined;
    pool->sample_bytes += r.alg_bytes;
    IM_CUDA(cudaStreamSynchronize(st));
    return IM_OK;
}

}  // namespace im
