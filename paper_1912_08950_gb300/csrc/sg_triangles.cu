// Triangle enumeration over the degree-ordered orientation E+ and the
// Triangle p-x-Reduction kernels of Slim Graph (Sec. 4.3; Listing 1
// p-1-reduction and p-1-reduction-EO; x = 2; the min-count "CT" choice of
// Sec. 7).
//
// Enumeration.  Every triangle {u, v, w} with u < v < w in the degree order
// (d, id) is found exactly once, at the oriented arc u->v, as w in
// N+(u) ∩ N+(v) (the forward algorithm behind the O(m^{3/2}) bound the paper
// quotes).  The intersection streams the shorter of the two lists through a
// shared-memory hash table of the longer one: every vertex x stages N+(x) in
// a table once and streams (a) N+(v) for its out-arcs x->v with
// d+(v) <= d+(x) and (b) N+(u) for its in-arcs u->x with d+(u) < d+(x); the
// in-arcs of kind (b) come from the reverse list.  Each arc
// is handled once, at the end with the longer list, so the probes number
// sum over arcs of min(d+(u), d+(v)) -- under half of the plain forward
// algorithm's sum of d+(v) on power-law graphs.  Vertices with a short N+(x)
// and few in-arcs get one warp each; the others get a whole CTA whose warps
// split the arcs; those with an N+(x) longer than one CTA's table (when there
// are at least as many as SMs) go first, to a launch of 32-warp CTAs, one per
// SM, whose larger table holds their N+(x) whole.
//
// Decisions.  A hit (a triangle) is pushed to a per-warp queue; whenever 32
// hits are queued the warp decides all of them at once with full lanes:
// Philox4x32-10 on the sorted original ids (a, b, c) selects the triangle
// (r0 < floor(p 2^32)) and picks the edge to delete (r1, the heaviest edge, or
// the edge in the fewest triangles of G, counted by an earlier EdgeCount pass);
// the p-2 kernel deletes the two edges r1 does not pick.  Union kernels set the
// arc's deletion flag (a bit, idempotent); where it pays they do so in two passes
// that leave out triangles whose edges are all deleted (tri_union_kernel).  The
// Edge-Once kernel instead reserves each edge of every live selected triangle
// with a 64-bit atomicMin of (r2 << 32 | third vertex); an edge pass then
// accepts every triangle that holds all three of its reservations.  Accepted
// triangles are edge-disjoint, mark their edges considered, delete their
// chosen edge, and the rounds repeat until no selected triangle is live.
// This reproduces exactly the sequential scan of the selected triangles in
// increasing (r2, a, b, c) order (for two triangles sharing an edge, the
// lexicographic order of (a, b, c) equals the order of their third vertices).
#include <climits>
#include <cstring>

#include "sg_internal.cuh"

namespace sg {

constexpr uint32_t kEmpty = 0xFFFFFFFFu;
constexpr int kLightMax = 64;     // largest out-degree processed by one warp
constexpr int kLightItems = 256;  // ... with at most this many lists to stream
constexpr int kLightSlots = 256;  // hash slots per warp (>= 4 * kLightMax)
constexpr int kTW = 8;            // warps per CTA
constexpr int kHeavyCap = 1024;  // largest phase-1 table (entries; 26 KB of shared memory)
constexpr int kHubTW = 32;        // warps per CTA of the hub launch (one CTA per SM)
constexpr int kHubCap = 4096;     // largest hub table (entries; 104 KB of shared memory)
constexpr int kQ = 128;           // per-warp hit ring (<= 31 left over + 2 slabs of hits fit)
// the two union passes (tri_union_kernel):
constexpr int kWindow = 32;       // list elements streamed before an arc is looked at again
constexpr int kWhole = 1 << 29;        // blocks of the window of a list streamed whole
constexpr int kFilterLog = 4;          // log2 of the filter bits per table slot (four slots per entry)
constexpr int kFilterBits = 4 << kFilterLog;  // per entry
constexpr int kUnionLightMax = 128;    // largest out-degree processed by one warp
constexpr int kUnionLightItems = 512;  // ... with at most this many lists to stream
// lists up to this long are always streamed whole (see tri_union_kernel): 256 on
// graphs with a hub launch, where the second pass costs more (R-MAT s26 at p =
// 0.5: both passes 528 ms against 551 at 128; s23 equal), 128 on the others
// (s22: 19.2 ms against 22.3 at 256; 64 leaves a third more arc ends to pass 2)
constexpr int kShortList = 128, kShortListHubs = 256;
// the second pass has no light vertices: their lists must all be short
static_assert(kUnionLightMax <= kShortList, "a light vertex's lists are streamed whole in the first pass");
constexpr int kEoBuckets = 6;     // edge-once list buckets (rounds 0..5 of the prefix schedule)
// context workspaces of the edge-once rounds: the list and the two active lists
constexpr int kWsList = 0, kWsActive0 = 1, kWsActive1 = 2;

// Count: totals only.  EdgeCount / VertexCount: add every triangle to the
// counters of its three edges / vertices.  Union*: the union-semantics TR
// kernels (in one pass, or in the two of tri_union_kernel: two_passes_pay).
// EoReserve: one edge-once bidding pass.  EoEmit: lists the live selected
// triangles for the edge-once list rounds.  BatchUnion: union kernels over a
// batch of graphs.
enum class Mode { Count, EdgeCount, VertexCount, UnionRandom, UnionMaxw, UnionP2, UnionMinCount, EoReserve, EoEmit,
                  BatchUnion };
template <Mode M>
constexpr bool kUnion = M == Mode::UnionRandom || M == Mode::UnionMaxw || M == Mode::UnionP2 ||
                        M == Mode::UnionMinCount || M == Mode::BatchUnion;
// the edge-once passes skip arcs that are already considered
template <Mode M>
constexpr bool kEdgeOnce = M == Mode::EoReserve || M == Mode::EoEmit;
// the passes that decide their triangles (the others only count them)
template <Mode M>
constexpr bool kDecides = kUnion<M> || kEdgeOnce<M>;

// Edge-once "considered" flags: one bit per oriented arc (m/8 bytes, so the
// flags stay in L2 while the triangle lists stream past them).
__device__ __forceinline__ bool considered_bit(const uint32_t *c, int64_t e) {
    return (__ldg(c + (e >> 5)) >> (e & 31)) & 1u;
}
__device__ __forceinline__ void set_considered(uint32_t *c, int64_t e) { atomicOr(c + (e >> 5), 1u << (e & 31)); }

// Deletion flags: one bit per oriented arc.  They only ever change from 0 to 1
// during a pass, so a stale read is a flag not seen yet.
__device__ __forceinline__ void delete_arc(uint32_t *del, uint32_t e) { atomicOr(del + (e >> 5), 1u << (e & 31)); }
__device__ __forceinline__ bool arc_deleted(const uint32_t *del, uint32_t e) {
    uint32_t w;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(w) : "l"(del + (e >> 5)) : "memory");
    return (w >> (e & 31)) & 1u;
}

// The same through the L1, where a line may have been there since before.
__device__ __forceinline__ bool arc_deleted_cached(const uint32_t *del, uint32_t e) {
    uint32_t w;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(w) : "l"(del + (e >> 5)));
    return (w >> (e & 31)) & 1u;
}

struct TriArgs {
    const int64_t *offp;
    const uint32_t *colp;
    const int64_t *offs;          // symmetric offsets: in-arcs of x live at inl[offs(x) - offp(x) ...]
    const uint32_t *din;          // in-arcs u->x with d+(u) < d+(x), per x
    const uint2 *inl;             // (u, arc u->x) of those in-arcs
    const float *wp;
    int64_t n;
    uint32_t k0, k1;
    unsigned long long tp;
    uint32_t *del;                // deletion flags, one bit per oriented arc
    bool look_first;              // one union pass: look at an arc's flag before setting it
    uint32_t dead_flag;           // two union passes: a bit no arc index uses (kArcDead), or 0
    const uint32_t *considered;  // edge-once flag bits (see considered_bit)
    unsigned long long *resv;
    uint32_t *tcnt;               // triangles of G through each arc of E+ (EdgeCount adds, min-count reads)
    unsigned long long *vcnt;     // triangles through each vertex (VertexCount adds)
    unsigned long long eo_theta;  // edge-once: only triangles with r2 < eo_theta bid this round
    unsigned long long *ctr;
    const uint32_t *heavy;
    int64_t n_heavy;
    int heavy_cap;               // entries of the phase-1 table; larger N+(u) go in chunks
    int light_max;               // out-degrees up to this go to the warp-per-vertex phase
    int light_claim;             // vertices a warp claims at a time in the light phase (at most 32)
    int short_max;               // two union passes: lists up to this long are always streamed whole
    const uint4 *arec;           // two union passes: off+, d+, and for the second first live arc, live arcs
    const uint2 *alive;
    int light_items;             // ... when they also have at most this many arcs to stream
    int *err;                    // device error word (a cuckoo stash overflow)
    unsigned long long *work;    // [0] next heavy vertex, [1] next light vertex block
    const unsigned long long *n_heavy_dev;  // if set, the heavy count is read on the device
    // batched union: per-graph parameters and the graph of every vertex
    const BatchParam *bparams;
    const uint32_t *vgid;
    // edge-once: list of the live selected triangles (EoEmit), split into
    // buckets by the round in which each first bids
    uint4 *list;
    unsigned long long *list_ctr;  // [kEoBuckets] slots handed out per bucket
    unsigned long long *list_dem;  // [kEoBuckets] triangles that belong in each bucket, listed or not
    unsigned long long list_base[kEoBuckets], list_cap[kEoBuckets];
    int eo_round;                  // this enumeration's round: earlier buckets fold into it
    int eo_shift;                  // list claims are halved this often (eo_chunk)
    int eo_hi;                     // buckets from this one on are not listed (counted only)
    int *list_overflow;            // bit b: bucket b ran out of room
};

// One live selected triangle of an active list: sorted original ids
// x0 < x1 < x2, its draws r1 (edge choice) and r2 (edge-once order), and the
// oriented arcs joining (x0,x1), (x0,x2), (x1,x2).  x0 == kSentinel marks an
// unused slot.  The enumeration writes the smaller record (a, e_ab, e_ac,
// e_bc) instead -- a < b < c in the degree order, so b and c are the heads of
// e_ab and e_ac -- and a triangle is expanded when it first bids.
struct __align__(16) TriRec {
    uint32_t x0, x1, x2, r1;
    uint32_t r2, e01, e02, e12;
};
constexpr uint32_t kSentinel = 0xFFFFFFFFu;

// Bucket b of the list holds the triangles whose r2 lies in
// [2^(26+b), 2^(27+b)) (bucket 0: r2 < 2^27), i.e. those that first bid in
// edge-once round b of the doubling prefix schedule.
__device__ __forceinline__ int eo_bucket(uint32_t r2) { return r2 < (1u << 27) ? 0 : (31 - __clz((int)r2)) - 26; }
// list slots a warp claims at a time, in proportion to the bucket's share: 2048
// over the buckets, halved `shift` times on graphs that fill less (to 32 each
// at least, a group's most), as what a warp leaves of a claim is read back as
// sentinels
__host__ __device__ constexpr int eo_chunk(int b, int shift) {
    return (b <= 1 ? 64 : (32 << b)) >> shift > 32 ? (b <= 1 ? 64 : (32 << b)) >> shift : 32;
}

// Per-warp list writer: per bucket it claims chunks of slots, fills them in
// order and seals the unused tail of a chunk with sentinels.  The cursors
// live in registers spread over the lanes: lane b holds the next free slot of
// bucket b, lane 8 + b the end of its chunk and lane 16 + b how many
// triangles belong in bucket b.  Buckets from hi on are counted but not
// written: those the caller left out, and any that ran out of room (the
// lower buckets stay complete, so the caller can still use them).
struct Emitter {
    unsigned long long cur = 0;  // this lane's cursor or count (see above)
    int hi = 0;                  // warp-uniform
};

__device__ __forceinline__ void emit_seal(const TriArgs &a, unsigned long long cur, unsigned long long end) {
    const int lane = threadIdx.x & 31;
    for (unsigned long long i = cur + lane; i < end; i += 32) a.list[i].x = kSentinel;
}

__device__ __forceinline__ void emit_push(const TriArgs &a, Emitter &em, bool want, const uint4 &rec, uint32_t r2) {
    const int lane = threadIdx.x & 31;
    const int mb = want ? max(eo_bucket(r2), min(a.eo_round, kEoBuckets - 1)) : -1;
    if (!__any_sync(kFull, want)) return;
    // lanes of my bucket, and (in lanes b and 16 + b) the count of bucket b
    unsigned mine = 0, cnt_b = 0;
#pragma unroll
    for (int b = 0; b < kEoBuckets; ++b) {
        const unsigned bm = __ballot_sync(kFull, mb == b);
        if (mb == b) mine = bm;
        if ((lane & 15) == b) cnt_b = (unsigned)__popc(bm);
    }
    if (lane >= 16) em.cur += cnt_b;  // zero outside lanes 16 .. 16 + kEoBuckets - 1
    // a bucket whose chunk is too short for this group claims a new chunk (rare)
    const unsigned long long end_b = __shfl_down_sync(kFull, em.cur, 8);  // lane b: end of bucket b
    unsigned need = __ballot_sync(kFull, lane < em.hi && end_b - em.cur < cnt_b);
    while (need) {
        const int b = __ffs(need) - 1;
        need &= need - 1;
        const unsigned long long cur = __shfl_sync(kFull, em.cur, b);
        const unsigned long long end = __shfl_sync(kFull, em.cur, 8 + b);
        emit_seal(a, cur, end);
        const unsigned long long chunk = (unsigned long long)eo_chunk(b, a.eo_shift);
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(a.list_ctr + b, chunk);
        base = __shfl_sync(kFull, base, 0);
        if (base + chunk > a.list_cap[b]) {
            // out of room: bucket b and the ones above it are no longer written
            if (lane == 0) atomicOr(a.list_overflow, 1 << b);
            em.hi = b;
            break;
        }
        if (lane == b) em.cur = a.list_base[b] + base;
        if (lane == 8 + b) em.cur = a.list_base[b] + base + chunk;
    }
    const unsigned long long cur = __shfl_sync(kFull, em.cur, mb < 0 ? 0 : mb);
    if (want && mb < em.hi) a.list[cur + __popc(mine & lanemask_lt())] = rec;
    if (lane < em.hi) em.cur += cnt_b;
}

// Per-warp ring of found triangles, waiting to be decided 32 at a time.  The
// table vertex u is the same for every entry (the ring is flushed before the
// warp moves to another table) and w is the head of the arc iuw, so an entry
// keeps v and the three arcs.  Oriented arcs are addressed with 32-bit
// indices (E+ holds fewer than 2^32 arcs).
struct HitQueue {
    uint32_t v[kQ], iuv[kQ], iuw[kQ], ivw[kQ];
};
struct QState {
    int head = 0, n = 0;
};

__device__ __forceinline__ uint32_t slot_of(uint32_t key, int log_slots) {
    return (key * 0x9E3779B1u) >> (32 - log_slots);
}

__device__ __forceinline__ int ceil_log2(int x) { return x <= 1 ? 0 : 32 - __clz(x - 1); }
template <typename T>
__device__ __forceinline__ void swap2(T &a, T &b) {
    const T t = a;
    a = b;
    b = t;
}

// The edge in the fewest triangles of G under (count, lo, hi).  The arcs are
// passed in the order (x0,x1), (x0,x2), (x1,x2) of the sorted endpoints, which
// is also their (lo, hi) order, so a tie keeps the earlier arc.
template <typename I>
__device__ __forceinline__ I mincount_arc(const uint32_t *tcnt, I e01, I e02, I e12) {
    const uint32_t c01 = __ldg(tcnt + e01), c02 = __ldg(tcnt + e02), c12 = __ldg(tcnt + e12);
    I best = e01;
    uint32_t bc = c01;
    if (c02 < bc) { best = e02; bc = c02; }
    if (c12 < bc) best = e12;
    return best;
}

// sort the vertices of a triangle, keeping e_ij = the arc joining x_i and x_j
__device__ __forceinline__ void sort_triangle(uint32_t &x0, uint32_t &x1, uint32_t &x2, uint32_t &e01, uint32_t &e02,
                                              uint32_t &e12) {
    if (x0 > x1) { swap2(x0, x1); swap2(e02, e12); }
    if (x1 > x2) { swap2(x1, x2); swap2(e01, e02); }
    if (x0 > x1) { swap2(x0, x1); swap2(e02, e12); }
}

// the heaviest of a sorted triangle's edges under (weight, lo, hi)
__device__ __forceinline__ uint32_t maxw_arc(const float *wp, uint32_t e01, uint32_t e02, uint32_t e12) {
    const float w01 = __ldg(wp + e01), w02 = __ldg(wp + e02), w12 = __ldg(wp + e12);
    // (x0, x1) < (x0, x2) < (x1, x2): of equal weights the later edge
    uint32_t best = e01;
    float bw = w01;
    if (w02 >= bw) { best = e02; bw = w02; }
    if (w12 >= bw) best = e12;
    return best;
}

// One triangle (u, v, w) with its three oriented arcs under a union kernel:
// selection, and kill(arc) for what it deletes.
template <Mode M, class Kill>
__device__ __forceinline__ void decide_union(const TriArgs &a, uint32_t u, uint32_t v, uint32_t w, uint32_t iuv,
                                             uint32_t iuw, uint32_t ivw, const Kill &kill) {
    uint32_t x0 = u, x1 = v, x2 = w, e01 = iuv, e02 = iuw, e12 = ivw;
    uint32_t k0 = a.k0, k1 = a.k1;
    unsigned long long tp = a.tp;
    bool maxw = M == Mode::UnionMaxw, p2 = M == Mode::UnionP2;
    if constexpr (M == Mode::BatchUnion) {
        // the triangle's graph: its own seed, p and kernel, local ids as keys
        const BatchParam &P = a.bparams[__ldg(a.vgid + u)];
        const uint32_t base = (uint32_t)P.vbase;
        x0 -= base;
        x1 -= base;
        x2 -= base;
        k0 = P.k0;
        k1 = P.k1;
        tp = P.tp;
        maxw = P.kernel == (int)SG_TR_MAXW;
        p2 = P.kernel == (int)SG_TR_P2;
    }
    sort_triangle(x0, x1, x2, e01, e02, e12);
    const uint4 r = philox4x32_10(make_uint4(x0, x1, x2, kTagTri), k0, k1);
    if ((unsigned long long)r.x >= tp) return;  // not selected
    uint32_t best;
    if constexpr (M == Mode::UnionMinCount) {
        best = mincount_arc(a.tcnt, e01, e02, e12);
    } else if (maxw) {
        best = maxw_arc(a.wp, e01, e02, e12);
    } else {
        const int k = (int)(((unsigned long long)r.y * 3ull) >> 32);
        if (p2) {  // x = 2: the drawn edge stays, the other two go
            if (k != 0) kill(e01);
            if (k != 1) kill(e02);
            if (k != 2) kill(e12);
            return;
        }
        best = k == 0 ? e01 : (k == 1 ? e02 : e12);
    }
    kill(best);
}

// One triangle under a one-pass union or an edge-once pass: deletion, or
// selection and bid or listing.  Warp-collective (the list writer uses
// ballots); lanes without a triangle pass valid = false.
template <Mode M>
__device__ __forceinline__ void decide(const TriArgs &a, bool valid, uint32_t u, uint32_t v, uint32_t w,
                                       uint32_t iuv, uint32_t iuw, uint32_t ivw, unsigned &live, Emitter &em,
                                       uint32_t head_uv = 0) {
    static_assert(kDecides<M>, "the counting passes decide nothing");
    if constexpr (kUnion<M>) {
        if (valid)
            decide_union<M>(a, u, v, w, iuv, iuw, ivw, [&](uint32_t e) {
                if (!a.look_first || !arc_deleted_cached(a.del, e)) delete_arc(a.del, e);
            });
    } else {
        bool emit = false;
        uint4 rec = make_uint4(0u, 0u, 0u, 0u);
        uint32_t rec_r2 = 0;
        if (valid) {
            uint32_t x0 = u, x1 = v, x2 = w;
            uint32_t e01 = iuv, e02 = iuw, e12 = ivw;
            sort_triangle(x0, x1, x2, e01, e02, e12);
            const uint4 r = philox4x32_10(make_uint4(x0, x1, x2, kTagTri), a.k0, a.k1);
            // the triangle is selected, and none of its edges is considered
            if ((unsigned long long)r.x < a.tp &&
                (a.considered == nullptr || !(considered_bit(a.considered, e01) | considered_bit(a.considered, e02) |
                                              considered_bit(a.considered, e12)))) {
                // the round's prefix of the (r2, a, b, c) order bids for its edges
                // (the listing pass too, in case the list overflows)
                if ((unsigned long long)r.z < a.eo_theta) {
                    const unsigned long long hi = (unsigned long long)r.z << 32;
                    atomicMin(a.resv + e01, hi | x2);
                    atomicMin(a.resv + e02, hi | x1);
                    atomicMin(a.resv + e12, hi | x0);
                }
                ++live;
                if constexpr (M == Mode::EoEmit) {  // list the live selected triangle
                    emit = true;
                    rec_r2 = r.z;
                    // w is last in the degree order; of u and v the head of iuv is the later one
                    const bool u_first = head_uv == v;
                    rec = make_uint4(u_first ? u : v, iuv, u_first ? iuw : ivw, u_first ? ivw : iuw);
                }
            }
        }
        if constexpr (M == Mode::EoEmit) emit_push(a, em, emit, rec, rec_r2);
    }
}

// Decide the 32 oldest queued triangles with all lanes.
template <Mode M>
__device__ __forceinline__ void drain32(const TriArgs &a, const HitQueue &q, int head, uint32_t u,
                                             unsigned &live, Emitter &em) {
    const int k = (head + (threadIdx.x & 31)) & (kQ - 1);
    const uint32_t iuw = q.iuw[k];
    const uint32_t iuv = q.iuv[k];
    // the listing pass needs the head of u-v too: load it with w, before the draw
    const uint32_t huv = M == Mode::EoEmit ? __ldg(a.colp + iuv) : 0u;
    decide<M>(a, true, u, q.v[k], __ldg(a.colp + iuw), iuv, iuw, q.ivw[k], live, em, huv);
    __syncwarp();
}
// Decide everything queued for the table vertex u (the last group with idle lanes).
template <Mode M>
__device__ __forceinline__ void flush_hits(const TriArgs &a, const HitQueue &q, QState &qs, uint32_t u,
                                           unsigned &live, Emitter &em) {
    if constexpr (kDecides<M>) {
        const int lane = threadIdx.x & 31;
        while (qs.n >= 32) {
            drain32<M>(a, q, qs.head, u, live, em);
            qs.head = (qs.head + 32) & (kQ - 1);
            qs.n -= 32;
        }
        const bool valid = lane < qs.n;
        const int k = (qs.head + lane) & (kQ - 1);
        const uint32_t iuw = valid ? q.iuw[k] : 0u;
        const uint32_t iuv = valid ? q.iuv[k] : 0u;
        const uint32_t huv = (M == Mode::EoEmit && valid) ? __ldg(a.colp + iuv) : 0u;
        decide<M>(a, valid, u, valid ? q.v[k] : 0u, valid ? __ldg(a.colp + iuw) : 0u, iuv, iuw,
                  valid ? q.ivw[k] : 0u, live, em, huv);
        __syncwarp();
    }
    qs.head = 0;
    qs.n = 0;
}

// Shared-memory cuckoo table of N+(u) (Pagh & Rodler's cuckoo hashing; the
// concurrent exchange-based insertion follows Alcantara et al.'s GPU tables):
// every key lives in one of two slots, so a lookup reads exactly two slots
// with no probe loop and no divergence.  Load <= 1/4.  An insertion that
// keeps displacing keys for kCuckooIters exchanges leaves its homeless entry
// in a small stash that lookups then scan; a full stash raises a device error.
//
// A table of 2^L slots puts key w in slot h_j(w) = (w * K_j) >> (32 - L),
// j = 1 or 2.  The slot's 32-bit word keeps the low 32 - L bits of w * K_j
// (the slot number holds the high L bits, and multiplying by an odd K_j is a
// bijection, so word and slot give w back), which hash placed it, and w's
// position in N+(u) (< 2^(L-2) at load 1/4):
//   bits [L, 32): low bits of w * K_j;  bit L-1: j - 1;  bit L-2: 0;  bits [0, L-2): position
// An empty slot is all ones (bit L-2 set), so it matches no key, and since
// the word and slot pin down w, kEmpty (past a list's end) matches none either.
constexpr uint32_t kSlotEmpty = 0xFFFFFFFFu;
constexpr uint32_t kH1 = 0x9E3779B1u, kH2 = 0x85EBCA77u;
// inverse of an odd k modulo 2^32 (Newton's iteration doubles the correct low bits)
constexpr uint32_t inv_mod32(uint32_t k) {
    uint32_t x = k;  // k * k == 1 mod 8
    for (int i = 0; i < 5; ++i) x *= 2u - k * x;
    return x;
}
constexpr uint32_t kH1Inv = inv_mod32(kH1), kH2Inv = inv_mod32(kH2);
static_assert(kH1 * kH1Inv == 1u && kH2 * kH2Inv == 1u, "hash multipliers must be invertible");
// a stash entry is (vertex << 32 | position); this marks "not in the stash"
constexpr unsigned long long kStashNone = 0xFFFFFFFEFFFFFFFFull;
constexpr int kCuckooIters = 32;
constexpr int kStash = 16;

struct Table {
    uint32_t *slot;
    unsigned long long *stash;
    int *stash_n;
    uint32_t *dead = nullptr;    // two union passes: deletion flags of the table's arcs, by position,
    uint32_t *filter = nullptr;  // and one bit per hash of kFilterBits per entry
};

__device__ __forceinline__ void table_insert(const Table &t, int log_slots, uint32_t w, int i, int *err) {
    const int L = log_slots, sh = 32 - L;
    const uint32_t pmask = (1u << (L - 2)) - 1u;
    uint32_t x = w * kH1;
    uint32_t pos = x >> sh;
    uint32_t cur = (x << L) | (uint32_t)i;
    for (int it = 0; it < kCuckooIters; ++it) {
        const uint32_t old = atomicExch(t.slot + pos, cur);
        if (old == kSlotEmpty) return;
        // the evicted key moves to its other slot
        const bool by2 = (old >> (L - 1)) & 1u;
        const uint32_t wo = ((pos << sh) | (old >> L)) * (by2 ? kH2Inv : kH1Inv);
        x = wo * (by2 ? kH1 : kH2);
        pos = x >> sh;
        cur = (x << L) | ((by2 ? 0u : 1u) << (L - 1)) | (old & pmask);
    }
    const bool by2 = (cur >> (L - 1)) & 1u;
    const uint32_t wo = ((pos << sh) | (cur >> L)) * (by2 ? kH2Inv : kH1Inv);
    const int s = atomicAdd(t.stash_n, 1);
    if (s < kStash) t.stash[s] = ((unsigned long long)wo << 32) | (cur & pmask);
    else atomicExch(err, (int)kDevTableFull);
}

// w in the table's two slots?  t receives its position in N+(u).
__device__ __forceinline__ bool table_find(const Table &tb, int sh, uint32_t w, uint32_t &t) {
    const int L = 32 - sh;
    const uint32_t lim = 1u << (L - 2);
    const uint32_t x1 = w * kH1, x2 = w * kH2;
    const uint32_t a = tb.slot[x1 >> sh];
    const uint32_t b = tb.slot[x2 >> sh];
    const bool ha = (a ^ (x1 << L)) < lim;
    const bool hb = (b ^ ((x2 << L) | (lim << 1))) < lim;
    t = (ha ? a : b) & (lim - 1u);
    return ha | hb;
}

// w in the stash (the rare table whose insertion left keys there)?  Returns
// the stash entry (vertex << 32 | position), or kStashNone.
__device__ __noinline__ unsigned long long stash_find(const unsigned long long *stash, int stash_n, uint32_t w) {
    for (int k = 0; k < stash_n; ++k) {
        const unsigned long long c = stash[k];
        if ((uint32_t)(c >> 32) == w) return c;
    }
    return kStashNone;
}

// First two 32-element slabs of the list colp[ov, ov + dv) (kEmpty past its end).
__device__ __forceinline__ void first_slabs(const TriArgs &a, uint32_t ov, int dv, uint32_t &na, uint32_t &nb) {
    const int lane = threadIdx.x & 31;
    na = lane < dv ? __ldg(a.colp + ov + lane) : kEmpty;
    nb = lane + 32 < dv ? __ldg(a.colp + ov + lane + 32) : kEmpty;
}

// Stream N+(v) = colp[ov, ov + dv) through the table of N+(u): two 32-element
// slabs per iteration, the next two loaded while these are probed.  The
// caller passes the first two slabs (na, nb) already loaded, so that it can
// issue them before finishing the previous list.  Hits go to the queue.
template <Mode M>
__device__ __forceinline__ void probe_list(const TriArgs &a, const Table &tb, int log_slots, int stash_n,
                                           uint32_t u, uint32_t iuv, uint32_t ou, uint32_t v, uint32_t ov, int dv,
                                           uint32_t na, uint32_t nb, HitQueue &q, QState &qs, unsigned &live,
                                           unsigned long long &tris, Emitter &em) {
    const int lane = threadIdx.x & 31;
    const uint32_t lt = lanemask_lt();
    const uint32_t *lst = a.colp + ov;
    const int sh = 32 - log_slots;
    unsigned huv = 0;  // EdgeCount: triangles found on the arc u->v
    for (int j0 = 0; j0 < dv; j0 += 64) {
        const int ja = j0 + lane, jb = ja + 32;
        const uint32_t wa = na, wb = nb;
        uint32_t ta = 0, tb2 = 0;
        // the next two slabs are in flight while these are probed
        na = kEmpty;
        nb = kEmpty;
        if (ja + 64 < dv) na = __ldg(lst + ja + 64);
        if (jb + 64 < dv) nb = __ldg(lst + jb + 64);
        // kEmpty is never a vertex, so out-of-range lanes miss
        bool ha = table_find(tb, sh, wa, ta);
        bool hb = table_find(tb, sh, wb, tb2);
        if (stash_n != 0) {  // warp-uniform and rare
            if (!ha) {
                const unsigned long long c = stash_find(tb.stash, stash_n, wa);
                ha = c != kStashNone;
                ta = (uint32_t)c;
            }
            if (!hb) {
                const unsigned long long c = stash_find(tb.stash, stash_n, wb);
                hb = c != kStashNone;
                tb2 = (uint32_t)c;
            }
        }
        const unsigned ma = __ballot_sync(kFull, ha), mb = __ballot_sync(kFull, hb);
        if constexpr (M == Mode::EdgeCount) {
            // each hit closes a triangle through u->w and v->w; u->v is summed once
            if (ha) { atomicAdd(a.tcnt + ou + ta, 1u); atomicAdd(a.tcnt + ov + (uint32_t)ja, 1u); }
            if (hb) { atomicAdd(a.tcnt + ou + tb2, 1u); atomicAdd(a.tcnt + ov + (uint32_t)jb, 1u); }
            huv += (unsigned)(__popc(ma) + __popc(mb));
            continue;
        }
        if constexpr (M == Mode::VertexCount) {
            // each hit is a triangle through w; u and v are summed once per list
            if (ha) atomicAdd(a.vcnt + wa, 1ull);
            if (hb) atomicAdd(a.vcnt + wb, 1ull);
            huv += (unsigned)(__popc(ma) + __popc(mb));
            continue;
        }
        if constexpr (M == Mode::Count) {
            if (lane == 0) tris += (unsigned)(__popc(ma) + __popc(mb));
            continue;
        }
        if constexpr (kDecides<M>) {
            if ((ma | mb) == 0) continue;
            const int pa = __popc(ma), pb = __popc(mb);
            const int tail = qs.head + qs.n;
            if (ha) {
                const int s0 = (tail + __popc(ma & lt)) & (kQ - 1);
                q.v[s0] = v; q.iuv[s0] = iuv; q.iuw[s0] = ou + ta; q.ivw[s0] = ov + (uint32_t)ja;
            }
            if (hb) {
                const int s0 = (tail + pa + __popc(mb & lt)) & (kQ - 1);
                q.v[s0] = v; q.iuv[s0] = iuv; q.iuw[s0] = ou + tb2; q.ivw[s0] = ov + (uint32_t)jb;
            }
            qs.n += pa + pb;
            if (lane == 0) tris += (unsigned)(pa + pb);
            __syncwarp();
            while (qs.n >= 32) {
                drain32<M>(a, q, qs.head, u, live, em);
                qs.head = (qs.head + 32) & (kQ - 1);
                qs.n -= 32;
            }
        }
    }
    if constexpr (M == Mode::EdgeCount) {
        if (lane == 0 && huv) {
            atomicAdd(a.tcnt + iuv, huv);
            tris += huv;
        }
    }
    if constexpr (M == Mode::VertexCount) {
        if (lane == 0 && huv) {
            atomicAdd(a.vcnt + u, (unsigned long long)huv);
            atomicAdd(a.vcnt + v, (unsigned long long)huv);
            tris += huv;
        }
    }
}

// Stream the in-lists [first, first + cnt) (cnt <= 32) of the table vertex u:
// the lanes load the arcs' records and list bounds in parallel, then the warp
// streams the lists one by one.
template <Mode M>
__device__ __forceinline__ void stream_in_group(const TriArgs &a, const Table &tb, int log_slots, int stash_n,
                                                uint32_t u, int du, uint32_t tbase, int64_t ib, int first, int cnt,
                                                HitQueue &q, QState &qs, unsigned &live, unsigned long long &probes,
                                                unsigned long long &tris, Emitter &em, bool count_probes) {
    const int lane = threadIdx.x & 31;
    uint32_t sv = 0, so = 0, se = 0;
    int sd = 0;
    if (lane < cnt) {
        const uint2 it = __ldg(a.inl + ib + first + lane);
        sv = it.x;
        se = it.y;
        const int64_t b0 = __ldg(a.offp + sv);
        so = (uint32_t)b0;
        // an in-arc v->u whose tail has d+(v) >= d+(u) is streamed from v's side
        const int dvv = (int)(__ldg(a.offp + sv + 1) - b0);
        sd = (dvv >= du || (kEdgeOnce<M> && a.considered != nullptr && considered_bit(a.considered, se))) ? 0 : dvv;
    }
    // the next list's first slabs load while the current one is probed
    uint32_t pa, pb;
    first_slabs(a, __shfl_sync(kFull, so, 0), __shfl_sync(kFull, sd, 0), pa, pb);
    for (int i = 0; i < cnt; ++i) {
        const uint32_t v = __shfl_sync(kFull, sv, i);
        const uint32_t ov = __shfl_sync(kFull, so, i);
        const uint32_t e = __shfl_sync(kFull, se, i);
        const int dv = __shfl_sync(kFull, sd, i);
        const uint32_t ca = pa, cb = pb;
        if (i + 1 < cnt) first_slabs(a, __shfl_sync(kFull, so, i + 1), __shfl_sync(kFull, sd, i + 1), pa, pb);
        if (lane == 0 && count_probes) probes += (unsigned)dv;
        probe_list<M>(a, tb, log_slots, stash_n, u, e, tbase, v, ov, dv, ca, cb, q, qs, live, tris, em);
    }
}

// Find the triangles on up to 32 arcs of a light table vertex u: its out-arcs
// [first, first + cnt) or entries of its in-list.  The lists are short (a few to
// 64 elements), so they are streamed as one sequence, a slab of 32 elements at a
// time: a lane finds its element's arc from the arcs that start inside the
// slab.  Counting: the first lane of an arc's run adds the run's hits to the
// arc's counters; otherwise the hits go to the queue.
//
// Bound by latency and idle lanes when a list is streamed at a time, 64 lanes
// wide, each waiting for the loads of the one before; against that, in ms:
// triangles per vertex of a geometric graph (2^20 vertices, 25 M edges, lists of
// 17 elements) 5.18 -> 2.15, of R-MAT s20, where most elements are in heavy
// vertices' lists, 9.33 -> 8.98; the edge-once listing pass at p = 0.5 on the
// geometric graph 7.90 -> 4.22, Chung-Lu 2^20 5.88 -> 4.99, R-MAT s21 23.1 ->
// 22.3; a union call at p = 0.5 on the geometric graph 7.74 -> 4.84.
// Returns the hits (all lanes).  arc: 32 entries of the warp's scratch.
template <Mode M>
__device__ __forceinline__ unsigned light_group(const TriArgs &a, const Table &tb, int sh, int stash_n, uint32_t u,
                                                int d, uint32_t ou, bool out, int64_t first, int cnt, uint4 *arc,
                                                HitQueue &q, QState &qs, unsigned &live, unsigned long long &probes,
                                                Emitter &em) {
    const int lane = threadIdx.x & 31;
    uint32_t sv = 0, se = 0, sp = 0;
    int sl = 0;
    if (lane < cnt) {
        if (out) {
            se = (uint32_t)first + lane;
            sv = __ldg(a.colp + se);
        } else {
            const uint2 it = __ldg(a.inl + first + lane);
            sv = it.x;
            se = it.y;
        }
        const int64_t b0 = __ldg(a.offp + sv);
        const int dv = (int)(__ldg(a.offp + sv + 1) - b0);
        sp = (uint32_t)b0;
        if (out ? dv <= d : dv < d) sl = dv;  // else streamed from the other end
        // a considered arc closes no live triangle
        if (kEdgeOnce<M> && a.considered != nullptr && considered_bit(a.considered, se)) sl = 0;
    }
    probes += (unsigned)sl;
    int inc = sl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += x;
    }
    const int total = __shfl_sync(kFull, inc, 31);
    const int start = sl > 0 ? inc - sl : INT_MIN;
    const unsigned wanted = __ballot_sync(kFull, sl > 0);
    if (sl > 0) arc[__popc(wanted & lanemask_lt())] = make_uint4(sv, se, sp - (uint32_t)start, 0u);
    __syncwarp();
    const uint32_t lt = lanemask_lt(), le = lt | (1u << lane);
    int before = -1;  // arcs that start before the slab, minus one
    unsigned hits = 0, nstarts = 0;
    int nk = 0;
    uint32_t nw = kEmpty, narc = 0;
    auto load = [&](int s) {
        const unsigned rel = (unsigned)start - (unsigned)s;
        nstarts = __reduce_or_sync(kFull, rel < 32u ? 1u << rel : 0u);
        nk = before + __popc(nstarts & le);
        before += __popc(nstarts);
        nw = kEmpty;
        if (s + lane < total) {
            narc = arc[nk].z + (uint32_t)(s + lane);
            nw = __ldg(a.colp + narc);
        }
    };
    if (total > 0) load(0);
    for (int s = 0; s < total; s += 32) {
        const uint32_t w = nw, ivw = narc;
        const unsigned starts = nstarts;
        const int k = nk;
        if (s + 32 < total) load(s + 32);  // the next slab's, while this one is probed
        uint32_t t = 0;
        bool h = table_find(tb, sh, w, t);
        if (stash_n != 0 && !h && w != kEmpty) {  // rare
            const unsigned long long c = stash_find(tb.stash, stash_n, w);
            h = c != kStashNone;
            t = (uint32_t)c;
        }
        const unsigned m = __ballot_sync(kFull, h);
        if (m == 0) continue;
        hits += (unsigned)__popc(m);
        if constexpr (M == Mode::Count) continue;
        if constexpr (kDecides<M>) {
            if (h) {
                const int s0 = (qs.head + qs.n + __popc(m & lt)) & (kQ - 1);
                const uint4 c = arc[k];
                q.v[s0] = c.x; q.iuv[s0] = c.y; q.iuw[s0] = ou + t; q.ivw[s0] = ivw;
            }
            qs.n += __popc(m);
            __syncwarp();
            if (qs.n >= 32) {  // fewer than 32 are left after each slab
                drain32<M>(a, q, qs.head, u, live, em);
                qs.head = (qs.head + 32) & (kQ - 1);
                qs.n -= 32;
            }
            continue;
        }
        // hits on this lane's arc, if its run starts here
        const unsigned later = starts & ~le;
        const unsigned run = (later ? (1u << (__ffs(later) - 1)) - 1u : kFull) & ~lt;
        const unsigned c = (lane == 0 || ((starts >> lane) & 1u)) ? (unsigned)__popc(m & run) : 0u;
        if constexpr (M == Mode::EdgeCount) {
            if (h) {
                atomicAdd(a.tcnt + ou + t, 1u);
                atomicAdd(a.tcnt + ivw, 1u);
            }
            if (c) atomicAdd(a.tcnt + arc[k].y, c);
        } else {
            if (h) atomicAdd(a.vcnt + w, 1ull);
            if (c) atomicAdd(a.vcnt + arc[k].x, (unsigned long long)c);
        }
    }
    __syncwarp();  // the entries are read before the next group writes them
    return hits;
}

template <Mode M>
__device__ __forceinline__ void finish(const TriArgs &a, unsigned live, unsigned long long probes,
                                       unsigned long long tris, Emitter &em) {
    if constexpr (M == Mode::EoEmit) {
        for (int b = 0; b < em.hi; ++b)
            emit_seal(a, __shfl_sync(kFull, em.cur, b), __shfl_sync(kFull, em.cur, 8 + b));
        const int lane = threadIdx.x & 31;
        if (lane >= 16 && lane < 16 + kEoBuckets && em.cur != 0) atomicAdd(a.list_dem + (lane - 16), em.cur);
    }
    const unsigned long long P = warp_sum(probes), T = warp_sum(tris);
    const unsigned L = warp_sum(live);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(a.ctr + kCtrProbes, P);
        atomicAdd(a.ctr + kCtrTriangles, T);
        if (L) atomicAdd(a.ctr + kCtrLive, (unsigned long long)L);
    }
}

// One persistent launch per enumeration pass.
// Phase 1: heavy vertices (large N+(u) or many lists to stream), largest work
// bound first; a CTA stages N+(u) in a shared-memory table (plus every
// out-neighbour's list bounds) and its warps claim out-arcs one at a time and
// in-arcs 32 at a time.  Phase 2: light vertices, a warp per vertex with its
// own small table; warps claim 32 vertex ids at a time.  Probe and triangle
// totals are counted per list and per found triangle.  The counting passes
// run 5 CTAs per SM at 48 registers; the passes that decide triangles keep 64
// (4 CTAs per SM): at 48 their queue drain and record assembly spill.
//
// The hub launch (TW = kHubTW) runs phase 1 alone, before the main launch,
// over the vertices whose N+(u) is too long for the main launch's table: one
// CTA of 32 warps per SM shares a table of up to kHubCap entries, so those
// lists are streamed once instead of once per table chunk.
template <Mode M>
constexpr int kEnumCtasPerSm = kDecides<M> ? 4 : 5;

template <Mode M, int TW>
__global__ void __launch_bounds__(TW * 32, TW == kTW ? kEnumCtasPerSm<M> : 1) tri_enum_kernel(TriArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_next;
    __shared__ long long s_h;
    __shared__ int s_stash_n[TW + 1];
    __shared__ unsigned long long s_stash[TW + 1][kStash];
    HitQueue *qs = reinterpret_cast<HitQueue *>(smem);
    unsigned char *tbl = smem + sizeof(HitQueue) * TW;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    HitQueue &q = qs[warp];
    QState qst;
    unsigned live = 0;
    unsigned long long probes = 0, tris = 0;
    Emitter em;
    em.hi = a.eo_hi;
    const int64_t n_heavy = a.n_heavy_dev ? (int64_t)*a.n_heavy_dev : a.n_heavy;

    // ---- phase 1: heavy vertices
    {
        const int cap = a.heavy_cap;  // table capacity: larger N+(u) is processed in chunks
        const int slots = 4 * cap;
        Table tb{reinterpret_cast<uint32_t *>(tbl), s_stash[TW], &s_stash_n[TW]};
        uint32_t *vv = tb.slot + slots;  // v, off+(v), d+(v) of N+(u)
        uint32_t *vo = vv + cap;
        unsigned short *vd = reinterpret_cast<unsigned short *>(vo + cap);  // d+(v) <= d+(u) <= cap, else 0
        for (;;) {
            if (threadIdx.x == 0) s_h = (long long)atomicAdd(a.work, 1ull);
            __syncthreads();
            const int64_t h = s_h;
            if (h >= n_heavy) break;
            const uint32_t u = __ldg(a.heavy + h);
            const uint32_t ou = (uint32_t)__ldg(a.offp + u);
            const int d = (int)(__ldg(a.offp + u + 1) - (int64_t)ou);
            const int nin = (int)__ldg(a.din + u);
            const int items = d + (nin + 31) / 32;                    // out-arcs, then groups of 32 in-arcs
            const int64_t ib = __ldg(a.offs + u) - (int64_t)ou;       // start of u's in-arcs in inl
            const bool staged = d <= cap;  // list bounds of N+(u) kept in shared memory
            for (int c0 = 0; c0 < d; c0 += cap) {
                const int cn = min(cap, d - c0);
                const int log_slots = ceil_log2(4 * cn) < 3 ? 3 : ceil_log2(4 * cn);
                for (int s2 = threadIdx.x; s2 < (1 << log_slots); s2 += blockDim.x) tb.slot[s2] = kSlotEmpty;
                if (threadIdx.x == 0) {
                    s_next = 0;
                    *tb.stash_n = 0;
                }
                __syncthreads();
                for (int k = threadIdx.x; k < cn; k += blockDim.x) {
                    const int i = c0 + k;
                    const uint32_t v = __ldg(a.colp + ou + i);
                    const bool dead = kEdgeOnce<M> && a.considered != nullptr &&
                                      considered_bit(a.considered, (int64_t)ou + i);
                    if (staged) {
                        const int64_t ov = __ldg(a.offp + v);
                        const int dv = (int)(__ldg(a.offp + v + 1) - ov);
                        vv[i] = v;
                        vo[i] = (uint32_t)ov;
                        // a considered arc u->v closes no live triangle; an arc
                        // with d+(v) > d+(u) is streamed from v's side
                        vd[i] = (unsigned short)((dead || dv > d) ? 0 : dv);
                    }
                    if (!dead) table_insert(tb, log_slots, v, k, a.err);
                }
                __syncthreads();
                const int stash_n = min(*tb.stash_n, kStash);
                for (;;) {
                    int i = 0;
                    if (lane == 0) i = atomicAdd(&s_next, 1);
                    i = __shfl_sync(kFull, i, 0);
                    if (i >= items) break;
                    {  // hand out the in-arc groups (the larger units) first, then the out-arcs
                        const int ng = items - d;
                        i = i < ng ? d + i : i - ng;
                    }
                    if (i >= d) {  // 32 in-arcs v->u with d+(v) < d+(u): stream each N+(v)
                        const int g0 = (i - d) * 32;
                        stream_in_group<M>(a, tb, log_slots, stash_n, u, d, ou + (uint32_t)c0, ib, g0,
                                           min(32, nin - g0), q, qst, live, probes, tris, em, c0 == 0);
                        continue;
                    }
                    // out-arc u->v: stream N+(v)
                    const uint32_t e = ou + (uint32_t)i;
                    uint32_t v, ov;
                    int dv;
                    if (staged) {
                        v = vv[i];
                        ov = vo[i];
                        dv = vd[i];
                    } else {
                        v = __ldg(a.colp + e);
                        const int64_t o64 = __ldg(a.offp + v);
                        ov = (uint32_t)o64;
                        dv = (int)(__ldg(a.offp + v + 1) - o64);
                        if (dv > d || (kEdgeOnce<M> && a.considered != nullptr && considered_bit(a.considered, e))) dv = 0;
                    }
                    // algorithmic probes: a chunked N+(u) re-reads the lists, which is not counted
                    if (lane == 0 && c0 == 0) probes += (unsigned)dv;
                    uint32_t ca, cb;
                    first_slabs(a, ov, dv, ca, cb);
                    probe_list<M>(a, tb, log_slots, stash_n, u, e, ou + (uint32_t)c0, v, ov, dv, ca, cb, q, qst,
                                  live, tris, em);
                }
                __syncthreads();  // the table is rebuilt for the next chunk or vertex
            }
            flush_hits<M>(a, q, qst, u, live, em);
        }
    }

    // ---- phase 2: light vertices
    if constexpr (TW == kTW) {
        Table tb{reinterpret_cast<uint32_t *>(tbl) + warp * kLightSlots, s_stash[warp], &s_stash_n[warp]};
        uint4 *arc = reinterpret_cast<uint4 *>(tbl + sizeof(uint32_t) * kLightSlots * TW) + warp * 32;
        for (;;) {
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(a.work + 1, (unsigned long long)a.light_claim);
            base = __shfl_sync(kFull, base, 0);
            if ((int64_t)base >= a.n) break;
            const int64_t ul = (int64_t)base + lane;
            uint32_t oul = 0;
            int dl = 0, nl = 0;
            if (lane < a.light_claim && ul < a.n) {
                const int64_t o0 = __ldg(a.offp + ul);
                oul = (uint32_t)o0;
                dl = (int)(__ldg(a.offp + ul + 1) - o0);
                nl = (int)__ldg(a.din + ul);
            }
            // d+(u) < 2 closes no triangle at u (and then u has no in-arcs to stream)
            unsigned lm = __ballot_sync(kFull, dl >= 2 && dl <= a.light_max && dl + nl <= a.light_items);
            while (lm) {
                const int src = __ffs(lm) - 1;
                lm &= lm - 1;
                const uint32_t u = (uint32_t)(base + src);
                const uint32_t ou = __shfl_sync(kFull, oul, src);
                const int d = __shfl_sync(kFull, dl, src);
                const int nin = __shfl_sync(kFull, nl, src);
                const int log_slots = max(3, ceil_log2(4 * d));
                for (int s2 = lane; s2 < (1 << log_slots); s2 += 32) tb.slot[s2] = kSlotEmpty;
                if (lane == 0) *tb.stash_n = 0;
                __syncwarp();
                for (int k = lane; k < d; k += 32) {
                    // the arc u->w may close a live triangle
                    if (!kEdgeOnce<M> || a.considered == nullptr || !considered_bit(a.considered, (int64_t)ou + k))
                        table_insert(tb, log_slots, __ldg(a.colp + ou + k), k, a.err);
                }
                __syncwarp();
                const int stash_n = min(*tb.stash_n, kStash);
                unsigned hits = 0;
                for (int c = 0; c < d; c += 32)
                    hits += light_group<M>(a, tb, 32 - log_slots, stash_n, u, d, ou, true, (int64_t)ou + c,
                                           min(32, d - c), arc, q, qst, live, probes, em);
                // in-arcs v->u with d+(v) < d+(u)
                const int64_t ib = nin > 0 ? __ldg(a.offs + u) - (int64_t)ou : 0;
                for (int c = 0; c < nin; c += 32)
                    hits += light_group<M>(a, tb, 32 - log_slots, stash_n, u, d, ou, false, ib + c, min(32, nin - c),
                                           arc, q, qst, live, probes, em);
                if (lane == 0) {
                    tris += hits;
                    if (M == Mode::VertexCount && hits) atomicAdd(a.vcnt + u, (unsigned long long)hits);
                }
                flush_hits<M>(a, q, qst, u, live, em);
                __syncwarp();
            }
        }
    }
    finish<M>(a, live, probes, tris, em);
}

// ------------------------------------------------------------ union passes
// The union kernels delete, for every selected triangle, the edge (or edges)
// its draw names, and deletions accumulate.  So a triangle whose three edges
// are already deleted need not be decided, and an arc whose edge is already
// deleted need not be streamed for triangles whose other two edges are deleted
// too.  Most edges die early: on R-MAT s22 at p = 0.5 an edge lies in 99
// triangles on average and each deletes it with probability 1/6.  Two passes
// use that and give the same flags as deciding every triangle:
//
//   first pass (kAlive = false)   every arc u->v streams the shorter list
//     through the table of the longer one as the counting passes do, but only
//     until its own edge is deleted: windows of 1, 2, 4, ... blocks of kWindow
//     elements, from a start spread over the list, between which the edge's
//     flag is looked at.  A list of at most short_max elements (kShortList) is
//     always streamed whole.  At the end a live arc has been streamed whole; a
//     long list not streamed whole belongs to a deleted arc.
//   second pass (kAlive = true)   for the deleted arcs u->v with two lists
//     longer than short_max, the triangles {u, v, w} that still matter have
//     u->w or v->w live after the first pass: the live arcs of v (compacted by
//     alive_build) stream through the table of N+(u) and the live arcs of u
//     through that of N+(v); where those together are no shorter than the
//     shorter list, that list streams whole instead.
//
// Bound by instruction issue (69% of the slots at s23, the integer pipe at
// 47%, DRAM at 19%): about half of the instructions are the list elements
// (mapping, filter, queue), a fifth the claims and windows, a fifth the
// decisions.  R-MAT at p = 0.5, elements streamed and triangles decided against
// all of them, and the enumeration's time before (one pass that decides every
// triangle) and now: s22 0.35 and 0.14, 41.8 -> 19.2 ms; s26 0.32 and 0.09,
// 1094 -> 525 ms.  Max-weight on a Chung-Lu graph of 2^21 vertices at p = 1,
// where light edges never die: 0.69 and 0.35, 11.5 -> 8.3 ms.

// The table vertex a warp works on.
struct TabCtx {
    Table tb;
    int sh;                 // 32 - log2(slots)
    int fsh;                // 32 - log2(filter bits)
    int stash_n;
    uint32_t u, tbase, cn;  // vertex, arc of table position 0, entries
    int d;                  // d+(u)
};

// A warp's scratch: the ring of list elements that may close a triangle --
// (v, arc u-v, w, arc v->w), one 16-byte store and load each -- the arcs whose
// lists it is streaming, (v, arc u-v, list start minus the elements before it,
// flags), and the arcs waiting for a free lane, (v, arc u-v, list start, length
// and flags).
constexpr int kPool = 64;
struct UnionScratch {
    uint4 ring[kQ];
    uint4 arc[32];
    uint4 pool[kPool];
};
// flags, beside the length in the pool: the arc's list is the live arcs of v;
// the arc was deleted before its list streamed (kept in the ring entry's arc
// v->w, when arc indices leave the bit free: TriArgs::dead_flag)
constexpr uint32_t kArcLive = 1u << 30, kArcDead = 1u << 31;
constexpr int kLenMask = (1 << 30) - 1;

// The table's filter: 2^L * kFilterBits / 4 bits, w's at the high bits of w *
// kH1.  Most list elements are in no triangle (R-MAT: 85-90%), and one
// shared-memory word and a bit test drop nearly all of them where the two
// cuckoo lookups take twice the instructions; what passes (the hits and about
// 1 / kFilterBits of the others) is looked up 32 at a time when it is decided.
__device__ __forceinline__ uint32_t filter_bit(const TabCtx &t, uint32_t w) { return (w * kH1) >> t.fsh; }
__device__ __forceinline__ bool filter_pass(const TabCtx &t, uint32_t w) {
    const uint32_t f = filter_bit(t, w);
    return (t.tb.filter[f >> 5] >> (f & 31)) & 1u;
}

// Look the oldest `cnt` (<= 32) queued elements up and decide the triangles
// they close that still have a live edge.
template <Mode M>
__device__ __forceinline__ void drain_union(const TriArgs &a, const TabCtx &t, const UnionScratch &q, int head, int cnt,
                                            unsigned long long &tris) {
    const int lane = threadIdx.x & 31;
    bool hit = false;
    if (lane < cnt) {
        const uint4 h = q.ring[(head + lane) & (kQ - 1)];  // v, arc u-v, w, arc v->w
        uint32_t k = 0;
        hit = table_find(t.tb, t.sh, h.z, k);
        if (t.stash_n != 0 && !hit) {  // rare
            const unsigned long long c = stash_find(t.tb.stash, t.stash_n, h.z);
            hit = c != kStashNone;
            k = (uint32_t)c;
        }
        // on an arc that was deleted before its list streamed, a triangle
        // matters while one of its other edges lives
        const uint32_t vw = h.w & ~a.dead_flag;
        if (hit && (h.w & a.dead_flag) && ((t.tb.dead[k >> 5] >> (k & 31)) & 1u)) hit = !arc_deleted(a.del, vw);
        if (hit)
            decide_union<M>(a, t.u, h.x, h.z, h.y, t.tbase + k, vw, [&](uint32_t e) {
                delete_arc(a.del, e);
                const uint32_t r = e - t.tbase;  // an arc of the table: its flag in shared memory too
                if (r < t.cn) atomicOr(t.tb.dead + (r >> 5), 1u << (r & 31));
            });
    }
    const unsigned m = __ballot_sync(kFull, hit);
    if (lane == 0) tris += (unsigned)__popc(m);
}

template <Mode M>
__device__ __forceinline__ void flush_union(const TriArgs &a, const TabCtx &t, const UnionScratch &q, QState &qs,
                                            unsigned long long &tris) {
    while (qs.n > 0) {
        drain_union<M>(a, t, q, qs.head, min(qs.n, 32), tris);
        qs.head = (qs.head + 32) & (kQ - 1);
        qs.n -= 32;
    }
    qs.head = 0;
    qs.n = 0;
}

// A list element: w (kEmpty: none), the arc v->w and the entry of v's arc in
// the scratch.
struct Elem {
    uint32_t w, arc;
    int k;
};

// Filter two list elements per lane, queue what passes, and decide what a full
// group has gathered.
template <Mode M>
__device__ __forceinline__ void probe_union(const TriArgs &a, const TabCtx &t, const Elem &x, const Elem &y,
                                            UnionScratch &q, QState &qs, unsigned long long &tris) {
    const bool hx = x.w != kEmpty && filter_pass(t, x.w);
    const bool hy = y.w != kEmpty && filter_pass(t, y.w);
    const unsigned mx = __ballot_sync(kFull, hx), my = __ballot_sync(kFull, hy);
    if (mx | my) {
        const uint32_t lt = lanemask_lt();
        const int px = __popc(mx);
        const int tail = qs.head + qs.n;
        if (hx) {
            const uint4 e = q.arc[x.k];
            q.ring[(tail + __popc(mx & lt)) & (kQ - 1)] = make_uint4(e.x, e.y, x.w, x.arc | (e.w & a.dead_flag));
        }
        if (hy) {
            const uint4 e = q.arc[y.k];
            q.ring[(tail + px + __popc(my & lt)) & (kQ - 1)] = make_uint4(e.x, e.y, y.w, y.arc | (e.w & a.dead_flag));
        }
        qs.n += px + __popc(my);
        __syncwarp();
        while (qs.n >= 32) {
            drain_union<M>(a, t, q, qs.head, 32, tris);
            qs.head = (qs.head + 32) & (kQ - 1);
            qs.n -= 32;
        }
    }
}

// Stream the wanted lists of the lanes' arcs (lane: sl elements from sp; none
// if 0) as one sequence of elements, 64 at a time: the lists are short (a
// window of 32, about ten live arcs), and a list at a time would leave most
// lanes idle.  A lane finds its element's arc from the arcs that start inside
// its slab of 32 (an OR over the lanes).
template <Mode M, bool kAlive>
__device__ __forceinline__ void stream_lists(const TriArgs &a, const TabCtx &t, uint32_t sv, uint32_t se, uint32_t sp,
                                             int sl, uint32_t flags, UnionScratch &q, QState &qs,
                                             unsigned long long &probes, unsigned long long &tris, bool count) {
    const int lane = threadIdx.x & 31;
    // number the elements consecutively
    int inc = sl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += x;
    }
    const int total = __shfl_sync(kFull, inc, 31);
    const int start = sl > 0 ? inc - sl : INT_MIN;
    const unsigned wanted = __ballot_sync(kFull, sl > 0);
    if (sl > 0) q.arc[__popc(wanted & lanemask_lt())] = make_uint4(sv, se, sp - (uint32_t)start, flags);
    __syncwarp();
    const uint32_t le = lanemask_lt() | (1u << lane);
    int before = -1;  // arcs that start before the slab, minus one
    auto element = [&](int s) {
        Elem x{kEmpty, 0u, 0};
        const unsigned rel = (unsigned)start - (unsigned)s;
        const unsigned starts = __reduce_or_sync(kFull, rel < 32u ? 1u << rel : 0u);
        x.k = before + __popc(starts & le);
        before += __popc(starts);
        if (s + lane < total) {
            const uint4 r = q.arc[x.k];
            x.arc = r.z + (uint32_t)(s + lane);
            if (kAlive && (r.w & kArcLive)) {
                const uint2 l = __ldg(a.alive + x.arc);
                x.w = l.x;
                x.arc = l.y;
            } else {
                x.w = __ldg(a.colp + x.arc);
            }
        }
        return x;
    };
    if (count) probes += (unsigned)sl;
    Elem nx = element(0), ny = element(32);
    for (int s = 64;; s += 64) {
        const Elem x = nx, y = ny;
        if (s < total) {
            nx = element(s);
            ny = element(s + 32);
        }
        probe_union<M>(a, t, x, y, q, qs, tris);
        if (s >= total) break;
    }
    __syncwarp();  // the scratch's arcs are read before they are written again
}

// Stream the lists of the table vertex's arcs: item i < nin is entry ib + i of
// the in-lists, item nin + i the out-arc ou + i.  The warp claims 32 items at
// a time (from the CTA's counter `next`, or its own); the lanes load their
// records, flags and list bounds, and the arcs that this pass wants from this
// end (fewer than half of them) wait in the pool until a lane is free.  A lane
// holds one arc: in the first pass a live arc with a long list streams windows
// of 1, 2, 4, ... blocks of kWindow until its edge is deleted (a kill takes
// about 40 elements on R-MAT graphs) and its lane takes the next arc.  The
// records of one claim load while the windows stream, the ids of the next with
// them.
template <Mode M, bool kAlive>
__device__ __forceinline__ void stream_arcs(const TriArgs &a, const TabCtx &t, int *next, uint32_t ou, int64_t ib, int nin,
                                            int ax, UnionScratch &q, QState &qs, unsigned long long &probes,
                                            unsigned long long &tris, bool count) {
    const int lane = threadIdx.x & 31;
    const int items = nin + t.d;
    auto claim = [&]() {
        int i = 0;
        if (lane == 0) i = atomicAdd(next, 32);
        return __shfl_sync(kFull, i, 0);
    };
    auto load_ids = [&](int c, uint32_t &v, uint32_t &e) {
        const int i = c + lane;
        if (i < nin) {
            const uint2 it = __ldg(a.inl + ib + i);
            v = it.x;
            e = it.y;
        } else if (i < items) {
            e = ou + (uint32_t)(i - nin);
            v = __ldg(a.colp + e);
        }
    };
    int c = claim();  // the claim whose ids are loaded
    uint32_t rv = 0, re = 0;
    load_ids(c, rv, re);
    int phead = 0, pn = 0;            // the pool
    uint32_t sv = 0, se = 0, lst = 0; // the lane's arc: other end, arc, list start,
    int len = 0, b = 0, left = 0;     // list length, next block, blocks not streamed yet
    int w = 0;                        // blocks of the next window
    for (;;) {
        // records of the claimed items, ids of the next claim
        const int gc = pn <= kPool - 32 ? c : items;  // the pool has room for a whole claim
        const bool got = gc + lane < items;
        bool dead = false;
        uint4 rec = make_uint4(0u, 0u, 0u, 0u);  // off+, d+, first live arc, live arcs
        const uint32_t gv = rv, ge = re;
        if (got) {
            dead = arc_deleted(a.del, ge);
            if constexpr (kAlive) {
                rec = __ldg(a.arec + gv);
            } else {
                const uint2 r = __ldg(reinterpret_cast<const uint2 *>(a.arec + gv));
                rec.x = r.x;
                rec.y = r.y;
            }
        }
        if (gc < items) {
            c = claim();
            load_ids(c, rv, re);
        }
        // the windows of the lanes' arcs
        if (__any_sync(kFull, left > 0)) {
            const int n = len & kLenMask;
            const int nb = (n + kWindow - 1) / kWindow;
            const int k = min(min(w, left), nb - b);  // up to the list's end, where it wraps
            const int sl = left > 0 ? min(k * kWindow, n - b * kWindow) : 0;
            stream_lists<M, kAlive>(a, t, sv, se, lst + (uint32_t)(b * kWindow), sl, (uint32_t)len, q, qs,
                                    probes, tris, count);
            if (left > 0) {
                left -= k;
                b = b + k == nb ? 0 : b + k;
                w *= 2;
            }
            if constexpr (!kAlive) {
                if (__any_sync(kFull, left > 0)) {
                    if (c >= items && pn == 0) flush_union<M>(a, t, q, qs, tris);  // nothing else to stream meanwhile
                    if (left > 0 && arc_deleted(a.del, se)) left = 0;
                }
            }
        }
        // the claimed arcs to stream from this end: the longer list's
        if (gc < items) {
            uint32_t sp = rec.x;
            int sl = 0;
            if (got) {
                const int dv = (int)rec.y;
                const bool own = gc + lane >= nin ? dv <= t.d : dv < t.d;
                if constexpr (!kAlive) {
                    if (own && (!dead || dv <= a.short_max)) sl = dead && dv > 0 ? (int)((uint32_t)dv | kArcDead) : dv;
                } else if (dead && min(dv, t.d) > a.short_max) {
                    if ((int)rec.w + ax >= min(dv, t.d)) {
                        if (own) sl = (int)((uint32_t)dv | kArcDead);
                    } else if (rec.w != 0) {
                        sp = rec.z;
                        sl = (int)(rec.w | kArcLive | kArcDead);
                    }
                }
            }
            const unsigned m = __ballot_sync(kFull, sl != 0);
            if (sl != 0) q.pool[(phead + pn + __popc(m & lanemask_lt())) & (kPool - 1)] = make_uint4(gv, ge, sp, (uint32_t)sl);
            pn += __popc(m);
        }
        __syncwarp();
        // free lanes take waiting arcs
        const unsigned idle = __ballot_sync(kFull, left == 0);
        const int take = min(pn, __popc(idle));
        const int rank = __popc(idle & lanemask_lt());
        if (left == 0 && rank < take) {
            const uint4 r = q.pool[(phead + rank) & (kPool - 1)];
            sv = r.x;
            se = r.y;
            lst = r.z;
            len = (int)r.w;
            const int n1 = len & kLenMask;
            left = (n1 + kWindow - 1) / kWindow;
            b = 0;
            w = kWhole;
            if (!kAlive && n1 > a.short_max) {
                b = (int)__umulhi(se * 0x9E3779B1u, (uint32_t)left);  // a start spread over the list
                w = 1;
            }
        }
        phead = (phead + take) & (kPool - 1);
        pn -= take;
        __syncwarp();
        if (take == 0 && idle == kFull && c >= items) break;
    }
}

// One launch of a union pass: the heavy vertices a CTA each (largest work bound
// first; the warps claim groups of 32 arcs), then the light ones a warp each.
// Bound by instruction issue on the integer pipe, like the counting passes:
// four CTAs of 8 warps per SM at 64 registers (the drain is inlined).  The second
// pass also waits for random reads of records and live lists, and is faster at
// three CTAs with more registers: s22 3.14 -> 2.84 ms, s26 51.6 -> 46.4,
// max-weight on the Chung-Lu graph 1.54 -> 1.38; the first pass is slower at
// three (s22 16.4 -> 17.0, s26 248 -> 276) and at five (17.0, 253).
template <Mode M, int TW, bool kAlive>
__global__ void __launch_bounds__(TW * 32, TW == kTW ? (kAlive ? 3 : 4) : 1) tri_union_kernel(TriArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_next;
    __shared__ long long s_h;
    __shared__ int s_stash_n[TW + 1];
    __shared__ unsigned long long s_stash[TW + 1][kStash];
    __shared__ uint32_t s_dead[TW][kUnionLightMax / 32];
    __shared__ int s_lnext[TW];
    __shared__ int s_bad;
    unsigned char *tbl = smem + sizeof(UnionScratch) * TW;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    UnionScratch &q = reinterpret_cast<UnionScratch *>(smem)[warp];
    QState qst;
    unsigned long long probes = 0, tris = 0;
    if constexpr (kAlive) {  // live lists of a scan that gave up are not followed
        if (threadIdx.x == 0) s_bad = *(volatile int *)a.err;
        __syncthreads();
        if (s_bad != 0) return;
    }

    // ---- heavy vertices
    {
        const int cap = a.heavy_cap;  // table capacity: larger N+(u) is processed in chunks
        TabCtx t;
        t.tb = Table{reinterpret_cast<uint32_t *>(tbl), s_stash[TW], &s_stash_n[TW],
                     reinterpret_cast<uint32_t *>(tbl) + 4 * cap,
                     reinterpret_cast<uint32_t *>(tbl) + 4 * cap + (cap + 31) / 32};
        for (;;) {
            if (threadIdx.x == 0) s_h = (long long)atomicAdd(a.work, 1ull);
            __syncthreads();
            const int64_t h = s_h;
            if (h >= a.n_heavy) break;
            t.u = __ldg(a.heavy + h);
            const int64_t ou = __ldg(a.offp + t.u);
            t.d = (int)(__ldg(a.offp + t.u + 1) - ou);
            const int nin = (int)__ldg(a.din + t.u);
            const int64_t ib = __ldg(a.offs + t.u) - ou;             // start of u's in-arcs in inl
            int ax = 0;
            if constexpr (kAlive) {
                if (t.d <= a.short_max) {
                    __syncthreads();  // s_h is read before it is written again
                    continue;
                }
                ax = (int)__ldg(a.arec + t.u).w;
            }
            for (int c0 = 0; c0 < t.d; c0 += cap) {
                const int cn = min(cap, t.d - c0);
                const int log_slots = ceil_log2(4 * cn) < 3 ? 3 : ceil_log2(4 * cn);
                t.sh = 32 - log_slots;
                t.fsh = t.sh - kFilterLog;
                t.tbase = (uint32_t)(ou + c0);
                t.cn = (uint32_t)cn;
                for (int s2 = threadIdx.x; s2 < (1 << log_slots); s2 += blockDim.x) t.tb.slot[s2] = kSlotEmpty;
                for (int s2 = threadIdx.x; s2 < (1 << (log_slots + kFilterLog - 5)); s2 += blockDim.x) t.tb.filter[s2] = 0;
                if (threadIdx.x == 0) {
                    s_next = 0;
                    *t.tb.stash_n = 0;
                }
                __syncthreads();
                for (int k0 = warp * 32; k0 < cn; k0 += TW * 32) {
                    const int k = k0 + lane;
                    bool dead = false;
                    if (k < cn) {
                        const uint32_t w = __ldg(a.colp + t.tbase + k), f = filter_bit(t, w);
                        atomicOr(t.tb.filter + (f >> 5), 1u << (f & 31));
                        table_insert(t.tb, log_slots, w, k, a.err);
                        dead = arc_deleted(a.del, t.tbase + (uint32_t)k);
                    }
                    const unsigned dm = __ballot_sync(kFull, dead);
                    if (lane == 0) t.tb.dead[k0 >> 5] = dm;
                }
                __syncthreads();
                t.stash_n = min(*t.tb.stash_n, kStash);
                stream_arcs<M, kAlive>(a, t, &s_next, (uint32_t)ou, ib, nin, ax, q, qst, probes, tris, c0 == 0);
                flush_union<M>(a, t, q, qst, tris);
                __syncthreads();  // the table is rebuilt for the next chunk or vertex
            }
        }
    }

    // ---- light vertices
    if constexpr (TW == kTW && !kAlive) {
        TabCtx t;
        constexpr int kWords = 4 * kUnionLightMax + 4 * kUnionLightMax * kFilterBits / 4 / 32;  // slots, filter
        uint32_t *own = reinterpret_cast<uint32_t *>(tbl) + warp * kWords;
        t.tb = Table{own, s_stash[warp], &s_stash_n[warp], s_dead[warp], own + 4 * kUnionLightMax};
        for (;;) {
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(a.work + 1, (unsigned long long)a.light_claim);
            base = __shfl_sync(kFull, base, 0);
            if ((int64_t)base >= a.n) break;
            const int64_t ul = (int64_t)base + lane;
            uint32_t oul = 0;
            int dl = 0, nl = 0;
            if (lane < a.light_claim && ul < a.n) {
                const int64_t o0 = __ldg(a.offp + ul);
                oul = (uint32_t)o0;
                dl = (int)(__ldg(a.offp + ul + 1) - o0);
                nl = (int)__ldg(a.din + ul);
            }
            // d+(u) < 2 closes no triangle at u (and then u has no in-arcs to stream)
            unsigned lm = __ballot_sync(kFull, dl >= 2 && dl <= a.light_max && dl + nl <= a.light_items);
            while (lm) {
                const int src = __ffs(lm) - 1;
                lm &= lm - 1;
                t.u = (uint32_t)(base + src);
                t.tbase = __shfl_sync(kFull, oul, src);
                t.d = __shfl_sync(kFull, dl, src);
                t.cn = (uint32_t)t.d;
                const int nin = __shfl_sync(kFull, nl, src);
                const int log_slots = max(3, ceil_log2(4 * t.d));
                t.sh = 32 - log_slots;
                t.fsh = t.sh - kFilterLog;
                for (int s2 = lane; s2 < (1 << log_slots); s2 += 32) t.tb.slot[s2] = kSlotEmpty;
                for (int s2 = lane; s2 < (1 << (log_slots + kFilterLog - 5)); s2 += 32) t.tb.filter[s2] = 0;
                if (lane == 0) {
                    *t.tb.stash_n = 0;
                    s_lnext[warp] = 0;
                }
                __syncwarp();
                for (int k0 = 0; k0 < t.d; k0 += 32) {
                    const int k = k0 + lane;
                    bool dead = false;
                    if (k < t.d) {
                        const uint32_t w = __ldg(a.colp + t.tbase + k), f = filter_bit(t, w);
                        atomicOr(t.tb.filter + (f >> 5), 1u << (f & 31));
                        table_insert(t.tb, log_slots, w, k, a.err);
                        dead = arc_deleted(a.del, t.tbase + (uint32_t)k);
                    }
                    const unsigned dm = __ballot_sync(kFull, dead);
                    if (lane == 0) t.tb.dead[k0 >> 5] = dm;
                }
                __syncwarp();
                t.stash_n = min(*t.tb.stash_n, kStash);
                stream_arcs<M, false>(a, t, &s_lnext[warp], t.tbase, nin > 0 ? __ldg(a.offs + t.u) - (int64_t)t.tbase : 0,
                                      nin, 0, q, qst, probes, tris, true);
                flush_union<M>(a, t, q, qst, tris);
                __syncwarp();
            }
        }
    }
    const unsigned long long P = warp_sum(probes), T = warp_sum(tris);
    if (lane == 0) {
        atomicAdd(a.ctr + kCtrProbes, P);
        atomicAdd(a.ctr + kCtrTriangles, T);
    }
}

// Heavy vertices in decreasing out-degree order, by log2 buckets: pass 1
// counts the vertices of each bucket (and the maximum out-degree), pass 2
// scatters them so that larger buckets come first.
constexpr int kBuckets = 52;  // floor(log2) of the work bound d+ (d+ + in-arcs)
// sort keys: the bucket, plus kBuckets for a hub (d+ > hub_min), so hubs come first
constexpr int kKeys = 2 * kBuckets;

__device__ __forceinline__ int bucket_of(unsigned long long d) { return 63 - __clzll(d); }

// A vertex goes to the CTA phase when its table or its arc count is too large
// for one warp; the bucket orders those vertices by the bound d+(x) * (d+(x) +
// in-arcs(x)) on the probes made there (every streamed list is at most d+(x)).
__device__ __forceinline__ bool is_heavy(int64_t d, int64_t nin, int light_max, int light_items) {
    return d >= 2 && (d > light_max || d + nin > light_items);
}
__device__ __forceinline__ int heavy_bucket(int64_t d, int64_t nin) {
    return min(bucket_of((unsigned long long)d * (unsigned long long)(d + nin)), kBuckets - 1);
}
__device__ __forceinline__ int heavy_key(int64_t d, int64_t nin, int64_t hub_min) {
    return heavy_bucket(d, nin) + (d > hub_min ? kBuckets : 0);
}

// Also writes every vertex's in-degree d(u) - d+(u): the length of its
// in-list in the reverse list (see Oriented::inl).  With bucket_cnt2, also
// counts the split of the two union passes (kUnionLightMax).
__global__ void classify_count_kernel(const int64_t *__restrict__ offp, const int64_t *__restrict__ offs,
                                      uint32_t *din, int64_t n, int light_max, int light_items, int64_t hub_min,
                                      unsigned long long *bucket_cnt, unsigned long long *bucket_cnt2,
                                      unsigned long long *ctr) {
    __shared__ unsigned int s_cnt[kKeys], s_cnt2[kKeys];
    static_assert(kKeys <= 256, "a thread per key");
    if (threadIdx.x < kKeys) s_cnt[threadIdx.x] = s_cnt2[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long dmax = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += stride) {
        const int64_t d = offp[u + 1] - offp[u];
        dmax = d > (int64_t)dmax ? (unsigned long long)d : dmax;
        int64_t nin = (offs[u + 1] - offs[u]) - d;
        nin = nin < 0 ? 0 : nin;
        din[u] = (uint32_t)nin;
        if (is_heavy(d, nin, light_max, light_items)) atomicAdd(&s_cnt[heavy_key(d, nin, hub_min)], 1u);
        if (bucket_cnt2 && is_heavy(d, nin, kUnionLightMax, kUnionLightItems))
            atomicAdd(&s_cnt2[heavy_key(d, nin, hub_min)], 1u);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(kFull, dmax, o);
        dmax = t > dmax ? t : dmax;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(ctr + kCtrMaxDeg, dmax);
    __syncthreads();
    if (threadIdx.x < kKeys && s_cnt[threadIdx.x]) atomicAdd(bucket_cnt + threadIdx.x, (unsigned long long)s_cnt[threadIdx.x]);
    if (threadIdx.x < kKeys && s_cnt2[threadIdx.x])
        atomicAdd(bucket_cnt2 + threadIdx.x, (unsigned long long)s_cnt2[threadIdx.x]);
}

// Also writes the vertex records of two union passes (off+, d+, no live arcs yet), if asked to.

__global__ void classify_scatter_kernel(const int64_t *__restrict__ offp, const uint32_t *__restrict__ din,
                                        int64_t n, int light_max, int light_items, int64_t hub_min,
                                        const unsigned long long *__restrict__ bucket_cnt,
                                        unsigned long long *bucket_fill, uint32_t *heavy, uint4 *arec,
                                        unsigned long long *total_out) {
    __shared__ unsigned long long s_off[kKeys];
    if (threadIdx.x == 0) {
        unsigned long long run = 0;
        for (int b = kKeys - 1; b >= 0; --b) {
            s_off[b] = run;
            run += bucket_cnt[b];
        }
        if (blockIdx.x == 0 && total_out) *total_out = run;
    }
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += stride) {
        const int64_t d = offp[u + 1] - offp[u];
        const int64_t nin = din[u];
        if (arec) arec[u] = make_uint4((uint32_t)offp[u], (uint32_t)d, 0u, 0u);
        if (is_heavy(d, nin, light_max, light_items)) {
            const int b = heavy_key(d, nin, hub_min);
            heavy[s_off[b] + atomicAdd(bucket_fill + b, 1ull)] = (uint32_t)u;
        }
    }
}

// Edge-Once acceptance: an oriented arc e = u->y holding reservation
// (r2, z) belongs to the accepted triangle {u, y, z} iff that triangle also
// holds the reservations of its two other edges.
// returns -1 when the arc is missing (never for a symmetric CSR)
__device__ __forceinline__ int64_t arc_between(const int64_t *off, const int64_t *offp, const uint32_t *colp,
                                               uint32_t p, uint32_t q) {
    const int64_t dp = __ldg(off + p + 1) - __ldg(off + p);
    const int64_t dq = __ldg(off + q + 1) - __ldg(off + q);
    const bool pq = dp < dq || (dp == dq && p < q);
    const uint32_t row = pq ? p : q, key = pq ? q : p;
    const int64_t end = __ldg(offp + row + 1);
    const int64_t i = lower_bound_u32(colp, __ldg(offp + row), end, key);
    return (i < end && __ldg(colp + i) == key) ? i : -1;
}

// Which edge an accepted triangle deletes.
enum Choice { kChoiceRandom = 0, kChoiceMaxw = 1, kChoiceMinCount = 2 };

template <int CH>
__global__ void eo_accept_kernel(TriArgs a, const int64_t *__restrict__ off, uint32_t *considered) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t u = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp; u < a.n; u += nw) {
        const int64_t ou = __ldg(a.offp + u), d = __ldg(a.offp + u + 1) - ou;
        for (int64_t i = lane; i < d; i += 32) {
            const int64_t e = ou + i;
            const unsigned long long r = a.resv[e];
            if (r == ~0ull) continue;
            const uint32_t y = __ldg(a.colp + e);
            const uint32_t z = (uint32_t)r;
            const unsigned long long hi = r & 0xFFFFFFFF00000000ull;
            const int64_t f1 = arc_between(off, a.offp, a.colp, (uint32_t)u, z);
            const int64_t f2 = arc_between(off, a.offp, a.colp, y, z);
            if (f1 < 0 || f2 < 0) continue;
            if (a.resv[f1] != (hi | y) || a.resv[f2] != (hi | (uint32_t)u)) continue;
            set_considered(considered, e);
            // which edge of the accepted triangle goes
            uint32_t x0 = (uint32_t)u, x1 = y, x2 = z;
            int64_t e01 = e, e02 = f1, e12 = f2;
            if (x0 > x1) { swap2(x0, x1); swap2(e02, e12); }
            if (x1 > x2) { swap2(x1, x2); swap2(e01, e02); }
            if (x0 > x1) { swap2(x0, x1); swap2(e02, e12); }
            int64_t chosen;
            if constexpr (CH == kChoiceMinCount) {
                chosen = mincount_arc(a.tcnt, e01, e02, e12);
            } else if constexpr (CH == kChoiceMaxw) {
                chosen = maxw_arc(a.wp, (uint32_t)e01, (uint32_t)e02, (uint32_t)e12);
            } else {
                const uint4 rr = philox4x32_10(make_uint4(x0, x1, x2, kTagTri), a.k0, a.k1);
                const int k = (int)(((unsigned long long)rr.y * 3ull) >> 32);
                chosen = k == 0 ? e01 : (k == 1 ? e02 : e12);
            }
            if (chosen == e) delete_arc(a.del, (uint32_t)e);
        }
    }
}

// the edge that a listed triangle deletes when it is accepted
template <int CH>
__device__ __forceinline__ uint32_t chosen_arc(const TriRec &r, const float *wp, const uint32_t *tcnt) {
    if constexpr (CH == kChoiceMinCount) {
        return mincount_arc(tcnt, r.e01, r.e02, r.e12);
    } else if constexpr (CH == kChoiceMaxw) {
        return maxw_arc(wp, r.e01, r.e02, r.e12);
    } else {
        const int k = (int)(((unsigned long long)r.r1 * 3ull) >> 32);
        return k == 0 ? r.e01 : (k == 1 ? r.e02 : r.e12);
    }
}

// Edge-once rounds over the list of live selected triangles.
// Accept: a triangle holding the reservations of all three of its edges is
// accepted; accepted triangles are edge-disjoint, so their stores never race.
template <int CH>
__global__ void eo_list_accept_kernel(const TriRec *__restrict__ L, int64_t len,
                                      const unsigned long long *__restrict__ resv, uint32_t *considered,
                                      uint32_t *del, const float *__restrict__ wp, const uint32_t *__restrict__ tcnt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += stride) {
        const TriRec r = L[i];
        if (r.x0 == kSentinel) continue;
        const unsigned long long hi = (unsigned long long)r.r2 << 32;
        if (resv[r.e01] != (hi | r.x2) || resv[r.e02] != (hi | r.x1) || resv[r.e12] != (hi | r.x0)) continue;
        set_considered(considered, (int64_t)r.e01);
        set_considered(considered, (int64_t)r.e02);
        set_considered(considered, (int64_t)r.e12);
        delete_arc(del, chosen_arc<CH>(r, wp, tcnt));
    }
}

// Reserve: drop every triangle that lost an edge to an accepted one, reserve
// the edges of the survivors (64-bit atomicMin of (r2, third vertex)) and
// compact the survivors into `out` (block-aggregated appends).
__global__ void __launch_bounds__(256) eo_list_reserve_kernel(const TriRec *__restrict__ L, int64_t len,
                                                              TriRec *__restrict__ out,
                                                              unsigned long long *out_len,
                                                              unsigned long long *resv,
                                                              const uint32_t *__restrict__ considered,
                                                              unsigned long long theta) {
    __shared__ int s_cnt[8];
    __shared__ unsigned long long s_base;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < len; base += stride) {
        const int64_t i = base + threadIdx.x;
        bool keep = false;
        TriRec r{kSentinel, 0, 0, 0, 0, 0, 0, 0};
        if (i < len) {
            r = L[i];
            if (r.x0 != kSentinel && !(considered_bit(considered, r.e01) | considered_bit(considered, r.e02) |
                                       considered_bit(considered, r.e12))) {
                keep = true;
                if ((unsigned long long)r.r2 < theta) {
                    const unsigned long long hi = (unsigned long long)r.r2 << 32;
                    atomicMin(resv + r.e01, hi | r.x2);
                    atomicMin(resv + r.e02, hi | r.x1);
                    atomicMin(resv + r.e12, hi | r.x0);
                }
            }
        }
        const unsigned bm = __ballot_sync(kFull, keep);
        if (lane == 0) s_cnt[warp] = __popc(bm);
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int k = 0; k < 8; ++k) {
                const int c = s_cnt[k];
                s_cnt[k] = tot;
                tot += c;
            }
            s_base = tot ? atomicAdd(out_len, (unsigned long long)tot) : 0ull;
        }
        __syncthreads();
        if (keep) out[s_base + s_cnt[warp] + __popc(bm & lanemask_lt())] = r;
        __syncthreads();
    }
}

// Reserve for a bucket written by the enumeration: drop the triangles that
// lost an edge, expand the survivors to full records (vertices from the arc
// heads, draws recomputed), bid and append them to `out`.  Each thread takes
// kFreshPer records per pass (their loads overlap) and a CTA appends its
// survivors with one atomic per pass.
constexpr int kFreshPer = 4;

__global__ void __launch_bounds__(256) eo_fresh_reserve_kernel(const uint4 *__restrict__ F, int64_t len,
                                                               TriRec *__restrict__ out, unsigned long long *out_len,
                                                               unsigned long long *resv,
                                                               const uint32_t *__restrict__ considered,
                                                               unsigned long long theta,
                                                               const uint32_t *__restrict__ colp, uint32_t k0,
                                                               uint32_t k1) {
    __shared__ int s_cnt[8];
    __shared__ unsigned long long s_base;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t span = (int64_t)blockDim.x * kFreshPer;
    for (int64_t base = (int64_t)blockIdx.x * span; base < len; base += (int64_t)gridDim.x * span) {
        uint4 f[kFreshPer];
        bool keep[kFreshPer];
#pragma unroll
        for (int r = 0; r < kFreshPer; ++r) {
            const int64_t i = base + r * blockDim.x + threadIdx.x;
            f[r] = i < len ? __ldg(F + i) : make_uint4(kSentinel, 0u, 0u, 0u);
        }
#pragma unroll
        for (int r = 0; r < kFreshPer; ++r)
            keep[r] = f[r].x != kSentinel && !(considered_bit(considered, f[r].y) | considered_bit(considered, f[r].z) |
                                               considered_bit(considered, f[r].w));
        int cnt = 0;
#pragma unroll
        for (int r = 0; r < kFreshPer; ++r) cnt += keep[r];
        int inc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) s_cnt[warp] = inc;
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int k = 0; k < 8; ++k) {
                const int c = s_cnt[k];
                s_cnt[k] = tot;
                tot += c;
            }
            s_base = tot ? atomicAdd(out_len, (unsigned long long)tot) : 0ull;
        }
        __syncthreads();
        unsigned long long slot = s_base + s_cnt[warp] + (inc - cnt);
#pragma unroll
        for (int r = 0; r < kFreshPer; ++r) {
            if (!keep[r]) continue;
            uint32_t x0 = f[r].x, x1 = __ldg(colp + f[r].y), x2 = __ldg(colp + f[r].z);
            uint32_t e01 = f[r].y, e02 = f[r].z, e12 = f[r].w;
            if (x0 > x1) { swap2(x0, x1); swap2(e02, e12); }
            if (x1 > x2) { swap2(x1, x2); swap2(e01, e02); }
            if (x0 > x1) { swap2(x0, x1); swap2(e02, e12); }
            const uint4 d = philox4x32_10(make_uint4(x0, x1, x2, kTagTri), k0, k1);
            if ((unsigned long long)d.z < theta) {
                const unsigned long long hi = (unsigned long long)d.z << 32;
                atomicMin(resv + e01, hi | x2);
                atomicMin(resv + e02, hi | x1);
                atomicMin(resv + e12, hi | x0);
            }
            out[slot++] = TriRec{x0, x1, x2, d.y, d.z, e01, e02, e12};
        }
        __syncthreads();
    }
}

// Clear the reservations of the listed triangles' edges (cheaper than a full
// reset once the list is short): every reserved edge belongs to a listed triangle.
__global__ void eo_list_reset_kernel(const TriRec *__restrict__ L, int64_t len, unsigned long long *resv) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += stride) {
        const TriRec r = L[i];
        if (r.x0 == kSentinel) continue;
        resv[r.e01] = ~0ull;
        resv[r.e02] = ~0ull;
        resv[r.e12] = ~0ull;
    }
}

// --------------------------------------------- list rounds in one launch
// On a small list a round's kernels take a few microseconds each, and the host's
// part -- three to five launches, a copy and a wait per round -- is most of the
// time.  This kernel runs all rounds of the list that are left: per round it
// reserves (last round's survivors and the round's bucket), accepts and resets,
// with a barrier after each.  The grid is one thread-block cluster: its CTAs are
// scheduled together and meet at the hardware's cluster barrier, so nothing
// spins, whatever else runs on the device.  What other CTAs wrote is read past
// the L1.
struct EoRun {
    const uint4 *fresh;     // the bucketed list
    int64_t base[kEoBuckets], used[kEoBuckets];
    TriRec *active[2];      // this round's bidders are written to active[1] first
    int64_t len;            // survivors in active[0]
    int next_bucket, top, sched;
    unsigned long long *out_len;  // [2], zero
    unsigned long long *rounds;   // rounds run
    unsigned long long *resv;
    uint32_t *considered, *del;
    const uint32_t *colp, *tcnt;
    const float *wp;
    uint32_t k0, k1;
};
constexpr int kEoCta = 1024, kEoCluster = 16;
// List slots up to which the rounds left run in one launch.  Edge-once TR on
// R-MAT graphs, per call with launches per round / with this (2^20): 4096
// vertices at p = 0.5 740 / 640 us, 16,384 at p = 0.2 853 / 779 us, 65,536 at
// 0.2 1247 / 1153 us.  Sixteen CTAs are slow on more: at 2^21 65,536 vertices take
// 1370 us, at 2^22 1566 us; eight CTAs instead of sixteen: 3454 against 3386
// us on s18, whose last rounds run here.
constexpr int64_t kEoOneLaunch = 1 << 20;

__device__ __forceinline__ bool considered_now(const uint32_t *c, uint32_t e) { return (__ldcg(c + (e >> 5)) >> (e & 31)) & 1u; }

// All threads of the cluster arrive, with what they wrote, before any leaves.
// Not the .aligned form, which needs whole warps: the lanes come from loops of
// their own lengths, and nothing makes them meet again before this.
__device__ __forceinline__ void cluster_barrier() {
    __threadfence();
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// Append the CTA's survivors: this thread's slot in the list (all threads call).
__device__ __forceinline__ unsigned long long append_slot(bool keep, unsigned long long *len) {
    __shared__ int s_cnt[kEoCta / 32];
    __shared__ unsigned long long s_base;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(kFull, keep);
    if (lane == 0) s_cnt[warp] = __popc(m);
    __syncthreads();
    if (warp == 0) {
        const int c = s_cnt[lane];
        int inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += t;
        }
        s_cnt[lane] = inc - c;
        if (lane == 31) s_base = inc ? atomicAdd(len, (unsigned long long)inc) : 0ull;
    }
    __syncthreads();
    const unsigned long long slot = s_base + s_cnt[warp] + __popc(m & lanemask_lt());
    __syncthreads();
    return slot;
}

template <int CH>
__global__ void __cluster_dims__(kEoCluster, 1, 1) __launch_bounds__(kEoCta, 1) eo_rounds_kernel(EoRun g) {
    const int64_t stride = (int64_t)gridDim.x * kEoCta, t0 = (int64_t)blockIdx.x * kEoCta;
    int64_t len = g.len;
    int nb = g.next_bucket, cur = 0;
    auto bid = [&](const TriRec &r, unsigned long long theta) {
        if ((unsigned long long)r.r2 < theta) {
            const unsigned long long hi = (unsigned long long)r.r2 << 32;
            atomicMin(g.resv + r.e01, hi | r.x2);
            atomicMin(g.resv + r.e02, hi | r.x1);
            atomicMin(g.resv + r.e12, hi | r.x0);
        }
    };
    auto load = [](const TriRec *p) {
        const uint4 a = __ldcg(reinterpret_cast<const uint4 *>(p)), b = __ldcg(reinterpret_cast<const uint4 *>(p) + 1);
        return TriRec{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    };
    unsigned long long done = 0;
    for (int sched = g.sched;; ++sched) {
        unsigned long long theta = 1ull << (27 + min(sched, kEoBuckets - 1));
        if (g.top < kEoBuckets) theta = min(theta, 1ull << (26 + g.top));  // the list's window
        TriRec *in = g.active[cur], *out = g.active[cur ^ 1];
        unsigned long long *out_len = g.out_len + cur;
        // reserve: drop the triangles that lost an edge, bid for the others
        for (int64_t b = t0; b < len; b += stride) {
            const int64_t i = b + threadIdx.x;
            TriRec r{kSentinel, 0, 0, 0, 0, 0, 0, 0};
            if (i < len) r = load(in + i);
            const bool keep = i < len && !(considered_now(g.considered, r.e01) || considered_now(g.considered, r.e02) ||
                                           considered_now(g.considered, r.e12));
            if (keep) bid(r, theta);
            const unsigned long long slot = append_slot(keep, out_len);
            if (keep) out[slot] = r;
        }
        const int64_t fresh = nb < g.top ? g.used[nb] : 0;
        for (int64_t b = t0; b < fresh; b += stride) {
            const int64_t i = b + threadIdx.x;
            uint4 f = make_uint4(kSentinel, 0u, 0u, 0u);
            if (i < fresh) f = __ldg(g.fresh + g.base[nb] + i);
            const bool keep = f.x != kSentinel && !(considered_now(g.considered, f.y) || considered_now(g.considered, f.z) ||
                                                    considered_now(g.considered, f.w));
            TriRec r{kSentinel, 0, 0, 0, 0, 0, 0, 0};
            if (keep) {  // expand: vertices from the arc heads, the draw again
                r.x0 = f.x;
                r.x1 = __ldg(g.colp + f.y);
                r.x2 = __ldg(g.colp + f.z);
                r.e01 = f.y;
                r.e02 = f.z;
                r.e12 = f.w;
                sort_triangle(r.x0, r.x1, r.x2, r.e01, r.e02, r.e12);
                const uint4 d = philox4x32_10(make_uint4(r.x0, r.x1, r.x2, kTagTri), g.k0, g.k1);
                r.r1 = d.y;
                r.r2 = d.z;
                bid(r, theta);
            }
            const unsigned long long slot = append_slot(keep, out_len);
            if (keep) out[slot] = r;
        }
        if (nb < g.top) ++nb;
        cluster_barrier();
        len = (int64_t)__ldcg(out_len);
        if (len > 0) ++done;
        // accept: a triangle that holds all three of its reservations
        for (int64_t i = t0 + threadIdx.x; i < len; i += stride) {
            const TriRec r = load(out + i);
            const unsigned long long hi = (unsigned long long)r.r2 << 32;
            if (__ldcg(g.resv + r.e01) != (hi | r.x2) || __ldcg(g.resv + r.e02) != (hi | r.x1) ||
                __ldcg(g.resv + r.e12) != (hi | r.x0))
                continue;
            set_considered(g.considered, (int64_t)r.e01);
            set_considered(g.considered, (int64_t)r.e02);
            set_considered(g.considered, (int64_t)r.e12);
            delete_arc(g.del, chosen_arc<CH>(r, g.wp, g.tcnt));
        }
        if (len == 0 && nb >= g.top) break;
        cluster_barrier();
        for (int64_t i = t0 + threadIdx.x; i < len; i += stride) {
            const TriRec r = load(out + i);
            g.resv[r.e01] = ~0ull;
            g.resv[r.e02] = ~0ull;
            g.resv[r.e12] = ~0ull;
        }
        if (t0 == 0 && threadIdx.x == 0) g.out_len[cur ^ 1] = 0;
        cur ^= 1;
        cluster_barrier();
    }
    if (t0 == 0 && threadIdx.x == 0) *g.rounds = done;
}

// -------------------------------------------------------------------- host
struct Plan {
    uint32_t *heavy = nullptr;
    unsigned long long *buckets = nullptr;  // counts [kKeys], those of the two passes' split [kKeys], fills [kKeys]
    uint32_t *din = nullptr;                // in-arcs streamed from the head's side, per vertex
    bool two = false;                       // two union passes
    uint4 *arec = nullptr;                  // ... their vertex records,
    void *rec_own = nullptr;                // the records' allocation, if they have one,
    AliveArcs al;                           // and the live arcs between them
    uint2 *inl = nullptr;                   // their (tail, arc), at offs(v) - offp(v) per vertex
    const int64_t *offs = nullptr;          // symmetric offsets of the graph
    int64_t n_heavy = 0, max_deg = 0;
    int64_t work = 0;    // W = sum over arcs of min(d+(u), d+(v)): the probes of one pass
    int64_t n_hubs = 0;  // the first n_hubs heavy vertices (d+ > kHeavyCap) go to the hub launch
    int hub_cap = 0;     // hub table entries
    size_t hub_smem = 0;
    int light_max = kLightMax;
    int light_items = kLightItems;
    size_t smem = 0;
    int heavy_cap = 8;  // phase-1 table entries
    size_t usmem = 0, uhub_smem = 0;  // shared memory of the union passes' launches
};

static sg_status read_ctr(Ctx *c, int first, int count, unsigned long long *out) {
    SG_CUDA(cudaMemcpyAsync(c->h_pinned, c->d_ctr + first, sizeof(unsigned long long) * count,
                            cudaMemcpyDeviceToHost, c->stream));
    SG_CUDA(cudaStreamSynchronize(c->stream));
    std::memcpy(out, c->h_pinned, sizeof(unsigned long long) * count);
    return SG_OK;
}

static void free_plan(Ctx *c, Plan *pl) {
    dfree(c, pl->heavy);
    dfree(c, pl->buckets);
    dfree(c, pl->din);
    dfree(c, pl->rec_own);
    alive_free(c, &pl->al);
    pl->rec_own = nullptr;
    pl->arec = nullptr;
    pl->heavy = nullptr;
    pl->buckets = nullptr;
    pl->din = nullptr;
    pl->inl = nullptr;
}


// a union table of `cap` entries: four slots each, one deletion flag bit, the filter
static size_t union_table_bytes(int cap) {
    return (size_t)cap * 4 * sizeof(uint32_t) + (size_t)(cap + 31) / 32 * 4 + (size_t)cap * kFilterBits / 8;
}

// A union call that may take two passes: its kernel, and the output graph, whose arrays they borrow.
struct UnionCall {
    sg_kernel kernel;
    unsigned long long tp;
    const Graph *h;
};

// Whether two union passes (tri_union_kernel) pay.  They drop what is streamed and
// decided for deleted edges, at the price of a pass over the vertices and arcs
// between them and of more instructions per element (the filter, the windows).
// So there have to be lists well above kShortList, as shorter ones are streamed
// whole whatever happens; the W elements of one pass have to outweigh the pass
// over the vertices; and edges have to be deleted while their lists stream: s = p W / m
// bounds the selected triangles per edge (about a sixth of the elements close
// one on R-MAT graphs, all of them in cliques, which the rule cannot tell).
// What can be dropped grows with s and W, what the second pass costs does not:
// s W is the rest of the rule.  Where a triangle deletes two edges (p-2), s
// counts double; where it always deletes its heaviest (max-weight), light edges
// live on and both lines lie higher.  Calls in ms, one pass / two passes:
//   random      s, s W
//     R-MAT s20            1.3, 2.5e9  8.49 / 10.3    R-MAT s20            13, 2.5e10  8.67 / 7.06
//     R-MAT s22            5.5, 6.6e10 45.1 / 45.5    Chung-Lu 2^21       6.0, 1.2e10  11.3 / 9.89
//     n = 100,000, ef 16   6.3, 5.4e8  0.74 / 0.93    n = 30,000, ef 40    17, 1.2e9   0.66 / 0.60
//     n = 400,000, ef 8    5.6, 9.5e8  1.29 / 1.53    n = 60,000, ef 24    36, 3.1e9   0.71 / 0.67
//     n = 200,000, ef 16   7.9, 1.8e9  1.36 / 1.51    n = 200,000, ef 24   11, 4.7e9   2.40 / 2.03
//   max-weight
//     R-MAT s20             13, 2.5e10 9.38 / 9.84    Chung-Lu 1.4 M       13, 2.4e10  10.9 / 10.4
//     R-MAT s22             18, 2.2e11 49.6 / 50.6    Chung-Lu 2^21        18, 3.6e10  12.1 / 11.0
//     n = 30,000, ef 40     83, 6.2e9  0.68 / 0.70    n = 200,000, ef 24   32, 1.4e10  2.52 / 2.39
//   longest list 199 to 234 (s from 9): cliques of 200 18.1 / 21.6, n = 200,000, ef 8  0.65 / 1.10
static bool two_passes_pay(const Oriented &o, int64_t max_deg, int64_t work, const UnionCall &u) {
    const double w = (double)work;
    if (o.m == 0 || max_deg <= 2 * kShortList || w < 32.0 * (double)o.n) return false;
    const double s = (double)u.tp / 4294967296.0 * w / (double)o.m * (u.kernel == SG_TR_P2 ? 2.0 : 1.0);
    return u.kernel == SG_TR_MAXW ? s >= 10.0 && s * w >= 1e10 : s >= 4.0 && s * w >= 1.2e9;
}

// What two passes need beside the plan; false (and nothing kept) where it does not fit.
static bool two_passes_fit(Ctx *c, const Oriented &o, const UnionCall &u, Plan *pl) {
    // the records in the unused half of E+'s column array (room for nnz = 2m
    // entries) if it holds them (16 n <= 4 m: a mean degree of 8), in memory of
    // their own otherwise
    const uintptr_t b = ((uintptr_t)(o.col + o.m) + 15) & ~(uintptr_t)15, e = (uintptr_t)(o.col + 2 * o.m);
    sg_status st = SG_OK;
    if (b + sizeof(uint4) * (size_t)o.n <= e)
        pl->arec = reinterpret_cast<uint4 *>(b);
    else if ((st = dalloc(c, &pl->rec_own, sizeof(uint4) * (size_t)o.n)) == SG_OK)
        pl->arec = static_cast<uint4 *>(pl->rec_own);
    if (st == SG_OK) st = alive_alloc(c, o, u.h, &pl->al);
    if (st == SG_OK) return true;
    set_error("");
    alive_free(c, &pl->al);  // what it got of it
    dfree(c, pl->rec_own);
    pl->rec_own = nullptr;
    pl->arec = nullptr;
    return false;
}

// How the vertices are split between warps, CTAs and the hub launch.  u: a union
// call that may take two passes, which split them their own way.
static sg_status make_plan(Ctx *c, const Oriented &o, const int64_t *offs, Plan *pl, const UnionCall *u = nullptr) {
    if (o.m >= (int64_t)0xFFFFFFFFll)
        return fail(SG_ERR_UNSUPPORTED, "triangle kernels address oriented arcs with 32 bits: m must be < 2^32");
    if (o.n >= (int64_t)0xFFFFFFFEll)
        return fail(SG_ERR_UNSUPPORTED, "triangle kernels reserve vertex ids 2^32 - 2 and 2^32 - 1");
    pl->offs = offs;
    sg_status st = dalloc(c, (void **)&pl->heavy, sizeof(uint32_t) * (size_t)std::max<int64_t>(o.n, 1));
    if (st == SG_OK) st = dalloc(c, (void **)&pl->buckets, sizeof(unsigned long long) * 3 * kKeys);
    if (st == SG_OK) st = dalloc(c, (void **)&pl->din, sizeof(uint32_t) * (size_t)std::max<int64_t>(o.n, 1));
    if (st != SG_OK) return st;
    pl->inl = o.inl;  // the orientation's reverse list (not owned by the plan)
    SG_CUDA(cudaMemsetAsync(pl->buckets, 0, sizeof(unsigned long long) * 3 * kKeys, c->stream));
    SG_CUDA(cudaMemsetAsync(c->d_ctr + kCtrMaxDeg, 0, sizeof(unsigned long long), c->stream));
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((o.n + 255) / 256, (int64_t)c->num_sms * 8));
    if (o.n > 0) {
        SG_LAUNCH(c, "tri_classify");
        classify_count_kernel<<<(unsigned)blocks, 256, 0, c->stream>>>(o.off, offs, pl->din, o.n, pl->light_max,
                                                                       pl->light_items, (int64_t)kHeavyCap,
                                                                       pl->buckets, u ? pl->buckets + kKeys : nullptr,
                                                                       c->d_ctr);
    }
    SG_CUDA(cudaGetLastError());
    SG_CUDA(cudaMemcpyAsync(c->h_pinned, pl->buckets, sizeof(unsigned long long) * 2 * kKeys, cudaMemcpyDeviceToHost,
                            c->stream));
    SG_CUDA(cudaMemcpyAsync(c->h_pinned + 2 * kKeys, c->d_ctr + kCtrMaxDeg, sizeof(unsigned long long),
                            cudaMemcpyDeviceToHost, c->stream));
    SG_CUDA(cudaMemcpyAsync(c->h_pinned + 2 * kKeys + 1, c->d_ctr + kCtrWork, sizeof(unsigned long long),
                            cudaMemcpyDeviceToHost, c->stream));
    SG_CUDA(cudaStreamSynchronize(c->stream));
    unsigned long long cnt[2 * kKeys + 2];
    std::memcpy(cnt, c->h_pinned, sizeof(cnt));
    pl->max_deg = (int64_t)cnt[2 * kKeys];
    pl->work = (int64_t)cnt[2 * kKeys + 1];
    pl->two = u && u->h && two_passes_pay(o, pl->max_deg, pl->work, *u) && two_passes_fit(c, o, *u, pl);
    if (pl->two) {
        pl->light_max = kUnionLightMax;
        pl->light_items = kUnionLightItems;
    }
    const int split = pl->two ? kKeys : 0;
    pl->n_heavy = 0;
    pl->n_hubs = 0;
    for (int b = 0; b < kKeys; ++b) pl->n_heavy += (int64_t)cnt[split + b];
    for (int b = kBuckets; b < kKeys; ++b) pl->n_hubs += (int64_t)cnt[split + b];
    // a hub launch with fewer hubs than SMs would leave most SMs idle: the
    // main launch then takes them first (they lead the list), in chunks
    if (pl->n_hubs < c->num_sms) pl->n_hubs = 0;
    if (pl->n_heavy > 0) {
        SG_LAUNCH(c, "tri_classify");
        classify_scatter_kernel<<<(unsigned)blocks, 256, 0, c->stream>>>(o.off, pl->din, o.n, pl->light_max,
                                                                         pl->light_items, (int64_t)kHeavyCap,
                                                                         pl->buckets + split, pl->buckets + 2 * kKeys,
                                                                         pl->heavy, pl->arec, nullptr);
    }
    SG_CUDA(cudaGetLastError());
    // shared memory: hit queues + the larger of the heavy table (4 slots per
    // entry, load <= 1/4, with the list bounds of N+(u)) and the light tables with
    // the entries of 32 arcs each
    const size_t queue_bytes = sizeof(HitQueue) * kTW;
    const size_t light_bytes = (size_t)kTW * (kLightSlots * sizeof(uint32_t) + 32 * sizeof(uint4));
    int cap = 8;
    while (cap < pl->max_deg && cap < kHeavyCap) cap *= 2;
    pl->heavy_cap = cap;
    const size_t entry_bytes = 4 * sizeof(uint32_t) + 2 * sizeof(uint32_t) + sizeof(unsigned short);
    pl->smem = queue_bytes + std::max(light_bytes, (size_t)cap * entry_bytes);
    pl->usmem = sizeof(UnionScratch) * kTW +
                std::max((size_t)kTW * kUnionLightMax * (4 * sizeof(uint32_t) + kFilterBits / 8), union_table_bytes(cap));
    if (pl->n_hubs > 0) {
        int hc = kHeavyCap;
        while (hc < pl->max_deg && hc < kHubCap) hc *= 2;
        pl->hub_cap = hc;
        pl->hub_smem = sizeof(HitQueue) * kHubTW + (size_t)hc * entry_bytes;
        pl->uhub_smem = sizeof(UnionScratch) * kHubTW + union_table_bytes(hc);
    }
    return SG_OK;
}

// Dynamic shared memory of a CTA of `warps` warps with tables of up to `cap`
// entries: the larger of the counting and edge-once passes' and the union passes'.
static int max_smem(int warps, int cap) {
    const size_t enumeration = sizeof(HitQueue) * warps + (size_t)cap * (6 * sizeof(uint32_t) + sizeof(unsigned short));
    const size_t light = warps == kTW ? (size_t)kTW * kUnionLightMax * (4 * sizeof(uint32_t) + kFilterBits / 8) : 0;
    const size_t unions = sizeof(UnionScratch) * warps + std::max(light, union_table_bytes(cap));
    return (int)std::max(enumeration, unions);
}

// One launch of `kernel`: as many CTAs per SM as fit (or grid_per_sm), which
// claim their vertices through the work counters.
static sg_status launch_tri(Ctx *c, void (*kernel)(TriArgs), int threads, size_t smem, const TriArgs &a,
                            const char *name, int grid_per_sm = 0) {
    TriArgs args = a;
    SG_CUDA(cudaMemsetAsync(a.work, 0, 2 * sizeof(unsigned long long), c->stream));
    // the limit is the function's, shared by all threads and contexts: always the
    // most any graph asks of it, never this launch's size
    const int limit = threads == kTW * 32 ? max_smem(kTW, kHeavyCap) : max_smem(kHubTW, kHubCap);
    SG_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, limit));
    int per_sm = 0;
    SG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
    per_sm = std::max(per_sm, 1);
    if (grid_per_sm > 0) per_sm = std::min(per_sm, grid_per_sm);
    // a light vertex takes some 10 us of one warp: on a small graph claims of 32
    // would leave most warps idle (n = 1000: 32 warps of 4864 busy, 283 us),
    // so a warp claims what gives every warp about four turns
    const int64_t warps = (int64_t)c->num_sms * per_sm * (threads / 32);
    args.light_claim = (int)std::max<int64_t>(1, std::min<int64_t>(32, a.n / (warps * 4)));
    {
        SG_LAUNCH(c, name);
        kernel<<<(unsigned)(c->num_sms * per_sm), threads, smem, c->stream>>>(args);
    }
    SG_CUDA(cudaGetLastError());
    return SG_OK;
}

// One pass over all vertices: the hubs first, in CTAs that share a large
// table, then everything else.
static sg_status launch_pass(Ctx *c, void (*hub)(TriArgs), void (*main)(TriArgs), size_t hub_smem, size_t smem,
                             const TriArgs &base, const Plan &pl, const char *hub_name, const char *main_name) {
    if (base.n == 0) return SG_OK;
    TriArgs a = base;
    a.heavy = pl.heavy;
    a.n_heavy = pl.n_heavy;
    a.heavy_cap = pl.heavy_cap;
    a.light_max = pl.light_max;
    a.light_items = pl.light_items;
    a.offs = pl.offs;
    a.din = pl.din;
    a.arec = pl.arec;
    a.inl = pl.inl;
    a.work = c->d_ctr + kCtrAux;
    if (pl.n_hubs > 0) {
        TriArgs h = a;
        h.n_heavy = pl.n_hubs;
        h.heavy_cap = pl.hub_cap;
        const sg_status st = launch_tri(c, hub, kHubTW * 32, hub_smem, h, hub_name);
        if (st != SG_OK) return st;
        a.heavy = pl.heavy + pl.n_hubs;
        a.n_heavy = pl.n_heavy - pl.n_hubs;
    }
    return launch_tri(c, main, kTW * 32, smem, a, main_name);
}

template <Mode M>
static sg_status launch_enum(Ctx *c, const TriArgs &a, const Plan &pl) {
    return launch_pass(c, tri_enum_kernel<M, kHubTW>, tri_enum_kernel<M, kTW>, pl.hub_smem, pl.smem, a, pl, "tri_hubs",
                       "tri_enum");
}

// The one pass of a union kernel, or its two (see tri_union_kernel).
template <Mode M>
static sg_status launch_union(Ctx *c, const Oriented &o, TriArgs a, const Plan &pl) {
    // where nearly every triangle deletes an edge, the atomics to edges deleted long
    // ago queue up (cliques of 200 at p = 1: random 23.0 against 18.1 ms, max-weight
    // 25.6 against 19.7); elsewhere looking costs more (geometric graph, 2^20
    // vertices, p = 0.5: 4.84 against 5.13)
    a.look_first = a.tp > 3ull << 30;
    if (!pl.two) return launch_enum<M>(c, a, pl);
    a.short_max = pl.n_hubs > 0 ? kShortListHubs : kShortList;
    sg_status st = launch_pass(c, tri_union_kernel<M, kHubTW, false>, tri_union_kernel<M, kTW, false>, pl.uhub_smem,
                               pl.usmem, a, pl, "tri_hubs", "tri_enum");
    if (st == SG_OK) st = alive_build(c, o, a.del, pl.al, pl.arec);
    a.alive = pl.al.list;
    if (st == SG_OK)
        st = launch_pass(c, tri_union_kernel<M, kHubTW, true>, tri_union_kernel<M, kTW, true>, pl.uhub_smem, pl.usmem, a,
                         pl, "tri_rest_hubs", "tri_rest");
    return st;
}

static TriArgs base_args(Ctx *c, const Oriented &o) {
    TriArgs a{};
    a.offp = o.off;
    a.colp = o.col;
    a.wp = o.w;
    a.n = o.n;
    a.dead_flag = o.m <= (int64_t)kArcDead ? kArcDead : 0u;
    a.ctr = c->d_ctr;
    a.err = c->d_err;
    return a;
}

struct EoBufs {
    uint32_t *considered = nullptr;
    // lctr: [kEoBuckets] bucket fills, [kEoBuckets] bucket counts, an out length, then the overflow bits
    unsigned long long *resv = nullptr, *lctr = nullptr;
};

// Whether the device (or the partition of it that this process has) can host
// eo_rounds_kernel's cluster: sixteen CTAs of a whole SM each are more than any
// device must take, so this is asked once per context, and the rounds' own
// launches do the work where the answer is no.
static bool eo_cluster_fits(Ctx *c, int choice, void (*kernel)(EoRun)) {
    signed char &fits = c->eo_cluster[choice];
    if (fits < 0) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(kEoCluster);
        cfg.blockDim = dim3(kEoCta);
        cfg.stream = c->stream;
        int clusters = 0;
        fits = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
               cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0;
        (void)cudaGetLastError();
    }
    return fits != 0;
}

// Edge-once rounds.  Round r lets the live selected triangles with
// r2 < theta_r = 2^(27+r) bid (all of them from round 5 on).  A bidder that
// holds all three reservations is the smallest live triangle on each of its
// edges (every non-bidder has a larger key), so the accepted set equals the
// unrestricted greedy scan's, while most triangles die before they ever bid.
//
// The first round enumerates the triangles once and lists every live selected
// one (16 bytes each, within a quarter of free memory), split into buckets by
// the round in which it first bids.  Each later round works on lists alone:
// the survivors of the last round plus this round's bucket are filtered
// (triangles that lost an edge are dropped), bid and are compacted into the
// next active list, so a listed triangle is read once before it bids.  The
// listing pass also bids for its round's prefix, so if the list does not fit,
// the round still completes from those bids, accepting from the edges' side;
// later rounds enumerate and bid directly and retry the list once the live
// triangles fit.
static sg_status eo_run(Ctx *c, const Graph *g, const Oriented &o, sg_kernel k, const Plan &pl, TriArgs a, EoBufs &buf) {
    const size_t m = (size_t)std::max<int64_t>(o.m, 1);
    const int choice = k == SG_TR_EO_MAXW ? kChoiceMaxw : (k == SG_TR_EO_MINCOUNT ? kChoiceMinCount : kChoiceRandom);
    uint32_t *&considered = buf.considered;
    const size_t cwords = (m + 31) / 32;
    unsigned long long *&resv = buf.resv, *&lctr = buf.lctr;
    const size_t lctr_bytes = (2 * kEoBuckets + 1) * sizeof(unsigned long long) + sizeof(int);
    int *lovf = nullptr;
    uint4 *L = nullptr;    // bucketed list written by the enumeration (workspace kWsList)
    TriRec *A = nullptr;   // active list: this round's bidders (workspace a_slot)
    int a_slot = kWsActive1;
    int64_t lenA = 0;
    int64_t ubase[kEoBuckets] = {}, used[kEoBuckets] = {};
    // live selected triangles per bucket at the last listing pass: a bound on them now
    unsigned long long dem[kEoBuckets] = {};
    bool have_dem = false;
    int next_bucket = kEoBuckets;  // next bucket to merge into the active list
    int top = kEoBuckets;          // the list holds every live triangle of the buckets below this one
    int sched = 0;                 // step of the prefix schedule: bids come from r2 below the top of bucket sched
    bool listed = false;
    bool no_small = false;         // the small graph's list size did not fit, or left no room for the active lists
    bool small_list = false;       // the list was allocated at that size
    bool try_list = o.m <= (int64_t)0xFFFFFFFFll && c->eo_list_cap >= 0;
    // warps of one enumeration launch, at most: each may leave a chunk per bucket part filled
    const int64_t emit_warps = (int64_t)c->num_sms * (8 * kTW + kHubTW);
    sg_status st = dalloc(c, (void **)&considered, cwords * sizeof(uint32_t));
    if (st == SG_OK) st = dalloc(c, (void **)&resv, m * sizeof(unsigned long long));
    if (st == SG_OK) st = dalloc(c, (void **)&lctr, lctr_bytes);
    if (st == SG_OK) {
        lovf = reinterpret_cast<int *>(lctr + 2 * kEoBuckets + 1);
        if (cudaMemsetAsync(considered, 0, cwords * sizeof(uint32_t), c->stream) != cudaSuccess)
            st = cuda_fail(cudaGetLastError(), "memset");
    }
    a.considered = considered;
    a.resv = resv;
    const int64_t acc_blocks = std::min<int64_t>((o.n + 7) / 8, (int64_t)c->num_sms * 8);
    if (st == SG_OK && cudaMemsetAsync(resv, 0xFF, m * sizeof(unsigned long long), c->stream) != cudaSuccess)
        st = cuda_fail(cudaGetLastError(), "memset");
    // a warp of the main launch lists about a sixth of its probes' share of p W
    // (R-MAT graphs); its claims together should be at most half of that
    const double per_warp = (double)a.tp / 4294967296.0 * (double)pl.work / 6.0 / ((double)c->num_sms * 4 * kTW);
    a.eo_shift = 0;
    while (a.eo_shift < 6 && (double)(2048 >> a.eo_shift) > 0.5 * per_warp) ++a.eo_shift;
    auto list_blocks = [&](int64_t len) { return std::min<int64_t>((len + 255) / 256, (int64_t)c->num_sms * 8); };
    cudaMemPool_t pool = nullptr;
    if (cudaDeviceGetMemPool(&pool, c->device) != cudaSuccess) {
        (void)cudaGetLastError();
        pool = nullptr;
    }
    auto list_capacity = [&]() -> int64_t {
        size_t fr = 0, tot = 0;
        if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) fr = 0;
        // memory the stream-ordered pool keeps from earlier calls but does not use is free too
        uint64_t reserved = 0, used = 0;  // the pool attributes are 64-bit counts
        if (pool && cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) == cudaSuccess &&
            cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess && reserved > used)
            fr += (size_t)(reserved - used);
        (void)cudaGetLastError();
        if (c->alloc_limit) fr = std::min(fr, c->alloc_limit - std::min(c->alloc_limit, c->alloc_live));
        for (int i = 0; i < 3; ++i) fr += c->ws_bytes[i];  // the context's workspaces are reused
        int64_t cap = (int64_t)(fr / 4 / sizeof(uint4));
        if (c->eo_list_cap > 0) cap = std::min<int64_t>(cap, c->eo_list_cap);
        return cap;
    };
    for (int round = 0; st == SG_OK; ++round, ++sched) {
        if (round > 100000) { st = fail(SG_ERR_TIMEOUT, "edge-once rounds did not converge"); break; }
        const int rb = std::min(sched, kEoBuckets - 1);
        unsigned long long theta = 1ull << (27 + rb);
        if (listed && top < kEoBuckets) theta = std::min(theta, 1ull << (26 + top));  // the list's window
        a.eo_theta = theta;
        unsigned long long live = 0;
        if (!listed) {
            bool bids_done = false;
            int hi = 0;  // buckets [rb, hi) get room in the list
            if (try_list) {
                // ---- one enumeration bids for this round and lists the live selected
                // triangles of as many buckets, from rb on, as the room allows
                // (asking how much memory is free takes longer than a small graph's
                // rounds: a list that is bounded by 2^24 records is not worth it)
                const double most = (double)a.tp / 4294967296.0 * (double)pl.work;
                const bool small = !no_small && !have_dem && c->eo_list_cap == 0 && most <= (double)(1 << 23);
                const int64_t cap = small ? (int64_t)1 << 24 : list_capacity();
                hi = kEoBuckets;
                int64_t run = 0;
                for (int b = 0; b < kEoBuckets; ++b) a.list_base[b] = a.list_cap[b] = 0;
                auto give = [&](int b, int64_t cb) {
                    a.list_base[b] = (unsigned long long)run;
                    a.list_cap[b] = (unsigned long long)cb;
                    ubase[b] = run;
                    run += cb;
                };
                // the shares of the draws r2 over the buckets: 1,1,2,4,8,16 of 32
                // (earlier buckets fold into rb)
                double w[kEoBuckets], wsum = 0.0;
                for (int b = 0; b < kEoBuckets; ++b) w[b] = b <= 1 ? 1.0 : (double)(1 << (b - 1));
                for (int b = 0; b < rb; ++b) { w[rb] += w[b]; w[b] = 0.0; }
                for (int b = 0; b < kEoBuckets; ++b) wsum += w[b];
                // no counts yet: a triangle is found by one probe, so at most
                // about p W are selected (W probes per pass)
                const double sel_max = (double)a.tp / 4294967296.0 * (double)pl.work;
                if (!have_dem && sel_max <= (double)cap) {
                    // everything fits: split the room by the shares
                    for (int b = rb; b < kEoBuckets; ++b) {
                        const int64_t cb = (int64_t)((double)cap * w[b] / wsum);
                        if (cb < 4 * eo_chunk(b, a.eo_shift)) { hi = b; break; }
                        give(b, cb);
                    }
                } else {
                    // Each bucket wants its bound: the last pass's count (live
                    // triangles only die) or, before the first pass, a quarter of p W
                    // (R-MAT graphs find a triangle in 12-18% of their probes), plus
                    // room for sealed chunk tails.  The bounds are loose -- deciding a
                    // window kills most of the triangles above it -- so when they do
                    // not all fit, this round's bucket gets its bound (up to half the
                    // room) and the rest is split in proportion to the bounds above:
                    // a bucket that overflows only narrows the window.
                    unsigned long long fold = 0;
                    for (int b = 0; b <= rb; ++b) fold += dem[b];
                    int64_t want[kEoBuckets] = {};
                    double above = 0.0;
                    for (int b = rb; b < kEoBuckets; ++b) {
                        const double d = have_dem ? (double)(b == rb ? fold : dem[b]) : 0.25 * sel_max * w[b] / wsum;
                        want[b] = (int64_t)(d * (1.0 + 16.0 / eo_chunk(b, a.eo_shift))) + emit_warps * eo_chunk(b, a.eo_shift);
                        if (b > rb) above += (double)want[b];
                    }
                    const int64_t first = std::min<int64_t>(want[rb], cap / 2);
                    const double rest = (double)(cap - first);
                    const double scale = above <= rest ? 1.0 : rest / above;
                    for (int b = rb; b < kEoBuckets; ++b) {
                        const int64_t cb = b == rb ? first : (int64_t)((double)want[b] * scale);
                        if (cb < 4 * eo_chunk(b, a.eo_shift)) { hi = b; break; }
                        give(b, cb);
                    }
                }
                if (hi <= rb) hi = 0;  // nothing to list: the pass only bids and counts
                if (hi > 0) {
                    const size_t lbytes = (size_t)std::max<int64_t>(run, 1) * sizeof(uint4);
                    small_list = small;
                    if (small) {
                        if (ws_get(c, kWsList, lbytes, (void **)&L) != SG_OK) {  // size it by the free memory then
                            set_error("");
                            L = nullptr;
                            no_small = true;
                            --round;
                            --sched;
                            continue;
                        }
                    } else if (ws_get(c, kWsList, lbytes, (void **)&L) != SG_OK && pool) {
                        // the pool's idle memory may be too fragmented: hand it back and retry
                        (void)cudaStreamSynchronize(c->stream);
                        (void)cudaMemPoolTrimTo(pool, 0);
                        (void)cudaGetLastError();
                        if (ws_get(c, kWsList, lbytes, (void **)&L) != SG_OK) L = nullptr;
                    }
                    if (L == nullptr) {
                        set_error("");
                        try_list = false;
                    }
                }
            }
            if (try_list) {
                a.list = L;
                a.list_ctr = lctr;
                a.list_dem = lctr + kEoBuckets;
                a.list_overflow = lovf;
                a.eo_round = rb;
                a.eo_hi = L != nullptr ? hi : 0;
                SG_CUDA(cudaMemsetAsync(lctr, 0, lctr_bytes, c->stream));
                SG_CUDA(cudaMemsetAsync(c->d_ctr + kCtrLive, 0, sizeof(unsigned long long), c->stream));
                // nothing is considered before the first acceptance: skip the flag reads
                a.considered = round == 0 ? nullptr : considered;
                st = launch_enum<Mode::EoEmit>(c, a, pl);
                ++c->eo_passes;
                a.considered = considered;
                a.list = nullptr;
                if (st != SG_OK) break;
                unsigned long long fill[2 * kEoBuckets + 1];
                int ovf = 0;
                SG_CUDA(cudaMemcpyAsync(c->h_pinned, lctr, 2 * kEoBuckets * sizeof(unsigned long long),
                                        cudaMemcpyDeviceToHost, c->stream));
                SG_CUDA(cudaMemcpyAsync(c->h_pinned + 2 * kEoBuckets, c->d_ctr + kCtrLive, sizeof(unsigned long long),
                                        cudaMemcpyDeviceToHost, c->stream));
                SG_CUDA(cudaMemcpyAsync(c->h_pinned + 2 * kEoBuckets + 1, lovf, sizeof(int), cudaMemcpyDeviceToHost,
                                        c->stream));
                SG_CUDA(cudaStreamSynchronize(c->stream));
                std::memcpy(fill, c->h_pinned, sizeof(fill));
                std::memcpy(&ovf, c->h_pinned + 2 * kEoBuckets + 1, sizeof(int));
                live = fill[2 * kEoBuckets];
                for (int b = 0; b < kEoBuckets; ++b) dem[b] = fill[kEoBuckets + b];
                have_dem = true;
                if (live == 0) break;  // no live selected triangle is left
                // the buckets below the first one that ran out of room are complete
                const int wtop = a.eo_hi > 0 ? std::min(a.eo_hi, ovf ? __builtin_ctz((unsigned)ovf) : kEoBuckets) : 0;
                if (wtop > rb) {
                    listed = true;
                    top = wtop;
                    for (int b = 0; b < kEoBuckets; ++b) used[b] = b >= rb && b < top ? (int64_t)fill[b] : 0;
                    for (int b = rb; b < top; ++b) c->eo_listed += dem[b];
                    ++c->eo_list_passes;
                    next_bucket = rb;
                } else {
                    // this round's bids are in: finish it from the edges' side
                    L = nullptr;
                    bids_done = true;
                }
            }
            if (!listed) {
                // ---- enumeration round that bids directly; acceptance from the edges' side
                if (!bids_done) {
                    SG_CUDA(cudaMemsetAsync(c->d_ctr + kCtrLive, 0, sizeof(unsigned long long), c->stream));
                    a.considered = round == 0 ? nullptr : considered;
                    st = launch_enum<Mode::EoReserve>(c, a, pl);
                    ++c->eo_passes;
                    a.considered = considered;
                    if (st != SG_OK) break;
                    st = read_ctr(c, kCtrLive, 1, &live);
                    if (st != SG_OK || live == 0) break;
                }
                ++c->eo_rounds;
                SG_LAUNCH(c, "tri_eo_accept");
                if (choice == kChoiceMaxw)
                    eo_accept_kernel<kChoiceMaxw><<<(unsigned)acc_blocks, 256, 0, c->stream>>>(a, g->off, considered);
                else if (choice == kChoiceMinCount)
                    eo_accept_kernel<kChoiceMinCount><<<(unsigned)acc_blocks, 256, 0, c->stream>>>(a, g->off,
                                                                                                  considered);
                else
                    eo_accept_kernel<kChoiceRandom><<<(unsigned)acc_blocks, 256, 0, c->stream>>>(a, g->off, considered);
                SG_CUDA(cudaGetLastError());
                SG_CUDA(cudaMemsetAsync(resv, 0xFF, m * sizeof(unsigned long long), c->stream));
                continue;
            }
        }
        // ---- a list this short: all rounds left in one launch
        int64_t rest = lenA;
        for (int b = next_bucket; b < top; ++b) rest += used[b];
        auto one = choice == kChoiceMaxw ? eo_rounds_kernel<kChoiceMaxw>
                   : choice == kChoiceMinCount ? eo_rounds_kernel<kChoiceMinCount>
                                               : eo_rounds_kernel<kChoiceRandom>;
        if (rest <= kEoOneLaunch && c->eo_one_launch && eo_cluster_fits(c, choice, one)) {
            TriRec *B = nullptr;
            const int bslot = a_slot == kWsActive0 ? kWsActive1 : kWsActive0;
            const size_t bytes = (size_t)std::max<int64_t>(rest, 1) * sizeof(TriRec);
            bool room = ws_get(c, bslot, bytes, (void **)&B) == SG_OK;
            // (the buffer that holds the survivors has room for them; the first
            // round reads it, later ones write at most what the round before kept)
            if (room && lenA == 0) room = ws_get(c, a_slot, bytes, (void **)&A) == SG_OK;
            if (!room) set_error("");  // a round's own launches need less
            if (room && c->ws_bytes[a_slot] >= bytes) {
                SG_CUDA(cudaMemsetAsync(lctr, 0, lctr_bytes, c->stream));
                EoRun r{};
                r.fresh = L;
                for (int b = 0; b < kEoBuckets; ++b) {
                    r.base[b] = ubase[b];
                    r.used[b] = used[b];
                }
                r.active[0] = A;
                r.active[1] = B;
                r.len = lenA;
                r.next_bucket = next_bucket;
                r.top = top;
                r.sched = sched;
                r.out_len = lctr;
                r.rounds = lctr + 2;
                r.resv = resv;
                r.considered = considered;
                r.del = a.del;
                r.colp = a.colp;
                r.tcnt = a.tcnt;
                r.wp = a.wp;
                r.k0 = a.k0;
                r.k1 = a.k1;
                {
                    SG_LAUNCH(c, "tri_eo_rounds");
                    one<<<kEoCluster, kEoCta, 0, c->stream>>>(r);
                }
                SG_CUDA(cudaGetLastError());
                SG_CUDA(cudaMemcpyAsync(c->h_pinned, r.rounds, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream));
                SG_CUDA(cudaStreamSynchronize(c->stream));
                c->eo_rounds += (uint64_t)c->h_pinned[0];
                lenA = 0;
                next_bucket = top;
                if (top >= kEoBuckets) break;
                for (int b = 0; b < top; ++b) dem[b] = 0;
                L = nullptr;
                listed = false;
                sched = top - 1;
                continue;
            }
        }
        // ---- list round: last round's survivors plus this round's bucket
        const int64_t fresh = next_bucket < top ? used[next_bucket] : 0;
        TriRec *B = nullptr;
        const int bslot = a_slot == kWsActive0 ? kWsActive1 : kWsActive0;
        st = ws_get(c, bslot, (size_t)std::max<int64_t>(lenA + fresh, 1) * sizeof(TriRec), (void **)&B);
        if (st == SG_ERR_OOM && small_list) {
            // the list was sized without asking for the free memory: give it back and
            // list what is live again, within a quarter of what there is
            set_error("");
            st = SG_OK;
            dfree(c, c->ws[kWsList]);
            c->ws[kWsList] = nullptr;
            c->ws_bytes[kWsList] = 0;
            L = nullptr;
            lenA = 0;
            listed = small_list = false;
            no_small = true;
            top = next_bucket = kEoBuckets;
            --round;
            --sched;
            continue;
        }
        if (st != SG_OK) break;
        unsigned long long *out_len = lctr + 2 * kEoBuckets;
        SG_CUDA(cudaMemsetAsync(out_len, 0, sizeof(unsigned long long), c->stream));
        if (lenA > 0) {
            SG_LAUNCH(c, "tri_eo_list_reserve");
            eo_list_reserve_kernel<<<(unsigned)list_blocks(lenA), 256, 0, c->stream>>>(A, lenA, B, out_len, resv,
                                                                                     considered, theta);
        }
        if (fresh > 0) {
            SG_LAUNCH(c, "tri_eo_fresh_reserve");
            eo_fresh_reserve_kernel<<<(unsigned)list_blocks((fresh + kFreshPer - 1) / kFreshPer), 256, 0,
                                      c->stream>>>(
                L + ubase[next_bucket], fresh, B, out_len, resv, considered, theta, a.colp, a.k0, a.k1);
        }
        if (next_bucket < top) ++next_bucket;
        SG_CUDA(cudaGetLastError());
        SG_CUDA(cudaMemcpyAsync(c->h_pinned, out_len, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream));
        SG_CUDA(cudaStreamSynchronize(c->stream));
        std::memcpy(&live, c->h_pinned, sizeof(live));
        A = B;
        a_slot = bslot;
        lenA = (int64_t)live;
        if (live == 0) {
            if (next_bucket < top) continue;  // nothing bid this round
            if (top >= kEoBuckets) break;     // no triangle left anywhere
            // every triangle of the list's window is decided: list the live ones
            // above it, starting the schedule at its first bucket
            for (int b = 0; b < top; ++b) dem[b] = 0;
            L = nullptr;
            listed = false;
            sched = top - 1;
            continue;
        }
        ++c->eo_rounds;
        // ---- accept: triangles holding all three reservations.  Judging from
        // the edge side costs a pass over m reservations plus a binary search
        // per reserved arc; once the list holds at most two triangles per
        // edge, read the list instead
        if ((double)lenA <= 2.0 * (double)m) {
            SG_LAUNCH(c, "tri_eo_list_accept");
            const unsigned blocks = (unsigned)list_blocks(lenA);
            if (choice == kChoiceMaxw)
                eo_list_accept_kernel<kChoiceMaxw><<<blocks, 256, 0, c->stream>>>(A, lenA, resv, considered, a.del,
                                                                                  a.wp, a.tcnt);
            else if (choice == kChoiceMinCount)
                eo_list_accept_kernel<kChoiceMinCount><<<blocks, 256, 0, c->stream>>>(A, lenA, resv, considered,
                                                                                      a.del, a.wp, a.tcnt);
            else
                eo_list_accept_kernel<kChoiceRandom><<<blocks, 256, 0, c->stream>>>(A, lenA, resv, considered, a.del,
                                                                                    a.wp, a.tcnt);
        } else {
            SG_LAUNCH(c, "tri_eo_accept");
            if (choice == kChoiceMaxw)
                eo_accept_kernel<kChoiceMaxw><<<(unsigned)acc_blocks, 256, 0, c->stream>>>(a, g->off, considered);
            else if (choice == kChoiceMinCount)
                eo_accept_kernel<kChoiceMinCount><<<(unsigned)acc_blocks, 256, 0, c->stream>>>(a, g->off, considered);
            else
                eo_accept_kernel<kChoiceRandom><<<(unsigned)acc_blocks, 256, 0, c->stream>>>(a, g->off, considered);
        }
        SG_CUDA(cudaGetLastError());
        // ---- reset the reservations for the next round: three scattered
        // writes per listed triangle beat clearing all m words only for short lists
        if ((double)lenA * 96.0 <= 8.0 * (double)m) {
            SG_LAUNCH(c, "tri_eo_list_reset");
            eo_list_reset_kernel<<<(unsigned)list_blocks(lenA), 256, 0, c->stream>>>(A, lenA, resv);
        } else {
            SG_CUDA(cudaMemsetAsync(resv, 0xFF, m * sizeof(unsigned long long), c->stream));
        }
        SG_CUDA(cudaGetLastError());
    }
    return st;
}

static sg_status eo_rounds(Ctx *c, const Graph *g, const Oriented &o, sg_kernel k, const Plan &pl, const TriArgs &a) {
    EoBufs buf;
    const sg_status st = eo_run(c, g, o, k, pl, a, buf);  // (which returns in its middle on an error)
    dfree(c, buf.lctr);
    dfree(c, buf.considered);
    dfree(c, buf.resv);
    return st;
}

sg_status tr_mark(Ctx *c, const Graph *g, const Oriented &o, sg_kernel k, double p, uint64_t seed, uint32_t *del,
                  const Graph *h) {
    Plan pl;
    TriArgs a = base_args(c, o);
    a.k0 = (uint32_t)(seed & 0xFFFFFFFFu);
    a.k1 = (uint32_t)(seed >> 32);
    a.tp = prob_threshold(p);
    a.del = del;
    const UnionCall u{k, a.tp, h};
    const bool choose = k == SG_TR_RANDOM || k == SG_TR_MAXW || k == SG_TR_P2;
    sg_status st = make_plan(c, o, g->off, &pl, choose ? &u : nullptr);
    uint32_t *tcnt = nullptr;
    if (st == SG_OK && (k == SG_TR_MINCOUNT || k == SG_TR_EO_MINCOUNT)) {
        // the min-count choice needs the triangle count of every edge of G first
        const size_t bytes = sizeof(uint32_t) * (size_t)std::max<int64_t>(o.m, 1);
        st = dalloc(c, (void **)&tcnt, bytes);
        if (st == SG_OK && cudaMemsetAsync(tcnt, 0, bytes, c->stream) != cudaSuccess)
            st = cuda_fail(cudaGetLastError(), "cudaMemsetAsync(tcnt)");
        a.tcnt = tcnt;
        if (st == SG_OK) st = launch_enum<Mode::EdgeCount>(c, a, pl);
        if (st == SG_OK && k == SG_TR_MINCOUNT && h && two_passes_pay(o, pl.max_deg, pl.work, u)) {
            free_plan(c, &pl);
            pl = Plan{};
            st = make_plan(c, o, g->off, &pl, &u);
        }
    }
    if (st == SG_OK) {
        switch (k) {
        case SG_TR_RANDOM: st = launch_union<Mode::UnionRandom>(c, o, a, pl); break;
        case SG_TR_MAXW: st = launch_union<Mode::UnionMaxw>(c, o, a, pl); break;
        case SG_TR_P2: st = launch_union<Mode::UnionP2>(c, o, a, pl); break;
        case SG_TR_MINCOUNT: st = launch_union<Mode::UnionMinCount>(c, o, a, pl); break;
        default: st = eo_rounds(c, g, o, k, pl, a); break;
        }
    }
    dfree(c, tcnt);
    free_plan(c, &pl);
    return st;
}

sg_status tr_count(Ctx *c, const Graph *g, const Oriented &o, int64_t *count, int64_t *probes, int64_t *maxdeg,
                   int64_t *in_arcs, int64_t *fwd_probes) {
    Plan pl;
    unsigned long long v0[kCtrCount] = {}, v1[kCtrCount] = {};
    sg_status st = read_ctr(c, 0, kCtrCount, v0);
    if (st == SG_OK) st = make_plan(c, o, g->off, &pl);
    if (st == SG_OK) st = launch_enum<Mode::Count>(c, base_args(c, o), pl);
    if (st == SG_OK) st = read_ctr(c, 0, kCtrCount, v1);
    if (count) *count = (int64_t)(v1[kCtrTriangles] - v0[kCtrTriangles]);
    if (probes) *probes = (int64_t)(v1[kCtrProbes] - v0[kCtrProbes]);
    if (maxdeg) *maxdeg = pl.max_deg;
    // summed afresh by this orientation's reverse list
    if (in_arcs) *in_arcs = (int64_t)v1[kCtrInArcs];
    if (fwd_probes) *fwd_probes = (int64_t)v1[kCtrWorkFwd];
    free_plan(c, &pl);
    return st;
}

// Triangles through every vertex (device uint64[n], overwritten).
sg_status tr_vertex_counts(Ctx *c, const Graph *g, const Oriented &o, unsigned long long *vcnt) {
    Plan pl;
    sg_status st = make_plan(c, o, g->off, &pl);
    if (st == SG_OK && cudaMemsetAsync(vcnt, 0, sizeof(unsigned long long) * (size_t)std::max<int64_t>(o.n, 1),
                                       c->stream) != cudaSuccess)
        st = cuda_fail(cudaGetLastError(), "cudaMemsetAsync(vcnt)");
    TriArgs a = base_args(c, o);
    a.vcnt = vcnt;
    if (st == SG_OK) st = launch_enum<Mode::VertexCount>(c, a, pl);
    free_plan(c, &pl);
    return st;
}

// ---------------------------------------------------------- batched union
sg_status batch_tr_prepare(Ctx *c, const Graph *u, const Oriented &o, BatchTri *bt) {
    Plan pl;
    pl.light_max = bt->light_max;
    pl.light_items = 4 * bt->light_max;
    sg_status st = make_plan(c, o, u->off, &pl);
    if (st == SG_OK) {
        bt->smem = pl.smem;
        bt->max_deg = pl.heavy_cap;
    }
    free_plan(c, &pl);
    if (st != SG_OK) return st;
    if (!bt->heavy) st = dalloc(c, (void **)&bt->heavy, sizeof(uint32_t) * (size_t)std::max<int64_t>(o.n, 1));
    if (st == SG_OK && !bt->buckets)
        st = dalloc(c, (void **)&bt->buckets, sizeof(unsigned long long) * (2 * kKeys + 1));
    if (st == SG_OK && !bt->din) st = dalloc(c, (void **)&bt->din, sizeof(uint32_t) * (size_t)std::max<int64_t>(o.n, 1));
    // Per call only the graphs with a triangle kernel are oriented, so E+ can
    // hold fewer than nnz/2 arcs and the in-list room off(v) - off+(v) then
    // reaches up to nnz: size the records for that.
    if (st == SG_OK && !bt->inl)
        st = dalloc(c, (void **)&bt->inl, sizeof(uint2) * (size_t)std::max<int64_t>(u->nnz, 1));
    return st;
}

void batch_tr_free(Ctx *c, BatchTri *bt) {
    dfree(c, bt->heavy);
    dfree(c, bt->buckets);
    dfree(c, bt->din);
    dfree(c, bt->inl);
    bt->heavy = nullptr;
    bt->buckets = nullptr;
    bt->din = nullptr;
    bt->inl = nullptr;
}

// No host synchronisation: the heavy-vertex count stays on the device.
sg_status batch_tr_mark(Ctx *c, const Graph *u, const Oriented &o, const BatchDev &b, const BatchTri &bt,
                        uint32_t *del) {
    if (o.n == 0) return SG_OK;
    const int light_items = 4 * bt.light_max;
    SG_CUDA(cudaMemsetAsync(bt.buckets, 0, sizeof(unsigned long long) * (2 * kKeys + 1), c->stream));
    sg_status st = SG_OK;  // the reverse list bt.inl was filled after the batch orientation
    if (st != SG_OK) return st;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((o.n + 255) / 256, (int64_t)c->num_sms * 8));
    {
        SG_LAUNCH(c, "tri_classify");
        // no hub launch in a batch: its graphs are small, and a long N+(u) is chunked
        classify_count_kernel<<<(unsigned)blocks, 256, 0, c->stream>>>(o.off, u->off, bt.din, o.n, bt.light_max,
                                                                       light_items, INT64_MAX, bt.buckets, nullptr,
                                                                       c->d_ctr);
    }
    {
        SG_LAUNCH(c, "tri_classify");
        classify_scatter_kernel<<<(unsigned)blocks, 256, 0, c->stream>>>(o.off, bt.din, o.n, bt.light_max,
                                                                         light_items, INT64_MAX, bt.buckets,
                                                                         bt.buckets + kKeys, bt.heavy, nullptr,
                                                                         bt.buckets + 2 * kKeys);
    }
    SG_CUDA(cudaGetLastError());
    TriArgs a = base_args(c, o);
    a.del = del;
    a.heavy = bt.heavy;
    a.n_heavy = 0;
    a.n_heavy_dev = bt.buckets + 2 * kKeys;
    a.heavy_cap = bt.max_deg;
    a.light_max = bt.light_max;
    a.light_items = light_items;
    a.offs = u->off;
    a.din = bt.din;
    a.inl = bt.inl;
    a.work = c->d_ctr + kCtrAux;
    a.bparams = b.params;
    a.vgid = b.vgid;
    return launch_tri(c, tri_enum_kernel<Mode::BatchUnion, kTW>, kTW * 32, bt.smem, a, "tri_enum", bt.grid_per_sm);
}

}  // namespace sg
