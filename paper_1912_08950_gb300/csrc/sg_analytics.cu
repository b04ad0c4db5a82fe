// Accuracy analytics of Slim Graph (Sec. 5): PageRank (Table 1), the
// Kullback-Leibler divergence of two PageRank distributions (Sec. 5.2.3) and
// the number of connected components (Table 1), plus CSR validation.
//
// PageRank is FP32 with a fixed reduction order (no floating-point atomics),
// so a graph always yields the same vector; the dangling mass and the final
// L1 residual are reduced in fixed block order.  KL is evaluated in FP64 from
// the FP32 vectors.  Connected components use concurrent union-find: roots
// hook to the smaller root with atomicCAS, then pointer jumping flattens the
// forest; the count of self-parented vertices is exact whatever the schedule.
// The edges are taken in the order of Sutton et al.'s Afforest (IPDPS'18):
// every vertex first links its first kCcSample neighbours, the most frequent
// root among sampled vertices is taken as the giant component, and then only
// the rows of vertices outside it link their remaining neighbours (an edge
// leaving the giant component is seen from its other end).
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "sg_internal.cuh"

namespace sg {

constexpr int kPrThreads = 256;
constexpr int kPrWarps = kPrThreads / 32;

// x'_v = (1-d)/n + d (sum_{u in N(v)} y_u + D/n), y_u = x_u / d_u, D the rank
// of the degree-0 vertices.
//
// An iteration is one gather of y per arc, and the gathers, not the bytes, are
// the bound: a warp's 32 loads fall into 32 sectors, and the L1 can only have as
// many misses in flight as it has lines.  So y is kept in order of falling
// degree -- the arcs' heads are translated to positions once per call (colx)
// -- and every CTA copies its first kPrHot entries (R-MAT s22: 0.8% of the
// vertices, the heads of 54% of the arcs) to shared memory when an iteration
// starts; the L1 keeps the next ones, which share lines.  The heads stream past
// it (evict-first).  One CTA of 32 warps per SM, eight slabs of 32 arcs in
// flight per warp.  Per iteration on R-MAT s22 (128 M arcs) 339 us, against 634
// with y in vertex order and launches of their own for hub rows and D; s20: 88
// against 172; n = 100,000: 26 against 41.  Half of the L1 for y is where the line lies: 373 us at 32 K
// entries before the heads were streamed, 403 at 16 K, 387 at 24 K and 389 at
// 40 K; 54 K entries (all of the shared memory) leave too few lines: 588.
//
// Row sums have a fixed order, so a graph always gives the same vector: rows
// of up to kShortRow arcs are summed 32 rows at a time -- their arcs are
// numbered consecutively and streamed in slabs of 32, a lane finds its arc's
// row among the rows' starts, a segmented shuffle scan sums each row's run
// inside the slab and the run's last lane adds it to the row's slot; longer
// rows by a warp (lanes stride the row, then a fixed shuffle tree); hub rows
// in chunks of kHubChunk arcs (eight interleaved runs per lane, each run's
// tree, then the eight in order), and the warp that finishes a hub's last chunk
// adds the chunks in order.
constexpr int kShortRow = 32;
constexpr int kHubRow = 1024;
constexpr int kHubChunk = 8192;
constexpr int kPrCta = 1024;              // threads of the iteration kernel
constexpr int kPrHot = 32 * 1024;         // entries of y in shared memory, at most
constexpr int kDegBuckets = 256;          // degree buckets: exact below 16, eighths of an octave above

__device__ __forceinline__ int degree_bucket(int64_t d) {
    if (d < 16) return (int)d;
    const int e = 63 - __clzll((unsigned long long)d);
    return min(16 + (e - 4) * 8 + (int)((d >> (e - 3)) & 7), kDegBuckets - 1);
}

struct PrHubs {
    const uint32_t *row;        // hub rows, in any order
    const unsigned long long *count;  // [0] hubs, [1] chunks, [2] rows of medium length
    const int *first;           // first chunk of hub h
    const uint32_t *chunk_hub;  // hub of chunk c
    float *part;                // sums of the chunks, or of their runs
    unsigned int *done;         // ... of hub h that are there in this iteration (0 between iterations)
};

struct PrArgs {
    const int64_t *off;
    const uint32_t *colx;  // position in y of every arc's head
    const uint32_t *pos;   // position of every vertex (NULL: its id)
    int64_t n;
    int hot;               // the first positions, which a CTA keeps in shared memory (0: none)
    float base, damping, inv_n;
    const float *y;
    float *y_new;
    float *x_prev;         // the values before the last iteration
    float *x_out;
    PrHubs hubs;
    const uint32_t *medium;  // rows of more than kShortRow arcs that are no hubs, in any order
    // the rank of the degree-0 vertices: how many each virtual lane sums, the
    // warp sums that give D of the last iteration and those of this one
    const uint32_t *lane_cnt;
    int vblocks;
    const float *wsum;
    float *wsum_new;
    unsigned int *work, *work_next;  // next unit of this iteration, of the next one
    int per_claim;         // 32-row groups per claim
};

// D of the last iteration from its warp sums: every virtual block's eight in
// order, then a fixed tree over 256 strided sums.  All threads call it.
__device__ float pr_dangling(const float *wsum, int vblocks, float *s) {
    if (threadIdx.x < kPrThreads) {
        float acc = 0.f;
        for (int i = threadIdx.x; i < vblocks; i += kPrThreads) {
            float bd = 0.f;
            for (int w = 0; w < kPrWarps; ++w) bd += __ldg(wsum + (size_t)i * kPrWarps + w);
            acc += bd;
        }
        s[threadIdx.x] = acc;
    }
    __syncthreads();
    for (int h = kPrThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
        __syncthreads();
    }
    return s[0];
}

// Warp sums of the rank of the degree-0 vertices, each of which holds `val`: a
// lane of the virtual warps adds its vertices' ranks one by one.
__device__ __forceinline__ void pr_dangling_sums(const uint32_t *lane_cnt, int vblocks, float val, float *wsum) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < (int64_t)vblocks * kPrWarps; w += nw) {
        float t = 0.f;
        for (uint32_t k = __ldg(lane_cnt + w * 32 + lane); k > 0; --k) t += val;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
        if (lane == 0) wsum[w] = t;
    }
}

// What an iteration stores: y, y and x (the one before the last), or x_out (the last).
enum class PrStore { kNone, kPrev, kLast };

template <bool kHot, PrStore S>
__global__ void __launch_bounds__(kPrCta, 1) pr_iter_kernel(PrArgs a) {
    extern __shared__ float s_y[];
    __shared__ float s_acc[kPrCta / 32][32];
    __shared__ longlong2 s_row[kPrCta / 32][32];  // first arc minus its number, and the row, of the short rows
    __shared__ float s_red[kPrThreads];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if constexpr (kHot) {
        const int quads = (a.hot + 3) >> 2;  // (y has room for whole ones)
        const float4 *src = reinterpret_cast<const float4 *>(a.y);
        for (int i = threadIdx.x; i < quads; i += kPrCta) reinterpret_cast<float4 *>(s_y)[i] = __ldg(src + i);
    }
    const float dterm = pr_dangling(a.wsum, a.vblocks, s_red) * a.inv_n;
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.work_next = 0;
    if (S != PrStore::kLast) pr_dangling_sums(a.lane_cnt, a.vblocks, a.base + a.damping * (0.f + dterm), a.wsum_new);
    // one generic load, from shared or global memory as the lane's position
    // says: two loads behind a branch would each wait for the other's
    auto rank_of = [&](uint32_t i) {
        float v;
        const float *base = kHot && i < (uint32_t)a.hot ? s_y : a.y;
        asm volatile("ld.f32 %0, [%1];" : "=f"(v) : "l"(base + i) : "memory");  // not before the barrier above
        return v;
    };
    auto finish = [&](int64_t v, int64_t deg, float s) {
        const float xv = a.base + a.damping * (s + dterm);
        if (S == PrStore::kPrev) a.x_prev[v] = xv;
        if (S == PrStore::kLast) {
            a.x_out[v] = xv;
        } else if (deg > 0) {
            a.y_new[a.pos ? __ldg(a.pos + v) : (uint32_t)v] = xv / (float)deg;
        }
    };
    // units, the longest first: chunks of hub rows, rows of medium length,
    // groups of 32 consecutive rows for their short ones.  With few chunks (or
    // medium rows) for the warps there are, a unit is one of a chunk's eight
    // runs (or fewer than 32 rows): one warp's walk over 8192 arcs takes 30 us,
    // most of an iteration on a small graph (R-MAT with 60,000 vertices: 54 us
    // an iteration with whole units, 20 with these; with the runs split up to
    // four times as many chunks, s20 takes 129 us instead of 92).
    const unsigned warps = gridDim.x * (kPrCta / 32);
    const unsigned nchunks = (unsigned)a.hubs.count[1];
    const bool split = nchunks < warps / 4;
    const unsigned hub_units = split ? nchunks * kPrWarps : nchunks;
    const unsigned nmed = (unsigned)a.hubs.count[2];
    const unsigned med_rows = max(1u, min(32u, 2 * nmed / warps));
    const unsigned med_units = (nmed + med_rows - 1) / med_rows;
    const unsigned groups = (unsigned)((a.n + 31) / 32);
    const unsigned units = hub_units + med_units + (groups + a.per_claim - 1) / a.per_claim;
    constexpr int kB = 8;  // slabs in flight
    for (;;) {
        unsigned u = 0;
        if (lane == 0) u = atomicAdd(a.work, 1u);
        u = __shfl_sync(kFull, u, 0);
        if (u >= units) break;
        if (u < hub_units) {  // one chunk of a hub row, or one run of it
            const unsigned chunk = split ? u / kPrWarps : u;
            const uint32_t h = __ldg(a.hubs.chunk_hub + chunk);
            const int first = __ldg(a.hubs.first + h);
            const int64_t v = __ldg(a.hubs.row + h);
            const int64_t rb = __ldg(a.off + v), re = __ldg(a.off + v + 1);
            const int64_t cb = rb + (int64_t)((int)chunk - first) * kHubChunk;
            const int64_t ce = min(cb + (int64_t)kHubChunk, re);
            static_assert(kB == kPrWarps, "a step of a chunk is one slab of each run");
            // a step: one slab of each of the eight runs, or eight of the unit's run
            auto sum_part = [&](int64_t from, auto next_slab, auto next_step, auto add) {
                uint32_t c[kB];
                auto load = [&](int64_t i) {
#pragma unroll
                    for (int w = 0; w < kB; ++w) c[w] = i + w * next_slab < ce ? __ldcs(a.colx + i + w * next_slab) : 0u;
                };
                load(from);
                for (int64_t i = from; i - lane < ce; i += next_step) {
                    float r[kB];
#pragma unroll
                    for (int w = 0; w < kB; ++w) {
                        r[w] = 0.f;
                        if (i + w * next_slab < ce) r[w] = rank_of(c[w]);
                    }
                    load(i + next_step);  // the next step's, while these are on their way
#pragma unroll
                    for (int w = 0; w < kB; ++w) add(w, r[w]);
                }
            };
            float acc = 0.f;
            if (split) {
                sum_part(cb + lane + (u % kPrWarps) * 32, std::integral_constant<int, kPrThreads>{},
                         std::integral_constant<int, kPrThreads * kB>{}, [&](int, float r) { acc += r; });
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
            } else {
                float t[kB];
#pragma unroll
                for (int w = 0; w < kB; ++w) t[w] = 0.f;
                sum_part(cb + lane, std::integral_constant<int, 32>{}, std::integral_constant<int, kPrThreads>{},
                         [&](int w, float r) { t[w] += r; });
#pragma unroll
                for (int w = 0; w < kB; ++w) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) t[w] += __shfl_xor_sync(kFull, t[w], o);
                    acc += t[w];
                }
            }
            // the warp that sums the row's last part adds the parts in order
            const int parts = (int)((re - rb + kHubChunk - 1) / kHubChunk) * (split ? kPrWarps : 1);
            bool last = false;
            if (lane == 0) {
                __stcg(a.hubs.part + u, acc);
                __threadfence();
                last = atomicAdd(a.hubs.done + h, 1u) == (unsigned)parts - 1;
                __threadfence();
            }
            if (__shfl_sync(kFull, (int)last, 0)) {
                __syncwarp();  // a shuffle orders no memory: the lanes' reads below come after lane 0's fence
                const float *part = a.hubs.part + (size_t)first * (split ? kPrWarps : 1);
                const int nch = split ? parts / kPrWarps : parts;
                float s = 0.f;
                for (int c0 = 0; c0 < nch; c0 += 32) {  // a lane adds a chunk's runs
                    float one = 0.f;
                    if (c0 + lane < nch) {
                        if (split) {
                            const float4 *run = reinterpret_cast<const float4 *>(part + (size_t)(c0 + lane) * kPrWarps);
                            static_assert(kPrWarps == 8, "two loads are a chunk's runs");
                            const float4 x = __ldcg(run), y = __ldcg(run + 1);
                            one = ((((((x.x + x.y) + x.z) + x.w) + y.x) + y.y) + y.z) + y.w;
                        } else {
                            one = __ldcg(part + c0 + lane);
                        }
                    }
                    // (one after another, but the shuffles do not wait for the sums; 0 past the last)
#pragma unroll
                    for (int j = 0; j < 32; ++j) s += __shfl_sync(kFull, one, j);
                }
                if (lane == 0) {
                    a.hubs.done[h] = 0;
                    finish(v, re - rb, s);
                }
            }
            continue;
        }
        u -= hub_units;
        if (u < med_units) {
            // a row per lane; the rows' slabs of 32 arcs as one sequence, kB of them in flight
            const unsigned mi = u * med_rows + lane;
            int64_t v = -1, b = 0, e = 0;
            if (lane < med_rows && mi < nmed) {
                v = __ldg(a.medium + mi);
                b = __ldg(a.off + v);
                e = __ldg(a.off + v + 1);
            }
            int vs = (int)((e - b + 31) / 32);  // this row's slabs, then the slabs before it
            const int mine = vs;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, vs, o);
                if (lane >= o) vs += t;
            }
            const int total = __shfl_sync(kFull, vs, 31);
            vs -= mine;
            float s = 0.f, t = 0.f;
            for (int w0 = 0; w0 < total; w0 += 32) {  // 32 slabs: a lane locates one
                const int sl = w0 + lane;
                int k = 0;  // the row of slab sl: the last one that starts at or before it
#pragma unroll
                for (int step = 16; step >= 1; step >>= 1) {
                    const int sk = __shfl_sync(kFull, vs, k + step);
                    if (sk <= sl) k += step;
                }
                const int64_t rb = __shfl_sync(kFull, b, k), re = __shfl_sync(kFull, e, k);
                const int64_t at = rb + (int64_t)(sl - __shfl_sync(kFull, vs, k)) * 32;
                // arcs of the slab; bit 8: the row's last; its row
                const int meta = sl < total ? (int)min((int64_t)32, re - at) | (re - at <= 32 ? 256 : 0) | (k << 9) : 0;
                const int m = min(32, total - w0);
                uint32_t c[kB];
                int mn[kB], mc[kB];
                auto load = [&](int q0) {  // (slabs past the last have no arcs)
                    int64_t p[kB];
#pragma unroll
                    for (int q = 0; q < kB; ++q) {
                        p[q] = __shfl_sync(kFull, at, (q0 + q) & 31) + lane;
                        mn[q] = q0 + q < m ? __shfl_sync(kFull, meta, (q0 + q) & 31) : 0;
                    }
#pragma unroll
                    for (int q = 0; q < kB; ++q) c[q] = lane < (mn[q] & 255) ? __ldcs(a.colx + p[q]) : 0u;
                };
                load(0);
                for (int q0 = 0; q0 < m; q0 += kB) {
                    float r[kB];
#pragma unroll
                    for (int q = 0; q < kB; ++q) {
                        mc[q] = mn[q];
                        r[q] = 0.f;
                        if (lane < (mc[q] & 255)) r[q] = rank_of(c[q]);
                    }
                    if (q0 + kB < m) load(q0 + kB);  // the next slabs', while these are on their way
#pragma unroll
                    for (int q = 0; q < kB; ++q) {
                        t += r[q];
                        if (mc[q] & 256) {  // (warp-uniform) the row's fixed tree over the lanes
#pragma unroll
                            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
                            if (lane == (mc[q] >> 9)) s = t;
                            t = 0.f;
                        }
                    }
                }
            }
            if (v >= 0) finish(v, e - b, s);
            continue;
        }
        const int64_t g0 = (int64_t)(u - med_units) * a.per_claim;
        const int64_t g1 = min(g0 + a.per_claim, (int64_t)groups);
        int64_t nb = 0, ne = 0;
        auto load_rows = [&](int64_t g) {
            const int64_t v = g * 32 + lane;
            nb = ne = 0;
            if (v < a.n) {
                nb = __ldg(a.off + v);
                ne = __ldg(a.off + v + 1);
            }
        };
        load_rows(g0);
        for (int64_t g = g0; g < g1; ++g) {
            const int64_t v = g * 32 + lane;
            const int64_t b = nb, e = ne;
            if (g + 1 < g1) load_rows(g + 1);
            const int64_t deg = e - b;
            const bool shortr = deg <= kShortRow;
            // consecutive numbering of the short rows' arcs
            const int sdeg = shortr ? (int)deg : 0;
            int vs = sdeg;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, vs, o);
                if (lane >= o) vs += t;
            }
            const int total = __shfl_sync(kFull, vs, 31);
            vs -= sdeg;  // exclusive start of this row's arcs
            s_acc[warp][lane] = 0.f;
            const unsigned full = __ballot_sync(kFull, sdeg > 0);
            const int start = sdeg > 0 ? vs : INT_MIN;
            if (sdeg > 0) s_row[warp][__popc(full & lanemask_lt())] = make_longlong2(b - vs, lane);
            __syncwarp();
            constexpr int kS = 4;  // slabs in flight
            const unsigned le = lanemask_lt() | (1u << lane);
            int before = -1;  // rows that start before the slab, minus one
            for (int s0 = 0; s0 < total; s0 += 32 * kS) {
                uint32_t c[kS];
                unsigned starts[kS];  // lanes of the slab where a row starts
                int row[kS];
                float r[kS];
#pragma unroll
                for (int q = 0; q < kS; ++q) {
                    const int i = s0 + q * 32 + lane;
                    const unsigned rel = (unsigned)start - (unsigned)(s0 + q * 32);
                    starts[q] = __reduce_or_sync(kFull, rel < 32u ? 1u << rel : 0u);
                    const longlong2 at = s_row[warp][(before + __popc(starts[q] & le)) & 31];
                    before += __popc(starts[q]);
                    row[q] = (int)at.y;
                    c[q] = i < total ? __ldcs(a.colx + at.x + i) : 0u;
                }
#pragma unroll
                for (int q = 0; q < kS; ++q) {
                    r[q] = 0.f;
                    if (s0 + q * 32 + lane < total) r[q] = rank_of(c[q]);
                }
#pragma unroll
                for (int q = 0; q < kS; ++q) {
                    if (s0 + q * 32 >= total) break;  // warp-uniform
                    // lanes since the row's start in this slab
                    const unsigned m = starts[q] & le;
                    const int d = m ? lane - (31 - __clz((int)m)) : lane;
                    float val = r[q];
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const float t = __shfl_up_sync(kFull, val, o);
                        if (d >= o) val += t;
                    }
                    const int i = s0 + q * 32 + lane;
                    if (i < total && (lane == 31 || ((starts[q] >> (lane + 1)) & 1u) || i + 1 >= total))
                        s_acc[warp][row[q]] += val;
                    __syncwarp();
                }
            }
            const float s = s_acc[warp][lane];
            __syncwarp();
            if (v < a.n && shortr) finish(v, deg, s);
        }
    }
}

// FP64 partial L1 residual |x - x_prev| per CTA: a thread adds the vertices a
// grid apart, then a fixed tree over lanes and warps.  (A pass of its own, 8n
// bytes once per call: in the last iteration the rows a lane gets, and so the
// order of the sum, depend on the schedule.  The sum is exact, and any order
// gives the same, only while the terms' bits fit 53, which damping near 1 or
// very many vertices exceed.)  Bound by the FP64 units (R-MAT s22: 64 us with two
// conversions and two additions a vertex, against 5 for the bytes), so differences
// that are exact in FP32 are taken there and widened by their bits, which leaves
// one addition, and none where the value did not change.
__device__ __forceinline__ double widen(float f) {  // (double)f of a value that is not negative
    const uint32_t b = __float_as_uint(f);
    if (b - 0x00800000u < 0x7F000000u)  // a normal number: its exponent and fraction moved
        return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
    return (double)f;
}

__global__ void __launch_bounds__(kPrThreads) pr_residual_kernel(const float *__restrict__ x,
                                                                const float *__restrict__ x_prev, int64_t n,
                                                                double *__restrict__ parts) {
    constexpr int kPer = 4;
    __shared__ double s[kPrWarps];
    const int64_t stride = (int64_t)gridDim.x * kPrThreads;
    double res = 0.0;
    for (int64_t v = (int64_t)blockIdx.x * kPrThreads + threadIdx.x; v < n; v += stride * kPer) {
        float a[kPer], b[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            a[j] = v + j * stride < n ? __ldg(x + v + j * stride) : 0.f;
            b[j] = v + j * stride < n ? __ldg(x_prev + v + j * stride) : 0.f;
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) {  // (0 past the last vertex)
            const float d = fabsf(a[j] - b[j]);
            // within a factor of two the FP32 difference is exact (Sterbenz)
            if (!(a[j] >= 0.5f * b[j] && a[j] <= 2.f * b[j]))
                res += fabs((double)a[j] - (double)b[j]);
            else if (d != 0.f)
                res += widen(d);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) res += __shfl_xor_sync(kFull, res, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = res;
    __syncthreads();
    if (threadIdx.x == 0) {
        double br = 0.0;
        for (int i = 0; i < kPrWarps; ++i) br += s[i];
        parts[blockIdx.x] = br;
    }
}

// Hub rows and their chunk count, the rows of medium length (in whatever order
// the atomics give), and the degree histogram.
__global__ void __launch_bounds__(kPrThreads) pr_degrees_kernel(const int64_t *__restrict__ off, int64_t n, uint32_t *hubs,
                                                               uint32_t *medium, unsigned long long *counts,
                                                               unsigned int *hist) {
    __shared__ unsigned int s_hist[kDegBuckets];
    for (int i = threadIdx.x; i < kDegBuckets; i += blockDim.x) s_hist[i] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x; v0 < n; v0 += stride) {
        const int64_t v = v0 + threadIdx.x;
        const int64_t deg = v < n ? off[v + 1] - off[v] : 0;
        const bool med = deg > kShortRow && deg <= kHubRow;
        const unsigned m = __ballot_sync(kFull, med);
        unsigned long long base = 0;
        if (lane == 0 && m) base = atomicAdd(counts + 2, (unsigned long long)__popc(m));
        base = __shfl_sync(kFull, base, 0);
        if (med) medium[base + __popc(m & lanemask_lt())] = (uint32_t)v;
        if (deg > kHubRow) {
            hubs[atomicAdd(counts, 1ull)] = (uint32_t)v;
            atomicAdd(counts + 1, (unsigned long long)((deg + kHubChunk - 1) / kHubChunk));
        }
        if (v < n) atomicAdd(&s_hist[degree_bucket(deg)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kDegBuckets; i += blockDim.x)
        if (s_hist[i]) atomicAdd(hist + i, s_hist[i]);
}

// One CTA: each hub's first chunk (a running block scan over the hub list, 1024
// hubs at a time) and the hub of every chunk; and the first position of every
// degree bucket in y (in place of its count), largest degrees first.
__global__ void __launch_bounds__(1024) pr_hub_chunks_kernel(const int64_t *__restrict__ off,
                                                             const uint32_t *__restrict__ hubs,
                                                             const unsigned long long *__restrict__ counts, int *first,
                                                             uint32_t *chunk_hub, unsigned int *hist) {
    __shared__ int s_warp[32];
    __shared__ int s_run;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int num_hubs = (int)counts[0];
    if (threadIdx.x == 0) s_run = 0;
    if (warp == 0) {  // the buckets' first positions, largest degrees first
        constexpr int kPer = kDegBuckets / 32;
        unsigned int cnt[kPer], sum = 0;
        for (int i = 0; i < kPer; ++i) sum += cnt[i] = hist[kDegBuckets - 1 - (lane * kPer + i)];
        unsigned int inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int t = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += t;
        }
        unsigned int run = inc - sum;
        for (int i = 0; i < kPer; ++i) {
            hist[kDegBuckets - 1 - (lane * kPer + i)] = run;
            run += cnt[i];
        }
    }
    __syncthreads();
    for (int h0 = 0; h0 < num_hubs; h0 += 1024) {
        const int h = h0 + threadIdx.x;
        int nch = 0;
        if (h < num_hubs) {
            const uint32_t v = hubs[h];
            nch = (int)((off[v + 1] - off[v] + kHubChunk - 1) / kHubChunk);
        }
        int inc = nch;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) s_warp[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            const int wv = s_warp[lane];
            int wi = wv;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, wi, o);
                if (lane >= o) wi += t;
            }
            s_warp[lane] = wi - wv;
        }
        __syncthreads();
        int slot = s_run + s_warp[warp] + inc - nch;
        if (h < num_hubs) {
            first[h] = slot;
            for (int c = 0; c < nch; ++c) chunk_hub[slot + c] = (uint32_t)h;
        }
        slot += nch;
        __syncthreads();
        if (threadIdx.x == 1023) s_run = slot;  // the last thread's next slot is the running total
        __syncthreads();
    }
}

// Positions in y, by falling degree bucket (in any order inside one: the
// values move with them, the sums don't change).  A CTA counts a tile of
// vertices by bucket and takes its places with one atomic per bucket.
__global__ void __launch_bounds__(kPrThreads) pr_positions_kernel(const int64_t *__restrict__ off, int64_t n,
                                                                 unsigned int *next, uint32_t *__restrict__ pos) {
    constexpr int kPer = 8;
    __shared__ unsigned int s_cnt[kDegBuckets], s_base[kDegBuckets];
    const int64_t stride = (int64_t)gridDim.x * kPrThreads * kPer;
    for (int64_t v0 = (int64_t)blockIdx.x * kPrThreads * kPer; v0 < n; v0 += stride) {
        for (int i = threadIdx.x; i < kDegBuckets; i += kPrThreads) s_cnt[i] = 0;
        __syncthreads();
        int bucket[kPer];
        unsigned int rank[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int64_t v = v0 + j * kPrThreads + threadIdx.x;
            if (v < n) {
                bucket[j] = degree_bucket(off[v + 1] - off[v]);
                rank[j] = atomicAdd(&s_cnt[bucket[j]], 1u);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < kDegBuckets; i += kPrThreads)
            if (s_cnt[i]) s_base[i] = atomicAdd(next + i, s_cnt[i]);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int64_t v = v0 + j * kPrThreads + threadIdx.x;
            if (v < n) pos[v] = s_base[bucket[j]] + rank[j];
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kPrThreads) pr_heads_kernel(const uint32_t *__restrict__ col, int64_t nnz,
                                                             const uint32_t *__restrict__ pos,
                                                             uint32_t *__restrict__ colx) {
    constexpr int kPer = 8;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * kPer;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x * kPer + threadIdx.x; i0 < nnz; i0 += stride) {
        uint32_t c[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) c[j] = i0 + j * kPrThreads < nnz ? __ldg(col + i0 + j * kPrThreads) : 0u;
#pragma unroll
        for (int j = 0; j < kPer; ++j) c[j] = __ldg(pos + c[j]);
#pragma unroll
        for (int j = 0; j < kPer; ++j)
            if (i0 + j * kPrThreads < nnz) colx[i0 + j * kPrThreads] = c[j];
    }
}

// y0 = x0/d, x0 itself when the first iteration is the last, and the degree-0
// vertices of every virtual lane: virtual warp w sums the rows w * 32 + lane,
// then those a whole virtual grid further, and so on.
__global__ void __launch_bounds__(kPrThreads) pr_init_kernel(PrArgs a, float x0, bool store_x, uint32_t *lane_cnt) {
    const int64_t stride = (int64_t)a.vblocks * kPrThreads;
    const int64_t l = (int64_t)blockIdx.x * kPrThreads + threadIdx.x;  // grid: vblocks
    uint32_t cnt = 0;
    for (int64_t v = l; v < a.n; v += stride) {
        const int64_t deg = __ldg(a.off + v + 1) - __ldg(a.off + v);
        if (deg > 0) a.y_new[a.pos ? __ldg(a.pos + v) : (uint32_t)v] = x0 / (float)deg;
        else ++cnt;
        if (store_x) a.x_prev[v] = x0;
    }
    lane_cnt[l] = cnt;
    const int lane = threadIdx.x & 31;
    float t = 0.f;
    for (uint32_t k = cnt; k > 0; --k) t += x0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
    if (lane == 0) a.wsum_new[l >> 5] = t;
}

// one block: sum the per-block partials in a fixed order
template <typename T>
__global__ void __launch_bounds__(kPrThreads) reduce_parts_kernel(const T *__restrict__ parts, int count,
                                                                  T *__restrict__ out) {
    __shared__ T s[kPrThreads];
    T acc = 0;
    for (int i = threadIdx.x; i < count; i += kPrThreads) acc += parts[i];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int h = kPrThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = s[0];
}

// Iterations that pay for the positions and the translated heads: they take
// 0.66 ms on R-MAT s22 and save about 0.2 ms an iteration.
constexpr int kPrMinIters = 4;
// Vertices above which they pay: below, most of y stays in the L1 without them,
// which the copy in shared memory takes space from (50 iterations in us, with /
// without: complete graph of 4000 1664 / 1333, R-MAT with n = 8000 687 / 639,
// 30,000 1081 / 1013, 60,000 951 / 917, 100,000 1322 / 1323; 2^20 4570 / 6351).
constexpr int64_t kPrMinVertices = 3 * (int64_t)kPrHot;

sg_status pagerank(Ctx *c, const Graph *g, float damping, int iters, float *x_out, double *resid) {
    const int64_t n = g->n, nnz = g->nnz;
    *resid = 0.0;
    if (n == 0) return SG_OK;
    const int vblocks = (int)std::min<int64_t>((n + kPrThreads - 1) / kPrThreads, (int64_t)c->num_sms * 8);
    const size_t nn = (size_t)n;
    PrArgs a{};
    a.off = g->off;
    a.colx = g->col;
    a.n = n;
    a.base = (float)((1.0 - (double)damping) / (double)n);
    a.damping = damping;
    a.inv_n = (float)(1.0 / (double)n);
    a.vblocks = vblocks;
    a.x_out = x_out;
    // one allocation: the arrays below, each aligned to 256 bytes
    // (rows of each length class: by their arcs, and no more than there are rows)
    const size_t max_hubs = std::min(nn, (size_t)(nnz / kHubRow + 1));
    const size_t max_chunks = (size_t)(nnz / kHubChunk) + max_hubs;
    // parts: the chunks' runs while there are few chunks, the chunks otherwise
    const size_t max_parts = std::max(max_chunks, std::min(max_chunks, (size_t)c->num_sms * (kPrCta / 32) / 4) * kPrWarps);
    const int hot_cap = (int)std::min<int64_t>(kPrHot, n);
    size_t total = 0;
    auto room = [&](size_t bytes) {
        const size_t at = total;
        total += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t zero_at = room((4 + kDegBuckets / 2 + 1) * sizeof(unsigned long long));  // counts, hist, work
    const size_t done_at = room(max_hubs * sizeof(unsigned int));
    // y of the degree-0 vertices is never written: an arc into one, which only a
    // CSR that is not symmetric has, adds nothing
    const size_t y_at[2] = {room(sizeof(float) * (nn + 4)), room(sizeof(float) * (nn + 4))};
    const size_t zero_end = total;
    const size_t x_at = room(sizeof(float) * nn), res_at = room(sizeof(double) * ((size_t)vblocks + 1));
    const size_t cnt_at = room(sizeof(uint32_t) * (size_t)vblocks * kPrThreads);
    const size_t w_at[2] = {room(sizeof(float) * (size_t)vblocks * kPrWarps), room(sizeof(float) * (size_t)vblocks * kPrWarps)};
    const size_t hubs_at = room(sizeof(uint32_t) * max_hubs), first_at = room(sizeof(int) * max_hubs);
    const size_t med_at = room(sizeof(uint32_t) * std::min(nn, (size_t)(nnz / kShortRow + 1)));
    const size_t chunk_at = room(sizeof(uint32_t) * max_chunks), part_at = room(sizeof(float) * max_parts);
    char *buf = nullptr;
    uint32_t *pos = nullptr, *colx = nullptr;
    sg_status st = dalloc(c, (void **)&buf, total);
    if (st != SG_OK) return st;
    // positions and translated heads: 4 (n + nnz) bytes, without which y stays in vertex order
    bool hot = iters >= kPrMinIters && nnz > 0 && n > kPrMinVertices;
    if (hot && (dalloc(c, (void **)&pos, sizeof(uint32_t) * nn) != SG_OK ||
                dalloc(c, (void **)&colx, sizeof(uint32_t) * (size_t)nnz) != SG_OK)) {
        set_error("");
        dfree(c, pos);
        pos = nullptr;
        hot = false;
    }
    unsigned long long *counts = reinterpret_cast<unsigned long long *>(buf + zero_at);
    unsigned int *hist = reinterpret_cast<unsigned int *>(counts + 4), *work = hist + kDegBuckets;
    a.hubs = PrHubs{reinterpret_cast<uint32_t *>(buf + hubs_at), counts, reinterpret_cast<int *>(buf + first_at),
                    reinterpret_cast<uint32_t *>(buf + chunk_at), reinterpret_cast<float *>(buf + part_at),
                    reinterpret_cast<unsigned int *>(buf + done_at)};
    a.medium = reinterpret_cast<uint32_t *>(buf + med_at);
    a.x_prev = reinterpret_cast<float *>(buf + x_at);
    double *parts = reinterpret_cast<double *>(buf + res_at);  // of the residual, then their sum
    a.lane_cnt = reinterpret_cast<uint32_t *>(buf + cnt_at);
    a.hot = hot ? hot_cap : 0;
    a.pos = pos;
    float *y[2] = {reinterpret_cast<float *>(buf + y_at[0]), reinterpret_cast<float *>(buf + y_at[1])};
    float *w[2] = {reinterpret_cast<float *>(buf + w_at[0]), reinterpret_cast<float *>(buf + w_at[1])};
    auto release = [&]() {
        dfree(c, colx);
        dfree(c, pos);
        dfree(c, buf);
    };
    cudaError_t e = cudaMemsetAsync(buf + zero_at, 0, zero_end - zero_at, c->stream);
    {
        SG_LAUNCH(c, "pr_setup");
        pr_degrees_kernel<<<vblocks, kPrThreads, 0, c->stream>>>(g->off, n, const_cast<uint32_t *>(a.hubs.row),
                                                                const_cast<uint32_t *>(a.medium), counts, hist);
    }
    {
        SG_LAUNCH(c, "pr_setup");
        pr_hub_chunks_kernel<<<1, 1024, 0, c->stream>>>(g->off, a.hubs.row, counts, const_cast<int *>(a.hubs.first),
                                                        const_cast<uint32_t *>(a.hubs.chunk_hub), hist);
    }
    if (hot) {
        {
            SG_LAUNCH(c, "pr_setup");
            pr_positions_kernel<<<vblocks, kPrThreads, 0, c->stream>>>(g->off, n, hist, pos);
        }
        SG_LAUNCH(c, "pr_setup");
        const int64_t hb = std::min<int64_t>((nnz + kPrThreads * 8 - 1) / (kPrThreads * 8), (int64_t)c->num_sms * 8);
        pr_heads_kernel<<<(unsigned)hb, kPrThreads, 0, c->stream>>>(g->col, nnz, pos, colx);
        a.colx = colx;
    }
    a.y_new = y[0];
    a.wsum_new = w[0];
    {
        SG_LAUNCH(c, "pr_init");
        pr_init_kernel<<<vblocks, kPrThreads, 0, c->stream>>>(a, a.inv_n, iters == 1, const_cast<uint32_t *>(a.lane_cnt));
    }
    const int64_t groups = (n + 31) / 32;
    const int grid = (int)std::min<int64_t>(std::max<int64_t>(groups, nnz / kHubChunk), (int64_t)c->num_sms);
    // groups of a claim, which hide each other's first loads: up to four, where that
    // leaves each warp eight claims, or four where the rows are so short that little
    // else is in flight (50 iterations, two groups of a claim / one: a star of 2 M
    // leaves 2.09 / 2.91 ms, a geometric graph of 1.8 M with 18 arcs a row 9.63 / 9.50)
    const int64_t claims = nnz < 8 * n ? 4 : 8;
    a.per_claim = (int)std::max<int64_t>(1, std::min<int64_t>(4, groups / ((int64_t)grid * 32 * claims)));
    const size_t smem = hot ? sizeof(float) * (((size_t)hot_cap + 3) / 4 * 4) : 0;
    void (*k[2][3])(PrArgs) = {{pr_iter_kernel<false, PrStore::kNone>, pr_iter_kernel<false, PrStore::kPrev>,
                                pr_iter_kernel<false, PrStore::kLast>},
                               {pr_iter_kernel<true, PrStore::kNone>, pr_iter_kernel<true, PrStore::kPrev>,
                                pr_iter_kernel<true, PrStore::kLast>}};
    // the limit is the function's, shared by all threads and contexts: always the
    // same value, never this call's
    for (int i = 0; i < 3 && hot && e == cudaSuccess; ++i)
        e = cudaFuncSetAttribute(k[1][i], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(float) * kPrHot));
    if (e != cudaSuccess) {
        release();
        return cuda_fail(e, "PageRank setup");
    }
    for (int it = 0; it < iters; ++it) {
        const int in = it & 1, s = it == iters - 1 ? 2 : (it == iters - 2 ? 1 : 0);
        a.y = y[in];
        a.y_new = y[in ^ 1];
        a.wsum = w[in];
        a.wsum_new = w[in ^ 1];
        a.work = work + in;
        a.work_next = work + (in ^ 1);
        SG_LAUNCH(c, "pr_iter");
        k[hot][s]<<<grid, kPrCta, smem, c->stream>>>(a);
    }
    {
        SG_LAUNCH(c, "pr_reduce");
        pr_residual_kernel<<<vblocks, kPrThreads, 0, c->stream>>>(x_out, a.x_prev, n, parts);
    }
    {
        SG_LAUNCH(c, "pr_reduce");
        reduce_parts_kernel<double><<<1, kPrThreads, 0, c->stream>>>(parts, vblocks, parts + vblocks);
    }
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->h_pinned, parts + vblocks, sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e == cudaSuccess) std::memcpy(resid, c->h_pinned, sizeof(double));
    release();
    return e == cudaSuccess ? SG_OK : cuda_fail(e, "PageRank");
}

// ---------------------------------------------------------------------- KL
__global__ void __launch_bounds__(kPrThreads) sum2_kernel(const float *__restrict__ P, const float *__restrict__ Q,
                                                          int64_t n, double *__restrict__ parts) {
    __shared__ double s[2][kPrThreads];
    double a = 0.0, b = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kPrThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kPrThreads) {
        a += (double)P[i];
        b += (double)Q[i];
    }
    s[0][threadIdx.x] = a;
    s[1][threadIdx.x] = b;
    __syncthreads();
    for (int h = kPrThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            s[0][threadIdx.x] += s[0][threadIdx.x + h];
            s[1][threadIdx.x] += s[1][threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        parts[2 * blockIdx.x] = s[0][0];
        parts[2 * blockIdx.x + 1] = s[1][0];
    }
}

// Per-vertex terms in FP32, summed in FP64.  With p_i = P_i / S_P and
// q_i = Q_i / S_Q (S the FP64 sums), sum_i p_i log2(p_i / q_i)
//   = (sum_i P_i log2(P_i / Q_i)) / S_P + log2(S_Q / S_P),
// so a term is the FP32 product P_i * log2f(P_i / Q_i) of the raw values and
// the normalisation enters once, in FP64, after the sum.
__global__ void __launch_bounds__(kPrThreads) kl_terms_kernel(const float *__restrict__ P, const float *__restrict__ Q,
                                                              int64_t n, double *__restrict__ parts) {
    __shared__ double s[kPrThreads];
    double acc = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kPrThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kPrThreads) {
        const float p = P[i];
        if (p > 0.f) acc += (double)(p * log2f(p / Q[i]));
    }
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int h = kPrThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) parts[blockIdx.x] = s[0];
}

__global__ void reduce_pairs_kernel(const double *__restrict__ parts, int count, double *__restrict__ out) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int i = 0; i < count; ++i) {
            a += parts[2 * i];
            b += parts[2 * i + 1];
        }
        out[0] = a;
        out[1] = b;
    }
}

sg_status kl_divergence(Ctx *c, int64_t n, const float *P, const float *Q, double *kl) {
    *kl = 0.0;
    if (n == 0) return SG_OK;
    const int blocks = (int)std::min<int64_t>((n + kPrThreads - 1) / kPrThreads, (int64_t)c->num_sms * 4);
    double *buf = nullptr;
    sg_status st = dalloc(c, (void **)&buf, sizeof(double) * (3 * (size_t)blocks + 4));
    if (st != SG_OK) return st;
    double *pairs = buf, *sums = buf + 2 * blocks, *terms = sums + 2, *tot = terms + blocks;
    {
        SG_LAUNCH(c, "kl_sums");
        sum2_kernel<<<blocks, kPrThreads, 0, c->stream>>>(P, Q, n, pairs);
    }
    {
        SG_LAUNCH(c, "kl_reduce");
        reduce_pairs_kernel<<<1, 32, 0, c->stream>>>(pairs, blocks, sums);
    }
    {
        SG_LAUNCH(c, "kl_terms");
        kl_terms_kernel<<<blocks, kPrThreads, 0, c->stream>>>(P, Q, n, terms);
    }
    {
        SG_LAUNCH(c, "kl_reduce");
        reduce_parts_kernel<double><<<1, kPrThreads, 0, c->stream>>>(terms, blocks, tot);
    }
    SG_CUDA(cudaGetLastError());
    // sums (S_P, S_Q) and the term total are adjacent: one copy
    static_assert(sizeof(double) == sizeof(int64_t), "pinned scratch holds doubles");
    SG_CUDA(cudaMemcpyAsync(c->h_pinned, sums, sizeof(double) * 2, cudaMemcpyDeviceToHost, c->stream));
    SG_CUDA(cudaMemcpyAsync(c->h_pinned + 2, tot, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    SG_CUDA(cudaStreamSynchronize(c->stream));
    double h[3];
    std::memcpy(h, c->h_pinned, sizeof(h));
    // FP64: the sum of the FP32 terms, normalised (see kl_terms_kernel)
    *kl = (h[0] > 0.0 && h[1] > 0.0) ? h[2] / h[0] + std::log2(h[1] / h[0]) : 0.0;
    dfree(c, buf);
    return SG_OK;
}

// ---------------------------------------------------------------------- CC
__global__ void cc_init_kernel(uint32_t *parent, int64_t n) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        parent[v] = (uint32_t)v;
}

__device__ __forceinline__ uint32_t cc_find(uint32_t *parent, uint32_t v) {
    uint32_t p = parent[v];
    while (p != v) {
        const uint32_t gp = parent[p];
        if (gp != p) parent[v] = gp;  // path halving; gp is still an ancestor of v
        v = p;
        p = gp;
    }
    return v;
}

constexpr int kCcSample = 2;     // neighbours every vertex links first
constexpr int kCcProbes = 1024;  // sampled vertices that name the giant component

// join the trees of x and y: the larger root hooks under the smaller
__device__ __forceinline__ void cc_link(uint32_t *parent, uint32_t x, uint32_t y) {
    uint32_t rx = cc_find(parent, x), ry = cc_find(parent, y);
    while (rx != ry) {
        const uint32_t hi = rx > ry ? rx : ry, lo = rx > ry ? ry : rx;
        const uint32_t old = atomicCAS(parent + hi, hi, lo);
        if (old == hi) break;
        rx = cc_find(parent, hi);
        ry = cc_find(parent, lo);
    }
}

// thread per vertex: link its first kCcSample neighbours
__global__ void cc_sample_kernel(const int64_t *__restrict__ off, const uint32_t *__restrict__ col, int64_t n,
                                 uint32_t *parent) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = __ldg(off + x), e = __ldg(off + x + 1);
        for (int64_t i = b; i < e && i < b + kCcSample; ++i) cc_link(parent, (uint32_t)x, __ldg(col + i));
    }
}

__global__ void cc_compress_kernel(uint32_t *parent, int64_t n) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        parent[v] = cc_find(parent, (uint32_t)v);
}

// roots of kCcProbes vertices spread over [0, n) by a fixed multiplicative hash
__global__ void cc_probe_kernel(const uint32_t *parent, int64_t n, uint32_t *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kCcProbes) {
        const uint64_t v = ((uint64_t)((uint32_t)i * 0x9E3779B1u) * (uint64_t)n) >> 32;
        out[i] = parent[v];
    }
}

// warp per row outside the giant component: link the neighbours after the sampled ones
__global__ void cc_rest_kernel(const int64_t *__restrict__ off, const uint32_t *__restrict__ col, int64_t n,
                               uint32_t *parent, uint32_t giant) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t x = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp; x < n; x += nw) {
        const int64_t b = __ldg(off + x), e = __ldg(off + x + 1);
        if (e - b <= kCcSample) continue;
        uint32_t r = 0;
        if (lane == 0) r = cc_find(parent, (uint32_t)x);
        if (__shfl_sync(0xFFFFFFFFu, r, 0) == giant) continue;
        for (int64_t i = b + kCcSample + lane; i < e; i += 32) cc_link(parent, (uint32_t)x, __ldg(col + i));
    }
}

__global__ void __launch_bounds__(256) cc_finish_kernel(uint32_t *parent, int64_t n, unsigned long long *roots) {
    unsigned long long cnt = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t r = cc_find(parent, (uint32_t)v);
        if (r == (uint32_t)v) ++cnt;
    }
    cnt = warp_sum(cnt);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(roots, cnt);
}

__global__ void cc_label_kernel(const uint32_t *parent, int64_t n, uint32_t *labels) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        uint32_t r = parent[v];
        while (parent[r] != r) r = parent[r];
        labels[v] = r;
    }
}

sg_status cc_count(Ctx *c, const Graph *g, int64_t *count, uint32_t *labels) {
    *count = 0;
    const int64_t n = g->n;
    if (n == 0) return SG_OK;
    uint32_t *parent = nullptr;
    unsigned long long *roots = nullptr;
    sg_status st = dalloc(c, (void **)&parent, sizeof(uint32_t) * (size_t)n);
    // roots: the root count, then kCcProbes sampled roots
    if (st == SG_OK) st = dalloc(c, (void **)&roots, sizeof(unsigned long long) + sizeof(uint32_t) * kCcProbes);
    if (st != SG_OK) {
        dfree(c, parent);
        return st;
    }
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, (int64_t)c->num_sms * 8);
    SG_CUDA(cudaMemsetAsync(roots, 0, sizeof(unsigned long long), c->stream));
    {
        SG_LAUNCH(c, "cc_init");
        cc_init_kernel<<<blocks, 256, 0, c->stream>>>(parent, n);
    }
    {
        SG_LAUNCH(c, "cc_sample");
        cc_sample_kernel<<<blocks, 256, 0, c->stream>>>(g->off, g->col, n, parent);
    }
    {
        SG_LAUNCH(c, "cc_compress");
        cc_compress_kernel<<<blocks, 256, 0, c->stream>>>(parent, n);
    }
    {
        SG_LAUNCH(c, "cc_probe");
        cc_probe_kernel<<<(kCcProbes + 255) / 256, 256, 0, c->stream>>>(parent, n, reinterpret_cast<uint32_t *>(roots + 1));
    }
    SG_CUDA(cudaGetLastError());
    SG_CUDA(cudaMemcpyAsync(c->h_pinned, roots + 1, sizeof(uint32_t) * kCcProbes, cudaMemcpyDeviceToHost, c->stream));
    SG_CUDA(cudaStreamSynchronize(c->stream));
    uint32_t giant = 0;
    {
        // the most frequent root among the probes (ties: the smaller root)
        std::vector<uint32_t> pr(kCcProbes);
        std::memcpy(pr.data(), c->h_pinned, sizeof(uint32_t) * kCcProbes);
        std::sort(pr.begin(), pr.end());
        int best = 0;
        for (int i = 0; i < kCcProbes;) {
            int j = i;
            while (j < kCcProbes && pr[j] == pr[i]) ++j;
            if (j - i > best) { best = j - i; giant = pr[i]; }
            i = j;
        }
    }
    {
        SG_LAUNCH(c, "cc_rest");
        const int hb = (int)std::min<int64_t>((n + 7) / 8, (int64_t)c->num_sms * 8);
        cc_rest_kernel<<<hb, 256, 0, c->stream>>>(g->off, g->col, n, parent, giant);
    }
    {
        SG_LAUNCH(c, "cc_finish");
        cc_finish_kernel<<<blocks, 256, 0, c->stream>>>(parent, n, roots);
    }
    if (labels) {
        SG_LAUNCH(c, "cc_label");
        cc_label_kernel<<<blocks, 256, 0, c->stream>>>(parent, n, labels);
    }
    SG_CUDA(cudaGetLastError());
    SG_CUDA(cudaMemcpyAsync(c->h_pinned, roots, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream));
    SG_CUDA(cudaStreamSynchronize(c->stream));
    unsigned long long r = 0;
    std::memcpy(&r, c->h_pinned, sizeof(r));
    *count = (int64_t)r;
    dfree(c, parent);
    dfree(c, roots);
    return SG_OK;
}

// ------------------------------------------------------ BFS levels (Sec. 5.3)
// Level-synchronous BFS over an int32 level array (-1 = unreached).  Each step
// is top-down (the frontier pushes L + 1 into unreached neighbours) or, once
// the frontier holds more than n/32 vertices, bottom-up (every unreached
// vertex looks for a neighbour on level L) -- the direction switch of Beamer,
// Asanovic and Patterson (SC'12).  Concurrent writes of L + 1 to one entry
// store the same value, so no atomics are needed; levels are unique, whatever
// the order of the writes.
__global__ void __launch_bounds__(256) bfs_top_down_kernel(const int64_t *__restrict__ off,
                                                           const uint32_t *__restrict__ col, int64_t n,
                                                           int *level, int L) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t base = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base < n;
         base += nw * 32) {
        const int64_t v = base + lane;
        unsigned fm = __ballot_sync(kFull, v < n && level[v] == L);
        while (fm) {
            const int src = __ffs(fm) - 1;
            fm &= fm - 1;
            const int64_t x = base + src;
            const int64_t o = __ldg(off + x), d = __ldg(off + x + 1) - o;
            for (int64_t i = lane; i < d; i += 32) {
                const uint32_t y = __ldg(col + o + i);
                if (level[y] < 0) level[y] = L + 1;
            }
        }
    }
}

__global__ void __launch_bounds__(256) bfs_bottom_up_kernel(const int64_t *__restrict__ off,
                                                            const uint32_t *__restrict__ col, int64_t n,
                                                            int *level, int L) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        if (level[v] >= 0) continue;
        const int64_t e = __ldg(off + v + 1);
        for (int64_t i = __ldg(off + v); i < e; ++i)
            if (level[__ldg(col + i)] == L) {
                level[v] = L + 1;
                break;
            }
    }
}

__global__ void __launch_bounds__(256) count_level_kernel(const int *__restrict__ level, int64_t n, int L,
                                                          unsigned long long *cnt) {
    unsigned long long k = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) k += level[v] == L;
    k = warp_sum(k);
    if ((threadIdx.x & 31) == 0 && k) atomicAdd(cnt, k);
}

__global__ void set_root_kernel(int *level, int64_t root) { level[root] = 0; }

sg_status bfs_levels(Ctx *c, const Graph *g, int64_t root, int *level) {
    if (g->n == 0) return SG_OK;
    SG_CUDA(cudaMemsetAsync(level, 0xFF, sizeof(int) * (size_t)g->n, c->stream));
    if (root < 0 || root >= g->n) return SG_OK;  // nothing is reached
    {
        SG_LAUNCH(c, "bfs_root");
        set_root_kernel<<<1, 1, 0, c->stream>>>(level, root);
    }
    unsigned long long *cnt = nullptr;
    sg_status st = dalloc(c, (void **)&cnt, sizeof(unsigned long long));
    if (st != SG_OK) return st;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((g->n + 255) / 256, (int64_t)c->num_sms * 8));
    unsigned long long frontier = 1;
    for (int L = 0; frontier > 0 && st == SG_OK; ++L) {
        if (L > (int)std::min<int64_t>(g->n, INT32_MAX - 1)) { st = fail(SG_ERR_CUDA, "BFS did not terminate"); break; }
        if (frontier * 32 > (unsigned long long)g->n) {
            SG_LAUNCH(c, "bfs_step");
            bfs_bottom_up_kernel<<<(unsigned)blocks, 256, 0, c->stream>>>(g->off, g->col, g->n, level, L);
        } else {
            SG_LAUNCH(c, "bfs_step");
            bfs_top_down_kernel<<<(unsigned)blocks, 256, 0, c->stream>>>(g->off, g->col, g->n, level, L);
        }
        if (cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), c->stream) != cudaSuccess) {
            st = cuda_fail(cudaGetLastError(), "cudaMemsetAsync");
            break;
        }
        {
            SG_LAUNCH(c, "bfs_count");
            count_level_kernel<<<(unsigned)blocks, 256, 0, c->stream>>>(level, g->n, L + 1, cnt);
        }
        if (cudaGetLastError() != cudaSuccess) { st = fail(SG_ERR_CUDA, "BFS launch"); break; }
        if (cudaMemcpyAsync(c->h_pinned, cnt, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(c->stream) != cudaSuccess) {
            st = cuda_fail(cudaGetLastError(), "BFS frontier count");
            break;
        }
        frontier = c->h_pinned[0];
    }
    dfree(c, cnt);
    return st;
}

// |E_cr| (Sec. 5.3): undirected edges joining BFS levels L and L + 1, each
// counted once from its lower end.
__global__ void __launch_bounds__(256) critical_kernel(const int64_t *__restrict__ off,
                                                       const uint32_t *__restrict__ col, int64_t n,
                                                       const int *__restrict__ level, unsigned long long *cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    unsigned long long k = 0;
    for (int64_t base = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base < n;
         base += nw * 32) {
        const int64_t v = base + lane;
        const int lv = v < n ? __ldg(level + v) : -1;
        unsigned fm = __ballot_sync(kFull, lv >= 0);
        while (fm) {
            const int src = __ffs(fm) - 1;
            fm &= fm - 1;
            const int64_t x = base + src;
            const int lx = __shfl_sync(kFull, lv, src);
            const int64_t o = __ldg(off + x), d = __ldg(off + x + 1) - o;
            for (int64_t i = lane; i < d; i += 32) k += __ldg(level + __ldg(col + o + i)) == lx + 1;
        }
    }
    k = warp_sum(k);
    if (lane == 0 && k) atomicAdd(cnt, k);
}

sg_status critical_edges(Ctx *c, const Graph *g, int64_t root, int64_t *count) {
    *count = 0;
    if (g->n == 0) return SG_OK;
    int *level = nullptr;
    unsigned long long *cnt = nullptr;
    sg_status st = dalloc(c, (void **)&level, sizeof(int) * (size_t)g->n);
    if (st == SG_OK) st = dalloc(c, (void **)&cnt, sizeof(unsigned long long));
    if (st == SG_OK) st = bfs_levels(c, g, root, level);
    if (st == SG_OK && cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), c->stream) != cudaSuccess)
        st = cuda_fail(cudaGetLastError(), "cudaMemsetAsync");
    if (st == SG_OK) {
        const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((g->n + 255) / 256, (int64_t)c->num_sms * 8));
        SG_LAUNCH(c, "critical_edges");
        critical_kernel<<<(unsigned)blocks, 256, 0, c->stream>>>(g->off, g->col, g->n, level, cnt);
        if (cudaGetLastError() != cudaSuccess) st = fail(SG_ERR_CUDA, "critical_edges launch");
    }
    if (st == SG_OK) {
        if (cudaMemcpyAsync(c->h_pinned, cnt, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(c->stream) != cudaSuccess)
            st = cuda_fail(cudaGetLastError(), "critical_edges read");
        else
            *count = (int64_t)c->h_pinned[0];
    }
    dfree(c, level);
    dfree(c, cnt);
    return st;
}

// ----------------------------------------------- A_REN (Sec. 5.2.2)
// Edges {u,v} of G (each once, from its smaller end) whose endpoint scores
// change relative order: sign(x_u - x_v) != sign(y_u - y_v), compared in the
// scores' own type.
template <typename T>
__device__ __forceinline__ int order_sign(T a, T b) {
    return (int)(a > b) - (int)(a < b);
}

template <typename T>
__global__ void __launch_bounds__(256) reordered_kernel(const int64_t *__restrict__ off,
                                                        const uint32_t *__restrict__ col, int64_t n,
                                                        const T *__restrict__ x, const T *__restrict__ y,
                                                        unsigned long long *cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    unsigned long long k = 0;
    for (int64_t u = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < n; u += nw) {
        const int64_t o = __ldg(off + u), d = __ldg(off + u + 1) - o;
        const T xu = x[u], yu = y[u];
        for (int64_t i = lane; i < d; i += 32) {
            const uint32_t v = __ldg(col + o + i);
            if ((int64_t)v > u) k += order_sign(xu, x[v]) != order_sign(yu, y[v]);
        }
    }
    k = warp_sum(k);
    if (lane == 0 && k) atomicAdd(cnt, k);
}

template <typename T>
sg_status reordered_neighbours(Ctx *c, const Graph *g, const T *x, const T *y, int64_t *count) {
    *count = 0;
    if (g->n == 0) return SG_OK;
    unsigned long long *cnt = nullptr;
    sg_status st = dalloc(c, (void **)&cnt, sizeof(unsigned long long));
    if (st == SG_OK && cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), c->stream) != cudaSuccess)
        st = cuda_fail(cudaGetLastError(), "cudaMemsetAsync");
    if (st == SG_OK) {
        const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((g->n + 7) / 8, (int64_t)c->num_sms * 8));
        SG_LAUNCH(c, "reordered");
        reordered_kernel<T><<<(unsigned)blocks, 256, 0, c->stream>>>(g->off, g->col, g->n, x, y, cnt);
        if (cudaGetLastError() != cudaSuccess) st = fail(SG_ERR_CUDA, "reordered launch");
    }
    if (st == SG_OK) {
        if (cudaMemcpyAsync(c->h_pinned, cnt, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(c->stream) != cudaSuccess)
            st = cuda_fail(cudaGetLastError(), "reordered read");
        else
            *count = (int64_t)c->h_pinned[0];
    }
    dfree(c, cnt);
    return st;
}
template sg_status reordered_neighbours<float>(Ctx *, const Graph *, const float *, const float *, int64_t *);
template sg_status reordered_neighbours<unsigned long long>(Ctx *, const Graph *, const unsigned long long *,
                                                            const unsigned long long *, int64_t *);

// The vertex of largest degree (smallest id on ties): the default BFS root.
__global__ void max_degree_kernel(const int64_t *__restrict__ off, int64_t n, unsigned long long *best) {
    unsigned long long b = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const unsigned long long d = (unsigned long long)(off[v + 1] - off[v]);
        const unsigned long long key = (d << 32) | (0xFFFFFFFFull - (unsigned long long)v);
        b = key > b ? key : b;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(kFull, b, o);
        b = t > b ? t : b;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(best, b);
}

sg_status max_degree_vertex(Ctx *c, const Graph *g, int64_t *v) {
    *v = -1;
    if (g->n == 0) return SG_OK;
    unsigned long long *best = nullptr;
    sg_status st = dalloc(c, (void **)&best, sizeof(unsigned long long));
    if (st == SG_OK && cudaMemsetAsync(best, 0, sizeof(unsigned long long), c->stream) != cudaSuccess)
        st = cuda_fail(cudaGetLastError(), "cudaMemsetAsync");
    if (st == SG_OK) {
        const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((g->n + 255) / 256, (int64_t)c->num_sms * 8));
        SG_LAUNCH(c, "max_degree");
        max_degree_kernel<<<(unsigned)blocks, 256, 0, c->stream>>>(g->off, g->n, best);
        if (cudaGetLastError() != cudaSuccess) st = fail(SG_ERR_CUDA, "max_degree launch");
    }
    if (st == SG_OK) {
        if (cudaMemcpyAsync(c->h_pinned, best, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream) !=
                cudaSuccess ||
            cudaStreamSynchronize(c->stream) != cudaSuccess)
            st = cuda_fail(cudaGetLastError(), "max_degree read");
        else
            *v = (int64_t)(0xFFFFFFFFull - (c->h_pinned[0] & 0xFFFFFFFFull));
    }
    dfree(c, best);
    return st;
}


// ---------------------------------------------------------------- validate
__global__ void validate_kernel(const int64_t *__restrict__ off, const uint32_t *__restrict__ col, int64_t n,
                                int64_t nnz, int *err) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = off[x], e = off[x + 1];
        bool bad = b < 0 || (x == 0 && b != 0) || e < b || (x == n - 1 && e != nnz) || e > nnz;
        for (int64_t i = b; !bad && i < e; ++i) {
            const uint32_t y = col[i];
            if (y >= (uint64_t)n || y == (uint32_t)x || (i > b && col[i - 1] >= y)) {
                bad = true;
                break;
            }
            // the reverse arc must exist
            const int64_t yb = off[y], ye = off[y + 1];
            if (yb < 0 || ye > nnz || ye < yb) { bad = true; break; }
            const int64_t k = lower_bound_u32(col, yb, ye, (uint32_t)x);
            if (k >= ye || col[k] != (uint32_t)x) bad = true;
        }
        if (bad) atomicExch(err, (int)kDevBadGraph);
    }
}

sg_status validate_graph(Ctx *c, const Graph *g) {
    if (g->n == 0) {
        if (g->nnz != 0) return fail(SG_ERR_INVALID_GRAPH, "an empty vertex set cannot hold arcs");
        return SG_OK;
    }
    const int blocks = (int)std::min<int64_t>((g->n + 255) / 256, (int64_t)c->num_sms * 8);
    {
        SG_LAUNCH(c, "validate");
        validate_kernel<<<blocks, 256, 0, c->stream>>>(g->off, g->col, g->n, g->nnz, c->d_err);
    }
    SG_CUDA(cudaGetLastError());
    return check_device_error(c);
}

}  // namespace sg
