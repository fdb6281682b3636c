// Grouping a graph's edges by a vertex id, in two partition passes staged in
// shared memory: the counting sort of the graph build.
//
// A counting sort with one global atomic and one scattered store per edge
// and array is bound by L2 transactions: on R-MAT 22 (67 M edges) 1.1 ms per
// histogram, 2.8 ms for the scatter into rows, 1.9 ms for the symmetrised
// copy's.  Here a tile of kPartTile edges is ranked in shared memory and
// written out in runs:
//   pass 1  by the id's high bits into buckets of 2^low_bits consecutive ids;
//   pass 2  each bucket's tiles by the low bits, i.e. by vertex, to the
//           vertex's final place.
// A tile counts its edges per digit with shared-memory atomics, reserves a
// run per digit with one global atomic each, and writes the runs in order, so
// that a run of r edges costs about r / 8 sectors per array instead of r.
// Both passes cut the edges into tiles of equal size whatever the digits, so
// that the few vertices that hold most edges of a skewed graph neither
// unbalance the work nor contend for a global counter.  The order of edges
// within a vertex is that of the atomics.
// R-MAT 22, with the weights: histogram 0.14 ms, pass 1 0.61 (1.47 GB of DRAM,
// 2.4 TB/s; a third of the stalls are shared memory's), counts 0.16, pass 2 1.09
// (1.29 GB; the warps wait for the random read of the renumbering, an edge
// each: 0.60 without one); pass 1 and 2 without the weights 0.45 and 0.57.
#pragma once

#include <algorithm>

#include "fg_internal.cuh"

namespace fg {
namespace {

constexpr int kPartThreads = 1024;
constexpr int kPartPer = 8;                             // edges a thread
constexpr int kPartTile = kPartThreads * kPartPer;      // 8192
constexpr int kPartRankBits = 13;                       // a rank within a tile
static_assert(kPartTile == 1 << kPartRankBits, "ranks take kPartRankBits");
// graphs with fewer edges, or more vertices than 4096 buckets of 4096 ids,
// keep the one-pass counting sort.  (A tile's runs shorten with the number of
// buckets; 1024 ids a bucket at least keep their number low on small graphs.)
constexpr int64_t kPartMinEdges = 1 << 20;
constexpr int32_t kPartMaxVertices = 1 << 24;
constexpr int kPartMinLow = 10, kPartMaxLow = 12;
constexpr int kPartMaxBuckets = kPartMaxVertices >> kPartMaxLow;

// How the ids 0..n-1 are cut: buckets of 2^low ids; sub-digits are the low
// bits, and below them the flag bit, if the edges carry one (flag = 1).
struct PartShape {
    int low = 0, nb = 0, flag = 0;
    __host__ __device__ int sub() const { return 1 << (low + flag); }
    __host__ __device__ int64_t counters() const { return (int64_t)nb << (low + flag); }
};
inline PartShape part_shape(int32_t n, int flag) {
    int bits = 1;
    while (((int64_t)1 << bits) < n) bits++;
    PartShape s;
    s.low = std::max(kPartMinLow, std::min(kPartMaxLow, bits - 11));
    s.nb = (int)(((int64_t)n + (1 << s.low) - 1) >> s.low);
    s.flag = flag;
    return s;
}
inline bool part_usable(int32_t n, int64_t m) { return m >= kPartMinEdges && n <= kPartMaxVertices; }

// Per grouping: edges per bucket, then the bucket's start; its pass-1 cursor;
// the first pass-2 tile of each bucket.
struct PartPlan {
    uint32_t *start = nullptr;    // [nb + 1]
    uint32_t *cursor = nullptr;   // [nb]
    uint32_t *tile0 = nullptr;    // [nb + 1]
};

// Edges per bucket of one or two id arrays (hist_t: of t), validated on the
// way (VALIDATE: ids inside [0, n), weights not negative; an edge with a bad
// id is not counted), with the sum of the weights.
template <bool VALIDATE>
__global__ void __launch_bounds__(kPartThreads)
    k_part_hist(int64_t m, int32_t n, const int32_t *__restrict__ s, const int32_t *__restrict__ t,
                const int32_t *__restrict__ w, PartShape sh, uint32_t *hist_s, uint32_t *hist_t, int *flags,
                unsigned long long *wsum) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *hs = reinterpret_cast<uint32_t *>(smem), *ht = hs + sh.nb;
    for (int i = threadIdx.x; i < 2 * sh.nb; i += kPartThreads) hs[i] = 0;
    __syncthreads();
    int bad = 0;
    unsigned long long sum = 0;
    const int64_t step = (int64_t)gridDim.x * kPartThreads;
    for (int64_t e0 = blockIdx.x * (int64_t)kPartThreads + threadIdx.x; e0 < m; e0 += 4 * step) {
        int32_t x[4], y[4], z[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int64_t e = e0 + j * step;
            x[j] = e < m ? __ldg(s + e) : 0;
            y[j] = t && e < m ? __ldg(t + e) : 0;
            z[j] = w && e < m ? __ldg(w + e) : 0;
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            if (e0 + j * step >= m) break;
            if (VALIDATE) {
                if (z[j] < 0) bad |= 2;
                if ((uint32_t)x[j] >= (uint32_t)n || (uint32_t)y[j] >= (uint32_t)n) {
                    bad |= 1;
                    continue;
                }
                sum += (uint32_t)z[j];
            }
            atomicAdd(hs + (x[j] >> sh.low), 1u);
            if (t) atomicAdd(ht + (y[j] >> sh.low), 1u);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < sh.nb; i += kPartThreads) {
        if (hs[i]) atomicAdd(hist_s + i, hs[i]);
        if (t && ht[i]) atomicAdd(hist_t + i, ht[i]);
    }
    if (VALIDATE) {
        bad = __reduce_or_sync(0xffffffffu, bad);
        if (bad && lane_id() == 0) atomicOr(flags, bad);
        sum = warp_sum(sum);
        if (sum && lane_id() == 0) atomicAdd(wsum, sum);
    }
}

// One CTA: exclusive prefix sums of the buckets' sizes (hist) and tiles.
__global__ void __launch_bounds__(1024) k_part_plan(const uint32_t *hist, int nb, PartPlan p) {
    __shared__ uint32_t s_sum[2][32];
    uint32_t run = 0, trun = 0;
    for (int b0 = 0; b0 < nb; b0 += 1024) {
        const int b = b0 + (int)threadIdx.x;
        const uint32_t c = b < nb ? hist[b] : 0u, tc = (c + kPartTile - 1) / kPartTile;
        const uint32_t ci = warp_inclusive_scan(c), ti = warp_inclusive_scan(tc);
        if (lane_id() == 31) {
            s_sum[0][threadIdx.x >> 5] = ci;
            s_sum[1][threadIdx.x >> 5] = ti;
        }
        __syncthreads();
        uint32_t before = run, tbefore = trun, all = 0, tall = 0;
        for (int w = 0; w < 32; w++) {
            const uint32_t x = s_sum[0][w], y = s_sum[1][w];
            if (w < (int)(threadIdx.x >> 5)) {
                before += x;
                tbefore += y;
            }
            all += x;
            tall += y;
        }
        if (b < nb) {
            p.start[b] = p.cursor[b] = before + ci - c;
            p.tile0[b] = tbefore + ti - tc;
        }
        run += all;
        trun += tall;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        p.start[nb] = run;
        p.tile0[nb] = trun;
    }
}

// Shared memory of a tile's ranking: a counter per digit, which becomes the
// digit's write position less its place in the tile, and that place.
struct PartTileMem {
    uint32_t *cnt;
    uint16_t *loc;
};
__device__ __forceinline__ void part_zero(const PartTileMem &s, int nd) {
    for (int d = threadIdx.x; d < nd; d += kPartThreads) s.cnt[d] = 0;
    __syncthreads();
}
// After every edge was counted: the digits' places in the tile, and a run of
// each reserved at its cursor.  cnt[d] + (place in the tile) is then the
// place to write to.
__device__ __forceinline__ void part_reserve(const PartTileMem &s, int nd, uint32_t *cursor) {
    __shared__ uint32_t s_warp[kPartThreads / 32];
    __syncthreads();
    const int per = (nd + kPartThreads - 1) / kPartThreads;
    const int d0 = min(nd, (int)threadIdx.x * per), d1 = min(nd, d0 + per);
    uint32_t sum = 0;
    for (int d = d0; d < d1; d++) sum += s.cnt[d];
    const uint32_t inc = warp_inclusive_scan(sum);
    if (lane_id() == 31) s_warp[threadIdx.x >> 5] = inc;
    __syncthreads();
    uint32_t run = inc - sum;
    for (int w = 0; w < (int)(threadIdx.x >> 5); w++) run += s_warp[w];
    for (int d = d0; d < d1; d++) {
        s.loc[d] = (uint16_t)run;
        run += s.cnt[d];
    }
    __syncthreads();
    for (int d = threadIdx.x; d < nd; d += kPartThreads) {
        const uint32_t c = s.cnt[d];
        if (c) s.cnt[d] = atomicAdd(cursor + d, c) - s.loc[d];
    }
    __syncthreads();
}

constexpr size_t part_smem(int nd, int bytes_per_edge) {
    return (size_t)nd * 4 + (((size_t)nd * 2 + 15) & ~(size_t)15) + (size_t)kPartTile * bytes_per_edge;
}
// The largest tile of either pass, over every shape.  A kernel's limit on
// dynamic shared memory belongs to the kernel in the whole process, so every
// caller sets it to this one value: a limit by the graph at hand could be
// lowered by another thread's build between the call that raised it and the
// launch that needs it.  (The histogram and the counts stay within the 48 KB
// that need no limit raised.)
constexpr size_t kPartMaxSmem =
    std::max(part_smem(kPartMaxBuckets, 12), part_smem(1 << (kPartMaxLow + 1), 10));
static_assert(2 * kPartMaxBuckets * sizeof(uint32_t) <= (48 << 10), "k_part_hist");
static_assert(sizeof(uint32_t) << (kPartMaxLow + 1) <= (48 << 10), "k_part_count");

// Pass 1: edges (key[e], a[e], b[e]) to their bucket; out_sub holds the low
// bits of the key and, with the shape's flag, whether b[e] >= split, or a[e]
// if by_a (b == nullptr: all ones).  WITH_B: b is carried along.
template <bool WITH_B>
__global__ void __launch_bounds__(kPartThreads, 2)
    k_part_pass1(int64_t m, const int32_t *__restrict__ key, const int32_t *__restrict__ a,
                 const int32_t *__restrict__ b, PartShape sh, int32_t split, bool by_a, uint32_t *cursor, uint16_t *out_sub,
                 int32_t *out_a, int32_t *out_b) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int nd = sh.nb;
    const PartTileMem s{reinterpret_cast<uint32_t *>(smem), reinterpret_cast<uint16_t *>(smem + (size_t)nd * 4)};
    unsigned char *stage = smem + (size_t)nd * 4 + (((size_t)nd * 2 + 15) & ~(size_t)15);
    int32_t *s_a = reinterpret_cast<int32_t *>(stage);
    int32_t *s_b = s_a + kPartTile;
    uint16_t *s_dig = reinterpret_cast<uint16_t *>(s_a + (WITH_B ? 2 : 1) * kPartTile);
    uint16_t *s_sub = s_dig + kPartTile;
    const int64_t e0 = (int64_t)blockIdx.x * kPartTile;
    const int cnt = (int)min((int64_t)kPartTile, m - e0);
    part_zero(s, nd);
    uint32_t dr[kPartPer];   // digit and rank
#pragma unroll
    for (int j = 0; j < kPartPer; j++) {
        const int i = j * kPartThreads + (int)threadIdx.x;
        dr[j] = i < cnt ? (uint32_t)__ldg(key + e0 + i) >> sh.low : 0u;
    }
#pragma unroll
    for (int j = 0; j < kPartPer; j++) {
        const int i = j * kPartThreads + (int)threadIdx.x;
        if (i < cnt) dr[j] = (dr[j] << kPartRankBits) | atomicAdd(s.cnt + dr[j], 1u);
    }
    part_reserve(s, nd, cursor);
#pragma unroll
    for (int j = 0; j < kPartPer; j++) {
        const int i = j * kPartThreads + (int)threadIdx.x;
        if (i < cnt) {
            const uint32_t d = dr[j] >> kPartRankBits;
            const int pos = s.loc[d] + (int)(dr[j] & (kPartTile - 1));
            const int32_t k = __ldg(key + e0 + i);
            uint32_t sub = (uint32_t)k & ((1u << sh.low) - 1u);
            s_a[pos] = __ldg(a + e0 + i);
            if (WITH_B) {
                const int32_t x = b ? __ldg(b + e0 + i) : 1;
                s_b[pos] = x;
                if (sh.flag) sub = 2 * sub + ((by_a ? s_a[pos] : x) >= split);
            }
            s_dig[pos] = (uint16_t)d;
            s_sub[pos] = (uint16_t)sub;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += kPartThreads) {
        const uint32_t g = s.cnt[s_dig[i]] + (uint32_t)i;
        out_sub[g] = s_sub[i];
        out_a[g] = s_a[i];
        if (WITH_B) out_b[g] = s_b[i];
    }
}

// Pass 2's tile of CTA blockIdx.x: its bucket and edges (false: none).
__device__ __forceinline__ bool part_tile(const PartPlan &p, int nb, int &bucket, uint32_t &e0, int &cnt) {
    const uint32_t tile = blockIdx.x;
    if (tile >= __ldg(p.tile0 + nb)) return false;
    int l = 0, r = nb - 1;   // the last bucket with tile0 <= tile that has a tile
    while (l < r) {
        const int mid = (l + r + 1) >> 1;
        if (__ldg(p.tile0 + mid) <= tile) l = mid;
        else r = mid - 1;
    }
    bucket = l;
    e0 = __ldg(p.start + l) + (tile - __ldg(p.tile0 + l)) * (uint32_t)kPartTile;
    cnt = (int)min((uint32_t)kPartTile, __ldg(p.start + l + 1) - e0);
    return true;
}

// Counts per sub-digit (a vertex, or a vertex and flag): count[bucket << ... | sub].
__global__ void __launch_bounds__(kPartThreads) k_part_count(PartPlan p, PartShape sh, const uint16_t *__restrict__ sub,
                                                             uint32_t *count) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *cnt_s = reinterpret_cast<uint32_t *>(smem);
    int bucket, cnt;
    uint32_t e0;
    if (!part_tile(p, sh.nb, bucket, e0, cnt)) return;
    const int nd = sh.sub();
    for (int d = threadIdx.x; d < nd; d += kPartThreads) cnt_s[d] = 0;
    __syncthreads();
    uint32_t x[kPartPer];   // every load before the first count
#pragma unroll
    for (int j = 0; j < kPartPer; j++) {
        const int i = j * kPartThreads + (int)threadIdx.x;
        x[j] = i < cnt ? __ldg(sub + e0 + i) : 0u;
    }
#pragma unroll
    for (int j = 0; j < kPartPer; j++)
        if (j * kPartThreads + (int)threadIdx.x < cnt) atomicAdd(cnt_s + x[j], 1u);
    __syncthreads();
    uint32_t *to = count + ((int64_t)bucket << (sh.low + sh.flag));
    for (int d = threadIdx.x; d < nd; d += kPartThreads)
        if (cnt_s[d]) atomicAdd(to + d, cnt_s[d]);
}

// Pass 2: a bucket's edges to their vertices' places (cursor: one per
// sub-digit, at its vertex's row).  map (or nullptr) renumbers a.
template <bool WITH_B>
__global__ void __launch_bounds__(kPartThreads, 2)
    k_part_pass2(PartPlan p, PartShape sh, const uint16_t *__restrict__ sub, const int32_t *__restrict__ a,
                 const int32_t *__restrict__ b, const int32_t *__restrict__ map, uint32_t *cursor, int32_t *out_a,
                 int32_t *out_b) {
    extern __shared__ __align__(16) unsigned char smem[];
    int bucket, cnt;
    uint32_t e0;
    if (!part_tile(p, sh.nb, bucket, e0, cnt)) return;
    const int nd = sh.sub();
    const PartTileMem s{reinterpret_cast<uint32_t *>(smem), reinterpret_cast<uint16_t *>(smem + (size_t)nd * 4)};
    unsigned char *stage = smem + (size_t)nd * 4 + (((size_t)nd * 2 + 15) & ~(size_t)15);
    int32_t *s_a = reinterpret_cast<int32_t *>(stage);
    int32_t *s_b = s_a + kPartTile;
    uint16_t *s_dig = reinterpret_cast<uint16_t *>(s_a + (WITH_B ? 2 : 1) * kPartTile);
    part_zero(s, nd);
    uint32_t dr[kPartPer];
#pragma unroll
    for (int j = 0; j < kPartPer; j++) {
        const int i = j * kPartThreads + (int)threadIdx.x;
        dr[j] = i < cnt ? __ldg(sub + e0 + i) : 0u;
    }
#pragma unroll
    for (int j = 0; j < kPartPer; j++) {
        const int i = j * kPartThreads + (int)threadIdx.x;
        if (i < cnt) dr[j] = (dr[j] << kPartRankBits) | atomicAdd(s.cnt + dr[j], 1u);
    }
    part_reserve(s, nd, cursor + ((int64_t)bucket << (sh.low + sh.flag)));
#pragma unroll
    for (int j = 0; j < kPartPer; j++) {
        const int i = j * kPartThreads + (int)threadIdx.x;
        if (i < cnt) {
            const uint32_t d = dr[j] >> kPartRankBits;
            const int pos = s.loc[d] + (int)(dr[j] & (kPartTile - 1));
            const int32_t x = __ldg(a + e0 + i);
            s_a[pos] = map ? __ldg(map + x) : x;
            if (WITH_B) s_b[pos] = __ldg(b + e0 + i);
            s_dig[pos] = (uint16_t)d;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += kPartThreads) {
        const uint32_t g = s.cnt[s_dig[i]] + (uint32_t)i;
        out_a[g] = s_a[i];
        if (WITH_B) out_b[g] = s_b[i];
    }
}

// src[e] = the row that holds edge e.  A CTA takes kRowTile consecutive
// edges, finds its first and last row by 32-ary searches, marks each row's
// first edge with its number and spreads the marks by a running maximum: the
// writes are whole 16-byte words whatever the degrees (a warp per row, as
// before, wrote 2-edge rows with 2 of 32 lanes: 0.54 ms for R-MAT 22's 67 M
// directed and 134 M symmetrised edges).
constexpr int kRowTile = 4096;
constexpr int kRowPer = kRowTile / kBlock;
__device__ __forceinline__ int last_row_at(const uint32_t *ro, int n, uint32_t e) {   // by one warp
    int l = 0, r = n - 1;   // ro[l] <= e throughout (ro[0] = 0)
    while (r - l > 31) {
        const int64_t span = (int64_t)(r - l);
        const bool le = __ldg(ro + l + (int)(span * lane_id() / 32)) <= e;
        const int k = __popc(__ballot_sync(0xffffffffu, le)) - 1;   // the true probes are a prefix
        const int nl = l + (int)(span * k / 32);
        r = k == 31 ? r : l + (int)(span * (k + 1) / 32);
        l = nl;
    }
    const bool le = l + (int)lane_id() <= r && __ldg(ro + l + lane_id()) <= e;
    return l + __popc(__ballot_sync(0xffffffffu, le)) - 1;
}
__global__ void __launch_bounds__(kBlock) k_row_sources(int32_t n, int64_t m, const uint32_t *__restrict__ ro,
                                                        int32_t *src) {
    __shared__ __align__(16) int32_t own[kRowTile];   // read four marks at a time
    __shared__ int s_row[2];
    __shared__ int32_t s_max[kWarps];
    const int64_t e0 = (int64_t)blockIdx.x * kRowTile;
    const int cnt = (int)min((int64_t)kRowTile, m - e0);
    const int wid = threadIdx.x >> 5;
    if (wid < 2) {
        const int row = last_row_at(ro, n, (uint32_t)(wid == 0 ? e0 : e0 + cnt - 1));
        if (lane_id() == 0) s_row[wid] = row;
    }
    for (int i = threadIdx.x; i < kRowTile; i += kBlock) own[i] = 0;
    __syncthreads();
    const int r0 = s_row[0], r1 = s_row[1];
    if (threadIdx.x == 0) own[0] = r0;
    // rows after r0 begin after e0; empty rows share the next one's first
    // edge, whose row is the last of them
    // (a tile of a skewed graph's last rows can span 10^5 of them: eight
    // loads in flight a thread)
    for (int r = r0 + 1 + (int)threadIdx.x; r <= r1; r += 8 * kBlock) {
        uint32_t at[8];
#pragma unroll
        for (int j = 0; j < 8; j++) at[j] = r + j * kBlock <= r1 ? __ldg(ro + r + j * kBlock) : 0u;
#pragma unroll
        for (int j = 0; j < 8; j++)
            if (r + j * kBlock <= r1) atomicMax(own + (int)(at[j] - (uint32_t)e0), r + j * kBlock);
    }
    __syncthreads();
    // a warp's 512 marks, four consecutive ones a lane at a time
    int32_t x[kRowPer], carry = 0;
#pragma unroll
    for (int k = 0; k < kRowPer; k += 4) {
        const int4 q = reinterpret_cast<const int4 *>(own)[wid * (kRowTile / kWarps / 4) + k * 8 + lane_id()];
        x[k] = q.x;
        x[k + 1] = max(x[k], q.y);
        x[k + 2] = max(x[k + 1], q.z);
        x[k + 3] = max(x[k + 2], q.w);
        int32_t inc = x[k + 3];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if ((int)lane_id() >= o) inc = max(inc, y);
        }
        int32_t before = __shfl_up_sync(0xffffffffu, inc, 1);
        before = lane_id() == 0 ? carry : max(carry, before);
#pragma unroll
        for (int j = 0; j < 4; j++) x[k + j] = max(x[k + j], before);
        carry = max(carry, __shfl_sync(0xffffffffu, inc, 31));
    }
    if (lane_id() == 0) s_max[wid] = carry;
    __syncthreads();
    int32_t before = 0;
    for (int w = 0; w < wid; w++) before = max(before, s_max[w]);
#pragma unroll
    for (int k = 0; k < kRowPer; k += 4) {
        const int i = (wid * (kRowTile / kWarps / 4) + k * 8 + (int)lane_id()) * 4;
        int32_t y[4];
#pragma unroll
        for (int j = 0; j < 4; j++) y[j] = max(x[k + j], before);
        if (i + 3 < cnt) {
            *reinterpret_cast<int4 *>(src + e0 + i) = make_int4(y[0], y[1], y[2], y[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (i + j < cnt) src[e0 + i + j] = y[j];
        }
    }
}

// CTAs that cover pass 2's tiles: every bucket's last tile may be short.
inline unsigned part_grid2(int64_t m, const PartShape &sh) {
    return (unsigned)((m + kPartTile - 1) / kPartTile + sh.nb);
}

}  // namespace
}  // namespace fg
