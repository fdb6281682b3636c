// Near-far SSSP with light and heavy edges: FG_BUCKET on a renumbered graph
// whose rows hold their light edges first (View::split).
//
// On a skewed graph label correcting without an order relaxes every edge
// several times: R-MAT 22 four times in the worklist modes, six in the
// synchronous ones.  Most of that is wasted on heavy edges: the hubs' final
// distances are a small fraction of the mean weight, so an edge much heavier
// than that matters only once its source is final.  As in Meyer and Sanders'
// delta-stepping, edges of weight below View::light are relaxed until no
// vertex below the threshold T changes, and only then the heavy edges of the
// vertices that did, each once:
//   light generations  vertices marked near (F) relax their light edges and
//                      are marked for the heavy pass (H); a target lowered
//                      below T is marked near for the next generation;
//   heavy pass         when a generation lowers nothing below T: the marked
//                      vertices relax their heavy edges; what that lowers
//                      below T goes through light generations again;
//   split              when a heavy pass lowers nothing below T: T moves to
//                      the smallest distance at or above it plus the width
//                      (which doubles), and the vertices in between are the
//                      next near ones.  A vertex at or above T was never
//                      expanded with its distance, so the distances
//                      themselves say who waits: there is no far list.
//                      When the vertices not below T hold less than a quarter
//                      of the edges, the rest runs as one phase over all
//                      their edges without a threshold.
// R-MAT 22: 1.1 relaxations per edge in about 28 generations, 0.89 ms, against
// 4.0 in 17 and 2.10 ms of the dense edge-async form (R-MAT 18 0.22 against
// 0.40 ms, R-MAT 16 0.18 against 0.32).  It is bound by latency: 0.26 ms are
// the one large heavy pass, a third the ten light generations that carry
// most of the frontier, a quarter the short ones before and after them.
//
// Marks are bytes, set by plain stores (all writers store 1) and read in the
// next generation; three near arrays rotate: read, filled, cleared.  A vertex
// is marked heavy by the generation that expands its light edges, after its
// distance was last lowered below T, so every distance's heavy edges follow;
// the two heavy arrays take turns, the idle one cleared after its pass.
#pragma once

#include "fg_device.cuh"

namespace fg {
namespace {

enum { kLight = 0, kHeavy = 1, kBoth = 2 };

__host__ __device__ __forceinline__ int64_t lh_pad(int32_t n) { return ((int64_t)n + 15) & ~(int64_t)15; }

// five mark arrays and the bitmap
inline int64_t lh_mark_bytes(int32_t n) { return 5 * lh_pad(n) + 4 * (((int64_t)n + 31) / 32); }

__device__ __forceinline__ void mark_byte(uint8_t *p) {
    asm volatile("st.global.cg.u8 [%0], %1;" ::"l"(p), "r"(1) : "memory");
}

struct LhOp {
    static constexpr bool kNextProbe = false;
    const int32_t *__restrict__ w;
    int32_t *D;
    uint8_t *near;     // marks of the next generation
    int32_t T;

    __device__ __forceinline__ bool cand(int32_t val, uint32_t e, int32_t &c, Acc &a) const {
        const uint32_t x = (uint32_t)val + (uint32_t)ld_edge(w + e);
        if (x >= (uint32_t)kInf) {
            a.overflow = 1;
            return false;
        }
        c = (int32_t)x;
        return true;
    }
    // an L1 copy is never below the current distance; what an old one lets
    // through costs a MIN without effect and perhaps a mark too many, less
    // than checking each against L2 first (R-MAT 22: 0.99 -> 0.91 ms)
    __device__ __forceinline__ int32_t probe(int32_t v) const { return ldca(D + v); }
    __device__ __forceinline__ bool commit(int32_t v, int32_t c, int32_t pv, Acc &a) const {
        if (c < pv) {
            red_min(D + v, c);
            a.updates++;
            if (c < T) {
                mark_byte(near + v);
                a.changed++;
            }
        }
        return false;
    }
};

// A heavy pass: its candidates are rarely below T (an edge of a vertex below T
// is at least a light bound longer), and such a candidate cannot lower a
// target that is.  One bit a vertex, set before the pass, says which are: the
// 32 times denser array answers from L1 what the distances would from L2, and
// on a skewed graph, whose edges mostly lead to the settled hubs, most probes
// end there (R-MAT 22's first heavy pass, 57 M edges: 311 -> 282 us, 10 of
// them for the bits).
struct LhHeavyOp : LhOp {
    const uint32_t *below;   // bit v: distance below T (null: not formed)
    __device__ __forceinline__ int32_t coarse(int32_t v) const {
        return below ? ldca(reinterpret_cast<const int32_t *>(below) + (v >> 5)) : 0;
    }
    __device__ __forceinline__ bool passes(int32_t x, int32_t v, int32_t c) const {
        return c < T || !(((uint32_t)x >> (v & 31)) & 1u);
    }
};

template <int PHASE>
__device__ __forceinline__ void lh_edges(const View &g, int32_t v, uint32_t &b, uint32_t &e) {
    b = __ldg((PHASE == kHeavy ? g.split : g.row_off) + v);
    e = PHASE == kLight ? __ldg(g.split + v) : __ldg(g.row_off + v + 1);
}

// One generation: the vertices marked in `marks` (the near marks, or the
// heavy ones in a heavy pass) and, if first, those at or above T_old and below
// op.T, relax their edges of the phase.  A light generation marks them in
// `heavy`.  High-degree vertices go by their 2048-edge chunks: a CTA per
// chunk, or in a light generation, where a chunk has some dozens of edges, a
// warp.  Mid-degree ones come from their list, strided over the warps (a
// renumbered graph holds them side by side), 32 to a warp with their edges
// spread over the lanes (a warp per vertex leaves most of its 128 edge slots
// empty: the heavy pass 282 -> 263 us), as those of the low-degree ones,
// which a scan of the marks finds.  Offsets and distances are loaded by the thread that
// tests a vertex, all at once, and handed on: loaded per vertex by the warp
// that expands it, the dependent loads made a light generation of 100 K
// vertices take 100 us.
// The compacted vertices' first edge, edge count and distance, per warp or (high
// class) of the CTA.  One set for all phases: an instantiation each took 24 KB
// more of what is L1 otherwise.
struct LhMem {
    uint32_t rb[kWarps][128], d[kWarps][128];
    int32_t v[kWarps][128];
    int n;
};
__device__ __forceinline__ LhMem &lh_mem() {
    __shared__ LhMem m;
    return m;
}

template <int PHASE, class OP>
__device__ __forceinline__ void lh_pass(const Team &t, const View &g, const uint8_t *marks, uint8_t *heavy, bool first,
                                        int32_t T_old, const OP &op, Acc &a) {
    auto &s_rb = lh_mem().rb;
    auto &s_d = lh_mem().d;
    auto &s_v = lh_mem().v;
    int &s_n = lh_mem().n;
    const unsigned lane = lane_id();
    const int wid = threadIdx.x >> 5;
    const int32_t T = op.T;
    auto is_active = [&](int32_t v) -> bool {
        if (__ldcg(marks + v)) return true;
        if (!first) return false;
        const int32_t d = ldcg(op.D + v);
        return d >= T_old && d < T;
    };
    const int64_t G = t.size;
    for (int64_t base = t.rank; base < g.n_high_chunks; base += G * kBlock) {
        const int64_t ci = base + (int64_t)threadIdx.x * G;
        bool act = false;
        uint32_t b = 0, e = 0;
        int32_t dv = 0;
        if (ci < g.n_high_chunks) {
            const int2 hc = __ldg(g.high + ci);
            if (is_active(hc.x)) {
                const uint32_t cb = (uint32_t)hc.y, rb = __ldg(g.row_off + hc.x);
                lh_edges<PHASE>(g, hc.x, b, e);
                dv = ldcg(op.D + hc.x);
                b = max(b, cb);
                e = min(e, cb + (uint32_t)kChunk);
                act = b < e;
                if (cb == rb) {
                    a.verts++;
                    if (PHASE == kLight) mark_byte(heavy + hc.x);
                }
            }
        }
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        const unsigned bal = __ballot_sync(0xffffffffu, act);
        int at = 0;
        if (lane == 0 && bal) at = atomicAdd(&s_n, __popc(bal));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & lanemask_lt());
        if (act) {
            (&s_rb[0][0])[at] = b;
            (&s_d[0][0])[at] = e;
            (&s_v[0][0])[at] = dv;
            a.edges += e - b;
        }
        __syncthreads();
        // in a light generation most chunks have a few dozen edges: those a warp each
        const int na = s_n;
        constexpr uint32_t kWarpChunk = 256;
        auto relax_range = [&](int i, int x, int lanes) {
            const uint32_t e0 = (&s_rb[0][0])[i], e1 = (&s_d[0][0])[i];
            const int32_t d0 = (&s_v[0][0])[i];
            for (uint32_t eb = e0; eb < e1; eb += lanes * kU) {
                uint32_t ee[kU];
                int32_t val[kU];
                bool in[kU];
#pragma unroll
                for (int j = 0; j < kU; j++) {
                    ee[j] = eb + j * lanes + x;
                    in[j] = ee[j] < e1;
                    val[j] = d0;
                }
                relax_batch(g.col, op, NoPush{}, ee, val, in, a);
            }
        };
        auto small = [&](int i) { return PHASE == kLight && (&s_d[0][0])[i] - (&s_rb[0][0])[i] <= kWarpChunk; };
        for (int i = 0; i < na; i++)
            if (!small(i)) relax_range(i, (int)threadIdx.x, kBlock);
        if (PHASE == kLight)
            for (int i = wid; i < na; i += kWarps)
                if (small(i)) relax_range(i, (int)lane, 32);
        __syncthreads();
    }
    const int gw = (int)((t.rank * (unsigned)kBlock + threadIdx.x) >> 5);
    const int nw = (int)(t.size * (unsigned)kWarps);
    int32_t next_mid = gw + (int)lane * nw < g.n_mid ? __ldg(g.mid + gw + (int)lane * nw) : 0;
    for (int base = gw; base < g.n_mid; base += nw * 32) {
        const int i = base + (int)lane * nw;
        const int32_t v = next_mid;
        if (i + nw * 32 < g.n_mid) next_mid = __ldg(g.mid + i + nw * 32);
        uint32_t vb = 0, ve = 0;
        int32_t vd = 0;
        bool act = false;
        if (i < g.n_mid) {
            act = is_active(v);
            if (act) {
                lh_edges<PHASE>(g, v, vb, ve);
                vd = ldcg(op.D + v);
                if (PHASE == kLight) mark_byte(heavy + v);
            }
        }
        unsigned bal = __ballot_sync(0xffffffffu, act);
        if (lane == 0) a.verts += __popc(bal);
        if (bal) relax_rows_of_warp(g.col, op, NoPush{}, vb, ve - vb, vd, a);
    }
    // four vertices a lane and step (one on small graphs); the marks of up to
    // four steps are loaded at once, and the vertices found are gathered over
    // several steps, so that a sparse generation's edges fill their batches
    const int32_t n = g.n;
    const int step = scan_step(n, nw);
    unsigned cnt = 0;   // vertices gathered
    auto flush = [&]() {
        __syncwarp();
        for (unsigned g0 = 0; g0 < cnt; g0 += 32) {
            const unsigned k = g0 + lane;
            uint32_t r0 = 0, dd = 0;
            int32_t vv = 0;
            if (k < cnt) {
                r0 = s_rb[wid][k];
                dd = s_d[wid][k];
                vv = s_v[wid][k];
            }
            relax_rows_of_warp(g.col, op, NoPush{}, r0, dd, vv, a);
        }
        __syncwarp();
        cnt = 0;
    };
    for (int64_t q0 = (int64_t)gw * step; q0 < n; q0 += 4 * (int64_t)nw * step) {
        uint32_t m4[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int64_t v0 = q0 + (int64_t)q * nw * step + (step == 128 ? 4 * lane : lane);
            m4[q] = 0;
            if (step == 128) {
                if (v0 < n) m4[q] = (uint32_t)__ldcg(reinterpret_cast<const int32_t *>(marks + v0));   // padded to 16
            } else if ((int)lane < step && v0 < n) {
                m4[q] = __ldcg(marks + v0);
            }
        }
#pragma unroll 1
        for (int q = 0; q < 4; q++) {
            const int64_t w0 = q0 + (int64_t)q * nw * step;
            if (w0 >= n) break;
            const int64_t v0 = w0 + (step == 128 ? 4 * lane : lane);
            uint32_t mk = q == 0 ? m4[0] : q == 1 ? m4[1] : q == 2 ? m4[2] : m4[3];
            if (lane == 0) a.scanned += min((int64_t)step, (int64_t)n - w0);
            if (first) {
                const int per = step == 128 ? 4 : (int)lane < step ? 1 : 0;
#pragma unroll
                for (int j = 0; j < 4; j++)
                    if (j < per && v0 + j < n) {
                        const int32_t d = ldcg(op.D + v0 + j);
                        if (d >= T_old && d < T) mk |= 1u << (8 * j);
                    }
            }
            if (!__ballot_sync(0xffffffffu, mk != 0)) continue;
            bool act[4];
            uint32_t rb[4], d[4];
            int32_t dv[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                act[j] = (mk >> (8 * j)) & 0xffu;
                rb[j] = d[j] = 0;
                dv[j] = 0;
                if (act[j]) {
                    const int32_t v = (int32_t)(v0 + j);
                    const uint32_t deg = __ldg(g.row_off + v + 1) - __ldg(g.row_off + v);
                    dv[j] = ldcg(op.D + v);
                    uint32_t e;
                    lh_edges<PHASE>(g, v, rb[j], e);
                    d[j] = e - rb[j];
                    act[j] = deg >= 1 && deg < (uint32_t)kLowMax;
                    if (act[j] && PHASE == kLight) mark_byte(heavy + v);
                    act[j] = act[j] && d[j] > 0;
                }
            }
            const unsigned cnt_lane = act[0] + act[1] + act[2] + act[3];
            if (!__ballot_sync(0xffffffffu, cnt_lane != 0)) continue;
            const unsigned incl = warp_inclusive_scan(cnt_lane);
            const unsigned tot = __shfl_sync(0xffffffffu, incl, 31);
            if (cnt + tot > 128) flush();
            unsigned slot = cnt + incl - cnt_lane;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                if (act[j]) {
                    s_rb[wid][slot] = rb[j];
                    s_d[wid][slot] = d[j];
                    s_v[wid][slot] = dv[j];
                    slot++;
                }
            }
            cnt += tot;
            if (lane == 0) a.verts += tot;
        }
    }
    if (cnt) flush();
}

__device__ __forceinline__ void light_heavy_body(const Params &p, const Team &t) {
    Ctrl *c = p.ctrl;
    const View &g = p.g;
    const int32_t n = g.n;
    const int64_t np = lh_pad(n);
    int32_t *D = p.A;
    uint8_t *F = p.marks;              // three near arrays, two heavy ones
    uint8_t *H = p.marks + 3 * np;
    uint32_t *below = reinterpret_cast<uint32_t *>(p.marks + 5 * np);   // a bit per vertex, in 16-byte units
    const int64_t tid = t.rank * (int64_t)kBlock + threadIdx.x;
    const int64_t nth = (int64_t)t.size * kBlock;
    Acc a;
    int rounds = 0, n_barriers = 0, work_gens = 0, splits = 0;
    bool done = false;
    stat_begin();
    auto sync_ = [&](int add = 0) -> bool {
        stat_flush(a);
        const bool r = team_sync(t, c, p.timeout_ns, add);
        if (tid == 0) {
            if (p.trace && n_barriers < p.trace_cap) p.trace[n_barriers] = global_ns();
            n_barriers++;
        }
        return r;
    };
    auto clear = [&](uint8_t *x) {
        for (int64_t i = tid; i < np / 16; i += nth) reinterpret_cast<int4 *>(x)[i] = make_int4(0, 0, 0, 0);
    };
    const int32_t source = p.new_of ? __ldg(p.new_of + p.source) : p.source;
    for (int64_t v = tid; v < n; v += nth) D[v] = v == source ? 0 : kInf;
    for (int64_t i = tid; i < 5 * np / 16; i += nth) {   // the source alone is near in generation 1
        const int64_t at = np + source - 16 * i;         // F[1]
        union {
            uint8_t b[16];
            int4 q;
        } z;
        z.q = make_int4(0, 0, 0, 0);
        if (at >= 0 && at < 16) z.b[at] = 1;
        reinterpret_cast<int4 *>(F)[i] = z.q;
    }
    if (tid == 0)
        for (int k = 0; k < 3; k++) c->far_min[k] = kInf;
    if (p.inject_missing_arrival && t.rank == 0) return;
    bool ok = sync_();
    int phase = kLight, hp = 0;
    bool first = false, h_used = false, fresh = true;
    int32_t T = p.delta, T_old = 0, width = p.delta;
    for (int gen = 1; ok; gen++) {
        if (work_gens >= p.max_rounds) {
            if (tid == 0) atomicOr(&c->status, kStRoundCap);
            break;
        }
        if (p.light_rounds && work_gens >= p.light_rounds) {
            if (tid == 0) atomicOr(&c->status, kStLong);
            break;
        }
        work_gens++;
        rounds++;
        const uint8_t *cur = F + (gen % 3) * np;
        const LhOp op{g.w, D, F + ((gen + 1) % 3) * np, T};
        clear(F + ((gen + 2) % 3) * np);
        uint8_t *heavy = H + (hp & 1) * np;
        if (phase == kLight) {
            if (h_used) clear(H + ((hp + 1) & 1) * np);   // the last heavy pass's marks
            h_used = false;
            lh_pass<kLight>(t, g, cur, heavy, first, T_old, op, a);
        } else if (phase == kHeavy) {
            if (fresh) {   // the epoch's first heavy pass, the large one
                for (int64_t i0 = tid - lane_id(); i0 < n; i0 += nth) {
                    const int64_t v = i0 + lane_id();
                    const unsigned bits = __ballot_sync(0xffffffffu, v < n && ldcg(D + v) < T);
                    if (lane_id() == 0) below[i0 >> 5] = bits;
                }
                if (!sync_()) break;
            }
            LhHeavyOp hop;
            static_cast<LhOp &>(hop) = op;
            hop.below = fresh ? below : nullptr;
            fresh = false;
            lh_pass<kHeavy>(t, g, heavy, nullptr, false, T_old, hop, a);
            hp++;
            h_used = true;
        } else {
            lh_pass<kBoth>(t, g, cur, nullptr, first, T_old, op, a);
        }
        first = false;
        if (!sync_(a.changed)) break;
        a.changed = 0;
        const bool more = team_total() != 0;
        if (more) {
            if (phase == kHeavy) phase = kLight;
            continue;
        }
        if (phase == kBoth || (phase == kHeavy && T >= kInf)) {
            done = true;
            break;
        }
        if (phase == kLight) {
            phase = kHeavy;
            continue;
        }
        // ---- split: the smallest distance not below T, and the edges of all vertices not below T
        rounds++;
        int32_t mn = kInf;
        uint32_t mass = 0;
        if (tid == 0) c->far_min[(splits + 1) % 3] = kInf;
        for (int64_t v = tid; v < n; v += nth) {
            const int32_t d = ldcg(D + v);
            if (d < T) continue;
            mn = min(mn, d);
            mass += __ldg(g.row_off + v + 1) - __ldg(g.row_off + v);
        }
        mn = block_min(mn);
        if (threadIdx.x == 0 && mn < kInf) atomicMin(&c->far_min[splits % 3], mn);
        if (!sync_((int)mass)) break;
        const int64_t left = team_total();
        mn = __ldcg(&c->far_min[splits % 3]);
        splits++;
        if (mn >= kInf) {
            done = true;
            break;
        }
        T_old = T;
        first = fresh = true;
        if (4 * left < g.m) {
            phase = kBoth;
            T = kInf;
        } else {
            phase = kLight;
            T = mn >= kInf - width ? kInf : mn + width;
            width = width > kInf / 2 ? kInf : 2 * width;
        }
    }
    stat_report(a, c);
    if (tid == 0) {
        c->rounds = rounds;
        c->barriers = n_barriers;
        c->splits = splits;
        c->done = done;
    }
    if (done && p.out)
        for (int64_t v = tid; v < n; v += nth) p.out[v] = ldcg(D + (p.new_of ? __ldg(p.new_of + v) : v));
}

}  // namespace
}  // namespace fg
