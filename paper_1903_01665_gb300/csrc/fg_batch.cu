// Batched queries: many sources over many resident graphs in one launch per
// (algorithm, mode) kind present -- the runtime counterpart of the paper's
// barrier-free kernels on separate streams (Sec. 3.2) and of its
// independent parallel sections (Sec. 3.4).
//
// The queries are first grouped into units: each query alone, or -- with
// fusion -- the queries on one graph merged (SSSP/BFS into multi-source
// sweeps of up to 8 sources, CC into one computation for all its outputs).
// Each launch is a persistent cooperative kernel whose CTAs are split into
// teams; every team pulls units from the queue of its size class and runs
// the whole fixpoint of each with a team-local barrier (a one-CTA team needs
// only __syncthreads).  The team sizes and their number come from a cost model
// of the units and a makespan common to all kinds (plan_teams).  Kinds run
// concurrently on forked streams, optionally captured in one CUDA graph.
#include <algorithm>
#include <map>
#include <vector>

#include "fg_batch_kernel.cuh"
#include "fg_team_plan.cuh"

namespace fg {

namespace {

using BatchFn = void (*)(BatchArgs);

// kind = algo * 16 + mode
BatchFn batch_kernel_for(int kind) {
    switch (kind) {
        case kSSSP * 16 + kVertexSync: return batch_kernel<kSSSP, kVertexSync>;
        case kSSSP * 16 + kVertexAsync: return batch_kernel<kSSSP, kVertexAsync>;
        case kSSSP * 16 + kEdgeSync: return batch_kernel<kSSSP, kEdgeSync>;
        case kSSSP * 16 + kEdgeAsync: return batch_kernel<kSSSP, kEdgeAsync>;
        case kBFS * 16 + kVertexSync: return batch_kernel<kBFS, kVertexSync>;
        case kBFS * 16 + kVertexAsync: return batch_kernel<kBFS, kVertexAsync>;
        case kBFS * 16 + kEdgeSync: return batch_kernel<kBFS, kEdgeSync>;
        case kBFS * 16 + kEdgeAsync: return batch_kernel<kBFS, kEdgeAsync>;
        case kCC * 16 + kVertexSync: return batch_kernel<kCC, kVertexSync>;
        case kCC * 16 + kVertexAsync: return batch_kernel<kCC, kVertexAsync>;
        case kCC * 16 + kEdgeSync: return batch_kernel<kCC, kEdgeSync>;
        case kCC * 16 + kEdgeAsync: return batch_kernel<kCC, kEdgeAsync>;
        case kSSSP * 16 + kPull: return batch_kernel<kSSSP, kPull>;
        case kBFS * 16 + kPull: return batch_kernel<kBFS, kPull>;
        case kCC * 16 + kPull: return batch_kernel<kCC, kPull>;
        case kSSSP * 16 + kBucket: return batch_kernel<kSSSP, kBucket>;
        case kSSSP * 16 + kLightHeavy: return batch_kernel<kSSSP, kLightHeavy>;
        case kBFS * 16 + kBucket: return batch_kernel<kBFS, kBucket>;
        case kCC * 16 + kBucket: return batch_kernel<kCC, kBucket>;
        case kAnyAlgo * 16 + kMulti: return batch_kernel<kAnyAlgo, kMulti>;
        case kSSSP * 16 + kMultiLight: return batch_kernel<kSSSP, kMultiLight>;
    }
    return nullptr;
}

// The cost model of the planner: a unit on a team of p CTAs takes about
// a + b / p ms.  a: its rounds, each a chain of dependent loads and a barrier;
// b: the edges it visits and the vertices its rounds scan, in CTA-ms.  Fitted to
// four-source sweeps and single queries on 152 to 608 CTAs (grids of 64^2 to
// 1484^2, R-MAT of 2^11 to 2^20 vertices; a 1484^2 grid's SSSP: 7.6, 4.6 and
// 3.2 ms on 152, 304 and 608 CTAs), b half as much again for the teams that
// run beside it (a batch of 24 units: measured 1.0 to 1.6 times the fit).
UnitCost unit_cost(const BatchUnit &u, const View &v, bool light) {
    int depth;
    {
        std::lock_guard<std::mutex> lk(u.g->mu);
        depth = u.g->diam_est;   // known if a query of the graph was FG_AUTO
    }
    const bool skew = u.g->degree_gini > 0.5;
    if (depth < 0) depth = skew ? 10 : 100;
    const bool deep = depth > kDeepLevels;
    const double k = (double)u.q.size(), m = (double)v.m, n = (double)v.n;
    double rounds, round_us, visits, visit_ns, scan;   // scan: vertices' words read per round, in int32
    if (u.mode == kMulti) {
        const bool sssp = u.algo == kSSSP;
        rounds = sssp ? (deep ? 1.5 * depth : light ? 40 : 17) : depth + 1;
        round_us = deep ? 7 : sssp ? 20 : 12;
        visits = m * (sssp ? (deep ? 1.2 + 2.2 * k : light ? 2.3 : 6.0) : (deep ? 0.97 * k : 2.2));
        visit_ns = deep ? (sssp ? 7.4 : 8.7) : (sssp ? 4.9 : 2.7);
        scan = sssp ? n : n / 2;
    } else {
        rounds = u.algo == kSSSP ? 1.4 * depth + 12 : u.algo == kBFS ? depth + 1 : 8;
        round_us = u.mode == kVertexSync || u.mode == kPull ? 6 : 9;
        visits = m * (u.algo == kBFS ? 1.0 : u.algo == kCC ? 2.0 : u.mode == kLightHeavy ? 1.2
                                                             : u.mode == kBucket         ? 2.2
                                                             : deep                      ? 9.0
                                                                                         : 5.0);
        visit_ns = 3.5;
        scan = u.mode == kVertexAsync || u.mode == kEdgeAsync || u.mode == kBucket ||
                       u.mode == kHook || u.mode == kHookBucket
                   ? 0
                   : n;
    }
    UnitCost c;
    c.a = 1e-3 * rounds * round_us;
    c.b = 1.5 * (1e-6 * visits * visit_ns + 6e-7 * rounds * scan);
    return c;
}

}  // namespace

// Groups the batch's queries into units.  Without fusion every query is a
// unit of its own.  With fusion, queries on the same graph are merged: CC
// queries into one unit (CC has no source: one result for every output),
// SSSP and BFS queries into multi-source sweeps of up to 8 sources (a lone
// query stays a plain unit in its own mode).  Units keep the order of their
// first query.
static std::vector<BatchUnit> plan_units(const fg_query *qs, int32_t nq, const std::vector<Mode> &mode,
                                         bool fuse) {
    std::vector<BatchUnit> units;
    if (!fuse) {
        for (int i = 0; i < nq; i++) {
            BatchUnit u;
            u.g = qs[i].g;
            u.algo = (Algo)qs[i].algo;
            u.mode = mode[i];
            u.q.push_back(i);
            units.push_back(u);
        }
        return units;
    }
    std::map<std::pair<const fg_graph *, int>, std::vector<int>> groups;
    std::vector<std::pair<const fg_graph *, int>> order;
    for (int i = 0; i < nq; i++) {
        auto key = std::make_pair(qs[i].g, (int)qs[i].algo);
        auto it = groups.find(key);
        if (it == groups.end()) {
            order.push_back(key);
            groups[key].push_back(i);
        } else {
            it->second.push_back(i);
        }
    }
    for (auto &key : order) {
        const std::vector<int> &qi = groups[key];
        const Algo algo = (Algo)key.second;
        if (algo == kCC || qi.size() == 1) {
            BatchUnit u;
            u.g = key.first;
            u.algo = algo;
            u.mode = mode[qi[0]];
            u.q = qi;
            units.push_back(u);
            continue;
        }
        for (size_t b = 0; b < qi.size(); b += 8) {
            BatchUnit u;
            u.g = key.first;
            u.algo = algo;
            const size_t e = std::min(qi.size(), b + 8);
            u.q.assign(qi.begin() + (long)b, qi.begin() + (long)e);
            u.mode = u.q.size() >= 2 ? kMulti : mode[u.q[0]];
            units.push_back(u);
        }
    }
    return units;
}

// Plans, allocates and enqueues a batch on opt->stream; nothing waits.  The
// results reach device outputs directly; host outputs go to device staging
// and, if enqueue_host_copies, are copied back on the stream (their contents
// are then unspecified for a failed query), as are the copies of a shared
// CC result to its other outputs.  cta_fraction scales the CTA budget so
// that several batches can be resident at once.  fuse merges queries on the
// same graph (plan_units).
fg_status batch_launch(const fg_query *qs, int32_t nq, const fg_batch_options *opt, double cta_fraction,
                       bool enqueue_host_copies, bool fuse, Ctrl *h_ctrls_pinned, BatchJob &job) {
    job.nq = nq;
    job.qs.assign(qs, qs + nq);
    int dev = 0;
    cudaGetDevice(&dev);
    cudaStream_t st = opt && opt->stream ? (cudaStream_t)opt->stream : (cudaStream_t)0;
    job.st = st;
    const int tmo = (opt && opt->wait_timeout_ms > 0) ? opt->wait_timeout_ms : 1000;
    int sms = 0, coop = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop) return fail(FG_ERR_CUDA, "device does not support cooperative launches");

    // ---- resolve modes, form units, group them by kind, plan teams
    std::vector<Mode> mode(nq);
    for (int i = 0; i < nq; i++) {
        const fg_query &q = qs[i];
        fg_mode m = (fg_mode)q.mode;
        if (m == FG_AUTO) {
            fg_status s = fg_select_mode(q.g, (fg_algo)q.algo, &m);
            if (s != FG_OK) return s;
        }
        mode[i] = kernel_mode(q.g, (Algo)q.algo, (Mode)m);
        fg_status vs = ensure_views(q.g, (Algo)q.algo, (int)m);   // lazily built parts, transposed view
        if (vs != FG_OK) return vs;
    }
    job.units = plan_units(qs, nq, mode, fuse);
    const int nu = (int)job.units.size();
    std::vector<BatchUnit> &units = job.units;
    std::vector<const View *> &view = job.view;
    view.resize(nu);
    job.qmode.assign(nq, kVertexSync);
    job.qunit.assign(nq, 0);
    std::map<int, KindPlan> kinds;
    std::vector<UnitCost> cost(nu);
    std::vector<int32_t> light(nu, 0);   // a fused SSSP sweep's first width in the light-heavy order
    for (int u = 0; u < nu; u++) {
        const BatchUnit &un = units[u];
        view[u] = (un.algo == kCC) ? &un.g->s : &un.g->g;
        for (int i : un.q) {
            job.qmode[i] = un.mode;
            job.qunit[i] = u;
        }
        // every multi-source sweep, SSSP or BFS, in one kernel (one launch), but for the light-heavy ones; CC by
        // hooking goes with them
        if (un.mode == kMulti) light[u] = ms_light_width(un.g, un.algo, (int)un.q.size(), 0, 0, true);
        const int kind = light[u]                                                       ? kSSSP * 16 + kMultiLight
                         : un.mode == kMulti || un.mode == kHook || un.mode == kHookBucket ? kAnyAlgo * 16 + kMulti
                                                                                       : un.algo * 16 + (int)un.mode;
        KindPlan &kp = kinds[kind];
        kp.kind = kind;
        kp.queries.push_back(u);
        cost[u] = unit_cost(un, *view[u], light[u] > 0);
    }
    for (auto &kv : kinds) {
        KindPlan &kp = kv.second;
        int per_sm = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, (const void *)batch_kernel_for(kp.kind), kBlock, 0);
        if (e != cudaSuccess) return cuda_fail(e, "occupancy query");
        kp.capacity = std::max(1, (int)(std::max(1, std::min(per_sm * sms, kMaxGrid)) * cta_fraction));
    }
    plan_teams(kinds, cost);

    // ---- one device allocation: zeroed region | tables | unit workspaces | staging
    size_t zero_bytes = Workspace::need(1, sizeof(Ctrl)) + Workspace::need(nu, sizeof(Ctrl));
    size_t table_bytes = Workspace::need(nu, sizeof(Params)) + Workspace::need(nu, sizeof(int));
    for (auto &kv : kinds) {
        KindPlan &kp = kv.second;
        int teams = 0;
        for (int t : kp.class_teams) teams += t;
        const int nc = (int)kp.class_size.size();
        zero_bytes += Workspace::need((int64_t)kBarWords * teams, 8) + Workspace::need(teams, 4) + Workspace::need(nc, 4);
        table_bytes += Workspace::need(kp.ctas, sizeof(int4)) + 2 * Workspace::need(nc, 4);
    }
    job.staged.assign(nq, false);
    size_t ws_bytes = 0;
    for (int u = 0; u < nu; u++) {
        ws_bytes += query_workspace_bytes(*view[u], units[u].algo, units[u].mode);
        if (units[u].algo == kCC && units[u].g->orig_of)   // the labels' smallest original ids
            ws_bytes += Workspace::need(view[u]->n, 4);
    }
    for (int i = 0; i < nq; i++) {
        job.staged[i] = !is_device_pointer(qs[i].out);
        if (job.staged[i]) ws_bytes += Workspace::need(view[job.qunit[i]]->n, 4);
    }
    const size_t total = zero_bytes + table_bytes + ws_bytes;
    job.device_bytes = total;
    cudaError_t e = cudaMallocAsync((void **)&job.base, total, st);
    if (e != cudaSuccess) {
        job.base = nullptr;
        return cuda_fail(e, "batch workspace");
    }
    char *base = job.base;

    // host image of the tables, copied in one transfer
    std::vector<char> img(table_bytes, 0);
    Workspace zw{base}, tw{base + zero_bytes}, hw{img.data()}, qw{base + zero_bytes + table_bytes};
    Ctrl *bctrl = zw.take<Ctrl>(1);
    job.d_ctrls = zw.take<Ctrl>(nu);
    Params *d_params = tw.take<Params>(nu);
    Params *h_params = hw.take<Params>(nu);
    int *d_order = tw.take<int>(nu);
    int *h_order = hw.take<int>(nu);
    job.dout.assign(nq, nullptr);
    for (int u = 0; u < nu; u++) {
        const BatchUnit &un = units[u];
        char *w = qw.base + qw.off;
        qw.off += query_workspace_bytes(*view[u], un.algo, un.mode);
        Params p;
        carve_query_workspace(w, *view[u], un.algo, un.mode, p);
        set_relabel(un.g, p);
        if (un.algo == kCC && un.g->orig_of) p.cc_min = qw.take<int32_t>(view[u]->n);
        h_params[u] = p;
    }
    for (int i = 0; i < nq; i++)
        job.dout[i] = job.staged[i] ? qw.take<int32_t>(view[job.qunit[i]]->n) : qs[i].out;
    for (int u = 0; u < nu; u++) {
        const BatchUnit &un = units[u];
        Params &p = h_params[u];
        if (un.mode == kPull) p.tv = (un.algo == kCC) ? un.g->s : un.g->t;
        p.delta = un.mode == kLightHeavy ? un.g->light : default_delta(un.g);
        p.light_rounds = kLightRounds;
        p.ctrl = job.d_ctrls + u;
        p.source = un.algo == kCC ? 0 : qs[un.q[0]].src;
        p.max_rounds = round_cap(un.mode, view[u]->n);
        p.timeout_ns = (unsigned long long)tmo * 1000000ull;
        if (un.mode == kMulti) {
            p.ms_k = (int32_t)un.q.size();
            p.ms_bfs = un.algo == kBFS ? 1 : 0;
            if (un.algo == kBFS && un.g->sym_built && un.g->new_of) p.tv = un.g->s;
            p.ms_light = light[u];
            p.max_rounds = ms_default_rounds(view[u]->n, p.ms_k, un.algo == kSSSP, p.ms_light > 0);
            for (size_t j = 0; j < un.q.size(); j++) {
                p.ms_src[j] = qs[un.q[j]].src;
                p.ms_out[j] = job.dout[un.q[j]];
            }
        } else {
            p.out = job.dout[un.q[0]];
            p.cc_hook = un.mode == kHook || un.mode == kHookBucket;
        }
    }
    job.params.assign(h_params, h_params + nu);
    std::vector<BatchArgs> args;
    std::vector<int> kind_ctas;
    std::vector<BatchFn> kind_fn;
    int order_pos = 0;
    for (auto &kv : kinds) {
        KindPlan &kp = kv.second;
        const int nc = (int)kp.class_size.size();
        int teams = 0;
        for (int t : kp.class_teams) teams += t;
        BatchArgs a;
        a.team_bar = zw.take<unsigned long long>((int64_t)kBarWords * teams);
        a.team_q = zw.take<int>(teams);
        a.cls_next = zw.take<int>(nc);
        int4 *d_ct = tw.take<int4>(kp.ctas);
        int4 *h_ct = hw.take<int4>(kp.ctas);
        int *d_cb = tw.take<int>(nc), *h_cb = hw.take<int>(nc);
        int *d_ce = tw.take<int>(nc), *h_ce = hw.take<int>(nc);
        int cta = 0, team = 0;
        for (int c = 0; c < nc; c++) {
            h_cb[c] = order_pos;
            for (int u : kp.class_q[c]) h_order[order_pos++] = u;
            h_ce[c] = order_pos;
            for (int k = 0; k < kp.class_teams[c]; k++, team++)
                for (int r = 0; r < kp.class_size[c]; r++) h_ct[cta++] = make_int4(team, r, kp.class_size[c], c);
        }
        a.cta_team = d_ct;
        a.cls_begin = d_cb;
        a.cls_end = d_ce;
        a.order = d_order;
        a.params = d_params;
        a.bctrl = bctrl;
        a.timeout_ns = (unsigned long long)tmo * 1000000ull;
        args.push_back(a);
        kind_ctas.push_back(kp.ctas);
        kind_fn.push_back(batch_kernel_for(kp.kind));
        job.teams += teams;
        job.ctas += kp.ctas;
    }

    // ---- enqueue: fork one stream per kind, join, optionally as a CUDA graph
    const int nk = (int)args.size();
    job.launches = nk;
    job.ks.assign(nk, nullptr);
    job.kev.assign(nk, nullptr);
    const bool use_graph = opt && opt->use_cuda_graph;
    auto ck = [&](cudaError_t err, const char *what) {
        if (err != cudaSuccess && job.status == FG_OK) {
            job.status = (err == cudaErrorMemoryAllocation) ? FG_ERR_OUT_OF_MEMORY : FG_ERR_CUDA;
            job.msg = std::string(what) + ": " + cudaGetErrorString(err);
        }
        return err == cudaSuccess;
    };
    ck(cudaEventCreateWithFlags(&job.fork, cudaEventDisableTiming), "event");
    ck(cudaEventCreate(&job.ev0), "event");
    ck(cudaEventCreate(&job.ev1), "event");
    ck(cudaEventCreateWithFlags(&job.done, cudaEventDisableTiming), "event");
    for (int k = 0; k < nk; k++) {
        ck(cudaStreamCreateWithFlags(&job.ks[k], cudaStreamNonBlocking), "stream");
        ck(cudaEventCreateWithFlags(&job.kev[k], cudaEventDisableTiming), "event");
    }
    ck(cudaMemcpyAsync(base + zero_bytes, img.data(), table_bytes, cudaMemcpyHostToDevice, st), "table upload");
    ck(cudaEventRecord(job.ev0, st), "event");
    // the launches are recorded on `cs`: the caller's stream itself, or for a
    // CUDA graph a private stream (the legacy default stream cannot capture)
    cudaStream_t cs = st;
    if (job.status == FG_OK && use_graph) {
        ck(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking), "stream");
        ck(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal), "capture");
    }
    ck(cudaMemsetAsync(base, 0, zero_bytes, cs), "memset");
    ck(cudaEventRecord(job.fork, cs), "event");
    for (int k = 0; k < nk && job.status == FG_OK; k++) {
        ck(cudaStreamWaitEvent(job.ks[k], job.fork, 0), "fork");
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kind_ctas[k]);
        cfg.blockDim = dim3(kBlock);
        cfg.stream = job.ks[k];
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (ck(cudaLaunchKernelEx(&cfg, kind_fn[k], args[k]), "batch launch")) count_launch();
        ck(cudaEventRecord(job.kev[k], job.ks[k]), "event");
        ck(cudaStreamWaitEvent(cs, job.kev[k], 0), "join");
    }
    if (use_graph && cs != st) {
        cudaError_t ce = cudaStreamEndCapture(cs, &job.graph);
        if (job.status == FG_OK) ck(ce, "capture");
        if (job.status == FG_OK) ck(cudaGraphInstantiate(&job.exec, job.graph, 0), "graph instantiate");
        if (job.status == FG_OK) ck(cudaGraphLaunch(job.exec, st), "graph launch");
        cudaStreamDestroy(cs);
    }
    ck(cudaEventRecord(job.ev1, st), "event");
    job.h_ctrls = h_ctrls_pinned;
    if (!job.h_ctrls) {
        job.own_ctrls.resize(nu);
        job.h_ctrls = job.own_ctrls.data();
    }
    ck(cudaMemcpyAsync(job.h_ctrls, job.d_ctrls, nu * sizeof(Ctrl), cudaMemcpyDeviceToHost, st), "status copy");
    if (enqueue_host_copies) {
        for (int u = 0; u < nu; u++) {
            const BatchUnit &un = units[u];
            const size_t bytes = (size_t)view[u]->n * sizeof(int32_t);
            for (size_t j = 0; j < un.q.size(); j++) {
                const int i = un.q[j];
                if (un.mode != kMulti && j > 0)   // the unit's one result, to its other outputs
                    ck(cudaMemcpyAsync(qs[i].out, job.dout[un.q[0]], bytes, cudaMemcpyDefault, st), "result copy");
                else if (job.staged[i])
                    ck(cudaMemcpyAsync(qs[i].out, job.dout[i], bytes, cudaMemcpyDeviceToHost, st), "result copy");
            }
        }
        job.host_copies_done = true;
    }
    ck(cudaEventRecord(job.done, st), "event");
    if (job.status != FG_OK) return fail(job.status, job.msg);
    return FG_OK;
}

// Waits for a launched batch, reports every query and releases the batch.
fg_status batch_finish(BatchJob &job, fg_status *status_out, fg_stats *stats_out, fg_batch_stats *bstats) {
    const int nq = job.nq;
    const int nu = (int)job.units.size();
    cudaStream_t st = job.st;
    auto ck = [&](cudaError_t err, const char *what) {
        if (err != cudaSuccess && job.status == FG_OK) {
            job.status = (err == cudaErrorMemoryAllocation) ? FG_ERR_OUT_OF_MEMORY : FG_ERR_CUDA;
            job.msg = std::string(what) + ": " + cudaGetErrorString(err);
        }
        return err == cudaSuccess;
    };
    if (job.done) ck(cudaEventSynchronize(job.done), "batch");
    float ms = 0.f;
    if (job.status == FG_OK && job.ev0 && job.ev1) cudaEventElapsedTime(&ms, job.ev0, job.ev1);
    std::vector<fg_status> qst(nq, FG_OK);
    std::vector<int> again;   // units whose light-heavy order reached its limit of generations
    for (int u = 0; u < nu && job.status == FG_OK; u++) {
        const Ctrl &hc = job.h_ctrls[u];
        const BatchUnit &un = job.units[u];
        const Params &p = job.params[u];
        const View &v = *job.view[u];
        const size_t bytes = (size_t)v.n * sizeof(int32_t);
        fg_status us = FG_OK;
        if (hc.status & kStTimeout) us = FG_ERR_TIMEOUT;
        else if (hc.status & kStRoundCap) us = FG_ERR_TIMEOUT;
        else if (hc.status & kStWorklist) us = FG_ERR_CUDA;
        else if (hc.status & kStLong) {
            again.push_back(u);
            continue;
        } else if (!hc.done) us = FG_ERR_TIMEOUT;
        for (int i : un.q) qst[i] = us;
        if (us == FG_OK && (hc.status & kStOverflow) && un.algo == kSSSP && un.mode != kMulti) {
            us = ensure_src(un.g);   // the check reads the edge sources, which a FG_GRAPH_LAZY graph may not have yet
            for (int i : un.q) qst[i] = us;
        }
        if (us == FG_OK && (hc.status & kStOverflow) && un.algo == kSSSP) {
            int *flag = reinterpret_cast<int *>(p.ctrl);
            int hf = 0;
            ck(cudaMemsetAsync(flag, 0, sizeof(int), st), "memset");
            if (un.mode == kMulti) {
                ms_overflow_check_launch(v, p.A, p.ms_k, flag, st);
            } else {   // on the result in internal order (p.out holds it in original order)
                overflow_check_launch(v, p.new_of ? ((hc.result_in_b && p.B) ? p.B : p.A) : p.out, flag, st);
            }
            ck(cudaMemcpyAsync(&hf, flag, sizeof(int), cudaMemcpyDeviceToHost, st), "copy");
            ck(cudaStreamSynchronize(st), "overflow check");
            if (un.mode == kMulti) {
                // the sweep wrote no output: write those of the sources that did not overflow
                MsOuts ok{};
                for (size_t j = 0; j < un.q.size(); j++) {
                    if ((hf >> j) & 1) qst[un.q[j]] = FG_ERR_OVERFLOW;
                    else ok.p[j] = job.dout[un.q[j]];
                }
                ms_output_launch(p.A, v.n, p.ms_k, ok, p.new_of, st);
                if (job.host_copies_done)   // the early copies carried no result: copy again
                    for (size_t j = 0; j < un.q.size(); j++) {
                        const int i = un.q[j];
                        if (qst[i] == FG_OK && job.staged[i])
                            ck(cudaMemcpyAsync(job.qs[i].out, job.dout[i], bytes, cudaMemcpyDeviceToHost, st),
                               "result copy");
                    }
            } else if (hf) {
                for (int i : un.q) qst[i] = FG_ERR_OVERFLOW;
            }
        }
        if (!job.host_copies_done)
            for (size_t j = 0; j < un.q.size(); j++) {
                const int i = un.q[j];
                if (qst[i] != FG_OK) continue;
                if (un.mode != kMulti && j > 0)
                    ck(cudaMemcpyAsync(job.qs[i].out, job.dout[un.q[0]], bytes, cudaMemcpyDefault, st),
                       "result copy");
                else if (job.staged[i])
                    ck(cudaMemcpyAsync(job.qs[i].out, job.dout[i], bytes, cudaMemcpyDeviceToHost, st),
                       "result copy");
            }
        if (stats_out)
            for (int i : un.q) {
                fg_stats &s = stats_out[i];
                s = fg_stats{};
                s.mode = un.mode == kMulti ? -1 : public_mode(un.mode);
                s.rounds = hc.rounds;
                s.jump_passes = hc.jump_passes;
                s.vertices_processed = (int64_t)hc.st_vertices;
                s.edges_relaxed = (int64_t)hc.st_edges;
                s.updates = (int64_t)hc.st_updates;
                s.pushes = (int64_t)hc.st_pushes;
                s.scanned = (int64_t)hc.st_scanned;
                s.barriers = hc.barriers;
                s.pull_rounds = hc.pull_rounds;
                s.edges_pulled = (int64_t)hc.st_pulled;
            }
    }
    ck(cudaStreamSynchronize(st), "result copies");
    if (job.exec) cudaGraphExecDestroy(job.exec);
    if (job.graph) cudaGraphDestroy(job.graph);
    for (size_t k = 0; k < job.ks.size(); k++) {
        if (job.kev[k]) cudaEventDestroy(job.kev[k]);
        if (job.ks[k]) cudaStreamDestroy(job.ks[k]);
    }
    if (job.fork) cudaEventDestroy(job.fork);
    if (job.ev0) cudaEventDestroy(job.ev0);
    if (job.ev1) cudaEventDestroy(job.ev1);
    if (job.done) cudaEventDestroy(job.done);
    if (job.base) cudaFreeAsync(job.base, st);
    job.exec = nullptr;
    job.graph = nullptr;
    job.ks.clear();
    job.kev.clear();
    job.fork = job.ev0 = job.ev1 = job.done = nullptr;
    job.base = nullptr;
    for (int u : again) {   // in the order of other graphs, with the batch's memory given back
        if (job.status != FG_OK) break;
        const BatchUnit &un = job.units[u];
        note_order(un.g, true);
        const int k = (int)un.q.size();
        int32_t srcs[kMsMax], *outs[kMsMax];
        fg_status each[kMsMax];
        for (int j = 0; j < k; j++) {
            srcs[j] = job.qs[un.q[j]].src;
            outs[j] = job.qs[un.q[j]].out;
        }
        fg_options o{};
        o.stream = st;
        o.wait_timeout_ms = (int32_t)(job.params[u].timeout_ns / 1000000ull);
        fg_stats s{};
        if (un.mode == kMulti) run_multi(un.g, un.algo, k, srcs, outs, &o, each, &s);
        else each[0] = run_query(un.g, un.algo, (Mode)public_mode(un.mode), srcs[0], outs[0], &o, &s);
        for (int j = 0; j < k; j++) {
            qst[un.q[j]] = each[un.mode == kMulti ? j : 0];
            if (stats_out) stats_out[un.q[j]] = s;
        }
    }
    if (job.status != FG_OK)
        for (int i = 0; i < nq; i++) qst[i] = job.status;
    fg_status first_err = FG_OK;
    std::string first_msg;
    for (int i = 0; i < nq; i++) {
        if (status_out) status_out[i] = qst[i];
        if (qst[i] != FG_OK && first_err == FG_OK) {
            first_err = qst[i];
            first_msg = "batch query " + std::to_string(i) + " failed: " + fg_status_string(qst[i]);
        }
    }
    if (bstats) {
        bstats->kernel_ms = ms;
        bstats->launches = job.launches;
        bstats->teams = job.teams;
        bstats->ctas = job.ctas;
    }
    if (job.status != FG_OK) return fail(job.status, job.msg);
    if (first_err != FG_OK) return fail(first_err, first_msg);
    return FG_OK;
}

fg_status run_batch(const fg_query *qs, int32_t nq, const fg_batch_options *opt, fg_status *status_out,
                    fg_stats *stats_out, fg_batch_stats *bstats) {
    BatchJob job;
    const bool fuse = opt && opt->fuse_same_graph;
    fg_status s = batch_launch(qs, nq, opt, 1.0, false, fuse, nullptr, job);
    fg_status f = batch_finish(job, status_out, stats_out, bstats);
    return s != FG_OK ? s : f;
}

}  // namespace fg
