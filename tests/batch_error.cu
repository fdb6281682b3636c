// Two units in the queue of one team of the batch kernel; the first one's worklists are given no room, so that it
// ends with a worklist error.
#include <vector>

#include "../paper_1903_01665_gb300/csrc/fg_batch_kernel.cuh"

// status[2], done[2]: each unit's; out: the second one's distances (device, n).  Returns a CUDA error code, 0 if none.
extern "C" int run_two_units(const fg_graph *g, int source, int team_size, int32_t *out, int *status, int *done) {
    using namespace fg;
    const size_t ws = query_workspace_bytes(g->g, kSSSP, kVertexAsync);
    const size_t zero = Workspace::need(3, sizeof(Ctrl)) + Workspace::need(kBarWords, 8) + 2 * Workspace::need(1, 4);
    const size_t tables = Workspace::need(team_size, sizeof(int4)) + Workspace::need(4, 4) + Workspace::need(2, sizeof(Params));
    char *base = nullptr;
    cudaError_t e = cudaMalloc(&base, zero + tables + 2 * ws);
    if (e != cudaSuccess) return (int)e;
    cudaMemset(base, 0, zero);
    Workspace w;
    w.base = base;
    Ctrl *ctrls = w.take<Ctrl>(3);
    BatchArgs a;
    a.bctrl = ctrls + 2;
    a.team_bar = w.take<unsigned long long>(kBarWords);
    a.team_q = w.take<int>(1);
    a.cls_next = w.take<int>(1);
    int4 *cta_team = w.take<int4>(team_size);
    int *ints = w.take<int>(4);
    Params *params = w.take<Params>(2);
    std::vector<int4> ct;
    for (int r = 0; r < team_size; r++) ct.push_back(make_int4(0, r, team_size, 0));
    const int queue[4] = {0, 2, 0, 1};   // first and end of the class, then the units in order
    Params p[2];
    for (int u = 0; u < 2; u++) {
        carve_query_workspace(w.base + w.off + u * ws, g->g, kSSSP, kVertexAsync, p[u]);
        set_relabel(g, p[u]);
        p[u].ctrl = ctrls + u;
        p[u].source = source;
        p[u].max_rounds = g->g.n + 2;
        p[u].timeout_ns = 500000000ull;
        p[u].out = u ? out : nullptr;
    }
    for (int k = 0; k < 3; k++) p[0].wl_cap[k] = 0;
    cudaMemcpy(cta_team, ct.data(), ct.size() * sizeof(int4), cudaMemcpyHostToDevice);
    cudaMemcpy(ints, queue, sizeof(queue), cudaMemcpyHostToDevice);
    cudaMemcpy(params, p, sizeof(p), cudaMemcpyHostToDevice);
    a.cta_team = cta_team;
    a.cls_begin = ints;
    a.cls_end = ints + 1;
    a.order = ints + 2;
    a.params = params;
    a.timeout_ns = 500000000ull;
    void *args[] = {&a};
    e = cudaLaunchCooperativeKernel((void *)batch_kernel<kSSSP, kVertexAsync>, dim3(team_size), dim3(kBlock), args, 0, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    Ctrl c[2];
    if (e == cudaSuccess) e = cudaMemcpy(c, ctrls, sizeof(c), cudaMemcpyDeviceToHost);
    for (int u = 0; u < 2 && e == cudaSuccess; u++) {
        status[u] = c[u].status;
        done[u] = c[u].done;
    }
    cudaFree(base);
    return (int)e;
}
