// The persistent kernel of a batch: teams of CTAs that pull units from the
// queue of their size class and run the whole fixpoint of each.
#pragma once

#include "fg_multi.cuh"

namespace fg {
namespace {

struct BatchArgs {
    const int4 *cta_team;     // per CTA: team, rank in team, team size, class
    unsigned long long *team_bar;   // kBarWords per team
    int *team_q;              // per team: the queue slot it is working on
    int *cls_next;            // per class: next queue slot
    const int *cls_begin;     // per class: queue range in `order`
    const int *cls_end;
    const int *order;         // unit indices, by class, largest work first
    const Params *params;     // per unit of the batch
    Ctrl *bctrl;              // status of the queue barriers
    unsigned long long timeout_ns;
};

template <int ALGO, int MODE>
__global__ void __launch_bounds__(kBlock, min_blocks<ALGO, MODE>()) batch_kernel(BatchArgs b) {
    const int4 ct = b.cta_team[blockIdx.x];
    const Team t{ct.y, ct.z, b.team_bar + (int64_t)kBarWords * ct.x};
    const int cls = ct.w;
    uint32_t ring_used;
    team_begin();
    fixpoint_prologue<ALGO, MODE>(ring_used);
    for (;;) {
        if (t.rank == 0 && threadIdx.x == 0) b.team_q[ct.x] = b.cls_begin[cls] + atomicAdd(&b.cls_next[cls], 1);
        if (!team_sync(t, b.bctrl, b.timeout_ns)) return;
        const int qi = __ldcg(&b.team_q[ct.x]);
        if (qi >= b.cls_end[cls]) return;
        query_body<ALGO, MODE>(b.params[b.order[qi]], t, ring_used);
        if (!team_next_query(t)) return;
        if (!team_sync(t, b.bctrl, b.timeout_ns)) return;
    }
}

}  // namespace
}  // namespace fg
