/* lb_resident_host.h -- launch arguments of the resident kernels, between the plan code
 * (lb_resident.cu) and the translation units that instantiate them. */
#pragma once

#include "lb_internal.h"

namespace lbk {

struct ResLaunch {
    const ResPlan *plan;
    const void *d_plan;
    const uint32_t *d_off;
    const void *params;
    const RingTab *tabs;
    int nsteps, base;
    uint32_t step0;
    int advance;
    unsigned int *queue;
    const void *osc;
    int blocks;
    bool force;
    void *stream;
    bool query;   /* nothing is launched: 0 if a block (a cluster) of it can be resident */
};
template <int ST, bool PAIR>
int launch_resident_store(const ResLaunch &a);

}  // namespace lbk
