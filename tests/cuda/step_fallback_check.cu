// ga_step's scheduling (ga_api.cu) over stand-ins for the launchers: a resident launch that is
// refused.  Prints, per case: the return code, the generations and launches that followed.
#include <cstdio>

#include "ga_internal.h"

namespace {
int resident_calls, step_calls, refuse_from;
uint32_t stepped;
}  // namespace

namespace ga {

bool step_supported(uint32_t, uint32_t, uint32_t) { return true; }
bool async_supported(uint32_t, uint32_t, uint32_t) { return true; }
size_t async_state_bytes(uint32_t, uint32_t) { return 0; }
cudaError_t async_clear(ga_run *, cudaStream_t) { return cudaSuccess; }
int async_step(ga_run *, uint32_t, cudaStream_t) { return GA_OK; }
cudaError_t launch_founder(ga_run *, void *) { return cudaSuccess; }
cudaError_t launch_counter_check(ga_run *, uint32_t, int *) { return cudaSuccess; }
cudaError_t launch_mrca(ga_run *, const uint32_t *, uint32_t, uint32_t *, uint32_t *, void *) { return cudaSuccess; }
size_t mrca_scratch_bytes(const ga_run *, uint32_t) { return 0; }
cudaError_t launch_curation_sites(uint32_t, uint32_t, uint32_t, uint32_t, int32_t *, cudaStream_t, uint32_t, uint2 *)
{
    return cudaSuccess;
}
size_t resident_state_bytes(uint32_t, uint32_t) { return 256; }
bool resident_eligible(const ga_run *) { return true; }
bool resident_pays(const ga_run *) { return true; }
bool resident_plan(const ga_run *, ResidentPlan &) { return true; }
cudaError_t launch_site_table(ga_run *, uint32_t, uint32_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_island_step(ga_run *, const void *, void *, uint32_t, uint32_t n_gens, bool, cudaStream_t)
{
    ++step_calls;
    stepped += n_gens;
    return cudaSuccess;
}
cudaError_t launch_resident(ga_run *, const ResidentPlan &, const void *, void *, uint32_t, uint32_t n_gens, cudaStream_t)
{
    if (resident_calls++ >= refuse_from) return cudaErrorCooperativeLaunchTooLarge;
    stepped += n_gens;
    return cudaSuccess;
}

}  // namespace ga

extern "C" int ga_batch_remove(ga_batch *, ga_run *) { return GA_OK; }

int main()
{
    const uint32_t modes[] = {GA_RESIDENT_AUTO, GA_RESIDENT_AUTO, GA_RESIDENT_ON};
    const int refusals[] = {0, 1, 0};
    for (int c = 0; c < 3; ++c) {
        ga_run run = {};
        run.cfg.mode = GA_SYNC;
        run.per_neighbor = 1;
        run.every_k = 1;
        run.resident_mode = modes[c];
        run.drop_island = 0xFFFFFFFFu;
        resident_calls = step_calls = 0;
        stepped = 0;
        refuse_from = refusals[c];
        const int rc = ga::step_run(&run, 5000, nullptr);
        std::printf("%d %u %llu %d %d\n", rc, stepped, static_cast<unsigned long long>(run.generation), resident_calls, step_calls);
    }
    return 0;
}
