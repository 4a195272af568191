// Stands between the library's host code and its launchers (linked with --wrap), for test_gpu_faults.py: a
// launch fails as the runtime would report it, without being made, or an advance leaves the error flag
// set as one whose wait ran out does.
#include "lbcm_internal.h"

using namespace lbcm;

static int g_fail_step = 0, g_fail_advance = 0, g_flag = 0;

// the n-th call from now fails (0: none); flag: every advance sets the flag
extern "C" __attribute__((visibility("default"))) void launch_faults(int fail_step, int fail_advance, int flag) {
    g_fail_step = fail_step;
    g_fail_advance = fail_advance;
    g_flag = flag;
}

extern "C" cudaError_t REAL_STEP(const StepArgs &, int, cudaStream_t, cudaEvent_t *, long long *, int);
extern "C" cudaError_t WRAP_STEP(const StepArgs &a, int storage, cudaStream_t s, cudaEvent_t *ev, long long *n, int passes) {
    if (g_fail_step > 0 && --g_fail_step == 0) return cudaErrorLaunchOutOfResources;
    return REAL_STEP(a, storage, s, ev, n, passes);
}
extern "C" cudaError_t REAL_ADVANCE(const StepArgs &, const AdvancePlan &, const AdvanceArgs &, cudaStream_t, long long *);
extern "C" cudaError_t WRAP_ADVANCE(const StepArgs &a, const AdvancePlan &p, const AdvanceArgs &v, cudaStream_t s, long long *n) {
    if (g_fail_advance > 0 && --g_fail_advance == 0) return cudaErrorLaunchOutOfResources;
    const cudaError_t e = REAL_ADVANCE(a, p, v, s, n);
    if (g_flag && e == cudaSuccess) return cudaMemsetAsync(v.err, 1, sizeof(int), s);
    return e;
}
