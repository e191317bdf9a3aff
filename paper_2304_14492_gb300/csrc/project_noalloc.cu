// Radial projection for callers that cannot allocate device memory.
//
// zm_project on a tensor-core plan keeps split-K partial sums in a workspace
// that the plan grows with cudaMalloc when a larger batch arrives.  Some callers
// cannot let the library allocate at call time: their device memory is already
// handed out by another allocator (a framework's caching pool that reserved the
// GPU up front), or they run in a loop where cudaMalloc's implicit device-wide
// synchronisation and unbounded latency are not acceptable.  zm_project_noalloc
// computes the same projection in FP32 (the kernel of zm_project's FP32 path,
// which holds its sums on chip), whatever the plan's precision; it allocates
// nothing.  There is no counterpart in the paper: this is an interface matter
// only.
#include "zm_internal.cuh"

using namespace zm;

// The largest request, P(n_max) * 2 * batch floats, that the interface takes: the
// size of the fixed scratch an earlier form of this call kept.  Nothing here needs
// the limit any more; it stays because requests that were refused stay refused.
constexpr size_t NOALLOC_FLOATS = (size_t)1 << 21;

extern "C" int zm_project_noalloc(zm_plan_t plan, const float* spectra, int batch, float* out, unsigned flags,
                                  void* stream) {
    if (!plan || !spectra || !out) return set_error(ZM_EINVAL, "NULL argument");
    if (batch < 1) return set_error(ZM_EINVAL, "batch must be >= 1 (got %d)", batch);
    if (flags & ~ZM_NEUMANN) return set_error(ZM_EINVAL, "unknown flags 0x%x", flags);
    const size_t floats = (size_t)plan->P * 2 * batch;
    if (floats > NOALLOC_FLOATS)
        return set_error(ZM_EINVAL,
                         "zm_project_noalloc: P(n_max) * 2 * batch = %zu floats exceeds the %zu floats this call takes (the "
                         "limit of the fixed scratch it once kept); use a smaller batch or zm_project",
                         floats, NOALLOC_FLOATS);
    DeviceGuard g(plan->device);
    if (!g.ok) return set_error(ZM_ECUDA, "cannot select device %d", plan->device);
    return launch_projection_fp32(plan, spectra, batch, out, flags, (cudaStream_t)stream);
}
