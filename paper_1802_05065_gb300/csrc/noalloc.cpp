// noalloc.cpp -- fpt_run_noalloc: one request, run to completion in a single launch, without device
// memory of the library's own.
//
// Who needs this: callers that must not allocate device memory while they run -- for example a
// host program that reserved the device memory for its own pool before loading this library,
// code inside a latency-critical loop where cudaMalloc's implicit synchronisation is not
// acceptable, or plugin hosts whose contract forbids allocation during execution.  The
// persistent engine (fpt_create / fpt_submit) allocates its lane state and accumulators;
// this entry point allocates nothing: the kernel's queues and accumulators live in shared memory,
// so calls on any streams and threads may overlap.
#include <string>

#include "engine_dev.h"
#include "internal.h"

using namespace fpt;

extern "C" fpt_status fpt_run_noalloc(const fpt_params *params, uint64_t n_traj, uint64_t seed,
                                      int64_t *d_steps, fpt_sums *d_sums, uint64_t *d_hist,
                                      void *stream) {
    Decoded d;
    std::string err;
    if (!decode(params, &d, &err)) {
        set_error(err);
        return FPT_EINVAL;
    }
    if (params->precision != FPT_FP32) {
        set_error("fpt_run_noalloc integrates in FP32 only");
        return FPT_EINVAL;
    }
    if (params->stop_rse != 0.0) {
        set_error("fpt_run_noalloc runs every trajectory: stop_rse must be 0");
        return FPT_EINVAL;
    }
    if (!d_sums || !d_hist) {
        set_error("d_sums and d_hist are required device outputs");
        return FPT_EINVAL;
    }
    if (n_traj > 0xFFFFFFFFull) {   // a CTA's per-bin counts are 32-bit
        set_error("fpt_run_noalloc: n_traj must be < 2^32");
        return FPT_EINVAL;
    }
    if (n_traj == 0) return FPT_OK;
    if (d.hist_bins > kSoloMaxBins) {
        set_error("fpt_run_noalloc: hist_bins must be <= 10240 (per-CTA histogram in shared memory)");
        return FPT_EINVAL;
    }
    const cudaError_t e = launch_solo(d, seed, params->traj_offset, n_traj, d_steps, d_sums,
                                      reinterpret_cast<unsigned long long *>(d_hist),
                                      static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) {
        set_error(std::string("fpt_run_noalloc: ") + cudaGetErrorString(e));
        return FPT_ECUDA;
    }
    return FPT_OK;
}
