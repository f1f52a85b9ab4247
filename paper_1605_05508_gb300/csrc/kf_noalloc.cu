// kf_noalloc.cu -- kf_fit_noalloc: the track fit for callers that must not
// allocate device memory.
//
// The fused launch keeps a track's state and status in registers through all
// layers, so it needs no per-track scratch whatever outputs the caller leaves
// out, and a call performs no allocation at all.
#include "kf_internal.h"

extern "C" int kf_fit_noalloc(kf_ctx* ctx, const kf_tracks* seeds, const kf_track_hits* hits, kf_tracks* out,
                              float* chi2, int32_t* status, void* stream) {
  const int rc = kfi::check_fit(ctx, seeds, hits, out);  // the checks of kf_fit
  if (rc) return rc;
  const int64_t n = seeds->n;
  if (n > KF_NOALLOC_MAX_TRACKS) return KF_EINVAL;  // the documented limit: split the batch
  if (n == 0) return KF_OK;
  KF_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  KF_CUDA_TRY(ctx, kfi::launch_fit_fused(kfi::fused_args(ctx, seeds, hits, out, chi2, status), ctx->tune.fit_block, static_cast<cudaStream_t>(stream)));
  return KF_OK;
}
