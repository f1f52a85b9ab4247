// kf_refit.cu -- the Kalman fit of built tracks over all layers with the hits
// the build chose (building, Sec. 3, followed by fitting, Sec. 2): the fused
// fit from the seed state, every track taking the seeding layers' hits from
// the seed's own and each building layer's by the hit id kf_build returned,
// from the raw hits of the seed's (event, layer) segment.
#include "kf_internal.h"

using namespace kfi;

extern "C" int kf_refit(kf_ctx* ctx, const kf_tracks* seeds, const kf_track_hits* seed_hits, const int64_t* seed_off,
                        const kf_layer_hits* build_hits, const int32_t* hit_idx, kf_tracks* out, float* chi2,
                        int32_t* status, void* stream) {
  if (!ctx || !seeds || !seed_hits || !build_hits || !out) return KF_EINVAL;
  const int64_t n = seeds->n;
  const int Ls = seed_hits->n_layers, Lb = build_hits->n_layers, E = build_hits->n_events;
  if (n < 0 || seed_hits->n_tracks != n || out->n != n) return KF_EINVAL;
  if (Ls < 0 || Lb < 1 || build_hits->first_layer != Ls || Ls + Lb > ctx->cfg.n_layers || E < 1) return KF_EINVAL;
  if (n == 0) return KF_OK;
  if (!seed_off || !hit_idx || !build_hits->xyz || !build_hits->seg_off || (Ls > 0 && !seed_hits->xyz) ||
      build_hits->n_hits < 0)
    return KF_EINVAL;
  KF_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  RefitGatherArgs g;
  g.seed_xyz = seed_hits->xyz;
  g.seed_valid = seed_hits->valid;
  g.seed_off = seed_off;
  g.hit_xyz = build_hits->xyz;
  g.seg_off = build_hits->seg_off;
  g.hit_idx = hit_idx;
  g.n = n;
  g.n_hits = build_hits->n_hits;
  g.Ls = Ls;
  g.Lb = Lb;
  g.E = E;
  kf_track_hits all;
  all.n_tracks = n;
  all.n_layers = Ls + Lb;
  all.xyz = nullptr;
  all.valid = nullptr;
  if (!seeds->par || !seeds->cov || !seeds->charge || !out->par || !out->cov) return KF_EINVAL;
  KF_CUDA_TRY(ctx, launch_fit_gather(fused_args(ctx, seeds, &all, out, chi2, status), g,
                                     static_cast<cudaStream_t>(stream)));
  return KF_OK;
}
