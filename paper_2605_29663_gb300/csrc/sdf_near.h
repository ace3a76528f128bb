// sdf_near.h -- the pruned paths of exact_sdf_batch (sdf_near.cu).
#pragma once

#include "internal.h"

namespace exact {

// Whether the pruned path is the faster one for this call.
bool sdf_near_fits(const exact_footprint *fp, int n_points, int n_poses, bool dist);
// Whether it can be for any footprint, at these sizes or smaller ones.
bool sdf_near_possible(int n_points, int n_poses);
// Device scratch of a call with n_points points.
size_t sdf_near_bytes(int n_points);
// keys: initialised per-pose keys for the minimum over several chunks, or NULL
// when one chunk holds every point (or without dist).
int sdf_near_launch(const float2 *pts, const uint8_t *mask, int N, const float *poses, int P, const exact_footprint *fp,
                    float *dist, float *dmin, int *argmin, unsigned long long *keys, void *scratch, int sms, int *err,
                    cudaStream_t st);
constexpr int kSdfChunk = 8192;   // points of a chunk

}  // namespace exact
