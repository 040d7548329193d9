// Launchers of the reduction kernels (gradient norms, relative state change).
#pragma once
#include "desloc_kernels.cuh"

namespace desloc {

// Entries of a row of partials: the rows are padded to whole 16-byte pieces.
inline long long reduce_row(long long items) { return (items + 3) & ~3LL; }

// partial: scratch of at least M * reduce_row(nchunks) floats; norms, scales: [M] floats, all on the device.
// scales[m] = min(1, max_norm / ||g^m||_2), or 1 when max_norm <= 0.  elems: parameters of a worker; *launches: one (small
// problems) or two.
// err, wait_limit: the flag a block sets when its bounded wait for a bulk copy runs out, and the
// bound (as for the step kernels).
cudaError_t launch_grad_norms(const Chunk *chunks, long long nchunks, int64_t elems, const void *const *g, int nt,
                              int M, bool bf16, float max_norm, float *partial, float *norms,
                              float *scales, int *err, int wait_limit, cudaStream_t stream, int *launches);

// partial: scratch of at least 2 * M * reduce_row(nchunks) floats; out[m] = ||now - then|| / ||then||
// (out may be host memory that the device can write to).  *released is written with a release at system
// scope, behind all that is in front in the stream.  Two launches.
cudaError_t launch_rel_change(const Chunk *chunks, long long nchunks, const float *const *now,
                              const float *const *then, int nt, int M, float *partial, float *out, float *released,
                              int *err, int wait_limit, cudaStream_t stream);

// Norms of a diagnostics step: partial [DIAG_KINDS][M][nchunks * *parts] sums of squares of the parts of a chunk,
// tstart [nt + 1] first chunk of every tensor; writes per_tensor [DIAG_KINDS][M][nt] and totals
// [DIAG_KINDS][M] (floats; may be host memory that the device can write to), and *released as above.  One launch.
cudaError_t launch_diag_norms(const float *partial, long long nchunks, const int *parts, const long long *tstart,
                              int nt, int M, float *per_tensor, float *totals, float *released,
                              cudaStream_t stream);

// Every element of the m_dst destination replicas := mean over the m_src source replicas.
// src / dst are device tables indexed [m * nt + tensor].
cudaError_t launch_mean_fill(const Chunk *chunks, long long nchunks, const float *const *src,
                             int m_src, float *const *dst, int m_dst, int nt, cudaStream_t stream);

}  // namespace desloc
