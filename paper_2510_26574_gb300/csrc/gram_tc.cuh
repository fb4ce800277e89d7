// Tensor-core (tcgen05) weighted Grams of an FP32 factor; see gram_tc.cu.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace kevd {

// True when F can be read by the tensor map (16-byte aligned, ldf a multiple
// of 4, N < 2^31) and KEVD_GRAM=ffma does not ask for the FFMA kernel.
bool gram_tc_eligible(const float* F, int64_t ldf, int64_t N, int rank);

// Rows per split (a multiple of 64) and the split count for ntri tile pairs.
int64_t gram_tc_per(int64_t N, int64_t ntri, int nsm, int* nsplit);

// Column maxima, magic numbers and the Gram kernel: gpart receives
// nsplit x ntri x 2 x 128 x 128 FP32 partials (A, then C) for the FP64 split
// reduction.  wa, wc: FP32 weights zero-padded to a multiple of 64 rows (wc
// NULL: the first Gram only); cmax, mag: 3 x rank scratch; flags bit 2 is set
// if a bounded wait gave up.
cudaError_t launch_gram_tc(const float* F, int64_t ldf, int64_t N, int rank, const float* wa, const float* wc,
                           unsigned* cmax, float* mag, float* gpart, uint16_t* planes, int* flags, int nb, int ntri,
                           int64_t per, int nsplit, int nsm, cudaStream_t s);
// Bytes of `planes` (16-byte aligned; 0: the kernel that slices its own tiles is used, as
// with planes == NULL).
size_t gram_tc_plane_bytes(int64_t N, int rank, int ngram, int nsm);

// FP64 factor: weighted Grams on the tensor cores at FP64 accuracy (gram_oz.cu),
// A = (sa F)^T (sa F) and C = (sc F)^T (sc F).  sa, sc: N row scales (sc NULL: A
// only); sa_hi, sc_hi: N words of scratch each; cmax, Ecol: 2 x rank scratch; gpart:
// gram_oz_partial_doubles(...); planes: gram_oz_plane_bytes(...) bytes, 16-byte aligned
// (the digit planes of one slab of rows).  Any ldf and alignment of F.  Writes A (and
// C) in full, exactly symmetric.
bool gram_oz_eligible(int64_t N, int rank);
size_t gram_oz_partial_doubles(int64_t N, int rank, int ngram, int nsm);
size_t gram_oz_plane_bytes(int64_t N, int rank, int ngram);
cudaError_t launch_gram_oz(const double* F, int64_t ldf, int64_t N, int rank, const double* sa, const double* sc,
                           uint32_t* sa_hi, uint32_t* sc_hi, uint32_t* cmax, int* Ecol, double* gpart,
                           uint16_t* planes, int* flags, double* A, double* C, int nsm, cudaStream_t s);

// The same for one panel of N <= P rows with seven digits (the error of the FP64-pipe
// kernel), acc adding to A and C; gpart and planes as sized for P rows.
size_t gram_oz_panel_partial_doubles(int64_t P, int rank, int nsm);
size_t gram_oz_panel_plane_bytes(int64_t P, int rank);
cudaError_t launch_gram_oz_panel(const double* F, int64_t ldf, int64_t P, int64_t N, int rank, const double* sa,
                                 const double* sc, uint32_t* sa_hi, uint32_t* sc_hi, uint32_t* cmax, int* Ecol,
                                 double* gpart, uint16_t* planes, int* flags, double* A, double* C, int acc, int nsm,
                                 cudaStream_t s);

}  // namespace kevd
