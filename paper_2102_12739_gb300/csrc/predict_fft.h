// The producer's fused transform (predict_fft.cu): internal interface.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

struct dg_predict_fft;

// Whether images of n x n pixels have a fused transform.
bool dg_predict_fft_supported(int n);
cudaError_t dg_predict_fft_create(dg_predict_fft **out, int n, int nz, int per_pass, int device);
void dg_predict_fft_destroy(dg_predict_fft *p);
cudaError_t dg_predict_fft_execute(dg_predict_fft *p, cudaStream_t st, double theta, const float *image,
                                   const float *taper, int n_subgrids, const int32_t *uv_offsets,
                                   const double *w_planes, float *subgrids_out);
