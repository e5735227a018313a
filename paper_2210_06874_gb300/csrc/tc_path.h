// tc_path.h -- entry points of the mixed-precision (tensor-core) path (internal).
#pragma once

#include <cuda_runtime.h>

#include "ctx.h"
#include "launch.h"

namespace hmc {

int tc_ctx_init(hmc_ctx* c);   // FP16 split of E, FP32 workspaces
void tc_ctx_free(hmc_ctx* c);
int tc_apply(hmc_ctx* c, const double* phi, const float2* in, float2* out, bool dag,
             cudaStream_t s);
int tc_cg(hmc_ctx* c, const double* phi, const double2* chi, double2* x, double tol,
          int max_iter, cudaStream_t s);
int tc_trajectory(hmc_ctx* c, const TrajArgs& a, cudaStream_t s);

// E by the series (series_kernels.cu): the automatic choice (operand_mode and
// cluster_mode 0) where it exists.
bool series_chosen(const hmc_ctx* c);
int series_ctx_init(hmc_ctx* c);
int series_apply(const ChainView& v, const double* phi, const float2* in, float2* out, bool dag,
                 cudaStream_t s);
int series_cg(hmc_ctx* c, const double* phi, const double2* chi, double2* x, double tol,
              int max_iter, cudaStream_t s);
int series_trajectory(hmc_ctx* c, const TrajArgs& a, cudaStream_t s);
// The series' batch kernel, its threads and the bytes of shared memory a CTA has for
// it; null on a CUDA error.
const void* series_batch_kernel(unsigned* smem, int* threads);

struct TcBatch;
int tc_batch_create(const hmc_params* p, int n, TcBatch** out);
void tc_batch_destroy(TcBatch* b);
void tc_batch_offsets(const TcBatch* b, long long* off);
int tc_batch_size(const TcBatch* b);
int tc_batch_trajectory(TcBatch* b, double* phi, uint64_t seed, uint64_t traj,
                        hmc_traj_out* out, cudaStream_t caller);

}  // namespace hmc
