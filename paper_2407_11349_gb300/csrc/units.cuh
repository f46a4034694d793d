// What the translation units use of one another, declared once.
#pragma once

#include <string>
#include <vector>

#include "common.cuh"

namespace hk {

// kernels.cu
__global__ void k_setup(double*, double*, double*, const int32_t*, int32_t, const double*, int64_t,
                        int64_t, int, double*, float*, int32_t*, int32_t*, double*, int*);
__global__ void k_prep(const __grid_constant__ EvalDesc, const EvalDesc*, const hawkes_params*,
                       const __grid_constant__ hawkes_params, int, int, int, int, const uint64_t*, int*);
void launch_finalize(cudaStream_t, dim3, const EvalDesc&, const EvalDesc*, int64_t, int64_t, int,
                     const double*, int, double*, double*, double*);
void launch_rows64(cudaStream_t, int, int, const EvalDesc&, const EvalDesc*, int, int, int64_t, double*, double*);
void launch_flushfix(cudaStream_t, int, int, const EvalDesc&, const EvalDesc*, int, int, int64_t, int64_t, double*,
                     double*, double*);
cudaError_t rows_setup_attributes();
__global__ void k_tri_area(const double*, int32_t, double*, int*);
__global__ void k_tri_county(const int32_t*, int32_t, int32_t, double*, int32_t*, int32_t*, int*);
__global__ void k_tri_check(const int32_t*, int32_t, int32_t, int*);
__global__ void k_resample(const __grid_constant__ EvalDesc, uint64_t);
__global__ void k_wait_selftest(int*);

// sweep.cu
cudaError_t sweep_setup_attributes();
int sweep_num_variants();
int sweep_blocks_per_sm(int v);
int sweep_variant_rows(int v);
SweepPlan sweep_plan(const int64_t* ns, size_t count, int sms, int v, int chunk, bool band);
std::string sweep_plans_key(const int64_t* ns, size_t count, int sms);
std::vector<int4> sweep_items(int64_t n, const SweepPlan& pl, int v);
std::vector<int4> sweep_items_batch(const std::vector<int64_t>& ns, const SweepPlan& pl, int v, int order);
std::vector<int4> sweep_band(const std::vector<int64_t>& ns, const SweepPlan& pl, int v);
cudaError_t launch_sweep(hawkes_ctx* c, bool sym, int64_t row_begin, int64_t row_end, bool bgt, bool ll);
cudaError_t launch_sweep_list(hawkes_ctx* c, const int4* items, int nitems, int nband, bool bgt, bool ll);
cudaError_t launch_sweep_batch(cudaStream_t st, const SweepPlan& pl, int sms, int variant, int grid,
                               const ProbDesc* probs, int nprobs, const int4* items, int nitems, int nband,
                               int* ctr, bool bgt, bool ll);

// sweep_split.cu
cudaError_t split_setup_attributes();
int split_rows();
cudaError_t launch_sweep_split(cudaStream_t st, int sms, const ProbDesc& one, const ProbDesc* probs,
                               int nprobs, const int4* items, int nitems, int* ctr, bool bgt, bool ll, bool band);

// sweep_group.cu
bool group_kc_supported(int kc);
int group_blocks_per_sm(int kc);
cudaError_t group_setup_attributes();
std::vector<int4> group_items(const std::vector<int64_t>& ns, int kc, int chunk);
cudaError_t launch_group_stage(cudaStream_t st, int sms, const GroupDesc& gd,
                               const Rec* const* recs, const double* t, int kc, float4* out);
cudaError_t launch_sweep_group(cudaStream_t st, int kc, int grid, const GroupDesc* groups,
                               int ngroups, const int4* items, int nitems, int* ctr);

// sweep_spatial.cu
cudaError_t spatial_setup_attributes();
int spatial_build(hawkes_ctx* c, const hawkes_params* p, const hawkes_params* d_p);
cudaError_t spatial_launch(hawkes_ctx* c, int model1, int llonly);
void spatial_free(hawkes_ctx* c);
int spatial_set_window(hawkes_ctx* c, int64_t window);
void spatial_invalidate(hawkes_ctx* c);

// rows64.cu
int rows64_segments(int64_t rows, int sms);
size_t rows64_scratch(int64_t n, int sms);
cudaError_t pairs64_setup_attributes();
cudaError_t launch_pairs64(const hawkes_ctx* c, bool model1, bool bgt, int64_t rb, int64_t re, double* out);

// tune_cache.cu
int tune_cache_get(const char* path, const char* key, int* variant, int* chunk, int* order, double* ms, int* kc);
int tune_cache_put(const char* path, const char* key, int variant, int chunk, int order, double ms, int kc);
int log2_ceil(double v);
std::string device_key();

}  // namespace hk
