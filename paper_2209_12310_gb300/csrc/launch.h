// launch.h -- host-side launchers of the device kernels (internal).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace ch {

struct Ctl;

// Launch of a kernel that may start before the stream's last kernel ends: as soon
// as every block of that one has executed griddepcontrol.launch_dependents (or
// ended).  The kernel itself ends with griddepcontrol.wait, so that what follows
// it in the stream follows both.
template <typename... KArgs, typename... Args>
inline void launch_beside(void (*kernel)(KArgs...), int grid, int threads, size_t smem, cudaStream_t s,
                          const Args&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

void launch_init(Ctl* ctl, int mode, cudaStream_t s);
void launch_sample(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, unsigned switch_at, int grid,
                   cudaStream_t s, int labels = 0);
void launch_main(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, uint64_t* raw_xy,
                 uint32_t* raw_idx, unsigned switch_at, uint32_t* keys, uint64_t* vals, int two_pass, int grid,
                 cudaStream_t s);
void launch_main_labels(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, uint64_t* raw_xy,
                        uint32_t* raw_idx, unsigned switch_at, uint32_t* keys, uint64_t* vals, int two_pass, int grid,
                        cudaStream_t s);
// The dense data's pass (star bins, star polygon, filter): the bins and the
// polygon live in the workspace.
void launch_dense(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, void* bins, void* poly,
                  uint64_t* raw_xy, uint32_t* raw_idx, uint32_t* keys, uint64_t* vals, int sms, cudaStream_t s);
void launch_small(const float* pts, long long n, Ctl* ctl, uint32_t* keys, uint64_t* vals, int32_t* out_idx,
                  int64_t* out_n, cudaStream_t s);
void launch_post(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, const uint64_t* raw_xy,
                 const uint32_t* raw_idx, uint32_t* keys, uint64_t* vals, unsigned* tiles, int32_t* out_idx,
                 int64_t* out_n, int grid, cudaStream_t s);
void launch_labels(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, const uint64_t* raw_xy,
                   const uint32_t* raw_idx, uint8_t* labels, int grid, cudaStream_t s);
size_t star_bins_bytes(int sms);   // a block's bins each, and the merged ones
size_t star_poly_bytes();
void launch_filter_output(const Ctl* ctl, long long n, int32_t* out_ext8, int64_t* out_counts4, cudaStream_t s);

// The large-survivor path without a sort (queues.cu); tiles: tiles_bytes() of
// the workspace, its first kPtGroups words the records per group, which the post
// pass clears when it picks the tiles.
void launch_large(Ctl* ctl, const uint32_t* kA, const uint64_t* vA, uint32_t* kB, uint64_t* vB, unsigned* tiles, int* cu,
                  int* cv, int* ci, long long n, int32_t* out_idx, int64_t* out_n, int grid, cudaStream_t s);
size_t tiles_bytes();
cudaError_t configure_large_kernel();
// The large-survivor path by radix sort and merge tree (sort.cuh, hull.cu).
void launch_sort(Ctl* ctl, uint32_t* kA, uint64_t* vA, uint32_t* kB, uint64_t* vB, unsigned long long* status, int* cu,
                 int* cv, int* ci, int* clen, int* counters, int ctcap, const float* pts, long long n, int32_t* out_idx,
                 int64_t* out_n, int grid, cudaStream_t s);
size_t chain_smem_bytes();
cudaError_t configure_hull_kernels();
cudaError_t configure_filter_kernels();
cudaError_t configure_post_kernel();
long long sample_tiles_host(long long ntiles);

// Occupancy (resident blocks per SM at each kernel's launch shape).
cudaError_t occupancy_filter(int* main_k, int* labels);
cudaError_t occupancy_post(int* post);
cudaError_t occupancy_sort(int* sort);

}  // namespace ch
