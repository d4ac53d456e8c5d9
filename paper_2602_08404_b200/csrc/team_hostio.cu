// Copies of team_moe_forward_host between the pinned staging block and its device mirror, as kernels.
//
// A copy node of a graph waits for the whole grid in front of it, is handed to a copy engine and hands back: 15 us from
// the end of the step's kernel to the end of the 32 KB copy of y, for 1 us of PCIe time.  A kernel that is chained with
// programmatic dependent launch reads or writes the pinned block (mapped into the device's address space) as soon as
// its predecessor is done: the call of 4 rows 70.5 -> 63.1 us.  Up to kHostIoMaxBytes per direction.  Both ways at hidden 2048
// and few experts, copy engine and kernel, us per call: 8 rows 76 and 60, 32 rows 93 and 79, 128 rows 202 and 184, 256 rows
// (1 MB of x, 2 MB of y) 345 and 322, 1024 rows 1189 and 1163, which is as much as two runs differ there: PCIe and the host's own
// copies bind larger blocks, and an engine moves those without taking SMs.
#include "team_common.cuh"

namespace team {

__global__ void __launch_bounds__(256) k_host_in(HostIn a) {
  asm volatile("griddepcontrol.wait;" ::: "memory");        // the preceding step's kernels have read the block
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int i = blockIdx.x * 256 + threadIdx.x; i < a.pieces[HostIn::kParts - 1]; i += gridDim.x * 256) {
    int part = 0;
#pragma unroll
    for (int q = 0; q + 1 < HostIn::kParts; ++q) part += i >= a.pieces[q];
    const int at = a.first[part] + i - (part > 0 ? a.pieces[part - 1] : 0);
    a.dst[at] = a.src[at];
  }
}

__global__ void __launch_bounds__(256) k_host_out(const uint4* __restrict__ src, uint4* __restrict__ dst, int n) {
  asm volatile("griddepcontrol.wait;" ::: "memory");        // y is complete
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) dst[i] = __ldcg(src + i);
}

static cudaLaunchConfig_t copy_launch(int pieces, cudaLaunchAttribute* attr, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  const int blocks = (pieces + 255) / 256;
  cfg.gridDim = dim3(blocks < 148 ? blocks : 148);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr->val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

cudaError_t launch_host_in(const HostIn& a, cudaStream_t s) {
  cudaLaunchAttribute attr;
  const cudaLaunchConfig_t cfg = copy_launch(a.pieces[HostIn::kParts - 1], &attr, s);
  return cudaLaunchKernelEx(&cfg, k_host_in, a);
}

cudaError_t launch_host_out(const void* src, void* dst, size_t bytes, cudaStream_t s) {
  cudaLaunchAttribute attr;
  const int n = (int)(bytes / 16);
  const cudaLaunchConfig_t cfg = copy_launch(n, &attr, s);
  return cudaLaunchKernelEx(&cfg, k_host_out, static_cast<const uint4*>(src), static_cast<uint4*>(dst), n);
}

}  // namespace team
