// nep_fallback.cu -- flags of the per-atom fallback from the student to the teacher model.
//
// The student's kernel flags every atom whose scaled descriptors leave the training range (Fallback in
// nep_descriptor.cuh), gives it a zero adjoint row and leaves only its LJ energy in the site energy.  The
// teacher (plain float32) is then evaluated on the flagged atoms by k_nep_wide_list (nep_wide.cu), so
// that E = sum_i U_i^(model of i) and F = -grad E with each atom's own model (the LJ term, shared by both
// models, stays in the student's kernels).  That kernel runs on a fixed grid and loops over the flagged list,
// whose length it reads on the device, so an MD step stays one CUDA graph.
#include <algorithm>

#include "nep_descriptor.cuh"

namespace nep {
namespace {

constexpr int FB_BLOCK = 128;

// flags[id[i]] = 1 for every flagged atom i (flags zeroed by the caller).
__global__ void k_fb_flags(const int *__restrict__ list, const int *__restrict__ count, int cap,
                           const int *__restrict__ id, int *__restrict__ flags) {
  const int m = min(*count, cap);
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < m; s += gridDim.x * blockDim.x) flags[id[list[s]]] = 1;
}

int fb_grid(int cap) { return std::max(1, std::min((cap + FB_BLOCK - 1) / FB_BLOCK, 152 * 8)); }

}  // namespace

cudaError_t launch_fallback_flags(const int *list, const int *count, int cap, const int *id, int *flags,
                                  cudaStream_t st) {
  if (cap <= 0) return cudaSuccess;
  k_fb_flags<<<fb_grid(cap), FB_BLOCK, 0, st>>>(list, count, cap, id, flags);
  return cudaGetLastError();
}

}  // namespace nep
