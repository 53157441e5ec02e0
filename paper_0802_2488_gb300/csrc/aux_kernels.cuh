// Launchers of the mask and labelling kernels (aux_kernels.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace epfft {
constexpr int GRID_SMS = 152;  // SMs of a GB300: caps of grid sizes, nothing depends on it
#ifdef __CUDACC__
// Pixel i is a void iff (SplitMix64 output i of `seed`) >> 11 < thr, where the
// i-th output of SplitMix64 is the 64-bit finaliser of seed + (i+1) gamma,
// gamma = 0x9e3779b97f4a7c15 (Steele, Lea & Flood's generator).
__device__ __forceinline__ uint8_t void_bit(int64_t i, uint64_t seed, uint64_t thr) {
  uint64_t z = seed + (uint64_t)(i + 1) * 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  z ^= z >> 31;
  return (uint8_t)((z >> 11) < thr);
}
#endif
cudaError_t launch_mask(uint8_t* mask, int64_t n, uint64_t seed, uint64_t thr, cudaStream_t s);
// n_img images of L*L flags -> labels (smallest linear index of the cluster,
// -1 off the flags) and counts_dev[n_img]; *err_dev set if a bound tripped.
// labels = false: the counts only (lab is scratch).  Three kernels.
cudaError_t launch_label(const uint8_t* flags, int32_t* lab, int64_t n_img, int L, int periodic,
                         int32_t* counts_dev, int32_t* err_dev, cudaStream_t s, bool labels = true);
// Scratch of the void-plastic clusters (Sec. 3), per pixel of every image,
// used at the roots of the first labelling; stats: 4 counts per image
// (clusters, pixels of the largest, clusters without a plastic pixel, plastic
// pixels), zeroed by the caller.
struct VpScratch {
  unsigned long long* best;  // nearest void of a void-free cluster: d^2 2^32 + index
  int32_t *target, *final_root, *size;
  uint8_t *has_void, *has_pl;
  int32_t* stats;
};
constexpr size_t VP_SCRATCH_BYTES = 22;  // per pixel
// Clusters of mask | plastic of n_img images (one mask) with the scratch
// initialised, clusters holding a void marked and the plastic pixels counted.
cudaError_t launch_vp_label(const uint8_t* mask, const uint8_t* plastic, int32_t* lab, int64_t n_img, int L,
                            const VpScratch& vp, int32_t* err_dev, cudaStream_t s);
// FP64 FMA throughput probe: `blocks` CTAs of 256 threads, each thread runs
// FMA_CHAINS independent chains of n dependent FMAs (2 flops each).
constexpr int FMA_CHAINS = 8, FMA_THREADS = 256;
cudaError_t launch_fp64_fma(int blocks, int n, double* sink, cudaStream_t s);
}  // namespace epfft
