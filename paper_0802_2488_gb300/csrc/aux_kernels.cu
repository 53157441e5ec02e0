// Void mask (Sec. 2) and plastic-cluster labelling (Sec. 3) kernels.
#include "aux_kernels.cuh"

namespace epfft {

__global__ void mask_kernel(uint8_t* __restrict__ mask, int64_t n, uint64_t seed, uint64_t thr) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    mask[i] = void_bit(i, seed, thr);
  }
}

// --- 4-connected clusters by concurrent union-find ------------------------
// lab[x] is a parent index (<= x) for flagged pixels and -1 otherwise; a
// root is its own parent.  Unions always hang the larger root below the
// smaller one, so each final root is the smallest linear index of its
// cluster, which makes the labels canonical.  Pointer chases are bounded by
// the image size; a chase that exceeds it raises *err and stops.
//
// Three kernels, all images of a call in each: the clusters of a tile in
// shared memory (a row's runs of 32 pixels come from a ballot, so that only
// vertical neighbours and run ends unite), the unions across tile borders in
// global memory, and the roots (labels and counts).  Against one union per
// neighbour pair in global memory and one count per root on a shared address
// (10 images of L = 1024, half flagged: 140 us an image) this leaves the
// traffic of a byte read and about three passes over the labels.

__device__ __forceinline__ int32_t find_root(const int32_t* lab, int32_t x, int32_t bound, int32_t* err) {
  for (int32_t it = 0; it < bound; it++) {
    const int32_t p = __ldcg(lab + x);
    if (p == x) return x;
    x = p;
  }
  atomicExch(err, 1);
  return x;
}

__device__ __forceinline__ void unite(int32_t* lab, int32_t a, int32_t b, int32_t bound, int32_t* err) {
  for (int32_t it = 0; it < bound; it++) {
    a = find_root(lab, a, bound, err);
    b = find_root(lab, b, bound, err);
    if (a == b) return;
    if (a > b) {
      const int32_t t = a;
      a = b;
      b = t;
    }
    const int32_t old = atomicMin(lab + b, a);
    if (old == b) return;
    b = old;
  }
  atomicExch(err, 1);
}

constexpr int CCL_NT = 256;

// The same on a tile's labels in shared memory.
__device__ __forceinline__ int tile_root(volatile int* s, int x, int bound, int32_t* err) {
  for (int it = 0; it < bound; it++) {
    const int p = s[x];
    if (p == x) return x;
    x = p;
  }
  atomicExch(err, 1);
  return x;
}
__device__ __forceinline__ void tile_unite(int* s, int a, int b, int bound, int32_t* err) {
  for (int it = 0; it < bound; it++) {
    a = tile_root(s, a, bound, err);
    b = tile_root(s, b, bound, err);
    if (a == b) return;
    if (a > b) {
      const int t = a;
      a = b;
      b = t;
    }
    const int old = atomicMin(s + b, a);
    if (old == b) return;
    b = old;
  }
  atomicExch(err, 1);
}

// Clusters within TW x TH tiles (one CTA each; blockIdx.x runs over the tiles
// of every image).  VP: the flags are mask | flags (void-plastic phase), the
// scratch of the tile's roots is initialised and the flags' pixels counted.
template <int TW, int TH, bool VP>
__global__ void __launch_bounds__(CCL_NT)
ccl_tile(const uint8_t* __restrict__ flags, const uint8_t* __restrict__ mask, int32_t* __restrict__ lab, int L,
         VpScratch vp, int32_t* err) {
  constexpr int PX = TW * TH, SEG = TW < 32 ? TW : 32;
  __shared__ int s[PX];
  const int tx = L / TW, per = tx * (L / TH);
  const int64_t img = blockIdx.x / per;
  const int t = (int)(blockIdx.x - img * per);
  const int x0 = (t % tx) * TW, y0 = (t / tx) * TH;
  const int64_t base = img * (int64_t)L * L;
  const int lane = threadIdx.x & 31, seg0 = lane & ~(SEG - 1);
  int n_fl = 0;
  for (int k0 = 0; k0 < PX; k0 += CCL_NT) {
    const int k = k0 + threadIdx.x;
    bool f = false;
    if (k < PX) {
      const int x = (y0 + k / TW) * L + x0 + k % TW;
      const bool p = flags[base + x] != 0;
      f = p || (VP && mask[x] != 0);
      if (VP) n_fl += p;
    }
    const unsigned m = __ballot_sync(0xffffffffu, f);
    // the lane after the last unflagged one below this in the run's segment
    const unsigned gap = ~m & ((1u << lane) - 1u) & (~0u << seg0);
    const int start = gap ? 32 - __clz((int)gap) : seg0;
    if (k < PX) s[k] = f ? k - (lane - start) : -1;
  }
  if (VP) {
    for (int o = 16; o > 0; o >>= 1) n_fl += __shfl_down_sync(0xffffffffu, n_fl, o);
    if (lane == 0 && n_fl) atomicAdd(vp.stats + 4 * img + 3, n_fl);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < PX; k += CCL_NT) {
    if (s[k] < 0) continue;
    const int lx = k % TW;
    if (lx > 0 && lx % SEG == 0 && s[k - 1] >= 0) tile_unite(s, k - 1, k, PX + 1, err);
    // the pair above; implied by the pair to the left when that joins the same runs
    if (k >= TW && s[k - TW] >= 0 && !(lx % SEG > 0 && s[k - 1] >= 0 && s[k - TW - 1] >= 0))
      tile_unite(s, k - TW, k, PX + 1, err);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < PX; k += CCL_NT) {
    const int x = (y0 + k / TW) * L + x0 + k % TW;
    if (s[k] < 0) {
      lab[base + x] = -1;
      continue;
    }
    const int r = tile_root(s, k, PX + 1, err);
    lab[base + x] = (y0 + r / TW) * L + x0 + r % TW;
    if (VP && r == k) {
      vp.best[base + x] = ~0ull;
      vp.final_root[base + x] = L * L;
      vp.size[base + x] = 0;
      vp.has_void[base + x] = 0;
      vp.has_pl[base + x] = 0;
    }
  }
}

// Unions across the tiles' right and lower borders (and the image's, where
// periodic).  A pair whose neighbour along the border is flagged on both sides
// too, in the same tiles, is implied by that one.
__global__ void __launch_bounds__(CCL_NT) ccl_border(int32_t* lab, int64_t n_img, int L, int TW, int TH, int periodic,
                                                     int32_t* err) {
  const int64_t LL = (int64_t)L * L;
  const int nv = (L / TW) * L, np = nv + (L / TH) * L;
  for (int64_t img = blockIdx.y; img < n_img; img += gridDim.y) {
    int32_t* l = lab + img * LL;
    for (int p = blockIdx.x * CCL_NT + threadIdx.x; p < np; p += gridDim.x * CCL_NT) {
      const bool vert = p < nv;
      const int q = vert ? p : p - nv;
      const int e = ((q / L) + 1) * (vert ? TW : TH), u = q % L;  // e: first line beyond the border
      if (e == L && !periodic) continue;
      const int a = vert ? u * L + e - 1 : (e - 1) * L + u;
      const int b = vert ? u * L + (e & (L - 1)) : (e & (L - 1)) * L + u;
      if (a == b || __ldcg(l + a) < 0 || __ldcg(l + b) < 0) continue;
      const int back = vert ? L : 1;
      if (u % (vert ? TH : TW) != 0 && __ldcg(l + a - back) >= 0 && __ldcg(l + b - back) >= 0) continue;
      unite(l, a, b, (int32_t)LL + 1, err);
    }
  }
}

// Roots: counts[img] = clusters; WRITE: every label becomes its root (a chain
// only ever shortens meanwhile, so concurrent chases stay valid); VP: clusters
// that hold a void are marked.
template <bool WRITE, bool VP>
__global__ void __launch_bounds__(CCL_NT) ccl_roots(int32_t* lab, const uint8_t* __restrict__ mask, int64_t n_img,
                                                    int L, VpScratch vp, int32_t* counts, int32_t* err) {
  const int64_t LL = (int64_t)L * L;
  const int32_t bound = (int32_t)(LL + 1);
  __shared__ int wc[CCL_NT / 32];
  for (int64_t img = blockIdx.y; img < n_img; img += gridDim.y) {
    int32_t* l = lab + img * LL;
    int n = 0;
    for (int64_t x = blockIdx.x * (int64_t)CCL_NT + threadIdx.x; x < LL; x += (int64_t)gridDim.x * CCL_NT) {
      const int32_t p = __ldcg(l + x);
      if (p < 0) continue;
      n += p == x;
      if (WRITE || VP) {
        const int32_t r = p == x ? p : find_root(l, p, bound, err);
        if (WRITE && r != p) l[x] = r;
        if (VP && mask[x]) vp.has_void[img * LL + r] = 1;
      }
    }
    if (counts) {
      n = __reduce_add_sync(0xffffffffu, n);
      if ((threadIdx.x & 31) == 0) wc[threadIdx.x >> 5] = n;
      __syncthreads();
      if (threadIdx.x == 0) {
        int s = 0;
        for (int w = 0; w < CCL_NT / 32; w++) s += wc[w];
        if (s) atomicAdd(counts + img, s);
      }
      __syncthreads();
    }
  }
}

static int grid_for(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > GRID_SMS * 32) g = GRID_SMS * 32;
  if (g < 1) g = 1;
  return (int)g;
}

cudaError_t launch_mask(uint8_t* mask, int64_t n, uint64_t seed, uint64_t thr, cudaStream_t s) {
  mask_kernel<<<grid_for(n), 256, 0, s>>>(mask, n, seed, thr);
  return cudaGetLastError();
}

template <bool VP>
static cudaError_t tile_launch(const uint8_t* flags, const uint8_t* mask, int32_t* lab, int64_t n_img, int L,
                               const VpScratch& vp, int32_t* err, int* tw, int* th, cudaStream_t s) {
  *tw = L < 64 ? L : 64;
  *th = L < 64 ? L : 32;
  const int64_t tiles = n_img * (L / *tw) * (L / *th);
  if (tiles > 0x7fffffff) return cudaErrorInvalidValue;
  const unsigned g = (unsigned)tiles;
  switch (*tw) {
    case 2: ccl_tile<2, 2, VP><<<g, CCL_NT, 0, s>>>(flags, mask, lab, L, vp, err); break;
    case 4: ccl_tile<4, 4, VP><<<g, CCL_NT, 0, s>>>(flags, mask, lab, L, vp, err); break;
    case 8: ccl_tile<8, 8, VP><<<g, CCL_NT, 0, s>>>(flags, mask, lab, L, vp, err); break;
    case 16: ccl_tile<16, 16, VP><<<g, CCL_NT, 0, s>>>(flags, mask, lab, L, vp, err); break;
    case 32: ccl_tile<32, 32, VP><<<g, CCL_NT, 0, s>>>(flags, mask, lab, L, vp, err); break;
    default: ccl_tile<64, 32, VP><<<g, CCL_NT, 0, s>>>(flags, mask, lab, L, vp, err); break;
  }
  return cudaGetLastError();
}

// CTAs over one image's pixels and over the images
static dim3 image_grid(int64_t px, int64_t n_img) {
  const int64_t y = n_img < 32768 ? n_img : 32768;
  int64_t x = (px + 4 * CCL_NT - 1) / (4 * CCL_NT), most = (GRID_SMS * 16 + y - 1) / y;
  if (x > most) x = most;
  return dim3((unsigned)(x < 1 ? 1 : x), (unsigned)y);
}

cudaError_t launch_label(const uint8_t* flags, int32_t* lab, int64_t n_img, int L, int periodic,
                         int32_t* counts_dev, int32_t* err_dev, cudaStream_t s, bool labels) {
  cudaError_t e = cudaMemsetAsync(counts_dev, 0, sizeof(int32_t) * n_img, s);
  if (e != cudaSuccess) return e;
  const int64_t LL = (int64_t)L * L;
  int tw, th;
  if ((e = tile_launch<false>(flags, nullptr, lab, n_img, L, VpScratch{}, err_dev, &tw, &th, s)) != cudaSuccess) return e;
  const int64_t borders = (int64_t)L * (L / tw) + (int64_t)L * (L / th);
  ccl_border<<<image_grid(borders, n_img), CCL_NT, 0, s>>>(lab, n_img, L, tw, th, periodic, err_dev);
  if (labels)
    ccl_roots<true, false><<<image_grid(LL, n_img), CCL_NT, 0, s>>>(lab, nullptr, n_img, L, VpScratch{}, counts_dev, err_dev);
  else
    ccl_roots<false, false><<<image_grid(LL, n_img), CCL_NT, 0, s>>>(lab, nullptr, n_img, L, VpScratch{}, counts_dev, err_dev);
  return cudaGetLastError();
}

cudaError_t launch_vp_label(const uint8_t* mask, const uint8_t* plastic, int32_t* lab, int64_t n_img, int L,
                            const VpScratch& vp, int32_t* err_dev, cudaStream_t s) {
  int tw, th;
  const cudaError_t e = tile_launch<true>(plastic, mask, lab, n_img, L, vp, err_dev, &tw, &th, s);
  if (e != cudaSuccess) return e;
  const int64_t borders = (int64_t)L * (L / tw) + (int64_t)L * (L / th);
  ccl_border<<<image_grid(borders, n_img), CCL_NT, 0, s>>>(lab, n_img, L, tw, th, 1, err_dev);
  ccl_roots<true, true><<<image_grid((int64_t)L * L, n_img), CCL_NT, 0, s>>>(lab, mask, n_img, L, vp, nullptr, err_dev);
  return cudaGetLastError();
}

// --- FP64 FMA throughput ---------------------------------------------------
// Every thread advances FMA_CHAINS independent chains x <- x a + b for n
// steps (a slightly below 1, so the values stay bounded); the sum is stored
// only if it equals an impossible value, so the chains cannot be removed.
__global__ void __launch_bounds__(FMA_THREADS) fp64_fma_kernel(int n, double a, double b, double* sink) {
  double x[FMA_CHAINS];
#pragma unroll
  for (int i = 0; i < FMA_CHAINS; i++) x[i] = 1e-3 * threadIdx.x + i;
#pragma unroll 4
  for (int k = 0; k < n; k++)
#pragma unroll
    for (int i = 0; i < FMA_CHAINS; i++) x[i] = fma(x[i], a, b);
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < FMA_CHAINS; i++) s += x[i];
  if (s == -1234.5) *sink = s;
}

cudaError_t launch_fp64_fma(int blocks, int n, double* sink, cudaStream_t s) {
  fp64_fma_kernel<<<blocks, FMA_THREADS, 0, s>>>(n, 0.999999, 1e-6, sink);
  return cudaGetLastError();
}

}  // namespace epfft
