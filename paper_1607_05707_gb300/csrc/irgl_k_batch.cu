// Batched kernels: admission (initial values + pending sources) and the
// persistent multi-query Iterate (one cooperative launch for all instances).
#include "irgl_launch.h"

namespace irgl {

// NF: near-far may be on; LOCAL: CTA-local sub-rounds. Sub-rounds without near-far have a
// kernel of their own: in the one with both, min-label CC of 24 meshes of 0.2 M vertices took
// 25.8 ms, 23.8 in its own (SSSP 12.7 and 12.2 ms).
template <int CTA, bool NF, bool LOCAL>
__global__ void __launch_bounds__(CTA, MinBlocks<CTA>::value) k_batch_iterate(BParams p) {
  __shared__ BatchSmem<CTA, NF, NF && LOCAL> bs;
  iterate_batch<CTA, NF, LOCAL>(p, bs);
}

__global__ void __launch_bounds__(256) k_batch_fill(AdmitParams a) { admit_fill(a); }
__global__ void __launch_bounds__(256) k_batch_sources(AdmitParams a) { admit_sources(a); }

// Results out of the packed arena: out[i] = ds[i] >> 32 (the value half),
// two entries per thread per step.
__global__ void __launch_bounds__(256) k_extract_values(const unsigned long long* __restrict__ ds,
                                                        uint32_t* __restrict__ out, uint64_t n) {
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride)
    __stcs(out + i, static_cast<uint32_t>(__ldcs(ds + i) >> 32));
}

namespace {

template <int CTA>
cudaError_t launch_b(uint32_t grid, const BParams& p, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(CTA);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (p.local_rounds != 0)
    return p.delta != 0 ? cudaLaunchKernelEx(&cfg, k_batch_iterate<CTA, true, true>, p)
                        : cudaLaunchKernelEx(&cfg, k_batch_iterate<CTA, false, true>, p);
  return p.delta != 0 ? cudaLaunchKernelEx(&cfg, k_batch_iterate<CTA, true, false>, p)
                      : cudaLaunchKernelEx(&cfg, k_batch_iterate<CTA, false, false>, p);
}

}  // namespace

cudaError_t launch_batch_iterate(uint32_t cta, uint32_t grid, const BParams& p, cudaStream_t s) {
  switch (cta) {
    case 128: return launch_b<128>(grid, p, s);
    case 256: return launch_b<256>(grid, p, s);
    case 512: return launch_b<512>(grid, p, s);
    case 1024: return launch_b<1024>(grid, p, s);
  }
  return cudaErrorInvalidValue;
}

template <bool NF, bool LOCAL>
cudaError_t occ_b(uint32_t cta, int* nb) {
  switch (cta) {
    case 128: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, k_batch_iterate<128, NF, LOCAL>, 128, 0);
    case 256: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, k_batch_iterate<256, NF, LOCAL>, 256, 0);
    case 512: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, k_batch_iterate<512, NF, LOCAL>, 512, 0);
    case 1024: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, k_batch_iterate<1024, NF, LOCAL>, 1024, 0);
  }
  return cudaErrorInvalidValue;
}

cudaError_t occupancy_batch(uint32_t cta, bool near_far, bool local, int* nb) {
  if (local) return near_far ? occ_b<true, true>(cta, nb) : occ_b<false, true>(cta, nb);
  return near_far ? occ_b<true, false>(cta, nb) : occ_b<false, false>(cta, nb);
}

cudaError_t launch_extract_values(const unsigned long long* ds, uint32_t* out, uint64_t n, uint32_t grid,
                                  cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_extract_values<<<grid, 256, 0, s>>>(ds, out, n);
  return cudaGetLastError();
}

cudaError_t launch_admit(const AdmitParams& a, uint32_t grid, cudaStream_t s) {
  if (a.nnew == 0) return cudaSuccess;
  k_batch_fill<<<grid, 256, 0, s>>>(a);
  k_batch_sources<<<grid, 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace irgl
