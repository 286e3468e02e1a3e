// Mixed form of the xi-march: FP32 ring and node arithmetic, float-float scans.
#include "march_tiles.cuh"
#include "pipeline.cuh"

namespace wake {

bool march_tile_mixed512(int nt, int ppt, TileFns *out, bool slab) {
  if (nt != 512) return false;
  if (slab) {
    switch (ppt) {
      case 1: *out = tile_fns<SlabOf<PolMixed>, 512, 1>(); return true;
      case 2: *out = tile_fns<SlabOf<PolMixed>, 512, 2>(); return true;
      case 4: *out = tile_fns<SlabOf<PolMixed>, 512, 4>(); return true;
      case 8: *out = tile_fns<SlabOf<PolMixed>, 512, 8>(); return true;
      default: return false;
    }
  }
  switch (ppt) {
    case 1: *out = tile_fns<PolMixed, 512, 1>(); return true;
    case 2: *out = tile_fns<PolMixed, 512, 2>(); return true;
    case 4: *out = tile_fns<PolMixed, 512, 4>(); return true;
    case 8: *out = tile_fns<PolMixed, 512, 8>(); return true;
    case 16: *out = tile_fns<PolMixed, 512, 16>(); return true;
    default: return false;
  }
}

using StepMixed = StepOf<PolMixed>;

template <class P, int PPT, bool kCorn = false>
static cudaError_t go_step(const PipeArgs &a, int ctas, cudaStream_t stream) {
  auto kern = step_kernel<P, StepMixed::NT, PPT, kCorn>;
  const size_t smem = step_smem_bytes<StepMixed, StepMixed::NT, PPT>(a.d.nr + 1);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  PipeArgs arg = a;
  void *args[] = {&arg};
  return cudaLaunchCooperativeKernel((const void *)kern, dim3(ctas), dim3(StepMixed::NT), args, smem, stream);
}
template <int PPT, bool kCorn = false>
static int ctas_step(int n1) {
  auto kern = step_kernel<StepMixed, StepMixed::NT, PPT, kCorn>;
  const size_t smem = step_smem_bytes<StepMixed, StepMixed::NT, PPT>(n1);
  if (smem > 227 * 1024) return 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
  int per_sm = 0, dev = 0, sms = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, StepMixed::NT, smem) != cudaSuccess) return 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return per_sm * sms;
}
static int ppt_for(int np) {
  const int ppt = (np + StepMixed::NT - 1) / StepMixed::NT;
  return ppt <= 1 ? 1 : ppt <= 2 ? 2 : ppt <= 4 ? 4 : ppt <= 8 ? 8 : ppt <= 16 ? 16 : 0;
}
static size_t step_bytes_for(int n1, int np) {
  switch (ppt_for(np)) {
    case 1: return step_smem_bytes<StepMixed, StepMixed::NT, 1>(n1);
    case 2: return step_smem_bytes<StepMixed, StepMixed::NT, 2>(n1);
    case 4: return step_smem_bytes<StepMixed, StepMixed::NT, 4>(n1);
    case 8: return step_smem_bytes<StepMixed, StepMixed::NT, 8>(n1);
    case 16: return step_smem_bytes<StepMixed, StepMixed::NT, 16>(n1);
    default: return (size_t)1 << 40;
  }
}
cudaError_t launch_step_mixed(const PipeArgs &a, int np, int ctas, cudaStream_t stream) {
  if (a.d.slab) {  // the slab geometry's kernels (up to 8 rings per thread)
    switch (ppt_for(np)) {
      case 1: return go_step<SlabOf<StepMixed>, 1>(a, ctas, stream);
      case 2: return go_step<SlabOf<StepMixed>, 2>(a, ctas, stream);
      case 4: return go_step<SlabOf<StepMixed>, 4>(a, ctas, stream);
      case 8: return go_step<SlabOf<StepMixed>, 8>(a, ctas, stream);
      default: return cudaErrorInvalidValue;
    }
  }
  if (a.corners) {
    switch (ppt_for(np)) {
      case 1: return go_step<StepMixed, 1, true>(a, ctas, stream);
      case 2: return go_step<StepMixed, 2, true>(a, ctas, stream);
      case 4: return go_step<StepMixed, 4, true>(a, ctas, stream);
      case 8: return go_step<StepMixed, 8, true>(a, ctas, stream);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (ppt_for(np)) {
    case 1: return go_step<StepMixed, 1>(a, ctas, stream);
    case 2: return go_step<StepMixed, 2>(a, ctas, stream);
    case 4: return go_step<StepMixed, 4>(a, ctas, stream);
    case 8: return go_step<StepMixed, 8>(a, ctas, stream);
    case 16: return go_step<StepMixed, 16>(a, ctas, stream);
    default: return cudaErrorInvalidValue;
  }
}
int step_ctas_mixed(int n1, int np) {
  if (step_bytes_for(n1, np) > 227 * 1024) return 0;
  switch (ppt_for(np)) {
    case 1: return ctas_step<1>(n1);
    case 2: return ctas_step<2>(n1);
    case 4: return ctas_step<4>(n1);
    case 8: return ctas_step<8>(n1);
    case 16: return ctas_step<16>(n1);
    default: return 0;
  }
}

// The same for the steps with density grids by cells (0: no such kernel).
int step_max_ctas_corners(int n1, int np) {
  if (step_bytes_for(n1, np) > 227 * 1024) return 0;
  switch (ppt_for(np)) {
    case 1: return ctas_step<1, true>(n1);
    case 2: return ctas_step<2, true>(n1);
    case 4: return ctas_step<4, true>(n1);
    case 8: return ctas_step<8, true>(n1);
    default: return 0;
  }
}

}  // namespace wake
