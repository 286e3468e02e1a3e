// Probes of the device arithmetic the marches are built from, for test_gpu_arith.py.
#include "../paper_1411_3246_gb300/csrc/march.cuh"

using namespace wake;

// one warp: lane l's pair (h[l], l[l]) summed over the lanes as the block scans do; the inclusive sums out
__global__ void ff_scan_kernel(const float *h, const float *l, float *oh, float *ol) {
  const int lane = threadIdx.x;
  FF v{h[lane], l[lane]};
  for (int o = 1; o < 32; o <<= 1) {
    const FF t = wide_shfl_up(v, o);
    if (lane >= o) v = wide_add(v, t);
  }
  oh[lane] = v.h;
  ol[lane] = v.l;
}

extern "C" int probe_ff_scan(const float *h, const float *l, float *oh, float *ol) {
  ff_scan_kernel<<<1, 32>>>(h, l, oh, ol);
  return (int)cudaDeviceSynchronize();
}
