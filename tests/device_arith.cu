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

// per element: 1/a, sqrt(a) and its reciprocal, 1/a and 1/b by one reciprocal, a / b
__global__ void fp64_kernel(int n, const double *a, const double *b, double *out) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    double r, ir, ia, ib;
    root64(a[i], r, ir);
    rcp_pair(a[i], b[i], ia, ib);
    out[i] = rcp64(a[i]);
    out[n + i] = r;
    out[2 * n + i] = ir;
    out[3 * n + i] = ia;
    out[4 * n + i] = ib;
    out[5 * n + i] = quot64(a[i], b[i], 1.0 / b[i]);
  }
}

extern "C" int probe_fp64(int n, const double *a, const double *b, double *out) {
  fp64_kernel<<<1, 256>>>(n, a, b, out);
  return (int)cudaDeviceSynchronize();
}
