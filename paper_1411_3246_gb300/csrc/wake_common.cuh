// Device-side helpers shared by the march and beam kernels of libwake.
//
// Grid conventions (Sec. II.A; readings stated in the library header): node-centred radial
// nodes r_i = i dr, i = 0..nr; xi nodes xi_k = k dxi, k = 0..nxi; linear hats in r with
// ring volumes V_0 = dr^2/6, V_i = r_i dr, V_nr = dr (r_nr/2 - dr/6) (per 2 pi).  Slab
// geometry (x, xi), x >= 0 with a mirror plane at x = 0: hat widths V_i = dx, halved at x = 0
// and at the wall (per unit area).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace wake {

// Sticky per-simulation status bits (device word), mapped to WAKE_E* codes on the host.
enum : int { ST_NUMERIC = 1, ST_ESCAPE = 2, ST_TIMEOUT = 4 };

constexpr unsigned kFull = 0xffffffffu;

// Shared memory of one CTA at most (sm_103a).
constexpr size_t kMaxSmemPerCta = 227 * 1024;

// Everything one CTA needs about one simulation.  Grids are (nxi+1) x (nr+1), slice-major;
// their element type is double (FP64) or float (mixed) as the kernel's policy says.
struct SimDesc {
  int nr, nxi, np, has_beam;
  double rmax, ximax, dr, dxi;
  const double *r0, *ur0, *lz, *G0, *w;  // ring constants (set by wake_load_plasma)
  void *ring_buf;                        // ring slot arrays in global memory (FP64 form)
  const void *nb;                        // beam density n_b on the nodes
  void *psi, *ez, *er, *bth;             // march output
  int *status;
  // trapping (march_trap_kernel): threshold, promotion list of trap_cap entries of 7 doubles
  double gamma_t;
  double *trap;
  int *trap_count;
  int trap_cap;
  int slab;  // slab geometry: r is x, lz holds the conserved u_y
};

// Cell index c in [0, nr-1] and offset f = r/dr - c (f in [0,1] for 0 <= r <= rmax).
// Clamped, so a non-finite r never indexes out of bounds.
template <class R>
__device__ __forceinline__ void locate(R r, R inv_dr, int nr, int &c, R &f) {
  R s = r * inv_dr;
  R fl = floor(s);
  int i = (int)fl;
  i = i < 0 ? 0 : (i > nr - 1 ? nr - 1 : i);
  c = i;
  f = s - (R)i;
}

template <class T, class R>
__device__ __forceinline__ R interp(const T *v, int c, R f) {
  return ((R)1 - f) * (R)v[c] + f * (R)v[c + 1];
}

__host__ __device__ __forceinline__ double node_volume(int i, int nr, double dr, bool slab = false) {
  if (slab) return (i == 0 || i == nr) ? 0.5 * dr : dr;
  return i == 0 ? dr * dr / 6.0 : (i == nr ? dr * ((double)nr * dr / 2.0 - dr / 6.0) : (double)i * dr * dr);
}

// Fraction of hat m's ring volume that lies inside r_m (1/2 - 1/(6m); 1 at the wall; slab 1/2).
__host__ __device__ __forceinline__ double node_alpha(int m, int nr, bool slab = false) {
  return m == nr ? 1.0 : (slab ? 0.5 : 0.5 - 1.0 / (6.0 * (double)m));
}

// Eq. 12: the two-bunch driver density.
__host__ __device__ __forceinline__ double nb_eq12(double r, double xi, double n_d, double n_w,
                                                   double sr, double szd, double szw, double xd,
                                                   double xw) {
  const double ad = (xi - xd) / szd;
  double lon = n_d * exp(-0.5 * ad * ad);
  if (n_w != 0.0) {
    const double aw = (xi - xw) / szw;
    lon += n_w * exp(-0.5 * aw * aw);
  }
  return exp(-r * r / (2.0 * sr * sr)) * lon;
}

__device__ __forceinline__ void flag(int *status, int bit) { atomicOr(status, bit); }

}  // namespace wake
