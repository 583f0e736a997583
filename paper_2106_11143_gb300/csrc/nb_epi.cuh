// nb_epi.cuh -- shared parts of the per-ion kernels that follow a pair kernel
// (nb_integrate.cu, nb_adjoint.cu): the eight-thread sum of an ion's partial
// slots, the FP32 parts of a position, and the step's launches.
#pragma once

#include "nb_verlet.cuh"

namespace nb {

// Eight threads per ion: warp u < 8 of a block of nine forms slot_sum3's running
// sum u (slots u, u + 8, ...) for the block's 32 ions, one ion per lane (each
// load of a warp reads 256 contiguous bytes), and leaves it in shared memory;
// the ninth warp takes the total after a barrier.  The dependent chain of the
// sum is spread over eight threads, and the FP64 tail serves 32 ions per warp
// instruction.  The kernels are latency chains (a few microseconds at any n up
// to 1e4): with eight lanes of one warp per ion, shuffles and the tail after
// them, a step took 23.9 us at n = 1024 (fp64) and, with the position split as
// a launch of its own, 20.3 us at n = 3001 (split); with the ninth warp and the
// fused split 23.1 and 17.6 us.
constexpr int EPI8_IONS = 32, EPI8_THREADS = 288;

__device__ __forceinline__ double (*epi8_shared())[8][32] {
  __shared__ double csum[3][8][32];
  return csum;
}

// The running sums of this thread's warp; true for the ninth warp (which has
// none).  The caller's __syncthreads() follows.
__device__ __forceinline__ bool epi8_slots(const double *__restrict__ part, int n_jc, int64_t n) {
  const int u = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (u == 8) return true;
  double(*csum)[8][32] = epi8_shared();
  const int64_t g = (int64_t)blockIdx.x * EPI8_IONS + l;
  double cs[3] = {0.0, 0.0, 0.0};
  const double *pi = part + (g < n ? g : n - 1);
  for (int jc = u; jc < n_jc; jc += 8) {
    const double *q = pi + (int64_t)jc * 3 * n;
    cs[0] += __ldcs(q);
    cs[1] += __ldcs(q + n);
    cs[2] += __ldcs(q + 2 * n);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) csum[c][u][l] = cs[c];
  return false;
}

// slot_sum3's pairing of the eight running sums, for the ninth warp's ion.
__device__ __forceinline__ void epi8_total(double cs[3]) {
  const int l = threadIdx.x & 31;
  double(*csum)[8][32] = epi8_shared();
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double(*s)[32] = csum[c];
    cs[c] = ((s[0][l] + s[1][l]) + (s[2][l] + s[3][l])) + ((s[4][l] + s[5][l]) + (s[6][l] + s[7][l]));
  }
}

// The FP32 (hi, lo) parts of a position as k_split_positions (nb_pair.cu) stores
// them.
__device__ __forceinline__ void store_split(float *out6, int64_t n, int64_t i, const double r[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float h = __double2float_rn(r[c]);
    out6[c * n + i] = h;
    out6[(3 + c) * n + i] = __double2float_rn(r[c] - (double)h);
  }
}

// launch_drift and launch_epi_step with the FP32 parts of the positions they
// write stored to `split` (nullptr: not).
cudaError_t launch_drift_split(const Phys &p, const StateView &s, double *px, double *py, double *pz, float *split,
                               cudaStream_t st);
cudaError_t launch_epi_step_split(const Phys &p, const StateView &s, const double *cx, const double *cy,
                                  const double *cz, const double *part, int n_jc, int64_t snew,
                                  double *nx, double *ny, double *nz, float *split, unsigned *err, cudaStream_t st,
                                  const int64_t *cin = nullptr, int64_t *cout = nullptr, int64_t cout_off = 0);

}  // namespace nb
