// nb_epi.cuh -- shared parts of the per-ion kernels that follow a pair kernel
// (nb_integrate.cu, nb_adjoint.cu): the eight-thread sum of an ion's partial
// slots, the FP32 parts of a position, and the step's launches.
#pragma once

#include "nb_pdl.cuh"
#include "nb_verlet.cuh"

namespace nb {

// Eight threads per ion: warp u < 8 of a block forms slot_sum1's running sum u
// (slots u, u + 8, ...) for the block's 32 ions, one ion per lane (each load of a
// warp reads 256 contiguous bytes), and leaves it in shared memory; after a
// barrier finishing warps take the totals: one warp for all three components, or
// warps 8, 9 and 10 for one each.
//
// These kernels are latency chains (a few microseconds at any n up to 1e4), and
// what makes the chain long is FP64: an SMSP issues one FP64 warp instruction per
// 64 cycles.  So the finishing work of a step goes to three warps, which sit on
// different SMSPs, and what does not depend on the sums is done before the
// barrier.  100 steps at n = 1024 (fp64) and n = 3001 (split): 2.39 and 2.03 ms
// with eight lanes of one warp per ion, shuffles and the tail after them (and the
// split of the positions as a launch of its own), 2.31 and 1.76 with one
// finishing warp; with three, 1.37 -> 1.09 (on nb_one.cu's pair kernel) and 1.76 ->
// 1.48 ms.
constexpr int EPI8_IONS = 32, EPI8_THREADS = 288, EPI8_THREADS_COMP = 352;

__device__ __forceinline__ double (*epi8_shared())[8][32] {
  __shared__ double csum[3][8][32];
  return csum;
}

// The running sums of this thread's warp; returns the finishing warps' number
// (0, 1, 2), which have none, and -1 for the others.  The caller's
// __syncthreads() follows.
__device__ __forceinline__ int epi8_slots(const double *__restrict__ part, int n_jc, int64_t n) {
  const int u = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (u >= 8) return u - 8;
  double(*csum)[8][32] = epi8_shared();
  const int64_t g = (int64_t)blockIdx.x * EPI8_IONS + l;
  double cs[3] = {0.0, 0.0, 0.0};
  const double *pi = part + (g < n ? g : n - 1);
  if (u < n_jc) {
    const double *q = pi + (int64_t)u * 3 * n;
    cs[0] = no_neg_zero(__ldcs(q));
    cs[1] = no_neg_zero(__ldcs(q + n));
    cs[2] = no_neg_zero(__ldcs(q + 2 * n));
  }
#pragma unroll 4
  for (int jc = u + 8; jc < n_jc; jc += 8) {
    const double *q = pi + (int64_t)jc * 3 * n;
    cs[0] += __ldcs(q);
    cs[1] += __ldcs(q + n);
    cs[2] += __ldcs(q + 2 * n);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) csum[c][u][l] = cs[c];
  return -1;
}

// slot_sum1's pairing of the eight running sums of component c of the lane's ion.
__device__ __forceinline__ double epi8_total(int c) {
  const int l = threadIdx.x & 31;
  const double(*s)[32] = epi8_shared()[c];
  return ((s[0][l] + s[1][l]) + (s[2][l] + s[3][l])) + ((s[4][l] + s[5][l]) + (s[6][l] + s[7][l]));
}

// The FP32 (hi, lo) parts of component c of ion i's position, as
// k_split_positions (nb_pair.cu) stores them.
__device__ __forceinline__ void store_split(float *out6, int64_t n, int64_t i, int c, double r) {
  const float h = __double2float_rn(r);
  out6[c * n + i] = h;
  out6[(3 + c) * n + i] = __double2float_rn(r - (double)h);
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
