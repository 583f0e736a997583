// nb_verlet.cuh -- per-ion pieces of the velocity-Verlet step (Sec. II) shared
// by every kernel that advances ions: the Langevin normals (Philox4x32-10 and
// Box-Muller), the Coulomb prefactor, the drift and the kick.  The
// multi-kernel step (nb_integrate.cu), the single-block step (nb_small.cu)
// and the ensemble kernel (nb_batched.cu) all inline these same functions, so
// an ion given the same inputs gets the same bits on every path.
#pragma once

#include <cmath>

#include "nb_common.cuh"

namespace nb {

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) from its definition:
// ten rounds of two 32x32 -> 64-bit products with the multipliers
// 0xD2511F53 and 0xCD9E8D57, key bumped by 0x9E3779B9 / 0xBB67AE85.
__device__ __forceinline__ void philox(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c[0]), lo0 = 0xD2511F53u * c[0];
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c[2]), lo1 = 0xCD9E8D57u * c[2];
    const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}

// Three N(0,1) draws for (seed, instance, step, ion): Box-Muller on the four
// Philox words mapped to (0,1) as (k + 1/2) 2^-32.
__device__ __forceinline__ void normals3(unsigned long long seed, unsigned instance,
                                         int64_t step, int64_t ion, double out[3]) {
  uint32_t c[4] = {(uint32_t)ion, (uint32_t)((uint64_t)step & 0xffffffffu),
                   (uint32_t)((uint64_t)step >> 32), instance};
  philox(c, (uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32));
  const double s = 2.3283064365386963e-10;
  const double u0 = ((double)c[0] + 0.5) * s, u1 = ((double)c[1] + 0.5) * s;
  const double u2 = ((double)c[2] + 0.5) * s, u3 = ((double)c[3] + 0.5) * s;
  const double m0 = sqrt(-2.0 * log(u0)), m1 = sqrt(-2.0 * log(u2));
  double s1, c1, s3, c3;
  sincospi(2.0 * u1, &s1, &c1);
  sincospi(2.0 * u3, &s3, &c3);
  out[0] = m0 * c1;
  out[1] = m0 * s1;
  out[2] = m1 * c3;
}

// Coulomb prefactor k_C q_i w / m_i, where the pair sums carry w_j = q_j when
// per-ion charges are given and w_j = 1 otherwise.
__device__ __forceinline__ double coulomb_pref(const Phys &p, const StateView &s, int64_t i) {
  const double m = ion_mass(p, s, i);
  return s.q ? p.k_coulomb * s.q[i] / m : p.k_coulomb * p.charge * p.charge / m;
}

// Sum of the n_jc chunk partials of one component of an ion, as eight interleaved
// running sums (chunk jc goes to sum jc mod 8, from zero) added pairwise at the
// end.  The dependent chain is n_jc/8 + 3 FP64 adds instead of n_jc: at small n
// the latency of that chain, not the bandwidth, bounds the epilogue.  ld(jc)
// returns chunk jc; the loads of eight chunks are issued before their adds.
// FP64 adds of zeros are left out (64 cycles of an SMSP each): 0 + v is v with -0
// made +0, and adding a running sum that no slot went to changes nothing, since
// none is ever -0.
__device__ __forceinline__ double no_neg_zero(double v) {
  return __double2hiint(v) == (int)0x80000000 && __double2loint(v) == 0 ? 0.0 : v;
}
template <class LD>
__device__ __forceinline__ double slot_sum1(int n_jc, LD ld) {
  double s[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const double v = u < n_jc ? ld(u) : 0.0;
    s[u] = no_neg_zero(v);
  }
  for (int jc = 8; jc < n_jc; jc += 8)
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (jc + u < n_jc) s[u] += ld(jc + u);
#pragma unroll
  for (int w = 1; w < 8; w <<= 1)
#pragma unroll
    for (int u = 0; u < 8; u += 2 * w)
      if (u + w < n_jc) s[u] += s[u + w];
  return s[0];
}

// Drift of one coordinate: r + v dt + a dt^2/2.
__device__ __forceinline__ double verlet_drift(double r, double v, double a, double dt) {
  return r + v * dt + 0.5 * dt * dt * a;
}

// The kick's per-ion constants, which depend only on the ion and the
// parameters: the Coulomb prefactor, the trap scale of its species, the
// friction factors 1 / (1 + gamma dt/(2 m_i)) and gamma/m_i, and the Langevin
// amplitude.  Several are FP64 divisions, long dependent chains on GB300, so a
// kernel that kicks the same ion many times forms them once; the values are
// the same wherever they are formed.
struct KickConst {
  double pref, ts, inv, g, sig;
};
__device__ __forceinline__ double kick_inv(const Phys &p, double mi) {
  return 1.0 / (1.0 + p.gamma * p.dt / (2.0 * mi));
}
__device__ __forceinline__ double kick_sig(const Phys &p, double mi) {
  return p.noise_T > 0.0 ? sqrt(2.0 * p.gamma * KB * p.noise_T * p.dt) / mi : 0.0;
}
__device__ __forceinline__ KickConst kick_consts(const Phys &p, const StateView &s, int64_t i) {
  const double mi = ion_mass(p, s, i);
  return KickConst{coulomb_pref(p, s, i), trap_scale(p, s, i), kick_inv(p, mi), p.gamma / mi, kick_sig(p, mi)};
}

// The same for all ions where they have the reference charge and mass, formed on
// the host: every operation is correctly rounded and none is an a b + c to fuse,
// so the bits are kick_consts'.
inline KickConst uniform_kick_consts(const Phys &p) {
  KickConst k;
  k.pref = p.k_coulomb * p.charge * p.charge / p.mass;
  k.ts = 1.0;
  k.inv = 1.0 / (1.0 + p.gamma * p.dt / (2.0 * p.mass));
  k.g = p.gamma / p.mass;
  k.sig = p.noise_T > 0.0 ? std::sqrt(2.0 * p.gamma * KB * p.noise_T * p.dt) / p.mass : 0.0;
  return k;
}

// The trap acceleration (Eq. 1) is linear in the position: a_k = f_k(t) r_k for
// the reference species, with the products of trap_accel.  The factors depend on
// the time alone; the RF trap's take an FP64 cosine, a long dependent chain, so a
// kernel forms them beside the pair sums, not after them.
struct TrapFactors {
  double f[3];
};
__device__ __forceinline__ TrapFactors trap_factors(const Phys &p, int64_t snew) {
  TrapFactors tf;
  const double t = p.t0 + (double)snew * p.dt;
  trap_accel(p, t, 1.0, 1.0, 1.0, tf.f[0], tf.f[1], tf.f[2]);
  return tf;
}
// Component c of them: a branch that a warp of one component takes as one.
__device__ __forceinline__ double trap_factor1(const Phys &p, int64_t snew, int c) {
  const TrapFactors tf = trap_factors(p, snew);
  return c == 0 ? tf.f[0] : c == 1 ? tf.f[1] : tf.f[2];
}

// The Langevin draws of ion i at step snew (zeros without noise).
__device__ __forceinline__ void kick_noise(const Phys &p, int64_t i, int64_t snew, double xi[3]) {
  xi[0] = xi[1] = xi[2] = 0.0;
  if (p.noise_T > 0.0) normals3(p.seed, p.instance, snew, i, xi);
}

// Kick of an ion at positions r (step index snew, time t0 + snew dt), given
// its pair sum cs = sum_j w_j (r_i - r_j) / s_ij^3, its constants kc, the trap's
// factors at that time and its draws xi:
//   a+_cons = k_C q_i/m_i cs + trap(r, t)   (Eq. 1)
//   v+ = (v + (a + a+_cons) dt/2) * [1 / (1 + gamma dt/(2 m_i))]  [+ Langevin kick]
//   a+ = a+_cons - (gamma/m_i) v+
// v and a hold the ion's velocity and acceleration on entry and the new ones
// on return, of one component.  Returns true if either is not finite.
__device__ __forceinline__ bool verlet_kick1(double dt, const KickConst &kc, double tf, double xi, double r, double cs,
                                             double &v, double &a) {
  const double tr = __dmul_rn(__dmul_rn(tf, r), kc.ts);
  const double ucons = __fma_rn(kc.pref, cs, tr);
  double vn = __fma_rn(0.5 * dt, a + ucons, v) * kc.inv;
  vn = __fma_rn(kc.sig, xi, vn);
  const double an = __fma_rn(-kc.g, vn, ucons);
  v = vn;
  a = an;
  return not_finite(vn) || not_finite(an);
}
}  // namespace nb
