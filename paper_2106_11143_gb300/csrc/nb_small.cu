// nb_small.cu -- velocity-Verlet steps (Sec. II) of a small system in one
// thread block: one launch runs many steps, with the positions in shared
// memory and each ion's velocity and acceleration in its own thread's
// registers.
//
// At small n a step of the multi-kernel path (pair kernel, epilogue) costs a
// few microseconds of launch and kernel latency whatever the work, so the
// step rate stops improving as n shrinks.  Here a step costs two block
// barriers on top of its arithmetic, but all of that arithmetic runs on one
// SM, so the path pays off only while one SM's share of the n^2 pair terms
// is shorter than that latency (the host picks it by n and precision).
//
// The block computes the same work items as the one-sided force kernel's
// plan: ion i against the partners of j-chunk jc, in tiles of the plan's
// block size, with the same pair term and the same per-tile flushes
// (nb_pairterm.cuh).  It keeps the chunk partials in shared memory and adds
// them in the epilogue's order (slot_sum1).  It then applies the same kick
// and drift (nb_verlet.cuh).  Each ion's result is therefore bitwise that of
// the multi-kernel path.
#include <mutex>

#include "nb_pairterm.cuh"
#include "nb_verlet.cuh"

namespace nb {

// Partial sum of ion i over the partners [jb, je), in tiles of `tile`
// partners: the arithmetic of one (i, j-chunk) item of k_pair_force.
template <int MODE, bool QARR>
__device__ __forceinline__ void chunk_partial(const D4 *pos, const float4 *sp, int i, int jb, int je,
                                              int tile, double soft2, float soft2f, float s2h,
                                              float s2l, double out[3]) {
  double ad[3] = {0.0, 0.0, 0.0}, cd[3] = {0.0, 0.0, 0.0};
  float af[3] = {0.0f, 0.0f, 0.0f};
  double xi = 0.0, yi = 0.0, zi = 0.0;
  float xh = 0.0f, yh = 0.0f, zh = 0.0f, xl = 0.0f, yl = 0.0f, zl = 0.0f;
  if (split_like(MODE)) {
    const float4 h = sp[2 * i], l = sp[2 * i + 1];
    xh = h.x; yh = h.y; zh = h.z;
    xl = l.x; yl = l.y; zl = l.z;
  } else {
    const D4 e = pos[i];
    xi = e.x; yi = e.y; zi = e.z;
  }
  for (int j0 = jb; j0 < je; j0 += tile) {
    const int cnt = min(tile, je - j0);
    if (MODE == MODE_FP64) {
#pragma unroll 4
      for (int k = 0; k < cnt; ++k) pair_f64<QARR>(xi, yi, zi, pos[j0 + k], soft2, ad[0], ad[1], ad[2]);
    } else if (ladder_mode(MODE)) {
#pragma unroll 4
      for (int k = 0; k < cnt; ++k)
        pair_ladder<MODE, QARR>(xi, yi, zi, pos[j0 + k], soft2, ad[0], ad[1], ad[2]);
    } else if (MODE == MODE_DF64) {
      float al[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll 4
      for (int k = 0; k < cnt; ++k) pair_df64<QARR>(xi, yi, zi, pos[j0 + k], s2h, s2l, af, al);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        ad[c] += f32_to_f64(af[c]) + f32_to_f64(al[c]);
        af[c] = 0.0f;
      }
    } else if (MODE == MODE_MIXED) {
#pragma unroll 4
      for (int k = 0; k < cnt; ++k) {
        const D4 pj = pos[j0 + k];
        const float qf = QARR ? (float)pj.w : 0.0f;
        const float fx = f64_to_f32_rn(xi - pj.x);
        const float fy = f64_to_f32_rn(yi - pj.y);
        const float fz = f64_to_f32_rn(zi - pj.z);
        pair_f32_bulk<QARR>(fx, fy, fz, qf, soft2f, af[0], af[1], af[2]);
      }
    } else {
#pragma unroll 4
      for (int k = 0; k < cnt; ++k) {
        const float4 ph = sp[2 * (j0 + k)];
        const float4 pl = sp[2 * (j0 + k) + 1];
        const float fx = (xh - ph.x) + (xl - pl.x);
        const float fy = (yh - ph.y) + (yl - pl.y);
        const float fz = (zh - ph.z) + (zl - pl.z);
        pair_f32_bulk<QARR, MODE == MODE_SPLIT_RSQ>(fx, fy, fz, ph.w, soft2f, af[0], af[1], af[2]);
      }
    }
    if (MODE == MODE_MIXED || split_like(MODE)) {
#pragma unroll
      for (int c = 0; c < 3; ++c) flush_tile(af[c], ad[c], cd[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) out[c] = (fp64_like(MODE) || MODE == MODE_DF64) ? ad[c] : ad[c] + cd[c];
}

// Stages ion i in the form the pair terms read: the FP64 position and weight (w =
// q_i, or its FP32 (hi, lo) pair for the double-float term), and for the split
// mode the FP32 (hi, lo) parts of the position as k_split_positions forms them,
// with the FP32 charge beside the high part.  stage_weight writes the weights,
// once; stage_comp component c at position r.
template <int MODE, bool QARR>
__device__ __forceinline__ void stage_weight(D4 *pos, float4 *sp, const StateView &s, int i) {
  pos[i].w = (QARR && MODE != MODE_DF64) ? s.q[i] : 0.0;
  if (MODE == MODE_DF64 && QARR) {
    float qh, ql;
    split_f64(s.q[i], qh, ql);
    *reinterpret_cast<float2 *>(&pos[i].w) = make_float2(qh, ql);
  }
  if (split_like(MODE)) {
    sp[2 * i].w = QARR ? (float)s.q[i] : 0.0f;
    sp[2 * i + 1].w = 0.0f;
  }
}
template <int MODE>
__device__ __forceinline__ void stage_comp(D4 *pos, float4 *sp, int i, int c, double r) {
  reinterpret_cast<double *>(pos + i)[c] = r;
  if (split_like(MODE)) {
    const float h = __double2float_rn(r);
    reinterpret_cast<float *>(sp + 2 * i)[c] = h;
    reinterpret_cast<float *>(sp + 2 * i + 1)[c] = __double2float_rn(r - (double)h);
  }
}

// One warp beyond the SMALL_THREADS of the pair items holds the trap's factors.
constexpr int SMALL_BLOCK = SMALL_THREADS + 32;
// Up to this many ions each component of an ion has a thread of its own.
constexpr int SMALL_COMP_N = SMALL_THREADS / 3 / 32 * 32;

// nsteps steps from (x, v, a) at step index step0.  Per step: [barrier] pair
// items -> chunk partials [barrier] kick and next drift.  Writes x, v, a back at
// the end.
//
// An SMSP issues one FP64 warp instruction per 64 cycles, whatever the number of
// active lanes, so up to SMALL_COMP_N ions the kick is laid out by component:
// thread (c, i) adds ion i's slots of component c, kicks and drifts it, and the
// three components run on warps of different SMSPs.  With all three on one warp
// the slot sums, kick and drift took 8900 of a step's 11000 cycles at n = 16, and
// 100 steps in the RF trap 592 us against 266 now.  Above, a thread has an ion (NC
// = 3): all SMSPs are busy either way.  The trap's factors of 32 steps are formed
// at a time, one step per lane of the last warp; the Langevin draws before the
// barrier, beside the pair items.
template <int MODE, bool QARR, int NC>
__global__ void __launch_bounds__(SMALL_BLOCK, 1)
    k_small_steps(Phys p, StateView s, int tile, int jchunk, int n_jc, int64_t step0, int64_t nsteps,
                  unsigned *err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = (int)s.n;
  const int tid = threadIdx.x;
  D4 *pos = reinterpret_cast<D4 *>(smem_raw);
  float4 *sp = reinterpret_cast<float4 *>(pos + n);
  double *part = reinterpret_cast<double *>(sp + (split_like(MODE) ? 2 * n : 0));
  TrapFactors *tf = reinterpret_cast<TrapFactors *>(part + 3 * n * n_jc);
  const int np = (n + 31) & ~31;
  const int c0 = NC == 1 ? tid / np : 0;  // the thread's first component
  const int ion = NC == 1 ? tid - c0 * np : tid;
  const bool own = ion < n && c0 < 3;
  const double dt = p.dt;
  const float soft2f = (float)p.soft2;
  float s2h = 0.0f, s2l = 0.0f;
  if (MODE == MODE_DF64) split_f64(p.soft2, s2h, s2l);

  double *const xs[3] = {s.x, s.y, s.z}, *const vs[3] = {s.vx, s.vy, s.vz}, *const as[3] = {s.ax, s.ay, s.az};
  double r[NC], v[NC], a[NC], xi[NC];
  const KickConst kc = kick_consts(p, s, own ? ion : 0);  // once for all the launch's steps
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    r[k] = v[k] = a[k] = xi[k] = 0.0;
    if (!own) continue;
    const int c = c0 + k;
    v[k] = (c == 0 ? vs[0] : c == 1 ? vs[1] : vs[2])[ion];
    a[k] = (c == 0 ? as[0] : c == 1 ? as[1] : as[2])[ion];
    r[k] = verlet_drift((c == 0 ? xs[0] : c == 1 ? xs[1] : xs[2])[ion], v[k], a[k], dt);
    stage_comp<MODE>(pos, sp, ion, c, r[k]);
    if (c == 0) stage_weight<MODE, QARR>(pos, sp, s, ion);
  }
  TrapFactors f = {};
  bool bad = false;
  const int items = n * n_jc;
  for (int64_t st = 0; st < nsteps; ++st) {
    __syncthreads();  // this step's positions are staged; last step's partials are read
    if (tid >= SMALL_THREADS) {
      const int lane = tid & 31, at = (int)(st & 31);
      if (at == 0) f = trap_factors(p, step0 + st + 1 + lane);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double fc = __shfl_sync(0xffffffffu, f.f[c], at);
        if (lane == 0) tf->f[c] = fc;
      }
    } else {
      for (int it = tid; it < items; it += SMALL_THREADS) {
        const int jc = it / n;
        const int i = it - jc * n;
        const int jb = jc * jchunk;
        double o[3];
        chunk_partial<MODE, QARR>(pos, sp, i, jb, min(jb + jchunk, n), tile, p.soft2, soft2f, s2h, s2l, o);
#pragma unroll
        for (int c = 0; c < 3; ++c) part[(jc * 3 + c) * n + i] = o[c];
      }
      if (p.noise_T > 0.0 && own) {
        double all[3];
        kick_noise(p, ion, step0 + st + 1, all);
#pragma unroll
        for (int k = 0; k < NC; ++k) xi[k] = NC == 3 ? all[k] : (c0 == 0 ? all[0] : c0 == 1 ? all[1] : all[2]);
      }
    }
    __syncthreads();  // partials complete; nobody reads the positions until the next barrier
    if (own) {
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const int c = c0 + k;
        const double cs = slot_sum1(n_jc, [&](int jc) { return part[(jc * 3 + c) * n + ion]; });
        bad |= verlet_kick1(dt, kc, tf->f[c], xi[k], r[k], cs, v[k], a[k]);
        if (st + 1 < nsteps) {
          r[k] = verlet_drift(r[k], v[k], a[k], dt);
          stage_comp<MODE>(pos, sp, ion, c, r[k]);
        }
      }
    }
  }
  if (own)
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const int c = c0 + k;
      (c == 0 ? xs[0] : c == 1 ? xs[1] : xs[2])[ion] = r[k];
      (c == 0 ? vs[0] : c == 1 ? vs[1] : vs[2])[ion] = v[k];
      (c == 0 ? as[0] : c == 1 ? as[1] : as[2])[ion] = a[k];
    }
  if (bad) atomicOr(err, ERR_NONFINITE);
}

size_t small_smem_bytes(const Plan &pl, int mode, int64_t n) {
  return (size_t)n * sizeof(D4) + (split_like(mode) ? (size_t)n * 2 * sizeof(float4) : 0) +
         (size_t)pl.n_jc * 3 * (size_t)n * sizeof(double) + sizeof(TrapFactors);
}

template <int MODE>
static cudaError_t launch_small_m(const Plan &pl, const Phys &p, const StateView &s, int64_t step0,
                                  int64_t nsteps, unsigned *err, cudaStream_t st) {
  static std::mutex mu;
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!done[dev]) {
      const void *const ks[4] = {(const void *)k_small_steps<MODE, true, 1>, (const void *)k_small_steps<MODE, false, 1>,
                                 (const void *)k_small_steps<MODE, true, 3>, (const void *)k_small_steps<MODE, false, 3>};
      for (const void *k : ks) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMALL_SMEM_MAX);
        if (e != cudaSuccess) return e;
      }
      done[dev] = true;
    }
  }
  const size_t smem = small_smem_bytes(pl, MODE, s.n);
#define NB_SMALL(QA, NC) \
  k_small_steps<MODE, QA, NC><<<1, SMALL_BLOCK, smem, st>>>(p, s, pl.block, (int)pl.jchunk, pl.n_jc, step0, nsteps, err)
  if (s.n <= SMALL_COMP_N) {
    if (s.q) NB_SMALL(true, 1); else NB_SMALL(false, 1);
  } else {
    if (s.q) NB_SMALL(true, 3); else NB_SMALL(false, 3);
  }
#undef NB_SMALL
  return cudaGetLastError();
}

cudaError_t launch_small_steps(const Plan &pl, int mode, const Phys &p, const StateView &s,
                               int64_t step0, int64_t nsteps, unsigned *err, cudaStream_t st) {
  if (s.n < 1 || s.n > SMALL_MAX_N || pl.sym || small_smem_bytes(pl, mode, s.n) > (size_t)SMALL_SMEM_MAX)
    return cudaErrorInvalidValue;
  switch (mode) {
    case MODE_FP64: return launch_small_m<MODE_FP64>(pl, p, s, step0, nsteps, err, st);
    case MODE_MIXED: return launch_small_m<MODE_MIXED>(pl, p, s, step0, nsteps, err, st);
    case MODE_SPLIT: return launch_small_m<MODE_SPLIT>(pl, p, s, step0, nsteps, err, st);
    case MODE_DF64: return launch_small_m<MODE_DF64>(pl, p, s, step0, nsteps, err, st);
    case MODE_SQRTDIV: return launch_small_m<MODE_SQRTDIV>(pl, p, s, step0, nsteps, err, st);
    case MODE_RSQ: return launch_small_m<MODE_RSQ>(pl, p, s, step0, nsteps, err, st);
    case MODE_RSQ_NR1: return launch_small_m<MODE_RSQ_NR1>(pl, p, s, step0, nsteps, err, st);
    case MODE_RSQ_NR2: return launch_small_m<MODE_RSQ_NR2>(pl, p, s, step0, nsteps, err, st);
    case MODE_SPLIT_RSQ: return launch_small_m<MODE_SPLIT_RSQ>(pl, p, s, step0, nsteps, err, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace nb
