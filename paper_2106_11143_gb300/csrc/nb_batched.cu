// nb_batched.cu -- persistent velocity-Verlet kernel for an ensemble of
// independent ion systems of uneven size (e.g. Kibble-Zurek quench
// realisations, Sec. I of the paper: many independent numerical experiments
// for defect statistics).
//
// One launch advances every instance by nsteps.  Each instance belongs to
// exactly one CTA, which keeps the instance's positions (and charges) in
// shared memory for the whole run, so no CTA ever waits on another CTA.
// Per step the CTA runs: drift of its ions, __syncthreads, the all-pairs
// Coulomb sum (the FP64 or the double-float pair term of the single-system
// kernels) and the
// kick/trap/friction/Langevin update of each ion, __syncthreads.  Velocities
// and accelerations stay in global memory (L2-resident).
//
// Load balance: instances are packed onto at most one CTA per SM by the
// longest-processing-time rule on N^2 (host side, nb_plan_batched); each
// CTA runs its instances one after another.  The schedule is passed to the
// kernel by value (__grid_constant__), so a launch needs no host-to-device
// copy and can be captured in a CUDA graph.
//
// Instances of at most 4096 ions use a half-pair force phase: btri_forces
// below, which has no FP64 in its pair loop, or bsym_forces for unusual
// scales; larger instances use the one-sided phase.
// Either way the arithmetic of an ion depends only on its instance (a fixed
// pair order and accumulation order per ion), not on the schedule or the block
// size, so results are bitwise reproducible.
#include <algorithm>
#include <mutex>
#include <vector>

#include "nb_tri.cuh"
#include "nb_verlet.cuh"

namespace nb {

struct __align__(16) BD4 {
  double x, y, z, w;
};

constexpr int BATCH_MAX_INST = 1024;
constexpr int BATCH_MAX_BINS = 1024;
static_assert(BATCH_MAX_INST == BATCH_LIMIT_INST, "schedule arrays sized for the validated instance limit");
// ions per instance (BATCH_LIMIT_N, checked on the host): 32 B each in shared memory
static_assert(sizeof(Phys) % 16 == 0 && sizeof(Phys) + BATCH_LIMIT_N * sizeof(BD4) <= 227 * 1024 - 1024,
              "an instance's parameters and positions fit one block's shared memory");

struct BatchSched {
  int n_inst;
  int n_bins;
  int off[BATCH_MAX_INST + 1];                      // ion offsets of the instances
  unsigned short order[BATCH_MAX_INST];             // instances, grouped by bin
  unsigned short bin_start[BATCH_MAX_BINS + 1];     // bin b = order[bin_start[b] .. bin_start[b+1])
};

// An instance's ions: positions in shared memory, charges in the caller's
// array (nullptr: one species).
struct BIons {
  const double *x, *y, *z, *q;
  int n;
};
// Ion i with its weight as the pair terms take it (an FP64 value for fp64, an
// FP32 (hi, lo) pair for df64); past the end a weight-0 dummy far away.
template <bool QARR, bool DF>
__device__ __forceinline__ BD4 bion(const BIons &v, int i) {
  BD4 r{1e18, 1e18, 1e18, 0.0};
  if (i < v.n) {
    r.x = v.x[i];
    r.y = v.y[i];
    r.z = v.z[i];
    r.w = QARR ? v.q[i] : 1.0;
    if (DF) {
      float qh = 1.0f, ql = 0.0f;
      if (QARR) split_f64(v.q[i], qh, ql);
      *reinterpret_cast<float2 *>(&r.w) = make_float2(qh, ql);
    }
  }
  return r;
}

// FP64 pair term, identical arithmetic to the single-system force kernel.
template <bool QARR>
__device__ __forceinline__ void bpair(double xi, double yi, double zi, const BD4 &pj, double soft2,
                                      double &ax, double &ay, double &az) {
  const double dx = xi - pj.x;
  const double dy = yi - pj.y;
  const double dz = zi - pj.z;
  double s = rinv3_fp64(dx, dy, dz, soft2);
  if (QARR) s *= pj.w;
  ax = fma(dx, s, ax);
  ay = fma(dy, s, ay);
  az = fma(dz, s, az);
}

// Double-float (FP64-class) pair term, as in the single-system df64 kernel;
// w carries q_j as an FP32 (hi, lo) pair in its bits.
template <bool QARR>
__device__ __forceinline__ void bpair_df64(double xi, double yi, double zi, const BD4 &pj,
                                           float s2h, float s2l, float ah[3], float al[3]) {
  float dh[3], dl[3];
  split_f64(xi - pj.x, dh[0], dl[0]);
  split_f64(yi - pj.y, dh[1], dl[1]);
  split_f64(zi - pj.z, dh[2], dl[2]);
  float sh, sl;
  df_rinv3(dh, dl, s2h, s2l, sh, sl);
  if (QARR) {
    const float2 q = *reinterpret_cast<const float2 *>(&pj.w);
    const float ph = sh * q.x;
    sl = fmaf(sh, q.y, fmaf(sl, q.x, fmaf(sh, q.x, -ph)));
    sh = ph;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float ph = dh[k] * sh;
    const float pl = fmaf(dh[k], sl, fmaf(dl[k], sh, fmaf(dh[k], sh, -ph)));
    float s, t;
    two_sum_f(ah[k], ph, s, t);
    ah[k] = s;
    al[k] += t + pl;
  }
}

// ---------------------------------------------------------------------------
// Half-pair (Newton's third law) force phase for instances of at most
// BATCH_SYM_N ions.  The instance is padded to whole 32-ion tiles with
// weight-0 dummies far away; the per-ion sums go to FP64 accumulators in
// shared memory.  A diagonal phase evaluates each tile against itself
// (one-sided); then Tp - 1 rounds of a round-robin schedule (circle method on
// Tp = T rounded up to even tiles, a bye for odd T) pair every two tiles once,
// each tile appearing once per round, so the warps of a round touch disjoint
// accumulators; a barrier separates the rounds.  Within a tile pair a lane
// holds one ion of tile a, reads tile b at the rotated index (lane + r) mod 32
// and rotates tile b's accumulators by shuffle.  The order of every sum is
// fixed by the schedule, not by the block size.
constexpr int BATCH_SYM_N = 4096;
constexpr int BATCH_THREADS_MAX = 512;
constexpr int BTRI_STAGE4 = 3 * 32;  // float4 per warp: a Q-tile's words
static_assert(sizeof(Phys) + BATCH_SYM_N * 6 * sizeof(double) + BATCH_THREADS_MAX / 32 * BTRI_STAGE4 * sizeof(float4) <=
                  227 * 1024 - 1024,
              "the half-pair phase's accumulators and staged tiles fit beside the positions");

__device__ __forceinline__ double bshfl_next(double v, int lane) {
  return __shfl_sync(0xffffffffu, v, (lane + 1) & 31);
}

template <bool W>
__device__ __forceinline__ void bsym_eval(const BD4 &p, const BD4 &q, double soft2, double a[3],
                                          double b[3]) {
  const double dx = p.x - q.x, dy = p.y - q.y, dz = p.z - q.z;
  const double s = rinv3_fp64(dx, dy, dz, soft2);
  const double sp = W ? s * q.w : s, sq = W ? s * p.w : s;
  a[0] = fma(dx, sp, a[0]);
  a[1] = fma(dy, sp, a[1]);
  a[2] = fma(dz, sp, a[2]);
  b[0] = fma(-dx, sq, b[0]);
  b[1] = fma(-dy, sq, b[1]);
  b[2] = fma(-dz, sq, b[2]);
}

// The double-float pair term for both ions (df64): P side (ah, al) += w_q d s,
// Q side (bh, bl) -= w_p d s, with the weights as FP32 (hi, lo) pairs in w.
__device__ __forceinline__ void df_scale(float sh, float sl, double w, float &oh, float &ol) {
  const float2 q = *reinterpret_cast<const float2 *>(&w);
  oh = sh * q.x;
  ol = fmaf(sh, q.y, fmaf(sl, q.x, fmaf(sh, q.x, -oh)));
}

template <bool W>
__device__ __forceinline__ void bsym_eval_df64(const BD4 &p, const BD4 &q, float s2h, float s2l,
                                               float ah[3], float al[3], float bh[3], float bl[3]) {
  float dh[3], dl[3];
  split_f64(p.x - q.x, dh[0], dl[0]);
  split_f64(p.y - q.y, dh[1], dl[1]);
  split_f64(p.z - q.z, dh[2], dl[2]);
  float sh, sl;
  df_rinv3(dh, dl, s2h, s2l, sh, sl);
  float sah = sh, sal = sl, sbh = sh, sbl = sl;
  if (W) {
    df_scale(sh, sl, q.w, sah, sal);
    df_scale(sh, sl, p.w, sbh, sbl);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float ph = dh[k] * sah;
    const float pl = fmaf(dh[k], sal, fmaf(dl[k], sah, fmaf(dh[k], sah, -ph)));
    float u, t;
    two_sum_f(ah[k], ph, u, t);
    ah[k] = u;
    al[k] += t + pl;
    float qh = ph, ql = pl;
    if (W) {
      qh = dh[k] * sbh;
      ql = fmaf(dh[k], sbl, fmaf(dl[k], sbh, fmaf(dh[k], sbh, -qh)));
    }
    two_sum_f(bh[k], -qh, u, t);
    bh[k] = u;
    bl[k] += t - ql;
  }
}

// Tiles (a, b) of round rho, pair k, for Tp tiles (circle method).
__device__ __forceinline__ void round_pair(int rho, int k, int Tp, int &a, int &b) {
  if (k == 0) {
    a = rho;
    b = Tp - 1;
  } else {
    a = (rho + k) % (Tp - 1);
    b = (rho - k + Tp - 1) % (Tp - 1);
  }
}

// The force phase: acc[c * npad + i] = sum_j w_j (r_i - r_j) / |r_i - r_j|^3
// for the instance's np32 staged entries (n real ions, weights in w: an FP64
// value for fp64, an FP32 (hi, lo) pair for df64).
template <bool QARR, bool W, bool DF>
__device__ __forceinline__ void bsym_tile_pair(const BIons &v, const BD4 &pp, int q0, int lane, double soft2,
                                               float s2h, float s2l, double a[3], double b[3]) {
  if (DF) {
    float ah[3] = {0, 0, 0}, al[3] = {0, 0, 0}, bh[3] = {0, 0, 0}, bl[3] = {0, 0, 0};
#pragma unroll 2
    for (int r = 0; r < 32; ++r) {
      bsym_eval_df64<W>(pp, bion<QARR, DF>(v, q0 + ((lane + r) & 31)), s2h, s2l, ah, al, bh, bl);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        bh[c] = __shfl_sync(0xffffffffu, bh[c], (lane + 1) & 31);
        bl[c] = __shfl_sync(0xffffffffu, bl[c], (lane + 1) & 31);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      a[c] = f32_to_f64(ah[c]) + f32_to_f64(al[c]);
      b[c] = f32_to_f64(bh[c]) + f32_to_f64(bl[c]);
    }
  } else {
    a[0] = a[1] = a[2] = b[0] = b[1] = b[2] = 0.0;
#pragma unroll 2
    for (int r = 0; r < 32; ++r) {
      bsym_eval<W>(pp, bion<QARR, DF>(v, q0 + ((lane + r) & 31)), soft2, a, b);
      b[0] = bshfl_next(b[0], lane);
      b[1] = bshfl_next(b[1], lane);
      b[2] = bshfl_next(b[2], lane);
    }
  }
}

template <bool QARR, bool DF>
__device__ __noinline__ void bsym_forces(const BIons v, double *acc, int npad, double soft2, float s2h, float s2l) {
  const int n = v.n, np32 = (n + 31) & ~31;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NW = blockDim.x >> 5;
  const int T = np32 >> 5;
  const bool ragged = (n & 31) != 0;
  // diagonal tiles, one-sided (the self pair gives 0)
  for (int t = warp; t < T; t += NW) {
    const int i = t * 32 + lane;
    const BD4 pi = bion<QARR, DF>(v, i);
    double a[3] = {0.0, 0.0, 0.0};
    const bool w = QARR || (ragged && t == T - 1);
    if (DF) {
      float ah[3] = {0, 0, 0}, al[3] = {0, 0, 0}, bh[3], bl[3];
      for (int j = 0; j < 32; ++j) {
        bh[0] = bh[1] = bh[2] = bl[0] = bl[1] = bl[2] = 0.0f;  // the partner side is not used
        if (w)
          bsym_eval_df64<true>(pi, bion<QARR, DF>(v, t * 32 + j), s2h, s2l, ah, al, bh, bl);
        else
          bsym_eval_df64<false>(pi, bion<QARR, DF>(v, t * 32 + j), s2h, s2l, ah, al, bh, bl);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) a[c] = f32_to_f64(ah[c]) + f32_to_f64(al[c]);
    } else {
      double dummy[3];
      if (w) {
        for (int j = 0; j < 32; ++j) bsym_eval<true>(pi, bion<QARR, DF>(v, t * 32 + j), soft2, a, dummy);
      } else {
        for (int j = 0; j < 32; ++j) bsym_eval<false>(pi, bion<QARR, DF>(v, t * 32 + j), soft2, a, dummy);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[c * npad + i] = a[c];
  }
  __syncthreads();
  const int Tp = T + (T & 1);
  for (int rho = 0; rho < Tp - 1; ++rho) {
    for (int k = warp; k < Tp / 2; k += NW) {
      int ta, tb;
      round_pair(rho, k, Tp, ta, tb);
      if (ta >= T || tb >= T) continue;  // the bye of an odd tile count
      const BD4 pp = bion<QARR, DF>(v, ta * 32 + lane);
      double a[3], b[3];
      if (QARR || (ragged && (ta == T - 1 || tb == T - 1)))
        bsym_tile_pair<QARR, true, DF>(v, pp, tb * 32, lane, soft2, s2h, s2l, a, b);
      else
        bsym_tile_pair<QARR, false, DF>(v, pp, tb * 32, lane, soft2, s2h, s2l, a, b);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        acc[c * npad + ta * 32 + lane] += a[c];
        acc[c * npad + tb * 32 + lane] += b[c];
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// The half-pair force phase on the FP32 pipe (nb_tri.cuh), both precisions.
//
// The instance is cut into S super-tiles of 128 ions, four 32-ion tiles each.
// A task (A, B, t) takes the 128 ions of A as the P side (four per lane) and
// tile t of B as the Q side; B = A is one-sided.  Tasks are numbered round by
// round: round 0 holds the S diagonal super-tiles, rounds 1 .. pair every two
// super-tiles once (circle method, as above), four tasks to a pair.  Each warp
// takes one task of every NW.  The arithmetic only reads positions; the sums
// are then added to the accumulators in the order of the rounds and, on a pair's
// A, of its four tasks, so that every ion's sum has one order whatever the
// number of warps.  That order is kept by a counter per super-tile of the tasks
// that have added to it: a task waits for its turn on A and, on B, for the
// earlier rounds, and no barrier stands between tasks, so a warp's FP64 adds
// overlap the others' pair arithmetic.  A task waits only for lower-numbered
// ones, which warps take in order, so the lowest unfinished never waits; the
// wait is bounded all the same (ERR_TIMEOUT).
//
// What bounds it: the FMA pipe, as in nb_tri.cu, 79 % busy with 152 instances of
// 4096 (issue 55 %, FP64 pipe 23 %) and 16 warps per SM (the registers' limit);
// units and words are formed from the FP64 positions at every task
// (600 instructions against 11 000 of pair arithmetic), diagonal super-tiles are
// one-sided, and below about 500 ions there are fewer tasks than warps.  Two
// steps of 512 instances of 32 .. 4096 ions: 15.6 ms (383 G pairs/s) against
// 59.9 (fp64) and 25.8 ms (df64) with bsym_forces; 152 instances of 4096: 11.2
// against 45.9 and 18.7 ms.  With the tasks' adds between barriers instead of
// counters the FP64 adds of all 16 warps coincided, a third slower.  With one
// unit per instance an ion far out, or a few kicked ones, sent every task to FP64
// (37.8 ms instead of 2.7 for 152 instances of 64 .. 2048 with one ion at 5 m; 3.7
// now).  Residues of cut coordinates (nb_tri.cuh) are formed before the turn too.
constexpr int BTRI_PI = 128;

// Bounded wait of a warp for counter c to reach v (about a second).
constexpr int BTRI_SPIN_LIMIT = 1 << 24;
__device__ __forceinline__ bool btri_wait(const int *c, int v) {
  bool ok = false;
  if ((threadIdx.x & 31) == 0)
    for (int k = 0; k < BTRI_SPIN_LIMIT && !ok; ++k) {
      ok = *(const volatile int *)c >= v;
      if (!ok) __nanosleep(32);
    }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  __threadfence_block();
  return ok;
}
// A task's turn: the counters of A and (two super-tiles) B and what to wait for.
struct BTurn {
  const int *a, *b;
  int va, vb;
  __device__ __forceinline__ bool wait(bool one) const {
    const bool ok = btri_wait(a, va);
    return (one || btri_wait(b, vb)) && ok;
  }
};

// A task in FP64 (nb_tri.cuh's limits): the P side's np ions (a multiple of 32, at
// most 128) against tile q0 .. q0 + 31, all of it before its turn.
template <bool QARR>
__device__ __noinline__ bool btri_task_fp64(const BIons v, int p0, int np, int q0, bool one, double soft2, double *acc,
                                            int npad, const BTurn turn) {
  const int lane = threadIdx.x & 31;
  double a[4][3], b[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    a[u][0] = a[u][1] = a[u][2] = 0.0;
    if (32 * u >= np) continue;
    const int i = p0 + 32 * u + lane;
#pragma unroll 1
    for (int r = 0; r < 32; ++r) {
      const int j = q0 + ((lane + r) & 31);
      if (i < v.n && j < v.n && i != j) {
        const BD4 pi = bion<QARR, false>(v, i), pj = bion<QARR, false>(v, j);
        bsym_eval<QARR>(pi, pj, soft2, a[u], b);
      }
      for (int c = 0; c < 3; ++c) b[c] = bshfl_next(b[c], lane);
    }
  }
  if (!turn.wait(one)) return false;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = p0 + 32 * u + lane;
    if (32 * u < np && i < v.n)
      for (int c = 0; c < 3; ++c) acc[c * npad + i] += a[u][c];
  }
  if (!one && q0 + lane < v.n)
    for (int c = 0; c < 3; ++c) acc[c * npad + q0 + lane] += b[c];
  return true;
}

// A task's residues (tri_residues): rs[u] those of ion p0 + 32 u + lane, rs[np / 32]
// those of ion q0 + lane.
template <bool QARR>
__device__ __noinline__ void btri_residues(const BIons v, int p0, int np, int q0, double soft2, const TriScale sc,
                                           double (*rs)[3]) {
  tri_residues<QARR, TRI_NEAR>(v.n, v.x, v.y, v.z, v.q, soft2, p0, np, q0, sc.ex, rs[np >> 5],
                               [&](int u, int c, double w) { rs[u >> 5][c] = w; });
}

// One task: the pair arithmetic of the P side's 64 V ions from p0 against tile
// q0 .. q0 + 31, then, in its turn, the adds to acc.  The units are the task's
// own, from its 64 V + 32 ions: an ion far out, or a coordinate small beside its
// instance's, concerns the tasks that hold it alone.  False: the wait gave up.
// self as in tri_tile, or -1 for two super-tiles.
template <int V, bool QARR>
__device__ __forceinline__ bool btri_task(const BIons &v, double *acc, int npad, float4 *st, int ew, double soft2, int p0,
                                          int q0, int self, const BTurn &turn) {
  const int lane = threadIdx.x & 31, n = v.n;
  const bool one = self >= 0;
  TriScale sc;
  sc.ew = ew;
  int mx[3] = {0, 0, 0};
  auto grow = [&](int i) {
    if (i < n) {
      mx[0] = max(mx[0], __double2hiint(v.x[i]) & 0x7fffffff);
      mx[1] = max(mx[1], __double2hiint(v.y[i]) & 0x7fffffff);
      mx[2] = max(mx[2], __double2hiint(v.z[i]) & 0x7fffffff);
    }
  };
  grow(q0 + lane);
#pragma unroll
  for (int u = 0; u < 2 * V; ++u) grow(p0 + 32 * u + lane);
#pragma unroll
  for (int c = 0; c < 3; ++c) mx[c] = __reduce_max_sync(0xffffffffu, mx[c]);
  bool done = tri_axes<QARR>(mx, soft2, sc);
  float w0[2][4], w1[2][4], w2[2][4];
  __syncwarp();  // every lane is done with the last tile
  const int qf = tri_ion<QARR, TRI_NEAR, false>(q0 + lane, q0 + lane < n, v.x, v.y, v.z, v.q, sc, -TRI_FAR, w0[0], w1[0],
                                                w2[0]);
  st[lane] = make_float4(w0[0][0], w0[0][1], w0[0][2], w0[0][3]);
  st[32 + lane] = make_float4(w1[0][0], w1[0][1], w1[0][2], w1[0][3]);
  st[64 + lane] = make_float4(w2[0][0], w2[0][1], w2[0][2], w2[0][3]);
  int pf = 0;
  TriIons<V> p;
#pragma unroll
  for (int u = 0; u < V; ++u) {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int i = p0 + u * 64 + b * 32 + lane;
      pf |= tri_ion<QARR, TRI_NEAR, false>(i, i < n, v.x, v.y, v.z, v.q, sc, TRI_FAR, w0[b], w1[b], w2[b]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      p.h[u][c] = pk(w0[0][c], w0[1][c]);
      p.m[u][c] = pk(w1[0][c], w1[1][c]);
      p.l[u][c] = pk(w2[0][c], w2[1][c]);
    }
    p.wh[u] = pk(w0[0][3], w0[1][3]);
    p.wl[u] = pk(w1[0][3], w1[1][3]);
  }
  const int fl = __reduce_or_sync(0xffffffffu, pf | qf << 6);
  int rot = 0;  // rotations with residues, where both sides are near on an axis
  if (done && fl & fl >> 6) {
    rot = tri_rotations<TRI_NEAR>(n, v.x, v.y, v.z, p0, 64 * V, q0, sc.ex);
    done = 2 * rot <= 64 * V;
  }
  TriSums<V> ts;
  if (done) {
    const f32x2 zero = pk1(0.0f);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ts.bh[c] = ts.bl[c] = zero;
#pragma unroll
      for (int u = 0; u < V; ++u) ts.ah[u][c] = ts.al[u][c] = zero;
    }
    __syncwarp();
    auto ld = [&](int r, float4 &f0, float4 &f1, float4 &f2) {
      const float4 *e = st + ((lane + r) & 31);
      f0 = e[0];
      f1 = e[32];
      f2 = e[64];
    };
    float ymax;
    if (soft2 != 0.0) {
      float sh, sl;
      split_f64_scaled(soft2, 2 * (sc.em - 1022), sh, sl);
      ymax = one ? tri_tile<V, QARR, true, true>(p, ld, lane, self, pk1(sh), pk1(sl), ts)
                 : tri_tile<V, QARR, false, true>(p, ld, lane, -1, pk1(sh), pk1(sl), ts);
    } else {
      ymax = one ? tri_tile<V, QARR, true, false>(p, ld, lane, self, zero, zero, ts)
                 : tri_tile<V, QARR, false, false>(p, ld, lane, -1, zero, zero, ts);
    }
    done = !__any_sync(0xffffffffu, !(ymax <= TRI_YMAX_GRID));
  }
  if (!done) return btri_task_fp64<QARR>(v, p0, 64 * V, q0, one, soft2, acc, npad, turn);
  double rs[2 * V + 1][3];
  if (rot) btri_residues<QARR>(v, p0, 64 * V, q0, soft2, sc, rs);
  if (!turn.wait(one)) return false;
  const double fwd = pow2d((ew - 1023) - 2 * (sc.em - 1022));  // from the task's units
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float h0, h1, l0, l1;
#pragma unroll
    for (int u = 0; u < V; ++u) {
      upk(ts.ah[u][c], h0, h1);
      upk(ts.al[u][c], l0, l1);
      const int i = p0 + u * 64 + lane;
      if (i < n) acc[c * npad + i] = fma((double)h0 + (double)l0, fwd, acc[c * npad + i]);
      if (i + 32 < n) acc[c * npad + i + 32] = fma((double)h1 + (double)l1, fwd, acc[c * npad + i + 32]);
    }
    if (!one && q0 + lane < n) {
      upk(ts.bh[c], h0, h1);
      upk(ts.bl[c], l0, l1);
      double &a = acc[c * npad + q0 + lane];
      a = fma(((double)h0 + (double)l0) + ((double)h1 + (double)l1), fwd, a);
    }
  }
  if (rot)
#pragma unroll 1
    for (int u = 0; u <= 2 * V; ++u) {
      const int i = u < 2 * V ? p0 + 32 * u + lane : q0 + lane;
      if (i < n && (u < 2 * V || !one))
        for (int c = 0; c < 3; ++c) acc[c * npad + i] += rs[u][c];
    }
  return true;
}

template <bool QARR>
__device__ __forceinline__ void btri_forces(const BIons &v, double *acc, int npad, float4 *stage, int *cnt,
                                            int ew, double soft2, unsigned *err) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NW = blockDim.x >> 5;
  const int n = v.n, S = (n + BTRI_PI - 1) / BTRI_PI, odd = S & 1;
  const int per = 4 * (S >> 1);  // tasks of a round
  const int M = 4 * S + (S > 1 ? (S - 1 + odd) * per : 0);
  float4 *st = stage + warp * BTRI_STAGE4;
  for (int m = warp; m < M; m += NW) {
    const int k = m & 3;  // 4 S and per are multiples of 4
    int A = m >> 2, B = A, rd = 0;
    if (m >= 4 * S) {
      const int u = m - 4 * S, rho = u / per;
      rd = 1 + rho;
      round_pair(rho, ((u - rho * per) >> 2) + odd, S + odd, A, B);  // an odd S: pair 0 is the bye
    }
    const int p0 = A * BTRI_PI, q0 = B * BTRI_PI + 32 * k;
    const bool one = A == B;
    // rounds before this one that X has taken part in: all but its own bye
    auto before = [&](int X) { return rd - (odd && X < rd - 1 ? 1 : 0); };
    const BTurn turn{cnt + A, cnt + B, 4 * before(A) + k, 4 * before(B)};
    // a super-tile of at most 64 ions (the last one, or a small instance) has
    // one pair of P-ions per lane: a third less time for 1024 instances of 16 ..
    // 64 ions
    bool ok;
    if (q0 >= n)
      ok = turn.wait(one);
    else if (p0 + 64 < n)
      ok = btri_task<2, QARR>(v, acc, npad, st, ew, soft2, p0, q0, one ? k : -1, turn);
    else
      ok = btri_task<1, QARR>(v, acc, npad, st, ew, soft2, p0, q0, one ? k : -1, turn);
    if (!ok && lane == 0) atomicOr(err, ERR_TIMEOUT);
    __threadfence_block();
    __syncwarp();
    if (lane == 0) {
      atomicAdd(cnt + A, 1);
      if (!one) atomicAdd(cnt + B, 1);
    }
  }
  __syncthreads();
}

// The largest (or with MIN the smallest) of a value over the block; red holds
// one int per warp and is free again after the caller's next barrier.
template <bool MIN>
__device__ __forceinline__ int block_extreme(int v, int *red) {
  v = MIN ? __reduce_min_sync(0xffffffffu, v) : __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v = MIN ? min(v, red[w]) : max(v, red[w]);
  return v;
}

template <bool QARR, bool DF, bool SYM>
__global__ void __launch_bounds__(512, 1) k_batched(Phys pall, const Phys *__restrict__ ptab, StateView s,
                                                  const __grid_constant__ BatchSched sch,
                                                  int64_t step0, int64_t nsteps, int npad, unsigned *err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Phys &pinst = *reinterpret_cast<Phys *>(smem_raw);  // the running instance's parameters
  double *sx = reinterpret_cast<double *>(smem_raw + sizeof(Phys)), *sy = sx + npad, *sz = sy + npad;
  double *acc = sz + npad;                                       // SYM: [3][npad]
  float4 *stage = reinterpret_cast<float4 *>(acc + 3 * npad);    // SYM: BTRI_STAGE4 per warp
  double *sw = sz + npad;                                        // one-sided: the weights
  __shared__ int red[2][BATCH_THREADS_MAX / 32];
  __shared__ int cnt[BATCH_SYM_N / BTRI_PI];  // tasks that have added to each super-tile
  const int T = blockDim.x;
  const int tid = threadIdx.x;
  bool bad = false;

  for (int kk = sch.bin_start[blockIdx.x]; kk < sch.bin_start[blockIdx.x + 1]; ++kk) {
    const int inst = sch.order[kk];
    const int64_t i0 = sch.off[inst];
    const int n = sch.off[inst + 1] - sch.off[inst];
    __syncthreads();  // the previous instance is done with shared memory
    if (tid == 0) {
      // the instance's own table entry, or the shared parameters with the
      // instance word offset by the instance's index
      if (ptab) {
        pinst = ptab[inst];
      } else {
        pinst = pall;
        pinst.instance = pall.instance + (unsigned)inst;
      }
    }
    const BIons ions{sx, sy, sz, QARR ? s.q + i0 : nullptr, n};
    int wx = 0, wn = 0x7fffffff;  // the weights' largest and smallest exponent words
    for (int i = tid; i < n; i += T) {
      sx[i] = s.x[i0 + i];
      sy[i] = s.y[i0 + i];
      sz[i] = s.z[i0 + i];
      if (SYM && QARR && s.q[i0 + i] != 0.0) {
        const int w = __double2hiint(s.q[i0 + i]) & 0x7fffffff;
        wx = max(wx, w);
        wn = min(wn, w);
      }
      if (!SYM) sw[i] = bion<QARR, DF>(ions, i).w;
    }
    int ew = 1023;
    bool tri_w = true;  // the weights' range suits the FP32 path
    if (SYM && QARR) {
      wx = block_extreme<false>(wx, red[0]);
      wn = block_extreme<true>(wn, red[1]);
      ew = wx >> 20;
      tri_w = ew >= 1023 - 400 && ew <= 1023 + 400 && ew - (wn >> 20) <= TRI_WSPREAD;
    }
    __syncthreads();
    const Phys &p = pinst;
    const unsigned inst_id = p.instance;
    const double dt = p.dt, hdt2 = 0.5 * dt * dt;
    const double inv = 1.0 / (1.0 + p.gamma * dt / (2.0 * p.mass)), g = p.gamma / p.mass;
    const double sig = p.noise_T > 0.0 ? sqrt(2.0 * p.gamma * KB * p.noise_T * dt) / p.mass : 0.0;
    const double pref_u = p.k_coulomb * p.charge * p.charge / p.mass;
    const double soft2 = p.soft2;
    float s2h = 0.0f, s2l = 0.0f;
    if (DF) split_f64(soft2, s2h, s2l);
    for (int64_t st = 0; st < nsteps; ++st) {
      const int64_t snew = step0 + st + 1;
      const double t = p.t0 + (double)snew * dt;
      // drift: r+ = r + v dt + a dt^2/2 (each thread its own ions)
      if (SYM)
        for (int i = tid; i < BATCH_SYM_N / BTRI_PI; i += T) cnt[i] = 0;
      for (int i = tid; i < n; i += T) {
        const double rx = sx[i] + s.vx[i0 + i] * dt + hdt2 * s.ax[i0 + i];
        const double ry = sy[i] + s.vy[i0 + i] * dt + hdt2 * s.ay[i0 + i];
        const double rz = sz[i] + s.vz[i0 + i] * dt + hdt2 * s.az[i0 + i];
        sx[i] = rx;
        sy[i] = ry;
        sz[i] = rz;
        if (SYM) acc[i] = acc[npad + i] = acc[2 * npad + i] = 0.0;
      }
      __syncthreads();
      // forces at r+ and the kick
      if (SYM) {
        if (tri_w)
          btri_forces<QARR>(ions, acc, npad, stage, cnt, ew, soft2, err);
        else
          bsym_forces<QARR, DF>(ions, acc, npad, soft2, s2h, s2l);
      }
      for (int ib = 0; ib < n; ib += T) {
        const int i = ib + tid;
        const int ic = min(i, n - 1);
        const BD4 ri{sx[ic], sy[ic], sz[ic], 0.0};
        double a0 = 0.0, a1 = 0.0, a2 = 0.0;
        if (SYM) {
          if (i < n) {
            a0 = acc[i];
            a1 = acc[npad + i];
            a2 = acc[2 * npad + i];
          }
        } else if (DF) {
          float ah[3] = {0.0f, 0.0f, 0.0f}, al[3] = {0.0f, 0.0f, 0.0f};
          for (int j0 = 0; j0 < n; j0 += 256) {  // double-float sums flushed every 256 partners
            const int j1 = min(n, j0 + 256);
            for (int j = j0; j < j1; ++j) bpair_df64<QARR>(ri.x, ri.y, ri.z, BD4{sx[j], sy[j], sz[j], sw[j]}, s2h, s2l, ah, al);
            a0 += f32_to_f64(ah[0]) + f32_to_f64(al[0]);
            a1 += f32_to_f64(ah[1]) + f32_to_f64(al[1]);
            a2 += f32_to_f64(ah[2]) + f32_to_f64(al[2]);
            ah[0] = ah[1] = ah[2] = al[0] = al[1] = al[2] = 0.0f;
          }
        } else {
#pragma unroll 2
          for (int j = 0; j < n; ++j) bpair<QARR>(ri.x, ri.y, ri.z, BD4{sx[j], sy[j], sz[j], sw[j]}, soft2, a0, a1, a2);
        }
        if (i < n) {
          const int64_t gi = i0 + i;
          const double pref = QARR ? p.k_coulomb * s.q[gi] / p.mass : pref_u;
          double tr[3];
          trap_accel(p, t, ri.x, ri.y, ri.z, tr[0], tr[1], tr[2]);
          double xi[3] = {0.0, 0.0, 0.0};
          if (sig > 0.0) normals3(p.seed, inst_id, snew, i, xi);
          const double acc[3] = {a0, a1, a2};
          double *vs[3] = {s.vx, s.vy, s.vz};
          double *as[3] = {s.ax, s.ay, s.az};
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const double u = pref * acc[k] + tr[k];
            double v = (vs[k][gi] + 0.5 * dt * (as[k][gi] + u)) * inv;
            v += sig * xi[k];
            const double a = u - g * v;
            vs[k][gi] = v;
            as[k][gi] = a;
            bad |= not_finite(v) || not_finite(a);
          }
        }
      }
      __syncthreads();
    }
    for (int i = tid; i < n; i += T) {
      s.x[i0 + i] = sx[i];
      s.y[i0 + i] = sy[i];
      s.z[i0 + i] = sz[i];
    }
  }
  if (bad) atomicOr(err, ERR_NONFINITE);
}

// ---------------------------------------------------------------------------
// Longest-processing-time packing of instances (cost n^2) onto n_bins bins:
// instances in decreasing cost (ties by index) go to the currently lightest
// bin (ties by bin index).  Deterministic.
int batched_plan(int n_inst, const int64_t *offsets, int n_bins, unsigned short *order,
                 unsigned short *bin_start, double *max_load, double *mean_load) {
  std::vector<int> idx(n_inst);
  for (int k = 0; k < n_inst; ++k) idx[k] = k;
  auto cost = [&](int k) { const double m = (double)(offsets[k + 1] - offsets[k]); return m * m; };
  std::stable_sort(idx.begin(), idx.end(), [&](int a, int b) { return cost(a) > cost(b); });
  std::vector<double> load(n_bins, 0.0);
  std::vector<std::vector<int>> bins(n_bins);
  for (int k : idx) {
    int best = 0;
    for (int b = 1; b < n_bins; ++b)
      if (load[b] < load[best]) best = b;
    load[best] += cost(k);
    bins[best].push_back(k);
  }
  int pos = 0;
  double mx = 0.0, sum = 0.0;
  for (int b = 0; b < n_bins; ++b) {
    bin_start[b] = (unsigned short)pos;
    for (int k : bins[b]) order[pos++] = (unsigned short)k;
    mx = std::max(mx, load[b]);
    sum += load[b];
  }
  bin_start[n_bins] = (unsigned short)pos;
  if (max_load) *max_load = mx;
  if (mean_load) *mean_load = n_bins ? sum / n_bins : 0.0;
  return pos;
}

cudaError_t launch_batched(const Phys &p, const Phys *ptab, const StateView &s, int n_inst, const int64_t *offsets,
                           int n_bins, int threads, bool allow_sym, int64_t step0, int64_t nsteps, unsigned *err,
                           cudaStream_t st) {
  BatchSched sch;
  sch.n_inst = n_inst;
  sch.n_bins = n_bins;
  int maxn = 0;
  for (int k = 0; k <= n_inst; ++k) sch.off[k] = (int)offsets[k];
  for (int k = 0; k < n_inst; ++k) maxn = std::max(maxn, (int)(offsets[k + 1] - offsets[k]));
  batched_plan(n_inst, offsets, n_bins, sch.order, sch.bin_start, nullptr, nullptr);
  // Instances of at most BATCH_SYM_N ions use the half-pair force phase,
  // which adds the [3][npad] FP64 accumulators to the positions in shared memory.
  const bool df = p.precision == MODE_DF64;
  const bool sym = allow_sym && maxn <= BATCH_SYM_N;
  const int npad = (std::max(maxn, 1) + 31) & ~31;
  const size_t need = sizeof(Phys) + (sym ? (size_t)npad * 6 * sizeof(double) +
                                                (size_t)(threads / 32) * BTRI_STAGE4 * sizeof(float4)
                                          : (size_t)npad * 4 * sizeof(double));
  // At least 120 KB of shared memory per CTA, so no SM holds two bins: each
  // bin then owns one SM, which is what the LPT packing assumes.
  const size_t smem = std::max(need, (size_t)120 * 1024);
  static std::mutex mu;
  static bool attr_done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_done[dev]) {
      const int lim = 227 * 1024 - 1024;  // beside the block's static shared memory
      const void *fns[8] = {(const void *)k_batched<true, false, false>, (const void *)k_batched<false, false, false>,
                            (const void *)k_batched<true, true, false>,  (const void *)k_batched<false, true, false>,
                            (const void *)k_batched<true, false, true>,  (const void *)k_batched<false, false, true>,
                            (const void *)k_batched<true, true, true>,   (const void *)k_batched<false, true, true>};
      for (int f = 0; f < 8 && e == cudaSuccess; ++f)
        e = cudaFuncSetAttribute(fns[f], cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
      if (e != cudaSuccess) return e;
      attr_done[dev] = true;
    }
  }
  if (sym && s.q && df)
    k_batched<true, true, true><<<n_bins, threads, smem, st>>>(p, ptab, s, sch, step0, nsteps, npad, err);
  else if (sym && df)
    k_batched<false, true, true><<<n_bins, threads, smem, st>>>(p, ptab, s, sch, step0, nsteps, npad, err);
  else if (sym && s.q)
    k_batched<true, false, true><<<n_bins, threads, smem, st>>>(p, ptab, s, sch, step0, nsteps, npad, err);
  else if (sym)
    k_batched<false, false, true><<<n_bins, threads, smem, st>>>(p, ptab, s, sch, step0, nsteps, npad, err);
  else if (s.q && df)
    k_batched<true, true, false><<<n_bins, threads, smem, st>>>(p, ptab, s, sch, step0, nsteps, npad, err);
  else if (s.q)
    k_batched<true, false, false><<<n_bins, threads, smem, st>>>(p, ptab, s, sch, step0, nsteps, npad, err);
  else if (df)
    k_batched<false, true, false><<<n_bins, threads, smem, st>>>(p, ptab, s, sch, step0, nsteps, npad, err);
  else
    k_batched<false, false, false><<<n_bins, threads, smem, st>>>(p, ptab, s, sch, step0, nsteps, npad, err);
  return cudaGetLastError();
}

}  // namespace nb
