// nb_tri.cu -- half-pair force kernels whose pair loop has no FP64
// instruction: the FP64-class precisions (fp64, df64) and the literal mixed
// form, from three-word positions on the FP32 pipe (nb_tri.cuh).
//
// Work items and output are those of the half-pair kernels (nb_symsched.cuh):
// a block pair (P, Q), P <= Q, of BI = 32 G ions.  Each warp owns one P-tile of
// 64 V ions, 2 V per lane as V packed pairs, whose words stay in its registers
// for the whole item, and visits Q-tiles of 32 ions.  Q words sit in shared
// memory, each tile twice back to back, so that rotation r of a tile is a fixed
// offset; the Q side's sums rotate one lane per iteration by shuffle, one
// packed double-float per component (the low half sums the terms of the even
// P-ions of the lane, the high half the odd ones).  32 rotations evaluate every
// pair of the two tiles once.  The sums are double-floats within a tile and are
// added to FP64 accumulators in shared memory after it: the warp's own for P,
// and for Q the block's, which the warps visit in a staggered order with a
// barrier between steps.  Everything is in units of L; the output applies L^-2.
//
// Diagonal items (P == Q) run the same tiles one-sided (ONE).
//
// What bounds it: the FMA pipe, 135 lane-cycles per evaluation (30 for the
// normalised d, 18 for r^2, 18 for r^-3, 12 for the products, 48 for the two ions'
// TwoSum sums, 9 to keep them normalised), 81 % busy at n = 32768 with issue at
// 51 %, ALU 10 % and the FP64 pipe 24 % (the tiles' sums into FP64).  A half-pair
// kernel on the FP64 pipe (10.3 FP64 instructions per evaluation in fp64, 3.4 in
// df64) took 91.0 ms (fp64) and 34.0 ms (df64) at n = 1e5; this one takes 20.6 ms
// for both (19.2 with d unnormalised, whose small components lost bits: nb_tri.cuh).
// Conditioned error over all ions at n = 1e5: rms 2^-50.4, largest 2^-45.2, against
// 2^-50.1 and 2^-44.9 (fp64) and 2^-49.2 and 2^-43.9 (df64) there; norm of the error
// over that of the force, which the closest pairs set, rms of 200 clouds of 700 ..
// 5003 ions and 250 of 16384: 6.8, 7.1, 6.5 and 6.3e-15 against 8.6, 7.5, 6.7 and
// 6.5e-15 (single clouds go either way by up to 2).
//
// Measured and not kept: one pair of P-ions per lane (V = 1: twice the
// shuffles per evaluation, 5-8 % slower; kept for 64-ion blocks, which it
// needs); ordering the summands by FSETP/FSEL so that a Fast2Sum does (18
// FMA lane-cycles fewer, 2-6 % slower: the halves of a packed pair are moved
// apart and together); 256 threads and two blocks per SM instead of 128 and
// four (3-4 % slower at 256-ion blocks); unrolling 4 or 8 rotations (level).
//
// The literal mixed form (MIX) takes the same words: its displacement, formed
// exactly and rounded once to FP32, is the FP64 difference cast to FP32, at 8
// FMA lane-cycles per component.  With 38 lane-cycles per evaluation it runs
// 6.95 ms at n = 1e5 (FMA pipe 67 %), where three FP64 differences per evaluation
// took 31.9 ms, and gives its sums to
// FP64 rounding: every FP32 operation and partial sum is the same, in the same
// order (norm of the difference at most 2e-11 of the result over n = 2000 ..
// 1e5; FP32 ties of a displacement may round the other way).  A pairwise
// order of the FP32 sums would be 20 % faster and as accurate, but would change
// results in their eighth digit.
#include <algorithm>
#include <mutex>

#include "nb_symsched.cuh"
#include "nb_tri.cuh"

namespace nb {

// The tile step of the literal mixed form, operation for operation that of the
// FP64-difference kernel (sym_step_mixed and the diagonal loop of nb_sym.cu):
// the displacement rounded once to FP32 (h + l is exact, so RN(h + l) is), the
// arithmetic of f32_rinv3, and one FP32 sum of 32 terms per ion and 32 x 32
// tile pair, in the order of the rotations, or (ONE) of the partners.  Q sums,
// with the sign reversed: bh for the ions of pair 0, bl for pair 1.
template <int V, bool W, bool ONE>
__device__ __forceinline__ float tri_tile_mixed(const TriIons<V> &p, const float4 *qt, int lane, int self,
                                                TriSums<V> &t) {
  static_assert(V <= 2, "one Q sum per pair of P-ions");
  float ymax = 0.0f;
  const int next = (lane + 1) & 31;
  const f32x2 m15 = pk1(-1.5f), p15 = pk1(1.5f);
#pragma unroll 4
  for (int r = 0; r < 32; ++r) {
    const float4 q0 = qt[r], q1 = qt[64 + r], q2 = qt[128 + r];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      f32x2 d[3], h, l;
      tri_diff(p.h[v][0], p.m[v][0], p.l[v][0], pk1(q0.x), pk1(q1.x), pk1(q2.x), h, l);
      d[0] = padd(h, l);
      tri_diff(p.h[v][1], p.m[v][1], p.l[v][1], pk1(q0.y), pk1(q1.y), pk1(q2.y), h, l);
      d[1] = padd(h, l);
      tri_diff(p.h[v][2], p.m[v][2], p.l[v][2], pk1(q0.z), pk1(q1.z), pk1(q2.z), h, l);
      d[2] = padd(h, l);
      const f32x2 r2 = pfma(d[0], d[0], pfma(d[1], d[1], pmul(d[2], d[2])));
      float ra, rb;
      upk(r2, ra, rb);
      float ya = rsqrt_approx(ra), yb = rsqrt_approx(rb);
      const bool me0 = ONE && r == lane && self == 2 * v, me1 = ONE && r == lane && self == 2 * v + 1;
      ymax = fmaxf(ymax, fmaxf(me0 ? 0.0f : ya, me1 ? 0.0f : yb));
      if (ONE) {
        ya = fminf(ya, TRI_YMAX_GRID);
        yb = fminf(yb, TRI_YMAX_GRID);
      }
      const f32x2 y = pk(ya, yb), y2 = pmul(y, y), y3 = pmul(y2, y);
      const f32x2 s = pfma(y3, pfma(pmul(m15, r2), y2, p15), y3);
      const f32x2 sp = W ? pmul(s, pk1(q0.w)) : s, sq = W && !ONE ? pmul(s, p.wh[v]) : s;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        t.ah[v][c] = pfma(d[c], sp, t.ah[v][c]);
        if (!ONE) {
          f32x2 &b = v == 0 ? t.bh[c] : t.bl[c];
          b = pshfl(pfma(d[c], sq, b), next);
        }
      }
    }
  }
  return ymax;
}

// The same tile step in FP64 from the caller's positions, for tiles the FP32
// path leaves: ions [i0, i0 + ni) (the P-tile) against [j0, j0 + 32), those
// below n.  `sc` takes a force from its own units to the accumulators'.
template <bool ONE>
__device__ __noinline__ void tri_tile_fp64(int64_t n, const double *x, const double *y, const double *z,
                                           const double *q, double soft2, int64_t i0, int ni, int64_t j0, double sc,
                                           double *accP, int ldp, double *accQ, int ldq) {
  const int lane = threadIdx.x & 31;
  for (int u = 0; u < ni; u += 32) {
    const int64_t i = i0 + u + lane;
    double a[3] = {0.0, 0.0, 0.0}, b[3] = {0.0, 0.0, 0.0};
    for (int r = 0; r < 32; ++r) {
      const int64_t j = j0 + ((lane + r) & 31);
      if (i < n && j < n && i != j) {
        const double dx = x[i] - x[j], dy = y[i] - y[j], dz = z[i] - z[j];
        const double s = rinv3_fp64(dx, dy, dz, soft2);
        const double sp = (q ? s * q[j] : s), sq = (q ? s * q[i] : s);
        a[0] = fma(dx, sp, a[0]);
        a[1] = fma(dy, sp, a[1]);
        a[2] = fma(dz, sp, a[2]);
        b[0] = fma(-dx, sq, b[0]);
        b[1] = fma(-dy, sq, b[1]);
        b[2] = fma(-dz, sq, b[2]);
      }
      if (!ONE)
        for (int c = 0; c < 3; ++c) b[c] = __shfl_sync(0xffffffffu, b[c], (lane + 1) & 31);
    }
    for (int c = 0; c < 3; ++c) {
      accP[c * ldp + u + lane] += a[c] * sc;
      if (!ONE) accQ[c * ldq + lane] += b[c] * sc;
    }
  }
}

// Adds a tile's residues (tri_residues) to the accumulators.
template <bool QARR, int NEAR>
__device__ __noinline__ void tri_tile_residues(int64_t n, const double *x, const double *y, const double *z,
                                               const double *q, double soft2, int64_t i0, int ni, int64_t j0,
                                               const int *ex, bool one, double sc, double *accP, int ldp, double *accQ,
                                               int ldq) {
  const int lane = threadIdx.x & 31;
  double b[3];
  tri_residues<QARR, NEAR>(n, x, y, z, q, soft2, i0, ni, j0, ex, b,
                           [&](int u, int c, double v) { accP[c * ldp + u + lane] += v * sc; });
  if (!one)
    for (int c = 0; c < 3; ++c) accQ[c * ldq + lane] += b[c] * sc;
}

// The item's in-place output of the mixed form (sym_commit, nb_symsched.cuh,
// laid out for short items): the sums are formed before the wait for the
// previous round, and all of a thread's old values are loaded before the first
// is stored, so that a commit costs one trip to L2 instead of one per value.
// At n = 40000 (157 rounds of 256-ion blocks) the chain of commits bounded the
// mixed form: 24 % per evaluation against sym_commit.  The fp64
// items are three times as long and hide the chain: there sym_commit, with
// fewer registers, is faster (19.2 against 19.7 ms at n = 1e5, before d was normalised).
template <int NT, class FP, class FQ>
__device__ __forceinline__ void tri_commit(const SymItem &it, int64_t n, int BI, int64_t p0, int np, int64_t q0,
                                           int nq, double *out, int *sync, unsigned *err, FP sumP, FQ sumQ) {
  __shared__ int s_ok;
  const int tid = threadIdx.x;
  const bool two = it.P != it.Q;
  const bool first = it.round == 0;
  for (int i0 = tid; i0 < BI; i0 += 2 * NT) {
    double vp[2][3], vq[2][3];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int i = i0 + k * NT;
        vp[k][c] = i < np ? sumP(c, i) : 0.0;
        vq[k][c] = two && i < nq ? sumQ(c, i) : 0.0;
      }
    if (i0 < 2 * NT) {  // the first pass, every thread: BI >= NT
      if (tid == 0) {
        bool ok = true;
        if (it.round > 0) ok = sym_wait(sync, it.P, it.round, err) && (!two || sym_wait(sync, it.Q, it.round, err));
        if (!ok) atomicOr(err, ERR_TIMEOUT);
        s_ok = ok;
      }
      __syncthreads();
    }
    if (!s_ok) continue;
    if (!first) {
      double op[2][3], oq[2][3];
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int i = i0 + k * NT;
          op[k][c] = i < np ? __ldcg(out + c * n + p0 + i) : 0.0;
          oq[k][c] = two && i < nq ? __ldcg(out + c * n + q0 + i) : 0.0;
        }
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          vp[k][c] += op[k][c];
          vq[k][c] += oq[k][c];
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int i = i0 + k * NT;
        if (i < np) __stcg(out + c * n + p0 + i, vp[k][c]);
        if (two && i < nq) __stcg(out + c * n + q0 + i, vq[k][c]);
      }
  }
  __syncthreads();  // every thread's adds happen before thread 0's release
  if (tid == 0) {
    __threadfence();
    st_release(sync + 1 + it.P, it.round + 1);
    if (two) st_release(sync + 1 + it.Q, it.round + 1);
  }
}

template <bool MIX, int V, bool QARR, int NT, int NB, bool INPLACE, bool SOFT>
__global__ void __launch_bounds__(NT, NB)
    k_pair_sym_tri(int64_t n, int nbk, int G, int SB, const double *__restrict__ x, const double *__restrict__ y,
                   const double *__restrict__ z, const double *__restrict__ q, double soft2, double *__restrict__ out,
                   int *__restrict__ sync, unsigned *err) {
  constexpr int NW = NT / 32, PI = 64 * V;  // warps; ions of a P-tile
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int BI = 32 * G;
  float4 *qs = reinterpret_cast<float4 *>(smem_raw);                 // [G][TRI_TILE4]
  double *accQ = reinterpret_cast<double *>(qs + G * TRI_TILE4);     // [3][BI]
  double *accP = accQ + 3 * BI;                                      // [NW][3][PI]
  __shared__ int qf[32];                                             // places of each Q-tile (G <= 32)
  __shared__ int ex[3];                                              // the axes' exponents, for tri_residues
  const SymItem it = sym_block_item(INPLACE, sync, nbk);
  const int64_t p0 = (int64_t)it.P * BI, q0 = (int64_t)it.Q * BI;
  const int np = (int)min((int64_t)BI, n - p0), nq = (int)min((int64_t)BI, n - q0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool diag = it.P == it.Q;
  TriScale sc;
  const bool fast = tri_scale<NT, QARR>(p0, np, q0, diag ? 0 : nq, x, y, z, q, soft2, sc);
  // units: a coordinate is L X with L = 2^(em - 1022), a weight 2^(ew - 1023) w
  const int kl = fast ? sc.em - 1022 : 0, kw = fast ? sc.ew - 1023 : 0;

  const int PT = BI / PI, NG = NW / PT, nqt = G / NG;  // P-tiles, warps per P-tile, Q-tiles per warp
  const int pt = warp % PT, grp = warp / PT;
  TriIons<V> p;
  int pf = 0;
  bool low;
  if (tid == 0) {
    ex[0] = sc.ex[0];
    ex[1] = sc.ex[1];
    ex[2] = sc.ex[2];
  }
  if (fast) pf = tri_load<V, QARR, NT, MIX ? TRI_NEAR_MIX : TRI_NEAR, false>(p, qs, qf, BI, pt, p0, np, q0, nq, x, y, z, q, sc, low);
  for (int i = tid; i < 3 * BI; i += NT) accQ[i] = 0.0;
  for (int i = tid; i < NW * 3 * PI; i += NT) accP[i] = 0.0;
  __syncthreads();
  f32x2 s2h = 0, s2l = 0;
  if (SOFT) {
    float sh, sl;
    split_f64_scaled(soft2, 2 * kl, sh, sl);
    s2h = pk1(sh);
    s2l = pk1(sl);
  }

  double *aP = accP + warp * 3 * PI;
  const double back = pow2d(2 * kl - kw);  // own units -> the accumulators'
  const bool live = pt * PI < np;          // the P-tile holds ions
  for (int k = 0; k < nqt; ++k) {
    // distinct over the P-tiles of a step: nqt >= PT
    const int t = grp * nqt + (k + pt) % nqt;
    if (k > 0) __syncthreads();  // the Q sums of the last step are written
    double *aQ = accQ + t * 32;
    if (!live || t * 32 >= nq) continue;
    // a diagonal item's tile pairs are one-sided; in the mixed form only within
    // a sub-block of SB tiles, and across sub-blocks each pair is taken once,
    // from the lower one
    const int sp = pt * 2 * V / SB, sq = t / SB;
    const bool one = diag && (!MIX || sp == sq);
    if (MIX && diag && sp > sq) continue;
    bool done = false;
    int rot = 0;  // rotations with residues, where both sides are near on an axis
    if (fast && (pf & qf[t]))
      rot = tri_rotations<MIX ? TRI_NEAR_MIX : TRI_NEAR>(n, x, y, z, p0 + pt * PI, PI, q0 + t * 32, ex);
    if (fast && 2 * rot <= PI) {
      TriSums<V> ts;
      const f32x2 zero = pk1(0.0f);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        ts.bh[c] = ts.bl[c] = zero;
#pragma unroll
        for (int v = 0; v < V; ++v) ts.ah[v][c] = ts.al[v][c] = zero;
      }
      const float4 *qt = qs + t * TRI_TILE4 + lane;
      auto ld = [&](int r, float4 &q0, float4 &q1, float4 &q2) {
        q0 = qt[r];
        q1 = qt[64 + r];
        q2 = qt[128 + r];
      };
      float ymax;
      if (one) {
        const int u = t - pt * 2 * V;  // the lane's own ion in this Q-tile, if any
        const int self = u >= 0 && u < 2 * V ? u : -1;
        ymax = MIX ? tri_tile_mixed<V, QARR, true>(p, qt - lane, lane, self, ts)
                   : tri_tile<V, QARR, true, SOFT>(p, ld, lane, self, s2h, s2l, ts);
      } else {
        ymax = MIX ? tri_tile_mixed<V, QARR, false>(p, qt, lane, -1, ts)
                   : tri_tile<V, QARR, false, SOFT>(p, ld, lane, -1, s2h, s2l, ts);
      }
      done = !__any_sync(0xffffffffu, !(ymax <= TRI_YMAX_GRID));
      if (done) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float h0, h1, l0, l1;
#pragma unroll
          for (int v = 0; v < V; ++v) {
            upk(ts.ah[v][c], h0, h1);
            upk(ts.al[v][c], l0, l1);
            double *d = aP + c * PI + v * 64 + lane;
            d[0] += MIX ? f32_to_f64(h0) : (double)h0 + (double)l0;
            d[32] += MIX ? f32_to_f64(h1) : (double)h1 + (double)l1;
          }
          if (!one) {
            upk(ts.bh[c], h0, h1);
            upk(ts.bl[c], l0, l1);
            if (MIX)
              aQ[c * BI + lane] -= (f32_to_f64(h0) + f32_to_f64(h1)) + (f32_to_f64(l0) + f32_to_f64(l1));
            else
              aQ[c * BI + lane] += ((double)h0 + (double)l0) + ((double)h1 + (double)l1);
          }
        }
        if (rot)
          tri_tile_residues<QARR, MIX ? TRI_NEAR_MIX : TRI_NEAR>(n, x, y, z, q, soft2, p0 + pt * PI, PI, q0 + t * 32, ex,
                                                                 one, back, aP, PI, aQ, BI);
      }
    }
    if (!done) {
      if (one)
        tri_tile_fp64<true>(n, x, y, z, q, soft2, p0 + pt * PI, PI, q0 + t * 32, back, aP, PI, aQ, BI);
      else
        tri_tile_fp64<false>(n, x, y, z, q, soft2, p0 + pt * PI, PI, q0 + t * 32, back, aP, PI, aQ, BI);
    }
  }
  __syncthreads();
  const double fwd = pow2d(kw - 2 * kl);
  auto sumP = [&](int c, int i) {
    double v = 0.0;
    const double *s = accP + (i / PI) * 3 * PI + c * PI + i % PI;
    for (int g = 0; g < NG; ++g) v += s[g * PT * 3 * PI];
    if (MIX && diag) v += accQ[c * BI + i];  // across its sub-blocks
    return v * fwd;
  };
  auto sumQ = [&](int c, int i) { return accQ[c * BI + i] * fwd; };
  if (MIX && INPLACE)
    tri_commit<NT>(it, n, BI, p0, np, q0, nq, out, sync, err, sumP, sumQ);
  else
    sym_output<NT>(INPLACE, it, n, p0, np, q0, nq, out, sync, err, sumP, sumQ);
}

// ---------------------------------------------------------------------------
template <int V, int NT>
static size_t tri_smem(int G) {
  return (size_t)G * TRI_TILE4 * sizeof(float4) + (size_t)3 * 32 * G * sizeof(double) +
         (size_t)(NT / 32) * 3 * 64 * V * sizeof(double);
}

template <bool MIX, int V, int NT, int NB, bool SOFT = false>
static cudaError_t launch_tri(int64_t n, int nbk, int G, int SB, const double *x, const double *y, const double *z,
                              const double *q, double soft2, double *part, int *sync, unsigned *err, bool inplace,
                              cudaStream_t st) {
  static std::mutex mu;
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!done[dev]) {
      const void *fns[4] = {(const void *)k_pair_sym_tri<MIX, V, true, NT, NB, true, SOFT>,
                            (const void *)k_pair_sym_tri<MIX, V, false, NT, NB, true, SOFT>,
                            (const void *)k_pair_sym_tri<MIX, V, true, NT, NB, false, SOFT>,
                            (const void *)k_pair_sym_tri<MIX, V, false, NT, NB, false, SOFT>};
      for (int k = 0; k < 4 && e == cudaSuccess; ++k)
        e = cudaFuncSetAttribute(fns[k], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tri_smem<V, NT>(32));
      if (e != cudaSuccess) return e;
      done[dev] = true;
    }
  }
  if (inplace) {
    e = cudaMemsetAsync(sync, 0, sizeof(int) * sym_sync_ints(nbk), st);
    if (e != cudaSuccess) return e;
  }
  const unsigned items = (unsigned)sym_items(nbk);
  const size_t smem = tri_smem<V, NT>(G);
#define NB_TRI_LAUNCH(QA, IP) \
  k_pair_sym_tri<MIX, V, QA, NT, NB, IP, SOFT><<<items, NT, smem, st>>>(n, nbk, G, SB, x, y, z, q, soft2, part, sync, err)
  if (inplace) {
    if (q) NB_TRI_LAUNCH(true, true); else NB_TRI_LAUNCH(false, true);
  } else {
    if (q) NB_TRI_LAUNCH(true, false); else NB_TRI_LAUNCH(false, false);
  }
#undef NB_TRI_LAUNCH
  return cudaGetLastError();
}

// The softened mixed form stays with nb_sym.cu, and so do 32-ion blocks (mixed
// below n = 2000, where 16-term FP32 sums are more accurate than 32-term ones at
// the same speed; elsewhere by set_tuning only).
static bool tri_sums(const Plan &pl, int mode, double soft2) {
  return pl.sym && (mode == MODE_FP64 || mode == MODE_DF64 || (mode == MODE_MIXED && soft2 == 0.0));
}
bool tri_serves(const Plan &pl, int mode, double soft2) { return tri_sums(pl, mode, soft2) && pl.G >= 2; }

// Block sizes, the fastest measured over n = 1500 .. 150000 (fp64): 64 ions below
// 2800 (us a step: 22.1 against 24.4 with 128 at n = 2000, 27.7 and 33.3 at 2600,
// 33.4 and 33.3 at 3000), 128 up to 12160 (us per nb_forces call: 90 against 115
// with 256 at 5003, 257 against 297 at 10000), where 96 blocks would take the
// in-place output, whose chain of commits these short items do not hide (631
// against 485 at 14000), 256 above (4 % faster than 512 at 1e5).  The mixed form's
// lines lie close by, from n = 2000; its FP32 sums run one-sided within a diagonal
// block, so its block (or sub-block, see launch_pair_tri) stays that of make_plan:
// 64 ions below 3000, 128 below 32768, 256 below 60000, 512 above.
Plan make_force_plan(int64_t n, int mode, double soft2) {
  Plan pl = make_plan(n, mode, 0);
  int tb = 0, tr = 0, tbps = 0;
  if (!tri_sums(pl, mode, soft2) || (mode == MODE_MIXED && n < 2000) || tuning_lookup(4, mode, n, &tb, &tr, &tbps)) return pl;
  int G = n > 12160 ? 8 : (n >= 2800 ? 4 : 2);
  if (mode == MODE_MIXED) G = n >= 60000 ? 16 : (n > 12160 ? 8 : (n >= 3000 ? 4 : 2));
  while (G < 32 && (n + 32 * G - 1) / (32 * G) > SYM_MAX_BLOCKS) G *= 2;  // the schedule's block limit
  pl.G = G;
  pl.nbk = (int)((n + 32 * G - 1) / (32 * G));
  // the output rule of the half-pair kernels: in place from 96 blocks or 1 GB of partials
  pl.n_jc = pl.nbk >= 96 || (double)pl.nbk * 3.0 * (double)n * 8.0 > 1e9 ? 1 : pl.nbk;
  return pl;
}

cudaError_t launch_pair_tri(const Plan &pl, int mode, int64_t n, const double *x, const double *y, const double *z,
                            const double *q, double soft2, double *part, unsigned *err, cudaStream_t st) {
  int *sync = part_sync(pl, part, n, 3);
  const bool inplace = pl.n_jc == 1;
  // softened: 8 more lane-cycles per evaluation, kernels of their own so that the
  // others' pair loop has no branch (2 % of it at n = 1e5)
#define NB_TRI(...) launch_tri<__VA_ARGS__>(n, pl.nbk, pl.G, SB, x, y, z, q, soft2, part, sync, err, inplace, st)
  // The mixed form's FP32 sums keep the order they have with make_plan's
  // blocks: one-sided within 128 ions for n < 32768 (whose items of 256 ions
  // from n = 12161 on only change where FP64 sums are added), else within the
  // item.  The fp64 form has no such order to keep; halving its diagonal items
  // this way cost 2 % at n = 1e5 (a second inlined tile step in the branch).
  const int SB = mode == MODE_MIXED && n < 32768 ? std::min(pl.G, 4) : pl.G;
  if (mode == MODE_MIXED) switch (pl.G) {
      case 2: return NB_TRI(true, 1, 64, 12);
      case 4:
      case 8: return NB_TRI(true, 2, 128, 4);
      case 16: return NB_TRI(true, 2, 128, 3);
      case 32: return NB_TRI(true, 2, 256, 2);
      default: return cudaErrorInvalidValue;
    }
  if (soft2 != 0.0) switch (pl.G) {
      case 2: return NB_TRI(false, 1, 64, 10, true);
      case 4:
      case 8: return NB_TRI(false, 2, 128, 4, true);
      case 16:
      case 32: return NB_TRI(false, 2, 256, 2, true);
      default: return cudaErrorInvalidValue;
    }
  switch (pl.G) {
    case 2: return NB_TRI(false, 1, 64, 10);
    case 4:
    case 8: return NB_TRI(false, 2, 128, 4);
    case 16:
    case 32: return NB_TRI(false, 2, 256, 2);
    default: return cudaErrorInvalidValue;
  }
#undef NB_TRI
}

}  // namespace nb
