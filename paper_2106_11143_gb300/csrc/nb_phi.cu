// nb_phi.cu -- the potential sums phi_i = sum_j w_j / s_ij (the energy's Coulomb
// term and nb_forces' phi) on the FP32 pipe: the half-pair kernel of nb_tri.cu
// with 1/r in place of r^-3 and one sum per ion in place of three.
//
// Both ions of a pair share 1/r, so each pair is evaluated once; the one-sided
// kernel (nb_pair.cu: k_pair_phi, five FP64 instructions per ordered pair) does
// it twice.  What bounds it: the FMA pipe, 68 lane-cycles per evaluation (21 for
// d, 18 for r^2, 10 for 1/r, 16 for the two sums, 3 to keep them normalised; d is left unnormalised, since 1/r needs
// no component), 77 % busy at n = 32768 with issue at 54 %.  An
// nb_energy call at n = 65537 takes 4.81 ms against 41.6, at 4097 92 us against
// 261; relative error of phi rms 5.3e-16 against 1.5e-15 at 65537.  Padding ions'
// terms are 2^-60 of a real one's, below the rounding of any sum.
//
// Output: part[X * n + i], one slot per partner block X, or a single slot with
// the round-ordered adds of nb_symsched.cuh.
#include <algorithm>
#include <mutex>

#include "nb_symsched.cuh"
#include "nb_tri.cuh"

namespace nb {

// 1/r as the double-float (y, sl) from r^2 = h + l and the seed y: with the
// residual rho = 1 - (h + l) y^2, 1/r = y (1 + rho/2 + 3/8 rho^2).
__device__ __forceinline__ void tri_rinv1(f32x2 h, f32x2 l, f32x2 y, f32x2 &sl) {
  const f32x2 w = pmul(y, y);
  const f32x2 e = pfma(y, y, pneg(w));
  const f32x2 rho = psub(pfma(h, pneg(w), pk1(1.0f)), pfma(l, w, pmul(h, e)));
  sl = pmul(pmul(y, pk1(0.5f)), pfma(pmul(rho, pk1(0.75f)), rho, rho));
}

// Half a tile step (tri_tile's conventions): rotations rs .. rs + 15, qt at the
// lane's entry of rotation rs; the sums are ah + al per P-ion and bh + bl per
// Q-ion, those of Q-ion (lane + rs + 16) mod 32 on return.  Halves, because all
// terms are positive: the rounding of a double-float sum of k terms grows with
// k, and with 32 rotations to a sum it passed that of FP64 sums below n = 6000
// (rms 9.7e-16 against 5.4e-16 at n = 1500).
template <int V, bool W, bool ONE, bool SOFT>
__device__ __forceinline__ float phi_tile(const TriIons<V> &p, const float4 *qt, int lane, int self, f32x2 s2h,
                                          f32x2 s2l, f32x2 ah[V], f32x2 al[V], f32x2 &bh, f32x2 &bl) {
  // self: the lane's P-ion that is Q-ion 0 of the first half's rotation itself, or -1
  float ymax = 0.0f, rmin = __int_as_float(0x7f800000);
  const int next = (lane + 1) & 31;
#pragma unroll 1
  for (int r0 = 0; r0 < 16; r0 += 2) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const float4 q0 = qt[r0 + s], q1 = qt[64 + r0 + s], q2 = qt[128 + r0 + s];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        f32x2 dh[3], dl[3], h, l, tl;
        tri_diff(p.h[v][0], p.m[v][0], p.l[v][0], pk1(q0.x), pk1(q1.x), pk1(q2.x), dh[0], dl[0]);
        tri_diff(p.h[v][1], p.m[v][1], p.l[v][1], pk1(q0.y), pk1(q1.y), pk1(q2.y), dh[1], dl[1]);
        tri_diff(p.h[v][2], p.m[v][2], p.l[v][2], pk1(q0.z), pk1(q1.z), pk1(q2.z), dh[2], dl[2]);
        tri_r2(dh, dl, h, l);
        float ha, hb;
        upk(h, ha, hb);
        const bool me0 = ONE && s == 0 && r0 == 0 && self == 2 * v;
        const bool me1 = ONE && s == 0 && r0 == 0 && self == 2 * v + 1;
        if (SOFT) {
          rmin = fminf(rmin, fminf(me0 ? rmin : ha, me1 ? rmin : hb));
          f32x2 e;
          ptwo_sum(h, s2h, h, e);
          l = padd(l, padd(e, s2l));
          upk(h, ha, hb);
        }
        float ya = rsqrt_approx(ha), yb = rsqrt_approx(hb);
        if (ONE) {  // y = 0: no term of the ion itself
          ya = me0 ? 0.0f : ya;
          yb = me1 ? 0.0f : yb;
        }
        if (!SOFT) ymax = fmaxf(ymax, fmaxf(ya, yb));
        f32x2 th = pk(ya, yb);
        tri_rinv1(h, l, th, tl);
        f32x2 uh = th, ul = tl;
        if (W) ptwo_prod(th, tl, pk1(q0.w), pk1(q1.w), uh, ul);
        pacc(ah[v], al[v], uh, ul);
        if (!ONE) {
          uh = th;
          ul = tl;
          if (W) ptwo_prod(th, tl, p.wh[v], p.wl[v], uh, ul);
          pacc(bh, bl, uh, ul);
        }
        if (s == 1) pfast2(ah[v], al[v]);
      }
      if (!ONE) {
        if (V == 2 || s == 1) pfast2(bh, bl);
        bh = pshfl(bh, next);
        bl = pshfl(bl, next);
      }
    }
  }
  return SOFT ? rsqrt_approx(rmin) : ymax;
}

// The same tile step in FP64 from the caller's positions (nb_tri.cuh's limits).
__device__ __noinline__ void phi_tile_fp64(int64_t n, const double *x, const double *y, const double *z,
                                           const double *q, double soft2, int64_t i0, int ni, int64_t j0, int rs,
                                           bool one, double sc, double *accP, double *accQ) {
  const int lane = threadIdx.x & 31;
  for (int u = 0; u < ni; u += 32) {
    const int64_t i = i0 + u + lane;
    double a = 0.0, b = 0.0;
    for (int r = rs; r < rs + 16; ++r) {
      const int64_t j = j0 + ((lane + r) & 31);
      if (i < n && j < n && i != j) {
        const double s = rinv1_fp64(x[i] - x[j], y[i] - y[j], z[i] - z[j], soft2);
        a += q ? s * q[j] : s;
        b += q ? s * q[i] : s;
      }
      b = __shfl_sync(0xffffffffu, b, (lane + 1) & 31);
    }
    accP[u + lane] += a * sc;
    if (!one) accQ[(lane + rs + 16) & 31] += b * sc;
  }
}

template <int V, bool QARR, int NT, int NB, bool INPLACE, bool SOFT>
__global__ void __launch_bounds__(NT, NB)
    k_phi_sym_tri(int64_t n, int nbk, int G, const double *__restrict__ x, const double *__restrict__ y,
                  const double *__restrict__ z, const double *__restrict__ q, double soft2, double *__restrict__ out,
                  int *__restrict__ sync, unsigned *err) {
  constexpr int NW = NT / 32, PI = 64 * V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int BI = 32 * G;
  float4 *qs = reinterpret_cast<float4 *>(smem_raw);              // [G][TRI_TILE4]
  double *accQ = reinterpret_cast<double *>(qs + G * TRI_TILE4);  // [BI]
  double *accP = accQ + BI;                                       // [NW][PI]
  __shared__ int qf[32];                                          // (the force kernel's; 1/r needs no component)
  const SymItem it = sym_block_item(INPLACE, sync, nbk);
  const int64_t p0 = (int64_t)it.P * BI, q0 = (int64_t)it.Q * BI;
  const int np = (int)min((int64_t)BI, n - p0), nq = (int)min((int64_t)BI, n - q0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool diag = it.P == it.Q;
  TriScale sc;
  const bool fast = tri_scale<NT, QARR>(p0, np, q0, diag ? 0 : nq, x, y, z, q, soft2, sc);
  const int kl = fast ? sc.em - 1022 : 0, kw = fast ? sc.ew - 1023 : 0;  // units: L = 2^kl, weights 2^kw
  const int PT = BI / PI, NG = NW / PT, nqt = G / NG;
  const int pt = warp % PT, grp = warp / PT;
  TriIons<V> p;
  bool low = false;
  if (fast) tri_load<V, QARR, NT, TRI_NEAR, true>(p, qs, qf, BI, pt, p0, np, q0, nq, x, y, z, q, sc, low);
  for (int i = tid; i < BI; i += NT) accQ[i] = 0.0;
  for (int i = tid; i < NW * PI; i += NT) accP[i] = 0.0;
  const float ylim = __syncthreads_or(low) ? TRI_YMAX : TRI_YMAX_GRID;
  f32x2 s2h = 0, s2l = 0;
  if (SOFT) {
    float sh, sl;
    split_f64_scaled(soft2, 2 * kl, sh, sl);
    s2h = pk1(sh);
    s2l = pk1(sl);
  }
  double *aP = accP + warp * PI;
  const double back = pow2d(kl - kw), fwd = pow2d(kw - kl);
  const bool live = pt * PI < np;
  for (int k = 0; k < nqt; ++k) {
    const int t = grp * nqt + (k + pt) % nqt;  // distinct over the P-tiles of a step: nqt >= PT
    if (k > 0) __syncthreads();                // the Q sums of the last step are written
    if (!live || t * 32 >= nq) continue;
#pragma unroll 1
    for (int rs = 0; rs < 32; rs += 16) {
      bool done = false;
      if (fast) {
        const f32x2 zero = pk1(0.0f);
        f32x2 ah[V], al[V], bh = zero, bl = zero;
#pragma unroll
        for (int v = 0; v < V; ++v) ah[v] = al[v] = zero;
        const float4 *qt = qs + t * TRI_TILE4 + lane + rs;
        float ymax;
        if (diag) {
          const int u = t - pt * 2 * V;
          ymax = phi_tile<V, QARR, true, SOFT>(p, qt, lane, rs == 0 && u >= 0 && u < 2 * V ? u : -1, s2h, s2l, ah, al,
                                               bh, bl);
        } else {
          ymax = phi_tile<V, QARR, false, SOFT>(p, qt, lane, -1, s2h, s2l, ah, al, bh, bl);
        }
        done = !__any_sync(0xffffffffu, !(ymax <= ylim));
        if (done) {
          float h0, h1, l0, l1;
#pragma unroll
          for (int v = 0; v < V; ++v) {
            upk(ah[v], h0, h1);
            upk(al[v], l0, l1);
            aP[v * 64 + lane] += (double)h0 + (double)l0;
            aP[v * 64 + 32 + lane] += (double)h1 + (double)l1;
          }
          if (!diag) {
            upk(bh, h0, h1);
            upk(bl, l0, l1);
            accQ[t * 32 + ((lane + rs + 16) & 31)] += ((double)h0 + (double)l0) + ((double)h1 + (double)l1);
          }
        }
      }
      if (!done)
        phi_tile_fp64(n, x, y, z, q, soft2, p0 + pt * PI, PI, q0 + t * 32, rs, diag, back, aP, accQ + t * 32);
    }
  }
  __syncthreads();
  auto sumP = [&](int i) {
    double v = 0.0;
    for (int g = 0; g < NG; ++g) v += accP[(g * PT + i / PI) * PI + i % PI];
    return v * fwd;
  };
  if (!INPLACE) {
    for (int i = tid; i < np; i += NT) out[(int64_t)it.Q * n + p0 + i] = sumP(i);
    if (!diag)
      for (int i = tid; i < nq; i += NT) out[(int64_t)it.P * n + q0 + i] = accQ[i] * fwd;
    return;
  }
  // round-ordered adds into one slot, as sym_commit (nb_symsched.cuh) for one sum per ion
  __shared__ int s_ok;
  if (tid == 0) {
    bool ok = true;
    if (it.round > 0) ok = sym_wait(sync, it.P, it.round, err) && (diag || sym_wait(sync, it.Q, it.round, err));
    if (!ok) atomicOr(err, ERR_TIMEOUT);
    s_ok = ok;
  }
  __syncthreads();
  if (s_ok) {
    const bool first = it.round == 0;
#pragma unroll 2
    for (int i = tid; i < BI; i += NT) {
      const bool a = i < np, b = !diag && i < nq;
      const double op = a && !first ? __ldcg(out + p0 + i) : 0.0, oq = b && !first ? __ldcg(out + q0 + i) : 0.0;
      if (a) __stcg(out + p0 + i, first ? sumP(i) : op + sumP(i));
      if (b) __stcg(out + q0 + i, first ? accQ[i] * fwd : oq + accQ[i] * fwd);
    }
  }
  __syncthreads();  // every thread's adds happen before thread 0's release
  if (tid == 0) {
    __threadfence();
    st_release(sync + 1 + it.P, it.round + 1);
    if (!diag) st_release(sync + 1 + it.Q, it.round + 1);
  }
}

template <int V, int NT, int NB, bool SOFT>
static cudaError_t launch_phi_t(int64_t n, int nbk, int G, const double *x, const double *y, const double *z,
                                const double *q, double soft2, double *part, int *sync, unsigned *err, bool inplace,
                                cudaStream_t st) {
  auto smem_of = [](int g) {
    return (size_t)g * TRI_TILE4 * sizeof(float4) + (size_t)32 * g * sizeof(double) +
           (size_t)(NT / 32) * 64 * V * sizeof(double);
  };
  static std::mutex mu;
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!done[dev]) {
      const void *fns[4] = {(const void *)k_phi_sym_tri<V, true, NT, NB, true, SOFT>,
                            (const void *)k_phi_sym_tri<V, false, NT, NB, true, SOFT>,
                            (const void *)k_phi_sym_tri<V, true, NT, NB, false, SOFT>,
                            (const void *)k_phi_sym_tri<V, false, NT, NB, false, SOFT>};
      for (int k = 0; k < 4 && e == cudaSuccess; ++k)
        e = cudaFuncSetAttribute(fns[k], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(16));
      if (e != cudaSuccess) return e;
      done[dev] = true;
    }
  }
  if (inplace) {
    e = cudaMemsetAsync(sync, 0, sizeof(int) * sym_sync_ints(nbk), st);
    if (e != cudaSuccess) return e;
  }
  const unsigned items = (unsigned)sym_items(nbk);
  const size_t smem = smem_of(G);
#define NB_PHI_LAUNCH(QA, IP) \
  k_phi_sym_tri<V, QA, NT, NB, IP, SOFT><<<items, NT, smem, st>>>(n, nbk, G, x, y, z, q, soft2, part, sync, err)
  if (inplace) {
    if (q) NB_PHI_LAUNCH(true, true); else NB_PHI_LAUNCH(false, true);
  } else {
    if (q) NB_PHI_LAUNCH(true, false); else NB_PHI_LAUNCH(false, false);
  }
#undef NB_PHI_LAUNCH
  return cudaGetLastError();
}

// Partials of at most PHI_SLOT_DOUBLES, so that they fit nb_energy_noalloc's
// fixed scratch (its results are those of nb_energy, bit for bit); above, the
// in-place output.
constexpr int64_t PHI_SLOT_DOUBLES = 1000000;
// From n = 2000, where its error is no larger than that of FP64 sums (rms 5.1e-16
// against 5.5e-16 of phi; an nb_energy call takes 75 us against 104).
constexpr int64_t PHI_FROM = 2000;

// Block sizes by measurement (us per nb_energy call): 128 ions below 10000 (92
// against 117 with 256 at n = 4097, 153 against 164 at 8192), 256 above (252
// against 275 with 128 at 12000, 4788 against 4994 with 512 at 65537).
PhiPlan make_phi_plan(int64_t n) {
  PhiPlan pl;
  pl.one = make_plan(n, MODE_FP64, 1);
  pl.n_slots = pl.one.n_jc;
  int tb = 0, tr = 0, tbps = 0;
  if (n < PHI_FROM || tuning_lookup(1, MODE_FP64, n, &tb, &tr, &tbps)) return pl;
  auto blocks = [&](int g) { return (n + 32 * g - 1) / (32 * g); };
  int G = n < 10000 ? 4 : 8;
  if (blocks(G) * n > PHI_SLOT_DOUBLES && blocks(16) * n <= PHI_SLOT_DOUBLES) G = 16;
  while (G < 16 && blocks(G) > SYM_MAX_BLOCKS) G *= 2;
  if (blocks(G) > SYM_MAX_BLOCKS) return pl;
  pl.G = G;
  pl.nbk = (int)blocks(G);
  pl.n_slots = blocks(G) * n > PHI_SLOT_DOUBLES ? 1 : pl.nbk;
  return pl;
}

cudaError_t launch_phi(const PhiPlan &pl, int64_t n, const double *x, const double *y, const double *z,
                       const double *q, double charge, double soft2, double *part, unsigned *err, cudaStream_t st) {
  if (!pl.G) return launch_pair_phi(pl.one, n, x, y, z, q, charge, soft2, part, st);
  int *sync = reinterpret_cast<int *>(part + (size_t)pl.n_slots * (size_t)n);
  const bool inplace = pl.n_slots == 1;
  if (soft2 != 0.0)
    return launch_phi_t<2, 128, 4, true>(n, pl.nbk, pl.G, x, y, z, q, soft2, part, sync, err, inplace, st);
  return launch_phi_t<2, 128, 4, false>(n, pl.nbk, pl.G, x, y, z, q, soft2, part, sync, err, inplace, st);
}

}  // namespace nb
