// nb_vjp.cu -- the pair-force VJP kernels.
//
// For a pair (i, j) with d = r_i - r_j and dl = lam_i - lam_j, the VJP term
//   T = dl r^-3 - 3 (d . dl) r^-5 d
// is formed in double-float on the FP32 pipe in the pair's own units
// (vjp_term) and summed per ion, g_i = sum_j w_j T_ij, in block-floating
// double-float sums widened into FP64 once per 32 partners
// (nb_vjpterm.cuh).  The only per-pair FP64 work is the six differences d and
// dl.  NB_FP64 and NB_DF64 share this arithmetic.
//
// One-sided kernel (k_pair_vjp, small n): the (i-tile, j-chunk) grid of the
// force kernel's plan; each thread owns one ion and sums the chunk's
// partners, staged in shared memory, into one partial per chunk.
//
// Half-pair kernel (k_vjp_sym): T changes sign under i <-> j (both d and dl
// do), so one evaluation serves both ions: g_i += w_j T and g_j -= w_i T.  The
// work is organised as in the force kernel (nb_tri.cu): block pairs (P, Q),
// P <= Q, of BI = 32 G ions, drawn from the round-robin schedule of
// nb_symsched.cuh; a warp owns a P-tile of 64 ions, one packed pair per lane,
// and visits the Q-tiles; positions and cotangents are three FP32 words each on
// the item's grids, one per axis (nb_tri.cuh), so d and dl are exact differences on
// the FP32 pipe, and T and the tile sums are double-floats in packed .f32x2
// instructions, added to FP64 sums after each tile.  What the words cut of
// small components is added in FP64 (vjp_tile_residues).  A tile with a pair too
// close for the words or many cut components, or an item of unusual scales, takes the
// pair's-own-units form of the one-sided kernel (vjp_tile_units), or FP64 where an
// axis is far shorter than the others (vjp_tile_fp64).
//
// What bounds it: the FMA pipe, 234 lane-cycles per evaluation (30 for d, 30 for
// dl, 18 for r^2, 16 for r^-3 and r^-2, 28 for d . dl, 7 for its
// product with 3 r^-2, 48 for T, 48 for the sums, 9 to keep them normalised), 81 %
// busy at n = 32768 with issue at 52 %.  The kernel it replaces formed d and dl
// with six FP64 subtractions per evaluation and scaled every pair's term to
// block-floating sums: 2.83 -> 1.61 ms at n = 20000, 16.6 -> 9.5 ms at 50000, 164
// -> 110 us at 4096 (per nb_forces_vjp call); conditioned error rms 2^-48.5
// against 2^-47.4.
#include <mutex>

#include "nb_symsched.cuh"
#include "nb_tri.cuh"
#include "nb_vjpterm.cuh"

namespace nb {

constexpr int VJP_THREADS = 128;
constexpr int VJP_W = VJP_THREADS / 32;
constexpr double VJP_FAR = 1e18;

// A staged ion: position, weight, cotangent.  The weight is an FP32 (hi, lo)
// pair in w's bits, scaled by its own exponent ew (vjp_weight).
struct __align__(16) VD8 {
  double x, y, z, w, lx, ly, lz;
  int ew, pad;
};

// One pair evaluation: P-ion p against Q-ion q; (ah, al, ea) += w_q T and,
// with BOTH, (bh, bl, eb) -= w_p T.
template <bool W, bool BOTH>
__device__ __forceinline__ void vjp_eval(const VD8 &p, const VD8 &q, double soft2, float ah[3], float al[3],
                                         int &ea, float bh[3], float bl[3], int &eb) {
  float th[3], tl[3];
  const int out = vjp_term(p.x - q.x, p.y - q.y, p.z - q.z, p.lx - q.lx, p.ly - q.ly, p.lz - q.lz, soft2, th, tl);
  if (W) {
    const float2 wq = *reinterpret_cast<const float2 *>(&q.w);
    const float2 wp = *reinterpret_cast<const float2 *>(&p.w);
    float uh[3], ul[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) dfmul(th[c], tl[c], wq.x, wq.y, uh[c], ul[c]);
    bf_acc(ah, al, ea, uh, ul, out + q.ew);
    if (BOTH) {
#pragma unroll
      for (int c = 0; c < 3; ++c) dfmul(th[c], tl[c], -wp.x, -wp.y, uh[c], ul[c]);
      bf_acc(bh, bl, eb, uh, ul, out + p.ew);
    }
  } else {
    bf_acc(ah, al, ea, th, tl, out);
    if (BOTH) {
      float nh[3], nl[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        nh[c] = -th[c];
        nl[c] = -tl[c];
      }
      bf_acc(bh, bl, eb, nh, nl, out);
    }
  }
}

// Staged entry i of a tile (g = global index).  Ions past n are weight-0, lam-0
// dummies far away.
template <bool QARR>
__device__ __forceinline__ void vjp_stage(VD8 *dst, int i, int64_t g, int64_t n, const double *x,
                                          const double *y, const double *z, const double *q,
                                          const double *lx, const double *ly, const double *lz) {
  VD8 e;
  float wh = 0.0f, wl = 0.0f;
  if (g < n) {
    e.x = x[g];
    e.y = y[g];
    e.z = z[g];
    e.lx = lx[g];
    e.ly = ly[g];
    e.lz = lz[g];
    wh = 1.0f;
    e.ew = 0;
    if (QARR) vjp_weight(q[g], wh, wl, e.ew);
  } else {
    e.x = e.y = e.z = VJP_FAR;
    e.lx = e.ly = e.lz = 0.0;
    e.ew = VJP_DEAD;
  }
  *reinterpret_cast<float2 *>(&e.w) = make_float2(wh, wl);
  e.pad = 0;
  dst[i] = e;
}

// ---------------------------------------------------------------------------
// One-sided kernel: part[(jc * 3 + c) * n + i] = sum over the chunk's
// partners j of w_j T_ij (c-th component).
template <bool QARR>
__global__ void __launch_bounds__(256) k_pair_vjp(int64_t n, int64_t jchunk, const double *__restrict__ x,
                                                  const double *__restrict__ y, const double *__restrict__ z,
                                                  const double *__restrict__ q, const double *__restrict__ lx,
                                                  const double *__restrict__ ly, const double *__restrict__ lz,
                                                  double soft2, double *__restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  VD8 *sj = reinterpret_cast<VD8 *>(smem_raw);
  const int B = blockDim.x;
  const int tid = threadIdx.x;
  const int64_t i = (int64_t)blockIdx.x * B + tid;
  const int64_t ic = min(i, n - 1);
  const int64_t jb = (int64_t)blockIdx.y * jchunk;
  const int64_t je = min(jb + jchunk, n);
  VD8 pi;
  pi.x = x[ic];
  pi.y = y[ic];
  pi.z = z[ic];
  pi.lx = lx[ic];
  pi.ly = ly[ic];
  pi.lz = lz[ic];
  pi.w = 0.0;  // the own weight is not used on the one side
  pi.ew = 0;
  pi.pad = 0;
  double g[3] = {0.0, 0.0, 0.0};
  for (int64_t j0 = jb; j0 < je; j0 += B) {
    __syncthreads();
    if (j0 + tid < je) vjp_stage<QARR>(sj, tid, j0 + tid, n, x, y, z, q, lx, ly, lz);
    __syncthreads();
    const int cnt = (int)min((int64_t)B, je - j0);
    for (int k0 = 0; k0 < cnt; k0 += 32) {
      float ah[3] = {0.0f, 0.0f, 0.0f}, al[3] = {0.0f, 0.0f, 0.0f};
      int ea = VJP_BF_EMPTY, eb = VJP_BF_EMPTY;
      const int k1 = min(cnt, k0 + 32);
      for (int k = k0; k < k1; ++k) vjp_eval<QARR, false>(pi, sj[k], soft2, ah, al, ea, nullptr, nullptr, eb);
      double t[3];
      bf_widen(ah, al, ea, t);
#pragma unroll
      for (int c = 0; c < 3; ++c) g[c] += t[c];
    }
  }
  if (i < n) {
#pragma unroll
    for (int c = 0; c < 3; ++c) part[((int64_t)blockIdx.y * 3 + c) * n + i] = g[c];
  }
}

// ---------------------------------------------------------------------------
// Half-pair kernel.

// A staged Q-ion: words 0-2 of the position (with the weight's high and low
// parts in the w of 0 and 1), then of the cotangent; word k of ion e at
// [k * 32 + e].  Stored once: twice (a fixed offset per rotation) would leave
// room for three blocks per SM instead of four.
constexpr int VJP_TILE4 = 6 * 32;

struct VjpIons {  // the lane's two P-ions
  TriIons<1> r, lam;
};

// r^-3 as the double-float (sh, sl) and r^-2 as (w, wl) from r^2 = h + l and the
// seed y: with the residual rho = 1 - (h + l) y^2, r^-3 = y^3 (1 + 3/2 rho + 15/8
// rho^2) and r^-2 = y^2 (1 + rho + rho^2).
__device__ __forceinline__ void vjp_rinv(f32x2 h, f32x2 l, f32x2 y, f32x2 &sh, f32x2 &sl, f32x2 &w, f32x2 &wl) {
  w = pmul(y, y);
  const f32x2 nw = pneg(w);
  const f32x2 e = pfma(y, y, nw);
  const f32x2 rho = psub(pfma(h, nw, pk1(1.0f)), pfma(l, w, pmul(h, e)));
  wl = pfma(w, pfma(rho, rho, rho), e);
  const f32x2 t = pfma(pmul(rho, pk1(1.25f)), rho, rho);
  sh = pmul(w, y);
  const f32x2 low = pfma(e, y, pfma(w, y, pneg(sh)));
  sl = pfma(sh, t, pfma(pmul(sh, pk1(0.5f)), t, low));
  pfast2(sh, sl);
}

// One tile step (tri_tile's conventions; qt: the tile): a += w_q T per P-ion, b
// -= w_p T per Q-ion, T = r^-3 (dl - 3 r^-2 (d . dl) d).  emin: the smallest
// |dl| met (its largest component).
template <bool W, bool ONE, bool SOFT>
__device__ __forceinline__ float vjp_tile(const VjpIons &p, const float4 *qt, int lane, int self, f32x2 s2h,
                                          f32x2 s2l, TriSums<1> &t, float &emin) {
  float ymax = 0.0f, rmin = __int_as_float(0x7f800000);
  emin = rmin;
  const int next = (lane + 1) & 31;
#pragma unroll 1
  for (int r0 = 0; r0 < 32; r0 += 2) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const float4 *qe = qt + ((lane + r0 + s) & 31);
      const float4 q0 = qe[0], q1 = qe[32], q2 = qe[64], u0 = qe[96], u1 = qe[128], u2 = qe[160];
      f32x2 dh[3], dl[3], eh[3], el[3], h, l, sh, sl, wh, wl;
      tri_diff_n(p.r.h[0][0], p.r.m[0][0], p.r.l[0][0], pk1(q0.x), pk1(q1.x), pk1(q2.x), dh[0], dl[0]);
      tri_diff_n(p.r.h[0][1], p.r.m[0][1], p.r.l[0][1], pk1(q0.y), pk1(q1.y), pk1(q2.y), dh[1], dl[1]);
      tri_diff_n(p.r.h[0][2], p.r.m[0][2], p.r.l[0][2], pk1(q0.z), pk1(q1.z), pk1(q2.z), dh[2], dl[2]);
      tri_r2(dh, dl, h, l);
      float ha, hb;
      upk(h, ha, hb);
      const bool me0 = ONE && s == 0 && r0 == 0 && self == 0, me1 = ONE && s == 0 && r0 == 0 && self == 1;
      if (SOFT) {
        rmin = fminf(rmin, fminf(me0 ? rmin : ha, me1 ? rmin : hb));
        f32x2 e;
        ptwo_sum(h, s2h, h, e);
        l = padd(l, padd(e, s2l));
        upk(h, ha, hb);
      }
      float ya = rsqrt_approx(ha), yb = rsqrt_approx(hb);
      if (!SOFT) ymax = fmaxf(ymax, fmaxf(me0 ? 0.0f : ya, me1 ? 0.0f : yb));
      if (ONE) {
        ya = fminf(ya, 0x1p30f);
        yb = fminf(yb, 0x1p30f);
      }
      vjp_rinv(h, l, pk(ya, yb), sh, sl, wh, wl);
      tri_diff_n(p.lam.h[0][0], p.lam.m[0][0], p.lam.l[0][0], pk1(u0.x), pk1(u1.x), pk1(u2.x), eh[0], el[0]);
      tri_diff_n(p.lam.h[0][1], p.lam.m[0][1], p.lam.l[0][1], pk1(u0.y), pk1(u1.y), pk1(u2.y), eh[1], el[1]);
      tri_diff_n(p.lam.h[0][2], p.lam.m[0][2], p.lam.l[0][2], pk1(u0.z), pk1(u1.z), pk1(u2.z), eh[2], el[2]);
      float m0[3], m1[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) upk(eh[c], m0[c], m1[c]);
      const float e0 = fmaxf(fmaxf(fabsf(m0[0]), fabsf(m0[1])), fabsf(m0[2]));
      const float e1 = fmaxf(fmaxf(fabsf(m1[0]), fabsf(m1[1])), fabsf(m1[2]));
      emin = fminf(emin, fminf(me0 ? emin : e0, me1 ? emin : e1));
      // d . dl
      const f32x2 p0 = pmul(dh[0], eh[0]), p1 = pmul(dh[1], eh[1]), p2 = pmul(dh[2], eh[2]);
      f32x2 low = padd(pfma(dh[0], eh[0], pneg(p0)), padd(pfma(dh[1], eh[1], pneg(p1)), pfma(dh[2], eh[2], pneg(p2))));
      f32x2 uh, ul, x1, x2;
      ptwo_sum(p0, p1, uh, x1);
      ptwo_sum(uh, p2, uh, x2);
      low = padd(low, padd(x1, x2));
#pragma unroll
      for (int c = 0; c < 3; ++c) low = pfma(dh[c], el[c], pfma(dl[c], eh[c], low));
      // k = 3 r^-2 (d . dl)
      ptwo_prod(uh, low, wh, wl, uh, ul);
      const f32x2 kh = pmul(pk1(3.0f), uh);
      const f32x2 kl = pfma(pk1(3.0f), ul, pfma(pk1(3.0f), uh, pneg(kh)));
      f32x2 sph = sh, spl = sl, sqh = sh, sql = sl;
      if (W) ptwo_prod(sh, sl, pk1(q0.w), pk1(q1.w), sph, spl);
      if (W && !ONE) ptwo_prod(sh, sl, p.r.wh[0], p.r.wl[0], sqh, sql);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        f32x2 xh, xl, vh, vl, th, tl;
        ptwo_prod(dh[c], dl[c], kh, kl, xh, xl);
        ptwo_diff(eh[c], xh, vh, vl);
        vl = padd(vl, psub(el[c], xl));
        ptwo_prod(vh, vl, sph, spl, th, tl);
        pacc(t.ah[0][c], t.al[0][c], th, tl);
        if (!ONE) {
          if (W) ptwo_prod(vh, vl, sqh, sql, th, tl);
          pacc_sub(t.bh[c], t.bl[c], th, tl);
        }
        if (s == 1) {
          pfast2(t.ah[0][c], t.al[0][c]);
          if (!ONE) pfast2(t.bh[c], t.bl[c]);
        }
      }
      if (!ONE)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          t.bh[c] = pshfl(t.bh[c], next);
          t.bl[c] = pshfl(t.bl[c], next);
        }
    }
  }
  return SOFT ? rsqrt_approx(rmin) : ymax;
}

// The same tile step with each pair in its own units and block-floating sums, as
// in the one-sided kernel: ions i0 .. i0 + 63 against j0 .. j0 + 31.
template <bool QARR>
__device__ __noinline__ void vjp_tile_units(int64_t n, const double *x, const double *y, const double *z,
                                            const double *q, const double *lx, const double *ly, const double *lz,
                                            double soft2, int64_t i0, int64_t j0, bool one, double sc, double *accP,
                                            int ldp, double *accQ, int ldq) {
  const int lane = threadIdx.x & 31;
  for (int u = 0; u < 64; u += 32) {
    VD8 pp;
    vjp_stage<QARR>(&pp, 0, i0 + u + lane, n, x, y, z, q, lx, ly, lz);
    float ah[3] = {0.0f, 0.0f, 0.0f}, al[3] = {0.0f, 0.0f, 0.0f};
    float bh[3] = {0.0f, 0.0f, 0.0f}, bl[3] = {0.0f, 0.0f, 0.0f};
    int ea = VJP_BF_EMPTY, eb = VJP_BF_EMPTY;
    for (int r = 0; r < 32; ++r) {
      const int64_t j = j0 + ((lane + r) & 31);
      VD8 pq;
      vjp_stage<QARR>(&pq, 0, j, n, x, y, z, q, lx, ly, lz);
      if (i0 + u + lane < n && j < n) vjp_eval<QARR, true>(pp, pq, soft2, ah, al, ea, bh, bl, eb);
      for (int c = 0; c < 3; ++c) {
        bh[c] = __shfl_sync(0xffffffffu, bh[c], (lane + 1) & 31);
        bl[c] = __shfl_sync(0xffffffffu, bl[c], (lane + 1) & 31);
      }
      eb = __shfl_sync(0xffffffffu, eb, (lane + 1) & 31);
    }
    double a[3], b[3];
    bf_widen(ah, al, ea, a);
    bf_widen(bh, bl, eb, b);
    for (int c = 0; c < 3; ++c) {
      accP[c * ldp + u + lane] += a[c] * sc;
      if (!one) accQ[c * ldq + lane] += b[c] * sc;
    }
  }
}

// The same in FP64, for the tiles of flat items (vjp_scale): a pair's own units lose
// a component below 2^-74 of its largest.
template <bool QARR>
__device__ __noinline__ void vjp_tile_fp64(int64_t n, const double *x, const double *y, const double *z, const double *q,
                                           const double *lx, const double *ly, const double *lz, double soft2,
                                           int64_t i0, int64_t j0, bool one, double sc, double *accP, int ldp,
                                           double *accQ, int ldq) {
  const int lane = threadIdx.x & 31;
  for (int u = 0; u < 64; u += 32) {
    const int64_t i = i0 + u + lane;
    double a[3] = {0.0, 0.0, 0.0}, b[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
    for (int r = 0; r < 32; ++r) {
      const int64_t j = j0 + ((lane + r) & 31);
      if (i < n && j < n && i != j) {
        const double d[3] = {x[i] - x[j], y[i] - y[j], z[i] - z[j]};
        const double l[3] = {lx[i] - lx[j], ly[i] - ly[j], lz[i] - lz[j]};
        const double s = rinv3_fp64(d[0], d[1], d[2], soft2), v = rinv1_fp64(d[0], d[1], d[2], soft2);
        const double k = 3.0 * (v * v) * fma(d[0], l[0], fma(d[1], l[1], d[2] * l[2]));
        for (int c = 0; c < 3; ++c) {
          const double t = s * fma(-k, d[c], l[c]);
          a[c] += QARR ? t * q[j] : t;
          b[c] -= QARR ? t * q[i] : t;
        }
      }
      for (int c = 0; c < 3; ++c) b[c] = __shfl_sync(0xffffffffu, b[c], (lane + 1) & 31);
    }
    for (int c = 0; c < 3; ++c) {
      accP[c * ldp + u + lane] += a[c] * sc;
      if (!one) accQ[c * ldq + lane] += b[c] * sc;
    }
  }
}

// Cotangents spread more than positions do (a loss that reads a few ions), so their
// rule allows a loss of 2^-44 of a pair's dl: residues are added for the pairs of a
// cut component below 2^-26 and one below 2^-24 of the largest, and in an item
// with a cut component (below 2^-17) a tile with a pair of |dl| below 2^-24 of it
// leaves its words.  A tile with residues in more than 16 of its 64 rotations (each
// costs about as much as four of the pair's-own-units form) leaves them too.
constexpr int VJP_NEAR = 24, VJP_ROT = 16;
constexpr float VJP_EMIN_CUT = 0x1p-24f;

// The same with the cotangents' places from bit 6 (ex: the positions' axes, then the
// cotangents').
struct VjpPlaces {
  const TriPlaces<TRI_NEAR> r;
  const TriPlaces<VJP_NEAR> l;
  __device__ __forceinline__ explicit VjpPlaces(int q) : r(q), l(q >> 6) {}
  __device__ __forceinline__ unsigned rotations(int p) const { return r.rotations(p) | l.rotations(p >> 6); }
};
__device__ __forceinline__ int vjp_places(int64_t n, int64_t g, const double *x, const double *y, const double *z,
                                          const double *lx, const double *ly, const double *lz, const int *ex) {
  return TriPlaces<TRI_NEAR>::of(n, g, x, y, z, ex) | TriPlaces<VJP_NEAR>::of(n, g, lx, ly, lz, ex + 3) << 6;
}
__device__ __noinline__ int vjp_rotations(int64_t n, const double *x, const double *y, const double *z, const double *lx,
                                          const double *ly, const double *lz, int64_t i0, int64_t j0, const int *ex) {
  const int lane = threadIdx.x & 31;
  const VjpPlaces pl(vjp_places(n, j0 + lane, x, y, z, lx, ly, lz, ex));
  int k = 0;
#pragma unroll 1
  for (int u = 0; u < 64; u += 32)
    k += __popc(__reduce_or_sync(0xffffffffu, pl.rotations(vjp_places(n, i0 + u + lane, x, y, z, lx, ly, lz, ex))));
  return k;
}

// What the words of a tile leave out (tri_residues): over the pairs of a cut
// component of a position or cotangent and a near one, r^-3 (de - 3 r^-2 (d . dl) e)
// with e and de what they leave out of d and dl.
template <bool QARR>
__device__ __noinline__ void vjp_tile_residues(int64_t n, const double *x, const double *y, const double *z,
                                               const double *q, const double *lx, const double *ly, const double *lz,
                                               double soft2, int64_t i0, int64_t j0, const int *ex, bool one, double sc,
                                               double *accP, int ldp, double *accQ, int ldq) {
  const int lane = threadIdx.x & 31;
  const VjpPlaces pl(vjp_places(n, j0 + lane, x, y, z, lx, ly, lz, ex));
  const double *const src[6] = {x, y, z, lx, ly, lz};
  double b[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
  for (int u = 0; u < 64; u += 32) {
    const int64_t i = i0 + u + lane;
    const unsigned m = pl.rotations(vjp_places(n, i, x, y, z, lx, ly, lz, ex));
    double a[3] = {0.0, 0.0, 0.0};
    for (unsigned w = __reduce_or_sync(0xffffffffu, m); w; w &= w - 1) {
      const int r = __ffs((int)w) - 1, home = (lane - r) & 31;
      const int64_t j = j0 + ((lane + r) & 31);
      double t[3] = {0.0, 0.0, 0.0};
      if (m >> r & 1) {  // both ions are below n
        double d[6], e[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          d[c] = src[c][i] - src[c][j];
          e[c] = tri_left_out(tri_residue(src[c][i], ex[c]), tri_residue(src[c][j], ex[c]), ex[c]);
        }
        const double s = rinv3_fp64(d[0], d[1], d[2], soft2), v = rinv1_fp64(d[0], d[1], d[2], soft2);
        const double k = 3.0 * (v * v) * fma(d[0], d[3], fma(d[1], d[4], d[2] * d[5]));
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          t[c] = s * fma(-k, e[c], e[c + 3]);
          a[c] += QARR ? t[c] * q[j] : t[c];
          if (QARR) t[c] *= q[i];
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) b[c] -= __shfl_sync(0xffffffffu, t[c], home);
    }
    for (int c = 0; c < 3; ++c) accP[c * ldp + u + lane] += a[c] * sc;
  }
  if (!one)
    for (int c = 0; c < 3; ++c) accQ[c * ldq + lane] += b[c] * sc;
}

// The item's scales: those of the positions and weights (nb_tri.cuh) and the
// largest biased exponents of the cotangents' components; false when the item is
// left to vjp_tile_units (lengths or cotangents beyond 2^+-100 and 2^+-200,
// components of a cotangent more than 2^40 apart, a position or weight scale that
// nb_tri.cuh leaves to FP64).  deep: an axis of the positions or cotangents is
// below 2^-30 of the longest, so that the tiles left to other forms need FP64.
// Ends with a barrier.
template <bool QARR>
__device__ __forceinline__ bool vjp_scale(int64_t p0, int np, int64_t q0, int nq, const double *x, const double *y,
                                          const double *z, const double *q, const double *lx, const double *ly,
                                          const double *lz, double soft2, TriScale &sc, int el[3], bool &deep) {
  __shared__ int red[3][VJP_W];
  int lm[3] = {0, 0, 0};
  auto mag = [](double v) { return __double2hiint(v) & 0x7fffffff; };
  for (int i = threadIdx.x; i < np + nq; i += VJP_THREADS) {
    const int64_t g = i < np ? p0 + i : q0 + (i - np);
    lm[0] = max(lm[0], mag(lx[g]));
    lm[1] = max(lm[1], mag(ly[g]));
    lm[2] = max(lm[2], mag(lz[g]));
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    lm[c] = __reduce_max_sync(0xffffffffu, lm[c]);
    if ((threadIdx.x & 31) == 0) red[c][threadIdx.x >> 5] = lm[c];
  }
  bool ok = tri_scale<VJP_THREADS, QARR>(p0, np, q0, nq, x, y, z, q, soft2, sc);  // holds the barrier
#pragma unroll
  for (int k = 0; k < VJP_W; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) lm[c] = max(lm[c], red[c][k]);
  const int top = max(lm[0], max(lm[1], lm[2])) >> 20;
  deep = false;
  const bool plain = sc.em >= 1023 - 100 && sc.em <= 1023 + 100 && top >= 1023 - 200 && top <= 1023 + 200;
  ok = ok && sc.em >= 1023 - 100 && sc.em <= 1023 + 100 && top <= 1023 + 200;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    deep = deep || (plain && (sc.em - sc.ex[c] > 30 || (lm[c] && top - (lm[c] >> 20) > 30)));
    el[c] = lm[c] ? lm[c] >> 20 : (top ? top : 1023);  // no cotangent at all: any unit
    ok = ok && el[c] >= 1023 - 200 && el[c] >= top - 40;
  }
  return ok;
}

// Largest 1/r of the FP32 path.
constexpr float VJP_YMAX = 0x1p24f;

// The words of ion g's cotangent (zeros past the end) on the components' own
// grids, in the unit of the largest; returns its place there (tri_place), and in
// bit 6 whether a component is cut.
__device__ __forceinline__ int vjp_lam(int64_t g, bool real, const double *lx, const double *ly, const double *lz,
                                       const int el[3], int top, float w0[3], float w1[3], float w2[3]) {
  int place = 0;
  const double *l[3] = {lx, ly, lz};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float t[3] = {0.0f, 0.0f, 0.0f};
    if (real) {
      tri_words(l[c][g], el[c], __int_as_float((127 + el[c] - top) << 23), t);
      place |= tri_place<VJP_NEAR>(l[c][g], el[c], c) | (tri_place<TRI_NEAR>(l[c][g], el[c], 0) & 1) << 6;
    }
    w0[c] = t[0];
    w1[c] = t[1];
    w2[c] = t[2];
  }
  return place;
}

template <bool QARR, bool INPLACE, bool SOFT>
__global__ void __launch_bounds__(VJP_THREADS, 4)
    k_vjp_sym(int64_t n, int nbk, int G, const double *__restrict__ x, const double *__restrict__ y,
              const double *__restrict__ z, const double *__restrict__ q, const double *__restrict__ lx,
              const double *__restrict__ ly, const double *__restrict__ lz, double soft2, double *__restrict__ acc,
              int *__restrict__ sync, unsigned *err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int BI = 32 * G;
  float4 *qs = reinterpret_cast<float4 *>(smem_raw);              // [G][VJP_TILE4]
  double *accQ = reinterpret_cast<double *>(qs + G * VJP_TILE4);  // [3][BI]
  double *accP = accQ + 3 * BI;                                   // [VJP_W][3][64]
  const SymItem it = sym_block_item(INPLACE, sync, nbk);
  const int64_t p0 = (int64_t)it.P * BI, q0 = (int64_t)it.Q * BI;
  const int np = (int)min((int64_t)BI, n - p0), nq = (int)min((int64_t)BI, n - q0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool diag = it.P == it.Q;
  __shared__ int qf[8];  // places of each Q-tile (G <= 8): positions, cotangents from bit 6, bit 12 cut
  __shared__ int ex[6];  // the axes' exponents, for vjp_tile_residues
  TriScale sc;
  int el[3];
  bool deep;
  const bool fast = vjp_scale<QARR>(p0, np, q0, diag ? 0 : nq, x, y, z, q, lx, ly, lz, soft2, sc, el, deep);
  const int ee = max(el[0], max(el[1], el[2]));
  // units: lengths 2^kl, cotangents 2^ke, weights 2^kw; T in 2^(ke - 3 kl + kw)
  const int kt = fast ? (ee - 1022) - 3 * (sc.em - 1022) + (sc.ew - 1023) : 0;
  const int PT = G >> 1, NG = VJP_W / PT, nqt = G / NG;  // P-tiles of 64 ions, warps and Q-tiles per P-tile
  const int pt = warp % PT, grp = warp / PT;
  VjpIons p;
  if (tid == 0)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ex[c] = sc.ex[c];
      ex[3 + c] = el[c];
    }
  int pf = 0;   // places of the warp's P-tile
  int cut = 0;  // a cotangent of the Q side is cut
  if (fast) {
    float w0[2][4], w1[2][4], w2[2][4];
    for (int i = tid; i < BI; i += VJP_THREADS) {
      const int64_t g = q0 + i;
      float4 *e = qs + (i >> 5) * VJP_TILE4 + (i & 31);
      int f = tri_ion<QARR>(g, i < nq, x, y, z, q, sc, -TRI_FAR, w0[0], w1[0], w2[0]);
      e[0] = make_float4(w0[0][0], w0[0][1], w0[0][2], w0[0][3]);
      e[32] = make_float4(w1[0][0], w1[0][1], w1[0][2], w1[0][3]);
      e[64] = make_float4(w2[0][0], w2[0][1], w2[0][2], 0.0f);
      f = __reduce_or_sync(0xffffffffu, f | vjp_lam(g, i < nq, lx, ly, lz, el, ee, w0[0], w1[0], w2[0]) << 6);
      cut |= f >> 12;
      if (lane == 0) qf[i >> 5] = f;
      e[96] = make_float4(w0[0][0], w0[0][1], w0[0][2], 0.0f);
      e[128] = make_float4(w1[0][0], w1[0][1], w1[0][2], 0.0f);
      e[160] = make_float4(w2[0][0], w2[0][1], w2[0][2], 0.0f);
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int i = pt * 64 + b * 32 + lane;
      pf |= tri_ion<QARR>(p0 + i, i < np, x, y, z, q, sc, TRI_FAR, w0[b], w1[b], w2[b]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      p.r.h[0][c] = pk(w0[0][c], w0[1][c]);
      p.r.m[0][c] = pk(w1[0][c], w1[1][c]);
      p.r.l[0][c] = pk(w2[0][c], w2[1][c]);
    }
    p.r.wh[0] = pk(w0[0][3], w0[1][3]);
    p.r.wl[0] = pk(w1[0][3], w1[1][3]);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int i = pt * 64 + b * 32 + lane;
      pf |= vjp_lam(p0 + i, i < np, lx, ly, lz, el, ee, w0[b], w1[b], w2[b]) << 6;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      p.lam.h[0][c] = pk(w0[0][c], w0[1][c]);
      p.lam.m[0][c] = pk(w1[0][c], w1[1][c]);
      p.lam.l[0][c] = pk(w2[0][c], w2[1][c]);
    }
    pf = __reduce_or_sync(0xffffffffu, pf);
  }
  for (int i = tid; i < 3 * BI; i += VJP_THREADS) accQ[i] = 0.0;
  for (int i = tid; i < VJP_W * 3 * 64; i += VJP_THREADS) accP[i] = 0.0;
  const float elim = __syncthreads_or(cut | pf >> 12) ? VJP_EMIN_CUT : 0.0f;
  f32x2 s2h = 0, s2l = 0;
  if (SOFT) {
    float sh, sl;
    split_f64_scaled(soft2, 2 * (sc.em - 1022), sh, sl);
    s2h = pk1(sh);
    s2l = pk1(sl);
  }
  double *aP = accP + warp * 3 * 64;
  const double back = pow2d(-kt), fwd = pow2d(kt);
  const bool live = pt * 64 < np;
  for (int k = 0; k < nqt; ++k) {
    const int t = grp * nqt + (k + pt) % nqt;  // distinct over the P-tiles of a step: nqt >= PT
    if (k > 0) __syncthreads();                // the Q sums of the last step are written
    if (!live || t * 32 >= nq) continue;
    double *aQ = accQ + t * 32;
    bool done = false;
    int rot = 0;  // rotations with residues, where both sides are near on an axis
    if (fast && (tri_fault(pf, qf[t]) || tri_fault(pf >> 6, qf[t] >> 6)))
      rot = vjp_rotations(n, x, y, z, lx, ly, lz, p0 + pt * 64, q0 + t * 32, ex);
    if (fast && rot <= VJP_ROT) {
      TriSums<1> ts;
      const f32x2 zero = pk1(0.0f);
#pragma unroll
      for (int c = 0; c < 3; ++c) ts.ah[0][c] = ts.al[0][c] = ts.bh[c] = ts.bl[c] = zero;
      const float4 *qt = qs + t * VJP_TILE4;
      const int u = t - 2 * pt;  // the lane's own ion in this Q-tile, if any
      float emin;
      const float ymax = diag ? vjp_tile<QARR, true, SOFT>(p, qt, lane, u == 0 || u == 1 ? u : -1, s2h, s2l, ts, emin)
                              : vjp_tile<QARR, false, SOFT>(p, qt, lane, -1, s2h, s2l, ts, emin);
      done = !__any_sync(0xffffffffu, !(ymax <= VJP_YMAX) || !(emin >= elim));
      if (done) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float h0, h1, l0, l1;
          upk(ts.ah[0][c], h0, h1);
          upk(ts.al[0][c], l0, l1);
          aP[c * 64 + lane] += (double)h0 + (double)l0;
          aP[c * 64 + 32 + lane] += (double)h1 + (double)l1;
          if (!diag) {
            upk(ts.bh[c], h0, h1);
            upk(ts.bl[c], l0, l1);
            aQ[c * BI + lane] += ((double)h0 + (double)l0) + ((double)h1 + (double)l1);
          }
        }
        if (rot)
          vjp_tile_residues<QARR>(n, x, y, z, q, lx, ly, lz, soft2, p0 + pt * 64, q0 + t * 32, ex, diag, back, aP, 64,
                                  aQ, BI);
      }
    }
    if (!done) {
      if (deep)
        vjp_tile_fp64<QARR>(n, x, y, z, q, lx, ly, lz, soft2, p0 + pt * 64, q0 + t * 32, diag, back, aP, 64, aQ, BI);
      else
        vjp_tile_units<QARR>(n, x, y, z, q, lx, ly, lz, soft2, p0 + pt * 64, q0 + t * 32, diag, back, aP, 64, aQ, BI);
    }
  }
  __syncthreads();
  sym_output<VJP_THREADS>(INPLACE, it, n, p0, np, q0, nq, acc, sync, err,
                          [&](int c, int i) {
                            double v = 0.0;
                            for (int g = 0; g < NG; ++g) v += accP[(g * PT + i / 64) * 192 + c * 64 + i % 64];
                            return v * fwd;
                          },
                          [&](int c, int i) { return accQ[c * BI + i] * fwd; });
}

static size_t vjp_smem_bytes(int G) {
  return (size_t)G * VJP_TILE4 * sizeof(float4) + (size_t)3 * 32 * G * sizeof(double) +
         (size_t)VJP_W * 3 * 64 * sizeof(double);
}

template <bool SOFT>
static cudaError_t launch_vjp_t(int64_t n, int nbk, int G, const double *x, const double *y,
                                const double *z, const double *q, const double *lx, const double *ly,
                                const double *lz, double soft2, double *part, int *sync, unsigned *err,
                                bool inplace, cudaStream_t st) {
  static std::mutex mu;
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!done[dev]) {
      const int lim = (int)vjp_smem_bytes(8);
      const void *fns[4] = {(const void *)k_vjp_sym<true, false, SOFT>, (const void *)k_vjp_sym<false, false, SOFT>,
                            (const void *)k_vjp_sym<true, true, SOFT>, (const void *)k_vjp_sym<false, true, SOFT>};
      for (int k = 0; k < 4 && e == cudaSuccess; ++k)
        e = cudaFuncSetAttribute(fns[k], cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
      if (e != cudaSuccess) return e;
      done[dev] = true;
    }
  }
  if (inplace) {
    e = cudaMemsetAsync(sync, 0, sizeof(int) * sym_sync_ints(nbk), st);
    if (e != cudaSuccess) return e;
  }
  const unsigned items = (unsigned)sym_items(nbk);
  const size_t smem = vjp_smem_bytes(G);
#define NB_VJP_LAUNCH(QA, IP) \
  k_vjp_sym<QA, IP, SOFT><<<items, VJP_THREADS, smem, st>>>(n, nbk, G, x, y, z, q, lx, ly, lz, soft2, part, sync, err)
  if (inplace) {
    if (q) NB_VJP_LAUNCH(true, true); else NB_VJP_LAUNCH(false, true);
  } else {
    if (q) NB_VJP_LAUNCH(true, false); else NB_VJP_LAUNCH(false, false);
  }
#undef NB_VJP_LAUNCH
  return cudaGetLastError();
}

cudaError_t launch_vjp_sym(int64_t n, int nbk, int G, const double *x, const double *y,
                           const double *z, const double *q, const double *lx, const double *ly,
                           const double *lz, double soft2, double *part, int *sync, unsigned *err,
                           bool inplace, cudaStream_t st) {
  if (G != 4 && G != 8) return cudaErrorInvalidValue;
  return soft2 != 0.0 ? launch_vjp_t<true>(n, nbk, G, x, y, z, q, lx, ly, lz, soft2, part, sync, err, inplace, st)
                      : launch_vjp_t<false>(n, nbk, G, x, y, z, q, lx, ly, lz, soft2, part, sync, err, inplace, st);
}

cudaError_t launch_pair_vjp(const Plan &pl, int64_t n, const double *x, const double *y,
                            const double *z, const double *q, const double *lx,
                            const double *ly, const double *lz, double soft2, double *part,
                            unsigned *err, cudaStream_t st) {
  if (pl.sym)
    return launch_vjp_sym(n, pl.nbk, pl.G, x, y, z, q, lx, ly, lz, soft2, part, part_sync(pl, part, n, 3), err,
                          pl.n_jc == 1, st);
  if (pl.block > 256) return cudaErrorInvalidValue;
  const dim3 grid(pl.n_it, pl.n_jc);
  const size_t smem = sizeof(VD8) * pl.block;
  if (q)
    k_pair_vjp<true><<<grid, pl.block, smem, st>>>(n, pl.jchunk, x, y, z, q, lx, ly, lz, soft2, part);
  else
    k_pair_vjp<false><<<grid, pl.block, smem, st>>>(n, pl.jchunk, x, y, z, q, lx, ly, lz, soft2, part);
  return cudaGetLastError();
}

}  // namespace nb
