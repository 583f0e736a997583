// nb_tri.cuh -- FP64-class pair terms (Eq. 1) formed entirely on the FP32
// pipe, from positions carried as three FP32 words on a common grid.
//
// GB300's FP64 pipe retires 2 lanes per clock per SM against 128 on the FP32
// pipe, so even the three FP64 subtractions of a displacement take longer than
// about 100 FP32 instructions.  Here a work item (two sets of ions) picks for
// each axis a power of two L_c above every coordinate of that axis it touches
// and cuts the coordinates' bits, in units of L_c, into
//   h: a multiple of 2^-22,  m: a multiple of 2^-45 below 2^-22,
//   l: a multiple of 2^-69 below 2^-45   (all with the coordinate's sign),
// which are then put in units of L = max L_c, an exact scaling.  The words'
// differences are exact in FP32, so d = dh + dm + dl is exact, and two Fast2Sums
// make it a double-float (RN(d), rest), whatever words it starts in: 10 FP32
// operations per component, all of which exist as packed .f32x2 instructions.
// Each component is right to 2^-48 of itself, as an FP64 difference is right to
// 2^-53 of itself, which the transverse forces of a thin chain need: its y may be
// 2^-40 of its z.  One unit for the three axes left y with its bits above 2^-69
// of the largest z, and an unnormalised (dh + dm, dl) with FP32 accuracy where
// dh and dm cancel.
//
// A coordinate of at least 2^-17 L_c is exact in its words, a smaller one if it
// has no bits below 2^-68 L_c (grids, zeros); else it is cut.  Against a partner
// of 2^-15 L_c or more a cut one is right to 2^-52 of the difference; for a pair of
// a cut one and one below 2^-15 L_c of the same axis, the force of what the words
// leave out of d is added in FP64 (tri_residues; one tile of 128 x 32 ions in 3000 of a
// random cloud has such a pair), and a tile where that would be more than half its
// rotations is done in FP64 as a whole.  Doing every such tile in FP64 took longer
// than the kernel's other tiles together below n = 5000: 62.3 against 55.7 us a step
// at n = 4096.
//
// What is left for FP32's range: pairs closer than 2^-40 L send their tile to
// FP64 too (the smallest r^2 met, one FMNMX per pair), and items whose scale,
// flatness or weights are far from the ordinary (below) take the FP64 path as a
// whole.
#pragma once

#include "nb_common.cuh"

namespace nb {

// Packed FP32 pairs (.f32x2): the same IEEE operation on both halves in one
// issue slot and two cycles of the FMA pipe.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f32x2 pk1(float v) { return pk(v, v); }
__device__ __forceinline__ void upk(f32x2 v, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 padd(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 psub(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 pmul(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 pfma(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 pneg(f32x2 v) {
  float a, b;
  upk(v, a, b);
  return pk(-a, -b);
}

// s + e = a + b and a - b exactly (Knuth TwoSum).
__device__ __forceinline__ void ptwo_sum(f32x2 a, f32x2 b, f32x2 &s, f32x2 &e) {
  s = padd(a, b);
  const f32x2 bb = psub(s, a);
  e = padd(psub(a, psub(s, bb)), psub(b, bb));
}
__device__ __forceinline__ void ptwo_diff(f32x2 a, f32x2 b, f32x2 &s, f32x2 &e) {
  s = psub(a, b);
  const f32x2 bb = psub(s, a);  // about -b
  e = psub(psub(a, psub(s, bb)), padd(b, bb));
}

// The words of coordinate x in units of 2^(em - 1022), em at least x's biased
// exponent, times f: w[0] + w[1] + w[2] = f x / 2^(em - 1022) to 2^-69 f.
__device__ __forceinline__ void tri_words(double x, int em, float f, float w[3]) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const unsigned t1 = e ? (0x80000000u | ((hi & 0xfffffu) << 11) | (lo >> 21)) : 0u, t0 = e ? lo << 11 : 0u;
  const int s = em - e, k = s & 31, j = s >> 5;  // the mantissa (t1:t0) moves down s bits
  const unsigned a0 = t1 >> k, a1 = __funnelshift_r(t0, t1, k), a2 = __funnelshift_r(0u, t0, k);
  const unsigned w0 = j == 0 ? a0 : 0u;
  const unsigned w1 = j == 0 ? a1 : (j == 1 ? a0 : 0u);
  const unsigned w2 = j == 0 ? a2 : (j == 1 ? a1 : (j == 2 ? a0 : 0u));
  const float sg = __uint_as_float(__float_as_uint(f) | (hi & 0x80000000u));
  w[0] = (float)(int)(w0 >> 10) * (sg * 0x1p-22f);
  w[1] = (float)(int)(((w0 & 0x3ffu) << 13) | (w1 >> 19)) * (sg * 0x1p-45f);
  w[2] = (float)(int)(((w1 & 0x7ffffu) << 5) | (w2 >> 27)) * (sg * 0x1p-69f);
}

// A coordinate's place on its axis's grid: bit 0, cut (it has bits below 2^-68,
// counted so that the difference of two uncut ones fits the words' 24 bits also
// where their signs differ, and is below 2^(-2 - NEAR)); bit 3, near the origin
// (below 2^-NEAR).  Shifted by the axis, 0 .. 2.
constexpr int TRI_NEAR = 15;      // a cut coordinate is right to 2^-52 of a difference
constexpr int TRI_NEAR_MIX = 38;  // .. to 2^-29, for FP32 displacements
template <int NEAR>
__device__ __forceinline__ int tri_place(double x, int em, int c) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ffu), s = em - e;
  if (s < NEAR) return 0;
  const int tz = lo ? __ffs((int)lo) - 1 : 31 + __ffs((int)((hi & 0xfffffu) | 0x100000u));
  const bool cut = s >= NEAR + 2 && ((hi << 1) | lo) != 0 && (e == 0 || tz < s - 15);
  return (cut ? 1 << c : 0) | (8 << c);
}
// Whether a pair of the two sides (OR of their ions' places) may lose bits.
__device__ __forceinline__ bool tri_fault(int p, int q) {
  return (((p >> 3) & q) | (p & (q >> 3))) & 7;
}

// A padding ion's coordinate, in units of L: far enough that every term with
// it underflows to zero (y^3 < 2^-149), near enough that r^2 stays finite.  The
// two sides use opposite signs, so two padding ions never coincide.
constexpr float TRI_FAR = 1e18f;

// Largest 1/r (units of 1/L) of the FP32 path: y^3 and its products stay in range.
constexpr float TRI_YMAX_GRID = 0x1p40f;
// The same where the displacement is left unnormalised (nb_phi.cu) and an l word
// is set or a coordinate cut.
constexpr float TRI_YMAX = 0x1p20f;

// Scales the path accepts: L within 2^+-150 (so that L^2, L^-2 and their products
// with any force the FP64 path can form stay inside FP64), weights within 2^40 of
// the item's largest (so that a double-float weight keeps its 48 bits), and an axis
// at least 2^-64 of the longest: its words are exact down to FP32's 2^-149, and the
// products' and sums' roundings there, 2^-149 each, are below 2^-57 of the terms its
// largest coordinate has with far partners (less 16 with weights, less 24 with a
// softening beyond L, by what these take off the terms).
constexpr int TRI_EMIN = 1023 - 150, TRI_EMAX = 1023 + 150, TRI_FLAT = 64, TRI_WSPREAD = 40;
// and a softening length up to 2^10 L (far above it the terms' low parts would
// leave FP32's range).
__device__ __forceinline__ bool tri_scale_ok(int em, double soft2) {
  return em >= TRI_EMIN && em <= TRI_EMAX && ((__double2hiint(soft2) >> 20) & 0x7ff) - 2 * (em - 1022) <= 1023 + 20;
}

// An item's scale: biased exponents of L and of the axes' L_c, and of the weights.
struct TriScale {
  int em, ex[3], ew;
  __device__ __forceinline__ float f(int c) const { return __int_as_float((127 + ex[c] - em) << 23); }
};
// From the largest high words of the coordinates of each axis; false: FP64.
template <bool QARR>
__device__ __forceinline__ bool tri_axes(const int mx[3], double soft2, TriScale &s) {
  s.em = max(mx[0], max(mx[1], mx[2])) >> 20;
  bool ok = tri_scale_ok(s.em, soft2);
  const int flat = TRI_FLAT - (QARR ? 16 : 0) - ((__double2hiint(soft2) >> 20) - 2 * (s.em - 1022) > 1023 ? 24 : 0);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    s.ex[c] = mx[c] ? mx[c] >> 20 : s.em;  // an axis of zeros: any unit
    ok = ok && s.em - s.ex[c] <= flat;
  }
  return ok;
}

// s + e = a + b exactly for |a| >= |b|, or a a multiple of ulp(s) (Fast2Sum).
__device__ __forceinline__ void pfast2(f32x2 &a, f32x2 &b) {
  const f32x2 s = padd(a, b);
  b = psub(b, psub(s, a));
  a = s;
}

// d = p - q as an unnormalised double-float: the word differences are exact, and
// so is the Fast2Sum of dh and dm: |dm| may reach 2^-21 (signs that differ), but
// dh is 0 or a multiple of 2^-22 and thus of the sum's last place.
__device__ __forceinline__ void tri_diff(f32x2 ph, f32x2 pm, f32x2 pl, f32x2 qh, f32x2 qm, f32x2 ql, f32x2 &h,
                                         f32x2 &l) {
  const f32x2 dh = psub(ph, qh), dm = psub(pm, qm), dl = psub(pl, ql);
  h = padd(dh, dm);
  l = padd(psub(dm, psub(h, dh)), dl);
}
// The same with h = RN(d): where dh and dm cancel, the leading bits of d stand in
// l, and a product with (h, l) would keep only 24 of them.
__device__ __forceinline__ void tri_diff_n(f32x2 ph, f32x2 pm, f32x2 pl, f32x2 qh, f32x2 qm, f32x2 ql, f32x2 &h,
                                           f32x2 &l) {
  tri_diff(ph, pm, pl, qh, qm, ql, h, l);
  pfast2(h, l);
}

// r^2 of the double-float displacement (dh, dl) as the double-float (h, l).
// The largest component's square comes first, so every partial sum a + b^2
// has a >= b^2 and its rounding error is one exact difference and one FMA
// (FMNMX runs on the ALU pipe, which the pair loop leaves idle).  The
// dl^2 terms are there against a bias: without them r^2 is short by 2^-50.
__device__ __forceinline__ void tri_r2(const f32x2 dh[3], const f32x2 dl[3], f32x2 &h, f32x2 &l) {
  float x[2], y[2], z[2], M[2], m1[2], m2[2];
  upk(dh[0], x[0], x[1]);
  upk(dh[1], y[0], y[1]);
  upk(dh[2], z[0], z[1]);
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const float t = fmaxf(fabsf(x[b]), fabsf(y[b]));
    m1[b] = fminf(fabsf(x[b]), fabsf(y[b]));
    M[b] = fmaxf(t, fabsf(z[b]));
    m2[b] = fminf(t, fabsf(z[b]));
  }
  const f32x2 A = pk(M[0], M[1]), B = pk(m1[0], m1[1]), C = pk(m2[0], m2[1]);
  const f32x2 p = pmul(A, A);
  const f32x2 e0 = pfma(A, A, pneg(p));
  const f32x2 h1 = pfma(B, B, p);
  const f32x2 t1 = pfma(B, B, psub(p, h1));
  h = pfma(C, C, h1);
  const f32x2 t2 = pfma(C, C, psub(h1, h));
  const f32x2 q = pfma(dh[2], dl[2], pfma(dh[1], dl[1], pmul(dh[0], dl[0])));
  const f32x2 d2 = pfma(dl[2], dl[2], pfma(dl[1], dl[1], pmul(dl[0], dl[0])));
  l = pfma(pk1(2.0f), q, padd(padd(e0, t1), padd(t2, d2)));
}

// r^-3 as the double-float (sh, sl) from r^2 = h + l and the seed y of
// 1/sqrt(h) (relative error below 2^-22.9).  With w = RN(y^2) and e = y^2 - w
// exactly, the residual is rho = 1 - (h + l) w (its first FMA is all but
// exact) and
//   r^-3 = w^(3/2) (1 - rho)^(-3/2),  w^(1/2) = y (1 - e / (2 y^2)) to e^2,
// so that r^-3 = (w y - y e / 2) (1 + 3/2 t), t = rho + 5/4 rho^2, with w y kept
// as a double-float.  3/2 t goes in as t + t/2 (a product 1.5 t would round
// once more), and (sh, sl) is left normalised, so that the products with it
// lose nothing to a long sl.
__device__ __forceinline__ void tri_rinv3(f32x2 h, f32x2 l, f32x2 y, f32x2 &sh, f32x2 &sl) {
  const f32x2 w = pmul(y, y), nw = pneg(w);
  const f32x2 e = pfma(y, y, nw);
  const f32x2 rho = pfma(l, nw, pfma(h, nw, pk1(1.0f)));
  const f32x2 t = pfma(pmul(rho, pk1(1.25f)), rho, rho);
  sh = pmul(w, y);
  f32x2 low = pfma(e, pmul(y, pk1(-0.5f)), pfma(w, y, pneg(sh)));
  low = pfma(pmul(low, pk1(1.5f)), rho, low);
  sl = pfma(sh, t, pfma(pmul(sh, pk1(0.5f)), t, low));
  pfast2(sh, sl);
}

// (h, l) = (ah + al) (bh + bl) as a double-float.
__device__ __forceinline__ void ptwo_prod(f32x2 ah, f32x2 al, f32x2 bh, f32x2 bl, f32x2 &h, f32x2 &l) {
  h = pmul(ah, bh);
  l = pfma(ah, bl, pfma(al, bh, pfma(ah, bh, pneg(h))));
}

// Double-float sums: (h, l) += (th, tl) and -= (th, tl).
__device__ __forceinline__ void pacc(f32x2 &h, f32x2 &l, f32x2 th, f32x2 tl) {
  f32x2 s, e;
  ptwo_sum(h, th, s, e);
  h = s;
  l = padd(l, padd(e, tl));
}
__device__ __forceinline__ void pacc_sub(f32x2 &h, f32x2 &l, f32x2 th, f32x2 tl) {
  f32x2 s, e;
  ptwo_diff(h, th, s, e);
  h = s;
  l = padd(l, psub(e, tl));
}

__device__ __forceinline__ f32x2 pshfl(f32x2 v, int lane) {
  float a, b;
  upk(v, a, b);
  return pk(__shfl_sync(0xffffffffu, a, lane), __shfl_sync(0xffffffffu, b, lane));
}

__device__ __forceinline__ float rsqrt_approx(float v) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(v));
  return y;
}

// 2^k as FP64 (|k| <= 1000).
__device__ __forceinline__ double pow2d(int k) { return __hiloint2double((1023 + k) << 20, 0); }

template <int V>
struct TriIons {  // 2 V ions of a lane: words and, with weights, the weight's (hi, lo)
  f32x2 h[V][3], m[V][3], l[V][3], wh[V], wl[V];
};

// The sums of a tile step: double-floats, or FP32 (MIX) in the high words.
template <int V>
struct TriSums {
  f32x2 ah[V][3], al[V][3], bh[3], bl[3];
};

// One tile step: this lane's P-ions against the 32 Q-ions of a tile;
// ld(r, q0, q1, q2) loads the three words (with the weight's parts in the w of
// q0 and q1) of Q-ion (lane + r) mod 32.  Returns the largest 1/r met
// (with a softening, of the distance without it).  self: the lane's P-ion (0 ..
// 2 V - 1) that is Q-ion 0 of the rotation itself, or -1 (ONE only).  SOFT: the
// softening soft2 L^-2 as the double-float (s2h, s2l).
template <int V, bool W, bool ONE, bool SOFT, class LD>
__device__ __forceinline__ float tri_tile(const TriIons<V> &p, LD ld, int lane, int self, f32x2 s2h, f32x2 s2l,
                                          TriSums<V> &t) {
  f32x2(&ah)[V][3] = t.ah, (&al)[V][3] = t.al, (&bh)[3] = t.bh, (&bl)[3] = t.bl;
  float ymax = 0.0f, rmin = __int_as_float(0x7f800000);
  const int next = (lane + 1) & 31;
#pragma unroll 1
  for (int r0 = 0; r0 < 32; r0 += 2) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      float4 q0, q1, q2;
      ld(r0 + s, q0, q1, q2);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        f32x2 dh[3], dl[3], h, l, sh, sl;
        tri_diff_n(p.h[v][0], p.m[v][0], p.l[v][0], pk1(q0.x), pk1(q1.x), pk1(q2.x), dh[0], dl[0]);
        tri_diff_n(p.h[v][1], p.m[v][1], p.l[v][1], pk1(q0.y), pk1(q1.y), pk1(q2.y), dh[1], dl[1]);
        tri_diff_n(p.h[v][2], p.m[v][2], p.l[v][2], pk1(q0.z), pk1(q1.z), pk1(q2.z), dh[2], dl[2]);
        tri_r2(dh, dl, h, l);
        float ha, hb;
        upk(h, ha, hb);
        // the ion itself is left out: its d = 0 gives a zero term with any finite y
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
        if (!SOFT) ymax = fmaxf(ymax, fmaxf(me0 ? 0.0f : ya, me1 ? 0.0f : yb));
        if (ONE) {
          ya = fminf(ya, TRI_YMAX_GRID);
          yb = fminf(yb, TRI_YMAX_GRID);
        }
        tri_rinv3(h, l, pk(ya, yb), sh, sl);
        f32x2 sph = sh, spl = sl, sqh = sh, sql = sl;
        if (W) ptwo_prod(sh, sl, pk1(q0.w), pk1(q1.w), sph, spl);
        if (W && !ONE) ptwo_prod(sh, sl, p.wh[v], p.wl[v], sqh, sql);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          f32x2 th, tl;
          ptwo_prod(dh[c], dl[c], sph, spl, th, tl);
          pacc(ah[v][c], al[v][c], th, tl);
          if (!ONE) {
            if (W) ptwo_prod(dh[c], dl[c], sqh, sql, th, tl);
            pacc_sub(bh[c], bl[c], th, tl);
          }
          // the low sums stay at an ulp of the high ones, so that adding to
          // them rounds at 2^-49 of the sum
          if (s == 1) pfast2(ah[v][c], al[v][c]);
        }
      }
      if (!ONE)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          if (V == 2 || s == 1) pfast2(bh[c], bl[c]);
          bh[c] = pshfl(bh[c], next);
          bl[c] = pshfl(bl[c], next);
        }
    }
  }
  return SOFT ? rsqrt_approx(rmin) : ymax;
}

// Words of ion g (or a padding ion on side `far`) with its weight; returns its place
// (without CUT the bits of the axes it is near on alone: no branches).
template <bool QARR, int NEAR = TRI_NEAR, bool CUT = true>
__device__ __forceinline__ int tri_ion(int64_t g, bool real, const double *x, const double *y, const double *z,
                                       const double *q, const TriScale &sc, float far, float w0[4], float w1[4],
                                       float w2[4]) {
  w0[3] = w1[3] = w2[3] = 0.0f;
  int place = 0;
  if (real) {
    const double r[3] = {x[g], y[g], z[g]};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float t[3];
      tri_words(r[c], sc.ex[c], sc.f(c), t);
      w0[c] = t[0];
      w1[c] = t[1];
      w2[c] = t[2];
      if (CUT)
        place |= tri_place<NEAR>(r[c], sc.ex[c], c);
      else
        place |= sc.ex[c] - ((__double2hiint(r[c]) >> 20) & 0x7ff) >= NEAR ? 8 << c : 0;
    }
    if (QARR && q[g] != 0.0) split_f64_scaled(q[g], sc.ew - 1023, w0[3], w1[3]);
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      w0[c] = far;
      w1[c] = w2[c] = 0.0f;
    }
  }
  return place;
}

// A staged tile: word k of entry e (64 entries, the tile twice) at
// [k * 64 + e], the weight's high and low parts in the w of words 0 and 1.
constexpr int TRI_TILE4 = 3 * 64;

// The item's scale over ions [p0, p0 + np) and [q0, q0 + nq); false when the item is
// left to FP64.  Ends with a barrier.
template <int NT, bool QARR>
__device__ __forceinline__ bool tri_scale(int64_t p0, int np, int64_t q0, int nq, const double *x, const double *y,
                                          const double *z, const double *q, double soft2, TriScale &sc) {
  __shared__ int red[5][NT / 32];
  int mx[3] = {0, 0, 0}, wx = 0, wn = 0x7fffffff;
  for (int i = threadIdx.x; i < np + nq; i += NT) {
    const int64_t g = i < np ? p0 + i : q0 + (i - np);
    mx[0] = max(mx[0], __double2hiint(x[g]) & 0x7fffffff);
    mx[1] = max(mx[1], __double2hiint(y[g]) & 0x7fffffff);
    mx[2] = max(mx[2], __double2hiint(z[g]) & 0x7fffffff);
    if (QARR) {
      const int w = __double2hiint(q[g]) & 0x7fffffff;
      wx = max(wx, w);
      if (q[g] != 0.0) wn = min(wn, w);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) mx[c] = __reduce_max_sync(0xffffffffu, mx[c]);
  if (QARR) {
    wx = __reduce_max_sync(0xffffffffu, wx);
    wn = __reduce_min_sync(0xffffffffu, wn);
  }
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int c = 0; c < 3; ++c) red[c][w] = mx[c];
    red[3][w] = wx;
    red[4][w] = wn;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NT / 32; ++k) {
#pragma unroll
    for (int c = 0; c < 3; ++c) mx[c] = max(mx[c], red[c][k]);
    wx = max(wx, red[3][k]);
    wn = min(wn, red[4][k]);
  }
  bool ok = tri_axes<QARR>(mx, soft2, sc);
  sc.ew = 1023;
  if (QARR) {
    sc.ew = wx >> 20;
    ok = ok && sc.ew >= 1023 - 400 && sc.ew <= 1023 + 400 && sc.ew - (wn >> 20) <= TRI_WSPREAD;
  }
  return ok;
}

// Cuts the Q block's ions into words in shared memory (BI entries), with the OR of
// each tile's places in qf, and loads the lane's ions of P-tile pt; returns the
// OR of that tile's places (CUT as in tri_ion).  low, with CUT: an l word is set or
// a coordinate cut.
template <int V, bool QARR, int NT, int NEAR, bool CUT>
__device__ __forceinline__ int tri_load(TriIons<V> &p, float4 *qs, int *qf, int BI, int pt, int64_t p0, int np,
                                        int64_t q0, int nq, const double *x, const double *y, const double *z,
                                        const double *q, const TriScale &sc, bool &low) {
  const int lane = threadIdx.x & 31;
  low = false;
  for (int i = threadIdx.x; i < BI; i += NT) {  // a warp takes a tile
    float w0[4], w1[4], w2[4];
    const int f = tri_ion<QARR, NEAR, CUT>(q0 + i, i < nq, x, y, z, q, sc, -TRI_FAR, w0, w1, w2);
    float4 *e = qs + (i >> 5) * TRI_TILE4 + (i & 31);
    e[0] = e[32] = make_float4(w0[0], w0[1], w0[2], w0[3]);
    e[64] = e[96] = make_float4(w1[0], w1[1], w1[2], w1[3]);
    e[128] = e[160] = make_float4(w2[0], w2[1], w2[2], w2[3]);
    low |= w2[0] != 0.0f || w2[1] != 0.0f || w2[2] != 0.0f || (f & 7);
    const int tf = __reduce_or_sync(0xffffffffu, f);
    if (lane == 0) qf[i >> 5] = tf;
  }
  int pf = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    float w0[2][4], w1[2][4], w2[2][4];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int i = pt * 64 * V + v * 64 + b * 32 + lane;
      pf |= tri_ion<QARR, NEAR, CUT>(p0 + i, i < np, x, y, z, q, sc, TRI_FAR, w0[b], w1[b], w2[b]);
      low |= w2[b][0] != 0.0f || w2[b][1] != 0.0f || w2[b][2] != 0.0f;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      p.h[v][c] = pk(w0[0][c], w0[1][c]);
      p.m[v][c] = pk(w1[0][c], w1[1][c]);
      p.l[v][c] = pk(w2[0][c], w2[1][c]);
    }
    p.wh[v] = pk(w0[0][3], w0[1][3]);
    p.wl[v] = pk(w1[0][3], w1[1][3]);
  }
  low |= pf & 7;
  return __reduce_or_sync(0xffffffffu, pf);
}

// The part of coordinate x below its words' last place, and its l word in units of
// that place.
struct TriRest {
  double e = 0.0;
  int l = 0;
};
__device__ __forceinline__ TriRest tri_residue(double x, int em) {
  TriRest t;
  const long long b = __double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff, s = em - e;
  if (e == 0 || s >= 69) {
    t.e = x;
    return t;
  }
  const long long m = (b & 0xfffffffffffffll) | 1ll << 52;
  if (s > 16) t.e = x - __longlong_as_double(b & (long long)(~0ull << (s - 16)));
  t.l = (int)(s > 16 ? m >> (s - 16) : m << (16 - s)) & 0xffffff;
  if (b < 0) t.l = -t.l;
  return t;
}
// What the words leave out of p - q: the residues' difference, and the last bit of a
// difference of l words of unlike sign, which has 25 (at 2^-42 L, the pairs' smallest
// components that lead a sum, 2^-27 of it).
__device__ __forceinline__ double tri_left_out(const TriRest &p, const TriRest &q, int em) {
  const int l = p.l - q.l;
  return p.e - q.e + (l - (int)(float)l) * pow2d(em - 1022 - 69);
}

// The pairs of a cut coordinate and a near one in a tile: ions [i0, i0 + ni) against
// [j0, j0 + 32), those below n; ex: the axes' exponents.  TriPlaces holds the Q
// side's places; rotations() gives, for the lane's ion i0 + u + lane, bit r for such a
// pair with Q-ion (lane + r) mod 32.
template <int NEAR>
struct TriPlaces {
  unsigned cut[3], near[3];
  __device__ __forceinline__ static int of(int64_t n, int64_t g, const double *x, const double *y, const double *z,
                                           const int *ex) {
    return g < n ? tri_place<NEAR>(x[g], ex[0], 0) | tri_place<NEAR>(y[g], ex[1], 1) | tri_place<NEAR>(z[g], ex[2], 2) : 0;
  }
  __device__ __forceinline__ TriPlaces(int q) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      cut[c] = __ballot_sync(0xffffffffu, q >> c & 1);
      near[c] = __ballot_sync(0xffffffffu, q >> (3 + c) & 1);
    }
  }
  __device__ __forceinline__ unsigned rotations(int p) const {
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) m |= (p >> (3 + c) & 1 ? cut[c] : 0u) | (p >> c & 1 ? near[c] : 0u);
    return __funnelshift_r(m, m, threadIdx.x & 31);
  }
};

// How many of the tile's ni rotations (32 for every 32 ions of the P side) hold such
// pairs.
template <int NEAR>
__device__ __noinline__ int tri_rotations(int64_t n, const double *x, const double *y, const double *z, int64_t i0,
                                          int ni, int64_t j0, const int *ex) {
  const int lane = threadIdx.x & 31;
  const TriPlaces<NEAR> pl(TriPlaces<NEAR>::of(n, j0 + lane, x, y, z, ex));
  int k = 0;
#pragma unroll 1
  for (int u = 0; u < ni; u += 32)
    k += __popc(__reduce_or_sync(0xffffffffu, pl.rotations(TriPlaces<NEAR>::of(n, i0 + u + lane, x, y, z, ex))));
  return k;
}

// What the words leave out of the tile's sums: over these pairs, with e what they leave
// out of d, r^-3 (e - 3 r^-2 (d . e) (d - e)); what remains is below 2^-54 of each
// component at the closest pairs the words serve.  addP(u, c, v) takes what falls to
// ion i0 + u + lane; b: the lane's Q-ion's sums.  Rotations without such pairs are
// skipped, and the Q side's terms go home by shuffle.
template <bool QARR, int NEAR, class ADD>
__device__ __forceinline__ void tri_residues(int64_t n, const double *x, const double *y, const double *z,
                                             const double *q, double soft2, int64_t i0, int ni, int64_t j0,
                                             const int *ex, double b[3], ADD addP) {
  const int lane = threadIdx.x & 31;
  const TriPlaces<NEAR> pl(TriPlaces<NEAR>::of(n, j0 + lane, x, y, z, ex));
  auto load = [&](int64_t g, double r[3], TriRest e[3], double &w) {
    r[0] = r[1] = r[2] = w = 0.0;
    if (g >= n) return;
    r[0] = x[g];
    r[1] = y[g];
    r[2] = z[g];
    if (QARR) w = q[g];
#pragma unroll
    for (int c = 0; c < 3; ++c) e[c] = tri_residue(r[c], ex[c]);
  };
  double xq[3], wq;
  TriRest eq[3];
  load(j0 + lane, xq, eq, wq);
  b[0] = b[1] = b[2] = 0.0;
#pragma unroll 1
  for (int u = 0; u < ni; u += 32) {
    const unsigned m = pl.rotations(TriPlaces<NEAR>::of(n, i0 + u + lane, x, y, z, ex));
    double a[3] = {0.0, 0.0, 0.0};
    unsigned w = __reduce_or_sync(0xffffffffu, m);
    if (w) {
      double xp[3], wp;
      TriRest ep[3];
      load(i0 + u + lane, xp, ep, wp);
      for (; w; w &= w - 1) {
        const int r = __ffs((int)w) - 1, from = (lane + r) & 31, home = (lane - r) & 31;
        double d[3], de[3], s = 0.0, k = 0.0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          d[c] = xp[c] - __shfl_sync(0xffffffffu, xq[c], from);
          TriRest t;
          t.e = __shfl_sync(0xffffffffu, eq[c].e, from);
          t.l = __shfl_sync(0xffffffffu, eq[c].l, from);
          de[c] = tri_left_out(ep[c], t, ex[c]);
        }
        const double wj = QARR ? __shfl_sync(0xffffffffu, wq, from) : 1.0;
        if (m >> r & 1) {
          s = rinv3_fp64(d[0], d[1], d[2], soft2);
          const double v = rinv1_fp64(d[0], d[1], d[2], soft2);
          k = 3.0 * (v * v) * fma(d[0], de[0], fma(d[1], de[1], d[2] * de[2]));
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const double t = s * fma(-k, d[c] - de[c], de[c]);
          a[c] += QARR ? t * wj : t;
          b[c] -= __shfl_sync(0xffffffffu, QARR ? t * wp : t, home);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) addP(u, c, a[c]);
  }
}

// The plan of a force evaluation: make_plan's, with this file's kernel's own
// block sizes where it serves the call (nb_tri.cu).
Plan make_force_plan(int64_t n, int mode, double soft2);
// Whether the kernel serves a plan, and its launch.
bool tri_serves(const Plan &pl, int mode, double soft2);
cudaError_t launch_pair_tri(const Plan &pl, int mode, int64_t n, const double *x, const double *y, const double *z,
                            const double *q, double soft2, double *part, unsigned *err, cudaStream_t st);

// The same for the one-sided sums of ions [i0, i0 + ni) (nb_one.cu).
bool one_serves(const Plan &pl, int mode, int64_t n);
cudaError_t launch_pair_one(const Plan &pl, int64_t n, int64_t i0, int64_t ni, const double *x, const double *y,
                            const double *z, const double *q, double soft2, double *part, cudaStream_t st);

// The potential by the same arithmetic (nb_phi.cu): blocks of 32 G ions, the
// block count and the output mode of a call at n ions (G = 0: the one-sided
// kernel of make_plan(n, mode, 1)); out[jc * n + i], out_doubles in all.
struct PhiPlan {
  int G = 0, nbk = 0;
  Plan one;  // the one-sided plan
  int n_slots = 0;  // partial slots of the output
  size_t out_doubles(int64_t n) const {
    return (size_t)n_slots * (size_t)n + (G ? (size_t)(nbk + 2) / 2 : 0);  // and the schedule's counters
  }
};
PhiPlan make_phi_plan(int64_t n);
cudaError_t launch_phi(const PhiPlan &pl, int64_t n, const double *x, const double *y, const double *z,
                       const double *q, double charge, double soft2, double *part, unsigned *err, cudaStream_t st);

}  // namespace nb
