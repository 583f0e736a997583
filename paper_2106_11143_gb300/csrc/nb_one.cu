// nb_one.cu -- one-sided FP64-class pair sums (Eq. 1) on the FP32 pipe, from
// positions cut into three FP32 words (nb_tri.cuh), for the sizes between the
// single-block steps and the half-pair kernels.
//
// Why: the one-sided kernel of nb_pair.cu takes seven FP64 instructions per
// evaluation (three subtractions, three FMAs, the widened r^-3), 16 cycles of
// the FP64 pipe each for a warp, and is bound by them: 17.2 us of a 23 us
// step at n = 1024.  Here an evaluation is about 103 lane-cycles of the FMA pipe
// and none of the FP64 pipe; the pipe is 43 % busy at n = 1024, where two blocks
// per SM leave latency bare.  100 steps at n = 1024: 2.31 -> 1.08 ms; with df64,
// whose pair term took 3 FP64 subtractions, and at 1499 and 1999 ions the same
// kernel; rms error 2^-49.2 of the sum of the magnitudes (the FP64 form 2^-48.9).
//
// Layout: 128 threads with one ion each against one j-chunk of the plan, staged
// in shared memory as pairs of partners (j, j + 1), which the two halves of the
// packed operations take; a warp reads each staged entry as one broadcast.  The
// units are the block's, from its 128 ions and its chunk without the few far out
// (one_scale): an ejected ion costs its own FP64 terms, not those of all ions.  What an ion gets depends on its
// group of 128 (ions 128 k .. 128 k + 127 of the system), its chunk and the
// positions alone: a range of ions (nb_forces_range) runs the groups it touches,
// whole, and gets the bits the full call gives it.
#include "nb_pairterm.cuh"
#include "nb_pdl.cuh"
#include "nb_tri.cuh"

namespace nb {

constexpr int ONE_NT = 128;        // threads, one ion each
constexpr int ONE_J = 256;         // partners staged at a time
constexpr int64_t ONE_MAX_N = 4096;

// Pair of partners k, staged as six float4: word h (x, y | z), m, l, weights;
// the floats of value v (0-2 h, 3-5 m, 6-8 l, 9 and 10 the weight's hi and lo
// part) stand at [24 k + 2 v], partner 2 k first.
constexpr int ONE_PAIR = 24;

// Sums over the partners [jb, je) in FP64, for the ions the FP32 path leaves: each
// lane its own ion i, or (WARP) the warp together for one ion, a partner per lane.
template <bool QARR, bool WARP>
__device__ __noinline__ void one_fp64(const double *x, const double *y, const double *z, const double *q, double soft2,
                                      int64_t i, int64_t jb, int64_t je, double out[3]) {
  double a[3] = {0.0, 0.0, 0.0};
  const double xi = x[i], yi = y[i], zi = z[i];
#pragma unroll 4
  for (int64_t j = jb + (WARP ? threadIdx.x & 31 : 0); j < je; j += WARP ? 32 : 1)
    pair_f64<QARR>(xi, yi, zi, make_d4(x[j], y[j], z[j], QARR ? q[j] : 0.0), soft2, a[0], a[1], a[2]);
  for (int c = 0; c < 3; ++c) {
    if (WARP) {
      __syncwarp();
      for (int o = 16; o > 0; o >>= 1) a[c] += __shfl_xor_sync(0xffffffffu, a[c], o);
    }
    out[c] = a[c];
  }
}

// The block's scale (tri_scale) over its ions [p0, p0 + np) and chunk [q0, q0 + nq).
// Where one warp's ions reach more than ONE_OUT bits beyond another's on an axis,
// and at most ONE_OUT_MAX ions in all are beyond that, the unit stops there (some
// are: `capped`) and those ions (one_out) take FP64.  100 steps at n = 1499 without
// and with an ion at 5 m: 1.55 and 1.79 ms, where a unit of all n ions took 1.53 and
// 5.16 and FP64 throughout 4.29.
constexpr int ONE_OUT = 4, ONE_OUT_MAX = 4;
__device__ __forceinline__ bool one_out(int64_t g, const double *x, const double *y, const double *z, const TriScale &sc) {
  return ((__double2hiint(x[g]) >> 20) & 0x7ff) > sc.ex[0] || ((__double2hiint(y[g]) >> 20) & 0x7ff) > sc.ex[1] ||
         ((__double2hiint(z[g]) >> 20) & 0x7ff) > sc.ex[2];
}
template <bool QARR>
__device__ __forceinline__ bool one_scale(int64_t p0, int np, int64_t q0, int nq, const double *x, const double *y,
                                          const double *z, const double *q, double soft2, TriScale &sc, bool &capped) {
  constexpr int NW = ONE_NT / 32;
  __shared__ int red[5][NW];
  int mx[3] = {0, 0, 0}, wx = 0, wn = 0x7fffffff;
  for (int i = threadIdx.x; i < ONE_NT + nq; i += ONE_NT) {
    if (i >= np && i < ONE_NT) continue;
    const int64_t g = i < ONE_NT ? p0 + i : q0 + (i - ONE_NT);
    mx[0] = max(mx[0], __double2hiint(x[g]) & 0x7fffffff);
    mx[1] = max(mx[1], __double2hiint(y[g]) & 0x7fffffff);
    mx[2] = max(mx[2], __double2hiint(z[g]) & 0x7fffffff);
    if (QARR) {
      const int w = __double2hiint(q[g]) & 0x7fffffff;
      wx = max(wx, w);
      if (q[g] != 0.0) wn = min(wn, w);
    }
  }
  const int warp = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 3; ++c) mx[c] = __reduce_max_sync(0xffffffffu, mx[c]);
  if (QARR) {
    wx = __reduce_max_sync(0xffffffffu, wx);
    wn = __reduce_min_sync(0xffffffffu, wn);
  }
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int c = 0; c < 3; ++c) red[c][warp] = mx[c];
    red[3][warp] = wx;
    red[4][warp] = wn;
  }
  __syncthreads();
  int lo[3];
  capped = false;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    lo[c] = 0x7fffffff;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const int v = red[c][w];
      mx[c] = max(mx[c], v);
      if (v) lo[c] = min(lo[c], v);
    }
    capped = capped || (mx[c] >> 20) - (lo[c] >> 20) > ONE_OUT;
  }
  if (capped) {  // the same for all threads
#pragma unroll
    for (int c = 0; c < 3; ++c) sc.ex[c] = mx[c] ? min(mx[c] >> 20, (lo[c] >> 20) + ONE_OUT) : 0;
    int k = 0;
    for (int i = threadIdx.x; i < ONE_NT + nq; i += ONE_NT)
      if (i < np || i >= ONE_NT) k += one_out(i < ONE_NT ? p0 + i : q0 + (i - ONE_NT), x, y, z, sc);
    __shared__ int outs[NW];
    k = __reduce_add_sync(0xffffffffu, k);
    if ((threadIdx.x & 31) == 0) outs[warp] = k;
    __syncthreads();
    k = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) k += outs[w];
    capped = k <= 2 * ONE_OUT_MAX;  // an ion of the group may be a partner too
    if (capped)
#pragma unroll
      for (int c = 0; c < 3; ++c) mx[c] = sc.ex[c] << 20;
  }
  bool ok = tri_axes<QARR>(mx, soft2, sc);
  sc.ew = 1023;
  if (QARR) {
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      wx = max(wx, red[3][w]);
      wn = min(wn, red[4][w]);
    }
    sc.ew = wx >> 20;
    ok = ok && sc.ew >= 1023 - 400 && sc.ew <= 1023 + 400 && sc.ew - (wn >> 20) <= TRI_WSPREAD;
  }
  return ok;
}

template <bool QARR, bool SOFT>
__global__ void __launch_bounds__(ONE_NT, 4)
    k_pair_one(int64_t n, int64_t jchunk, int64_t i0, int64_t ni, const double *__restrict__ x,
               const double *__restrict__ y, const double *__restrict__ z, const double *__restrict__ q, double soft2,
               double *__restrict__ part) {
  __shared__ __align__(16) float qs[ONE_J / 2 * ONE_PAIR];
  __shared__ int qf[ONE_J / 32];       // places of each 32 staged partners
  __shared__ unsigned qo[ONE_J / 32];  // and those beyond the unit
  pdl_wait();
  const int tid = threadIdx.x;
  const int64_t gb = (i0 / ONE_NT + blockIdx.x) * ONE_NT;  // the group's first ion
  const int64_t g = gb + tid;
  const bool own = g < n;
  const int64_t c0 = (int64_t)blockIdx.y * jchunk, c1 = min(n, c0 + jchunk);
  TriScale sc;
  bool capped;
  const bool ok = one_scale<QARR>(gb, (int)min((int64_t)ONE_NT, n - gb), c0, (int)(c1 - c0), x, y, z, q, soft2, sc, capped);
  double tot[3] = {0.0, 0.0, 0.0};
  if (!ok) {
    if (own) one_fp64<QARR, false>(x, y, z, q, soft2, g, c0, c1, tot);
  } else {
    const int kl = sc.em - 1022, kw = sc.ew - 1023;
    const double fwd = pow2d(kw - 2 * kl);
    f32x2 s2h = 0, s2l = 0;
    if (SOFT) {
      float h, l;
      split_f64(soft2 * pow2d(-2 * kl), h, l);
      s2h = pk1(h);
      s2l = pk1(l);
    }
    float w0[4], w1[4], w2[4];
    const bool far = capped && own && one_out(g, x, y, z, sc);
    const int pf = tri_ion<false>(g, own && !far, x, y, z, q, sc, TRI_FAR, w0, w1, w2);
    f32x2 ph[3], pm[3], pl[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ph[c] = pk1(w0[c]);
      pm[c] = pk1(w1[c]);
      pl[c] = pk1(w2[c]);
    }
    for (int64_t jb = c0; jb < c1; jb += ONE_J) {
      const int cnt = (int)min((int64_t)ONE_J, c1 - jb), padded = (cnt + 3) & ~3;
      if (jb > c0) __syncthreads();
      for (int j = tid; j < ONE_J; j += ONE_NT) {  // a warp takes 32 partners
        if ((j & ~31) >= padded) break;
        float v0[4], v1[4], v2[4];
        const bool out = capped && j < cnt && one_out(jb + j, x, y, z, sc);
        const int tf = __reduce_or_sync(
            0xffffffffu, tri_ion<QARR>(jb + j, j < cnt && !out, x, y, z, q, sc, -TRI_FAR, v0, v1, v2));
        const unsigned to = __ballot_sync(0xffffffffu, out);
        if ((j & 31) == 0) {
          qf[j >> 5] = tf;
          qo[j >> 5] = to;
        }
        float *e = qs + (j >> 1) * ONE_PAIR + (j & 1);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          e[2 * c] = v0[c];
          e[6 + 2 * c] = v1[c];
          e[12 + 2 * c] = v2[c];
        }
        e[18] = v0[3];
        e[20] = v1[3];
      }
      __syncthreads();
      int cf = 0;  // the partners' places
      for (int k = 0; k < padded; k += 32) cf |= qf[k >> 5];
      const int self = (int)(g - jb);  // the ion's own place among the staged partners, if any
      f32x2 ah[3] = {0, 0, 0}, al[3] = {0, 0, 0};
      float ymax = 0.0f, rmin = __int_as_float(0x7f800000);
      bool left = far || (own && tri_fault(pf, cf));  // to FP64
      const int jend = __all_sync(0xffffffffu, left || !own) ? 0 : padded;
#pragma unroll 1
      for (int j0 = 0; j0 < jend; j0 += 4) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const int j = j0 + 2 * s;
          const ulonglong2 *e = reinterpret_cast<const ulonglong2 *>(qs + (j >> 1) * ONE_PAIR);
          const ulonglong2 a = e[0], b = e[1], c2 = e[2], d = e[3], f = e[4];
          f32x2 dh[3], dl[3], h, l, sh, sl;
          tri_diff_n(ph[0], pm[0], pl[0], a.x, b.y, d.x, dh[0], dl[0]);
          tri_diff_n(ph[1], pm[1], pl[1], a.y, c2.x, d.y, dh[1], dl[1]);
          tri_diff_n(ph[2], pm[2], pl[2], b.x, c2.y, f.x, dh[2], dl[2]);
          tri_r2(dh, dl, h, l);
          float ha, hb;
          upk(h, ha, hb);
          // the ion itself is left out: its d = 0 gives a zero term with any finite y
          const bool me0 = self == j, me1 = self == j + 1;
          if (SOFT) {
            rmin = fminf(rmin, fminf(me0 ? rmin : ha, me1 ? rmin : hb));
            f32x2 t;
            ptwo_sum(h, s2h, h, t);
            l = padd(l, padd(t, s2l));
            upk(h, ha, hb);
          }
          float ya = rsqrt_approx(ha), yb = rsqrt_approx(hb);
          if (!SOFT) ymax = fmaxf(ymax, fmaxf(me0 ? 0.0f : ya, me1 ? 0.0f : yb));
          ya = fminf(ya, TRI_YMAX_GRID);
          yb = fminf(yb, TRI_YMAX_GRID);
          tri_rinv3(h, l, pk(ya, yb), sh, sl);
          if (QARR) {
            f32x2 th, tl;
            ptwo_prod(sh, sl, f.y, e[5].x, th, tl);
            sh = th;
            sl = tl;
          }
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            f32x2 th, tl;
            ptwo_prod(dh[c], dl[c], sh, sl, th, tl);
            pacc(ah[c], al[c], th, tl);
            if (s == 1) pfast2(ah[c], al[c]);  // as in tri_tile
          }
        }
      }
      if (SOFT) ymax = rsqrt_approx(rmin);
      double r[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float h0, h1, l0, l1;
        upk(ah[c], h0, h1);
        upk(al[c], l0, l1);
        r[c] = ((f32_to_f64(h0) + f32_to_f64(h1)) + (f32_to_f64(l0) + f32_to_f64(l1))) * fwd;
      }
      left = left || (own && !(ymax <= TRI_YMAX_GRID));
      for (int k = 0; capped && k < padded; k += 32)
        for (unsigned o = qo[k >> 5]; o; o &= o - 1) {
          const int64_t j = jb + k + __ffs((int)o) - 1;
          double t[3];
          if (own) one_fp64<QARR, false>(x, y, z, q, soft2, g, j, j + 1, t);
          if (own)
            for (int c = 0; c < 3; ++c) r[c] += t[c];
        }
      // one by one by the warp (7 FP64 instructions per 32 partners and 15 adds of
      // lanes each), or every lane its own (7 per partner), whichever is fewer
      const unsigned m = __ballot_sync(0xffffffffu, left);
      if (__popc(m) * (7 * ((cnt + 31) >> 5) + 15) < 7 * cnt) {
        for (unsigned k = m; k; k &= k - 1) {
          const int l = __ffs((int)k) - 1;
          double t[3];
          one_fp64<QARR, true>(x, y, z, q, soft2, g - (tid & 31) + l, jb, jb + cnt, t);
          if ((tid & 31) == l)
            for (int c = 0; c < 3; ++c) r[c] = t[c];
        }
      } else if (left) {
        one_fp64<QARR, false>(x, y, z, q, soft2, g, jb, jb + cnt, r);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) tot[c] += r[c];
    }
  }
  if (g >= i0 && g < i0 + ni)
#pragma unroll
    for (int c = 0; c < 3; ++c) part[((int64_t)blockIdx.y * 3 + c) * ni + g - i0] = tot[c];
}

// The kernel serves the one-sided FP64-class sums above the single-block steps'
// limit, whose bits up to there are those of nb_pair.cu's kernel, to 4096 ions
// (whole calls are half-pair from 1500 or 2000), unless a tuned launch shape asks
// for that kernel.  us a
// step with the FP64 kernel and this one: 15.6 and 9.9 at n = 600 (df64 13.1),
// 23.8 and 11.2 at 1024 (df64 16.6), 42.9 and 15.6 at 1499 (df64 25.9).
bool one_serves(const Plan &pl, int mode, int64_t n) {
  int tb = 0, tr = 0, tbps = 0;
  return !pl.sym && (mode == MODE_FP64 || mode == MODE_DF64) && n > SMALL_MAX_N && n <= ONE_MAX_N &&
         !tuning_lookup(0, mode, n, &tb, &tr, &tbps);
}

cudaError_t launch_pair_one(const Plan &pl, int64_t n, int64_t i0, int64_t ni, const double *x, const double *y,
                            const double *z, const double *q, double soft2, double *part, cudaStream_t st) {
  const dim3 grid((unsigned)((i0 + ni + ONE_NT - 1) / ONE_NT - i0 / ONE_NT), (unsigned)pl.n_jc);
#define NB_ONE(QA, SO) launch_pdl(k_pair_one<QA, SO>, grid, dim3(ONE_NT), 0, st, n, pl.jchunk, i0, ni, x, y, z, q, soft2, part)
  if (soft2 != 0.0) return q ? NB_ONE(true, true) : NB_ONE(false, true);
  return q ? NB_ONE(true, false) : NB_ONE(false, false);
#undef NB_ONE
}

}  // namespace nb
