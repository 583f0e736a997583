// nb_one.cu -- one-sided FP64-class pair sums (Eq. 1) on the FP32 pipe, from
// positions cut into three FP32 words (nb_tri.cuh), for the sizes between the
// single-block steps and the half-pair kernels.
//
// Why: the one-sided kernel of nb_pair.cu takes seven FP64 instructions per
// evaluation (three subtractions, three FMAs, the widened r^-3), 16 cycles of
// the FP64 pipe each for a warp, and is bound by them: 17.2 us of a 23 us
// step at n = 1024.  Here an evaluation is about 94 lane-cycles of the FMA pipe
// and none of the FP64 pipe.  100 steps at n = 1024: 2.31 -> 1.37 ms; with df64,
// whose pair term took 3 FP64 subtractions, and at 1499 and 1999 ions the same
// kernel; rms error 2^-49.2 of the sum of the magnitudes (the FP64 form 2^-48.9).
//
// Layout: 128 threads with one ion each against one j-chunk of the plan, staged
// in shared memory as pairs of partners (j, j + 1), which the two halves of the
// packed operations take; a warp reads each staged entry as one broadcast.
// What an ion gets depends on the ion, its chunk and the scale only, so a range
// of ions (nb_forces_range) gets the bits the full call gives it.  For the same
// reason the scale L is taken over all n ions, not over the block's: up to 4096
// ions that scan is at most 96 loads per thread.
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

// Ion i's sums over the partners [jb, je) in FP64, for the ions the FP32 path leaves.
template <bool QARR>
__device__ __noinline__ void one_fp64(const double *x, const double *y, const double *z, const double *q, double soft2,
                                      int64_t i, int64_t jb, int64_t je, double out[3]) {
  double a[3] = {0.0, 0.0, 0.0};
  const double xi = x[i], yi = y[i], zi = z[i];
  for (int64_t j = jb; j < je; ++j)
    pair_f64<QARR>(xi, yi, zi, make_d4(x[j], y[j], z[j], QARR ? q[j] : 0.0), soft2, a[0], a[1], a[2]);
  for (int c = 0; c < 3; ++c) out[c] = a[c];
}

template <bool QARR, bool SOFT>
__global__ void __launch_bounds__(ONE_NT, 4)
    k_pair_one(int64_t n, int64_t jchunk, int64_t i0, int64_t ni, const double *__restrict__ x,
               const double *__restrict__ y, const double *__restrict__ z, const double *__restrict__ q, double soft2,
               double *__restrict__ part) {
  __shared__ __align__(16) float qs[ONE_J / 2 * ONE_PAIR];
  __shared__ int qf[ONE_J / 32];  // places of each 32 staged partners
  pdl_wait();
  const int tid = threadIdx.x;
  const int64_t i = (int64_t)blockIdx.x * ONE_NT + tid;
  const bool own = i < ni;
  const int64_t g = i0 + i;
  TriScale sc;
  const bool ok = tri_scale<ONE_NT, QARR>(0, 0, 0, (int)n, x, y, z, q, soft2, sc);
  const int64_t c0 = (int64_t)blockIdx.y * jchunk, c1 = min(n, c0 + jchunk);
  double tot[3] = {0.0, 0.0, 0.0};
  if (!ok) {
    if (own) one_fp64<QARR>(x, y, z, q, soft2, g, c0, c1, tot);
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
    const int pf = tri_ion<false>(g, own, x, y, z, q, sc, TRI_FAR, w0, w1, w2);
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
        const int tf = __reduce_or_sync(0xffffffffu, tri_ion<QARR>(jb + j, j < cnt, x, y, z, q, sc, -TRI_FAR, v0, v1, v2));
        if ((j & 31) == 0) qf[j >> 5] = tf;
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
#pragma unroll 1
      for (int j0 = 0; j0 < padded; j0 += 4) {
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
      if (own && (tri_fault(pf, cf) || !(ymax <= TRI_YMAX_GRID))) one_fp64<QARR>(x, y, z, q, soft2, g, jb, jb + cnt, r);
#pragma unroll
      for (int c = 0; c < 3; ++c) tot[c] += r[c];
    }
  }
  if (own)
#pragma unroll
    for (int c = 0; c < 3; ++c) part[((int64_t)blockIdx.y * 3 + c) * ni + i] = tot[c];
}

// The kernel serves the one-sided FP64-class sums above the single-block steps'
// limit, whose bits up to there are those of nb_pair.cu's kernel, to 4096 ions
// (the scan above), unless a tuned launch shape asks for that kernel.  us per
// nb_forces call with its host part, FP64 kernel and this one: n = 513 30.2 and
// 28.4, 1024 31.4 and 27.9, 1499 48.3 and 30.2 (df64 31.6 and 29.1), 1999 df64
// 40.7 and 32.0.
bool one_serves(const Plan &pl, int mode, int64_t n) {
  int tb = 0, tr = 0, tbps = 0;
  return !pl.sym && (mode == MODE_FP64 || mode == MODE_DF64) && n > SMALL_MAX_N && n <= ONE_MAX_N &&
         !tuning_lookup(0, mode, n, &tb, &tr, &tbps);
}

cudaError_t launch_pair_one(const Plan &pl, int64_t n, int64_t i0, int64_t ni, const double *x, const double *y,
                            const double *z, const double *q, double soft2, double *part, cudaStream_t st) {
  const dim3 grid((unsigned)((ni + ONE_NT - 1) / ONE_NT), (unsigned)pl.n_jc);
#define NB_ONE(QA, SO) launch_pdl(k_pair_one<QA, SO>, grid, dim3(ONE_NT), 0, st, n, pl.jchunk, i0, ni, x, y, z, q, soft2, part)
  if (soft2 != 0.0) return q ? NB_ONE(true, true) : NB_ONE(false, true);
  return q ? NB_ONE(true, false) : NB_ONE(false, false);
#undef NB_ONE
}

}  // namespace nb
