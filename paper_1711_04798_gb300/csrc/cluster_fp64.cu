// FP64 pieces of the projector step on one thread-block cluster.
//
// GB300 executes FP64 at a small fraction of its FP32 rate per SM, so a
// k x k Jacobi SVD or Cholesky factorisation on a single CTA is bound by one
// SM's FP64 units, while spreading it over a grid pays a global-memory
// barrier per step.  Here the rows are distributed over the CTAs of one
// cluster (row i lives in the shared memory of CTA i mod csize), warps read
// and write partner rows through distributed shared memory, and steps are
// separated by the hardware cluster barrier.  The pair schedule is that of the
// grid-wide kernels (kernels.cu), over the rows that take part; angles, carried
// norms and the blocked Cholesky are this file's own.
#include <cooperative_groups.h>

#include <algorithm>

#include "ctm_internal.h"
#include "dfloat.h"

namespace cg = cooperative_groups;

namespace {

constexpr int CL_THREADS = 256;         // 8 warps per CTA (Cholesky): FP64 pipe occupancy
constexpr int CL_SMEM = 200 * 1024;     // dynamic shared memory bound per CTA
int g_csize = 0;                        // CTAs per cluster (16 if schedulable, else 8)
int g_clusters = 0;                     // clusters of 16 with CL_SMEM that the device holds at once

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ void pair_of(int r, int p, int np, int rounds, int* i, int* j) {
  int a, b;
  if (p == 0) {
    a = np - 1;
    b = r;
  } else {
    a = (r + p) % rounds;
    b = (r - p + rounds) % rounds;
  }
  if (a > b) { const int t = a; a = b; b = t; }
  *i = a;
  *j = b;
}

// a complex element of a row: (Re hi, Re lo, Im hi, Im lo)
__device__ __forceinline__ float4 df_elem(cplx x) {
  const df2 r = df_of(x.x), i = df_of(x.y);
  return make_float4(r.h, r.l, i.h, i.l);
}

// the sums of a and b over the warp, in every lane: after the first butterfly
// level each half of the warp carries one of them
__device__ __forceinline__ void warp_sum2(double& a, double& b) {
  const bool up = threadIdx.x & 16;
  double k = up ? b : a;
  k += __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  a = __shfl_sync(0xffffffffu, k, 0);
  b = __shfl_sync(0xffffffffu, k, 16);
}

__device__ __forceinline__ void warp_sum2(df2& a, df2& b) {
  const bool up = threadIdx.x & 16;
  df2 k = up ? b : a;
  const df2 o = up ? a : b;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, d == 16 ? o.h : k.h, d);
    const float ol = __shfl_xor_sync(0xffffffffu, d == 16 ? o.l : k.l, d);
    float s, t;
    two_sum(k.h, oh, s, t);
    k.h = s;
    k.l = __fadd_rn(k.l, __fadd_rn(ol, t));
  }
  k = df_norm(k);
  a = {__shfl_sync(0xffffffffu, k.h, 0), __shfl_sync(0xffffffffu, k.l, 0)};
  b = {__shfl_sync(0xffffffffu, k.h, 16), __shfl_sync(0xffffffffu, k.l, 16)};
}

// A rotation of rows i, j (the form of jac_rotate): a' = c a - q b,
// b' = c b + conj(q) a with q = s e^{-i phi}, c^2 + |q|^2 = 1.
template <class S>
struct Rot {
  S c, qr, qi;
};

// Row element types: FP64 complex, or two double-floats (Re hi, Re lo, Im hi,
// Im lo) in the same 16 bytes.
template <bool DF>
struct RowT {
  typedef double S;
  typedef cplx E;
};
template <>
struct RowT<true> {
  typedef df2 S;
  typedef float4 E;
};

__device__ __forceinline__ void dot_acc(double& gr, double& gi, cplx x, cplx y) {  // conj(x) y
  gr = fma(x.x, y.x, gr);
  gr = fma(x.y, y.y, gr);
  gi = fma(x.x, y.y, gi);
  gi = fma(-x.y, y.x, gi);
}
__device__ __forceinline__ void dot_acc(df2& gr, df2& gi, float4 x, float4 y) {
  const df2 xr = {x.x, x.y}, xi = {x.z, x.w}, yr = {y.x, y.y}, yi = {y.z, y.w};
  acc_mul(gr, xr, yr);
  acc_mul(gr, xi, yi);
  acc_mul(gi, xr, yi);
  acc_mul(gi, df_negate(xi), yr);
}
__device__ __forceinline__ void norm_acc(double& a, cplx x) {
  a = fma(x.x, x.x, a);
  a = fma(x.y, x.y, a);
}
__device__ __forceinline__ void norm_acc(df2& a, float4 x) {
  acc_mul(a, {x.x, x.y}, {x.x, x.y});
  acc_mul(a, {x.z, x.w}, {x.z, x.w});
}
__device__ __forceinline__ void rotate_elem(const Rot<double>& r, cplx& a, cplx& b) {
  const cplx x = a, y = b;
  a.x = fma(-r.qr, y.x, fma(r.qi, y.y, r.c * x.x));
  a.y = fma(-r.qr, y.y, fma(-r.qi, y.x, r.c * x.y));
  b.x = fma(r.qr, x.x, fma(r.qi, x.y, r.c * y.x));
  b.y = fma(r.qr, x.y, fma(-r.qi, x.x, r.c * y.y));
}
__device__ __forceinline__ void rotate_elem(const Rot<df2>& r, float4& a, float4& b) {
  const df2 xr = {a.x, a.y}, xi = {a.z, a.w}, yr = {b.x, b.y}, yi = {b.z, b.w};
  const df2 nr = df_negate(r.qr), ni = df_negate(r.qi);
  df2 ar = df_mul(r.c, xr), ai = df_mul(r.c, xi), br = df_mul(r.c, yr), bi = df_mul(r.c, yi);
  acc_mul(ar, nr, yr);
  acc_mul(ar, r.qi, yi);
  acc_mul(ai, nr, yi);
  acc_mul(ai, ni, yr);
  acc_mul(br, r.qr, xr);
  acc_mul(br, r.qi, xi);
  acc_mul(bi, r.qr, xi);
  acc_mul(bi, ni, xr);
  ar = df_norm(ar);
  ai = df_norm(ai);
  br = df_norm(br);
  bi = df_norm(bi);
  a = make_float4(ar.h, ar.l, ai.h, ai.l);
  b = make_float4(br.h, br.l, bi.h, bi.l);
}

// The rotation that makes rows of squared norms al, be and inner product
// g = x^H y orthogonal: t = tan, c = 1/sqrt(1 + t^2), q = c t conj(g)/|g|; tg
// = t |g| (the squared norms become al - tg, be + tg).  Returns 0: left alone
// (|g| <= tol sqrt(al be)), 1: off-orthogonality and angle at most 1e-8, 2:
// larger.  g is scaled by a power of two into [1, 2) first, so nothing under-
// or overflows that the test does not settle.
__device__ __forceinline__ int rotation(df2 al, df2 be, df2 gr, df2 gi, float tol, Rot<df2>& rot, df2& tg) {
  const float big = fmaxf(fabsf(gr.h), fabsf(gi.h));
  const int e = (int)(__float_as_uint(big) >> 23);
  if (!(big > 0.f) || e >= 255 || e < 8) return 0;
  const float S = __uint_as_float((unsigned)(254 - e) << 23);  // 2^(127-e)
  const float iS = __uint_as_float((unsigned)e << 23);         // 1/S
  gr = {gr.h * S, gr.l * S};
  gi = {gi.h * S, gi.l * S};
  df2 g2 = df_mul(gr, gr);
  acc_mul(g2, gi, gi);
  g2 = df_norm(g2);
  const float as = al.h * S, bs = be.h * S;
  if (!(g2.h > (tol * as) * (tol * bs))) return 0;
  const df2 ig = df_rsqrt(g2);
  const df2 d = df_add(be, df_negate(al));
  const float zf = 0.5f * (d.h * S) * ig.h;
  // the tangent in FP32: an angle off by 2^-24 leaves that share of g behind
  const float az = fabsf(zf);
  const float t = copysignf(az < 1e15f ? 1.0f / (az + sqrtf(fmaf(zf, zf, 1.0f))) : 0.5f / az, zf);
  const df2 tt = {t, 0.f};
  df2 w = df_mul(tt, tt), one;
  two_sum(1.0f, w.h, one.h, one.l);
  one.l = __fadd_rn(one.l, w.l);
  rot.c = df_rsqrt(df_norm(one));
  const df2 u = df_norm(df_mul(df_norm(df_mul(rot.c, tt)), ig));
  rot.qr = df_norm(df_mul(u, gr));
  rot.qi = df_negate(df_norm(df_mul(u, gi)));
  tg = df_mul(df_norm(df_mul(g2, ig)), tt);
  tg = {tg.h * iS, tg.l * iS};
  return (g2.h > (1e-8f * as) * (1e-8f * bs) || fabsf(t) > 1e-8f) ? 2 : 1;
}

// FP64 rows: the angle in double-float on the FP32 pipe (its tangent good to
// 2^-45; FP32 alone raised the corner spectra's noise from 2e-11 to 1e-10),
// then c and q from that tangent in FP64, so c^2 + |q|^2 = 1 to FP64 rounding
// whatever the tangent's error.  Some 20 FP64 instructions instead of the
// 100 of FP64 roots and divides, each of which holds the SM's FP64 unit for
// about 18 cycles.
__device__ __forceinline__ int rotation(double al, double be, double gr, double gi, float tol, Rot<double>& rot,
                                        double& tg) {
  // exponent of the larger part, by integer operations
  const unsigned long long br = (unsigned long long)__double_as_longlong(gr) & 0x7fffffffffffffffull;
  const unsigned long long bi = (unsigned long long)__double_as_longlong(gi) & 0x7fffffffffffffffull;
  const int e = (int)((br > bi ? br : bi) >> 52);
  if (e >= 2047 || e < 64) return 0;  // |g| below 2^-960 (or not finite): nothing to rotate
  const int sh = 1023 - e;
  auto scaled = [&](double v) {  // v 2^sh for v >= 0, clamped (v is a squared norm: compared and subtracted only)
    const long long b = __double_as_longlong(v);
    const int ev = (int)(b >> 52) + sh;
    return b <= 0 || ev <= 0 ? 0.0 : (ev >= 2046 ? 1e308 : __longlong_as_double(b + ((long long)sh << 52)));
  };
  auto scale_s = [&](double v) {  // signed, |v| <= |g|'s larger part
    const long long b = __double_as_longlong(v);
    const int ev = (int)((b >> 52) & 0x7ff) + sh;
    return (b << 1) == 0 || ev <= 0 ? 0.0 : __longlong_as_double(b + ((long long)sh << 52));
  };
  const double xr = scale_s(gr), xi = scale_s(gi), as = scaled(al), bs = scaled(be);
  const float hr = d2f_bits(xr), hi = d2f_bits(xi);
  const df2 dr = {hr, d2f_bits(xr - f2d_bits(hr))}, di = {hi, d2f_bits(xi - f2d_bits(hi))};
  df2 g2 = df_mul(dr, dr);
  acc_mul(g2, di, di);
  g2 = df_norm(g2);
  const float af = d2f_bits(as), bf = d2f_bits(bs);
  if (!(g2.h > (tol * af) * (tol * bf))) return 0;
  const df2 ig = df_rsqrt(g2);
  const double dd = bs - as;
  const float dh = d2f_bits(dd);
  df2 z = df_norm(df_mul({dh, fabsf(dh) < 1e30f ? d2f_bits(dd - f2d_bits(dh)) : 0.f}, ig));
  z = {0.5f * fabsf(z.h), dh >= 0.f ? 0.5f * z.l : -0.5f * z.l};
  df2 t;
  if (z.h < 1e8f) {
    // 1 / (|z| + sqrt(1 + z^2)): the root as w / sqrt(w), the reciprocal refined once
    df2 w = df_mul(z, z), w1;
    two_sum(1.0f, w.h, w1.h, w1.l);
    w1.l = __fadd_rn(w1.l, w.l);
    w1 = df_norm(w1);
    const df2 den = df_add(z, df_norm(df_mul(w1, df_rsqrt(w1))));
    const float r0 = 1.0f / den.h;
    const df2 p = df_norm(df_mul(den, {r0, 0.f}));
    t = {r0, __fmul_rn(r0, __fadd_rn(__fadd_rn(1.0f, -p.h), -p.l))};
  } else {
    t = {0.5f / z.h, 0.f};  // 1/(2 z): below 5e-9, good to 2^-23 of itself
  }
  if (dh < 0.f) t = df_negate(t);
  const df2 u = df_norm(df_mul(df_norm(t), ig));
  const df2 ur = df_norm(df_mul(u, dr)), ui = df_norm(df_mul(u, di));
  const double er = f2d_bits(ur.h) + f2d_bits(ur.l), ei = f2d_bits(ui.h) + f2d_bits(ui.l);  // t conj(phase), exactly
  const double w = fma(er, er, fma(ei, ei, 1.0));
  rot.c = rsqrt64_normal(w);  // 1 <= w <= 2
  rot.qr = rot.c * er;
  rot.qi = -(rot.c * ei);
  tg = fma(er, gr, ei * gi);
  return (g2.h > (1e-8f * af) * (1e-8f * bf) || fabsf(t.h) > 1e-8f) ? 2 : 1;
}

__device__ __forceinline__ double s_zero(double) { return 0.0; }
__device__ __forceinline__ df2 s_zero(df2) { return {0.f, 0.f}; }
__device__ __forceinline__ double s_val(double x) { return x; }
__device__ __forceinline__ double s_val(df2 x) { return df_val(x); }
__device__ __forceinline__ double s_add(double a, double b) { return a + b; }
__device__ __forceinline__ df2 s_add(df2 a, df2 b) { return df_add(a, b); }
__device__ __forceinline__ double s_neg(double a) { return neg_bits(a); }
__device__ __forceinline__ df2 s_neg(df2 a) { return df_negate(a); }
__device__ __forceinline__ bool s_less(double a, double b) { return a < b; }       // for squared norms
__device__ __forceinline__ bool s_less(df2 a, df2 b) { return a.h < b.h; }
__device__ __forceinline__ double s_quarter(double a) { return 0.25 * a; }
__device__ __forceinline__ df2 s_quarter(df2 a) { return {0.25f * a.h, 0.25f * a.l}; }

constexpr int JC_MAXP = 32;  // row pairs of one round per CTA (n <= 2 * 16 * 32 with 16 CTAs, half with 8)

// One-sided Jacobi (Hestenes) on the n rows of G (length m), one matrix per
// cluster (cluster b: G + b * strideG), rows in the cluster's shared memory
// (active row a in CTA a mod cs).  One warp per row pair: it holds both rows in
// registers between the inner product and the rotation (NE elements per lane;
// NE = 0: any length, read twice) and needs no block barrier; a cluster
// barrier ends each round.  Rows below 1e-15 ||G||_F are rounding noise and
// take part in no rotation: they are left out of the schedule, which covers
// the other rows only.  The squared norms stay with their rows and follow the
// rotations (al - t|g|, be + t|g|), formed anew at every sweep and where a
// rotation takes most of one away, so a round's inner product is x^H y alone.
//
// Bound: FP64 rows by the FP64 units of the cluster's SMs (about 18 cycles per
// warp instruction and SM: 16 for the inner product, 48 for the rotation and
// some 25 for the reduction and angle, per pair and 128 columns); double-float
// rows by the latency of a round (loads from the partner CTAs, reduction,
// angle, rotation, cluster barrier).
//
// With a log: the rotations are logged and replayed onto Vt by
// jacobi_replay_kernel across the GPU (rotating FP64 rows of V here would double
// the FP64 work of these 16 SMs).  With Vt: the second half of the warps rotates
// the rows of V (from Vt, in the rows' arithmetic), one round behind the first
// half; for double-float rows in cycles that the rounds leave idle.  V = false:
// without that half's code, which costs the FP64 kernel 5 % by its registers.
template <bool DF, int NE, bool V>
__global__ void __launch_bounds__(512, 1)
    jacobi_cluster_kernel(cplx* __restrict__ G0, int n, int m, long long ldg, long long strideG,
                          cplx* __restrict__ Vt, int max_sweeps, float tol, double4_16a* __restrict__ log,
                          int* __restrict__ amap, int* sweeps_used, DevStatus* st, int warm) {
  typedef typename RowT<DF>::S S;
  typedef typename RowT<DF>::E E;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), cs = (int)cl.num_blocks();
  cplx* __restrict__ G = G0 + (long long)(blockIdx.x / cs) * strideG;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int R = (n + cs - 1) / cs;   // row slots per CTA
  const bool with_v = V && Vt != nullptr;
  const int gwarps = with_v ? nwarps / 2 : nwarps;
  extern __shared__ cplx sm[];       // [R x m] rows of G, then (with_v) [R x n] rows of V
  __shared__ S s_nrm[JC_MAXP * 2];   // squared norm of each row slot
  __shared__ int s_act[JC_MAXP * 2 * 16], s_nact;  // original row of each active row
  __shared__ double s_fro;
  __shared__ int s_rot, s_big;
  __shared__ Rot<S> s_rec[2][JC_MAXP];  // with_v: the last rounds' rotations
  __shared__ int s_recij[2][JC_MAXP];     // their rows, i << 16 | j, or -1
  __shared__ double s_w[16];
  E* gl = (E*)sm;
  E* vl = (E*)(sm + (long long)R * m);
  // squared row norms of the whole matrix by every CTA: the Frobenius norm and
  // the active rows, the same in each
  double* rn = (double*)sm;  // n doubles before the rows arrive
  for (int i = warp; i < n; i += nwarps) {
    double f = 0.0;
    for (int t = lane; t < m; t += 32) {
      const cplx x = G[(long long)i * ldg + t];
      f = fma(x.x, x.x, f);
      f = fma(x.y, x.y, f);
    }
    f = warp_sum(f);
    if (lane == 0) rn[i] = f;
  }
  __syncthreads();
  double f = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) f += rn[i];
  f = warp_sum(f);
  if (lane == 0) s_w[warp] = f;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < nwarps; ++w) t += s_w[w];
    s_fro = t;
    s_rot = 0;
    s_big = 0;
  }
  __syncthreads();
  const double fro2 = s_fro;
  if (warp == 0) {
    int cnt = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
      const bool on = i0 + lane < n && rn[i0 + lane] > fro2 * 1e-30;
      const unsigned mask = __ballot_sync(0xffffffffu, on);
      if (on) s_act[cnt + __popc(mask & ((1u << lane) - 1u))] = i0 + lane;
      cnt += __popc(mask);
    }
    if (lane == 0) s_nact = cnt;
  }
  __syncthreads();
  const int na = s_nact;
  // double-float rows are scaled by a power of two so that ||G||_F lies near
  // 2^20: every squared norm that takes part is then far inside FP32's range
  double sc = 1.0, isc = 1.0;
  if (DF && fro2 > 0.0 && fro2 < 1e300) {
    const int ef = ((int)(__double_as_longlong(fro2) >> 52) - 1023) / 2;
    sc = __longlong_as_double((long long)(1023 + 20 - ef) << 52);
    isc = __longlong_as_double((long long)(1023 - 20 + ef) << 52);
  }
  const double fros = DF ? fro2 * sc * sc : fro2;
  for (int l = 0; l < R; ++l) {
    const int a = l * cs + rank;
    if (a >= na) break;
    const int i = s_act[a];
    for (int t = threadIdx.x; t < m; t += blockDim.x) {
      const cplx x = G[(long long)i * ldg + t];
      if constexpr (DF)
        gl[(long long)l * m + t] = df_elem(make_double2(x.x * sc, x.y * sc));
      else
        gl[(long long)l * m + t] = x;
    }
    if (with_v)
      for (int t = threadIdx.x; t < n; t += blockDim.x) {
        const cplx v = warm ? Vt[(long long)i * n + t] : make_double2(t == i ? 1.0 : 0.0, 0.0);
        if constexpr (DF)
          vl[(long long)l * n + t] = df_elem(v);
        else
          vl[(long long)l * n + t] = v;
      }
  }
  if (with_v)
    for (int q = threadIdx.x; q < 2 * JC_MAXP; q += blockDim.x) (&s_recij[0][0])[q] = -1;
  const float neg = DF ? (float)(fros * 1e-30) : 0.f;
  const double negd = fros * 1e-30;
  auto negligible = [&](S x) {
    if constexpr (DF)
      return !(x.h > neg);
    else
      return !(x > negd);
  };
  auto grow = [&](int a) { return cl.map_shared_rank(gl, a % cs) + (long long)(a / cs) * m; };
  auto vrow = [&](int a) { return cl.map_shared_rank(vl, a % cs) + (long long)(a / cs) * n; };
  auto nrm = [&](int a) { return cl.map_shared_rank(s_nrm, a % cs) + a / cs; };
  const int np = (na + 1) & ~1;
  const int rounds = np - 1, npairs = np / 2;
  const int own = (npairs + cs - 1) / cs;  // pairs of this CTA: p = slot * cs + rank
  bool converged = na < 2;
  int sweep = 0, par = 0;
  // with_v: the second half of the warps applies the rotations recorded in buffer b
  auto rotate_v = [&](int b) {
    if constexpr (!V) return;
    for (int slot = warp - gwarps; slot < own; slot += gwarps) {
      const int ij = s_recij[b][slot];
      if (ij < 0) continue;
      E* vi = vrow(ij >> 16);
      E* vj = vrow(ij & 0xffff);
      const Rot<S> rot = s_rec[b][slot];
      for (int q = lane; q < n; q += 32) {
        E x = vi[q], y = vj[q];
        rotate_elem(rot, x, y);
        vi[q] = x;
        vj[q] = y;
      }
    }
  };
  cl.sync();
  for (; sweep < max_sweeps && !converged; ++sweep) {
    // squared norms formed anew
    for (int l = warp; l < R; l += nwarps) {
      if (l * cs + rank >= na) break;
      S a = s_zero(S());
      for (int t = lane; t < m; t += 32) norm_acc(a, gl[(long long)l * m + t]);
      S b = a;
      warp_sum2(a, b);
      if (lane == 0) s_nrm[l] = a;
    }
    cl.sync();
    for (int r = 0; r < rounds; ++r) {
      if (warp < gwarps) {
        for (int slot = warp; slot < own; slot += gwarps) {
          const int p = slot * cs + rank;
          int i = 0, j = na, kind = 0;
          if (p < npairs) pair_of(r, p, np, rounds, &i, &j);
          Rot<S> rot;
          if (p < npairs && j < na) {
            E* gi = grow(i);
            E* gj = grow(j);
            const S al = *nrm(i), be = *nrm(j);
            S gr = s_zero(S()), gim = s_zero(S()), tg = s_zero(S());
            constexpr int NR = NE > 0 ? NE : 1;
            E x[NR], y[NR];
            if constexpr (NE > 0) {
#pragma unroll
              for (int q = 0; q < NE; ++q) {
                const int t = lane + 32 * q;
                x[q] = E();
                y[q] = E();
                if (t < m) {
                  x[q] = gi[t];
                  y[q] = gj[t];
                }
              }
#pragma unroll
              for (int q = 0; q < NE; ++q) dot_acc(gr, gim, x[q], y[q]);
            } else {
              for (int t = lane; t < m; t += 32) dot_acc(gr, gim, gi[t], gj[t]);
            }
            warp_sum2(gr, gim);
            if (!negligible(al) && !negligible(be)) kind = rotation(al, be, gr, gim, tol, rot, tg);
            if (kind) {
              S na_i = s_add(al, s_neg(tg)), na_j = s_add(be, tg);
              const bool anew = !s_less(s_quarter(al), na_i) || !s_less(s_quarter(be), na_j);
              S ni = s_zero(S()), nj = s_zero(S());
              if constexpr (NE > 0) {
#pragma unroll
                for (int q = 0; q < NE; ++q) {
                  const int t = lane + 32 * q;
                  rotate_elem(rot, x[q], y[q]);
                  if (t < m) {
                    gi[t] = x[q];
                    gj[t] = y[q];
                  }
                }
                if (anew) {
#pragma unroll
                  for (int q = 0; q < NE; ++q) {
                    norm_acc(ni, x[q]);
                    norm_acc(nj, y[q]);
                  }
                }
              } else {
                for (int t = lane; t < m; t += 32) {
                  E u = gi[t], v = gj[t];
                  rotate_elem(rot, u, v);
                  gi[t] = u;
                  gj[t] = v;
                  if (anew) {
                    norm_acc(ni, u);
                    norm_acc(nj, v);
                  }
                }
              }
              if (anew) {
                warp_sum2(ni, nj);
                na_i = ni;
                na_j = nj;
              }
              if (lane == 0) {
                *nrm(i) = na_i;
                *nrm(j) = na_j;
                atomicAdd(&s_rot, 1);
                if (kind == 2) s_big = 1;
              }
            }
          }
          if (lane == 0) {
            if (with_v) {
              s_recij[par][slot] = kind ? (i << 16 | j) : -1;
              s_rec[par][slot] = rot;
            }
            if (log && p < npairs) {
              double4_16a rec = make_double4_16a(2.0, 0.0, 0.0, 0.0);
              if (kind) rec = make_double4_16a(s_val(rot.c), s_val(rot.qr), s_val(rot.qi), 0.0);
              log[((long long)sweep * rounds + r) * npairs + p] = rec;
            }
          }
        }
      } else {
        rotate_v(par ^ 1);
      }
      par ^= 1;
      cl.sync();
    }
    int total = 0, big = 0;
    for (int r = 0; r < cs; ++r) {
      total += *cl.map_shared_rank(&s_rot, r);
      big |= *cl.map_shared_rank(&s_big, r);
    }
    cl.sync();  // every CTA has read every count
    if (threadIdx.x == 0) {
      s_rot = 0;
      s_big = 0;
    }
    // No rotation: converged.  Only rotations with off-orthogonality and angle
    // <= 1e-8: each later rotation changed an earlier pair's inner product by at
    // most 1e-16 relative, so the rows are orthogonal to ~k * 1e-16 (the
    // m * eps tolerance) and the confirming sweep is skipped.
    if (total == 0 || big == 0) converged = true;
  }
  if (with_v) {
    if (warp >= gwarps) rotate_v(par ^ 1);  // the last round's rotations
    cl.sync();
  }
  for (int l = 0; l < R; ++l) {
    const int a = l * cs + rank;
    if (a >= na) break;
    const int i = s_act[a];
    for (int t = threadIdx.x; t < m; t += blockDim.x) {
      if constexpr (DF) {
        const float4 x4 = gl[(long long)l * m + t];
        G[(long long)i * ldg + t] = make_double2(df_val({x4.x, x4.y}) * isc, df_val({x4.z, x4.w}) * isc);
      } else {
        G[(long long)i * ldg + t] = gl[(long long)l * m + t];
      }
    }
    if (with_v)
      for (int t = threadIdx.x; t < n; t += blockDim.x) {
        if constexpr (DF) {
          const float4 x4 = vl[(long long)l * n + t];
          Vt[(long long)i * n + t] = make_double2(df_val({x4.x, x4.y}), df_val({x4.z, x4.w}));
        } else {
          Vt[(long long)i * n + t] = vl[(long long)l * n + t];
        }
      }
  }
  if (with_v && !warm)  // rows that took part in no rotation: the identity's
    for (int i = rank; i < n; i += cs) {
      bool on = false;
      for (int a = threadIdx.x; a < na; a += blockDim.x) on |= s_act[a] == i;
      if (!__syncthreads_or(on))
        for (int t = threadIdx.x; t < n; t += blockDim.x)
          Vt[(long long)i * n + t] = make_double2(t == i ? 1.0 : 0.0, 0.0);
    }
  if (rank == 0) {
    if (amap) {
      for (int a = threadIdx.x; a < na; a += blockDim.x) amap[1 + a] = s_act[a];
      if (threadIdx.x == 0) amap[0] = na;
    }
    if (threadIdx.x == 0) {
      if (sweeps_used) *sweeps_used = sweep;
      atomicAdd(&st->jacobi_calls, 1);
      atomicAdd(&st->jacobi_sweeps, sweep);
      if (!converged) atomicAdd(&st->jacobi_unconverged, 1);
    }
  }
  cl.sync();  // no CTA leaves while another may still read its shared memory
}

// Vt (n x n) = the logged rotations applied to the identity (warm: to Vt as
// it is, in place), one CTA per column q (columns are independent: a CTA
// reads and writes its own column only): thread p applies pair p of every
// round, rounds in order, the column held in shared memory.  The log covers
// the active rows (amap[0] of them, amap[1 + a] the row of active row a).
// Rotation c = 2 marks a pair that was not rotated.  The next LOOK rounds'
// records are on their way while one is applied: a round is a load from
// memory, a rotation and a block barrier, and the load is the longest.
__global__ void jacobi_replay_kernel(cplx* __restrict__ Vt, int n, const double4_16a* __restrict__ log,
                                     const int* __restrict__ amap, const int* __restrict__ sweeps_used, int warm) {
  extern __shared__ cplx col[];
  const int q = blockIdx.x;
  const int na = amap[0];
  for (int a = threadIdx.x; a < na; a += blockDim.x) {
    const int i = amap[1 + a];
    col[a] = warm ? Vt[(long long)i * n + q] : make_double2(i == q ? 1.0 : 0.0, 0.0);
  }
  if (!warm)  // rows left out keep the identity's
    for (int i = threadIdx.x; i < n; i += blockDim.x) Vt[(long long)i * n + q] = make_double2(i == q ? 1.0 : 0.0, 0.0);
  __syncthreads();
  const int sweeps = *sweeps_used;
  const int np = (na + 1) & ~1;
  const int rounds = np - 1, npairs = np / 2;
  const int p = threadIdx.x;
  const long long steps = na < 2 ? 0 : (long long)sweeps * rounds;
  constexpr int LOOK = 8;
  double4_16a rec[LOOK];
#pragma unroll
  for (int u = 0; u < LOOK; ++u) {
    rec[u] = make_double4_16a(2.0, 0.0, 0.0, 0.0);
    if (p < npairs && u < steps) rec[u] = log[(long long)u * npairs + p];
  }
  int r = 0;
  for (long long st0 = 0; st0 < steps; st0 += LOOK) {
#pragma unroll
    for (int u = 0; u < LOOK; ++u) {
      const long long st = st0 + u;
      if (st < steps) {
        const double4_16a c = rec[u];
        if (p < npairs && st + LOOK < steps) rec[u] = log[(st + LOOK) * npairs + p];
        if (p < npairs && c.x < 1.5) {
          int i, j;
          pair_of(r, p, np, rounds, &i, &j);
          rotate_elem(Rot<double>{c.x, c.y, c.z}, col[i], col[j]);
        }
        if (++r == rounds) r = 0;
        __syncthreads();
      }
    }
  }
  for (int a = threadIdx.x; a < na; a += blockDim.x) Vt[(long long)amap[1 + a] * n + q] = col[a];
}

// Right-looking Cholesky G = R^H R of the Hermitian n x n G (upper triangle
// used) with dropped pivots (d <= tol * max diagonal: row of R zero), carried
// out on the augmented rows [G | I], which leaves L^{-1} = R^{-H} beside R (zero
// rows and columns for dropped pivots): row j of the working matrix holds the
// Schur complement right of its diagonal and its row of L^{-1} left of it, so
// the augmented part costs no storage and no further steps (a back
// substitution of its own took 35 us, with no pivot dropped 196 us at n = 116,
// a serial chain of n warp reductions per column).
//
// Blocked by CH_NB rows.  Rows of the working copy W live in the cluster's
// shared memory (row i in CTA i mod csize, csize a power of two).  For the
// block of rows j0 .. j0+nb-1 each CTA factors the nb x nb diagonal block
// (every CTA the same arithmetic, so the same pivots) and the block's entries
// in the other columns it owns (l mod csize = rank), one barrier of four warps per row, and
// writes its scaled columns into every CTA's copy of the block's rows; after a
// cluster barrier every CTA updates its own rows below the block and writes
// those of the next block straight to the CTAs that factor them.  Bound: the
// serial chain of pivots (each an FP64 reciprocal and a rank-one update, some
// 0.3 us) and the trailing update on the FP64 units of the cluster's SMs.
// Written by its maker, a row needs no round trip through the cluster to be
// gathered (n = 116: 132 -> 98 us, 209 -> 163 us where no pivot is dropped).
constexpr int CH_NB = 8;
constexpr int CH_PANEL = 128;  // threads of the panel's barrier

__global__ void __launch_bounds__(CL_THREADS)
    chol_cluster_kernel(const cplx* __restrict__ G, cplx* __restrict__ Rout, cplx* __restrict__ Lout, int n,
                        double tol) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), cs = (int)cl.num_blocks();
  const int R = (n + cs - 1) / cs;
  extern __shared__ cplx sm[];  // [R x n] own rows of W, then [CH_NB x n] the block's rows of W, then of [L^{-1} R]
  cplx* pan = sm + (long long)R * n;
  cplx* rpan = pan + (long long)CH_NB * n;
  __shared__ double s_max, s_rjj[CH_NB], s_inv[CH_NB];
  __shared__ unsigned s_kept;  // pivots of the block that were not dropped
  for (int l = 0; l < R; ++l) {
    const int i = l * cs + rank;
    if (i >= n) break;
    for (int t = threadIdx.x; t < n; t += CL_THREADS)
      sm[(long long)l * n + t] = t >= i ? G[(long long)i * n + t] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double mx = 0.0;
    for (int l = 0; l < R; ++l) {
      const int i = l * cs + rank;
      if (i >= n) break;
      mx = fmax(mx, sm[(long long)l * n + i].x);
    }
    s_max = mx;
  }
  cl.sync();
  double dmax = 0.0;
  for (int r = 0; r < cs; ++r) dmax = fmax(dmax, *cl.map_shared_rank(&s_max, r));
  const double thr = tol * dmax;
  const int own = cs - 1;  // l & own: the owner of column (or row) l
  for (int j0 = 0; j0 < n; j0 += CH_NB) {
    const int nb = min(CH_NB, n - j0), jn = j0 + nb;
    // columns this CTA works on: the diagonal block (c < nb), then its own
    // columns outside it, left ones (L^{-1}) first
    const int nleft = Lout && j0 > rank ? (j0 - 1 - rank) / cs + 1 : 0;
    const int off = (rank - jn) & own;  // first own column at or after jn is jn + off
    const int nright = jn + off < n ? (n - 1 - (jn + off)) / cs + 1 : 0;
    const int ncol = nb + nleft + nright;
    const unsigned rec = 65536u / ncol + 1;  // e / ncol = e rec >> 16 for e ncol < 65536
    auto col = [&](int c) {
      c -= nb;
      return c < 0 ? jn + c : (c < nleft ? rank + c * cs : jn + off + (c - nleft) * cs);
    };
    if (j0 == 0) {  // the first block's rows of W on those columns, from their owners
      for (int e = threadIdx.x; e < nb * ncol; e += CL_THREADS) {
        const int jj = e / ncol, l = col(e % ncol);
        pan[(long long)jj * n + l] = cl.map_shared_rank(sm, jj & own)[(long long)(jj / cs) * n + l];
      }
      __syncthreads();
    }
    if (threadIdx.x < CH_PANEL) {
      // rows i > j of the block on every column: W[i,l] -= conj(W[j,i]) W[j,l] / d,
      // for l >= i (the Schur complement) and l <= j (L^{-1}, whose column j
      // starts here from 0 with a one in W[j,j]'s place).  Every warp with an
      // element forms 1/d itself: four FP64 instructions against a second barrier.
      for (int jj = 0; jj < nb - 1; ++jj) {
        const int j = j0 + jj, todo = (nb - 1 - jj) * ncol;
        const cplx* pj = pan + (long long)jj * n;
        const double d = pj[j].x;
        // d > thr: the same in every thread; a dropped direction updates nothing
        if (d > thr && (int)(threadIdx.x & ~31u) < todo) {
          auto update = [&](auto over_d) {
            for (int e = threadIdx.x; e < todo; e += CH_PANEL) {
              const int q = (int)((unsigned)e * rec >> 16), i = j + 1 + q, l = col(e - q * ncol);
              if (l > j && l < i) continue;
              cplx* w = pan + (long long)(i - j0) * n + l;
              const bool diag = l == j;
              const cplx g = pj[i], h = diag ? make_double2(1.0, 0.0) : pj[l];
              const cplx v = diag ? make_double2(0.0, 0.0) : *w;
              const double ax = over_d(g.x), ay = over_d(g.y);
              *w = make_double2(fma(-ax, h.x, fma(-ay, h.y, v.x)), fma(-ax, h.y, fma(ay, h.x, v.y)));
            }
          };
          if ((unsigned)(__double2hiint(d) >> 20) - 3u < 2040u) {  // 2^-1020 <= d < 2^1020, on the integer pipe
            const double inv = rcp64_pos(d);
            update([inv](double x) { return x * inv; });
          } else {  // 1/d overflows or loses bits where x / d does not
            const double inv = rsqrt(d);
            update([inv](double x) { return x * inv * inv; });
          }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(CH_PANEL) : "memory");
      }
      if (threadIdx.x < nb) {  // r = d / sqrt(d) and 1/r, zero for a dropped direction
        const double d = pan[(long long)threadIdx.x * n + j0 + threadIdx.x].x;
        const bool keep = d > thr;
        const double inv = keep ? rsqrt64(d) : 0.0;
        s_inv[threadIdx.x] = inv;
        s_rjj[threadIdx.x] = keep ? d * inv : 0.0;
        const unsigned mask = __ballot_sync((1u << nb) - 1u, keep);
        if (threadIdx.x == 0) s_kept = mask;
      }
      asm volatile("bar.sync 1, %0;" ::"n"(CH_PANEL) : "memory");
      // the block's rows scaled: R right of the diagonal, L^{-1} left of it and on
      // it; the diagonal block is every CTA's own, the other columns go to all
      for (int e = threadIdx.x; e < nb * ncol; e += CH_PANEL) {
        const int jj = (int)((unsigned)e * rec >> 16), c = e - jj * ncol, l = col(c);
        const double inv = s_inv[jj];
        const cplx g = pan[(long long)jj * n + l];
        cplx v = make_double2(g.x * inv, g.y * inv);
        if (l == j0 + jj) v = make_double2(inv, 0.0);
        if (!(s_kept >> jj & 1u)) v = make_double2(0.0, 0.0);
        cplx* to = rpan + (long long)jj * n + l;
        if (c < nb) {
          *to = v;
        } else {
#pragma unroll 8
          for (int r = 0; r < cs; ++r) *cl.map_shared_rank(to, r) = v;
        }
      }
    }
    cl.sync();  // the block's rows are complete in every CTA, and pan is free
    // the owners store their rows of R and L^{-1}
    for (int jj = 0; jj < nb; ++jj) {
      const int j = j0 + jj;
      if ((j & own) != rank) continue;
      for (int l = threadIdx.x; l < n; l += CL_THREADS) {
        const cplx v = rpan[(long long)jj * n + l], z = make_double2(0.0, 0.0);
        if (Rout) Rout[(long long)j * n + l] = l < j ? z : (l == j ? make_double2(s_rjj[jj], 0.0) : v);
        if (Lout) Lout[(long long)j * n + l] = l > j ? z : v;
      }
    }
    // below the next block's diagonal nothing has been written yet: zero, which
    // is what L^{-1} keeps there for a dropped pivot
    if (threadIdx.x < CH_NB * CH_NB) {
      const int jj = threadIdx.x / CH_NB, c = threadIdx.x % CH_NB;
      if (c < jj && jn + jj < n) pan[(long long)jj * n + jn + c] = make_double2(0.0, 0.0);
    }
    // own rows below the block, on the columns l < jn (L^{-1}: the block's own
    // columns start here, from the rows at and below them) and l >= i: the
    // (row, column) pairs of all own rows, row after row, spread over the threads
    const unsigned kept = s_kept;
    const int left = Lout ? jn : 0;
    int lr = jn > rank ? (jn - rank + cs - 1) / cs : 0;  // first own row at or after jn
    int i = lr * cs + rank, len = left + n - i, e = threadIdx.x;
    while (true) {
      while (i < n && e >= len) {
        e -= len;
        len -= cs;
        i += cs;
        ++lr;
      }
      if (i >= n) break;
      const int l = e < left ? e : i + (e - left);
      cplx* w = sm + (long long)lr * n + l;
      const bool fresh = l >= j0 && l < jn;
      cplx v = fresh ? make_double2(0.0, 0.0) : *w;
      const unsigned use = fresh ? kept & ~((1u << (l - j0)) - 1u) : kept;
#pragma unroll
      for (int jj = 0; jj < CH_NB; ++jj) {
        if (!(use >> jj & 1u)) continue;
        const cplx a = rpan[(long long)jj * n + i], b = rpan[(long long)jj * n + l];
        v.x = fma(-a.x, b.x, fma(-a.y, b.y, v.x));
        v.y = fma(-a.x, b.y, fma(a.y, b.x, v.y));
      }
      if (i >= jn + CH_NB) {
        *w = v;
      } else {  // a row of the next block: to the CTAs that work on its column
        cplx* to = pan + (long long)(i - jn) * n + l;
        if (l >= jn && l < jn + CH_NB) {
#pragma unroll 8
          for (int r = 0; r < cs; ++r) *cl.map_shared_rank(to, r) = v;
        } else {
          *cl.map_shared_rank(to, l & own) = v;
        }
      }
      e += CL_THREADS;
    }
    cl.sync();  // the next block's rows have arrived; rpan is read no more
  }
}

}  // namespace

template <bool DF, bool V>
static const void* jacobi_fn(int m) {
  if (m <= 128) return (const void*)jacobi_cluster_kernel<DF, 4, V>;
  return m <= 256 ? (const void*)jacobi_cluster_kernel<DF, 8, V> : (const void*)jacobi_cluster_kernel<DF, 0, V>;
}

// the kernel for rows of m elements; v: Vt beside the rows
static const void* jacobi_fn(bool df, bool v, int m) {
  return df ? jacobi_fn<true, true>(m) : (v ? jacobi_fn<false, true>(m) : jacobi_fn<false, false>(m));
}

static cudaError_t cluster_init() {
  if (g_csize) return cudaSuccess;
  cudaError_t e;
  auto prepare = [](const void* f) {
    cudaError_t r = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return r != cudaSuccess ? r : cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, CL_SMEM);
  };
  for (int m : {128, 256, 257})
    for (const void* f : {jacobi_fn(false, false, m), jacobi_fn(false, true, m), jacobi_fn(true, true, m)})
      if ((e = prepare(f)) != cudaSuccess) return e;
  if ((e = prepare((const void*)chol_cluster_kernel)) != cudaSuccess) return e;
  // 16 CTAs per cluster when the hardware can place such a cluster, else 8
  int csize = 8;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 16;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = CL_SMEM;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int nclusters = 0;
  if (cudaOccupancyMaxActiveClusters(&nclusters, jacobi_fn(false, false, 257), &cfg) == cudaSuccess && nclusters >= 1)
    csize = 16;
  g_clusters = nclusters;
  cudaGetLastError();  // a refused query leaves no error behind
  g_csize = csize;
  return cudaSuccess;
}

cudaError_t fp64_cluster_init() { return cluster_init(); }

static cudaError_t launch_cluster(const void* fn, void** args, size_t smem, cudaStream_t s, int threads = CL_THREADS,
                                  int csize = 0, int nclusters = 1) {
  if (csize == 0) csize = g_csize;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = csize;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.gridDim = dim3(csize * nclusters);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

// dynamic shared memory of a CTA, 0 where the rows do not fit a cluster of cs
static size_t jacobi_smem(int n, int m, bool vt_in_smem, int cs) {
  const long long R = (n + cs - 1) / cs, npairs = (n + 1) / 2;
  if (R > 2 * JC_MAXP || (npairs + cs - 1) / cs > JC_MAXP || n > JC_MAXP * 2 * 16) return 0;
  const long long b =
      std::max(R * ((long long)m + (vt_in_smem ? n : 0)) * (long long)sizeof(cplx), n * (long long)sizeof(double));
  return b <= CL_SMEM ? (size_t)b : 0;
}

bool jacobi_cluster_fits(int n, int m, bool vt_in_smem) {
  if (n < 32) return false;
  if (cluster_init() != cudaSuccess) return false;
  return jacobi_smem(n, m, vt_in_smem, g_csize) > 0;
}

// the rotation records (one double4_16a = two complex slots per pair), then
// the map of the active rows
static long long jacobi_log_slots(int n, int max_sweeps) {
  const long long np = (n + 1) & ~1;
  return (long long)max_sweeps * (np - 1) * (np / 2) * 2;
}
long long jacobi_log_elems(int n, int max_sweeps) {
  return jacobi_log_slots(n, max_sweeps) + (n + 1 + 3) / 4;
}

static int jacobi_threads(int n, int cs, bool with_v) {
  const int own = ((n + 1) / 2 + cs - 1) / cs;  // pairs per CTA, a warp each (two with V)
  return (with_v ? 2 * own : own) <= 8 ? 256 : 512;
}

cudaError_t jacobi_cluster(cudaStream_t s, cplx* G, int n, int m, long long ldg, cplx* Vt, int max_sweeps,
                           DevStatus* st, cplx* rotlog, int* sweeps_used, bool warm_v, bool dfloat) {
  cudaError_t e;
  if ((e = cluster_init()) != cudaSuccess) return e;
  // double-float rows only where a V comes with them (the projector cores);
  // their dot products resolve orthogonality to about m 2^-48, so pairs are
  // left alone below m 2^-44 (FP64: m eps)
  const bool df = dfloat && Vt;
  // V beside the rows (double-float, or no log to replay it from)
  const bool v_in = Vt && (df || !rotlog) && jacobi_smem(n, m, true, g_csize) > 0;
  if (Vt && !v_in && !rotlog) return cudaErrorInvalidValue;
  const bool replay = Vt && !v_in;
  cplx* Vin = v_in ? Vt : nullptr;
  double4_16a* logp = replay ? (double4_16a*)rotlog : nullptr;
  int* amap = replay ? (int*)(rotlog + jacobi_log_slots(n, max_sweeps)) : nullptr;
  int* su = replay ? sweeps_used : nullptr;
  size_t smem = jacobi_smem(n, m, v_in, g_csize);
  float tol = df ? (float)((double)m * 0x1p-44) : (float)((double)m * 2.220446049250313e-16);
  int warm = warm_v && Vt ? 1 : 0;
  long long stride = 0;
  void* args[] = {&G, &n, &m, &ldg, &stride, &Vin, &max_sweeps, &tol, &logp, &amap, &su, &st, &warm};
  e = launch_cluster(jacobi_fn(df, v_in, m), args, smem, s, jacobi_threads(n, g_csize, v_in));
  count_launch();
  if (e != cudaSuccess || !replay) return e;
  const int npairs = ((n + 1) & ~1) / 2;
  const int threads = (npairs + 31) / 32 * 32;
  jacobi_replay_kernel<<<n, threads, n * sizeof(cplx), s>>>(Vt, n, (const double4_16a*)rotlog, amap, sweeps_used,
                                                          warm);
  count_launch();
  return cudaGetLastError();
}

bool jacobi_batch_fits(int n) {
  return n >= 1 && cluster_init() == cudaSuccess && jacobi_smem(n, n, false, g_csize) > 0;
}

// Singular values only of `count` matrices (matrix b at G + b * strideG), one
// cluster each in one launch.  Clusters of 8 where the device does not hold as
// many of 16 at once: the FP64 units of the SMs in use bound the kernel, and the
// 16 corners of a 2x2 cell on 8 CTAs each take 128 SMs in one wave.
cudaError_t jacobi_cluster_batch(cudaStream_t s, cplx* G, int n, int m, long long ldg, long long strideG, int count,
                                 int max_sweeps, DevStatus* st) {
  cudaError_t e;
  if ((e = cluster_init()) != cudaSuccess) return e;
  int cs = g_csize;
  if (cs == 16 && count > g_clusters && jacobi_smem(n, m, false, 8) > 0) cs = 8;
  size_t smem = jacobi_smem(n, m, false, cs);
  cplx* Vin = nullptr;
  double4_16a* logp = nullptr;
  int *amap = nullptr, *su = nullptr, warm = 0;
  float tol = (float)((double)m * 2.220446049250313e-16);
  void* args[] = {&G, &n, &m, &ldg, &strideG, &Vin, &max_sweeps, &tol, &logp, &amap, &su, &st, &warm};
  e = launch_cluster(jacobi_fn(false, false, m), args, smem, s, jacobi_threads(n, cs, false), cs, count);
  count_launch();
  return e;
}

bool chol_cluster_fits(int n) {
  if (n < 32) return false;
  if (cluster_init() != cudaSuccess) return false;
  const long long R = (n + g_csize - 1) / g_csize;
  return (R + 2 * CH_NB) * n * (long long)sizeof(cplx) <= CL_SMEM;
}

cudaError_t chol_cluster(cudaStream_t s, const cplx* G, cplx* R, cplx* Linv, int n, double tol) {
  cudaError_t e;
  if ((e = cluster_init()) != cudaSuccess) return e;
  const long long rows = (n + g_csize - 1) / g_csize;
  const size_t smem = (size_t)((rows + 2 * CH_NB) * n * sizeof(cplx));
  void* args[] = {&G, &R, &Linv, &n, &tol};
  e = launch_cluster((const void*)chol_cluster_kernel, args, smem, s);
  count_launch();
  return e;
}
