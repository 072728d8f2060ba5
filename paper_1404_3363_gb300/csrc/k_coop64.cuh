// Stage 3 of FP64 frames with few active pixels: sixteen lanes per ray (see
// k_coop.cuh).
//
// GB300 has half a double unit per SM sub-partition: a double instruction of
// a warp occupies it for 64 cycles however many of its lanes need it, so what
// counts is the number of double instructions per right-hand side, and that
// every sub-partition has a ray.  A lane therefore owns one entry of
// everything: row (i, j) of the control points, one direction's basis (its
// coordinate's), one entry of (phi, J), one component of the cross products of
// the solve, one sample of a step and one sub-sample of an interval; shuffles,
// which do not use that unit, carry the rest.  About 95 double instructions
// per right-hand side instead of 780 in the one-lane form (and 170 with eight
// lanes that only share the contraction).  Clamps compare the bits as
// integers, the degree and the element counts scale the slope W once, and the
// step control starts its cube root from FP32 and refines it.
//
// 64 x 64 cube at tol 1e-8 (1111 rays, 441 k right-hand sides): 37.4 ms with
// one lane per ray, 15.4 with eight that share the contraction, 12.8 with one
// coordinate per lane, 8.1 in this form.  What is left is the longest ray's
// chain: an SM is busy 36 % of the kernel, and then at half the FP64 rate.
#pragma once

#include "k_coop.cuh"
#include "step_factor.h"

namespace ivv {

// Four doubles with one 256-bit read-only load (32-byte aligned).
__device__ __forceinline__ Dbl4 ldg_d4(const Dbl4* p) {
  Dbl4 r;
  asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(r.x), "=d"(r.y), "=d"(r.z), "=d"(r.w) : "l"(p));
  return r;
}

// x clamped to [0, 1] by integer compares (NaN of either sign ends at a bound).
__device__ __forceinline__ double clamp01_bits(double x) {
  const long long b = __double_as_longlong(x);
  return b < 0 ? 0.0 : (b > 0x3ff0000000000000ll ? 1.0 : x);
}

// Element and local coordinate of x in [0, 1] in direction d.
__device__ __forceinline__ int coop_locate64(const DevVolume& V, const BlockInfo& B, int d, double x, double& loc,
                                             double& sc) {
  const int nseg = d == 0 ? B.nseg[0] : (d == 1 ? B.nseg[1] : B.nseg[2]);
  const int off = d == 0 ? B.brk_off[0] : (d == 1 ? B.brk_off[1] : B.brk_off[2]);
  if ((B.uniform >> d) & 1) {
    sc = (double)nseg;
    if (nseg == 1) {
      loc = x;
      return 0;
    }
    const double xs = x * sc;
    int k = (int)xs;
    k = k < nseg - 1 ? k : nseg - 1;
    loc = xs - (double)k;
    return k;
  }
  return locate<double>(V.brk64 + off, nseg, x, loc, sc);
}

// Bernstein values and, without the factor P, derivatives by de Casteljau.
template <int P>
__device__ __forceinline__ void bernstein_dc(double x, double b[4], double d[4]) {
  const double y = 1.0 - x;
  if (P == 2) {
    const double xy = x * y;
    b[0] = y * y; b[1] = xy + xy; b[2] = x * x; b[3] = 0.0;
    d[0] = -y; d[1] = y - x; d[2] = x; d[3] = 0.0;
  } else {
    const double xy = x * y, q0 = y * y, q1 = xy + xy, q2 = x * x;
    b[0] = y * q0; b[1] = fma(y, q1, x * q0); b[2] = fma(y, q2, x * q1); b[3] = x * q2;
    d[0] = -q0; d[1] = q0 - q1; d[2] = q1 - q2; d[3] = q2;
  }
}

// v[m] for a lane-dependent m, by selects.
__device__ __forceinline__ double pick4(const double v[4], int m) {
  const double lo = m & 1 ? v[1] : v[0], hi = m & 1 ? v[3] : v[2];
  return m & 2 ? hi : lo;
}

// W_c at the point whose coordinate c this lane holds in x (c = min(g mod 4,
// 2); gm: the group's lanes of the warp, g: this lane in it).
template <int P>
__device__ __forceinline__ double coop_rhs64(const DevVolume& V, const BlockInfo& B, double x, double g_in, double d,
                                             double cc, unsigned gm, int g) {
  constexpr int N = P + 1, G = kCoopLanes64;
  const int a = g >> 2, c4 = g & 3, c = c4 < 2 ? c4 : 2;
  double loc, sc, b[4], db[4];
  const int ed = coop_locate64(V, B, c, x, loc, sc);
  bernstein_dc<P>(loc, b, db);
  const int e0 = __shfl_sync(gm, ed, 0, G), e1 = __shfl_sync(gm, ed, 1, G), e2 = __shfl_sync(gm, ed, 2, G);
  const size_t eid = (size_t)(B.elem_off + (e2 * B.nseg[1] + e1) * B.nseg[0] + e0);
  // this lane's row: u index a, v index c4 (a valid row with weight zero past
  // the last index); lane 4 m + r holds index m of direction r's basis
  const Dbl4* cp = V.elem64 + ((eid * N + (a < N ? a : N - 1)) * N + (c4 < N ? c4 : N - 1)) * N;
  const double bm = pick4(b, a), dm = pick4(db, a);
  const double bu = __shfl_sync(gm, bm, 4 * a, G), du = __shfl_sync(gm, dm, 4 * a, G);
  const double bv = __shfl_sync(gm, bm, 4 * c4 + 1, G), dv = __shfl_sync(gm, dm, 4 * c4 + 1, G);
  double t0[3] = {0, 0, 0}, t1[3] = {0, 0, 0};
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const Dbl4 p4 = ldg_d4(cp + k);
    const double bw = __shfl_sync(gm, b[k], 2, G), dw = __shfl_sync(gm, db[k], 2, G);
    const double cr[3] = {p4.x, p4.y, p4.z};
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      t0[r] = k ? fma(bw, cr[r], t0[r]) : bw * cr[r];
      t1[r] = k ? fma(dw, cr[r], t1[r]) : dw * cr[r];
    }
  }
  const double w00 = bu * bv, w10 = du * bv, w01 = bu * dv;
  // sums over the group: lane (a, c4) ends with entry a of (phi, phi_u, phi_v,
  // phi_w) in coordinate c
  const bool h3 = g & 8, h2 = g & 4, h1 = g & 2, h0 = g & 1;
  double q[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const double f = w00 * t0[r], fu = w10 * t0[r], fv = w01 * t0[r], fw = w00 * t1[r];
    const double s0 = (h3 ? fv : f) + __shfl_xor_sync(gm, h3 ? f : fv, 8, G);
    const double s1 = (h3 ? fw : fu) + __shfl_xor_sync(gm, h3 ? fu : fw, 8, G);
    q[r] = (h2 ? s1 : s0) + __shfl_xor_sync(gm, h2 ? s0 : s1, 4, G);
  }
  const double m0 = (h1 ? q[2] : q[0]) + __shfl_xor_sync(gm, h1 ? q[0] : q[2], 2, G);
  const double m1 = q[1] + __shfl_xor_sync(gm, q[1], 2, G);
  const double val = (!h1 && h0 ? m1 : m0) + __shfl_xor_sync(gm, h1 || h0 ? m0 : m1, 1, G);
  // V = d + c (e - (e.d) d), e = g_in - phi
  const double phi = __shfl_sync(gm, val, c, G) + __ldg(reinterpret_cast<const double*>(V.org64 + eid) + c);
  const double e = g_in - phi, p_ed = e * d;
  const double dot = __shfl_sync(gm, p_ed, 0, G) + __shfl_sync(gm, p_ed, 1, G) + __shfl_sync(gm, p_ed, 2, G);
  const double v = fma(cc, fma(-dot, d, e), d);
  // W = (v_0 (J_1 x J_2) + v_1 (J_2 x J_0) + v_2 (J_0 x J_1)) / det, J_r row r:
  // this lane takes component m of the product without row c
  const int m = a == 0 ? 0 : a - 1;
  const int n1 = c == 2 ? 0 : c + 1, n2 = c == 0 ? 2 : c - 1, k1 = m == 2 ? 1 : m + 2, k2 = m == 0 ? 3 : m;
  const double j11 = __shfl_sync(gm, val, 4 * k1 + n1, G), j22 = __shfl_sync(gm, val, 4 * k2 + n2, G);
  const double j12 = __shfl_sync(gm, val, 4 * k2 + n1, G), j21 = __shfl_sync(gm, val, 4 * k1 + n2, G);
  const double xm = fma(j11, j22, -(j12 * j21));
  const double td = val * xm, y = v * xm;
  const double det = __shfl_sync(gm, td, 4, G) + __shfl_sync(gm, td, 8, G) + __shfl_sync(gm, td, 12, G);
  const int src = 4 * (c + 1);
  const double num = __shfl_sync(gm, y, src, G) + __shfl_sync(gm, y, src + 1, G) + __shfl_sync(gm, y, src + 2, G);
  return num / (det * (P * sc));          // the slopes above lack the factors P and the element counts
}

// The scalar at p (in [0,1]^3), evaluated by one lane.
template <int P>
__device__ __forceinline__ double coop_scalar(const DevVolume& V, const BlockInfo& B, const double p[3]) {
  constexpr int N = P + 1;
  if (V.mode == IVV_SCALAR_CP) {
    double loc[3], sc[3];
    int e[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) e[d] = coop_locate64(V, B, d, p[d], loc[d], sc[d]);
    const size_t eid = (size_t)(B.elem_off + (e[2] * B.nseg[1] + e[1]) * B.nseg[0] + e[0]);
    double bu[N], bv[N], bw[N], s = 0;
    bernstein_v<P, double>(loc[0], bu);
    bernstein_v<P, double>(loc[1], bv);
    bernstein_v<P, double>(loc[2], bw);
    const Dbl4* cp = V.elem64 + eid * (N * N * N);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      double si = 0;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        double sj = 0;
#pragma unroll
        for (int k = 0; k < N; ++k) sj += bw[k] * __ldg(&cp[(i * N + j) * N + k].w);
        si += bv[j] * sj;
      }
      s += bu[i] * si;
    }
    return s;
  }
  double phi[3], J[3][3], rc;
  eval_block<P, double, false>(V, B, p, phi, J, rc);
  return scalar_at<P, double>(V, B, V.mode, p, J, 0.0);
}

// Sub-sample k of the K of an interval of Alg. 1 (composite_interval_k): its
// opacity, and its colour in col.
__device__ __forceinline__ double coop_subsample(const TfView& t, const DevTF& tf, int K, int k, double rho0,
                                                 double rho1, double dsi, float4& col) {
  const double invK = 1.0 / (double)K, x0 = tf_coord<double>(tf, rho0), x1 = tf_coord<double>(tf, rho1);
  const float x = (float)fma(((double)k + 0.5) * invK, x1 - x0, x0);
  const int e = tf_piece(t, tf.n, x);
  const float4 a = t.a[e], d = t.d[e];
  const float u = x - t.lo[e];
  col = make_float4(fmaf(d.x, u, a.x), fmaf(d.y, u, a.y), fmaf(d.z, u, a.z), fmaf(d.w, u, a.w));
  return 1.0 - exp(-((double)tf.sigma * dsi * invK) * (double)col.w);
}

// n_active beyond coop_max: the frame is left to k5_integrate, which leaves
// frames up to coop_max to this one.
template <int P>
__global__ void __launch_bounds__(32) k5_coop64(DevVolume V, DevCamera<double> cam, DevTF tf, IntegrateArgs args,
                                                const Dbl4* __restrict__ pair_in, const Dbl4* __restrict__ pair_out,
                                                const int* __restrict__ pair_block,
                                                const int* __restrict__ pair_count, const int* __restrict__ active,
                                                const int* __restrict__ n_active, int* __restrict__ queue_head,
                                                float4* __restrict__ out, DevStats* __restrict__ st) {
  constexpr int G = kCoopLanes64, kGroups = 32 / G;
  __shared__ TfTable s_tf;
  tf_load(s_tf, tf);
  pdl_wait();
  const int nact = *n_active;
  if (nact == 0 || nact > args.coop_max) return;
  const int lane = threadIdx.x, g = lane & (G - 1);
  const int c = (g & 3) < 2 ? (g & 3) : 2;          // this lane's coordinate
  const unsigned gm = ((1u << G) - 1u) << (lane - g);
  const int npix = args.npix;
  const double tol = args.rk_tol, cc = args.c, early = args.early_alpha, ds = args.ds;
  const double tail_eps = 1e-12 * (double)V.diag, hmin = 1e-7 * ds, hmax = (double)args.max_step_samples * ds;
  const int K = args.K;
  unsigned long long c_cap = 0;
  // the first items in the order of the warps (neighbouring pixels share a
  // warp), further ones from the queue
  int item = blockIdx.x * kGroups + lane / G;
  while (item < nact) {
    const int pix = __ldg(active + item);
    double o3[3], d3[3];
    make_ray<double>(cam, cam.x0 + pix % cam.w, cam.y0 + pix / cam.w, o3, d3);
    const double o = c == 0 ? o3[0] : (c == 1 ? o3[1] : o3[2]), d = c == 0 ? d3[0] : (c == 1 ? d3[1] : d3[2]);
    double C[3] = {0, 0, 0}, alpha = 0;
    const int np = __ldg(pair_count + pix);
    bool done = false;
    for (int q = 0; q < np && !done; ++q) {
      const size_t slot = (size_t)q * npix + pix;
      const Dbl4 pi = pair_in[slot], po = pair_out[slot];
      const double L = po.x - pi.x;
      if (!(L > 0)) continue;
      const BlockInfo B = V.blocks[__ldg(pair_block + slot)];
      const double fl = floor(L / ds);
      const int nsamp = (int)fl, nlast = nsamp + ((L - fl * ds > tail_eps) ? 1 : 0);
      const double g_in = o + pi.x * d;
      double p = c == 0 ? pi.y : (c == 1 ? pi.z : pi.w), k1 = 0, ka = 0, kb = 0;
      double s = 0, s_last = 0, h = ds, hh = 0, rho_prev = 0;
      int j = 1, steps = 0, stage = 0;
      for (;;) {
        const double x = clamp01_bits(stage == 0   ? p
                                      : stage == 1 ? bs3_q2<double>(p, hh, k1)
                                      : stage == 2 ? bs3_q3<double>(p, hh, ka)
                                                   : ka);
        const double W = coop_rhs64<P>(V, B, x, g_in, d, cc, gm, g);
        if (stage == 0) {
          k1 = W;
          if (j > nlast) break;                         // zero-length remainder: pair done
          const double x3[3] = {__shfl_sync(gm, x, 0, G), __shfl_sync(gm, x, 1, G), __shfl_sync(gm, x, 2, G)};
          rho_prev = coop_scalar<P>(V, B, x3);
        } else if (stage == 1) {
          ka = W;
          stage = 2;
          continue;
        } else if (stage == 2) {
          const double k2 = ka;
          ka = bs3_pn<double>(p, hh, k1, k2, W);
          kb = bs3_e3<double>(k1, k2, W);
          stage = 3;
          continue;
        } else {
          // the largest component of the error: non-negative doubles order as integers
          const long long ae = __double_as_longlong(fabs(bs3_err<double>(hh, kb, W)));
          long long em = 0;
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            const long long t = __shfl_sync(gm, ae, r, G);
            em = t > em && t <= 0x7ff0000000000000ll ? t : em;
          }
          const double err = __longlong_as_double(em);
          ++steps;
          const bool capped = steps >= args.max_steps;
          if (err <= tol || hh <= hmin || capped) {
            if (capped) {
              ++c_cap;                                  // the rest of the pair is left out
              break;
            }
            const double s1 = last_end(s, hh, L);
            // the samples in (s, s1], one per lane, then Alg. 1 through them
            for (;;) {
              const int jl = j + g;
              const double st_ = (jl <= nsamp) ? (double)jl * ds : L;
              const bool in = jl <= nlast && !(st_ > s1);
              const unsigned have = __ballot_sync(gm, in) >> (lane - g);
              const int n = __popc(have & ((1u << G) - 1u));
              if (n == 0) break;
              double xs[3], rho = 0;
              const double th = (st_ - s) / hh;
#pragma unroll
              for (int r = 0; r < 3; ++r) {
                const double pr = __shfl_sync(gm, p, r, G), kr = __shfl_sync(gm, k1, r, G),
                             xr = __shfl_sync(gm, x, r, G), wr = __shfl_sync(gm, W, r, G);
                xs[r] = clamp01_bits(st_ >= s1 ? xr : hermite<double>(th, hh, pr, kr, xr, wr));
              }
              if (in) rho = coop_scalar<P>(V, B, xs);
              __syncwarp(gm);
              // the n intervals' sub-samples, one per lane, then front to back
              const double rho_left = __shfl_up_sync(gm, rho, 1, G);
              const double s_left = g == 0 ? s_last : (double)(jl - 1) * ds;
              const double r0 = g == 0 ? rho_prev : rho_left, dsi = st_ - s_left;
              for (int base = 0; base < n * K && !done; base += G) {
                const int it = base + g, t = it / K, k = it - t * K;
                const double a0 = __shfl_sync(gm, r0, t, G), a1 = __shfl_sync(gm, rho, t, G),
                             al = __shfl_sync(gm, dsi, t, G);
                double w1 = 0;
                float4 col = make_float4(0.f, 0.f, 0.f, 0.f);
                if (it < n * K) w1 = coop_subsample(s_tf.view(), tf, K, k, a0, a1, al, col);
                __syncwarp(gm);
                const int most = n * K - base < G ? n * K - base : G;
                for (int u = 0; u < most && !done; ++u) {
                  const double w = __shfl_sync(gm, w1, u, G) * (1.0 - alpha);
                  C[0] += w * (double)__shfl_sync(gm, col.x, u, G);
                  C[1] += w * (double)__shfl_sync(gm, col.y, u, G);
                  C[2] += w * (double)__shfl_sync(gm, col.z, u, G);
                  alpha += w;
                  if ((base + u + 1) % K == 0) done = alpha >= early;
                }
              }
              rho_prev = __shfl_sync(gm, rho, n - 1, G);
              s_last = __shfl_sync(gm, st_, n - 1, G);
              j += n;
              if (done || n < G) break;
            }
            if (done || j > nlast) break;               // early termination, or the pair is done
            p = x;
            k1 = W;
            s = s1;
            double fac = err > 0 ? coop_step_factor(tol, err) : 5.0;
            fac = fac < 0.2 ? 0.2 : (fac > 5.0 ? 5.0 : fac);
            h = hh * fac;
          } else {
            const double fac = coop_step_factor(tol, err);
            h = hh * (fac < 0.2 ? 0.2 : fac);
          }
        }
        const double rem = L - s;
        hh = h < hmax ? h : hmax;
        hh = hh < rem ? hh : rem;
        stage = 1;
      }
    }
    if (g == 0) {
      out[pix] = make_float4((float)C[0], (float)C[1], (float)C[2], (float)alpha);
      item = (int)gridDim.x * kGroups + atomicAdd(queue_head, 1);
    }
    item = __shfl_sync(gm, item, 0, G);
  }
  if (g == 0 && c_cap) atomicAdd(&st->step_cap, c_cap);
}

}  // namespace ivv
