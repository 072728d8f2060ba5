// Stage 3 of small frames: a group of lanes per ray.
//
// A frame with few active pixels leaves most of the chip idle, and its time is
// one ray's chain of right-hand sides.  Here the lanes of a group share a ray:
// each takes a slab of the control points, the slabs' sums are exchanged by
// shuffles, and all lanes follow the ray's steps.  The samples of an accepted
// step are independent of each other, so each lane evaluates the scalar of one
// of them, and Alg. 1 then runs through them in order.  Same steps, samples
// and compositing as K5, or K5t and the shading pass (SPLIT).
//
// FP32 (k5_coop): four lanes, one u index each; the sums keep their order (k,
// then j within a lane, then i), so the image is that of the one-lane kernels.
// Bound by latency: a quarter of the loads and multiply-adds per right-hand
// side.  A 64 x 64 tile of the cube: 515 us a frame before, 279 with it, 243
// since the later cull and transfer function; the 256 x 256 bar 255 -> 197,
// then 165 (frames among others).  FP64 is in k_coop64.cuh.
#pragma once

#include "k_integrate.cuh"

namespace ivv {

constexpr int kCoopLanes32 = 4, kCoopLanes64 = 16;    // lanes per ray

// Element, local coordinate and scale of one direction (as eval_block).
__device__ __forceinline__ int coop_locate(const DevVolume& V, const BlockInfo& B, int d, float x, float& loc,
                                           float& sc) {
  if ((B.uniform >> d) & 1) {
    const float xs = x * (float)B.nseg[d];
    int k = (int)xs;
    k = k < B.nseg[d] - 1 ? k : B.nseg[d] - 1;
    loc = xs - (float)k;
    sc = (float)B.nseg[d];
    return k;
  }
  return locate<float>(V.brk32 + B.brk_off[d], B.nseg[d], x, loc, sc);
}

// phi and J at p (in [0,1]^3), the slabs shared by the group's lanes (gm: its lanes of the
// warp, g: this lane in it); every lane gets the result.
template <int P>
__device__ __forceinline__ void coop_map(const DevVolume& V, const BlockInfo& B, const float p[3], unsigned gm, int g,
                                         float phi[3], float J[3][3]) {
  constexpr int N = P + 1, G = kCoopLanes32;
  float loc[3], sc[3];
  int e[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) e[d] = coop_locate(V, B, d, p[d], loc[d], sc[d]);
  const size_t eid = (size_t)(B.elem_off + (e[2] * B.nseg[1] + e[1]) * B.nseg[0] + e[0]);
  float bu[N], dbu[N], bv[N], dbv[N], bw[N], dbw[N];
  bernstein<P, float>(loc[0], bu, dbu);
  bernstein<P, float>(loc[1], bv, dbv);
  bernstein<P, float>(loc[2], bw, dbw);
  // the slab of u index g (the last lane repeats one where there are fewer)
  const float4* cp = V.elem32 + (eid * N + (g < N ? g : N - 1)) * (N * N);
  float s00[3] = {0, 0, 0}, s01[3] = {0, 0, 0}, s10[3] = {0, 0, 0};
#pragma unroll
  for (int j = 0; j < N; ++j) {
    float4 row[N];
    ldg_row<N>(cp + j * N, row);
    float t0[3] = {0, 0, 0}, t1[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const float c[3] = {row[k].x, row[k].y, row[k].z};
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        t0[r] = __fmaf_rn(bw[k], c[r], t0[r]);
        t1[r] = __fmaf_rn(dbw[k], c[r], t1[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      s00[r] = __fmaf_rn(bv[j], t0[r], s00[r]);
      s01[r] = __fmaf_rn(dbv[j], t0[r], s01[r]);
      s10[r] = __fmaf_rn(bv[j], t1[r], s10[r]);
    }
  }
  const float4 og = ElemPtr<float>::org(V, eid);
  const float o[3] = {og.x, og.y, og.z};
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    float f = 0.f, fu = 0.f, fv = 0.f, fw = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) {                     // the u sums in their order
      const float a = __shfl_sync(gm, s00[r], i, G), b = __shfl_sync(gm, s01[r], i, G),
                  c = __shfl_sync(gm, s10[r], i, G);
      f = __fmaf_rn(bu[i], a, f);
      fu = __fmaf_rn(dbu[i], a, fu);
      fv = __fmaf_rn(bu[i], b, fv);
      fw = __fmaf_rn(bu[i], c, fw);
    }
    phi[r] = f + o[r];
    J[r][0] = fu * sc[0];
    J[r][1] = fv * sc[1];
    J[r][2] = fw * sc[2];
  }
}

// The scalar at p, evaluated by one lane: as the shading pass rounds it
// (SPLIT), or the fused integrator.
template <int P, bool SPLIT>
__device__ __forceinline__ float coop_scalar(const DevVolume& V, const BlockInfo& B, const float p[3]) {
  if (V.mode == IVV_SCALAR_CP) return eval_rho_cp<P>(V, B, p);
  float phi[3], J[3][3], rc;
  eval_block<P, float, false>(V, B, p, phi, J, rc);
  if (SPLIT && V.mode == IVV_SCALAR_DETJ) return det_cofactor(J);
  if (SPLIT && V.mode == IVV_SCALAR_QUALITY) return quality_cofactor(J);
  return scalar_at<P, float>(V, B, V.mode, p, J, 0.f);
}
// n_active beyond coop_max: the frame is left to the one-lane-per-ray kernels,
// which in turn leave frames up to coop_max to this one.
template <int P, bool MIXED, bool SPLIT>
__global__ void __launch_bounds__(32) k5_coop(DevVolume V, DevCamera<float> cam, DevTF tf, IntegrateArgs args,
                                              const float4* __restrict__ pair_in, const float4* __restrict__ pair_out,
                                              const int* __restrict__ pair_block, const int* __restrict__ pair_count,
                                              const int* __restrict__ active, const int* __restrict__ n_active,
                                              int* __restrict__ queue_head, float4* __restrict__ out,
                                              DevStats* __restrict__ st) {
  typedef float R;
  typedef float4 V4;
  constexpr int G = kCoopLanes32, kGroups = 32 / G;
  __shared__ TfTable s_tf;
  tf_load(s_tf, tf);
  pdl_wait();
  const int nact = *n_active;
  if (nact == 0 || nact > args.coop_max) return;
  const int lane = threadIdx.x, g = lane & (G - 1);
  const unsigned gm = ((1u << G) - 1u) << (lane - g);
  const int npix = args.npix;
  const R tol = R(args.rk_tol), cc = R(args.c), early = R(args.early_alpha), ds = R(args.ds);
  const R tail_eps = R(1e-12) * R(V.diag);
  const R hmin = R(1e-7) * ds, hmax = R(args.max_step_samples) * ds;
  unsigned long long c_fp64 = 0, c_cap = 0;
  // the first items in the order of the warps (neighbouring pixels share a
  // warp, and one warp per SM fills first), further ones from the queue
  int item = blockIdx.x * kGroups + lane / G;
  while (item < nact) {
    const int pix = __ldg(active + item);
    R o[3], d[3];
    make_ray<R>(cam, cam.x0 + pix % cam.w, cam.y0 + pix / cam.w, o, d);
    Acc<R> acc;
    acc.C[0] = acc.C[1] = acc.C[2] = acc.a = R(0);
    const int np = __ldg(pair_count + pix);
    bool done = false;
    for (int q = 0; q < np && !done; ++q) {
      const size_t slot = (size_t)q * npix + pix;
      const V4 pi = pair_in[slot], po = pair_out[slot];
      const R L = R(po.x) - R(pi.x);
      if (!(L > R(0))) continue;
      const BlockInfo B = V.blocks[__ldg(pair_block + slot)];
      const R fl = floor(L / ds);
      const int nsamp = (int)fl, nlast = nsamp + ((L - fl * ds > tail_eps) ? 1 : 0);
      R g_in[3], p[3] = {R(pi.y), R(pi.z), R(pi.w)}, k1[3], ka[3], kb[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) g_in[r] = o[r] + R(pi.x) * d[r];
      R s = R(0), s_last = R(0), h = ds, hh = R(0), rho_prev = R(0);
      int j = 1, steps = 0, stage = 0;
      for (;;) {
        R x[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          R v;
          if (stage == 0) v = p[r];
          else if (stage == 1) v = bs3_q2<R>(p[r], hh, k1[r]);
          else if (stage == 2) v = bs3_q3<R>(p[r], hh, ka[r]);
          else v = ka[r];
          x[r] = v < R(0) ? R(0) : (v > R(1) ? R(1) : v);
        }
        R W[3], phi[3], J[3][3];
        coop_map<P>(V, B, x, gm, g, phi, J);
        rhs_solve<R, MIXED>(B, phi, J, g_in, d, cc, W, c_fp64);
        if (stage == 0) {
          k1[0] = W[0]; k1[1] = W[1]; k1[2] = W[2];
          if (j > nlast) break;                         // zero-length remainder: pair done
          rho_prev = coop_scalar<P, SPLIT>(V, B, x);
        } else if (stage == 1) {
          ka[0] = W[0]; ka[1] = W[1]; ka[2] = W[2];
          stage = 2;
          continue;
        } else if (stage == 2) {
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            const R k2 = ka[r];
            ka[r] = bs3_pn<R>(p[r], hh, k1[r], k2, W[r]);
            kb[r] = bs3_e3<R>(k1[r], k2, W[r]);
          }
          stage = 3;
          continue;
        } else {
          R err = R(0);
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            const R ae = fabs(bs3_err<R>(hh, kb[r], W[r]));
            err = ae > err ? ae : err;
          }
          ++steps;
          const bool capped = steps >= args.max_steps;
          if (err <= tol || hh <= hmin || capped) {
            if (capped) ++c_cap;
            const R s1 = last_end(s, hh, L);
            if (capped && !SPLIT) break;                // the fused integrator leaves the rest of the pair out
            // the samples in (s, s1], one per lane (capped: all that are left,
            // at the step's end), then Alg. 1 through them in order
            for (;;) {
              const int jl = j + g;
              const R st_ = (jl <= nsamp) ? R(jl) * ds : L;
              const bool in = jl <= nlast && (capped || !(st_ > s1));
              const unsigned have = __ballot_sync(gm, in) >> (lane - g);
              const int m = __popc(have & ((1u << G) - 1u));
              if (m == 0) break;
              R rho = R(0);
              if (in) {
                R xs[3] = {x[0], x[1], x[2]};
                if (!(capped || st_ >= s1)) {
                  const R th = (st_ - s) / hh;
#pragma unroll
                  for (int r = 0; r < 3; ++r) {
                    const R v = hermite<R>(th, hh, p[r], k1[r], x[r], W[r]);
                    xs[r] = v < R(0) ? R(0) : (v > R(1) ? R(1) : v);
                  }
                }
                rho = coop_scalar<P, SPLIT>(V, B, xs);
              }
              __syncwarp(gm);
              for (int t = 0; t < m && !done; ++t) {
                const R rj = __shfl_sync(gm, rho, t, G);
                const R sj = (j + t <= nsamp) ? R(j + t) * ds : L;
                composite_interval<R>(s_tf.view(), tf, args.K, rho_prev, rj, sj - s_last, acc);
                rho_prev = rj;
                s_last = sj;
                done = acc.a >= early;
              }
              j += m;
              if (done || m < G) break;
            }
            if (done || j > nlast) break;               // early termination, or the pair is done
#pragma unroll
            for (int r = 0; r < 3; ++r) {
              p[r] = x[r];
              k1[r] = W[r];
            }
            s = s1;
            R fac = err > R(0) ? R(0.9) * pow_third<R>(tol / err) : R(5);
            fac = fac < R(0.2) ? R(0.2) : (fac > R(5) ? R(5) : fac);
            h = hh * fac;
          } else {
            const R fac = R(0.9) * pow_third<R>(tol / err);
            h = hh * (fac < R(0.2) ? R(0.2) : fac);
          }
        }
        const R rem = L - s;
        hh = h < hmax ? h : hmax;
        hh = hh < rem ? hh : rem;
        stage = 1;
      }
    }
    if (g == 0) out[pix] = make_float4((float)acc.C[0], (float)acc.C[1], (float)acc.C[2], (float)acc.a);
    if (g == 0) item = (int)gridDim.x * kGroups + atomicAdd(queue_head, 1);
    item = __shfl_sync(gm, item, 0, G);
  }
  if (g == 0) {
    if (MIXED && c_fp64) atomicAdd(&st->fp64_solves, c_fp64);
    if (c_cap) atomicAdd(&st->step_cap, c_cap);
  }
}

template <typename K, typename R, typename V4>
void launch_coop_k(K kern, int& per_sm, const DevVolume& V, const DevCamera<R>& cam, const DevTF& tf,
                   const IntegrateArgs& a, const V4* pin, const V4* pout, const int* pblk, const int* pcnt,
                   const int* active, const int* n_active, int* queue_head, float4* out, DevStats* st, int num_sms,
                   cudaStream_t s) {
  if (per_sm < 0) {
    int n = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, 32, 0);
    per_sm = n < 1 ? 1 : n;
  }
  const int groups = 32 / (sizeof(R) == 4 ? kCoopLanes32 : kCoopLanes64);
  const int most = a.npix < a.coop_max ? a.npix : a.coop_max;
  int grid = num_sms * per_sm;
  const int useful = (most + groups - 1) / groups;
  grid = grid < useful ? grid : (useful > 0 ? useful : 1);
  launch_pdl(kern, dim3(grid), dim3(32), s, V, cam, tf, a, pin, pout, pblk, pcnt, active, n_active, queue_head, out,
             st);
}

}  // namespace ivv
