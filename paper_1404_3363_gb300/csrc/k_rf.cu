// Root-finding ray integration (§5.1, Eqs. 6-7).  Every sample's preimage is
// solved from a start of its own, by damped Newton on F(p) = phi(p) - g_j with
// a halving line search and clamping to [0,1]^3, stopped when ||F|| is below
// rf_tol times the half width of the pixel at the sample's depth (the paper's
// pixel-accuracy criterion).  The samples of a frame are laid out by groups of
// 32 neighbouring active pixels: sample i (over a pixel's pairs, front to
// back) of lane l of group g has the place base[g] + 32 i + l, every group
// padded to its longest pixel.
//   k_rf_groups    -- the samples of every pixel, the longest and the base of
//                     every group (one warp, one atomic per group)
//   k_rf_points    -- learned guess only: world point and block of every place
//                     for the inference (k_mlp_tc.cu), which writes the starts
//   k_rf_solve     -- a warp per group and chunk of samples: start (the block's
//                     parameter centre, the chord point p_in + (s_j / L)
//                     (p_out - p_in), or the learned guess), Newton, scalar
//   k_rf_composite -- per pixel, Alg. 1 with supersampling over its samples
//   k_rf_count, k_scan_* -- samples per active pixel and their scan for the
//                     split ODE integration after stage-2 fix-ups, and batches
//   k_rf_newton    -- the same Newton for a list of points (point location)
#include <cuda_runtime.h>

#include "k_integrate.cuh"

namespace ivv {

namespace {

constexpr int kScanBlock = 1024;

struct PairView {
  float L, t_in;
  float pin[3], pout[3];
  int blk;
  int nsamp, nlast;
};

__device__ __forceinline__ bool load_pair(const float4* pair_in, const float4* pair_out, const int* pair_block,
                                          size_t slot, float ds, float tail_eps, PairView& v) {
  const float4 pi = pair_in[slot], po = pair_out[slot];
  v.L = po.x - pi.x;
  if (!(v.L > 0.f)) return false;
  v.t_in = pi.x;
  v.pin[0] = pi.y; v.pin[1] = pi.z; v.pin[2] = pi.w;
  v.pout[0] = po.y; v.pout[1] = po.z; v.pout[2] = po.w;
  v.blk = pair_block[slot];
  const float fl = floorf(v.L / ds);
  v.nsamp = (int)fl;
  v.nlast = v.nsamp + ((v.L - fl * ds > tail_eps) ? 1 : 0);
  return true;
}

__global__ void k_rf_count(const float4* __restrict__ pair_in, const float4* __restrict__ pair_out,
                           const int* __restrict__ pair_block, const int* __restrict__ pair_count,
                           const int* __restrict__ active, const int* __restrict__ n_active, int npix, float ds,
                           float tail_eps, int* __restrict__ cnt) {
  pdl_wait();
  const int nact = *n_active;
  for (int item = blockIdx.x * blockDim.x + threadIdx.x; item < nact; item += gridDim.x * blockDim.x) {
    const int pix = active[item];
    const int np = pair_count[pix];
    int c = 0;
    for (int q = 0; q < np; ++q) {
      PairView v;
      if (load_pair(pair_in, pair_out, pair_block, (size_t)q * npix + pix, ds, tail_eps, v)) c += v.nlast + 1;
    }
    cnt[item] = c;
  }
}

// exclusive scan within each CTA of kScanBlock items; CTA totals to sums[]
__global__ void __launch_bounds__(kScanBlock) k_scan_local(const int* __restrict__ in, const int* __restrict__ n_ptr,
                                                           int* __restrict__ out, int* __restrict__ sums) {
  __shared__ int warp_tot[kScanBlock / 32];
  pdl_wait();
  const int n = *n_ptr;
  const int i = blockIdx.x * kScanBlock + threadIdx.x;
  if (blockIdx.x * kScanBlock >= n) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x = i < n ? in[i] : 0;
  int v = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  if (lane == 31) warp_tot[warp] = v;
  __syncthreads();
  if (warp == 0) {
    int w = warp_tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    warp_tot[lane] = w;
  }
  __syncthreads();
  const int incl = v + (warp > 0 ? warp_tot[warp - 1] : 0);
  if (i < n) out[i] = incl - x;
  if (threadIdx.x == kScanBlock - 1) sums[blockIdx.x] = incl;
}

// exclusive scan of the CTA sums (one CTA, chunks of kScanBlock) and total;
// the running total is kept in 64 bits, so a total beyond cap (at most
// INT_MAX) is reported as cap with the excess in total[1]
__global__ void __launch_bounds__(kScanBlock) k_scan_sums(int* __restrict__ sums, const int* __restrict__ n_ptr,
                                                          int cap, int* __restrict__ total) {
  __shared__ int warp_tot[kScanBlock / 32];
  __shared__ long long carry;
  pdl_wait();
  const int n = (*n_ptr + kScanBlock - 1) / kScanBlock;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < n; base += kScanBlock) {
    const int i = base + threadIdx.x;
    const int x = i < n ? sums[i] : 0;
    int v = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    if (lane == 31) warp_tot[warp] = v;
    __syncthreads();
    if (warp == 0) {
      int w = warp_tot[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += y;
      }
      warp_tot[lane] = w;
    }
    __syncthreads();
    const int incl = v + (warp > 0 ? warp_tot[warp - 1] : 0);
    const long long c = carry;
    if (i < n) sums[i] = (int)(c + incl - x);
    __syncthreads();
    if (threadIdx.x == kScanBlock - 1) carry = c + incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    *total = carry < (long long)cap ? (int)carry : cap;
    if (carry > (long long)cap) {                                  // overflow count
      const long long ex = carry - cap;
      total[1] = ex < 0x7fffffffll ? (int)ex : 0x7fffffff;
    }
  }
}

__global__ void k_scan_add(int* __restrict__ out, const int* __restrict__ n_ptr, const int* __restrict__ sums) {
  pdl_wait();
  const int n = *n_ptr;
  const int i = blockIdx.x * kScanBlock + threadIdx.x;
  if (i < n) out[i] += sums[blockIdx.x];
}

// Samples of the pixel's pairs.
__device__ __forceinline__ int pixel_samples(const float4* pair_in, const float4* pair_out, const int* pair_block,
                                             int pix, int np, int npix, float ds, float tail_eps) {
  int c = 0;
  for (int q = 0; q < np; ++q) {
    PairView v;
    if (load_pair(pair_in, pair_out, pair_block, (size_t)q * npix + pix, ds, tail_eps, v)) c += v.nlast + 1;
  }
  return c;
}

// cnt: the pixels' samples, counted here unless K4 did (counted).
// ctr->places: the places handed out; ctr->longest: the largest group;
// ctr->samples: the samples counted here (adding up those that K4 counted, and
// has the total of, cost 3 us of a 500 us frame).
__global__ void __launch_bounds__(256) k_rf_groups(const float4* __restrict__ pair_in,
                                                   const float4* __restrict__ pair_out,
                                                   const int* __restrict__ pair_block,
                                                   const int* __restrict__ pair_count, const int* __restrict__ active,
                                                   const int* __restrict__ n_active, int npix, float ds,
                                                   float tail_eps, bool counted, int* __restrict__ cnt,
                                                   RfGroup* __restrict__ grp, RfCounters* __restrict__ ctr) {
  pdl_wait();
  const int nact = *n_active, lane = threadIdx.x & 31;
  const int groups = (nact + 31) / 32, warps = (gridDim.x * blockDim.x) >> 5;
  int longest = 0;
  unsigned long long samples = 0;
  for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < groups; w += warps) {
    const int item = 32 * w + lane;
    int c = 0;
    if (item < nact && counted) {
      c = cnt[item];
    } else if (item < nact) {
      const int pix = active[item];
      c = pixel_samples(pair_in, pair_out, pair_block, pix, pair_count[pix], npix, ds, tail_eps);
      cnt[item] = c;
    }
    const int m = (int)__reduce_max_sync(0xffffffffu, (unsigned)c);
    longest = m > longest ? m : longest;
    if (!counted) samples += (unsigned)c;
    if (lane == 0) {
      RfGroup r;
      r.base = (long long)atomicAdd(&ctr->places, 32ull * (unsigned)m);
      r.m = m;
      r.pad = 0;
      grp[w] = r;
    }
  }
  if (lane == 0 && longest > 0) atomicMax(&ctr->longest, longest);
  if (!counted) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) samples += __shfl_down_sync(0xffffffffu, samples, o);
    if (lane == 0 && samples > 0) atomicAdd(&ctr->samples, samples);
  }
}

// A lane's walk through the samples of its pixel's pairs.
struct SampleWalk {
  PairView v;
  int q, j;
  __device__ __forceinline__ bool next_pair(const float4* pair_in, const float4* pair_out, const int* pair_block,
                                            int pix, int np, int npix, float ds, float tail_eps) {
    while (++q < np)
      if (load_pair(pair_in, pair_out, pair_block, (size_t)q * npix + pix, ds, tail_eps, v)) return true;
    return false;
  }
  // the pixel's sample i (false past the last)
  __device__ __forceinline__ bool seek(int i, const float4* pair_in, const float4* pair_out, const int* pair_block,
                                       int pix, int np, int npix, float ds, float tail_eps) {
    q = -1;
    while (next_pair(pair_in, pair_out, pair_block, pix, np, npix, ds, tail_eps)) {
      if (i <= v.nlast) {
        j = i;
        return true;
      }
      i -= v.nlast + 1;
    }
    return false;
  }
  __device__ __forceinline__ float s(float ds) const { return j <= v.nsamp ? (float)j * ds : v.L; }
};

// Learned guess: the places' world points and blocks, written in whole lines
// (a list in pixel order wrote every lane to a line of its own: 84 us on the
// 1080p beam, 19 here).  A lane past its last sample repeats it.
__global__ void __launch_bounds__(256) k_rf_points(DevCamera<float> cam, const float4* __restrict__ pair_in,
                                                   const float4* __restrict__ pair_out,
                                                   const int* __restrict__ pair_block,
                                                   const int* __restrict__ pair_count, const int* __restrict__ active,
                                                   const int* __restrict__ n_active, const RfGroup* __restrict__ grp,
                                                   int npix, float ds, float tail_eps, long long cap,
                                                   float4* __restrict__ sg, int* __restrict__ sblk) {
  pdl_wait();
  const int nact = *n_active, lane = threadIdx.x & 31;
  const int groups = (nact + 31) / 32, warps = (gridDim.x * blockDim.x) >> 5;
  for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < groups; w += warps) {
    const int item = 32 * w + lane;
    const RfGroup r = grp[w];
    if (r.base + 32ll * r.m > cap) continue;
    const int pix = item < nact ? active[item] : -1, np = pix >= 0 ? pair_count[pix] : 0;
    float o[3] = {0.f, 0.f, 0.f}, d[3] = {0.f, 0.f, 0.f};
    if (pix >= 0) make_ray<float>(cam, cam.x0 + pix % cam.w, cam.y0 + pix / cam.w, o, d);
    SampleWalk k;
    k.q = -1;
    k.j = 0;
    bool more = pix >= 0 && k.next_pair(pair_in, pair_out, pair_block, pix, np, npix, ds, tail_eps);
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
    int blk = 0;
    for (int i = 0; i < r.m; ++i) {
      if (more) {
        const float s = k.s(ds), t = k.v.t_in + s;
        g = make_float4(o[0] + t * d[0], o[1] + t * d[1], o[2] + t * d[2], s);
        blk = k.v.blk;
        if (++k.j > k.v.nlast) {
          more = k.next_pair(pair_in, pair_out, pair_block, pix, np, npix, ds, tail_eps);
          k.j = 0;
        }
      }
      sg[r.base + 32ll * i + lane] = g;
      sblk[r.base + 32ll * i + lane] = blk;
    }
  }
}

// One lane's Newton solve, one map evaluation per call of step(): the start, a
// full step or a halved one.  Only an accepted point's J is needed (for the
// next step, and for the scalar at the end: every way out follows an accepted
// point).
struct NewtonState {
  float q[3], p[3], dx[3];      // point to evaluate, last accepted point, Newton step
  float nF, lam;
  int it, ls;                   // it: iterations, -1 before the start's evaluation
  __device__ __forceinline__ void start(float x, float y, float z) {
    q[0] = p[0] = fminf(fmaxf(x, 0.f), 1.f);
    q[1] = p[1] = fminf(fmaxf(y, 0.f), 1.f);
    q[2] = p[2] = fminf(fmaxf(z, 0.f), 1.f);
    nF = 3.4e38f;
    it = -1;
    ls = 0;
  }
  // phi, J: the map at q.  True when the solve is over (at p).
  template <bool MIXED>
  __device__ __forceinline__ bool step(const BlockInfo& B, const float phi[3], const float J[3][3], const float g[3],
                                       float tol, int max_newton, unsigned long long& c_64) {
    const float F[3] = {phi[0] - g[0], phi[1] - g[1], phi[2] - g[2]};
    const float nG = sqrtf(F[0] * F[0] + F[1] * F[1] + F[2] * F[2]);
    if (it < 0 || nG < nF || ls == 5) {
      const bool moved = it < 0 || nG < nF;
      p[0] = q[0]; p[1] = q[1]; p[2] = q[2];
      nF = nG;
      if (!moved) return true;
      ++it;
      if (!(it < max_newton && nF > tol)) return true;
      const float rhs[3] = {-F[0], -F[1], -F[2]};
      const float det = solve3<float>(J, rhs, dx);
      if constexpr (MIXED) {
        if (fabsf(det) < B.tau_det) {
          double Jd[3][3], bd[3], xd[3];
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            bd[r] = rhs[r];
#pragma unroll
            for (int c = 0; c < 3; ++c) Jd[r][c] = J[r][c];
          }
          solve3<double>(Jd, bd, xd);
#pragma unroll
          for (int r = 0; r < 3; ++r) dx[r] = (float)xd[r];
          ++c_64;
        }
      }
      lam = 1.f;
      ls = 0;
    } else {
      lam *= 0.5f;
      ++ls;
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) q[r] = fminf(fmaxf(p[r] + lam * dx[r], 0.f), 1.f);
    return false;
  }
};

// A task is a group and a chunk of its samples: the lanes of a warp are
// neighbouring pixels at the same sample, so their control-point loads meet one
// or two elements, and the chunks keep every SM busy whatever the number of
// pixels.  (One lane per sample over a list in pixel order needed a sort by
// element for that, and a pass that wrote every sample's point and start; one
// lane per pixel through all its samples left the chip to the longest pixels:
// 974 us a frame on the 1367 x 769 step against 835 with the list and 584
// here.)  Four samples a chunk (eight: small frames 10 % slower, the rest
// even), four CTAs per SM (128 registers; three: even to 3 % slower).  A task
// past the end of its group is empty; where one group is so much longer than
// the others that there would be more than sixteen tasks for every four
// samples of a group, or 2^30 of them, the chunks are longer.
// sp: the learned guess's starts by place (null otherwise).  VM: the von Mises
// scalar of §6.2, in an instance of its own.
constexpr int kRfChunk = 4;
template <int P, bool MIXED, bool STATS, bool VM>
__global__ void __launch_bounds__(128, 4) k_rf_solve(DevVolume V, DevCamera<float> cam, float rf_tol, int guess,
                                                     const float4* __restrict__ pair_in,
                                                     const float4* __restrict__ pair_out,
                                                     const int* __restrict__ pair_block,
                                                     const int* __restrict__ pair_count,
                                                     const int* __restrict__ active, const int* __restrict__ n_active,
                                                     const int* __restrict__ cnt, const RfGroup* __restrict__ grp,
                                                     RfCounters* __restrict__ ctr, const float4* __restrict__ sp,
                                                     long long cap, int npix, float ds, float tail_eps,
                                                     float* __restrict__ srho, DevStats* __restrict__ st) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int nact = *n_active, groups = (nact + 31) / 32;
  const unsigned longest = (unsigned)ctr->longest;
  unsigned chunk = kRfChunk;
  {
    const unsigned long long all = (unsigned long long)groups * ((longest + chunk - 1) / chunk);
    const unsigned long long most = min(16 * (ctr->places / (32 * kRfChunk)) + groups, 1ull << 30);
    if (all > most) chunk *= (unsigned)((all + most - 1) / most);
  }
  const int tasks = groups * (int)((longest + chunk - 1) / chunk);
  // half width of a pixel per unit depth (perspective) or absolute (ortho)
  const float px_half = cam.sy / (float)cam.H;
  unsigned long long c_it = 0, c_ev = 0, c_fail = 0, c_64 = 0;
  for (;;) {
    int t0 = 0;
    if (lane == 0) t0 = atomicAdd(&ctr->head, 1);
    t0 = __shfl_sync(0xffffffffu, t0, 0);
    if (t0 >= tasks) break;
    // chunk after chunk over all groups: neighbouring warps share elements
    const int w = t0 % groups, i0 = t0 / groups * (int)chunk;
    const RfGroup gr = grp[w];
    if (i0 >= gr.m || gr.base + 32ll * gr.m > cap) continue;
    const int item = 32 * w + lane;
    const int left = item < nact ? cnt[item] - i0 : 0;
    const int last = left > 0 ? i0 + min(left, (int)chunk) : 0;            // one past the lane's samples
    int i = i0;
    if (i < last) {
      const int pix = active[item], np = pair_count[pix];
      float o[3], d[3];
      make_ray<float>(cam, cam.x0 + pix % cam.w, cam.y0 + pix / cam.w, o, d);
      SampleWalk k;
      k.seek(i, pair_in, pair_out, pair_block, pix, np, npix, ds, tail_eps);
      BlockInfo B = V.blocks[k.v.blk];
      NewtonState nw;
      float g[3], tol = 0.f;
      bool fresh = true;              // the next evaluation is a sample's start
      while (i < last) {
        if (fresh) {
          fresh = false;
          const float s = k.s(ds), t = k.v.t_in + s;
#pragma unroll
          for (int r = 0; r < 3; ++r) g[r] = o[r] + t * d[r];
          float depth = 1.f;
          if (!cam.ortho)
            depth = (g[0] - cam.eye[0]) * cam.f[0] + (g[1] - cam.eye[1]) * cam.f[1] + (g[2] - cam.eye[2]) * cam.f[2];
          tol = rf_tol * px_half * depth;
          // never below FP32 resolution of the coordinates
          tol = fmaxf(tol, 2e-7f * (fabsf(g[0]) + fabsf(g[1]) + fabsf(g[2]) + V.diag));
          if (sp != nullptr) {
            const float4 p4 = sp[gr.base + 32ll * i + lane];
            nw.start(p4.x, p4.y, p4.z);
          } else if (guess != 0) {
            const float a = s / k.v.L;
            nw.start(k.v.pin[0] + a * (k.v.pout[0] - k.v.pin[0]), k.v.pin[1] + a * (k.v.pout[1] - k.v.pin[1]),
                     k.v.pin[2] + a * (k.v.pout[2] - k.v.pin[2]));
          } else {
            nw.start(0.5f, 0.5f, 0.5f);
          }
        }
        float phi[3], J[3][3], rc;
        eval_block<P, float, false>(V, B, nw.q, phi, J, rc);
        if (STATS) ++c_ev;
        if (!nw.template step<MIXED>(B, phi, J, g, tol, V.max_newton, c_64)) continue;
        if (STATS) c_it += nw.it;
        if (nw.nF > tol) ++c_fail;
        float rho;
        if constexpr (VM)
          rho = scalar_at<P, float>(V, B, IVV_SCALAR_VONMISES, nw.p, J, 0.f);
        else
          rho = V.mode == IVV_SCALAR_CP ? eval_rho_cp<P>(V, B, nw.p)
                : V.mode == IVV_SCALAR_DETJ ? det3<float>(J)
                                            : quality_det3<float>(J);
        srho[gr.base + 32ll * i + lane] = rho;
        fresh = true;
        ++i;
        if (++k.j > k.v.nlast && i < last) {
          k.next_pair(pair_in, pair_out, pair_block, pix, np, npix, ds, tail_eps);
          k.j = 0;
          B = V.blocks[k.v.blk];
        }
      }
    }
    __syncwarp();
  }
  if (STATS) {
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) {
      c_it += __shfl_down_sync(0xffffffffu, c_it, o2);
      c_ev += __shfl_down_sync(0xffffffffu, c_ev, o2);
      c_fail += __shfl_down_sync(0xffffffffu, c_fail, o2);
    }
    if (lane == 0) {
      atomicAdd(&st->rf_newton_iters, c_it);
      atomicAdd(&st->rhs_evals, c_ev);
      atomicAdd(&st->rf_unconverged, c_fail);
    }
  } else if (c_fail) {
    atomicAdd(&st->rf_unconverged, c_fail);         // a cap counter: kept by every render
  }
  if (MIXED && c_64) atomicAdd(&st->fp64_solves, c_64);
}

// One lane per pixel; the lanes of a warp are the group's, so a sample's
// scalars are one line (in a list in pixel order they were 32).
__global__ void __launch_bounds__(128) k_rf_composite(DevTF tf, int K, float early, const float4* __restrict__ pair_in,
                                                      const float4* __restrict__ pair_out,
                                                      const int* __restrict__ pair_block,
                                                      const int* __restrict__ pair_count,
                                                      const int* __restrict__ active,
                                                      const int* __restrict__ n_active, const int* __restrict__ cnt,
                                                      const RfGroup* __restrict__ grp, int npix, float ds,
                                                      float tail_eps, long long cap, const float* __restrict__ srho,
                                                      float4* __restrict__ out, DevStats* __restrict__ st, bool stats) {
  __shared__ TfTable s_tf;
  tf_load(s_tf, tf);
  pdl_wait();
  const int nact = *n_active, lane = threadIdx.x & 31;
  unsigned long long c_samp = 0;
  for (int item = blockIdx.x * blockDim.x + threadIdx.x; item < nact; item += gridDim.x * blockDim.x) {
    const RfGroup gr = grp[item >> 5];
    const int pix = active[item], np = pair_count[pix];
    Acc<float> acc;
    acc.C[0] = acc.C[1] = acc.C[2] = acc.a = 0.f;
    if (gr.base + 32ll * gr.m <= cap) {
      c_samp += cnt[item];
      // flat over the pixel's (pair, sample) sequence: lanes whose pairs end
      // at different samples stay together
      const float* rho_at = srho + gr.base + lane;
      const int n = cnt[item];
      SampleWalk k;
      k.q = -1;
      k.j = 0;
      k.v.nlast = -1;                               // no pair yet
      float rho_prev = 0.f, s_prev = 0.f;
      for (int i = 0; i < n; ++i) {
        const float rho = rho_at[32ll * i];
        if (k.j > k.v.nlast) {
          k.next_pair(pair_in, pair_out, pair_block, pix, np, npix, ds, tail_eps);
          k.j = 0;
        }
        const float s = k.s(ds);
        if (k.j > 0) {
          composite_interval<float>(s_tf.view(), tf, K, rho_prev, rho, s - s_prev, acc);
          if (acc.a >= early) break;
        }
        rho_prev = rho;
        s_prev = s;
        ++k.j;
      }
    }
    out[pix] = make_float4(acc.C[0], acc.C[1], acc.C[2], acc.a);
  }
  if (stats) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c_samp += __shfl_down_sync(0xffffffffu, c_samp, o);
    if (lane == 0) atomicAdd(&st->samples, c_samp);
  }
}

// Point location: damped Newton for listed points to a fixed tolerance.
// Four CTAs per SM (128 registers), as k_rf_solve.
template <int P>
__global__ void __launch_bounds__(128, 4) k_rf_newton(DevVolume V, float abs_tol, const int* __restrict__ n_ptr,
                                                      const float4* __restrict__ sg, const int* __restrict__ sblk,
                                                      const float4* __restrict__ sp, float4* __restrict__ p_out,
                                                      int* __restrict__ it_out, DevStats* __restrict__ st) {
  pdl_wait();
  const int n = *n_ptr;
  unsigned long long c_fail = 0, c_64 = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float4 g4 = sg[i];
    const float g[3] = {g4.x, g4.y, g4.z};
    const BlockInfo B = V.blocks[sblk[i]];
    // never below FP32 resolution of the coordinates
    const float tol = fmaxf(abs_tol, 2e-7f * (fabsf(g[0]) + fabsf(g[1]) + fabsf(g[2]) + V.diag));
    const float4 p4 = sp[i];
    NewtonState nw;
    nw.start(p4.x, p4.y, p4.z);
    for (;;) {
      float phi[3], J[3][3], rc;
      eval_block<P, float, false>(V, B, nw.q, phi, J, rc);
      if (nw.step<false>(B, phi, J, g, tol, V.max_newton, c_64)) break;
    }
    if (nw.nF > tol) ++c_fail;
    p_out[i] = make_float4(nw.p[0], nw.p[1], nw.p[2], nw.nF);
    if (it_out) it_out[i] = nw.nF <= tol ? nw.it : -1 - nw.it;
  }
  if (c_fail) atomicAdd(&st->rf_unconverged, c_fail);       // a cap counter
}

}  // namespace

namespace {
__global__ void k_fill_center(float4* __restrict__ p, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = make_float4(0.5f, 0.5f, 0.5f, 0.f);
}
}  // namespace

void launch_fill_center(float4* p, int n, cudaStream_t s) {
  if (n > 0) k_fill_center<<<(n + 255) / 256, 256, 0, s>>>(p, n);
}

void launch_rf_count(const float4* pin, const float4* pout, const int* pblk, const int* pcnt, const int* active,
                     const int* n_active, int npix, float ds, float tail_eps, int* cnt, int num_sms, cudaStream_t s) {
  launch_pdl(k_rf_count, dim3(num_sms * 8), dim3(256), s, pin, pout, pblk, pcnt, active, n_active, npix, ds, tail_eps,
             cnt);
}

void launch_rf_scan(const int* cnt, const int* n_active, int npix, int* off, int* sums, int cap, int* total,
                    cudaStream_t s) {
  const int blocks = (npix + kScanBlock - 1) / kScanBlock;
  launch_pdl(k_scan_local, dim3(blocks), dim3(kScanBlock), s, cnt, n_active, off, sums);
  launch_pdl(k_scan_sums, dim3(1), dim3(kScanBlock), s, sums, n_active, cap, total);
  launch_pdl(k_scan_add, dim3(blocks), dim3(kScanBlock), s, off, n_active, (const int*)sums);
}

void launch_rf_groups(const float4* pin, const float4* pout, const int* pblk, const int* pcnt, const int* active,
                      const int* n_active, int npix, float ds, float tail_eps, bool counted, int* cnt, RfGroup* grp,
                      RfCounters* ctr, int num_sms, cudaStream_t s) {
  launch_pdl(k_rf_groups, dim3(num_sms * 8), dim3(256), s, pin, pout, pblk, pcnt, active, n_active, npix, ds, tail_eps,
             counted, cnt, grp, ctr);
}

void launch_rf_points(const DevCamera<float>& cam, const float4* pin, const float4* pout, const int* pblk,
                      const int* pcnt, const int* active, const int* n_active, const RfGroup* grp, int npix, float ds,
                      float tail_eps, long long cap, float4* sg, int* sblk, int num_sms, cudaStream_t s) {
  launch_pdl(k_rf_points, dim3(num_sms * 8), dim3(256), s, cam, pin, pout, pblk, pcnt, active, n_active, grp, npix, ds,
             tail_eps, cap, sg, sblk);
}

namespace {
template <int P, bool MIXED, bool STATS, bool VM>
void launch_rf_solve_k(const DevVolume& V, const DevCamera<float>& cam, float rf_tol, int guess, const float4* pin,
                       const float4* pout, const int* pblk, const int* pcnt, const int* active, const int* n_active,
                       const int* cnt, const RfGroup* grp, RfCounters* ctr, const float4* sp, long long cap, int npix,
                       float ds, float tail_eps, float* srho, DevStats* st, int num_sms, cudaStream_t s) {
  static int per_sm = -1;
  if (per_sm < 0) {
    int n = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_rf_solve<P, MIXED, STATS, VM>, 128, 0);
    per_sm = n < 1 ? 1 : n;
  }
  launch_pdl(k_rf_solve<P, MIXED, STATS, VM>, dim3(num_sms * per_sm), dim3(128), s, V, cam, rf_tol, guess, pin, pout,
             pblk, pcnt, active, n_active, cnt, grp, ctr, sp, cap, npix, ds, tail_eps, srho, st);
}
}  // namespace

void launch_rf_solve(const DevVolume& V, const DevCamera<float>& cam, float rf_tol, int guess, const float4* pin,
                     const float4* pout, const int* pblk, const int* pcnt, const int* active, const int* n_active,
                     const int* cnt, const RfGroup* grp, RfCounters* ctr, const float4* sp, long long cap, int npix,
                     float ds, float tail_eps, float* srho, bool mixed, bool stats, DevStats* st, int num_sms,
                     cudaStream_t s) {
#define IVV_RFS(PP, MM, SS, VV)                                                                                  \
  launch_rf_solve_k<PP, MM, SS, VV>(V, cam, rf_tol, guess, pin, pout, pblk, pcnt, active, n_active, cnt, grp, ctr, sp, \
                                    cap, npix, ds, tail_eps, srho, st, num_sms, s)
#define IVV_RFS2(PP, VV)                                                                        \
  do {                                                                                          \
    if (mixed) { if (stats) IVV_RFS(PP, true, true, VV); else IVV_RFS(PP, true, false, VV); }   \
    else { if (stats) IVV_RFS(PP, false, true, VV); else IVV_RFS(PP, false, false, VV); }       \
  } while (0)
  const bool vm = V.mode == IVV_SCALAR_VONMISES;
  if (V.P == 2) { if (vm) IVV_RFS2(2, true); else IVV_RFS2(2, false); }
  else { if (vm) IVV_RFS2(3, true); else IVV_RFS2(3, false); }
#undef IVV_RFS2
#undef IVV_RFS
}

void launch_rf_composite(const DevTF& tf, int K, float early, const float4* pin, const float4* pout, const int* pblk,
                         const int* pcnt, const int* active, const int* n_active, const int* cnt, const RfGroup* grp,
                         int npix, float ds, float tail_eps, long long cap, const float* srho, float4* out,
                         DevStats* st, bool stats, int num_sms, cudaStream_t s) {
  launch_pdl(k_rf_composite, dim3(num_sms * 8), dim3(128), s, tf, K, early, pin, pout, pblk, pcnt, active, n_active,
             cnt, grp, npix, ds, tail_eps, cap, srho, out, st, stats);
}

void launch_rf_newton(const DevVolume& V, float abs_tol, const int* n_ptr, const float4* sg, const int* sblk,
                      const float4* sp, float4* p_out, int* it_out, DevStats* st, int num_sms, cudaStream_t s) {
  if (V.P == 2)
    launch_pdl(k_rf_newton<2>, dim3(num_sms * 16), dim3(128), s, V, abs_tol, n_ptr, sg, sblk, sp, p_out, it_out, st);
  else
    launch_pdl(k_rf_newton<3>, dim3(num_sms * 16), dim3(128), s, V, abs_tol, n_ptr, sg, sblk, sp, p_out, it_out, st);
}

}  // namespace ivv
