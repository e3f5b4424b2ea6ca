// pf_adjoint.cu -- kernels of pf_backward: the gradient of log Z = sum_k
// log c_k with respect to theta = (sigma_psf, A, b, sigma_pos, sigma_v) with
// the resampling ancestry of the forward run held fixed.
//
// Paper: Demirel et al., "An Adaptive Distributed Resampling Algorithm with
// Non-Proportional Allocation" (arXiv:1310.4624).  With the ancestry fixed
// the filter (Alg. 3) is a smooth function of theta:
//   X_k(i)   = NCV(X_{k-1}(p_k(i)); theta)            (Alg. 1 step P)
//   lw_k(i)  = lbar_{k-1}(o(i)) - log Np + l_k(i)      (steps 4-5, U)
//   L_k,m    = LSE_{i in m} lw_k(i)                    (step 6)
//   log c_k  = LSE_m L_k,m,  lbar_k = L_k - log c_k    (steps 9-10)
// with o(i) = p_k(i) div Np the origin group of the slot (the exchange puts
// a particle of group o into slot i).  Reverse mode, seed s = d out / d log Z:
//   dL_{T-1,m} = s pi_m,  dL_{k,m} = sum_{i : o_{k+1}(i) = m} dlw_{k+1}(i)
//   dlw_k(i)   = dL_{k,m(i)} exp(lw_k(i) - L_k,m(i))
// (the softmax terms of lbar cancel because sum_m dL_k,m = s at every k);
// states back-propagate through the NCV Jacobian to their recorded parents.
// The forward pass is replayed from the initial population and the recorded
// parents with the same Philox streams; the replay leaves the log-weights and
// the likelihood's derivatives of each step (24 bytes a particle), which is
// all that the reverse sweep needs of it.  Where those of every step would
// take more than ADJ_STORE_MAX, they are kept for a segment at a time and
// replayed from checkpoints of the states.
#include <cuda_runtime.h>

#include <climits>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "pf_device.cuh"
#include "pf_launch.h"
#include "pf_math.cuh"

namespace pf {

constexpr int RG_GROUP_THREADS = 1024;

// --------------------------------------------- likelihood and its derivatives
// Where a tile's pixels come from: the caller's frame (raw: y = z - bg inside,
// 0 outside) or the track's padded frame (bg = 0, every access inside).
// Patch coordinates are those of the padded frame; sub converts them.
struct PixelSource {
  const float* z;
  int w, h, sub;
  float bg;
  __device__ __forceinline__ float at(int u, int v) const {
    const int x = u - sub, y = v - sub;
    return ((unsigned)x < (unsigned)w && (unsigned)y < (unsigned)h) ? __fsub_rn(__ldg(z + (long long)y * w + x), bg)
                                                                    : 0.0f;
  }
};

// A patch's pixels from the staged box (from the frame: FramePatch).
struct StagedRows {
  const float* base;
  __device__ __forceinline__ float operator()(int b, int a) const { return base[b * ROI_W + a]; }
};

// Log-likelihood (Sec. V model) and its partial derivatives for the
// adjoint: d[0..4] = dl/dx, dl/dy, dl/dI, dl/dsigma_psf, dl/db.  One pass
// over the patch with separable row sums: per row v with r = y - I gx gy,
// R0 = sum r gx, R1 = sum r gx a, R2 = sum r gx a^2 (a the column offset), so
// that sum r gx (u - x) = R1 + du0 R0 and sum r gx (u - x)^2 = R2 + 2 du0 R1
// + du0^2 R0 with du0 = cx - R - x.  Pixels outside the frame count as
// background, so only inside pixels depend on b.
// The replay's group log-weights come from patch_sum's order of the same
// pixels; both orders are part of the result's rounding and are kept.
// ROLLED: a loop over the rows (gy from memory, every patch masked), for
// patches read from the frame, whose loads would otherwise be hoisted into
// more registers than there are; the sums and their order are the same.
template <int R, bool ROLLED, class Rows, class Gy>
__device__ __forceinline__ float loglik_grad(const Rows& px, const Gy& gy, int H, int W, float x, float y, float I,
                                             const TrackParams& P, float (&d)[5]) {
  constexpr int D = 2 * R + 1;
  const float cxf = floorf(x + 0.5f), cyf = floorf(y + 0.5f);
  float gx[D];
  gauss_row<R>(cxf, x, P.c_psf, P.kappa, gx);
  // inside-the-frame column / row ranges of the (true) patch
  const float ulo = fmaxf(0.0f, (float)R - cxf), uhi = fminf((float)(2 * R), (float)(W - 1) + (float)R - cxf);
  const float vlo = fmaxf(0.0f, (float)R - cyf), vhi = fminf((float)(2 * R), (float)(H - 1) + (float)R - cyf);
  float ss = 0.0f, SI = 0.0f, S1 = 0.0f, Sy = 0.0f, Ss = 0.0f, Sb = 0.0f, Y2 = 0.0f, Y1 = 0.0f;
  const float du0 = cxf - (float)R - x;
  // patches wholly inside the frame (almost all) sum the b-derivative's
  // residuals without per-pixel masks
  const bool inside = ulo == 0.0f && uhi == (float)(2 * R) && vlo == 0.0f && vhi == (float)(2 * R);
  auto rows = [&](auto inside_tag) {
    constexpr bool IN = decltype(inside_tag)::value;
#pragma unroll(ROLLED ? 1 : D)
    for (int b = 0; b < D; ++b) {
      asm volatile("" ::: "memory");  // (a row's pixels at a time)
      const float gyb = gy(b);
      const float Igy = I * gyb;
      float R0 = 0.0f, R1 = 0.0f, R2 = 0.0f, Rb = 0.0f;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const float yv = px(b, a);  // y = z - b, 0 outside the frame
        const float r = fmaf(-gx[a], Igy, yv);
        ss = fmaf(r, r, ss);
        Y2 = fmaf(yv, yv, Y2);
        Y1 += yv;
        const float t = r * gx[a];
        R0 += t;
        R1 = fmaf(t, (float)a, R1);
        R2 = fmaf(t, (float)(a * a), R2);
        if constexpr (IN)
          Rb += r;
        else
          Rb += ((float)a >= ulo && (float)a <= uhi) ? r : 0.0f;
      }
      const float dv = (cyf - (float)R + (float)b) - y;
      const float sx1 = R1 + du0 * R0;
      const float sx2 = R2 + 2.0f * du0 * R1 + du0 * du0 * R0;
      SI = fmaf(gyb, R0, SI);
      S1 = fmaf(gyb, sx1, S1);
      Sy = fmaf(gyb * dv, R0, Sy);
      Ss = fmaf(gyb, fmaf(dv * dv, R0, sx2), Ss);
      if (IN || ((float)b >= vlo && (float)b <= vhi)) Sb += Rb;
    }
  };
  if (!ROLLED && inside)
    rows(std::true_type{});
  else
    rows(std::false_type{});
  const float iso2 = 2.0f * P.inv2so2;  // 1 / sigma_obs^2
  const float s2 = P.spsf * P.spsf;
  d[0] = I * S1 / s2 * iso2;
  d[1] = I * Sy / s2 * iso2;
  d[2] = SI * iso2;
  d[3] = I * Ss / (s2 * P.spsf) * iso2;
  d[4] = Sb * iso2;
  if (P.obs_model == 1) {
    // frame likelihood ratio: + sum y^2 / (2 sigma_obs^2), whose only
    // parameter is b (dy/db = -1 inside the frame, y = 0 outside)
    d[4] -= Y1 * iso2;
    return -(ss - Y2) * P.inv2so2;
  }
  return -ss * P.inv2so2;
}

// ------------------------------------------------------------------ replay
// A particle's log-weight into the thread's running (max, sum exp), and what
// the reverse sweep takes of it (log-weight `lwg`, derivatives d).
__device__ __forceinline__ void weigh(float lw, float& mx, float& sm) {
  if (lw == lw && lw > -INFINITY) {
    if (lw > mx) {
      sm = sm * __expf(mx - lw) + 1.0f;
      mx = lw;
    } else {
      sm += __expf(lw - mx);
    }
  }
}
__device__ __forceinline__ void keep_derivatives(const ReplayArgs& a, long long i, const float (&d)[5], float lwg) {
  a.dl_pv[i] = make_float4(d[0], d[1], d[2], d[3]);
  a.dl_b[i] = d[4];
  a.dl_lw[i] = lwg;
}

// The pixels that patches are taken from, of a single track's frame or of
// the track's padded frame.
template <int R>
__device__ __forceinline__ PixelSource pixel_source(const ReplayArgs& a, const TrackParams& P) {
  constexpr int PAD = 2 * R + 1;
  return a.zraw ? PixelSource{a.zraw, P.W, P.H, PAD, P.bg}
                : PixelSource{a.ypad + P.ypad_off, P.pitch, P.H + 2 * PAD, 0, 0.0f};
}

// A patch's corner in padded-frame coordinates (centre clamped so that a
// patch wholly off the frame reads background).
template <int R>
__device__ __forceinline__ int patch_corner(float x, int n) {
  return (int)fminf(fmaxf(floorf(x + 0.5f), -(float)(R + 1)), (float)(n + R)) - R + (2 * R + 1);
}

// The weights of a tile whose patches do not fit one staging box (a spread
// population): the patches are read from the frame.  Out of line, and from
// the states the tile has just stored, so that nothing of it takes registers
// of the staged path; gy of the rolled row loop lies in s_gy (one float per
// thread and row, of the staging buffer that such a tile does not use).  Bound
// by L1: a lane's pixel is a line of its own, in both passes over a patch.
// The gradient over two frames of 64 x 16384 spread particles: 1939 us with
// the patch's rows and arrays spilled under the staged path's registers, 1052
// from prepared frames without bounds checks, 739 here.
template <int R>
__device__ __noinline__ float2 replay_off_box(const ReplayArgs& a, const TrackParams& P, int4 td, float* s_gy) {
  constexpr int D = 2 * R + 1;
  const int g = td.y, Np = P.Np, k = a.k;
  const float log_G = logf((float)P.G), log_Np = logf((float)Np);
  const PixelSource px = pixel_source<R>(a, P);
  const uint32_t* __restrict__ par_t =
      a.parent + P.parent_off + (long long)(k % a.history) * ((long long)P.G * Np);
  float mx = -INFINITY, sm = 0.0f;
  for (int jj = threadIdx.x; jj < td.w; jj += K1_THREADS) {
    const long long il = (long long)g * Np + td.z + jj, i = P.part_off + il;
    const float4 s = a.pv_out[i];
    const float I = a.I_out[i];
    const float lb = k >= 1 ? a.lbar_prev[P.group_off + (int)fastdiv(par_t[il], P.m_Np)] : -log_G;
    const FramePatch rows(px.z, px.w, px.h, px.bg, patch_corner<R>(s.x, P.W) - px.sub,
                          patch_corner<R>(s.y, P.H) - px.sub, D);
    float ss;
    {
      float gxI[D];
      gauss_row<R>(floorf(s.x + 0.5f), s.x, P.c_psf, P.kappa, gxI);
#pragma unroll
      for (int c = 0; c < D; ++c) gxI[c] *= I;
      const float dy = floorf(s.y + 0.5f) - s.y;
      ss = P.obs_model == 1 ? patch_sum<R, true>(rows, gxI, dy, P.c_psf, P.kappa)
                            : patch_sum<R, false>(rows, gxI, dy, P.c_psf, P.kappa);
    }
    weigh(lb - log_Np - ss * P.inv2so2, mx, sm);
    if (a.dl_pv) {
      float gy[D], d[5];
      gauss_row<R>(floorf(s.y + 0.5f), s.y, P.c_psf, P.kappa, gy);
#pragma unroll
      for (int b = 0; b < D; ++b) s_gy[b * K1_THREADS + threadIdx.x] = gy[b];
      const float l = loglik_grad<R, true>(rows, [&](int b) { return s_gy[b * K1_THREADS + threadIdx.x]; }, P.H, P.W,
                                           s.x, s.y, I, P, d);
      keep_derivatives(a, i, d, lb - log_Np + l);
    }
  }
  return make_float2(mx, sm);
}

// Replay of step k for every slot: the state (propagate: NCV from the
// recorded parent and the step's normals; else as given in pv_out), the
// log-weights' (max, sum exp) per tile for the group log-weights and, where
// dl_pv is given, the log-weight and the likelihood's derivatives for the
// reverse sweep, which then never looks at a frame.
// One CTA per tile; the box of the tile's patches is staged in shared memory
// twice (the copy shifted by one float makes every patch row a row of aligned
// pairs), a tile whose patches do not fit reads the frame through L1.  Bound
// by FP32 issue (the two patch sums are ~1200 instructions a particle) and the
// latency of the gathers before them: 84 us a million particles, a gradient of
// 16 x 65536 particles over 20 frames 7.7 ms when each step's patches were
// summed by the replay and again by the reverse sweep, 4.1 now.  Derivatives
// by column sums in packed pairs would take 55 us.  They are in another order,
// which moves the gradient by up to 2e-5 of its largest component (and nearer
// to the 64-bit value): a library update would then change the iterates of a
// parameter fit, so the order of the sums is kept as part of the result.
// SINGLE: one track, its parameters and round keys in the constant bank.
template <int R, bool SINGLE>
__global__ void __launch_bounds__(K1_THREADS, 4) k_replay(const __grid_constant__ ReplayArgs a) {
  constexpr int D = 2 * R + 1, NW = K1_THREADS / 32;
  __shared__ __align__(16) float s_roi[2][ROI_FLOATS + 4];
  __shared__ int s_box[NW][4];
  __shared__ float s_m[NW], s_s[NW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int k = a.k, tile = blockIdx.x;
  grid_dep_wait();
  grid_dep_launch();
  const int4 td = a.tiles[tile];
  const TrackParams& P = SINGLE ? a.p0 : a.trk[td.x];
  const int g = td.y, Np = P.Np;
  const long long Nt = (long long)P.G * Np;
  const uint32_t* __restrict__ par_t = a.parent + P.parent_off + (long long)(k % a.history) * Nt;
  float4 s[K1_PPT];
  float I[K1_PPT];
  int o[K1_PPT], pu[K1_PPT], pv[K1_PPT];
  int umin = INT_MAX, umax = INT_MIN, vmin = INT_MAX, vmax = INT_MIN;
#pragma unroll
  for (int q = 0; q < K1_PPT; ++q) {
    const int jj = threadIdx.x + q * K1_THREADS, j = td.z + jj;
    const long long il = (long long)g * Np + j, i = P.part_off + il;
    o[q] = g;
    if (jj >= td.w) continue;
    uint32_t par = 0;
    if (k >= 1) {
      par = par_t[il];
      o[q] = (int)fastdiv(par, P.m_Np);  // origin group
    }
    if (a.propagate) {
      s[q] = a.pv_in[P.part_off + par];
      I[q] = a.I_in[P.part_off + par];
      uint4 w0 = make_uint4(j, g, k, P.tag | (ST_PROP << 4) | 0u);
      uint4 w1 = make_uint4(j, g, k, P.tag | (ST_PROP << 4) | 1u);
      if constexpr (SINGLE)
        philox2_rk(P.rk, w0, w1);
      else
        philox2(P.key0, P.key1, w0, w1);
      float e0, e1, e2, e3, e4, e5;
      box_muller_fast(w0.x, w0.y, e0, e1);
      box_muller_fast(w0.z, w0.w, e2, e3);
      box_muller_fast(w1.x, w1.y, e4, e5);
      s[q].x = fmaf(P.spos, e0, s[q].x + s[q].z);
      s[q].y = fmaf(P.spos, e1, s[q].y + s[q].w);
      s[q].z = fmaf(P.sv, e2, s[q].z);
      s[q].w = fmaf(P.sv, e3, s[q].w);
      I[q] = fmaf(P.sI, e4, I[q]);
      a.pv_out[i] = s[q];
      a.I_out[i] = I[q];
    } else {
      s[q] = a.pv_out[i];
      I[q] = a.I_out[i];
    }
    if (a.ck_pv) {
      a.ck_pv[i] = s[q];
      a.ck_I[i] = I[q];
    }
    if (a.zero_pv) {
      a.zero_pv[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      a.zero_I[i] = 0.0f;
    }
    pu[q] = patch_corner<R>(s[q].x, P.W);
    pv[q] = patch_corner<R>(s[q].y, P.H);
    umin = min(umin, pu[q]);
    umax = max(umax, pu[q]);
    vmin = min(vmin, pv[q]);
    vmax = max(vmax, pv[q]);
  }

  // the box of the tile's patches, staged as y values
  const PixelSource px = pixel_source<R>(a, P);
  umin = __reduce_min_sync(0xffffffffu, umin);
  umax = __reduce_max_sync(0xffffffffu, umax);
  vmin = __reduce_min_sync(0xffffffffu, vmin);
  vmax = __reduce_max_sync(0xffffffffu, vmax);
  if (lane == 0) {
    s_box[warp][0] = umin;
    s_box[warp][1] = umax;
    s_box[warp][2] = vmin;
    s_box[warp][3] = vmax;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    umin = min(umin, s_box[w][0]);
    umax = max(umax, s_box[w][1]);
    vmin = min(vmin, s_box[w][2]);
    vmax = max(vmax, s_box[w][3]);
  }
  const int cols = umax + D - umin, nrows = vmax + D - vmin;
  const bool staged = cols <= ROI_W && nrows <= ROI_ROWS;
  if (staged) {
    // eight threads a row, 32 rows a pass: sector-sized reads
    const int c0 = threadIdx.x & 7;
    for (int r = threadIdx.x >> 3; r < nrows; r += K1_THREADS / 8)
#pragma unroll
      for (int i = 0; i < ROI_W / 8; ++i) {
        const int c = c0 + 8 * i;
        if (c < cols) {
          const float v = px.at(umin + c, vmin + r);
          s_roi[0][r * ROI_W + c] = v;
          if (r * ROI_W + c > 0) s_roi[1][r * ROI_W + c - 1] = v;
        }
      }
    __syncthreads();
  }

  float mx = -INFINITY, sm = 0.0f;
  if (staged) {
    const float log_G = logf((float)P.G), log_Np = logf((float)Np);
    const bool frame_model = P.obs_model == 1;
#pragma unroll
    for (int q = 0; q < K1_PPT; ++q) {
      const int jj = threadIdx.x + q * K1_THREADS;
      if (jj >= td.w) continue;
      const long long i = P.part_off + (long long)g * Np + td.z + jj;
      const int c = pu[q] - umin, off = (pv[q] - vmin) * ROI_W + c;
      const float* base = (c & 1) ? &s_roi[1][off - 1] : &s_roi[0][off];
      float ss;
      {
        float gxI[D];
        gauss_row<R>(floorf(s[q].x + 0.5f), s[q].x, P.c_psf, P.kappa, gxI);
#pragma unroll
        for (int x = 0; x < D; ++x) gxI[x] *= I[q];
        const float dy = floorf(s[q].y + 0.5f) - s[q].y;
        ss = frame_model ? patch_ss_pairs<R, true>(base, gxI, dy, P.c_psf, P.kappa)
                         : patch_ss_pairs<R, false>(base, gxI, dy, P.c_psf, P.kappa);
      }
      const float lb = k >= 1 ? a.lbar_prev[P.group_off + o[q]] : -log_G;
      asm volatile("" ::: "memory");  // (the pixels are read again, not held in registers)
      if (a.dl_pv) {
        float gy[D], d[5];
        gauss_row<R>(floorf(s[q].y + 0.5f), s[q].y, P.c_psf, P.kappa, gy);
        const float l = loglik_grad<R, false>(StagedRows{base}, [&](int b) { return gy[b]; }, P.H, P.W, s[q].x, s[q].y,
                                              I[q], P, d);
        keep_derivatives(a, i, d, lb - log_Np + l);
      }
      weigh(lb - log_Np - ss * P.inv2so2, mx, sm);
    }
  } else {
    const float2 ms = replay_off_box<R>(a, P, td, &s_roi[0][0]);
    mx = ms.x;
    sm = ms.y;
  }
  // block (max, sum exp) of the tile
  const float m2 = warp_max(mx);
  const float s2 = warp_sum((mx > -INFINITY) ? sm * __expf(mx - m2) : 0.0f);
  if (lane == 0) {
    s_m[warp] = m2;
    s_s[warp] = s2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < NW; ++w) M = fmaxf(M, s_m[w]);
    float S = 0.0f;
#pragma unroll
    for (int w = 0; w < NW; ++w)
      if (s_m[w] > -INFINITY) S += s_s[w] * __expf(s_m[w] - M);
    *reinterpret_cast<float2*>(&a.tile_part[(long long)tile * 8]) = make_float2(M, S);
  }
}

// Per track: the replayed group log-weights of step k, log c_k, lbar_k, and
// at the last step the seed of the reverse sweep, dL = s pi.  FP64 (G-sized).
// The sweep's accumulators are prepared here: the gradient's copies and the
// second dL buffer start at zero at step 0, log Z is set there.
__global__ void __launch_bounds__(RG_GROUP_THREADS) k_replay_groups(ReplayGroupArgs a) {
  grid_dep_wait();
  grid_dep_launch();
  const int t = blockIdx.x;
  const TrackParams& P = a.trk[t];
  const int G = P.G;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
  __shared__ double s_lam[MAX_G];
  __shared__ float s_lamf[MAX_G], s_f[32];
  __shared__ double s_d[32];
  __shared__ double s_lc;
  // L_k,m = LSE over the group's slots, from its tiles' (max, sum exp): a
  // warp per group, its lanes over the tiles
  for (int m = warp; m < G; m += nw) {
    const int t0 = a.gd[P.group_off + m].tile_begin, nt = a.gd[P.group_off + m].tile_count;
    float M = -INFINITY;
    for (int q = lane; q < nt; q += 32) M = fmaxf(M, __ldcg(&a.tile_part[(long long)(t0 + q) * 8]));
    M = warp_max(M);
    float S = 0.0f;
    if (M > -INFINITY)
      for (int q = lane; q < nt; q += 32) {
        const float2 ms = __ldcg(reinterpret_cast<const float2*>(&a.tile_part[(long long)(t0 + q) * 8]));
        if (ms.x > -INFINITY) S = fmaf(ms.y, expf(ms.x - M), S);
      }
    S = warp_sum(S);
    if (lane == 0) {
      const double l = (M > -INFINITY && S > 0.0f) ? (double)M + log((double)S) : -INFINITY;
      s_lam[m] = l;
      s_lamf[m] = (float)l;
    }
  }
  __syncthreads();
  // log c_k = LSE over the groups: the maximum in FP32 (any value near it
  // serves as the scale), FP64 by the warps that hold groups only -- an FP64
  // instruction holds the SM's one pipe for 19 cycles
  float mf = -INFINITY;
  for (int m = threadIdx.x; m < G; m += blockDim.x) mf = fmaxf(mf, s_lamf[m]);
  mf = warp_max(mf);
  if (lane == 0) s_f[warp] = mf;
  __syncthreads();
  const int nwa = nw < (G + 31) / 32 ? nw : (G + 31) / 32;
  mf = -INFINITY;
  for (int w = 0; w < nwa; ++w) mf = fmaxf(mf, s_f[w]);
  const double mx = (double)mf;
  if (warp < nwa) {
    double e = 0.0;
    for (int m = threadIdx.x; m < G; m += blockDim.x) e += s_lam[m] > -INFINITY ? exp(s_lam[m] - mx) : 0.0;
    e = warp_sum_d(e);
    if (lane == 0) s_d[warp] = e;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int w = 0; w < nwa; ++w) tot += s_d[w];
    s_lc = mx + log(tot);
    a.logZ[t] = (a.k > 0 ? a.logZ[t] : 0.0) + s_lc;
  }
  if (a.k == 0) {
    for (int i = threadIdx.x; i < GRAD_COPIES * 5; i += blockDim.x)
      a.grad[((long long)(i / 5) * gridDim.x + t) * GRAD_STRIDE + i % 5] = 0.0;
    for (int m = threadIdx.x; m < G; m += blockDim.x) a.dlam1[P.group_off + m] = 0.0;
  }
  __syncthreads();
  const double lc = s_lc;
  for (int m = threadIdx.x; m < G; m += blockDim.x) {
    const double lam = s_lam[m];
    const long long gm = P.group_off + m;
    a.lam[(long long)a.k * a.G_total + gm] = (float)lam;
    a.lbar[(long long)a.k * a.G_total + gm] = (float)(lam - lc);
    if (a.last) a.dlam[gm] = (double)(a.seed ? a.seed[t] : a.seed0) * exp(lam - lc);
  }
}

// ------------------------------------------------------------------ adjoint
// Adds four neighbouring floats in one L2 operation.
__device__ __forceinline__ void red_add_v4(float4* p, float x, float y, float z, float w) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(__cvta_generic_to_global(p)), "f"(x), "f"(y), "f"(z), "f"(w)
               : "memory");
}

// Reverse step k: the softmax weights from the replay's log-weights, the
// state adjoint (the likelihood's derivatives, stored by the replay, plus the
// children's) and its transposed dynamics onto the recorded parents.  One CTA
// per tile; the particle data is read once, coalesced.  Children of one
// parent sit in neighbouring slots (resampling is monotone), so a segmented
// sum over the warp's runs of equal parents leaves one vector reduction per
// run; any other order is right too, with more of them.  Weight adjoints go
// to the origin group per tile, gradient terms to one of GRAD_COPIES
// accumulators, so that no address takes an atomic per warp.  Bound by the
// 90 bytes a particle it moves and the step's normals it draws again.
template <bool SINGLE>
__global__ void __launch_bounds__(K1_THREADS, 4) k_adjoint(const __grid_constant__ AdjointArgs a) {
  constexpr int NW = K1_THREADS / 32;
  constexpr unsigned FULL = 0xffffffffu;
  const int k = a.k;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ float s_red[NW][8];
  __shared__ int s_other[NW];
  grid_dep_wait();
  grid_dep_launch();
  for (int m = blockIdx.x * K1_THREADS + threadIdx.x; m < a.G_total; m += gridDim.x * K1_THREADS)
    a.dlam_clear[m] = 0.0;
  const int4 td = a.tiles[blockIdx.x];
  const TrackParams& P = SINGLE ? a.p0 : a.trk[td.x];
  const int g = td.y, Np = P.Np;
  const uint32_t* __restrict__ par_t =
      a.parent + P.parent_off + (long long)(k % a.history) * ((long long)P.G * Np);
  const float lam = a.lam_k[P.group_off + g], dlam = (float)a.dlam_k[P.group_off + g];
  uint32_t par[K1_PPT];
  int o[K1_PPT], other = -1;
  float dlw[K1_PPT], cI[K1_PPT];
  float4 c[K1_PPT];
  // sums over the warp: the gradient terms (0 .. 4), and for dL_{k-1} the
  // weight adjoints that came from g (OWN) and from `other` (PRE), one FP32
  // sum per 32 particles and FP64 from there on; the term of A (1) has a value
  // at step 0 only, which has no dL before it
  static_assert(K1_PPT == 2, "one sum per particle of a thread");
  constexpr int OWN[K1_PPT] = {5, 7}, PRE[K1_PPT] = {6, 1};
  float v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
  for (int q = 0; q < K1_PPT; ++q) {
    const int jj = threadIdx.x + q * K1_THREADS;
    const long long il = (long long)g * Np + td.z + jj, i = P.part_off + il;
    par[q] = 0xffffffffu;
    o[q] = g;
    dlw[q] = 0.0f;
    cI[q] = 0.0f;
    c[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (jj < td.w) {
      const float4 d = __ldcs(&a.dl_pv[i]);
      const float db = __ldcs(&a.dl_b[i]), lw = __ldcs(&a.dl_lw[i]);
      if (!a.last) {
        c[q] = __ldcs(&a.Cc_pv[i]);
        cI[q] = __ldcs(&a.Cc_I[i]);
      }
      if (k >= 1) {
        par[q] = par_t[il];
        o[q] = (int)fastdiv(par[q], P.m_Np);  // origin group
      }
      const float wbar = (lw == lw && lw - lam > -87.0f) ? __expf(lw - lam) : 0.0f;
      dlw[q] = dlam * wbar;
      c[q].x = fmaf(dlw[q], d.x, c[q].x);
      c[q].y = fmaf(dlw[q], d.y, c[q].y);
      cI[q] = fmaf(dlw[q], d.z, cI[q]);
      v[0] = fmaf(dlw[q], d.w, v[0]);  // sigma_psf
      v[2] = fmaf(dlw[q], db, v[2]);   // background
    }
    other = max(other, o[q] != g ? o[q] : -1);
  }
  if (k >= 1) {
    // dL_{k-1} of the origin groups: the tile's slots originate in g or in
    // its ring predecessor (slots of any third origin add theirs directly)
    other = __reduce_max_sync(FULL, other);
#pragma unroll
    for (int q = 0; q < K1_PPT; ++q) {
      if (o[q] == g)
        v[OWN[q]] = dlw[q];
      else if (o[q] == other)
        v[PRE[q]] = dlw[q];
      else if (dlw[q] != 0.0f)
        atomicAdd(&a.D[P.group_off + o[q]], (double)dlw[q]);
      const int jj = threadIdx.x + q * K1_THREADS;
      float t[5] = {c[q].x, c[q].y, c[q].x + c[q].z, c[q].y + c[q].w, cI[q]};
      if (jj < td.w) {
        const int j = td.z + jj;
        uint4 w0 = make_uint4(j, g, k, P.tag | (ST_PROP << 4) | 0u);
        uint4 w1 = make_uint4(j, g, k, P.tag | (ST_PROP << 4) | 1u);
        if constexpr (SINGLE)
          philox2_rk(P.rk, w0, w1);
        else
          philox2(P.key0, P.key1, w0, w1);
        float e0, e1, e2, e3;
        box_muller_fast(w0.x, w0.y, e0, e1);
        box_muller_fast(w0.z, w0.w, e2, e3);
        v[3] = fmaf(c[q].x, e0, fmaf(c[q].y, e1, v[3]));  // sigma_pos
        v[4] = fmaf(c[q].z, e2, fmaf(c[q].w, e3, v[4]));  // sigma_v
      }
      // NCV Jacobian transposed onto the parent (x <- x, vx <- x + vx, ...),
      // summed over the run of lanes that share it
      const uint32_t prev = __shfl_up_sync(FULL, par[q], 1);
      const unsigned heads = __ballot_sync(FULL, lane == 0 || par[q] != prev);
      const unsigned above = lane < 31 ? heads >> (lane + 1) : 0u;
      const int left = above ? __ffs(above) - 1 : 31 - lane;  // lanes of the run after this one
#pragma unroll
      for (int dd = 1; dd < 32; dd *= 2) {
        if (!__any_sync(FULL, left >= dd)) break;
#pragma unroll
        for (int x = 0; x < 5; ++x) {
          const float up = __shfl_down_sync(FULL, t[x], dd);
          if (left >= dd) t[x] += up;
        }
      }
      if (((heads >> lane) & 1u) && jj < td.w) {
        const long long pi = P.part_off + par[q];
        red_add_v4(&a.Cp_pv[pi], t[0], t[1], t[2], t[3]);
        atomicAdd(&a.Cp_I[pi], t[4]);
      }
    }
  } else if ((P.init_kind == INIT_POINT) || (P.init_kind == INIT_SHARING && g == 0)) {
#pragma unroll
    for (int q = 0; q < K1_PPT; ++q) v[1] += cI[q];  // the initial intensity is A
  }
  int slot;
  const float x = warp_reduce8(v, lane, slot);
  if ((lane & 3) == 0) s_red[warp][slot] = x;
  if (lane == 0) s_other[warp] = other;
  // the adjoints read above make way for the step before last.  Cleared only
  // now: a store into a line whose load is in flight holds up the load unit
  // (a million particles: 137 us with the stores behind the loads, 27 us here)
#pragma unroll
  for (int q = 0; q < K1_PPT; ++q) {
    const int jj = threadIdx.x + q * K1_THREADS;
    const long long i = P.part_off + (long long)g * Np + td.z + jj;
    if (jj < td.w) {
      a.Cc_pv[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      a.Cc_I[i] = 0.0f;
    }
  }
  __syncthreads();
  // FP64 from here, where an instruction holds the SM's one pipe for 19
  // cycles: a warp's lanes share the sums, four to a slot, and a second warp
  // takes the other origins (one lane summing all eight warps, twice for the
  // second sums, took 7 us more for a million particles)
  static_assert(NW == 8, "two warps' sums per lane");
  if (warp == 0) {
    const int at = lane & 7, w = lane >> 3;
    double r = (double)s_red[w][at] + (double)s_red[w + 4][at];
    r += __shfl_xor_sync(FULL, r, 8);
    r += __shfl_xor_sync(FULL, r, 16);
    const double second = __shfl_down_sync(FULL, r, OWN[1] - OWN[0]);
    if (lane == OWN[0]) r += second;
    if (lane < OWN[0] && r != 0.0 && (lane != PRE[1] || k == 0))
      atomicAdd(&a.grad[((long long)(blockIdx.x % GRAD_COPIES) * a.n_tracks + td.x) * GRAD_STRIDE + lane], r);
    else if (lane == OWN[0] && r != 0.0)
      atomicAdd(&a.D[P.group_off + g], r);
  } else if (warp == 1 && k >= 1) {
    // the warps' second origins, as a rule one group
    const int ow = lane < NW ? s_other[lane] : -1, m = __reduce_max_sync(FULL, ow);
    if (m < 0) return;
    double r = 0.0;
    if (ow >= 0) r = (double)s_red[lane][PRE[0]] + (double)s_red[lane][PRE[1]];
    if (__all_sync(FULL, ow < 0 || ow == m)) {
#pragma unroll
      for (int d = 1; d < NW; d *= 2) r += __shfl_xor_sync(FULL, r, d);
      if (lane != 0) r = 0.0;
      if (r != 0.0) atomicAdd(&a.D[P.group_off + m], r);
    } else if (r != 0.0) {
      atomicAdd(&a.D[P.group_off + ow], r);
    }
  }
}

// The gradient and log Z out of their accumulators.
__global__ void k_grad_out(const double* __restrict__ g, const double* __restrict__ lz, float* __restrict__ out,
                           double* __restrict__ lz_out, int n) {
  grid_dep_wait();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * 5; i += gridDim.x * blockDim.x) {
    double v = 0.0;
#pragma unroll
    for (int c = 0; c < GRAD_COPIES; ++c) v += g[((long long)c * n + i / 5) * GRAD_STRIDE + i % 5];
    out[i] = (float)v;
    if (lz_out && i % 5 == 0) lz_out[i / 5] = lz[i / 5];
  }
}

// ------------------------------------------------------------------ launchers
template <typename Arg, typename... Params>
static cudaError_t launch_pdl(void (*kernel)(Params...), int grid, int block, bool pdl, cudaStream_t s,
                              const Arg& arg) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, arg);
}

template <int R>
static cudaError_t launch_replay_r(const ReplayArgs& a, int n_tiles, bool pdl, cudaStream_t s) {
  if (a.n_tracks == 1) return launch_pdl(k_replay<R, true>, n_tiles, K1_THREADS, pdl, s, a);
  return launch_pdl(k_replay<R, false>, n_tiles, K1_THREADS, pdl, s, a);
}

cudaError_t launch_replay(const ReplayArgs& a, int R, int n_tiles, bool pdl, cudaStream_t s) {
  switch (R) {
    case 1: return launch_replay_r<1>(a, n_tiles, pdl, s);
    case 2: return launch_replay_r<2>(a, n_tiles, pdl, s);
    case 3: return launch_replay_r<3>(a, n_tiles, pdl, s);
    case 4: return launch_replay_r<4>(a, n_tiles, pdl, s);
    case 5: return launch_replay_r<5>(a, n_tiles, pdl, s);
    case 6: return launch_replay_r<6>(a, n_tiles, pdl, s);
    case 7: return launch_replay_r<7>(a, n_tiles, pdl, s);
    default: return cudaErrorInvalidValue;
  }
}

// A warp per group up to 32 groups: with few groups 256 threads suffice.
cudaError_t launch_replay_groups(const ReplayGroupArgs& a, int n_tracks, int max_G, bool pdl, cudaStream_t s) {
  return launch_pdl(k_replay_groups, n_tracks, max_G <= 8 ? 256 : RG_GROUP_THREADS, pdl, s, a);
}

cudaError_t launch_adjoint(const AdjointArgs& a, int n_tiles, bool pdl, cudaStream_t s) {
  if (a.n_tracks == 1) return launch_pdl(k_adjoint<true>, n_tiles, K1_THREADS, pdl, s, a);
  return launch_pdl(k_adjoint<false>, n_tiles, K1_THREADS, pdl, s, a);
}

// Caller-supplied ancestry for the replay (pf_set_replay): for steps k = 1 ..
// T-1 (blockIdx.y + 1), parents[k * n_total + part_off + il] (track-local
// slot of X_{k-1} that slot il of step k was propagated from) into the
// ancestry record the replay reads.  An index outside the track is counted
// in *bad and recorded as the slot itself, so that no later kernel reads
// outside the track.
__global__ void k_set_replay(const TrackParams* __restrict__ trk, const int4* __restrict__ tiles, int n_tiles,
                             const uint32_t* __restrict__ parents, long long n_total, uint32_t* __restrict__ parent,
                             int history, int* __restrict__ bad) {
  const int k = (int)blockIdx.y + 1;
  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int4 td = tiles[tile];
    const TrackParams& P = trk[td.x];
    if (!P.record) continue;
    const long long Nt = (long long)P.G * P.Np;
    for (int jj = threadIdx.x; jj < td.w; jj += blockDim.x) {
      const long long il = (long long)td.y * P.Np + td.z + jj;
      uint32_t v = parents[(long long)k * n_total + P.part_off + il];
      if ((long long)v >= Nt) {
        atomicAdd(bad, 1);
        v = (uint32_t)il;
      }
      parent[P.parent_off + (long long)(k % history) * Nt + il] = v;
    }
  }
}

cudaError_t launch_set_replay(const TrackParams* trk, const int4* tiles, int n_tiles, const uint32_t* parents,
                              long long n_total, uint32_t* parent, int history, int T, int* bad, int grid,
                              cudaStream_t s) {
  if (T < 2) return cudaSuccess;
  k_set_replay<<<dim3(grid, T - 1), 256, 0, s>>>(trk, tiles, n_tiles, parents, n_total, parent, history, bad);
  return cudaGetLastError();
}

cudaError_t launch_grad_out(const double* g, const double* lz, float* out, double* lz_out, int n, cudaStream_t s) {
  k_grad_out<<<(n * 5 + 255) / 256, 256, 0, s>>>(g, lz, out, lz_out, n);
  return cudaGetLastError();
}

}  // namespace pf
