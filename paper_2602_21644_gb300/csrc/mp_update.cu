// Spatiotemporal motion-probability update (Sec. IV-A, Eq. (17)) on sm_103a.
//
//   mp_pixel_sum_kernel   per pixel: residual e(p) between the observed and
//                         the rendered RGB-D, stored; per-region count and sum
//                         (shared-memory partials, one FP64 atomic per region
//                         per CTA)
//   mp_pixel_var_kernel   per pixel: centred squares (e - mean_k)^2 summed per
//                         region the same way (two passes: no cancellation)
//   mp_pixel_map_kernel   per pixel: the fused MP M_p, Eqs. (2)-(7), from
//                         the region statistics; Gamma_geo of a pixel that no
//                         instance claims uses the dispersion of e over the
//                         pixel's own disk of radius r_s (its associated
//                         neighbourhood); stored for the gather
//   mp_pyramid_kernel     per pixel of pyramid level s >= 1 (only when the
//                         association uses S > 1 levels): the 2x2 box mean
//                         of level s - 1 for M_p and e, the 2x2 max for the
//                         rendered depth
//   mp_gauss_kernel       per Gaussian: projection, the association N(G),
//                         Eq. (1), the union over the levels of the disks of
//                         radius r_s around pi(G) / 2^s, over the stored M_p
//                         (or the caller's map); M_hat, Eq. (8), with weights
//                         2^-s exp(-d^2 / (2 sigma_w^2)); Var{M_p}; sigma_e,G;
//                         U, Eq. (10); min/max of U; the observed Gaussians
//                         as a compact list (in no particular order)
//   mp_apply_kernel       one cooperative launch over that list: normalised U,
//                         C, alpha, Eqs. (11), (17); M^t, Eq. (9), written
//                         into the records; exact lower medians of M^t and
//                         U_tilde by radix select (bits 31-21, 20-10, 9-0 of
//                         the non-negative floats, a grid barrier per level);
//                         tau, U_bar; labels, Eq. (12); region statistics
#include <cuda_bf16.h>
#include <math.h>

#include "common.cuh"

namespace dags {

namespace {

constexpr int kMpBlock = 256;
constexpr int kSelBins = 2048;
constexpr int kSelLevels = 3;

struct MpCfg {
  float kappa_c, lam, sigma_min, e_floor, sigma_g, sigma_c, lam_u, eps, alpha_min, alpha_max, rho, r_s, sigma_w,
      vis_tol, z_near, tau_floor;
  int fusion_mode, seg_refreshed, n_regions, scales;
};

constexpr int kMaxScales = DAGS_MP_MAX_SCALES;

// Workspace of the update (carved from the ctx's MP buffers).
struct MpWs {
  float *e;              // [P] residual per pixel
  double *acc;           // [256][4] region count, sum, centred sum of squares, -
  // the observed Gaussians, compact: index, M_hat, sigma_e, U; Mt: their MP,
  // then M^t; Ut: U_tilde
  uint32_t *idx;         // [N]
  float *mhat, *sige, *U, *Mt, *Ut;  // [N]
  uint32_t *hist;        // [kSelLevels][2][kSelBins]
  uint32_t *sel;         // [0] n_obs, [1] Umin bits, [2] Umax bits, [3] arrivals at the grid barriers
  double *stats;         // caller's output
  const float *mp_map;   // [P] external per-pixel MP replacing M_p, or null
  float *mp_pixel;       // [P] out: the fused M_p, or null
  uint32_t *status;      // the ctx's status word (index checks of a DAGS_CHECK build)
  // association pyramid, level s: (M_p or the external map, e, rendered depth,
  // -) per pixel of a row-major Ws x Hs map (level 0: the frame itself), so
  // that the gather takes a pixel with one load instead of three
  float4 *lv[kMaxScales];
  int lw[kMaxScales], lh[kMaxScales];
};

// The region of pixel p (its instance label; checked against the table size
// in a DAGS_CHECK build, where an out-of-range label counts as background).
__device__ __forceinline__ int region_of(const uint8_t *inst, size_t p, int n_regions, uint32_t *status) {
  int k = inst[p];
  if (!DAGS_IN_BOUNDS(k < n_regions, status)) k = 0;
  (void)status;
  return k;
}

// Order-preserving map of floats to uint32 (for atomic min/max of values
// that may be slightly negative).
__device__ __forceinline__ uint32_t f2o(float x) {
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float o2f(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

__device__ __forceinline__ float residual(const float4 tg, const float *img, size_t P, size_t p, float kappa_c) {
  const float dr = img[3 * P + p];
  float e = tg.w > 0.f ? fabsf(tg.w - dr) : 0.f;
  e += kappa_c * (fabsf(tg.x - img[p]) + fabsf(tg.y - img[P + p]) + fabsf(tg.z - img[2 * P + p]));
  return e;
}

__global__ void __launch_bounds__(kMpBlock)
mp_pixel_sum_kernel(MpWs m, const float4 *__restrict__ targets, const float *__restrict__ image,
                    const uint8_t *__restrict__ inst, int P, MpCfg c) {
  pdl_wait();
  __shared__ float s_cnt[DAGS_MP_MAX_REGIONS], s_sum[DAGS_MP_MAX_REGIONS];
  for (int k = threadIdx.x; k < c.n_regions; k += blockDim.x) { s_cnt[k] = 0.f; s_sum[k] = 0.f; }
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  // select state and histograms start cleared (used from mp_gauss_kernel on)
  for (int k = p; k < kSelLevels * 2 * kSelBins; k += gridDim.x * blockDim.x) m.hist[k] = 0u;
  if (p == 0) {
    m.sel[0] = 0u;            // observed count
    m.sel[1] = 0xFFFFFFFFu;   // min of U (ordered key)
    m.sel[2] = 0u;            // max of U (ordered key)
    m.sel[3] = 0u;            // barrier arrivals
  }
  __syncthreads();
  float e = 0.f;
  int k = -1;
  if (p < P) {
    e = residual(targets[p], image, (size_t)P, (size_t)p, c.kappa_c);
    m.e[p] = e;
    k = region_of(inst, p, c.n_regions, m.status);
  }
  // most pixels of a warp share a region: sum per region over the warp
  // first, then one shared atomic per region per warp
  unsigned pending = __ballot_sync(0xffffffffu, k >= 0);
  while (pending) {
    const int leader = __ffs(pending) - 1;
    const int key = __shfl_sync(0xffffffffu, k, leader);
    const bool mine = k == key;
    const unsigned grp = __ballot_sync(0xffffffffu, mine);
    const float sum = warp_sum(mine ? e : 0.f);
    if ((int)(threadIdx.x & 31) == leader) {
      atomicAdd(&s_cnt[key], (float)__popc(grp));
      atomicAdd(&s_sum[key], sum);
    }
    pending &= ~grp;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < c.n_regions; k += blockDim.x)
    if (s_cnt[k] > 0.f) {
      atomicAdd(&m.acc[4 * k + 0], (double)s_cnt[k]);
      atomicAdd(&m.acc[4 * k + 1], (double)s_sum[k]);
    }
}

__global__ void __launch_bounds__(kMpBlock)
mp_pixel_var_kernel(MpWs m, const uint8_t *__restrict__ inst, const float *__restrict__ depth, int P, MpCfg c) {
  pdl_wait();
  __shared__ float s_mean[DAGS_MP_MAX_REGIONS], s_sq[DAGS_MP_MAX_REGIONS];
  for (int k = threadIdx.x; k < c.n_regions; k += blockDim.x) {
    const double cnt = m.acc[4 * k + 0];
    s_mean[k] = cnt > 0.0 ? (float)(m.acc[4 * k + 1] / cnt) : 0.f;
    s_sq[k] = 0.f;
  }
  __syncthreads();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  float sq = 0.f;
  int k = -1;
  if (p < P) {
    k = region_of(inst, p, c.n_regions, m.status);
    const float e = m.e[p], d = e - s_mean[k];
    sq = d * d;
    if (m.mp_map) m.lv[0][p] = make_float4(m.mp_map[p], e, depth[p], 0.f);
  }
  // per-region sums over the warp first, as in the pixel-sum pass
  unsigned pending = __ballot_sync(0xffffffffu, k >= 0);
  while (pending) {
    const int leader = __ffs(pending) - 1;
    const int key = __shfl_sync(0xffffffffu, k, leader);
    const bool mine = k == key;
    const unsigned grp = __ballot_sync(0xffffffffu, mine);
    const float sum = warp_sum(mine ? sq : 0.f);
    if ((int)(threadIdx.x & 31) == leader) atomicAdd(&s_sq[key], sum);
    pending &= ~grp;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < c.n_regions; k += blockDim.x)
    if (s_sq[k] != 0.f) atomicAdd(&m.acc[4 * k + 2], (double)s_sq[k]);
}

// Region parameters used per pixel: mean, e_ub, Gamma_geo, use-mean flag.
__device__ __forceinline__ void region_params(const MpWs &m, const MpCfg &c, int k, float4 *out) {
  const double cnt = m.acc[4 * k + 0];
  const float mean = cnt > 0.0 ? (float)(m.acc[4 * k + 1] / cnt) : 0.f;
  const float sd = cnt > 0.0 ? sqrtf((float)(m.acc[4 * k + 2] / cnt)) : 0.f;
  const float eub = fmaxf(mean + c.lam * sd, c.e_floor);
  const float ggeo = expf(-sd / c.sigma_g);
  const float use_mean = (k >= 1 && sd < c.sigma_min) ? 1.f : 0.f;
  *out = make_float4(mean, eub, ggeo, use_mean);
}

__device__ __forceinline__ float pixel_mp(float e, const float4 reg, const float2 tab, int fusion_mode) {
  const float e_used = reg.w != 0.f ? reg.x : e;
  const float mp_geo = fminf(fmaxf(e_used / reg.y, 0.f), 1.f);
  float K = reg.z / (tab.y + reg.z);
  if (fusion_mode == 1) K = 0.f;
  else if (fusion_mode == 2) K = 1.f;
  return (1.f - K) * tab.x + K * mp_geo;
}

// Population std of e over the disk {(di, dj): di^2 + dj^2 <= r_s^2} around
// pixel (x, y), clipped to the image; two passes (mean, then centred squares).
__device__ __forceinline__ float disk_std(const float *__restrict__ e, int x, int y, int W, int H, float r_s) {
  const int R = (int)floorf(r_s);
  const float rs2 = r_s * r_s;
  const int y0 = max(y - R, 0), y1 = min(y + R, H - 1), x0 = max(x - R, 0), x1 = min(x + R, W - 1);
  float s = 0.f;
  int cnt = 0;
  for (int yy = y0; yy <= y1; ++yy)
    for (int xx = x0; xx <= x1; ++xx) {
      const int di = xx - x, dj = yy - y;
      if ((float)(di * di + dj * dj) > rs2) continue;
      s += __ldg(e + (size_t)yy * W + xx);
      ++cnt;
    }
  const float mean = s / (float)cnt;
  float sq = 0.f;
  for (int yy = y0; yy <= y1; ++yy)
    for (int xx = x0; xx <= x1; ++xx) {
      const int di = xx - x, dj = yy - y;
      if ((float)(di * di + dj * dj) > rs2) continue;
      const float d = __ldg(e + (size_t)yy * W + xx) - mean;
      sq += d * d;
    }
  return sqrtf(sq / (float)cnt);
}

// The same for a disk of at most 5 x 5 pixels (floor(r_s) = 2, the default
// radius): the box unrolled, one pass over the values less the centre's
// (sums of d and d^2, whose mean square less the squared mean is the
// population variance; the shift keeps both sums small).
__device__ __forceinline__ float disk_std_r2(const float *__restrict__ e, int x, int y, int W, int H, float rs2) {
  const float c = __ldg(e + (size_t)y * W + x);
  float s = 0.f, s2 = 0.f, cnt = 0.f;
#pragma unroll
  for (int dj = -2; dj <= 2; ++dj) {
    const int yy = y + dj;
    const bool row = yy >= 0 && yy < H;
#pragma unroll
    for (int di = -2; di <= 2; ++di) {
      const int xx = x + di;
      if (row && xx >= 0 && xx < W && (float)(di * di + dj * dj) <= rs2) {
        const float d = __ldg(e + (size_t)yy * W + xx) - c;
        s += d;
        s2 = fmaf(d, d, s2);
        cnt += 1.f;
      }
    }
  }
  const float m = s / cnt;
  return sqrtf(fmaxf(s2 / cnt - m * m, 0.f));
}

// The fused per-pixel M_p map, Eqs. (2)-(7): read by the gather and, when
// asked for, returned to the caller (who may train or evaluate a learned
// proposal against the method). Gamma_geo = exp(-sigma / sigma_g) takes the
// region's sigma_e inside an instance and, for a pixel that no instance
// claims, the dispersion over the pixel's associated neighbourhood (the
// sentence after Eq. (7)), read as its disk of radius r_s.
__global__ void __launch_bounds__(kMpBlock)
mp_pixel_map_kernel(MpWs m, const uint8_t *__restrict__ inst, const float2 *__restrict__ table,
                    const float *__restrict__ depth, int W, int H, MpCfg c) {
  pdl_wait();
  __shared__ float4 s_reg[DAGS_MP_MAX_REGIONS];
  __shared__ float2 s_tab[DAGS_MP_MAX_REGIONS];
  for (int k = threadIdx.x; k < c.n_regions; k += blockDim.x) {
    region_params(m, c, k, &s_reg[k]);
    s_tab[k] = table[k];
  }
  __syncthreads();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < W * H) {
    const int k = region_of(inst, p, c.n_regions, m.status);
    float4 reg = s_reg[k];
    if (k == 0) {
      const float sd = floorf(c.r_s) == 2.f ? disk_std_r2(m.e, p % W, p / W, W, H, c.r_s * c.r_s)
                                            : disk_std(m.e, p % W, p / W, W, H, c.r_s);
      reg.z = expf(-sd / c.sigma_g);
    }
    const float e = m.e[p], mp = pixel_mp(e, reg, s_tab[k], c.fusion_mode);
    if (!m.mp_map) m.lv[0][p] = make_float4(mp, e, depth[p], 0.f);
    if (m.mp_pixel) m.mp_pixel[p] = mp;
  }
}

// Level s of the association pyramid from level s - 1: each pixel covers a
// 2x2 block; M_p and e take the block's mean, the rendered depth its maximum
// (the occlusion test's maximum over a level-s pixel is then the maximum over
// the full-resolution pixels it covers).
__global__ void __launch_bounds__(kMpBlock)
mp_pyramid_kernel(MpWs m, int s) {
  pdl_wait();
  const int W = m.lw[s], H = m.lh[s], Wp = m.lw[s - 1];
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= W * H) return;
  const int x = q % W, y = q / W;
  const float4 *in = m.lv[s - 1] + (size_t)(2 * y) * Wp + 2 * x;
  const float4 a = in[0], b = in[1], c = in[Wp], d = in[Wp + 1];
  m.lv[s][q] = make_float4(((a.x + b.x) + (c.x + d.x)) * 0.25f, ((a.y + b.y) + (c.y + d.y)) * 0.25f,
                           fmaxf(fmaxf(a.z, b.z), fmaxf(c.z, d.z)), 0.f);
}

// The pixel rectangle of the disk of radius r_s around (us, vs) clipped to a
// Ws x Hs level; false when it is empty (or the centre is not finite).
__device__ __forceinline__ bool disk_rect(float us, float vs, int Ws, int Hs, float r_s, int *i0, int *i1, int *j0,
                                          int *j1) {
  if (!(us > -r_s - 1.f && us < (float)Ws + r_s && vs > -r_s - 1.f && vs < (float)Hs + r_s)) return false;
  *i0 = (int)fmaxf(ceilf(us - r_s), 0.f);
  *i1 = (int)fminf(floorf(us + r_s), (float)(Ws - 1));
  *j0 = (int)fmaxf(ceilf(vs - r_s), 0.f);
  *j1 = (int)fminf(floorf(vs + r_s), (float)(Hs - 1));
  return *i0 <= *i1 && *j0 <= *j1;
}

// Sums over the members of N(G): f(level weight, dx^2 + dy^2, pixel, level).
// kSmall: r_s <= 2, so a row of the disk has at most five pixels: the row is
// unrolled with its loads side by side (a member outside the disk adds zero,
// which leaves the sums' bits as they are). The squared distance is rounded
// explicitly: a pixel on the disk's rim is in or out alike in both forms and
// whatever else the compiler contracts.
template <bool kSmall, typename F>
__device__ __forceinline__ void for_disk(const MpWs &m, const MpCfg &c, float u, float v, F &&f) {
  const float rs2 = c.r_s * c.r_s;
#pragma unroll
  for (int s = 0; s < kMaxScales; ++s) {
    if (s >= c.scales) break;
    const float sc = 1.f / (float)(1 << s);              // 2^-s: exact
    const float us = u * sc, vs = v * sc;
    const int Ws = m.lw[s];
    int i0, i1, j0, j1;
    if (!disk_rect(us, vs, Ws, m.lh[s], c.r_s, &i0, &i1, &j0, &j1)) continue;
    for (int jj = j0; jj <= j1; ++jj) {
      const size_t row = (size_t)jj * Ws;
      const float dy = (float)jj - vs;
      if (kSmall) {
#pragma unroll
        for (int t = 0; t < 5; ++t) {
          const int ii = i0 + t;
          const float dx = (float)ii - us, d2 = __fmaf_rn(dx, dx, __fmul_rn(dy, dy));
          f(sc, d2, row + (size_t)min(ii, i1), s, ii <= i1 && !(d2 > rs2));
        }
      } else {
        for (int ii = i0; ii <= i1; ++ii) {
          const float dx = (float)ii - us, d2 = __fmaf_rn(dx, dx, __fmul_rn(dy, dy));
          if (!(d2 > rs2)) f(sc, d2, row + (size_t)ii, s, true);
        }
      }
    }
  }
}

// A thread per Gaussian, bound by the latency of the gathers (up to 13 pixels x
// 3 levels, twice). With M_p, e and depth of a pixel in one 16-byte load instead
// of three maps: 75 -> 55 us for 1M Gaussians and three levels. Maps are appended frame by frame, so Gaussians in view
// come in runs and fill their warps: compacting them per CTA first made the
// CTAs uneven (300k Gaussians: 42 us against 17).
template <bool kSmall>
__global__ void __launch_bounds__(kMpBlock)
mp_gauss_kernel(MpWs m, const float4 *__restrict__ gauss, int64_t n, const double *__restrict__ pose, Raster r,
                MpCfg c) {
  pdl_wait();
  __shared__ float sp[12];
  __shared__ uint32_t s_min, s_max, s_obs, s_base;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 12) sp[threadIdx.x] = (float)pose[threadIdx.x];
  if (threadIdx.x == 0) { s_min = 0xFFFFFFFFu; s_max = 0u; s_obs = 0u; }
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool observed = false;
  float mhat = 0.f, sige = 0.f, U = 0.f, M0 = 0.f;
  if (i < n) {
    const float4 g0 = __ldg(gauss + 4 * i);
    const float x = sp[0] * g0.x + sp[1] * g0.y + sp[2] * g0.z + sp[3];
    const float y = sp[4] * g0.x + sp[5] * g0.y + sp[6] * g0.z + sp[7];
    const float z = depth_key(g0, sp);
    const float u = r.fx * x / z + r.cx, v = r.fy * y / z + r.cy;
    if (z > c.z_near) {
      const float inv2s2 = 1.f / (2.f * c.sigma_w * c.sigma_w);
      float sw = 0.f, swm = 0.f, sm = 0.f, se = 0.f, dmax = -INFINITY;
      int cnt = 0;
      for_disk<kSmall>(m, c, u, v, [&](float sc, float d2, size_t p, int s, bool ok) {
        const float4 t = ok ? __ldg(m.lv[s] + p) : make_float4(0.f, 0.f, -INFINITY, 0.f);
        const float w = ok ? sc * expf(-d2 * inv2s2) : 0.f;
        sw += w; swm = __fmaf_rn(w, t.x, swm); sm += t.x; se += t.y; cnt += ok;
        dmax = fmaxf(dmax, t.z);
      });
      observed = cnt > 0 && !(c.vis_tol > 0.f && dmax > 0.f && z > dmax + c.vis_tol);
      if (observed) {
        mhat = swm / sw;
        const float mm = sm / cnt, me = se / cnt;
        float vm = 0.f, ve = 0.f;
        for_disk<kSmall>(m, c, u, v, [&](float, float, size_t p, int s, bool ok) {
          const float4 t = ok ? __ldg(m.lv[s] + p) : make_float4(mm, me, 0.f, 0.f);
          const float de = ok ? t.y - me : 0.f, dm = ok ? t.x - mm : 0.f;
          vm = __fmaf_rn(dm, dm, vm);
          ve = __fmaf_rn(de, de, ve);
        });
        sige = sqrtf(ve / cnt);
        M0 = __ldg(reinterpret_cast<const float *>(gauss + 4 * i) + 11);
        U = -M0 * logf(M0 + c.eps) - (1.f - M0) * logf(1.f - M0 + c.eps) + c.lam_u * (vm / cnt);
        atomicMin(&s_min, f2o(U));
        atomicMax(&s_max, f2o(U));
      }
    }
  }
  const unsigned b = __ballot_sync(0xffffffffu, observed);
  uint32_t at = 0u;
  if (lane == 0 && b) at = atomicAdd(&s_obs, (uint32_t)__popc(b));
  at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & ((1u << lane) - 1u));
  __syncthreads();
  if (threadIdx.x == 0 && s_obs) {
    atomicMin(&m.sel[1], s_min);
    atomicMax(&m.sel[2], s_max);
    s_base = atomicAdd(&m.sel[0], s_obs);
  }
  __syncthreads();
  if (observed) {
    const size_t q = (size_t)s_base + at;
    m.idx[q] = (uint32_t)i;
    m.U[q] = U;
    m.sige[q] = sige;
    m.mhat[q] = mhat;
    m.Mt[q] = M0;
  }
}

constexpr int kApplyBlock = 1024;
constexpr int kApplyHeld = 8;      // list entries that a thread keeps in registers
constexpr int kBarrierSpins = 1 << 22;

// All CTAs of the grid (a cooperative launch) have arrived `round` times;
// false, with the timeout recorded, if one did not within `spins` iterations.
__device__ bool grid_barrier(uint32_t *arrivals, uint32_t round, int spins, uint32_t *status) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(arrivals, 1u);
    bool ok = false;
    for (int it = 0; it < spins && !ok; ++it) {
      uint32_t v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(arrivals) : "memory");
      ok = v >= round * gridDim.x;
    }
    if (!ok) atomicOr(status, kStatusTimeout);
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Failure-path self-test: the one CTA waits for a second arrival that nothing
// makes. scratch[0] counts arrivals, [1] is the status that an earlier wait
// recorded its timeout in, [2] this one's; the ctx's status gets the timeout if
// both did.
__global__ void selftest_barrier_kernel(uint32_t *scratch, int spins, uint32_t *status) {
  const bool ok = grid_barrier(scratch, 2u, spins, scratch + 2);
  if (threadIdx.x == 0 && !ok && (__ldcg(scratch + 1) & __ldcg(scratch + 2) & kStatusTimeout))
    atomicOr(status, kStatusTimeout);
}

// Radix-select level l of the floats' bits: 31-21, 20-10, 9-0.
__device__ __forceinline__ int select_shift(int level) { return level == 0 ? 21 : level == 1 ? 10 : 0; }

// For the ranks rank[0], rank[1]: the bins of the two histograms (kSelBins
// each, contiguous) that hold them, and the ranks within those bins. The
// CTA's halves take a histogram each, a thread four bins.
__device__ void find_bins(const uint32_t *hist, uint32_t *rank, uint32_t *bin) {
  __shared__ uint32_t s_sum[32], s_bin[2], s_rank[2];
  const int h = threadIdx.x / (kApplyBlock / 2), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  static_assert(kSelBins == 4 * (kApplyBlock / 2), "four bins per thread");
  const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(hist) + threadIdx.x);
  const uint32_t mine = v.x + v.y + v.z + v.w;
  uint32_t inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_sum[warp] = inc;
  __syncthreads();
  uint32_t before = inc - mine;
  for (int w = 16 * h; w < warp; ++w) before += s_sum[w];
  const uint32_t r = rank[h];
  if (before <= r && r < before + mine) {
    uint32_t b = 4u * (threadIdx.x % (kApplyBlock / 2)), run = before;
    const uint32_t cnt[3] = {v.x, v.y, v.z};
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (b % 4u == (uint32_t)k && r >= run + cnt[k]) { run += cnt[k]; ++b; }
    s_bin[h] = b;
    s_rank[h] = r - run;
  }
  __syncthreads();
  for (int k = 0; k < 2; ++k) { bin[k] = s_bin[k]; rank[k] = s_rank[k]; }
  __syncthreads();
}

// The list is read once; each thread keeps its entries' M^t and U_tilde in
// registers over the three select levels and the labels (entries past
// kApplyHeld per thread, above 1.2M observed, are read again). Every CTA finds
// the bins for itself after a barrier, so that no level waits for one CTA.
// In place of five launches that each walked all N Gaussians and ended on one
// CTA's serial search: 51 -> 23 us at 300k Gaussians, each launch alone.
__global__ void __launch_bounds__(kApplyBlock, 1)
mp_apply_kernel(MpWs m, float *__restrict__ gauss, uint8_t *__restrict__ labels, MpCfg c) {
  __shared__ uint32_t s_h[2 * kSelBins];
  const uint32_t nobs = m.sel[0];
  const float umin = o2f(m.sel[1]), umax = o2f(m.sel[2]);
  const size_t T = (size_t)gridDim.x * kApplyBlock, first = (size_t)blockIdx.x * kApplyBlock + threadIdx.x;
  if (blockIdx.x == gridDim.x - 1)
    for (int k = threadIdx.x; k < c.n_regions; k += kApplyBlock) {
      float4 reg;
      region_params(m, c, k, &reg);
      const double cnt = m.acc[4 * k + 0];
      double *o = m.stats + DAGS_MP_STATS_HEAD + 4 * k;
      o[0] = cnt;
      o[1] = cnt > 0.0 ? m.acc[4 * k + 1] / cnt : 0.0;
      o[2] = cnt > 0.0 ? sqrt(m.acc[4 * k + 2] / cnt) : 0.0;
      o[3] = reg.y;
    }
  if (nobs == 0u) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      m.stats[0] = (double)c.tau_floor;
      m.stats[1] = 0.0;
      m.stats[2] = nanf("");
      m.stats[3] = m.stats[4] = m.stats[5] = 0.0;
    }
    return;
  }
  uint32_t id[kApplyHeld];
  float Mt[kApplyHeld], Ut[kApplyHeld];
  auto apply = [&](size_t q, uint32_t *i, float *M, float *Un) {
    const float ut = umax > umin ? (m.U[q] - umin) / (umax - umin) : 0.f;
    const float C = expf(-m.sige[q] / c.sigma_c);
    float a = c.alpha_min + (c.alpha_max - c.alpha_min) * (1.f - ut) * C;
    a = fminf(fmaxf(a, c.alpha_min), c.alpha_max);
    if (!c.seg_refreshed) a *= c.rho;
    *i = m.idx[q];
    *Un = ut;
    *M = (1.f - a) * m.Mt[q] + a * m.mhat[q];
    gauss[16 * (size_t)*i + 11] = *M;
  };
#pragma unroll
  for (int j = 0; j < kApplyHeld; ++j) {
    const size_t q = first + j * T;
    id[j] = 0u;
    Mt[j] = Ut[j] = 0.f;
    if (q < nobs) apply(q, &id[j], &Mt[j], &Ut[j]);
  }
  for (size_t q = first + kApplyHeld * T; q < nobs; q += T) {
    uint32_t i;
    float M, Un;
    apply(q, &i, &M, &Un);
    m.Mt[q] = M;
    m.Ut[q] = Un;
  }
  uint32_t rank[2] = {(nobs - 1u) / 2u, (nobs - 1u) / 2u}, prefix[2] = {0u, 0u};
  for (int level = 0; level < kSelLevels; ++level) {
    for (int k = threadIdx.x; k < 2 * kSelBins; k += kApplyBlock) s_h[k] = 0u;
    __syncthreads();
    const int shift = select_shift(level);
    const uint32_t mask = level == 2 ? 0x3FFu : 0x7FFu;
    auto count = [&](float M, float Un) {
      // the bits above this level equal the prefix
      const uint32_t bm = __float_as_uint(M), bu = __float_as_uint(Un);
      if (level == 0 || ((bm ^ prefix[0]) >> shift) <= mask) atomicAdd(&s_h[(bm >> shift) & mask], 1u);
      if (level == 0 || ((bu ^ prefix[1]) >> shift) <= mask) atomicAdd(&s_h[kSelBins + ((bu >> shift) & mask)], 1u);
    };
#pragma unroll
    for (int j = 0; j < kApplyHeld; ++j)
      if (first + j * T < nobs) count(Mt[j], Ut[j]);
    for (size_t q = first + kApplyHeld * T; q < nobs; q += T) count(m.Mt[q], m.Ut[q]);
    __syncthreads();
    uint32_t *hist = m.hist + level * 2 * kSelBins;
    for (int k = threadIdx.x; k < 2 * kSelBins; k += kApplyBlock)
      if (s_h[k]) atomicAdd(&hist[k], s_h[k]);
    if (!grid_barrier(m.sel + 3, (uint32_t)level + 1u, kBarrierSpins, m.status)) return;
    uint32_t bin[2];
    find_bins(hist, rank, bin);
    prefix[0] |= bin[0] << shift;
    prefix[1] |= bin[1] << shift;
  }
  const float medM = __uint_as_float(prefix[0]);
  const double tau = fmax((double)medM, (double)c.tau_floor);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    m.stats[0] = tau;
    m.stats[1] = __uint_as_float(prefix[1]);
    m.stats[2] = medM;
    m.stats[3] = (double)umin;
    m.stats[4] = (double)umax;
    m.stats[5] = (double)nobs;
  }
#pragma unroll
  for (int j = 0; j < kApplyHeld; ++j)
    if (first + j * T < nobs) labels[id[j]] = (double)Mt[j] > tau ? 1 : 0;
  for (size_t q = first + kApplyHeld * T; q < nobs; q += T) labels[m.idx[q]] = (double)m.Mt[q] > tau ? 1 : 0;
}

// Semantic-on-demand trigger, Eqs. (13)-(16): one thread reads the frame's
// U_bar and background residual mean from the MP statistics.
__global__ void semantic_trigger_kernel(const double *__restrict__ stats, double w_u, double w_r, double theta,
                                        double e_ref, int n_max, int seg_refreshed, int32_t *state,
                                        double *score) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double u_bar = stats[1];
  const double cnt0 = stats[DAGS_MP_STATS_HEAD + 0];
  const double e_bar = cnt0 > 0.0 ? stats[DAGS_MP_STATS_HEAD + 1] : 0.0;
  const double R = fmin(fmax(e_bar / e_ref, 0.0), 1.0);
  const double S = w_u * u_bar + w_r * R;
  const int since = seg_refreshed ? 0 : state[0] + 1;
  state[0] = since;
  state[1] = (S > theta || since + 1 >= n_max) ? 1 : 0;
  if (score) {
    score[0] = e_bar;
    score[1] = R;
    score[2] = S;
  }
}

}  // namespace

cudaError_t launch_selftest_barrier(uint32_t *scratch, int spins, uint32_t *status, cudaStream_t s) {
  selftest_barrier_kernel<<<1, 32, 0, s>>>(scratch, spins < kBarrierSpins ? spins : kBarrierSpins, status);
  return cudaGetLastError();
}

cudaError_t launch_mp_update(const MpBuffers &b, float *gauss, int64_t n, const double *pose, const Raster &r,
                             const float4 *targets, const float *image, const uint8_t *inst, const float *table,
                             int n_regions, const dags_mp_cfg &cfg, int seg_refreshed, uint8_t *labels,
                             double *stats, const float *mp_map, float *mp_pixel, uint32_t *status,
                             int num_sms, cudaStream_t s) {
  MpWs m;
  m.status = status;
  m.mp_map = mp_map;
  m.mp_pixel = mp_pixel;
  m.e = b.e; m.acc = b.acc; m.mhat = b.mhat; m.sige = b.sige; m.U = b.U; m.Mt = b.Mt; m.Ut = b.Ut;
  m.idx = b.idx; m.hist = b.hist; m.sel = b.sel; m.stats = stats;
  MpCfg c;
  c.kappa_c = cfg.kappa_c; c.lam = cfg.lam; c.sigma_min = cfg.sigma_min; c.e_floor = cfg.e_floor;
  c.sigma_g = cfg.sigma_g; c.sigma_c = cfg.sigma_c; c.lam_u = cfg.lam_u; c.eps = cfg.eps;
  c.alpha_min = cfg.alpha_min; c.alpha_max = cfg.alpha_max; c.rho = cfg.rho; c.r_s = cfg.r_s;
  c.sigma_w = cfg.sigma_w; c.vis_tol = cfg.vis_tol; c.z_near = cfg.z_near; c.tau_floor = cfg.tau_floor;
  c.fusion_mode = cfg.fusion_mode; c.seg_refreshed = seg_refreshed; c.n_regions = n_regions;
  c.scales = cfg.scales < 1 ? 1 : (cfg.scales > kMaxScales ? kMaxScales : cfg.scales);
  const int P = r.W * r.H;
  float4 *level = b.levels;
  for (int l = 0; l < kMaxScales; ++l) {
    m.lw[l] = r.W >> l;
    m.lh[l] = r.H >> l;
    m.lv[l] = level;
    level += (size_t)m.lw[l] * m.lh[l];
  }
  const float *depth = image + 3 * (size_t)P;
  // the region accumulators start at zero (the select state is cleared by
  // the first kernel)
  cudaError_t e = cudaMemsetAsync(b.acc, 0, DAGS_MP_MAX_REGIONS * 4 * sizeof(double), s);
  if (e != cudaSuccess) return e;
  const unsigned gp = (unsigned)((P + kMpBlock - 1) / kMpBlock);
  const unsigned gg = (unsigned)((n + kMpBlock - 1) / kMpBlock > 0 ? (n + kMpBlock - 1) / kMpBlock : 1);
  const int64_t blocks = (n + kApplyBlock - 1) / kApplyBlock;
  const unsigned ga = (unsigned)(blocks < 1 ? 1 : blocks < num_sms ? blocks : num_sms);
  mp_pixel_sum_kernel<<<gp, kMpBlock, 0, s>>>(m, targets, image, inst, P, c);
  if (e == cudaSuccess) e = launch_pdl(mp_pixel_var_kernel, dim3(gp), dim3(kMpBlock), 0, s, m, inst, depth, P, c);
  if (!mp_map || mp_pixel)
    if (e == cudaSuccess)
      e = launch_pdl(mp_pixel_map_kernel, dim3(gp), dim3(kMpBlock), 0, s, m, inst,
                     reinterpret_cast<const float2 *>(table), depth, r.W, r.H, c);
  for (int l = 1; l < c.scales; ++l) {
    const int Pl = m.lw[l] * m.lh[l];
    if (Pl > 0 && e == cudaSuccess)
      e = launch_pdl(mp_pyramid_kernel, dim3((unsigned)((Pl + kMpBlock - 1) / kMpBlock)), dim3(kMpBlock), 0, s, m, l);
  }
  if (e == cudaSuccess)
    e = launch_pdl(c.r_s <= 2.f ? mp_gauss_kernel<true> : mp_gauss_kernel<false>, dim3(gg), dim3(kMpBlock), 0, s, m,
                   reinterpret_cast<const float4 *>(gauss), n, pose, r, c);
  if (e == cudaSuccess) {
    // cooperative: its CTAs (one per SM at most) wait for one another
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ga);
    cfg.blockDim = dim3(kApplyBlock);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, mp_apply_kernel, m, gauss, labels, c);
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

cudaError_t launch_semantic_trigger(const double *stats, const dags_sched_cfg &cfg, int seg_refreshed,
                                    int32_t *state, double *score, cudaStream_t s) {
  semantic_trigger_kernel<<<1, 32, 0, s>>>(stats, cfg.w_u, cfg.w_r, cfg.theta, cfg.e_ref, cfg.n_max,
                                           seg_refreshed ? 1 : 0, state, score);
  return cudaGetLastError();
}

}  // namespace dags

namespace dags {

namespace {

__device__ __forceinline__ uint32_t bf16x2_bits(float lo, float hi) {
  const uint32_t a = __bfloat16_as_ushort(__float2bfloat16_rn(lo));
  const uint32_t b = __bfloat16_as_ushort(__float2bfloat16_rn(hi));
  return a | (b << 16);
}

// Per-pixel input of the learned MP network: rendered MP, |dC| (3), |dD|
// where the observed depth is valid, observed depth, rendered opacity, the
// MP_ins of the pixel's region (Eq. (2)); one 16-byte BF16 row per pixel.
__global__ void __launch_bounds__(kMpBlock)
mpnet_features_kernel(const float *__restrict__ image, const float4 *__restrict__ targets,
                      const uint8_t *__restrict__ inst, const float2 *__restrict__ table, int n_regions, int P,
                      uint4 *__restrict__ feats, uint32_t *status) {
  __shared__ float s_mu[DAGS_MP_MAX_REGIONS];
  for (int k = threadIdx.x; k < n_regions; k += blockDim.x) s_mu[k] = table[k].x;
  __syncthreads();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const size_t Q = (size_t)P;
  const float4 t = __ldg(targets + p);
  const float cr = __ldg(image + p), cg = __ldg(image + Q + p), cb = __ldg(image + 2 * Q + p);
  const float d = __ldg(image + 3 * Q + p), o = __ldg(image + 4 * Q + p), rmp = __ldg(image + 5 * Q + p);
  const bool valid = t.w > 0.f;
  const int k = region_of(inst, p, n_regions, status);
  feats[p] = make_uint4(bf16x2_bits(rmp, fabsf(t.x - cr)), bf16x2_bits(fabsf(t.y - cg), fabsf(t.z - cb)),
                        bf16x2_bits(valid ? fabsf(t.w - d) : 0.f, valid ? t.w : 0.f), bf16x2_bits(o, s_mu[k]));
}

}  // namespace

cudaError_t launch_mpnet_features(const float *image, const float4 *targets, const uint8_t *inst, const float *table,
                                  int n_regions, int P, uint16_t *feats, uint32_t *status, cudaStream_t s) {
  if (P <= 0) return cudaSuccess;
  mpnet_features_kernel<<<(P + kMpBlock - 1) / kMpBlock, kMpBlock, 0, s>>>(
      image, targets, inst, reinterpret_cast<const float2 *>(table), n_regions, P, reinterpret_cast<uint4 *>(feats),
      status);
  return cudaGetLastError();
}

}  // namespace dags
