// Levenberg-Marquardt pose refinement (Sec. V-A(c)) on sm_103a.
//
// The tracking objective is the MP-weighted L1 loss of Eqs. (20)-(22) with
// the static weight w(u) held constant in the linearisation. Its L1 terms
// enter a weighted least-squares problem by iterative reweighting: channel
// residual r with coefficient c (lambda_pho w for r, g, b; lambda_depth w
// where the observed depth is valid) gets the weight W = c / max(|r|, delta).
// One iteration:
//
//   preprocess, tile scan, emit    as for the forward (splat_fwd.cu)
//   pose_tangent_kernel   per visible Gaussian, the derivative of its 2D
//                         record (centre, conic in log2 units, depth) along
//                         the six twist directions xi = (rho, phi) of the
//                         left perturbation T <- exp(xi^) T; beside it, one CTA
//                         per tile depth-sorts the tile's bucket
//   render_jac_kernel     one warp per 8x4 pixel block: the forward compositing
//                         with forward-mode tangents (the derivative of alpha,
//                         of the transmittance and of the composited colour
//                         and depth, 30 accumulators per pixel), then per
//                         pixel the loss and W J J^T, W r J; summed per block
//                         and tile in FP32 and over tiles in FP64, each in a
//                         fixed order, into (L, H, g)
//   LM step               FP64, one warp: accept the linearisation point if its
//                         loss is lower, adapt the damping, solve the damped
//                         6x6 system by Cholesky and step the pose, spread over
//                         the lanes; inside the tracking loop it is the last
//                         warp of render_jac_kernel, on its own lm_step_kernel
//
// The kernels use programmatic dependent launch like the other splatting
// kernels: each waits for its predecessor's memory before its first access.
#include "common.cuh"
#include "tile_sort.cuh"

namespace dags {

namespace {

constexpr int kJacChunk = 8;    // entries a warp stages at a time
constexpr int kTan4 = 9;         // float4 per Gaussian tangent record (36 floats)
constexpr int kNormal = 28;      // L, the upper triangle of H (21), g (6)
constexpr int kTanBlock = kTilePix;      // threads per CTA of the tangents and the sort
constexpr int kBlocks = kTilePix / 32;   // pixel blocks per tile
constexpr int kTileGroup = kLmTileGroup; // tiles whose partials one warp sums in FP64

// Tangent record of a visible Gaussian: for twist direction k = 0..5 the six
// floats (du, dv, da', db', dc', dz), where (a', b', c') are the exponent
// coefficients of the projected record (log2 units). Directions 2p and 2p + 1
// are interleaved, so that a component of both is one aligned register pair.
__host__ __device__ constexpr int tan_at(int k, int c) { return (k >> 1) * 12 + 2 * c + (k & 1); }

// The grid: (tracking loop) one CTA that ranks the tiles by the previous
// Jacobian render's counts into this iteration's render order, dispatched
// first; one CTA per tile that sorts its bucket (an overflowed one is left);
// CTAs that stride over the visible Gaussians. The sort needs nothing of the
// tangents, so it fills the SMs beside them, and the render after it runs
// without a CTA per tile.
__global__ void __launch_bounds__(kTanBlock, 3)
pose_tangent_kernel(Workspace ws, const float4 *__restrict__ gauss, int64_t n, Raster r,
                    float4 *__restrict__ tan) {
  pdl_wait();
  const int ordering = ws.order_next != nullptr ? 1 : 0;
  if (ordering && blockIdx.x == 0) {
    rank_tiles(ws.prev_count, r.T, ws.order_next, ws.band);
    return;
  }
  const int64_t lead = ordering + (int64_t)r.T;
  if ((int64_t)blockIdx.x < lead) {
    __shared__ __align__(16) uint64_t s_key[kSortSmallCap];
    const int tile = (int)blockIdx.x - ordering;
    if (ws.bucket_cap ? ws.tile_count[tile] > ws.bucket_cap : pairs_overflow_ws(ws)) return;
    uint32_t s, e;
    tile_range(ws, tile, s, e);
    sort_tile_bucket(ws, s, (int)(e - s), s_key);
    return;
  }
  const int64_t nb = (int64_t)gridDim.x - lead;
  const int64_t bid = (int64_t)blockIdx.x - lead;
  // the tracking loop's bucket layout: the visible list is still the
  // preprocess's append cursor
  const uint32_t nv = ws.bucket_cap ? ws.vis_append[0] : ws.vis_n[0];
  float P[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) P[k] = ws.pose32[k];
  for (int64_t t = bid * blockDim.x + threadIdx.x; t < (int64_t)nv; t += nb * blockDim.x) {
    const uint32_t id = ws.vis_ids[t];
    if (!DAGS_IN_BOUNDS(id < (uint64_t)n, ws.counters + CNT_STATUS)) continue;
    const float4 g0 = __ldg(gauss + 4 * id), g1 = __ldg(gauss + 4 * id + 1), g2 = __ldg(gauss + 4 * id + 2);
    Proj q;
    float out[36];
    if (!project_gaussian(g0, g1, g2, P, r, q)) {
#pragma unroll
      for (int k = 0; k < 36; ++k) out[k] = 0.f;
    } else {
      const float x = q.x, y = q.y, z = q.z;
      const float iz = 1.f / z, iz2 = iz * iz;
      const bool clx = q.txz > r.limx || q.txz < -r.limx;
      const bool cly = q.tyz > r.limy || q.tyz < -r.limy;
      const float idet = 1.f / q.det;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        // camera mean: e_k (rho), phi x p (phi); K = R_cw Rq S: [phi]x K
        float dp[3] = {0.f, 0.f, 0.f}, dK[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) dK[e] = 0.f;
        if (k < 3) {
          dp[k] = 1.f;
        } else if (k == 3) {
          dp[1] = -z; dp[2] = y;
#pragma unroll
          for (int s = 0; s < 3; ++s) { dK[3 + s] = -q.K[6 + s]; dK[6 + s] = q.K[3 + s]; }
        } else if (k == 4) {
          dp[0] = z; dp[2] = -x;
#pragma unroll
          for (int s = 0; s < 3; ++s) { dK[s] = q.K[6 + s]; dK[6 + s] = -q.K[s]; }
        } else {
          dp[0] = -y; dp[1] = x;
#pragma unroll
          for (int s = 0; s < 3; ++s) { dK[s] = -q.K[3 + s]; dK[3 + s] = q.K[s]; }
        }
        // the guard clamp freezes x/z (y/z) in the Jacobian
        const float dtx = clx ? 0.f : (dp[0] * z - x * dp[2]) * iz2;
        const float dty = cly ? 0.f : (dp[1] * z - y * dp[2]) * iz2;
        const float dj00 = -r.fx * dp[2] * iz2, dj02 = -r.fx * (dtx * z - q.tx * dp[2]) * iz2;
        const float dj11 = -r.fy * dp[2] * iz2, dj12 = -r.fy * (dty * z - q.ty * dp[2]) * iz2;
        float dA = 0.f, dB = 0.f, dC = 0.f;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          const float dm0 = dj00 * q.K[s] + q.j00 * dK[s] + dj02 * q.K[6 + s] + q.j02 * dK[6 + s];
          const float dm1 = dj11 * q.K[3 + s] + q.j11 * dK[3 + s] + dj12 * q.K[6 + s] + q.j12 * dK[6 + s];
          dA += 2.f * q.m0[s] * dm0;
          dC += 2.f * q.m1[s] * dm1;
          dB += dm0 * q.m1[s] + q.m0[s] * dm1;
        }
        // conic (ca, cb, cc) = (C, -B, A) / det
        const float ddet = dA * q.C + q.A * dC - 2.f * q.B * dB;
        const float dca = (dC - q.ca * ddet) * idet;
        const float dcb = (-dB - q.cb * ddet) * idet;
        const float dcc = (dA - q.cc * ddet) * idet;
        out[tan_at(k, 0)] = r.fx * (dp[0] * z - x * dp[2]) * iz2;
        out[tan_at(k, 1)] = r.fy * (dp[1] * z - y * dp[2]) * iz2;
        out[tan_at(k, 2)] = -0.5f * kLog2e * dca;
        out[tan_at(k, 3)] = -kLog2e * dcb;
        out[tan_at(k, 4)] = -0.5f * kLog2e * dcc;
        out[tan_at(k, 5)] = dp[2];
      }
    }
    float4 *o = tan + (size_t)id * kTan4;
#pragma unroll
    for (int w = 0; w < kTan4; ++w) o[w] = make_float4(out[4 * w], out[4 * w + 1], out[4 * w + 2], out[4 * w + 3]);
  }
}

// Index of H[a][b] (a <= b) in the packed upper triangle.
__host__ __device__ constexpr int tri(int a, int b) { return a * 6 - a * (a - 1) / 2 + (b - a); }

// LM state (DAGS_LM_STATE doubles): T_best[12], L_best, mu, H_best[21],
// g_best[6], accepted count, iteration count, last L, last accepted flag.
enum { ST_T = 0, ST_L = 12, ST_MU = 13, ST_H = 14, ST_G = 35, ST_ACC = 41, ST_IT = 42, ST_LAST_L = 43,
       ST_LAST_A = 44 };

// The LM step by one warp (all lanes must call it): decide, solve the damped
// system and step the pose, on shared-memory copies of the normal equations at
// the linearisation point, the state and the pose. FP64 instructions are what
// it costs (each occupies the pipe as long for one lane as for 32, and they
// depend on one another), so the factorisation, the solves and the exponential
// are spread over the lanes: 7 us against 10 for one lane.
__device__ void lm_step_warp(const double *nrm, double *state, double *pose_try, double *pose_best,
                             const dags_lm_cfg &c) {
  __shared__ double s_st[DAGS_LM_STATE], s_A[6][6], s_x[6], s_sc[3];
  const unsigned FULL = 0xffffffffu;
  const int t = threadIdx.x & 31;
  const bool accept = nrm[0] < state[ST_L];
  double mu = state[ST_MU];
  mu = accept ? fmax(mu * c.down, c.mu_min) : fmin(mu * c.up, c.mu_max);
  for (int k = t; k < DAGS_LM_STATE; k += 32) s_st[k] = state[k];
  __syncwarp();
  if (accept) {
    if (t < 12) s_st[ST_T + t] = pose_try[t];
    if (t < 21) s_st[ST_H + t] = nrm[1 + t];
    if (t < 6) s_st[ST_G + t] = nrm[22 + t];
  }
  if (t == 0) {
    if (accept) {
      s_st[ST_L] = nrm[0];
      s_st[ST_ACC] += 1.0;
    }
    s_st[ST_MU] = mu;
    s_st[ST_IT] += 1.0;
    s_st[ST_LAST_L] = nrm[0];
    s_st[ST_LAST_A] = accept ? 1.0 : 0.0;
  }
  __syncwarp();
  // (H + mu diag(H) + floor tr(H)/6 I) delta = -g by Cholesky: lane (i, j) of
  // the lower triangle holds A[i][j]; column k's lanes are scaled by the
  // reciprocal square root of the pivot, then every lane to their right
  // subtracts its product (the diagonal holds 1 / l_jj)
  double tr = 0.0;
  for (int a = 0; a < 6; ++a) tr += s_st[ST_H + tri(a, a)];
  bool ok = tr > 0.0;
  int i = 0, j = t;                 // lane t < 21: row i, column j <= i
  while (i < 5 && j > i) { j -= i + 1; ++i; }
  const bool mine = t < 21;
  double v = 0.0;
  if (mine) {
    v = s_st[ST_H + tri(j, i)];
    if (i == j) v += mu * v + c.floor * (tr / 6.0);
  }
  for (int k = 0; k < 6; ++k) {
    const int diag = k * (k + 1) / 2 + k;   // lane of A[k][k]
    const double piv = __shfl_sync(FULL, v, diag);
    if (!(piv > 0.0)) ok = false;
    const double inv = rsqrt(piv);
    if (mine && j == k) {
      v = i == k ? inv : v * inv;
      s_A[i][k] = v;
    }
    __syncwarp();
    if (mine && j > k) v -= s_A[i][k] * s_A[j][k];
  }
  // forward and back substitution: lane i holds row i's running sum
  double x = t < 6 ? -s_st[ST_G + t] : 0.0;
  for (int k = 0; k < 6; ++k) {
    const double y = __shfl_sync(FULL, x, k) * s_A[k][k];
    if (t == k) x = y;
    else if (t > k && t < 6) x -= s_A[t][k] * y;
  }
  for (int k = 5; k >= 0; --k) {
    const double d = __shfl_sync(FULL, x, k) * s_A[k][k];
    if (t == k) x = d;
    else if (t < k) x -= s_A[k][t] * d;
  }
  if (t < 6) s_x[t] = ok ? x : 0.0;
  __syncwarp();
  // T <- exp(delta^) T, an entry to a lane
  se3_exp_coeffs(s_x, s_sc, t);
  __syncwarp();
  const double out = t < 12 ? se3_exp_entry(s_st + ST_T, s_x, s_sc, t) : 0.0;
  for (int k = t; k < DAGS_LM_STATE; k += 32) state[k] = s_st[k];
  if (t < 12) {
    pose_try[t] = out;
    pose_best[t] = s_st[ST_T + t];
  }
}

// One warp arrives at `counter`; true for the last of `count`, which then sees
// what the others wrote before they arrived, and leaves the counter at zero.
__device__ __forceinline__ bool arrive_last(uint32_t *counter, uint32_t count) {
  __syncwarp();
  uint32_t t = 0;
  if ((threadIdx.x & 31) == 0) {
    __threadfence();
    t = atomicAdd(counter, 1u);
    if (t == count - 1u) {
      *counter = 0u;
      __threadfence();
    }
  }
  __syncwarp();   // the fence orders lane 0's view; this passes it on to the other lanes
  return __shfl_sync(0xffffffffu, t, 0) == count - 1u;
}

// One warp, and one CTA, per 8 x 4 pixel block, as in the adjoint of the
// first-order loop: bound by the latency of a warp's own chain (59% of the
// issue slots used, FP32 pipe next) and by the number of warps that 30 tangent
// accumulators per pixel leave room for (20 per SM at 96 registers; 24 spill
// and are slower, as are 16 and 18). The six twist directions run in pairs on
// the packed FP32 operations, so a pair's 84 operations issue as 42. 300k
// Gaussians, 640x480, per launch: 122 us and 64M warp instructions; 146 us with
// a CTA of 8 warps per tile that sorts its bucket, scalar (93M) or packed (77M:
// its warps wait on one another). The sort went beside the tangents, the sums
// and the step over warps and lanes, and the next entry is read ahead.
__global__ void __launch_bounds__(32, 20)
render_jac_kernel(Workspace ws, Raster r, Loss l, float delta, const float4 *__restrict__ targets,
                  const float4 *__restrict__ tan, LmBuffers buf, double *__restrict__ normal,
                  float *__restrict__ jac, float *__restrict__ image, int32_t *__restrict__ last, LmFuse fuse) {
  pdl_wait();
  // records and tangent records of a chunk's entries, double-buffered: word w of
  // entry j at w * kJacChunk + j
  __shared__ float4 s_rec[2][(4 + kTan4) * kJacChunk];
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x;
  const int warp = (int)(blockIdx.x % kBlocks);   // the tile's pixel block
  // the tracking loop's fixed-capacity buckets: a tile whose list overflowed
  // its bucket is skipped and reported, and the render publishes the counts
  // and the visible count as the forward of the first-order loop does;
  // otherwise an overflow anywhere skips every tile
  bool ovf;
  int tile;
  if (ws.bucket_cap) {
    tile = (int)ws.tile_order[blockIdx.x / kBlocks];
    const uint32_t c = ws.tile_count[tile];
    ovf = c > ws.bucket_cap;
    if (warp == 0 && lane == 0) {
      ws.prev_count[tile] = c;
      atomicMax(reinterpret_cast<unsigned long long *>(ws.counters + CNT_REQ_LO), (unsigned long long)c * r.T);
      if (ovf) atomicOr(ws.counters + CNT_STATUS, kStatusCapacity);
      if (blockIdx.x == 0) {
        ws.vis_n[0] = ws.vis_append[0];
        ws.vis_append[0] = 0u;
      }
    }
  } else {
    ovf = pairs_overflow_ws(ws);
    tile = (int)(ovf ? blockIdx.x / kBlocks : ws.tile_order[blockIdx.x / kBlocks]);
  }
  const int tx = tile % r.tiles_x, ty = tile / r.tiles_x;
  const int bx0 = tx * kTile + (warp & 1) * 8, by0 = ty * kTile + (warp >> 1) * 4;
  const int px = bx0 + (lane & 7), py = by0 + (lane >> 3);
  const bool inside = px < r.W && py < r.H;
  uint32_t s = 0u, e = 0u;
  if (!ovf) tile_range(ws, tile, s, e);
  const float bcx = (float)bx0 + 3.5f, bcy = (float)by0 + 1.5f;
  const int len = (int)(e - s);

  float T = 1.f, cr = 0.f, cg = 0.f, cb = 0.f, dd = 0.f, oo = 0.f, rm = 0.f;
  // tangents of T and of the composited channels, directions in pairs
  f32x2 dT2[3], jr2[3], jg2[3], jb2[3], jd2[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) dT2[k] = jr2[k] = jg2[k] = jb2[k] = jd2[k] = 0ull;
  const f32x2 minus1 = dup2(-1.f);
  int lastk = 0;
  bool done = !inside;
  const float fpx = (float)px, fpy = (float)py;
  // The list in groups of 32 entries, in depth order; of a group, the entries
  // whose box meets the block, in chunks of up to kJacChunk. While a chunk is
  // worked on, the records and tangents of the next are on their way to shared
  // memory; the boxes of the next group and the ids of the one after are on
  // their way to registers.
  auto load_id = [&](int g) -> uint32_t {
    const int k = g * 32 + lane;
    if (k >= len) return 0u;
    const uint32_t id = __ldg(ws.sorted_ids + s + k);
    return DAGS_IN_BOUNDS(id < (uint32_t)ws.max_n, ws.counters + CNT_STATUS) ? id : 0u;
  };
  auto load_box = [&](uint32_t id) {   // {u, v, ex, ey}
    const float4 r0 = __ldg(ws.rec2d + (size_t)id * 4), r3 = __ldg(ws.rec2d + (size_t)id * 4 + 3);
    return make_float4(r0.x, r0.y, r3.y, r3.z);
  };
  const int groups = (len + 31) >> 5;
  int pg = -1;                     // the group being staged
  unsigned pend = 0u;              // its entries that are still to be staged
  uint32_t pid = 0u, nid = load_id(0), nnid = load_id(1);
  float4 nbox = load_box(nid);
  // stages the next chunk; its entries as bits of group pg (0: the list's end)
  auto stage = [&](int b) -> unsigned {
    while (pend == 0u && pg + 1 < groups) {
      ++pg;
      pid = nid;
      const float4 box = nbox;
      nid = nnid;
      nnid = load_id(pg + 2);
      nbox = load_box(nid);
      pend = __ballot_sync(FULL, pg * 32 + lane < len && fabsf(box.x - bcx) <= box.z + 3.5f &&
                                     fabsf(box.y - bcy) <= box.w + 1.5f);
    }
    const int rank = __popc(pend & ((1u << lane) - 1u));
    const bool take = ((pend >> lane) & 1u) != 0u && rank < kJacChunk;
    if (take) {
      const float4 *rec = ws.rec2d + (size_t)pid * 4, *tg = tan + (size_t)pid * kTan4;
#pragma unroll
      for (int w = 0; w < 4; ++w) cp_async16(&s_rec[b][w * kJacChunk + rank], rec + w);
#pragma unroll
      for (int w = 0; w < kTan4; ++w) cp_async16(&s_rec[b][(4 + w) * kJacChunk + rank], tg + w);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const unsigned chunk = __ballot_sync(FULL, take);
    pend ^= chunk;
    return chunk;
  };
  unsigned mask_next = groups > 0 ? stage(0) : 0u;
  for (int cur = 0; mask_next; cur ^= 1) {
    unsigned mask = mask_next;
    const int kbase = pg * 32 + 1;
    mask_next = stage(cur ^ 1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
    const float4 *const rec = s_rec[cur];
    float4 a = rec[0], b = rec[kJacChunk];
    for (int j = 0; mask; ++j) {
      const int bit = __ffs((int)mask) - 1;
      mask &= mask - 1;
      // alpha is evaluated by every lane; a lane that is done, or whose alpha
      // is below alpha_min, or that would stop here leaves the sums alone (a
      // zero weight would not: a Gaussian's colour may be infinite)
      const float dx = (a.x - fpx) + a.z, dy = (a.y - fpy) + a.w;
      const float p = fmaf(b.x * dx, dx, fmaf(b.y * dx, dy, fmaf(b.z * dy, dy, b.w)));
      const bool live = !done && p >= r.log2_alpha_min;
      const float ag = hw_exp2(p);
      const bool clamped = ag > r.alpha_max;
      const float alpha = clamped ? r.alpha_max : ag;
      const float tt = T * (1.f - alpha);
      const bool stop = live && tt < r.t_min;
      const bool contrib = live && !stop;
      done = done || stop;
      const float gxs = fmaf(2.f * b.x, dx, b.y * dy), gys = fmaf(b.y, dx, 2.f * b.z * dy);
      // the next entry's centre and conic (past the chunk's last, the buffer's
      // following word, which nothing uses)
      a = rec[j + 1];
      b = rec[kJacChunk + j + 1];
      if (contrib) {
        const float w = alpha * T;
        const float4 c = rec[2 * kJacChunk + j];
        const float blue = rec[3 * kJacChunk + j].x;
        cr += c.z * w; cg += c.w * w; cb += blue * w;
        dd += c.x * w; oo += w; rm += c.y * w;
        // tangents: p' = da' dx^2 + db' dx dy + dc' dy^2 + dp/du du + dp/dv dv,
        // alpha' = alpha ln2 p' (0 where clamped), weight' = alpha' T + alpha T';
        // the next entry's T = T - weight, so its T' = T' - weight'
        const f32x2 gx = dup2(gxs), gy = dup2(gys);
        const f32x2 pdx = dup2(dx), pdy = dup2(dy);
        const f32x2 dx2 = mul2(pdx, pdx), dxy = mul2(pdx, pdy), dy2 = mul2(pdy, pdy);
        const f32x2 aln = dup2(clamped ? 0.f : alpha * kLn2), al2 = dup2(alpha);
        const f32x2 T2 = dup2(T), w2 = dup2(w);
        const f32x2 cz2 = dup2(c.x), cr2 = dup2(c.z), cg2 = dup2(c.w), cb2 = dup2(blue);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const ulonglong2 uv = *reinterpret_cast<const ulonglong2 *>(&rec[(4 + 3 * k) * kJacChunk + j]);
          const ulonglong2 ab = *reinterpret_cast<const ulonglong2 *>(&rec[(5 + 3 * k) * kJacChunk + j]);
          const ulonglong2 cz = *reinterpret_cast<const ulonglong2 *>(&rec[(6 + 3 * k) * kJacChunk + j]);
          const f32x2 dp = fma2(ab.x, dx2, fma2(ab.y, dxy, fma2(cz.x, dy2, fma2(gx, uv.x, mul2(gy, uv.y)))));
          const f32x2 da = mul2(aln, dp);
          const f32x2 dw = fma2(da, T2, mul2(al2, dT2[k]));
          jr2[k] = fma2(cr2, dw, jr2[k]);
          jg2[k] = fma2(cg2, dw, jg2[k]);
          jb2[k] = fma2(cb2, dw, jb2[k]);
          jd2[k] = fma2(cz2, dw, fma2(w2, cz.y, jd2[k]));
          dT2[k] = fma2(dw, minus1, dT2[k]);
        }
        T = tt;
        lastk = kbase + bit;
      }
    }
    __syncwarp();   // the chunk's buffer is staged again in the next round
    if (__all_sync(FULL, done)) break;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");   // no copy outlives the warp

  float jr[6], jg[6], jb[6], jd[6];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    unpack2(jr2[k], jr[2 * k], jr[2 * k + 1]);
    unpack2(jg2[k], jg[2 * k], jg[2 * k + 1]);
    unpack2(jb2[k], jb[2 * k], jb[2 * k + 1]);
    unpack2(jd2[k], jd[2 * k], jd[2 * k + 1]);
  }
  float acc[kNormal];
#pragma unroll
  for (int k = 0; k < kNormal; ++k) acc[k] = 0.f;
  if (inside) {
    const size_t P = (size_t)r.W * r.H;
    const size_t pix = (size_t)py * r.W + px;
    float wgt;
    if (l.weight_mode == 0) wgt = oo > l.o_eps ? (oo - rm) / oo : 0.f;
    else wgt = oo - rm;
    const float4 tg = targets[pix];
    const bool dvalid = tg.w > 0.f;
    if (tg.x >= 0.f) {
      const float res[4] = {cr - tg.x, cg - tg.y, cb - tg.z, dd - tg.w};
      const float coef[4] = {l.lambda_pho * wgt, l.lambda_pho * wgt, l.lambda_pho * wgt,
                             dvalid ? l.lambda_depth * wgt : 0.f};
      const float l1 = fabsf(res[0]) + fabsf(res[1]) + fabsf(res[2]);
      acc[0] = wgt * (l.lambda_pho * l1 + (dvalid ? l.lambda_depth * fabsf(res[3]) : 0.f));
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        const float *J = ch == 0 ? jr : ch == 1 ? jg : ch == 2 ? jb : jd;
        const float W = coef[ch] / fmaxf(fabsf(res[ch]), delta);
#pragma unroll
        for (int a = 0; a < 6; ++a) {
          const float wa = W * J[a];
          acc[22 + a] = fmaf(wa, res[ch], acc[22 + a]);
#pragma unroll
          for (int b2 = a; b2 < 6; ++b2) acc[1 + tri(a, b2)] = fmaf(wa, J[b2], acc[1 + tri(a, b2)]);
        }
      }
    }
    if (jac) {
      float4 *jp = reinterpret_cast<float4 *>(jac + pix * 24);
      jp[0] = make_float4(jr[0], jr[1], jr[2], jr[3]);
      jp[1] = make_float4(jr[4], jr[5], jg[0], jg[1]);
      jp[2] = make_float4(jg[2], jg[3], jg[4], jg[5]);
      jp[3] = make_float4(jb[0], jb[1], jb[2], jb[3]);
      jp[4] = make_float4(jb[4], jb[5], jd[0], jd[1]);
      jp[5] = make_float4(jd[2], jd[3], jd[4], jd[5]);
    }
    if (image) {
      float *img = image + pix;
      img[0 * P] = cr; img[1 * P] = cg; img[2 * P] = cb; img[3 * P] = dd;
      img[4 * P] = oo; img[5 * P] = rm; img[6 * P] = T; img[7 * P] = wgt;
    }
    if (last) last[pix] = lastk;
  }
  // block sums, the tile's eight in order, a group's tiles and the groups: the
  // last warp to arrive at each level sums the level below in a fixed order
  // (FP64 additions run at two per cycle and SM, so they are spread over the
  // groups' last warps)
  {
    const float v = warp_reduce_scatter<kNormal, 16>(acc, lane);
    const int comp = rs_component<kNormal>(lane);
    if (__ffs(__match_any_sync(FULL, (unsigned)comp)) - 1 == lane)
      buf.block_partial[((size_t)tile * kBlocks + warp) * kNormal + comp] = v;
  }
  if (!arrive_last(buf.done + tile, kBlocks)) return;
  if (lane < kNormal) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kBlocks; ++w) t += __ldcg(buf.block_partial + ((size_t)tile * kBlocks + w) * kNormal + lane);
    buf.partial[(size_t)tile * kNormal + lane] = t;
  }
  // the bucket is empty again for the next iteration's binning (the tile's
  // warps have read its range)
  if (ws.bucket_cap && lane == 0) ws.tile_count[tile] = 0u;
  const int group = tile / kTileGroup, ngroups = (r.T + kTileGroup - 1) / kTileGroup;
  const int first = group * kTileGroup, in_group = min(kTileGroup, r.T - first);
  if (!arrive_last(buf.done + r.T + group, (uint32_t)in_group)) return;
  if (lane < kNormal) {
    double a4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int k = 0; k < in_group; ++k) a4[k & 3] += (double)__ldcg(buf.partial + (size_t)(first + k) * kNormal + lane);
    buf.group_partial[(size_t)group * kNormal + lane] = (a4[0] + a4[1]) + (a4[2] + a4[3]);
  }
  if (!arrive_last(buf.done + r.T + ngroups, (uint32_t)ngroups)) return;
  __shared__ double s_nrm[kNormal];
  // a pair-capacity overflow leaves tiles unrendered (all of them in the
  // general layout; in the bucket layout those whose list exceeded its
  // bucket, which the largest requirement of this iteration tells)
  bool any_ovf = ovf;
  if (ws.bucket_cap)
    any_ovf = __ldcg(reinterpret_cast<const unsigned long long *>(ws.counters + CNT_REQ_LO)) >
              (unsigned long long)ws.bucket_cap * (unsigned long long)r.T;
  if (lane < kNormal) {
    double a4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int k = 0; k < ngroups; ++k) a4[k & 3] += __ldcg(buf.group_partial + (size_t)k * kNormal + lane);
    double t = (a4[0] + a4[1]) + (a4[2] + a4[3]);
    // then the loss is NaN, so the LM step rejects this point
    if (any_ovf && lane == 0) t = __longlong_as_double(0x7ff8000000000000ll);
    normal[lane] = t;
    s_nrm[lane] = t;
  }
  __syncwarp();
  // inside the LM loop the step runs here, in the last warp
  if (fuse.state) {
    lm_step_warp(s_nrm, fuse.state, fuse.pose_try, fuse.pose_best, fuse.cfg);
    // the bucket layout: if the next linearisation point (as the preprocess
    // stages it in FP32) has left the bounds the candidates were culled for,
    // move the culling pose to it and empty the list; the next preprocess
    // then takes every Gaussian once and re-culls
    if (ws.bucket_cap && ws.cand_n && ws.cull_pose) {
      __shared__ float s_np[12];
      __syncwarp();
      if (lane < 12) s_np[lane] = __double2float_rn(fuse.pose_try[lane]);
      __syncwarp();
      const bool out = !within_cull_bounds(s_np, ws.cull_pose);
      __syncwarp();
      if (out && lane < 12) ws.cull_pose[lane] = s_np[lane];
      if (lane == 0) {
        if (out) *ws.cand_n = 0u;
        ws.counters[CNT_RECULL] = out ? 1u : 0u;
      }
    }
  }
}

__global__ void lm_init_kernel(const double *__restrict__ pose, double *__restrict__ state,
                               double *__restrict__ pose_try, double mu0) {
  pdl_wait();
  const int t = threadIdx.x;
  if (t < 12) {
    state[ST_T + t] = pose[t];
    pose_try[t] = pose[t];
  }
  if (t >= 12 && t < DAGS_LM_STATE) state[t] = 0.0;
  __syncthreads();
  if (t == 0) {
    state[ST_L] = __longlong_as_double(0x7ff0000000000000ll);   // +inf: the first point is accepted
    state[ST_MU] = mu0;
  }
}

__global__ void lm_step_kernel(const double *__restrict__ normal, double *__restrict__ state,
                               double *__restrict__ pose_try, double *__restrict__ pose_best, dags_lm_cfg c) {
  pdl_wait();
  lm_step_warp(normal, state, pose_try, pose_best, c);
}

}  // namespace

cudaError_t launch_pose_tangents(const Workspace &ws, const float4 *gauss, int64_t n, const Raster &r, float4 *tan,
                                 int num_sms, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int64_t need = (n + kTanBlock - 1) / kTanBlock;
  const unsigned grid = (unsigned)(need < (int64_t)num_sms * 3 ? need : (int64_t)num_sms * 3);
  // the visible Gaussians' CTAs, the tiles' and, in the tracking loop, the
  // ranking one
  return launch_pdl(pose_tangent_kernel, dim3(grid + (unsigned)r.T + (ws.order_next ? 1u : 0u)), dim3(kTanBlock), 0, s,
                    ws, gauss, n, r, tan);
}

cudaError_t launch_render_jac(const Workspace &ws, const Raster &r, const Loss &l, float delta,
                              const float4 *targets, const LmBuffers &buf, double *normal, float *jac, float *image,
                              int32_t *last, const LmFuse &fuse, cudaStream_t s) {
  return launch_pdl(render_jac_kernel, dim3((unsigned)r.T * kBlocks), dim3(32), 0, s, ws, r, l, delta, targets,
                    (const float4 *)buf.tan, buf, normal, jac, image, last, fuse);
}

cudaError_t launch_lm_init(const double *pose, double *state, double *pose_try, double mu0, cudaStream_t s) {
  return launch_pdl(lm_init_kernel, dim3(1), dim3(64), 0, s, pose, state, pose_try, mu0);
}

cudaError_t launch_lm_step(const double *normal, double *state, double *pose_try, double *pose_best,
                           const dags_lm_cfg &c, cudaStream_t s) {
  return launch_pdl(lm_step_kernel, dim3(1), dim3(32), 0, s, normal, state, pose_try, pose_best, c);
}

}  // namespace dags
