// Backward half of the MP-aware splatting path (sm_103a).
//
//   render_bwd_kernel      one warp per 8x4 pixel block: walks its tile's sorted
//                          list back to front from the furthest recorded
//                          contributor, re-deriving each pixel's
//                          transmittance from its final value (T_k =
//                          T_{k+1} / (1 - alpha_k)) with running suffix sums,
//                          so no per-pair state is stored; the 2D-gradient
//                          moments of the 32 pixels of a warp are summed with
//                          shuffles and added with one atomic per word per
//                          (warp, Gaussian) pair.
//   preprocess_bwd_kernel  per Gaussian over all views: chains the 2D
//                          gradients through conic, EWA covariance, Jacobian,
//                          camera transform, scale and rotation to the record's
//                          parameters, and to the pose twist (mean and
//                          covariance paths); per-view pose partials are summed
//                          per CTA and then, by the last CTA, in a fixed order
//                          in FP64.
#include "common.cuh"
#include "tile_sort.cuh"

namespace dags {

namespace {

constexpr int kMaxViewsSmem = 64;
// the pose path's words are the first two float4 (the preprocess zeroes only those)
static_assert(G2_E == 0 && G2_YY == 4 && G2_Z == 5 && G2_BL == 9 && kGradWords >= 10, "2D-gradient word order");

// Warp sums of an entry's moments over the warp's 8 x 4 pixels (lane = 8 row +
// column). dy depends on the row only, so m0, m1, m2 = g, g e, g e^2 and the
// depth and colour terms are first reduce-scattered over each row's 8 lanes, and
// the y factors are applied to the row sums: 7 + 2 shuffles for the ten words
// and 4 + 2 for the pose path's six (a reduce-scatter of all words over 32 lanes
// takes 12 and 8, and needs every word formed per pixel). The terms are given as
// x = (m1, m2, z, r, g, b, m0), or (m1, m2, z, m0) for the pose path; after the
// row stage lane l8 = lane & 7 holds
//   FULL:      m1, m2, z, m0, r, g, b, m0
//   pose only: m1, m1, m2, m2, z, z, m0, m0
// and the rows are summed as is by the lanes below 16, weighted with dy by the
// others, with l8 = 7 taking dy^2. moment_word: the word a lane ends up with
// (-1: it writes none).
template <bool FULL>
__device__ __forceinline__ int moment_word(int lane) {
  const int l8 = lane & 7;
  if (lane & 8) return -1;
  if (lane & 16) return l8 == 0 ? G2_EY : (l8 == (FULL ? 3 : 6) ? G2_Y : -1);
  if (l8 == 0) return G2_E;
  if (l8 == 7) return G2_YY;
  if (FULL) return l8 == 1 ? G2_EE : l8 == 2 ? G2_Z : l8 == 3 ? G2_S0 : l8 == 4 ? G2_R : l8 == 5 ? G2_G : G2_BL;
  return l8 == 2 ? G2_EE : l8 == 4 ? G2_Z : -1;
}

template <int K>
__device__ __forceinline__ float moment_sums(const float (&x)[K], float dy, int lane) {
  const unsigned FULLM = 0xffffffffu;
  const float v = warp_reduce_scatter<K, 4>(x, lane);
  const float b = v * dy;
  const float a = (lane & 7) == 7 ? b * dy : v;
  const bool hi = (lane & 16) != 0;
  const float keep = hi ? b : a, send = hi ? a : b;
  const float s = keep + __shfl_xor_sync(FULLM, send, 16);
  return s + __shfl_xor_sync(FULLM, s, 8);
}

// FULL: every parameter's 2D gradients (else the pose path's six words);
// MOMENTS: words 0-4 as moments (see G2_E), else as gradients formed per pixel;
// MASKS: visit only the entries the forward recorded as taken by the warp
// (ws.warp_masks); COUNT: count evaluations and contributions (ws.evals).
// One warp, and one CTA, per 8 x 4 pixel block: no barrier joins the blocks of a
// tile, a block with few entries leaves its slot at once, and the short blocks
// launched last even out the SMs (with a CTA of 8 warps per tile, a frame's
// 1,200 CTAs kept the SMs busy for 77% of the kernel and half of a busy SM's
// warp slots). The warp stages the taken entries of a 32-entry group with
// cp.async while it works on the group before, and works on two entries at a
// time. 300k Gaussians, 640x480, pose only: 67 us per CTA of 8 warps, 58 and 54
// per warp in CTAs of two and one, 52 with two entries at a time; all
// gradients: 74 -> 66 us; 2,000 Gaussians, 160x120: 60 -> 42 us.
constexpr int kBlocks = kTilePix / 32;   // pixel blocks per tile

template <bool FULL, bool MOMENTS, bool MASKS, bool COUNT>
__global__ void __launch_bounds__(32, 32)
render_bwd_kernel(Workspace ws, Raster r, Loss l, const float4 *__restrict__ targets,
                  const float *__restrict__ image, const int32_t *__restrict__ last,
                  const float *__restrict__ upstream) {
  pdl_wait();
  pdl_trigger();
  __shared__ float4 s_rec[2][4][32];   // projected records, double-buffered
  const unsigned FULLM = 0xffffffffu;
  const int lane = threadIdx.x;
  const int warp = (int)(blockIdx.x % kBlocks);   // the tile's pixel block
  // an overflow of the packed layout leaves every tile out; in the
  // fixed-bucket layout a tile that overflowed has no contributors
  if (!ws.bucket_cap) {
    const uint64_t tot = (uint64_t)ws.counters[CNT_REQ_LO] | ((uint64_t)ws.counters[CNT_REQ_HI] << 32);
    if (tot > (uint64_t)ws.max_pairs) return;
  }
  // the 2D-gradient word whose warp sum this lane adds, if any (of the lanes
  // that hold one word, the lowest)
  int word;
  if constexpr (MOMENTS) {
    word = moment_word<FULL>(lane);
  } else {
    word = rs_component<10>(lane);
    if (__ffs(__match_any_sync(FULLM, (unsigned)word)) - 1 != lane) word = -1;
  }
  const bool writer = word >= 0;
  const int tile = (int)ws.tile_order[blockIdx.x / kBlocks];   // longest lists first
  const int v = tile / r.T, tv = tile - v * r.T;
  const int tx = tv % r.tiles_x, ty = tv / r.tiles_x;
  const int bx0 = tx * kTile + (warp & 1) * 8, by0 = ty * kTile + (warp >> 1) * 4;
  const int px = bx0 + (lane & 7), py = by0 + (lane >> 3);
  const bool inside = px < r.W && py < r.H;
  const uint32_t s = ws.bucket_cap ? (uint32_t)tile * ws.bucket_cap : ws.tile_start[tile];
  // the forward's record of the entries this warp's pixels took (groups of
  // 32 entries; later groups fall back to the box test)
  const uint32_t *const wmask = MASKS ? ws.warp_masks + (size_t)tile * kMaskGroups * 8 + warp : nullptr;
  const float4 *const recs = ws.rec2d + (size_t)v * ws.max_n * 4;
  float *const gdst = ws.grad2d + (size_t)v * ws.max_n * kGradWords + (writer ? word : 0);
  const size_t P = (size_t)r.W * r.H;
  const float bcx = (float)bx0 + 3.5f, bcy = (float)by0 + 1.5f;

  float T = 1.f;
  float g0 = 0.f, g1 = 0.f, g2 = 0.f, g3 = 0.f, g4 = 0.f, g5 = 0.f;  // upstream per channel
  int lastp = 0;
  if (inside && upstream) {
    // the caller's gradients of its own function of the six composited
    // channels take the place of the loss's
    const size_t pix = (size_t)py * r.W + px;
    const float *up = upstream + (size_t)v * 6 * P + pix;
    g0 = up[0]; g1 = up[P]; g2 = up[2 * P]; g3 = up[3 * P]; g4 = up[4 * P]; g5 = up[5 * P];
    T = image[(size_t)v * DAGS_IMG_CHANNELS * P + 6 * P + pix];
    lastp = last[(size_t)v * P + pix];
  } else if (inside) {
    // a pixel whose target has negative red is outside the loss (no gradient)
    const size_t pix = (size_t)py * r.W + px;
    const float *img = image + (size_t)v * DAGS_IMG_CHANNELS * P + pix;
    const float cr = img[0], cg = img[P], cb = img[2 * P], dd = img[3 * P];
    const float oo = img[4 * P], rm = img[5 * P];
    T = img[6 * P];
    const float w = img[7 * P];
    const float4 tg = targets[(size_t)v * P + pix];
    lastp = tg.x >= 0.f ? last[(size_t)v * P + pix] : 0;
    const float rc0 = cr - tg.x, rc1 = cg - tg.y, rc2 = cb - tg.z, rd = dd - tg.w;
    const bool dvalid = tg.w > 0.f;
    auto sgn = [](float x) { return (float)((x > 0.f) - (x < 0.f)); };
    g0 = l.lambda_pho * w * sgn(rc0);
    g1 = l.lambda_pho * w * sgn(rc1);
    g2 = l.lambda_pho * w * sgn(rc2);
    g3 = dvalid ? l.lambda_depth * w * sgn(rd) : 0.f;
    if (l.weight_grad) {
      const float lw = l.lambda_pho * (fabsf(rc0) + fabsf(rc1) + fabsf(rc2)) +
                       (dvalid ? l.lambda_depth * fabsf(rd) : 0.f);
      if (l.weight_mode == 0) {
        if (oo > l.o_eps) { g4 = lw * rm / (oo * oo); g5 = -lw / oo; }
      } else {
        g4 = lw;
        g5 = -lw;
      }
    }
  }
  const int wmax = (int)__reduce_max_sync(FULLM, (unsigned)lastp);

  // Sg = sum over channels of g_ch * S_ch, S_ch the channel's composited sum
  // behind the current Gaussian: dL/dalpha needs only this contraction
  float Sg = 0.f;
  unsigned n_eval = 0, n_contrib = 0;
  const float fpx = (float)px, fpy = (float)py;
  // this lane's entry of group g, and the group's entries to visit: those the
  // forward recorded, or all up to the last contributor
  auto group = [&](int g, uint32_t &id, unsigned &mask) {
    const int k = g * 32 + lane;
    id = 0u;
    if (k < wmax && DAGS_IN_BOUNDS((uint64_t)s + k < (uint64_t)ws.max_pairs, ws.counters + CNT_STATUS)) {
      id = __ldg(ws.sorted_ids + s + k);
      if (!DAGS_IN_BOUNDS(id < (uint32_t)ws.max_n, ws.counters + CNT_STATUS)) id = 0u;
    }
    mask = MASKS && g < kMaskGroups ? __ldg(wmask + g * 8) : FULLM;
    const int lim = wmax - g * 32;
    if (lim < 32) mask &= (1u << lim) - 1u;
  };
  auto stage = [&](int b, uint32_t id, unsigned mask) {
    if ((mask >> lane) & 1u) {
      const float4 *src = recs + (size_t)id * 4;
#pragma unroll
      for (int w = 0; w < 4; ++w) cp_async16(&s_rec[b][w][lane], src + w);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // One entry: advances T and Sg and gives the terms x of its 2D gradient for
  // this lane's pixel; whether any lane takes it (a recorded entry has one: the
  // forward took it for the same pixels by the same arithmetic).
  constexpr int kTerms = !FULL ? 4 : MOMENTS ? 7 : 10;
  auto entry = [&](const float4 (*rec)[32], int j, int k, bool recorded, float (&x)[kTerms], float &dy, uint32_t &id) {
    // evaluated by every lane, without branches: a lane past its last
    // contributor or below alpha_min keeps T and Sg and carries zero
    // gradients, so each contributing lane's values are those of the
    // branching form, operation for operation
    const float4 a = rec[0][j], b = rec[1][j];
    const float dx = (a.x - fpx) + a.z;
    dy = (a.y - fpy) + a.w;
    const float bxdx = b.x * dx, bydx = b.y * dx, bzdy = b.z * dy;
    const float p = fmaf(bxdx, dx, fmaf(bydx, dy, fmaf(bzdy, dy, b.w)));
    const bool contrib = k < lastp && p >= r.log2_alpha_min;
    if (COUNT) { n_eval += k < lastp ? 1u : 0u; n_contrib += contrib ? 1u : 0u; }
    const float ag = hw_exp2(p);
    // zero for a lane that does not take the entry: the weight and the suffix
    // update vanish without a select
    const float alpha = contrib ? fminf(r.alpha_max, ag) : 0.f;
    const float inv = hw_rcp(1.f - alpha);
    // transmittance in front of this Gaussian; kept, whatever the approximate
    // reciprocal makes of 1, by a lane that does not take it
    if (contrib) T *= inv;
    const float wk = alpha * T;
    const float4 c = rec[2][j], d = rec[3][j];
    // dL/dalpha = sum_ch g_ch (c_ch T - S_ch / (1 - alpha))
    const float gcv = fmaf(g0, c.z, fmaf(g1, c.w, fmaf(g2, d.x, fmaf(g3, c.x, fmaf(g5, c.y, g4)))));
    const float dal = fmaf(gcv, T, -Sg * inv);
    // below the clamp, d alpha / d(natural exponent) = alpha (at the clamp
    // alpha does not move with the exponent)
    const float dpw = contrib && ag <= r.alpha_max ? dal * alpha : 0.f;
    const float gz = g3 * wk;
    Sg = fmaf(gcv, wk, Sg);
    id = __float_as_uint(d.w);
    if constexpr (MOMENTS) {
      const float e = fmaf(d.y, dy, dx), te = dpw * e;
      x[0] = te; x[1] = te * e; x[2] = gz; x[kTerms - 1] = dpw;
      if constexpr (FULL) { x[3] = g0 * wk; x[4] = g1 * wk; x[5] = g2 * wk; }
    } else {
      // the exponent in log2 units is p, so d/dx of the natural exponent is
      // ln2 dp/dx: d p / d(u, v) = (2 a' dx + b' dy, b' dx + 2 c' dy) from the
      // exponent's products; d(natural exponent) / d(conic) = -(dx^2 / 2,
      // dx dy, dy^2 / 2)
      const float hl = dpw * kLn2, tx = dpw * dx, ty = dpw * dy;
      x[0] = hl * fmaf(2.f, bxdx, b.y * dy); x[1] = hl * fmaf(2.f, bzdy, bydx); x[2] = -0.5f * (tx * dx);
      x[3] = -(tx * dy); x[4] = -0.5f * (ty * dy); x[5] = gz; x[6] = dpw; x[7] = g0 * wk; x[8] = g1 * wk;
      x[9] = g2 * wk;
    }
    return recorded || __any_sync(FULLM, contrib);
  };
  // the warp sum of this lane's word
  auto sums = [&](const float (&x)[kTerms], float dy) {
    if constexpr (MOMENTS) return moment_sums<kTerms>(x, dy, lane);
    else return warp_reduce_scatter<kTerms, 16>(x, lane);
  };
  // groups from the last contributor's down; the ids of the group after next
  // and the records of the next are in flight while a group is worked on
  int g = wmax > 0 ? (wmax - 1) >> 5 : -1, cur = 0;
  uint32_t id_next = 0u;
  unsigned mask_cur = 0u, mask_next = 0u;
  if (g >= 0) {
    uint32_t id;
    group(g, id, mask_cur);
    if (g > 0) group(g - 1, id_next, mask_next);
    stage(0, id, mask_cur);
  }
  for (; g >= 0; --g, cur ^= 1) {
    stage(cur ^ 1, id_next, mask_next);      // (nothing when g is 0)
    unsigned mask = mask_cur;
    mask_cur = mask_next;
    mask_next = 0u;
    if (g > 1) group(g - 2, id_next, mask_next);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    // the lane's own entry: whether its box meets the block, and the conic's
    // shear in place of the box's half width
    const float4(*const rec)[32] = s_rec[cur];
    const bool recorded = MASKS && g < kMaskGroups;
    bool hit = false;
    if ((mask >> lane) & 1u) {
      const float4 a = rec[0][lane], b = rec[1][lane], d = rec[3][lane];
      hit = fabsf(a.x - bcx) <= d.y + 3.5f && fabsf(a.y - bcy) <= d.z + 1.5f;
      if (MOMENTS) s_rec[cur][3][lane].y = conic_shear(b.x, b.y);
    }
    // without a record (later groups, or none): the entries that passed
    if (!recorded) mask = __ballot_sync(FULLM, hit);
    __syncwarp();
    // two entries at a time: the second's arithmetic and reduction fill the
    // latencies of the first's
    while (mask) {
      float x0[kTerms], x1[kTerms], dy0, dy1;
      uint32_t id0, id1;
      const int j0 = 31 - __clz((int)mask);
      mask &= ~(1u << j0);
      const bool any0 = entry(rec, j0, g * 32 + j0, recorded, x0, dy0, id0);
      if (mask) {
        const int j1 = 31 - __clz((int)mask);
        mask &= ~(1u << j1);
        const bool any1 = entry(rec, j1, g * 32 + j1, recorded, x1, dy1, id1);
        const float s0 = sums(x0, dy0), s1 = sums(x1, dy1);
        if (any0 && writer) atomicAdd(gdst + (size_t)id0 * kGradWords, s0);
        if (any1 && writer) atomicAdd(gdst + (size_t)id1 * kGradWords, s1);
      } else if (any0) {
        const float s0 = sums(x0, dy0);
        if (writer) atomicAdd(gdst + (size_t)id0 * kGradWords, s0);
      }
    }
    __syncwarp();   // the group's buffer is staged again in the next round
  }
  if (COUNT) add_eval_counts(ws, 1, n_eval, n_contrib);
  // the fixed-bucket layout's counts start at zero for the next preprocess
  // (the adjoint is the last reader of the tile's range)
  if (ws.bucket_cap && warp == 0 && lane == 0) ws.tile_count[tile] = 0u;
}

// A projection with what the chain makes of its conic. The exponent is
// -(d^T Q d) / 2 over the offset d = (dx, dy) with the conic Q = [[a, b], [b, c]],
// and Q d = (a e + h dy, b e + s dy) with e = dx + k dy: k is b / a up to its
// rounding, so h = b - a k is that rounding's remainder and s = c - b k is 1 / C,
// the inverse of a covariance entry. Neither is formed as a difference of conic
// entries, which cancels as the square of the splat's aspect ratio.
struct ChainProj : Proj {
  float h, s;
};
__device__ __forceinline__ void chain_factors(ChainProj &q) {
  const float k = conic_shear(__fmul_rn(-0.5f * kLog2e, q.ca), __fmul_rn(-kLog2e, q.cb));
  const float rem = fmaf(-k, q.C, -q.B);
  q.h = rem * __fdiv_rn(1.f, q.det);
  q.s = fmaf(q.cb, rem, 1.f) / q.C;
}

// Chains the 2D gradients of the Gaussian projected as q in view slot `slot`
// (pose Pm) to the pose twist (pg, added) and, FULL, to the record's
// parameters (acc, added).
template <bool FULL, bool MOMENTS>
__device__ __forceinline__ void chain_proj(const Workspace &ws, const Raster &r, const ChainProj &q, const float *Pm,
                                           size_t slot, float *pg, float *acc) {
  const float *gd = ws.grad2d + slot * kGradWords;
  const float4 ga4 = *reinterpret_cast<const float4 *>(gd);
  const float4 gb4 = *reinterpret_cast<const float4 *>(gd + 4);
  const float gzz = gb4.y;
  float gu, gv, d00, d01, d11;   // gradients of the centre and of the 2D covariance
  if constexpr (MOMENTS) {
    // d/d(u, v) = -sum g Q d
    gu = -fmaf(q.ca, ga4.x, q.h * ga4.y);
    gv = -fmaf(q.cb, ga4.x, q.s * ga4.y);
    // dS = sum g (Q d)(Q d)^T / 2: the sums of g (Q d)_u (e, dy) and of g (Q d)_v (e, dy)
    const float t0e = q.ca * ga4.z + q.h * ga4.w, t0y = q.ca * ga4.w + q.h * gb4.x;
    const float t1e = q.cb * ga4.z + q.s * ga4.w, t1y = q.cb * ga4.w + q.s * gb4.x;
    d00 = 0.5f * (t0e * q.ca + t0y * q.h);
    d01 = 0.5f * (t0e * q.cb + t0y * q.s);
    d11 = 0.5f * (t1e * q.cb + t1y * q.s);
  } else {
    gu = ga4.x;
    gv = ga4.y;
    // conic -> 2D covariance: dS = -Q Gq Q with Gq the symmetric-matrix form of
    // the conic gradient (the off-diagonal appears twice in the quadratic form)
    const float gA = ga4.z, gB = ga4.w, gC = gb4.x;
    const float qa = q.ca, qb = q.cb, qc = q.cc;
    const float h = 0.5f * gB;
    const float t00 = qa * gA + qb * h, t01 = qa * h + qb * gC;
    const float t10 = qb * gA + qc * h, t11 = qb * h + qc * gC;
    d00 = -(t00 * qa + t01 * qb);
    d01 = -(t00 * qb + t01 * qc);
    d11 = -(t10 * qb + t11 * qc);
  }
  // Sigma' = M2 M2^T + d I with M2 = J K: dM2 = 2 dS M2
  float dm0[3], dm1[3];
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    dm0[s] = 2.f * (d00 * q.m0[s] + d01 * q.m1[s]);
    dm1[s] = 2.f * (d01 * q.m0[s] + d11 * q.m1[s]);
  }
  const float dj00 = dm0[0] * q.K[0] + dm0[1] * q.K[1] + dm0[2] * q.K[2];
  const float dj02 = dm0[0] * q.K[6] + dm0[1] * q.K[7] + dm0[2] * q.K[8];
  const float dj11 = dm1[0] * q.K[3] + dm1[1] * q.K[4] + dm1[2] * q.K[5];
  const float dj12 = dm1[0] * q.K[6] + dm1[1] * q.K[7] + dm1[2] * q.K[8];
  float dK[9];
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    dK[s] = q.j00 * dm0[s];
    dK[3 + s] = q.j11 * dm1[s];
    dK[6 + s] = q.j02 * dm0[s] + q.j12 * dm1[s];
  }
  // camera-space mean
  const float z = q.z, iz = 1.f / z, iz2 = iz * iz;
  float dpx = gu * r.fx * iz;
  float dpy = gv * r.fy * iz;
  float dpz = -gu * r.fx * q.x * iz2 - gv * r.fy * q.y * iz2 + gzz;
  dpz += -dj00 * r.fx * iz2 - dj11 * r.fy * iz2;
  const bool clx = q.txz > r.limx || q.txz < -r.limx;
  const bool cly = q.tyz > r.limy || q.tyz < -r.limy;
  if (!clx) { dpx += -dj02 * r.fx * iz2; dpz += dj02 * 2.f * r.fx * q.x * iz2 * iz; }
  else { dpz += dj02 * r.fx * q.tx * iz2; }
  if (!cly) { dpy += -dj12 * r.fy * iz2; dpz += dj12 * 2.f * r.fy * q.y * iz2 * iz; }
  else { dpz += dj12 * r.fy * q.ty * iz2; }
  // pose twist (left perturbation): rho += dp, phi += p x dp + the covariance
  // term from K' = (I + [phi]x) K: B = K dK^T
  pg[0] += dpx; pg[1] += dpy; pg[2] += dpz;
  pg[3] += q.y * dpz - z * dpy;
  pg[4] += z * dpx - q.x * dpz;
  pg[5] += q.x * dpy - q.y * dpx;
  float Bm[9];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
      Bm[3 * a + b] = q.K[3 * a] * dK[3 * b] + q.K[3 * a + 1] * dK[3 * b + 1] + q.K[3 * a + 2] * dK[3 * b + 2];
  pg[3] += Bm[5] - Bm[7];
  pg[4] += Bm[6] - Bm[2];
  pg[5] += Bm[1] - Bm[3];
  if (FULL) {
    const float4 gc4 = *reinterpret_cast<const float4 *>(gd + 8);
    const float s0 = gb4.z;   // o dL/do: alpha is proportional to the opacity
    acc[0] += Pm[0] * dpx + Pm[4] * dpy + Pm[8] * dpz;
    acc[1] += Pm[1] * dpx + Pm[5] * dpy + Pm[9] * dpz;
    acc[2] += Pm[2] * dpx + Pm[6] * dpy + Pm[10] * dpz;
    acc[3] += s0 * (1.f - q.o);
    // K = R M, M = Rq diag(S): dM = R^T dK
    float dRq[9];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      float dS = 0.f;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float dM = Pm[a] * dK[s] + Pm[4 + a] * dK[3 + s] + Pm[8 + a] * dK[6 + s];
        dS += q.Rq[3 * a + s] * dM;
        dRq[3 * a + s] = dM * q.S[s];
      }
      acc[8 + s] += dS * q.S[s];
    }
    const float w = q.nq[0], x = q.nq[1], y = q.nq[2], zq = q.nq[3];
    const float dn0 = -2.f * zq * dRq[1] + 2.f * y * dRq[2] + 2.f * zq * dRq[3] - 2.f * x * dRq[5] -
                      2.f * y * dRq[6] + 2.f * x * dRq[7];
    const float dn1 = 2.f * y * dRq[1] + 2.f * zq * dRq[2] + 2.f * y * dRq[3] - 4.f * x * dRq[4] -
                      2.f * w * dRq[5] + 2.f * zq * dRq[6] + 2.f * w * dRq[7] - 4.f * x * dRq[8];
    const float dn2 = -4.f * y * dRq[0] + 2.f * x * dRq[1] + 2.f * w * dRq[2] + 2.f * x * dRq[3] +
                      2.f * zq * dRq[5] - 2.f * w * dRq[6] + 2.f * zq * dRq[7] - 4.f * y * dRq[8];
    const float dn3 = -4.f * zq * dRq[0] - 2.f * w * dRq[1] + 2.f * x * dRq[2] + 2.f * w * dRq[3] -
                      4.f * zq * dRq[4] + 2.f * y * dRq[5] + 2.f * x * dRq[6] + 2.f * y * dRq[7];
    const float ndn = w * dn0 + x * dn1 + y * dn2 + zq * dn3;
    const float iq = 1.f / q.qlen;
    acc[4] += (dn0 - w * ndn) * iq;
    acc[5] += (dn1 - x * ndn) * iq;
    acc[6] += (dn2 - y * ndn) * iq;
    acc[7] += (dn3 - zq * ndn) * iq;
    acc[12] += gb4.w;   // colour: slots G2_R, G2_G, G2_BL
    acc[13] += gc4.x;
    acc[14] += gc4.y;
  }
}

// Whether the Gaussian of view slot `slot` has a non-empty tile range, and if
// so its projection.
template <bool MOMENTS>
__device__ __forceinline__ bool visible_proj(const Workspace &ws, const Raster &r, const float4 &g0,
                                             const float4 &g1, const float4 &g2, const float *Pm, size_t slot,
                                             ChainProj &q) {
  const uint2 rc = ws.rect[slot];
  if ((rc.x >> 16) <= (rc.x & 0xFFFF) || !project_gaussian(g0, g1, g2, Pm, r, q)) return false;
  if (MOMENTS) chain_factors(q);
  return true;
}

// chain_proj of Gaussian (g0, g1, g2) when it is visible.
template <bool FULL, bool MOMENTS>
__device__ __forceinline__ void chain_one(const Workspace &ws, const Raster &r, const float4 &g0, const float4 &g1,
                                          const float4 &g2, const float *Pm, size_t slot, float *pg, float *acc) {
  ChainProj q;
  if (visible_proj<MOMENTS>(ws, r, g0, g1, g2, Pm, slot, q)) chain_proj<FULL, MOMENTS>(ws, r, q, Pm, slot, pg, acc);
}

// Compensated (double-FP32) addition: (h, l) += (bh, bl) through two-sum,
// the high words' rounding error carried into the low word.
__device__ __forceinline__ void cadd(float &h, float &l, float bh, float bl) {
  float sh, se;
  two_sum(h, bh, sh, se);
  h = sh;
  l = __fadd_rn(__fadd_rn(l, bl), se);
}

// Sums pg[6] over the CTA in compensated FP32 (a fixed shuffle tree, then
// the warps in order) and stores the (high, low) partial of (view v, CTA b).
__device__ __forceinline__ void store_pose_partial(const Workspace &ws, float *pg, int v, int b, int nb,
                                                   float2 (*s_red)[6]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    float h = pg[c], l = 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      cadd(h, l, __shfl_xor_sync(0xffffffffu, h, o), __shfl_xor_sync(0xffffffffu, l, o));
    if (lane == 0) s_red[wid][c] = make_float2(h, l);
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    float h = 0.f, l = 0.f;
    for (int w = 0; w < kBwdPrepBlock / 32; ++w) cadd(h, l, s_red[w][threadIdx.x].x, s_red[w][threadIdx.x].y);
    ws.pose_partial[((size_t)v * nb + b) * 6 + threadIdx.x] = make_float2(h, l);
  }
  __syncthreads();
}

// FULL: one thread per Gaussian, all views, parameter gradients written.
// !FULL (pose only): a fixed grid strides over the Gaussians of each view.
// The last CTA sums the pose partials in a fixed order in FP64 (one warp per
// twist component) and, if ps.poses is set, applies the pose step.
// The pose-only form keeps to 96 registers, five CTAs per SM: its grid of four
// per SM and the ranking CTA are then one wave (at 104 registers and four CTAs
// per SM the ranking CTA pushes one out, and an iteration of the tracking loop
// takes 3 us more).
template <bool FULL, bool MOMENTS>
__global__ void __launch_bounds__(kBwdPrepBlock, FULL ? 1 : 5)
preprocess_bwd_kernel(Workspace ws, const float4 *__restrict__ gauss, int64_t n, int views, Raster r,
                      float *__restrict__ grad_gauss, double *__restrict__ grad_pose, PoseStep ps) {
  // pose only, tracking loop: the grid's first CTA (dispatched first, so
  // that it runs beside the chain CTAs from the start) ranks the tiles by
  // this iteration's counts for the next iteration's render order; the
  // chain CTAs are numbered from the second
  const bool ordering = !FULL && ws.order_next != nullptr;
  if (ordering && blockIdx.x == 0) {
    pdl_wait();
    pdl_trigger();
    rank_tiles(ws.prev_count, r.T, ws.order_next, ws.band);
    return;
  }
  __shared__ float sp[kMaxViewsSmem * 12];
  __shared__ float2 s_red[kBwdPrepBlock / 32][6];
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nb = gridDim.x - (ordering ? 1 : 0);
  const int bid = blockIdx.x - (ordering ? 1 : 0);
  // pose only, one view: the visible list, the records, their tile ranges
  // and the FP32 pose were written two or more launches before this one, so
  // each thread projects its first visible Gaussian before waiting for the
  // adjoint, whose 2D gradients it reads after the wait
  ChainProj q0;
  bool pre = false, pre_vis = false;
  // the pose step's bias corrections depend only on the Adam step count,
  // written by the previous iteration's step (three launches back): every
  // CTA forms them before its wait, and the last one uses its own
  __shared__ double s_presc[2];
  const bool presc = !FULL && views == 1 && ps.poses != nullptr;
  if (presc && (tid == 6 || tid == 7)) {
    const double k = __ldcg(ps.state + 12) + 1.0;
    s_presc[tid - 6] = tid == 6 ? adam_bias1(ps.cfg, k) : adam_bias2(ps.cfg, k);
  }
  int64_t pre_k = 0;
  size_t pre_slot = 0;
  if (!FULL && views == 1) {
    for (int k = tid; k < 12; k += blockDim.x) sp[k] = __ldcg(ws.pose32 + k);
    __syncthreads();
    pre = true;
    pre_k = (int64_t)bid * blockDim.x + tid;
    if (pre_k < (int64_t)__ldcg(ws.vis_n)) {
      const int64_t i = __ldcg(ws.vis_ids + pre_k);
      if (DAGS_IN_BOUNDS(i >= 0 && i < n, ws.counters + CNT_STATUS)) {
        pre_slot = (size_t)i;
        const float4 g0 = __ldg(gauss + 4 * i + 0), g1 = __ldg(gauss + 4 * i + 1), g2 = __ldg(gauss + 4 * i + 2);
        pre_vis = visible_proj<MOMENTS>(ws, r, g0, g1, g2, sp, pre_slot, q0);
      }
    }
  }
  pdl_wait();
  pdl_trigger();
  if (!pre) {
    for (int k = threadIdx.x; k < views * 12; k += blockDim.x) sp[k] = ws.pose32[k];
    __syncthreads();
  }
  if (FULL) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float4 g0 = make_float4(0.f, 0.f, 0.f, 0.f), g1 = g0, g2 = g0;
    if (i < n) {
      g0 = __ldg(gauss + 4 * i + 0);
      g1 = __ldg(gauss + 4 * i + 1);
      g2 = __ldg(gauss + 4 * i + 2);
    }
    float acc[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = 0.f;
    for (int v = 0; v < views; ++v) {
      float pg[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (i < n) chain_one<true, MOMENTS>(ws, r, g0, g1, g2, sp + v * 12, (size_t)v * ws.max_n + i, pg, acc);
      if (grad_pose) store_pose_partial(ws, pg, v, blockIdx.x, nb, s_red);
    }
    if (i < n) {
      float4 *out = reinterpret_cast<float4 *>(grad_gauss + 16 * i);
      out[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      out[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
      out[2] = make_float4(acc[8], acc[9], acc[10], 0.f);
      out[3] = make_float4(acc[12], acc[13], acc[14], 0.f);
    }
  } else {
    // pose only: the visible Gaussians of each view (the others have no
    // 2D gradient)
    for (int v = 0; v < views; ++v) {
      float pg[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      const int64_t nv = ws.vis_n[v];
      const uint32_t *vis = ws.vis_ids + (size_t)v * ws.max_n;
      for (int64_t k = (int64_t)bid * blockDim.x + tid; k < nv; k += (int64_t)nb * blockDim.x) {
        if (pre && k == pre_k) {
          if (pre_vis) chain_proj<false, MOMENTS>(ws, r, q0, sp, pre_slot, pg, nullptr);
          continue;
        }
        int64_t i = vis[k];
        if (!DAGS_IN_BOUNDS(i >= 0 && i < n, ws.counters + CNT_STATUS)) continue;
        const float4 g0 = __ldg(gauss + 4 * i + 0), g1 = __ldg(gauss + 4 * i + 1), g2 = __ldg(gauss + 4 * i + 2);
        chain_one<false, MOMENTS>(ws, r, g0, g1, g2, sp + v * 12, (size_t)v * ws.max_n + i, pg, nullptr);
      }
      store_pose_partial(ws, pg, v, bid, nb, s_red);
    }
  }
  if (!grad_pose) return;
  // last CTA: barrier, then one thread's fence and counter increment
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    const unsigned t = atomicAdd(ws.counters + CNT_DONE_BWDPREP, 1u);
    s_last = (t == (unsigned)nb - 1u);
    if (s_last) __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  // the CTA partials of each view, summed by every thread of the last CTA:
  // thread t takes CTAs t, t + 128, ... (all loads of a round issued before
  // they are added), each component in compensated FP32 in a fixed order,
  // then a fixed shuffle tree and the warps in order; the result is the
  // FP64 sum of the high and low words
  for (int v = 0; v < views; ++v) {
    const float2 *src = ws.pose_partial + (size_t)v * nb * 6;
    float h[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, l[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int b0 = tid; b0 < nb; b0 += kBwdPrepBlock * 4) {
      float2 t[4][6];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int b = b0 + kBwdPrepBlock * u;
#pragma unroll
        for (int c = 0; c < 6; ++c) t[u][c] = b < nb ? __ldcg(src + (size_t)b * 6 + c) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int c = 0; c < 6; ++c) cadd(h[c], l[c], t[u][c].x, t[u][c].y);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        cadd(h[c], l[c], __shfl_xor_sync(0xffffffffu, h[c], o), __shfl_xor_sync(0xffffffffu, l[c], o));
      if (lane == 0) s_red[wid][c] = make_float2(h[c], l[c]);
    }
    __syncthreads();
    if (tid < 6) {
      float hh = 0.f, ll = 0.f;
      for (int w = 0; w < kBwdPrepBlock / 32; ++w) cadd(hh, ll, s_red[w][tid].x, s_red[w][tid].y);
      grad_pose[v * 6 + tid] = (double)hh + (double)ll;
    }
    __syncthreads();
  }
  if (tid == 0) ws.counters[CNT_DONE_BWDPREP] = 0u;
  if (ps.poses) {
    __shared__ double s_xi[6], s_sc[3];
    for (int v = 0; v < views; ++v)
      pose_adam_exp_cta(ps.poses + 12 * v, grad_pose + 6 * v, ps.state + 13 * v, ps.cfg, s_xi, s_sc,
                        presc ? s_presc : nullptr);
    // the tracking loop: if the new pose (as the preprocess stages it in
    // FP32) has left the bounds the candidates were culled for, move the
    // culling pose to it and empty the list; the next preprocess then takes
    // every Gaussian once and re-culls
    if (ordering && ws.cand_n && ws.cull_pose) {
      __shared__ float s_np[12];
      __shared__ int s_out;
      __syncthreads();
      if (tid < 12) s_np[tid] = __double2float_rn(ps.poses[tid]);
      __syncthreads();
      if (tid == 0) s_out = within_cull_bounds(s_np, ws.cull_pose) ? 0 : 1;
      __syncthreads();
      if (s_out && tid < 12) ws.cull_pose[tid] = s_np[tid];
      if (tid == 0) {
        if (s_out) *ws.cand_n = 0u;
        ws.counters[CNT_RECULL] = s_out ? 1u : 0u;
      }
    }
  }
}

}  // namespace

// Whether the 2D gradients are accumulated as moments: not where the Gaussian
// and the twist gradients are both asked for. Moments are the faster form (the
// adjoint of one frame, 300k Gaussians, 640x480, all gradients over recorded
// entries: 59 against 66 us) and no less exact: against 64 bits the twist of
// 2,000 Gaussians is 2.5e-7 off from moments and 2.9e-7 from words per pixel
// (means of six scenes), that of discs seen edge-on with a standard deviation
// of 2 to 110 px 1e-6 .. 1e-5 and 1e-6 .. 7e-4. But the two differ by what
// either is off, 3e-7 there and 4e-8 on the 300k frame, three times what the
// order of the atomics does, and a caller of both takes the twist as FP64:
// those results stay as they were.
static bool backward_moments(bool full, bool pose) { return !(full && pose); }

cudaError_t launch_render_bwd(const Workspace &ws, int views, int64_t n, const Raster &r, const Loss &l,
                              const float4 *targets, const float *image, const int32_t *last, bool full, bool pose,
                              cudaStream_t s, const float *upstream) {
  (void)n;
  const dim3 grid((unsigned)(views * r.T) * kBlocks);
  const bool masks = ws.warp_masks != nullptr, count = ws.count_evals != 0;
#define DAGS_BWD(F, M, K, C) \
  launch_pdl(render_bwd_kernel<F, M, K, C>, grid, dim3(32), 0, s, ws, r, l, targets, image, last, upstream)
#define DAGS_BWD_KC(F, M) \
  (masks ? (count ? DAGS_BWD(F, M, true, true) : DAGS_BWD(F, M, true, false)) \
         : (count ? DAGS_BWD(F, M, false, true) : DAGS_BWD(F, M, false, false)))
  if (full) return backward_moments(full, pose) ? DAGS_BWD_KC(true, true) : DAGS_BWD_KC(true, false);
  return DAGS_BWD_KC(false, true);
#undef DAGS_BWD_KC
#undef DAGS_BWD
}

cudaError_t launch_preprocess_bwd(const Workspace &ws, const float4 *gauss, int64_t n, int views,
                                  const Raster &r, float *grad_gauss, double *grad_pose, const PoseStep &ps,
                                  cudaStream_t s) {
  if (views > kMaxViewsSmem) return cudaErrorInvalidValue;
  const unsigned gx = (unsigned)((n + kBwdPrepBlock - 1) / kBwdPrepBlock);
  unsigned grid = gx > 0 ? gx : 1u;
  if (grad_gauss) {
    if (backward_moments(true, grad_pose != nullptr))
      return launch_pdl(preprocess_bwd_kernel<true, true>, dim3(grid), dim3(kBwdPrepBlock), 0, s, ws, gauss, n, views,
                        r, grad_gauss, grad_pose, ps);
    return launch_pdl(preprocess_bwd_kernel<true, false>, dim3(grid), dim3(kBwdPrepBlock), 0, s, ws, gauss, n, views,
                      r, grad_gauss, grad_pose, ps);
  } else {
    // pose only: a fixed grid of 4 CTAs per SM (one wave) strides over the
    // visible Gaussians (at most one per thread at the tracking size); the
    // tracking loop adds one CTA that ranks the tiles for the next
    // iteration's render order
    const unsigned cap = (unsigned)(4 * (ws.band > 0 ? ws.band : 1));
    if (grid > cap) grid = cap;
    if (ws.order_next) grid += 1;
    return launch_pdl(preprocess_bwd_kernel<false, true>, dim3(grid), dim3(kBwdPrepBlock), 0, s, ws, gauss, n, views, r,
                      grad_gauss, grad_pose, ps);
  }
  return cudaGetLastError();
}

}  // namespace dags
