// Epipolar verification and static recovery (Sec. IV-C, Eqs. (18), (19)) on
// sm_103a:
//
//   epi_dist_kernel     F = K^-T [t]x R K^-1 from the two poses, FP64, per CTA;
//                       per match: the point-to-epipolar-line distance d of
//                       Eq. (18) in FP64, and the match's
//                       rank inside its Gaussian's group (one atomic per
//                       match on the Gaussian's count)
//   epi_offsets_kernel  group offsets: a scan of 1024 counts per CTA, placed
//                       behind one another by an atomic cursor (the groups'
//                       order does not matter)
//   epi_scatter_kernel  d into its group's slot (offset + rank)
//   epi_median_kernel   per Gaussian with matches: the lower median of its
//                       group by rank counting (the groups hold a few values;
//                       the result does not depend on the order the atomics
//                       gave), the consistency test dbar < eps of Eq. (19),
//                       and the recovery of a dynamic-labelled consistent
//                       Gaussian: label 0, M <- min(M, m_static)
//
// Gaussian ids come from the caller: an id >= n is skipped and recorded as
// an index error in the status word (DAGS_E_BOUNDS at the next sync).
#include "common.cuh"

namespace dags {

namespace {

constexpr int kEpiBlock = 256;
constexpr int kScanItems = 4;                  // counts per thread in the block scan
constexpr int kScanTile = kEpiBlock * kScanItems;

// F = K^-T [t]x R K^-1 of the relative pose (R, t) = T_2W T_1W^-1, in FP64 by
// the first nine threads of a CTA (FP64 instructions are scarce on GB300, but
// a launch of its own costs more than every CTA's few dozen).
__device__ __forceinline__ void epi_F(const Raster &r, const double *__restrict__ pose_1,
                                      const double *__restrict__ pose_2, double *F) {
  __shared__ double s_R[9], s_EK[9], s_t[3];
  const int k = threadIdx.x, a = k / 3, b = k % 3;
  // R = R2 R1^T, t = t2 - R t1, E = [t]x R, F = K^-T E K^-1
  if (k < 9)
    s_R[k] = pose_2[4 * a] * pose_1[4 * b] + pose_2[4 * a + 1] * pose_1[4 * b + 1] +
             pose_2[4 * a + 2] * pose_1[4 * b + 2];
  __syncthreads();
  if (k < 3)
    s_t[k] = pose_2[4 * k + 3] - (s_R[3 * k] * pose_1[3] + s_R[3 * k + 1] * pose_1[7] + s_R[3 * k + 2] * pose_1[11]);
  __syncthreads();
  // K^-1 = [[1/fx, 0, -cx/fx], [0, 1/fy, -cy/fy], [0, 0, 1]]
  const double ifx = 1.0 / (double)r.fx, ify = 1.0 / (double)r.fy;
  const double kx = -(double)r.cx * ifx, ky = -(double)r.cy * ify;
  if (k < 3) {   // row k of E K^-1
    const double tx[9] = {0.0, -s_t[2], s_t[1], s_t[2], 0.0, -s_t[0], -s_t[1], s_t[0], 0.0};
    double E[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double t0 = k == 0 ? tx[0] : k == 1 ? tx[3] : tx[6], t1 = k == 0 ? tx[1] : k == 1 ? tx[4] : tx[7],
                   t2 = k == 0 ? tx[2] : k == 1 ? tx[5] : tx[8];
      E[j] = t0 * s_R[j] + t1 * s_R[3 + j] + t2 * s_R[6 + j];
    }
    s_EK[3 * k + 0] = E[0] * ifx;
    s_EK[3 * k + 1] = E[1] * ify;
    s_EK[3 * k + 2] = E[0] * kx + E[1] * ky + E[2];
  }
  __syncthreads();
  // K^-T (E K^-1): rows 0, 1 scale, row 2 combines
  if (k < 3) F[k] = s_EK[k] * ifx;
  else if (k < 6) F[k] = s_EK[k] * ify;
  else if (k < 9) F[k] = s_EK[b] * kx + s_EK[3 + b] * ky + s_EK[6 + b];
}

__global__ void __launch_bounds__(kEpiBlock)
epi_dist_kernel(Raster r, const double *__restrict__ pose_1, const double *__restrict__ pose_2,
                const float2 *__restrict__ p1, const float2 *__restrict__ p2, const int32_t *__restrict__ gid,
                int64_t m, int64_t n, float *__restrict__ dist, uint32_t *__restrict__ count,
                uint32_t *__restrict__ rank, uint32_t *__restrict__ cursor, uint32_t *status) {
  pdl_wait();
  __shared__ double s_F[9];
  if (blockIdx.x == 0 && threadIdx.x == 0) *cursor = 0u;
  epi_F(r, pose_1, pose_2, s_F);
  __syncthreads();
  const int64_t k = (int64_t)blockIdx.x * kEpiBlock + threadIdx.x;
  if (k >= m) return;
  const float2 a1 = p1[k], a2 = p2[k];
  const double u1 = a1.x, v1 = a1.y, u2 = a2.x, v2 = a2.y;
  const double la = s_F[0] * u1 + s_F[1] * v1 + s_F[2];
  const double lb = s_F[3] * u1 + s_F[4] * v1 + s_F[5];
  const double lc = s_F[6] * u1 + s_F[7] * v1 + s_F[8];
  const double num = fabs(u2 * la + v2 * lb + lc);
  const double den = sqrt(la * la + lb * lb);
  dist[k] = den > 0.0 ? (float)(num / den) : 0.f;
  const int32_t g = gid[k];
  if (g < 0 || (int64_t)g >= n) {
    atomicOr(status, kStatusBounds);
    rank[k] = 0xFFFFFFFFu;
    return;
  }
  rank[k] = atomicAdd(count + g, 1u);
}

// The first slot of every group: per CTA an exclusive scan of 1024 counts (four
// per thread, a warp scan of the thread sums, the eight warp sums), offset by
// the CTA's share of a global cursor. Three launches (tile scans, their sums,
// the addition) gave the groups in order, which nothing needs.
__global__ void __launch_bounds__(kEpiBlock)
epi_offsets_kernel(const uint32_t *__restrict__ count, int64_t n, uint32_t *__restrict__ off,
                   uint32_t *__restrict__ cursor) {
  pdl_wait();
  __shared__ uint32_t s_warp[kEpiBlock / 32], s_base;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)tid * kScanItems;
  uint32_t v[kScanItems], acc = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    v[j] = base + j < n ? count[base + j] : 0u;
    acc += v[j];
  }
  uint32_t inc = acc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t add = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += add;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  uint32_t run = inc - acc;
#pragma unroll
  for (int w = 0; w < kEpiBlock / 32; ++w) run += w < warp ? s_warp[w] : 0u;
  if (tid == kEpiBlock - 1) s_base = run + acc ? atomicAdd(cursor, run + acc) : 0u;
  __syncthreads();
  run += s_base;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    if (v[j]) off[base + j] = run;
    run += v[j];
  }
}

__global__ void __launch_bounds__(kEpiBlock)
epi_scatter_kernel(const int32_t *__restrict__ gid, const uint32_t *__restrict__ rank, const float *__restrict__ dist,
                   int64_t m, const uint32_t *__restrict__ off, float *__restrict__ vals) {
  pdl_wait();
  const int64_t k = (int64_t)blockIdx.x * kEpiBlock + threadIdx.x;
  if (k >= m) return;
  const uint32_t rk = rank[k];
  if (rk == 0xFFFFFFFFu) return;
  vals[off[gid[k]] + rk] = dist[k];
}

__global__ void __launch_bounds__(kEpiBlock)
epi_median_kernel(const uint32_t *__restrict__ count, const uint32_t *__restrict__ off,
                  const float *__restrict__ vals, int64_t n, float eps, float m_static, float4 *__restrict__ gauss,
                  uint8_t *__restrict__ labels, float *__restrict__ dbar) {
  pdl_wait();
  const int64_t g = (int64_t)blockIdx.x * kEpiBlock + threadIdx.x;
  if (g >= n) return;
  const uint32_t c = count[g];
  if (c == 0) {
    if (dbar) dbar[g] = __int_as_float(0x7fc00000);
    return;
  }
  const float *v = vals + off[g];
  const uint32_t want = (c - 1) / 2;
  float med = v[0];
  for (uint32_t i = 0; i < c; ++i) {
    // rank of v[i] in the ascending order (ties broken by position)
    const float x = v[i];
    uint32_t rk = 0;
    for (uint32_t j = 0; j < c; ++j) {
      const float y = v[j];
      rk += (y < x || (y == x && j < i)) ? 1u : 0u;
    }
    if (rk == want) { med = x; break; }
  }
  if (dbar) dbar[g] = med;
  if (med < eps && labels[g] == 1) {
    labels[g] = 0;
    float4 w = gauss[4 * g + 2];
    w.w = fminf(w.w, m_static);
    gauss[4 * g + 2] = w;
  }
}

}  // namespace

cudaError_t launch_epipolar(const Raster &r, const double *pose_1, const double *pose_2, const float2 *p1,
                            const float2 *p2, const int32_t *gid, int64_t m, float4 *gauss, int64_t n,
                            uint8_t *labels, float eps, float m_static, float *dist, float *dbar, const EpiBuffers &b,
                            uint32_t *status, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(b.count, 0, (size_t)(n > 0 ? n : 1) * sizeof(uint32_t), s);
  if (e != cudaSuccess) return e;
  const unsigned gm = (unsigned)((m + kEpiBlock - 1) / kEpiBlock);
  const unsigned gn = (unsigned)((n + kEpiBlock - 1) / kEpiBlock);
  // programmatic launches after the first: each kernel waits for its
  // predecessor's memory before its first access, and its launch overlaps
  // the predecessor's last wave
  if (m > 0) {
    epi_dist_kernel<<<gm, kEpiBlock, 0, s>>>(r, pose_1, pose_2, p1, p2, gid, m, n, dist, b.count, b.rank, b.cursor,
                                             status);
    if (n > 0)
      e = launch_pdl(epi_offsets_kernel, dim3((unsigned)((n + kScanTile - 1) / kScanTile)), dim3(kEpiBlock), 0, s,
                     (const uint32_t *)b.count, n, b.off, b.cursor);
  }
  if (m > 0 && e == cudaSuccess)
    e = launch_pdl(epi_scatter_kernel, dim3(gm), dim3(kEpiBlock), 0, s, gid, (const uint32_t *)b.rank,
                   (const float *)dist, m, (const uint32_t *)b.off, b.vals);
  if (n > 0 && e == cudaSuccess)
    e = launch_pdl(epi_median_kernel, dim3(gn), dim3(kEpiBlock), 0, s, (const uint32_t *)b.count,
                   (const uint32_t *)b.off, (const float *)b.vals, n, eps, m_static, gauss, labels, dbar);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace dags
