// The conventional pipeline of Fig. 1(a), the comparator that the
// instance-specific projection of Sec. 3.3 replaces: every step moves the
// Gaussians of each dynamic instance k to the world frame by the instance's
// pose (R_k = R(q_k/|q_k|), t_k):
//   mu_w = R_k mu + t_k,   q_w = (q_k/|q_k|) (x) (q/|q|)   (Hamilton product),
// and rotates their SH coefficients so that the world-frame view direction
// gives the colour the object-frame direction gives (band l: c'_l = D_l^T c_l
// with Y_l(R_k^T d) = D_l Y_l(d)); its backward maps the adjoints of the
// world-frame parameters back to the object frame and to the poses.
//
// D_l is the projection of the rotated basis on the basis,
//   (D_l)_ij = integral over the sphere of Y_li(R^T d) Y_lj(d) dd,
// evaluated exactly (the integrand is a polynomial of degree <= 6 on the
// sphere) with Lebedev's 26-point rule of degree 7: the 6 axis directions
// (weight 1/21), the 12 edge midpoints of the cube (weight 4/105) and its 8
// corners (weight 9/280), weights summing to 1, times 4 pi.
//
// Only the rows of dynamic Gaussians are read or written: static Gaussians
// do not move, so the caller copies their rows once. The backward works in
// place on the gradient buffers (the world-frame adjoints of the renderer's
// backward become the object-frame ones) and sums the pose terms per
// instance in the workspace before a warp per instance maps them to the
// pose quaternion and translation.
//
// Both kernels should stream at the HBM rate (440 B per Gaussian forward, 700
// backward at degree 3), so the work beside the copies is kept small. A CTA is
// one warp with a contiguous range of rows, taken 32 at a time and never across
// an instance's end, so a chunk has one pose and one set of D_l in shared
// memory. The next chunk's SH rows are already on their way (cp.async into the
// other buffer) while this one is rotated, a lane per Gaussian. The backward's
// sums over an instance (the 83 entries of dD_l, dR, dt, dp) stay in each
// lane's registers until the warp leaves the instance, and only then cross the
// lanes. At 1M Gaussians in 80 instances, degree 3, both calls with the copy of
// the incoming adjoints took 0.291 ms, against 0.712 ms with two-warp CTAs that
// loaded each chunk before working on it, summed dD over each warp's staged rows
// (a loop of 32 Gaussians per entry) and mapped an instance's sums to its pose
// in one thread.
#include "s3r_math.cuh"

namespace s3r {
namespace {

constexpr int kWorldThreads = 32;            // one warp per CTA: a chunk is 32 Gaussians
constexpr int kRotFloats = 9 + 25 + 49;      // D_1, D_2, D_3 row-major
constexpr int kPoseTerms = 9 + 3 + 4;        // dR, dt, dp
constexpr int kWorldAcc = kPoseTerms + kRotFloats;   // and dD, per instance

// entries of D_1..D_deg
__host__ __device__ constexpr int rot_count(int deg) {
  return deg <= 0 ? 0 : (deg == 1 ? 9 : (deg == 2 ? 34 : 83));
}

__device__ __forceinline__ void lebedev26(int m, float d[3], float& w) {
  const float s2 = 0.70710678118654752f, s3 = 0.57735026918962576f;
  if (m < 6) {
    d[0] = d[1] = d[2] = 0.f;
    d[m >> 1] = (m & 1) ? -1.f : 1.f;
    w = 1.f / 21.f;
  } else if (m < 18) {
    const int e = m - 6, pair = e >> 2;            // axes (0,1), (0,2), (1,2)
    const int a = pair == 2 ? 1 : 0, b = pair == 0 ? 1 : 2;
    d[0] = d[1] = d[2] = 0.f;
    d[a] = (e & 1) ? -s2 : s2;
    d[b] = (e & 2) ? -s2 : s2;
    w = 4.f / 105.f;
  } else {
    const int e = m - 18;
    d[0] = (e & 1) ? -s3 : s3;
    d[1] = (e & 2) ? -s3 : s3;
    d[2] = (e & 4) ? -s3 : s3;
    w = 9.f / 280.f;
  }
}

// first basis function of band l, and the offset of D_l in the packed matrices
__host__ __device__ constexpr int band_start(int l) { return l * l; }
__host__ __device__ constexpr int rot_off(int l) { return l <= 1 ? 0 : (l == 2 ? 9 : 34); }

__device__ __forceinline__ int segment_of_gid(const int64_t* __restrict__ off, int n_inst, int64_t g) {
  int lo = 0, hi = n_inst + 1;   // off[lo] <= g < off[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= g) lo = mid; else hi = mid;
  }
  return lo;
}

struct WorldArgs {
  int64_t n;
  const float* means;
  const float4* quats;
  const float* sh;
  const int64_t* inst_off;
  int n_inst;
  const float4* pose_q;
  const float* pose_t;
  float* means_out;
  float4* quats_out;
  float* sh_out;        // null: SH not rotated
  // backward
  float* g_means;
  float4* g_quats;
  float* g_sh;
  float* acc;           // [n_inst + 1][kWorldAcc]
  float* g_pose_q;
  float* g_pose_t;
};

// The SH basis at the 26 Lebedev points, [26][16] (once per CTA).
template <int DEG>
__device__ void lebedev_basis(float* s_Yd) {
  constexpr int K = sh_count(DEG);
  const int m = (int)threadIdx.x;
  if (m < 26) {
    float d[3], w, Y[16];
    lebedev26(m, d, w);
    sh_basis<DEG>(d[0], d[1], d[2], Y);
#pragma unroll
    for (int i = 0; i < K; ++i) s_Yd[m * 16 + i] = Y[i];
  }
}

// D_1..D_DEG of rotation R into s_D: first 4 pi w_m Y(R^T d_m) at the 26 points
// (a lane per point, in s_Yu), then a matrix entry per lane for its 26-term sum.
// Synchronises the warp before and after.
template <int DEG>
__device__ void instance_rotation(const float (&R)[9], const float* s_Yd, float* s_Yu, float* s_D) {
  constexpr int K = sh_count(DEG), E = rot_count(DEG);
  __syncwarp();
  const int m = (int)threadIdx.x;
  if (m < 26) {
    float d[3], w, Y[16];
    lebedev26(m, d, w);
    sh_basis<DEG>(R[0] * d[0] + R[3] * d[1] + R[6] * d[2], R[1] * d[0] + R[4] * d[1] + R[7] * d[2],
                  R[2] * d[0] + R[5] * d[1] + R[8] * d[2], Y);   // R^T d
    const float sw = 12.566370614359172f * w;
#pragma unroll
    for (int i = 0; i < K; ++i) s_Yu[m * 16 + i] = sw * Y[i];
  }
  __syncwarp();
  for (int r = (int)threadIdx.x; r < E; r += 32) {
    const int l = r < 9 ? 1 : (r < 34 ? 2 : 3);
    const int nb = 2 * l + 1, idx = r - rot_off(l), i = idx / nb, j = idx - i * nb, b = band_start(l);
    float acc = 0.f;
    for (int q = 0; q < 26; ++q) acc = fmaf(s_Yu[q * 16 + b + i], s_Yd[q * 16 + b + j], acc);
    s_D[r] = acc;
  }
  __syncwarp();
}

// A lane's own staged SH row (kFloatPitch floats from `row`) to and from
// registers: as float4s where the rows are (conflict-free across a quarter
// warp with the odd float4 pitch), else as floats.
template <int DEG>
__device__ __forceinline__ void row_get(const float* row, float (&c)[3 * sh_count(DEG)]) {
  using St = ShStage<DEG>;
  if constexpr (St::kVec) {
#pragma unroll
    for (int q = 0; q < St::kRow; ++q) {
      const float4 v = reinterpret_cast<const float4*>(row)[q];
      c[4 * q] = v.x; c[4 * q + 1] = v.y; c[4 * q + 2] = v.z; c[4 * q + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < 3 * sh_count(DEG); ++q) c[q] = row[q];
  }
}
template <int DEG>
__device__ __forceinline__ void row_put(float* row, const float (&c)[3 * sh_count(DEG)]) {
  using St = ShStage<DEG>;
  if constexpr (St::kVec) {
#pragma unroll
    for (int q = 0; q < St::kRow; ++q)
      reinterpret_cast<float4*>(row)[q] = make_float4(c[4 * q], c[4 * q + 1], c[4 * q + 2], c[4 * q + 3]);
  } else {
#pragma unroll
    for (int q = 0; q < 3 * sh_count(DEG); ++q) row[q] = c[q];
  }
}

// Coalesced copy of n_here staged rows to the consecutive rows g0.. of `sh`
// (the inverse of stage_sh_rows for consecutive Gaussians).
template <int DEG>
__device__ __forceinline__ void unstage_sh_rows(float* __restrict__ sh, const float* stage, int64_t g0,
                                                int n_here, uint32_t lane) {
  using St = ShStage<DEG>;
  if constexpr (St::kVec) {
    float4* dst = reinterpret_cast<float4*>(sh) + g0 * St::kRow;
    const float4* src = reinterpret_cast<const float4*>(stage);
    for (int idx = (int)lane; idx < n_here * St::kRow; idx += 32) {
      const int g = idx / St::kRow, q = idx - g * St::kRow;
      dst[idx] = src[g * St::kPitch + q];
    }
  } else {
    float* dst = sh + g0 * St::kRow;
    for (int idx = (int)lane; idx < n_here * St::kRow; idx += 32) {
      const int g = idx / St::kRow, q = idx - g * St::kRow;
      dst[idx] = stage[g * St::kPitch + q];
    }
  }
}

// Asynchronous copy of n consecutive SH rows from row g0 into `stage` (the
// layout of stage_sh_rows), 16 bytes per copy where the rows are float4s, else 4.
template <int DEG>
__device__ __forceinline__ void fetch_rows(float* stage, const float* __restrict__ sh, int64_t g0, int n,
                                           uint32_t lane) {
  using St = ShStage<DEG>;
  constexpr int kUnit = St::kVec ? 4 : 1;
  const float* src = sh + g0 * (St::kRow * kUnit);
  const uint32_t dst = (uint32_t)__cvta_generic_to_shared(stage);
#pragma unroll
  for (int it = 0; it < St::kRow; ++it) {
    const int idx = it * 32 + (int)lane;
    const int g = idx / St::kRow, q = idx - g * St::kRow;
    if (g < n) {
      const uint32_t d = dst + (uint32_t)(g * St::kPitch + q) * (4u * kUnit);
      if constexpr (St::kVec)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src + 4 * idx) : "memory");
      else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src + idx) : "memory");
    }
  }
}
__device__ __forceinline__ void fetch_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kLeft>
__device__ __forceinline__ void fetch_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kLeft) : "memory");
}

// A warp's walk over its contiguous range of dynamic rows: chunks of at most 32
// rows that end at an instance's last row at the latest.
struct RowWalk {
  const int64_t* off;
  int64_t g, end, inst_end;
  int k;              // instance of row g
  __device__ __forceinline__ void settle() {
    while (g < end && g >= inst_end) inst_end = off[++k + 1];
  }
  __device__ __forceinline__ RowWalk(const WorldArgs& a) {
    off = a.inst_off;
    const int64_t first = off[1], rows = a.n - first;
    // ranges are whole chunks of 32 rows (the last one is ragged)
    const int64_t chunks = (rows + 31) / 32, per = (chunks + gridDim.x - 1) / gridDim.x;
    g = min(a.n, first + (int64_t)blockIdx.x * per * 32);
    end = min(a.n, g + per * 32);
    k = 0;
    inst_end = 0;
    if (g < end) {
      k = segment_of_gid(off, a.n_inst, g);
      inst_end = off[k + 1];
      settle();
    }
  }
  __device__ __forceinline__ bool more() const { return g < end; }
  __device__ __forceinline__ int rows() const { return (int)min((int64_t)32, min(end, inst_end) - g); }
  __device__ __forceinline__ void next() {
    g += rows();
    settle();
  }
};

template <int DEG>
__global__ void __launch_bounds__(kWorldThreads) k_to_world(WorldArgs a) {
  using St = ShStage<DEG>;
  constexpr int K = sh_count(DEG);
  __shared__ float s_D[kRotFloats];
  __shared__ float s_Yd[26 * 16], s_Yu[26 * 16];
  __shared__ __align__(16) float s_rows[2][St::kWords];
  const uint32_t lane = threadIdx.x;
  const bool sh = a.sh_out != nullptr;
  const bool rotate = DEG > 0 && sh;
  RowWalk at(a);
  if (rotate) lebedev_basis<DEG>(s_Yd);   // read after instance_rotation's barriers
  if (sh && at.more()) fetch_rows<DEG>(s_rows[0], a.sh, at.g, at.rows(), lane);
  fetch_commit();
  int cur = 0, k_now = -1;
  float R[9], t[3] = {0.f, 0.f, 0.f};
  float4 p = make_float4(1.f, 0.f, 0.f, 0.f);   // the instance's unit quaternion
#pragma unroll
  for (int i = 0; i < 9; ++i) R[i] = 0.f;
  while (at.more()) {
    const int64_t g = at.g + lane;
    const int n = at.rows(), k = at.k;
    const int64_t g0 = at.g;
    const bool live = (int)lane < n;
    float m0 = 0.f, m1 = 0.f, m2 = 0.f;
    float4 q = make_float4(1.f, 0.f, 0.f, 0.f);
    if (live) {
      m0 = a.means[3 * g]; m1 = a.means[3 * g + 1]; m2 = a.means[3 * g + 2];
      q = a.quats[g];
    }
    at.next();
    if (sh && at.more()) fetch_rows<DEG>(s_rows[cur ^ 1], a.sh, at.g, at.rows(), lane);
    fetch_commit();
    if (k != k_now) {
      k_now = k;
      const float4 qp = a.pose_q[k - 1];
      quat_to_rot(qp, R);
      const float ip = rsqrtf(qp.x * qp.x + qp.y * qp.y + qp.z * qp.z + qp.w * qp.w);
      p = make_float4(qp.x * ip, qp.y * ip, qp.z * ip, qp.w * ip);
#pragma unroll
      for (int r = 0; r < 3; ++r) t[r] = a.pose_t[3 * (k - 1) + r];
      if (rotate) instance_rotation<DEG>(R, s_Yd, s_Yu, s_D);
    }
    if (live) {
      a.means_out[3 * g] = fmaf(R[0], m0, fmaf(R[1], m1, fmaf(R[2], m2, t[0])));
      a.means_out[3 * g + 1] = fmaf(R[3], m0, fmaf(R[4], m1, fmaf(R[5], m2, t[1])));
      a.means_out[3 * g + 2] = fmaf(R[6], m0, fmaf(R[7], m1, fmaf(R[8], m2, t[2])));
      const float iq = rsqrtf(q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w);
      const float w2 = q.x * iq, x2 = q.y * iq, y2 = q.z * iq, z2 = q.w * iq;
      a.quats_out[g] = make_float4(p.x * w2 - p.y * x2 - p.z * y2 - p.w * z2,
                                   p.x * x2 + p.y * w2 + p.z * z2 - p.w * y2,
                                   p.x * y2 - p.y * z2 + p.z * w2 + p.w * x2,
                                   p.x * z2 + p.y * y2 - p.z * x2 + p.w * w2);
    }
    if (sh) {
      fetch_wait<1>();   // this chunk's rows; the next chunk's may be in flight
      __syncwarp();
      float* rows = s_rows[cur];
      if (DEG > 0 && live) {
        // c'_l = D_l^T c_l per channel; degree 0 as is
        float c[3 * K], o[3 * K];
        float* row = rows + lane * St::kFloatPitch;
        row_get<DEG>(row, c);
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) o[ch] = c[ch];
#pragma unroll
        for (int l = 1; l <= DEG; ++l) {
          const int nb = 2 * l + 1, b = band_start(l);
#pragma unroll
          for (int j = 0; j < nb; ++j)
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
              float v = 0.f;
#pragma unroll
              for (int i = 0; i < nb; ++i) v = fmaf(s_D[rot_off(l) + i * nb + j], c[3 * (b + i) + ch], v);
              o[3 * (b + j) + ch] = v;
            }
        }
        row_put<DEG>(row, o);
      }
      __syncwarp();
      unstage_sh_rows<DEG>(a.sh_out, rows, g0, n, lane);
      __syncwarp();   // the buffer is refilled by the chunk after next
    }
    cur ^= 1;
  }
}

// The warp's sums of the lanes' values v[0..N), added to dst[0..N): 32 values
// at a time through shared memory (`s`, 32 x 33 floats), a lane per value.
template <int N>
__device__ __forceinline__ void flush_sums(float (&v)[N], float* s, float* dst, uint32_t lane) {
#pragma unroll
  for (int b = 0; b < N; b += 32) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (b + i < N) {
        s[i * 33 + lane] = v[b + i];
        v[b + i] = 0.f;
      }
    __syncwarp();
    if (b + (int)lane < N) {
      float x = 0.f, y = 0.f;
#pragma unroll
      for (int i = 0; i < 32; i += 2) {
        x += s[lane * 33 + i];
        y += s[lane * 33 + i + 1];
      }
      if (x + y != 0.f) atomicAdd(dst + b + lane, x + y);
    }
  }
  __syncwarp();
}

// Adjoint of the world transform for the dynamic rows, in place. Per
// Gaussian: dmu = R^T dmu_w; dq from q_w = p (x) q^ (dq^ = p* (x) dq_w, then
// through the normalisation); dc_l = D_l dc'_l. Per instance (summed): dR
// from the means and dD_l = sum c_l dc'_l^T, dt = sum dmu_w, dp = sum dq_w (x) q^*.
template <int DEG>
__global__ void __launch_bounds__(kWorldThreads) k_to_world_bwd(WorldArgs a) {
  using St = ShStage<DEG>;
  constexpr int E = rot_count(DEG);
  __shared__ float s_D[kRotFloats];
  __shared__ float s_Yd[26 * 16];
  __shared__ float s_tmp[32 * 33];    // the quadrature's values, and the lanes' sums when they are flushed
  __shared__ __align__(16) float s_c[2][St::kWords];
  __shared__ __align__(16) float s_g[2][St::kWords];
  static_assert(32 * 33 >= 26 * 16, "the quadrature's values fit the flush buffer");
  const uint32_t lane = threadIdx.x;
  const bool rotate = DEG > 0 && a.g_sh;
  RowWalk at(a);
  if (rotate) lebedev_basis<DEG>(s_Yd);
  auto fetch = [&](int buf) {
    if (rotate && at.more()) {
      fetch_rows<DEG>(s_c[buf], a.sh, at.g, at.rows(), lane);
      fetch_rows<DEG>(s_g[buf], a.g_sh, at.g, at.rows(), lane);
    }
    fetch_commit();
  };
  fetch(0);
  int cur = 0, k_now = -1;
  float R[9], sum[kPoseTerms], dD[E > 0 ? E : 1];
  float4 p = make_float4(1.f, 0.f, 0.f, 0.f);
  float np = 1.f;
#pragma unroll
  for (int i = 0; i < 9; ++i) R[i] = 0.f;
#pragma unroll
  for (int i = 0; i < kPoseTerms; ++i) sum[i] = 0.f;
#pragma unroll
  for (int i = 0; i < (E > 0 ? E : 1); ++i) dD[i] = 0.f;
  auto flush = [&]() {
    float* acc = a.acc + (size_t)k_now * kWorldAcc;
    flush_sums(sum, s_tmp, acc, lane);
    if (E > 0 && rotate) flush_sums(dD, s_tmp, acc + kPoseTerms, lane);
  };
  while (at.more()) {
    const int64_t g = at.g + lane;
    const int n = at.rows(), k = at.k;
    const int64_t g0 = at.g;
    const bool live = (int)lane < n;
    const bool do_m = live && a.g_means, do_q = live && a.g_quats;
    float d[3] = {0.f, 0.f, 0.f}, m[3] = {0.f, 0.f, 0.f};
    float4 q = make_float4(1.f, 0.f, 0.f, 0.f), G = make_float4(0.f, 0.f, 0.f, 0.f);
    if (do_m) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        d[i] = a.g_means[3 * g + i];
        m[i] = a.means[3 * g + i];
      }
    }
    if (do_q) {
      q = a.quats[g];
      G = a.g_quats[g];
    }
    at.next();
    fetch(cur ^ 1);
    if (k != k_now) {
      if (k_now >= 0) flush();
      k_now = k;
      const float4 qp = a.pose_q[k - 1];
      quat_to_rot(qp, R);
      np = sqrtf(qp.x * qp.x + qp.y * qp.y + qp.z * qp.z + qp.w * qp.w);
      p = make_float4(qp.x / np, qp.y / np, qp.z / np, qp.w / np);
      if (rotate) instance_rotation<DEG>(R, s_Yd, s_tmp, s_D);
    }
    if (do_m) {
      a.g_means[3 * g] = R[0] * d[0] + R[3] * d[1] + R[6] * d[2];
      a.g_means[3 * g + 1] = R[1] * d[0] + R[4] * d[1] + R[7] * d[2];
      a.g_means[3 * g + 2] = R[2] * d[0] + R[5] * d[1] + R[8] * d[2];
#pragma unroll
      for (int r = 0; r < 3; ++r) {
#pragma unroll
        for (int c = 0; c < 3; ++c) sum[3 * r + c] = fmaf(d[r], m[c], sum[3 * r + c]);
        sum[9 + r] += d[r];
      }
    }
    if (do_q) {
      const float nq = sqrtf(q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w);
      const float qw = q.x / nq, qx = q.y / nq, qy = q.z / nq, qz = q.w / nq;
      // dq^ = p* (x) G, then through the normalisation of q
      const float aw = p.x * G.x + p.y * G.y + p.z * G.z + p.w * G.w;
      const float ax = p.x * G.y - p.y * G.x - p.z * G.w + p.w * G.z;
      const float ay = p.x * G.z + p.y * G.w - p.z * G.x - p.w * G.y;
      const float az = p.x * G.w - p.y * G.z + p.z * G.y - p.w * G.x;
      const float dot = aw * qw + ax * qx + ay * qy + az * qz;
      a.g_quats[g] = make_float4((aw - qw * dot) / nq, (ax - qx * dot) / nq, (ay - qy * dot) / nq,
                                 (az - qz * dot) / nq);
      // dp^ = G (x) q^*
      sum[12] += G.x * qw + G.y * qx + G.z * qy + G.w * qz;
      sum[13] += -G.x * qx + G.y * qw - G.z * qz + G.w * qy;
      sum[14] += -G.x * qy + G.y * qz + G.z * qw - G.w * qx;
      sum[15] += -G.x * qz - G.y * qy + G.z * qx + G.w * qw;
    }
    if (rotate) {
      fetch_wait<1>();
      __syncwarp();
      if (live) {
        // a band at a time: its coefficients and adjoints in registers, the
        // rotated adjoints back over the staged row
        const float* crow = s_c[cur] + lane * St::kFloatPitch;
        float* grow = s_g[cur] + lane * St::kFloatPitch;
#pragma unroll
        for (int l = 1; l <= DEG; ++l) {
          constexpr int kMax = 3 * (2 * DEG + 1);
          const int nb = 2 * l + 1, b = band_start(l), o = rot_off(l);
          float c[kMax], gw[kMax];
#pragma unroll
          for (int i = 0; i < 3 * nb; ++i) {
            c[i] = crow[3 * b + i];
            gw[i] = grow[3 * b + i];
          }
#pragma unroll
          for (int i = 0; i < nb; ++i) {
            float v[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int j = 0; j < nb; ++j) {
              const float D = s_D[o + i * nb + j];
              float& e = dD[o + i * nb + j];
#pragma unroll
              for (int ch = 0; ch < 3; ++ch) {
                v[ch] = fmaf(D, gw[3 * j + ch], v[ch]);
                e = fmaf(c[3 * i + ch], gw[3 * j + ch], e);
              }
            }
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) grow[3 * (b + i) + ch] = v[ch];
          }
        }
      }
      __syncwarp();
      unstage_sh_rows<DEG>(a.g_sh, s_g[cur], g0, n, lane);
      __syncwarp();
    }
    cur ^= 1;
  }
  if (k_now >= 0) flush();
}

// Per instance, one warp: the pose adjoints from the sums (written), then the
// sums cleared. The quadrature's 26 points are a lane each. All sums are loaded
// before the first is cleared: with a load, a store, the next load of the row in
// turn, the loads waited for the stores (100,000 instances 0.30 ms, 0.06 so;
// in one thread per instance 0.07, but 80 instances several times longer).
constexpr int kPoseWarps = 4;
template <int DEG>
__global__ void __launch_bounds__(32 * kPoseWarps) k_world_pose(WorldArgs a) {
  __shared__ float s_accs[kPoseWarps][kWorldAcc];
  const int warp = (int)threadIdx.x >> 5, k = 1 + (int)blockIdx.x * kPoseWarps + warp;
  if (k > a.n_inst) return;   // whole warps; no barrier of the CTA follows
  float* s_acc = s_accs[warp];
  const uint32_t lane = threadIdx.x & 31u;
  float* acc = a.acc + (size_t)k * kWorldAcc;
  constexpr int kRounds = (kWorldAcc + 31) / 32;
  float sums[kRounds];
#pragma unroll
  for (int j = 0; j < kRounds; ++j) {
    const int i = 32 * j + (int)lane;
    sums[j] = i < kWorldAcc ? acc[i] : 0.f;
  }
#pragma unroll
  for (int j = 0; j < kRounds; ++j) {
    const int i = 32 * j + (int)lane;
    if (i < kWorldAcc) s_acc[i] = sums[j];
    if (sums[j] != 0.f) acc[i] = 0.f;
  }
  __syncwarp();
  const float4 qp = a.pose_q[k - 1];
  float dR[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) dR[i] = lane == 0 ? s_acc[i] : 0.f;
  if (DEG > 0) {
    // dD -> dR through D_ij = 4 pi sum_m w_m Y_i(R^T d_m) Y_j(d_m): with
    // u_m = R^T d_m, dL/du_m = 4 pi w_m grad(sum_i W_i Y_i)(u_m), W_i = sum_j dD_ij Y_j(d_m)
    float R[9];
    quat_to_rot(qp, R);
    if (lane < 26) {
      float d[3], w;
      lebedev26((int)lane, d, w);
      const float u[3] = {R[0] * d[0] + R[3] * d[1] + R[6] * d[2],
                          R[1] * d[0] + R[4] * d[1] + R[7] * d[2],
                          R[2] * d[0] + R[5] * d[1] + R[8] * d[2]};
      float Yd[16], W[16];
      sh_basis<DEG>(d[0], d[1], d[2], Yd);
#pragma unroll
      for (int i = 0; i < 16; ++i) W[i] = 0.f;
#pragma unroll
      for (int l = 1; l <= DEG; ++l) {
        const int nb = 2 * l + 1, b = band_start(l);
#pragma unroll
        for (int i = 0; i < nb; ++i) {
          float v = 0.f;
#pragma unroll
          for (int j = 0; j < nb; ++j) v = fmaf(s_acc[kPoseTerms + rot_off(l) + i * nb + j], Yd[b + j], v);
          W[b + i] = v;
        }
      }
      float gu[3];
      sh_dir_grad<DEG>(u[0], u[1], u[2], W, gu);
      const float s = 12.566370614359172f * w;
      // u_a = sum_b R_ba d_b
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c) dR[3 * b + c] = fmaf(s * gu[c], d[b], dR[3 * b + c]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < 9; ++i) dR[i] += __shfl_xor_sync(0xffffffffu, dR[i], o);
  if (lane != 0) return;
  float4 gq = quat_backward(qp, dR);
  const float np = sqrtf(qp.x * qp.x + qp.y * qp.y + qp.z * qp.z + qp.w * qp.w);
  const float pw = qp.x / np, px = qp.y / np, py = qp.z / np, pz = qp.w / np;
  const float dp[4] = {s_acc[12], s_acc[13], s_acc[14], s_acc[15]};
  const float dot = dp[0] * pw + dp[1] * px + dp[2] * py + dp[3] * pz;
  gq.x += (dp[0] - pw * dot) / np;
  gq.y += (dp[1] - px * dot) / np;
  gq.z += (dp[2] - py * dot) / np;
  gq.w += (dp[3] - pz * dot) / np;
  if (a.g_pose_q) {
    float* o = a.g_pose_q + 4 * (k - 1);
    o[0] = gq.x; o[1] = gq.y; o[2] = gq.z; o[3] = gq.w;
  }
  if (a.g_pose_t) {
    float* o = a.g_pose_t + 3 * (k - 1);
    o[0] = s_acc[9]; o[1] = s_acc[10]; o[2] = s_acc[11];
  }
}

}  // namespace

int world_acc_floats() { return kWorldAcc; }

namespace {
// CTAs of a world-transform launch: one resident wave (each CTA takes a
// contiguous range of chunks), fewer for a small scene. The occupancy of each
// kernel is queried once.
int64_t world_grid(const void* fn, int* cache, int64_t n_rows, int num_sms) {
  if (*cache == 0 &&
      (cudaOccupancyMaxActiveBlocksPerMultiprocessor(cache, fn, kWorldThreads, 0) != cudaSuccess || *cache < 1))
    *cache = 1;
  int64_t blocks = (n_rows + kWorldThreads - 1) / kWorldThreads;
  if (blocks > (int64_t)num_sms * *cache) blocks = (int64_t)num_sms * *cache;
  return blocks < 1 ? 1 : blocks;
}
}  // namespace

cudaError_t launch_to_world(const s3r_scene* sc, const s3r_poses* poses, float* means_out,
                            float* quats_out, float* sh_out, int64_t n_dynamic, int num_sms,
                            cudaStream_t st) {
  if (n_dynamic <= 0) return cudaSuccess;
  WorldArgs a = {};
  a.n = sc->n;
  a.means = sc->means;
  a.quats = reinterpret_cast<const float4*>(sc->quats);
  a.sh = sc->sh;
  a.inst_off = sc->inst_offsets;
  a.n_inst = sc->n_inst;
  a.pose_q = reinterpret_cast<const float4*>(poses->quat);
  a.pose_t = poses->trans;
  a.means_out = means_out;
  a.quats_out = reinterpret_cast<float4*>(quats_out);
  a.sh_out = sh_out;
  static thread_local int occ[4] = {0, 0, 0, 0};
  switch (sc->sh_degree) {
    case 0:
      k_to_world<0><<<(unsigned)world_grid((const void*)k_to_world<0>, &occ[0], n_dynamic, num_sms),
                      kWorldThreads, 0, st>>>(a);
      break;
    case 1:
      k_to_world<1><<<(unsigned)world_grid((const void*)k_to_world<1>, &occ[1], n_dynamic, num_sms),
                      kWorldThreads, 0, st>>>(a);
      break;
    case 2:
      k_to_world<2><<<(unsigned)world_grid((const void*)k_to_world<2>, &occ[2], n_dynamic, num_sms),
                      kWorldThreads, 0, st>>>(a);
      break;
    default:
      k_to_world<3><<<(unsigned)world_grid((const void*)k_to_world<3>, &occ[3], n_dynamic, num_sms),
                      kWorldThreads, 0, st>>>(a);
      break;
  }
  return cudaGetLastError();
}

cudaError_t launch_to_world_bwd(const s3r_scene* sc, const s3r_poses* poses, const s3r_grads* g,
                                float* acc, int64_t n_dynamic, int num_sms, cudaStream_t st) {
  if (sc->n_inst <= 0) return cudaSuccess;
  WorldArgs a = {};
  a.n = sc->n;
  a.means = sc->means;
  a.quats = reinterpret_cast<const float4*>(sc->quats);
  a.sh = sc->sh;
  a.inst_off = sc->inst_offsets;
  a.n_inst = sc->n_inst;
  a.pose_q = reinterpret_cast<const float4*>(poses->quat);
  a.pose_t = poses->trans;
  a.g_means = g->means;
  a.g_quats = reinterpret_cast<float4*>(g->quats);
  a.g_sh = g->sh;
  a.acc = acc;
  a.g_pose_q = g->inst_quat;
  a.g_pose_t = g->inst_trans;
  const unsigned pose_blocks = (unsigned)((sc->n_inst + kPoseWarps - 1) / kPoseWarps);
  static thread_local int occ[4] = {0, 0, 0, 0};
  switch (sc->sh_degree) {
    case 0:
      k_to_world_bwd<0><<<(unsigned)world_grid((const void*)k_to_world_bwd<0>, &occ[0], n_dynamic, num_sms),
                          kWorldThreads, 0, st>>>(a);
      k_world_pose<0><<<pose_blocks, 32 * kPoseWarps, 0, st>>>(a);
      break;
    case 1:
      k_to_world_bwd<1><<<(unsigned)world_grid((const void*)k_to_world_bwd<1>, &occ[1], n_dynamic, num_sms),
                          kWorldThreads, 0, st>>>(a);
      k_world_pose<1><<<pose_blocks, 32 * kPoseWarps, 0, st>>>(a);
      break;
    case 2:
      k_to_world_bwd<2><<<(unsigned)world_grid((const void*)k_to_world_bwd<2>, &occ[2], n_dynamic, num_sms),
                          kWorldThreads, 0, st>>>(a);
      k_world_pose<2><<<pose_blocks, 32 * kPoseWarps, 0, st>>>(a);
      break;
    default:
      k_to_world_bwd<3><<<(unsigned)world_grid((const void*)k_to_world_bwd<3>, &occ[3], n_dynamic, num_sms),
                          kWorldThreads, 0, st>>>(a);
      k_world_pose<3><<<pose_blocks, 32 * kPoseWarps, 0, st>>>(a);
      break;
  }
  return cudaGetLastError();
}

}  // namespace s3r
