// inner_krylov.cu -- FP32 kernels of the inner GMRES(d) that preconditions the flexible
// outer GMRES in mixed precision.  The inner solve is a fixed number of Arnoldi steps on
// J M^-1 (M: the 3x3 block diagonal) whose small Hessenberg bookkeeping also stays on the
// device, so it needs no host round trip; the outer Krylov method keeps FP64 dots,
// orthogonalisation and basis (Sec. 4.1's Newton-Krylov, with the bulk work in FP32).
#include <algorithm>
#include <cstdint>

#include "dot4.cuh"
#include "kernels.h"
#include "last_block.cuh"

namespace {

inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t); }

constexpr int kMaxInner = 64;
constexpr int kGsSums = kMaxInner + 2;

__device__ __forceinline__ float warp_sum4f(const float (&s)[4], int lane) {
  const bool hi4 = lane & 16, hi3 = lane & 8;
  const float a0 = (hi4 ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, hi4 ? s[0] : s[2], 16);
  const float a1 = (hi4 ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, hi4 ? s[1] : s[3], 16);
  float b = (hi3 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, hi3 ? a0 : a1, 8);
  b += __shfl_xor_sync(0xffffffffu, b, 4);
  b += __shfl_xor_sync(0xffffffffu, b, 2);
  b += __shfl_xor_sync(0xffffffffu, b, 1);
  return b;
}

__device__ __forceinline__ double block_sum_d(double v, double* sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  const double r = sh[0];
  __syncthreads();
  return r;
}

// The inner basis has rows padded to a multiple of four floats (zeros beyond the
// vector's length), so its kernels move float4: four entries per load.

// Arnoldi bookkeeping of the inner process.  Basis vectors u_i are kept unnormalised
// with norms s_i (q_i = u_i / s_i).  The steps only store the Hessenberg columns
// h_i = d_i / s_i, h_(j+1) = s_(j+1); the Givens rotations wait for the least-squares
// kernel at the end, where the columns rotate in parallel.  (Rotating column j as it
// arrived kept one thread busy with up to 2 d dependent FP64 operations between two steps:
// 11 us per step at d = 24, as a launch of its own.)
// Scalar layout: H [(d+1) x d] row-major.
struct InnerStep {
  int j, d;            // column j of d; j < 0: the start vector
  double *sv, *dinv;   // norms s_i and 1 / s_i^2
  float* inv_s;        // 1 / s_i
  double* H;
  double* sums;        // [2][kGsSums] projections and w . w, of even and of odd steps
  unsigned* arrived;   // blocks at the step's barrier (zero between launches)
};
__device__ __forceinline__ void axpy4(float c, const float4& u, float4& a) {
  a.x = fmaf(c, u.x, a.x);
  a.y = fmaf(c, u.y, a.y);
  a.z = fmaf(c, u.z, a.z);
  a.w = fmaf(c, u.w, a.w);
}

__device__ __forceinline__ void finish_norm(const InnerStep& S, double ww) {
  const double s = sqrt(ww);
  S.sv[S.j + 1] = s;
  S.dinv[S.j + 1] = s > 0 ? 1.0 / (s * s) : 0.0;
  S.inv_s[S.j + 1] = s > 0 ? (float)(1.0 / s) : 0.0f;
  if (S.j >= 0) S.H[(int64_t)(S.j + 1) * S.d + S.j] = s;
}

// The start vector's norm; clears the first step's sums
__global__ void __launch_bounds__(256) k_inner_start(int64_t n4, const float4* __restrict__ u, double* part,
                                                     unsigned* ticket, InnerStep S) {
  __shared__ double sh[256];
  float ss = 0.0f;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n4; t += (int64_t)gridDim.x * blockDim.x)
    ss = dot4(u[t], u[t], ss);
  double tot = block_sum_d((double)ss, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = tot;
  if (!last_block(ticket, gridDim.x)) return;
  tot = 0.0;
#pragma unroll 4
  for (int b = threadIdx.x; b < (int)gridDim.x; b += 256) tot += __ldcg(part + b);
  tot = block_sum_d(tot, sh);
  if (threadIdx.x == 0) finish_norm(S, tot);
  for (int i = threadIdx.x; i < kGsSums; i += 256) S.sums[i] = 0.0;
}

// One Gram-Schmidt step in one cooperative launch: d_i = U_i . w, a grid barrier, then
// w -= sum_i (d_i / s_i^2) U_i and w . w, for k FP32 vectors of n4 float4.  Each block walks
// its chunks of 256 float4 up for the sums and down for the update, so that the rows it ends
// the sums with come from L1 and L2 again.  The sums of the blocks meet in FP64 atomics (one
// per vector and block).  The barrier's wait is bounded: a block that gives up sets err (pinned
// host memory) and skips the update, but arrives at the end as the others do, so the counters
// are left as they were.
// What bounds it, a step's mean over 24: 163,000 nodes (the basis in L2) latency, 16 us, 27 us as
// a dot and an update kernel; 1,047,407 nodes memory, 57 us, 81 us as two (the basis read
// twice: 51 us at HBM rate, 13 vectors each way).
constexpr int kGsGroup = 24, kGsBatch = 8;
__global__ void __launch_bounds__(256, 3) k_inner_gs(int64_t n4, int k, const float4* __restrict__ Ub, int64_t ld4,
                                                     float4* w, unsigned* ticket, int* err, int polls, InnerStep S) {
  __shared__ float sh[kGsGroup][8];
  __shared__ float cf[kMaxInner];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t chunks = (n4 + 255) / 256;
  double *cur = S.sums + (S.j & 1) * kGsSums, *next = S.sums + (~S.j & 1) * kGsSums;
  for (int g0 = 0; g0 < k; g0 += kGsGroup) {
    float s[kGsGroup];
#pragma unroll
    for (int q = 0; q < kGsGroup; ++q) s[q] = 0.0f;
    for (int64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
      const int64_t t = c * 256 + tid;
      if (t >= n4) break;
      const float4 wv = w[t];
#pragma unroll
      for (int b = 0; b < kGsGroup; b += kGsBatch) {
        if (g0 + b >= k) break;
        float4 u[kGsBatch];
#pragma unroll
        for (int q = 0; q < kGsBatch; ++q) u[q] = __ldg(Ub + (int64_t)min(g0 + b + q, k - 1) * ld4 + t);
#pragma unroll
        for (int q = 0; q < kGsBatch; ++q) s[b + q] = dot4(u[q], wv, s[b + q]);
      }
    }
#pragma unroll
    for (int q = 0; q < kGsGroup; q += 4) {
      const float v[4] = {s[q], s[q + 1], s[q + 2], s[q + 3]};
      const float tot = warp_sum4f(v, lane);
      if ((lane & 7) == 0) sh[q + (lane >> 3)][wid] = tot;
    }
    __syncthreads();
    if (tid < kGsGroup && g0 + tid < k) {
      double t = 0.0;
#pragma unroll
      for (int v = 0; v < 8; ++v) t += (double)sh[tid][v];
      atomicAdd(cur + g0 + tid, t);
    }
    __syncthreads();
  }
  const bool passed = grid_barrier(S.arrived, err, polls);
  float ss = 0.0f;
  if (passed) {
    if (tid < k) {
      const double d = __ldcg(cur + tid);
      cf[tid] = -(float)(d * S.dinv[tid]);
      if (blockIdx.x == 0) S.H[(int64_t)tid * S.d + S.j] = S.sv[tid] > 0 ? d / S.sv[tid] : 0.0;
    }
    if (blockIdx.x == 0)
      for (int i = tid; i < kGsSums; i += 256) next[i] = 0.0;
    __syncthreads();
    const int64_t mine = blockIdx.x < chunks ? (chunks - 1 - blockIdx.x) / gridDim.x : -1;
    for (int64_t m = mine; m >= 0; --m) {
      const int64_t t = (blockIdx.x + m * gridDim.x) * 256 + tid;
      if (t >= n4) continue;
      float4 a = w[t];
      int i = 0;
      for (; i + kGsBatch <= k; i += kGsBatch) {
        float4 u[kGsBatch];
#pragma unroll
        for (int q = 0; q < kGsBatch; ++q) u[q] = __ldg(Ub + (int64_t)(i + q) * ld4 + t);
#pragma unroll
        for (int q = 0; q < kGsBatch; ++q) axpy4(cf[i + q], u[q], a);
      }
      if (i < k) {
        float4 u[kGsBatch];
#pragma unroll
        for (int q = 0; q < kGsBatch; ++q) u[q] = __ldg(Ub + (int64_t)min(i + q, k - 1) * ld4 + t);
#pragma unroll
        for (int q = 0; q < kGsBatch; ++q)
          if (i + q < k) axpy4(cf[i + q], u[q], a);
      }
      w[t] = a;
      ss = dot4(a, a, ss);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (lane == 0) sh[0][wid] = ss;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
#pragma unroll
    for (int v = 0; v < 8; ++v) t += (double)sh[0][v];
    atomicAdd(cur + kMaxInner, t);
  }
  if (!last_block(ticket, gridDim.x) || tid) return;
  *S.arrived = 0;  // every block has passed the barrier
  finish_norm(S, __ldcg(cur + kMaxInner));
}

// y_i = Dinv_i (inv_s[0] u_i) per node, FP32 3x3 blocks
__global__ void k_block_apply32(int64_t N, const float* __restrict__ Dinv, const float* __restrict__ u,
                                const float* __restrict__ inv_s, float* __restrict__ y) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float sc = inv_s ? inv_s[0] : 1.0f;
  const float* B = Dinv + 9 * i;
  const float a = sc * u[3 * i], b = sc * u[3 * i + 1], c = sc * u[3 * i + 2];
  y[3 * i] = fmaf(B[0], a, fmaf(B[1], b, B[2] * c));
  y[3 * i + 1] = fmaf(B[3], a, fmaf(B[4], b, B[5] * c));
  y[3 * i + 2] = fmaf(B[6], a, fmaf(B[7], b, B[8] * c));
}

// Least squares of the inner process and coef_i = y_i / s_i, so that sum_i y_i q_i = sum_i
// coef_i u_i.  Thread l holds column l: step j makes rotation j from column j and applies it
// to the columns after it; then a column-oriented back-substitution over the columns before
// the first breakdown (a zero rotated column).
__global__ void __launch_bounds__(kMaxInner) k_inner_lsq(int d, const double* __restrict__ sv,
                                                         const double* __restrict__ Hg, double* __restrict__ coef) {
  __shared__ double H[kMaxInner + 1][kMaxInner + 1], g[kMaxInner + 1], cs[kMaxInner], sn[kMaxInner], y[kMaxInner];
  __shared__ int kv;
  const int l = threadIdx.x;
  for (int t = l; t < (d + 1) * d; t += kMaxInner) {
    const int r = t / d, c = t - r * d;
    H[r][c] = r <= c + 1 ? Hg[t] : 0.0;
  }
  for (int t = l; t <= d; t += kMaxInner) g[t] = t == 0 ? sv[0] : 0.0;
  if (l == 0) kv = 0;
  __syncthreads();
  for (int j = 0; j < d; ++j) {
    if (l == j) {
      const double rr = hypot(H[j][j], H[j + 1][j]);
      cs[j] = 1.0;
      sn[j] = 0.0;
      if (rr > 0) {
        cs[j] = H[j][j] / rr;
        sn[j] = H[j + 1][j] / rr;
        H[j][j] = rr;
        g[j + 1] = -sn[j] * g[j];
        g[j] = cs[j] * g[j];
        if (kv == j) kv = j + 1;
      }
    }
    __syncthreads();
    if (l > j && l < d) {
      const double t = cs[j] * H[j][l] + sn[j] * H[j + 1][l];
      H[j + 1][l] = -sn[j] * H[j][l] + cs[j] * H[j + 1][l];
      H[j][l] = t;
    }
  }
  const int k = kv;
  for (int i = k - 1; i >= 0; --i) {
    if (l == i) y[i] = g[i] / H[i][i];
    __syncthreads();
    if (l < i) g[l] -= H[l][i] * y[i];
  }
  if (l < d) coef[l] = l < k ? y[l] / sv[l] : 0.0;
}

// out = sum_i coef_i U_i (FP32 vectors of n4 float4, coefficients on the device)
__global__ void k_combine_f32(int64_t n4, int k, const float4* __restrict__ Ub, int64_t ld4,
                              const double* __restrict__ coef, float4* __restrict__ out) {
  extern __shared__ float cf[];
  for (int i = threadIdx.x; i < k; i += blockDim.x) cf[i] = (float)coef[i];
  __syncthreads();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n4; t += (int64_t)gridDim.x * blockDim.x) {
    float4 v[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
#pragma unroll 4
    for (int i = 0; i < k; ++i) {
      const float4 u = Ub[(int64_t)i * ld4 + t];
      float4& a = v[i & 1];
      a.x = fmaf(cf[i], u.x, a.x);
      a.y = fmaf(cf[i], u.y, a.y);
      a.z = fmaf(cf[i], u.z, a.z);
      a.w = fmaf(cf[i], u.w, a.w);
    }
    out[t] = make_float4(v[0].x + v[1].x, v[0].y + v[1].y, v[0].z + v[1].z, v[0].w + v[1].w);
  }
}

// x += sum_i coef_i Z_i: FP32 vectors combined in FP32, added to an FP64 vector
__global__ void k_combine_f32_add_f64(int64_t n, int k, const float* __restrict__ Zb, int64_t ld,
                                      const double* __restrict__ coef, double* __restrict__ x) {
  extern __shared__ float cf[];
  for (int i = threadIdx.x; i < k; i += blockDim.x) cf[i] = (float)coef[i];
  __syncthreads();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    float v0 = 0.0f, v1 = 0.0f;
    int i = 0;
    for (; i + 2 <= k; i += 2) {
      v0 = fmaf(cf[i], Zb[(int64_t)i * ld + t], v0);
      v1 = fmaf(cf[i + 1], Zb[(int64_t)(i + 1) * ld + t], v1);
    }
    if (i < k) v0 = fmaf(cf[i], Zb[(int64_t)i * ld + t], v0);
    x[t] += (double)(v0 + v1);
  }
}

// y = scale * (double) x
__global__ void k_to_f64_scaled(int64_t n, const float* __restrict__ x, double scale, double* __restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = scale * (double)x[i];
}

}  // namespace

int inner_max_depth() { return kMaxInner; }
int inner_sum_doubles() { return 2 * kGsSums; }

cudaError_t launch_inner_start(int64_t n, int d, const float* u0, double* part, unsigned* ticket, double* sv,
                               double* dinv, float* inv_s, double* sums, cudaStream_t s) {
  if (n & 3) return cudaErrorInvalidValue;  // rows padded to float4
  const int nb = (int)std::min<int64_t>(kInnerBlocks, std::max<int64_t>(1, (n / 4 + 255) / 256));
  k_inner_start<<<nb, 256, 0, s>>>(n / 4, (const float4*)u0, part, ticket,
                                   InnerStep{-1, d, sv, dinv, inv_s, nullptr, sums, nullptr});
  note_launch();
  return cudaGetLastError();
}
cudaError_t launch_inner_gs(int64_t n, int j, int d, const float* Ub, int64_t ld, float* w, unsigned* ticket,
                            double* sv, double* dinv, float* inv_s, double* H, double* sums, unsigned* arrived, int* err,
                            int polls, cudaStream_t s) {
  if ((n | ld) & 3 || j + 1 > kMaxInner) return cudaErrorInvalidValue;  // rows padded to float4
  int dev = 0, n_sm = 0, per = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_inner_gs, 256, 0);
  if (e != cudaSuccess) return e;
  // chunks in equal shares of as many blocks as are resident together
  const int64_t chunks = std::max<int64_t>(1, (n / 4 + 255) / 256), most = (int64_t)n_sm * std::max(1, per);
  const int64_t share = (chunks + most - 1) / most, nb = (chunks + share - 1) / share;
  int64_t n4 = n / 4, ld4 = ld / 4;
  int k = j + 1;
  const float4* U = (const float4*)Ub;
  float4* w4 = (float4*)w;
  InnerStep S{j, d, sv, dinv, inv_s, H, sums, arrived};
  void* args[] = {&n4, &k, &U, &ld4, &w4, &ticket, &err, &polls, &S};
  e = cudaLaunchCooperativeKernel(k_inner_gs, dim3((unsigned)nb), dim3(256), args, 0, s);
  note_launch();
  return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t launch_block_apply32(int64_t N, const float* Dinv32, const float* u, const float* inv_s, float* y,
                                 cudaStream_t s) {
  if (N) {
    k_block_apply32<<<nblk(N, 256), 256, 0, s>>>(N, Dinv32, u, inv_s, y);
    note_launch();
  }
  return cudaGetLastError();
}

cudaError_t launch_inner_lsq(int d, const double* sv, const double* H, double* coef, cudaStream_t s) {
  k_inner_lsq<<<1, kMaxInner, 0, s>>>(d, sv, H, coef);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_combine_f32(int64_t n, int k, const float* Ub, int64_t ld, const double* coef, float* out,
                               cudaStream_t s) {
  if ((n | ld) & 3) return cudaErrorInvalidValue;  // rows padded to float4
  const unsigned nb = (unsigned)std::min<int64_t>(2 * kRedBlocks, std::max<int64_t>(1, (n / 4 + 255) / 256));
  k_combine_f32<<<nb, 256, (k > 0 ? k : 1) * sizeof(float), s>>>(n / 4, k, (const float4*)Ub, ld / 4, coef, (float4*)out);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_combine_f32_add_f64(int64_t n, int k, const float* Zb, int64_t ld, const double* coef, double* x,
                                       cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  k_combine_f32_add_f64<<<kRedBlocks, 256, k * sizeof(float), s>>>(n, k, Zb, ld, coef, x);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_to_f64_scaled(int64_t n, const float* x, double scale, double* y, cudaStream_t s) {
  k_to_f64_scaled<<<kRedBlocks, 256, 0, s>>>(n, x, scale, y);
  note_launch();
  return cudaGetLastError();
}
