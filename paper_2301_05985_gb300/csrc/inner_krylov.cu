// inner_krylov.cu -- FP32 kernels of the inner GMRES(d) that preconditions the flexible
// outer GMRES in mixed precision.  The inner solve is a fixed number of Arnoldi steps on
// J M^-1 (M: the 3x3 block diagonal) whose small Hessenberg bookkeeping also stays on the
// device, so it needs no host round trip; the outer Krylov method keeps FP64 dots,
// orthogonalisation and basis (Sec. 4.1's Newton-Krylov, with the bulk work in FP32).
#include <algorithm>
#include <cstdint>

#include "kernels.h"
#include "last_block.cuh"

namespace {

inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t); }

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
// vector's length), so both Gram-Schmidt kernels move float4: four entries per load.

// d_i = U_i . w (i < k) for FP32 vectors of n4 float4.  At most kInnerBlocks blocks (8 per
// SM) stride over chunks of 256 x kRows float4; for every group of four basis vectors a
// thread accumulates its rows of all chunks (w re-read from L2 per group), then one warp
// reduce-scatter and a fixed-order block sum give the block's partials part[i][block].
// Long vectors stream at HBM rate (89 %).  Short ones (a 163 k-node mesh: 240 chunks, the
// basis in L2) are latency: there blockIdx.y takes a share of the groups, and the last block
// adds the partials (`ticket` given) instead of a second launch.
constexpr int kRows = 2;
__device__ __forceinline__ float dot4(float4 a, float4 b, float s) {
  return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, s))));
}
__global__ void __launch_bounds__(256, 8) k_multi_dot_f32(int64_t n4, int k, const float4* __restrict__ Ub,
                                                          int64_t ld4, const float4* __restrict__ w, double* part,
                                                          unsigned* ticket, double* __restrict__ d) {
  __shared__ float sh[4][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t chunk = 256 * kRows;
  const int nb = gridDim.x;
  const int per = ((k + 3) / 4 + gridDim.y - 1) / gridDim.y * 4;  // vectors of this block
  const int je = min(k, ((int)blockIdx.y + 1) * per);
  for (int j0 = blockIdx.y * per; j0 < je; j0 += 4) {
    const int cnt = min(4, je - j0);
    float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int64_t c0 = (int64_t)blockIdx.x * chunk; c0 < n4; c0 += (int64_t)gridDim.x * chunk) {
      float4 wv[kRows];
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const int64_t t = c0 + threadIdx.x + r * 256;
        wv[r] = t < n4 ? w[t] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (q < cnt) {
          const float4* ui = Ub + (int64_t)(j0 + q) * ld4;
#pragma unroll
          for (int r = 0; r < kRows; ++r) {
            const int64_t t = c0 + threadIdx.x + r * 256;
            if (t < n4) s[q] = dot4(__ldg(ui + t), wv[r], s[q]);
          }
        }
      }
    }
    const float tot = warp_sum4f(s, lane);
    if ((lane & 7) == 0) sh[(lane >> 3) & 3][wid] = tot;
    __syncthreads();
    if (threadIdx.x < cnt) {
      double t = 0.0;
#pragma unroll
      for (int v = 0; v < 8; ++v) t += (double)sh[threadIdx.x][v];
      part[(int64_t)(j0 + threadIdx.x) * nb + blockIdx.x] = t;
    }
    __syncthreads();
  }
  if (!ticket || !last_block(ticket, gridDim.x * gridDim.y)) return;
  for (int j = wid; j < k; j += 8) {
    double t = 0.0;
#pragma unroll 4
    for (int b = lane; b < nb; b += 32) t += __ldcg(part + (int64_t)j * nb + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) d[j] = t;
  }
}

// Arnoldi bookkeeping of the inner process.  Basis vectors u_i are kept unnormalised
// with norms s_i (q_i = u_i / s_i).  The steps only store the Hessenberg columns
// h_i = d_i / s_i, h_(j+1) = s_(j+1); the Givens rotations wait for the least-squares
// kernel at the end, where the columns rotate in parallel.  (Rotating column j as it
// arrived kept one thread busy with up to 2 d dependent FP64 operations between two steps:
// 11 us per step at d = 24, as a launch of its own.)
// Scalar layout: H [(d+1) x d] row-major.
struct InnerStep {
  int j, d;            // column j of d; j < 0: the start vector
  const double* dd;    // projections of the step
  double *sv, *dinv;   // norms s_i and 1 / s_i^2
  float* inv_s;        // 1 / s_i
  double* H;
};

// w -= sum_i (d_i dinv_i) U_i (i < k) in FP32 on n4 float4, and w . w: at most kUpdBlocks
// blocks (6 per SM); the last one adds the partials and ends the Arnoldi step.
constexpr int kUpdBlocks = 6 * 152;
__global__ void __launch_bounds__(256, 6) k_multi_axpy_norm_f32(int64_t n4, int k, const float4* __restrict__ Ub,
                                                             int64_t ld4, float4* __restrict__ w, double* part,
                                                             unsigned* ticket, InnerStep S) {
  extern __shared__ float cf[];
  __shared__ double sh[256];
  for (int i = threadIdx.x; i < k; i += blockDim.x) cf[i] = (float)(S.dd[i] * S.dinv[i]);
  __syncthreads();
  float ss = 0.0f;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n4; t += (int64_t)gridDim.x * blockDim.x) {
    float4 a = w[t];
#pragma unroll 4
    for (int i = 0; i < k; ++i) {
      const float4 u = Ub[(int64_t)i * ld4 + t];
      const float c = -cf[i];
      a.x = fmaf(c, u.x, a.x);
      a.y = fmaf(c, u.y, a.y);
      a.z = fmaf(c, u.z, a.z);
      a.w = fmaf(c, u.w, a.w);
    }
    if (k > 0) w[t] = a;
    ss = fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(a.z, a.z, fmaf(a.w, a.w, ss))));
  }
  double tot = block_sum_d((double)ss, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = tot;
  if (!last_block(ticket, gridDim.x)) return;
  tot = 0.0;
#pragma unroll 4
  for (int b = threadIdx.x; b < (int)gridDim.x; b += 256) tot += __ldcg(part + b);
  tot = block_sum_d(tot, sh);
  const int i = threadIdx.x;
  if (i == 0) {
    const double s = sqrt(tot);
    S.sv[S.j + 1] = s;
    S.dinv[S.j + 1] = s > 0 ? 1.0 / (s * s) : 0.0;
    S.inv_s[S.j + 1] = s > 0 ? (float)(1.0 / s) : 0.0f;
    if (S.j >= 0) S.H[(int64_t)(S.j + 1) * S.d + S.j] = s;
  }
  if (i <= S.j) S.H[(int64_t)i * S.d + S.j] = S.sv[i] > 0 ? S.dd[i] / S.sv[i] : 0.0;
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
constexpr int kMaxInner = 64;
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

int inner_dot_blocks(int64_t n) {
  const int64_t chunk = 4 * 256 * kRows;
  return (int)std::min<int64_t>(kInnerBlocks, std::max<int64_t>(1, (n + chunk - 1) / chunk));
}
int inner_max_depth() { return kMaxInner; }

cudaError_t launch_multi_dot_f32(int64_t n, int k, const float* Ub, int64_t ld, const float* w, double* part,
                                 unsigned* ticket, double* d, cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  if ((n | ld) & 3) return cudaErrorInvalidValue;  // rows padded to float4
  const int nb = inner_dot_blocks(n), groups = (k + 3) / 4;
  const int gy = std::min(groups, std::max(1, kInnerBlocks / nb));
  // the last block adds up to 16 k partials; beyond that a block per vector does
  const bool fused = (int64_t)nb * k <= 16384;
  k_multi_dot_f32<<<dim3(nb, gy), 256, 0, s>>>(n / 4, k, (const float4*)Ub, ld / 4, (const float4*)w, part,
                                               fused ? ticket : nullptr, d);
  note_launch();
  return fused ? cudaGetLastError() : launch_reduce_cols(nb, k, part, d, s);
}

static cudaError_t launch_update(int64_t n, int k, const float* Ub, int64_t ld, float* w, double* part,
                                 unsigned* ticket, const InnerStep& S, cudaStream_t s) {
  if ((n | ld) & 3) return cudaErrorInvalidValue;  // rows padded to float4
  const int nb = (int)std::min<int64_t>(kUpdBlocks, std::max<int64_t>(1, (n / 4 + 255) / 256));
  k_multi_axpy_norm_f32<<<nb, 256, (k > 0 ? k : 1) * sizeof(float), s>>>(n / 4, k, (const float4*)Ub, ld / 4, (float4*)w,
                                                                        part, ticket, S);
  note_launch();
  return cudaGetLastError();
}
cudaError_t launch_inner_start(int64_t n, int d, float* u0, double* part, unsigned* ticket, double* sv, double* dinv,
                               float* inv_s, cudaStream_t s) {
  return launch_update(n, 0, u0, n, u0, part, ticket, InnerStep{-1, d, nullptr, sv, dinv, inv_s, nullptr}, s);
}
cudaError_t launch_inner_update(int64_t n, int j, int d, const float* Ub, int64_t ld, const double* dd, float* w,
                                double* part, unsigned* ticket, double* sv, double* dinv, float* inv_s, double* H,
                                cudaStream_t s) {
  return launch_update(n, j + 1, Ub, ld, w, part, ticket, InnerStep{j, d, dd, sv, dinv, inv_s, H}, s);
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
