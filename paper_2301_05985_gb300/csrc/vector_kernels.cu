// vector_kernels.cu -- streaming kernels of the Newton-Krylov loop (history, conversions,
// deterministic FP64 reductions, Gram-Schmidt multi-dot / multi-axpy, 3x3 block Jacobi).
// All of these are HBM-bound: one coalesced pass over their operands.
#include <algorithm>
#include <atomic>

#include "kernels.h"
#include "last_block.cuh"

static std::atomic<int64_t> g_launches{0};
void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
void note_launches(int64_t n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
int64_t launch_count() { return g_launches.load(); }
extern "C" int64_t pnp_kernel_launches(void) { return g_launches.load(); }
static std::atomic<int64_t> g_captures{0};
void note_capture() { g_captures.fetch_add(1, std::memory_order_relaxed); }
extern "C" int64_t pnp_graph_captures(void) { return g_captures.load(); }

namespace {

inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t); }
inline int gs_blocks(int64_t n, int t) {
  const int64_t b = (n + t - 1) / t;
  return (int)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

__global__ void k_history(int64_t N, const double* __restrict__ Uk, const double* __restrict__ Ukm1, double b1,
                          double b2, double inv_dt, double* __restrict__ hs) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  hs[2 * i + 0] = (b1 * Uk[3 * i + 0] + b2 * Ukm1[3 * i + 0]) * inv_dt;
  hs[2 * i + 1] = (b1 * Uk[3 * i + 1] + b2 * Ukm1[3 * i + 1]) * inv_dt;
}

__global__ void k_to_f32(int64_t n, const double* __restrict__ x, float* __restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = (float)x[i];
}
__global__ void k_to_f64(int64_t n, const float* __restrict__ x, double* __restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = (double)x[i];
}
// b = 0 does not read y (it may hold any bit pattern, NaN included: 0 * NaN is NaN)
__global__ void k_axpby(int64_t n, double a, const double* __restrict__ x, double b, double* __restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = b == 0.0 ? a * x[i] : a * x[i] + b * y[i];
}
__global__ void k_axpbyz(int64_t n, double a, const double* __restrict__ x, double b, const double* __restrict__ y,
                         double* __restrict__ z) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    z[i] = b == 0.0 ? a * x[i] : a * x[i] + b * y[i];
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
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

// partial sums of x . y per block; the last block adds them (fixed order) and writes the sum,
// or its square root, to the device and (host, may be null) to mapped pinned memory: one
// launch where the partials, their sum and a copy to the host were three operations
__global__ void __launch_bounds__(kRedThreads) k_dot(int64_t n, const double* __restrict__ x,
                                                     const double* __restrict__ y, double* part, unsigned* ticket,
                                                     int take_sqrt, double* __restrict__ out,
                                                     double* __restrict__ host) {
  __shared__ double sh[kRedThreads];
  double s = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s += x[i] * y[i];
  s = block_sum(s, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
  if (!last_block(ticket, gridDim.x)) return;
  s = 0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) s += __ldcg(part + b);
  s = block_sum(s, sh);
  if (threadIdx.x == 0) {
    const double r = take_sqrt ? sqrt(s) : s;
    out[0] = r;
    if (host) host[0] = r;
  }
}

// one block per output: out[j] = sum_b part[b * sb + j * sj]
__global__ void __launch_bounds__(kRedThreads) k_reduce_parts(int nparts, int64_t sb, int64_t sj,
                                                              const double* __restrict__ part,
                                                              double* __restrict__ out) {
  __shared__ double sh[kRedThreads];
  const int j = blockIdx.x;
  double s = 0;
  for (int b = threadIdx.x; b < nparts; b += blockDim.x) s += part[b * sb + j * sj];
  s = block_sum(s, sh);
  if (threadIdx.x == 0) out[j] = s;
}

// Sum over the warp of four per-lane values at once (reduce-scatter: 6 adds per lane
// instead of 4 x 5); lanes 8q .. 8q+7 end with the total of s[q].  Fixed order.
__device__ __forceinline__ double warp_sum4(const double (&s)[4], int lane) {
  const bool hi4 = lane & 16, hi3 = lane & 8;
  const double a0 = (hi4 ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, hi4 ? s[0] : s[2], 16);
  const double a1 = (hi4 ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, hi4 ? s[1] : s[3], 16);
  double b = (hi3 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, hi3 ? a0 : a1, 8);
  b += __shfl_xor_sync(0xffffffffu, b, 4);
  b += __shfl_xor_sync(0xffffffffu, b, 2);
  b += __shfl_xor_sync(0xffffffffu, b, 1);
  return b;
}

// d_i = V_i . w (i < k).  A block owns 256 R rows: w's rows stay in registers while the block
// sweeps its share of the basis four vectors at a time (4 R independent loads per thread,
// one reduce-scatter over the warp, fixed order).  The partials go to part[i][block]; with
// `ticket`, the last block adds them (a warp per vector).
// Rows and split by size (multi_dot_shape): for long vectors the FP64 pipe bounds the kernel
// (84 % of its peak) and R = 16 rows per thread keep the reduction adds small next to the
// FMAs; for short ones it is latency, and with R = 16 a 3,267-entry vector was one block
// that swept the whole basis alone (28 us at up to 30 vectors).  Short vectors take one row
// per thread and a block per four vectors.
template <int R>
__global__ void __launch_bounds__(256, 4) k_multi_dot(int64_t n, int k, const double* __restrict__ Vb, int64_t ld,
                                                      const double* __restrict__ w, double* part, unsigned* ticket,
                                                      double* __restrict__ d) {
  __shared__ double sh[4][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t base = (int64_t)blockIdx.x * (256 * R) + threadIdx.x;
  const int nb = gridDim.x;
  const int per = ((k + 3) / 4 + gridDim.y - 1) / gridDim.y * 4;  // vectors of this block
  const int jb = blockIdx.y * per, je = min(k, jb + per);
  double wv[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t t = base + r * 256;
    wv[r] = t < n ? w[t] : 0.0;
  }
  for (int j0 = jb; j0 < je; j0 += 4) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (j0 + q < je) {
        const double* vi = Vb + (int64_t)(j0 + q) * ld;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int64_t t = base + r * 256;
          if (t < n) s[q] = fma(__ldg(vi + t), wv[r], s[q]);
        }
      }
    }
    const double tot = warp_sum4(s, lane);
    if ((lane & 7) == 0) sh[(lane >> 3) & 3][wid] = tot;
    __syncthreads();
    if (threadIdx.x < 4 && j0 + (int)threadIdx.x < je) {
      double t = 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q) t += sh[threadIdx.x][q];
      part[(int64_t)(j0 + threadIdx.x) * nb + blockIdx.x] = t;
    }
    __syncthreads();
  }
  if (!ticket || !last_block(ticket, gridDim.x * gridDim.y)) return;
  for (int j = wid; j < k; j += 8) {
    double t = 0.0;
    for (int b = lane; b < nb; b += 32) t += __ldcg(part + (int64_t)j * nb + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) d[j] = t;
  }
}

__device__ __forceinline__ void finish_step(const GsFinish& f, int k, double ss) {
  if (threadIdx.x == 0) {
    f.nrm2[0] = ss;
    if (f.dinv_next) f.dinv_next[0] = ss > 0.0 ? 1.0 / ss : 0.0;
    if (f.inv_s_next) f.inv_s_next[0] = ss > 0.0 ? 1.0 / sqrt(ss) : 0.0;
    if (f.host_nrm2) f.host_nrm2[0] = ss;
  }
  if (f.host0)
    for (int i = threadIdx.x; i < k; i += blockDim.x) f.host0[i] = __ldcg(f.d0 + i);
  if (f.host1)
    for (int i = threadIdx.x; i < k; i += blockDim.x) f.host1[i] = __ldcg(f.d1 + i);
}

// w -= sum_i (d_i * dinv_i) V_i and w . w of the updated w; the last block adds the partials
// and finishes the Krylov step: w . w and its reciprocal for the next vector on the device,
// and what the host needs of the step into mapped pinned memory (GsFinish)
__global__ void __launch_bounds__(kRedThreads) k_multi_axpy_norm(int64_t n, int k, const double* __restrict__ Vb,
                                                                 int64_t ld, const double* __restrict__ d,
                                                                 const double* __restrict__ dinv,
                                                                 double* __restrict__ w, double* part,
                                                                 unsigned* ticket, GsFinish f) {
  extern __shared__ double cf[];
  __shared__ double sh[kRedThreads];
  for (int i = threadIdx.x; i < k; i += blockDim.x) cf[i] = d[i] * dinv[i];
  __syncthreads();
  double ss = 0.0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    // two independent chains; eight loads in flight
    double v0 = w[t], v1 = 0.0;
    int i = 0;
#pragma unroll 4
    for (; i + 2 <= k; i += 2) {
      v0 -= cf[i] * Vb[(int64_t)i * ld + t];
      v1 -= cf[i + 1] * Vb[(int64_t)(i + 1) * ld + t];
    }
    if (i < k) v0 -= cf[i] * Vb[(int64_t)i * ld + t];
    const double v = v0 + v1;
    w[t] = v;
    ss += v * v;
  }
  ss = block_sum(ss, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = ss;
  if (!last_block(ticket, gridDim.x)) return;
  ss = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) ss += __ldcg(part + b);
  ss = block_sum(ss, sh);
  finish_step(f, k, ss);
}

// One Gram-Schmidt step of short vectors in one cooperative launch: d_i = V_i . w, a grid
// barrier, w -= sum_i (d_i dinv_i) V_i and w . w, and the step's end (GsFinish).  Sums: a block
// per four vectors and chunk of rows (at most kGsChunks chunks), partials to
// part[i][chunk], added in order by every block.  Update: a block per 32 rows, its warps
// sharing the vectors.  The barrier's wait is bounded.  Latency, all of it.
constexpr int kGsChunks = 64;
constexpr int64_t kGsShort = int64_t(1) << 16;
__global__ void __launch_bounds__(256) k_gs_step(int64_t n, int k, const double* __restrict__ Vb, int64_t ld,
                                                 double* d, const double* __restrict__ dinv, double* w, double* part,
                                                 unsigned* ticket, unsigned* arrived, int* err, int polls,
                                                 GsFinish f) {
  extern __shared__ double cf[];
  __shared__ double sh[8][33];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int groups = (k + 3) / 4;
  const int xb = (int)((n + 255) / 256 < kGsChunks ? (n + 255) / 256 : kGsChunks);
  const int64_t rows = ((n + xb - 1) / xb + 255) / 256 * 256;
  for (int task = blockIdx.x; task < xb * groups; task += gridDim.x) {
    const int x = task % xb, j0 = task / xb * 4;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    const int64_t t1 = (x + 1) * rows < n ? (x + 1) * rows : n;
#pragma unroll 2
    for (int64_t t = x * rows + threadIdx.x; t < t1; t += 256) {
      const double wv = w[t];
#pragma unroll
      for (int q = 0; q < 4; ++q) s[q] = fma(__ldg(Vb + (int64_t)min(j0 + q, k - 1) * ld + t), wv, s[q]);
    }
    const double tot = warp_sum4(s, lane);
    if ((lane & 7) == 0) sh[lane >> 3][wid] = tot;
    __syncthreads();
    if (threadIdx.x < 4 && j0 + (int)threadIdx.x < k) {
      double t = 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q) t += sh[threadIdx.x][q];
      part[(int64_t)(j0 + threadIdx.x) * xb + x] = t;
    }
    __syncthreads();
  }
  const bool passed = grid_barrier(arrived, err, polls);
  double ss = 0.0;
  if (passed) {
    // four lanes per vector
    for (int j0 = 0; j0 < k; j0 += 64) {
      const int j = j0 + (threadIdx.x >> 2);
      double t = 0.0;
      if (j < k) {
#pragma unroll 4
        for (int b = threadIdx.x & 3; b < xb; b += 4) t += __ldcg(part + (int64_t)j * xb + b);
      }
      t += __shfl_xor_sync(0xffffffffu, t, 1);
      t += __shfl_xor_sync(0xffffffffu, t, 2);
      if (j < k && (threadIdx.x & 3) == 0) {
        cf[j] = t * dinv[j];
        if (blockIdx.x == 0) d[j] = t;
      }
    }
    __syncthreads();
    for (int64_t r0 = (int64_t)blockIdx.x * 32; r0 < n; r0 += (int64_t)gridDim.x * 32) {
      const int64_t t = r0 + lane;
      double v = 0.0;
      if (t < n) {
#pragma unroll 4
        for (int i = wid; i < k; i += 8) v = fma(cf[i], __ldg(Vb + (int64_t)i * ld + t), v);
      }
      sh[wid][lane] = v;
      __syncthreads();
      if (wid == 0 && t < n) {
        double a = w[t];
#pragma unroll
        for (int q = 0; q < 8; ++q) a -= sh[q][lane];
        w[t] = a;
        ss = fma(a, a, ss);
      }
      __syncthreads();
    }
  }
  grid_dependency_release();
  if (wid == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (lane == 0) part[(int64_t)k * xb + blockIdx.x] = ss;
  }
  if (!last_block(ticket, gridDim.x)) return;
  if (threadIdx.x == 0) *arrived = 0;  // every block has passed the barrier
  ss = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += 256) ss += __ldcg(part + (int64_t)k * xb + b);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  __syncthreads();
  if (lane == 0) sh[0][wid] = ss;
  __syncthreads();
  ss = 0.0;
#pragma unroll
  for (int q = 0; q < 8; ++q) ss += sh[0][q];
  finish_step(f, k, ss);
}

__global__ void __launch_bounds__(256) k_multi_axpy(int64_t n, int k, const double* __restrict__ Vb, int64_t ld,
                                                    const double* __restrict__ h, double* __restrict__ w) {
  extern __shared__ double hs[];
  for (int i = threadIdx.x; i < k; i += blockDim.x) hs[i] = h[i];
  __syncthreads();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    double v = w[t];
    for (int i = 0; i < k; ++i) v -= hs[i] * Vb[(int64_t)i * ld + t];
    w[t] = v;
  }
}

__global__ void k_block_apply(int64_t N, const double* __restrict__ Dinv, const double* __restrict__ v, double scale,
                              const double* __restrict__ scale_dev, double* __restrict__ z, float* __restrict__ z32) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  if (scale_dev) scale = *scale_dev;
  const double* B = Dinv + 9 * i;
  const double a = scale * v[3 * i], b = scale * v[3 * i + 1], c = scale * v[3 * i + 2];
  const double r0 = B[0] * a + B[1] * b + B[2] * c;
  const double r1 = B[3] * a + B[4] * b + B[5] * c;
  const double r2 = B[6] * a + B[7] * b + B[8] * c;
  if (z) {
    z[3 * i] = r0;
    z[3 * i + 1] = r1;
    z[3 * i + 2] = r2;
  }
  if (z32) {
    z32[3 * i] = (float)r0;
    z32[3 * i + 1] = (float)r1;
    z32[3 * i + 2] = (float)r2;
  }
}

template <typename T>
__global__ void k_block_invert(int64_t N, const T* D, double* Dinv, int* __restrict__ flag) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  double a[3][6];
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) {
      a[r][c] = (double)D[9 * i + 3 * r + c];
      a[r][3 + c] = (r == c) ? 1.0 : 0.0;
    }
  for (int col = 0; col < 3; ++col) {
    int piv = col;
    for (int r = col + 1; r < 3; ++r)
      if (fabs(a[r][col]) > fabs(a[piv][col])) piv = r;
    if (a[piv][col] == 0.0 || !isfinite(a[piv][col])) {
      atomicOr(flag, 1);
      return;
    }
    if (piv != col)
      for (int c = 0; c < 6; ++c) {
        const double t = a[col][c];
        a[col][c] = a[piv][c];
        a[piv][c] = t;
      }
    const double inv = 1.0 / a[col][col];
    for (int c = 0; c < 6; ++c) a[col][c] *= inv;
    for (int r = 0; r < 3; ++r)
      if (r != col) {
        const double f = a[r][col];
        for (int c = 0; c < 6; ++c) a[r][c] -= f * a[col][c];
      }
  }
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) Dinv[9 * i + 3 * r + c] = a[r][3 + c];
}

__global__ void k_set_dirichlet(int64_t N, const uint8_t* __restrict__ faces, BcTable bc, double* __restrict__ U) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  const uint8_t fm = faces[i];
  if (fm & 0x80) return;
  for (int f = 0; f < 3; ++f) {
    const unsigned msk = fm & bc.dir_faces[f] & 0x3F;
    if (msk) U[3 * i + f] = bc.val[31 - __clz(msk)][f];
  }
}

__global__ void k_interp_hanging(int64_t H, const int32_t* __restrict__ hnode, const int32_t* __restrict__ hpar,
                                 const uint8_t* __restrict__ hnp, double* __restrict__ U) {
  const int64_t h = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (h >= H) return;
  const int np = hnp[h];
  const double wgt = np == 2 ? 0.5 : 0.25;
  for (int f = 0; f < 3; ++f) {
    double s = 0;
    for (int p = 0; p < np; ++p) s += wgt * U[3 * (int64_t)hpar[4 * h + p] + f];
    U[3 * (int64_t)hnode[h] + f] = s;
  }
}

__global__ void k_vel_pack(int64_t N, int dim, const double* __restrict__ src, double* __restrict__ dst3) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  for (int k = 0; k < 3; ++k) dst3[3 * i + k] = k < dim ? src[dim * i + k] : 0.0;
}
__global__ void k_vel_unpack(int64_t N, int dim, const double* __restrict__ src3, double* __restrict__ dst) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  for (int k = 0; k < dim; ++k) dst[dim * i + k] = src3[3 * i + k];
}

}  // namespace

cudaError_t launch_history(int64_t N, const double* Uk, const double* Ukm1, double b1, double b2, double dt,
                           double* hs, cudaStream_t s) {
  if (N) { k_history<<<nblk(N, 256), 256, 0, s>>>(N, Uk, Ukm1, b1, b2, 1.0 / dt, hs); note_launch(); }
  return cudaGetLastError();
}
cudaError_t launch_to_f32(int64_t n, const double* x, float* y, cudaStream_t s) {
  if (n) { k_to_f32<<<gs_blocks(n, 256), 256, 0, s>>>(n, x, y); note_launch(); }
  return cudaGetLastError();
}
cudaError_t launch_to_f64(int64_t n, const float* x, double* y, cudaStream_t s) {
  if (n) { k_to_f64<<<gs_blocks(n, 256), 256, 0, s>>>(n, x, y); note_launch(); }
  return cudaGetLastError();
}
cudaError_t launch_axpby(int64_t n, double a, const double* x, double b, double* y, cudaStream_t s) {
  if (n) { k_axpby<<<gs_blocks(n, 256), 256, 0, s>>>(n, a, x, b, y); note_launch(); }
  return cudaGetLastError();
}
cudaError_t launch_axpbyz(int64_t n, double a, const double* x, double b, const double* y, double* z, cudaStream_t s) {
  if (n) { k_axpbyz<<<gs_blocks(n, 256), 256, 0, s>>>(n, a, x, b, y, z); note_launch(); }
  return cudaGetLastError();
}
// threads and blocks of a reduction over n entries: at most kRedBlocks blocks of 256, for
// short vectors (fewer than 64 kRedBlocks entries) blocks of 64
static int red_threads(int64_t n) { return n < int64_t(64) * kRedBlocks ? 64 : kRedThreads; }
static int red_blocks(int64_t n) {
  const int t = red_threads(n);
  return (int)std::min<int64_t>(kRedBlocks, std::max<int64_t>(1, (n + t - 1) / t));
}

cudaError_t launch_dot(int64_t n, const double* x, const double* y, double* part, unsigned* ticket, double* result,
                       double* host, cudaStream_t s) {
  k_dot<<<red_blocks(n), red_threads(n), 0, s>>>(n, x, y, part, ticket, 0, result, host);
  note_launch();
  return cudaGetLastError();
}
cudaError_t launch_norm2(int64_t n, const double* x, double* part, unsigned* ticket, double* result, double* host,
                         cudaStream_t s) {
  k_dot<<<red_blocks(n), red_threads(n), 0, s>>>(n, x, x, part, ticket, 1, result, host);
  note_launch();
  return cudaGetLastError();
}
cudaError_t launch_multi_axpy(int64_t n, int k, const double* Vb, int64_t ld, const double* h, double* w,
                              cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  k_multi_axpy<<<gs_blocks(n, 256), 256, k * sizeof(double), s>>>(n, k, Vb, ld, h, w); note_launch();
  return cudaGetLastError();
}
__global__ void k_node_records(int64_t N, const double* __restrict__ U, const double* __restrict__ hs,
                               const double* __restrict__ adv, float4* __restrict__ rec) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  rec[2 * i] = make_float4((float)U[3 * i], (float)U[3 * i + 1], (float)U[3 * i + 2], (float)hs[2 * i]);
  rec[2 * i + 1] = make_float4((float)hs[2 * i + 1], (float)adv[3 * i], (float)adv[3 * i + 1], (float)adv[3 * i + 2]);
}

cudaError_t launch_node_records(int64_t N, const double* U, const double* hs, const double* adv, float4* rec,
                                cudaStream_t s) {
  if (N) {
    k_node_records<<<nblk(N, 256), 256, 0, s>>>(N, U, hs, adv, rec);
    note_launch();
  }
  return cudaGetLastError();
}

cudaError_t launch_reduce_parts(int nparts, int k, const double* part, double* out, cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  k_reduce_parts<<<k, kRedThreads, 0, s>>>(nparts, k, 1, part, out);
  note_launch();
  return cudaGetLastError();
}
cudaError_t launch_reduce_cols(int nparts, int k, const double* part, double* out, cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  k_reduce_parts<<<k, kRedThreads, 0, s>>>(nparts, 1, nparts, part, out);
  note_launch();
  return cudaGetLastError();
}

// rows per thread: 16 while that leaves two blocks per SM (vectors of 1.2 M entries and
// more), 4 down to 155 k entries, 1 below
static int multi_dot_rows(int64_t n) { return n >= int64_t(304) * 4096 ? 16 : n >= int64_t(152) * 1024 ? 4 : 1; }
int multi_dot_blocks(int64_t n) {
  const int64_t rows = 256 * multi_dot_rows(n);
  return (int)std::max<int64_t>(1, (n + rows - 1) / rows);
}

cudaError_t launch_multi_dot(int64_t n, int k, const double* Vb, int64_t ld, const double* w, double* part,
                             unsigned* ticket, double* d, cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  const int nb = multi_dot_blocks(n), rows = multi_dot_rows(n), groups = (k + 3) / 4;
  // short vectors: a block per four vectors until the chip has eight blocks per SM
  const int gy = rows == 16 ? 1 : (int)std::min<int64_t>(groups, std::max<int64_t>(1, 1216 / nb));
  // the last block adds up to 16 k partials (about 4 us); beyond that a block per vector does
  const bool fused = (int64_t)nb * k <= 16384;
  unsigned* tk = fused ? ticket : nullptr;
  const dim3 grid(nb, gy);
  if (rows == 16) k_multi_dot<16><<<grid, 256, 0, s>>>(n, k, Vb, ld, w, part, tk, d);
  else if (rows == 4) k_multi_dot<4><<<grid, 256, 0, s>>>(n, k, Vb, ld, w, part, tk, d);
  else k_multi_dot<1><<<grid, 256, 0, s>>>(n, k, Vb, ld, w, part, tk, d);
  note_launch();
  return fused ? cudaGetLastError() : launch_reduce_cols(nb, k, part, d, s);
}
cudaError_t launch_multi_axpy_norm(int64_t n, int k, const double* Vb, int64_t ld, const double* d, const double* dinv,
                                   double* w, double* part, unsigned* ticket, const GsFinish& f, cudaStream_t s) {
  k_multi_axpy_norm<<<red_blocks(n), red_threads(n), (k > 0 ? k : 1) * sizeof(double), s>>>(n, k, Vb, ld, d, dinv, w,
                                                                                           part, ticket, f);
  note_launch();
  return cudaGetLastError();
}
// Short vectors: one cooperative launch (k_gs_step).  GMRES(50) iterations with it and with the
// two kernels (none of an iteration's launches dependent), 2D: 867 unknowns 26.4 and 31.8 us, 3,267 27.4 and 32.5, 12,675 35.5 and 38.1,
// 49,923 59.1 and 62.5, 198,147 137 and 131, 789,507 485 and 435 (the FP64 pipe; the barrier
// and the sums in every block add to it).
bool gs_step_short(int64_t n) { return n <= kGsShort; }
size_t gs_step_part(int64_t n, int m) { return gs_step_short(n) ? (size_t)kGsChunks * (m + 2) + 2048 : 0; }
cudaError_t launch_gs_step(int64_t n, int k, const double* Vb, int64_t ld, double* d, const double* dinv, double* w,
                           double* part, unsigned* ticket, int* err, int polls, const GsFinish& f, cudaStream_t s) {
  int dev = 0, n_sm = 0, per = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = sizeof(double) * (size_t)k;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_gs_step, 256, smem);
  if (e != cudaSuccess) return e;
  const int64_t xb = std::min<int64_t>(kGsChunks, (n + 255) / 256);
  const int64_t most = std::min<int64_t>((int64_t)n_sm * std::max(1, std::min(per, 4)), 2048);
  const unsigned nb = (unsigned)std::min(most, std::max(xb * ((k + 3) / 4), (n + 31) / 32));
  unsigned* arrived = ticket + 1;
  GsFinish fin = f;
  void* args[] = {&n, &k, &Vb, &ld, &d, &dinv, &w, &part, &ticket, &arrived, &err, &polls, &fin};
  e = cudaLaunchCooperativeKernel(k_gs_step, dim3(nb), dim3(256), args, smem, s);
  note_launch();
  return e == cudaSuccess ? cudaGetLastError() : e;
}
cudaError_t launch_block_apply(int64_t N, const double* Dinv, const double* v, double scale, const double* scale_dev,
                               double* z, float* z32, cudaStream_t s) {
  if (N) {
    const int t = block_threads(N);
    k_block_apply<<<block_count(N, t), t, 0, s>>>(N, Dinv, v, scale, scale_dev, z, z32);
    note_launch();
  }
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_block_invert(int64_t N, const T* D, double* Dinv, int* flag, cudaStream_t s) {
  if (N) { k_block_invert<T><<<nblk(N, 128), 128, 0, s>>>(N, D, Dinv, flag); note_launch(); }
  return cudaGetLastError();
}
template cudaError_t launch_block_invert<double>(int64_t, const double*, double*, int*, cudaStream_t);
template cudaError_t launch_block_invert<float>(int64_t, const float*, double*, int*, cudaStream_t);
cudaError_t launch_make_consistent(const RowArgs& R, double* U, cudaStream_t s) {
  if (R.n_nodes) { k_set_dirichlet<<<nblk(R.n_nodes, 256), 256, 0, s>>>(R.n_nodes, R.faces, R.bc, U); note_launch(); }
  if (R.n_hanging) { k_interp_hanging<<<nblk(R.n_hanging, 256), 256, 0, s>>>(R.n_hanging, R.hnode, R.hpar, R.hnp, U); note_launch(); }
  return cudaGetLastError();
}
cudaError_t launch_vel_pack(int64_t N, int dim, const double* src, double* dst3, cudaStream_t s) {
  if (N) { k_vel_pack<<<nblk(N, 256), 256, 0, s>>>(N, dim, src, dst3); note_launch(); }
  return cudaGetLastError();
}
cudaError_t launch_vel_unpack(int64_t N, int dim, const double* src3, double* dst, cudaStream_t s) {
  if (N) { k_vel_unpack<<<nblk(N, 256), 256, 0, s>>>(N, dim, src3, dst); note_launch(); }
  return cudaGetLastError();
}
