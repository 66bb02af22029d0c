// mlp_train.cu -- loss and gradient of the learned-start network for a batch of rows, in
// three launches:
//   k_mlp_fwd_bwd   forward, loss and backward of 32-row tiles, one tile at a time per CTA;
//   k_mlp_wgrad     the four weight gradients A^T dZ, split over the rows;
//   k_mlp_reduce    the partial sums of both, in a fixed order.
// BF16 operands, FP32 accumulation by mma.sync m16n8k16.  The work is small (1.3 GFLOP for
// 4096 rows, under a microsecond at the tensor cores' rate), so what bounds it is latency:
// launches, chains of dependent tiles, and too few blocks.  4096 rows took 18 launches and
// 2.04 ms when every GEMM was a launch of its own with 64 x 64 tiles and the whole batch as
// one k loop (the weight gradients: 4 to 8 blocks, 0.69 ms each).
#include "mlp_train.h"

#include <algorithm>
#include <mutex>

#include "kernels.h"
#include "pnp.h"

namespace {

using bf16 = __nv_bfloat16;

constexpr int kIn = 216, kInP = 224, kHid = 128, kNo = 3, kNoP = 8;
constexpr int64_t oW1 = 0, ob1 = oW1 + kIn * kHid, oW2 = ob1 + kHid, ob2 = oW2 + kHid * kHid, oW3 = ob2 + kHid,
                  ob3 = oW3 + kHid * kHid, oW4 = ob3 + kHid, ob4 = oW4 + kHid * kNo, kParams = ob4 + kNo;
static_assert(kParams == PNP_MLP_PARAMS, "packed parameter count");

// ---- forward + backward.  A CTA keeps the BF16 weights in shared memory (rows of 136 and
// 232 elements: ldmatrix without bank conflicts) and walks 32-row tiles; 8 warps, each 16
// columns of the 128.  A warp's accumulators of a layer and of the gradient that comes back
// to it have one layout, so GELU' of the pre-activations stays in registers (48 floats per
// thread) between the two passes.  32 rows a tile: 4096 rows are 128 CTAs, one wave.
constexpr int kTile = 32, kFbThreads = 256, kFbCtas = 152;
constexpr int kLdW = kHid + 8, kLdX = kInP + 8, kLdA = kHid + 8, kLdO = 24;
constexpr size_t sW1 = 0, sW2 = sW1 + sizeof(bf16) * kInP * kLdW, sW3 = sW2 + sizeof(bf16) * kHid * kLdW,
                 sW4 = sW3 + sizeof(bf16) * kHid * kLdW, sX = sW4 + sizeof(bf16) * kHid * kNoP,
                 sA = sX + sizeof(bf16) * kTile * kLdX, sO = sA + 3 * sizeof(bf16) * kTile * kLdA,
                 sOut = sO + sizeof(bf16) * kTile * kLdO,
                 kFbSmem = sOut + sizeof(float) * kTile * kNoP;
static_assert(sX % 16 == 0 && sA % 16 == 0 && sO % 16 == 0, "aligned regions");
constexpr int kBias = 3 * kHid + kNo;  // bias-gradient partials per CTA

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool live) {
  const int n = live ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N));
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// GELU x Phi(x) and its derivative (one erf for both)
__device__ __forceinline__ void gelu_both(float z, float& y, float& dy) {
  const float e = 1.f + erff(z * 0.70710678118654752f);
  y = 0.5f * z * e;
  dy = 0.5f * e + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// acc[2][2] = 32 rows of A [32][lda] times 16 columns of B: B from rows [k][n] (T = true,
// n0 the warp's first column) or from rows [n][k]
template <int K, bool T>
__device__ __forceinline__ void warp_gemm(float (&acc)[2][2][4], const bf16* A, int lda, const bf16* B, int ldb, int n0,
                                          int lane) {
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
  const uint32_t a0 = smem_addr(A + (lane & 15) * lda + (lane >> 4) * 8);
  const uint32_t b0 = T ? smem_addr(B + (lane & 15) * ldb + n0 + (lane >> 4) * 8)
                        : smem_addr(B + (n0 + (lane & 7) + (lane >> 4) * 8) * ldb + ((lane >> 3) & 1) * 8);
#pragma unroll
  for (int k = 0; k < K; k += 16) {
    uint32_t a[2][4], b[4];
    ldsm4(a[0], a0 + 2 * k);
    ldsm4(a[1], a0 + 2 * (16 * lda + k));
    if (T) ldsm4_t(b, b0 + 2 * k * ldb);
    else ldsm4(b, b0 + 2 * k);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      mma(acc[i][0], a[i], b[0], b[1]);
      mma(acc[i][1], a[i], b[2], b[3]);
    }
  }
}

__global__ void __launch_bounds__(kFbThreads, 1) k_mlp_fwd_bwd(MlpGradArgs g) {
  extern __shared__ __align__(128) uint8_t sm[];
  bf16* W1 = reinterpret_cast<bf16*>(sm + sW1);
  bf16* W2 = reinterpret_cast<bf16*>(sm + sW2);
  bf16* W3 = reinterpret_cast<bf16*>(sm + sW3);
  bf16* W4 = reinterpret_cast<bf16*>(sm + sW4);
  bf16* X = reinterpret_cast<bf16*>(sm + sX);
  bf16* Ah[3];
#pragma unroll
  for (int l = 0; l < 3; ++l) Ah[l] = reinterpret_cast<bf16*>(sm + sA) + l * kTile * kLdA;
  bf16* dO = reinterpret_cast<bf16*>(sm + sO);
  float* out = reinterpret_cast<float*>(sm + sOut);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  const int n0 = warp * 16;

  // weights: the first layer's in one group, the others behind it
  for (int i = tid; i < kInP * 16; i += kFbThreads)
    cp16(smem_addr(W1 + (i >> 4) * kLdW + (i & 15) * 8), g.W1 + i * 8, true);
  cp_commit();
  for (int i = tid; i < kHid * 16; i += kFbThreads) {
    cp16(smem_addr(W2 + (i >> 4) * kLdW + (i & 15) * 8), g.W2 + i * 8, true);
    cp16(smem_addr(W3 + (i >> 4) * kLdW + (i & 15) * 8), g.W3 + i * 8, true);
  }
  if (tid < kHid) cp16(smem_addr(W4 + tid * kNoP), g.W4 + tid * kNoP, true);
  cp_commit();
  for (int i = tid; i < kTile * kLdO; i += kFbThreads) dO[i] = __float2bfloat16(0.f);

  float db[3][2][2];  // bias-gradient sums of this thread's rows (columns n0 + 8 j + 2 tig + q)
  float db4 = 0.f;
  double loss = 0.0;
#pragma unroll
  for (int l = 0; l < 3; ++l)
#pragma unroll
    for (int j = 0; j < 2; ++j) db[l][j][0] = db[l][j][1] = 0.f;
  const double scale = 2.0 / (3.0 * (double)g.rows);
  bool first = true;
  for (int64_t r0 = (int64_t)blockIdx.x * kTile; r0 < g.rows; r0 += (int64_t)gridDim.x * kTile) {
    const int live = (int)(g.rows - r0 < kTile ? g.rows - r0 : kTile);
    // input rows (BF16, 216 columns padded with zeros to 224)
    if (g.Xf) {
      const bool vec = (reinterpret_cast<uintptr_t>(g.Xf) & 15) == 0;  // rows are 864 bytes
      for (int i = tid; i < kTile * (kInP / 8); i += kFbThreads) {
        const int r = i / (kInP / 8), c = (i % (kInP / 8)) * 8;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (r < live && c < kIn) {
          const float* p = g.Xf + (r0 + r) * kIn + c;
          float x[8];
          if (vec) {
            *reinterpret_cast<float4*>(x) = __ldg(reinterpret_cast<const float4*>(p));
            *reinterpret_cast<float4*>(x + 4) = __ldg(reinterpret_cast<const float4*>(p) + 1);
          } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) x[q] = __ldg(p + q);
          }
          v = make_uint4(pack2(x[0], x[1]), pack2(x[2], x[3]), pack2(x[4], x[5]), pack2(x[6], x[7]));
        }
        *reinterpret_cast<uint4*>(X + r * kLdX + c) = v;
        if (r < live) *reinterpret_cast<uint4*>(g.Xb + (r0 + r) * kInP + c) = v;
      }
    } else {
      for (int i = tid; i < kTile * (kInP / 8); i += kFbThreads) {
        const int r = i / (kInP / 8), c = (i % (kInP / 8)) * 8;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (r < live) v = *reinterpret_cast<const uint4*>(g.Xb + (r0 + r) * kInP + c);
        *reinterpret_cast<uint4*>(X + r * kLdX + c) = v;
      }
    }
    if (first) cp_wait<1>();
    __syncthreads();

    float acc[2][2][4], gp[3][2][2][4];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      if (l == 0) warp_gemm<kInP, true>(acc, X, kLdX, W1, kLdW, n0, lane);
      else warp_gemm<kHid, true>(acc, Ah[l - 1], kLdA, l == 1 ? W2 : W3, kLdW, n0, lane);
      const float* bias = l == 0 ? g.b1 : l == 1 ? g.b2 : g.b3;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int c = n0 + 8 * j + 2 * tig;
        const float bb[2] = {__ldg(bias + c), __ldg(bias + c + 1)};
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int r = 16 * i + gid + 8 * h;
            float y[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) gelu_both(acc[i][j][2 * h + q] + bb[q], y[q], gp[l][i][j][2 * h + q]);
            const uint32_t p = pack2(y[0], y[1]);
            *reinterpret_cast<uint32_t*>(Ah[l] + r * kLdA + c) = p;
            if (r < live) *reinterpret_cast<uint32_t*>(g.A[l] + (r0 + r) * kHid + c) = p;
          }
      }
      if (l == 0 && first) cp_wait<0>();
      __syncthreads();
    }
    first = false;
    // output layer: warps 0 and 1, 16 rows each
    if (warp < 2) {
      float o[4] = {0.f, 0.f, 0.f, 0.f};
      const uint32_t a0 = smem_addr(Ah[2] + (16 * warp + (lane & 15)) * kLdA + (lane >> 4) * 8);
#pragma unroll
      for (int k = 0; k < kHid; k += 32) {
        uint32_t a[4], b[4];
        ldsm4_t(b, smem_addr(W4 + (k + lane) * kNoP));  // 32 rows of k, 8 columns
        ldsm4(a, a0 + 2 * k);
        mma(o, a, b[0], b[1]);
        ldsm4(a, a0 + 2 * (k + 16));
        mma(o, a, b[2], b[3]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int c = 2 * tig + (q & 1);
        out[(16 * warp + gid + 8 * (q >> 1)) * kNoP + c] = o[q] + (c < kNo ? __ldg(g.b4 + c) : 0.f);
      }
    }
    __syncthreads();
    if (tid < kTile) {
      // loss and its gradient at the outputs, one row per thread of warp 0
      double s = 0.0;
      float d[4] = {0.f, 0.f, 0.f, 0.f};
      if (tid < live)
#pragma unroll
        for (int f = 0; f < kNo; ++f) {
          const double e = (double)out[tid * kNoP + f] - (double)__ldg(g.Y + (r0 + tid) * g.ldy + f);
          s += e * e;
          d[f] = (float)(scale * e);
        }
      const uint2 p = make_uint2(pack2(d[0], d[1]), pack2(d[2], 0.f));
      *reinterpret_cast<uint2*>(dO + tid * kLdO) = p;
      if (tid < live) *reinterpret_cast<uint4*>(g.dO + (r0 + tid) * kNoP) = make_uint4(p.x, p.y, 0u, 0u);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      loss += s;
#pragma unroll
      for (int f = 0; f < kNo; ++f) {
        float t = d[f];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (tid == f) db4 += t;
      }
    }
    __syncthreads();
    // backward: dZ_l = (gradient at A_l) GELU'(Z_l), the layer above's dZ in Ah[l]
#pragma unroll
    for (int l = 2; l >= 0; --l) {
      if (l == 2) {
        // dO [32][16] (columns past 2 zero) times W4^T
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          uint32_t a[4];
          ldsm4(a, smem_addr(dO + (16 * i + (lane & 15)) * kLdO + (lane >> 4) * 8));
#pragma unroll
          for (int j = 0; j < 2; ++j) {
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
            mma(acc[i][j], a, *reinterpret_cast<const uint32_t*>(W4 + (n0 + 8 * j + gid) * kNoP + 2 * tig), 0u);
          }
        }
      } else {
        warp_gemm<kHid, false>(acc, Ah[l + 1], kLdA, l == 1 ? W3 : W2, kLdW, n0, lane);
      }
      // dZ_l goes where A_l was: its last reader is behind a barrier
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int c = n0 + 8 * j + 2 * tig;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int r = 16 * i + gid + 8 * h;
            const float z0 = acc[i][j][2 * h] * gp[l][i][j][2 * h], z1 = acc[i][j][2 * h + 1] * gp[l][i][j][2 * h + 1];
            db[l][j][0] += z0;
            db[l][j][1] += z1;
            const uint32_t p = pack2(z0, z1);
            if (l > 0) *reinterpret_cast<uint32_t*>(Ah[l] + r * kLdA + c) = p;
            if (r < live) *reinterpret_cast<uint32_t*>(g.dZ[l] + (r0 + r) * kHid + c) = p;
          }
      }
      __syncthreads();
    }
  }
  // this CTA's bias gradients (sums over the row groups of the warp) and loss
  float* bp = g.part + (int64_t)blockIdx.x * kBias;
#pragma unroll
  for (int l = 0; l < 3; ++l)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float t = db[l][j][q];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (gid == 0) bp[l * kHid + n0 + 8 * j + 2 * tig + q] = t;
      }
  if (tid < kNo) bp[3 * kHid + tid] = db4;
  if (tid == 0) g.loss_part[blockIdx.x] = loss;
}

// ---- weight gradients.  Block (tile, split): a 64 x 64 tile of one layer's A^T dZ over
// the rows of its split, staged 32 rows at a time (cp.async, two stages), 4 warps of 32 x 32;
// both operands lie with the rows as k, so both come through ldmatrix.trans.  The split
// gives 17 tiles enough blocks: about 256 rows each, at most kSplits.
constexpr int kSplits = 32, kWgThreads = 128, kWgRows = 32, kLdT = 72;
constexpr int kWgTiles = 8 + 4 + 4 + 2;
// more rows than this: the splits as one accumulation (1e-5 apart without at 8,192 rows)
constexpr int64_t kThroughRows = 8192;

// THROUGH: a split's accumulators start from the sum of the splits before it, and what it
// adds to that is its partial.  The tensor core truncates its FP32 sums, so a sum over all
// rows that runs through loses up to 1e-4 of itself at 65,536 rows against one in 32 short
// pieces; with the base the gradient is that of one accumulation over the rows, whatever the
// split, as it has been (1.1e-4 apart without, under 1e-6 with it).
template <bool THROUGH>
__global__ void __launch_bounds__(kWgThreads) k_mlp_wgrad(MlpGradArgs g, float* __restrict__ part,
                                                          const float* __restrict__ base) {
  __shared__ __align__(16) bf16 At[2][kWgRows][kLdT], Bt[2][kWgRows][kLdT];
  int t = blockIdx.x;
  const bf16 *A, *B;
  int lda, ldb, m0, n0, m_end, n_end, ldw;
  int64_t off;
  if (t < 8) {
    A = g.Xb; lda = kInP; B = g.dZ[0]; ldb = kHid; off = oW1;
    m0 = 64 * (t >> 1); n0 = 64 * (t & 1); m_end = kIn; n_end = kHid; ldw = kHid;
  } else if (t < 16) {
    const int l = t < 12 ? 1 : 2;
    t &= 3;
    A = g.A[l - 1]; lda = kHid; B = g.dZ[l]; ldb = kHid; off = l == 1 ? oW2 : oW3;
    m0 = 64 * (t >> 1); n0 = 64 * (t & 1); m_end = kHid; n_end = kHid; ldw = kHid;
  } else {
    A = g.A[2]; lda = kHid; B = g.dO; ldb = kNoP; off = oW4;
    m0 = 64 * (t - 16); n0 = 0; m_end = kHid; n_end = kNo; ldw = kNo;
  }
  const int64_t per = ((g.rows + gridDim.y - 1) / gridDim.y + kWgRows - 1) / kWgRows * kWgRows;
  const int64_t k0 = per * blockIdx.y, k1 = k0 + per < g.rows ? k0 + per : g.rows;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  float acc[2][4][4];
  // entry of acc[i][j][q] in the split's parameters, -1 outside
  auto entry = [&](int i, int j, int q) -> int64_t {
    const int m = m0 + wm + 16 * i + gid + 8 * (q >> 1), n = n0 + wn + 8 * j + 2 * tig + (q & 1);
    return m < m_end && n < n_end ? (int64_t)blockIdx.y * kParams + off + m * ldw + n : -1;
  };
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t at = THROUGH ? entry(i, j, q) : -1;
        acc[i][j][q] = at >= 0 ? base[at] : 0.f;
      }
  // 32 rows x 64 columns of each operand; what lies outside is filled with zeros
  auto stage = [&](int64_t k, int st) {
#pragma unroll
    for (int i = tid; i < kWgRows * 8; i += kWgThreads) {
      const int r = i >> 3, c = (i & 7) * 8;
      const bool row = k + r < k1;
      const bool la = row && m0 + c < lda, lb = row && n0 + c < ldb;
      cp16(smem_addr(&At[st][r][c]), la ? A + (k + r) * lda + m0 + c : A, la);
      cp16(smem_addr(&Bt[st][r][c]), lb ? B + (k + r) * ldb + n0 + c : B, lb);
    }
    cp_commit();
  };
  if (k0 < k1) stage(k0, 0);
  int st = 0;
  for (int64_t k = k0; k < k1; k += kWgRows, st ^= 1) {
    if (k + kWgRows < k1) {
      stage(k + kWgRows, st ^ 1);
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
#pragma unroll
    for (int ks = 0; ks < kWgRows; ks += 16) {
      uint32_t a[2][4], b[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i)  // (m lo, k lo) (m hi, k lo) (m lo, k hi) (m hi, k hi)
        ldsm4_t(a[i], smem_addr(&At[st][ks + (lane & 7) + (lane >> 4) * 8][wm + 16 * i + ((lane >> 3) & 1) * 8]));
#pragma unroll
      for (int j = 0; j < 2; ++j)
        ldsm4_t(b[j], smem_addr(&Bt[st][ks + (lane & 15)][wn + 16 * j + (lane >> 4) * 8]));
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma(acc[i][j], a[i], b[j >> 1][2 * (j & 1)], b[j >> 1][2 * (j & 1) + 1]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t at = entry(i, j, q);
        if (at >= 0) part[at] = THROUGH ? acc[i][j][q] - base[at] : acc[i][j][q];
      }
}
// base of a split: the sum of the splits before it
__global__ void __launch_bounds__(256) k_mlp_base(int splits, const float* __restrict__ part, float* __restrict__ base) {
  const int64_t i = blockIdx.x * 256 + threadIdx.x;
  if (i >= kParams) return;
  float s = 0.f;
#pragma unroll 8
  for (int k = 0; k < splits; ++k) {
    base[k * kParams + i] = s;
    s += part[k * kParams + i];
  }
}

// ---- the partials, summed in a fixed order: weights over the splits, biases and the loss
// over the first kernel's CTAs
__global__ void __launch_bounds__(256) k_mlp_reduce(int64_t rows, int splits, int ctas, const float* __restrict__ wpart,
                                                    const float* __restrict__ bpart,
                                                    const double* __restrict__ loss_part, float* __restrict__ grad,
                                                    double* __restrict__ loss) {
  const int64_t i = blockIdx.x * 256 + threadIdx.x;
  if (i == 0) {
    double s = 0.0;
    for (int b = 0; b < ctas; ++b) s += loss_part[b];
    *loss = s / (3.0 * (double)rows);
  }
  if (i >= kParams) return;
  int b = -1;  // bias column
  if (i >= ob1 && i < oW2) b = (int)(i - ob1);
  else if (i >= ob2 && i < oW3) b = kHid + (int)(i - ob2);
  else if (i >= ob3 && i < oW4) b = 2 * kHid + (int)(i - ob3);
  else if (i >= ob4) b = 3 * kHid + (int)(i - ob4);
  const float* p = b < 0 ? wpart + i : bpart + b;
  const int64_t ld = b < 0 ? kParams : kBias;
  const int n = b < 0 ? splits : ctas;
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
  int k = 0;
  for (; k + 4 <= n; k += 4) {
    s0 += p[k * ld];
    s1 += p[(k + 1) * ld];
    s2 += p[(k + 2) * ld];
    s3 += p[(k + 3) * ld];
  }
  for (; k < n; ++k) s0 += p[k * ld];
  grad[i] = (s0 + s1) + (s2 + s3);
}

}  // namespace

size_t mlp_grad_part_floats() { return (size_t)kFbCtas * kBias + 2 * (size_t)kSplits * kParams; }
int mlp_grad_max_ctas() { return kFbCtas; }

cudaError_t launch_mlp_grad(const MlpGradArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaErrorInvalidValue;
  // the shared-memory attribute is a per-device setting; only a success is remembered
  static std::mutex mu;
  static bool ready[128] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 128) return cudaErrorInvalidDevice;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!ready[dev]) {
      e = cudaFuncSetAttribute(k_mlp_fwd_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFbSmem);
      if (e != cudaSuccess) return e;
      ready[dev] = true;
    }
  }
  const int ctas = (int)std::min<int64_t>(kFbCtas, (a.rows + kTile - 1) / kTile);
  const int splits = (int)std::min<int64_t>(kSplits, std::max<int64_t>(1, a.rows / 256));
  float* wpart = a.part + (size_t)kFbCtas * kBias;
  k_mlp_fwd_bwd<<<ctas, kFbThreads, kFbSmem, s>>>(a);
  k_mlp_wgrad<false><<<dim3(kWgTiles, splits), kWgThreads, 0, s>>>(a, wpart, nullptr);
  if (a.rows > kThroughRows) {
    float* base = wpart + (size_t)kSplits * kParams;
    k_mlp_base<<<(unsigned)((kParams + 255) / 256), 256, 0, s>>>(splits, wpart, base);
    k_mlp_wgrad<true><<<dim3(kWgTiles, splits), kWgThreads, 0, s>>>(a, wpart, base);
    note_launches(2);
  }
  k_mlp_reduce<<<(unsigned)((kParams + 255) / 256), 256, 0, s>>>(a.rows, splits, ctas, wpart, a.part, a.loss_part,
                                                                 a.grad, a.loss);
  note_launches(3);
  return cudaGetLastError();
}
