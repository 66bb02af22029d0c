// element_tiles.cu -- the FP32 Jacobian action of the PNP block on node tiles (tiles.h), and
// the row initialisation that goes before the element kernels.  One block per tile: its
// nodes come into shared memory once, threads take their corners' values from there,
// evaluate the Gauss points and put their shares of the element vectors into shared
// memory, and one thread per node and field adds the shares and issues the atomic.
#include <algorithm>
#include <cstdint>

#include "pnp_lane.cuh"
#include "tiles.h"

namespace {

// adds r to node id's rows but the Dirichlet ones (0 there): two atomics, the pair that is
// 8-byte aligned and the third field
__device__ __forceinline__ void add_node(const TileMesh& M, int64_t id, uint8_t face, const float (&r)[3], float w,
                                         float* __restrict__ out) {
  float x[3];
#pragma unroll
  for (int f = 0; f < 3; ++f) x[f] = face & (M.dir >> (8 * f)) & 0x3F ? 0.f : w * r[f];
  float* p = out + 3 * id;
  const int odd = (int)(reinterpret_cast<uintptr_t>(p) >> 2 & 1);
  atomicAdd(reinterpret_cast<float2*>(p + odd), odd ? make_float2(x[1], x[2]) : make_float2(x[0], x[1]));
  atomicAdd(p + 2 - 2 * odd, odd ? x[0] : x[2]);
}
// adds r to the rows of entry u: its node, or a hanging node's parents by their weights
__device__ __forceinline__ void add_entry(const TileMesh& M, const TileView& v, int u, const float (&r)[3],
                                          float* __restrict__ out) {
  const int32_t id = v.id(M.tab, u);
  if (id >= 0) {
    add_node(M, id, v.face(M.tab, u), r, 1.0f, out);
    return;
  }
  const int4 p = v.parents(M.tab, u);
  const uchar4 fm = v.parent_faces(M.tab, u);
  const float w = p.z < 0 ? 0.5f : 0.25f;
  add_node(M, p.x, fm.x, r, w, out);
  add_node(M, p.y, fm.y, r, w, out);
  if (p.z >= 0) {
    add_node(M, p.z, fm.z, r, w, out);
    add_node(M, p.w, fm.w, r, w, out);
  }
}

// ---- FP32 J V ------------------------------------------------------------------------
// The state comes from the 32-byte FP32 node records {c+, c-, phi, h+, h-, v0, v1, v2} of
// the linearisation.  A persistent grid walks the tiles; thread 0 brings the next tile's
// record into the other of two stages by a bulk copy (TMA, cp.async.bulk) that completes on
// the stage's mbarrier, so the mesh tables' latency is off the path; the waits are bounded.
//
// Hexahedra: two threads per element, the one with z-bit z holding the four corners there
// and the four Gauss points next to them.  The z factors of the interpolation and of the
// tests take a shuffle per scalar and corner, the x and y factors run in registers; species,
// (phi, dphi) and (v0, v1) as packed pairs.  Quadrilaterals: a lane per corner (pnp_lane.cuh).
//
// What bounds it: latency, with 16 warps of 118 registers on an SM (IPC 2.3, shared memory
// 66 %).  Uniform level-7 cube (2,097,152 elements) with advection 174 us a launch, 0.25 GB of
// DRAM traffic; from a state stored per Gauss point (64 bytes a lane, 1.1 GB a launch) 262 us.
// Membrane-band octree of 971,776 elements 94 us (115 stored), of 143,872 elements 19 us (24),
// without advection 17 (five blocks fit an SM; 18 with four).  Other layouts, level-7 cube: a
// lane per corner 340 us; tiles of 128 elements (two blocks per SM) 248; slots in the order of
// the entries and nodes' values through registers 187.
struct JvArgs {
  const float4* rec;
  const float* V;
  float* out;
};

// try_wait polls before a wait on a stage gives up (about a second by default; a launch
// argument), and the longer limit of the drain that follows a give-up: the block waits
// for the copies it issued before it exits
constexpr int kWaitPolls = 1 << 22;
constexpr int kDrainPolls = 1 << 24;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// bounded wait for the phase of the given parity to complete; false when it did not
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int polls) {
  const uint32_t a = smem_u32(bar);
  for (int i = 0; i < polls; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
// global -> shared bulk copy of `bytes` (multiple of 16, both addresses 16-byte aligned)
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// value and derivatives of a pair of fields on the way to the Gauss points; z: scaled value
// and reflected derivative of the four corner columns (x + 2 y) at this thread's z
struct ZPair {
  f2 v[4], d[4];
};
// after the y factor, at a row qy: per x
struct YPair {
  f2 v[2], dy[2], dz[2];
};
__device__ __forceinline__ f2 partner(f2 a) { return pair(__shfl_xor_sync(kFull, a.v.x, 1), __shfl_xor_sync(kFull, a.v.y, 1)); }
__device__ __forceinline__ float partner(float a) { return __shfl_xor_sync(kFull, a, 1); }
__device__ __forceinline__ void z_factor(f2 u, f2 rho, f2& v, f2& d) {
  const f2 p = partner(u);
  d = u - p;
  v = fma(rho, p, u);
}
template <typename T>
__device__ __forceinline__ T z_value(T u, T rho) {
  return fma(rho, partner(u), u);
}
__device__ __forceinline__ void y_factor(const ZPair& z, int qy, f2 rho, YPair& o) {
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    o.v[x] = fma(rho, z.v[x + 2 * (1 - qy)], z.v[x + 2 * qy]);
    o.dy[x] = z.v[x + 2] - z.v[x];
    o.dz[x] = fma(rho, z.d[x + 2 * (1 - qy)], z.d[x + 2 * qy]);
  }
}
__device__ __forceinline__ void x_factor(const YPair& y, int qx, f2 rho, f2& v, f2 (&g)[3]) {
  v = fma(rho, y.v[1 - qx], y.v[qx]);
  g[0] = y.v[1] - y.v[0];
  g[1] = fma(rho, y.dy[1 - qx], y.dy[qx]);
  g[2] = fma(rho, y.dz[1 - qx], y.dz[qx]);
}
template <typename T>
__device__ __forceinline__ T xy_value(const T (&z)[4], int qx, int qy, T rho) {
  T a[2];
#pragma unroll
  for (int x = 0; x < 2; ++x) a[x] = fma(rho, z[x + 2 * (1 - qy)], z[x + 2 * qy]);
  return fma(rho, a[1 - qx], a[qx]);
}
// the tests of a row's two Gauss points with the x factors: per corner column x the value
// part (S and the x derivative), and what the y and z derivatives multiply
template <typename T>
__device__ __forceinline__ void test_x(const T (&S)[2], const T (&P)[2][3], T rho, T (&A)[2], T (&Y)[2], T (&Z)[2]) {
  const T px = P[0][0] + P[1][0];
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const T s = fma(rho, S[1 - x], S[x]);
    A[x] = x ? s + px : s - px;
    Y[x] = fma(rho, P[1 - x][1], P[x][1]);
    Z[x] = fma(rho, P[1 - x][2], P[x][2]);
  }
}

// J V at an element's z half: nodal values of the four corners (x + 2 y) of this thread's z
// (nodal arrays as in lane_pnp), to the element vector's entries of these corners without
// the factor lane_weight_c(3) 2^lane_weight_e(3, lev)
template <bool ADV>
__device__ __forceinline__ void half_jv(const float4 (&n0)[4], const float4 (&n1)[4], const float4 (&n2)[4], int zb,
                                        int lev, const LaneParams<float>& K, f2 (&rs)[4], float (&rp)[4]) {
  constexpr int D = 3;
  const float rho = (float)kRho;
  const f2 rho2 = both<float>(rho);
  ZPair zc, zp, zd;  // (c+, c-), (phi, dphi), (dc+, dc-)
  f2 zh[4], zv[4];   // (h+, h-), (v0, v1)
  float zw[4];       // v2
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 a = n0[j], b = n1[j];
    const float d0 = ADV ? n2[j].x : b.y, d1 = ADV ? n2[j].y : b.z, d2 = ADV ? n2[j].z : b.w;
    z_factor(pair(a.x, a.y), rho2, zc.v[j], zc.d[j]);
    z_factor(pair(a.z, d2), rho2, zp.v[j], zp.d[j]);
    z_factor(pair(d0, d1), rho2, zd.v[j], zd.d[j]);
    zh[j] = z_value(pair(a.w, b.x), rho2);
    if constexpr (ADV) {
      zv[j] = z_value(pair(b.y, b.z), rho2);
      zw[j] = z_value(b.w, rho);
    }
  }
  const float beta = const_pow2(kVal, 2 * lev, 0.0f), delta = const_pow2(kVal * kVal, -2 * lev, 0.0f);
  const float tau0 = times_pow2(K.cid, 4 * lev + 4) + K.tau_t;
  const f2 zb2 = pair(-beta, beta), kap2 = both<float>(K.kappa);
  const uint32_t sz = zb ? 0u : 0x80000000u;  // reflection of the z component
  constexpr double alpha = ipow(kVal, D);
  f2 A0[2], Y0[2], Z0[2], A1[2], Y1[2], Z1[2];
  float a0[2], y0[2], z0[2], a1[2], y1[2], z1[2];
#pragma unroll
  for (int qy = 0; qy < 2; ++qy) {
    YPair yc, yp, yd;
    y_factor(zc, qy, rho2, yc);
    y_factor(zp, qy, rho2, yp);
    y_factor(zd, qy, rho2, yd);
    f2 S[2], P[2][3];
    float Sp[2], Pp[2][3];
#pragma unroll
    for (int qx = 0; qx < 2; ++qx) {
      f2 cv, gc[3], pv, gp[3], dcv, dgc[3];
      x_factor(yc, qx, rho2, cv, gc);
      x_factor(yp, qx, rho2, pv, gp);
      x_factor(yd, qx, rho2, dcv, dgc);
      float V[3], tau;
      if constexpr (ADV) {
        const f2 v01 = xy_value(zv, qx, qy, rho2);
        const float v2 = xy_value(zw, qx, qy, rho);
        const float vv = fmaf(v2, v2, fmaf(second(v01), second(v01), first(v01) * first(v01)));
        tau = rsqrtf(fmaf(const_pow2(ipow(kVal, 6), 2 * lev + 2, 0.0f), vv, tau0));
        const f2 V01 = times_const2(v01, ipow(kVal, 2), lev);
        V[0] = first(V01);
        V[1] = second(V01);
        V[2] = reflect(times_const(v2, ipow(kVal, 2), lev), sz);
      } else {
        tau = rsqrtf(tau0);
      }
      f2 sv = fma(kap2, cv, xy_value(zh, qx, qy, rho2));
      f2 dsv = kap2 * dcv;
      f2 gg = both<float>(first(gp[0])) * gc[0], dgg = both<float>(first(gp[0])) * dgc[0];
#pragma unroll
      for (int k = 1; k < 3; ++k) {
        gg = fma(both<float>(first(gp[k])), gc[k], gg);
        dgg = fma(both<float>(first(gp[k])), dgc[k], dgg);
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        dgg = fma(both<float>(second(gp[k])), gc[k], dgg);
        if constexpr (ADV) {
          sv = fma(both<float>(V[k]), gc[k], sv);
          dsv = fma(both<float>(V[k]), dgc[k], dsv);
        }
      }
      const f2 R = fma(zb2, gg, sv), dR = fma(zb2, dgg, dsv), mt = both<float>(-tau);
      const f2 q1 = times_pm(fma(mt, R, cv), alpha), q2 = times_pm(fma(mt, dR, dcv), alpha);
      const f2 p = both<float>(tau * delta) * dR;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        P[qx][k] = fma(q2, both<float>(first(gp[k])), fma(q1, both<float>(second(gp[k])), dgc[k]));
        if constexpr (ADV) P[qx][k] = fma(p, both<float>(V[k]), P[qx][k]);
        Pp[qx][k] = K.e2 * second(gp[k]);
      }
      S[qx] = times_const2(dsv, kVal * kVal, -2 * lev);
      Sp[qx] = times_const(fmaf(tau, first(dR) - second(dR), second(dcv) - first(dcv)), kVal * kVal, -2 * lev);
    }
    if (qy == 0) {
      test_x(S, P, rho2, A0, Y0, Z0);
      test_x(Sp, Pp, rho, a0, y0, z0);
    } else {
      test_x(S, P, rho2, A1, Y1, Z1);
      test_x(Sp, Pp, rho, a1, y1, z1);
    }
  }
  // y factors of the tests, then z: own corners T + Z, the partner's rho T - Z
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const f2 py = Y0[x] + Y1[x];
    const float fy = y0[x] + y1[x];
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      const f2 t = fma(rho2, y ? A0[x] : A1[x], y ? A1[x] : A0[x]);
      const f2 T = y ? t + py : t - py;
      const f2 Z = fma(rho2, y ? Z0[x] : Z1[x], y ? Z1[x] : Z0[x]);
      rs[x + 2 * y] = (T + Z) + partner(fma(rho2, T, f2{make_float2(-Z.v.x, -Z.v.y)}));
      const float tp = fmaf(rho, y ? a0[x] : a1[x], y ? a1[x] : a0[x]);
      const float Tp = y ? tp + fy : tp - fy;
      const float Zp = fmaf(rho, y ? z0[x] : z1[x], y ? z1[x] : z0[x]);
      rp[x + 2 * y] = (Tp + Zp) + partner(fmaf(rho, Tp, -Zp));
    }
  }
}

// shared memory: mbarriers, two records, per slot (c+, c-, phi, h+), with advection
// (h-, v0, v1, v2) and (d0, d1, d2), without (h-, d0, d1, d2), and the corners' shares and a 0
size_t jv_smem_bytes(const TileTab& t, bool adv) {
  return 16 + 2 * (size_t)t.bytes + 16 * ((size_t)(adv ? 3 : 2) * t.slots + t.corners + 1);
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// the nodal values of an entry on their way into its slot: a node's by asynchronous copies
// (no registers, no wait), a hanging node's from its parents
template <bool ADV>
__device__ __forceinline__ void fetch_entry(const TileMesh& M, const JvArgs& A, const TileView& t, int u, float4* n0,
                                            float4* n1, float4* n2) {
  const int32_t id = t.id(M.tab, u);
  const int slot = t.slot(M.tab, u);
  float* d = ADV ? &n2[slot].x : &n1[slot].y;
  if (id >= 0) {
    const float4* rec = A.rec + 2 * (int64_t)id;
    cp_async16(n0 + slot, rec);
    if (ADV) cp_async16(n1 + slot, rec + 1);
    else cp_async4(n1 + slot, rec + 1);
#pragma unroll
    for (int f = 0; f < 3; ++f) cp_async4(d + f, A.V + 3 * (int64_t)id + f);
    return;
  }
  const int4 p4 = t.parents(M.tab, u);
  const bool four = p4.z >= 0;
  const float w = four ? 0.25f : 0.5f;
  // all loads in flight together; two parents: those twice, the second time unused
  const int32_t p[4] = {p4.x, p4.y, four ? p4.z : p4.x, four ? p4.w : p4.y};
  float4 y[4], z[4];
  float g[4][3];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    y[i] = __ldg(A.rec + 2 * (int64_t)p[i]);
    z[i] = __ldg(A.rec + 2 * (int64_t)p[i] + 1);
#pragma unroll
    for (int f = 0; f < 3; ++f) g[i][f] = __ldg(A.V + 3 * (int64_t)p[i] + f);
  }
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
  float x[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (i >= 2 && !four) break;
    a.x += w * y[i].x; a.y += w * y[i].y; a.z += w * y[i].z; a.w += w * y[i].w;
    b.x += w * z[i].x; b.y += w * z[i].y; b.z += w * z[i].z; b.w += w * z[i].w;
#pragma unroll
    for (int f = 0; f < 3; ++f) x[f] += w * g[i][f];
  }
  n0[slot] = a;
  if (ADV) n1[slot] = b;
  else n1[slot].x = b.x;
#pragma unroll
  for (int f = 0; f < 3; ++f) d[f] = x[f];
}

// Per tile: barrier, Gauss points, barrier, sums.  The next tile's record is under way while
// the Gauss points are evaluated, and its nodal values while the sums are made (the slots are
// free then).
template <int D, bool ADV>
__global__ void __launch_bounds__(D == 3 ? 128 : 256, D == 3 && !ADV ? 5 : 4)
    k_jv_tiles(TileMesh M, JvArgs A, LaneParams<float> K, int* err, int polls) {
  constexpr int NC = 1 << D;
  extern __shared__ __align__(128) uint8_t tile_smem[];
  const int tl = blockDim.x, tid = threadIdx.x, nk = M.tab.corners;
  uint64_t* bar = reinterpret_cast<uint64_t*>(tile_smem);
  uint8_t* stage = tile_smem + 16;
  float4* n0 = reinterpret_cast<float4*>(stage + 2 * M.tab.bytes);
  float4 *n1 = n0 + M.tab.slots, *n2 = n1 + (ADV ? M.tab.slots : 0);
  float4* r = n2 + M.tab.slots;
  const int64_t G = gridDim.x;
  auto issue = [&](int64_t tile, int st) {
    mbar_expect_tx(&bar[st], (uint32_t)M.tab.bytes);
    bulk_g2s(stage + st * M.tab.bytes, M.tab.rec + tile * M.tab.bytes, (uint32_t)M.tab.bytes, &bar[st]);
  };
  auto fetch = [&](const TileView& t) {
    for (int u = tid; u < t.cnt; u += tl) fetch_entry<ADV>(M, A, t, u, n0, n1, n2);
  };
  // the copy into stage st of the block's k-th tile did not complete: flag it, let it land
  auto give_up = [&](int k) {
    if (tid == 0) {
      *reinterpret_cast<volatile int*>(err) = 1;  // pinned host memory
      mbar_wait(&bar[k & 1], (uint32_t)(k >> 1) & 1u, kDrainPolls);
    }
  };
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    r[nk] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  if (tid == 0) issue(blockIdx.x, 0);
  if (__syncthreads_or(!mbar_wait(&bar[0], 0, polls))) {
    grid_dependency_wait();
    give_up(0);
    return;
  }
  TileView v = tile_view(stage, M.tab);
  grid_dependency_wait();  // so far only the mesh's tables
  fetch(v);
  for (int k = 0;; ++k) {
    const int64_t tile = blockIdx.x + k * G;
    const bool more = tile + G < M.tab.n;
    cp_async_wait();
    __syncthreads();  // the slots are filled; the other stage is read
    if (tid == 0 && more) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(tile + G, (k + 1) & 1);
    }
    if constexpr (D == 3) {
      const int lev = v.level(M.tab, tid >> 1);
      const ushort4 l4 = *reinterpret_cast<const ushort4*>(v.loc(M.tab) + 4 * tid);
      const int l[4] = {l4.x, l4.y, l4.z, l4.w};
      float4 a[4], b[4], d[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        a[j] = n0[l[j]];
        b[j] = n1[l[j]];
        if (ADV) d[j] = n2[l[j]];
      }
      f2 rs[4];
      float rp[4];
      half_jv<ADV>(a, b, d, tid & 1, lev, K, rs, rp);
      const float p2 = pow2i(lane_weight_e(3, lev), 0.0f);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        r[tile_share(4 * tid + j, NC, nk)] = make_float4(p2 * first(rs[j]), p2 * second(rs[j]), p2 * rp[j], 0.f);
    } else {
      const int u = v.loc(M.tab)[tid], lev = v.level(M.tab, tid / NC), c = tid & (NC - 1);
      const float4 a = n0[u], b = n1[u];
      const float un[3] = {a.x, a.y, a.z}, hn[2] = {a.w, b.x};
      float vn[3] = {0.f, 0.f, 0.f}, dn[3];
      if (ADV) {
        const float4 d = n2[u];
        vn[0] = b.y; vn[1] = b.z; vn[2] = b.w;
        dn[0] = d.x; dn[1] = d.y; dn[2] = d.z;
      } else {
        dn[0] = b.y; dn[1] = b.z; dn[2] = b.w;
      }
      f2 rs;
      float rp;
      lane_pnp<float, D, true, ADV>(un, hn, vn, dn, c, lev, K, rs, rp);
      const float p2 = pow2i(lane_weight_e(D, lev), 0.0f);
      r[tid] = make_float4(p2 * first(rs), p2 * second(rs), p2 * rp, 0.f);
    }
    const bool ok = !more || mbar_wait(&bar[(k + 1) & 1], (uint32_t)((k + 1) >> 1) & 1u, polls);
    if (__syncthreads_or(!ok)) {
      give_up(k + 1);
      return;
    }
    const TileView w = tile_view(stage + ((k + 1) & 1) * M.tab.bytes, M.tab);
    if (more) fetch(w);
    for (int u = tid; u < v.cnt; u += tl) {
      const int e = u + 1 < v.cnt ? (int)v.seg(M.tab)[u + 1] : v.corners;
      float x[3] = {0.f, 0.f, 0.f};
      for (int q = v.seg(M.tab)[u]; q < e; q += 4) {
        float4 y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) y[i] = r[q + i < e ? (int)v.ord(M.tab)[q + i] : nk];
#pragma unroll
        for (int i = 0; i < 4; ++i) { x[0] += y[i].x; x[1] += y[i].y; x[2] += y[i].z; }
      }
#pragma unroll
      for (int f = 0; f < 3; ++f) x[f] = times_const(x[f], lane_weight_c(D), 0);
      add_entry(M, v, u, x, A.out);
    }
    if (!more) return;
    v = w;
  }
}

// ---- rows that the element kernels leave alone, before them --------------------------
// out = 0 on weak-form rows, in - g (mode 0, the residual) or in (mode 1, J V) on Dirichlet
// rows, the constraint in_h - sum_p w_p in_p on hanging rows; with Uk also the history
// hs = (b1 c^k + b2 c^{k-1}) / dt.  One pass and launch in place of a memset, the history
// and a row kernel after the operator.
struct HistoryArgs {
  const double *Uk, *Ukm1;
  double b1, b2, inv_dt;
  double* hs;
};
template <typename T>
__global__ void k_init_rows(RowArgs R, const T* __restrict__ in, T* __restrict__ out, int mode, HistoryArgs H) {
  const int64_t i = row_last_first();
  if (i < R.n_nodes) {
    if (H.hs) {
      H.hs[2 * i + 0] = H.Uk ? (H.b1 * H.Uk[3 * i + 0] + H.b2 * H.Ukm1[3 * i + 0]) * H.inv_dt : 0.0;
      H.hs[2 * i + 1] = H.Uk ? (H.b1 * H.Uk[3 * i + 1] + H.b2 * H.Ukm1[3 * i + 1]) * H.inv_dt : 0.0;
    }
    const uint8_t fm = R.faces[i];
    if (fm & 0x80) return;  // hanging: written by a thread past N
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      const unsigned msk = fm & R.bc.dir_faces[f] & 0x3F;
      T x = T(0);
      if (msk) x = mode == 0 ? T(double(in[3 * i + f]) - R.bc.val[31 - __clz(msk)][f]) : in[3 * i + f];
      out[3 * i + f] = x;
    }
    return;
  }
  const int64_t h = i - R.n_nodes;
  if (h >= R.n_hanging) return;
  const int np = R.hnp[h];
  const T wgt = np == 2 ? T(0.5) : T(0.25);
  const int64_t id = R.hnode[h];
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    T s = in[3 * id + f];
    for (int p = 0; p < np; ++p) s -= wgt * in[3 * (int64_t)R.hpar[4 * h + p] + f];
    out[3 * id + f] = s;
  }
}

// block-Jacobi apply y = Dinv (scale u), and the rows of the J V of y that follows (as
// k_init_rows, mode 1; a hanging node's thread makes its parents' y again)
template <typename T>
__device__ __forceinline__ void apply3(const T (&B)[9], const T* u, T sc, int64_t i, T (&y)[3]) {
  const T a = sc * u[3 * i], b = sc * u[3 * i + 1], c = sc * u[3 * i + 2];
  y[0] = fma(B[0], a, fma(B[1], b, B[2] * c));
  y[1] = fma(B[3], a, fma(B[4], b, B[5] * c));
  y[2] = fma(B[6], a, fma(B[7], b, B[8] * c));
}
template <typename T>
__device__ __forceinline__ void load_block(const T* __restrict__ Dinv, int64_t i, T (&B)[9]) {
#pragma unroll
  for (int q = 0; q < 9; ++q) B[q] = __ldg(Dinv + 9 * i + q);
}
// The blocks and the mesh's tables are older than the launch before; u and the scale are its
// results.  FP64: a dependent launch, in the stream of small GMRES iterations (a 2D time step
// with 3,267 unknowns 14.4 ms without any, 13.4 with the element kernel's, 12.4 with both).
// FP32: not, nor the J V after it: between the nodes of the inner solve's graph dependent
// launches cost more than they hide (17.3 ms a step on 143,872 elements, 17.8 with this one,
// 18.0 with both).
template <typename T>
__global__ void k_block_apply_rows(RowArgs R, const T* __restrict__ Dinv, const T* u, T scale, const T* scale_dev,
                                   T* __restrict__ y, T* __restrict__ out) {
  const int64_t i = row_last_first();
  const int64_t h = i - R.n_nodes;
  const bool node = i < R.n_nodes, hanging = !node && h < R.n_hanging;
  T B[9], v[3];
  uint8_t fm = 0;
  int np = 0;
  int64_t id = i;
  if (node) {
    load_block(Dinv, i, B);
    fm = R.faces[i];
  }
  if (hanging) {
    id = R.hnode[h];
    np = R.hnp[h];
    load_block(Dinv, id, B);
  }
  grid_dependency_wait();
  grid_dependency_release();
  const T sc = scale_dev ? scale_dev[0] : scale;
  if (node) {
    apply3(B, u, sc, i, v);
#pragma unroll
    for (int f = 0; f < 3; ++f) y[3 * i + f] = v[f];
    if (fm & 0x80) return;
#pragma unroll
    for (int f = 0; f < 3; ++f) out[3 * i + f] = (fm & R.bc.dir_faces[f] & 0x3F) ? v[f] : T(0);
  } else if (hanging) {
    const T wgt = np == 2 ? T(0.5) : T(0.25);
    apply3(B, u, sc, id, v);
    for (int p = 0; p < np; ++p) {
      T w[3];
      const int64_t pid = R.hpar[4 * h + p];
      load_block(Dinv, pid, B);
      apply3(B, u, sc, pid, w);
#pragma unroll
      for (int f = 0; f < 3; ++f) v[f] -= wgt * w[f];
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) out[3 * id + f] = v[f];
  }
}

constexpr int kMaxSmem = 200 * 1024;  // a tile of 512 different nodes needs 68 KB
template <int D, bool ADV>
cudaError_t plan_jv(TileTab& t) {
  const size_t smem = jv_smem_bytes(t, ADV);
  if (smem > kMaxSmem) return cudaErrorInvalidConfiguration;
  int dev = 0, n_sm = 0, per = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_jv_tiles<D, ADV>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_jv_tiles<D, ADV>, t.threads, smem);
  if (e != cudaSuccess) return e;
  t.blocks[ADV] = (int)std::min<int64_t>(t.n, (int64_t)n_sm * std::max(1, per));
  return cudaSuccess;
}
template <int D, bool ADV>
cudaError_t launch_jv(const TileMesh& M, const JvArgs& A, const LaneParams<float>& K, bool dependent, int* err,
                      int polls, cudaStream_t s) {
  const cudaError_t e = launch_kernel(dependent, k_jv_tiles<D, ADV>, (unsigned)M.tab.blocks[ADV], M.tab.threads,
                                      jv_smem_bytes(M.tab, ADV), s, M, A, K, err, polls);
  note_launch();
  return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace

cudaError_t plan_jv_tiles(int dim, TileTab& t) {
  const cudaError_t e = dim == 2 ? plan_jv<2, false>(t) : plan_jv<3, false>(t);
  if (e != cudaSuccess) return e;
  return dim == 2 ? plan_jv<2, true>(t) : plan_jv<3, true>(t);
}

cudaError_t launch_jv_tiles(int dim, const TileMesh& M, const float4* rec, bool advection, const float* V,
                            const PhysParams& P, float* out, bool dependent, int* err, int polls, cudaStream_t s) {
  if (polls < 0) polls = kWaitPolls;
  if (M.tab.n == 0) return cudaSuccess;
  const JvArgs A{rec, V, out};
  const LaneParams<float> K = lane_params<float>(P, dim);
  if (dim == 2)
    return advection ? launch_jv<2, true>(M, A, K, dependent, err, polls, s)
                     : launch_jv<2, false>(M, A, K, dependent, err, polls, s);
  return advection ? launch_jv<3, true>(M, A, K, dependent, err, polls, s)
                   : launch_jv<3, false>(M, A, K, dependent, err, polls, s);
}

template <typename T>
cudaError_t launch_init_rows(const RowArgs& R, const T* in, T* out, int mode, cudaStream_t s) {
  const int64_t n = R.n_nodes + R.n_hanging;
  if (n) {
    const int t = block_threads(n);
    k_init_rows<T><<<block_count(n, t), t, 0, s>>>(R, in, out, mode, HistoryArgs{});
    note_launch();
  }
  return cudaGetLastError();
}
template cudaError_t launch_init_rows<double>(const RowArgs&, const double*, double*, int, cudaStream_t);
template cudaError_t launch_init_rows<float>(const RowArgs&, const float*, float*, int, cudaStream_t);

cudaError_t launch_init_residual(const RowArgs& R, const double* U, double* F, const double* Uk, const double* Ukm1,
                                 double b1, double b2, double inv_dt, double* hs, cudaStream_t s) {
  const int64_t n = R.n_nodes + R.n_hanging;
  if (n) {
    const int t = block_threads(n);
    k_init_rows<double><<<block_count(n, t), t, 0, s>>>(R, U, F, 0, HistoryArgs{Uk, Ukm1, b1, b2, inv_dt, hs});
    note_launch();
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_block_apply_rows(const RowArgs& R, const T* Dinv, const T* u, T scale, const T* scale_dev, T* y,
                                    T* out, cudaStream_t s) {
  const int64_t n = R.n_nodes + R.n_hanging;
  if (n) {
    const int t = block_threads(n);
    const cudaError_t e =
        launch_kernel(sizeof(T) == 8, k_block_apply_rows<T>, block_count(n, t), t, 0, s, R, Dinv, u, scale, scale_dev, y,
                      out);
    note_launch();
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}
template cudaError_t launch_block_apply_rows<double>(const RowArgs&, const double*, const double*, double,
                                                     const double*, double*, double*, cudaStream_t);
template cudaError_t launch_block_apply_rows<float>(const RowArgs&, const float*, const float*, float, const float*,
                                                    float*, float*, cudaStream_t);

// floating-point operations per element of the FP32 J V (an FMA counts 2).  Hexahedra, of a
// half with advection: z factors 112, y factors 120, Gauss points 4 x 216, tests x 90, y and z
// 114, weights 12; 24 for the element's corners in the sums.  Without advection 4 x 68 + 24
// fewer a half.  Quadrilaterals: the lane form, less the advection's part when it is zero.
double jv_tiles_flops(int D, bool advection) {
  if (D == 3) return 2 * (advection ? 1312 : 1016) + 24;
  const double v = 2 * D;
  const double adv = D * v + (2 * D - 1) + D + 2 + 2 * (2 * D) + 2 * (2 * D) + 2 * (2 * D);
  return element_kernel_flops(D, true) - (advection ? 0.0 : (1 << D) * adv);
}
