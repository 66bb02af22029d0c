// element_lanes.cu -- element kernels of the VMS PNP block with one lane group per element
// (2^d lanes of a warp share an element, lane c holds corner c and the Gauss point next to
// it) that gather and scatter lane by lane: the residual and the J V of FP64 vectors
// (pnp_lane.cuh) and the block diagonal of the Jacobian.  The FP32 J V runs on node tiles
// (element_tiles.cu).  The FP32 kernels execute no FP64
// instruction (GB300 runs FP64 at 1/64 of the FP32 rate): powers of two come from the
// exponent bits and the parameters arrive converted.
#include <cstdint>
#include <type_traits>

#include "pnp_lane.cuh"

namespace {

// nodal values of NF interleaved fields at node id (hanging: the parents' mean)
template <typename T, int NF>
__device__ __forceinline__ void load_node(const ElemArgs<T>& A, int32_t id, bool valid, const T* __restrict__ src,
                                          int stride, T (&dst)[NF]) {
#pragma unroll
  for (int f = 0; f < NF; ++f) dst[f] = T(0);
  if (!valid) return;
  if (id >= 0) {
#pragma unroll
    for (int f = 0; f < NF; ++f) dst[f] = __ldg(src + (int64_t)stride * id + f);
  } else {
    const int32_t h = -id - 1;
    const int np = A.hang_np[h];
    const T wgt = np == 2 ? T(0.5) : T(0.25);
    for (int p = 0; p < np; ++p) {
      const int32_t pid = A.hang_par[4 * h + p];
#pragma unroll
      for (int f = 0; f < NF; ++f) dst[f] += wgt * __ldg(src + (int64_t)stride * pid + f);
    }
  }
}

// the FP32 state of node id from its 32-byte record (two 16-byte loads; hanging: the
// parents' mean)
template <typename T>
__device__ __forceinline__ void load_record(const ElemArgs<T>& A, int32_t id, bool valid, float (&un)[3],
                                            float (&hn)[2], float (&vn)[3]) {
  float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
  if (valid) {
    if (id >= 0) {
      r0 = __ldg(A.rec + 2 * (int64_t)id);
      r1 = __ldg(A.rec + 2 * (int64_t)id + 1);
    } else {
      const int32_t h = -id - 1;
      const int np = A.hang_np[h];
      const float wgt = np == 2 ? 0.5f : 0.25f;
      for (int p = 0; p < np; ++p) {
        const int64_t pid = A.hang_par[4 * h + p];
        const float4 a = __ldg(A.rec + 2 * pid), b = __ldg(A.rec + 2 * pid + 1);
        r0.x += wgt * a.x; r0.y += wgt * a.y; r0.z += wgt * a.z; r0.w += wgt * a.w;
        r1.x += wgt * b.x; r1.y += wgt * b.y; r1.z += wgt * b.z; r1.w += wgt * b.w;
      }
    }
  }
  un[0] = r0.x; un[1] = r0.y; un[2] = r0.z;
  hn[0] = r0.w; hn[1] = r1.x;
  vn[0] = r1.y; vn[1] = r1.z; vn[2] = r1.w;
}

// U-dependent quantities at this lane's Gauss point: values and gradients of c+-, grad
// phi, the advection v, the history h, tau_c, R_s and P_s = v - z_s grad phi
template <typename T, int D>
__device__ __forceinline__ void lane_state(const T (&un)[3], const T (&vn)[3], const T (&hn)[2], T nb,
                                           const T (&sh)[3], T kappa, T tau0, T G2, T (&cv)[2], T (&gc)[2][3],
                                           T (&gp)[3], T (&v)[3], T (&hq)[2], T& tau, T (&R)[2], T (&P)[2][3]) {
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    interp_vg<T, D>(un[s], nb, sh, cv[s], gc[s]);
    hq[s] = interp_v<T, D>(hn[s], nb);
  }
  interp_g<T, D>(un[2], nb, sh, gp);
  T vv = T(0);
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = T(0);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    v[k] = interp_v<T, D>(vn[k], nb);
    vv = fma(v[k], v[k], vv);
  }
  tau = inv_sqrt(tau0 + G2 * vv);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const T z = s == 0 ? T(1) : T(-1);
    T pg = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      P[s][k] = v[k] - z * gp[k];
      pg = fma(P[s][k], gc[s][k], pg);
    }
    R[s] = fma(kappa, cv[s], hq[s] + pg);
  }
}

// loaded nodal values in the arithmetic type C
template <typename C, int NF>
__device__ __forceinline__ void load_node_c(const ElemArgs<double>& A, int32_t id, bool valid,
                                            const double* __restrict__ src, int stride, C (&dst)[NF]) {
  double x[NF];
  load_node<double, NF>(A, id, valid, src, stride, x);
#pragma unroll
  for (int f = 0; f < NF; ++f) dst[f] = to_compute<C>(x[f]);
}

// The operators on FP64 vectors, arithmetic C (double, or double-float).  They add to the
// weak-form rows only (Dirichlet and hanging rows were written by the row initialisation).
// What bounds it, on the membrane-band octree (971,776 elements) with advection:
//   double-float residual: the FMA pipe (77 % of its cycles; 460 M warp instructions, packed
//   ones two cycles each): 0.56 ms a launch, 1.47 ms with accurate operations throughout and
//   conversions on the FP64 pipe.  (On node tiles as the FP32 J V: no gain, the barriers
//   between its phases cost what the fewer loads and atomics save.)
//   FP64 J V: the FP64 pipe (86 %); uniform level-6 cube 0.76 ms a launch, 1.03 ms with
//   unscaled operators (318 instead of 230 FP64 instructions per lane).
template <typename C, int D, bool JV>
__global__ void __launch_bounds__(256, sizeof(C) == 8 && !std::is_same<C, double>::value ? 4 : 3)
    k_element_lanes(ElemArgs<double> A, LaneParams<C> K) {
  constexpr int NC = 1 << D;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  // warps whose first element is past the end leave together (shuffles need the warp)
  if ((t & ~int64_t(31)) / NC >= A.n_elem) return;
  const int64_t e = t / NC;
  const int c = (int)(t & (NC - 1));
  const bool valid = e < A.n_elem;
  const int32_t id = valid ? __ldg(A.conn + e * NC + c) : 0;
  const int lev = valid ? A.level[e] : 0;
  grid_dependency_wait();  // so far only the mesh's tables
  C un[3], vn[3], hn[2], dn[3];
  load_node_c<C, 3>(A, id, valid, A.U, 3, un);
  load_node_c<C, 3>(A, id, valid, A.adv, 3, vn);
  load_node_c<C, 2>(A, id, valid, A.hs, 2, hn);
  if constexpr (JV) load_node_c<C, 3>(A, id, valid, A.V, 3, dn);
  pair_t<C> rs;
  C rp;
  lane_pnp<C, D, JV, true>(un, hn, vn, dn, c, lev, K, rs, rp);
  if (!valid) return;
  const double w = const_pow2(lane_weight_c(D), lane_weight_e(D, lev), 0.0);
  const double r[3] = {w * to_storage<double>(first(rs)), w * to_storage<double>(second(rs)), w * to_storage<double>(rp)};
  if (id >= 0) {
    const uint32_t fm = A.faces[id] & 0x3Fu;
#pragma unroll
    for (int f = 0; f < 3; ++f)
      if (!(fm & (A.dir >> (8 * f)))) atomicAdd(A.out + 3 * (int64_t)id + f, r[f]);
  } else {
    const int32_t hh = -id - 1;
    const int np = A.hang_np[hh];
    const double wgt = np == 2 ? 0.5 : 0.25;
    for (int p = 0; p < np; ++p) {
      const int32_t pid = A.hang_par[4 * hh + p];
      const uint32_t fm = A.faces[pid] & 0x3Fu;
#pragma unroll
      for (int f = 0; f < 3; ++f)
        if (!(fm & (A.dir >> (8 * f)))) atomicAdd(A.out + 3 * (int64_t)pid + f, wgt * r[f]);
    }
  }
}

// ---- block diagonal of the Jacobian (block-Jacobi preconditioner) ----------------
// D_n = sum over elements, Gauss points and local pairs (i, j) whose constraint targets
// both reach node n of t_i(n) t_j(n) B_ij, B_ij the 3x3 block (test N_i, trial N_j) of
// the linearised element operator and t the constraint weight (1 for a regular node, 1/2
// or 1/4 for a hanging node's parents).  Regular corners only pair with themselves; the
// pairs i != j arise only through hanging corners.  Lane c of an element group holds
// Gauss point c.  A block has seven nonzero entries, stored in this order:
// (+,+) (+,phi) (-,-) (-,phi) (phi,+) (phi,-) (phi,phi).
constexpr int kBlk = 7;
__device__ __forceinline__ int blk_slot(int k) {  // position in the row-major 3x3 block
  return k == 0 ? 0 : k == 1 ? 2 : k == 2 ? 4 : k == 3 ? 5 : k == 4 ? 6 : k == 5 ? 7 : 8;
}

// the seven entries of B_ij at this Gauss point (without the quadrature weight):
// derivatives of the species rows S_s, Phi_s and the Poisson row with respect to the
// trial field N_j, tested with N_i (Def. 3 linearised, as in the J V)
template <typename T>
__device__ __forceinline__ void pair_block(T Ni, const T (&dNi)[3], T Nj, const T (&dNj)[3], T kappa, T e2, T tau,
                                           const T (&cv)[2], const T (&gc)[2][3], const T (&gp)[3], const T (&v)[3],
                                           const T (&R)[2], const T (&P)[2][3], T (&B)[kBlk]) {
  T gij = T(0), gip = T(0), vgj = T(0);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    gij = fma(dNi[k], dNj[k], gij);
    gip = fma(dNi[k], gp[k], gip);
    vgj = fma(v[k], dNj[k], vgj);
  }
  T pp = T(0);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const T z = s == 0 ? T(1) : T(-1);
    T pgj = T(0), giP = T(0), gcj = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      pgj = fma(P[s][k], dNj[k], pgj);
      giP = fma(dNi[k], P[s][k], giP);
      gcj = fma(gc[s][k], dNj[k], gcj);
    }
    const T dRdc = fma(kappa, Nj, pgj);  // d R_s / d c_s
    const T dRdp = -z * gcj;             // d R_s / d phi
    B[2 * s] = Ni * fma(kappa, Nj, vgj) + gij + z * Nj * gip + tau * dRdc * giP;
    B[2 * s + 1] = z * cv[s] * gij + tau * dRdp * giP - tau * R[s] * z * gij;
    B[4 + s] = z * Ni * (tau * dRdc - Nj);
    pp = fma(z * tau, dRdp, pp);
  }
  B[6] = fma(e2, gij, Ni * pp);
}

// constraint targets of a corner: itself, or a hanging node's parents with their weights
template <typename T>
__device__ __forceinline__ int corner_targets(const int32_t* __restrict__ hpar, const uint8_t* __restrict__ hnp,
                                              int32_t id, int32_t (&tg)[4], T& wt) {
  if (id >= 0) {
    tg[0] = id;
    tg[1] = tg[2] = tg[3] = -1;
    wt = T(1);
    return 1;
  }
  const int32_t h = -id - 1;
  const int np = hnp[h];
#pragma unroll
  for (int p = 0; p < 4; ++p) tg[p] = p < np ? hpar[4 * h + p] : -1;
  wt = np == 2 ? T(0.5) : T(0.25);
  return np;
}

template <typename T, int D>
__global__ void __launch_bounds__(256) k_block_diag_lanes(ElemArgs<T> A, LaneParams<T> K, T* __restrict__ Dout) {
  constexpr int NC = 1 << D;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if ((t & ~int64_t(31)) / NC >= A.n_elem) return;
  const int64_t e = t / NC;
  const int c = (int)(t & (NC - 1));
  const int lane = threadIdx.x & 31, gb = lane & ~(NC - 1);
  const bool valid = e < A.n_elem;
  const int32_t id = valid ? __ldg(A.conn + e * NC + c) : 0;
  const int lev = valid ? A.level[e] : 0;
  const T inv_h = pow2i(lev, T(0));
  const T w = pow2i(-D * (lev + 1), T(0));
  const T nb = T(-0.5 * (1.0 - kG));
  T sh[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) sh[k] = ((c >> k) & 1) ? inv_h : -inv_h;
  const T G2 = pow2i(2 * lev + 2, T(0));
  const T tau0 = fma(K.cid * G2, G2, K.tau_t);
  T un[3], vn[3], hn[2];
  bool have = false;
  if constexpr (sizeof(T) == 4) {
    if (A.rec) {
      load_record(A, id, valid, un, hn, vn);
      have = true;
    }
  }
  if (!have) {
    load_node<T, 3>(A, id, valid, A.U, 3, un);
    load_node<T, 3>(A, id, valid, A.adv, 3, vn);
    load_node<T, 2>(A, id, valid, A.hs, 2, hn);
  }
  T cv[2], gc[2][3], gp[3], v[3], hq[2], tau, R[2], P[2][3];
  lane_state<T, D>(un, vn, hn, nb, sh, K.kappa, tau0, G2, cv, gc, gp, v, hq, tau, R, P);

  // diagonal pairs: B_ii at this Gauss point for every corner i, then a reduce-scatter
  // over the group leaves lane c with sum_q B_cc
  T a[NC][kBlk];
#pragma unroll
  for (int i = 0; i < NC; ++i) {
    T Ni, dNi[3];
    shape_at<T, D>(i, c, inv_h, Ni, dNi);
    pair_block<T>(Ni, dNi, Ni, dNi, K.kappa, K.e2, tau, cv, gc, gp, v, R, P, a[i]);
  }
  T b[(NC + 1) / 2][kBlk];
  {
    const bool hi = c & 1;
#pragma unroll
    for (int m = 0; m < NC / 2; ++m)
#pragma unroll
      for (int x = 0; x < kBlk; ++x) {
        const T keep = hi ? a[2 * m + 1][x] : a[2 * m][x];
        const T send = hi ? a[2 * m][x] : a[2 * m + 1][x];
        b[m][x] = keep + flip(send, 0);
      }
  }
  T r[kBlk];
  if constexpr (D == 2) {
    const bool hi = (c >> 1) & 1;
#pragma unroll
    for (int x = 0; x < kBlk; ++x) {
      const T keep = hi ? b[1][x] : b[0][x];
      const T send = hi ? b[0][x] : b[1][x];
      r[x] = keep + flip(send, 1);
    }
  } else {
    T b2[2][kBlk];
    const bool hi1 = (c >> 1) & 1, hi2 = (c >> 2) & 1;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int x = 0; x < kBlk; ++x) {
        const T keep = hi1 ? b[2 * m + 1][x] : b[2 * m][x];
        const T send = hi1 ? b[2 * m][x] : b[2 * m + 1][x];
        b2[m][x] = keep + flip(send, 1);
      }
#pragma unroll
    for (int x = 0; x < kBlk; ++x) {
      const T keep = hi2 ? b2[1][x] : b2[0][x];
      const T send = hi2 ? b2[0][x] : b2[1][x];
      r[x] = keep + flip(send, 2);
    }
  }
  int32_t tg[4] = {-1, -1, -1, -1};
  T wt = T(0);
  const int nt = valid ? corner_targets<T>(A.hang_par, A.hang_np, id, tg, wt) : 0;
  for (int p = 0; p < nt; ++p) {
    const T ww = w * wt * wt;
#pragma unroll
    for (int x = 0; x < kBlk; ++x) atomicAdd(Dout + 9 * (int64_t)tg[p] + blk_slot(x), ww * r[x]);
  }

  // pairs i != j through hanging corners: lane gb + i owns the pair's scatter.  First every
  // lane finds its partners j (bits), then the warp evaluates the pairs that some element of
  // it has.  (With the 56 pairs tested one after another a launch took 169 us on the octree of
  // 143,872 elements, now 118.)
  if (!__any_sync(kFull, valid && id < 0)) return;
  unsigned mine = 0;
#pragma unroll 1
  for (int j = 0; j < NC; ++j) {
    const int32_t id_j = __shfl_sync(kFull, id, gb + j);
    bool share = false;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int32_t tj = __shfl_sync(kFull, tg[q], gb + j);
#pragma unroll
      for (int p = 0; p < 4; ++p) share |= p < nt && tg[p] == tj;
    }
    if (share && j != c && valid && (id < 0 || id_j < 0)) mine |= 1u << j;
  }
#pragma unroll 1
  for (int j = 0; j < NC; ++j) {
    unsigned rows = __ballot_sync(kFull, mine >> j & 1);  // lanes gb + i
#pragma unroll
    for (int o = 16; o >= NC; o >>= 1) rows |= rows >> o;
    rows &= (1u << NC) - 1;
    if (!rows) continue;
    int32_t tj[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) tj[p] = __shfl_sync(kFull, tg[p], gb + j);
    const T wj = __shfl_sync(kFull, wt, gb + j);
    T Nj, dNj[3];
    shape_at<T, D>(j, c, inv_h, Nj, dNj);
#pragma unroll 1
    for (; rows; rows &= rows - 1) {
      const int i = __ffs(rows) - 1;
      T Ni, dNi[3], B[kBlk];
      shape_at<T, D>(i, c, inv_h, Ni, dNi);
      pair_block<T>(Ni, dNi, Nj, dNj, K.kappa, K.e2, tau, cv, gc, gp, v, R, P, B);
#pragma unroll
      for (int k = 0; k < D; ++k)
#pragma unroll
        for (int x = 0; x < kBlk; ++x) B[x] += flip(B[x], k);
      if (c == i && (mine >> j & 1))
        for (int p = 0; p < nt; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (tg[p] == tj[q]) {
              const T ww = w * wt * wj;
#pragma unroll
              for (int x = 0; x < kBlk; ++x) atomicAdd(Dout + 9 * (int64_t)tg[p] + blk_slot(x), ww * B[x]);
            }
    }
  }
}

}  // namespace

template <typename C, bool JV>
static cudaError_t launch_lanes(int dim, const ElemArgs<double>& A, cudaStream_t s) {
  if (A.n_elem == 0) return cudaSuccess;
  const int t = block_threads(A.n_elem << dim);
  const unsigned blocks = block_count(A.n_elem << dim, t);
  const LaneParams<C> K = lane_params<C>(A.P, dim);
  const cudaError_t e = dim == 2 ? launch_kernel(true, k_element_lanes<C, 2, JV>, blocks, t, 0, s, A, K)
                                 : launch_kernel(true, k_element_lanes<C, 3, JV>, blocks, t, 0, s, A, K);
  note_launch();
  return e == cudaSuccess ? cudaGetLastError() : e;
}
cudaError_t launch_residual_lanes(int dim, bool double_float, const ElemArgs<double>& A, cudaStream_t s) {
  return double_float ? launch_lanes<df, false>(dim, A, s) : launch_lanes<double, false>(dim, A, s);
}
cudaError_t launch_jv64_lanes(int dim, const ElemArgs<double>& A, cudaStream_t s) {
  return launch_lanes<double, true>(dim, A, s);
}

template <typename T>
cudaError_t launch_block_diag_lanes(int dim, const ElemArgs<T>& A, T* Dout, cudaStream_t s) {
  if (A.n_elem == 0) return cudaSuccess;
  const int t = block_threads(A.n_elem << dim);
  const unsigned blocks = block_count(A.n_elem << dim, t);
  const LaneParams<T> K = lane_params<T>(A.P, dim);
  if (dim == 2) k_block_diag_lanes<T, 2><<<blocks, t, 0, s>>>(A, K, Dout);
  else k_block_diag_lanes<T, 3><<<blocks, t, 0, s>>>(A, K, Dout);
  note_launch();
  return cudaGetLastError();
}
template cudaError_t launch_block_diag_lanes<double>(int, const ElemArgs<double>&, double*, cudaStream_t);
template cudaError_t launch_block_diag_lanes<float>(int, const ElemArgs<float>&, float*, cudaStream_t);

// per element of the block-diagonal kernel, hanging pairs not counted: per lane the
// state at its Gauss point (as in the residual), per corner the shape function (8) and
// the seven block entries (114), the reduce-scatter (7 adds per stage and entry over
// 2^d - 1 entries in all) and the scaling
double block_diag_flops(int D) {
  const double NC = 1 << D;
  const double tri = D * (D - 1) / 2.0;
  const double vg = 3 * tri + 4 * D, g = vg - 2, v = 3 * D;
  const double state = 2 * vg + 2 * v + g + D * v + 2 * D + 3 + 30;
  return NC * (state + NC * (8 + 114) + 7 * (NC - 1) + 7);
}
