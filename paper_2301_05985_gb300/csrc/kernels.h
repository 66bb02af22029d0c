// kernels.h -- launch interfaces of the library's CUDA kernels.
#pragma once

#include "patches.h"
#include "pnp_internal.h"
#include "tiles.h"

// Arguments of the fused element kernels (residual / Jv / block diagonal).
template <typename T>
struct ElemArgs {
  int64_t n_elem;
  const int32_t* conn;     // [E][2^dim]
  const uint8_t* level;    // [E]
  const int32_t* hang_par; // [H][4]
  const uint8_t* hang_np;  // [H]
  const T* U;              // [N][3]
  const T* V;              // [N][3] direction (Jv only)
  const T* hs;             // [N][2] (beta1 c^k + beta2 c^{k-1}) / dt
  const T* adv;            // [N][3] advection velocity
  T* out;                  // [N][3] accumulated (must be zeroed first)
  PhysParams P;
  // lane kernels on FP64 vectors: the nodes' boundary faces, and the Dirichlet faces of field
  // f in byte f (those rows are not added to)
  const uint8_t* faces = nullptr;
  uint32_t dir = 0;
  // FP32 block diagonal only (may be null): per node {c+, c-, phi, h+, h-, v0, v1, v2}, 32 B
  // aligned, the same values as U, hs and adv in one sector
  const float4* rec = nullptr;
};

// What the tile kernel (element_tiles.cu) needs of the mesh: the node tables and which rows
// are Dirichlet rows.
struct TileMesh {
  TileTab tab;
  uint32_t dir;  // byte f: the faces on which field f is Dirichlet (bit per face)
};

// Arguments of the Dirichlet / hanging row kernels.
struct RowArgs {
  int64_t n_nodes, n_hanging;
  const uint8_t* faces;    // [N] boundary-face bits; bit 7 = hanging
  const int32_t* hnode;
  const int32_t* hpar;
  const uint8_t* hnp;
  BcTable bc;
};

// Launches a kernel; with `dependent` it may start while the one before it on the stream ends
// (programmatic dependent launch): it calls grid_dependency_wait() before it touches anything that launch
// makes or reads, and the other may call grid_dependency_release() when its blocks need no
// more of the chip.
template <typename... P, typename... A>
inline cudaError_t launch_kernel(bool dependent, void (*kernel)(P...), unsigned blocks, int threads, size_t smem,
                                 cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
#ifdef __CUDACC__
// This thread's row of n_nodes nodes and the hanging nodes after them, the last rows first: a
// hanging node's row is a chain of loads through its parents, and in the last blocks it was
// the end of the launch (block apply with rows on 1,047,407 nodes 20.9 us, now 16.9).
__device__ __forceinline__ int64_t row_last_first() {
  return (gridDim.x - 1 - blockIdx.x) * (int64_t)blockDim.x + threadIdx.x;
}
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_release() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif

// Counts every kernel the library launches (read by pnp_kernel_launches).
void note_launch();
// adds n launches (a replayed graph's kernels) and reads the counter
void note_launches(int64_t n);
int64_t launch_count();
// counts a capture of the inner solve (read by pnp_graph_captures)
void note_capture();

// Threads per block for n independent threads: 256, and fewer (down to a warp) while that
// leaves less than two blocks per SM.  A small mesh's kernels otherwise sit on a few SMs: the
// FP64 J V of 1,024 quadrilaterals as 16 blocks of 8 warps shared 16 FP64 pipes (16 clocks
// per warp instruction) and took 14 us, as 128 blocks of one warp 5 us.
inline int block_threads(int64_t n) {
  int t = 256;
  while (t > 32 && (n + t - 1) / t < 304) t /= 2;
  return t;
}
inline unsigned block_count(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Arguments of the shared-memory patch kernels (residual / Jv over Morton patches).
template <typename T>
struct PatchArgs {
  DevPatches pt;
  const uint8_t* level;    // [E]
  const uint8_t* faces;    // [N]
  BcTable bc;
  const T* U;              // [N][3]
  const T* V;              // [N][3] (Jv)
  const T* hs;             // [N][2]
  const T* adv;            // [N][3]
  T* out;                  // [N][3]: every non-hanging row written (no zeroing needed)
  T* partial;              // [n_partials][3]
  PhysParams P;
};
template <typename T>
cudaError_t launch_patch(int dim, bool jv, const PatchArgs<T>& A, cudaStream_t s);

// one thread per element; out zeroed first, Dirichlet and hanging rows left to
// launch_row_fixups
template <typename T>
cudaError_t launch_element(int dim, bool jv, const ElemArgs<T>& A, cudaStream_t s);
// ---- kernels that add to the weak-form rows of `out` only: the rows are initialised first
// (launch_init_rows or a kernel that does the same).
// The residual of FP64 vectors with 2^dim lanes per element (element_lanes.cu), in
// double-float arithmetic (pairs of floats, about 48 bits, on the FP32 pipe) or in FP64
cudaError_t launch_residual_lanes(int dim, bool double_float, const ElemArgs<double>& A, cudaStream_t s);
// J V in FP64, the same lanes
cudaError_t launch_jv64_lanes(int dim, const ElemArgs<double>& A, cudaStream_t s);
// floating-point operations per element (an FMA counts 2) of the residual or J V, counted
// from the formulation that runs (lanes, or one thread per element)
double element_kernel_flops(int dim, bool jv);
// FP32 J V [N][3] on node tiles (element_tiles.cu) at the state of the node records
// (launch_node_records); `advection` false when the advection field is zero.  err[0] = 1
// (mapped pinned memory) when a wait on a staged table gave up after `polls` polls (< 0: the
// default, about a second).  dependent: as launch_kernel; the tables (tab.rec) must be older
// than the launch before, as the kernel reads them before its wait.  plan_jv_tiles: the grids
// for a table (t.blocks), once.
cudaError_t plan_jv_tiles(int dim, TileTab& t);
cudaError_t launch_jv_tiles(int dim, const TileMesh& M, const float4* rec, bool advection, const float* V,
                            const PhysParams& P, float* out, bool dependent, int* err, int polls, cudaStream_t s);
double jv_tiles_flops(int dim, bool advection);
// out = 0 on weak-form rows, in - g (mode 0) or in (mode 1) on Dirichlet rows, the
// constraint of in on hanging rows
template <typename T>
cudaError_t launch_init_rows(const RowArgs& R, const T* in, T* out, int mode, cudaStream_t s);
// the rows of the residual F at U (mode 0) and the history hs = (b1 c^k + b2 c^{k-1}) / dt
// (Uk null: zero)
cudaError_t launch_init_residual(const RowArgs& R, const double* U, double* F, const double* Uk, const double* Ukm1,
                                 double b1, double b2, double inv_dt, double* hs, cudaStream_t s);
// y = Dinv (scale u) per node, scale = scale_dev[0] when given, and the rows of J V of y
// (mode 1) into out
template <typename T>
cudaError_t launch_block_apply_rows(const RowArgs& R, const T* Dinv, const T* u, T scale, const T* scale_dev, T* y,
                                    T* out, cudaStream_t s);
// true when launch_element runs the lane-group kernel (not PNP_ELEMENT_KERNEL=thread)
bool element_kernel_is_lanes();
// true when the FP64 residual runs in double-float arithmetic (lane-group kernel, unless
// PNP_RESIDUAL_ARITH=f64 selects FP64 arithmetic)
bool residual_double_float();
// FP32 operations per FP64 operation of the double-float arithmetic: a quick fused
// multiply-add (2 FP64 flops) costs 18, a quick sum 11, the accurate sums 20, a product 10
constexpr double kDfFlopsPerFlop = 10.0;
// Dout [N][9] += the 3x3 diagonal blocks of the Jacobian (lane-group kernel; Dout zeroed
// first, Dirichlet and hanging rows left to launch_diag_rows)
template <typename T>
cudaError_t launch_block_diag_lanes(int dim, const ElemArgs<T>& A, T* Dout, cudaStream_t s);
double block_diag_flops(int dim);
template <typename T>
cudaError_t launch_row_fixups(const RowArgs& R, const T* in, T* out, int mode, cudaStream_t s);
template <typename T>
cudaError_t launch_diag_rows(const RowArgs& R, T* Dg, cudaStream_t s);

// ------------------------------------------------------------------ vector kernels
// FP64 reductions are deterministic: fixed grid, per-block partials, added in a fixed order.
// The inner FP32 solve's are not: its Gram-Schmidt steps add the blocks' sums with FP64 atomics
// as they arrive.  (A mixed-precision solve depends on the order of atomics on every element
// path: the block diagonal is summed with them.)
constexpr int kRedBlocks = 608;  // 4 x 152 SMs
// blocks at most of the inner FP32 solve's start norm (partials in `part`)
constexpr int kInnerBlocks = 6 * 152;
constexpr int kRedThreads = 256;

// history h_s = (b1 c^k + b2 c^{k-1}) / dt, [N][2]
cudaError_t launch_history(int64_t N, const double* Uk, const double* Ukm1, double b1, double b2, double dt,
                           double* hs, cudaStream_t s);
// y[i] = (float) x[i]
cudaError_t launch_to_f32(int64_t n, const double* x, float* y, cudaStream_t s);
// rec[i] = {U[i][0..2], hs[i][0..1], adv[i][0..2]} in FP32 (two float4 per node)
cudaError_t launch_node_records(int64_t N, const double* U, const double* hs, const double* adv, float4* rec,
                                cudaStream_t s);
cudaError_t launch_to_f64(int64_t n, const float* x, double* y, cudaStream_t s);
// y = a x + b y
cudaError_t launch_axpby(int64_t n, double a, const double* x, double b, double* y, cudaStream_t s);
// z = a x + b y
cudaError_t launch_axpbyz(int64_t n, double a, const double* x, double b, const double* y, double* z, cudaStream_t s);
// result[0] = x . y or ||x||_2 on the device, and in mapped pinned memory at host (may be
// null); part: kRedBlocks doubles; ticket: a zeroed counter of the stream
cudaError_t launch_dot(int64_t n, const double* x, const double* y, double* part, unsigned* ticket, double* result,
                       double* host, cudaStream_t s);
cudaError_t launch_norm2(int64_t n, const double* x, double* part, unsigned* ticket, double* result, double* host,
                         cudaStream_t s);
// w -= sum_i h[i] Vb[i*ld + .], i < k
cudaError_t launch_multi_axpy(int64_t n, int k, const double* Vb, int64_t ld, const double* h, double* w,
                              cudaStream_t s);
// z_i = Dinv_i v_i per node (3x3 blocks) in FP64 and / or as floats z32 (either may be null).
// The factor of v is `scale`, or *scale_dev when that is given.
cudaError_t launch_block_apply(int64_t N, const double* Dinv, const double* v, double scale, const double* scale_dev,
                               double* z, float* z32, cudaStream_t s);
// blocks (= partials per vector) of the multi-dot for vectors of n entries
int multi_dot_blocks(int64_t n);
// d[i] = V_i . w for i < k (part: [k][multi_dot_blocks(n)])
cudaError_t launch_multi_dot(int64_t n, int k, const double* Vb, int64_t ld, const double* w, double* part,
                             unsigned* ticket, double* d, cudaStream_t s);
// What ends a Gram-Schmidt pass: w . w (nrm2) and, where given, its reciprocal (dinv_next)
// and that of its root (inv_s_next) on the device; to mapped pinned memory w . w (host_nrm2) and the k projections of one or
// two passes (host0 <- d0, host1 <- d1).  Null: not written.
struct GsFinish {
  double* nrm2;
  double* dinv_next = nullptr;
  double* inv_s_next = nullptr;
  double* host_nrm2 = nullptr;
  const double* d0 = nullptr;
  double* host0 = nullptr;
  const double* d1 = nullptr;
  double* host1 = nullptr;
};
// w -= sum_i d[i] dinv[i] V_i (i < k), then what `f` says
cudaError_t launch_multi_axpy_norm(int64_t n, int k, const double* Vb, int64_t ld, const double* d, const double* dinv,
                                   double* w, double* part, unsigned* ticket, const GsFinish& f, cudaStream_t s);
// Both in one cooperative launch, for short vectors (gs_step_short): d_i = V_i . w first.
// part: gs_step_part(n, m) doubles for k <= m + 1; ticket[0 .. 1] zeroed counters; err[0] = 1
// (pinned host memory) when its bounded wait gave up after `polls` polls (< 0: the default).
bool gs_step_short(int64_t n);
size_t gs_step_part(int64_t n, int m);
cudaError_t launch_gs_step(int64_t n, int k, const double* Vb, int64_t ld, double* d, const double* dinv, double* w,
                           double* part, unsigned* ticket, int* err, int polls, const GsFinish& f, cudaStream_t s);
// Dinv = inverse of the 3x3 blocks of D (Gauss-Jordan with partial pivoting, FP64);
// flag[0] |= 1 on a singular or non-finite block.  D may alias Dinv when T = double.
template <typename T>
cudaError_t launch_block_invert(int64_t N, const T* D, double* Dinv, int* flag, cudaStream_t s);
// hanging interpolation + Dirichlet values on U
cudaError_t launch_make_consistent(const RowArgs& R, double* U, cudaStream_t s);
// out[j] = sum_b part[b*k + j] for j < k (one block per output, fixed order)
cudaError_t launch_reduce_parts(int nparts, int k, const double* part, double* out, cudaStream_t s);
// out[j] = sum_b part[j*nparts + b]
cudaError_t launch_reduce_cols(int nparts, int k, const double* part, double* out, cudaStream_t s);

// ---------------------------------------------- inner FP32 GMRES (inner_krylov.cu)
// All on FP32 vectors of n entries, n and ld multiples of 4, 16-byte aligned (rows padded
// with zeros); ticket, arrived: zeroed counters of the stream; part: kInnerBlocks doubles;
// sums: inner_sum_doubles() doubles.
int inner_max_depth();
int inner_sum_doubles();
// The Arnoldi bookkeeping stays on the device: norms s_i (sv), 1 / s_i^2 (dinv), 1 / s_i
// (inv_s) and the Hessenberg matrix H [(d+1) x d].  start: s_0 = ||u0||; gs: step j,
// w -= sum_{i <= j} (U_i . w) dinv_i U_i, s_(j+1) = ||w|| and column j of H, in one cooperative
// launch whose bounded wait sets err[0] = 1 (pinned host memory) when it gives up after `polls`
// polls (< 0: the default); lsq: the least squares, coef_i = y_i / s_i.
cudaError_t launch_inner_start(int64_t n, int d, const float* u0, double* part, unsigned* ticket, double* sv,
                               double* dinv, float* inv_s, double* sums, cudaStream_t s);
cudaError_t launch_inner_gs(int64_t n, int j, int d, const float* Ub, int64_t ld, float* w, unsigned* ticket,
                            double* sv, double* dinv, float* inv_s, double* H, double* sums, unsigned* arrived, int* err,
                            int polls, cudaStream_t s);
inline size_t inner_scalar_doubles(int d) { return (size_t)(d + 1) * d; }
cudaError_t launch_inner_lsq(int d, const double* sv, const double* H, double* coef, cudaStream_t s);
// y = Dinv32 (inv_s[0] u) per node (inv_s may be null: scale 1)
cudaError_t launch_block_apply32(int64_t N, const float* Dinv32, const float* u, const float* inv_s, float* y,
                                 cudaStream_t s);
// out = sum_i coef_i U_i (FP32, n and ld multiples of 4); x += sum_i coef_i Z_i (FP32 vectors
// into FP64)
cudaError_t launch_combine_f32(int64_t n, int k, const float* Ub, int64_t ld, const double* coef, float* out,
                               cudaStream_t s);
cudaError_t launch_combine_f32_add_f64(int64_t n, int k, const float* Zb, int64_t ld, const double* coef, double* x,
                                       cudaStream_t s);
// y = scale * x
cudaError_t launch_to_f64_scaled(int64_t n, const float* x, double scale, double* y, cudaStream_t s);
// out[s] = int_face n . (grad c_s + z_s c_s grad phi) dS (s = +, -) over boundary face
// `face` (boundary.cu); part: kRedBlocks x 2 partials; out: 2 device doubles
cudaError_t launch_element_gradient(int dim, int64_t n_elem, const int32_t* conn, const uint8_t* level,
                                    const int32_t* hpar, const uint8_t* hnp, const double* U, double* out,
                                    cudaStream_t s);
cudaError_t launch_boundary_flux(int dim, int64_t n_elem, const int32_t* conn, const uint8_t* level,
                                 const uint8_t* faces, const int32_t* hnode, const int32_t* hpar, const uint8_t* hnp,
                                 const double* U, int face, double* part, double* out, cudaStream_t s);
// out[f] = integral of field f over the plane x_ax = coord 2^-L (boundary.cu); anchor:
// element anchors [E][dim] on the device; part: kRedBlocks x 3 partials
cudaError_t launch_plane_integral(int dim, int L, int64_t n_elem, const int32_t* conn, const uint8_t* level,
                                  const int32_t* anchor, const int32_t* hnode, const int32_t* hpar, const uint8_t* hnp,
                                  const double* U, int ax, int64_t coord, double* part, double* out, cudaStream_t s);
// copy with layout change: [N][dim] <-> [N][3]
cudaError_t launch_vel_pack(int64_t N, int dim, const double* src, double* dst3, cudaStream_t s);
cudaError_t launch_vel_unpack(int64_t N, int dim, const double* src3, double* dst, cudaStream_t s);
