// Eulerian solves of the coupled loop (Sect. 3.2), FP64 throughout.  The per-node and
// per-element arithmetic lives in eulerian_ops.h; these kernels map threads onto it and
// carry the reductions.
//
// * The local right-hand side of the elliptic relaxation and its length scale (Eqs. 12-18),
//   one thread per node.  H_ijkl of Eq. 13 is applied in contracted form:
//       H_ijkl G_kl = (C2 A_v + g5/3) G_ij - (g5/3) G_ji + g5 (b G)_ij - g5 (b G^T)_ij
//   with G_kl = d<U_k>/dx_l (zero for l = z).
// * Galerkin matrices of linear triangles in CSR.  Fixed matrices (consistent mass,
//   laplacian stiffness) come from the host.  The elliptic-relaxation matrix M + L_e^2 K
//   changes with L every call, so each CSR entry sums its element contributions in
//   ascending element order.
// * Conjugate gradients with the Jacobi preconditioner for C right-hand sides at once
//   (vectors [C][nn]), with per-component Dirichlet masks.  Every reduction is two-stage:
//   block partials, then one block per component summing them in a fixed order.  Results
//   therefore repeat bit for bit.
// * The pressure projection's source (Eq. 33), the increment's normal derivative (Eq. 61),
//   node-transferred gradients (Sect. 3.4) and the Galerkin load.
#include "pdfx_device.cuh"
#include "pdfx_internal.h"

namespace pdfx {
namespace {

constexpr int kEB = 256;   // threads per block
constexpr int kRowChunk = 8;   // CSR entries whose loads a row issues together

unsigned blocks_for(int64_t n) { return static_cast<unsigned>((n + kEB - 1) / kEB); }

// Sum of v over the block's threads (kEB threads); the result is valid in thread 0.
__device__ double block_sum(double v, double* sh) {
  const int t = threadIdx.x;
  sh[t] = v;
  __syncthreads();
  for (int w = kEB / 2; w > 0; w >>= 1) {
    if (t < w) sh[t] += sh[t + w];
    __syncthreads();
  }
  const double r = sh[0];
  __syncthreads();
  return r;
}

template <typename T>
__global__ void wp_rhs_kernel(const T* __restrict__ f, int nn, WpConst k, double* __restrict__ rhs,
                              double* __restrict__ L, int* __restrict__ err) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  if (!eops::wp_rhs_node(f + static_cast<size_t>(n) * kNF, k, rhs + n, static_cast<size_t>(nn), L + n))
    atomicExch(err, 1);
}

// The fields' wp_ij (slots 14-22) as the initial guess x[9][nn].
template <typename T>
__global__ void read_wp_kernel(int nn, const T* __restrict__ f, double* __restrict__ x) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  for (int c = 0; c < 9; ++c) x[static_cast<size_t>(c) * nn + n] = f[static_cast<size_t>(n) * kNF + 14 + c];
}

// Dirichlet conditions of the nine components (Eq. 59 at no-slip nodes, zero off-diagonal
// components at free-slip nodes) written into x[9][nn], which holds the initial guess.
template <typename T>
__global__ void wp_bc_kernel(const T* __restrict__ f, int nn, WpConst k, const int8_t* __restrict__ ncls,
                             const double* __restrict__ nrm, uint8_t* __restrict__ fixed,
                             double* __restrict__ x, int* __restrict__ err) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  if (!eops::wp_bc_node(f + static_cast<size_t>(n) * kNF, k, ncls[n], nrm[2 * n], nrm[2 * n + 1], fixed + n,
                        x + n, static_cast<size_t>(nn)))
    atomicExch(err, 1);
}

__global__ void assemble_wp_kernel(int nnz, const int32_t* __restrict__ cptr, const int32_t* __restrict__ clist,
                                   const double* __restrict__ fe, const int32_t* __restrict__ tri,
                                   const double* __restrict__ L, double* __restrict__ aval) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nnz) return;
  aval[i] = eops::wp_entry(cptr[i], cptr[i + 1], clist, fe, tri, L);
}

// y[c][n] = sum_k val[k] x[c][col[k]] over row n, for C components.
__global__ void spmv_kernel(int nn, int C, const int32_t* __restrict__ row, const int32_t* __restrict__ col,
                            const double* __restrict__ val, const double* __restrict__ x,
                            double* __restrict__ y) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= static_cast<int64_t>(nn) * C) return;
  const int c = static_cast<int>(i / nn), n = static_cast<int>(i % nn);
  y[i] = eops::csr_row(n, row, col, val, x + static_cast<size_t>(c) * nn);
}

// Scalars of component c: sc[c * kSc + .].
constexpr int kSc = kPcgScalars;
using eops::S_ALPHA;

// Sums over nodes of the block's slice: grid (nblk, C); part[(c * nblk + blk) * 2 + m].
// mode 0: zb = free ? (b - q) / diag : 0, sums zb^2 (the reduced load's norm)
// mode 1: r = free ? b - q : 0, z = r / diag, d = z, sums r z and z z (initial residual)
// mode 2: q = free ? q : 0, sums d q
// mode 3: x += alpha d, r -= alpha q, z = free ? r / diag : 0, sums r z and z z
__global__ void pcg_pass_kernel(int mode, int nn, const uint8_t* __restrict__ fixed, const double* __restrict__ diag,
                                const double* __restrict__ b, double* __restrict__ x, double* __restrict__ r,
                                double* __restrict__ z, double* __restrict__ d, double* __restrict__ q,
                                const double* __restrict__ sc, double* __restrict__ part) {
  __shared__ double sh[kEB];
  const int c = blockIdx.y, nblk = gridDim.x;
  const size_t base = static_cast<size_t>(c) * nn;
  const double alpha = sc[c * kSc + S_ALPHA];
  double s0 = 0.0, s1 = 0.0;
  for (int n = blockIdx.x * kEB + threadIdx.x; n < nn; n += nblk * kEB) {
    const size_t o = base + n;
    const bool fr = !fixed || !fixed[o];
    eops::pcg_node(mode, fr, diag[n], alpha, b + o, x + o, r + o, z + o, d + o, q + o, &s0, &s1);
  }
  const double t0 = block_sum(s0, sh);
  const double t1 = block_sum(s1, sh);
  if (threadIdx.x == 0) {
    part[(static_cast<size_t>(c) * nblk + blockIdx.x) * 2] = t0;
    part[(static_cast<size_t>(c) * nblk + blockIdx.x) * 2 + 1] = t1;
  }
}

// One block per component: the partial sums in block order, then the scalars.
// step 0: bnorm; step 1: rz, zz, active, iters = 0; step 2: alpha; step 3: beta, rz, zz,
// iters, active.
__global__ void pcg_scalar_kernel(int step, int nblk, const double* __restrict__ part, double tol,
                                  double* __restrict__ sc) {
  __shared__ double sh[kEB];
  const int c = blockIdx.x;
  double a0 = 0.0, a1 = 0.0;
  for (int j = threadIdx.x; j < nblk; j += kEB) {
    a0 += part[(static_cast<size_t>(c) * nblk + j) * 2];
    a1 += part[(static_cast<size_t>(c) * nblk + j) * 2 + 1];
  }
  const double t0 = block_sum(a0, sh);
  const double t1 = block_sum(a1, sh);
  if (threadIdx.x == 0) eops::pcg_scalars(step, t0, t1, tol, sc + c * kSc);
}

// d = free ? z + beta d : 0 for the components still iterating.
__global__ void pcg_direction_kernel(int nn, int C, const uint8_t* __restrict__ fixed, const double* __restrict__ z,
                                     double* __restrict__ d, const double* __restrict__ sc) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= static_cast<int64_t>(nn) * C) return;
  const int c = static_cast<int>(i / nn);
  eops::pcg_direction(!fixed || !fixed[i], sc + c * kSc, z[i], d + i);
}

// ---------------------------------------------------------------------------------------
// The conjugate-gradient iterations of a solve in one launch.  The grids here hold 1e3 to
// 1e5 nodes, so an iteration is a chain of latencies (two sums over all nodes, each needed by
// every block before the next pass) on a narrow FP64 pipe (a warp instruction holds its
// scheduler's for 64 cycles), not a stream of bytes: as two kernels per iteration, each
// finished by its last block to arrive, it took about 20 us at 1,104 nodes and 23 us at
// 25,200.
//
// * A block owns K items, each 256 / P nodes of one component, a node per thread, and keeps
//   their rows and vectors in shared memory for the whole solve:
//     direction pass: d1 = z + beta d0, q = A d1, sums d1 q; a row forms the new direction
//       at its neighbours itself, so that d alternates between two buffers;
//     update pass: x += alpha d1, r -= alpha q, z = r / diag, sums r z and z z.
// * The sums keep the order of the setup's two-stage sums (slices of 256 nodes, a halving
//   tree in a slice, then one over the slices), so a solve has the bits and the iteration
//   count of separate passes.  An item is a slice (P = 1) or, where there are
//   multiprocessors for twice as many, the even or the odd nodes of one (P = 2: the tree's
//   last level joins the two), so that each scheduler has one warp.
// * CLUSTER, where a component fits one cluster of 16 blocks: a cluster per component, no
//   traffic beyond it.  Neighbours' z and d are read from, and item sums pushed to, the
//   other blocks' shared memory, with a hardware cluster barrier per pass.
// * Otherwise a cooperative launch: z and d in global memory, item sums in slots (three sets,
//   since blocks read a pass's sums after they have arrived: eops::pcg_sum_slot), one arrival
//   counter for all blocks.  (A counter costs 2,900 cycles at any block count;
//   polling every block's slot instead 2,600 at 5 blocks but 7,600 at 99, since writers and
//   pollers share the slots' lines.)  The wait is bounded: a block that gives up leaves its
//   mark in the scalars and returns, and so do the others, whose own waits then run out.
// ---------------------------------------------------------------------------------------
constexpr int kMaxSystems = 9;
constexpr int kClusterBlocks = 16;
constexpr int kPollLimit = 1 << 22;   // a second or more
constexpr int S_FAILED = kPcgScalars - 1;   // unused by the arithmetic; component 0: a wait ran out
static_assert(eops::S_ITERS < S_FAILED, "scalar slots");
static_assert(kRedBlocks <= 256, "a lane holds at most eight slices");

struct SolveArgs {
  int nn, C, nvb, limit, K;   // nvb slices of 256 nodes, K items per block
  const int32_t* row;
  const int32_t* col;
  const double* val;
  const uint8_t* fixed;
  const double* diag;
  double *x, *r, *z, *q, *d0, *d1;
  double tol;
  double* sc;
  double* slots;         // [kPcgSumSets][C][nvb P] item sums (eops::pcg_sum_slot)
  unsigned* arrived;     // blocks that have published, over all passes (zero at the start)
};

// The halving tree over a[m] of lane l at place l + 32 m, m < M (the rest zero): the levels
// above 32 in the lane, the others across lanes.
__device__ __forceinline__ double tree256(const double (&a)[8], int M) {
  double v = a[0];
  if (M > 4) v = ((a[0] + a[4]) + (a[2] + a[6])) + ((a[1] + a[5]) + (a[3] + a[7]));
  else if (M > 2) v = (a[0] + a[2]) + (a[1] + a[3]);
  else if (M > 1) v = a[0] + a[1];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Orders what this thread has written, read or seen through a barrier before its later
// accesses, for the whole GPU.
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(r) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
  return r;
}
__device__ __forceinline__ double cluster_load(uint32_t addr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_store(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// r / d from y = 1 / d rounded to nearest: Markstein's correction (1990) applied twice, each
// step an exact remainder by fused multiply-add; the first makes the quotient faithful, the
// second correctly rounded, so the bits are the division's in half its FP64 operations.
// Magnitudes far from the ends of the range only (ok: |d| is); else the division itself.
__device__ __forceinline__ bool mid_range(double v) {
  const int e = (__double2hiint(v) >> 20) & 0x7ff;
  return e > 600 && e < 1450;
}
__device__ __forceinline__ double divide(double r, double d, double y, bool ok) {
  if (!(ok && mid_range(r))) return r / d;
  double q = r * y;
  q = fma(fma(-q, d, r), y, q);
  return fma(fma(-q, d, r), y, q);
}

// The cooperative launch's exchange: the block's vectors and sums, complete at its barrier,
// become visible with its arrival; the warps that go on to read the sums (reads) wait for
// every block's.  False for a lane whose wait ran out.
__device__ __forceinline__ bool grid_exchange(const SolveArgs& a, unsigned target, bool reads) {
  __syncthreads();
  if (threadIdx.x == 0) {
    fence_gpu();
    atomicAdd(a.arrived, 1u);
  }
  bool ok = true;
  if (reads) {
    if ((threadIdx.x & 31) == 0) {
      int tries = 0;
      unsigned v;
      do {
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.arrived) : "memory");
      } while (v < target && ++tries < kPollLimit);
      ok = v >= target;
      fence_gpu();
    }
    __syncwarp();
  }
  return ok;
}

// Totals of a pass's item sums and the scalars from them (eops::pcg_scalars steps 2 and 3,
// its two sums apart), one component and sum per warp; every block forms them all.  sums: the
// cluster's sums of the pass, [which][item], or the slots.
template <int P, int W, bool CLUSTER>
__device__ __forceinline__ void solve_totals(const SolveArgs& a, int pass, int c0, int c1, const double* sums,
                                             double* ssc, const int* on, int* on_next) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int per = a.nvb * P, M = (a.nvb + 31) >> 5;
  constexpr int V = P == 1 ? 8 : 1;   // P = 2: few slices, one per lane
  static_assert(P == 1 || kClusterBlocks / P <= 32, "a cluster's slices by lane");
  const int tasks = (c1 - c0) * (pass + 1);
  double v[V][P];
  auto fetch = [&](int t) {
    const int c = c0 + (pass ? t >> 1 : t), which = pass ? t & 1 : 0;
    const double* src = sums + (CLUSTER ? static_cast<size_t>(which) * kRedBlocks
                                        : eops::pcg_sum_slot(pass, which, a.C, per, c, 0));
#pragma unroll
    for (int m = 0; m < V; ++m) {
      const int vb = lane + 32 * m;
#pragma unroll
      for (int j = 0; j < P; ++j)
        v[m][j] = vb < a.nvb ? (CLUSTER ? src[vb * P + j] : __ldcg(src + vb * P + j)) : 0.0;
    }
  };
  if (warp < tasks) fetch(warp);
  for (int t = warp; t < tasks; t += W) {
    const int c = c0 + (pass ? t >> 1 : t), which = pass ? t & 1 : 0;
    double w[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) w[m] = m < V ? (P == 2 ? v[m % V][0] + v[m % V][P - 1] : v[m % V][0]) : 0.0;
    if (t + W < tasks) fetch(t + W);   // the next sum's slots are read under this one's tree
    if (!on[c]) continue;
    const double total = tree256(w, P == 2 ? 1 : M);
    double* s = ssc + c * kSc;
    if (lane == 0) {
      if (!pass) {
        s[S_ALPHA] = s[eops::S_RZ] / total;
      } else if (which == 0) {
        s[eops::S_BETA] = total / s[eops::S_RZ];
        s[eops::S_RZ] = total;
        s[eops::S_ITERS] += 1.0;
      } else {
        s[eops::S_ZZ] = total;
        on_next[c] = sqrt(total) > a.tol * s[eops::S_BNORM];
      }
    }
  }
}

// Scalars of components [c0, c1) back to global memory (by one block).
__device__ __forceinline__ void solve_store_scalars(const SolveArgs& a, int c0, int c1, const double* ssc,
                                                    const int* on0, const int* on1) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int i = c0 * kSc + tid; i < c1 * kSc; i += nt)
    if (i % kSc != eops::S_ACTIVE && i % kSc != eops::S_BETA && i != S_FAILED) a.sc[i] = ssc[i];
  for (int c = c0 + tid; c < c1; c += nt) {
    const bool on = on0[c] && on1[c];
    a.sc[c * kSc + eops::S_ACTIVE] = on ? 1.0 : 0.0;
    a.sc[c * kSc + eops::S_BETA] = on ? ssc[c * kSc + eops::S_BETA] : 0.0;
  }
}

// One item's rows and vectors in shared memory.  (The waits' fences empty the L1, so reads
// through it would come from the L2 in every pass.)  Rows of up to kSolveRow entries; a
// longer row is read from global memory.  nb: the neighbours' nodes, or (CLUSTER) the
// addresses of their z in the cluster.
constexpr int kSolveRow = 9;   // the longest row of these grids (a node of eight neighbours)
template <int NT>
struct SolveRows {
  double val[kSolveRow][NT];
  uint32_t nb[kSolveRow][NT];
  double diag[NT], inv[NT];
  int32_t len[NT];
  int most;                 // the longest of the rows
};
template <int NT>
struct SolveItem {
  double z[NT], d[2][NT];   // d: the direction, and (CLUSTER) the previous one
  double x[NT], r[NT], q[NT];
  double sums[2][NT];
  uint8_t fr[NT];           // the node is free for this component
};

template <int P, bool CLUSTER>
__global__ void __launch_bounds__(kEB / P) pcg_solve_kernel(SolveArgs a) {
  constexpr int NT = kEB / P, W = NT / 32;
  extern __shared__ __align__(16) unsigned char solve_smem[];
  __shared__ double ssc[kMaxSystems * kSc];
  __shared__ int act[2][kMaxSystems];   // components still iterating, this pass and the next
  __shared__ double csum[3][CLUSTER ? kRedBlocks : 1];   // CLUSTER: item sums of a pass (d q; r z, z z)
  __shared__ int failed;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int per = a.nvb * P;            // items of a component
  // CLUSTER: block `rank` of a component's cluster holds the component's items from rank K.
  // Otherwise the blocks take K consecutive items each in slice-major order.
  const int rank = static_cast<int>(blockIdx.x) % kClusterBlocks;
  const int c0 = CLUSTER ? static_cast<int>(blockIdx.x) / kClusterBlocks : 0, c1 = CLUSTER ? c0 + 1 : a.C;
  const int b0 = (CLUSTER ? rank : static_cast<int>(blockIdx.x)) * a.K;
  const int nb = max(0, min(a.K, (CLUSTER ? per : a.C * per) - b0));
  auto comp_of = [&](int k) { return CLUSTER ? c0 : (b0 + k) % a.C; };
  auto part_of = [&](int k) { return CLUSTER ? b0 + k : (b0 + k) / a.C; };
  auto node_of = [&](int part) { return (part / P) * kEB + part % P + P * tid; };
  const int part0 = part_of(0);
  const int nrows = nb > 0 ? part_of(nb - 1) - part0 + 1 : 0;
  SolveItem<NT>* const item = reinterpret_cast<SolveItem<NT>*>(solve_smem);
  SolveRows<NT>* const rows = reinterpret_cast<SolveRows<NT>*>(solve_smem + sizeof(SolveItem<NT>) * a.K);
  // CLUSTER: address of node n's z in the block that holds it
  auto node_addr = [&](int n) -> uint32_t {
    const int part = (n / kEB) * P + n % P, at = (n % kEB) / P;
    return cluster_addr(&item[part % a.K].z[at], static_cast<uint32_t>(part / a.K));
  };
  constexpr uint32_t kDirAt = offsetof(SolveItem<NT>, d);   // of d[0] behind z (z comes first)

  for (int i = tid; i < a.C * kSc; i += NT) ssc[i] = a.sc[i];
  if (tid < a.C) act[0][tid] = act[1][tid] = a.sc[tid * kSc + eops::S_ACTIVE] != 0.0;
  if (tid == 0) failed = 0;
  if (CLUSTER)
    for (int i = tid; i < 3 * kRedBlocks; i += NT) csum[i / kRedBlocks][i % kRedBlocks] = 0.0;
  if (tid < nrows) rows[tid].most = 0;
  __syncthreads();
  for (int k = 0; k < nrows; ++k) {
    SolveRows<NT>& R = rows[k];
    const int n = node_of(part0 + k);
    const bool in = n < a.nn;
    const int r0 = in ? a.row[n] : 0, len = in ? a.row[n + 1] - r0 : 0;
    R.len[tid] = len;
    atomicMax(&R.most, len);
    for (int u = 0; u < kSolveRow; ++u) {
      const int m = u < len ? a.col[r0 + u] : (in ? n : 0);
      R.nb[u][tid] = CLUSTER ? node_addr(m) : static_cast<uint32_t>(m);
      R.val[u][tid] = u < len ? a.val[r0 + u] : 0.0;
    }
    R.diag[tid] = in ? a.diag[n] : 1.0;
    R.inv[tid] = 1.0 / R.diag[tid];
  }
  for (int k = 0; k < nb; ++k) {
    SolveItem<NT>& S = item[k];
    const int n = node_of(part_of(k));
    const size_t o = static_cast<size_t>(comp_of(k)) * a.nn + n;
    const bool in = n < a.nn;
    S.x[tid] = in ? a.x[o] : 0.0;
    S.r[tid] = in ? a.r[o] : 0.0;
    S.z[tid] = in ? a.z[o] : 0.0;
    S.d[0][tid] = in ? a.d0[o] : 0.0;
    S.fr[tid] = in && (!a.fixed || !a.fixed[o]);
  }
  if (CLUSTER) cluster_barrier();
  else __syncthreads();

  unsigned target = 0;
  int it = 0;
  for (; it < a.limit; ++it) {
    const int cur = it & 1;
    bool any = false;
    for (int c = c0; c < c1; ++c) any |= act[cur][c] != 0;
    if (!any) break;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      if (pass == 0) {
        // z and d of an item's rows, in flight together and (cooperative launch) one item
        // ahead of the products; a fixed node has z = d = 0
        double zj[kSolveRow], dj[kSolveRow];
        auto fetch = [&](int k) {
          const SolveRows<NT>& R = rows[part_of(k) - part0];
          const size_t base = static_cast<size_t>(comp_of(k)) * a.nn;
          const int most = R.most;
#pragma unroll
          for (int u = 0; u < kSolveRow; ++u) {
            if (u >= most) break;
            const uint32_t m = R.nb[u][tid];
            if (CLUSTER) {
              zj[u] = cluster_load(m);
              dj[u] = cluster_load(m + kDirAt + static_cast<uint32_t>(sizeof(double) * NT) * cur);
            } else {   // other blocks': past the L1
              zj[u] = __ldcg(a.z + base + m);
              dj[u] = __ldcg(a.d0 + base + m);
            }
          }
        };
#pragma unroll
        for (int u = 0; u < kSolveRow; ++u) zj[u] = dj[u] = 0.0;
        if (nb > 0) fetch(0);
#pragma unroll 1
        for (int k = 0; k < nb; ++k) {
          const int c = comp_of(k), part = part_of(k), n = node_of(part);
          SolveItem<NT>& S = item[k];
          const SolveRows<NT>& R = rows[part - part0];
          const double beta = ssc[c * kSc + eops::S_BETA];
          const int len = R.len[tid], most = R.most;
          // in entry order; the entries past a shorter row's end are 0 times a finite value,
          // and the loop ends at the item's longest row (an FP64 instruction with its lanes
          // switched off takes the pipe as long)
          double dir[kSolveRow];
#pragma unroll
          for (int u = 0; u < kSolveRow; ++u) {
            if (u >= most) break;
            dir[u] = zj[u] + beta * dj[u];
          }
          if (k + 1 < nb) fetch(k + 1);
          if (!act[cur][c]) continue;
          double acc = 0.0;
#pragma unroll
          for (int u = 0; u < kSolveRow; ++u) {
            if (u >= most) break;
            acc += R.val[u][tid] * (u < len ? dir[u] : 0.0);
          }
          if (len > kSolveRow) {
            const int r0 = a.row[n];
            const size_t base = static_cast<size_t>(c) * a.nn;
            for (int u = kSolveRow; u < len; ++u) {
              const int m = a.col[r0 + u];
              double zm, dm;
              if (CLUSTER) {
                const uint32_t ad = node_addr(m);
                zm = cluster_load(ad);
                dm = cluster_load(ad + kDirAt + static_cast<uint32_t>(sizeof(double) * NT) * cur);
              } else {
                zm = __ldcg(a.z + base + m);
                dm = __ldcg(a.d0 + base + m);
              }
              acc += a.val[r0 + u] * (zm + beta * dm);
            }
          }
          const bool fr = S.fr[tid];
          const double dn = fr ? S.z[tid] + beta * S.d[CLUSTER ? cur : 0][tid] : 0.0;
          const double qn = fr ? acc : 0.0;
          S.d[CLUSTER ? 1 - cur : 0][tid] = dn;
          S.q[tid] = qn;
          if (!CLUSTER && n < a.nn) a.d1[static_cast<size_t>(c) * a.nn + n] = dn;
          S.sums[0][tid] = dn * qn;
        }
      } else {
#pragma unroll 1
        for (int k = 0; k < nb; ++k) {
          const int c = comp_of(k), part = part_of(k), n = node_of(part);
          if (!act[cur][c]) continue;
          SolveItem<NT>& S = item[k];
          const SolveRows<NT>& R = rows[part - part0];
          const double alpha = ssc[c * kSc + S_ALPHA];
          double r = S.r[tid], zz = 0.0;
          if (S.fr[tid]) {
            const double d = R.diag[tid];
            S.x[tid] += alpha * S.d[CLUSTER ? 1 - cur : 0][tid];
            r -= alpha * S.q[tid];
            S.r[tid] = r;
            zz = divide(r, d, R.inv[tid], mid_range(d));
          }
          S.z[tid] = zz;
          if (!CLUSTER && n < a.nn) a.z[static_cast<size_t>(c) * a.nn + n] = zz;
          S.sums[0][tid] = r * zz;
          S.sums[1][tid] = zz * zz;
        }
      }
      __syncthreads();
      // each item's sum by one warp, in the tree's order
      for (int t = warp; t < nb * (pass + 1); t += W) {
        const int k = pass ? t >> 1 : t, which = pass ? t & 1 : 0, c = comp_of(k);
        if (!act[cur][c]) continue;
        double v[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = m < W ? item[k].sums[which][lane + 32 * m] : 0.0;
        const double sum = tree256(v, W);
        if (CLUSTER) {
          if (lane < kClusterBlocks)
            cluster_store(cluster_addr(&csum[pass + which][part_of(k)], static_cast<uint32_t>(lane)), sum);
        } else if (lane == 0) {
          __stcg(a.slots + eops::pcg_sum_slot(pass, which, a.C, per, c, part_of(k)), sum);
        }
      }
      if (CLUSTER) {
        cluster_barrier();
      } else {
        if (!grid_exchange(a, target += gridDim.x, warp < (c1 - c0) * (pass + 1))) failed = 1;
      }
      solve_totals<P, W, CLUSTER>(a, pass, c0, c1, CLUSTER ? &csum[pass][0] : a.slots, ssc, act[cur], act[1 - cur]);
      __syncthreads();
      if (!CLUSTER && failed) {
        if (tid == 0) a.sc[S_FAILED] = 1.0;
        return;
      }
    }
    // a component that has stopped stays so in both halves
    if (tid < a.C && !act[cur][tid]) act[1 - cur][tid] = 0;
    __syncthreads();
    double* t = a.d0;
    a.d0 = a.d1;
    a.d1 = t;
  }
  for (int k = 0; k < nb; ++k) {
    const int n = node_of(part_of(k));
    const size_t o = static_cast<size_t>(comp_of(k)) * a.nn + n;
    if (n < a.nn) {
      a.x[o] = item[k].x[tid];
      a.r[o] = item[k].r[tid];
      if (CLUSTER) {   // for a launch that goes on from here
        a.z[o] = item[k].z[tid];
        a.d0[o] = item[k].d[it & 1][tid];
      }
    }
  }
  if (CLUSTER ? rank == 0 : blockIdx.x == 0) solve_store_scalars(a, c0, c1, ssc, act[0], act[1]);
  if (CLUSTER) cluster_barrier();   // no block leaves while another may still read its memory
}

// The same with rows and vectors in global memory, for systems whose share does not fit
// shared memory or of more than 256 kRedBlocks nodes (a slice's threads then take every
// kRedBlocks-th slice's nodes in turn, as in the setup): there the FP64 work of a pass
// outweighs its latency.  Cooperative launch, kStreamRound items' sums at a time.
constexpr int kStreamRound = 4;
__global__ void __launch_bounds__(kEB) pcg_stream_kernel(SolveArgs a) {
  constexpr int W = kEB / 32;
  __shared__ double ssc[kMaxSystems * kSc];
  __shared__ int act[2][kMaxSystems];
  __shared__ double sums[kStreamRound][2][kEB];
  __shared__ int failed;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int items = a.C * a.nvb;
  for (int i = tid; i < a.C * kSc; i += kEB) ssc[i] = a.sc[i];
  if (tid < a.C) act[0][tid] = act[1][tid] = a.sc[tid * kSc + eops::S_ACTIVE] != 0.0;
  if (tid == 0) failed = 0;
  __syncthreads();
  unsigned target = 0;
  for (int it = 0; it < a.limit; ++it) {
    const int cur = it & 1;
    bool any = false;
    for (int c = 0; c < a.C; ++c) any |= act[cur][c] != 0;
    if (!any) break;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      for (int i0 = blockIdx.x; i0 < items; i0 += gridDim.x * kStreamRound) {
        int nr = 0;
#pragma unroll 1
        for (int i = i0; i < items && nr < kStreamRound; i += gridDim.x, ++nr) {
          const int c = i / a.nvb, vb = i - c * a.nvb;
          if (!act[cur][c]) continue;
          const size_t base = static_cast<size_t>(c) * a.nn;
          const double beta = ssc[c * kSc + eops::S_BETA], alpha = ssc[c * kSc + S_ALPHA];
          double s0 = 0.0, s1 = 0.0;
          for (int n = vb * kEB + tid; n < a.nn; n += a.nvb * kEB) {
            const size_t o = base + n;
            const bool fr = !a.fixed || !a.fixed[o];
            if (pass) {
              eops::pcg_node(3, fr, a.diag[n], alpha, nullptr, a.x + o, a.r + o, a.z + o, a.d1 + o, a.q + o, &s0, &s1);
              continue;
            }
            double acc = 0.0;
            const int r0 = a.row[n], r1 = a.row[n + 1];
#pragma unroll 1
            for (int k0 = r0; k0 < r1; k0 += kRowChunk) {
              int32_t cj[kRowChunk];
              double vk[kRowChunk], zj[kRowChunk], dj[kRowChunk];
#pragma unroll
              for (int u = 0; u < kRowChunk; ++u) cj[u] = k0 + u < r1 ? a.col[k0 + u] : n;
#pragma unroll
              for (int u = 0; u < kRowChunk; ++u) {
                vk[u] = k0 + u < r1 ? a.val[k0 + u] : 0.0;
                zj[u] = __ldcg(a.z + base + cj[u]);
                dj[u] = __ldcg(a.d0 + base + cj[u]);
              }
#pragma unroll
              for (int u = 0; u < kRowChunk; ++u)
                if (k0 + u < r1) acc += vk[u] * (zj[u] + beta * dj[u]);
            }
            double dn = fr ? a.z[o] + beta * a.d0[o] : 0.0, unused = 0.0;
            eops::pcg_node(2, fr, 1.0, 0.0, nullptr, nullptr, nullptr, nullptr, &dn, &acc, &s0, &unused);
            a.d1[o] = dn;
            a.q[o] = acc;
          }
          sums[nr][0][tid] = s0;
          if (pass) sums[nr][1][tid] = s1;
        }
        __syncthreads();
        for (int t = warp; t < nr * (pass + 1); t += W) {
          const int q = pass ? t >> 1 : t, which = pass ? t & 1 : 0;
          const int i = i0 + q * static_cast<int>(gridDim.x), c = i / a.nvb;
          if (!act[cur][c]) continue;
          double v[8];
#pragma unroll
          for (int m = 0; m < 8; ++m) v[m] = sums[q][which][lane + 32 * m];
          const double sum = tree256(v, W);
          if (lane == 0) __stcg(a.slots + eops::pcg_sum_slot(pass, which, a.C, a.nvb, c, i - c * a.nvb), sum);
        }
        __syncthreads();
      }
      if (!grid_exchange(a, target += gridDim.x, warp < a.C * (pass + 1))) failed = 1;
      solve_totals<1, W, false>(a, pass, 0, a.C, a.slots, ssc, act[cur], act[1 - cur]);
      __syncthreads();
      if (failed) {
        if (tid == 0) a.sc[S_FAILED] = 1.0;
        return;
      }
    }
    if (tid < a.C && !act[cur][tid]) act[1 - cur][tid] = 0;
    __syncthreads();
    double* t = a.d0;
    a.d0 = a.d1;
    a.d1 = t;
  }
  if (blockIdx.x == 0) solve_store_scalars(a, 0, a.C, ssc, act[0], act[1]);
}

// xD = fixed ? x : 0 (the Dirichlet columns of the reduced load).
__global__ void dirichlet_part_kernel(int64_t n, const uint8_t* __restrict__ fixed, const double* __restrict__ x,
                                      double* __restrict__ xd) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  xd[i] = (fixed && fixed[i]) ? x[i] : 0.0;
}

// A component whose reduced load is zero has the zero solution on its free nodes.
__global__ void trivial_kernel(int nn, int C, const uint8_t* __restrict__ fixed, const double* __restrict__ sc,
                               double* __restrict__ x) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= static_cast<int64_t>(nn) * C) return;
  const int c = static_cast<int>(i / nn);
  eops::pcg_trivial(!(fixed && fixed[i]), sc + c * kSc, x + i);
}

// Element gradients (Eq. 39 with Eq. 40's derivatives) of nq nodal quantities q[nq][nn]:
// eg[nq][ne][2].
__global__ void egrad_kernel(int ne, int nn, int nq, const double* __restrict__ fe, const int32_t* __restrict__ tri,
                             const double* __restrict__ q, double* __restrict__ eg) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= static_cast<int64_t>(ne) * nq) return;
  const int j = static_cast<int>(i / ne), e = static_cast<int>(i % ne);
  eops::elem_gradient(e, fe, tri, q + static_cast<size_t>(j) * nn, &eg[2 * i], &eg[2 * i + 1]);
}

// Node transfer (Sect. 3.4): the mean over the elements around each node: gn[nq][nn][2].
__global__ void nmean_kernel(int nn, int ne, int nq, const int32_t* __restrict__ ne_off,
                             const int32_t* __restrict__ ne_list, const double* __restrict__ eg,
                             double* __restrict__ gn) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= static_cast<int64_t>(nn) * nq) return;
  const int j = static_cast<int>(i / nn), n = static_cast<int>(i % nn);
  eops::node_mean(n, ne_off, ne_list, eg + 2 * static_cast<size_t>(j) * ne, &gn[2 * i], &gn[2 * i + 1]);
}

// Inputs of the first derivative pass: <U>*, <V>* (from nmom or a caller's [nn][3]), P and
// <uu>, <vv>, <uv> from the fields: q6[6][nn].
template <typename T>
__global__ void pressure_inputs_kernel(int nn, const double* __restrict__ ustar, int ustride, int uoff,
                                       const double* __restrict__ P, const T* __restrict__ f,
                                       double* __restrict__ q6) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  const T* fn = f + static_cast<size_t>(n) * kNF;
  q6[n] = ustar[static_cast<size_t>(n) * ustride + uoff];
  q6[static_cast<size_t>(nn) + n] = ustar[static_cast<size_t>(n) * ustride + uoff + 1];
  q6[2 * static_cast<size_t>(nn) + n] = P[n];
  q6[3 * static_cast<size_t>(nn) + n] = fn[23];
  q6[4 * static_cast<size_t>(nn) + n] = fn[24];
  q6[5 * static_cast<size_t>(nn) + n] = fn[26];
}

__global__ void second_inputs_kernel(int nn, const double* __restrict__ g6, double* __restrict__ q2) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  const double* gp = g6 + 2 * (2 * static_cast<size_t>(nn));   // gradient of P
  q2[n] = gp[2 * n];
  q2[static_cast<size_t>(nn) + n] = gp[2 * n + 1];
}

// Eq. 33's source and the increment's outward normal derivative at no-slip nodes (Eq. 61
// from the fields minus n . grad P).
template <typename T>
__global__ void pressure_src_kernel(int nn, const double* __restrict__ g6, const double* __restrict__ g2,
                                    const T* __restrict__ f, const int8_t* __restrict__ ncls,
                                    const double* __restrict__ nrm, double nu, double dt, double Cp,
                                    double* __restrict__ src, double* __restrict__ flux) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  const size_t N2 = 2 * static_cast<size_t>(nn);
  const double lapP = g2[2 * n] + g2[N2 + 2 * n + 1];
  eops::pressure_node(g6 + 2 * n, g6 + N2 + 2 * n, g6 + 2 * N2 + 2 * n, g6 + 3 * N2 + 2 * n,
                      g6 + 4 * N2 + 2 * n, g6 + 5 * N2 + 2 * n, lapP, f + static_cast<size_t>(n) * kNF, ncls[n],
                      nrm[2 * n], nrm[2 * n + 1], nu, dt, Cp, &src[n], &flux[n]);
}

// Galerkin load of Eq. 33: b = -M src + the no-slip edge integrals of the normal derivative.
__global__ void pressure_load_kernel(int nn, const int32_t* __restrict__ row, const int32_t* __restrict__ col,
                                     const double* __restrict__ mval, const double* __restrict__ src,
                                     const double* __restrict__ flux, const int32_t* __restrict__ boff,
                                     const int32_t* __restrict__ bnb, const double* __restrict__ blen,
                                     double* __restrict__ b) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  b[n] = eops::pressure_load_node(n, row, col, mval, src, flux, boff, bnb, blen);
}

// v -= sum[0] / div (a sum the dot kernels left in device memory).
__global__ void sub_mean_kernel(int nn, const double* __restrict__ sum, double div, double* __restrict__ v) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  v[n] -= sum[0] / div;
}

// part[blk] = sum over the block's slice of w[n] v[n] (w = NULL: 1).
__global__ void dot_part_kernel(int nn, const double* __restrict__ w, const double* __restrict__ v,
                                double* __restrict__ part) {
  __shared__ double sh[kEB];
  double s = 0.0;
  for (int n = blockIdx.x * kEB + threadIdx.x; n < nn; n += gridDim.x * kEB) s += (w ? w[n] : 1.0) * v[n];
  const double t = block_sum(s, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = t;
}

__global__ void dot_finish_kernel(int nblk, const double* __restrict__ part, double* __restrict__ out) {
  __shared__ double sh[kEB];
  double s = 0.0;
  for (int j = threadIdx.x; j < nblk; j += kEB) s += part[j];
  const double t = block_sum(s, sh);
  if (threadIdx.x == 0) out[0] = t;
}

template <typename T>
__global__ void write_wp_kernel(int nn, const double* __restrict__ x, T* __restrict__ f) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  for (int c = 0; c < 9; ++c) f[static_cast<size_t>(n) * kNF + 14 + c] = static_cast<T>(x[static_cast<size_t>(c) * nn + n]);
}

template <typename T>
__global__ void write_pgrad_kernel(int nn, const double* __restrict__ gp, T* __restrict__ f) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  f[static_cast<size_t>(n) * kNF + 3] = static_cast<T>(gp[2 * n]);
  f[static_cast<size_t>(n) * kNF + 4] = static_cast<T>(gp[2 * n + 1]);
}

__global__ void diag_kernel(int nn, const int32_t* __restrict__ dpos, const double* __restrict__ val,
                            double* __restrict__ diag) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n < nn) diag[n] = val[dpos[n]];
}

__global__ void add_kernel(int nn, const double* __restrict__ a, double* __restrict__ b) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n < nn) b[n] += a[n];
}

}  // namespace

// Blocks of the reduction passes: one node per thread up to kRedBlocks blocks (the passes
// are latency-bound at these sizes, so every SM should take part).
int pcg_blocks(int nn) {
  const int nb = static_cast<int>(blocks_for(nn));
  return nb < kRedBlocks ? nb : kRedBlocks;
}

// Partial sums and scalars of the setup passes, the solve kernel's slots and counter.
size_t pcg_scratch_doubles(int nn, int C) {
  const size_t nb = static_cast<size_t>(C) * static_cast<size_t>(pcg_blocks(nn));
  return 2 * nb + static_cast<size_t>(C) * kSc + eops::kPcgSumSets * nb + 1;
}

template <typename T>
void launch_wp_rhs(const T* fields, int nn, const WpConst& k, double* rhs, double* L, int* err, cudaStream_t s) {
  wp_rhs_kernel<T><<<blocks_for(nn), kEB, 0, s>>>(fields, nn, k, rhs, L, err);
}

template <typename T>
void launch_wp_bc(const T* fields, int nn, const WpConst& k, const int8_t* ncls, const double* nrm,
                  uint8_t* fixed, double* x, int* err, cudaStream_t s) {
  wp_bc_kernel<T><<<blocks_for(nn), kEB, 0, s>>>(fields, nn, k, ncls, nrm, fixed, x, err);
}

template <typename T>
void launch_read_wp(int nn, const T* fields, double* x, cudaStream_t s) {
  read_wp_kernel<T><<<blocks_for(nn), kEB, 0, s>>>(nn, fields, x);
}

// The elliptic-relaxation matrix M + L_e^2 K into aval[nnz] and its diagonal into adiag[nn].
void launch_assemble_wp(const FemDev& m, const double* L, double* aval, double* adiag, cudaStream_t s) {
  assemble_wp_kernel<<<blocks_for(m.nnz), kEB, 0, s>>>(m.nnz, m.cptr, m.clist, m.fe, m.tri, L, aval);
  diag_kernel<<<blocks_for(m.nn), kEB, 0, s>>>(m.nn, m.dpos, aval, adiag);
}

void launch_spmv(const FemDev& m, const double* val, int C, const double* x, double* y, cudaStream_t s) {
  spmv_kernel<<<blocks_for(static_cast<int64_t>(m.nn) * C), kEB, 0, s>>>(m.nn, C, m.row, m.col, val, x, y);
}

// Jacobi-PCG setup for C systems sharing one matrix: the reduced load's norm, the zero
// solution of components with a zero reduced load, the initial residual and direction.
void launch_pcg_setup(const FemDev& m, const PcgArgs& a, cudaStream_t s) {
  const int nn = m.nn, C = a.C, nblk = pcg_blocks(nn);
  const int64_t n = static_cast<int64_t>(nn) * C;
  double* part = a.scratch;
  double* sc = a.scratch + 2 * static_cast<size_t>(C) * nblk;
  const dim3 grid(static_cast<unsigned>(nblk), static_cast<unsigned>(C));
  dirichlet_part_kernel<<<blocks_for(n), kEB, 0, s>>>(n, a.fixed, a.x, a.d);
  spmv_kernel<<<blocks_for(n), kEB, 0, s>>>(nn, C, m.row, m.col, a.val, a.d, a.q);
  pcg_pass_kernel<<<grid, kEB, 0, s>>>(0, nn, a.fixed, a.diag, a.b, a.x, a.r, a.z, a.d, a.q, sc, part);
  pcg_scalar_kernel<<<C, kEB, 0, s>>>(0, nblk, part, a.tol, sc);
  trivial_kernel<<<blocks_for(n), kEB, 0, s>>>(nn, C, a.fixed, sc, a.x);
  spmv_kernel<<<blocks_for(n), kEB, 0, s>>>(nn, C, m.row, m.col, a.val, a.x, a.q);
  pcg_pass_kernel<<<grid, kEB, 0, s>>>(1, nn, a.fixed, a.diag, a.b, a.x, a.r, a.z, a.d, a.q, sc, part);
  pcg_scalar_kernel<<<C, kEB, 0, s>>>(1, nblk, part, a.tol, sc);
}

const double* pcg_scalars(const PcgArgs& a, int nn) {
  return a.scratch + 2 * static_cast<size_t>(a.C) * pcg_blocks(nn);
}

namespace {

constexpr size_t kMaxSolveSmem = 220 * 1024;   // dynamic, beside the kernel's own arrays

OncePerDevice solve_configured;
cudaError_t configure_solves() {
  return once_on_device(solve_configured, [] {
    const void* const kernels[] = {reinterpret_cast<const void*>(pcg_solve_kernel<2, true>),
                                   reinterpret_cast<const void*>(pcg_solve_kernel<1, true>),
                                   reinterpret_cast<const void*>(pcg_solve_kernel<1, false>)};
    for (int k = 0; k < 3; ++k) {
      cudaError_t e = allow_shared(kernels[k], kMaxSolveSmem);
      if (e == cudaSuccess && k < 2) e = cudaFuncSetAttribute(kernels[k], cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  });
}

template <int P, bool CLUSTER>
size_t solve_smem(const SolveArgs& k) {
  constexpr int NT = kEB / P;
  const int rows = CLUSTER ? k.K : (k.K + k.C - 2) / k.C + 1;   // slice parts that K items touch, at most
  return sizeof(SolveItem<NT>) * k.K + sizeof(SolveRows<NT>) * rows;
}

cudaError_t start_solve(void (*f)(SolveArgs), SolveArgs k, int blocks, int threads, size_t smem, bool cluster,
                        cudaStream_t s) {
  cudaLaunchAttribute at{};
  if (cluster) {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kClusterBlocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
  } else {
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(blocks));
  cfg.blockDim = dim3(static_cast<unsigned>(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (cluster) {   // none fits where the context has a share of the device without 16 multiprocessors together
    int fit = 0;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&fit, f, &cfg);
    if (e != cudaSuccess || fit < 1) return e != cudaSuccess ? e : cudaErrorInvalidClusterSize;
  }
  return cudaLaunchKernelEx(&cfg, f, k);
}

// A launch that the context's share of the device does not grant, and nothing worse: nothing has
// run and a smaller one may.
bool refused(cudaError_t e) {
  if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorInvalidClusterSize &&
      e != cudaErrorLaunchOutOfResources && e != cudaErrorInvalidConfiguration && e != cudaErrorNotSupported)
    return false;
  cudaGetLastError();   // it was the launch's alone
  return true;
}

// Iterations of every component still iterating as six plain kernels each, for a context that is
// granted no launch whose blocks may wait for one another: the same bits.
void launch_pcg_iterations(const FemDev& m, const PcgArgs& a, int n, cudaStream_t s) {
  const int nn = m.nn, C = a.C, nblk = pcg_blocks(nn);
  const int64_t all = static_cast<int64_t>(nn) * C;
  double* part = a.scratch;
  double* sc = a.scratch + 2 * static_cast<size_t>(C) * nblk;
  const dim3 grid(static_cast<unsigned>(nblk), static_cast<unsigned>(C));
  for (int it = 0; it < n; ++it) {
    pcg_direction_kernel<<<blocks_for(all), kEB, 0, s>>>(nn, C, a.fixed, a.z, a.d, sc);
    spmv_kernel<<<blocks_for(all), kEB, 0, s>>>(nn, C, m.row, m.col, a.val, a.d, a.q);
    for (int step = 2; step <= 3; ++step) {
      pcg_pass_kernel<<<grid, kEB, 0, s>>>(step, nn, a.fixed, a.diag, a.b, a.x, a.r, a.z, a.d, a.q, sc, part);
      pcg_scalar_kernel<<<C, kEB, 0, s>>>(step, nblk, part, a.tol, sc);
    }
  }
}
constexpr int kPlainChunk = 16;   // iterations between two looks at the scalars

}  // namespace

// Up to `limit` (even) iterations of every component still iterating, in one launch.  After
// a launch that ran them all the direction is back in a.d.  Where the context is not granted
// that launch (a share of the device's multiprocessors), the next form down is taken, from a.form
// on: cluster, cooperative with the rows in shared memory, streamed with as many blocks as are
// granted, plain kernels.  Every form forms the same sums in the same order, so the bits and the
// iterations do not depend on it.  *ran: the iterations that may have run, *launches: kernels.
//
// A component takes a cluster where that leaves a block at most two slices: beyond, the FP64
// work of 16 multiprocessors (and the eight clusters of 16 that the GPU holds apart) outweighs
// the cheaper exchange.  us per iteration, cluster / cooperative (rows in shared memory) /
// streamed: 1 component 5.8 / 8.8 / 10.9 at 1,104 nodes, 8.9 / 9.3 / 10.1 at 6,600, 13.1 /
// 10.0 / 10.9 at 12,600, - / 10.0 / 11.0 at 25,200; 9 components 6.8 / 14.4 / 15.4, 11.5 /
// 18.1 / 20.5, 26.2 / 21.1 / 24.9, - / 29 / 38 (two kernels per iteration: 20 and 23 at 1,104
// and 25,200 nodes with 1 component).
cudaError_t launch_pcg_solve(const FemDev& m, const PcgArgs& a, int limit, int num_sms, int* ran, int* launches,
                             cudaStream_t s) {
  if (a.C > kMaxSystems) return cudaErrorInvalidValue;
  *ran = limit;
  *launches = 1;
  SolveArgs k{};
  k.nn = m.nn;
  k.C = a.C;
  k.nvb = pcg_blocks(m.nn);
  k.limit = limit;
  k.row = m.row;
  k.col = m.col;
  k.val = a.val;
  k.fixed = a.fixed;
  k.diag = a.diag;
  k.x = a.x;
  k.r = a.r;
  k.z = a.z;
  k.q = a.q;
  k.d0 = a.d;
  k.d1 = a.d2;
  k.tol = a.tol;
  k.sc = a.scratch + 2 * static_cast<size_t>(a.C) * k.nvb;
  k.slots = k.sc + static_cast<size_t>(a.C) * kSc;
  k.arrived = reinterpret_cast<unsigned*>(k.slots + eops::kPcgSumSets * static_cast<size_t>(a.C) * k.nvb);
  cudaError_t e = configure_solves();
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(k.arrived, 0, sizeof(double), s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(k.sc + S_FAILED, 0, sizeof(double), s);
  if (e != cudaSuccess) return e;
  const int sms = num_sms > 0 ? num_sms : 1;
  const bool node_per_thread = m.nn <= kEB * kRedBlocks;
  const int P = 2 * k.nvb <= kClusterBlocks ? 2 : 1;
  k.K = (k.nvb * P + kClusterBlocks - 1) / kClusterBlocks;
  if (a.form <= kSolveCluster && node_per_thread && k.K <= 2) {
    const int blocks = k.C * kClusterBlocks;
    e = P == 2 ? start_solve(pcg_solve_kernel<2, true>, k, blocks, kEB / 2, solve_smem<2, true>(k), true, s)
               : start_solve(pcg_solve_kernel<1, true>, k, blocks, kEB, solve_smem<1, true>(k), true, s);
    if (!refused(e)) return e;
  }
  const int items = k.C * k.nvb;
  k.K = (items + sms - 1) / sms;
  if (a.form <= kSolveRows && node_per_thread && solve_smem<1, false>(k) <= kMaxSolveSmem) {
    e = start_solve(pcg_solve_kernel<1, false>, k, (items + k.K - 1) / k.K, kEB, solve_smem<1, false>(k), false, s);
    if (!refused(e)) return e;
  }
  if (a.form <= kSolveStream) {
    for (int blocks = items < sms ? items : sms; blocks > 0; blocks /= 2) {
      e = start_solve(pcg_stream_kernel, k, blocks, kEB, 0, false, s);
      if (!refused(e)) return e;
    }
  }
  *ran = limit < kPlainChunk ? limit : kPlainChunk;
  *launches = 6 * *ran;
  launch_pcg_iterations(m, a, *ran, s);
  return cudaSuccess;
}

bool pcg_solve_failed(const double* h) { return h[S_FAILED] != 0.0; }

// Node-transferred gradients (Sect. 3.4) of nq quantities q[nq][nn] into gn[nq][nn][2];
// eg is scratch of 2 nq ne doubles.
void launch_node_gradients(const FemDev& m, const int32_t* ne_off, const int32_t* ne_list, int nq,
                           const double* q, double* eg, double* gn, cudaStream_t s) {
  egrad_kernel<<<blocks_for(static_cast<int64_t>(m.ne) * nq), kEB, 0, s>>>(m.ne, m.nn, nq, m.fe, m.tri, q, eg);
  nmean_kernel<<<blocks_for(static_cast<int64_t>(m.nn) * nq), kEB, 0, s>>>(m.nn, m.ne, nq, ne_off, ne_list, eg, gn);
}

template <typename T>
void launch_pressure_rhs(const FemDev& m, const int32_t* ne_off, const int32_t* ne_list, const double* ustar,
                         int ustride, int uoff, const double* P, const T* fields, double nu, double dt,
                         double Cp, double* work, double* src, double* flux, cudaStream_t s) {
  const size_t nn = static_cast<size_t>(m.nn), ne = static_cast<size_t>(m.ne);
  double* q6 = work;                 // 6 nn
  double* g6 = q6 + 6 * nn;          // 12 nn
  double* q2 = g6 + 12 * nn;         // 2 nn
  double* g2 = q2 + 2 * nn;          // 4 nn
  double* eg = g2 + 4 * nn;          // 12 ne
  pressure_inputs_kernel<T><<<blocks_for(m.nn), kEB, 0, s>>>(m.nn, ustar, ustride, uoff, P, fields, q6);
  launch_node_gradients(m, ne_off, ne_list, 6, q6, eg, g6, s);
  second_inputs_kernel<<<blocks_for(m.nn), kEB, 0, s>>>(m.nn, g6, q2);
  launch_node_gradients(m, ne_off, ne_list, 2, q2, eg, g2, s);
  pressure_src_kernel<T><<<blocks_for(m.nn), kEB, 0, s>>>(m.nn, g6, g2, fields, m.ncls, m.nrm, nu, dt, Cp, src, flux);
  (void)ne;
}

size_t pressure_rhs_scratch_doubles(int nn, int ne) {
  return 24 * static_cast<size_t>(nn) + 12 * static_cast<size_t>(ne);
}

// The Galerkin load of Eq. 33 with its nodal mean removed; red holds kRedBlocks + 1 doubles.
void launch_pressure_load(const FemDev& m, const double* src, const double* flux, double* b, double* red,
                          cudaStream_t s) {
  pressure_load_kernel<<<blocks_for(m.nn), kEB, 0, s>>>(m.nn, m.row, m.col, m.mval, src, flux, m.boff, m.bnb,
                                                        m.blen, b);
  const int nblk = pcg_blocks(m.nn);
  dot_part_kernel<<<nblk, kEB, 0, s>>>(m.nn, nullptr, b, red);
  dot_finish_kernel<<<1, kEB, 0, s>>>(nblk, red, red + kRedBlocks);
  sub_mean_kernel<<<blocks_for(m.nn), kEB, 0, s>>>(m.nn, red + kRedBlocks, static_cast<double>(m.nn), b);
}

// Zero integral: x -= (sum_n mlump_n x_n) / (domain area).
void launch_zero_mean(const FemDev& m, double* x, double* red, cudaStream_t s) {
  const int nblk = pcg_blocks(m.nn);
  dot_part_kernel<<<nblk, kEB, 0, s>>>(m.nn, m.mlump, x, red);
  dot_finish_kernel<<<1, kEB, 0, s>>>(nblk, red, red + kRedBlocks);
  sub_mean_kernel<<<blocks_for(m.nn), kEB, 0, s>>>(m.nn, red + kRedBlocks, m.area, x);
}

template <typename T>
void launch_write_wp(int nn, const double* x, T* fields, cudaStream_t s) {
  write_wp_kernel<T><<<blocks_for(nn), kEB, 0, s>>>(nn, x, fields);
}

template <typename T>
void launch_write_pgrad(const FemDev& m, const int32_t* ne_off, const int32_t* ne_list, const double* P,
                        double* eg, double* gp, T* fields, cudaStream_t s) {
  launch_node_gradients(m, ne_off, ne_list, 1, P, eg, gp, s);
  write_pgrad_kernel<T><<<blocks_for(m.nn), kEB, 0, s>>>(m.nn, gp, fields);
}

void launch_add(int nn, const double* a, double* b, cudaStream_t s) {
  add_kernel<<<blocks_for(nn), kEB, 0, s>>>(nn, a, b);
}

#define PDFX_INSTANTIATE(T)                                                                         \
  template void launch_wp_rhs<T>(const T*, int, const WpConst&, double*, double*, int*, cudaStream_t); \
  template void launch_wp_bc<T>(const T*, int, const WpConst&, const int8_t*, const double*, uint8_t*, \
                                double*, int*, cudaStream_t);                                        \
  template void launch_pressure_rhs<T>(const FemDev&, const int32_t*, const int32_t*, const double*,  \
                                       int, int, const double*, const T*, double, double, double,     \
                                       double*, double*, double*, cudaStream_t);                      \
  template void launch_write_wp<T>(int, const double*, T*, cudaStream_t);                             \
  template void launch_read_wp<T>(int, const T*, double*, cudaStream_t);                              \
  template void launch_write_pgrad<T>(const FemDev&, const int32_t*, const int32_t*, const double*,   \
                                      double*, double*, T*, cudaStream_t);
PDFX_INSTANTIATE(float)
PDFX_INSTANTIATE(double)
#undef PDFX_INSTANTIATE

}  // namespace pdfx
