// solve_kernels.cu -- supernodal forward and back substitution on the device.
//
// Sec. 1 and Sec. 2 of the paper: the solve phase solves L y = b and then L^T x = y.  With
// the supernodal factor both run over the level sets: the forward solve goes from the
// leaves up (a supernode's rows are final once all of its descendants are done), the back
// solve from the root down (a supernode needs the solution on its off-diagonal rows, which
// belong to ancestors).
//
// Vectors are n x nrhs column-major in the permuted numbering, ld = n, stored in FP64.  The
// arithmetic runs in the precision of the panels: FP64 for an FP64 factor; FP32 for the
// FP32 factor of the mixed path, whose solves only produce refinement corrections (the
// FP64 residual of the refinement loop restores FP64 accuracy).
//   forward  task {s, r0}: y_s <- L11^{-1} y_s (redundantly in every task of s; the task
//            with r0 = 0 stores it in w), then y[rows[n+i]] -= L21[i, :] y_s for its rows,
//            by atomics, or (owner order) staged and summed per row in a fixed order.
//   backward task {s, r0}: part_q[j, c] = sum_{i in block} L21[i, j] x[rows[n+i], c] into
//            a staging slot q; the supernode's last task to finish then forms
//            x_s = L11^{-T} (w_s - sum_q part_q), the partials summed in task order
//            (deterministic).
// Where the factor keeps the inverses Y = L11^{-1} of its diagonal blocks (formed once per
// factorization), L11^{-1} y_s and L11^{-T} r_s are products with Y and Y^T, parallel over
// the block's rows; otherwise they are substitutions, one step per column.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "chol_internal.h"
#include "device_common.cuh"
#include "kernels.h"
#include "launch_util.h"
#include "solve_shape.h"

namespace chol {

// y[i, c] = B[perm[i], c] (* scale[perm[i]] when scale is given: the equilibrated system)
__global__ void k_gather_perm(const double* __restrict__ B, int64_t ldb,
                              const int32_t* __restrict__ perm, const double* __restrict__ scale,
                              int64_t n, int nrhs, double* __restrict__ y) {
  const int64_t total = n * nrhs;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = q / n, i = q - c * n;
    const int32_t o = perm[i];
    y[q] = scale ? B[c * ldb + o] * scale[o] : B[c * ldb + o];
  }
}

// X[perm[i], c] = w[i, c] (* scale[perm[i]])
__global__ void k_scatter_perm(const double* __restrict__ w, const int32_t* __restrict__ perm,
                               const double* __restrict__ scale, int64_t n, int nrhs,
                               double* __restrict__ X, int64_t ldx) {
  const int64_t total = n * nrhs;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = q / n, i = q - c * n;
    const int32_t o = perm[i];
    X[c * ldx + o] = scale ? w[q] * scale[o] : w[q];
  }
}

constexpr int kSolveThreads = kSolveRows;  // one off-diagonal row per thread

// Warp-level triangular solve of the n x n lower L11 (smem, column-major ld n) against
// xs (smem, n x nrhs, ld n).  Forward: xs <- L11^{-1} xs.  Backward: xs <- L11^{-T} xs.
// Lane l owns rows l, l+32, l+64, l+96 (n <= 128).
template <bool FORWARD, typename CT>
__device__ void warp_trisolve(const CT* L11, const CT* rdiag, CT* xs, int n, int nrhs) {
  const int lane = threadIdx.x & 31;
  // the CTA's warps share the right-hand sides: warp w solves columns w, w + nwarps, ...
  const int nwarps = blockDim.x >> 5;
  for (int c = threadIdx.x >> 5; c < nrhs; c += nwarps) {
    CT v[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int r = lane + 32 * q;
      v[q] = r < n ? xs[c * n + r] : CT(0);
    }
    for (int jj = 0; jj < n; jj++) {
      const int j = FORWARD ? jj : n - 1 - jj;
      const int qj = j >> 5, lj = j & 31;
      CT own = v[0];
      if (qj == 1) own = v[1];
      if (qj == 2) own = v[2];
      if (qj == 3) own = v[3];
      const CT xj = __shfl_sync(0xffffffffu, own, lj) * rdiag[j];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int r = lane + 32 * q;
        if (r == j) v[q] = xj;
        else if (FORWARD ? (r > j && r < n) : (r < j)) {
          // forward: row r of column j of L11; backward: (L^T)_{r j} = L_{j r}
          const CT l = FORWARD ? L11[j * n + r] : L11[r * n + j];
          v[q] -= l * xj;
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int r = lane + 32 * q;
      if (r < n) xs[c * n + r] = v[q];
    }
  }
}

// The lower triangle of L11 (the only part warp_trisolve reads) with every copy in flight
// at once, then the reciprocals of its diagonal.
template <typename P>
__device__ void load_l11(const SnDev& d, P* L11, P* rdiag) {
  stage_diag_block(L11, reinterpret_cast<const P*>(d.L), d.n, d.m);
  cp_async_wait_all();
  __syncthreads();
  const int n = d.n;
  for (int j = threadIdx.x; j < n; j += blockDim.x) rdiag[j] = P(1) / L11[j * n + j];
  __syncthreads();
}

// Y (row-major, lower triangle) into shared memory with leading dimension n + 1 (odd: the
// threads of a warp reading one column of Y hit distinct banks), every copy in flight.
template <typename P>
__device__ void stage_dinv(P* Ys, const P* __restrict__ Y, int n) {
  const int ld = n + 1, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  for (int r = threadIdx.x >> 5; r < n; r += nwarp)
    for (int k = lane; k <= r; k += 32) cp_async_elem(Ys + r * ld + k, Y + r * n + k);
}

// Panel block of a solve task in shared memory: X[j * kXld + i] = L21[r0 + i, j] for the
// task's rb rows (warps along the columns, lanes along the rows: coalesced reads; odd kXld:
// a warp reading one row across the columns hits distinct banks), every copy in flight.
constexpr int kXld = kSolveRows + 1;
template <typename P>
__device__ void stage_rows(P* X, const P* __restrict__ L21, int64_t m, int n, int rb) {
  const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  for (int j = threadIdx.x >> 5; j < n; j += nwarp)
    for (int i = lane; i < rb; i += 32) cp_async_elem(X + j * kXld + i, L21 + (int64_t)j * m + i);
}

// ---- solves of factors that keep Y = L11^-1 ------------------------------------------------
// A CTA serves one task (128 panel rows) for NR right-hand sides, those of its blockIdx.y
// (missing ones are zeros).  Vectors in shared memory hold the right-hand sides of a row
// next to one another, V[row * NR + c], so that one or a few wide loads feed NR
// multiply-adds; with them apart (V[c * n + row]) every multiply-add had a load of its own.
// Measured, one solve: 48^3 27-point FP64, 1 right-hand side 11.0 -> 7.9 ms, 16 right-hand sides
// 68.0 -> 38.2 ms (the FP64 unit's floor is 31 ms); 96^3 diffusion, three FP32 solves of 16
// right-hand sides with their residuals 123.7 -> 38.4 ms.
//  * kNarrow (levels whose tasks, times their groups of right-hand sides, fit in one wave):
//    kWideThreads threads, the task's panel block and Y staged in shared memory with every
//    copy in flight at once.  A task alone on its SM is bound by its FP64 work and the length of
//    its dependent FMA chains: the threads split the right-hand sides first (no sums to add
//    up), then the columns (forward) or rows (backward), and the launch splits the right-hand
//    sides over CTAs while SMs are idle (solve_shape).
//  * kSplit (wider levels whose supernodes have several tasks): the product with Y is a kernel of
//    its own, one CTA per supernode and group of right-hand sides, before the forward's or
//    after the backward's panel product.  In one kernel every forward task repeats it (27 % of the FP64
//    work of a full task, and FP64 throughput is what bounds these levels), and in the
//    backward the last task alone adds up the partial sums of all tasks (96^3, 16 right-hand
//    sides: 97 us on a level of two supernodes, almost all of it that sum).  kWideThreads threads,
//    the panel block staged.
//  * kLeaf (wider levels of supernodes of one or two tasks): kSolveThreads threads and a small
//    footprint, many CTAs per SM: the
//    forward reads the panel from global memory (rows contiguous: coalesced, eight or more
//    loads in flight), the backward stages it (a thread per column reading down the rows would
//    fetch each cache line several times) and Y in the supernode's last task only.
// Both kernels are launched with programmatic dependent launch: a level's CTAs start while the
// previous level still runs, fetch what no solve kernel writes (descriptors, row lists, Y and,
// where staged, the panel block) and wait for the previous level only then.
constexpr int kWideThreads = 4 * kSolveRows;
template <int MODE>
__host__ __device__ constexpr int y_threads() { return MODE != kLeaf ? kWideThreads : kSolveThreads; }

// Lets the next level's CTAs start: on levels of one wave, and with a single right-hand side (with
// more, a wide level's own work fills the SMs that the next one's waiting CTAs would take: 48^3,
// 16 right-hand sides, 38.2 ms instead of 39.0, and the 96^3 FP32 refinement of 16 38.4 instead of
// 39.7; never: 8.8 instead of 7.9 ms for one).
__device__ __forceinline__ void start_next_level(int nrhs) {
  if (nrhs == 1 || gridDim.x * gridDim.y <= kWave) pdl_launch_dependents();
}

// NR consecutive shared-memory values by the widest loads their row alignment allows.
template <typename P, int NR>
__device__ __forceinline__ void load_vec(const P* p, P (&v)[NR]) {
  constexpr int B = NR * (int)sizeof(P);
  if constexpr (B % 16 == 0) {
    constexpr int E = 16 / (int)sizeof(P);
#pragma unroll
    for (int q = 0; q < NR / E; q++) {
      if constexpr (sizeof(P) == 8) {
        const double2 t = reinterpret_cast<const double2*>(p)[q];
        v[2 * q] = t.x;
        v[2 * q + 1] = t.y;
      } else {
        const float4 t = reinterpret_cast<const float4*>(p)[q];
        v[4 * q] = t.x;
        v[4 * q + 1] = t.y;
        v[4 * q + 2] = t.z;
        v[4 * q + 3] = t.w;
      }
    }
  } else {
#pragma unroll
    for (int q = 0; q < NR; q++) v[q] = p[q];
  }
}

// Right-hand sides per thread and column segments of dinv_apply: one item per thread at n = 64.
template <int NR, int T>
__host__ __device__ constexpr int dinv_cv() { return (64 * NR + T - 1) / T; }
template <int NR, int T>
__host__ __device__ constexpr int dinv_seg() {
  return 64 * NR >= T ? 1 : (T / (64 * NR) < 8 ? T / (64 * NR) : 8);
}

// xs = Y bin (FORWARD) or Y^T bin, n x NR, Y staged by stage_dinv.  Each output is a dot product
// over the triangle's part of a row (forward: k <= r) or column (backward: k >= r) of Y; with
// fewer outputs than threads the k range is cut into segments whose partial sums are added in
// segment order through red (T entries); a thread's single output keeps four interleaved
// partial sums.  Ends with a barrier.
template <bool FORWARD, typename P, int NR, int T>
__device__ void dinv_apply(const P* Ys, const P* bin, P* xs, P* red, int n) {
  constexpr int CV = dinv_cv<NR, T>(), SEG = dinv_seg<NR, T>(), NG = NR / CV;
  const int ld = n + 1, items = n * NG;
  const int seg = (n + SEG - 1) / SEG;
  for (int idx = threadIdx.x; idx < items * SEG; idx += T) {
    const int sg = SEG > 1 ? idx / items : 0, it = idx - sg * items;
    const int g = it / n, r = it - g * n;
    int k0 = sg * seg, k1 = min(n, k0 + seg);
    if (FORWARD) k1 = min(k1, r + 1);
    else k0 = max(k0, r);
    const P* b = bin + g * CV;
    if constexpr (CV == 1) {
      // four independent chains: an FP64 FMA's result is available only tens of cycles later
      P a[4] = {P(0), P(0), P(0), P(0)};
      int k = k0;
      for (; k + 4 <= k1; k += 4)
#pragma unroll
        for (int q = 0; q < 4; q++)
          a[q] += (FORWARD ? Ys[r * ld + k + q] : Ys[(k + q) * ld + r]) * b[(k + q) * NR];
      for (; k < k1; k++) a[0] += (FORWARD ? Ys[r * ld + k] : Ys[k * ld + r]) * b[k * NR];
      const P v = (a[0] + a[1]) + (a[2] + a[3]);
      if (SEG == 1) xs[r * NR + g] = v;
      else red[idx] = v;
    } else {
      P a[CV];
#pragma unroll
      for (int c = 0; c < CV; c++) a[c] = P(0);
      for (int k = k0; k < k1; k++) {
        const P l = FORWARD ? Ys[r * ld + k] : Ys[k * ld + r];
        P bv[CV];
        load_vec<P, CV>(b + k * NR, bv);
#pragma unroll
        for (int c = 0; c < CV; c++) a[c] += l * bv[c];
      }
#pragma unroll
      for (int c = 0; c < CV; c++) xs[r * NR + g * CV + c] = a[c];
    }
  }
  __syncthreads();
  if (SEG > 1) {  // then CV = 1: an item is one output
    for (int it = threadIdx.x; it < items; it += T) {
      P v = red[it];
      for (int sg = 1; sg < SEG; sg++) v += red[sg * items + it];
      const int g = it / n, r = it - g * n;
      xs[r * NR + g] = v;
    }
    __syncthreads();
  }
}

// Shared memory (P elements, every array 16-byte aligned).  Forward: [Y n(n+1) unless kSplit],
// [X n*kXld unless kLeaf], bin n*NR (kSplit: xs itself), [xs n*NR], red max(T, 3*kSolveRows).
// Backward: [Y if kNarrow], X, xg kSolveRows*NR, hred 96*NR + 448, and unless kSplit r, xo n*NR
// each and red T; kLeaf: the last task stages Y over X.  Products with Y: Y, r, xo, the
// partial sums' sums (T doubles), red T.
__host__ __device__ constexpr int up4(int e) { return (e + 3) & ~3; }
template <int NR, int MODE>
__host__ __device__ constexpr int fwd_y_elems(int n) {
  return (MODE != kSplit ? up4(n * (n + 1)) + up4(n * NR) : 0) + (MODE != kLeaf ? up4(n * kXld) : 0) +
         up4(n * NR) + (y_threads<MODE>() > 3 * kSolveRows ? y_threads<MODE>() : 3 * kSolveRows);
}
template <int NR, int MODE>
__host__ __device__ constexpr int bwd_y_elems(int n) {
  return (MODE == kNarrow ? up4(n * (n + 1)) : 0) + up4(n * kXld) + kSolveRows * NR + 96 * NR + 448 +
         (MODE != kSplit ? 2 * up4(n * NR) + y_threads<MODE>() : 0);
}
template <int NR>
__host__ __device__ constexpr int diag_y_elems(int n) {
  return up4(n * (n + 1)) + 2 * up4(n * NR) + 3 * kWideThreads;
}

// Forward step of a level, one CTA per task {s, r0} and group of NR right-hand sides:
// x_s = Y y_s (in every task of s; the task with r0 = 0 stores it in w; kSplit: k_fwd_diag has
// stored it), then y[rows[n + r0 + i]] -= L21[r0 + i, :] x_s for the task's rows, by
// reductions or (fstage) into the level's staging slots (q * kSolveRows + i) * nrhs + c.
template <typename P, int NR, int MODE>
__global__ void __launch_bounds__(y_threads<MODE>())
    k_fwd_y(const int4* __restrict__ tasks, const SnDev* __restrict__ sns, int64_t ldv, int nrhs,
            double* y, double* w, double* fstage) {
  constexpr int T = y_threads<MODE>();
  constexpr bool STAGED = MODE != kLeaf;
  // threads split the right-hand sides RS ways and the columns CS ways (staged)
  constexpr int RS = !STAGED ? 1 : (NR >= 4 ? 4 : NR), CS = STAGED ? 4 / RS : 1, RG = NR / RS;
  constexpr int IL = NR == 1 ? 4 : 1;  // interleaved partial sums per right-hand side
  extern __shared__ __align__(16) double sm[];
  P* Ys = reinterpret_cast<P*>(sm);
  start_next_level(nrhs);
  const int4 tk = tasks[blockIdx.x];
  const SnDev d = sns[tk.x];
  const int n = d.n, m = d.m, u = m - n;
  const int rb = min(kSolveRows, u - tk.y);  // <= 0 for a supernode without rows below
  const int c0 = blockIdx.y * NR, nr = min(NR, nrhs - c0);
  const P* L = reinterpret_cast<const P*>(d.L) + n + tk.y;
  P* X = Ys + (MODE != kSplit ? up4(n * (n + 1)) : 0);
  P* bin = X + (STAGED ? up4(n * kXld) : 0);
  P* xs = bin + (MODE != kSplit ? up4(n * NR) : 0);
  P* red = xs + up4(n * NR);
  const int i = threadIdx.x % kSolveRows, g = threadIdx.x / kSolveRows;
  if (MODE != kSplit) stage_dinv(Ys, reinterpret_cast<const P*>(d.dinv), n);
  if (STAGED && rb > 0) stage_rows(X, L, m, n, rb);
  const int64_t grow = i < rb ? d.rows[n + tk.y + i] : 0;
  pdl_wait();  // the levels below are done: y is final for s
  const double* src = MODE == kSplit ? w : y;
  for (int idx = threadIdx.x; idx < n * NR; idx += T) {
    const int c = idx / n, j = idx - c * n;
    bin[j * NR + c] = c < nr ? (P)src[(int64_t)(c0 + c) * ldv + d.col0 + j] : P(0);
  }
  cp_async_wait_all();
  __syncthreads();
  if constexpr (MODE != kSplit) {
    dinv_apply<true, P, NR, T>(Ys, bin, xs, red, n);
    if (tk.y == 0)
      for (int idx = threadIdx.x; idx < n * nr; idx += T) {
        const int c = idx / n, j = idx - c * n;
        w[(int64_t)(c0 + c) * ldv + d.col0 + j] = xs[j * NR + c];
      }
  }
  // off-diagonal rows: row i, right-hand sides RG (g % RS) .., columns of group g / RS
  const int cg = g / RS, r0 = RG * (g % RS);
  P acc[RG][IL];
#pragma unroll
  for (int c = 0; c < RG; c++)
#pragma unroll
    for (int q = 0; q < IL; q++) acc[c][q] = P(0);
  if (i < rb) {
    if (STAGED) {
      const int cw = (n + CS - 1) / CS, j0 = min(n, cg * cw), j1 = min(n, j0 + cw);
      const P* xr = xs + r0;
      int j = j0;
      for (; j + 4 <= j1; j += 4)
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const P l = X[(j + q) * kXld + i];
          P xv[RG];
          load_vec<P, RG>(xr + (j + q) * NR, xv);
#pragma unroll
          for (int c = 0; c < RG; c++) acc[c][q % IL] += l * xv[c];
        }
      for (; j < j1; j++) {
        const P l = X[j * kXld + i];
#pragma unroll
        for (int c = 0; c < RG; c++) acc[c][0] += l * xr[j * NR + c];
      }
    } else {
      // independent panel loads per step: the loads are the latency here
      const P* Li = L + i;
      constexpr int QB = sizeof(P) == 4 ? 16 : 8;
      int j = 0;
      for (; j + QB <= n; j += QB) {
        P l[QB];
#pragma unroll
        for (int q = 0; q < QB; q++) l[q] = Li[(int64_t)(j + q) * m];
#pragma unroll
        for (int q = 0; q < QB; q++) {
          P xv[RG];
          load_vec<P, RG>(xs + (j + q) * NR, xv);
#pragma unroll
          for (int c = 0; c < RG; c++) acc[c][q % IL] += l[q] * xv[c];
        }
      }
      for (; j < n; j++) {
        const P l = Li[(int64_t)j * m];
#pragma unroll
        for (int c = 0; c < RG; c++) acc[c][0] += l * xs[j * NR + c];
      }
    }
  }
  P v[RG];
#pragma unroll
  for (int c = 0; c < RG; c++) {
    if constexpr (IL == 4) v[c] = (acc[c][0] + acc[c][1]) + (acc[c][2] + acc[c][3]);
    else v[c] = acc[c][0];
  }
  if constexpr (CS > 1) {  // then RG = 1: the column groups' sums, added in group order
    if (cg > 0) red[((cg - 1) * RS + g % RS) * kSolveRows + i] = v[0];
    __syncthreads();
    if (cg == 0)
      for (int gg = 1; gg < CS; gg++) v[0] += red[((gg - 1) * RS + g) * kSolveRows + i];
  }
  if (cg == 0 && i < rb) {
#pragma unroll
    for (int c = 0; c < RG; c++) {
      const int cc = r0 + c;
      if (cc >= nr) continue;
      if (fstage)
        fstage[((int64_t)blockIdx.x * kSolveRows + i) * nrhs + c0 + cc] = (double)v[c];
      else
        red_add(&y[(int64_t)(c0 + cc) * ldv + grow], -(double)v[c]);
    }
  }
}

// x_s = Y y_s of every supernode of a level (POTRF tasks) into w: the forward's kSplit.
template <typename P, int NR>
__global__ void __launch_bounds__(kWideThreads)
    k_fwd_diag(const int4* __restrict__ tasks, const SnDev* __restrict__ sns, int64_t ldv, int nrhs,
               const double* y, double* w) {
  extern __shared__ __align__(16) double sm[];
  start_next_level(nrhs);
  const SnDev d = sns[tasks[blockIdx.x].x];
  const int n = d.n, c0 = blockIdx.y * NR, nr = min(NR, nrhs - c0);
  P* Ys = reinterpret_cast<P*>(sm);
  P* bin = Ys + up4(n * (n + 1));
  P* xs = bin + up4(n * NR);
  P* red = xs + up4(n * NR);
  stage_dinv(Ys, reinterpret_cast<const P*>(d.dinv), n);
  pdl_wait();  // the levels below are done: y is final for s
  for (int idx = threadIdx.x; idx < n * NR; idx += kWideThreads) {
    const int c = idx / n, j = idx - c * n;
    bin[j * NR + c] = c < nr ? (P)y[(int64_t)(c0 + c) * ldv + d.col0 + j] : P(0);
  }
  cp_async_wait_all();
  __syncthreads();
  dinv_apply<true, P, NR, kWideThreads>(Ys, bin, xs, red, n);
  for (int idx = threadIdx.x; idx < n * nr; idx += kWideThreads) {
    const int c = idx / n, j = idx - c * n;
    w[(int64_t)(c0 + c) * ldv + d.col0 + j] = xs[j * NR + c];
  }
}

// Owner-ordered forward update: row fg_row[i] of y subtracts its staged contributions in
// the fixed order of fg_ent (ascending source supernode).
__global__ void k_fwd_gather(const int32_t* __restrict__ fg_row, const int64_t* __restrict__ fg_ptr,
                             const int32_t* __restrict__ fg_ent, int64_t nrows, int64_t ldv,
                             int nrhs, const double* __restrict__ fstage, double* __restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nrows;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = fg_row[i];
    for (int c = 0; c < nrhs; c++) {
      double s = 0.0;
      for (int64_t e = fg_ptr[i]; e < fg_ptr[i + 1]; e++) s += fstage[(int64_t)fg_ent[e] * nrhs + c];
      y[(int64_t)c * ldv + r] -= s;
    }
  }
}

// Counts this CTA into its supernode's arrivals once its partials are published; true in every
// thread of the last of the nq CTAs, which also puts the counter back to zero (the next
// launch that uses it starts after this one has ended).
__device__ __forceinline__ bool last_arrival(int* counter, int nq) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(counter, 1) == nq - 1;
    if (s_last) *counter = 0;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last;
}

// r = w_s - sum of the supernode's nq partial sums (slots pp0 + q ps, each [c][W]) for NR
// right-hand sides from c0 on, with eight loads in flight per thread (from L2: other CTAs wrote
// them); with fewer sums than threads QG threads share one, every QG-th task each, through hd
// (T doubles), added in order.  The caller's next barrier publishes r.
template <typename P, int NR, int T>
__device__ void sum_partials(const SnDev& d, const double* w, int64_t ldv, int c0, int nr,
                             const double* pp0, int64_t ps, int W, int nq, double* hd, P* r) {
  const int n = d.n;
  constexpr int QG = 64 * NR >= T ? 1 : (T / (64 * NR) < 8 ? T / (64 * NR) : 8);
  const int items = n * NR;
  for (int idx = threadIdx.x; idx < items * QG; idx += T) {
    const int qg = QG > 1 ? idx / items : 0, it = idx - qg * items;
    const int c = it / n, jj = it - c * n;
    double a[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    double wv = 0.0;
    if (c < nr) {
      const double* pp = pp0 + (int64_t)c * W + jj;
      if (qg == 0) wv = w[(int64_t)(c0 + c) * ldv + d.col0 + jj];
      int q = qg;
      for (; q + 7 * QG < nq; q += 8 * QG) {
#pragma unroll
        for (int t = 0; t < 8; t++) a[t] += __ldcg(pp + (int64_t)(q + t * QG) * ps);
      }
      double b[7];  // the remaining tasks' loads in flight together
#pragma unroll
      for (int t = 0; t < 7; t++)
        b[t] = q + t * QG < nq ? __ldcg(pp + (int64_t)(q + t * QG) * ps) : 0.0;
#pragma unroll
      for (int t = 0; t < 7; t++)
        if (q + t * QG < nq) a[t] += b[t];
    }
    const double s = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
    if (QG == 1) r[jj * NR + c] = (P)(wv - s);
    else hd[idx] = wv - s;
  }
  if (QG > 1) {
    __syncthreads();
    for (int it = threadIdx.x; it < items; it += T) {
      const int c = it / n, jj = it - c * n;
      double s = hd[it];
      for (int qg = 1; qg < QG; qg++) s += hd[qg * items + it];
      r[jj * NR + c] = (P)s;
    }
  }
}

// Backward step of a level, one CTA per task {s, r0} (a supernode's tasks are consecutive in
// the level's list, r0 = 0, kSolveRows, ...; every supernode has at least one) and group of NR
// right-hand sides.  Each CTA writes its partial part[q][c][j] = sum_{i in block} L21[r0 + i, j]
// x[rows[n + r0 + i], c] to the slot of its task's index q in the level; the last of the
// supernode's CTAs of a group to finish (last_arrival; kSplit: k_bwd_diag, the next launch)
// sums the slots and finishes x_s = Y^T (w_s - sum_q part_q): the same arithmetic whichever
// comes last, and no CTA waits for another.
// Thread (j, h): column j; h splits the right-hand sides (unless kLeaf) and the rows.
template <typename P, int NR, int MODE>
__global__ void __launch_bounds__(y_threads<MODE>())
    k_bwd_y(const int4* __restrict__ tasks, const SnDev* __restrict__ sns, int64_t ldv, int nrhs,
            int cfirst, int W, double* w, double* part, int* arrive) {
  constexpr int T = y_threads<MODE>();
  constexpr int RS = MODE == kLeaf ? 1 : (NR >= 4 ? 4 : NR), RG = NR / RS, IL = NR == 1 ? 4 : 1;
  extern __shared__ __align__(16) double sm[];
  P* Ys = reinterpret_cast<P*>(sm);
  start_next_level(nrhs);
  const int4 tk = tasks[blockIdx.x];
  const SnDev d = sns[tk.x];
  const int n = d.n, m = d.m, u = m - n;
  const int rb = max(0, min(kSolveRows, u - tk.y));
  const int c0 = cfirst + blockIdx.y * NR, nr = min(NR, nrhs - c0);
  P* X = Ys + (MODE == kNarrow ? up4(n * (n + 1)) : 0);
  P* xg = X + up4(n * kXld);          // rb x NR
  P* hred = xg + kSolveRows * NR;     // row groups' partial sums
  if (MODE == kNarrow) stage_dinv(Ys, reinterpret_cast<const P*>(d.dinv), n);
  if (rb > 0) stage_rows(X, reinterpret_cast<const P*>(d.L) + n + tk.y, m, n, rb);
  const int gi = threadIdx.x % kSolveRows;
  const int64_t grow = gi < rb ? d.rows[n + tk.y + gi] : 0;
  pdl_wait();  // the levels above are done: x is final on s's rows
  if (gi < rb)
    for (int c = threadIdx.x / kSolveRows; c < NR; c += T / kSolveRows)
      xg[gi * NR + c] = c < nr ? (P)w[(int64_t)(c0 + c) * ldv + grow] : P(0);
  cp_async_wait_all();
  __syncthreads();
  // column slots rounded up to whole warps, so that no warp straddles two groups; T / ns is
  // 2 or 4 (8 or 16 unless kLeaf): the groups' partial sums take at most 96 NR + 448 entries
  const int ns = (n + 31) & ~31, ng = T / ns;
  const int nh = min(NR == 1 ? 8 : 4, ng / RS);  // row groups
  const int j = threadIdx.x % ns, h = threadIdx.x / ns, hr = h / RS, r0 = RG * (h % RS);
  const int rw = (rb + nh - 1) / nh, ib = min(rb, hr * rw), ie = min(rb, ib + rw);
  const bool act = hr < nh && j < n;
  P acc[RG][IL];
#pragma unroll
  for (int c = 0; c < RG; c++)
#pragma unroll
    for (int q = 0; q < IL; q++) acc[c][q] = P(0);
  if (act) {
    const P* col = X + j * kXld;
    const P* xr = xg + r0;
    int i = ib;
    for (; i + 4 <= ie; i += 4)
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const P l = col[i + q];
        P xv[RG];
        load_vec<P, RG>(xr + (i + q) * NR, xv);
#pragma unroll
        for (int c = 0; c < RG; c++) acc[c][q % IL] += l * xv[c];
      }
    for (; i < ie; i++) {
      const P l = col[i];
#pragma unroll
      for (int c = 0; c < RG; c++) acc[c][0] += l * xr[i * NR + c];
    }
  }
  P v[RG];
#pragma unroll
  for (int c = 0; c < RG; c++) {
    if constexpr (IL == 4) v[c] = (acc[c][0] + acc[c][1]) + (acc[c][2] + acc[c][3]);
    else v[c] = acc[c][0];
  }
  if (act && hr > 0)
#pragma unroll
    for (int c = 0; c < RG; c++) hred[((hr - 1) * NR + r0 + c) * ns + j] = v[c];
  __syncthreads();
  if (act && hr == 0) {
    double* out = part + ((int64_t)blockIdx.x * nrhs + c0) * W;
    for (int hh = 1; hh < nh; hh++)
#pragma unroll
      for (int c = 0; c < RG; c++) v[c] += hred[((hh - 1) * NR + r0 + c) * ns + j];
#pragma unroll
    for (int c = 0; c < RG; c++)
      if (r0 + c < nr) out[(int64_t)(r0 + c) * W + j] = (double)v[c];
  }
  if constexpr (MODE != kSplit) {
    P* r = hred + 96 * NR + 448;  // w_s - sum of the partials
    P* xo = r + up4(n * NR);
    P* red = xo + up4(n * NR);
    const int nq = (max(u, 1) + kSolveRows - 1) / kSolveRows;
    const int first = (int)blockIdx.x - tk.y / kSolveRows;
    // one group: the supernode's own counter; several: its first task's, per group (solve_shape
    // launches several only where that many counters exist)
    int* counter = arrive + (gridDim.y == 1 ? tk.x : (int)(blockIdx.y * gridDim.x) + first);
    if (!last_arrival(counter, nq)) return;
    // kLeaf: Y over X, no longer read (kNarrow: X is free and holds the sums' parts)
    if (MODE == kLeaf) stage_dinv(Ys, reinterpret_cast<const P*>(d.dinv), n);
    sum_partials<P, NR, T>(d, w, ldv, c0, nr, part + ((int64_t)first * nrhs + c0) * W,
                           (int64_t)W * nrhs, W, nq,
                           reinterpret_cast<double*>(MODE == kNarrow ? X : hred), r);
    if (MODE == kLeaf) cp_async_wait_all();
    __syncthreads();
    dinv_apply<false, P, NR, T>(Ys, r, xo, red, n);
    for (int idx = threadIdx.x; idx < n * nr; idx += T) {
      const int c = idx / n, jj = idx - c * n;
      w[(int64_t)(c0 + c) * ldv + d.col0 + jj] = xo[jj * NR + c];
    }
  }
}

// x_s = Y^T (w_s - sum of s's partial sums) of every supernode of a level (POTRF tasks
// {s, first backward task, backward tasks, -}; bwd0: the level's first): the backward's kSplit.
template <typename P, int NR>
__global__ void __launch_bounds__(kWideThreads)
    k_bwd_diag(const int4* __restrict__ tasks, const SnDev* __restrict__ sns, int64_t ldv, int nrhs,
               int W, int64_t bwd0, double* w, const double* part) {
  constexpr int T = kWideThreads;
  extern __shared__ __align__(16) double sm[];
  start_next_level(nrhs);
  const int4 tk = tasks[blockIdx.x];
  const SnDev d = sns[tk.x];
  const int n = d.n, c0 = blockIdx.y * NR, nr = min(NR, nrhs - c0);
  double* hd = sm;  // T sums
  P* Ys = reinterpret_cast<P*>(sm + T);
  P* r = Ys + up4(n * (n + 1));
  P* xo = r + up4(n * NR);
  P* red = xo + up4(n * NR);
  stage_dinv(Ys, reinterpret_cast<const P*>(d.dinv), n);
  pdl_wait();  // the level's partial sums are in place
  sum_partials<P, NR, T>(d, w, ldv, c0, nr, part + ((tk.y - bwd0) * nrhs + c0) * W, (int64_t)W * nrhs,
                         W, tk.z, hd, r);
  cp_async_wait_all();
  __syncthreads();
  dinv_apply<false, P, NR, T>(Ys, r, xo, red, n);
  for (int idx = threadIdx.x; idx < n * nr; idx += T) {
    const int c = idx / n, jj = idx - c * n;
    w[(int64_t)(c0 + c) * ldv + d.col0 + jj] = xo[jj * NR + c];
  }
}

// ---- solves by substitution: factors without Y (wider than kDinvMaxWidth) ------------------
// The same tasks and arithmetic by a warp-level substitution with L11, NR right-hand sides per
// pass, kSolveThreads threads, the panel read from global memory with eight or more loads in
// flight per thread.
// Shared memory in P elements: forward L11 n*n, rdiag n, xs n*nrhs; backward the larger of
// that and xg kSolveRows*nrhs, hred T*NR.
static inline size_t fwd_sub_elems(int n, int nrhs) { return (size_t)n * n + n + (size_t)n * nrhs; }
static inline size_t bwd_sub_elems(int n, int nrhs, int nr) {
  return std::max((size_t)kSolveRows * nrhs + (size_t)kSolveThreads * nr, fwd_sub_elems(n, nrhs));
}

template <typename P, bool OWNER, int NR>
__global__ void __launch_bounds__(kSolveThreads)
    k_fwd_sub(const int4* __restrict__ tasks, const SnDev* __restrict__ sns, int64_t ldv, int nrhs,
              double* __restrict__ y, double* __restrict__ w, double* __restrict__ fstage) {
  constexpr int T = kSolveThreads, IL = NR == 1 ? 4 : 1;
  extern __shared__ __align__(16) double sm[];
  const int4 tk = tasks[blockIdx.x];
  const SnDev d = sns[tk.x];
  const int n = d.n, m = d.m, u = m - n;
  const int rb = min(kSolveRows, u - tk.y);  // <= 0 for a supernode without rows below
  P* L11 = reinterpret_cast<P*>(sm);
  P* rdiag = L11 + n * n;
  P* xs = rdiag + n;
  for (int idx = threadIdx.x; idx < n * nrhs; idx += T) {
    const int c = idx / n, j = idx - c * n;
    xs[idx] = (P)y[c * ldv + d.col0 + j];
  }
  load_l11<P>(d, L11, rdiag);
  warp_trisolve<true>(L11, rdiag, xs, n, nrhs);
  __syncthreads();
  if (tk.y == 0)
    for (int idx = threadIdx.x; idx < n * nrhs; idx += T) {
      const int c = idx / n, j = idx - c * n;
      w[c * ldv + d.col0 + j] = xs[idx];
    }
  const int i = threadIdx.x;
  if (i >= rb) return;
  const int64_t grow = d.rows[n + tk.y + i];
  const P* L = reinterpret_cast<const P*>(d.L) + n + tk.y + i;
  for (int c0 = 0; c0 < nrhs; c0 += NR) {
    P acc[NR][IL];
#pragma unroll
    for (int c = 0; c < NR; c++)
#pragma unroll
      for (int q = 0; q < IL; q++) acc[c][q] = P(0);
    constexpr int QB = (sizeof(P) == 4 && NR == 1) ? 16 : 8;  // independent loads per step
    int j = 0;
    for (; j + QB <= n; j += QB) {
      P l[QB];
#pragma unroll
      for (int q = 0; q < QB; q++) l[q] = L[(int64_t)(j + q) * m];
#pragma unroll
      for (int q = 0; q < QB; q++)
#pragma unroll
        for (int c = 0; c < NR; c++)
          if (c0 + c < nrhs) acc[c][q % IL] += l[q] * xs[(c0 + c) * n + j + q];
    }
    for (; j < n; j++) {
      const P l = L[(int64_t)j * m];
#pragma unroll
      for (int c = 0; c < NR; c++)
        if (c0 + c < nrhs) acc[c][0] += l * xs[(c0 + c) * n + j];
    }
#pragma unroll
    for (int c = 0; c < NR; c++) {
      if (c0 + c >= nrhs) continue;
      P v = acc[c][0];
      if constexpr (IL == 4) v = (acc[c][0] + acc[c][1]) + (acc[c][2] + acc[c][3]);
      if (OWNER) fstage[((int64_t)blockIdx.x * kSolveRows + i) * nrhs + c0 + c] = (double)v;
      else red_add(&y[(int64_t)(c0 + c) * ldv + grow], -(double)v);
    }
  }
}

template <typename P, int NR>
__global__ void __launch_bounds__(kSolveThreads)
    k_bwd_sub(const int4* __restrict__ tasks, const SnDev* __restrict__ sns, int64_t ldv, int nrhs,
              int W, double* __restrict__ w, double* __restrict__ part, int* __restrict__ arrive) {
  constexpr int T = kSolveThreads, IL = NR == 1 ? 4 : 1;
  extern __shared__ __align__(16) double sm[];
  const int4 tk = tasks[blockIdx.x];
  const SnDev d = sns[tk.x];
  const int n = d.n, m = d.m, u = m - n;
  const int rb = max(0, min(kSolveRows, u - tk.y));
  P* xg = reinterpret_cast<P*>(sm);  // rb x nrhs
  P* hred = xg + kSolveRows * nrhs;   // row groups' partial sums
  for (int idx = threadIdx.x; idx < rb * nrhs; idx += T) {
    const int c = idx / rb, i = idx - c * rb;
    xg[idx] = (P)w[c * ldv + d.rows[n + tk.y + i]];
  }
  __syncthreads();
  double* out = part + (int64_t)blockIdx.x * W * nrhs;
  // column slots rounded up to whole warps, so that no warp straddles two row groups
  const int ns = (n + 31) & ~31, ng = max(1, min(8, T / ns));
  const int j = threadIdx.x % ns, h = threadIdx.x / ns;
  const int rw = (rb + ng - 1) / ng, ib = min(rb, h * rw), ie = min(rb, ib + rw);
  const bool act = h < ng && j < n;
  for (int c0 = 0; c0 < nrhs; c0 += NR) {
    P acc[NR][IL];
#pragma unroll
    for (int c = 0; c < NR; c++)
#pragma unroll
      for (int q = 0; q < IL; q++) acc[c][q] = P(0);
    if (act) {
      const P* col = reinterpret_cast<const P*>(d.L) + (int64_t)j * m + n + tk.y;
      constexpr int QB = (sizeof(P) == 4 && NR == 1) ? 16 : 8;  // independent loads per step
      int i = ib;
      for (; i + QB <= ie; i += QB) {
        P l[QB];
#pragma unroll
        for (int q = 0; q < QB; q++) l[q] = col[i + q];
#pragma unroll
        for (int q = 0; q < QB; q++)
#pragma unroll
          for (int c = 0; c < NR; c++)
            if (c0 + c < nrhs) acc[c][q % IL] += l[q] * xg[(c0 + c) * rb + i + q];
      }
      for (; i < ie; i++) {
        const P l = col[i];
#pragma unroll
        for (int c = 0; c < NR; c++)
          if (c0 + c < nrhs) acc[c][0] += l * xg[(c0 + c) * rb + i];
      }
    }
    P v[NR];
#pragma unroll
    for (int c = 0; c < NR; c++) {
      if constexpr (IL == 4) v[c] = (acc[c][0] + acc[c][1]) + (acc[c][2] + acc[c][3]);
      else v[c] = acc[c][0];
    }
    if (ng > 1) {
      if (act && h > 0)
#pragma unroll
        for (int c = 0; c < NR; c++) hred[((h - 1) * NR + c) * n + j] = v[c];
      __syncthreads();
      if (act && h == 0)
        for (int hh = 1; hh < ng; hh++)
#pragma unroll
          for (int c = 0; c < NR; c++) v[c] += hred[((hh - 1) * NR + c) * n + j];
    }
    if (act && h == 0) {
#pragma unroll
      for (int c = 0; c < NR; c++)
        if (c0 + c < nrhs) out[(c0 + c) * W + j] = (double)v[c];
    }
    if (ng > 1) __syncthreads();
  }
  const int nq = (max(u, 1) + kSolveRows - 1) / kSolveRows;
  if (!last_arrival(&arrive[tk.x], nq)) return;
  P* r = reinterpret_cast<P*>(sm) + n * n + n;  // after L11 and rdiag, over the arrays above
  const double* pp0 = part + (int64_t)((int)blockIdx.x - tk.y / kSolveRows) * W * nrhs;
  const int64_t ps = (int64_t)W * nrhs;
  for (int idx = threadIdx.x; idx < n * nrhs; idx += T) {
    const int c = idx / n, jj = idx - c * n;
    const double* pp = pp0 + c * W + jj;
    double a[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int q = 0;
    for (; q + 8 <= nq; q += 8) {
#pragma unroll
      for (int t = 0; t < 8; t++) a[t] += __ldcg(pp + (q + t) * ps);
    }
    for (; q < nq; q++) a[0] += __ldcg(pp + q * ps);
    r[idx] = (P)(w[c * ldv + d.col0 + jj] -
                 (((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]))));
  }
  load_l11<P>(d, reinterpret_cast<P*>(sm), reinterpret_cast<P*>(sm) + n * n);
  warp_trisolve<false>(reinterpret_cast<const P*>(sm), reinterpret_cast<const P*>(sm) + n * n, r, n,
                       nrhs);
  __syncthreads();
  for (int idx = threadIdx.x; idx < n * nrhs; idx += T) {
    const int c = idx / n, jj = idx - c * n;
    w[c * ldv + d.col0 + jj] = r[idx];
  }
}

// ---- launchers ---------------------------------------------------------------------------------
static inline int grid_for(int64_t total) {
  return (int)std::min<int64_t>((total + 255) / 256, 152 * 8);
}

void launch_gather_perm(const double* B, int64_t ldb, const int32_t* perm, const double* scale,
                        int64_t n, int nrhs, double* y, cudaStream_t st) {
  if (n <= 0) return;
  k_gather_perm<<<grid_for(n * nrhs), 256, 0, st>>>(B, ldb, perm, scale, n, nrhs, y);
}

void launch_scatter_perm(const double* w, const int32_t* perm, const double* scale, int64_t n,
                         int nrhs, double* X, int64_t ldx, cudaStream_t st) {
  if (n <= 0) return;
  k_scatter_perm<<<grid_for(n * nrhs), 256, 0, st>>>(w, perm, scale, n, nrhs, X, ldx);
}

struct FwdArgs {
  const int4 *tasks, *diag;
  int ntasks, nsup;
  const SnDev* sns;
  int64_t ldv;
  int nrhs, W;
  double *y, *w, *fstage;
  cudaStream_t st;
};
struct BwdArgs {
  const int4 *tasks, *diag;
  int ntasks, nsup;
  int64_t bwd0;
  const SnDev* sns;
  int64_t ldv;
  int nrhs, W, wl;
  double *w, *part;
  int* arrive;
  cudaStream_t st;
};

template <typename P, int NR>
static void fwd_y_nr(const FwdArgs& a, const SolveShape& s) {
  auto go = [&](auto mode) {
    constexpr int M = decltype(mode)::value;
    launch_pdl(k_fwd_y<P, NR, M>, dim3(a.ntasks, s.groups), y_threads<M>(),
               fwd_y_elems<NR, M>(a.W) * sizeof(P), a.st, a.tasks, a.sns, a.ldv, a.nrhs, a.y, a.w,
               a.fstage);
  };
  if (s.mode == kSplit) go(std::integral_constant<int, kSplit>());
  else if (s.mode == kNarrow) go(std::integral_constant<int, kNarrow>());
  else go(std::integral_constant<int, kLeaf>());
}
template <typename P, int NR>
static void bwd_y_nr(const BwdArgs& a, const SolveShape& s) {
  auto go = [&](auto mode, int groups, int cfirst) {
    constexpr int M = decltype(mode)::value;
    launch_pdl(k_bwd_y<P, NR, M>, dim3(a.ntasks, groups), y_threads<M>(),
               bwd_y_elems<NR, M>(a.wl) * sizeof(P), a.st, a.tasks, a.sns, a.ldv, a.nrhs, cfirst, a.W,
               a.w, a.part, a.arrive);
  };
  for (int p = 0; p < s.groups; p += s.bwd_groups) {
    if (s.mode == kSplit) go(std::integral_constant<int, kSplit>(), s.bwd_groups, p * NR);
    else if (s.mode == kNarrow) go(std::integral_constant<int, kNarrow>(), s.bwd_groups, p * NR);
    else go(std::integral_constant<int, kLeaf>(), s.bwd_groups, p * NR);
  }
}

// f(integral constant NR) for the shape's NR
template <typename F>
static void with_nr(int nr, F f) {
  switch (nr) {
    case 1: f(std::integral_constant<int, 1>()); break;
    case 2: f(std::integral_constant<int, 2>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 8: f(std::integral_constant<int, 8>()); break;
    case 12: f(std::integral_constant<int, 12>()); break;
    default: f(std::integral_constant<int, 16>()); break;
  }
}

// Right-hand sides per pass of the substitution kernels: all of them, so that a task reads its panel
// once (27-point 20^3, widths up to 128, FP64: 16 right-hand sides 13.2 ms in one pass, 13.9 in
// two; 32 26.3 ms in one, 27.3 in four).
static inline int rhs_pass(int nrhs) {
  return nrhs <= 1 ? 1 : nrhs <= 4 ? 4 : nrhs <= 8 ? 8 : nrhs <= 16 ? 16 : 32;
}
template <typename P, int NR>
static void fwd_sub_nr(const FwdArgs& a) {
  const size_t sm = fwd_sub_elems(a.W, a.nrhs) * sizeof(P);
  if (a.fstage)
    k_fwd_sub<P, true, NR><<<a.ntasks, kSolveThreads, sm, a.st>>>(a.tasks, a.sns, a.ldv, a.nrhs, a.y,
                                                                  a.w, a.fstage);
  else
    k_fwd_sub<P, false, NR><<<a.ntasks, kSolveThreads, sm, a.st>>>(a.tasks, a.sns, a.ldv, a.nrhs,
                                                                   a.y, a.w, nullptr);
}
template <typename P, int NR>
static void bwd_sub_nr(const BwdArgs& a) {
  const size_t sm = bwd_sub_elems(a.wl, a.nrhs, NR) * sizeof(P);
  k_bwd_sub<P, NR><<<a.ntasks, kSolveThreads, sm, a.st>>>(a.tasks, a.sns, a.ldv, a.nrhs, a.W, a.w,
                                                          a.part, a.arrive);
}

template <typename P>
static void fwd_p(const FwdArgs& a, bool inv, int64_t counters) {
  if (!inv) {
    switch (rhs_pass(a.nrhs)) {
      case 1: fwd_sub_nr<P, 1>(a); break;
      case 4: fwd_sub_nr<P, 4>(a); break;
      case 8: fwd_sub_nr<P, 8>(a); break;
      case 16: fwd_sub_nr<P, 16>(a); break;
      default: fwd_sub_nr<P, 32>(a); break;
    }
    return;
  }
  const SolveShape s = solve_shape(a.nrhs, a.ntasks, a.nsup, counters);
  if (s.mode == kSplit)
    with_nr(fill_nr(a.nrhs, a.nsup, 2 * kWave), [&](auto nr) {
      constexpr int NR = decltype(nr)::value;
      launch_pdl(k_fwd_diag<P, NR>, dim3(a.nsup, (a.nrhs + NR - 1) / NR), kWideThreads,
                 diag_y_elems<NR>(a.W) * sizeof(P), a.st, a.diag, a.sns, a.ldv, a.nrhs, a.y, a.w);
    });
  with_nr(s.nr, [&](auto nr) { fwd_y_nr<P, decltype(nr)::value>(a, s); });
}
template <typename P>
static void bwd_p(const BwdArgs& a, bool inv, int64_t counters) {
  if (!inv) {
    switch (rhs_pass(a.nrhs)) {
      case 1: bwd_sub_nr<P, 1>(a); break;
      case 4: bwd_sub_nr<P, 4>(a); break;
      case 8: bwd_sub_nr<P, 8>(a); break;
      case 16: bwd_sub_nr<P, 16>(a); break;
      default: bwd_sub_nr<P, 32>(a); break;
    }
    return;
  }
  const SolveShape s = solve_shape(a.nrhs, a.ntasks, a.nsup, counters);
  with_nr(s.nr, [&](auto nr) { bwd_y_nr<P, decltype(nr)::value>(a, s); });
  if (s.mode == kSplit)
    with_nr(fill_nr(a.nrhs, a.nsup, 2 * kWave), [&](auto nr) {
      constexpr int NR = decltype(nr)::value;
      launch_pdl(k_bwd_diag<P, NR>, dim3(a.nsup, (a.nrhs + NR - 1) / NR), kWideThreads,
                 diag_y_elems<NR>(a.wl) * sizeof(P), a.st, a.diag, a.sns, a.ldv, a.nrhs, a.W, a.bwd0,
                 a.w, a.part);
    });
}

void launch_fwd(const int4* tasks, int ntasks, const int4* diag, int nsup, const SnDev* sns,
                int64_t ldv, int nrhs, int W, double* y, double* w, double* fstage,
                int64_t counters, bool inv, bool f32, cudaStream_t st) {
  if (ntasks <= 0) return;
  const FwdArgs a{tasks, diag, ntasks, nsup, sns, ldv, nrhs, W, y, w, fstage, st};
  if (f32) fwd_p<float>(a, inv, counters);
  else fwd_p<double>(a, inv, counters);
}

void launch_fwd_gather(const int32_t* fg_row, const int64_t* fg_ptr, const int32_t* fg_ent,
                       int64_t nrows, int64_t ldv, int nrhs, const double* fstage, double* y,
                       cudaStream_t st) {
  if (nrows <= 0) return;
  int blocks = (int)std::min<int64_t>((nrows + 127) / 128, 152 * 8);
  k_fwd_gather<<<blocks, 128, 0, st>>>(fg_row, fg_ptr, fg_ent, nrows, ldv, nrhs, fstage, y);
}

void launch_bwd(const int4* tasks, int ntasks, const int4* diag, int nsup, int64_t bwd0,
                const SnDev* sns, int64_t ldv, int nrhs, int W, int wl, double* w, double* part,
                int* arrive, int64_t counters, bool inv, bool f32, cudaStream_t st) {
  if (ntasks <= 0) return;
  const BwdArgs a{tasks, diag, ntasks, nsup, bwd0, sns, ldv, nrhs, W, wl, w, part, arrive, st};
  if (f32) bwd_p<float>(a, inv, counters);
  else bwd_p<double>(a, inv, counters);
}

template <typename K>
static bool set_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) ==
         cudaSuccess;
}

template <typename P, int NR, int MODE>
static bool set_y_mode() {
  return set_smem(k_fwd_y<P, NR, MODE>, fwd_y_elems<NR, MODE>(kDinvMaxWidth) * sizeof(P)) &&
         set_smem(k_bwd_y<P, NR, MODE>, bwd_y_elems<NR, MODE>(kDinvMaxWidth) * sizeof(P));
}
template <typename P, int NR>
static bool set_y_nr() {
  const size_t dg = diag_y_elems<NR>(kDinvMaxWidth) * sizeof(P);
  return set_y_mode<P, NR, kLeaf>() && set_y_mode<P, NR, kNarrow>() && set_y_mode<P, NR, kSplit>() &&
         set_smem(k_fwd_diag<P, NR>, dg) && set_smem(k_bwd_diag<P, NR>, dg);
}

template <typename P, int NR>
static bool set_sub_nr(int W, int max_nrhs) {
  const size_t f = fwd_sub_elems(W, max_nrhs) * sizeof(P);
  return set_smem(k_fwd_sub<P, false, NR>, f) && set_smem(k_fwd_sub<P, true, NR>, f) &&
         set_smem(k_bwd_sub<P, NR>, bwd_sub_elems(W, max_nrhs, NR) * sizeof(P));
}

template <typename P>
static bool set_solve_p(int W, int max_nrhs) {
  bool ok = set_sub_nr<P, 1>(W, max_nrhs) && set_sub_nr<P, 4>(W, max_nrhs) &&
            set_sub_nr<P, 8>(W, max_nrhs) && set_sub_nr<P, 16>(W, max_nrhs) &&
            set_sub_nr<P, 32>(W, max_nrhs);
  for (int nr : kNrList)
    with_nr(nr, [&](auto c) {
      ok = ok && set_y_nr<P, decltype(c)::value>();
    });
  return ok;
}

int set_solve_kernel_attrs(int W, int max_nrhs) {
  return set_solve_p<double>(W, max_nrhs) && set_solve_p<float>(W, max_nrhs) ? CHOL_OK
                                                                             : CHOL_E_CUDA;
}

}  // namespace chol
