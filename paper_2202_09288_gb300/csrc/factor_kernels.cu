// factor_kernels.cu -- sm_103a kernels of the per-level supernodal factorization.
//
// The paper's factorization (Sec. 3, Listing 1) applies to every supernode the SYRK and
// GEMM updates of the supernodes that precede it, serializes their assembly with a lock,
// then runs POTRF on the diagonal block and TRSM on the rows below.  Here the same
// arithmetic is reorganized right-looking over the level sets of the supernodal
// elimination tree (Sec. 3, Fig. 1): all supernodes of a level are independent, so one
// launch factors every diagonal block of the level (POTRF), one solves all off-diagonal
// rows (TRSM), and one forms every Schur update U_s = L21 L21^T in tiles (the SYRK and
// GEMM of Listing 1) and subtracts it from the ancestor panels.  The lock becomes either
// device atomics or an owner-pulls assembly in a fixed order.
//
// FP64 throughput on GB300 is ~1 TFLOP/s for both FMA instructions and the FP64 `mma.sync` (DMMA);
// the 64-, 32- and 16-wide Schur tiles here use m8n8k4 DMMA (an eighth of the instructions and of the
// shared-memory loads), the 128-wide ones the bf16 tensor cores (oz_kernels.cu).
#include <cuda_runtime.h>

#include <algorithm>

#include "chol_internal.h"
#include "kernels.h"
#include "launch_util.h"
#include "device_common.cuh"
#include "oz_common.cuh"

namespace chol {

// ---- assembly of A into the zeroed panels ------------------------------------------------
template <typename T>
__global__ void k_assemble(const double* __restrict__ vals, const int64_t* __restrict__ amap,
                           int64_t nnz, T* __restrict__ L) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nnz;
       p += (int64_t)gridDim.x * blockDim.x)
    L[amap[p]] = (T)vals[p];
}

// ---- diagonal-block Cholesky ---------------------------------------------------------------
// Cost model on this part (measured): a warp's FP64 instruction takes ~65 cycles, dependent or not;
// an SM's FP64 unit takes one per 19 cycles from all its warps together (so eight busy warps wait
// ~150 cycles each); the library's double sqrt and reciprocal take ~690 and ~440 cycles.  The
// factorization is therefore organized so that (a) the serial per-column chain holds as
// few FP64 instructions as possible and (b) the bulk of the work runs with every lane busy.

// FMA in the block's precision.
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }

// y = p^{-1/2} of a positive normal pivot: an FP32 seed y0 and one third-order correction.
// With r = 1 - p y0^2, p^{-1/2} = y0 (1 - r)^{-1/2} = y0 (1 + r/2 + 3r^2/8 + O(r^3)); the seed
// has |r| < 2^-20, so the dropped term is below 2^-58 relative, and the result is within an
// ulp or so.  p is first scaled by an even power of two into [1, 4) with integer exponent
// arithmetic (no FP32 overflow or underflow) and the result scaled back the same way; the
// FP32 <-> FP64 conversions are integer arithmetic too (exact, but for the seed's argument,
// truncated to 24 bits): four FP64 instructions in all, where each conversion would be one more
// of ~64 cycles on the serial chain.  Subnormal, infinite and NaN p take the library path.
__device__ __forceinline__ double widen_normal(float x) {  // a positive normal float
  const uint32_t b = __float_as_uint(x);
  return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}
__device__ __forceinline__ double pivot_rsqrt(double p) {
  const int hi = __double2hiint(p), lo = __double2loint(p);
  const int ebits = (hi >> 20) & 0x7ff;
  if (ebits == 0 || ebits == 0x7ff) return 1.0 / sqrt(p);
  const int s = (ebits - 1023) & ~1;  // even, so that p 2^-s lies in [1, 4)
  const int his = hi - s * (1 << 20);
  const double ps = __hiloint2double(his, lo);
  const float y0f = rsqrtf(__uint_as_float((((uint32_t)his - 0x38000000u) << 3) | ((uint32_t)lo >> 29)));
  const double y0 = widen_normal(y0f), c1 = widen_normal(0.5f * y0f), c2 = widen_normal(0.375f * y0f);
  const double h = ps * y0;
  const double r = fma(-h, y0, 1.0);
  const double q = fma(r, c2, c1);  // y0/2 + 3 y0 r / 8
  const double y = fma(q, r, y0);
  return __hiloint2double(__double2hiint(y) - (s / 2) * (1 << 20), __double2loint(y));
}
// FP32: the hardware estimate and one Newton step.
__device__ __forceinline__ float pivot_rsqrt(float p) {
  const float y0 = rsqrtf(p);
  const float r = fmaf(-p * y0, y0, 1.f);
  return fmaf(0.5f * y0, r, y0);
}
// p > 0 without the FP64 unit (NaN and zero of either sign are not)
__device__ __forceinline__ bool positive(double p) {
  const long long b = __double_as_longlong(p);
  return b > 0 && b <= 0x7ff0000000000000ll;
}

// Threads of a POTRF CTA: warp 0 finishes the next column, the others update the trailing
// triangle (potrf_lookahead).
constexpr int kPotrfThreads = 256;
// POTRF launches of at most this many CTAs, one per SM, let the next kernel start early.  A larger
// one still has CTAs to place, and the next kernel's would take the places of its second wave: 200
// supernodes of 40 columns 78 us per factorization in FP64 (79 in FP32) with the early start, 65
// (61) without.
constexpr unsigned kPotrfEarly = 152;

// Position table of the trailing update: the lower triangle of columns 2..n-1 taken column by
// column from the last (column n-1: 1 entry, column n-2: 2, ...), entry (C << 8) | R.  At step j
// the entries of columns j+2..n-1 are the first (n-j-2)(n-j-1)/2, so every step's work is a
// prefix, dealt evenly over the threads, and no index arithmetic is repeated per step.
__device__ __forceinline__ void build_update_table(uint16_t* tab, int n) {
  const int mm = n - 2, tot = mm > 0 ? mm * (mm + 1) / 2 : 0;
  for (int e = threadIdx.x; e < tot; e += blockDim.x) {
    int cc = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    if (cc * (cc + 1) / 2 > e) cc--;
    else if ((cc + 1) * (cc + 2) / 2 <= e) cc++;
    const int C = n - 1 - cc, R = C + (e - cc * (cc + 1) / 2);
    tab[e] = (uint16_t)((C << 8) | R);
  }
}
__host__ __device__ constexpr size_t update_table_bytes(int w) {
  return w > 2 ? (size_t)(w - 2) * (w - 1) / 2 * sizeof(uint16_t) : 0;
}

// The mixed kernel's table follows the FP64 block of a redo, which overlays the FP32 one (leading
// dimension 64 up to 64 columns: 64 n floats)
__host__ __device__ constexpr size_t potrf_mixed_tab_offset(int w) {
  return (size_t)w * w * sizeof(double) > (size_t)64 * 64 * sizeof(float)
             ? (size_t)w * w * sizeof(double)
             : (size_t)64 * 64 * sizeof(float);
}

// Right-looking Cholesky of the n x n block A (shared memory, column-major A[c * n + r]; only
// the lower triangle is read or written; n <= 128) with a one-column lookahead and one barrier
// per column: blocks wider than 64, and the FP64 redo of the mixed factor.  Step j (column j
// final and scaled): warp 0 finishes column j+1 in registers --
// its update by column j, the pivot (a shuffle from the lane holding the diagonal), its
// reciprocal square root, the scaling (the diagonal becomes p y = sqrt(p)) -- while the other
// warps apply column j to columns j+2..n-1 through the position table (build_update_table),
// four elements per thread in flight.  Returns the first column whose pivot fails accept(p),
// else n.  A failed pivot does not stop the loop (every thread passes the same barriers); the
// caller discards the block.
template <typename T, typename Accept>
__device__ int potrf_lookahead(T* A, int n, const uint16_t* tab, Accept accept) {
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nupd = blockDim.x - 32;  // threads of the trailing update
  int bad = n;
  if (warp == 0) {
    T v[4];
#pragma unroll
    for (int g = 0; g < 4; g++) {
      if (32 * g >= n) break;
      const int r = 32 * g + lane;
      v[g] = r < n ? A[r] : T(0);
    }
    const T p = __shfl_sync(0xffffffffu, v[0], 0);
    const T y = pivot_rsqrt(p);
    if (!accept(p)) bad = 0;
#pragma unroll
    for (int g = 0; g < 4; g++) {
      if (32 * g >= n) break;
      const int r = 32 * g + lane;
      if (r < n) A[r] = v[g] * y;
    }
  }
  __syncthreads();
  for (int j = 0; j + 1 < n; j++) {
    const T* lj = A + j * n;
    if (warp == 0) {
      const int c = j + 1;
      T* ac = A + c * n;
      const T lc = lj[c];
      T v[4];
#pragma unroll
      for (int g = 0; g < 4; g++) {
        if (c + 32 * g >= n) break;
        const int r = c + 32 * g + lane;
        v[g] = r < n ? fma_t(-lj[r], lc, ac[r]) : T(0);
      }
      const T p = __shfl_sync(0xffffffffu, v[0], 0);  // lane 0 holds row c
      const T y = pivot_rsqrt(p);
      if (bad == n && !accept(p)) bad = c;
#pragma unroll
      for (int g = 0; g < 4; g++) {
        if (c + 32 * g >= n) break;
        const int r = c + 32 * g + lane;
        if (r < n) ac[r] = v[g] * y;
      }
    } else {
      const int m = n - j - 2, tot = m * (m + 1) / 2;
      for (int e0 = tid - 32; e0 < tot; e0 += 4 * nupd) {
        int pos[4];
        T lr[4], lcv[4], av[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const int e = e0 + q * nupd;
          pos[q] = -1;
          if (e < tot) {
            const int ent = tab[e], C = ent >> 8, R = ent & 255;
            pos[q] = C * n + R;
            lr[q] = lj[R];
            lcv[q] = lj[C];
            av[q] = A[pos[q]];
          }
        }
#pragma unroll
        for (int q = 0; q < 4; q++)
          if (pos[q] >= 0) A[pos[q]] = fma_t(-lr[q], lcv[q], av[q]);
      }
    }
    __syncthreads();
  }
  if (tid == 0) s_bad = bad;
  __syncthreads();
  return s_bad;
}

// What potrf_blocks leaves of Y = L11^-1 beside L11.
enum PotrfInverse { kInvBlocks, kInvFull };  // its 16 x 16 diagonal blocks, all of it

// ---- FP64 blocks up to 64 wide: 8 x 8 blocks on the FP64 matrix instruction -----------------------
// An SM's FP64 unit takes one FMA warp instruction per 16 to 19 cycles from all warps together and
// holds a single warp 65 cycles for each; an m8n8k4 product (256 multiply-adds, eight instructions'
// worth) takes 146 of the unit: no more arithmetic per cycle, but an eighth of the instructions and
// operand loads.  So the block is cut into 8 x 8 blocks: warp 0
// factors a diagonal block in registers, in the fewest dependent FP64 instructions, and everything
// else is 8 x 8 x 8 products, dealt over the other warps.  Layout: A[c * kPld + r], L in the
// lower triangle, Y in the blocks above it (Y[r, c] at A[r * kPld + c]), Y's diagonal 8 x 8
// blocks in Dv (row-major, zeros above the diagonal); kPld = 4 mod 16 doubles: the matrix
// operands' four columns of eight rows hit distinct banks.
constexpr int kPotrfWorkers = 4;
constexpr int kPld = 68;
constexpr size_t kPotrfBlkSmem = (64 * kPld + 8 * 64) * sizeof(double);

__device__ __forceinline__ void dmma_884(double (&c)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
               : "+d"(c[0]), "+d"(c[1])
               : "d"(a), "d"(b));
}

// 1 / p of a positive p with an exponent field in 3 .. 2043, in integer arithmetic (the FP64 unit is what the chain of pivots
// and the other warps' products compete for): with p = P 2^-52 2^x in [1, 2) 2^x and the FP32
// reciprocal z0 = m 2^-24 of p's leading bits, e = 1 - p z0 = E 2^-76 exactly, E = -P m mod 2^64
// (|e| < 2^-21, so |E| < 2^55), and 1/p = z0 (1 + e + e^2 + ...): z0 e in units of 2^-60 from
// E's upper bits, z0 e^2 from 24 x 23 bits, the dropped z0 e^3 < 2^-63; rounded to nearest (an error
// below 0.51 ulp).
__device__ __forceinline__ double pivot_rcp(double p) {
  const uint32_t hi = (uint32_t)__double2hiint(p), lo = (uint32_t)__double2loint(p);
  const int ebits = (int)(hi >> 20);
  const uint32_t ph = (hi & 0xfffffu) | 0x100000u;  // P = ph 2^32 + lo
  float z0;
  asm("rcp.approx.ftz.f32 %0, %1;"
      : "=f"(z0)
      : "f"(__uint_as_float(((hi << 3) & 0x7fffffu) | (lo >> 29) | 0x3f800000u)));
  const uint32_t zb = __float_as_uint(z0);  // in [0.5, 1]: exponent 126, or 1.0
  const uint32_t m = ((zb & 0x7fffffu) | 0x800000u) << ((zb >> 23) - 126u);
  unsigned long long pm = (unsigned long long)lo * m;
  pm += (unsigned long long)(ph * m) << 32;
  const long long E = -(long long)pm;
  const long long E16 = E >> 16;  // e in units of 2^-60
  const long long c1 = (long long)((unsigned long long)(uint32_t)E16 * m +
                                   ((unsigned long long)((uint32_t)(E16 >> 32) * m) << 32)) >> 24;
  const long long c2 = ((long long)(int)(c1 >> 14) * (int)(E >> 32)) >> 30;
  const unsigned long long Z = ((unsigned long long)m << 36) + (unsigned long long)(c1 + c2) + 64ull;
  // Z 2^-60 in [0.5, 1]: the 53-bit integer part of Z / 2^7 carries into the exponent
  const long long bits = (long long)(Z >> 7) + (1021ll << 52) - ((long long)(ebits - 1023) << 52);
  return __longlong_as_double(bits);
}

// One warp: Cholesky of the 8 x 8 diagonal block at column b of A, and its inverse into Dv.
// Lane (r, g): row r, columns g and g + 4.  Gaussian elimination with the pivots' reciprocals
// z_j: row r > j takes v_rc -= t u_c, t = v_rj z_j, where u_c is the pivot row's value: a_jc = a_cj
// right of column j; left of it the register of the eliminated column c holds M^-1 (M the unit
// lower factor), whose row j gives u_c, and v_rj becomes -t.  The square roots come at the end,
// all eight at once: L_rj = a_rj y_j and (L^-1)_rc = y_r (M^-1)_rc with y = p^{-1/2}.
// nc: the block's columns from b on (past them it is padded, which takes no steps: the
// factorization of 5,000 one-column supernodes 75 -> 48 us; column by column it took 57).  Returns the first j whose pivot is not positive, else 8;
// *lossy (shared memory): a pivot fell below half of its diagonal entry (see refined_quotient).
__device__ __forceinline__ int potrf_diag8(double* A, double* Dv, int b, int nc, int* lossy) {
  const int lane = threadIdx.x & 31, r = lane & 7, g = lane >> 3;
  constexpr unsigned full = 0xffffffffu;
  double v[2], raw[2] = {0.0, 0.0}, prow = 1.0;
#pragma unroll
  for (int s = 0; s < 2; s++) {
    const int c = g + 4 * s;
    v[s] = r >= c ? A[(b + c) * kPld + b + r] : A[(b + r) * kPld + b + c];
  }
  const int dlo = __shfl_sync(full, __double2hiint(v[0]), 8 * (r & 3) + r);  // (r, r), r < 4
  const int dhi = __shfl_sync(full, __double2hiint(v[1]), 8 * (r & 3) + r);
  int bad = 8;
#pragma unroll
  for (int j = 0; j < 8; j++) {
    const int sj = j >> 2, gj = 8 * (j & 3);  // column j: register sj of the lanes gj + row
    const double p = __shfl_sync(full, v[sj], gj + j);
    double u[2];
#pragma unroll
    for (int s = 0; s < 2; s++) {
      const int c = g + 4 * s;
      const double right = __shfl_sync(full, v[sj], gj + c);
      const double left = __shfl_sync(full, v[s], 8 * g + j);
      u[s] = c > j ? right : left;
    }
    const double arj = __shfl_sync(full, v[sj], gj + r);
#pragma unroll
    for (int s = 0; s < 2; s++)
      if (g + 4 * s == j) raw[s] = v[s];
    if (r == j) prow = p;
    if (bad == 8 && !positive(p)) bad = j;
    if (j + 1 >= nc) break;
    // t = v_rj / p can neither overflow (v_rj^2 <= p v_rr) nor underflow for pivots and nonzero
    // v_rj in the middle of the exponent range
    const uint32_t phi = (uint32_t)__double2hiint(p) >> 20, ahi = (uint32_t)__double2hiint(arj) << 1;
    const bool tiny = ahi < (300u << 21) && (ahi | (uint32_t)__double2loint(arj)) != 0u;
    if (phi - 823u <= 400u && !__any_sync(full, tiny)) {
      const double t = arj * pivot_rcp(p);
#pragma unroll
      for (int q = 0; q < 2; q++) {
        const int s = q ^ ((j + 1) >> 2);  // the next pivot's column first
        const double x = fma(-t, u[s], v[s]);
        if (r > j) v[s] = g + 4 * s == j ? -t : x;
      }
    } else {  // by the square roots, over the whole range
      const double y = pivot_rsqrt(p), l = arj * y, t = l * y;
#pragma unroll
      for (int s = 0; s < 2; s++) {
        const int c = g + 4 * s;
        const double x = c > j ? fma(-l, u[s] * y, v[s]) : fma(-t, u[s], v[s]);
        if (r > j) v[s] = c == j ? -t : x;
      }
    }
  }
  const double y = pivot_rsqrt(prow);
#pragma unroll
  for (int s = 0; s < 2; s++) {
    const int c = g + 4 * s;
    const double l = raw[s] * __shfl_sync(full, y, c);
    const double w = v[s] * y;
    if (c <= r) A[(b + c) * kPld + b + r] = l;
    Dv[r * 8 + c] = c < r ? w : c == r ? y : 0.0;
  }
  // (high words: one exponent step is a factor of two)
  const bool small = __any_sync(full, __double2hiint(prow) + 0x100000ll < (r < 4 ? dlo : dhi));
  if (lane == 0) *lossy = small;
  return bad;
}

// One warp: the 8 x 8 x 8 product C += sgn P Q with P[r][k] at P[r * pr + k * pk] and
// Q[k][n] at Q[k * qk + n * qn]; C[r][n] at C[r * cr + n * cn], loaded first if ADD.
template <bool ADD, bool NEG>
__device__ __forceinline__ void block_product(double* C, int cr, int cn, const double* P, int pr,
                                              int pk, const double* Q, int qk, int qn) {
  const int lane = threadIdx.x & 31, r = lane >> 2, k = lane & 3;
  double a[2], b[2], c[2] = {0.0, 0.0};
#pragma unroll
  for (int s = 0; s < 2; s++) {
    a[s] = P[r * pr + (4 * s + k) * pk];
    b[s] = Q[(4 * s + k) * qk + r * qn];
    if (NEG) a[s] = -a[s];
  }
  double* c0 = C + r * cr + 2 * k * cn;
  if (ADD) {
    c[0] = c0[0];
    c[1] = c0[cn];
  }
  __syncwarp();  // C may be P or Q: every lane has read before any writes
  dmma_884(c, a[0], b[0]);
  dmma_884(c, a[1], b[1]);
  c0[0] = c[0];
  c0[cn] = c[1];
}

// One warp: X <- X D^{-T}, X[r][c] at X[r + c * kPld], D a diagonal block of L and W its inverse, as
// X0 = X W^T, R = X - X0 D^T, X0 + R W^T.  The product with the computed inverse alone leaves R of the
// order of 2^-53 |X| |D| |W| instead of substitution's 2^-53 |X0| |D|: for 16 columns with pairs
// dependent to 10^-5, |A - L L^T| was 5.5e-12 of the diagonal, 2.8e-16 by substitution, and is
// 3.3e-16 refined.  Taken where a pivot fell below half of its diagonal entry;
// otherwise the rows of D, scaled to unit length, have diagonals of at least 0.7 and the two
// agree to a small factor.  (Ratios of the 2D, 3D and 27-point workloads: 0.74 and more, so that
// their blocks never come here and their times are as before; diffusion with lognormal coefficients:
// a few blocks in a thousand.)
__device__ __noinline__ void refined_quotient(double* X, const double* W, const double* D) {
  const int lane = threadIdx.x & 31, r = lane >> 2, k = lane & 3;
  double* x = X + r + 2 * k * kPld;  // this lane's two entries of a product
  double c[2] = {x[0], x[kPld]}, x0[2], a[2], b[2];
  block_product<false, false>(X, 1, kPld, X, 1, kPld, W, 1, 8);
  __syncwarp();
#pragma unroll
  for (int s = 0; s < 2; s++) {
    x0[s] = x[s * kPld];
    a[s] = -X[r + (4 * s + k) * kPld];
    b[s] = r >= 4 * s + k ? D[(4 * s + k) * kPld + r] : 0.0;
  }
  __syncwarp();
  dmma_884(c, a[0], b[0]);
  dmma_884(c, a[1], b[1]);
  x[0] = c[0];
  x[kPld] = c[1];
  __syncwarp();
#pragma unroll
  for (int s = 0; s < 2; s++) {
    a[s] = X[r + (4 * s + k) * kPld];
    b[s] = W[r * 8 + 4 * s + k];
  }
  __syncwarp();
  dmma_884(x0, a[0], b[0]);
  dmma_884(x0, a[1], b[1]);
  x[0] = x0[0];
  x[kPld] = x0[1];
}

// Cholesky of the n x n block (n <= 64, padded to whole 8 x 8 blocks with the identity, the
// upper blocks zero) and Y.  Per block column p, one barrier of the CTA:
//   warp 0: the block below the diagonal one, L_{p+1,p} = A_{p+1,p} D_p^{-T} (D_p the diagonal
//   block, its inverse from potrf_diag8), then the next diagonal block's update and factor;
//   kPotrfWorkers warps: the other blocks of the column and the block row p of Y, Y_pc =
//   D_p^{-1} S_pc; then (a barrier of theirs that warp 0 only arrives at) the trailing update
//   A_ij -= L_ip L_jp^T and S_ic -= L_ip Y_pc (S_ic starts at 0, Y_pp = D_p^{-1}).
// More workers finish their products sooner but delay warp 0's chain at the FP64 unit they share.
// kInvBlocks: of Y only the blocks (p, p-1) of odd p, which complete 16 x 16 diagonal blocks.
// Returns the first column whose pivot is not positive, else n.
// Measured, one 64-wide block (one CTA): kInvBlocks 31 us, kInvFull 41 us with four workers (34 /
// 45 with three, 34 / 46 with seven); a column-by-column factorization at one barrier per
// column took 42 us, its in-place inverse 35 more.  Per 48^3 27-point factorization POTRF 19.8 ->
// 15.6 ms; 64 x 64 2D Laplacian step 0.70 -> 0.62 ms.
template <int INV, int WORKERS>
__device__ int potrf_blocks(double* A, double* Dv, int n) {
  __shared__ int s_bad, s_lossy[8];
  const int warp = threadIdx.x >> 5, nb = (n + 7) / 8;
  int bad = n;
  if (warp == 0) {
    const int q = potrf_diag8(A, Dv, 0, n, s_lossy);
    if (q < 8) bad = min(n, q);
  }
  __syncthreads();
  for (int p = 0; p < nb; p++) {
    const int below = nb - 1 - p;
    const double *D = Dv + 64 * p, *Lp = A + 8 * p * kPld + 8 * p;
    const bool lossy = s_lossy[p];
    if (warp == 0) {
      if (below > 0) {
        const int b = 8 * (p + 1);
        double* X = A + 8 * p * kPld + b;
        if (lossy) refined_quotient(X, D, Lp);
        else block_product<false, false>(X, 1, kPld, X, 1, kPld, D, 1, 8);
        __threadfence_block();
        __syncwarp();
        asm volatile("bar.arrive 1, %0;" ::"n"(32 * (WORKERS + 1)) : "memory");
        block_product<true, true>(A + b * kPld + b, 1, kPld, X, 1, kPld, X, kPld, 1);
        __syncwarp();
        const int q = potrf_diag8(A, Dv + 64 * (p + 1), b, n - b, s_lossy + p + 1);
        if (q < 8 && bad == n) bad = min(n, b + q);
      }
    } else if (warp <= WORKERS) {
      const int c0 = INV == kInvFull ? 0 : p & ~1;  // first block column of Y's row p
      const int nx = below > 0 ? below - 1 : 0;
      for (int q = warp - 1; q < nx + p - c0; q += WORKERS) {
        if (lossy) {  // (D^{-1} S = (S^T D^{-T})^T: the same strides)
          refined_quotient(A + 8 * p * kPld + 8 * (q < nx ? p + 2 + q : c0 + q - nx), D, Lp);
        } else if (q < nx) {
          double* X = A + 8 * p * kPld + 8 * (p + 2 + q);
          block_product<false, false>(X, 1, kPld, X, 1, kPld, D, 1, 8);
        } else {
          double* S = A + 8 * p * kPld + 8 * (c0 + q - nx);
          block_product<false, false>(S, kPld, 1, D, 8, 1, S, kPld, 1);
        }
      }
      if (below > 0) {
        asm volatile("bar.sync 1, %0;" ::"n"(32 * (WORKERS + 1)) : "memory");
        // the trailing blocks (i, j), p < j <= i, without the next diagonal block, then Y's
        const int tri = below * (below + 1) / 2, cols = INV == kInvFull ? p + 1 : (p & 1) ^ 1;
        const int ny = INV == kInvFull ? below * cols : cols;
        for (int q = warp; q < tri + ny; q += WORKERS) {
          if (q < tri) {
            int i = 0;
            while ((i + 1) * (i + 2) / 2 <= q) i++;
            const int j = p + 1 + q - i * (i + 1) / 2;
            i += p + 1;
            block_product<true, true>(A + 8 * j * kPld + 8 * i, 1, kPld, A + 8 * p * kPld + 8 * i, 1,
                                      kPld, A + 8 * p * kPld + 8 * j, kPld, 1);
          } else {
            const int f = q - tri, i = p + 1 + f / cols, c = INV == kInvFull ? f % cols : p;
            double* S = A + 8 * i * kPld + 8 * c;
            const double* X = A + 8 * p * kPld + 8 * i;
            if (c < p)
              block_product<true, true>(S, kPld, 1, X, 1, kPld, A + 8 * p * kPld + 8 * c, kPld, 1);
            else
              block_product<true, true>(S, kPld, 1, X, 1, kPld, D, 8, 1);
          }
        }
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) s_bad = bad;
  __syncthreads();
  return s_bad;
}

// Entry (r, c) of Y as potrf_blocks leaves it, c <= r.
__device__ __forceinline__ double potrf_y(const double* A, const double* Dv, int r, int c) {
  return r >> 3 == c >> 3 ? Dv[64 * (r >> 3) + 8 * (r & 7) + (c & 7)] : A[r * kPld + c];
}

// FP32 Cholesky of the n x n block A (n <= 64, column-major, leading dimension 64, lower
// triangle), in panels of 8 columns: warp 0 factors a panel in registers (two rows per lane,
// pivots and multipliers by shuffles), then the 256 threads apply it to the columns after it,
// a 4 x 4 block each.  Every element sees the same operations in the same order as in
// potrf_lookahead; that one's barrier and dependent shared-memory loads per column took 33 us at
// n = 64, where the FP32 arithmetic itself is short (96^3 diffusion: POTRF 13.2 -> 6.0 ms).
template <typename Accept>
__device__ int potrf_f32_panels(float* A, int n, Accept accept) {
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int bad = n;
  for (int k0 = 0; k0 < n; k0 += 8) {
    if (warp == 0) {
      float v[2][8];
#pragma unroll
      for (int g = 0; g < 2; g++)
#pragma unroll
        for (int j = 0; j < 8; j++) {
          const int r = k0 + 32 * g + lane;
          v[g][j] = r < n && k0 + j < n ? A[(k0 + j) * 64 + r] : 0.f;
        }
#pragma unroll
      for (int j = 0; j < 8; j++) {
        if (k0 + j >= n) break;
        const float p = __shfl_sync(0xffffffffu, v[0][j], j);
        const float y = pivot_rsqrt(p);
        if (bad == n && !accept(p)) bad = k0 + j;
        v[0][j] *= y;
        v[1][j] *= y;
#pragma unroll
        for (int q = 0; q < 8; q++)
          if (q > j) {
            const float l = __shfl_sync(0xffffffffu, v[0][j], q);
            v[0][q] = fmaf(-v[0][j], l, v[0][q]);
            v[1][q] = fmaf(-v[1][j], l, v[1][q]);
          }
      }
#pragma unroll
      for (int g = 0; g < 2; g++)
#pragma unroll
        for (int j = 0; j < 8; j++) {
          const int r = k0 + 32 * g + lane;
          if (r < n && r >= k0 + j) A[(k0 + j) * 64 + r] = v[g][j];
        }
    }
    __syncthreads();
    const int r0 = 4 * (tid & 15), c0 = 4 * (tid >> 4);
    if (c0 >= k0 + 8 && c0 < n && r0 >= c0 && r0 < n) {
      float4 x[4];
#pragma unroll
      for (int c = 0; c < 4; c++) x[c] = *reinterpret_cast<const float4*>(A + (c0 + c) * 64 + r0);
#pragma unroll
      for (int k = 0; k < 8; k++) {
        const float4 a = *reinterpret_cast<const float4*>(A + (k0 + k) * 64 + r0);
        const float4 b = *reinterpret_cast<const float4*>(A + (k0 + k) * 64 + c0);
        const float bc[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int c = 0; c < 4; c++) {
          x[c].x = fmaf(-a.x, bc[c], x[c].x);
          x[c].y = fmaf(-a.y, bc[c], x[c].y);
          x[c].z = fmaf(-a.z, bc[c], x[c].z);
          x[c].w = fmaf(-a.w, bc[c], x[c].w);
        }
      }
#pragma unroll
      for (int c = 0; c < 4; c++) *reinterpret_cast<float4*>(A + (c0 + c) * 64 + r0) = x[c];
    }
    __syncthreads();
  }
  if (tid == 0) s_bad = bad;
  __syncthreads();
  return s_bad;
}

// The inverses of the 16 x 16 diagonal blocks of L11 (shared memory, leading dimension ld) into
// Y (row-major n x n, global): warp b inverts block b, lane (i, h) column i and every other row,
// by forward substitution on the columns of the identity in registers.
template <typename T, typename S>
__device__ void invert_blocks(const S* A, int ld, int n, T* __restrict__ Y) {
  const int b0 = 16 * (threadIdx.x >> 5);
  if (b0 >= n) return;
  const int lane = threadIdx.x & 31, i = lane & 15, h = lane >> 4, bw = min(16, n - b0);
  T x[8];  // rows 2 q + h of column i
#pragma unroll
  for (int q = 0; q < 8; q++) x[q] = 2 * q + h == i ? T(1) : T(0);
#pragma unroll
  for (int j = 0; j < 16; j++) {
    if (j >= bw) break;
    const T rj = T(1) / (T)A[(b0 + j) * ld + b0 + j];
    T yj = x[j >> 1] * rj;  // row j is complete: its lane pair's half j & 1 holds it
    yj = __shfl_sync(0xffffffffu, yj, i + 16 * (j & 1));
    if (h == (j & 1)) {
      x[j >> 1] = yj;
      if (i <= j && b0 + i < n) Y[(int64_t)(b0 + j) * n + b0 + i] = yj;
    }
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int r = 2 * q + h;
      if (r > j && r < bw) x[q] = fma_t(-(T)A[(b0 + j) * ld + b0 + r], yj, x[q]);
    }
  }
}

template <typename T, typename S>
__device__ __forceinline__ void store_diag_block(T* __restrict__ L, const S* A, int lda, int n, int m) {
  const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  for (int c = threadIdx.x >> 5; c < n; c += nwarp)
    for (int r = c + lane; r < n; r += 32) L[(int64_t)c * m + r] = (T)A[c * lda + r];
}

// The kOzInvRows slice rows of Y S (Y as potrf_blocks leaves it; rows and columns past n are zero;
// S = diag(2^t_k), t_k the exponent of L11[k,k]) at slice rows y0 .. y0+63 of the scratch oy
// (planes oy_rows rows apart, then the rows' exponents, then the column shifts t_k): the
// right-hand operand of the supernode's tensor-core TRSM, A21 Y^T = (A21 S^-1)(Y S)^T.  The
// shift balances the operands: a column k of Y scales like 1/L_kk and the same column of A21
// like L_kk (rows and columns of A may span many decades), while Y S is the inverse of the
// unit-diagonal factor (exact: powers of two).  t: the n shifts; e: kOzInvRows ints.
__device__ void slice_inverse(const double* A, const double* Dv, int n, const int* t, uint8_t* oy,
                              int64_t oy_rows, int64_t y0, int* e) {
  const size_t stride = (size_t)oy_rows * kOzRowBytes;
  int32_t* oexp = reinterpret_cast<int32_t*>(oy + kOzSlices * stride);
  static_assert(kPotrfThreads == 4 * kOzInvRows, "four threads per row");
  {
    const int r = threadIdx.x >> 2;
    int f = 0;  // the largest exponent field of the row of Y S (fields shifted by t_k)
    if (r < n)
      for (int c = threadIdx.x & 3; c <= r; c += 4) {
        const int fc = oz_exp_field(potrf_y(A, Dv, r, c));
        if (fc > 0) f = max(f, fc + t[c]);
      }
    f = max(f, __shfl_xor_sync(0xffffffffu, f, 1));
    f = max(f, __shfl_xor_sync(0xffffffffu, f, 2));
    if ((threadIdx.x & 3) == 0) {
      e[r] = oz_row_exponent(f);
      oexp[y0 + r] = e[r];
      oexp[oy_rows + y0 + r] = r < n ? t[r] : 0;
    }
  }
  __syncthreads();
  for (int item = threadIdx.x; item < kOzInvRows * 8; item += blockDim.x) {
    const int r = item >> 3, pc = item & 7;  // row, physical 16-byte chunk
    const int c = pc ^ (int)((y0 + r) & 7);  // logical chunk: columns 8c .. 8c+7
    long long R[8];
#pragma unroll
    for (int j = 0; j < 8; j++) {
      const int k = 8 * c + j;
      R[j] = r < n && k <= r ? oz_fixed(potrf_y(A, Dv, r, k), e[r] - t[k]) : 0;  // Y[r,k] 2^t_k
    }
    oz_write_chunk(R, oy + (size_t)(y0 + r) * kOzRowBytes + pc * 16, stride);
  }
}

// ---- POTRF of each diagonal block ---------------------------------------------------------
// One CTA (kPotrfThreads threads) per supernode, in shared memory.  A non-positive pivot is an
// error (not SPD), recorded with its column.
// Factors that keep the inverses (d.dinv, widths up to 64) use potrf_blocks and get the inverses
// of the 16 x 16 diagonal blocks, in their places of the row-major Y, for the FP64 TRSM
// (k_diag_inverse completes Y later); with oy, a task whose y field is set (a 128-tile supernode
// of the FP64 factor) all of Y, for the solves, and Y's slices at rows y .. y+63 of oy, the
// operand of its tensor-core TRSM.
__global__ void __launch_bounds__(kPotrfThreads)
    k_potrf(const int4* __restrict__ tasks, const SnDev* __restrict__ sns,
            const MatDev* __restrict__ mats, uint8_t* oy, int64_t oy_rows) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* A = reinterpret_cast<double*>(smem_raw);
  __shared__ int s_e[kOzInvRows], s_t[kOzInvRows];
  if (gridDim.x <= kPotrfEarly) pdl_launch_dependents();
  const int4 tk = tasks[blockIdx.x];
  const SnDev d = sns[tk.x];
  const int n = d.n, m = d.m;
  double* L = reinterpret_cast<double*>(d.L);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  if (!d.dinv) {
    uint16_t* tab = reinterpret_cast<uint16_t*>(smem_raw + (size_t)n * n * sizeof(double));
    build_update_table(tab, n);
    pdl_wait();  // the levels below are done: the block is final but for this
    stage_diag_block(A, L, n, m);
    cp_async_wait_all();
    __syncthreads();
    const int bad = potrf_lookahead<double>(A, n, tab, [](double p) { return positive(p); });
    if (bad < n && threadIdx.x == 0) record_error(mats[d.mat], d.col0 + bad);
    store_diag_block(L, A, n, n, m);
    return;
  }
  double* Dv = A + 64 * kPld;
  const int n8 = (n + 7) & ~7;
  for (int c = warp; c < n8; c += nwarp)  // what the block does not fill: see potrf_blocks
    for (int r = lane; r < n8; r += 32)
      if (r < c || r >= n) A[c * kPld + r] = r == c ? 1.0 : 0.0;
  pdl_wait();
  stage_diag_block_ld(A, kPld, L, n, m);
  cp_async_wait_all();
  __syncthreads();
  const bool full = oy && tk.w >= 0;
  const int bad = full ? potrf_blocks<kInvFull, kPotrfWorkers>(A, Dv, n)
                        : potrf_blocks<kInvBlocks, kPotrfWorkers>(A, Dv, n);
  if (bad < n && threadIdx.x == 0) record_error(mats[d.mat], d.col0 + bad);
  store_diag_block(L, A, kPld, n, m);
  double* Y = reinterpret_cast<double*>(d.dinv);
  if (full) {
    // column shifts t_k: the exponent of L11[k,k] (|L_kk| in [2^t, 2^(t+1)))
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const int f = oz_exp_field(A[k * kPld + k]);
      s_t[k] = f > 0 ? f - 1023 : 0;
    }
    for (int r = warp; r < n; r += nwarp)
      for (int c = lane; c < n; c += 32) Y[r * n + c] = c <= r ? potrf_y(A, Dv, r, c) : 0.0;
    __syncthreads();
    slice_inverse(A, Dv, n, s_t, oy, oy_rows, tk.w, s_e);
  } else {
    for (int e = threadIdx.x; e < n * 16; e += blockDim.x) {
      const int r = e >> 4, c = (r & ~15) + (e & 15);
      if (c <= r) Y[r * n + c] = potrf_y(A, Dv, r, c);
    }
  }
}

// ---- TRSM of the off-diagonal rows --------------------------------------------------------
// Task {s, r0}: rows r0 .. r0+kTrsmRows-1 of L21 (panel rows n + r0 + lane), L21 = A21 L11^{-T},
// i.e. for each row x_j = (a_j - sum_{k<j} x_k L_jk) / L_jj.
//   k_trsm (any W <= 128): the substitution itself, one thread per row, partial rows in
//     shared memory.
// k_trsm_blk (W <= 64): the rows of a task (lane = row, or a part of the lanes per row when ROWS is
//   below 32) are solved by all the CTA's warps at once, 16 columns at a time.  Block b (columns
//   16b .. 16b+15, diagonal block D_b of L11): every lane group takes QC of the block's columns
//   and subtracts the products with the solved columns of the earlier blocks, acc_k = a_k -
//   sum_{j<16b} x_j L_kj; the partial vectors are exchanged through shared memory and the block
//   is finished as x_b = D_b^{-1} acc_b with D_b^{-1} from POTRF (in d.dinv).  On this part an FP64 warp
//   instruction holds its warp for ~64 cycles and 32 rows are 66,000 multiply-adds, 16 us of
//   one SM's FP64 units: levels with SMs to spare take ROWS = 16 or 8 per CTA (launch_trsm).
//   Wide levels do `per` tasks in turn in one CTA, so that L11 is staged once for them.
//   Measured per factorization: 64 x 64 2D Laplacian 0.21 -> 0.11 ms, 48^3 27-point (levels without
//   the tensor-core TRSM) 4.5 -> 3.3 ms, 96^3 diffusion in FP32 13.4 -> 9.7 ms.
template <int ROWS>
__host__ __device__ constexpr int trsm_warps() { return ROWS == 8 ? 4 : 8; }
template <typename T, int ROWS>
constexpr size_t trsm_blk_smem() { return (64 * 64 + 64 * ROWS + 16 * ROWS + 4 * 16 * 16) * sizeof(T); }

template <typename T, int ROWS>
__global__ void __launch_bounds__(32 * trsm_warps<ROWS>())
    k_trsm_blk(const int4* __restrict__ tasks, int ntasks, int per, const SnDev* __restrict__ sns) {
  constexpr int NG = 32 / ROWS, NC = trsm_warps<ROWS>() * NG, QC = 16 / NC;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* Ls = reinterpret_cast<T*>(smem_raw);  // Ls[c * 64 + r] = L11[r][c]
  T* Xs = Ls + 64 * 64;                     // Xs[k * ROWS + r]: solved column k of the rows
  T* Acc = Xs + 64 * ROWS;                  // Acc[kk * ROWS + r]: block column kk before D_b^{-1}
  T* Dv = Acc + 16 * ROWS;                  // Dv[b * 256 + k * 16 + i] = (D_b^{-1})[k][i], k >= i
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, r = lane % ROWS;
  const int w = (threadIdx.x >> 5) * NG + lane / ROWS;  // this lane group's first column of a block
  int cur = -1;
  const int e0 = blockIdx.x * per, e1 = min(ntasks, e0 + per);
  for (int e = e0; e < e1; e++) {
    const int4 tk = tasks[e];
    const SnDev d = sns[tk.x];
    const int n = d.n, m = d.m;
    T* L = reinterpret_cast<T*>(d.L);
    if (e == e0) pdl_wait();  // the diagonal blocks are factored
    if (tk.x != cur) {
      if (cur >= 0) __syncthreads();
      cur = tk.x;
      stage_diag_block_ld(Ls, 64, L, n, m);
      const T* Y = reinterpret_cast<const T*>(d.dinv);
      for (int q = threadIdx.x; q < n * 16; q += blockDim.x) {
        const int k = q >> 4, i = q & 15;
        if (i <= (k & 15)) cp_async_elem(Dv + (k >> 4) * 256 + (k & 15) * 16 + i, Y + k * n + (k & ~15) + i);
      }
    }
    // the lane group's own columns k = 16 b + w + NC q of this task's row
    const int row = n + tk.y + (int)blockIdx.y * ROWS + r;
    const bool live = row < m;
    T a[4 * QC];
#pragma unroll
    for (int b = 0; b < 4; b++)
#pragma unroll
      for (int q = 0; q < QC; q++) {
        const int k = 16 * b + w + NC * q;
        a[b * QC + q] = (live && k < n) ? L[(int64_t)k * m + row] : T(0);
      }
    cp_async_wait_all();
    __syncthreads();
#pragma unroll
    for (int b = 0; b < 4; b++) {
      if (16 * b >= n) break;
      T acc[QC];
#pragma unroll
      for (int q = 0; q < QC; q++) acc[q] = a[b * QC + q];
      const T* lrow = Ls + 16 * b + w;  // + j * 64 + NC q: L11[16b + w + NC q][j]
      for (int j = 0; j < 16 * b; j++) {
        const T xj = Xs[j * ROWS + r];
#pragma unroll
        for (int q = 0; q < QC; q++) acc[q] = fma_t(-xj, lrow[j * 64 + NC * q], acc[q]);
      }
#pragma unroll
      for (int q = 0; q < QC; q++) Acc[(w + NC * q) * ROWS + r] = acc[q];
      __syncthreads();
      const T* dv = Dv + b * 256;
#pragma unroll
      for (int q = 0; q < QC; q++) {
        const int kk = w + NC * q, k = 16 * b + kk;
        T s = T(0);
        if (k < n) {
          for (int i = 0; i <= kk; i++) s = fma_t(Acc[i * ROWS + r], dv[kk * 16 + i], s);
          if (live) L[(int64_t)k * m + row] = s;
        }
        Xs[k * ROWS + r] = s;
      }
      __syncthreads();
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(32) k_trsm(const int4* __restrict__ tasks, int ntasks, int* __restrict__ queue,
                                             const SnDev* __restrict__ sns) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_next_task;
  for (int tq = blockIdx.x; tq < ntasks;) {
    const int4 tk = tasks[tq];
    const SnDev d = sns[tk.x];
    const int n = d.n, m = d.m;
    T* L = reinterpret_cast<T*>(d.L);
    T* L11 = reinterpret_cast<T*>(smem_raw);  // n x n, column-major, ld n
    T* rdiag = L11 + n * n;                   // n
    T* X = rdiag + n;                         // n x 32: X[k * 32 + t]
    for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
      int c = idx / n, r = idx - c * n;
      L11[idx] = r >= c ? L[(int64_t)c * m + r] : T(0);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += blockDim.x) rdiag[j] = T(1) / L11[j * n + j];
    __syncthreads();
    const int t = threadIdx.x;
    for (int sub = 0; sub < kTrsmRows; sub += 32) {
      const int row = n + tk.y + sub + t;
      if (row < m) {
        for (int j = 0; j < n; j++) {
          T acc = L[(int64_t)j * m + row];
          for (int k = 0; k < j; k++) acc -= X[k * 32 + t] * L11[k * n + j];
          acc *= rdiag[j];
          X[j * 32 + t] = acc;
          L[(int64_t)j * m + row] = acc;
        }
      }
      __syncwarp();
    }
    __syncthreads();
    if (gridDim.x >= ntasks) break;
    if (threadIdx.x == 0) s_next_task = gridDim.x + atomicAdd(queue, 1);
    __syncthreads();
    tq = s_next_task;
  }
}

// ---- Schur update tiles ---------------------------------------------------------------------
// Task {s, i0, k0}: the T x T tile of U_s = L21 L21^T at rows i0.., columns k0.. (offsets
// into the off-diagonal rows of s), computed with FP64 m8n8k4 DMMA, then handed to
// schur_tile_epilogue.
template <int TILE>
struct SchurCfg {
  // four warps on every tile, one per FP64 unit of an SM: a 32 x 32 tile with K = 64 is 65,536
  // multiply-adds, 52 us on the one unit of a single warp.  64 x 64 2D Laplacian, 11 levels of
  // 32-tiles: 0.57 ms with one warp, 0.13 ms with four and the few-tile rule of schur_cls.
  static constexpr int WARPS_M = 2;
  static constexpr int WARPS_N = 2;
  static constexpr int WT = TILE / WARPS_M;       // warp tile edge: 32, 16 or 8
  static constexpr int MB = WT / 8;               // 8x8 blocks per warp edge
  static constexpr int THREADS = 32 * WARPS_M * WARPS_N;
  static constexpr int KC = TILE == 64 ? 32 : 64;  // K chunk staged in shared memory
  static constexpr int LDS = TILE + 8;            // padded stride (bank spread)
};

template <int TILE, bool OWNER>
__global__ void __launch_bounds__(SchurCfg<TILE>::THREADS)
    k_schur_f64(const int4* __restrict__ tasks, int ntasks, int* __restrict__ queue, const SnDev* __restrict__ sns,
                const MatDev* __restrict__ mats, int vsplit) {
  using Cfg = SchurCfg<TILE>;
  constexpr int KC = Cfg::KC, LDS = Cfg::LDS, MB = Cfg::MB;
  __shared__ __align__(16) double sh[2 * KC * LDS > TILE * (TILE + 1) ? 2 * KC * LDS
                                                                      : TILE * (TILE + 1)];
  double* As = sh;              // [KC][LDS]: As[kk][ii] = L21[i0 + ii][kc + kk]
  double* Bs = sh + KC * LDS;   // [KC][LDS]: Bs[kk][jj] = L21[k0 + jj][kc + kk]

  __shared__ int s_next_task;
  pdl_wait();
  // with vsplit > 0 every task is 2^vsplit virtual tasks, one per sub-tile
  const int nv = ntasks << vsplit;
  for (int tq = blockIdx.x; tq < nv;) {
    const int4 tk = tasks[tq >> vsplit];
    const SnDev d = sns[tk.x];
    const int n = d.n, m = d.m, u = m - n;
    // a task covers a (tk.w x tk.w) block of U_s (128 x 128 for the 128 class, whose .w
    // holds the slice offset instead); blocks larger than this kernel's tile are done as
    // TILE x TILE sub-tiles, skipping those wholly above the diagonal
    const int span = vsplit ? TILE << (vsplit >> 1) : (tk.w > TILE ? tk.w : TILE);
    const int sub_lo = vsplit ? (tq & ((1 << vsplit) - 1)) : 0;
    const int sub_hi = vsplit ? sub_lo + 1 : (span / TILE) * (span / TILE);
    for (int sub = sub_lo; sub < sub_hi; sub++) {
    const int i0 = tk.y + (sub / (span / TILE)) * TILE, k0 = tk.z + (sub % (span / TILE)) * TILE;
    if (i0 + TILE - 1 < k0 || i0 >= u || k0 >= u) continue;
    const double* L = reinterpret_cast<const double*>(d.L);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp / Cfg::WARPS_N, wn = warp % Cfg::WARPS_N;

    double acc[MB][MB][2];
  #pragma unroll
    for (int a = 0; a < MB; a++)
  #pragma unroll
      for (int b = 0; b < MB; b++) acc[a][b][0] = acc[a][b][1] = 0.0;

    for (int kc = 0; kc < n; kc += KC) {
      const int kw = min(KC, n - kc);
      for (int idx = tid; idx < KC * TILE; idx += Cfg::THREADS) {
        const int kk = idx / TILE, ii = idx - kk * TILE;
        double va = 0.0, vb = 0.0;
        if (kk < kw) {
          const int64_t col = (int64_t)(kc + kk) * m + n;
          if (i0 + ii < u) va = L[col + i0 + ii];
          if (k0 + ii < u) vb = L[col + k0 + ii];
        }
        As[kk * LDS + ii] = va;
        Bs[kk * LDS + ii] = vb;
      }
      __syncthreads();
      const int ksteps = (kw + 3) >> 2;
      for (int ks = 0; ks < ksteps; ks++) {
        const int kr = ks * 4 + (lane & 3);
        double af[MB], bf[MB];
  #pragma unroll
        for (int a = 0; a < MB; a++) af[a] = As[kr * LDS + wm * Cfg::WT + a * 8 + (lane >> 2)];
  #pragma unroll
        for (int b = 0; b < MB; b++) bf[b] = Bs[kr * LDS + wn * Cfg::WT + b * 8 + (lane >> 2)];
  #pragma unroll
        for (int a = 0; a < MB; a++)
  #pragma unroll
          for (int b = 0; b < MB; b++) dmma_884(acc[a][b], af[a], bf[b]);
      }
      __syncthreads();
    }
    // accumulators -> shared tile Cs[kk][ii] (ld TILE + 1)
    double* Cs = sh;
  #pragma unroll
    for (int a = 0; a < MB; a++)
  #pragma unroll
      for (int b = 0; b < MB; b++)
  #pragma unroll
        for (int e = 0; e < 2; e++) {
          const int ii = wm * Cfg::WT + a * 8 + (lane >> 2);
          const int kk = wn * Cfg::WT + b * 8 + (lane & 3) * 2 + e;
          Cs[kk * (TILE + 1) + ii] = acc[a][b][e];
        }
    __syncthreads();

    schur_tile_epilogue<double, TILE, Cfg::THREADS, OWNER>(
        Cs, d, i0, k0, sns, mats, static_cast<double*>(mats[d.mat].stage));
    __syncthreads();
    }
    __syncthreads();
    // a CTA's first task is its block index; only a grid smaller than the task list makes
    // CTAs take further tasks from this launch's work queue
    if (gridDim.x >= nv) break;
    if (threadIdx.x == 0) s_next_task = gridDim.x + atomicAdd(queue, 1);
    __syncthreads();
    tq = s_next_task;
  }
}

// ---- FP32 Schur tiles (mixed precision) -------------------------------------------------------
// The same task and epilogue as k_schur_f64 on FP32 panels: each of the (T/4)^2 threads
// accumulates a 4 x 4 block of the tile in FP32 registers (rows ty + q T/4, columns
// tx + p T/4) from K chunks staged in shared memory.
template <int TILE>
struct SchurF32Cfg {
  static constexpr int S = TILE / 4;
  static constexpr int THREADS = S * S;
  static constexpr int KC = 32;
  static constexpr int LDS = TILE + 4;
};

template <int TILE, bool OWNER>
__global__ void __launch_bounds__(SchurF32Cfg<TILE>::THREADS)
    k_schur_f32(const int4* __restrict__ tasks, int ntasks, int* __restrict__ queue, const SnDev* __restrict__ sns,
                const MatDev* __restrict__ mats, int vsplit) {
  using Cfg = SchurF32Cfg<TILE>;
  constexpr int KC = Cfg::KC, LDS = Cfg::LDS, S = Cfg::S;
  __shared__ __align__(16) float sh[2 * KC * LDS > TILE * (TILE + 1) ? 2 * KC * LDS
                                                                     : TILE * (TILE + 1)];
  float* As = sh;
  float* Bs = sh + KC * LDS;
  __shared__ int s_next_task;
  pdl_wait();
  // with vsplit > 0 every task is 2^vsplit virtual tasks, one per sub-tile
  const int nv = ntasks << vsplit;
  for (int tq = blockIdx.x; tq < nv;) {
    const int4 tk = tasks[tq >> vsplit];
    const SnDev d = sns[tk.x];
    const int n = d.n, m = d.m, u = m - n;
    // a task covers a (tk.w x tk.w) block of U_s (128 x 128 for the 128 class, whose .w
    // holds the slice offset instead); blocks larger than this kernel's tile are done as
    // TILE x TILE sub-tiles, skipping those wholly above the diagonal
    const int span = vsplit ? TILE << (vsplit >> 1) : (tk.w > TILE ? tk.w : TILE);
    const int sub_lo = vsplit ? (tq & ((1 << vsplit) - 1)) : 0;
    const int sub_hi = vsplit ? sub_lo + 1 : (span / TILE) * (span / TILE);
    for (int sub = sub_lo; sub < sub_hi; sub++) {
    const int i0 = tk.y + (sub / (span / TILE)) * TILE, k0 = tk.z + (sub % (span / TILE)) * TILE;
    if (i0 + TILE - 1 < k0 || i0 >= u || k0 >= u) continue;
    const float* L = reinterpret_cast<const float*>(d.L);
    const int tid = threadIdx.x, tx = tid % S, ty = tid / S;
    float acc[4][4];
  #pragma unroll
    for (int q = 0; q < 4; q++)
  #pragma unroll
      for (int p = 0; p < 4; p++) acc[q][p] = 0.f;
    for (int kc = 0; kc < n; kc += KC) {
      const int kw = min(KC, n - kc);
      for (int idx = tid; idx < KC * TILE; idx += Cfg::THREADS) {
        const int kk = idx / TILE, ii = idx - kk * TILE;
        float va = 0.f, vb = 0.f;
        if (kk < kw) {
          const int64_t col = (int64_t)(kc + kk) * m + n;
          if (i0 + ii < u) va = L[col + i0 + ii];
          if (k0 + ii < u) vb = L[col + k0 + ii];
        }
        As[kk * LDS + ii] = va;
        Bs[kk * LDS + ii] = vb;
      }
      __syncthreads();
      for (int kk = 0; kk < kw; kk++) {
        float a[4], b[4];
  #pragma unroll
        for (int q = 0; q < 4; q++) a[q] = As[kk * LDS + ty + q * S];
  #pragma unroll
        for (int p = 0; p < 4; p++) b[p] = Bs[kk * LDS + tx + p * S];
  #pragma unroll
        for (int q = 0; q < 4; q++)
  #pragma unroll
          for (int p = 0; p < 4; p++) acc[q][p] = fmaf(a[q], b[p], acc[q][p]);
      }
      __syncthreads();
    }
    float* Cs = sh;
  #pragma unroll
    for (int q = 0; q < 4; q++)
  #pragma unroll
      for (int p = 0; p < 4; p++) Cs[(tx + p * S) * (TILE + 1) + ty + q * S] = acc[q][p];
    __syncthreads();
    schur_tile_epilogue<float, TILE, Cfg::THREADS, OWNER>(
        Cs, d, i0, k0, sns, mats, static_cast<float*>(mats[d.mat].stage));
    __syncthreads();
    }
    __syncthreads();
    // a CTA's first task is its block index; only a grid smaller than the task list makes
    // CTAs take further tasks from this launch's work queue
    if (gridDim.x >= nv) break;
    if (threadIdx.x == 0) s_next_task = gridDim.x + atomicAdd(queue, 1);
    __syncthreads();
    tq = s_next_task;
  }
}

// ---- POTRF of the mixed-precision factor ---------------------------------------------------
// FP32 panels of the equilibrated matrix (unit diagonal before updates).  The block is
// factored in FP32; if any pivot falls below tau (tau times the original diagonal, which
// is 1 after equilibration), the block is factored again in FP64 from the panel's values,
// which are still unchanged in global memory, and the FP64 result is rounded into the panel.
// err[2] counts such redos.  The FP64 block overlays the FP32 one in shared memory.
__global__ void __launch_bounds__(kPotrfThreads)
    k_potrf_mixed(const int4* __restrict__ tasks, const SnDev* __restrict__ sns,
                  const MatDev* __restrict__ mats, float tau) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* A = reinterpret_cast<float*>(smem_raw);    // FP32 work block, leading dimension lda
  double* D = reinterpret_cast<double*>(smem_raw);  // n x n FP64 block of a redo
  if (gridDim.x <= kPotrfEarly) pdl_launch_dependents();
  const int4 tk = tasks[blockIdx.x];
  const SnDev d = sns[tk.x];
  const int n = d.n, m = d.m, lda = n <= 64 ? 64 : n;
  float* L = reinterpret_cast<float*>(d.L);
  float* Y = reinterpret_cast<float*>(d.dinv);
  uint16_t* tab = reinterpret_cast<uint16_t*>(smem_raw + potrf_mixed_tab_offset(n));
  pdl_wait();  // the levels below are done: the block is final but for this
  stage_diag_block_ld(A, lda, L, n, m);
  if (n > 64) build_update_table(tab, n);
  cp_async_wait_all();
  __syncthreads();
  const auto accept = [&](float p) { return p >= tau; };
  const int stop = n <= 64 ? potrf_f32_panels(A, n, accept)
                           : potrf_lookahead<float>(A, n, tab, accept);
  if (stop < n) {
    // a small FP32 pivot: the whole block again in FP64 (the barrier that ended the FP32
    // pass is behind every thread, so D may overwrite A)
    if (threadIdx.x == 0) atomicAdd(mats[d.mat].err + 2, 1ull);
    const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    for (int c = threadIdx.x >> 5; c < n; c += nwarp)
      for (int r = c + lane; r < n; r += 32) D[c * n + r] = (double)L[(int64_t)c * m + r];
    if (n <= 64) build_update_table(tab, n);
    __syncthreads();
    const int bad = potrf_lookahead<double>(D, n, tab, [](double p) { return positive(p); });
    if (bad < n && threadIdx.x == 0) record_error(mats[d.mat], d.col0 + bad);
    store_diag_block(L, D, n, n, m);
    __syncthreads();
    // the diagonal blocks' inverses of the rounded factor, as without the redo
    if (Y)
      for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) D[idx] = (double)(float)D[idx];
    __syncthreads();
    if (Y) invert_blocks<float, double>(D, n, n, Y);
  } else {
    store_diag_block(L, A, lda, n, m);
    if (Y) invert_blocks<float, float>(A, lda, n, Y);
  }
}

// ---- owner assembly -----------------------------------------------------------------------
// Group {t, cb, first, end}: every staged U_s entry of this level that falls into columns
// [32 cb, 32 cb + 32) of target t is subtracted, sources in ascending s: each panel entry sees its
// updates in a fixed order, so the result is bitwise reproducible.  A warp owns whole target
// columns and takes the sources one after another on its own (its lanes' writes ordered by
// __syncwarp), so no barrier and no idle warp stands between two sources: only once per
// kAsmBatch sources do all threads look up which column of a source is which of the target's
// (a barrier pair per source and 1,024 of its rows took 138 us a level at 24^3, 27 points; now
// 58 us, the step 19.4 -> 13.8 ms).
constexpr int kAsmThreads = 256;
constexpr int kAsmBatch = 32;
constexpr int kAsmInFlight = 4;  // rows per lane with loads in flight

template <typename T>
__global__ void __launch_bounds__(kAsmThreads)
    k_assemble_owner(const int4* __restrict__ groups, const int4* __restrict__ srcs,
                     const SnDev* __restrict__ sns, const MatDev* __restrict__ mats) {
  __shared__ int kmap[kAsmBatch][32];  // the source's row position of target column c, or -1
  __shared__ const T* s_U[kAsmBatch];
  __shared__ const int32_t* s_rel[kAsmBatch];
  __shared__ int s_u[kAsmBatch];
  pdl_wait();
  const int4 g = groups[blockIdx.x];
  const SnDev td = sns[g.x];
  const MatDev md = mats[td.mat];
  T* Lt = reinterpret_cast<T*>(td.L);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int q0 = g.z; q0 < g.w; q0 += kAsmBatch) {
    const int nb = min(kAsmBatch, g.w - q0);
    __syncthreads();
    for (int idx = threadIdx.x; idx < nb * 32; idx += kAsmThreads) kmap[idx >> 5][idx & 31] = -1;
    __syncthreads();
    for (int idx = threadIdx.x; idx < nb * 32; idx += kAsmThreads) {
      const int q = idx >> 5, j = idx & 31;
      const int4 sr = srcs[q0 + q];  // {s, kb, ke, -}: at most 32 columns
      const SnDev& sd = sns[sr.x];
      const int n = sd.n;
      if (sr.y + j < sr.z) kmap[q][sd.rows[n + sr.y + j] - td.col0 - 32 * g.y] = sr.y + j;
      if (j == 0) {
        s_U[q] = static_cast<const T*>(md.stage) + sd.ustage;
        s_rel[q] = md.relmap + md.run_base[find_run(md, sd, sr.y)];
        s_u[q] = sd.m - n;
      }
    }
    __syncthreads();
    for (int c = warp; c < 32; c += nwarp) {
      T* col = Lt + (int64_t)(32 * g.y + c) * td.m;
      for (int q = 0; q < nb; q++) {
        const int k = kmap[q][c];
        if (k < 0) continue;
        const int u = s_u[q];
        const T* U = s_U[q] + (int64_t)k * u;
        const int32_t* rel = s_rel[q];
        for (int i0 = k + lane; i0 < u; i0 += 32 * kAsmInFlight) {
          int p[kAsmInFlight];
          T v[kAsmInFlight], x[kAsmInFlight];
#pragma unroll
          for (int e = 0; e < kAsmInFlight; e++) {
            const int i = i0 + 32 * e;
            p[e] = i < u ? rel[i] : -1;
            v[e] = i < u ? U[i] : T(0);
          }
#pragma unroll
          for (int e = 0; e < kAsmInFlight; e++)
            if (p[e] >= 0) x[e] = col[p[e]];
#pragma unroll
          for (int e = 0; e < kAsmInFlight; e++)
            if (p[e] >= 0) col[p[e]] = x[e] - v[e];
        }
        __syncwarp();
      }
    }
  }
}

// ---- relative map -------------------------------------------------------------------------
// One CTA per supernode s: for every target run q of s (rows from run_a[q] on belong to the
// run's target t or to later targets, all of them rows of t by the elimination-tree
// property) the position of each row inside t's sorted row list; a row missing from t (an
// internal inconsistency) is stored as -1 and counted in *miss.
__global__ void k_build_relmap(const int32_t* __restrict__ sn_start, const int64_t* __restrict__ sn_rowptr,
                               const int32_t* __restrict__ rows, const int32_t* __restrict__ sn_run0,
                               const int32_t* __restrict__ run_a, const int32_t* __restrict__ run_t,
                               const int64_t* __restrict__ run_base, int32_t* __restrict__ relmap,
                               unsigned long long* __restrict__ miss) {
  const int s = blockIdx.x;
  const int n = sn_start[s + 1] - sn_start[s];
  const int64_t rp = sn_rowptr[s];
  const int u = (int)(sn_rowptr[s + 1] - rp) - n;
  const int32_t* r = rows + rp + n;
  for (int q = sn_run0[s]; q < sn_run0[s + 1]; q++) {
    const int t = run_t[q];
    const int tn = sn_start[t + 1] - sn_start[t], tcol0 = sn_start[t];
    const int64_t trp = sn_rowptr[t];
    const int tm = (int)(sn_rowptr[t + 1] - trp);
    const int32_t* tr = rows + trp;
    for (int i = run_a[q] + threadIdx.x; i < u; i += blockDim.x) {
      const int key = r[i];
      int p;
      if (key - tcol0 < tn) {
        p = key - tcol0;  // one of t's own columns
      } else {
        p = lower_bound_dev(tr, tm, key);
        if (p >= tm || tr[p] != key) {
          p = -1;
          atomicAdd(miss, 1ull);
        }
      }
      relmap[run_base[q] + i] = p;
    }
  }
}

void launch_build_relmap(int32_t ns, const int32_t* sn_start, const int64_t* sn_rowptr,
                         const int32_t* rows, const int32_t* sn_run0, const int32_t* run_a,
                         const int32_t* run_t, const int64_t* run_base, int32_t* relmap,
                         unsigned long long* miss, cudaStream_t st) {
  if (ns <= 0) return;
  k_build_relmap<<<ns, 256, 0, st>>>(sn_start, sn_rowptr, rows, sn_run0, run_a, run_t, run_base,
                                     relmap, miss);
}

// ---- launchers --------------------------------------------------------------------------------
void launch_assemble(const double* vals, const int64_t* amap, int64_t nnz, void* L, bool f32,
                     cudaStream_t st) {
  if (nnz <= 0) return;
  int blocks = (int)std::min<int64_t>((nnz + 255) / 256, 152 * 16);
  if (f32) k_assemble<float><<<blocks, 256, 0, st>>>(vals, amap, nnz, (float*)L);
  else k_assemble<double><<<blocks, 256, 0, st>>>(vals, amap, nnz, (double*)L);
}

static size_t potrf_smem(int w) {  // potrf_blocks, or the block and potrf_lookahead's table
  return std::max((size_t)w * w * sizeof(double) + update_table_bytes(w), kPotrfBlkSmem);
}

constexpr int kDinvThreads = 256;
template <typename P>
constexpr size_t dinv_smem() {
  return ((size_t)kDinvMaxWidth * kDinvMaxWidth + kDinvMaxWidth) * sizeof(P);
}

// Y = L11^-1 of the supernode of each task (POTRF tasks, one CTA per task) into d.dinv,
// row-major n x n (dinv[r * n + c] = Y[r, c], zeros above the diagonal), in the panel's
// precision; supernodes without dinv are skipped.  Forward substitution on all columns of
// the identity at once, right-looking: with l'_ij = L_ij / L_jj and Z = I, step j (one
// barrier) takes Z[i, c] -= l'_ij Z[j, c] for the rows i > j and columns c <= j (row j is
// final by then); Y[i, c] = Z[i, c] / L_ii at the end: n (n^2 - 1) / 6 multiply-adds, the n
// reciprocals once.  One n x n shared array holds both factors of each step: l' in the
// strict lower triangle (column-major, S[c * n + r]) and the lower-triangular Z transposed
// in the upper triangle and the diagonal (Z[i, c] at S[i * n + c]), so a warp's threads
// update consecutive words.  The solves apply Y instead of substituting serially (each FP64
// instruction holds its warp ~64 cycles, so a 64-step substitution chain costs ~10 us).
template <typename P>
__global__ void __launch_bounds__(kDinvThreads)
    k_diag_inverse(const int4* __restrict__ tasks, const SnDev* __restrict__ sns,
                   bool skip_sliced) {
  extern __shared__ __align__(16) double dsm[];
  const int4 tk = tasks[blockIdx.x];
  const SnDev d = sns[tk.x];
  pdl_wait();
  if (!d.dinv || (skip_sliced && tk.w >= 0)) return;
  const int n = d.n;
  P* S = reinterpret_cast<P*>(dsm);
  P* rd = S + n * n;
  stage_diag_block(S, reinterpret_cast<const P*>(d.L), n, d.m);
  cp_async_wait_all();
  __syncthreads();
  for (int j = threadIdx.x; j < n; j += blockDim.x) rd[j] = P(1) / S[j * n + j];
  __syncthreads();
  for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
    const int c = idx / n, r = idx - c * n;
    if (r > c) S[idx] *= rd[c];          // l'_rc
    else S[idx] = r == c ? P(1) : P(0);  // Z[c, r] = I
  }
  __syncthreads();
  for (int j = 0; j + 1 < n; j++) {
    const int cols = j + 1, rows = n - 1 - j;
    for (int idx = threadIdx.x; idx < rows * cols; idx += blockDim.x) {
      const int ii = idx / cols, c = idx - ii * cols, i = j + 1 + ii;
      S[i * n + c] -= S[j * n + i] * S[j * n + c];
    }
    __syncthreads();
  }
  P* Y = reinterpret_cast<P*>(d.dinv);
  for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
    const int r = idx / n, c = idx - r * n;
    Y[idx] = c <= r ? S[idx] * rd[r] : P(0);
  }
}

void launch_diag_inverse(const int4* tasks, int ntasks, const SnDev* sns, bool f32,
                         bool skip_sliced, cudaStream_t st) {
  if (ntasks <= 0) return;
  if (f32)
    launch_pdl(k_diag_inverse<float>, ntasks, kDinvThreads, dinv_smem<float>(), st, tasks, sns, false);
  else
    launch_pdl(k_diag_inverse<double>, ntasks, kDinvThreads, dinv_smem<double>(), st, tasks, sns,
               skip_sliced);
}
static size_t potrf_mixed_smem(int w) { return potrf_mixed_tab_offset(w) + update_table_bytes(w); }
static size_t trsm_smem(int w) { return ((size_t)w * w + w + (size_t)w * 32) * sizeof(double); }

void launch_potrf(const int4* tasks, int ntasks, const SnDev* sns, const MatDev* mats,
                  int max_width, bool f32, float tau, void* oy, int64_t oy_rows, cudaStream_t st) {
  if (ntasks <= 0) return;
  if (f32)
    launch_pdl(k_potrf_mixed, ntasks, kPotrfThreads, potrf_mixed_smem(max_width), st, tasks, sns, mats,
               tau);
  else
    launch_pdl(k_potrf, ntasks, kPotrfThreads, potrf_smem(max_width), st, tasks, sns, mats,
               static_cast<uint8_t*>(oy), oy_rows);
}

template <typename T, int ROWS>
static void trsm_blk_t(const int4* tasks, int ntasks, int per, const SnDev* sns, cudaStream_t st) {
  launch_pdl(k_trsm_blk<T, ROWS>, dim3((ntasks + per - 1) / per, kTrsmRows / ROWS),
             32 * trsm_warps<ROWS>(), trsm_blk_smem<T, ROWS>(), st, tasks, ntasks, per, sns);
}

template <typename T>
static void trsm_t(const int4* tasks, int ntasks, int* queue, const SnDev* sns, int max_width,
                   cudaStream_t st) {
  if (max_width <= 64) {
    // rows per CTA: as few as keep the CTAs within one wave (152 SMs); wide levels four tasks
    // per CTA while three CTAs per SM are left
    if (4 * ntasks <= 152) trsm_blk_t<T, 8>(tasks, ntasks, 1, sns, st);
    else if (2 * ntasks <= 152) trsm_blk_t<T, 16>(tasks, ntasks, 1, sns, st);
    else trsm_blk_t<T, 32>(tasks, ntasks, ntasks >= 4 * 3 * 152 ? 4 : 1, sns, st);
    return;
  }
  const size_t sm = trsm_smem(max_width);
  k_trsm<T><<<task_grid(k_trsm<T>, 32, sm, ntasks), 32, sm, st>>>(tasks, ntasks, queue, sns);
}

void launch_trsm(const int4* tasks, int ntasks, int* queue, const SnDev* sns, int max_width,
                 bool f32, cudaStream_t st) {
  if (ntasks <= 0) return;
  if (f32) trsm_t<float>(tasks, ntasks, queue, sns, max_width, st);
  else trsm_t<double>(tasks, ntasks, queue, sns, max_width, st);
}

template <int T, bool OWNER>
static void schur_f64_t(const int4* tasks, int ntasks, int* queue, const SnDev* sns,
                        const MatDev* mats, cudaStream_t st, int vsplit = 0) {
  constexpr int th = SchurCfg<T>::THREADS;
  launch_pdl(k_schur_f64<T, OWNER>, task_grid(k_schur_f64<T, OWNER>, th, 0, ntasks << vsplit), th, 0,
             st, tasks, ntasks, queue, sns, mats, vsplit);
}

template <int T, bool OWNER>
static void schur_f32_t(const int4* tasks, int ntasks, int* queue, const SnDev* sns,
                        const MatDev* mats, cudaStream_t st, int vsplit = 0) {
  constexpr int th = SchurF32Cfg<T>::THREADS;
  launch_pdl(k_schur_f32<T, OWNER>, task_grid(k_schur_f32<T, OWNER>, th, 0, ntasks << vsplit), th, 0,
             st, tasks, ntasks, queue, sns, mats, vsplit);
}

template <bool OWNER>
static void schur_cls(int cls, bool f32, const int4* tasks, int ntasks, int* queue,
                      const SnDev* sns, const MatDev* mats, cudaStream_t st) {
  if (f32) {
    // 128-wide tasks without the tensor-core scratch: four 64 x 64 virtual tasks
    if (cls == kTile128) schur_f32_t<64, OWNER>(tasks, ntasks, queue, sns, mats, st, 2);
    else if (cls == kTile64) schur_f32_t<64, OWNER>(tasks, ntasks, queue, sns, mats, st);
    else if (cls == kTile32) schur_f32_t<32, OWNER>(tasks, ntasks, queue, sns, mats, st);
    else schur_f32_t<16, OWNER>(tasks, ntasks, queue, sns, mats, st);
  } else {
    // FP64 128-wide tasks run as four 64 x 64 virtual tasks of the DMMA kernel
    if (cls == kTile128) schur_f64_t<64, OWNER>(tasks, ntasks, queue, sns, mats, st, 2);
    else if (cls == kTile64) schur_f64_t<64, OWNER>(tasks, ntasks, queue, sns, mats, st);
    else if (cls == kTile32 && 4 * ntasks > 3 * 152)
      schur_f64_t<32, OWNER>(tasks, ntasks, queue, sns, mats, st);
    // few 32-tiles: as 16 x 16 virtual tasks, which spread over the idle SMs' FP64 units (20 us
    // a 32-tile on one SM, 5 us a 16-tile) while there are at most three of them per SM
    else if (cls == kTile32) schur_f64_t<16, OWNER>(tasks, ntasks, queue, sns, mats, st, 2);
    else schur_f64_t<16, OWNER>(tasks, ntasks, queue, sns, mats, st);
  }
}

void launch_schur(int cls, const int4* tasks, int ntasks, int* queue, const SnDev* sns,
                  const MatDev* mats, bool owner, bool f32, cudaStream_t st) {
  if (ntasks <= 0) return;
  if (owner) schur_cls<true>(cls, f32, tasks, ntasks, queue, sns, mats, st);
  else schur_cls<false>(cls, f32, tasks, ntasks, queue, sns, mats, st);
}

template <typename T>
static void asm_owner_t(const int4* groups, int ngroups, const int4* srcs, const SnDev* sns,
                        const MatDev* mats, cudaStream_t st) {
  launch_pdl(k_assemble_owner<T>, ngroups, kAsmThreads, 0, st, groups, srcs, sns, mats);
}

void launch_assemble_owner(const int4* groups, int ngroups, const int4* srcs, const SnDev* sns,
                           const MatDev* mats, bool f32, cudaStream_t st) {
  if (ngroups <= 0) return;
  if (f32) asm_owner_t<float>(groups, ngroups, srcs, sns, mats, st);
  else asm_owner_t<double>(groups, ngroups, srcs, sns, mats, st);
}

template <typename K>
static bool set_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) ==
         cudaSuccess;
}

int set_factor_kernel_attrs(int max_width) {
  bool ok = set_smem(k_diag_inverse<double>, dinv_smem<double>()) &&
            set_smem(k_diag_inverse<float>, dinv_smem<float>()) &&
            set_smem(k_potrf, potrf_smem(max_width)) &&
            set_smem(k_potrf_mixed, potrf_mixed_smem(max_width)) &&
            set_smem(k_trsm_blk<double, 32>, trsm_blk_smem<double, 32>()) &&
            set_smem(k_trsm_blk<double, 16>, trsm_blk_smem<double, 16>()) &&
            set_smem(k_trsm_blk<double, 8>, trsm_blk_smem<double, 8>()) &&
            set_smem(k_trsm_blk<float, 32>, trsm_blk_smem<float, 32>()) &&
            set_smem(k_trsm_blk<float, 16>, trsm_blk_smem<float, 16>()) &&
            set_smem(k_trsm_blk<float, 8>, trsm_blk_smem<float, 8>()) &&
            set_smem(k_trsm<double>, trsm_smem(max_width)) &&
            set_smem(k_trsm<float>, trsm_smem(max_width));
  return ok ? CHOL_OK : CHOL_E_CUDA;
}

}  // namespace chol
