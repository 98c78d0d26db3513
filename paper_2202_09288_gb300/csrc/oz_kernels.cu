// oz_kernels.cu -- FP64 Schur update tiles of the FP64 factor on the bf16 tcgen05 tensor
// cores by operand splitting (Ozaki's error-free splitting of a dot product).
//
// The update U_s = L21 L21^T (Sec. 3, Listing 1: SYRK + GEMM) of a 128-tile supernode is
// computed in two steps per level:
//   k_oz_slice  every row r of L21 gets an exponent e_r (max_k |L21[r,k]| < 2^e_r) and
//               kOzSlices integer slices s_p[r,k] of 8 bits with
//               L21[r,k] = 2^e_r sum_p s_p[r,k] 2^(-7-8p) + (error <= 2^(e_r-56)),
//               stored as bf16 (exact) in units of 32 columns, rows of 64 bytes whose 16-byte
//               chunks are pre-swizzled for the tensor cores' 64-byte swizzle;
//   k_schur_oz  a 128 x 128 task is done as four 128 x 32 quarters.  The units of the task's 128 A
//               rows and of each quarter's 32 B rows (7 slices each) are brought into
//               shared memory by tiled TMA copies issued by a load thread, which
//               also claims the tasks; an MMA thread issues, for every slice pair p + q < 7,
//               the bf16 MMAs of D_{p+q} += S_p S_q^T into the quarter's set of tensor-memory
//               accumulators (one per diagonal p + q, 7 x 32 columns; two sets).  K is the
//               supernode's columns (<= 64) or those of two merged chunks (<= 128): every partial
//               sum of a diagonal is an integer of at most 7 2^21, so FP32 accumulation is exact.
//               Consumer warps read a finished
//               set (lane = tile row), release it, form U[i,k] = 2^(e_i+e_k)
//               sum_d 2^(-14-8d) D_d[i,k] as an FP64 value (integer combination, one
//               int64 -> double conversion) and add it into the ancestors with FP64
//               reductions (or write the owner staging buffer) while the tensor cores compute
//               the next quarter; metadata warps prepare the next task's targets ahead.
// What bounds it (80^3 27-point, 23,400 cycles per K = 128 tile): the MMAs (15,400 alone, 16,800 as the
// MMA thread issues them, 17,500 with the copies, 19,900 with the conversions) and the latency of the
// copies while the reductions fill the L2 (the rest).  In tiles of K = 64 with one chunk per task
// the same work took 32,800.
// Every wait is bounded in time (kOzWaitCycles SM clock cycles, about a second): then the
// kernel records a timeout in err[3] of every factor with work in the launch,
// waits (bounded) for its copies and MMAs in flight, frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "chol_internal.h"
#include "device_common.cuh"
#include "kernels.h"
#include "oz_combine.h"
#include "oz_common.cuh"
#include "launch_util.h"

namespace chol {

namespace {

constexpr int kOzConsumers = 512;                          // 16 warps: drain + scatter
constexpr int kOzMetaThreads = 128;                        // 4 warps: per-task metadata
constexpr int kOzMmaWarp = kOzConsumers / 32;              // issues the MMAs (one thread)
constexpr int kOzLoadWarp = kOzMmaWarp + 1;                // issues the TMA copies (one thread)
constexpr int kOzMetaBase = kOzConsumers + 64;             // first metadata thread
constexpr int kOzThreads = kOzMetaBase + kOzMetaThreads;
constexpr int kOzRing = 16;
constexpr int kOzM = 128;                                  // tile rows (UMMA M)
constexpr uint32_t kOzASlice = kOzM * kOzRowBytes;         // 16 KB (TRSM)
constexpr uint32_t kOzABytes = kOzSlices * kOzASlice;      // 112 KB (TRSM)
// Schur tiles: operands in units of 32 columns of K (64-byte rows)
constexpr int kOzQ = 32;                                   // columns per quarter
constexpr int kOzUnitRow = 64;                             // bytes of a row's unit
constexpr uint32_t kOzUASlice = kOzM * kOzUnitRow;         // 8 KB
constexpr uint32_t kOzUBSlice = kOzQ * kOzUnitRow;         // 2 KB
constexpr uint32_t kOzUA = kOzSlices * kOzUASlice;         // 56 KB: a unit of A
constexpr uint32_t kOzUB = kOzSlices * kOzUBSlice;         // 14 KB: a unit of a quarter's B
constexpr int kOzABufs = 3, kOzBBufs = 3;
constexpr int kOzSetCols = kOzSlices * kOzQ;               // 224: TMEM columns of a set
constexpr size_t kOzSmem = 512 + kOzABufs * kOzUA + kOzBBufs * kOzUB;  // + alignment slack
constexpr uint32_t kOzTmemCols = 512;                     // two sets of 7 diagonals (448)
static_assert(kOzABufs == 3, "the load thread's replacement looks at three buffers");
// A step as the load thread describes it: A buffer, K steps of 16 (1 or 2), first and last of its
// quarter, stop.
constexpr int kStepK = 2, kStepFirst = 4, kStepLast = 5, kStepStop = 6;
// Bound of every wait in SM clock cycles (~1 s at 2 GHz; the waits of a working launch last
// microseconds).  Counted with clock64(), not in polls: a poll of mbarrier.try_wait may suspend
// the thread for a hardware-defined time.
constexpr long long kOzWaitCycles = 1ll << 31;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor, K-major, 128-byte swizzle: 8-row groups 1024 bytes
// apart (stride byte offset), descriptor version 1, leading byte offset unused (16).
__device__ __forceinline__ uint64_t oz_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)(16 >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// The same with the 64-byte swizzle: 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t oz_desc64(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | (uint64_t)(16 >> 4) << 16 | (uint64_t)(512 >> 4) << 32 |
         (uint64_t)1 << 46 | (uint64_t)4 << 61;
}

// Instruction descriptor of kind::f16: FP32 accumulator, bf16 A and B (format 1), both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__device__ __forceinline__ uint32_t oz_idesc(int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(kOzM >> 4) << 24);
}

__device__ __forceinline__ bool oz_wait(uint32_t bar, uint32_t parity,
                                        long long limit = kOzWaitCycles) {
  long long t0 = 0;
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (t0 == 0) t0 = clock64();
    else if (clock64() - t0 > limit) return false;
  }
}

// Whether the phase is complete, without waiting.
__device__ __forceinline__ bool oz_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}

__device__ __forceinline__ void oz_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void oz_bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                             uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

// Tiled copy of a unit: all slices of the 8-row groups from g8 on, half h (see oz_unit_map).
__device__ __forceinline__ void oz_unit_load(uint32_t dst, const CUtensorMap* map, int g8, int h,
                                             uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], "
      "[%1, {%2, %3, %4, %2}], [%5];" ::"r"(dst),
      "l"(map), "r"(0), "r"(g8), "r"(h), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void oz_mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

// True in one thread of the (converged) warp.
__device__ __forceinline__ bool oz_elect() {
  uint32_t e;
  asm volatile(
      "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(e));
  return e != 0;
}

__device__ __forceinline__ void oz_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}

}  // namespace

constexpr int kOzSliceThreads = 256;
constexpr int kOzSliceLd = kOzM + 1;  // padded column stride of the staged block

// Slices of the L21 rows r0 .. r0+127 of supernode s, at slice rows oz + r (rows u ..
// roundup(u, 8) get zero slices).  The block is staged column by column through shared
// memory (cp.async, all copies in flight); a row's exponent e_r is that of its largest entry; each
// entry becomes the integer x 2^(55-e_r), rounded to nearest and cut into 7 balanced digits
// of 8 bits (|s_p| <= 128, exact); thread t writes the
// 16-byte chunk t % 8 of row t / 8 of every slice (coalesced, pre-swizzled).
// With oy (the tensor-core TRSM's operand A21 S^-1, sliced before that TRSM), column k is
// scaled by 2^-t_k, the shift POTRF stored with the supernode's inverse slices in oy, and the planes
// have rows of 128 bytes.  Without it (the Schur tiles) plane p is two planes of 64-byte rows, its
// columns 0 .. 31 and 32 .. 63, swizzled by 64 bytes: 16-byte chunk c of slice row R sits at chunk c ^
// ((R >> 1) & 3).  A task with w = -2 or -3 is one of two merged chunks whose rows get one exponent
// (their products are summed in tensor memory): w = -2, the chunk before s is the other, w =
// -3 the one after it; the other's largest exponents are read straight from its panel (a second pass
// over it, 80^3 27-point: the level's slicing 62 -> 67.5 ms, of 1,434).
__global__ void __launch_bounds__(kOzSliceThreads)
    k_oz_slice(const int4* __restrict__ tasks, const SnDev* __restrict__ sns,
               uint8_t* oz, int64_t oz_rows, const uint8_t* oy,
               int64_t oy_rows) {
  extern __shared__ __align__(16) double xs[];  // [n][kOzSliceLd]
  __shared__ int s_e[kOzM], s_t[kOzInvRows], s_f[kOzSliceThreads];
  const int4 tk = tasks[blockIdx.x];
  pdl_wait();
  if (oy && tk.w < 0) return;  // A21 slices only for the tensor-core TRSM's supernodes
  const SnDev d = sns[tk.x];
  const int n = d.n, m = d.m, u = m - n;
  const int r0 = tk.y;
  const int rows = min(kOzM, ((u + 7) & ~7) - r0);  // slice rows this block owns
  const double* L = reinterpret_cast<const double*>(d.L) + n + r0;  // L21[r0 + i, k] = L[k m + i]
  static_assert(kOzM == 128, "stage_row_block stages 128 rows");
  stage_row_block(xs, kOzSliceLd, L, m, n, u - r0);
  if (threadIdx.x < kOzInvRows) {
    // the shifts follow the inverse slices' row exponents in oy
    const int32_t* shift =
        oy ? reinterpret_cast<const int32_t*>(oy + kOzSlices * (size_t)oy_rows * kOzRowBytes) +
                 oy_rows + tk.w
           : nullptr;
    s_t[threadIdx.x] = shift && threadIdx.x < n ? shift[threadIdx.x] : 0;
  }
  int fmax = 0;  // largest exponent field of the other chunk's row, half of its columns
  static_assert(kMergeChunks == 2, "a merged chunk has one other");
  if (!oy && tk.w <= -2) {
    const SnDev o = sns[tk.w == -2 ? tk.x - 1 : tk.x + 1];
    const int i = threadIdx.x & (kOzM - 1);
    if (i < u - r0) {
      const int off = tk.w == -2 ? r0 + n : r0 - o.n;  // row r0 of s among the other's rows below
      const double* P = reinterpret_cast<const double*>(o.L) + o.n + off + i;
#pragma unroll 8
      for (int k = threadIdx.x / kOzM; k < o.n; k += kOzSliceThreads / kOzM)
        fmax = max(fmax, oz_exp_field(P[(int64_t)k * o.m]));
    }
  }
  s_f[threadIdx.x] = fmax;
  cp_async_wait_all();
  __syncthreads();
  const int64_t row0 = tk.z + (int64_t)r0;
  const size_t stride = (size_t)oz_rows * kOzRowBytes;
  static_assert(kOzSliceThreads == 2 * kOzM, "two threads a row");
  if (threadIdx.x < kOzM) {
    const int i = threadIdx.x;
    // the largest entry's exponent field by integer comparison (the FP64 unit is slow):
    // max |x| = f 2^e with f in [0.5, 1) has e = field - 1022 (0 for rows of zeros and
    // subnormals, whose slices are zero)
    int emax = max(s_f[i], s_f[i + kOzM]);  // of the row scaled by 2^-t_k (exponent fields shifted by -t_k)
    for (int k = 0; k < n; k++) {
      const int f = oz_exp_field(xs[k * kOzSliceLd + i]);
      if (f > 0) emax = max(emax, f - s_t[k]);
    }
    const int e = oz_row_exponent(emax);
    s_e[i] = e;
    if (i < rows) reinterpret_cast<int32_t*>(oz + kOzSlices * stride)[row0 + i] = e;
  }
  __syncthreads();
  for (int item = threadIdx.x; item < kOzM * 8; item += kOzSliceThreads) {
    const int i = item >> 3, pc = item & 7;  // row, physical 16-byte chunk
    if (i >= rows) continue;
    const int R7 = (int)((row0 + i) & 7);
    const int c = pc ^ (oy ? R7 : R7 >> 1);  // logical chunk: columns 8c .. 8c+7
    uint8_t* dst = oy ? oz + (size_t)(row0 + i) * kOzRowBytes + pc * 16
                      : oz + ((size_t)(pc >> 2) * oz_rows + row0 + i) * kOzUnitRow + (pc & 3) * 16;
    const int e = s_e[i];
    long long R[8];
#pragma unroll
    for (int j = 0; j < 8; j++) {
      const int k = 8 * c + j;
      R[j] = k < n ? oz_fixed(xs[k * kOzSliceLd + i], e + s_t[k]) : 0;  // x 2^-t_k
    }
    oz_write_chunk(R, dst, stride);
  }
}

// Eight accumulator columns of this warp's 32 TMEM lanes (one row per thread); the caller
// waits (tcgen05.wait::ld) before using them.
__device__ __forceinline__ void oz_tmem_load8(uint32_t addr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(addr));
}

__device__ __forceinline__ void oz_tmem_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The FP32 bits of x + 1.5 * 2^23 for an accumulator x holding an integer of magnitude at most
// 2^22: 0x4B400000 + x, i.e. the integer plus a fixed offset in the low mantissa bits.
__device__ __forceinline__ uint32_t oz_fbits(uint32_t acc) {
  return __float_as_uint(__uint_as_float(acc) + 12582912.0f);
}
__device__ __forceinline__ int oz_int(uint32_t acc) { return __float2int_rn(__uint_as_float(acc)); }

// s d 2^E with a subnormal or infinite result (out of line: the consumers' code is long enough)
template <bool NEG>
__device__ __noinline__ double oz_scale(double d, int E) {
  const double r = ldexp(d, E);
  return NEG ? -r : r;
}

// s W 2^E as a double (s = -1 when NEG), rounded to nearest (ties to even): the FP64 unit's
// int64 -> double conversion, then an add to the exponent field and, for NEG, to the sign bit
// (exact inside the normal range; a signed zero for W = 0, ldexp outside the range).  The FP64 unit is otherwise
// idle in this kernel, and one conversion there costs the consumer warps far fewer issue slots
// than normalizing and rounding the 64-bit integer with integer operations.
template <bool NEG>
__device__ __forceinline__ double oz_to_double(long long W, int E) {
  const double d = __ll2double_rn(W);
  const uint32_t hi = (uint32_t)__double2hiint(d);
  const int be = (int)((hi >> 20) & 0x7ffu) + E;
  if (hi == 0u) return NEG ? -0.0 : 0.0;  // W = 0: adds nothing (-0.0 leaves every sum as it is)
  if ((unsigned)(be - 1) < 2046u)
    return __hiloint2double((int)(hi + (uint32_t)E * 1048576u + (NEG ? 0x80000000u : 0u)),
                            __double2loint(d));
  return oz_scale<NEG>(d, E);
}

constexpr int kOzMaxRuns = 8;  // column targets per task whose relative rows are cached
constexpr int kOzMetaBufs = 2;  // metadata buffers: the metadata warps run up to one task ahead

// Per-task metadata, in kOzMetaBufs buffers: the metadata warps build the next task's copy
// while the consumers scatter with the current one.
struct OzMeta {
  double* cp[kOzM];  // each column's target panel column (its relative rows are added)
  long long rb[kOzM];  // relative-map base of every run
  int eA[kOzM], eB[kOzM];  // row exponents e_i; column exponents e_k - 55
  int rp[kOzMaxRuns][kOzM];  // relative rows (while building, rp[0]: each column's target)
  uint8_t run[kOzM];
  int u, uc, i0, k0;       // the task: update order, end of its columns, tile origin
  const int32_t* relmap;   // for runs beyond the cached ones
  double* ustage;          // owner assembly: this supernode's staged U
};
// ... and what only its construction needs
static_assert(kOzM == 128, "the run count sums four 32-column words; a run index fits a byte");
struct OzMetaWork {
  uint8_t run_start[kOzM];
  int wcnt[kOzM / 32];  // run starts per 32 columns
  int fcnt[kOzMetaThreads / 32];  // the supernode's runs before the tile, per warp
};

// A task as the load thread hands it to the other roles.
struct OzTask {
  int s, i0, k0;  // supernode, tile origin in its off-diagonal rows
  int oz;         // slice row of its off-diagonal row 0
  int oz0;        // a merged chunk before it (n0 > 0): slice row of the same row
  int kend;       // columns from here on are not this task's (the update's order, or a group's inner columns)
  int n0, n;      // K: columns of the chunk before (0: none) and of s; n < 0: stop
};

// Task ti of segment g (SchurSeg); sns: the descriptors.  A strip's tiles
// follow one another, so that later ones reuse the A rows.
__device__ __forceinline__ OzTask oz_task(const SchurSeg& g, int ti, const SnDev* __restrict__ sns) {
  const SnDev& d = sns[g.s];
  int y = ti - g.first, a = 0;
  OzTask t;
  t.s = g.s;
  t.oz = g.oz;
  t.oz0 = g.w;
  t.n = d.n;
  t.n0 = 0;
  t.kend = d.m - d.n;
  if (g.kind == kSegInner) {
    const int nc = (g.w + 127) >> 7;  // column tiles: strip a has min(a + 1, nc)
    while (a + 1 < nc && y > a) y -= ++a;
    if (a + 1 == nc) {
      a += y / nc;
      y %= nc;
    }
    t.kend = g.w;
  } else {
    if (g.kind == kSegOuter) t.n0 = sns[g.s - 1].n;
    // strip a: a + 1 tiles after a (a + 1) / 2
    a = (int)((sqrtf(8.f * (float)y + 1.f) - 1.f) * 0.5f);
    while (a * (a + 1) / 2 > y) a--;
    while ((a + 1) * (a + 2) / 2 <= y) a++;
    y -= a * (a + 1) / 2;
  }
  t.i0 = 128 * a;
  t.k0 = 128 * y;
  return t;
}

// barrier among the metadata warps only
__device__ __forceinline__ void oz_meta_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kOzMetaThreads) : "memory");
}

__device__ __forceinline__ void oz_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// A task is done as 128 x 32 quarters, a quarter in steps of one unit of K (32 columns).  A load
// thread (its own warp) claims the tasks, hands each one to the other roles through a ring as soon
// as it has claimed it, and bulk-copies per step the quarter's B slices of the unit into one of
// kOzBBufs buffers and the unit's A slices into one of kOzABufs, unless they are still there: the
// units of K = 128 (4 x 56 KB) do not fit, so successive quarters take them in alternating
// directions and the buffer used longest ago is replaced, one unit of four per quarter; at K = 64
// every unit stays for a whole strip of tiles.  An MMA thread (its own warp) issues each
// step's MMAs into one of two TMEM sets of 7
// diagonals x 32 columns, slice by slice; the 16 consumer warps drain a finished set (and
// release it) while the tensor cores compute the next quarter, then scatter; four metadata
// warps build each task's exponents, column targets and relative rows one task ahead.
// Barriers: b_full[] / b_empty[] (a step's B, and its A if that was copied for it, in / the step's
// MMAs done, which also frees its A buffer), acc_full[2] (a set's MMAs done), acc_empty[2] (a set
// drained), meta_full[] / meta_empty[] (a metadata buffer built / released), ring_full[]
// (the task order).
template <bool OWNER>
__global__ void __launch_bounds__(kOzThreads, 1)
    k_schur_oz(const SchurSeg* __restrict__ segs, int nsegs, int ntasks, int* __restrict__ queue,
               const SnDev* __restrict__ sns, const MatDev* __restrict__ mats,
               const uint8_t* oz, int64_t oz_rows, long long acc_wait,
               const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b) {
  extern __shared__ __align__(512) unsigned char oz_sm[];
  unsigned char* A =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(oz_sm) + 511) & ~uintptr_t(511));
  unsigned char* Bq0 = A + kOzABufs * kOzUA;
  __shared__ __align__(8) uint64_t b_full[kOzBBufs], b_empty[kOzBBufs];
  __shared__ int step[kOzBBufs];  // the step in a B buffer: see kStep...
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2];
  __shared__ __align__(8) uint64_t ring_full[kOzRing];
  __shared__ OzTask ring[kOzRing];
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t meta_full[kOzMetaBufs], meta_empty[kOzMetaBufs];
  __shared__ OzMeta meta[kOzMetaBufs];
  __shared__ OzMetaWork mw;
  __shared__ __align__(8) uint64_t never;  // test hook: a barrier nothing completes
  __shared__ int s_mgo;  // the metadata warps go on with the next task (0: stop)
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  pdl_wait();
  // a launch of this factorization already gave up on a wait: its updates are missing and the
  // factorization is reported failed, so skip the work below -- the whole CTA, or none of it
  // (another CTA may be recording a timeout of this launch): decided at the set-up's barrier, which the
  // loads' way there overlaps (a barrier of its own took 1 us a launch, 49.5 -> 49.75 ms at 48^3)
  const bool gave_up = *(volatile unsigned long long*)(mats[sns[segs[0].s].mat].err + 3) != 0;
  const size_t stride = (size_t)oz_rows * kOzRowBytes;
  const int32_t* exps = reinterpret_cast<const int32_t*>(oz + kOzSlices * stride);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base)),
                 "r"(kOzTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    s_fail = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&never)));
    for (int i = 0; i < kOzBBufs; i++) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&b_full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&b_empty[i])));
    }
    for (int i = 0; i < 2; i++) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&acc_full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&acc_empty[i])),
                   "r"(kOzConsumers / 64));  // the 8 warps of the set's consumer group
    }
    for (int i = 0; i < kOzRing; i++)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&ring_full[i])));
    for (int i = 0; i < kOzMetaBufs; i++) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&meta_full[i])),
                   "r"(kOzMetaThreads));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&meta_empty[i])),
                   "r"(kOzConsumers / 32));
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  const bool skip = __syncthreads_or(gave_up);
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  if (skip) {
    record_timeout(nsegs, sns, mats, [&](int i) { return segs[i].s; });
    __syncwarp();
    if (warp == 0)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"(kOzTmemCols));
    return;
  }

  if (warp == kOzLoadWarp) {
    // ---------------- loads: task claims, ring, tiled copies; one thread ----------------
    if (lane == 0) {
      int st = 0;                            // steps issued (B buffer st % kOzBBufs)
      // the A buffers: the unit in each (slice row, half) and the last step that reads it
      int arow[kOzABufs] = {-1, -1, -1}, ahalf[kOzABufs] = {0, 0, 0};
      int alast[kOzABufs] = {-3, -2, -1};
      bool down = false;                     // the next quarter takes its units from the last on
      int ord = 0;                           // ring entries published
      bool ok = true;
      // Tasks are claimed in runs (g0 per CTA at first, then from the queue): four while more
      // than 16 per CTA remain, then two while more than 4 do, then singles: the tasks of a
      // row strip are consecutive in the list, so the later tasks of a run usually have the
      // first one's A rows, which stay in shared memory.
      const int g0 = ntasks >= 8 * (int)gridDim.x ? 4 : (ntasks >= 4 * (int)gridDim.x ? 2 : 1);
      int tq = g0 * (int)blockIdx.x;         // a CTA's first run follows its block index
      int tend = min(tq + g0, ntasks);       // end of the claimed run
      // The ring runs one task ahead of the copies: a task is published (and the next one
      // claimed) before the current task's copies are issued, so that the metadata warps
      // can build its targets while the current task is still being copied and computed.
      int sg = -1;  // the segment of the last published task
      SchurSeg seg;
      seg.first = seg.count = 0;
      auto publish = [&](int ti) -> OzTask {
        OzTask t;
        t.n = -1;
        if (ti < ntasks) {
          if (ti >= seg.first + seg.count) {  // the next segment, or a search among the later ones
            int lo = sg + 1, hi = nsegs - 1;
            if (lo < hi && ti < segs[lo + 1].first) hi = lo;
            while (lo < hi) {
              const int mid = (lo + hi + 1) >> 1;
              if (segs[mid].first <= ti) lo = mid; else hi = mid - 1;
            }
            sg = lo;
            seg = segs[sg];
          }
          t = oz_task(seg, ti, sns);
        }
        const int rs = ord % kOzRing;
        ring[rs] = t;
        oz_arrive(smem_u32(&ring_full[rs]));
        ord++;
        return t;
      };
      // the B buffer of the next step, once the MMAs of the step before it there are done
      auto b_wait = [&]() -> bool {
        return st < kOzBBufs ||
               oz_wait(smem_u32(&b_empty[st % kOzBBufs]), (uint32_t)((st / kOzBBufs - 1) & 1));
      };
      int cur = tq;
      OzTask t = publish(cur);
      while (cur < ntasks) {
        if (++tq >= tend) {  // the run is done: claim the next one
          const int g = tq < ntasks - 16 * (int)gridDim.x ? 4
                        : (tq < ntasks - 4 * (int)gridDim.x ? 2 : 1);
          tq = g0 * (int)gridDim.x >= ntasks ? ntasks
                                             : g0 * (int)gridDim.x + atomicAdd(queue, g);
          tend = min(tq + g, ntasks);
        }
        const OzTask next = publish(tq);  // the next task (or the stop entry)
        const int nq = min(4, (t.kend - t.k0 + kOzQ - 1) / kOzQ);
        const int z0 = (t.n0 + 31) >> 5, nz = z0 + ((t.n + 31) >> 5);  // units
        for (int j = 0; j < nq && ok; j++, down = !down)
          for (int zz = 0; zz < nz; zz++, st++) {
            const int z = down ? nz - 1 - zz : zz;
            const int row = z < z0 ? t.oz0 : t.oz, h = z < z0 ? z : z - z0;
            const int left = (z < z0 ? t.n0 : t.n) - 32 * h;
            ok = b_wait();
            if (!ok) break;
            int ab = 0;
            bool hit = false;
#pragma unroll
            for (int i = 0; i < kOzABufs; i++)
              if (arow[i] == row + t.i0 && ahalf[i] == h) {
                ab = i;
                hit = true;
              }
            if (!hit) {  // replace the unit used longest ago, once its last MMAs are done
#pragma unroll
              for (int i = 1; i < kOzABufs; i++)
                if (alast[i] < (ab == 0 ? alast[0] : alast[1])) ab = i;
            }
            const int b = st % kOzBBufs;
            const uint32_t bar = smem_u32(&b_full[b]);
            if (!hit) {
              const int last = ab == 0 ? alast[0] : (ab == 1 ? alast[1] : alast[2]);
              // (steps up to st - kOzBBufs are done: the wait for the B buffer)
              if (last > st - kOzBBufs && last >= 0 &&
                  !oz_wait(smem_u32(&b_empty[last % kOzBBufs]), (uint32_t)((last / kOzBBufs) & 1))) {
                ok = false;
                break;
              }
            }
#pragma unroll
            for (int i = 0; i < kOzABufs; i++)
              if (ab == i) {
                arow[i] = row + t.i0;
                ahalf[i] = h;
                alast[i] = st;
              }
            step[b] = ab | (left > 16 ? 2 : 1) << kStepK | (zz == 0 ? 1 << kStepFirst : 0) |
                      (zz == nz - 1 ? 1 << kStepLast : 0);
            // a unit of A counts on its first step's barrier: the later steps that find it come after
            oz_expect(bar, hit ? kOzUB : kOzUA + kOzUB);
            oz_unit_load(smem_u32(Bq0 + b * kOzUB), &map_b, (row + t.k0 + kOzQ * j) >> 3, h, bar);
            if (!hit) oz_unit_load(smem_u32(A + ab * kOzUA), &map_a, (row + t.i0) >> 3, h, bar);
          }
        if (!ok) break;
        t = next;
        cur = tq;
      }
      if (ok && b_wait()) {  // the stop step
        step[st % kOzBBufs] = 1 << kStepStop;
        oz_arrive(smem_u32(&b_full[st % kOzBBufs]));
        st++;
      } else {
        ok = false;
      }
      if (!ok) {
        s_fail = 1;
        const int rs = ord % kOzRing;
        ring[rs].n = -1;
        oz_arrive(smem_u32(&ring_full[rs]));
      }
      // bounded waits for the copies still in flight: the last steps'
      for (int q = max(0, st - kOzBBufs); q < st; q++)
        oz_wait(smem_u32(&b_full[q % kOzBBufs]), (uint32_t)((q / kOzBBufs) & 1));
    }
  } else if (warp == kOzMmaWarp) {
    // ---------------- MMAs: one elected thread ----------------
    // The loop over a step's MMAs is rolled and short: it shares its scheduler's instruction
    // cache with consumer warps that run through long unrolled code, and an unrolled loop was
    // refetched line by line (2,800 cycles of issuing per quarter whose MMAs take 1,930).
    if (oz_elect()) {
      // N = (7 - p) x 32: the MMA of slice p against slices 0 .. 6-p of a quarter
      const uint32_t idesc0 = oz_idesc(kOzSlices * kOzQ);
      constexpr uint32_t kIdStep = (uint32_t)(kOzQ >> 3) << 17, kAStep = kOzUASlice >> 4;
      const uint64_t da0 = oz_desc64(smem_u32(A)), db0 = oz_desc64(smem_u32(Bq0));
      bool ok = true;
      int q = 0;            // quarters issued (TMEM set q & 1)
      int bb = 0, bpar = 0;  // the step's B buffer and the parity of its use
      int st = 0;           // steps issued
      bool ready = false, drained = false;  // the next step is in / its set drained
      int snext = 0;
      uint32_t acc = 0;
      for (;; st++) {
        ok = ready || oz_wait(smem_u32(&b_full[bb]), (uint32_t)bpar);
        if (!ok) break;
        const int s = ready ? snext : *(volatile int*)&step[bb];
        if (s >> kStepStop & 1) break;
        const int ab = s & ((1 << kStepK) - 1), b = q & 1;
        if (s >> kStepFirst & 1) {
          // the set was drained (quarter q - 2)
          ok = q < 2 || drained || oz_wait(smem_u32(&acc_empty[b]), (uint32_t)(((q >> 1) - 1) & 1));
          if (!ok) break;
          acc = 0;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        // K step outer, slice inner: consecutive MMAs start at different diagonals (measured
        // 2.3x faster than issuing one slice's K steps back to back into the same columns).  The second
        // K step takes the slices from the last to the first: the largest MMAs (N = 160 to 224) then end a
        // step and, queued, keep the tensor cores busy over the commit and the next step's waits.
        uint64_t da = da0 + (uint64_t)((ab * kOzUA) >> 4), db = db0 + (uint64_t)((bb * kOzUB) >> 4);
        uint32_t col = tmem + (uint32_t)(b * kOzSetCols), id = idesc0;
#pragma unroll 1
        for (int p = 0; p < kOzSlices; p++) {
          oz_mma(col, da, db, id, acc);
          acc = 1;
          da += kAStep;
          col += kOzQ;
          id -= kIdStep;
        }
        // the next step's waits, if they are over, while these MMAs run
        const int nb = bb + 1 == kOzBBufs ? 0 : bb + 1, npar = nb == 0 ? bpar ^ 1 : bpar;
        ready = oz_test(smem_u32(&b_full[nb]), (uint32_t)npar);
        drained = false;
        if (ready) {
          snext = *(volatile int*)&step[nb];
          drained = (s >> kStepLast & 1) && q >= 1 &&
                    oz_test(smem_u32(&acc_empty[b ^ 1]), (uint32_t)(((q + 1) >> 1) - 1) & 1);
        }
        if ((s >> kStepK & 3) == 2) {
          da += 2;
          db += 2;
#pragma unroll 1
          for (int p = 0; p < kOzSlices; p++) {
            da -= kAStep;
            col -= kOzQ;
            id += kIdStep;
            oz_mma(col, da, db, id, 1u);
          }
        }
        if (s >> kStepLast & 1) {
          oz_commit(smem_u32(&acc_full[b]));
          q++;
        }
        oz_commit(smem_u32(&b_empty[bb]));
        bb = nb;
        bpar = npar;
      }
      if (!ok) s_fail = 1;
      // bounded wait for the MMAs in flight (the last step's commit covers all earlier ones)
      if (st >= 1)
        oz_wait(smem_u32(&b_empty[(st - 1) % kOzBBufs]), (uint32_t)(((st - 1) / kOzBBufs) & 1));
    }
    __syncwarp();
  } else if (warp >= kOzMetaBase / 32) {
    // ---------------- metadata warps: one thread per tile row / column ----------------
    // For each task in ring order, into meta[ord % kOzMetaBufs] once the consumers have released it:
    // the rows' and columns' slice exponents, every column's target supernode, the runs of
    // equal target (ballot per 32 columns), each column's run and column inside its target,
    // per run the relative-map base and target panel, and the relative rows of the first
    // kOzMaxRuns runs.  Thread 0 alone waits on the ring and on the buffer, so that the
    // group's decisions are uniform.
    const int mt = tid - kOzMetaBase, mwarp = mt >> 5;
    for (int ord = 0;; ord++) {
      const int buf = ord % kOzMetaBufs;
      if (mt == 0) {
        const int rs = ord % kOzRing;
        int go = 0;
        if (!oz_wait(smem_u32(&ring_full[rs]), (uint32_t)((ord / kOzRing) & 1)) ||
            (ring[rs].n >= 0 && ord >= kOzMetaBufs &&
             !oz_wait(smem_u32(&meta_empty[buf]), (uint32_t)((ord / kOzMetaBufs - 1) & 1))))
          s_fail = 1;
        else
          go = ring[rs].n >= 0;
        s_mgo = go;
      }
      oz_meta_sync();
      const int go = s_mgo;
      const OzTask tk = ring[ord % kOzRing];
      oz_meta_sync();  // s_mgo is rewritten only after every thread has read it
      if (!go) break;
      OzMeta& M = meta[buf];
      const SnDev d = sns[tk.s];
      const int n = d.n, u = d.m - n, i0 = tk.i0, k0 = tk.k0, uc = tk.kend;
      const MatDev md = mats[d.mat];
      const int gk = k0 + mt;
      // (merged chunks have the same exponents)
      M.eA[mt] = (i0 + mt < u) ? exps[tk.oz + i0 + mt] : 0;
      M.eB[mt] = (gk < uc ? exps[tk.oz + gk] : 0) - 55;  // U = W 2^(e_i + e_k - 55)
      if (mt == 0) {
        M.u = u;
        M.uc = uc;
        M.i0 = i0;
        M.k0 = k0;
        M.relmap = md.relmap;
        M.ustage = OWNER ? static_cast<double*>(md.stage) + d.ustage : nullptr;
      }
      if (!OWNER) {
        const int32_t* rows = d.rows + n;
        const int grow = gk < uc ? rows[gk] : 0;
        const int tc = gk < uc ? md.col2sn[grow] : -1;
        M.rp[0][mt] = tc;
        // the supernode's runs that start after position 0 and at or before k0: their count
        // is the index (from run0) of the run holding the tile's first column; the tile's
        // runs are that run and the ones after it, in order (runs split where the target
        // changes, and so do the tile's)
        int before = 0;
        for (int t = 1 + mt; t < d.nrun; t += kOzMetaThreads) before += md.run_a[d.run0 + t] <= k0 ? 1 : 0;
        before = __reduce_add_sync(0xffffffffu, before);
        if (lane == 0) mw.fcnt[mwarp] = before;
        oz_meta_sync();
        // a column starts a run when its target differs from its left neighbour's; its run
        // index is the number of starts up to it, less one
        const bool start = gk < uc && (mt == 0 || M.rp[0][mt - 1] != tc);
        const unsigned bl = __ballot_sync(0xffffffffu, start);
        if (lane == 0) mw.wcnt[mwarp] = __popc(bl);
        oz_meta_sync();
        int off = 0;
        for (int w2 = 0; w2 < mwarp; w2++) off += mw.wcnt[w2];
        const int first = d.run0 + mw.fcnt[0] + mw.fcnt[1] + mw.fcnt[2] + mw.fcnt[3];
        if (gk < uc) {
          const int r = off + __popc(bl & ((2u << lane) - 1u)) - 1;
          const SnDev& td = sns[md.sn_base + tc];
          M.run[mt] = (uint8_t)r;
          M.cp[mt] = reinterpret_cast<double*>(td.L) + (int64_t)(grow - td.col0) * td.m;
          if (start) {  // the run's first column fetches its map base
            mw.run_start[r] = (uint8_t)mt;
            M.rb[r] = md.run_base[first + r];
          }
        }
        oz_meta_sync();
        // relative rows of the cached runs: this thread's tile row in each, all loads in flight
        static_assert(kOzMetaThreads == kOzM, "one metadata thread per tile row");
        const int nrc = min(mw.wcnt[0] + mw.wcnt[1] + mw.wcnt[2] + mw.wcnt[3], kOzMaxRuns), g = i0 + mt;
        int rpv[kOzMaxRuns];
#pragma unroll
        for (int r = 0; r < kOzMaxRuns; r++)
          rpv[r] = (r < nrc && g < u && g >= k0 + mw.run_start[r]) ? md.relmap[M.rb[r] + g] : -1;
#pragma unroll
        for (int r = 0; r < kOzMaxRuns; r++)
          if (r < nrc) M.rp[r][mt] = rpv[r];
      }
      oz_arrive(smem_u32(&meta_full[buf]));  // each thread after its own writes
    }
  } else {
    // ---------------- consumers: set drain and scatter ----------------
    // Two groups of 8 warps, one per TMEM set: group g takes the quarters on set g (global
    // quarter index q with q & 1 == g), a warp 32 rows x 16 columns of it as two chunks of 8
    // columns.  The groups work half a quarter apart, so one group's conversions (FP64 unit)
    // overlap the other's atomics (memory pipe) instead of all 16 warps running each phase
    // at once.  A set is released after the warp's second chunk is drained.  Each wait's
    // outcome is made uniform over the warp (tcgen05.ld is warp-collective).
    const int grp = warp >> 3;
    const int i = 32 * (warp & 3) + lane;     // this thread's tile row
    const int c16 = 16 * ((warp >> 2) & 1);   // this warp's 16 columns of a quarter
    long long q0 = 0;                         // global index of the task's first quarter
    for (int ord = 0;; ord++) {
      const int rs = ord % kOzRing, buf = ord % kOzMetaBufs;
      if (!__all_sync(0xffffffffu, oz_wait(smem_u32(&ring_full[rs]), (uint32_t)((ord / kOzRing) & 1)))) {
        s_fail = 1;
        break;
      }
      if (ring[rs].n < 0) break;
      const OzMeta& M = meta[buf];
      if (!__all_sync(0xffffffffu, oz_wait(smem_u32(&meta_full[buf]), (uint32_t)((ord / kOzMetaBufs) & 1)))) {
        s_fail = 1;
        break;
      }
      const int u = M.u, uc = M.uc, i0 = M.i0, k0 = M.k0;
      const int nq = min(4, (uc - k0 + kOzQ - 1) / kOzQ);
      const int gi = i0 + i;
      const int eA = M.eA[i];
      bool stop = false;
      for (int j = 0; j < nq && !stop; j++) {
        const long long q = q0 + j;
        if ((int)(q & 1) != grp) continue;
        const int b = grp;
        // acc_wait > 0 (a test hook): wait that long on a barrier that never completes instead,
        // standing in for an accumulator that never finishes
        const bool got = acc_wait > 0 ? oz_wait(smem_u32(&never), 0u, acc_wait)
                                      : oz_wait(smem_u32(&acc_full[b]), (uint32_t)((q >> 1) & 1));
        if (!__all_sync(0xffffffffu, got)) {
          s_fail = 1;
          stop = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        for (int c = 0; c < 2; c++) {
          const int c8 = c16 + 8 * c;  // this chunk's 8 columns of the quarter
          const int kb = kOzQ * j + c8, gk0 = k0 + kb;
          const int r0w = i0 + 32 * (warp & 3);  // the warp's first tile row
          // warp-uniform: no entry of the chunk in the lower triangle of the update (past
          // its order, or above the diagonal): nothing to read but the release
          const bool dead = r0w >= u || gk0 >= uc || r0w + 31 < gk0;
          double val[8];
          if (!dead) {
            // the 7 diagonals of the chunk's columns -> W (exact integer) -> U = W 2^(e_i +
            // e_k - 55)
            const uint32_t ta =
                tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(b * kOzSetCols + c8);
            long long w[8];
            {
              uint32_t v[3][8];
#pragma unroll
              for (int dd = 0; dd < 3; dd++)
                oz_tmem_load8(ta + (uint32_t)((4 + dd) * kOzQ), v[dd]);
              oz_tmem_wait();
#pragma unroll
              for (int jj = 0; jj < 8; jj++)
                w[jj] = oz_low(oz_int(v[0][jj]), oz_int(v[1][jj]), oz_int(v[2][jj]));
            }
            {
              uint32_t v[4][8];
#pragma unroll
              for (int dd = 0; dd < 4; dd++) oz_tmem_load8(ta + (uint32_t)(dd * kOzQ), v[dd]);
              oz_tmem_wait();
#pragma unroll
              for (int jj = 0; jj < 8; jj++)
                w[jj] = oz_high(w[jj], oz_fbits(v[0][jj]), oz_fbits(v[1][jj]), oz_int(v[2][jj]),
                                oz_int(v[3][jj]));
            }
            if (c == 1) {  // the warp's last reads of this set
              asm volatile("tcgen05.fence::before_thread_sync;");
              __syncwarp();
              if (lane == 0) oz_arrive(smem_u32(&acc_empty[b]));
            }
#pragma unroll
            for (int jj = 0; jj < 8; jj++)  // -U for the atomics, U for the staging buffer
              val[jj] = oz_to_double<!OWNER>(w[jj], eA + M.eB[kb + jj]);
          } else if (c == 1) {
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) oz_arrive(smem_u32(&acc_empty[b]));
          }
          if (dead) continue;
          // scatter this thread's row of the chunk
          if (OWNER) {
            if (gi < u) {
              double* U = M.ustage;
#pragma unroll
              for (int jj = 0; jj < 8; jj++) {
                const int gk = gk0 + jj;
                if (gk < uc && gk <= gi) U[(int64_t)gk * u + gi] = val[jj];
              }
            }
          } else if (r0w + 31 < u && gk0 + 7 < uc && gk0 + 7 <= r0w &&
                     M.run[kb] == M.run[kb + 7]) {
            // warp-uniform fast path: every entry live, one target run for all 8 columns
            const int r = M.run[kb];
            const int p = r < kOzMaxRuns ? M.rp[r][i] : M.relmap[M.rb[r] + gi];
            if (p >= 0) {
#pragma unroll
              for (int jj = 0; jj < 8; jj++) red_add(M.cp[kb + jj] + p, val[jj]);
            }
          } else if (gi < u) {
            // the relative row changes only with the run, which is the same for every lane
            int rprev = -1, p = -1;
#pragma unroll
            for (int jj = 0; jj < 8; jj++) {
              const int kk = kb + jj, gk = k0 + kk;
              if (gk >= uc || gk > gi) continue;
              const int r = M.run[kk];
              if (r != rprev) {
                rprev = r;
                p = r < kOzMaxRuns ? M.rp[r][i] : M.relmap[M.rb[r] + gi];
              }
              if (p >= 0) red_add(M.cp[kk] + p, val[jj]);
            }
          }
        }
      }
      if (stop) break;
      q0 += nq;
      __syncwarp();
      if (lane == 0) oz_arrive(smem_u32(&meta_empty[buf]));
    }
  }
  __syncthreads();
  if (s_fail) record_timeout(nsegs, sns, mats, [&](int i) { return segs[i].s; });
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kOzTmemCols));
}

// ---- TRSM of the 128-tile supernodes on the tensor cores ----------------------------------
// L21 = A21 L11^{-T} = A21 Y^T with Y = L11^{-1}, formed by POTRF, which also stored the
// slices of Y S (S = diag(2^t_k), t_k the exponent of L11[k,k]) and the shifts t_k in oy; the
// slices of A21 S^-1 come from the slicing kernel run on the panel just before.  L21 =
// (A21 S^-1)(Y S)^T is a product of row-sliced operands of exactly the Schur tiles' form,
// L21[i, j] = 2^(e_i + e_j) sum_{p+q<7} 2^(-14-8(p+q)) sum_k a_p[i,k] y_q[j,k], K = n <= 64, so
// every diagonal's partial sums are exact in FP32 and the combination is
// the same integer one.  A task is 128 rows of A21.  A CTA per SM takes consecutive tasks: a load and
// MMA thread (its own warp) bulk-copies a task's 7 A slices (112 KB) and, for another supernode than
// before, Y's 7 slices (64 rows each, 56 KB), then issues, per K step and A
// slice p, the MMAs of A_p against Y slices 0 .. 6-p in one go (N = (7-p) 64, at most 256 per
// MMA): diagonal p + q lands at TMEM columns (p + q) 64.
// Eight warps read the accumulators (warp w: TMEM lanes 32 (w & 3) .., columns
// 32 (w >> 2) ..), combine them exactly, round once to FP64 and store L21 into the panel, while the
// next task's slices are on their way.  A CTA per task did these one after another, each at its
// latency: per 80^3 27-point factorization 47.3 -> 29.9 ms, 48^3 6.4 -> 4.6 ms.
// (Forming the slices inside this kernel as well was measured slower: one CTA per SM then
// serializes the slicing, the copies and the tensor work, which separate launches overlap.)
// Waits are bounded as in the Schur tiles; a timeout is recorded in err[3] and ends the CTA.
constexpr int kToWarps = 8;                       // of the epilogue
constexpr int kToThreads = 32 * (kToWarps + 1);
constexpr uint32_t kToBSlice = kOzInvRows * kOzRowBytes;  // 8 KB: one slice of Y's rows
constexpr uint32_t kToBBytes = kOzSlices * kToBSlice;      // 56 KB
constexpr size_t kToSmem = 1024 + kOzABytes + kToBBytes;   // + alignment slack
constexpr uint32_t kToTmemCols = 512;                      // 7 diagonals of 64 columns

__global__ void __launch_bounds__(kToThreads, 1)
    k_trsm_oz(const int4* __restrict__ tasks, int ntasks, const SnDev* __restrict__ sns,
              const MatDev* __restrict__ mats, const uint8_t* oz, int64_t oz_rows, const uint8_t* oy,
              int64_t oy_rows) {
  extern __shared__ __align__(1024) unsigned char to_sm[];
  unsigned char* A =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(to_sm) + 1023) & ~uintptr_t(1023));
  unsigned char* B = A + kOzABytes;
  __shared__ __align__(8) uint64_t full, done, drained;
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int e0 = (int)((long long)ntasks * blockIdx.x / gridDim.x);
  const int e1 = (int)((long long)ntasks * (blockIdx.x + 1) / gridDim.x);
  pdl_wait();
  // a launch of this factorization already gave up on a wait: skip (as in k_schur_oz)
  const bool gave_up = *(volatile unsigned long long*)(mats[sns[tasks[e0].x].mat].err + 3) != 0;
  const size_t sa = (size_t)oz_rows * kOzRowBytes, sb = (size_t)oy_rows * kOzRowBytes;
  const int32_t* ea = reinterpret_cast<const int32_t*>(oz + kOzSlices * sa);
  const int32_t* ey = reinterpret_cast<const int32_t*>(oy + kOzSlices * sb);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base)),
                 "r"(kToTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    s_fail = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&done)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&drained)), "r"(kToWarps));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  const bool skip = __syncthreads_or(gave_up);
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  if (skip) {
    record_timeout(e1 - e0, sns, mats, [&](int i) { return tasks[e0 + i].x; });
    __syncwarp();
    if (warp == 0)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"(kToTmemCols));
    return;
  }
  if (warp == kToWarps) {
    if (lane == 0) {
      const uint32_t fb = smem_u32(&full), db = smem_u32(&done);
      const uint64_t ad = oz_desc(smem_u32(A)), bd = oz_desc(smem_u32(B));
      bool ok = true;
      int it = 0, yrow = -1;  // tasks issued; the supernode whose Y is in B
      for (int e = e0; e < e1 && ok; e++) {
        const int4 tk = tasks[e];
        if (tk.w < 0) continue;  // the supernode keeps the FP64 TRSM
        // the MMAs of the task before have read A and B
        if (it > 0 && !oz_wait(db, (uint32_t)((it - 1) & 1))) {
          ok = false;
          break;
        }
        const bool newy = tk.w != yrow;
        yrow = tk.w;
        oz_expect(fb, newy ? kOzABytes + kToBBytes : kOzABytes);
        const uint8_t* arow = oz + (size_t)((int64_t)tk.z + tk.y) * kOzRowBytes;
        for (int p = 0; p < kOzSlices; p++)
          oz_bulk_load(smem_u32(A + p * kOzASlice), arow + p * sa, kOzASlice, fb);
        if (newy)
          for (int p = 0; p < kOzSlices; p++)
            oz_bulk_load(smem_u32(B + p * kToBSlice), oy + p * sb + (size_t)yrow * kOzRowBytes,
                         kToBSlice, fb);
        const int ks = (sns[tk.x].n + 15) >> 4;
        ok = oz_wait(fb, (uint32_t)(it & 1));
        if (!ok) {
          oz_wait(fb, (uint32_t)(it & 1));  // bounded: the copies in flight
          break;
        }
        if (it > 0 && !oz_wait(smem_u32(&drained), (uint32_t)((it - 1) & 1))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        // K step outer, A slice inner (consecutive MMAs start at different diagonals); the
        // first K step of slice 0 writes every diagonal, everything after accumulates
        for (int k = 0; k < ks; k++)
          for (int p = 0; p < kOzSlices; p++)
            for (int q0 = 0; q0 < kOzSlices - p; q0 += 4) {
              const int nq = min(4, kOzSlices - p - q0);
              oz_mma(tmem + (uint32_t)((p + q0) * kOzInvRows),
                     ad + (uint64_t)((p * kOzASlice) >> 4) + 2 * k,
                     bd + (uint64_t)((q0 * kToBSlice) >> 4) + 2 * k, oz_idesc(nq * kOzInvRows),
                     (p > 0 || k > 0) ? 1u : 0u);
            }
        oz_commit(db);
        it++;
      }
      if (!ok) s_fail = 1;
      if (it > 0) oz_wait(db, (uint32_t)((it - 1) & 1));  // bounded: the MMAs in flight
    }
    __syncwarp();
  } else {
    const int lq = warp & 3, ch = warp >> 2;
    const int i = 32 * lq + lane;  // this thread's row of a task
    int it = 0;
    for (int e = e0; e < e1; e++) {
      const int4 tk = tasks[e];
      if (tk.w < 0) continue;
      const SnDev d = sns[tk.x];
      const int n = d.n, m = d.m, r0 = tk.y, rb = min(kOzM, m - n - r0);
      const int eA = i < rb ? ea[(int64_t)tk.z + r0 + i] - 55 : 0;
      const int eY = ey[tk.w + 32 * ch + lane];  // of column 32 ch + lane
      double* out = reinterpret_cast<double*>(d.L) + n + r0 + i;
      if (!__all_sync(0xffffffffu, oz_wait(smem_u32(&done), (uint32_t)(it & 1)))) {
        s_fail = 1;
        break;
      }
      it++;
      asm volatile("tcgen05.fence::after_thread_sync;");
      for (int c8 = 0; c8 < 4; c8++) {
        const int col0 = 32 * ch + 8 * c8;
        uint32_t v[kOzSlices][8];
#pragma unroll
        for (int dd = 0; dd < kOzSlices; dd++)
          oz_tmem_load8(tmem + ((uint32_t)(32 * lq) << 16) + (uint32_t)(dd * kOzInvRows + col0), v[dd]);
        oz_tmem_wait();
        if (c8 == 3) {  // the warp's last reads
          asm volatile("tcgen05.fence::before_thread_sync;");
          __syncwarp();
          if (lane == 0) oz_arrive(smem_u32(&drained));
        }
#pragma unroll
        for (int j = 0; j < 8; j++) {
          const int col = col0 + j;
          const int E = eA + __shfl_sync(0xffffffffu, eY, 8 * c8 + j);
          if (i < rb && col < n) {
            const long long lo = oz_low(oz_int(v[4][j]), oz_int(v[5][j]), oz_int(v[6][j]));
            const long long W =
                oz_high(lo, oz_fbits(v[0][j]), oz_fbits(v[1][j]), oz_int(v[2][j]), oz_int(v[3][j]));
            out[(int64_t)col * m] = oz_to_double<false>(W, E);
          }
        }
      }
    }
  }
  __syncthreads();
  if (s_fail) record_timeout(e1 - e0, sns, mats, [&](int i) { return tasks[e0 + i].x; });
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kToTmemCols));
}

static int oz_sms() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

void launch_trsm_oz(const int4* tasks, int ntasks, const SnDev* sns, const MatDev* mats,
                    const void* oz, int64_t oz_rows, const void* oy, int64_t oy_rows,
                    cudaStream_t st) {
  if (ntasks <= 0) return;
  launch_pdl(k_trsm_oz, std::min(ntasks, oz_sms()), kToThreads, kToSmem, st, tasks, ntasks, sns, mats,
             static_cast<const uint8_t*>(oz), oz_rows, static_cast<const uint8_t*>(oy), oy_rows);
}

void launch_oz_slice(const int4* tasks, int ntasks, const SnDev* sns, void* oz, int64_t oz_rows,
                     const void* oy, int64_t oy_rows, cudaStream_t st) {
  if (ntasks <= 0) return;
  launch_pdl(k_oz_slice, ntasks, kOzSliceThreads, (size_t)64 * kOzSliceLd * sizeof(double), st, tasks,
             sns, static_cast<uint8_t*>(oz), oz_rows, static_cast<const uint8_t*>(oy), oy_rows);
}

size_t oy_scratch_bytes(int64_t oy_rows) {
  return oz_scratch_bytes(oy_rows) + (size_t)oy_rows * sizeof(int32_t);
}

// The slices as units for tiled copies: dimensions {8 rows of a unit (512 bytes, as FP64 elements),
// groups of 8 rows, halves of K, slices}, boxes of `rows` rows and all slices.  One copy per unit: with
// bulk copies (one per slice and unit, 144 a tile at K = 128) the load thread issued for 22,000 of a
// tile's 28,800 cycles.
static decltype(&cuTensorMapEncodeTiled) tensor_map_encode() {
  static const auto fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult r;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &r) !=
            cudaSuccess ||
        r != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<decltype(&cuTensorMapEncodeTiled)>(p);
  }();
  return fn;
}
static bool oz_unit_map(CUtensorMap* map, const void* oz, int64_t oz_rows, int rows) {
  const cuuint64_t dim[4] = {64, (cuuint64_t)(oz_rows / 8), 2, kOzSlices};
  const cuuint64_t stride[3] = {8 * kOzUnitRow, (cuuint64_t)oz_rows * kOzUnitRow,
                                (cuuint64_t)oz_rows * kOzRowBytes};
  const cuuint32_t box[4] = {64, (cuuint32_t)(rows / 8), 1, kOzSlices}, one[4] = {1, 1, 1, 1};
  const auto fn = tensor_map_encode();
  return fn && fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4, const_cast<void*>(oz), dim, stride, box, one,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int launch_schur_oz(const int4* segs, int nsegs, int ntasks, int* queue, const SnDev* sns,
                    const MatDev* mats, bool owner, const void* oz, int64_t oz_rows,
                    long long acc_wait, cudaStream_t st) {
  if (ntasks <= 0) return CHOL_OK;
  CUtensorMap map_a, map_b;
  if (!oz_unit_map(&map_a, oz, oz_rows, kOzM) || !oz_unit_map(&map_b, oz, oz_rows, kOzQ))
    return CHOL_E_CUDA;
  const int grid = std::min(ntasks, oz_sms());  // one resident CTA per SM, tasks by queue
  const uint8_t* z = static_cast<const uint8_t*>(oz);
  const SchurSeg* sg = reinterpret_cast<const SchurSeg*>(segs);
  launch_pdl(owner ? k_schur_oz<true> : k_schur_oz<false>, grid, kOzThreads, kOzSmem, st, sg, nsegs, ntasks,
             queue, sns, mats, z, oz_rows, acc_wait, map_a, map_b);
  return CHOL_OK;
}

int64_t oz_stride_rows(int64_t oz_rows) {
  return (int64_t)(oz_scratch_bytes(oz_rows) / (kOzSlices * kOzRowBytes + sizeof(int32_t)));
}

size_t oz_scratch_bytes(int64_t oz_rows) {
  return (size_t)oz_rows * (kOzPlanes * kOzRowBytes + sizeof(int32_t));
}

int set_oz_kernel_attrs() {
  if (!tensor_map_encode()) return CHOL_E_CUDA;
  if (cudaFuncSetAttribute(k_oz_slice, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(64 * kOzSliceLd * sizeof(double))) != cudaSuccess ||
      cudaFuncSetAttribute(k_schur_oz<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kOzSmem) != cudaSuccess ||
      cudaFuncSetAttribute(k_schur_oz<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kOzSmem) != cudaSuccess ||
      cudaFuncSetAttribute(k_trsm_oz, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kToSmem) != cudaSuccess)
    return CHOL_E_CUDA;
  return CHOL_OK;
}

}  // namespace chol
