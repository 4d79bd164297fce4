// sp_dense.cu -- continuous-input projections (Section 2.3: for continuous
// inputs the INT8 weights are converted to FP32, multiplied with the FP32
// activations and accumulated, and the row scale is applied after; Section
// 2.2: these projections keep row-major weights, one contiguous dot product
// per output):
//
//   y[b][m] = s_m * sum_k float(W[m * ldw + k]) * x[b][k]
//
// for B <= 4 activation rows and up to 128 problems per launch (e.g. the
// query/key/value, attention-output and FFN up projections of every block of a
// decode step).  The weights stream from HBM once per call, so the kernel is
// HBM-bound: algorithmic bytes = sum over problems of N * K.
//
// Two forms.
//
// dense_mma_kernel<B>: the products run on the tensor cores and stay exact.
// An INT8 weight is a bf16 value exactly, and a normal FP32 activation is the
// exact sum of three bf16 values (its 24 significant bits in three runs of 8:
// x = hi + mid + lo), so every bf16 x bf16 product of mma.sync m16n8k16 is an
// exact part of the FP32 product and only the additions round.  Per warp: 16
// weight rows as the MMA's M, the split activations of all B rows as its N
// (columns 4 b + {0, 1, 2} = hi, mid, lo of row b), 64 weight columns per
// chunk.  Every MMA starts from zero, the sums of a chunk's four meet in pairs
// and are added to the running FP32 sums of the lane; at the end
// y = s * (hi + (mid + lo)).  How an MMA rounds its sum of 16 products is not
// specified; on this device each product is cut to a multiple of 2^-24 of the
// largest one's leading power of two and the sum to 24 bits.  So 16 products
// lose at most 17 units u = 2^-24 of sum |W x|, the two additions of a chunk 2,
// the running sum one per chunk and the three parts 2: depth 22 + ceil(K / 64).
// (With the four MMAs of a chunk chained through their accumulator a large
// product cost 63 others their last bits: 24.5 units measured at K = 64, 8.6 this way,
// 10.7 with FMAs.  The additions are packed two to an instruction: for
// four rows 1 to 2 us a call, nothing for one.)  Relative error (2-norm, K =
// 1536, N(0, 1) activations) 8.2e-8, against 1.4e-7 with FMAs.
// Bounds and layout:
//   - with FP32 FMAs the kernel is bound by instructions and L1 (per weight a
//     byte permute, an FADD and B FFMAs, and every lane re-reads the
//     activations).  The MMA takes the multiplications for all B rows at
//     once; what is left per 4 weights is 5 logic operations and 2 packed
//     subtractions (byte -> bf16: 128 + low 7 bits, minus 128 or 256).
//   - lane (g, t) copies 16 bytes of rows g and g + 8 (four lanes share 64
//     bytes of a row) with cp.async into its own slots of an 8-chunk ring and
//     reads them back itself: 128 KB in flight per SM, no barrier, and no
//     registers held by loads (a register ring of the same depth was slower,
//     83 and 91 us against 72 and 75 for one and four rows below: it shares
//     the six load scoreboards of a warp).  The K order inside a chunk is
//     permuted alike on both operands.
//   - the split activations of the CTA's problems are made once, in shared
//     memory, in the order of the MMA's B operand (1 KB per 64 columns and two
//     activation rows), while the first ring is in flight.
//   - one 512-thread CTA per SM takes an equal, contiguous share of the
//     launch's chunks, so that it meets one or two activation tables.
// Measured on 66 projections (4608 / 1536 / 6144 x 1536, 415 MB), by the machine:
// 70.8 to 74.8 us for one activation row (5.9 to 5.6 TB/s) and 74.0 to 78.2 for
// four; with dense_kernel 81 and 260 us.
//
// dense_kernel<B> (small launches, and K whose table does not fit): a unit
// is 4 consecutive rows of one problem, owned by one warp.  Lane l
// covers the 16-column chunks l, l + 32, l + 64, ... of the row (16-byte
// weight loads, 512 contiguous bytes per warp instruction), issuing the loads
// of one chunk of all 4 rows before any arithmetic.  A weight byte
// becomes a float exactly through its bias (w + 128 in the low byte of 2^23's
// mantissa, minus 2^23 + 128).  Each lane accumulates with fmaf in ascending
// k, the 32 lane sums meet in a 5-level butterfly, and one FP32 multiply by s_m
// gives y: an FP32 sum of K products of depth at most 16 * ceil(K / 512) + 5.
// Its small CTAs start while the previous kernel drains: 2.2 us a call at
// 0.5 MB, where the tensor-core form, which fills its SM, takes 4.1.
// dense_mma_kernel runs an activation row with FMAs too when one of its values
// is not finite or outside 2^-100 .. 2^100 (its three parts would not be exact).
//
// In both forms the order of a sum depends on K alone, so the result is the
// same on every run, and a row's does not depend on the other rows of the call
// or on the other problems of the launch, but through the choice of the form,
// which goes by the sizes of the whole launch.
#include <algorithm>

#include "sp_ptx.cuh"
#include "sp_rows.cuh"
#include "sp_spikes.cuh"

namespace sp {
namespace {

constexpr int kDenseRows = 4;        // rows per unit (one warp)
constexpr int kDenseThreads = 256;
// Per activation count B: 16-column chunks per lane loaded per round, and
// CTAs per SM the registers must allow.  One chunk of 4 rows per round: the
// converted weights stay in registers for the B activation rows, and more
// warps with less in flight each stream faster than fewer warps with three
// chunks (measured on 415 MB of weights: B = 1 at 32 warps per SM 5.1 TB/s
// against 3.6 with three chunks; B = 2 / 3 / 4 at 16 warps per SM 2.9 / 2.3 /
// 1.7 TB/s against 2.5 / 1.6 / 1.3).
template <int B> struct DenseShape { static constexpr int batch = 1, min_ctas = 2; };
template <> struct DenseShape<1> { static constexpr int batch = 1, min_ctas = 4; };

template <int B> constexpr uint32_t kAllRows = (1u << B) - 1u;

struct DenseParams {
  int32_t count, B;
  int32_t units;                       // total over problems
  DenseProblem prob[kDenseMaxProblems];
  int32_t unit_end[kDenseMaxProblems]; // prefix sums of each problem's units
};

// y of rows row0 .. row0 + nrows - 1 (nrows <= 4) of P for the activation rows
// in `rows` (bit b: row b), by one warp with FP32 FMAs.
template <int B>
__device__ __forceinline__ void dense_rows(const DenseProblem& P, int row0, int nrows, uint32_t rows) {
  constexpr int kDenseBatch = DenseShape<B>::batch;
  const int lane = threadIdx.x & 31;
  const int nch = (P.K + 511) / 512;        // chunk rounds of the whole warp
  float acc[kDenseRows][B];
#pragma unroll
  for (int r = 0; r < kDenseRows; ++r)
#pragma unroll
    for (int b = 0; b < B; ++b) acc[r][b] = 0.f;

  for (int i0 = 0; i0 < nch; i0 += kDenseBatch) {
    // weights: one chunk x 4 rows of 16 bytes in flight
    uint4 w[kDenseRows][kDenseBatch];
#pragma unroll
    for (int c = 0; c < kDenseBatch; ++c) {
      const int k = 16 * (lane + 32 * (i0 + c));
#pragma unroll
      for (int r = 0; r < kDenseRows; ++r) {
        w[r][c] = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);   // biased zeros
        if (k < P.K && r < nrows) {
          // the row is ldw >= K bytes with ldw % 16 == 0: the 16 bytes at k
          // lie inside it; bytes at or past K meet a zero activation
          const uint4 v = ld_weights16(P.W + (int64_t)(row0 + r) * P.ldw + k);
          w[r][c] = make_uint4(v.x ^ 0x80808080u, v.y ^ 0x80808080u, v.z ^ 0x80808080u,
                               v.w ^ 0x80808080u);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < kDenseBatch; ++c) {
      const int k = 16 * (lane + 32 * (i0 + c));
      if (k >= P.K) continue;
#pragma unroll
      for (int b = 0; b < B; ++b) {
        float xv[16];
        load_x16(P.x + (int64_t)b * P.ldx, k, P.K, xv);
#pragma unroll
        for (int r = 0; r < kDenseRows; ++r) {
          const uint32_t ww[4] = {w[r][c].x, w[r][c].y, w[r][c].z, w[r][c].w};
#pragma unroll
          for (int e = 0; e < 16; ++e)
            acc[r][b] = fmaf(byte_to_float(ww[e >> 2], (uint32_t)(e & 3)), xv[e], acc[r][b]);
        }
      }
    }
  }
  // butterfly over the 32 lanes; every lane ends with the full sums
#pragma unroll
  for (int r = 0; r < kDenseRows; ++r)
#pragma unroll
    for (int b = 0; b < B; ++b)
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) acc[r][b] += __shfl_xor_sync(0xffffffffu, acc[r][b], d);
#pragma unroll
  for (int r = 0; r < kDenseRows; ++r)
#pragma unroll
    for (int b = 0; b < B; ++b)
      if (lane == r * B + b && r < nrows && (rows >> b & 1u))
        P.y[(int64_t)b * P.ldy + row0 + r] = __fmul_rn(__ldg(P.scale + row0 + r), acc[r][b]);
}

template <int B>
__global__ void __launch_bounds__(kDenseThreads, DenseShape<B>::min_ctas)
dense_kernel(const __grid_constant__ DenseParams p) {
  pdl_launch_dependents();
  pdl_wait();
  const int nwarps = gridDim.x * (kDenseThreads / 32);
  int j = 0;                                   // problem of the current unit (units ascend)
  for (int u = blockIdx.x * (kDenseThreads / 32) + (threadIdx.x >> 5); u < p.units; u += nwarps) {
    while (u >= p.unit_end[j]) ++j;
    const DenseProblem& P = p.prob[j];
    const int row0 = (u - (j ? p.unit_end[j - 1] : 0)) * kDenseRows;
    dense_rows<B>(P, row0, min(kDenseRows, P.N - row0), kAllRows<B>);
  }
}

// ---- tensor-core form -----------------------------------------------------------
constexpr int kMmaRows = 16;                 // weight rows per unit (MMA M)
constexpr int kMmaChunk = 64;                // weight columns per chunk (16 bytes per lane and row)
constexpr int kMmaThreads = 512;
constexpr int kMmaWarps = kMmaThreads / 32;
constexpr int kMmaRing = 8;                  // chunks in flight per warp (1 KB each)

// activation table: per chunk and 8-column tile, 2 x 32 16-byte groups
constexpr int kMmaTile = 1024;
constexpr int kMmaRingBytes = kMmaWarps * kMmaRing * kMmaRows * kMmaChunk;
constexpr int kMmaTableBytes = 224 * 1024 - kMmaRingBytes;

// d = A B for one 16 x 16 x 8 step.
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%10, %10, %10, %10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// Two FP32 values, added each by itself (round to nearest) in one instruction.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair(const float (&d)[4], int e) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(d[2 * e]), "f"(d[2 * e + 1]));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__device__ __forceinline__ void cp_async16(uint4* dst, const int8_t* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Bytes 0 and 2 of w (INT8) as two bf16: 128 + (low 7 bits), whose bf16
// pattern is 0x4300 | bits, minus 128 (or 256 where the sign bit is set:
// 0x4380).  Exact.  one28 = 0x43004300, in a register: with the mask as the
// immediate each and-or is one instruction (as two immediates it is two).
__device__ __forceinline__ uint32_t bytes02_bf16(uint32_t w, uint32_t one28) {
  uint32_t m, c, r;
  asm("lop3.b32 %0, %1, 0x007f007f, %2, 0xEA;" : "=r"(m) : "r"(w), "r"(one28));
  asm("lop3.b32 %0, %1, 0x00800080, %2, 0xEA;" : "=r"(c) : "r"(w), "r"(one28));
  asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(m), "r"(c));
  return r;
}

// The three bf16 parts of a and b packed as (a, b) pairs: out[0] hi, out[1]
// mid, out[2] lo.  Each part takes the leading 8 significant bits of what is
// left (truncation), so the parts sum to the value exactly.
__device__ __forceinline__ void split3(float a, float b, uint32_t (&out)[3]) {
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const uint32_t ua = __float_as_uint(a) & 0xffff0000u, ub = __float_as_uint(b) & 0xffff0000u;
    out[s] = (ua >> 16) | ub;
    a = __fsub_rn(a, __uint_as_float(ua));
    b = __fsub_rn(b, __uint_as_float(ub));
  }
}

// The parts of v are exact bf16 values (0, or 2^-100 <= |v| <= 2^100).
__device__ __forceinline__ bool splits_exactly(float v) {
  const float a = fabsf(v);
  return a == 0.f || (a >= 0x1p-100f && a <= 0x1p100f);
}

struct DenseMmaParams {
  int32_t count;
  int32_t table_bytes;                 // shared memory for activation tables
  uint32_t one28;                      // two bf16 128 (bytes02_bf16)
  int64_t cost;                        // chunks of all units
  DenseProblem prob[kDenseMaxProblems];
  int32_t unit_end[kDenseMaxProblems]; // prefix sums of each problem's 16-row units
  int64_t cost_end[kDenseMaxProblems]; // prefix sums of each problem's chunks
};

// One unit of the tensor-core form with FP32 FMAs, for some activation rows.
template <int B>
__device__ __forceinline__ void dense_unit_fma(const DenseProblem& P, int row0, uint32_t rows) {
  for (int r = row0; r < row0 + kMmaRows && r < P.N; r += kDenseRows)
    dense_rows<B>(P, r, min(kDenseRows, P.N - r), rows);
}

template <int B>
__global__ void __launch_bounds__(kMmaThreads, 1)
dense_mma_kernel(const __grid_constant__ DenseMmaParams p) {
  constexpr int NT = (B + 1) / 2;      // 8-column MMA tiles: two activation rows each
  extern __shared__ __align__(16) uint8_t smem[];
  uint8_t* s_tab = smem + kMmaRingBytes;
  __shared__ uint32_t s_fma[kDenseMaxProblems];  // problem j0 + i: activation rows that do not split exactly
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const uint32_t one28 = p.one28;
  // this lane's landing slots: each lane reads only what it copied
  uint4* ring = reinterpret_cast<uint4*>(smem) + warp * (64 * kMmaRing) + lane;
  pdl_launch_dependents();

  // this CTA's units: an equal share of the launch's chunks (a unit belongs
  // to the CTA that its first chunk falls to)
  int range[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int64_t c = p.cost * ((int)blockIdx.x + e) / (int)gridDim.x;
    int lo = 0, hi = p.count - 1;      // the problem holding chunk c
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (c < p.cost_end[mid]) hi = mid;
      else lo = mid + 1;
    }
    const int nch = (p.prob[lo].K + kMmaChunk - 1) / kMmaChunk;
    const int64_t at = c - (lo ? p.cost_end[lo - 1] : 0);
    const int u = (lo ? p.unit_end[lo - 1] : 0) + (int)((at + nch - 1) / nch);
    range[e] = min(u, p.unit_end[p.count - 1]);
  }
  pdl_wait();

  int j0 = 0;
  for (int u0 = range[0]; u0 < range[1];) {
    // ---- a segment: the units of the problems whose tables fit together ----
    while (u0 >= p.unit_end[j0]) ++j0;
    int used = 0, j1 = j0;
    while (j1 < p.count && (j1 == j0 || range[1] > p.unit_end[j1 - 1])) {
      const bool same = j1 > j0 && p.prob[j1].x == p.prob[j1 - 1].x && p.prob[j1].K == p.prob[j1 - 1].K &&
                        p.prob[j1].ldx == p.prob[j1 - 1].ldx;
      if (!same) {
        const int bytes = (p.prob[j1].K + kMmaChunk - 1) / kMmaChunk * (NT * kMmaTile);
        if (used + bytes > p.table_bytes) break;
        used += bytes;
      }
      ++j1;
    }
    const int u1 = min(range[1], p.unit_end[j1 - 1]);

    bool any_fma = false;
    // ---- the weight ring: chunks of this warp's units, kMmaRing ahead --------
    // Units are padded to whole rings, so slot s always holds a chunk s mod
    // kMmaRing.  Rows past N and columns past K are clamped to the last row and
    // the row's last 16 bytes: such a row's sums are not written and such a
    // column meets zero activations.
    int lu = u0 + warp, lj = j0, lc = 0, lch = 0, lK = 0;
    const int8_t *q0 = nullptr, *q1 = nullptr;
    auto open_unit = [&]() {
      while (lu < u1) {                  // the next unit of this warp that runs here
        while (lu >= p.unit_end[lj]) ++lj;
        if (!any_fma || s_fma[lj - j0] != kAllRows<B>) break;
        lu += kMmaWarps;
      }
      lc = lch = 0;
      if (lu >= u1) return;
      const DenseProblem& P = p.prob[lj];
      const int row = (lu - (lj ? p.unit_end[lj - 1] : 0)) * kMmaRows + g;
      lK = P.K;
      lch = (lK + kMmaChunk - 1) / kMmaChunk;
      q0 = P.W + (int64_t)min(row, P.N - 1) * P.ldw + 16 * t;
      q1 = P.W + (int64_t)min(row + 8, P.N - 1) * P.ldw + 16 * t;
    };
    // slot s of the ring that starts at chunk lc of the open unit
    auto load = [&](int s) {
      if (lc + s < lch) {
        const int over = max(0, (lc + s) * kMmaChunk + 16 * t - (lK - 1) / 16 * 16);
        cp_async16(ring + 64 * s, q0 + (s * kMmaChunk - over));
        cp_async16(ring + 64 * s + 32, q1 + (s * kMmaChunk - over));
      }
      cp_async_commit();
      if (s == kMmaRing - 1) {           // the next ring of the unit, or the next unit
        lc += kMmaRing;
        q0 += kMmaRing * kMmaChunk;
        q1 += kMmaRing * kMmaChunk;
        if (lc >= lch && lch > 0) {
          lu += kMmaWarps;
          open_unit();
        }
      }
    };
    open_unit();
#pragma unroll
    for (int s = 0; s < kMmaRing; ++s) load(s);

    // ---- the activation tables of the segment --------------------------------
    for (int i = threadIdx.x; i < kDenseMaxProblems; i += kMmaThreads) s_fma[i] = 0;
    __syncthreads();
    int bad = 0;
    {
      int base = 0;
      for (int j = j0; j < j1; ++j) {
        const DenseProblem& P = p.prob[j];
        if (j > j0 && P.x == p.prob[j - 1].x && P.K == p.prob[j - 1].K && P.ldx == p.prob[j - 1].ldx) continue;
        const int nch = (P.K + kMmaChunk - 1) / kMmaChunk;
        for (int i = threadIdx.x; i < nch * 4 * B; i += kMmaThreads) {
          const int tt = i & 3, b = (i >> 2) % B, c = (i >> 2) / B;
          float x[16];
          load_x16(P.x + (int64_t)b * P.ldx, c * kMmaChunk + 16 * tt, P.K, x);
          uint4* dst = reinterpret_cast<uint4*>(s_tab + base + (c * NT + (b >> 1)) * kMmaTile) +
                       (b & 1) * 16 + tt;
          bool exact = true;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            // MMAs 2 h and 2 h + 1 of the chunk: columns (0, 2), (1, 3) of each
            uint32_t o[4][3];
#pragma unroll
            for (int m = 0; m < 2; ++m) {
              const float* xm = x + 8 * h + 4 * m;
              split3(xm[0], xm[2], o[2 * m]);
              split3(xm[1], xm[3], o[2 * m + 1]);
#pragma unroll
              for (int e = 0; e < 4; ++e) exact = exact && splits_exactly(xm[e]);
            }
#pragma unroll
            for (int s = 0; s < 3; ++s)
              dst[32 * h + 4 * s] = make_uint4(o[0][s], o[1][s], o[2][s], o[3][s]);
          }
          if (!exact) {
            bad = 1;
            atomicOr(&s_fma[j - j0], 1u << b);
          }
        }
        base += nch * NT * kMmaTile;
      }
    }
    any_fma = __syncthreads_or(bad) != 0;
    if (any_fma) {
      // rare: those activation rows (of each problem that shares them) with
      // FP32 FMAs; the loops below do not write them, and leave out a problem
      // of none but such rows.  (A row's products stay in its own columns of
      // the MMA: what they are does not reach the other rows.)
      if (threadIdx.x == 0)
        for (int j = j0 + 1; j < j1; ++j)
          if (p.prob[j].x == p.prob[j - 1].x && p.prob[j].K == p.prob[j - 1].K && p.prob[j].ldx == p.prob[j - 1].ldx)
            s_fma[j - j0] = s_fma[j - 1 - j0];
      __syncthreads();
      for (int u = u0 + warp, j = j0; u < u1; u += kMmaWarps) {
        while (u >= p.unit_end[j]) ++j;
        const int row0 = (u - (j ? p.unit_end[j - 1] : 0)) * kMmaRows;
        if (s_fma[j - j0]) dense_unit_fma<B>(p.prob[j], row0, s_fma[j - j0]);
      }
      // the ring again, without them
      cp_async_wait<0>();
      lu = u0 + warp;
      lj = j0;
      open_unit();
#pragma unroll 1
      for (int s = 0; s < kMmaRing; ++s) load(s);
    }

    // ---- the units -------------------------------------------------------------
    int j = j0, base = 0;
    for (int u = u0 + warp; u < u1; u += kMmaWarps) {
      while (u >= p.unit_end[j]) {
        const DenseProblem &P = p.prob[j], &Q = p.prob[j + 1];
        if (!(P.x == Q.x && P.K == Q.K && P.ldx == Q.ldx)) {
          base += (P.K + kMmaChunk - 1) / kMmaChunk * (NT * kMmaTile);
        }
        ++j;
      }
      const uint32_t skip = any_fma ? s_fma[j - j0] : 0u;
      if (skip == kAllRows<B>) continue;
      const DenseProblem& P = p.prob[j];
      const int row0 = (u - (j ? p.unit_end[j - 1] : 0)) * kMmaRows;
      const int nch = (P.K + kMmaChunk - 1) / kMmaChunk;
      f32x2 run[NT][2];
#pragma unroll
      for (int n = 0; n < NT; ++n) run[n][0] = run[n][1] = 0ull;
      const uint4* tab = reinterpret_cast<const uint4*>(s_tab + base) + lane;
      for (int c0 = 0; c0 < nch; c0 += kMmaRing) {
#pragma unroll
        for (int s = 0; s < kMmaRing; ++s) {
          cp_async_wait<kMmaRing - 1>();   // this lane's copies of the chunk have landed
          if (c0 + s < nch) {
            const uint4 w0 = ring[64 * s], w1 = ring[64 * s + 32];
            const uint32_t wa[4] = {w0.x, w0.y, w0.z, w0.w};
            const uint32_t wb[4] = {w1.x, w1.y, w1.z, w1.w};
            const uint4* tc = tab + (c0 + s) * NT * (kMmaTile / 16);
            f32x2 chunk[NT][2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              float part[2][NT][4];
              uint4 bf[NT];
#pragma unroll
              for (int n = 0; n < NT; ++n) bf[n] = tc[n * (kMmaTile / 16) + 32 * h];
#pragma unroll
              for (int m = 0; m < 2; ++m) {
                const uint32_t va = wa[2 * h + m], vb = wb[2 * h + m];
                const uint32_t a0 = bytes02_bf16(va, one28), a1 = bytes02_bf16(vb, one28);
                const uint32_t a2 = bytes02_bf16(va >> 8, one28), a3 = bytes02_bf16(vb >> 8, one28);
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                  const uint32_t b0 = m ? bf[n].z : bf[n].x, b1 = m ? bf[n].w : bf[n].y;
                  mma_bf16(part[m][n], a0, a1, a2, a3, b0, b1);
                }
              }
#pragma unroll
              for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                  const f32x2 sum = add2(pair(part[0][n], e), pair(part[1][n], e));
                  if (h == 0) chunk[n][e] = sum;
                  else run[n][e] = add2(run[n][e], add2(chunk[n][e], sum));
                }
            }
          }
          load(s);
        }
      }
      // lanes t = 0, 2 hold hi and mid of activation row 2 n + t / 2, lanes
      // t = 1, 3 its lo
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float a0 = __uint_as_float((uint32_t)run[n][e]), a1 = __uint_as_float((uint32_t)(run[n][e] >> 32));
          const float lo = __shfl_xor_sync(0xffffffffu, a0, 1);
          const float sum = __fadd_rn(a0, __fadd_rn(a1, lo));
          const int b = 2 * n + (t >> 1), row = row0 + g + 8 * e;
          if ((t & 1) == 0 && b < B && row < P.N && !(skip >> b & 1u))
            P.y[(int64_t)b * P.ldy + row] = __fmul_rn(__ldg(P.scale + row), sum);
        }
    }
    __syncthreads();                   // the tables are rebuilt by the next segment
    u0 = u1;
  }
}

// Resident CTAs of dense_kernel<B> per SM.
template <int B>
int dense_ctas_per_sm(int dev) {
  static PerDevice ctas;
  return ctas.get(dev, []() {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, dense_kernel<B>, kDenseThreads, 0) != cudaSuccess)
      (void)cudaGetLastError();
    return n > 0 ? n : 1;
  });
}

template <int B>
cudaError_t launch_dense_t(const DenseParams& p, int dev, int sms, cudaStream_t s) {
  // one wave of resident CTAs (never more than the units need): every unit a
  // warp takes from the grid-stride sequence starts without waiting for a CTA
  const int warps_per_cta = kDenseThreads / 32;
  int grid = sms * dense_ctas_per_sm<B>(dev);
  const int need = (p.units + warps_per_cta - 1) / warps_per_cta;
  if (grid > need) grid = need;
  if (grid < 1) grid = 1;
  return launch_pdl(dense_kernel<B>, dim3(grid), dim3(kDenseThreads), 0, s, p);
}

template <int B>
cudaError_t launch_dense_mma(const DenseMmaParams& p, int dev, int sms, cudaStream_t s) {
  static PerDevice attr;
  const cudaError_t e = attr.once(dev, []() {
    return cudaFuncSetAttribute(dense_mma_kernel<B>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kMmaRingBytes + kMmaTableBytes);
  });
  if (e != cudaSuccess) return e;
  return launch_pdl(dense_mma_kernel<B>, dim3(sms), dim3(kMmaThreads),
                    (size_t)(kMmaRingBytes + p.table_bytes),
                    s, p);
}

// Whether two consecutive problems share one activation table.
bool same_table(const DenseProblem& a, const DenseProblem& b) {
  return a.x == b.x && a.K == b.K && a.ldx == b.ldx;
}

// Bytes of shared memory for the activation tables: two of the largest where
// they fit.
int table_bytes(int largest) { return 2 * largest <= kMmaTableBytes ? 2 * largest : largest; }

// The faster form by a model of both, or the tensor cores where FMAs win by less
// than 15 % (their sums err 0.6 times as much), us per call:
//   FMAs          a + b (K rounds of a warp) + c (warp rounds per SM) + d MB, by B
//   tensor cores  3.4 + 0.136 per chunk that a warp takes one after another + 0.134 MB
//                 + 2.2 where a CTA meets a second activation table, + 2.6 (three rows
//                 or four) where the two do not fit together
// A unit is 16 rows of one warp, so the tensor-core form pays for few units per
// warp (a warp alone reads a wide row from a ring of 8 KB) and for uneven ones
// (16.1 units a CTA take two rounds of 16 warps), and a launch of many small
// problems for its tables.  Fitted on 2153 launches of 1.5 to 200 MB (K = 64 to
// 6144, 1 to 66 problems, weights in L2 and from HBM), each timed in both forms:
// error 9 %, and 0.997 of the rate of always taking the faster one.  (By a line on
// the bytes alone 0.987, with launches at up to twice their time: 64 problems of 52
// x 3000, three rows, 14.2 us by FMAs and 24.8; 64 of 66 x 6144, one row, 14.4 and 35.3.
// The 66 problems of a decode step, one row and four, take 81 and 260 by FMAs, 71
// to 75 and 74 to 78 on the tensor cores.)
bool mma_is_faster(const DenseProblem* probs, int count, int B, int sms) {
  constexpr double kFma[SPIKE_PROJ_DENSE_MAX_B][4] = {
      {3.4, 0.70, 0.044, -0.015}, {3.2, 0.83, 0.059, 0.021}, {2.9, 1.28, 0.058, 0.076}, {3.0, 1.57, 0.070, 0.121}};
  const auto ring = [](int nch) { return ceil_div(nch, kMmaRing) * kMmaRing; };
  int64_t cost = 0, quads = 0, rounds = 0;                 // chunks; units of 4 rows, their K rounds
  double mb = 0;
  int most = 0, wide = 0;
  for (int j = 0; j < count; ++j) {
    const DenseProblem& P = probs[j];
    const int nch = ceil_div(P.K, kMmaChunk);
    cost += (int64_t)ceil_div(P.N, kMmaRows) * nch;
    quads += ceil_div(P.N, kDenseRows);
    rounds += (int64_t)ceil_div(P.N, kDenseRows) * ceil_div(P.K, 512);
    mb += 1e-6 * P.N * P.K;
    if (nch > most) most = nch;
    if (ceil_div(P.K, 512) > wide) wide = ceil_div(P.K, 512);
  }
  const int64_t warps = (int64_t)sms * (kDenseThreads / 32) * (B == 1 ? DenseShape<1>::min_ctas : DenseShape<2>::min_ctas);
  const double serial_fma =
      quads <= warps ? wide : (double)((quads + warps - 1) / warps) * rounds / quads;
  const double* f = kFma[B - 1];
  const double fma = f[0] + f[1] * serial_fma + f[2] * rounds / sms + f[3] * mb;

  const int tiles = (B + 1) / 2;
  const int fits = table_bytes(most * tiles * kMmaTile);
  int64_t serial = cost / ((int64_t)sms * kMmaWarps);
  bool second = false, apart = false;
  int64_t at = 0;                                          // chunk at which problem j + 1 begins
  for (int j = 0; j < count; ++j) {
    const int nch = ceil_div(probs[j].K, kMmaChunk);
    const int64_t mine = ceil_div(probs[j].N, kMmaRows);
    const int64_t units = std::min(mine, (cost + (int64_t)sms * nch - 1) / ((int64_t)sms * nch));   // of one CTA
    serial = std::max(serial, (units + kMmaWarps - 1) / kMmaWarps * ring(nch));
    at += mine * nch;
    if (j + 1 == count || same_table(probs[j], probs[j + 1])) continue;
    const int next = ceil_div(probs[j + 1].K, kMmaChunk);
    const int64_t cta = at * sms / cost;                   // the CTA whose share that chunk is in
    const int64_t before = std::min(mine, (at - cost * cta / sms) / nch);   // its units of the two problems
    const int64_t after = std::min<int64_t>(ceil_div(probs[j + 1].N, kMmaRows),
                                            (cost * (cta + 1) / sms - at + next - 1) / next);
    if (before < 1 || after < 1) continue;
    second = true;
    if ((nch + next) * tiles * kMmaTile > fits) {
      apart = true;
      serial = std::max(serial, (before + kMmaWarps - 1) / kMmaWarps * ring(nch) +
                                    (after + kMmaWarps - 1) / kMmaWarps * ring(next));
    }
  }
  const double mma = 3.4 + 0.136 * serial + 0.134 * mb + (second ? 2.2 : 0.0) + (apart && B > 2 ? 2.6 : 0.0);
  return mma < 1.15 * fma;
}

}  // namespace

cudaError_t launch_dense(const DenseProblem* probs, int count, int B, cudaStream_t s) {
  int dev = 0, sms = 0;
  const cudaError_t e = current_device(&dev, &sms);
  if (e != cudaSuccess) return e;
  // The tensor-core form where an activation table fits in shared memory, the
  // weights outweigh its start (it holds a whole SM, so it cannot start beside
  // the previous kernel), and it is modelled to be the faster one.
  constexpr int64_t kMmaMinBytes[SPIKE_PROJ_DENSE_MAX_B] = {24 << 20, 9 << 20, 3 << 20, 3 << 19};
  int maxK = 0;
  int64_t bytes = 0;
  for (int j = 0; j < count; ++j) {
    maxK = probs[j].K > maxK ? probs[j].K : maxK;
    bytes += (int64_t)probs[j].N * probs[j].K;
  }
  const int table = ceil_div(maxK, kMmaChunk) * ((B + 1) / 2) * kMmaTile;
  if (table <= kMmaTableBytes && bytes >= kMmaMinBytes[B - 1] && mma_is_faster(probs, count, B, sms)) {
    DenseMmaParams p;
    p.count = count;
    p.one28 = 0x43004300u;
    p.table_bytes = table_bytes(table);
    int units = 0;
    int64_t cost = 0;
    for (int j = 0; j < count; ++j) {
      const int n = ceil_div(probs[j].N, kMmaRows);
      p.prob[j] = probs[j];
      units += n;
      cost += (int64_t)n * ceil_div(probs[j].K, kMmaChunk);
      p.unit_end[j] = units;
      p.cost_end[j] = cost;
    }
    p.cost = cost;
    switch (B) {
      case 1: return launch_dense_mma<1>(p, dev, sms, s);
      case 2: return launch_dense_mma<2>(p, dev, sms, s);
      case 3: return launch_dense_mma<3>(p, dev, sms, s);
      default: return launch_dense_mma<4>(p, dev, sms, s);
    }
  }
  DenseParams p;
  p.count = count;
  p.B = B;
  int units = 0;
  for (int j = 0; j < count; ++j) {
    p.prob[j] = probs[j];
    units += (probs[j].N + kDenseRows - 1) / kDenseRows;
    p.unit_end[j] = units;
  }
  for (int j = count; j < kDenseMaxProblems; ++j) p.unit_end[j] = units;
  p.units = units;
  switch (B) {
    case 1: return launch_dense_t<1>(p, dev, sms, s);
    case 2: return launch_dense_t<2>(p, dev, sms, s);
    case 3: return launch_dense_t<3>(p, dev, sms, s);
    default: return launch_dense_t<4>(p, dev, sms, s);
  }
}

}  // namespace sp
