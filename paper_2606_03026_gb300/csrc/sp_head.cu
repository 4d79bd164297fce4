// sp_head.cu -- vocabulary head with INT8 activations and candidate-row
// verification (Section 5, trace configuration; Appendix D), two launches per
// call for up to 4 hidden states:
//
//   1. s_x = max(max_k |h_k|, 1e-8) / 127, q_k = clip(rint(h_k / s_x), +-127)
//      (the weight quantiser of Section 2.3 read onto the hidden vector)
//   2. a_m = sum_k Q[m][k] q_k (exact INT32), z_m = s_m * (s_x * float(a_m))
//   3. order by z descending (equal z: lower row first); gap = z_(1) - z_(2)
//   4. gate: verification when gap < tau
//   5. the k_sel first rows are recomputed with the FP32 activations,
//      r_m = s_m * sum_k float(Q[m][k]) h_k (the continuous-input rule)
//   6. token = the candidate with the largest r (equal r: lower row), or,
//      without verification, the first row of the order.
//
// Steps 1-4 reach exactly the definition's values: the codes and the scale
// come from the same IEEE operations, the integer sums are order-free and z
// is two RN multiplies, so z, the gap, the gate and the candidate rows are
// bit-identical to the definition's.  r is an FP32 sum (per lane in ascending
// k, then a 5-level butterfly: depth 16 * ceil(K / 512) + 5), within the
// usual FP32 dot-product bound of the exact value.
//
// Layout of the work.  The weights stream from HBM once (V * K bytes) and
// dominate the traffic.  Projection (head_kernel, one 512-thread CTA per SM):
// every CTA builds the INT8 codes of all hidden states in shared memory.  A
// pair of warps owns units of 16 consecutive rows, each warp half of the
// unit's 64-column chunks: lane (g, t) copies 16 bytes of rows g and g + 8
// with cp.async into its own slots of a 6-chunk ring (96 KB in flight per SM,
// no barrier and no registers held by loads) and reads them back itself.  One
// hidden state takes __dp4a; several take mma.sync m16n8k32 on INT8 with the
// weights as A and the states as B, so that a weight byte is read from shared
// memory once whatever B.  (Units of whole rows per warp left the last of 1.5
// rounds to half the warps: 8 us of 29; halves make about three rounds.)  A
// per-B dp4a form cost 61 us at B = 4: 128 registers, 16 warps, and 80
// shuffles and 4 list insertions per 4 rows.
//
// Each z becomes a 64-bit key (z's order-preserving bits, then the complement
// of the row, so that one unsigned comparison orders by z descending and row
// ascending; keys are distinct).  A pair keeps its best 64 keys: the first 64
// as they come (a vocabulary of 57,344 has 48 rows per pair, and sorting
// them cost 8 us a call at B = 4), later ones by a bitonic sort and merge.
// At the end every list goes to the workspace, and the 8 best keys of each
// CTA beside it.
//
// Selection (head_select_kernel, a cluster of 4 CTAs per hidden state, the
// programmatic dependent of the projection): the bound T is the 64th largest
// of the CTAs' best keys; the leading keys >= T (about eighty) are gathered
// (the lists of a CTA are fetched only when all 8 of its leading keys pass),
// ordered by counting, gated, and the candidates recomputed, two rows per
// warp.  Its CTAs are small enough in registers, shared memory and carve-out
// to run beside a projection CTA: a projection CTA that had to wait for a
// selection's SM held up the call by 7 us.
//
// Projection of one state beyond L2 (head_wide_kernel): there the ring's stream is
// the slower one (5.3 TB/s at the margin, whatever its depth, its lane layout or
// the work per chunk; the register loads 7), and the call takes register loads.
//
// Measured on 57,344 x 1536, us a call through the binding: four states 31.7
// (60.4 with a dp4a form per state and one selecting CTA), one state 23.1 to 24.1
// (23.6: no gain; the weights are 14 of it, the codes 1.3, the selection and the
// two hand-offs 6).
#include "sp_internal.h"
#include "sp_ptx.cuh"
#include "sp_rows.cuh"
#include "sp_spikes.cuh"

namespace sp {
namespace {

constexpr int kHeadThreads = 512;
constexpr int kHeadWarps = kHeadThreads / 32;
constexpr int kHeadRegs = 80;                 // registers per thread: the selection's CTAs fit beside the projection's
constexpr int kHeadRows = 16;                 // rows per unit (a pair of warps)
constexpr int kHeadChunk = 64;                // columns of one ring slot (a 16-byte vector of two rows per lane)
constexpr int kHeadRing = 6;                  // slots in flight per warp (1 KB each)
constexpr int kCodePad = 64;                  // bytes between the states' codes (their reads then miss each other's banks)
constexpr size_t kHeadRingBytes = (size_t)kHeadWarps * kHeadRing * kHeadRows * kHeadChunk;
constexpr int kHeadLists = kHeadWarps / 2;    // lists of a projection CTA (one per pair of warps)
constexpr int kHeadList = SPIKE_PROJ_HEAD_MAX_CAND;   // keys per list
constexpr int kHeadMaxGrid = 160;             // projection CTAs of one call
constexpr int kWideThreads = 1024;            // head_wide_kernel: a CTA per SM, 4 rows and a list per warp
constexpr int kWideWarps = kWideThreads / 32;
constexpr int kWideRows = 4;
constexpr int64_t kWideBytes = (int64_t)110 << 20;
constexpr int kSelThreads = 256;              // threads of a selection CTA
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelCluster = 4;                // selection CTAs of one hidden state
constexpr int kCtaLead = 8;                   // leading keys of each projection CTA read first
constexpr int kSelCand = 512;                 // keys that the bound may pass
constexpr int kSelLong = 16;                  // projection CTAs read in full
static_assert(kHeadList == 64, "a list is two keys per lane");
static_assert(kHeadRingBytes + SPIKE_PROJ_HEAD_MAX_B * (SPIKE_PROJ_HEAD_MAX_K + kCodePad) <= 212 * 1024, "shared memory per CTA");
static_assert((size_t)SPIKE_PROJ_HEAD_MAX_B * kHeadLists * kHeadList * 8 <= kHeadRingBytes, "the lists fit the ring");
static_assert(kHeadLists * kCtaLead == 64, "the pairs' leading keys: two per lane of one warp");
static_assert(kWideWarps <= SPIKE_PROJ_HEAD_MAX_B * kHeadLists, "one state's lists fit the workspace");
static_assert(SPIKE_PROJ_HEAD_MAX_CAND * kCtaLead <= kSelCand, "the leading keys of 64 CTAs");
static_assert(kHeadMaxGrid <= kSelThreads, "one projection CTA per selection thread");
static_assert(kHeadList == 2 * kSelWarps * kSelCluster, "two candidates per selection warp");

typedef unsigned long long hkey;

// Workspace: the lists (list q of projection CTA c, hidden state b: list
// (b * nctas + c) * nlists + q), then each CTA's leading keys; all of it
// is rewritten by every call.
constexpr size_t kListBytes = (size_t)SPIKE_PROJ_HEAD_MAX_B * kHeadMaxGrid * kHeadLists * kHeadList * 8;
constexpr size_t kLeadBytes = (size_t)SPIKE_PROJ_HEAD_MAX_B * kHeadMaxGrid * kCtaLead * 8;

struct HeadParams {
  const int8_t* W;
  int64_t ldw;
  const float* scale;
  int32_t V, K, Kpad, units;
  const float* h;
  int64_t ldh;
  float tau;
  int32_t k_sel;
  int32_t* token;
  int32_t* verified;
  float* gap;
  int32_t* cand;
  float* r;
  float* z;
  int64_t ld_z;
  int32_t B;
  hkey* lists;             // 64 keys each: one per pair of projection warps (or warp) and hidden state
  hkey* lead;              // the kCtaLead best keys of each projection CTA and hidden state
  int32_t nctas;           // CTAs of the projection kernel
  int32_t nlists;          // lists of one of them
};

// Order-preserving bits of z (both zeros map to the bits of +0).
__device__ __forceinline__ uint32_t order_bits(float z) {
  const uint32_t u = z == 0.0f ? 0u : __float_as_uint(z);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float from_order_bits(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}
// Larger key = larger z, or equal z and lower row; 0 is below every key.
__device__ __forceinline__ hkey make_key(float z, int m) {
  return ((hkey)order_bits(z) << 32) | (hkey)(0xffffffffu - (uint32_t)m);
}
__device__ __forceinline__ int key_row(hkey k) { return (int)(0xffffffffu - (uint32_t)k); }
__device__ __forceinline__ float key_z(hkey k) { return from_order_bits((uint32_t)(k >> 32)); }
__device__ __forceinline__ hkey kmax(hkey a, hkey b) { return a > b ? a : b; }
__device__ __forceinline__ hkey kmin(hkey a, hkey b) { return a < b ? a : b; }

// The warp's 32 keys (one per lane) sorted descending: lane l gets the l-th.
__device__ __forceinline__ hkey warp_sort32(hkey v, int lane) {
#pragma unroll
  for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const hkey o = __shfl_xor_sync(0xffffffffu, v, j);
      const bool lower = (lane & j) == 0;
      const bool desc = (lane & k) == 0;    // k == 32: every lane
      v = (lower == desc) ? kmax(v, o) : kmin(v, o);
    }
  return v;
}

// Sorts a bitonic sequence of 64 keys, element l in a and 32 + l in b of lane
// l, into descending order (half-cleaners of stride 32, 16, ..., 1).
__device__ __forceinline__ void warp_merge64(hkey& a, hkey& b, int lane) {
  const hkey hi = kmax(a, b), lo = kmin(a, b);
  a = hi;
  b = lo;
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    const bool lower = (lane & j) == 0;
    const hkey oa = __shfl_xor_sync(0xffffffffu, a, j);
    const hkey ob = __shfl_xor_sync(0xffffffffu, b, j);
    a = lower ? kmax(a, oa) : kmin(a, oa);
    b = lower ? kmax(b, ob) : kmin(b, ob);
  }
}

// The 64 keys of (a, b), any order, sorted descending.
__device__ __forceinline__ void sort64(hkey& a, hkey& b, int lane) {
  a = warp_sort32(a, lane);
  b = __shfl_sync(0xffffffffu, warp_sort32(b, lane), 31 - lane);   // descending, then ascending: bitonic
  warp_merge64(a, b, lane);
}

// The kCtaLead largest of the 64 keys of (a, b), any order: lane r < kCtaLead
// gets the r-th (the warp's maximum by two integer reductions each time).
__device__ __forceinline__ hkey best_of64(hkey a, hkey b, int lane) {
  hkey mine = 0ull;
#pragma unroll
  for (int r = 0; r < kCtaLead; ++r) {
    const hkey m = kmax(a, b);
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(m >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(m >> 32) == hi ? (uint32_t)m : 0u);
    const hkey best = (hkey)hi << 32 | lo;
    if (lane == r) mine = best;
    if (a == best) a = 0ull;                     // keys are distinct, the empty one apart
    else if (b == best) b = 0ull;
  }
  return mine;
}

// List (a, b) <- the best 64 of the list and the 32 keys n (one per lane), the
// insert number `held`.  The first 64 keys stay as they come; from the third
// insert on the list is kept sorted, and 32 keys below its last one are
// dropped at once.  For descending A and B of equal length, max(A_i, B_{63-i})
// holds the best 64 of both as a bitonic sequence; n is B with 32 empty keys
// appended.
__device__ __forceinline__ void list_add32(hkey& a, hkey& b, hkey n, int held, int lane) {
  if (held == 0) {
    a = n;
  } else if (held == 1) {
    b = n;
  } else {
    if (held == 2) sort64(a, b, lane);
    if (!__any_sync(0xffffffffu, n > __shfl_sync(0xffffffffu, b, 31))) return;
    n = warp_sort32(n, lane);
    b = kmax(b, __shfl_sync(0xffffffffu, n, 31 - lane));
    warp_merge64(a, b, lane);
  }
}

// (a, b) <- the best 64 of the two sorted lists (a, b) and (c, d), sorted.
__device__ __forceinline__ void list_merge(hkey& a, hkey& b, hkey c, hkey d, int lane) {
  a = kmax(a, __shfl_sync(0xffffffffu, d, 31 - lane));
  b = kmax(b, __shfl_sync(0xffffffffu, c, 31 - lane));
  warp_merge64(a, b, lane);
}

// Keys of buf[0 .. C) above k.
__device__ __forceinline__ int count_larger(const hkey* buf, int C, hkey k) {
  int larger = 0;
  int j = 0;
  for (; j + 8 <= C; j += 8) {                   // 8 loads in flight
    hkey v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = buf[j + e];
#pragma unroll
    for (int e = 0; e < 8; ++e) larger += v[e] > k;
  }
  for (; j < C; ++j) larger += buf[j] > k;
  return larger;
}

// out[0 .. 64) <- the best min(C, 64) of the C distinct keys buf[0 .. C),
// descending (each placed by counting the larger ones), 0 past C.
__device__ void rank_place(const hkey* buf, int C, hkey* out) {
  const int t = threadIdx.x, nt = blockDim.x;
  for (int i = C + t; i < kHeadList; i += nt) out[i] = 0ull;
  for (int i = t; i < C; i += nt) {
    const int larger = count_larger(buf, C, buf[i]);
    if (larger < kHeadList) out[larger] = buf[i];
  }
  __syncthreads();
}

// r of up to 2 candidate rows (rows[j], j < n) for hidden state hb, by one
// warp: per row, lane l sums the 16-byte chunks l, l + 32, ... in ascending k
// with fmaf, then the 5-level butterfly (the continuous-input kernel's
// order); the loads of all the rows and of up to 4 chunks are in flight
// together.
__device__ __forceinline__ void verify_rows2(const HeadParams& p, const float* hb, const int (&rows)[2],
                                             int n, int lane, float (&out)[2]) {
  const int nch = (p.K + 511) / 512;
  float acc[2] = {0.f, 0.f};
  for (int c0 = 0; c0 < nch; c0 += 4) {
    uint4 v[2][4];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int k = 16 * (lane + 32 * (c0 + t));
        if (j < n && c0 + t < nch && k < p.K) v[j][t] = ld_weights16(p.W + (int64_t)rows[j] * p.ldw + k);
      }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int k = 16 * (lane + 32 * (c0 + t));
      if (c0 + t < nch && k < p.K) {
        float x[16];
        load_x16(hb, k, p.K, x);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (j < n) {
            const uint32_t ww[4] = {v[j][t].x ^ 0x80808080u, v[j][t].y ^ 0x80808080u,
                                    v[j][t].z ^ 0x80808080u, v[j][t].w ^ 0x80808080u};
#pragma unroll
            for (int e = 0; e < 16; ++e)
              acc[j] = fmaf(byte_to_float(ww[e >> 2], (uint32_t)(e & 3)), x[e], acc[j]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], d);
    out[j] = j < n ? __fmul_rn(__ldg(p.scale + rows[j]), acc[j]) : 0.f;
  }
}

// Step 1: the CTA's NT threads are dealt out over the hidden states (NT / G
// each, G = B rounded up to a power of two); each group finds its
// state's maximum |h|, and after one barrier every thread derives s_x and
// writes codes four to a word, zero from K to Kpad.  h is read again for the
// codes (from L1): kept in registers it made the code larger, and as the code
// runs once per CTA its size showed (2.3 us instead of 1.3).
template <int B, int NT, class Ring>
__device__ __forceinline__ void head_codes(const HeadParams& p, int8_t* s_codes, float* s_red, float* s_sx,
                                           const Ring& issue_ring) {
  constexpr int G = B == 1 ? 1 : B == 2 ? 2 : 4;
  constexpr int T = NT / G;                      // threads of one hidden state
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = (int)threadIdx.x / T, tt = (int)threadIdx.x % T;
  const float* hb = p.h + (int64_t)(b < B ? b : 0) * p.ldh;
  const auto load4 = [&](int k) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k + 4 <= p.K) {
      v = __ldg(reinterpret_cast<const float4*>(hb + k));   // h 16-byte aligned, ldh % 4 == 0
    } else if (k < p.K) {
      v.x = __ldg(hb + k);
      if (k + 1 < p.K) v.y = __ldg(hb + k + 1);
      if (k + 2 < p.K) v.z = __ldg(hb + k + 2);
    }
    return v;
  };
  const auto pack = [&](const float4& v, int k, float sx) {
    const float e[4] = {v.x, v.y, v.z, v.w};
    uint32_t packed = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = k + j < p.K ? (int)fminf(fmaxf(rintf(__fdiv_rn(e[j], sx)), -127.0f), 127.0f) : 0;
      packed |= ((uint32_t)c & 0xffu) << (8 * j);
    }
    *reinterpret_cast<uint32_t*>(s_codes + b * (p.Kpad + kCodePad) + k) = packed;
  };
  const auto max4 = [&](float m, const float4& v) {
    return fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
  };
  // h is requested ahead of the weight ring, whose 96 KB per SM it would
  // otherwise queue behind (25.9 against 25.3 us a call)
  const float4 v0 = load4(4 * tt);
  issue_ring();
  float mx = max4(0.f, v0);
#pragma unroll 4
  for (int k = 4 * tt + 4 * T; k < p.K; k += 4 * T) mx = max4(mx, load4(k));
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
  if (lane == 0) s_red[warp] = mx;
  __syncthreads();
  float a = s_red[b * (T / 32)];
#pragma unroll
  for (int w = 1; w < T / 32; ++w) a = fmaxf(a, s_red[b * (T / 32) + w]);
  const float sx = __fdiv_rn(fmaxf(a, 1e-8f), 127.0f);
  if (b < B) {
    if (tt == 0) s_sx[b] = sx;
#pragma unroll 1
    for (int k = 4 * tt; k < p.Kpad; k += 4 * T) pack(k == 4 * tt ? v0 : load4(k), k, sx);
  }
  __syncthreads();
}

__device__ __forceinline__ void cp_async16(uint4* dst, const int8_t* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// d += A B for 16 rows x 32 columns of weights and 32 columns of 8 states.
__device__ __forceinline__ void mma_s8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                       uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Steps 1-2 and the CTA's lists.
template <int B>
__global__ void __maxnreg__(kHeadRegs)
head_kernel(const __grid_constant__ HeadParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint4* s_ring = reinterpret_cast<uint4*>(smem);          // [warp][slot][2][32 lanes]
  int8_t* s_codes = reinterpret_cast<int8_t*>(smem + kHeadRingBytes);   // [B][Kpad]
  __shared__ float s_red[kHeadWarps];
  __shared__ float s_sx[B];
  __shared__ hkey s_lead[B][kHeadLists * kCtaLead];
  __shared__ int4 s_sum[2][kHeadWarps / 2][32];

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int nch = p.Kpad / kHeadChunk;
  // this lane's codes: of the one state, or of the MMA column g (any state for
  // the columns past B)
  const int8_t* codes = s_codes + (B == 1 ? 0 : g % B) * (p.Kpad + kCodePad) + 16 * t;
  uint4* ring = s_ring + warp * (kHeadRing * 64) + lane;

  // The weight ring: a pair of warps takes a unit, each warp half of its
  // chunks, so that the units of a call fill about three rounds (rows past V
  // and columns past K are clamped: their logits are not kept, their codes
  // are 0).
  const int half = warp & 1;
  const int c0 = half ? (nch + 1) / 2 : 0;                 // this warp's chunks c0 .. c0 + nc - 1
  const int nc = half ? nch / 2 : (nch + 1) / 2;
  const int nslot = max(nc, kHeadRing);                    // ring slots of a unit: the loader is at most one unit ahead
  const int first = (warp >> 1) * (int)gridDim.x + (int)blockIdx.x;
  const int stride = (int)gridDim.x * (kHeadWarps / 2);
  int lu = first, lc = 0, lslot = 0;                       // the loader's unit, chunk and slot
  const int last16 = (p.K - 1) / 16 * 16;
  const int8_t *lrow0, *lrow1;                             // this lane's rows of the loader's unit
  const auto open_unit = [&]() {
    lrow0 = p.W + (int64_t)min(lu * kHeadRows + g, p.V - 1) * p.ldw;
    lrow1 = p.W + (int64_t)min(lu * kHeadRows + g + 8, p.V - 1) * p.ldw;
  };
  open_unit();
  const auto load = [&]() {
    if (lu < p.units && lc < nc) {
      const int k = min((c0 + lc) * kHeadChunk + 16 * t, last16);
      uint4* dst = ring + lslot * 64;
      cp_async16(dst, lrow0 + k);
      cp_async16(dst + 32, lrow1 + k);
    }
    cp_async_commit();
    if (++lslot == kHeadRing) lslot = 0;
    if (++lc == nslot) {                                   // on to the next unit
      lc = 0;
      lu += stride;
      open_unit();
    }
  };
  // Nothing is read before the wait: the weights are the caller's, and an
  // earlier kernel of the stream may have written them.
  pdl_wait();

  // 1. activation scale and INT8 codes of each hidden state
  head_codes<B, kHeadThreads>(p, s_codes, s_red, s_sx, [&]() {
#pragma unroll 1
    for (int s = 0; s < kHeadRing; ++s) load();
  });

  // 2. approximate logits; the even warp of each pair keeps the pair's best 64
  // keys per hidden state
  hkey la[B], lb[B], pend[B];
#pragma unroll
  for (int b = 0; b < B; ++b) la[b] = lb[b] = pend[b] = 0ull;
  int nu = 0;                                    // units since the last insert
  int held = 0;                                  // inserts
  int cslot = 0, buf = 0;
  for (int u = first; u < p.units; u += stride) {
    const int row0 = u * kHeadRows + g, row1 = row0 + 8;
    const float sc0 = __ldg(p.scale + min(row0, p.V - 1)), sc1 = __ldg(p.scale + min(row1, p.V - 1));
    // one state: each lane's share of rows g, g + 8; several: the MMA's
    // accumulators (state 2 t + e of row g + 8 h in acc[2 h + e])
    int acc[4] = {0, 0, 0, 0};
#pragma unroll 1
    for (int c = 0; c < nslot; ++c) {
      cp_async_wait<kHeadRing - 1>();            // this lane's copies of the chunk have landed
      if (c < nc) {
        const uint4 w0 = ring[cslot * 64], w1 = ring[cslot * 64 + 32];
        const uint4 q = *reinterpret_cast<const uint4*>(codes + (c0 + c) * kHeadChunk);
        if constexpr (B == 1) {
          acc[0] = __dp4a((int)w0.x, (int)q.x, acc[0]);
          acc[1] = __dp4a((int)w1.x, (int)q.x, acc[1]);
          acc[0] = __dp4a((int)w0.y, (int)q.y, acc[0]);
          acc[1] = __dp4a((int)w1.y, (int)q.y, acc[1]);
          acc[0] = __dp4a((int)w0.z, (int)q.z, acc[0]);
          acc[1] = __dp4a((int)w1.z, (int)q.z, acc[1]);
          acc[0] = __dp4a((int)w0.w, (int)q.w, acc[0]);
          acc[1] = __dp4a((int)w1.w, (int)q.w, acc[1]);
        } else {
          mma_s8(acc, w0.x, w1.x, w0.y, w1.y, q.x, q.y);
          mma_s8(acc, w0.z, w1.z, w0.w, w1.w, q.z, q.w);
        }
      }
      if (++cslot == kHeadRing) cslot = 0;
      load();
    }
    // the halves meet: the odd warp hands its sums to the even one (two
    // buffers: a buffer is written again only after the even warp has reached
    // the next unit's barrier)
    int4* sum = &s_sum[buf][warp >> 1][lane];
    buf ^= 1;
    if (half) *sum = make_int4(acc[0], acc[1], acc[2], acc[3]);
    asm volatile("bar.sync %0, 64;" ::"r"(1 + (warp >> 1)) : "memory");
    if (half) continue;
    {
      const int4 o = *sum;
      acc[0] += o.x;
      acc[1] += o.y;
      acc[2] += o.z;
      acc[3] += o.w;
    }
    if constexpr (B == 1) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        acc[h] += __shfl_xor_sync(0xffffffffu, acc[h], 1);
        acc[h] += __shfl_xor_sync(0xffffffffu, acc[h], 2);
      }
    }
#pragma unroll
    for (int b = 0; b < B; ++b) {
      int a0 = acc[0], a1 = acc[1];
      if constexpr (B > 1) {
        const int src = (lane & ~3) | (b >> 1);
        a0 = __shfl_sync(0xffffffffu, acc[b & 1], src);
        a1 = __shfl_sync(0xffffffffu, acc[2 + (b & 1)], src);
      }
      const float z0 = __fmul_rn(sc0, __fmul_rn(s_sx[b], __int2float_rn(a0)));
      const float z1 = __fmul_rn(sc1, __fmul_rn(s_sx[b], __int2float_rn(a1)));
      if (p.z && t == b) {
        float* zb = p.z + (int64_t)b * p.ld_z;
        if (row0 < p.V) zb[row0] = z0;
        if (row1 < p.V) zb[row1] = z1;
      }
      // lanes t = 0, 1 keep the rows g, g + 8 of the first of two units, lanes
      // t = 2, 3 those of the second
      const int row = t & 1 ? row1 : row0;
      if ((t >> 1) == nu && row < p.V) pend[b] = make_key(t & 1 ? z1 : z0, row);
    }
    if (++nu == 2) {                             // 32 pending keys
#pragma unroll
      for (int b = 0; b < B; ++b) {
        list_add32(la[b], lb[b], pend[b], held, lane);
        pend[b] = 0ull;
      }
      ++held;
      nu = 0;
    }
  }
  if (nu) {
#pragma unroll
    for (int b = 0; b < B; ++b) list_add32(la[b], lb[b], pend[b], held, lane);
  }
  // 3. every pair's list into the workspace; the CTA's best keys (of the
  // pairs' best) into its leading keys.  With several states all the warps
  // share the pairs' lists, through shared memory (the ring is idle).
  pdl_launch_dependents();
  if constexpr (B > 1) {
    cp_async_wait<0>();
    __syncthreads();
  }
  if (!half) {
    const int pair = warp >> 1;
#pragma unroll
    for (int b = 0; b < B; ++b) {
      hkey* list = p.lists + (((int64_t)b * p.nctas + blockIdx.x) * kHeadLists + pair) * kHeadList;
      __stcg(list + lane, la[b]);
      __stcg(list + 32 + lane, lb[b]);
      if constexpr (B == 1) {
        const hkey k = best_of64(la[b], lb[b], lane);
        if (lane < kCtaLead) s_lead[b][pair * kCtaLead + lane] = k;
      } else {
        hkey* mine = reinterpret_cast<hkey*>(smem) + (b * kHeadLists + pair) * kHeadList;
        mine[lane] = la[b];
        mine[32 + lane] = lb[b];
      }
    }
  }
  __syncthreads();
  if constexpr (B > 1) {
    for (int i = warp; i < B * kHeadLists; i += kHeadWarps) {
      const hkey* list = reinterpret_cast<const hkey*>(smem) + i * kHeadList;
      const hkey k = best_of64(list[lane], list[32 + lane], lane);
      if (lane < kCtaLead) s_lead[i / kHeadLists][i % kHeadLists * kCtaLead + lane] = k;
    }
    __syncthreads();
  }
  if (warp < B) {
    const hkey k = best_of64(s_lead[warp][lane], s_lead[warp][32 + lane], lane);
    if (lane < kCtaLead) __stcg(p.lead + ((int64_t)warp * p.nctas + blockIdx.x) * kCtaLead + lane, k);
  }
}

// Steps 1-2 and the CTA's lists for one hidden state whose weights exceed what L2
// keeps (kWideBytes): a warp owns units of 4 consecutive rows, lane l reads the
// 16-byte chunks l, l + 32, ... of each row into registers (512 contiguous bytes
// per instruction, 64 KB in flight per SM) and accumulates __dp4a products; every
// warp has a list of its own.
__global__ void __launch_bounds__(kWideThreads, 1)
head_wide_kernel(const __grid_constant__ HeadParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  int8_t* s_codes = reinterpret_cast<int8_t*>(smem);       // [Kpad]
  __shared__ float s_red[kWideWarps];
  __shared__ float s_sx[1];
  __shared__ hkey s_lead[kWideWarps * kCtaLead], s_lead2[kWideWarps];
  static_assert(kWideWarps * kCtaLead == 256 && kWideWarps == 32, "leading keys in two steps of one warp each");

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wg = (int)blockIdx.x * kWideWarps + warp, nwarps = (int)gridDim.x * kWideWarps;
  // the rows of the warp's first unit into L2 while the previous kernel ends
  // (a prefetch hands no data to this kernel)
  for (int r = wg * kWideRows; r < min((wg + 1) * kWideRows, p.V); ++r)
    for (int off = lane * 128; off < p.K; off += 32 * 128)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(p.W + (int64_t)r * p.ldw + off));
  pdl_wait();
  head_codes<1, kWideThreads>(p, s_codes, s_red, s_sx, []() {});

  hkey la = 0ull, lb = 0ull, pend = 0ull;
  int slot = 0, held = 0;                        // units since the last insert; inserts
  const int nch = (p.K + 511) / 512;
  for (int row0 = wg * kWideRows; row0 < p.V; row0 += nwarps * kWideRows) {
    const int nrows = min(kWideRows, p.V - row0);
    int acc[kWideRows] = {};
    for (int c = 0; c < nch; ++c) {
      const int k = 16 * (lane + 32 * c);
      if (k >= p.K) continue;
      // the row is ldw >= K bytes with ldw % 16 == 0: the 16 bytes at k lie
      // inside it; bytes at or past K meet zero codes
      uint4 w[kWideRows];
#pragma unroll
      for (int r = 0; r < kWideRows; ++r)
        w[r] = r < nrows ? ld_weights16(p.W + (int64_t)(row0 + r) * p.ldw + k) : make_uint4(0u, 0u, 0u, 0u);
      const uint4 q = *reinterpret_cast<const uint4*>(s_codes + k);
#pragma unroll
      for (int r = 0; r < kWideRows; ++r) {
        acc[r] = __dp4a((int)w[r].x, (int)q.x, acc[r]);
        acc[r] = __dp4a((int)w[r].y, (int)q.y, acc[r]);
        acc[r] = __dp4a((int)w[r].z, (int)q.z, acc[r]);
        acc[r] = __dp4a((int)w[r].w, (int)q.w, acc[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < kWideRows; ++r) {
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], d);
      if (r < nrows) {
        const float z = __fmul_rn(__ldg(p.scale + row0 + r), __fmul_rn(s_sx[0], __int2float_rn(acc[r])));
        if (p.z && lane == r) p.z[row0 + r] = z;
        if (lane == slot * kWideRows + r) pend = make_key(z, row0 + r);
      }
    }
    if (++slot == 32 / kWideRows) {              // 32 pending keys
      list_add32(la, lb, pend, held, lane);
      pend = 0ull;
      ++held;
      slot = 0;
    }
  }
  if (slot) list_add32(la, lb, pend, held, lane);
  pdl_launch_dependents();
  hkey* list = p.lists + ((int64_t)blockIdx.x * kWideWarps + warp) * kHeadList;
  __stcg(list + lane, la);
  __stcg(list + 32 + lane, lb);
  const hkey k1 = best_of64(la, lb, lane);
  if (lane < kCtaLead) s_lead[warp * kCtaLead + lane] = k1;
  __syncthreads();
  if (warp < kWideWarps * kCtaLead / 64) {
    const hkey k2 = best_of64(s_lead[64 * warp + lane], s_lead[64 * warp + 32 + lane], lane);
    if (lane < kCtaLead) s_lead2[warp * kCtaLead + lane] = k2;
  }
  __syncthreads();
  if (warp == 0) {
    const hkey k3 = best_of64(s_lead2[lane], 0ull, lane);
    if (lane < kCtaLead) __stcg(p.lead + (int64_t)blockIdx.x * kCtaLead + lane, k3);
  }
}

// s_best <- the best 64 keys, descending, of s_cand[0 .. nshort) and of the lists
// of n projection CTAs (those in s_long, or CTAs 0 .. n - 1); by a whole
// selection CTA, with s_merge as scratch.  (A rare path: out of the way of the
// code that every call runs through once.)
__device__ __noinline__ void merge_lists(const hkey* lists, int nlists, const int* s_long, int n, const hkey* s_cand,
                                         int nshort, hkey (*s_merge)[kHeadList], hkey* s_best) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  hkey a = 0ull, c = 0ull;
  for (int i = 64 * warp; i < nshort; i += 64 * kSelWarps) {
    hkey la = i + lane < nshort ? s_cand[i + lane] : 0ull;
    hkey lb = i + 32 + lane < nshort ? s_cand[i + 32 + lane] : 0ull;
    sort64(la, lb, lane);
    list_merge(a, c, la, lb, lane);
  }
  for (int l = warp; l < n * nlists; l += kSelWarps) {
    const hkey* L = lists + (int64_t)(s_long ? s_long[l / nlists] * nlists + l % nlists : l) * kHeadList;
    hkey la = __ldcg(L + lane), lb = __ldcg(L + 32 + lane);
    sort64(la, lb, lane);                        // (lists of up to 64 keys are as they came)
    list_merge(a, c, la, lb, lane);
  }
  s_merge[warp][lane] = a;
  s_merge[warp][32 + lane] = c;
  __syncthreads();
  if (warp == 0) {
    for (int w = 1; w < kSelWarps; ++w) list_merge(a, c, s_merge[w][lane], s_merge[w][32 + lane], lane);
    s_best[lane] = a;
    s_best[32 + lane] = c;
  }
  __syncthreads();
}

// A sharper bound for the selection: *s_bound <- the 64th largest of the m keys
// s_cand[0 .. m) (also a rare path).
__device__ __noinline__ void sharper_bound(const hkey* s_cand, int m, hkey* s_bound) {
  for (int i = threadIdx.x; i < m; i += kSelThreads)
    if (s_cand[i] != 0ull && count_larger(s_cand, m, s_cand[i]) == kHeadList - 1) *s_bound = s_cand[i];
  __syncthreads();
}

// Steps 3-6, a cluster of kSelCluster CTAs per hidden state.  Every CTA of
// the cluster makes the same selection: the bound T (the 64th largest of the
// projection CTAs' best keys, so at least 64 keys reach it), the keys >= T,
// the best 64 of them by counting, the gate.  A projection CTA whose kCtaLead
// leading keys all pass may have others in its lists, which are then read in
// full.  The candidates are shared out (warp w of rank r recomputes 8 r + w
// and 32 + 8 r + w), their logits meet in rank 0's shared memory, and rank 0
// picks the token.  Where more than kSelLong CTAs would be read in full a sharper
// bound is taken; where more than kSelCand keys reach the bound the warps merge
// the lists that hold them (or every list, when there is no bound): slower, and
// exact either way.
__global__ void __launch_bounds__(kSelThreads)
head_select_kernel(const __grid_constant__ HeadParams p) {
  __shared__ hkey s_cand[kSelCand];
  __shared__ hkey s_best[kHeadList];
  __shared__ hkey s_merge[kSelWarps][kHeadList];
  __shared__ float s_r[kHeadList];
  __shared__ int s_long[kSelLong];
  __shared__ hkey s_bound;
  __shared__ int s_nc, s_nlong;

  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int b = (int)blockIdx.x / kSelCluster;
  const int rank = (int)blockIdx.x - b * kSelCluster;
  const int ks = p.k_sel, nc = p.nctas;
  asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");   // waited for before the first remote store
  pdl_wait();                                    // every list and count is written
  hkey lead[kCtaLead];                           // of projection CTA t
  if (t < nc) {
    const ulonglong2* src =
        reinterpret_cast<const ulonglong2*>(p.lead + ((int64_t)b * nc + t) * kCtaLead);
#pragma unroll
    for (int q = 0; q < kCtaLead / 2; ++q) {
      const ulonglong2 k = __ldcg(src + q);
      lead[2 * q] = k.x;
      lead[2 * q + 1] = k.y;
    }
  }
  if (t == 0) {
    s_nc = 0;
    s_nlong = 0;
    s_bound = 1ull;                              // no bound: every key passes
  }
  // the bound: the 64th largest of the CTAs' best keys (of all their leading
  // keys where there are fewer than 64 CTAs), found by counting the larger ones
  const int per = nc >= kHeadList ? 1 : kCtaLead;
  if (t < nc) {
#pragma unroll
    for (int e = 0; e < kCtaLead; ++e)
      if (e < per) s_cand[t * per + e] = lead[e];
  }
  __syncthreads();
  for (int i = t; i < nc * per; i += kSelThreads)
    if (count_larger(s_cand, nc * per, s_cand[i]) == kHeadList - 1 && s_cand[i] != 0ull) s_bound = s_cand[i];
  __syncthreads();
  // The next call's projection waits for this kernel in any case; started at
  // this kernel's start its idle CTAs slowed the call (57,344 rows, one state,
  // tau 0.5: 24.6 against 24.0 us; four states 31.7 against 31.3).
  pdl_launch_dependents();
  hkey T = s_bound;
  // the leading keys >= T into s_cand; the CTAs whose lists may hold more
  const auto gather_leads = [&]() {
    if (t < nc) {
      int n = 0;
#pragma unroll
      for (int e = 0; e < kCtaLead; ++e) n += lead[e] >= T;
      if (n == kCtaLead) {
        const int j = atomicAdd(&s_nlong, 1);
        if (j < kSelLong) s_long[j] = t;
      } else if (n > 0) {
        const int i = atomicAdd(&s_nc, n);
#pragma unroll
        for (int e = 0; e < kCtaLead - 1; ++e)
          if (e < n && i + e < kSelCand) s_cand[i + e] = lead[e];
      }
    }
    __syncthreads();
  };
  gather_leads();
  if (s_nlong > kSelLong) {
    // Best rows that are spread evenly, eight and more to a CTA, as equal logits
    // are (3000 of them: 191 us a call by merging every list, 20 so): the bound is
    // the 64th largest of all leading keys instead.  Those of 64 CTAs at most
    // reach the first one, and at most eight CTAs reach this one in full.
    __syncthreads();                             // every thread has read s_nlong
    if (t == 0) s_nc = s_nlong = 0;
    __syncthreads();
    if (t < nc && lead[0] >= T) {
      const int i = atomicAdd(&s_nc, kCtaLead);
#pragma unroll
      for (int e = 0; e < kCtaLead; ++e)
        if (i + e < kSelCand) s_cand[i + e] = lead[e];
    }
    __syncthreads();
    sharper_bound(s_cand, min(s_nc, kSelCand), &s_bound);   // (a barrier: s_nc and s_cand are read)
    T = s_bound;
    if (t == 0) s_nc = 0;
    __syncthreads();
    gather_leads();
  }
  const hkey* lists = p.lists + (int64_t)b * nc * p.nlists * kHeadList;
  const int nlong = s_nlong, nshort = s_nc;      // (s_cand[0 .. nshort) are leading keys)
  if (nlong > 0 && nlong <= kSelLong) {
    __syncthreads();                             // every thread has read s_nc
    for (int j = 0; j < nlong; ++j) {
      const hkey* L = lists + (int64_t)s_long[j] * p.nlists * kHeadList;
#pragma unroll 2
      for (int e = t; e < p.nlists * kHeadList; e += kSelThreads) {
        const hkey k = __ldcg(L + e);
        if (k >= T) {
          const int i = atomicAdd(&s_nc, 1);
          if (i < kSelCand) s_cand[i] = k;
        }
      }
    }
    __syncthreads();
  }
  const int C = s_nc;
  if (C <= kSelCand && nlong <= kSelLong && C >= min(p.V, kHeadList)) {
    rank_place(s_cand, C, s_best);
  } else {
    // the lists of the CTAs that pass in full and the leading keys of the others,
    // or every list
    if (nlong <= kSelLong && C > kSelCand)
      merge_lists(lists, p.nlists, s_long, nlong, s_cand, nshort, s_merge, s_best);
    else
      merge_lists(lists, p.nlists, nullptr, nc, s_cand, 0, s_merge, s_best);
  }
  const float g = __fsub_rn(key_z(s_best[0]), key_z(s_best[1]));
  const bool open = g < p.tau;
  asm volatile("barrier.cluster.wait;" ::: "memory");   // rank 0 is running
  if (open) {
    const float* hb = p.h + (int64_t)b * p.ldh;
    const int i0 = rank * kSelWarps + warp, i1 = i0 + kHeadList / 2;
    const int n = i1 < ks ? 2 : i0 < ks ? 1 : 0;
    if (n > 0) {
      const int rows[2] = {key_row(s_best[i0]), n > 1 ? key_row(s_best[i1]) : 0};
      float rv[2];
      verify_rows2(p, hb, rows, n, lane, rv);
      if (lane < n)
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr(&s_r[lane ? i1 : i0], 0)),
                     "f"(lane ? rv[1] : rv[0])
                     : "memory");
    }
  }
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  if (rank != 0) return;
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // every logit is in
  if (warp == 0) {
    int token = key_row(s_best[0]);
    if (open) {
      // largest r, equal r: lower row (starting from candidate 0, so the
      // token is always a candidate)
      float br = s_r[0];
      int bm = token;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i = lane + 32 * q;
        if (i < ks) {
          const float rv = s_r[i];
          const int m = key_row(s_best[i]);
          if (rv > br || (rv == br && m < bm)) {
            br = rv;
            bm = m;
          }
          if (p.r) p.r[(int64_t)b * ks + i] = rv;
        }
      }
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) {
        const float orv = __shfl_xor_sync(0xffffffffu, br, d);
        const int om = __shfl_xor_sync(0xffffffffu, bm, d);
        if (orv > br || (orv == br && om < bm)) {
          br = orv;
          bm = om;
        }
      }
      token = bm;
    }
    if (lane == 0) {
      p.token[b] = token;
      if (p.verified) p.verified[b] = open ? 1 : 0;
      if (p.gap) p.gap[b] = g;
    }
  }
  if (p.cand && t < ks) p.cand[(int64_t)b * ks + t] = key_row(s_best[t]);
}

template <int B>
cudaError_t launch_head_t(HeadParams p, int dev, int sms, cudaStream_t s) {
  // The largest shared-memory carve-out for the selection too: with a smaller
  // one its SM could not take a projection CTA beside it (the next call's,
  // which starts while the selection runs), and the late CTA held up the call.
  static PerDevice carve, ring;  // per instance: head_kernel<B> is a kernel of its own
  cudaError_t e = carve.once(dev, []() {
    return cudaFuncSetAttribute(head_select_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                (int)cudaSharedmemCarveoutMaxShared);
  });
  if (e != cudaSuccess) return e;
  e = ring.once(dev, []() {
    return cudaFuncSetAttribute(head_kernel<B>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(kHeadRingBytes + (size_t)B * (SPIKE_PROJ_HEAD_MAX_K + kCodePad)));
  });
  if (e != cudaSuccess) return e;
  const size_t smem = kHeadRingBytes + (size_t)B * (p.Kpad + kCodePad);
  // one wave, one CTA per SM
  int grid = sms;
  if (grid > p.units) grid = p.units;
  if (grid > kHeadMaxGrid) grid = kHeadMaxGrid;
  p.nctas = grid;
  p.nlists = kHeadLists;
  // One state whose weights exceed what L2 keeps streams faster into registers,
  // given two rounds of units for every warp.  us a call, ring / registers, gate
  // closed: 57,344 x 2048 28.0 / 24.5, 57,344 x 4096 50.9 / 41.0, 150,000 x 1536
  // 48.8 / 46.0, 128,256 x 2048 55.8 / 49.3 to 52.4, 151,936 x 1024 36.3 / 33.3;
  // below, in L2, the ring: 70,000 x 1536 22.9 / 24.1; with few rows too: 13,000 x
  // 8192 from HBM 31.2 / 36.7.
  if (B == 1 && (int64_t)p.V * p.K >= kWideBytes && p.V >= 2 * kWideRows * kWideWarps * sms) {
    p.nlists = kWideWarps;
    e = launch_pdl(head_wide_kernel, dim3((unsigned)grid), dim3(kWideThreads), (size_t)p.Kpad + kCodePad, s, p);
  } else {
    e = launch_pdl(head_kernel<B>, dim3((unsigned)grid), dim3(kHeadThreads), smem, s, p);
  }
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(B * kSelCluster, 1, 1);
  cfg.blockDim = dim3(kSelThreads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kSelCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, head_select_kernel, p);
}

}  // namespace

size_t head_workspace_bytes() { return kListBytes + kLeadBytes; }

cudaError_t launch_head(const HeadArgs& a, cudaStream_t s) {
  int dev = 0, sms = 0;
  const cudaError_t e = current_device(&dev, &sms);
  if (e != cudaSuccess) return e;
  HeadParams p;
  p.W = a.W;
  p.ldw = a.ldw;
  p.scale = a.scale;
  p.V = a.V;
  p.K = a.K;
  p.Kpad = (a.K + kHeadChunk - 1) / kHeadChunk * kHeadChunk;
  p.units = (a.V + kHeadRows - 1) / kHeadRows;
  p.h = a.h;
  p.ldh = a.ldh;
  p.tau = a.tau;
  p.k_sel = a.k_sel;
  p.token = a.token;
  p.verified = a.verified;
  p.gap = a.gap;
  p.cand = a.cand;
  p.r = a.r;
  p.z = a.z;
  p.ld_z = a.ld_z;
  p.B = a.B;
  p.lists = static_cast<hkey*>(a.ws);
  p.lead = reinterpret_cast<hkey*>(static_cast<unsigned char*>(a.ws) + kListBytes);
  p.nctas = p.nlists = 0;
  switch (a.B) {
    case 1: return launch_head_t<1>(p, dev, sms, s);
    case 2: return launch_head_t<2>(p, dev, sms, s);
    case 3: return launch_head_t<3>(p, dev, sms, s);
    default: return launch_head_t<4>(p, dev, sms, s);
  }
}

}  // namespace sp
