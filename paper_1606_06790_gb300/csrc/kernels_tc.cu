// Mixed-precision H_eff psi on the 5th-generation tensor cores (Step 3).
//
// Every FP64 operand x is split into two TF32 numbers, hi = x rounded to TF32
// and lo = x - hi (also used at TF32 precision), and a product is formed from
// three tcgen05.mma of kind::tf32 (hi.hi + hi.lo + lo.hi) accumulated in FP32
// in tensor memory: about 21 significant bits per product.  The BF16 variant
// splits into two BF16 numbers the same way and issues kind::f16 MMAs: about
// 16 significant bits per product at twice the K per instruction.  Both use
// the same byte layout (a K block is 128 bytes of every row: 32 TF32 or 64
// BF16 elements), so the GEMM kernel differs only in the MMA it issues.
//
//  pack      : splits FP64 or FP32 source blocks into packed hi/lo tiles in the
//              tensor-core operand layout (K-major, no swizzle, core matrices
//              of 8 rows x 16 bytes), so that a K block of a tile is one
//              contiguous range that a single bulk (TMA) copy moves.
//  wstage_tc : T3[c] = sum W12 T1[a] from the FP32 stage-1 output, written
//              straight into the packed A operand of stage 3.
//  tc_gemm   : persistent grouped GEMM over a list of 128 x TN output tiles
//              (TN = 64, 128 or 256, picked per list by the context's tuner),
//              one CTA per SM: a producer warp streams the hi/lo tiles
//              of A and B through a ring of shared-memory stages with
//              cp.async.bulk, an MMA warp issues the tcgen05.mma chain into one
//              of two tensor-memory accumulators, four epilogue warps read the
//              other out (tcgen05.ld) and store it as FP32 (stage 1) or,
//              through a row map, as FP64 into the output wavefunction
//              (stage 3).  Every mbarrier wait is bounded; a timeout sets the
//              context's error word and ends every role's loop, the copies in
//              flight are waited for (bounded), and tensor memory is released
//              unless the wait for the MMAs themselves ran out (they may still
//              write it).
#include <cuda_bf16.h>
#include <stdint.h>

#include "common.h"
#include "tc_ptx.h"

namespace idmrg {

namespace {

// streaming multiprocessors of the current device (0: query failed)
int sm_count() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return 0;
    sms = n;
  }
  return sms;
}

__device__ __forceinline__ float tf32_round(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}

__device__ __forceinline__ int64_t packed_off(int row, int k, int KB, int G) {
  const int rows_per_tile = 8 * G;
  const int rt = row / rows_per_tile, rr = row - rt * rows_per_tile;
  const int kb = k >> 5, kc = (k & 31) >> 2;
  const int64_t tile_floats = (int64_t)rows_per_tile * 32;
  return ((int64_t)rt * KB + kb) * 2 * tile_floats + (((int64_t)kc * G + (rr >> 3)) * 8 + (rr & 7)) * 4 + (k & 3);
}

// The same position for 16-bit elements (in units of 16 bits): 64 per K
// block, core matrices 8 rows x 8 elements.
__device__ __forceinline__ int64_t packed_off_h(int row, int k, int KB, int G) {
  const int rows_per_tile = 8 * G;
  const int rt = row / rows_per_tile, rr = row - rt * rows_per_tile;
  const int kb = k >> 6, kc = (k & 63) >> 3;
  const int64_t tile_h = (int64_t)rows_per_tile * 64;
  return ((int64_t)rt * KB + kb) * 2 * tile_h + (((int64_t)kc * G + (rr >> 3)) * 8 + (rr & 7)) * 8 + (k & 7);
}

// hi/lo split of an FP32 value: hi its BF16 (bf16 = 1) or TF32 rounding, lo the
// rest, which is exact
__device__ __forceinline__ void split(float x, int bf16, float &hi, float &lo) {
  hi = bf16 ? __bfloat162float(__float2bfloat16_rn(x)) : tf32_round(x);
  lo = x - hi;
}

// The same of an FP64 value: hi from x rounded to FP32, lo = x - hi rounded to
// FP32.  The FP64 pipe takes 4 operations per element for it (two narrowings, a
// widening and the difference) at 2 lanes per clock and SM, which is more time
// than the memory traffic; so integers round x to f, and x - hi = (f - hi) + r,
// r = +-E 2^(e-52) with |E| <= 2^28, is formed in FP32 with one rounding: f - hi
// and the part of E above its low 21 bits make 24 significant bits at most (hi
// leaves 2^44 + 2^28 units at most), so the first fma is exact.  Values whose
// rest could leave the normal FP32 range take the FP64 operations.
__device__ __forceinline__ void split(double x, int bf16, float &hi, float &lo) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int e = (int)((h >> 20) & 2047u) - 1023;
  if (((h << 1) | l) == 0) {
    hi = __uint_as_float(h);
    lo = 0.0f;
    return;
  }
  if (e < -74 || e > 100) {
    hi = bf16 ? __bfloat162float(__float2bfloat16_rn((float)x)) : tf32_round((float)x);
    lo = (float)(x - (double)hi);
    return;
  }
  const uint32_t trunc = ((uint32_t)(e + 127) << 23) | ((h & 0xFFFFFu) << 3) | (l >> 29);
  const uint32_t rest = l & 0x1FFFFFFFu;
  const bool up = rest > 0x10000000u || (rest == 0x10000000u && (trunc & 1u));
  const float f = __uint_as_float((h & 0x80000000u) | (trunc + (up ? 1u : 0u)));
  const int E = (int)rest - (up ? 0x20000000 : 0);
  hi = bf16 ? __bfloat162float(__float2bfloat16_rn(f)) : tf32_round(f);
  // integers below 2^23 to FP32 through the mantissa of 1.5 * 2^23
  const float Eh = __int_as_float(0x4B400000 + (E >> 21)) - 12582912.0f;
  const float El = __int_as_float(0x4B400000 + (E & 0x1FFFFF)) - 12582912.0f;
  const float u = __uint_as_float((h & 0x80000000u) | ((uint32_t)(e - 52 + 127) << 23));
  lo = fmaf(El, u, fmaf(Eh, u * 2097152.0f, f - hi));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);  // (exact for hi parts)
  return (uint32_t)__bfloat16_as_ushort(v.x) | ((uint32_t)__bfloat16_as_ushort(v.y) << 16);
}

// one 16-byte group (8 BF16 or 4 TF32 elements from packed K kg on) of packed
// row `row`
template <class T>
__device__ __forceinline__ void put_group(float *dst, int row, int kg, int KB, int G, int bf16, const T *v) {
  float hi[8], lo[8];
  if (bf16) {
#pragma unroll
    for (int j = 0; j < 8; ++j) split(v[j], 1, hi[j], lo[j]);
    __nv_bfloat16 *h = reinterpret_cast<__nv_bfloat16 *>(dst) + packed_off_h(row, kg, KB, G);
    *reinterpret_cast<uint4 *>(h) = make_uint4(pack_bf16x2(hi[0], hi[1]), pack_bf16x2(hi[2], hi[3]),
                                               pack_bf16x2(hi[4], hi[5]), pack_bf16x2(hi[6], hi[7]));
    *reinterpret_cast<uint4 *>(h + (int64_t)8 * G * 64) =
        make_uint4(pack_bf16x2(lo[0], lo[1]), pack_bf16x2(lo[2], lo[3]), pack_bf16x2(lo[4], lo[5]),
                   pack_bf16x2(lo[6], lo[7]));
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) split(v[j], 0, hi[j], lo[j]);
    float *f = dst + packed_off(row, kg, KB, G);
    *reinterpret_cast<float4 *>(f) = make_float4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<float4 *>(f + (int64_t)8 * G * 32) = make_float4(lo[0], lo[1], lo[2], lo[3]);
  }
}

// the elements of a group that fall into packed K [ka, kb), one by one: a group
// that a neighbouring segment shares
__device__ __forceinline__ void put_part(float *dst, int row, int kg, int ka, int kb, int KB, int G, int bf16,
                                         const double *v) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int k = kg + j;
    if (k < ka || k >= kb || (!bf16 && j >= 4)) continue;
    float hi, lo;
    split(v[j], bf16, hi, lo);
    if (bf16) {
      __nv_bfloat16 *h = reinterpret_cast<__nv_bfloat16 *>(dst) + packed_off_h(row, k, KB, G);
      h[0] = __float2bfloat16_rn(hi);
      h[(int64_t)8 * G * 64] = __float2bfloat16_rn(lo);
    } else {
      float *f = dst + packed_off(row, k, KB, G);
      f[0] = hi;
      f[(int64_t)8 * G * 32] = lo;
    }
  }
}

// Packing runs through windows of 32 rows and 64 packed K columns (aligned to
// 64) held in shared memory: read with the lanes along whatever is contiguous
// in the source, written a 16-byte group of a row per thread with the lanes
// along the rows, so that a warp fills 512 contiguous bytes.
constexpr int OP_ROWS = PACK_ROWS, OP_K = PACK_K, OP_LD = OP_K + 2;

// SCALED: alpha is not 1 (a multiplication is as long on the FP64 pipe as the
// element's memory traffic)
template <bool SCALED>
__device__ __forceinline__ double pack_src(const PackSeg &s, const double *src, int r, int k) {
  const double x = src[s.trans ? (int64_t)k * s.src_ld + r : (int64_t)r * s.src_ld + k];
  return SCALED ? s.alpha * x : x;
}

// rows r0 .. r0 + nr - 1 of a segment, packed K columns kw .. kw + 63, zeros
// where the segment has none (256 threads)
template <bool SCALED>
__device__ __forceinline__ void pack_load_window(const PackSeg &s, const double *src, int r0, int nr, int kw,
                                                 double *tile) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k1 = s.k0 + s.ks;
  if (s.trans) {
#pragma unroll
    for (int i = 0; i < OP_K / 8; ++i) {
      const int kk = warp + 8 * i, k = kw + kk;
      if (lane < nr)
        tile[lane * OP_LD + kk] = k >= s.k0 && k < k1 ? pack_src<SCALED>(s, src, r0 + lane, k - s.k0) : 0.0;
    }
  } else {
#pragma unroll
    for (int i = 0; i < OP_ROWS / 8; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = warp + 8 * i, kk = lane + 32 * h, k = kw + kk;
        if (r < nr)
          tile[r * OP_LD + kk] = k >= s.k0 && k < k1 ? pack_src<SCALED>(s, src, r0 + r, k - s.k0) : 0.0;
      }
  }
}

// Split operands, one window per block: memory bound, 8 bytes in and 4 (BF16) or
// 8 (TF32) out per element.  Measured (GB300, kagome cylinder at m = 1000, BF16,
// under a profiler): R of all superblocks, 13 300 windows, 178 us by a thread per
// element, its 16-bit stores and FP64 operations; 123 us through windows with the
// split in integers; 99 us without the multiplication by alpha = 1.  What is left
// are the rectangles' partly filled windows and the chain of loads in front of
// each (unit, segment, data).
__global__ void __launch_bounds__(256) pack_kernel(const int4 *__restrict__ units, const PackSeg *__restrict__ segs,
                                                   double *const *__restrict__ bufs, const int *__restrict__ active,
                                                   int bf16) {
  __shared__ __align__(16) double tile[OP_ROWS * OP_LD];
  const int4 u = units[blockIdx.x];  // segment, first row, first packed K column
  const PackSeg s = segs[u.x];
  if (active && !active[s.sb]) return;
  const int nr = min(OP_ROWS, s.rows - u.y), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pack_load_window<false>(s, bufs[s.sb * NBUF + s.src_buf] + s.src_off, u.y, nr, u.z, tile);
  __syncthreads();
  if (lane >= nr) return;
  float *dst = (float *)bufs[s.sb * NBUF + s.dst_buf] + s.dst_off;
  const int gw = bf16 ? 8 : 4, ka = s.k0, kb = s.k0 + s.ks + s.kpad, row = s.row0 + u.y + lane;
  for (int k = gw * warp; k < OP_K; k += 8 * gw) {
    const int kg = u.z + k;
    if (kg + gw <= ka || kg >= kb) continue;
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; j += 2)
      if (j < gw) *reinterpret_cast<double2 *>(v + j) = *reinterpret_cast<const double2 *>(tile + lane * OP_LD + k + j);
    if (kg >= ka && kg + gw <= kb)
      put_group(dst, row, kg, s.KB, s.G, bf16, v);
    else
      put_part(dst, row, kg, ka, kb, s.KB, s.G, bf16, v);
  }
}

// T3 = sum W12 T1 into the packed stage-3 A operand.  The two-site MPO is
// mostly pass-through (T3 copies one T1 rectangle per channel; the completed
// channel sums many), so the stage streams T1 in and T3 out.  A unit is 32 rows
// and 64 packed K columns, across however many channels' rectangles these fall
// into: the many small rectangles of the outer charge sectors share a window,
// and the terms that reach into it are one run of the term list.  Phase 1:
// warps read T1 rows with the lanes along K (coalesced) and accumulate the
// terms.  Phase 2: through a shared-memory tile, each thread takes one row and
// one 16-byte group of the packed layout, the lanes along the rows, so that a
// warp's stores fill 512 contiguous bytes; columns that no rectangle covers,
// and the K padding inside the window, are zeros.
// A window is a microsecond of work behind a chain of dependent loads (unit,
// its terms, T1), which is what bounded one CTA per window; the CTAs are
// persistent instead, and while one window is worked on the next one's terms
// are on their way to shared memory and the one after that's unit to registers.
// Measured (GB300, kagome cylinder at m = 1000, all superblocks, under a
// profiler; before: a CTA per window of a single rectangle): 180 -> 171 us, two
// thirds of the issue slots taken; the FP64 form's two passes 419 + 608 -> 338 +
// 407 us.
constexpr int W_BATCH = 64;  // terms in shared memory at a time

struct __align__(16) WStage {  // the shared-memory part of one unit
  WTaskP task;
  WTerm term[W_BATCH];
};
static_assert(sizeof(WTerm) == 32 && sizeof(WTaskP) == 48, "copied in 16-byte pieces");

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}

// Walks the units of this CTA (blockIdx.x, + gridDim.x, ...): body(u, S) for
// each, S holding its task and first W_BATCH terms; every thread of the block
// takes part, and body is free to use barriers.
template <class Body>
__device__ __forceinline__ void w_walk(const WUnit *__restrict__ units, int nunits, const WTaskP *__restrict__ tasks,
                                       const WTerm *__restrict__ terms, WStage (&S)[2], Body body) {
  auto fetch = [&](const WUnit &u, WStage &to) {
    const int n = 2 * min(u.nterm, W_BATCH);
    const char *t = reinterpret_cast<const char *>(terms + u.term0), *k = reinterpret_cast<const char *>(tasks + u.task);
    if (threadIdx.x < n) cp_async16(reinterpret_cast<char *>(to.term) + 16 * threadIdx.x, t + 16 * threadIdx.x);
    if (threadIdx.x >= 128 && threadIdx.x < 131)
      cp_async16(reinterpret_cast<char *>(&to.task) + 16 * (threadIdx.x - 128), k + 16 * (threadIdx.x - 128));
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  int i = blockIdx.x, buf = 0;
  if (i >= nunits) return;
  WUnit u = units[i], next{};
  if (i + gridDim.x < nunits) next = units[i + gridDim.x];
  fetch(u, S[0]);
  for (; i < nunits; i += gridDim.x, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // this unit's terms are there; the other buffer is free
    WUnit after{};
    if (i + gridDim.x < nunits) fetch(next, S[buf ^ 1]);
    if (i + 2 * gridDim.x < nunits) after = units[i + 2 * gridDim.x];
    body(u, S[buf]);
    u = next;
    next = after;
  }
}

template <class T>
__device__ __forceinline__ T w_coef(const WTerm &w);
template <>
__device__ __forceinline__ float w_coef<float>(const WTerm &w) {
  return w.coef32;
}
template <>
__device__ __forceinline__ double w_coef<double>(const WTerm &w) {
  return w.coef;
}
// comparisons that stay off the FP64 pipe, where one holds its unit for 64 cycles a warp
__device__ __forceinline__ bool is_one(float x) { return x == 1.0f; }
__device__ __forceinline__ bool is_one(double x) { return __double_as_longlong(x) == 0x3FF0000000000000ll; }
__device__ __forceinline__ bool is_zero(double x) { return ((unsigned long long)__double_as_longlong(x) << 1) == 0; }

// The window's sums: warp w holds rows w, w + 8, w + 16, w + 24, lane l the
// columns l and l + 32.  Most elements have one term of coefficient 1, which is
// copied (an FMA in FP64 holds its unit for 64 cycles); halves of the window
// that a narrow rectangle does not reach issue nothing.
template <class T>
__device__ __forceinline__ void w_accumulate(const WUnit &u, const WTerm *__restrict__ terms, const T *in, int nr,
                                             WTerm *st, T (&acc)[4][2]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = T(0);
  const int nrow = (nr - warp + 7) >> 3;  // rows of this warp (may be <= 0)
  int last = -1;  // first column of the last term's rectangle: terms of one rectangle are consecutive
  for (int b = 0; b < u.nterm; b += W_BATCH) {
    const int n = min(W_BATCH, u.nterm - b);
    if (b > 0) {
      __syncthreads();
      const double *from = reinterpret_cast<const double *>(terms + u.term0 + b);
      for (int j = threadIdx.x; j < 4 * n; j += blockDim.x) reinterpret_cast<double *>(st)[j] = from[j];
      __syncthreads();
    }
    for (int q = 0; q < n; ++q) {
      const WTerm w = st[q];
      const int k = u.k0 - w.k0;  // the window's first column in the rectangle
      const T cf = w_coef<T>(w);
      const bool copy = w.k0 != last && is_one(cf);
      last = w.k0;
      const bool on[2] = {(unsigned)(k + lane) < (unsigned)w.cols, (unsigned)(k + lane + 32) < (unsigned)w.cols};
      const bool half[2] = {k + 31 >= 0 && k < w.cols, k + 32 < w.cols};  // (every term reaches the window)
      const T *src = in + (w.in_off + (int64_t)(u.r0 + warp) * w.in_ld + (k + lane));
      const int64_t step = 8 * (int64_t)w.in_ld;
      T x[4][2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (half[h]) {
          const T *row = src + 32 * h;
#pragma unroll
          for (int i = 0; i < 4; ++i, row += step) {
            x[i][h] = T(0);
            if (on[h] && i < nrow) x[i][h] = *row;
          }
        }
      }
      if (copy) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (half[h]) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (on[h]) acc[i][h] = x[i][h];
          }
      } else {
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (half[h]) {
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i][h] = fma(cf, x[i][h], acc[i][h]);
          }
      }
    }
  }
}

constexpr int WT_LD = W_K + 4;  // row stride of the tile (floats)

constexpr int W_TC_CTAS = 6;  // resident per SM
__global__ void __launch_bounds__(256, W_TC_CTAS) wstage_tc_kernel(const WUnit *__restrict__ units, int nunits,
                                                                   const WTaskP *__restrict__ tasks,
                                                                   const WTerm *__restrict__ terms,
                                                                   double *const *__restrict__ bufs,
                                                                   const int *__restrict__ active, int bf16) {
  __shared__ __align__(16) float tile[W_ROWS * WT_LD];
  __shared__ WStage S[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  w_walk(units, nunits, tasks, terms, S, [&](const WUnit &u, WStage &st) {
    const WTaskP &t = st.task;
    if (active && !active[t.sb]) return;
    const int nr = min(W_ROWS, t.rows - u.r0);
    float *dst = (float *)bufs[t.sb * NBUF + t.dst_buf] + t.dst_off;
    float acc[4][2];
    w_accumulate<float>(u, terms, (const float *)bufs[t.sb * NBUF + t.in_buf], nr, st.term, acc);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      tile[(warp + 8 * i) * WT_LD + lane] = acc[i][0];
      tile[(warp + 8 * i) * WT_LD + lane + 32] = acc[i][1];
    }
    __syncthreads();  // (the walk's barrier keeps the next window off the tile)
    if (lane >= nr) return;
    const int gw = bf16 ? 8 : 4, kend = min(W_K, (bf16 ? 64 : 32) * t.KB - u.k0);
    for (int k = gw * warp; k < kend; k += 8 * gw) {
      float v[8];
      *reinterpret_cast<float4 *>(v) = *reinterpret_cast<const float4 *>(tile + lane * WT_LD + k);
      if (bf16) *reinterpret_cast<float4 *>(v + 4) = *reinterpret_cast<const float4 *>(tile + lane * WT_LD + k + 4);
      put_group(dst, t.row0 + u.r0 + lane, u.k0 + k, t.KB, t.G, bf16, v);
    }
  });
}

constexpr int TM = 128;
constexpr int A_TILE = TM * 32;         // floats per A tile (one of hi/lo)
constexpr long long WAIT_BUDGET = 4000000000LL;  // clock cycles (about 2 s)

// Shapes of the persistent GEMM for an N tile of TN columns: a ring stage
// holds one K block of the A tile and of the B tile, hi and lo; as many
// stages as fit in 192 KB of shared memory (4, 3, 2 for TN = 64, 128, 256).
// Behind the ring, each epilogue warp has a 32 x 32 staging block (row
// stride 33 floats) through which its accumulator rows reach global memory
// as whole-row segments.
constexpr int EPI_COLS = 32, EPI_LD = EPI_COLS + 1;
constexpr int EPI_FLOATS = 4 * 32 * EPI_LD;
template <int TN>
struct PsShape {
  static_assert(TN == 64 || TN == 128 || TN == 256, "N tile");
  static constexpr int B_TILE = TN * 32;  // floats per B tile (one of hi/lo)
  static constexpr int STAGE_FLOATS = 2 * A_TILE + 2 * B_TILE;
  static constexpr int STAGES = (192 * 1024) / (STAGE_FLOATS * 4);
  static constexpr int SMEM = STAGES * STAGE_FLOATS * 4 + EPI_FLOATS * 4;
  static_assert(STAGES >= 2, "ring depth");
};

// ---------------------------------------------- persistent grouped GEMM
// Output tiles of 128 rows x TN columns, one CTA per SM looping over the
// tile list (tile t = blockIdx.x + i gridDim.x), with three roles:
// warp 0 streams the K blocks of successive tiles through a PS_STAGES-deep
// ring of shared memory (bulk copies), warp 1 issues the MMA chain of a tile
// into one of two TMEM accumulators, warps 2-5 read the other accumulator out
// (tcgen05.ld) and store it.  Set-up, pipeline fill and epilogue of a tile
// thereby overlap the next tile's copies and MMAs, which matters when K is a
// few blocks (stage 1 of H_eff psi: K = one sector of the left block).
// Ring and accumulator buffers are handed over by mbarriers whose phases
// follow from running counters; every wait is bounded, a timeout sets the
// error word and makes every role leave its loop, and the accumulators are
// released only once every MMA issued has completed.  The N tile (64, 128
// or 256 columns) is chosen per GEMM list by the plan's tuner: a wider tile
// reads each A tile from L2 fewer times, a narrower one wastes less of a
// ragged N.
constexpr int PS_THREADS = 192;

template <bool BF16, int TN>
__global__ void __launch_bounds__(PS_THREADS, 1) tc_gemm_ps_kernel(const TcTile *__restrict__ tiles, int ntiles,
                                                                   const TcTask *__restrict__ tasks,
                                                                   double *const *__restrict__ bufs,
                                                                   const int *__restrict__ active, int *err) {
  using Sh = PsShape<TN>;
  constexpr int PS_STAGES = Sh::STAGES;
  constexpr int B_TILE = Sh::B_TILE;
  constexpr int STAGE_FLOATS = Sh::STAGE_FLOATS;
  extern __shared__ __align__(1024) float sm[];
  float *epi = sm + PS_STAGES * STAGE_FLOATS;  // epilogue staging, EPI_FLOATS
  __shared__ __align__(8) uint64_t full[PS_STAGES], empty[PS_STAGES], accf[2], acce[2], done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) {
    tc::tmem_alloc(&tmem_base, 2 * TN);
    tc::tmem_relinquish();
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < PS_STAGES; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      tc::mbar_init(&accf[a], 1);
      tc::mbar_init(&acce[a], 4);  // one arrival per epilogue warp
    }
    tc::mbar_init(&done, 1);
    abort_flag = 0;
    tc::fence_mbar_init();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_base;
  volatile int *abort_v = &abort_flag;
  constexpr uint32_t stage_bytes = 4u * STAGE_FLOATS;

  if (warp == 0) {
    if (lane == 0) {  // ---- producer
      long long it = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const TcTile tile = tiles[t];
        const TcTask T = tasks[tile.task];
        if (active && !active[T.sb]) continue;
        const float *A = (const float *)bufs[T.sb * NBUF + T.a_buf] + T.a_off + (int64_t)tile.mt * T.KB * 2 * A_TILE;
        const float *B = (const float *)bufs[T.sb * NBUF + T.b_buf] + T.b_off + (int64_t)tile.nt * T.KB * 2 * B_TILE;
        for (int kb = 0; kb < T.KB; ++kb, ++it) {
          const int s = (int)(it % PS_STAGES);
          const long long u = it / PS_STAGES;
          if (*abort_v || (u > 0 && !tc::mbar_wait(&empty[s], (uint32_t)((u - 1) & 1), WAIT_BUDGET))) {
            ok = false;
            break;
          }
          float *st = sm + s * STAGE_FLOATS;
          tc::mbar_arrive_expect_tx(&full[s], stage_bytes);
          tc::bulk_g2s(st, A + (int64_t)kb * 2 * A_TILE, 4u * 2 * A_TILE, &full[s]);
          tc::bulk_g2s(st + 2 * A_TILE, B + (int64_t)kb * 2 * B_TILE, 4u * 2 * B_TILE, &full[s]);
        }
      }
      if (!ok) {
        atomicOr(err, IDMRG_DEV_ERR_TIMEOUT);
        atomicOr(&abort_flag, 1);
      }
      // the copies of the last ring window may still be in flight: wait for them
      for (long long j = it > PS_STAGES ? it - PS_STAGES : 0; j < it; ++j)
        tc::mbar_wait(&full[j % PS_STAGES], (uint32_t)((j / PS_STAGES) & 1), WAIT_BUDGET);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ---- MMA issuer
      constexpr uint32_t idesc = tc::instr_desc(TM, TN, BF16 ? 1u : 2u);
      constexpr uint32_t lboA = (TM / 8) * 128, lboB = (TN / 8) * 128, sbo = 128;
      long long it = 0;
      int lt = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const TcTile tile = tiles[t];
        const TcTask T = tasks[tile.task];
        if (active && !active[T.sb]) continue;
        const int a = lt & 1, v = lt >> 1;
        if (*abort_v || (v > 0 && !tc::mbar_wait(&acce[a], (uint32_t)((v - 1) & 1), WAIT_BUDGET))) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
        const uint32_t d = tmem + (uint32_t)(a * TN);
        for (int kb = 0; kb < T.KB; ++kb, ++it) {
          const int s = (int)(it % PS_STAGES);
          if (!tc::mbar_wait(&full[s], (uint32_t)((it / PS_STAGES) & 1), WAIT_BUDGET)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint32_t sa = tc::smem_u32(sm + s * STAGE_FLOATS);
          const uint32_t sb = sa + 4u * 2 * A_TILE;
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const uint64_t ahi = tc::smem_desc(sa + kk * 2 * lboA, lboA, sbo);
            const uint64_t alo = tc::smem_desc(sa + 4u * A_TILE + kk * 2 * lboA, lboA, sbo);
            const uint64_t bhi = tc::smem_desc(sb + kk * 2 * lboB, lboB, sbo);
            const uint64_t blo = tc::smem_desc(sb + 4u * B_TILE + kk * 2 * lboB, lboB, sbo);
            const uint32_t acc0 = (kb > 0 || kk > 0) ? 1u : 0u;
            if (BF16) {
              tc::mma_f16(d, ahi, bhi, idesc, acc0);
              tc::mma_f16(d, ahi, blo, idesc, 1u);
              tc::mma_f16(d, alo, bhi, idesc, 1u);
            } else {
              tc::mma_tf32(d, ahi, bhi, idesc, acc0);
              tc::mma_tf32(d, ahi, blo, idesc, 1u);
              tc::mma_tf32(d, alo, bhi, idesc, 1u);
            }
          }
          tc::mma_commit(&empty[s]);
        }
        if (!ok) break;
        tc::mma_commit(&accf[a]);  // the accumulator of this tile is complete
        ++lt;
      }
      if (!ok) {
        atomicOr(err, IDMRG_DEV_ERR_TIMEOUT);
        atomicOr(&abort_flag, 1);
      }
      tc::mma_commit(&done);  // fires once every MMA issued above has completed
    }
  } else {  // ---- epilogue, warps 2..5: TMEM lane quarter q = warp % 4
    const int q = warp & 3;
    int lt = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
      const TcTile tile = tiles[t];
      const TcTask T = tasks[tile.task];
      if (active && !active[T.sb]) continue;
      const int a = lt & 1, v = lt >> 1;
      // every lane waits; the warp goes on only together (tcgen05.ld is warp-wide)
      const bool got = !*abort_v && tc::mbar_wait(&accf[a], (uint32_t)(v & 1), WAIT_BUDGET);
      if (!__all_sync(0xffffffffu, got)) {
        if (lane == 0) {
          atomicOr(err, IDMRG_DEV_ERR_TIMEOUT);
          atomicOr(&abort_flag, 1);
        }
        break;
      }
      tc::fence_after_sync();
      // lane l holds accumulator row r0 + l; 32 columns at a time go through
      // the warp's staging block, then out row by row with the lanes along
      // the columns (one 128-byte FP32 or 256-byte FP64 store per row)
      const int r0 = tile.mt * TM + 32 * q;
      const int col0 = tile.nt * TN;
      const int nrows = min(32, T.M - r0);
      double *cbase = bufs[T.sb * NBUF + T.c_buf];
      int64_t obase = 0;
      if (T.mode == 1 && lane < nrows) obase = ((const int64_t *)bufs[T.sb * NBUF + T.rmap_buf])[T.rmap_off + r0 + lane];
      float *stg = epi + q * 32 * EPI_LD;
      for (int c = 0; c < TN && col0 + c < T.N; c += EPI_COLS) {
#pragma unroll
        for (int h = 0; h < EPI_COLS; h += 16) {
          float vv[16];
          if (T.KB > 0) {
            tc::tmem_ld16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(a * TN + c + h), vv);
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) vv[i] = 0.f;
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) stg[lane * EPI_LD + h + i] = vv[i];
        }
        __syncwarp();
        const int col = col0 + c + lane;
        if (T.mode == 0) {
          float *out = (float *)cbase + T.c_off + (int64_t)r0 * T.ldc + col;
          for (int r = 0; r < nrows; ++r)
            if (col < T.N) out[(int64_t)r * T.ldc] = stg[r * EPI_LD + lane];
        } else {
          for (int r = 0; r < nrows; ++r) {
            const int64_t ob = __shfl_sync(0xffffffffu, obase, r);
            if (col < T.N) cbase[ob + col] = (double)stg[r * EPI_LD + lane];
          }
        }
        __syncwarp();
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acce[a]);  // this quarter of the accumulator is free
      ++lt;
    }
  }
  __syncthreads();
  const bool ready = tc::mbar_wait(&done, 0, WAIT_BUDGET);
  if (!ready) {
    atomicOr(&abort_flag, 2);
    if (lane == 0) atomicOr(err, IDMRG_DEV_ERR_TIMEOUT);
  }
  tc::fence_before_sync();
  __syncthreads();
  const int aborted = abort_flag;
  if (warp == 0 && !(aborted & 2)) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, 2 * TN);
  }
}

// ------------------------------------------- FP64-accurate digit-slice form
// The Ozaki scheme (Ozaki, Ogita, Oishi, Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and
// its applications", Numer. Algorithms 59, 2012), here with BF16 slices:
// every packed row r (a row of A, or a column of B) gets an exponent e_r with
// |x| < 2^(e_r - 1) for all its elements, and each element becomes
//   x = sum_{p<8} d_p 2^(e_r - 7 (p + 1)),  d_p integer, |d_p| <= 64,
// exact in BF16 (balanced base-128 digits, 56 bits in all; the rest,
// below 2^(e_r - 57), is dropped).  A product of digits is an integer of at
// most 2^12, so the K-sum of the digit products of one level t = p + q is an
// exact FP32 integer while (t + 1) K 2^12 < 2^24; for K <= OZ_MAX_K that holds
// up to t = 4, and the rounding of the higher levels is below 2^-53 of the
// leading terms.  Levels t <= 7 are kept (one 64-column TMEM accumulator
// each); the epilogue sums them with their power-of-two scales.
constexpr int OZ_GA = 16;  // row groups of a packed A tile (128 rows); B tiles have TC_TN / 8
static_assert(OZ_KBLK == 16, "a K block is one kind::f16 MMA step");
// Digit p of element (row, k): K blocks of 16 (one MMA step), row tiles of 8 G
// rows.  A operands (G = 16) keep plane after plane, so that a plane of a block
// is one M = 128 operand; B operands (G = 8) keep the planes of a K chunk one
// after the other, so that consecutive planes read as one operand of 64 rows
// each: A_p against B_q, B_q+1, ... is one MMA, and its output columns are the
// consecutive levels p + q, p + q + 1, ... (see oz_order.h)
__device__ __forceinline__ int64_t oz_off(int row, int k, int KB, int G, int p) {
  const int rows_per_tile = 8 * G;
  const int rt = row / rows_per_tile, rr = row - rt * rows_per_tile;
  const int64_t block = (int64_t)rt * KB + k / OZ_KBLK;
  const int kc = (k & (OZ_KBLK - 1)) >> 3;
  const int64_t run = G == OZ_GA ? (block * OZ_PLANES + p) * 2 + kc : (block * 2 + kc) * OZ_PLANES + p;
  return ((run * G + (rr >> 3)) * 8 + (rr & 7)) * 8 + (k & 7);
}

// exponent of the expansion for a non-zero x: |x| < 2^(e - 1)
__device__ __forceinline__ int oz_exp_of(double x) {
  const int be = (int)((__double_as_longlong(x) >> 52) & 0x7FF);
  return be ? be - 1023 + 2 : ilogb(x) + 2;
}

// Digits of eight consecutive K elements, from the bits of x in integer
// arithmetic (FP64 instructions are scarce here): Y = round(x 2^(56 - e)),
// |Y| <= 2^55, then balanced base-128 digits (-64 .. 63; the leading one takes
// what is left, |d_0| <= 64): Y = sum_p d_p 128^(7 - p).  Adding 64 to every
// digit but the leading one makes them plain 7-bit fields u_p = d_p + 64 of
// Y + 64 sum_{j<7} 128^j.  BF16 128 + u is 0x4300 + u, and subtracting 192 leaves
// d, exactly.  out[p]: plane p, the eight elements in order.
__device__ __forceinline__ uint32_t oz_sub192(uint32_t w) {
  const __nv_bfloat162 r =
      __hsub2(*reinterpret_cast<const __nv_bfloat162 *>(&w), __floats2bfloat162_rn(192.0f, 192.0f));
  return *reinterpret_cast<const uint32_t *>(&r);
}
__device__ __forceinline__ void oz_digits8(const double *v, int e, uint4 (&out)[OZ_PLANES]) {
  constexpr long long bias = 64ll * ((1ll << 49) - 1) / 127;
  uint32_t w[OZ_PLANES][4];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v[i]);
    unsigned long long u = 0;
    if (e != OZ_EXP_EMPTY && (bits << 1) != 0) {
      const int be = (int)((bits >> 52) & 0x7FF);
      unsigned long long mant = bits & ((1ull << 52) - 1);
      int ex = -1074;  // x = mant 2^ex
      if (be) {
        mant |= 1ull << 52;
        ex = be - 1075;
      }
      const int sh = ex + 56 - e;
      if (sh >= 0)
        u = mant << sh;  // sh <= 2 since |x| < 2^(e - 1)
      else if (sh > -62)
        u = (mant + (1ull << (-sh - 1))) >> (-sh);
    }
    const long long Y = ((bits >> 63) ? -(long long)u : (long long)u) + bias;
    const uint32_t lo = (uint32_t)Y, mid = (uint32_t)(Y >> 28), top = (uint32_t)((int)(Y >> 49) + 64);
    const uint32_t d[OZ_PLANES] = {top,               (mid >> 14) & 127u, (mid >> 7) & 127u, mid & 127u,
                                   (lo >> 21) & 127u, (lo >> 14) & 127u,  (lo >> 7) & 127u,  lo & 127u};
#pragma unroll
    for (int p = 0; p < OZ_PLANES; ++p)
      w[p][i >> 1] = (i & 1) ? w[p][i >> 1] + (d[p] << 16) : 0x43004300u + d[p];
  }
#pragma unroll
  for (int p = 0; p < OZ_PLANES; ++p)
    out[p] = make_uint4(oz_sub192(w[p][0]), oz_sub192(w[p][1]), oz_sub192(w[p][2]), oz_sub192(w[p][3]));
}

// Digit packing goes through the windows of pack_kernel, eight K elements of a
// row per thread (a warp fills 512 contiguous bytes of every plane, 128 of a B
// plane).  It is memory bound: 8 bytes in, 16 out per element.  (Before, a
// thread per element stored 16 bits per plane; environments and prediction of
// the kagome cylinder at m = 1000 11.6 -> 8.2 ms a step with it.)
static_assert(W_ROWS == PACK_ROWS && W_K == PACK_K, "windows of oz_store_window");

// The thread's share of a window: packed row row0 + lane (lane < nr), K group
// kw + 8 warp; elements outside [ka, kb) belong to a neighbour.
__device__ __forceinline__ void oz_store_window(__nv_bfloat16 *dst, const double *tile, int e, int row0, int nr, int kw,
                                                int ka, int kb, int KB, int G) {
  const int g = threadIdx.x >> 5, r = threadIdx.x & 31;
  const int kg = kw + 8 * g;
  if (r >= nr || kg + 8 <= ka || kg >= kb) return;
  double v[8];
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    const double2 x = *reinterpret_cast<const double2 *>(tile + r * OP_LD + 8 * g + j);
    v[j] = x.x;
    v[j + 1] = x.y;
  }
  uint4 d[OZ_PLANES];
  oz_digits8(v, e, d);
  const int64_t step = oz_off(0, 0, KB, G, 1);  // from plane to plane
  __nv_bfloat16 *o = dst + oz_off(row0 + r, kg, KB, G, 0);
  if (kg >= ka && kg + 8 <= kb) {
#pragma unroll
    for (int p = 0; p < OZ_PLANES; ++p) *reinterpret_cast<uint4 *>(o + p * step) = d[p];
  } else {
#pragma unroll
    for (int p = 0; p < OZ_PLANES; ++p) {
      const uint32_t w[4] = {d[p].x, d[p].y, d[p].z, d[p].w};
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (kg + j >= ka && kg + j < kb)
          o[p * step + j] = __ushort_as_bfloat16((unsigned short)(w[j >> 1] >> (16 * (j & 1))));
    }
  }
}

// exponents of the rows r0 .. r0 + nr - 1 of a segment into rexp[32] (every
// thread of the block takes part)
template <bool SCALED>
__device__ __forceinline__ void oz_row_exps(const PackSeg &s, const double *src, int r0, int nr, int *rexp) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < OP_ROWS) rexp[threadIdx.x] = OZ_EXP_EMPTY;
  __syncthreads();
  // several loads in flight per thread: the source is read at memory latency
  if (s.trans) {
    int m = OZ_EXP_EMPTY;
    if (lane < nr) {
#pragma unroll 8
      for (int k = warp; k < s.ks; k += 8) {
        const double x = pack_src<SCALED>(s, src, r0 + lane, k);
        if (!is_zero(x)) m = max(m, oz_exp_of(x));
      }
    }
    if (m != OZ_EXP_EMPTY) atomicMax(&rexp[lane], m);
  } else {
    int m[4] = {OZ_EXP_EMPTY, OZ_EXP_EMPTY, OZ_EXP_EMPTY, OZ_EXP_EMPTY};
#pragma unroll 2
    for (int k = lane; k < s.ks; k += 32) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const double x = warp + 8 * i < nr ? pack_src<SCALED>(s, src, r0 + warp + 8 * i, k) : 0.0;
        if (!is_zero(x)) m[i] = max(m[i], oz_exp_of(x));
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      m[i] = __reduce_max_sync(0xffffffffu, m[i]);
      if (lane == 0) rexp[warp + 8 * i] = m[i];
    }
  }
  __syncthreads();
}

// exponents of rows whose K range spans several segments
__global__ void __launch_bounds__(256) oz_exp_kernel(const int2 *__restrict__ units, const PackSeg *__restrict__ segs,
                                                     double *const *__restrict__ bufs,
                                                     const int *__restrict__ active) {
  __shared__ int rexp[OP_ROWS];
  const int2 u = units[blockIdx.x];  // (segment, first row)
  const PackSeg s = segs[u.x];
  if (s.whole || (active && !active[s.sb])) return;
  const int nr = min(OP_ROWS, s.rows - u.y);
  const double *src = bufs[s.sb * NBUF + s.src_buf] + s.src_off;
  if (is_one(s.alpha))
    oz_row_exps<false>(s, src, u.y, nr, rexp);
  else
    oz_row_exps<true>(s, src, u.y, nr, rexp);
  int *ex = (int *)bufs[s.sb * NBUF + s.exp_buf] + s.exp_off + s.row0 + u.y;
  if (threadIdx.x < nr && rexp[threadIdx.x] != OZ_EXP_EMPTY) atomicMax(ex + threadIdx.x, rexp[threadIdx.x]);
}

// digits; a segment that holds the whole K range of its rows finds their
// exponents itself (and stores them), the others read them
__global__ void __launch_bounds__(256, 3) oz_pack_kernel(const int2 *__restrict__ units,
                                                      const PackSeg *__restrict__ segs,
                                                      double *const *__restrict__ bufs,
                                                      const int *__restrict__ active) {
  __shared__ __align__(16) double tile[OP_ROWS * OP_LD];
  __shared__ int rexp[OP_ROWS];
  const int2 u = units[blockIdx.x];  // (segment, first row)
  const PackSeg s = segs[u.x];
  if (active && !active[s.sb]) return;
  const int r0 = u.y, nr = min(OP_ROWS, s.rows - r0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int *ex = (int *)bufs[s.sb * NBUF + s.exp_buf] + s.exp_off + s.row0 + r0;
  const double *src = bufs[s.sb * NBUF + s.src_buf] + s.src_off;
  __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(bufs[s.sb * NBUF + s.dst_buf]) + s.dst_off;
  if (s.whole) {
    if (is_one(s.alpha))
      oz_row_exps<false>(s, src, r0, nr, rexp);
    else
      oz_row_exps<true>(s, src, r0, nr, rexp);
    if (threadIdx.x < nr) ex[threadIdx.x] = rexp[threadIdx.x];
  } else {
    if (threadIdx.x < nr) rexp[threadIdx.x] = ex[threadIdx.x];
  }
  const bool scaled = !is_one(s.alpha);
  const int k1 = s.k0 + s.ks, kend = k1 + s.kpad;  // zeros up to the end of the last K block
  for (int kw = s.k0 & ~(OP_K - 1); kw < kend; kw += OP_K) {
    __syncthreads();
    if (scaled)
      pack_load_window<true>(s, src, r0, nr, kw, tile);
    else
      pack_load_window<false>(s, src, r0, nr, kw, tile);
    __syncthreads();
    oz_store_window(dst, tile, lane < nr ? rexp[lane] : 0, s.row0 + r0, nr, kw, s.k0, kend, s.KB, s.G);
  }
}

// T3 = sum W12 T1 in FP64 from the FP64 stage-1 output, in the windows of
// wstage_tc_kernel.  Pass 0 takes the row exponents of T3, which need all of a
// row (every channel's rectangle); pass 1 writes the digits.  Where T3 copies
// T1 pass 1 reads T1 again, which moves less than storing T3 would; windows
// with sums (the completed channel's, about one in w, of up to 2 w terms, bound
// by the FP64 units) are kept by pass 0 in `keep`, 16 KB each.
constexpr int W_OZ_CTAS[2] = {4, 3};  // resident per SM
template <int PASS>
__global__ void __launch_bounds__(256, W_OZ_CTAS[PASS]) wstage_oz_kernel(const WUnit *__restrict__ units, int nunits,
                                                                         const WTaskP *__restrict__ tasks,
                                                                         const WTerm *__restrict__ terms,
                                                                         double *const *__restrict__ bufs,
                                                                         double *__restrict__ keep,
                                                                         const int *__restrict__ active) {
  __shared__ __align__(16) double tile[PASS ? W_ROWS * OP_LD : 2];
  __shared__ WStage S[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  w_walk(units, nunits, tasks, terms, S, [&](const WUnit &u, WStage &st) {
    const WTaskP &t = st.task;
    if (active && !active[t.sb]) return;
    const int nr = min(W_ROWS, t.rows - u.r0);
    int *ex = (int *)bufs[t.sb * NBUF + BUF_OEXP] + t.exp_off + t.row0 + u.r0;
    const int e = PASS && lane < nr ? ex[lane] : 0;
    double *kept = u.slot >= 0 ? keep + (int64_t)u.slot * (W_ROWS * W_K) + warp * W_K + lane : nullptr;
    double acc[4][2];
    if (PASS == 0 || !kept) {
      w_accumulate<double>(u, terms, bufs[t.sb * NBUF + t.in_buf], nr, st.term, acc);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        acc[i][0] = kept[8 * i * W_K];
        acc[i][1] = kept[8 * i * W_K + 32];
      }
    }
    if (PASS == 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        int m = OZ_EXP_EMPTY;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (!is_zero(acc[i][h])) m = max(m, oz_exp_of(acc[i][h]));
          if (kept) kept[8 * i * W_K + 32 * h] = acc[i][h];
        }
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0 && m != OZ_EXP_EMPTY) atomicMax(ex + warp + 8 * i, m);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        tile[(warp + 8 * i) * OP_LD + lane] = acc[i][0];
        tile[(warp + 8 * i) * OP_LD + lane + 32] = acc[i][1];
      }
      __syncthreads();
      __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(bufs[t.sb * NBUF + t.dst_buf]) + t.dst_off;
      oz_store_window(dst, tile, e, t.row0 + u.r0, nr, u.k0, u.k0, min(u.k0 + W_K, OZ_KBLK * t.KB), t.KB, t.G);
    }
  });
}

constexpr int OZ_A_PLANE = TM * OZ_KBLK * 2;       // bytes of one A digit plane of a K block
constexpr int OZ_B_PLANE = TC_TN * OZ_KBLK * 2;
constexpr int OZ_B_HALF = OZ_B_PLANE / 2;           // of it, one K chunk of 8
constexpr int OZ_B_RUN = (OZ_ZERO + OZ_PLANES) * OZ_B_HALF;  // the stack of a K chunk: zero planes, then the digits
constexpr int OZ_COPY = OZ_PLANES * (OZ_A_PLANE + OZ_B_PLANE);  // bytes copied per K block
constexpr int OZ_STAGE = OZ_PLANES * OZ_A_PLANE + 2 * OZ_B_RUN;
constexpr int OZ_STAGES = 3;
constexpr int OZ_CH = OZ_MAX_K / OZ_KBLK;           // K blocks of one K chunk
constexpr int OZ_TMEM_COLS = 512;                  // 8 levels x 64 columns
constexpr int OZ_EPI_WARPS = 8;                    // two per TMEM lane quarter, 32 columns each
constexpr int OZ_THREADS = 64 + 32 * OZ_EPI_WARPS;
constexpr int OZ_STG_LD = 17;                      // staging block of an epilogue warp: 32 rows x 16 columns
constexpr int OZ_SMEM = OZ_STAGES * OZ_STAGE + OZ_EPI_WARPS * 32 * OZ_STG_LD * 8;
static_assert(OZ_SMEM <= 227 * 1024, "shared memory of a CTA");

// Persistent: one CTA per SM walks the tile list (128 x 64 outputs each, the
// longest K first) with three roles, as tc_gemm_ps_kernel does.  A K block is 36
// digit products of 128 x 64 x 16, issued as 15 MMAs of 128 or 192 columns in
// fixed windows of levels (oz_order.h): 1376 cycles of the tensor pipe with the
// zero planes, and 146 KB of operand reads beside 48 KB of copies, 1515 cycles
// of shared memory; 36 MMAs of 64 columns read 216 KB.  All 512 TMEM columns
// hold one tile, so the MMAs of the next one wait until this one has been read:
// the epilogue warps first take all eight levels into registers (integers, see
// below), release the accumulators, and only then scale, round and store, beside
// the next tile's MMAs.  Tasks longer than OZ_MAX_K have one tile per K chunk, so
// that few but long outputs still fill the chip; these store into the task's
// partial results, which oz_sum_kernel adds up in the order of K.
// Measured (GB300; before: one CTA per tile of 32-element K blocks, 36 MMAs of 64
// columns per 16 of K, the epilogue in FP64 by the row): the two stages of the
// kagome cylinder's H_eff psi at m = 1500 13.1 -> 4.4 ms (39 TFLOP/s
// FP64-accurate), of the J1-J2 cylinder at m = 500 0.81 -> 0.28 ms.  By ncu
// (kagome, m = 1000) the tensor pipe is active 87 % of the cycles in stage 3 (long
// K), close to what the operand reads allow (0.91), and 70 % in stage 1, whose
// tiles have few K blocks beside their read-out (FP64 pipe 29 %); L2 at 26 %.
__global__ void __launch_bounds__(OZ_THREADS, 1) oz_gemm_kernel(const TcTile *__restrict__ tiles, int ntiles,
                                                                const TcTask *__restrict__ tasks,
                                                                double *const *__restrict__ bufs,
                                                                const int *__restrict__ active, int *err) {
  extern __shared__ __align__(1024) uint8_t osm[];
  __shared__ __align__(8) uint64_t full[OZ_STAGES], empty[OZ_STAGES], accf, acce, done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) {
    tc::tmem_alloc(&tmem_base, OZ_TMEM_COLS);
    tc::tmem_relinquish();
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < OZ_STAGES; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
    }
    tc::mbar_init(&accf, 1);
    tc::mbar_init(&acce, OZ_EPI_WARPS);
    tc::mbar_init(&done, 1);
    abort_flag = 0;
    tc::fence_mbar_init();
  }
  // the zero planes of B: no copy touches them
  for (int e = threadIdx.x; e < OZ_STAGES * 2 * OZ_ZERO * (OZ_B_HALF / 16); e += OZ_THREADS) {
    const int run = e / (OZ_ZERO * (OZ_B_HALF / 16)), i = e - run * (OZ_ZERO * (OZ_B_HALF / 16));
    *reinterpret_cast<uint4 *>(osm + (run >> 1) * OZ_STAGE + OZ_PLANES * OZ_A_PLANE + (run & 1) * OZ_B_RUN + 16 * i) =
        make_uint4(0u, 0u, 0u, 0u);
  }
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_base;
  volatile int *abort_v = &abort_flag;

  if (warp == 0) {
    if (lane == 0) {  // ---- producer
      long long it = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const TcTile tile = tiles[t];
        const TcTask T = tasks[tile.task];
        if (active && !active[T.sb]) continue;
        const uint8_t *A = reinterpret_cast<const uint8_t *>(bufs[T.sb * NBUF + T.a_buf]) + 2 * T.a_off +
                           (int64_t)tile.mt * T.KB * OZ_PLANES * OZ_A_PLANE;
        const uint8_t *B = reinterpret_cast<const uint8_t *>(bufs[T.sb * NBUF + T.b_buf]) + 2 * T.b_off +
                           (int64_t)tile.nt * T.KB * OZ_PLANES * OZ_B_PLANE;
        const int kend = min(T.KB, (tile.chunk + 1) * OZ_CH);
        for (int kb = tile.chunk * OZ_CH; kb < kend; ++kb, ++it) {
          const int s = (int)(it % OZ_STAGES);
          const long long u = it / OZ_STAGES;
          if (*abort_v || (u > 0 && !tc::mbar_wait(&empty[s], (uint32_t)((u - 1) & 1), WAIT_BUDGET))) {
            ok = false;
            break;
          }
          uint8_t *st = osm + s * OZ_STAGE;
          tc::mbar_arrive_expect_tx(&full[s], (uint32_t)OZ_COPY);
          tc::bulk_g2s(st, A + (int64_t)kb * OZ_PLANES * OZ_A_PLANE, OZ_PLANES * OZ_A_PLANE, &full[s]);
          for (int kc = 0; kc < 2; ++kc)
            tc::bulk_g2s(st + OZ_PLANES * OZ_A_PLANE + kc * OZ_B_RUN + OZ_ZERO * OZ_B_HALF,
                         B + ((int64_t)kb * 2 + kc) * OZ_PLANES * OZ_B_HALF, OZ_PLANES * OZ_B_HALF, &full[s]);
        }
      }
      if (!ok) {
        atomicOr(err, IDMRG_DEV_ERR_TIMEOUT);
        atomicOr(&abort_flag, 1);
      }
      // the copies of the last ring window may still be in flight: wait for them
      for (long long j = it > OZ_STAGES ? it - OZ_STAGES : 0; j < it; ++j)
        tc::mbar_wait(&full[j % OZ_STAGES], (uint32_t)((j / OZ_STAGES) & 1), WAIT_BUDGET);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ---- MMA issuer
      constexpr uint32_t lboA = (TM / 8) * 128, lboB = OZ_B_RUN, sbo = 128;
      long long it = 0;
      int v = 0;  // tiles so far
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const TcTile tile = tiles[t];
        const TcTask T = tasks[tile.task];
        if (active && !active[T.sb]) continue;
        if (*abort_v || (v > 0 && !tc::mbar_wait(&acce, (uint32_t)((v - 1) & 1), WAIT_BUDGET))) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
        const int kc = tile.chunk * OZ_CH, kend = min(T.KB, kc + OZ_CH);
        for (int kb = kc; kb < kend; ++kb, ++it) {
          const int s = (int)(it % OZ_STAGES);
          if (!tc::mbar_wait(&full[s], (uint32_t)((it / OZ_STAGES) & 1), WAIT_BUDGET)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint32_t sa = tc::smem_u32(osm + s * OZ_STAGE);
          const uint32_t sb = sa + OZ_PLANES * OZ_A_PLANE;
          oz_for_each_mma([&](int p, int q0, int level, int n) {
            tc::mma_f16(tmem + (uint32_t)(TC_TN * level), tc::smem_desc(sa + p * OZ_A_PLANE, lboA, sbo),
                        tc::smem_desc(sb + (OZ_ZERO + q0) * OZ_B_HALF, lboB, sbo), tc::instr_desc(TM, n * TC_TN, 1u),
                        (kb > kc || p > 0) ? 1u : 0u);
          });
          tc::mma_commit(&empty[s]);
        }
        if (!ok) break;
        tc::mma_commit(&accf);  // the levels of this tile are complete
        ++v;
      }
      if (!ok) {
        atomicOr(err, IDMRG_DEV_ERR_TIMEOUT);
        atomicOr(&abort_flag, 1);
      }
      tc::mma_commit(&done);  // fires once every MMA issued above has completed
    }
  } else {  // ---- epilogue: TMEM lane quarter warp % 4, columns 32 w .. 32 w + 31
    const int quarter = warp & 3, cb = 32 * ((warp - 2) >> 2);
    double *stg = reinterpret_cast<double *>(osm + OZ_STAGES * OZ_STAGE) + (warp - 2) * 32 * OZ_STG_LD;
    int v = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
      const TcTile tile = tiles[t];
      const TcTask T = tasks[tile.task];
      if (active && !active[T.sb]) continue;
      const int r0 = tile.mt * TM + 32 * quarter, col0 = tile.nt * TC_TN + cb;
      const int nrows = min(32, T.M - r0);  // may be <= 0
      const int *ex = (const int *)bufs[T.sb * NBUF + T.exp_buf];
      const int ea = lane < nrows ? ex[T.a_exp + r0 + lane] : OZ_EXP_EMPTY;
      const int ebl = col0 + lane < T.N ? ex[T.b_exp + col0 + lane] : OZ_EXP_EMPTY;
      // this lane's output row: of the task's output, or of this chunk's partial results
      double *cbase = bufs[T.sb * NBUF + (T.nch > 1 ? T.part_buf : T.c_buf)];
      const bool accum = T.accum && T.nch == 1;
      int64_t obase = 0;
      if (lane < nrows) {
        if (T.nch > 1)
          obase = T.part_off + ((int64_t)tile.chunk * T.M + r0 + lane) * T.N;
        else if (T.mode == 1)
          obase = ((const int64_t *)bufs[T.sb * NBUF + T.rmap_buf])[T.rmap_off + r0 + lane];
        else
          obase = T.c_off + (int64_t)(r0 + lane) * T.ldc;
      }
      // every lane waits; the warp goes on only together (tcgen05.ld is warp-wide)
      const bool got = !*abort_v && tc::mbar_wait(&accf, (uint32_t)(v & 1), WAIT_BUDGET);
      if (!__all_sync(0xffffffffu, got)) {
        if (lane == 0) {
          atomicOr(err, IDMRG_DEV_ERR_TIMEOUT);
          atomicOr(&abort_flag, 1);
        }
        break;
      }
      tc::fence_after_sync();
      // Levels 0..4 are exact integers, |L_t| <= (t + 1) 768 2^12 < 2^24, and
      // are summed as such: H = sum_t L_t 128^(4-t) in units of 2^-42, with
      // L_0 128 + L_1 and L_2 128 + L_3 within 32 bits and |H| < 2^50.
      // Levels 5..7 carry FP32 rounding anyway: Tl = L_5 2^14 + L_6 2^7 + L_7
      // in FP32, in units of 2^-63 (its error lies below 2^-58 of the leading
      // term).
      long long H[32];
      float Tl[32];
      const uint32_t ta = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)cb;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float x[4][16];
        if (T.KB > 0) {
#pragma unroll
          for (int l = 0; l < 4; ++l) tc::tmem_ld16_async(ta + (uint32_t)(TC_TN * l + 16 * h), x[l]);
          tc::tmem_ld_wait();
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          tc::tmem_ld_fence(x[0][i], x[1][i], x[2][i], x[3][i]);
          const int p01 = __float2int_rn(x[0][i]) * 128 + __float2int_rn(x[1][i]);
          const int p23 = __float2int_rn(x[2][i]) * 128 + __float2int_rn(x[3][i]);
          H[16 * h + i] = T.KB > 0 ? (long long)p01 * (1 << 21) + (long long)p23 * 128 : 0;
        }
        if (T.KB > 0) {
#pragma unroll
          for (int l = 0; l < 4; ++l) tc::tmem_ld16_async(ta + (uint32_t)(TC_TN * (4 + l) + 16 * h), x[l]);
          tc::tmem_ld_wait();
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          tc::tmem_ld_fence(x[0][i], x[1][i], x[2][i], x[3][i]);
          if (T.KB > 0) H[16 * h + i] += __float2int_rn(x[0][i]);
          Tl[16 * h + i] = T.KB > 0 ? fmaf(fmaf(x[1][i], 128.0f, x[2][i]), 128.0f, x[3][i]) : 0.0f;
        }
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acce);  // this warp's part of the accumulators is free
      // value = (H 2^-42 + Tl 2^-63) 2^(ea + eb), one rounding: H 2^(k - 42)
      // exactly (1.5 2^52 + H is H in the low mantissa bits; the FMA takes
      // the offset away), Tl 2^(k - 63) by its exponent bits, one addition.
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int eb = __shfl_sync(0xffffffffu, ebl, 16 * h + i);
          double val = 0.0;
          if (ea != OZ_EXP_EMPTY && eb != OZ_EXP_EMPTY) {
            const int k = ea + eb;
            const long long Hi = H[16 * h + i];
            const float Ti = Tl[16 * h + i];
            if (k - 63 > -1000 && k - 42 < 960) {  // every power of two below is a normal double
              const double s42 = __longlong_as_double((long long)(k - 42 + 1023) << 52);
              const double off = __longlong_as_double(((long long)(k + 10 + 1023) << 52) | (1ll << 51));
              const double hv = fma(__longlong_as_double(0x4338000000000000ll + Hi), s42, -off);
              const uint32_t tb = __float_as_uint(Ti);
              const long long tm = ((long long)(tb & 0x7fffffffu) << 29) + ((long long)(896 + k - 63) << 52);
              const double tv = Ti == 0.0f ? 0.0 : __longlong_as_double(tm | ((long long)(tb >> 31) << 63));
              val = hv + tv;
            } else {
              val = scalbn(fma((double)Ti, 0x1p-21, (double)Hi), k - 42);
            }
          }
          stg[lane * OZ_STG_LD + i] = val;
        }
        __syncwarp();
        // two rows of 16 columns per pass
        const int cl = lane & 15, col = col0 + 16 * h + cl;
#pragma unroll 4
        for (int r = 0; r < 32; r += 2) {
          const int rr = r + (lane >> 4);
          const int64_t ob = __shfl_sync(0xffffffffu, obase, rr);
          if (rr < nrows && col < T.N) {
            double *dst = cbase + ob + col;
            const double val = stg[rr * OZ_STG_LD + cl];
            *dst = accum ? *dst + val : val;
          }
        }
        __syncwarp();
      }
      ++v;
    }
  }
  __syncthreads();
  const bool ready = tc::mbar_wait(&done, 0, WAIT_BUDGET);
  if (!ready) {
    atomicOr(&abort_flag, 2);
    if (lane == 0) atomicOr(err, IDMRG_DEV_ERR_TIMEOUT);
  }
  tc::fence_before_sync();
  __syncthreads();
  const int aborted = abort_flag;
  if (warp == 0 && !(aborted & 2)) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, OZ_TMEM_COLS);
  }
}

// Sums the partial results of the tasks in K chunks, in the order of K; a warp
// per output row, memory bound (8 bytes read per output and chunk).
constexpr int OZ_SUM_ROWS = 8;
__global__ void __launch_bounds__(32 * OZ_SUM_ROWS) oz_sum_kernel(const int *__restrict__ ids,
                                                                  const TcTask *__restrict__ tasks,
                                                                  double *const *__restrict__ bufs,
                                                                  const int *__restrict__ active) {
  const TcTask T = tasks[ids[blockIdx.x]];
  const int row = blockIdx.y * OZ_SUM_ROWS + (threadIdx.x >> 5);
  if (row >= T.M || (active && !active[T.sb])) return;
  const double *part = bufs[T.sb * NBUF + T.part_buf] + T.part_off + (int64_t)row * T.N;
  double *out = bufs[T.sb * NBUF + T.c_buf] +
                (T.mode == 1 ? ((const int64_t *)bufs[T.sb * NBUF + T.rmap_buf])[T.rmap_off + row]
                             : T.c_off + (int64_t)row * T.ldc);
  for (int col = threadIdx.x & 31; col < T.N; col += 32) {
    double x = T.accum ? out[col] + part[col] : part[col];
    for (int c = 1; c < T.nch; ++c) x += part[(int64_t)c * T.M * T.N + col];
    out[col] = x;
  }
}

}  // namespace

cudaError_t launch_oz_exp(const int2 *units, int nunits, const PackSeg *segs, double *const *bufs, const int *active,
                          cudaStream_t st) {
  if (nunits > 0) oz_exp_kernel<<<nunits, 256, 0, st>>>(units, segs, bufs, active);
  return cudaGetLastError();
}

cudaError_t launch_oz_pack(const int2 *units, int nunits, const PackSeg *segs, double *const *bufs, const int *active,
                           cudaStream_t st) {
  if (nunits > 0) oz_pack_kernel<<<nunits, 256, 0, st>>>(units, segs, bufs, active);
  return cudaGetLastError();
}

cudaError_t launch_wstage_oz(const WUnit *units, int nunits, const WTaskP *tasks, const WTerm *terms,
                             double *const *bufs, double *keep, const int *active, int pass, cudaStream_t st) {
  if (nunits <= 0) return cudaGetLastError();
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidValue;
  const int most = W_OZ_CTAS[pass ? 1 : 0] * sms, grid = nunits < most ? nunits : most;
  (pass ? wstage_oz_kernel<1> : wstage_oz_kernel<0>)<<<grid, 256, 0, st>>>(units, nunits, tasks, terms, bufs, keep,
                                                                             active);
  return cudaGetLastError();
}

cudaError_t launch_oz_gemm(const TcTile *tiles, int ntiles, const TcTask *tasks, double *const *bufs,
                           const int *active, int *err, cudaStream_t st) {
  if (ntiles <= 0) return cudaGetLastError();
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(oz_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM);
  if (e != cudaSuccess) return e;
  oz_gemm_kernel<<<ntiles < sms ? ntiles : sms, OZ_THREADS, OZ_SMEM, st>>>(tiles, ntiles, tasks, bufs, active, err);
  return cudaGetLastError();
}

cudaError_t launch_oz_sum(const int *ids, int n, int max_rows, const TcTask *tasks, double *const *bufs,
                          const int *active, cudaStream_t st) {
  if (n > 0 && max_rows > 0) {
    dim3 grid(n, (max_rows + OZ_SUM_ROWS - 1) / OZ_SUM_ROWS);
    oz_sum_kernel<<<grid, 32 * OZ_SUM_ROWS, 0, st>>>(ids, tasks, bufs, active);
  }
  return cudaGetLastError();
}

cudaError_t launch_pack(const int4 *units, int nunits, const PackSeg *segs, double *const *bufs, const int *active,
                        int bf16, cudaStream_t st) {
  if (nunits > 0) pack_kernel<<<nunits, 256, 0, st>>>(units, segs, bufs, active, bf16);
  return cudaGetLastError();
}

cudaError_t launch_wstage_tc(const WUnit *units, int nunits, const WTaskP *tasks, const WTerm *terms,
                             double *const *bufs, const int *active, int bf16, cudaStream_t st) {
  if (nunits <= 0) return cudaGetLastError();
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidValue;
  const int most = W_TC_CTAS * sms;
  wstage_tc_kernel<<<nunits < most ? nunits : most, 256, 0, st>>>(units, nunits, tasks, terms, bufs, active, bf16);
  return cudaGetLastError();
}

template <int TN>
static cudaError_t launch_tc_gemm_tn(const TcTile *tiles, int ntiles, const TcTask *tasks, double *const *bufs,
                                     const int *active, int *err, int bf16, int sms, cudaStream_t st) {
  constexpr int smem = PsShape<TN>::SMEM;
  auto kern = bf16 ? tc_gemm_ps_kernel<true, TN> : tc_gemm_ps_kernel<false, TN>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int grid = ntiles < sms ? ntiles : sms;
  kern<<<grid, PS_THREADS, smem, st>>>(tiles, ntiles, tasks, bufs, active, err);
  return cudaGetLastError();
}

cudaError_t launch_tc_gemm(const TcTile *tiles, int ntiles, const TcTask *tasks, double *const *bufs,
                           const int *active, int *err, int bf16, int tn, cudaStream_t st) {
  if (ntiles <= 0) return cudaGetLastError();
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidValue;
  switch (tn) {
    case 64: return launch_tc_gemm_tn<64>(tiles, ntiles, tasks, bufs, active, err, bf16, sms, st);
    case 128: return launch_tc_gemm_tn<128>(tiles, ntiles, tasks, bufs, active, err, bf16, sms, st);
    case 256: return launch_tc_gemm_tn<256>(tiles, ntiles, tasks, bufs, active, err, bf16, sms, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace idmrg
