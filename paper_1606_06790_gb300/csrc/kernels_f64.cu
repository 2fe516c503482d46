// FP64 block-sparse contraction kernels of the iDMRG hot path.
//
//  * gemm_f64: the grouped block GEMM used for H_eff psi (Step 3: L . psi and
//    T3 . R^T), the block-spin transformation (Step 6, Eqs. L and R) and the
//    prediction (Step 3', Eq. wfprediction).  A task is one output block;
//    several (A, B) segments may be summed into it (MPO channels folded into
//    the contraction index).
//  * wstage_f64: the two-site MPO stage T3[c] = sum W_{c1} W_{c2} T1[a] and the
//    one-site stage of Step 6, as weighted sums of equally shaped sub-blocks.
//  * dot_terms: weighted sub-block dot products (centre-bond energies).
//  * rand_blocks: SplitMix64 start vectors (Step 3, n = 1, 2).
//  * scale_tasks: diagonal scalings by lambda and 1/lambda (Eq. wfprediction).
#include "common.h"

namespace idmrg {

namespace {

// Grouped GEMM.  The FP64 units bound it, by far: an SM retires one warp-wide
// FMA per 16 cycles (2 FMA lanes per clock), each holding its sub-partition's
// unit for 64, whereas the operands of even a 16 x 16 tile come to 2 bytes per
// clock and SM.  So the split serves the FP64 units alone:
//  * 16 x 16 outputs per CTA, one 8 x 8 quadrant per warp (2 outputs a lane):
//    a warp on each sub-partition, 128 cycles per k whatever the problem, and
//    no more padding than a ragged 8 x 8 quadrant (quadrants outside the task
//    issue nothing).  The 64 x 64 .. 32 x 32 tiles before it (4 x 4 outputs a
//    lane) took 1024 cycles per k on the two sub-partitions they occupied when
//    the chip was not full, and padded every sector to their size.
//  * exact trip counts in k: sectors of a few states are common, and a padded
//    k costs as much as a real one.
//  * the next K step is on its way to registers while the current one is
//    multiplied out of shared memory (two buffers, one barrier per step).
// The k order of every output is the segments' order, so the results do not
// depend on the tiling.  Task lists hold 32 x 32 tiles; a CTA takes a quarter
// of one (four times less list to build and upload).
// Measured (GB300), the tuned 64 x 64 .. 32 x 32 tiles before -> now: H_eff psi
// of one superblock at m = 32 77 -> 26 us (the call), of the J1-J2 cylinder at
// m = 200 1.13 -> 0.61 ms, of the 16-site chain at m = 500 3.74 -> 2.96 ms
// (0.98 of 1.26 TFLOP/s), of the kagome cylinder at m = 700 21.6 -> 18.1 ms.
constexpr int TK = 16, TS = 16;

__global__ void __launch_bounds__(128) gemm_f64_kernel(const GemmTile *__restrict__ tiles,
                                                       const GemmTask *__restrict__ tasks,
                                                       const GemmSeg *__restrict__ segs,
                                                       double *const *__restrict__ bufs,
                                                       const int *__restrict__ active) {
  __shared__ double As[2][TK][TS + 1];
  __shared__ __align__(16) double Bs[2][TK][TS + 2];
  const GemmTile tile = tiles[blockIdx.x >> 2];
  const GemmTask task = tasks[tile.task];
  const int m0 = tile.m0 + TS * ((blockIdx.x >> 1) & 1), n0 = tile.n0 + TS * (blockIdx.x & 1);
  if (m0 >= task.M || n0 >= task.N || (active && !active[task.sb])) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wr = 8 * (warp >> 1), wc = 8 * (warp & 1);
  const int r = wr + (lane >> 2), c = wc + 2 * (lane & 3);
  const bool live = m0 + wr < task.M && n0 + wc < task.N;
  double acc0 = 0.0, acc1 = 0.0;
  double ra[2], rb[2];  // the step being fetched
  GemmSeg sg{};
  const double *A = nullptr, *B = nullptr;
  int s = task.seg0 - 1, k0 = 0, kn = 0;  // segment, first k and length of the step being fetched
  const int s_end = task.seg0 + task.nseg;
  auto fetch = [&]() {
    k0 += TK;
    if (s < task.seg0 || k0 >= sg.K) {
      k0 = 0;
      do {
        if (++s >= s_end) {
          kn = 0;
          return;
        }
        sg = segs[s];
      } while (sg.K <= 0);
      A = bufs[task.sb * NBUF + sg.a_buf] + sg.a_off;
      B = bufs[task.sb * NBUF + sg.b_buf] + sg.b_off;
    }
    kn = min(TK, sg.K - k0);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int hi = (tid + 128 * q) >> 4, lo = tid & 15;
      {
        const int m = m0 + ((sg.flags & 1) ? lo : hi), k = (sg.flags & 1) ? hi : lo;
        ra[q] = 0.0;
        if (m < task.M && k < kn)
          ra[q] = (sg.flags & 1) ? A[(int64_t)(k0 + k) * sg.lda + m] : A[(int64_t)m * sg.lda + k0 + k];
      }
      {
        const int n = n0 + ((sg.flags & 2) ? hi : lo), k = (sg.flags & 2) ? lo : hi;
        rb[q] = 0.0;
        if (n < task.N && k < kn)
          rb[q] = (sg.flags & 2) ? B[(int64_t)n * sg.ldb + k0 + k] : B[(int64_t)(k0 + k) * sg.ldb + n];
      }
    }
  };
  fetch();
  for (int buf = 0; kn > 0; buf ^= 1) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int hi = (tid + 128 * q) >> 4, lo = tid & 15;
      const double va = sg.alpha != 1.0 ? ra[q] * sg.alpha : ra[q];
      if (sg.flags & 1) As[buf][hi][lo] = va;
      else As[buf][lo][hi] = va;
      if (sg.flags & 2) Bs[buf][lo][hi] = rb[q];
      else Bs[buf][hi][lo] = rb[q];
    }
    const int n = kn;
    __syncthreads();
    fetch();
    if (live) {
#pragma unroll 4
      for (int k = 0; k < n; ++k) {
        const double a = As[buf][k][r];
        const double2 b = *reinterpret_cast<const double2 *>(&Bs[buf][k][c]);
        acc0 = fma(a, b.x, acc0);
        acc1 = fma(a, b.y, acc1);
      }
    }
  }
  const int gm = m0 + r, gn = n0 + c;
  if (gm >= task.M) return;
  double *C = bufs[task.sb * NBUF + task.c_buf] + task.c_off + (int64_t)gm * task.ldc + gn;
  if (gn < task.N) C[0] = task.accumulate ? C[0] + acc0 : acc0;
  if (gn + 1 < task.N) C[1] = task.accumulate ? C[1] + acc1 : acc1;
}

constexpr int WROWS = 16;

__global__ void wstage_f64_kernel(const WTask *__restrict__ tasks, const WTerm *__restrict__ terms,
                                  double *const *__restrict__ bufs, const int *__restrict__ active) {
  const WTask t = tasks[blockIdx.x];
  if (active && !active[t.sb]) return;
  const int r0 = blockIdx.y * WROWS;
  if (r0 >= t.rows) return;
  const int r1 = min(t.rows, r0 + WROWS);
  double *out = bufs[t.sb * NBUF + t.out_buf] + t.out_off;
  const double *in = bufs[t.sb * NBUF + t.in_buf];
  const int n = (r1 - r0) * t.cols;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int r = r0 + e / t.cols, c = e % t.cols;
    double acc = 0.0;
    for (int q = 0; q < t.nterm; ++q) {
      const WTerm w = terms[t.term0 + q];
      acc = fma(w.coef, in[w.in_off + (int64_t)r * w.in_ld + c], acc);
    }
    out[(int64_t)r * t.out_ld + c] = acc;
  }
}

__global__ void dot_terms_kernel(const DotTerm *__restrict__ terms, double *const *__restrict__ bufs,
                                 double *__restrict__ partial) {
  const DotTerm t = terms[blockIdx.x];
  const double *a = bufs[t.sb * NBUF + t.buf] + t.off1;
  const double *b = bufs[t.sb * NBUF + t.buf] + t.off2;
  double acc = 0.0;
  const int n = t.rows * t.cols;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int r = e / t.cols, c = e % t.cols;
    acc = fma(a[(int64_t)r * t.ld1 + c], b[(int64_t)r * t.ld2 + c], acc);
  }
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (threadIdx.x == 0) partial[blockIdx.x] = t.coef * acc;
  }
}

// SplitMix64: output k of the stream with state s is mix(s + (k+1) * GAMMA).
__device__ __forceinline__ uint64_t sm64_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void rand_blocks_kernel(const RandBlock *__restrict__ blocks, double *const *__restrict__ bufs,
                                   int buf) {
  const RandBlock b = blocks[blockIdx.x];
  const int r0 = blockIdx.y * WROWS;
  if (r0 >= b.rows) return;
  const int r1 = min(b.rows, r0 + WROWS);
  double *out = bufs[b.sb * NBUF + buf] + b.off;
  const int n = (r1 - r0) * b.cols;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int r = r0 + e / b.cols, c = e % b.cols;
    const uint64_t k = (uint64_t)(b.dense0 + (int64_t)r * b.dense_rs + c);
    const uint64_t z = sm64_mix(b.state + (k + 1ull) * 0x9E3779B97F4A7C15ull);
    const double u = (double)(z >> 11) * 0x1.0p-53;
    out[(int64_t)r * b.ld + c] = 2.0 * u - 1.0;
  }
}

__global__ void scale_tasks_kernel(const ScaleTask *__restrict__ tasks, const double *__restrict__ table,
                                   double zero_rel, double *const *__restrict__ bufs) {
  const ScaleTask t = tasks[blockIdx.x];
  const int r0 = blockIdx.y * WROWS;
  if (r0 >= t.rows) return;
  const int r1 = min(t.rows, r0 + WROWS);
  const double *src = bufs[t.sb * NBUF + t.src_buf] + t.off;
  double *dst = bufs[t.sb * NBUF + t.dst_buf] + t.off;
  const double thr = t.rs_inv ? zero_rel * table[t.max_off] : 0.0;
  const int n = (r1 - r0) * t.cols;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int r = r0 + e / t.cols, c = e % t.cols;
    double f = 1.0;
    if (t.rs_off >= 0) {
      const double l = table[t.rs_off + r];
      f = t.rs_inv ? (l > thr ? 1.0 / l : 0.0) : l;
    }
    if (t.cs_off >= 0) f *= table[t.cs_off + c];
    dst[(int64_t)r * t.ld + c] = src[(int64_t)r * t.ld + c] * f;
  }
}

}  // namespace

cudaError_t launch_gemm_f64(const GemmTile *tiles, int ntiles, const GemmTask *tasks, const GemmSeg *segs,
                            double *const *bufs, const int *active, cudaStream_t st) {
  static_assert(GEMM_TILE == 2 * TS, "a list tile is four CTA tiles");
  if (ntiles > 0) gemm_f64_kernel<<<4 * ntiles, 128, 0, st>>>(tiles, tasks, segs, bufs, active);
  return cudaGetLastError();
}

cudaError_t launch_wstage_f64(const WTask *tasks, int ntasks, int max_rows, const WTerm *terms,
                              double *const *bufs, const int *active, cudaStream_t st) {
  if (ntasks > 0 && max_rows > 0) {
    dim3 grid(ntasks, (max_rows + WROWS - 1) / WROWS);
    wstage_f64_kernel<<<grid, 256, 0, st>>>(tasks, terms, bufs, active);
  }
  return cudaGetLastError();
}

cudaError_t launch_dot_terms(const DotTerm *terms, int nterms, double *const *bufs, double *partial,
                             cudaStream_t st) {
  if (nterms > 0) dot_terms_kernel<<<nterms, 256, 0, st>>>(terms, bufs, partial);
  return cudaGetLastError();
}

cudaError_t launch_rand_blocks(const RandBlock *blocks, int nblocks, int max_rows, double *const *bufs, int buf,
                               cudaStream_t st) {
  if (nblocks > 0 && max_rows > 0) {
    dim3 grid(nblocks, (max_rows + WROWS - 1) / WROWS);
    rand_blocks_kernel<<<grid, 256, 0, st>>>(blocks, bufs, buf);
  }
  return cudaGetLastError();
}

cudaError_t launch_scale_tasks(const ScaleTask *tasks, int ntasks, int max_rows, const double *table,
                               double zero_rel, double *const *bufs, cudaStream_t st) {
  if (ntasks > 0 && max_rows > 0) {
    dim3 grid(ntasks, (max_rows + WROWS - 1) / WROWS);
    scale_tasks_kernel<<<grid, 256, 0, st>>>(tasks, table, zero_rel, bufs);
  }
  return cudaGetLastError();
}

}  // namespace idmrg
