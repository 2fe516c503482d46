// The MMAs of one K block of the digit-slice GEMM (kernels_tc.cu): which digit
// planes each multiplies and which accumulators it adds to.
//
// tcgen05.mma instructions run asynchronously; two of them are only ordered if
// they name the same accumulator and the same shape.  So the eight levels
// t = p + q lie in windows, and every MMA covers exactly one window: digit
// plane p of A against as many planes of B, from q0 = (first level of the
// window) - p on.  Where that is below plane 0 the stack of B planes begins with
// OZ_ZERO planes of zeros, which add exactly nothing.
//
// Windows of 2, 3 and 3 levels take 15 MMAs and 43 plane products a K block (36
// without the zeros) and read 146 KB of operands from shared memory, the least
// of the splits into a few windows.  Measured (GB300, H_eff psi of the kagome
// cylinder at m = 1500 on the digit slices): 6.08 ms; windows of 1, 3 and 4
// levels 6.15, of 4 and 4 6.34, of 2 each 6.28, of 1 each 7.89.  MMAs that each
// take the levels their plane reaches, on accumulators that partly overlap (12 a
// block, no zeros), were 5.8 ms, but nothing orders them.
#pragma once

#ifdef __CUDACC__
#define OZ_ORDER_FN __device__ __forceinline__
#else
#define OZ_ORDER_FN inline
#endif

namespace idmrg {

constexpr int OZ_PLANES = 8;  // digits of an element, levels kept
constexpr int OZ_NWIN = 3;    // windows
OZ_ORDER_FN constexpr int oz_first(int w) {  // first level of window w
  return w <= 0 ? 0 : w == 1 ? 2 : w == 2 ? 5 : OZ_PLANES;
}
constexpr int OZ_ZERO = 2;    // zero planes before plane 0 of B: levels of the widest window - 1

// mma(p, q0, level, n): planes q0 .. q0 + n - 1 of B, levels from `level` on, in
// the order of issue; the first one of a window has p = 0
template <class F>
OZ_ORDER_FN void oz_for_each_mma(F mma) {
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int p = 0; p < OZ_PLANES; ++p) {
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int w = 0; w < OZ_NWIN; ++w)
      if (p < oz_first(w + 1)) mma(p, oz_first(w) - p, oz_first(w), oz_first(w + 1) - oz_first(w));
  }
}

}  // namespace idmrg
