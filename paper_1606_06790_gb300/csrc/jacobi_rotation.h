// The rotation of the FP32 block tournament (kernels_svd.cu), in a header of its
// own so that the host can check its arithmetic.
#pragma once
#include <float.h>
#include <math.h>

#ifdef __CUDACC__
#define JACOBI_FN __device__ __forceinline__
#else
#define JACOBI_FN inline
static inline float rsqrtf(float x) { return 1.0f / sqrtf(x); }
static inline float __frcp_rn(float x) { return 1.0f / x; }
#endif

namespace idmrg {

// The rotation that makes columns of squared norms a, b and overlap g
// orthogonal, in FP32 with correctly rounded divisions and square roots: false if
// their relative overlap is at most tol.  Approximate ones (__fdividef, products
// with rsqrtf) shorten the tournament's sub-rounds by a tenth (GB300, J1-J2
// cylinder at m = 1024: 20.5 ms against 22.5 a step) and lose two bits of the
// angle.
JACOBI_FN bool js_rotation(float a, float b, float g, float tol, float &ratio, float &t, float &c, float &sn) {
  if (!(a > 0.f) || !(b > 0.f)) return false;
  ratio = fabsf(g) / (sqrtf(a) * sqrtf(b));
  if (!(ratio > tol)) return false;
  const float z = (b - a) / (2.0f * g);
  t = z == 0.f ? 1.0f : copysignf(__frcp_rn(fabsf(z) + sqrtf(fmaf(z, z, 1.0f))), z);
  if (!(fabsf(t) >= FLT_MIN) || !(fabsf(t) <= FLT_MAX)) return false;
  c = rsqrtf(fmaf(t, t, 1.0f));
  sn = c * t;
  return true;
}

}  // namespace idmrg
