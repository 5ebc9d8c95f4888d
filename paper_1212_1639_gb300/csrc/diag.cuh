// The cycle's correctly rounded arithmetic on arrays of the caller's, for tests
// (pf_diag_arith): one thread per pair of binary32 values or per binary64 value.
#pragma once
#include "kernels.cuh"

namespace pfk {

enum ArithOp : int {
  OP_RCP2 = 0,     // 1 / a
  OP_DIV2 = 1,     // a / b
  OP_SQRT2 = 2,    // sqrt a
  OP_SQRT1 = 3,    // the same for one value
  OP_QUOT2 = 4,    // a / b of the predictive weights, any operands
  OP_IG2 = 5,      // a / b of the inverse-gamma draws, shapes below 2^60
  OP_IG2_WIDE = 6, // and from there on
  OP_SCALE_R = 7,  // the propagation's 1 / (a + b)
  OP_SCALE_S = 8,  // and sqrt((a b) / (a + b))
  OP_F32_COUNT = 9,
  OP_DIV64 = 16,
  OP_SQRT64 = 17
};

static __global__ void __launch_bounds__(BLOCK) k_arith32(int op, const float2* a, const float2* b, float2* out,
                                                          uint64_t pairs) {
  const uint64_t i = (uint64_t)blockIdx.x * BLOCK + threadIdx.x;
  if (i >= pairs) return;
  const float2 x = a[i], y = b[i];
  float2 r = make_float2(0.0f, 0.0f), ri, sv;
  switch (op) {
    case OP_RCP2: r = rcp_rn2(x); break;
    case OP_DIV2: r = div_rn2(x, y); break;
    case OP_SQRT2: r = sqrt_rn2(x); break;
    case OP_SQRT1: r = make_float2(sqrt_rn1(x.x), sqrt_rn1(x.y)); break;
    case OP_QUOT2: r = quot2(x, y); break;
    case OP_IG2: r = ig2(x, y, false); break;
    case OP_IG2_WIDE: r = ig2(x, y, true); break;
    default:
      state_scale2(x, y, addp(x, y), &ri, &sv);
      r = op == OP_SCALE_R ? ri : sv;
  }
  out[i] = r;
}
static __global__ void __launch_bounds__(BLOCK) k_arith64(int op, const double* a, const double* b, double* out,
                                                          uint64_t n) {
  const uint64_t i = (uint64_t)blockIdx.x * BLOCK + threadIdx.x;
  if (i < n) out[i] = op == OP_DIV64 ? div_rn(a[i], b[i]) : sqrt_rn(a[i]);
}

}  // namespace pfk
