// pft_records.cuh -- FP32 face records without FP64 arithmetic (GB300's FP64 pipe is a small fraction
// of its FP32 rate), for the batched prep kernels of the forward call and the adjoint.
#pragma once

#include "pft_common.cuh"
#include "pft_kernels.cuh"

namespace pft {

// Record of a face with corners x about the centre c = chi + clo (float pairs), and its largest corner
// distance (raised by a relative 1e-6 to stay above the exact one).  Each centred corner is a float pair
// s + t (TwoSum of the vertex and the centre's high part, less its low part); the centroid is rounded
// once from the pair sum over 3 (the remainder of the rounded quotient is exact through its FMA), q0, q1
// and the edges from TwoSum differences, N = e1 x e2 with Kahan's FMA form of each 2 x 2 determinant.
// kUnrounded: q0 and q1 relative to the centroid before its rounding (the adjoint's records: its errors
// are those of records rounded once from FP64; relative to the rounded centroid they are 1.4 times that).
template <bool kUnrounded>
__device__ __forceinline__ Face32 face_record32(const float (&x)[3][3], const float (&chi)[3], const float (&clo)[3],
                                                float& far) {
  auto det2 = [](float a, float b, float cc, float dd) {   // a b - cc dd
    const float w = cc * dd;
    return fmaf(a, b, -w) + fmaf(-cc, dd, w);
  };
  float sp[3][3], tp[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float e;
      two_sum(x[k][d], -chi[d], sp[k][d], e);
      tp[k][d] = e - clo[d];
    }
  float G[3], Q0[3], Q1[3], e1[3], e2[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    float a, ea, b, eb;
    two_sum(sp[0][d], sp[1][d], a, ea);
    two_sum(a, sp[2][d], b, eb);
    const float lo = (ea + eb) + (tp[0][d] + tp[1][d] + tp[2][d]);
    const float gh = b / 3.0f;
    const float rest = (fmaf(-gh, 3.0f, b) + lo) / 3.0f;
    G[d] = gh + rest;
    const float glo = kUnrounded ? rest - (G[d] - gh) : 0.f;
    float y, ey;
    two_sum(sp[0][d], -G[d], y, ey);
    Q0[d] = y + (ey + (kUnrounded ? tp[0][d] - glo : tp[0][d]));
    two_sum(sp[1][d], -G[d], y, ey);
    Q1[d] = y + (ey + (kUnrounded ? tp[1][d] - glo : tp[1][d]));
    two_sum(sp[1][d], -sp[0][d], y, ey);
    e1[d] = y + (ey + (tp[1][d] - tp[0][d]));
    two_sum(sp[2][d], -sp[0][d], y, ey);
    e2[d] = y + (ey + (tp[2][d] - tp[0][d]));
  }
  far = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k)
    far = fmaxf(far, sqrtf(fmaf(sp[k][0], sp[k][0], fmaf(sp[k][1], sp[k][1], sp[k][2] * sp[k][2]))) * 1.000001f);
  return Face32{G[0], G[1], G[2], Q0[0], Q0[1], Q0[2], Q1[0], Q1[1], Q1[2], det2(e1[1], e2[2], e1[2], e2[1]),
                det2(e1[2], e2[0], e1[0], e2[2]), det2(e1[0], e2[1], e1[1], e2[0])};
}

}  // namespace pft
