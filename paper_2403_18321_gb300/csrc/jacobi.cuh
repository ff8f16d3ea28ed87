// jacobi.cuh -- device code shared by the two Jacobi kernels: the rotation of a
// pair and the thread-block-cluster primitives.
#pragma once

#include "tma.cuh"

namespace gbpca {

__device__ __forceinline__ float rcp_nr(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return fmaf(r, fmaf(-x, r, 1.f), r);
}
__device__ __forceinline__ float rsqrt_nr(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return fmaf(y, fmaf(-0.5f * x * y, y, 0.5f), y);
}
__device__ __forceinline__ float sqrt_est(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Eqs. 2-5: small root t of Eq. 3 as t = sgn(tau)/(|tau| + sqrt(1+tau^2)),
// tau = (aqq - app)/(2 apq); an off-diagonal below 2^-24 sqrt(|app aqq|) is
// dropped without rotating (c = 1, s = 0).  Returns the record of the pair:
// (c, s) and the two diagonal values after the rotation and position swap.
// With d = aqq - app and n = 2 apq the same root is
// t = sgn(tau) |n| / (|d| + sqrt(d^2 + n^2)) (sgn 0 = +1): three dependent
// reciprocal/root steps instead of four (the step's critical path runs
// through this record).  Where d^2 + n^2 could leave the FP32 range (|d| or
// |n| beyond 1e18, or both below 1e-18) the scale-free tau form is taken.
// The drop test runs beside the root, and one rotation follows either root.  With the
// test before the root and a rotation for each in the cluster kernel (the same values) a step
// takes, in us: 144 bands 0.757 for 0.762 here, 188 bands 0.810 / 0.795, 224 bands 0.817 /
// 0.805, 246 bands 0.846 / 0.837, 252 bands 0.881 / 0.894, 256 bands 0.900 / 0.910; the Jacobi
// stage of 256 tiles 7.2 to 7.7 ms in both.
__device__ __forceinline__ float4 pair_record(float app, float aqq, float apq) {
  const float thr = 5.9604645e-08f * sqrt_est(fabsf(app)) * sqrt_est(fabsf(aqq));
  const bool keep = fabsf(apq) > thr;
  const float d = aqq - app, n = 2.f * apq;
  const float ad = fabsf(d), an = fabsf(n);
  auto root = [&]() {
    const float q = fmaf(d, d, n * n);
    const float t = an * rcp_nr(ad + q * rsqrt_nr(q));
    return (d != 0.f && ((d < 0.f) != (n < 0.f))) ? -t : t;
  };
  auto root_scale_free = [&]() {
    const float tau = (aqq - app) * rcp_nr(2.f * apq);
    const float at = fabsf(tau);
    float t;
    if (at > 1e18f) {
      t = 0.5f * rcp_nr(at);
    } else {
      const float u = fmaf(tau, tau, 1.f);
      t = rcp_nr(at + u * rsqrt_nr(u));
    }
    return (tau >= 0.f) ? t : -t;
  };
  auto rotation = [&](float t) {
    const float c = rsqrt_nr(fmaf(t, t, 1.f));
    return make_float4(c, t * c, fmaf(t, apq, aqq), fmaf(-t, apq, app));
  };
  const bool in_range = ad < 1e18f && an < 1e18f && (ad > 1e-18f || an > 1e-18f);
  float t;
  if (!keep || in_range) t = root();
  else t = root_scale_free();
  const float4 r = rotation(t);
  return keep ? r : make_float4(1.f, 0.f, aqq, app);
}

// M' = G_I M G_J, G = [[s, c], [c, -s]].
__device__ __forceinline__ void rot_block(float2 csI, float2 csJ, float& m00, float& m01,
                                          float& m10, float& m11) {
  const float cI = csI.x, sI = csI.y, cJ = csJ.x, sJ = csJ.y;
  const float t00 = fmaf(m00, sJ, m01 * cJ), t01 = fmaf(m00, cJ, -m01 * sJ);
  const float t10 = fmaf(m10, sJ, m11 * cJ), t11 = fmaf(m10, cJ, -m11 * sJ);
  m00 = fmaf(sI, t00, cI * t10);
  m01 = fmaf(sI, t01, cI * t11);
  m10 = fmaf(cI, t00, -sI * t10);
  m11 = fmaf(cI, t01, -sI * t11);
}

// Shared-memory address a (this CTA's window) in the window of CTA `rank`.
__device__ __forceinline__ uint32_t mapa(uint32_t a, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// Phase test with cluster-scope acquire (the data other CTAs sent).
__device__ __forceinline__ bool mbar_try_cluster(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

}  // namespace gbpca
