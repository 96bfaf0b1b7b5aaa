// The correction of one column pair in the refinement of a sector SVD (k_refine.cu on the tensor cores,
// svd_small_kernel of k_svd.cu inside one CTA).
#pragma once

namespace mps {

struct RefinePair {
  float2 pq, qp;      // s_p E_pq / s_q and s_q E_qp / s_p
  float size;         // the larger of the relative change of the smaller column and of the other's rotation
};

// A step's diagonal is E_pp = (R_pp - sum_k |E_kp|^2) / 2: with the second-order term V's columns keep their norm
// to third order, which the singular values see directly (orthogonality errors only at second order).
//
// al, be: |a_p|^2 / s_p^2 and |a_q|^2 / s_q^2; rho = s_q / s_p; g = a_p^dag a_q / (s_p s_q); r = R_pq of
// R = I - V^dag V; tol: columns with |g| <= tol |a_p| |a_q| count as orthogonal.
__device__ __forceinline__ RefinePair refine_pair(float al, float be, float rho, float gr, float gi, float rr,
                                                  float ri, float tol) {
  RefinePair out;
  const float br = be * rho * rho;                  // lambda_q / s_p^2
  const float dif = br - al;
  if (fabsf(dif) > 0.03f * fmaxf(al, br)) {
    const float ip = 1.f / dif, brq = be * rho;
    out.pq = make_float2((gr + brq * rr) * ip, (gi + brq * ri) * ip);
    // E_qp = conj(S_pq + lambda_p R_pq) / (lambda_p - lambda_q)
    const float f = -rho * ip;
    out.qp = make_float2((gr * rho + al * rr) * f, -(gi * rho + al * ri) * f);
  } else {      // close values: orthonormalise by R / 2 and turn by the Jacobi angle
    const float mean = 0.5f * (al / rho + be * rho);
    const float hr = gr + mean * rr, hi = gi + mean * ri, ag = hypotf(hr, hi);
    float tx = 0.f, ty = 0.f;
    if (ag > tol * sqrtf(al * be)) {      // orthogonal to rounding otherwise
      const float z = dif / (2.f * rho * ag), az = fabsf(z);
      const float tt = copysignf(1.f, z) / (az + (az < 1e18f ? sqrtf(fmaf(z, z, 1.f)) : az));
      const float c = rsqrtf(fmaf(tt, tt, 1.f));
      tx = c * tt * hr / ag;
      ty = c * tt * hi / ag;
    }
    out.pq = make_float2((0.5f * rr + tx) / rho, (0.5f * ri + ty) / rho);
    out.qp = make_float2((0.5f * rr - tx) * rho, -(0.5f * ri - ty) * rho);
  }
  const float a1 = hypotf(out.pq.x, out.pq.y), a2 = hypotf(out.qp.x, out.qp.y);
  out.size = rho <= 1.f ? fmaxf(a1, a2 / rho) : fmaxf(a2, a1 * rho);
  return out;
}

// Whether a step of size th settles K columns of n rows: its second-order error K th^2 is below half the
// orthogonality threshold eps max(n, 32) of the FP64 sweeps.
__device__ __forceinline__ bool refine_settles(float th, int K, int n) {
  return (double)K * th * th < 0.5 * 2.220446049250313e-16 * (n > 32 ? n : 32);
}
// Whether the steps do not contract (step counts from 0): leave the sector to the FP64 sweeps.
__device__ __forceinline__ bool refine_fails(float th, int step) { return !(th < (step > 0 ? 0.3f : 1.6f)); }

}  // namespace mps
