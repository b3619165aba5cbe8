// The tube frame of the warm start's per-site kernels (features in mlp.cu,
// initial populations in kernels.cu), included inside their namespaces.
#pragma once

// A frame with the reciprocals its kernels multiply by.
struct WarmDev {
  lbm_warm_frame f;
  double inv_length, inv_radius, inv_rho, inv_u;
};
inline WarmDev warm_dev(const lbm_warm_frame& f) {
  return WarmDev{f, 1.0 / f.length, 1.0 / f.radius, 1.0 / f.rho_scale, 1.0 / f.u_scale};
}

struct SiteFrame {
  double s, r;     // axial coordinate from the inlet plane, distance from the axis
  double er[3];    // outward radial unit vector (0 on the axis)
};

// Its kernels are bound by the FP64 pipe (one warp instruction per SM
// in 16 cycles), so FP64 divisions and square roots, each a dozen or more of
// them, are kept out: 1 / r comes from the FP32 estimate by two Newton steps
// (relative errors 2^-22, 2^-43, then rounding), and r = r^2 (1 / r).
__device__ __forceinline__ SiteFrame site_frame(const int32_t* coords, int64_t i,
                                                const lbm_warm_frame& f) {
  const double p[3] = {coords[3 * i] - f.centre[0], coords[3 * i + 1] - f.centre[1],
                       coords[3 * i + 2] - f.centre[2]};
  const double a = p[0] * f.axis[0] + p[1] * f.axis[1] + p[2] * f.axis[2];
  const double q[3] = {p[0] - a * f.axis[0], p[1] - a * f.axis[1], p[2] - a * f.axis[2]};
  const double r2 = q[0] * q[0] + q[1] * q[1] + q[2] * q[2];
  SiteFrame sf;
  sf.s = a - f.z0;
  double ir = 0.0;
  if (r2 > 1e-24 && r2 < 1e30) {
    ir = (double)rsqrtf((float)r2);
    ir *= fma(-0.5 * r2, ir * ir, 1.5);
    ir *= fma(-0.5 * r2, ir * ir, 1.5);
    sf.r = r2 * ir;
  } else {
    sf.r = sqrt(r2);
    if (sf.r > 1e-12) ir = 1.0 / sf.r;
  }
  for (int k = 0; k < 3; ++k) sf.er[k] = q[k] * ir;
  return sf;
}
