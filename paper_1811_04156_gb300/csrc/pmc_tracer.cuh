// Forward photon transport of the comparison tracer (Collin,
// arXiv:1811.04156, appendix "Ray tracer"): one photon from the point source
// through the medium to the first sensor crossing.  Shared by every tracer
// kernel of the library (pmc_trace, pmc_trace_lengths, pmc_trace_paths, the
// chain seeding and the allocation-free pmc_trace_noalloc), so there is one
// copy of the photon's physics.
//
// Transport model: the photon leaves the source in a direction drawn from the
// emission law.  Each flight draws an optical depth tau ~ Exp(1) for the next
// scattering; the next event is whichever comes first of the scattering point
// (where the scattering depth along the ray reaches tau) and the first
// crossing of the sensor sphere.  The flight's absorption depth lowers the
// photon's log weight ln w (w = exp(-integrated absorption), starting at
// w = 1).  At the sensor the photon is detected with weight w rho.  Otherwise
// it scatters (cos theta from the phase function, azimuth uniform) unless
// it started the flight farther than r_reject from the sensor centre or has
// used its max_scatter scatterings.
//
// Random numbers: Philox4x32-10 with key (k0, k1) and counter (photon low,
// photon high, i, PUR_TRACE): block i = 0 gives the emission direction
// (x, y), block i + 1 the flight after i scatterings (x: optical depth, y:
// cos theta, z: azimuth, w: the phase-mixture choice; y doubles as the
// thinning uniform of a detected photon).
#pragma once

#include "pmc_internal.h"

namespace pmc {

// Quotients by a divisor that a photon's flights share, correctly rounded.
// With y = 1/d correctly rounded, a quotient within one unit in the last
// place is rounded correctly by one residual step (P. Markstein,
// "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990, theorem on quotients from a correctly rounded
// reciprocal); the first residual step brings a * y within that unit.  So
// the result is a / d for operands and quotients away from the range's ends
// (here a is an optical depth in [2^-24, 17] or of order 1, and trace_lean
// bounds d), in five operations without the division's range checks.
struct SharedDivisor {
  float d, y;
  __device__ explicit SharedDivisor(float divisor) : d(divisor), y(1.0f / divisor) {}
  __device__ __forceinline__ float quotient(float a) const {
    float q = __fmul_rn(a, y);
    q = __fmaf_rn(__fmaf_rn(-d, q, a), y, q);
    return __fmaf_rn(__fmaf_rn(-d, q, a), y, q);
  }
};

// What the flights of a thread's photons share (b: lean photons only).
struct FlightConsts {
  SharedDivisor by_b, by_2g;
  __device__ explicit FlightConsts(const DMedium& M) : by_b(M.b), by_2g(2.0f * M.g) {}
};

// Distance along direction (0, 0, nz) component nz from height z_abs at
// which the scattering depth reaches tau: tau / b in a homogeneous medium;
// layered media walk the horizontal layers the ray crosses.
template <bool kLean>
__device__ inline float free_path(const DMedium& M, const FlightConsts& C, float z_abs, float nz, float tau) {
  if constexpr (kLean) return C.by_b.quotient(tau);
  if (M.kind == 0) return tau / M.b;
  float walked = 0.f, z = z_abs;
  int l = layer_of(M, z);
  for (int guard = 0; guard < (1 << 16); ++guard) {
    const float b = __ldg(M.lb + l);
    // distance to the layer's boundary in the ray's vertical direction (end
    // layers extend to infinity)
    float to_edge = __int_as_float(0x7f800000);
    int next = l;
    if (nz > 0.f && l < M.n_layers - 1) {
      to_edge = (M.z0 + (l + 1) * M.dz - z) / nz;
      next = l + 1;
    } else if (nz < 0.f && l > 0) {
      to_edge = (M.z0 + l * M.dz - z) / nz;
      next = l - 1;
    }
    to_edge = fmaxf(to_edge, 0.f);
    if (tau <= b * to_edge) return walked + tau / b;
    tau -= b * to_edge;
    walked += to_edge;
    z += to_edge * nz;
    l = next;
  }
  return walked;
}

// Distance along unit direction nh from x to the first crossing of the sphere
// |p - c|^2 = R2 ahead of x (infinity when the ray misses it).
__device__ inline float sphere_crossing(float3 x, float3 nh, float3 c, float R2) {
  const float3 w = x - c;
  const float half_b = dot(w, nh);
  const float disc = half_b * half_b - (dot(w, w) - R2);
  if (disc < 0.f) return __int_as_float(0x7f800000);
  const float t = -half_b - sqrtf(disc);
  return t > 0.f ? t : __int_as_float(0x7f800000);
}

// cos theta drawn from the phase mixture f_sl p_SL + (1 - f_sl) p_HG by
// inversion of each component's CDF (umix picks the component).
template <bool kLean>
__device__ inline float draw_cos_theta(const DMedium& M, const FlightConsts& C, float u, float umix) {
  if (!kLean && M.f_sl > 0.f && umix < M.f_sl) {
    // simplified Liu: density proportional to (1 + cos)^alpha
    return 2.0f * powf(u, 1.0f / (M.sl_alpha + 1.0f)) - 1.0f;
  }
  const float g = M.g;
  if (!kLean && fabsf(g) < 1e-6f) return 2.0f * u - 1.0f;
  const float q = (1.0f - g * g) / (1.0f - g + 2.0f * g * u);
  return fminf(fmaxf(C.by_2g.quotient(1.0f + g * g - q * q), -1.0f), 1.0f);
}

// Unit vector at polar cosine ct and azimuth (sin, cos) = (sp, cp) about axis.
__device__ inline float3 turn_about(float3 axis, float ct, float sp, float cp) {
  float3 e1, e2;
  onb(axis, e1, e2);
  const float st = sqrtf(fmaxf(0.f, 1.0f - ct * ct));
  return ct * axis + st * (cp * e1 + sp * e2);
}

struct PhotonResult {
  bool hit;     // reached the sensor
  float lw;     // ln(w rho) of a detected photon
  float L;      // path length of a detected photon
  int nsc;      // scatterings before detection
  float u_acc;  // spare uniform of the detecting flight (thinning by w rho)
};

// kLean instances leave out the parts that a homogeneous medium with a pure
// Henyey-Greenstein phase function (g not 0), isotropic emission and rho = 1
// never takes, and divide by b and 2 g through their reciprocals; what they
// compute is the same.  8e6 photons of 255 flights in the detector geometry:
// 18.6 ms with the one general kernel, 15.7 ms with the lean one on the same
// grid, 15.4 on the grid of trace_grid (the issue slots bind: 290 warp
// instructions per flight at 80 % issue before).
inline bool trace_lean(const DMedium& M, const DPair& S) {
  return M.kind == 0 && M.b > 1e-20f && M.b < 1e20f && !(M.f_sl > 0.f) && !(M.g > -1e-6f && M.g < 1e-6f) &&
         S.emission == 0 && S.rho == 0;
}

// A photon in flight.
struct Photon {
  float3 x, nh;       // where it starts its next flight (frame coordinates) and the direction
  float lnw, walked;  // log weight and path length so far
  int i;              // scatterings so far
};

// The photon as it leaves the source: isotropic, or von Mises-Fisher about
// S.dir (inverse CDF in cos).
template <bool kLean>
__device__ __forceinline__ Photon emit_photon(const DPair& S, uint32_t k0, uint32_t k1, unsigned long long ph) {
  const uint4 r = philox4x32_10(make_uint4(static_cast<uint32_t>(ph), static_cast<uint32_t>(ph >> 32), 0u, PUR_TRACE),
                                k0, k1);
  float sp, cp;
  sincospif(2.0f * u01(r.y), &sp, &cp);
  const float u0 = u01(r.x);
  float3 nh;
  if (!kLean && S.emission != 0) {
    const float ct = 1.0f + logf(fmaf(1.0f - u0, expf(-2.0f * S.kappa), u0)) / S.kappa;
    nh = turn_about(f3(S.dir[0], S.dir[1], S.dir[2]), ct, sp, cp);
  } else {
    const float ct = 2.0f * u0 - 1.0f;
    const float st = sqrtf(fmaxf(0.f, 1.0f - ct * ct));
    nh = f3(st * cp, st * sp, ct);
  }
  return Photon{f3(0.f, 0.f, 0.f), nh, 0.f, 0.f, 0};
}

// One flight of photon ph: true when it was the last (detected, escaped or
// out of scatterings; `res` is filled), else the photon has scattered.
// `next` receives the flight's end point.
template <bool kLean>
__device__ __forceinline__ bool fly_photon(const DMedium& M, const DPair& S, const FlightConsts& C, uint32_t k0,
                                           uint32_t k1, unsigned long long ph, float r_reject, int max_scatter,
                                           Photon& p, PhotonResult& res, float3& next) {
  const float3 c = f3(S.c[0], S.c[1], S.c[2]);
  const uint4 r = philox4x32_10(make_uint4(static_cast<uint32_t>(ph), static_cast<uint32_t>(ph >> 32),
                                           static_cast<uint32_t>(p.i + 1), PUR_TRACE), k0, k1);
  const float3 x = p.x, nh = p.nh;
  const float to_scatter = free_path<kLean>(M, C, x.z + S.zoff, nh.z, -logf(u01(r.x)));
  const float to_sensor = sphere_crossing(x, nh, c, S.R2);
  const bool detect = to_sensor < to_scatter;
  const float flight = detect ? to_sensor : to_scatter;
  next = x + flight * nh;
  float ta, tb;
  if constexpr (kLean) ta = M.a * flight;
  else seg_tau(M, x.z + S.zoff, next.z + S.zoff, flight, ta, tb);
  p.lnw -= ta;
  if (detect) {
    float lr = 0.f;
    if (!kLean && S.rho != 0) {
      const float xx = dot(sensor_normal(S, next), f3(S.rho_hat[0], S.rho_hat[1], S.rho_hat[2]));
      lr = fmaf(3.0f, xx, -1.0f) - logf(coshf(fmaf(2.0f, xx, 0.7f)));
    }
    res = PhotonResult{true, p.lnw + lr, p.walked + to_sensor, p.i, u01(r.y)};
    return true;
  }
  const float3 from_c = x - c;
  const bool escaped = dot(from_c, from_c) > r_reject * r_reject;
  if (escaped || p.i == max_scatter) {
    res = PhotonResult{false, 0.f, 0.f, 0, 1.f};
    return true;
  }
  p.x = next;
  p.walked += to_scatter;
  float sp, cp;
  sincospif(2.0f * u01(r.z), &sp, &cp);
  const float3 out = turn_about(nh, draw_cos_theta<kLean>(M, C, u01(r.y), u01(r.w)), sp, cp);
  p.nh = rsqrtf(dot(out, out)) * out;
  ++p.i;
  return false;
}

// One photon (index ph) with its vertices (source, scattering points, sensor
// crossing) recorded to (ox, oy, oz) in absolute coordinates (frame
// coordinates + S.org).
__device__ inline PhotonResult record_photon(const DMedium& M, const DPair& S, uint32_t k0, uint32_t k1,
                                             unsigned long long ph, float r_reject, int max_scatter, float* ox,
                                             float* oy, float* oz) {
  const FlightConsts C(M);
  Photon p = emit_photon<false>(S, k0, k1, ph);
  PhotonResult res;
  float3 at = p.x;
  for (;;) {
    const int i = p.i;
    if (i == 0) {
      ox[0] = at.x + S.org[0];
      oy[0] = at.y + S.org[1];
      oz[0] = at.z + S.org[2];
    }
    const bool done = fly_photon<false>(M, S, C, k0, k1, ph, r_reject, max_scatter, p, res, at);
    ox[i + 1] = at.x + S.org[0];
    oy[i + 1] = at.y + S.org[1];
    oz[i + 1] = at.z + S.org[2];
    if (done) return res;
  }
}

// Photons photon0 .. photon0 + n_photons - 1, one per thread and trip; `done`
// runs on the photon's thread when it ends, with its index and result.
// (Lanes that take the next photon as soon as theirs ends gain nothing: most
// photons use all their scatterings, and the refill's votes at every flight
// cost 14 % in the two-sensor scene.)
template <bool kLean, class F>
__device__ __forceinline__ void trace_photons(const DMedium& M, const DPair& S, uint32_t k0, uint32_t k1,
                                              unsigned long long photon0, unsigned long long n_photons, float r_reject,
                                              int max_scatter, F&& done) {
  const unsigned long long stride = static_cast<unsigned long long>(gridDim.x) * blockDim.x;
  const FlightConsts C(M);
  for (unsigned long long q = blockIdx.x * blockDim.x + threadIdx.x; q < n_photons; q += stride) {
    const unsigned long long ph = photon0 + q;
    Photon p = emit_photon<kLean>(S, k0, k1, ph);
    PhotonResult res;
    float3 next;
    while (!fly_photon<kLean>(M, S, C, k0, k1, ph, r_reject, max_scatter, p, res, next)) {}
    done(ph, res);
  }
}

}  // namespace pmc
