// Pieces shared by the chain kernels that keep a path in a warp's shared memory
// (pmc_chain.cu: one warp per chain, or a team of warps; pmc_group.cuh: several chains
// per warp): the path's arrays, the staged random numbers of a step, and the
// lane-parallel gradient of a vertex.
#pragma once

#include "pmc_internal.h"

namespace pmc {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRefreshSteps = 256;  // recompute the running sums from the caches
constexpr int kFlushAccepts = 64;   // FP32 partials -> FP64 accumulators
constexpr int kRngWords = 8;        // staged words per step
constexpr int kPairWords = 64;      // shared slot for the pair constants (floats)
static_assert(sizeof(DPair) <= kPairWords * sizeof(float), "pair slot too small");
constexpr int kMedWords = 48;       // wavelength sampling: the medium at the chain's wavelength (floats)
static_assert(sizeof(DMedium) <= kMedWords * sizeof(float), "medium slot too small");

enum Move { MV_INTERIOR = 0, MV_END = 1, MV_BIRTH = 2, MV_DEATH = 3 };

// View of one chain's path: entries [0, S) of every array live in the warp's
// shared memory, entries [S, cap) in the chain's global block (same layout:
// array a at offset a * stride).  kTb: tau_b per segment is cached (layered
// media); otherwise it is b * length.  kGt: d log sigma / dg per vertex is
// cached (gradients requested).  kSpill = false: the whole cap fits (S >= cap)
// and every access goes to shared memory.  kRoll: loops over the path are kept
// rolled (path_loop in pmc_chain.cu).
template <bool kTb, bool kGt, bool kSpill, bool kRoll = true>
struct WarpPath {
  static constexpr bool kRolled = kRoll;
  static constexpr int kArrays = 6 + (kTb ? 1 : 0) + (kGt ? 1 : 0);
  static constexpr int kX = 0, kY = 1, kZ = 2, kSeg = 3, kLen = 4, kVt = 5, kTbA = 6, kGtA = 6 + (kTb ? 1 : 0);
  float* sm;   // shared arrays, stride S
  float* gm;   // global block of the chain, stride cap
  int S, cap;
  float b;
  template <int a>
  __device__ __forceinline__ float ld(int i) const {
    if (kSpill && i >= S) return gm[a * cap + i];
    return sm[a * S + i];
  }
  template <int a>
  __device__ __forceinline__ void st(int i, float v) const {
    if (kSpill && i >= S) gm[a * cap + i] = v;
    else sm[a * S + i] = v;
  }
  __device__ float3 pos(int i) const { return f3(ld<kX>(i), ld<kY>(i), ld<kZ>(i)); }
  __device__ void set_pos(int i, float3 p) const {
    st<kX>(i, p.x);
    st<kY>(i, p.y);
    st<kZ>(i, p.z);
  }
  __device__ float seg(int i) const { return ld<kSeg>(i); }
  __device__ float len(int i) const { return ld<kLen>(i); }
  __device__ float vt(int i) const { return ld<kVt>(i); }
  __device__ void set_seg(int i, float v) const { st<kSeg>(i, v); }
  __device__ void set_len(int i, float v) const { st<kLen>(i, v); }
  __device__ void set_vt(int i, float v) const { st<kVt>(i, v); }
  __device__ float tb(int i) const {
    if constexpr (kTb) return ld<kTbA>(i);
    else return b * ld<kLen>(i);
  }
  __device__ float gt(int i) const {
    if constexpr (kGt) return ld<kGtA>(i);
    else return 0.f;
  }
  __device__ void set_tb(int i, float v) const {
    if constexpr (kTb) st<kTbA>(i, v);
  }
  __device__ void set_gt(int i, float v) const {
    if constexpr (kGt) st<kGtA>(i, v);
  }
};

// d log p / d f_v with the terms spread over lanes: lanes 0-1 the two segment
// factors that end / start at v, lanes 2-4 the scattering angles at v-1, v,
// v+1, lane 5 the emission and detection factors; a shuffle tree sums them
// and every lane returns the total.  Same formulas as grad_vertex.
template <class PosF>
__device__ float3 grad_vertex_warp(const DMedium& M, const DPair& S, float zoff, PosF pos, int n, int v, int lane) {
  float3 pv[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int k = min(max(v - 2 + i, 0), n - 1);
    pv[i] = pos(k);
  }
  float3 rh[4];
  float el[4];
  bool ex[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = v - 2 + i;
    ex[i] = (k >= 0 && k <= n - 2);
    const float3 r = pv[i + 1] - pv[i];
    const float rr = dot(r, r);
    const float ir = ex[i] ? rsqrtf(rr) : 1.0f;
    el[i] = ex[i] ? rr * ir : 1.0f;
    rh[i] = ir * r;
  }
  float3 g = f3(0.f, 0.f, 0.f);
  if (lane < 2) {
    const bool e = (lane == 0) ? ex[1] : ex[2];
    const float3 P = (lane == 0) ? pv[1] : pv[2];
    const float3 Q = (lane == 0) ? pv[2] : pv[3];
    const float3 r = (lane == 0) ? rh[1] : rh[2];
    const float l = (lane == 0) ? el[1] : el[2];
    if (e) {
      float3 dP, dQ;
      dtau_dends(M, zoff, P, Q, l, r, dP, dQ);
      g = (lane == 0) ? (f3(0.f, 0.f, 0.f) - dQ - (2.0f / l) * r) : ((2.0f / l) * r - dP);
    }
  } else if (lane < 5) {
    const int k = v - 3 + lane;
    if (k >= 1 && k <= n - 2) {
      const float3 A = (lane == 2) ? rh[0] : ((lane == 3) ? rh[1] : rh[2]);
      const float3 B = (lane == 2) ? rh[1] : ((lane == 3) ? rh[2] : rh[3]);
      const float lA = (lane == 2) ? el[0] : ((lane == 3) ? el[1] : el[2]);
      const float lB = (lane == 2) ? el[1] : ((lane == 3) ? el[2] : el[3]);
      const float alpha = (lane == 2) ? 0.f : ((lane == 3) ? 1.f : -1.f);
      const float beta = (lane == 2) ? 1.f : ((lane == 3) ? -1.f : 0.f);
      const float w = phase_dlogdc(M, A, B);
      g = w * (alpha * drdot(A, lA, B) + beta * drdot(B, lB, A));
    }
  } else if (lane == 5) {
    if (S.emission != 0) {
      const float3 ed = f3(S.dir[0], S.dir[1], S.dir[2]);
      if (v == 1) g = g + S.kappa * drdot(rh[1], el[1], ed);
      if (v == 0 && ex[2]) g = g - S.kappa * drdot(rh[2], el[2], ed);
    }
    if (v == n - 2 || v == n - 1) {
      const float3 e = (v == n - 1) ? pv[2] : pv[3];
      const float3 rhat = (v == n - 1) ? rh[1] : rh[2];
      const float ell = (v == n - 1) ? el[1] : el[2];
      float3 nu = (e - f3(S.c[0], S.c[1], S.c[2])) - f3(S.c_lo[0], S.c_lo[1], S.c_lo[2]);
      const float dn = sqrtf(dot(nu, nu));
      nu = (1.0f / dn) * nu;
      const float u = -dot(rhat, nu);
      const float3 t1 = drdot(rhat, ell, nu);
      if (v == n - 2) {
        g = g + (1.0f / u) * t1;
      } else {
        const float3 t2 = drdot(nu, dn, rhat);
        g = g - (1.0f / u) * (t1 + t2);
        if (S.rho != 0) {
          const float3 rh_ = f3(S.rho_hat[0], S.rho_hat[1], S.rho_hat[2]);
          const float x = dot(nu, rh_);
          const float dl = 3.0f - 2.0f * tanhf(fmaf(2.0f, x, 0.7f));
          g = g + dl * drdot(nu, dn, rh_);
        }
      }
    }
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    g.x += __shfl_xor_sync(kFull, g.x, o);
    g.y += __shfl_xor_sync(kFull, g.y, o);
    g.z += __shfl_xor_sync(kFull, g.z, o);
  }
  return f3(__shfl_sync(kFull, g.x, 0), __shfl_sync(kFull, g.y, 0), __shfl_sync(kFull, g.z, 0));
}

// Point of a birth: mid-point of the foci + sc * t.  In a homogeneous medium the
// rounding of the z coordinate follows `fuse_z` (product and sum rounded once,
// or each), so that the paths do not depend on which instance of which kernel
// runs a chain.
template <bool kGen>
__device__ __forceinline__ float3 birth_point(float3 A, float3 B, float sc, float3 t, int fuse_z) {
  if constexpr (kGen) {
    return 0.5f * (A + B) + sc * t;
  } else {
    const float3 m = 0.5f * (A + B);
    const float pz = __fmul_rn(sc, t.z);
    return f3(__fadd_rn(m.x, __fmul_rn(sc, t.x)), __fadd_rn(m.y, __fmul_rn(sc, t.y)),
              fuse_z ? __fmaf_rn(sc, t.z, m.z) : __fadd_rn(m.z, pz));
  }
}

// Pre-transformed random numbers of one step (8 staged words):
//   lo.x = 23-bit index draw | move type << 24, lo.y = log u (accept),
//   within: lo.z, lo.w, hi.x = standard normals, hi.y = vMF cosine,
//           hi.z, hi.w = cos, sin of the vMF azimuth
//   birth:  lo.z = u for cos s, lo.w = sinh t, hi.x = cosh t, hi.y, hi.z = cos, sin of phi
// Returns the move type (0 within, 2 birth, 3 death).
__device__ __forceinline__ uint32_t stage_step(const DRun& R, const DPair& S, unsigned long long t, uint32_t cid,
                                               uint32_t key0, uint32_t key1, uint4& lo, uint4& hi) {
  const uint4 ra = philox4x32_10(make_uint4(static_cast<uint32_t>(t), static_cast<uint32_t>(t >> 32), cid, PUR_STEP_A),
                                 key0, key1);
  const uint4 rb = philox4x32_10(make_uint4(static_cast<uint32_t>(t), static_cast<uint32_t>(t >> 32), cid, PUR_STEP_B),
                                 key0, key1);
  const uint32_t um = ra.x >> 9;
  const uint32_t type = um < R.thr_within ? 0u : (um < R.thr_birth ? 2u : 3u);
  lo = make_uint4((ra.y >> 9) | (type << 24), __float_as_uint(__logf(u01(ra.z))), 0u, 0u);
  const float ub0 = u01(rb.x), ub1 = u01(rb.y), ub2 = u01(rb.z), ub3 = u01(rb.w);
  if (type == 0u) {
    float s1, c1, s2, c2;
    const float r1 = m_sqrt<true>(-2.0f * __logf(ub0));
    sincospif(2.0f * ub1, &s1, &c1);
    const float r2 = m_sqrt<true>(-2.0f * __logf(ub2));
    sincospif(2.0f * ub3, &s2, &c2);
    lo.z = __float_as_uint(r1 * c1);
    lo.w = __float_as_uint(r1 * s1);
    const float wv = 1.0f + __fdividef(__logf(fmaf(1.0f - ub0, S.exp_m2ke, ub0)), S.kappa_end);
    hi = make_uint4(__float_as_uint(r2 * c2), __float_as_uint(wv), __float_as_uint(c1), __float_as_uint(s1));
  } else {
    const float et = __fdividef(ub1, 1.0f - ub1);
    const float iet = __fdividef(1.0f - ub1, ub1);
    float s3, c3;
    sincospif(2.0f * ub2, &s3, &c3);
    lo.z = __float_as_uint(ub0);
    lo.w = __float_as_uint(0.5f * (et - iet));
    hi = make_uint4(__float_as_uint(0.5f * (et + iet)), __float_as_uint(c3), __float_as_uint(s3), 0u);
  }
  return type;
}

}  // namespace pmc
