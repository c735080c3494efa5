// Density, adjoint, score, normalisation, estimator and forward-tracer kernels
// (Collin, arXiv:1811.04156).
#include <algorithm>

#include "pmc_internal.h"
#include "pmc_tracer.cuh"

namespace pmc {

namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Batch accessor: SoA [3][batch][cap] positions, evaluated in the caller's
// absolute frame (the pair struct passed to these kernels uses that frame).
struct BatchPos {
  const float* xyz;
  size_t plane, off;
  __device__ float3 operator()(int i) const {
    return f3(xyz[off + i], xyz[plane + off + i], xyz[2 * plane + off + i]);
  }
};

// ---------------------------------------------------------------------------
// Density of a batch of paths.  A block takes a tile of kP
// consecutive paths and spreads the concatenated list of their vertices over
// its threads, item f of the list on thread f mod kTile, so that no lane idles
// because its path is shorter than a warp; a path's terms meet again in
// shared memory.
//
// Bound by instruction issue (304 warp instructions per 32 vertices, 78 % issue,
// against 12 bytes per vertex).  One warp per path ran at 16.6 active lanes on
// paths of 21 vertices: 131,072 paths (cap 64) took 60 us, in tiles 31 us.
// ---------------------------------------------------------------------------
constexpr int kTile = 128;          // threads of a block
constexpr int kTileItems = 1024;    // vertices whose terms a block holds at once
constexpr int kTilePaths = 32;      // paths of a tile, and of a small batch's or long paths' tile
constexpr int kTilePathsFew = 4;

// Tiles of 4 paths (a warp each for their sums) where 32 would leave fewer than
// three blocks per SM, eight where paths are longer than 64 (paths of 21 vertices: 5,000 3.75 us in tiles of 4 and
// 6.69 in tiles of 32, 12,000 6.34 and 7.30, 14,500 7.07 and 7.40; 8,000 of 65
// vertices 8.4 and 17.4, 14,700 12.3 and 17.8, 30,000 21.2 and 25.6, 65,536 as
// fast in either), or where the cap exceeds 128 (tiles of 32 were not measured there).
inline bool tile_few(int batch, int cap, int n_sm) {
  return cap > 128 || batch < (cap > 64 ? 8 : 3) * kTilePaths * n_sm;
}

// First item of each of the tile's paths (invalid vertex counts: no items),
// in offs[0 .. kP]; returns the number of items.
template <int kP>
__device__ __forceinline__ int tile_offsets(const int* __restrict__ nn, int b0, int batch, int cap, int* offs) {
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    const int n = (lane < kP && b0 + lane < batch) ? nn[b0 + lane] : 0;
    int incl = (n >= 2 && n <= cap) ? n : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 0) offs[0] = 0;
    if (lane < kP) offs[lane + 1] = incl;
  }
  __syncthreads();
  return offs[kP];
}

// Path of item f.
template <int kP>
__device__ __forceinline__ int tile_path(const int* offs, int f) {
  int p = 0;
#pragma unroll
  for (int h = kP / 2; h > 0; h >>= 1)
    if (offs[p + h] <= f) p += h;
  return p;
}

// Sum of a chunk's items [c0, c1) of the path that this thread helps to add up
// (kTile / kP threads per path): term i of the path goes to partial sum i mod 32
// (mod 64 in tiles of 4 paths), and a thread's partial sums meet in pairs, then the
// threads', as 32 lanes would add the path up.  So a path of at most 32 vertices
// has the same log p whatever tile it is in.  (Eight partial sums per path in tiles of
// 32 lost accuracy: 4.07e-8 from 64 bits on 131,072 paths of 21 vertices, against
// 4.02e-8 with 32 at the same time, 31 us.)
template <int kP>
__device__ __forceinline__ float tile_partial(const int* offs, const float* term, int c0, int c1) {
  constexpr int kT = kTile / kP, kA = kT < 32 ? 32 / kT : 2, kS = kT * kA;
  const int p = threadIdx.x / kT, part = threadIdx.x % kT;
  const int o = offs[p], hi = min(offs[p + 1], c1);
  float v[kA];
#pragma unroll
  for (int j = 0; j < kA; ++j) v[j] = 0.f;
  int f = o + part;
  if (o < c0) {  // the path began in an earlier chunk: its stride that holds c0
    f += (c0 - o) / kS * kS;
#pragma unroll
    for (int j = 0; j < kA; ++j) {
      const int q = f + j * kT;
      if (q >= c0 && q < hi) v[j] += term[q - c0];
    }
    f += kS;
  }
  for (; f + (kA - 1) * kT < hi; f += kS) {
#pragma unroll
    for (int j = 0; j < kA; ++j) v[j] += term[f + j * kT - c0];
  }
#pragma unroll
  for (int j = 0; j < kA - 1; ++j) {
    if (f + j * kT >= hi) break;
    v[j] += term[f + j * kT - c0];
  }
#pragma unroll
  for (int h = kA / 2; h > 0; h >>= 1)
#pragma unroll
    for (int j = 0; j < h; ++j) v[j] += v[j + h];
  return v[0];
}
template <int kP>
__device__ __forceinline__ float tile_total(float v) {
#pragma unroll
  for (int o = kTile / kP / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Factors of vertex i of an n-vertex path and of the segment that leaves it,
// as vertex_term and segment_term give them, without branches between the
// source, the scattering vertices and the end vertex: one logarithm serves
// the phase function and the detection factor.
template <bool kGen>
__device__ __forceinline__ float tile_term(const DMedium& M, const DPair& S, float zoff, float3 Pp, float3 P, float3 Pn,
                                           int i, int n) {
  const bool first = i == 0, last = i == n - 1;
  const float3 r = Pn - P, a0 = P - Pp;
  const float l2 = dot(r, r);
  const float3 b = rsqrtf(l2) * r;
  const float3 a = rsqrtf(dot(a0, a0)) * a0;
  // detection: cos of the arrival angle
  float3 nu = f3(0.f, 0.f, 0.f);
  float arg;
  const float3 dm = a - b;
  const float omc = 0.5f * dot(dm, dm);
  arg = fmaf(M.two_g, omc, M.omg2);
  if (last) {
    nu = sensor_normal(S, P);
    arg = -dot(a, nu);
  }
  const float lg = logf(arg);
  float vt;
  if (last) {
    vt = arg > 0.0f ? lg : kNegInf;
    if (kGen && S.rho != 0 && arg > 0.0f) {
      const float x = dot(nu, f3(S.rho_hat[0], S.rho_hat[1], S.rho_hat[2]));
      vt += fmaf(3.0f, x, -1.0f) - logf(coshf(fmaf(2.0f, x, 0.7f)));
    }
    return vt;
  }
  if (first) {
    vt = kGen ? emission_term(S, b) : -kLog4Pi;
  } else {
    const float lhg = fmaf(-1.5f, lg, M.hg_lognorm);
    float ph = lhg;
    if (kGen && M.f_sl > 0.0f) {
      const float3 dp = a + b;
      const float opc = 0.5f * dot(dp, dp);
      const float lsl = fmaf(M.sl_alpha, logf(0.5f * opc), M.sl_lognorm);
      const float mx = fmaxf(lhg, lsl);
      ph = mx + logf((1.0f - M.f_sl) * expf(lhg - mx) + M.f_sl * expf(lsl - mx));
    }
    vt = (kGen ? log_b_at(M, P.z + zoff) : M.log_b) + ph;
  }
  const float ell = sqrtf(l2);
  float ta = M.a * ell, tb = M.b * ell;
  if constexpr (kGen) seg_tau(M, P.z + zoff, Pn.z + zoff, ell, ta, tb);
  float seg = -(ta + tb) - logf(l2);
  if (!(l2 > 0.0f)) seg = kNegInf;
  if (i <= n - 3 && hits_ball(S, P, r)) seg = kNegInf;
  return vt + seg;
}

// log p of each path (NaN marks an invalid vertex count).
template <int kP, bool kGen>
__global__ void __launch_bounds__(kTile) logp_kernel(const DMedium M, const DPair S, const float* __restrict__ xyz,
                                                     const int* __restrict__ nn, int batch, int cap,
                                                     float* __restrict__ out_logp) {
  __shared__ int offs[kP + 1];
  __shared__ float term[kTileItems];
  const int b0 = blockIdx.x * kP;
  const size_t plane = static_cast<size_t>(batch) * cap;
  const int total = tile_offsets<kP>(nn, b0, batch, cap, offs);
  float lp = 0.f;
  for (int c0 = 0; c0 < total; c0 += kTileItems) {
    const int c1 = min(total, c0 + kTileItems);
    for (int f = c0 + threadIdx.x; f < c1; f += kTile) {
      const int p = tile_path<kP>(offs, f);
      const int i = f - offs[p], n = offs[p + 1] - offs[p];
      const BatchPos pos{xyz, plane, static_cast<size_t>(b0 + p) * cap};
      const float3 P = pos(i);
      const float3 Pp = (i >= 1) ? pos(i - 1) : P;
      const float3 Pn = (i <= n - 2) ? pos(i + 1) : P;
      term[f - c0] = tile_term<kGen>(M, S, S.zoff, Pp, P, Pn, i, n);
    }
    __syncthreads();
    lp += tile_partial<kP>(offs, term, c0, c1);
    __syncthreads();
  }
  lp = tile_total<kP>(lp);
  constexpr int kT = kTile / kP;
  const int p = threadIdx.x / kT;
  if (threadIdx.x % kT == 0 && b0 + p < batch)
    out_logp[b0 + p] = offs[p + 1] > offs[p] ? lp : __int_as_float(0x7fc00000);
}

// log p of each path and d log p / d xyz (one warp per path).  (Tiles of paths
// as in logp_kernel, with the phase function's derivative shared through
// shared memory instead of taken three times per vertex, measured no faster
// on 32,768 paths of 49 vertices in the two-sensor scene: 139 us against 137.)
__global__ void logp_grad_kernel(const DMedium M, const DPair S, const float* __restrict__ xyz,
                            const int* __restrict__ nn, int batch, int cap, float* __restrict__ out_logp,
                            float* __restrict__ out_grad) {
  const int lane = threadIdx.x & 31;
  const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (b >= batch) return;
  const int n = nn[b];
  const float zoff = S.zoff;
  BatchPos pos{xyz, static_cast<size_t>(batch) * cap, static_cast<size_t>(b) * cap};
  float lp = 0.f;
  if (n >= 2 && n <= cap) {
    for (int i = lane; i < n; i += 32) {
      const float3 P = pos(i);
      const float3 Pp = (i >= 1) ? pos(i - 1) : P;
      const float3 Pn = (i <= n - 2) ? pos(i + 1) : P;
      float g;
      lp += vertex_term(M, S, zoff, Pp, P, Pn, i, n, g);
      if (i <= n - 2) lp += segment_term(M, S, zoff, P, Pn, i <= n - 3).seg;
    }
    lp = warp_sum(lp);
  } else {
    lp = __int_as_float(0x7fc00000);  // NaN marks an invalid vertex count
  }
  if (lane == 0 && out_logp) out_logp[b] = lp;
  const size_t plane = static_cast<size_t>(batch) * cap;
  const size_t off = static_cast<size_t>(b) * cap;
  const bool ok = n >= 2 && n <= cap && isfinite(lp);
  for (int i = lane; i < cap; i += 32) {
    float3 g = f3(0.f, 0.f, 0.f);
    if (ok && i < n) g = grad_vertex(M, S, zoff, pos, n, i);
    out_grad[off + i] = g.x;
    out_grad[plane + off + i] = g.y;
    out_grad[2 * plane + off + i] = g.z;
  }
}

// d log p / d theta per path.  Homogeneous theta = (lambda_s, lambda_a, g):
//   (L b^2 - (n-2) b, L a^2, sum_k d log sigma/d g);  layered theta =
// (lambda_s[l], lambda_a[l]): (len_l b_l^2 - n_l b_l, len_l a_l^2), with len_l
// the path length inside layer l and n_l its scattering vertices.
// Layered media: the warp clears its path's row of `out`, then adds the
// per-layer terms atomically (a separate clearing pass cost 5 of 27 us for
// 32,768 paths of 41 vertices and 100 layers; adding runs of one layer up over
// the lanes first, or gathering the row in shared memory, measured slower).
// 12 blocks per SM: the kernel waits on its loads.
__global__ void __launch_bounds__(128, 12) score_kernel(const DMedium M, const DPair S, const float* __restrict__ xyz,
                             const int* __restrict__ nn, int batch, int cap, float* __restrict__ out,
                             int n_theta) {
  const int lane = threadIdx.x & 31;
  const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (b >= batch) return;
  float* o = out + static_cast<size_t>(b) * n_theta;
  if (M.kind != 0) {
    for (int k = lane; k < n_theta; k += 32) o[k] = 0.f;
    __syncwarp();  // orders the zeros before the other lanes' additions
  }
  const int n = nn[b];
  if (n < 2 || n > cap) {  // an invalid vertex count scores zero
    if (M.kind == 0 && lane < n_theta) o[lane] = 0.f;
    return;
  }
  const float zoff = S.zoff;
  BatchPos pos{xyz, static_cast<size_t>(batch) * cap, static_cast<size_t>(b) * cap};
  if (M.kind == 0) {
    float L = 0.f, G = 0.f;
    for (int i = lane; i < n; i += 32) {
      const float3 P = pos(i);
      if (i <= n - 2) {
        const float3 r = pos(i + 1) - P;
        L += sqrtf(dot(r, r));
      }
      if (i >= 1 && i <= n - 2) {
        const float3 a0 = P - pos(i - 1), b0 = pos(i + 1) - P;
        float g;
        phase_term(M, rsqrtf(dot(a0, a0)) * a0, rsqrtf(dot(b0, b0)) * b0, g);
        G += g;
      }
    }
    L = warp_sum(L);
    G = warp_sum(G);
    if (lane == 0) {
      o[0] = L * M.b * M.b - static_cast<float>(n - 2) * M.b;
      o[1] = L * M.a * M.a;
      o[2] = G;
    }
    return;
  }
  const int NL = M.n_layers;
  for (int i = lane; i < n; i += 32) {
    const float3 P = pos(i);
    if (i >= 1 && i <= n - 2) {
      const int l = layer_of(M, P.z + zoff);
      atomicAdd(o + l, -__ldg(M.lb + l));
    }
    if (i <= n - 2) {
      const float3 Q = pos(i + 1);
      const float3 r = Q - P;
      const float ell = sqrtf(dot(r, r));
      const float zP = P.z + zoff, zQ = Q.z + zoff;
      const int lP = layer_of(M, zP), lQ = layer_of(M, zQ);
      const int l0 = min(lP, lQ), l1 = max(lP, lQ);
      const float zlo = fminf(zP, zQ), zhi = fmaxf(zP, zQ);
#pragma unroll 1
      for (int l = l0; l <= l1; ++l) {
        float frac = 1.0f;
        if (l0 != l1) {
          const float lo = (l == l0) ? zlo : M.z0 + l * M.dz;
          const float hi = (l == l1) ? zhi : M.z0 + (l + 1) * M.dz;
          frac = fmaxf(hi - lo, 0.f) / (zhi - zlo);
        }
        const float len = ell * frac;
        const float bl = __ldg(M.lb + l), al = __ldg(M.la + l);
        atomicAdd(o + l, len * bl * bl);
        atomicAdd(o + NL + l, len * al * al);
      }
    }
  }
}

// Block-wide sum of K doubles held by every thread (blockDim.x == 256).
template <int K>
__device__ void block_sum(double (&v)[K], double* sh) {
  const int t = threadIdx.x;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    double x = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    if ((t & 31) == 0) sh[k * 8 + (t >> 5)] = x;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    double x = 0.0;
    for (int i = 0; i < 8; ++i) x += sh[k * 8 + i];
    v[k] = x;
  }
  __syncthreads();
}

// Direct-sector integral Z2 = int over the sensor seen from the source of
// eps(omega) exp(-tau) rho dOmega, with theta = theta_max (1 - v^2) to remove
// the square-root behaviour at the rim; FP32 integrand, FP64 sums.
__global__ void __launch_bounds__(256) z2_kernel(const DMedium M, const DPair* __restrict__ pairs, int n_v,
                                                 int n_phi, double* __restrict__ out) {
  __shared__ double sh[8 * 1];
  const DPair S = pairs[blockIdx.x];
  const float3 c = f3(S.c[0], S.c[1], S.c[2]);
  const float D = sqrtf(dot(c, c));
  const float3 ax = (1.0f / D) * c;
  float3 e1, e2;
  onb(ax, e1, e2);
  const float R = S.R;
  const float thmax = asinf(R / D);
  double acc = 0.0;
  const int total = n_v * n_phi;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int iv = idx / n_phi, ip = idx % n_phi;
    const float v = (iv + 0.5f) / n_v;
    const float th = thmax * (1.0f - v * v);
    const float jac = 2.0f * thmax * v / n_v;
    float st, ct, sp, cp;
    sincosf(th, &st, &ct);
    sincospif(2.0f * (ip + 0.5f) / n_phi, &sp, &cp);
    const float disc = fmaxf((R - D * st) * (R + D * st), 0.0f);
    const float r = D * ct - sqrtf(disc);
    const float3 om = ct * ax + st * (cp * e1 + sp * e2);
    const float3 h = r * om;
    float ta, tb;
    seg_tau(M, S.zoff, h.z + S.zoff, r, ta, tb);
    float lv = emission_term(S, om) - ta - tb;
    if (S.rho != 0) {
      const float3 nu = sensor_normal(S, h);
      const float x = dot(nu, f3(S.rho_hat[0], S.rho_hat[1], S.rho_hat[2]));
      lv += fmaf(3.0f, x, -1.0f) - logf(coshf(fmaf(2.0f, x, 0.7f)));
    }
    acc += static_cast<double>(expf(lv) * st * jac) * (2.0 * 3.14159265358979323846 / n_phi);
  }
  double vv[1] = {acc};
  block_sum<1>(vv, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = vv[0];
}

// Sum over the warp's lanes of each of `K` values (K a power of two, at most
// 32) by recursive halving: at every step a lane hands half of its values to
// its partner and adds the partner's copy of the other half, so that K values
// cost K - 1 + log2(32 / K) additions per lane instead of the 5 K of a
// butterfly.  Afterwards v[0] of a lane is the warp's total of the value whose
// index is the lane's top log2(K) bits.
template <int K>
__device__ __forceinline__ void warp_scatter_sum(double* v, int lane) {
  int o = 16;
#pragma unroll
  for (int m = K; m > 1; m >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < m / 2; ++k) {
      const double give = up ? v[k] : v[k + m / 2];
      const double keep = up ? v[k + m / 2] : v[k];
      v[k] = keep + __shfl_xor_sync(kFull, give, o);
    }
  }
  for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(kFull, v[0], o);
}

// Per-pair moments of the chain accumulators, first pass: one block per chunk
// of at most kMomChunk chains of one pair, one chain per thread, each chain's
// terms from add_chain_moments.  A pair of one chunk is finished here, the
// partial sums of the others go to part[chunk][MOM_USED].
//
// Bound by the FP64 pipe (about 80 FP64 operations per chain): with one block
// per pair a single pair of 65,536 chains kept one SM busy for 1,359 us; in
// chunks of 128 chains over all SMs (and 51 additions per lane for the
// block's sums instead of 180) both passes take 27 us.
__global__ void __launch_bounds__(kMomChunk) moments_kernel(const double* __restrict__ acc,
                                                            const MomChunk* __restrict__ chunks, double ls, double la,
                                                            double* __restrict__ part, double* __restrict__ out) {
  constexpr int kWarps = kMomChunk / 32;
  __shared__ double sh[kWarps][MOM_USED];
  const MomChunk C = chunks[blockIdx.x];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double v[MOM_USED];
#pragma unroll
  for (int k = 0; k < MOM_USED; ++k) v[k] = 0.0;
  if (static_cast<int>(threadIdx.x) < C.n)
    add_chain_moments(acc + static_cast<size_t>(C.first + threadIdx.x) * ACC_WORDS, ls, la, v);
  static_assert(MOM_USED == 36, "32 + 4 values");
  warp_scatter_sum<32>(v, lane);
  sh[w][lane] = v[0];
  warp_scatter_sum<4>(v + 32, lane);
  if ((lane & 7) == 0) sh[w][32 + (lane >> 3)] = v[32];
  __syncthreads();
  const int k = threadIdx.x;
  if (k >= PMC_MOMENT_WORDS) return;
  double x = 0.0;
  if (k < MOM_USED)
    for (int i = 0; i < kWarps; ++i) x += sh[i][k];
  if (C.last) out[static_cast<size_t>(C.pair) * PMC_MOMENT_WORDS + k] = x;
  else if (k < MOM_USED) part[static_cast<size_t>(blockIdx.x) * MOM_USED + k] = x;
}

// Second pass: one block per pair of several chunks, kMomGroups groups of
// threads over the pair's partial sums.
constexpr int kMomGroups = 8;
__global__ void __launch_bounds__(kMomGroups * MOM_USED) moments_total_kernel(const double* __restrict__ part,
                                                                              const MomPair* __restrict__ pairs,
                                                                              double* __restrict__ out) {
  __shared__ double sh[kMomGroups][MOM_USED];
  const MomPair C = pairs[blockIdx.x];
  const int g = threadIdx.x / MOM_USED, k = threadIdx.x % MOM_USED;
  double x = 0.0;
  for (int i = g; i < C.n; i += kMomGroups) x += part[static_cast<size_t>(C.first + i) * MOM_USED + k];
  sh[g][k] = x;
  __syncthreads();
  if (threadIdx.x >= PMC_MOMENT_WORDS) return;
  x = 0.0;
  if (threadIdx.x < MOM_USED)
    for (int i = 0; i < kMomGroups; ++i) x += sh[i][threadIdx.x];
  out[static_cast<size_t>(C.pair) * PMC_MOMENT_WORDS + threadIdx.x] = x;
}

// ---------------------------------------------------------------------------
// Forward tracer (appendix, "Ray tracer"; the photons in pmc_tracer.cuh):
// one thread per photon.
// ---------------------------------------------------------------------------
// Grid of the tracer kernels: 16 blocks per SM (3 or 4 are resident), so that
// several waves even out the ends of the blocks: 8e6 lean photons took 16.5 ms
// with 4 per SM, 15.7 with 8, 15.4 with 16; two-sensor photons 34.6, 30.8, 30.1.
static unsigned trace_grid(unsigned long long n_photons, int n_sm) {
  return static_cast<unsigned>(std::min((n_photons + 255) / 256, static_cast<unsigned long long>(n_sm) * 16ull));
}

template <bool kLean>
__global__ void __launch_bounds__(256)
    trace_kernel(const DMedium M, const DPair S, unsigned long long seed, unsigned long long photon0,
                 unsigned long long n_photons, float r_reject, int max_scatter, double* __restrict__ out5,
                 double* __restrict__ hist, double l_lo, double bins_per_m, int n_bins) {
  __shared__ double sh[8 * 5];
  const uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
  double v[5] = {0, 0, 0, 0, 0};
  unsigned int emitted = 0;
  trace_photons<kLean>(M, S, k0, k1, photon0, n_photons, r_reject, max_scatter,
                [&](unsigned long long, const PhotonResult& pr) {
                  if (++emitted == 0u) v[3] += 4294967296.0;
                  if (!pr.hit) return;
                  const double W = static_cast<double>(expf(pr.lw));
                  v[0] += W;
                  v[1] += W * W;
                  v[2] += 1.0;
                  v[4] += W * static_cast<double>(pr.L);
                  if (hist != nullptr) {
                    const double fb = (static_cast<double>(pr.L) - l_lo) * bins_per_m;
                    if (fb >= 0.0 && fb < static_cast<double>(n_bins)) atomicAdd(hist + static_cast<int>(fb), W);
                  }
                });
  v[3] += static_cast<double>(emitted);
  block_sum<5>(v, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < 5; ++k) atomicAdd(out5 + k, v[k]);
  }
}

// Detected photons thinned by their weight w rho (<= 1): an accepted path is an
// exact draw from the normalised path density (cap-truncated by max_scatter).
// Accepted paths are written to out_xyz [3][max_paths][stride] (absolute) and
// out_n; *count counts every accepted path (also those beyond max_paths).
__global__ void __launch_bounds__(256)
    trace_paths_kernel(const DMedium M, const DPair S, unsigned long long seed, unsigned long long photon0,
                       unsigned long long n_photons, float r_reject, int max_scatter, int max_paths, int stride,
                       float* __restrict__ out_xyz, int* __restrict__ out_n, unsigned int* __restrict__ count) {
  const uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
  const size_t plane = static_cast<size_t>(max_paths) * stride;
  trace_photons<false>(M, S, k0, k1, photon0, n_photons, r_reject, max_scatter,
                [&](unsigned long long ph, const PhotonResult& pr) {
                  if (!pr.hit || !(pr.u_acc < expf(pr.lw))) return;
                  const unsigned int slot = atomicAdd(count, 1u);
                  if (slot >= static_cast<unsigned int>(max_paths)) return;
                  float* ox = out_xyz + static_cast<size_t>(slot) * stride;
                  record_photon(M, S, k0, k1, ph, r_reject, max_scatter, ox, ox + plane, ox + 2 * plane);
                  out_n[slot] = pr.nsc + 2;
                });
}

// Choice of a class's kernel by its chains' vertex counts (pmc_internal.h): the last
// block to have counted its share decides and leaves the counters at zero.
constexpr int kChooseThreads = 256, kChooseBlocks = 64;
__global__ void __launch_bounds__(kChooseThreads) choose_kernel(const int* __restrict__ n,
                                                                const int* __restrict__ order, int chains,
                                                                ChoiceRule rule, ChoiceState* state,
                                                                unsigned int* queue) {
  int past[2] = {0, 0};
  for (int i = blockIdx.x * kChooseThreads + threadIdx.x; i < chains; i += gridDim.x * kChooseThreads) {
    const int k = n[order[i]];
    past[0] += k > rule.past[0];
    past[1] += k > rule.past[1];
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    past[j] = __reduce_add_sync(kFull, past[j]);
    if ((threadIdx.x & 31) == 0 && past[j] > 0) atomicAdd(&state->past[j], past[j]);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x != 0 || atomicAdd(&state->blocks, 1u) != gridDim.x - 1) return;
  __threadfence();
  const int a = atomicExch(&state->past[0], 0), b = atomicExch(&state->past[1], 0);
  state->blocks = 0u;
  state->choice = a <= rule.max_past[0] ? 0 : (b <= rule.max_past[1] ? 1 : 2);
  *queue = 0u;
}

// Per-layer scores of every chain's current path, summed per pair (layered
// media): theta = (lambda_s[l], lambda_a[l]) with d log p / d lambda_s[l] =
// len_l b_l^2 - n_l b_l and d log p / d lambda_a[l] = len_l a_l^2 (len_l: path
// length in layer l, n_l: scattering vertices in it).  One warp per chain; the
// chain's 2L scores are gathered in shared memory, then added (and squared)
// into the pair's FP64 sums.
__global__ void __launch_bounds__(128) chain_layer_score_kernel(const DMedium M, const DPair* __restrict__ pairs,
                                                                const int* __restrict__ chain_pair,
                                                                const long long* __restrict__ chain_base,
                                                                const float* __restrict__ xyz, const int* __restrict__ nn,
                                                                int total, double* __restrict__ sums) {
  extern __shared__ float sc[];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int NL = M.n_layers;
  float* s = sc + static_cast<size_t>(wib) * 2 * NL;
  const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (c >= total) return;
  for (int j = lane; j < 2 * NL; j += 32) s[j] = 0.f;
  __syncwarp();
  const int pair = chain_pair[c];
  const DPair S = pairs[pair];
  const int n = nn[c];
  const float* gx = xyz + chain_base[c];
  const float* gy = gx + S.cap;
  const float* gz = gy + S.cap;
  const float zoff = S.zoff;
  for (int i = lane; i < n; i += 32) {
    const float3 P = f3(gx[i], gy[i], gz[i]);
    if (i >= 1 && i <= n - 2) {
      const int l = layer_of(M, P.z + zoff);
      atomicAdd(s + l, -__ldg(M.lb + l));
    }
    if (i <= n - 2) {
      const float3 Q = f3(gx[i + 1], gy[i + 1], gz[i + 1]);
      const float3 r = Q - P;
      const float ell = sqrtf(dot(r, r));
      const float zP = P.z + zoff, zQ = Q.z + zoff;
      const int lP = layer_of(M, zP), lQ = layer_of(M, zQ);
      const int l0 = min(lP, lQ), l1 = max(lP, lQ);
      const float zlo = fminf(zP, zQ), zhi = fmaxf(zP, zQ);
#pragma unroll 1
      for (int l = l0; l <= l1; ++l) {
        float frac = 1.0f;
        if (l0 != l1) {
          const float lo = (l == l0) ? zlo : M.z0 + l * M.dz;
          const float hi = (l == l1) ? zhi : M.z0 + (l + 1) * M.dz;
          frac = fmaxf(hi - lo, 0.f) / (zhi - zlo);
        }
        const float len = ell * frac;
        const float bl = __ldg(M.lb + l), al = __ldg(M.la + l);
        atomicAdd(s + l, len * bl * bl);
        atomicAdd(s + NL + l, len * al * al);
      }
    }
  }
  __syncwarp();
  double* out = sums + static_cast<size_t>(pair) * 4 * NL;
  for (int j = lane; j < 2 * NL; j += 32) {
    const double v = s[j];
    if (v != 0.0) {
      atomicAdd(out + j, v);
      atomicAdd(out + 2 * NL + j, v * v);
    }
  }
}

}  // namespace

cudaError_t launch_choose(const int* n, const int* order, int chains, const ChoiceRule& rule, ChoiceState* state,
                          unsigned int* queue, cudaStream_t s) {
  const int blocks = std::min(kChooseBlocks, (chains + kChooseThreads - 1) / kChooseThreads);
  choose_kernel<<<blocks, kChooseThreads, 0, s>>>(n, order, chains, rule, state, queue);
  return cudaGetLastError();
}

cudaError_t launch_logp(const DMedium& M, const DPair& S, const float* xyz, const int* n, int batch, int cap,
                        float* out_logp, float* out_grad, int n_sm, cudaStream_t s) {
  if (batch == 0) return cudaSuccess;
  if (out_grad != nullptr) {
    logp_grad_kernel<<<(batch + 3) / 4, 128, 0, s>>>(M, S, xyz, n, batch, cap, out_logp, out_grad);
    return cudaGetLastError();
  }
  const bool few = tile_few(batch, cap, n_sm), gen = M.kind != 0 || M.f_sl > 0.f || S.emission != 0 || S.rho != 0;
  const int paths = few ? kTilePathsFew : kTilePaths;
  const auto kernel = few ? (gen ? logp_kernel<kTilePathsFew, true> : logp_kernel<kTilePathsFew, false>)
                          : (gen ? logp_kernel<kTilePaths, true> : logp_kernel<kTilePaths, false>);
  kernel<<<(batch + paths - 1) / paths, kTile, 0, s>>>(M, S, xyz, n, batch, cap, out_logp);
  return cudaGetLastError();
}

cudaError_t launch_score(const DMedium& M, const DPair& S, const float* xyz, const int* n, int batch, int cap,
                         float* out, int n_theta, const double*, const double*, cudaStream_t s) {
  if (batch == 0) return cudaSuccess;
  const int grid = (batch + 3) / 4;
  score_kernel<<<grid, 128, 0, s>>>(M, S, xyz, n, batch, cap, out, n_theta);
  return cudaGetLastError();
}

cudaError_t launch_z2(const DMedium& M, const DPair* pairs, int n_pairs, int n_v, int n_phi, double* out,
                      cudaStream_t s) {
  if (n_pairs == 0) return cudaSuccess;
  z2_kernel<<<n_pairs, 256, 0, s>>>(M, pairs, n_v, n_phi, out);
  return cudaGetLastError();
}

cudaError_t launch_moments(const double* acc, const MomChunk* chunks, int n_chunks, const MomPair* pairs, int n_pairs,
                           double ls, double la, double* part, double* out, cudaStream_t s) {
  if (n_chunks <= 0) return cudaSuccess;
  moments_kernel<<<n_chunks, kMomChunk, 0, s>>>(acc, chunks, ls, la, part, out);
  if (n_pairs > 0) moments_total_kernel<<<n_pairs, kMomGroups * MOM_USED, 0, s>>>(part, pairs, out);
  return cudaGetLastError();
}

cudaError_t launch_trace(const DMedium& M, const DPair& S, unsigned long long seed, unsigned long long photon0,
                         unsigned long long n_photons, float r_reject, int max_scatter, double* out5, int n_sm,
                         cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out5, 0, 5 * sizeof(double), s);
  if (e != cudaSuccess) return e;
  if (n_photons == 0) return cudaSuccess;
  const auto kernel = trace_lean(M, S) ? trace_kernel<true> : trace_kernel<false>;
  kernel<<<trace_grid(n_photons, n_sm), 256, 0, s>>>(M, S, seed, photon0, n_photons, r_reject,
                                                             max_scatter, out5, nullptr, 0.0, 0.0, 0);
  return cudaGetLastError();
}

cudaError_t launch_trace_lengths(const DMedium& M, const DPair& S, unsigned long long seed,
                                 unsigned long long photon0, unsigned long long n_photons, float r_reject,
                                 int max_scatter, double l_lo, double l_hi, int n_bins, double* out5, double* hist,
                                 int n_sm, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out5, 0, 5 * sizeof(double), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(hist, 0, static_cast<size_t>(n_bins) * sizeof(double), s);
  if (e != cudaSuccess) return e;
  if (n_photons == 0) return cudaSuccess;
  const auto kernel = trace_lean(M, S) ? trace_kernel<true> : trace_kernel<false>;
  kernel<<<trace_grid(n_photons, n_sm), 256, 0, s>>>(M, S, seed, photon0, n_photons, r_reject,
                                                             max_scatter, out5, hist, l_lo,
                                                             static_cast<double>(n_bins) / (l_hi - l_lo), n_bins);
  return cudaGetLastError();
}

cudaError_t launch_layer_scores(const DMedium& M, const DPair* pairs, const int* chain_pair, const long long* chain_base,
                                const float* xyz, const int* n, int total, double* sums, cudaStream_t s) {
  if (total == 0) return cudaSuccess;
  const size_t smem = 4u * 2u * static_cast<size_t>(M.n_layers) * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(chain_layer_score_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  chain_layer_score_kernel<<<(total + 3) / 4, 128, smem, s>>>(M, pairs, chain_pair, chain_base, xyz, n, total, sums);
  return cudaGetLastError();
}

// Chain seeding, first pass: the indices of the photons in [photon0,
// photon0 + n_photons) whose detection survives the thinning by w rho (the
// same test as trace_paths_kernel), in any order, into idx[0 .. cap_idx);
// *count receives how many there were (also beyond cap_idx).
template <bool kLean>
__global__ void __launch_bounds__(256)
    seed_count_kernel(const DMedium M, const DPair S, unsigned long long seed, unsigned long long photon0,
                      unsigned long long n_photons, float r_reject, int max_scatter,
                      unsigned long long* __restrict__ idx, unsigned int cap_idx, unsigned int* __restrict__ count) {
  const uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
  trace_photons<kLean>(M, S, k0, k1, photon0, n_photons, r_reject, max_scatter,
                [&](unsigned long long ph, const PhotonResult& pr) {
                  if (!pr.hit || !(pr.u_acc < expf(pr.lw))) return;
                  const unsigned int slot = atomicAdd(count, 1u);
                  if (slot < cap_idx) idx[slot] = ph;
                });
}

// Chain seeding, second pass: chain chain0 + i of pair S (i < n) takes the
// path of photon sel[i], traced again (the same photon gives the same path)
// and written straight into the chain's block in the source frame.
__global__ void __launch_bounds__(128) seed_record_kernel(const DMedium M, DPair S, unsigned long long seed,
                                                          float r_reject, const unsigned long long* __restrict__ sel,
                                                          int chain0, int n, const long long* __restrict__ chain_base,
                                                          float* __restrict__ xyz, int* __restrict__ nv,
                                                          int* __restrict__ status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int c = chain0 + i;
  S.org[0] = S.org[1] = S.org[2] = 0.f;  // record frame coordinates
  const uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
  float* gx = xyz + chain_base[c];
  const PhotonResult pr = record_photon(M, S, k0, k1, sel[i], r_reject, S.cap - 2, gx, gx + S.cap, gx + 2 * S.cap);
  nv[c] = pr.hit ? pr.nsc + 2 : 2;
  status[c] = pr.hit ? 0 : ST_BAD_N;
}

cudaError_t launch_seed_count(const DMedium& M, const DPair& S, unsigned long long seed, unsigned long long photon0,
                              unsigned long long n_photons, float r_reject, int max_scatter, unsigned long long* idx,
                              unsigned int cap_idx, unsigned int* count, int n_sm, cudaStream_t s) {
  if (n_photons == 0) return cudaSuccess;
  const auto kernel = trace_lean(M, S) ? seed_count_kernel<true> : seed_count_kernel<false>;
  kernel<<<trace_grid(n_photons, n_sm), 256, 0, s>>>(M, S, seed, photon0, n_photons, r_reject,
                                                                  max_scatter, idx, cap_idx, count);
  return cudaGetLastError();
}

cudaError_t launch_seed_record(const DMedium& M, const DPair& S, unsigned long long seed, float r_reject,
                               const unsigned long long* sel, int chain0, int n, const long long* chain_base,
                               float* xyz, int* nv, int* status, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  seed_record_kernel<<<(n + 127) / 128, 128, 0, s>>>(M, S, seed, r_reject, sel, chain0, n, chain_base, xyz, nv,
                                                     status);
  return cudaGetLastError();
}

cudaError_t launch_trace_paths(const DMedium& M, const DPair& S, unsigned long long seed, unsigned long long photon0,
                               unsigned long long n_photons, float r_reject, int max_scatter, int max_paths, int stride,
                               float* out_xyz, int* out_n, unsigned int* count, int n_sm, cudaStream_t s) {
  if (n_photons == 0) return cudaSuccess;
  trace_paths_kernel<<<trace_grid(n_photons, n_sm), 256, 0, s>>>(M, S, seed, photon0, n_photons, r_reject,
                                                                   max_scatter, max_paths, stride, out_xyz, out_n,
                                                                   count);
  return cudaGetLastError();
}

}  // namespace pmc
