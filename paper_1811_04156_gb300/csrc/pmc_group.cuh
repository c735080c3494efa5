// RJMCMC chain kernel with a group of kG = 8 lanes of a warp per chain (Collin,
// arXiv:1811.04156: section "Numerical path integration", Eq. acceptFact;
// appendix "Jump proposal" and "Dimension matching transformation"), for the general
// physics with Gaussian vertex moves.  The same Markov chains as the
// warp-per-chain kernel in pmc_chain.cu, decision for decision: the same
// Philox counters, the same factors, and every sum over a path (T_b, the choice
// of a birth's segment, the path length) taken in the order in which 32 lanes
// would take it, each lane standing in for 32 / kG of them.
//
// Why: one warp per chain issues the proposal's scalar arithmetic, the change of
// the log density (3 lanes busy) and the acceptance for 32 lanes, some 400 warp
// instructions per proposal, at 58 to 81 % of the issue slots.  With kG = 8, four
// chains share those instructions; only the O(n) parts (sums and shifts) take
// more trips per chain.  The four chains draw different kinds of moves, so a
// step runs as straight-line code with each kind's part behind a vote of the
// warp rather than as four branches in turn.  30,720 chains of 44 vertices in
// 100 layers, 500 steps: 10.3 ms with one warp per chain, 6.9 in groups (6.2
// flushing subnormals).
#pragma once

#include <type_traits>

#include "pmc_warp.cuh"

namespace pmc {
namespace PMC_VARIANT {

namespace {

// View of one chain's path: entries [0, S) live in the warp's shared memory,
// [vertex] float4 (position and vertex factor), then [segment] float2 (factor
// and length), then tau_b per segment and the optional array; entries [S, cap) in
// the chain's global block, array a at offset a * cap.  kGt: d log sigma / dg per vertex is
// cached (gradients requested).  kSpill = false: the whole cap fits (S >= cap)
// and every access goes to shared memory.
template <bool kGt, bool kSpill>
struct GroupPath {
  static constexpr int kArrays = 7 + (kGt ? 1 : 0);
  static constexpr int kX = 0, kY = 1, kZ = 2, kSeg = 3, kLen = 4, kVt = 5, kTbA = 6, kGtA = 7;
  float* sm;   // shared block
  float* gm;   // global block of the chain, stride cap
  int S, cap;
  __device__ __forceinline__ float4* va(int i) const { return reinterpret_cast<float4*>(sm) + i; }
  __device__ __forceinline__ float2* vb(int i) const { return reinterpret_cast<float2*>(sm + 4 * S) + i; }
  template <int a>
  __device__ __forceinline__ float* at(int i) const {
    if constexpr (a <= kZ) return reinterpret_cast<float*>(va(i)) + a;
    else if constexpr (a == kVt) return reinterpret_cast<float*>(va(i)) + 3;
    else if constexpr (a == kSeg || a == kLen) return reinterpret_cast<float*>(vb(i)) + (a - kSeg);
    else return sm + a * S + i;
  }
  template <int a>
  __device__ __forceinline__ float ld(int i) const {
    if (kSpill && i >= S) return gm[a * cap + i];
    return *at<a>(i);
  }
  template <int a>
  __device__ __forceinline__ void st(int i, float v) const {
    if (kSpill && i >= S) gm[a * cap + i] = v;
    else *at<a>(i) = v;
  }
  // position and vertex factor; segment factor and length
  __device__ __forceinline__ float4 vertex(int i) const {
    if (kSpill && i >= S) return make_float4(gm[kX * cap + i], gm[kY * cap + i], gm[kZ * cap + i], gm[kVt * cap + i]);
    return *va(i);
  }
  __device__ __forceinline__ void set_vertex(int i, float4 v) const {
    if (kSpill && i >= S) {
      gm[kX * cap + i] = v.x;
      gm[kY * cap + i] = v.y;
      gm[kZ * cap + i] = v.z;
      gm[kVt * cap + i] = v.w;
    } else {
      *va(i) = v;
    }
  }
  __device__ __forceinline__ float2 segment(int i) const {
    if (kSpill && i >= S) return make_float2(gm[kSeg * cap + i], gm[kLen * cap + i]);
    return *vb(i);
  }
  __device__ __forceinline__ void set_segment(int i, float2 v) const {
    if (kSpill && i >= S) {
      gm[kSeg * cap + i] = v.x;
      gm[kLen * cap + i] = v.y;
    } else {
      *vb(i) = v;
    }
  }
  __device__ __forceinline__ float3 pos(int i) const {
    if (kSpill && i >= S) return f3(gm[kX * cap + i], gm[kY * cap + i], gm[kZ * cap + i]);
    const float4 v = *va(i);
    return f3(v.x, v.y, v.z);
  }
  __device__ __forceinline__ void set_pos(int i, float3 p) const {
    st<kX>(i, p.x);
    st<kY>(i, p.y);
    st<kZ>(i, p.z);
  }
  __device__ __forceinline__ float seg(int i) const { return ld<kSeg>(i); }
  __device__ __forceinline__ float len(int i) const { return ld<kLen>(i); }
  __device__ __forceinline__ float vt(int i) const { return ld<kVt>(i); }
  __device__ __forceinline__ void set_vt(int i, float v) const { st<kVt>(i, v); }
  __device__ __forceinline__ float tb(int i) const { return ld<kTbA>(i); }
  __device__ __forceinline__ float gt(int i) const {
    if constexpr (kGt) return ld<kGtA>(i);
    else return 0.f;
  }
  __device__ __forceinline__ void set_tb(int i, float v) const { st<kTbA>(i, v); }
  __device__ __forceinline__ void set_gt(int i, float v) const {
    if constexpr (kGt) st<kGtA>(i, v);
  }
  // entry i of the arrays that move with a birth or a death
  struct Entry {
    float4 v;
    float2 s;
    float tb, gt;
  };
  __device__ __forceinline__ Entry entry(int i, bool segment_too) const {
    Entry e;
    e.v = vertex(i);
    e.gt = gt(i);
    e.s = make_float2(0.f, 0.f);
    e.tb = 0.f;
    if (segment_too) {
      e.s = segment(i);
      e.tb = tb(i);
    }
    return e;
  }
  __device__ __forceinline__ void set_entry(int i, const Entry& e, bool segment_too) const {
    set_vertex(i, e.v);
    set_gt(i, e.gt);
    if (segment_too) {
      set_segment(i, e.s);
      set_tb(i, e.tb);
    }
  }
};

constexpr int kG = kGroupLanes;

__device__ __forceinline__ float group_get(float v, int from) {
  return __shfl_sync(kFull, v, from, kG);
}

// Sum over the 32 virtual lanes of a group (virtual lane gl + kG * j holds
// part[j]) in the order of a 32-lane butterfly.
__device__ __forceinline__ float group_sum(float (&part)[32 / kG]) {
#pragma unroll
  for (int h = 32 / kG / 2; h > 0; h >>= 1)
#pragma unroll
    for (int j = 0; j < h; ++j) part[j] += part[j + h];
  float v = part[0];
#pragma unroll
  for (int o = kG / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Sum of f(i) over i < m, the terms spread over 32 virtual lanes by i mod 32.
template <class F>
__device__ __forceinline__ float group_sum_of(int m, int gl, F&& f) {
  float part[32 / kG];
#pragma unroll
  for (int j = 0; j < 32 / kG; ++j) part[j] = 0.f;
#pragma unroll 1
  for (int base = 0; base < m; base += 32) {
#pragma unroll
    for (int j = 0; j < 32 / kG; ++j) {
      const int i = base + kG * j + gl;
      if (i < m) part[j] += f(i);
    }
  }
  return group_sum(part);
}

// Segment chosen for a birth: smallest k with cumsum_k(tau_b) > u * T_b, the
// cumulative sums as 32 lanes form them: each virtual lane v (v = gl * kV + j)
// adds up m consecutive segments, then an inclusive scan over the lanes.
template <class WP>
__device__ __forceinline__ int group_select(const WP& w, int nseg, float u, float& total, int gl) {
  constexpr int kV = 32 / kG;
  const int m = (nseg + 31) >> 5;
  float own[kV], incl[kV];
#pragma unroll
  for (int j = 0; j < kV; ++j) {
    const int lo = (gl * kV + j) * m, hi = min(lo + m, nseg);
    float s = 0.f;
#pragma unroll 1
    for (int i = lo; i < hi; ++i) s += w.tb(i);
    own[j] = incl[j] = s;
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    float y[kV];
#pragma unroll
    for (int j = 0; j < kV; ++j) {
      if (o < kV) y[j] = (j >= o) ? incl[(j - o) & (kV - 1)] : __shfl_up_sync(kFull, incl[(j - o) & (kV - 1)], 1, kG);
      else y[j] = __shfl_up_sync(kFull, incl[j], o / kV, kG);
    }
#pragma unroll
    for (int j = 0; j < kV; ++j)
      if (gl * kV + j >= o) incl[j] += y[j];
  }
  total = group_get(incl[kV - 1], kG - 1);
  const float target = u * total;
  // first virtual lane past the target, else the last one that holds a segment
  int first = kV, last = -1;
#pragma unroll
  for (int j = kV - 1; j >= 0; --j) {
    const bool has = (gl * kV + j) * m < nseg;
    if (has && incl[j] > target) first = j;
    if (has && last < 0) last = j;
  }
  const int shift = (threadIdx.x & 31) - gl;
  constexpr unsigned kMask = (1u << kG) - 1u;
  const unsigned over = (__ballot_sync(kFull, first < kV) >> shift) & kMask;
  const unsigned has = (__ballot_sync(kFull, last >= 0) >> shift) & kMask;
  const int owner = over ? (__ffs(over) - 1) : (31 - __clz(has));
  int k = nseg - 1;
  if (gl == owner) {
    const int j = over ? first : last;
    float cum = 0.f;
#pragma unroll
    for (int q = 0; q < kV; ++q)
      if (q == j) cum = incl[q] - own[q];
    const int lo = (gl * kV + j) * m, hi = min(lo + m, nseg);
    k = hi - 1;
#pragma unroll 1
    for (int i = lo; i < hi; ++i) {
      cum += w.tb(i);
      if (cum > target) {
        k = i;
        break;
      }
    }
  }
  return __shfl_sync(kFull, k, owner, kG);
}

// Recording state of a chain, the same on every lane that works on it.
struct GroupAcc {
  unsigned long long pn2, pn, t_a;
  float pL, pL2, pG;
  unsigned int nflush;
  unsigned int prop_w, prop_end, prop_b, prop_d;
  unsigned int acc_i, acc_e, acc_b, acc_d;
};

// The state current since step t_a is recorded at every step in [t_a, t_b) at
// or after burn-in.
__device__ __forceinline__ void group_close(GroupAcc& a, unsigned long long t_b, unsigned long long burn_in, int n,
                                            float L, float G) {
  const unsigned long long from = a.t_a > burn_in ? a.t_a : burn_in;
  a.t_a = t_b;
  if (t_b <= from) return;
  const unsigned long long d = t_b - from;
  const float dw = static_cast<float>(d);
  a.pn2 += (n == 2) ? d : 0ull;
  a.pn += static_cast<unsigned long long>(n) * d;
  a.pL = fmaf(L, dw, a.pL);
  a.pL2 = fmaf(L * L, dw, a.pL2);
  a.pG = fmaf(G, dw, a.pG);
  a.nflush++;
}

// FP32 partials into the chain's FP64 accumulators (one lane writes).
__device__ __forceinline__ void group_flush(GroupAcc& a, double* acc, bool writes) {
  if (writes) {
    acc[ACC_NDIRECT] += static_cast<double>(a.pn2);
    acc[ACC_SUMN] += static_cast<double>(a.pn);
    acc[ACC_SUML] += static_cast<double>(a.pL);
    acc[ACC_SUML2] += static_cast<double>(a.pL2);
    acc[ACC_SUMG] += static_cast<double>(a.pG);
  }
  a.pn2 = a.pn = 0ull;
  a.pL = a.pL2 = a.pG = 0.f;
  a.nflush = 0;
}

// Words of shared memory per chain: its arrays, the staged random numbers, the
// pair constants, and a remainder that sets neighbouring chains kG banks apart.
__host__ __device__ constexpr int group_words(int arrays, int cap_s) {
  const int w = arrays * cap_s + kG * kRngWords + kPairWords;
  return w + (kG - w % 32 + 32) % 32;
}

template <bool kGrad, bool kSpill>
__global__ void __launch_bounds__(128, 4) group_chain_kernel(const ChainParams P) {
  if (P.choice != nullptr && *P.choice != P.option) return;
  using WP = GroupPath<kGrad, kSpill>;
  constexpr int kChains = 32 / kG;  // chains of a warp
  constexpr int kBatch = kG;        // steps whose random numbers are staged at once
  extern __shared__ float4 group_smem4[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int gl = lane % kG, gi = lane / kG;
  const int cap_s = P.smem_cap;
  const int words = group_words(WP::kArrays, cap_s);
  WP w;
  w.sm = reinterpret_cast<float*>(group_smem4) + static_cast<size_t>(wib * kChains + gi) * words;
  w.S = cap_s;
  uint4* rng = reinterpret_cast<uint4*>(w.sm + WP::kArrays * cap_s);  // [kBatch][2]
  DPair* spair = reinterpret_cast<DPair*>(rng + 2 * kBatch);
  const DMedium& M = P.M;
  const DRun& R = P.R;
  const uint32_t key0 = static_cast<uint32_t>(R.seed), key1 = static_cast<uint32_t>(R.seed >> 32);
  const unsigned gmask = ((1u << kG) - 1u) << (gi * kG);  // this chain's lanes

  for (;;) {
    int item = 0;
    if (lane == 0) item = static_cast<int>(atomicAdd(P.queue, 1u));
    item = __shfl_sync(kFull, item, 0);
    const long long base = static_cast<long long>(P.chain_lo) + static_cast<long long>(item) * kChains;
    if (base >= P.chain_hi) break;
    // a group past the last chain, or whose chain cannot run, follows the
    // warp's votes and shuffles on a two-vertex path of its own shared memory
    // and writes nothing else
    bool own = base + gi < P.chain_hi;
    const int c = P.order[own ? base + gi : base];
    {
      const int* src = reinterpret_cast<const int*>(P.pairs + P.chain_pair[c]);
      int* dst = reinterpret_cast<int*>(spair);
#pragma unroll 1
      for (int q = gl; q < static_cast<int>(sizeof(DPair) / sizeof(int)); q += kG) dst[q] = src[q];
      __syncwarp();
    }
    const DPair& S = *spair;
    const float zoff = S.zoff;
    const int cap = S.cap;
    const uint32_t cid = static_cast<uint32_t>(c) + P.chain_id0;  // global chain index
    int n = P.n[c];
    const unsigned long long step0 = P.step[c];
    if (n < 2 || n > cap || (!kSpill && cap > cap_s)) {
      if (own && gl == 0) {
        P.status[c] |= ST_BAD_N;
        atomicOr(P.any_status, ST_BAD_N);
      }
      own = false;
    }
    if (!own) n = 2;
    float* gx = P.xyz + P.chain_base[c];
    float* gy = gx + cap;
    float* gz = gy + cap;
    w.gm = gx;
    w.cap = cap;
    const GroupPath<kGrad, false> w_in{w.sm, w.gm, w.S, w.cap};  // the same path, all of it in the window
#pragma unroll 1
    for (int i = gl; i < min(n, cap_s); i += kG) {
      *w.va(i) = make_float4(gx[i], gy[i], gz[i], 0.f);
    }
    __syncwarp();
    // cached factors of the whole path
    bool finite = true;
#pragma unroll 1
    for (int i = gl; i < n; i += kG) {
      const float3 Pc = w.pos(i);
      const float3 Pp = (i >= 1) ? w.pos(i - 1) : Pc;
      const float3 Pn = (i <= n - 2) ? w.pos(i + 1) : Pc;
      float vt, gt, seg, tb, len;
      vertex_and_segment<true>(M, S, zoff, Pp, Pc, Pn, i, n, vt, gt, seg, tb, len);
      w.set_vt(i, vt);
      w.set_gt(i, gt);
      finite = finite && isfinite(vt);
      if (i <= n - 2) {
        w.set_segment(i, make_float2(seg, len));
        w.set_tb(i, tb);
        finite = finite && isfinite(seg);
      }
    }
    __syncwarp();
    {
      const unsigned bad = __ballot_sync(kFull, !finite);
      if (own && (bad & gmask)) {
        if (gl == 0) {
          P.status[c] |= ST_NONFINITE;
          atomicOr(P.any_status, ST_NONFINITE);
        }
        own = false;
      }
    }
    if (!__any_sync(kFull, own)) continue;
    if (!own) n = 2;
    float L = 0.f, G = 0.f;
    auto refresh_sums = [&]() {
      L = group_sum_of(n - 1, gl, [&](int i) { return w.len(i); });
      if constexpr (kGrad) G = group_sum_of(n, gl, [&](int i) { return w.gt(i); });
    };
    refresh_sums();

    GroupAcc A;
    A.pn2 = A.pn = 0;
    A.pL = A.pL2 = A.pG = 0.f;
    A.t_a = step0;
    A.nflush = 0;
    A.prop_w = A.prop_end = A.prop_b = A.prop_d = 0;
    A.acc_i = A.acc_e = A.acc_b = A.acc_d = 0;
    double* acc = P.acc + static_cast<size_t>(c) * ACC_WORDS;
    const float3 cS = f3(S.c[0], S.c[1], S.c[2]);
    unsigned long long done = 0;
    bool aborted = false;
    for (unsigned long long s0 = 0; s0 < P.n_steps; s0 += kBatch) {
      if ((s0 & 1023ull) == 0 && P.abort_flag != nullptr && __any_sync(kFull, *P.abort_flag != 0)) {
        aborted = true;
        break;
      }
      {
        // random numbers of steps step0 + s0 .. + kBatch - 1, one step per lane
        uint4 lo, hi;
        const uint32_t type = stage_step(R, S, step0 + s0 + gl, cid, key0, key1, lo, hi);
        __syncwarp();
        rng[2 * gl] = lo;
        rng[2 * gl + 1] = hi;
        __syncwarp();
        const bool live = s0 + gl < P.n_steps;
        A.prop_w += __popc(__ballot_sync(kFull, live && type == 0u) & gmask);
        A.prop_b += __popc(__ballot_sync(kFull, live && type == 2u) & gmask);
        A.prop_d += __popc(__ballot_sync(kFull, live && type == 3u) & gmask);
      }
      const int cnt = static_cast<int>(min(static_cast<unsigned long long>(kBatch), P.n_steps - s0));
      auto some = [](bool x) { return __any_sync(kFull, x); };
      // step i of the batch on the path view `w`
      auto step = [&](const auto& w, const int i) {
        using WQ = std::remove_cv_t<std::remove_reference_t<decltype(w)>>;
        const uint4 lo = rng[2 * i];
        const uint4 hi = rng[2 * i + 1];
        const uint32_t mtype = lo.x >> 24;
        const uint32_t v23 = lo.x & 0x7fffffu;
        const float logu = __uint_as_float(lo.y);
        const bool within = mtype == 0u, birth = mtype == 2u, death = mtype == 3u;
        const int jw = 1 + static_cast<int>((static_cast<unsigned long long>(v23) * (n - 1)) >> 23);
        const bool end = within && jw == n - 1;
        const bool born = birth && n < cap, dead = death && n > 2;
        const int jd = 1 + static_cast<int>((static_cast<unsigned long long>(v23) * (n - 2)) >> 23);
        // births: the segment, T_b and its share; deaths: T_b afresh
        int k = 0;
        float total = 1.f;
        if (some(born)) {
          const float ui = __fadd_rn(__uint_as_float(v23 + 0x3f800000u), -0.999999940395355224609375f);
          k = group_select(w, born ? n - 1 : 1, ui, total, gl);
        }
        // the moved vertex (within), the segment's ends (birth), the removed
        // vertex between its neighbours (death)
        const int ia = birth ? k : max(jd - 1, 0), ib = birth ? k + 1 : min(jd + 1, n - 1);
        const float3 V = w.pos(within ? jw : min(jd, n - 1));
        const float3 Af = w.pos(ia), Bf = w.pos(ib);
        float3 fnew = f3(0.f, 0.f, 0.f);
        float extra = 0.f;
        if (within) {
          const float3 z = f3(__uint_as_float(lo.z), __uint_as_float(lo.w), __uint_as_float(hi.x));
          fnew = V + R.sigma * z;
        }
        if (some(end)) {
          const float3 nu = sensor_normal(S, V);
          float3 e1, e2;
          onb(nu, e1, e2);
          const float wv = __uint_as_float(hi.y);
          const float sw = m_sqrt<true>(fmaxf(0.f, 1.0f - wv * wv));
          const float3 nn = wv * nu + sw * (__uint_as_float(hi.z) * e1 + __uint_as_float(hi.w) * e2);
          const float3 at = cS + (f3(S.c_lo[0], S.c_lo[1], S.c_lo[2]) + S.R * nn);
          if (end) fnew = at;
        }
        if (some(born)) {
          const float3 r = Bf - Af;
          const float rr = dot(r, r);
          const float irl = rsqrtf(rr);
          const float gamma = 0.5f * rr * irl;
          const float3 rh = irl * r;
          float3 xi, ze;
          onb(rh, xi, ze);
          const float beta = insertion_beta(M, R, zoff, Af, Bf, gamma);
          const float u0 = __uint_as_float(lo.z);
          float cs = -1.0f - __fdividef(__logf(fmaf(-u0, 1.0f - __expf(-2.0f * beta), 1.0f)), beta);
          cs = fminf(fmaxf(cs, -1.0f), 1.0f);
          const float sn = m_sqrt<true>(fmaxf(0.f, (1.0f - cs) * (1.0f + cs)));
          const float sc = __fdividef(gamma, __uint_as_float(hi.x) - cs);
          const float3 at = birth_point<true>(
              Af, Bf, sc, __uint_as_float(lo.w) * rh + sn * (__uint_as_float(hi.y) * xi + __uint_as_float(hi.z) * ze),
              false);
          const float tbk = w.tb(k);
          const float ex = R.log_pd - __logf(static_cast<float>(n - 1)) - R.log_pb - __logf(__fdividef(tbk, total));
          if (born) {
            fnew = at;
            extra = ex;
          }
        }
        // insertion density of a birth's new or a death's removed vertex
        float lid = 0.f;
        if (some(born || dead)) lid = log_insert_density<true>(M, R, zoff, Af, Bf, birth ? fnew : V);
        if (born) extra -= lid;

        // the changed vertex and segment factors, one slot per lane
        const bool proposed = within || born || dead;
        const int n_new = birth ? n + 1 : (death ? n - 1 : n);
        const int wlo = end ? n - 2 : (within ? jw - 1 : (birth ? k : jd - 1));
        const int nc = (end || death) ? 2 : 3, onc = (end || birth) ? 2 : 3;
        const int inew = within ? jw : (birth ? k + 1 : -1);
        const int sh_from = birth ? k + 2 : (death ? jd : 0x7fffffff), sh_by = birth ? -1 : 1;
        auto newpos = [&](int idx) -> float3 {
          int o = idx + ((idx >= sh_from) ? sh_by : 0);
          o = min(max(o, 0), n - 1);
          const float3 q = w.pos(o);
          return (idx == inew) ? fnew : q;
        };
        float nvt = 0.f, ngt = 0.f, nseg = 0.f, ntb = 0.f, nlen = 0.f;
        float ovt = 0.f, ogt = 0.f, oseg = 0.f, otb = 0.f, olen = 0.f;
        if (proposed && gl < nc) {
          const int v = wlo + gl;
          const float3 Pc = newpos(v);
          const float3 Pp = newpos(v - 1);
          const float3 Pn = newpos(v + 1);
          float seg_, tb_, len_;
          vertex_and_segment<true>(M, S, zoff, Pp, Pc, Pn, v, n_new, nvt, ngt, seg_, tb_, len_);
          if (gl < nc - 1) {
            nseg = seg_;
            ntb = tb_;
            nlen = len_;
          }
        }
        if (proposed && gl < onc) {
          const int o = wlo + gl;
          ovt = w.vt(o);
          ogt = w.gt(o);
          if (gl < onc - 1) {
            const float2 sl = w.segment(o);
            oseg = sl.x;
            olen = sl.y;
            otb = w.tb(o);
          }
        }
        __syncwarp();
        float dlp = (nvt + nseg) - (ovt + oseg);
        dlp += __shfl_xor_sync(kFull, dlp, 1);
        dlp += __shfl_xor_sync(kFull, dlp, 2);
        dlp = group_get(dlp, 0);
        if (some(dead)) {
          float dtb = ntb - otb;
          dtb += __shfl_xor_sync(kFull, dtb, 1);
          dtb += __shfl_xor_sync(kFull, dtb, 2);
          dtb = group_get(dtb, 0);
          const float tb_new = group_get(ntb, 0);
          const float Tb = group_sum_of(dead ? n - 1 : 0, gl, [&](int i) { return w.tb(i); });
          const float Tb_red = Tb + dtb;
          if (dead)
            extra = -R.log_pd + __logf(static_cast<float>(n - 2)) + R.log_pb + __logf(__fdividef(tb_new, Tb_red)) + lid;
        }
        const bool accept = own && proposed && logu < dlp + extra;
        A.prop_end += end;
        if (__any_sync(kFull, accept)) {
          // births move entries k+1 .. n-1 up by one (highest first), deaths
          // entries jd+1 .. n-1 down by one (lowest first); segment arrays only
          // below n-1
          const int a0 = birth ? k + 1 : jd + 1;
          const int most = __reduce_max_sync(kFull, accept && !within ? n - a0 : 0);
          const int d = birth ? 1 : -1;
#pragma unroll 1
          for (int q = 0; q < most; q += kG) {
            const int from = birth ? n - 1 - q - gl : a0 + q + gl;
            const bool ok = accept && !within && q + gl < n - a0;
            const bool oks = ok && from < n - 1;
            typename WQ::Entry e;
            if (ok) e = w.entry(from, oks);
            __syncwarp();
            if (ok) w.set_entry(from + d, e, oks);
            __syncwarp();
          }
          float dlen = nlen - olen;
          dlen += __shfl_xor_sync(kFull, dlen, 1);
          dlen += __shfl_xor_sync(kFull, dlen, 2);
          float dg = 0.f;
          if constexpr (kGrad) {
            dg = ngt - ogt;
            dg += __shfl_xor_sync(kFull, dg, 1);
            dg += __shfl_xor_sync(kFull, dg, 2);
          }
          if (accept && gl < nc) {
            const int v = wlo + gl;
            w.set_vt(v, nvt);
            w.set_gt(v, ngt);
            if (gl < nc - 1) {
              w.set_segment(v, make_float2(nseg, nlen));
              w.set_tb(v, ntb);
            }
          }
          if (accept && gl == 0 && !death) w.set_pos(inew, fnew);
          dlen = group_get(dlen, 0);
          if constexpr (kGrad) dg = group_get(dg, 0);
          __syncwarp();
          if (accept) {
            A.acc_i += within && !end;
            A.acc_e += end;
            A.acc_b += birth;
            A.acc_d += death;
            group_close(A, step0 + s0 + i, R.burn_in, n, L, G);
            n = n_new;
            L += dlen;
            G += dg;
            if (A.nflush >= kFlushAccepts) group_flush(A, acc, gl == 0);
          }
        }
      };
#pragma unroll 1
      for (int i = 0; i < cnt; ++i) {
        if constexpr (kSpill) {
          // paths that stay within the window even after a birth need no test at their accesses
          if (__all_sync(kFull, n < cap_s)) step(w_in, i);
          else step(w, i);
        } else {
          step(w, i);
        }
      }
      done += cnt;
      if (((s0 + kBatch) & (kRefreshSteps - 1)) == 0) refresh_sums();
    }
    // batches of 32 steps end on a refresh where the last, partial one does
    if (!aborted && (((P.n_steps + 31) & ~31ull) & (kRefreshSteps - 1)) == 0 &&
        (((P.n_steps + kBatch - 1) & ~static_cast<unsigned long long>(kBatch - 1)) & (kRefreshSteps - 1)) != 0)
      refresh_sums();
    if (own) {
      group_close(A, step0 + done, R.burn_in, n, L, G);
      group_flush(A, acc, gl == 0);
      // recorded states, proposal and acceptance counts
      const unsigned long long t_end = step0 + done;
      const unsigned long long first = step0 > R.burn_in ? step0 : R.burn_in;
#pragma unroll 1
      for (int i = gl; i < min(n, cap_s); i += kG) {
        const float4 v = *w.va(i);
        gx[i] = v.x;
        gy[i] = v.y;
        gz[i] = v.z;
      }
      if (gl == 0) {
        acc[ACC_NREC] += t_end > first ? static_cast<double>(t_end - first) : 0.0;
        acc[ACC_PROP + 0] += static_cast<double>(A.prop_w - A.prop_end);
        acc[ACC_PROP + 1] += static_cast<double>(A.prop_end);
        acc[ACC_PROP + 2] += static_cast<double>(A.prop_b);
        acc[ACC_PROP + 3] += static_cast<double>(A.prop_d);
        acc[ACC_ACC + 0] += static_cast<double>(A.acc_i);
        acc[ACC_ACC + 1] += static_cast<double>(A.acc_e);
        acc[ACC_ACC + 2] += static_cast<double>(A.acc_b);
        acc[ACC_ACC + 3] += static_cast<double>(A.acc_d);
        P.n[c] = n;
        P.step[c] = t_end;
        if (aborted) {
          P.status[c] |= ST_ABORTED;
          atomicOr(P.any_status, ST_ABORTED);
        }
      }
    }
    __syncwarp();
  }
}

// The dynamic shared-memory limit and carve-out of a kernel, once per device.
template <bool kGrad, bool kSpill>
cudaError_t group_attributes() {
  static int done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
  int optin = 0;
  e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  const auto kernel = group_chain_kernel<kGrad, kSpill>;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = 1;
  return e;
}

// Launch (blocks_per_sm == nullptr) or occupancy query of one instance.
template <bool kGrad, bool kSpill>
cudaError_t group_call(const ChainParams* p, int grid, int warps_per_block, size_t smem, int* blocks_per_sm,
                       cudaStream_t s) {
  cudaError_t e = group_attributes<kGrad, kSpill>();
  if (e != cudaSuccess) return e;
  const auto kernel = group_chain_kernel<kGrad, kSpill>;
  if (blocks_per_sm != nullptr)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, warps_per_block * 32, smem);
  kernel<<<grid, warps_per_block * 32, smem, s>>>(*p);
  return cudaGetLastError();
}

}  // namespace

}  // namespace PMC_VARIANT
}  // namespace pmc
