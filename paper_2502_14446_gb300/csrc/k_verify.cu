// Candidate verification (the distance check of Algorithm 1's inner loop).
//
// Per pair: the z-normalised Euclidean distance of Eq. (zned) in every
// dimension, computed directly from the centred windows,
//   dist_f^2 = sum_t ((x_a[t] - mu_a) / sigma_a - (x_b[t] - mu_b) / sigma_b)^2,
// then dist_d = the sum of the d smallest (Definition distdims, ties to the
// lower dimension), dims_d as a mask and dist_d^max (Eq. distdmax).  One
// warp per pair, lanes over t, in float32 (the traversal) or float64 (the
// final re-verification).
#include "internal.h"

#include <algorithm>
#include <cstdint>

namespace momenti {

namespace {

__device__ __forceinline__ float warp_sum(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <typename T>
__device__ __forceinline__ T warp_max(T v) {
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

struct VerifyOut {
  double dist_d, dist_max;
  uint64_t mask;
};

// Distances of one pair; lane f (and f - 32) ends up holding dimension f.
template <typename T>
__device__ void pair_distances(const Index& ix, uint32_t a, uint32_t b, T dist[2]) {
  const int lane = threadIdx.x & 31;
  dist[0] = dist[1] = T(0);
  for (int f = 0; f < ix.D; ++f) {
    const int64_t oa = int64_t(f) * ix.M + a, ob = int64_t(f) * ix.M + b;
    const float* xa = ix.xs_hi + int64_t(f) * ix.n + a;
    const float* xb = ix.xs_hi + int64_t(f) * ix.n + b;
    const float* la = ix.has_lo ? ix.xs_lo + int64_t(f) * ix.n + a : nullptr;
    const float* lb = ix.has_lo ? ix.xs_lo + int64_t(f) * ix.n + b : nullptr;
    T s = T(0);
    if constexpr (sizeof(T) == 4) {
      const float m0a = ix.mu_hi[oa], m1a = ix.mu_lo[oa], isa = ix.inv_sig[oa];
      const float m0b = ix.mu_hi[ob], m1b = ix.mu_lo[ob], isb = ix.inv_sig[ob];
      for (int t = lane; t < ix.w; t += 32) {
        float za = ((xa[t] - m0a) + ((la ? la[t] : 0.f) - m1a)) * isa;
        float zb = ((xb[t] - m0b) + ((lb ? lb[t] : 0.f) - m1b)) * isb;
        float dd = za - zb;
        s = fmaf(dd, dd, s);
      }
    } else {
      const double ma = ix.mu[oa], mb = ix.mu[ob];
      const double sa = ix.sig[oa], sb = ix.sig[ob];
      const bool fa = sa <= kFlatRel * (1.0 + fabs(ma)), fb = sb <= kFlatRel * (1.0 + fabs(mb));
      const double isa = fa ? 0.0 : 1.0 / sa, isb = fb ? 0.0 : 1.0 / sb;
      for (int t = lane; t < ix.w; t += 32) {
        double va = double(xa[t]) + (la ? double(la[t]) : 0.0);
        double vb = double(xb[t]) + (lb ? double(lb[t]) : 0.0);
        double dd = (va - ma) * isa - (vb - mb) * isb;
        s = fma(dd, dd, s);
      }
    }
    s = warp_sum(s);
    if (lane == (f & 31)) dist[f >> 5] = sqrt(s);
  }
}

// Sum of the d smallest of D per-lane distances (ties to the lower index).
template <typename T>
__device__ VerifyOut select_d(const T dist[2], int D, int d) {
  const int lane = threadIdx.x & 31;
  int rank[2] = {0, 0};
  for (int g = 0; g < D; ++g) {
    T vg = __shfl_sync(0xffffffffu, dist[g >> 5], g & 31);
    for (int h = 0; h < 2; ++h) {
      int f = lane + 32 * h;
      if (f < D && (vg < dist[h] || (vg == dist[h] && g < f))) ++rank[h];
    }
  }
  T sum = 0, mx = 0;
  bool sel0 = lane < D && rank[0] < d, sel1 = lane + 32 < D && rank[1] < d;
  if (sel0) { sum += dist[0]; mx = dist[0]; }
  if (sel1) { sum += dist[1]; mx = max(mx, dist[1]); }
  sum = warp_sum(sum);
  mx = warp_max(mx);
  uint64_t m0 = __ballot_sync(0xffffffffu, sel0), m1 = __ballot_sync(0xffffffffu, sel1);
  return VerifyOut{double(sum), double(mx), m0 | (m1 << 32)};
}

// Per-dimension distances of one pair in FP32 with all dims' partial sums
// kept per lane (loads of every dim in flight together), then the D warp
// reductions interleaved; lane f (and f - 32) ends with dimension f.
template <int DM>
__device__ __forceinline__ void pair_distances_fast(const Index& ix, uint32_t a, uint32_t b,
                                                    float dist[2]) {
  const int lane = threadIdx.x & 31;
  float acc[DM];
#pragma unroll
  for (int f = 0; f < DM; ++f) acc[f] = 0.f;
#pragma unroll
  for (int f = 0; f < DM; ++f) {
    if (f < ix.D) {
      const int64_t oa = int64_t(f) * ix.M + a, ob = int64_t(f) * ix.M + b;
      const float m0a = ix.mu_hi[oa], m1a = ix.mu_lo[oa], isa = ix.inv_sig[oa];
      const float m0b = ix.mu_hi[ob], m1b = ix.mu_lo[ob], isb = ix.inv_sig[ob];
      const float* xa = ix.xs_hi + int64_t(f) * ix.n + a;
      const float* xb = ix.xs_hi + int64_t(f) * ix.n + b;
      const float* la = ix.has_lo ? ix.xs_lo + int64_t(f) * ix.n + a : nullptr;
      const float* lb = ix.has_lo ? ix.xs_lo + int64_t(f) * ix.n + b : nullptr;
      float s = 0.f;
      for (int t = lane; t < ix.w; t += 32) {
        float za = ((xa[t] - m0a) + ((la ? la[t] : 0.f) - m1a)) * isa;
        float zb = ((xb[t] - m0b) + ((lb ? lb[t] : 0.f) - m1b)) * isb;
        float dd = za - zb;
        s = fmaf(dd, dd, s);
      }
      acc[f] = s;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int f = 0; f < DM; ++f) acc[f] += __shfl_xor_sync(0xffffffffu, acc[f], o);
  dist[0] = dist[1] = 0.f;
#pragma unroll
  for (int f = 0; f < DM; ++f)
    if (f < ix.D && lane == (f & 31)) dist[f >> 5] = sqrtf(acc[f]);
}

template <int DP>
__device__ __forceinline__ void load_row(const float* __restrict__ base, int64_t t, float (&v)[DP]) {
  const float4* p = reinterpret_cast<const float4*>(base + t * DP);
#pragma unroll
  for (int q = 0; q < DP / 4; ++q) {
    const float4 u = p[q];
    v[4 * q] = u.x; v[4 * q + 1] = u.y; v[4 * q + 2] = u.z; v[4 * q + 3] = u.w;
  }
}

// dist_d of a pair from per-dim distances (registers), the d smallest.
template <int DM>
__device__ __forceinline__ float sum_d_smallest(const float (&v)[DM], int D, int d) {
  float best[DM];
#pragma unroll
  for (int q = 0; q < DM; ++q) best[q] = INFINITY;
#pragma unroll
  for (int f = 0; f < DM; ++f) {
    if (f < D) {
      float x = v[f];
      // insert x into the sorted prefix best[0..d)
#pragma unroll
      for (int q = DM - 1; q >= 0; --q) {
        if (q < d) {
          float prev = q > 0 ? best[q - 1] : -INFINITY;
          if (x < best[q]) best[q] = x >= prev ? x : prev;
        }
      }
    }
  }
  float s = 0.f;
#pragma unroll
  for (int q = 0; q < DM; ++q)
    if (q < d) s += best[q];
  return s;
}

// Window statistics of window a from the point-major copy: 3 rows of DP.
template <int DP>
__device__ __forceinline__ void load_stats(const Index& ix, uint32_t a, float (&mh)[DP],
                                           float (&ml)[DP], float (&is)[DP]) {
  const float* base = ix.stT + int64_t(a) * 3 * DP;
  load_row<DP>(base, 0, mh);
  load_row<DP>(base + DP, 0, ml);
  load_row<DP>(base + 2 * DP, 0, is);
}

// Point-major form (D <= 8): each lane reads all dims of a time point of
// both windows with float4 loads.  Padding dims have 1/sigma = 0 and add 0.
template <int DP, bool LO>
__device__ __forceinline__ void pair_distances_pm(const Index& ix, uint32_t a, uint32_t b,
                                                  float dist[2]) {
  const int lane = threadIdx.x & 31;
  float m0a[DP], m1a[DP], isa[DP], m0b[DP], m1b[DP], isb[DP], acc[DP];
  load_stats<DP>(ix, a, m0a, m1a, isa);
  load_stats<DP>(ix, b, m0b, m1b, isb);
#pragma unroll
  for (int f = 0; f < DP; ++f) acc[f] = 0.f;
  const float4* pa = reinterpret_cast<const float4*>(ix.xT + int64_t(a) * DP);
  const float4* pb = reinterpret_cast<const float4*>(ix.xT + int64_t(b) * DP);
  const float4* la = LO ? reinterpret_cast<const float4*>(ix.xlT + int64_t(a) * DP) : nullptr;
  const float4* lb = LO ? reinterpret_cast<const float4*>(ix.xlT + int64_t(b) * DP) : nullptr;
  for (int t = lane; t < ix.w; t += 32) {
    float xa[DP], xb[DP], ya[DP], yb[DP];
#pragma unroll
    for (int v = 0; v < DP / 4; ++v) {
      const float4 qa = pa[int64_t(t) * (DP / 4) + v], qb = pb[int64_t(t) * (DP / 4) + v];
      xa[4 * v] = qa.x; xa[4 * v + 1] = qa.y; xa[4 * v + 2] = qa.z; xa[4 * v + 3] = qa.w;
      xb[4 * v] = qb.x; xb[4 * v + 1] = qb.y; xb[4 * v + 2] = qb.z; xb[4 * v + 3] = qb.w;
      if (LO) {
        const float4 ra = la[int64_t(t) * (DP / 4) + v], rb = lb[int64_t(t) * (DP / 4) + v];
        ya[4 * v] = ra.x; ya[4 * v + 1] = ra.y; ya[4 * v + 2] = ra.z; ya[4 * v + 3] = ra.w;
        yb[4 * v] = rb.x; yb[4 * v + 1] = rb.y; yb[4 * v + 2] = rb.z; yb[4 * v + 3] = rb.w;
      }
    }
#pragma unroll
    for (int f = 0; f < DP; ++f) {
      const float za = ((xa[f] - m0a[f]) + ((LO ? ya[f] : 0.f) - m1a[f])) * isa[f];
      const float zb = ((xb[f] - m0b[f]) + ((LO ? yb[f] : 0.f) - m1b[f])) * isb[f];
      const float dd = za - zb;
      acc[f] = fmaf(dd, dd, acc[f]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int f = 0; f < DP; ++f) acc[f] += __shfl_xor_sync(0xffffffffu, acc[f], o);
  dist[0] = dist[1] = 0.f;
#pragma unroll
  for (int f = 0; f < DP; ++f)
    if (f < ix.D && lane == f) dist[0] = sqrtf(acc[f]);
}

// Lower bound of dist_d from segment means (piecewise aggregate
// approximation): for 16-point segments of both windows,
//   sum_t (z_a - z_b)^2 >= sum_k 16 (mean_k z_a - mean_k z_b)^2
// (Cauchy-Schwarz on every segment; the points after the last full
// segment are left out, which only lowers the bound), and the sum of the d
// smallest per-dim bounds is below dist_d.  Reads w/16 rows per window.
template <int DP>
__device__ __forceinline__ float dist_d_lower_bound(const Index& ix, uint32_t a, uint32_t b, int d) {
  const int lane = threadIdx.x & 31;
  float m0a[DP], m1a[DP], isa[DP], m0b[DP], m1b[DP], isb[DP], acc[DP];
  load_stats<DP>(ix, a, m0a, m1a, isa);
  load_stats<DP>(ix, b, m0b, m1b, isb);
#pragma unroll
  for (int f = 0; f < DP; ++f) acc[f] = 0.f;
  const int segs = ix.w / 16;
  for (int k = lane; k < segs; k += 32) {
    float ua[DP], ub[DP];
    load_row<DP>(ix.smT, int64_t(a) + 16 * k, ua);
    load_row<DP>(ix.smT, int64_t(b) + 16 * k, ub);
#pragma unroll
    for (int f = 0; f < DP; ++f) {
      const float za = ((ua[f] - m0a[f]) - m1a[f]) * isa[f];
      const float zb = ((ub[f] - m0b[f]) - m1b[f]) * isb[f];
      const float dd = za - zb;
      acc[f] = fmaf(dd, dd, acc[f]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int f = 0; f < DP; ++f) acc[f] += __shfl_xor_sync(0xffffffffu, acc[f], o);
  float lb[DP];
#pragma unroll
  for (int f = 0; f < DP; ++f) lb[f] = f < ix.D ? sqrtf(16.f * acc[f]) : INFINITY;
  return sum_d_smallest<DP>(lb, ix.D, d);
}

// One warp per candidate event (each warp a contiguous range of events):
// distances; a pair with dist_d < tau is recorded (with its repetition) and
// offered to the set of close pairs.
// DM: dims held per lane (0 = any D); PM: the point-major copies (DP = DM)
template <int DM, bool PM, bool LO>
__global__ void __launch_bounds__(256)
k_verify_events(Index ix, int d, HashSet hs, const Event* __restrict__ ev,
                unsigned long long* __restrict__ counters, uint64_t ev_cap, float tau,
                PairRec* __restrict__ rec, uint64_t rec_cap) {
  const int lane = threadIdx.x & 31;
  uint64_t cnt = counters[0];
  if (cnt > ev_cap) cnt = ev_cap;
  const uint64_t nw = uint64_t(gridDim.x) * (blockDim.x >> 5);
  const uint64_t w = (blockIdx.x * uint64_t(blockDim.x) + threadIdx.x) >> 5;
  const uint64_t q0 = cnt * w / nw, q1 = cnt * (w + 1) / nw;
  for (uint64_t q = q0; q < q1; ++q) {
    const Event e = ev[q];
    if (PM && ix.smT) {
      const float lb = dist_d_lower_bound<(PM ? DM : 4)>(ix, e.a, e.b, d);
      if (lb > tau * (1.f + 1e-3f) + 1e-3f) {          // provably not below tau
        if (lane == 0) atomicAdd(&counters[3], 1ull);
        continue;
      }
    }
    float dist[2];
    if (PM) pair_distances_pm<(PM ? DM : 4), LO>(ix, e.a, e.b, dist);
    else if (DM > 0) pair_distances_fast<(DM > 0 ? DM : 1)>(ix, e.a, e.b, dist);
    else pair_distances<float>(ix, e.a, e.b, dist);
    VerifyOut v = select_d<float>(dist, ix.D, d);
    if (lane != 0) continue;
    if (!(float(v.dist_d) < tau)) {
      atomicAdd(&counters[4], 1ull);
      continue;
    }
    const unsigned long long pos = atomicAdd(&counters[1], 1ull);
    if (pos < rec_cap) {
      PairRec r;
      r.a = e.a;
      r.b = e.b;
      r.j = e.j;
      r.dist_d = float(v.dist_d);
      r.dist_max = float(v.dist_max);
      r.pad = 0;
      r.dims = v.mask;
      rec[pos] = r;
    }
    const uint64_t key = (uint64_t(e.a) << 32) | e.b;
    uint64_t h = set_hash(key) & (hs.cap - 1);
    for (int probe = 0; probe < kSetMaxProbe; ++probe) {
      uint64_t cur = hs.keys[h];
      if (cur == key) break;
      if (cur == kSetEmpty) {
        cur = atomicCAS(reinterpret_cast<unsigned long long*>(&hs.keys[h]), kSetEmpty, key);
        if (cur == kSetEmpty) {
          atomicAdd(&counters[2], 1ull);
          break;
        }
        if (cur == key) break;
      }
      h = (h + 1) & (hs.cap - 1);
    }
  }
}

__global__ void __launch_bounds__(256)
k_verify_pairs(Index ix, int d, const uint64_t* __restrict__ pairs, int64_t m, int fp64,
               double* __restrict__ per_dim, double* __restrict__ dist_d,
               uint64_t* __restrict__ dims) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = int64_t(gridDim.x) * (blockDim.x >> 5);
  for (int64_t q = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; q < m; q += nw) {
    const uint32_t a = uint32_t(pairs[q] >> 32), b = uint32_t(pairs[q]);
    VerifyOut v;
    double dd[2];
    if (fp64) {
      double dist[2];
      pair_distances<double>(ix, a, b, dist);
      v = select_d<double>(dist, ix.D, d);
      dd[0] = dist[0];
      dd[1] = dist[1];
    } else {
      float dist[2];
      pair_distances<float>(ix, a, b, dist);
      v = select_d<float>(dist, ix.D, d);
      dd[0] = dist[0];
      dd[1] = dist[1];
    }
    if (per_dim) {
      if (lane < ix.D) per_dim[q * ix.D + lane] = dd[0];
      if (lane + 32 < ix.D) per_dim[q * ix.D + lane + 32] = dd[1];
    }
    if (lane == 0) {
      if (dist_d) dist_d[q] = v.dist_d;
      if (dims) dims[q] = v.mask;
    }
  }
}

}  // namespace

cudaError_t launch_verify_events(const Index& ix, int d, const HashSet& hs,
                                 const CollideScratch& cs, float tau, PairRec* rec,
                                 uint64_t rec_cap, cudaStream_t s) {
#define MOMENTI_VE(DM, PM, LO) MOMENTI_LAUNCH("verify_events", s, k_verify_events<DM, PM, LO><<<sm_count() * 8, 256, 0, s>>>(ix, d, hs, cs.events, cs.counters, cs.ev_cap, tau, rec, rec_cap))
  const bool lo = ix.has_lo;
  if (ix.xT && ix.Dp == 4) { if (lo) MOMENTI_VE(4, true, true); else MOMENTI_VE(4, true, false); }
  else if (ix.xT && ix.Dp == 8) { if (lo) MOMENTI_VE(8, true, true); else MOMENTI_VE(8, true, false); }
  else if (ix.xT && ix.Dp == 16) { if (lo) MOMENTI_VE(16, true, true); else MOMENTI_VE(16, true, false); }
  else if (ix.D <= 16) MOMENTI_VE(16, false, false);
  else MOMENTI_VE(0, false, false);
#undef MOMENTI_VE
  return cudaGetLastError();
}

cudaError_t launch_verify_pairs(const Index& ix, int d, const uint64_t* pairs, int64_t m,
                                int fp64, double* per_dim, double* dist_d, uint64_t* dims,
                                cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  int64_t g = (m + 7) / 8;
  if (g > sm_count() * 16) g = sm_count() * 16;
  MOMENTI_LAUNCH("verify_pairs", s, k_verify_pairs<<<unsigned(g), 256, 0, s>>>(ix, d, pairs, m, fp64, per_dim, dist_d, dims));
  return cudaGetLastError();
}

// Recorded pairs whose approximate distance lies in (lo, hi], compacted.
__global__ void k_select_pairs(const uint64_t* __restrict__ pairs, const float* __restrict__ dd,
                               uint64_t m, float lo, float hscale, int b0, int b1, uint64_t* __restrict__ out,
                               unsigned long long* __restrict__ count) {
  const int lane = threadIdx.x & 31;
  for (uint64_t q0 = blockIdx.x * uint64_t(blockDim.x); q0 < m; q0 += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t q = q0 + threadIdx.x;
    const int bin = q < m ? ap_bin(dd[q], lo, hscale) : -1;
    const bool keep = bin >= b0 && bin < b1;
    const unsigned mask = __ballot_sync(0xffffffffu, keep);
    if (!mask) continue;
    unsigned long long base = 0;
    if (lane == __ffs(mask) - 1) base = atomicAdd(count, (unsigned long long)__popc(mask));
    base = __shfl_sync(0xffffffffu, base, __ffs(mask) - 1);
    if (keep) out[base + __popc(mask & ((1u << lane) - 1u))] = pairs[q];
  }
}

cudaError_t launch_select_pairs(const ApRec& rc, uint64_t m, int b0, int b1, uint64_t* out,
                                unsigned long long* count, cudaStream_t s) {
  if (m == 0) return cudaSuccess;
  uint64_t g = (m + 255) / 256;
  if (g > sm_count() * 8) g = sm_count() * 8;
  MOMENTI_LAUNCH("select_pairs", s, k_select_pairs<<<unsigned(g), 256, 0, s>>>(rc.out, rc.out_d, m, rc.lo, rc.hscale, b0, b1, out, count));
  return cudaGetLastError();
}

}  // namespace momenti
