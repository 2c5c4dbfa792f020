// The recording sweep of the exact all-pairs path (the final fallback of
// Algorithm 1): every non-trivial pair of windows whose approximate dist_d
// lies in (lo, thr] is appended to a list, with a histogram of the
// distances.  One form for every series (float32 and float64 input, 1 to
// 64 dimensions).
//
// Recurrence.  Along a diagonal b = a + delta of the distance matrix the
// centred cross product of two windows,
//   C(a, b) = sum_t (x_{a+t} - mu_a) (x_{b+t} - mu_b),
// satisfies exactly
//   C(a, b) = C(a - 1, b - 1) + df_a dg_b + dg_a df_b,
//   df_a = (x_{a+w-1} - x_{a-1}) / 2,
//   dg_a = (x_{a+w-1} - mu_a) + (x_{a-1} - mu_{a-1})
// (the mean-centred streaming update of the matrix-profile literature:
// Zimmerman et al., "Matrix Profile XIV", SoCC 2019).  df, dg and sigma
// are per-window values: they are computed once per search in float64 and
// rounded (k_sweep_table), so a pair and dimension costs two FMA for the
// recurrence and one for the threshold test, and nothing of the state
// depends on the series' level: it is C itself, in float32, restarted
// directly every `seg` rows and after every cut.  Its error per step is one rounding of C and
// of the two products; a form that slides products centred on a constant
// carries those and the centring offset's on top.
//
// Test.  dist_f <= t  <=>  corr >= c(t) = 1 - t^2 / 2w  <=>
// C >= c(t) w sigma_a sigma_b.  dist_d <= thr needs one dimension with
// dist <= thr / d (the smallest of d values is at most their mean): one FMA
// per dimension against a row factor, whose sign bits are combined over the
// 8 rows x 8 diagonals a lane runs between two branches.  A group in which
// one passed runs again with a test of all dimensions together (sw_redo).
//
// Layout.  A lane holds 2 P dimensions (P = 2, or 1: sw_pairs) of 8
// neighbouring diagonals; G = ceil(D / 2P) lanes share a diagonal (32 / G
// diagonal groups in a warp).  Per row a lane reads the row's record from
// shared memory (one address per g: a broadcast) and one new column record,
// which the 8 diagonals use in the next 8 rows: the 8 columns in flight
// live in registers, indexed statically by unrolling 8 rows.  Both sides
// then read 96 bytes per 32 pair-dimensions, a quarter of what one diagonal
// per lane reads.  Neighbouring lanes' columns are 8 windows apart, which
// in window order would put them on the same banks: the table stores blocks
// of 64 windows transposed (8 x 8), so that they are consecutive.
//
// What bounds it (D = 8, w = 300, 5e9 pairs, edge below the background):
// 7.0 ms, 4.5 pair-dimensions per cycle and scheduler of the 10.7 that three
// FMA on the FP32 lanes allow; 8 warps per SM, fixed-latency dependencies
// first.  The form before, one diagonal per lane sliding centred products,
// took 35.6 ms; at D = 32, w = 500, n = 2e5, 136 against 848 ms.
//
// Windows that C cannot resolve (flat ones, and the 7 where the series falls
// quiet: k_sweep_cuts) are marked and listed when the table is built.  The
// sweep leaves their pairs out; a kernel of its own computes them directly
// (k_sweep_marked).
#include "internal.h"

#include <algorithm>
#include <cstdint>

namespace momenti {

namespace {

constexpr int kSwThreads = 128;
constexpr int kSwWarps = kSwThreads / 32;
constexpr int kSwR = 8;                 // diagonals per lane
constexpr int kSwPad = 2048;            // records after the last window / point
constexpr int kSwSegMax = 2048;         // most rows between direct starts
constexpr int kSwAtCut = 1, kSwMarked = 2;   // bits of a window's byte

// P pairs of dims: 2 P floats of one kind, loaded with one instruction.
template <int P>
struct __align__(8 * P) SwVec {
  float2 v[P];
};

// CTAs per SM: what the registers of 8 diagonals x 2 P dims leave without
// spilling in the loop (255 and 168 registers a thread).
template <int P>
constexpr int kSwBlocks = P == 2 ? 2 : 3;

// Position of point b in its array: 8 x 8 transposed blocks.
__host__ __device__ __forceinline__ int64_t sw_pos(int64_t b) {
  return (b & ~int64_t(63)) + ((b & 7) << 3) + ((b >> 3) & 7);
}
// Offset of window b in the table, in units of G vectors: blocks of 64
// windows with their df, dg and sigma planes (64 units each) one after
// another, so that a warp's load of one kind touches whole cache lines (12
// lines a load when the three lay together: L1 was the limit).  1/sigma, which
// only the queued pairs need, follows in an array of its own, ordered by
// sw_pos.
__host__ __device__ __forceinline__ int64_t sw_off(int64_t b) {
  return (b >> 6) * 192 + ((b & 7) << 3) + ((b >> 3) & 7);
}

// Pairs of dims per lane for a series of D dims.  Two pairs read half the
// instructions per pair-dimension; one pair wastes at most one dimension
// instead of three, which pays at D = 1, 2, 5, 6 (a sweep of n = 1e5, w =
// 300: 6.3 ms at D = 5, with two pairs as at D = 8 7.0; 2.1 at D = 1, with
// two as at D = 4 4.4).
int sw_pairs(int D) { return D <= 2 || D == 5 || D == 6 ? 1 : 2; }
int64_t sw_round(int64_t m) { return ((m + 63) & ~int64_t(63)) + 64 + kSwPad; }

// Rows staged in shared memory at a time.
template <int P>
__host__ __device__ __forceinline__ int sw_rows(int G) { return G * P <= 8 ? 64 : (G * P <= 16 ? 32 : 16); }
// A warp's queue of hits: 32 plus what one row can add (8 per group of
// lanes); an entry holds C per dim, row and column in an odd number of
// 16-byte units, so that lanes reading their own entries spread over the
// banks.
__host__ __device__ __forceinline__ int sw_queue(int G) { return 32 + kSwR * (32 / G); }
template <int P>
__host__ __device__ __forceinline__ int sw_entry(int G) { return 4 * (((G * 2 * P + 2 + 3) / 4) | 1); }
template <int P>
size_t sw_smem(int G) {
  return size_t(2) * sw_rows<P>(G) * G * 3 * sizeof(SwVec<P>) +
         size_t(kSwWarps) * (size_t(2) * kSwR * 32 * sizeof(SwVec<P>) + size_t(sw_queue(G)) * sw_entry<P>(G) * 4);
}
size_t sw_smem(const SweepView& v) { return v.P == 2 ? sw_smem<2>(v.G) : sw_smem<1>(v.G); }

// Error of the recurrence.  C is a float32 running sum: what is rounded away
// in a loud stretch stays when both windows have become quiet.  Between a
// direct start and window x the rounding of C, relative to w sigma_a sigma_b,
// stays below kSwErr e_a e_b with
//   e_x^4 = sum of sigma^4 over the windows since the start / sigma_x^4
// (a rounding step is at most 2^-24 of |C| <= w sigma_a sigma_b; steps add in
// squares, and Cauchy-Schwarz parts the two windows; emulated in float32 on
// walks, noise, sinusoids, spikes and repeated stretches at w = 50 to 1000:
// at most 2.7 2^-24 e_a e_b).  Three things keep it harmless, all decided per
// window here, so that they depend on no pass and no block:
//   - sigma is stored less kappa = kSwErr (e^2 + sqrt w) of itself (the root:
//     the direct start's own error), so that a pair's correlation, and with it
//     its recorded distance, errs to the near side;
//   - where e would exceed kSwLoud (sum over at least the 2047 windows back),
//     the sum starts anew and the window is a cut: the sweep starts C again
//     after the 8-row group in which a cut falls (walks reach e = 47, even
//     noise 8: no cuts there);
//   - the rest of such a group still has the old C, so a cut and the 6 windows
//     after it are marked.  Their sigma is NaN: a test against it gives NaN,
//     whose sign bit is clear, so a group with a cut always reaches the slow
//     branch, which knows the cut by its byte and sends the warp to a new start.
// One warp per dimension and 256 windows (a warp's scan is serial: 2048 took
// 90 us); the sum starts with that of the 2048 windows before, whatever cuts
// lie there.  kappa goes where 1/sigma will lie.  With the table 0.12 ms at
// D = 8, n = 1e5 (0.05 without).
constexpr float kSwErr = 4.f / 16777216.f;
constexpr double kSwLoud = 64.0;
constexpr int kSwCutRun = 256;
template <int P>
__global__ void __launch_bounds__(128) k_sweep_cuts(Index ix, SweepView v, float* __restrict__ kap,
                                                    uint8_t* __restrict__ cut) {
  const int lane = threadIdx.x & 31, f = blockIdx.y;
  const int64_t M = ix.M, x0 = (blockIdx.x * int64_t(4) + (threadIdx.x >> 5)) * kSwCutRun;
  if (x0 >= M) return;                           // warp-uniform
  const double* sig = ix.sig + int64_t(f) * M;
  const float* isg = ix.inv_sig + int64_t(f) * M;
  auto fourth = [&](int64_t x) {                 // flat windows have no part in this: they are always computed directly
    const double s2 = isg[x] == 0.f ? 0.0 : sig[x] * sig[x];
    return s2 * s2;
  };
  double S = 0.0;                                // since the last cut
  #pragma unroll 8
  for (int64_t x = max(int64_t(0), x0 - kSwSegMax) + lane; x < x0; x += 32) S += fourth(x);
  for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
  const double limit = kSwLoud * kSwLoud * kSwLoud * kSwLoud;
  const int64_t x1 = min(M, x0 + kSwCutRun);
  for (int64_t xb = x0; xb < x1; xb += 32) {
    const int64_t x = xb + lane;
    const double q = x < x1 ? fourth(x) : 0.0;
    double part = q, run = 0.0;                  // lanes before the last cut: 0
    int from = 0;
    for (;;) {
      double p = part;
      for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, p, o);
        if (lane >= o) p += u;
      }
      if (lane >= from) run = S + p;
      const uint32_t loud = __ballot_sync(0xffffffffu, lane >= from && q > 0.0 && run > limit * q);
      if (!loud) break;
      const int c = __ffs(int(loud)) - 1;
      if (lane < 7 && xb + c + lane < M) cut[xb + c + lane] = 1;
      S = 0.0;                                   // the sum starts anew with window c
      from = c;
      if (lane < c) part = 0.0;
    }
    if (q > 0.0)
      kap[(sw_pos(x) * v.G + f / (2 * P)) * (2 * P) + f % (2 * P)] =
          kSwErr * (sqrtf(float(run / q)) + sqrtf(float(ix.w)));
    S = __shfl_sync(0xffffffffu, run, 31);
  }
}

// Table of an index: per window and group of 2 P dims {df, dg, sigma,
// 1/sigma}, each computed in float64 and rounded once; per point the values
// (and their low parts for float64 input).  A block
// builds 64 windows and points: first the marks (flat in some dim, or at a
// cut), which also go to a list, then the records.  A flat window that is not
// at a cut has a sigma no correlation reaches, as the windows past the end.
template <int P>
__global__ void __launch_bounds__(256) k_sweep_table(Index ix, SweepView v, SwVec<P>* tab, SwVec<P>* __restrict__ xp,
                                                     SwVec<P>* __restrict__ xl, uint8_t* cut,
                                                     uint32_t* __restrict__ marked) {
  __shared__ int mark[64];                       // kSwAtCut, kSwMarked
  const int64_t B = int64_t(blockIdx.x) * 64;
  const int64_t M = ix.M, n = ix.n;
  if (threadIdx.x < 64) mark[threadIdx.x] = 0;
  __syncthreads();
  for (int q = threadIdx.x; q < 64 * (ix.D + 1); q += 256) {
    const int c = q & 63, f = q >> 6;
    if (B + c >= M) continue;
    if (f == ix.D) {
      if (cut[B + c]) atomicOr(&mark[c], kSwAtCut | kSwMarked);
    } else if (ix.inv_sig[int64_t(f) * M + B + c] == 0.f) {
      atomicOr(&mark[c], kSwMarked);
    }
  }
  __syncthreads();
  if (threadIdx.x < 64 && mark[threadIdx.x]) {   // (the first 64 threads: 2 warps)
    const uint32_t act = __activemask();
    const int lane = threadIdx.x & 31, lead = __ffs(act) - 1;
    uint32_t at = 0;
    if (lane == lead) at = atomicAdd(&marked[0], uint32_t(__popc(act)));
    at = __shfl_sync(act, at, lead) + __popc(act & ((1u << lane) - 1u));
    marked[1 + at] = uint32_t(B) + threadIdx.x;
    cut[B + threadIdx.x] = uint8_t(mark[threadIdx.x]);
  }
  const int G = v.G;
  const float* kap = reinterpret_cast<const float*>(tab + 3 * v.Mpad * G);   // replaced by 1/sigma below
  for (int q = threadIdx.x; q < 64 * G; q += 256) {
    const int c = q & 63, g = q >> 6;
    const int64_t b = B + c;
    const bool in = b < M;
    SwVec<P> df, dg, sg, is, xh, xlo;
#pragma unroll
    for (int e = 0; e < 2 * P; ++e) {
      const int f = 2 * P * g + e;
      float vdf = 0.f, vdg = 0.f, vx = 0.f, vl = 0.f;
      // past the last window: a sigma no correlation reaches; no such dim: 0
      float vs = f < ix.D ? 1e30f : 0.f, vi = f < ix.D ? 1e-30f : INFINITY;
      if (f < ix.D) {
        const float* h = ix.xs_hi + int64_t(f) * n;
        const float* l = ix.has_lo ? ix.xs_lo + int64_t(f) * n : nullptr;
        auto X = [&](int64_t t) { return double(h[t]) + (l ? double(l[t]) : 0.0); };
        if (in) {
          if (b > 0) {
            const double xi = X(b + ix.w - 1), xo = X(b - 1);
            vdf = float(0.5 * (xi - xo));
            vdg = float((xi - ix.mu[int64_t(f) * M + b]) + (xo - ix.mu[int64_t(f) * M + b - 1]));
          }
          const double kappa = mark[c] ? 0.0 : double(kap[(sw_pos(b) * G + g) * (2 * P) + e]);
          const double sd = ix.sig[int64_t(f) * M + b] * (1.0 - kappa);
          if (mark[c] & kSwAtCut) vs = vi = __int_as_float(0x7fc00000);
          else if (!mark[c]) vs = float(sd), vi = float(1.0 / sd);
        }
        if (b < n) {
          vx = h[b];
          if (l) vl = l[b];
        }
      }
      float2* o[6] = {&df.v[e / 2], &dg.v[e / 2], &sg.v[e / 2], &is.v[e / 2], &xh.v[e / 2], &xlo.v[e / 2]};
      const float val[6] = {vdf, vdg, vs, vi, vx, vl};
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        if (e & 1) o[k]->y = val[k];
        else o[k]->x = val[k];
      }
    }
    const int64_t p = sw_pos(b) * G + g;
    if (b < v.Mpad) {
      SwVec<P>* t = tab + sw_off(b) * G + g;
      t[0] = df;
      t[64 * G] = dg;
      t[128 * G] = sg;
      tab[3 * v.Mpad * G + p] = is;
    }
    if (b < v.npad) {
      xp[p] = xh;
      if (xl) xl[p] = xlo;
    }
  }
}

// A pair whose approximate dist_d lies in (rc.lo, thr]: appended (with its
// approximate distance) while there is room, and counted in the histogram
// of (rc.lo, thr] either way.
__device__ __forceinline__ void sw_record(const ApRec& rc, uint32_t a, uint32_t b, float dd) {
  // one counter atomic per group of converged lanes
  const unsigned act = __activemask();
  const int lane = threadIdx.x & 31, leader = __ffs(act) - 1;
  unsigned long long base = 0;
  if (lane == leader) base = atomicAdd(rc.count, (unsigned long long)__popc(act));
  base = __shfl_sync(act, base, leader);
  const unsigned long long pos = base + __popc(act & ((1u << lane) - 1u));
  if (pos < rc.cap) {
    rc.out[pos] = (uint64_t(a) << 32) | uint64_t(b);
    rc.out_d[pos] = dd;
  }
  if (rc.hist) atomicAdd(&rc.hist[ap_bin(dd, rc.lo, rc.hscale)], 1u);
}

// Sorts N registers (a power of two) descending: bitonic network.
template <int N>
__device__ __forceinline__ void sort_desc(float (&c)[N]) {
#pragma unroll
  for (int k = 2; k <= N; k <<= 1)
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int l = i ^ j;
        if (l > i) {
          const float hi = fmaxf(c[i], c[l]), lo = fminf(c[i], c[l]);
          c[i] = (i & k) ? lo : hi;
          c[l] = (i & k) ? hi : lo;
        }
      }
}

// dist_d of one hit from its correlations: the sum of the distances of the d
// largest.  N >= D values in registers.
template <int N>
__device__ __forceinline__ float sw_dist(const float* e, int D, int d, float wf) {
  float c[N];
#pragma unroll
  for (int f = 0; f < N; ++f) c[f] = f < D ? e[f] : -INFINITY;
  sort_desc<N>(c);
  float sm = 0.f;
#pragma unroll
  for (int f = 0; f < N; ++f)
    if (f < d) sm += sqrtf(fmaxf(2.f * wf * (1.f - c[f]), 0.f));
  return sm;
}

// The joint test.  With lambda = q thr / d, dist_d <= thr gives
//   sum over the d best dims of (lambda - x_f) >= d lambda - thr,
// and lambda - x_f, as a function of the correlation y_f = 1 - x_f^2 / 2w,
// is convex above y_l = 1 - lambda^2 / 2w, where it is 0, so below its chord
// to (1, lambda).  Hence
//   sum over all dims of max(0, y_f - y_l) >= (d - d / q) (1 - y_l).
// At q = 1.5 this passes a tenth of the pairs that have one dimension
// within thr / d on the sensor workload (0.3 % against 3.3 %); for d = 1,
// where the one-dimension test is the exact one, q is near 1.
//
// Both tests are necessary conditions of the distance that is recorded: they
// give way by more than that distance's rounding (kSwSlack in the
// correlation: a few units in the last place of values up to 2, from the
// product, the square root and the sum), so that what a sweep records
// depends on the distance alone and consecutive slices leave no pair out.
constexpr float kSwSlack = 2e-6f;
struct SwJoint {
  float yl, need;
};
__device__ __forceinline__ SwJoint sw_joint(const SweepJob* jb) {
  const float q = jb->d > 1 ? 1.5f : 1.02f;
  const float lam = q * jb->thr / float(jb->d);
  SwJoint j;
  j.yl = 1.f - lam * lam / (2.f * float(jb->v.w));
  j.need = (float(jb->d) * (1.f - 1.f / q) - 1e-3f) * (1.f - j.yl) - kSwSlack * float(jb->v.D);
  return j;
}

// The queued hits of a warp, the last 32 at a time (all of them when
// `all`), one per lane: pairs that exist, are not trivial and hold no marked
// window get their distance.  Returns the number left.
template <int P>
__device__ __noinline__ int sw_drain(const SweepJob* jb, float* queue, int qn, bool all) {
  const SweepView& v = jb->v;
  const int lane = threadIdx.x & 31;
  const int D = v.D, d = jb->d, QS = sw_entry<P>(v.G);
  const float thr = jb->thr, wf = float(v.w);
  __syncwarp();
  while (qn >= 32 || (all && qn > 0)) {
    const int n = min(32, qn);
    qn -= n;
    float* e = queue + (qn + lane) * QS;
    uint32_t a = 0, b = 0;
    bool pair = false;
    if (lane < n) {
      a = __float_as_uint(e[QS - 2]);
      b = __float_as_uint(e[QS - 1]);
      pair = int64_t(b) < v.M && int64_t(b) - int64_t(a) > int64_t(v.excl) && !((v.cut[a] | v.cut[b]) & kSwMarked);
    }
    if (pair) {
      float sm = 0.f;
      if (D <= 8) sm = sw_dist<8>(e, D, d, wf);
      else if (D <= 16) sm = sw_dist<16>(e, D, d, wf);
      else {
        for (int q = 0; q < d && sm <= thr; ++q) {
          float best = -INFINITY;
          int at = 0;
          for (int f = 0; f < D; ++f) {
            const float c = e[f];
            if (c > best) {
              best = c;
              at = f;
            }
          }
          e[at] = -INFINITY;
          sm += sqrtf(fmaxf(2.f * wf * (1.f - best), 0.f));
        }
      }
      if (sm <= thr && sm > jb->rc.lo) sw_record(jb->rc, a, b, sm);
    }
    __syncwarp();
  }
  return qn;
}

template <int P>
__device__ __forceinline__ void cp_async(uint32_t dst, const void* src) {
  if constexpr (P == 2)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// Where a lane works: group g of dims of the warp's diagonal group ld.
struct SwLane {
  int g, base;
  uint32_t below, group;   // lanes of the diagonal groups before this one's, and of its own
  bool live, lead;
  int ld;
};
__device__ __forceinline__ SwLane sw_lane(int G) {
  const int lane = threadIdx.x & 31, LPW = 32 / G;
  SwLane l;
  l.g = lane % G;
  l.ld = min(lane / G, LPW - 1);
  l.base = l.ld * G;
  l.below = (1u << l.base) - 1u;
  l.group = G == 32 ? ~0u : (((1u << G) - 1u) << l.base);
  l.live = lane / G < LPW;
  l.lead = l.live && l.g == 0;
  return l;
}

// One row of the recurrence and the test for the lane's 8 diagonals (row i
// of an 8-row group, column a + i + r in slot (i + r) & 7); t[r] has the
// sign bit clear when a dim of diagonal r passes.  After diagonal 0, the
// slot of its column takes the column 8 further.
template <int P>
__device__ __forceinline__ void sw_row(float2 (&C)[kSwR][P], SwVec<P> (&df)[kSwR], SwVec<P> (&dg)[kSwR],
                                       SwVec<P> (&sg)[kSwR], const SwVec<P>& rf, const SwVec<P>& rg,
                                       const float2 (&nt)[P], int i, const SwVec<P>* pc, int G, uint32_t (&t)[kSwR]) {
#pragma unroll
  for (int r = 0; r < kSwR; ++r) {
    const int k = (i + r) & 7;
    uint32_t sb = ~0u;
#pragma unroll
    for (int p = 0; p < P; ++p) {
      C[r][p] = __ffma2_rn(rf.v[p], dg[k].v[p], C[r][p]);
      C[r][p] = __ffma2_rn(rg.v[p], df[k].v[p], C[r][p]);
      const float2 e = __ffma2_rn(nt[p], sg[k].v[p], C[r][p]);
      sb &= __float_as_uint(e.x) & __float_as_uint(e.y);
    }
    t[r] = sb;
    if (r == 0) {
      df[i] = pc[0];
      dg[i] = pc[64 * G];
      sg[i] = pc[128 * G];
    }
  }
}

// Loads the 8 columns from b0 (a multiple of 8) into the slots.
template <int P>
__device__ __forceinline__ void sw_cols(const SwVec<P>* tab, int64_t b0, int G, int g, SwVec<P> (&df)[kSwR],
                                        SwVec<P> (&dg)[kSwR], SwVec<P> (&sg)[kSwR]) {
  const SwVec<P>* p = tab + sw_off(b0) * G + g;
#pragma unroll
  for (int r = 0; r < kSwR; ++r, p += 8 * G) {
    df[r] = p[0];
    dg[r] = p[64 * G];
    sg[r] = p[128 * G];
  }
}

// Direct start: C(a, b + r) of the lane's 8 columns (a, b multiples of 8) into
// C.  The columns are centred on the first one's mean c and corrected by
// (c - mu_b) sum_t u_t, u_t = x_{a+t} - mu_a (a sum that is zero but for
// rounding).
template <int P>
__device__ __forceinline__ void sw_start(const SweepView& v, int G, int g, int64_t a, int64_t b, float2 (&C)[kSwR][P]) {
  const int D = v.D, w = v.w;
  const int64_t M = v.M;
  SwVec<P> mah, mal, cc;
#pragma unroll
  for (int e = 0; e < (2 * P); ++e) {
    const int f = (2 * P) * g + e;
    const bool in = f < D;
    const double ma = in ? v.mu[int64_t(f) * M + a] : 0.0;
    const float hi = float(ma), lo = float(ma - double(hi));
    const float c = in ? float(v.mu[int64_t(f) * M + min(b, M - 1)]) : 0.f;
    if (e & 1) { mah.v[e / 2].y = hi; mal.v[e / 2].y = lo; cc.v[e / 2].y = c; }
    else { mah.v[e / 2].x = hi; mal.v[e / 2].x = lo; cc.v[e / 2].x = c; }
  }
  const SwVec<P>* px = static_cast<const SwVec<P>*>(v.xp) + g;
  const SwVec<P>* pl = v.xl ? static_cast<const SwVec<P>*>(v.xl) + g : nullptr;
  auto value = [&](int64_t pos, const SwVec<P>& m) {
    SwVec<P> x = px[pos * G];
#pragma unroll
    for (int p = 0; p < P; ++p) x.v[p] = __fadd2_rn(x.v[p], make_float2(-m.v[p].x, -m.v[p].y));
    if (pl) {
      const SwVec<P> l = pl[pos * G];
#pragma unroll
      for (int p = 0; p < P; ++p) x.v[p] = __fadd2_rn(x.v[p], l.v[p]);
    }
    return x;
  };
  SwVec<P> col[kSwR];
  float2 su[P];
#pragma unroll
  for (int p = 0; p < P; ++p) su[p] = make_float2(0.f, 0.f);
#pragma unroll
  for (int r = 0; r < kSwR; ++r) {
#pragma unroll
    for (int p = 0; p < P; ++p) C[r][p] = make_float2(0.f, 0.f);
    col[r] = value(sw_pos(b + r), cc);
  }
  for (int t = 0; t < w; t += 8) {
    const int64_t pr = sw_pos(a + t), pc = sw_pos(b + t + 8);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      SwVec<P> u = value(pr + 8 * i, mah);
#pragma unroll
      for (int p = 0; p < P; ++p) {
        u.v[p] = __fadd2_rn(u.v[p], make_float2(-mal.v[p].x, -mal.v[p].y));
        if (t + i >= w) u.v[p] = make_float2(0.f, 0.f);
        su[p] = __fadd2_rn(su[p], u.v[p]);
      }
#pragma unroll
      for (int r = 0; r < kSwR; ++r)
#pragma unroll
        for (int p = 0; p < P; ++p) C[r][p] = __ffma2_rn(u.v[p], col[(i + r) & 7].v[p], C[r][p]);
      col[i] = value(pc + 8 * i, cc);
    }
  }
#pragma unroll
  for (int r = 0; r < kSwR; ++r) {
#pragma unroll
    for (int p = 0; p < P; ++p) {
      float dm[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int f = (2 * P) * g + 2 * p + h;
        const float c = h ? cc.v[p].y : cc.v[p].x;
        dm[h] = f < D ? float(double(c) - v.mu[int64_t(f) * M + min(b + r, M - 1)]) : 0.f;
      }
      C[r][p] = __ffma2_rn(make_float2(dm[0], dm[1]), su[p], C[r][p]);
      // a dim that does not exist: negative, against sigma 0
      if ((2 * P) * g + 2 * p >= D) C[r][p].x = -1.f;
      if ((2 * P) * g + 2 * p + 1 >= D) C[r][p].y = -1.f;
    }
  }
}

// An 8-row group in which some dim of some pair passed the first test,
// again from its start (the cross products in ck), up to its last hot row
// (bits of hot), with the joint test in the hot rows: the correlations of
// the lane's dims, their part of the sum, the sum over the
// diagonal's lanes.  Passing pairs go to the queue, one entry per pair, with
// their correlations (which depend on no threshold).
// Returns the queue's length, with kSwCut where a row or column of the group
// is at a cut.  Two rows per turn, with the columns moved
// along in registers: unrolled over all 8 rows, the code fell out of the
// instruction cache (a sweep of n = 2e4 at a
// loose threshold took 7.3 ms against 3.4).
constexpr int kSwCut = 1 << 30;
template <int P, int GT>
__device__ __noinline__ int sw_redo(const SweepJob* jb, const SwVec<P>* rows, SwVec<P>* ck, float* queue,
                                    int64_t a, int64_t b, uint32_t hot, int qn) {
  const int G = GT ? GT : jb->v.G, QS = sw_entry<P>(G), lane = threadIdx.x & 31;
  const SwLane L = sw_lane(G);
  const SwVec<P>* tab = static_cast<const SwVec<P>*>(jb->v.tab);
  const SwVec<P>* inv = tab + 3 * jb->v.Mpad * G + L.g;          // 1 / sigma
  const float wf = float(jb->v.w), iw = 1.f / wf;
  const SwJoint J = sw_joint(jb);
  const float2 nyl = make_float2(-J.yl, -J.yl);
  int top = 0;                                                   // the largest power of two below G
  for (int o = 1; o < G; o <<= 1) top = o;
  float2 C[kSwR][P];
  SwVec<P> df[kSwR + 1], dg[kSwR + 1], ib[kSwR + 1];             // columns b + i .. b + i + 8; ib: 1 / sigma
  // the test's own quotients, to two units in the last place
  auto quot = [](const SwVec<P>& s) {
    SwVec<P> o;
#pragma unroll
    for (int p = 0; p < P; ++p) o.v[p] = make_float2(__fdividef(1.f, s.v[p].x), __fdividef(1.f, s.v[p].y));
    return o;
  };
  // b is a multiple of 8: its 8 columns, and the next 8, are 8 G apart
  const SwVec<P>* pb = tab + sw_off(b) * G + L.g;
  const SwVec<P>* pn = tab + sw_off(b + 8) * G + L.g;
  auto load = [&](const SwVec<P>* p0, int slot) {
    df[slot] = p0[0];
    dg[slot] = p0[64 * G];
    ib[slot] = quot(p0[128 * G]);
  };
#pragma unroll
  for (int r = 0; r < kSwR; ++r) {
    const SwVec<P> c = ck[r * 32 + lane];
#pragma unroll
    for (int p = 0; p < P; ++p) C[r][p] = c.v[p];
    load(pb + r * 8 * G, r);
  }
#pragma unroll 1
  for (int i2 = 0; hot >> i2; i2 += 2) {
    load(pn + i2 * 8 * G, 8);
#pragma unroll
    for (int h = 0; h < 2; ++h, rows += 3 * G) {
      const int i = i2 + h;
      const SwVec<P> rf = rows[0], rg = rows[G];
#pragma unroll
      for (int r = 0; r < kSwR; ++r)
#pragma unroll
        for (int p = 0; p < P; ++p) {
          C[r][p] = __ffma2_rn(rf.v[p], dg[h + r].v[p], C[r][p]);
          C[r][p] = __ffma2_rn(rg.v[p], df[h + r].v[p], C[r][p]);
        }
      if (!((hot >> i) & 1u)) continue;
      SwVec<P> ws = rows[2 * G];
#pragma unroll
      for (int p = 0; p < P; ++p) ws.v[p] = make_float2(wf * ws.v[p].x, wf * ws.v[p].y);
      const SwVec<P> ia = quot(ws);                              // 1 / (w sigma_a)
      float sum[kSwR];
      uint32_t hit = 0;
#pragma unroll
      for (int r = 0; r < kSwR; ++r) {
        float2 part = make_float2(0.f, 0.f), y[P];
#pragma unroll
        for (int p = 0; p < P; ++p) {
          y[p] = __ffma2_rn(__fmul2_rn(C[r][p], ib[h + r].v[p]), ia.v[p], nyl);
          part = __fadd2_rn(part, make_float2(fmaxf(y[p].x, 0.f), fmaxf(y[p].y, 0.f)));
        }
        sum[r] = part.x + part.y;                                // (a window at a cut: 0, no hit)
      }
      if (G == 2) {                                              // over the diagonal's lanes
#pragma unroll
        for (int r = 0; r < kSwR; ++r) sum[r] += __shfl_xor_sync(0xffffffffu, sum[r], 1);
      } else
      // (to its first one, in a tree that takes any G)
#pragma unroll 1
      for (int o = top, len = G; o > 0; len = o, o >>= 1) {
        const bool add = L.g < o && L.g + o < len;
#pragma unroll
        for (int r = 0; r < kSwR; ++r) {
          const float u = __shfl_down_sync(0xffffffffu, sum[r], o);
          if (add) sum[r] += u;
        }
      }
#pragma unroll
      for (int r = 0; r < kSwR; ++r)
        if (!(sum[r] < J.need)) hit |= 1u << r;
      if (!L.lead) hit = 0;
      uint32_t rmask = __reduce_or_sync(0xffffffffu, hit);
      if (!rmask) continue;
      __syncwarp();
      const SwVec<P> sa = inv[sw_pos(a + i) * G];
#pragma unroll
      for (int r = 0; r < kSwR; ++r) {                           // the checkpoint has been read: room for the correlations
        SwVec<P> c = inv[sw_pos(b + i + r) * G];
#pragma unroll
        for (int p = 0; p < P; ++p)
          c.v[p] = __fmul2_rn(__fmul2_rn(C[r][p], c.v[p]), __fmul2_rn(sa.v[p], make_float2(iw, iw)));
        ck[r * 32 + lane] = c;
      }
#pragma unroll 1
      while (rmask) {
        const int r = __ffs(rmask) - 1;
        rmask &= rmask - 1u;
        const uint32_t gm = __ballot_sync(0xffffffffu, (hit >> r) & 1u);
        if (L.live && ((gm >> L.base) & 1u)) {
          float* e = queue + (qn + __popc(gm & L.below)) * QS;
          reinterpret_cast<SwVec<P>*>(e)[L.g] = ck[r * 32 + lane];
          if (L.lead) {
            e[QS - 2] = __uint_as_float(uint32_t(a + i));
            e[QS - 1] = __uint_as_float(uint32_t(b + i + r));
          }
        }
        qn += __popc(gm);
      }
      if (qn >= 32) qn = sw_drain<P>(jb, queue, qn, false);
    }
#pragma unroll
    for (int r = 0; r + 2 <= kSwR; ++r) {
      df[r] = df[r + 2];
      dg[r] = dg[r + 2];
      ib[r] = ib[r + 2];
    }
    load(pn + (i2 + 1) * 8 * G, 7);
  }
  const unsigned long long* cuts = reinterpret_cast<const unsigned long long*>(jb->v.cut);
  if (__any_sync(0xffffffffu, ((cuts[a >> 3] | cuts[b >> 3] | cuts[(b >> 3) + 1]) & (kSwAtCut * 0x0101010101010101ull)) != 0ull))
    qn |= kSwCut;
  return qn;
}

// One block of the sweep: row windows [bx seg, bx seg + seg), the
// diagonals of row `by` of the grid (kSwWarps * (32 / G) * 8 of them, from
// a multiple of 8 at or below eps + 1).
template <int P, int GT>
__device__ __forceinline__ void sw_block(const SweepJob* jb, int64_t bx, int64_t by) {
  extern __shared__ __align__(16) unsigned char sw_mem[];
  const SweepView& v = jb->v;
  const int G = GT ? GT : v.G, w = v.w;
  const int64_t M = v.M;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int LPW = 32 / G;
  const SwLane L = sw_lane(G);
  const int g = L.g;
  const int a0 = int(bx * jb->seg);    // rows and columns in 32 bits (fewer than 2^27 windows): 7.0 ms against 7.4 at D = 8, n = 1e5
  const int64_t dlo = ((int64_t(v.excl) + 1) & ~int64_t(7)) + by * (kSwWarps * LPW * kSwR);
  const int64_t dfirst = max(dlo, int64_t(v.excl) + 1);          // the block's first diagonal
  if (dfirst >= M || a0 >= M - dfirst) return;                   // block-uniform
  const int nrow = int(min(int64_t(jb->seg), M - dfirst - a0));
  const int b0 = int(a0 + dlo) + (warp * LPW + L.ld) * kSwR;     // this lane's first column, a multiple of 8
  const int RS = sw_rows<P>(G);
  SwVec<P>* rows = reinterpret_cast<SwVec<P>*>(sw_mem);                // [2][RS][3][G]
  SwVec<P>* ck = rows + 2 * RS * G * 3 + warp * (2 * kSwR * 32); // [warps][2][8][32]: C at an 8-row group's start
  float* queue = reinterpret_cast<float*>(rows + 2 * RS * G * 3 + kSwWarps * 2 * kSwR * 32) +
                 warp * sw_queue(G) * sw_entry<P>(G);
  const SwVec<P>* __restrict__ tab = static_cast<const SwVec<P>*>(v.tab);
  auto stage = [&](int s) {                                      // rows [s RS, s RS + RS) of the block
    const int rn = min(RS, ((nrow + 7) & ~7) - s * RS);
    const uint32_t dst = uint32_t(__cvta_generic_to_shared(rows + (s & 1) * RS * G * 3));
    for (int q = threadIdx.x; q < rn * G * 3; q += kSwThreads) {
      const int r = q / (3 * G), c = q - r * 3 * G;
      const int k = c / G;                                       // plane, then group
      cp_async<P>(dst + uint32_t(q) * uint32_t(sizeof(SwVec<P>)),
                  tab + (sw_off(a0 + s * RS + r) + 64 * k) * G + (c - k * G));
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  __syncthreads();                  // a previous block of this CTA is done with the row buffers
  stage(0);

  // ---- the state: C, the columns in flight
  float2 C[kSwR][P];
  const int cstep = 8 * G;                                       // vectors between the columns of an 8-row group
  SwVec<P> df[kSwR], dg[kSwR], sg[kSwR];
  const float t1 = jb->thr / float(jb->d);
  const float nk = -(1.f - t1 * t1 / (2.f * float(w)) - kSwSlack) * float(w);
  const float2 nk2 = make_float2(nk, nk);
  int qn = 0, cb = 0, redone = 0;   // queued hits, this group's checkpoint, groups run twice
  int ro = 0;                       // the group's first row
start:
  // C started anew for the group at row ro, and its columns: back by one row
  // from the direct value, which the group's first row then takes again; into
  // the group's checkpoint.  The slow branch comes back here after a cut: a
  // flag asked for at the head of every group, or a second copy of the start
  // in the branch, cost the loop registers (7.6 ms against 7.2 at D = 8,
  // n = 1e5; 24.6 against 23.4 at D = 64, n = 6e4)
  {
    sw_start<P>(v, G, g, a0 + ro, b0 + ro, C);
    sw_cols<P>(tab, b0 + ro, G, g, df, dg, sg);
    const SwVec<P>* ra = tab + sw_off(a0 + ro) * G + g;
    const SwVec<P> rf = ra[0], rg = ra[64 * G];
#pragma unroll
    for (int r = 0; r < kSwR; ++r) {
      SwVec<P> c;
#pragma unroll
      for (int p = 0; p < P; ++p) {
        C[r][p] = __ffma2_rn(make_float2(-rg.v[p].x, -rg.v[p].y), df[r].v[p], C[r][p]);
        C[r][p] = __ffma2_rn(make_float2(-rf.v[p].x, -rf.v[p].y), dg[r].v[p], C[r][p]);
        c.v[p] = C[r][p];
      }
      ck[cb + r * 32 + lane] = c;
    }
  }
  while (ro < nrow) {
    if ((ro & (RS - 1)) == 0) {     // (RS: a power of two)
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();              // this stage's rows are here, the other buffer is free
      if (ro + RS < nrow) stage(ro / RS + 1);
    }
    const int rend = min((ro | (RS - 1)) + 1, (nrow + 7) & ~7);   // of the stage
    const SwVec<P>* rp = rows + (ro & (2 * RS - 1)) * G * 3 + g;
    SwVec<P> nf = rp[0], ng = rp[G], ns = rp[2 * G];                    // the next row's record
    // 8 rows at a time without a branch: the tests' sign bits of all their
    // pairs are combined, and a group in which one passed runs once more
    // from its start (a branch after every row, with what it kept from
    // overlapping, took 185 ms on the wide workload against 145)
    for (; ro < rend; ro += 8) {
      const SwVec<P>* pc = tab + sw_off(b0 + ro + 8) * G + g;
      const SwVec<P>* r8 = rp;
      uint32_t quiet = ~0u;                                      // bit 7 - i: no dim of row i's pairs passed
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const SwVec<P> rf = nf, rg = ng;
        float2 nt[P];
#pragma unroll
        for (int p = 0; p < P; ++p) nt[p] = __fmul2_rn(ns.v[p], nk2);
        if (i < 7 || ro + 8 < rend) rp += G * 3;                 // (the last row of the stage is read again)
        nf = rp[0];
        ng = rp[G];
        ns = rp[2 * G];
        uint32_t t[kSwR];
        sw_row<P>(C, df, dg, sg, rf, rg, nt, i, pc, G, t);
        pc += cstep;
        const uint32_t all = ((t[0] & t[1] & t[2]) & (t[3] & t[4])) & ((t[5] & t[6]) & t[7]);
        quiet = __funnelshift_l(all, quiet, 1);
      }
      cb ^= kSwR * 32;
#pragma unroll
      for (int r = 0; r < kSwR; ++r) {                           // C at the next group's start
        SwVec<P> c;
#pragma unroll
        for (int p = 0; p < P; ++p) c.v[p] = C[r][p];
        ck[cb + r * 32 + lane] = c;
      }
      if (__any_sync(0xffffffffu, quiet != ~0u)) {
        ++redone;
        const uint32_t hot = __brev(__reduce_or_sync(0xffffffffu, ~quiet)) >> 24;   // bit i: row i
        qn = sw_redo<P, GT>(jb, r8, ck + (cb ^ (kSwR * 32)), queue, a0 + ro, b0 + ro, hot, qn);
        if (qn >= kSwCut && ro + 8 < nrow) {                     // a cut in the group, warp-uniform
          qn &= kSwCut - 1;
          ro += 8;
          goto start;
        }
        qn &= kSwCut - 1;
        // the state again from memory, so that none of it lives across the call
#pragma unroll
        for (int r = 0; r < kSwR; ++r) {
          const SwVec<P> c = ck[cb + r * 32 + lane];
#pragma unroll
          for (int p = 0; p < P; ++p) C[r][p] = c.v[p];
        }
        sw_cols<P>(tab, b0 + ro + 8, G, g, df, dg, sg);
        nf = rp[0];
        ng = rp[G];
        ns = rp[2 * G];
      }
    }
  }
  sw_drain<P>(jb, queue, qn, true);
  if (jb->groups && lane == 0) {
    atomicAdd(&jb->groups[0], (unsigned long long)((nrow + 7) / 8));
    atomicAdd(&jb->groups[1], (unsigned long long)redone);
  }
}

template <int P, int GT>
__global__ void __launch_bounds__(kSwThreads, kSwBlocks<P>)
k_sweep(const __grid_constant__ SweepJob jb, int64_t ybase) {
  sw_block<P, GT>(&jb, int64_t(blockIdx.x), ybase + int64_t(blockIdx.y));
}

// Every stride-th block of the sweep's grid, at a varying offset.
__host__ __device__ __forceinline__ int64_t sw_sampled(int64_t q, int64_t stride) {
  return q * stride + int64_t((uint64_t(q) * 2654435761ull) % uint64_t(stride));
}
template <int P>
__global__ void __launch_bounds__(kSwThreads, kSwBlocks<P>)
k_sweep_sample(const __grid_constant__ SweepJob jb, int64_t nbx, int64_t stride) {
  const int64_t q = sw_sampled(int64_t(blockIdx.x), stride);
  sw_block<P, 0>(&jb, q % nbx, q / nbx);
}

// The sweeps of several series in one persistent launch: each CTA takes
// (series, row block, diagonal block) items from a device queue in order
// (largest series first) until the queue is empty; an item is one block of
// the sweep above on that series' index, threshold and record buffers.
template <int P>
__global__ void __launch_bounds__(kSwThreads, kSwBlocks<P>)
k_sweep_batch(const SweepJob* __restrict__ jobs, const SweepItem* __restrict__ items, int nitems,
              int* __restrict__ next) {
  __shared__ int cur;
  for (;;) {
    __syncthreads();                // every thread has read the previous item
    if (threadIdx.x == 0) cur = atomicAdd(next, 1);
    __syncthreads();
    const int it = cur;
    if (it >= nitems) return;       // block-uniform
    const SweepItem q = items[it];
    sw_block<P, 0>(jobs + q.job, int64_t(q.bx), int64_t(q.by));
  }
}

// The pairs with a marked window: a marked window against 256 others per
// turn, a pair per thread, point by point as the verification does (a pair of
// two marked windows from the first).  Distances err to the near side by
// 1e-5.  Bound by the FP32 lanes: about 8 operations per point and dim.  With
// 2% of the windows of n = 3e4, D = 8 flat, an exact search takes 36 ms; 2.9 s
// when a warp computed such a pair in the sweep's own queue, 2.4 s when they
// were candidates at distance 0 (with 30% flat 0.30 s, 8.4 and 42).
template <int P>
__global__ void __launch_bounds__(256) k_sweep_marked(const __grid_constant__ SweepJob jb) {
  extern __shared__ __align__(16) unsigned char sw_mem[];
  float* dist = reinterpret_cast<float*>(sw_mem) + threadIdx.x;  // [D][256]
  const SweepView& v = jb.v;
  const uint32_t n = v.marked[0];
  const int64_t M = v.M, ny = (M + 255) / 256, items = int64_t(n) * ny;
  const int G = v.G, D = v.D, w = v.w;
  const SwVec<P>* px = static_cast<const SwVec<P>*>(v.xp);
  const SwVec<P>* pl = static_cast<const SwVec<P>*>(v.xl);
  for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const int64_t x = v.marked[1 + it / ny], y = (it % ny) * 256 + threadIdx.x;
    const int64_t a = min(x, y), b = max(x, y);
    if (y >= M || b - a <= int64_t(v.excl) || (y < x && (v.cut[y] & kSwMarked))) continue;
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
      float2 ma[P], la[P], ia[P], mb[P], lb[P], ib[P], acc[P];
      auto stats = [&](int64_t q, float2 (&hi)[P], float2 (&lo)[P], float2 (&is)[P]) {
#pragma unroll
        for (int k = 0; k < 2 * P; ++k) {
          const int f = 2 * P * g + k;
          const int64_t o = int64_t(f) * M + q;
          const double m = f < D ? v.mu[o] : 0.0, sd = f < D ? v.sig[o] : 0.0;
          const float h = float(m), l = float(m - double(h));
          const float r = sd <= kFlatRel * (1.0 + fabs(m)) ? 0.f : float(1.0 / sd);   // flat: the zero vector
          if (k & 1) hi[k / 2].y = -h, lo[k / 2].y = -l, is[k / 2].y = r;
          else hi[k / 2].x = -h, lo[k / 2].x = -l, is[k / 2].x = r;
        }
      };
      stats(a, ma, la, ia);
      stats(b, mb, lb, ib);
#pragma unroll
      for (int p = 0; p < P; ++p) acc[p] = make_float2(0.f, 0.f);
#pragma unroll 4
      for (int t = 0; t < w; ++t) {
        const int64_t pa = sw_pos(a + t) * G + g, pb = sw_pos(b + t) * G + g;
        const SwVec<P> xa = px[pa], xb = px[pb];
#pragma unroll
        for (int p = 0; p < P; ++p) {
          const float2 ua = pl ? __fadd2_rn(pl[pa].v[p], la[p]) : la[p], ub = pl ? __fadd2_rn(pl[pb].v[p], lb[p]) : lb[p];
          const float2 za = __fmul2_rn(__fadd2_rn(__fadd2_rn(xa.v[p], ma[p]), ua), ia[p]);
          const float2 zb = __fmul2_rn(__fadd2_rn(__fadd2_rn(xb.v[p], mb[p]), ub), ib[p]);
          const float2 d = __fadd2_rn(za, make_float2(-zb.x, -zb.y));
          acc[p] = __ffma2_rn(d, d, acc[p]);
        }
      }
#pragma unroll
      for (int k = 0; k < 2 * P; ++k) {
        const int f = 2 * P * g + k;
        if (f < D) dist[256 * f] = sqrtf((k & 1) ? acc[k / 2].y : acc[k / 2].x) * 0.99999f;
      }
    }
    float sm = 0.f;                                              // the d smallest
    for (int q = 0; q < jb.d && sm <= jb.thr; ++q) {
      float best = INFINITY;
      int at = 0;
      for (int f = 0; f < D; ++f) {
        const float c = dist[256 * f];
        if (c < best) {
          best = c;
          at = f;
        }
      }
      dist[256 * at] = INFINITY;
      sm += best;
    }
    if (sm <= jb.thr && sm > jb.rc.lo) sw_record(jb.rc, uint32_t(a), uint32_t(b), sm);
  }
}

int64_t sw_diags(int G) { return int64_t(kSwWarps) * (32 / G) * kSwR; }   // per block

// Diagonal blocks of the whole sweep (0: no non-trivial pair).
int64_t sw_gy(const SweepView& v) {
  const int64_t first = int64_t(v.excl) + 1;
  if (first >= v.M) return 0;
  const int64_t lo = first & ~int64_t(7), nd = sw_diags(v.G);
  return (v.M - lo + nd - 1) / nd;
}

// Rows per block.  A block pays a direct start of w points (about 22
// issue slots each) before its rows (about 78 each); a launch runs two or
// three blocks per SM at a time.  Long blocks where there are many of them,
// shorter ones where waves would be partly empty.  At most 2048: the error of
// C grows with the root of the rows (blocks of 4096 took 128 ms where this
// takes 136, n = 2e5, D = 32, w = 500, at 1.4 times the error).
int sw_seg(const SweepView& v) {
  const int64_t slots = int64_t(sm_count()) * (v.P == 2 ? kSwBlocks<2> : kSwBlocks<1>), nd = sw_diags(v.G), gy = sw_gy(v);
  int best = kSwSegMax;
  double best_cost = 1e300;
  for (int seg = kSwSegMax; seg >= 32; seg >>= 1) {
    int64_t blocks = 0;
    for (int64_t by = 0; by < gy; ++by) {
      const int64_t d0 = ((int64_t(v.excl) + 1) & ~int64_t(7)) + by * nd;
      blocks += std::max<int64_t>(0, (v.M - d0 + seg - 1) / seg);
    }
    const double waves = std::max(1.0, double(blocks) / double(slots));
    const double cost = (waves > 16.0 ? waves : std::ceil(waves)) * (22.0 * v.w + 78.0 * seg);
    if (cost < best_cost) {
      best_cost = cost;
      best = seg;
    }
  }
  return best;
}

}  // namespace

size_t sweep_table_bytes(const Index& ix) {
  const int P = sw_pairs(ix.D);
  const size_t G = size_t((ix.D + 2 * P - 1) / (2 * P));
  return (size_t(sw_round(ix.M)) * 4 + size_t(sw_round(ix.n)) * (ix.has_lo ? 2 : 1)) * G * (8 * size_t(P)) +
         size_t(sw_round(ix.M)) * 5 + 16;
}

template <int P>
static cudaError_t sweep_table(const Index& ix, SweepView& v, void* buf, cudaStream_t s) {
  SwVec<P>* tab = static_cast<SwVec<P>*>(buf);
  SwVec<P>* xp = tab + v.Mpad * v.G * 4;
  SwVec<P>* xl = ix.has_lo ? xp + v.npad * v.G : nullptr;
  v.tab = tab;
  v.xp = xp;
  v.xl = xl;
  uint8_t* cut = reinterpret_cast<uint8_t*>(xp + v.npad * v.G * (ix.has_lo ? 2 : 1));
  v.cut = cut;
  uint32_t* marked = reinterpret_cast<uint32_t*>(cut + v.Mpad);      // (Mpad: a multiple of 64)
  v.marked = marked;
  const cudaError_t e = cudaMemsetAsync(cut, 0, size_t(v.Mpad) + 4, s);
  if (e != cudaSuccess) return e;
  const dim3 gc{unsigned((ix.M + 4 * kSwCutRun - 1) / (4 * kSwCutRun)), unsigned(ix.D), 1u};
  MOMENTI_LAUNCH("sweep_cuts", s, k_sweep_cuts<P><<<gc, 128, 0, s>>>(ix, v, reinterpret_cast<float*>(tab + v.Mpad * v.G * 3), cut));
  MOMENTI_LAUNCH("sweep_table", s, k_sweep_table<P><<<unsigned(v.npad / 64), 256, 0, s>>>(ix, v, tab, xp, xl, cut, marked));
  return cudaGetLastError();
}

cudaError_t launch_sweep_table(const Index& ix, void* buf, SweepView* out, cudaStream_t s) {
  SweepView v;
  v.M = ix.M;
  v.Mpad = sw_round(ix.M);
  v.npad = sw_round(ix.n);
  v.D = ix.D;
  v.P = sw_pairs(ix.D);
  v.G = (ix.D + 2 * v.P - 1) / (2 * v.P);
  v.w = ix.w;
  v.excl = ix.excl;
  v.mu = ix.mu;
  v.sig = ix.sig;
  const cudaError_t e = v.P == 2 ? sweep_table<2>(ix, v, buf, s) : sweep_table<1>(ix, v, buf, s);
  *out = v;
  return e;
}

template <int P>
static cudaError_t sweep_marked(const SweepJob& jb, cudaStream_t s) {
  const size_t smem = size_t(jb.v.D) * 256 * sizeof(float);
  const cudaError_t e = allow_smem(reinterpret_cast<const void*>(k_sweep_marked<P>), smem);
  if (e != cudaSuccess) return e;
  // (as many blocks as stay resident; they find the marked windows' number on the device)
  MOMENTI_LAUNCH("sweep_marked", s, k_sweep_marked<P><<<unsigned(sm_count() * 3), 256, smem, s>>>(jb));
  return cudaGetLastError();
}

template <int P, int GT>
static cudaError_t sweep(const SweepJob& jb, int64_t gy, cudaStream_t s) {
  const size_t smem = sw_smem<P>(jb.v.G);
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(k_sweep<P, GT>), smem);
  if (e != cudaSuccess) return e;
  for (int64_t y0 = 0; y0 < gy; y0 += 65535) {
    dim3 grid{unsigned((jb.v.M + jb.seg - 1) / jb.seg), unsigned(std::min<int64_t>(65535, gy - y0)), 1u};
    MOMENTI_LAUNCH("allpairs", s, k_sweep<P, GT><<<grid, kSwThreads, smem, s>>>(jb, y0));
  }
  return cudaGetLastError();
}

cudaError_t launch_allpairs(const SweepView& v, int d, float thr, const ApRec& rc, cudaStream_t s) {
  const int64_t gy = sw_gy(v);
  if (gy <= 0) return cudaSuccess;
  SweepJob jb;
  jb.v = v;
  jb.rc = rc;
  jb.thr = thr;
  jb.d = d;
  jb.seg = sw_seg(v);
  // offsets of the lanes' groups as constants where D is common (n = 1e5, w =
  // 300: 6.3 ms against 8.3 at D = 5, 14.0 against 16.8 at D = 16, 30.3 against
  // 36.2 at D = 32); D = 25 to 28 (36.3 at 27) and 33 to 60 take the runtime form
  cudaError_t e = cudaSuccess;
  if (v.P == 1) e = v.G == 1 ? sweep<1, 1>(jb, gy, s) : sweep<1, 3>(jb, gy, s);
  else switch (v.G) {
    case 1: e = sweep<2, 1>(jb, gy, s); break;
    case 2: e = sweep<2, 2>(jb, gy, s); break;
    case 3: e = sweep<2, 3>(jb, gy, s); break;
    case 4: e = sweep<2, 4>(jb, gy, s); break;
    case 5: e = sweep<2, 5>(jb, gy, s); break;
    case 6: e = sweep<2, 6>(jb, gy, s); break;
    case 8: e = sweep<2, 8>(jb, gy, s); break;
    case 16: e = sweep<2, 16>(jb, gy, s); break;
    default: e = sweep<2, 0>(jb, gy, s);
  }
  if (e != cudaSuccess) return e;
  return v.P == 2 ? sweep_marked<2>(jb, s) : sweep_marked<1>(jb, s);
}

template <int P>
static cudaError_t sweep_sample(const SweepJob& jb, int64_t nbx, int64_t blocks, int64_t stride, cudaStream_t s) {
  const size_t smem = sw_smem<P>(jb.v.G);
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(k_sweep_sample<P>), smem);
  if (e != cudaSuccess) return e;
  MOMENTI_LAUNCH("allpairs_sample", s, k_sweep_sample<P><<<unsigned(blocks), kSwThreads, smem, s>>>(jb, nbx, stride));
  return cudaGetLastError();
}

cudaError_t launch_allpairs_sample(const SweepView& v, int d, float thr, const ApRec& rc, double fraction,
                                   int seg, double* pairs, unsigned long long* groups, cudaStream_t s) {
  *pairs = 0.0;
  const int64_t gy = sw_gy(v), nd = sw_diags(v.G);
  if (gy <= 0) return cudaSuccess;
  SweepJob jb;
  jb.v = v;
  jb.rc = rc;
  jb.thr = thr;
  jb.d = d;
  jb.seg = seg;
  jb.groups = groups;
  const int64_t nbx = (v.M + seg - 1) / seg, total = nbx * gy;
  const int64_t stride = std::max<int64_t>(1, std::min<int64_t>(int64_t(1.0 / fraction), total));
  const int64_t blocks = std::min<int64_t>((total + stride - 1) / stride, int64_t(1) << 30);
  // pairs the sampled blocks hold
  for (int64_t q = 0; q < blocks; ++q) {
    const int64_t lin = sw_sampled(q, stride);
    if (lin >= total) continue;
    const int64_t a0 = (lin % nbx) * seg, dlo = ((int64_t(v.excl) + 1) & ~int64_t(7)) + (lin / nbx) * nd;
    const int64_t d0 = std::max(dlo, int64_t(v.excl) + 1), d1 = std::min(dlo + nd, v.M);
    // rows a0 .. a0 + seg - 1 against diagonals d0 .. d1 - 1 with a + delta < M
    for (int64_t dl = d0; dl < d1; dl += 64) {
      const int64_t c = std::min<int64_t>(64, d1 - dl);
      *pairs += double(c) * double(std::max<int64_t>(0, std::min<int64_t>(seg, v.M - (dl + c / 2) - a0)));
    }
  }
  const cudaError_t e = v.P == 2 ? sweep_sample<2>(jb, nbx, blocks, stride, s) : sweep_sample<1>(jb, nbx, blocks, stride, s);
  if (e != cudaSuccess || stride > 1) return e;
  return v.P == 2 ? sweep_marked<2>(jb, s) : sweep_marked<1>(jb, s);
}

template <int P>
static cudaError_t sweep_batch(const SweepJob* jobs, const std::vector<SweepItem>& items, size_t smem,
                               cudaStream_t s) {
  if (items.empty()) return cudaSuccess;
  SweepItem* ditems = nullptr;
  int* dnext = nullptr;
  cudaError_t e = cudaMallocAsync(&ditems, items.size() * sizeof(SweepItem), s);
  if (e == cudaSuccess) e = cudaMallocAsync(&dnext, sizeof(int), s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(ditems, items.data(), items.size() * sizeof(SweepItem), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(dnext, 0, sizeof(int), s);
  if (e == cudaSuccess) e = allow_smem(reinterpret_cast<const void*>(k_sweep_batch<P>), smem);
  if (e == cudaSuccess) {
    const int64_t grid = std::min<int64_t>(int64_t(sm_count()) * kSwBlocks<P>, int64_t(items.size()));
    MOMENTI_LAUNCH("allpairs_batch", s, k_sweep_batch<P><<<unsigned(grid), kSwThreads, smem, s>>>(jobs, ditems, int(items.size()), dnext));
    e = cudaGetLastError();
  }
  if (ditems) cudaFreeAsync(ditems, s);
  if (dnext) cudaFreeAsync(dnext, s);
  return e;
}

cudaError_t launch_allpairs_batch(std::vector<SweepJob> jobs, cudaStream_t s) {
  if (jobs.empty()) return cudaSuccess;
  // items of every job, largest series first; one launch per form
  std::stable_sort(jobs.begin(), jobs.end(), [](const SweepJob& x, const SweepJob& y) { return x.v.M > y.v.M; });
  std::vector<SweepItem> items[2];
  size_t smem[2] = {0, 0};
  for (size_t q = 0; q < jobs.size(); ++q) {
    SweepJob& j = jobs[q];
    const int64_t gy = sw_gy(j.v);
    if (gy <= 0) continue;
    const int f = j.v.P - 1;
    j.seg = sw_seg(j.v);
    smem[f] = std::max(smem[f], sw_smem(j.v));
    for (int64_t by = 0; by < gy; ++by) {
      const int64_t dfirst = std::max(((int64_t(j.v.excl) + 1) & ~int64_t(7)) + by * sw_diags(j.v.G),
                                      int64_t(j.v.excl) + 1);
      for (int64_t bx = 0; bx * j.seg < j.v.M - dfirst; ++bx)
        items[f].push_back(SweepItem{uint32_t(q), uint32_t(bx), uint32_t(by)});
    }
  }
  SweepJob* djobs = nullptr;
  cudaError_t e = cudaMallocAsync(&djobs, jobs.size() * sizeof(SweepJob), s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(djobs, jobs.data(), jobs.size() * sizeof(SweepJob), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = sweep_batch<1>(djobs, items[0], smem[0], s);
  if (e == cudaSuccess) e = sweep_batch<2>(djobs, items[1], smem[1], s);
  for (size_t q = 0; q < jobs.size() && e == cudaSuccess; ++q)
    if (sw_gy(jobs[q].v) > 0) e = jobs[q].v.P == 2 ? sweep_marked<2>(jobs[q], s) : sweep_marked<1>(jobs[q], s);
  if (djobs) cudaFreeAsync(djobs, s);
  return e;
}

}  // namespace momenti
