// Runs the exact path's recording sweep on a series and returns what it
// records, for the tests: the public calls only return the final top-k.
#include "internal.h"

#include <vector>

using namespace momenti;

namespace {

struct Held {
  std::vector<void*> bufs;
  ~Held() {
    for (void* p : bufs) cudaFree(p);
  }
  template <typename T>
  T* get(size_t count) {
    void* p = nullptr;
    if (cudaMalloc(&p, count * sizeof(T) + 16) != cudaSuccess) return nullptr;
    bufs.push_back(p);
    return static_cast<T*>(p);
  }
};

}  // namespace

// Pairs whose approximate distance lies in (lo, thr], with that distance;
// at most cap of them are stored.  form: 0 the plain launch, 1 the batching
// form's, beside a second copy of the series, from 8 on the sample's with a
// share of 1 and that many rows per block (a multiple of 8, at most 2048).
// Returns how many there are, or a negative CUDA error.
extern "C" long long sweep_pairs(const void* series, int dtype, long long n, int D, int w, int excl, int d, float lo,
                                 float thr, int form, unsigned long long* pairs, float* dist, long long cap) {
  Held m;
  Index ix;
  ix.n = n;
  ix.M = n - w + 1;
  ix.D = D;
  ix.w = w;
  ix.excl = excl;
  ix.has_lo = dtype == 1;
  const size_t e = size_t(D) * size_t(n), em = size_t(D) * size_t(ix.M), elem = dtype == 1 ? 8 : 4;
  void* src = m.get<char>(e * elem);
  ix.xs_hi = m.get<float>(e);
  ix.xs_lo = ix.has_lo ? m.get<float>(e) : nullptr;
  ix.mu = m.get<double>(em);
  ix.sig = m.get<double>(em);
  ix.mu_hi = m.get<float>(em);
  ix.mu_lo = m.get<float>(em);
  ix.inv_sig = m.get<float>(em);
  void* tab = m.get<char>(sweep_table_bytes(ix));
  ApRec rc[2];
  for (ApRec& r : rc) {
    r.out = reinterpret_cast<decltype(r.out)>(m.get<unsigned long long>(size_t(cap)));
    r.out_d = m.get<float>(size_t(cap));
    r.count = m.get<unsigned long long>(1);
    r.hist = m.get<uint32_t>(kApBins);
    r.cap = uint64_t(cap);
    r.lo = lo;
    r.hscale = float(kApBins) / (thr - lo);
    if (!r.out || !r.out_d || !r.count || !r.hist) return -2;
    cudaMemset(r.count, 0, 8);
    cudaMemset(r.hist, 0, kApBins * 4);
  }
  if (!src || !ix.xs_hi || !ix.mu || !ix.sig || !ix.mu_hi || !ix.mu_lo || !ix.inv_sig || !tab ||
      (ix.has_lo && !ix.xs_lo))
    return -2;
  cudaMemcpy(src, series, e * elem, cudaMemcpyHostToDevice);
  cudaError_t er = launch_split_series(src, dtype, n, D, n, ix.xs_hi, ix.xs_lo, nullptr);
  if (er == cudaSuccess) er = launch_window_stats(ix, nullptr);
  SweepView v;
  if (er == cudaSuccess) er = launch_sweep_table(ix, tab, &v, nullptr);
  if (er == cudaSuccess) {
    if (form >= 8) {
      double held = 0.0;
      er = launch_allpairs_sample(v, d, thr, rc[0], 1.0, form, &held, nullptr, nullptr);
    } else if (form) {
      std::vector<SweepJob> jobs(2);
      for (int q = 0; q < 2; ++q) {
        jobs[size_t(q)].v = v;
        jobs[size_t(q)].rc = rc[q];
        jobs[size_t(q)].thr = thr;
        jobs[size_t(q)].d = d;
      }
      er = launch_allpairs_batch(jobs, nullptr);
    } else {
      er = launch_allpairs(v, d, thr, rc[0], nullptr);
    }
  }
  if (er == cudaSuccess) er = cudaDeviceSynchronize();
  if (er != cudaSuccess) return -1000 - int(er);
  unsigned long long cnt = 0;
  cudaMemcpy(&cnt, rc[0].count, 8, cudaMemcpyDeviceToHost);
  const unsigned long long k = cnt < (unsigned long long)cap ? cnt : (unsigned long long)cap;
  cudaMemcpy(pairs, rc[0].out, k * 8, cudaMemcpyDeviceToHost);
  cudaMemcpy(dist, rc[0].out_d, k * 4, cudaMemcpyDeviceToHost);
  return (long long)cnt;
}
