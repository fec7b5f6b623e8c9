// Single steps of the residual minimisation (Alg. 1) for test_gpu_minimisation_kernels.py: the
// library's kernels on vectors and a level state that the test sets.  Host pointers throughout.
#include "kcmg_internal.h"

#include <cmath>
#include <vector>

using namespace kcmg;

namespace step_test {

template <typename T>
struct Dev {
  T* p = nullptr;
  size_t n = 0;
  Dev(const T* h, size_t n) : n(n) {
    cudaMalloc((void**)&p, n * sizeof(T) + 16);
    if (h) cudaMemcpy(p, h, n * sizeof(T), cudaMemcpyHostToDevice);
    else cudaMemset(p, 0, n * sizeof(T));
  }
  ~Dev() { cudaFree(p); }
  void get(T* h) const { cudaMemcpy(h, p, n * sizeof(T), cudaMemcpyDeviceToHost); }
};

// the new column with l columns stored: w_l = gamma (w - W h), r -= alpha w_l; returns ||r||
template <typename T>
int update(int N, int l, T* W, const T* w, const T* z, const double* h, double gamma, double alpha, T* r, int nblk,
           double* rnorm) {
  const int lcap = l + 1;
  Dev<T> dW(W, (size_t)lcap * N), dZ(nullptr, (size_t)lcap * N), dw(w, N), dz(z, N), dr(r, N);
  Dev<double> dh(h, lcap), part(nullptr, (size_t)(nblk + 1) * 8), gm(nullptr, lcap), al(nullptr, lcap),
      y(nullptr, lcap), R(nullptr, (size_t)lcap * lcap + 1);
  LevelState st{};
  st.l = l;
  st.lcap = lcap;
  st.gamma = gamma;
  st.alpha = alpha;
  Dev<LevelState> ds(&st, 1);
  EpiArgs e;
  e.st = ds.p;
  e.kind = EPI_FINISH;
  e.h = e.h2 = dh.p;
  const RmCoef co{gm.p, al.p, y.p, R.p};
  launch_gram_update<T>(dW.p, dZ.p, N, dw.p, dw.p, dz.p, co, dr.p, lcap, nblk, part.p, e, 0);
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  ds.get(&st);
  dW.get(W);
  dr.get(r);
  *rnorm = st.rnorm;
  return st.l == l + 1 ? 0 : 2;
}

}  // namespace step_test

using namespace step_test;

extern "C" {

int update_f32(int N, int l, float* W, const float* w, const float* z, const double* h, double gamma, double alpha,
               float* r, int nblk, double* rnorm) {
  return update<float>(N, l, W, w, z, h, gamma, alpha, r, nblk, rnorm);
}
int update_f64(int N, int l, double* W, const double* w, const double* z, const double* h, double gamma, double alpha,
               double* r, int nblk, double* rnorm) {
  return update<double>(N, l, W, w, z, h, gamma, alpha, r, nblk, rnorm);
}

}  // extern "C"
