// Single steps of the residual minimisation (Alg. 1) for test_gpu_minimisation_kernels.py: the
// library's kernels on vectors and a level state that the test sets.  Host pointers throughout.
#include "coarse_cycle.cuh"
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

// a second Gram-Schmidt pass over w' and the step after it; returns the new column's gamma and alpha
template <typename T>
int second_pass(int N, int l, T* W, const T* w, const T* z, double naz2, T* r, int nblk, double* gamma, double* alpha,
                double* rnorm) {
  const int lcap = l + 1;
  Dev<T> dW(W, (size_t)lcap * N), dZ(nullptr, (size_t)lcap * N), dw(w, N), dz(z, N), dr(r, N);
  Dev<double> h(nullptr, lcap), h2(nullptr, lcap), part(nullptr, (size_t)(nblk + 1) * (lcap + 8)), gm(nullptr, lcap),
      al(nullptr, lcap), y(nullptr, lcap), R(nullptr, (size_t)lcap * lcap + 1);
  LevelState st{};
  st.l = l;
  st.lcap = lcap;
  st.naz2 = naz2;
  st.brk = 1e-14;
  st.flags = F_REORTH;
  Dev<LevelState> ds(&st, 1);
  EpiArgs e;
  e.st = ds.p;
  e.kind = EPI_GRAM2;
  e.h = h.p;
  e.h2 = h2.p;
  launch_gram_dots<T>(dW.p, N, dw.p, dr.p, lcap, nblk, part.p, e, 1, 0);
  e.kind = EPI_FINISH;
  const RmCoef co{gm.p, al.p, y.p, R.p};
  launch_gram_update<T>(dW.p, dZ.p, N, dw.p, dw.p, dz.p, co, dr.p, lcap, nblk, part.p, e, 0);
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  ds.get(&st);
  dW.get(W);
  dr.get(r);
  std::vector<double> g(lcap), a(lcap);
  gm.get(g.data());
  al.get(a.data());
  *gamma = g[l];
  *alpha = a[l];
  *rnorm = st.rnorm;
  return st.l == l + 1 ? 0 : 2;
}

// the persistent kernel's sums over a block that is alone on its level: W^T w, w . w, w . r, r . r, and
// the last column's with r
constexpr int kNP = 3;
template <typename T>
__global__ void k_dots(const __grid_constant__ CoarseArgs a, const T* W, int N, int l, const T* w, const T* r,
                       double* out) {
  __shared__ double sh[32 * 8];
  __shared__ RmScal rms;
  __shared__ int nbs[5];
  __shared__ long long tph[kCoarsePhases + KCMG_MAX_LEVELS];
  double* red_s = reinterpret_cast<double*>(smem_cc + a.sm_red);
  CoarseCycle<T, T, T, kNP, 2, false> cc{a, sh, red_s, red_s + a.cols + 4, &rms, nbs, tph, nullptr};
  cc.rows = N;
  cc.rs_off = a.lv[0].sm_r;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    cc.ws()[i] = w[i];
    cc.rs_()[i] = r[i];
  }
  __syncthreads();
  cc.dots(W, N, l);
  for (int i = threadIdx.x; i < l + 4; i += blockDim.x) out[i] = l > 0 || i < 3 ? red_s[i] : 0.0;
}

// what the persistent kernel does after a Gram pass with these sums (l coefficients, the last of them h)
__global__ void k_decide(const __grid_constant__ CoarseArgs a, int l, int pass, double naz2, double n2, double h,
                         int* verdict) {
  __shared__ double red_s[64];
  __shared__ RmScal rms;
  CoarseCycle<double, double, double, kNP, 2, false> cc{a, nullptr, red_s, nullptr, &rms, nullptr, nullptr, nullptr};
  for (int p = 0; p <= pass; p += max(1, pass)) {   // the first pass leaves ||A z||^2
    __syncthreads();
    for (int i = threadIdx.x; i < l + 4; i += blockDim.x) red_s[i] = 0.0;
    __syncthreads();
    if (threadIdx.x == 0) {
      red_s[l] = p == 0 && pass > 0 ? naz2 : n2;
      red_s[l + 1] = red_s[l + 2] = 1.0;
      if (l > 0) red_s[l - 1] = h;
    }
    __syncthreads();
    cc.decide(l, p);
  }
  __syncthreads();
  if (threadIdx.x == 0) *verdict = rms.verdict;
}

template <typename T>
int dots(int N, int l, const T* W, const T* w, const T* r, double* out) {
  Dev<T> dW(W, (size_t)(l + 1) * N), dw(w, N), dr(r, N);
  Dev<double> dout(nullptr, l + 4);
  CoarseArgs a{};
  a.nlev = 2;
  a.cols = l + 1;
  a.lv[0].N = N;
  a.lv[0].sm_r = (int)(N * sizeof(T) + 15) / 16 * 16;
  a.sm_red = 2 * a.lv[0].sm_r;
  a.sm_bytes = a.sm_red + (int)((2 * a.cols + 4) * sizeof(double));
  k_dots<T><<<1, kCoarseThreads, a.sm_bytes>>>(a, dW.p, N, l, dw.p, dr.p, dout.p);
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  dout.get(out);
  return 0;
}

}  // namespace step_test

using namespace step_test;

extern "C" {

int decide(int l, int pass, double naz2, double n2, double h) {
  Dev<int> v(nullptr, 1);
  CoarseArgs a{};
  a.brk = 1e-14;
  k_decide<<<1, 64>>>(a, l, pass, naz2, n2, h, v.p);
  int r = -1;
  if (cudaDeviceSynchronize() == cudaSuccess) v.get(&r);
  return r;
}
int dots_f32(int N, int l, const float* W, const float* w, const float* r, double* out) { return dots<float>(N, l, W, w, r, out); }
int dots_f64(int N, int l, const double* W, const double* w, const double* r, double* out) { return dots<double>(N, l, W, w, r, out); }

int second_pass_f32(int N, int l, float* W, const float* w, const float* z, double naz2, float* r, int nblk,
                    double* gamma, double* alpha, double* rnorm) {
  return second_pass<float>(N, l, W, w, z, naz2, r, nblk, gamma, alpha, rnorm);
}
int second_pass_f64(int N, int l, double* W, const double* w, const double* z, double naz2, double* r, int nblk,
                    double* gamma, double* alpha, double* rnorm) {
  return second_pass<double>(N, l, W, w, z, naz2, r, nblk, gamma, alpha, rnorm);
}
int update_f32(int N, int l, float* W, const float* w, const float* z, const double* h, double gamma, double alpha,
               float* r, int nblk, double* rnorm) {
  return update<float>(N, l, W, w, z, h, gamma, alpha, r, nblk, rnorm);
}
int update_f64(int N, int l, double* W, const double* w, const double* z, const double* h, double gamma, double alpha,
               double* r, int nblk, double* rnorm) {
  return update<double>(N, l, W, w, z, h, gamma, alpha, r, nblk, rnorm);
}

}  // extern "C"
