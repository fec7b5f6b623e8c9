// A step of the batched residual minimisation for test_gpu_minimisation_kernels.py: the second
// Gram-Schmidt pass and the update, by the batched solve's kernels, on bases, vectors and a state that
// the test sets.  Vectors [N][R], bases [l + 1][N][R]; host pointers.  The kernels are local to their
// translation unit, which is therefore part of this one.
#include "mrhs.cu"

using namespace kcmg;

namespace step_test {

struct Dev {
  double* p = nullptr;
  size_t n = 0;
  Dev(const double* h, size_t n) : n(n) {
    cudaMalloc((void**)&p, n * sizeof(double) + 16);
    if (h) cudaMemcpy(p, h, n * sizeof(double), cudaMemcpyHostToDevice);
    else cudaMemset(p, 0, n * sizeof(double));
  }
  ~Dev() { cudaFree(p); }
  void get(double* h) const { cudaMemcpy(h, p, n * sizeof(double), cudaMemcpyDeviceToHost); }
};

}  // namespace step_test

// in_kernel: the reductions' last blocks run the control, else k_mreduce launches
extern "C" int batched_second_pass(int N, int R, int l, double* W, double* Z, const double* w, const double* z,
                                   double naz2, double* x, double* r, const int* reorth, int in_kernel, int blocks,
                                   int* lnew, double* rnorm) {
  using step_test::Dev;
  const int lcap = l + 1, ps = lcap + 2, thr = kGramWarps * 32;
  const size_t NR = (size_t)N * R;
  Dev dW(W, lcap * NR), dZ(Z, lcap * NR), dw(w, NR), dz(z, NR), dx(x, NR), dr(r, NR);
  Dev part(nullptr, (size_t)blocks * ps * 32), sums(nullptr, ps * 32), cw(nullptr, ps * 32), cz(nullptr, ps * 32);
  MState h;
  memset(&h, 0, sizeof h);
  h.R = R;
  h.lcap = lcap;
  h.cap = lcap;
  h.brk_tol = 1e-14;
  h.any_reorth = 1;
  for (int k = 0; k < R; ++k) {
    h.act[k] = 1;
    h.l[k] = l;
    h.flags[k] = reorth[k] ? MF_REORTH : MF_DISCARD;
    h.naz2[k] = naz2;
  }
  MState* st = nullptr;
  cudaMalloc((void**)&st, sizeof h);
  cudaMemcpy(st, &h, sizeof h, cudaMemcpyHostToDevice);
  CtlArgs g2{st, nullptr, CTL_GRAM2, sums.p, cw.p, cz.p, nullptr, 0u, {dW.p, dZ.p, dx.p, dr.p, N}}, fin = g2, none = g2;
  fin.steps = CTL_FINISH;
  none.steps = CTL_NONE;
  k_mdots<<<blocks, thr>>>(dW.p, dw.p, dr.p, N, R, lcap, part.p, 1, in_kernel ? g2 : none);
  if (!in_kernel) k_mreduce<<<ps, 256>>>(part.p, blocks, ps, lcap, 1, g2);
  auto update = in_kernel ? k_mupdate<8> : k_mupdate<4>;
  update<<<blocks, thr>>>(dW.p, dZ.p, N, R, dw.p, dw.p, dz.p, dx.p, dr.p, cw.p, cz.p, part.p, in_kernel ? fin : none);
  if (!in_kernel) k_mreduce<<<2, 256>>>(part.p, blocks, 2, 0, 0, fin);
  const bool ok = cudaDeviceSynchronize() == cudaSuccess;
  cudaMemcpy(&h, st, sizeof h, cudaMemcpyDeviceToHost);
  cudaFree(st);
  dW.get(W);
  dZ.get(Z);
  dx.get(x);
  dr.get(r);
  for (int k = 0; k < R; ++k) {
    lnew[k] = h.l[k];
    rnorm[k] = h.rnorm[k];
  }
  return ok ? 0 : 1;
}
