// One small step (csrc/bodies.cuh, small_body) outside a program: 32 rows of A times two columns of B over
// 2^rk contracted indices, with B zero for whole warps of outputs. Prints, per rk, the number of outputs
// that differ from the host's sums, and with one infinity in A the number of outputs of its row that are
// finite and of other rows that changed.
#include <cuda_runtime.h>

#include <cmath>
#include <complex>
#include <cstdio>
#include <limits>
#include <vector>

#include "bodies.cuh"

using namespace ajf;
using C = std::complex<double>;

__global__ void __launch_bounds__(kSmallThreads) step(const StepDev* steps, int blocks, double* arena) {
  extern __shared__ int64_t tab[];
  __shared__ StepDev st;
  small_body<double, double, SyncBlock, kSmallThreads>(steps, 1, blocks, arena, blockIdx.x, tab, st);
}

int main() {
  for (int rk = 0; rk <= 5; ++rk) {
    const int nk = 1 << rk;
    StepDev st{};
    st.pa = 32 << rk;
    st.b = 2 * st.pa;
    st.pb = 2 << rk;
    st.c = st.b + 2 * st.pb;
    st.pc = 64;
    st.rc = 6;
    st.rk = rk;
    st.scalar_slot = -1;
    st.oa.nbits = st.ob.nbits = 6;
    st.ka.nbits = st.kb.nbits = rk;
    for (int i = 0; i < 6; ++i) {
      st.oa.pos[i] = i < 5 ? rk + i : -1;
      st.ob.pos[i] = i < 5 ? -1 : rk;
    }
    for (int i = 0; i < rk; ++i) st.ka.pos[i] = st.kb.pos[i] = i;
    std::vector<double> h(st.c + 2 * 64, 0.0);
    auto A = [&](int r, int k) { return C(0.5 + r - 0.25 * k, 1.0 / (1 + r + k)); };
    auto B = [&](int n, int k) { return nk > 1 && k % 2 != n ? C(0, 0) : C(1 + k, n ? 0.0 : 0.125 * k); };
    for (int r = 0; r < 32; ++r)
      for (int k = 0; k < nk; ++k) {
        h[(r << rk) + k] = A(r, k).real();
        h[st.pa + (r << rk) + k] = A(r, k).imag();
      }
    for (int n = 0; n < 2; ++n)
      for (int k = 0; k < nk; ++k) {
        h[st.b + (n << rk) + k] = B(n, k).real();
        h[st.b + st.pb + (n << rk) + k] = B(n, k).imag();
      }
    double* d = nullptr;
    StepDev* ds = nullptr;
    if (cudaMalloc(&d, h.size() * 8) != cudaSuccess || cudaMalloc(&ds, sizeof(st)) != cudaSuccess) return 1;
    cudaMemcpy(ds, &st, sizeof(st), cudaMemcpyHostToDevice);
    int wrong = 0, finite = 0, changed = 0;
    std::vector<double> first(128), out(128);
    for (int pass = 0; pass < 2; ++pass) {
      if (pass) h[(3 << rk) + nk - 1] = std::numeric_limits<double>::infinity();  // row 3, last contracted index
      cudaMemcpy(d, h.data(), h.size() * 8, cudaMemcpyHostToDevice);
      step<<<1, kSmallThreads, 4 * 256 * 8>>>(ds, 1, d);
      auto& o = pass ? out : first;
      if (cudaMemcpy(o.data(), d + st.c, 128 * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    }
    for (int n = 0; n < 2; ++n)
      for (int r = 0; r < 32; ++r) {
        C ref = 0;
        double mag = 0;
        for (int k = 0; k < nk; ++k) {
          ref += A(r, k) * B(n, k);
          mag += std::abs(A(r, k)) * std::abs(B(n, k));
        }
        const int o = 32 * n + r;
        // 2 nk roundings of partial sums and products, on either side
        if (std::abs(C(first[o], first[64 + o]) - ref) > 4 * nk * 0x1p-52 * mag) ++wrong;
        if (r == 3) finite += std::isfinite(out[o]) || std::isfinite(out[64 + o]);
        else changed += out[o] != first[o] || out[64 + o] != first[64 + o];
      }
    std::printf("%d %d %d %d\n", rk, wrong, finite, changed);
    cudaFree(d);
    cudaFree(ds);
  }
  return 0;
}
