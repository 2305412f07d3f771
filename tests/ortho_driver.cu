// One step of the Arnoldi process by ortho_kernel on given vectors, for tests/test_gpu_ortho_kernel.py.
// stdin: n (entries), kk (basis vectors), blocks, wait limit, then (kk + 1) n words of 64 bits (doubles) in binary; the
// launch is made twice: with the limit given, then on fresh exchange words with a limit that is not reached.
// stdout, per launch: status (int32), kk + 1 doubles (coefficients, squared norm), n doubles (the new vector).
#include <cstdio>
#include <vector>

#include "ortho.cuh"

using namespace vms;

int main() {
  long long head[4];
  if (fread(head, sizeof head, 1, stdin) != 1) return 2;
  int64_t n = head[0];
  int kk = (int)head[1];
  const int blocks = (int)head[2];
  std::vector<double> v((size_t)(kk + 1) * n);
  if (n < 4 || n % 4 || kk < 1 || kk > OG_MAX || blocks < 1 || blocks > OG_BLOCKS ||
      fread(v.data(), sizeof(double), v.size(), stdin) != v.size())
    return 2;
  double *V, *X, *out;
  if (cudaMalloc(&V, sizeof(double) * v.size()) != cudaSuccess || cudaMalloc(&X, sizeof(double) * 2 * OG_SET) != cudaSuccess ||
      cudaMallocHost(&out, sizeof(double) * (OG_MAX + 2)) != cudaSuccess)
    return 3;
  for (int pass = 0; pass < 2; ++pass) {
    uint32_t lim = pass ? 1u << 22 : (uint32_t)head[3];
    cudaMemcpy(V, v.data(), sizeof(double) * v.size(), cudaMemcpyHostToDevice);
    cudaMemset(X, 0xff, sizeof(double) * 2 * OG_SET);
    out[kk + 1] = 0.0;
    double* Y = X + OG_SET;
    int kprev = 0, gprev = 0;
    void* args[] = {&V, &n, &kk, &X, &Y, &kprev, &gprev, &lim, &out};
    if (cudaLaunchCooperativeKernel((const void*)ortho_kernel<double>, dim3(blocks), dim3(OG_THREADS), args, 0, 0) != cudaSuccess ||
        cudaDeviceSynchronize() != cudaSuccess)
      return 3;
    std::vector<double> w(n);
    cudaMemcpy(w.data(), V + (size_t)kk * n, sizeof(double) * n, cudaMemcpyDeviceToHost);
    const int status = (int)out[kk + 1];
    fwrite(&status, sizeof status, 1, stdout);
    fwrite(out, sizeof(double), kk + 1, stdout);
    fwrite(w.data(), sizeof(double), n, stdout);
  }
  return 0;
}
