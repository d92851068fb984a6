// The fixed-point apply of one dense matrix: y = M v, from libfeti.so's own launchers.
#include "feti_internal.h"

#include <vector>

extern "C" int symv_fixed_probe(int m, int C, const double* M, const double* v, double* y) {
  feti::SubLayout L{};
  L.nbp = m;
  const int order = 0, zero = 0;
  double *dM = nullptr, *dv = nullptr, *dy = nullptr;
  int2 *dp = nullptr, *de = nullptr;
  int32_t* dorder = nullptr;
  int* dzero = nullptr;
  feti::SubLayout* dl = nullptr;
  auto up = [](auto** d, const void* h, size_t bytes) {
    const cudaError_t e = cudaMalloc(reinterpret_cast<void**>(d), bytes);
    return e != cudaSuccess || !h ? e : cudaMemcpy(*d, h, bytes, cudaMemcpyHostToDevice);
  };
  cudaError_t e = up(&dM, M, sizeof(double) * m * m);
  if (e == cudaSuccess) e = up(&dv, v, sizeof(double) * m);
  if (e == cudaSuccess) e = up(&dy, nullptr, sizeof(double) * m);
  if (e == cudaSuccess) e = up(&dp, nullptr, sizeof(int2) * feti::fix_entries(m));
  if (e == cudaSuccess) e = up(&de, nullptr, sizeof(int2) * m);
  if (e == cudaSuccess) e = up(&dorder, &order, sizeof(order));
  if (e == cudaSuccess) e = up(&dzero, &zero, sizeof(zero));
  if (e == cudaSuccess) e = up(&dl, &L, sizeof(L));
  if (e == cudaSuccess) {
    feti::launch_fix_operator(1, m, dl, 0, dM, de, dp, nullptr);
    e = feti::launch_symv_fixed(C, 1, dorder, m, dl, 0, dp, de, dM, dv, dy, dzero, nullptr);
  }
  if (e == cudaSuccess) e = cudaMemcpy(y, dy, sizeof(double) * m, cudaMemcpyDeviceToHost);
  for (void* p : {(void*)dM, (void*)dv, (void*)dy, (void*)dp, (void*)de, (void*)dorder, (void*)dzero, (void*)dl}) cudaFree(p);
  return (int)e;
}
