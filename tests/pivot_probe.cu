// The pivot of csrc/pivot_fp64.cuh for arrays of (x0, tail), and from S itself.
#include "pivot_fp64.cuh"

using namespace slqr;

__global__ void pivot_kernel(const double *x0, const double *tail, const int *E, int n,
                             double *out, int from_S) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  PivotFp64 r = {0.0, 0.0, 0.0, true};
  if (from_S) pivot_fp64(tail[i], x0[i], &r.cl, &r.up, &r.rb);
  else r = pivot_fp64(x0[i], tail[i], E[i] != 0, E[i]);
  out[4 * i] = r.cl;
  out[4 * i + 1] = r.up;
  out[4 * i + 2] = r.rb;
  out[4 * i + 3] = r.defined ? 1.0 : 0.0;
}

extern "C" int pivot_probe(const double *x0, const double *tail, const int *E, int n, double *out,
                           int from_S) {
  pivot_kernel<<<(n + 127) / 128, 128>>>(x0, tail, E, n, out, from_S);
  return (int)cudaDeviceSynchronize();
}
