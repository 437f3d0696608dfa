// The float64 eigenvalue search of csrc/eigen.cu on its own: called by test_gpu_eigen_search.py.
#include "eigen.cu"

template <int NN>
static cudaError_t search(const double* M, int batch, int r, double* lam) {
  using HL = spr::HhLayout<NN>;
  double* ws;
  cudaError_t e = spr::init_eigen();
  if (e == cudaSuccess) e = cudaMalloc(&ws, spr::eig_scratch_doubles(batch, NN) * sizeof(double));
  if (e != cudaSuccess) return e;
  spr::k_householder<NN, double><<<batch, (spr::kHhThreads<NN>)>>>(M, (spr::i64)NN * NN, ws, 0);
  spr::k_eig_vectors<NN, double><<<dim3((r + spr::kVecsOf<double> - 1) / spr::kVecsOf<double>, batch), spr::kLanesOf<double> * spr::kVecsOf<double>,
                                   (spr::VecSmem<NN, double>::total)>>>(ws, r);
  e = cudaMemcpy2D(lam, r * sizeof(double), ws + HL::lam, HL::stride * sizeof(double), r * sizeof(double), batch, cudaMemcpyDeviceToDevice);
  const cudaError_t run = cudaDeviceSynchronize();
  cudaFree(ws);
  return e != cudaSuccess ? e : run;
}

// M [batch][n][n] of largest magnitude 1, lam [batch][r]: device memory
extern "C" int largest_eigenvalues(const double* M, int batch, int n, int r, double* lam) {
  return n == 128 ? search<128>(M, batch, r, lam) : search<64>(M, batch, r, lam);
}
