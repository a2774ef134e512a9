// Panel Cholesky factorisation and triangular inverse of the blocks of a
// block-diagonal matrix: reads (nb, stacked, threads, lengths[4]) as int32 and
// the n x n matrix as doubles from stdin; writes the n x n factor, the n x n
// inverse (lower triangles of the blocks, zero elsewhere) and the flag.
#include <cstdio>
#include <vector>
#include "../paper_1507_04789_gb300/csrc/mra_device.cuh"

using namespace mra;

template <int NTH>
__global__ void __launch_bounds__(NTH) factor(const double* M, int nb, int stk, const int* segs, double* out, int* flag) {
  extern __shared__ double sm[];
  __shared__ int bad, seg[LGRP_MAX + 1];
  if (threadIdx.x == 0) bad = 0;
  if (threadIdx.x <= nb) seg[threadIdx.x] = segs[threadIdx.x];
  __syncthreads();
  const int n = seg[nb];
  int most = 0;
  for (int b = 0; b < nb; ++b) most = max(most, seg[b + 1] - seg[b]);
  const int lda = (stk ? most : n) + 1;
  double* A = sm;
  double* scr = A + n * lda;
  auto at = [&](int i, int j) -> double& { return A[i * lda + j - (stk ? seg[seg_block(seg, nb, i)] : 0)]; };
  auto in = [&](int i, int j) { return j <= i && j >= seg[seg_block(seg, nb, i)]; };
  for (int t = threadIdx.x; t < n * n; t += NTH)
    if (in(t / n, t % n)) at(t / n, t % n) = M[t];
  auto store = [&](double* o) {
    __syncthreads();
    for (int t = threadIdx.x; t < n * n; t += NTH) o[t] = in(t / n, t % n) ? at(t / n, t % n) : 0.0;
    __syncthreads();
  };
  if (nb == 1 && !stk) chol_smem<NTH>(A, n, lda, &bad);
  else if (stk) chol_seg<true, NTH>(A, lda, seg, nb, &bad);
  else chol_seg<false, NTH>(A, lda, seg, nb, &bad);
  store(out);
  if (nb == 1 && !stk) trinv_smem<NTH>(A, n, lda, scr);
  else if (stk) trinv_seg<true, NTH>(A, lda, seg, nb, scr);
  else trinv_seg<false, NTH>(A, lda, seg, nb, scr);
  store(out + n * n);
  if (threadIdx.x == 0) *flag = bad;
}

int main() {
  int h[7];
  cudaFuncSetAttribute(factor<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160000);
  cudaFuncSetAttribute(factor<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160000);
  while (fread(h, 4, 7, stdin) == 7) {
    const int nb = h[0];
    if (nb < 1 || nb > LGRP_MAX) return 2;
    int seg[LGRP_MAX + 1] = {0};
    for (int b = 0; b < nb; ++b) seg[b + 1] = seg[b] + h[3 + b];
    const int n = seg[nb];
    if (n < 1 || n > FAC_MAX_N) return 2;
    std::vector<double> A((size_t)n * n), out(2 * A.size());
    if (fread(A.data(), 8, A.size(), stdin) != A.size()) return 2;
    double *dA, *dO;
    int *ds, *df, flag = 0;
    cudaMalloc(&dA, A.size() * 8);
    cudaMalloc(&dO, out.size() * 8);
    cudaMalloc(&ds, sizeof(seg));
    cudaMalloc(&df, 4);
    cudaMemcpy(dA, A.data(), A.size() * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(ds, seg, sizeof(seg), cudaMemcpyHostToDevice);
    const size_t sm = sizeof(double) * ((size_t)n * (n + 1) + FAC_SCRATCH);
    if (h[2] == 512) factor<512><<<1, 512, sm>>>(dA, nb, h[1], ds, dO, df);
    else factor<256><<<1, 256, sm>>>(dA, nb, h[1], ds, dO, df);
    if (cudaMemcpy(out.data(), dO, out.size() * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    cudaMemcpy(&flag, df, 4, cudaMemcpyDeviceToHost);
    fwrite(out.data(), 8, out.size(), stdout);
    fwrite(&flag, 4, 1, stdout);
    cudaFree(dA); cudaFree(dO); cudaFree(ds); cudaFree(df);
  }
  return 0;
}
