// One product of the FP64-emulation engine on the GPU: reads
//   na nb K layoutA layoutB tables   (int32)  then A (na x K) and B (nb x K), row-major doubles
// from stdin and writes the na x nb result.  layout 0: rows K-contiguous, even
// stride (vector loads); 1: rows K-contiguous, odd stride; 2: K-major.  tables:
// 1 passes the row scales of every 128-column group, 0 lets the engine form them.
#include <cstdio>
#include <vector>
#include "../paper_1507_04789_gb300/csrc/mra_emu.cuh"

using namespace mra;

__global__ void __launch_bounds__(EM_NT) product(const double* A, long sai, long sak, int na, const double* B, long sbj,
                                                 long sbk, int nb, int K, const int* pa, const int* pb, double* C,
                                                 int* failed) {
  extern __shared__ __align__(1024) unsigned char dsm[];
  __shared__ __align__(8) uint64_t mbar[EM_MBARS];
  __shared__ uint32_t slot;
  __shared__ int fail;
  __shared__ __align__(16) int rexp[EM_REXP], cexp[EM_CEXP];
  EmCtx cx;
  cx.stage = reinterpret_cast<uint16_t*>(dsm);
  cx.rexp = rexp;
  cx.cexp = cexp;
  cx.mbar = mbar;
  cx.fail = &fail;
  em_init(cx, &slot);
  EmAcc acc;
  bool ok = true;
  for (int rep = 0; rep < 3 && ok; ++rep)   // (the barriers' phases carry over from product to product)
    ok = em_mma(cx, acc, A, sai, sak, na, B, sbj, sbk, nb, K, pa, na, pb, nb);
  if (ok && acc.row() < na)
    for (int c = 0; c < EmAcc::NC; ++c)
      if (acc.col0() + c < nb) C[acc.row() * nb + acc.col0() + c] = acc.v[c];
  em_release(cx);
  if (!ok && threadIdx.x == 0) *failed = 1;
}

static std::vector<double> lay(const std::vector<double>& X, int n, int K, int layout, long& si, long& sk) {
  const long ld = layout == 2 ? n + 3 : (layout == 1 ? (K | 1) : ((K + 1) & ~1) + 2);
  std::vector<double> out((size_t)ld * (layout == 2 ? K : n), 1e30);
  si = layout == 2 ? 1 : ld;
  sk = layout == 2 ? ld : 1;
  for (int i = 0; i < n; ++i)
    for (int k = 0; k < K; ++k) out[i * si + k * sk] = X[(size_t)i * K + k];
  return out;
}
static std::vector<int> scales(const std::vector<double>& X, int n, int K) {
  const int ng = (K + EM_KG - 1) / EM_KG;
  std::vector<int> e((size_t)ng * n, -2000);
  for (int i = 0; i < n; ++i)
    for (int k = 0; k < K; ++k)
      if (X[(size_t)i * K + k] != 0.0) e[(k / EM_KG) * n + i] = std::max(e[(k / EM_KG) * n + i], std::ilogb(X[(size_t)i * K + k]) + 1);
  return e;
}
template <typename T>
static T* up(const std::vector<T>& v) {
  T* p;
  cudaMalloc(&p, v.size() * sizeof(T));
  cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  return p;
}

int main() {
  int h[6];
  cudaFuncSetAttribute(product, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)EM_SOLO_SMEM);
  int* failed;
  cudaMalloc(&failed, 4);
  cudaMemset(failed, 0, 4);
  while (fread(h, 4, 6, stdin) == 6) {
    const int na = h[0], nb = h[1], K = h[2];
    if (na < 1 || na > TC_M || nb < 1 || nb > TC_N || K < 1 || K > 2048) return 2;
    std::vector<double> A((size_t)na * K), B((size_t)nb * K), C((size_t)na * nb);
    if (fread(A.data(), 8, A.size(), stdin) != A.size() || fread(B.data(), 8, B.size(), stdin) != B.size()) return 2;
    long sai, sak, sbj, sbk;
    double *dA = up(lay(A, na, K, h[3], sai, sak)), *dB = up(lay(B, nb, K, h[4], sbj, sbk)), *dC = up(C);
    int *ea = up(scales(A, na, K)), *eb = up(scales(B, nb, K));
    product<<<1, EM_NT, EM_SOLO_SMEM>>>(dA, sai, sak, na, dB, sbj, sbk, nb, K, h[5] ? ea : nullptr, h[5] ? eb : nullptr,
                                        dC, failed);
    if (cudaMemcpy(C.data(), dC, C.size() * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    int bad = 0;
    cudaMemcpy(&bad, failed, 4, cudaMemcpyDeviceToHost);
    if (bad) return 4;
    fwrite(C.data(), 8, C.size(), stdout);
    cudaFree(dA); cudaFree(dB); cudaFree(dC); cudaFree(ea); cudaFree(eb);
  }
  return 0;
}
