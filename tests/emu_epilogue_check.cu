// The FP64-emulation engine's product and what its kernels do with it, on the GPU:
//   out(i, j) = P(i, j)  or  out(i, j) -= P(i, j),   P = A B'
// written by the inlined row helpers (form 0) and by em_rows, a call, into global
// (form 1) or shared memory (form 2).  Reads from stdin
//   na nb K ldo off sub form xe0 gcol   (int32), then A (na x K), B (nb x K) and out (na x nb), row-major doubles;
// out lies at its buffer + off with row stride ldo, GUARD doubles of POISON around it and POISON between its rows.
// Writes the whole buffer, then (form 1, 2) xe (128) and ge (2 x 128) as int32.
#include <cstdio>
#include <vector>
#include "../paper_1507_04789_gb300/csrc/mra_emu.cuh"

using namespace mra;

constexpr int GUARD = 4096;
constexpr double POISON = -1.2345678901234567e+250;
constexpr int OUT_SMEM_DOUBLES = TC_M * (TC_N + 5) + 8;      // form 2: the rows in shared memory
constexpr int SMEM = EM_STAGE_BYTES + OUT_SMEM_DOUBLES * 8;

__global__ void __launch_bounds__(EM_NT) product(const double* A, int na, const double* B, int nb, int K, double* out,
                                                 int ldo, int off, int sub, int form, int xe0, int gcol, int* xe, int* failed) {
  extern __shared__ __align__(1024) unsigned char dsm[];
  __shared__ __align__(8) uint64_t mbar[EM_MBARS];
  __shared__ uint32_t slot;
  __shared__ int fail;
  __shared__ __align__(16) int rexp[EM_REXP], cexp[EM_CEXP];
  __shared__ int xs[TC_M], gs[2 * TC_M];
  EmCtx cx;
  cx.stage = reinterpret_cast<uint16_t*>(dsm);
  cx.rexp = rexp;
  cx.cexp = cexp;
  cx.mbar = mbar;
  cx.fail = &fail;
  em_init(cx, &slot);
  for (int t = threadIdx.x; t < TC_M; t += EM_NT) xs[t] = gs[t] = gs[TC_M + t] = -2000;
  double* o = out + GUARD + off;
  double* so = reinterpret_cast<double*>(dsm + EM_STAGE_BYTES) + (off & 3);
  if (form == 2)
    for (int t = threadIdx.x; t < na * ldo; t += EM_NT) so[t] = o[t];
  __syncthreads();
  bool ok;
  if (form == 0) {
    EmAcc acc;
    ok = em_mma(cx, acc, A, K, 1, na, B, K, 1, nb, K);
    const int row = acc.row(), c0 = acc.col0();
    if (ok && row < na) {
      double* const p = o + (long)row * ldo + c0;
      if (sub) {
        double v[EmAcc::NC];
        em_get<EmAcc::NC>(p, nb - c0, v);
#pragma unroll
        for (int c = 0; c < EmAcc::NC; ++c) acc.v[c] = v[c] - acc.v[c];
      }
      em_put<EmAcc::NC>(p, nb - c0, acc.v);
    }
  } else {
    const EmRows q{A, K, 1, na, B, K, 1, nb, K, nullptr, 0, nullptr, 0, form == 2 ? so : o, ldo, sub != 0, xs, xe0, gs, gcol};
    ok = em_rows(&cx, &q);
  }
  __syncthreads();
  if (form == 2)
    for (int t = threadIdx.x; t < na * ldo; t += EM_NT) o[t] = so[t];
  for (int t = threadIdx.x; t < TC_M; t += EM_NT) {
    xe[t] = xs[t];
    xe[TC_M + t] = gs[t];
    xe[2 * TC_M + t] = gs[TC_M + t];
  }
  em_release(cx);
  if (!ok && threadIdx.x == 0) *failed = 1;
}

template <typename T>
static T* up(const std::vector<T>& v) {
  T* p = nullptr;
  if (cudaMalloc(&p, v.size() * sizeof(T)) || cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice)) exit(3);
  return p;
}

int main() {
  int h[9];
  if (cudaFuncSetAttribute(product, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM)) return 3;
  while (fread(h, 4, 9, stdin) == 9) {
    const int na = h[0], nb = h[1], K = h[2], ldo = h[3], off = h[4], sub = h[5], form = h[6], xe0 = h[7], gcol = h[8];
    // (the rows' group exponents reach groups gcol / 128 .. (gcol + nb - 1) / 128 of two)
    if (na < 1 || na > TC_M || nb < 1 || nb > TC_N || K < 1 || K > 1024 || ldo < nb || ldo > TC_N + 5 || off < 0 || off > 3 ||
        form < 0 || form > 2 || gcol < 0 || gcol + nb > 2 * EM_KG)
      return 2;
    std::vector<double> A((size_t)na * K), B((size_t)nb * K), C((size_t)na * nb), buf(2 * GUARD + 4 + (size_t)na * ldo, POISON);
    if (fread(A.data(), 8, A.size(), stdin) != A.size() || fread(B.data(), 8, B.size(), stdin) != B.size() ||
        fread(C.data(), 8, C.size(), stdin) != C.size())
      return 2;
    for (int i = 0; i < na; ++i)
      for (int j = 0; j < nb; ++j) buf[GUARD + off + (size_t)i * ldo + j] = C[(size_t)i * nb + j];
    std::vector<int> xe(3 * TC_M), zero(1, 0);
    double *dA = up(A), *dB = up(B), *dC = up(buf);
    int *dx = up(xe), *df = up(zero);
    product<<<1, EM_NT, SMEM>>>(dA, na, dB, nb, K, dC, ldo, off, sub, form, xe0, gcol, dx, df);
    if (cudaMemcpy(buf.data(), dC, buf.size() * 8, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(xe.data(), dx, xe.size() * 4, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(zero.data(), df, 4, cudaMemcpyDeviceToHost))
      return 3;
    if (zero[0]) return 4;
    fwrite(buf.data(), 8, buf.size(), stdout);
    fwrite(xe.data(), 4, xe.size(), stdout);
    cudaFree(dA); cudaFree(dB); cudaFree(dC); cudaFree(dx); cudaFree(df);
  }
  return 0;
}
