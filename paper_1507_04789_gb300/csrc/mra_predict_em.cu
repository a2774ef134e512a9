// mra_predict_em.cu -- posterior predictive mean and variance (Sec. 3.4, Prop. 2)
// with the products on the emulation engine, for handles of MRA_PREC_EMU.
//
// The same quantities as predict_kernel (mra_predict.cu), whose 2^18 points at
// n = 2^18, r = 64 take 121 ms of the FP64 pipe (0.86 of its 1.06 TFLOP/s) and
// 29 ms here, where the digit splitting (integer pipe) bounds the products.  One
// CTA takes up to 128 points of one level-(M-1) region: the chain and the
// posterior recursion read the region's ancestors, which its leaves share, as
// one 128-row product per block; only the leaf term goes leaf by leaf.
#include <algorithm>

#include "mra_emu.cuh"
#include "mra_launch.h"

namespace mra {

constexpr int PE_GMAX = 6;   // 128-column groups of a row of at most MRA_MAX_M x MAX_R_DEV = 768 columns

__global__ void __launch_bounds__(EM_NT) predict_kernel_em(const Desc* __restrict__ D, PredState ps, int tiles,
                                                           int* status) {
  constexpr int NTH = EM_NT;
  extern __shared__ __align__(1024) unsigned char dsm[];
  __shared__ __align__(8) uint64_t mbar[EM_MBARS];
  __shared__ uint32_t tmem_slot;
  __shared__ int fail;
  __shared__ __align__(16) int rexp[EM_REXP], cexp[EM_CEXP];
  // row scales: of Uhat per 128-column group, of the current X^l, C0, P or Y rows, of the Bhat block the
  // recursion takes next; of the leaf's rows of H per group
  __shared__ int usc[PE_GMAX * TC_M], xsc[TC_M], bsc[TC_M], hs[PE_GMAX * TC_N];
  __shared__ double px[TC_M], py[TC_M], mu[TC_M], va[TC_M], ax[MAX_R_DEV], ay[MAX_R_DEV], c0gp[TC_M], c0gq[C0_GMAX];
  __shared__ unsigned char qcol[MAX_R_DEV], qrow[MAX_R_DEV];
  const Desc& ds = D[ps.desc];
  const Shape sh = ds.sh;
  const Cov cv = ds.cv;
  const LevelState& st = ds.st;
  const LeafState& lf = ds.lf;
  const int M = sh.M, r = sh.r, Mr = M * r, ng = (Mr + EM_KG - 1) / EM_KG, lb = leaf_bits(sh);
  const long pm = (ps.leaf0 >> lb) + blockIdx.x / tiles;   // Morton id of the region
  const long row1 = ps.off[(pm + 1) << lb];
  const long t0 = ps.off[pm << lb] + (long)(blockIdx.x % tiles) * TC_M;
  if (t0 >= row1) return;
  const int na = (int)min((long)TC_M, row1 - t0);
  const int dM = lvl_depth(sh.hx, sh.hy, M - 1);
  for (int l = 0; l < M; ++l)
    if (st.cid[l][pm >> (dM - lvl_depth(sh.hx, sh.hy, l))] < 0) {   // pruned tree: no data above these points
      long F = pm << lb;
      while (ps.off[F + 1] <= t0) ++F;
      if (threadIdx.x == 0) flag_error(status, ST_ARG, l, F);
      return;
    }
  const long P = st.cid[M - 1][pm];
  const int ldp = ds.nlmax + 1;
  double* Ps = reinterpret_cast<double*>(dsm + EM_STAGE_BYTES);   // rows x ldp: C0(S^P, S_F), then P
  // c0_fast in the chain (Ps is free then): squared scaled offsets of the points to the knot grid's columns and rows
  double* c0dx = Ps;
  double* c0dy = c0dx + TC_M * C0_GMAX;
  const int gx = sh.gx, gy = sh.gy;
  const bool fast = c0_fast_ok(cv, gx, gy);
  const double c0s = c0_scale(cv), c0s2 = c0s * c0s;
  for (int q = threadIdx.x; q < r; q += NTH) {
    qcol[q] = (unsigned char)(q % gx);
    qrow[q] = (unsigned char)(q / gx);
  }
  for (int t = threadIdx.x; t < na; t += NTH) {
    px[t] = ps.xs[t0 + t];
    py[t] = ps.ys[t0 + t];
    c0gp[t] = cv.sigma2 * c0_vfac(cv, px[t]);
  }
  for (int t = threadIdx.x; t < PE_GMAX * TC_M; t += NTH) usc[t] = -2000;
  for (int t = threadIdx.x; t < TC_M; t += NTH) bsc[t] = -2000;
  EmCtx cx;
  cx.stage = reinterpret_cast<uint16_t*>(dsm);
  cx.rexp = rexp;
  cx.cexp = cexp;
  cx.mbar = mbar;
  cx.fail = &fail;
  em_init(cx, &tmem_slot);
  double* U = ps.U + t0 * Mr;
  bool ok = true;
  EmRows q{};
  // four lanes a row: sums over columns [0, n) of x(c) w(c) and x(c)^2, to the row's four lanes (every lane calls it)
  const int srow = threadIdx.x >> 2, sq = threadIdx.x & 3;
  auto row_sums = [&](const double* x, const double* w, int n, double& s1, double& s2) {
    s1 = s2 = 0.0;
    for (int c = sq; c < n; c += 4) {
      const double v = x[c];
      if (w) s1 = fma(v, w[c], s1);
      s2 = fma(v, v, s2);
    }
    s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
    s2 += __shfl_xor_sync(0xffffffffu, s2, 1);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 2);
    s2 += __shfl_xor_sync(0xffffffffu, s2, 2);
  };
  // ---- Uhat chain --------------------------------------------------------------
  for (int l = 0; l < M && ok; ++l) {
    const long a = ancestor(st, M - 1, P, l);
    __syncthreads();
    load_knots<NTH>(sh, l, st.mort[l][a], ax, ay);
    const double* Vanc = st.V[l] + a * (long)r * (l * r);
    for (int t = threadIdx.x; t < TC_M; t += NTH) xsc[t] = -2000;
    __syncthreads();
    if (fast) {
      const int gs = gx + gy;
      for (int t = threadIdx.x; t < na * gs; t += NTH) {
        const int i = t / gs, c = t - i * gs;
        const double d = c < gx ? c0s * (px[i] - ax[c]) : c0s * (py[i] - ay[(c - gx) * gx]);
        (c < gx ? c0dx + i * gx + c : c0dy + i * gy + (c - gx))[0] = d * d;
      }
      for (int c = threadIdx.x; c < gx; c += NTH) c0gq[c] = c0_vfac(cv, ax[c]);
      __syncthreads();
    }
    for (int t = threadIdx.x; t < na * r; t += NTH) {
      const int i = t / r, j = t - i * r;
      const double v = fast ? c0_fast(cv.family, c0dx[i * gx + qcol[j]] + c0dy[i * gy + qrow[j]],
                                      cv.nonstat ? c0gp[i] * c0gq[qcol[j]] : cv.sigma2)
                            : cov0(cv, px[i], py[i], ax[j], ay[j]);
      U[(long)i * Mr + l * r + j] = v;
      if (l == 0) atomicMax(xsc + i, xexp_of(v));
    }
    if (l > 0) {
      const int* vsa = st.vexp[l] + a * (long)((l * r + 127) / 128) * r;
      q = EmRows{U, Mr, 1, na, Vanc, l * r, 1, r, l * r, usc, TC_M, vsa, r, U + l * r, Mr, true, xsc, 0, nullptr, 0};
      ok = em_rows(&cx, &q);
      if (!ok) break;
    }
    q = EmRows{U + l * r, Mr, 1, na, st.Li[l] + a * (long)r * r, r, 1, r, r, xsc, 0, st.liexp[l] + a * r, 0, U + l * r, Mr,
               false, nullptr, 0, usc, l * r};
    ok = em_rows(&cx, &q);
  }
  __syncthreads();
  // ---- prior variance v^P = C0(s, s) - |Uhat row|^2 --------------------------
  {
    double s1 = 0.0, s2 = 0.0;
    row_sums(U + (long)srow * Mr, nullptr, srow < na ? Mr : 0, s1, s2);
    if (srow < na && sq == 0) {
      va[srow] = cov0(cv, px[srow], py[srow], px[srow], py[srow]) - s2;
      mu[srow] = 0.0;
    }
  }
  // ---- leaf term, leaf by leaf: P = C0(S^P, S_F) L_Sigma^{-T} - Uhat H_F', then Bhat^M = Uhat - P H_F ----
  for (long F = pm << lb; F < (pm + 1) << lb && ok; ++F) {
    const int ra = (int)(max(ps.off[F], t0) - t0), rb = (int)(min(ps.off[F + 1], t0 + na) - t0), nP = rb - ra;
    if (nP <= 0) continue;                       // (uniform)
    const long o0 = lf.off[F];
    const int nF = (int)(lf.off[F + 1] - o0);
    double* Us = U + (long)ra * Mr;
    if (nF == 0) {                               // the scales of Bhat^{M,M-1} = Uhat^{M-1}
      for (int t = threadIdx.x; t < nP * r; t += NTH)
        atomicMax(bsc + ra + t / r, xexp_of(Us[(long)(t / r) * Mr + (M - 1) * r + t % r]));
      continue;
    }
    const double* LS = lf.LS + lf.sq_off[F];
    const double* HF = lf.H + o0 * Mr;
    const long cl = st.cid[M][F];
    __syncthreads();                             // the previous leaf's P and scales are no longer read
    for (int t = threadIdx.x; t < TC_M; t += NTH) xsc[t] = -2000;
    __syncthreads();
    const bool ff = c0_fast_ok(cv, 1, 1);
    for (int t = threadIdx.x; t < nP * nF; t += NTH) {
      const int i = t / nF, k = t - i * nF;
      const double x = lf.xs[o0 + k], y = lf.ys[o0 + k];
      double v;
      if (ff) {
        const double dx = px[ra + i] - x, dy = py[ra + i] - y;
        v = c0_fast(cv.family, c0s2 * fma(dx, dx, dy * dy), cv.nonstat ? c0gp[ra + i] * c0_vfac(cv, x) : cv.sigma2);
      } else {
        v = cov0(cv, px[ra + i], py[ra + i], x, y);
      }
      Ps[i * ldp + k] = v;
      atomicMax(xsc + i, xexp_of(v));
    }
    // column tiles from the last: L_Sigma^{-1} is lower triangular, so a tile's product reads the columns of
    // C0 up to its own, which its result replaces
    for (int ct = (nF - 1) / TC_N; ct >= 0 && ok; --ct) {
      const int b0 = ct * TC_N, nb = min(TC_N, nF - b0);
      q = EmRows{Ps, ldp, 1, nP, LS + (long)b0 * nF, nF, 1, nb, b0 + nb, xsc, 0, nullptr, 0, Ps + b0, ldp, false, nullptr, 0,
                 nullptr, 0};
      ok = em_rows(&cx, &q);
      if (!ok) break;
      for (int t = threadIdx.x; t < ng * TC_N; t += NTH) {
        const int g = t / TC_N, j = t - g * TC_N;
        hs[t] = j < nb ? lf.hrow[(o0 + b0 + j) * ng + g] : -2000;
      }
      q = EmRows{Us, Mr, 1, nP, HF + (long)b0 * Mr, Mr, 1, nb, Mr, usc + ra, TC_M, hs, TC_N, Ps + b0, ldp, true, nullptr, 0,
                 nullptr, 0};
      ok = em_rows(&cx, &q);
    }
    if (!ok) break;
    __syncthreads();
    for (int t = threadIdx.x; t < TC_M; t += NTH) xsc[t] = -2000;
    __syncthreads();
    for (int t = threadIdx.x; t < nP * nF; t += NTH) atomicMax(xsc + t / nF, xexp_of(Ps[(t / nF) * ldp + t % nF]));
    {
      double s1 = 0.0, s2 = 0.0;
      row_sums(Ps + srow * ldp, lf.z + o0, srow < nP ? nF : 0, s1, s2);
      if (srow < nP && sq == 0) {
        mu[ra + srow] += s1;
        va[ra + srow] -= s2;
      }
    }
    for (int cb = 0; cb < Mr && ok; cb += TC_N) {
      const int nbc = min(TC_N, Mr - cb);
      q = EmRows{Ps, ldp, 1, nP, HF + cb, 1, Mr, nbc, nF, xsc, 0, lf.hcol + cl * (long)Mr + cb, 0, Us + cb, Mr, true,
                 bsc + ra, Mr - r - cb, nullptr, 0};
      ok = em_rows(&cx, &q);
    }
  }
  // ---- posterior basis recursion, l = M-1..0 -----------------------------------
  for (int l = M - 1; l >= 0 && ok; --l) {
    const long a = ancestor(st, M - 1, P, l);
    __syncthreads();
    for (int t = threadIdx.x; t < TC_M; t += NTH) xsc[t] = -2000;
    // Y_l, in place of Bhat^l (no longer read)
    q = EmRows{U + l * r, Mr, 1, na, st.Lt[l] + a * (long)r * r, r, 1, r, r, bsc, 0, nullptr, 0, U + l * r, Mr, false, xsc, 0,
               nullptr, 0};
    ok = em_rows(&cx, &q);
    if (!ok) break;
    for (int t = threadIdx.x; t < TC_M; t += NTH) bsc[t] = -2000;
    __syncthreads();
    {
      double s1 = 0.0, s2 = 0.0;
      row_sums(U + (long)srow * Mr + l * r, st.gv[l] + a * r, srow < na ? r : 0, s1, s2);
      if (srow < na && sq == 0) {
        mu[srow] += s1;
        va[srow] += s2;
      }
    }
    const int lr = l * r;
    const double* Gl = st.G[l] + a * (long)r * lr;
    for (int cb = 0; cb < lr && ok; cb += TC_N) {
      const int nbc = min(TC_N, lr - cb);
      q = EmRows{U + lr, Mr, 1, na, Gl + cb, 1, lr, nbc, r, xsc, 0, st.gcol[l] + a * (long)lr + cb, 0, U + cb, Mr, true, bsc,
                 lr - r - cb, nullptr, 0};                       // (block l - 1: its last update)
      ok = em_rows(&cx, &q);
    }
  }
  em_release(cx);
  if (!ok) {
    if (threadIdx.x == 0) flag_error(status, ST_TIMEOUT, M - 1, P);
    return;
  }
  for (int t = threadIdx.x; t < na; t += NTH) {
    const long orig = ps.perm[t0 + t];
    ps.mean[orig] = mu[t];
    ps.var[orig] = va[t];
  }
}

static size_t predict_em_smem(int nlmax) {
  return EM_STAGE_BYTES + sizeof(double) * std::max((size_t)TC_M * (nlmax + 1), (size_t)2 * TC_M * C0_GMAX);
}

// Whether the marginal prediction of np points on an emulated handle (n observations) runs on the engine.
// A product costs the engine about the same for one row as for 128, the FP64 kernel pays by 16-row tiles (of
// 32 columns for r <= 32, else 64) and by the observations a leaf, and a region is one CTA where its leaves
// are four: few points a leaf, small blocks on sparse leaves and trees with fewer regions than SMs stay on the
// FP64 kernel.  The line is where the engine is first faster for points over the whole domain and (to a tenth
// of a millisecond) over a sixteenth of it.  FP64 / engine, kernel times at so many points a leaf (domain,
// sixteenth):
//   1024 regions: r = 17: 24 1.20, 1.39, 16 0.97, 1.41;  25: 16 1.14, 1.70, 4 0.82, 1.21;  33: 1 1.27, 1.48, 0.5
//     1.02, 0.91;  49: 0.5 1.19, 1.00;  64: 0.5 1.28, 1.44.
//   256 regions: 25: 16 1.13, 1.86, 4 0.75, 1.21;  33: 4 1.41, 1.86, 2 1.17, 0.96, 1 1.09, 0.80;
//     49: 1 1.25, 0.88;  64: 2 1.54, 1.22, 1 1.42, 0.98.
//   64 regions: 17: 96 1.10, 1.21, 64 0.96, 1.58;  25: 64 0.96 to 1.08, 1.64;  33: 16 1.20, 2.76, 8 0.73, 1.38;
//     64: 16 1.63, 1.78, 8 0.94, 1.79.
//   16 regions: 32: 256 1.62, 1.75, 128 1.01, 1.38;  33: 64 1.17, 1.42, 32 0.74, 1.45.
//   4 regions: 33: 1024 2.18, 2.86, 512 (6 observations a leaf) 0.94;  49: 256 1.33, 1.66.
//   1 region: 33: 4096 1.67, 2.53 (6 observations a leaf 1.17), 1024 0.92, 1.32;  48: 1024 (6) 0.73.
// r <= 32 stays on the FP64 kernel below M r = 96 columns (r = 17, M = 4 or 5, 24 to 30 observations a leaf: 0.90
// to 0.95 at the line and above), with fewer than 16 regions (0.77 to 1.5 whatever the points) and on leaves of
// few observations (6: 64 regions, r = 17 0.81, 512 regions 0.78; but 1024 regions, r = 25 1.27).  Regions of two
// leaves (J_M = 2) hold half the points: r = 33, 256 regions 16 1.55, 8 0.92, 1024 regions 4 1.10, 2 0.98; r = 17,
// 256 regions 64 1.22, 16 0.85: eight times the line.
//   The grid holds the tiles of the fullest leaf for every region, and an empty CTA costs about 25 ns (one
// of the FP64 kernel's 1 ns): points crowded into so few regions that more than 64 times the tiles needed
// would be launched stay on the FP64 kernel (r = 17, 16 a leaf of 4096, all in one: engine 13.0 ms, FP64 8.9).
// The flat grid is 31 bits.
bool predict_on_engine(int M, int r, int lb, int max_per_leaf, long nleaf, long np, long n) {
  constexpr long NEVER = 1L << 40;
  // half points a leaf; rows: regions from 1024, 256, 64, 16, 4, 1 on; columns: r <= 24, <= 32, < 48, up to 64
  constexpr long LINE[6][4] = {{48, 32, 2, 1},       {48, 32, 5, 3},            {192, 192, 32, 32},
                               {512, 512, 128, 128}, {NEVER, NEVER, 2048, 512}, {NEVER, NEVER, 8192, 8192}};
  if (M < 1 || r <= 16 || max_per_leaf <= 0) return false;
  const long regions = nleaf >> lb;
  if (r <= 32 && (M * r < 96 || (n < 24 * nleaf && (r <= 24 || regions < 1024)))) return false;
  const int row = regions >= 1024 ? 0 : regions >= 256 ? 1 : regions >= 64 ? 2 : regions >= 16 ? 3 : regions >= 4 ? 4 : 5;
  const long line = LINE[row][r <= 24 ? 0 : r <= 32 ? 1 : r < 48 ? 2 : 3];
  if (2 * np < (lb < 2 ? 8 * line : line) * nleaf) return false;
  const long tiles = (((long)max_per_leaf << lb) + TC_M - 1) / TC_M;
  return regions * tiles <= 64 * (np / TC_M + regions) && regions * tiles < (1L << 31);
}

cudaError_t launch_predict_em(const Desc* d_desc, int lb, int nlmax, const PredState& ps, int max_per_leaf, long nleaf,
                              int* status, cudaStream_t s, int64_t* launches, Timer* tm) {
  const int tiles = (int)((((long)max_per_leaf << lb) + TC_M - 1) / TC_M);
  const size_t sm = std::max(predict_em_smem(nlmax), EM_SOLO_SMEM);
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(predict_kernel_em, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm))) return e;
  tm->start(5, s);
  predict_kernel_em<<<(unsigned)((nleaf >> lb) * tiles), EM_NT, sm, s>>>(d_desc, ps, tiles, status);
  tm->stop(s);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace mra
