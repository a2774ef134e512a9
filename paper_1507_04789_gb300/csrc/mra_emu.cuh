// mra_emu.cuh -- FP64-grade tile product on the tcgen05 tensor cores.
//
// GB300 retires 2 FP64 FMA per clock per SM, so FP64 contractions are emulated
// with the error-free splitting of Ozaki et al. (2012, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications"), written here for f16 tensor cores:
//
//  * every row of A and of B is scaled, per group of 128 K-columns, by a power
//    of two 2^e with |x| < 2^e over the group, rounded to the nearest multiple
//    of 2^(e - 48) and cut into S = 6 signed digits of 8 bits: x = sum_p d_p
//    2^(e - 8p), d_p integer, |d_1| <= 256, |d_p| <= 128 for p > 1, exact in
//    f16 (integers to 2048);
//  * d_p d_q products are exact and the FP32 sums of every pair with the same
//    weight t = p + q over a group stay at or below 128 (2 256 128 + 4 128^2)
//    = 2^24, so the tensor-memory accumulation is exact too; the 26 pairs with
//    t <= 8 go to 7 accumulators (one per t, up to 64 TMEM columns each);
//  * every group is drained: the 7 accumulators of a column are combined in
//    units of the leading weight (double-float, Fast2Sum for the two largest
//    corrections), scaled by 2^(e_i + f_j - 16) (exact) and added to a
//    double-float register accumulator, converted to FP64 once at the end.
//
// Signed digits carry 8 bits a slice where sign-and-magnitude slices of the
// same magnitude (|a| < 128) carry 7: 6 slices and 26 products against 7 and 28,
// with the operand error (at most 2^(e - 49)) rounded instead of truncated.  The pairs of weight 8 matter: without them (21 products,
// 2 % of an evaluation) the squares d_4^2 a Gram product drops are all positive,
// and the gradient at n = 2^16 is off by 2e-11 to 3e-10 instead of 6e-13 to 3e-12.
// So a term a b is off by at most 2^-46.5 2^(e + f) and a product by about 1e-15 of
// sum |a b| where 2^e and 2^f are within a few times the elements, while running on
// the tensor cores; only rare sums touch the FP64 pipe.  (2^e is at most twice the
// group's largest element when it comes from the scale pass; a producer's scale may
// cover more than the group, as H's column scales a whole leaf, and rows of wide
// dynamic range keep fewer bits of their small elements.)
// Range: the running sums are FP32 pairs, so |results| < 2^127, and a group
// whose scale product 2^(e_i + f_j) is below 2^-110 is dropped.
//
// Pipeline: the K range is staged in chunks of 16 (one MMA K-step) into two
// shared-memory buffers.  Warps 1..15 split: the work of a chunk is cut into
// slots of 16 rows x 16 columns, one warp each, and the warps take the slots
// of all chunks in turn, each loading its next slot's elements before it splits
// the current one.  Warp 0 issues the MMAs.  They meet in mbarriers per buffer
// (staged, free) and per group (accumulators complete, accumulators read), so
// no barrier of the whole CTA stands between two chunks.
#pragma once
#include "mra_tc.cuh"

namespace mra {

constexpr int EM_NT = 512;                    // threads per CTA of the engine's kernels
constexpr int EM_S = 6;                       // digits per operand
constexpr int EM_T = EM_S + 2;                // digit pairs (p, q) with p + q <= EM_T are formed
constexpr int EM_NA = EM_T - 1;               // accumulators, one per p + q
constexpr int EM_KC = 16;                     // staged K chunk (f16 elements) = one MMA K-step
constexpr int EM_KG = 128;                    // K group sharing one scale per row (drain period)
constexpr int EM_GCH = EM_KG / EM_KC;         // chunks per group
constexpr int EM_MAXG = 4;                    // groups whose scales one pass finds
constexpr int EM_CC = EM_KC / 8;              // 16-byte core columns (8 f16) per chunk
constexpr int EM_A_HALFS = TC_M * EM_KC;      // f16 per digit plane of A (4 KB)
constexpr int EM_B_HALFS = TC_N * EM_KC;      // (2 KB)
constexpr int EM_BUF_HALFS = EM_S * (EM_A_HALFS + EM_B_HALFS);
constexpr int EM_STAGE_BYTES = 2 * 2 * EM_BUF_HALFS;                    // two buffers: 73728
constexpr int EM_REXP = EM_MAXG * TC_M;       // ints of row scales of A (shared)
constexpr int EM_CEXP = EM_MAXG * TC_N;       // ints of row scales of B (shared)
constexpr uint32_t EM_TMEM_COLS = 512;
constexpr int EM_SLOT = 16;                   // rows of one warp's slot
constexpr int EM_SLOTS = (TC_M + TC_N) / EM_SLOT;   // slots of a full chunk, and its arrivals
constexpr int EM_EMIN = -900;                 // scales below 2^-900 are raised to it (the elements become zero)
// mbarriers: buffer b staged / free, group accumulated / read, and the last
// resort of a timed-out product
enum : int { EM_FULL = 0, EM_FREE = 2, EM_DONE = 4, EM_READ = 5, EM_LAST = 6, EM_MBARS = 7 };
// The engine takes all 512 TMEM columns of an SM; its kernels ask for more than
// half of the SM's shared memory so that a second CTA is never resident (it
// would only wait in tcgen05.alloc).
constexpr size_t EM_SOLO_SMEM = 116 * 1024;
static_assert(EM_KG * (2 * 256 * 128 + 4 * 128 * 128) <= (1 << 24), "group sums (but the least significant) must stay exact in FP32");
static_assert(EM_NA * TC_N <= (int)EM_TMEM_COLS, "accumulators exceed the tensor-memory allocation");

// kind::f16 instruction descriptor: D = F32, A = B = F16, both K-major, 128 x n.
__device__ __forceinline__ uint32_t em_idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}

// Shared-memory matrix descriptor, no swizzle, K-major core matrices of 8 rows x
// 16 bytes: 128 B between K-adjacent cores, EM_CC * 128 B between 8-row groups.
__device__ __forceinline__ uint64_t em_desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((128u >> 4) & 0x3FFF) << 16) |
         ((uint64_t)(((EM_CC * 128u) >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// Binary exponent e with |x| < 2^e (x != 0, normal); -2000 for zero.
__device__ __forceinline__ int em_exp(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int be = (int)((u >> 52) & 0x7FF);
  return be == 0 ? -2000 : be - 1022;
}

// Output ownership: thread (warp w, lane l) holds row 32 (w % 4) + l and the
// 16 columns starting at 16 (w / 4) of the 128 x 64 tile.
struct EmAcc {
  static constexpr int NC = 16;
  double v[NC];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int c = 0; c < NC; ++c) v[c] = 0.0;
  }
  __device__ __forceinline__ int row() const { return (((threadIdx.x >> 5) & 3) << 5) | (threadIdx.x & 31); }
  __device__ __forceinline__ int col0() const { return (threadIdx.x >> 7) * NC; }
};
static_assert((EM_NT / 128) * EmAcc::NC == TC_N, "the warps cover the tile's columns");

struct EmCtx {
  uint16_t* stage;   // EM_STAGE_BYTES of shared memory: two buffers of 6 A planes, then 6 B planes (of nb rows, to 16)
  int* rexp;         // EM_REXP row scales of A, [group][row], when the scale pass forms them
  int* cexp;         // EM_CEXP row scales of B
  const int* ra;     // row scales of A in use: ra[g * rs + i] (rexp or a producer's table)
  const int* cb;     // row scales of B in use: cb[g * cs + j] (the drains: cexp[g * TC_N + j])
  int rs, cs;
  uint64_t* mbar;    // EM_MBARS mbarriers
  uint32_t tmem;
  uint32_t chunks;   // chunks staged and groups drained by the products so far (uniform): the barriers' phases
  uint32_t groups;
  int* fail;
};

__device__ inline void em_init(EmCtx& cx, uint32_t* tmem_slot) {
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                 "r"(EM_TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    for (int b = 0; b < EM_MBARS; ++b) {
      const int count = b < EM_FREE ? EM_SLOTS : (b == EM_READ ? EM_NT / 32 : (b == EM_DONE ? 2 : 1));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(cx.mbar + b)), "r"(count));
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    *cx.fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  cx.tmem = *tmem_slot;
  cx.chunks = cx.groups = 0;
}

__device__ inline void em_release(EmCtx& cx) {
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(cx.tmem), "r"(EM_TMEM_COLS));
}

// Wait (bounded) until the phase of the given parity of mbarrier k completed.
// False after the limit, or once another warp gave up.
constexpr int EM_WAIT_LIMIT = 1 << 22;
__device__ __forceinline__ bool em_wait(const EmCtx& cx, int k, uint32_t parity) {
  const uint32_t a = smem_addr(cx.mbar + k);
  uint32_t done = 0;
  for (int it = 0; it < EM_WAIT_LIMIT && !done; ++it) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (!done && (it & 63) == 63 && *(volatile int*)cx.fail) break;
  }
  if (__all_sync(0xffffffffu, done != 0)) return true;   // (whole warps wait)
  *(volatile int*)cx.fail = 1;
  return false;
}

__device__ __forceinline__ void em_arrive(const EmCtx& cx, int k, uint32_t count) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(cx.mbar + k)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void em_commit(const EmCtx& cx, int k) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_addr(cx.mbar + k))
               : "memory");
}

// Row scales of the groups of K columns [K0, K0 + KS), KS <= EM_MAXG * EM_KG:
// rexp[g * TC_M + i] = max exponent of row i < na of A over group g (cexp for
// B, rows < nb).  The high words of the doubles (sign, exponent, top of the
// mantissa) are brought into the idle staging buffers with asynchronous
// copies, a slab of 64 K columns of every kept row at a time, so that one
// memory latency covers a slab; one thread per row then scans its words.
constexpr int EM_SLAB = 64;                    // K columns per slab (a divisor of EM_KG)
constexpr int EM_SLAB_LD = EM_SLAB + 1;        // padded words per row in shared memory
static_assert((TC_M + TC_N) * EM_SLAB_LD * 4 <= EM_STAGE_BYTES, "slab exceeds the staging buffers");

__device__ __forceinline__ void em_cp4(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

__device__ inline void em_scales(EmCtx& cx, const double* A, long sai, long sak, int na, const double* B, long sbj,
                                 long sbk, int nb, int K0, int KS) {
  uint32_t* words = reinterpret_cast<uint32_t*>(cx.stage);   // [row][EM_SLAB_LD]; rows of A, then of B
  const uint32_t wbase = smem_addr(words);
  const int rows = na + nb;                  // na (nb) = 0: that operand's scales come from its producer
  if (rows == 0) {
    __syncthreads();
    return;
  }
  for (int s0 = 0; s0 < KS; s0 += EM_SLAB) {
    const int sn = min(EM_SLAB, KS - s0);
    __syncthreads();                         // scratch (and, on the first slab, earlier scales) no longer read
    if (s0 == 0) {
      const int ng = (KS + EM_KG - 1) / EM_KG;
      for (int t = threadIdx.x; t < ng * (TC_M + TC_N); t += EM_NT) {
        if (t < ng * TC_M) cx.rexp[t] = -2000;
        else cx.cexp[t - ng * TC_M] = -2000;
      }
    }
    // copies: along K for row-major operands, along rows otherwise (coalesced
    // either way); an operand that already lives in shared memory is read
    // directly (the asynchronous copy takes global sources only)
    for (int q = 0; q < 2; ++q) {
      const double* X = q == 0 ? A : B;
      const long si = q == 0 ? sai : sbj, sk = q == 0 ? sak : sbk;
      const int n = q == 0 ? na : nb, r0 = q == 0 ? 0 : na;
      const bool in_smem = __isShared(X);
      const int cnt = n * sn;
      for (int t = threadIdx.x; t < cnt; t += EM_NT) {
        int i, k;
        if (sk == 1) { i = t / sn; k = t - i * sn; }
        else { k = t / n; i = t - k * n; }
        const unsigned* src = reinterpret_cast<const unsigned*>(X + (long)i * si + (long)(K0 + s0 + k) * sk) + 1;
        if (in_smem) words[(r0 + i) * EM_SLAB_LD + k] = *src;
        else em_cp4(wbase + 4u * (uint32_t)((r0 + i) * EM_SLAB_LD + k), src);
      }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_all;" ::: "memory");
    __syncthreads();
    const int g = s0 / EM_KG;
    for (int i = threadIdx.x; i < rows; i += EM_NT) {   // (the scanned rows are the kept ones)
      const uint32_t* wr = words + i * EM_SLAB_LD;
      int be = 0;
      for (int k = 0; k < sn; ++k) be = max(be, (int)((wr[k] >> 20) & 0x7FFu));
      if (be) {
        int* slot = i < na ? cx.rexp + g * TC_M + i : cx.cexp + g * TC_N + (i - na);
        *slot = max(*slot, be - 1022);       // one thread per row: no race
      }
    }
  }
  __syncthreads();
}

// |x| in units of 2^(E - 1022 - 56) (E = 1022 + e, |x| < 2^e) plus the digit
// bias: the magnitude's 56-bit window plus 128 at every digit, so that the low
// six bytes are the digits 6 (rounding, dropped) .. 2 plus 128 and the top 16
// bits the first digit plus 0x6400 (f16 1024).  Zero and subnormal x shift out
// entirely (E >= 122); shr.b64 clamps shifts of 64 and more.
__device__ __forceinline__ uint64_t em_window(double x, int E) {
  const uint32_t hw = (uint32_t)__double2hiint(x), lw = (uint32_t)__double2loint(x);
  const uint32_t d = (uint32_t)(E - (int)((hw >> 20) & 0x7FFu));
  const uint32_t mh = (__funnelshift_l(lw, hw, 3) & 0x7FFFFFu) | 0x800000u;   // (1.mantissa) 2^55
  uint64_t m = ((uint64_t)mh << 32) | (lw << 3);
  asm("shr.b64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(d));
  return m + 0x6400808080808080ull;
}

// f16x2 fused multiply-add: exact here (small integers).
__device__ __forceinline__ uint32_t em_hfma2(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// The 6 digit planes of a pair of elements (x0 low half, x1 high half) as f16x2
// words: a byte b of the window joins 0x64 to the f16 1024 + b, and one f16x2
// FMA with the signs gives sg (1024 + b) - sg 1152 = sg (b - 128) exactly (the
// first digit: minus 1024).
__device__ __forceinline__ void em_split_pair(double x0, double x1, int E, uint32_t* w) {
  const uint64_t y0 = em_window(x0, E), y1 = em_window(x1, E);
  const uint32_t h0 = (uint32_t)(y0 >> 32), l0 = (uint32_t)y0, h1 = (uint32_t)(y1 >> 32), l1 = (uint32_t)y1;
  const uint32_t sgn = __byte_perm((uint32_t)__double2hiint(x0), (uint32_t)__double2hiint(x1), 0x7632) & 0x80008000u;
  const uint32_t sg = 0x3C003C00u | sgn;              // (+-1, +-1) in f16
  const uint32_t n1 = 0xE400E400u ^ sgn;              // -1024 sg
  const uint32_t nb = 0xE480E480u ^ sgn;              // -1152 sg
  const uint32_t k64 = 0x64646464u;
  const uint32_t a = __byte_perm(h0, h1, 0x5410);     // bytes: digits 3, 2 of x0, then of x1
  const uint32_t b = __byte_perm(l0, l1, 0x7632);     // digits 5, 4
  const uint32_t c = __byte_perm(l0, l1, 0x0501);     // digit 6 (in bytes 0 and 2)
  w[0] = em_hfma2(__byte_perm(h0, h1, 0x7632), sg, n1);
  w[1] = em_hfma2(__byte_perm(a, k64, 0x4341), sg, nb);
  w[2] = em_hfma2(__byte_perm(a, k64, 0x4240), sg, nb);
  w[3] = em_hfma2(__byte_perm(b, k64, 0x4341), sg, nb);
  w[4] = em_hfma2(__byte_perm(b, k64, 0x4240), sg, nb);
  w[5] = em_hfma2((c & 0x00FF00FFu) | 0x64006400u, sg, nb);
}

// One operand of a product as its slots see it.
//
// A slot is 16 rows x 16 columns, a warp's 8 elements per lane.  Rows that are
// contiguous along K and aligned are read four elements a lane in two loads, four
// lanes to a row's 128 bytes (lane: row l / 4 and row l / 4 + 8, columns 4 (l % 4) ..):
// 8 cache lines a load, where a lane to a row took 16 and kept the L1's tag
// stage busier than anything else in the engine.  Other operands give every
// lane 8 columns of one row (row l % 16, columns 8 (l / 16) ..), so that loads
// of a K-major operand run along its rows.
struct EmOperand {
  const double* p;
  long si, sk;      // element (i, k) at p[i * si + k * sk]
  int n;            // rows kept
  bool vec;         // rows contiguous and 16-byte aligned (else: any layout)
};

__device__ __forceinline__ EmOperand em_operand(const double* p, long si, long sk, int n) {
  return EmOperand{p, si, sk, n, sk == 1 && (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (si & 1) == 0};
}

// This lane's 8 elements of the slot with first row i0 and first column k0 (zero
// beyond the kept rows and beyond the K range, k1), and the scales of its rows
// from tab (0 beyond).
__device__ __forceinline__ void em_load(const EmOperand& o, const int* tab, int i0, int k0, int k1, double* x, int* e) {
  const int lane = threadIdx.x & 31;
  if (o.vec) {
    const int k = k0 + 4 * (lane & 3), kn = k1 - k;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int i = i0 + (lane >> 2) + 8 * j;
      const double* p = o.p + (long)i * o.si + k;
      double* y = x + 4 * j;
      const bool in = i < o.n;
      e[j] = in ? tab[i] : 0;
      if (in && kn >= 4) {
        const double2 u = *reinterpret_cast<const double2*>(p), v = *reinterpret_cast<const double2*>(p + 2);
        y[0] = u.x;
        y[1] = u.y;
        y[2] = v.x;
        y[3] = v.y;
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) y[c] = in && c < kn ? p[c] : 0.0;
      }
    }
  } else {
    const int i = i0 + (lane & 15), k = k0 + 8 * (lane >> 4), kn = i < o.n ? k1 - k : 0;
    const double* p = o.p + (long)i * o.si + (long)k * o.sk;
    e[0] = e[1] = i < o.n ? tab[i] : 0;
    if (kn >= 8) {
#pragma unroll
      for (int c = 0; c < 8; ++c) x[c] = p[(long)c * o.sk];
    } else {
#pragma unroll
      for (int c = 0; c < 8; ++c) x[c] = c < kn ? p[(long)c * o.sk] : 0.0;
    }
  }
}

// Split a slot's elements and store their digit planes (pstride f16 apart) from
// `planes`, where the operand's row 0 lies.
__device__ __forceinline__ void em_split_slot(const EmOperand& o, int i0, const double* x, const int* e,
                                              uint16_t* planes, int pstride) {
  const int lane = threadIdx.x & 31;
  const int E0 = max(e[0], EM_EMIN) + 1022, E1 = max(e[1], EM_EMIN) + 1022;
  uint32_t w[4][EM_S];
  em_split_pair(x[0], x[1], E0, w[0]);
  em_split_pair(x[2], x[3], E0, w[1]);
  em_split_pair(x[4], x[5], E1, w[2]);
  em_split_pair(x[6], x[7], E1, w[3]);
  uint16_t* d = planes + (i0 >> 3) * EM_CC * 64;   // (i0 is a multiple of 16)
  if (o.vec) {
    const int l = lane & 3;
    d += (l >> 1) * 64 + (lane >> 2) * 8 + (l & 1) * 4;
#pragma unroll
    for (int s = 0; s < EM_S; ++s) {
      const uint32_t q = smem_addr(d + s * pstride);
      asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(q), "r"(w[0][s]), "r"(w[1][s]) : "memory");
      asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(q + EM_CC * 128), "r"(w[2][s]), "r"(w[3][s]) : "memory");
    }
  } else {
    d += ((lane >> 3) & 1) * EM_CC * 64 + (lane >> 4) * 64 + (lane & 7) * 8;
#pragma unroll
    for (int s = 0; s < EM_S; ++s)
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(smem_addr(d + s * pstride)), "r"(w[0][s]), "r"(w[1][s]),
                   "r"(w[2][s]), "r"(w[3][s])
                   : "memory");
  }
}

__device__ __forceinline__ void em_issue(uint32_t tmem, uint64_t da, uint64_t db, uint32_t accumulate,
                                         uint32_t idesc = em_idesc(TC_N)) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Issue the digit-pair products of one staged chunk (one thread; stage: the
// buffer's shared-memory address).  The B planes of nbp rows follow each other,
// and so do the accumulators of nbp columns: digit p of A times the digits
// 1 .. min(6, 8 - p) of B is one product of that many times nbp columns into the
// accumulators from p on, cut at 256 columns.  So 10 MMAs of up to 256 columns do
// the work of 26 of 64, which took the issuing thread 86 cycles each on a busy
// SM and read A from shared memory 26 times.  (A group's first chunk sets the
// accumulators: the last one, which digit 2 is the first to touch, by its own MMA.)
__device__ __forceinline__ void em_issue_chunk(const EmCtx& cx, uint32_t stage, int nbp, bool gfirst) {
  // plane descriptors differ only in the start-address field (addr >> 4, 14 bits; shared memory
  // addresses stay below 2^18, so the offsets below never carry out of the field)
  const uint64_t da0 = em_desc(stage), db0 = em_desc(stage + 2 * EM_S * EM_A_HALFS);
#pragma unroll
  for (int p = 1; p <= EM_S; ++p) {
    const uint64_t da = da0 + (uint64_t)(((p - 1) * EM_A_HALFS * 2) >> 4);
    const uint32_t dt = cx.tmem + (uint32_t)((p - 1) * nbp), ac = gfirst && p == 1 ? 0u : 1u;
    const bool own = gfirst && p == EM_T - EM_S;
    const int cols = nbp * (min(EM_S, EM_T - p) - (own ? 1 : 0));
    em_issue(dt, da, db0, ac, em_idesc(min(cols, 256)));
    if (p <= EM_T - 5 && cols > 256)               // (a row of a plane is 32 bytes)
      em_issue(dt + 256, da, db0 + 256 * 2, ac, em_idesc(cols - 256));
    if (own) em_issue(dt + cols, da, db0 + (uint64_t)(cols * 2), 0u, em_idesc(nbp));
  }
}

__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float v) {
  const float s = hi + v;
  const float bb = s - hi;
  const float err = (hi - (s - bb)) + (v - bb);
  hi = s;
  lo += err;
}

__device__ __forceinline__ void em_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// Add the group with row scale ei and column scales cexp[c0 + c] (shared memory,
// 16-byte aligned; columns beyond nb are discarded) to the running double-float
// sums (hi, lo) of this thread's 16 columns (first: the sums are set).
__device__ inline void em_drain(const EmCtx& cx, const int* cexp, int ei, int c0, int na, int nb, int nbp, bool first,
                                float* hi, float* lo) {
  const int wq = (threadIdx.x >> 5) & 3;
  if (wq * 32 >= na) return;                         // warp-uniform: every row of this warp is discarded
  const uint32_t base = cx.tmem + ((uint32_t)wq << 21);
#pragma unroll
  for (int cb = 0; cb < EmAcc::NC; cb += 8) {
    if (c0 + cb >= nb) break;                        // warp-uniform
    uint32_t v[EM_NA][8];
#pragma unroll
    for (int t = 0; t < EM_NA; ++t) em_ld8(base + (uint32_t)(t * nbp + c0 + cb), v[t]);
    int f[8];
    *reinterpret_cast<int4*>(f) = *reinterpret_cast<const int4*>(cexp + c0 + cb);
    *reinterpret_cast<int4*>(f + 4) = *reinterpret_cast<const int4*>(cexp + c0 + cb + 4);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      // group value in units of 2^(e_i + f_j - 16): sum_t v_t 2^(-8 (t - 2)).  The v_t are integers of at
      // most 2^24, so that Fast2Sum (Dekker 1971) is exact in both steps whichever operand is larger: where
      // the second one is, both lie on a grid that leaves their sum's rounding representable
      const float v0 = __uint_as_float(v[0][c]), v1 = __uint_as_float(v[1][c]), v2 = __uint_as_float(v[2][c]);
      const float s1 = fmaf(v1, 0x1p-8f, v0), r1 = fmaf(v1, 0x1p-8f, -(s1 - v0));
      const float gh = fmaf(v2, 0x1p-16f, s1), r2 = fmaf(v2, 0x1p-16f, -(gh - s1));
      float tail = __uint_as_float(v[EM_NA - 1][c]);
#pragma unroll
      for (int t = EM_NA - 2; t >= 3; --t) tail = fmaf(tail, 0x1p-8f, __uint_as_float(v[t][c]));
      const float gl = fmaf(tail, 0x1p-24f, r1 + r2);
      const int e = ei + f[c] + (127 - 16);
      const float s = (uint32_t)(e - 1) < 254u ? __int_as_float(e << 23) : 0.0f;
      if (first) {
        hi[cb + c] = gh * s;
        lo[cb + c] = gl * s;
      } else {
        two_sum_add(hi[cb + c], lo[cb + c], gh * s);
        lo[cb + c] = fmaf(gl, s, lo[cb + c]);
      }
    }
  }
}

// Exact float -> double by bit moves (subnormal floats, below 2^-126, become 0).
__device__ __forceinline__ double em_widen(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t e = (u >> 23) & 0xFFu;
  if (e == 0) return 0.0;
  const uint32_t de = e == 0xFFu ? 0x7FFu : e + 896u;          // 1023 - 127
  const uint32_t hi = (u & 0x80000000u) | (de << 20) | ((u >> 3) & 0xFFFFFu);
  return __hiloint2double((int)hi, (int)(u << 29));
}

// hi + lo rounded to FP64, on the FP32 and integer pipes: after a TwoSum |lo| is
// at most half an ulp of hi, so lo is an integer number k of FP64 ulps of hi
// (|k| <= 2^28, rounded to nearest even) and the sum's bits are hi's plus or minus
// k.  (8192 DADD take 2.5 us on the narrow FP64 pipe.)  Powers of two, below
// which the ulp halves, and |hi| < 2^-75 take the DADD.
__device__ __forceinline__ double em_sum(float a, float b) {
  const float hi = a + b, t = hi - a;
  const float lo = (a - (hi - t)) + (b - t);
  const uint32_t u = __float_as_uint(hi), m = u & 0x7FFFFFFFu;
  if (m == 0u) return 0.0;
  if ((m & 0x7FFFFFu) == 0u || m < (52u << 23) || m >= 0x7F800000u) return em_widen(hi) + em_widen(lo);
  const float ulps = lo * __uint_as_float((306u << 23) - (m & 0x7F800000u));   // lo 2^(52 - exponent of hi)
  const int k = __float2int_rn(__uint_as_float(__float_as_uint(ulps) ^ (u & 0x80000000u)));
  const long long d = ((long long)m << 29) + (896LL << 52) + k;
  return __longlong_as_double(d | (long long)((unsigned long long)(u & 0x80000000u) << 32));
}

// acc(i, j) = sum_k A(i, k) B(j, k) with FP64-grade accuracy, i < na <= 128,
// j < nb <= 64 (acc is overwritten).  Returns false (uniformly) if a
// tensor-core wait timed out.  Opens and ends with a barrier of the CTA.
//
// pa / pb, when not null, hold the operands' row scales from their producers:
// pa[g * pas + i] = the exponent e with |A(i, k)| < 2^e over K group g (any
// upper bound a producer can form cheaply, e.g. a maximum over a superset of
// the group's columns); the scale pass then skips that operand.
__device__ inline bool em_mma(EmCtx& cx, EmAcc& acc, const double* A, long sai, long sak, int na, const double* B,
                              long sbj, long sbk, int nb, int K, const int* pa = nullptr, int pas = 0,
                              const int* pb = nullptr, int pbs = 0) {
  const int row = acc.row(), c0 = acc.col0();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float hi[EmAcc::NC], lo[EmAcc::NC];
#pragma unroll
  for (int c = 0; c < EmAcc::NC; ++c) hi[c] = lo[c] = 0.f;
  const EmOperand oa = em_operand(A, sai, sak, na), ob = em_operand(B, sbj, sbk, nb);
  const int sa = (na + EM_SLOT - 1) / EM_SLOT, ns = sa + (nb + EM_SLOT - 1) / EM_SLOT;   // slots of a chunk
  const int nbp = ((nb + 15) >> 4) << 4;           // rows of a B plane, columns of an accumulator
  bool ok = true;
  for (int K0 = 0; K0 < K && ok; K0 += EM_MAXG * EM_KG) {
    const int KS = min(EM_MAXG * EM_KG, K - K0);
    const int g0 = K0 / EM_KG;
    cx.ra = pa ? pa + g0 * pas : cx.rexp;
    cx.rs = pa ? pas : TC_M;
    cx.cb = pb ? pb + g0 * pbs : cx.cexp;
    cx.cs = pb ? pbs : TC_N;
    em_scales(cx, A, sai, sak, pa ? 0 : na, B, sbj, sbk, pb ? 0 : nb, K0, KS);
    const int nch = (KS + EM_KC - 1) / EM_KC, ngr = (KS + EM_KG - 1) / EM_KG;
    const uint32_t n0 = cx.chunks, m0 = cx.groups;
    // the accumulators of group g: wait, add them to the sums, hand them back
    auto drain = [&](int g) {
      if (!em_wait(cx, EM_DONE, (m0 + g) & 1u)) return false;
      asm volatile("tcgen05.fence::after_thread_sync;");
      em_drain(cx, cx.cexp + g * TC_N, row < na ? cx.ra[g * cx.rs + row] : -2000, c0, na, nb, nbp, K0 + g == 0,
               hi, lo);
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0) em_arrive(cx, EM_READ, 1);
      return true;
    };
    if (warp == 0) {
      if (pb) {                                  // the drains read the column scales from shared memory
        for (int t = lane; t < ngr * TC_N; t += 32)
          if ((t & (TC_N - 1)) < nb) cx.cexp[t] = cx.cb[(t / TC_N) * cx.cs + (t & (TC_N - 1))];
        __syncwarp();
      }
      for (int c = 0; c < nch && ok; ++c) {
        const uint32_t n = n0 + c;
        const int b = (int)(n & 1u), g = c / EM_GCH;
        const bool gfirst = c % EM_GCH == 0;
        ok = em_wait(cx, EM_FULL + b, (n >> 1) & 1u);
        if (ok && gfirst && m0 + g > 0) ok = em_wait(cx, EM_READ, (m0 + g - 1) & 1u);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const bool glast = (c + 1) % EM_GCH == 0 || c + 1 == nch;
        if (lane == 0) {
          em_issue_chunk(cx, smem_addr(cx.stage) + (uint32_t)(b * 2 * EM_BUF_HALFS), nbp, gfirst);
          em_commit(cx, EM_FREE + b);
          if (glast) {
            em_commit(cx, EM_DONE);
            em_arrive(cx, EM_DONE, 1);           // (releases the column scales written above)
          }
        }
        __syncwarp();
        if (glast) ok = drain(g);
      }
    } else {
      // The warps share out the operands in the ratio of their slots (a warp keeps
      // to one operand): slot q of chunk c is rows 16 q .. of it.  An operand of
      // sx slots a chunk gets at most 2 sx warps: a warp's next slot then lies at
      // most two chunks on, and since its own arrival held back the MMAs of the
      // chunk it staged last, the buffer's barrier is within one phase of the one
      // it waits for (a parity tells neighbouring phases apart only).
      const int wa = max(1, min(EM_NT / 32 - 2, ((EM_NT / 32 - 1) * sa + ns / 2) / ns));
      const bool isA = warp <= wa;
      const EmOperand o = isA ? oa : ob;
      const int* tab = isA ? cx.ra : cx.cb;
      const int ts = isA ? cx.rs : cx.cs, sx = isA ? sa : ns - sa;
      const int nw = min(isA ? wa : EM_NT / 32 - 1 - wa, 2 * sx), w0 = isA ? warp - 1 : warp - 1 - wa;
      const int pstride = isA ? EM_A_HALFS : nbp * EM_KC;
      uint16_t* const planes = cx.stage + (isA ? 0 : EM_S * EM_A_HALFS);
      int g = 0;
      int c = w0 >= nw ? nch : 0, q = w0;          // the slot to stage
      while (q >= sx) q -= sx, ++c;
      int cn = c, qn = q;                          // the slot to load next
      double x[8];                                 // its elements, in flight while the slot before is stored
      int e[2] = {0, 0};                           // and the scales of their rows
      auto load = [&] {
        if (cn < nch) {
          em_load(o, tab + (cn / EM_GCH) * ts, qn * EM_SLOT, K0 + cn * EM_KC, K0 + KS, x, e);
          qn += nw;
          while (qn >= sx) qn -= sx, ++cn;
        }
      };
      auto step = [&] {
        const uint32_t n = n0 + c;
        const int b = (int)(n & 1u);
        // the buffer is free once the MMAs of chunk n - 2 are done
        if (n >= 2 && !em_wait(cx, EM_FREE + b, ((n >> 1) - 1) & 1u)) return false;
        em_split_slot(o, q * EM_SLOT, x, e, planes + b * EM_BUF_HALFS, pstride);
        load();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        // (A's last slot makes up the arrivals of the slots that the product does not have)
        if (lane == 0) em_arrive(cx, EM_FULL + b, isA && q == sa - 1 ? EM_SLOTS + 1 - ns : 1);
        q += nw;
        while (q >= sx) q -= sx, ++c;
        return true;
      };
      load();
      while (c < nch && ok) {
        // (one chunk of the next group is staged before this group is drained)
        const int stop = min(nch, (g + 1) * EM_GCH + 1);
        while (ok && c < stop) ok = step();
        if (c < nch && ok) ok = drain(g++);
      }
      while (g < ngr && ok) ok = drain(g++);
    }
    cx.chunks += nch;
    cx.groups += ngr;
    if (__syncthreads_or(!ok)) {                           // uniform: every thread leaves
      if (threadIdx.x == 0) {
        *cx.fail = 0;
        em_commit(cx, EM_LAST);
      }
      __syncthreads();
      if (warp == 0) em_wait(cx, EM_LAST, 0);              // one more bounded wait for the MMAs in flight
      if (threadIdx.x == 0) *cx.fail = 1;
      __syncthreads();
      ok = false;
    }
  }
  // hi + lo to FP64 (warps whose rows or columns are all discarded leave it out)
  if ((warp & 3) * 32 < na && c0 < nb) {
#pragma unroll
    for (int c = 0; c < EmAcc::NC; ++c) acc.v[c] = em_sum(hi[c], lo[c]);
  }
  return ok;
}

// A thread's N consecutive doubles at p, in any memory, n of them kept: two at a
// time where all are and p allows.  The 32 lanes of a warp hold 32 rows, so every
// access touches 32 lines: a row's 128 bytes go in 8 instructions instead of 16.
// (32-byte accesses in inline PTX, ld/st.global.v4.f64, here and in em_load were up to
// 3 % faster: n = 2^20 103.0 against 105.2 ms, n = 2^14 3.04 against 3.06, the gradient
// at n = 2^18 77.1 against 78.9, predictions there 29.2 against 29.4.  But where a
// product was a call they once left rows of a ragged tile unwritten; rows of every
// alignment come out right in isolation, called or inlined, and no cause was found, so
// the engine reads and writes by plain accesses only.)
template <int N>
__device__ __forceinline__ void em_get(const double* p, int n, double* v) {
  if (n >= N && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
#pragma unroll
    for (int c = 0; c < N; c += 2) {
      const double2 d = *reinterpret_cast<const double2*>(p + c);
      v[c] = d.x;
      v[c + 1] = d.y;
    }
  } else {
#pragma unroll
    for (int c = 0; c < N; ++c) v[c] = c < n ? p[c] : 0.0;
  }
}
template <int N>
__device__ __forceinline__ void em_put(double* p, int n, const double* v) {
  if (n >= N && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
#pragma unroll
    for (int c = 0; c < N; c += 2) *reinterpret_cast<double2*>(p + c) = make_double2(v[c], v[c + 1]);
  } else {
#pragma unroll
    for (int c = 0; c < N; ++c)
      if (c < n) p[c] = v[c];
  }
}

// A product and what becomes of it, for kernels with many products: one call,
// since inlined at every product the engine's state and the kernel's own crowd
// each other out of the 128 registers a thread has.
//   out(i, j) = P(i, j)  or, with sub, out(i, j) -= P(i, j),  i < na, j < nb,
// row-major with stride ldo; the exponents of the results' rows go to xe[i]
// (columns j >= xe0; null: none), and per 128-column group, counted from column
// gcol for j = 0, to ge[group * TC_M + i] (null: none).
struct EmRows {
  const double* A;
  long sai, sak;
  int na;
  const double* B;
  long sbj, sbk;
  int nb, K;
  const int* pa;
  int pas;
  const int* pb;
  int pbs;
  double* out;
  long ldo;
  bool sub;
  int* xe;
  int xe0;
  int* ge;
  int gcol;
};
static __device__ __noinline__ bool em_rows(EmCtx* pcx, const EmRows* pq) {
  EmCtx cx = *pcx;
  // (out of line the compiler no longer sees that these lie in shared memory)
  __builtin_assume(__isShared(cx.stage));
  __builtin_assume(__isShared(cx.rexp));
  __builtin_assume(__isShared(cx.cexp));
  __builtin_assume(__isShared(cx.mbar));
  __builtin_assume(__isShared(cx.fail));
  EmAcc acc;
  const bool ok = em_mma(cx, acc, pq->A, pq->sai, pq->sak, pq->na, pq->B, pq->sbj, pq->sbk, pq->nb, pq->K, pq->pa,
                         pq->pas, pq->pb, pq->pbs);
  pcx->chunks = cx.chunks;
  pcx->groups = cx.groups;
  const int row = acc.row(), c0 = acc.col0(), nb = pq->nb;
  if (ok && row < pq->na && c0 < nb) {
    double* const o = pq->out + (long)row * pq->ldo + c0;
    if (pq->sub) {
      double v[EmAcc::NC];
      em_get<EmAcc::NC>(o, nb - c0, v);
#pragma unroll
      for (int c = 0; c < EmAcc::NC; ++c) acc.v[c] = v[c] - acc.v[c];
    }
    em_put<EmAcc::NC>(o, nb - c0, acc.v);
    int e0 = -2000, e1 = -2000, ex = -2000;      // a thread's columns touch at most two groups
    const int x0 = pq->xe0 - c0, g0 = EM_KG - ((pq->gcol + c0) & (EM_KG - 1));
#pragma unroll
    for (int c = 0; c < EmAcc::NC; ++c)
      if (c0 + c < nb) {
        const int e = xexp_of(acc.v[c]);
        if (c < g0) e0 = max(e0, e);
        else e1 = max(e1, e);
        if (c >= x0) ex = max(ex, e);
      }
    if (pq->xe && ex > -2000) atomicMax(pq->xe + row, ex);
    if (pq->ge) {
      int* const g = pq->ge + ((pq->gcol + c0) / EM_KG) * TC_M + row;
      if (e0 > -2000) atomicMax(g, e0);
      if (e1 > -2000) atomicMax(g + TC_M, e1);
    }
  }
  return ok;
}

// Row blocks of r rows stacked into one 128-row tile.
__host__ __device__ inline int em_stack(int r) { return r > 64 ? 1 : TC_M / r; }

// Tiles of the packed lower blocks (l, k), k <= l < M, stacked S high along l:
// per column block k, the diagonal tile (l = k) alone, then l = k+1.. in
// stacks of S (the leaf and prior partial sums, whose diagonal tiles take
// another operand).
__host__ __device__ inline int partial_tiles(int M, int S) {
  int n = 0;
  for (int k = 0; k < M; ++k) n += 1 + (M - 1 - k + S - 1) / S;
  return n;
}
__device__ inline bool partial_tile(int t, int M, int S, int& k, int& l0, int& nl) {
  for (k = 0; k < M; ++k) {
    const int nt = 1 + (M - 1 - k + S - 1) / S;
    if (t < nt) {
      l0 = t == 0 ? k : k + 1 + (t - 1) * S;
      nl = t == 0 ? 1 : min(S, M - l0);
      return true;
    }
    t -= nt;
  }
  return false;
}

}  // namespace mra
