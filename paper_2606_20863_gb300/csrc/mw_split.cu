// Steps 1-2 of the error-free summation (Section 2): a shared exponent per row
// of the logical operand, then every entry cut into S balanced pieces of w bits.
//
// Logical operand: R rows (output dimension) x K columns (reduction).  trans = 0
// reads X[r*ld + k] (k contiguous), trans = 1 reads X[k*ld + r] (r contiguous)
// and transposes through shared memory so that the pieces are written with k
// contiguous either way.
//
// Pass 1 (exponents): E'_r = max over nonzero words of ilogb+1, e'_r = min over
//   nonzero entries of the entry exponent, kept biased in int32 so that zero
//   means "nothing seen" and a memset initialises them.
// Finalize: E_r (0 for an all-zero row), spread_r = E_r - e_r, warning check.
// Pass 2 (pieces): T = sum_j trunc(x_j 2^(wS-2-E_r)) in NL 64-bit limbs (two's
//   complement), then the balanced base-2^w digits from the least significant
//   end with a carry, written as bfloat16 or double.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdio>
#include <type_traits>

#include "mw_device.cuh"
#include "mw_pieces.cuh"

namespace mw {
namespace {

constexpr int kBias = 1 << 20;  // E and -e stored as value + kBias (> 0 for any double)

__device__ __forceinline__ void entry_exps(const double *x, int64_t plane_stride, int m,
                                           int &e_entry, bool &nonfinite) {
  e_entry = kExpZero;
  for (int j = 0; j < m; ++j) {
    const int e = exp_plus1(x[j * plane_stride]);
    if (e == kExpNonFinite) nonfinite = true;
    else if (e > e_entry) e_entry = e;
  }
}

// ---- pass 1 ------------------------------------------------------------------
// m words per entry (m = 1: the leading words only).  Kernels given a gate return
// at once while *gate == 0; their blocks loop over the work, so that a launch
// that turns out not to be needed costs few blocks.
// trans = 0: block = 256 threads along 1024 k of one row; work unit (r, k chunk).
constexpr int kRowChunk = 1024;
// operands of at least this many entries take their exponents from the leading
// words first (below it the extra launches cost more than the words saved)
constexpr int64_t kLeadMinEntries = 1 << 22;
__global__ void exps_rows_kernel(const double *__restrict__ X, int m, int64_t R, int64_t K,
                                 int64_t ld, int64_t ps, int *Eb, int *eminb,
                                 unsigned int *status, const int32_t *gate) {
  if (gate && *gate == 0) return;
  const int64_t nkc = (K + kRowChunk - 1) / kRowChunk;
  bool bad = false;
  for (int64_t u = blockIdx.x; u < R * nkc; u += gridDim.x) {
    const int64_t r = u / nkc, kc = u - r * nkc;
    int emax = kExpZero, emin = -kExpZero;
    for (int64_t k = kc * kRowChunk + threadIdx.x; k < K && k < (kc + 1) * kRowChunk;
         k += blockDim.x) {
      int e;
      entry_exps(X + r * ld + k, ps, m, e, bad);
      if (e != kExpZero) {
        emax = max(emax, e);
        emin = min(emin, e);
      }
    }
    for (int o = 16; o; o >>= 1) {
      emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
      emin = min(emin, __shfl_xor_sync(0xffffffffu, emin, o));
    }
    if ((threadIdx.x & 31) == 0 && emax != kExpZero) {
      atomicMax(Eb + r, emax + kBias);
      atomicMax(eminb + r, kBias - emin);
    }
  }
  if (bad) raise_status(status, MW_ENONFINITE);
}

// trans = 1: block = 32 (r) x 8 (k) threads; work unit: 32 columns x
// kRowsPerBlock rows of the stored K x R matrix.
constexpr int kRowsPerBlock = 32;
__global__ void exps_cols_kernel(const double *__restrict__ X, int m, int64_t R, int64_t K,
                                 int64_t ld, int64_t ps, int *Eb, int *eminb,
                                 unsigned int *status, const int32_t *gate) {
  if (gate && *gate == 0) return;
  __shared__ int smax[8][32], smin[8][32];
  const int64_t nrb = (R + 31) / 32, nkb = (K + kRowsPerBlock - 1) / kRowsPerBlock;
  bool bad = false;
  for (int64_t u = blockIdx.x; u < nrb * nkb; u += gridDim.x) {
    const int64_t kb = u / nrb, rb = u - kb * nrb;  // neighbouring blocks: neighbouring r
    const int64_t r = rb * 32 + threadIdx.x;
    const int64_t k0 = kb * kRowsPerBlock;
    int emax = kExpZero, emin = -kExpZero;
    if (r < R) {
      for (int64_t k = k0 + threadIdx.y; k < K && k < k0 + kRowsPerBlock; k += 8) {
        int e;
        entry_exps(X + k * ld + r, ps, m, e, bad);
        if (e != kExpZero) {
          emax = max(emax, e);
          emin = min(emin, e);
        }
      }
    }
    smax[threadIdx.y][threadIdx.x] = emax;
    smin[threadIdx.y][threadIdx.x] = emin;
    __syncthreads();
    if (threadIdx.y == 0 && r < R) {
      for (int i = 1; i < 8; ++i) {
        emax = max(emax, smax[i][threadIdx.x]);
        emin = min(emin, smin[i][threadIdx.x]);
      }
      if (emax != kExpZero) {
        atomicMax(Eb + r, emax + kBias);
        atomicMax(eminb + r, kBias - emin);
      }
    }
    __syncthreads();
  }
  if (bad) raise_status(status, MW_ENONFINITE);
}

// E_r and the spread from the biased maxima, then the largest spread and the
// warning (MW_WRANGE).  mode 1: the conversion only (exponents from the leading
// words, checked later); mode 2, after that check: when the operand was not
// passed over again (*redo == 0) the largest spread and the warning from the
// values already converted.
__global__ void exps_finalize_kernel(int64_t R, int *E, int *spread, int *max_spread, int range,
                                     unsigned int *status, const int32_t *redo, int mode) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= R) return;
  int Er = E[r], sp = spread[r];
  if (mode != 2 || *redo) {
    const int eb = Er, mb = sp;
    Er = eb > 0 ? eb - kBias : 0;
    sp = eb > 0 ? Er - (kBias - mb) : 0;
    E[r] = Er;
    spread[r] = sp;
  }
  if (mode == 1) return;
  if (max_spread) atomicMax(max_spread, sp);
  if (range >= 0 && sp > range) raise_status(status, MW_WRANGE);
}

// Pass 1 of both operands of a product in one launch: no atomics on the rows, no
// clearing, no finalize, no second stream.  trans = 0: a warp per row, eight rows a
// block; trans = 1: 8 columns x 32 rows of the stored matrix at a time; either way
// the threads that see a row or column see all of it, one entry in 32 each, so
// reductions are short (pair_max_k) and, in a product, operands small (kPairMaxWords:
// 384^3 quad doubles 120 -> 114 us, 512^3 149 -> 159, 256^3 octo doubles 150 -> 137,
// 384^3 236 -> 246; above that the two-stream passes over chunks keep more loads in
// flight).  The limits on the reduction, us a call apart / together, 32 x 32 outputs:
//   products   m = 2  K = 1,024  106 / 99   2,048  170 / 172 (128 x 128: 176 / 181)
//              m = 4  K = 1,024  172 / 170  2,048  299 / 310 (residues: 63 / 61, 78 / 88)
//              m = 8  K = 512    190 / 183  1,024  313 / 315  2,048  568 / 588
//              m = 16 K = 512    643 / 630  1,024  1,130 / 1,126
//   the spread measurement (16 to 1,024 rows), which waits for the result:
//              m = 2  K = 2,048  53 / 48    m = 4  1,024  56 / 47, 2,048  58 / 59
//              m = 8  K = 1,024  61 / 58, 2,048  61 / 71
//              m = 16 K = 1,024  62 / 57 (1,000 + 1,000 rows: 150 / 109), 2,048  62 / 72
// Many rows (more than kPairMaxRows): a warp a short row, or eight columns of few rows,
// leaves loads unused: 2^19 columns of 1..16 double doubles 84-125 / 117-158, of 64
// 281 / 234; 2^19 rows of 2 580 / 172, of 128 773 / 730, of 256 872 / 1,055.
// The first block clears the product kernel's work counter.
inline int64_t pair_max_k(int m, bool exponents_only) {
  if (m <= 2) return exponents_only ? 2048 : 1536;
  return m <= 4 || exponents_only ? 1024 : 512;
}
constexpr int64_t kPairMaxRows = 1 << 17;
constexpr int64_t kPairMaxWords = 3 << 19;
constexpr int kPairCols = 8;
struct ExpsArgs {
  const double *X;
  int64_t R, K, ld, ps;
  int trans, range;
  int32_t *E, *spread, *max_spread;
};
__host__ __device__ __forceinline__ int64_t exps_pair_blocks(const ExpsArgs &a) { return (a.R + 7) / 8; }

template <int MW>
__device__ __forceinline__ void exps_entry(const double *x, int64_t ps, int &emax, int &emin,
                                           bool &bad) {
  double v[MW];
  uint32_t h = 0;                                  // largest high word without its sign
#pragma unroll
  for (int j = 0; j < MW; ++j) v[j] = x[j * ps];
#pragma unroll
  for (int j = 0; j < MW; ++j) h = max(h, (uint32_t)__double2hiint(v[j]) << 1);
  int e = (int)(h >> 21) - 1022;
  if ((h >> 21) == 0 || (h >> 21) == 0x7ff) {      // zero, subnormal or not finite
    e = kExpZero;
#pragma unroll
    for (int j = 0; j < MW; ++j) {
      const int u = exp_plus1(v[j]);
      if (u == kExpNonFinite) bad = true;
      else e = max(e, u);
    }
  }
  if (e != kExpZero) {
    emax = max(emax, e);
    emin = min(emin, e);
  }
}

template <int MW>
__global__ void __launch_bounds__(256) exps_pair_kernel(ExpsArgs a, ExpsArgs b, unsigned blocks_a,
                                                        unsigned long long *counter,
                                                        unsigned int *status) {
  if (blockIdx.x == 0 && threadIdx.x == 0 && counter) *counter = 0;
  const bool second = blockIdx.x >= blocks_a;
  const ExpsArgs &p = second ? b : a;
  const int64_t r0 = 8 * (int64_t)(blockIdx.x - (second ? blocks_a : 0u));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int emax = kExpZero, emin = -kExpZero;
  bool bad = false;
  auto finish = [&](int64_t r) {                   // one thread per row
    const int Er = emax == kExpZero ? 0 : emax, sp = emax == kExpZero ? 0 : emax - emin;
    p.E[r] = Er;
    p.spread[r] = sp;
    if (sp > 0) atomicMax(p.max_spread, sp);
    if (p.range >= 0 && sp > p.range) raise_status(status, MW_WRANGE);
  };
  if (!p.trans) {
    const int64_t r = r0 + warp;
    if (r < p.R)
#pragma unroll(MW <= 4 ? 4 : 1)
      for (int64_t k = lane; k < p.K; k += 32)
        exps_entry<MW>(p.X + r * p.ld + k, p.ps, emax, emin, bad);
    for (int o = 16; o; o >>= 1) {
      emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
      emin = min(emin, __shfl_xor_sync(0xffffffffu, emin, o));
    }
    if (lane == 0 && r < p.R) finish(r);
  } else {
    __shared__ int smax[32][kPairCols], smin[32][kPairCols];
    const int tx = threadIdx.x % kPairCols, ty = threadIdx.x / kPairCols;
    const int64_t r = r0 + tx;
    if (r < p.R)
#pragma unroll(MW <= 4 ? 4 : 1)
      for (int64_t k = ty; k < p.K; k += 32)
        exps_entry<MW>(p.X + k * p.ld + r, p.ps, emax, emin, bad);
    smax[ty][tx] = emax;
    smin[ty][tx] = emin;
    __syncthreads();
    if (threadIdx.x < kPairCols && r < p.R) {
      for (int i = 1; i < 32; ++i) {
        emax = max(emax, smax[i][tx]);
        emin = min(emin, smin[i][tx]);
      }
      finish(r);
    }
  }
  if (bad) raise_status(status, MW_ENONFINITE);
}

// ---- pass 2 ------------------------------------------------------------------
// trans = 0: one thread per (row, pair of columns), pairs cover the padded width.
template <int MW, int NL, typename Out>
__device__ __forceinline__ void pieces_rows(const double *__restrict__ X, int64_t R, int64_t K,
                                            int64_t ld, int64_t ps, int w, int S, Out *digits,
                                            int64_t dld, const int *E, unsigned int *status,
                                            int64_t block) {
  const int64_t npair = dld / 2;
  const int64_t idx = block * 256 + threadIdx.x;
  if (idx >= R * npair) return;
  const int64_t r = idx / npair, k = 2 * (idx % npair);
  double a[MW], b[MW];
  const bool v0 = k < K, v1 = k + 1 < K;
  const double *row = X + r * ld;
  const bool vec = v1 && ((((uintptr_t)(row + k)) & 15) == 0) && ((ps & 1) == 0);
#pragma unroll
  for (int j = 0; j < MW; ++j) {
    if (vec) {
      const double2 v = *reinterpret_cast<const double2 *>(row + j * ps + k);  // 128-bit load
      a[j] = v.x;
      b[j] = v.y;
    } else {
      a[j] = v0 ? row[j * ps + k] : 0.0;
      b[j] = v1 ? row[j * ps + k + 1] : 0.0;
    }
  }
  const int F = w * S - 2 - E[r];
  if (w == 8)
    cut_pair_w8<MW, NL, Out>(a, b, F, S, digits + r * dld + k, R * dld, status);
  else
    cut_pair<MW, NL, Out>(a, b, F, w, S, digits + r * dld + k, R * dld, status);
}

template <int MW, int NL, typename Out>
__global__ void pieces_rows_kernel(const double *__restrict__ X, int64_t R, int64_t K,
                                   int64_t ld, int64_t ps, int w, int S, Out *digits,
                                   int64_t dld, const int *E, unsigned int *status) {
  pieces_rows<MW, NL, Out>(X, R, K, ld, ps, w, S, digits, dld, E, status, blockIdx.x);
}

// trans = 1: 32 x 32 tiles (32 rows r, 32 columns k of the logical operand)
// staged through shared memory as doubles (m planes), then cut like trans = 0.
template <int MW, int NL, typename Out>
__device__ __forceinline__ void pieces_cols(const double *__restrict__ X, int64_t R, int64_t K,
                                            int64_t ld, int64_t ps, int w, int S, Out *digits,
                                            int64_t dld, const int *E, unsigned int *status,
                                            int64_t r0, int64_t k0, double *tile) {
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8; tile [m][32 k][33]
#pragma unroll
  for (int j = 0; j < MW; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int kl = ty + 8 * i;
      const int64_t k = k0 + kl, r = r0 + tx;
      tile[(j * 32 + kl) * 33 + tx] = (k < K && r < R) ? X[j * ps + k * ld + r] : 0.0;
    }
  __syncthreads();
  const int tid = ty * 32 + tx;
  for (int it = 0; it < 2; ++it) {
    const int e = tid + 256 * it;      // 512 pairs per tile
    const int rl = e >> 4, kl = 2 * (e & 15);
    const int64_t r = r0 + rl, k = k0 + kl;
    if (r >= R || k >= dld) continue;
    double a[MW], b[MW];
#pragma unroll
    for (int j = 0; j < MW; ++j) {
      a[j] = tile[(j * 32 + kl) * 33 + rl];
      b[j] = tile[(j * 32 + kl + 1) * 33 + rl];
    }
    const int F = w * S - 2 - E[r];
    if (w == 8)
      cut_pair_w8<MW, NL, Out>(a, b, F, S, digits + r * dld + k, R * dld, status);
    else
      cut_pair<MW, NL, Out>(a, b, F, w, S, digits + r * dld + k, R * dld, status);
  }
}

template <int MW, int NL, typename Out>
__global__ void __launch_bounds__(256)
    pieces_cols_kernel(const double *__restrict__ X, int64_t R, int64_t K, int64_t ld, int64_t ps,
                       int w, int S, Out *digits, int64_t dld, const int *E, unsigned int *status) {
  extern __shared__ double tile[];
  pieces_cols<MW, NL, Out>(X, R, K, ld, ps, w, S, digits, dld, E, status, blockIdx.x * (int64_t)32,
                           blockIdx.y * (int64_t)32, tile);
}

// Pieces of both operands in one launch, for small products (kPairMaxEntries), where
// a second stream's fork and join cost more than the kernels beside each other save:
// with the exponents together 64^3 double doubles 45.6 -> 31.9 us a call (37 -> 25
// replayed from a graph).  Only for entries of up to kPairMaxBits bits: the wider
// kernels take minutes to compile twice, and their two launches belong beside each
// other on two streams (64^3, one after the other / beside each other: octo doubles
// 77 / 67 us, hexa doubles 237 / 194, 50-bit spreads of quad doubles 53 / 50; 32 x 32 x
// 512 hexa doubles with A transposed 728 / 628).  One after the other again from
// kRowMinEntries on when A and B are as stored (k contiguous in A only), where each
// kernel fills the GPU: 290^3 quad doubles of wide spread 106 / 112, 300^3 octo doubles
// 178 / 184, equal at 256^3; with a transpose beside each other stays faster (98-100 /
// 106-107, 159-170 / 169-182).
constexpr int64_t kPairMaxEntries = 1 << 18;
constexpr int kPairMaxBits = 256;
constexpr int64_t kRowMinEntries = 1 << 17;
inline int piece_bits(int w, int S) { return w * S + 3; }   // |T| < m 2^(wS-2) < 2^(wS+1), one sign bit
template <typename Out> struct PieceArgs {
  const double *X;
  int64_t R, K, ld, ps, dld;
  int trans, S;
  Out *digits;
  const int32_t *E;
};
template <int MW, int NL, typename Out>
__global__ void __launch_bounds__(256) pieces_pair_kernel(PieceArgs<Out> a, PieceArgs<Out> b,
                                                          unsigned blocks_a, int w,
                                                          unsigned int *status) {
  extern __shared__ double tile[];
  const bool second = blockIdx.x >= blocks_a;
  const PieceArgs<Out> &p = second ? b : a;
  const int64_t u = blockIdx.x - (second ? blocks_a : 0u);
  if (!p.trans) {
    pieces_rows<MW, NL, Out>(p.X, p.R, p.K, p.ld, p.ps, w, p.S, p.digits, p.dld, p.E, status, u);
  } else {
    const int64_t nr = (p.R + 31) / 32, kb = u / nr;
    pieces_cols<MW, NL, Out>(p.X, p.R, p.K, p.ld, p.ps, w, p.S, p.digits, p.dld, p.E, status,
                             (u - kb * nr) * 32, kb * 32, tile);
  }
}

template <int MW, typename Out, int NL>
int launch_pieces_pair(const SplitArgs &a, const SplitArgs &b, cudaStream_t s) {
  auto args = [](const SplitArgs &x) {
    return PieceArgs<Out>{x.X, x.R, x.K, x.ld, x.plane_stride, x.digit_ld, x.trans, x.S,
                          static_cast<Out *>(x.digits), x.exps};
  };
  auto blocks = [](const SplitArgs &x) {
    return (unsigned)(x.trans ? (x.R + 31) / 32 * ((x.digit_ld + 31) / 32)
                              : (x.R * (x.digit_ld / 2) + 255) / 256);
  };
  const size_t sm = a.trans || b.trans ? (size_t)MW * 32 * 33 * sizeof(double) : 0;
  static std::atomic<uint64_t> granted{0};
  cudaError_t e = allow_smem(granted, pieces_pair_kernel<MW, NL, Out>, MW * 32 * 33 * sizeof(double));
  if (e != cudaSuccess) return cuda_fail(e, "split smem attribute");
  pieces_pair_kernel<MW, NL, Out><<<blocks(a) + blocks(b), 256, sm, s>>>(args(a), args(b), blocks(a),
                                                                        a.w, status_ptr());
  return cuda_fail(cudaGetLastError(), "split pieces launch");
}

template <int MW, typename Out, int NL>
int launch_pieces(const SplitArgs &a, cudaStream_t s) {
  Out *dig = static_cast<Out *>(a.digits);
  if (!a.trans) {
    const int64_t n = a.R * (a.digit_ld / 2);
    const int threads = 256;
    pieces_rows_kernel<MW, NL, Out><<<(unsigned)((n + threads - 1) / threads), threads, 0, s>>>(
        a.X, a.R, a.K, a.ld, a.plane_stride, a.w, a.S, dig, a.digit_ld, a.exps, status_ptr());
  } else {
    dim3 grid((unsigned)((a.R + 31) / 32), (unsigned)((a.digit_ld + 31) / 32));
    const size_t sm = (size_t)MW * 32 * 33 * sizeof(double);
    static std::atomic<uint64_t> granted{0};
    cudaError_t e = allow_smem(granted, pieces_cols_kernel<MW, NL, Out>, sm);
    if (e != cudaSuccess) return cuda_fail(e, "split smem attribute");
    pieces_cols_kernel<MW, NL, Out><<<grid, 256, sm, s>>>(
        a.X, a.R, a.K, a.ld, a.plane_stride, a.w, a.S, dig, a.digit_ld, a.exps, status_ptr());
  }
  return cuda_fail(cudaGetLastError(), "split pieces launch");
}

// The pieces of a (b: of both operands, of at most kPairMaxBits bits).
template <int MW, typename Out, int NL>
int launch_pieces_ab(const SplitArgs &a, const SplitArgs *b, cudaStream_t s) {
  if (!b) return launch_pieces<MW, Out, NL>(a, s);
  if constexpr (64 * NL <= kPairMaxBits) return launch_pieces_pair<MW, Out, NL>(a, *b, s);
  return fail(MW_EUNSUPPORTED, "pieces of both operands in one launch: %d limbs", NL);
}

template <int MW, typename Out>
int launch_pieces_nl(const SplitArgs &a, const SplitArgs *b, cudaStream_t s) {
  const int S = b ? std::max(a.S, b->S) : a.S;
  const int bits = piece_bits(a.w, S);
  if (bits <= 128) return launch_pieces_ab<MW, Out, 2>(a, b, s);
  if (bits <= 256) return launch_pieces_ab<MW, Out, 4>(a, b, s);
  if (bits <= 384) return launch_pieces_ab<MW, Out, 6>(a, b, s);
  if (bits <= 512) return launch_pieces_ab<MW, Out, 8>(a, b, s);
  if (bits <= 640) return launch_pieces_ab<MW, Out, 10>(a, b, s);
  return fail(MW_EUNSUPPORTED, "w*S = %d too large (at most 637 bits)", a.w * S);
}

template <typename Out>
int launch_pieces_m(const SplitArgs &a, const SplitArgs *b, cudaStream_t s) {
  switch (a.m) {
    case 2: return launch_pieces_nl<2, Out>(a, b, s);
    case 4: return launch_pieces_nl<4, Out>(a, b, s);
    case 8: return launch_pieces_nl<8, Out>(a, b, s);
    case 16:
      // hexa doubles: bfloat16 pieces (MW_OZAKI) only
      if constexpr (std::is_same<Out, __nv_bfloat16>::value) {
        const int S = b ? std::max(a.S, b->S) : a.S;
        const int bits = piece_bits(a.w, S);
        if (bits <= 768) return launch_pieces_ab<16, Out, 12>(a, b, s);
        if (bits <= 896) return launch_pieces_ab<16, Out, 14>(a, b, s);
        if (bits <= 1024) return launch_pieces_ab<16, Out, 16>(a, b, s);
        return fail(MW_EUNSUPPORTED, "w*S = %d too large (at most 1021 bits)", a.w * S);
      } else {
        return fail(MW_EUNSUPPORTED, "m = 16 is cut into bfloat16 pieces only");
      }
  }
  return fail(MW_EINVAL, "m must be 2, 4, 8 or 16");
}

}  // namespace

// Exponents of the operand from m words per entry.  gate: the pass over every
// word after the leading words' check (runs only if *gate != 0, on a small grid:
// it is rarely needed); it accumulates onto the converted values of the first
// pass, which every biased maximum exceeds.
int launch_exps(const SplitArgs &a, int m, int mode, const int32_t *gate, cudaStream_t s) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int64_t cap = (int64_t)(gate ? 2 : 16) * std::max(nsm, 1);
  if (!a.trans) {
    const int64_t units = a.R * ((a.K + kRowChunk - 1) / kRowChunk);
    exps_rows_kernel<<<(unsigned)std::min(units, cap), 256, 0, s>>>(
        a.X, m, a.R, a.K, a.ld, a.plane_stride, a.exps, a.spread, status_ptr(), gate);
  } else {
    const int64_t units = ((a.R + 31) / 32) * ((a.K + kRowsPerBlock - 1) / kRowsPerBlock);
    exps_cols_kernel<<<(unsigned)std::min(units, cap), dim3(32, 8), 0, s>>>(
        a.X, m, a.R, a.K, a.ld, a.plane_stride, a.exps, a.spread, status_ptr(), gate);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "split exponent launch");
  exps_finalize_kernel<<<(unsigned)((a.R + 255) / 256), 256, 0, s>>>(
      a.R, a.exps, a.spread, a.max_spread, a.range, status_ptr(), a.redo, mode);
  return cuda_fail(cudaGetLastError(), "split finalize launch");
}

int launch_split(const SplitArgs &a, bool exponents_only, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(a.exps, 0, sizeof(int32_t) * a.R, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.spread, 0, sizeof(int32_t) * a.R, s);
  if (e != cudaSuccess) return cuda_fail(e, "split memset");
  if (a.nmod > 0 && a.redo && !exponents_only && a.R * a.K >= kLeadMinEntries) {
    // residue form, large operands: exponents from the leading words (1/m of the
    // data), checked entry by entry by the split; only if an entry failed do the
    // exponents over every word and the split run again
    if ((e = cudaMemsetAsync(a.redo, 0, sizeof(int32_t), s)) != cudaSuccess)
      return cuda_fail(e, "split memset");
    SplitArgs b = a;
    b.gate = nullptr;
    int rc = launch_exps(b, 1, 1, nullptr, s);
    if (!rc) rc = launch_residues(b, s);
    if (!rc) rc = launch_exps(b, a.m, 2, a.redo, s);
    if (rc) return rc;
    b.redo = nullptr;
    b.gate = a.redo;
    return launch_residues(b, s);
  }
  SplitArgs b = a;
  b.redo = nullptr;
  b.gate = nullptr;
  int rc = launch_exps(b, a.m, 0, nullptr, s);
  if (rc || exponents_only) return rc;
  if (a.nmod > 0) return launch_residues(b, s);
  return launch_digits(a, nullptr, s);
}

int launch_digits(const SplitArgs &a, const SplitArgs *b, cudaStream_t s) {
  if (a.format == MW_DIGITS_BF16) return launch_pieces_m<__nv_bfloat16>(a, b, s);
  return launch_pieces_m<double>(a, b, s);
}

bool exps_together(const SplitArgs &a, const SplitArgs &b, bool exponents_only) {
  auto few_rows = [](const SplitArgs &x) {
    return x.R <= kPairMaxRows || (x.trans ? x.K >= 64 : x.K <= 128);
  };
  if (a.K > pair_max_k(a.m, exponents_only) || !few_rows(a) || !few_rows(b) ||
      (a.R + 7) / 8 + (b.R + 7) / 8 > 0x7fffffff)
    return false;
  return exponents_only || a.m * (a.R + b.R) * a.K <= kPairMaxWords;
}

bool digits_together(const SplitArgs &a, const SplitArgs &b) {
  // (the narrowest kernel for m = 16 takes 768 bits, also for a plan of fewer)
  return a.nmod == 0 && a.m <= 8 && (a.R + b.R) * a.K <= kPairMaxEntries &&
         piece_bits(a.w, std::max(a.S, b.S)) <= kPairMaxBits;
}

bool digits_in_a_row(const SplitArgs &a, const SplitArgs &b) {
  const int64_t entries = (a.R + b.R) * a.K;
  return a.nmod == 0 && entries > kRowMinEntries && entries <= kPairMaxEntries && !a.trans && b.trans;
}

int launch_exps_pair(const SplitArgs &a, const SplitArgs &b, unsigned long long *counter,
                     cudaStream_t s) {
  auto args = [](const SplitArgs &x) {
    return ExpsArgs{x.X, x.R, x.K, x.ld, x.plane_stride, x.trans, x.range,
                    x.exps, x.spread, x.max_spread};
  };
  const ExpsArgs ea = args(a), eb = args(b);
  const unsigned na = (unsigned)exps_pair_blocks(ea), nb = (unsigned)exps_pair_blocks(eb);
  switch (a.m) {
    case 2: exps_pair_kernel<2><<<na + nb, 256, 0, s>>>(ea, eb, na, counter, status_ptr()); break;
    case 4: exps_pair_kernel<4><<<na + nb, 256, 0, s>>>(ea, eb, na, counter, status_ptr()); break;
    case 8: exps_pair_kernel<8><<<na + nb, 256, 0, s>>>(ea, eb, na, counter, status_ptr()); break;
    case 16: exps_pair_kernel<16><<<na + nb, 256, 0, s>>>(ea, eb, na, counter, status_ptr()); break;
    default: return fail(MW_EINVAL, "m must be 2, 4, 8 or 16");
  }
  return cuda_fail(cudaGetLastError(), "split exponent launch");
}

}  // namespace mw
