// MW_PLAIN: step 3 and 4 of the error-free summation on the FP64 pipe.
//
// Section 2 computes, for double doubles cut into 13-bit quarters,
//   s_i = sum_k sum_{j=0..i} x_{k,j} y_{k,i-j}
// in double arithmetic -- exact because the pieces have zero high bits and the
// number of terms stays below a threshold -- and then adds s_0 + s_1 + ... in
// double double arithmetic.  Here the pieces are balanced integers of w bits
// held in doubles (mw_split, format MW_DIGITS_F64) and the threshold is
// (pairs on a diagonal) * K * 2^(2w-2) <= 2^53, which mw_plan_gemm enforces, so
// every diagonal sum s_t below is exact.  Each s_t, scaled by its weight
// 2^(E_i + E_j + 4 - w(t+2)), is added into an (m+1)-word accumulator with a
// two-sum cascade (postponing renormalisation, Section 4); the accumulator is
// renormalised into m nonoverlapping words once, at the end.
//
// Tiling: a block of 16 x 16 threads computes a (16 TH) x (16 TH) tile of C,
// thread (ty, tx) the outputs (ty + 16 a, tx + 16 b); pieces are staged in
// shared memory 16 columns of the reduction at a time.  This kernel takes any plan;
// plain_split_kernel below (4 x 8 outputs a CTA) takes the plans whose pieces fit in
// its shared memory where it is the faster one (split_clocks, tile_clocks).
#include <algorithm>

#include "mw_device.cuh"
#include "mw_eft.cuh"

namespace mw {
namespace {

constexpr int BKP = 16;

// Add x into the (W)-word accumulator s: top-down two-sum cascade (the error of
// each word moves to the next, the last rounding error is dropped), then a
// bottom-up sweep that keeps the words ordered by magnitude.
template <int W>
__device__ __forceinline__ void accumulate(double (&s)[W], double x) {
  double e = x;
#pragma unroll
  for (int j = 0; j < W; ++j) s[j] = two_sum(s[j], e, e);
#pragma unroll
  for (int j = W - 1; j >= 1; --j) s[j - 1] = two_sum(s[j - 1], s[j], s[j]);
}

// Renormalise W terms into M nonoverlapping words: each pass sums the remaining
// terms bottom-up with two-sum, keeps the top as the next word and the exact
// rounding errors as the terms of the next pass.
template <int W, int M>
__device__ __forceinline__ void renormalize(double (&x)[W], double (&r)[M]) {
#pragma unroll
  for (int j = 0; j < M; ++j) {
    double s = x[W - 1];
#pragma unroll
    for (int i = W - 2; i >= 0; --i) {
      double e;
      s = two_sum(x[i], s, e);
      x[i + 1] = e;
    }
    r[j] = s;
#pragma unroll
    for (int i = 0; i < W - 1; ++i) x[i] = x[i + 1];
    x[W - 1] = 0.0;
  }
}

template <int MW, int TH>
__global__ void __launch_bounds__(256, 1) plain_kernel(PlainArgs a) {
  constexpr int BT = 16 * TH;
  __shared__ double As[BKP][BT + 1];
  __shared__ double Bs[BKP][BT + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int64_t i0 = (int64_t)blockIdx.y * BT, j0 = (int64_t)blockIdx.x * BT;

  double st[TH][TH][MW + 1];
#pragma unroll
  for (int u = 0; u < TH; ++u)
#pragma unroll
    for (int v = 0; v < TH; ++v)
#pragma unroll
      for (int j = 0; j <= MW; ++j) st[u][v][j] = 0.0;

  int ei[TH], ej[TH];
#pragma unroll
  for (int u = 0; u < TH; ++u) {
    const int64_t i = i0 + ty + 16 * u, j = j0 + tx + 16 * u;
    ei[u] = i < a.M ? a.eA[i] : 0;
    ej[u] = j < a.N ? a.eB[j] : 0;
  }

  // load mapping: thread -> (kk = t % 16, row = t / 16 + 16 r)
  const int lk = threadIdx.x & 15, lr = threadIdx.x >> 4;
  for (int t = 0; t < a.D; ++t) {
    double acc[TH][TH];
#pragma unroll
    for (int u = 0; u < TH; ++u)
#pragma unroll
      for (int v = 0; v < TH; ++v) acc[u][v] = 0.0;
    const int plo = max(0, t - a.S_B + 1), phi = min(t, a.S_A - 1);
    for (int p = plo; p <= phi; ++p) {
      const int q = t - p;
      const double *pa = a.dA + (int64_t)p * a.M * a.Kp;
      const double *pb = a.dB + (int64_t)q * a.N * a.Kp;
      for (int64_t k0 = 0; k0 < a.K; k0 += BKP) {       // zeros from K up
#pragma unroll
        for (int r = 0; r < TH; ++r) {
          const int row = lr + 16 * r;
          const int64_t gi = i0 + row, gj = j0 + row;
          As[lk][row] = gi < a.M ? pa[gi * a.Kp + k0 + lk] : 0.0;
          Bs[lk][row] = gj < a.N ? pb[gj * a.Kp + k0 + lk] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BKP; ++kk) {
          double x[TH], y[TH];
#pragma unroll
          for (int u = 0; u < TH; ++u) {
            x[u] = As[kk][ty + 16 * u];
            y[u] = Bs[kk][tx + 16 * u];
          }
#pragma unroll
          for (int u = 0; u < TH; ++u)
#pragma unroll
            for (int v = 0; v < TH; ++v) acc[u][v] = __fma_rn(x[u], y[v], acc[u][v]);
        }
        __syncthreads();
      }
    }
    // s_t is exact; scale by its weight (a power of two) and accumulate
#pragma unroll
    for (int u = 0; u < TH; ++u)
#pragma unroll
      for (int v = 0; v < TH; ++v)
        accumulate<MW + 1>(st[u][v], scalbn(acc[u][v], ei[u] + ej[v] + 4 - a.w * (t + 2)));
  }
#pragma unroll
  for (int u = 0; u < TH; ++u)
#pragma unroll
    for (int v = 0; v < TH; ++v) {
      const int64_t i = i0 + ty + 16 * u, j = j0 + tx + 16 * v;
      double r[MW];
      renormalize<MW + 1, MW>(st[u][v], r);
      if (i < a.M && j < a.N)
#pragma unroll
        for (int w = 0; w < MW; ++w) a.C[w * a.psc + i * a.ldc + j] = r[w];
    }
}

// 4 x 8 outputs a CTA.  The FP64 pipe takes 2 multiply-adds a clock and SM, so
// loads need no reuse in registers; what counts is that every SM has its share of
// the work.  A lane holds one output and the CTA's 8 warps take every eighth k of a
// chunk of KC (all pieces of the chunk's 4 rows and 8 columns in shared memory,
// rows KC + 2 apart: lanes read distinct banks or the same word).  Every partial
// diagonal sum is exact, so the warps' sums add up to the same s_t in any order;
// warp 0 then adds the s_t into the m-double accumulator, t in order, as
// plain_kernel does.  plain_kernel against this one, us (FP64 floor), the call: dd 64^3
// 1,400 / 36 (9), dd 384^3 10,290 / 2,530 (2,420), qd 640^3 37,390 / 33,080
// (32,770), od 256^3 17,380 / 8,010 (6,930).
constexpr int SR = 4, SC = 8, SWARPS = 8;

// Where plain_kernel is the faster one: many tiles for the SMs and a chunk that a warp's
// share of k (every eighth) does not divide into fours, or so many pieces that one CTA
// fills an SM.  Clocks of an SM per pair of pieces, both kernels at two multiply-adds a
// clock: plain_kernel pays whole rounds of tiles and k in sixteens; this kernel the share
// of the rate that chunks of 8, 16, .. 64 columns reach (measured), 0.6 of it with one CTA
// an SM.  us, plain_kernel / this one: qd 512 x 512 x 64 2,304 / 2,761 (S = 10, chunks of 48
// and 16), qd 512 x 512 x 300 10,300 / 11,150, w = 8 (S = 27) 14,310 / 21,580, w = 5 (S = 44)
// 35,300 / 62,670, od w = 16 1024 x 1024 x 40 39,430 / 54,070.  Of 240 plans and sizes
// the rule took the slower kernel for four, 3-6 % slower (K = 40, 1,024 tiles).
inline double tile_clocks(const PlainArgs &a, int BT, int nsm) {
  const int64_t tiles = (a.M + BT - 1) / BT * ((a.N + BT - 1) / BT);
  return 0.5 * BT * BT * (double)((tiles + nsm - 1) / nsm * ((a.K + 15) / 16 * 16));
}
inline double split_clocks(const PlainArgs &a, int KC, size_t smem, int64_t tiles, int nsm) {
  static const double rate[] = {0.79, 0.57, 0.88, 0.92, 0.85, 0.80, 0.88, 0.96};   // by columns / 8
  const int64_t full = a.K / KC, rest = (a.K % KC + 7) / 8;
  const double columns = (double)full * KC / rate[KC / 8 - 1] + (rest ? 8.0 * rest / rate[rest - 1] : 0.0);
  const double one_cta = 2 * (smem + 1024) > 233472 ? 0.6 : 1.0;
  return 0.5 * SR * SC * std::max((double)tiles / nsm, 1.0) * columns / one_cta;
}

inline size_t plain_split_smem(int S_A, int S_B, int D, int KC) {
  return 8 * ((size_t)(SR * S_A + SC * S_B) * (KC + 2) + (size_t)SWARPS * D * 32);
}

template <int MW>
__global__ void __launch_bounds__(32 * SWARPS) plain_split_kernel(PlainArgs a, int KC) {
  extern __shared__ double sm[];
  const int LD = KC + 2;
  double *As = sm, *Bs = As + SR * a.S_A * LD, *st = Bs + SC * a.S_B * LD;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = lane >> 3, c = lane & 7;
  const int64_t tiles_n = (a.N + SC - 1) / SC, ti = blockIdx.x / tiles_n;
  const int64_t i0 = ti * SR, j0 = (blockIdx.x - ti * tiles_n) * SC;
  for (int64_t k0 = 0; k0 < a.K; k0 += KC) {
    const int kc = (int)(a.K - k0 < KC ? (a.K - k0 + 7) & ~(int64_t)7 : KC);   // zeros from K up
    if (k0) __syncthreads();                       // the previous chunk was read
    for (int u = warp; u < SR * a.S_A; u += SWARPS) {
      const int64_t i = i0 + (u & (SR - 1));
      const double *src = a.dA + ((int64_t)(u / SR) * a.M + i) * a.Kp + k0;
      for (int k = lane; k < kc; k += 32) As[u * LD + k] = i < a.M ? src[k] : 0.0;
    }
    for (int u = warp; u < SC * a.S_B; u += SWARPS) {
      const int64_t j = j0 + (u & (SC - 1));
      const double *src = a.dB + ((int64_t)(u / SC) * a.N + j) * a.Kp + k0;
      for (int k = lane; k < kc; k += 32) Bs[u * LD + k] = j < a.N ? src[k] : 0.0;
    }
    __syncthreads();
    for (int t = 0; t < a.D; ++t) {
      const int plo = max(0, t - a.S_B + 1), phi = min(t, a.S_A - 1);
      double acc = k0 ? st[(warp * a.D + t) * 32 + lane] : 0.0;
      for (int p = plo; p <= phi; ++p) {
        const double *x = As + (p * SR + r) * LD, *y = Bs + ((t - p) * SC + c) * LD;
#pragma unroll 4
        for (int k = warp; k < kc; k += SWARPS) acc = __fma_rn(x[k], y[k], acc);
      }
      st[(warp * a.D + t) * 32 + lane] = acc;
    }
  }
  __syncthreads();
  for (int t = warp; t < a.D; t += SWARPS) {       // the warps' sums of s_t into warp 0's
    double v = st[t * 32 + lane];
#pragma unroll
    for (int w = 1; w < SWARPS; ++w) v = __dadd_rn(v, st[(w * a.D + t) * 32 + lane]);
    st[t * 32 + lane] = v;
  }
  __syncthreads();
  const int64_t i = i0 + r, j = j0 + c;
  if (warp || i >= a.M || j >= a.N) return;
  double acc[MW + 1], out[MW];
#pragma unroll
  for (int w = 0; w <= MW; ++w) acc[w] = 0.0;
  const int e = a.eA[i] + a.eB[j] + 4;
  for (int t = 0; t < a.D; ++t) accumulate<MW + 1>(acc, scalbn(st[t * 32 + lane], e - a.w * (t + 2)));
  renormalize<MW + 1, MW>(acc, out);
#pragma unroll
  for (int w = 0; w < MW; ++w) a.C[w * a.psc + i * a.ldc + j] = out[w];
}

template <int MW, int TH>
int launch(const PlainArgs &a, cudaStream_t s) {
  // the longest chunk that leaves room for 3 CTAs an SM, from 32 on for 2 (many
  // pieces: short chunks cost more than the third CTA gives)
  int KC = 64;
  while (KC > 32 && plain_split_smem(a.S_A, a.S_B, a.D, KC) > 75776) KC -= 16;
  while (KC > 8 && plain_split_smem(a.S_A, a.S_B, a.D, KC) > 115712) KC -= 8;
  const size_t smem = plain_split_smem(a.S_A, a.S_B, a.D, KC);
  const int64_t tiles = (a.N + SC - 1) / SC * ((a.M + SR - 1) / SR);
  constexpr int BT = 16 * TH;
  int dev = 0, nsm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (smem <= 232448 && tiles <= 0x7fffffff &&
      (split_clocks(a, KC, smem, tiles, nsm) <= 1.02 * tile_clocks(a, BT, nsm) ||
       (a.M + BT - 1) / BT > 65535)) {               // rows of plain_kernel's grid
    static std::atomic<uint64_t> granted{0};
    cudaError_t e = allow_smem(granted, plain_split_kernel<MW>, 232448);
    if (e != cudaSuccess) return cuda_fail(e, "plain kernel smem attribute");
    plain_split_kernel<MW><<<(unsigned)tiles, 32 * SWARPS, smem, s>>>(a, KC);
    return cuda_fail(cudaGetLastError(), "plain kernel launch");
  }
  dim3 grid((unsigned)((a.N + BT - 1) / BT), (unsigned)((a.M + BT - 1) / BT));
  plain_kernel<MW, TH><<<grid, 256, 0, s>>>(a);
  return cuda_fail(cudaGetLastError(), "plain kernel launch");
}

}  // namespace

int launch_plain(const PlainArgs &a, cudaStream_t s) {
  if (a.Kp % BKP) return fail(MW_EINVAL, "padded K must be a multiple of %d", BKP);
  switch (a.m) {
    case 2: return launch<2, 4>(a, s);
    case 4: return launch<4, 2>(a, s);
    case 8: return launch<8, 2>(a, s);
  }
  return fail(MW_EINVAL, "m must be 2, 4 or 8");
}

}  // namespace mw
