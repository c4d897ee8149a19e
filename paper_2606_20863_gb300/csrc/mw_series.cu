// mw_convolve_batched for series whose digits fit in shared memory: products of
// truncated power series, c_i = sum_{k<=i} a_k b_{i-k} (Section 2's diagonal
// sums s_i are these convolutions), the same words as one inner product per
// coefficient (mw_dot.cu) gives.
//
// Coefficient i is cut on the grids of its own vectors: E_a(i), the largest
// exponent of a_0..a_i, and E_b(i) likewise.  Both only grow with i, so the
// coefficients fall into segments of equal (E_a, E_b), a few for ordinary series
// (as many as there are new largest entries), and one cut of a_0..a_i1 and
// b_0..b_i1 serves a segment's coefficients i0..i1.  A CTA works on one series:
//   1. exponents of all entries (every word), prefix maxima, segment starts;
//   2. per segment, the 24-bit balanced digits of the entries into shared memory
//      (only those not cut yet on the same grid);
//   3. a warp takes 32 consecutive coefficients (a row), one a lane: for every k
//      the digits of a_k are read as a broadcast, those of b_{i-k} at consecutive
//      addresses, and S^2/2 products go into int64 diagonal sums in registers
//      (|d d| <= 2^46 and S n < 2^17 terms at most: far below 2^63);
//   4. each lane fuses and rounds its own coefficient.
// Row r has 32 (r + 1) steps, so a warp takes rows r and R - 1 - r; with few
// series `ks` warps share a row's k and add their sums in shared memory.
//
// A row whose coefficients lie in many segments would be walked once for each with
// most lanes idle, and with few series the rows are fewer than the SMs.  There (the
// cheaper of the two by their steps) a segment's coefficients are taken one a warp, or
// one by several warps: the lanes take every 32nd k, their sums are added by shuffles,
// and `ctas` CTAs share the segments of a series.
//
// Bound by the 32 x 32 -> 64 bit multiply-adds (133 M warp instructions for 2,000
// octo-double pairs of degree 127, about four cycles each and SM sub-partition:
// 0.45 ms, their pipe 77 % busy): those pairs take 0.62 ms, and took 17.25 ms with one CTA per coefficient
// (which cuts i + 1 entries of both series again for each).  Exponents that grow along
// the series cost more cuts.  us, entries growing by 0 / 20 / 45 binades in one operand /
// 45 in both, with one CTA a coefficient, with rows alone, and now:
//   od 2,000 x 128   17,260 / 17,380 / 17,760 / 18,450   623 / 4,450 / 9,330 / 16,390   620 / 1,240 / 1,910 / 3,210
//   od 300 x 512     12,570 / 12,710 / 12,970 / 14,160   1,100 / 5,810 / 11,890 / 41,420   1,090 / 1,440 / 1,760 / 3,160
//   dd 300 x 600      4,410 / 4,710 / 5,210 / 5,370      516 / 2,370 / 5,300 / 9,070   380 / 548 / 708 / 931
//   od 40 x 64          179 / 183 / 189 / 193            39 / 199 / 398 / 585   25 / 48 / 76 / 103
//   od 1 x 1,200        144 / 146 / 151 / 156            476 / 958 / 1,217 / 2,187   70 / 84 / 112 / 130
// So few coefficients that inner products fill the SMs once go there (one_wave).  Slower
// than one CTA a coefficient were, growing by 45 binades in both operands, 12 octo-double
// series of 24 (24.9 / 27.0; of one magnitude 22.8 / 14.3) and 4 double-double ones of 128
// (18.7 / 20.9; 13.0 / 12.8).
#include <cuda.h>

#include <algorithm>

#include "mw_column.cuh"
#include "mw_dot.cuh"

namespace mw {
namespace {

constexpr int kSeriesWarps = 8;                    // most warps of a CTA
constexpr size_t kSeriesSmem = 232448;             // shared memory a CTA can have

constexpr int kSegMask = 0x1fff;                   // n <= 4096

template <int MW, int S> struct SeriesShape {
  static constexpr int DC = S + kDotExtraD;
  static constexpr int SP = (S + 3) / 4 * 4;       // a's digits of one entry, in int4
  static constexpr int NL32 = (kDotW * (DC - 1) + 65 + 31) / 32;   // |X| < 2^(64 + w (D-1))
  // column of a thread: the slots of cut_column (m >= 8), then the rounding's limbs
  static constexpr int COL = (MW >= 8 && S + 3 > NL32) ? S + 3 : NL32;
  // issue cycles of a warp, about: one step of k, the sums of 32 lanes, fusion and rounding
  static constexpr int kStep = 2 * S * (S + 1) + 2 * S + 30, kSum = 30 * DC + 100,
                       kRound = 600 + 150 * MW;
  // coefficients whose sums fit over the columns, one a lane at most
  static __host__ __device__ int most(int warps) {
    static_assert(COL * 16 >= DC, "one a warp fits");
    return COL * 16 / DC * warps < 32 ? COL * 16 / DC * warps : 32;
  }
};

__host__ __device__ inline int64_t series_round32(int64_t n) { return (n + 31) & ~(int64_t)31; }

template <int MW, int S>
size_t series_smem(int64_t n, int warps, int ks) {
  using SH = SeriesShape<MW, S>;
  const size_t nr = (size_t)series_round32(n);
  return 4 * (nr * SH::SP + S * (nr + 32) + 2 * nr + nr + 32 + (size_t)SH::COL * 32 * warps) + 64 +
         (size_t)(warps / ks) * (ks - 1) * SH::DC * 32 * 8;
}

// SINGLE: segments may be taken by coefficients; otherwise one warp does a series, row by
// row (ks = pairs = ctas = 1).
template <int MW, int S, bool SINGLE>
__global__ void __launch_bounds__(SINGLE ? 32 * kSeriesWarps : 32, SINGLE ? (MW == 16 ? 1 : 2) : (MW == 16 ? 8 : 16))
    series_kernel(const DotArgs a, int ks_, int pairs_, int ctas_) {
  const int ks = SINGLE ? ks_ : 1, pairs = SINGLE ? pairs_ : 1, ctas = SINGLE ? ctas_ : 1;
  using SH = SeriesShape<MW, S>;
  constexpr int DC = SH::DC, SP = SH::SP, NL32 = SH::NL32;
  const int n = (int)a.K, nr = (int)series_round32(n), rows = nr / 32;
  const int row_pairs = SINGLE ? (rows + 1) / 2 : 1, nthr = SINGLE ? blockDim.x : 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  extern __shared__ int4 smem4[];
  int64_t *red = reinterpret_cast<int64_t *>(smem4);           // [pairs][ks - 1][DC][32]
  int32_t *da = reinterpret_cast<int32_t *>(red + (size_t)pairs * (ks - 1) * DC * 32);  // [nr][SP]
  int32_t *db = da + (size_t)nr * SP;                          // [S][32 zeros, nr]
  int32_t *pe = db + (size_t)S * (nr + 32);                    // prefix exponents [2][nr]
  int32_t *segs = pe + 2 * nr;                                 // first coefficient of a segment
  int32_t *flags = segs + nr + 32;         // [0] segments, [1..2] smallest exponents, [3] bits
  uint32_t *col = reinterpret_cast<uint32_t *>(flags + 16) + tid;
  // [coefficients of a chunk x q][DC] their sums: over the columns, between their uses
  int64_t *one = reinterpret_cast<int64_t *>(flags + 16);
  const int warps = nthr / 32;
  const int ldb_ = nr + 32;
  for (int t = tid; t < S * 32; t += nthr) db[(t >> 5) * ldb_ + (t & 31)] = 0;

  // the parts with rows come first
  for (int64_t task = blockIdx.x; task < a.count * ctas; task += gridDim.x) {
    const int part = SINGLE ? (int)(task / a.count) : 0;
    const int64_t s_idx = SINGLE ? task - part * a.count : task;
    const double *px[2] = {a.A + s_idx * a.lda, a.B + s_idx * a.ldb};
    const int64_t ps[2] = {a.psa, a.psb};
    // 1. exponents
    __syncthreads();                               // the previous task's flags were read
    if (tid < 4) flags[tid] = tid == 3 ? 0 : -kExpZero;
    __syncthreads();
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      int emin = -kExpZero;
      for (int k = tid; k < nr; k += nthr) {
        int e = kExpZero;
        if (k < n) {
          double x[MW];
#pragma unroll
          for (int j = 0; j < MW; ++j) x[j] = px[o][j * ps[o] + k];
          e = entry_exp<MW>(x);
          if (e == kExpNonFinite) {
            atomicOr(&flags[3], MW_ENONFINITE);
            e = kExpZero;
          }
          if (e != kExpZero) emin = min(emin, e);
        }
        pe[o * nr + k] = e;
      }
      if (emin != -kExpZero) atomicMin(&flags[1 + o], emin);
    }
    __syncthreads();
    if (warp == 0) {                               // prefix maxima and segment starts
      int carry[2] = {kExpZero, kExpZero}, nseg = 0;
      for (int k0 = 0; k0 < nr; k0 += 32) {
        bool first = k0 + lane == 0;
#pragma unroll
        for (int o = 0; o < 2; ++o) {
          int e = max(pe[o * nr + k0 + lane], carry[o]);
          for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, e, d);
            if (lane >= d) e = max(e, y);
          }
          pe[o * nr + k0 + lane] = e;
          int before = __shfl_up_sync(0xffffffffu, e, 1);
          if (lane == 0) before = carry[o];
          first |= before != e;
          carry[o] = __shfl_sync(0xffffffffu, e, 31);
        }
        first &= k0 + lane < n;
        const unsigned m = __ballot_sync(0xffffffffu, first);
        if (first) segs[nseg + __popc(m & ((1u << lane) - 1u))] = k0 + lane;
        nseg += __popc(m);
      }
      if (lane == 0) {
        segs[nseg] = n;
        flags[0] = nseg;
        const int ma = carry[0], mb = carry[1];
        const int sa = ma == kExpZero ? 0 : ma - flags[1], sb = mb == kExpZero ? 0 : mb - flags[2];
        if ((a.range_A >= 0 && sa > a.range_A) || (a.range_B >= 0 && sb > a.range_B))
          raise_status(a.status, MW_WRANGE);
        if (flags[3]) raise_status(a.status, (unsigned)flags[3]);
      }
    }
    __syncthreads();
    const int nseg = flags[0];
    if constexpr (SINGLE) {
      // a segment's way, one thread a segment: bit 23 by rows, whose cost is the steps of
      // the warp with most of them; else `per` coefficients in a chunk (bits 13..18), one
      // a warp at a time, or fewer than the warps with q warps each (bits 19..22), chunk
      // j on CTA (bits 24..31 + j) mod ctas: the segments' chunks, at most one every
      // `warps` coefficients and one more, follow each other.  Rows where neither is
      // much cheaper.
      for (int g = tid; g < nseg; g += nthr) {
        const int i0 = segs[g] & kSegMask, i1 = (segs[g + 1] & kSegMask) - 1, len = i1 + 1 - i0;
        const int r0 = i0 >> 5, r1 = i1 >> 5;
        const int row_steps = min((r1 - r0 < row_pairs ? 1 : 2) * (i1 + 1), 32 * (rows + 1)) / ks;
        const float row_cost = 0.8f * (float)(row_steps * SH::kStep + SH::kRound);
        const int per = min(len, max(warps, min(SH::most(warps), (len + ctas - 1) / ctas)));
        const int q = max(warps / per, 1), chunks = (len + per - 1) / per;
        const int turns = (per * q + warps - 1) / warps;
        const float cost = (float)(turns * (((r1 + q) / q) * SH::kStep + SH::kSum) + SH::kRound);
        const bool by_rows = row_cost * (float)min(ctas, nseg + chunks - 1) <= cost * (float)chunks;
        segs[g] = i0 | per << 13 | q << 19 | (by_rows ? 1 << 23 : 0) | (g + i0 / warps) % ctas << 24;
      }
      __syncthreads();
    }
    const int rp = part * pairs + warp / ks, kw = warp - (warp / ks) * ks;
    // entries 0 .. done[o] - 1 hold digits on the grid of exponent cutE[o]
    int done[2] = {0, 0}, cutE[2] = {0, 0};
    for (int g = 0; g < nseg; ++g) {
      const uint32_t way = (uint32_t)segs[g];
      const int i0 = (int)(way & kSegMask), i1 = (segs[g + 1] & kSegMask) - 1;
      const int r0 = i0 >> 5, r1 = i1 >> 5;
      const bool by_rows = !SINGLE || (way >> 23 & 1);
      const int per = way >> 13 & 63, q = by_rows ? 1 : way >> 19 & 15;
      int first = part - (int)(way >> 24);         // this CTA's first chunk
      if (first < 0) first += ctas;
      if (!by_rows && i0 + first * per > i1) continue;
      const int E[2] = {pe[i0] == kExpZero ? 0 : pe[i0], pe[nr + i0] == kExpZero ? 0 : pe[nr + i0]};
      int kmax, c0 = i0, cstep = i1 + 1;           // entries 0 .. kmax are needed
      if (by_rows) {
        // the rows of this CTA's pairs that the segment touches
        const int plo = part * pairs, phi = min(plo + pairs, row_pairs) - 1;
        const int lo_max = min(phi, r1), hi_max = min(rows - 1 - plo, r1);   // largest row touched
        const bool lo_in = lo_max >= plo && lo_max >= r0;
        const bool hi_in = hi_max >= rows - 1 - phi && hi_max >= r0;
        if (!lo_in && !hi_in) continue;
        kmax = min(i1, 32 * (hi_in ? hi_max : lo_max) + 31);
      } else {
        c0 = i0 + first * per;
        cstep = ctas * per;
        kmax = min(c0 + (i1 - c0) / cstep * cstep + per - 1, i1);
      }
      for (; c0 <= i1; c0 += cstep) {
        const int c1 = by_rows ? i1 : min(c0 + per - 1, i1);
        __syncthreads();                           // the previous digits and sums were read
        // 2. digits
        const int base[2] = {cutE[0] == E[0] ? done[0] : 0, cutE[1] == E[1] ? done[1] : 0};
        const int na = max(kmax + 1 - base[0], 0), nb = max(kmax + 1 - base[1], 0);
        if (MW >= 8 && na + nb > 0)
          for (int c = 0; c < S + 3; ++c) col[c * nthr] = 0u;    // cut_column leaves it zero
        bool ok = true;
        for (int u = tid; u < na + nb; u += nthr) {
          const int o = u >= na, k = o ? base[1] + u - na : base[0] + u;
          const double *p = (o ? px[1] : px[0]) + k;
          const int64_t pst = o ? ps[1] : ps[0];
          const int F = kDotW * S - 2 - (o ? E[1] : E[0]);
          double x[MW];
#pragma unroll
          for (int j = 0; j < MW; ++j) x[j] = p[j * pst];
          // digit p of entry k: a's at da[k SP + p], b's at db[p (nr + 32) + 32 + k]
          int32_t *dst = o ? db + 32 + k : da + k * SP;
          const int step = o ? ldb_ : 1;
          if constexpr (MW >= 8) {
            ok &= cut_column<MW, kDotW, false>(x, F, S, col, nthr,
                                               [&](int p, int32_t d) { dst[(S - 1 - p) * step] = d; });
          } else {
            int32_t d[S];
            ok &= dot_cut<MW, S>(x, F, d);
#pragma unroll
            for (int p = 0; p < S; ++p) dst[p * step] = d[p];
          }
        }
        if (!ok) raise_status(a.status, MW_ERANGE);
        done[0] = max(kmax + 1, base[0]);
        done[1] = max(kmax + 1, base[1]);
        cutE[0] = E[0];
        cutE[1] = E[1];
        if (na + nb > 0) __syncthreads();
        // 3. diagonal sums of rows rp and rows - 1 - rp, or of coefficients c0 .. c1
        const int at_once = by_rows ? 0 : warps / q, at = by_rows ? 0 : warp / q;
        const int turns = by_rows ? 2 : (c1 - c0 + at_once) / at_once;
#pragma unroll 1
        for (int turn = 0; turn < turns; ++turn) {
          const int r = turn ? rows - 1 - rp : rp;
          int i, k, kstep, kend;                   // b_{i-k} is zero for i < k <= i + 31
          bool mine;
          if (by_rows) {
            mine = rp < row_pairs && !(turn && r == rp) && r >= r0 && r <= r1;
            i = 32 * r + lane;
            k = kw;
            kstep = ks;
            kend = min(i1, 32 * r + 31);
          } else {
            i = c0 + turn * at_once + at;
            mine = at < at_once && i <= c1;
            k = 32 * (warp - at * q) + lane;
            kstep = 32 * q;
            kend = i | 31;
          }
          int64_t s[DC];
#pragma unroll
          for (int t = 0; t < DC; ++t) s[t] = 0;
          if (mine) {
#pragma unroll 1
            for (; k <= kend; k += kstep) {
              int32_t x[SP], y[S];
              const int4 *xa = reinterpret_cast<const int4 *>(da + k * SP);
#pragma unroll
              for (int p = 0; p < SP / 4; ++p) {
                const int4 v = xa[p];
                x[4 * p] = v.x; x[4 * p + 1] = v.y; x[4 * p + 2] = v.z; x[4 * p + 3] = v.w;
              }
              const int32_t *yb = db + 32 + i - k;
#pragma unroll
              for (int p = 0; p < S; ++p) y[p] = yb[p * ldb_];
#pragma unroll
              for (int p = 0; p < S; ++p)
#pragma unroll
                for (int p2 = 0; p2 < S - p; ++p2) s[p + p2] += (int64_t)x[p] * (int64_t)y[p2];
#pragma unroll
              for (int t = S; t < DC; ++t)
                if (t < a.D) {
#pragma unroll
                  for (int p = t - S + 1; p < S; ++p) s[t] += (int64_t)x[p] * (int64_t)y[t - p];
                }
            }
          }
          if (by_rows && ks > 1) {
            int64_t *rd = red + (size_t)(warp / ks) * (ks - 1) * DC * 32 + lane;
            if (kw > 0 && mine)
#pragma unroll
              for (int t = 0; t < DC; ++t) rd[((kw - 1) * DC + t) * 32] = s[t];
            __syncthreads();
            if (kw == 0 && mine)
              for (int w = 1; w < ks; ++w)
#pragma unroll
                for (int t = 0; t < DC; ++t) s[t] += rd[((w - 1) * DC + t) * 32];
            mine = mine && kw == 0;
          }
          if (!by_rows) {
            if (mine)
#pragma unroll
              for (int t = 0; t < DC; ++t) {
                for (int o = 16; o; o >>= 1) s[t] += __shfl_xor_sync(0xffffffffu, s[t], o);
                if (lane == t % 32) one[(size_t)((i - c0) * q + warp - at * q) * DC + t] = s[t];
              }
            if (turn + 1 < turns) continue;
            __syncthreads();
            mine = warp == 0 && lane <= c1 - c0;   // one coefficient a lane from here on
            i = c0 + lane;
            if (mine)
#pragma unroll
              for (int t = 0; t < DC; ++t) {
                s[t] = one[lane * q * DC + t];
                for (int w = 1; w < q; ++w) s[t] += one[(lane * q + w) * DC + t];
              }
            __syncwarp();                          // the columns are written next
          }
          // 4. fusion and rounding: X = sum_t s_t 2^(w (DC-1-t)) in 24-bit fields from
          // the least significant end, joined into 32-bit limbs (diagonals D.. are zero)
          if (mine) {
            uint32_t f[DC + 4];
            int64_t carry = 0;
#pragma unroll
            for (int j = 0; j < DC; ++j) {
              if (DC - 1 - j < a.D) carry += s[DC - 1 - j];
              f[j] = (uint32_t)carry & 0xFFFFFFu;
              carry >>= 24;
            }
#pragma unroll
            for (int j = DC; j < DC + 4; ++j) {
              f[j] = (uint32_t)carry & 0xFFFFFFu;
              carry >>= 24;
            }
            uint32_t U[NL32];
#pragma unroll
            for (int l = 0; l < NL32; ++l) {
              const int j = 32 * l / 24, o = 32 * l % 24;
              static_assert((32 * (NL32 - 1)) / 24 + 2 < DC + 4, "fields cover the limbs");
              uint32_t v = (f[j] >> o) | (f[j + 1] << (24 - o));
              if (48 - o < 32) v |= f[j + 2] << (48 - o);
              U[l] = v;
            }
            if (i >= i0 && i <= i1) {
              double *c = a.C + s_idx * a.ldc + i;
              const int64_t psc = a.psc;
              round_column<MW, NL32>(U, col, nthr, E[0] + E[1] + 4 - kDotW * (DC + 1),
                                     [&](int w, double v) { c[w * psc] = v; });
            }
          }
          if (by_rows && ks > 1) __syncthreads();  // red and the columns are reused
        }
      }
    }
  }
}

template <int MW, int S>
int launch_series_s(const DotArgs &a, cudaStream_t st) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int row_pairs = (int)((a.K + 63) / 64);
  // warps sharing a row's k: more while the rows of all series leave SMs with
  // fewer than eight warps
  auto smem_of = [&](int pairs, int ks) { return series_smem<MW, S>(a.K, pairs * ks, ks); };
  int ks = 1;
  while (ks < kSeriesWarps && a.count * row_pairs * ks < (int64_t)8 * nsm) ks *= 2;
  while (ks > 1 && smem_of(1, ks) > kSeriesSmem) ks /= 2;
  int pairs = std::min(row_pairs, kSeriesWarps / ks);
  while (pairs > 1 && smem_of(pairs, ks) > kSeriesSmem) --pairs;
  // few rows for the SMs: coefficients one by one, for which warps count, not a row's share;
  // likewise where the sums of shared rows leave room for two or three warps only (8
  // quad-double series of 2,000, growing: two warps 1,712 us, seven 474; from four warps
  // on a row's share counts again, series of one magnitude 322 with four, 390 with eight)
  const int least = a.count * row_pairs * 4 <= nsm ? pairs * ks + 1 : pairs * ks < 4 ? 4 : kSeriesWarps + 1;
  for (int k = ks / 2; k >= 1; k /= 2) {
    int p = std::min(row_pairs, kSeriesWarps / k);
    while (p > 1 && smem_of(p, k) > kSeriesSmem) --p;
    if (p * k >= least && p * k > pairs * ks && smem_of(p, k) <= kSeriesSmem) {
      ks = k;
      pairs = p;
    }
  }
  const size_t smem = smem_of(pairs, ks);
  if (smem > kSeriesSmem) return fail(MW_EUNSUPPORTED, "series of %lld coefficients", (long long)a.K);
  // CTAs a series: all its rows, and with few series more, for the segments that are taken
  // by coefficients: two an SM while a series is short (40 octo-double series of 64
  // growing coefficients 185 -> 103 us), one an SM for longer ones, whose rows the exponent
  // pass of idle CTAs would slow down (8 double-double series of 1,000: 46 -> 66 us);
  // at most one a chunk's place (the kernel's `way` of a segment g starts at g + i0 / warps)
  const int ctas = (int)std::max<int64_t>((row_pairs + pairs - 1) / pairs,
                                          std::min<int64_t>({a.K + (a.K - 1) / (pairs * ks), (MW < 16 && a.K <= 256 ? 2 : 1) * nsm / a.count, 255}));
  const unsigned grid = (unsigned)std::min<int64_t>(a.count * ctas, 1 << 30);
  auto launch = [&](auto kernel, std::atomic<uint64_t> &granted) {
    cudaError_t e = allow_smem(granted, kernel, kSeriesSmem);
    if (e != cudaSuccess) return cuda_fail(e, "series kernel smem attribute");
    kernel<<<grid, 32 * pairs * ks, smem, st>>>(a, ks, pairs, ctas);
    return cuda_fail(cudaGetLastError(), "series kernel launch");
  };
  static std::atomic<uint64_t> granted[2];
  if (row_pairs == 1 && ks == 1 && ctas == 1) return launch(series_kernel<MW, S, false>, granted[0]);
  return launch(series_kernel<MW, S, true>, granted[1]);
}

template <int MW, int S>
int launch_series_m(int s_req, const DotArgs &a, cudaStream_t st) {
  if constexpr (S > DotS<MW>::hi) {
    return fail(MW_EUNSUPPORTED, "series need %d pieces, at most %d supported", s_req,
                DotS<MW>::hi);
  } else {
    if (s_req == S) return launch_series_s<MW, S>(a, st);
    return launch_series_m<MW, S + 1>(s_req, a, st);
  }
}

// Digits in shared memory beside the columns of four warps.  With fewer a CTA, the only one
// of its SM, is slower than the inner products where exponents grow (us, inner products /
// one to three warps: 200 quad-double series of 2,100 33,230 / 74,390, 600 double-double
// ones of 3,000 100,710 / 285,670, 76 octo-double ones of 1,150 9,310 / 12,020).
template <int MW, int S>
bool series_fits_m(int s_req, int64_t n) {
  if constexpr (S > DotS<MW>::hi) {
    return false;
  } else {
    if (s_req == S) return n <= 4096 && series_smem<MW, S>(n, 4, 1) <= kSeriesSmem;
    return series_fits_m<MW, S + 1>(s_req, n);
  }
}

// So few coefficients that a CTA each fills the SMs once: the inner products take the time
// of one, the series kernel that of a chain of passes where exponents grow (us, inner
// products / series kernel, series of one magnitude and growing by 45 binades: dd 1 x 200
// 13.0 / 12.5 and 12.9 / 18.9, qd 1 x 128 12.7 / 12.5 and 13.6 / 18.8, 12 x 24 13.4 / 13.2
// and 14.9 / 18.6, od 1 x 200 23.0 / 20.9 and 25.1 / 33.1; short octo-double series stay
// with the series kernel, 1 x 64 18.7 / 14.2 and 20.7 / 20.8).
bool one_wave(int m, int64_t count, int64_t n) {
  int dev = 0, nsm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  return m <= 4 ? count * n <= (m == 2 ? 3 : 2) * nsm : m == 8 && n > 64 && count * n <= 2 * nsm;
}

}  // namespace

bool series_fits(int m, int S, int64_t count, int64_t n) {
  if (one_wave(m, count, n)) return false;
  switch (m) {
    case 2: return series_fits_m<2, DotS<2>::lo>(S, n);
    case 4: return series_fits_m<4, DotS<4>::lo>(S, n);
    case 8: return series_fits_m<8, DotS<8>::lo>(S, n);
    case 16: return series_fits_m<16, DotS<16>::lo>(S, n);
  }
  return false;
}

int launch_series(int m, int S, const DotArgs &a, cudaStream_t st) {
  switch (m) {
    case 2: return launch_series_m<2, DotS<2>::lo>(S, a, st);
    case 4: return launch_series_m<4, DotS<4>::lo>(S, a, st);
    case 8: return launch_series_m<8, DotS<8>::lo>(S, a, st);
    case 16: return launch_series_m<16, DotS<16>::lo>(S, a, st);
  }
  return fail(MW_EINVAL, "m must be 2, 4, 8 or 16");
}

}  // namespace mw
