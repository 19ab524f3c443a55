// D_c = R D P assembly (Alg. 5, Eq. cgo via Alg. 7's D P) on the tensor cores, by exact products of slices
// (the Ozaki scheme: Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59 (2012); on tensor cores Mukunoki,
// Ozaki, Ogita and Imamura, ISC 2020).
//
// One forward hop x -> x+mu contributes A(x)^dagger Bt(x) with A = u^dagger P(x) and
// Bt = u^dagger U_mu(x) P(x+mu), both 6 x 2 ntv (see setup.cu); per (block, job) that is a product of
// two matrices of K = 6 Vb rows.  Every column of A and Bt becomes fixed-point numbers relative to a power
// of two that bounds the column on its block, cut into DIG signed digits of 8 bits, which FP16 holds
// exactly.  Products of digits i and j have the weight of i + j = s; those of equal s < DIG are summed by
// the tensor cores in one FP32 accumulator in tensor memory.  For s <= 4 a sum of 12 K steps is an integer
// below 5 x 192 x 128^2 < 2^24, which FP32 holds exactly in any order; every 12 K steps these are added, with
// their weights, to 64-bit integers in shared memory.  The sums of s >= 5 carry at most 2^-40 of the
// result each; they stay in FP32 to the end.  Lost are the pairs of s >= DIG, the cut of the columns (56 bits for
// DIG 7, 64 for DIG 8) and of the 64-bit result: about 2^-52 (DIG 8) of the product of the two columns' bounds.  Where the
// largest product of one site lies far below that, as with test vectors that are small on a face of the block, the (block,
// job) is left to the kernels that add up in floating point (tc_left_kernel).
//
// U_mu P (self: (4 + m0 + C) P) is formed in integers too: coefficients of 62 bits and entries of 61 as two words
// of 31 bits each, the three leading partial products summed in 64 bits (a 32 x 32 bit multiply-add takes a
// sixteenth of the time of one in FP64).  The block's coefficients are converted once, into shared memory.
//
// Real arithmetic: rows 2 c, 2 c + 1 of A are the real and imaginary part of its column c (at most 128 rows, the
// instruction's M), columns of B likewise for the columns of one chirality (N = 2 round8(ntv)); the four
// real products meet in neighbouring lanes when the tile is written.  A_i times all of B_0 .. B_(DIG-1-i) is one
// product of up to 256 columns: B's slices and the accumulators of i, i + 1, .. both follow each other.
//
// One CTA per (block, job, chirality of the columns), one per SM (DIG accumulators of N columns of tensor memory).
// Roles: warps 0-3 read the accumulators (lane quadrant = warp) and write the blocks; then kBuildWarps warps turn
// entries into digits; the last warp issues the products.  A builder's item is 4 columns at 4 sites, a pair of
// lanes a column's 6 entries of one site: 96 contiguous bytes to read, and 6 consecutive rows of K of one real
// column to store per lane (in B the lanes form a spin each and exchange parts), as pairs of FP16 that
// fall on 32 banks.  The ring's unit is half a K step (8 rows), a quad of sites fills three.
// Items go round the builder warps without regard to stages.  Every wait is bounded; a wait that runs out raises
// the CTA's abort flag and sets the timeout bit of the error word.
//
// Bounds: issue slots (fixed-point conversion and digits: 60 % busy over the CTA's life) together with the
// products, 9 per K step at Ntv 24 that take 1500 cycles alone and 2100 beside the builders' shared-memory traffic (each
// product reads 4 KB of A; one product per pair of slices, 28 of them, takes 3000), and the reading of the sums, 18 % of
// the time, in which no product runs.  4^4 blocks of 16^4 sites, assembly altogether: Ntv 24, DIG 7, 3.5 ms (in pairs
// of FP32 numbers on the FP32 pipes 11.4 ms); Ntv 20, DIG 8, 3.5 ms (in FP64 22.0 ms); error of D_c against 64-bit
// references 2.0e-15 with DIG 8 as with sums in FP64.  Measured slower: U_mu P in FP64 (2 x), the block's coefficients
// converted by each item (1.2 x), 8 warps on the sums and 11 or 12 builders (1.04 x).
#include "fixed.cuh"
#include "tcgen05.cuh"

#include <limits.h>
#include <string.h>

namespace {
using namespace amgfix;
using namespace amgtc5;

constexpr int kExact = 5;          // accumulators s < kExact hold exact integers
constexpr int kChunk = 12;         // K steps between two readings of them
constexpr int kSumWarps = 4, kBuildWarps = 15;
constexpr int kTcThreads = 32 * (kSumWarps + kBuildWarps + 1);
constexpr int kTcCols = 512;
constexpr int kMaxPairs = 12;
constexpr int kNoScale = 1 << 20;  // exponent of a column with a non-finite entry
constexpr int kMaxVb = 352;        // sites per block: the Gram-Schmidt takes at most 2048 entries

struct TcBars {
  uint64_t full[kMaxPairs], empty[kMaxPairs];  // K step built / its products complete
  uint64_t accfull, accempty;                  // accumulators complete / read
  uint64_t done;                               // last product complete
  uint32_t tmem;
};
constexpr int kBarBytes = 256;
constexpr int kMaxProducts = 16;   // a K step's products
static_assert(sizeof(TcBars) <= kBarBytes, "barriers");

constexpr int kHopCoef = 18;   // numbers per site: a link
// The clover term of one chirality is [[G, M], [M^dagger, -G]] with Hermitian G: diagonals of 4 + m0 + G and
// 4 + m0 - G, entries 01, 02, 12 of G, M
constexpr int kSelfCoef = 30;

struct TcPlan {
  int N, mrows, pairs;          // columns of B, rows of A (multiples of 8), K steps in the ring
  int itemsB, items, builders;  // items of 8 columns per quad of sites, of B and together; builder warps at work
  unsigned half, acc, head;     // bytes: half a K step, integer sums, barriers and tables
  size_t smem() const { return head + (size_t)pairs * 2 * half + acc; }
};
template <int DIG, bool SELF>
__host__ __device__ inline TcPlan tc_plan(int ntv, int Vb) {
  TcPlan p;
  p.N = (ntv + 7) / 8 * 16;
  p.mrows = ((SELF ? 2 : 4) * ntv + 7) / 8 * 8;
  p.half = (unsigned)DIG * (p.mrows + p.N) * 16;
  p.acc = (unsigned)p.N * 128 * 8;
  p.head = kPipeBytes + kBarBytes + kMaxProducts * 16 + (64 + 64) * sizeof(int) + kMaxVb * 2 + (unsigned)Vb * (SELF ? kSelfCoef : kHopCoef) * 8;
  p.head = (p.head + 127) / 128 * 128;
  p.pairs = kMaxPairs;
  while (p.pairs > 2 && p.head + 2 * p.pairs * p.half + p.acc > 227 * 1024) --p.pairs;
  // A warp that waits for a K step of its next quad, d quads on, has seen the one `pairs` before its last quad
  // complete; the barrier's parity tells the two K steps before in that slot apart if ceil(1.5 d) <= pairs.
  p.itemsB = (ntv + 7) / 8;
  p.items = p.itemsB + ((SELF ? 1 : 2) * ntv + 7) / 8;
  p.builders = min(kBuildWarps, p.items * (2 * p.pairs / 3));
  return p;
}

// ------------------------------------------------------------------ bounds
// e with 1.015 v < 2^e for finite v >= 0 (0 for v = 0; the margin covers roundings and the largest digit),
// kNoScale otherwise; at least -900 (smaller numbers lose bits)
__device__ inline int bound_exp(double v) {
  const int f = (__double2hiint(v * 1.015625) >> 20) & 0x7FF;
  if (f == 0x7FF) return kNoScale;
  return v == 0 ? 0 : max(f - 1022, -900);
}
// exps[blk]: [2 mu + face] bound of sum_b |Re U_ab| + |Im U_ab| over the block's links of direction mu that stay
// inside (face 0) or leave it (1), [8] of |4 + m0| + sum_b |C_ab| over the clover, then [2][ntv] of the columns of
// P.  Largest magnitude by its bits, so that a NaN wins.
constexpr int kLinkExps = 9;
// mags[blk]: [k][site] the exponent of the largest number at a site: k = 0, 1 of P's l and r columns, 2 + mu of the
// row sums of U_mu, 6 of those of the self term
constexpr int kMags = 7;
__global__ void __launch_bounds__(256) tc_bounds_kernel(const double2* __restrict__ R, const double2* __restrict__ U,
                                                        const double2* __restrict__ clov, int* __restrict__ exps,
                                                        int* __restrict__ mags, Geom g, double m0) {
  __shared__ unsigned long long red[kLinkExps + 2 * AMG_MAX_NTV];
  __shared__ int mag[kMags * kMaxVb];
  const long long blk = blockIdx.x;
  const int n = kLinkExps + 2 * g.ntv, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, Vb = (int)g.Vb;
  for (int i = threadIdx.x; i < n; i += blockDim.x) red[i] = 0;
  for (int i = threadIdx.x; i < kMags * Vb; i += blockDim.x) mag[i] = 0;
  __syncthreads();
  auto bits = [](double v) { return (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull; };
  for (int row = warp; row < 2 * g.ntv; row += 8) {
    const double2* p = R + (blk * 2 * g.ntv + row) * (long long)g.nagg;
    unsigned long long m = 0;
    for (int i = lane; i < g.nagg; i += 32) {
      const unsigned long long v = max(bits(p[i].x), bits(p[i].y));
      atomicMax(&mag[(row >= g.ntv ? Vb : 0) + i / 6], (int)(v >> 52));
      m = max(m, v);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) red[kLinkExps + row] = m;
  }
  const long long origin = block_origin(g, blk);
  for (int i = threadIdx.x; i < Vb * 24; i += blockDim.x) {  // 12 rows of links, 12 of the clover
    const int sl = i / 24, q = i % 24;
    const long long s = block_site_fast(g, origin, sl);
    double sum = q < 12 ? 0 : fabs(4.0 + m0);
    const double2* p = q < 12 ? U + (s * 12 + q) * 3 : clov + (s * 12 + q - 12) * 6;
    for (int b = 0; b < (q < 12 ? 3 : 6); ++b) sum += fabs(p[b].x) + fabs(p[b].y);
    int slot = 8;
    if (q < 12) {
      const int mu = q / 3;
      int l = sl;
      for (int m = 0; m < mu; ++m) l /= g.B[m];
      slot = 2 * mu + (l % g.B[mu] == g.B[mu] - 1);
    }
    atomicMax(&red[slot], bits(sum));
    atomicMax(&mag[(q < 12 ? 2 + q / 3 : 6) * Vb + sl], (int)(bits(sum) >> 52));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) exps[blk * n + i] = bound_exp(__longlong_as_double((long long)red[i]));
  for (int i = threadIdx.x; i < kMags * Vb; i += blockDim.x) mags[blk * kMags * Vb + i] = mag[i];
}
// left[blk][job]: 1 where, for a pair of chiralities and one kind of links (inside the block, or through the face), the
// largest product of a site's numbers lies more than kProductBits bits below the product of the largest ones.
// Gaussian test vectors and SU(3) links: at most 3 bits.  Products that are all 0 are exact, and where a number is not
// finite the result is not either.
constexpr int kProductBits = 6;
__global__ void __launch_bounds__(160) tc_left_kernel(const int* __restrict__ mags, int* __restrict__ left, Geom g) {
  const int job = threadIdx.x >> 5, lane = threadIdx.x & 31, Vb = (int)g.Vb;
  const long long blk = blockIdx.x;
  const int* M = mags + blk * kMags * Vb;
  auto wide = [](int best, int top, bool finite) {
    return best > 0 && best < top - kProductBits && finite;
  };
  bool any = false;
  if (job < 4) {
    int X[4], stride = 1, Bmu = 1;
    long long r = blk;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      X[m] = (int)(r % g.Lc[m]);
      r /= g.Lc[m];
      if (m < job) stride *= g.B[m];
      if (m == job) {
        Bmu = g.B[m];
        X[m] = X[m] + 1 < g.Lc[m] ? X[m] + 1 : 0;
      }
    }
    const long long fwd = ((long long)(X[3] * g.Lc[2] + X[2]) * g.Lc[1] + X[1]) * g.Lc[0] + X[0];
    for (int p = 0; p < 2; ++p) {  // links inside, links through the face
      const int *N = p ? mags + fwd * kMags * Vb : M, step = p ? -(Bmu - 1) * stride : stride;
      int best[2][2] = {}, ta[2] = {}, tb[2] = {}, tu = 0;
      for (int s = lane; s < Vb; s += 32) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          ta[h] = max(ta[h], M[h * Vb + s]);
          tb[h] = max(tb[h], N[h * Vb + s]);
        }
        if ((s / stride % Bmu == Bmu - 1) != (p == 1)) continue;
        const int u = M[(2 + job) * Vb + s];
        tu = max(tu, u);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const int a = M[h * Vb + s], b = N[k * Vb + s + step];
            if (a > 0 && b > 0 && u > 0) best[h][k] = max(best[h][k], a + b + u);
          }
      }
      tu = __reduce_max_sync(0xffffffffu, tu);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        ta[h] = __reduce_max_sync(0xffffffffu, ta[h]);
        tb[h] = __reduce_max_sync(0xffffffffu, tb[h]);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int k = 0; k < 2; ++k)
          any |= wide(__reduce_max_sync(0xffffffffu, best[h][k]), ta[h] + tb[k] + tu, max(max(ta[h], tb[k]), tu) < 0x7FF);
    }
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int best = 0, ta = 0, tc = 0;
      for (int s = lane; s < Vb; s += 32) {
        const int a = M[h * Vb + s], c = M[6 * Vb + s];
        ta = max(ta, a);
        tc = max(tc, c);
        if (a > 0 && c > 0) best = max(best, 2 * a + c);
      }
      ta = __reduce_max_sync(0xffffffffu, ta);
      tc = __reduce_max_sync(0xffffffffu, tc);
      any |= wide(__reduce_max_sync(0xffffffffu, best), 2 * ta + tc, max(ta, tc) < 0x7FF);
    }
  }
  if (lane == 0) left[blk * 5 + job] = any;
}

// ------------------------------------------------------------------ digits
// The factor of -b_mu in row a (see setup.cu), i, -i, -1 or 1: whether it swaps the parts, and the sign bits of
// the new real and imaginary part
struct Phase {
  bool swap;
  int re, im;
};
__device__ __forceinline__ Phase phase(int mu, int a) {
  const bool swap = !(mu & 1), minus = mu == 2 ? a == 1 : mu == 1 ? a == 1 : mu == 3;
  const int sg = minus ? INT_MIN : 0;
  return swap ? Phase{true, sg ^ INT_MIN, sg} : Phase{false, sg, sg};
}
// the digits of two consecutive K rows as pairs of FP16, most significant first, `pitch` bytes apart
template <int DIG>
__device__ __forceinline__ void put_digits(long long x0, long long x1, unsigned char* dst, unsigned pitch) {
  constexpr unsigned long long kBias = DIG == 8 ? 0x8080808080808080ull : 0x80808080808080ull;
  const unsigned long long u0 = (unsigned long long)x0 + kBias, u1 = (unsigned long long)x1 + kBias;
  __half2 c;
  const unsigned cu = 0x64806480u;  // 1152
  memcpy(&c, &cu, 4);
#pragma unroll
  for (int q = 0; q < 4; ++q) {  // bytes 2 q, 2 q + 1
    const unsigned a = q < 2 ? (unsigned)u0 : (unsigned)(u0 >> 32), b = q < 2 ? (unsigned)u1 : (unsigned)(u1 >> 32);
    const unsigned w = __byte_perm(a, b, q & 1 ? 0x7362 : 0x5140);
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      const int byte = 2 * q + o;
      if (byte >= DIG) continue;
      const unsigned h = __byte_perm(w, 0x64646464u, o ? 0x4342 : 0x4140);  // FP16 1024 + byte
      __half2 v;
      memcpy(&v, &h, 4);
      v = __hsub2(v, c);
      *reinterpret_cast<__half2*>(dst + (DIG - 1 - byte) * pitch) = v;
    }
  }
}

struct TcArgs {
  const double2 *R, *U, *clov;
  const int *exps, *left;
  double2* part;
  unsigned* err;
  Geom g;
  double m0;
};

template <int DIG, bool SELF>
__global__ void __launch_bounds__(kTcThreads, 1) assemble_tc_kernel(const TcArgs a) {
  if (a.left[blockIdx.x * 5 + (SELF ? 4 : blockIdx.y)]) return;
  extern __shared__ __align__(128) unsigned char sm[];
  const Geom& g = a.g;
  const int ntv = g.ntv, nc = g.nc, nagg = g.nagg, Vb = (int)g.Vb;
  const TcPlan pl = tc_plan<DIG, SELF>(ntv, Vb);
  Pipe* pp = reinterpret_cast<Pipe*>(sm);
  TcBars* tb = reinterpret_cast<TcBars*>(sm + kPipeBytes);
  int4* prods = reinterpret_cast<int4*>(sm + kPipeBytes + kBarBytes);
  int* eA = reinterpret_cast<int*>(prods + kMaxProducts);                // exponents of A's columns
  int* eB = eA + 64;                                              // [phase][ntv] of P's in B
  unsigned short* site_at = reinterpret_cast<unsigned short*>(eB + 64);  // local site of visiting order t
  int2* coefs = reinterpret_cast<int2*>(site_at + kMaxVb);  // [visiting order][kCoef]
  constexpr int kCoef = SELF ? kSelfCoef : kHopCoef;
  unsigned char* ring = sm + pl.head;
  long long* acc = reinterpret_cast<long long*>(ring + (size_t)pl.pairs * 2 * pl.half);  // [N][128 rows]
  const long long blk = blockIdx.x;
  const int hc = blockIdx.z, job = SELF ? 4 : blockIdx.y, mu = SELF ? 0 : job;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, N = pl.N;
  int stride = 1, Bmu = 1;
  long long fwd;
  {
    int X[4];
    long long r = blk;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      X[m] = (int)(r % g.Lc[m]);
      r /= g.Lc[m];
      if (m < mu) stride *= g.B[m];
      if (m == mu) {
        Bmu = g.B[m];
        X[m] = X[m] + 1 < g.Lc[m] ? X[m] + 1 : 0;
      }
    }
    fwd = ((long long)(X[3] * g.Lc[2] + X[2]) * g.Lc[1] + X[1]) * g.Lc[0] + X[0];
  }
  // phase 0: the links inside the block (self: all sites), phase 1: those through the face
  const int nface = SELF ? 0 : Vb / Bmu, inside = Vb - nface;
  const int quads0 = (inside + 7) / 8 * 2, quads = quads0 + (nface + 7) / 8 * 2;  // an even number: whole K steps
  const int ncolA = SELF ? ntv : nc, nB = pl.itemsB, items = pl.items;
  const int ne = kLinkExps + 2 * ntv;
  const int eu[2] = {a.exps[blk * ne + 2 * job], SELF ? 0 : a.exps[blk * ne + 2 * job + 1]};  // per phase
  for (int c = threadIdx.x; c < ncolA; c += kTcThreads) eA[c] = a.exps[blk * ne + kLinkExps + (SELF ? hc * ntv : 0) + c];
  for (int i = threadIdx.x; i < 2 * ntv; i += kTcThreads)
    eB[i] = a.exps[(i < ntv ? blk : fwd) * ne + kLinkExps + hc * ntv + (i < ntv ? i : i - ntv)];
  for (int t = threadIdx.x; t < Vb; t += kTcThreads) {  // the sites with l_mu = B_mu - 1 last
    const int r = SELF ? 0 : t % nface;
    site_at[t] = (unsigned short)(SELF ? t : r / stride * (stride * Bmu) + t / nface * stride + r % stride);
  }
  __syncthreads();
  {
    const long long origin = block_origin(g, blk);
#pragma unroll 4
    for (int i = threadIdx.x; i < Vb * kCoef; i += kTcThreads) {
      const int t = i / kCoef, q = i - t * kCoef;
      const long long site = origin + __ldg(g.soff + site_at[t]);
      double u;
      if (!SELF) {
        u = __ldg(reinterpret_cast<const double*>(a.U) + (site * 4 + mu) * 18 + q);
      } else {
        const double* C = reinterpret_cast<const double*>(a.clov) + (site * 2 + hc) * 72;
        const int k = q < 6 ? 14 * q : q < 8 ? q - 4 : q < 10 ? q - 4 : q < 12 ? q + 6 : (q - 12) / 6 * 12 + 6 + (q - 12) % 6;
        u = __ldg(C + k);
        if (q < 6) u += 4.0 + a.m0;
      }
      coefs[i] = words31(fixed<61>(u, t < inside ? eu[0] : eu[1]));
    }
  }
  // The products of a K step: accumulator column, slices of A and of B in units of 16 bytes, descriptor; bit 16 of the
  // first word: the first A slice of the exact sums, bit 17: of the others (these start from zero)
  int nprod = 0;
  for (int i = 0, wide = 256 / N; i < DIG; ++i)
    for (int s = i; s < DIG; ++nprod) {
      int n = min(DIG - s, wide);
      if (i == 0 && s < kExact) n = min(n, kExact - s);
      if (threadIdx.x == 0)
        prods[nprod] = make_int4(s * N | (i == 0 ? (s < kExact ? 1 << 16 : 1 << 17) : 0), i * pl.mrows, (s - i) * N,
                                 (int)tc5_idesc(n * N));
      s += n;
    }
  if (threadIdx.x == 0) {
    for (int s = 0; s < pl.pairs; ++s) {
      mbar_init(&tb->full[s], 2 * items);
      mbar_init(&tb->empty[s], 1);
    }
    mbar_init(&tb->accfull, 1);
    mbar_init(&tb->accempty, kSumWarps);
    mbar_init(&tb->done, 1);
    pp->abort = 0;
    fence_mbar_init();
  }
  if (warp == kSumWarps + kBuildWarps) tc5_alloc(&tb->tmem, kTcCols);
  tc5_fence_before();
  __syncthreads();
  tc5_fence_after();
  const uint32_t tmem = tb->tmem;
  const unsigned inv = 65536u / pl.pairs + 1;  // k / pairs = k inv >> 16 for the k that occur

  if (warp >= kSumWarps && warp < kSumWarps + pl.builders) {
    // ---------------------------------------------------------------- digits of A and B
    const int s = (lane >> 1) & 3, cl = lane >> 3, sa = lane & 1;
    const Phase turn0 = phase(mu, 0), turn1 = phase(mu, 1);  // of rows 0-2 and 3-5 of the r columns
    const Phase turn = sa ? turn1 : turn0;
    const double2 *own = a.R + blk * 2 * ntv * (long long)nagg, *next = a.R + fwd * 2 * ntv * (long long)nagg;
    const int shift = stride * 6, back = (Bmu - 1) * stride * 6;
    // What item i of quad t reads: A, one part (of the turned column: see Phase) of a site's 6 entries; B, the 3
    // entries of one spin.  -b_mu takes spin 1 - a to row a for mu < 2.
    auto fetch = [&](int t, int i, int part, double (&z)[6]) {
      const int p = t >= quads0, n = p ? nface : inside, x = 4 * (p ? t - quads0 : t) + s;
      const bool isB = i < nB;
      const int c = 8 * (isB ? i : i - nB) + 4 * part + cl;
#pragma unroll
      for (int k = 0; k < 6; ++k) z[k] = 0;
      if (x >= n || c >= (isB ? ntv : ncolA)) return;
      const int sl = site_at[(p ? inside : 0) + x] * 6;
      if (isB) {
        const int cross = !SELF && hc == 1 && mu < 2;
        const double2* src = (!SELF && p ? next - back : SELF ? own : own + shift) + (hc * ntv + c) * nagg + sl + 3 * (sa ^ cross);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const double2 v = __ldg(src + k);
          z[2 * k] = v.x;
          z[2 * k + 1] = v.y;
        }
      } else {
        const bool turned = !SELF && c >= ntv;
        const double* src = reinterpret_cast<const double*>(own + (SELF ? hc * ntv + c : c) * nagg + sl) +
                            (sa ^ (int)(turned && turn.swap));
        const int r0 = turned && mu < 2 ? 6 : 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          z[k] = __ldg(src + r0 + 2 * k);
          z[3 + k] = __ldg(src + 6 - r0 + 2 * k);
        }
      }
    };
    int t = 0, i = warp - kSumWarps, part = 0, slot0 = 0, slot1 = 0;
    unsigned at[3] = {0, 0, 0};  // where this lane's three pairs of rows go
    while (i >= items) {
      i -= items;
      ++t;
    }
    double zn[6];
    if (t < quads) fetch(t, i, 0, zn);
    while (t < quads) {
      double z[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) z[k] = zn[k];
      int t1 = t, i1 = i;
      if (part) {
        i1 += pl.builders;
        while (i1 >= items) {
          i1 -= items;
          ++t1;
        }
      }
      if (t1 < quads) fetch(t1, i1, part ^ 1, zn);

      const int p = t >= quads0;
      const bool isB = i < nB;
      const int c = 8 * (isB ? i : i - nB) + 4 * part + cl;
      const bool valid = c < (isB ? ntv : ncolA);
      long long v[6];
      if (isB) {
        const int ej = valid ? eB[p * ntv + c] : 0;
        int2 rx[3], ry[3];  // conj(r), turned
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if (!SELF && hc == 1) {  // phase x (re - i im)
            const double re = turn.swap ? z[2 * k + 1] : z[2 * k], im = turn.swap ? z[2 * k] : z[2 * k + 1];
            rx[k] = words31(fixed<60>(re, ej, turn.swap ? turn.re ^ INT_MIN : turn.re));
            ry[k] = words31(fixed<60>(im, ej, turn.swap ? turn.im : turn.im ^ INT_MIN));
          } else {
            rx[k] = words31(fixed<60>(z[2 * k], ej));
            ry[k] = words31(fixed<60>(z[2 * k + 1], ej, INT_MIN));
          }
        }
        const int2* cf = coefs + ((p ? inside : 0) + min(4 * (p ? t - quads0 : t) + s, (p ? nface : inside) - 1)) * kCoef;
        long long xr[3], xi[3];
        int2 ox[3], oy[3];  // self: the other spin's
        if (SELF)
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            ox[k] = make_int2(__shfl_xor_sync(0xffffffffu, rx[k].x, 1), __shfl_xor_sync(0xffffffffu, rx[k].y, 1));
            oy[k] = make_int2(__shfl_xor_sync(0xffffffffu, ry[k].x, 1), __shfl_xor_sync(0xffffffffu, ry[k].y, 1));
          }
#pragma unroll
        for (int col = 0; col < 3; ++col) {
          long long hr = 0, hi = 0, lr = 0, li = 0;  // high x high, high x low words
          auto cmac = [&](int2 ur, int2 ui, int2 x, int2 y) {
            mac(hr, lr, ur, x);
            mac(hr, lr, minus(ui), y);
            mac(hi, li, ur, y);
            mac(hi, li, ui, x);
          };
          if (!SELF) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const int4 w = *reinterpret_cast<const int4*>(cf + (col * 3 + k) * 2);
              cmac(make_int2(w.x, w.y), make_int2(w.z, w.w), rx[k], ry[k]);
            }
          } else {
            auto signed_words = [](int2 u, bool neg) { return neg ? minus(u) : u; };
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              if (k == col) {
                const int2 d = cf[3 * sa + k];
                mac(hr, lr, d, rx[k]);
                mac(hi, li, d, ry[k]);
              } else {  // +-G, its lower triangle the conjugate of the upper
                const int4 w = *reinterpret_cast<const int4*>(cf + 4 + 2 * (col + k));
                cmac(signed_words(make_int2(w.x, w.y), sa), signed_words(make_int2(w.z, w.w), (k < col) != (sa != 0)), rx[k], ry[k]);
              }
              // M from the upper rows, M^dagger from the lower
              const int4 w = *reinterpret_cast<const int4*>(cf + 12 + 2 * (sa ? k * 3 + col : col * 3 + k));
              cmac(make_int2(w.x, w.y), signed_words(make_int2(w.z, w.w), sa), ox[k], oy[k]);
            }
          }
          if (DIG == 8) {
            xr[col] = (hr << 4) + (lr >> 27);
            xi[col] = (hi << 4) + (li >> 27);
          } else {
            xr[col] = (hr + (lr >> 31) + 8) >> 4;
            xi[col] = (hi + (li >> 31) + 8) >> 4;
          }
        }
        // lane 0 of the pair takes the real parts of the site's 6 rows, lane 1 the imaginary parts
#pragma unroll
        for (int col = 0; col < 3; ++col) {
          const long long keep = sa ? xi[col] : xr[col];
          const long long got = __shfl_xor_sync(0xffffffffu, sa ? xr[col] : xi[col], 1);
          v[col] = sa ? got : keep;
          v[3 + col] = sa ? keep : got;
        }
      } else {
        const int e = valid ? eA[c] : 0;
        const bool turned = !SELF && c >= ntv;
        const int conj = sa ? INT_MIN : 0;  // of the part read: phase x (re - i im)
        // the part that goes to lane sa: re of row a is re, or (swapped) im of the entry
        const int n0 = turned ? (sa ? turn0.im : turn0.re) ^ (turn0.swap ? conj ^ INT_MIN : conj) : conj;
        const int n1 = turned ? (sa ? turn1.im : turn1.re) ^ (turn1.swap ? conj ^ INT_MIN : conj) : conj;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          v[k] = fixed<8 * DIG - 1>(z[k], e, n0);
          v[3 + k] = fixed<8 * DIG - 1>(z[3 + k], e, n1);
        }
      }
      if (!part) {  // halves 3 t .. 3 t + 2 lie in K steps k0 and k0 + 1
        const int k0 = (3 * t) >> 1, q0 = (int)((unsigned)k0 * inv >> 16), q1 = (int)((unsigned)(k0 + 1) * inv >> 16);
        slot0 = k0 - q0 * pl.pairs;
        slot1 = k0 + 1 - q1 * pl.pairs;
        bool ok = q0 == 0 || wait_phase(&tb->empty[slot0], (unsigned)((q0 - 1) & 1), pp);
        ok = ok && (q1 == 0 || wait_phase(&tb->empty[slot1], (unsigned)((q1 - 1) & 1), pp));
        if (!__all_sync(0xffffffffu, ok)) {
          abort_cta(pp, a.err);
          break;
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int e = 6 * s + 2 * q, n = (t & 1) + (e >> 3);  // half, counted from K step k0
          at[q] = (2 * (n < 2 ? slot0 : slot1) + (n & 1)) * pl.half + (isB ? DIG * pl.mrows * 16 : 0) + (e & 7) * 2 + sa * 16;
        }
      }
      if (valid) {
        const unsigned pitch = (unsigned)(isB ? N : pl.mrows) * 16;
#pragma unroll
        for (int q = 0; q < 3; ++q) put_digits<DIG>(v[2 * q], v[2 * q + 1], ring + at[q] + c * 32, pitch);
      }
      if (part) {
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&tb->full[slot0]);
          mbar_arrive(&tb->full[slot1]);
          mbar_arrive(&tb->full[t & 1 ? slot1 : slot0]);
        }
      }
      t = t1;
      i = i1;
      part ^= 1;
    }
  } else if (warp == kSumWarps + kBuildWarps) {
    // ---------------------------------------------------------------- products
    if (lane == 0) {
      const int k0 = quads0 / 2 * 3, k1 = quads / 2 * 3;
      int chunk = 0, in = 0;
      for (int k = 0; k < k1; ++k) {
        const bool start = k == 0 || k == k0;
        if (start) in = 0;
        const bool first = in == 0, last = in == kChunk - 1 || k == k0 - 1 || k == k1 - 1;
        const int use = (int)((unsigned)k * inv >> 16), slot = k - use * pl.pairs;
        bool ok = !first || chunk == 0 || wait_phase(&tb->accempty, (unsigned)((chunk - 1) & 1), pp);
        ok = ok && wait_phase(&tb->full[slot], (unsigned)(use & 1), pp);
        if (!ok) {
          abort_cta(pp, a.err);
          break;
        }
        tc5_fence_after();
        const unsigned char* A = ring + (size_t)slot * 2 * pl.half;
        const uint64_t da = tc5_desc(A, pl.half, 128u), db = tc5_desc(A + DIG * pl.mrows * 16, pl.half, 128u);
        const int fresh = (first ? 1 << 16 : 0) | (start ? 1 << 17 : 0);
        int4 q = prods[0];
        for (int i = 0; i < nprod; ++i) {
          const int4 next = prods[i + 1 < nprod ? i + 1 : 0];
          tc5_mma_ss(tmem + (uint32_t)(q.x & 0xFFFF), da + (unsigned)q.y, db + (unsigned)q.z, (uint32_t)q.w, q.x & fresh ? 0u : 1u);
          q = next;
        }
        tc5_commit(&tb->empty[slot]);
        if (++in == kChunk) in = 0;
        if (last) {
          tc5_commit(&tb->accfull);
          ++chunk;
        }
      }
      tc5_commit(&tb->done);  // every product issued has completed before tensor memory is freed
      const long long t0 = clock64();
      while (!mbar_test(&tb->done, 0) && clock64() - t0 < kWaitCycles) {
      }
    }
    __syncwarp();
  } else if (warp < kSumWarps) {
    // ---------------------------------------------------------------- sums
    const int row = warp * 32 + lane, c = row >> 1, ri = row & 1;
    const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
    double* P = reinterpret_cast<double*>(a.part + (blk * 5 + job) * 2 * (long long)nc * nc);
    const int m = SELF ? hc * ntv + c : c;
    int chunk = 0;
    bool ok = true;
    for (int p = 0; p < (SELF ? 1 : 2) && ok; ++p, P += 2 * (long long)nc * nc) {
      const int steps = (p ? quads - quads0 : quads0) / 2 * 3;
      const int ea = c < ncolA ? eA[c] : 0;
      // entry j from the sum of its real products, in units of 2^(ea + eb - 52)
      auto write = [&](int j, long long x) {
        if (c >= ncolA || j >= ntv) return;
        const int ej = eB[p * ntv + j];
        const int el = p ? eu[1] : eu[0], k = ea + ej + el - 52;
        double v = (double)x;
        if (k >= -1022 && k < 1024)
          v *= __hiloint2double((k + 1023) << 20, 0);
        else  // a column with a non-finite entry, or far from one
          v = ea == kNoScale || ej == kNoScale || el == kNoScale ? nan("") : scalbn(v, k);
        P[((long long)m * nc + hc * ntv + j) * 2 + ri] = v;
      };
      if (steps == 0)
        for (int j = 0; j < ntv; ++j) write(j, 0);
      for (int step = 0; step < steps; step += kChunk, ++chunk) {
        if (!__all_sync(0xffffffffu, wait_phase(&tb->accfull, (unsigned)(chunk & 1), pp))) {
          abort_cta(pp, a.err);
          ok = false;
          break;
        }
        tc5_fence_after();
        const bool last = step + kChunk >= steps;
        for (int n0 = 0; n0 < N; n0 += 16) {
          __syncwarp();  // converged for the collective loads
          long long sum[16];
          uint32_t v[2][16];
          tc5_ld16(taddr + (uint32_t)n0, v[0]);
#pragma unroll
          for (int d = 0; d < kExact; ++d) {
            tc5_wait_ld();
            if (d + 1 < kExact) tc5_ld16(taddr + (uint32_t)((d + 1) * N + n0), v[(d + 1) & 1]);
#pragma unroll
            for (int n = 0; n < 16; ++n) {
              const int x = __float2int_rn(__uint_as_float(v[d & 1][n]));
              const long long w = (long long)x * (long long)(1u << (d ? 32 - 8 * d : 0));
              sum[n] = d == 0 ? (long long)((unsigned long long)(unsigned)x << 32) : sum[n] + w;
            }
          }
          long long* q = acc + (size_t)n0 * 128 + row;
          if (step > 0)
#pragma unroll
            for (int n = 0; n < 16; ++n) sum[n] += q[n * 128];
          if (!last) {
#pragma unroll
            for (int n = 0; n < 16; ++n) q[n * 128] = sum[n];
            continue;
          }
          __syncwarp();
          float low[16];
#pragma unroll
          for (int d = kExact; d < DIG; ++d) {
            uint32_t v[16];
            tc5_ld16(taddr + (uint32_t)(d * N + n0), v);
            tc5_wait_ld();
            const float w = d == 5 ? 0.25f : d == 6 ? 0.25f / 256 : 0.25f / 65536;
#pragma unroll
            for (int n = 0; n < 16; ++n) low[n] = d == kExact ? __uint_as_float(v[n]) * w : fmaf(__uint_as_float(v[n]), w, low[n]);
          }
          // (Re A - i Im A)^T (Re B + i Im B): lanes of Re A write the real part, of Im A the imaginary part
#pragma unroll
          for (int n = 0; n < 16; n += 2) {
            const long long x0 = (sum[n] << 6) + __float2int_rn(low[n]), x1 = (sum[n + 1] << 6) + __float2int_rn(low[n + 1]);
            const long long got = __shfl_xor_sync(0xffffffffu, x1, 1);
            write((n0 + n) / 2, ri ? got - x0 : x0 + got);
          }
        }
        tc5_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tb->accempty);
      }
    }
  }
  tc5_fence_before();
  __syncthreads();
  tc5_fence_after();
  if (warp == kSumWarps + kBuildWarps) tc5_dealloc(tmem, kTcCols);
}

template <int DIG, bool SELF>
amg_status launch_tc(const TcArgs& a, cudaStream_t st) {
  const TcPlan pl = tc_plan<DIG, SELF>(a.g.ntv, (int)a.g.Vb);
  const size_t smem = pl.smem();
  if (smem > 227 * 1024) return AMG_ERR_UNSUPPORTED;
  AMG_CUDA_TRY(cudaFuncSetAttribute(assemble_tc_kernel<DIG, SELF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  assemble_tc_kernel<DIG, SELF><<<dim3((unsigned)a.g.Vc, SELF ? 1 : 4, 2), kTcThreads, smem, st>>>(a);
  AMG_LAUNCH_CHECK();
  return AMG_OK;
}
}  // namespace

size_t amg_internal_assemble_tc_ints(const Geom& g) {
  return (size_t)g.Vc * (5 + kLinkExps + 2 * g.ntv + kMags * g.Vb);
}

// Partial sums of the assembly (the layout the combine step reads), but those of the (block, job)s marked in work[blk 5 +
// job], which another kernel takes; work: amg_internal_assemble_tc_ints() ints
amg_status amg_internal_assemble_tc(const Geom& g, const double2* R, const double2* U, const double2* clov, int* work,
                                    double2* part, double m0, bool pair, unsigned* err, cudaStream_t st) {
  if (g.Vb > kMaxVb || 4 * g.ntv > 128) return AMG_ERR_UNSUPPORTED;
  int *left = work, *exps = left + g.Vc * 5, *mags = exps + g.Vc * (kLinkExps + 2 * g.ntv);
  tc_bounds_kernel<<<(unsigned)g.Vc, 256, 0, st>>>(R, U, clov, exps, mags, g, m0);
  AMG_LAUNCH_CHECK();
  tc_left_kernel<<<(unsigned)g.Vc, 160, 0, st>>>(mags, left, g);
  AMG_LAUNCH_CHECK();
  const TcArgs a{R, U, clov, exps, left, part, err, g, m0};
  const amg_status s = pair ? launch_tc<7, false>(a, st) : launch_tc<8, false>(a, st);
  if (s != AMG_OK) return s;
  return pair ? launch_tc<7, true>(a, st) : launch_tc<8, true>(a, st);
}
