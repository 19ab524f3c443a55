// Gram-Schmidt on aggregates (Sec. 3, "Gram-Schmidt on aggregates") in fixed point.
//
// The algorithm is that of the FP64 kernel (setup.cu): block classical Gram-Schmidt on column blocks of 4, each
// projection applied twice, then the block's columns one by one, again twice.  A column w is held as 60-bit integers
// relative to a power of two 2^ew >= ||w||, an orthonormal one relative to 1.  By the Cauchy-Schwarz inequality no
// sum over the aggregate then exceeds 2^58 in units of its products' high words, so that sums of any order
// fit 64 bits; entries are good to 2^-60 ||w|| (FP64: 2^-53 of each).  After every projection the norm is taken
// anew and the column shifted up, so that what is left of a nearly dependent column is again good to 2^-60 of
// its norm where it is projected for the second time.  Products are of words of 31 bits: high x high and the
// two high x low ones; FULL adds low x low.
//
// What is relative to a column's norm loses a site whose entries are far below the column's.  An aggregate where a test
// vector has such a site (kSiteBits bits or more, entries of 0 apart) is left to the kernels that work in floating
// point, where every entry is good relative to itself; the others' sites keep at least 47 bits.
//
// One CTA of up to 512 threads per aggregate, element n of the aggregate in thread n mod T (E per thread).  Finished
// columns wait in R as words and become doubles at the end, each element by the thread that wrote it.
//
// Bound: integer multiply-adds (12 or, FULL, 16 per complex one, at a quarter of the FP32 rate) and, with one CTA of
// 128 registers per thread on an SM, the latency of the columns' reads and of the sums' two barriers.  16^4, 4^4 blocks,
// Ntv 20, FULL: 3.24 ms, in FP64 5.49 ms; finding what to leave, a pass over the test vectors, 0.08 ms.
#include "fixed.cuh"

namespace {
using namespace amgfix;

constexpr int kNB = 4;  // columns per block
constexpr int kKG = 2;  // earlier columns per round of dots
constexpr int kSiteBits = 7;  // Gaussian entries: 4 bits between the largest and the smallest of 200,000 sites
constexpr long long kSmall = 1 << 18;

struct cw {  // complex number in words
  int2 re, im;
};
template <bool FULL>
struct Sum {  // of real products
  long long h = 0, l = 0, ll = 0;
  __device__ __forceinline__ void add(int2 a, int2 b) {
    mac(h, l, a, b);
    if (FULL) ll += (long long)a.y * b.y;
  }
  // in sixteenths of the high products' unit, rounded: the sums over the aggregate still fit, and what the threads'
  // roundings leave of a column after the second projection is as small as in FP64
  __device__ __forceinline__ long long value() const { return (h << 4) + ((l + (FULL ? ll >> 31 : 0) + (1 << 26)) >> 27); }
  // in quarters
  __device__ __forceinline__ long long fine() const { return (h << 2) + ((l + (FULL ? ll >> 31 : 0) + (1 << 28)) >> 29); }
};

// CTA sums of NV integers (a power of two, at most 16; at most 16 warps): left in out[0 .. NV - 1] (shared, valid
// after the call).  The values are halved as they go down the lanes.  red: [16][NV].
template <int NV>
__device__ __forceinline__ void totals(long long (&v)[NV], long long* red, long long* out) {
  constexpr int sh = NV == 16 ? 1 : NV == 8 ? 2 : NV == 4 ? 3 : NV == 2 ? 4 : 5;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int o = 16;
#pragma unroll
  for (int n = NV / 2; n > 0; n /= 2, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < NV / 2; ++i)
      if (i < n) {
        const long long give = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
  }
  for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  if ((lane & ((1 << sh) - 1)) == 0) red[warp * NV + (lane >> sh)] = v[0];
  __syncthreads();
  for (int t = threadIdx.x; t < (NV > 1 ? 16 * NV : 32); t += blockDim.x) {
    const int i = t >> 4, w = t & 15;
    long long x = w < nw && i < NV ? red[w * NV + i] : 0;
#pragma unroll
    for (int q = 8; q; q >>= 1) x += __shfl_xor_sync(0xffffffffu, x, q);
    if (w == 0 && i < NV) out[i] = x;
  }
  __syncthreads();
}

// left[agg]: 1 where a test vector has a site kSiteBits bits or more below its largest entry on the aggregate.  Reads the test
// vectors once.  One CTA per aggregate; thread t takes column t mod Ntv of every step-th entry.
__global__ void __launch_bounds__(512) gs_left_kernel(const double2* __restrict__ tv, int* __restrict__ left, Geom g) {
  extern __shared__ int site[];  // [sites][ntv]: exponent of a column's largest entry at a site
  __shared__ int top[AMG_MAX_NTV];
  const long long agg = blockIdx.x, origin = block_origin(g, agg >> 1);
  const int h = (int)(agg & 1), T = blockDim.x, tid = threadIdx.x, ntv = g.ntv, nagg = g.nagg, n = nagg / 6 * ntv;
  for (int i = tid; i < n; i += T) site[i] = 0;
  if (tid < ntv) top[tid] = 0;
  __syncthreads();
  const int step = T / ntv, j = tid % ntv;
  if (tid < step * ntv) {
    int f = 0;
#pragma unroll 4
    for (int i = tid / ntv; i < nagg; i += step) {
      const double2 v = __ldg(tv + (block_site_fast(g, origin, i / 6) * 12 + 6 * h + i % 6) * ntv + j);
      const int fe = max((__double2hiint(v.x) >> 20) & 0x7FF, (__double2hiint(v.y) >> 20) & 0x7FF);
      atomicMax(&site[i / 6 * ntv + j], fe);
      f = max(f, fe);
    }
    atomicMax(&top[j], f);
  }
  __syncthreads();
  bool wide = false;
  for (int i = tid; i < n; i += T) {
    const int t = top[i % ntv];
    wide |= site[i] > 0 && t != 0x7FF && t - site[i] >= kSiteBits;
  }
  wide = __syncthreads_or(wide);
  if (tid == 0) left[agg] = wide;
}

template <int E, bool FULL>
__global__ void __launch_bounds__(512) gs_fixed_kernel(const double2* __restrict__ tv, double2* __restrict__ R, Geom g,
                                                       const int* __restrict__ left, unsigned* err) {
  if (left[blockIdx.x]) return;
  __shared__ long long red[16 * 2 * kKG * kNB], tot[2 * kKG * kNB];
  __shared__ int4 coef[AMG_MAX_NTV * kNB];  // minus the coefficients
  __shared__ int top[kNB];
  __shared__ long long scal;
  const long long agg = blockIdx.x, blk = agg >> 1;
  const int h = (int)(agg & 1);
  const int T = blockDim.x, tid = threadIdx.x, ntv = g.ntv, nagg = g.nagg;
  const double2* src[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int n = tid + e * T;
    src[e] = nullptr;
    if (n < nagg) {
      const int sl = n / 6, a = (n % 6) / 3, col = n % 3;
      src[e] = tv + ((block_site(g, blk, sl) * 4 + 2 * h + a) * 3 + col) * (long long)ntv;
    }
  }
  int4* Q = reinterpret_cast<int4*>(R + agg * (long long)ntv * nagg);  // words of conj(q_k) until the end
  int bad_from = ntv;  // first column with a non-finite entry: it and what follows is not a number
  cw w[E][kNB];
  int ew[kNB] = {0, 0, 0, 0};
  double n0[kNB];
  // Shifts column c, given its norm^2 z in units of 2^(2 ew - 62), to a bound within a factor of two; by 20 bits if z is
  // too small to tell (the products of low words left out make up to 2^14 units).
  auto lift = [&](int c, long long z) {
    const int b = 64 - __clzll(z), s = z < kSmall ? 20 : b < 61 ? (62 - b) >> 1 : 0;
    if (s > 0) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        w[e][c].re = words31(joined(w[e][c].re) << s);
        w[e][c].im = words31(joined(w[e][c].im) << s);
      }
      ew[c] -= s;
    }
    return z << (2 * s);
  };
  auto norm = [&](int c) {
    Sum<FULL> s;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      s.add(w[e][c].re, w[e][c].re);
      s.add(w[e][c].im, w[e][c].im);
    }
    return s.value();
  };
  for (int j0 = 0; j0 < ntv; j0 += kNB) {
    const int nb = min(kNB, ntv - j0);
    // exponents: first 2^6 times the largest entry (at most 4096 parts), then by the norm
    if (tid < kNB) top[tid] = 0;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kNB; ++c) {
      int f = 0;
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (src[e] && c < nb) {
          const double2 v = __ldg(src[e] + j0 + c);
          f = max(f, max((__double2hiint(v.x) >> 20) & 0x7FF, (__double2hiint(v.y) >> 20) & 0x7FF));
        }
      f = __reduce_max_sync(0xffffffffu, f);
      if ((tid & 31) == 0) atomicMax(&top[c], f);
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kNB; ++c) {
      if (top[c] == 0x7FF) bad_from = min(bad_from, j0 + c);
      ew[c] = max(top[c] - 1022, -900) + 6;
    }
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
      for (int e = 0; e < E; ++e)
#pragma unroll
        for (int c = 0; c < kNB; ++c) {
          double2 v = make_double2(0, 0);
          if (src[e] && c < nb && top[c] != 0x7FF) v = __ldg(src[e] + j0 + c);
          w[e][c].re = words31(fixed<60>(v.x, ew[c]));
          w[e][c].im = words31(fixed<60>(v.y, ew[c]));
        }
      if (pass) break;
      long long v[kNB];
#pragma unroll
      for (int c = 0; c < kNB; ++c) v[c] = norm(c);
      totals<kNB>(v, red, tot);
#pragma unroll
      for (int c = 0; c < kNB; ++c) {
        const long long z = tot[c];
        n0[c] = scalbn((double)z, 2 * ew[c] - 62);
        const int b = 64 - __clzll(z);
        if (z > 0 && b < 61) ew[c] -= (62 - b) >> 1;
      }
      __syncthreads();  // tot is read
    }
    // projection against the earlier column blocks (all coefficients from the same vectors), twice
    for (int pass = 0; pass < 2 && j0 > 0; ++pass) {
      for (int k0 = 0; k0 < j0; k0 += kKG) {
        long long v[2 * kKG * kNB];
#pragma unroll
        for (int kk = 0; kk < kKG; ++kk) {
          Sum<FULL> dr[kNB], di[kNB];
#pragma unroll
          for (int e = 0; e < E; ++e) {
            if (!src[e]) continue;
            const int4 r = Q[(long long)(k0 + kk) * nagg + tid + e * T];
            const int2 rr = make_int2(r.x, r.y), ri = make_int2(r.z, r.w), ni = minus(ri);
#pragma unroll
            for (int c = 0; c < kNB; ++c) {
              dr[c].add(rr, w[e][c].re);
              dr[c].add(ni, w[e][c].im);
              di[c].add(rr, w[e][c].im);
              di[c].add(ri, w[e][c].re);
            }
          }
#pragma unroll
          for (int c = 0; c < kNB; ++c) {
            v[(kk * kNB + c) * 2] = dr[c].value();
            v[(kk * kNB + c) * 2 + 1] = di[c].value();
          }
        }
        totals<2 * kKG * kNB>(v, red, tot);
        if (tid < kKG * kNB) {
          const int2 a = words31(-((tot[2 * tid] + 2) >> 2)), b = words31(-((tot[2 * tid + 1] + 2) >> 2));
          coef[k0 * kNB + tid] = make_int4(a.x, a.y, b.x, b.y);
        }
      }
      __syncthreads();
      // w -= q_k coef_k, kUp columns to a sum: by Cauchy-Schwarz and |low words| <= 2^30 it fits
      constexpr int kUp = FULL ? 3 : 8;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        if (!src[e]) continue;
        for (int k0 = 0; k0 < j0; k0 += kUp) {
          Sum<FULL> ur[kNB], ui[kNB];
          for (int k = k0; k < min(k0 + kUp, j0); ++k) {
            const int4 r = Q[(long long)k * nagg + tid + e * T];
            const int2 rr = make_int2(r.x, r.y), ri = make_int2(r.z, r.w), ni = minus(ri);
#pragma unroll
            for (int c = 0; c < kNB; ++c) {
              const int4 f = coef[k * kNB + c];
              const int2 fr = make_int2(f.x, f.y), fi = make_int2(f.z, f.w);
              ur[c].add(rr, fr);
              ur[c].add(ri, fi);
              ui[c].add(rr, fi);
              ui[c].add(ni, fr);
            }
          }
#pragma unroll
          for (int c = 0; c < kNB; ++c) {
            w[e][c].re = words31(joined(w[e][c].re) + ur[c].fine());
            w[e][c].im = words31(joined(w[e][c].im) + ui[c].fine());
          }
        }
      }
#pragma unroll 1
      for (int tries = 0; tries < 4; ++tries) {
        long long v[kNB];
#pragma unroll
        for (int c = 0; c < kNB; ++c) v[c] = norm(c);
        totals<kNB>(v, red, tot);
        bool small = false;
#pragma unroll
        for (int c = 0; c < kNB; ++c)
          if (c < nb) {
            small |= tot[c] < kSmall;
            lift(c, tot[c]);
          }
        __syncthreads();  // tot and coef are read
        if (!small) break;
      }
    }
    // orthonormalise inside the block
#pragma unroll
    for (int c = 0; c < kNB; ++c) {
      if (c >= nb) break;
      long long z = 0;
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        if (c > 0) {
          long long v[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = 0;
#pragma unroll
          for (int cp = 0; cp < kNB - 1; ++cp)
            if (cp < c) {
              Sum<FULL> dr, di;
#pragma unroll
              for (int e = 0; e < E; ++e) {
                dr.add(w[e][cp].re, w[e][c].re);
                dr.add(w[e][cp].im, w[e][c].im);
                di.add(w[e][cp].re, w[e][c].im);
                di.add(minus(w[e][cp].im), w[e][c].re);
              }
              v[2 * cp] = dr.value();
              v[2 * cp + 1] = di.value();
            }
          totals<8>(v, red, tot);
          Sum<FULL> ur[E], ui[E];
#pragma unroll
          for (int cp = 0; cp < kNB - 1; ++cp)
            if (cp < c) {
              const int2 fr = words31(-((tot[2 * cp] + 2) >> 2)), fi = words31(-((tot[2 * cp + 1] + 2) >> 2));
#pragma unroll
              for (int e = 0; e < E; ++e) {
                ur[e].add(w[e][cp].re, fr);
                ur[e].add(minus(w[e][cp].im), fi);
                ui[e].add(w[e][cp].re, fi);
                ui[e].add(w[e][cp].im, fr);
              }
            }
#pragma unroll
          for (int e = 0; e < E; ++e) {
            w[e][c].re = words31(joined(w[e][c].re) + ur[e].fine());
            w[e][c].im = words31(joined(w[e][c].im) + ui[e].fine());
          }
          __syncthreads();  // tot is read
        } else if (pass == 0) {
          continue;
        }
#pragma unroll 1
        for (int tries = 0; tries < 4; ++tries) {
          long long v[1] = {norm(c)};
          totals<1>(v, red, tot);
          const bool small = tot[0] < kSmall;
          z = lift(c, tot[0]);
          __syncthreads();  // tot is read
          if (!small) break;
          z = 0;
        }
      }
      // q = w / ||w||: the factor 2^ew / ||w|| (1 to 2) in units of 2^-60, by one warp
      if (tid < 32) {
        const double nrm = sqrt(scalbn((double)z, 2 * ew[c] - 62));
        const double f = nrm > 0 ? 1.0 / sqrt((double)z * 0x1p-62) : 0.0;
        if (tid == 0) {
          if (!(nrm > 1e-12 * sqrt(n0[c])) || j0 + c >= bad_from) atomicOr(err, AMG_EBIT_RANK);
          scal = __double2ll_rn(f * 0x1p60);
        }
      }
      __syncthreads();
      const int2 f = words31(scal);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        Sum<FULL> sr, si;
        sr.add(w[e][c].re, f);
        si.add(w[e][c].im, f);
        w[e][c].re = words31(sr.fine());
        w[e][c].im = words31(si.fine());
      }
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if (!src[e]) continue;
#pragma unroll
      for (int c = 0; c < kNB; ++c)
        if (c < nb) {
          const int2 a = w[e][c].re, b = minus(w[e][c].im);
          Q[(long long)(j0 + c) * nagg + tid + e * T] = make_int4(a.x, a.y, b.x, b.y);
        }
    }
    __syncthreads();  // scal is read
  }
  double2* out = reinterpret_cast<double2*>(Q);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    if (!src[e]) continue;
    for (int j = 0; j < ntv; ++j) {
      const long long o = (long long)j * nagg + tid + e * T;
      const int4 r = Q[o];
      double2 v = make_double2((double)joined(make_int2(r.x, r.y)) * 0x1p-60, (double)joined(make_int2(r.z, r.w)) * 0x1p-60);
      if (j >= bad_from) v = make_double2(nan(""), nan(""));
      out[o] = v;
    }
  }
}

template <int E, bool FULL>
amg_status launch(const Geom& g, const double2* tv, double2* R, int* left, unsigned* err, cudaStream_t st) {
  const int T = (g.nagg + E * 32 - 1) / (E * 32) * 32;
  gs_left_kernel<<<(unsigned)(g.Vc * 2), 512, (size_t)g.Vb * g.ntv * sizeof(int), st>>>(tv, left, g);
  AMG_LAUNCH_CHECK();
  gs_fixed_kernel<E, FULL><<<(unsigned)(g.Vc * 2), T, 0, st>>>(tv, R, g, left, err);
  AMG_LAUNCH_CHECK();
  return AMG_OK;
}
}  // namespace

// Gram-Schmidt of every aggregate in fixed point but those marked in `left` (one int per aggregate), which another kernel
// takes; AMG_ERR_UNSUPPORTED where another kernel serves altogether: above 1536 entries per aggregate, and
//   in FP64, up to 4 test vectors of large aggregates (16^4, 4^4 blocks, Ntv 2: 0.125 ms, the FP64 kernel 0.105 ms; Ntv
//     8: 0.75 and 0.97 ms),
//   in pairs, large aggregates, where FP32 pairs are as fast and need less latency hiding (4^4 blocks, Ntv 24: 3.65 ms,
//     pairs 3.61 ms; Ntv 8: 0.65 and 0.53 ms; 64-site blocks, Ntv 20: 2.27 and 2.50 ms; 2^4 blocks, Ntv 24: 3.53 and 9.63 ms).
amg_status amg_internal_gs_fixed(const Geom& g, const double2* tv, double2* R, int* left, bool pair, unsigned* err,
                                 cudaStream_t st) {
  if (pair && g.nagg <= 512)
    return g.nagg <= 256 ? launch<1, false>(g, tv, R, left, err, st) : launch<2, false>(g, tv, R, left, err, st);
  if (pair || g.nagg > 1536 || (g.ntv <= 4 && g.nagg > 512)) return AMG_ERR_UNSUPPORTED;
  if (g.nagg <= 256) return launch<1, true>(g, tv, R, left, err, st);
  return g.nagg <= 1024 ? launch<2, true>(g, tv, R, left, err, st) : launch<3, true>(g, tv, R, left, err, st);
}
