// Fine-grid part of the two-level method around the coarse-grid correction:
//   D        the Wilson-clover operator (the fine operator whose blocks Eq. cgo restricts),
//   SAP      the domain-decomposition smoother of Alg. 3 (multiplicative Schwarz over two block
//            colours, each block system solved by minimal-residual steps),
//   V-cycle  Alg. 1: the smoother started from the coarse-grid correction of Alg. 2,
//   solve    the outer FGMRES of Sec. 1, right-preconditioned with the V-cycle.
//
// D psi(x) = (4 + m0) psi(x) + C(x) psi(x)
//            - 1/2 sum_mu [(1 - g_mu) U_mu(x) psi(x + mu) + (1 + g_mu) U_mu(x - mu)^dag psi(x - mu)],
// periodic, chiral basis g_mu = [[0, A_mu], [A_mu^dag, 0]] with A = -i sigma_1, -i sigma_2, -i sigma_3, 1.
// Each hop is spin-projected: with psi = (u, d) (spins 0,1 and 2,3),
//   (1 - g) psi = (h, -A^dag h), h = u - A d;   (1 + g) psi = (h', A^dag h'), h' = u + A d,
// so a hop costs two colour mat-vecs (on h) instead of four.  The clover term acts on the two
// chirality halves with the handle's 6x6 blocks C^{ll}, C^{rr}.
//
// The smoother's blocks are the aggregation blocks.  One half sweep (colour c) is one launch: one
// CTA per block of colour c and group of right-hand sides (FP64: per right-hand side), one thread
// per site.  The CTA forms the residual r = y - D x on its sites (the neighbours outside the block
// have the other colour and are not written in this launch), runs n_mr MR steps on B e = r with
// B = D without the hops that cross the block face (rho in shared memory, block-wide sums), and
// adds e to x.
//
// FP32 keeps the links and the clover of the fine lattice in an order of its own (see kLinkQ).
#include "fixed.cuh"
#include "pipe.cuh"

#include <limits.h>
#include <math.h>

#include <algorithm>
#include <complex>
#include <type_traits>
#include <vector>

namespace {

template <typename T> struct Cx;
template <> struct Cx<double> { using type = double2; };
template <> struct Cx<float> { using type = float2; };

template <typename C> __device__ __forceinline__ C zadd(C a, C b) { a.x += b.x; a.y += b.y; return a; }
template <typename C> __device__ __forceinline__ C zsub(C a, C b) { a.x -= b.x; a.y -= b.y; return a; }
template <typename C> __device__ __forceinline__ C zneg(C a) { a.x = -a.x; a.y = -a.y; return a; }
template <typename C> __device__ __forceinline__ C zi(C a) { C r; r.x = -a.y; r.y = a.x; return r; }    // i a
template <typename C> __device__ __forceinline__ C zmi(C a) { C r; r.x = a.y; r.y = -a.x; return r; }   // -i a
template <typename C> __device__ __forceinline__ C zzero() { C r; r.x = 0; r.y = 0; return r; }
template <typename C, typename T> __device__ __forceinline__ C zscale(C a, T s) { a.x *= s; a.y *= s; return a; }
template <typename C> __device__ __forceinline__ void zfma(C& acc, C a, C b) {  // acc += a b
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}
template <typename C> __device__ __forceinline__ void zfmac(C& acc, C a, C b) {  // acc += conj(a) b
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(-a.y, b.x, acc.y);
}

// (A_mu d)_s, s = 0, 1
template <typename C>
__device__ __forceinline__ void amul(int mu, C d0, C d1, C& o0, C& o1) {
  if (mu == 0) { o0 = zmi(d1); o1 = zmi(d0); }          // -i sigma_1
  else if (mu == 1) { o0 = zneg(d1); o1 = d0; }         // -i sigma_2 = [[0, -1], [1, 0]]
  else if (mu == 2) { o0 = zmi(d0); o1 = zi(d1); }      // -i sigma_3
  else { o0 = d0; o1 = d1; }                            // 1
}
// (A_mu^dag v)_s
template <typename C>
__device__ __forceinline__ void adagmul(int mu, C v0, C v1, C& o0, C& o1) {
  if (mu == 0) { o0 = zi(v1); o1 = zi(v0); }            // i sigma_1
  else if (mu == 1) { o0 = v1; o1 = zneg(v0); }         // i sigma_2 = [[0, 1], [-1, 0]]
  else if (mu == 2) { o0 = zi(v0); o1 = zmi(v1); }      // i sigma_3
  else { o0 = v0; o1 = v1; }
}

// out += -1/2 (1 - g_mu) U p   (FWD) or   out += -1/2 (1 + g_mu) U^dag p   (!FWD); p, out: [spin][colour];
// u: the link's 3x3 entries
template <bool FWD, int mu, typename C>
__device__ __forceinline__ void hop_u(const C u[9], const C p[12], C out[12]) {
  C h[2][3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    C a0, a1;
    amul(mu, p[6 + c], p[9 + c], a0, a1);
    h[0][c] = FWD ? zsub(p[c], a0) : zadd(p[c], a0);
    h[1][c] = FWD ? zsub(p[3 + c], a1) : zadd(p[3 + c], a1);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    C w0 = zzero<C>(), w1 = zzero<C>();
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      if (FWD) {
        zfma(w0, u[a * 3 + b], h[0][b]);
        zfma(w1, u[a * 3 + b], h[1][b]);
      } else {
        zfmac(w0, u[b * 3 + a], h[0][b]);
        zfmac(w1, u[b * 3 + a], h[1][b]);
      }
    }
    C d0, d1;
    adagmul(mu, w0, w1, d0, d1);
    // upper half -1/2 W; lower half +1/2 A^dag W (forward) or -1/2 A^dag W (backward)
    out[a] = zsub(out[a], zscale(w0, 0.5));
    out[3 + a] = zsub(out[3 + a], zscale(w1, 0.5));
    if (FWD) {
      out[6 + a] = zadd(out[6 + a], zscale(d0, 0.5));
      out[9 + a] = zadd(out[9 + a], zscale(d1, 0.5));
    } else {
      out[6 + a] = zsub(out[6 + a], zscale(d0, 0.5));
      out[9 + a] = zsub(out[9 + a], zscale(d1, 0.5));
    }
  }
}

// The 3x3 link at U9 = U + (s 4 + mu) 9 (FP64)
__device__ __forceinline__ void load_link(const double2* __restrict__ U9, double2 u[9]) {
#pragma unroll
  for (int k = 0; k < 9; ++k) u[k] = __ldg(U9 + k);
}

template <bool FWD, int mu>
__device__ __forceinline__ void hop(const double2* __restrict__ U, const double2 p[12], double2 out[12]) {
  double2 u[9];
  load_link(U, u);
  hop_u<FWD, mu>(u, p, out);
}

// Row of six clover entries (FP64 blocks)
__device__ __forceinline__ void clover_row(const double2* __restrict__ row, double2 c[6]) {
#pragma unroll
  for (int b = 0; b < 6; ++b) c[b] = __ldg(row + b);
}

// out = (4 + m0) p + C(x) p for the site whose clover blocks start at Cl ([2][6][6])
template <typename C, typename T>
__device__ __forceinline__ void site_term(const C* __restrict__ Cl, T mass, const C p[12], C out[12]) {
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      C acc = zscale(p[hh * 6 + a], mass), c[6];
      clover_row(Cl + (hh * 6 + a) * 6, c);
#pragma unroll
      for (int b = 0; b < 6; ++b) zfma(acc, c[b], p[hh * 6 + b]);
      out[hh * 6 + a] = acc;
    }
  }
}

// FP32 links and clover in HBM: per site kLinkQ 16-byte words of links (36 entries, two per word,
// direction mu at entries 9 mu .. 9 mu + 8) and kClovQ words of clover, block by block: word q of the
// site with local index t in block b at (b NQ + q) Vb + t.  A block's links (and its clover) are one
// contiguous run, which one bulk copy moves, and consecutive lanes read consecutive words; with one
// record per site in lattice order (strides of 288 and 352 bytes) every load of a warp touched up to
// 32 lines, and the line look-ups in L1 bounded D.
//
// The clover of a chirality is [[H, X], [X^dag, -H]] with H = H^dag (spin blocks sigma_m (x) G_m with
// Hermitian G_m): 27 real numbers instead of 36, as 14 complex words (H00, H11), (H22, 0), H01, H02,
// H12, X row by row.  The links are stored halved (exactly), so that the hops have weight one and the
// sums below are D psi itself: with sums of 2 D psi, halved at the end, D psi and <B rho, B rho> left
// the FP32 range by a factor of 2 and 4 sooner.
constexpr int kLinkQ = 18, kClovQ = 14;

__device__ __forceinline__ float2 lo2(float4 f) { return make_float2(f.x, f.y); }
__device__ __forceinline__ float2 hi2(float4 f) { return make_float2(f.z, f.w); }
// The link of direction mu of a site whose first word is U, words `stride` apart: four 16-byte words
// and half of a fifth
template <int mu>
__device__ __forceinline__ void load_link(const float4* __restrict__ U, int stride, float2 u[9]) {
  constexpr int e0 = 9 * mu, o = e0 & 1, p0 = e0 >> 1;
  u[o ? 0 : 8] = __ldg(reinterpret_cast<const float2*>(U + (o ? p0 : p0 + 4) * stride) + o);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 f = __ldg(U + (p0 + o + k) * stride);
    u[o + 2 * k] = lo2(f);
    u[o + 2 * k + 1] = hi2(f);
  }
}

// N 16-byte words, `stride` words apart, of shared memory or (load_words) read-only global memory
template <int N>
__device__ __forceinline__ void put_words(float4* S, int stride, const float2 p[2 * N]) {
#pragma unroll
  for (int k = 0; k < N; ++k) S[k * stride] = make_float4(p[2 * k].x, p[2 * k].y, p[2 * k + 1].x, p[2 * k + 1].y);
}
template <int N>
__device__ __forceinline__ void get_words(const float4* S, int stride, float2 p[2 * N]) {
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const float4 f = S[k * stride];
    p[2 * k] = lo2(f);
    p[2 * k + 1] = hi2(f);
  }
}
template <int N>
__device__ __forceinline__ void load_words(const float4* __restrict__ G, int stride, float2 p[2 * N]) {
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const float4 f = __ldg(G + k * stride);
    p[2 * k] = lo2(f);
    p[2 * k + 1] = hi2(f);
  }
}
// 16-byte global -> shared copy that bypasses the registers (and L1)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// load_link from shared memory
template <int mu>
__device__ __forceinline__ void shared_link(const float4* U, int stride, float2 u[9]) {
  constexpr int e0 = 9 * mu, o = e0 & 1, p0 = e0 >> 1;
  u[o ? 0 : 8] = reinterpret_cast<const float2*>(U + (o ? p0 : p0 + 4) * stride)[o];
  get_words<4>(U + (p0 + o) * stride, stride, u + o);
}

// h = (1 -+ g_mu) p on the upper half: u - A d (FWD), u + A d; h[3 s + colour]
template <bool FWD, int mu>
__device__ __forceinline__ void half_spinor(const float2 p[12], float2 h[6]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float2 a0, a1;
    amul(mu, p[6 + c], p[9 + c], a0, a1);
    h[c] = FWD ? zsub(p[c], a0) : zadd(p[c], a0);
    h[3 + c] = FWD ? zsub(p[3 + c], a1) : zadd(p[3 + c], a1);
  }
}
// row a of U h (FWD) or U^dag h for both spins
template <bool FWD>
__device__ __forceinline__ void colour_row(const float2* u, const float2 h[6], int a, float2& w0, float2& w1) {
  w0 = w1 = make_float2(0.f, 0.f);
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    if (FWD) {
      zfma(w0, u[a * 3 + b], h[b]);
      zfma(w1, u[a * 3 + b], h[3 + b]);
    } else {
      zfmac(w0, u[b * 3 + a], h[b]);
      zfmac(w1, u[b * 3 + a], h[3 + b]);
    }
  }
}
// o += -(1 -+ g_mu)-hop for colour a of the product w: -w on the upper half, +- A^dag w on
// the lower
template <bool FWD, int mu>
__device__ __forceinline__ void add_hop(float2 w0, float2 w1, int a, float2 o[12]) {
  float2 d0, d1;
  adagmul(mu, w0, w1, d0, d1);
  o[a] = zsub(o[a], w0);
  o[3 + a] = zsub(o[3 + a], w1);
  o[6 + a] = FWD ? zadd(o[6 + a], d0) : zsub(o[6 + a], d0);
  o[9 + a] = FWD ? zadd(o[9 + a], d1) : zsub(o[9 + a], d1);
}
template <bool FWD, int mu>
__device__ __forceinline__ void hop2(const float2* u, const float2 p[12], float2 o[12]) {
  float2 h[6], w0, w1;
  half_spinor<FWD, mu>(p, h);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    colour_row<FWD>(u, h, a, w0, w1);
    add_hop<FWD, mu>(w0, w1, a, o);
  }
}

// out = (mass + C) p from the site's clover words c (14 complex per chirality)
__device__ __forceinline__ void site_term_words(const float2 c[2 * kClovQ], float mass, const float2 p[12], float2 out[12]) {
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    const float2* k = c + hh * kClovQ;
    const float2 *u = p + hh * 6, *d = u + 3;
    const float dg[3] = {k[0].x, k[0].y, k[1].x};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float2 s0 = zscale(u[a], mass), s1 = zscale(d[a], mass);
      s0.x = fmaf(dg[a], u[a].x, s0.x);
      s0.y = fmaf(dg[a], u[a].y, s0.y);
      s1.x = fmaf(-dg[a], d[a].x, s1.x);
      s1.y = fmaf(-dg[a], d[a].y, s1.y);
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (a < b) {
          const float2 hab = k[1 + a + b];  // H01, H02, H12 at words 2, 3, 4
          zfma(s0, hab, u[b]);
          zfma(s1, zneg(hab), d[b]);
        } else if (a > b) {
          const float2 hba = k[1 + a + b];
          zfmac(s0, hba, u[b]);
          zfmac(s1, zneg(hba), d[b]);
        }
        zfma(s0, k[5 + 3 * a + b], d[b]);
        zfmac(s1, k[5 + 3 * b + a], u[b]);
      }
      out[hh * 6 + a] = s0;
      out[hh * 6 + 3 + a] = s1;
    }
  }
}
// Division by an invariant d of n < 2^31: n / d = (mulhi(m, n) + n) >> l with l = ceil(log2 d) and
// m = floor(2^32 (2^l - d) / d) + 1 (Granlund and Montgomery 1994)
struct FastDiv {
  unsigned d, m, l;
};
FastDiv fast_div(unsigned d) {
  FastDiv f{d, 0, 0};
  while ((1ull << f.l) < d) ++f.l;
  f.m = (unsigned)((((1ull << f.l) - d) << 32) / d + 1);
  return f;
}
// n / d; rem: n % d
__device__ __forceinline__ unsigned divide(unsigned n, const FastDiv& f, int& rem) {
  const unsigned q = (__umulhi(f.m, n) + n) >> f.l;
  rem = (int)(n - q * f.d);
  return q;
}

struct FineGeom {
  int L[4];
  long long V;
  int B[4];
  int Lc[4];
  int Vb;
  FastDiv dL[3], dB[3], dLc[3], dVb;
};

__device__ __forceinline__ void coords_of(unsigned s, const FastDiv d[3], int x[4]) {
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) s = divide(s, d[mu], x[mu]);
  x[3] = (int)s;
}
__device__ __forceinline__ void site_coords(const FineGeom& g, long long s, int x[4]) { coords_of((unsigned)s, g.dL, x); }

__device__ __forceinline__ long long site_of(const FineGeom& g, const int x[4]) {
  return (((long long)x[3] * g.L[2] + x[2]) * g.L[1] + x[1]) * g.L[0] + x[0];
}

// Lattice site of local index t in the block at coordinates X
__device__ __forceinline__ long long local_site(const FineGeom& g, const int X[4], int t) {
  int c[4];
  coords_of((unsigned)t, g.dB, c);
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) c[mu] += X[mu] * g.B[mu];
  return site_of(g, c);
}

template <typename C>
__device__ __forceinline__ void load12(const C* __restrict__ v, long long site, int nrhs, int r, C p[12]) {
  if (nrhs == 1 && sizeof(C) == 8) {  // one column of FP32: six 16-byte loads
    const float4* q = reinterpret_cast<const float4*>(v + site * 12);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float4 f = __ldg(q + k);
      p[2 * k].x = f.x;
      p[2 * k].y = f.y;
      p[2 * k + 1].x = f.z;
      p[2 * k + 1].y = f.w;
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < 12; ++k) p[k] = v[(site * 12 + k) * nrhs + r];
}

// site +- mu (periodic) from the coordinates of site s
template <int mu, int dir>
__device__ __forceinline__ long long nbr_site(const FineGeom& g, long long s, const int x[4]) {
  long long st = 1;
#pragma unroll
  for (int k = 0; k < mu; ++k) st *= g.L[k];
  if (dir > 0) return x[mu] + 1 < g.L[mu] ? s + st : s - st * (g.L[mu] - 1);
  return x[mu] > 0 ? s - st : s + st * (g.L[mu] - 1);
}

// out += all 8 hops of D at site s (neighbour spinors from v), FP64
__device__ __forceinline__ void all_hops(const FineGeom& g, const double2* __restrict__ U, const double2* __restrict__ v,
                                         long long s, const int x[4], int nrhs, int r, double2 o[12]) {
  double2 p[12];
#define AMG_HOPS(MU)                                      \
  {                                                       \
    const long long sf = nbr_site<MU, 1>(g, s, x);        \
    load12(v, sf, nrhs, r, p);                            \
    hop<true, MU>(U + (s * 4 + MU) * 9, p, o);            \
    const long long sb = nbr_site<MU, -1>(g, s, x);       \
    load12(v, sb, nrhs, r, p);                            \
    hop<false, MU>(U + (sb * 4 + MU) * 9, p, o);          \
  }
  AMG_HOPS(0)
  AMG_HOPS(1)
  AMG_HOPS(2)
  AMG_HOPS(3)
#undef AMG_HOPS
}

// out = D psi (SUB: out = y - D psi), one thread per (site, right-hand side); FP64
template <bool SUB>
__global__ void __launch_bounds__(128) dirac_kernel(const double2* __restrict__ U, const double2* __restrict__ Cl,
                                                    const double2* __restrict__ psi, const double2* __restrict__ y,
                                                    double2* __restrict__ out, FineGeom g, double mass, int nrhs) {
  const long long total = g.V * nrhs;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long s = e / nrhs;
    const int r = (int)(e % nrhs);
    int x[4];
    site_coords(g, s, x);
    double2 p[12], o[12];
    load12(psi, s, nrhs, r, p);
    site_term(Cl + s * 72, mass, p, o);
    all_hops(g, U, psi, s, x, nrhs, r, o);
    if (SUB) {
      load12(y, s, nrhs, r, p);
#pragma unroll
      for (int k = 0; k < 12; ++k) o[k] = zsub(p[k], o[k]);
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) out[(s * 12 + k) * nrhs + r] = o[k];
  }
}

// Block coordinates of block k, and the block one step along mu
__device__ __forceinline__ int block_of(const FineGeom& g, const int X[4]) {
  return ((X[3] * g.Lc[2] + X[2]) * g.Lc[1] + X[1]) * g.Lc[0] + X[0];
}
template <int mu, int dir>
__device__ __forceinline__ int block_next(const FineGeom& g, const int X[4]) {
  int Y[4] = {X[0], X[1], X[2], X[3]};
  Y[mu] = dir > 0 ? (X[mu] + 1 < g.Lc[mu] ? X[mu] + 1 : 0) : (X[mu] > 0 ? X[mu] - 1 : g.Lc[mu] - 1);
  return block_of(g, Y);
}

// First word of the site below along mu (its link of direction mu carries the backward hop)
template <int mu>
__device__ __forceinline__ const float4* link_below(const FineGeom& g, const float4* U, const float4* Us, const int X[4],
                                                    const int lc[4], int t, int stride) {
  if (lc[mu] > 0) return Us - stride;
  return U + (long long)block_next<mu, -1>(g, X) * kLinkQ * g.Vb + t + (g.B[mu] - 1) * stride;
}

// The same in FP32, several columns: lanes over (site in block order, group of NC columns), so that the
// columns of a site are read together and its links and clover are broadcast.  With an even number of
// columns a thread takes two (16-byte loads, half as many link and clover loads per column) where that
// needs less time by waves (dirac32_columns).  FAST: fewer than 2^31 threads.
template <int NC>
__device__ __forceinline__ void load_cols(const float2* __restrict__ v, long long site, int nrhs, int r, float2 p[NC][12]) {
  if constexpr (NC == 1) {
    load12(v, site, nrhs, r, p[0]);
  } else {
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const float4 f = __ldg(reinterpret_cast<const float4*>(v + (site * 12 + k) * nrhs + r));
      p[0][k] = lo2(f);
      p[1][k] = hi2(f);
    }
  }
}
constexpr int dirac32_ctas(int nc) { return nc == 1 ? 4 : 3; }  // per SM
template <bool SUB, bool FAST, int NC>
__global__ void __launch_bounds__(128, dirac32_ctas(NC)) dirac32_kernel(const float4* __restrict__ U,
                                                                       const float4* __restrict__ Cl,
                                                                       const float2* __restrict__ psi,
                                                                       const float2* __restrict__ y,
                                                                       float2* __restrict__ out, FineGeom g, float mass,
                                                                       FastDiv dn) {
  const int groups = (int)dn.d, nrhs = groups * NC;
  const long long total = g.V * groups;
  const int Vb = g.Vb;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    int r, t, X[4], lc[4], x[4];
    unsigned i;
    if (FAST) {
      i = divide((unsigned)e, dn, r);
    } else {
      i = (unsigned)(e / groups);
      r = (int)(e % groups);
    }
    r *= NC;
    const unsigned b = divide(i, g.dVb, t);
    coords_of(b, g.dLc, X);
    coords_of((unsigned)t, g.dB, lc);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) x[mu] = X[mu] * g.B[mu] + lc[mu];
    const long long s = site_of(g, x);
    float2 p[NC][12], o[NC][12];
    load_cols<NC>(psi, s, nrhs, r, p);
    {
      float2 c[2 * kClovQ];
      load_words<kClovQ>(Cl + (long long)b * kClovQ * Vb + t, Vb, c);
#pragma unroll
      for (int k = 0; k < NC; ++k) site_term_words(c, mass, p[k], o[k]);
    }
    const float4* Us = U + (long long)b * kLinkQ * Vb + t;
    int stride = 1;
#define AMG_HOPS2(MU)                                                                              \
  {                                                                                                \
    float2 u[9];                                                                                   \
    load_cols<NC>(psi, nbr_site<MU, 1>(g, s, x), nrhs, r, p);                                      \
    load_link<MU>(Us, Vb, u);                                                                      \
    _Pragma("unroll") for (int k = 0; k < NC; ++k) hop2<true, MU>(u, p[k], o[k]);                  \
    load_cols<NC>(psi, nbr_site<MU, -1>(g, s, x), nrhs, r, p);                                     \
    load_link<MU>(link_below<MU>(g, U, Us, X, lc, t, stride), Vb, u);                              \
    _Pragma("unroll") for (int k = 0; k < NC; ++k) hop2<false, MU>(u, p[k], o[k]);                 \
    stride *= g.B[MU];                                                                             \
  }
    AMG_HOPS2(0)
    AMG_HOPS2(1)
    AMG_HOPS2(2)
    AMG_HOPS2(3)
#undef AMG_HOPS2
    if (SUB) load_cols<NC>(y, s, nrhs, r, p);
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int k = 0; k < 12; ++k)
        if (SUB) o[c][k] = zsub(p[c][k], o[c][k]);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      float2* q = out + (s * 12 + k) * nrhs + r;
      if constexpr (NC == 1) *q = o[0][k];
      else *reinterpret_cast<float4*>(q) = make_float4(o[0][k].x, o[0][k].y, o[1][k].x, o[1][k].y);
    }
  }
}

// One column: a CTA takes nb whole blocks (at most kDiracSites sites, one thread each, in the block order
// of the links and the clover).  Their spinors are copied to shared memory in runs and serve the hops
// inside a block; a neighbour across a block face is read from global memory, through the same
// (generic) load, so that the hops have no branches and their loads overlap.  The links and the clover
// are read as they are needed, consecutive words by consecutive lanes.  The result goes out through
// the spinor tile.
//
// Bounds: HBM (696 bytes per site), reached as far as two CTAs per SM cover each other's waits.
// 32^3 x 64: 305 us, 70 % of the copy bandwidth.  One thread per site in lattice order with records of 288
// and 352 bytes took 509 us (3,150 line look-ups in L1 per warp of sites).
constexpr int kDiracSites = 256;
constexpr int kRec = 7;  // words per record in the tile: 16-byte accesses of 8 consecutive sites hit all banks
template <bool SUB>
__global__ void __launch_bounds__(kDiracSites, 2) dirac32_block_kernel(const float4* __restrict__ U,
                                                                       const float4* __restrict__ Cl, const float2* psi,
                                                                       const float2* __restrict__ y, float2* out,
                                                                       FineGeom g, float mass, int nb, int nblocks) {
  __shared__ float4 tile[kDiracSites * kRec];
  __shared__ unsigned lex[kDiracSites];
  const int Vb = g.Vb, b0 = blockIdx.x * nb, n = min(nb, nblocks - b0) * Vb, i = threadIdx.x;
  const bool act = i < n;
  int t, X[4], lc[4], x[4];
  const int b = b0 + (int)divide((unsigned)(act ? i : 0), g.dVb, t);
  coords_of((unsigned)b, g.dLc, X);
  coords_of((unsigned)t, g.dB, lc);
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) x[mu] = X[mu] * g.B[mu] + lc[mu];
  const long long s = site_of(g, x);
  if (act) lex[i] = (unsigned)s;
  __syncthreads();
  for (int e = i; e < n * 6; e += blockDim.x)
    cp_async16(tile + e / 6 * kRec + e % 6, reinterpret_cast<const float4*>(psi) + (long long)lex[e / 6] * 6 + e % 6);
  float2 o[12], p[12];
  float2 c[2 * kClovQ];
  load_words<kClovQ>(Cl + (long long)b * kClovQ * Vb + t, Vb, c);
  cp_async_wait_all();
  __syncthreads();
  if (act) {
    const float4* own = tile + i * kRec;
    get_words<6>(own, 1, p);
    site_term_words(c, mass, p, o);
    const float4* Us = U + (long long)b * kLinkQ * Vb + t;
    int stride = 1;
#define AMG_HOPS2(MU)                                                                                          \
  {                                                                                                            \
    float2 u[9];                                                                                               \
    const float4* q = lc[MU] + 1 < g.B[MU] ? own + stride * kRec                                               \
                                           : reinterpret_cast<const float4*>(psi + nbr_site<MU, 1>(g, s, x) * 12); \
    load_link<MU>(Us, Vb, u);                                                                                  \
    get_words<6>(q, 1, p);                                                                                     \
    hop2<true, MU>(u, p, o);                                                                                   \
    q = lc[MU] > 0 ? own - stride * kRec : reinterpret_cast<const float4*>(psi + nbr_site<MU, -1>(g, s, x) * 12); \
    load_link<MU>(link_below<MU>(g, U, Us, X, lc, t, stride), Vb, u);                                          \
    get_words<6>(q, 1, p);                                                                                     \
    hop2<false, MU>(u, p, o);                                                                                  \
    stride *= g.B[MU];                                                                                         \
  }
    AMG_HOPS2(0)
    AMG_HOPS2(1)
    AMG_HOPS2(2)
    AMG_HOPS2(3)
#undef AMG_HOPS2
    if (SUB) {
      load12(y, s, 1, 0, p);
#pragma unroll
      for (int k = 0; k < 12; ++k) o[k] = zsub(p[k], o[k]);
    }
  }
  __syncthreads();
  if (act) put_words<6>(tile + i * kRec, 1, o);
  __syncthreads();
  for (int e = i; e < n * 6; e += blockDim.x)
    reinterpret_cast<float4*>(out)[(long long)lex[e / 6] * 6 + e % 6] = tile[e / 6 * kRec + e % 6];
}

// MR coefficient alpha = <p, rho> / <p, p> from per-thread partial sums v = (<p,p>, Re, Im <p,rho>):
// warp sums, then the CTA sum and the division by one thread (FP64 is slow on this GPU: every thread
// summing and dividing would keep the FP64 pipe busy), alpha broadcast through shared memory.
// ok = false when <p, p> = 0.  red: 3 doubles per warp + 3 doubles.  FP64.
__device__ __forceinline__ void cta_alpha(double v[3], double* red, double2& al, bool& ok) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  __syncthreads();  // red may still be read by the previous call
  if (lane == 0)
    for (int k = 0; k < 3; ++k) red[warp * 3 + k] = v[k];
  __syncthreads();
  double* out = red + 3 * nw;
  if (threadIdx.x == 0) {
    double sp = 0, sr = 0, si = 0;
    for (int w = 0; w < nw; ++w) {
      sp += red[w * 3];
      sr += red[w * 3 + 1];
      si += red[w * 3 + 2];
    }
    out[0] = sp > 0 ? sr / sp : 0.0;
    out[1] = sp > 0 ? si / sp : 0.0;
    red[3 * nw + 2] = sp > 0 ? 1.0 : 0.0;
  }
  __syncthreads();
  al.x = out[0];
  al.y = out[1];
  ok = out[2] != 0.0;
}

// The same coefficient in FP32 with one barrier: each warp's lane 0 writes the warp's partial sums to its
// slot of red (3 values per warp, FP32), and after the barrier every thread sums the slots in warp
// order and divides, so that all threads hold the same alpha (the order and the arithmetic of
// cta_alpha, hence the same value).  Callers alternate between two red buffers from one step to the
// next, so that a step's writes never meet the previous step's reads.
__device__ __forceinline__ void cta_alpha_all(float v[3], float* red, float2& al, bool& ok) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  if (lane == 0)
    for (int k = 0; k < 3; ++k) red[warp * 3 + k] = v[k];
  __syncthreads();
  float sp = 0, sr = 0, si = 0;
  for (int w = 0; w < nw; ++w) {
    sp += red[w * 3];
    sr += red[w * 3 + 1];
    si += red[w * 3 + 2];
  }
  ok = sp > 0;
  al.x = ok ? sr / sp : 0.f;
  al.y = ok ? si / sp : 0.f;
}

// The same for `lanes` lanes of a warp (a power of two) that hold a whole block
__device__ __forceinline__ void lanes_alpha(float v[3], int lanes, float2& al, bool& ok) {
#pragma unroll
  for (int k = 0; k < 3; ++k)
    for (int o = lanes / 2; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  ok = v[0] > 0;
  al.x = ok ? v[1] / v[0] : 0.f;
  al.y = ok ? v[2] / v[0] : 0.f;
}

// Intra-block hops of the block operator B at local site t: neighbours' rho from shared memory
// (component-major: rho[q * Vb + t]), links from global memory; FP64.
template <int mu>
__device__ __forceinline__ void block_hops_mu(const FineGeom& g, const double2* __restrict__ U, const double2* rho,
                                              int t, long long s, const int x[4], const int lc[4], int stride,
                                              double2 o[12]) {
  double2 p[12];
  if (lc[mu] + 1 < g.B[mu]) {
#pragma unroll
    for (int q = 0; q < 12; ++q) p[q] = rho[q * g.Vb + t + stride];
    hop<true, mu>(U + (s * 4 + mu) * 9, p, o);
  }
  if (lc[mu] > 0) {
#pragma unroll
    for (int q = 0; q < 12; ++q) p[q] = rho[q * g.Vb + t - stride];
    const long long sb = nbr_site<mu, -1>(g, s, x);
    hop<false, mu>(U + (sb * 4 + mu) * 9, p, o);
  }
}

// Coordinates of the k-th block of a colour: rows of Lc[0] / 2 blocks, X of the colour's parity in
// each row
__device__ __forceinline__ void colour_block(const FineGeom& g, int k, int colour, int X[4]) {
  const int half = g.Lc[0] / 2;
  int row = k / half;
  X[1] = row % g.Lc[1];
  row /= g.Lc[1];
  X[2] = row % g.Lc[2];
  X[3] = row / g.Lc[2];
  X[0] = 2 * (k % half) + ((colour + X[1] + X[2] + X[3]) & 1);
}

// Words of the links and the clover of an FP64 handle for the MR steps (fixed.cuh), block by block, word q of the site
// with local index t in block b at (b kFixQ + q) Vb + t: 36 link entries (re, im), then per chirality the diagonal
// of 4 + m0 + C (6 numbers, two per word), C's entries 01, 02, 12 and its upper right 3 x 3 block (see kClovQ).
// All of a block relative to 2^exps[b], a bound of every row's and column's sum of |re| + |im|, in units of 2^-61.
// exps[b] = INT_MAX, and no words: a number that is not finite, or a link more than kFixBits bits below the bound.
constexpr int kFixQ = 66, kFixClov = 36;
constexpr int kFixBits = 8;
__global__ void __launch_bounds__(256) fixed_words_kernel(const double2* __restrict__ U, const double2* __restrict__ clov,
                                                          int4* __restrict__ W, int* __restrict__ exps, FineGeom g,
                                                          double mass) {
  __shared__ unsigned long long top;
  __shared__ int low;  // exponent of the smallest link
  const int b = blockIdx.x;
  int X[4], row = b;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    X[mu] = (row % g.Lc[mu]) * g.B[mu];
    row /= g.Lc[mu];
  }
  auto site = [&](int t) {
    int x[4];
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      x[mu] = X[mu] + t % g.B[mu];
      t /= g.B[mu];
    }
    return site_of(g, x);
  };
  if (threadIdx.x == 0) {
    top = 0;
    low = 0x7FF;
  }
  __syncthreads();
  auto mag = [](double2 z) { return fabs(z.x) + fabs(z.y); };
  for (int i = threadIdx.x; i < g.Vb * 5; i += blockDim.x) {
    const int t = i % g.Vb, mu = i / g.Vb;
    const long long s = site(t);
    unsigned long long m = 0;
    auto bound = [&](double v) { m = max(m, (unsigned long long)__double_as_longlong(v)); };  // a NaN wins
    if (mu < 4) {
      const double2* u = U + (s * 4 + mu) * 9;
      for (int k = 0; k < 3; ++k) {
        bound(mag(u[3 * k]) + mag(u[3 * k + 1]) + mag(u[3 * k + 2]));
        bound(mag(u[k]) + mag(u[3 + k]) + mag(u[6 + k]));
      }
      if (m > 0) atomicMin(&low, (int)(m >> 52));
    } else {
      for (int k = 0; k < 12; ++k) {
        double v = fabs(mass);
        for (int q = 0; q < 6; ++q) v += mag(clov[s * 72 + k * 6 + q]);
        bound(v);
      }
    }
    atomicMax(&top, m);
  }
  __syncthreads();
  const double v = __longlong_as_double((long long)top) * 1.015625;  // |v| < 2^e with room for roundings
  const int f = (__double2hiint(v) >> 20) & 0x7FF, e = max(f - 1022, -900);
  const bool none = f == 0x7FF || f - low > kFixBits;
  if (threadIdx.x == 0) exps[b] = none ? INT_MAX : e;
  if (none) return;
  for (int i = threadIdx.x; i < g.Vb * kFixQ; i += blockDim.x) {
    const int t = i % g.Vb, q = i / g.Vb;
    const long long s = site(t);
    double2 z;
    if (q < kFixClov) {
      z = U[s * 36 + q];
    } else {
      const int h = (q - kFixClov) / 15, k = (q - kFixClov) % 15;
      const double2* c = clov + (s * 2 + h) * 36;
      if (k < 3)
        z = make_double2(mass + c[14 * k].x, mass + c[14 * k + 7].x);
      else
        z = c[k < 5 ? k - 2 : k == 5 ? 8 : (k - 6) / 3 * 6 + 3 + (k - 6) % 3];
    }
    const int2 re = amgfix::words31(amgfix::fixed<61>(z.x, e)), im = amgfix::words31(amgfix::fixed<61>(z.y, e));
    W[(long long)b * kFixQ * g.Vb + i] = make_int4(re.x, re.y, im.x, im.y);
  }
}

struct fx2 {  // complex fixed-point number
  long long x, y;
};
__device__ __forceinline__ fx2 joined(int4 w) {
  return fx2{amgfix::joined(make_int2(w.x, w.y)), amgfix::joined(make_int2(w.z, w.w))};
}
struct FixSum {  // sum of products in units of their high words' products
  long long h = 0, l = 0;
  __device__ __forceinline__ void add(int2 a, int2 b) { amgfix::mac(h, l, a, b); }
  __device__ __forceinline__ long long value() const { return h + ((l + (1 << 30)) >> 31); }
};
// out += -(1 -+ g_mu) U p for the hop of one site in fixed point (hop_u without the factor 1/2).  W: the link's words, Vb
// apart; rho: the neighbour's entries, Vb apart
template <bool FWD, int mu>
__device__ __forceinline__ void hop_fixed(const int4* __restrict__ W, const int4* rho, int Vb, fx2 (&out)[12]) {
  int2 hr[2][3], hi[2][3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    fx2 a0, a1;
    amul(mu, joined(rho[(6 + c) * Vb]), joined(rho[(9 + c) * Vb]), a0, a1);
    const fx2 p0 = joined(rho[c * Vb]), p1 = joined(rho[(3 + c) * Vb]);
    const fx2 h0 = FWD ? zsub(p0, a0) : zadd(p0, a0), h1 = FWD ? zsub(p1, a1) : zadd(p1, a1);
    hr[0][c] = amgfix::words31(h0.x);
    hi[0][c] = amgfix::words31(h0.y);
    hr[1][c] = amgfix::words31(h1.x);
    hi[1][c] = amgfix::words31(h1.y);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    FixSum r0, i0, r1, i1;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int4 u = __ldg(W + (mu * 9 + (FWD ? a * 3 + b : b * 3 + a)) * Vb);
      const int2 ur = make_int2(u.x, u.y), ui = make_int2(u.z, u.w), ni = amgfix::minus(ui);
      const int2 pi = FWD ? ui : ni, mi = FWD ? ni : ui;  // backward: conj(u)
      r0.add(ur, hr[0][b]);
      r0.add(mi, hi[0][b]);
      i0.add(ur, hi[0][b]);
      i0.add(pi, hr[0][b]);
      r1.add(ur, hr[1][b]);
      r1.add(mi, hi[1][b]);
      i1.add(ur, hi[1][b]);
      i1.add(pi, hr[1][b]);
    }
    const fx2 w0{r0.value(), i0.value()}, w1{r1.value(), i1.value()};
    fx2 d0, d1;
    adagmul(mu, w0, w1, d0, d1);
    out[a] = zsub(out[a], w0);
    out[3 + a] = zsub(out[3 + a], w1);
    out[6 + a] = FWD ? zadd(out[6 + a], d0) : zsub(out[6 + a], d0);
    out[9 + a] = FWD ? zadd(out[9 + a], d1) : zsub(out[9 + a], d1);
  }
}
template <int mu>
__device__ __forceinline__ void block_hops_fixed(const FineGeom& g, const int4* __restrict__ W, const int4* rho, int t,
                                                 const int lc[4], int stride, fx2 (&out)[12]) {
  if (lc[mu] + 1 < g.B[mu]) hop_fixed<true, mu>(W + t, rho + t + stride, g.Vb, out);
  if (lc[mu] > 0) hop_fixed<false, mu>(W + t - stride, rho + t - stride, g.Vb, out);
}
// out = 2 (4 + m0 + C) rho at site t
__device__ __forceinline__ void site_fixed(const int4* __restrict__ W, const int4* rho, int Vb, fx2 (&out)[12]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    int2 x[6], y[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int4 p = rho[(6 * h + k) * Vb];
      x[k] = make_int2(p.x, p.y);
      y[k] = make_int2(p.z, p.w);
    }
    FixSum r[6], i[6];
    auto cadd = [&](int a, int2 ur, int2 ui, int b) {
      r[a].add(ur, x[b]);
      r[a].add(amgfix::minus(ui), y[b]);
      i[a].add(ur, y[b]);
      i[a].add(ui, x[b]);
    };
    const int4* c = W + (kFixClov + 15 * h) * Vb;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int4 d = __ldg(c + k * Vb), u = __ldg(c + (3 + k) * Vb);
      r[2 * k].add(make_int2(d.x, d.y), x[2 * k]);
      i[2 * k].add(make_int2(d.x, d.y), y[2 * k]);
      r[2 * k + 1].add(make_int2(d.z, d.w), x[2 * k + 1]);
      i[2 * k + 1].add(make_int2(d.z, d.w), y[2 * k + 1]);
      const int a = k < 2 ? 0 : 1, b = k < 1 ? 1 : 2;  // G_ab and, conjugated, G_ba; -G for the lower rows
      const int2 ur = make_int2(u.x, u.y), ui = make_int2(u.z, u.w), nr = amgfix::minus(ur), ni = amgfix::minus(ui);
      cadd(a, ur, ui, b);
      cadd(b, ur, ni, a);
      cadd(3 + a, nr, ni, 3 + b);
      cadd(3 + b, nr, ui, 3 + a);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const int4 u = __ldg(c + (6 + a * 3 + b) * Vb);
        const int2 ur = make_int2(u.x, u.y), ui = make_int2(u.z, u.w);
        cadd(a, ur, ui, 3 + b);
        cadd(3 + b, ur, amgfix::minus(ui), a);
      }
#pragma unroll
    for (int a = 0; a < 6; ++a) out[6 * h + a] = fx2{r[a].value() << 1, i[a].value() << 1};
  }
}

// One SAP half sweep on the blocks of one colour: x += MR_{n_mr}(B_b, (y - D x)|_b) per block; FP64.
// grid (Vc / 2, nrhs); blockDim >= Vb (threads past Vb only join the sums); dynamic smem: rho
// [12][Vb] + 3 doubles per warp + 3 doubles + 4 ints.
//
// Bound: the FP64 pipes (one warp instruction in 64 cycles per sub-partition).  FIXED: the MR steps apply B in fixed
// point (a multiply-add takes a sixteenth of that): rho as 59-bit integers relative to its largest entry in the block, links and
// clover as words prepared once, sums of 64 bits; the sums over the block and the updates stay in FP64.  An
// application is then good to 2^-57 of the block's largest entry.  A step takes FP64, where every site's sums are good
// relative to its own terms, if an entry is not finite or a site's largest one (unless 0) lies more than kFixBits
// bits below the block's.  12 x 8 x 24 x 16, blocks 3 x 4 x 4 x 2, 3 columns: 451 us a half sweep, in FP64 703 us; 16^4 in
// 2^4 blocks 468 and 944 us.
template <bool FIXED>
__global__ void __launch_bounds__(256) sap_kernel(const double2* __restrict__ U, const double2* __restrict__ Cl,
                                                  const int4* __restrict__ words, const int* __restrict__ exps,
                                                  const double2* __restrict__ y, double2* __restrict__ x, FineGeom g,
                                                  double mass, int nrhs, int colour, int n_mr) {
  using C = double2;
  extern __shared__ __align__(16) unsigned char smem[];
  C* rho = reinterpret_cast<C*>(smem);
  int4* rhow = reinterpret_cast<int4*>(smem);
  double* red = reinterpret_cast<double*>(smem + (size_t)g.Vb * 12 * sizeof(C));
  // largest exponent of rho, and the smallest of the sites', by parity of the step
  int *top = reinterpret_cast<int*>(red + 3 * ((blockDim.x + 31) / 32) + 3), *low = top + 2;
  const int r = blockIdx.y;
  int X[4];
  colour_block(g, blockIdx.x, colour, X);
  const int t = threadIdx.x;
  const bool act = t < g.Vb;
  int lc[4] = {0, 0, 0, 0}, xs[4] = {0, 0, 0, 0};
  long long s = 0;
  if (act) {
    lc[0] = t % g.B[0];
    lc[1] = (t / g.B[0]) % g.B[1];
    lc[2] = (t / (g.B[0] * g.B[1])) % g.B[2];
    lc[3] = t / (g.B[0] * g.B[1] * g.B[2]);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) xs[mu] = X[mu] * g.B[mu] + lc[mu];
    s = site_of(g, xs);
  }
  const int st1 = g.B[0], st2 = g.B[0] * g.B[1], st3 = g.B[0] * g.B[1] * g.B[2];
  const int4* W = nullptr;
  int eb = 0;
  bool words_ok = FIXED;
  if (FIXED) {
    const long long b = ((long long)(X[3] * g.Lc[2] + X[2]) * g.Lc[1] + X[1]) * g.Lc[0] + X[0];
    W = words + b * kFixQ * g.Vb;
    eb = __ldg(exps + b);
    words_ok = eb != INT_MAX;
    if (t < 2) {
      top[t] = 0;
      low[t] = 0x7FF;
    }
    __syncthreads();
  }
  // residual r = y - D x on this site (full D: neighbours outside the block have the other colour)
  C rr[12], e[12];
#pragma unroll
  for (int q = 0; q < 12; ++q) rr[q] = e[q] = zzero<C>();
  if (act) {
    C p[12], o[12];
    load12(x, s, nrhs, r, p);
    site_term(Cl + s * 72, mass, p, o);
    all_hops(g, U, x, s, xs, nrhs, r, o);
    load12(y, s, nrhs, r, p);
#pragma unroll
    for (int q = 0; q < 12; ++q) rr[q] = zsub(p[q], o[q]);
  }
#pragma unroll 1
  for (int it = 0; it < n_mr; ++it) {
    // p = B rho at this site: site term plus the hops that stay inside the block
    double v[3] = {0, 0, 0}, unit = 1;
    C o[12];
    int er = 0;
    bool fixed = words_ok;
    if (FIXED && words_ok) {
      int f = 0;
#pragma unroll
      for (int q = 0; q < 12; ++q)
        f = max(f, max((__double2hiint(rr[q].x) >> 20) & 0x7FF, (__double2hiint(rr[q].y) >> 20) & 0x7FF));
      const int l = __reduce_min_sync(0xffffffffu, f > 0 ? f : 0x7FF);
      f = __reduce_max_sync(0xffffffffu, f);
      if ((t & 31) == 0) {
        atomicMax(&top[it & 1], f);
        atomicMin(&low[it & 1], l);
      }
      __syncthreads();
      f = top[it & 1];
      fixed = f != 0x7FF && f - low[it & 1] <= kFixBits;
      if (t == 0) {  // last read before the previous step's coefficient
        top[(it + 1) & 1] = 0;
        low[(it + 1) & 1] = 0x7FF;
      }
      er = max(f - 1022, -900);
    }
    if (FIXED && fixed) {
      if (act)
#pragma unroll
        for (int q = 0; q < 12; ++q) {
          const int2 a = amgfix::words31(amgfix::fixed<59>(rr[q].x, er)), b = amgfix::words31(amgfix::fixed<59>(rr[q].y, er));
          rhow[q * g.Vb + t] = make_int4(a.x, a.y, b.x, b.y);
        }
      __syncthreads();
      unit = scalbn(1.0, eb + er - 59);
      if (act) {
        fx2 p[12];
        site_fixed(W + t, rhow + t, g.Vb, p);
        block_hops_fixed<0>(g, W, rhow, t, lc, 1, p);
        block_hops_fixed<1>(g, W, rhow, t, lc, st1, p);
        block_hops_fixed<2>(g, W, rhow, t, lc, st2, p);
        block_hops_fixed<3>(g, W, rhow, t, lc, st3, p);
#pragma unroll
        for (int q = 0; q < 12; ++q) o[q] = make_double2((double)p[q].x, (double)p[q].y);
      }
    } else {
      if (act)
#pragma unroll
        for (int q = 0; q < 12; ++q) rho[q * g.Vb + t] = rr[q];
      __syncthreads();
      if (act) {
        site_term(Cl + s * 72, mass, rr, o);
        block_hops_mu<0>(g, U, rho, t, s, xs, lc, 1, o);
        block_hops_mu<1>(g, U, rho, t, s, xs, lc, st1, o);
        block_hops_mu<2>(g, U, rho, t, s, xs, lc, st2, o);
        block_hops_mu<3>(g, U, rho, t, s, xs, lc, st3, o);
      }
    }
    if (act) {
#pragma unroll
      for (int q = 0; q < 12; ++q) {  // in units of p's
        v[0] = fma(o[q].x, o[q].x, fma(o[q].y, o[q].y, v[0]));       // <p, p>
        v[1] = fma(o[q].x, rr[q].x, fma(o[q].y, rr[q].y, v[1]));     // Re <p, rho>
        v[2] = fma(o[q].x, rr[q].y, fma(-o[q].y, rr[q].x, v[2]));    // Im <p, rho>
      }
      v[0] = v[0] * unit * unit;
      v[1] *= unit;
      v[2] *= unit;
    }
    C al;
    bool ok;
    cta_alpha(v, red, al, ok);  // also orders every read of rho before the writes below
    if (act && ok) {
      const C na = make_double2(-al.x * unit, -al.y * unit);
#pragma unroll
      for (int q = 0; q < 12; ++q) {
        zfma(e[q], al, rr[q]);
        zfma(rr[q], na, o[q]);
      }
    }
  }
  if (act) {
#pragma unroll
    for (int q = 0; q < 12; ++q) {
      const long long idx = (s * 12 + q) * nrhs + r;
      x[idx] = zadd(x[idx], e[q]);
    }
  }
}

// The same half sweep in FP32: a CTA takes a block of the colour and a group of nr right-hand sides, one
// thread per site.  The block's links and clover come to shared memory by bulk copy, once for the
// group; residual and MR steps read them, rho and the neighbours' rho from there.  The hops across the
// block face appear in the residual only: a list of face sites, spread over all threads, fetches the
// outside neighbours and leaves half spinors (from above) and finished products (from below) in
// halo, so that no lane of the residual waits for a gather of its own.  x and y are in the block order
// of the links (BLOCKED): one bulk copy, and 16-byte words of consecutive sites for the face
// neighbours; otherwise in the caller's order, entry by entry.  LANES: blocks of up to 16 sites,
// several in a warp (`lanes` lanes and a part of shared memory each), their sums by shuffles.
//
// Bounds: the FP32 pipes (about 1,330 operations per site and application of D or B, five of them: 13 K
// cycles per block of 4^4 and column) and shared memory (1.4 KB read per site and application, 2.9 K
// cycles), of which two warps per sub-partition (the registers, at 4^4 also shared memory) overlap
// little: 5.8 K cycles per MR step.  Half sweep with 4 MR steps: 273 us at 32^4 and one column, 340 us at
// 16^3 x 32 and 12 columns, 37 us at 24^2 8 20 in 2^4 blocks.  Links and clover staged again for every block
// and column from records gathered site by site, the neighbours by each thread: 367, 1,424, 56 us.
// Measured and not kept (32^4 / 12 columns): links in registers, backward hops handed over as half
// spinors, the next block's links fetched ahead 270 / 364 and slower for small blocks; links and
// clover in registers 277 / 379; two threads per site 314 / 397; own links in registers 278 / 344.
//
// Shared memory (float4 words) per block: x, then rho [6][Vb] (12 entries), links [18][Vb], clover
// [14][Vb], and per direction the hops from outside ([3][f] half spinors, [3][f] products, f: its face
// sites).
__host__ __device__ inline int face_sites(const FineGeom& g, int mu) { return g.Vb / g.B[mu]; }
__host__ __device__ inline int sap_words(const FineGeom& g) {
  return (6 + kLinkQ + kClovQ) * g.Vb +
         6 * (face_sites(g, 0) + face_sites(g, 1) + face_sites(g, 2) + face_sites(g, 3));
}
constexpr int kSapRed = 12;  // words of the MR coefficient's warp sums: 2 buffers x 3 sums x 8 warps of floats
inline size_t sap_smem(const FineGeom& g, int subs) {
  return amgpipe::kPipeBytes + (size_t)(kSapRed + subs * sap_words(g)) * sizeof(float4);
}
inline int sap_lanes(const FineGeom& g) {  // lanes per block, a power of two; 0: one block per CTA
  if (g.Vb > 16) return 0;
  int w = 4;
  while (w < g.Vb) w *= 2;
  return w;
}

// Column r of x and y: in block order word q of (block b, site t) at r V 6 + (b 6 + q) Vb + t, else
// entry k of lattice site s at (s 12 + k) nrhs + r
template <bool BLOCKED>
__device__ __forceinline__ void load_site(const FineGeom& g, const float2* __restrict__ v, int b, const int X[4], int t,
                                          int nrhs, int r, float2 p[12]) {
  if (BLOCKED) {
    const float4* q = reinterpret_cast<const float4*>(v) + r * g.V * 6 + (long long)b * 6 * g.Vb + t;
    load_words<6>(q, g.Vb, p);
  } else {
    load12(v, local_site(g, X, t), nrhs, r, p);
  }
}

// The hops of face site f of direction mu to its outside neighbours on both sides (t: its local index
// at lc[mu] = 0; the block's site at lc[mu] = B - 1 is (B - 1) stride further): the half spinor from
// above to halo[f], the product from below to halo[3 nf + f]
template <int mu, bool BLOCKED>
__device__ __forceinline__ void face_hops(const FineGeom& g, const float4* __restrict__ U, const float2* __restrict__ x,
                                          const int X[4], int f, int stride, int nrhs, int r, float4* halo) {
  const int Vb = g.Vb, nf = face_sites(g, mu);
  const int t = f / stride * (stride * g.B[mu]) + f % stride, tt = t + (g.B[mu] - 1) * stride;
  int Xf[4] = {X[0], X[1], X[2], X[3]}, Xb[4] = {X[0], X[1], X[2], X[3]};
  Xf[mu] = X[mu] + 1 < g.Lc[mu] ? X[mu] + 1 : 0;
  Xb[mu] = X[mu] > 0 ? X[mu] - 1 : g.Lc[mu] - 1;
  const int bf = block_of(g, Xf), bb = block_of(g, Xb);
  float2 pf[12], pb[12], h[6], u[9], w[6];
  load_site<BLOCKED>(g, x, bf, Xf, t, nrhs, r, pf);
  load_site<BLOCKED>(g, x, bb, Xb, tt, nrhs, r, pb);
  load_link<mu>(U + (long long)bb * kLinkQ * Vb + tt, Vb, u);
  half_spinor<true, mu>(pf, h);
  put_words<3>(halo + f, nf, h);
  half_spinor<false, mu>(pb, h);
#pragma unroll
  for (int a = 0; a < 3; ++a) colour_row<false>(u, h, a, w[a], w[3 + a]);
  put_words<3>(halo + 3 * nf + f, nf, w);
}
// face_hops of every face site of the block, spread over its threads (t of threads)
template <bool BLOCKED>
__device__ __forceinline__ void all_face_hops(const FineGeom& g, const float4* __restrict__ U, const float2* __restrict__ x,
                                              const int X[4], const int nf[4], const int st[4], int nrhs, int r, int t,
                                              int threads, float4* halo) {
  const int n = nf[0] + nf[1] + nf[2] + nf[3];
  for (int i = t; i < n; i += threads) {
    int f = i;
    if (f < nf[0]) face_hops<0, BLOCKED>(g, U, x, X, f, st[0], nrhs, r, halo);
    else if ((f -= nf[0]) < nf[1]) face_hops<1, BLOCKED>(g, U, x, X, f, st[1], nrhs, r, halo + 6 * nf[0]);
    else if ((f -= nf[1]) < nf[2]) face_hops<2, BLOCKED>(g, U, x, X, f, st[2], nrhs, r, halo + 6 * (nf[0] + nf[1]));
    else face_hops<3, BLOCKED>(g, U, x, X, f - nf[2], st[3], nrhs, r, halo + 6 * (nf[0] + nf[1] + nf[2]));
  }
}
// both hops of direction mu: neighbours in the block from R with the links in us; from outside the
// half spinors and products in halo (FULL), or none
template <int mu, bool FULL>
__device__ __forceinline__ void site_hops(const float4* us, const float4* R, const float4* halo, int nf, int f, bool inside,
                                           bool below, int Vb, int t, int stride, float2 o[12]) {
  float2 p[12], h[6], u[9], w0, w1;
  if (FULL || inside) {
    if (!FULL || inside) {
      get_words<6>(R + t + stride, Vb, p);
      half_spinor<true, mu>(p, h);
    } else {
      get_words<3>(halo + f, nf, h);
    }
    shared_link<mu>(us + t, Vb, u);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      colour_row<true>(u, h, a, w0, w1);
      add_hop<true, mu>(w0, w1, a, o);
    }
  }
  if (below) {
    get_words<6>(R + t - stride, Vb, p);
    shared_link<mu>(us + t - stride, Vb, u);
    hop2<false, mu>(u, p, o);
  } else if (FULL) {
    get_words<3>(halo + 3 * nf + f, nf, h);
#pragma unroll
    for (int a = 0; a < 3; ++a) add_hop<false, mu>(h[a], h[3 + a], a, o);
  }
}

template <bool BLOCKED, bool LANES>
__global__ void __launch_bounds__(256, 1) sap32_kernel(const float4* __restrict__ U, const float4* __restrict__ Cl,
                                                       const float2* __restrict__ y, float2* x, FineGeom g, float mass,
                                                       int nrhs, int nr, int groups, int nblk, int lanes, int colour,
                                                       int n_mr, unsigned* err) {
  using namespace amgpipe;
  extern __shared__ __align__(128) unsigned char sm[];
  Pipe* pp = reinterpret_cast<Pipe*>(sm);  // full[0]: links and clover, full[1]: x
  const int Vb = g.Vb, W = LANES ? lanes : (int)blockDim.x, subs = LANES ? 32 / lanes : 1;
  const int t = LANES ? (int)threadIdx.x & (lanes - 1) : (int)threadIdx.x, sub = LANES ? (int)threadIdx.x / lanes : 0;
  const int ta = t < Vb ? t : 0, item = blockIdx.x;
  float* red = reinterpret_cast<float*>(sm + kPipeBytes);
  float4* xr = reinterpret_cast<float4*>(sm + kPipeBytes) + kSapRed + sub * sap_words(g);
  float4* us = xr + 6 * Vb;
  float4* cs = us + kLinkQ * Vb;
  float4* halo = cs + kClovQ * Vb;
  const int nf[4] = {face_sites(g, 0), face_sites(g, 1), face_sites(g, 2), face_sites(g, 3)};
  const int st[4] = {1, g.B[0], g.B[0] * g.B[1], g.B[0] * g.B[1] * g.B[2]};
  const int k = item / groups * subs + sub;  // block of the colour (past the last: the last, not written)
  int X[4];
  colour_block(g, min(k, nblk - 1), colour, X);
  const int b = block_of(g, X);
  if (threadIdx.x == 0) {
    mbar_init(&pp->full[0], subs);
    mbar_init(&pp->full[1], subs);
    pp->abort = 0;
    fence_mbar_init();
  }
  __syncthreads();
  if (t == 0) {
    mbar_expect_tx(&pp->full[0], (unsigned)((kLinkQ + kClovQ) * Vb * sizeof(float4)));
    bulk_load(us, U + (long long)b * kLinkQ * Vb, (unsigned)(kLinkQ * Vb * sizeof(float4)), &pp->full[0]);
    bulk_load(cs, Cl + (long long)b * kClovQ * Vb, (unsigned)(kClovQ * Vb * sizeof(float4)), &pp->full[0]);
  }
  const bool act = t < Vb && k < nblk;
  bool in[4], below[4];
  int fi[4];
  {
    int lc[4];
    coords_of((unsigned)ta, g.dB, lc);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      in[mu] = lc[mu] + 1 < g.B[mu];
      below[mu] = lc[mu] > 0;
      fi[mu] = ta / (st[mu] * g.B[mu]) * st[mu] + ta % st[mu];
    }
  }
  const int r0 = item % groups * nr, r1 = min(nrhs, r0 + nr);
  unsigned phx = 0;
  for (int r = r0; r < r1; ++r) {
    float2 p[12], o[12], e[12], x0[12];
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // rho before the next copy of x
    __syncthreads();  // the previous column's rho is read
    if (BLOCKED) {
      if (t == 0) {
        const unsigned bytes = (unsigned)(6 * Vb * sizeof(float4));
        mbar_expect_tx(&pp->full[1], bytes);
        bulk_load(xr, reinterpret_cast<const float4*>(x) + r * g.V * 6 + (long long)b * 6 * Vb, bytes, &pp->full[1]);
      }
    } else if (act) {
      const long long s = local_site(g, X, t);
#pragma unroll
      for (int q = 0; q < 12; ++q) reinterpret_cast<float2*>(xr + (q >> 1) * Vb + t)[q & 1] = x[(s * 12 + q) * nrhs + r];
    }
    // the hops across the faces: half spinors from above, products from below
    all_face_hops<BLOCKED>(g, U, x, X, nf, st, nrhs, r, t, W, halo);
    load_site<BLOCKED>(g, y, b, X, ta, nrhs, r, e);
    if (BLOCKED && !wait_phase(&pp->full[1], phx, pp)) abort_cta(pp, err);
    phx ^= 1u;
    if (r == r0 && !wait_phase(&pp->full[0], 0, pp)) abort_cta(pp, err);
    __syncthreads();
    if (pp->abort) return;
    const float4 *h0 = halo, *h1 = h0 + 6 * nf[0], *h2 = h1 + 6 * nf[1], *h3 = h2 + 6 * nf[2];
    {
      float2 cl[2 * kClovQ];
      get_words<kClovQ>(cs + ta, Vb, cl);
      get_words<6>(xr + ta, Vb, x0);
      site_term_words(cl, mass, x0, o);
    }
    site_hops<0, true>(us, xr, h0, nf[0], fi[0], in[0], below[0], Vb, ta, st[0], o);
    site_hops<1, true>(us, xr, h1, nf[1], fi[1], in[1], below[1], Vb, ta, st[1], o);
    site_hops<2, true>(us, xr, h2, nf[2], fi[2], in[2], below[2], Vb, ta, st[2], o);
    site_hops<3, true>(us, xr, h3, nf[3], fi[3], in[3], below[3], Vb, ta, st[3], o);
#pragma unroll
    for (int q = 0; q < 12; ++q) {  // rho = y - D x
      p[q] = zsub(e[q], o[q]);
      e[q] = zzero<float2>();
    }
    __syncthreads();  // x is read
#pragma unroll 1
    for (int it = 0; it < n_mr; ++it) {
      if (act) put_words<6>(xr + t, Vb, p);
      __syncthreads();
      {
        float2 cl[2 * kClovQ];
        get_words<kClovQ>(cs + ta, Vb, cl);
        site_term_words(cl, mass, p, o);  // o = B rho
      }
      site_hops<0, false>(us, xr, h0, 0, 0, in[0], below[0], Vb, ta, st[0], o);
      site_hops<1, false>(us, xr, h1, 0, 0, in[1], below[1], Vb, ta, st[1], o);
      site_hops<2, false>(us, xr, h2, 0, 0, in[2], below[2], Vb, ta, st[2], o);
      site_hops<3, false>(us, xr, h3, 0, 0, in[3], below[3], Vb, ta, st[3], o);
      float v[3] = {0, 0, 0};
      if (t < Vb) {
#pragma unroll
        for (int q = 0; q < 12; ++q) {
          v[0] += o[q].x * o[q].x + o[q].y * o[q].y;  // <o, o>
          v[1] += o[q].x * p[q].x + o[q].y * p[q].y;  // Re <o, rho>
          v[2] += o[q].x * p[q].y - o[q].y * p[q].x;  // Im <o, rho>
        }
      }
      float2 al;
      bool ok;
      // the barrier (inside) also orders every read of rho before the next step's writes
      if (LANES) {
        lanes_alpha(v, lanes, al, ok);
        __syncwarp();
      } else {
        cta_alpha_all(v, red + (it & 1) * 24, al, ok);
      }
      if (ok) {  // e += alpha rho, rho -= alpha B rho
#pragma unroll
        for (int q = 0; q < 12; ++q) {
          zfma(e[q], al, p[q]);
          float2 ap = zzero<float2>();
          zfma(ap, al, o[q]);
          p[q] = zsub(p[q], ap);
        }
      }
    }
    if (act) {
#pragma unroll
      for (int q = 0; q < 12; ++q) p[q] = zadd(x0[q], e[q]);
      if (BLOCKED) {
        put_words<6>(reinterpret_cast<float4*>(x) + r * g.V * 6 + (long long)b * 6 * Vb + t, Vb, p);
      } else {
        const long long s = local_site(g, X, t);
#pragma unroll
        for (int q = 0; q < 12; ++q) x[(s * 12 + q) * nrhs + r] = p[q];
      }
    }
  }
}

// Columns j0 .. j0 + N groups - 1 of v ([V][12][nrhs]) <-> w ([column][block][6 words][Vb], block order).
// One CTA per kTileSites sites (in block order) and N columns, through shared memory: v is read and written
// in runs (the B[0] sites of a row; N neighbouring columns), w in runs of consecutive sites.  Bound:
// HBM; many small CTAs keep it busy (32^4, one column: 36 us a copy, 5.6 TB/s; a CTA per block with the
// site index computed by divisions took 86 us).
constexpr int kTileSites = 64;
template <bool TO, int N>
__global__ void __launch_bounds__(256) blocked_kernel(float2* __restrict__ v, float2* __restrict__ w, FineGeom g,
                                                      const int* __restrict__ soff, int nrhs, int j0, int groups) {
  constexpr int P = kTileSites + 1;
  __shared__ float2 sc[N * 12 * P];           // [column][entry][site]
  __shared__ unsigned lex[kTileSites];        // the sites' places in the lattice
  __shared__ long long wof[kTileSites];       // and of their first words in w
  const int Vb = g.Vb, grp = (int)(blockIdx.x % groups);
  const long long i0 = (long long)(blockIdx.x / groups) * kTileSites;
  const int ts = (int)min((long long)kTileSites, g.V - i0);
  if (threadIdx.x < ts) {
    int t, X[4];
    const unsigned b = divide((unsigned)(i0 + threadIdx.x), g.dVb, t);
    coords_of(b, g.dLc, X);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) X[mu] *= g.B[mu];
    lex[threadIdx.x] = (unsigned)(site_of(g, X) + __ldg(soff + t));
    wof[threadIdx.x] = (long long)b * 6 * Vb + t;
  }
  __syncthreads();
  float4* wg = reinterpret_cast<float4*>(w) + (long long)grp * N * g.V * 6;
  auto caller = [&](auto&& body) {  // e = (site, entry, column), the column fastest
#pragma unroll 6
    for (int e = threadIdx.x; e < ts * 12 * N; e += 256) {
      const int c = e % N, k = e / N % 12, t = e / (12 * N);
      body(v + ((long long)lex[t] * 12 + k) * nrhs + j0 + grp * N + c, sc + (c * 12 + k) * P + t);
    }
  };
  auto caller_words = [&](auto&& body) {  // one column: e = (site, word)
#pragma unroll 2
    for (int e = threadIdx.x; e < ts * 6; e += 256)
      body(reinterpret_cast<float4*>(v) + (long long)lex[e / 6] * 6 + e % 6, sc + e % 6 * 2 * P + e / 6);
  };
  auto blocked = [&](auto&& body) {  // e = (column, word, site)
#pragma unroll 2
    for (int e = threadIdx.x; e < N * 6 * kTileSites; e += 256) {
      const int t = e % kTileSites, q = e / kTileSites % 6, c = e / (6 * kTileSites);
      if (t < ts) body(wg + (long long)c * g.V * 6 + wof[t] + q * Vb, sc + (c * 12 + 2 * q) * P + t);
    }
  };
  auto word_in = [](const float4* a, float2* s) {
    const float4 f = *a;
    s[0] = lo2(f);
    s[P] = hi2(f);
  };
  auto word_out = [](float4* a, const float2* s) { *a = make_float4(s[0].x, s[0].y, s[P].x, s[P].y); };
  if (!TO) blocked(word_in);
  else if (N == 1 && nrhs == 1) caller_words(word_in);
  else caller([](const float2* a, float2* s) { *s = *a; });
  __syncthreads();
  if (TO) blocked(word_out);
  else if (N == 1 && nrhs == 1) caller_words(word_out);
  else caller([](float2* a, const float2* s) { *a = *s; });
}

// ------------------------------------------------------------------ outer FGMRES vector kernels
constexpr int FT = 256;

// Arithmetic of the outer FGMRES vector kernels: per element in the vectors' precision (FP64 is
// slow on this GPU; an FP32 vector gains nothing from FP64 products), per-thread partial sums in
// that precision (a few dozen elements each), sums across threads and CTAs in FP64.  The per-column
// coefficients are converted to the vectors' precision once per CTA, in shared memory.
template <typename C> struct Real;
template <> struct Real<float2> { using type = float; };
template <> struct Real<double2> { using type = double; };

template <typename C>
__device__ __forceinline__ C to_c(double2 v) {
  C o;
  o.x = (typename Real<C>::type)v.x;
  o.y = (typename Real<C>::type)v.y;
  return o;
}

// part[i][r] += sum_n conj(V_i[n, r]) w[n, r] for i < nv (one FP64 atomic per CTA and pair)
template <typename C>
__global__ void __launch_bounds__(FT) fdots_kernel(const C* __restrict__ Vb, long long vstride, int nv,
                                                   const C* __restrict__ w, long long n, int nrhs, double2* out) {
  using R = typename Real<C>::type;
  __shared__ double2 red[FT];
  const int i = blockIdx.y;
  const C* v = Vb + vstride * i;
  const int per = FT / nrhs * nrhs;  // threads per CTA that take part (a multiple of nrhs)
  R ax = 0, ay = 0;
  if (threadIdx.x < per) {
    for (long long e = blockIdx.x * (long long)per + threadIdx.x; e < n * nrhs; e += (long long)gridDim.x * per) {
      const C a = v[e], b = w[e];
      ax = fma(a.x, b.x, fma(a.y, b.y, ax));
      ay = fma(a.x, b.y, fma(-a.y, b.x, ay));
    }
  }
  red[threadIdx.x] = make_double2((double)ax, (double)ay);
  __syncthreads();
  if (threadIdx.x < nrhs) {
    double2 s = make_double2(0, 0);
    for (int q = threadIdx.x; q < per; q += nrhs) {
      s.x += red[q].x;
      s.y += red[q].y;
    }
    atomicAdd(&out[i * nrhs + threadIdx.x].x, s.x);
    atomicAdd(&out[i * nrhs + threadIdx.x].y, s.y);
  }
}

constexpr int kFMaxCoef = 1024;  // coefficients cached per CTA (nv x nrhs); more are read from global memory

template <typename C>
__device__ __forceinline__ C coef_at(const C* cached, const double2* __restrict__ g, bool use_cache, int k) {
  return use_cache ? cached[k] : to_c<C>(g[k]);
}

// w -= sum_{i < nv} h[i][r] V_i ; nrm2[r] += |w|^2 (after the update)
template <typename C>
__global__ void __launch_bounds__(FT) fupdate_kernel(const C* __restrict__ Vb, long long vstride, int nv,
                                                     const double2* __restrict__ h, C* __restrict__ w, long long n,
                                                     int nrhs, double* nrm2) {
  using R = typename Real<C>::type;
  __shared__ double red[FT];
  __shared__ C hc[kFMaxCoef];
  const bool cached = nv * nrhs <= kFMaxCoef;
  if (cached)
    for (int k = threadIdx.x; k < nv * nrhs; k += blockDim.x) hc[k] = to_c<C>(h[k]);
  __syncthreads();
  const int per = FT / nrhs * nrhs;
  R acc = 0;
  if (threadIdx.x < per) {
    for (long long e = blockIdx.x * (long long)per + threadIdx.x; e < n * nrhs; e += (long long)gridDim.x * per) {
      const int r = (int)(e % nrhs);
      C a = w[e];
      for (int i = 0; i < nv; ++i) {
        const C v = Vb[vstride * i + e];
        const C c = coef_at(hc, h, cached, i * nrhs + r);
        a.x -= c.x * v.x - c.y * v.y;
        a.y -= c.x * v.y + c.y * v.x;
      }
      w[e] = a;
      acc = fma(a.x, a.x, fma(a.y, a.y, acc));
    }
  }
  red[threadIdx.x] = (double)acc;
  __syncthreads();
  if (threadIdx.x < nrhs) {
    double s = 0;
    for (int q = threadIdx.x; q < per; q += nrhs) s += red[q];
    atomicAdd(&nrm2[threadIdx.x], s);
  }
}

// y = a[r] * x (a per column, complex); y may be x
template <typename C>
__global__ void fscale_kernel(const C* x, C* y, const double2* __restrict__ a, long long n, int nrhs) {
  __shared__ C ac[64];  // nrhs <= 64
  if (threadIdx.x < nrhs) ac[threadIdx.x] = to_c<C>(a[threadIdx.x]);
  __syncthreads();
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * nrhs;
       e += (long long)gridDim.x * blockDim.x) {
    const C c = ac[e % nrhs];
    const C v = x[e];
    C o;
    o.x = c.x * v.x - c.y * v.y;
    o.y = c.x * v.y + c.y * v.x;
    y[e] = o;
  }
}

// y += sum_{i < nv} c[i][r] X_i
template <typename C>
__global__ void fcombine_kernel(const C* __restrict__ Xb, long long vstride, int nv, const double2* __restrict__ c,
                                C* __restrict__ y, long long n, int nrhs) {
  __shared__ C cc[kFMaxCoef];
  const bool cached = nv * nrhs <= kFMaxCoef;
  if (cached)
    for (int k = threadIdx.x; k < nv * nrhs; k += blockDim.x) cc[k] = to_c<C>(c[k]);
  __syncthreads();
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * nrhs;
       e += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(e % nrhs);
    C a = y[e];
    for (int i = 0; i < nv; ++i) {
      const C v = Xb[vstride * i + e];
      const C k = coef_at(cc, c, cached, i * nrhs + r);
      a.x += k.x * v.x - k.y * v.y;
      a.y += k.x * v.y + k.y * v.x;
    }
    y[e] = a;
  }
}

// nrm2[r] += |v|^2
template <typename C>
__global__ void __launch_bounds__(FT) fnorm_kernel(const C* __restrict__ v, long long n, int nrhs, double* nrm2) {
  using R = typename Real<C>::type;
  __shared__ double red[FT];
  const int per = FT / nrhs * nrhs;
  R acc = 0;
  if (threadIdx.x < per)
    for (long long e = blockIdx.x * (long long)per + threadIdx.x; e < n * nrhs; e += (long long)gridDim.x * per)
      acc = fma(v[e].x, v[e].x, fma(v[e].y, v[e].y, acc));
  red[threadIdx.x] = (double)acc;
  __syncthreads();
  if (threadIdx.x < nrhs) {
    double s = 0;
    for (int q = threadIdx.x; q < per; q += nrhs) s += red[q];
    atomicAdd(&nrm2[threadIdx.x], s);
  }
}

FineGeom fine_geom(const amg_coarse* h) {
  FineGeom g;
  for (int mu = 0; mu < 4; ++mu) {
    g.L[mu] = h->g.L[mu];
    g.B[mu] = h->g.B[mu];
    g.Lc[mu] = h->g.Lc[mu];
  }
  g.V = h->g.V;
  g.Vb = (int)h->g.Vb;
  for (int mu = 0; mu < 3; ++mu) {
    g.dL[mu] = fast_div(g.L[mu]);
    g.dB[mu] = fast_div(g.B[mu]);
    g.dLc[mu] = fast_div(g.Lc[mu]);
  }
  g.dVb = fast_div(g.Vb);
  return g;
}

// Links [V][36] and clover blocks [V][2][6][6] in FP64 -> the FP32 words in block order (see kLinkQ)
__global__ void links_words_kernel(const double2* __restrict__ in, float4* __restrict__ out, Geom g) {
  const long long n = g.V * kLinkQ;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const long long b = e / (kLinkQ * g.Vb);
    const int q = (int)(e / g.Vb % kLinkQ);
    const double2* U = in + block_site_fast(g, block_origin(g, b), (int)(e % g.Vb)) * 36 + 2 * q;
    out[e] = make_float4(0.5f * (float)U[0].x, 0.5f * (float)U[0].y, 0.5f * (float)U[1].x, 0.5f * (float)U[1].y);
  }
}
__global__ void clover_words_kernel(const double2* __restrict__ in, float4* __restrict__ out, Geom g) {
  const long long n = g.V * kClovQ;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const long long b = e / (kClovQ * g.Vb);
    const int q = (int)(e / g.Vb % kClovQ), hh = q / 7;
    const double2* C = in + (block_site_fast(g, block_origin(g, b), (int)(e % g.Vb)) * 2 + hh) * 36;
    float2 v[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int w = 2 * (q % 7) + k;  // complex word of the chirality
      if (w < 2) {
        v[k].x = (float)C[w * 2 * 7].x;                      // H00, H22
        v[k].y = w == 0 ? (float)C[7].x : 0.f;               // H11
      } else {
        const int a = w < 5 ? (w == 4 ? 1 : 0) : (w - 5) / 3;
        const int c = w < 5 ? (w == 2 ? 1 : 2) : 3 + (w - 5) % 3;
        v[k] = make_float2((float)C[a * 6 + c].x, (float)C[a * 6 + c].y);
      }
    }
    out[e] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  }
}

bool fine_fp64(const amg_coarse* h) { return h->p.vec_prec == AMG_FP64; }

// Columns per thread: two if their waves, 1.35 times as long (a thread's loads and sums in series), take less time than
// those of one.  us with one and two: 8^4 and 2 columns 8.6 and 10.8 (one wave each), 12^4 and 6 18.8 and 21.5 (two
// each), 8^3 x 16 and 12 15.1 and 12.9 (two and one), 16^3 x 32 and 2 55.6 and 58.4 (four and three), 12 columns 174
// and 160.
int dirac32_columns(long long V, int nrhs) {
  if (nrhs % 2) return 1;
  auto waves = [&](int nc) {
    const long long per = 128LL * dirac32_ctas(nc) * amg_sm_count();
    return (V * (nrhs / nc) + per - 1) / per;
  };
  return 1.35 * waves(2) < waves(1) ? 2 : 1;
}

template <int NC>
auto* pick_dirac32(bool sub, bool fast) {
  return sub ? (fast ? dirac32_kernel<true, true, NC> : dirac32_kernel<true, false, NC>)
             : (fast ? dirac32_kernel<false, true, NC> : dirac32_kernel<false, false, NC>);
}

amg_status dirac_any(amg_coarse* h, const void* psi, const void* y, void* out, int nrhs, cudaStream_t st) {
  const long long total = h->g.V * nrhs;
  const long long want = (total + 127) / 128;
  const int grid = (int)(want < 16LL * amg_sm_count() ? want : 16LL * amg_sm_count());
  const FineGeom g = fine_geom(h);
  if (fine_fp64(h)) {
    const double mass = 4.0 + h->p.m0;
    auto* U = (const double2*)h->fU;
    auto* C = (const double2*)h->fC;
    if (y)
      dirac_kernel<true><<<grid, 128, 0, st>>>(U, C, (const double2*)psi, (const double2*)y, (double2*)out, g, mass, nrhs);
    else
      dirac_kernel<false><<<grid, 128, 0, st>>>(U, C, (const double2*)psi, nullptr, (double2*)out, g, mass, nrhs);
  } else {
    const float mass = (float)(4.0 + h->p.m0);
    auto* U = (const float4*)h->fU;
    auto* C = (const float4*)h->fC;
    const float2 *p = (const float2*)psi, *yy = (const float2*)y;
    const int nb = g.Vb <= kDiracSites ? kDiracSites / g.Vb : 0, nblocks = (int)h->g.Vc;
    const int ctas = nb ? (nblocks + nb - 1) / nb : 0;
    // fewer tiles than SMs: one thread per site in lattice order spreads over more of them
    if (nrhs == 1 && ctas >= amg_sm_count()) {
      const int threads = (nb * g.Vb + 31) / 32 * 32;
      auto* k = y ? dirac32_block_kernel<true> : dirac32_block_kernel<false>;
      k<<<ctas, threads, 0, st>>>(U, C, p, yy, (float2*)out, g, mass, nb, nblocks);
    } else {
      const int nc = dirac32_columns(g.V, nrhs), groups = nrhs / nc;
      const FastDiv dn = fast_div(groups);
      const long long threads = h->g.V * groups;
      auto* k = nc == 1 ? pick_dirac32<1>(y != nullptr, threads < (1LL << 31)) : pick_dirac32<2>(y != nullptr, threads < (1LL << 31));
      k<<<(unsigned)std::min((threads + 127) / 128, 16LL * amg_sm_count()), 128, 0, st>>>(U, C, p, yy, (float2*)out, g, mass, dn);
    }
  }
  AMG_LAUNCH_CHECK();
  h->launches++;
  return AMG_OK;
}

// CTAs of the FP32 half sweep resident at once: the register file holds 256 of its threads
int sap_slots(int threads, size_t smem) {
  return amg_sm_count() * std::max(1, std::min(256 / threads, (int)(227 * 1024 / smem)));
}

// Columns per item of the FP32 half sweep: an item loads its block's links and clover once and sweeps a
// group of columns with them (about a quarter of a column's time), so larger groups repeat fewer
// loads and smaller ones fill the last wave; the group with the least waves x (load + columns).
int sap_columns(long long nblk, int nrhs, int slots) {
  int best = 1;
  double best_cost = 0;
  for (int c = 1; c <= nrhs; ++c) {
    const long long ctas = nblk * ((nrhs + c - 1) / c);
    const double cost = (double)((ctas + slots - 1) / slots) * (0.25 + c);
    if (c == 1 || cost < best_cost) {
      best = c;
      best_cost = cost;
    }
  }
  return best;
}

template <bool BLOCKED>
amg_status sweep32(amg_coarse* h, const float2* y, float2* x, int nrhs, int n_cycles, int n_mr, cudaStream_t st) {
  const FineGeom g = fine_geom(h);
  const int nblk = (int)(h->g.Vc / 2);
  // Small blocks share a warp unless the launch's warps find an SM sub-partition each anyway: then a block's
  // faces are spread over more lanes (8^4 in 2^4 blocks, one column, 4 cycles: 141 us, 150 with two blocks to a warp).
  int lanes = sap_lanes(g);
  while (lanes && lanes < 32 && (long long)nblk * (2 * lanes) / 32 * nrhs <= 4LL * amg_sm_count()) lanes *= 2;
  const int subs = lanes ? 32 / lanes : 1, threads = lanes ? 32 : (g.Vb + 31) / 32 * 32;
  const size_t smem = sap_smem(g, subs);
  if (threads > 256 || smem > 227 * 1024) return AMG_ERR_UNSUPPORTED;
  auto* k = lanes ? sap32_kernel<BLOCKED, true> : sap32_kernel<BLOCKED, false>;
  AMG_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int units = (nblk + subs - 1) / subs;
  const int nr = sap_columns(units, nrhs, sap_slots(threads, smem)), groups = (nrhs + nr - 1) / nr;
  const float mass = (float)(4.0 + h->p.m0);
  for (int c = 0; c < n_cycles; ++c)
    for (int colour = 0; colour < 2; ++colour) {
      k<<<units * groups, threads, smem, st>>>((const float4*)h->fU, (const float4*)h->fC, y, x, g, mass, nrhs, nr, groups,
                                              nblk, lanes, colour, n_mr, h->err);
      AMG_LAUNCH_CHECK();
      h->launches++;
    }
  return AMG_OK;
}

// The sweeps run on copies of x and y in block order, one vector per column; x is copied back.  The
// copies come from the handle's pool, at most kColBytes at a time but one column at least (columns are
// independent).  While the stream is captured, or without memory for them, the sweeps work on the
// caller's vectors; so they do where the copies cost more than they save (sap_copies).
constexpr size_t kColBytes = (size_t)2 << 30;
constexpr size_t kPoolStep = (size_t)64 << 20;  // more than what a pool adds to an allocation (32 MB pieces)
// us with and without copies (4 MR steps).  One column gains little from the block order: 32^4 1220 and 1202 for two
// cycles, 2297 and 2382 for four; in blocks of up to 16 sites 8^4 151 and 145, 16^4 191 and 188, 24^4 893 and 972 for four.
// One cycle of two columns: 16^4 102 and 98, 32^4 1239 and 1271; of more: 12^4 and three 94 and 90, 8^3 x 16 and eight
// 65 and 61, but 12^4 and eight 160 and 176, 16^4 and four 177 and 198.  Two cycles of two columns 16^4 171 and 189.
bool sap_copies(const FineGeom& g, int nrhs, int n_cycles) {
  constexpr long long kSmall = 1 << 16;  // elements (sites times columns) that one cycle does not copy
  if (nrhs == 1) return n_cycles > 2 && (sap_lanes(g) == 0 || g.V > kSmall);
  return n_cycles > 1 || (nrhs > 2 && g.V * nrhs > kSmall);
}
int sap_copy_columns(const amg_coarse* h, int nrhs) {
  return (int)std::max<size_t>(1, std::min<size_t>(nrhs, kColBytes / (2 * h->g.V * 12 * sizeof(float2))));
}
size_t sap_copy_bytes(const amg_coarse* h, int nrhs) {
  return 2 * (size_t)h->g.V * 12 * sizeof(float2) * sap_copy_columns(h, nrhs);
}

// Columns j0 .. j0 + nc - 1 of v to (TO) or from w; four columns per CTA (a 32-byte sector), the rest
// in a launch of their own
template <bool TO>
amg_status blocked_copy(amg_coarse* h, const float2* v, const float2* w, int nrhs, int j0, int nc, cudaStream_t st) {
  float2 *vv = const_cast<float2*>(v), *ww = const_cast<float2*>(w);
  const unsigned tiles = (unsigned)((h->g.V + kTileSites - 1) / kTileSites);
  const int groups = nc / 4, rest = nc % 4;
  const FineGeom g = fine_geom(h);
  const int* so = h->soff;
  if (groups) blocked_kernel<TO, 4><<<tiles * groups, 256, 0, st>>>(vv, ww, g, so, nrhs, j0, groups);
  j0 += 4 * groups;
  ww += (size_t)4 * groups * h->g.V * 12;
  if (rest == 1) blocked_kernel<TO, 1><<<tiles, 256, 0, st>>>(vv, ww, g, so, nrhs, j0, 1);
  else if (rest == 2) blocked_kernel<TO, 2><<<tiles, 256, 0, st>>>(vv, ww, g, so, nrhs, j0, 1);
  else if (rest == 3) blocked_kernel<TO, 3><<<tiles, 256, 0, st>>>(vv, ww, g, so, nrhs, j0, 1);
  h->launches += (groups > 0) + (rest > 0);
  AMG_LAUNCH_CHECK();
  return AMG_OK;
}

// The pool, with the copies of max_nrhs columns allocated once here rather than in the first sweep; the pool
// keeps them until the handle goes.  Without it (a device without pools) the sweeps do without copies.
void sap_pool(amg_coarse* h, cudaStream_t st) {
  if (h->fpool) return;  // links set again: the lattice, and so the copies' size, are the same
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  uint64_t keep = std::max(kColBytes, sap_copy_bytes(h, h->p.max_nrhs) + kPoolStep);
  void* w = nullptr;
  if (cudaGetDevice(&props.location.id) != cudaSuccess || cudaMemPoolCreate(&h->fpool, &props) != cudaSuccess) {
    h->fpool = nullptr;
  } else if (cudaMemPoolSetAttribute(h->fpool, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess &&
             cudaMallocFromPoolAsync(&w, sap_copy_bytes(h, h->p.max_nrhs), h->fpool, st) == cudaSuccess) {
    cudaFreeAsync(w, st);
  }
  cudaGetLastError();
}

amg_status launch_sap32(amg_coarse* h, const void* yv, void* xv, int nrhs, int n_cycles, int n_mr, cudaStream_t st) {
  const float2* y = (const float2*)yv;
  float2* x = (float2*)xv;
  const size_t n = (size_t)h->g.V * 12;
  if (n_cycles < 1) return AMG_OK;
  if (!sap_copies(fine_geom(h), nrhs, n_cycles)) return sweep32<false>(h, y, x, nrhs, n_cycles, n_mr, st);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  AMG_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
  const int chunk = sap_copy_columns(h, nrhs);
  float2* w = nullptr;
  if (h->fpool && cap == cudaStreamCaptureStatusNone &&
      cudaMallocFromPoolAsync((void**)&w, sap_copy_bytes(h, nrhs), h->fpool, st) != cudaSuccess) {
    cudaGetLastError();
    w = nullptr;
  }
  if (!w) return sweep32<false>(h, y, x, nrhs, n_cycles, n_mr, st);
  float2* wx = w + n * chunk;
  amg_status s = AMG_OK;
  for (int j0 = 0; j0 < nrhs && s == AMG_OK; j0 += chunk) {
    const int nc = std::min(chunk, nrhs - j0);
    s = blocked_copy<true>(h, y, w, nrhs, j0, nc, st);
    if (s == AMG_OK) s = blocked_copy<true>(h, x, wx, nrhs, j0, nc, st);
    if (s == AMG_OK) s = sweep32<true>(h, w, wx, nc, n_cycles, n_mr, st);
    if (s == AMG_OK) s = blocked_copy<false>(h, x, wx, nrhs, j0, nc, st);
  }
  cudaFreeAsync(w, st);
  return s;
}

amg_status launch_sap64(amg_coarse* h, const void* y, void* x, int nrhs, int n_cycles, int n_mr, cudaStream_t st) {
  const int threads = (h->g.Vb + 31) / 32 * 32;
  const size_t smem = (size_t)h->g.Vb * 12 * sizeof(double2) + (size_t)(threads / 32 + 1) * 3 * sizeof(double) + 16;
  if (threads > 256 || smem > 227 * 1024) return AMG_ERR_UNSUPPORTED;
  auto* kernel = h->fW ? sap_kernel<true> : sap_kernel<false>;
  AMG_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const dim3 grid((unsigned)(h->g.Vc / 2), (unsigned)nrhs);
  for (int c = 0; c < n_cycles; ++c)
    for (int colour = 0; colour < 2; ++colour) {
      kernel<<<grid, threads, smem, st>>>((const double2*)h->fU, (const double2*)h->fC, (const int4*)h->fW, h->fE,
                                          (const double2*)y, (double2*)x, fine_geom(h), 4.0 + h->p.m0, nrhs, colour,
                                          n_mr);
      AMG_LAUNCH_CHECK();
      h->launches++;
    }
  return AMG_OK;
}

amg_status sap_any(amg_coarse* h, const void* y, void* x, int nrhs, int n_cycles, int n_mr, cudaStream_t st) {
  return fine_fp64(h) ? launch_sap64(h, y, x, nrhs, n_cycles, n_mr, st) : launch_sap32(h, y, x, nrhs, n_cycles, n_mr, st);
}

amg_status check_fine(amg_coarse* h, const void* a, const void* b, int nrhs) {
  if (!h || !a || !b || !aligned16(a) || !aligned16(b)) return AMG_ERR_INVALID_ARG;
  if (nrhs < 1 || nrhs > h->p.max_nrhs) return AMG_ERR_INVALID_ARG;
  if (!h->fU) return AMG_ERR_UNSUPPORTED;  // amg_setup_fine not called
  return AMG_OK;
}

// Allocates by alloc(), which returns a cudaError_t; where memory runs out once more after giving back what the smoother
// holds for its speed: the fixed-point words (its steps then take FP64) and the pool's idle copies (the sweeps then
// allocate them again or do without).
template <typename F>
cudaError_t alloc_or_give_back(amg_coarse* h, F&& alloc) {
  cudaError_t e = alloc();
  if (e != cudaErrorMemoryAllocation) return e;
  cudaGetLastError();
  cudaFree(h->fW);
  cudaFree(h->fE);
  h->fW = nullptr;
  h->fE = nullptr;
  if (h->fpool) cudaMemPoolTrimTo(h->fpool, 0);
  e = alloc();
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

bool sap_supported(const amg_coarse* h) {
  for (int mu = 0; mu < 4; ++mu)
    if (h->g.Lc[mu] % 2) return false;
  return h->g.Vb <= 256;
}

amg_status check_vp(const amg_vcycle_params* vp) {
  if (!vp || !(vp->coarse_tol >= 0) || vp->coarse_restart < 1 || vp->coarse_max_applies < 1 || vp->n_smoother < 0 ||
      vp->n_mr < 1)
    return AMG_ERR_INVALID_ARG;
  return AMG_OK;
}

amg_status vcycle_impl(amg_coarse* h, const amg_vcycle_params* vp, const void* y, void* x, int nrhs,
                       cudaStream_t st) {
  if (h->next)  // three levels: one two-grid cycle on level 1 in place of the coarse solve
    AMG_TRY_INTERNAL(amg_internal_cgc3(h, y, x, nrhs, st));
  else
    AMG_TRY_INTERNAL(amg_cgc(h, y, x, nrhs, vp->coarse_tol, vp->coarse_restart, vp->coarse_max_applies, st, nullptr));
  if (vp->n_smoother > 0) AMG_TRY_INTERNAL(sap_any(h, y, x, nrhs, vp->n_smoother, vp->n_mr, st));
  return AMG_OK;
}

// ------------------------------------------------------------------ outer FGMRES (host-driven)
// Right-preconditioned flexible GMRES(m) of Saad Alg. 9.6 from u = 0, every right-hand side
// independently: classical Gram-Schmidt Arnoldi, Givens rotations, convergence on the implicit
// residual |g_{j+1}| <= tol ||f||; every restart after the first recomputes the true residual
// (one more application of D), as the coarse solve counts them.  Scalars live on the host: each
// Arnoldi step synchronises once, which is small against the V-cycle it waits for.
template <typename T>
amg_status solve_impl(amg_coarse* h, const amg_vcycle_params* vp, const void* f, void* u, int nrhs, double tol,
                      int m, int max_applies, cudaStream_t st, double* info) {
  using C = typename Cx<T>::type;
  const long long n = h->g.V * 12;
  const long long vs = n * nrhs;  // elements of one multi-column vector
  const size_t vbytes = (size_t)vs * sizeof(C);
  // workspace: V_0..V_m, Z_0..Z_{m-1}, r, and (m + 1) x nrhs double2 + nrhs doubles of sums
  const size_t need = (size_t)(2 * m + 2) * vbytes + ((size_t)(m + 1) * nrhs * 2 + nrhs) * sizeof(double) + 256;
  if (need > h->fwork_bytes) {
    AMG_CUDA_TRY(cudaStreamSynchronize(st));
    cudaFree(h->fwork);
    h->fwork = nullptr;
    h->fwork_bytes = 0;
    AMG_CUDA_TRY(alloc_or_give_back(h, [&] { return cudaMalloc(&h->fwork, need); }));
    h->fwork_bytes = need;
  }
  C* Vb = (C*)h->fwork;
  C* Zb = Vb + (size_t)(m + 1) * vs;
  C* R = Zb + (size_t)m * vs;
  double2* dh = (double2*)(R + vs);
  double* dn = (double*)(dh + (size_t)(m + 1) * nrhs);
  C* U = (C*)u;
  const int vgrid = 4 * amg_sm_count();
  const dim3 fblk(FT);

  auto colnorm = [&](const C* v, std::vector<double>& out) -> amg_status {
    AMG_CUDA_TRY(cudaMemsetAsync(dn, 0, nrhs * sizeof(double), st));
    fnorm_kernel<C><<<vgrid, fblk, 0, st>>>(v, n, nrhs, dn);
    AMG_LAUNCH_CHECK();
    h->launches++;
    AMG_CUDA_TRY(cudaMemcpyAsync(out.data(), dn, nrhs * sizeof(double), cudaMemcpyDeviceToHost, st));
    AMG_CUDA_TRY(cudaStreamSynchronize(st));
    for (auto& x : out) x = sqrt(x);
    return AMG_OK;
  };

  std::vector<double> fnorm(nrhs), beta(nrhs), tmp(nrhs);
  std::vector<int> applies(nrhs, 0), done(nrhs, 0);
  std::vector<double> relres(nrhs, 1.0);
  AMG_CUDA_TRY(cudaMemsetAsync(U, 0, vbytes, st));
  AMG_CUDA_TRY(cudaMemcpyAsync(R, f, vbytes, cudaMemcpyDeviceToDevice, st));
  AMG_TRY_INTERNAL(colnorm((const C*)f, fnorm));
  for (int r = 0; r < nrhs; ++r)
    if (fnorm[r] == 0) {
      done[r] = 1;
      relres[r] = 0;
    }
  int total_applies = 0;
  const size_t hs = (size_t)(m + 1) * m;
  std::vector<std::complex<double>> H(hs * nrhs), cs(m * nrhs), sn(m * nrhs), g((m + 1) * nrhs);
  std::vector<double2> coef((m + 1) * nrhs);
  while (true) {
    AMG_TRY_INTERNAL(colnorm(R, beta));
    bool any = false;
    for (int r = 0; r < nrhs; ++r) {
      if (!done[r] && beta[r] <= tol * fnorm[r]) done[r] = 1;
      any = any || !done[r];
    }
    const int mm = std::min(m, max_applies - total_applies);
    if (!any || mm <= 0) break;
    // V_0 = r / beta (columns already converged get 0 and stay 0)
    for (int r = 0; r < nrhs; ++r) coef[r] = make_double2(done[r] ? 0.0 : 1.0 / beta[r], 0.0);
    AMG_CUDA_TRY(cudaMemcpyAsync(dh, coef.data(), nrhs * sizeof(double2), cudaMemcpyHostToDevice, st));
    fscale_kernel<C><<<vgrid, fblk, 0, st>>>(R, Vb, dh, n, nrhs);
    AMG_LAUNCH_CHECK();
    h->launches++;
    std::fill(H.begin(), H.end(), 0.0);
    std::fill(g.begin(), g.end(), 0.0);
    for (int r = 0; r < nrhs; ++r) g[r * (m + 1)] = beta[r];
    std::vector<int> k(nrhs, 0), active(nrhs);
    for (int r = 0; r < nrhs; ++r) active[r] = !done[r];
    for (int j = 0; j < mm; ++j) {
      C* Vj = Vb + (size_t)j * vs;
      C* Zj = Zb + (size_t)j * vs;
      C* W = Vb + (size_t)(j + 1) * vs;
      AMG_TRY_INTERNAL(vcycle_impl(h, vp, Vj, Zj, nrhs, st));        // Z_j = M V_j
      AMG_TRY_INTERNAL(dirac_any(h, Zj, nullptr, W, nrhs, st));      // w = D Z_j
      total_applies++;
      AMG_CUDA_TRY(cudaMemsetAsync(dh, 0, (size_t)(j + 1) * nrhs * sizeof(double2), st));
      fdots_kernel<C><<<dim3(vgrid, j + 1), fblk, 0, st>>>(Vb, vs, j + 1, W, n, nrhs, dh);
      AMG_LAUNCH_CHECK();
      AMG_CUDA_TRY(cudaMemsetAsync(dn, 0, nrhs * sizeof(double), st));
      fupdate_kernel<C><<<vgrid, fblk, 0, st>>>(Vb, vs, j + 1, dh, W, n, nrhs, dn);
      AMG_LAUNCH_CHECK();
      h->launches += 2;
      std::vector<double2> hc((size_t)(j + 1) * nrhs);
      AMG_CUDA_TRY(cudaMemcpyAsync(hc.data(), dh, hc.size() * sizeof(double2), cudaMemcpyDeviceToHost, st));
      AMG_CUDA_TRY(cudaMemcpyAsync(tmp.data(), dn, nrhs * sizeof(double), cudaMemcpyDeviceToHost, st));
      AMG_CUDA_TRY(cudaStreamSynchronize(st));
      bool more = false;
      for (int r = 0; r < nrhs; ++r) {
        coef[r] = make_double2(0, 0);
        if (!active[r]) continue;
        applies[r]++;
        std::complex<double>* Hr = H.data() + hs * r;  // Hr[i * m + j]
        for (int i = 0; i <= j; ++i) Hr[i * m + j] = std::complex<double>(hc[i * nrhs + r].x, hc[i * nrhs + r].y);
        const double hnext = sqrt(tmp[r]);
        Hr[(j + 1) * m + j] = hnext;
        std::complex<double>* c = cs.data() + (size_t)m * r;
        std::complex<double>* s = sn.data() + (size_t)m * r;
        std::complex<double>* gr = g.data() + (size_t)(m + 1) * r;
        for (int i = 0; i < j; ++i) {
          const std::complex<double> a = c[i] * Hr[i * m + j] + s[i] * Hr[(i + 1) * m + j];
          Hr[(i + 1) * m + j] = -std::conj(s[i]) * Hr[i * m + j] + std::conj(c[i]) * Hr[(i + 1) * m + j];
          Hr[i * m + j] = a;
        }
        const std::complex<double> a = Hr[j * m + j], b = Hr[(j + 1) * m + j];
        const double den = sqrt(std::norm(a) + std::norm(b));
        c[j] = std::conj(a) / den;
        s[j] = std::conj(b) / den;
        Hr[j * m + j] = den;
        Hr[(j + 1) * m + j] = 0.0;
        gr[j + 1] = -std::conj(s[j]) * gr[j];
        gr[j] = c[j] * gr[j];
        k[r] = j + 1;
        relres[r] = std::abs(gr[j + 1]) / fnorm[r];
        if (std::abs(gr[j + 1]) <= tol * fnorm[r] || hnext == 0) {
          active[r] = 0;
          done[r] = 1;
        } else {
          coef[r] = make_double2(1.0 / hnext, 0.0);
          more = true;
        }
      }
      if (!more) break;
      // V_{j+1} = w / h_{j+1,j} (columns that stopped get 0 and drop out of later sums)
      AMG_CUDA_TRY(cudaMemcpyAsync(dh, coef.data(), nrhs * sizeof(double2), cudaMemcpyHostToDevice, st));
      AMG_CUDA_TRY(cudaStreamSynchronize(st));
      fscale_kernel<C><<<vgrid, fblk, 0, st>>>(W, W, dh, n, nrhs);
      AMG_LAUNCH_CHECK();
      h->launches++;
    }
    // u += Z y, y from the k x k triangular systems
    std::vector<double2> yv((size_t)m * nrhs, make_double2(0, 0));
    int kmax = 0;
    for (int r = 0; r < nrhs; ++r) {
      const std::complex<double>* Hr = H.data() + hs * r;
      const std::complex<double>* gr = g.data() + (size_t)(m + 1) * r;
      std::vector<std::complex<double>> yy(k[r]);
      for (int i = k[r] - 1; i >= 0; --i) {
        std::complex<double> acc = gr[i];
        for (int q = i + 1; q < k[r]; ++q) acc -= Hr[i * m + q] * yy[q];
        yy[i] = acc / Hr[i * m + i];
      }
      for (int i = 0; i < k[r]; ++i) yv[i * nrhs + r] = make_double2(yy[i].real(), yy[i].imag());
      kmax = std::max(kmax, k[r]);
    }
    if (kmax > 0) {
      AMG_CUDA_TRY(cudaMemcpyAsync(dh, yv.data(), (size_t)kmax * nrhs * sizeof(double2), cudaMemcpyHostToDevice, st));
      fcombine_kernel<C><<<vgrid, fblk, 0, st>>>(Zb, vs, kmax, dh, U, n, nrhs);
      AMG_LAUNCH_CHECK();
      h->launches++;
    }
    bool all = true;
    for (int r = 0; r < nrhs; ++r) all = all && done[r];
    if (all || total_applies >= max_applies) break;
    // true residual r = f - D u
    AMG_TRY_INTERNAL(dirac_any(h, u, f, R, nrhs, st));
    total_applies++;
    for (int r = 0; r < nrhs; ++r)
      if (!done[r]) applies[r]++;
  }
  AMG_CUDA_TRY(cudaStreamSynchronize(st));
  if (info)
    for (int r = 0; r < nrhs; ++r) {
      info[2 * r] = applies[r];
      info[2 * r + 1] = relres[r];
    }
  return AMG_OK;
}

// Columns j0 .. j0 + nc - 1 of the FP64 test vectors tv ([V][12][ntv]) <-> a fine vector of nc
// columns in the vector precision ([V][12][nc]).
template <typename C>
__global__ void tv_gather_kernel(const double2* __restrict__ tv, C* __restrict__ out, long long n12, int ntv, int j0,
                                 int nc) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n12 * nc;
       e += (long long)gridDim.x * blockDim.x) {
    const double2 v = tv[(e / nc) * ntv + j0 + (int)(e % nc)];
    C o;
    o.x = v.x;
    o.y = v.y;
    out[e] = o;
  }
}

template <typename C>
__global__ void tv_scatter_kernel(const C* __restrict__ in, double2* __restrict__ tv, long long n12, int ntv, int j0,
                                  int nc) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n12 * nc;
       e += (long long)gridDim.x * blockDim.x)
    tv[(e / nc) * ntv + j0 + (int)(e % nc)] = make_double2((double)in[e].x, (double)in[e].y);
}

// Alg. 4 on the handle: see amg_adaptive_setup in amg.h.  The test vectors go through the smoother
// and the V-cycle in column chunks of at most min(max_nrhs, 16); R and D_c are rebuilt in place.
template <typename T>
amg_status adaptive_impl(amg_coarse* h, const amg_vcycle_params* vp, const double2* U, double2* tv, int n_setup,
                         cudaStream_t st) {
  using C = typename Cx<T>::type;
  const int ntv = h->g.ntv;
  const int chunk = std::min(h->p.max_nrhs, 16);
  const long long n12 = h->g.V * 12;
  const size_t vbytes = (size_t)n12 * chunk * sizeof(C);
  void* buf = nullptr;
  AMG_CUDA_TRY(alloc_or_give_back(
      h, [&] { return cudaMallocAsync(&buf, 2 * vbytes + 256 + (size_t)ntv * (sizeof(double) + sizeof(double2)), st); }));
  C* y = (C*)buf;
  C* x = y + (size_t)n12 * chunk;
  double* dn = (double*)(x + (size_t)n12 * chunk);
  double2* dc = (double2*)(dn + ntv);
  const int vgrid = 4 * amg_sm_count();
  amg_status s = AMG_OK;
  auto each_chunk = [&](auto&& body) -> amg_status {
    for (int j0 = 0; j0 < ntv; j0 += chunk) {
      const int nc = std::min(chunk, ntv - j0);
      tv_gather_kernel<C><<<vgrid, 256, 0, st>>>(tv, y, n12, ntv, j0, nc);
      AMG_LAUNCH_CHECK();
      AMG_TRY_INTERNAL(body(nc));
      tv_scatter_kernel<C><<<vgrid, 256, 0, st>>>(x, tv, n12, ntv, j0, nc);
      AMG_LAUNCH_CHECK();
      h->launches += 2;
    }
    return AMG_OK;
  };
  // initial phase: v <- S_k(v; 0), k = 1, 2, 3
  s = each_chunk([&](int nc) -> amg_status {
    for (int k = 1; k <= 3; ++k) {
      AMG_CUDA_TRY(cudaMemsetAsync(x, 0, (size_t)n12 * nc * sizeof(C), st));
      AMG_TRY_INTERNAL(sap_any(h, y, x, nc, k, vp->n_mr, st));
      if (k < 3) AMG_CUDA_TRY(cudaMemcpyAsync(y, x, (size_t)n12 * nc * sizeof(C), cudaMemcpyDeviceToDevice, st));
    }
    return AMG_OK;
  });
  if (s == AMG_OK) s = amg_internal_rebuild(h, U, tv, st);
  if (s == AMG_OK) {  // v_j <- v_j / ||v_j||
    cudaMemsetAsync(dn, 0, ntv * sizeof(double), st);
    fnorm_kernel<double2><<<vgrid, FT, 0, st>>>(tv, n12, ntv, dn);
    std::vector<double> nrm(ntv);
    cudaMemcpyAsync(nrm.data(), dn, ntv * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) s = AMG_ERR_CUDA;
    std::vector<double2> inv(ntv);
    for (int j = 0; j < ntv; ++j) inv[j] = make_double2(nrm[j] > 0 ? 1.0 / sqrt(nrm[j]) : 0.0, 0.0);
    if (s == AMG_OK && cudaMemcpyAsync(dc, inv.data(), ntv * sizeof(double2), cudaMemcpyHostToDevice, st) != cudaSuccess)
      s = AMG_ERR_CUDA;
    if (s == AMG_OK) {
      fscale_kernel<double2><<<vgrid, 256, 0, st>>>(tv, tv, dc, n12, ntv);
      if (cudaGetLastError() != cudaSuccess) s = AMG_ERR_CUDA;
      h->launches += 2;
    }
  }
  // iterative passes: v_j <- S(v_j; CGC(v_j)) with the current R and D_c, then rebuild
  for (int pass = 0; pass < n_setup && s == AMG_OK; ++pass) {
    s = each_chunk([&](int nc) -> amg_status { return vcycle_impl(h, vp, y, x, nc, st); });
    if (s == AMG_OK) s = amg_internal_rebuild(h, U, tv, st);
  }
  cudaFreeAsync(buf, st);
  cudaStreamSynchronize(st);
  return s;
}

// All but the pool
void free_fields(amg_coarse* h) {
  cudaFree(h->fU);
  if (h->fC != (void*)h->clover) cudaFree(h->fC);
  cudaFree(h->fwork);
  cudaFree(h->fW);
  cudaFree(h->fE);
  h->fW = nullptr;
  h->fE = nullptr;
  h->fU = h->fC = h->fwork = nullptr;
  h->fwork_bytes = 0;
}

}  // namespace

void amg_internal_free_fine(amg_coarse* h) {
  free_fields(h);
  if (h->fpool) cudaMemPoolDestroy(h->fpool);
  h->fpool = nullptr;
}

extern "C" {

amg_status amg_setup_fine(amg_handle h, const void* d_U, void* stream) {
  if (!h || !d_U || !aligned16(d_U)) return AMG_ERR_INVALID_ARG;
  if (h->level != 1) return AMG_ERR_UNSUPPORTED;  // a level-2 handle has no fine lattice
  if (h->p.vec_prec != AMG_FP64 && h->p.vec_prec != AMG_FP32) return AMG_ERR_UNSUPPORTED;
  cudaStream_t st = (cudaStream_t)stream;
  h->last_stream = st;
  free_fields(h);
  const long long nU = h->g.V * 36;
  if (fine_fp64(h)) {
    AMG_CUDA_TRY(cudaMalloc(&h->fU, nU * sizeof(double2)));
    AMG_CUDA_TRY(cudaMemcpyAsync(h->fU, d_U, nU * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    h->fC = h->clover;
    // words for the smoother's MR steps; without memory for them these run in FP64
    if (sap_supported(h)) {
      if (cudaMalloc(&h->fW, h->g.V * kFixQ * sizeof(int4)) == cudaSuccess &&
          cudaMalloc(&h->fE, h->g.Vc * sizeof(int)) == cudaSuccess) {
        fixed_words_kernel<<<(unsigned)h->g.Vc, 256, 0, st>>>((const double2*)h->fU, h->clover, (int4*)h->fW, h->fE,
                                                              fine_geom(h), 4.0 + h->p.m0);
        AMG_LAUNCH_CHECK();
        h->launches++;
      } else {
        cudaGetLastError();
        cudaFree(h->fW);
        h->fW = nullptr;
      }
    }
  } else {
    AMG_CUDA_TRY(cudaMalloc(&h->fU, h->g.V * kLinkQ * sizeof(float4)));
    if (cudaMalloc(&h->fC, h->g.V * kClovQ * sizeof(float4)) != cudaSuccess) {
      cudaGetLastError();
      amg_internal_free_fine(h);
      return AMG_ERR_OOM;
    }
    if (sap_supported(h)) sap_pool(h, st);
    links_words_kernel<<<8 * amg_sm_count(), 256, 0, st>>>((const double2*)d_U, (float4*)h->fU, h->g);
    AMG_LAUNCH_CHECK();
    clover_words_kernel<<<8 * amg_sm_count(), 256, 0, st>>>(h->clover, (float4*)h->fC, h->g);
    AMG_LAUNCH_CHECK();
    h->launches += 2;
  }
  return AMG_OK;
}

amg_status amg_dirac_apply(amg_handle h, const void* d_psi, void* d_out, int nrhs, void* stream) {
  AMG_TRY_INTERNAL(check_fine(h, d_psi, d_out, nrhs));
  if (d_psi == d_out) return AMG_ERR_INVALID_ARG;
  h->last_stream = (cudaStream_t)stream;
  return dirac_any(h, d_psi, nullptr, d_out, nrhs, (cudaStream_t)stream);
}

amg_status amg_sap(amg_handle h, const void* d_y, void* d_x, int nrhs, int n_cycles, int n_mr, void* stream) {
  AMG_TRY_INTERNAL(check_fine(h, d_y, d_x, nrhs));
  if (d_y == d_x || n_cycles < 0 || n_mr < 1) return AMG_ERR_INVALID_ARG;
  if (!sap_supported(h)) return AMG_ERR_UNSUPPORTED;
  h->last_stream = (cudaStream_t)stream;
  return sap_any(h, d_y, d_x, nrhs, n_cycles, n_mr, (cudaStream_t)stream);
}

amg_status amg_vcycle(amg_handle h, const amg_vcycle_params* vp, const void* d_y, void* d_x, int nrhs,
                      void* stream) {
  AMG_TRY_INTERNAL(check_fine(h, d_y, d_x, nrhs));
  AMG_TRY_INTERNAL(check_vp(vp));
  if (d_y == d_x) return AMG_ERR_INVALID_ARG;
  if (!sap_supported(h)) return AMG_ERR_UNSUPPORTED;
  h->last_stream = (cudaStream_t)stream;
  return vcycle_impl(h, vp, d_y, d_x, nrhs, (cudaStream_t)stream);
}

amg_status amg_adaptive_setup(amg_handle h, const amg_vcycle_params* vp, const void* d_U, void* d_tv, int n_setup,
                              void* stream) {
  if (!h || !d_U || !d_tv || !aligned16(d_U) || !aligned16(d_tv) || n_setup < 0) return AMG_ERR_INVALID_ARG;
  AMG_TRY_INTERNAL(check_vp(vp));
  if (h->next) return AMG_ERR_INVALID_ARG;  // an attached level 2 would keep D_cc of the old D_c
  if (!h->fU) return AMG_ERR_UNSUPPORTED;
  if (!sap_supported(h)) return AMG_ERR_UNSUPPORTED;
  cudaStream_t st = (cudaStream_t)stream;
  h->last_stream = st;
  return fine_fp64(h) ? adaptive_impl<double>(h, vp, (const double2*)d_U, (double2*)d_tv, n_setup, st)
                      : adaptive_impl<float>(h, vp, (const double2*)d_U, (double2*)d_tv, n_setup, st);
}

amg_status amg_solve(amg_handle h, const amg_vcycle_params* vp, const void* d_f, void* d_u, int nrhs, double tol,
                     int restart, int max_applies, void* stream, double* info) {
  AMG_TRY_INTERNAL(check_fine(h, d_f, d_u, nrhs));
  AMG_TRY_INTERNAL(check_vp(vp));
  if (d_f == d_u || !(tol >= 0) || restart < 1 || restart > 64 || max_applies < 1) return AMG_ERR_INVALID_ARG;
  if (!sap_supported(h)) return AMG_ERR_UNSUPPORTED;
  cudaStream_t st = (cudaStream_t)stream;
  h->last_stream = st;
  return fine_fp64(h) ? solve_impl<double>(h, vp, d_f, d_u, nrhs, tol, restart, max_applies, st, info)
                      : solve_impl<float>(h, vp, d_f, d_u, nrhs, tol, restart, max_applies, st, info);
}

}  // extern "C"
