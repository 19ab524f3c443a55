// Setup of the restriction and the coarse-grid operator (Alg. 5): the FP64 kernels, the clover in fixed point, and
// the driver, which chooses between these and the kernels of setup_gs.cu, setup_tc.cu and setup_ds.cu.
//
//   clover_kernel    C(x) = c_sw (i/4) sum sigma_{mu nu} F_{mu nu}(x), per chirality (Alg. 7's C^{hh})
//   gs_kernel        block classical Gram-Schmidt per aggregate (Sec. 3, "Gram-Schmidt on aggregates"), where
//                    those in fixed point (setup_gs.cu) and in pairs of floats (setup_ds.cu) do not serve
//   assemble_kernel  self and forward blocks of D_c = R D P (Eq. cgo via Alg. 7's D P), as sums
//                    over links of small rank-6 products: small blocks and few test vectors, and
//                    what the kernel on the tensor cores (setup_tc.cu) leaves of the others
//   combine_kernel   D_c blocks from the partial sums; backward blocks by Eq. dagger
//   quantize_*       D_c and R to the storage precisions of the applies (Sec. 3: half precision D_c)
#include "fixed.cuh"

#include <stdio.h>
#include <stdlib.h>
#include <algorithm>
#include <vector>

namespace {
using namespace amgfix;

// ------------------------------------------------------------------ clover term
// Products of links in fixed point: entry = (h 2^31 + l) 2^(e - 60) with |h| <= 2^29, |l| <= 2^30 and one exponent for
// the matrix, taken from its largest entry.
struct I3 {
  int2 re[9], im[9];
  int e;
};
// U, or its adjoint; `bad` is set if an entry is not finite
__device__ __forceinline__ I3 load_link(const double2* __restrict__ p, bool dagger, bool& bad) {
  double2 u[9];
  int f = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double2 v = __ldg(p + (dagger ? j * 3 + i : i * 3 + j));
      f = max(f, max((__double2hiint(v.x) >> 20) & 0x7FF, (__double2hiint(v.y) >> 20) & 0x7FF));
      u[i * 3 + j] = v;
    }
  bad |= f == 0x7FF;
  I3 m;
  m.e = max(f - 1022, -900);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    m.re[k] = words31(fixed<60>(u[k].x, m.e));
    m.im[k] = words31(fixed<60>(u[k].y, m.e, dagger ? (int)0x80000000 : 0));
  }
  return m;
}
// z = a b in units of 2^(a.e + b.e - 58): |z| < 6 2^58, the product of the low words left out (3 units at most)
__device__ __forceinline__ void mul(const I3& a, const I3& b, long long (&re)[9], long long (&im)[9]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      long long hr = 0, lr = 0, hi = 0, li = 0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int2 ar = a.re[i * 3 + k], ai = a.im[i * 3 + k], br = b.re[k * 3 + j], bi = b.im[k * 3 + j];
        mac(hr, lr, ar, br);
        mac(hr, lr, minus(ai), bi);
        mac(hi, li, ar, bi);
        mac(hi, li, ai, br);
      }
      re[i * 3 + j] = hr + (lr >> 31);
      im[i * 3 + j] = hi + (li >> 31);
    }
}
// z 2^(unit) with the largest entry brought to 60 bits
__device__ __forceinline__ I3 scaled(const long long (&re)[9], const long long (&im)[9], int unit) {
  int top = 0;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int r = (int)(re[k] >> 32), i = (int)(im[k] >> 32);
    top |= (r ^ (r >> 31)) | (i ^ (i >> 31));
  }
  const int s = __clz(top) - 3;  // bits to shift left after one to the right: highest bit 59 (at most 28 bits)
  I3 m;
  m.e = unit + 61 - s;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    m.re[k] = words31((re[k] << s) >> 1);
    m.im[k] = words31((im[k] << s) >> 1);
  }
  return m;
}

// Step s of leaf `leaf` of plane (mu, nu) from y: the leaf follows the steps +mu, +nu, -mu, -nu from the leaf-th on, round.
// Returns the link passed (its adjoint is meant if `back`) and moves y on.
__device__ __forceinline__ const double2* leaf_link(const double2* __restrict__ U, const Geom& g, int (&y)[4], int mu, int nu,
                                                    int leaf, int s, bool& back) {
  const int k = (leaf + s) & 3, d = k & 1 ? nu : mu;
  back = k >= 2;
  long long site = 0;
  int step = 0;
#pragma unroll
  for (int m = 3; m >= 0; --m) {
    const int fwd = y[m] + 1 < g.L[m] ? y[m] + 1 : 0, bwd = y[m] > 0 ? y[m] - 1 : g.L[m] - 1;
    if (m == d) step = back ? bwd : fwd;
    if (m == d && back) y[m] = bwd;
    site = site * g.L[m] + y[m];
  }
#pragma unroll
  for (int m = 0; m < 4; ++m)
    if (m == d) y[m] = step;
  return U + (site * 4 + d) * 9;
}

// field_strength in FP64, where every part keeps the accuracy of its own size.  Out of line: links close to 1, whose F
// is far below them, are the exception.
__device__ __noinline__ void field_strength_fp64(const double2* __restrict__ U, const Geom& g, int x0, int x1, int x2, int x3,
                                                 int mu, int nu, double* f) {
  double2 q[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) q[k] = make_double2(0, 0);
#pragma unroll 1
  for (int leaf = 0; leaf < 4; ++leaf) {
    int y[4] = {x0, x1, x2, x3};
    double2 t[9] = {};
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
      bool back;
      const double2* p = leaf_link(U, g, y, mu, nu, leaf, s, back);
      double2 u[9], z[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        u[k] = __ldg(p + (back ? k % 3 * 3 + k / 3 : k));
        if (back) u[k].y = -u[k].y;
      }
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          z[i * 3 + j] = make_double2(0, 0);
#pragma unroll
          for (int k = 0; k < 3; ++k) cfma(z[i * 3 + j], t[i * 3 + k], u[k * 3 + j]);
        }
#pragma unroll
      for (int k = 0; k < 9; ++k) t[k] = s ? z[k] : u[k];
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) q[k] = cadd(q[k], t[k]);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) f[i] = 0.25 * q[4 * i].y;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = k < 2 ? 0 : 1, j = k < 1 ? 1 : 2;
    f[3 + 2 * k] = 0.125 * (q[i * 3 + j].x - q[j * 3 + i].x);
    f[4 + 2 * k] = 0.125 * (q[i * 3 + j].y + q[j * 3 + i].y);
  }
}

// F_{mu nu}(x) = (Q - Q^dagger)/8 with Q the four counter-clockwise leaves at x.  f: imaginary parts of the diagonal, real and
// imaginary parts of (0,1), (0,2), (1,2); F is anti-Hermitian.  The fixed-point sums are good to about 2^-57 of the links'
// products; returns true if F lies below 2^-kWeakBits of these.
constexpr int kWeakBits = 7;  // spread 0.2 of the links: F about 0.1
__device__ __forceinline__ bool field_strength(const double2* __restrict__ U, const Geom& g, const int (&x)[4], int mu,
                                               int nu, double* f) {
  long long qr[9], qi[9];
  int unit = 0;  // of Q
  bool bad = false;
#pragma unroll 1
  for (int leaf = 0; leaf < 4; ++leaf) {
    int y[4] = {x[0], x[1], x[2], x[3]};
    I3 t;
    long long zr[9], zi[9];
    int uz = 0;
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
      bool back;
      const double2* p = leaf_link(U, g, y, mu, nu, leaf, s, back);
      const I3 u = load_link(p, back, bad);
      if (s == 0) {
        t = u;
      } else {
        mul(t, u, zr, zi);
        uz = t.e + u.e - 58;
        if (s < 3) t = scaled(zr, zi, uz);
      }
    }
    if (leaf == 0) {
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        qr[k] = zr[k];
        qi[k] = zi[k];
      }
      unit = uz;
    } else {  // in the larger of the two units; four times 6 2^58 fits
      const int top = max(unit, uz), sq = min(top - unit, 63), sz = min(top - uz, 63);
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        qr[k] = (qr[k] >> sq) + (zr[k] >> sz);
        qi[k] = (qi[k] >> sq) + (zi[k] >> sz);
      }
      unit = top;
    }
  }
  // halves, for the sums to fit
  auto value = [&](long long a) { return bad ? nan("") : scalbn((double)a, unit - 2); };
#pragma unroll
  for (int i = 0; i < 3; ++i) f[i] = value(qi[4 * i]);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = k < 2 ? 0 : 1, j = k < 1 ? 1 : 2;
    f[3 + 2 * k] = value((qr[i * 3 + j] >> 1) - (qr[j * 3 + i] >> 1));
    f[4 + 2 * k] = value((qi[i * 3 + j] >> 1) + (qi[j * 3 + i] >> 1));
  }
  int top = 0;
#pragma unroll
  for (int k = 0; k < 9; ++k) top = max(top, (__double2hiint(f[k]) >> 20) & 0x7FF);
  return top < unit + 58 - kWeakBits + 1022 && !bad;
}

// In the chiral basis sigma_{mu nu} = diag(s^l, s^r) with 2x2 blocks
//   s_{kl} = -eps_{klm} sigma_m (both chiralities), s_{k4} = +sigma_k (l), -sigma_k (r).
// Hence C^{hh} = c_sw (i/2) sum_m sigma_m (x) G^h_m with
//   G^h_m = -B_m + s_h E_m,  B = (F_yz, F_zx, F_xy),  E_m = F_{m t},  s_l = +1, s_r = -1.
//
// Bound: integer multiply-adds and the fixed-point conversions: 72 products of 3 x 3 matrices per site, 12 multiply-adds
// per complex one (a sixteenth of the time of 4 in FP64 each).  One body for all planes, leaves and steps
// stays in the instruction cache (links close to 1 take a second one, in FP64).  16^3 x 32: 1.02 ms (with 255 registers and two CTAs per SM 1.09 ms), in FP64 1.99 ms.
__global__ void __launch_bounds__(128, 3) clover_kernel(const double2* __restrict__ U, double2* __restrict__ C, Geom g,
                                                     double csw) {
  const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int c[4];
  long long r = s;
  c[0] = (int)(r % g.L[0]);
  r /= g.L[0];
  c[1] = (int)(r % g.L[1]);
  r /= g.L[1];
  c[2] = (int)(r % g.L[2]);
  c[3] = (int)(r / g.L[2]);
  double F[6][9];  // planes (0,1), (0,2), (1,2), (0,3), (1,3), (2,3)
  unsigned weak = 0;
#pragma unroll 1
  for (int p = 0; p < 6; ++p)
    weak |= (unsigned)field_strength(U, g, c, p < 2 ? 0 : p == 2 ? 1 : p - 3, p == 0 ? 1 : p < 3 ? 2 : 3, F[p]) << p;
#pragma unroll 1
  for (int p = 0; p < 6; ++p)
    if (weak >> p & 1)
      field_strength_fp64(U, g, c[0], c[1], c[2], c[3], p < 2 ? 0 : p == 2 ? 1 : p - 3, p == 0 ? 1 : p < 3 ? 2 : 3, F[p]);
  auto entry = [&](int p, int k) {
    const int i = k / 3, j = k % 3, o = 2 * (i + j) + 1;
    return i == j ? make_double2(0, F[p][i]) : make_double2(i < j ? F[p][o] : -F[p][o], F[p][o + 1]);
  };
  for (int h = 0; h < 2; ++h) {
    const double sh = h == 0 ? 1.0 : -1.0;
    double2 G[3][9];  // -B_m +- E_m, B = (F_12, -F_02, F_01)
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const double2 b = entry(2 - m, k), e = entry(3 + m, k);
        const double sb = m == 1 ? 1.0 : -1.0;
        G[m][k] = make_double2(sb * b.x + sh * e.x, sb * b.y + sh * e.y);
      }
    // spin blocks: (0,0) = G_z, (1,1) = -G_z, (0,1) = G_x - i G_y, (1,0) = G_x + i G_y
    double2* out = C + (s * 2 + h) * 36;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const int k = i * 3 + j;
            double2 v;
            if (a == 0 && b == 0) v = G[2][k];
            else if (a == 1 && b == 1) v = cscale(G[2][k], -1.0);
            else if (a == 0) v = make_double2(G[0][k].x + G[1][k].y, G[0][k].y - G[1][k].x);
            else v = make_double2(G[0][k].x - G[1][k].y, G[0][k].y + G[1][k].x);
            // times c_sw (i/2)
            out[(a * 3 + i) * 6 + b * 3 + j] = make_double2(-0.5 * csw * v.y, 0.5 * csw * v.x);
          }
  }
}

// ------------------------------------------------------------------ block reductions
// Sum of NV values (a power of two, at most 32) over the warp's lanes; lane l gets the total of value
// l >> (5 - log2 NV).  Halving the values with the distance takes NV - 1 + (5 - log2 NV) FP64 additions
// instead of 5 NV.
template <int NV>
__device__ inline double warp_totals(double (&v)[NV]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int n = NV / 2; n > 0; n /= 2, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < NV / 2; ++i)
      if (i < n) {
        const double give = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
  }
  for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}
// CTA sums of NV values: left in out[0 .. NV - 1] (shared; valid after this call's last barrier).
// sm: [warps][NV]
template <int NV>
__device__ inline void block_totals(double (&v)[NV], double* sm, double* out) {
  constexpr int sh = NV == 32 ? 0 : NV == 16 ? 1 : NV == 8 ? 2 : NV == 4 ? 3 : NV == 2 ? 4 : 5;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const double t = warp_totals<NV>(v);
  if ((lane & ((1 << sh) - 1)) == 0) sm[warp * NV + (lane >> sh)] = t;
  __syncthreads();
  if (threadIdx.x < NV) {
    double sum = 0;
    for (int w = 0; w < nw; ++w) sum += sm[w * NV + threadIdx.x];
    out[threadIdx.x] = sum;
  }
  __syncthreads();
}

// ------------------------------------------------------------------ Gram-Schmidt
// One CTA per aggregate (blk, h).  The aggregate's test vectors (6 Vb x ntv) are processed in
// column blocks of NB = 4: each block is projected against all earlier columns with classical
// Gram-Schmidt (all coefficients from the same vectors), twice, then orthonormalised column by
// column, again classically and twice.  Element n of the aggregate lives in thread n mod T, E elements
// per thread.  Output row j of R_i^h = conj(q_j).
//
// Bound: the FP64 pipes (one warp instruction in 64 cycles per sub-partition): 4 instructions per element and pair
// of columns in every dot and every update, and as little else as possible: updates add the negated
// coefficients, sums halve their values as they go down the lanes, one warp takes the roots and
// reciprocals.  It serves up to 4 test vectors of large aggregates, those beyond the fixed-point kernel (setup_gs.cu) and
// those that it leaves.
// 16^4, Ntv 2: 0.105 ms; Ntv 20: 5.5 ms; with a multiplication, a fused one and a subtraction per update,
// 5 additions per value and lane and roots in every thread 8.8 ms.
constexpr int GS_NB = 4;
constexpr int GS_EMAX = 8;

template <int E>
__global__ void __launch_bounds__(256) gs_kernel(const double2* __restrict__ tv, double2* __restrict__ R,
                                                 Geom g, const int* __restrict__ only, unsigned* err) {
  if (only && !only[blockIdx.x]) return;
  __shared__ double sm[8 * 32], tot[32], n0[GS_NB], scal;
  __shared__ double2 coef[AMG_MAX_NTV * GS_NB];  // minus the coefficients
  const long long agg = blockIdx.x;
  const long long blk = agg >> 1;
  const int h = (int)(agg & 1);
  const int T = blockDim.x, tid = threadIdx.x, ntv = g.ntv, nagg = g.nagg;
  long long tvoff[E];
  bool valid[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int n = tid + e * T;
    valid[e] = n < nagg;
    tvoff[e] = 0;
    if (valid[e]) {
      const int sl = n / 6, a = (n % 6) / 3, col = n % 3;
      const long long site = block_site(g, blk, sl);
      tvoff[e] = ((site * 4 + 2 * h + a) * 3 + col) * (long long)ntv;
    }
  }
  double2* Rblk = R + agg * (long long)ntv * nagg;
  double2 w[E][GS_NB];
  for (int j0 = 0; j0 < ntv; j0 += GS_NB) {
    const int nb = min(GS_NB, ntv - j0);
#pragma unroll
    for (int e = 0; e < E; ++e)
#pragma unroll
      for (int c = 0; c < GS_NB; ++c)
        w[e][c] = (valid[e] && c < nb) ? tv[tvoff[e] + j0 + c] : make_double2(0, 0);
    {
      double v[GS_NB];
#pragma unroll
      for (int c = 0; c < GS_NB; ++c) {
        v[c] = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) v[c] = fma(w[e][c].x, w[e][c].x, fma(w[e][c].y, w[e][c].y, v[c]));
      }
      block_totals<GS_NB>(v, sm, tot);
      if (tid < GS_NB) n0[tid] = tot[tid];
    }
    // projection against the earlier column blocks (block classical GS), twice
    for (int pass = 0; pass < 2 && j0 > 0; ++pass) {
      for (int k0 = 0; k0 < j0; k0 += GS_NB) {
        double2 d[GS_NB * GS_NB];
#pragma unroll
        for (int q = 0; q < GS_NB * GS_NB; ++q) d[q] = make_double2(0, 0);
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if (!valid[e]) continue;
          const int n = tid + e * T;
#pragma unroll
          for (int kk = 0; kk < GS_NB; ++kk) {
            const double2 r = Rblk[(long long)(k0 + kk) * nagg + n];  // conj(q_k)
#pragma unroll
            for (int c = 0; c < GS_NB; ++c) cfma(d[kk * GS_NB + c], r, w[e][c]);
          }
        }
        double v[2 * GS_NB * GS_NB];
#pragma unroll
        for (int q = 0; q < GS_NB * GS_NB; ++q) {
          v[2 * q] = d[q].x;
          v[2 * q + 1] = d[q].y;
        }
        block_totals<2 * GS_NB * GS_NB>(v, sm, tot);
        if (tid < GS_NB * GS_NB) coef[k0 * GS_NB + tid] = make_double2(-tot[2 * tid], -tot[2 * tid + 1]);
        __syncthreads();
      }
      for (int k0 = 0; k0 < j0; k0 += GS_NB) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if (!valid[e]) continue;
          const int n = tid + e * T;
#pragma unroll
          for (int kk = 0; kk < GS_NB; ++kk) {
            const double2 r = Rblk[(long long)(k0 + kk) * nagg + n];
#pragma unroll
            for (int c = 0; c < GS_NB; ++c) cfmac(w[e][c], r, coef[(k0 + kk) * GS_NB + c]);  // w -= q_k coef
          }
        }
      }
      __syncthreads();
    }
    // orthonormalise inside the block
#pragma unroll
    for (int c = 0; c < GS_NB; ++c) {
      if (c >= nb) break;
      for (int pass = 0; pass < 2 && c > 0; ++pass) {
        double v[2 * GS_NB];
#pragma unroll
        for (int cp = 0; cp < GS_NB; ++cp) {
          double2 d = make_double2(0, 0);
          if (cp < c)
#pragma unroll
            for (int e = 0; e < E; ++e) cfmac(d, w[e][cp], w[e][c]);
          v[2 * cp] = d.x;
          v[2 * cp + 1] = d.y;
        }
        block_totals<2 * GS_NB>(v, sm, tot);
#pragma unroll
        for (int cp = 0; cp < GS_NB; ++cp)
          if (cp < c) {
            const double2 m = make_double2(-tot[2 * cp], -tot[2 * cp + 1]);
#pragma unroll
            for (int e = 0; e < E; ++e) cfma(w[e][c], w[e][cp], m);
          }
        __syncthreads();  // tot is read
      }
      double v[1] = {0};
#pragma unroll
      for (int e = 0; e < E; ++e) v[0] = fma(w[e][c].x, w[e][c].x, fma(w[e][c].y, w[e][c].y, v[0]));
      block_totals<1>(v, sm, tot);
      if (tid < 32) {
        const double nrm = sqrt(tot[0]);
        if (tid == 0) {
          if (!(nrm > 1e-12 * sqrt(n0[c]))) atomicOr(err, AMG_EBIT_RANK);
          scal = nrm > 0 ? 1.0 / nrm : 0.0;
        }
      }
      __syncthreads();
      const double inv = scal;
#pragma unroll
      for (int e = 0; e < E; ++e) w[e][c] = cscale(w[e][c], inv);
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if (!valid[e]) continue;
      const int n = tid + e * T;
#pragma unroll
      for (int c = 0; c < GS_NB; ++c)
        if (c < nb) Rblk[(long long)(j0 + c) * nagg + n] = cconj(w[e][c]);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ D_c = R D P assembly
// With (1 - gamma_mu) = u u^dagger, u^dagger = [1, -b_mu] (b_mu the upper-right 2x2 block of
// gamma_mu in the chiral basis), one forward hop x -> x+mu contributes to R_i D P_j
//     -1/2 P(x)^dagger u u^dagger U_mu(x) P(x+mu) = -1/2 A(x)^dagger Bt(x)
// with A = u^dagger P(x) and Bt = u^dagger U_mu(x) P(x+mu), both 6 x 2ntv.  Job mu sums
// A^dagger Bt over the links of block i: links inside the block go to S_mu, links leaving through
// the +mu face to F_mu.  Job 4 sums P(x)^dagger ((4+m0) + C(x)) P(x) with both chiralities
// stacked in the same 6 rows (only the chirality-diagonal quadrants are kept).
// b_mu: -i sigma_x, -i sigma_y, -i sigma_z, 1.
//
// Bound: the FP64 pipes (one warp instruction in 64 cycles per SM sub-partition), so what counts is the
// number of FP64 warp instructions per sub-partition.  Each thread keeps a TA x TC tile of the sum; the
// CTA has a multiple of four warps, and where the tiles fill fewer, groups of warps share out the
// sites; the tile shape is the one that needs the fewest instructions so, links leaving through the face come last so that one set of
// accumulators serves S_mu and F_mu, the self job works on the tiles that its quadrants need, and the
// factors b_mu (+-1, +-i) only move words and flip signs in the integer pipe.  16^4 in 2^4 blocks, Ntv 8: 4.5 ms, Ntv 6:
// 3.2 ms; 2 x 4 tiles in two accumulator sets, all tiles of the self job and b_mu as products took 8.6 and 8.3 ms.
__device__ inline double flip(double v) {  // -v off the FP64 pipe
  return __hiloint2double(__double2hiint(v) ^ (int)0x80000000, __double2loint(v));
}
__device__ inline double2 conj_i(double2 z) { return make_double2(z.x, flip(z.y)); }
// row a of -b_mu z, z the entry of spin b(a) = 1 - a (mu < 2), a (mu >= 2)
__device__ inline double2 neg_b(int mu, int a, double2 z) {
  if (mu == 0 || (mu == 2 && a == 0)) return make_double2(flip(z.y), z.x);  // i z
  if (mu == 2) return make_double2(z.y, flip(z.x));                         // -i z
  if (mu == 1 && a == 0) return z;
  return make_double2(flip(z.x), flip(z.y));
}
// visiting order t -> local site: the sites with l_mu = B_mu - 1 last
__device__ inline int face_last(int t, int nface, int stride, int Bmu) {
  const int lmu = t / nface, r = t % nface;
  return (r / stride) * (stride * Bmu) + lmu * stride + (r % stride);
}

// The TA x TC tiles of the nc x nc sum that a job needs: all, or (self) those that meet a
// chirality-diagonal quadrant
struct Tiles {
  int nta, ntc, TA, TC, ntv;
  bool self;
  __host__ __device__ int first(int ta) const { return self && ta * TA >= ntv ? ntv / TC : 0; }
  __host__ __device__ int last(int ta) const { return self && ta * TA + TA <= ntv ? (ntv + TC - 1) / TC : ntc; }
  __host__ __device__ int count() const {
    if (!self) return nta * ntc;
    int n = 0;
    for (int ta = 0; ta < nta; ++ta) n += last(ta) - first(ta);
    return n;
  }
  __host__ __device__ bool at(int k, int& ta, int& tc) const {  // the k-th of them
    tc = 0;
    for (ta = 0; ta < nta; ++ta) {
      const int n = last(ta) - first(ta);
      if (k < n) {
        tc = first(ta) + k;
        return true;
      }
      k -= n;
    }
    return false;
  }
};

template <int TA, int TC>
__global__ void __launch_bounds__(256) assemble_kernel(const double2* __restrict__ R, const double2* __restrict__ U,
                                const double2* __restrict__ clov, double2* __restrict__ part, Geom g,
                                double m0, int ncp, int sb_max, const int* __restrict__ only) {
  if (only && !only[blockIdx.x * 5 + blockIdx.y]) return;
  extern __shared__ double2 smem[];
  const long long blk = blockIdx.x;
  const int job = blockIdx.y;
  const int nc = g.nc, ntv = g.ntv, nagg = g.nagg, Vb = (int)g.Vb;
  double2* As = smem;                        // [sb][6][ncp]
  double2* Bs = smem + (size_t)sb_max * 6 * ncp;
  const int nta = (nc + TA - 1) / TA, ntc = (nc + TC - 1) / TC;
  const int tid = threadIdx.x, nwarp = blockDim.x >> 5;
  // tiles of this job over tw warps; the CTA's warps form KG groups that share out the sites
  const Tiles need{nta, ntc, TA, TC, ntv, job == 4};
  const int tw = (need.count() + 31) / 32, KG = max(1, nwarp / tw), kg = (tid >> 5) / tw, lt = tid - kg * tw * 32;
  int ta, tc;
  const bool active = need.at(lt, ta, tc) && kg < KG;
  double2 acc[TA][TC];
#pragma unroll
  for (int i = 0; i < TA; ++i)
#pragma unroll
    for (int j = 0; j < TC; ++j) acc[i][j] = make_double2(0, 0);
  double2* P0 = part + ((blk * 5 + job) * 2 + 0) * (long long)nc * nc;
  auto write = [&](double2* P) {  // sum over the groups (through shared memory), then out; clears the tiles
    if (active && kg > 0)
#pragma unroll
      for (int i = 0; i < TA; ++i)
#pragma unroll
        for (int jj = 0; jj < TC; ++jj) smem[(((kg - 1) * TA + i) * TC + jj) * tw * 32 + lt] = acc[i][jj];
    __syncthreads();
    for (int q = 1; active && kg == 0 && q < KG; ++q)
#pragma unroll
      for (int i = 0; i < TA; ++i)
#pragma unroll
        for (int jj = 0; jj < TC; ++jj) acc[i][jj] = cadd(acc[i][jj], smem[(((q - 1) * TA + i) * TC + jj) * tw * 32 + lt]);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TA; ++i)
#pragma unroll
      for (int jj = 0; jj < TC; ++jj) {
        const int a = ta * TA + i, c = tc * TC + jj;
        if (active && kg == 0 && a < nc && c < nc) P[a * nc + c] = acc[i][jj];
        acc[i][jj] = make_double2(0, 0);
      }
  };
  // coarse coordinates of this block and stride of direction mu inside a block
  int X[4];
  {
    long long r = blk;
    for (int m = 0; m < 4; ++m) {
      X[m] = (int)(r % g.Lc[m]);
      r /= g.Lc[m];
    }
  }
  const int mu = job < 4 ? job : 0;
  int stride_mu = 1;
  for (int m = 0; m < mu; ++m) stride_mu *= g.B[m];
  X[mu] = (X[mu] + 1) % g.Lc[mu];
  const long long blk_fwd = ((long long)(X[3] * g.Lc[2] + X[2]) * g.Lc[1] + X[1]) * g.Lc[0] + X[0];
  const int Bmu = g.B[mu], nface = job < 4 ? Vb / Bmu : 0;
  int end = Vb - nface;  // the links inside the block first
  if (end == 0) {
    write(P0);  // S_mu of a block of extent 1: none
    end = Vb;
  }
  for (int s0 = 0, nsb = 0; s0 < Vb; s0 += nsb) {
    nsb = min(sb_max, end - s0);
    for (int pr = tid; pr < nsb * ncp; pr += blockDim.x) {
      const int sb = pr / ncp, c = pr % ncp;
      double2 *Ao = As + (size_t)sb * 6 * ncp + c, *Bo = Bs + (size_t)sb * 6 * ncp + c;
      if (c >= nc) {
#pragma unroll
        for (int k = 0; k < 6; ++k) Ao[k * ncp] = Bo[k * ncp] = make_double2(0, 0);
        continue;
      }
      const int sl = job < 4 ? face_last(s0 + sb, nface, stride_mu, Bmu) : s0 + sb;
      const long long site = block_site(g, blk, sl);
      const int hc = c / ntv, j = c % ntv;
      const double2* Rc = R + ((blk * 2 + hc) * (long long)ntv + j) * nagg + sl * 6;
      double2 q[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) q[k] = conj_i(Rc[k]);
      if (job < 4) {
        // A = u^dagger P(x): l columns keep the l rows, r columns give -b_mu P_r; Bt the same of
        // U_mu(x) P(x + mu), with the neighbour and its block
        const bool face = s0 + sb >= Vb - nface;
        const int sn = face ? sl - (Bmu - 1) * stride_mu : sl + stride_mu;
        const double2* Rn = R + (((face ? blk_fwd : blk) * 2 + hc) * (long long)ntv + j) * nagg + sn * 6;
        const double2* Ul = U + (site * 4 + mu) * 9;
        double2 qn[6], z[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) qn[k] = conj_i(Rn[k]);
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int col = 0; col < 3; ++col) {
            double2 t = make_double2(0, 0);
#pragma unroll
            for (int cp = 0; cp < 3; ++cp) cfma(t, Ul[col * 3 + cp], qn[b * 3 + cp]);
            z[b * 3 + col] = t;
          }
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
          for (int col = 0; col < 3; ++col) {
            const int k = a * 3 + col, kb = (1 - a) * 3 + col;
            Ao[k * ncp] = hc == 0 ? q[k] : neg_b(mu, a, mu < 2 ? q[kb] : q[k]);
            Bo[k * ncp] = hc == 0 ? z[k] : neg_b(mu, a, mu < 2 ? z[kb] : z[k]);
          }
      } else {
        const double2* C6 = clov + (site * 2 + hc) * 36;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          Ao[k * ncp] = q[k];
          double2 t = cscale(q[k], 4.0 + m0);
#pragma unroll
          for (int kp = 0; kp < 6; ++kp) cfma(t, C6[k * 6 + kp], q[kp]);
          Bo[k * ncp] = t;
        }
      }
    }
    __syncthreads();
    if (active) {
      for (int sb = kg; sb < nsb; sb += KG) {
#pragma unroll 1
        for (int k = 0; k < 6; ++k) {
          double2 av[TA], bv[TC];
#pragma unroll
          for (int i = 0; i < TA; ++i) av[i] = As[((size_t)sb * 6 + k) * ncp + ta * TA + i];
#pragma unroll
          for (int jj = 0; jj < TC; ++jj) bv[jj] = Bs[((size_t)sb * 6 + k) * ncp + tc * TC + jj];
#pragma unroll
          for (int i = 0; i < TA; ++i)
#pragma unroll
            for (int jj = 0; jj < TC; ++jj) cfmac(acc[i][jj], av[i], bv[jj]);
        }
      }
    }
    __syncthreads();
    if (s0 + nsb == end && end < Vb) {
      write(P0);  // S_mu
      end = Vb;
    }
  }
  write(job < 4 ? P0 + (long long)nc * nc : P0);  // F_mu, or the self block
}

// D_c blocks from the partial sums:
//   self:  Diag (chirality-diagonal part) - 1/2 sum_mu (S_mu + g5c S_mu^dagger g5c)
//   +mu:   -1/2 F_mu(i)
//   -mu:   g5c (D_c[i-mu][+mu])^dagger g5c            (Eq. dagger)
// where g5c S^dagger g5c accounts for the backward hops inside the block (gamma_5-hermiticity).
__global__ void combine_kernel(const double2* __restrict__ part, const int* __restrict__ nbr,
                               double2* __restrict__ Dc, Geom g) {
  const long long nc = g.nc;
  const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long total = g.Vc * 9 * nc * nc;
  if (idx >= total) return;
  const int c = (int)(idx % nc);
  const int a = (int)((idx / nc) % nc);
  const int d = (int)((idx / (nc * nc)) % 9);
  const long long i = idx / (9 * nc * nc);
  const double sa = a < g.ntv ? 1.0 : -1.0, sc = c < g.ntv ? 1.0 : -1.0;
  auto P = [&](long long site, int job, int slot) {
    return part + ((site * 5 + job) * 2 + slot) * nc * nc;
  };
  double2 v;
  if (d == 0) {
    v = ((a < g.ntv) == (c < g.ntv)) ? P(i, 4, 0)[a * nc + c] : make_double2(0, 0);
    for (int mu = 0; mu < 4; ++mu) {
      const double2* S = P(i, mu, 0);
      const double2 s1 = S[a * nc + c], s2 = cconj(S[c * nc + a]);
      v.x -= 0.5 * (s1.x + sa * sc * s2.x);
      v.y -= 0.5 * (s1.y + sa * sc * s2.y);
    }
  } else if (d & 1) {
    const int mu = (d - 1) >> 1;
    v = cscale(P(i, mu, 1)[a * nc + c], -0.5);
  } else {
    const int mu = (d - 2) >> 1;
    const long long j = nbr[i * 9 + d];
    v = cscale(cconj(P(j, mu, 1)[c * nc + a]), -0.5 * sa * sc);
  }
  Dc[idx] = v;
}

// D_c to the apply layout At[i][d][col][row] in FP64 / FP32, or FP16 with one FP32 scale per
// (site, direction): s = maxabs / 2^15, stored = value / s rounded to nearest (Sec. 3: half
// precision storage of D_c).
template <int MODE>
__global__ void quantize_dc_kernel(const double2* __restrict__ Dc, void* __restrict__ out,
                                   float* __restrict__ scale, int nc) {
  __shared__ double red[32];
  const long long blk = blockIdx.x;  // (i, d)
  const double2* src = Dc + blk * (long long)nc * nc;
  const int n2 = nc * nc;
  double inv = 1.0;
  float sf = 1.0f;
  if (MODE == 2) {
    double m = 0;
    for (int e = threadIdx.x; e < n2; e += blockDim.x) m = fmax(m, fmax(fabs(src[e].x), fabs(src[e].y)));
    for (int o = 16; o; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmax(t, red[w]);
      red[0] = t;
    }
    __syncthreads();
    const double maxabs = red[0];
    sf = maxabs > 0 ? (float)(maxabs / 32768.0) : 1.0f;
    inv = 1.0 / (double)sf;
    if (threadIdx.x == 0) scale[blk] = sf;
  }
  for (int e = threadIdx.x; e < n2; e += blockDim.x) {
    const int col = e / nc, row = e % nc;
    const double2 v = src[row * nc + col];
    const long long o = blk * (long long)n2 + e;
    if (MODE == 0) {
      ((double2*)out)[o] = v;
    } else if (MODE == 1) {
      ((float2*)out)[o] = make_float2((float)v.x, (float)v.y);
    } else {
      __half2 hv;
      hv.x = __double2half(v.x * inv);
      hv.y = __double2half(v.y * inv);
      ((__half2*)out)[o] = hv;
    }
  }
}

__global__ void r_to_fp32_kernel(const double2* __restrict__ R, float2* __restrict__ out, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = make_float2((float)R[i].x, (float)R[i].y);
}

}  // namespace

// ------------------------------------------------------------------ host driver
static int round_up(int a, int b) { return (a + b - 1) / b * b; }

// Warps of the assembly's CTA: the hop jobs' tiles, rounded up to a multiple of four
static int assemble_warps(int nc, int ta, int tc) {
  return round_up((((nc + ta - 1) / ta) * ((nc + tc - 1) / tc) + 31) / 32, 4);
}

template <int TA, int TC>
static amg_status launch_assemble_tile(const Geom& g, const double2* R, const double2* U, const double2* clov,
                                       double2* part, double m0, const int* only, cudaStream_t st) {
  const int ncp = std::max(round_up(g.nc, TA), round_up(g.nc, TC));
  const int nta = (g.nc + TA - 1) / TA, ntc = (g.nc + TC - 1) / TC, W = assemble_warps(g.nc, TA, TC), T = 32 * W;
  if (T > 256) return AMG_ERR_UNSUPPORTED;
  int sb = 8;  // sites per chunk: several CTAs per SM, so that one builds while others contract
  while (sb > 4 && (size_t)sb * 12 * ncp * sizeof(double2) > 40 * 1024) sb >>= 1;
  size_t words = (size_t)sb * 12 * ncp;
  for (int self = 0; self < 2; ++self) {  // the groups' tiles on their way to the first group
    const int tw = (Tiles{nta, ntc, TA, TC, g.ntv, self != 0}.count() + 31) / 32;
    words = std::max(words, (size_t)(std::max(1, W / tw) - 1) * TA * TC * tw * 32);
  }
  const size_t sm = words * sizeof(double2);
  AMG_CUDA_TRY(cudaFuncSetAttribute(assemble_kernel<TA, TC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  assemble_kernel<TA, TC><<<dim3((unsigned)g.Vc, 5), T, sm, st>>>(R, U, clov, part, g, m0, ncp, sb, only);
  AMG_LAUNCH_CHECK();
  return AMG_OK;
}

// The tile shape with the fewest FP64 instructions per row and sub-partition (2 Ntv = 16: 2 x 4, four groups of one
// warp; for blocks that the tensor cores leave also 40: 5 x 5, two groups of two warps, and 48: 3 x 6, four warps).
static amg_status launch_assemble(const Geom& g, const double2* R, const double2* U, const double2* clov, double2* part,
                                  double m0, const int* only, cudaStream_t st) {
  constexpr int shapes[][2] = {{5, 5}, {6, 4}, {4, 4}, {3, 6}, {2, 4}, {3, 2}, {2, 2}};
  int best = -1;
  double cost = 0;
  for (int k = 0; k < 7; ++k) {
    const int ta = shapes[k][0], tc = shapes[k][1], W = assemble_warps(g.nc, ta, tc);
    if (W > 8) continue;
    const int tw = (((g.nc + ta - 1) / ta) * ((g.nc + tc - 1) / tc) + 31) / 32;
    const double c = (double)(W / 4) * ta * tc / (W / tw);
    if (best < 0 || c < cost) {
      best = k;
      cost = c;
    }
  }
  switch (best) {
    case 0: return launch_assemble_tile<5, 5>(g, R, U, clov, part, m0, only, st);
    case 1: return launch_assemble_tile<6, 4>(g, R, U, clov, part, m0, only, st);
    case 2: return launch_assemble_tile<4, 4>(g, R, U, clov, part, m0, only, st);
    case 3: return launch_assemble_tile<3, 6>(g, R, U, clov, part, m0, only, st);
    case 4: return launch_assemble_tile<2, 4>(g, R, U, clov, part, m0, only, st);
    case 5: return launch_assemble_tile<3, 2>(g, R, U, clov, part, m0, only, st);
    case 6: return launch_assemble_tile<2, 2>(g, R, U, clov, part, m0, only, st);
    default: return AMG_ERR_UNSUPPORTED;
  }
}

// Whether the assembly runs on the tensor cores (setup_tc.cu).  That kernel has a fixed cost of about 10 us per block
// and job and grows slowly with Ntv; the tiled ones grow with Vb Ntv^2.  In FP64 the two meet near
// Vb Ntv^2 = 1800 (tiled / slices in ms, 10^4 sites: Vb 16, Ntv 8: 1.44 / 1.50, Ntv 11: 2.41 / 1.94; Vb 81, Ntv 4: 0.75 /
// 0.85, Ntv 6: 1.10 / 0.87; Vb 8, Ntv 12: 2.13 / 2.26, Ntv 16: 3.08 / 2.46).  In pairs of FP32 numbers the tiles are
// several times cheaper and good at Ntv 11 and below (Vb 54, Ntv 11: 1.05 / 1.16; Vb 81, Ntv 11: 1.07 / 1.00; Vb 16, Ntv 12:
// 1.36 / 1.90, Ntv 16: 2.15 / 2.10; Vb 8, Ntv 16: 1.84 / 2.39, Ntv 20: 3.12 / 2.97).
static bool assemble_by_slices(const Geom& g, bool pair) {
  const long long work = g.Vb * g.ntv * g.ntv;
  return pair ? g.Vb >= 64 || (g.ntv >= 16 && work >= 3200) : work >= 1800;
}

// The setup's steps; the caller owns the timing events and frees `part` if a step fails.  The Gram-Schmidt and the
// assembly run twice where a fixed-point kernel serves: that one marks the aggregates and (block, job)s whose numbers
// differ too widely for it, the floating-point kernel of the arithmetic takes these (none: its CTAs return at once).
static amg_status setup_body(amg_coarse* h, const double2* U, const double2* tv, cudaStream_t st, cudaEvent_t (&ev)[5],
                             double2*& part) {
  const Geom& g = h->g;
  AMG_CUDA_TRY(cudaEventRecord(ev[0], st));
  // clover
  {
    const int T = 128;
    const long long nb = (g.V + T - 1) / T;
    clover_kernel<<<(unsigned)nb, T, 0, st>>>(U, h->clover, g, h->p.csw);
    AMG_LAUNCH_CHECK();
  }
  AMG_CUDA_TRY(cudaEventRecord(ev[1], st));
  // Gram-Schmidt, one CTA per aggregate
  const bool pair = h->p.setup_arith == AMG_SETUP_F32PAIR;
  // what the fixed-point kernel leaves (all, where it does not serve) goes to the kernel of the arithmetic asked for; the
  // marks, 2 Vc ints, are kept where D_c will be
  int* left = (int*)h->Dc64;
  amg_status gs = amg_internal_gs_fixed(g, tv, h->R64, left, pair, h->err, st);
  if (gs == AMG_ERR_UNSUPPORTED) left = nullptr;
  else if (gs != AMG_OK) return gs;
  gs = pair ? amg_internal_gs_pair(g, tv, h->R64, left, h->err, st) : AMG_ERR_UNSUPPORTED;
  if (gs == AMG_ERR_UNSUPPORTED) {
    int T = round_up(g.nagg < 256 ? g.nagg : 256, 32);
    if ((g.nagg + T - 1) / T > GS_EMAX) return AMG_ERR_UNSUPPORTED;
    void (*const kernels[GS_EMAX])(const double2*, double2*, Geom, const int*, unsigned*) = {
        gs_kernel<1>, gs_kernel<2>, gs_kernel<3>, gs_kernel<4>, gs_kernel<5>, gs_kernel<6>, gs_kernel<7>, gs_kernel<8>};
    kernels[(g.nagg + T - 1) / T - 1]<<<(unsigned)(g.Vc * 2), T, 0, st>>>(tv, h->R64, g, left, h->err);
    AMG_LAUNCH_CHECK();
  } else if (gs != AMG_OK) {
    return gs;
  }
  AMG_CUDA_TRY(cudaEventRecord(ev[2], st));
  // assembly
  const bool slices = assemble_by_slices(g, pair);
  const size_t part_elems = (size_t)g.Vc * 5 * 2 * g.nc * g.nc, work = slices ? amg_internal_assemble_tc_ints(g) : 0;
  AMG_CUDA_TRY(cudaMallocAsync((void**)&part, part_elems * sizeof(double2) + work * sizeof(int), st));
  left = slices ? (int*)(part + part_elems) : nullptr;
  if (slices)
    AMG_TRY_INTERNAL(amg_internal_assemble_tc(g, h->R64, U, h->clover, left, part, h->p.m0, pair, h->err, st));
  if (pair)
    AMG_TRY_INTERNAL(amg_internal_assemble_pair(g, h->R64, U, h->clover, part, h->p.m0, left, h->err, st));
  else
    AMG_TRY_INTERNAL(launch_assemble(g, h->R64, U, h->clover, part, h->p.m0, left, st));
  {
    const long long total = g.Vc * 9LL * g.nc * g.nc;
    combine_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(part, h->nbr, h->Dc64, g);
    AMG_LAUNCH_CHECK();
  }
  AMG_CUDA_TRY(cudaEventRecord(ev[3], st));
  AMG_CUDA_TRY(cudaFreeAsync(part, st));
  part = nullptr;
  // storage precisions
  {
    const unsigned nblk = (unsigned)(g.Vc * 9);
    switch (h->p.link_prec) {
      case AMG_FP64: quantize_dc_kernel<0><<<nblk, 256, 0, st>>>(h->Dc64, h->Dq, nullptr, g.nc); break;
      case AMG_FP32: quantize_dc_kernel<1><<<nblk, 256, 0, st>>>(h->Dc64, h->Dq, nullptr, g.nc); break;
      case AMG_FP16_SCALED: quantize_dc_kernel<2><<<nblk, 256, 0, st>>>(h->Dc64, h->Dq, h->Dscale, g.nc); break;
      default: break;
    }
    AMG_LAUNCH_CHECK();
    if (h->p.r_prec == AMG_FP32) {
      const long long n = g.Vc * 2LL * g.ntv * g.nagg;
      r_to_fp32_kernel<<<1216, 256, 0, st>>>(h->R64, (float2*)h->Rq, n);
      AMG_LAUNCH_CHECK();
    }
    if (h->p.link_prec == AMG_BF16 || h->p.r_prec == AMG_BF16 ||
        ((h->p.link_prec == AMG_FP32 || h->p.link_prec == AMG_FP16_SCALED) && h->p.max_nrhs >= 4)) {
      amg_status s = amg_internal_tc_prepare(h, st);
      if (s != AMG_OK) return s;
    }
  }
  AMG_CUDA_TRY(cudaEventRecord(ev[4], st));
  AMG_CUDA_TRY(cudaEventSynchronize(ev[4]));
  for (int k = 0; k < 4; ++k) cudaEventElapsedTime(&h->setup_ms[k], ev[k], ev[k + 1]);
  unsigned e = 0;
  AMG_CUDA_TRY(cudaMemcpy(&e, h->err, sizeof(unsigned), cudaMemcpyDeviceToHost));
  if (e & AMG_EBIT_RANK) return AMG_ERR_RANK_DEFICIENT;
  if (e) {
    amg_note_cuda_error(__FILE__, __LINE__, cudaErrorUnknown);
    return AMG_ERR_CUDA;
  }
  return AMG_OK;
}

amg_status amg_internal_setup(amg_coarse* h, const double2* U, const double2* tv, cudaStream_t st) {
  cudaEvent_t ev[5] = {};
  double2* part = nullptr;
  amg_status s = AMG_OK;
  for (int k = 0; k < 5 && s == AMG_OK; ++k) {
    const cudaError_t c = cudaEventCreate(&ev[k]);
    if (c != cudaSuccess) {
      amg_note_cuda_error(__FILE__, __LINE__, c);
      ev[k] = nullptr;
      s = AMG_ERR_CUDA;
    }
  }
  if (s == AMG_OK) s = setup_body(h, U, tv, st, ev, part);
  if (part) cudaFreeAsync(part, st);  // a step failed between the allocation and its release
  for (int k = 0; k < 5; ++k)
    if (ev[k]) cudaEventDestroy(ev[k]);
  return s;
}
