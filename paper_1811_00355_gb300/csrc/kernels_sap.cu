// Schwarz alternating procedure (SAP) smoother, paper Sec. 2: a
// multiplicative Schwarz sweep over the blocks of one colour, the block
// system solved approximately by site even-odd preconditioned minimal
// residual with a fixed number of iterations.  Loops over blocks are the
// parallel dimension (Sec. 4); here one CTA owns one block.  Two kernels: the
// general one (any block shape, FP64 and FP32, one right-hand side per CTA,
// the block's links in shared memory), and the FP32 block kernel further down.
//
// Per CTA (block B of colour c):
//   r   = b - D x on the block's sites (full operator, neighbours from global
//         memory; r = b when x is known to be zero)
//   rhs = r_e - D_eo A_oo^-1 r_o                      (D_B restricted to B)
//   MR on S = A_ee - D_eo A_oo^-1 D_oe from e_e = 0:
//         p = S res; alpha = <p,res>/<p,p>; e_e += alpha res; res -= alpha p
//   e_o = A_oo^-1 (r_o - D_oe e_e)
//   x  += e
// with D_eo, D_oe the hops that stay inside the block (-1/2 (1 -+ g) U).
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "half.cuh"
#include "kernels.h"

namespace ddamg {

namespace {

// Four threads per site: thread sub = 0..3 of a site applies the two hops
// of direction mu = sub and owns the three colour components of spin sub of
// every site vector (res, e, p, ...).  Hop partial sums of the four threads
// are combined by a reduce-scatter of warp shuffles.

constexpr int LPAD = 2;   // padding of the staged link rows (bank groups)

template <class R>
using T16 = typename U16<R>::T;

// link mu of local site q from the staged block links (rows of Vb + LPAD units)
template <class R>
__device__ __forceinline__ void smem_link(const T16<R>* sl, int Vbp, int q, int mu, Link<R>& U) {
  using LY = Layout<R, GAUGE_NR>;
  constexpr int NUL = LINK_NR / LY::PER;
  R v[LINK_NR];
#pragma unroll
  for (int u = 0; u < NUL; ++u) {
    T16<R> t = sl[(mu * NUL + u) * Vbp + q];
    if constexpr (LY::PER == 4) {
      v[4 * u] = t.x; v[4 * u + 1] = t.y; v[4 * u + 2] = t.z; v[4 * u + 3] = t.w;
    } else {
      v[2 * u] = t.x; v[2 * u + 1] = t.y;
    }
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) U.m[k / 3][k % 3] = mk(v[2 * k], v[2 * k + 1]);
  complete_link(U);
}

template <class R>
__device__ __forceinline__ void smem_spinor(const cpx<R>* buf, int Vh, int h, Spinor<R>& s) {
#pragma unroll
  for (int k = 0; k < 12; ++k) s.c[k] = buf[k * Vh + h];
}

// one complex component k of site d in a global spinor field
template <class R>
__device__ __forceinline__ size_t comp_off(int d, int Vb, int k) {
  using LY = Layout<R, SPINOR_NR>;
  constexpr int CPU = LY::PER / 2;   // complex numbers per 16-byte unit
  int B = d / Vb, q = d - B * Vb;
  return (((size_t)B * LY::NU + k / CPU) * Vb + q) * LY::PER + (k % CPU) * 2;
}
__device__ __forceinline__ cpx<float> ld_comp(const float* f, size_t off) {
  float2 t = __ldcg(reinterpret_cast<const float2*>(f + off));
  return mk(t.x, t.y);
}
__device__ __forceinline__ cpx<double> ld_comp(const double* f, size_t off) {
  double2 t = __ldcg(reinterpret_cast<const double2*>(f + off));
  return mk(t.x, t.y);
}
__device__ __forceinline__ void st_comp(float* f, size_t off, cpx<float> v) {
  *reinterpret_cast<float2*>(f + off) = make_float2(v.re, v.im);
}
__device__ __forceinline__ void st_comp(double* f, size_t off, cpx<double> v) {
  *reinterpret_cast<double2*>(f + off) = make_double2(v.re, v.im);
}

template <class R>
__device__ __forceinline__ cpx<R> shfl_x(cpx<R> v, int m) {
  return mk(__shfl_xor_sync(0xffffffffu, v.re, m), __shfl_xor_sync(0xffffffffu, v.im, m));
}

// reduce-scatter of a 12-component partial sum over the 4 threads of a site:
// thread sub receives the full sum of components 3 sub .. 3 sub + 2
template <class R>
__device__ __forceinline__ void reduce_scatter(const Spinor<R>& acc, int sub, cpx<R> out[3]) {
  const bool hi = sub >= 2;      // chirality block of this thread
  cpx<R> keep[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    cpx<R> send = hi ? acc.c[i] : acc.c[6 + i];
    keep[i] = (hi ? acc.c[6 + i] : acc.c[i]) + shfl_x(send, 2);
  }
  const bool odd = sub & 1;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cpx<R> send = odd ? keep[i] : keep[3 + i];
    out[i] = (odd ? keep[3 + i] : keep[i]) + shfl_x(send, 1);
  }
}

// the 6 components of this thread's chirality block: own 3 + partner's 3
template <class R>
__device__ __forceinline__ void chiral6(const cpx<R> own[3], int sub, cpx<R> v6[6]) {
  const bool odd = sub & 1;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cpx<R> other = shfl_x(own[i], 1);
    v6[i] = odd ? other : own[i];
    v6[3 + i] = odd ? own[i] : other;
  }
}

// own 3 rows of the packed Hermitian block (chirality sub / 2) times v6
template <class R>
__device__ __forceinline__ void clover_rows(const R* __restrict__ clov, int d, int Vb, int sub,
                                            const cpx<R> v6[6], cpx<R> y[3]) {
  using LY = Layout<R, CLOVER_NR>;
  constexpr int NUB = 36 / LY::PER;
  R P[36];
  load_units<R, CLOVER_NR>(clov, d, Vb, (sub >> 1) * NUB, NUB, P);
  cpx<R> y6[6];
  herm6<R>(P, v6, y6);
  const bool odd = sub & 1;
#pragma unroll
  for (int i = 0; i < 3; ++i) y[i] = odd ? y6[3 + i] : y6[i];
}

// Runtime direction: with g_mu = [[0, B], [B^H, 0]] every B_mu has one
// non-zero per row, B[r][pi(r)] = c_r with pi the identity (z, t) or the
// swap (x, y) and c_r in {+-1, +-i}.  Writing the projector this way keeps
// the four threads of a site (four directions) in one instruction stream.
// A factor c in {+-1, +-i} is held as (rot, a): c = a when rot is false and
// c = -i a when it is true, so c t = rot ? (a t.im, -a t.re) : (a t.re, a t.im)
// costs two selects and no multiplications.
template <class R>
struct Dir {
  bool swp;          // pi swaps the spin pairs
  bool rot0, rot1;   // c_0, c_1 imaginary
  R a0, a1;
};
template <class R>
__device__ __forceinline__ Dir<R> make_dir(int mu) {
  Dir<R> d;
  d.swp = mu < 2;
  d.rot0 = d.rot1 = (mu == 0 || mu == 2);
  d.a0 = (mu == 1) ? R(-1) : R(1);      // c_0: -i, -1, -i, 1
  d.a1 = (mu == 2) ? R(-1) : R(1);      // c_1: -i,  1,  i, 1
  return d;
}
// acc += s c t for c = (rot, a) and a real scale s (sa = s a)
template <class R>
__device__ __forceinline__ void add_ct(cpx<R>& acc, bool rot, R sa, cpx<R> t) {
  const R u = rot ? t.im : t.re, v = rot ? t.re : t.im;
  const R sb = rot ? -sa : sa;
  acc.re += sa * u;
  acc.im += sb * v;
}
// h_r = s_r + sigma c_r s_{2 + pi(r)}
template <class R>
__device__ __forceinline__ void project_rt(const Spinor<R>& p, const Dir<R>& dr, R sigma, cpx<R> h[2][3]) {
  const R s0 = sigma * dr.a0, s1 = sigma * dr.a1;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cpx<R> s2 = p.c[6 + a], s3 = p.c[9 + a];
    cpx<R> t0 = dr.swp ? s3 : s2, t1 = dr.swp ? s2 : s3;
    h[0][a] = p.c[a];
    h[1][a] = p.c[3 + a];
    add_ct(h[0][a], dr.rot0, s0, t0);
    add_ct(h[1][a], dr.rot1, s1, t1);
  }
}
// acc += sc [y; sigma B^H y],  (B^H y)_r = conj(c_pi(r)) y_pi(r); the
// conjugate of (rot, a) is (rot, -a) when rot is true
template <class R>
__device__ __forceinline__ void accumulate_rt(Spinor<R>& acc, const cpx<R> y[2][3], const Dir<R>& dr,
                                              R sigma, R sc) {
  const bool r2 = dr.swp ? dr.rot1 : dr.rot0, r3 = dr.swp ? dr.rot0 : dr.rot1;
  R a2 = dr.swp ? dr.a1 : dr.a0, a3 = dr.swp ? dr.a0 : dr.a1;
  if (r2) a2 = -a2;
  if (r3) a3 = -a3;
  const R s2 = sigma * sc * a2, s3 = sigma * sc * a3;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const cpx<R> y0 = y[0][a], y1 = y[1][a];
    acc.c[a].re += sc * y0.re;
    acc.c[a].im += sc * y0.im;
    acc.c[3 + a].re += sc * y1.re;
    acc.c[3 + a].im += sc * y1.im;
    add_ct(acc.c[6 + a], r2, s2, dr.swp ? y1 : y0);
    add_ct(acc.c[9 + a], r3, s3, dr.swp ? y0 : y1);
  }
}

// own 3 components of the sum of the block-internal hops at local site q;
// this thread applies the two hops of direction mu = sub
template <class R>
__device__ __forceinline__ void hop_block(const int16_t* __restrict__ bnbr, const T16<R>* sl,
                                          const cpx<R>* buf, int Vb, int Vbp, int Vh, int q, int sub,
                                          cpx<R> out[3]) {
  Spinor<R> acc;
#pragma unroll
  for (int k = 0; k < 12; ++k) acc.c[k] = mk(R(0), R(0));
  const Dir<R> dr = make_dir<R>(sub);
  cpx<R> hh[2][3], y[2][3];
  Spinor<R> nb;
  int qf = __ldg(bnbr + (2 * sub) * Vb + q);
  if (qf >= 0) {   // (1 - g_mu) U_mu(x) x(x + mu)
    smem_spinor<R>(buf, Vh, qf >= Vh ? qf - Vh : qf, nb);
    project_rt<R>(nb, dr, R(-1), hh);
    Link<R> U;
    smem_link<R>(sl, Vbp, q, sub, U);
    su3_mul(U, hh, y);
    accumulate_rt<R>(acc, y, dr, R(-1), R(1));
  }
  int qb = __ldg(bnbr + (2 * sub + 1) * Vb + q);
  if (qb >= 0) {   // (1 + g_mu) U_mu(x - mu)^H x(x - mu)
    smem_spinor<R>(buf, Vh, qb >= Vh ? qb - Vh : qb, nb);
    project_rt<R>(nb, dr, R(1), hh);
    Link<R> U;
    smem_link<R>(sl, Vbp, qb, sub, U);
    su3_mul_dag(U, hh, y);
    accumulate_rt<R>(acc, y, dr, R(1), R(1));
  }
  reduce_scatter<R>(acc, sub, out);
}

// own 3 components of the full (global) hopping sum at device site d
template <class R>
__device__ __forceinline__ void hop_global(const Geom& g, const R* x, const R* gauge, int d, int sub,
                                           cpx<R> out[3]) {
  Spinor<R> acc;
#pragma unroll
  for (int k = 0; k < 12; ++k) acc.c[k] = mk(R(0), R(0));
  const Dir<R> dr = make_dir<R>(sub);
  cpx<R> hh[2][3], y[2][3];
  Spinor<R> nb;
  {
    uint32_t e = __ldg(g.nbr + (size_t)(2 * sub) * g.V + d);
    int n = (int)(e & ~NEG_BIT);
    load_spinor_cg<R>(x, n, g.Vb, nb);
    project_rt<R>(nb, dr, R(-1), hh);
    Link<R> U;
    load_link<R>(gauge, d, g.Vb, sub, U);
    su3_mul(U, hh, y);
    accumulate_rt<R>(acc, y, dr, R(-1), (e & NEG_BIT) ? R(-1) : R(1));
  }
  {
    uint32_t e = __ldg(g.nbr + (size_t)(2 * sub + 1) * g.V + d);
    int n = (int)(e & ~NEG_BIT);
    load_spinor_cg<R>(x, n, g.Vb, nb);
    project_rt<R>(nb, dr, R(1), hh);
    Link<R> U;
    load_link<R>(gauge, n, g.Vb, sub, U);
    su3_mul_dag(U, hh, y);
    accumulate_rt<R>(acc, y, dr, R(1), (e & NEG_BIT) ? R(-1) : R(1));
  }
  reduce_scatter<R>(acc, sub, out);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <class R>
__device__ __forceinline__ R warp_sum_r(R v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// block sum of three per-thread partials in the working precision (warp
// trees, then one warp over the per-warp sums), broadcast to every thread
template <class R>
__device__ __forceinline__ void block_sum3(R ra, R rb, R rc, R& a, R& b, R& c, R* sh) {
  ra = warp_sum_r<R>(ra);
  rb = warp_sum_r<R>(rb);
  rc = warp_sum_r<R>(rc);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int nw = blockDim.x >> 5;
  if (l == 0) { sh[3 * w] = ra; sh[3 * w + 1] = rb; sh[3 * w + 2] = rc; }
  __syncthreads();
  if (w == 0) {
    R x = l < nw ? sh[3 * l] : R(0), y = l < nw ? sh[3 * l + 1] : R(0), z = l < nw ? sh[3 * l + 2] : R(0);
    x = warp_sum_r<R>(x);
    y = warp_sum_r<R>(y);
    z = warp_sum_r<R>(z);
    if (l == 0) { sh[96] = x; sh[97] = y; sh[98] = z; }
  }
  __syncthreads();
  a = sh[96];
  b = sh[97];
  c = sh[98];
}

// block index of the k-th block of colour c (block-grid extent 0 even)
__device__ __forceinline__ int block_of_colour(const Geom& g, int c, int k) {
  int t = 2 * k;
  int b0 = t % g.grid[0];
  int r = t / g.grid[0];
  int b1 = r % g.grid[1];
  r /= g.grid[1];
  int b2 = r % g.grid[2];
  int b3 = r / g.grid[2];
  b0 += (c + b1 + b2 + b3) & 1;
  return b0 + g.grid[0] * (b1 + g.grid[1] * (b2 + g.grid[2] * b3));
}

template <class R>
__global__ void __launch_bounds__(512) k_sap_sweep(Geom g, int colour, int mr_iters, int x_is_zero,
                                                   const R* __restrict__ b, R* __restrict__ x,
                                                   const R* __restrict__ gauge, const R* __restrict__ clov,
                                                   const R* __restrict__ clov_inv) {
  using LYG = Layout<R, GAUGE_NR>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int Vb = g.Vb, Vh = Vb / 2, Vbp = Vb + LPAD;
  T16<R>* sl = reinterpret_cast<T16<R>*>(smem_raw);                      // [NU][Vb + LPAD]
  cpx<R>* E = reinterpret_cast<cpx<R>*>(sl + (size_t)LYG::NU * Vbp);      // [12][Vh]
  cpx<R>* O = E + 12 * Vh;                                                // [12][Vh]
  R* red = reinterpret_cast<R*>(O + 12 * Vh);                             // [3 * warps + 3]

  const int B = block_of_colour(g, colour, blockIdx.x);
  const size_t off = (size_t)blockIdx.y * g.V * SPINOR_NR;
  b += off;
  x += off;
  const int h = threadIdx.x >> 2, sub = threadIdx.x & 3;
  const bool act = h < Vh;
  const int hs = act ? h : 0;                 // inactive lanes shadow site 0 (no stores)
  const int de = B * Vb + hs, dO = B * Vb + Vh + hs;

  // stage the block's links (contiguous in the block-major layout)
  {
    // (two rows of each link; FP64 links have a third one in between)
    constexpr int NUL = LYG::NU / 4, NULG = sizeof(R) == 8 ? LINK64_NR / 2 : NUL;
    const T16<R>* src = reinterpret_cast<const T16<R>*>(gauge) + (size_t)B * 4 * NULG * Vb;
    for (int i = threadIdx.x; i < LYG::NU * Vb; i += blockDim.x) {
      int u = i / Vb, q = i - u * Vb;
      sl[u * Vbp + q] = __ldg(src + (size_t)((u / NUL) * NULG + u % NUL) * Vb + q);
    }
  }

  // residual r = b - D x on the own components of both sites
  cpx<R> re[3], ro[3];
  {
#pragma unroll
    for (int par = 0; par < 2; ++par) {
      const int d = par ? dO : de;
      cpx<R> r[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) r[i] = ld_comp(b, comp_off<R>(d, Vb, 3 * sub + i));
      if (!x_is_zero) {
        cpx<R> hop[3], x6[6], ax[3];
        hop_global<R>(g, x, gauge, d, sub, hop);
        const int c0 = 6 * (sub >> 1);
#pragma unroll
        for (int i = 0; i < 6; ++i) x6[i] = ld_comp(x, comp_off<R>(d, Vb, c0 + i));
        clover_rows<R>(clov, d, Vb, sub, x6, ax);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          r[i].re -= ax[i].re - R(0.5) * hop[i].re;
          r[i].im -= ax[i].im - R(0.5) * hop[i].im;
        }
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (par) ro[i] = r[i];
        else re[i] = r[i];
      }
    }
    // u_o = A_oo^-1 r_o
    cpx<R> v6[6], u[3];
    chiral6<R>(ro, sub, v6);
    clover_rows<R>(clov_inv, dO, Vb, sub, v6, u);
    if (act)
#pragma unroll
      for (int i = 0; i < 3; ++i) O[(3 * sub + i) * Vh + h] = u[i];
  }
  __syncthreads();

  // rhs_e = r_e - D_eo u_o = r_e + 1/2 hop(u_o)
  cpx<R> res[3], xe[3];
  {
    cpx<R> t[3];
    hop_block<R>(g.bnbr, sl, O, Vb, Vbp, Vh, hs, sub, t);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      res[i].re = fma_r(R(0.5), t[i].re, re[i].re);
      res[i].im = fma_r(R(0.5), t[i].im, re[i].im);
      xe[i] = mk(R(0), R(0));
    }
  }

  for (int it = 0; it < mr_iters; ++it) {
    __syncthreads();       // readers of E / O from the previous step are done
    if (act)
#pragma unroll
      for (int i = 0; i < 3; ++i) E[(3 * sub + i) * Vh + h] = res[i];
    __syncthreads();
    {  // odd: w = A_oo^-1 D_oe res = A_oo^-1 (-1/2 hop(res))
      cpx<R> t[3], v6[6], w[3];
      hop_block<R>(g.bnbr, sl, E, Vb, Vbp, Vh, Vh + hs, sub, t);
#pragma unroll
      for (int i = 0; i < 3; ++i) t[i] = R(-0.5) * t[i];
      chiral6<R>(t, sub, v6);
      clover_rows<R>(clov_inv, dO, Vb, sub, v6, w);
      if (act)
#pragma unroll
        for (int i = 0; i < 3; ++i) O[(3 * sub + i) * Vh + h] = w[i];
    }
    __syncthreads();
    R pr_re = 0, pr_im = 0, pp_r = 0;
    cpx<R> p[3];
    {  // even: p = A_ee res - D_eo w = A_ee res + 1/2 hop(w)
      cpx<R> t[3], v6[6];
      chiral6<R>(res, sub, v6);
      clover_rows<R>(clov, de, Vb, sub, v6, p);
      hop_block<R>(g.bnbr, sl, O, Vb, Vbp, Vh, hs, sub, t);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        p[i].re = fma_r(R(0.5), t[i].re, p[i].re);
        p[i].im = fma_r(R(0.5), t[i].im, p[i].im);
        if (act) {
          pr_re += p[i].re * res[i].re + p[i].im * res[i].im;
          pr_im += p[i].re * res[i].im - p[i].im * res[i].re;
          pp_r += p[i].re * p[i].re + p[i].im * p[i].im;
        }
      }
    }
    R dpr_re, dpr_im, pp;
    block_sum3<R>(pr_re, pr_im, pp_r, dpr_re, dpr_im, pp, red);
    if (pp > R(0)) {
      cpx<R> a = mk(dpr_re / pp, dpr_im / pp);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        fma(xe[i], a, res[i]);
        res[i] = res[i] - a * p[i];
      }
    }
  }

  // e_o = A_oo^-1 (r_o - D_oe e_e) = A_oo^-1 (r_o + 1/2 hop(e_e))
  __syncthreads();
  if (act)
#pragma unroll
    for (int i = 0; i < 3; ++i) E[(3 * sub + i) * Vh + h] = xe[i];
  __syncthreads();
  cpx<R> eo[3];
  {
    cpx<R> t[3], v6[6];
    hop_block<R>(g.bnbr, sl, E, Vb, Vbp, Vh, Vh + hs, sub, t);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      t[i].re = fma_r(R(0.5), t[i].re, ro[i].re);
      t[i].im = fma_r(R(0.5), t[i].im, ro[i].im);
    }
    chiral6<R>(t, sub, v6);
    clover_rows<R>(clov_inv, dO, Vb, sub, v6, eo);
  }
  if (act) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      size_t oe = comp_off<R>(de, Vb, 3 * sub + i), oo = comp_off<R>(dO, Vb, 3 * sub + i);
      cpx<R> ve = xe[i], vo = eo[i];
      if (!x_is_zero) {
        ve = ve + ld_comp(x, oe);
        vo = vo + ld_comp(x, oo);
      }
      st_comp(x, oe, ve);
      st_comp(x, oo, vo);
    }
  }
}

// ---------------------------------------------------------------------------
// Block kernel (FP32 arithmetic) for Schwarz blocks of 64, 128, 192 or 256
// sites: a thread per site, the site's links and its clover block (A_ee on an
// even site, A_oo^-1 on an odd one) in registers for the whole launch.
//
// What bounds it: instruction issue and latency of few warps.  The block
// solve has about 3 MFLOP but 36 half-spinor exchanges with barriers between
// them; a block's operators (120 KB) come from L2 or DRAM once per launch.
// The form before (four threads per site, operators read from shared memory
// at every hop, the residual b - D x recomputed from global memory in every
// sweep) spent 640 instructions per thread and hop phase on selects, shuffles
// and shared-memory reads: 34 us per sweep of one right-hand side on 16^4,
// 35 us per block solve on 24^3 x 48.  This one: 21 us and 17.6 us.
//  * A thread multiplies only with its own four links: forward hops as the
//    receiver, backward ones as the sender, so a link is held once and both
//    parities work at the same time (half steps below).
//  * Hops leaving the block read a place of zeros instead of branching.
//  * The residual is carried: after a block solve it is zero on the odd sites
//    and the MR residual on the even ones, and only hops across block faces
//    change it until the block's next sweep.  Every sweep leaves those hops as
//    half spinors (msg) for the other colour, a quarter of the hops of a 4^4
//    block and no clover product.  (Error of the smoother against 64 bits on
//    the lattices above 1.8e-7, with recomputed residuals 1.5e-7.)
//  * What the next right-hand side needs arrives by bulk copies while this one
//    is solved.
//  * The loop's parts exist once each, or the code would not stay in the
//    instruction cache: with every use inlined the same algorithm took 26 us.
// Two threads per site (two links and one chirality each, 512 threads) were
// slower, 24 us: twice the shared-memory traffic, and registers spilled.
// ---------------------------------------------------------------------------
namespace blk {

using f2 = cpx<float>;

struct SapArgs {
  Geom g;
  int colour, mr_iters, nrhs, per;   // right-hand sides of the call and per CTA
  int first, take, give, keep;
  const float* b;
  float* x;
  float4* res;
  float4* msg;
  const void* gauge;
  const void* clov;
  const void* clov_inv;
  int* status;
  long long wait_limit;
};

// staged operator units of site q (half h) -> links (halved) and clover block
template <class S>
struct Ops;
template <>
struct Ops<float> {
  using T = float4;
  static constexpr int LU = 12, CU = 18;
  __device__ __forceinline__ static void links(const T* sl, int Vb, int q, Link<float> (&U)[4]) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const float4 a = sl[(3 * m) * Vb + q], b = sl[(3 * m + 1) * Vb + q], c = sl[(3 * m + 2) * Vb + q];
      U[m].m[0][0] = mk(a.x, a.y); U[m].m[0][1] = mk(a.z, a.w); U[m].m[0][2] = mk(b.x, b.y);
      U[m].m[1][0] = mk(b.z, b.w); U[m].m[1][1] = mk(c.x, c.y); U[m].m[1][2] = mk(c.z, c.w);
    }
  }
  __device__ __forceinline__ static void clover(const T* A, int Vh, int h, float (&P)[72]) {
#pragma unroll
    for (int u = 0; u < 18; ++u) {
      const float4 a = A[u * Vh + h];
      P[4 * u] = a.x; P[4 * u + 1] = a.y; P[4 * u + 2] = a.z; P[4 * u + 3] = a.w;
    }
  }
};
template <class S>
struct OpsHalf {
  using T = uint4;
  static constexpr int LU = HGAUGE_NU, CU = HCLOV_NU;
  __device__ __forceinline__ static void links(const T* sl, int Vb, int q, Link<float> (&U)[4]) {
    float v[48];
#pragma unroll
    for (int u = 0; u < 6; ++u) unpack8<S>(sl[u * Vb + q], v + 8 * u);
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int k = 0; k < 6; ++k) U[m].m[k / 3][k % 3] = mk(v[12 * m + 2 * k], v[12 * m + 2 * k + 1]);
  }
  __device__ __forceinline__ static void clover(const T* A, int Vh, int h, float (&P)[72]) {
#pragma unroll
    for (int u = 0; u < 9; ++u) unpack8<S>(A[u * Vh + h], P + 8 * u);
  }
};
template <>
struct Ops<__half> : OpsHalf<__half> {};
template <>
struct Ops<__nv_bfloat16> : OpsHalf<__nv_bfloat16> {};

__device__ __forceinline__ void put_half(float4* p, int stride, const f2 (&h)[2][3]) {
  p[0] = make_float4(h[0][0].re, h[0][0].im, h[0][1].re, h[0][1].im);
  p[stride] = make_float4(h[0][2].re, h[0][2].im, h[1][0].re, h[1][0].im);
  p[2 * stride] = make_float4(h[1][1].re, h[1][1].im, h[1][2].re, h[1][2].im);
}
__device__ __forceinline__ void as_half(const float4& a, const float4& b, const float4& c, f2 (&h)[2][3]) {
  h[0][0] = mk(a.x, a.y); h[0][1] = mk(a.z, a.w); h[0][2] = mk(b.x, b.y);
  h[1][0] = mk(b.z, b.w); h[1][1] = mk(c.x, c.y); h[1][2] = mk(c.z, c.w);
}
__device__ __forceinline__ void get_half(const float4* p, int stride, f2 (&h)[2][3]) {
  as_half(p[0], p[stride], p[2 * stride], h);
}

// U^H (1 + g_MU) psi for the site ahead, one direction after the other
template <int MU>
__device__ __forceinline__ void ahead_dir(const Spinor<float>& psi, const Link<float>& U, float4* gx, int row, int h) {
  f2 hh[2][3], y[2][3];
  project<MU, +1>(psi, hh);
  su3_mul_dag(U, hh, y);
  put_half(gx + (size_t)(3 * MU) * row + h, row, y);
}
__device__ __forceinline__ void send_ahead(const Spinor<float>& psi, const Link<float> (&U)[4], float4* gx, int row, int h) {
  ahead_dir<0>(psi, U[0], gx, row, h);
  ahead_dir<1>(psi, U[1], gx, row, h);
  ahead_dir<2>(psi, U[2], gx, row, h);
  ahead_dir<3>(psi, U[3], gx, row, h);
}
// acc += (1 - g_MU) U psi(ahead) from the published spinors (n: the
// neighbours' places); a direction's spinor is loaded while the one before is
// multiplied
__device__ __forceinline__ void load6(const float4* p, int stride, Spinor<float>& s) {
#pragma unroll
  for (int u = 0; u < 6; ++u) {
    const float4 a = p[u * stride];
    s.c[2 * u] = mk(a.x, a.y);
    s.c[2 * u + 1] = mk(a.z, a.w);
  }
}
template <int MU>
__device__ __forceinline__ void fwd_dir(Spinor<float>& acc, const Link<float>& U, const Spinor<float>& nb) {
  f2 hh[2][3], y[2][3];
  project<MU, -1>(nb, hh);
  su3_mul(U, hh, y);
  accumulate<MU, -1>(acc, y, 1.f);
}
__device__ __forceinline__ void take_ahead(Spinor<float>& acc, const Link<float> (&U)[4], const float4* pub, int row,
                                           unsigned n0, unsigned n1) {
  Spinor<float> p, q;
  load6(pub + (n0 & 255u), row, p);
  load6(pub + ((n0 >> 16) & 255u), row, q);
  fwd_dir<0>(acc, U[0], p);
  load6(pub + (n1 & 255u), row, p);
  fwd_dir<1>(acc, U[1], q);
  load6(pub + ((n1 >> 16) & 255u), row, q);
  fwd_dir<2>(acc, U[2], p);
  fwd_dir<3>(acc, U[3], q);
}
// acc += the half spinors that the sites behind sent ahead
template <int MU>
__device__ __forceinline__ void bwd_dir(Spinor<float>& acc, const float4* gx, int row, unsigned n) {
  f2 hh[2][3];
  get_half(gx + (size_t)(3 * MU) * row + n, row, hh);
  accumulate<MU, +1>(acc, hh, 1.f);
}
__device__ __forceinline__ void take_behind(Spinor<float>& acc, const float4* gx, int row, unsigned n0, unsigned n1) {
  bwd_dir<0>(acc, gx, row, (n0 >> 8) & 255u);
  bwd_dir<1>(acc, gx, row, n0 >> 24);
  bwd_dir<2>(acc, gx, row, (n1 >> 8) & 255u);
  bwd_dir<3>(acc, gx, row, n1 >> 24);
}

__device__ __forceinline__ void clover12(const float (&P)[72], const Spinor<float>& v, Spinor<float>& y) {
  herm6<float>(P, v.c, y.c);
  herm6<float>(P + 36, v.c + 6, y.c + 6);
}

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }


// the hops of direction MU from the neighbouring blocks: their messages, the
// lower face of the block ahead and the upper face of the block behind (sites
// inside the block take zeros)
template <int MU>
__device__ __forceinline__ void outer_dir(Spinor<float>& r, const Link<float>& U, const float4* m, const float4* zero,
                                          bool lower, bool upper, int F, float sf, float sb) {
  f2 hh[2][3], y[2][3], bb[2][3];
  const float4 *pf = upper ? m : zero, *pb = lower ? m + 3 * F : zero;
  get_half(pf, upper ? F : 0, hh);
  get_half(pb, lower ? F : 0, bb);
  su3_mul(U, hh, y);
  accumulate<MU, -1>(r, y, MU == 3 ? sf : 1.f);
  accumulate<MU, +1>(r, bb, MU == 3 ? sb : 1.f);
}
// and what this site sends them
template <int MU>
__device__ __forceinline__ void give_dir(const Spinor<float>& v, const Link<float>& U, float4* m, bool lower, bool upper,
                                         int F) {
  f2 hh[2][3], y[2][3];
  if (lower) {
    project<MU, -1>(v, hh);
    put_half(m, F, hh);
  }
  if (upper) {
    project<MU, +1>(v, hh);
    su3_mul_dag(U, hh, y);
    put_half(m + 3 * F, F, y);
  }
}

// float4 units of a block's messages: three per site of each face
__host__ __device__ __forceinline__ int msg_units(const Geom& g) {
  return 6 * (g.Vb / g.b[0] + g.Vb / g.b[1] + g.Vb / g.b[2] + g.Vb / g.b[3]);
}

// VB: the block's sites (constant strides take 10 % off the solve)
template <class S, int VB>
__global__ void __launch_bounds__(VB, 256 / VB) k_sap_block(SapArgs a) {
  using T = typename Ops<S>::T;
  constexpr int LU = Ops<S>::LU, CU = Ops<S>::CU;
  constexpr unsigned UB = sizeof(T);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Geom& g = a.g;
  constexpr int Vb = VB, Vh = Vb / 2, row = Vh + 1;
  const int S3 = msg_units(g);
  float4* pub = reinterpret_cast<float4*>(smem_raw);       // [parity][6][Vh + 1] published spinors
  float4* gx = pub + 12 * row;                             // [parity][12][Vh + 1] sent ahead
  float4* red = gx + 24 * row;                             // [warps of one parity]
  float4* area = red + Vh / 32;                            // staged operators, then:
  float4* kp = area;                                       // [6][Vb] kept -r_o / e_e
  float4* base = kp + 6 * Vb;                              // [6][Vb] b, or [6][Vh] the even residual
  float4* xs = base + 6 * Vb;                              // [6][Vb] x
  float4* ms = xs + 6 * Vb;                                // [S3] the neighbours' messages
  T* sl = reinterpret_cast<T*>(area);                      // [LU][Vb]
  T* Aee = sl + LU * Vb;                                   // [CU][Vh]
  T* Aoi = Aee + CU * Vh;                                  // [CU][Vh]

  const int t = threadIdx.x;
  const bool odd = t >= Vh;
  const int h = odd ? t - Vh : t;
  const int slices = gridDim.x / (g.nb / 2);
  const int B = block_of_colour(g, a.colour, blockIdx.x / slices);
  const int rhs0 = (blockIdx.x % slices) * a.per, rhs1 = min(a.nrhs, rhs0 + a.per);

  __shared__ __align__(8) uint64_t bar_ops, bar_in, bar_x;
  __shared__ float2 alpha;                                 // the last MR step's
  if (t < 32) {
    if (t == 0) {
      mbar_init(&bar_ops, 1);
      mbar_init(&bar_in, 1);
      mbar_init(&bar_x, 1);
      mbar_fence_init();
    }
    __syncwarp();
    const unsigned links = (unsigned)(LU * Vb) * UB, half = (unsigned)Vh * UB;
    if (t == 0) {
      mbar_expect_tx(&bar_ops, links + 2u * CU * half);
      bulk_g2s(sl, reinterpret_cast<const T*>(a.gauge) + (size_t)B * LU * Vb, links, &bar_ops);
    }
    const T* ca = reinterpret_cast<const T*>(a.clov) + (size_t)B * CU * Vb;
    const T* ci = reinterpret_cast<const T*>(a.clov_inv) + (size_t)B * CU * Vb + Vh;
    for (int u = t; u < 2 * CU; u += 32) {
      if (u < CU) bulk_g2s(Aee + u * Vh, ca + (size_t)u * Vb, half, &bar_ops);
      else bulk_g2s(Aoi + (u - CU) * Vh, ci + (size_t)(u - CU) * Vb, half, &bar_ops);
    }
  }
  // the place past the last one stands for a neighbour outside the block
  if (t < 36) pub[t * row + Vh] = make_float4(0.f, 0.f, 0.f, 0.f);
  launch_dependents();
  // places of the eight block-internal neighbours among the other parity's sites
  unsigned n0 = 0, n1 = 0;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    int f = __ldg(g.bnbr + (2 * m) * Vb + t), b = __ldg(g.bnbr + (2 * m + 1) * Vb + t);
    f = f < 0 ? Vh : (f >= Vh ? f - Vh : f);
    b = b < 0 ? Vh : (b >= Vh ? b - Vh : b);
    const unsigned w = (unsigned)f | ((unsigned)b << 8);
    if (m < 2) n0 |= w << (16 * m);
    else n1 |= w << (16 * (m - 2));
  }
  auto outside = [&](unsigned n, int sh) { return ((n >> sh) & 255u) == (unsigned)Vh; };
  // this site's place among the messages of a face, by direction
  int pos[4];
  const int F0 = Vb / g.b[0], F1 = Vb / g.b[1], F2 = Vb / g.b[2], F3 = Vb / g.b[3];
  {
    int l[4], r = h;
    l[0] = 2 * (r % (g.b[0] / 2)); r /= g.b[0] / 2;
    l[1] = r % g.b[1]; r /= g.b[1];
    l[2] = r % g.b[2]; l[3] = r / g.b[2];
    l[0] += ((odd ? 1 : 0) + l[1] + l[2] + l[3]) & 1;
    pos[0] = l[1] + g.b[1] * (l[2] + g.b[2] * l[3]);
    pos[1] = 6 * F0 + l[0] + g.b[0] * (l[2] + g.b[2] * l[3]);
    pos[2] = 6 * (F0 + F1) + l[0] + g.b[0] * (l[1] + g.b[1] * l[3]);
    pos[3] = 6 * (F0 + F1 + F2) + l[0] + g.b[0] * (l[1] + g.b[1] * l[2]);
  }
  // b or the even residual (lane 8) and the messages (lanes 0 .. 7, a face each)
  const int face = t & 7, fF = Vb / g.b[face >> 1];
  int foff = 3 * fF * (face & 1);
  for (int m = 0; m < (face >> 1); ++m) foff += 6 * (Vb / g.b[m]);
  const int fY = __ldg(g.cnbr + (1 + face) * g.nb + B);
  // sign of the hops across the time boundary (t runs slowest over the blocks)
  const float sf = __ldg(g.cnbr + 7 * g.nb + B) < B ? -1.f : 1.f, sb = __ldg(g.cnbr + 8 * g.nb + B) > B ? -1.f : 1.f;
  __syncthreads();
  // false when a copy did not land in time: the status is set and every copy
  // in flight has been waited for
  auto landed = [&](uint64_t* bar, unsigned phase, int in_phase, int x_phase) -> bool {
    const bool ok = mbar_wait_bounded(bar, phase, a.wait_limit);
    if (!__syncthreads_or(!ok)) return true;
    if (t == 0) atomicExch(a.status, 6);
    mbar_wait_bounded(&bar_ops, 0, MBAR_POLL_LIMIT);
    if (in_phase >= 0) mbar_wait_bounded(&bar_in, in_phase & 1, MBAR_POLL_LIMIT);
    if (x_phase >= 0) mbar_wait_bounded(&bar_x, x_phase & 1, MBAR_POLL_LIMIT);
    return false;
  };
  if (!landed(&bar_ops, 0, -1, -1)) {
    // not before the sweep before: the next one waits for this grid only
    grid_dependency_wait();
    return;
  }
  Link<float> U[4];
  float P[72];
  Ops<S>::links(sl, Vb, t, U);
  Ops<S>::clover(odd ? Aoi : Aee, Vh, h, P);
  if (odd)
#pragma unroll
    for (int k = 0; k < 72; ++k) P[k] = -P[k];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    complete_link(U[m]);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) U[m].m[i][j] = 0.5f * U[m].m[i][j];
  }
  __syncthreads();       // the staged operators are in registers: their place is free
  grid_dependency_wait();

  auto fetch_in = [&](int rhs) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (t == 8) {
      const size_t blk = (size_t)rhs * g.nb + B;
      const unsigned nb = (unsigned)(a.first ? 6 * Vb : 6 * Vh) * 16u;
      mbar_expect_tx(&bar_in, nb + (a.take ? (unsigned)S3 * 16u : 0u));
      bulk_g2s(base, a.first ? reinterpret_cast<const float4*>(a.b) + blk * 6 * Vb : a.res + blk * 6 * Vh, nb, &bar_in);
    } else if (a.take) {
      bulk_g2s(ms + foff, a.msg + ((size_t)rhs * g.nb + fY) * S3 + foff, 3u * fF * 16u, &bar_in);
    }
  };
  if (t < 9) fetch_in(rhs0);
  for (int rhs = rhs0; rhs < rhs1; ++rhs) {
    const size_t blk = (size_t)rhs * g.nb + B;
    float4* xb = reinterpret_cast<float4*>(a.x) + blk * 6 * Vb;
    if (t == 0 && !a.first) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_expect_tx(&bar_x, 6u * Vb * 16u);
      bulk_g2s(xs, xb, 6u * Vb * 16u, &bar_x);
    }
    const int n = rhs - rhs0;
    if (!landed(&bar_in, n & 1, n, a.first ? -1 : n)) return;
    Spinor<float> v, out;
    if (a.first || !odd) {
      const float4* p = a.first ? base + t : base + h;
      const int st = a.first ? Vb : Vh;
#pragma unroll
      for (int u = 0; u < 6; ++u) {
        const float4 q = p[u * st];
        out.c[2 * u] = mk(q.x, q.y);
        out.c[2 * u + 1] = mk(q.z, q.w);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 12; ++k) out.c[k] = mk(0.f, 0.f);
    }
    if (a.take) {
      outer_dir<0>(out, U[0], ms + pos[0], pub + Vh, outside(n0, 8), outside(n0, 0), F0, sf, sb);
      outer_dir<1>(out, U[1], ms + pos[1], pub + Vh, outside(n0, 24), outside(n0, 16), F1, sf, sb);
      outer_dir<2>(out, U[2], ms + pos[2], pub + Vh, outside(n1, 8), outside(n1, 0), F2, sf, sb);
      outer_dir<3>(out, U[3], ms + pos[3], pub + Vh, outside(n1, 24), outside(n1, 16), F3, sf, sb);
    }
    if (odd)
#pragma unroll
      for (int k = 0; k < 12; ++k) out.c[k] = -out.c[k];
#pragma unroll
    for (int u = 0; u < 6; ++u)
      kp[u * Vb + t] = odd ? make_float4(out.c[2 * u].re, out.c[2 * u].im, out.c[2 * u + 1].re, out.c[2 * u + 1].im)
                           : make_float4(0.f, 0.f, 0.f, 0.f);
    v = out;
    // The even-odd solve in half steps: at an even one the even sites receive
    // a hop from the odd ones, at an odd one the odd sites from the even ones.
    // While the receivers multiply their own links with the spinors ahead,
    // the senders multiply theirs for the sites ahead of them, so all warps
    // work; then the receivers add what was sent and make the next vector.
    //   odd   -1: w = A_oo^-1 r_o      2 i - 1: q_i = 1/2 hop res, w = -A_oo^-1 q_i
    //   even  0: res = r_e + 1/2 hop w      2 i: p = A_ee res + 1/2 hop w, MR step alpha_i
    //   odd   2 m + 1: e_o = A_oo^-1 (r_o + sum alpha_i q_i), the hop of e_e
    //         being the sum of the alpha_i times those of the residuals
    // with -A_oo^-1 as the odd block and -r_o in its place, so that every hop
    // is added.  One copy of each part's code serves both parities: the loop
    // has to stay in the instruction cache.
    const int m = a.mr_iters;
    float4* my_pub = odd ? pub + 6 * row : pub;
    float4* my_gx = odd ? gx + 12 * row : gx;
    const float4* th_pub = odd ? pub : pub + 6 * row;
    const float4* th_gx = odd ? gx : gx + 12 * row;
    // odd: q_i (in out) joins the kept vector once alpha_i is known
    auto keep_q = [&]() {
      const f2 al = mk(alpha.x, alpha.y);
#pragma unroll
      for (int u = 0; u < 6; ++u) {
        const float4 z = kp[u * Vb + t];
        f2 x0 = mk(z.x, z.y), x1 = mk(z.z, z.w);
        x0 = x0 - al * out.c[2 * u];
        x1 = x1 - al * out.c[2 * u + 1];
        kp[u * Vb + t] = make_float4(x0.re, x0.im, x1.re, x1.im);
      }
    };
    for (int hs = -1;; ++hs) {
      const bool rx = ((hs & 1) != 0) == odd;
      if (hs > 1 && odd && rx) keep_q();
      if (hs >= 0 && hs <= 2 * m) {
        if (!rx) {
          send_ahead(v, U, my_gx, row, h);
        } else {
          if (odd)
#pragma unroll
            for (int k = 0; k < 12; ++k) out.c[k] = mk(0.f, 0.f);
          take_ahead(out, U, th_pub, row, n0, n1);
        }
        __syncthreads();
        if (rx) take_behind(out, th_gx, row, n0, n1);
      }
      if (hs == 2 * m + 1 && odd) {
#pragma unroll
        for (int u = 0; u < 6; ++u) {
          const float4 q = kp[u * Vb + t];
          out.c[2 * u] = mk(q.x, q.y);
          out.c[2 * u + 1] = mk(q.z, q.w);
        }
      }
      if (hs & 1) {
        // both parities multiply their own block: w or e_o, and A_ee res
        if (odd) clover12(P, out, v);
        else if (hs > 0 && hs < 2 * m + 1) clover12(P, v, out);
      } else if (!odd) {
        if (hs == 0) {
          v = out;
        } else {
          load6(my_pub + h, row, v);        // res
          float d[6] = {};
#pragma unroll
          for (int k = 0; k < 12; ++k) {
            const int e = 3 * (k & 1);
            d[e] = fmaf(out.c[k].re, v.c[k].re, fmaf(out.c[k].im, v.c[k].im, d[e]));
            d[e + 1] = fmaf(out.c[k].re, v.c[k].im, fmaf(-out.c[k].im, v.c[k].re, d[e + 1]));
            d[e + 2] = fmaf(out.c[k].re, out.c[k].re, fmaf(out.c[k].im, out.c[k].im, d[e + 2]));
          }
          float sre = d[0] + d[3], sim = d[1] + d[4], spp = d[2] + d[5];
          sre = warp_sum_r<float>(sre);
          sim = warp_sum_r<float>(sim);
          spp = warp_sum_r<float>(spp);
          if ((t & 31) == 0) red[t >> 5] = make_float4(sre, sim, spp, 0.f);
          bar_sync(1, Vh);
          sre = sim = spp = 0.f;
          for (int w = 0; w < Vh / 32; ++w) {
            const float4 q = red[w];
            sre += q.x; sim += q.y; spp += q.z;
          }
          if (spp > 0.f) {
            // (residuals down to 1e-21 a component: the reciprocal of a sum
            // below 2^-128 is infinite, so small sums are scaled first)
            const float up = spp < 0x1p-100f ? 0x1p64f : 1.f, inv = 1.f / (spp * up);
            const f2 al = mk(sre * up * inv, sim * up * inv);
            if (t == 0) alpha = make_float2(al.re, al.im);
#pragma unroll
            for (int u = 0; u < 6; ++u) {
              const float4 q = kp[u * Vb + t];
              f2 x0 = mk(q.x, q.y), x1 = mk(q.z, q.w);
              fma(x0, al, v.c[2 * u]);
              fma(x1, al, v.c[2 * u + 1]);
              kp[u * Vb + t] = make_float4(x0.re, x0.im, x1.re, x1.im);
            }
#pragma unroll
            for (int k = 0; k < 12; ++k) v.c[k] = v.c[k] - al * out.c[k];
          } else if (t == 0) {
            alpha = make_float2(0.f, 0.f);
          }
        }
        if (hs == 2 * m) {
          if (a.keep) {
            float4* rb = a.res + blk * 6 * Vh + h;
#pragma unroll
            for (int u = 0; u < 6; ++u)
              rb[u * Vh] = make_float4(v.c[2 * u].re, v.c[2 * u].im, v.c[2 * u + 1].re, v.c[2 * u + 1].im);
          }
#pragma unroll
          for (int u = 0; u < 6; ++u) {
            const float4 q = kp[u * Vb + t];
            v.c[2 * u] = mk(q.x, q.y);
            v.c[2 * u + 1] = mk(q.z, q.w);
          }
        }
      }
      if (hs == 2 * m + 1) break;
      if (rx && hs < 2 * m)
#pragma unroll
        for (int u = 0; u < 6; ++u)
          my_pub[u * row + h] = make_float4(v.c[2 * u].re, v.c[2 * u].im, v.c[2 * u + 1].re, v.c[2 * u + 1].im);
      __syncthreads();
      if (hs < 0 && t < 9 && rhs + 1 < rhs1) fetch_in(rhs + 1);     // everyone has read this one's
    }
    // v = e_o or e_e
    if (a.give) {
      float4* to = a.msg + blk * S3;
      give_dir<0>(v, U[0], to + pos[0], outside(n0, 8), outside(n0, 0), F0);
      give_dir<1>(v, U[1], to + pos[1], outside(n0, 24), outside(n0, 16), F1);
      give_dir<2>(v, U[2], to + pos[2], outside(n1, 8), outside(n1, 0), F2);
      give_dir<3>(v, U[3], to + pos[3], outside(n1, 24), outside(n1, 16), F3);
    }
    if (!a.first && !landed(&bar_x, n & 1, n + 1 < rhs1 - rhs0 ? n + 1 : n, n)) return;
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      float4 q = a.first ? make_float4(0.f, 0.f, 0.f, 0.f) : xs[u * Vb + t];
      q.x += v.c[2 * u].re;
      q.y += v.c[2 * u].im;
      q.z += v.c[2 * u + 1].re;
      q.w += v.c[2 * u + 1].im;
      xb[u * Vb + t] = q;
    }
    if (rhs + 1 < rhs1) __syncthreads();       // x and the sent half spinors have been read
  }
}

}  // namespace blk

namespace stg {

using f2 = cpx<float>;

// loads and stores by storage type: FP32, or BF16 / FP16 (half.cuh; spinors
// divided by their site norms)
template <class S>
struct IO;
template <>
struct IO<float> {
  // complex component k of the spinor at site d
  __device__ __forceinline__ static f2 comp(const float* f, const float*, int d, int Vb, int k) {
    return ld_comp(f, comp_off<float>(d, Vb, k));
  }
  __device__ __forceinline__ static void spinor(const float* f, const float*, int d, int Vb, Spinor<float>& s) {
    load_spinor_cg<float>(f, d, Vb, s);
  }
  __device__ __forceinline__ static void link(const float* g, int d, int Vb, int mu, Link<float>& U) {
    load_link<float>(g, d, Vb, mu, U);
  }
  // 36 values of chirality block cb of site d of a clover field
  __device__ __forceinline__ static void block36(const float* c, int d, int Vb, int cb, float* P) {
    load_units<float, CLOVER_NR>(c, d, Vb, cb * 9, 9, P);
  }
  // write this thread's 3 components (k0 = 3 sub) of site d
  __device__ __forceinline__ static void store3(float* f, float*, int d, int Vb, int sub, const f2 v[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) st_comp(f, comp_off<float>(d, Vb, 3 * sub + i), v[i]);
  }
};

template <class S>
struct IOH {
  // 32-bit word of complex component k: unit k / 4, position k % 4
  __device__ __forceinline__ static size_t word(int d, int Vb, int k) {
    return hunit<HSPIN_NU>(d, Vb, k >> 2) * 4 + (k & 3);
  }
  __device__ __forceinline__ static f2 comp(const S* f, const float* nrm, int d, int Vb, int k) {
    const uint32_t w = __ldcg(reinterpret_cast<const unsigned int*>(f) + word(d, Vb, k));
    const float2 v = H2<S>::unpack(w);
    const float m = __ldcg(nrm + d);
    return mk(v.x * m, v.y * m);
  }
  __device__ __forceinline__ static void spinor(const S* f, const float* nrm, int d, int Vb, Spinor<float>& s) {
    load_spinor_h_cg<S>(f, nrm, d, Vb, s);
  }
  __device__ __forceinline__ static void link(const S* g, int d, int Vb, int mu, Link<float>& U) {
    load_link_h<S>(g, d, Vb, mu, U);
  }
  __device__ __forceinline__ static void block36(const S* c, int d, int Vb, int cb, float* P) {
    load_block36_h<S>(c, d, Vb, cb, P);
  }
  // the site norm is the largest magnitude over the four threads of the
  // site (adjacent lanes, combined by shuffles); thread 0 of the site
  // writes it.  Every lane of the warp must call this.
  __device__ __forceinline__ static void store3(S* f, float* nrm, int d, int Vb, int sub, const f2 v[3]) {
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) m = fmaxf(m, fmaxf(fabsf(v[i].re), fabsf(v[i].im)));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    const float inv = m > 0.f ? 1.f / m : 0.f;
    unsigned int* w = reinterpret_cast<unsigned int*>(f);
#pragma unroll
    for (int i = 0; i < 3; ++i) w[word(d, Vb, 3 * sub + i)] = H2<S>::pack(v[i].re * inv, v[i].im * inv);
    if (sub == 0) nrm[d] = m;
  }
};
template <>
struct IO<__half> : IOH<__half> {};
template <>
struct IO<__nv_bfloat16> : IOH<__nv_bfloat16> {};

// own 3 components of the full (global) hopping sum at device site d
template <class S>
__device__ __forceinline__ void hop_global_s(const Geom& g, const S* x, const float* xn, const S* gauge, int d,
                                             int sub, f2 out[3]) {
  Spinor<float> acc;
#pragma unroll
  for (int k = 0; k < 12; ++k) acc.c[k] = mk(0.f, 0.f);
  const Dir<float> dr = make_dir<float>(sub);
  f2 hh[2][3], y[2][3];
  Spinor<float> nb;
  {
    const uint32_t e = __ldg(g.nbr + (size_t)(2 * sub) * g.V + d);
    const int n = (int)(e & ~NEG_BIT);
    IO<S>::spinor(x, xn, n, g.Vb, nb);
    project_rt<float>(nb, dr, -1.f, hh);
    Link<float> U;
    IO<S>::link(gauge, d, g.Vb, sub, U);
    su3_mul(U, hh, y);
    accumulate_rt<float>(acc, y, dr, -1.f, (e & NEG_BIT) ? -1.f : 1.f);
  }
  {
    const uint32_t e = __ldg(g.nbr + (size_t)(2 * sub + 1) * g.V + d);
    const int n = (int)(e & ~NEG_BIT);
    IO<S>::spinor(x, xn, n, g.Vb, nb);
    project_rt<float>(nb, dr, 1.f, hh);
    Link<float> U;
    IO<S>::link(gauge, n, g.Vb, sub, U);
    su3_mul_dag(U, hh, y);
    accumulate_rt<float>(acc, y, dr, 1.f, (e & NEG_BIT) ? -1.f : 1.f);
  }
  reduce_scatter<float>(acc, sub, out);
}

// ---------------------------------------------------------------------------
// Wilson-clover D on the whole lattice with four threads per site (the
// thread layout of the general SAP kernel): thread sub applies the two hops of
// direction mu = sub and the three rows of its chiral clover block that it
// owns; the hop sums are combined by warp shuffles.  A quarter of the
// loads per thread and four times the threads of the one-thread-per-site
// kernel keep more memory requests in flight.
//   y = A x - 1/2 hop(x)                       (DSLASH_D)
// ---------------------------------------------------------------------------
template <class S>
__global__ void __launch_bounds__(256) k_dslash4(Geom g, const S* __restrict__ x, const float* __restrict__ xn,
                                                 S* __restrict__ y, float* __restrict__ yn,
                                                 const S* __restrict__ gauge, const S* __restrict__ clov) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (size_t)4 * g.V) return;        // whole warps (4 V is a multiple of 32)
  const int d = (int)(t >> 2), sub = (int)(t & 3);
  const int cb = sub >> 1, half = sub & 1;
  const size_t off = (size_t)blockIdx.y * g.V * SPINOR_NR;
  const size_t noff = (size_t)blockIdx.y * g.V;
  x += off;
  y += off;
  if (xn) xn += noff;        // site norms exist for half storage only
  if (yn) yn += noff;
  f2 hop[3];
  hop_global_s<S>(g, x, xn, gauge, d, sub, hop);
  f2 x6[6], ax[3];
#pragma unroll
  for (int i = 0; i < 6; ++i) x6[i] = IO<S>::comp(x, xn, d, g.Vb, 6 * cb + i);
  {
    float P[36];
    IO<S>::block36(clov, d, g.Vb, cb, P);
    f2 y6[6];
    herm6<float>(P, x6, y6);
#pragma unroll
    for (int i = 0; i < 3; ++i) ax[i] = half ? y6[3 + i] : y6[i];
  }
  f2 out[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) out[i] = mk(fmaf(-0.5f, hop[i].re, ax[i].re), fmaf(-0.5f, hop[i].im, ax[i].im));
  IO<S>::store3(y, yn, d, g.Vb, sub, out);
}

}  // namespace stg

}  // namespace

static int sap_threads(const Geom& g) { return ((4 * (g.Vb / 2) + 31) / 32) * 32; }

size_t sap_smem_bytes(const Geom& g, int real_size) {
  size_t units = (size_t)GAUGE_NR * real_size / 16 * (g.Vb + LPAD);   // staged links
  size_t bufs = 2 * 12 * (size_t)(g.Vb / 2) * 2 * real_size;          // E, O
  return units * 16 + bufs + 100 * sizeof(double);
}

// shared memory of the block kernel: published spinors and half spinors sent
// ahead, the reduction slots, and the staged operators or, once these are in
// registers, the kept vectors, x, b or the residual, and the messages
static size_t sap_block_smem(const Geom& g, int LU, int CU) {
  const size_t Vh = g.Vb / 2, ops = (size_t)LU * g.Vb * 16 + (size_t)2 * CU * Vh * 16;
  const size_t after = ((size_t)18 * g.Vb + blk::msg_units(g)) * 16;
  return 36 * (Vh + 1) * 16 + 16 * (Vh / 32) + (ops > after ? ops : after);
}

bool sap_block_ok(const Geom& g) { return g.Vb % 64 == 0 && g.Vb <= 256; }
size_t sap_res_bytes(const Geom& g) { return (size_t)g.V / 2 * 96; }
size_t sap_msg_bytes(const Geom& g) {      // 48 bytes per site of each of a block's eight faces
  size_t sites = 0;
  for (int mu = 0; mu < 4; ++mu) sites += 2 * (size_t)(g.Vb / g.b[mu]);
  return (size_t)g.nb * sites * 48;
}

template <class S, int VB>
static cudaError_t launch_block(const Geom& g, const blk::SapArgs& args, cudaStream_t st, bool overlap) {
  const size_t need = sap_block_smem(g, blk::Ops<S>::LU, blk::Ops<S>::CU);
  cudaError_t e = raise_smem_limit((const void*)blk::k_sap_block<S, VB>, need);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  // right-hand sides per CTA: a CTA loads its block's operators once for all
  // of them (about a quarter of a right-hand side's time), but few CTAs of
  // many right-hand sides leave SMs idle in the last wave
  blk::SapArgs a = args;
  const long long slots = (long long)sms * (256 / g.Vb), blocks = g.nb / 2;
  double best = 0.0;
  for (int slices = 1; slices <= a.nrhs; ++slices) {
    const int per = (a.nrhs + slices - 1) / slices;
    if ((a.nrhs + per - 1) / per != slices) continue;
    const double cost = (double)((blocks * slices + slots - 1) / slots) * (per + 0.25);
    if (slices == 1 || cost < best) {
      best = cost;
      a.per = per;
    }
  }
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)(blocks * ((a.nrhs + a.per - 1) / a.per)));
  lc.blockDim = dim3(g.Vb);
  lc.dynamicSmemBytes = need;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // prologue overlaps the previous kernel
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = overlap ? 1 : 0;
  e = cudaLaunchKernelEx(&lc, blk::k_sap_block<S, VB>, a);
  ++g_launches;
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t sap_block_sweep(const Geom& g, int half_kind, int colour, int mr_iters, const SapStep& step, const float* b,
                            float* x, void* res, void* msg, const void* gauge, const void* clover,
                            const void* clover_inv, int nrhs, int* status, long long wait_limit, cudaStream_t st) {
  if (!sap_block_ok(g)) return cudaErrorInvalidValue;
  blk::SapArgs a{g, colour, mr_iters, nrhs, nrhs, step.first, step.take, step.give, step.keep, b, x,
                 static_cast<float4*>(res), static_cast<float4*>(msg), gauge, clover, clover_inv, status, wait_limit};
  auto launch = [&](auto vb) -> cudaError_t {
    constexpr int VB = decltype(vb)::value;
    if (half_kind == 0) return launch_block<__half, VB>(g, a, st, step.overlap);
    if (half_kind == 1) return launch_block<__nv_bfloat16, VB>(g, a, st, step.overlap);
    return launch_block<float, VB>(g, a, st, step.overlap);
  };
  switch (g.Vb) {
    case 64: return launch(std::integral_constant<int, 64>{});
    case 128: return launch(std::integral_constant<int, 128>{});
    case 192: return launch(std::integral_constant<int, 192>{});
    default: return launch(std::integral_constant<int, 256>{});
  }
}

template <class S>
cudaError_t dslash4(const Geom& g, const void* x, const float* xn, void* y, float* yn, const void* gauge,
                    const void* clover, int nrhs, cudaStream_t st) {
  if (g.V % 8) return cudaErrorInvalidValue;
  const size_t threads = (size_t)4 * g.V;
  stg::k_dslash4<S><<<dim3((unsigned)((threads + 255) / 256), nrhs), 256, 0, st>>>(
      g, static_cast<const S*>(x), xn, static_cast<S*>(y), yn, static_cast<const S*>(gauge),
      static_cast<const S*>(clover));
  ++g_launches;
  return cudaGetLastError();
}
template cudaError_t dslash4<float>(const Geom&, const void*, const float*, void*, float*, const void*, const void*,
                                    int, cudaStream_t);
template cudaError_t dslash4<__half>(const Geom&, const void*, const float*, void*, float*, const void*, const void*,
                                     int, cudaStream_t);
template cudaError_t dslash4<__nv_bfloat16>(const Geom&, const void*, const float*, void*, float*, const void*,
                                            const void*, int, cudaStream_t);

template <class R>
cudaError_t sap_sweep(const Geom& g, int colour, int mr_iters, bool x_is_zero, const R* b, R* x,
                      const R* gauge, const R* clover, const R* clover_inv, int nrhs,
                      cudaStream_t st) {
  int threads = sap_threads(g);
  size_t smem = sap_smem_bytes(g, sizeof(R));
  {
    static std::mutex mu;
    static size_t configured[64][2] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (configured[dev][sizeof(R) == 8] < smem) {
      cudaError_t e = cudaFuncSetAttribute(k_sap_sweep<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      configured[dev][sizeof(R) == 8] = smem;
    }
  }
  dim3 grid(g.nb / 2, nrhs);
  k_sap_sweep<R><<<grid, threads, smem, st>>>(g, colour, mr_iters, x_is_zero ? 1 : 0, b, x, gauge,
                                               clover, clover_inv);
  ++g_launches;
  return cudaGetLastError();
}

template cudaError_t sap_sweep<float>(const Geom&, int, int, bool, const float*, float*, const float*,
                                      const float*, const float*, int, cudaStream_t);
template cudaError_t sap_sweep<double>(const Geom&, int, int, bool, const double*, double*,
                                       const double*, const double*, const double*, int, cudaStream_t);

}  // namespace ddamg
