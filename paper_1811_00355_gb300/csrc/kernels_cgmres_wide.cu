// The coarse even-odd GMRES of kernels_cgmres.cu for many right-hand sides
// (FP32, five or more, coarse blocks of 32 to 64 rows; the rule and its one
// exception stand at choose_uncached there): the same method,
// CTA ownership and grid barriers, with everything else arranged for 8 or 12
// right-hand sides in lockstep.
//
// What bounds it: per iteration D_c's blocks are read once (17 blocks a pair of
// sites; 406 MB on 6^3 x 12 coarse sites with n_v 24, 61 us of DRAM time) and
// 8 (2n)^2 real multiply-adds per block and four right-hand sides run on the
// FP32 pipe (64 us for 12).  So:
//  * block products: a site's 2n x 2n blocks come through a ring of
//    shared-memory slots (bulk copies, no CTA barrier per block); each of the 16
//    warps takes every 16th column and multiplies all 2n rows with all right-hand sides, lane (g, j) the row
//    pairs j, j + 8, .. and a quarter of the right-hand sides: per column
//    UT + RQ shared-memory loads for 8 UT RQ multiply-adds.  The warps' sums
//    meet in shared memory once per site.  (1.1 us per block: the pipes' own
//    times are 0.42 us of multiply-adds and 0.5 us of shared memory; mma.sync in
//    3xTF32 would need 0.45 us of the tensor pipe.)
//  * the next site's vectors are copied (cp.async) while this site is
//    multiplied; scales and signs are applied to the sums instead.
//  * Gram-Schmidt: a warp keeps a right-hand side's piece of w in registers for
//    eight basis vectors at a time; the basis stays in L2.
//  * the partial sums of all CTAs are FP32 pairs, four of them per warp in flight.
// The form before (two row pairs and four right-hand sides per thread, a CTA
// barrier per block, vectors staged before each site, passes of eight) took
// 530 us per iteration of 12 right-hand sides there; this one 268.
#include <algorithm>

#include "cgmres.cuh"

namespace ddamg {

namespace {

constexpr int TPB = 512;
constexpr int NWARP = TPB / 32;
constexpr int RING_MAX = 8;

// shared memory, identical on host and device
struct WidePlan {
  size_t sv, sv_bytes, ring, hc, h2, cs, sn, gv, yv, beta, bnorm, hn, scale, act, kd, tot, conv, nbo, bytes;
  int slots;
};
__host__ __device__ inline int wide_svs(int n2) { return n2 + 2; }     // even: 16-byte rows
__host__ __device__ inline int wide_ut(int n2) { return (n2 / 2 + 7) / 8; }
__host__ __device__ inline WidePlan wide_plan(int NR, int n2, int m, int per, int slots) {
  WidePlan p;
  size_t o = 0;
  auto put = [&](size_t bytes) { const size_t r = o; o = al16(o + bytes); return r; };
  const size_t vec = (size_t)9 * NR * wide_svs(n2) * 8, red = (size_t)(NWARP / 2) * NR * 16 * wide_ut(n2) * 8;
  p.sv_bytes = al16(vec > red ? vec : red);
  p.sv = put(2 * p.sv_bytes);
  p.slots = slots;
  p.ring = put((size_t)slots * n2 * n2 * 8);
  p.hc = put((size_t)NR * 2 * (m + 1) * 4);
  p.h2 = put((size_t)NR * 4);
  p.cs = put((size_t)NR * m * 4);
  p.sn = put((size_t)NR * 2 * m * 4);
  p.gv = put((size_t)NR * 2 * (m + 1) * 4);
  p.yv = put((size_t)NR * 2 * m * 4);
  p.beta = put((size_t)NR * 4);
  p.bnorm = put((size_t)NR * 4);
  p.hn = put((size_t)NR * 4);
  p.scale = put((size_t)NR * 4);
  p.act = put((size_t)NR * 4);
  p.kd = put((size_t)NR * 4);
  p.tot = put((size_t)NR * 4);
  p.conv = put((size_t)NR * 4);
  p.nbo = put((size_t)2 * per * 8 * 4);
  p.bytes = o;
  return p;
}
// global scratch of a CTA: basis, x, right-hand side, w, and the R factors
__host__ __device__ inline size_t wide_local(int NR, int n2, int m, int per) {
  return al16((size_t)(m + 4) * NR * per * n2 * 8) + al16((size_t)NR * m * (m + 1) * 4);
}

struct WideArgs {
  Geom g;
  const cpx<float>*Dc, *Ainv, *AD;
  int n2, m, max_iter, nrhs, NE, per, slots;
  float tol;
  const cpx<float>* b;
  cpx<float>* x;
  cpx<float>*wg, *to, *xg;       // [NR][NE][n2]
  unsigned char* lglob;
  size_t lstride;
  float2* part;                  // [(m + 2) * NR][G]
  unsigned* bar;
  int *iters, *iters_acc, *status;
  long long spin_limit;
};

__device__ __forceinline__ void cp16_cg(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
// sum of 16 values over a warp as a reduce-scatter: lane l ends with the total
// of value (l >> 1) & 15
__device__ __forceinline__ float warp_reduce_scatter16(float (&v)[16]) {
  const int l = threadIdx.x & 31;
#pragma unroll
  for (int lev = 0; lev < 4; ++lev) {
    const int half = 8 >> lev, off = 16 >> lev;
    const bool up = (l & off) != 0;
#pragma unroll
    for (int k = 0; k < half; ++k) {
      const float send = up ? v[k] : v[k + half], keep = up ? v[k + half] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// what a phase of block products multiplies: A_oo^-1 of the odd sites; A_oo^-1 D_c
// of the odd sites; the even sites' blocks with and without the self block
enum Kind { K_INV, K_ODD, K_EVEN, K_EVEN_HOPS };

template <int NR, int UT>
__global__ void __launch_bounds__(TPB, 1) k_cgmres_wide(WideArgs a) {
  constexpr int RQ = NR / 4;
  extern __shared__ __align__(16) unsigned char sm[];
  const int n2 = a.n2, m = a.m, NE = a.NE, L = a.per * n2, svs = wide_svs(n2);
  const unsigned nn = (unsigned)(n2 * n2);
  const WidePlan P = wide_plan(NR, n2, m, a.per, a.slots);
  const unsigned RING = (unsigned)a.slots;
  cpx<float>* ringbuf = reinterpret_cast<cpx<float>*>(sm + P.ring);
  float* hc = reinterpret_cast<float*>(sm + P.hc);      // [NR][2(m+1)]
  float* h2 = reinterpret_cast<float*>(sm + P.h2);      // [NR]
  float* cs = reinterpret_cast<float*>(sm + P.cs);      // [NR][m]
  float* sn = reinterpret_cast<float*>(sm + P.sn);      // [NR][2m]
  float* gv = reinterpret_cast<float*>(sm + P.gv);      // [NR][2(m+1)]
  float* yv = reinterpret_cast<float*>(sm + P.yv);      // [NR][2m]
  float* beta = reinterpret_cast<float*>(sm + P.beta);
  float* bnorm = reinterpret_cast<float*>(sm + P.bnorm);
  float* hnv = reinterpret_cast<float*>(sm + P.hn);
  float* scl = reinterpret_cast<float*>(sm + P.scale);
  int* act = reinterpret_cast<int*>(sm + P.act);        // active in this cycle
  int* kd = reinterpret_cast<int*>(sm + P.kd);          // basis size of this cycle
  int* tot = reinterpret_cast<int*>(sm + P.tot);        // iterations so far
  int* conv = reinterpret_cast<int*>(sm + P.conv);      // converged (or gave up)
  int* nbo = reinterpret_cast<int*>(sm + P.nbo);
  unsigned char* lbase = a.lglob + (size_t)blockIdx.x * a.lstride;
  cpx<float>* V = reinterpret_cast<cpx<float>*>(lbase);           // [m+1][NR][L]
  cpx<float>* xl = V + (size_t)(m + 1) * NR * L;                  // [NR][L]
  cpx<float>* rl = xl + (size_t)NR * L;
  cpx<float>* wl = rl + (size_t)NR * L;
  float* Rf = reinterpret_cast<float*>(lbase + al16((size_t)(m + 4) * NR * L * 8));   // [NR][m(m+1)] packed columns
  __shared__ int any_s, any_act_s, exn[NR];
  __shared__ __align__(8) uint64_t full[RING_MAX], empty[RING_MAX];   // a slot's block has landed / is done with
  __shared__ signed char sent[RING_MAX];      // the phase parity of `full` that a slot's last copy completes; -1: no copy yet

  const int G = gridDim.x, tx = threadIdx.x, wid = tx >> 5, lane = tx & 31;
  const int gq = lane >> 3, jq = lane & 7;          // right-hand-side quarter, row-pair slot
  grid_barrier_reset();
  const int lo = min(NE, (int)blockIdx.x * a.per), hi = min(NE, lo + a.per), nown = hi - lo;
  const int Lo = nown * n2;
  const size_t vstr = (size_t)NE * n2;
  const int TRI = m * (m + 1) / 2;
  const size_t NX = a.g.nb;

  for (int i = tx; i < 2 * nown * 8; i += TPB) {
    const int par = i / (nown * 8), rem = i - par * nown * 8, kk = rem / 8, d = 1 + rem % 8;
    const int X = par ? a.g.ceven[lo + kk] : a.g.codd[lo + kk];
    nbo[(par * a.per + kk) * 8 + d - 1] = a.g.cpos[a.g.cnbr[d * a.g.nb + X]] * n2;
  }
  if (tx == 0) {
    for (unsigned q = 0; q < RING; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], NWARP);
      sent[q] = -1;
    }
    mbar_fence_init();
  }
  __syncthreads();
  auto Vk = [&](int k, int r) { return V + ((size_t)k * NR + r) * L; };
  // this warp's columns of a block; the lane's last row pair, one of the block's
  // (its sums are left out where the block has fewer); the sums this thread
  // adds up over the warps: (right-hand side, row) outr[i], outw[i]
  const int np = n2 / 2, ncol = (n2 - wid + NWARP - 1) / NWARP;
  const int last = min(8 * (UT - 1), np - 1 - jq);
  int outr[2], outw[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int idx = tx + i * TPB;
    outr[i] = idx / n2;
    outw[i] = idx - outr[i] * n2;
  }

  // ---- block products ---------------------------------------------------------
  // Blocks of a launch are numbered in the order of their use, block i goes
  // through slot i % RING.  A phase's first RING blocks are copied by thread 0;
  // the block RING after block b follows into its slot once all warps have
  // taken b, sent by one warp in turn when it is done with block b + 1.
  unsigned used = 0;                       // blocks of the phases before
  unsigned primed = 0;                     // of the next phase's blocks, those on their way
  unsigned slot = 0, turn = 0;             // block `used`: its slot, and the parity of the slot's use
  auto blk = [&](int kind, unsigned i) -> const cpx<float>* {
    if (kind == K_INV) return a.Ainv + (size_t)a.g.codd[lo + i] * nn;
    if (kind == K_ODD) return a.AD + ((size_t)lo * 8 + i) * nn;
    const unsigned nd = kind == K_EVEN ? 9 : 8;
    return a.Dc + ((size_t)a.g.ceven[lo + i / nd] * 9 + (9 - nd) + i % nd) * nn;
  };
  // (parity: that of block i's use of slot q)
  auto copy = [&](int kind, unsigned base, unsigned q, unsigned parity, unsigned i) {
    sent[q] = (signed char)parity;
    mbar_expect_tx(&full[q], nn * 8);
    bulk_g2s(ringbuf + (size_t)q * nn, blk(kind, i - base), nn * 8, &full[q]);
  };
  // the first blocks of the next phase, which has to be of this kind, travel
  // while the CTA waits for the others (all slots are free between phases)
  auto prime = [&](int kind) {
    const unsigned nd = kind == K_INV ? 1 : kind == K_EVEN ? 9 : 8, n = min(RING, nown * nd);
    if (tx == 0)
      for (unsigned i = primed; i < n; ++i) {
        const unsigned at = slot + i;         // (at most RING - 1 past the last slot)
        copy(kind, used, at % RING, at < RING ? turn : turn ^ 1u, used + i);
      }
    primed = n;
  };
  // before the CTA leaves early (all threads past a CTA barrier): every copy
  // that was sent has landed, each wait bounded
  auto drain = [&]() {
    if (tx == 0)
      for (unsigned q = 0; q < RING; ++q)
        if (sent[q] >= 0) mbar_wait_bounded(&full[q], (unsigned)sent[q], MBAR_POLL_LIMIT);
  };
  // the grid barriers; false (copies on their way waited for) when one gives up
  auto others = [&]() -> bool {
    if (grid_wait(a.bar, a.status, a.spin_limit)) return true;
    drain();
    return false;
  };
  auto meet = [&]() -> bool {
    grid_arrive(a.bar);
    return others();
  };
  // vectors that block d0 + t of site si multiplies, into buffer `buf`:
  // src(si, t, r) is the address of n2 entries (16-byte pieces)
  auto stage = [&](int nd, int si, int buf, auto&& src) {
    cpx<float>* sv = reinterpret_cast<cpx<float>*>(sm + P.sv + buf * P.sv_bytes);
#pragma unroll 4
    for (int row = wid; row < nd * NR; row += NWARP) {
      const cpx<float>* s = src(si, row / NR, row % NR);
      if (s)
        for (int c = lane; c < np; c += 32) cp16_cg(sv + (size_t)row * svs + 2 * c, s + 2 * c);
      else
        for (int c = lane; c < np; c += 32)
          *reinterpret_cast<float4*>(sv + (size_t)row * svs + 2 * c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // emit(si, r, row, sum) for every site, right-hand side and row; false when
  // a copy did not land in time (status set, copies in flight waited for)
  auto products = [&](int kind, auto&& src, auto&& emit) -> bool {
    const int nd = kind == K_INV ? 1 : kind == K_EVEN ? 9 : 8;
    const unsigned base = used, end = base + (unsigned)(nown * nd);
    bool ok = true;
    prime(kind);
    primed = 0;
    if (nown) stage(nd, 0, 0, src);
    for (int si = 0; si < nown; ++si) {
      const int buf = si & 1;
      if (si + 1 < nown) {
        if (wid == NWARP - 1) prefetch_l2(blk(kind, (unsigned)((si + 1) * nd)), (size_t)nd * nn * 8);
        stage(nd, si + 1, buf ^ 1, src);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncthreads();
      const cpx<float>* sv = reinterpret_cast<const cpx<float>*>(sm + P.sv + buf * P.sv_bytes) + (size_t)gq * RQ * svs;
      cpx<float> acc[UT][2][RQ];
#pragma unroll
      for (int u = 0; u < UT; ++u)
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
          for (int q = 0; q < RQ; ++q) acc[u][e][q] = mk(0.f, 0.f);
      for (int t = 0; t < nd; ++t) {
        const unsigned b = base + (unsigned)(si * nd + t);
        if (ok) ok = mbar_wait_bounded(&full[slot], turn, a.spin_limit);
        // columns wid + 16 i: the lane's row pairs and right-hand sides
        const float4 *M = reinterpret_cast<const float4*>(ringbuf + (size_t)slot * nn) + wid * np + jq, *Ml = M + last;
        const cpx<float>* vt = sv + (size_t)t * NR * svs + wid;
        auto column = [&](int i) {
          cpx<float> v[RQ];
          float4 e[UT];
#pragma unroll
          for (int q = 0; q < RQ; ++q) v[q] = vt[q * svs + i * NWARP];
#pragma unroll
          for (int u = 0; u < UT; ++u) e[u] = u + 1 < UT ? M[i * NWARP * np + 8 * u] : Ml[i * NWARP * np];
#pragma unroll
          for (int u = 0; u < UT; ++u)
#pragma unroll
            for (int q = 0; q < RQ; ++q) {
              fma(acc[u][0][q], mk(e[u].x, e[u].y), v[q]);
              fma(acc[u][1][q], mk(e[u].z, e[u].w), v[q]);
            }
        };
        // (every warp has UT - 1 columns, 16 (UT - 1) <= n2 <= 16 UT, some one more)
#pragma unroll
        for (int i = 0; i + 1 < UT; ++i) column(i);
        if (UT - 1 < ncol) column(UT - 1);
        // (a warp that has given up neither frees a slot nor fills one: a
        // slot's copies follow one another, each after the one before landed)
        ok = __all_sync(0xffffffffu, ok);
        if (lane == 0 && ok) {
          mbar_arrive(&empty[slot]);
          if (wid == (int)(b % NWARP) && b > base && b - 1 + RING < end) {
            const unsigned before = slot ? slot - 1 : RING - 1, p = slot ? turn : turn ^ 1u;
            ok = mbar_wait_bounded(&empty[before], p, a.spin_limit);
            if (ok) copy(kind, base, before, p ^ 1u, b - 1 + RING);
          }
        }
        if (++slot == RING) {
          slot = 0;
          turn ^= 1u;
        }
      }
      if (__syncthreads_or(!ok)) {
        if (tx == 0) atomicExch(a.status, 6);
        drain();
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        return false;
      }
      // sum over the warps in this site's (now free) buffer: eight warps, then all
      float4* red = reinterpret_cast<float4*>(sm + P.sv + buf * P.sv_bytes);   // [8][NR][8 UT] row pairs
      auto at = [&](int w, int u, int q) { return ((w * NR + gq * RQ + q) * UT + u) * 8 + jq; };
      if (wid >= NWARP / 2)
#pragma unroll
        for (int u = 0; u < UT; ++u)
#pragma unroll
          for (int q = 0; q < RQ; ++q)
            red[at(wid - NWARP / 2, u, q)] = make_float4(acc[u][0][q].re, acc[u][0][q].im, acc[u][1][q].re, acc[u][1][q].im);
      __syncthreads();
      if (wid < NWARP / 2)
#pragma unroll
        for (int u = 0; u < UT; ++u)
#pragma unroll
          for (int q = 0; q < RQ; ++q) {
            float4 z = red[at(wid, u, q)];
            z.x += acc[u][0][q].re; z.y += acc[u][0][q].im;
            z.z += acc[u][1][q].re; z.w += acc[u][1][q].im;
            red[at(wid, u, q)] = z;
          }
      __syncthreads();
      const float2* rs = reinterpret_cast<const float2*>(red);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = outr[i], row = outw[i];
        if (r >= NR) break;
        float re = 0.f, im = 0.f;
#pragma unroll
        for (int w = 0; w < NWARP / 2; ++w) {
          const float2 z = rs[(size_t)(w * NR + r) * 16 * UT + row];
          re += z.x;
          im += z.y;
        }
        emit(si, r, row, mk(re, im));
      }
      __syncthreads();
    }
    used = end;
    return true;
  };

  // to = f A_oo^-1 D_oe src (f = scl, the scale of the unnormalised src)
  auto phase_odd = [&](const cpx<float>* srcv) -> bool {
    return products(
        K_ODD, [&](int si, int t, int r) { return srcv + r * vstr + nbo[si * 8 + t]; },
        [&](int si, int r, int row, cpx<float> s) { a.to[r * vstr + (size_t)(lo + si) * n2 + row] = scl[r] * s; });
  };
  // w = A_ee v - D_eo to: the self block's vector enters negated, the sum is negated
  auto phase_even = [&](const cpx<float>* vself, cpx<float>* out) -> bool {
    return products(
        K_EVEN,
        [&](int si, int t, int r) -> const cpx<float>* {
          return t == 0 ? vself + (size_t)r * L + si * n2 : a.to + r * vstr + nbo[(a.per + si) * 8 + t - 1];
        },
        [&](int si, int r, int row, cpx<float> s) { out[(size_t)r * L + si * n2 + row] = mk(-s.re, -s.im); });
  };
  // out = A_oo^-1 b_o of right-hand sides r < nr (zero for the others)
  auto phase_inv = [&](const cpx<float>* bb, int nr, auto&& emit) -> bool {
    return products(
        K_INV,
        [&](int si, int, int r) -> const cpx<float>* {
          return r < nr ? bb + (size_t)r * NX * n2 + (size_t)a.g.codd[lo + si] * n2 : nullptr;
        },
        emit);
  };

  // f(r, e) for the CTA's pairs e of entries of every right-hand side
  auto each_pair = [&](auto&& f) {
    const int half = Lo / 2;
    if (!half) return;
    int r = tx / half, e = tx - r * half;
    while (r < NR) {
      f(r, e);
      e += TPB;
      while (e >= half) {
        e -= half;
        ++r;
      }
    }
  };

  // ---- Gram-Schmidt -------------------------------------------------------------
  // sums over this CTA of <V_j[r], w[r]> for j < kcount (slot (s0 + j) NR + r)
  // and, in slot (s0 + kcount) NR + r, ||w[r]||^2: a warp takes a right-hand
  // side and eight vectors at a time.  Other CTAs may still be gathering the
  // reduction before: where no grid barrier lies between that gather and this
  // call, s0 has to lead past its slots
  auto partial = [&](int s0, int kcount) {
    float2* part = a.part + (size_t)s0 * NR * G;
    const int groups = (kcount + 7) / 8 > 0 ? (kcount + 7) / 8 : 1;
    for (int un = wid; un < groups * NR; un += NWARP) {
      const int r = un % NR, j0 = (un / NR) * 8;
      float d[16], nn2 = 0.f;
#pragma unroll
      for (int q = 0; q < 16; ++q) d[q] = 0.f;
      if (act[r]) {
        const float4* ww = reinterpret_cast<const float4*>(wl + (size_t)r * L);
        // (vectors past the last one: the last one again, their sums unused)
        const float4* vv[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) vv[q] = reinterpret_cast<const float4*>(Vk(max(0, min(j0 + q, kcount - 1)), r));
        for (int e = lane; e < Lo / 2; e += 32) {
          const float4 w = ww[e];
          float4 v[8];
          if (kcount)
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = vv[q][e];
          nn2 += w.x * w.x + w.y * w.y + w.z * w.z + w.w * w.w;
          if (kcount)
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              d[2 * q] += v[q].x * w.x + v[q].y * w.y + v[q].z * w.z + v[q].w * w.w;
              d[2 * q + 1] += v[q].x * w.y - v[q].y * w.x + v[q].z * w.w - v[q].w * w.z;
            }
        }
      }
      if (kcount) {
        const float sum = warp_reduce_scatter16(d);      // value (lane / 2) % 16 in lanes 2 i, 2 i + 1
        const int q = lane >> 2;
        const float im = __shfl_down_sync(0xffffffffu, sum, 2);
        if ((lane & 3) == 0 && j0 + q < kcount)
          part[(size_t)((j0 + q) * NR + r) * G + blockIdx.x] = make_float2(sum, im);
      }
      if (j0 == 0) {
        nn2 = wsum(nn2);
        if (lane == 0) part[(size_t)(kcount * NR + r) * G + blockIdx.x] = make_float2(nn2, 0.f);
      }
    }
  };
  // the slots' sums over all CTAs: dots to dst[r][2 j], squared norms to nrm[r]
  auto gather = [&](int s0, int kcount, float* dst, float* nrm) {
    const float2* part = a.part + (size_t)s0 * NR * G;
    const int pairs = (kcount + 1) * NR;
    for (int p0 = 4 * wid; p0 < pairs; p0 += 4 * NWARP) {
      float re[4] = {}, im[4] = {};
      for (int c = lane; c < G; c += 32)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (p0 + q < pairs) {
            const float2 z = __ldcg(part + (size_t)(p0 + q) * G + c);
            re[q] += z.x;
            im[q] += z.y;
          }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        re[q] = wsum(re[q]);
        im[q] = wsum(im[q]);
        const int p = p0 + q, j = p / NR, r = p - j * NR;
        if (lane == 0 && p < pairs) {
          if (j < kcount) {
            dst[(size_t)r * 2 * (m + 1) + 2 * j] = re[q];
            dst[(size_t)r * 2 * (m + 1) + 2 * j + 1] = im[q];
          } else {
            nrm[r] = re[q];
          }
        }
      }
    }
    __syncthreads();
  };

  for (int r0 = 0; r0 < a.nrhs; r0 += NR) {
    const int nr = min(NR, a.nrhs - r0);
    const cpx<float>* bb = a.b + (size_t)r0 * NX * n2;
    cpx<float>* xx = a.x + (size_t)r0 * NX * n2;
    if (tx < NR) {
      act[tx] = tx < nr ? 1 : 0;
      conv[tx] = tx < nr ? 0 : 1;
      tot[tx] = 0;
      scl[tx] = 1.f;
    }
    __syncthreads();
    // to = A_oo^-1 b_o
    if (!phase_inv(bb, nr, [&](int si, int r, int row, cpx<float> s) {
          a.to[r * vstr + (size_t)(lo + si) * n2 + row] = s;
        }))
      return;
    prime(K_EVEN_HOPS);
    if (!meet()) return;
    // rhs_e = b_e - D_eo to; x_e = 0; w = rhs_e
    if (!products(
            K_EVEN_HOPS, [&](int si, int t, int r) { return a.to + r * vstr + nbo[(a.per + si) * 8 + t]; },
            [&](int si, int r, int row, cpx<float> s) {
              cpx<float> v = mk(0.f, 0.f);
              if (r < nr) v = bb[(size_t)r * NX * n2 + (size_t)a.g.ceven[lo + si] * n2 + row] - s;
              const size_t o = (size_t)r * L + si * n2 + row;
              rl[o] = v;
              wl[o] = v;
              xl[o] = mk(0.f, 0.f);
            }))
      return;
    partial(0, 0);
    if (!meet()) return;
    gather(0, 0, hc, bnorm);
    if (tx < NR) {
      bnorm[tx] = sqrtf(bnorm[tx]);
      beta[tx] = bnorm[tx];
      if (!(bnorm[tx] > 0.f)) { conv[tx] = 1; act[tx] = 0; }
    }
    __syncthreads();

    while (true) {
      // start a cycle for every right-hand side that is not done
      if (tx < NR) {
        const bool go = !conv[tx] && tot[tx] < a.max_iter;
        act[tx] = go ? 1 : 0;
        if (!go) conv[tx] = 1;
        kd[tx] = 0;
        gv[tx * 2 * (m + 1)] = beta[tx];
        gv[tx * 2 * (m + 1) + 1] = 0.f;
        scl[tx] = beta[tx] > 0.f ? 1.f / beta[tx] : 0.f;
      }
      __syncthreads();
      if (tx == 0) {
        int any = 0;
        for (int r = 0; r < NR; ++r) any |= act[r];
        any_s = any;
      }
      __syncthreads();
      if (!any_s) break;
      // V_0 = w / beta (own sites) and the global copy of w for the neighbours
      for (int idx = tx; idx < NR * Lo; idx += TPB) {
        const int r = idx / Lo, e = idx - r * Lo;
        const cpx<float> v = wl[(size_t)r * L + e];
        Vk(0, r)[e] = scl[r] * v;
        a.wg[r * vstr + (size_t)lo * n2 + e] = v;
      }
      if (!meet()) return;
      for (int k = 0; k < m; ++k) {
        // w = S V_k: odd phase from the neighbours' unnormalised w (scale 1/h)
        if (!phase_odd(a.wg)) return;
        prime(K_EVEN);
        // the self block's vector, negated, for the even phase
        each_pair([&](int r, int e) {
          const float4 v = reinterpret_cast<const float4*>(Vk(k, r))[e];
          reinterpret_cast<float4*>(wl + (size_t)r * L)[e] = make_float4(-v.x, -v.y, -v.z, -v.w);
        });
        if (!meet()) return;
        if (!phase_even(wl, wl)) return;
        prime(K_ODD);
        // Givens rotation of right-hand side r's new Hessenberg column (one
        // thread), new residual estimate, scale 1/h of V_{k+1}, convergence
        auto givens = [&](int r) {
          const float hn = sqrtf(hnv[r]);
          const float* __restrict__ col = hc + (size_t)r * 2 * (m + 1);   // this column of the Hessenberg matrix
          float* __restrict__ csr = cs + (size_t)r * m;
          float* __restrict__ snr = sn + (size_t)r * 2 * m;
          float* __restrict__ Rr = Rf + (size_t)r * 2 * TRI;
          const int base = k * (k + 1) / 2;          // packed column k: entries 0..k
          float ar = col[0], ai = col[1];            // runs down the column through the rotations so far
#pragma unroll 4
          for (int j = 0; j < k; ++j) {
            const float c = csr[j], sr = snr[2 * j], si = snr[2 * j + 1], br = col[2 * j + 2], bi = col[2 * j + 3];
            Rr[2 * (base + j)] = c * ar + (sr * br - si * bi);
            Rr[2 * (base + j) + 1] = c * ai + (sr * bi + si * br);
            const float ur = c * br - (sr * ar + si * ai), ui = c * bi - (sr * ai - si * ar);
            ar = ur;
            ai = ui;
          }
          const float br = hn, bi = 0.f;
          const float a1 = sqrtf(ar * ar + ai * ai), a2 = sqrtf(br * br + bi * bi);
          float c, sr, si, rr, ri;
          if (a2 == 0.f) { c = 1.f; sr = 0.f; si = 0.f; rr = ar; ri = ai; }
          else if (a1 == 0.f) { c = 0.f; sr = br / a2; si = -bi / a2; rr = a2; ri = 0.f; }
          else {
            const float rho = hypotf(a1, a2), pr = ar / a1, pi = ai / a1;
            c = a1 / rho;
            sr = (pr * br + pi * bi) / rho;
            si = (pi * br - pr * bi) / rho;
            rr = pr * rho; ri = pi * rho;
          }
          csr[k] = c; snr[2 * k] = sr; snr[2 * k + 1] = si;
          Rr[2 * (base + k)] = rr; Rr[2 * (base + k) + 1] = ri;
          float* g = gv + (size_t)r * 2 * (m + 1);
          const float gr = g[2 * k], gi = g[2 * k + 1];
          g[2 * (k + 1)] = -(sr * gr + si * gi);
          g[2 * (k + 1) + 1] = -(sr * gi - si * gr);
          g[2 * k] = c * gr;
          g[2 * k + 1] = c * gi;
          const float res = sqrtf(g[2 * (k + 1)] * g[2 * (k + 1)] + g[2 * (k + 1) + 1] * g[2 * (k + 1) + 1]);
          kd[r] = k + 1;
          tot[r] += 1;
          scl[r] = hn > 0.f ? 1.f / hn : 0.f;
          hnv[r] = hn;
          if (res <= a.tol * bnorm[r] || hn == 0.f || tot[r] >= a.max_iter) act[r] = 0;
        };
        // one classical Gram-Schmidt pass whose reduction also carries ||w||^2,
        // so ||w_new||^2 = ||w||^2 - sum_j |h_j|^2 (Pythagoras); an explicit
        // norm is taken only if that difference has cancelled
        partial(0, k + 1);
        if (!meet()) return;
        gather(0, k + 1, hc, hnv);
        if (tx < NR) {
          const float* hr = hc + (size_t)tx * 2 * (m + 1);
          float s2 = hnv[tx];
          for (int j = 0; j <= k; ++j) s2 -= hr[2 * j] * hr[2 * j] + hr[2 * j + 1] * hr[2 * j + 1];
          exn[tx] = (act[tx] && !(s2 > 1e-3f * hnv[tx])) ? 1 : 0;
          hnv[tx] = s2 > 0.f ? s2 : 0.f;
        }
        __syncthreads();
        if (tx == 0) {
          int any = 0;
          for (int r = 0; r < NR; ++r) any |= exn[r];
          any_s = any;
        }
        each_pair([&](int r, int e) {
          if (!act[r]) return;
          float4 w = reinterpret_cast<const float4*>(wl + (size_t)r * L)[e];
          const float2* hr = reinterpret_cast<const float2*>(hc + (size_t)r * 2 * (m + 1));
#pragma unroll 8
          for (int j = 0; j <= k; ++j) {
            const float4 v = reinterpret_cast<const float4*>(Vk(j, r))[e];
            const float2 c = hr[j];
            w.x -= c.x * v.x - c.y * v.y;
            w.y -= c.x * v.y + c.y * v.x;
            w.z -= c.x * v.z - c.y * v.w;
            w.w -= c.x * v.w + c.y * v.z;
          }
          reinterpret_cast<float4*>(wl + (size_t)r * L)[e] = w;
          reinterpret_cast<float4*>(a.wg + r * vstr + (size_t)lo * n2)[e] = w;
        });
        __syncthreads();
        const int any_explicit = any_s;
        if (any_explicit) {
          partial(k + 2, 0);       // (past the dots' slots, which others may still read)
          if (!meet()) return;
          gather(k + 2, 0, hc, h2);
          if (tx < NR && exn[tx]) hnv[tx] = h2[tx];
          __syncthreads();
        } else {
          // publish w for the next odd phase; the Givens step and the new
          // basis vector are local work done while the other CTAs arrive
          grid_arrive(a.bar);
        }
        if (tx < NR && act[tx]) givens(tx);
        __syncthreads();
        each_pair([&](int r, int e) {
          const float f = scl[r];
          const float4 w = reinterpret_cast<const float4*>(wl + (size_t)r * L)[e];
          reinterpret_cast<float4*>(Vk(k + 1, r))[e] = make_float4(f * w.x, f * w.y, f * w.z, f * w.w);
        });
        if (tx == 0) {
          int any = 0;
          for (int r = 0; r < NR; ++r) any |= act[r];
          any_act_s = any;
        }
        if (!any_explicit) {
          if (!others()) return;
        } else {
          __syncthreads();
        }
        if (!any_act_s) break;
      }
      // y = R^-1 g; x_e += V y (every right-hand side of this cycle)
      if (tx < NR && !conv[tx]) {
        const int r = tx, kk = kd[r];
        const float* Rr = Rf + (size_t)r * 2 * TRI;
        const float* g = gv + (size_t)r * 2 * (m + 1);
        float* y = yv + (size_t)r * 2 * m;
        for (int i = kk - 1; i >= 0; --i) {
          float accr = g[2 * i], acci = g[2 * i + 1];
          for (int j = i + 1; j < kk; ++j) {
            const int pj = j * (j + 1) / 2 + i;
            const float rr = Rr[2 * pj], ri = Rr[2 * pj + 1];
            accr -= rr * y[2 * j] - ri * y[2 * j + 1];
            acci -= rr * y[2 * j + 1] + ri * y[2 * j];
          }
          const int pd = i * (i + 1) / 2 + i;
          const float dr = Rr[2 * pd], di = Rr[2 * pd + 1], dn = dr * dr + di * di;
          y[2 * i] = (accr * dr + acci * di) / dn;
          y[2 * i + 1] = (acci * dr - accr * di) / dn;
        }
      }
      __syncthreads();
      for (int idx = tx; idx < NR * Lo; idx += TPB) {
        const int r = idx / Lo, e = idx - r * Lo;
        if (conv[r]) continue;
        const float* y = yv + (size_t)r * 2 * m;
        cpx<float> s = xl[(size_t)r * L + e];
        for (int j = 0; j < kd[r]; ++j) fma(s, mk(y[2 * j], y[2 * j + 1]), Vk(j, r)[e]);
        xl[(size_t)r * L + e] = s;
        a.xg[r * vstr + (size_t)lo * n2 + e] = s;
        wl[(size_t)r * L + e] = mk(-s.re, -s.im);      // the self block's vector below
      }
      if (tx < NR) scl[tx] = 1.f;
      if (!meet()) return;
      // true residual w = rhs_e - S x_e
      if (!phase_odd(a.xg)) return;
      prime(K_EVEN);
      if (!meet()) return;
      if (!phase_even(wl, wl)) return;
      for (int idx = tx; idx < NR * Lo; idx += TPB) {
        const int r = idx / Lo, e = idx - r * Lo;
        wl[(size_t)r * L + e] = rl[(size_t)r * L + e] - wl[(size_t)r * L + e];
      }
      if (tx < NR) act[tx] = conv[tx] ? 0 : 1;
      __syncthreads();
      partial(0, 0);
      if (!meet()) return;
      gather(0, 0, hc, beta);
      if (tx < NR && !conv[tx]) {
        beta[tx] = sqrtf(beta[tx]);
        if (beta[tx] <= a.tol * bnorm[tx]) conv[tx] = 1;
      }
      __syncthreads();
    }
    // x_o = A_oo^-1 b_o - A_oo^-1 D_oe x_e; write x
    for (int idx = tx; idx < NR * Lo; idx += TPB) {
      const int r = idx / Lo, e = idx - r * Lo;
      const cpx<float> v = xl[(size_t)r * L + e];
      a.xg[r * vstr + (size_t)lo * n2 + e] = v;
      if (r < nr) xx[(size_t)r * NX * n2 + (size_t)a.g.ceven[lo + e / n2] * n2 + e % n2] = v;
    }
    if (tx < NR) scl[tx] = 1.f;
    if (!meet()) return;
    auto xo = [&](int si, int r, int row) { return xx + (size_t)r * NX * n2 + (size_t)a.g.codd[lo + si] * n2 + row; };
    if (!phase_inv(bb, nr, [&](int si, int r, int row, cpx<float> s) {
          if (r < nr) *xo(si, r, row) = s;
        }))
      return;
    if (!products(
            K_ODD, [&](int si, int t, int r) { return a.xg + r * vstr + nbo[si * 8 + t]; },
            [&](int si, int r, int row, cpx<float> s) {
              if (r < nr) *xo(si, r, row) = *xo(si, r, row) - s;
            }))
      return;
    if (blockIdx.x == 0 && tx < nr) {
      if (a.iters) a.iters[r0 + tx] = tot[tx];
      if (a.iters_acc) atomicAdd(a.iters_acc, tot[tx]);
    }
    if (!meet()) return;
  }
}

template <int NR>
const void* wide_kernel(int ut) {
  switch (ut) {
    case 2: return (const void*)k_cgmres_wide<NR, 2>;
    case 3: return (const void*)k_cgmres_wide<NR, 3>;
    default: return (const void*)k_cgmres_wide<NR, 4>;
  }
}
const void* wide_fn(int NR, int n2) { return NR == 8 ? wide_kernel<8>(wide_ut(n2)) : wide_kernel<12>(wide_ut(n2)); }

}  // namespace

// NR: 12 right-hand sides in lockstep for nine or more, else 8; as many ring
// slots (at most eight) as fit beside two sites' vectors; one CTA per SM
WideChoice cgmres_wide_choose(int dev, const Geom& g, int n2, int m, int nrhs) {
  WideChoice c{};
  if (nrhs < 5 || n2 < 32 || n2 > 64) return c;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return c;
  const int NE = g.nb / 2, per = (NE + sms - 1) / sms;
  for (int NR = nrhs > 8 ? 12 : 8; NR >= 8; NR -= 4)
    for (int slots = RING_MAX; slots >= 2; --slots) {
      const WidePlan p = wide_plan(NR, n2, m, per, slots);
      int occ = 0;
      if (p.bytes > 226 * 1024 || raise_smem_limit(wide_fn(NR, n2), p.bytes) != cudaSuccess ||
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, wide_fn(NR, n2), TPB, p.bytes) != cudaSuccess || occ < 1) {
        cudaGetLastError();
        continue;
      }
      c.NR = NR;
      c.per = per;
      c.G = (NE + per - 1) / per;
      c.slots = slots;
      c.smem_bytes = p.bytes;
      c.work_bytes = al16(3 * (size_t)NR * NE * n2 * 8) + al16((size_t)(m + 2) * NR * c.G * 8) + 256 +
                     (size_t)c.G * wide_local(NR, n2, m, per);
      return c;
    }
  return c;
}

cudaError_t cgmres_wide_launch(const WideChoice& c, const Geom& g, const CoarseSolveArgs& ca, const float* b, float* x,
                               int nrhs, void* work, int* iters, int* iters_acc, int* status, cudaStream_t st) {
  WideArgs a{};
  a.g = g;
  a.Dc = reinterpret_cast<const cpx<float>*>(ca.Dc);
  a.Ainv = reinterpret_cast<const cpx<float>*>(ca.Ainv);
  a.AD = reinterpret_cast<const cpx<float>*>(ca.AinvD);
  a.n2 = 2 * ca.n;
  a.m = ca.restart;
  a.max_iter = ca.max_iter;
  a.nrhs = nrhs;
  a.NE = g.nb / 2;
  a.per = c.per;
  a.slots = c.slots;
  a.tol = (float)ca.tol;
  a.b = reinterpret_cast<const cpx<float>*>(b);
  a.x = reinterpret_cast<cpx<float>*>(x);
  const size_t vec = (size_t)c.NR * a.NE * a.n2;
  unsigned char* w = static_cast<unsigned char*>(work);
  a.wg = reinterpret_cast<cpx<float>*>(w);
  a.to = a.wg + vec;
  a.xg = a.to + vec;
  w += al16(3 * vec * 8);
  a.part = reinterpret_cast<float2*>(w);
  w += al16((size_t)(a.m + 2) * c.NR * c.G * 8);
  a.bar = reinterpret_cast<unsigned*>(w);
  a.lglob = w + 256;
  a.lstride = wide_local(c.NR, a.n2, a.m, c.per);
  a.iters = iters;
  a.iters_acc = iters_acc;
  a.status = status;
  a.spin_limit = ca.wait_limit;
  cudaError_t e = cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  e = raise_smem_limit(wide_fn(c.NR, a.n2), c.smem_bytes);
  if (e != cudaSuccess) return e;
  void* args[] = {&a};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c.G);
  cfg.blockDim = dim3(TPB);
  cfg.dynamicSmemBytes = c.smem_bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;   // all CTAs co-resident (grid barrier)
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, wide_fn(c.NR, a.n2), args);
}

}  // namespace ddamg
