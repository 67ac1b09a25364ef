// M psi in the W form (Eq. minFlopForm): one thread per site gathers the on-site spinor and the
// 26 neighbour spinors (x +- mu, x +- 2i, x +- i +- j) and multiplies them by the stored forward
// matrices at x, or by the backward ones obtained on the fly from the forward matrices stored at
// the neighbour (Eqs. conjugate and opp_diag_pre_mat: W^-_{mu,x} = gamma5 W^{+ dagger}_{mu,x-mu}
// gamma5 and so on).
//
// Spin handling.  With psi = (u, l) its upper and lower 2-spin halves, the nearest spatial hops are
// block diagonal in h+- = u +- l: the stored (D +- S) / 2 act on h+- and add to
//   acc+ = (out_u + out_l) / 2,   acc- = (out_u - out_l) / 2.
// W^0 is block diagonal in u -+ i l.  The temporal, two-hop and diagonal hops are [[A, B], [B, D]] with
// A, B, D spin matrices times one colour matrix, so they act on u and l as they are and add to the
// half outputs D_u = out_u / 2, D_l = out_l / 2 (the stored matrices hold the 1/2).  In these bases the
// 148 colour matrix-vector products per site are the only dense work.
//
// Precision R = double or float: loads, arithmetic and stores in R.  Fused epilogues feed the
// BiCGStab reductions (ok_reduce.cuh) without a second pass over the output.
#include "ok_hops.cuh"

#include <type_traits>

namespace okgb {

// ---------------------------------------------------------------------------- hop kernels
// acc0 += B00 h0 + B01 h1, acc1 += B10 h0 + B11 h1 (blocks at matrices m .. m+3 of `site`);
// DAG: acc0 += B00^dag h0 + B10^dag h1, acc1 += B01^dag h0 + B11^dag h1.
template <typename R, bool DAG>
__device__ __forceinline__ void block2(const cx<R>* __restrict__ W, int site, int m, const Half<R>& h, Half<R>& acc) {
  M3<R> b;
  b = wmat(W, site, m + 0);
  if (DAG) mdv_add(acc.v[0], b, h.v[0]); else mv_add(acc.v[0], b, h.v[0]);
  b = wmat(W, site, m + 1);
  if (DAG) mdv_add(acc.v[1], b, h.v[0]); else mv_add(acc.v[0], b, h.v[1]);
  b = wmat(W, site, m + 2);
  if (DAG) mdv_add(acc.v[0], b, h.v[1]); else mv_add(acc.v[1], b, h.v[0]);
  b = wmat(W, site, m + 3);
  if (DAG) mdv_add(acc.v[1], b, h.v[1]); else mv_add(acc.v[1], b, h.v[1]);
}

// Spatial nearest neighbours in direction I.
template <typename R, int I>
__device__ __forceinline__ void hop_spatial(const cx<R>* __restrict__ W, const cx<R>* __restrict__ psi, const int (&c)[4],
                                            const Geom& g, int s, Half<R>& ap, Half<R>& am) {
  constexpr int mp = M_WP + 8 * I, mm = mp + 4;
  Half<R> hp, hm;
  // forward: acc+ += (P+ / 2) h+, acc- += (P- / 2) h-, P at x
  gather_h<R, I == 0, I == 1, I == 2, 0>(psi, c, g, hp, hm);
  block2<R, false>(W, s, mp, hp, ap);
  block2<R, false>(W, s, mm, hm, am);
  // backward: acc+ += (P- / 2)^dag h+, acc- += (P+ / 2)^dag h-, P at x - I
  int n = gather_h<R, -(I == 0), -(I == 1), -(I == 2), 0>(psi, c, g, hp, hm);
  block2<R, true>(W, n, mm, hp, ap);
  block2<R, true>(W, n, mp, hm, am);
}

// The halves u, l of the neighbour at offset d, with the boundary sign.
template <typename R, int D0, int D1, int D2, int D3>
__device__ __forceinline__ int gather_ul(const cx<R>* __restrict__ psi, const int (&c)[4], const Geom& g, Half<R>& u, Half<R>& l) {
  bool neg;
  const int n = nbr_site<D0, D1, D2, D3>(c, g, neg);
  cx<R> v[12];
  load_spinor<R>(psi, n, v);
  if (neg) {
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = -v[k];
  }
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      u.v[s][a] = v[3 * s + a];
      l.v[s][a] = v[3 * (s + 2) + a];
    }
  return n;
}

// Temporal nearest neighbours on (u, l): W^+_4 = [[0, S], [S, -U]] at x, W^-_4 = [[-U^dag, -S^dag], [-S^dag, 0]]
// from x - t, S = [[s3, n1], [n2, -s3]].
template <typename R>
__device__ __forceinline__ void hop_time(const cx<R>* __restrict__ W, const cx<R>* __restrict__ psi, const int (&c)[4],
                                         const Geom& g, int s, Half<R>& du, Half<R>& dl) {
  Half<R> u, l;
  gather_ul<R, 0, 0, 0, 1>(psi, c, g, u, l);
  M3<R> A = wmat(W, s, M_UT);
  mv_sub(dl.v[0], A, l.v[0]); mv_sub(dl.v[1], A, l.v[1]);
  A = wmat(W, s, M_ST + 0);
  mv_add(du.v[0], A, l.v[0]); mv_sub(du.v[1], A, l.v[1]);
  mv_add(dl.v[0], A, u.v[0]); mv_sub(dl.v[1], A, u.v[1]);
  A = wmat(W, s, M_ST + 1);
  mv_add(du.v[0], A, l.v[1]); mv_add(dl.v[0], A, u.v[1]);
  A = wmat(W, s, M_ST + 2);
  mv_add(du.v[1], A, l.v[0]); mv_add(dl.v[1], A, u.v[0]);
  const int n = gather_ul<R, 0, 0, 0, -1>(psi, c, g, u, l);
  // S^dag = [[s3^dag, n2^dag], [n1^dag, -s3^dag]]
  A = wmat(W, n, M_UT);
  mdv_sub(du.v[0], A, u.v[0]); mdv_sub(du.v[1], A, u.v[1]);
  A = wmat(W, n, M_ST + 0);
  mdv_sub(du.v[0], A, l.v[0]); mdv_add(du.v[1], A, l.v[1]);
  mdv_sub(dl.v[0], A, u.v[0]); mdv_add(dl.v[1], A, u.v[1]);
  A = wmat(W, n, M_ST + 2);
  mdv_sub(du.v[0], A, l.v[1]); mdv_sub(dl.v[0], A, u.v[1]);
  A = wmat(W, n, M_ST + 1);
  mdv_sub(du.v[1], A, l.v[0]); mdv_sub(dl.v[1], A, u.v[0]);
}

// sigma_k y.
template <typename R>
__device__ __forceinline__ void sigma_half(int k, const Half<R>& y, Half<R>& s) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    s.v[0][a] = k == 0 ? y.v[1][a] : k == 1 ? tmi(y.v[1][a]) : y.v[0][a];
    s.v[1][a] = k == 0 ? y.v[0][a] : k == 1 ? ti(y.v[0][a]) : -y.v[1][a];
  }
}

// The spin part of a straight two-hop term, applied to the spinor before the colour matrix:
// a u + b sigma l = big (u + r sigma l) when |a| >= |b| (a_big), else big (r u + sigma l), |r| <= 1.  One
// multiply-add per component; the factor big multiplies the sum of the six terms once.
template <typename R> struct TwoHop { R big, r; bool a_big; };
template <typename R>
__device__ __forceinline__ Half<R> two_combine(const TwoHop<R>& q, R r, const Half<R>& u, const Half<R>& sl, bool minus) {
  Half<R> w;
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const cx<R> b = minus ? -sl.v[s][a] : sl.v[s][a];
      const cx<R> x = q.a_big ? u.v[s][a] : b, y = q.a_big ? b : u.v[s][a];
      w.v[s][a] = mk<R>(fma(r, y.re, x.re), fma(r, y.im, x.im));
    }
  return w;
}

// Straight two-hop neighbours x +- 2I: [[a, +-b sigma_i], [+-b sigma_i, a]] (x) V (at x), V^dag (at x - 2I),
// without the factor q.big.
template <typename R, int I>
__device__ __forceinline__ void hop_two(const cx<R>* __restrict__ W, const cx<R>* __restrict__ psi, const int (&c)[4],
                                        const Geom& g, int s, const TwoHop<R>& q, Half<R>& du, Half<R>& dl) {
  Half<R> u, l, t;
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    int n = s;
    if (f == 0) gather_ul<R, 2 * (I == 0), 2 * (I == 1), 2 * (I == 2), 0>(psi, c, g, u, l);
    else n = gather_ul<R, -2 * (I == 0), -2 * (I == 1), -2 * (I == 2), 0>(psi, c, g, u, l);
    const M3<R> V = wmat(W, n, M_VII + I);
    sigma_half(I, l, t);
    const Half<R> wu = two_combine(q, q.r, u, t, f == 1);
    sigma_half(I, u, t);
    const Half<R> wl = two_combine(q, q.r, l, t, f == 1);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      if (f == 0) { mv_add(du.v[p], V, wu.v[p]); mv_add(dl.v[p], V, wl.v[p]); }
      else { mdv_add(du.v[p], V, wu.v[p]); mdv_add(dl.v[p], V, wl.v[p]); }
    }
  }
}

// w = (sigma_I + SG sigma_J) y, I < J.
template <typename R, int I, int J, int SG>
__device__ __forceinline__ Half<R> sigma_sum(const Half<R>& y) {
  Half<R> w;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const cx<R> p = y.v[0][a], q = y.v[1][a];
    if constexpr (I == 0 && J == 1) {
      w.v[0][a] = SG > 0 ? q + tmi(q) : q + ti(q);
      w.v[1][a] = SG > 0 ? p + ti(p) : p + tmi(p);
    } else if constexpr (I == 0) {
      w.v[0][a] = SG > 0 ? q + p : q - p;
      w.v[1][a] = SG > 0 ? p - q : p + q;
    } else {
      w.v[0][a] = SG > 0 ? tmi(q) + p : tmi(q) - p;
      w.v[1][a] = SG > 0 ? ti(p) - q : ti(p) + q;
    }
  }
  return w;
}

// Diagonal neighbours of the pair (I, J), I < J, P = pair index: [[0, S], [S, 0]] with
// S = (s_I + s_J) (x) V from x+I+J and (s_I - s_J) (x) X from x+I-J, minus the adjoints from x-I-J, x-I+J.
template <typename R, int I, int J, int P>
__device__ __forceinline__ void hop_diag(const cx<R>* __restrict__ W, const cx<R>* __restrict__ psi, const int (&c)[4],
                                         const Geom& g, int s, Half<R>& du, Half<R>& dl) {
  constexpr int A0 = (I == 0) + (J == 0), A1 = (I == 1) + (J == 1), A2 = (I == 2) + (J == 2);
  constexpr int B0 = (I == 0) - (J == 0), B1 = (I == 1) - (J == 1), B2 = (I == 2) - (J == 2);
  Half<R> u, l, w;
  gather_ul<R, A0, A1, A2, 0>(psi, c, g, u, l);
  M3<R> V = wmat(W, s, M_VIJ + P);
  w = sigma_sum<R, I, J, 1>(l); mv_add(du.v[0], V, w.v[0]); mv_add(du.v[1], V, w.v[1]);
  w = sigma_sum<R, I, J, 1>(u); mv_add(dl.v[0], V, w.v[0]); mv_add(dl.v[1], V, w.v[1]);
  int n = gather_ul<R, -A0, -A1, -A2, 0>(psi, c, g, u, l);
  V = wmat(W, n, M_VIJ + P);
  w = sigma_sum<R, I, J, 1>(l); mdv_sub(du.v[0], V, w.v[0]); mdv_sub(du.v[1], V, w.v[1]);
  w = sigma_sum<R, I, J, 1>(u); mdv_sub(dl.v[0], V, w.v[0]); mdv_sub(dl.v[1], V, w.v[1]);
  gather_ul<R, B0, B1, B2, 0>(psi, c, g, u, l);
  V = wmat(W, s, M_XIJ + P);
  w = sigma_sum<R, I, J, -1>(l); mv_add(du.v[0], V, w.v[0]); mv_add(du.v[1], V, w.v[1]);
  w = sigma_sum<R, I, J, -1>(u); mv_add(dl.v[0], V, w.v[0]); mv_add(dl.v[1], V, w.v[1]);
  n = gather_ul<R, -B0, -B1, -B2, 0>(psi, c, g, u, l);
  V = wmat(W, n, M_XIJ + P);
  w = sigma_sum<R, I, J, -1>(l); mdv_sub(du.v[0], V, w.v[0]); mdv_sub(du.v[1], V, w.v[1]);
  w = sigma_sum<R, I, J, -1>(u); mdv_sub(dl.v[0], V, w.v[0]); mdv_sub(dl.v[1], V, w.v[1]);
}

// ---------------------------------------------------------------------------- the kernel
// One thread per site, for FP64: the FP64 pipe runs at 1/58 of the FP32 rate and bounds the kernel, so
// what counts is the number of FP64 operations.  5328 of them per site are the products'
// multiply-adds; acting on u and l wherever a hop allows leaves about 750 additions beside them, where
// the h+- basis throughout took about 1600 (16^3 x 32: 1625 us before, 1401 us now).
template <typename R, int EPI>
__global__ void __launch_bounds__(APPLY_THREADS) apply_kernel(const cx<R>* __restrict__ W, const cx<R>* __restrict__ psi,
                                                              cx<R>* __restrict__ out, Geom g, R c0q, TwoHop<R> two,
                                                              EpiArgs<R> ep) {
  if (ep.halt && *ep.halt) return;
  const int s = blockIdx.x * APPLY_THREADS + threadIdx.x;
  double red[3] = {0.0, 0.0, 0.0};
  if (s < g.V) {
    int c[4];
    {
      int r = s;
      c[0] = r % g.L[0]; r /= g.L[0];
      c[1] = r % g.L[1]; r /= g.L[1];
      c[2] = r % g.L[2]; c[3] = r / g.L[2];
    }
    Half<R> ap, am;
    {
      Half<R> du, dl;
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 3; ++k) du.v[q][k] = dl.v[q][k] = mk<R>(0, 0);
      hop_two<R, 0>(W, psi, c, g, s, two, du, dl);
      hop_two<R, 1>(W, psi, c, g, s, two, du, dl);
      hop_two<R, 2>(W, psi, c, g, s, two, du, dl);
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          du.v[q][k] = two.big * du.v[q][k];
          dl.v[q][k] = two.big * dl.v[q][k];
        }
      hop_time<R>(W, psi, c, g, s, du, dl);
      hop_diag<R, 0, 1, 0>(W, psi, c, g, s, du, dl);
      hop_diag<R, 0, 2, 1>(W, psi, c, g, s, du, dl);
      hop_diag<R, 1, 2, 2>(W, psi, c, g, s, du, dl);
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          ap.v[q][k] = du.v[q][k] + dl.v[q][k];
          am.v[q][k] = du.v[q][k] - dl.v[q][k];
        }
    }
    // on-site: a = u - i l, b = u + i l; A = Y+ a, B = Y- b; acc+- += (A + B) +- i (A - B)
    {
      cx<R> x0[12];
      load_spinor<R>(psi, s, x0);
      Half<R> a, b, A, B;
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          a.v[q][k] = x0[3 * q + k] - ti(x0[3 * (q + 2) + k]);
          b.v[q][k] = x0[3 * q + k] + ti(x0[3 * (q + 2) + k]);
          A.v[q][k] = c0q * a.v[q][k];
          B.v[q][k] = c0q * b.v[q][k];
        }
      M3<R> y = wmat(W, s, M_Y0P + 0);
      mv_add(A.v[0], y, a.v[0]); mv_sub(A.v[1], y, a.v[1]);
      y = wmat(W, s, M_Y0P + 1);
      mv_add(A.v[0], y, a.v[1]);
      y = wmat(W, s, M_Y0P + 2);
      mv_add(A.v[1], y, a.v[0]);
      y = wmat(W, s, M_Y0M + 0);
      mv_add(B.v[0], y, b.v[0]); mv_sub(B.v[1], y, b.v[1]);
      y = wmat(W, s, M_Y0M + 1);
      mv_add(B.v[0], y, b.v[1]);
      y = wmat(W, s, M_Y0M + 2);
      mv_add(B.v[1], y, b.v[0]);
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const cx<R> P = A.v[q][k] + B.v[q][k], Q = A.v[q][k] - B.v[q][k];
          ap.v[q][k] = ap.v[q][k] + (P + ti(Q));
          am.v[q][k] = am.v[q][k] + (P - ti(Q));
        }
    }
    hop_spatial<R, 0>(W, psi, c, g, s, ap, am);
    hop_spatial<R, 1>(W, psi, c, g, s, ap, am);
    hop_spatial<R, 2>(W, psi, c, g, s, ap, am);

    cx<R> o[12];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        o[3 * q + k] = ap.v[q][k] + am.v[q][k];
        o[3 * (q + 2) + k] = ap.v[q][k] - am.v[q][k];
      }
    if (EPI == EPI_RESID) {
      cx<R> bv[12];
      load_spinor<R>(ep.b, s, bv);
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        o[k] = bv[k] - o[k];
        const double ore = (double)o[k].re, oim = (double)o[k].im;
        const double bre = (double)bv[k].re, bim = (double)bv[k].im;
        red[0] += ore * ore + oim * oim;
        red[1] += bre * bre + bim * bim;
      }
    }
    store_spinor<R>(out, s, o);
    if constexpr (EPI == EPI_DOT) {
      cx<R> rh[12];
      load_spinor<R>(ep.rhat, s, rh);
      cx<R> d = mk<R>(0, 0);
#pragma unroll
      for (int k = 0; k < 12; ++k) d = fma_cj(rh[k], o[k], d);
      red[0] = d.re;
      red[1] = d.im;
    } else if constexpr (EPI == EPI_TS) {
      cx<R> x0[12];
      load_spinor<R>(psi, s, x0);
      cx<R> d = mk<R>(0, 0);
      R n2 = 0;
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        d = fma_cj(o[k], x0[k], d);
        n2 += o[k].re * o[k].re + o[k].im * o[k].im;
      }
      red[0] = d.re;
      red[1] = d.im;
      red[2] = n2;
    }
  }
  if (EPI == EPI_DOT || EPI == EPI_RESID) {
    double v2[2] = {red[0], red[1]};
    grid_reduce<2, APPLY_THREADS>(v2, ep.ra, ep.ticket);
  } else if (EPI == EPI_TS) {
    grid_reduce<3, APPLY_THREADS>(red, ep.ra, ep.ticket);
  }
}

// ============================================================================ staged split kernel
// FP32 arithmetic, the alternative to the pipelined kernel of ok_apply_pipe.cu that ok_autotune times
// (and ok_set_launch_shape pins).  A block of 128 threads covers 32 sites.  Warps 0-1 (thread pairs as in
// ok_pair.cuh) do the on-site term and the 13 forward hops, warps 2-3 the 13 backward hops of the same
// sites; the backward half hands its partial sums over through shared memory.
//
// The forward half reads its own tile's W record from shared memory.  The record of a 32-site tile is
// contiguous in the site-blocked layout, so the Tensor Memory Accelerator streams it (cp.async.bulk:
// one thread issues, an mbarrier counts the bytes) in NCHUNK chunks, one per group of hops, through
// OK_STAGES shared-memory slots.  The copy of chunk q + OK_STAGES is issued as soon as both forward
// warps are done with chunk q, across the block's tiles, so the DRAM stream of W is kept in flight by
// the copy engine instead of by registers.  The backward half gathers the neighbours' matrices with
// ordinary loads: the block that owns that tile streamed them shortly before, so they are L2 hits.
constexpr int SPLIT_THREADS = 128;
constexpr int SPLIT_SITES = 32;
static_assert(SPLIT_SITES == LANES, "a tile is one site block of the W layout");

#ifndef OK_STAGES
#define OK_STAGES 2
#endif
constexpr int NCHUNK = 7;     // W+t | W++ii | W++ij, W+-ij | W0 | W+x | W+y | W+z (the order of use)
constexpr int CHUNK_MAX = 8;  // matrices in the largest chunk
__device__ __forceinline__ int chunk_first(int c) {
  return c == 0 ? M_UT : c == 1 ? M_VII : c == 2 ? M_VIJ : c == 3 ? M_Y0P : M_WP + 8 * (c - 4);
}
__device__ __forceinline__ int chunk_count(int c) { return c == 0 ? 4 : c == 1 ? 3 : c == 2 || c == 3 ? 6 : 8; }
// A staged matrix occupies its own 9 x 32 elements plus 16 bytes: the two threads of a pair read
// matrices 4 apart, which this shift puts in different shared-memory banks.
template <typename WT> constexpr int smat_elems() { return 9 * LANES + 16 / (int)sizeof(cx<WT>); }
template <typename WT> constexpr int slot_elems() { return CHUNK_MAX * smat_elems<WT>(); }
template <typename WT> constexpr size_t staged_smem() { return (size_t)OK_STAGES * slot_elems<WT>() * sizeof(cx<WT>); }

// Bounded waits: a wait that has not completed after about 2^30 SM cycles (half a second) gives
// up, counts itself here and lets the kernel run to its end (the result is then invalid).
__device__ unsigned g_wait_timeouts;
// Failure injection for the bounded waits: extra bytes that block 0 declares for its first chunk
// (which its copies never deliver, so that wait runs out).  0 outside the failure-detection test.
__device__ unsigned g_stage_test_bytes;

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
// Waits until phase `parity` of `bar` completes or `limit` SM cycles pass; a wait that runs out
// is counted in g_wait_timeouts when `count` is set.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, long long limit = 1LL << 30,
                                          bool count = true) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > limit) {
      if (count) atomicAdd(&g_wait_timeouts, 1u);
      return false;
    }
  }
  return true;
}
// Global -> shared bulk copy completing on `bar` (both addresses 16-byte aligned, bytes % 16 == 0).
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}
// Named barrier 1 over the 64 forward threads (non-aligned form: lanes may arrive diverged).
__device__ __forceinline__ void fwd_bar_sync() { asm volatile("barrier.sync 1, 64;" ::: "memory"); }

// W source reading the tile's own matrices [m0, m0 + count) from a staged chunk.
template <typename WT> struct StagedW {
  const cx<WT>* slot;
  int m0;
  __device__ __forceinline__ M3<typename WReal<WT>::type> operator()(int site, int m) const {
    const cx<WT>* q = slot + (m - m0) * smat_elems<WT>();
    const int l = site & (LANES - 1);
    M3<typename WReal<WT>::type> a;
    if constexpr (std::is_same<WT, __half>::value) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const uint4 u = reinterpret_cast<const uint4*>(q)[k * LANES + l];
        a.e[4 * k] = widen(u.x);
        a.e[4 * k + 1] = widen(u.y);
        a.e[4 * k + 2] = widen(u.z);
        a.e[4 * k + 3] = widen(u.w);
      }
      a.e[8] = widen(reinterpret_cast<const unsigned*>(q)[8 * LANES + l]);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 f = reinterpret_cast<const float4*>(q)[k * LANES + l];
        a.e[2 * k] = mk<float>(f.x, f.y);
        a.e[2 * k + 1] = mk<float>(f.z, f.w);
      }
      const float2 f = reinterpret_cast<const float2*>(q)[8 * LANES + l];
      a.e[8] = mk<float>(f.x, f.y);
    }
    return a;
  }
};

#ifndef OK_TILE_SWIZZLE
#define OK_TILE_SWIZZLE 1
#endif
// First tile of this block; the block then walks every gridDim.x-th tile.  With OK_TILE_SWIZZLE,
// on a grid of G = k S blocks (S multiprocessors) the blocks b, b + S, b + 2S, ..., which a full
// persistent grid places on one SM, take consecutive tiles, so that their neighbour gathers (the
// rows above and below a tile) can share L1.
__device__ __forceinline__ int tile_rank(int sms) {
  const int b = blockIdx.x, G = gridDim.x;
  if (OK_TILE_SWIZZLE && sms > 0 && G % sms == 0) return (b % sms) * (G / sms) + b / sms;
  return b;
}

// Issue the copies of chunk q of this block (tile tile_rank + (q / NCHUNK) gridDim.x) into slot
// q % OK_STAGES.  Called by one thread.
template <typename WT>
__device__ __forceinline__ void issue_chunk(const cx<WT>* __restrict__ W, cx<WT>* stage, unsigned long long* full, int q,
                                            int rank) {
  const int tile = rank + (q / NCHUNK) * gridDim.x;
  const int c = q % NCHUNK, slot = q % OK_STAGES;
  const int m0 = chunk_first(c), n = chunk_count(c);
  constexpr unsigned mbytes = 9 * LANES * sizeof(cx<WT>);
  // The slot was last read through the generic proxy; order those reads before the async writes.
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  const unsigned extra = (q == 0 && blockIdx.x == 0) ? g_stage_test_bytes : 0u;
  mbar_expect_tx(&full[slot], n * mbytes + extra);
  for (int j = 0; j < n; ++j)
    bulk_g2s(stage + (size_t)slot * slot_elems<WT>() + (size_t)j * smat_elems<WT>(),
             W + ((size_t)tile * NMAT + m0 + j) * (9 * LANES), mbytes, &full[slot]);
}

template <typename WT>
__global__ void __launch_bounds__(SPLIT_THREADS, 4)
    apply_staged_kernel(const cx<WT>* __restrict__ W, const cx<float>* __restrict__ psi, cx<float>* __restrict__ out, Geom g,
                        float c0q, float a_ii, float b_ii, const int* halt) {
  using R = float;
  if (halt && *halt) return;
  // Persistent: each block walks tiles rank, rank + gridDim.x, ...  The hand-off buffer is
  // double-buffered by tile parity, so one barrier per tile suffices: the backward half writes
  // buffer k & 1 for tile k only after the barrier of tile k - 1, which the forward half passes
  // only after it has read buffer (k - 2) & 1 = k & 1.
  __shared__ cx<R> xch[2][64][6];
  __shared__ __align__(8) unsigned long long full[OK_STAGES];
  extern __shared__ __align__(128) unsigned char stage_raw[];
  cx<WT>* stage = reinterpret_cast<cx<WT>*>(stage_raw);
  const int half = threadIdx.x >> 6;  // warp-uniform: 0 forward, 1 backward
  const int t = threadIdx.x & 63;
  Pair pr;
  pr.p = t & 1;
  pr.mask = 3u << (threadIdx.x & 30);
  const GlobalW<WT> Wg{W};
  const int ntiles = (g.V + SPLIT_SITES - 1) / SPLIT_SITES;
  const int rank = tile_rank(g.sms);
  const int nq = rank < ntiles ? ((ntiles - 1 - rank) / (int)gridDim.x + 1) * NCHUNK : 0;
  int qc = 0;  // next chunk (forward warps)
  bool staged_ok = true;
  // Failure path: a wait that runs out sets stage_abort; no further chunk is issued, the block
  // finishes without waiting (its results are invalid and the timeout is counted), and thread 0
  // waits once more, briefly, for every chunk it issued but did not see arrive, so that no bulk
  // copy is in flight when the block exits.
  __shared__ int stage_abort;
  int issued = 0, unwaited_from = -1;
  if (threadIdx.x == 0) {
    for (int k = 0; k < OK_STAGES; ++k) mbar_init(&full[k], 1);
    mbar_fence_init();
    stage_abort = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (; issued < OK_STAGES && issued < nq; ++issued) issue_chunk<WT>(W, stage, full, issued, rank);
  // Wait for chunk qc; the forward warps then read it through a StagedW.
  auto chunk = [&](int m0) {
    const int slot = qc % OK_STAGES;
    if (staged_ok) {
      staged_ok = mbar_wait(&full[slot], (qc / OK_STAGES) & 1);
      if (!staged_ok) {
        stage_abort = 1;
        unwaited_from = qc;
      }
    }
    return StagedW<WT>{stage + (size_t)slot * slot_elems<WT>(), m0};
  };
  // Both forward warps are done with chunk qc: its slot takes chunk qc + OK_STAGES.
  auto release = [&]() {
    fwd_bar_sync();
    if (threadIdx.x == 0 && qc + OK_STAGES < nq && !stage_abort) {
      issue_chunk<WT>(W, stage, full, qc + OK_STAGES, rank);
      ++issued;
    }
    ++qc;
  };
  int kb = 0;
  for (int tile = rank; tile < ntiles; tile += gridDim.x, kb ^= 1) {
  const int s = tile * SPLIT_SITES + (t >> 1);
  const bool active = s < g.V;
  H6<R> acc;
#pragma unroll
  for (int qq = 0; qq < 2; ++qq)
#pragma unroll
    for (int k = 0; k < 3; ++k) acc.v[qq][k] = mk<R>(0, 0);
  int c[4] = {0, 0, 0, 0};
  if (active) {
    int r = s;
    c[0] = r % g.L[0]; r /= g.L[0];
    c[1] = r % g.L[1]; r /= g.L[1];
    c[2] = r % g.L[2]; c[3] = r / g.L[2];
  }
  if (half == 0) {
    Halves<R> hs;
    zero_halves(hs);
    // Every forward thread takes part in the waits and barriers, active or not.
    { auto w = chunk(M_UT); if (active) pair_time<R, true>(w, psi, c, g, s, pr, hs); release(); }
    {
      auto w = chunk(M_VII);
      if (active) {
        pair_two<R, 0, true>(w, psi, c, g, s, pr, a_ii, b_ii, hs);
        pair_two<R, 1, true>(w, psi, c, g, s, pr, a_ii, b_ii, hs);
        pair_two<R, 2, true>(w, psi, c, g, s, pr, a_ii, b_ii, hs);
      }
      release();
    }
    {
      auto w = chunk(M_VIJ);
      if (active) {
        pair_diag<R, 0, 1, 0, true>(w, psi, c, g, s, pr, hs);
        pair_diag<R, 0, 2, 1, true>(w, psi, c, g, s, pr, hs);
        pair_diag<R, 1, 2, 2, true>(w, psi, c, g, s, pr, hs);
        to_h(hs, pr, acc);
      }
      release();
    }
    { auto w = chunk(M_Y0P); if (active) pair_onsite<R>(w, psi, s, pr, c0q, acc); release(); }
    { auto w = chunk(M_WP + 0); if (active) pair_spatial<R, 0, true>(w, psi, c, g, s, pr, acc); release(); }
    { auto w = chunk(M_WP + 8); if (active) pair_spatial<R, 1, true>(w, psi, c, g, s, pr, acc); release(); }
    { auto w = chunk(M_WP + 16); if (active) pair_spatial<R, 2, true>(w, psi, c, g, s, pr, acc); release(); }
  } else if (active) {
    Halves<R> hs;
    zero_halves(hs);
    pair_time<R, false>(Wg, psi, c, g, s, pr, hs);
    pair_two<R, 0, false>(Wg, psi, c, g, s, pr, a_ii, b_ii, hs);
    pair_two<R, 1, false>(Wg, psi, c, g, s, pr, a_ii, b_ii, hs);
    pair_two<R, 2, false>(Wg, psi, c, g, s, pr, a_ii, b_ii, hs);
    pair_diag<R, 0, 1, 0, false>(Wg, psi, c, g, s, pr, hs);
    pair_diag<R, 0, 2, 1, false>(Wg, psi, c, g, s, pr, hs);
    pair_diag<R, 1, 2, 2, false>(Wg, psi, c, g, s, pr, hs);
    to_h(hs, pr, acc);
    pair_spatial<R, 0, false>(Wg, psi, c, g, s, pr, acc);
    pair_spatial<R, 1, false>(Wg, psi, c, g, s, pr, acc);
    pair_spatial<R, 2, false>(Wg, psi, c, g, s, pr, acc);
#pragma unroll
    for (int qq = 0; qq < 2; ++qq)
#pragma unroll
      for (int k = 0; k < 3; ++k) xch[kb][t][3 * qq + k] = acc.v[qq][k];
  }
  __syncthreads();
  if (half == 0 && active) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int k = 0; k < 3; ++k) acc.v[q][k] = acc.v[q][k] + xch[kb][t][3 * q + k];
    // out_u = acc+ + acc- (p = 0 writes it), out_l = acc+ - acc- (p = 1)
    H6<R> ap = partner(acc, pr.mask), o;
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int k = 0; k < 3; ++k) o.v[q][k] = pr.p ? ap.v[q][k] - acc.v[q][k] : acc.v[q][k] + ap.v[q][k];
    store_half<R>(out, s, pr.p, o);
  }
  }  // tiles
  if (threadIdx.x == 0 && unwaited_from >= 0)
    for (int q = unwaited_from; q < issued; ++q) mbar_wait(&full[q % OK_STAGES], (q / OK_STAGES) & 1, 1LL << 24, false);
}

// ---------------------------------------------------------------------------- launchers
// Persistent grid: as many blocks as fit on the device at once, at most one per tile.
template <typename WT>
static void launch_staged(const cx<WT>* W, const cx<float>* psi, cx<float>* out, const Geom& g, float c0q, float a, float b,
                          const int* halt, cudaStream_t st) {
  static int resident = 0;
  const size_t dyn = staged_smem<WT>();
  auto kern = apply_staged_kernel<WT>;
  if (resident == 0) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, SPLIT_THREADS, dyn) != cudaSuccess || nb < 1) nb = 1;
    resident = nb * sm_count();
  }
  const int tiles = grid_for(g.V, SPLIT_SITES);
  Geom gs = g;
  gs.sms = sm_count();
  kern<<<tiles < resident ? tiles : resident, SPLIT_THREADS, dyn, st>>>(W, psi, out, gs, c0q, a, b, halt);
}

// The staged form runs when the handle's tuning record says so (ok_autotune); the default, the
// pipelined kernel, reads W with ordinary loads (16^3 x 32: 92 us against 128 us staged, whose slots take
// L1 capacity that the neighbour spinors use).
template <typename WT>
static void launch_f32(const cx<WT>* W, const cx<float>* psi, cx<float>* out, const Geom& g, float c0q, float a, float b,
                       const int* halt, bool staged, cudaStream_t st) {
  if (staged) launch_staged<WT>(W, psi, out, g, c0q, a, b, halt, st);
  else launch_pipe<WT>(W, psi, out, g, c0q, a, b, halt, st);
}

static void launch_f64(const cx<double>* W, const cx<double>* psi, cx<double>* out, const Geom& g, const WScalars& sc, int epi,
                       const EpiArgs<double>& ep, cudaStream_t st) {
  const double a = sc.a_ii, b = sc.b_ii;
  const bool a_big = fabs(a) >= fabs(b);
  const double big = a_big ? a : b, small = a_big ? b : a;
  const TwoHop<double> two{big, big != 0.0 ? small / big : 0.0, a_big};
  const int nb = grid_for(g.V, APPLY_THREADS);
  switch (epi) {
    case EPI_NONE: apply_kernel<double, EPI_NONE><<<nb, APPLY_THREADS, 0, st>>>(W, psi, out, g, sc.c0q, two, ep); break;
    case EPI_DOT: apply_kernel<double, EPI_DOT><<<nb, APPLY_THREADS, 0, st>>>(W, psi, out, g, sc.c0q, two, ep); break;
    case EPI_TS: apply_kernel<double, EPI_TS><<<nb, APPLY_THREADS, 0, st>>>(W, psi, out, g, sc.c0q, two, ep); break;
    default: apply_kernel<double, EPI_RESID><<<nb, APPLY_THREADS, 0, st>>>(W, psi, out, g, sc.c0q, two, ep); break;
  }
}

template <typename R>
int launch_apply(const ok_W* Wh, const cx<R>* psi, cx<R>* out, int epi, const EpiArgs<R>& ep, cudaStream_t st) {
  const cx<R>* W = (const cx<R>*)(sizeof(R) == 8 ? Wh->W64 : Wh->W32);
  if (!W) return OK_EINVAL;
  // FP32: no fused epilogue (the inner products run in passes of their own, launch_dots)
  if (epi < EPI_NONE || epi > (sizeof(R) == 8 ? EPI_RESID : EPI_NONE)) return OK_EINVAL;
  static const char* n64[4] = {"apply_f64", "apply_f64_dot", "apply_f64_ts", "apply_f64_resid"};
  {
    TraceScope ts(sizeof(R) == 8 ? n64[epi] : "apply_f32", st);
    if constexpr (sizeof(R) == 8) launch_f64(W, psi, out, Wh->g, Wh->sc, epi, ep, st);
    else launch_f32<R>(W, psi, out, Wh->g, (R)Wh->sc.c0q, (R)Wh->sc.a_ii, (R)Wh->sc.b_ii, ep.halt, Wh->tune.staged[0] == 1, st);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

// Upper bound of the grid size of any apply variant (sizes the reduction partials).
int apply_blocks_needed(const ok_W* Wh) { return grid_for(Wh->g.V, SPLIT_SITES); }

// FP32 fields and arithmetic with the half-precision copy of W.
int launch_apply_w16(const ok_W* Wh, const cx<float>* psi, cx<float>* out, int epi, const EpiArgs<float>& ep, cudaStream_t st) {
  const cx<__half>* W = (const cx<__half>*)Wh->W16;
  if (!W || epi != EPI_NONE) return OK_EINVAL;
  {
    TraceScope ts("apply_w16", st);
    launch_f32<__half>(W, psi, out, Wh->g, (float)Wh->sc.c0q, (float)Wh->sc.a_ii, (float)Wh->sc.b_ii, ep.halt,
                       Wh->tune.staged[1] == 1, st);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

// Failure injection for the bounded waits (see g_stage_test_bytes).
int set_stage_test_bytes(unsigned bytes) {
  if (bytes % 16 != 0 || bytes > (1u << 16)) return OK_EINVAL;
  if (cudaMemcpyToSymbol(g_stage_test_bytes, &bytes, sizeof(unsigned)) != cudaSuccess) return OK_ECUDA;
  return OK_SUCCESS;
}

// Bounded waits that gave up since the last reset (see g_wait_timeouts).
int read_wait_timeouts(unsigned* n, bool reset) {
  if (cudaMemcpyFromSymbol(n, g_wait_timeouts, sizeof(unsigned)) != cudaSuccess) return OK_ECUDA;
  if (reset) {
    const unsigned zero = 0;
    if (cudaMemcpyToSymbol(g_wait_timeouts, &zero, sizeof(unsigned)) != cudaSuccess) return OK_ECUDA;
  }
  return OK_SUCCESS;
}

template int launch_apply<double>(const ok_W*, const cx<double>*, cx<double>*, int, const EpiArgs<double>&, cudaStream_t);
template int launch_apply<float>(const ok_W*, const cx<float>*, cx<float>*, int, const EpiArgs<float>&, cudaStream_t);

}  // namespace okgb
