// Device helpers shared by the apply kernels: W element loads, colour algebra, lattice
// geometry and the thread-pair hop functions (two threads per site, one per spin projection).
#pragma once

#include "ok_launch.cuh"

#include <type_traits>

namespace okgb {

// Matrix m of the site record of `site` (FP64: nine 16-byte loads; FP32: four and one of 8 bytes).
template <typename R>
__device__ __forceinline__ M3<R> wmat(const cx<R>* __restrict__ W, int site, int m) {
  const cx<R>* p = W + ((size_t)(site >> 5) * NMAT + m) * (9 * LANES);
  const int l = site & 31;
  M3<R> a;
  if constexpr (std::is_same<R, double>::value) {
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const double2 d = __ldg(reinterpret_cast<const double2*>(p) + e * LANES + l);
      a.e[e] = mk<R>(d.x, d.y);
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 d = __ldg(reinterpret_cast<const float4*>(p) + q * LANES + l);
      a.e[2 * q] = mk<R>(d.x, d.y);
      a.e[2 * q + 1] = mk<R>(d.z, d.w);
    }
    const float2 d = __ldg(reinterpret_cast<const float2*>(p) + 8 * LANES + l);
    a.e[8] = mk<R>(d.x, d.y);
  }
  return a;
}

// The same from the half-precision copy, widened to FP32 (two 16-byte loads and one of 4 bytes).
__device__ __forceinline__ cx<float> widen(unsigned u) {
  const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&u));
  return mk<float>(f.x, f.y);
}
__device__ __forceinline__ M3<float> wmat(const cx<__half>* __restrict__ W, int site, int m) {
  const cx<__half>* p = W + ((size_t)(site >> 5) * NMAT + m) * (9 * LANES);
  const int l = site & 31;
  M3<float> a;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(p) + q * LANES + l);
    a.e[4 * q] = widen(u.x);
    a.e[4 * q + 1] = widen(u.y);
    a.e[4 * q + 2] = widen(u.z);
    a.e[4 * q + 3] = widen(u.w);
  }
  a.e[8] = widen(__ldg(reinterpret_cast<const unsigned*>(p) + 8 * LANES + l));
  return a;
}

// Arithmetic type of a stored W element type (FP16 elements are widened to FP32).
template <typename WT> struct WReal { using type = WT; };
template <> struct WReal<__half> { using type = float; };

// W source reading any site's record from global memory.
template <typename WT> struct GlobalW {
  const cx<WT>* __restrict__ p;
  __device__ __forceinline__ M3<typename WReal<WT>::type> operator()(int site, int m) const { return wmat(p, site, m); }
};

// ---------------------------------------------------------------------------- colour algebra
// y += A v, y -= A v, y += A^dag v, y -= A^dag v
template <typename R> __device__ __forceinline__ void mv_add(cx<R> (&y)[3], const M3<R>& A, const cx<R> (&v)[3]) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) y[r] = fma_c(A.e[3 * r + c], v[c], y[r]);
}
template <typename R> __device__ __forceinline__ void mv_sub(cx<R> (&y)[3], const M3<R>& A, const cx<R> (&v)[3]) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) y[r] = fma_c(-A.e[3 * r + c], v[c], y[r]);
}
template <typename R> __device__ __forceinline__ void mdv_add(cx<R> (&y)[3], const M3<R>& A, const cx<R> (&v)[3]) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) y[r] = fma_cj(A.e[3 * c + r], v[c], y[r]);
}
template <typename R> __device__ __forceinline__ void mdv_sub(cx<R> (&y)[3], const M3<R>& A, const cx<R> (&v)[3]) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) y[r] = fma_cj(-A.e[3 * c + r], v[c], y[r]);
}
template <typename R> __device__ __forceinline__ void mv(cx<R> (&y)[3], const M3<R>& A, const cx<R> (&v)[3]) {
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    y[r] = A.e[3 * r] * v[0];
    y[r] = fma_c(A.e[3 * r + 1], v[1], y[r]);
    y[r] = fma_c(A.e[3 * r + 2], v[2], y[r]);
  }
}
template <typename R> __device__ __forceinline__ void mdv(cx<R> (&y)[3], const M3<R>& A, const cx<R> (&v)[3]) {
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    y[r] = cj(A.e[r]) * v[0];
    y[r] = fma_cj(A.e[3 + r], v[1], y[r]);
    y[r] = fma_cj(A.e[6 + r], v[2], y[r]);
  }
}

// ---------------------------------------------------------------------------- geometry
// Neighbour x + d with fermion boundary sign; |d_mu| <= 2.  The coordinate is wrapped by at most
// two conditional subtractions (two are needed only when L_mu < |d_mu|, on lattices of extent 1
// or 2); the sign flips once per wrap across an antiperiodic boundary (AP false: none that this hop can cross).
template <int D0, int D1, int D2, int D3, bool AP = true>
__device__ __forceinline__ int nbr_site(const int (&c)[4], const Geom& g, bool& neg) {
  const int d[4] = {D0, D1, D2, D3};
  int idx = 0;
  neg = false;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    int x = c[mu];
    if (d[mu] != 0) {
      const int L = g.L[mu];
      x += d[mu];
      int wraps = 0;
      if (d[mu] > 0) {
        if (x >= L) { x -= L; wraps = 1; if (x >= L) { x -= L; wraps = 2; } }
      } else {
        if (x < 0) { x += L; wraps = 1; if (x < 0) { x += L; wraps = 2; } }
      }
      if (AP && ((g.bcneg >> mu) & 1) && (wraps & 1)) neg = !neg;
    }
    idx += x * g.S[mu];
  }
  return idx;
}


// ============================================================================ two threads per site
// The pair (lanes 2k, 2k+1) shares one site.  Thread p = 0 loads the upper spin half u of every
// spinor it needs, thread p = 1 the lower half l.  Two bases are used:
//   * The temporal, two-hop and diagonal hops need no exchange between the threads.  W^+-_4,
//     W^{++}_ii and W^{++}_ij, W^{+-}_ij are [[A, B], [B, D]] on (u, l) with the same B both ways, so a
//     thread multiplies its own half only and adds the result to `same` (its own half of the output)
//     or to `cross` (the partner's half).  to_h exchanges the two sums once per site.
//   * The nearest spatial hops and W^0 work on h+- = u +- l (u -+ i l for W^0): p = 0 accumulates
//     acc+ with (D + S)/2 forward and (D - S)/2 backward, p = 1 acc- with the other two, so no matrix
//     is read twice; the partner's half arrives through one shuffle per component.
// With every hop in the h+- basis a site took 27 exchanges of 12 shuffles instead of 10, and each
// diagonal product 48 additions instead of 24: 48.4 M warp instructions for an FP32 application at
// 16^3 x 32, now 39 M.  Six right-hand sides at 12^3 x 24 in FP32 (apply_mrhs_kernel, whose unrolled code
// overflowed the instruction caches): 169 us before, 137 us now.

template <typename R> struct H6 { cx<R> v[2][3]; };

template <typename R>
__device__ __forceinline__ void load_half(const cx<R>* __restrict__ psi, int site, int p, H6<R>& h) {
  if constexpr (sizeof(R) == 8) {
    const double2* q = reinterpret_cast<const double2*>(psi) + (size_t)site * 12 + 6 * p;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      double2 d = __ldg(q + k);
      h.v[k / 3][k % 3] = mk<R>(d.x, d.y);
    }
  } else {
    const float4* q = reinterpret_cast<const float4*>(psi) + (size_t)site * 6 + 3 * p;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float4 d = __ldg(q + k);
      h.v[(2 * k) / 3][(2 * k) % 3] = mk<R>(d.x, d.y);
      h.v[(2 * k + 1) / 3][(2 * k + 1) % 3] = mk<R>(d.z, d.w);
    }
  }
}

template <typename R>
__device__ __forceinline__ void store_half(cx<R>* __restrict__ out, int site, int p, const H6<R>& h) {
  if constexpr (sizeof(R) == 8) {
    double2* q = reinterpret_cast<double2*>(out) + (size_t)site * 12 + 6 * p;
#pragma unroll
    for (int k = 0; k < 6; ++k) q[k] = make_double2(h.v[k / 3][k % 3].re, h.v[k / 3][k % 3].im);
  } else {
    float4* q = reinterpret_cast<float4*>(out) + (size_t)site * 6 + 3 * p;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const cx<R>& a = h.v[(2 * k) / 3][(2 * k) % 3];
      const cx<R>& b = h.v[(2 * k + 1) / 3][(2 * k + 1) % 3];
      q[k] = make_float4(a.re, a.im, b.re, b.im);
    }
  }
}

template <typename R>
__device__ __forceinline__ H6<R> partner(const H6<R>& h, unsigned mask) {
  H6<R> o;
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      o.v[s][a].re = __shfl_xor_sync(mask, h.v[s][a].re, 1);
      o.v[s][a].im = __shfl_xor_sync(mask, h.v[s][a].im, 1);
    }
  return o;
}

struct Pair {
  int p;          // 0: acc+ thread, 1: acc- thread
  unsigned mask;  // the two lanes of the pair
};

// The thread's own half of the neighbour at offset D, with the boundary sign (a multiplication, not a
// branch: the hops stay one basic block, so the loads of the next hop can be issued early).
template <typename R, int D0, int D1, int D2, int D3>
__device__ __forceinline__ int gather_mine(const cx<R>* __restrict__ psi, const int (&c)[4], const Geom& g, const Pair& pr,
                                           H6<R>& mine) {
  bool neg;
  const int n = nbr_site<D0, D1, D2, D3>(c, g, neg);
  load_half<R>(psi, n, pr.p, mine);
  const R sg = neg ? R(-1) : R(1);
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) mine.v[s][a] = sg * mine.v[s][a];
  return n;
}

// h+ = u + l (p = 0) or h- = u - l (p = 1) from the threads' halves.
template <typename R>
__device__ __forceinline__ void halves_to_h(const H6<R>& mine, const Pair& pr, H6<R>& h) {
  const H6<R> oth = partner(mine, pr.mask);
  const R sg = pr.p ? R(-1) : R(1);
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      h.v[s][a].re = fma(sg, mine.v[s][a].re, oth.v[s][a].re);
      h.v[s][a].im = fma(sg, mine.v[s][a].im, oth.v[s][a].im);
    }
}

// h+ (p = 0) or h- (p = 1) of the neighbour at offset D.
template <typename R, int D0, int D1, int D2, int D3>
__device__ __forceinline__ int gather_pair(const cx<R>* __restrict__ psi, const int (&c)[4], const Geom& g, const Pair& pr,
                                           H6<R>& h) {
  H6<R> mine;
  const int n = gather_mine<R, D0, D1, D2, D3>(psi, c, g, pr, mine);
  halves_to_h(mine, pr, h);
  return n;
}

// Sums of the hops without exchange: same goes to the thread's own half of the output, cross to the
// partner's.
template <typename R> struct Halves { H6<R> same, cross; };

template <typename R>
__device__ __forceinline__ void zero_halves(Halves<R>& d) {
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) d.same.v[s][a] = d.cross.v[s][a] = mk<R>(0, 0);
}

// acc+ += D_u + D_l (p = 0), acc- += D_u - D_l (p = 1) of the half outputs D = same + partner's cross.
template <typename R>
__device__ __forceinline__ void to_h(const Halves<R>& d, const Pair& pr, H6<R>& acc) {
  const H6<R> oc = partner(d.cross, pr.mask);
  H6<R> m;
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) m.v[s][a] = d.same.v[s][a] + oc.v[s][a];
  H6<R> h;
  halves_to_h(m, pr, h);
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) acc.v[s][a] = acc.v[s][a] + h.v[s][a];
}

template <typename R, bool DAG, typename WS>
__device__ __forceinline__ void block2h(const WS& W, int site, int m, const H6<R>& h, H6<R>& acc) {
  M3<R> b;
  b = W(site, m + 0);
  if (DAG) mdv_add(acc.v[0], b, h.v[0]); else mv_add(acc.v[0], b, h.v[0]);
  b = W(site, m + 1);
  if (DAG) mdv_add(acc.v[1], b, h.v[0]); else mv_add(acc.v[0], b, h.v[1]);
  b = W(site, m + 2);
  if (DAG) mdv_add(acc.v[0], b, h.v[1]); else mv_add(acc.v[1], b, h.v[0]);
  b = W(site, m + 3);
  if (DAG) mdv_add(acc.v[1], b, h.v[1]); else mv_add(acc.v[1], b, h.v[1]);
}

template <typename R>
__device__ __forceinline__ void add_sigma_h(H6<R>& acc, int k, const H6<R>& y, R f) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (k == 0) {
      acc.v[0][a] = acc.v[0][a] + f * y.v[1][a];
      acc.v[1][a] = acc.v[1][a] + f * y.v[0][a];
    } else if (k == 1) {
      acc.v[0][a] = acc.v[0][a] + f * tmi(y.v[1][a]);
      acc.v[1][a] = acc.v[1][a] + f * ti(y.v[0][a]);
    } else {
      acc.v[0][a] = acc.v[0][a] + f * y.v[0][a];
      acc.v[1][a] = acc.v[1][a] - f * y.v[1][a];
    }
  }
}

template <typename R, bool DAG>
__device__ __forceinline__ void colour2h(H6<R>& y, const M3<R>& V, const H6<R>& h) {
  if (DAG) { mdv(y.v[0], V, h.v[0]); mdv(y.v[1], V, h.v[1]); }
  else { mv(y.v[0], V, h.v[0]); mv(y.v[1], V, h.v[1]); }
}

// Each hop function does the forward (FWD) or the backward half of its part of the stencil; the two
// run in different warps.
template <typename R, int I, bool FWD, typename WS>
__device__ __forceinline__ void pair_spatial(const WS& W, const cx<R>* __restrict__ psi, const int (&c)[4],
                                             const Geom& g, int s, const Pair& pr, H6<R>& acc) {
  constexpr int base = M_WP + 8 * I, f = FWD ? 1 : -1;
  H6<R> h;
  const int n = gather_pair<R, f * (I == 0), f * (I == 1), f * (I == 2), 0>(psi, c, g, pr, h);
  if constexpr (FWD) block2h<R, false>(W, s, base + 4 * pr.p, h, acc);
  else block2h<R, true>(W, n, base + 4 * (1 - pr.p), h, acc);
}

// m, or zero for the thread whose half a term does not act on (selects instead of a branch).
template <typename R>
__device__ __forceinline__ void only(H6<R>& m, bool mine) {
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) m.v[s][a] = mk<R>(mine ? m.v[s][a].re : R(0), mine ? m.v[s][a].im : R(0));
}

// On (u, l): W^+_4 = [[0, S], [S, -U]] with the matrices at x, W^-_4 = [[-U^dag, -S^dag], [-S^dag, 0]]
// with those at x - t (halves stored); S = [[s3, n1], [n2, -s3]].
template <typename R, bool FWD, typename WS>
__device__ __forceinline__ void pair_time(const WS& W, const cx<R>* __restrict__ psi, const int (&c)[4],
                                          const Geom& g, int s, const Pair& pr, Halves<R>& d) {
  H6<R> m;
  if constexpr (FWD) {
    gather_mine<R, 0, 0, 0, 1>(psi, c, g, pr, m);
    M3<R> A = W(s, M_ST + 0);
    mv_add(d.cross.v[0], A, m.v[0]);
    mv_sub(d.cross.v[1], A, m.v[1]);
    A = W(s, M_ST + 1);
    mv_add(d.cross.v[0], A, m.v[1]);
    A = W(s, M_ST + 2);
    mv_add(d.cross.v[1], A, m.v[0]);
    only(m, pr.p == 1);  // U multiplies l
    A = W(s, M_UT);
    mv_sub(d.same.v[0], A, m.v[0]);
    mv_sub(d.same.v[1], A, m.v[1]);
  } else {
    // S^dag = [[s3^dag, n2^dag], [n1^dag, -s3^dag]]
    const int n = gather_mine<R, 0, 0, 0, -1>(psi, c, g, pr, m);
    M3<R> A = W(n, M_ST + 0);
    mdv_sub(d.cross.v[0], A, m.v[0]);
    mdv_add(d.cross.v[1], A, m.v[1]);
    A = W(n, M_ST + 2);
    mdv_sub(d.cross.v[0], A, m.v[1]);
    A = W(n, M_ST + 1);
    mdv_sub(d.cross.v[1], A, m.v[0]);
    only(m, pr.p == 0);  // U^dag multiplies u
    A = W(n, M_UT);
    mdv_sub(d.same.v[0], A, m.v[0]);
    mdv_sub(d.same.v[1], A, m.v[1]);
  }
}

template <typename R>
__device__ __forceinline__ void add_scaled_h(H6<R>& acc, R a, const H6<R>& y) {
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      acc.v[q][k].re = fma(a, y.v[q][k].re, acc.v[q][k].re);
      acc.v[q][k].im = fma(a, y.v[q][k].im, acc.v[q][k].im);
    }
}

// W^{++}_ii = [[a, b sigma_i], [b sigma_i, a]] (x) V forward, [[a, -b sigma_i], [-b sigma_i, a]] (x) V^dag backward.
template <typename R, int I, bool FWD, typename WS>
__device__ __forceinline__ void pair_two(const WS& W, const cx<R>* __restrict__ psi, const int (&c)[4],
                                         const Geom& g, int s, const Pair& pr, R a, R b, Halves<R>& d) {
  constexpr int f = FWD ? 1 : -1;
  H6<R> m, y;
  const int n = gather_mine<R, 2 * f * (I == 0), 2 * f * (I == 1), 2 * f * (I == 2), 0>(psi, c, g, pr, m);
  const M3<R> V = W(FWD ? s : n, M_VII + I);
  colour2h<R, !FWD>(y, V, m);
  add_scaled_h(d.same, a, y);
  add_sigma_h(d.cross, I, y, FWD ? b : -b);
}

// s = (sigma_I + SG sigma_J) m, I < J.
template <typename R, int I, int J, int SG>
__device__ __forceinline__ void sigma_pair(const H6<R>& m, H6<R>& s) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const cx<R> x = m.v[0][a], y = m.v[1][a];
    if constexpr (I == 0 && J == 1) {       // [[0, 1 - SG i], [1 + SG i, 0]]
      s.v[0][a] = SG > 0 ? y + tmi(y) : y + ti(y);
      s.v[1][a] = SG > 0 ? x + ti(x) : x + tmi(x);
    } else if constexpr (I == 0) {          // [[SG, 1], [1, -SG]]
      s.v[0][a] = SG > 0 ? y + x : y - x;
      s.v[1][a] = SG > 0 ? x - y : x + y;
    } else {                                // [[SG, -i], [i, -SG]]
      s.v[0][a] = SG > 0 ? tmi(y) + x : tmi(y) - x;
      s.v[1][a] = SG > 0 ? ti(x) - y : ti(x) + y;
    }
  }
}

template <typename R, bool DAG>
__device__ __forceinline__ void colour2h_acc(H6<R>& y, const M3<R>& V, const H6<R>& h) {
  if (DAG) { mdv_sub(y.v[0], V, h.v[0]); mdv_sub(y.v[1], V, h.v[1]); }
  else { mv_add(y.v[0], V, h.v[0]); mv_add(y.v[1], V, h.v[1]); }
}

// Diagonal pair (I, J): [[0, S], [S, 0]] with S = (s_I + s_J) (x) V from x+I+J and (s_I - s_J) (x) X from
// x+I-J (forward), minus their adjoints from x-I-J and x-I+J (backward).
template <typename R, int I, int J, int P, bool FWD, typename WS>
__device__ __forceinline__ void pair_diag(const WS& W, const cx<R>* __restrict__ psi, const int (&c)[4],
                                          const Geom& g, int s, const Pair& pr, Halves<R>& d) {
  constexpr int f = FWD ? 1 : -1;
  constexpr int A0 = (I == 0) + (J == 0), A1 = (I == 1) + (J == 1), A2 = (I == 2) + (J == 2);
  constexpr int B0 = (I == 0) - (J == 0), B1 = (I == 1) - (J == 1), B2 = (I == 2) - (J == 2);
  H6<R> m, y;
  int n = gather_mine<R, f * A0, f * A1, f * A2, 0>(psi, c, g, pr, m);
  sigma_pair<R, I, J, 1>(m, y);
  M3<R> V = W(FWD ? s : n, M_VIJ + P);
  colour2h_acc<R, !FWD>(d.cross, V, y);
  n = gather_mine<R, f * B0, f * B1, f * B2, 0>(psi, c, g, pr, m);
  sigma_pair<R, I, J, -1>(m, y);
  V = W(FWD ? s : n, M_XIJ + P);
  colour2h_acc<R, !FWD>(d.cross, V, y);
}

// On-site term W^0 psi_x (both halves of the pair): p = 0 forms A = Y+ (u - i l), p = 1 forms
// B = Y- (u + i l); acc += (A + B) + i (A - B) for p = 0 and (A + B) - i (A - B) for p = 1.
template <typename R, typename WS>
__device__ __forceinline__ void pair_onsite(const WS& W, const cx<R>* __restrict__ psi, int s, const Pair& pr, R c0q,
                                            H6<R>& acc) {
  H6<R> mine, oth, v, Rm;
  load_half<R>(psi, s, pr.p, mine);
  oth = partner(mine, pr.mask);
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      cx<R> u = pr.p ? oth.v[q][k] : mine.v[q][k];
      cx<R> l = pr.p ? mine.v[q][k] : oth.v[q][k];
      v.v[q][k] = pr.p ? u + ti(l) : u - ti(l);
      Rm.v[q][k] = c0q * v.v[q][k];
    }
  const int m0 = pr.p ? M_Y0M : M_Y0P;
  M3<R> y = W(s, m0 + 0);
  mv_add(Rm.v[0], y, v.v[0]); mv_sub(Rm.v[1], y, v.v[1]);
  y = W(s, m0 + 1);
  mv_add(Rm.v[0], y, v.v[1]);
  y = W(s, m0 + 2);
  mv_add(Rm.v[1], y, v.v[0]);
  H6<R> Rp = partner(Rm, pr.mask);
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 3; ++k)
      acc.v[q][k] = acc.v[q][k] + ((Rm.v[q][k] + Rp.v[q][k]) + ti(Rm.v[q][k] - Rp.v[q][k]));
}

}  // namespace okgb
