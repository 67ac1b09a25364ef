// FP64-accurate M psi on the FP32 pipes: double-float W (OK_W_DF64) and fields.
//
// A block takes a 32-site tile of W; its four warps take the four sums per site of ok_dd_entries.cuh, lane
// = site, and walk their 37 products with one compact loop body: gather one or two spin components of
// the neighbour, combine them, multiply by the matrix, add to the warp's one sum.  All of a warp's
// lanes walk the same entry, so the table reads and the branches on an entry's fields are uniform.
//
// Double-float: a row of a product sums six real products with TwoProd and TwoSum, deferring the
// renormalisation to the addition of the row to the sum (Joldes, Muller, Popescu, ACM TOMS 44 (2017),
// the building blocks of ok_internal.cuh).  Real and imaginary parts go through the same sequence
// side by side, as the two halves of packed FP32 operations.
//
// What bounds it: the FP32 pipe, about 520 slots of packed operations per product and lane.  One thread
// per site with four sums, up to two destinations and a scalar per product, and scalar operations took
// 120 k instructions per site (issue 72 % busy): 602 us at 16^3 x 32 with x's conversion, now 475 us, and
// the error against 64 bits 3.2e-15 instead of 8.9e-15 (fewer sums).
#include "ok_dd.cuh"
#include "ok_dd_entries.cuh"
#include "ok_split.cuh"

namespace okgb {

namespace {

constexpr int DD_THREADS = 128;
#ifndef OK_DD_MINB
#define OK_DD_MINB 5   // 475 us at 16^3 x 32 with x's conversion; 482 and 516 us at 4 and 3 blocks per SM
#endif

using namespace ddent;

// ---------------------------------------------------------------------------- packed double-float
// A complex double-float: hi = (re.hi, im.hi), lo = (re.lo, im.lo).
struct P2 {
  float2 hi, lo;
};
__device__ __forceinline__ float2 f2(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a - b (one rounding: the product by -1 is exact)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ P2 norm2(float2 s, float2 e) {
  P2 r;
  r.hi = add2(s, e);
  r.lo = sub2(e, sub2(r.hi, s));
  return r;
}
// a + (s, e), e the unnormalised low part
__device__ __forceinline__ P2 add_row(P2 a, float2 s, float2 e) {
  const float2 t = add2(a.hi, s), bb = sub2(t, a.hi);
  float2 r = add2(sub2(a.hi, sub2(t, bb)), sub2(s, bb));
  r = add2(r, add2(a.lo, e));
  return norm2(t, r);
}
__device__ __forceinline__ P2 add(P2 a, P2 b) { return add_row(a, b.hi, b.lo); }
__device__ __forceinline__ float2 flip2(float2 a, unsigned mx, unsigned my) {
  return f2(__uint_as_float(__float_as_uint(a.x) ^ mx), __uint_as_float(__float_as_uint(a.y) ^ my));
}
__device__ __forceinline__ P2 flip(P2 a, unsigned mx, unsigned my) { return P2{flip2(a.hi, mx, my), flip2(a.lo, mx, my)}; }
// i^k a (exact)
__device__ __forceinline__ P2 times_i(P2 a, int k) {
  const bool sw = k & 1;
  const unsigned mr = ((k + 1) & 2) ? 0x80000000u : 0u, mi = (k & 2) ? 0x80000000u : 0u;
  const P2 b = sw ? P2{f2(a.hi.y, a.hi.x), f2(a.lo.y, a.lo.x)} : a;
  return flip(b, mr, mi);
}
// a times the real double-float f
__device__ __forceinline__ P2 scale(P2 a, dd f) {
  const float2 fh = f2(f.hi, f.hi), fl = f2(f.lo, f.lo), q = __fmul2_rn(a.hi, f2(-f.hi, -f.hi));  // -product
  float2 e = __ffma2_rn(a.hi, fh, q);
  e = __ffma2_rn(a.hi, fl, e);
  e = __ffma2_rn(a.lo, fh, e);
  return norm2(f2(-q.x, -q.y), e);
}
// (s, t) = or += a b by components: q is the negated product of the high parts (na = -a.hi).
__device__ __forceinline__ void prod_first(float2& s, float2& t, float2 ah, float2 na, float2 al, float2 bh, float2 bl) {
  s = __fmul2_rn(ah, bh);
  const float2 q = __fmul2_rn(na, bh);
  t = __ffma2_rn(ah, bh, q);
  t = __ffma2_rn(ah, bl, t);
  t = __ffma2_rn(al, bh, t);
}
__device__ __forceinline__ void prod_acc(float2& s, float2& t, float2 ah, float2 na, float2 al, float2 bh, float2 bl) {
  const float2 q = __fmul2_rn(na, bh);
  float2 e = __ffma2_rn(ah, bh, q);
  e = __ffma2_rn(ah, bl, e);
  e = __ffma2_rn(al, bh, e);
  const float2 s2 = sub2(s, q), bb = sub2(s2, s);
  t = add2(t, sub2(sub2(s, sub2(s2, bb)), add2(q, bb)));  // (s - (s2 - bb)) + (p - bb)
  t = add2(t, e);
  s = s2;
}

// Neighbour x + d with the fermion sign of every wrap across an antiperiodic boundary (|d_mu| <= 2, so at
// most two wraps per direction).
__device__ __forceinline__ int nbr_of(const int (&c)[4], const Geom& g, const signed char* d, bool& neg) {
  int n = 0;
  neg = false;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    const int L = g.L[mu];
    int x = c[mu] + d[mu];
    int wraps = 0;
    if (x >= L) { x -= L; wraps = 1; if (x >= L) { x -= L; wraps = 2; } }
    if (x < 0) { x += L; wraps = 1; if (x < 0) { x += L; wraps = 2; } }
    if (((g.bcneg >> mu) & 1) && (wraps & 1)) neg = !neg;
    n += x * g.S[mu];
  }
  return n;
}

// Fields of the apply: per block of 32 sites, component k = 3 spin + colour of lane l is the 16-byte word
// (re.hi, im.hi, re.lo, im.lo) at (blk * 12 + k) * 32 + l, so a warp's gather of one component is a run of
// consecutive words.
__device__ __forceinline__ const float4* field(const float4* psi, int n, int spin) {
  return psi + ((size_t)(n >> 5) * 12 + 3 * spin) * LANES + (n & 31);
}
__device__ __forceinline__ P2 unpack(float4 v) { return P2{f2(v.x, v.y), f2(v.z, v.w)}; }

// ---------------------------------------------------------------------------- the kernel
template <int EPI>
__global__ void __launch_bounds__(DD_THREADS, OK_DD_MINB)
    apply_dd_kernel(const float4* __restrict__ W, const float4* __restrict__ psi, double2* __restrict__ out, Geom g,
                    dd c0q4, dd two_big, dd two_r, int a_big, const double2* __restrict__ rhs, RedArgs ra, unsigned* ticket,
                    const int* halt, const __grid_constant__ Table tab) {
  if (EPI != EPI_NONE && halt && *halt) return;
  __shared__ float4 sh[2][4][3][LANES];   // the S and O sums of the four warps
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int s0 = blockIdx.x * LANES + lane;
  const int s = s0 < g.V ? s0 : g.V - 1;   // lanes past the last site repeat it and store nothing
  int c[4];
  {
    int r = s;
    c[0] = r % g.L[0]; r /= g.L[0];
    c[1] = r % g.L[1]; r /= g.L[1];
    c[2] = r % g.L[2]; c[3] = r / g.L[2];
  }
  P2 acc[3], D[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) acc[k] = P2{f2(0.f, 0.f), f2(0.f, 0.f)};
  int hop = -1, n = s;
  bool neg = false;
#pragma unroll 1
  for (int i = 0; i < N_ALL; ++i) {
    const Entry E = tab.e[w][i];
    if (E.hop != hop) {
      hop = E.hop;
      n = nbr_of(c, g, tab.d[hop], neg);
    }
    const bool adj = E.flags & 1;
    const int site = adj ? n : s;
    const float4* wp = W + ((size_t)(site >> 5) * NMAT + E.m) * (9 * LANES) + (site & 31);
    const int unit = E.src >> 4;
    float4 ve[9];
    // the matrix in the order of use: row r's elements (r, c), of the adjoint (c, r)
    const int sr = adj ? 1 : 3, sc = adj ? 3 : 1;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int k = 0; k < 3; ++k) ve[3 * r + k] = __ldg(wp + (r * sr + k * sc) * LANES);
    P2 v[3];
    {
      const float4* p1 = field(psi, n, E.src & 3);
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] = unpack(__ldg(p1 + k * LANES));
      if (unit) {
        const float4* p2 = field(psi, n, (E.src >> 2) & 3);
        P2 y[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) y[k] = times_i(unpack(__ldg(p2 + k * LANES)), unit - 1);
        if (i < N_TWO) {
          // a psi_s1 + b y = two_big (psi_s1 + r y), or two_big (r psi_s1 + y) when b is the larger
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            if (a_big) y[k] = scale(y[k], two_r);
            else v[k] = scale(v[k], two_r);
          }
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) v[k] = add(v[k], y[k]);
      }
      const unsigned m = (neg != ((E.flags & 2) != 0)) ? 0x80000000u : 0u;
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] = flip(v[k], m, m);
    }
    const unsigned cj = adj ? 0x80000000u : 0u;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      float2 S, T;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float4 e = ve[3 * r + k];   // (re.hi, re.lo, im.hi, im.lo)
        const float ih = __uint_as_float(__float_as_uint(e.z) ^ cj), il = __uint_as_float(__float_as_uint(e.w) ^ cj);
        const float2 ah = f2(e.x, e.x), an = f2(-e.x, -e.x), al = f2(e.y, e.y);
        if (k == 0) prod_first(S, T, ah, an, al, v[k].hi, v[k].lo);
        else prod_acc(S, T, ah, an, al, v[k].hi, v[k].lo);
        // i im times (re, im) = im times (-im, re)
        prod_acc(S, T, f2(-ih, ih), f2(ih, -ih), f2(-il, il), f2(v[k].hi.y, v[k].hi.x), f2(v[k].lo.y, v[k].lo.x));
      }
      acc[r] = add_row(acc[r], S, T);
    }
    if (i == N_TWO - 1) {
#pragma unroll
      for (int k = 0; k < 3; ++k) acc[k] = scale(acc[k], two_big);
    } else if (i == N_D - 1) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        D[k] = acc[k];
        acc[k] = P2{f2(0.f, 0.f), f2(0.f, 0.f)};
      }
    } else if (i == N_S - 1) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        sh[0][w][k][lane] = make_float4(acc[k].hi.x, acc[k].hi.y, acc[k].lo.x, acc[k].lo.y);
        acc[k] = P2{f2(0.f, 0.f), f2(0.f, 0.f)};
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) sh[1][w][k][lane] = make_float4(acc[k].hi.x, acc[k].hi.y, acc[k].lo.x, acc[k].lo.y);
  __syncthreads();
  // out_u = S+ + S- + 2 D + 2 (A + B) + 4 c0q u,  out_l = S+ - S- + 2 D + 2 i (A - B) + 4 c0q l
  double red[2] = {0.0, 0.0};
  const int h = w >> 1, q = w & 1;
  const float4* pp = field(psi, s, w);
  double2* op = out + (size_t)s * 12 + 3 * w;
  const double2* bp = EPI == EPI_RESID ? rhs + (size_t)s * 12 + 3 * w : nullptr;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const unsigned m = h ? 0x80000000u : 0u;
    const P2 S = add(unpack(sh[0][q][k][lane]), flip(unpack(sh[0][2 + q][k][lane]), m, m));
    P2 O = add(unpack(sh[1][q][k][lane]), flip(unpack(sh[1][2 + q][k][lane]), m, m));
    if (h) O = times_i(O, 1);
    P2 X = add(D[k], O);
    X = P2{add2(X.hi, X.hi), add2(X.lo, X.lo)};
    X = add(X, add(S, scale(unpack(__ldg(pp + k * LANES)), c0q4)));
    double2 o = make_double2((double)X.hi.x + (double)X.lo.x, (double)X.hi.y + (double)X.lo.y);
    if (EPI == EPI_RESID) {
      const double2 b = bp[k];
      o = make_double2(b.x - o.x, b.y - o.y);
      if (s0 < g.V) {
        red[0] += o.x * o.x + o.y * o.y;
        red[1] += b.x * b.x + b.y * b.y;
      }
    }
    if (s0 < g.V) op[k] = o;
  }
  if (EPI == EPI_RESID) grid_reduce<2, DD_THREADS>(red, ra, ticket);
}

// FP64 canonical field -> the apply's fields (zero past the last site).
__global__ void __launch_bounds__(384) to_dd_field_kernel(const double2* __restrict__ in, float4* __restrict__ out, int V) {
  __shared__ float4 t[12 * LANES + 12];
  const int i = threadIdx.x;                         // site i / 12 of the block, component i % 12
  const size_t base = (size_t)blockIdx.x * (12 * LANES);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (base + i < (size_t)V * 12) {
    const double2 d = in[base + i];
    const dd re = split_df(d.x), im = split_df(d.y);
    v = make_float4(re.hi, im.hi, re.lo, im.lo);
  }
  t[(i % 12) * (LANES + 1) + i / 12] = v;
  __syncthreads();
  out[base + i] = t[(i / LANES) * (LANES + 1) + (i & 31)];
}

const Table& dd_entries() {
  static const Table t = build();
  return t;
}

}  // namespace

size_t dd_field_bytes(const ok_W* W) { return (size_t)W->g.nblk * 12 * LANES * 16; }

int launch_to_dd_field(const ok_W* W, const cx<double>* in, void* out, cudaStream_t st) {
  {
    TraceScope ts("to_df64", st);
    to_dd_field_kernel<<<W->g.nblk, 12 * LANES, 0, st>>>((const double2*)in, (float4*)out, W->g.V);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

int launch_apply_dd(const ok_W* Wh, const void* psi_dd, cx<double>* out, int epi, const EpiArgs<dd>& ep, cudaStream_t st) {
  if (!Wh->Wdf || (epi != EPI_NONE && epi != EPI_RESID)) return OK_EINVAL;
  if (epi == EPI_RESID && !ep.b) return OK_EINVAL;
  const Table& tab = dd_entries();
  const Geom& g = Wh->g;
  const double a = Wh->sc.a_ii, b = Wh->sc.b_ii;
  const int a_big = fabs(a) >= fabs(b);
  const double big = a_big ? a : b, small = a_big ? b : a;
  const dd c0q4(4.0 * Wh->sc.c0q), two_big(big), two_r(big != 0.0 ? small / big : 0.0);
  const float4* W = reinterpret_cast<const float4*>(Wh->Wdf);
  const float4* psi = reinterpret_cast<const float4*>(psi_dd);
  double2* o = reinterpret_cast<double2*>(out);
  const double2* rhs = reinterpret_cast<const double2*>(ep.b);
  {
    TraceScope ts(epi == EPI_RESID ? "apply_df64_resid" : "apply_df64", st);
    if (epi == EPI_RESID)
      apply_dd_kernel<EPI_RESID><<<g.nblk, DD_THREADS, 0, st>>>(W, psi, o, g, c0q4, two_big, two_r, a_big, rhs, ep.ra, ep.ticket,
                                                                ep.halt, tab);
    else
      apply_dd_kernel<EPI_NONE><<<g.nblk, DD_THREADS, 0, st>>>(W, psi, o, g, c0q4, two_big, two_r, a_big, rhs, ep.ra, ep.ticket,
                                                               ep.halt, tab);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

}  // namespace okgb
