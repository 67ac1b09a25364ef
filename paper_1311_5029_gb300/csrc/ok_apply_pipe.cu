// The plain FP32 application of M (FP32 or FP16 W), software-pipelined by hand.
//
// A block of 128 threads covers 32 sites, two threads per site (ok_pair.cuh).  Warps 0-1 do the on-site
// term and the forward hops, warps 2-3 the backward hops, whose sums they hand over through shared memory.
// A half of the stencil is a fixed sequence of steps, one colour matrix each; the matrix of step k + LA and
// the half-spinor of a hop PLA steps ahead are requested before step k is computed, so several loads of
// every warp are always in flight.
//
// What bounds it: memory latency (16^3 x 32, FP32: 5.4 warps waiting for loads per issue and 0.2 at the barrier where the
// halves meet, issue 35 %, L1 57 %, DRAM 56 %; FP16: 3.8 and 0.4, issue 49 %, L1 45 %, DRAM 35 %).  Every tile starts with
// nothing in flight; requests over the tile boundary have not been tried.  More warps with fewer registers take as long or
// longer.  Left to itself the compiler keeps about one hop's loads in flight once the hops form one basic block (122 us at
// 16^3 x 32); a __syncwarp between a step's requests and its arithmetic keeps it from sinking the loads to their use.
// 16^3 x 32 / 28^3 x 96, FP32: 98 / 1735 us with the split kernel before, 92 / 1450 us now; FP16: 86 / 1610 us before, 74 /
// 1375 us now.  14x18x11x27 and 14^3 x 28 in FP32 were 1 to 2 % faster with the split kernel: their 2339 and 2401 tiles fill
// its four rounds of 608 blocks, and 5.1 and 5.3 rounds of this kernel's 456.
#include "ok_pair.cuh"

namespace okgb {
namespace {

constexpr int PIPE_THREADS = 128;
constexpr int PIPE_SITES = 32;

// ---------------------------------------------------------------------------- loads
__device__ __forceinline__ float4 ldv4(const void* p) {
  float4 d;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(d.x), "=f"(d.y), "=f"(d.z), "=f"(d.w) : "l"(p));
  return d;
}
__device__ __forceinline__ float2 ldv2(const void* p) {
  float2 d;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(d.x), "=f"(d.y) : "l"(p));
  return d;
}
__device__ __forceinline__ uint4 ldu4(const void* p) {
  uint4 d;
  asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(d.x), "=r"(d.y), "=r"(d.z), "=r"(d.w) : "l"(p));
  return d;
}
__device__ __forceinline__ unsigned ldu1(const void* p) {
  unsigned d;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(d) : "l"(p));
  return d;
}

// A matrix as loaded: FP32 elements, or FP16 words widened when used.
template <typename WT> struct Raw;
template <> struct Raw<float> {
  float4 a[4];
  float2 b;
  __device__ __forceinline__ void load(const cx<float>* W, int site, int m) {
    const cx<float>* p = W + ((size_t)(site >> 5) * NMAT + m) * (9 * LANES);
    const int l = site & 31;
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = ldv4(p + 2 * (q * LANES + l));
    b = ldv2(p + 8 * LANES + l);
  }
  __device__ __forceinline__ M3<float> get() const {
    M3<float> r;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      r.e[2 * q] = mk<float>(a[q].x, a[q].y);
      r.e[2 * q + 1] = mk<float>(a[q].z, a[q].w);
    }
    r.e[8] = mk<float>(b.x, b.y);
    return r;
  }
};
template <> struct Raw<__half> {
  uint4 a[2];
  unsigned b;
  __device__ __forceinline__ void load(const cx<__half>* W, int site, int m) {
    const cx<__half>* p = W + ((size_t)(site >> 5) * NMAT + m) * (9 * LANES);
    const int l = site & 31;
#pragma unroll
    for (int q = 0; q < 2; ++q) a[q] = ldu4(p + 4 * (q * LANES + l));
    b = ldu1(p + 8 * LANES + l);
  }
  __device__ __forceinline__ M3<float> get() const {
    M3<float> r;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      r.e[4 * q] = widen(a[q].x);
      r.e[4 * q + 1] = widen(a[q].y);
      r.e[4 * q + 2] = widen(a[q].z);
      r.e[4 * q + 3] = widen(a[q].w);
    }
    r.e[8] = widen(b);
    return r;
  }
};

// ---------------------------------------------------------------------------- the step sequence
// Hops: 0 on-site, 1..3 spatial, 4 temporal, 5..7 two-hop, 8..13 diagonal (2 pair + (0: I+J, 1: I-J)).
// A step is one matrix: on-site 3, spatial 4 each, temporal 4, the others 1.
constexpr int hop_steps(int h) { return h == 0 ? 3 : h <= 4 ? 4 : 1; }
constexpr int NHOPS = 14;
// Steps of the hops from h0 on: the first of hop h, the hop of step k and its place in the hop.
constexpr int first_step(int h, int h0) {
  int k = 0;
  for (int q = h0; q < h; ++q) k += hop_steps(q);
  return k;
}
constexpr int hop_of(int k, int h0) {
  int h = h0;
  while (k >= hop_steps(h)) { k -= hop_steps(h); ++h; }
  return h;
}
constexpr int sub_of(int k, int h0) { return k - first_step(hop_of(k, h0), h0); }
struct Off { int d[4]; };
constexpr Off hop_off(int h, bool fwd) {
  Off o{{0, 0, 0, 0}};
  const int f = fwd ? 1 : -1;
  if (h >= 1 && h <= 3) o.d[h - 1] = f;
  else if (h == 4) o.d[3] = f;
  else if (h >= 5 && h <= 7) o.d[h - 5] = 2 * f;
  else if (h >= 8) {
    const int P = (h - 8) / 2, I = P == 2 ? 1 : 0, J = P == 0 ? 1 : 2;
    o.d[I] = f;
    o.d[J] = (h - 8) % 2 ? -f : f;
  }
  return o;
}
// Matrix of sub-step j of hop h for thread p.
template <int H, int J, bool FWD>
__device__ __forceinline__ int mat_of(int p) {
  if constexpr (H == 0) return (p ? M_Y0M : M_Y0P) + J;
  else if constexpr (H <= 3) return M_WP + 8 * (H - 1) + 4 * (FWD ? p : 1 - p) + J;
  else if constexpr (H == 4) return J == 3 ? M_UT : M_ST + (J == 0 ? 0 : FWD ? J : 3 - J);
  else if constexpr (H <= 7) return M_VII + H - 5;
  else return M_VIJ + (H - 8) / 2 + 3 * ((H - 8) % 2);
}

// Antiperiodic directions (BC): none, time alone (physics runs), any.  Hop h can cross such a boundary.
enum : int { BC_NONE = 0, BC_TIME = 1, BC_ANY = 2 };
constexpr bool signed_hop(int h, int bc) { return bc == BC_ANY ? h != 0 : bc == BC_TIME && h == 4; }

template <typename SH, bool FWD, int BC, int H0, int H1>
struct Ctx {
  using WT = typename SH::W;

  const cx<WT>* W;
  const cx<float>* psi;
  int s, p;
  int c[4];
  Pair pr;
};

// The shape of the pipeline for W elements of type T: resident blocks per SM, and how many steps ahead a
// matrix (LA) and a half-spinor (PLA) are requested.  An FP16 matrix waits in half the registers, so it is
// requested earlier at four blocks per SM.
template <typename T, int N> struct PipeShape;
template <int N> struct PipeShape<float, N> { using W = float; static constexpr int MINB = 3, LA = N, PLA = 2; };
template <int N> struct PipeShape<__half, N> { using W = __half; static constexpr int MINB = 4, LA = N, PLA = 1; };

template <typename SH>
struct Bufs {
  static constexpr int LA = SH::LA;
  Raw<typename SH::W> v[LA + 1];
  H6<float> m[(SH::PLA + 1)];
  int n[8];       // neighbour site by hop (a backward hop's matrices and half-spinor)
  bool neg[8];
};

// Step at which the half-spinor of hop h is requested.
constexpr int psi_step(int h, int h0, int pla) {
  const int k = first_step(h, h0) - pla;
  return k < 0 ? -1 : k;
}

template <int H, typename SH, bool FWD, int BC, int H0, int H1>
__device__ __forceinline__ int site_of(const Ctx<SH, FWD, BC, H0, H1>& C, const Geom& g, bool& neg) {
  constexpr Off o = hop_off(H, FWD);
  return nbr_site<o.d[0], o.d[1], o.d[2], o.d[3], signed_hop(H, BC)>(C.c, g, neg);
}

template <int K, typename SH, bool FWD, int BC, int H0, int H1>
__device__ __forceinline__ void request(const Ctx<SH, FWD, BC, H0, H1>& C, const Geom& g, Bufs<SH>& B) {
  // matrix of step K
  if constexpr (K < first_step(H1, H0)) {
    constexpr int H = hop_of(K, H0), J = sub_of(K, H0);
    int w = C.s;
    if constexpr (!FWD) {
      bool neg;
      if constexpr (J == 0) {
        B.n[H & 7] = site_of<H>(C, g, neg);
        B.neg[H & 7] = neg;
      }
      w = B.n[H & 7];
    }
    B.v[K % (SH::LA + 1)].load(C.W, w, mat_of<H, J, FWD>(C.p));
  }
}
template <int H, typename SH, bool FWD, int BC, int H0, int H1>
__device__ __forceinline__ void request_psi(const Ctx<SH, FWD, BC, H0, H1>& C, const Geom& g, Bufs<SH>& B) {
  bool neg = false;
  int n = C.s;
  if constexpr (!FWD && psi_step(H, H0, SH::PLA) >= first_step(H, H0) - SH::LA) n = B.n[H & 7];  // its matrix request came first
  else if constexpr (H != 0) {
    n = site_of<H>(C, g, neg);
    B.neg[H & 7] = neg;
  }
  const float4* q = reinterpret_cast<const float4*>(C.psi) + (size_t)n * 6 + 3 * C.p;
  H6<float>& m = B.m[H % (SH::PLA + 1)];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float4 d = ldv4(q + k);
    m.v[(2 * k) / 3][(2 * k) % 3] = mk<float>(d.x, d.y);
    m.v[(2 * k + 1) / 3][(2 * k + 1) % 3] = mk<float>(d.z, d.w);
  }
}

struct Accs {
  H6<float> acc;    // h+- sums
  Halves<float> d;  // (u, l) sums
  H6<float> t;      // the hop's working half-spinor
  H6<float> y;      // on-site: the sum of the thread's Y term
};

template <int H, int BC>
__device__ __forceinline__ void take(H6<float>& m, bool neg) {
  if constexpr (signed_hop(H, BC)) {
    const float sg = neg ? -1.f : 1.f;
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int a = 0; a < 3; ++a) m.v[q][a] = sg * m.v[q][a];
  }
}

template <int K, typename SH, bool FWD, int BC, int H0, int H1>
__device__ __forceinline__ void compute(const Ctx<SH, FWD, BC, H0, H1>& C, Bufs<SH>& B, Accs& A, float c0q, float a_ii, float b_ii) {
  constexpr int H = hop_of(K, H0), J = sub_of(K, H0);
  const M3<float> V = B.v[K % (SH::LA + 1)].get();
  if constexpr (J == 0) take<H, BC>(B.m[H % (SH::PLA + 1)], B.neg[H & 7]);
  const H6<float>& m = B.m[H % (SH::PLA + 1)];
  if constexpr (H == 0) {
    if constexpr (J == 0) {
      // p = 0: u - i l, p = 1: u + i l
      const H6<float> oth = partner(m, C.pr.mask);
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const cx<float> u = C.p ? oth.v[q][k] : m.v[q][k], l = C.p ? m.v[q][k] : oth.v[q][k];
          A.t.v[q][k] = C.p ? u + ti(l) : u - ti(l);
          A.y.v[q][k] = c0q * A.t.v[q][k];
        }
      mv_add(A.y.v[0], V, A.t.v[0]);
      mv_sub(A.y.v[1], V, A.t.v[1]);
    } else if constexpr (J == 1) {
      mv_add(A.y.v[0], V, A.t.v[1]);
    } else {
      mv_add(A.y.v[1], V, A.t.v[0]);
      const H6<float> Rp = partner(A.y, C.pr.mask);
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 3; ++k) A.acc.v[q][k] = (A.y.v[q][k] + Rp.v[q][k]) + ti(A.y.v[q][k] - Rp.v[q][k]);
    }
  } else if constexpr (H <= 3) {
    if constexpr (J == 0) halves_to_h(m, C.pr, A.t);
    // forward: rows (J >> 1), columns (J & 1); backward: the adjoint
    if constexpr (FWD) mv_add(A.acc.v[J >> 1], V, A.t.v[J & 1]);
    else mdv_add(A.acc.v[J & 1], V, A.t.v[J >> 1]);
  } else if constexpr (H == 4) {
    if constexpr (FWD) {
      if constexpr (J == 0) { mv_add(A.d.cross.v[0], V, m.v[0]); mv_sub(A.d.cross.v[1], V, m.v[1]); }
      else if constexpr (J == 1) mv_add(A.d.cross.v[0], V, m.v[1]);
      else if constexpr (J == 2) mv_add(A.d.cross.v[1], V, m.v[0]);
      else {
        A.t = m;
        only(A.t, C.p == 1);
        mv_sub(A.d.same.v[0], V, A.t.v[0]);
        mv_sub(A.d.same.v[1], V, A.t.v[1]);
      }
    } else {
      if constexpr (J == 0) { mdv_sub(A.d.cross.v[0], V, m.v[0]); mdv_add(A.d.cross.v[1], V, m.v[1]); }
      else if constexpr (J == 1) mdv_sub(A.d.cross.v[0], V, m.v[1]);   // n2 (mat_of: M_ST + 2)
      else if constexpr (J == 2) mdv_sub(A.d.cross.v[1], V, m.v[0]);   // n1
      else {
        A.t = m;
        only(A.t, C.p == 0);
        mdv_sub(A.d.same.v[0], V, A.t.v[0]);
        mdv_sub(A.d.same.v[1], V, A.t.v[1]);
      }
    }
  } else if constexpr (H <= 7) {
    colour2h<float, !FWD>(A.t, V, m);
    add_scaled_h(A.d.same, a_ii, A.t);
    add_sigma_h(A.d.cross, H - 5, A.t, FWD ? b_ii : -b_ii);
  } else {
    constexpr int P = (H - 8) / 2, I = P == 2 ? 1 : 0, JJ = P == 0 ? 1 : 2;
    sigma_pair<float, I, JJ, (H - 8) % 2 ? -1 : 1>(m, A.t);
    colour2h_acc<float, !FWD>(A.d.cross, V, A.t);
  }
}

template <int H, int K, typename SH, bool FWD, int BC, int H0, int H1>
__device__ __forceinline__ void psi_due(const Ctx<SH, FWD, BC, H0, H1>& C, const Geom& g, Bufs<SH>& B) {
  if constexpr (H < H1) {
    if constexpr (psi_step(H, H0, SH::PLA) == K) request_psi<H>(C, g, B);
    psi_due<H + 1, K>(C, g, B);
  }
}

template <int K, typename SH, bool FWD, int BC, int H0, int H1>
__device__ __forceinline__ void steps(const Ctx<SH, FWD, BC, H0, H1>& C, const Geom& g, Bufs<SH>& B, Accs& A, float c0q, float a_ii,
                                      float b_ii) {
  if constexpr (K < first_step(H1, H0)) {
    request<K + SH::LA>(C, g, B);
    psi_due<H0, K>(C, g, B);
    __syncwarp();
    compute<K>(C, B, A, c0q, a_ii, b_ii);
    steps<K + 1>(C, g, B, A, c0q, a_ii, b_ii);
  }
}

template <int K, typename SH, bool FWD, int BC, int H0, int H1>
__device__ __forceinline__ void prologue(const Ctx<SH, FWD, BC, H0, H1>& C, const Geom& g, Bufs<SH>& B) {
  if constexpr (K < SH::LA) {
    request<K>(C, g, B);
    prologue<K + 1>(C, g, B);
  }
}

template <typename SH, bool FWD, int BC, int H0, int H1>
__device__ __forceinline__ void run_part(const Ctx<SH, FWD, BC, H0, H1>& C, const Geom& g, Accs& A, float c0q, float a_ii, float b_ii) {
  Bufs<SH> B;
#pragma unroll
  for (int k = 0; k < 8; ++k) B.neg[k] = false;
  prologue<0>(C, g, B);
  psi_due<H0, -1>(C, g, B);
  steps<0>(C, g, B, A, c0q, a_ii, b_ii);
}

template <typename SH, int BC>
__global__ void __launch_bounds__(PIPE_THREADS, SH::MINB)
    apply_pipe_kernel(const cx<typename SH::W>* __restrict__ W, const cx<float>* __restrict__ psi, cx<float>* __restrict__ out, Geom g,
                      float c0q, float a_ii, float b_ii, int spread, const int* halt) {
  if (halt && *halt) return;
  __shared__ cx<float> xch[2][64][6];
  const int half = threadIdx.x >> 6, t = threadIdx.x & 63;
  Pair pr;
  pr.p = t & 1;
  pr.mask = 0xffffffffu;
  const int ntiles = (g.V + PIPE_SITES - 1) / PIPE_SITES;
  const int b = blockIdx.x, G = gridDim.x;
  const int rank = (g.sms > 0 && G % g.sms == 0) ? (b % g.sms) * (G / g.sms) + b / g.sms : b;
  int kb = 0;
  // The last round, if it does not need every block, takes them in launch order, which spreads it over
  // the multiprocessors.  spread: the first tile of that round, a multiple of G (no tile's when the round
  // is nearly full).
  for (int r0 = 0; r0 < ntiles; r0 += G, kb ^= 1) {
    const int tile = r0 + (r0 == spread ? b : rank);
    if (tile >= ntiles) break;
    const int s = tile * PIPE_SITES + (t >> 1);
    const int sc = s < g.V ? s : g.V - 1;   // threads past the end repeat the last site and store nothing
    Accs A;
    zero_halves(A.d);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int k = 0; k < 3; ++k) A.acc.v[q][k] = mk<float>(0.f, 0.f);
    int r = sc, c[4];
    c[0] = r % g.L[0]; r /= g.L[0];
    c[1] = r % g.L[1]; r /= g.L[1];
    c[2] = r % g.L[2]; c[3] = r / g.L[2];
    if (half == 0) {
      const Ctx<SH, true, BC, 0, NHOPS> C{W, psi, sc, pr.p, {c[0], c[1], c[2], c[3]}, pr};
      run_part(C, g, A, c0q, a_ii, b_ii);
      to_h(A.d, pr, A.acc);
    } else {
      const Ctx<SH, false, BC, 1, NHOPS> C{W, psi, sc, pr.p, {c[0], c[1], c[2], c[3]}, pr};
      run_part(C, g, A, c0q, a_ii, b_ii);
      to_h(A.d, pr, A.acc);
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 3; ++k) xch[kb][t][3 * q + k] = A.acc.v[q][k];
    }
    __syncthreads();
    if (half == 0) {
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 3; ++k) A.acc.v[q][k] = A.acc.v[q][k] + xch[kb][t][3 * q + k];
      const H6<float> ap = partner(A.acc, pr.mask);
      H6<float> o;
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 3; ++k) o.v[q][k] = pr.p ? ap.v[q][k] - A.acc.v[q][k] : A.acc.v[q][k] + ap.v[q][k];
      if (s < g.V) store_half<float>(out, s, pr.p, o);
    }
  }
}

// ---------------------------------------------------------------------------- small lattices
// When the lattice has fewer tiles than the device has room for, a tile's latency is the kernel's time:
// one warp walks 25 or 28 steps, at one warp per scheduler mostly waiting for its instructions and
// loads.  Here a block takes 16 sites and its eight warps a part of the stencil each (4 to 8 steps), and
// the eight sums meet in shared memory, in a fixed order.
constexpr int SMALL_THREADS = 256;
constexpr int SMALL_SITES = 16;
template <typename WT, bool FWD, int H0, int H1>
__device__ __forceinline__ void small_part(const cx<WT>* W, const cx<float>* psi, int s, const int (&c)[4], const Pair& pr,
                                           const Geom& g, Accs& A, float c0q, float a_ii, float b_ii) {
  const Ctx<PipeShape<WT, sizeof(WT) == 2 ? 5 : 3>, FWD, BC_ANY, H0, H1> C{W, psi, s, pr.p, {c[0], c[1], c[2], c[3]}, pr};
  run_part(C, g, A, c0q, a_ii, b_ii);
}

template <typename WT>
__global__ void __launch_bounds__(SMALL_THREADS, 2)
    apply_small_kernel(const cx<WT>* __restrict__ W, const cx<float>* __restrict__ psi, cx<float>* __restrict__ out, Geom g,
                       float c0q, float a_ii, float b_ii, const int* halt) {
  if (halt && *halt) return;
  __shared__ float part[8][12][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  Pair pr;
  pr.p = lane & 1;
  pr.mask = 0xffffffffu;
  const int s0 = blockIdx.x * SMALL_SITES + (lane >> 1);
  const int s = s0 < g.V ? s0 : g.V - 1;   // threads past the end repeat the last site and store nothing
  int r = s, c[4];
  c[0] = r % g.L[0]; r /= g.L[0];
  c[1] = r % g.L[1]; r /= g.L[1];
  c[2] = r % g.L[2]; c[3] = r / g.L[2];
  Accs A;
  zero_halves(A.d);
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 3; ++k) A.acc.v[q][k] = mk<float>(0.f, 0.f);
  switch (w) {
    case 0: small_part<WT, true, 0, 2>(W, psi, s, c, pr, g, A, c0q, a_ii, b_ii); break;
    case 1: small_part<WT, true, 2, 4>(W, psi, s, c, pr, g, A, c0q, a_ii, b_ii); break;
    case 2: small_part<WT, true, 4, 8>(W, psi, s, c, pr, g, A, c0q, a_ii, b_ii); break;
    case 3: small_part<WT, true, 8, 14>(W, psi, s, c, pr, g, A, c0q, a_ii, b_ii); break;
    case 4: small_part<WT, false, 1, 3>(W, psi, s, c, pr, g, A, c0q, a_ii, b_ii); break;
    case 5: small_part<WT, false, 3, 5>(W, psi, s, c, pr, g, A, c0q, a_ii, b_ii); break;
    case 6: small_part<WT, false, 5, 9>(W, psi, s, c, pr, g, A, c0q, a_ii, b_ii); break;
    default: small_part<WT, false, 9, 14>(W, psi, s, c, pr, g, A, c0q, a_ii, b_ii); break;
  }
  to_h(A.d, pr, A.acc);
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      part[w][2 * (3 * q + k)][lane] = A.acc.v[q][k].re;
      part[w][2 * (3 * q + k) + 1][lane] = A.acc.v[q][k].im;
    }
  __syncthreads();
  float* sum = &part[0][0][0];
  for (int i = threadIdx.x; i < 12 * 32; i += SMALL_THREADS) {
    float v = sum[i];
#pragma unroll
    for (int k = 1; k < 8; ++k) v += sum[k * 384 + i];
    sum[i] = v;   // word i belongs to this thread alone
  }
  __syncthreads();
  if (w) return;
  H6<float> a, o;
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 3; ++k) a.v[q][k] = mk<float>(part[0][2 * (3 * q + k)][lane], part[0][2 * (3 * q + k) + 1][lane]);
  const H6<float> ap = partner(a, pr.mask);
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 3; ++k) o.v[q][k] = pr.p ? ap.v[q][k] - a.v[q][k] : a.v[q][k] + ap.v[q][k];
  if (s0 < g.V) store_half<float>(out, s, pr.p, o);
}

template <typename SH, int BC>
void launch(const cx<typename SH::W>* W, const cx<float>* psi, cx<float>* out, const Geom& g, float c0q, float a, float b, const int* halt,
            cudaStream_t st) {
  static int resident = 0;
  auto kern = apply_pipe_kernel<SH, BC>;
  if (resident == 0) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, PIPE_THREADS, 0) != cudaSuccess || nb < 1) nb = 1;
    resident = nb * sm_count();
  }
  const int tiles = grid_for(g.V, PIPE_SITES);
  Geom gs = g;
  gs.sms = sm_count();
  const int G = tiles < resident ? tiles : resident, rem = tiles % G;
  const int spread = rem > 0 && rem <= G - gs.sms ? tiles - rem : -1;
  kern<<<G, PIPE_THREADS, 0, st>>>(W, psi, out, gs, c0q, a, b, spread, halt);
}

}  // namespace

template <typename WT>
void launch_pipe(const cx<WT>* W, const cx<float>* psi, cx<float>* out, const Geom& g, float c0q, float a, float b,
                 const int* halt, cudaStream_t st) {
  // Small lattices: up to half a block of 16 sites per SM (us, pipelined / small: 5.5 / 4.1 at 512 sites,
  // 5.9 / 5.3 at 1024, 6.2 / 6.7 at 1536).
  const int small = grid_for(g.V, SMALL_SITES);
  if (2 * small <= sm_count()) {
    apply_small_kernel<WT><<<small, SMALL_THREADS, 0, st>>>(W, psi, out, g, c0q, a, b, halt);
    return;
  }
  // The form of the boundaries and the lookahead.  The requests are the same in all forms, but the compiler schedules
  // each in its own way, and which is the fastest was found by measurement.  The form, us: before the slash every hop's sign
  // is a multiplication, behind it only the temporal hop's (BC_TIME, for periodic lattices too).
  //   FP32, time antiperiodic: 14x18x11x27 63.0 / 60.6; 20^3 x 64 350 / 337; 28^3 x 96 1532 / 1445.  Periodic, against the
  //   form without signs: 61.6 / 60.6; 343 / 337; 1461 / 1445.
  //   FP16, time antiperiodic: 14x18x11x27 47.0 / 45.1; 18^3 x 36 126 / 117; 20^3 x 64 296 / 282; 28^3 x 48 663 / 648 and 647 /
  //   660 in two runs.  Periodic: 45.1 / 45.1; 117 / 117; 276 / 282; 24^3 x 64 480 / 506, so there the form without signs stays.
  // LA against the bytes of a time slice of W (us, LA 2 / 3 and 4 / 5; the crossover lies between the two nearest):
  //   FP32 BC_TIME: 9 MB (14^3 x 28) 61.5 / 63.0; 43 MB (24^3 x 64) 578 / 590; 68 MB (28^3 x 48) 797 / 729.
  //   FP32 BC_ANY the other way round: 43 MB 627 / 593; 28^3 x 96 (68 MB) 1533 / 1585; against the rule 28^3 x 48 770 / 755.
  //   FP16 BC_NONE: 4.2 MB (14^3 x 28) 46.6 / 45.2, 11x15x9x40 43.3 / 41.7; 6.3 MB (16^3 x 32) 74.1 / 79.4, 12 MB (20^3 x 64)
  //   276 / 305, 34 MB (28^3 x 96) 1349 / 1417; against the rule 10^3 x 20 19.9 / 21.1 and 18^3 x 36 117.1 / 116.1.
  //   FP16 BC_ANY: 4.2 MB 49.2 / 47.2; 6.3 MB 78.9 / 82.3; 12 MB 301 / 331; against the rule 18^3 x 36 125.8 / 121.6.
  //   FP16 BC_TIME: LA 4 from 1 % slower (14x14x16x59 104.5 / 103.3) to 5 % faster (12^3 x 24 32.9 / 34.6) everywhere.
  const size_t slice = (size_t)g.L[0] * g.L[1] * g.L[2] * SITE_ELEMS * sizeof(cx<WT>);
  const bool time_only = (g.bcneg & ~8) == 0;
  if constexpr (sizeof(WT) == 4) {
    const bool wide = slice > (size_t)56 << 20;
    if (time_only) {
      if (wide) launch<PipeShape<WT, 3>, BC_TIME>(W, psi, out, g, c0q, a, b, halt, st);
      else launch<PipeShape<WT, 2>, BC_TIME>(W, psi, out, g, c0q, a, b, halt, st);
    } else {
      if (wide) launch<PipeShape<WT, 2>, BC_ANY>(W, psi, out, g, c0q, a, b, halt, st);
      else launch<PipeShape<WT, 3>, BC_ANY>(W, psi, out, g, c0q, a, b, halt, st);
    }
  } else {
    const bool wide = slice > (size_t)5 << 20;
    if (g.bcneg == 8) {
      launch<PipeShape<WT, 4>, BC_TIME>(W, psi, out, g, c0q, a, b, halt, st);
    } else if (g.bcneg == 0) {
      if (wide) launch<PipeShape<WT, 4>, BC_NONE>(W, psi, out, g, c0q, a, b, halt, st);
      else launch<PipeShape<WT, 5>, BC_NONE>(W, psi, out, g, c0q, a, b, halt, st);
    } else {
      if (wide) launch<PipeShape<WT, 4>, BC_ANY>(W, psi, out, g, c0q, a, b, halt, st);
      else launch<PipeShape<WT, 5>, BC_ANY>(W, psi, out, g, c0q, a, b, halt, st);
    }
  }
}
template void launch_pipe<float>(const cx<float>*, const cx<float>*, cx<float>*, const Geom&, float, float, float, const int*, cudaStream_t);
template void launch_pipe<__half>(const cx<__half>*, const cx<float>*, cx<float>*, const Geom&, float, float, float, const int*, cudaStream_t);

}  // namespace okgb
