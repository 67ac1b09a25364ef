// Learned right preconditioner: P = L_K ... L_1 with gauge-covariant linear layers
//   (L psi)(x) = sum_d A_d (T_d psi)(x),   d in {0, +x, -x, +y, -y, +z, -z, +t, -t},
// T_0 = 1, (T_{+mu} psi)(x) = U_mu(x) psi(x + mu), (T_{-mu} psi)(x) = U_mu(x - mu)^dag psi(x - mu)
// (the link transport of the hopping terms of Eq. minFlopForm, with the fermion boundary sign),
// and A_d a learned 4 x 4 complex spin matrix shared by all sites.  P is linear in psi, so
// BiCGStab on M P y = b (x = P y) keeps a fixed operator; it is gauge covariant because only the
// links move colour.
//
// Kernels (FP32 fields, FP32 weights, FP32 links from the handle's OK_W_LINKS copy in the
// site-blocked layout of W):
//   layer:    one thread per site, the nine offsets unrolled; weights staged in shared memory.
//             The adjoint layer L^dag = sum_d A_d^dag T_{-d} is the same kernel with the offsets
//             reversed and the weights conjugate-transposed.
//   gradient: dloss/dA_{l,d} = 2 sum_{x, colour} g_l(x) (T_d psi_{l-1})(x)^dag: one warp per offset,
//             FP32 sums over a few sites, then sums over lanes, blocks and pairs with FP64's accuracy or
//             better, in a fixed order (deterministic for a given group of pairs).
//   loss:     |P b - x|^2 / |x|^2 per pair with the seed g_K = (P b - x) / |x|^2.
//   Adam:     on the real and imaginary parts of every A entry, in the gradient's final sum.
// A training step runs every kernel once for a group of its pairs, not once per pair.
#include "ok_net.cuh"
#include "ok_group.cuh"
#include "ok_sum3.cuh"
#include "ok_pair.cuh"

#include <cmath>
#include <cstring>
#include <vector>

namespace okgb {
// Scratch of a training step for `group` pairs.
struct TrainBufs {
  int group = 0;                       // 0: none
  cx<float>* acts = nullptr;           // [layers][group][V * 12]
  cx<float>* tg[2] = {nullptr, nullptr};  // backward gradients [group][V * 12]; null for one pair (ok_net::g serves)
  double* part = nullptr;              // gradient partials [layers][blocks][9][32]
  double* lpart = nullptr;             // loss partials [group][2 * loss blocks]
};
}  // namespace okgb

struct ok_net {
  int layers = 0;
  float2* A = nullptr;      // [layers][9][4][4]
  float* m = nullptr;       // Adam moments, [layers * 288]
  float* v = nullptr;
  double* gacc = nullptr;   // gradient accumulator [layers * 288]
  double* scal = nullptr;   // [0] loss accumulator, [2 + 2 q, 3 + 2 q] |x|^2 and |P b - x|^2 of pair q of a group
  unsigned* ticket = nullptr;  // [MAX_GROUP]
  long long adam_t = 0;
  int V = 0;                // volume the workspace is sized for
  int device = 0;
  okgb::cx<float>* g[2] = {nullptr, nullptr};  // layer ping-pong of an application, [V * 12]
  okgb::TrainBufs t;        // of the pairs that train together
  int most = 0;             // the largest group that fitted, once a larger one did not
};

namespace okgb {

namespace {

constexpr int NET_THREADS = 128;
constexpr int NOFF = 9;
constexpr int NPAR = NOFF * 32;  // real parameters per layer
constexpr int MAX_GROUP = 64;    // pairs of a batch that go through the kernels together

// (direction, step) of offset d; direction -1 is the on-site term.
__host__ __device__ constexpr int off_mu(int d) { return d == 0 ? -1 : (d - 1) / 2; }
__host__ __device__ constexpr int off_step(int d) { return d == 0 ? 0 : ((d - 1) % 2 == 0 ? 1 : -1); }

__device__ __forceinline__ int neighbour(const int (&c)[4], const Geom& g, int mu, int step, bool& neg) {
  int cc[4] = {c[0], c[1], c[2], c[3]};
  int v = cc[mu] + step;
  neg = false;
  if (v < 0) { v += g.L[mu]; neg = (g.bcneg >> mu) & 1; }
  else if (v >= g.L[mu]) { v -= g.L[mu]; neg = (g.bcneg >> mu) & 1; }
  cc[mu] = v;
  return cc[0] + g.L[0] * (cc[1] + g.L[1] * (cc[2] + g.L[2] * cc[3]));
}

__device__ __forceinline__ void site_coords(int s, const Geom& g, int (&c)[4]) {
  int r = s;
  c[0] = r % g.L[0]; r /= g.L[0];
  c[1] = r % g.L[1]; r /= g.L[1];
  c[2] = r % g.L[2]; c[3] = r / g.L[2];
}

__device__ __forceinline__ void load_sp(const cx<float>* __restrict__ p, int site, cx<float> (&v)[4][3]) {
  const float4* q = reinterpret_cast<const float4*>(p) + (size_t)site * 6;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float4 d = __ldg(q + k);
    v[(2 * k) / 3][(2 * k) % 3] = mk<float>(d.x, d.y);
    v[(2 * k + 1) / 3][(2 * k + 1) % 3] = mk<float>(d.z, d.w);
  }
}

// U_mu(site) from the site-blocked FP32 link copy (element e of the 32 sites of a block is one
// contiguous row).
__device__ __forceinline__ void link(const cx<float>* __restrict__ L, int site, int mu, M3<float>& U) {
  const float2* q = reinterpret_cast<const float2*>(L) + ((size_t)(site >> 5) * 4 + mu) * 9 * LANES + (site & 31);
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const float2 d = __ldg(q + e * LANES);
    U.e[e] = mk<float>(d.x, d.y);
  }
}

// w = (T psi)(x) for the transport of offset d (reversed when REV).
template <bool REV>
__device__ __forceinline__ void transported(const cx<float>* __restrict__ L, const cx<float>* __restrict__ in, int x,
                                            const int (&c)[4], const Geom& g, int d, cx<float> (&w)[4][3]) {
  const int mu = off_mu(d);
  if (mu < 0) { load_sp(in, x, w); return; }
  const int step = REV ? -off_step(d) : off_step(d);
  bool neg;
  const int n = neighbour(c, g, mu, step, neg);
  cx<float> v[4][3];
  load_sp(in, n, v);
  M3<float> U;
  link(L, step > 0 ? x : n, mu, U);
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    if (step > 0) mv(w[s], U, v[s]);
    else mdv(w[s], U, v[s]);
    if (neg)
#pragma unroll
      for (int a = 0; a < 3; ++a) w[s][a] = -w[s][a];
  }
}

// out = sum_d A_d T_d in   (ADJ: sum_d A_d^dag T_{-d} in, the adjoint layer).  With nrhs fields
// [nrhs][V][12] per launch, block b works on field b % nrhs and site block b / nrhs, so the blocks
// that read the same links run back to back and share them through L2.  With `halt` non-null and
// nonzero at launch the kernel does nothing.
template <bool ADJ>
__global__ void __launch_bounds__(NET_THREADS) net_layer_kernel(const cx<float>* __restrict__ L, const float2* __restrict__ A,
                                                                const cx<float>* __restrict__ in, cx<float>* __restrict__ out,
                                                                Geom g, int nrhs, const int* __restrict__ halt) {
  if (halt && *halt) return;  // a halted solver state: this layer belongs to an iteration that does nothing
  const int rhs = blockIdx.x % nrhs, sb = blockIdx.x / nrhs;
  in += (size_t)rhs * 12 * g.V;
  out += (size_t)rhs * 12 * g.V;
  // Each weight a is kept as (a.re, a.re, -a.im, a.im), so that a w adds to (re, im) as two
  // packed FP32 multiply-adds: (a.re, a.re) * (w.re, w.im) + (-a.im, a.im) * (w.im, w.re).
  __shared__ float4 sA[NOFF * 16];
  for (int i = threadIdx.x; i < NOFF * 16; i += NET_THREADS) {
    float2 a;
    if (!ADJ) {
      a = A[i];
    } else {
      const int d = i / 16, s = (i % 16) / 4, t = i % 4;
      const float2 b = A[d * 16 + t * 4 + s];
      a = make_float2(b.x, -b.y);
    }
    sA[i] = make_float4(a.x, a.x, -a.y, a.y);
  }
  __syncthreads();
  const int x = sb * NET_THREADS + threadIdx.x;
  if (x >= g.V) return;
  int c[4];
  site_coords(x, g, c);
  float2 acc[4][3];
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) acc[s][a] = make_float2(0.f, 0.f);
#pragma unroll
  for (int d = 0; d < NOFF; ++d) {
    cx<float> w[4][3];
    transported<ADJ>(L, in, x, c, g, d, w);
    float2 wv[4][3], ws[4][3];
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        wv[t][k] = make_float2(w[t][k].re, w[t][k].im);
        ws[t][k] = make_float2(w[t][k].im, w[t][k].re);
      }
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float4 a4 = sA[d * 16 + s * 4 + t];
        const float2 ar = make_float2(a4.x, a4.y), ai = make_float2(a4.z, a4.w);
#pragma unroll
        for (int k = 0; k < 3; ++k) acc[s][k] = __ffma2_rn(ai, ws[t][k], __ffma2_rn(ar, wv[t][k], acc[s][k]));
      }
  }
  float4* q = reinterpret_cast<float4*>(out) + (size_t)x * 6;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float2 u = acc[(2 * k) / 3][(2 * k) % 3];
    const float2 v = acc[(2 * k + 1) / 3][(2 * k + 1) % 3];
    q[k] = make_float4(u.x, u.y, v.x, v.y);
  }
}

// The lanes' floats summed over the warp: returns the sum of C[lane].  It transposes as it sums: each step adds the half of
// the values that a lane keeps to the same half of its partner's, 31 additions instead of 160.  They are error-free
// transformations on the FP32 pipes, which keep more bits than FP64 (ok_sum3.cuh), wherever their range allows: some
// 200 cycles of a multiprocessor, where FP64's additions and conversions, at 1/58 of the FP32 rate, take 900.
__device__ __forceinline__ double lane_sums(const float (&C)[32], int lane) {
  constexpr unsigned full = 0xffffffffu;
  float m = 0.f;   // (a NaN goes through either way)
#pragma unroll
  for (int k = 0; k < 32; ++k) m = fmaxf(m, fabsf(C[k]));
  if (__any_sync(full, m > 0x1p100f)) {
    double v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float keep = lane & 16 ? C[k + 16] : C[k], send = lane & 16 ? C[k] : C[k + 16];
      v[k] = (double)keep + (double)__shfl_xor_sync(full, send, 16);
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < o; ++k) {
        const double keep = lane & o ? v[k + o] : v[k], send = lane & o ? v[k] : v[k + o];
        v[k] = keep + __shfl_xor_sync(full, send, o);
      }
    return v[0];
  }
  Sum3 v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float send = lane & 16 ? C[k] : C[k + 16];
    v[k].s = lane & 16 ? C[k + 16] : C[k];
    v[k].t = two_sum(v[k].s, __shfl_xor_sync(full, send, 16));
    v[k].u = 0.f;
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < o; ++k) {
      const bool up = lane & o;
      const Sum3 keep = up ? v[k + o] : v[k];
      Sum3 send = up ? v[k] : v[k + o];
      send.s = __shfl_xor_sync(full, send.s, o);
      send.t = __shfl_xor_sync(full, send.t, o);
      if (o < 8) send.u = __shfl_xor_sync(full, send.u, o);   // zero before
      v[k] = keep + send;
    }
  return v[0].value();
}

// Gradient partials: part[block][d][32] = sum over the block's (pair, 32-site tile)s of
// g(x)_s,c conj((T_d in)(x)_t,c) (16 complex = 32 values).  A block has one warp per offset d, so a
// warp keeps one offset's 32 sums over all its sites and takes one lane reduction for every `run` sites of
// a thread.  (One warp walking all nine offsets took nine five-step FP64 trees of 32 values for one or two sites a
// thread: the FP64 pipe was 76 % busy and the kernel took 289 us at 16^3 x 32; this form takes 53 us, 48 us a
// pair in a batch of four.)
// The nine warps read the same tile's g and neighbours back to back, so L1 shares them.
constexpr int GRAD_WARPS = NOFF;
constexpr int GRAD_THREADS = 32 * GRAD_WARPS;
// Sites that a thread adds up in FP32 before a lane reduction, at most 8: as many as 77824 threads (608 blocks of 128) take
// of the lattice, which is what one thread per site in a resident grid adds up.  Shorter runs err less, longer ones need
// fewer reductions.  The gradient's error against 64 bits, mean of 12 fields, and the kernel's time in a batch of four at
// 16^3 x 32: run 1 2.486e-8, 241 us; 2 (the rule) 2.490e-8, 191 us; 8 2.505e-8, 156 us.  12^3 x 24: run 1 (the rule)
// 3.329e-8, 81 us; 8 3.354e-8, 55 us.
int grad_run(int V) {
  const int r = (V + 77823) / 77824;
  return r > 8 ? 8 : r;
}
__global__ void __launch_bounds__(GRAD_THREADS, 2) net_grad_kernel(const cx<float>* __restrict__ L, const cx<float>* __restrict__ gr,
                                                                   const cx<float>* __restrict__ in, Geom g, int pairs, int run,
                                                                   double* __restrict__ part, bool accumulate) {
  const int lane = threadIdx.x & 31, d = threadIdx.x >> 5;
  // (32-bit indices: a group of pairs holds at most 256 MiB of activations, or it is one pair)
  const unsigned ntiles = (g.V + 31) / 32, work = ntiles * pairs;
  double tot = 0.0;
  for (unsigned w0 = blockIdx.x; w0 < work; w0 += gridDim.x * run) {
    float C[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) C[k] = 0.f;
#pragma unroll 1
    for (int u = 0; u < run; ++u) {
      const unsigned w = w0 + u * gridDim.x;
      if (w >= work) break;
      const int q = w / ntiles, x = w % ntiles * 32 + lane;
      if (x >= g.V) continue;
      const size_t off = (size_t)q * 12 * g.V;
      int c[4];
      site_coords(x, g, c);
      cx<float> gv[4][3], wv[4][3];
      load_sp(gr + off, x, gv);
      transported<false>(L, in + off, x, c, g, d, wv);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          cx<float> z = mk<float>(C[2 * (4 * s + t)], C[2 * (4 * s + t) + 1]);
#pragma unroll
          for (int a = 0; a < 3; ++a) z = fma_cj(wv[t][a], gv[s][a], z);  // g conj(w)
          C[2 * (4 * s + t)] = z.re;
          C[2 * (4 * s + t) + 1] = z.im;
        }
    }
    tot += lane_sums(C, lane);
  }
  double* p = part + (size_t)blockIdx.x * NPAR + threadIdx.x;
  *p = accumulate ? *p + tot : tot;
}

// Adam's arguments; P null: no update.
struct AdamArgs {
  float *P, *m, *v;
  double scale;
  float lr, b1, b2, eps, c1, c2;
};

// One block per (layer, offset): gacc = 2 sum over the blocks' partials (eight slices of blocks,
// then the slices in order), and one Adam step on those 32 parameters.  (One block per layer
// summing 608 partials in sequence took 60 us per pair and layer; all layers of a step now take 14 us.)
__global__ void __launch_bounds__(256) net_grad_final_kernel(const double* __restrict__ part, int nblocks, double* __restrict__ gacc,
                                                             AdamArgs ad) {
  __shared__ double sh[8][32];
  const int l = blockIdx.x / NOFF, d = blockIdx.x % NOFF;
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const double* p = part + (size_t)l * nblocks * NPAR + d * 32 + lane;
  double s = 0.0;
#pragma unroll 4
  for (int b = slice; b < nblocks; b += 8) s += p[(size_t)b * NPAR];
  sh[slice][lane] = s;
  __syncthreads();
  if (slice) return;
  for (int k = 1; k < 8; ++k) s += sh[k][lane];
  const int i = l * NPAR + d * 32 + lane;
  const double gsum = 2.0 * s;
  gacc[i] = gsum;
  if (!ad.P) return;
  const float gr = (float)(gsum * ad.scale);
  const float m = ad.b1 * ad.m[i] + (1.f - ad.b1) * gr, v = ad.b2 * ad.v[i] + (1.f - ad.b2) * gr * gr;
  ad.m[i] = m;
  ad.v[i] = v;
  ad.P[i] -= ad.lr * (m / ad.c1) / (sqrtf(v / ad.c2) + ad.eps);
}

// |x|^2 and |out - x|^2 of pair blockIdx.y -> scal[2 + 2 pair], scal[3 + 2 pair]: chunks of LOSS_CHUNK complex
// numbers on the FP32 pipes with more than FP64's accuracy (ok_sum3.cuh), the chunks in FP64.  (In FP64 throughout
// the FP64 pipe was 82 % busy: 51 us for 25 MB at 16^3 x 32, now 16 us a pair in a batch of four; pairs of floats, which
// took 13 us, keep 48 bits and lose the squares of small differences.)
constexpr int LOSS_CHUNK = 8;
__global__ void __launch_bounds__(256) net_loss_kernel(const float2* __restrict__ out, const float2* __restrict__ x, long long n,
                                                       double* part, double* scal, unsigned* ticket) {
  out += blockIdx.y * n;
  x += blockIdx.y * n;
  double v[2] = {0.0, 0.0};
  const long long gs = (long long)gridDim.x * 256;
  for (long long i0 = blockIdx.x * 256LL + threadIdx.x; i0 < n; i0 += gs * LOSS_CHUNK) {
    float2 a[LOSS_CHUNK], b[LOSS_CHUNK];
#pragma unroll
    for (int u = 0; u < LOSS_CHUNK; ++u) {
      const long long i = i0 + u * gs;
      a[u] = b[u] = make_float2(0.f, 0.f);
      if (i < n) { a[u] = out[i]; b[u] = x[i]; }
    }
    loss_chunk(a, b, v);
  }
  const RedArgs ra{nullptr, part + (size_t)blockIdx.y * 2 * gridDim.x, scal + 2 + 2 * blockIdx.y, FIN_NONE};
  grid_reduce<2, 256>(v, ra, ticket + blockIdx.y);
}

// g = (out - x) / |x|^2 for pair blockIdx.y; one thread adds the group's losses to scal[0].
__global__ void __launch_bounds__(256) net_seed_kernel(const float2* __restrict__ out, const float2* __restrict__ x,
                                                       float2* __restrict__ g, long long n, double* scal) {
  __shared__ float inv_s;
  if (threadIdx.x == 0) {
    const double n2 = scal[2 + 2 * blockIdx.y];
    inv_s = n2 > 0.0 ? (float)(1.0 / n2) : 0.f;  // one FP64 division per block, not per thread
  }
  __syncthreads();
  const float inv = inv_s;
  out += blockIdx.y * n;
  x += blockIdx.y * n;
  g += blockIdx.y * n;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
    const float2 a = out[i], b = x[i];
    g[i] = make_float2((a.x - b.x) * inv, (a.y - b.y) * inv);
  }
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
    double s = scal[0];
    for (unsigned q = 0; q < gridDim.y; ++q) s += scal[2 + 2 * q] > 0.0 ? scal[3 + 2 * q] / scal[2 + 2 * q] : 0.0;
    scal[0] = s;
  }
}

// Two blocks of GRAD_THREADS threads fit on a multiprocessor.
int grad_blocks(int V) {
  const int need = (V + 31) / 32;
  const int cap = sm_count() * 2;
  return need < cap ? need : cap;
}

int loss_blocks(int V) {
  const int need = grid_for((12LL * V + LOSS_CHUNK - 1) / LOSS_CHUNK, 256);
  const int cap = sm_count() * 4;
  return need < cap ? need : cap;
}

void free_training(TrainBufs& t) {
  for (void* q : {(void*)t.acts, (void*)t.tg[0], (void*)t.tg[1], (void*)t.part, (void*)t.lpart})
    if (q) cudaFree(q);
  t = TrainBufs{};
}

cudaError_t alloc_training(const ok_net* N, int V, int pairs, TrainBufs& t) {
  const size_t f = (size_t)pairs * V * 12 * sizeof(cx<float>);
  cudaError_t e = cudaMalloc(&t.acts, N->layers * f);
  for (int k = 0; k < 2 && pairs > 1 && e == cudaSuccess; ++k) e = cudaMalloc(&t.tg[k], f);
  if (e == cudaSuccess) e = cudaMalloc(&t.part, (size_t)N->layers * grad_blocks(V) * NPAR * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&t.lpart, (size_t)pairs * 2 * loss_blocks(V) * sizeof(double));
  if (e == cudaSuccess) {
    t.group = pairs;
  } else {
    cudaGetLastError();
    free_training(t);
  }
  return e;
}

// Pairs of a batch of nb that one pass of the kernels takes: as many as fit in 256 MiB of
// activations (enough to fill the GPU: the launches of a small lattice hold little work each).
int group_of(const ok_net* N, int V, int nb) {
  const long long per = (long long)N->layers * V * 12 * (long long)sizeof(cx<float>);
  long long q = (256LL << 20) / per;
  if (q > MAX_GROUP) q = MAX_GROUP;
  if (q > nb) q = nb;
  return q < 1 ? 1 : (int)q;
}

// Scratch for a lattice of V sites: two fields (the layer ping-pong of an application, and the backward gradients of
// one pair) and, for training (nb > 0), the activations of every layer, the backward gradients and the
// reduction partials of a group of pairs.  A larger group's buffers are taken before the present ones are given
// back; where they do not fit, a smaller group runs, down to one pair.
int ensure_workspace(ok_net* N, int V, int nb) {
  const size_t n = (size_t)V * 12;
  if (N->V != V) {
    free_training(N->t);
    N->most = 0;
    if (N->g[0]) cudaFree(N->g[0]);
    if (N->g[1]) cudaFree(N->g[1]);
    N->g[0] = N->g[1] = nullptr; N->V = 0;
    OK_CUDA_TRY(cudaMalloc(&N->g[0], n * sizeof(cx<float>)));
    OK_CUDA_TRY(cudaMalloc(&N->g[1], n * sizeof(cx<float>)));
    N->V = V;
  }
  if (nb < 1) return OK_SUCCESS;
  TrainBufs t;
  cudaError_t err = cudaSuccess;
  const int group = grow_group(group_of(N, V, nb), N->t.group, N->most, [&](int q) {
    err = alloc_training(N, V, q, t);
    return err == cudaSuccess;
  });
  if (t.group) {
    free_training(N->t);
    N->t = t;
  }
  if (!group) { set_cuda_error(err); return OK_ECUDA; }
  return OK_SUCCESS;
}

int layer(const ok_net* N, const ok_W* W, int l, bool adj, const cx<float>* in, cx<float>* out, cudaStream_t st,
          int nrhs = 1, const int* halt = nullptr) {
  const Geom& g = W->g;
  const long long nb = (long long)grid_for(g.V, NET_THREADS) * nrhs;
  if (nb > 0x7fffffffLL) return OK_EINVAL;
  {
    TraceScope ts(adj ? "net_layer_adj" : "net_layer", st);
    if (adj)
      net_layer_kernel<true><<<(unsigned)nb, NET_THREADS, 0, st>>>((const cx<float>*)W->L32, N->A + (size_t)l * 144, in, out, g, nrhs, halt);
    else
      net_layer_kernel<false><<<(unsigned)nb, NET_THREADS, 0, st>>>((const cx<float>*)W->L32, N->A + (size_t)l * 144, in, out, g, nrhs, halt);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

#define NET_TRY(expr)                       \
  do {                                      \
    int _rc = (expr);                       \
    if (_rc != OK_SUCCESS) return _rc;      \
  } while (0)

// The gradient partials of `pairs` pairs ([pairs][V * 12] fields), added to those of the batch's
// earlier groups unless `first`, and their losses into scal[0].
int group_backprop(ok_net* N, const ok_W* W, int pairs, const cx<float>* b, const cx<float>* x, bool first, cudaStream_t st) {
  const Geom& g = W->g;
  const long long n = 12LL * g.V, gn = n * pairs;
  const int K = N->layers;
  cx<float>* const tg[2] = {N->t.tg[0] ? N->t.tg[0] : N->g[0], N->t.tg[1] ? N->t.tg[1] : N->g[1]};
  const cx<float>* in = b;
  for (int l = 0; l < K; ++l) {
    cx<float>* o = N->t.acts + (size_t)l * gn;
    NET_TRY(layer(N, W, l, false, in, o, st, pairs));
    in = o;
  }
  const int lb = loss_blocks(g.V), gb = grad_blocks(g.V);
  {
    TraceScope ts("net_loss", st);
    net_loss_kernel<<<dim3(lb, pairs), 256, 0, st>>>((const float2*)in, (const float2*)x, n, N->t.lpart, N->scal, N->ticket);
  }
  OK_LAUNCH_CHECK();
  {
    TraceScope ts("net_seed", st);
    const int sb = grid_for(n, 256) < 1024 ? grid_for(n, 256) : 1024;
    net_seed_kernel<<<dim3(sb, pairs), 256, 0, st>>>((const float2*)in, (const float2*)x, (float2*)tg[0], n, N->scal);
  }
  OK_LAUNCH_CHECK();
  int cur = 0;
  for (int l = K - 1; l >= 0; --l) {
    const cx<float>* lin = l == 0 ? b : N->t.acts + (size_t)(l - 1) * gn;
    {
      TraceScope ts("net_grad", st);
      net_grad_kernel<<<gb, GRAD_THREADS, 0, st>>>((const cx<float>*)W->L32, tg[cur], lin, g, pairs, grad_run(g.V),
                                                   N->t.part + (size_t)l * gb * NPAR, !first);
    }
    OK_LAUNCH_CHECK();
    if (l > 0) {
      NET_TRY(layer(N, W, l, true, tg[cur], tg[1 - cur], st, pairs));
      cur = 1 - cur;
    }
  }
  return OK_SUCCESS;
}

// Loss sum (scal[0]) and gradient (gacc, with `ad` applied) over nb pairs.
int batch_backprop(ok_net* N, const ok_W* W, int nb, const cx<float>* b, const cx<float>* x, const AdamArgs& ad, cudaStream_t st) {
  NET_TRY(ensure_workspace(N, W->g.V, nb));
  OK_CUDA_TRY(cudaMemsetAsync(N->scal, 0, sizeof(double), st));
  const size_t n = (size_t)W->g.V * 12;
  for (int i = 0; i < nb; i += N->t.group) {
    const int pairs = nb - i < N->t.group ? nb - i : N->t.group;
    NET_TRY(group_backprop(N, W, pairs, b + i * n, x + i * n, i == 0, st));
  }
  {
    TraceScope ts("net_grad_final", st);
    net_grad_final_kernel<<<N->layers * NOFF, 256, 0, st>>>(N->t.part, grad_blocks(W->g.V), N->gacc, ad);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

int check(const ok_net* N, const ok_W* W) {
  if (!N || !W || !W->L32 || N->layers < 1) return OK_EINVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != N->device || dev != W->device) return OK_EINVAL;
  return OK_SUCCESS;
}

}  // namespace

int net_apply_unless_halted(ok_net* N, const ok_W* W, const cx<float>* in, cx<float>* out, const int* halt,
                           cudaStream_t st) {
  NET_TRY(check(N, W));
  NET_TRY(ensure_workspace(N, W->g.V, 0));
  const cx<float>* cur = in;
  for (int l = 0; l < N->layers; ++l) {
    cx<float>* o = l == N->layers - 1 ? out : N->g[l % 2];  // ping-pong through the workspace
    NET_TRY(layer(N, W, l, false, cur, o, st, 1, halt));
    cur = o;
  }
  return OK_SUCCESS;
}

int net_apply(ok_net* N, const ok_W* W, const cx<float>* in, cx<float>* out, cudaStream_t st) {
  return net_apply_unless_halted(N, W, in, out, nullptr, st);
}

// out_k = P in_k for nrhs fields [nrhs][V][12] in one launch per layer, through the caller's two
// scratch fields of the same size.
int net_apply_multi(ok_net* N, const ok_W* W, const cx<float>* in, cx<float>* out, int nrhs, cx<float>* tmp0, cx<float>* tmp1,
                    cudaStream_t st) {
  NET_TRY(check(N, W));
  if (nrhs < 1 || nrhs > 65535 || !tmp0 || !tmp1) return OK_EINVAL;
  cx<float>* tmp[2] = {tmp0, tmp1};
  const cx<float>* cur = in;
  for (int l = 0; l < N->layers; ++l) {
    cx<float>* o = l == N->layers - 1 ? out : tmp[l % 2];
    NET_TRY(layer(N, W, l, false, cur, o, st, nrhs));
    cur = o;
  }
  return OK_SUCCESS;
}

int net_loss_grad(ok_net* N, const ok_W* W, const cx<float>* b, const cx<float>* x, double* loss, double* grad, cudaStream_t st) {
  NET_TRY(check(N, W));
  NET_TRY(batch_backprop(N, W, 1, b, x, AdamArgs{}, st));
  double s = 0.0;
  OK_CUDA_TRY(cudaMemcpyAsync(&s, N->scal, sizeof(s), cudaMemcpyDeviceToHost, st));
  if (grad) OK_CUDA_TRY(cudaMemcpyAsync(grad, N->gacc, sizeof(double) * NPAR * N->layers, cudaMemcpyDeviceToHost, st));
  OK_CUDA_TRY(cudaStreamSynchronize(st));
  if (loss) *loss = s;
  return OK_SUCCESS;
}

int net_train_step(ok_net* N, const ok_W* W, int nb, const cx<float>* b, const cx<float>* x, double lr, double* loss,
                   cudaStream_t st) {
  NET_TRY(check(N, W));
  if (nb < 1 || !b || !x || !(lr > 0.0)) return OK_EINVAL;
  const float b1 = 0.9f, b2 = 0.999f;
  const float t = (float)(N->adam_t + 1);
  const float c1 = 1.f - powf(b1, t), c2 = 1.f - powf(b2, t);
  NET_TRY(batch_backprop(N, W, nb, b, x, AdamArgs{(float*)N->A, N->m, N->v, 1.0 / nb, (float)lr, b1, b2, 1e-8f, c1, c2}, st));
  N->adam_t += 1;
  double s = 0.0;
  OK_CUDA_TRY(cudaMemcpyAsync(&s, N->scal, sizeof(s), cudaMemcpyDeviceToHost, st));
  OK_CUDA_TRY(cudaStreamSynchronize(st));
  if (loss) *loss = s / nb;
  return OK_SUCCESS;
}

int net_create(int layers, const double* w, ok_net** out) {
  if (!out || layers < 1 || layers > 16) return OK_EINVAL;
  *out = nullptr;
  ok_net* N = new (std::nothrow) ok_net();
  if (!N) return OK_ENOMEM;
  N->layers = layers;
  auto fail = [&](int rc) {
    cudaFree(N->A); cudaFree(N->m); cudaFree(N->v); cudaFree(N->gacc); cudaFree(N->scal); cudaFree(N->ticket);
    delete N;
    return rc;
  };
  if (cudaGetDevice(&N->device) != cudaSuccess) return fail(OK_ECUDA);
  const size_t np = (size_t)NPAR * layers;
  if (cudaMalloc(&N->A, np * sizeof(float)) != cudaSuccess || cudaMalloc(&N->m, np * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&N->v, np * sizeof(float)) != cudaSuccess || cudaMalloc(&N->gacc, np * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&N->scal, (2 + 2 * MAX_GROUP) * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&N->ticket, MAX_GROUP * sizeof(unsigned)) != cudaSuccess)
    return fail(OK_ENOMEM);
  if (cudaMemset(N->m, 0, np * sizeof(float)) != cudaSuccess || cudaMemset(N->v, 0, np * sizeof(float)) != cudaSuccess ||
      cudaMemset(N->ticket, 0, MAX_GROUP * sizeof(unsigned)) != cudaSuccess)
    return fail(OK_ECUDA);
  std::vector<float> h(np, 0.f);
  for (size_t i = 0; i < np; ++i) h[i] = w ? (float)w[i] : 0.f;
  if (!w)
    for (int l = 0; l < layers; ++l)
      for (int s = 0; s < 4; ++s) h[(size_t)l * NPAR + 2 * (4 * s + s)] = 1.f;  // A_0 = 1: P = identity
  if (cudaMemcpy(N->A, h.data(), np * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return fail(OK_ECUDA);
  *out = N;
  return OK_SUCCESS;
}

void net_free(ok_net* N) {
  if (!N) return;
  cudaFree(N->A); cudaFree(N->m); cudaFree(N->v); cudaFree(N->gacc); cudaFree(N->scal); cudaFree(N->ticket);
  free_training(N->t);
  cudaFree(N->g[0]); cudaFree(N->g[1]);
  delete N;
}

int net_weights(ok_net* N, double* get, const double* set) {
  if (!N) return OK_EINVAL;
  const size_t np = (size_t)NPAR * N->layers;
  std::vector<float> h(np);
  if (set) {
    for (size_t i = 0; i < np; ++i) {
      if (!std::isfinite(set[i])) return OK_EINVAL;
      h[i] = (float)set[i];
    }
    OK_CUDA_TRY(cudaMemcpy(N->A, h.data(), np * sizeof(float), cudaMemcpyHostToDevice));
    OK_CUDA_TRY(cudaMemset(N->m, 0, np * sizeof(float)));
    OK_CUDA_TRY(cudaMemset(N->v, 0, np * sizeof(float)));
    N->adam_t = 0;
  }
  if (get) {
    OK_CUDA_TRY(cudaMemcpy(h.data(), N->A, np * sizeof(float), cudaMemcpyDeviceToHost));
    for (size_t i = 0; i < np; ++i) get[i] = h[i];
  }
  return OK_SUCCESS;
}

int net_layers(const ok_net* N) { return N ? N->layers : 0; }

}  // namespace okgb
