// BiCGStab vector updates with fused inner products (the "vector addition" work the paper times
// in Table 1c).  Vectors are complex arrays of n = 12 V entries, processed in 16-byte units
// (one complex double or two complex floats).  Every kernel first reads the solver's halt flag
// so that iterations enqueued after convergence are no-ops; scalars (alpha, omega, beta) are read
// from the device-resident state, so no host round trip is needed between kernels.
//
// The three iteration kernels (update_s, update_xr, update_p) also run batched over several
// right-hand sides: grid row blockIdx.y works on vectors offset by blockIdx.y * n with state
// st[blockIdx.y] and its own reduction partials (one launch for all systems of a multi-RHS solve).
#include "ok_launch.cuh"
#include "ok_reduce_dd.cuh"

#include <mutex>
#include <utility>
#include <vector>

namespace okgb {

constexpr int BLAS_THREADS = 256;

template <typename R> struct Unit;
template <> struct Unit<double> {
  using T = double2;
  static constexpr int NC = 1;
  __device__ static __forceinline__ void get(const T& u, cx<double> (&c)[1]) { c[0] = mk(u.x, u.y); }
  __device__ static __forceinline__ T put(const cx<double> (&c)[1]) { return make_double2(c[0].re, c[0].im); }
};
template <> struct Unit<float> {
  using T = float4;
  static constexpr int NC = 2;
  __device__ static __forceinline__ void get(const T& u, cx<float> (&c)[2]) { c[0] = mk(u.x, u.y); c[1] = mk(u.z, u.w); }
  __device__ static __forceinline__ T put(const cx<float> (&c)[2]) { return make_float4(c[0].re, c[0].im, c[1].re, c[1].im); }
};

template <typename R> __device__ __forceinline__ cx<R> scal(dcx z) { return mk<R>((R)z.re, (R)z.im); }

// The grid reduction of the precision R's kernels.
template <typename R, int NP>
__device__ __forceinline__ void grid_reduce_r(typename RedT<R>::T (&v)[NP], const RedArgs& ra, unsigned* ticket) {
  if constexpr (sizeof(R) == 4) grid_reduce_dd<NP, BLAS_THREADS>(v, ra, ticket);
  else grid_reduce<NP, BLAS_THREADS>(v, ra, ticket);
}

#define OK_GRID_STRIDE(i, n) for (long long i = blockIdx.x * (long long)BLAS_THREADS + threadIdx.x; i < (n); i += (long long)gridDim.x * BLAS_THREADS)

// The reducing kernels sum RED_CHUNK units per thread in the vectors' own precision and add each
// chunk's sums into the thread's FP64 totals: FP64 arithmetic runs at a small fraction of the FP32
// rate on this part, so an FP64 conversion and add per unit would bound the kernel.  A chunk's
// units (stride: the grid) are loaded together.  The order of every sum is fixed by the launch
// shape, so results are reproducible.
constexpr int RED_CHUNK = 8;
#define OK_CHUNK_STRIDE(i0, n) \
  for (long long i0 = blockIdx.x * (long long)BLAS_THREADS + threadIdx.x; i0 < (n); i0 += (long long)gridDim.x * BLAS_THREADS * RED_CHUNK)
#define OK_CHUNK_UNITS(i, i0, n)                   \
  _Pragma("unroll") for (int u_ = 0; u_ < RED_CHUNK; ++u_) \
    if (const long long i = (i0) + (long long)u_ * gridDim.x * BLAS_THREADS; i < (n))

// s = r - alpha v
template <typename R>
__global__ void __launch_bounds__(BLAS_THREADS) update_s_kernel(const typename Unit<R>::T* __restrict__ r,
                                                                const typename Unit<R>::T* __restrict__ v,
                                                                typename Unit<R>::T* __restrict__ s, long long nu,
                                                                const SolverState* __restrict__ st) {
  const long long off = (long long)blockIdx.y * nu;
  r += off; v += off; s += off; st += blockIdx.y;
  if (st->halt) return;
  using U = Unit<R>;
  const cx<R> al = scal<R>(st->alpha);
  OK_GRID_STRIDE(i, nu) {
    cx<R> a[U::NC], b[U::NC];
    U::get(r[i], a);
    U::get(v[i], b);
#pragma unroll
    for (int k = 0; k < U::NC; ++k) a[k] = a[k] - al * b[k];
    s[i] = U::put(a);
  }
}

// x += alpha p + omega s;  r = s - omega t;  sums <rhat, r>, <r, r>  ->  FIN_XR.  With sx set (right
// preconditioning: p and sx are the preconditioned directions P p and P s) x += alpha p + omega sx.
template <typename R>
__global__ void __launch_bounds__(BLAS_THREADS) update_xr_kernel(typename Unit<R>::T* __restrict__ x,
                                                                 const typename Unit<R>::T* __restrict__ p,
                                                                 const typename Unit<R>::T* __restrict__ s,
                                                                 const typename Unit<R>::T* __restrict__ t,
                                                                 typename Unit<R>::T* __restrict__ r,
                                                                 const typename Unit<R>::T* __restrict__ rhat,
                                                                 long long nu, SolverState* __restrict__ st,
                                                                 RedArgs ra, long long pstride,
                                                                 const typename Unit<R>::T* __restrict__ sx) {
  const long long off = (long long)blockIdx.y * nu;
  x += off; p += off; s += off; t += off; r += off; rhat += off; st += blockIdx.y;
  if (sx) sx += off;
  ra.st = st;
  ra.part += (long long)blockIdx.y * pstride;
  if (st->halt) return;
  using U = Unit<R>;
  const cx<R> al = scal<R>(st->alpha), om = scal<R>(st->omega);
  typename RedT<R>::T red[3] = {0, 0, 0};
  OK_CHUNK_STRIDE(i0, nu) {
    cx<R> d = mk<R>(0, 0);
    R n2 = 0;
    OK_CHUNK_UNITS(i, i0, nu) {
      cx<R> xv[U::NC], pv[U::NC], sv[U::NC], tv[U::NC], hv[U::NC], zv[U::NC];
      U::get(x[i], xv);
      U::get(p[i], pv);
      U::get(s[i], sv);
      U::get(t[i], tv);
      U::get(rhat[i], hv);
      if (sx) U::get(sx[i], zv);
#pragma unroll
      for (int k = 0; k < U::NC; ++k) {
        xv[k] = xv[k] + al * pv[k] + om * (sx ? zv[k] : sv[k]);
        sv[k] = sv[k] - om * tv[k];
        d = fma_cj(hv[k], sv[k], d);
        n2 += sv[k].re * sv[k].re + sv[k].im * sv[k].im;
      }
      x[i] = U::put(xv);
      r[i] = U::put(sv);
    }
    red_add(red[0], d.re);
    red_add(red[1], d.im);
    red_add(red[2], n2);
  }
  grid_reduce_r<R, 3>(red, ra, &st->ticket[2]);
}

// p = r + beta (p - omega v)
template <typename R>
__global__ void __launch_bounds__(BLAS_THREADS) update_p_kernel(typename Unit<R>::T* __restrict__ p,
                                                                const typename Unit<R>::T* __restrict__ r,
                                                                const typename Unit<R>::T* __restrict__ v,
                                                                long long nu, const SolverState* __restrict__ st) {
  const long long off = (long long)blockIdx.y * nu;
  p += off; r += off; v += off; st += blockIdx.y;
  if (st->halt) return;
  using U = Unit<R>;
  const cx<R> be = scal<R>(st->beta), om = scal<R>(st->omega);
  OK_GRID_STRIDE(i, nu) {
    cx<R> pv[U::NC], rv[U::NC], vv[U::NC];
    U::get(p[i], pv);
    U::get(r[i], rv);
    U::get(v[i], vv);
#pragma unroll
    for (int k = 0; k < U::NC; ++k) pv[k] = rv[k] + be * (pv[k] - om * vv[k]);
    p[i] = U::put(pv);
  }
}

// The inner products a BiCGStab half-iteration takes from its application of M, in a pass of their
// own (the FP32 applications run without a fused epilogue; the separate pass over two vectors
// costs less than the epilogue did): ALPHA: <a, b> (a = rhat, b = v) -> FIN_ALPHA;
// OMEGA: <a, b>, <a, a> (a = t, b = s) -> FIN_OMEGA.  S: the type of the totals.
template <typename R, bool OMEGA, typename S = typename RedT<R>::T>
__global__ void __launch_bounds__(BLAS_THREADS) dots_kernel(const typename Unit<R>::T* __restrict__ a,
                                                            const typename Unit<R>::T* __restrict__ b, long long nu,
                                                            SolverState* __restrict__ st, RedArgs ra, unsigned* ticket) {
  if (st->halt) return;
  using U = Unit<R>;
  S red[3] = {0, 0, 0};
  OK_CHUNK_STRIDE(i0, nu) {
    cx<R> d = mk<R>(0, 0);
    R n2 = 0;
    OK_CHUNK_UNITS(i, i0, nu) {
      cx<R> av[U::NC], bv[U::NC];
      U::get(a[i], av);
      U::get(b[i], bv);
#pragma unroll
      for (int k = 0; k < U::NC; ++k) {
        d = fma_cj(av[k], bv[k], d);
        if (OMEGA) n2 += av[k].re * av[k].re + av[k].im * av[k].im;
      }
    }
    red_add(red[0], d.re);
    red_add(red[1], d.im);
    red_add(red[2], n2);
  }
  constexpr int NP = OMEGA ? 3 : 2;
  S v[NP];
#pragma unroll
  for (int k = 0; k < NP; ++k) v[k] = red[k];
  if constexpr (std::is_same<S, double>::value) grid_reduce<NP, BLAS_THREADS>(v, ra, ticket);
  else grid_reduce_dd<NP, BLAS_THREADS>(v, ra, ticket);
}

// ---------------------------------------------------------------------------- small systems
// On a small lattice the five vector kernels of an FP32 iteration cost their launches, their grid
// completions and their last block's tail, not their bytes (4^3 x 8: 43 us an iteration, 12 us of it
// update_xr; now 25 us).  There one cluster of up to eight blocks does the work between two applications
// in one launch: it takes the inner products, finalises the scalars and streams the update, with cluster
// barriers in the place of kernel boundaries.  Block sums meet in the first block's shared memory and are
// added in a fixed tree, so a solve is reproducible; the state is worked on in shared memory as well, as
// its finalisation is one thread's chain of dependent accesses (18.2 -> 16.0 us for small_xrp).
constexpr int CL_THREADS = 1024;
constexpr int CL_MAX = 8;
__device__ __forceinline__ unsigned cl_rank() { unsigned r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ unsigned cl_size() { unsigned r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
struct ClusterShared {
  dd warp[3][CL_THREADS / 32];
  dd part[3];
  float sc[4];
  int halt;
  SolverState st;  // the first block's copy of the system's state: the finalisations work on it
};
static_assert(sizeof(SolverState) % 4 == 0 && sizeof(SolverState) / 4 <= CL_THREADS, "one word per thread");
// Copies the state into the first block's shared memory, or back; every thread of the block calls it.
__device__ __forceinline__ void cl_state(ClusterShared& sh, SolverState* st, bool load) {
  if (cl_rank() != 0) return;
  if (!load) __syncthreads();
  if (threadIdx.x < sizeof(SolverState) / 4) {
    unsigned* a = reinterpret_cast<unsigned*>(&sh.st) + threadIdx.x;
    unsigned* b = reinterpret_cast<unsigned*>(st) + threadIdx.x;
    if (load) *a = *b; else *b = *a;
  }
}
// The form that counts threads, not warps: lane 0 alone finalises, and the last round of a loop over units need not take
// a whole warp, so the lanes of a warp may arrive here apart (`.aligned` would want them converged).
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
// A 32-bit word of shared memory at the same place in block `rank` of the cluster.
__device__ __forceinline__ float cl_load(const void* p, unsigned rank) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), b;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(b) : "memory");
  return v;
}

// Sums v over the cluster and finalises on sh.st; sc[0..3] and the halt flag as `publish` leaves them in the
// first block's shared memory reach every block's.  Every thread of the cluster takes part.
template <int NP, typename Publish>
__device__ __forceinline__ void cl_finalise(dd (&v)[NP], ClusterShared& sh, int fin, Publish&& publish) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    dd x = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = x + shfl_xor_dd(x, o);
    if (lane == 0) sh.warp[k][warp] = x;
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      dd x = sh.warp[k][lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x = x + shfl_xor_dd(x, o);
      if (lane == 0) sh.part[k] = x;
    }
  }
  cl_sync();
  const unsigned rank = cl_rank();
  if (rank == 0 && warp == 0) {
    double tot[4] = {0.0, 0.0, 0.0, 0.0};
    dd x[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) {   // lane r takes block r's sum
      x[k] = dd(0.f, 0.f);
      if (lane < (int)cl_size()) x[k] = dd(cl_load(&sh.part[k].hi, lane), cl_load(&sh.part[k].lo, lane));
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) {
#pragma unroll
      for (int o = CL_MAX / 2; o > 0; o >>= 1) x[k] = x[k] + shfl_xor_dd(x[k], o);
      tot[k] = (double)x[k];
    }
    if (lane == 0) {
      finalise(&sh.st, fin, tot);
      publish(sh.sc);
      sh.halt = sh.st.halt;
    }
  }
  cl_sync();
  if (rank != 0 && threadIdx.x < 5) {
    if (threadIdx.x < 4) sh.sc[threadIdx.x] = cl_load(&sh.sc[threadIdx.x], 0);
    else sh.halt = __float_as_int(cl_load(&sh.halt, 0));
  }
  __syncthreads();
}

// <rhat, v> -> alpha;  s = r - alpha v.
__global__ void __launch_bounds__(CL_THREADS, 1) small_s_kernel(const float4* __restrict__ rhat, const float4* __restrict__ v,
                                                                const float4* __restrict__ r, float4* __restrict__ s, int nu,
                                                                SolverState* __restrict__ st) {
  __shared__ ClusterShared sh;
  if (st->halt) return;  // set before this launch, so the same for every block
  cl_state(sh, st, true);
  using U = Unit<float>;
  const int i0 = cl_rank() * CL_THREADS + threadIdx.x, step = cl_size() * CL_THREADS;
  dd red[2] = {dd(0.f, 0.f), dd(0.f, 0.f)};
  for (int i = i0; i < nu; i += step) {
    cx<float> a[2], b[2], d = mk<float>(0, 0);
    U::get(rhat[i], a);
    U::get(v[i], b);
#pragma unroll
    for (int k = 0; k < 2; ++k) d = fma_cj(a[k], b[k], d);
    red_add(red[0], d.re);
    red_add(red[1], d.im);
  }
  cl_finalise<2>(red, sh, FIN_ALPHA, [&](float* sc) { sc[0] = (float)sh.st.alpha.re; sc[1] = (float)sh.st.alpha.im; });
  cl_state(sh, st, false);
  if (!sh.halt) {
    const cx<float> al = mk(sh.sc[0], sh.sc[1]);
    for (int i = i0; i < nu; i += step) {
      cx<float> a[2], b[2];
      U::get(r[i], a);
      U::get(v[i], b);
#pragma unroll
      for (int k = 0; k < 2; ++k) a[k] = a[k] - al * b[k];
      s[i] = U::put(a);
    }
  }
  cl_sync();  // the first block's shared memory is read until here
}

// <t, s>, <t, t> -> omega;  x += alpha p + omega sx, r = s - omega t, <rhat, r>, <r, r> -> beta, convergence;
// p = r + beta (p - omega v).  px, sx: the directions of the solution update (p and s, or P p and P s with a
// right preconditioner P).
__global__ void __launch_bounds__(CL_THREADS, 1) small_xrp_kernel(float4* __restrict__ x, float4* p, const float4* px,
                                                                  const float4* __restrict__ s, const float4* sx,
                                                                  const float4* __restrict__ t, float4* __restrict__ r,
                                                                  const float4* __restrict__ rhat, const float4* __restrict__ v, int nu,
                                                                  SolverState* __restrict__ st) {
  __shared__ ClusterShared sh;
  if (st->halt) return;
  cl_state(sh, st, true);
  using U = Unit<float>;
  const int i0 = cl_rank() * CL_THREADS + threadIdx.x, step = cl_size() * CL_THREADS;
  const cx<float> al = mk((float)st->alpha.re, (float)st->alpha.im);
  dd red[3] = {dd(0.f, 0.f), dd(0.f, 0.f), dd(0.f, 0.f)};
  for (int i = i0; i < nu; i += step) {
    cx<float> a[2], b[2], d = mk<float>(0, 0);
    float n2 = 0.f;
    U::get(t[i], a);
    U::get(s[i], b);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      d = fma_cj(a[k], b[k], d);
      n2 += a[k].re * a[k].re + a[k].im * a[k].im;
    }
    red_add(red[0], d.re);
    red_add(red[1], d.im);
    red_add(red[2], n2);
  }
  cl_finalise<3>(red, sh, FIN_OMEGA, [&](float* sc) { sc[0] = (float)sh.st.omega.re; sc[1] = (float)sh.st.omega.im; });
  const cx<float> om = mk(sh.sc[0], sh.sc[1]);
  if (sh.halt) {  // the same in every block
    cl_state(sh, st, false);
    cl_sync();
    return;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) red[k] = dd(0.f, 0.f);
  for (int i = i0; i < nu; i += step) {
    cx<float> xv[2], pv[2], sv[2], zv[2], tv[2], hv[2], d = mk<float>(0, 0);
    float n2 = 0.f;
    U::get(x[i], xv);
    U::get(px[i], pv);
    U::get(s[i], sv);
    U::get(sx[i], zv);
    U::get(t[i], tv);
    U::get(rhat[i], hv);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      xv[k] = xv[k] + al * pv[k] + om * zv[k];
      sv[k] = sv[k] - om * tv[k];
      d = fma_cj(hv[k], sv[k], d);
      n2 += sv[k].re * sv[k].re + sv[k].im * sv[k].im;
    }
    x[i] = U::put(xv);
    r[i] = U::put(sv);
    red_add(red[0], d.re);
    red_add(red[1], d.im);
    red_add(red[2], n2);
  }
  cl_sync();  // sc of omega is read; the sums' shared memory is free again
  cl_finalise<3>(red, sh, FIN_XR, [&](float* sc) { sc[2] = (float)sh.st.beta.re; sc[3] = (float)sh.st.beta.im; });
  cl_state(sh, st, false);
  if (!sh.halt) {
    const cx<float> be = mk(sh.sc[2], sh.sc[3]);
    for (int i = i0; i < nu; i += step) {
      cx<float> pv[2], rv[2], vv[2];
      U::get(p[i], pv);
      U::get(r[i], rv);
      U::get(v[i], vv);
#pragma unroll
      for (int k = 0; k < 2; ++k) pv[k] = rv[k] + be * (pv[k] - om * vv[k]);
      p[i] = U::put(pv);
    }
  }
  cl_sync();
}

// Restart: rhat = p = r (same precision), sum <r, r> -> FIN_RESTART.
template <typename R>
__global__ void __launch_bounds__(BLAS_THREADS) restart_kernel(const typename Unit<R>::T* __restrict__ r,
                                                               typename Unit<R>::T* __restrict__ rhat,
                                                               typename Unit<R>::T* __restrict__ p, long long nu,
                                                               SolverState* __restrict__ st, RedArgs ra) {
  using U = Unit<R>;
  typename RedT<R>::T red[1] = {0};
  OK_CHUNK_STRIDE(i0, nu) {
    R n2 = 0;
    OK_CHUNK_UNITS(i, i0, nu) {
      typename U::T u = r[i];
      rhat[i] = u;
      p[i] = u;
      cx<R> a[U::NC];
      U::get(u, a);
#pragma unroll
      for (int k = 0; k < U::NC; ++k) n2 += a[k].re * a[k].re + a[k].im * a[k].im;
    }
    red_add(red[0], n2);
  }
  grid_reduce_r<R, 1>(red, ra, &st->ticket[3]);
}

// Mixed precision: r32 = (float) r64; RESTART: rhat = p = r32 and FIN_RESTART on <r, r>;
// otherwise FIN_CONTINUE on <rhat, r32>, <r32, r32>.  Units are complex doubles here.
template <bool RESTART>
__global__ void __launch_bounds__(BLAS_THREADS) demote_kernel(const double2* __restrict__ r64, float2* __restrict__ r32,
                                                              float2* __restrict__ rhat, float2* __restrict__ p,
                                                              long long n, SolverState* __restrict__ st, RedArgs ra) {
  double red[3] = {0.0, 0.0, 0.0};
  OK_CHUNK_STRIDE(i0, n) {
    float c[3] = {0.f, 0.f, 0.f};
    OK_CHUNK_UNITS(i, i0, n) {
      double2 d = r64[i];
      float2 f = make_float2((float)d.x, (float)d.y);
      r32[i] = f;
      if (RESTART) {
        rhat[i] = f;
        p[i] = f;
        c[0] += f.x * f.x + f.y * f.y;
      } else {
        float2 h = rhat[i];
        c[0] += h.x * f.x + h.y * f.y;
        c[1] += h.x * f.y - h.y * f.x;
        c[2] += f.x * f.x + f.y * f.y;
      }
    }
    red[0] += c[0];
    red[1] += c[1];
    red[2] += c[2];
  }
  if (RESTART) {
    double v1[1] = {red[0]};
    grid_reduce<1, BLAS_THREADS>(v1, ra, &st->ticket[4]);
  } else {
    grid_reduce<3, BLAS_THREADS>(red, ra, &st->ticket[4]);
  }
}

// Mixed precision: x64 += x32, x32 = 0.
__global__ void __launch_bounds__(BLAS_THREADS) accum_x_kernel(double2* __restrict__ x64, float2* __restrict__ x32, long long n) {
  OK_GRID_STRIDE(i, n) {
    float2 f = x32[i];
    double2 d = x64[i];
    d.x += (double)f.x;
    d.y += (double)f.y;
    x64[i] = d;
    x32[i] = make_float2(0.f, 0.f);
  }
}

// <x, x> and <b, b> (FP64 vectors, complex-double units).
__global__ void __launch_bounds__(BLAS_THREADS) norms_kernel(const double2* __restrict__ x, const double2* __restrict__ b,
                                                             long long n, SolverState* __restrict__ st, RedArgs ra) {
  double red[2] = {0.0, 0.0};
  OK_GRID_STRIDE(i, n) {
    double2 u = x[i], v = b[i];
    red[0] += u.x * u.x + u.y * u.y;
    red[1] += v.x * v.x + v.y * v.y;
  }
  grid_reduce<2, BLAS_THREADS>(red, ra, &st->ticket[6]);
}

// ---------------------------------------------------------------------------- launchers
static int g_sms = 0;

int sm_count() {
  if (g_sms == 0) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 132;
    g_sms = sms;
  }
  return g_sms;
}

// Upper bound of every vector kernel's grid width (sizes the reduction partials).
int blas_blocks(long long units) {
  long long need = (units + BLAS_THREADS - 1) / BLAS_THREADS;
  long long cap = (long long)sm_count() * 8;
  return (int)(need < cap ? (need > 0 ? need : 1) : cap);
}

// Grid width for one vector kernel: one full wave of the blocks that fit on the device at once
// (from the occupancy calculator; a grid-stride loop covers the rest).  A wider grid would leave a
// partial second wave that every thread of the first must wait for: the kernels that hold more
// registers (update_xr at 48) fit 5 blocks of 256 threads per SM, not 8.
// Kernels that end in a grid reduction take at most this many blocks per multiprocessor: every
// block's partial ends in a fence and an atomic on one completion counter, and at a full wave
// (up to 8 x 152 blocks) those serialised atomics cost more than the few extra loads in flight.
#ifndef OK_RED_BLOCKS_PER_SM
#define OK_RED_BLOCKS_PER_SM 4
#endif
template <typename K>
static int wave_blocks(K kern, long long units, bool reduces = false) {
  static std::mutex mu;
  static std::vector<std::pair<const void*, int>> cache;
  int per_sm = 0;
  {
    std::lock_guard<std::mutex> lk(mu);
    for (const auto& e : cache)
      if (e.first == (const void*)kern) per_sm = e.second;
    if (per_sm == 0) {
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, BLAS_THREADS, 0) != cudaSuccess || per_sm < 1)
        per_sm = 1;
      if (per_sm > 8) per_sm = 8;
      cache.emplace_back((const void*)kern, per_sm);
    }
  }
  if (reduces && per_sm > OK_RED_BLOCKS_PER_SM) per_sm = OK_RED_BLOCKS_PER_SM;
  const long long need = (units + BLAS_THREADS - 1) / BLAS_THREADS;
  const long long cap = (long long)sm_count() * per_sm;
  return (int)(need < cap ? (need > 0 ? need : 1) : cap);
}

template <typename R> long long units_of(long long ncomplex) { return ncomplex / Unit<R>::NC; }

// One cluster of blocks, as many as give every thread a unit and a half, at most CL_MAX.
// Up to 49152 units (8192 sites).  One solve, separate kernels / one cluster (us): 512 sites 2473 / 2088,
// 4096 sites 2974 / 2516, 8192 sites 3192 / 3029, 16000 sites 3868 / 4347.
constexpr long long CL_UNITS = 49152;
bool small_system(long long n) { return units_of<float>(n) <= CL_UNITS; }

template <typename... P, typename... A>
static cudaError_t launch_cluster(void (*kern)(P...), int nu, cudaStream_t strm, A... args) {
  int nr = (nu + CL_THREADS + CL_THREADS / 2 - 1) / (CL_THREADS + CL_THREADS / 2);
  if (nr > CL_MAX) nr = CL_MAX;
  if (nr < 1) nr = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nr);
  cfg.blockDim = dim3(CL_THREADS);
  cfg.stream = strm;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nr;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

int launch_small_s(const cx<float>* rhat, const cx<float>* v, const cx<float>* r, cx<float>* s, long long n, SolverState* st,
                   cudaStream_t strm) {
  const int nu = (int)units_of<float>(n);
  {
    TraceScope ts("small_s_f32", strm);
    OK_CUDA_TRY(launch_cluster(small_s_kernel, nu, strm, (const float4*)rhat, (const float4*)v, (const float4*)r, (float4*)s, nu, st));
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

int launch_small_xrp(cx<float>* x, cx<float>* p, const cx<float>* px, const cx<float>* s, const cx<float>* sx, const cx<float>* t,
                     cx<float>* r, const cx<float>* rhat, const cx<float>* v, long long n, SolverState* st, cudaStream_t strm) {
  const int nu = (int)units_of<float>(n);
  {
    TraceScope ts("small_xrp_f32", strm);
    OK_CUDA_TRY(launch_cluster(small_xrp_kernel, nu, strm, (float4*)x, (float4*)p, (const float4*)px, (const float4*)s,
                               (const float4*)sx, (const float4*)t, (float4*)r, (const float4*)rhat, (const float4*)v, nu, st));
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

template <typename R>
int launch_update_s(const cx<R>* r, const cx<R>* v, cx<R>* s, long long n, const SolverState* st, cudaStream_t strm) {
  using T = typename Unit<R>::T;
  long long nu = units_of<R>(n);
  {
    TraceScope ts(sizeof(R) == 8 ? "update_s_f64" : "update_s_f32", strm);
    update_s_kernel<R><<<wave_blocks(update_s_kernel<R>, nu), BLAS_THREADS, 0, strm>>>((const T*)r, (const T*)v, (T*)s, nu, st);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

template <typename R>
int launch_update_xr(cx<R>* x, const cx<R>* p, const cx<R>* s, const cx<R>* t, cx<R>* r, const cx<R>* rhat, long long n,
                     SolverState* st, double* part, cudaStream_t strm, const cx<R>* sx) {
  using T = typename Unit<R>::T;
  long long nu = units_of<R>(n);
  RedArgs ra{st, part, nullptr, FIN_XR};
  {
    TraceScope ts(sizeof(R) == 8 ? "update_xr_f64" : "update_xr_f32", strm);
    update_xr_kernel<R><<<wave_blocks(update_xr_kernel<R>, nu, true), BLAS_THREADS, 0, strm>>>((T*)x, (const T*)p, (const T*)s, (const T*)t, (T*)r,
                                                                  (const T*)rhat, nu, st, ra, 0, (const T*)sx);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

template <typename R>
int launch_dots(const cx<R>* a, const cx<R>* b, long long n, bool omega, SolverState* st, double* part, cudaStream_t strm) {
  using T = typename Unit<R>::T;
  long long nu = units_of<R>(n);
  RedArgs ra{st, part, nullptr, omega ? FIN_OMEGA : FIN_ALPHA};
  {
    TraceScope ts(omega ? (sizeof(R) == 8 ? "dots_ts_f64" : "dots_ts_f32") : (sizeof(R) == 8 ? "dot_rv_f64" : "dot_rv_f32"), strm);
    if (omega)
      dots_kernel<R, true><<<wave_blocks(dots_kernel<R, true>, nu, true), BLAS_THREADS, 0, strm>>>((const T*)a, (const T*)b, nu, st, ra,
                                                                                          &st->ticket[omega ? 1 : 0]);
    else
      dots_kernel<R, false><<<wave_blocks(dots_kernel<R, false>, nu, true), BLAS_THREADS, 0, strm>>>((const T*)a, (const T*)b, nu, st, ra,
                                                                                            &st->ticket[0]);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

int launch_sums(const cx<float>* a, const cx<float>* b, long long n, bool norm, SolverState* st, double* part, cudaStream_t strm) {
  const long long nu = units_of<float>(n);
  const RedArgs ra{st, part, nullptr, FIN_NONE};
  auto kern = norm ? dots_kernel<float, true, double> : dots_kernel<float, false, double>;
  {
    TraceScope ts("sums_f32", strm);
    kern<<<wave_blocks(kern, nu, true), BLAS_THREADS, 0, strm>>>((const float4*)a, (const float4*)b, nu, st, ra, &st->ticket[0]);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

template <typename R>
int launch_update_p(cx<R>* p, const cx<R>* r, const cx<R>* v, long long n, const SolverState* st, cudaStream_t strm) {
  using T = typename Unit<R>::T;
  long long nu = units_of<R>(n);
  {
    TraceScope ts(sizeof(R) == 8 ? "update_p_f64" : "update_p_f32", strm);
    update_p_kernel<R><<<wave_blocks(update_p_kernel<R>, nu), BLAS_THREADS, 0, strm>>>((T*)p, (const T*)r, (const T*)v, nu, st);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

template <typename R>
int launch_restart(const cx<R>* r, cx<R>* rhat, cx<R>* p, long long n, SolverState* st, double* part, cudaStream_t strm) {
  using T = typename Unit<R>::T;
  long long nu = units_of<R>(n);
  RedArgs ra{st, part, nullptr, FIN_RESTART};
  {
    TraceScope ts(sizeof(R) == 8 ? "restart_f64" : "restart_f32", strm);
    restart_kernel<R><<<wave_blocks(restart_kernel<R>, nu), BLAS_THREADS, 0, strm>>>((const T*)r, (T*)rhat, (T*)p, nu, st, ra);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

// Batched over nrhs systems (vectors [nrhs][n], states [nrhs]); reductions use part + k * pstride
// for system k, pstride >= 3 * blas_blocks(n / units).
int launch_update_s_multi(const cx<float>* r, const cx<float>* v, cx<float>* s, long long n, int nrhs, const SolverState* st,
                          cudaStream_t strm) {
  using T = Unit<float>::T;
  const long long nu = units_of<float>(n);
  {
    TraceScope ts("update_s_multi", strm);
    update_s_kernel<float><<<dim3(wave_blocks(update_s_kernel<float>, nu), nrhs), BLAS_THREADS, 0, strm>>>((const T*)r, (const T*)v, (T*)s, nu, st);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

int launch_update_xr_multi(cx<float>* x, const cx<float>* p, const cx<float>* s, const cx<float>* t, cx<float>* r,
                           const cx<float>* rhat, long long n, int nrhs, SolverState* st, double* part, long long pstride,
                           cudaStream_t strm, const cx<float>* sx) {
  using T = Unit<float>::T;
  const long long nu = units_of<float>(n);
  if (pstride < 3LL * blas_blocks(nu)) return OK_EINVAL;
  RedArgs ra{st, part, nullptr, FIN_XR};
  {
    TraceScope ts("update_xr_multi", strm);
    update_xr_kernel<float><<<dim3(wave_blocks(update_xr_kernel<float>, nu), nrhs), BLAS_THREADS, 0, strm>>>(
        (T*)x, (const T*)p, (const T*)s, (const T*)t, (T*)r, (const T*)rhat, nu, st, ra, pstride, (const T*)sx);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

int launch_update_p_multi(cx<float>* p, const cx<float>* r, const cx<float>* v, long long n, int nrhs, const SolverState* st,
                          cudaStream_t strm) {
  using T = Unit<float>::T;
  const long long nu = units_of<float>(n);
  {
    TraceScope ts("update_p_multi", strm);
    update_p_kernel<float><<<dim3(wave_blocks(update_p_kernel<float>, nu), nrhs), BLAS_THREADS, 0, strm>>>((T*)p, (const T*)r, (const T*)v, nu, st);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

int launch_demote(const cx<double>* r64, cx<float>* r32, cx<float>* rhat, cx<float>* p, long long n, bool restart,
                  SolverState* st, double* part, cudaStream_t strm) {
  if (restart) {
    const int nb = wave_blocks(demote_kernel<true>, n);
    RedArgs ra{st, part, nullptr, FIN_RESTART};
    {
    TraceScope ts("demote_restart", strm);
    demote_kernel<true><<<nb, BLAS_THREADS, 0, strm>>>((const double2*)r64, (float2*)r32, (float2*)rhat, (float2*)p, n, st, ra);
  }
  } else {
    const int nb = wave_blocks(demote_kernel<false>, n);
    RedArgs ra{st, part, nullptr, FIN_CONTINUE};
    {
    TraceScope ts("demote_continue", strm);
    demote_kernel<false><<<nb, BLAS_THREADS, 0, strm>>>((const double2*)r64, (float2*)r32, (float2*)rhat, (float2*)p, n, st, ra);
  }
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

int launch_accum_x(cx<double>* x64, cx<float>* x32, long long n, cudaStream_t strm) {
  {
    TraceScope ts("accum_x", strm);
    accum_x_kernel<<<wave_blocks(accum_x_kernel, n), BLAS_THREADS, 0, strm>>>((double2*)x64, (float2*)x32, n);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

int launch_norms(const cx<double>* x, const cx<double>* b, long long n, SolverState* st, double* part, cudaStream_t strm) {
  RedArgs ra{st, part, nullptr, FIN_RESID};
  {
    TraceScope ts("norms_f64", strm);
    norms_kernel<<<wave_blocks(norms_kernel, n), BLAS_THREADS, 0, strm>>>((const double2*)x, (const double2*)b, n, st, ra);
  }
  OK_LAUNCH_CHECK();
  return OK_SUCCESS;
}

template int launch_update_s<double>(const cx<double>*, const cx<double>*, cx<double>*, long long, const SolverState*, cudaStream_t);
template int launch_update_s<float>(const cx<float>*, const cx<float>*, cx<float>*, long long, const SolverState*, cudaStream_t);
template int launch_dots<float>(const cx<float>*, const cx<float>*, long long, bool, SolverState*, double*, cudaStream_t);
template int launch_dots<double>(const cx<double>*, const cx<double>*, long long, bool, SolverState*, double*, cudaStream_t);
template int launch_update_xr<double>(cx<double>*, const cx<double>*, const cx<double>*, const cx<double>*, cx<double>*, const cx<double>*, long long, SolverState*, double*, cudaStream_t, const cx<double>*);
template int launch_update_xr<float>(cx<float>*, const cx<float>*, const cx<float>*, const cx<float>*, cx<float>*, const cx<float>*, long long, SolverState*, double*, cudaStream_t, const cx<float>*);
template int launch_update_p<double>(cx<double>*, const cx<double>*, const cx<double>*, long long, const SolverState*, cudaStream_t);
template int launch_update_p<float>(cx<float>*, const cx<float>*, const cx<float>*, long long, const SolverState*, cudaStream_t);
template int launch_restart<double>(const cx<double>*, cx<double>*, cx<double>*, long long, SolverState*, double*, cudaStream_t);
template int launch_restart<float>(const cx<float>*, cx<float>*, cx<float>*, long long, SolverState*, double*, cudaStream_t);

}  // namespace okgb
