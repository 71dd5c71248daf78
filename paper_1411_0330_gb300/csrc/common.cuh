// common.cuh -- device-side types and helpers shared by the liblsh kernels.
//
// Precision-generic complex arithmetic (float2 / double2), the device-resident
// CG state, and deterministic block / grid reductions (per-block partials in
// FP64, summed in block-index order by the last block to finish: no spin
// waits, bit-identical results run to run).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lsh {

template <typename T> struct cplx_of;
template <> struct cplx_of<float> { typedef float2 type; };
template <> struct cplx_of<double> { typedef double2 type; };
template <typename T> using C2 = typename cplx_of<T>::type;

template <typename T> __device__ __forceinline__ C2<T> mkc(T a, T b) {
  C2<T> r;
  r.x = a;
  r.y = b;
  return r;
}
template <typename T> __device__ __forceinline__ C2<T> cadd(C2<T> a, C2<T> b) { return mkc<T>(a.x + b.x, a.y + b.y); }
template <typename T> __device__ __forceinline__ C2<T> csub(C2<T> a, C2<T> b) { return mkc<T>(a.x - b.x, a.y - b.y); }
// a * b
template <typename T> __device__ __forceinline__ C2<T> cmul(C2<T> a, C2<T> b) {
  return mkc<T>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
template <typename T> __device__ __forceinline__ C2<T> cmulc(C2<T> a, C2<T> b) {
  return mkc<T>(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
// a * (-i)  and  a * (+i)
template <typename T> __device__ __forceinline__ C2<T> cmul_mi(C2<T> a) { return mkc<T>(a.y, -a.x); }
template <typename T> __device__ __forceinline__ C2<T> cmul_pi(C2<T> a) { return mkc<T>(-a.y, a.x); }
template <typename T> __device__ __forceinline__ C2<T> cscale(C2<T> a, T s) { return mkc<T>(a.x * s, a.y * s); }

// Device-resident state of one Krylov solve.  Scalars are always FP64.
struct SolverState {
  double rr;        // (r_k, r_k)
  double rz;        // (r_k, D r_k), D the preconditioner (rr where there is none)
  double bb;        // (b, b) of the system being solved
  double tol2;      // stop when rr <= tol2 (= tol^2 bb)
  double alpha;     // alpha of the last completed iteration (0 after breakdown)
  double beta;      // beta_{k-1}
  double pq;        // (p_k, K p_k)
  double aux[4];    // extra reduction results: residual norm; in a CG solve of the fused plane
                    // schedule (p, M p), (z, M z), (z, M p) (kernels_plane.cu)
  int iter;         // completed CG iterations
  int done;         // nonzero: converged or failed, later kernels return at once
  int status;       // lsh_status-compatible code set on device (0, breakdown)
  int pad;          // setup scan: largest phase id; solves in a cluster: timed iterations
  unsigned int counter[4];  // last-block counters, reset by the last block
};

// The flag as the kernel ahead left it.  A kernel that may start before the one ahead has
// ended (griddep_wait, chain_wait) reads the state through a volatile pointer: a load of
// const __restrict__ data may come from a cache that such a kernel's start has not emptied.
__device__ __forceinline__ bool is_done(const SolverState* st) {
  return *reinterpret_cast<const volatile int*>(&st->done) != 0;
}

// Per-thread accumulator for inner products.  FP64 fields: plain double sum.
// FP32 fields: Kahan-compensated float sum (the FP64 pipe of GB300 is 64x
// slower than the FP32 one), handed to the FP64 block / grid reduction.
template <typename T> struct Acc;
template <> struct Acc<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ void mac(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ double get() const { return s; }
};
template <> struct Acc<float> {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float v) {
    const float y = v - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
  }
  // add(a * b) with one rounding for the product and the compensation together
  __device__ __forceinline__ void mac(float a, float b) {
    const float y = fmaf(a, b, -c);
    const float t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ double get() const { return (double)s - (double)c; }
};

// Two FP32 accumulators side by side for products that come in pairs (the two parts of a
// complex value, neighbouring voxels): the operations of Acc<float>::mac on both halves of
// packed registers.
struct Acc2 {
  float2 s = {0.0f, 0.0f}, n = {0.0f, 0.0f};  // n: minus the compensation
  __device__ __forceinline__ void mac(float2 a, float2 b) {
    const float2 m = make_float2(-1.0f, -1.0f);
    const float2 y = __ffma2_rn(a, b, n);
    const float2 t = __fadd2_rn(s, y);
    n = __ffma2_rn(m, __ffma2_rn(m, s, t), y);  // y - (t - s)
    s = t;
  }
  // both sums times w (a power of two) as one compensated pair
  __device__ __forceinline__ Acc<float> fold(float w = 1.0f) const {
    Acc<float> a;
    a.s = s.x + s.y;
    const float bp = a.s - s.x;
    a.c = -(n.x + n.y) - ((s.x - (a.s - bp)) + (s.y - bp));  // s.x + s.y = a.s + the bracket exactly
    a.s *= w;
    a.c *= w;
    return a;
  }
};

// Block sum of per-thread accumulators; result valid in thread 0.  FP32
// compensated pairs are first merged across the warp in FP32 (TwoSum keeps
// the rounding error of each merge), so only one value per warp touches the
// FP64 pipe.
__device__ __forceinline__ double block_sum(double v);
__device__ __forceinline__ double block_reduce(const Acc<double>& a) { return block_sum(a.get()); }
__device__ __forceinline__ void warp_merge_pair(float& s, float& c) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float s2 = __shfl_down_sync(0xffffffffu, s, o);
    const float c2 = __shfl_down_sync(0xffffffffu, c, o);
    const float t = s + s2;
    const float bp = t - s;
    const float e = (s - (t - bp)) + (s2 - bp);  // s + s2 = t + e exactly
    s = t;
    c = c + c2 - e;
  }
}
__device__ __forceinline__ double block_reduce(const Acc<float>& a) {
  __shared__ float pair_sh[2][32];
  float s = a.s, c = a.c;  // value = s - c
  warp_merge_pair(s, c);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) {
    pair_sh[0][w] = s;
    pair_sh[1][w] = c;
  }
  __syncthreads();
  double out = 0.0;
  if (w == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    s = l < nw ? pair_sh[0][l] : 0.0f;
    c = l < nw ? pair_sh[1][l] : 0.0f;
    warp_merge_pair(s, c);
    if (l == 0) out = (double)s - (double)c;
  }
  return out;
}

// Quotients by a divisor that is uniform across the block: one multiplication with
// ceil(2^32 / d), exact for dividends and divisors below 2^16 (every index inside a
// block's shared-memory tile).  The mixed-radix stages spend most of their integer
// work on such splits; an integer division is some twenty instructions.
struct FastDiv {
  unsigned d, m;
  __host__ __device__ __forceinline__ static unsigned magic(int d) { return d == 1 ? 0u : 0xffffffffu / (unsigned)d + 1u; }
  __device__ __forceinline__ explicit FastDiv(int d_) : d((unsigned)d_), m(magic(d_)) {}
  __device__ __forceinline__ FastDiv(int d_, unsigned m_) : d((unsigned)d_), m(m_) {}
  __device__ __forceinline__ int div(int a) const { return d == 1u ? a : (int)__umulhi((unsigned)a, m); }
};

// FFT plan of one axis: length n = product of the radices, DIF stage order.
#define LSH_MAX_STAGES 8
struct Plan1D {
  int n;
  int nst;
  int radix[LSH_MAX_STAGES];
  int m[LSH_MAX_STAGES];             // distance between a butterfly's inputs: span / radix
  int tws[LSH_MAX_STAGES];           // twiddle stride n / span
  unsigned mag_m[LSH_MAX_STAGES];    // FastDiv factors of m and of n / radix
  unsigned mag_nb[LSH_MAX_STAGES];
};

// The cheapest sequence of radices (descending, each at most 12) whose product is n, by
// the sum of cost(radix) over the stages; its length in *nst, 0 if there is none.
template <typename Cost> inline void lsh_best_radices(int left, int from, int k, double c, const Cost& cost, int* cur,
                                                      double* best, int* bestr, int* nst) {
  if (left == 1) {
    if (c < *best) {
      *best = c;
      *nst = k;
      for (int i = 0; i < k; ++i) bestr[i] = cur[i];
    }
    return;
  }
  if (k == LSH_MAX_STAGES) return;
  for (int r = from; r >= 2; --r) {
    if (r == 11 || left % r != 0) continue;
    cur[k] = r;
    lsh_best_radices(left / r, r, k + 1, c + cost(r), cost, cur, best, bestr, nst);
  }
}

// A length whose factors 8, 4, 2, 3, 5, 7 number more than LSH_MAX_STAGES is not taken.
inline bool lsh_plan_length(int n) {
  if (n < 1) return false;
  int small = 0;
  for (int q : {8, 4, 2, 3, 5, 7})
    while (n % q == 0) { n /= q; ++small; }
  return n == 1 && small <= LSH_MAX_STAGES;
}

inline void lsh_fill_plan(int n, const int* radix, int nst, Plan1D* p) {
  *p = Plan1D{};
  p->n = n;
  p->nst = nst;
  int span = n;
  for (int i = 0; i < nst; ++i) {
    const int r = radix[i];
    p->radix[i] = r;
    p->m[i] = span / r;
    p->tws[i] = n / span;
    p->mag_m[i] = FastDiv::magic(p->m[i]);
    p->mag_nb[i] = FastDiv::magic(n / r);
    span /= r;
  }
}

// Plan of length n (factors 2, 3, 5, 7), false if there is none.  Every stage is a
// round trip through shared memory with a barrier, so the fewest stages win, then
// the fewest operations; larger radices first.  Radices up to 12 keep an FP64
// butterfly in 128 registers.  The lengths with compile-time schedules (fft.cuh) come
// out as those expect.
inline bool lsh_make_plan(int n, Plan1D* p) {
  if (!lsh_plan_length(n)) return false;
  // cost per point: a stage's own (shared-memory round trip, indices, twiddles) of 16 and
  // the butterfly's operations
  const auto cost = [](int r) {
    const double c[13] = {0, 0, 18, 21, 20, 23, 23, 26, 22, 28, 25, 0, 26};
    return c[r];
  };
  double best = 1e30;
  int cur[LSH_MAX_STAGES], r[LSH_MAX_STAGES] = {0}, nst = 0;
  switch (n) {
    case 128: nst = 3; r[0] = 4; r[1] = 8; r[2] = 4; break;
    case 256: nst = 3; r[0] = 8; r[1] = 8; r[2] = 4; break;
    case 96: nst = 2; r[0] = 12; r[1] = 8; break;
    case 64: nst = 2; r[0] = r[1] = 8; break;
    case 48: nst = 2; r[0] = 8; r[1] = 6; break;
    case 32: nst = 2; r[0] = 8; r[1] = 4; break;
    case 16: nst = 2; r[0] = r[1] = 4; break;
    default: lsh_best_radices(n, 12, 0, 0.0, cost, cur, &best, r, &nst);
  }
  lsh_fill_plan(n, r, nst, p);
  return true;
}

// Plan for `lines` lines in one block of `threads` threads, by the cycles of a stage: a
// barrier and the shared-memory round trip, and the instructions of a butterfly times
// the rounds of the threads.  FP64: a warp instruction holds its scheduler's share of the
// unit for 64 cycles, and radix 2 runs on two lanes per butterfly.  Measured, us per
// iteration of the cluster solver: 32 x 32 in radices 4, 4, 2 23.7, in 2s 20.9; 64 x 64
// rows in 8, 8 30.5, in 2s 29.5, in 4, 4, 4 26.9; 96 x 96 columns in 12, 8 42.8, in
// 6, 4, 4 39.8; 16^3 in 4, 4 27.8, in 8, 2 35.
inline bool lsh_make_plan_lines(int n, int lines, int threads, bool fp64, Plan1D* p) {
  if (!lsh_plan_length(n)) return false;
  const auto cost = [&](int r) {
    const double instr[13] = {0, 0, 16, 30, 36, 60, 66, 100, 92, 130, 140, 0, 160};
    const double instr64[13] = {0, 0, 5, 24, 28, 56, 60, 100, 84, 150, 136, 0, 156};
    const double items = (double)lines * n / r * (fp64 && r == 2 ? 2 : 1);
    const double warps = (double)(long long)((items + 31) / 32);
    const double rounds = (double)(long long)((items + threads - 1) / threads);
    if (fp64) return 250.0 + 100.0 * rounds + 16.0 * instr64[r] * (warps > 4.0 ? warps : 4.0);
    return 200.0 + instr[r] * (4.0 * rounds + warps / 4.0);
  };
  double best = 1e30;
  int cur[LSH_MAX_STAGES], r[LSH_MAX_STAGES] = {0}, nst = 0;
  lsh_best_radices(n, 12, 0, 0.0, cost, cur, &best, r, &nst);
  lsh_fill_plan(n, r, nst, p);
  return true;
}

// ---------------------------------------------------------------- reductions
// Sum of one double per thread; result valid in thread 0.  Deterministic for a
// fixed block size.  Every thread of the block must call it.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double red_sh[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red_sh[w] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  v = (threadIdx.x < (unsigned)nw) ? red_sh[threadIdx.x] : 0.0;
  if (w == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  }
  return v;
}

// Publish this block's partial and report whether the block is the last one
// of the grid to do so.  The last block then owns partials[0..nblocks).
__device__ __forceinline__ bool publish_partial(double* partials, double v, unsigned int* counter) {
  __shared__ int is_last;
  const unsigned int nb = gridDim.x * gridDim.y * gridDim.z;
  const unsigned int b = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  if (threadIdx.x == 0) {
    partials[b] = v;
    __threadfence();
    unsigned int t = atomicAdd(counter, 1u);
    is_last = (t == nb - 1);
  }
  __syncthreads();
  return is_last != 0;
}

// In the last block: ordered sum of the partials (result in thread 0), and
// counter reset for the next launch.
__device__ __forceinline__ double gather_partials(const double* partials, unsigned int* counter) {
  __threadfence();
  const unsigned int nb = gridDim.x * gridDim.y * gridDim.z;
  double s = 0.0;
  for (unsigned int i = threadIdx.x; i < nb; i += blockDim.x) s += __ldcg(partials + i);
  s = block_sum(s);
  if (threadIdx.x == 0) *counter = 0u;
  return s;
}

// Variants for a reduction over `nb` blocks of one system out of many in the
// grid: block `b` (0..nb-1 within its system) publishes to partials[b].
__device__ __forceinline__ bool publish_partial_sys(double* partials, unsigned int b, unsigned int nb, double v,
                                                    unsigned int* counter) {
  __shared__ int is_last_sys;
  if (threadIdx.x == 0) {
    partials[b] = v;
    __threadfence();
    unsigned int t = atomicAdd(counter, 1u);
    is_last_sys = (t == nb - 1);
  }
  __syncthreads();
  return is_last_sys != 0;
}

__device__ __forceinline__ double gather_partials_sys(const double* partials, unsigned int nb, unsigned int* counter) {
  __threadfence();
  double s = 0.0;
  for (unsigned int i = threadIdx.x; i < nb; i += blockDim.x) s += __ldcg(partials + i);
  s = block_sum(s);
  if (threadIdx.x == 0) *counter = 0u;
  return s;
}

// The same for two sums of one block: the second one's partials sit `off` further on.
__device__ __forceinline__ bool publish_partial_sys2(double* partials, long long off, unsigned int b, unsigned int nb,
                                                     double v, double w, unsigned int* counter) {
  if (threadIdx.x == 0) partials[off + b] = w;  // ordered before the ticket by publish_partial_sys's fence
  return publish_partial_sys(partials, b, nb, v, counter);
}

// Scalars of one system's MINRES recurrence (Lanczos + Givens, Paige-Saunders),
// kept on the device next to its SolverState.
struct MinresScalars {
  double beta1, beta, oldb, alfa;
  double dbar, epsln, oldeps, phibar;
  double cs, sn, phi, delta, denom;
  int pending;  // converged after this iteration's update of x
  int pad;
};

// Scalars of one system's SYMMLQ recurrence (Lanczos as for MINRES, whose
// MinresScalars keep beta1, beta, oldb and alfa; LQ factorisation of the
// tridiagonal matrix by rotations from the right, Paige-Saunders 1975).
struct SymmlqScalars {
  double gbar, dbar, rhs1, rhs2;
  double bstep, snprod;     // step along the first Lanczos vector, product of the sines
  double s, t, cs, sn;      // this iteration's update x += s w + t v, w <- sn w - cs v
  double zbar, cb;          // at exit: x += zbar w + cb b (the CG point)
  int pending;
  int pad;
};

}  // namespace lsh
