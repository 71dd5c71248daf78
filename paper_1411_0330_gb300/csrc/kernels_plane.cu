// kernels_plane.cu -- the x and y transforms of one z plane in one kernel
// (FP32, square planes nx = ny = N with N in {16, 32, 48, 64, 96, 128}).
//
// The operator of Eq. (13) transforms along x, y and z around the per-
// frequency Gamma^h product.  A z plane of one component (N^2 reals, at most
// 68 KB as a half spectrum) fits in shared memory, so both in-plane axes are
// done by one block and the spectrum makes one HBM round trip less per axis
// than with separate x and y passes.
//
// Forward (k_xyfwd): the CG prologue (x += alpha p_old, p = r + beta p_old) or
// the projection on I0 runs on coalesced 16-byte global accesses and leaves
// the real plane in shared memory.  Rows 2l and 2l+1 form one complex line,
// transformed along x by the two-level register FFT with the exchange inside
// the pair's own storage, and split into two Hermitian half rows
// X(kx) = (Z(kx) + conj Z(N-kx)) / 2, (Z(kx) - conj Z(N-kx)) / 2i.  Then the
// columns are transformed along y; columns 0 and N/2 hold real sequences and
// travel as one complex column X0 + i XN, separated afterwards.  The plane
// leaves as N rows of the half spectrum, one bulk copy per row, in the
// ky-major layout H[S][c][ky][z][hs]: the z pass then reads each (system,
// component, ky) slab [z][kx] as one contiguous range.  The Nyquist column
// kx = N/2 also goes to a compact array NQ[S][c][z][ky], so the z pass reads
// that column as 8 consecutive ky per z instead of one complex per row.
//
// Inverse (k_xyinv): the rows come back by bulk copies (bounded wait), the
// Nyquist column from NQ, the y and x inverse transforms run the same steps
// backwards (unnormalised: the Gamma table carries 1/V), and the epilogue
// adds the local term M_beta x_beta of Eq. (7), projects on I0 (zero where
// A_beta = A0, Eq. (4)) and, in a CG iteration, reduces this block's part of
// (p, K p) in FP64; k_dot_finalize sums the blocks of a system into alpha.
#include <algorithm>

#include "common.cuh"
#include "fft.cuh"
#include "internal.h"
#include "regfft.cuh"
#include "tma.cuh"

namespace lsh {

template <int N> struct PlaneCfg {
  typedef RegLine<float, N> RL;
  static constexpr int P = RL::P, R1 = RL::R1, Q = RL::Q;
  // row stride of the plane in shared memory (complex values, even: 16-byte
  // rows for the bulk copies), at least N/2 + 1.  A warp of the x phases holds
  // 32 / P row pairs; their bases, 2 RS apart, must fall on distinct banks for
  // the accesses along a line (stride 1 in t): RS = 4 (mod 8) for P = 8 (row
  // pairs 8 complex values apart modulo 16), RS = 2 (mod 8) for P = 4 (4 apart).
  // The global rows keep the handle's stride hs >= RS (32-byte rows for the z
  // pass); a bulk copy moves the first RS values of a row.
  static constexpr int RS = P >= 8 ? (N / 2 + 1 + 3) / 8 * 8 + 4 : (N / 2 + 6) / 8 * 8 + 2;
  static constexpr int LINES = N / 2;  // row pairs along x, packed columns along y
  static constexpr int TH = LINES * P < 256 ? LINES * P : 256;
  static constexpr int LPR = TH / P;   // lines per round
  static constexpr int ROUNDS = LINES / LPR;
  static constexpr int NV = N / 4;     // float4 groups per real row
  static constexpr int IT = N * NV / TH;
  static constexpr size_t SMEM = sizeof(float2) * ((size_t)N * RS + N);
  // resident blocks per SM the register budget must allow (three 70 KB planes at 128^2)
  static constexpr int MINB = N == 128 ? 3 : 4;
  static_assert(LINES % LPR == 0 && (N * NV) % TH == 0, "tiling");
  static_assert(N + N / R1 <= 2 * RS, "padded exchange fits in a row pair");
};

// x transform of the row pairs of the plane: real rows in, half rows out.
template <int N> __device__ __forceinline__ void plane_x_fwd(float2* PL, const float2* tw) {
  typedef PlaneCfg<N> PC;
  typedef typename PC::RL RL;
  constexpr int P = PC::P, R1 = PC::R1, RS = PC::RS;
  constexpr int NK = (RS + P - 1) / P;
  const int t = threadIdx.x % P, lr = threadIdx.x / P;
#pragma unroll 1
  for (int rd = 0; rd < PC::ROUNDS; ++rd) {
    float2* pair = PL + 2 * (lr + rd * PC::LPR) * RS;
    const float* ra = reinterpret_cast<const float*>(pair);
    const float* rb = ra + 2 * RS;
    float2 v[R1];
#pragma unroll
    for (int j = 0; j < R1; ++j) v[j] = make_float2(ra[t + P * j], rb[t + P * j]);
    __syncwarp();
    RL::fwd_a_p(v, t, tw, pair);
    __syncwarp();
    RL::fwd_b_p(v, t, tw, pair);
    __syncwarp();
#pragma unroll
    for (int m = 0; m < R1; ++m) pair[RL::freq(t, m)] = v[m];
    __syncwarp();
    // kx = t + P i lies in [P i, P (i + 1)): inside 0..N/2 for every t while
    // P (i + 1) <= N/2, for t = 0 only at i = N / (2P), outside beyond; kx = 0
    // pairs with itself
    float2 xa[NK], xb[NK];
#pragma unroll
    for (int i = 0; i < NK; ++i) {
      const int kx = t + P * i;
      xa[i] = make_float2(0.f, 0.f);
      xb[i] = xa[i];
      const bool in = P * (i + 1) <= N / 2 || (P * i <= N / 2 && kx <= N / 2);
      if (in) {
        const float2 z1 = pair[kx], z2 = pair[(i == 0 && t == 0) ? 0 : N - kx];
        xa[i] = make_float2(0.5f * (z1.x + z2.x), 0.5f * (z1.y - z2.y));
        xb[i] = make_float2(0.5f * (z1.y + z2.y), 0.5f * (z2.x - z1.x));
      }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NK; ++i) {
      const int kx = t + P * i;
      if (P * (i + 1) <= RS || kx < RS) {
        pair[kx] = xa[i];
        pair[RS + kx] = xb[i];
      }
    }
  }
}

// y transform of the columns 0 .. N/2 (0 and N/2 packed), forward.
template <int N> __device__ __forceinline__ void plane_y_fwd(float2* PL, const float2* tw) {
  typedef PlaneCfg<N> PC;
  typedef typename PC::RL RL;
  constexpr int P = PC::P, R1 = PC::R1, RS = PC::RS, LPR = PC::LPR;
  const int t = threadIdx.x / LPR, cl = threadIdx.x % LPR;
#pragma unroll 1
  for (int rd = 0; rd < PC::ROUNDS; ++rd) {
    const int col = cl + rd * LPR;
    float2* cp = PL + col;
    float2 v[R1];
    if (col == 0) {  // columns 0 and N/2 (real) as one complex column
#pragma unroll
      for (int j = 0; j < R1; ++j) v[j] = make_float2(PL[(t + P * j) * RS].x, PL[(t + P * j) * RS + N / 2].x);
    } else {
#pragma unroll
      for (int j = 0; j < R1; ++j) v[j] = cp[(t + P * j) * RS];
    }
    __syncthreads();
    RL::template fwd_a_s<RS>(v, t, tw, cp);
    __syncthreads();
    RL::template fwd_b_s<RS>(v, t, tw, cp);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < R1; ++m) cp[RL::freq(t, m) * RS] = v[m];
  }
  __syncthreads();
  // W = X0 + i XN with X0, XN Hermitian in ky: X0 = (W(k) + conj W(-k)) / 2,
  // XN = (W(k) - conj W(-k)) / 2i; the thread of ky also writes N - ky
  for (int ky = threadIdx.x; ky <= N / 2; ky += PC::TH) {
    const int km = ky == 0 ? 0 : N - ky;
    const float2 w1 = PL[ky * RS], w2 = PL[km * RS];
    const float2 x0 = make_float2(0.5f * (w1.x + w2.x), 0.5f * (w1.y - w2.y));
    const float2 xn = make_float2(0.5f * (w1.y + w2.y), 0.5f * (w2.x - w1.x));
    PL[ky * RS] = x0;
    PL[ky * RS + N / 2] = xn;
    if (km != ky) {
      PL[km * RS] = make_float2(x0.x, -x0.y);
      PL[km * RS + N / 2] = make_float2(xn.x, -xn.y);
    }
  }
  __syncthreads();
}

// y inverse transform of the columns (0 and N/2 packed), unnormalised.
template <int N> __device__ __forceinline__ void plane_y_inv(float2* PL, const float2* tw) {
  typedef PlaneCfg<N> PC;
  typedef typename PC::RL RL;
  constexpr int P = PC::P, R1 = PC::R1, RS = PC::RS, LPR = PC::LPR;
  const int t = threadIdx.x / LPR, cl = threadIdx.x % LPR;
#pragma unroll 1
  for (int rd = 0; rd < PC::ROUNDS; ++rd) {
    const int col = cl + rd * LPR;
    float2* cp = PL + col;
    float2 v[R1];
    if (col == 0) {
#pragma unroll
      for (int m = 0; m < R1; ++m) {
        const int f = RL::freq(t, m);
        const float2 x0 = PL[f * RS], xn = PL[f * RS + N / 2];
        v[m] = make_float2(x0.x - xn.y, x0.y + xn.x);  // X0 + i XN
      }
    } else {
#pragma unroll
      for (int m = 0; m < R1; ++m) v[m] = cp[RL::freq(t, m) * RS];
    }
    __syncthreads();
    RL::template inv_a_s<RS>(v, t, tw, cp);
    __syncthreads();
    RL::template inv_b_s<RS>(v, t, tw, cp);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < R1; ++j) {
      const int y = t + P * j;
      if (col == 0) {
        // the inverse of X0 + i XN is x0 + i xN with x0, xN real
        PL[y * RS] = make_float2(v[j].x, 0.f);
        PL[y * RS + N / 2] = make_float2(v[j].y, 0.f);
      } else {
        cp[y * RS] = v[j];
      }
    }
  }
  __syncthreads();
}

// x inverse transform of the row pairs: half rows in, N x real rows out.
template <int N> __device__ __forceinline__ void plane_x_inv(float2* PL, const float2* tw) {
  typedef PlaneCfg<N> PC;
  typedef typename PC::RL RL;
  constexpr int P = PC::P, R1 = PC::R1, Q = PC::Q, RS = PC::RS;
  const int t = threadIdx.x % P, lr = threadIdx.x / P;
#pragma unroll 1
  for (int rd = 0; rd < PC::ROUNDS; ++rd) {
    float2* pair = PL + 2 * (lr + rd * PC::LPR) * RS;
    float2 v[R1];
    // frequency f = t Q + q + R1 u lies in [R1 u, R1 (u + 1)): below N/2 for u < P/2,
    // read at N - f from u = P/2 on (f = N/2 included: X(N/2) of a row is real)
    const float2* up = pair + t * Q;      // X(f) at up[q + R1 u]
    const float2* dn = pair + N - t * Q;  // X(N - f) at dn[-(q + R1 u)]
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int u = 0; u < P; ++u) {
        const int c = q + R1 * u;
        // Z(f) = X_a(f) + i X_b(f), X(N - k) = conj X(k)
        if (u < P / 2) {
          const float2 xa = up[c], xb = up[RS + c];
          v[q * P + u] = make_float2(xa.x - xb.y, xa.y + xb.x);
        } else {
          const float2 xa = dn[-c], xb = dn[RS - c];
          v[q * P + u] = make_float2(xa.x + xb.y, xb.x - xa.y);
        }
      }
    __syncwarp();
    RL::inv_a_p(v, t, tw, pair);
    __syncwarp();
    RL::inv_b_p(v, t, tw, pair);
    __syncwarp();
    float* ra = reinterpret_cast<float*>(pair);
    float* rb = ra + 2 * RS;
#pragma unroll
    for (int j = 0; j < R1; ++j) {
      ra[t + P * j] = v[j].x;
      rb[t + P * j] = v[j].y;
    }
  }
}

// MODE 0: spectrum of P in (apply).  MODE 1 (CG): x += alpha p_old, p = r +
// beta p_old (p = r at the first iteration), spectrum of p.
template <int N, int MODE>
__global__ void __launch_bounds__(PlaneCfg<N>::TH, PlaneCfg<N>::MINB) k_xyfwd(OpArgs<float> a, const float* __restrict__ in,
                                                           float* __restrict__ x, const float* __restrict__ r,
                                                           float* __restrict__ p, const SolverState* __restrict__ st) {
  typedef PlaneCfg<N> PC;
  constexpr int RS = PC::RS, TH = PC::TH, NV = PC::NV;
  const int cnz = a.c * a.nz;
  const int s = blockIdx.x / cnz;
  const int blk = blockIdx.x - s * cnz;  // comp * nz + z
  const int comp = blk / a.nz, z = blk - comp * a.nz;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* PL = reinterpret_cast<float2*>(smem_raw);  // [N][RS]
  float2* tw = PL + N * RS;
  // the state is written by the kernel ahead: read after the wait, never from a cache of
  // invariant data
  const volatile SolverState* vst = st + s;
  if (MODE == 1) {
    griddep_wait();
    griddep_launch();
    if (vst->done) return;
  }
  float* PR = reinterpret_cast<float*>(PL);  // real row y at PR + 2 RS y
  __shared__ unsigned char aloc[256];
  for (int u = threadIdx.x; u < N; u += TH) tw[u] = a.twx[u];
  if (MODE == 0)
    for (int u = threadIdx.x; u < a.nphase; u += TH) aloc[u] = a.act[u];
  const long long plane = (long long)blockIdx.x * N * N;  // [S][c][nz] planes of N^2
  const long long pbase = (long long)((a.sys0 + s) / a.sys_per_ms) * a.V + (long long)z * N * N;
  int k = 0;
  float alpha = 0.f, beta = 0.f;
  if (MODE == 1) {
    k = vst->iter;
    alpha = (float)vst->alpha;
    beta = (float)vst->beta;
  }
  if (MODE == 0) {
    __syncthreads();  // aloc
#pragma unroll 4
    for (int it = 0; it < PC::IT; ++it) {
      const int idx = threadIdx.x + it * TH;
      const int row = idx / NV, xx = (idx - row * NV) * 4;
      const long long g = plane + (long long)row * N + xx;
      float4 v = *reinterpret_cast<const float4*>(in + g);
      const uchar4 ph = *reinterpret_cast<const uchar4*>(a.phase + pbase + row * N + xx);
      if (!aloc[ph.x]) v.x = 0.f;
      if (!aloc[ph.y]) v.y = 0.f;
      if (!aloc[ph.z]) v.z = 0.f;
      if (!aloc[ph.w]) v.w = 0.f;
      *reinterpret_cast<float4*>(PR + 2 * RS * row + xx) = v;
    }
  } else {
    // The r plane comes into the real rows of the plane buffer by one bulk copy
    // per row; p and x go through registers in batches of B groups of four
    // reals, each batch's loads in flight while the previous batch is combined.
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
      mbar_init(&bar, 1);
      mbar_init_fence();
      mbar_expect_tx(&bar, (uint32_t)(sizeof(float) * N * N));
    }
    __syncthreads();
    for (int row = threadIdx.x; row < N; row += TH)
      bulk_load_1d(PR + 2 * RS * row, r + plane + (long long)row * N, (uint32_t)(sizeof(float) * N), &bar);
    constexpr int B = PC::IT % 4 == 0 ? 4 : (PC::IT % 3 == 0 ? 3 : (PC::IT % 2 == 0 ? 2 : 1));
    static_assert(PC::IT % B == 0, "batches");
    float4 pb[B], xb[B];
    auto load_batch = [&](int it0) {
#pragma unroll
      for (int b = 0; b < B; ++b) {
        const int idx = threadIdx.x + (it0 + b) * TH;
        const int row = idx / NV, xx = (idx - row * NV) * 4;
        const long long g = plane + (long long)row * N + xx;
        pb[b] = *reinterpret_cast<const float4*>(p + g);
        xb[b] = *reinterpret_cast<const float4*>(x + g);
      }
    };
    if (k > 0) load_batch(0);
    if (__syncthreads_or(!mbar_wait(&bar, 0))) {
      if (threadIdx.x == 0) {
        mbar_wait(&bar, 0);  // no copy may still be writing this block's shared memory
        atomicOr(a.fault, 1);
      }
      return;
    }
#pragma unroll
    for (int it0 = 0; it0 < PC::IT; it0 += B) {
      float4 pc[B], xc[B];
#pragma unroll
      for (int b = 0; b < B; ++b) {
        pc[b] = pb[b];
        xc[b] = xb[b];
      }
      if (k > 0 && it0 + B < PC::IT) load_batch(it0 + B);
#pragma unroll
      for (int b = 0; b < B; ++b) {
        const int idx = threadIdx.x + (it0 + b) * TH;
        const int row = idx / NV, xx = (idx - row * NV) * 4;
        const long long g = plane + (long long)row * N + xx;
        float4* rs = reinterpret_cast<float4*>(PR + 2 * RS * row + xx);
        const float4 r4 = *rs;
        float4 v = r4;
        if (k > 0) {
          const float4 p4 = pc[b];
          float4 x4 = xc[b];
          x4.x += alpha * p4.x;
          x4.y += alpha * p4.y;
          x4.z += alpha * p4.z;
          x4.w += alpha * p4.w;
          *reinterpret_cast<float4*>(x + g) = x4;
          v = make_float4(r4.x + beta * p4.x, r4.y + beta * p4.y, r4.z + beta * p4.z, r4.w + beta * p4.w);
          *rs = v;
        }
        *reinterpret_cast<float4*>(p + g) = v;
      }
    }
  }
  __syncthreads();
  plane_x_fwd<N>(PL, tw);
  __syncthreads();
  plane_y_fwd<N>(PL, tw);
  // N rows of the half spectrum to H[s][comp][ky][z][:]; the Nyquist column to NQ
  fence_proxy_async();
  __syncthreads();
  const long long slab = (long long)(s * a.c + comp) * N;
  for (int ky = threadIdx.x; ky < N; ky += TH) {
    bulk_store_1d(a.H + ((slab + ky) * a.nz + z) * a.hs, PL + ky * RS, (uint32_t)(sizeof(float2) * RS));
    a.nq[(long long)blockIdx.x * N + ky] = PL[ky * RS + N / 2];
  }
  bulk_commit();
  bulk_wait_read_all();
}

// MODE 0: out = P (M xin + g).  MODE 4 (CG): q = P (M p + g) and this block's
// part of (p, q) in partials[s * c nz + block of the system].
// MODE 5 (CG, alpha known before this pass): q is not stored, z -= alpha D q is formed
// here (z = D r in `out`, D the preconditioner, 1 without one) and this block's parts of
// (r, r), (r, z), (z, M z), (z, M p) go to partials + {0, 1, 2, 3} off; k_cg_beta sums
// them.  Against MODE 4 and the CG update kernel the q field is neither written nor read
// and r is read where p and the phases already are: 12.5 instead of 14.25 field passes
// per iteration.  MODE 6: the same for two phases that are both in I0 and no voxel field,
// without the general forms of the local term in its epilogue.
template <int N, int MODE>
__global__ void __launch_bounds__(PlaneCfg<N>::TH, PlaneCfg<N>::MINB) k_xyinv(OpArgs<float> a, const float* __restrict__ xin,
                                                           float* __restrict__ out, const SolverState* __restrict__ st,
                                                           double* __restrict__ partials, long long off) {
  typedef PlaneCfg<N> PC;
  constexpr int RS = PC::RS, TH = PC::TH, NV = PC::NV;
  const int cnz = a.c * a.nz;
  const int s = blockIdx.x / cnz;
  const int blk = blockIdx.x - s * cnz;
  const int comp = blk / a.nz, z = blk - comp * a.nz;
  if (MODE >= 5) {
    griddep_wait();
    griddep_launch();
  }
  const volatile SolverState* vst = st + s;  // as in the forward pass
  if (MODE >= 4 && vst->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* PL = reinterpret_cast<float2*>(smem_raw);
  float2* tw = PL + N * RS;
  float* PR = reinterpret_cast<float*>(PL);
  // this component's per-phase values after the plane (sized by the launch): M, D, activity
  float* mloc = reinterpret_cast<float*>(tw + N);
  float* dloc = mloc + a.nphase;
  unsigned char* aloc = reinterpret_cast<unsigned char*>(dloc + a.nphase);
  __shared__ __align__(8) uint64_t bar;
  const long long slab = (long long)(s * a.c + comp) * N;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
    mbar_expect_tx(&bar, (uint32_t)(sizeof(float2) * N * RS));
  }
  __syncthreads();
  for (int ky = threadIdx.x; ky < N; ky += TH)
    bulk_load_1d(PL + ky * RS, a.H + ((slab + ky) * a.nz + z) * a.hs, (uint32_t)(sizeof(float2) * RS), &bar);
  for (int u = threadIdx.x; u < N; u += TH) tw[u] = a.twx[u];
  for (int u = threadIdx.x; u < a.nphase; u += TH) {
    mloc[u] = a.mtab[u * a.c + comp];
    dloc[u] = MODE >= 5 && a.pre == 1 ? a.dtab[u * a.c + comp] : 1.f;
    aloc[u] = a.act[u];
  }
  // the epilogue's p plane and phase plane go to L2 while the transforms run
  const long long plane = (long long)blockIdx.x * N * N;
  const long long pbase = (long long)((a.sys0 + s) / a.sys_per_ms) * a.V + (long long)z * N * N;
  if ((a.l2pf & 2) && threadIdx.x < (MODE >= 5 ? 17 : 9)) {
    constexpr uint32_t PB = (uint32_t)(sizeof(float) * N * N);
    if (threadIdx.x < 8) bulk_prefetch_l2(reinterpret_cast<const char*>(xin + plane) + threadIdx.x * (PB / 8), PB / 8);
    else if (threadIdx.x > 8) bulk_prefetch_l2(reinterpret_cast<const char*>(out + plane) + (threadIdx.x - 9) * (PB / 8), PB / 8);
    else if ((pbase & 15) == 0) bulk_prefetch_l2(a.phase + pbase, (uint32_t)(N * N));
  }
  float2 nqv = make_float2(0.f, 0.f);
  if (threadIdx.x < N) nqv = a.nq[(long long)blockIdx.x * N + threadIdx.x];
  if (__syncthreads_or(!mbar_wait(&bar, 0))) {
    if (threadIdx.x == 0) {
      mbar_wait(&bar, 0);  // no copy may still be writing this block's shared memory
      atomicOr(a.fault, 1);
    }
    return;
  }
  for (int ky = threadIdx.x; ky < N; ky += TH)
    PL[ky * RS + N / 2] = ky == (int)threadIdx.x ? nqv : a.nq[(long long)blockIdx.x * N + ky];
  __syncthreads();
  plane_y_inv<N>(PL, tw);
  // the epilogue's p and phase loads go out in batches of B groups of four
  // voxels, each batch in flight while the previous one is worked on; two
  // register sets take the batches in turn (no copies between them)
  constexpr int B = PC::IT % 2 == 0 && MODE < 5 ? 2 : 1;
  constexpr int ZB = MODE >= 5 ? B : 1;
  float4 xb0[B], xb1[B], zb0[ZB], zb1[ZB];
  uchar4 hb0[B], hb1[B];
  auto load_batch = [&](int it0, float4* xb, uchar4* hb, float4* zb) {
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int idx = threadIdx.x + (it0 + b) * TH;
      const int row = idx / NV, xx = (idx - row * NV) * 4;
      xb[b] = *reinterpret_cast<const float4*>(xin + plane + (long long)row * N + xx);
      hb[b] = *reinterpret_cast<const uchar4*>(a.phase + pbase + (long long)row * N + xx);
      if (MODE >= 5) zb[b] = *reinterpret_cast<const float4*>(out + plane + (long long)row * N + xx);
    }
  };
  plane_x_inv<N>(PL, tw);
  if (MODE == 0 && a.mandel) {
    // Mandel components: M acts as m_d on the deviatoric part and m_h on the spherical
    // part, so a normal component takes (m_h - m_d) / 3 of the trace too
    __syncthreads();
    const long long nv = (long long)a.nz * N * N;  // one component
    const float* x0 = xin + plane - (comp < 3 ? (long long)comp * nv : 0);
    constexpr int MB = PC::IT % 2 == 0 ? 2 : 1;
#pragma unroll 1
    for (int it0 = 0; it0 < PC::IT; it0 += MB) {
      float4 v[MB][3];
      uchar4 hc[MB];
#pragma unroll
      for (int b = 0; b < MB; ++b) {
        const int idx = threadIdx.x + (it0 + b) * TH;
        const int row = idx / NV, xx = (idx - row * NV) * 4;
        const long long o = (long long)row * N + xx;
        hc[b] = *reinterpret_cast<const uchar4*>(a.phase + pbase + o);
        v[b][0] = *reinterpret_cast<const float4*>(x0 + o);
        v[b][1] = v[b][2] = v[b][0];
        if (comp < 3) {
          v[b][1] = *reinterpret_cast<const float4*>(x0 + nv + o);
          v[b][2] = *reinterpret_cast<const float4*>(x0 + 2 * nv + o);
        }
      }
#pragma unroll
      for (int b = 0; b < MB; ++b) {
        const int idx = threadIdx.x + (it0 + b) * TH;
        const int row = idx / NV, xx = (idx - row * NV) * 4;
        const long long o = (long long)row * N + xx, vox = pbase + o;
        const float4 g4 = *reinterpret_cast<const float4*>(PR + 2 * RS * row + xx);
        const float4 q4 = comp == 1 ? v[b][1] : (comp == 2 ? v[b][2] : v[b][0]);
        const float xq[4] = {q4.x, q4.y, q4.z, q4.w}, gv[4] = {g4.x, g4.y, g4.z, g4.w};
        const float tr[4] = {v[b][0].x + v[b][1].x + v[b][2].x, v[b][0].y + v[b][1].y + v[b][2].y,
                             v[b][0].z + v[b][1].z + v[b][2].z, v[b][0].w + v[b][1].w + v[b][2].w};
        const unsigned char ph[4] = {hc[b].x, hc[b].y, hc[b].z, hc[b].w};
        float ov[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int pp = ph[u];
          const float mh = a.mfld ? a.mfld[vox + u] : a.mtab[pp * 6];
          const float md = a.mfld ? a.mfld[a.fstride + vox + u] : a.mtab[pp * 6 + 1];
          const float local = comp < 3 ? fmaf((mh - md) * (1.f / 3.f), tr[u], md * xq[u]) : md * xq[u];
          ov[u] = aloc[pp] ? local + gv[u] : 0.f;
        }
        *reinterpret_cast<float4*>(out + plane + o) = make_float4(ov[0], ov[1], ov[2], ov[3]);
      }
    }
    return;
  }
  load_batch(0, xb0, hb0, zb0);
  __syncthreads();
  Acc<float> acc;
  Acc2 acc2[MODE >= 5 ? 4 : 1];  // (r, r), (r, z), (z, M z), (z, M p)
  const float al = MODE >= 5 ? (float)vst->alpha : 0.f;
  // two phases without a voxel field (the common case): both phases' M and
  // activity in registers, selected per voxel instead of read from the tables;
  // both active (A0 differs from both phases): no projection to apply
  const bool two = MODE == 6 || (a.nphase <= 2 && !a.mfld);
  const float m0 = mloc[0], m1 = a.nphase > 1 ? mloc[1] : m0;
  const float d0 = dloc[0], d1 = a.nphase > 1 ? dloc[1] : d0;
  const float e0 = 1.f / d0, e1 = 1.f / d1;
  const bool act0 = aloc[0] != 0, act1 = a.nphase > 1 ? aloc[1] != 0 : act0;
  const bool both = MODE == 6 || (two && act0 && act1);
  auto work = [&](int it0, const float4* xc, const uchar4* hc, const float4* zc) {
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int idx = threadIdx.x + (it0 + b) * TH;
      const int row = idx / NV, xx = (idx - row * NV) * 4;
      const long long g = plane + (long long)row * N + xx;
      const long long vox = pbase + (long long)row * N + xx;
      const float4 g4 = *reinterpret_cast<const float4*>(PR + 2 * RS * row + xx);
      const float xq[4] = {xc[b].x, xc[b].y, xc[b].z, xc[b].w};
      float4 f4 = make_float4(0.f, 0.f, 0.f, 0.f);  // M of the voxels
      if (MODE != 6 && a.mfld) f4 = *reinterpret_cast<const float4*>(a.mfld + field_class(a, comp) * a.fstride + vox);
      const float field[4] = {f4.x, f4.y, f4.z, f4.w};
      const unsigned char ph[4] = {hc[b].x, hc[b].y, hc[b].z, hc[b].w};
      const float gv[4] = {g4.x, g4.y, g4.z, g4.w};
      float ov[4];
      if constexpr (MODE >= 5) {
        float z[4] = {zc[b].x, zc[b].y, zc[b].z, zc[b].w};
        float r[4], zm[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float m, d, e;
          bool active = true;
          if (two) {
            const bool p1 = ph[u] != 0;
            m = p1 ? m1 : m0;
            d = p1 ? d1 : d0;
            e = p1 ? e1 : e0;
            if (!both) active = p1 ? act1 : act0;
          } else {
            active = aloc[ph[u]] != 0;
            m = mloc[ph[u]];
            d = dloc[ph[u]];
            e = 1.f / d;
            if (a.mfld) {
              m = field[u];
              e = a.pre ? fabsf(m) + a.gpre[comp] : 1.f;
              d = 1.f / e;
            }
          }
          const float q = active ? fmaf(m, xq[u], gv[u]) : 0.f;
          z[u] = fmaf(-al, d * q, z[u]);
          r[u] = z[u] * e;
          zm[u] = z[u] * m;
        }
#pragma unroll
        for (int u = 0; u < 4; u += 2) {
          const float2 r2 = make_float2(r[u], r[u + 1]), zm2 = make_float2(zm[u], zm[u + 1]),
                       z2 = make_float2(z[u], z[u + 1]);
          acc2[0].mac(r2, r2);
          acc2[1].mac(r2, z2);
          acc2[2].mac(zm2, z2);
          acc2[3].mac(zm2, make_float2(xq[u], xq[u + 1]));
        }
        *reinterpret_cast<float4*>(out + g) = make_float4(z[0], z[1], z[2], z[3]);
        continue;
      }
      if (both) {
#pragma unroll
        for (int u = 0; u < 4; ++u) ov[u] = fmaf(ph[u] != 0 ? m1 : m0, xq[u], gv[u]);
      } else if (two) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool p1 = ph[u] != 0;
          ov[u] = (p1 ? act1 : act0) ? fmaf(p1 ? m1 : m0, xq[u], gv[u]) : 0.f;
        }
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int pp = ph[u];
          const bool active = aloc[pp] != 0;
          float m = mloc[pp];
          if (a.mfld) m = field[u];
          ov[u] = active ? m * xq[u] + gv[u] : 0.f;
        }
      }
      // (p, K p): the group's four products summed in FP32, then one compensated add
      if (MODE == 4) acc.add(fmaf(xq[3], ov[3], fmaf(xq[2], ov[2], fmaf(xq[1], ov[1], xq[0] * ov[0]))));
      *reinterpret_cast<float4*>(out + g) = make_float4(ov[0], ov[1], ov[2], ov[3]);
    }
  };
#pragma unroll 1
  for (int it0 = 0; it0 < PC::IT; it0 += 2 * B) {
    if (it0 + B < PC::IT) load_batch(it0 + B, xb1, hb1, zb1);
    work(it0, xb0, hb0, zb0);
    if (it0 + B >= PC::IT) break;
    if (it0 + 2 * B < PC::IT) load_batch(it0 + 2 * B, xb0, hb0, zb0);
    work(it0 + B, xb1, hb1, zb1);
  }
  if constexpr (MODE >= 5) {
    double* part = partials + (long long)s * cnz + blk;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double tot = block_reduce(acc2[k].fold());
      if (threadIdx.x == 0) part[k * off] = tot;
      __syncthreads();
    }
  }
  if (MODE == 4) {
    const double tot = block_reduce(acc);
    if (threadIdx.x == 0) partials[(long long)s * cnz + blk] = tot;
  }
}

// Scalars of a CG iteration whose inverse pass updates z (MODE 5).  One block per
// system; partials summed in block order.
//
// alpha = (r, z) / (p, K p) before the inverse pass: (p, Gamma p) from the z pass's
// tiles, (p, M p) from its recurrence under p = z + beta p_old,
//   (p, M p) = (z, M z) + 2 beta (z, M p_old) + beta^2 (p_old, M p_old),
// whose sums the previous inverse pass (at the start, the start kernel) left in aux.
// Against 64 bits, on the FP32 iterates of 64 x 64 conductivity at contrast 10 to 10^4, this
// (p, K p) is off by 2.5e-9 to 1.7e-8 in the root mean square (the sum of p q in space by
// 2e-9 to 5e-9): less than the 6e-8 of alpha's own rounding to FP32.
__global__ void __launch_bounds__(256) k_cg_alpha(SolverState* __restrict__ st, const double* __restrict__ partials,
                                                  int nb) {
  const int s = blockIdx.x;
  SolverState* sst = st + s;
  griddep_wait();
  griddep_launch();
  if (sst->done) return;
  const double* part = partials + (long long)s * nb;
  double v = 0.0;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) v += __ldcg(part + i);
  const double sum = block_sum(v);
  if (threadIdx.x == 0) {
    const double b = sst->beta;
    const double pmp = sst->iter == 0 ? sst->aux[1] : sst->aux[1] + 2.0 * b * sst->aux[2] + b * b * sst->aux[0];
    const double pq = pmp + sum;
    sst->aux[0] = pmp;
    sst->pq = pq;
    if (!(fabs(pq) > 0.0) || !isfinite(pq) || !isfinite(sst->rr)) {
      sst->status = 5;  // LSH_ERR_BREAKDOWN
      sst->alpha = 0.0;
      sst->done = 1;
    } else {
      sst->alpha = sst->rz / pq;
    }
  }
}

// beta, (r, r), the sums of the next (p, M p), convergence.
__global__ void __launch_bounds__(256) k_cg_beta(SolverState* __restrict__ st, const double* __restrict__ partials,
                                                 long long off, int nb) {
  const int s = blockIdx.x;
  SolverState* sst = st + s;
  griddep_wait();
  griddep_launch();
  if (sst->done) return;
  // two warps per sum, one barrier
  __shared__ double part[8];
  const int w = threadIdx.x >> 5, k = w & 3;
  double t = 0.0;
  for (int i = threadIdx.x & 31 | (w >> 2) << 5; i < nb; i += 64) t += __ldcg(partials + k * off + (long long)s * nb + i);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0) part[w] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    const double v[4] = {part[0] + part[4], part[1] + part[5], part[2] + part[6], part[3] + part[7]};
    sst->beta = v[1] / sst->rz;
    sst->rr = v[0];
    sst->rz = v[1];
    sst->aux[1] = v[2];
    sst->aux[2] = v[3];
    sst->iter += 1;
    if (!isfinite(v[0])) {
      sst->status = 5;
      sst->done = 1;
    } else if (v[0] <= sst->tol2) {
      sst->done = 1;
    }
  }
}

namespace {

// dynamic shared memory of the inverse kernel: the plane, the twiddles and the phase tables
template <int N> size_t plane_inv_smem(const OpArgs<float>& a) {
  return PlaneCfg<N>::SMEM + (((size_t)a.nphase * 9 + 15) & ~(size_t)15);
}

template <int N> void plane_attrs() {
  const int sm = (int)PlaneCfg<N>::SMEM;
  const int smi = (int)(PlaneCfg<N>::SMEM + 256 * 9);  // up to 256 phases
  cudaFuncSetAttribute(k_xyfwd<N, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  cudaFuncSetAttribute(k_xyfwd<N, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  cudaFuncSetAttribute(k_xyinv<N, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, smi);
  cudaFuncSetAttribute(k_xyinv<N, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smi);
  cudaFuncSetAttribute(k_xyinv<N, 5>, cudaFuncAttributeMaxDynamicSharedMemorySize, smi);
  cudaFuncSetAttribute(k_xyinv<N, 6>, cudaFuncAttributeMaxDynamicSharedMemorySize, smi);
}

template <int N> bool plane_fwd_n(const OpArgs<float>& a, int mode, const float* in, float* x, const float* r,
                                  float* p, const SolverState* st, cudaStream_t s) {
  typedef PlaneCfg<N> PC;
  if (a.hs < PC::RS || (a.hs & 1) != 0) return false;
  const unsigned grid = (unsigned)((long long)a.S * a.c * a.nz);
  if (mode == 0) k_xyfwd<N, 0><<<grid, PC::TH, PC::SMEM, s>>>(a, in, x, r, p, st);
  else launch_dep(a.pdl != 0, k_xyfwd<N, 1>, dim3(grid), dim3(PC::TH), PC::SMEM, s, a, in, x, r, p, st);
  return true;
}

template <int N> bool plane_inv_n(const OpArgs<float>& a, int mode, const float* xin, float* out, SolverState* st,
                                  double* partials, long long off, cudaStream_t s) {
  typedef PlaneCfg<N> PC;
  if (a.hs < PC::RS || (a.hs & 1) != 0) return false;
  const unsigned grid = (unsigned)((long long)a.S * a.c * a.nz);
  const size_t smem = plane_inv_smem<N>(a);
  if (mode == 0) {
    k_xyinv<N, 0><<<grid, PC::TH, smem, s>>>(a, xin, out, st, partials, 0);
  } else if (mode == 1) {
    k_xyinv<N, 4><<<grid, PC::TH, smem, s>>>(a, xin, out, st, partials, 0);
    launch_dot_finalize(st, partials, a.c * a.nz, a.S, s);
  } else {
    launch_dep(a.pdl != 0, a.both ? k_xyinv<N, 6> : k_xyinv<N, 5>, dim3(grid), dim3(PC::TH), smem, s, a, xin, out,
               (const SolverState*)st, partials, off);
    launch_dep(a.pdl != 0, k_cg_beta, dim3(a.S), dim3(256), 0, s, st, (const double*)partials, off, a.c * a.nz);
  }
  return true;
}

}  // namespace

bool plane_length(int n) { return n == 16 || n == 32 || n == 48 || n == 64 || n == 96 || n == 128; }

bool launch_xyfwd(const OpArgs<float>& a, int mode, const float* in, float* x, const float* r, float* p,
                  const SolverState* st, cudaStream_t s) {
  if (a.nx != a.ny || mode < 0 || mode > 1) return false;
  switch (a.nx) {
    case 16: return plane_fwd_n<16>(a, mode, in, x, r, p, st, s);
    case 32: return plane_fwd_n<32>(a, mode, in, x, r, p, st, s);
    case 48: return plane_fwd_n<48>(a, mode, in, x, r, p, st, s);
    case 64: return plane_fwd_n<64>(a, mode, in, x, r, p, st, s);
    case 96: return plane_fwd_n<96>(a, mode, in, x, r, p, st, s);
    case 128: return plane_fwd_n<128>(a, mode, in, x, r, p, st, s);
    default: return false;
  }
}

namespace {
bool xyinv_n(const OpArgs<float>& a, int mode, const float* xin, float* out, SolverState* st, double* partials,
             long long off, cudaStream_t s) {
  if (a.nx != a.ny) return false;
  switch (a.nx) {
    case 16: return plane_inv_n<16>(a, mode, xin, out, st, partials, off, s);
    case 32: return plane_inv_n<32>(a, mode, xin, out, st, partials, off, s);
    case 48: return plane_inv_n<48>(a, mode, xin, out, st, partials, off, s);
    case 64: return plane_inv_n<64>(a, mode, xin, out, st, partials, off, s);
    case 96: return plane_inv_n<96>(a, mode, xin, out, st, partials, off, s);
    case 128: return plane_inv_n<128>(a, mode, xin, out, st, partials, off, s);
    default: return false;
  }
}
}  // namespace

bool launch_xyinv(const OpArgs<float>& a, int mode, const float* xin, float* out, SolverState* st, double* partials,
                  cudaStream_t s) {
  return mode >= 0 && mode <= 1 && xyinv_n(a, mode, xin, out, st, partials, 0, s);
}

bool launch_xyinv_update(const OpArgs<float>& a, const float* p, float* z, SolverState* st, double* partials,
                         long long off, cudaStream_t s) {
  return xyinv_n(a, 2, p, z, st, partials, off, s);
}

void launch_cg_beta(SolverState* st, const double* partials, long long off, int nb, int S, bool pdl, cudaStream_t s) {
  launch_dep(pdl, k_cg_beta, dim3(S), dim3(256), 0, s, st, partials, off, nb);
}

void launch_cg_alpha(SolverState* st, const double* partials, int nb, int S, bool pdl, cudaStream_t s) {
  launch_dep(pdl, k_cg_alpha, dim3(S), dim3(256), 0, s, st, partials, nb);
}

void plane_prepare() {
  plane_attrs<16>();
  plane_attrs<32>();
  plane_attrs<48>();
  plane_attrs<64>();
  plane_attrs<96>();
  plane_attrs<128>();
}

}  // namespace lsh
