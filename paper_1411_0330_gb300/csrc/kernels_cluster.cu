// kernels_cluster.cu -- a whole CG solve of one small system in one thread-block
// cluster.
//
// On small grids a CG iteration of separate passes is bound by latency, not by
// bandwidth or arithmetic: five to seven launches, each a chain of dependent
// global loads (state, tables, spectrum, fields), a ticket and a drain.  Here the
// CTAs of one cluster hold a system's direction p, preconditioned residual z and
// half spectrum in their shared memory and iterate to convergence in one launch;
// data crosses CTAs through distributed shared memory.
//
// Decomposition: slices along the slowest axis (z; y of a 2D grid).  CTA r owns ps
// slices of every component, does their x (and in 3D y) transforms by itself, then
// takes the lines along the slowest axis of pp of the (ky, kx) positions: gathers
// them from all CTAs, transforms, applies Gamma^h (Eq. (13)), transforms back and
// writes them where they came from.  Three cluster barriers per iteration: before
// the gather, after the scatter, after the sums of the update.  (p, K p) is known
// at the second one -- (p, Gamma p) from the spectrum by Parseval, (p, M p) from the
// prologue -- so that the update of z follows the inverse transforms directly.
//
// FFTs are the in-place mixed-radix stages of fft.cuh on strided lines.  Plans are
// this kernel's own (lsh_make_plan_lines): with a few lines per CTA, small radices
// keep more lanes busy -- an FP64 instruction holds the SM's FP64 unit for 16 cycles
// however few of its lanes work.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fft.cuh"
#include "gamma_onfly.cuh"
#include "internal.h"

namespace lsh {

namespace cg = cooperative_groups;

namespace {

constexpr int kMaxCluster = 16;
// FP64 butterflies of up to 12 points need more than 128 registers
template <typename T> constexpr int kThreadsOf = sizeof(T) == 8 ? 256 : 512;
constexpr int kGroup = 4;  // items a thread carries over a barrier where rows change layout

template <typename T, bool INV, int R, typename A>
__device__ __forceinline__ void line_stage_r(C2<T>* __restrict__ buf, int nlines, const FastDiv& dl, const A& at,
                                             const Plan1D& pl, int st, const C2<T>* __restrict__ tw) {
  const int m = pl.m[st], total = pl.n / R * nlines, tws = pl.tws[st];
  const FastDiv dm(m, pl.mag_m[st]);
  for (int w = threadIdx.x; w < total; w += blockDim.x) {
    const int b = dl.div(w), line = w - b * nlines;
    const int sp = dm.div(b), j = b - sp * m, e0 = sp * (m * R) + j, te = j * tws;
    C2<T> a[R];
#pragma unroll
    for (int q = 0; q < R; ++q) a[q] = buf[at(line, e0 + q * m)];
    if (INV && te != 0) {
#pragma unroll
      for (int p = 1; p < R; ++p) a[p] = cmulc<T>(a[p], tw[p * te]);
    }
    Dft<T, R, INV>::run(a, tw, pl.n);
    if (!INV && te != 0) {
#pragma unroll
      for (int p = 1; p < R; ++p) a[p] = cmul<T>(a[p], tw[p * te]);
    }
#pragma unroll
    for (int q = 0; q < R; ++q) buf[at(line, e0 + q * m)] = a[q];
  }
}

// Radix 2 in FP64 on two lanes per butterfly, one for the real and one for the imaginary
// parts.  A scheduler's FP64 unit is busy some 64 cycles with any warp instruction; where
// a stage is a warp or two, four times as many instructions per butterfly are on the
// critical path of a radix-4 stage as here per level (32 x 32, two systems: 23.7 -> 20.9 us
// per iteration; 12^3, radices 3, 2, 2 for one 12: 30.5 -> 28.3).
template <bool INV, typename A>
__device__ __forceinline__ void line_stage_pair(double2* __restrict__ buf, int nlines, const FastDiv& dl, const A& at,
                                                const Plan1D& pl, int st, const double2* __restrict__ tw) {
  const int m = pl.m[st], total = pl.n * nlines, tws = pl.tws[st];  // lanes: two per butterfly
  const FastDiv dm(m, pl.mag_m[st]);
  double* f = reinterpret_cast<double*>(buf);
  const int im = threadIdx.x & 1;  // the block is a whole number of warps
  const double sg = im ? 1.0 : -1.0;
  for (int w = threadIdx.x; w < total; w += blockDim.x) {
    const int i = w >> 1, b = dl.div(i), line = i - b * nlines;
    const int sp = dm.div(b), j = b - sp * m, e0 = sp * (2 * m) + j, te = j * tws;
    const int i0 = 2 * at(line, e0), i1 = 2 * at(line, e0 + m);
    const double a = f[i0 + im], c = f[i1 + im];
    double y0, y1;
    if (te == 0) {
      y0 = a + c;
      y1 = a - c;
    } else if (INV) {
      // t = b conj(w): re b.x w.x + b.y w.y, im b.y w.x - b.x w.y
      const double o = f[i1 + (im ^ 1)];
      const double2 wv = tw[te];
      const double t = fma(-sg * o, wv.y, c * wv.x);
      y0 = a + t;
      y1 = a - t;
    } else {
      // (a - b) w: re d.x w.x - d.y w.y, im d.y w.x + d.x w.y
      const double ao = f[i0 + (im ^ 1)], co = f[i1 + (im ^ 1)];
      const double2 wv = tw[te];
      y0 = a + c;
      y1 = fma(sg * (ao - co), wv.y, (a - c) * wv.x);
    }
    // Both lanes of a pair have read before either writes.  The mask is the lanes with an
    // element left, known from the indices: __activemask() would name whichever lanes happen
    // to be together after the branches, and a partner may be missing from those.  One mask
    // per warp, not one per pair, so that the barrier is a single instruction for all.
    const int left = total - (w - (int)(threadIdx.x & 31));
    __syncwarp(left >= 32 ? 0xffffffffu : (1u << left) - 1u);
    f[i0 + im] = y0;
    f[i1 + im] = y1;
  }
}

// In-place transform of nlines lines, element e of a line at buf[at(line, e)]: DIF
// (natural in, digit-reversed out) or DIT.  Ends synchronised.
template <typename T, bool INV, typename A>
__device__ __forceinline__ void line_fft(C2<T>* __restrict__ buf, int nlines, const A& at, const Plan1D& pl,
                                         const C2<T>* __restrict__ tw) {
  const FastDiv dl(nlines);
  for (int k = 0; k < pl.nst; ++k) {
    const int st = INV ? pl.nst - 1 - k : k;
    switch (pl.radix[st]) {
      case 12: line_stage_r<T, INV, 12>(buf, nlines, dl, at, pl, st, tw); break;
      case 10: line_stage_r<T, INV, 10>(buf, nlines, dl, at, pl, st, tw); break;
      case 9: line_stage_r<T, INV, 9>(buf, nlines, dl, at, pl, st, tw); break;
      case 8: line_stage_r<T, INV, 8>(buf, nlines, dl, at, pl, st, tw); break;
      case 7: line_stage_r<T, INV, 7>(buf, nlines, dl, at, pl, st, tw); break;
      case 6: line_stage_r<T, INV, 6>(buf, nlines, dl, at, pl, st, tw); break;
      case 5: line_stage_r<T, INV, 5>(buf, nlines, dl, at, pl, st, tw); break;
      case 4: line_stage_r<T, INV, 4>(buf, nlines, dl, at, pl, st, tw); break;
      case 3: line_stage_r<T, INV, 3>(buf, nlines, dl, at, pl, st, tw); break;
      default:
        if constexpr (sizeof(T) == 8) line_stage_pair<INV>(buf, nlines, dl, at, pl, st, tw);
        else line_stage_r<T, INV, 2>(buf, nlines, dl, at, pl, st, tw);
        break;
    }
    __syncthreads();
  }
}

__device__ __forceinline__ int dif_pos(const Plan1D& p, int k) {
  int pos = 0;
  for (int s = 0; s < p.nst; ++s) {
    pos += (k % p.radix[s]) * p.m[s];
    k /= p.radix[s];
  }
  return pos;
}

// Gamma^h at the frequencies of the CTA's lines, and their share of (p, Gamma p).
template <typename T, int NC>
__device__ __forceinline__ void cluster_gamma(const OpArgs<T>& a, C2<T>* __restrict__ G, int ns, int pp, int np,
                                              int pos0, const FastDiv& dpp, const FastDiv& dxh, bool flat,
                                              const int* yfreq, const int* yrow, const int* sfreq, const int* srow,
                                              Acc<T>& acc) {
  for (int w = threadIdx.x; w < ns * pp; w += blockDim.x) {
    const int sp = dpp.div(w), t = w - sp * pp;
    if (t >= np) continue;
    const int pos = pos0 + t, y = dxh.div(pos), kx = pos - y * a.nxh;
    // 2D: the slowest axis is y; 3D: y and z
    const int ky = flat ? sfreq[sp] : yfreq[y], kz = flat ? 0 : sfreq[sp];
    const long long f = flat ? (long long)srow[sp] * a.ts + kx : ((long long)srow[sp] * a.ny + yrow[y]) * a.ts + kx;
    C2<T> v[NC], u[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) v[i] = u[i] = G[(i * ns + sp) * pp + t];
    if (a.onfly) {
      gamma_trunc_onfly<T, NC>(a, kx, ky, kz, v);
    } else {
      if (a.fdphase) fd_rotate<T, NC>(a, kx, ky, kz, v, (T)-1);
      gamma_table_apply<T, NC>(a.gtab, f, v);
      if (a.fdphase) fd_rotate<T, NC>(a, kx, ky, kz, v, (T)1);
    }
    // columns other than kx = 0 and nx/2 stand for their mirror images too
    const T w2 = (kx == 0 || 2 * kx == a.nx) ? (T)1 : (T)2;
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      acc.mac(w2 * u[i].x, v[i].x);
      acc.mac(w2 * u[i].y, v[i].y);
      G[(i * ns + sp) * pp + t] = v[i];
    }
  }
}

// Sum of two accumulators over the CTA, sent to slot `rank` of every CTA's arrays: one
// barrier, then warp 0 merges the warps' sums and its lanes store to the CTAs.
__device__ __forceinline__ double2 warp_sums(const Acc<double>& a, const Acc<double>& b) {
  double x = a.s, y = b.s;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    x += __shfl_xor_sync(0xffffffffu, x, o);
    y += __shfl_xor_sync(0xffffffffu, y, o);
  }
  return make_double2(x, y);
}
__device__ __forceinline__ double2 warp_sums(const Acc<float>& a, const Acc<float>& b) {
  float s0 = a.s, c0 = a.c, s1 = b.s, c1 = b.c;
  warp_merge_pair(s0, c0);
  warp_merge_pair(s1, c1);
  return make_double2((double)s0 - (double)c0, (double)s1 - (double)c1);
}
template <typename T>
__device__ __forceinline__ void cluster_share(cg::cluster_group& cluster, const Acc<T>& a, const Acc<T>& b,
                                              double2* warps, double2* slots, int rank, int CS) {
  const double2 v = warp_sums(a, b);
  const int lane = threadIdx.x & 31;
  if (lane == 0) warps[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double2 w = lane < (int)(blockDim.x >> 5) ? warps[lane] : make_double2(0.0, 0.0);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {  // at most 16 warps
      w.x += __shfl_xor_sync(0xffffffffu, w.x, o);
      w.y += __shfl_xor_sync(0xffffffffu, w.y, o);
    }
    if (lane < CS) *cluster.map_shared_rank(slots + rank, lane) = w;
  }
}
// Sums of the CTAs' slots, on every lane of the calling warp, in an order that does not
// depend on the CTA.
__device__ __forceinline__ double2 cluster_total(const double2* slots, int CS) {
  const int lane = threadIdx.x & 31;
  double2 w = lane < CS ? slots[lane] : make_double2(0.0, 0.0);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    w.x += __shfl_xor_sync(0xffffffffu, w.x, o);
    w.y += __shfl_xor_sync(0xffffffffu, w.y, o);
  }
  return w;
}

// N consecutive values of a row (aligned where N > 1)
template <typename T, int N> struct alignas(sizeof(T) * N) Pack {
  T v[N];
};

}  // namespace

// One cluster per system.  x: the iterate, updated in place; z: D r on entry.
// st: states begun by k_cg_begin / k_d2f_begin.  prof (or null): ns of the six pass
// kinds summed over system 0's iterations in every prof_every-th chunk of `check`.
template <typename T>
__global__ void __launch_bounds__(kThreadsOf<T>, 1) k_cluster_cg(ClusterCg<T> c) {
  const OpArgs<T>& a = c.a;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), CS = (int)cluster.num_blocks();
  const int s = blockIdx.x / CS;
  SolverState* sst = c.st + s;
  if (sst->done) return;  // uniform over the cluster, before any barrier
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double2 red_pq[kMaxCluster], red_r[kMaxCluster], red_w[2][16];
  __shared__ double sc_rr, sc_rz;
  __shared__ T sc_alpha, sc_beta;
  __shared__ int sc_done, sc_status;
  const int nx = a.nx, nxh = a.nxh, ns = c.ns, ry = c.ry, ps = c.ps, pp = c.pp, hs = c.hs, LP = c.LP;
  const bool flat = c.flat != 0;
  const int nrow = a.c * ps * ry, npair = (nrow + 1) >> 1;
  // shared memory: spectrum rows (pairs of rows, LP apart), gathered lines, twiddles,
  // p, z, tables, phases
  C2<T>* H = reinterpret_cast<C2<T>*>(smem_raw);
  C2<T>* G = H + npair * LP;
  C2<T>* twx = G + a.c * ns * pp;
  C2<T>* twy = twx + nx;
  C2<T>* tws = twy + (flat ? 0 : a.ny);
  T* P = reinterpret_cast<T*>(smem_raw + ((reinterpret_cast<unsigned char*>(tws + ns) - smem_raw + 15) & ~(ptrdiff_t)15));
  T* Z = P + 2 * npair * nx;
  T* mt = Z + 2 * npair * nx;
  T* dt = mt + a.nphase * a.c;
  T* et = dt + a.nphase * a.c;
  int* posx = reinterpret_cast<int*>(et + a.nphase * a.c);
  int* rowg = posx + nx;              // row of the system a local row is (-1: none)
  int* yfreq = rowg + 2 * npair;
  int* yrow = yfreq + (flat ? 0 : a.ny);
  int* sfreq = yrow + (flat ? 0 : a.ny);
  int* srow = sfreq + ns;
  unsigned char* ph = reinterpret_cast<unsigned char*>(srow + ns);  // [ps][ry][nx]
  unsigned char* act = ph + ps * ry * nx;
  const int slice0 = rank * ps, nsl = max(0, min(ps, ns - slice0));
  const int pos0 = rank * pp, np = max(0, min(pp, ry * nxh - pos0));
  const long long pbase = (long long)((a.sys0 + s) / a.sys_per_ms) * a.V;

  // ---- tables
  for (int i = threadIdx.x; i < nx; i += blockDim.x) {
    twx[i] = a.twx[i];
    posx[i] = dif_pos(c.qx, i);
  }
  const int* kofs = flat ? a.kofy : a.kofz;
  const C2<T>* gtws = flat ? a.twy : a.twz;
  for (int i = threadIdx.x; i < ns; i += blockDim.x) {
    tws[i] = gtws[i];
    sfreq[dif_pos(c.qs, i)] = i;
  }
  if (!flat)
    for (int i = threadIdx.x; i < a.ny; i += blockDim.x) {
      twy[i] = a.twy[i];
      yfreq[dif_pos(c.qy, i)] = i;
    }
  for (int i = threadIdx.x; i < a.nphase * a.c; i += blockDim.x) {
    mt[i] = a.mtab[i];
    dt[i] = a.pre == 1 ? a.dtab[i] : (T)1;
    et[i] = a.pre == 1 ? a.etab[i] : (T)1;
  }
  for (int i = threadIdx.x; i < a.nphase; i += blockDim.x) act[i] = a.act[i];
  for (int i = threadIdx.x; i < nsl * ry * nx; i += blockDim.x) ph[i] = a.phase[pbase + (long long)slice0 * ry * nx + i];
  for (int r = threadIdx.x; r < 2 * npair; r += blockDim.x) {
    const int comp = r / (ps * ry), o = r - comp * ps * ry, sl = o / ry;
    rowg[r] = (comp < a.c && sl < nsl) ? (comp * ns + slice0 + sl) * ry + (o - sl * ry) : -1;
  }
  __syncthreads();
  // table rows of the frequencies at this kernel's positions: kof*[row] = frequency
  for (int i = threadIdx.x; i < ns; i += blockDim.x) {
    const int f = kofs[i];
    srow[dif_pos(c.qs, f)] = i;
  }
  if (!flat)
    for (int i = threadIdx.x; i < a.ny; i += blockDim.x) {
      const int f = a.kofy[i];
      yrow[dif_pos(c.qy, f)] = i;
    }
  const long long fbase = (long long)s * a.c * a.V;
  const FastDiv dnx(nx), dxh(nxh), dpp(pp);
  for (int w = threadIdx.x; w < 2 * npair * nx; w += blockDim.x) {
    const int r = dnx.div(w), i = w - r * nx;
    P[w] = (T)0;
    Z[w] = rowg[r] >= 0 ? c.z[fbase + (long long)rowg[r] * nx + i] : (T)0;
  }
  if (threadIdx.x == 0) {
    sc_rr = sst->rr;
    sc_rz = sst->rz;
    sc_alpha = sc_beta = (T)0;
    sc_done = sc_status = 0;
  }
  __syncthreads();
  cluster.sync();  // every CTA's shared memory is live before the first remote access

  const auto row_at = [&](int r) { return (r >> 1) * LP + (r & 1) * hs; };  // row r of the half spectrum
  const auto x_at = [&](int l, int e) { return l * LP + e; };              // packed line of row pair l
  const auto y_at = [&](int l, int e) {
    const int q = dxh.div(l);
    return row_at(q * ry + e) + (l - q * nxh);
  };
  const auto s_at = [&](int l, int e) {
    const int q = dpp.div(l);
    return (q * ns + e) * pp + (l - q * pp);
  };
  // M, D, 1 / D of voxel o of the CTA's slab (component comp)
  const long long vox0 = pbase + (long long)slice0 * ry * nx;
  const int slab = ps * ry;
  const auto local = [&](int comp, int o, T* m, T* d, T* e) -> bool {
    const int p = ph[o];
    if (a.mfld) {
      const long long f = (a.physics != 0 ? (comp > 0) : comp) * a.fstride + vox0 + o;
      *m = a.mfld[f];
      *e = a.pre ? (T)fabs(*m) + a.gpre[comp] : (T)1;
      *d = a.pre ? (sizeof(T) == 8 ? a.dfld[f] : (T)1 / *e) : (T)1;
      return act[p] != 0;
    }
    *m = mt[p * a.c + comp];
    *d = dt[p * a.c + comp];
    *e = et[p * a.c + comp];
    return act[p] != 0;
  };
  const FastDiv dslab(slab), dns(ns), dps(ps);
  const double tol2 = sst->tol2;
  // rows in 16-byte pieces where they are whole (P, Z and the system's x start aligned then)
  const bool wide = nx % (16 / (int)sizeof(T)) == 0;
  // where element w of the gathered lines lives (null: a line beyond the CTA's positions)
  const auto remote = [&](int w) -> C2<T>* {
    const int cs2 = dpp.div(w), t = w - cs2 * pp;
    if (t >= np) return nullptr;
    const int comp = dns.div(cs2), sl = cs2 - comp * ns, own = dps.div(sl);
    const int pos = pos0 + t, y = dxh.div(pos);
    return cluster.map_shared_rank(H, own) + row_at((comp * ps + sl - own * ps) * ry + y) + (pos - y * nxh);
  };
  unsigned long long tm[6] = {0, 0, 0, 0, 0, 0}, t0 = 0;
  const bool timer = c.prof != nullptr && blockIdx.x == 0 && threadIdx.x == 0;
  int timed_iters = 0, iter = 0;
  auto tick = [&](int k, bool on) {
    if (!on) return;
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (k >= 0) tm[k] += t - t0;
    t0 = t;
  };

  for (; iter < c.maxit; ++iter) {
    const bool on = timer && ((c.chunk0 + iter / c.check) % c.prof_every) == 0;
    tick(-1, on);
    timed_iters += (c.prof != nullptr && ((c.chunk0 + iter / c.check) % c.prof_every) == 0) ? 1 : 0;
    const T alpha = sc_alpha, beta = sc_beta;
    Acc<T> accm;
    // ---- x += alpha p_old, p = z + beta p_old, rows packed in pairs
    const auto prologue = [&](auto width) {
      constexpr int N = decltype(width)::value;
      typedef Pack<T, N> V;
      const int nxv = nx / N;
      const FastDiv dxv(nxv);
#pragma unroll 2
      for (int w = threadIdx.x; w < npair * nxv; w += blockDim.x) {
        const int l = dxv.div(w), i = (w - l * nxv) * N;
        V v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = 2 * l + h, g = rowg[r];
          V po = *reinterpret_cast<const V*>(P + r * nx + i);
          v[h] = *reinterpret_cast<const V*>(Z + r * nx + i);
          if (iter > 0 && g >= 0) {
            V* xg = reinterpret_cast<V*>(c.x + fbase + (long long)g * nx + i);
            V xv = *xg;
#pragma unroll
            for (int u = 0; u < N; ++u) xv.v[u] += alpha * po.v[u];
            *xg = xv;
          }
#pragma unroll
          for (int u = 0; u < N; ++u) v[h].v[u] += beta * po.v[u];
          *reinterpret_cast<V*>(P + r * nx + i) = v[h];
          if (g >= 0) {
            const int comp = dslab.div(r), o = (r - comp * slab) * nx + i;
            T m, d, e;
#pragma unroll
            for (int u = 0; u < N; ++u)
              if (local(comp, o + u, &m, &d, &e)) accm.add(m * v[h].v[u] * v[h].v[u]);
          }
        }
#pragma unroll
        for (int u = 0; u < N; ++u) H[l * LP + i + u] = mkc<T>(v[0].v[u], v[1].v[u]);
      }
    };
    if (wide) prologue(std::integral_constant<int, 16 / (int)sizeof(T)>());
    else prologue(std::integral_constant<int, 1>());
    __syncthreads();
    line_fft<T, false>(H, npair, x_at, c.qx, twx);
    // Z = X_a + i X_b into the two Hermitian half rows, in place: a thread reads its
    // frequencies of a group of pairs before any of them is overwritten
    const int group = max(1, kGroup * (int)blockDim.x / nxh);
    for (int l0 = 0; l0 < npair; l0 += group) {
      const int n = min(group, npair - l0) * nxh;
      C2<T> xa[kGroup], xb[kGroup];
#pragma unroll
      for (int u = 0; u < kGroup; ++u) {
        const int w = threadIdx.x + u * blockDim.x;
        if (w < n) {
          const int l = dxh.div(w), kx = w - l * nxh;
          const C2<T>* line = H + (l0 + l) * LP;
          const C2<T> z1 = line[posx[kx]], z2 = line[posx[kx == 0 ? 0 : nx - kx]];
          xa[u] = mkc<T>((T)0.5 * (z1.x + z2.x), (T)0.5 * (z1.y - z2.y));
          xb[u] = mkc<T>((T)0.5 * (z1.y + z2.y), (T)0.5 * (z2.x - z1.x));
        }
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kGroup; ++u) {
        const int w = threadIdx.x + u * blockDim.x;
        if (w < n) {
          const int l = dxh.div(w), kx = w - l * nxh;
          H[(l0 + l) * LP + kx] = xa[u];
          H[(l0 + l) * LP + hs + kx] = xb[u];
        }
      }
    }
    __syncthreads();
    tick(0, on);
    if (!flat) line_fft<T, false>(H, a.c * ps * nxh, y_at, c.qy, twy);
    tick(1, on);
    cluster.sync();
    // ---- lines along the slowest axis
    const int ngath = a.c * ns * pp;
    for (int w0 = threadIdx.x; w0 < ngath; w0 += kGroup * blockDim.x) {
      C2<T> v[kGroup];
#pragma unroll
      for (int u = 0; u < kGroup; ++u) {
        const int w = w0 + u * blockDim.x;
        const C2<T>* p = w < ngath ? remote(w) : nullptr;
        if (p) v[u] = *p;
      }
#pragma unroll
      for (int u = 0; u < kGroup; ++u)
        if (w0 + u * (int)blockDim.x < ngath) G[w0 + u * blockDim.x] = v[u];
    }
    __syncthreads();
    if (np > 0) line_fft<T, false>(G, a.c * pp, s_at, c.qs, tws);
    Acc<T> accg;
    if (np > 0) {
      if (a.c == 6) cluster_gamma<T, 6>(a, G, ns, pp, np, pos0, dpp, dxh, flat, yfreq, yrow, sfreq, srow, accg);
      else if (a.c == 3) cluster_gamma<T, 3>(a, G, ns, pp, np, pos0, dpp, dxh, flat, yfreq, yrow, sfreq, srow, accg);
      else cluster_gamma<T, 2>(a, G, ns, pp, np, pos0, dpp, dxh, flat, yfreq, yrow, sfreq, srow, accg);
    }
    __syncthreads();
    if (np > 0) line_fft<T, true>(G, a.c * pp, s_at, c.qs, tws);
    for (int w = threadIdx.x; w < ngath; w += blockDim.x) {
      C2<T>* p = remote(w);
      if (p) *p = G[w];
    }
    cluster_share(cluster, accg, accm, red_w[0], red_pq, rank, CS);
    cluster.sync();
    if (threadIdx.x >= blockDim.x - 32) {  // a warp the next stage hardly needs
      const double2 w = cluster_total(red_pq, CS);
      const double pq = w.x + w.y;
      if (threadIdx.x == blockDim.x - 1) {
        if (!(fabs(pq) > 0.0) || !isfinite(pq) || !isfinite(sc_rr)) {
          sc_status = 5;  // LSH_ERR_BREAKDOWN
          sc_alpha = (T)0;
        } else {
          sc_alpha = (T)(sc_rz / pq);
        }
      }
    }
    tick(2, on);
    // ---- inverse transforms
    if (!flat) line_fft<T, true>(H, a.c * ps * nxh, y_at, c.qy, twy);
    tick(3, on);
    for (int l0 = 0; l0 < npair; l0 += group) {
      const int n = min(group, npair - l0) * nxh;
      C2<T> xa[kGroup], xb[kGroup];
#pragma unroll
      for (int u = 0; u < kGroup; ++u) {
        const int w = threadIdx.x + u * blockDim.x;
        if (w < n) {
          const int l = dxh.div(w), kx = w - l * nxh;
          xa[u] = H[(l0 + l) * LP + kx];
          xb[u] = H[(l0 + l) * LP + hs + kx];
        }
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kGroup; ++u) {
        const int w = threadIdx.x + u * blockDim.x;
        if (w < n) {
          const int l = dxh.div(w), kx = w - l * nxh;
          C2<T>* line = H + (l0 + l) * LP;
          line[posx[kx]] = mkc<T>(xa[u].x - xb[u].y, xa[u].y + xb[u].x);
          if (kx >= 1 && kx <= nx - nxh) line[posx[nx - kx]] = mkc<T>(xa[u].x + xb[u].y, xb[u].x - xa[u].y);
        }
      }
    }
    __syncthreads();
    if (sc_status) break;  // uniform over the cluster: every CTA summed the same values
    line_fft<T, true>(H, npair, x_at, c.qx, twx);
    // ---- q = M p + g, z -= alpha D q, (r, r), (r, z)
    const T al = sc_alpha;
    Acc<T> accr, accz;
    for (int w = threadIdx.x; w < npair * nx; w += blockDim.x) {
      const int l = dnx.div(w), i = w - l * nx;
      const C2<T> g2 = H[l * LP + i];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = 2 * l + h;
        if (rowg[r] < 0) continue;
        const int comp = dslab.div(r);
        T m, d, e;
        if (!local(comp, (r - comp * slab) * nx + i, &m, &d, &e)) continue;  // off I0: q = 0
        const T q = m * P[r * nx + i] + (h ? g2.y : g2.x);
        T& zr = Z[r * nx + i];
        const T zn = zr - al * (d * q);
        zr = zn;
        const T rr = zn * e;
        accr.add(rr * rr);
        accz.add(rr * zn);
      }
    }
    tick(4, on);
    cluster_share(cluster, accr, accz, red_w[1], red_r, rank, CS);
    cluster.sync();
    if (threadIdx.x < 32) {
      const double2 w = cluster_total(red_r, CS);
      if (threadIdx.x == 0) {
        sc_beta = (T)(w.y / sc_rz);
        sc_rr = w.x;
        sc_rz = w.y;
        if (!isfinite(w.x)) {
          sc_status = 5;
          sc_done = 1;
        } else if (w.x <= tol2) {
          sc_done = 1;
        }
      }
    }
    __syncthreads();
    tick(5, on);
    if (sc_done) {
      ++iter;
      break;
    }
  }
  // the last step's share of x (none after a breakdown)
  __syncthreads();
  const T alpha = sc_alpha;
  if (iter > 0 && alpha != (T)0)
    for (int w = threadIdx.x; w < 2 * npair * nx; w += blockDim.x) {
      const int r = dnx.div(w), i = w - r * nx;
      if (rowg[r] >= 0) c.x[fbase + (long long)rowg[r] * nx + i] += alpha * P[w];
    }
  if (rank == 0 && threadIdx.x == 0) {
    sst->iter = iter;
    sst->rr = sc_rr;
    sst->rz = sc_rz;
    sst->alpha = 0.0;  // x is complete
    sst->status = sc_status;
    sst->done = (sc_done || sc_status) ? 1 : 0;
    sst->pad = timed_iters;
  }
  if (timer)
    for (int k = 0; k < 6; ++k) c.prof[k] = tm[k];
}

// ------------------------------------------------------------------ host side
namespace {

template <typename T> size_t cluster_smem(const OpArgs<T>& a, const ClusterCg<T>& c) {
  const int npair = (a.c * c.ps * c.ry + 1) / 2;
  size_t b = sizeof(C2<T>) * ((size_t)npair * c.LP + (size_t)a.c * c.ns * c.pp + a.nx + c.ns + (c.flat ? 0 : a.ny));
  b = (b + 15) & ~(size_t)15;
  b += sizeof(T) * (4 * (size_t)npair * a.nx + 3 * (size_t)a.nphase * a.c);
  b += sizeof(int) * ((size_t)a.nx + 2 * npair + 2 * c.ns + (c.flat ? 0 : 2 * a.ny));
  b += (size_t)c.ps * c.ry * a.nx + a.nphase;
  return (b + 15) & ~(size_t)15;
}

template <typename T> void cluster_launch_config(const ClusterCg<T>& c, int S, cudaLaunchConfig_t* cfg,
                                                 cudaLaunchAttribute* at, cudaStream_t s) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3((unsigned)(S * c.CS));
  cfg->blockDim = dim3((unsigned)c.threads);
  cfg->dynamicSmemBytes = c.smem;
  cfg->stream = s;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = (unsigned)c.CS;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = 1;
}

}  // namespace

// Whether the cluster solver takes this problem (nsys systems in the handle), and how.
// The cluster size depends on the grid, the type and the handle's systems only, not on
// the wave, so that waves of any size give the same sums.
template <typename T> bool cluster_plan(const OpArgs<T>& a, int nsys, ClusterCg<T>* out) {
  ClusterCg<T> c{};
  c.flat = a.nz == 1 ? 1 : 0;
  c.ns = c.flat ? a.ny : a.nz;
  c.ry = c.flat ? 1 : a.ny;
  const long long n = (long long)a.c * a.V;
  if (n > (1 << 20) || a.nx > 1024 || c.ns > 2048 || c.ry > 2048) return false;
  const int npos = c.ry * a.nxh;
  c.hs = a.nxh;
  c.LP = (2 * c.hs) | 1;  // odd: lanes over row pairs fall on distinct banks
  static bool attrs = []() {
    return cudaFuncSetAttribute(k_cluster_cg<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024) == cudaSuccess &&
           cudaFuncSetAttribute(k_cluster_cg<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  }();
  if (!attrs) {
    cudaGetLastError();
    return false;
  }
  for (int CS = kMaxCluster; CS >= 1; CS /= 2) {
    if (CS > c.ns || (long long)nsys * CS > 152) continue;
    c.CS = CS;
    c.ps = (c.ns + CS - 1) / CS;
    c.pp = (npos + CS - 1) / CS;
    const int npair = (a.c * c.ps * c.ry + 1) / 2;
    c.threads = std::min(kThreadsOf<T>, std::max(sizeof(T) == 8 ? 128 : 64, (npair * a.nx / 2 + 31) / 32 * 32));
    c.smem = cluster_smem(a, c);
    if (c.smem > 223 * 1024) return false;  // smaller clusters need more still
    // elements a CTA carries through an iteration: beyond these the separate passes,
    // which use the whole chip, are as fast.  us per iteration, cluster / separate: FP64
    // 32^2 conductivity 21 / 42, 16^3 28 / 69, 16^3 elasticity (1536 a CTA) 40 / 66; FP32
    // 24^3 elasticity 39 / 58; on grids with the plane passes 32^3 conductivity (6144) 34
    // / 36, 32^3 elasticity (12288) 51 / 49; off them 20^3 elasticity, four
    // microstructures (12000) 68 / 93.
    if (n / CS > (sizeof(T) == 8 ? 1536 : (a.plane ? 6144 : 12288))) return false;
    if (!lsh_make_plan_lines(a.nx, npair, c.threads, sizeof(T) == 8, &c.qx) ||
        !lsh_make_plan_lines(c.ns, a.c * c.pp, c.threads, sizeof(T) == 8, &c.qs) ||
        !lsh_make_plan_lines(a.ny, a.c * c.ps * a.nxh, c.threads, sizeof(T) == 8, &c.qy))
      return false;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    cluster_launch_config(c, nsys, &cfg, &at, nullptr);
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k_cluster_cg<T>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      clusters = 0;
    }
    if (clusters < nsys) continue;  // all systems at once
    *out = c;
    return true;
  }
  return false;
}

template <typename T> bool launch_cluster_cg(const ClusterCg<T>& c, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  cluster_launch_config(c, c.a.S, &cfg, &at, s);
  return cudaLaunchKernelEx(&cfg, k_cluster_cg<T>, c) == cudaSuccess;
}

template bool cluster_plan<double>(const OpArgs<double>&, int, ClusterCg<double>*);
template bool cluster_plan<float>(const OpArgs<float>&, int, ClusterCg<float>*);
template bool launch_cluster_cg<double>(const ClusterCg<double>&, cudaStream_t);
template bool launch_cluster_cg<float>(const ClusterCg<float>&, cudaStream_t);

}  // namespace lsh
