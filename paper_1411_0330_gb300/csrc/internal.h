// internal.h -- host-side declarations shared by the liblsh translation units.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"

namespace lsh {

// Launch with or without programmatic dependence on the kernel ahead in the stream.
template <typename... P, typename... A>
inline void launch_dep(bool pdl, void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, args...);
}

// Everything an operator pass needs, passed by value to the kernels.
//
// A launch covers S independent systems (one microstructure, one load each)
// that share the grid, the reference medium, the twiddles and the Gamma^h
// table.  Fields are stored system-major: [S][c][nz][ny][nx] (real) and
// [S][c][nz][ny][nxh] (half spectrum), so the rows of all systems are one
// contiguous range; each x-pass block works inside one system (RY divides the
// rows of a system) which keeps the per-system reductions block-aligned.
template <typename T> struct OpArgs {
  int nx, ny, nz, nxh, c;
  int hs;            // row stride of the half spectrum H (nxh rounded up to 4: 32-byte FP32 rows)
  int ts;            // row stride of the Gamma table (nxh rounded up to 8: 32-byte FP32 rows)
  long long V;       // voxels per system
  int S;             // systems in this launch
  int sys0;          // global index of system 0 of this launch
  int sys_per_ms;    // systems per microstructure (phase map index = (sys0 + s) / sys_per_ms)
  int rps;           // rows per system: c * nz * ny
  int bps;           // x-pass blocks per system: rps / RY
  int RY;            // rows per block in the x passes
  int TY, TZ;        // kx columns per block in the y / z passes
  int lsx, lsy, lsz; // shared-memory line strides (complex elements)
  Plan1D px, py, pz;
  const C2<T>* twx;
  const C2<T>* twy;
  const C2<T>* twz;
  const int* posx;   // frequency kx -> position after the x DIF
  C2<T>* H;          // half spectrum [S][c][nz][ny][hs] (kx < nxh used; y, z positions per kofy / kofz)
  const T* gtab;     // Gamma^h (internal basis, scaled by 1/V): blocks of 8 frequencies, see gamma_elem
  int ncoef;
  // local term M_beta = (A_beta - A0)^{-1}, diagonal in the internal basis
  const unsigned char* phase;  // [nbatch][V]
  const float* scale;          // [nbatch][V] or null
  int frac;                    // 1: scale holds the volume fraction of phase 1 (Eq. (def_ah))
  const unsigned char* act;    // per phase: 1 if A_phase != A0 (voxel in I0)
  int nphase;
  int both;                    // two phases, both in I0, no voxel field (the common case)
  const T* mtab;               // per phase * c: diagonal of M (no scale field)
  const T* modtab;             // per phase * c: diagonal of A_phase (scale field)
  T ref[6];                    // diagonal of A0 (internal basis)
  // diagonal preconditioner of the CG iterations, D = 1 / (|M_beta| + gpre).  pre: 0 none,
  // 1 per phase, 2 per voxel (scale or fraction field).  The residual buffer then
  // holds z = D r, so that p = z + beta p needs no phase map.
  int pre;
  const T* dtab;               // per phase * c: D (1 outside I0)
  const T* etab;               // per phase * c: 1 / D
  // per-voxel local operator of handles with a scale or fraction field, formed once when
  // the field is set (a division per voxel instead of one per voxel, component, system
  // and pass): M, and D in FP64; [class][nbatch * V], class 0 / 1 the spherical /
  // deviatoric components of elasticity, else the component.  Null (no such field, or a call
  // without a handle): formed where used.
  const T* mfld;
  const T* dfld;
  long long fstride;           // nbatch * V
  T gpre[6];                   // g per component: 0 or what stands for the Green operator's diagonal
  const T* loads;              // [S][6] macroscopic load per system (internal basis)
  // Green operator computed in the z pass instead of read from gtab (truncated
  // operator, FP32): physics, grid lengths, signed-frequency tables, constants
  int onfly;                   // 1: compute Gamma^h_k on the fly
  int fdphase;                 // finite-difference operator: the table holds the real part
                               // u u^T / (u^T A0 u); components rotate by -/+ pi k_i / N_i around it
  const C2<T>* fdw;            // its factors (cos, sin)(pi k / N), x then y then z (null: computed)
  int physics;
  const int* kofy;             // y position -> frequency
  const int* kofz;             // z position -> frequency
  T g0[6];                     // elastic: 1/(2 mu0 V), cb/V, 1/(3 K0 V), 1/(2 mu0 V); scalar: A0 diagonal
  T invV;
  // register-FFT passes (natural-order y / z frequencies) for lengths 16..256
  int yreg, zreg;
  // FP32 y and z passes through the Tensor Memory Accelerator (host pointers
  // to the maps)
  int ytma;           // 1: TMA y pass
  int ztma;           // 0: register z pass; 1..5: the variant of launch_zgamma_tma; 6: register, 4 columns;
                      // 7: persistent register z pass with staged prefetch; 8: register, 16 columns;
                      // 9: register, coefficients loaded when used; 10: pipelined TMA tiles on the
                      // ky-major spectrum (kernels_zpipe.cu); 11: the same on the plan N = R1 x 4
                      // with the 4-point DFTs and Gamma^h fused
  const CUtensorMap* tmy;
  const CUtensorMap* tmz;   // z boxes of 4 columns
  const CUtensorMap* tmz8;  // z boxes of 8 columns
  const CUtensorMap* tmz16; // z boxes of 16 columns
  const CUtensorMap* tmzp;  // ky-major spectrum, boxes of 8 columns (variant 10)
  const CUtensorMap* tmzq;  // Nyquist columns of the ky-major spectrum, boxes of 8 ky
  int* fault;  // set by a kernel whose bounded wait ran out
  int xreg;    // FP32 inverse x pass: 0 shared-memory stages, 1 register FFT, 2 register FFT persistent,
               // 3 register FFT in blocks of 128 threads
  int xfreg;   // 1: FP32 forward x pass on the register FFT (kernels_x.cu)
  // FP32 plane passes (kernels_plane.cu): x and y transforms of a z plane in one
  // kernel; the spectrum is then ky-major, H[S][c][ky][z][hs] (tlay = 1), and the
  // Nyquist column kx = nx/2 also lives in nq[S][c][z][ky]
  int plane;
  int tlay;
  C2<T>* nq;
  int mandel;  // apply on the plane passes: fields are Mandel components, the z pass takes
               // the internal basis around Gamma^h and the local term couples the normals
  double* dot; // FP32 z passes: each block's share of (p, Gamma p), zdot_blocks() of them per
               // system (null: not wanted)
  int pdl;     // the kernels of the fused plane iteration start before the one ahead has drained
  int fuse;  // the CG update runs in the inverse pass: plane passes with z variant 11; separate
             // passes with inverse x variants 0, 1 and 3 and z variants 0 and 9
  int l2pf;  // plane passes, input planes requested into L2 at a block's start: bit 0 the
             // forward pass's x, r, p; bit 1 the inverse pass's p and phase planes
};

// Row of the voxel fields for component comp: one per component, or the bulk and the
// shear part of isotropic elasticity.
template <typename T> __host__ __device__ __forceinline__ int field_class(const OpArgs<T>& a, int comp) {
  return a.physics != 0 ? (comp > 0) : comp;
}

// Thread-block sizes and tile shapes, chosen at setup for one system count.
struct LaunchCfg {
  int thr_x, thr_y, thr_z;  // threads per block of the shared-memory x, y and z passes
  int RY, TY, TZ, VEC;
  size_t smem_x, smem_y, smem_z;
  int grid_x, grid_yx, grid_yy, grid_zx, grid_zy, grid_zz;
  int ew_per_sys;  // blocks per system of the elementwise kernels
};

// Threads per block of a shared-memory pass over nlines lines of plan p, `blocks` of them
// in the launch: the largest number of blocks in flight per SM over the time of one,
// where a stage of radix R takes ceil(butterflies / threads) rounds of R values.  Larger
// radices leave few butterflies per block, and 256 threads for 56 of them hold the
// registers of 200 idle ones: at 90 x 100 x 84, six systems, the y pass went from 89 to
// 65 us in FP32 and from 755 to 707 us in FP64 with blocks of 64, at 63 x 45 x 50 the FP64
// z pass from 81 to 61 us with tiles of 2 columns in blocks of 96.
inline int pass_threads(int nlines, const Plan1D& p, size_t smem, int max_resident, long long blocks) {
  int best = 256;
  double best_rate = 0.0;
  const long long share = (blocks + 151) / 152;  // blocks an SM gets
  for (int t = 256; t >= 64; t -= 32) {
    const long long fit = std::min<long long>(
        {32LL, (long long)(max_resident / t), (long long)(226 * 1024 / (smem + 1024)), share});
    if (fit < 1) continue;
    const long long pts = (long long)nlines * p.n;
    double time = 8.0 + 2.0 * 4.0 * (double)((pts / 4 + t) / t);  // barriers; loads and stores, four in flight
    for (int s = 0; s < p.nst; ++s) time += (double)p.radix[s] * (double)((pts / p.radix[s] + t - 1) / t);
    const double rate = (double)fit / time;
    if (rate > best_rate * 1.02) {
      best_rate = rate;
      best = t;
    }
  }
  return best;
}

// Tiles and block sizes of the shared-memory passes for S systems: blocks of about 32 KB,
// fewer lines where that would leave the 152 SMs without some four blocks each (two for
// the x passes, whose tables and barriers cost more than the idle SMs).
template <typename T>
LaunchCfg pass_cfg(int nx, int ny, int nz, int c, const Plan1D& px, const Plan1D& py, const Plan1D& pz, int S) {
  LaunchCfg L{};
  const size_t cs = sizeof(C2<T>);
  const int nxh = nx / 2 + 1, lsx = nx | 1, lsy = ny | 1, lsz = nz | 1;
  const int rps = c * nz * ny;
  const int resident = sizeof(T) == 8 ? 512 : 768;  // threads per SM at the passes' register counts
  constexpr long long kBlocks = 608;                // four per SM
  // rows per x block: an even divisor of the rows of a system where there is one
  const int cap = std::max(2, 2 * (int)(32768 / (lsx * cs)));
  const bool fixed = nx == 16 || nx == 32 || nx == 48 || nx == 64 || nx == 96 || nx == 128 || nx == 256;
  L.RY = 0;
  if (sizeof(T) == 8 && fixed && cap < rps) {
    // FP64 at the lengths with a compile-time schedule, blocks of 256 threads, two to an SM:
    // the divisor of the least time, a wave of blocks costing its chain of barriers (the
    // time of some 1280 elements) and an SM the elements of its blocks; among equals the
    // larger.  us per iteration with RY = 8 (384 blocks, two waves) / 12 (256, one): 32^3
    // conductivity, one load, 68 / 55; 16 x 64 x 64 75 / 61; 32^3 elasticity, six loads, 96
    // (384) / 64 (576) 180 / 173; 96^3 conductivity 36 (768) / 32 (864) 502 / 474.
    long long best = 0;
    for (int d = cap & ~1; d >= 2; d -= 2) {
      if (rps % d != 0) continue;
      const long long blocks = (long long)S * (rps / d);
      const long long t = (blocks + 303) / 304 * 1280 + (blocks + 151) / 152 * d * nx;
      if (!L.RY || t < best) {
        best = t;
        L.RY = d;
      }
    }
  }
  if (!L.RY) {
    const int target = std::min(cap, std::max(2, (int)((long long)rps * S / (kBlocks / 2))));
    if (target >= rps) {
      L.RY = rps;
    } else {
      int odd = 1;
      for (int d = target; d >= 1 && !L.RY; --d)
        if (rps % d == 0) {
          if (d % 2 == 0) L.RY = d;
          else if (odd == 1) odd = d;
        }
      if (!L.RY) L.RY = odd;
    }
  }
  constexpr int VV = 16 / (int)sizeof(T);
  L.VEC = nx % VV == 0 ? VV : (nx % 2 == 0 ? 2 : 1);
  const int npair = (L.RY + 1) / 2;
  L.smem_x = nx * cs + (size_t)npair * lsx * cs + nx * sizeof(int);
  // the FP32 x passes stream three fields in and two out: the loads want every thread; the
  // lengths with a compile-time schedule are bound by the FP64 pipe at any block size
  L.thr_x = sizeof(T) == 4 || fixed ? 256 : pass_threads(npair, px, L.smem_x, resident, (long long)S * (rps / L.RY));
  // y columns per block: up to 16 (8 in FP64), evenly shared among a plane's blocks
  int TY = std::min(sizeof(T) == 8 ? 8 : 16, nxh);
  while (TY > 2 && (long long)S * c * nz * ((nxh + TY - 1) / TY) < kBlocks) TY /= 2;
  const int nty = (nxh + TY - 1) / TY;
  L.TY = (nxh + nty - 1) / nty;
  L.smem_y = ny * cs + (size_t)L.TY * lsy * cs;
  L.thr_y = pass_threads(L.TY, py, L.smem_y, resident, (long long)S * c * nz * nty);
  // z columns per block (32-byte segments at least)
  int TZ = std::min(8, nxh);
  while (TZ > 1 && (size_t)c * TZ * lsz * cs > 100 * 1024) TZ /= 2;
  while (TZ > 32 / (int)cs && (long long)S * ny * ((nxh + TZ - 1) / TZ) < kBlocks) TZ /= 2;
  L.TZ = TZ;
  L.smem_z = nz * cs + (size_t)c * TZ * lsz * cs;
  L.thr_z = pass_threads(c * TZ, pz, L.smem_z, resident, (long long)S * ny * ((nxh + TZ - 1) / TZ));
  L.grid_x = rps / L.RY;  // per system
  L.grid_yx = nty;
  L.grid_yy = c * nz;  // per system
  L.grid_zx = (nxh + TZ - 1) / TZ;
  L.grid_zy = ny;
  const long long n = (long long)rps * nx, want = (n + 2047) / 2048;
  L.ew_per_sys = (int)std::max(1LL, std::min(want, std::max(1LL, 2432LL / S)));
  return L;
}

// A CG solve of every system of a wave in one cluster each (kernels_cluster.cu).
template <typename T> struct ClusterCg {
  OpArgs<T> a;
  Plan1D qx, qy, qs;  // the kernel's own plans: x, y (3D), slowest axis
  int flat;           // 2D grid: y is the slowest axis
  int ns, ry;         // slices along the slowest axis, rows per slice
  int CS, ps, pp;     // cluster size, slices and (row, kx) positions per CTA
  int hs, LP;         // half rows and row pairs in shared memory (complex elements)
  int threads;
  size_t smem;
  T* x;
  const T* z;
  SolverState* st;
  int maxit;
  // per-pass device time of system 0's iterations in every prof_every-th chunk of `check`
  unsigned long long* prof;
  int check, prof_every;
  long long chunk0;
};
template <typename T> bool cluster_plan(const OpArgs<T>& a, int nsys, ClusterCg<T>* out);
template <typename T> bool launch_cluster_cg(const ClusterCg<T>& c, cudaStream_t s);

template <typename T>
void launch_xfwd(const OpArgs<T>& a, const LaunchCfg& L, int mode, const T* in, T* x, const T* r, T* p,
                 const SolverState* st, cudaStream_t s);
template <typename T>
void launch_yfft(const OpArgs<T>& a, const LaunchCfg& L, bool inv, const SolverState* st, cudaStream_t s);
template <typename T>
void launch_zgamma(const OpArgs<T>& a, const LaunchCfg& L, const SolverState* st, cudaStream_t s);
template <typename T>
void launch_xinv(const OpArgs<T>& a, const LaunchCfg& L, int mode, const T* xin, T* out, SolverState* st,
                 double* partials, cudaStream_t s);
template <typename T>
void launch_cg_update(const OpArgs<T>& a, T* r, const T* q, SolverState* st, double* partials, long long off2, int G,
                      cudaStream_t s);
template <typename T>
void launch_cg_finalize(T* x, const T* p, long long n, int S, const SolverState* st, int G, cudaStream_t s);
template <typename T>
void launch_cg_begin(const OpArgs<T>& a, T* r, SolverState* st, double* partials, long long off2, double tol,
                     const double* bb_given, int G, cudaStream_t s);
template <typename T>
void launch_fill_rhs(const OpArgs<T>& a, T* r, T* x, int G, cudaStream_t s);
template <typename T>
void launch_rotate(const T* in, T* out, long long V, int nsys, int to_internal, cudaStream_t s);
template <typename T>
void launch_comp_sums(const T* x, int c, long long V, int S, double* partials, int nblk, double* out, cudaStream_t s);
template <typename T>
void launch_gamma_table(const OpArgs<T>& a, int dim, int physics, int green, const double* ref_mandel,
                        const int* kofy, const int* kofz, cudaStream_t s, const double* a0full = nullptr,
                        const double* rot = nullptr);
template <typename T>
void launch_rotate_scalar(const T* in, T* out, long long V, int nsys, int d, const double* R, int to_internal,
                          cudaStream_t s);
template <typename T>
void launch_voxel_fields(const OpArgs<T>& a, T* mfld, T* dfld, unsigned* range, int B, cudaStream_t s);
void launch_gamma_diag(const OpArgs<double>& a, double* partials, int nblk, double* out, cudaStream_t s);
void launch_d2f_begin(const OpArgs<float>& a, const double* r64, int src, float* r32, float* x32, SolverState* st,
                      double* partials, long long off2, double tol, const unsigned char* active, int G,
                      cudaStream_t s);
void launch_f2d_axpy(double* x64, const float* x32, const float* p, long long n, int S, const SolverState* st,
                     bool first, int G, cudaStream_t s);
void launch_scan_phase(const unsigned char* phase, long long V, int B, const unsigned char* act, int nphase,
                       SolverState* st, double* partials, int G, cudaStream_t s);
void launch_scale_grad(const double* tau_all, const double* W, const unsigned char* phase, const float* scale,
                       const double* modtab, const double* ref, int c, int elastic, long long V, int B,
                       double* grad, cudaStream_t s);

// FP32 CG iteration of the separate passes with the update of z in the inverse x pass.
// Blocks per system of the z pass, each of which leaves its share of (p, Gamma p): register
// kernel in tiles of 8 columns (z variants 0 and 9), pointwise kernel of a scalar 2D grid,
// else the shared-memory tiles, grids of one z layer with six components among them.  The
// workspace holds as many partials for every system, at the tiles of a single one (the
// most): the layout asks the same function.
inline long long zdot_blocks(bool zreg, int nxh, int ny, int nz, int c, const LaunchCfg& L) {
  if (zreg) {
    const int TZ = 8, nrt = nxh / TZ;
    return (long long)ny * nrt + ((long long)ny * (nxh - nrt * TZ) + TZ - 1) / TZ;
  }
  if (nz == 1 && c != 6) return ((nxh + 31) / 32) * (long long)((ny + 7) / 8);
  return (long long)L.grid_zx * L.grid_zy;
}
void launch_xinv_update(const OpArgs<float>& a, const LaunchCfg& L, const float* p, float* z, SolverState* st,
                        double* partials, long long off, cudaStream_t s);
void launch_cg_beta(SolverState* st, const double* partials, long long off, int nb, int S, bool pdl, cudaStream_t s);
void launch_dot_finalize(SolverState* st, const double* partials, int nb, int S, cudaStream_t s);
void launch_basic_update(const OpArgs<double>& a, double* x, const double* r, const unsigned char* flags, int G,
                         cudaStream_t s);
void launch_minres_begin(SolverState* st, MinresScalars* ms, const double* rhs2, const double* bb, double tol, int S,
                         cudaStream_t s);
void launch_minres_step(double* x, double* r1, double* r2, double* q, double* wa, double* wb, long long n, int S,
                        SolverState* st, MinresScalars* ms, double* partials, int G, cudaStream_t s);
void launch_symmlq_begin(SymmlqScalars* sq, int S, cudaStream_t s);
void launch_symmlq_step(double* x, double* r1, double* r2, double* q, double* w, const double* b, long long n, int S,
                        SolverState* st, MinresScalars* ms, SymmlqScalars* sq, double* partials, int G,
                        cudaStream_t s);
template <typename T> void set_smem_attrs();
template <typename T> void set_smem_attrs_reg();
template <typename T> void launch_yfft_reg(const OpArgs<T>& a, bool inv, const SolverState* st, cudaStream_t s);
template <typename T> void launch_zgamma_reg(const OpArgs<T>& a, const SolverState* st, cudaStream_t s, int tz);
bool reg_length(int n);
void launch_yfft_tma(const OpArgs<float>& a, bool inv, const SolverState* st, cudaStream_t s);
bool encode_y_map(CUtensorMap* out, void* H, int hs, int ny, long long planes);
bool launch_zgamma_tma(const OpArgs<float>& a, int var, const SolverState* st, cudaStream_t s);
bool tma_z_variant_fits(const OpArgs<float>& a, int var);
bool launch_zgamma_regp(const OpArgs<float>& a, const SolverState* st, cudaStream_t s);
bool launch_zgamma_pipe(const OpArgs<float>& a, bool fused, const SolverState* st, cudaStream_t s,
                        double* partials = nullptr);
int zdot_count(const OpArgs<float>& a);
bool encode_zpipe_maps(CUtensorMap* th, CUtensorMap* tq, void* H, void* NQ, int hs, int ny, int nz, int c,
                       long long nsys);
void zpipe_prepare();
int multiprocessors();
// double-float passes (kernels_df.cu); DF and DF2 come from df.cuh
struct DF;
struct DF2;
bool df_supported(const OpArgs<double>& a);
void launch_d2df(const double* in, DF* out, long long n, cudaStream_t s);
void launch_d2df_inplace(void* buf, long long n, cudaStream_t s);
void launch_df_x(const OpArgs<double>& a, const DF2* twx, int mode, const double* in, double* out, SolverState* st,
                 double* partials, cudaStream_t s);
void launch_df_z(const OpArgs<DF>& a, cudaStream_t s);
void df_prepare();
bool encode_z_map(CUtensorMap* out, void* H, int hs, int ny, int nz, int c, long long nsys, int tz);
void tma_prepare();
void launch_wait_probe(int* fault, unsigned long long limit_ns, cudaStream_t s);
bool launch_xinv_reg(const OpArgs<float>& a, int mode, const float* xin, float* out, SolverState* st,
                     double* partials, cudaStream_t s, bool persistent, bool small = false, long long off = 0);
void xreg_prepare();
bool xinv_reg_fits(const OpArgs<float>& a);
bool launch_xfwd_reg(const OpArgs<float>& a, int mode, const float* in, float* x, const float* r, float* p,
                     const SolverState* st, cudaStream_t s);
bool xfwd_reg_fits(const OpArgs<float>& a);
bool plane_length(int n);
bool launch_xyfwd(const OpArgs<float>& a, int mode, const float* in, float* x, const float* r, float* p,
                  const SolverState* st, cudaStream_t s);
bool launch_xyinv(const OpArgs<float>& a, int mode, const float* xin, float* out, SolverState* st, double* partials,
                  cudaStream_t s);
// CG iteration with the update of z fused into the inverse pass (kernels_plane.cu)
void launch_cg_alpha(SolverState* st, const double* partials, int nb, int S, bool pdl, cudaStream_t s);
bool launch_xyinv_update(const OpArgs<float>& a, const float* p, float* z, SolverState* st, double* partials,
                         long long off, cudaStream_t s);
void plane_prepare();

}  // namespace lsh
