// fft.cuh -- batched in-place mixed-radix FFT of lines held in shared memory.
//
// Forward transforms are decimation-in-frequency (DIF): natural-order input,
// digit-reversed output.  Inverse transforms are decimation-in-time (DIT):
// digit-reversed input, natural-order output, unnormalised.  Because the
// Green-operator product between them is per frequency, the spectrum is never
// permuted: the kernels only need the frequency k stored at each position.
//
// Stage s of a DIF with radix r acts on spans of length L (L = n for the
// first stage, divided by r after each stage), m = L / r.  For j < m:
//   y_p = (sum_q a_q w_r^{pq}) w_L^{pj},  a_q = x[j + q m],  y_p -> x[j + p m],
// with w_N = exp(-2 i pi / N).  The frequency k of an n-point transform ends up
// at position pos(k) = sum_s d_s m_s, where k = d_1 + r_1 (d_2 + r_2 (...)).
// The DIT stage is the exact inverse of the DIF stage up to the factor r.
//
// All threads of the block cooperate; each stage ends with __syncthreads().
// Twiddles come from a per-axis table tw[t] = exp(-2 i pi t / n), t < n.
#pragma once

#include "common.cuh"

namespace lsh {

template <typename T, int R, bool INV> struct Dft;

template <typename T, bool INV> struct Dft<T, 2, INV> {
  static __device__ __forceinline__ void run(C2<T>* a, const C2<T>*, int) {
    C2<T> t = a[1];
    a[1] = csub<T>(a[0], t);
    a[0] = cadd<T>(a[0], t);
  }
};

template <typename T, bool INV> struct Dft<T, 4, INV> {
  static __device__ __forceinline__ void run(C2<T>* a, const C2<T>*, int) {
    C2<T> t0 = cadd<T>(a[0], a[2]), t1 = csub<T>(a[0], a[2]);
    C2<T> t2 = cadd<T>(a[1], a[3]), t3 = csub<T>(a[1], a[3]);
    C2<T> r3 = INV ? cmul_pi<T>(t3) : cmul_mi<T>(t3);  // w_4^{1} t3
    a[0] = cadd<T>(t0, t2);
    a[2] = csub<T>(t0, t2);
    a[1] = cadd<T>(t1, r3);
    a[3] = csub<T>(t1, r3);
  }
};

template <typename T, bool INV> struct Dft<T, 8, INV> {
  static __device__ __forceinline__ void run(C2<T>* a, const C2<T>* tw, int n) {
    const T h = (T)0.70710678118654752440084436210484903928;  // 1/sqrt(2)
    C2<T> e[4] = {a[0], a[2], a[4], a[6]};
    C2<T> o[4] = {a[1], a[3], a[5], a[7]};
    Dft<T, 4, INV>::run(e, tw, n);
    Dft<T, 4, INV>::run(o, tw, n);
    // o_p *= w_8^p
    C2<T> o1 = o[1], o3 = o[3];
    if (!INV) {
      o[1] = mkc<T>((o1.x + o1.y) * h, (o1.y - o1.x) * h);
      o[2] = cmul_mi<T>(o[2]);
      o[3] = mkc<T>((o3.y - o3.x) * h, -(o3.x + o3.y) * h);
    } else {
      o[1] = mkc<T>((o1.x - o1.y) * h, (o1.x + o1.y) * h);
      o[2] = cmul_pi<T>(o[2]);
      o[3] = mkc<T>(-(o3.x + o3.y) * h, (o3.x - o3.y) * h);
    }
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      a[p] = cadd<T>(e[p], o[p]);
      a[p + 4] = csub<T>(e[p], o[p]);
    }
  }
};

template <typename T, bool INV> struct Dft<T, 3, INV> {
  static __device__ __forceinline__ void run(C2<T>* a, const C2<T>*, int) {
    const T s3 = (T)0.86602540378443864676372317075293618347;  // sqrt(3)/2
    C2<T> s = cadd<T>(a[1], a[2]), d = csub<T>(a[1], a[2]);
    C2<T> m = mkc<T>(a[0].x - (T)0.5 * s.x, a[0].y - (T)0.5 * s.y);
    C2<T> rd = INV ? cmul_pi<T>(d) : cmul_mi<T>(d);  // +-i d
    a[0] = cadd<T>(a[0], s);
    a[1] = mkc<T>(m.x + s3 * rd.x, m.y + s3 * rd.y);
    a[2] = mkc<T>(m.x - s3 * rd.x, m.y - s3 * rd.y);
  }
};

template <typename T, bool INV> struct Dft<T, 5, INV> {
  static __device__ __forceinline__ void run(C2<T>* a, const C2<T>*, int) {
    const T c1 = (T)0.30901699437494742410229341718281905886;   // cos(2pi/5)
    const T c2 = (T)-0.80901699437494742410229341718281905886;  // cos(4pi/5)
    const T s1 = (T)0.95105651629515357211643933337938214340;   // sin(2pi/5)
    const T s2 = (T)0.58778525229247312916870595463907276860;   // sin(4pi/5)
    C2<T> p14 = cadd<T>(a[1], a[4]), m14 = csub<T>(a[1], a[4]);
    C2<T> p23 = cadd<T>(a[2], a[3]), m23 = csub<T>(a[2], a[3]);
    C2<T> b1 = mkc<T>(a[0].x + c1 * p14.x + c2 * p23.x, a[0].y + c1 * p14.y + c2 * p23.y);
    C2<T> b2 = mkc<T>(a[0].x + c2 * p14.x + c1 * p23.x, a[0].y + c2 * p14.y + c1 * p23.y);
    C2<T> u1 = mkc<T>(s1 * m14.x + s2 * m23.x, s1 * m14.y + s2 * m23.y);
    C2<T> u2 = mkc<T>(s2 * m14.x - s1 * m23.x, s2 * m14.y - s1 * m23.y);
    // forward: y1 = b1 - i u1, y4 = b1 + i u1, y2 = b2 - i u2, y3 = b2 + i u2
    C2<T> iu1 = INV ? cmul_pi<T>(u1) : cmul_mi<T>(u1);
    C2<T> iu2 = INV ? cmul_pi<T>(u2) : cmul_mi<T>(u2);
    a[0] = mkc<T>(a[0].x + p14.x + p23.x, a[0].y + p14.y + p23.y);
    a[1] = cadd<T>(b1, iu1);
    a[4] = csub<T>(b1, iu1);
    a[2] = cadd<T>(b2, iu2);
    a[3] = csub<T>(b2, iu2);
  }
};

// 16 = 4 x 4: x[n2 + 4 n1] -> X[k1 + 4 k2] = sum_n2 w4^(n2 k2) w16^(n2 k1) sum_n1 x[n2 + 4 n1] w4^(n1 k1)
template <typename T, bool INV> struct Dft<T, 16, INV> {
  static __device__ __forceinline__ void run(C2<T>* a, const C2<T>* tw, int n) {
    const T c1 = (T)0.92387953251128675612818318939678828682;  // cos(pi/8)
    const T s1 = (T)0.38268343236508977172845998403039886676;  // sin(pi/8)
    const T h = (T)0.70710678118654752440084436210484903928;   // cos(pi/4)
    C2<T> b[4][4];
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
      C2<T> c[4] = {a[n2], a[n2 + 4], a[n2 + 8], a[n2 + 12]};
      Dft<T, 4, INV>::run(c, tw, n);
#pragma unroll
      for (int k1 = 0; k1 < 4; ++k1) b[n2][k1] = c[k1];
    }
    // twiddles w16^m, m = n2 k1: (cos, -+sin) of 2 pi m / 16
    const T sg = INV ? (T)1 : (T)-1;
    const C2<T> w1 = mkc<T>(c1, sg * s1), w2 = mkc<T>(h, sg * h), w3 = mkc<T>(s1, sg * c1);
    const C2<T> w6 = mkc<T>(-h, sg * h), w9 = mkc<T>(-c1, -sg * s1);
    b[1][1] = cmul<T>(b[1][1], w1);
    b[1][2] = cmul<T>(b[1][2], w2);
    b[1][3] = cmul<T>(b[1][3], w3);
    b[2][1] = cmul<T>(b[2][1], w2);
    b[2][2] = INV ? cmul_pi<T>(b[2][2]) : cmul_mi<T>(b[2][2]);  // w16^4 = -+i
    b[2][3] = cmul<T>(b[2][3], w6);
    b[3][1] = cmul<T>(b[3][1], w3);
    b[3][2] = cmul<T>(b[3][2], w6);
    b[3][3] = cmul<T>(b[3][3], w9);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      C2<T> d[4] = {b[0][k1], b[1][k1], b[2][k1], b[3][k1]};
      Dft<T, 4, INV>::run(d, tw, n);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) a[k1 + 4 * k2] = d[k2];
    }
  }
};

// 32 = 2 x 16: X[k] = E[k] + w32^k O[k], X[k + 16] = E[k] - w32^k O[k] with E, O
// the 16-point DFTs of the even and odd samples (w32 = exp(-+2 i pi / 32)).
template <typename T, bool INV> struct Dft<T, 32, INV> {
  static __device__ __forceinline__ void run(C2<T>* a, const C2<T>* tw, int n) {
    // cos(pi k / 16), k = 0..8 (sin(pi k / 16) = cos(pi (8 - k) / 16))
    const T cs[9] = {(T)1.0,
                     (T)0.98078528040323044912618223613424,
                     (T)0.92387953251128675612818318939679,
                     (T)0.83146961230254523707878837761791,
                     (T)0.70710678118654752440084436210485,
                     (T)0.55557023301960222474283081394853,
                     (T)0.38268343236508977172845998403040,
                     (T)0.19509032201612826784828486847702,
                     (T)0.0};
    C2<T> e[16], o[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      e[j] = a[2 * j];
      o[j] = a[2 * j + 1];
    }
    Dft<T, 16, INV>::run(e, tw, n);
    Dft<T, 16, INV>::run(o, tw, n);
    const T sg = INV ? (T)1 : (T)-1;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      C2<T> w;
      if (k <= 8) w = mkc<T>(cs[k], sg * cs[8 - k]);
      else w = mkc<T>(-cs[16 - k], sg * cs[k - 8]);
      const C2<T> ow = k == 0 ? o[k] : cmul<T>(o[k], w);
      a[k] = cadd<T>(e[k], ow);
      a[k + 16] = csub<T>(e[k], ow);
    }
  }
};

// 7 points from the sums and differences of the pairs (q, 7 - q)
template <typename T, bool INV> struct Dft<T, 7, INV> {
  static __device__ __forceinline__ void run(C2<T>* a, const C2<T>*, int) {
    const T c[3] = {(T)0.62348980185873353052500488400424, (T)-0.22252093395631440428890256449679,
                    (T)-0.90096886790241912623610231950745};  // cos(2 pi k / 7)
    const T s[3] = {(T)0.78183148246802980870844452667406, (T)0.97492791218182360701813168299393,
                    (T)0.43388373911755812047576833284836};  // sin(2 pi k / 7)
    C2<T> p[3], m[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      p[q] = cadd<T>(a[q + 1], a[6 - q]);
      m[q] = csub<T>(a[q + 1], a[6 - q]);
    }
    const C2<T> a0 = a[0];
    a[0] = mkc<T>(a0.x + p[0].x + p[1].x + p[2].x, a0.y + p[0].y + p[1].y + p[2].y);
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
      C2<T> b = a0, u = mkc<T>((T)0, (T)0);
#pragma unroll
      for (int q = 1; q <= 3; ++q) {
        const int e = (k * q) % 7, f = e <= 3 ? e : 7 - e;  // angle 2 pi e / 7, folded
        const T sn = e <= 3 ? s[f - 1] : -s[f - 1];
        b.x += c[f - 1] * p[q - 1].x;
        b.y += c[f - 1] * p[q - 1].y;
        u.x += sn * m[q - 1].x;
        u.y += sn * m[q - 1].y;
      }
      const C2<T> iu = INV ? cmul_pi<T>(u) : cmul_mi<T>(u);
      a[k] = cadd<T>(b, iu);
      a[7 - k] = csub<T>(b, iu);
    }
  }
};

// Composite lengths with coprime factors R = A * B in registers, by the Chinese
// remainder theorem (Good-Thomas): with n = (B n1 + A n2) mod R and k = (B B' k1 +
// A A' k2) mod R, B' = B^{-1} mod A and A' = A^{-1} mod B, w_R^(nk) = w_A^(n1 k1)
// w_B^(n2 k2): A- and B-point DFTs with no twiddles between them.
__host__ __device__ constexpr int inverse_mod(int a, int m) {
  for (int x = 1; x < m; ++x)
    if ((a * x) % m == 1) return x;
  return 0;
}
template <typename T, int A, int B, bool INV> struct DftPFA {
  static __device__ __forceinline__ void run(C2<T>* a, const C2<T>* tw, int n) {
    constexpr int R = A * B;
    constexpr int eb = B * inverse_mod(B % A, A), ea = A * inverse_mod(A % B, B);
    C2<T> b[B][A];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) b[n2][n1] = a[(B * n1 + A * n2) % R];
      Dft<T, A, INV>::run(b[n2], tw, n);
    }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      C2<T> d[B];
#pragma unroll
      for (int n2 = 0; n2 < B; ++n2) d[n2] = b[n2][k1];
      Dft<T, B, INV>::run(d, tw, n);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) a[(eb * k1 + ea * k2) % R] = d[k2];
    }
  }
};
template <typename T, bool INV> struct Dft<T, 6, INV> : DftPFA<T, 2, 3, INV> {};
template <typename T, bool INV> struct Dft<T, 10, INV> : DftPFA<T, 2, 5, INV> {};
template <typename T, bool INV> struct Dft<T, 12, INV> : DftPFA<T, 4, 3, INV> {};
template <typename T, bool INV> struct Dft<T, 24, INV> : DftPFA<T, 8, 3, INV> {};

// 9 = 3 x 3: x[3 n1 + n2] -> X[k1 + 3 k2] = sum_n2 w3^(n2 k2) w9^(n2 k1) sum_n1 x w3^(n1 k1)
template <typename T, bool INV> struct Dft<T, 9, INV> {
  static __device__ __forceinline__ void run(C2<T>* a, const C2<T>* tw, int n) {
    const T sg = INV ? (T)1 : (T)-1;
    // w9^1, w9^2, w9^4
    const C2<T> w1 = mkc<T>((T)0.76604444311897803520239265055542, sg * (T)0.64278760968653932632264340990726);
    const C2<T> w2 = mkc<T>((T)0.17364817766693034885171662676931, sg * (T)0.98480775301220805936674302458952);
    const C2<T> w4 = mkc<T>((T)-0.93969262078590838405410927732473, sg * (T)0.34202014332566873304409961468226);
    C2<T> b[3][3];
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 3; ++n1) b[n2][n1] = a[3 * n1 + n2];
      Dft<T, 3, INV>::run(b[n2], tw, n);
    }
    b[1][1] = cmul<T>(b[1][1], w1);
    b[1][2] = cmul<T>(b[1][2], w2);
    b[2][1] = cmul<T>(b[2][1], w2);
    b[2][2] = cmul<T>(b[2][2], w4);
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      C2<T> d[3] = {b[0][k1], b[1][k1], b[2][k1]};
      Dft<T, 3, INV>::run(d, tw, n);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) a[k1 + 3 * k2] = d[k2];
    }
  }
};

template <typename T, int R, bool INV>
__device__ __forceinline__ void butterfly(C2<T>* base, int m, int te, const C2<T>* tw, int n) {
  C2<T> a[R];
#pragma unroll
  for (int q = 0; q < R; ++q) a[q] = base[q * m];
  if (!INV) {
    Dft<T, R, false>::run(a, tw, n);
    if (te != 0) {
#pragma unroll
      for (int p = 1; p < R; ++p) a[p] = cmul<T>(a[p], tw[p * te]);
    }
  } else {
    if (te != 0) {
#pragma unroll
      for (int p = 1; p < R; ++p) a[p] = cmulc<T>(a[p], tw[p * te]);
    }
    Dft<T, R, true>::run(a, tw, n);
  }
#pragma unroll
  for (int q = 0; q < R; ++q) base[q * m] = a[q];
}

// Stage `st` of plan pl (radix R) over nlines lines (line stride ls, element stride 1).
template <typename T, bool INV, int R>
__device__ __forceinline__ void fft_stage_r(C2<T>* __restrict__ buf, int nlines, const FastDiv& dl, int ls,
                                            const Plan1D& pl, int st, const C2<T>* __restrict__ tw) {
  const int m = pl.m[st], nb = pl.n / R, total = nb * nlines, tws = pl.tws[st];
  const bool jmajor = m >= 16;
  const FastDiv dm(m, pl.mag_m[st]), dnb(nb, pl.mag_nb[st]);
  for (int w = threadIdx.x; w < total; w += blockDim.x) {
    int line, b;
    if (jmajor) {
      line = dnb.div(w);
      b = w - line * nb;
    } else {
      b = dl.div(w);
      line = w - b * nlines;
    }
    const int sp = dm.div(b), j = b - sp * m;
    butterfly<T, R, INV>(buf + line * ls + sp * (m * R) + j, m, j * tws, tw, pl.n);
  }
}

template <typename T, bool INV>
__device__ __forceinline__ void fft_stage(C2<T>* __restrict__ buf, int nlines, const FastDiv& dl, int ls,
                                          const Plan1D& pl, int st, const C2<T>* __restrict__ tw) {
  switch (pl.radix[st]) {
    case 12: fft_stage_r<T, INV, 12>(buf, nlines, dl, ls, pl, st, tw); break;
    case 10: fft_stage_r<T, INV, 10>(buf, nlines, dl, ls, pl, st, tw); break;
    case 9: fft_stage_r<T, INV, 9>(buf, nlines, dl, ls, pl, st, tw); break;
    case 8: fft_stage_r<T, INV, 8>(buf, nlines, dl, ls, pl, st, tw); break;
    case 7: fft_stage_r<T, INV, 7>(buf, nlines, dl, ls, pl, st, tw); break;
    case 6: fft_stage_r<T, INV, 6>(buf, nlines, dl, ls, pl, st, tw); break;
    case 5: fft_stage_r<T, INV, 5>(buf, nlines, dl, ls, pl, st, tw); break;
    case 4: fft_stage_r<T, INV, 4>(buf, nlines, dl, ls, pl, st, tw); break;
    case 3: fft_stage_r<T, INV, 3>(buf, nlines, dl, ls, pl, st, tw); break;
    default: fft_stage_r<T, INV, 2>(buf, nlines, dl, ls, pl, st, tw); break;
  }
}

// ---------------------------------------------------------------- compile-time schedules
// For the common lengths the radix sequence is a template argument: every
// index split becomes a shift or a mask and the stage loop unrolls.
template <typename T, bool INV, int N, int R, int L>
__device__ __forceinline__ void stage_ct(C2<T>* __restrict__ buf, int nlines, int ls, const C2<T>* __restrict__ tw) {
  constexpr int m = L / R, nb = N / R, tws = N / L;
  constexpr bool jmajor = m >= 16;
  const int total = nb * nlines;
  const FastDiv dl(nlines);
  for (int w = threadIdx.x; w < total; w += blockDim.x) {
    int line, b;
    if (jmajor) {
      line = w / nb;
      b = w - line * nb;
    } else {
      b = dl.div(w);
      line = w - b * nlines;
    }
    const int sp = b / m, j = b - sp * m;
    butterfly<T, R, INV>(buf + line * ls + sp * L + j, m, j * tws, tw, N);
  }
}

template <typename T, int N, int L, int... Rs> struct DifStages {
  static __device__ __forceinline__ void run(C2<T>*, int, int, const C2<T>*) {}
};
template <typename T, int N, int L, int R, int... Rs> struct DifStages<T, N, L, R, Rs...> {
  static __device__ __forceinline__ void run(C2<T>* buf, int nlines, int ls, const C2<T>* tw) {
    stage_ct<T, false, N, R, L>(buf, nlines, ls, tw);
    __syncthreads();
    DifStages<T, N, L / R, Rs...>::run(buf, nlines, ls, tw);
  }
};
// DIT stages run the DIF radices in reverse; the span of a stage is its radix
// times the product of the radices after it.
template <typename T, int N, int... Rs> struct DitStages {
  static constexpr int P = 1;
  static __device__ __forceinline__ void run(C2<T>*, int, int, const C2<T>*) {}
};
template <typename T, int N, int R, int... Rs> struct DitStages<T, N, R, Rs...> {
  static constexpr int P = R * DitStages<T, N, Rs...>::P;
  static __device__ __forceinline__ void run(C2<T>* buf, int nlines, int ls, const C2<T>* tw) {
    DitStages<T, N, Rs...>::run(buf, nlines, ls, tw);
    stage_ct<T, true, N, R, P>(buf, nlines, ls, tw);
    __syncthreads();
  }
};

template <int... Rs> __device__ __forceinline__ bool plan_is(const Plan1D& pl) {
  constexpr int r[] = {Rs...};
  constexpr int k = sizeof...(Rs);
  if (pl.nst != k) return false;
#pragma unroll
  for (int i = 0; i < k; ++i)
    if (pl.radix[i] != r[i]) return false;
  return true;
}

template <typename T, bool INV, int N, int... Rs>
__device__ __forceinline__ bool try_fixed(C2<T>* buf, int nlines, int ls, const Plan1D& pl, const C2<T>* tw) {
  if (pl.n != N || !plan_is<Rs...>(pl)) return false;
  if (INV) DitStages<T, N, Rs...>::run(buf, nlines, ls, tw);
  else DifStages<T, N, N, Rs...>::run(buf, nlines, ls, tw);
  return true;
}

template <typename T, bool INV>
__device__ void fft_lines_generic(C2<T>* buf, int nlines, int ls, const Plan1D& pl, const C2<T>* tw);

// Forward (DIF) or inverse (DIT) transform of nlines lines; ends synchronised.
// The fixed schedules mirror the host's radix choice (lsh_make_plan); any other
// plan runs the generic stage loop.
template <typename T, bool INV>
__device__ void fft_lines(C2<T>* buf, int nlines, int ls, const Plan1D& pl, const C2<T>* tw) {
  if (try_fixed<T, INV, 128, 4, 8, 4>(buf, nlines, ls, pl, tw)) return;
  if (try_fixed<T, INV, 64, 8, 8>(buf, nlines, ls, pl, tw)) return;
  if (try_fixed<T, INV, 256, 8, 8, 4>(buf, nlines, ls, pl, tw)) return;
  if (try_fixed<T, INV, 32, 8, 4>(buf, nlines, ls, pl, tw)) return;
  if (try_fixed<T, INV, 96, 12, 8>(buf, nlines, ls, pl, tw)) return;
  if (try_fixed<T, INV, 48, 8, 6>(buf, nlines, ls, pl, tw)) return;
  if (try_fixed<T, INV, 16, 4, 4>(buf, nlines, ls, pl, tw)) return;
  fft_lines_generic<T, INV>(buf, nlines, ls, pl, tw);
}

template <typename T, bool INV>
__device__ void fft_lines_generic(C2<T>* buf, int nlines, int ls, const Plan1D& pl, const C2<T>* tw) {
  const FastDiv dl(nlines);
  for (int k = 0; k < pl.nst; ++k) {
    fft_stage<T, INV>(buf, nlines, dl, ls, pl, INV ? pl.nst - 1 - k : k, tw);
    __syncthreads();
  }
}

}  // namespace lsh
