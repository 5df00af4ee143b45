// Objective, gradient and Hessian-vector product of Sec. 2.2 (eq_chi,
// eq_cost) on grids of any side lengths whose prime factors are 2, 3, 5 and 7
// (up to 1024 pixels a side), for callers whose maps are not powers of two.
//
//   chi^2(s) = |s|^2 + (d - x)^T W (d - x),  x = U^-1 R(k) sqrt(P) s,
//   grad     = 2 (s - sqrt(P) R(k)^T U W (d - x)),
//
// with s the half-plane unitary spectrum [C][ny][nx/2+1] of a real field, U
// the unitary 2-D DFT ((ny nx)^-1/2), W = mask * Ninv per pixel and, for the
// joint E/B pair (C = 2), R(k) the Kaiser-Squires rotation of App. C at the
// wavevector (mx / nx, my / ny) with s = 0 on the Nyquist lines.  With d
// omitted the data term sees d = 0, so grad = 2 (I + A^T W A) s: the
// Hessian-vector product.
//
// Kernels:
//   k_any_prep    once per call: sqrt(P), the rotation's cosine and sine per mode
//                 and the roots of unity of both lengths, shared by all maps;
//   k_any_colinv  per column tile: R sqrt(P) s, inverse DFT along y -> scratch;
//   k_any_row     per pair of rows, a warp or a block each: c2r along x, r = d - x, W r, sum r W r,
//                 r2c along x -> scratch;
//   k_any_colfwd  per column tile: forward DFT along y, sqrt(P) R^T / sqrt N,
//                 grad, sum of |s|^2 with the half-plane weights;
// then k_any_final adds the partial sums of each map in a fixed order.
//
// The DFTs are Stockham autosort transforms (pass with radix R, span Ns:
// butterfly j reads j + r L/R, multiplies by exp(+-2 pi i r (j mod Ns) / (Ns R)),
// does a length-R DFT and writes (j - j mod Ns) R + j mod Ns + r Ns) of two to
// four passes with radices up to 16, composite ones included, done in registers.
// The first pass reads global memory with the per-mode operator applied, the last
// one hands its values to the stage's epilogue, and the passes between exchange
// through two shared-memory buffers.  Two rows a, b of a map are one complex
// sequence a + i b, which carries both real transforms.
//
// What bounds them: HBM and instruction issue for FP32, the FP64 units for FP64
// (two lanes a clock and SM): so every transcendental, square root and division is taken
// out of the maps' passes, and the FP32 path's FP64-accurate sums run in FP32
// (WfSum).  One value per thread and pass with sincospi twiddles and radices up to
// 7 had taken, 64 maps of 768^2 FP32: 0.40 + 1.64 + 0.61 + 0.08 ms; 8 E/B maps of
// 375 x 315 FP64: 0.64 + 2.35 + 0.66 + 0.04 ms.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "wf_api_internal.h"
#include "wf_fft.cuh"
#include "wf_reg.cuh"

#define WF_ANY_MAXP 4     // passes of one transform at most (7-smooth lengths up to 1024)
#define WF_ANY_MAXN 1024
#define WF_ANY_THREADS 512  // most threads of a column block
#define WF_ANY_ROWW 8       // most warps of a row block
#define WF_ANY_TEAMT 128    // most threads of a row block of one pair

// One transform length: its passes, with the spans and their reciprocals
// ceil(2^32 / d) (n / d = umulhi(n, m), exact for n d < 2^32).
struct WfAnyPlan {
  int L, np;
  int R[WF_ANY_MAXP], Ns[WF_ANY_MAXP], LR[WF_ANY_MAXP];
  unsigned mNs[WF_ANY_MAXP];
};
struct WfAnyGeo {
  int B, C, ny, nx, h1;  // h1 = nx / 2 + 1 half-plane columns
  int tc, lgtc, gx;      // columns of a tile (a power of two), tiles: ceil(h1 / tc)
  int roww, nrb;         // row pairs of a row block, row blocks
  int roww_t;            // threads of a row block: a warp a pair, or all for one
  int rpitch;            // shared-memory places of a row sequence
  double inv_sqrt_n;     // (ny nx)^-1/2
  WfAnyPlan py, px;
};

// cos and sin of 2 pi n / d at compile time: Taylor series of the angle brought
// into [-pi, pi], summed until the terms vanish.
constexpr double wf_any_series(double x, double term, int k) {
  double sum = term;
  for (; k < 60; k += 2) {
    term *= -x * x / ((double)k * (k + 1));
    sum += term;
  }
  return sum;
}
constexpr double wf_any_angle(int n, int d) {
  n %= d;
  if (2 * n > d) n -= d;
  return 6.283185307179586476925286766559 * (double)n / (double)d;
}
constexpr double wf_any_cos(int n, int d) { return wf_any_series(wf_any_angle(n, d), 1.0, 1); }
constexpr double wf_any_sin(int n, int d) { return wf_any_series(wf_any_angle(n, d), wf_any_angle(n, d), 2); }
template <int R> struct WfAnyRoots {  // of length R
  double c[R], s[R];
  constexpr WfAnyRoots() : c(), s() {
    for (int t = 0; t < R; ++t) {
      c[t] = wf_any_cos(t, R);
      s[t] = wf_any_sin(t, R);
    }
  }
};

// Odd prime length R: sums and differences of the pairs r, R - r.
template <typename T, int R, int DIR>
__device__ __forceinline__ void wf_any_prime(V2<T>* v) {
  constexpr int H = (R - 1) / 2;
  constexpr WfAnyRoots<R> w;
  V2<T> p[H], m[H], x0 = v[0];
#pragma unroll
  for (int r = 1; r <= H; ++r) {
    p[r - 1] = cadd<T>(v[r], v[R - r]);
    m[r - 1] = csub<T>(v[r], v[R - r]);
    x0 = cadd<T>(x0, p[r - 1]);
  }
#pragma unroll
  for (int q = 1; q <= H; ++q) {
    V2<T> a = v[0], b = mk<T>((T)0, (T)0);
#pragma unroll
    for (int r = 1; r <= H; ++r) {
      const T c = (T)w.c[r * q % R], s = (T)(DIR * w.s[r * q % R]);
      a = mk<T>(wf_fma(c, p[r - 1].x, a.x), wf_fma(c, p[r - 1].y, a.y));
      b = mk<T>(wf_fma(s, m[r - 1].x, b.x), wf_fma(s, m[r - 1].y, b.y));
    }
    v[q] = mk<T>(a.x - b.y, a.y + b.x);  // a + i b
    v[R - q] = mk<T>(a.x + b.y, a.y - b.x);
    // v[q] and v[R - q] (q >= 1) are no longer needed: p and m hold them
  }
  v[0] = x0;
}
template <int R> struct WfAnySplit;  // R = P Q
template <> struct WfAnySplit<6> { static constexpr int P = 2, Q = 3; };
template <> struct WfAnySplit<9> { static constexpr int P = 3, Q = 3; };
template <> struct WfAnySplit<10> { static constexpr int P = 2, Q = 5; };
template <> struct WfAnySplit<12> { static constexpr int P = 4, Q = 3; };
template <> struct WfAnySplit<14> { static constexpr int P = 2, Q = 7; };
template <> struct WfAnySplit<15> { static constexpr int P = 3, Q = 5; };

// Multiply by exp(DIR 2 pi i N / D), N and D known at compile time.
template <typename T, int DIR, int N, int D>
__device__ __forceinline__ V2<T> wf_any_rot(V2<T> v) {
  if constexpr (N % D == 0) return v;
  else if constexpr (4 * (N % D) == D) return DIR > 0 ? mul_i<T>(v) : mk<T>(v.y, -v.x);
  else {
    constexpr WfAnyRoots<D> w;
    constexpr double c = w.c[N % D], s = DIR * w.s[N % D];
    return cmul<T>(v, mk<T>((T)c, (T)s));
  }
}
template <typename T, int R, int DIR> __device__ __forceinline__ void wf_any_dft(V2<T>* v);
template <typename T, int P, int Q, int DIR, int N2, int K1>
__device__ __forceinline__ void wf_any_twist(V2<T>* y) {  // y[k1] *= w_R^(n2 k1), k1 = K1 ..
  if constexpr (K1 < P) {
    y[K1] = wf_any_rot<T, DIR, N2 * K1, P * Q>(y[K1]);
    wf_any_twist<T, P, Q, DIR, N2, K1 + 1>(y);
  }
}
template <typename T, int P, int Q, int DIR, int N2>
__device__ __forceinline__ void wf_any_ct1(const V2<T>* v, V2<T>* y) {  // columns n2 = N2 ..: y[n2 P + k1]
  if constexpr (N2 < Q) {
    V2<T> u[P];
#pragma unroll
    for (int n1 = 0; n1 < P; ++n1) u[n1] = v[Q * n1 + N2];
    wf_any_dft<T, P, DIR>(u);
    wf_any_twist<T, P, Q, DIR, N2, 1>(u);
#pragma unroll
    for (int k1 = 0; k1 < P; ++k1) y[N2 * P + k1] = u[k1];
    wf_any_ct1<T, P, Q, DIR, N2 + 1>(v, y);
  }
}
// Length-R DFT in registers, natural order in and out.
template <typename T, int R, int DIR>
__device__ __forceinline__ void wf_any_dft(V2<T>* v) {
  if constexpr (R == 2 || R == 4 || R == 8 || R == 16) {
    wf_rg_dft<T, R, DIR, 1>(v);
  } else if constexpr (R == 3 || R == 5 || R == 7) {
    wf_any_prime<T, R, DIR>(v);
  } else {  // Cooley-Tukey: n = Q n1 + n2, k = k1 + P k2
    constexpr int P = WfAnySplit<R>::P, Q = WfAnySplit<R>::Q;
    V2<T> y[R];
    wf_any_ct1<T, P, Q, DIR, 0>(v, y);
#pragma unroll
    for (int k1 = 0; k1 < P; ++k1) {
      V2<T> u[Q];
#pragma unroll
      for (int n2 = 0; n2 < Q; ++n2) u[n2] = y[n2 * P + k1];
      wf_any_dft<T, Q, DIR>(u);
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2) v[k1 + P * k2] = u[k2];
    }
  }
}

// One pass of radix R.  TILE: the block's threads over 1 << lgS interleaved
// sequences, consecutive lanes in consecutive sequences (column tiles); else the
// lanes of a warp over one sequence (rows).  ld(t, e) gives element e of sequence
// t; st(t, o, Ns, v) takes the elements o + q Ns.
template <typename T, int R, int DIR, bool TILE, class LD, class ST>
__device__ __forceinline__ void wf_any_pass(const WfAnyPlan& P, int p, int lgS, const V2<T>* tw, LD& ld, ST& st) {
  const int LR = P.LR[p], Ns = P.Ns[p];
  const int b0 = TILE ? threadIdx.x : (threadIdx.x & 31), db = TILE ? blockDim.x : 32, nbf = TILE ? LR << lgS : LR;
  for (int b = b0; b < nbf; b += db) {
    const int t = TILE ? b & ((1 << lgS) - 1) : 0, j = TILE ? b >> lgS : b;
    V2<T> v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = ld(t, j + r * LR);
    int k = 0;
    if (p > 0) {
      k = j - (int)__umulhi(j, P.mNs[p]) * Ns;
      const int step = k * (LR / Ns);  // exp(2 pi i r k / (Ns R)) = root r k L / (Ns R) of the L-th
      int x = step;
#pragma unroll
      for (int r = 1; r < R; ++r, x += step) v[r] = cmul<T>(v[r], twid<T, DIR>(tw, WF_CHK(x, P.L)));
    }
    wf_any_dft<T, R, DIR>(v);
    st(t, (j - k) * R + k, Ns, v, std::integral_constant<int, R>());
  }
}
template <typename T, int DIR, bool TILE, class LD, class ST>
__device__ __forceinline__ void wf_any_radix(const WfAnyPlan& P, int p, int lgS, const V2<T>* tw, LD& ld, ST& st) {
  switch (P.R[p]) {
    case 2: wf_any_pass<T, 2, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 3: wf_any_pass<T, 3, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 4: wf_any_pass<T, 4, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 5: wf_any_pass<T, 5, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 6: wf_any_pass<T, 6, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 7: wf_any_pass<T, 7, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 8: wf_any_pass<T, 8, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 9: wf_any_pass<T, 9, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 10: wf_any_pass<T, 10, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 12: wf_any_pass<T, 12, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 14: wf_any_pass<T, 14, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    case 15: wf_any_pass<T, 15, DIR, TILE>(P, p, lgS, tw, ld, st); break;
    default: wf_any_pass<T, 16, DIR, TILE>(P, p, lgS, tw, ld, st); break;
  }
}
// All passes: ld0 feeds the first, stl takes the last one's values, A and Bf the
// buffers between (place at(t, e)).  Returns the buffer the last pass did not read,
// where stl may write (out, called first).
template <typename T> __device__ __forceinline__ V2<T>* wf_any_out(const WfAnyPlan& P, V2<T>* A, V2<T>* Bf) {
  return (P.np & 1) ? A : Bf;  // pass p reads A for odd p, Bf for even p >= 2
}
template <typename T, int DIR, bool TILE, class AT, class LD0, class STL>
__device__ __forceinline__ void wf_any_fft(const WfAnyPlan& P, int lgS, V2<T>* A, V2<T>* Bf, const V2<T>* tw,
                                           AT& at, LD0& ld0, STL& stl) {
  const int np = P.np;
  if (np == 1) {
    wf_any_radix<T, DIR, TILE>(P, 0, lgS, tw, ld0, stl);
    return;
  }
  V2<T> *in = Bf, *out = A;
  auto ld = [&](int t, int e) { return in[at(t, e)]; };
  auto st = [&](int t, int o, int Ns, V2<T>* v, auto rt) {
#pragma unroll
    for (int q = 0; q < decltype(rt)::value; ++q) out[at(t, o + q * Ns)] = v[q];
  };
  wf_any_radix<T, DIR, TILE>(P, 0, lgS, tw, ld0, st);
  for (int p = 1; p < np; ++p) {
    if constexpr (TILE) __syncthreads();
    else __syncwarp();
    V2<T>* x = in;
    in = out;
    out = x;
    if (p + 1 < np) wf_any_radix<T, DIR, TILE>(P, p, lgS, tw, ld, st);
    else wf_any_radix<T, DIR, TILE>(P, p, lgS, tw, ld, stl);
  }
}

// Sum of many products a b (WfSum), two at a time; a pair that FP32 does not hold is
// taken in FP64, out of line: inlined it is predicated, and instructions that do nothing
// hold the FP64 unit all the same (64 maps of 768^2: 908 us a call against 751).
template <typename T> static __device__ __noinline__ double wf_any_far(double far, T a0, T b0, T a1, T b1) {
  return fma((double)a1, (double)b1, fma((double)a0, (double)b0, far));
}
template <typename T> struct WfAnySum {
  WfSum<T> near;
  double far = 0.0;
  __device__ __forceinline__ void add(const T (&a)[2], const T (&b)[2]) {
    if (!wf_sum_products(near, a, b)) far = wf_any_far<T>(far, a[0], b[0], a[1], b[1]);
  }
  __device__ __forceinline__ double get() const { return near.get() + far; }
};

// Tables of a call.
template <typename T> struct WfAnyTab {
  T* amp;         // [C][ny][h1] sqrt(P)
  V2<T>* rot;     // [ny][h1] (cosine, sine), two channels only
  V2<T>* twy;     // exp(-2 pi i k / ny)
  V2<T>* twx;     // exp(-2 pi i k / nx)
};

// Kaiser-Squires cosine and sine at half-plane mode (ky, kx): wavevector
// (mx / nx, my / ny) scaled by nx ny to the integers (mx ny, my nx); signed
// mode numbers, R = I at k = 0, sine 0 on the Nyquist line of an even side.
__device__ __forceinline__ void wf_any_ks(const WfAnyGeo& G, int ky, int kx, double* c, double* s) {
  const int my = ky <= (G.ny - 1) / 2 ? ky : ky - G.ny;
  const double qx = (double)kx * G.ny, qy = (double)my * G.nx;
  const double k2 = qx * qx + qy * qy;
  if (k2 == 0.0) {
    *c = 1.0;
    *s = 0.0;
    return;
  }
  *c = (qx * qx - qy * qy) / k2;
  const bool nyq = ((G.nx % 2) == 0 && 2 * kx == G.nx) || ((G.ny % 2) == 0 && 2 * ky == G.ny);
  *s = nyq ? 0.0 : 2.0 * qx * qy / k2;
}

// The tables: what the maps' passes share, computed once (a division, a square
// root or a sine costs the FP64 path tens of its two lanes' cycles).
template <typename T>
__global__ void __launch_bounds__(256) k_any_prep(const __grid_constant__ WfAnyGeo G, const T* P, WfAnyTab<T> tab) {
  const int nm = G.ny * G.h1, stride = gridDim.x * blockDim.x, i0 = blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = i0; i < G.C * nm; i += stride) tab.amp[i] = sqrt(P[i]);
  if (G.C == 2)
    for (int i = i0; i < nm; i += stride) {
      const int ky = i / G.h1, kx = i - ky * G.h1;
      double c, s;
      wf_any_ks(G, ky, kx, &c, &s);
      tab.rot[i] = mk<T>((T)c, (T)s);
    }
  for (int i = i0; i < G.ny + G.nx; i += stride) {
    const bool y = i < G.ny;
    const int k = y ? i : i - G.ny;
    double s, c;
    sincospi(2.0 * k / (y ? G.ny : G.nx), &s, &c);
    (y ? tab.twy : tab.twx)[k] = mk<T>((T)c, (T)-s);
  }
}

// Inverse column stage: tile of tc half-plane columns of map blockIdx.y, all
// channels; the per-mode operator R(k) sqrt(P) on the way in, then the inverse
// DFT along y into scratch [B][C][ny][h1].  Sequence t = channel tc + column; a
// column beyond h1 repeats the last one and is not stored.
template <typename T, int C>
__global__ void __launch_bounds__(WF_ANY_THREADS)
k_any_colinv(const __grid_constant__ WfAnyGeo G, const V2<T>* s, WfAnyTab<T> tab, V2<T>* scr) {
  extern __shared__ __align__(16) unsigned char wf_smem[];
  const int b = blockIdx.y, kx0 = blockIdx.x * G.tc, ny = G.ny, h1 = G.h1, tc = G.tc, lgS = G.lgtc + (C == 2), S = 1 << lgS;
  V2<T>* tw = (V2<T>*)wf_smem;
  V2<T>* A = tw + ny;
  V2<T>* Bf = A + S * ny;
  const size_t vsz = (size_t)C * ny * h1;
  const V2<T>* sb = s + (size_t)b * vsz;
  V2<T>* out = scr + (size_t)b * vsz;
  for (int i = threadIdx.x; i < ny; i += blockDim.x) tw[i] = tab.twy[i];
  const int nm = ny * h1;
  auto at = [&](int t, int e) { return (int)WF_CHK((e << lgS) + t, S * ny); };
  auto ld0 = [&](int t, int e) -> V2<T> {
    const int col = t & (tc - 1), kx = min(kx0 + col, h1 - 1), m = (int)WF_CHK(e * h1 + kx, nm);
    if constexpr (C == 1) {
      return cscale<T>(__ldg(sb + m), __ldg(tab.amp + m));
    } else {
      const V2<T> a0 = cscale<T>(__ldg(sb + m), __ldg(tab.amp + m)), a1 = cscale<T>(__ldg(sb + nm + m), __ldg(tab.amp + nm + m));
      const V2<T> r = __ldg(tab.rot + m);
      return t < tc ? mk<T>(r.x * a0.x - r.y * a1.x, r.x * a0.y - r.y * a1.y)
                    : mk<T>(r.y * a0.x + r.x * a1.x, r.y * a0.y + r.x * a1.y);
    }
  };
  auto stl = [&](int t, int o, int Ns, V2<T>* v, auto rt) {
    const int col = t & (tc - 1), c = C == 2 ? t >> G.lgtc : 0;
    if (kx0 + col < h1) {
#pragma unroll
      for (int q = 0; q < decltype(rt)::value; ++q) out[WF_CHK(c * nm + (o + q * Ns) * h1 + kx0 + col, vsz)] = v[q];
    }
  };
  wf_any_fft<T, +1, true>(G.py, lgS, A, Bf, tw, at, ld0, stl);
}

// Row stage: every warp takes one pair of rows of map blockIdx.y (rows of all
// channels, in order), with no barrier but its own.  Z[k] = A[k] + i B[k] over
// k <= nx/2 and conj A[nx-k] + i conj B[nx-k] beyond; its inverse DFT is a + i b.
// Then r = d - x, W r and sum r W r, and the forward DFT Z of W r: A[k] = (Z[k] +
// conj Z[nx-k]) / 2, B[k] = -i (Z[k] - conj Z[nx-k]) / 2.  An odd last row pairs
// with itself, its partner's weights 0.  Element e sits at e + e / 16 of the warp's
// places: the first pass writes with stride R.
// TEAM: a block takes one pair, its threads in place of the warp's lanes.  With few
// pairs a warp each leaves most of the chip idle and the stage lasts as long as one
// warp's chain of passes.
template <typename T, bool TEAM>
__global__ void __launch_bounds__(TEAM ? WF_ANY_TEAMT : WF_ANY_ROWW * 32, sizeof(T) == 4 && !TEAM ? 2 : 1)
k_any_row(const __grid_constant__ WfAnyGeo G, const T* d, const uint8_t* mask, const T* Ninv, const V2<T>* twx, V2<T>* scr,
          double* dpart) {
  extern __shared__ __align__(16) unsigned char wf_smem[];
  const int b = blockIdx.y, ny = G.ny, nx = G.nx, h1 = G.h1, rows = G.C * ny, rp = G.rpitch;
  const int nteam = TEAM ? 1 : blockDim.x >> 5, team = TEAM ? blockDim.x : 32;  // teams, and threads of one
  const int lane = TEAM ? threadIdx.x : threadIdx.x & 31, wid = TEAM ? 0 : threadIdx.x >> 5;
  V2<T>* tw = (V2<T>*)wf_smem;
  V2<T>* A = tw + nx + 2 * wid * rp;
  V2<T>* Bf = A + rp;
  const int pair = blockIdx.x * nteam + wid, ra = 2 * pair;
  const bool on = ra < rows, two = ra + 1 < rows;  // a warp beyond the last pair only meets the block's barriers
  WfAnySum<T> acc;
  if (on) {
    // this pair's pixels start towards L2
    const size_t pix = ((size_t)b * rows + ra) * nx;
    const char* pw = (const char*)(Ninv + pix);
    const char* pd = (const char*)(d + pix);
    for (int i = lane * 128; i < (two ? 2 : 1) * nx * (int)sizeof(T); i += team * 128) {
      asm volatile("prefetch.global.L2 [%0];" ::"l"(pw + i));
      if (d) asm volatile("prefetch.global.L2 [%0];" ::"l"(pd + i));
    }
  }
  for (int i = threadIdx.x; i < nx; i += blockDim.x) tw[i] = twx[i];
  __syncthreads();
  auto sync = [] {
    if constexpr (TEAM) __syncthreads();  // a block's only pair is never beyond the last
    else __syncwarp();
  };
  if (on) {
    const size_t vsz = (size_t)rows * h1, psz = (size_t)rows * nx;
    V2<T>* rowa = scr + (size_t)b * vsz + (size_t)ra * h1;
    V2<T>* rowb = two ? rowa + h1 : rowa;
    const size_t pix = (size_t)b * psz + (size_t)ra * nx;
    const T *wa = Ninv + pix, *wb = two ? wa + nx : wa, *da = d + pix, *db = two ? da + nx : da;
    const int ya = ra < ny ? ra : ra - ny, yb = !two ? ya : ra + 1 < ny ? ra + 1 : ra + 1 - ny;
    const uint8_t *ma = mask + ((size_t)b * ny + ya) * nx, *mb = mask + ((size_t)b * ny + yb) * nx;
    const T onb = two ? (T)1 : (T)0;
    auto at = [&](int, int e) { return (int)WF_CHK(e + (e >> 4), rp); };
    auto ld0 = [&](int, int e) -> V2<T> {
      const bool lo = e < h1;
      const int m = (int)WF_CHK(lo ? e : nx - e, h1);
      const V2<T> x = __ldcg(rowa + m), y = __ldcg(rowb + m);
      return lo ? mk<T>(x.x - y.y, x.y + y.x) : mk<T>(x.x + y.y, y.x - x.y);
    };
    const T sc = (T)G.inv_sqrt_n;
    V2<T>* O = wf_any_out<T>(G.px, A, Bf);
    auto stpix = [&](int, int o, int Ns, V2<T>* v, auto rt) {
      constexpr int R = decltype(rt)::value, U = R > 8 ? (R + 1) / 2 : R;  // at most eight values' loads at once
#pragma unroll
      for (int q0 = 0; q0 < R; q0 += U) {
        T xa[U], xb[U], fa[U], fb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (q0 + u >= R) break;
          const int e = (int)WF_CHK(o + (q0 + u) * Ns, nx);
          const uint8_t ka = __ldg(ma + e), kb = __ldg(mb + e);
          const T na = __ldg(wa + e), nb = __ldg(wb + e);
          xa[u] = ka ? na : (T)0;
          xb[u] = kb ? nb * onb : (T)0;
          fa[u] = d ? __ldg(da + e) : (T)0;
          fb[u] = d ? __ldg(db + e) : (T)0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (q0 + u >= R) break;
          const V2<T> x = v[q0 + u];
          const T r0 = fa[u] - x.x * sc, r1 = fb[u] - x.y * sc, w0 = xa[u] * r0, w1 = xb[u] * r1;
          acc.add({r0, r1}, {w0, w1});
          O[at(0, o + (q0 + u) * Ns)] = mk<T>(w0, w1);
        }
      }
    };
    wf_any_fft<T, +1, TEAM>(G.px, 0, A, Bf, tw, at, ld0, stpix);
    sync();
    // forward: the first pass reads O, so the buffers swap roles where O is A
    V2<T>* A2 = O == A ? Bf : A;
    auto ldO = [&](int, int e) { return O[at(0, e)]; };
    V2<T>* Z = wf_any_out<T>(G.px, A2, O);
    auto stZ = [&](int, int o, int Ns, V2<T>* v, auto rt) {
#pragma unroll
      for (int q = 0; q < decltype(rt)::value; ++q) Z[at(0, o + q * Ns)] = v[q];
    };
    wf_any_fft<T, -1, TEAM>(G.px, 0, A2, O, tw, at, ldO, stZ);
    sync();
    for (int k = lane; k < h1; k += team) {
      const V2<T> zk = Z[at(0, k)], zm = Z[at(0, k == 0 ? 0 : nx - k)];
      rowa[k] = mk<T>((T)0.5 * (zk.x + zm.x), (T)0.5 * (zk.y - zm.y));
      if (two) rowb[k] = mk<T>((T)0.5 * (zk.y + zm.y), (T)0.5 * (zm.x - zk.x));
    }
  }
  const double tot = wf_rg_block_sum(acc.get(), blockDim.x >> 5);
  if (threadIdx.x == 0) dpart[(size_t)b * G.nrb + blockIdx.x] = tot;
}

// Forward column stage: the forward DFT along y of a tile of the row stage's
// output, then per mode g = 2 (s - sqrt(P) R(k)^T G / sqrt(N)) and the prior
// sum of |s|^2 with the half-plane weights (1 on column 0 and on the Nyquist
// column of an even nx, 2 elsewhere).  ppart[b gx + tile] = the tile's sum.  One
// channel takes the last pass's values as they come; two meet in shared memory.
template <typename T, int C>
__global__ void __launch_bounds__(WF_ANY_THREADS, sizeof(T) == 4 ? 2 : 0)
k_any_colfwd(const __grid_constant__ WfAnyGeo G, const V2<T>* s, WfAnyTab<T> tab, const V2<T>* scr, V2<T>* grad,
             double* ppart) {
  extern __shared__ __align__(16) unsigned char wf_smem[];
  const int b = blockIdx.y, kx0 = blockIdx.x * G.tc, ny = G.ny, h1 = G.h1, tc = G.tc, lgS = G.lgtc + (C == 2), S = 1 << lgS;
  V2<T>* tw = (V2<T>*)wf_smem;
  V2<T>* A = tw + ny;
  V2<T>* Bf = A + S * ny;
  const size_t vsz = (size_t)C * ny * h1;
  const int nm = ny * h1;
  const V2<T>* in = scr + (size_t)b * vsz;
  const V2<T>* sb = s + (size_t)b * vsz;
  V2<T>* gb = grad + (size_t)b * vsz;
  for (int i = threadIdx.x; i < ny; i += blockDim.x) tw[i] = tab.twy[i];
  auto at = [&](int t, int e) { return (int)WF_CHK((e << lgS) + t, S * ny); };
  auto ld0 = [&](int t, int e) -> V2<T> {
    const int col = t & (tc - 1), c = C == 2 ? t >> G.lgtc : 0, kx = min(kx0 + col, h1 - 1);
    return __ldcg(in + WF_CHK(c * nm + e * h1 + kx, vsz));
  };
  const T sc = (T)G.inv_sqrt_n;
  // a thread's column is fixed: its stride is a multiple of the tile's width
  const int kxt = kx0 + (threadIdx.x & (tc - 1));
  const double wm = kxt >= h1 ? 0.0 : (kxt == 0 || ((G.nx % 2) == 0 && 2 * kxt == G.nx)) ? 1.0 : 2.0;
  WfAnySum<T> acc;
  if constexpr (C == 1) {
    auto stl = [&](int t, int o, int Ns, V2<T>* v, auto rt) {
      constexpr int R = decltype(rt)::value;
      const int kx = kx0 + t;
      if (kx >= h1) return;
      constexpr int U = sizeof(T) == 4 && R > 4 ? 4 : R;  // FP32: four values' loads at once, 64 registers
#pragma unroll
      for (int q0 = 0; q0 < R; q0 += U) {
        V2<T> sv[U];
        T a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (q0 + u >= R) break;
          const int m = (int)WF_CHK((o + (q0 + u) * Ns) * h1 + kx, nm);
          sv[u] = __ldg(sb + m);
          a[u] = __ldg(tab.amp + m);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (q0 + u >= R) break;
          const V2<T> g = cscale<T>(v[q0 + u], sc);
          gb[(o + (q0 + u) * Ns) * h1 + kx] = mk<T>((T)2 * (sv[u].x - a[u] * g.x), (T)2 * (sv[u].y - a[u] * g.y));
          acc.add({sv[u].x, sv[u].y}, {sv[u].x, sv[u].y});
        }
      }
    };
    wf_any_fft<T, -1, true>(G.py, lgS, A, Bf, tw, at, ld0, stl);
  } else {
    V2<T>* O = wf_any_out<T>(G.py, A, Bf);
    auto stl = [&](int t, int o, int Ns, V2<T>* v, auto rt) {
#pragma unroll
      for (int q = 0; q < decltype(rt)::value; ++q) O[at(t, o + q * Ns)] = v[q];
    };
    wf_any_fft<T, -1, true>(G.py, lgS, A, Bf, tw, at, ld0, stl);
    __syncthreads();
    for (int i = threadIdx.x; i < (ny << G.lgtc); i += blockDim.x) {
      const int col = i & (tc - 1), ky = i >> G.lgtc, kx = kx0 + col;
      if (kx >= h1) continue;
      const int m = (int)WF_CHK(ky * h1 + kx, nm);
      const V2<T> g0 = cscale<T>(O[at(col, ky)], sc), g1 = cscale<T>(O[at(tc + col, ky)], sc), r = __ldg(tab.rot + m);
      const V2<T> s0 = __ldg(sb + m), s1 = __ldg(sb + nm + m);
      const T a0 = __ldg(tab.amp + m), a1 = __ldg(tab.amp + nm + m);
      const V2<T> d0 = mk<T>(r.x * g0.x + r.y * g1.x, r.x * g0.y + r.y * g1.y);   // R^T: first row (c, s)
      const V2<T> d1 = mk<T>(r.x * g1.x - r.y * g0.x, r.x * g1.y - r.y * g0.y);   // second row (-s, c)
      gb[m] = mk<T>((T)2 * (s0.x - a0 * d0.x), (T)2 * (s0.y - a0 * d0.y));
      gb[nm + m] = mk<T>((T)2 * (s1.x - a1 * d1.x), (T)2 * (s1.y - a1 * d1.y));
      acc.add({s0.x, s0.y}, {s0.x, s0.y});
      acc.add({s1.x, s1.y}, {s1.x, s1.y});
    }
  }
  const double tot = wf_rg_block_sum(wm * acc.get(), blockDim.x >> 5);
  if (threadIdx.x == 0) ppart[(size_t)b * G.gx + blockIdx.x] = tot;
}

// chi2[b] = prior sums of the column tiles + data sums of the row blocks: each
// lane of the map's warp adds its share in index order, then the lanes pairwise.
__global__ void k_any_final(int gx, int nrb, const double* ppart, const double* dpart, double* chi2) {
  const int b = blockIdx.x;
  double v = 0.0;
  for (int i = threadIdx.x; i < gx; i += 32) v += ppart[(size_t)b * gx + i];
  for (int i = threadIdx.x; i < nrb; i += 32) v += dpart[(size_t)b * nrb + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (threadIdx.x == 0) chi2[b] = v;
}

// Passes of a transform of length L: the fewest, and among those the ones with
// the smallest largest radix, larger radices first.  False if L has a prime factor
// above 7.
static bool wf_any_plan(int L, WfAnyPlan* P) {
  static const int rad[] = {16, 15, 14, 12, 10, 9, 8, 7, 6, 5, 4, 3, 2};
  int best[WF_ANY_MAXP] = {0}, nbest = 0, cur[WF_ANY_MAXP] = {0};
  auto search = [&](auto&& self, int rest, int n, int from) -> void {
    if (rest == 1) {
      if (n > 0 && (!nbest || n < nbest || (n == nbest && cur[0] < best[0]))) {
        nbest = n;
        for (int i = 0; i < n; ++i) best[i] = cur[i];
      }
      return;
    }
    if (n == WF_ANY_MAXP || (nbest && n + 1 > nbest)) return;
    for (int i = from; i < (int)(sizeof rad / sizeof rad[0]); ++i)
      if (rest % rad[i] == 0) {
        cur[n] = rad[i];
        self(self, rest / rad[i], n + 1, i);
      }
  };
  search(search, L, 0, 0);
  if (!nbest) return false;
  P->L = L;
  P->np = nbest;
  int Ns = 1;
  auto recip = [](int d) { return d > 1 ? (unsigned)(((1ull << 32) + d - 1) / d) : 0u; };
  for (int p = 0; p < nbest; ++p) {
    P->R[p] = best[p];
    P->Ns[p] = Ns;
    P->LR[p] = L / best[p];
    P->mNs[p] = recip(Ns);
    Ns *= best[p];
  }
  return true;
}

// Shared memory of the column and row kernels: two blocks an SM where two fit
// (113 KB each), else one.
template <typename T> static size_t any_col_smem(const WfAnyGeo& G, int tc) {
  return ((size_t)G.ny + 2 * (size_t)G.C * tc * G.ny) * sizeof(V2<T>);
}
template <typename T> static size_t any_row_smem(const WfAnyGeo& G) {
  return ((size_t)G.nx + 2 * (size_t)G.roww * G.rpitch) * sizeof(V2<T>);
}
// Butterflies of a transform's widest pass, and the threads for n of them.
static int any_butterflies(const WfAnyPlan& P) {
  int n = 0;
  for (int p = 0; p < P.np; ++p) n = P.LR[p] > n ? P.LR[p] : n;
  return n;
}
static int any_threads(int n, int most) { return n >= most ? most : (n + 31) / 32 * 32; }
// Row blocks of one pair each up to this many pairs an SM (us a call, a warp a pair -> a
// block a pair: FP32 12 x 1024 115 -> 106, 600 x 1000 145 -> 128; FP64 60 x 875 210 -> 136,
// 600 x 1000 300 -> 232); at 480 pairs, 375 values, FP64, it was slower: 191 -> 206.
#define WF_ANY_TEAM 2
#define WF_ANY_SMEM2 (113u << 10)
#define WF_ANY_SMEM1 (226u << 10)
template <typename T> static void any_tiles(WfAnyGeo& G) {
  // columns: the widest of 16 .. 1 (FP64 8 .. 1) with two blocks an SM; a tile under
  // 64 bytes takes the whole SM for one block instead
  const int wide = sizeof(T) == 4 ? 16 : 8, fair = sizeof(T) == 4 ? 8 : 4;
  int tc = wide;
  while (tc > 1 && any_col_smem<T>(G, tc) > WF_ANY_SMEM2) tc /= 2;
  while (tc < fair && any_col_smem<T>(G, 2 * tc) <= WF_ANY_SMEM1) tc *= 2;
  while (tc > 1 && tc / 2 >= G.h1) tc /= 2;
  while (tc > 1 && (long long)G.B * ((G.h1 + tc - 1) / tc) < 2 * WF_SMS) tc /= 2;  // a small batch: more tiles
  G.tc = tc;
  G.lgtc = 0;
  while ((1 << G.lgtc) < tc) ++G.lgtc;
  G.gx = (G.h1 + tc - 1) / tc;
  G.rpitch = G.nx + G.nx / 16 + 1;
  const int pairs = (G.C * G.ny + 1) / 2;
  G.roww = sizeof(T) == 4 ? WF_ANY_ROWW : WF_ANY_ROWW / 2;  // FP64: four warps of 255 registers, two blocks
  if (G.roww > pairs) G.roww = pairs;
  while (G.roww > 1 && any_row_smem<T>(G) > WF_ANY_SMEM2) --G.roww;
  while (G.roww > 1 && (long long)G.B * ((pairs + G.roww - 1) / G.roww) < 2 * WF_SMS) G.roww = (G.roww + 1) / 2;
  G.nrb = (pairs + G.roww - 1) / G.roww;
  G.roww_t = 32 * G.roww;
  if (G.roww == 1 && (long long)G.B * pairs <= WF_ANY_TEAM * WF_SMS && any_butterflies(G.px) > 32)
    G.roww_t = any_threads(any_butterflies(G.px), WF_ANY_TEAMT);
}

static size_t any_up(size_t x) { return (x + 255) & ~(size_t)255; }

template <typename T>
static cudaError_t wf_any_launch(const WfAnyGeo& G, const void* d, const uint8_t* mask, const void* Ninv,
                                 const void* P, const void* s, void* grad, double* chi2, void* scr, char* work,
                                 cudaStream_t st) {
  const size_t nm = (size_t)G.ny * G.h1;
  WfAnyTab<T> tab;
  double* ppart = (double*)work;
  work += any_up(sizeof(double) * (size_t)G.B * G.gx);
  double* dpart = (double*)work;
  work += any_up(sizeof(double) * (size_t)G.B * G.nrb);
  tab.twy = (V2<T>*)work;
  work += any_up(sizeof(V2<T>) * G.ny);
  tab.twx = (V2<T>*)work;
  work += any_up(sizeof(V2<T>) * G.nx);
  tab.amp = (T*)work;
  work += any_up(sizeof(T) * G.C * nm);
  tab.rot = (V2<T>*)work;
  const size_t smc = any_col_smem<T>(G, G.tc), smr = any_row_smem<T>(G);
  auto ki = G.C == 1 ? k_any_colinv<T, 1> : k_any_colinv<T, 2>;
  auto kf = G.C == 1 ? k_any_colfwd<T, 1> : k_any_colfwd<T, 2>;
  cudaError_t e = cudaFuncSetAttribute(ki, cudaFuncAttributeMaxDynamicSharedMemorySize, WF_ANY_SMEM1);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, WF_ANY_SMEM1);
  auto kr = G.roww_t > 32 * G.roww ? k_any_row<T, true> : k_any_row<T, false>;
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kr, cudaFuncAttributeMaxDynamicSharedMemorySize, WF_ANY_SMEM1);
  if (e != cudaSuccess) return e;
  // FP32 threads take 64 registers, so two blocks of 512 fit; FP64 ones up to 128.  No
  // more than the widest pass has butterflies: every further warp adds the FP64 steps of
  // its sums (one map of 12 x 1024, tiles of one column: 134 -> 115 us a call).
  const int tcol = any_threads(any_butterflies(G.py) * G.C * G.tc, sizeof(T) == 4 || smc > WF_ANY_SMEM2 ? 512 : 256);
  size_t pb = (G.C * nm + 255) / 256;
  if (pb > 8 * WF_SMS) pb = 8 * WF_SMS;
  k_any_prep<T><<<(unsigned)pb, 256, 0, st>>>(G, (const T*)P, tab);
  ki<<<dim3(G.gx, G.B), tcol, smc, st>>>(G, (const V2<T>*)s, tab, (V2<T>*)scr);
  kr<<<dim3(G.nrb, G.B), G.roww_t, smr, st>>>(G, (const T*)d, mask, (const T*)Ninv, tab.twx, (V2<T>*)scr, dpart);
  kf<<<dim3(G.gx, G.B), tcol, smc, st>>>(G, (const V2<T>*)s, tab, (const V2<T>*)scr, (V2<T>*)grad, ppart);
  k_any_final<<<G.B, 32, 0, st>>>(G.gx, G.nrb, ppart, dpart, chi2);
  return cudaGetLastError();
}
template <typename T> static size_t any_work_bytes(const WfAnyGeo& G) {
  const size_t nm = (size_t)G.ny * G.h1;
  return any_up(sizeof(double) * (size_t)G.B * G.gx) + any_up(sizeof(double) * (size_t)G.B * G.nrb) +
         any_up(sizeof(V2<T>) * G.ny) + any_up(sizeof(V2<T>) * G.nx) + any_up(sizeof(T) * G.C * nm) +
         (G.C == 2 ? any_up(sizeof(V2<T>) * nm) : 0);
}

extern "C" wf_status wf_eval_any(wf_handle* h, int B, int C, int ny, int nx, int precision, const void* d,
                                 const uint8_t* mask, const void* Ninv, const void* P, const void* s, void* grad,
                                 double* chi2, void* stream) {
  if (!h || !mask || !Ninv || !P || !s || !grad || !chi2) return wf_fail(WF_EINVAL, "wf_eval_any: null argument");
  if (s == grad) return wf_fail(WF_EINVAL, "wf_eval_any: s and grad must not alias");
  if (B < 1 || (C != 1 && C != 2)) return wf_fail(WF_EINVAL, "wf_eval_any: need count >= 1 and C = 1 or 2");
  if (precision != WF_FP64 && precision != WF_MIXED) return wf_fail(WF_EINVAL, "wf_eval_any: unknown precision");
  WfAnyGeo G = {};
  if (ny < 2 || nx < 2 || ny > WF_ANY_MAXN || nx > WF_ANY_MAXN || !wf_any_plan(ny, &G.py) || !wf_any_plan(nx, &G.px))
    return wf_fail(WF_EINVAL, "wf_eval_any: ny = %d, nx = %d: each side must be in [2, %d] with no prime factor "
                   "above 7", ny, nx, WF_ANY_MAXN);
  G.B = B;
  G.C = C;
  G.ny = ny;
  G.nx = nx;
  G.h1 = nx / 2 + 1;
  G.inv_sqrt_n = 1.0 / sqrt((double)ny * (double)nx);
  const bool f64 = precision == WF_FP64;
  if (f64) any_tiles<double>(G);
  else any_tiles<float>(G);
  const size_t vsz = (size_t)C * ny * G.h1;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;  // the call synchronises: refuse before it allocates
  cudaError_t ce = cudaStreamIsCapturing((cudaStream_t)stream, &cap);
  if (ce == cudaSuccess && cap != cudaStreamCaptureStatusNone) ce = cudaErrorStreamCaptureUnsupported;
  if (ce != cudaSuccess) return wf_cuda_fail(ce, "wf_eval_any");
  void* scr = nullptr;
  char* work = nullptr;
  wf_status rs = wf_alloc(h, &scr, (size_t)B * vsz * (f64 ? sizeof(double2) : sizeof(float2)), "wf_eval_any scratch");
  if (rs == WF_OK)
    rs = wf_alloc(h, (void**)&work, f64 ? any_work_bytes<double>(G) : any_work_bytes<float>(G), "wf_eval_any tables and sums");
  if (rs == WF_OK) {
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = f64 ? wf_any_launch<double>(G, d, mask, Ninv, P, s, grad, chi2, scr, work, st)
                        : wf_any_launch<float>(G, d, mask, Ninv, P, s, grad, chi2, scr, work, st);
    const cudaError_t es = cudaStreamSynchronize(st);  // also after a failed launch: earlier ones may still run
    if (e == cudaSuccess) e = es;
    if (e != cudaSuccess) rs = wf_cuda_fail(e, "wf_eval_any");
  }
  if (rs == WF_OK) {
    wf_free_idle(h, work);
    wf_free_idle(h, scr);
  } else {
    void* ptrs[] = {work, scr};
    wf_free_all(h, ptrs, 2);
  }
  return rs;
}

WF_DBG_READER(any)
