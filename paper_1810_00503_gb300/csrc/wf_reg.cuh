// Register-resident two-pass transforms: the FFT stages of every operator pass.
//
// A sequence of N values is held by G = N / NV threads, NV values each: thread
// g holds the elements g + G m, m < NV.  N = R1 R2, both at most NV, so a
// transform is two passes of in-register DFTs with one exchange through shared
// memory between them (the three-pass forms of wf_fft.cuh and wf_fft_pp.cuh
// exchange twice and keep their values in shared memory):
//   pass 1: butterfly j (< N / R1) takes the elements j + r N / R1, gives
//           y_q(j), multiplied by exp(+-2 pi i q j / N);
//   exchange: y_q(j) is written at (q, j) and read back by butterfly q;
//   pass 2: butterfly q (< R1) takes y_q(j) over j < R2 and gives the
//           elements q + R1 r.
// Both passes read and write the same elements per thread (g + G m), so a
// thread's inputs and outputs stay in its registers, a second transform needs
// no exchange before it, and the thread that holds element e has a partner
// (G - g) that holds N - e at index NV - 1 - m: the reflections of a real
// transform are exchanges between fixed lanes.
//
// What bounds them: HBM and L2.  A value costs about 30 FP instructions per
// transform (radix-32 passes: 12.1 each with fused butterflies, 4 for the
// twiddle) and six shared- or global-memory instructions, all at immediate
// offsets: the exchange's pitches are compile-time constants padded so that
// every access of a warp is conflict-free.  The three-pass forms executed 97,
// 222 and 217 instructions a value (inverse column, row, forward column stage),
// 45% of them integer work, and met 2 to 8 block barriers.
//
// Measured, 120 maps of 1024^2, FP32 (bytes at 6.78 TB/s: 0.15, 0.30 and 0.22
// ms): inverse column stage 0.466 -> 0.248 ms, row stage with data 0.533 -> 0.330
// ms, forward column stage 0.626 -> 0.393 ms; the objective pass 1.637 -> 1.00
// ms.  53 E/B maps of 512^2, Hessian-vector product: 0.448 -> 0.272 ms.
#pragma once
#include "wf_ops.cuh"

// Passes of a length-N transform: a thread holds the larger radix (32 values, 64
// registers in FP32, at 512 and 1024).
template <int N> struct WfReg;
template <> struct WfReg<1024> { static constexpr int NV = 32, RA = 32, RB = 32; };
template <> struct WfReg<512> { static constexpr int NV = 32, RA = 16, RB = 32; };
template <> struct WfReg<256> { static constexpr int NV = 16, RA = 16, RB = 16; };
template <> struct WfReg<128> { static constexpr int NV = 16, RA = 8, RB = 16; };
template <> struct WfReg<64> { static constexpr int NV = 8, RA = 8, RB = 8; };
template <> struct WfReg<32> { static constexpr int NV = 8, RA = 4, RB = 8; };
template <> struct WfReg<16> { static constexpr int NV = 4, RA = 4, RB = 4; };
template <> struct WfReg<8> { static constexpr int NV = 4, RA = 2, RB = 4; };
// Passes in the working type: R1, R2 of the column and the forward row transforms,
// I1, I2 of the inverse row transform (the radices the other way round).  At the
// lengths of wf_rg_split a thread holds half as many values and pass 2 splits its
// butterflies, of twice as many, over two threads (wf_rg_read), for 20 operations
// more per pair of values: twice the warps.
//   FP64, 32, 128 and 512: a warp's FP64 instruction holds its unit for 64 cycles,
//     so a pass over few maps takes as long as one warp's instructions.  Objective
//     pass of one map, us: 32^2 45 -> 32, 128^2 87 -> 60, 512^2 186 -> 111; 40 maps
//     of 512^2 1650 -> 1597.  (Where the units are busy the extra work shows: 100
//     maps of 128^2 224 -> 257.)  8 gained nothing; 64, 256 and 1024 have no such split.
//   FP32 columns of 512: 80 registers and three blocks an SM against 128 and two.
//     Hessian-vector product of 53 E/B maps 302 -> 272 us, 20 E/B solves 2.42 ->
//     2.08 ms, objective of one map 44 -> 38 us, of 256 maps 515 -> 521.
// FP32 rows of 512 and the shorter FP32 lengths were slower split (300 maps of 32 x
// 512: 58.6 against 70.1 us; 300 E/B maps of 128^2: 98.7 against 105.4).
template <typename T, int N, bool ROW> struct WfRegT {
  static constexpr bool SPLIT = wf_rg_split(N, sizeof(T) == 8, ROW);
  static constexpr int NV = SPLIT ? WfReg<N>::NV / 2 : WfReg<N>::NV;
  static constexpr int R1 = SPLIT ? NV : WfReg<N>::RB, R2 = SPLIT ? 2 * NV : WfReg<N>::RA;
  static constexpr int I1 = SPLIT ? R1 : R2, I2 = SPLIT ? R2 : R1;
};

__device__ __forceinline__ float wf_fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double wf_fma(double a, double b, double c) { return fma(a, b, c); }

// Butterfly (a, b) <- (a + w b, a - w b), w = exp(DIR 2 pi i Q / 32), in six
// fused multiply-adds: w b = s (t b.x - b.y, t b.y + b.x) with t = cot, or the
// tangent form c (b.x - t b.y, b.y + t b.x), whichever has the smaller factor
// outside.  Four multiplications and additions would take eight.  The factor's
// rounding is a gain error common to every transform, which adds up in the
// modes of small k; the smaller factor carries less of it (FP32, 512^2 Hessian-
// vector product against FP64: 5.5e-8 this way, 1.3e-7 with the larger factor
// outside, 6.8e-8 for radix-8 passes of plain multiplications).
template <typename T, int DIR, int Q>
__device__ __forceinline__ void wf_bf(V2<T>& a, V2<T>& b) {
  static_assert(Q >= 0 && Q < 16, "root index");
  if constexpr (Q == 0) {
    const V2<T> t = b;
    b = csub<T>(a, t);
    a = cadd<T>(a, t);
  } else if constexpr (Q == 8) {
    const V2<T> t = (DIR > 0) ? mul_i<T>(b) : mk<T>(b.y, -b.x);
    b = csub<T>(a, t);
    a = cadd<T>(a, t);
  } else {
    constexpr double cs[16] = {1.0,   WF_C16,  WF_C1,  WF_C3,  WF_R2,  WF_S3,  WF_S1,  WF_S16,
                               0.0,  -WF_S16, -WF_S1, -WF_S3, -WF_R2, -WF_C3, -WF_C1, -WF_C16};
    constexpr double sn[16] = {0.0,  WF_S16, WF_S1, WF_S3, WF_R2, WF_C3, WF_C1, WF_C16,
                               1.0,  WF_C16, WF_C1, WF_C3, WF_R2, WF_S3, WF_S1, WF_S16};
    constexpr double c = cs[Q], s = DIR * sn[Q];
    constexpr bool tangent = (c < 0 ? -c : c) < (s < 0 ? -s : s);
    if constexpr (tangent) {
      constexpr double t = s / c;
      const T t1 = wf_fma((T)-t, b.y, b.x), t2 = wf_fma((T)t, b.x, b.y);
      b = mk<T>(wf_fma((T)-c, t1, a.x), wf_fma((T)-c, t2, a.y));
      a = mk<T>(wf_fma((T)c, t1, a.x), wf_fma((T)c, t2, a.y));
    } else {
      constexpr double t = (Q == 4) ? (double)DIR : (Q == 12) ? -(double)DIR : c / s;
      const T t1 = wf_fma((T)t, b.x, -b.y), t2 = wf_fma((T)t, b.y, b.x);
      b = mk<T>(wf_fma((T)-s, t1, a.x), wf_fma((T)-s, t2, a.y));
      a = mk<T>(wf_fma((T)s, t1, a.x), wf_fma((T)s, t2, a.y));
    }
  }
}

template <typename T, int R, int DIR, int LEN, int Q>
__device__ __forceinline__ void wf_rg_q(V2<T>* v) {
  if constexpr (Q < LEN / 2) {
#pragma unroll
    for (int s = 0; s < R; s += LEN) wf_bf<T, DIR, Q * (32 / LEN)>(v[s + Q], v[s + Q + LEN / 2]);
    wf_rg_q<T, R, DIR, LEN, Q + 1>(v);
  }
}
template <typename T, int R, int DIR, int LEN>
__device__ __forceinline__ void wf_rg_stages(V2<T>* v) {
  if constexpr (LEN <= R) {
    wf_rg_q<T, R, DIR, LEN, 0>(v);
    wf_rg_stages<T, R, DIR, LEN * 2>(v);
  }
}
// Length-R DFT of v[0], v[STEP], .., natural order in and out.
template <typename T, int R, int DIR, int STEP>
__device__ __forceinline__ void wf_rg_dft(V2<T>* v) {
  V2<T> u[R];
#pragma unroll
  for (int r = 0; r < R; ++r) u[bitrev_c(r, Log2R<R>::v)] = v[r * STEP];
  wf_rg_stages<T, R, DIR, 2>(u);
#pragma unroll
  for (int r = 0; r < R; ++r) v[r * STEP] = u[r];
}

// Exchange layout of S interleaved sequences (sequence fastest): (q, j) of
// sequence t at q P + j S + t.  A write of one q covers consecutive places; a
// read of one j strides over q by P, padded so that the 16 (FP64: 8) accesses
// served together fall in different banks.
template <typename T, int S, int R2> struct WfXch {
  static constexpr int BK = sizeof(T) == 4 ? 16 : 8;
  static constexpr int PITCH = R2 * S + (S < BK ? S : 0);
};

// Pass 1, twiddles, write of the exchange.  tw: roots exp(-2 pi i k / N) laid out
// [q][j] (wf_rg_stage_tw).  sm: this sequence's place of the exchange buffer.
template <typename T, int N, int R1, int R2, int NV, int DIR, int PITCH, int S>
__device__ __forceinline__ void wf_rg_pass1(V2<T>* v, V2<T>* sm, const V2<T>* tw, int g) {
  constexpr int G = N / NV, NB = NV / R1;
  static_assert(R1 * R2 == N && NV % R1 == 0 && (NV % R2 == 0 || R2 == 2 * NV), "passes");
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    wf_rg_dft<T, R1, DIR, NB>(v + i);
    const int j = g + G * i;
    sm[j * S] = v[i];
#pragma unroll
    for (int q = 1; q < R1; ++q) sm[q * PITCH + j * S] = cmul<T>(v[i + q * NB], twid<T, DIR>(tw, q * R2 + j));
  }
}
// Place of the exchange that a thread's value m of pass 2 is read from (a split
// butterfly's two threads read both halves: this thread's half).
template <int N, int R2, int NV, int PITCH, int S>
__device__ __forceinline__ int wf_rg_place(int g, int m) {
  if constexpr (R2 > NV) {
    constexpr int R1 = N / R2;
    return (g & (R1 - 1)) * PITCH + (m + NV * (g / R1)) * S;
  } else {
    constexpr int G = N / NV, NB = NV / R2;
    return (g + G * (m % NB)) * PITCH + (m / NB) * S;
  }
}
// Read of the exchange.  A butterfly of R2 = 2 NV values is split over the threads
// q and q + R1: they form y_j + y_{j+NV} and (y_j - y_{j+NV}) w^j, whose length-NV
// transforms are the outputs of even and odd index, elements g + G k of both.
template <typename T, int N, int R1, int R2, int NV, int DIR, int PITCH, int S>
__device__ __forceinline__ void wf_rg_read(V2<T>* v, const V2<T>* sm, const V2<T>* tw, int g) {
  if constexpr (R2 > NV) {
    const V2<T>* y = sm + (g & (R1 - 1)) * PITCH;
    if (g < R1) {
#pragma unroll
      for (int m = 0; m < NV; ++m) v[m] = cadd<T>(y[m * S], y[(m + NV) * S]);
    } else {  // w^j = the pass-1 root of (q, j) = (j, R1)
#pragma unroll
      for (int m = 0; m < NV; ++m) v[m] = cmul<T>(csub<T>(y[m * S], y[(m + NV) * S]), twid<T, DIR>(tw, m * R2 + R1));
    }
  } else {
#pragma unroll
    for (int m = 0; m < NV; ++m) v[m] = sm[wf_rg_place<N, R2, NV, PITCH, S>(g, m)];
  }
}
template <typename T, int N, int R1, int R2, int NV, int DIR>
__device__ __forceinline__ void wf_rg_pass2(V2<T>* v) {
  if constexpr (R2 > NV) {  // half a butterfly (wf_rg_read has done its first step)
    wf_rg_dft<T, NV, DIR, 1>(v);
  } else {
    constexpr int NB = NV / R2;
#pragma unroll
    for (int i = 0; i < NB; ++i) wf_rg_dft<T, R2, DIR, NB>(v + i);
  }
}

// Pass-1 twiddles of a length-N transform with radices R1, R2 into shared
// memory: tw[q R2 + j] = exp(-2 pi i q j / N), from the table of WF_NT-th roots.
template <typename T, int N, int R2>
__device__ __forceinline__ void wf_rg_stage_tw(V2<T>* s_tw, const void* tw_, int threads) {
  const V2<T>* roots = (const V2<T>*)tw_;
  for (int i = threadIdx.x; i < N; i += threads) {
    const int q = i / R2, j = i - q * R2;
    s_tw[i] = roots[(q * j) * (WF_NT / N)];
  }
}

// 8- or 16-byte asynchronous copy global -> shared.
template <typename T>
__device__ __forceinline__ void wf_cp_async(V2<T>* dst, const V2<T>* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(V2<T>) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void wf_cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Kaiser-Squires cosine and sine (wf_ks) of column kx at signed row frequency ky.
template <typename T>
__device__ __forceinline__ void wf_rg_ks(int kx, int ky, const WfGeo& g, T& c, T& s) {
  const int qx = kx * g.ksx, qy = ky * g.ksy;
  const int k2 = qx * qx + qy * qy;
  const T inv = (T)1 / (T)(k2 == 0 ? 1 : k2);
  c = k2 == 0 ? (T)1 : (T)(qx * qx - qy * qy) * inv;
  s = (kx == g.h || 2 * ky == -g.n) ? (T)0 : (T)(2 * qx * qy) * inv;
}

// Blocks per SM asked of the compiler for `threads` threads of NV values: FP32
// threads get 128 registers (32 values) or 80 (fewer), FP64 ones up to 255.
template <typename T, int NV> __host__ __device__ constexpr int wf_rg_minb(int threads) {
  return sizeof(T) == 8 ? 1 : (NV == 32 ? 512 : 768) / threads;
}

// ---------------------------------------------------------------------------
// Column stages.  A block holds TC packed columns of C channels: thread
// (sequence t = c TC + column, g), t fastest, rows g + G m.  A tile wider than
// the map (h < TC) has idle columns: they load the last one and store nothing.
// ---------------------------------------------------------------------------
template <typename T, int C, int N, int TC> struct WfRegCol {
  static constexpr int NV = WfRegT<T, N, false>::NV, G = N / NV, S = C * TC, THREADS = S * G;
  static constexpr int R1 = WfRegT<T, N, false>::R1, R2 = WfRegT<T, N, false>::R2;
  static constexpr int PITCH = WfXch<T, S, R2>::PITCH;
  static constexpr size_t XCH = (size_t)R1 * PITCH;            // values of the exchange buffer
  static constexpr size_t SMEM = (XCH + N) * sizeof(V2<T>);    // and the twiddles
};


// Per-mode operator on this thread's rows of its column, every lane of the warp
// (with two channels their values are exchanged between lanes TC apart):
//   forward (ADJ = false): v <- R(k) diag(amp) v     (step A1)
//   adjoint (ADJ = true):  v <- diag(amp) R(k)^T v   (step A5)
// skip: a thread of the packed column 0, whose values pass unchanged (they are
// done by wf_rg_mode0).
template <typename T, int C, int N, int TC, bool ADJ>
__device__ __forceinline__ void wf_rg_modes(V2<T>* v, int c, int g, int kx, bool skip, const WfGeo& geo, const T* sp,
                                            T extra) {
  typedef WfRegCol<T, C, N, TC> K;
  constexpr int U = K::NV < 8 ? K::NV : 8;
  const unsigned p0 = (unsigned)(c * N + g) * (unsigned)(geo.h + 1) + (unsigned)kx;
  const unsigned step = (unsigned)K::G * (unsigned)(geo.h + 1);
#pragma unroll
  for (int m0 = 0; m0 < K::NV; m0 += U) {
    T a[U];
#pragma unroll
    for (int u = 0; u < U; ++u) a[u] = sp[WF_CHK(p0 + (m0 + u) * step, (unsigned)(C * N) * (geo.h + 1))];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int m = m0 + u;
      const T am = skip ? (T)1 : a[u] * extra;
      if constexpr (C == 1) {
        v[m] = cscale<T>(v[m], am);
      } else {
        const int j = g + K::G * m;
        T cs, sn;
        wf_rg_ks<T>(kx, m < K::NV / 2 ? j : j - N, geo, cs, sn);
        if (skip) cs = (T)1, sn = (T)0;
        V2<T> own = v[m];
        if constexpr (!ADJ) own = cscale<T>(own, am);
        const V2<T> oth = mk<T>(__shfl_xor_sync(0xffffffffu, own.x, TC), __shfl_xor_sync(0xffffffffu, own.y, TC));
        const T so = ((c == 0) != ADJ) ? -sn : sn;
        V2<T> r = mk<T>(cs * own.x + so * oth.x, cs * own.y + so * oth.y);
        if constexpr (ADJ) r = cscale<T>(r, am);
        v[m] = r;
      }
    }
  }
}

// Operator at the packed column 0: X0 (kx = 0) and Xh (kx = nx/2) of row j,
// packed again.  The rotation's sine is 0 there, so the channels do not mix.
template <typename T, int C>
__device__ __forceinline__ V2<T> wf_rg_mode0(V2<T> X0, V2<T> Xh, int c, int j, const WfGeo& g, const T* sp, T extra) {
  const unsigned o = (unsigned)(c * g.n + j) * (unsigned)(g.h + 1);
  T a0 = sp[o] * extra, ah = sp[o + g.h] * extra;
  if constexpr (C == 2) {
    T cs, sn;
    wf_ks<T>(0, j, g, cs, sn);
    a0 *= cs;
    wf_ks<T>(g.h, j, g, cs, sn);
    ah *= cs;
  }
  return wf_pack0<T>(cscale<T>(X0, a0), cscale<T>(Xh, ah));
}

// Column 0 of a forward transform (the first tile's only; every thread of the
// block calls it): rows j and ny - j are unpacked together through shared
// memory, the operator applied and the column packed again.
template <typename T, int C, int N, int TC>
__device__ __forceinline__ void wf_rg_col0(V2<T>* v, V2<T>* xch, bool col0, int c, int g, const WfGeo& geo,
                                           const T* sp, T extra) {
  typedef WfRegCol<T, C, N, TC> K;
  __syncthreads();  // the exchange buffer has been read
  if (col0) {
#pragma unroll
    for (int m = 0; m < K::NV; ++m) xch[c * N + g + K::G * m] = v[m];
  }
  __syncthreads();
  if (col0) {
#pragma unroll
    for (int m = 0; m < K::NV; ++m) {
      const int j = g + K::G * m;
      V2<T> X0, Xh;
      wf_unpack0<T>(v[m], xch[c * N + ((N - j) & (N - 1))], X0, Xh);
      v[m] = wf_rg_mode0<T, C>(X0, Xh, c, j, geo, sp, extra);
    }
  }
}

// Pass 1 and the exchange of a block's column transforms (pass 2 is the
// caller's: it needs no shared memory).  s_tw is staged before.
template <typename T, int C, int N, int TC, int DIR>
__device__ __forceinline__ void wf_rg_cols(V2<T>* v, V2<T>* xch_t, const V2<T>* s_tw, int g) {
  typedef WfRegCol<T, C, N, TC> K;
  __syncthreads();  // twiddles staged; an earlier exchange has been read
  wf_rg_pass1<T, N, K::R1, K::R2, K::NV, DIR, K::PITCH, K::S>(v, xch_t, s_tw, g);
  __syncthreads();
  wf_rg_read<T, N, K::R1, K::R2, K::NV, DIR, K::PITCH, K::S>(v, xch_t, s_tw, g);
}

// Inverse column stage of the tile at packed column kx0: spectrum (packed or
// standard layout) -> R sqrt(P)/n -> inverse FFT along y -> scratch (packed).
template <typename T, int C, int IN, int N, int TC>
__device__ __forceinline__ void wf_rg_colinv(const WfGeo& geo, const V2<T>* src, const T* sp, V2<T>* scr,
                                             const void* tw_, int kx0) {
  typedef WfRegCol<T, C, N, TC> K;
  extern __shared__ __align__(16) unsigned char wf_smem[];
  V2<T>* xch = (V2<T>*)wf_smem;
  V2<T>* s_tw = xch + K::XCH;
  const int t = threadIdx.x & (K::S - 1), g = threadIdx.x / K::S;
  const int c = t / TC, h = geo.h, kxt = kx0 + (t & (TC - 1)), kx = kxt < h ? kxt : h - 1;
  const unsigned pitch = IN == WF_IN_PK ? h : h + 1;
  const bool col0 = kx == 0;
  V2<T> v[K::NV];
  const unsigned o0 = (unsigned)(c * N + g) * pitch + (unsigned)kx, step = K::G * pitch;
#pragma unroll
  for (int m = 0; m < K::NV; ++m) v[m] = __ldcg(src + WF_CHK(o0 + m * step, C * N * pitch));
  wf_rg_stage_tw<T, N, K::R2>(s_tw, tw_, K::THREADS);
  if (kx0 == 0 && col0) {
#pragma unroll
    for (int m = 0; m < K::NV; ++m) {
      const int j = g + K::G * m;
      V2<T> X0 = v[m], Xh;
      if constexpr (IN == WF_IN_STD) Xh = src[WF_CHK(o0 + m * step + h, C * N * pitch)];
      else wf_unpack0<T>(v[m], src[WF_CHK((unsigned)(c * N + ((N - j) & (N - 1))) * pitch, C * N * pitch)], X0, Xh);
      v[m] = wf_rg_mode0<T, C>(X0, Xh, c, j, geo, sp, (T)1);
    }
  }
  wf_rg_modes<T, C, N, TC, false>(v, c, g, kx, col0, geo, sp, (T)1);
  wf_rg_cols<T, C, N, TC, +1>(v, xch + t, s_tw, g);
  wf_rg_pass2<T, N, K::R1, K::R2, K::NV, +1>(v);
  const unsigned d0 = (unsigned)(c * N + g) * h + (unsigned)kx, dstep = K::G * h;
#pragma unroll
  for (int m = 0; m < K::NV; ++m)
    if (kxt < h) scr[WF_CHK(d0 + m * dstep, C * N * h)] = v[m];
}

// Data synthesis: the row r2c of a white field z (scratch) -> forward FFT along
// y -> 1/sqrt(ny nx) (unitary U z) -> R sqrt(P)/n -> inverse FFT along y -> scratch.
template <typename T, int C, int N, int TC>
__device__ __forceinline__ void wf_rg_colsim(const WfGeo& geo, const T* sp, V2<T>* scr, const void* tw_, int kx0) {
  typedef WfRegCol<T, C, N, TC> K;
  extern __shared__ __align__(16) unsigned char wf_smem[];
  V2<T>* xch = (V2<T>*)wf_smem;
  V2<T>* s_tw = xch + K::XCH;
  const int t = threadIdx.x & (K::S - 1), g = threadIdx.x / K::S;
  const int c = t / TC, h = geo.h, kxt = kx0 + (t & (TC - 1)), kx = kxt < h ? kxt : h - 1;
  const bool col0 = kx == 0;
  V2<T> v[K::NV];
  const unsigned d0 = (unsigned)(c * N + g) * h + (unsigned)kx, dstep = K::G * h;
#pragma unroll
  for (int m = 0; m < K::NV; ++m) v[m] = __ldcg(scr + WF_CHK(d0 + m * dstep, C * N * h));
  wf_rg_stage_tw<T, N, K::R2>(s_tw, tw_, K::THREADS);
  wf_rg_cols<T, C, N, TC, -1>(v, xch + t, s_tw, g);
  wf_rg_pass2<T, N, K::R1, K::R2, K::NV, -1>(v);
  const T unit = (T)(1.0 / sqrt((double)N * (double)geo.nx));
  if (kx0 == 0) wf_rg_col0<T, C, N, TC>(v, xch, col0, c, g, geo, sp, unit);
  wf_rg_modes<T, C, N, TC, false>(v, c, g, kx, col0, geo, sp, unit);
  wf_rg_cols<T, C, N, TC, +1>(v, xch + t, s_tw, g);
  wf_rg_pass2<T, N, K::R1, K::R2, K::NV, +1>(v);
#pragma unroll
  for (int m = 0; m < K::NV; ++m)
    if (kxt < h) scr[WF_CHK(d0 + m * dstep, C * N * h)] = v[m];
}

// Forward column stage up to the adjoint: scratch tile -> forward FFT along y ->
// sqrt(P) R^T / n, in v.  aux (packed or standard rows of `pitch` values): the
// epilogue's vector; its values are copied asynchronously into the exchange
// places this thread has finished reading, while pass 2 runs
// (wf_rg_aux reads them).
template <typename T, int C, int N, int TC>
__device__ __forceinline__ void wf_rg_colfwd_front(V2<T>* v, const WfGeo& geo, const V2<T>* scr, const T* sp,
                                                   const V2<T>* aux, unsigned pitch, const void* tw_, int kx0, int kx,
                                                   int t, int g) {
  typedef WfRegCol<T, C, N, TC> K;
  extern __shared__ __align__(16) unsigned char wf_smem[];
  V2<T>* xch = (V2<T>*)wf_smem;
  V2<T>* s_tw = xch + K::XCH;
  const int c = t / TC, h = geo.h;
  const bool col0 = kx == 0;
  const unsigned d0 = (unsigned)(c * N + g) * h + (unsigned)kx, dstep = K::G * h;
#pragma unroll
  for (int m = 0; m < K::NV; ++m) v[m] = __ldcg(scr + WF_CHK(d0 + m * dstep, C * N * h));
  wf_rg_stage_tw<T, N, K::R2>(s_tw, tw_, K::THREADS);
  wf_rg_cols<T, C, N, TC, -1>(v, xch + t, s_tw, g);
  const unsigned a0 = (unsigned)(c * N + g) * pitch + (unsigned)kx, astep = K::G * pitch;
  auto fetch = [&]() {
    if constexpr (K::R2 > K::NV) __syncthreads();  // two threads read a value
    else __syncwarp();
#pragma unroll
    for (int m = 0; m < K::NV; ++m)
      wf_cp_async<T>(xch + t + wf_rg_place<N, K::R2, K::NV, K::PITCH, K::S>(g, m),
                     aux + WF_CHK(a0 + m * astep, C * N * pitch));
  };
  if (kx0 != 0) fetch();
  wf_rg_pass2<T, N, K::R1, K::R2, K::NV, -1>(v);
  if (kx0 == 0) {
    wf_rg_col0<T, C, N, TC>(v, xch, col0, c, g, geo, sp, (T)1);
    __syncthreads();  // column 0's rows have been read
    fetch();
  }
  wf_rg_modes<T, C, N, TC, true>(v, c, g, kx, col0, geo, sp, (T)1);
  wf_cp_async_wait();
}
template <typename T, int C, int N, int TC>
__device__ __forceinline__ V2<T> wf_rg_aux(int t, int g, int m) {
  typedef WfRegCol<T, C, N, TC> K;
  extern __shared__ __align__(16) unsigned char wf_smem[];
  return ((V2<T>*)wf_smem)[t + wf_rg_place<N, K::R2, K::NV, K::PITCH, K::S>(g, m)];
}

// Sum over the block's first `warps` warps (the others have left) of one double
// per thread; valid in thread 0.
__device__ __forceinline__ double wf_rg_block_sum(double v, int warps) {
  __shared__ double red[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < warps; ++i) r += red[i];
  return r;
}

// Forward column stage of the objective: out = 2 (src - a), the prior partial
// sum |src|^2 and |out|^2 (half-plane weights) to slot `bx` of part_b.
template <typename T, int C, int IN, int N, int TC>
__device__ __forceinline__ void wf_rg_colfwd(const WfGeo& geo, const V2<T>* src, const T* sp, const V2<T>* scr,
                                             V2<T>* dst, double* part_b, const void* tw_, int kx0, int bx) {
  typedef WfRegCol<T, C, N, TC> K;
  const int t = threadIdx.x & (K::S - 1), g = threadIdx.x / K::S;
  const int c = t / TC, h = geo.h, kxt = kx0 + (t & (TC - 1)), kx = kxt < h ? kxt : h - 1;
  const bool ok = kxt < h;
  const unsigned pitch = IN == WF_IN_PK ? h : h + 1;
  V2<T> v[K::NV];
  wf_rg_colfwd_front<T, C, N, TC>(v, geo, scr, sp, src, pitch, tw_, kx0, kx, t, g);
  const unsigned o0 = (unsigned)(c * N + g) * pitch + (unsigned)kx, step = K::G * pitch;
  const bool split = IN == WF_IN_STD && kxt == 0;  // kx = 0 and kx = nx/2 stored separately
  const T wk = !ok ? (T)0 : kx == 0 ? (T)1 : (T)2;
  constexpr int A16 = K::NV < 16 ? K::NV : 16;
  double prior = 0.0, out2 = 0.0;
#pragma unroll
  for (int m0 = 0; m0 < K::NV; m0 += A16) {  // 16 terms in the working type, then FP64
    WfAcc<T> a1 = 0, a2 = 0;
#pragma unroll
    for (int m = m0; m < m0 + A16; ++m) {
      V2<T> sv = wf_rg_aux<T, C, N, TC>(t, g, m);
      if (split) sv = wf_pack0<T>(sv, src[WF_CHK(o0 + m * step + h, C * N * pitch)]);
      const V2<T> o = mk<T>((T)2 * (sv.x - v[m].x), (T)2 * (sv.y - v[m].y));
      a1 += sv.x * sv.x + sv.y * sv.y;
      a2 += o.x * o.x + o.y * o.y;
      if (split) v[m] = o;
      else if (ok) dst[WF_CHK(o0 + m * step, C * N * pitch)] = o;
    }
    prior += (double)(wk * a1);
    out2 += (double)(wk * a2);
  }
  if (IN == WF_IN_STD && kx0 == 0) {  // unpack column 0 of the output
    extern __shared__ __align__(16) unsigned char wf_smem[];
    V2<T>* xch = (V2<T>*)wf_smem;
    __syncthreads();
    if (split) {
#pragma unroll
      for (int m = 0; m < K::NV; ++m) xch[c * N + g + K::G * m] = v[m];
    }
    __syncthreads();
    if (split) {
#pragma unroll
      for (int m = 0; m < K::NV; ++m) {
        const int j = g + K::G * m;
        V2<T> X0, Xh;
        wf_unpack0<T>(v[m], xch[c * N + ((N - j) & (N - 1))], X0, Xh);
        dst[WF_CHK(o0 + m * step, C * N * pitch)] = X0;
        dst[WF_CHK(o0 + m * step + h, C * N * pitch)] = Xh;
      }
    }
  }
  const double s1 = wf_rg_block_sum(prior, K::THREADS / 32);
  if (threadIdx.x == 0) part_b[(size_t)WF_SLOT_PRIOR * geo.maxblk + bx] = s1;
  const double s2 = wf_rg_block_sum(out2, K::THREADS / 32);
  if (threadIdx.x == 0) part_b[(size_t)WF_SLOT_OUT2 * geo.maxblk + bx] = s2;
}

// Forward column stage of the Hessian-vector product: q = 2 (p - a), and <q,q>,
// <p,q>, <p,p>, <g,q>, <g,p> (half-plane weights) to slot `bx` of part_b.
template <typename T, int C, int N, int TC>
__device__ __forceinline__ void wf_rg_lb_colfwd(const WfGeo& geo, const V2<T>* Pn, const V2<T>* gv, V2<T>* Qn,
                                                const T* sp, const V2<T>* scr, double* part_b, const void* tw_,
                                                int kx0, int bx) {
  typedef WfRegCol<T, C, N, TC> K;
  const int t = threadIdx.x & (K::S - 1), g = threadIdx.x / K::S;
  const int c = t / TC, h = geo.h, kxt = kx0 + (t & (TC - 1)), kx = kxt < h ? kxt : h - 1;
  const bool ok = kxt < h;
  V2<T> v[K::NV];
  wf_rg_colfwd_front<T, C, N, TC>(v, geo, scr, sp, Pn, h, tw_, kx0, kx, t, g);
  const unsigned o0 = (unsigned)(c * N + g) * h + (unsigned)kx, step = K::G * h;
  const double wk = !ok ? 0.0 : kx == 0 ? 1.0 : 2.0;
  double d[5] = {0, 0, 0, 0, 0};
  constexpr int U = K::NV < 8 ? K::NV : 8, A16 = K::NV < 16 ? K::NV : 16;
#pragma unroll
  for (int m0 = 0; m0 < K::NV; m0 += A16) {  // 16 terms in the working type, then FP64
    WfAcc<T> qq = 0, pq = 0, pp = 0, gq = 0, gp = 0;
#pragma unroll
    for (int m1 = m0; m1 < m0 + A16; m1 += U) {
      V2<T> gl[U];
#pragma unroll
      for (int u = 0; u < U; ++u) gl[u] = __ldcg(gv + WF_CHK(o0 + (m1 + u) * step, C * N * h));
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int m = m1 + u;
        const V2<T> p = wf_rg_aux<T, C, N, TC>(t, g, m);
        const V2<T> q = mk<T>((T)2 * (p.x - v[m].x), (T)2 * (p.y - v[m].y));
        if (ok) Qn[WF_CHK(o0 + m * step, C * N * h)] = q;
        qq += q.x * q.x + q.y * q.y;
        pq += p.x * q.x + p.y * q.y;
        pp += p.x * p.x + p.y * p.y;
        gq += gl[u].x * q.x + gl[u].y * q.y;
        gp += gl[u].x * p.x + gl[u].y * p.y;
      }
    }
    d[0] += wk * (double)qq;
    d[1] += wk * (double)pq;
    d[2] += wk * (double)pp;
    d[3] += wk * (double)gq;
    d[4] += wk * (double)gp;
  }
  constexpr int NW = K::THREADS / 32;
  __shared__ double red[5 * NW];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    double x = d[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) red[i * NW + (threadIdx.x >> 5)] = x;
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    const int slot[5] = {WF_SLOT_QQ, WF_SLOT_PQ, WF_SLOT_PP, WF_SLOT_GQN, WF_SLOT_GPN};
    double x = 0.0;
    for (int i = 0; i < NW; ++i) x += red[threadIdx.x * NW + i];
    part_b[(size_t)slot[threadIdx.x] * geo.maxblk + bx] = x;
  }
}

// ---------------------------------------------------------------------------
// Row stage.  Two rows a, b of one channel are one complex sequence a + i b of
// length nx: its transform carries both real transforms, A[k] = (Z[k] + conj
// Z[nx-k]) / 2 and B[k] = -i (Z[k] - conj Z[nx-k]) / 2, with no roots beyond the
// passes' own.  A warp takes 32 / G pairs of rows (lane = sequence, then g) and
// meets no barrier but its own: load the packed rows, c2r, the pixel step on the
// values in registers, r2c from there, store.
// ---------------------------------------------------------------------------
template <typename T, int NX> struct WfRegRow {
  static constexpr int NV = WfRegT<T, NX, true>::NV, G = NX / NV, SEQ = 32 / G;
  static constexpr int I1 = WfRegT<T, NX, true>::I1, I2 = WfRegT<T, NX, true>::I2, F1 = WfRegT<T, NX, true>::R1, F2 = WfRegT<T, NX, true>::R2;
  static constexpr int PI = WfXch<T, 1, I2>::PITCH, PF = WfXch<T, 1, F2>::PITCH;  // inverse, forward
  static constexpr int XI = I1 * PI, XF = F1 * PF, XM = XI > XF ? XI : XF;
  // a sequence's exchange places; the sequences of a half-warp sit G values apart
  // modulo 16
  static constexpr int XCH = G >= 16 ? XM : (XM + 15) / 16 * 16 + G;
  static constexpr int NTW = I1 == F1 ? NX : 2 * NX;  // twiddles of both directions
  static constexpr size_t smem(int warps) { return ((size_t)warps * SEQ * XCH + NTW) * sizeof(V2<T>); }
};

template <typename T, int NX, int DIR>
__device__ __forceinline__ void wf_rg_row_fft(V2<T>* v, V2<T>* xch, const V2<T>* s_tw, int g) {
  typedef WfRegRow<T, NX> K;
  __syncwarp();  // an earlier exchange has been read
  if constexpr (DIR > 0) {
    wf_rg_pass1<T, NX, K::I1, K::I2, K::NV, DIR, K::PI, 1>(v, xch, s_tw, g);
    __syncwarp();
    wf_rg_read<T, NX, K::I1, K::I2, K::NV, DIR, K::PI, 1>(v, xch, s_tw, g);
    wf_rg_pass2<T, NX, K::I1, K::I2, K::NV, DIR>(v);
  } else {
    const V2<T>* tw = s_tw + (K::I1 == K::F1 ? 0 : NX);
    wf_rg_pass1<T, NX, K::F1, K::F2, K::NV, DIR, K::PF, 1>(v, xch, tw, g);
    __syncwarp();
    wf_rg_read<T, NX, K::F1, K::F2, K::NV, DIR, K::PF, 1>(v, xch, tw, g);
    wf_rg_pass2<T, NX, K::F1, K::F2, K::NV, DIR>(v);
  }
}

//   MODE DATA / NODATA: c2r, r = d - x (or -x), wr = w r, data partial sum
//     r.wr, r2c of wr, store packed rows back to scratch.
//   MODE SIGNAL: c2r, write x to out (pixel layout).
//   MODE SIM: c2r, out = (w > 0) ? x + aux : 0 (aux = noise).
//   MODE RFFT: r2c of the pixel rows of aux (a white field), store to scratch.
// Row block rb of map b, on the block's first `warps` warps; d, w, aux, out: whole
// arrays.
template <typename T, int MODE, int NX>
__device__ __forceinline__ void wf_rg_row(const WfGeo& geo, V2<T>* scratch, const T* d, const T* w, const T* aux,
                                          T* out, double* part, const void* tw_, int b, int rb, int warps) {
  typedef WfRegRow<T, NX> K;
  constexpr int h = NX / 2, NV = K::NV, G = K::G;
  extern __shared__ __align__(16) unsigned char wf_smem[];
  V2<T>* s_tw = (V2<T>*)wf_smem;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, g = lane & (G - 1), t = lane / G;
  V2<T>* xch = s_tw + K::NTW + (wid * K::SEQ + t) * K::XCH;
  const int rows = geo.C * geo.n;
  const int rt = 2 * ((rb * warps + wid) * K::SEQ + t), nth = 32 * warps;
  const bool ok = rt < rows;     // a sequence beyond the map computes on the first rows and stores nothing
  const int r0 = ok ? rt : 0;    // this sequence's rows r0, r0 + 1
  V2<T>* sc = scratch + ((size_t)b * rows + r0) * h;
  const size_t poff = ((size_t)b * rows + r0) * NX;
  const int part_lane = (lane & ~(G - 1)) | ((G - g) & (G - 1));  // holds the reflections nx - e
  constexpr unsigned FULL = 0xffffffffu;
  V2<T> v[NV];
  if constexpr (MODE == WF_ROW_RFFT) {
    const T* za = aux + poff;
#pragma unroll
    for (int m = 0; m < NV; ++m) {
      const unsigned e = g + G * m;
      v[m] = mk<T>(__ldcg(za + WF_CHK(e, NX)), __ldcg(za + NX + e));
    }
  } else {
    // Z[k] = A[k] + i B[k] and its reflection Z[nx-k] = conj A[k] + i conj B[k],
    // which the partner lane holds at index NV - 1 - m (lane 0, its own partner:
    // at NV - m; there k = 0 and k = nx/2 are the packed real pairs)
    V2<T> s[NV / 2];
    V2<T> ny0 = mk<T>((T)0, (T)0);
#pragma unroll
    for (int m = 0; m < NV / 2; ++m) {
      const unsigned e = g + G * m;
      const V2<T> A = __ldcg(sc + WF_CHK(e, h)), B = __ldcg(sc + h + e);
      v[m] = mk<T>(A.x - B.y, A.y + B.x);
      s[m] = mk<T>(A.x + B.y, B.x - A.y);
      if (m == 0 && g == 0) {
        v[0] = mk<T>(A.x, B.x);
        ny0 = mk<T>(A.y, B.y);
      }
    }
#pragma unroll
    for (int m = 0; m < NV / 2; ++m) {
      const V2<T> nx_ = m + 1 < NV / 2 ? s[m + 1 < NV / 2 ? m + 1 : m] : ny0;
      const V2<T> snd = g == 0 ? nx_ : s[m];
      v[NV - 1 - m] = mk<T>(__shfl_sync(FULL, snd.x, part_lane), __shfl_sync(FULL, snd.y, part_lane));
    }
  }
  {
    const V2<T>* roots = (const V2<T>*)tw_;
    if constexpr (MODE != WF_ROW_RFFT) {
      for (int i = threadIdx.x; i < NX; i += nth) s_tw[i] = roots[((i / K::I2) * (i % K::I2)) * (WF_NT / NX)];
    }
    if constexpr (K::I1 != K::F1 && (MODE == WF_ROW_RFFT || MODE == WF_ROW_DATA || MODE == WF_ROW_NODATA)) {
      for (int i = threadIdx.x; i < NX; i += nth)
        s_tw[NX + i] = roots[((i / K::F2) * (i % K::F2)) * (WF_NT / NX)];
    } else if constexpr (MODE == WF_ROW_RFFT) {
      for (int i = threadIdx.x; i < NX; i += nth) s_tw[i] = roots[((i / K::F2) * (i % K::F2)) * (WF_NT / NX)];
    }
  }
  if constexpr (MODE == WF_ROW_DATA || MODE == WF_ROW_NODATA || MODE == WF_ROW_SIM) {
    // the pixel step reads these after the c2r: start them towards L2 (the
    // sequence's two rows, one request per 128-byte line)
    constexpr int LINES = 2 * NX * (int)sizeof(T) / 128;
    const char* wp = (const char*)(w + poff);
    const char* dp = (const char*)((MODE == WF_ROW_SIM ? aux : d) + poff);
#pragma unroll
    for (int l = 0; l < LINES; l += G) {
      if (l + g < LINES) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(wp + (l + g) * 128));
        if (MODE != WF_ROW_NODATA) asm volatile("prefetch.global.L2 [%0];" ::"l"(dp + (l + g) * 128));
      }
    }
  }
  __syncthreads();  // twiddles staged
  double acc = 0.0;
  if constexpr (MODE != WF_ROW_RFFT) {
    wf_rg_row_fft<T, NX, +1>(v, xch, s_tw, g);
    // v[m] = pixels e = g + G m of the two rows
    if constexpr (MODE == WF_ROW_SIGNAL) {
      T* o = out + poff;
#pragma unroll
      for (int m = 0; m < NV; ++m) {
        if (ok) {
          o[WF_CHK(g + G * m, NX)] = v[m].x;
          o[NX + g + G * m] = v[m].y;
        }
      }
      return;
    } else if constexpr (MODE == WF_ROW_SIM) {
      T* o = out + poff;
      const T *wp = w + poff, *np = aux + poff;
      constexpr int U = NV < 8 ? NV : 8;
#pragma unroll
      for (int m0 = 0; m0 < NV; m0 += U) {
        T wa[U], wb[U], na[U], nb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const unsigned e = WF_CHK(g + G * (m0 + u), NX);
          wa[u] = __ldcg(wp + e);
          wb[u] = __ldcg(wp + NX + e);
          na[u] = __ldcg(np + e);
          nb[u] = __ldcg(np + NX + e);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const unsigned e = g + G * (m0 + u);
          if (ok) {
            o[e] = wa[u] > (T)0 ? v[m0 + u].x + na[u] : (T)0;
            o[NX + e] = wb[u] > (T)0 ? v[m0 + u].y + nb[u] : (T)0;
          }
        }
      }
      return;
    } else {
      const T *wp = w + poff, *dp = MODE == WF_ROW_DATA ? d + poff : nullptr;
      constexpr int U = NV < 8 ? NV : 8, A16 = NV < 16 ? NV : 16;
#pragma unroll
      for (int m0 = 0; m0 < NV; m0 += A16) {
        WfAcc<T> a16 = 0;  // 32 terms in the working type, then FP64
#pragma unroll
        for (int m1 = m0; m1 < m0 + A16; m1 += U) {
          T wa[U], wb[U], da[U], db[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const unsigned e = WF_CHK(g + G * (m1 + u), NX);
            wa[u] = __ldcg(wp + e);
            wb[u] = __ldcg(wp + NX + e);
            if constexpr (MODE == WF_ROW_DATA) {
              da[u] = __ldcg(dp + e);
              db[u] = __ldcg(dp + NX + e);
            }
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const V2<T> x = v[m1 + u];
            V2<T> r;
            if constexpr (MODE == WF_ROW_DATA) r = mk<T>(da[u] - x.x, db[u] - x.y);
            else r = mk<T>(-x.x, -x.y);
            const V2<T> wr = mk<T>(wa[u] * r.x, wb[u] * r.y);
            a16 += r.x * wr.x + r.y * wr.y;
            v[m1 + u] = wr;
          }
        }
        if (ok) acc += (double)a16;
      }
    }
  }
  wf_rg_row_fft<T, NX, -1>(v, xch, s_tw, g);
#pragma unroll
  for (int m = 0; m < NV / 2; ++m) {
    const V2<T> own0 = m == 0 ? v[0] : v[(NV - m) & (NV - 1)];
    const V2<T> snd = g == 0 ? own0 : v[NV - 1 - m];
    const V2<T> zm = mk<T>(__shfl_sync(FULL, snd.x, part_lane), __shfl_sync(FULL, snd.y, part_lane)), zk = v[m];
    V2<T> A = mk<T>((T)0.5 * (zk.x + zm.x), (T)0.5 * (zk.y - zm.y));
    V2<T> B = mk<T>((T)0.5 * (zk.y + zm.y), (T)0.5 * (zm.x - zk.x));
    if (m == 0 && g == 0) {
      A = mk<T>(v[0].x, v[NV / 2].x);
      B = mk<T>(v[0].y, v[NV / 2].y);
    }
    const unsigned e = WF_CHK(g + G * m, h);
    if (ok) {
      sc[e] = A;
      sc[h + e] = B;
    }
  }
  if constexpr (MODE == WF_ROW_DATA || MODE == WF_ROW_NODATA) {
    const double s = wf_rg_block_sum(acc, warps);
    if (threadIdx.x == 0) part[((size_t)b * WF_NSLOT + WF_SLOT_DATA) * geo.maxblk + rb] = s;
  }
}

// ---------------------------------------------------------------------------
// The stages of the L-BFGS iteration on the direction P[next] of map bm, for a
// block at column tile (row block) bx of its problem's own grid.
// ---------------------------------------------------------------------------
template <typename T, int C, int N, int TC>
__device__ __forceinline__ void wf_rg_lb_colinv_map(const WfGeo& g, const WfBufs& b, const WfLbBufs& lb, int bm, int bx) {
  const WfLbMap* M = lb.st + bm;
  if (!M->active) return;
  const size_t vsz = (size_t)C * N * g.h;
  wf_rg_colinv<T, C, WF_IN_PK, N, TC>(g, (const V2<T>*)lb.ring + ((size_t)M->next * b.B + bm) * vsz,
                                      (const T*)b.sp + (size_t)bm * b.sp_stride, (V2<T>*)b.scratch + (size_t)bm * vsz,
                                      b.tw, bx * TC);
}
template <typename T, int NX>
__device__ __forceinline__ void wf_rg_lb_row_map(const WfGeo& g, const WfBufs& b, const WfLbBufs& lb, int bm, int bx) {
  if (!lb.st[bm].active) return;
  wf_rg_row<T, WF_ROW_NODATA, NX>(g, (V2<T>*)b.scratch, nullptr, (const T*)b.w, nullptr, nullptr, b.part, b.tw, bm, bx,
                                  g.RB / wf_rg_rows(NX, sizeof(T) == 8));
}
template <typename T, int C, int N, int TC>
__device__ __forceinline__ void wf_rg_lb_colfwd_map(const WfGeo& g, const WfBufs& b, const WfLbBufs& lb, int bm, int bx) {
  const WfLbMap* M = lb.st + bm;
  if (!M->active) return;
  const size_t vsz = (size_t)C * N * g.h;
  const int nx = M->next;
  V2<T>* ring = (V2<T>*)lb.ring;
  wf_rg_lb_colfwd<T, C, N, TC>(g, ring + ((size_t)nx * b.B + bm) * vsz, (const V2<T>*)lb.g + (size_t)bm * vsz,
                               ring + ((size_t)(lb.m + nx) * b.B + bm) * vsz, (const T*)b.sp + (size_t)bm * b.sp_stride,
                               (const V2<T>*)b.scratch + (size_t)bm * vsz,
                               b.part + (size_t)bm * WF_NSLOT * g.maxblk, b.tw, bx * TC, bx);
}
