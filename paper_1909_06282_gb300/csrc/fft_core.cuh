// In-CTA FFT engine for the 2LPT pass kernels (sm_103a).
//
// A pencil of N complex points is owned by TPP = N / RMAX threads; thread t of
// the pencil holds RMAX values in registers.  The first and the last stage use
// the same radix R0, so the input of the first stage and the output of the last
// stage sit at the same element n = elem(t, j) = t + (j / R0) TPP + (j mod R0) N/R0
// (= t + j TPP when R0 = RMAX): prologue/epilogue code sees natural-order
// indices without an extra shared memory round trip.  Stages follow the Stockham autosort formulation (radix-R
// butterflies on inputs b + r N/R, twiddle W_{Ns R}^{r (b mod Ns)}, outputs at
// (b / Ns) Ns R + b mod Ns + r Ns) with one shared-memory exchange between
// consecutive stages.  Twiddles come from a table exp(-2 pi i m / N) computed in
// FP64 on the host and rounded once to FP32, stored per stage in the order the lanes of a
// pencil read them (twiddle_exponent).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "packed.cuh"

namespace lpt2 {

// ---------------------------------------------------------------- complex ops
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// The radix butterflies add with padd / psub (packed.cuh).  A packed add has the arithmetic rate
// of two scalar adds but takes one issue slot instead of two (measured: 0.53 against 1.04
// instructions per cycle and scheduler), and the passes with several transforms per field are
// bound by issue and shared-memory slots: z_source at 512^3 1141 -> 1071 us, z_final 636 -> 617.
// (Its aligned register pairs cost x_delta and x_source at 512 spills of 132 and 68 bytes.)  Products stay scalar: a packed complex product needs swapped or
// doubled operands, whose moves cost what it saves.
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 mul_i(float2 a) { return make_float2(-a.y, a.x); }    // i a
__device__ __forceinline__ float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }   // -i a

// ------------------------------------------------------------ radix schedules
// V = 0: radix sequences with the same radix first and last (so that stage-0 input and
// last-stage output share one element pattern); every radix divides RMAX.
// V = 1 (32, 128, 512): twice the values per thread and two stages, so one shared-memory exchange
// per transform instead of two, half the twiddle loads and half the threads per pencil.  fft()
// brings the outputs back into the input's pattern (a renaming of registers).
// Rule (YCfg, XCfg): passes that hold one array of values, where the registers allow it.  The z
// passes, x_delta, the adjoint x passes and the summing y passes keep V = 0: 16-8 in all passes at
// 128 costs the batch of 96 mixed grids 16.7 ms a call, 8-2-8 in all 15.5, by the rule 15.4.
template <int N, int V = 0> struct Cfg;
template <> struct Cfg<96>   { static constexpr int NS = 3, RMAX = 12; static __host__ __device__ constexpr int rad(int s) { return s == 1 ? 6 : 4; } };
template <> struct Cfg<192>  { static constexpr int NS = 3, RMAX = 12; static __host__ __device__ constexpr int rad(int s) { return s == 1 ? 12 : 4; } };
template <> struct Cfg<16>   { static constexpr int NS = 2, RMAX = 4;  static __host__ __device__ constexpr int rad(int s) { return 4; } };
template <> struct Cfg<32>   { static constexpr int NS = 3, RMAX = 4;  static __host__ __device__ constexpr int rad(int s) { return s == 1 ? 2 : 4; } };
template <> struct Cfg<64>   { static constexpr int NS = 2, RMAX = 8;  static __host__ __device__ constexpr int rad(int s) { return 8; } };
template <> struct Cfg<128>  { static constexpr int NS = 3, RMAX = 8;  static __host__ __device__ constexpr int rad(int s) { return s == 1 ? 2 : 8; } };
template <> struct Cfg<256>  { static constexpr int NS = 2, RMAX = 16; static __host__ __device__ constexpr int rad(int s) { return 16; } };
#ifndef LPT2_R512
#define LPT2_R512 16   // N = 512: radix 16-2-16 (16 values per thread) or 8-8-8 (8 values)
#endif
template <> struct Cfg<512>  { static constexpr int NS = 3, RMAX = LPT2_R512;
  static __host__ __device__ constexpr int rad(int s) { return LPT2_R512 == 8 ? 8 : (s == 1 ? 2 : 16); } };
template <> struct Cfg<1024> { static constexpr int NS = 3, RMAX = 16; static __host__ __device__ constexpr int rad(int s) { return s == 1 ? 4 : 16; } };
template <> struct Cfg<128, 1> { static constexpr int NS = 2, RMAX = 16; static __host__ __device__ constexpr int rad(int s) { return s == 0 ? 16 : 8; } };
template <> struct Cfg<32, 1>  { static constexpr int NS = 2, RMAX = 8;  static __host__ __device__ constexpr int rad(int s) { return s == 0 ? 8 : 4; } };
template <> struct Cfg<512, 1> { static constexpr int NS = 2, RMAX = 32; static __host__ __device__ constexpr int rad(int s) { return s == 0 ? 32 : 16; } };

// element index held in register slot j by lane t (first-stage input, and output of fft())
template <int N, int V = 0> __host__ __device__ __forceinline__ constexpr int elem(int t, int j) {
  constexpr int R0 = Cfg<N, V>::rad(0), TPP = N / Cfg<N, V>::RMAX;
  return t + (j / R0) * TPP + (j % R0) * (N / R0);
}

// i mod N for i in [0, 2N) (periodic neighbour index)
template <int N> __host__ __device__ __forceinline__ constexpr int wrap_idx(int i) {
  return ((N & (N - 1)) == 0) ? (i & (N - 1)) : (i >= N ? i - N : i);
}

template <int N, int V = 0> __host__ __device__ constexpr int ns_before(int s) {
  int p = 1;
  for (int i = 0; i < s; ++i) p *= Cfg<N, V>::rad(i);
  return p;
}

// Twiddle table: entry i, NS <= i < NS R of a stage with radix R after NS = ns_before points,
// is exp(-2 pi i r j / (NS R)) for r = i / NS, j = i mod NS (a thread's butterfly b reads j = b
// mod NS): the lanes of a pencil, whose b are consecutive, read consecutive entries.  The
// stages' ranges tile [ns_before(1), N).  A table in the order of the exponent puts the lanes
// r entries apart, up to 16 to a bank (512^3: z_source 1257 -> 1141 us, z_adj_source 2223 ->
// 1907 us, x_pkadj 438 -> 367 us by this order).  Returns the exponent m of exp(-2 pi i m / N).
template <int N> __host__ __device__ constexpr int twiddle_exponent(int i) {
  for (int s = 1; s < Cfg<N>::NS; ++s) {
    const int ns = ns_before<N>(s), R = Cfg<N>::rad(s);
    if (i >= ns && i < ns * R) return (i / ns) * (i % ns) * (N / (ns * R));
  }
  return 0;
}

// Whether schedule V reads its twiddles from that table, which is laid out for V = 0: each of its
// twiddled stages starts after the same number of points, with the same radix, as one of V = 0's
// (32-16 as 16-2-16, 16-8 as 8-2-8, 8-4 as 4-2-4; 32-16 not as 8-8-8).
template <int N, int V> __host__ __device__ constexpr bool shares_twiddles() {
  for (int s = 1; s < Cfg<N, V>::NS; ++s) {
    bool found = false;
    for (int u = 1; u < Cfg<N>::NS; ++u)
      found = found || (ns_before<N>(u) == ns_before<N, V>(s) && Cfg<N>::rad(u) == Cfg<N, V>::rad(s));
    if (!found) return false;
  }
  return true;
}
// Whether N has a two-stage schedule V = 1 that a pass may take.
template <int N> __host__ __device__ constexpr bool two_stage() {
  if constexpr (N == 32 || N == 128 || N == 512) return shares_twiddles<N, 1>();
  else return false;
}

// ------------------------------------------------------- in-register DFTs
// Forward: X[k] = sum_n x[n] exp(-2 pi i n k / R); INV flips the sign.
// Roots of unity of order 96 (covers R = 2, 3, 4, 6, 8, 12, 16, 32): cos / sin of
// 2 pi j / 96, from cos(j * 3.75 deg) for j = 0..24.
__device__ __forceinline__ float2 root96(int j, bool inv) {
  // j in [0, 96); value exp(-+ 2 pi i j / 96)
  const float c[25] = {1.0f, 0.99785892323860348f, 0.99144486137381038f,
                       0.98078528040323043f, 0.96592582628906831f, 0.94693012949510569f,
                       0.92387953251128674f, 0.89687274153268826f, 0.86602540378443871f,
                       0.83146961230254524f, 0.79335334029123517f, 0.75183980747897738f,
                       0.70710678118654757f, 0.65934581510006884f, 0.60876142900872066f,
                       0.55557023301960229f, 0.5f, 0.44228869021900125f,
                       0.38268343236508984f, 0.3214394653031617f, 0.25881904510252074f,
                       0.19509032201612833f, 0.13052619222005171f, 0.065403129230143048f,
                       0.0f};
  float cs, sn;
  const int q = j % 24, quad = j / 24;
  const float cq = c[q], sq = c[24 - q];
  switch (quad) {
    case 0: cs = cq; sn = sq; break;
    case 1: cs = -sq; sn = cq; break;
    case 2: cs = -cq; sn = -sq; break;
    default: cs = sq; sn = -cq; break;
  }
  return make_float2(cs, inv ? sn : -sn);
}

template <int R, bool INV> struct Dft;

template <bool INV> struct Dft<1, INV> { static __device__ __forceinline__ void run(float2*) {} };

template <bool INV> struct Dft<3, INV> {
  static __device__ __forceinline__ void run(float2* v) {
    const float h = 0.86602540378443865f;   // sin(60 deg)
    const float2 a = v[0], s = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const float2 t = make_float2(a.x - 0.5f * s.x, a.y - 0.5f * s.y);
    const float2 u = INV ? cscale(mul_i(d), h) : cscale(mul_mi(d), h);
    v[0] = cadd(a, s);
    v[1] = cadd(t, u);
    v[2] = csub(t, u);
  }
};

template <bool INV> struct Dft<2, INV> {
  static __device__ __forceinline__ void run(float2* v) {
    const float2 a = v[0];
    const float2 b = v[1];
    v[0] = padd(a, b);
    v[1] = psub(a, b);
  }
};

template <int R, bool INV> struct Dft {   // even R: split into even and odd halves
  static_assert(R % 2 == 0 && 96 % R == 0, "radix must be 2, 4, 6, 8, 12, 16, 24 or 32 here");
  static __device__ __forceinline__ void run(float2* v) {
    float2 e[R / 2], o[R / 2];
#pragma unroll
    for (int i = 0; i < R / 2; ++i) { e[i] = v[2 * i]; o[i] = v[2 * i + 1]; }
    Dft<R / 2, INV>::run(e);
    Dft<R / 2, INV>::run(o);
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      const int j = k * (96 / R);   // exponent in units of 2 pi / 96
      float2 t;
      if (j == 0) t = o[k];
      else if (j == 24) t = INV ? mul_i(o[k]) : mul_mi(o[k]);
      else t = cmul(o[k], root96(j, INV));
      if (j == 24) {   // t is o with its parts swapped: scalar adds read the swap in place
        v[k] = cadd(e[k], t);
        v[k + R / 2] = csub(e[k], t);
      } else {
        v[k] = padd(e[k], t);
        v[k + R / 2] = psub(e[k], t);
      }
    }
  }
};

// Three-stage sequences R0-2-R0 with R0 values per thread: the inputs e, e + R0 TPP / 2 of a radix-2
// butterfly are the same register of threads t and t + TPP / 2.  Where those are lanes of one warp
// (partner(): the lane mask, 0 where they are not), the middle stage can run on shuffles: one exchange
// through shared memory per transform instead of two, which is what bounds the z passes (70 % of
// their cycles) and whose CTA barriers the x passes wait at.
// Rule: z passes of 32, 128 and 512 (512^3: z_source 1099 -> 1043 us, z_adj_source 1766 -> 1672) and,
// at 512, the shell sums and the adjoint x passes (x_pk 251 -> 240, x_adj_delta 833 -> 769).  Not
// where they spill more than the pass does without them (x_delta, 132 bytes a thread as it stands,
// 740 -> 863 us; x_source 702 -> 723; the summing y passes 1065 -> 1141), nor in z_final at
// 512, whose independent warps miss the instruction cache (499 -> 512).
template <int N, int V> inline constexpr bool kPaired =
    Cfg<N, V>::NS == 3 && Cfg<N, V>::rad(1) == 2 && Cfg<N, V>::RMAX == Cfg<N, V>::rad(0);

// --------------------------------------------------------- shared accessors
// Z layout: one pencil per row of N + N/16 complex (one pad slot per 16).  The row is
// private to its pencil; when the pencil's threads lie in one warp (WARP), the exchange
// between stages needs only a warp barrier.
template <bool WARP = false> struct SmemRowT {
  float2* base;
  __device__ __forceinline__ void st(int n, float2 v) const { base[n + (n >> 4)] = v; }
  __device__ __forceinline__ float2 ld(int n) const { return base[n + (n >> 4)]; }
  __device__ __forceinline__ void sync() const {
    if (WARP) __syncwarp();
    else __syncthreads();
  }
  static __host__ __device__ constexpr int words(int n) { return n + n / 16; }
  template <int N, int V> static constexpr int partner() { return WARP && kPaired<N, V> ? N / Cfg<N, V>::RMAX / 2 : 0; }
  // where element n lies between the paired stages: stores from and loads into all lanes at once
  // fall in different banks
  template <int N> static __device__ __forceinline__ int paired_slot(int n) { return n + (n >> (N == 512 ? 5 : 4)); }
};
using SmemRow = SmemRowT<false>;
// z-pass pencils of N points lie in one warp when N / RMAX <= 32 threads hold one
template <int N> inline constexpr bool kRowWarp = (N / Cfg<N>::RMAX) <= 32;
// The same row for a group of GT threads that runs on its own: a warp, or GT / 32 warps that meet
// at the CTA's named barrier `bar`.
template <int GT, bool PAIR = true> struct SmemRowG {
  float2* base;
  int bar;
  __device__ __forceinline__ void st(int n, float2 v) const { base[n + (n >> 4)] = v; }
  __device__ __forceinline__ float2 ld(int n) const { return base[n + (n >> 4)]; }
  __device__ __forceinline__ void sync() const {
    if constexpr (GT == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(GT) : "memory");
  }
  template <int N, int V> static constexpr int partner() {
    return PAIR && GT == 32 && kPaired<N, V> ? N / Cfg<N, V>::RMAX / 2 : 0;
  }
  template <int N> static __device__ __forceinline__ int paired_slot(int n) { return n + (n >> (N == 512 ? 5 : 4)); }
};
// Column layout: W pencils interleaved, element (n, w) at n * W + w (a pencil spans warps).
template <int W, bool PAIR = false> struct SmemCol {
  float2* base;   // already offset by w
  __device__ __forceinline__ void st(int n, float2 v) const { base[n * W] = v; }
  __device__ __forceinline__ float2 ld(int n) const { return base[n * W]; }
  __device__ __forceinline__ void sync() const { __syncthreads(); }
  // N = 512, W = 8: pencil_thread() puts t + 16 sixteen lanes from t
  template <int N, int V> static constexpr int partner() { return PAIR && N == 512 && W == 8 && kPaired<N, V> ? 16 : 0; }
  template <int N> static __device__ __forceinline__ int paired_slot(int n) { return (n ^ ((n >> 5) & 1)) * W; }
};
// Pencil position t of this thread in a CTA of W interleaved pencils (w = threadIdx.x % W).
template <int N, int V, int W, bool PAIR> __device__ __forceinline__ int pencil_thread() {
  if constexpr (SmemCol<W, PAIR>::template partner<N, V>() != 0) {   // lanes 0-15: t, t + 1; 16-31: t + 16, t + 17
    return (int)((threadIdx.x >> 5) << 1) + (int)((threadIdx.x >> 3) & 1) + (int)(threadIdx.x & 16);
  } else {
    return threadIdx.x / W;
  }
}

// ------------------------------------------------------------ stage engine
// Runs all stages on v (in: x[t + r TPP], out: X[t + r TPP]).  Every thread of
// the CTA (of the warp, for a warp-private row layout) must call this the same number
// of times (it contains the layout's barriers).
template <int N, bool INV, int S, int V, class SM>
__device__ __forceinline__ void fft_stages(float2 (&v)[Cfg<N, V>::RMAX], int t, const SM& sm,
                                           const float2* __restrict__ tw) {
  using C = Cfg<N, V>;
  static_assert(shares_twiddles<N, V>(), "the twiddle table has no entries in this schedule's order");
  constexpr int RMAX = C::RMAX;
  constexpr int TPP = N / RMAX;
  constexpr int R = C::rad(S);
  constexpr int NS = ns_before<N, V>(S);
  constexpr int NB = RMAX / R;
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int b = t + q * TPP;
    if (S > 0) {
      const int j = b % NS;
#pragma unroll
      for (int r = 1; r < R; ++r) {
        float2 w = tw[r * NS + j];
        if (INV) w.y = -w.y;
        v[q * R + r] = cmul(v[q * R + r], w);
      }
    }
    Dft<R, INV>::run(&v[q * R]);
  }
  if constexpr (S == 0 && SM::template partner<N, V>() != 0) {
    // radix 2 with the partner lane (its twiddles are constants of the register), then one exchange
    constexpr int M = SM::template partner<N, V>();
    const bool up = (t & (TPP / 2)) != 0;
    if (up) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], root96(r * (96 / (2 * R)), INV));
    }
    const float2 sg = pair(up ? -1.f : 1.f);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float2 o = make_float2(__shfl_xor_sync(0xffffffffu, v[r].x, M), __shfl_xor_sync(0xffffffffu, v[r].y, M));
      v[r] = pfma(v[r], sg, o);
    }
    const int d = (t & (TPP / 2 - 1)) * (2 * R) + (up ? R : 0);
#pragma unroll
    for (int r = 0; r < R; ++r) sm.base[SM::template paired_slot<N>(d + r)] = v[r];
    sm.sync();
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = sm.base[SM::template paired_slot<N>(t + r * TPP)];
    sm.sync();
    fft_stages<N, INV, S + 2, V, SM>(v, t, sm, tw);
  } else if constexpr (S + 1 < C::NS) {
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int b = t + q * TPP;
      const int d = (b / NS) * NS * R + (b % NS);
#pragma unroll
      for (int r = 0; r < R; ++r) sm.st(d + r * NS, v[q * R + r]);
    }
    sm.sync();
    constexpr int R2 = C::rad(S + 1);
#pragma unroll
    for (int q = 0; q < RMAX / R2; ++q) {
      const int b = t + q * TPP;
#pragma unroll
      for (int r = 0; r < R2; ++r) v[q * R2 + r] = sm.ld(b + r * (N / R2));
    }
    sm.sync();
    fft_stages<N, INV, S + 1, V, SM>(v, t, sm, tw);
  } else if constexpr (R != C::rad(0)) {
    // output (q, r) is element t + q TPP + r NS: back into the order of elem()
    constexpr int R0 = C::rad(0);
    float2 o[RMAX];
#pragma unroll
    for (int i = 0; i < RMAX; ++i) {
      const int m = i / R + (i % R) * (NS / TPP);          // element t + m TPP
      o[(m % (N / R0 / TPP)) * R0 + m / (N / R0 / TPP)] = v[i];
    }
#pragma unroll
    for (int i = 0; i < RMAX; ++i) v[i] = o[i];
  }
}

template <int N, bool INV, int V = 0, class SM>
__device__ __forceinline__ void fft(float2 (&v)[Cfg<N, V>::RMAX], int t, const SM& sm,
                                    const float2* __restrict__ tw) {
  fft_stages<N, INV, 0, V, SM>(v, t, sm, tw);
}

// Copy the N-entry twiddle table to shared memory (all threads participate).
__device__ __forceinline__ void load_twiddles(float2* s_tw, const float2* __restrict__ g_tw, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) s_tw[i] = g_tw[i];
}

// ---------------------------------------------------------------- k helpers
__device__ __forceinline__ int mode_of(int i, int n) { return i < (n >> 1) ? i : i - n; }

}  // namespace lpt2
