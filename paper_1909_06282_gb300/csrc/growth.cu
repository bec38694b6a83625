// FP64 set-up kernels: Eisenstein-Hu constants and sigma_8 normalisation of
// P(k), and the batched RK4 integration of the growth tables D1(k,a), D2(k,a)
// (T1 triangle by default, or another triangle of the Sec. 3 comparison) with
// their ln|f_R0| tangents.
//
// Equations (units h/Mpc, s = ln a, flat E^2 = Om a^-3 + OL):
//   D1_ss + (2 - 1.5 Om(a)) D1_s = 1.5 Om(a) mu(k,a) D1                    (Eq. d1)
//   D2_ss + (2 - 1.5 Om(a)) D2_s - 1.5 Om(a) mu(k) D2
//       = -1.5 Om(a) D1(k/sqrt2)^2 [mu(k) - B(k,a)],                     (Eq. full-d2, T1)
//   B = (2/27) 4 pi G rho (k^2/a^2) M2(a) / (Pi(k) Pi(k/sqrt2)^2),
//   mu = 1 + (k^2/a^2) / (3 Pi), Pi = k^2/a^2 + m^2, m^2 = M1/3    (Eq. mihusawicki, Sec. 2.4)
// with D2 taken with the sign that gives -3/7 D1^2 in GR, the EdS growing mode at
// a_init and D1 normalised to the GR solution at a = 1.  Tangents use
// dm^2/dln|fR0| = -m^2 and dM2/dln|fR0| = -2 M2.
// Other triangles (k1 = r k2 at angle theta between k1 and k2, |k1 + k2| = k): the
// source is -1.5 Om D1(k1) D1(k2) times the Eq. full-d2 braces
//   mu - c^2 (mu1 + mu2 - mu) + m^2/Pi [2 c^2 (mu1 + mu2 - 2) + (c/r)(mu1 - 1) + r c (mu2 - 1)]
//   - (2/27) 4piGrho (k^2/a^2) M2 / (Pi Pi1 Pi2),   c = cos theta,
// divided by sin^2 theta so that every triangle keeps the GR limit; Winther's variant
// takes D1(k)^2 with the T1 braces; the GR variant solves the D2 equation with mu = 1.
#include <math.h>

#include "passes.h"

namespace lpt2 {

static constexpr double kH0c = 1.0 / 2997.92458;   // H0 / c in h/Mpc
static constexpr int kSigmaPts = 20001;            // Simpson points in ln k on [1e-5, 1e3]
static constexpr int kPartBlocks = 64;

struct EhConst { double theta2, omh, alpha, s; };

__device__ EhConst eh_constants(const GrowthParams& p) {
  const double h = p.h, wm = p.omega_m * h * h, wb = p.omega_b * h * h, fb = p.omega_b / p.omega_m;
  const double theta = p.t_cmb / 2.7;
  EhConst c;
  c.theta2 = theta * theta;
  c.s = 44.5 * log(9.83 / wm) / sqrt(1.0 + 10.0 * pow(wb, 0.75));                 // EH Eq. 26
  c.alpha = 1.0 - 0.328 * log(431.0 * wm) * fb + 0.38 * log(22.3 * wm) * fb * fb;   // EH Eq. 31
  c.omh = p.omega_m * h;
  return c;
}

__device__ double eh_T64(const EhConst& c, double k, double h) {
  const double sk = 0.43 * k * h * c.s;
  const double gamma = c.omh * (c.alpha + (1.0 - c.alpha) / (1.0 + sk * sk * sk * sk));  // Eq. 30
  const double q = k * c.theta2 / gamma;                                                  // Eq. 28
  const double L0 = log(2.0 * 2.718281828459045 + 1.8 * q);                              // Eq. 29
  const double C0 = 14.2 + 731.0 / (1.0 + 62.5 * q);
  return L0 / (L0 + C0 * q * q);
}

__global__ void k_sigma_partial(GrowthParams p, double* part) {
  const EhConst c = eh_constants(p);
  const double lo = log(1e-5), hi = log(1e3), dl = (hi - lo) / (kSigmaPts - 1);
  double acc = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kSigmaPts; i += gridDim.x * blockDim.x) {
    const double k = exp(lo + i * dl);
    const double T = eh_T64(c, k, p.h);
    const double x = 8.0 * k;
    const double W = 3.0 * (sin(x) - x * cos(x)) / (x * x * x);
    const double f = k * k * k * pow(k, p.n_s) * T * T * W * W / (2.0 * M_PI * M_PI);
    const double w = (i == 0 || i == kSigmaPts - 1) ? 1.0 : ((i & 1) ? 4.0 : 2.0);
    acc += w * f;
  }
  __shared__ double s[256];
  s[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = s[0] * dl / 3.0;
}

__global__ void k_sigma_final(GrowthParams p, const double* part, DevCosmo* out) {
  if (threadIdx.x != 0) return;
  double s2 = 0.0;
  for (int b = 0; b < kPartBlocks; ++b) s2 += part[b];
  const EhConst c = eh_constants(p);
  DevCosmo d;
  d.sigma_sq = s2;
  d.amp = p.sigma8 * p.sigma8 / s2;
  d.sqrt_amp = (float)sqrt(d.amp);
  d.ns_half = (float)(0.5 * p.n_s);
  d.theta2 = (float)c.theta2;
  d.omh = (float)c.omh;
  d.alpha = (float)c.alpha;
  d.s043h = (float)(0.43 * c.s * p.h);
  d.lnkmin = (float)log(p.k_min);
  d.inv_dlnk = (float)((p.nk - 1) / (log(p.k_max) - log(p.k_min)));
  d.nk = p.nk;
  *out = d;
}

int cosmo_partial_blocks() { return kPartBlocks; }

cudaError_t launch_cosmo_setup(const GrowthParams& p, double* partials, DevCosmo* out, cudaStream_t s) {
  k_sigma_partial<<<kPartBlocks, 256, 0, s>>>(p, partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_sigma_final<<<1, 32, 0, s>>>(p, partials, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ growth RK4
// Background at every half step, shared by the block: 1/a^2, 1.5 Om(a),
// 2 - 1.5 Om(a), m^2(a), (2/27) 4 pi G rho M2(a).
struct Bg { double inv_a2, cc, damp, m2, bfac; };

__device__ Bg background(const GrowthParams& p, double s, bool gr) {
  const double a = exp(s);
  const double a3 = 1.0 / (a * a * a);
  const double e2 = p.omega_m * a3 + p.omega_l;
  const double om = p.omega_m * a3 / e2;
  Bg b;
  b.inv_a2 = 1.0 / (a * a);
  b.cc = 1.5 * om;
  b.damp = 2.0 - 1.5 * om;
  if (gr) {
    b.m2 = 0.0;
    b.bfac = 0.0;
  } else {
    const double x = p.omega_m * a3 + 4.0 * p.omega_l, x0 = p.omega_m + 4.0 * p.omega_l;
    const double x2 = x * x, x02 = x0 * x0;
    b.m2 = 0.5 * kH0c * kH0c * x2 * x / (p.fr0_abs * x02);
    const double M2 = 2.25 * kH0c * kH0c * x2 * x2 * x / (p.fr0_abs * p.fr0_abs * x02 * x02);
    b.bfac = (2.0 / 27.0) * 1.5 * p.omega_m * a3 * kH0c * kH0c * M2;
  }
  return b;
}

// Triangle of a D2 variant: fa, fb = (k1/k)^2, (k2/k)^2, c = cos theta, r = k1/k2.
struct D2Geo {
  double fa, fb, c, c2, inv_s2, r;
  int winther, gr2;
  int fit;   // D2 from the LCDM fit Eq. lcdm-fit with the scale-dependent D1 (no D2 equation)
};

__host__ __device__ inline D2Geo d2_geo(int variant) {
  // (r, theta in degrees) of the Sec. 3 comparison; Winther and GR use the T1 geometry
  double r = 1.0, th = 90.0;
  switch (variant) {
    case 1: th = 80.0; break;
    case 2: th = 70.0; break;
    case 3: r = 2.0; th = 80.0; break;
    case 4: r = 2.0; th = 70.0; break;
    case 7: th = 60.0; break;    // isosceles 60 deg (the text's "equilateral")
    case 8: r = 1e-3; break;     // squeezed: k1 = 1e-3 k2 at 90 deg (k1 ~ 0, k2 ~ k)
    default: break;              // T1; Winther, GR and the LCDM fit use its geometry
  }
  D2Geo g;
  g.c = th == 90.0 ? 0.0 : cos(th * (M_PI / 180.0));
  g.c2 = g.c * g.c;
  g.inv_s2 = 1.0 / (1.0 - g.c2);
  g.r = r;
  const double k2sq = 1.0 / (r * r + 1.0 + 2.0 * r * g.c);   // (k2/k)^2
  g.fb = k2sq;
  g.fa = r * r * k2sq;
  g.winther = variant == 5;
  g.gr2 = variant == 6;
  g.fit = variant == 9;
  return g;
}

// GEO 0: r = 1, c = 0 (T1, Winther, GR): the T1 braces mu - B.
// GEO 1: r = 1, c != 0: k1 = k2, full braces.
// GEO 2: r != 1: full braces at k1 and k2.
//
// The integration.  Per k there are eight second-order chains
//   y_ss = -damp y_s + c(s) y + src(s):
// D1(k), Da = D1(k1), Db = D1(k2) (no source); D2 (source: -W Pa Pb) and the ln|fR0| tangents
// Z1, Za, Zb (source: T times the chain's own primal); Z2 (source: T2 D2 - W (Pat Pb + Pa Pbt)
// - Wt Pa Pb).  One warp integrates four k, a lane per chain.
//
// What bounds it: an FP64 instruction occupies an SM sub-partition of this GPU for 64 cycles
// whatever the active lanes (measured: 64.3 cycles per dependent or independent DFMA), so the
// time is the number of FP64 instructions a warp issues per step.  A lane does only what
// depends on its own state, 21 of them: the coefficients, which depend on (k, a) alone, and the
// sources, which depend on chains integrated earlier, come from the block's other three warps
// (one per remaining sub-partition) through shared memory.  The lanes of one warp are at
// different times: a level (primal chains; D2 and the first tangents; Z2) runs two chunks of
// GR_CH steps behind the one whose stage values its sources need, so in an iteration the chain
// warp advances level l by chunk it - 2 l while the other warps fill the coefficients of chunk
// it + 1, the level-1 sources of chunk it - 1 and the level-2 sources of chunk it - 3.
// Measured (512 k, 1024 steps): 12.4 ms with a thread per k doing all of it, 0.87 ms now (the
// chain warp alone would take 0.76 ms: 21 instructions x 64 cycles x 1056 steps).
constexpr int GR_KPB = 4;            // k per block: 4 x 8 chains fill the chain warp
constexpr int GR_CH = 8;             // RK4 steps per chunk
constexpr int GR_HS = 2 * GR_CH + 1; // half steps of a chunk, both ends included
constexpr int GR_THREADS = 128;      // the chain warp and three warps for coefficients and sources
constexpr int GR_NC = 10;            // coefficients per (half step, k): c x 4, tangent x 4, W, Wt
constexpr int GR_VRING = 4, GR_SRING = 2, GR_CRING = 6;   // chunks kept: stage values, sources, coefficients
enum { CH_D1 = 0, CH_DA = 1, CH_DB = 2, CH_D2 = 3, CH_Z1 = 4, CH_ZA = 5, CH_ZB = 6, CH_Z2 = 7 };
struct GrowthSmem {
  double val[GR_VRING][GR_CH][4][32];             // y at the four stages of each step, per chain lane
  double src[GR_SRING][GR_CH][4][32];             // h^2 src at the four stages
  double coef[GR_CRING][GR_HS][GR_KPB][GR_NC];    // h^2 times the coefficients
  double damp[GR_CRING][GR_HS];                   // -h damp
  double red[8][4];                               // norm reduction
  double out[32];
};

// Coefficients of (k, half step), times h2: c of D1, Da, Db, D2; their tangents; W, Wt.
template <int GEO>
__device__ __forceinline__ void growth_coef(const Bg& b, double k2, bool gr, const D2Geo& g, double h2, double* o) {
  const double q = k2 * b.inv_a2, qa = q * g.fa, qb = q * g.fb;
  double mu_k = 1.0, mu_a = 1.0, mu_b = 1.0, mu_kt = 0.0, mu_at = 0.0, mu_bt = 0.0, br = 1.0, brt = 0.0;
  if (!gr) {
    const double rpk = 1.0 / (q + b.m2), rpa = 1.0 / (qa + b.m2);
    const double rpb = GEO == 2 ? 1.0 / (qb + b.m2) : rpa;
    mu_k = 1.0 + q * rpk * (1.0 / 3.0);
    mu_a = 1.0 + qa * rpa * (1.0 / 3.0);
    mu_b = GEO == 2 ? 1.0 + qb * rpb * (1.0 / 3.0) : mu_a;
    mu_kt = q * b.m2 * rpk * rpk * (1.0 / 3.0);
    mu_at = qa * b.m2 * rpa * rpa * (1.0 / 3.0);
    mu_bt = GEO == 2 ? qb * b.m2 * rpb * rpb * (1.0 / 3.0) : mu_at;
    const double B = b.bfac * q * rpk * rpa * rpb;
    if (g.gr2) {             // the GR D2 variant: mu = 1 in its chains and equation
      mu_a = mu_b = 1.0;
      mu_at = mu_bt = 0.0;
    } else if (GEO == 0) {
      br = mu_k - B;
      brt = mu_kt - B * (-2.0 + b.m2 * rpk + 2.0 * b.m2 * rpa);
    } else {
      const double G = b.m2 * rpk, Gt = -G * q * rpk;
      const double lin = 2.0 * g.c2 * (mu_a + mu_b - 2.0) + (g.c / g.r) * (mu_a - 1.0) + g.r * g.c * (mu_b - 1.0);
      const double lint = 2.0 * g.c2 * (mu_at + mu_bt) + (g.c / g.r) * mu_at + g.r * g.c * mu_bt;
      const double Bt = B * (-2.0 + b.m2 * rpk + b.m2 * rpa + b.m2 * rpb);
      br = (mu_k - g.c2 * (mu_a + mu_b - mu_k) + G * lin - B) * g.inv_s2;
      brt = (mu_kt - g.c2 * (mu_at + mu_bt - mu_kt) + Gt * lin + G * lint - Bt) * g.inv_s2;
    }
  }
  const double w = h2 * b.cc;
  o[CH_D1] = w * mu_k;
  o[CH_DA] = w * mu_a;
  o[CH_DB] = w * mu_b;
  o[CH_D2] = g.gr2 ? w : w * mu_k;
  o[CH_Z1] = w * mu_kt;
  o[CH_ZA] = w * mu_at;
  o[CH_ZB] = w * mu_bt;
  o[CH_Z2] = g.gr2 ? 0.0 : w * mu_kt;
  o[8] = w * br;
  o[9] = w * brt;
}

// s = ln a at half step j of steps of size h from s0
__device__ __forceinline__ double half_step_s(double s0, double h, int j) {
  const int i = j >> 1;
  return (j & 1) ? (s0 + i * h) + 0.5 * h : s0 + i * h;
}

// One RK4 step of (y, u = h y_s): coefficients C and damping D (scaled) at the step's ends and
// middle, stage sources s0..s3; the stage values of y go to st.
struct Rk4Stage { double y0, y1, y2, y3; };
__device__ __forceinline__ Rk4Stage rk4_step(double& y, double& u, double D0, double Dm, double D1, double C0, double Cm,
                                             double C1, double s0, double s1, double s2, double s3) {
  Rk4Stage r;
  r.y0 = y;
  const double f0 = fma(D0, u, fma(C0, y, s0));
  r.y1 = fma(0.5, u, y);
  const double u1 = fma(0.5, f0, u);
  const double f1 = fma(Dm, u1, fma(Cm, r.y1, s1));
  r.y2 = fma(0.5, u1, y);
  const double u2 = fma(0.5, f1, u);
  const double f2 = fma(Dm, u2, fma(Cm, r.y2, s2));
  r.y3 = y + u2;
  const double u3 = u + f2;
  const double f3 = fma(D1, u3, fma(C1, r.y3, s3));
  const double f12 = f1 + f2, f012 = f0 + f12;
  y = fma(1.0 / 6.0, f012, y + u);
  u = fma(1.0 / 6.0, (f012 + f12) + f3, u);
  return r;
}

// D1 of GR at a = 1 from the Einstein-de Sitter mode at a_init, by the whole block: the RK4
// step is a 2x2 matrix on (y, u), each thread multiplies those of its share of the steps, and
// the shares are multiplied in order.
__device__ double gr_norm(const GrowthParams& p, double s0, GrowthSmem& sm) {
  const double h = (0.0 - s0) / p.n_steps;
  const int per = (p.n_steps + GR_THREADS - 1) / GR_THREADS;
  const int i0 = threadIdx.x * per, i1 = min(p.n_steps, i0 + per);
  double a0 = 1.0, a1 = 0.0, b0 = 0.0, b1 = 1.0;   // columns: (y, u) images of (1, 0) and (0, 1)
  if (i0 < i1) {
    Bg e = background(p, half_step_s(s0, h, 2 * i0), true);
    for (int i = i0; i < i1; ++i) {
      const Bg m = background(p, half_step_s(s0, h, 2 * i + 1), true), f = background(p, half_step_s(s0, h, 2 * i + 2), true);
      const double D0 = -h * e.damp, Dm = -h * m.damp, D1 = -h * f.damp;
      const double C0 = h * h * e.cc, Cm = h * h * m.cc, C1 = h * h * f.cc;
      rk4_step(a0, a1, D0, Dm, D1, C0, Cm, C1, 0.0, 0.0, 0.0, 0.0);
      rk4_step(b0, b1, D0, Dm, D1, C0, Cm, C1, 0.0, 0.0, 0.0, 0.0);
      e = f;
    }
  }
  // lane l holds the product of the shares l .. l + 2^k - 1 after k rounds
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double c0 = __shfl_down_sync(0xffffffffu, a0, o), c1 = __shfl_down_sync(0xffffffffu, a1, o);
    const double d0 = __shfl_down_sync(0xffffffffu, b0, o), d1 = __shfl_down_sync(0xffffffffu, b1, o);
    const double n0 = fma(c0, a0, d0 * a1), n1 = fma(c1, a0, d1 * a1);
    const double m0 = fma(c0, b0, d0 * b1), m1 = fma(c1, b0, d1 * b1);
    a0 = n0; a1 = n1; b0 = m0; b1 = m1;
  }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    sm.red[warp][0] = a0;
    sm.red[warp][1] = a1;
    sm.red[warp][2] = b0;
    sm.red[warp][3] = b1;
  }
  __syncthreads();
  double y = p.a_init, u = h * p.a_init;   // EdS growing mode: D = a, dD/ds = a
  for (int w = 0; w < GR_THREADS / 32; ++w) {
    const double ny = fma(sm.red[w][0], y, sm.red[w][2] * u);
    u = fma(sm.red[w][1], y, sm.red[w][3] * u);
    y = ny;
  }
  return y;
}

template <int GEO>
__global__ void __launch_bounds__(GR_THREADS) k_growth(GrowthParams p, double* tab, float* tabf) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  GrowthSmem& sm = *reinterpret_cast<GrowthSmem*>(s_raw);
  if (p.fr0s) p.fr0_abs = p.fr0s[blockIdx.y];     // instance blockIdx.y
  tab += (size_t)blockIdx.y * 4 * p.nk;
  tabf += (size_t)blockIdx.y * 4 * p.nk;
  const bool gr = (p.fr0_abs == 0.0);
  const D2Geo geo = d2_geo(p.d2_variant);
  const double s0 = log(p.a_init);
  const double norm = gr_norm(p, s0, sm);
  const double h = (log(p.a_out) - s0) / p.n_steps, h2 = h * h;
  const int k0 = blockIdx.x * GR_KPB;
  const int n_half = 2 * p.n_steps;
  const int nch = (p.n_steps + GR_CH - 1) / GR_CH;
  // coefficients of chunk c: threads t, t + stride, ... of a group of `stride` threads, t and
  // stride congruent to threadIdx.x and 0 mod GR_KPB, so a thread keeps to one k
  const int kf = threadIdx.x % GR_KPB;
  const double k = p.k_min * pow(p.k_max / p.k_min, (double)min(k0 + kf, p.nk - 1) / (double)(p.nk - 1));
  auto fill_coef = [&](int c, int t, int stride) {
    for (; t < GR_HS * GR_KPB; t += stride) {
      const int j = t / GR_KPB;
      const Bg b = background(p, half_step_s(s0, h, min(c * 2 * GR_CH + j, n_half)), gr);
      growth_coef<GEO>(b, k * k, gr, geo, h2, sm.coef[c % GR_CRING][j][kf]);
      if (kf == 0) sm.damp[c % GR_CRING][j] = -h * b.damp;
    }
  };
  fill_coef(0, threadIdx.x, GR_THREADS);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // chain lane: k = lane / 8, chain = lane % 8
  const int chain = lane & 7, kk = lane >> 3;
  const int level = chain < CH_D2 ? 0 : (chain == CH_Z2 ? 2 : 1);
  double y = chain < CH_D2 ? p.a_init : (chain == CH_D2 ? -3.0 / 7.0 * p.a_init * p.a_init : 0.0);
  double u = h * (chain < CH_D2 ? p.a_init : (chain == CH_D2 ? -6.0 / 7.0 * p.a_init * p.a_init : 0.0));
  __syncthreads();
  for (int it = 0; it < nch + 4; ++it) {
    if (warp == 0) {
      const int c = it - 2 * level;
      if (c >= 0 && c < nch) {
        const double* cf = &sm.coef[c % GR_CRING][0][kk][chain & 3];
        const double* dm = sm.damp[c % GR_CRING];
        double* va = &sm.val[c % GR_VRING][0][0][lane];
        const double* sr = &sm.src[c % GR_SRING][0][0][lane];
        double D0 = dm[0], C0 = cf[0];
#pragma unroll 2
        for (int i = 0; i < GR_CH; ++i) {
          const double Dm = dm[2 * i + 1], D1 = dm[2 * i + 2];
          const double Cm = cf[(2 * i + 1) * GR_KPB * GR_NC], C1 = cf[(2 * i + 2) * GR_KPB * GR_NC];
          double s[4] = {0.0, 0.0, 0.0, 0.0};
          if (level > 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] = sr[(i * 4 + q) * 32];
          }
          double ny = y, nu = u;
          const Rk4Stage r = rk4_step(ny, nu, D0, Dm, D1, C0, Cm, C1, s[0], s[1], s[2], s[3]);
          va[(i * 4 + 0) * 32] = r.y0;
          va[(i * 4 + 1) * 32] = r.y1;
          va[(i * 4 + 2) * 32] = r.y2;
          va[(i * 4 + 3) * 32] = r.y3;
          if (c * GR_CH + i < p.n_steps) {   // the last chunk may be partial
            y = ny;
            u = nu;
          }
          D0 = D1;
          C0 = C1;
        }
      }
    } else {
      const int t0 = threadIdx.x - 32, stride = GR_THREADS - 32;
      if (it + 1 < nch) fill_coef(it + 1, t0, stride);
      // sources: task (step, stage, k); the half step of stages 0, 1, 2, 3 is 2 i + {0, 1, 1, 2}
      for (int lev = 1; lev <= 2; ++lev) {
        const int c = it + 1 - 2 * lev;
        if (c < 0 || c >= nch) continue;
        for (int t = t0; t < GR_CH * 4 * GR_KPB; t += stride) {
          const int kt = t % GR_KPB, q = (t / GR_KPB) & 3, i = t / (4 * GR_KPB);
          const int j = 2 * i + ((q + 1) >> 1);
          const double* cf = sm.coef[c % GR_CRING][j][kt];
          const double* v = &sm.val[c % GR_VRING][i][q][kt * 8];
          double* o = &sm.src[c % GR_SRING][i][q][kt * 8];
          const double Pa = v[geo.winther ? CH_D1 : CH_DA], Pb = v[geo.winther ? CH_D1 : CH_DB];
          if (lev == 1) {
            o[CH_D2] = -cf[8] * (Pa * Pb);
            o[CH_Z1] = cf[4] * v[CH_D1];
            o[CH_ZA] = cf[5] * v[CH_DA];
            o[CH_ZB] = cf[6] * v[CH_DB];
          } else {
            const double Pat = v[geo.winther ? CH_Z1 : CH_ZA], Pbt = v[geo.winther ? CH_Z1 : CH_ZB];
            o[CH_Z2] = fma(cf[7], v[CH_D2], -fma(cf[8], fma(Pat, Pb, Pa * Pbt), cf[9] * (Pa * Pb)));
          }
        }
      }
    }
    __syncthreads();
  }
  if (warp == 0) sm.out[lane] = y;
  __syncthreads();
  const int t = k0 + threadIdx.x;
  if (threadIdx.x >= GR_KPB || t >= p.nk) return;
  const double* o = sm.out + threadIdx.x * 8;
  const int nk = p.nk;
  tab[t] = o[CH_D1] / norm;
  tab[nk + t] = o[CH_D2] / (norm * norm);
  tab[2 * nk + t] = o[CH_Z1] / norm;
  tab[3 * nk + t] = o[CH_Z2] / (norm * norm);
  if (geo.fit) {   // D2 = -(3/7) D1^2 Omega_m(a)^(-1/143), tangent -(6/7) D1 dD1 Omega_m(a)^(-1/143)
    const double a3 = 1.0 / (p.a_out * p.a_out * p.a_out);
    const double f = pow(p.omega_m * a3 / (p.omega_m * a3 + p.omega_l), -1.0 / 143.0);
    tab[nk + t] = -3.0 / 7.0 * tab[t] * tab[t] * f;
    tab[3 * nk + t] = -6.0 / 7.0 * tab[t] * tab[2 * nk + t] * f;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) tabf[i * nk + t] = (float)tab[i * nk + t];
}

template <int GEO>
static cudaError_t launch_growth_geo(const GrowthParams& p, double* tab, float* tabf, cudaStream_t s) {
  const int blocks = (p.nk + GR_KPB - 1) / GR_KPB;
  cudaFuncSetAttribute(k_growth<GEO>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GrowthSmem));
  k_growth<GEO><<<dim3(blocks, p.n_inst > 0 ? p.n_inst : 1), GR_THREADS, sizeof(GrowthSmem), s>>>(p, tab, tabf);
  return cudaGetLastError();
}

cudaError_t launch_growth(const GrowthParams& p, double* tab, float* tabf, cudaStream_t s) {
  const D2Geo g = d2_geo(p.d2_variant);
  if (g.r != 1.0) return launch_growth_geo<2>(p, tab, tabf, s);
  if (g.c != 0.0) return launch_growth_geo<1>(p, tab, tabf, s);
  return launch_growth_geo<0>(p, tab, tabf, s);
}

// ------------------------------------------------------------- mode tables
// For every integer |n|^2 of an n^3 grid: k = (2 pi / L) sqrt(|n|^2),
//   x = sqrt(P_lin(k) N^3 / V)  (EH no-wiggle, sigma_8 amplitude),
//   y = 1 / (k^2 N^3),
//   z, w = D1(k), D2(k), linear in ln k between the growth-table nodes and clamped at the
// ends - all in FP64, rounded once; and mt1 (where given) the FP32 products of D1, D2 and their
// derivatives by ln|fR0| with y, the four values the adjoint source pass multiplies by.
__device__ double interp_lnk64(const double* t, int nk, double lnkmin, double dlnk, double lnk) {
  double x = (lnk - lnkmin) / dlnk;
  if (x <= 0.0) return t[0];
  if (x >= (double)(nk - 1)) return t[nk - 1];
  int i = (int)x;
  if (i > nk - 2) i = nk - 2;
  const double f = x - (double)i;
  return t[i] + f * (t[i + 1] - t[i]);
}

__global__ void k_mode_tables(GrowthParams p, const DevCosmo* cosmo, const double* tab, int inst0, int n, double box,
                              float4* mt0, float4* mt1) {
  const int len = mode_table_len(n);
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= len) return;
  const int inst = inst0 + blockIdx.y;
  const double* tb = tab + (size_t)inst * 4 * p.nk;
  float4* o0 = mt0 + (size_t)blockIdx.y * len;
  if (idx == 0) {
    o0[0] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (mt1) mt1[(size_t)blockIdx.y * len] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const double nd = n, kf = 2.0 * M_PI / box;
  const double k = kf * sqrt((double)idx);
  const EhConst c = eh_constants(p);
  const double T = eh_T64(c, k, p.h);
  const double sp = sqrt(cosmo->amp) * pow(k, 0.5 * p.n_s) * T * sqrt(nd * nd * nd / (box * box * box));
  const double inv = 1.0 / (k * k * nd * nd * nd);
  const double lnkmin = log(p.k_min), dlnk = (log(p.k_max) - log(p.k_min)) / (p.nk - 1), lk = log(k);
  const double d1 = interp_lnk64(tb, p.nk, lnkmin, dlnk, lk);
  const double d2 = interp_lnk64(tb + p.nk, p.nk, lnkmin, dlnk, lk);
  const double t1 = interp_lnk64(tb + 2 * p.nk, p.nk, lnkmin, dlnk, lk);
  const double t2 = interp_lnk64(tb + 3 * p.nk, p.nk, lnkmin, dlnk, lk);
  o0[idx] = make_float4((float)sp, (float)inv, (float)d1, (float)d2);
  if (!mt1) return;
  const float iv = (float)inv;
  mt1[(size_t)blockIdx.y * len + idx] = make_float4((float)d1 * iv, (float)d2 * iv, (float)t1 * iv, (float)t2 * iv);
}

cudaError_t launch_mode_tables(const GrowthParams& p, const DevCosmo* cosmo, const double* tab, int inst0, int count,
                               int n, double box, float4* mt0, float4* mt1, cudaStream_t s) {
  const int len = mode_table_len(n);
  k_mode_tables<<<dim3((len + 127) / 128, count), 128, 0, s>>>(p, cosmo, tab, inst0, n, box, mt0, mt1);
  return cudaGetLastError();
}

}  // namespace lpt2
