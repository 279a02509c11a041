// Depth march for the reference Green's function g(k_n, z_j; omega~_f).
//
// g solves g'' + (omega~^2/c0(z)^2 - k^2) g = -delta(z) (the Green's-function equation of
// Section "Two dimensions" after a lateral Fourier transform; G~ = g / sqrt(2 pi)).  The
// paper does not say how to evaluate it in layers; this is the stable reflectivity
// recursion:
//   kappa_j = sqrt(omega~^2/c_j^2 - k^2), Im kappa_j >= 0,
//   upward:   r_{J-1} = 0, y = kappa_{j+1}(1 - r_{j+1})/(1 + r_{j+1}),
//             rho_j = (kappa_j - y)/(kappa_j + y), r_j = rho_j exp(2 i kappa_j h_j),
//   downward: A_0 = i/(2 kappa_0), A_{j+1} = A_j exp(i kappa_j h_j)(1 + rho_j)/(1 + r_{j+1}),
//   field:    g(z) = A_j [exp(i kappa_j (z - t_j)) + rho_j exp(i kappa_j (2 h_j - (z - t_j)))]
// in which no exponential grows.  Within a layer the two exponentials advance from one
// depth sample to the next by multiplication with exp(+-i kappa_j dz) (error ~ n ulp),
// re-anchored by a direct evaluation at every layer entry and chunk start.
//
// Kernels: green_layer (one thread per (f, n, layer): vertical wavenumber, the layer's phase
// factors and the interface's recursion coefficients, fully parallel), green_recursion (one
// thread per (f, n): the two recursions in a division-free form, FP64), then one of two
// evaluations:
//   green_eval64  (FP64 table, and/or the FP32 table sqrt|s_f| g rounded from it, with the
//                 rounding remainder as a second FP32 table for a double-float pair):
//                 a warp per 32 rows (f, n) and 16 depths marches them by the recurrence and
//                 stages its tile in shared memory so the table rows are written coalesced;
//   green_eval32  (FP32 table sqrt|s_f| g for the mixed path; green_coef32 rounds the layers'
//                 coefficients for it): one thread per (f, n, z);
//                 each exponential's phase and decay are formed and range-reduced in FP64
//                 (Cody-Waite for the phase, integer/fraction split for the decay) and
//                 evaluated with FP32 sincos/exp2 of the reduced arguments, ~1e-7 relative.
// For the line inversion with the FP32 residual (GREEN_G32F) and at most 32 layers,
// green_kap32 (one thread per (f, n, layer)) and green_rec32 (one thread per (f, n)) replace
// green_layer and green_recursion: each kappa_j by an FP32 complex square root and one Newton
// step on the FP64 residual w - kappa^2 (the square of the FP32 root is exact in FP64, so the
// (hi, lo) pair carries kappa to ~1e-14 with four FP64 products instead of a complex FP64
// root), exp(i kappa_j h_j) by double-float phase reduction, and both recursions in FP32
// complex arithmetic; the outputs are the FP32 coefficients green_eval32 reads.  GB300's FP64
// rate made the FP64 transcendentals of green_layer and the recursion's FP64 divisions most of
// the depth march.
#include "edt_internal.h"
#include "cplx.cuh"
#include "green_coef.cuh"

namespace edt {

namespace {

// FP32 copies for the fast evaluation: kappa.x and kappa.y as (hi, lo) pairs, amp, rho
constexpr int NCOEF32 = 8;

// sqrt(w) on the branch Im >= 0, FP64: the FP32 root (relative error ~1e-7) and two Newton steps
// k + (w - k^2) / (2 k) whose residual is formed in FP64 and whose divisor is the FP32 root's (it
// only scales the correction): 1e-14, then FP64 rounding, in about 20 FP64 operations instead of
// the hundred of a complex FP64 root.  Values outside the FP32 range take that root.
__device__ __forceinline__ double2 kappa_of(double2 w) {
  const double m = fmax(fabs(w.x), fabs(w.y));
  if (!(m > 1e-25 && m < 1e25)) return csqrt_upper(w);
  const float2 k32 = csqrt_upper32(make_float2(float(w.x), float(w.y)));
  const float2 inv = cinv32(make_float2(2.f * k32.x, 2.f * k32.y));
  double2 k = cmk(double(k32.x), double(k32.y));
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const double rr = fma(k.y, k.y, fma(-k.x, k.x, w.x)), ri = fma(-2.0 * k.x, k.y, w.y);
    const float2 dk = make_float2(float(rr), float(ri)) * inv;
    k.x += double(dk.x);
    k.y += double(dk.y);
  }
  return k;
}

// 2^-e of a positive double's exponent e (|v| in [2^e, 2^(e+1))), by its bits
__device__ __forceinline__ double pow2_down(double v) {
  const int e = (__double2hiint(v) >> 20) & 0x7ff;
  return __hiloint2double(min(max(2046 - e, 1), 2046) << 20, 0);
}

// Per (f, n) and LRUN consecutive layers: kappa_j, exp(i kappa_j h_j), the step factors
// exp(+-i kappa_j dz) of layers that may hold two depth samples, and the interface's recursion
// coefficients sigma = lambda (kappa_j + kappa_{j+1}), delta = lambda (kappa_j - kappa_{j+1}) and
// tau = 2 kappa_j lambda exp(i kappa_j h_j), lambda the power of two that puts sigma near 1.
// LRUN = 4 forms five kappa for four layers instead of eight; with few layers one per thread
// spreads better beside the data transform that runs at the same time (13 layers over 9675
// (f, n): a 256-point line takes 1.13 ms with 1, 1.19 with 4).
constexpr int LBLOCK = 128;
template <int LRUN>
__global__ void __launch_bounds__(LBLOCK) green_layer_kernel(Dev d, int want_steps) {
  const long long gid = (long long)blockIdx.x * LBLOCK + threadIdx.x;
  const int J = d.nlayer, nrun = (J + LRUN - 1) / LRUN;
  if (gid >= (long long)d.nf * d.nk * nrun) return;
  const int n = int(gid % d.nk);                   // wavenumber fastest: coalesced stores
  const long long fj = gid / d.nk;
  const int j0 = int(fj % nrun) * LRUN, f = int(fj / nrun);
  const FreqConst fc = d.fc[f];
  const double k = d.kval ? d.kval[n] : double(n) * (2.0 * M_PI / (double(d.N) * d.dx));
  const double2 om = cmk(fc.om_re, fc.om_im);
  const double2 om2 = om * om;
  double2* c = d.coef;
  auto kappa = [&](int j) {
    const double inv_c2 = 1.0 / (d.layer_vel[j] * d.layer_vel[j]);
    return kappa_of(cmk(om2.x * inv_c2 - k * k, om2.y * inv_c2));
  };
  double2 kap = kappa(j0);
#pragma unroll 1
  for (int j = j0; j < min(J, j0 + LRUN); ++j) {
    c[cix(d, f, n, j, C_KAP)] = kap;
    double h = 2.0 * d.dz;
    double2 kn = kap;
    if (j < J - 1) {
      h = d.layer_top[j + 1] - d.layer_top[j];
      const double2 eh = cexp(cmk(-kap.y * h, kap.x * h));
      kn = kappa(j + 1);
      const double2 sg = kap + kn;
      const double lam = pow2_down(fmax(fabs(sg.x), fabs(sg.y)));
      c[cix(d, f, n, j, C_EH)] = eh;
      c[cix(d, f, n, j, C_SIG)] = lam * sg;
      c[cix(d, f, n, j, C_DEL)] = lam * (kap - kn);
      c[cix(d, f, n, j, C_AMP)] = (2.0 * lam) * (kap * eh);
    }
    // samples are dz apart, so a thinner layer holds one at most
    if (want_steps && h > 0.999 * d.dz) {
      const double2 E = cexp(cmk(-kap.y * d.dz, kap.x * d.dz));
      c[cix(d, f, n, j, C_E)] = E;
      c[cix(d, f, n, j, C_EI)] = cinv(E);
    }
    kap = kn;
  }
}

__device__ __forceinline__ double2 shfl2(double2 v, int src) {
  return cmk(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ double cmax(double2 v) { return fmax(fabs(v.x), fabs(v.y)); }
// s = 2^-e of the exponent e of v (bits), e added to ex
__device__ __forceinline__ double rescale(double v, int& ex) {
  const double s = pow2_down(v);
  ex += 1023 - ((__double2hiint(s) >> 20) & 0x7ff);
  return s;
}

// The recursions over the layers.  With r_j = N_j / D_j the upward recursion of the header is linear,
//   M_j = delta_j D_{j+1} + sigma_j N_{j+1},  D_j = sigma_j D_{j+1} + delta_j N_{j+1},
//   N_j = exp(2 i kappa_j h_j) M_j,   rho_j = M_j / D_j,
// from N = 0, D = 1 at the half-space, and the downward one telescopes:
//   A_j = (i / (2 kappa_0)) prod_{i < j} (2 kappa_i exp(i kappa_i h_i)) D_j / D_0
// (the powers of two lambda_i cancel against tau_i).  No division is left on the chains.  Every
// eighth layer the pair is rescaled by a power of two (into tau too), so that thousands of
// layers neither overflow nor vanish.  Leaves M_j (C_MUP), D_j (C_DEN) and T_j = A_j / D_j (C_AMP).
//
// S lanes share the layers of one (f, n), a run of layers each.  One warp takes 64 cycles of its
// quarter of an SM for an FP64 instruction however few lanes work, so a stack of many layers over
// few (f, n) (257 layers, 1056 of them: 33 warps on 608 quarters) has to be split: each lane
// forms the 2 x 2 matrix of its run, a suffix scan of the matrices over the lanes gives every run
// its incoming pair, then the run is walked as usual; the amplitudes take a prefix product.
template <int S>
__global__ void __launch_bounds__(32) green_recursion_kernel(Dev d) {
  constexpr int RPW = 32 / S;                             // (f, n) per warp
  const int lane = threadIdx.x, seg = lane / RPW;
  const long long row0 = (long long)blockIdx.x * RPW + lane % RPW, nrow = (long long)d.nf * d.nk;
  const bool live = row0 < nrow;                          // the others only take part in the shuffles
  const long long row = live ? row0 : nrow - 1;
  const int f = int(row / d.nk), n = int(row - (long long)f * d.nk);
  const int J = d.nlayer;
  const int ja = int((long long)(J - 1) * seg / S), jb = int((long long)(J - 1) * (seg + 1) / S);
  const size_t nk = d.nk, lst = size_t(NCOEF) * nk;       // from a layer to the next
  double2* c = d.coef + cix(d, f, n, 0, 0);
  const double2 zero = cmk(0.0, 0.0), one = cmk(1.0, 0.0);
  constexpr int U = 4;                                    // layers loaded ahead of the chain
  double2 N = zero, D = one;                              // what enters the run from below
  int ein = 0;                                            // true pair: times 2^ein
  if (S > 1) {
    // columns (Nu, Du), (Nv, Dv): the images of (1, 0) and (0, 1); true matrix: times 2^e
    double2 Nu = one, Du = zero, Nv = zero, Dv = one;
    int e = 0;
    auto norm = [&]() {
      const double s = rescale(fmax(fmax(cmax(Nu), cmax(Du)), fmax(cmax(Nv), cmax(Dv))), e);
      Nu = s * Nu; Du = s * Du; Nv = s * Nv; Dv = s * Dv;
    };
    for (int j1 = jb; j1 > ja; j1 -= U) {
      double2 sg[U], de[U], eh[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j1 - 1 - u;
        if (j < ja) continue;
        const double2* cl = c + lst * j;
        sg[u] = cl[C_SIG * nk]; de[u] = cl[C_DEL * nk]; eh[u] = cl[C_EH * nk];
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j1 - 1 - u;
        if (j < ja) continue;
        const double2 E = eh[u] * eh[u];
        const double2 Mu = de[u] * Du + sg[u] * Nu, Mv = de[u] * Dv + sg[u] * Nv;
        Du = sg[u] * Du + de[u] * Nu;
        Dv = sg[u] * Dv + de[u] * Nv;
        Nu = E * Mu;
        Nv = E * Mv;
        if ((j & 7) == 0) norm();
      }
    }
    norm();
#pragma unroll
    for (int o = 1; o < S; o <<= 1) {                     // times the product of the o runs below
      const int src = min(lane + o * RPW, 31);
      const double2 a = shfl2(Nu, src), b = shfl2(Nv, src), x = shfl2(Du, src), y = shfl2(Dv, src);
      const int eo = __shfl_sync(0xffffffffu, e, src);
      if (seg + o < S) {
        const double2 nu = Nu * a + Nv * x, nv = Nu * b + Nv * y;
        const double2 du = Du * a + Dv * x, dv = Du * b + Dv * y;
        Nu = nu; Nv = nv; Du = du; Dv = dv;
        e += eo;
        norm();
      }
    }
    const int src = min(lane + RPW, 31);
    const double2 bn = shfl2(Nv, src), bd = shfl2(Dv, src);
    const int eb = __shfl_sync(0xffffffffu, e, src);
    if (seg + 1 < S) { N = bn; D = bd; ein = eb; }
  }
  if (live && seg == S - 1) {
    double2* cl = c + lst * (J - 1);
    cl[C_MUP * nk] = zero;
    cl[C_DEN * nk] = one;
  }
  double2 prod = one;                                     // of the run's tau (rescaled)
  int er = 0;                                             // exponents taken out inside the run
  for (int j1 = jb; j1 > ja; j1 -= U) {
    double2 sg[U], de[U], eh[U], ta[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j1 - 1 - u;
      if (j < ja) continue;
      const double2* cl = c + lst * j;
      sg[u] = cl[C_SIG * nk]; de[u] = cl[C_DEL * nk]; eh[u] = cl[C_EH * nk];
      if (S > 1) ta[u] = cl[C_AMP * nk];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j1 - 1 - u;
      if (j < ja) continue;
      double2* cl = c + lst * j;
      double2 M = de[u] * D + sg[u] * N;
      D = sg[u] * D + de[u] * N;
      const double2 E = eh[u] * eh[u];
      if ((j & 7) == 0) {
        const double s = rescale(cmax(D), er);
        D = s * D;
        M = s * M;
        const double2 t = s * (S > 1 ? ta[u] : cl[C_AMP * nk]);
        if (live) cl[C_AMP * nk] = t;
        if (S > 1) ta[u] = t;
      }
      if (S > 1) prod = prod * ta[u];
      N = E * M;
      if (live) {
        cl[C_MUP * nk] = M;
        cl[C_DEN * nk] = D;
      }
    }
  }
  // T at the run's first layer: T_0 = A_0 / D_0 times the runs above; a run's stored D is off the
  // true one by 2^(ein + er), its product of tau by 2^-er
  double2 T = cmk(0.0, 0.5) * cinv(c[C_KAP * nk] * D);
  if (S > 1) {
    T = shfl2(T, lane % RPW);
    const int e0 = __shfl_sync(0xffffffffu, ein + er, lane % RPW);
    int x = er;
#pragma unroll
    for (int o = 1; o < S; o <<= 1) {                     // inclusive prefix over the runs
      const int src = max(lane - o * RPW, 0);
      const double2 q = shfl2(prod, src);
      const int xo = __shfl_sync(0xffffffffu, x, src);
      if (seg >= o) { prod = prod * q; x += xo; }
    }
    const int src = max(lane - RPW, 0);
    const double2 q = shfl2(prod, src);
    const int xo = __shfl_sync(0xffffffffu, x, src);
    if (seg > 0) {
      T = T * q;
      const int k = xo + ein + er - e0;
      T = cmk(scalbn(T.x, k), scalbn(T.y, k));
    }
  }
  const int je = seg == S - 1 ? J : jb;                   // the half-space belongs to the last run
  for (int j0 = ja; j0 < je; j0 += 2 * U) {
    double2 tau[2 * U];
#pragma unroll
    for (int u = 0; u < 2 * U; ++u)
      if (j0 + u < min(je, J - 1)) tau[u] = c[lst * (j0 + u) + C_AMP * nk];
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      if (j0 + u >= je) continue;
      if (live) c[lst * (j0 + u) + C_AMP * nk] = T;
      if (j0 + u < J - 1) T = T * tau[u];
    }
  }
}

// the FP32 coefficients green_eval32 reads, per (f, n, layer)
__global__ void __launch_bounds__(128) green_coef32_kernel(Dev d) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int J = d.nlayer;
  if (gid >= (long long)d.nf * d.nk * J) return;
  const int n = int(gid % d.nk);
  const long long fj = gid / d.nk;
  const int j = int(fj % J), f = int(fj / J);
  double2 a, r;
  layer_waves(d, f, n, j, a, r);
  const double2 kap = d.coef[cix(d, f, n, j, C_KAP)];
  float4 k4;
  split_ff(kap.x, k4.x, k4.y);
  split_ff(kap.y, k4.z, k4.w);
  float4* o = reinterpret_cast<float4*>(d.coef32 + ((size_t(f) * d.nk + n) * J + j) * NCOEF32);
  o[0] = k4;
  o[1] = make_float4(float(a.x), float(a.y), float(r.x), float(r.y));
}

// The FP32 recursion's rounding errors (and those of its FP32 exponentials) compound over the
// layers, about a few FP32 ulps per layer in the amplitudes: deeper stacks keep the FP64 march.
constexpr int COEF32_MAX_LAYERS = 32;

// FP32 coefficients, pass 1: one thread per (f, n, layer) -- kappa_j (FP32 root, one Newton
// step on the FP64 residual) and exp(i kappa_j h_j), the latter parked in the amplitude slots
// until the recursion replaces it.
__global__ void green_kap32_kernel(Dev d) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int J = d.nlayer;
  const long long total = (long long)d.nf * d.nk * J;
  if (gid >= total) return;
  const int j = int(gid % J);
  const long long fn = gid / J;
  const int n = int(fn % d.nk), f = int(fn / d.nk);
  const FreqConst fc = d.fc[f];
  const double L = double(d.N) * d.dx;
  const double k = d.kval ? d.kval[n] : 2.0 * M_PI * double(n) / L;
  const double om2r = fc.om_re * fc.om_re - fc.om_im * fc.om_im, om2i = 2.0 * fc.om_re * fc.om_im;
  const double ic2 = 1.0 / (d.layer_vel[j] * d.layer_vel[j]);
  const double wr2 = om2r * ic2 - k * k, wi2 = om2i * ic2;
  const float2 k32 = csqrt_upper32(make_float2(float(wr2), float(wi2)));
  const double rr = wr2 - (double(k32.x) * k32.x - double(k32.y) * k32.y);
  const double ri = wi2 - 2.0 * double(k32.x) * k32.y;
  const float2 dk = (k32.x == 0.f && k32.y == 0.f)
                        ? make_float2(0.f, 0.f)
                        : make_float2(float(rr), float(ri)) * cinv32(make_float2(2.f * k32.x, 2.f * k32.y));
  float2 eh = make_float2(1.f, 0.f);
  if (j + 1 < J) {
    float hh, hl;
    split_ff(d.layer_top[j + 1] - d.layer_top[j], hh, hl);
    eh = expi_ff(k32.x, dk.x, k32.y, hh, hl);            // exp(i kappa_j h_j)
  }
  float4* o = reinterpret_cast<float4*>(d.coef32 + size_t(gid) * NCOEF32);
  o[0] = make_float4(k32.x, dk.x, k32.y, dk.y);
  o[1] = make_float4(eh.x, eh.y, 0.f, 0.f);
}

// Pass 2: one thread per (f, n) -- the upward recursion for rho_j (stored; the amplitude slot
// takes exp(i kappa_j h_j) / (1 + r_{j+1})), then the downward one for the amplitudes, in FP32.
__global__ void __launch_bounds__(128) green_rec32_kernel(Dev d) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  const int f = blockIdx.y;
  if (n >= d.nk) return;
  const int J = d.nlayer;
  float4* c4 = reinterpret_cast<float4*>(d.coef32 + (size_t(f) * d.nk + n) * size_t(J) * NCOEF32);
  const float2 one = make_float2(1.f, 0.f);
  // upward: r_{J-1} = 0; y = kappa_{j+1}(1 - r_{j+1})/(1 + r_{j+1}); rho_j = (kappa_j - y)/(kappa_j + y)
  float2 r = make_float2(0.f, 0.f);
  float4 kn4 = c4[2 * (J - 1)];
  float2 kn = make_float2(kn4.x + kn4.y, kn4.z + kn4.w);
  c4[2 * (J - 1) + 1] = make_float4(0.f, 0.f, 0.f, 0.f);   // amplitude set below; rho_{J-1} = 0
  for (int j = J - 2; j >= 0; --j) {
    const float4 kj4 = c4[2 * j], ah = c4[2 * j + 1];
    const float2 kj = make_float2(kj4.x + kj4.y, kj4.z + kj4.w), eh = make_float2(ah.x, ah.y);
    const float2 inv1r = cinv32(one + r);
    const float2 y = kn * (one - r) * inv1r;
    const float2 rho = (kj - y) * cinv32(kj + y);
    r = rho * (eh * eh);
    const float2 ehi = eh * inv1r;                            // exp(i kappa_j h_j) / (1 + r_{j+1})
    c4[2 * j + 1] = make_float4(ehi.x, ehi.y, rho.x, rho.y);
    kn = kj;
  }
  // downward: A_0 = i / (2 kappa_0), A_{j+1} = A_j exp(i kappa_j h_j)(1 + rho_j)/(1 + r_{j+1})
  const float4 k04 = c4[0];
  float2 amp = make_float2(0.f, 0.5f) * cinv32(make_float2(k04.x + k04.y, k04.z + k04.w));
  for (int j = 0; j < J; ++j) {
    const float4 ah = c4[2 * j + 1];                          // (ehi, rho)
    c4[2 * j + 1] = make_float4(amp.x, amp.y, ah.z, ah.w);
    if (j + 1 < J) amp = amp * make_float2(ah.x, ah.y) * (one + make_float2(ah.z, ah.w));
  }
}

// One warp per 32 table rows (of any frequencies) and EV_ZC depths: the FP64 unit is the bound, so
// the lanes are filled across frequencies; 16 depths share the anchors where the rows alone fill
// the GPU, 4 where they do not (a 64-point line: 33 row blocks for 608 quarters of an SM).
template <int EV_ZC>
__global__ void __launch_bounds__(32) green_eval64_kernel(Dev d) {
  __shared__ double2 tile[32][EV_ZC + 1];
  const int lane = threadIdx.x;
  const long long nrow = (long long)d.nf * d.nk;
  const long long r0 = (long long)blockIdx.x * 32;
  const long long row = min(r0 + lane, nrow - 1);
  const int f = int(row / d.nk), n = int(row - (long long)f * d.nk);
  const int J = d.nlayer;
  const double2* c = d.coef;
  const int zc = blockIdx.y * EV_ZC;
  // both waves carry the amplitude (and, where only sqrt|s_f| g is wanted, sqrt|s_f|) from their anchors,
  // so a depth takes two products and a sum, 10 FP64 operations instead of 18 (256 points, 150 depths,
  // 75 frequencies: an inversion takes 0.985 ms, 1.000 with 18)
  const double sq_own = d.g32 ? sqrt(d.fc[f].s_abs) : 0.0;
  const bool fold = d.g32 && !d.g64;
  {
    int cur = -1;
    double2 e1 = cmk(0.0, 0.0), e2 = e1, E = e1, Ei = e1;
    for (int i = 0; i < EV_ZC && zc + i < d.nz; ++i) {
      const int z = zc + i;
      const int l = d.z_layer[z];
      if (l != cur) {             // anchor: direct evaluation at layer entry / chunk start
        cur = l;
        const double2 kap = c[cix(d, f, n, l, C_KAP)];
        double2 amp, rho;
        layer_waves(d, f, n, l, amp, rho);
        if (fold) amp = sq_own * amp;
        if (z + 1 < d.nz && d.z_layer[z + 1] == l) {
          E = c[cix(d, f, n, l, C_E)];
          Ei = c[cix(d, f, n, l, C_EI)];
        }
        const double off = d.z_off[z];
        e1 = amp * cexp(cmk(-kap.y * off, kap.x * off));
        if (l < J - 1) {
          const double a = 2.0 * (d.layer_top[l + 1] - d.layer_top[l]) - off;
          e2 = (amp * rho) * cexp(cmk(-kap.y * a, kap.x * a));
        } else {
          e2 = cmk(0.0, 0.0);
        }
      } else {
        e1 = e1 * E;
        e2 = e2 * Ei;
      }
      tile[lane][i] = e1 + e2;
    }
  }
  __syncwarp();
  constexpr int RP = 32 / EV_ZC;                          // rows written together
  const int z = zc + lane % EV_ZC;
  for (int rr = 0; rr < 32; rr += RP) {
    const int nl = rr + lane / EV_ZC;
    const double sq = __shfl_sync(0xffffffffu, sq_own, nl);
    const long long r = r0 + nl;
    if (r < nrow && z < d.nz) {
      const double2 v = tile[nl][lane % EV_ZC];
      if (d.g64) d.g64[size_t(r) * d.nz + z] = v;
      if (d.g32) {
        // sqrt|s_f| g rounded to FP32, and (double-float table) the FP32 rounding of the rest
        const double sx = fold ? v.x : sq * v.x, sy = fold ? v.y : sq * v.y;
        const float hx = float(sx), hy = float(sy);
        const size_t o32 = size_t(r) * d.nzs + z;
        d.g32[o32] = make_float2(hx, hy);
        if (d.g32lo) d.g32lo[o32] = make_float2(float(sx - double(hx)), float(sy - double(hy)));
      }
    }
  }
}

// One CTA per table row (f, n), threads over depth; the row's largest |value| goes to rowmax
// (when present) for the FP16 operand scales of the Gram, so that no pass re-reads the table.
__global__ void __launch_bounds__(256) green_eval32_kernel(Dev d) {
  __shared__ float red[8];
  const long long fn = blockIdx.x;
  const int J = d.nlayer;
  const int f = int(fn / d.nk);
  const float sq = d.fc32_sqrt_s[f];
  float mx = 0.f;
  for (int z = threadIdx.x; z < d.nz; z += blockDim.x) {
    const int l = d.z_layer[z];
    const float4 zo = reinterpret_cast<const float4*>(d.z_off32)[z];   // off (hi, lo), 2h - off (hi, lo)
    const float4* c4 = reinterpret_cast<const float4*>(d.coef32 + (fn * J + l) * NCOEF32);
    const float4 k4 = c4[0], ar = c4[1];
    float2 e = expi_ff(k4.x, k4.y, k4.z, zo.x, zo.y);
    if (l < J - 1) {
      const float2 e2 = expi_ff(k4.x, k4.y, k4.z, zo.z, zo.w);
      e = e + make_float2(ar.z, ar.w) * e2;
    }
    const float2 g = make_float2(ar.x, ar.y) * e;
    const float2 v = make_float2(sq * g.x, sq * g.y);
    d.g32[size_t(fn) * d.nzs + z] = v;
    mx = fmaxf(mx, sqrtf(v.x * v.x + v.y * v.y));
  }
  if (!d.rowmax) return;                           // the same in the whole CTA
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < int(blockDim.x >> 5); ++w) mx = fmaxf(mx, red[w]);
    d.rowmax[fn] = mx;
  }
}

}  // namespace

int green_launches(const Dev& d, int tables) {
  if (tables == GREEN_COEF) return 2;
  if (tables == GREEN_G32F && d.nlayer <= COEF32_MAX_LAYERS) return 3;
  return tables == GREEN_G32 || tables == GREEN_G32F ? 4 : 3;
}

cudaError_t launch_green(const Dev& d, cudaStream_t s, int tables) {
  const bool fast32 = tables == GREEN_G32 || tables == GREEN_G32F;
  dim3 g1((d.nk + 127) / 128, d.nf);
  if (tables == GREEN_G32F && d.coef32 && d.nlayer <= COEF32_MAX_LAYERS) {
    const long long nl = (long long)d.nf * d.nk * d.nlayer;
    green_kap32_kernel<<<unsigned((nl + 255) / 256), 256, 0, s>>>(d);
    green_rec32_kernel<<<g1, 128, 0, s>>>(d);
  } else {
    const long long rows = (long long)d.nf * d.nk, nl = rows * d.nlayer;
    const int run = d.nlayer > 64 ? 4 : 1, steps = fast32 || tables == GREEN_COEF ? 0 : 1;
    const unsigned lb = unsigned((rows * ((d.nlayer + run - 1) / run) + LBLOCK - 1) / LBLOCK);
    if (run == 4) green_layer_kernel<4><<<lb, LBLOCK, 0, s>>>(d, steps);
    else green_layer_kernel<1><<<lb, LBLOCK, 0, s>>>(d, steps);
    // the split walks every layer twice (2 x 2 matrices, then the run): only for stacks of at
    // least four layers per run over too few (f, n) to fill the SMs' quarters (257 layers over 1056: an
    // inversion takes 0.37 ms, 0.70 with one lane; one and 16 lanes are what was measured)
    if (d.nlayer > 4 * 16 && rows < 32 * 304) green_recursion_kernel<16><<<unsigned((rows + 1) / 2), 32, 0, s>>>(d);
    else green_recursion_kernel<1><<<unsigned((rows + 31) / 32), 32, 0, s>>>(d);
    if (fast32) green_coef32_kernel<<<unsigned((nl + 127) / 128), 128, 0, s>>>(d);
  }
  if (tables == GREEN_COEF) return cudaGetLastError();
  if (fast32) {
    green_eval32_kernel<<<unsigned((long long)d.nf * d.nk), 256, 0, s>>>(d);
  } else {
    Dev e = d;
    if (!(tables & (GREEN_G32 | GREEN_G32DF))) e.g32 = nullptr;
    if (!(tables & GREEN_G32DF)) e.g32lo = nullptr;
    if (!(tables & GREEN_G64)) e.g64 = nullptr;
    const long long rows = (long long)d.nf * d.nk;
    const unsigned rb = unsigned((rows + 31) / 32);
    if ((long long)rb * ((d.nz + 15) / 16) < 608) green_eval64_kernel<4><<<dim3(rb, (d.nz + 3) / 4), 32, 0, s>>>(e);
    else green_eval64_kernel<16><<<dim3(rb, (d.nz + 15) / 16), 32, 0, s>>>(e);
  }
  return cudaGetLastError();
}

}  // namespace edt
