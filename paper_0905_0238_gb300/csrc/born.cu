// Spectral Born operator of the line geometry on the folded table index.
//
// The operator (eqs. DMV and M read forward) is F(p, q) = s_f sum_j g_p g_q Vhat(p - q) over the
// depths j, with g_n = g(|k_n|, z_j) even in n and Vhat(-m) = conj Vhat(m) for a real model.  The
// N^2 entries of a frequency plane therefore come from the pairs k >= l of the table index
// 0..H, H = N/2, eight entries to a pair.  With a = g_k g_l and the real sums' shorthand
//   P = sum a Re Vhat(k - l),  Q = sum a Im Vhat(k - l)   (complex times real: 4 multiply-adds)
//   P2, Q2 the same with Vhat(k + l),
//   F(k, l) = F(-l, -k) = s_f (P + iQ),      F(l, k) = F(-k, -l) = s_f (P - iQ),
//   F(k, -l) = F(l, -k) = s_f (P2 + iQ2),    F(-k, l) = F(-l, k) = s_f (P2 - iQ2),
// so a pair and depth take 12 multiply-adds where the eight entries one by one take 64 (complex
// a times complex Vhat each).  A pair with k = H has -k = k and needs P and Q only (edge
// kernels); l = 0 and k = l name some entries twice, with the same value.
//
// Three arithmetics of the same tile (32 x 32 pairs, 2 x 2 per thread, depths staged in shared
// memory 8 at a time):
//   F32   the misfit's residual (the FP32 table sqrt|s_f| g);
//   F64   the forward model of the FP64 path, bound by the FP64 unit;
//   DF    the forward model of the mixed path, FP64 table and sums carried as float pairs on
//         the FP32 pipes (an FP64 multiply-add costs 64 FP32 ones here).  Table rows are scaled by
//         powers of two to a 2-norm of at most 1 and Vhat rows to components of at most 1, so every
//         sum stays within 1 (Cauchy-Schwarz) and is accumulated on a bias C = 4: s keeps to [3, 5],
//         s - s' is exact for s' = fma(a, v, s), and fma(a, v, s - s') is the rounding error of s'
//         up to its own rounding to 24 bits; one multiply-add of pairs takes 6 FP32 operations
//         instead of the 12 of an unordered TwoSum.  The captured errors are summed in FP32 and carried
//         back into s after every 32 depths (3 operations), so that this sum stays within a few units
//         of C's last place, 2^-21.  The error of a sum is then that of some 3 nz roundings to 2^-45 or
//         finer: sqrt(nz) 2^-43 of the bound 1 is taken for it, whatever the sum itself comes to.
//
// The depth sums of a smooth model, or of a deep one under strong decay, come to far less than their
// bound.  The mixed forward model holds a plane's error to 2^-27 of its 2-norm, below the 1.2e-7 of
// the FP32 transforms behind it: every tile leaves the squares of its sums and of their bounds, and the planes
// whose ratio falls short (born_pick_kernel) are formed again in FP64 from the same pairs (49 bits of the
// FP64 table, as many as the march's rounding leaves right).  A Gaussian perturbation of 120 m in a
// homogeneous reference, 20 to 60 Hz: up to 1.1e-2 off by pairs alone, at most 1.9e-7 so.
//
// Measured at N = 512, 128 frequencies, 256 depths (GB300): the forward contraction 3.61 ms in DF, where
// the 512^2 entries one by one in FP64 took 153 ms (FP64-bound); the operation count (87 FP32
// operations per pair and depth) allows 2.3 ms.  The planes formed again take 0.23 ms each (30 ms for
// all 128); finding none takes 9 us.  Against a 64-bit restatement the data are 1.2e-7 to 1.6e-7 off: the
// FP32 transforms set the error.
//
// The gradients read the residual plane R2 (or the data plane) only through the sums over the
// entries of a class, so the residual kernel leaves, per pair, the folded values
//   E[k][l] = (S, S'),  S = R(k, l) + R(-l, -k),   S' = R(l, k) + R(-k, -l),
//   T[k][l] = (T, T'),  T = R(k, -l) + R(l, -k),   T' = R(-k, l) + R(-l, k),
// times conj(s_f)/|s_f|, for every ordered (k, l) (E[l][k] = (S', S), T[l][k] = (T, T')).
#include "edt_internal.h"
#include "cplx.cuh"
#include "dfloat.cuh"

namespace edt {

namespace {

constexpr int BT = 32, BZ = 8;              // pairs per tile side, depths per staged chunk
constexpr int BKS = BT + 1, BVS = 2 * BT + 1;   // odd rows: the transposing stores spread over banks
constexpr int BTHREADS = 256;
constexpr int BSETTLE = 4;                  // chunks after which the DF form's low sums are carried up

// ---- arithmetics -------------------------------------------------------------------------
struct ArF32 {
  using E = float2;                        // as staged
  using S = float2;                        // as stored
  __device__ __forceinline__ static E of(S v) { return v; }
  float s[8];
  __device__ __forceinline__ void init(float) {
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = 0.f;
  }
  __device__ __forceinline__ void mac(E k, E l, E v, E w) {
    const E a = k * l;
    s[0] = fmaf(a.x, v.x, s[0]); s[1] = fmaf(a.y, v.x, s[1]);
    s[2] = fmaf(a.x, v.y, s[2]); s[3] = fmaf(a.y, v.y, s[3]);
    s[4] = fmaf(a.x, w.x, s[4]); s[5] = fmaf(a.y, w.x, s[5]);
    s[6] = fmaf(a.x, w.y, s[6]); s[7] = fmaf(a.y, w.y, s[7]);
  }
  __device__ __forceinline__ void settle() {}
};

template <class Src> struct ArF64 {
  using E = double2;
  using S = Src;                           // doubles, or the pairs of the DF form
  __device__ __forceinline__ static E of(double2 v) { return v; }
  __device__ __forceinline__ static E of(float4 v) {
    return make_double2(double(v.x) + double(v.z), double(v.y) + double(v.w));
  }
  double s[8];
  __device__ __forceinline__ void init(float) {
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = 0.0;
  }
  __device__ __forceinline__ void mac(E k, E l, E v, E w) {
    const E a = k * l;
    s[0] = fma(a.x, v.x, s[0]); s[1] = fma(a.y, v.x, s[1]);
    s[2] = fma(a.x, v.y, s[2]); s[3] = fma(a.y, v.y, s[3]);
    s[4] = fma(a.x, w.x, s[4]); s[5] = fma(a.y, w.x, s[5]);
    s[6] = fma(a.x, w.y, s[6]); s[7] = fma(a.y, w.y, s[7]);
  }
  __device__ __forceinline__ void settle() {}
};

// complex pairs (re hi, im hi, re lo, im lo), scaled as above
constexpr float DF_BIAS = 4.f;
struct ArDF {
  using E = float4;
  using S = float4;
  __device__ __forceinline__ static E of(S v) { return v; }
  float s[8], lo[8];
  __device__ __forceinline__ void init(float) {
#pragma unroll
    for (int i = 0; i < 8; ++i) { s[i] = DF_BIAS; lo[i] = 0.f; }
  }
  // the low sums' high parts into s
  __device__ __forceinline__ void settle() {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float t = __fadd_rn(s[i], lo[i]);
      lo[i] = __fsub_rn(lo[i], __fsub_rn(t, s[i]));
      s[i] = t;
    }
  }
  __device__ __forceinline__ void acc(int i, float ah, float al, float vh, float vl) {
    const float t = fmaf(ah, vh, s[i]);
    const float e = fmaf(ah, vh, __fsub_rn(s[i], t));      // the rounding error of t, rounded
    s[i] = t;
    lo[i] = fmaf(al, vh, fmaf(ah, vl, __fadd_rn(lo[i], e)));
  }
  __device__ __forceinline__ void mac(E k, E l, E v, E w) {
    float2 ah, al;
    cmul_df(make_float2(k.x, k.y), make_float2(k.z, k.w), make_float2(l.x, l.y), make_float2(l.z, l.w), ah, al);
    acc(0, ah.x, al.x, v.x, v.z); acc(1, ah.y, al.y, v.x, v.z);
    acc(2, ah.x, al.x, v.y, v.w); acc(3, ah.y, al.y, v.y, v.w);
    acc(4, ah.x, al.x, w.x, w.z); acc(5, ah.y, al.y, w.x, w.z);
    acc(6, ah.x, al.x, w.y, w.w); acc(7, ah.y, al.y, w.y, w.w);
  }
};

template <class E> __device__ __forceinline__ E zero_of();
template <> __device__ __forceinline__ float2 zero_of<float2>() { return make_float2(0.f, 0.f); }
template <> __device__ __forceinline__ double2 zero_of<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float4 zero_of<float4>() { return make_float4(0.f, 0.f, 0.f, 0.f); }

// tile pair (tk >= tl) of the lower triangle, row-major
__device__ __forceinline__ void tile_of(int t, int& tk, int& tl) {
  tk = int((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
  while (tk * (tk + 1) / 2 > t) --tk;
  while ((tk + 1) * (tk + 2) / 2 <= t) ++tk;
  tl = t - tk * (tk + 1) / 2;
}
inline int tile_count(int H) { const int T = (H + BT - 1) / BT; return T * (T + 1) / 2; }

// A warp covers 8 x 4 pairs, so that each of its shared reads touches at most 11 consecutive
// elements; pair (a, b) of a thread is k = tx + 16 a, l = ty + 16 b.
__device__ __forceinline__ void thread_xy(int& tx, int& ty) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  tx = (w & 1) * 8 + (lane & 7);
  ty = (w >> 1) * 4 + (lane >> 3);
}

template <class E> constexpr size_t tile_smem() { return size_t(BZ) * (2 * BKS + 2 * BVS) * sizeof(E); }

// Sums of the tile's pairs over the depths.  g: table row n at g + n gs; v: Vhat row m at
// v + m vs.  Rows k, l >= H are not part of the tile (their pairs are not used).
template <class Ar>
__device__ __forceinline__ void fold_tile(const typename Ar::S* g, size_t gs, const typename Ar::S* v, size_t vs,
                                          int nz, int N, int k0, int l0, typename Ar::E* sm, Ar (&acc)[2][2]) {
  using E = typename Ar::E;
  E* sk = sm;                       // [BZ][BKS] rows k0 + i
  E* sl = sk + BZ * BKS;            // [BZ][BKS] rows l0 + i
  E* s1 = sl + BZ * BKS;            // [BZ][BVS] rows k0 - l0 - 31 + i
  E* s2 = s1 + BZ * BVS;            // [BZ][BVS] rows k0 + l0 + i
  const int H = N / 2, msk = N - 1;
  int tx, ty;
  thread_xy(tx, ty);
  const bool diag = k0 == l0;
  for (int z0 = 0; z0 < nz; z0 += BZ) {
    for (int e = threadIdx.x; e < BT * BZ; e += BTHREADS) {
      const int i = e / BZ, zz = e - i * BZ;
      const bool in = z0 + zz < nz;
      sk[zz * BKS + i] = in && k0 + i < H ? Ar::of(g[size_t(k0 + i) * gs + z0 + zz]) : zero_of<E>();
      sl[zz * BKS + i] = in && l0 + i < H ? Ar::of(g[size_t(l0 + i) * gs + z0 + zz]) : zero_of<E>();
    }
    for (int e = threadIdx.x; e < 2 * BT * BZ; e += BTHREADS) {
      const int i = e / BZ, zz = e - i * BZ;
      const bool in = z0 + zz < nz;
      s1[zz * BVS + i] = in ? Ar::of(v[size_t((k0 - l0 - (BT - 1) + i) & msk) * vs + z0 + zz]) : zero_of<E>();
      s2[zz * BVS + i] = in ? Ar::of(v[size_t((k0 + l0 + i) & msk) * vs + z0 + zz]) : zero_of<E>();
    }
    __syncthreads();
#pragma unroll 2
    for (int zz = 0; zz < BZ; ++zz) {
      E gk[2], gl[2], v1[3], v2[3];
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        gk[a] = sk[zz * BKS + tx + 16 * a];
        gl[a] = sl[zz * BKS + ty + 16 * a];
      }
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        v1[t] = s1[zz * BVS + tx - ty + 16 * (t - 1) + BT - 1];
        v2[t] = s2[zz * BVS + tx + ty + 16 * t];
      }
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
          if (!(diag && a < b)) acc[a][b].mac(gk[a], gl[b], v1[a - b + 1], v2[a + b]);   // a < b: k < l
    }
    if ((z0 / BZ) % BSETTLE == BSETTLE - 1) {
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) acc[a][b].settle();
    }
    __syncthreads();
  }
}

// ---- preparation of the double-float forward model ---------------------------------------
// One row of nz <= 256 FP64 complex values per warp, replaced in place by float pairs of
// value * c * 2^-e; e goes to exps[row].  Green's table (per_f rows to a frequency): the row's 2-norm in
// [1/2, 1), c = sqrt(s_f) = omega~ sqrt(dz/dx), so the products carry s_f.  Vhat (per_f = 0): the largest
// component in [1/2, 1), c = 1.
constexpr int PREP_THREADS = 128, PREP_Q = 8;
__global__ void __launch_bounds__(PREP_THREADS) born_prep_kernel(Dev d, double2* rows, long long nrow, int per_f, int* exps) {
  const int lane = threadIdx.x & 31;
  const long long row = (long long)blockIdx.x * (PREP_THREADS / 32) + (threadIdx.x >> 5);
  if (row >= nrow) return;
  double2 c = make_double2(1.0, 0.0);
  if (per_f) {
    const FreqConst fc = d.fc[row / per_f];
    const double q = sqrt(d.dz / d.dx);
    c = make_double2(q * fc.om_re, q * fc.om_im);
  }
  double2* r = rows + size_t(row) * d.nz;
  double2 v[PREP_Q];
  int e = -1022;
#pragma unroll
  for (int i = 0; i < PREP_Q; ++i) {
    const int z = lane + 32 * i;
    v[i] = z < d.nz ? r[z] : make_double2(0.0, 0.0);
  }
#pragma unroll
  for (int i = 0; i < PREP_Q; ++i) {
    if (per_f) v[i] = c * v[i];
    e = max(e, exp_above(v[i]));
  }
  e = max(-1000, min(1000, __reduce_max_sync(0xffffffffu, e)));
  const double sc = __hiloint2double((1023 - e) << 20, 0);                  // 2^-e
  float4 o[PREP_Q];
  float q = 0.f;
#pragma unroll
  for (int i = 0; i < PREP_Q; ++i) {
    const double x = v[i].x * sc, y = v[i].y * sc;
    const float xh = float(x), yh = float(y);
    o[i] = make_float4(xh, yh, float(x - double(xh)), float(y - double(yh)));
    q = fmaf(xh, xh, fmaf(yh, yh, q));
  }
  float un = 1.f;
  if (per_f) {
    for (int w = 16; w > 0; w >>= 1) q += __shfl_xor_sync(0xffffffffu, q, w);
    int en = 0;
    if (q > 0.f && isfinite(q)) frexpf(sqrtf(q), &en);
    e += en;
    un = __int_as_float((127 - en) << 23);                                  // 2^-en
  }
#pragma unroll
  for (int i = 0; i < PREP_Q; ++i) {
    const int z = lane + 32 * i;
    if (z < d.nz) reinterpret_cast<float4*>(r)[z] = make_float4(un * o[i].x, un * o[i].y, un * o[i].z, un * o[i].w);
  }
  if (lane == 0) exps[row] = e;
}

// Vhat for the misfit: FP32 in place (row m's float2 values at the start of its FP64 row), all of it
// times one power of two 2^-e with the largest component just under 1, e in exps[0].  The products
// residual x Vhat x table then neither vanish nor overflow where their sum does not: with Vhat as it
// is, dJ/dc lost digits for models and data 1e-17 of the usual size and was not finite at 1e20 times.
__global__ void __launch_bounds__(PREP_THREADS) born_v32_kernel(Dev d, const int* tile, int ntile, int* exps) {
  static_assert(PREP_THREADS == 128, "four warps");
  __shared__ int red[PREP_THREADS / 32];
  constexpr int Q = 2;                  // nz <= 256
  double2* r = d.vfull + size_t(blockIdx.x) * d.nz;
  double2 v[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int z = threadIdx.x + PREP_THREADS * i;
    v[i] = z < d.nz ? r[z] : make_double2(0.0, 0.0);
  }
  int e = -1022;
  for (int i = threadIdx.x; i < ntile; i += PREP_THREADS) e = max(e, tile[i]);
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
  __syncthreads();                      // and every element of the row has been read
  // a factor that stays normal in FP32 on either side; values beyond it have their own rounding
  e = max(-100, min(100, max(max(red[0], red[1]), max(red[2], red[3]))));
  const double sc = __hiloint2double((1023 - e) << 20, 0);                  // 2^-e
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int z = threadIdx.x + PREP_THREADS * i;
    if (z < d.nz) reinterpret_cast<float2*>(r)[z] = make_float2(float(sc * v[i].x), float(sc * v[i].y));
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) exps[0] = e;
}

// ---- forward model -----------------------------------------------------------------------
// one rounding of (xh + xl) + sg (yh + yl), scaled by 2^e
__device__ __forceinline__ float df_comb(float xh, float xl, float yh, float yl, float sg, int e) {
  const float2 t = two_sum(xh, sg * yh);
  return ldexpf(t.x + (t.y + (xl + sg * yl)), e);
}
// f1 = A + iB, f2 = A - iB for A = (s[o], s[o+1]), B = (s[o+2], s[o+3])
__device__ __forceinline__ void df_result(const ArDF& a, int o, int e, float2& f1, float2& f2) {
  const float a0 = a.s[o] - DF_BIAS, a1 = a.s[o + 1] - DF_BIAS, b0 = a.s[o + 2] - DF_BIAS, b1 = a.s[o + 3] - DF_BIAS;
  f1 = make_float2(df_comb(a0, a.lo[o], b1, a.lo[o + 3], -1.f, e), df_comb(a1, a.lo[o + 1], b0, a.lo[o + 2], 1.f, e));
  f2 = make_float2(df_comb(a0, a.lo[o], b1, a.lo[o + 3], 1.f, e), df_comb(a1, a.lo[o + 1], b0, a.lo[o + 2], -1.f, e));
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < nw; ++i) t += red[i];
  return t;
}

// the eight entries of pair (k, l): f1, f2 of k - l, h1, h2 of k + l
template <class T2>
__device__ __forceinline__ void put_pair(T2* X, int N, int k, int l, T2 f1, T2 f2, T2 h1, T2 h2) {
  const int msk = N - 1, nk_ = (N - k) & msk, nl_ = (N - l) & msk;
  X[size_t(l) * N + k] = f1;
  X[size_t(nk_) * N + nl_] = f1;
  X[size_t(k) * N + l] = f2;
  X[size_t(nl_) * N + nk_] = f2;
  X[size_t(nl_) * N + k] = h1;
  X[size_t(nk_) * N + l] = h1;
  X[size_t(l) * N + nk_] = h2;
  X[size_t(k) * N + nl_] = h2;
}
// the four of (H, l)
template <class T2>
__device__ __forceinline__ void put_edge(T2* X, int N, int l, T2 f1, T2 f2) {
  const int H = N / 2, nl_ = (N - l) & (N - 1);
  X[size_t(l) * N + H] = f1;
  X[size_t(H) * N + nl_] = f1;
  X[size_t(H) * N + l] = f2;
  X[size_t(nl_) * N + H] = f2;
}

// X[fi][q][p] = F(p, q) for the pairs of one tile (mixed path: FP32 planes), and into born_part[fi][tile]
// the sums over its entries of |F|^2 and of the squared bounds 2^e of F
__global__ void __launch_bounds__(BTHREADS, 2) born_fwd_df_kernel(Dev d, int f0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ float2 red[BTHREADS / 32];
  __shared__ int emax[BTHREADS / 32];
  const int N = d.N, H = N / 2, msk = N - 1, fi = blockIdx.y, f = f0 + fi;
  int tk, tl;
  tile_of(blockIdx.x, tk, tl);
  const int k0 = tk * BT, l0 = tl * BT;
  ArDF acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b].init(0.f);
  fold_tile<ArDF>(reinterpret_cast<const float4*>(d.g64) + size_t(f) * d.nk * d.nz, d.nz,
                  reinterpret_cast<const float4*>(d.vfull), d.nz, d.nz, N, k0, l0,
                  reinterpret_cast<float4*>(smem_raw), acc);
  int tx, ty;
  thread_xy(tx, ty);
  float2* X = reinterpret_cast<float2*>(d.X) + size_t(fi) * N * N;
  const int* eg = d.born_exp + size_t(f) * d.nk;
  const int* ev = d.born_exp + size_t(d.nf) * d.nk;
  // the tile's largest exponent, to which its squares are scaled
  int em = -4000;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int k = k0 + tx + 16 * a, l = l0 + ty + 16 * b;
      if (k < H && l <= k) em = max(em, eg[k] + eg[l] + max(ev[(k - l) & msk], ev[(k + l) & msk]));
    }
  em = __reduce_max_sync(0xffffffffu, em);
  if ((threadIdx.x & 31) == 0) emax[threadIdx.x >> 5] = em;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < BTHREADS / 32; ++w) em = max(em, emax[w]);
  float sf = 0.f, sb = 0.f;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int k = k0 + tx + 16 * a, l = l0 + ty + 16 * b;
      if (k >= H || l > k) continue;
      const int e = eg[k] + eg[l], e1 = e + ev[(k - l) & msk], e2 = e + ev[(k + l) & msk];
      const float w1 = exp2f(float(max(-120, 2 * (e1 - em)))), w2 = exp2f(float(max(-120, 2 * (e2 - em))));
      float q[2] = {0.f, 0.f};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float x = acc[a][b].s[i] - DF_BIAS + acc[a][b].lo[i];
        q[i / 4] = fmaf(x, x, q[i / 4]);
      }
      sf = fmaf(w1, q[0], fmaf(w2, q[1], sf));
      sb += w1 + w2;
      float2 f1, f2, h1, h2;
      df_result(acc[a][b], 0, e1, f1, f2);
      df_result(acc[a][b], 4, e2, h1, h2);
      put_pair(X, N, k, l, f1, f2, h1, h2);
    }
  for (int o = 16; o > 0; o >>= 1) {
    sf += __shfl_down_sync(0xffffffffu, sf, o);
    sb += __shfl_down_sync(0xffffffffu, sb, o);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float2(sf, sb);
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < BTHREADS / 32; ++w) { sf += red[w].x; sb += red[w].y; }
    d.born_part[size_t(fi) * gridDim.x + blockIdx.x] = make_float4(sf, sb, __int_as_float(em), 0.f);
  }
}

__global__ void __launch_bounds__(BTHREADS, 2) born_fwd_f64_kernel(Dev d, int f0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = d.N, H = N / 2, fi = blockIdx.y, f = f0 + fi;
  int tk, tl;
  tile_of(blockIdx.x, tk, tl);
  const int k0 = tk * BT, l0 = tl * BT;
  ArF64<double2> acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b].init(0.f);
  fold_tile<ArF64<double2>>(d.g64 + size_t(f) * d.nk * d.nz, d.nz, d.vfull, d.nz, d.nz, N, k0, l0,
                   reinterpret_cast<double2*>(smem_raw), acc);
  int tx, ty;
  thread_xy(tx, ty);
  double2* X = reinterpret_cast<double2*>(d.X) + size_t(fi) * N * N;
  const FreqConst fc = d.fc[f];
  const double2 om = make_double2(fc.om_re, fc.om_im), sf = (d.dz / d.dx) * (om * om);
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int k = k0 + tx + 16 * a, l = l0 + ty + 16 * b;
      if (k >= H || l > k) continue;
      const double* s = acc[a][b].s;
      put_pair(X, N, k, l, sf * make_double2(s[0] - s[3], s[1] + s[2]), sf * make_double2(s[0] + s[3], s[1] - s[2]),
               sf * make_double2(s[4] - s[7], s[5] + s[6]), sf * make_double2(s[4] + s[7], s[5] - s[6]));
    }
}

// Pairs (H, l), l = 0..H: one warp per (plane, l), lanes over the depths.
// F(H, l) = F(-l, H) = s_f (P + iQ), F(l, H) = F(H, -l) = s_f (P - iQ).
template <typename T> struct EdgeSum;
template <> struct EdgeSum<float> {                       // double-float partial sums
  float2 s[4];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < 4; ++i) s[i] = make_float2(0.f, 0.f);
  }
  __device__ __forceinline__ void mac(float4 k, float4 l, float4 v) {
    float2 ah, al;
    cmul_df(make_float2(k.x, k.y), make_float2(k.z, k.w), make_float2(l.x, l.y), make_float2(l.z, l.w), ah, al);
    const float2 ar = make_float2(ah.x, al.x), ai = make_float2(ah.y, al.y);
    df_acc(s[0], ar, make_float2(v.x, v.z)); df_acc(s[1], ai, make_float2(v.x, v.z));
    df_acc(s[2], ar, make_float2(v.y, v.w)); df_acc(s[3], ai, make_float2(v.y, v.w));
  }
  __device__ __forceinline__ void warp_sum() {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s[i] = df_norm(s[i]);
      for (int o = 16; o > 0; o >>= 1)
        s[i] = df_add(s[i], make_float2(__shfl_xor_sync(0xffffffffu, s[i].x, o), __shfl_xor_sync(0xffffffffu, s[i].y, o)));
    }
  }
};

__global__ void __launch_bounds__(256) born_fwd_edge_df_kernel(Dev d, int f0) {
  const int N = d.N, H = N / 2, lane = threadIdx.x & 31;
  const int l = blockIdx.x * 8 + (threadIdx.x >> 5), fi = blockIdx.y, f = f0 + fi;
  if (l > H) return;
  const float4* g = reinterpret_cast<const float4*>(d.g64) + size_t(f) * d.nk * d.nz;
  const float4* v = reinterpret_cast<const float4*>(d.vfull) + size_t(H - l) * d.nz;
  EdgeSum<float> a;
  a.init();
  for (int z = lane; z < d.nz; z += 32) a.mac(g[size_t(H) * d.nz + z], g[size_t(l) * d.nz + z], v[z]);
  a.warp_sum();
  if (lane != 0) return;
  const int e = d.born_exp[size_t(f) * d.nk + H] + d.born_exp[size_t(f) * d.nk + l] +
                d.born_exp[size_t(d.nf) * d.nk + (H - l)];
  auto out = [&](float2 x, float2 y, float sg) { return df_comb(x.x, x.y, y.x, y.y, sg, e); };
  const float2 f1 = make_float2(out(a.s[0], a.s[3], -1.f), out(a.s[1], a.s[2], 1.f));
  const float2 f2 = make_float2(out(a.s[0], a.s[3], 1.f), out(a.s[1], a.s[2], -1.f));
  put_edge(reinterpret_cast<float2*>(d.X) + size_t(fi) * N * N, N, l, f1, f2);
}

// sums over the depths of a (H, l) pair by a warp: (P, Q) in every lane
template <class Src>
__device__ __forceinline__ void edge_sums(const Src* gh, const Src* gl, const Src* v, int nz, int lane, double2& p, double2& q) {
  using A = ArF64<Src>;
  p = q = make_double2(0.0, 0.0);
  for (int z = lane; z < nz; z += 32) {
    const double2 a = A::of(gh[z]) * A::of(gl[z]), b = A::of(v[z]);
    p = p + b.x * a;
    q = q + b.y * a;
  }
  for (int o = 16; o > 0; o >>= 1) {
    p.x += __shfl_xor_sync(0xffffffffu, p.x, o); p.y += __shfl_xor_sync(0xffffffffu, p.y, o);
    q.x += __shfl_xor_sync(0xffffffffu, q.x, o); q.y += __shfl_xor_sync(0xffffffffu, q.y, o);
  }
}

__global__ void __launch_bounds__(256) born_fwd_edge_f64_kernel(Dev d, int f0) {
  const int N = d.N, H = N / 2, lane = threadIdx.x & 31;
  const int l = blockIdx.x * 8 + (threadIdx.x >> 5), fi = blockIdx.y, f = f0 + fi;
  if (l > H) return;
  const double2* g = d.g64 + size_t(f) * d.nk * d.nz;
  double2 p, q;
  edge_sums(g + size_t(H) * d.nz, g + size_t(l) * d.nz, d.vfull + size_t(H - l) * d.nz, d.nz, lane, p, q);
  if (lane != 0) return;
  const FreqConst fc = d.fc[f];
  const double2 om = make_double2(fc.om_re, fc.om_im), sf = (d.dz / d.dx) * (om * om);
  put_edge(reinterpret_cast<double2*>(d.X) + size_t(fi) * N * N, N, l, sf * make_double2(p.x - q.y, p.y + q.x),
           sf * make_double2(p.x + q.y, p.y - q.x));
}

// flags of the planes to form again, behind the partial sums
__device__ __forceinline__ int* redo_flags(const Dev& d, int ntile) {
  return reinterpret_cast<int*>(d.born_part + size_t(d.fchunk) * ntile);
}

// Flags plane fi if its sums by pairs are not 2^-27 of the plane accurate: their sum of squares falls
// below (sqrt(nz) 2^-43 2^27)^2 times that of the bounds.  One warp per plane.
__global__ void __launch_bounds__(32) born_pick_kernel(Dev d, int ntile) {
  const int fi = blockIdx.x, lane = threadIdx.x;
  const float4* part = d.born_part + size_t(fi) * ntile;
  int em = -4000;
  for (int i = lane; i < ntile; i += 32) em = max(em, __float_as_int(part[i].z));
  em = __reduce_max_sync(0xffffffffu, em);
  float sf = 0.f, sb = 0.f;
  for (int i = lane; i < ntile; i += 32) {
    const float4 p = part[i];
    const float w = exp2f(float(max(-120, 2 * (__float_as_int(p.z) - em))));
    sf = fmaf(w, p.x, sf);
    sb = fmaf(w, p.y, sb);
  }
  for (int o = 16; o > 0; o >>= 1) {
    sf += __shfl_xor_sync(0xffffffffu, sf, o);
    sb += __shfl_xor_sync(0xffffffffu, sb, o);
  }
  if (lane == 0) redo_flags(d, ntile)[fi] = !(sf >= float(d.nz) * 0x1p-32f * sb);
}

// These planes in FP64.  CTAs below ntile take a tile, the others eight edge pairs, of every
// gridDim.y-th of the planes.
__device__ __forceinline__ void redo_part(const Dev& d, int f0, int fi, int ntile, double2* sm) {
  const int N = d.N, H = N / 2, msk = N - 1, f = f0 + fi;
  const float4* g = reinterpret_cast<const float4*>(d.g64) + size_t(f) * d.nk * d.nz;
  const float4* v = reinterpret_cast<const float4*>(d.vfull);
  const int* eg = d.born_exp + size_t(f) * d.nk;
  const int* ev = d.born_exp + size_t(d.nf) * d.nk;
  float2* X = reinterpret_cast<float2*>(d.X) + size_t(fi) * N * N;
  auto out = [](double x, double y, int e) { return make_float2(float(scalbn(x, e)), float(scalbn(y, e))); };
  if (int(blockIdx.x) >= ntile) {
    const int l = (int(blockIdx.x) - ntile) * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (l > H) return;
    double2 p, q;
    edge_sums(g + size_t(H) * d.nz, g + size_t(l) * d.nz, v + size_t(H - l) * d.nz, d.nz, lane, p, q);
    if (lane != 0) return;
    const int e = eg[H] + eg[l] + ev[H - l];
    put_edge(X, N, l, out(p.x - q.y, p.y + q.x, e), out(p.x + q.y, p.y - q.x, e));
    return;
  }
  int tk, tl;
  tile_of(blockIdx.x, tk, tl);
  const int k0 = tk * BT, l0 = tl * BT;
  ArF64<float4> acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b].init(0.f);
  fold_tile<ArF64<float4>>(g, d.nz, v, d.nz, d.nz, N, k0, l0, sm, acc);
  int tx, ty;
  thread_xy(tx, ty);
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int k = k0 + tx + 16 * a, l = l0 + ty + 16 * b;
      if (k >= H || l > k) continue;
      const int e = eg[k] + eg[l], e1 = e + ev[(k - l) & msk], e2 = e + ev[(k + l) & msk];
      const double* s = acc[a][b].s;
      put_pair(X, N, k, l, out(s[0] - s[3], s[1] + s[2], e1), out(s[0] + s[3], s[1] - s[2], e1),
               out(s[4] - s[7], s[5] + s[6], e2), out(s[4] + s[7], s[5] - s[6], e2));
    }
}

constexpr int REDO_Y = 8;
__global__ void __launch_bounds__(BTHREADS, 2) born_redo_kernel(Dev d, int f0, int nfc, int ntile) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31;
  const int* flag = redo_flags(d, ntile);
  int n = 0;                                 // planes met so far
  for (int b = 0; b < nfc; b += 32) {
    unsigned m = __ballot_sync(0xffffffffu, b + lane < nfc && flag[b + lane]);
    for (; m; m &= m - 1, ++n)
      if (n % REDO_Y == int(blockIdx.y)) redo_part(d, f0, b + __ffs(m) - 1, ntile, reinterpret_cast<double2*>(smem_raw));
  }
}

// ---- residual and folding ----------------------------------------------------------------
__device__ __forceinline__ float4 pack2(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }

// Sum of squares as a float pair times 2^(2 e), e the largest exponent met: the squares of FP32 values
// leave the FP32 range long before their FP64 sum would.
struct SumSq {
  float2 acc = make_float2(0.f, 0.f);
  int e = -126;
  __device__ __forceinline__ static float pow2(int n) { return __int_as_float((127 + n) << 23); }   // |n| <= 126
  // w1 times the squares of the first half of r, w2 times those of the second (powers of two)
  template <int K>
  __device__ __forceinline__ void add(const float2 (&r)[K], float w1, float w2) {
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < K; ++i) m = fmaxf(m, fmaxf(fabsf(r[i].x), fabsf(r[i].y)));
    const int en = min(126, (__float_as_int(m) >> 23) - 126);
    if (en > e) {
      const float k = pow2(max(e - en, -126));
      acc = k * (k * acc);
      e = en;
    }
    const float sc = pow2(-e);
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const float w = i < K / 2 ? w1 : w2, x = sc * r[i].x, y = sc * r[i].y;
      df_acc(acc, make_float2(w * x, 0.f), make_float2(x, 0.f));
      df_acc(acc, make_float2(w * y, 0.f), make_float2(y, 0.f));
    }
  }
  __device__ __forceinline__ double value() const {
    // (an infinite sum: its error terms are NaN)
    return (isfinite(acc.x) ? df_val(acc) : double(acc.x)) * __hiloint2double((1023 + 2 * e) << 20, 0);
  }
};

// RES: R = F - D2 with the FP32 table and Vhat, sum |R|^2 into gacc[0] and R folded;
// else R = D2 (the adjoint operator).  X[fi][q][p] = D2(p, q) is only read.
template <bool RES>
__global__ void __launch_bounds__(BTHREADS, 3) born_resid_kernel(Dev d, int f0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[BTHREADS / 32];
  const int N = d.N, H = N / 2, msk = N - 1, nk = d.nk, fi = blockIdx.y, f = f0 + fi;
  int tk, tl;
  tile_of(blockIdx.x, tk, tl);
  const int k0 = tk * BT, l0 = tl * BT;
  ArF32 acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b].init(0.f);
  if (RES)
    fold_tile<ArF32>(d.g32 + size_t(f) * nk * d.nzs, d.nzs, reinterpret_cast<const float2*>(d.vfull),
                     2 * size_t(d.nz), d.nz, N, k0, l0, reinterpret_cast<float2*>(smem_raw), acc);
  int tx, ty;
  thread_xy(tx, ty);
  const float2* X = reinterpret_cast<const float2*>(d.X) + size_t(fi) * N * N;
  float4* E = d.born_fold + size_t(fi) * 2 * nk * nk;
  float4* T = E + size_t(nk) * nk;
  const FreqConst fc = d.fc[f];
  const float2 rot = make_float2(float(fc.rot_re), float(fc.rot_im));   // conj(s_f) / |s_f|
  const float ve = RES ? __int_as_float((127 + d.born_exp[0]) << 23) : 1.f;      // the scale of Vhat
  SumSq jp;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int k = k0 + tx + 16 * a, l = l0 + ty + 16 * b;
      if (k >= H || l > k) continue;
      const int nk_ = (N - k) & msk, nl_ = (N - l) & msk;
      float2 r[8] = {X[size_t(l) * N + k],   X[size_t(nk_) * N + nl_], X[size_t(k) * N + l],   X[size_t(nl_) * N + nk_],
                     X[size_t(nl_) * N + k], X[size_t(nk_) * N + l],   X[size_t(l) * N + nk_], X[size_t(k) * N + nl_]};
      if (RES) {
        const float2 ph = cconj(rot);
        const float* s = acc[a][b].s;
        const float2 f1 = ve * (ph * make_float2(s[0] - s[3], s[1] + s[2]));
        const float2 f2 = ve * (ph * make_float2(s[0] + s[3], s[1] - s[2]));
        const float2 h1 = ve * (ph * make_float2(s[4] - s[7], s[5] + s[6]));
        const float2 h2 = ve * (ph * make_float2(s[4] + s[7], s[5] - s[6]));
        r[0] = f1 - r[0]; r[1] = f1 - r[1]; r[2] = f2 - r[2]; r[3] = f2 - r[3];
        r[4] = h1 - r[4]; r[5] = h1 - r[5]; r[6] = h2 - r[6]; r[7] = h2 - r[7];
        // every distinct entry once: l = 0 names its entries twice, k = l the two of each kind
        const float w1 = k == l ? (l == 0 ? 0.25f : 0.5f) : 1.f, w2 = l == 0 ? 0.f : w1;
        jp.add(r, w1, w2);
      }
      const float2 S = rot * (r[0] + r[1]), S2 = rot * (r[2] + r[3]);
      const float2 U = rot * (r[4] + r[5]), U2 = rot * (r[6] + r[7]);
      E[size_t(k) * nk + l] = pack2(S, S2);
      E[size_t(l) * nk + k] = pack2(S2, S);
      T[size_t(k) * nk + l] = pack2(U, U2);
      T[size_t(l) * nk + k] = pack2(U, U2);
    }
  if (RES) {
    const double t = block_sum(jp.value(), red);
    if (threadIdx.x == 0) atomicAdd(d.gacc, t);
  }
}

// the pairs (H, l): E[H][l], E[l][H] and T[H][l] = E[l][H] (the entries of -l against H = -H)
template <bool RES>
__global__ void __launch_bounds__(256) born_resid_edge_kernel(Dev d, int f0) {
  __shared__ double red[8];
  const int N = d.N, H = N / 2, msk = N - 1, nk = d.nk, lane = threadIdx.x & 31;
  const int l = blockIdx.x * 8 + (threadIdx.x >> 5), fi = blockIdx.y, f = f0 + fi;
  double jp = 0.0;
  if (l <= H) {
    float2 p = make_float2(0.f, 0.f), q = p;
    if (RES) {
      const float2* g = d.g32 + size_t(f) * nk * d.nzs;
      const float2* v = reinterpret_cast<const float2*>(d.vfull) + size_t(H - l) * 2 * d.nz;
      for (int z = lane; z < d.nz; z += 32) {
        const float2 a = g[size_t(H) * d.nzs + z] * g[size_t(l) * d.nzs + z], b = v[z];
        p.x = fmaf(a.x, b.x, p.x); p.y = fmaf(a.y, b.x, p.y);
        q.x = fmaf(a.x, b.y, q.x); q.y = fmaf(a.y, b.y, q.y);
      }
      for (int o = 16; o > 0; o >>= 1) {
        p.x += __shfl_xor_sync(0xffffffffu, p.x, o); p.y += __shfl_xor_sync(0xffffffffu, p.y, o);
        q.x += __shfl_xor_sync(0xffffffffu, q.x, o); q.y += __shfl_xor_sync(0xffffffffu, q.y, o);
      }
    }
    if (lane == 0) {
      const float2* X = reinterpret_cast<const float2*>(d.X) + size_t(fi) * N * N;
      const FreqConst fc = d.fc[f];
      const float2 rot = make_float2(float(fc.rot_re), float(fc.rot_im));
      const int nl_ = (N - l) & msk;
      float2 r[4] = {X[size_t(l) * N + H], X[size_t(H) * N + nl_], X[size_t(H) * N + l], X[size_t(nl_) * N + H]};
      if (RES) {
        const float2 ph = cconj(rot);
        const float ve = __int_as_float((127 + d.born_exp[0]) << 23);            // the scale of Vhat
        const float2 f1 = ve * (ph * make_float2(p.x - q.y, p.y + q.x));
        const float2 f2 = ve * (ph * make_float2(p.x + q.y, p.y - q.x));
        r[0] = f1 - r[0]; r[1] = f1 - r[1]; r[2] = f2 - r[2]; r[3] = f2 - r[3];
        const float w = l == 0 ? 0.5f : (l == H ? 0.25f : 1.f);
        SumSq sq;
        sq.add(r, w, w);
        jp = sq.value();
      }
      float4* E = d.born_fold + size_t(fi) * 2 * nk * nk;
      float4* T = E + size_t(nk) * nk;
      const float2 S = rot * (r[0] + r[1]), S2 = rot * (r[2] + r[3]);
      E[size_t(H) * nk + l] = pack2(S, S2);
      E[size_t(l) * nk + H] = pack2(S2, S);
      T[size_t(H) * nk + l] = pack2(S2, S);
    }
  }
  if (RES) {
    const double t = block_sum(jp, red);
    if (threadIdx.x == 0) atomicAdd(d.gacc, t);
  }
}

}  // namespace

// elements of one plane in born_part
int born_tiles(int N) { return tile_count(N / 2); }

cudaError_t prepare_born() {
  cudaError_t e = allow_smem(born_fwd_df_kernel, int(tile_smem<float4>()));
  if (e != cudaSuccess) return e;
  if ((e = allow_smem(born_fwd_f64_kernel, int(tile_smem<double2>()))) != cudaSuccess) return e;
  return allow_smem(born_redo_kernel, int(tile_smem<double2>()));
}

cudaError_t launch_born_prep(const Dev& d, cudaStream_t s) {
  constexpr int W = PREP_THREADS / 32;
  const long long rows = (long long)d.nf * d.nk;
  born_prep_kernel<<<unsigned((rows + W - 1) / W), PREP_THREADS, 0, s>>>(d, d.g64, rows, d.nk, d.born_exp);
  born_prep_kernel<<<(d.N + W - 1) / W, PREP_THREADS, 0, s>>>(d, d.vfull, d.N, 0, d.born_exp + rows);
  return cudaGetLastError();
}

int* born_v32_exps(const Dev& d) { return d.born_exp + 1; }

cudaError_t launch_born_v32(const Dev& d, cudaStream_t s) {
  born_v32_kernel<<<d.N, PREP_THREADS, 0, s>>>(d, born_v32_exps(d), lateral_tiles(d.nz), d.born_exp);
  return cudaGetLastError();
}

cudaError_t launch_born_forward(const Dev& d, int f0, int nfc, cudaStream_t s) {
  const dim3 g(tile_count(d.N / 2), nfc), ge((d.nk + 7) / 8, nfc);
  if (d.precision == EDT_FP64) {
    born_fwd_f64_kernel<<<g, BTHREADS, tile_smem<double2>(), s>>>(d, f0);
    born_fwd_edge_f64_kernel<<<ge, 256, 0, s>>>(d, f0);
  } else {
    born_fwd_df_kernel<<<g, BTHREADS, tile_smem<float4>(), s>>>(d, f0);
    born_fwd_edge_df_kernel<<<ge, 256, 0, s>>>(d, f0);
    born_pick_kernel<<<nfc, 32, 0, s>>>(d, int(g.x));
    born_redo_kernel<<<dim3(g.x + ge.x, REDO_Y), BTHREADS, tile_smem<double2>(), s>>>(d, f0, nfc, int(g.x));
  }
  return cudaGetLastError();
}

cudaError_t launch_born_residual(const Dev& d, int f0, int nfc, bool model, cudaStream_t s) {
  const dim3 g(tile_count(d.N / 2), nfc), ge((d.nk + 7) / 8, nfc);
  if (model) {
    born_resid_kernel<true><<<g, BTHREADS, tile_smem<float2>(), s>>>(d, f0);
    born_resid_edge_kernel<true><<<ge, 256, 0, s>>>(d, f0);
  } else {
    born_resid_kernel<false><<<g, BTHREADS, 0, s>>>(d, f0);
    born_resid_edge_kernel<false><<<ge, 256, 0, s>>>(d, f0);
  }
  return cudaGetLastError();
}

}  // namespace edt
