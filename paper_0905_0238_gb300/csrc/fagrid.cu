// Kernel rows of the window geometry on a grid (nx = ny = N): for every kept row (f, j) of a pair
// {k, -k} and every depth z
//   M(k; j) = c_f sum_w e^{-2 pi i j.w/W} F_w(k),   F_w(k) = sum_y e^{i k.y} P_w(y),
//   P_w(y)  = G(y - w) G(y + w)
// (csrc/fa.cu derives the rows; there the window sum comes first, here the transform over y).
// G is even in each coordinate, so with |w| = (a, b)
//   F_{-w}(k) = F_w(k) = F_w(-k),   F_{(-a, b)}(kx, ky) = F_{(a, b)}(-kx, ky):
// the planes of the (WX/2 + 1)(WY/2 + 1) windows a, b >= 0 hold them all, against one plane per active
// j (up to WX WY) when the window sum is taken first, and where the spacings and the window are the same
// in x and y, F_{(b, a)}(ky, kx) = F_{(a, b)}(kx, ky) leaves only a >= b.  With
//   E_ab = F_ab(kx, ky) + F_ab(-kx, ky),   O_ab = F_ab(kx, ky) - F_ab(-kx, ky)
// (twice the even and odd parts), h = (WX/2, WY/2) and s = sign, the window sum is
//   2 M(+-kx, ky; j) = A(|jx|, |jy|) +- [ -s(jx) s(jy) B(|jx|, |jy|) + i (-1)^jy s(jx) X(|jx|)
//                                         + i (-1)^jx s(jy) Y(|jy|) + (-1)^(jx + jy) O_hh ],
// A the cosine transform of E in both directions (ends weighted 1, the rest 2), B the sine transform of
// O over 0 < a < hx, 0 < b < hy, X that of O_{a, hy} over a, Y that of O_{hx, b} over b (the window's
// end -h has no partner +h; s(0) = s(-h) = 0).  Both pairs (kx, ky), (-kx, ky) share the transforms.
// Against the window sum first (per offset wavenumber j: products, 16-point transforms and one plane
// FFT), at 128 x 128 midpoints, 16 x 16 half-offsets, 64 frequencies and 200 depths: 45 planes per
// (f, z) instead of 138 on average, 46 ms of kernels instead of 144; 64 x 64, 8 x 8, 12 frequencies, 100
// depths: 0.55 ms instead of 1.36.
// Per frequency, for all depths at once (slabs of depths whose planes stay in L2 lost more to short
// launches than they saved: 134 ms per inversion at 80 MB, 123 at 240 MB, 115 with none; the largest
// accepted grid, window and depth count have 1.3 GB of planes):
//   grid_gspace  G on the quadrant, by a half-plane inverse FFT of the |k| table;
//   grid_planes  P_ab from G in shared memory, its half-plane FFT, E and O at the quadrant points q
//                = (kx, ky) that have kept rows, as tiles of 8 q x 8 z: F[q / 8][z / 8][slot][z % 8][q % 8];
//   grid_rows    per tile, one bulk copy: the cosine and sine transforms in shared memory, then the
//                kept rows of the tile's pairs, 8 depths (64 bytes) at a time.
//                With F[z][slot][q] and 8-byte copies the kernel waited for its loads (37 % of L1, 25 % of
//                DRAM): 103 ms per inversion of the 128 x 128 grid against 87.
#include "edt_internal.h"
#include "cplx.cuh"
#include "fadft.cuh"
#include "tc_ptx.cuh"

#include <algorithm>

namespace edt {

namespace {

// ---- half-plane FFT -----------------------------------------------------------------------
// 2D transform of a centrosymmetric N x N plane (its transform X is centrosymmetric too) from rows
// 0..H, H = N/2, in place in H + 3 rows of LD = N + 1 complex slots:
//   row pass:    rows r = 0..H; V(r, k) for k > H equals V(N - r, N - k) of the rows not stored.
//   column pass: columns c = 0..H only (X(ky, kx) = X(-ky, -kx) gives the rest).  Element e of column
//                c is V(e, c) for e < H, else V(N - e, N - c).  Its N slots: e < H at (e, c); e >= H
//                at (e - H, N - c) for 0 < c < H, and in the spare rows H + 1 (c = 0) and H + 2
//                (c = H).  Columns touch disjoint slots, so they need no barrier among them.
// A line is transformed by 8 threads with V = N/8 values each: element 8 a + t in register a of
// thread t; V-point DFTs over a, the twiddle W_N^{t k1}, one exchange through the line's own slots,
// 8-point DFTs over t, outputs X[k1 + V k2].  No shuffles, and an element crosses shared memory
// three times in a row, four in a column.  LD = 1 mod 16 makes element i of a row and of a column
// bank pair i mod 16 apart from a line constant; the exchange stores (k1, t) at 8 k1 + (t ^ (k1 & 7)),
// so that every access of the 8 threads hits 8 different bank pairs mod 8, and the two lines of a
// half-warp lie 8 apart: no bank conflicts (the spare rows aside).
template <int N> struct Half {
  static constexpr int H = N / 2, V = N / 8, LD = N + 1, QD = H + 1;
  static constexpr int THREADS = N == 32 ? 160 : 288;     // 2 lines per half-warp; H + 1 lines in one
                                                          // round, two for N = 128 (33 units, 18 a round)
  static constexpr int PLANE = (H + 3) * LD, TW = N, QUAD = QD * QD;
  static constexpr int SMEM = (PLANE + TW + QUAD) * int(sizeof(float2));
  // slot of X(ky, kx), 0 <= ky < N, 0 <= kx <= H
  __device__ static __forceinline__ int at(int ky, int kx) {
    if (ky < H) return ky * LD + kx;
    if (kx == 0) return (H + 1) * LD + ky - H;
    if (kx == H) return (H + 2) * LD + ky - H;
    return (ky - H) * LD + N - kx;
  }
};

// W_N^{t k1} (sign -) at 8 k1 + t
template <int N> __device__ __forceinline__ void half_twiddles(float2* tw, const float2* tw32) {
  for (int e = threadIdx.x; e < N; e += blockDim.x) tw[e] = tw_at(tw32, (e & 7) * (e >> 3), N);
}

template <int N> struct RowSlots {
  int base;
  __device__ __forceinline__ int ex(int k1, int low) const { return base + 8 * k1 + low; }
  __device__ __forceinline__ int out(int k1, int k2) const { return base + k1 + Half<N>::V * k2; }
};
template <int N> struct ColSlots {
  int lo, hi, hs;                       // slot of element 0; of element H; step from there on
  __device__ __forceinline__ int ex(int k1, int low) const {
    return k1 < Half<N>::V / 2 ? lo + (8 * k1 + low) * Half<N>::LD : hi + (8 * k1 - Half<N>::H + low) * hs;
  }
  __device__ __forceinline__ int out(int k1, int k2) const {
    return k2 < 4 ? lo + (k1 + Half<N>::V * k2) * Half<N>::LD : hi + (k1 + Half<N>::V * (k2 - 4)) * hs;
  }
};

// one line by threads t = 0..7 of a group (all 32 lanes of the warp call it; act: the line exists)
template <int N, class Slots>
__device__ __forceinline__ void line_fft(float2 (&v)[Half<N>::V], float2* s, const float2* tw, const Slots& sl, int t,
                                         bool act) {
  constexpr int V = Half<N>::V, I = V >= 8 ? V / 8 : 1;
  Dft<V, +1>::run(v);
#pragma unroll
  for (int k1 = 1; k1 < V; ++k1) v[k1] = v[k1] * tw_sg<+1>(tw[8 * k1 + t]);
  __syncwarp();                         // the group's loads precede its stores
  if (act) {
#pragma unroll
    for (int k1 = 0; k1 < V; ++k1) s[sl.ex(k1, t ^ (k1 & 7))] = v[k1];
  }
  __syncwarp();
  float2 u[I][8];
#pragma unroll
  for (int i = 0; i < I; ++i) {
    const int k1 = V >= 8 ? t + 8 * i : t & (V - 1);
#pragma unroll
    for (int j = 0; j < 8; ++j) u[i][j] = s[sl.ex(k1, j ^ (k1 & 7))];
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < I; ++i) {
    const int k1 = t + 8 * i;
    dft8<+1>(u[i]);
    if (act && k1 < V) {
#pragma unroll
      for (int k2 = 0; k2 < 8; ++k2) s[sl.out(k1, k2)] = u[i][k2];
    }
  }
}

// src(r, t, v): v[a] = element 8 a + t of row r.  Only columns 0..cmax are transformed.  Ends with a
// block barrier.
template <int N, class Src>
__device__ __forceinline__ void half_fft(float2* s, const float2* tw, int cmax, const Src& src) {
  using S = Half<N>;
  constexpr int H = S::H, V = S::V, LD = S::LD;
  const int t = threadIdx.x & 7, h = (threadIdx.x >> 3) & 1, hw = (threadIdx.x >> 4) & 1;
  const int nu = blockDim.x >> 4;       // half-warps: two lines each, 8 apart
  for (int ub = (threadIdx.x >> 5) * 2; ub <= H / 2; ub += nu) {
    const int u = ub + hw, r = 16 * (u >> 3) + (u & 7) + 8 * h;
    const bool act = r <= H;
    float2 v[V];
    src(act ? r : 0, t, v);
    line_fft<N>(v, s, tw, RowSlots<N>{(act ? r : 0) * LD}, t, act);
  }
  __syncthreads();
  for (int ub = (threadIdx.x >> 5) * 2; ub <= H / 2; ub += nu) {
    if (16 * (ub >> 3) + (ub & 7) > cmax) continue;          // the warp's first column
    const int u = ub + hw, cc = 16 * (u >> 3) + (u & 7) + 8 * h;
    const bool act = cc <= cmax;
    const int c = act ? cc : 0, cm = (N - c) & (N - 1);
    const bool spec = c == 0 || c == H;
    float2 v[V];
#pragma unroll
    for (int a = 0; a < V; ++a) v[a] = s[a < V / 2 ? (8 * a + t) * LD + c : (N - 8 * a - t) * LD + cm];
    const ColSlots<N> sl = spec ? ColSlots<N>{c, (c == 0 ? H + 1 : H + 2) * LD, 1} : ColSlots<N>{c, cm, LD};
    line_fft<N>(v, s, tw, sl, t, act);
  }
  __syncthreads();
}

constexpr int GT_Q = 8, GT_Z = 8, GT_P = GT_Q * GT_Z;    // points of a tile of F

// ---- G on the quadrant ----------------------------------------------------------------------
// G(y, z) of one frequency for 0 <= yx, yy <= H, CTA per z: Gs[z][yy][yx].
template <int N>
__global__ void __launch_bounds__(Half<N>::THREADS) grid_gspace_kernel(Dev d, int f) {
  using S = Half<N>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* s = reinterpret_cast<float2*>(smem_raw);
  float2* tw = s + S::PLANE;
  float2* tab = tw + S::TW;
  const int z = blockIdx.x;
  const float2* g = d.g32 + size_t(f) * d.nk * d.nzs + z;
  half_twiddles<N>(tw, d.tw32);
  for (int e = threadIdx.x; e < S::QUAD; e += blockDim.x) tab[e] = g[size_t(e) * d.nzs];
  __syncthreads();
  half_fft<N>(s, tw, S::H, [&](int r, int t, float2 (&v)[S::V]) {
#pragma unroll
    for (int a = 0; a < S::V; ++a) {
      const int x = 8 * a + t;
      v[a] = tab[r * S::QD + (a < S::V / 2 ? x : N - x)];
    }
  });
  const float sc = float(1.0 / (double(N) * N * d.dx * d.dy));
  float2* G = d.Gs + size_t(z) * S::QUAD;
  for (int e = threadIdx.x; e < S::QUAD; e += blockDim.x) {
    const int y = e / S::QD, x = e - y * S::QD;
    const float2 v = s[S::at(y, x)];
    G[e] = make_float2(sc * v.x, sc * v.y);
  }
}

// ---- products and planes --------------------------------------------------------------------
// CTA per (z, every gridDim.x-th plane).  swap: only a >= b, the other half of the
// windows from the transposed points.  cmax: the largest column among the points (transposed ones
// included); at low frequencies the cut keeps no point beyond it, and the rest is not transformed (128 x
// 128 midpoints, 4-50 Hz: 84.6 ms per inversion, 85.4 with all columns).
template <int N>
__global__ void __launch_bounds__(Half<N>::THREADS, N == 128 ? 2 : 3)
grid_planes_kernel(Dev d, const int* qxy, int nq, int hx, int hy, int swap, int nplane, int cmax) {
  using S = Half<N>;
  constexpr int H = S::H, V = S::V, QD = S::QD;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* s = reinterpret_cast<float2*>(smem_raw);
  float2* tw = s + S::PLANE;
  float2* gq = tw + S::TW;
  const float2* G = d.Gs + size_t(blockIdx.y) * S::QUAD;
  half_twiddles<N>(tw, d.tw32);
  for (int e = threadIdx.x; e < S::QUAD; e += blockDim.x) gq[e] = G[e];
  const int nE = (hx + 1) * (hy + 1);
  // slot stride GT_P within a tile
  const size_t ns = size_t(nE + hx * hy), zt = (d.nz + GT_Z - 1) / GT_Z;
  float2* F = d.U + (size_t(blockIdx.y / GT_Z) * ns) * GT_P + (blockIdx.y % GT_Z) * GT_Q;
  for (int pl = blockIdx.x; pl < nplane; pl += gridDim.x) {
    int a, b;
    if (swap) {
      a = 0;
      while ((a + 1) * (a + 2) / 2 <= pl) ++a;
      b = pl - a * (a + 1) / 2;
    } else {
      b = pl / (hx + 1);
      a = pl - b * (hx + 1);
    }
    __syncthreads();                    // gq loaded; the last plane's points read
    half_fft<N>(s, tw, cmax, [&](int r, int t, float2 (&v)[V]) {
      const int rp = r + b;
      const float2* gm = gq + abs(r - b) * QD;
      const float2* gp = gq + (rp > H ? N - rp : rp) * QD;
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const int x = 8 * i + t;
        // |x - a| and |x + a| folded to 0..H
        const int xm = i < V / 2 ? abs(x - a) : H - abs(x - a - H);
        const int xp = i < V / 2 ? H - abs(x + a - H) : abs(N - x - a);
        v[i] = gm[xm] * gp[xp];
      }
    });
    float2* e0 = F + (b * (hx + 1) + a) * GT_P;
    float2* o0 = a > 0 && b > 0 ? F + (nE + (b - 1) * hx + a - 1) * GT_P : nullptr;
    float2* e1 = swap && a != b ? F + (a * (hx + 1) + b) * GT_P : nullptr;
    float2* o1 = e1 && o0 ? F + (nE + (a - 1) * hx + b - 1) * GT_P : nullptr;
    for (int q = threadIdx.x; q < nq; q += blockDim.x) {
      const int xy = qxy[q], x = xy & 0xffff, y = xy >> 16;
      const float2 p = s[S::at(y, x)], m = s[S::at((N - y) & (N - 1), x)];
      const size_t at = size_t(q / GT_Q) * zt * ns * GT_P + q % GT_Q;
      e0[at] = p + m;
      if (o0) o0[at] = p - m;
      if (e1) {
        const float2 pt = s[S::at(x, y)], mt = s[S::at((N - x) & (N - 1), y)];
        e1[at] = pt + mt;
        if (o1) o1[at] = pt - mt;
      }
    }
  }
}

// ---- window transforms and rows -------------------------------------------------------------
constexpr float C1 = 0.92387953251128674f, C2 = 0.70710678118654752f, C3 = 0.38268343236508977f;   // cos(k pi/8)

__device__ __forceinline__ float2 sc2(float c, float2 v) { return make_float2(c * v.x, c * v.y); }
__device__ __forceinline__ float2 mad2(float c, float2 v, float2 w) { return make_float2(fmaf(c, v.x, w.x), fmaf(c, v.y, w.y)); }

// x_j <- x_0 + (-1)^j x_H + 2 sum_{0<a<H} cos(pi j a/H) x_a
template <int H> struct Dct {
  __device__ static __forceinline__ void run(float2 (&x)[H + 1]) {
    constexpr int M = H / 2;
    float2 u[M + 1], v[M];
#pragma unroll
    for (int a = 0; a < M; ++a) { u[a] = x[a] + x[H - a]; v[a] = x[a] - x[H - a]; }
    u[M] = x[M] + x[M];
    Dct<M>::run(u);
#pragma unroll
    for (int j = 0; j <= M; ++j) x[2 * j] = u[j];
    if constexpr (H == 2) {
      x[1] = v[0];
    } else if constexpr (H == 4) {
      x[1] = mad2(2.f * C2, v[1], v[0]);
      x[3] = mad2(-2.f * C2, v[1], v[0]);
    } else {
      static_assert(H == 8, "windows of at most 16");
      const float2 e = mad2(2.f * C2, v[2], v[0]), g = mad2(-2.f * C2, v[2], v[0]);
      const float2 p = mad2(2.f * C3, v[3], sc2(2.f * C1, v[1])), r = mad2(-2.f * C1, v[3], sc2(2.f * C3, v[1]));
      x[1] = e + p; x[7] = e - p;
      x[3] = g + r; x[5] = g - r;
    }
  }
};
template <> struct Dct<1> {
  __device__ static __forceinline__ void run(float2 (&x)[2]) {
    const float2 u = x[0], v = x[1];
    x[0] = u + v; x[1] = u - v;
  }
};
template <> struct Dct<0> {
  __device__ static __forceinline__ void run(float2 (&)[1]) {}
};

// x_{j-1} <- 2 sum_{0<a<H} sin(pi j a/H) x_{a-1}, 0 < j < H
template <int H> struct Dst {
  __device__ static __forceinline__ void run(float2 (&x)[H - 1]) {
    if constexpr (H == 2) {
      x[0] = x[0] + x[0];
    } else if constexpr (H == 4) {
      const float2 s = sc2(2.f * C2, x[0] + x[2]), d = x[0] - x[2], m = x[1] + x[1];
      x[0] = s + m; x[2] = s - m; x[1] = d + d;
    } else {
      static_assert(H == 8, "windows of at most 16");
      float2 d[3];
      const float2 s1 = x[0] + x[6], s2 = x[1] + x[5], s3 = x[2] + x[4], x4 = x[3] + x[3];
      d[0] = x[0] - x[6]; d[1] = x[1] - x[5]; d[2] = x[2] - x[4];
      Dst<4>::run(d);
      const float2 p = mad2(2.f * C1, s3, sc2(2.f * C3, s1)), r = mad2(-2.f * C3, s3, sc2(2.f * C1, s1));
      const float2 q = sc2(2.f * C2, s2);
      x[0] = p + (q + x4); x[6] = p - (q + x4);
      x[2] = r + (q - x4); x[4] = r - (q - x4);
      x[1] = d[0]; x[3] = d[1]; x[5] = d[2];
    }
  }
};

// A tile in shared memory is v[slot][point].  It arrives as point 8 z + q; the x pass leaves each
// half (4 depths, g = z / 4) as 32 g + ((4 q + z % 4) ^ 8 g), so that the 8 depths of a row, for an even
// and an odd q side by side, fall on 16 different bank pairs.
constexpr int RT_THREADS = 256;
__device__ __forceinline__ int rt_at(int q, int z) { return 32 * (z >> 2) + ((4 * q + (z & 3)) ^ (2 * (z & 4))); }

template <int WX, int WY>
__global__ void __launch_bounds__(RT_THREADS, 3)
grid_rows_kernel(Dev d, const int4* qrows, int nq, float2 cf) {
  constexpr int HX = WX / 2, HY = WY / 2, NE = (HX + 1) * (HY + 1), NS = NE + HX * HY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* v = reinterpret_cast<float2*>(smem_raw);
  __shared__ uint64_t bar;
  const int q0 = blockIdx.y * GT_Q, zb = blockIdx.x * GT_Z;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = RT_THREADS / 32;
  if (threadIdx.x == 0) {
    tcx::mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    constexpr uint32_t bytes = NS * GT_P * sizeof(float2);
    tcx::mbar_expect_tx(&bar, bytes);
    tcx::bulk_g2s(v, d.U + (size_t(blockIdx.y) * gridDim.x + blockIdx.x) * NS * GT_P, bytes, &bar);
  }
  __syncthreads();
  // the wait is bounded; on expiry the copy gets as long again before the CTA leaves
  bool ok = tcx::mbar_drain(&bar, 0u);
  if (!ok) {
    if (threadIdx.x == 0) atomicOr(&d.flags[0], 1u);
    tcx::mbar_drain(&bar, 0u);
  }
  if (!__syncthreads_and(ok)) return;
  // over x: cosine transforms of E's rows b = 0..HY, sine transforms of O's rows b = 1..HY; a warp
  // takes a row's 8 points x 4 depths, which it reads before it stores
  for (int tk = warp; tk < 2 * (2 * HY + 1); tk += nw) {
    const int ln = tk >> 1;
    const float2* p = v + (tk & 1) * 32 + lane;
    float2* o = v + rt_at(lane & 7, 4 * (tk & 1) + (lane >> 3));
    if (ln <= HY) {
      float2 x[HX + 1];
#pragma unroll
      for (int a = 0; a <= HX; ++a) x[a] = p[(ln * (HX + 1) + a) * GT_P];
      Dct<HX>::run(x);
      __syncwarp();
#pragma unroll
      for (int a = 0; a <= HX; ++a) o[(ln * (HX + 1) + a) * GT_P] = x[a];
    } else if constexpr (HX > 0) {
      const int s0 = NE + (ln - HY - 1) * HX;
      float2 x[HX > 1 ? HX - 1 : 1];
      const float2 e = p[(s0 + HX - 1) * GT_P];
#pragma unroll
      for (int a = 0; a < HX - 1; ++a) x[a] = p[(s0 + a) * GT_P];
      if constexpr (HX > 1) Dst<HX>::run(x);
      __syncwarp();
#pragma unroll
      for (int a = 0; a < HX - 1; ++a) o[(s0 + a) * GT_P] = x[a];
      o[(s0 + HX - 1) * GT_P] = e;
    }
  }
  __syncthreads();
  // over y: E's columns 0..HX, O's columns 1..HX (the last one Y)
  for (int tk = warp; tk < 2 * (2 * HX + 1); tk += nw) {
    const int ln = tk >> 1;
    float2* p = v + (tk & 1) * 32 + lane;
    if (ln <= HX) {
      float2 x[HY + 1];
#pragma unroll
      for (int b = 0; b <= HY; ++b) x[b] = p[(b * (HX + 1) + ln) * GT_P];
      Dct<HY>::run(x);
#pragma unroll
      for (int b = 0; b <= HY; ++b) p[(b * (HX + 1) + ln) * GT_P] = x[b];
    } else if constexpr (HY > 1) {
      float2 x[HY - 1];
      float2* o = p + (NE + ln - HX - 1) * GT_P;
#pragma unroll
      for (int b = 0; b < HY - 1; ++b) x[b] = o[b * HX * GT_P];
      Dst<HY>::run(x);
#pragma unroll
      for (int b = 0; b < HY - 1; ++b) o[b * HX * GT_P] = x[b];
    }
  }
  __syncthreads();
  // the kept rows of both pairs of every point, 8 lanes (depths) per row, four groups per point
  const int z = lane & 7, g = warp * 4 + (lane >> 3), q = g & 7;
  if (q0 + q >= nq || zb + z >= d.nz) return;
  const int4 R = qrows[q0 + q];
  const int n = R.y + R.w;
  float2* A = d.A32 + zb + z;
  const float2* p = v + rt_at(q, z);
  const float2 ohh = p[(NS - 1) * GT_P];
  constexpr int STEP = RT_THREADS / 64, AHEAD = 4;        // rows' j read ahead
  auto row_of = [&](int i) { return i < R.y ? R.x + i : R.z + i - R.y; };
  auto j_of = [&](int i) { return i < n ? int(d.rows[row_of(i)] & 0xffffu) : 0; };
  int jn[AHEAD];
#pragma unroll
  for (int u = 0; u < AHEAD; ++u) jn[u] = j_of((g >> 3) + u * STEP);
  for (int i = g >> 3; i < n; i += STEP) {
    const bool mir = i >= R.y;
    const int row = row_of(i);
    const int j = jn[0], jy = j / WX - HY, jx = j - (j / WX) * WX - HX;
#pragma unroll
    for (int u = 0; u + 1 < AHEAD; ++u) jn[u] = jn[u + 1];
    jn[AHEAD - 1] = j_of(i + AHEAD * STEP);
    const int ax = abs(jx), ay = abs(jy);
    float2 m = p[(ay * (HX + 1) + ax) * GT_P];
    if constexpr (HX > 0 && HY > 0) {
      const bool ix = jx != 0 && ax < HX, iy = jy != 0 && ay < HY;
      float2 o = (jx + jy) & 1 ? make_float2(-ohh.x, -ohh.y) : ohh;
      if (ix) {                       // i (-1)^jy s(jx) X
        const float2 X = p[(NE + (HY - 1) * HX + ax - 1) * GT_P];
        const float c = ((jy & 1) != 0) != (jx < 0) ? -1.f : 1.f;
        o = make_float2(fmaf(-c, X.y, o.x), fmaf(c, X.x, o.y));
      }
      if (iy) {                       // i (-1)^jx s(jy) Y
        const float2 Y = p[(NE + (ay - 1) * HX + HX - 1) * GT_P];
        const float c = ((jx & 1) != 0) != (jy < 0) ? -1.f : 1.f;
        o = make_float2(fmaf(-c, Y.y, o.x), fmaf(c, Y.x, o.y));
      }
      if (ix && iy) {
        const float2 B = p[(NE + (ay - 1) * HX + ax - 1) * GT_P];
        o = (jx < 0) != (jy < 0) ? o + B : o - B;
      }
      m = mir ? m - o : m + o;
    }
    A[size_t(row) * d.nzs] = cf * m;
  }
}

template <int WX, int WY>
constexpr int rows_smem() { return ((WX / 2 + 1) * (WY / 2 + 1) + (WX / 2) * (WY / 2)) * GT_P * int(sizeof(float2)); }

#define GRID_WINDOWS(X) X(1, 1) X(2, 1) X(4, 1) X(8, 1) X(16, 1) X(2, 2) X(4, 4) X(8, 8) X(16, 16) X(4, 2) X(8, 4) X(16, 8)

template <int N>
cudaError_t planes_for(const Dev& d, const int* qxy, int nq, int2 qmax, cudaStream_t s) {
  const int hx = d.wx / 2, hy = d.wy / 2, swap = d.wx == d.wy && d.dx == d.dy;
  const int npl = swap ? (hx + 1) * (hx + 2) / 2 : (hx + 1) * (hy + 1);
  // about four rounds of CTAs where there are planes enough; each loads its depth's quadrant once
  const int nx = std::min(npl, std::max(1, (4 * 304 + d.nz - 1) / d.nz));
  grid_planes_kernel<N><<<dim3(nx, d.nz), Half<N>::THREADS, Half<N>::SMEM, s>>>(
      d, qxy, nq, hx, hy, swap, npl, swap ? std::max(qmax.x, qmax.y) : qmax.x);
  return cudaGetLastError();
}

template <int N>
cudaError_t prepare_n() {
  cudaError_t e = allow_smem(grid_gspace_kernel<N>, Half<N>::SMEM);
  return e != cudaSuccess ? e : allow_smem(grid_planes_kernel<N>, Half<N>::SMEM);
}

}  // namespace

int fa_grid_slots(int wx, int wy) { return (wx / 2 + 1) * (wy / 2 + 1) + (wx / 2) * (wy / 2); }

size_t fa_grid_bytes(int nz, int slots, int nq) {
  return size_t((std::max(nq, 1) + GT_Q - 1) / GT_Q) * ((nz + GT_Z - 1) / GT_Z) * slots * GT_P * sizeof(float2);
}

cudaError_t launch_fa_grid(const Dev& d, int f, int qoff, int nq, int2 qmax, double2 cf, cudaStream_t s) {
  if (nq == 0) return cudaSuccess;       // no kept row at this frequency
  cudaError_t e;
  if (d.N == 32) grid_gspace_kernel<32><<<d.nz, Half<32>::THREADS, Half<32>::SMEM, s>>>(d, f);
  else if (d.N == 64) grid_gspace_kernel<64><<<d.nz, Half<64>::THREADS, Half<64>::SMEM, s>>>(d, f);
  else grid_gspace_kernel<128><<<d.nz, Half<128>::THREADS, Half<128>::SMEM, s>>>(d, f);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const float2 c = make_float2(float(0.5 * cf.x), float(0.5 * cf.y));
  e = d.N == 32 ? planes_for<32>(d, d.q_xy + qoff, nq, qmax, s)
      : d.N == 64 ? planes_for<64>(d, d.q_xy + qoff, nq, qmax, s)
                  : planes_for<128>(d, d.q_xy + qoff, nq, qmax, s);
  if (e != cudaSuccess) return e;
  // the depth tiles of a point side by side: its rows' neighbouring 64-byte pieces meet in L2
  const dim3 g((d.nz + GT_Z - 1) / GT_Z, (nq + GT_Q - 1) / GT_Q);
  switch (d.wx * 32 + d.wy) {
#define GR(WX, WY) case WX * 32 + WY: \
    grid_rows_kernel<WX, WY><<<g, RT_THREADS, rows_smem<WX, WY>(), s>>>(d, d.q_rows + qoff, nq, c); break;
    GRID_WINDOWS(GR)
#undef GR
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t prepare_fa_grid(const Dev& d) {
  cudaError_t e = d.N == 32 ? prepare_n<32>() : d.N == 64 ? prepare_n<64>() : prepare_n<128>();
  if (e != cudaSuccess) return e;
  switch (d.wx * 32 + d.wy) {
#define GA(WX, WY) case WX * 32 + WY: \
    return allow_smem(grid_rows_kernel<WX, WY>, rows_smem<WX, WY>());
    GRID_WINDOWS(GA)
#undef GA
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace edt
