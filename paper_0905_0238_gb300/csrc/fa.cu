// Window geometry: finite half-offset aperture on an nx x ny periodic midpoint grid
// (Section "A practical 3D geometry", with the aperture sinc of eq. M kept as the window's
// Dirichlet kernel).  ny = 1 is the 2D line survey with a finite aperture.
//
// Kernel rows (per frequency f, for every kept row (pair, f, j) and depth z):
//   M(k_m; f, j, z) = c_f sum_y exp(i k_m.y) U_j(y, z),
//   U_j(y, z)       = sum_w exp(-2 pi i j.w/W) G(y - w, z) G(y + w, z),
// with G(y, z) = (1/(L_x L_y)) sum_a exp(i k_a.y) g(|k_a|, z) and c_f = omega~^2 dx dy dz.
// This is the row of the decoupled system (eq. DMV): summing the midpoint transform of the
// Born data over the window, y -> y + w turns the product G(2w - y) G(y) of the kernel of
// half-offset w into G(y - w) G(y + w) and the midpoint phase exp(-i k_m.w) cancels, so the
// window transform acts on U before one transform over y gives every k_m at once.
// Stages per frequency of a line: fa_gspace (spectrum from the table, inverse FFT -> G), fa_u
// (products and the window transform per y), fa_mrows (FFT of U_j per (j, z); clusters of ZC
// consecutive depths, then the kept rows of (f, j) are written into the row table A32[row][z]
// ZC depths at a time from the cluster's distributed shared memory).  A grid takes the
// transform over y first (csrc/fagrid.cu).
//
// Data: the window transform of D[f][m][w] per midpoint (fa_dwin, written transposed as
// Dw[f][j][m]), then per (f, j) plane the midpoint FFT and the split right-hand sides of
// the kept rows, d_+ = (d(k_m) + d(-k_m))/2, d_- = (d(k_m) - d(-k_m))/(2i) (eq. Split).
//
// Inverse: Vhat(k_m) = x_+ + i x_- of each pair, Vhat(-k_m) = conj (eq. VSym), inverse 2D
// FFT per depth in FP64, V[y][x][z] = Re / (nx ny).
#include "edt_internal.h"
#include "cplx.cuh"
#include "wfft.cuh"
#include "fadft.cuh"

#include <algorithm>
#include <cooperative_groups.h>

namespace edt {

namespace {

// threads of the plane kernels: a 2D plane fills shared memory (one CTA per SM), so it takes
// the most warps a CTA can have; a line is one warp's FFT
template <int PY> __host__ __device__ constexpr int plane_threads() { return PY > 0 ? 1024 : 128; }
constexpr int LINE_THREADS = plane_threads<0>();
constexpr int FW_THREADS = 256;   // window-transform kernels

// Plane layout in shared memory: element (y, x) at y * ld + 2 (y/16) + x + 2 (x/16) with
// ld = 1 mod 16, so that along a row and along a column element i sits at i + 2 (i/16)
// modulo 16 complex slots (32 banks).  Every access pattern of the 16-thread line FFT below
// (stride-16 loads, the paired reads of its second pass, the natural-order stores) then
// sends the 16 lanes of each 8-byte phase to 16 distinct slot pairs: no bank conflicts.
__host__ __device__ constexpr int plane_ld(int nx) { return (nx + 2 * (nx / 16) + 15) / 16 * 16 + 1; }
__host__ __device__ constexpr int plane_words(int nx, int ny) {
  return (ny - 1) * plane_ld(nx) + 2 * ((ny - 1) / 16) + (nx - 1) + 2 * ((nx - 1) / 16) + 1;
}
__device__ __forceinline__ int paddr(int y, int x, int ld) { return y * ld + 2 * (y >> 4) + x + 2 * (x >> 4); }


// 2D transform of one plane in shared memory (layout above), nx = 32 PX, ny = 32 PY (PY = 0:
// ny = 1).  Warps take rows, then columns, each line a register-resident warp FFT; the
// twiddle table is that of length nx (ny == nx when PY > 0).
// Load a contiguous [NY][NX] plane into the shared layout: every thread issues all of its loads
// before its shared stores, so a CTA keeps the whole plane's reads in flight.
template <int NX, int NY, int LD, int T>
__device__ __forceinline__ void load_plane(float2* s, const float2* P) {
  constexpr int TOT = NX * NY;
  if (TOT % T == 0) {
    constexpr int PER = TOT % T == 0 ? TOT / T : 1;
    float2 r[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) r[i] = P[threadIdx.x + i * T];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int e = threadIdx.x + i * T, y = e / NX, x = e - y * NX;
      s[paddr(y, x, LD)] = r[i];
    }
  } else {
    for (int e = threadIdx.x; e < TOT; e += blockDim.x) {
      const int y = e / NX, x = e - y * NX;
      s[paddr(y, x, LD)] = P[e];
    }
  }
}

// in-register DFTs of the window (sign -, natural order)
template <int W> __device__ __forceinline__ void reg_dft(float2 (&a)[W]) {
  if constexpr (W > 1) Dft<W, -1>::run(a);
}

// N-point FFT (N = 16 R, R in {2, 4, 8}) of one line by a group of 16 threads, t = 0..15,
// in place in shared memory (element i at s[addr(i)]).  With n = 16 a + t and
// k = k1 + R k2: pass 1 takes the R-point DFT over a of x[16 a + t] and applies W_N^{t k1},
// keeping the result in the slots 16 k1 + t; pass 2 takes the 16-point DFT over t for each
// k1, split between the thread pair (2 k1, 2 k1 + 1) as the 8-point DFTs of the even and the
// odd t (the odd half times W_16^k2), exchanged by one shuffle per value, and writes
// X[k1 + R k2] in natural order.  tw: W_N^e (sign -1) for e < N.  A group is a half-warp.
// src: where pass 1 reads the line (null: the shared slots themselves).
template <int R, int SG, class Addr>
__device__ __forceinline__ void group_fft(float2* s, const Addr& addr, int t, const float2* tw,
                                          const float2* src = nullptr) {
  const unsigned gm = 0xffffu << (threadIdx.x & 16);         // this half-warp
  // slot addresses are affine along each pass (the layout's skew steps at multiples of 16):
  // pass 1 reads slots 16 a + t, pass 2 reads 16 k1 + 2 i + h
  const int a1 = addr(t), s1 = addr(16) - addr(0), s2 = addr(2) - addr(0);
  float2 v[R];
  if (src) {
#pragma unroll
    for (int a = 0; a < R; ++a) v[a] = src[16 * a + t];
  } else {
#pragma unroll
    for (int a = 0; a < R; ++a) v[a] = s[a1 + a * s1];
  }
  Dft<R, SG>::run(v);
#pragma unroll
  for (int k1 = 1; k1 < R; ++k1) v[k1] = v[k1] * tw_sg<SG>(tw[t * k1]);
#pragma unroll
  for (int k1 = 0; k1 < R; ++k1) s[a1 + k1 * s1] = v[k1];
  __syncwarp(gm);
  const int k1 = t >> 1, h = t & 1;
  const bool act = k1 < R;
  const int a2 = addr(16 * (act ? k1 : 0) + h);
  float2 u[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) u[i] = act ? s[a2 + i * s2] : make_float2(0.f, 0.f);
  dft8<SG>(u);
  if (h) {
#pragma unroll
    for (int k2 = 1; k2 < 8; ++k2) u[k2] = u[k2] * tw_sg<SG>(w16(k2));
  }
  float2 p[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    p[i].x = __shfl_xor_sync(gm, u[i].x, 1);
    p[i].y = __shfl_xor_sync(gm, u[i].y, 1);
  }
  __syncwarp(gm);                                            // pass-2 reads before the writes
  if (act) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float2 e = h ? p[i] : u[i], o = h ? u[i] : p[i];
      s[addr(k1 + R * (i + 8 * h))] = h ? e - o : e + o;
    }
  }
  __syncwarp(gm);
}

struct RowAddr {
  int r, ld;
  __device__ __forceinline__ int operator()(int i) const { return paddr(r, i, ld); }
};
struct ColAddr {
  int c, ld;
  __device__ __forceinline__ int operator()(int i) const { return paddr(i, c, ld); }
};

// gsrc: a row-major plane in global memory that the row pass reads directly (its loads then
// overlap other groups' arithmetic); null: the plane is already in s.
template <int PX, int PY, int SG>
__device__ void plane_fft2(float2* s, int ld, const float2* tw, const float2* tws,
                           const float2* gsrc = nullptr) {
  constexpr int NX = 32 * PX, NY = PY > 0 ? 32 * PY : 1;
  if constexpr (PY > 0) {
    // square plane: one group of 16 threads per line, rows then columns
    constexpr int R = NX / 16;
    const int t = threadIdx.x & 15, grp = threadIdx.x >> 4, ng = blockDim.x >> 4;
    for (int r = grp; r < NY; r += ng) group_fft<R, SG>(s, RowAddr{r, ld}, t, tws, gsrc ? gsrc + size_t(r) * NX : nullptr);
    __syncthreads();
    for (int c = grp; c < NX; c += ng) group_fft<R, SG>(s, ColAddr{c, ld}, t, tws);
    __syncthreads();
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int r = warp; r < NY; r += nw) {
    float2 v[PX];
#pragma unroll
    for (int a = 0; a < PX; ++a) v[a] = s[paddr(r, 32 * a + lane, ld)];
    warp_fft<PX>(v, tw, NX, SG, lane);
    const int br = rbits(lane, 5) * PX;
#pragma unroll
    for (int k = 0; k < PX; ++k) s[paddr(r, k + br, ld)] = v[k];
  }
  __syncthreads();
}

// W_N^e (sign -1) for e < N in shared memory, from the context's table of length N
__device__ __forceinline__ void plane_twiddles(float2* tws, const float2* tw32, int N) {
  for (int e = threadIdx.x; e < N; e += blockDim.x) tws[e] = tw_at(tw32, e, N);
}

// signed-index DFT over a window of W samples: out[j] = sum_w exp(-2 pi i j w/W) in[w] with
// j, w in [-W/2, W/2): the plain DFT of (-1)^w in[w], times (-1)^j (-1)^(W/2) (W >= 2).
__host__ __device__ constexpr bool alt_sign_end(int W) { return W >= 2 && ((W / 2) & 1); }
__device__ __forceinline__ float2 neg_if(float2 v, bool n) { return n ? make_float2(-v.x, -v.y) : v; }

// ---- kernel rows of a line -----------------------------------------------------------------
// (a grid's are formed in csrc/fagrid.cu, the transform over y first)
// G(y, z) for one frequency: CTA per z.
template <int PX>
__global__ void __launch_bounds__(LINE_THREADS) fa_gspace_kernel(Dev d, int f) {
  constexpr int NX = 32 * PX, LD = plane_ld(NX);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* s = reinterpret_cast<float2*>(smem_raw);
  const int z = blockIdx.x;
  const float2* g = d.g32 + size_t(f) * d.nk * d.nzs + z;
  float2* tws = s + plane_words(NX, 1);
  plane_twiddles(tws, d.tw32, NX);
  for (int x = threadIdx.x; x < NX; x += blockDim.x) s[paddr(0, x, LD)] = g[size_t(min(x, NX - x)) * d.nzs];
  __syncthreads();
  plane_fft2<PX, 0, +1>(s, LD, d.tw32, tws);
  const float sc = float(1.0 / (double(NX) * d.dx * d.dy));
  float2* G = d.Gs + size_t(z) * NX;
  for (int x = threadIdx.x; x < NX; x += blockDim.x) {
    const float2 v = s[paddr(0, x, LD)];
    G[x] = make_float2(sc * v.x, sc * v.y);
  }
}

// U_j(y, z) for one frequency: thread per (y, z), the window transform in registers, stored for
// the offset wavenumbers j with kept rows only (compacted).
template <int WX>
__global__ void __launch_bounds__(FW_THREADS) fa_u_kernel(Dev d, int f) {
  const int* jmap = d.jmap + size_t(f) * WX;
  const int nx = d.N, x = blockIdx.x * FW_THREADS + threadIdx.x, z = blockIdx.y;
  if (x >= nx) return;
  const float2* G = d.Gs + size_t(z) * nx;
  float2 a[WX];
#pragma unroll
  for (int ix = 0; ix < WX; ++ix) {
    const int w = ix - WX / 2;                             // nx is a power of two
    a[ix] = neg_if(G[(x - w + nx) & (nx - 1)] * G[(x + w + nx) & (nx - 1)], WX >= 2 && (ix & 1));
  }
  reg_dft<WX>(a);
#pragma unroll
  for (int jx = 0; jx < WX; ++jx) {
    const int ja = jmap[jx];
    if (ja >= 0) d.U[(size_t(ja) * d.nz + z) * nx + x] = neg_if(a[jx], WX >= 2 && ((jx & 1) != alt_sign_end(WX)));
  }
}

// Exchange buffer of the two-pass window transforms: [jx][unit][wy] with an odd unit stride
// when WY > 1, so that both the row-wise writes and the column-wise reads spread over banks.
template <int WX, int WY> struct ExLayout {
  static constexpr int UPB = FW_THREADS / WY, US = WY > 1 ? WY + 1 : 1, S = UPB * US;
  static constexpr int SIZE = WX * S;
  __device__ static __forceinline__ int at(int jx, int u, int iwy) { return jx * S + u * US + iwy; }
};

// M(k_m; f, j, z) for ZC consecutive depths of one j: a cluster of ZC CTAs, one (j, z) line
// each (FFT of U_j in shared memory); then every CTA takes a share of the kept rows of
// (f, j) and reads the ZC depths of each from the cluster's lines (distributed shared
// memory), so each row's depths z0..z0+ZC-1 are written together (8 ZC contiguous bytes).
// ZC: depths per cluster, 2, 4 or 8 (the autotuner's choice).
template <int PX, int ZC>
__global__ void __cluster_dims__(1, ZC, 1) __launch_bounds__(LINE_THREADS) fa_mrows_kernel(Dev d, int f, float2 cf) {
  namespace cg = cooperative_groups;
  constexpr int NX = 32 * PX, LD = plane_ld(NX);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* s = reinterpret_cast<float2*>(smem_raw);
  float2* tws = s + plane_words(NX, 1);
  cg::cluster_group cluster = cg::this_cluster();
  // blockIdx.x: position among the frequency's active offset wavenumbers
  const int ja = blockIdx.x, j = d.jact[size_t(f) * d.W + ja];
  const int z = blockIdx.y, rank = int(cluster.block_rank()), z0 = z - rank;
  if (z < d.nz) {                        // every CTA reaches both cluster barriers below
    plane_twiddles(tws, d.tw32, NX);
    load_plane<NX, 1, LD, LINE_THREADS>(s, d.U + (size_t(ja) * d.nz + z) * NX);
    __syncthreads();
    plane_fft2<PX, 0, +1>(s, LD, d.tw32, tws);
  }
  cluster.sync();
  const float2* ps[ZC];
#pragma unroll
  for (int k = 0; k < ZC; ++k) ps[k] = cluster.map_shared_rank(s, k);
  const int e0 = d.fj_off[f * d.W + j], e1 = d.fj_off[f * d.W + j + 1];
  const int n = e1 - e0, per = (n + ZC - 1) / ZC;
  const int a0 = e0 + rank * per, a1 = min(e1, a0 + per);
  for (int e = a0 + threadIdx.x; e < a1; e += blockDim.x) {
    const int2 ent = d.fj_ent[e];
    const int off = paddr(0, ent.x, LD);
    float2 v[ZC];
#pragma unroll
    for (int k = 0; k < ZC; ++k) v[k] = z0 + k < d.nz ? cf * ps[k][off] : make_float2(0.f, 0.f);
    float2* dst = d.A32 + size_t(ent.y) * d.nzs + z0;
    if (z0 + ZC <= d.nzs) {
#pragma unroll
      for (int k = 0; k < ZC; k += 2)
        reinterpret_cast<float4*>(dst)[k / 2] = make_float4(v[k].x, v[k].y, v[k + 1].x, v[k + 1].y);
    } else {
#pragma unroll
      for (int k = 0; k < ZC; ++k) if (z0 + k < d.nzs) dst[k] = v[k];
    }
  }
  cluster.sync();                        // peers may still read this CTA's plane
}

// ---- data ------------------------------------------------------------------------------
// Window transform of D[f][m][wy][wx] for UPB consecutive midpoints, written as Dw[f][j][m].
template <int WX, int WY, typename TIN>
__global__ void __launch_bounds__(FW_THREADS) fa_dwin_kernel(Dev d, const TIN* D) {
  using L = ExLayout<WX, WY>;
  constexpr int W = WX * WY, UPB = L::UPB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* ex = reinterpret_cast<float2*>(smem_raw);
  const int f = blockIdx.y, m0 = blockIdx.x * UPB;
  {
    const int um = threadIdx.x / WY, iwy = threadIdx.x - um * WY, m = m0 + um;
    if (m < d.nxy) {
      const TIN* src = D + ((size_t(f) * d.nxy + m) * WY + iwy) * WX;
      float2 a[WX];
#pragma unroll
      for (int ix = 0; ix < WX; ++ix) {
        const TIN v = src[ix];
        a[ix] = neg_if(make_float2(float(v.x), float(v.y)), WX >= 2 && (ix & 1));
      }
      reg_dft<WX>(a);
#pragma unroll
      for (int jx = 0; jx < WX; ++jx)
        ex[L::at(jx, um, iwy)] = neg_if(a[jx], WX >= 2 && ((jx & 1) != alt_sign_end(WX)));
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < UPB * WX; t += blockDim.x) {
    const int jx = t / UPB, um = t - jx * UPB, m = m0 + um;   // consecutive threads: consecutive m
    if (m >= d.nxy) continue;
    float2 b[WY];
#pragma unroll
    for (int iwy = 0; iwy < WY; ++iwy) b[iwy] = neg_if(ex[L::at(jx, um, iwy)], WY >= 2 && (iwy & 1));
    reg_dft<WY>(b);
#pragma unroll
    for (int jy = 0; jy < WY; ++jy)
      d.Dw[(size_t(f) * W + jy * WX + jx) * d.nxy + m] =
          neg_if(b[jy], WY >= 2 && ((jy & 1) != alt_sign_end(WY)));
  }
}

// Midpoint FFT of one (f, j) plane of Dw and the split right-hand sides of its kept rows.
template <int PX, int PY>
__global__ void __launch_bounds__(plane_threads<PY>()) fa_drhs_kernel(Dev d) {
  constexpr int NX = 32 * PX, NY = PY > 0 ? 32 * PY : 1, LD = plane_ld(NX);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* s = reinterpret_cast<float2*>(smem_raw);
  const int j = blockIdx.x, f = blockIdx.y;
  float2* tws = s + plane_words(NX, NY);
  const float2* P = d.Dw + (size_t(f) * d.W + j) * (NX * NY);
  plane_twiddles(tws, d.tw32, NX);
  if (PY > 0) {
    __syncthreads();
    plane_fft2<PX, PY, -1>(s, LD, d.tw32, tws, P);
  } else {
    load_plane<NX, NY, LD, plane_threads<PY>()>(s, P);
    __syncthreads();
    plane_fft2<PX, PY, -1>(s, LD, d.tw32, tws);
  }
  const int e0 = d.fj_off[f * d.W + j], e1 = d.fj_off[f * d.W + j + 1];
  for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const int2 ent = d.fj_ent[e];
    const int y = ent.x / NX, x = ent.x - y * NX;
    const int ny2 = (NY - y) % NY, nx2 = (NX - x) % NX;
    const float2 a = s[paddr(y, x, LD)], b = s[paddr(ny2, nx2, LD)];
    reinterpret_cast<float4*>(d.rhs)[ent.y] =
        make_float4(0.5f * (a.x + b.x), 0.5f * (a.y + b.y), 0.5f * (a.y - b.y), -0.5f * (a.x - b.x));
  }
}

// ---- inverse ---------------------------------------------------------------------------
// Vhat of every pair and its conjugate at -k_m into vfull[z][m] (FP64), Vhat[pair][z] kept.
__global__ void fa_vfull_kernel(Dev d) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)d.nsub * d.nz) return;
  const int p = int(t / d.nz), z = int(t - (long long)p * d.nz);
  const double* xm = d.x + (size_t(p) * d.nz + z) * 2;
  double re = xm[0], im = xm[1];
  if (d.status[p] != EDT_OK) { re = 0.0; im = 0.0; }
  const int m = d.pair_m[p], nx = d.N, y = m / nx, x = m - y * nx;
  const int mneg = ((d.ny - y) % d.ny) * nx + (nx - x) % nx;
  if (mneg == m) im = 0.0;
  d.vhat[size_t(p) * d.nz + z] = make_double2(re, im);
  d.vfull[size_t(z) * d.nxy + m] = make_double2(re, im);
  d.vfull[size_t(z) * d.nxy + mneg] = make_double2(re, -im);
}

__global__ void fa_vout_kernel(Dev d, void* V, int V_dtype) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)d.nxy * d.nz) return;
  const int m = int(t / d.nz), z = int(t - (long long)m * d.nz);
  const double v = d.vfull[size_t(z) * d.nxy + m].x / double(d.nxy);
  if (V_dtype == EDT_F64) reinterpret_cast<double*>(V)[t] = v;
  else reinterpret_cast<float*>(V)[t] = float(v);
}

// Gram metadata of window rows: row r of the kernel table times the ones row, weight 1;
// the ones row itself.
__global__ void fa_setup_kernel(Dev d, long long nrows) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < nrows) {
    GramRow g;
    g.rp = unsigned(t);
    g.rq = unsigned(d.ones_row);
    g.bp = (unsigned long long)t * d.nzs * sizeof(float2);
    g.bq = (unsigned long long)d.ones_row * d.nzs * sizeof(float2);
    g.sw = 1.f;
    g.pad = 0.f;
    d.gent[t] = g;
  }
  if (t < d.nz) d.A32[size_t(d.ones_row) * d.nzs + t] = make_float2(1.f, 0.f);
}

template <int PX, int PY>
size_t plane_smem() { return size_t(plane_words(32 * PX, PY > 0 ? 32 * PY : 1) + 32 * PX) * sizeof(float2); }
template <int PX>
cudaError_t rows_for(const Dev& d, int f, int nact, float2 cf, cudaStream_t s) {
  if (nact == 0) return cudaSuccess;     // no kept row at this frequency
  const size_t sm = plane_smem<PX, 0>();
  fa_gspace_kernel<PX><<<d.nz, LINE_THREADS, sm, s>>>(d, f);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const dim3 gu((d.N + FW_THREADS - 1) / FW_THREADS, d.nz);
  switch (d.wx) {
#define FA_U(WX) case WX: fa_u_kernel<WX><<<gu, FW_THREADS, 0, s>>>(d, f); break;
    FA_U(1) FA_U(2) FA_U(4) FA_U(8) FA_U(16)
#undef FA_U
    default: return cudaErrorInvalidValue;
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int zc = d.tune_zc;
  const dim3 gm(nact, (d.nz + zc - 1) / zc * zc);
  if (zc == 2) fa_mrows_kernel<PX, 2><<<gm, LINE_THREADS, sm, s>>>(d, f, cf);
  else if (zc == 8) fa_mrows_kernel<PX, 8><<<gm, LINE_THREADS, sm, s>>>(d, f, cf);
  else fa_mrows_kernel<PX, 4><<<gm, LINE_THREADS, sm, s>>>(d, f, cf);
  return cudaGetLastError();
}

template <typename TIN>
cudaError_t dwin_for(const Dev& d, const TIN* D, cudaStream_t s) {
  const unsigned nb = unsigned((d.nxy + FW_THREADS / d.wy - 1) / (FW_THREADS / d.wy));
  dim3 g(nb, d.nf);
  switch (d.wx * 32 + d.wy) {
#define FA_D(WX, WY) case WX * 32 + WY: fa_dwin_kernel<WX, WY, TIN><<<g, FW_THREADS, ExLayout<WX, WY>::SIZE * sizeof(float2), s>>>(d, D); break;
    FA_D(1, 1) FA_D(2, 1) FA_D(4, 1) FA_D(8, 1) FA_D(16, 1)
    FA_D(2, 2) FA_D(4, 4) FA_D(8, 8) FA_D(16, 16) FA_D(4, 2) FA_D(8, 4) FA_D(16, 8)
#undef FA_D
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <int PX, int PY>
cudaError_t prepare_plane() {
  const int sm = int(plane_smem<PX, PY>());
  cudaError_t e;
  if constexpr (PY == 0) {
    if ((e = allow_smem(fa_gspace_kernel<PX>, sm)) != cudaSuccess) return e;
    if ((e = allow_smem(fa_mrows_kernel<PX, 2>, sm)) != cudaSuccess) return e;
    if ((e = allow_smem(fa_mrows_kernel<PX, 4>, sm)) != cudaSuccess) return e;
    if ((e = allow_smem(fa_mrows_kernel<PX, 8>, sm)) != cudaSuccess) return e;
  }
  return allow_smem(fa_drhs_kernel<PX, PY>, sm);
}

// plane shapes: (nx, ny) = (32 PX, 32 PY), PY = 0 for a line
#define FA_LINES(X) X(1, 0) X(2, 0) X(4, 0) X(8, 0) X(16, 0)
#define FA_SHAPES(X) FA_LINES(X) X(1, 1) X(2, 2) X(4, 4)

}  // namespace

bool fa_supported(int nx, int ny, int wx, int wy) {
  const int px = nx / 32, py = ny == 1 ? 0 : ny / 32;
  bool shape = false;
#define FA_S(PX, PY) shape |= (px == PX && py == PY && nx == 32 * PX && (PY == 0 ? ny == 1 : ny == 32 * PY));
  FA_SHAPES(FA_S)
#undef FA_S
  const int k = wx * 32 + wy;
  const bool win = k == 1 * 32 + 1 || k == 2 * 32 + 1 || k == 4 * 32 + 1 || k == 8 * 32 + 1 ||
                   k == 16 * 32 + 1 || k == 2 * 32 + 2 || k == 4 * 32 + 4 || k == 8 * 32 + 8 ||
                   k == 16 * 32 + 16 || k == 4 * 32 + 2 || k == 8 * 32 + 4 || k == 16 * 32 + 8;
  return shape && win && wx <= nx && wy <= ny;
}

cudaError_t launch_fa_line(const Dev& d, int f, int nact, double2 cf, cudaStream_t s) {
  const float2 c = make_float2(float(cf.x), float(cf.y));
  const int px = d.N / 32;
#define FA_R(PX, PY) if (px == PX) return rows_for<PX>(d, f, nact, c, s);
  FA_LINES(FA_R)
#undef FA_R
  return cudaErrorInvalidValue;
}

cudaError_t launch_fa_data(const Dev& d, const void* D, int D_dtype, cudaStream_t s) {
  cudaError_t e = D_dtype == EDT_C64 ? dwin_for<float2>(d, static_cast<const float2*>(D), s)
                                     : dwin_for<double2>(d, static_cast<const double2*>(D), s);
  if (e != cudaSuccess) return e;
  const int px = d.N / 32, py = d.ny == 1 ? 0 : d.ny / 32;
#define FA_DR(PX, PY) \
  if (px == PX && py == PY) { \
    fa_drhs_kernel<PX, PY><<<dim3(d.W, d.nf), plane_threads<PY>(), plane_smem<PX, PY>(), s>>>(d); \
    return cudaGetLastError(); \
  }
  FA_SHAPES(FA_DR)
#undef FA_DR
  return cudaErrorInvalidValue;
}

cudaError_t launch_fa_inverse(const Dev& d, void* V, int V_dtype, cudaStream_t s) {
  const long long n1 = (long long)d.nsub * d.nz;
  fa_vfull_kernel<<<unsigned((n1 + 255) / 256), 256, 0, s>>>(d);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if ((e = fft2_f64(d, d.vfull, d.nz, d.ny, +1, 1.0, s)) != cudaSuccess) return e;
  const long long n2 = (long long)d.nxy * d.nz;
  fa_vout_kernel<<<unsigned((n2 + 255) / 256), 256, 0, s>>>(d, V, V_dtype);
  return cudaGetLastError();
}

cudaError_t launch_fa_setup(const Dev& d, long long nrows, cudaStream_t s) {
  const long long n = std::max<long long>(nrows, d.nz);
  fa_setup_kernel<<<unsigned((n + 255) / 256), 256, 0, s>>>(d, nrows);
  return cudaGetLastError();
}

cudaError_t prepare_fa(const Dev& d) {
  const int px = d.N / 32, py = d.ny == 1 ? 0 : d.ny / 32;
  cudaError_t e = cudaSuccess;
  switch (d.wx * 32 + d.wy) {
#define FA_A(WX, WY) case WX * 32 + WY: \
    e = allow_smem(fa_dwin_kernel<WX, WY, float2>, int(ExLayout<WX, WY>::SIZE * sizeof(float2))); \
    if (e == cudaSuccess) e = allow_smem(fa_dwin_kernel<WX, WY, double2>, int(ExLayout<WX, WY>::SIZE * sizeof(float2))); \
    break;
    FA_A(1, 1) FA_A(2, 1) FA_A(4, 1) FA_A(8, 1) FA_A(16, 1)
    FA_A(2, 2) FA_A(4, 4) FA_A(8, 8) FA_A(16, 16) FA_A(4, 2) FA_A(8, 4) FA_A(16, 8)
#undef FA_A
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  if (d.ny > 1 && (e = prepare_fa_grid(d)) != cudaSuccess) return e;
#define FA_P(PX, PY) if (px == PX && py == PY) return prepare_plane<PX, PY>();
  FA_SHAPES(FA_P)
#undef FA_P
  return cudaErrorInvalidValue;
}

}  // namespace edt
