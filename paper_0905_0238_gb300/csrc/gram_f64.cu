// Plain FP64 normal matrices of the split systems (the FP64 comparison path).
//
// For midpoint index m with rows r = (f, p), q = (p - m) mod N and weights w_r:
//   a_r(z) = |s_f| g(k_p, z) g(k_q, z)                           (kernel row of eq. M)
//   G(z, z') = sum_r w_r [Re a_r(z) Re a_r(z') + Im a_r(z) Im a_r(z')]   = Re(A^H W A)
//   b_+-(z)  = sum_r w_r Re(conj(a_r(z)) d~_+-,r)                       = Re(A^H W d~)
// i.e. Ahat^T Ahat and Ahat^T dhat of the real-stacked system [Re A; Im A].  The kernel
// row is regenerated from the FP64 Green's-function table; nothing of size rows x nz is stored.
//
// The FP64 unit (one warp instruction per 16 cycles of an SM) bounds the kernel, so what matters
// is how many FP64 operations are issued and over how many SMs they are spread:
//   * the lower triangle is cut into 2 x 2 tiles, dealt out to the threads of a CTA (up to
//     8 each; a group of 2048 tiles, depths up to 126, per CTA), so an nz of 65 computes 2 244
//     entries of its 2 145 (64 x 64 tiles computed 12 288) and each row is generated once per
//     group;
//   * a subproblem's rows are split over up to 16 CTAs when the grid would leave SMs idle (33
//     subproblems of a 64-point line ran on 33 of 152 SMs, the longest of them setting the
//     time); the parts are added in order by gram_f64_sum.  The split depends on nx, nz and the
//     subproblem's own rows only, so a context restricted to some subproblems adds alike.
// Measured (GB300): 64-point line, 32 frequencies, nz 64: 0.84 -> about 0.11 ms; 256-point line, 10
// frequencies, nz 65: 2.04 -> 0.49 ms.
#include "edt_internal.h"
#include "cplx.cuh"

#include <algorithm>

namespace edt {

namespace {

constexpr int G_THREADS = 256, G_MT = 8, G_TILES = G_THREADS * G_MT;
constexpr int G_SPLIT_MAX = 16, G_MIN_ROWS = 24;      // parts of a subproblem, rows per part at least
constexpr int G_CTAS = 4 * 152;                       // CTAs wanted before the rows are left whole

__host__ __device__ inline int micro_rows(int nz) { return (nz + 1) / 2; }
__host__ __device__ inline int tile_groups(int nz) {
  const int mr = micro_rows(nz), n = mr * (mr + 1) / 2;
  return (n + G_TILES - 1) / G_TILES;
}
// sums one part of a group leaves: whole rounds of the CTA's threads over the most tiles a group has
__host__ __device__ inline int part_doubles(int nz) {
  const int mr = micro_rows(nz), n = mr * (mr + 1) / 2;
  return 4 * G_THREADS * ((min(n, G_TILES) + G_THREADS - 1) / G_THREADS);
}
__device__ __forceinline__ void tri_of(int t, int& r, int& c) {      // tile (r >= c), row-major
  r = int((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
  while (r * (r + 1) / 2 > t) --r;
  while ((r + 1) * (r + 2) / 2 <= t) ++r;
  c = t - r * (r + 1) / 2;
}
// parts the nr rows of a subproblem are added in
__device__ __forceinline__ int parts_of(long long nr, int nsplit) {
  return int(max(1LL, min((long long)nsplit, nr / G_MIN_ROWS)));
}
inline int rows_per_chunk(int nz) { return std::max(2, std::min(16, 2048 / ((nz + 1) & ~1))); }
inline size_t gram_smem(int nz) {
  return size_t(rows_per_chunk(nz)) * (2 * size_t((nz + 1) & ~1) + 2) * sizeof(double2);
}

__device__ __forceinline__ void put_tile(const Dev& d, int m, int r, int c, const double (&v)[4]) {
  double* G = d.G + size_t(m) * d.nz * d.nz;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int zi = 2 * r + i, zj = 2 * c + j;
      if (zi < d.nz && zj <= zi) {
        G[size_t(zi) * d.nz + zj] = v[2 * i + j];
        G[size_t(zj) * d.nz + zi] = v[2 * i + j];
      }
    }
}

// CTA (group, m, part); the last group, which holds every depth, also forms b.
__global__ void __launch_bounds__(G_THREADS, 2) gram_f64_kernel(Dev d, int kc) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nz = d.nz, nze = (nz + 1) & ~1, N = d.N, msk = N - 1;
  double2* A = reinterpret_cast<double2*>(smem_raw);      // [kc][nze] a_r
  double2* B = A + size_t(kc) * nze;                      // [kc][nze] w_r a_r
  double2* rh = B + size_t(kc) * nze;                     // [kc][2]
  const int grp = blockIdx.x, m = blockIdx.y, part = blockIdx.z;
  const long long r00 = d.row_off[m], nr = d.row_off[m + 1] - r00;
  const int np = parts_of(nr, d.g64_split);
  if (part >= np) return;
  const long long r0 = r00 + nr * part / np, r1 = r00 + nr * (part + 1) / np;
  const int mr = micro_rows(nz), ntile = mr * (mr + 1) / 2;
  const int t0 = grp * G_TILES, t1 = min(ntile, t0 + G_TILES);
  const bool last = t1 == ntile;
  int rl, cl;
  tri_of(t1 - 1, rl, cl);
  const int zmax = 2 * rl + 2;                            // depths this group reads (<= nze)
  int tr[G_MT], tc[G_MT], nq = 0;
  double acc[G_MT][4];
#pragma unroll
  for (int q = 0; q < G_MT; ++q) {
    const int t = t0 + q * G_THREADS + int(threadIdx.x);
    tr[q] = tc[q] = 0;
    if (t < t1) { tri_of(t, tr[q], tc[q]); nq = q + 1; }
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[q][i] = 0.0;
  }
  constexpr int BQ = 4;                                   // (z, side) of b per thread: 2 nz <= 1024
  double bacc[BQ] = {};
  for (long long c0 = r0; c0 < r1; c0 += kc) {
    const int nk = int(min((long long)kc, r1 - c0));
    for (int e = threadIdx.x; e < nk * zmax; e += G_THREADS) {
      const int k = e / zmax, z = e - k * zmax;
      const uint32_t row = d.rows[c0 + k];
      const int f = row_f(row), p = row_p(row), q = (p - m) & msk;
      const int kp = p <= N / 2 ? p : N - p, kq = q <= N / 2 ? q : N - q;
      const double2* g = d.g64 + size_t(f) * d.nk * nz;
      double2 v = make_double2(0.0, 0.0);
      if (z < nz) v = d.fc[f].s_abs * (g[size_t(kp) * nz + z] * g[size_t(kq) * nz + z]);
      A[k * nze + z] = v;
      B[k * nze + z] = row_w2(row) ? v + v : v;
    }
    if (last && int(threadIdx.x) < 2 * nk)
      rh[threadIdx.x] = reinterpret_cast<const double2*>(d.rhs)[2 * c0 + threadIdx.x];
    __syncthreads();
    for (int k = 0; k < nk; ++k) {
#pragma unroll
      for (int q = 0; q < G_MT; ++q)
        if (q < nq) {
          const double2 a0 = A[k * nze + 2 * tr[q]], a1 = A[k * nze + 2 * tr[q] + 1];
          const double2 b0 = B[k * nze + 2 * tc[q]], b1 = B[k * nze + 2 * tc[q] + 1];
          acc[q][0] = fma(a0.x, b0.x, fma(a0.y, b0.y, acc[q][0]));
          acc[q][1] = fma(a0.x, b1.x, fma(a0.y, b1.y, acc[q][1]));
          acc[q][2] = fma(a1.x, b0.x, fma(a1.y, b0.y, acc[q][2]));
          acc[q][3] = fma(a1.x, b1.x, fma(a1.y, b1.y, acc[q][3]));
        }
      if (last) {
#pragma unroll
        for (int i = 0; i < BQ; ++i) {
          const int e = threadIdx.x + i * G_THREADS;
          if (e < 2 * nz) {
            const double2 x = B[k * nze + (e >> 1)], y = rh[2 * k + (e & 1)];
            bacc[i] = fma(x.x, y.x, fma(x.y, y.y, bacc[i]));
          }
        }
      }
    }
    __syncthreads();
  }
  if (np == 1) {
#pragma unroll
    for (int q = 0; q < G_MT; ++q)
      if (q < nq) put_tile(d, m, tr[q], tc[q], acc[q]);
  } else {
    double* P = d.g64part + ((size_t(m) * gridDim.x + grp) * d.g64_split + part) * part_doubles(nz) + threadIdx.x;
#pragma unroll
    for (int q = 0; q < G_MT; ++q)
      if (q < nq)
#pragma unroll
        for (int i = 0; i < 4; ++i) P[size_t(4 * q + i) * G_THREADS] = acc[q][i];
  }
  if (last) {
    double* b = np == 1 ? d.b + size_t(m) * nz * 2 : d.b64part + (size_t(m) * d.g64_split + part) * nz * 2;
#pragma unroll
    for (int i = 0; i < BQ; ++i) {
      const int e = threadIdx.x + i * G_THREADS;
      if (e < 2 * nz) b[e] = bacc[i];
    }
  }
}

// the parts of subproblem m's group added in order
__global__ void __launch_bounds__(G_THREADS) gram_f64_sum_kernel(Dev d) {
  const int grp = blockIdx.x, m = blockIdx.y, nz = d.nz;
  const int np = parts_of(d.row_off[m + 1] - d.row_off[m], d.g64_split);
  if (np == 1) return;
  const int mr = micro_rows(nz), ntile = mr * (mr + 1) / 2;
  const double* P = d.g64part + (size_t(m) * gridDim.x + grp) * d.g64_split * part_doubles(nz) + threadIdx.x;
  for (int q = 0; q < G_MT; ++q) {
    const int t = grp * G_TILES + q * G_THREADS + int(threadIdx.x);
    if (t >= ntile) break;
    double v[4] = {};
    for (int s = 0; s < np; ++s)
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] += P[size_t(s) * part_doubles(nz) + size_t(4 * q + i) * G_THREADS];
    int r, c;
    tri_of(t, r, c);
    put_tile(d, m, r, c, v);
  }
  if (grp == 0)
    for (int e = threadIdx.x; e < 2 * nz; e += G_THREADS) {
      const double* bp = d.b64part + size_t(m) * d.g64_split * nz * 2 + e;
      double v = 0.0;
      for (int s = 0; s < np; ++s) v += bp[size_t(s) * nz * 2];
      d.b[size_t(m) * nz * 2 + e] = v;
    }
}

}  // namespace

int gram_f64_split(int nz, int nsub) {
  const int ctas = nsub * tile_groups(nz);
  return std::max(1, std::min(G_SPLIT_MAX, (G_CTAS + ctas - 1) / ctas));
}

size_t gram_f64_part_doubles(int nz, int nsub) {
  return size_t(nsub) * tile_groups(nz) * gram_f64_split(nz, nsub) * part_doubles(nz);
}

cudaError_t prepare_gram_f64() {
  size_t most = 0;
  for (int nz = 1; nz <= MAX_NZ; ++nz) most = std::max(most, gram_smem(nz));
  return allow_smem(gram_f64_kernel, most);
}

cudaError_t launch_gram_f64(const Dev& d, cudaStream_t s) {
  const int ng = tile_groups(d.nz);
  gram_f64_kernel<<<dim3(ng, d.nsub, d.g64_split), G_THREADS, gram_smem(d.nz), s>>>(d, rows_per_chunk(d.nz));
  if (d.g64_split > 1) gram_f64_sum_kernel<<<dim3(ng, d.nsub), G_THREADS, 0, s>>>(d);
  return cudaGetLastError();
}

}  // namespace edt
