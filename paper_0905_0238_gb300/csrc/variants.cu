// The paper's solver variants (Section "Numerical Examples") on the FP64 path.
//
//  * Vertical-wavenumber disk: the unknowns of midpoint wavenumber k_m are restricted to the
//    depth vectors whose vertical wavenumber k_z satisfies k_m^2 + k_z^2 <= K^2,
//    K = factor omega_max / c0.  With the orthonormal real basis P (constant, cos and sin of
//    2 pi l j / nz for l = 1, 2, ..., and (-1)^j for even nz, in that order) the kept columns are
//    a leading block P_p, and the restricted normal equations are
//        G' = P_p^T G P_p,   b' = P_p^T b,   x = P_p x'.
//  * Truncated SVD: with Ahat^T Ahat = W Lambda W^T (Lambda = S^2 for the singular values S of
//    Ahat, W its right singular vectors) the solution V S~^-1 U^T dhat is
//        x = sum over lambda_j >= sigma^2 of w_j (w_j^T Ahat^T dhat) / lambda_j,
//    computed from the eigenpairs of the FP64 normal matrix by cyclic two-sided Jacobi rotations
//    in parallel (round-robin) order, the matrix in shared memory and the rotations logged.
#include "edt_internal.h"

namespace edt {

namespace {

// T[m] = G[m] P_p (nz x p), one thread per element
__global__ void kzv_t_kernel(Dev d) {
  const int m = blockIdx.y;
  const int n = d.nz, p = d.kz_p[m];
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * p) return;
  const int i = e / p, c = e - i * p;
  const double* G = d.G + size_t(m) * n * n + size_t(i) * n;
  double s = 0.0;
  for (int k = 0; k < n; ++k) s = fma(G[k], d.kz_P[size_t(k) * n + c], s);
  d.kz_T[size_t(m) * n * n + size_t(i) * p + c] = s;
}

// G'[m] = P_p^T T[m] (p x p) and b'[m] = P_p^T b[m] (p x 2)
__global__ void kzv_g_kernel(Dev d) {
  const int m = blockIdx.y;
  const int n = d.nz, p = d.kz_p[m];
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < p * p) {
    const int a = e / p, c = e - a * p;
    const double* T = d.kz_T + size_t(m) * n * n;
    double s = 0.0;
    for (int i = 0; i < n; ++i) s = fma(d.kz_P[size_t(i) * n + a], T[size_t(i) * p + c], s);
    d.kz_G[size_t(m) * n * n + size_t(a) * p + c] = s;
  } else if (e < p * p + 2 * p) {
    const int a = (e - p * p) >> 1, side = (e - p * p) & 1;
    const double* b = d.b + size_t(m) * n * 2;
    double s = 0.0;
    for (int i = 0; i < n; ++i) s = fma(d.kz_P[size_t(i) * n + a], b[i * 2 + side], s);
    d.kz_b[(size_t(m) * n + a) * 2 + side] = s;
  }
}

// x[m] = P_p x'[m] (nz x 2)
__global__ void kzv_back_kernel(Dev d) {
  const int m = blockIdx.y;
  const int n = d.nz, p = d.kz_p[m];
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 2 * n) return;
  const int i = e >> 1, side = e & 1;
  double s = 0.0;
  for (int a = 0; a < p; ++a) s = fma(d.kz_P[size_t(i) * n + a], d.kz_x[(size_t(m) * n + a) * 2 + side], s);
  d.x[(size_t(m) * n + i) * 2 + side] = s;
}

constexpr int JAC_THREADS = 512;
constexpr int JAC_MAX_SWEEPS = 20;
constexpr int JAC_BLOCKS = 3;      // 2 x 2 blocks per thread: (TSVD_MAX_NZ / 2)(TSVD_MAX_NZ / 2 + 1) / 2 in all
static_assert((TSVD_MAX_NZ / 2) * (TSVD_MAX_NZ / 2 + 1) / 2 <= JAC_THREADS * JAC_BLOCKS, "blocks fit the threads");

// cosine of the rotation of tangent t, 1 / sqrt(1 + t^2) to FP64 (q = 1 + t^2): the FP32 estimate
// y0 and one third-order step on e = 1 - q y0^2 (y = y0 (1 + e/2 + 3 e^2 / 8), error ~ e^3)
__device__ __forceinline__ double cos_of(double t, double q) {
  const double y0 = double(rsqrtf(float(q)));
  const double e = fma(-q * y0, y0, 1.0);
  return fma(y0 * e, fma(0.375, e, 0.5), y0);
}
__device__ __forceinline__ double cos_of(double t) { return cos_of(t, fma(t, t, 1.0)); }
// tangent of the rotation that zeroes apq between diagonal entries that differ by dd = aqq - app, in
// FP32: an inexact angle leaves |apq| 1e-7 of what it was (the next sweep takes the rest), the
// rotation itself is orthogonal to FP64 because the cosine is formed from the tangent that is used
__device__ __forceinline__ float tan_of(float dd, float apq) {
  if (dd == 0.f) return 1.f;
  const float tau = dd / (2.f * apq);
  if (fabsf(tau) > 1e9f) return 0.5f / tau;
  return copysignf(1.f / (fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f))), tau);
}

// players of the round-robin (a dummy when p is odd); round r: player 0 fixed, the others
// rotate; pair k = (position k, position P2 - 1 - k), a < b, b == p: the dummy
__device__ __forceinline__ void jac_pair(int k, int r, int P2, int& a, int& b) {
  auto pos = [&](int t) {
    if (t == 0) return 0;
    const int v = t + r;                       // 1 + (t - 1 + r) mod (P2 - 1), r < P2 - 1
    return v >= P2 ? v - (P2 - 1) : v;
  };
  a = pos(k);
  b = pos(P2 - 1 - k);
  if (a > b) { const int t = a; a = b; b = t; }
}

// One CTA per subproblem: eigen-decomposition of the p x p normal matrix (G, or G' of the disk)
// by cyclic Jacobi, then the truncated-SVD solution for both right-hand sides.
// src: matrices at m * nz * nz with leading dimension p; rhs, out: [m][nz][2].
//
// The FP64 unit (one warp instruction per 64 cycles of each of an SM's four parts) bounds the
// rounds, so a round does no more FP64 work than it has to:
//   * the matrix is kept as its lower triangle and updated two-sidedly in one pass, block (K, L) of
//     the pairs K <= L at a time, where a pass over the columns and one over the rows of the whole
//     matrix do it twice; blocks of two pairs that do not rotate are left alone;
//   * it is kept scaled, A = S B S with S diagonal: a rotation by c [1, -t; t, 1] then is one
//     multiply-add per entry, B_p' = B_p - (t s_q / s_p) B_q, B_q' = B_q + (t s_p / s_q) B_p, with
//     s_p' = c s_p, s_q' = c s_q (fast rotations: 8 operations per block instead of 16); S goes
//     back into the matrix after every sweep (c >= 1/sqrt 2, so it shrinks by 2^-48 at most);
//   * the eigenvectors are not accumulated: with W = J_1 J_2 ... J_n, W^T b is formed by applying
//     each rotation to b as it is found, and W z by applying them in reverse order from the log
//     of their tangents (tlog, written once and read once);
//   * the angles are chosen in FP32 (tan_of);
//   * only what the threshold needs is rotated (below), which ends the sweeps earlier.
// One barrier after the angles and one after the update.  Measured on the paper's acquisition (129
// systems of 65 unknowns): the kernel 14.0 ms with W accumulated over the whole
// matrix and every pair rotated (13 to 20 sweeps), 6.1 with the half matrix and the log, 3.5 ms now (8 to 14
// sweeps).
__global__ void __launch_bounds__(JAC_THREADS) tsvd_jacobi_kernel(Dev d, const double* src, const double* rhs,
                                                                 double* out) {
  extern __shared__ __align__(16) double sm[];
  const int m = blockIdx.x;
  const int n = d.nz;
  const int p = d.kz_p ? d.kz_p[m] : n;
  const int ld = p + 1;
  const int P2 = (p + 1) & ~1, npair = P2 / 2;
  double* A = sm;                         // [p][ld] lower triangle (row >= column) of B
  double* bv = A + size_t(p) * ld;        // [p][2] S^-1 W^T b, later W z
  double* al = bv + 2 * p;                // [2][npair] a round's t s_q / s_p and t s_p / s_q
  double* rt = al + P2;                   // [2][npair] the next round's s_q / s_p and s_p / s_q
  double* sv = rt + P2;                   // [p] S
  double* si = sv + p;                    // [p] S^-1
  double* red = si + p;                   // [32]
  int* pj = reinterpret_cast<int*>(red + 32);   // [2][npair] pair indices a < b (b == p: alone)
  int* rotated = pj + P2;
  const bool has_rows = d.row_off[m + 1] > d.row_off[m];
  double* xo = out + size_t(m) * n * 2;
  if (!has_rows || p == 0) {
    for (int i = threadIdx.x; i < 2 * n; i += blockDim.x) xo[i] = 0.0;
    if (threadIdx.x == 0) d.status[m] = EDT_OK;
    return;
  }
  const double* S = src + size_t(m) * n * n;
  const double* bm = rhs + size_t(m) * n * 2;
  // the matrix times a power of two that puts its largest diagonal entry in [0.5, 1)
  double dmax = 0.0;
  for (int i = threadIdx.x; i < p; i += blockDim.x) dmax = fmax(dmax, fabs(S[size_t(i) * p + i]));
  auto block_max = [&](double v) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0.0;
    for (int w = 0; w < JAC_THREADS / 32; ++w) v = fmax(v, red[w]);
    return v;
  };
  dmax = block_max(dmax);
  int ex = 0;
  if (dmax > 0.0 && isfinite(dmax)) frexp(dmax, &ex);
  const double sc = scalbn(1.0, -ex);
  for (int e = threadIdx.x; e < p * p; e += blockDim.x) {
    const int i = e / p, j = e - i * p;
    if (j <= i) A[i * ld + j] = sc * S[size_t(i) * p + j];
  }
  for (int i = threadIdx.x; i < 2 * p; i += blockDim.x) bv[i] = bm[i];
  for (int i = threadIdx.x; i < p; i += blockDim.x) sv[i] = si[i] = 1.0;
  // this thread's blocks (K <= L), the same in every round
  int bK[JAC_BLOCKS], bL[JAC_BLOCKS];
  const int nblk = npair * (npair + 1) / 2;
#pragma unroll
  for (int q = 0; q < JAC_BLOCKS; ++q) {
    const int e = threadIdx.x + q * JAC_THREADS;
    int L = int((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
    while (L * (L + 1) / 2 > e) --L;
    while ((L + 1) * (L + 2) / 2 <= e) ++L;
    bL[q] = e < nblk ? L : -1;
    bK[q] = e - L * (L + 1) / 2;
  }
  float* tl = d.tlog + size_t(m) * d.tlog_stride;
  // Which pairs to rotate.  Without a threshold: while |a_ij| > 1e-14 sqrt(a_ii a_jj) (relative to
  // its own diagonal, which keeps small eigenvalues of the positive semi-definite matrix accurate;
  // well above the FP64 rounding of a rotation, so the sweeps end).  With one, only the
  // eigenvalues at or above it and their vectors are wanted; th <= the threshold (the largest
  // diagonal entry is at most the largest eigenvalue) stands for it:
  //   both entries >= th / 2: as above;
  //   one of them: decoupled to the FP64 rounding of the larger, |a_ij| <= 1e-15 a_ii;
  //   both below: |a_ij| <= th / (4 p), so that no eigenvalue of that block reaches th (Gershgorin:
  //   below th / 2 + p th / (4 p)); its eigenvalues below th need not be resolved.
  // The small ones are mostly rounding noise, whose relative off-diagonals die down last.
  const double tol = d.tsvd_tol;
  const double th64 = tol > 0.0 ? tol * tol * sc : tol * tol * (sc * dmax);
  const float wanted = tol != 0.0 ? float(0.5 * th64) : -1.f, apart = float(0.25 * th64 / double(p));
  int nround = 0;
  for (int sweep = 0; sweep < JAC_MAX_SWEEPS; ++sweep) {
    if (threadIdx.x == 0) *rotated = 0;
    for (int k = threadIdx.x; k < P2; k += blockDim.x) rt[k] = 1.0;
    __syncthreads();
    for (int r = 0; r < P2 - 1; ++r, ++nround) {
      for (int k = threadIdx.x; k < npair; k += blockDim.x) {
        int a, b;
        jac_pair(k, r, P2, a, b);
        float t = 0.f;
        const double rab = rt[k], rba = rt[npair + k];     // s_b / s_a, s_a / s_b
        if (b < p) {
          const double Bab = A[b * ld + a], Baa = A[a * ld + a], Bbb = A[b * ld + b];
          const float fab = float(Bab), faa = fabsf(float(Baa)), fbb = fabsf(float(Bbb));
          const float sa = float(sv[a]), sb = float(sv[b]);
          const float taa = sa * sa * faa, tbb = sb * sb * fbb, tab = sa * sb * fabsf(fab);   // true entries
          const float hi = fmaxf(taa, tbb), lo = fminf(taa, tbb);
          const bool want = lo >= wanted ? fabsf(fab) > 1e-14f * (sqrtf(faa) * sqrtf(fbb))
                                         : (hi >= wanted ? tab > 1e-15f * hi : tab > apart);
          if (want) t = tan_of(float(rab * Bbb - rba * Baa), fab);
          if (!(fabsf(t) <= 2.f)) t = 0.f;     // outside the estimates' range: nothing to rotate
        }
        pj[k] = a; pj[npair + k] = b;
        tl[size_t(nround) * npair + k] = t;
        double alpha = 0.0, beta = 0.0;
        if (t != 0.f) {
          *rotated = 1;
          const double t64 = double(t), q = fma(t64, t64, 1.0), c = cos_of(t64, q), ic = q * c;
          alpha = t64 * rab;
          beta = t64 * rba;
          sv[a] *= c; sv[b] *= c;
          si[a] *= ic; si[b] *= ic;
        }
        al[k] = alpha; al[npair + k] = beta;
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < JAC_BLOCKS; ++q) {
        const int K = bK[q], L = bL[q];
        if (L < 0) continue;
        const double aK = al[K], eK = al[npair + K], aL = al[L], eL = al[npair + L];
        if (aK == 0.0 && aL == 0.0) continue;
        const int a = pj[K], b = pj[npair + K], u = pj[L], v = pj[npair + L];
        auto at = [&](int i, int j) -> double& { return i >= j ? A[i * ld + j] : A[j * ld + i]; };
        const bool hb = b < p, hv = v < p;
        const double xau = at(a, u), xav = hv ? at(a, v) : 0.0;
        const double xbu = hb ? at(b, u) : 0.0, xbv = hb && hv ? at(b, v) : 0.0;
        const double yau = fma(-aL, xav, xau), yav = fma(eL, xau, xav);
        const double ybu = fma(-aL, xbv, xbu), ybv = fma(eL, xbu, xbv);
        at(a, u) = fma(-aK, ybu, yau);
        if (hv) at(a, v) = fma(-aK, ybv, yav);
        if (K != L && hb) at(b, u) = fma(eK, yau, ybu);     // K == L: the entry (a, v) again
        if (hb && hv) at(b, v) = fma(eK, yav, ybv);
      }
      for (int e = JAC_THREADS - 1 - int(threadIdx.x); e < 3 * npair; e += JAC_THREADS) {
        if (e < 2 * npair) {                               // b; the last warps have the fewest blocks
          const int k = e >> 1, a = pj[k], b = pj[npair + k];
          if (al[k] == 0.0) continue;
          const double x = bv[2 * a + (e & 1)], y = bv[2 * b + (e & 1)];
          bv[2 * a + (e & 1)] = fma(-al[k], y, x);
          bv[2 * b + (e & 1)] = fma(al[npair + k], x, y);
        } else if (r + 1 < P2 - 1) {                       // the next round's ratios
          const int k = e - 2 * npair;
          int a, b;
          jac_pair(k, r + 1, P2, a, b);
          if (b < p) {
            rt[k] = sv[b] * si[a];
            rt[npair + k] = sv[a] * si[b];
          }
        }
      }
      __syncthreads();
    }
    const bool more = *rotated != 0;
    for (int e = threadIdx.x; e < p * p; e += blockDim.x) {      // S back into the matrix and b
      const int i = e / p, j = e - i * p;
      if (j <= i) A[i * ld + j] *= sv[i] * sv[j];
    }
    for (int e = threadIdx.x; e < 2 * p; e += blockDim.x) bv[e] *= sv[e >> 1];
    __syncthreads();
    for (int i = threadIdx.x; i < p; i += blockDim.x) sv[i] = si[i] = 1.0;
    __syncthreads();
    if (!more) break;
  }
  // threshold on the eigenvalues lambda = s^2: tol > 0 absolute on s, < 0 relative to s_max,
  // 0: every positive s
  double lmax = 0.0;
  for (int i = threadIdx.x; i < p; i += blockDim.x) lmax = fmax(lmax, A[i * ld + i]);
  lmax = block_max(lmax);
  const double un = scalbn(1.0, ex);                       // eigenvalues of the unscaled matrix
  const double thr = tol > 0.0 ? tol * tol : (tol < 0.0 ? tol * tol * (un * lmax) : 0.0);
  for (int e = threadIdx.x; e < 2 * p; e += blockDim.x) {  // z = Lambda~^-1 W^T b
    const int i = e >> 1;
    const double lam = un * A[i * ld + i];
    bv[e] = (thr > 0.0 ? lam >= thr : lam > 0.0) ? bv[e] / lam : 0.0;
  }
  // x' = W z: the rotations in reverse order, a batch of rounds' tangents at a time (the matrix
  // is no longer needed; its storage holds their cosines and sines)
  const int batch = max(1, (p * ld) / (2 * npair));
  double* lc = A;
  for (int r1 = nround; r1 > 0; r1 -= batch) {
    const int r0 = max(0, r1 - batch), cnt = (r1 - r0) * npair;
    double* ls = lc + cnt;
    __syncthreads();
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
      const double t = double(tl[size_t(r0) * npair + e]);
      const double c = t != 0.0 ? cos_of(t) : 1.0;
      lc[e] = c;
      ls[e] = t * c;
    }
    __syncthreads();
    if (threadIdx.x < 2 * TSVD_MAX_NZ / 2) {               // the threads of one named barrier
      for (int r = r1 - 1; r >= r0; --r) {
        for (int e = threadIdx.x; e < 2 * npair; e += TSVD_MAX_NZ) {
          const int k = e >> 1;
          const double c = lc[(r - r0) * npair + k], s = ls[(r - r0) * npair + k];
          int a, b;
          jac_pair(k, r % (P2 - 1), P2, a, b);
          if (s == 0.0 || b >= p) continue;
          const double x = bv[2 * a + (e & 1)], y = bv[2 * b + (e & 1)];
          bv[2 * a + (e & 1)] = c * x + s * y;
          bv[2 * b + (e & 1)] = c * y - s * x;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(TSVD_MAX_NZ) : "memory");
      }
    }
  }
  __syncthreads();
  bool bad = false;
  for (int e = threadIdx.x; e < 2 * p; e += blockDim.x) {
    xo[e] = bv[e];
    if (!isfinite(bv[e])) bad = true;
  }
  for (int e = 2 * p + threadIdx.x; e < 2 * n; e += blockDim.x) xo[e] = 0.0;
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) d.status[m] = bad ? EDT_ENONFINITE : EDT_OK;
}

}  // namespace

size_t tsvd_smem_bytes(int p) {
  const size_t P2 = (p + 1) & ~1;
  return (size_t(p) * (p + 1) + 4 * p + 2 * P2 + 32) * sizeof(double) + (P2 + 1) * sizeof(int);
}

// one subproblem's rotation log: the tangent, which is chosen in FP32, of every pair of every round of the
// most sweeps
size_t tsvd_log_floats(int p) {
  const size_t P2 = (p + 1) & ~1;
  return size_t(JAC_MAX_SWEEPS) * (P2 - 1) * (P2 / 2);
}

cudaError_t prepare_variants() {
  return allow_smem(tsvd_jacobi_kernel, tsvd_smem_bytes(TSVD_MAX_NZ));
}

cudaError_t launch_solve_variant(const Dev& d, cudaStream_t s) {
  const int n = d.nz;
  if (d.kz_p) {
    // lam = alpha trace(G) of the unrestricted system
    cudaError_t e = launch_trace_diag(d, s);
    if (e != cudaSuccess) return e;
    kzv_t_kernel<<<dim3((n * n + 255) / 256, d.nsub), 256, 0, s>>>(d);
    kzv_g_kernel<<<dim3((n * n + 2 * n + 255) / 256, d.nsub), 256, 0, s>>>(d);
    if (d.solver == EDT_SOLVE_TSVD) {
      tsvd_jacobi_kernel<<<d.nsub, JAC_THREADS, tsvd_smem_bytes(n), s>>>(d, d.kz_G, d.kz_b, d.kz_x);
    } else {
      // damped: per-subproblem Cholesky of G' + lam I (size p(m)) in the projected arrays
      Dev v = d;
      v.G = d.kz_G; v.b = d.kz_b; v.x = d.kz_x; v.dinv = d.kz_T; v.L32 = nullptr; v.dinv32 = nullptr;
      v.sub_n = d.kz_p; v.sub_goff = d.kz_goff; v.sub_voff = d.kz_voff; v.sub_order = nullptr;
      e = launch_chol_var(v, n, s);
      if (e != cudaSuccess) return e;
    }
    kzv_back_kernel<<<dim3((2 * n + 255) / 256, d.nsub), 256, 0, s>>>(d);
  } else {
    tsvd_jacobi_kernel<<<d.nsub, JAC_THREADS, tsvd_smem_bytes(n), s>>>(d, d.G, d.b, d.x);
  }
  return cudaGetLastError();
}

}  // namespace edt
