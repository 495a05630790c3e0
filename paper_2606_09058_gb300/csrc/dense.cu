// Small dense kernels around the GEMM core: diagonal-block Cholesky, triangular solves
// against a diagonal block, the two-sided reduction of a diagonal block, the compact-WY
// T factor, and elementwise helpers (phase application, Hermitian mirror, eigenvector
// phase, spinor overlap).
#include "dense.h"

#include <algorithm>
#include <cmath>

namespace gks {

// acc -= a * b, acc -= a * conj(b): two fused operations per component.
__device__ __forceinline__ void msub(double& acc, double a, double b) { acc = fma(-a, b, acc); }
__device__ __forceinline__ void msub(zc& acc, zc a, zc b) {
  acc.x = fma(-a.x, b.x, acc.x);
  acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(-a.x, b.y, acc.y);
  acc.y = fma(-a.y, b.x, acc.y);
}
__device__ __forceinline__ void msubc(double& acc, double a, double b) { acc = fma(-a, b, acc); }
__device__ __forceinline__ void msubc(zc& acc, zc a, zc b) { msub(acc, a, conjg(b)); }

// the value of lane src of each group of G lanes
template <int G>
__device__ __forceinline__ double shfl_g(double v, int src) { return __shfl_sync(0xffffffffu, v, src, G); }
template <int G>
__device__ __forceinline__ zc shfl_g(zc v, int src) { return zc{shfl_g<G>(v.x, src), shfl_g<G>(v.y, src)}; }

// Diagonal blocks (64 x 64) on a cluster of C CTAs, in sub-blocks (32 columns of the
// Cholesky factorization, 8 of the two-sided reduction).  One SM does 1.7 FP64 multiply-adds
// per clock: the 64^3 operations of a complex two-sided reduction alone keep it busy for 0.3
// ms, so the panel rows and the trailing updates are spread over the cluster (data in global
// memory, L2 reads), with two cluster barriers per sub-block; the diagonal parts, a serial
// chain of 67-clock operations, are done by every CTA for itself.
// Measured, one block (complex / real): two-sided reduction 794 / 265 us on one CTA column by
// column, 163 / 80 us here (190 / 90 with sub-blocks of 16, 420 / 153 on one CTA); Cholesky 207 / 103 us on one CTA,
// 110 / 76 us with sub-blocks of 8, 83 / 59 us here.
constexpr int kDiagThreads = 256;
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Cholesky of the nb x nb diagonal block of A at (k0, k0) in place (lower, A = L L^H), one
// cluster per batch item.  A non-positive or non-finite pivot records GKS_ENOTSPD with the
// global column; the block is then left part way.
// A 32-column sub-block's own part: thread (i, q) holds row i, columns q + 8 t in registers; a
// step scales the pivot column (one warp), then every element takes its rank-one update, the
// next pivot's owner going on to its reciprocal square root while the others still update.
template <typename T, int C>
__global__ void __launch_bounds__(kDiagThreads) potf2_kernel(T* A, int lda, long long sA, int k0, int nb,
                                                             DevStatus* st) {
  constexpr int SB = 32;
  __shared__ T l11[SB][SB + 1], raw[SB], v[SB][SB + 1];
  __shared__ double rd[SB], s_d;
  __shared__ int fail;
  const int z = blockIdx.y, rank = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  A += z * sA + (size_t)k0 * lda + k0;
  if (tid == 0) fail = -1;
  for (int c0 = 0; c0 < nb; c0 += SB) {
    const int kb = min(SB, nb - c0), m = nb - c0 - kb;
    T* Ab = A + (size_t)c0 * lda + c0;
    const int i = tid >> 3, q = tid & 7;
    T a[4];
#pragma unroll
    for (int t = 0; t < 4; t++) {
      const int j = q + 8 * t;
      a[t] = (i < kb && j <= i) ? ldcg(Ab + (size_t)i * lda + j) : zero<T>();
    }
    // pivot: 1 / sqrt, then sqrt with one correction step (half the chain of a square root and a
    // division on this pipe, 434 + 686 clocks)
    auto pivot = [&](int k, double piv) {
      if (!(piv > 0.0) || !isfinite(piv)) {
        fail = c0 + k;
      } else {
        const double inv = rsqrt(piv), d0 = piv * inv;
        rd[k] = inv;
        s_d = fma(0.5 * inv, fma(-d0, d0, piv), d0);
      }
    };
    __syncthreads();
    if (q == 0) raw[i] = a[0];
    if (tid == 0) pivot(0, re(a[0]));
    __syncthreads();
    for (int k = 0; k < kb && fail < 0; k++) {
      if (warp == 0 && lane < kb) {
        if (lane > k) l11[lane][k] = raw[lane] * rd[k];
        if (lane == k) l11[k][k] = from_real<T>(s_d);
        if (lane < k) l11[lane][k] = zero<T>();
      }
      __syncthreads();
      if (i > k && i < kb) {
        const T li = l11[i][k];
#pragma unroll
        for (int t = 0; t < 4; t++) {
          const int j = q + 8 * t;
          if (j > k && j <= i) {
            msubc(a[t], li, l11[j][k]);
            if (j == k + 1) {
              raw[i] = a[t];
              if (i == j) pivot(j, re(a[t]));
            }
          }
        }
      }
      __syncthreads();
    }
    if (fail >= 0) break;  // the same in every CTA of the cluster
    // rows below, one per warp, row r of CTA r % C: x L11^H = a
    if (m > 0) {
      for (int r = rank + C * warp; r < m; r += C * 8) {
        T* ar = A + (size_t)(c0 + kb + r) * lda + c0;
        T x = lane < kb ? ldcg(ar + lane) : zero<T>();
#pragma unroll 1
        for (int j = 0; j < kb; j++) {
          const T xj = shfl_g<32>(x * rd[j], j);
          if (lane > j && lane < kb) msubc(x, xj, l11[lane][j]);
          if (lane == j) x = xj;
        }
        if (lane < kb) ar[lane] = x;
      }
    }
    cluster_barrier();  // every CTA has read the diagonal part
    if (rank == 0)
      for (int e = tid; e < SB * SB; e += kDiagThreads) {
        const int r = e >> 5, c = e & 31;
        if (r < kb && c <= r) Ab[(size_t)r * lda + c] = l11[r][c];
      }
    if (m <= 0) break;
    for (int e = tid; e < m * SB; e += kDiagThreads) {
      const int r = e >> 5, g = e & 31;
      v[r][g] = g < kb ? ldcg(A + (size_t)(c0 + kb + r) * lda + c0 + g) : zero<T>();
    }
    __syncthreads();
    for (int e = rank * kDiagThreads + tid; e < m * m; e += C * kDiagThreads) {
      const int r = e / m, j = e - r * m;
      if (j > r) continue;
      T* p = A + (size_t)(c0 + kb + r) * lda + c0 + kb + j;
      T x = ldcg(p), y = zero<T>();
#pragma unroll 4
      for (int g = 0; g < SB; g += 2) {  // two chains
        msubc(x, v[r][g], v[j][g]);
        msubc(y, v[r][g + 1], v[j][g + 1]);
      }
      *p = x + y;
    }
    cluster_barrier();
  }
  if (fail >= 0 && rank == 0 && tid == 0) set_status(st ? st + z : nullptr, ST_ENOTSPD, k0 + fail);
}

// Triangular solves against one nb x nb lower-triangular block L (nb <= 64), by substitution
// (no explicit inverse: the diagonal blocks of the Cholesky factor of an overcomplete
// basis have condition numbers near 1e5).
//   TRSM_RIGHT_CONJ : B (nrhs x nb rows)  <- B L^-H   (x L^H = b: conj(L) x = b per row)
//   TRSM_LEFT       : B (nb x nrhs cols)  <- L^-1 B
//   TRSM_LEFT_CONJ  : B (nb x nrhs cols)  <- L^-H B   (backward: the reversed conj(L)^T)
// Every mode is forward substitution with one lower matrix, kept in shared memory by
// columns (conjugated or reversed while loading, padded to 64 with the identity).  G lanes
// share a right-hand side, each holding 64 / G of its entries in registers (entry G i +
// lane): a step broadcasts the solved entry by shuffles and every lane updates its own
// entries, so nothing but the columns of L is read.  The steps are a rolled loop on rotating
// registers (unrolled they are 30 to 100 KB of code that each launch runs through once).
// The FP64 pipe bounds it: one warp instruction per 64 clocks and SM partition whatever its
// active lanes, 19 clocks over the four: trsm_pick.
// Measured against 832 real right-hand sides: 184 us with a thread per right-hand side and
// 64 of them per CTA, 20 us here.
template <typename T, int MODE, int G>
__global__ void __launch_bounds__(512) trsm_block_kernel(const T* L, int ldl, long long sL, T* B, int ldb,
                                                         long long sB, int nb, int nrhs) {
  constexpr int E = 64 / G;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* lc = reinterpret_cast<T*>(smem_raw);                    // [column][64]
  double* rd = reinterpret_cast<double*>(lc + 64 * 64);       // 1 / diagonal
  const int z = blockIdx.y, tid = threadIdx.x, nt = blockDim.x;
  L += z * sL;
  B += z * sB;
  const int g = tid % G, r = (blockIdx.x * nt + tid) / G;
  const bool ok = r < nrhs;
  auto at = [&](int i) -> T* {  // entry i of this right-hand side, in solving order
    const int e = MODE == TRSM_LEFT_CONJ ? nb - 1 - i : i;
    return MODE == TRSM_RIGHT_CONJ ? B + (size_t)r * ldb + e : B + (size_t)e * ldb + r;
  };
  T x[E];
#pragma unroll
  for (int i = 0; i < E; i++) x[i] = (ok && G * i + g < nb) ? *at(G * i + g) : zero<T>();
#pragma unroll 8
  for (int e = tid; e < 64 * 64; e += nt) {
    const int i = e >> 6, j = e & 63;  // stored element (i, j), j <= i
    T v = (i == j) ? from_real<T>(1.0) : zero<T>();
    if (i < nb && j <= i) v = L[(size_t)i * ldl + j];
    if (MODE != TRSM_LEFT) v = conjg(v);
    // lower matrix by columns; backward: (i, j) of L is (nb - 1 - j, nb - 1 - i) of its reverse
    if (MODE == TRSM_LEFT_CONJ && i < nb && j < nb) lc[(nb - 1 - i) * 64 + nb - 1 - j] = v;
    else lc[j * 64 + i] = v;
  }
  __syncthreads();
  for (int i = tid; i < 64; i += nt) rd[i] = 1.0 / re(lc[i * 65]);
  __syncthreads();
#pragma unroll 1
  for (int J = 0; G * J < nb; J++) {  // x[i]: entries G (J + i) + g
    const T* col = lc + G * J * 64 + G * J + g;
#pragma unroll 1
    for (int jj = 0; jj < G; jj++, col += 64) {
      const T y = x[0] * rd[G * J + jj];
      const T xj = shfl_g<G>(y, jj);
      if (g > jj) msub(x[0], xj, col[0]);
      if (g == jj) x[0] = xj;
#pragma unroll
      for (int i = 1; i < E; i++) {
        if (i + J >= E) break;
        msub(x[i], xj, col[G * i]);
      }
    }
    if (ok && G * J + g < nb) *at(G * J + g) = x[0];
#pragma unroll
    for (int i = 0; i < E - 1; i++) x[i] = x[i + 1];
  }
}

// One cluster per batch item: the nb x nb diagonal block A <- L^-1 A L^-H (read from its lower
// triangle) with the diagonal block L, in sub-blocks of kSub columns: A11 by the two-sided
// column recurrence
//   alpha_k = a_kk / l_kk^2,  v = a(k+1:, k)/l_kk - (alpha_k/2) l(k+1:, k),
//   A(k+1:, k+1:) -= l v^H + v l^H,  r_k = v - (alpha_k/2) l(k+1:, k),
// and its in-block solve, then W = A21 L11^-H, V = W - L21 A11/2, A22 -= L21 V^H + V L21^H,
// R = V - L21 A11/2, and finally L^-1 [R_0 R_1 ...] by forward substitution, a warp per
// column.  Writes the lower triangle back into A and the full Hermitian block into F (ldF).
constexpr int kSub = 8;
__device__ __forceinline__ void diag_bar() { asm volatile("bar.sync 1, 64;\n" ::: "memory"); }
template <typename T, int C>
__global__ void __launch_bounds__(kDiagThreads) hegst_diag_kernel(T* A, int lda, long long sA, const T* L, int ldl,
                                                                  long long sL, int k0, int nb, T* F, int ldF,
                                                                  long long sF) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* l = reinterpret_cast<T*>(smem_raw);  // [64][65]
  __shared__ T s11[kSub][kSub + 1];
  __shared__ double rd[64];
  T* v = l + 64 * 65;  // [64][kSub + 1]
  constexpr int LD = 65, LV = kSub + 1;
  const int z = blockIdx.y, rank = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  A += z * sA + (size_t)k0 * lda + k0;
  L += z * sL + (size_t)k0 * ldl + k0;
  F += z * sF;
#pragma unroll 4
  for (int e = tid; e < nb * nb; e += kDiagThreads) {
    const int i = e / nb, j = e - i * nb;
    const T x = j <= i ? L[(size_t)i * ldl + j] : zero<T>();
    l[i * LD + j] = x;
  }
  __syncthreads();
  if (tid < nb) rd[tid] = 1.0 / re(l[tid * 66]);
  for (int c0 = 0; c0 < nb; c0 += kSub) {
    const int kb = min(kSub, nb - c0), m = nb - c0 - kb;
    const T* lb = l + c0 * LD + c0;
    __syncthreads();
    if (tid < kSub * kSub) {  // two warps (two SM partitions), one element each
      const int i = tid >> 3, j = tid & 7;
      T a = (i < kb && j <= i) ? ldcg(A + (size_t)(c0 + i) * lda + c0 + j) : zero<T>();
      s11[i][j] = a;
      diag_bar();
      for (int k = 0; k < kb; k++) {
        const double rk = rd[c0 + k], alpha = re(s11[k][k]) * rk * rk;
        const T hl = (0.5 * alpha) * lb[min(i, kb - 1) * LD + k];
        if (j == k && i > k) {
          a = a * rk - hl;
          s11[i][k] = a;
        }
        diag_bar();
        if (j > k && j <= i && i < kb) {
          msubc(a, lb[i * LD + k], s11[j][k]);
          msubc(a, s11[i][k], lb[j * LD + k]);
          if (j == k + 1 && i == j) s11[i][j] = a;  // the next step's alpha
        }
        diag_bar();
        if (j == k && i > k) a = a - hl;
        if (j == k && i == k) a = from_real<T>(alpha);
      }
      // strictly lower part: forward substitution with L11, rows top down
      s11[i][j] = a;
      diag_bar();
      for (int k = 1; k < kb; k++) {
        if (i == k && j < k) {
          a = a * rd[c0 + k];
          s11[k][j] = a;
        }
        diag_bar();
        if (i > k && i < kb && j < k) msub(a, lb[i * LD + k], s11[k][j]);
      }
      diag_bar();
      if (i > j) s11[j][i] = conjg(s11[i][j]);  // the full Hermitian 8 x 8
    }
    __syncthreads();
    // rows below, one per 8 lanes: W, V
    constexpr int NR = (56 + 32 * C - 1) / (32 * C);  // rows per 8 lanes
    const int g = tid & 7;
    T x[NR], h[NR];
#pragma unroll
    for (int q = 0; q < NR; q++) {
      const int r = rank + C * ((tid >> 3) + 32 * q);
      T* ar = A + (size_t)(c0 + kb + r) * lda + c0;
      x[q] = (r < m && g < kb) ? ldcg(ar + g) : zero<T>();
      h[q] = zero<T>();
      if (__any_sync(0xffffffffu, r < m)) {
        for (int j = 0; j < kb; j++) {
          const T xj = shfl_g<8>(x[q] * rd[c0 + j], j);
          if (g > j && g < kb) msubc(x[q], xj, lb[g * LD + j]);
          if (g == j) x[q] = xj;
        }
        if (r < m && g < kb) {
          const T* lr = l + (c0 + kb + r) * LD + c0;
          for (int j = 0; j < kb; j++) mac(h[q], lr[j], s11[j][g]);
          h[q] = 0.5 * h[q];
          x[q] = x[q] - h[q];
          ar[g] = x[q];
        }
      }
    }
    cluster_barrier();  // every CTA has read the 8 x 8 block
    if (rank == 0 && tid < kSub * kSub) {
      const int i = tid >> 3, j = tid & 7;
      if (i < kb && j < kb) {
        F[(size_t)(c0 + i) * ldF + c0 + j] = s11[i][j];
        if (j <= i) A[(size_t)(c0 + i) * lda + c0 + j] = s11[i][j];
      }
    }
    if (m <= 0) break;
    for (int e = tid; e < m * kSub; e += kDiagThreads) {
      const int i = e >> 3, q = e & 7;
      v[i * LV + q] = q < kb ? ldcg(A + (size_t)(c0 + kb + i) * lda + c0 + q) : zero<T>();
    }
    __syncthreads();
    for (int e = rank * kDiagThreads + tid; e < m * m; e += C * kDiagThreads) {
      const int i = e / m, j = e - i * m;
      if (j > i) continue;
      T* p = A + (size_t)(c0 + kb + i) * lda + c0 + kb + j;
      T a = ldcg(p);
      const T *li = l + (c0 + kb + i) * LD + c0, *lj = l + (c0 + kb + j) * LD + c0;
#pragma unroll
      for (int q = 0; q < kSub; q++) {  // columns past kb of L are other data: v is zero there
        if (q >= kb) break;
        msubc(a, li[q], v[j * LV + q]);
        msubc(a, v[i * LV + q], lj[q]);
      }
      *p = a;
    }
    cluster_barrier();
#pragma unroll
    for (int q = 0; q < NR; q++) {
      const int r = rank + C * ((tid >> 3) + 32 * q);
      if (r < m && g < kb) A[(size_t)(c0 + kb + r) * lda + c0 + g] = x[q] - h[q];
    }
  }
  cluster_barrier();  // every R is in place
  // column c: rows from its sub-block's end, x_i = (g_i - sum L_ik x_k) / l_ii
  for (int c = rank + C * warp; c < nb; c += C * (kDiagThreads / 32)) {
    const int s0 = min(nb, (c / kSub + 1) * kSub);
    T x0 = zero<T>(), x1 = zero<T>();
    if (lane >= s0 && lane < nb) x0 = ldcg(A + (size_t)lane * lda + c);
    if (lane + 32 >= s0 && lane + 32 < nb) x1 = ldcg(A + (size_t)(lane + 32) * lda + c);
#pragma unroll 1
    for (int i = s0; i < nb; i++) {
      const T xi = shfl_g<32>(i < 32 ? x0 : x1, i & 31) * rd[i];
      if (i < 31 && lane > i && lane < nb) msub(x0, l[lane * LD + i], xi);
      if (lane + 32 > i && lane + 32 < nb) msub(x1, l[(lane + 32) * LD + i], xi);
      if (lane == (i & 31)) {
        if (i < 32) x0 = xi;
        else x1 = xi;
      }
    }
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int i = lane + 32 * h;
      const T xv = h ? x1 : x0;
      if (i >= s0 && i < nb) {
        A[(size_t)i * lda + c] = xv;
        F[(size_t)i * ldF + c] = xv;
        F[(size_t)c * ldF + i] = conjg(xv);
      }
    }
  }
}

// Compact WY T factor for H_1 H_2 ... H_k = I - V T V^H with H_i = I - tau_i v_i v_i^H:
// T upper triangular, T_ii = tau_i, and T^-1 = diag(1 / tau) + the strictly upper part of
// G = V^H V, so each column is a back substitution of its own,
//   t_i = tau_i,  t_r = -tau_r sum_{r < c <= i} G_rc t_c  (r = i - 1 .. 0),
// a warp per column (lanes hold rows lane and lane + 32; k <= 64), 4 columns per CTA.  The
// column-by-column form T[0:i, i] = -tau_i T[0:i, 0:i] G[0:i, i] on one CTA took 372 us
// (complex, k = 64) and 144 us (real); this one 38 and 26 us.
template <typename T>
__global__ void __launch_bounds__(128) larft_kernel(const T* G, int ldG, long long sG, const double* tau,
                                                    long long stau, int k, T* Tm, int ldT, long long sT) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* gs = reinterpret_cast<T*>(smem_raw);  // [64][65], column c of G in row c
  __shared__ double ts[64];
  const int z = blockIdx.y, tid = threadIdx.x, lane = tid & 31, i = blockIdx.x * 4 + (tid >> 5);
  G += z * sG;
  tau += z * stau;
  Tm += z * sT;
#pragma unroll 8
  for (int e = tid; e < 64 * 64; e += 128) {
    const int r = e >> 6, c = e & 63;
    if (r < c && c < k) gs[c * 65 + r] = G[(size_t)r * ldG + c];
  }
  if (tid < k && tid < 64) ts[tid] = tau[tid];
  __syncthreads();
  if (i >= k) return;
  T a0 = zero<T>(), a1 = zero<T>();  // sums of rows lane, lane + 32, then the entries
  if (lane == (i & 31)) (i < 32 ? a0 : a1) = from_real<T>(ts[i]);
#pragma unroll 1
  for (int c = i; c > 0; c--) {
    const T tc = shfl_g<32>(c < 32 ? a0 : a1, c & 31);
    if (lane < c) mac(a0, gs[c * 65 + lane], tc);
    if (lane + 32 < c) mac(a1, gs[c * 65 + lane + 32], tc);
    if (lane == ((c - 1) & 31)) {
      T& a = c - 1 < 32 ? a0 : a1;
      a = (-ts[c - 1]) * a;
    }
  }
  if (lane < k) Tm[(size_t)lane * ldT + i] = lane <= i ? a0 : zero<T>();
  if (lane + 32 < k) Tm[(size_t)(lane + 32) * ldT + i] = lane + 32 <= i ? a1 : zero<T>();
}

// X[b][i][c] = ph[b][i] * Z[b][i][c] for the leading `cols` columns (Z real, X of type T)
template <typename T>
__global__ void apply_phase_kernel(T* X, int ldx, long long sX, const double* Z, int ldz, long long sZ,
                                   const T* ph, long long sph, int n, int cols) {
  const int z = blockIdx.z;
  X += z * sX;
  Z += z * sZ;
  ph += z * sph;
  for (int i = blockIdx.y; i < n; i += gridDim.y) {
    T p = ph[i];
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < cols; c += gridDim.x * blockDim.x)
      X[(size_t)i * ldx + c] = p * Z[(size_t)i * ldz + c];
  }
}

// Upper triangle <- conj(lower triangle); diagonal made real.  One CTA per 32 x 32 tile of the
// lower triangle, transposed through shared memory so that both sides move in whole lines
// (element by element, the writes down the columns took 93 us for four of order 1664; 29 us).
template <typename T>
__global__ void __launch_bounds__(256) mirror_lower_kernel(T* A, int lda, long long sA, int n) {
  if (blockIdx.x > blockIdx.y) return;
  __shared__ T tile[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  A += blockIdx.z * sA;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const int r = warp + 8 * q;
    if (r0 + r < n && c0 + lane <= r0 + r) tile[r][lane] = A[(size_t)(r0 + r) * lda + c0 + lane];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const int c = warp + 8 * q;  // row of the mirrored tile
    const int i = c0 + c, j = r0 + lane;
    if (j >= n || j < i) continue;
    const T v = tile[lane][c];
    A[(size_t)i * lda + j] = i == j ? from_real<T>(re(v)) : conjg(v);
  }
}

// Column phase convention: the entry of largest modulus (lowest row on ties) becomes
// real and positive.  One CTA of 32 warps per 32 columns: lanes along the columns (the
// contiguous direction), each warp every 32nd row.
template <typename T>
__global__ void __launch_bounds__(1024) column_phase_kernel(T* C, int ldc, long long sC, int rows, int cols) {
  __shared__ double sb[32][33];
  __shared__ int si[32][33];
  __shared__ T sf[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, col = blockIdx.x * 32 + lane;
  C += blockIdx.y * sC + col;
  double best = -1.0;
  int bi = 0;
  if (col < cols)
#pragma unroll 4
    for (int i = warp; i < rows; i += 32) {
      const double a = abs2(C[(size_t)i * ldc]);
      if (a > best) { best = a; bi = i; }
    }
  sb[warp][lane] = best;
  si[warp][lane] = bi;
  __syncthreads();
  {  // warp w: column w, lanes over the warps' candidates
    best = sb[lane][warp];
    bi = si[lane][warp];
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if (lane == 0 && blockIdx.x * 32 + warp < cols) {
      const T p = C[(size_t)bi * ldc - col + blockIdx.x * 32 + warp];
      const double mag = sqrt(abs2(p));
      sf[warp] = mag > 0.0 ? conjg(p) * (1.0 / mag) : from_real<T>(1.0);
    }
  }
  __syncthreads();
  if (col >= cols) return;
  const T f = sf[lane];
#pragma unroll 4
  for (int i = warp; i < rows; i += 32) C[(size_t)i * ldc] = C[(size_t)i * ldc] * f;
}

// Fill dst (2n x 2n) with diag(S, S) from the n x n S (lower triangle valid).
template <typename T>
__global__ void spinor_overlap_kernel(T* dst, long long sd, const T* S, int lds, long long ss, int n) {
  const int z = blockIdx.z;
  dst += z * sd;
  S += z * ss;
  const int m = 2 * n;
  for (int i = blockIdx.y; i < m; i += gridDim.y)
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < m; j += gridDim.x * blockDim.x) {
      T v = zero<T>();
      if ((i < n) == (j < n)) {
        int a = i % n, b = j % n;
        v = (b <= a) ? S[(size_t)a * lds + b] : conjg(S[(size_t)b * lds + a]);
      }
      dst[(size_t)i * m + j] = v;
    }
}

// Loewdin factor V = U diag(s)^-1/2 (paper Sec. 3.1 Part 2-2) from the eigenvectors U
// (ldu, sU) and eigenvalues s (ss per item) of S; a non-positive eigenvalue reports
// GKS_ENOTSPD with its index and zeroes the column.
template <typename T>
__global__ void lowdin_factor_kernel(const T* U, int ldu, long long sU, const double* sv, long long ss, T* V, int ldv,
                                     long long sV, int n, DevStatus* st) {
  const int z = blockIdx.z;
  U += z * sU;
  V += z * sV;
  sv += z * ss;
  for (int i = blockIdx.y; i < n; i += gridDim.y)
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
      const double sj = sv[j];
      if (!(sj > 0.0)) {
        if (i == 0) set_status(st ? st + z : nullptr, ST_ENOTSPD, j);
        V[(size_t)i * ldv + j] = zero<T>();
      } else {
        V[(size_t)i * ldv + j] = U[(size_t)i * ldu + j] * (1.0 / sqrt(sj));
      }
    }
}

// ------------------------------------------------------------------ launchers

static dim3 grid2d(int rows, int cols, int count) {
  int gx = (cols + 255) / 256;
  if (gx > 16) gx = 16;
  if (gx < 1) gx = 1;
  int gy = rows < 2048 ? (rows > 0 ? rows : 1) : 2048;
  return dim3(gx, gy, count);
}

// CTAs per diagonal block: the largest cluster with all items side by side (clusters of 8 and 4
// do not fill every processing cluster's SMs).  A second wave costs more than a wider cluster
// gains.  Two-sided reduction of 64 x 64 blocks, complex, in us on 8 / 4 / 2 / 1 CTAs: 8 items
// 163 / 194 / 266 / 421, 19 items 208 / 194 / 266 / 421, 76 items 585 / 448 / 266 / 423, 1000
// items 5779 / 3760 / 2837 / 2552; Cholesky 85 / 89 / 110 / 154, 112 / 90 / 111 / 153, 218 / 165 /
// 112 / 155, 2129 / 1306 / 956 / 784.  Real blocks cross at the same counts.
static int diag_ctas(int count) { return count <= 8 ? 8 : count <= 32 ? 4 : count <= 76 ? 2 : 1; }

// Launch of a diagonal-block kernel on one cluster per item.
template <typename... P, typename... Q>
static void diag_launch(void (*k)(P...), int ctas, int count, size_t sm, cudaStream_t s, Q... args) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  cfg.gridDim = dim3(ctas, count);
  cfg.blockDim = dim3(kDiagThreads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ctas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  count_launch();
  cudaLaunchKernelEx(&cfg, k, args...);
}

template <typename T>
void potf2(T* A, int lda, long long sA, int k0, int nb, DevStatus* st, int count, cudaStream_t s) {
  auto run = [&](auto k, int c) { diag_launch(k, c, count, 0, s, A, lda, sA, k0, nb, st); };
  const int c = diag_ctas(count);
  if (c == 8) run(potf2_kernel<T, 8>, c);
  else if (c == 4) run(potf2_kernel<T, 4>, c);
  else if (c == 2) run(potf2_kernel<T, 2>, c);
  else run(potf2_kernel<T, 1>, c);
}

template <typename T, int MODE, int G>
static void trsm_launch(const T* L, int ldl, long long sL, T* B, int ldb, long long sB, int nb, int nrhs, int count,
                        int w, cudaStream_t s) {
  const int sm = (int)(64 * 64 * sizeof(T) + 64 * sizeof(double)), per = 32 * w / G;
  cudaFuncSetAttribute(trsm_block_kernel<T, MODE, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  count_launch();
  trsm_block_kernel<T, MODE, G><<<dim3((nrhs + per - 1) / per, count), 32 * w, sm, s>>>(L, ldl, sL, B, ldb, sB, nb,
                                                                                        nrhs);
}

// Lanes per right-hand side and warps per CTA (4 to 16): those with the least FP64 pipe time
// of the fullest SM, which is the instructions of a step (four right-hand sides: 20 / 24 / 32
// for 8 / 16 / 32 lanes complex, 5.5 / 7 / 10 real) times 19 clocks for each of its warps or 64
// for each on its fullest partition.  A last wave of a few CTAs costs as much as a full one
// (4992 right-hand sides in CTAs of 32 are 156 on 152 SMs).
// Measured, all launches of a call (32 lanes up to 1216 right-hand sides, 8 above, 4 or 8
// warps, against this rule): order 4992 complex 32.2 / 29.1 ms, eight of order 832 complex
// 5.5 / 5.0, a spinor problem of order 2496 12.2 / 11.2; order 832 real unchanged.
template <typename T, int MODE>
static void trsm_pick(const T* L, int ldl, long long sL, T* B, int ldb, long long sB, int nb, int nrhs, int count,
                      cudaStream_t s) {
  int G = 8, w = 4;
  double best = 1e300;
  for (int g = 8; g <= 32; g *= 2) {
    const int e = 64 / g - 1;
    const double instr = sizeof(T) == 16 ? 6.0 + 2.0 * e : 2.0 + 0.5 * e;
    for (int v = 4; v <= 16; v++) {
      const long long per = 32 * v / g, ctas = (nrhs + per - 1) / per * count;
      const double warps = (double)((ctas + 151) / 152) * v;
      const double t = instr * std::max(19.0 * warps, 64.0 * std::ceil(warps / 4.0));
      if (t < best) {
        best = t;
        G = g;
        w = v;
      }
    }
  }
  if (G == 8) trsm_launch<T, MODE, 8>(L, ldl, sL, B, ldb, sB, nb, nrhs, count, w, s);
  else if (G == 16) trsm_launch<T, MODE, 16>(L, ldl, sL, B, ldb, sB, nb, nrhs, count, w, s);
  else trsm_launch<T, MODE, 32>(L, ldl, sL, B, ldb, sB, nb, nrhs, count, w, s);
}

template <typename T>
void trsm_block(int mode, const T* L, int ldl, long long sL, T* B, int ldb, long long sB, int nb, int nrhs,
                int count, cudaStream_t s) {
  if (nrhs <= 0 || nb <= 0 || count <= 0) return;
  if (mode == TRSM_RIGHT_CONJ) trsm_pick<T, TRSM_RIGHT_CONJ>(L, ldl, sL, B, ldb, sB, nb, nrhs, count, s);
  else if (mode == TRSM_LEFT) trsm_pick<T, TRSM_LEFT>(L, ldl, sL, B, ldb, sB, nb, nrhs, count, s);
  else trsm_pick<T, TRSM_LEFT_CONJ>(L, ldl, sL, B, ldb, sB, nb, nrhs, count, s);
}

template <typename T>
void hegst_diag(T* A, int lda, long long sA, const T* L, int ldl, long long sL, int k0, int nb, T* F, int ldF,
                long long sF, int count, cudaStream_t s) {
  const size_t sm = sizeof(T) * (64 * 65 + 64 * (kSub + 1));
  auto run = [&](auto k, int c) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    diag_launch(k, c, count, sm, s, A, lda, sA, L, ldl, sL, k0, nb, F, ldF, sF);
  };
  const int c = diag_ctas(count);
  if (c == 8) run(hegst_diag_kernel<T, 8>, c);
  else if (c == 4) run(hegst_diag_kernel<T, 4>, c);
  else if (c == 2) run(hegst_diag_kernel<T, 2>, c);
  else run(hegst_diag_kernel<T, 1>, c);
}

template <typename T>
void larft(const T* G, int ldG, long long sG, const double* tau, long long stau, int k, T* Tm, int ldT,
           long long sT, int count, cudaStream_t s) {
  const size_t sm = sizeof(T) * 64 * 65;
  cudaFuncSetAttribute(larft_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  count_launch();
  larft_kernel<T><<<dim3((k + 3) / 4, count), 128, sm, s>>>(G, ldG, sG, tau, stau, k, Tm, ldT, sT);
}

template <typename T>
void apply_phase(T* X, int ldx, long long sX, const double* Z, int ldz, long long sZ, const T* ph, long long sph,
                 int n, int cols, int count, cudaStream_t s) {
  count_launch();
  apply_phase_kernel<T><<<grid2d(n, cols, count), 256, 0, s>>>(X, ldx, sX, Z, ldz, sZ, ph, sph, n, cols);
}

template <typename T>
void lowdin_factor(const T* U, int ldu, long long sU, const double* sv, long long ss, T* V, int ldv, long long sV,
                   int n, DevStatus* st, int count, cudaStream_t s) {
  count_launch();
  lowdin_factor_kernel<T><<<grid2d(n, n, count), 256, 0, s>>>(U, ldu, sU, sv, ss, V, ldv, sV, n, st);
}

template <typename T>
void mirror_lower(T* A, int lda, long long sA, int n, int count, cudaStream_t s) {
  if (n <= 0) return;
  count_launch();
  const int t = (n + 31) / 32;
  mirror_lower_kernel<T><<<dim3(t, t, count), 256, 0, s>>>(A, lda, sA, n);
}

template <typename T>
void column_phase(T* C, int ldc, long long sC, int rows, int cols, int count, cudaStream_t s) {
  if (cols <= 0) return;
  count_launch();
  column_phase_kernel<T><<<dim3((cols + 31) / 32, count), 1024, 0, s>>>(C, ldc, sC, rows, cols);
}

template <typename T>
void spinor_overlap(T* dst, long long sd, const T* S, int lds, long long ss, int n, int count, cudaStream_t s) {
  count_launch();
  spinor_overlap_kernel<T><<<grid2d(2 * n, 2 * n, count), 256, 0, s>>>(dst, sd, S, lds, ss, n);
}

// Seeded test pencils for the width tuner (no input data needed): splitmix64 of the
// element index gives uniform numbers.  hermitian = 1: entries in [-1, 1] (both parts);
// hermitian = 0: S = I + entries in [-0.5, 0.5]/m off the diagonal (diagonally dominant).
__device__ __forceinline__ double tune_uniform(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  x ^= x >> 31;
  return (double)(x >> 11) * 0x1.0p-53;
}

template <typename T>
__global__ void tune_pencil_kernel(T* A, int m, int hermitian) {
  const int z = blockIdx.z;
  A += (size_t)z * m * m;
  for (int i = blockIdx.y; i < m; i += gridDim.y)
    for (int jj = blockIdx.x * blockDim.x + threadIdx.x; jj <= i; jj += gridDim.x * blockDim.x) {
      const unsigned long long id = (((unsigned long long)z * m + i) * m + jj) * 2ull;
      const double a = 2.0 * tune_uniform(id) - 1.0, b = 2.0 * tune_uniform(id + 1) - 1.0;
      T v;
      if constexpr (sizeof(T) == 16) v = zc{a, i == jj ? 0.0 : b};
      else v = a;
      if (!hermitian) v = (i == jj) ? from_real<T>(1.0) : (0.5 / m) * v;
      A[(size_t)i * m + jj] = v;
    }
}

template <typename T>
void tune_pencil(T* A, int m, int count, int hermitian, cudaStream_t s) {
  count_launch();
  tune_pencil_kernel<T><<<grid2d(m, m, count), 256, 0, s>>>(A, m, hermitian);
}

#define INST(T)                                                                                         \
  template void potf2<T>(T*, int, long long, int, int, DevStatus*, int, cudaStream_t);                   \
  template void trsm_block<T>(int, const T*, int, long long, T*, int, long long, int, int, int,         \
                              cudaStream_t);                                                            \
  template void hegst_diag<T>(T*, int, long long, const T*, int, long long, int, int, T*, int, long long, \
                              int, cudaStream_t);                                                       \
  template void larft<T>(const T*, int, long long, const double*, long long, int, T*, int, long long,    \
                         int, cudaStream_t);                                                            \
  template void apply_phase<T>(T*, int, long long, const double*, int, long long, const T*, long long,   \
                               int, int, int, cudaStream_t);                                            \
  template void mirror_lower<T>(T*, int, long long, int, int, cudaStream_t);                            \
  template void lowdin_factor<T>(const T*, int, long long, const double*, long long, T*, int, long long, int, \
                                 DevStatus*, int, cudaStream_t);                                           \
  template void column_phase<T>(T*, int, long long, int, int, int, cudaStream_t);                      \
  template void spinor_overlap<T>(T*, long long, const T*, int, long long, int, int, cudaStream_t);         \
  template void tune_pencil<T>(T*, int, int, int, cudaStream_t);
INST(double)
INST(zc)

}  // namespace gks
