// One-stage Householder reduction of a Hermitian matrix to real-phased tridiagonal form
// (the dense -> tridiagonal half of the standard eigensolve of H', paper Sec. 3.1 Part
// 2-4 / Sec. 3.2 Part 3-5).
//
// Storage: lower triangle, row-major.  The reduction runs upward: step j (j = m-1 .. 2)
// annihilates column j above its super-diagonal, i.e. row j left of its sub-diagonal,
// which is one contiguous row segment in this storage.  With a = A[0:j, j],
//   u = a + ph |a| e_{j-1},  ph = a_{j-1}/|a_{j-1}|,  P_j = I - tau u' u'^H,  u' = u/u_{j-1},
// and the leading j x j block becomes P_j A P_j = A - u q^H - q u^H with
//   p = tau A u,  q = p - (tau/2)(u^H p) u.
// u' (without its unit entry) is stored in row j left of the sub-diagonal.
//
// On GB300 the Hermitian matrix-vector product that dominates each step is bound by the
// FP64 pipe, not by HBM: a complex element read once feeds two complex multiply-adds
// (16 flops per 16 bytes), above the DFMA pipe's balance point of ~0.15 flop/byte.  It runs
// as exact 8-bit integer dot products on digits of the panel's stale block (the persistent
// panel kernel below; two launches per step in FP64 or single precision are the other form),
// and the rank-2 updates are deferred over panels of steps and applied as products, which
// the product dispatcher can send to the tensor cores.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "dense.h"

namespace gks {

// Reflector for step j (one CTA): reads row j left of the diagonal (through L2: in the
// fused form other CTAs have just written it), writes u', tau[j] and the sub-diagonal.
// uw (complex only, nullable): per element (Re u, Im u - Re u, Re u + Im u), the vector form
// of the three-multiplication complex products of the panel matrix-vector step.
__device__ __forceinline__ void put_uw(double* uw, int i, double ur, double ui) {
  if (uw) {
    uw[3 * i] = ur;
    uw[3 * i + 1] = ui - ur;
    uw[3 * i + 2] = ur + ui;
  }
}

// Scale exponent from the bits of a non-negative double (0 for zero): the e with the value
// below 2^e, i.e. ilogb + 1 (subnormals are counted at the smallest normal exponent).
__device__ __forceinline__ int bscale(unsigned long long bits) {
  return bits ? (int)((bits >> 52) & 0x7ff) - 1022 : 0;
}
// Equilibration exponent d_i = ceil(g_i / 2) of a row whose maximum (bits) lies below 2^{g_i}.
__device__ __forceinline__ int deq(unsigned long long bits) { return (bscale(bits) + 1) >> 1; }

// Digit format of the matrix-vector step: kDig balanced base-256 digits (signed 8-bit,
// in [-128, 127]) of the integer round(|x| 2^{54 - e}) with the sign of x, for |x| < 2^e:
// x = sum_s d_s 2^{e - 6 - 8s} up to 2^{e - 55}.
constexpr int kDig = 7;
constexpr int kMaxLevel = 7;  // digit pairs s + t <= kMaxLevel

// The digits of x below 2^e as the bytes of one word.  Integer operations on
// the bits of x only (the FP64 pipe is slow on this GPU): |x| = m 2^{x_e - 1075} with the
// 53-bit significand m, so trunc(|x| 2^{55 - e}) = m shifted by x_e - 1020 - e, and
// rounding halves it with a carry.  The balanced digits d_s, least significant d_{kDig-1} in
// byte 0, are the bytes of v + sum 128 256^i less 128 each (a flipped top bit); the leading
// one, in byte 6, stays within [-65, 65] and needs neither.
__device__ __forceinline__ unsigned long long digit_bytes(double x, int e) {
  constexpr unsigned long long bias = 0x0000808080808080ull;
  static_assert(kDig == 7, "six balanced bytes below the leading one");
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int xe = (int)((b >> 52) & 0x7ff);
  const unsigned long long m = (b & 0xfffffffffffffull) | (xe ? (1ull << 52) : 0ull);
  const int sh = (xe ? xe : 1) - 1020 - e;
  const unsigned long long q2 = sh >= 0 ? (m << sh) : (sh > -64 ? (m >> -sh) : 0ull);
  const unsigned long long q = (q2 + 1) >> 1;
  return (((b >> 63) ? 0ull - q : q) + bias) ^ bias;
}

// |Re|, |Im| maximum of a value as the bits of a non-negative double (bits of non-negative
// doubles order like the values).
__device__ __forceinline__ unsigned long long absbits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
template <typename T>
__device__ __forceinline__ unsigned long long maxbits(T a) {
  if constexpr (std::is_same<T, double>::value || std::is_same<T, float>::value) return absbits((double)a);
  else return max(absbits((double)re(a)), absbits((double)im(a)));
}

// Digits of 16 consecutive entries of a row, NPL planes of 16 bytes (the kDig Re planes, then
// the Im planes for complex) stored 32 rows apart (the tile's plane stride).  Entry el is cut
// below 2^{e[el]} (the scale and the equilibration folded into one exponent).
template <typename T, int NPL>
__device__ __forceinline__ void store_digit_block(const T (&vals)[16], const int (&e)[16], signed char* dst) {
  uint4 o[NPL];
  auto put = [&](int plane, int w, uint32_t v) {
    if (w == 0) o[plane].x = v;
    else if (w == 1) o[plane].y = v;
    else if (w == 2) o[plane].z = v;
    else o[plane].w = v;
  };
  // digits first .. first - 3 of four elements, whose bytes are 0 .. 3 of x0 .. x3: a 4 x 4
  // byte transpose, one word per plane
  auto put4 = [&](int base, int first, int w, uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3) {
    const uint32_t a = __byte_perm(x0, x1, 0x5140), b = __byte_perm(x2, x3, 0x5140);
    const uint32_t c = __byte_perm(x0, x1, 0x7362), d = __byte_perm(x2, x3, 0x7362);
    put(base + first, w, __byte_perm(a, b, 0x5410));
    put(base + first - 1, w, __byte_perm(a, b, 0x7632));
    put(base + first - 2, w, __byte_perm(c, d, 0x5410));
    if (first > 2) put(base + first - 3, w, __byte_perm(c, d, 0x7632));
  };
  auto put7 = [&](int base, int w, const unsigned long long (&d)[4]) {
    put4(base, 6, w, (uint32_t)d[0], (uint32_t)d[1], (uint32_t)d[2], (uint32_t)d[3]);
    put4(base, 2, w, (uint32_t)(d[0] >> 32), (uint32_t)(d[1] >> 32), (uint32_t)(d[2] >> 32), (uint32_t)(d[3] >> 32));
  };
#pragma unroll
  for (int w = 0; w < 4; w++) {
    unsigned long long d[4];
#pragma unroll
    for (int q = 0; q < 4; q++) d[q] = digit_bytes((double)re(vals[4 * w + q]), e[4 * w + q]);
    put7(0, w, d);
    if constexpr (NPL == 2 * kDig) {
#pragma unroll
      for (int q = 0; q < 4; q++) d[q] = digit_bytes((double)im(vals[4 * w + q]), e[4 * w + q]);
      put7(kDig, w, d);
    }
  }
  uint4* out = reinterpret_cast<uint4*>(dst);
#pragma unroll
  for (int q = 0; q < NPL; q++) out[32 * q] = o[q];
}

template <typename T>
__device__ void reflector_body(T* A, int lda, int j, T* u, double* tau, double* uw) {
  __shared__ double redd[32];
  const int tid = threadIdx.x, nt = blockDim.x;
  T* row = A + (size_t)j * lda;
  double s2 = 0.0;
  for (int i0 = tid; i0 < j; i0 += 8 * nt) {  // eight independent loads in flight per thread
    T v[8];
#pragma unroll
    for (int q = 0; q < 8; q++) v[q] = i0 + q * nt < j ? ldcg(row + i0 + q * nt) : zero<T>();
#pragma unroll
    for (int q = 0; q < 8; q++) s2 += abs2(v[q]);
  }
  const double xnorm2 = block_sum(s2, redd);
  const T alpha = conjg(ldcg(row + j - 1));
  const double tail = xnorm2 - abs2(alpha);
  if (!(tail > 0.0)) {  // nothing to annihilate: P_j = I
    for (int i = tid; i < j; i += nt) {
      u[i] = (i == j - 1) ? from_real<T>(1.0) : zero<T>();
      put_uw(uw, i, i == j - 1 ? 1.0 : 0.0, 0.0);
    }
    if (tid == 0) tau[j] = 0.0;
    return;
  }
  const double xn = sqrt(xnorm2);
  const double aa = sqrt(abs2(alpha));
  const T ph = aa > 0.0 ? alpha * (1.0 / aa) : from_real<T>(1.0);
  const T upiv = ph * (aa + xn);                       // alpha + ph * xn
  const double beta = 2.0 / (tail + abs2(upiv));
  const T inv = conjg(upiv) * (1.0 / abs2(upiv));       // 1 / upiv
  __syncthreads();
  for (int i0 = tid; i0 < j - 1; i0 += 8 * nt) {
    T v[8];
#pragma unroll
    for (int q = 0; q < 8; q++) v[q] = i0 + q * nt < j - 1 ? ldcg(row + i0 + q * nt) : zero<T>();
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int i = i0 + q * nt;
      if (i < j - 1) {
        const T w = conjg(v[q]) * inv;  // u'_i = a_i / u_{j-1}
        u[i] = w;
        row[i] = w;
        put_uw(uw, i, re(w), im(w));
      }
    }
  }
  if (tid == 0) {
    u[j - 1] = from_real<T>(1.0);
    put_uw(uw, j - 1, 1.0, 0.0);
    tau[j] = beta * abs2(upiv);
    row[j - 1] = conjg(ph) * (-xn);                     // lower-storage sub-diagonal
  }
}

template <typename T>
__global__ void hetrd_reflector_kernel(T* A, int lda, long long sA, int j, T* u, long long sv, double* tau,
                                       long long stau, double* uw) {
  const int z = blockIdx.x;
  reflector_body<T>(A + z * sA, lda, j, u + z * sv, tau + z * stau, uw ? uw + z * 3 * sv : nullptr);
}

// Sg[r][c] = Re A[r][c] + Im A[r][c] over the lower triangle of the leading n x n block
// (the stale block of a panel), for the three-multiplication products.
__global__ void hetrd_sums_kernel(const zc* A, int lda, long long sA, int n, double* Sg) {
  const int z = blockIdx.z;
  A += z * sA;
  Sg += z * sA;
  for (int r = blockIdx.y; r < n; r += gridDim.y)
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c <= r; c += gridDim.x * blockDim.x) {
      const zc a = A[(size_t)r * lda + c];
      Sg[(size_t)r * lda + c] = a.x + a.y;
    }
}

// The step's second part once this CTA's p_raw rows [c0, cend) are in prow (shared, one
// per row): p, the CTA's shares of Q^H u, U^H u and u^H p_raw, and in the last CTA (atomic
// ticket after a fence) their sums y1, y2, u^H p and kq.  Pointers are the item's.
template <typename T>
__device__ void phemv_tail(const T* prow, int c0, int cend, const T* u, T* p, double t, const T* U, const T* Q,
                           int ldu, int k, T* part, T* y, int* ticket) {
  __shared__ T red[32];
  __shared__ T gsum[256];
  __shared__ int last;
  const int tid = threadIdx.x;
  const int pst = 2 * ldu + 2;
  T d0 = zero<T>();
  if (tid < cend - c0) {
    const T pr = prow[tid];
    p[c0 + tid] = pr;
    macc(d0, u[c0 + tid], pr);
  }
  d0 = block_sum(d0, red);
  T* mine = part + (size_t)blockIdx.x * pst;
  if (tid == 0) mine[2 * ldu] = d0;
  for (int s = tid; s < k; s += blockDim.x) {
    T a1 = zero<T>(), a2 = zero<T>();
    for (int r0 = c0; r0 < cend; r0 += 8) {  // eight rows' loads in flight
      T qv[8], uv[8], ur[8];
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int r = min(r0 + q, cend - 1);
        qv[q] = Q[(size_t)r * ldu + s];
        uv[q] = U[(size_t)r * ldu + s];
        ur[q] = r0 + q < cend ? u[r] : zero<T>();
      }
#pragma unroll
      for (int q = 0; q < 8; q++) {
        macc(a1, qv[q], ur[q]);
        macc(a2, uv[q], ur[q]);
      }
    }
    mine[s] = a1;
    mine[ldu + s] = a2;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last = (atomicAdd(ticket, 1) == (int)gridDim.x - 1);
  __syncthreads();
  if (!last) return;
  if (tid == 0) *ticket = 0;
  // Sums over the CTAs' shares of the E = 2k + 1 entries (Q^H u, U^H u, u^H p_raw): G groups
  // of threads per entry take every G-th CTA with eight loads in flight, then one thread per
  // entry adds the groups in order.
  const int nb = gridDim.x, nt = blockDim.x, E = 2 * k + 1;
  const int G = E <= nt ? nt / E : 1;
  for (int t0 = tid; t0 < G * E; t0 += nt) {
    const int e = t0 % E, g = t0 / E;
    const size_t off = e < k ? e : (e < 2 * k ? ldu + (e - k) : 2 * ldu);
    T a = zero<T>();
    for (int b0 = g; b0 < nb; b0 += 8 * G) {
      T v[8];
#pragma unroll
      for (int q = 0; q < 8; q++) v[q] = b0 + q * G < nb ? ldcg(part + (size_t)(b0 + q * G) * pst + off) : zero<T>();
#pragma unroll
      for (int q = 0; q < 8; q++) a += v[q];
    }
    if (G > 1) gsum[t0] = a;
    else if (e < k) y[e] = a;
    else if (e < 2 * k) y[ldu + e - k] = a;
    else red[0] = a;
  }
  __syncthreads();
  if (G > 1 && tid < E) {
    T a = gsum[tid];
    for (int g = 1; g < G; g++) a += gsum[g * E + tid];
    if (tid < k) y[tid] = a;
    else if (tid < 2 * k) y[ldu + tid - k] = a;
    else red[0] = a;
  }
  __syncthreads();
  const T tot = red[0];
  __syncthreads();
  T w = zero<T>();
  for (int e = tid; e < k; e += blockDim.x) {
    macc(w, y[ldu + e], y[e]);
    macc(w, y[e], y[ldu + e]);
  }
  w = block_sum(w, red);
  if (tid == 0) {
    const T uhp = t * (tot - w);
    y[2 * ldu] = tot;
    y[2 * ldu + 1] = (0.5 * t) * uhp;
  }
}

// Panel (blocked) form.  A panel of steps keeps the trailing block A[0:j,0:j] as it was
// at the panel's start; the panel buffers U and Q (M x ldu per item, row r holds u_s[r]
// and q_s[r] for the panel's earlier steps s < k) carry what it has not seen yet:
//   A_true = A - U Q^H - Q U^H   on [0:j, 0:j].
// The panel ends with that rank-2k update as two GEMMs.
//
// Step j, first half: p_raw = A[0:j,0:j] u over the stale block.  CTA b owns rows/columns
// [RB b, RB b + RB): its row panel left of the diagonal plus its column panel below, so every
// CTA reads the same number of elements.  It adds its rows' shares of Q^H u, U^H u and
// u^H p_raw.  The last CTA (atomic ticket after a fence; nothing waits) sums the shares:
//   y1 = Q^H u,  y2 = U^H u,  u^H p = tau (u^H p_raw - y2^H y1 - y1^H y2),
//   kq = (tau/2) u^H p,
// since p = tau A_true u = tau (p_raw - U y1 - Q y2).
// y layout per item: y1 at [0, k), y2 at [ldu, ldu + k), u^H p_raw at 2 ldu, kq at 2 ldu + 1;
// the shares use the same layout per CTA with stride 2 ldu + 2.
template <typename T, int RB>
__global__ void __launch_bounds__(256) hetrd_phemv_kernel(const T* A, int lda, long long sA, int j, const T* u,
                                                          T* p, long long sv, const double* tau, long long stau,
                                                          const T* U, const T* Q, int ldu, long long sU, int k,
                                                          T* part, long long spart, T* y, long long sy,
                                                          int* ticket, const double* Sg, const double* uw) {
  // RB rows/columns per CTA (64, or 16 when the grid would not fill the GPU)
  constexpr int NG = 256 / RB;
  __shared__ T colpart[NG][RB];
  __shared__ T rowacc[RB];
  const int z = blockIdx.y, tid = threadIdx.x;
  A += z * sA;
  u += z * sv;
  p += z * sv;
  U += z * sU;
  Q += z * sU;
  part += z * spart;
  y += z * sy;
  const double t = tau[z * stau + j];
  const int c0 = blockIdx.x * RB;
  const int cend = min(c0 + RB, j);
  const int warp = tid >> 5, lane = tid & 31;
  bool done = false;
  if constexpr (sizeof(T) == 16) {
    if (Sg) {
      // Three real multiply-adds per complex product (Gauss): with s = Re a + Im a (Sg) and
      // the vector form (c, d - c, c + d) of u_c = c + i d (uw),
      //   a u    = (c s - Im a (c + d)) + i (c s + Re a (d - c)),
      //   a* u   = (c s + Im a (d - c)) + i (Re a (c + d) - c s).
      Sg += z * sA;
      uw += z * 3 * sv;
      for (int r = c0 + warp; r < cend; r += 8) {
        const zc* ar = reinterpret_cast<const zc*>(A) + (size_t)r * lda;
        const double* sr = Sg + (size_t)r * lda;
        double k1 = 0.0, k2 = 0.0, k3 = 0.0;
        for (int c = lane; c <= r; c += 32) {
          const zc a = ar[c];
          k1 = fma(uw[3 * c], sr[c], k1);
          k2 = fma(a.x, uw[3 * c + 1], k2);
          k3 = fma(a.y, uw[3 * c + 2], k3);
        }
        k1 = warp_sum(k1);
        k2 = warp_sum(k2);
        k3 = warp_sum(k3);
        if (lane == 0) rowacc[r - c0] = T{k1 - k3, k1 + k2};
      }
      const int cc = tid % RB, g = tid / RB;
      const int c = c0 + cc;
      double l1 = 0.0, l3 = 0.0, l4 = 0.0;
      if (c < cend) {
        for (int r = c0 + g; r < j; r += NG)
          if (r > c) {
            const zc a = reinterpret_cast<const zc*>(A)[(size_t)r * lda + c];
            l1 = fma(uw[3 * r], Sg[(size_t)r * lda + c], l1);
            l3 = fma(a.y, uw[3 * r + 1], l3);
            l4 = fma(a.x, uw[3 * r + 2], l4);
          }
      }
      colpart[g][cc] = T{l1 + l3, l4 - l1};
      done = true;
    }
  }
  if (!done) {
    // row part: rows r in [c0, cend), columns 0..r; one warp per row
    for (int r = c0 + warp; r < cend; r += 8) {
      const T* ar = A + (size_t)r * lda;
      T s = zero<T>();
      for (int c = lane; c <= r; c += 32) mac(s, ar[c], u[c]);
      s = warp_sum(s);
      if (lane == 0) rowacc[r - c0] = s;
    }
    // column part: columns c in [c0, cend), rows r > c
    const int cc = tid % RB, g = tid / RB;
    const int c = c0 + cc;
    T s = zero<T>();
    if (c < cend) {
      for (int r = c0 + g; r < j; r += NG)
        if (r > c) macc(s, A[(size_t)r * lda + c], u[r]);
    }
    colpart[g][cc] = s;
  }
  __syncthreads();
  if (tid < RB && c0 + tid < cend) {
    T pr = rowacc[tid];
#pragma unroll
    for (int g = 0; g < NG; g++) pr += colpart[g][tid];
    rowacc[tid] = pr;
  }
  phemv_tail<T>(rowacc, c0, cend, u, p, t, U, Q, ldu, k, part, y, ticket + z);
}

// ------------------------------------------------------------------ digit form of the step
//
// hetrd_dmax_kernel: row maxima of |Re|, |Im| over the full Hermitian rows of the stale
// block from its lower triangle, where element (r, c) counts for rows r and c.  One CTA per
// 64 x 64 tile of the lower triangle (each element read once, 8 warps of 8 rows, a lane per
// column pair): row maxima by warp reduction, column maxima over the warps, one atomic max
// per row, column and tile (on the bits of non-negative doubles, which order like the
// values).  One CTA per 64 rows walking their columns twice took 777 us at order 4992.
__device__ __forceinline__ unsigned long long umax(unsigned long long a, unsigned long long b) { return a > b ? a : b; }
template <typename T>
__global__ void __launch_bounds__(256) hetrd_dmax_kernel(const T* A, int lda, long long sA, int n,
                                                         unsigned long long* rmax, int ldr) {
  if (blockIdx.x > blockIdx.y) return;
  __shared__ unsigned long long cm[8][64];
  const int z = blockIdx.z, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 64;
  A += z * sA;
  rmax += (size_t)z * ldr;
  unsigned long long m0 = 0ull, m1 = 0ull, b[8][2];
#pragma unroll
  for (int q = 0; q < 8; q++) {
    const int r = r0 + warp * 8 + q, c = c0 + lane;
    b[q][0] = (r < n && c <= r) ? maxbits(A[(size_t)r * lda + c]) : 0ull;
    b[q][1] = (r < n && c + 32 <= r) ? maxbits(A[(size_t)r * lda + c + 32]) : 0ull;
  }
#pragma unroll
  for (int q = 0; q < 8; q++) {
    const int r = r0 + warp * 8 + q;
    m0 = umax(m0, b[q][0]);
    m1 = umax(m1, b[q][1]);
    unsigned long long m = umax(b[q][0], b[q][1]);
    for (int o = 16; o > 0; o >>= 1) m = umax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0 && m) atomicMax(rmax + r, m);
  }
  cm[warp][lane] = m0;
  cm[warp][lane + 32] = m1;
  __syncthreads();
  if (tid < 64) {
    unsigned long long m = 0ull;
#pragma unroll
    for (int w = 0; w < 8; w++) m = umax(m, cm[w][tid]);
    if (m) atomicMax(rmax + c0 + tid, m);
  }
}

// hetrd_digits_kernel: 32 x 32 tiles of the full Hermitian [0:n16, 0:n16] (zero outside
// [0:n, 0:n]); tiles above the diagonal come from the transposed lower tile through shared
// memory, conjugated.  64 threads: thread t packs row t / 2, columns 16 (t % 2) .. + 15.
// Bound by integer operations and HBM once the tile's loads are in flight together (order 4992
// complex: 349 us with one load at a time, 246 us with eight, 144 us with the digits as the bytes of one
// biased word and byte transposes).
template <typename T>
__global__ void __launch_bounds__(64) hetrd_digits_kernel(const T* A, int lda, long long sA, int n, HemvDigits hd) {
  constexpr int NPL = sizeof(T) == 16 ? 2 * kDig : kDig;
  __shared__ T tile[32][33];
  const int z = blockIdx.z, tid = threadIdx.x;
  const int R0 = blockIdx.y * 32, C0 = blockIdx.x * 32;
  const int n16 = (n + 15) & ~15;
  if (R0 >= n16 || C0 >= n16) return;
  A += z * sA;
  const bool upper = C0 > R0;
  // source tile: (R0, C0) itself, or (C0, R0) for tiles above the diagonal
  const int sr0 = upper ? C0 : R0, sc0 = upper ? R0 : C0;
#pragma unroll 8
  for (int e = tid; e < 32 * 32; e += 64) {  // eight loads in flight
    const int yy = e >> 5, xx = e & 31;
    const int r = sr0 + yy, c = sc0 + xx;
    tile[yy][xx] = (r < n && c < n && c <= r) ? A[(size_t)r * lda + c] : zero<T>();
  }
  __syncthreads();
  const unsigned long long* rm = hd.rmax + (size_t)z * hd.ldd;
  const int rr = tid >> 1, cbk = tid & 1;
  const int r = R0 + rr;
  if (r < n16 && C0 + 16 * cbk < n16) {
    const int dr = r < n ? deq(rm[r]) : 0;
    T vals[16];
    int ex[16];
#pragma unroll
    for (int el = 0; el < 16; el++) {
      const int cc = 16 * cbk + el, c = C0 + cc;
      T v;
      if (upper) v = conjg(tile[cc][rr]);
      else if (c <= r) v = tile[rr][cc];
      else v = (r < n && c < n) ? conjg(tile[cc][rr]) : zero<T>();  // diagonal tile, upper part
      vals[el] = v;
      ex[el] = dr + (c < n ? deq(rm[c]) : 0);  // ã = a 2^{-d_r - d_c}, cut below 1
    }
    const size_t tile = (size_t)(r >> 5) * (hd.ldd >> 4) + (C0 >> 4) + cbk;
    store_digit_block<T, NPL>(vals, ex, hd.D + z * hd.sD + tile * (32 * NPL * 16) + (size_t)(r & 31) * 16);
  }
}

__device__ __forceinline__ int dp4(unsigned a, unsigned b, int c) { return __dp4a((int)a, (int)b, c); }
__device__ __forceinline__ int dp4x4(uint4 a, uint4 b, int c) {
  return dp4(a.w, b.w, dp4(a.z, b.z, dp4(a.y, b.y, dp4(a.x, b.x, c))));
}

// 16-byte asynchronous global -> shared copies (L2 only), their groups and waits.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Sum over aligned groups of 8 lanes (every lane of the warp takes part).
__device__ __forceinline__ double group8_sum(double v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ zc group8_sum(zc v) { return zc{group8_sum(v.x), group8_sum(v.y)}; }
__device__ __forceinline__ float group8_sum(float v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ cf group8_sum(cf v) { return cf{group8_sum(v.x), group8_sum(v.y)}; }
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ zc shfl_xor(zc v, int o) { return zc{shfl_xor(v.x, o), shfl_xor(v.y, o)}; }

// Step j, second half: q = tau (p_raw - U y1 - Q y2) - kq u for the rows of this CTA (64
// per CTA), stored with u as column k of Q and U.  With rowupd, row j-1 of A (columns
// 0..j-1) receives the panel's updates so far,
//   A[j-1][c] -= sum_{s<=k} U[j-1][s] conj(Q[c][s]) + Q[j-1][s] conj(U[c][s]),
// (each CTA computes the single q_k[j-1] it needs itself), and the last CTA forms the
// reflector of step j-1 from that row.  Dynamic shared memory: 4 (ldu + 1) elements.
template <typename T>
__global__ void __launch_bounds__(256) hetrd_pupdate_kernel(T* A, int lda, long long sA, int j, T* u,
                                                            const T* p, long long sv, double* tau, long long stau,
                                                            T* U, T* Q, int ldu, long long sU, int k, const T* y,
                                                            long long sy, int rowupd, int* ticket, double* uw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* y1s = reinterpret_cast<T*>(smem_raw);
  T* y2s = y1s + (ldu + 1);
  T* ujs = y2s + (ldu + 1);
  T* qjs = ujs + (ldu + 1);
  __shared__ int last;
  const int z = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  A += z * sA;
  u += z * sv;
  p += z * sv;
  U += z * sU;
  Q += z * sU;
  y += z * sy;
  tau += z * stau;
  if (uw) uw += z * 3 * sv;
  const double t = tau[j];
  const T kq = y[2 * ldu + 1];
  for (int s = tid; s < k; s += blockDim.x) {
    y1s[s] = y[s];
    y2s[s] = y[ldu + s];
    if (rowupd) {
      ujs[s] = U[(size_t)(j - 1) * ldu + s];
      qjs[s] = Q[(size_t)(j - 1) * ldu + s];
    }
  }
  __syncthreads();
  if (rowupd && warp == 0) {
    T corr = zero<T>();
    for (int s = lane; s < k; s += 32) {
      mac(corr, ujs[s], y1s[s]);
      mac(corr, qjs[s], y2s[s]);
    }
    corr = warp_sum(corr);
    if (lane == 0) {
      const T uj = u[j - 1];
      ujs[k] = uj;
      qjs[k] = t * (p[j - 1] - corr) - kq * uj;
    }
  }
  __syncthreads();
  // 32 groups of 8 lanes, two columns per group (more columns in flight, short reductions)
  const int c0 = blockIdx.x * 64, cend = min(c0 + 64, j);
  const int grp = tid >> 3, gl = tid & 7;
  for (int it = 0; it < 2; it++) {
    const int c = c0 + grp + 32 * it;
    const bool ok = c < cend;
    T corr = zero<T>(), rs = zero<T>();
    if (ok) {
      const T* Uc = U + (size_t)c * ldu;
      const T* Qc = Q + (size_t)c * ldu;
      for (int s0 = gl; s0 < k; s0 += 32) {  // four steps' loads in flight
        T ucv[4], qcv[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const int sq = min(s0 + 8 * q, k - 1);
          ucv[q] = Uc[sq];
          qcv[q] = Qc[sq];
        }
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const int sq = s0 + 8 * q;
          if (sq < k) {
            mac(corr, ucv[q], y1s[sq]);
            mac(corr, qcv[q], y2s[sq]);
            if (rowupd) {
              mac(rs, ujs[sq], conjg(qcv[q]));
              mac(rs, qjs[sq], conjg(ucv[q]));
            }
          }
        }
      }
    }
    corr = group8_sum(corr);
    if (rowupd) rs = group8_sum(rs);
    if (ok && gl == 0) {
      const T uc = u[c];
      const T qc = t * (p[c] - corr) - kq * uc;
      U[(size_t)c * ldu + k] = uc;
      Q[(size_t)c * ldu + k] = qc;
      if (rowupd) {
        mac(rs, ujs[k], conjg(qc));
        mac(rs, qjs[k], conjg(uc));
        T* a = A + (size_t)(j - 1) * lda + c;
        *a = *a - rs;
      }
    }
  }
  if (!rowupd) return;
  __threadfence();
  __syncthreads();
  if (tid == 0) last = (atomicAdd(ticket + z, 1) == (int)gridDim.x - 1);
  __syncthreads();
  if (!last) return;
  if (tid == 0) ticket[z] = 0;
  __syncthreads();
  reflector_body<T>(A, lda, j - 1, u, tau, uw);
}

// ------------------------------------------------------------------ persistent panel (digit form)
//
// All steps of a panel in one cooperative launch, G CTAs per item.  A step is a chain of
// short dependent parts (norm and reflector, matrix-vector product, the panel's corrections,
// the next row); as two launches per step with the reductions in a last CTA it took 32 us at
// order 832 and 127 us at 4992 (one item), against 6 and 25 us of digit traffic and
// arithmetic.  Here two barriers over all CTAs of the item separate the parts, the vector warps
// have one or two more of their own, and every part is spread over all CTAs:
//   1. every CTA forms the reflector's scalars from the CTAs' shares of the norm.  Warps 0-7
//      multiply the CTA's share of the digit tiles (the R x C tiles of the block in row-tile
//      order, cut into G equal runs, so every CTA streams the same bytes at any order) with
//      v = conj(a) (the pivot replaced by upiv; u' = v / upiv is applied to the sums), whose
//      digits each warp makes for the 16 columns it is about to use.  Warps 8-11 meanwhile
//      store u' for the CTA's rows, form the rows' shares of y1 = Q^H u and y2 = U^H u and,
//      after a barrier of their own, add the shares of a few entries each over the CTAs.
//      Where the product is long enough to hide it (a.early) they also wait for y and form
//      U y1 + Q y2 and row j-1 with the panel's earlier updates, which takes the panel's FP64
//      work off the chain (order 4992: 44 -> 40 us per step; order 832: 13 -> 16 us, the
//      product being shorter than that work).
//   2. barrier; p from the runs that touch each row, those corrections unless done, q, row j-1
//      with this step's update, and the shares of its norm; barrier.
// The digit tiles of the next step do not depend on this one: their first copies are issued
// before the barriers.  Partial sums are added in a fixed order: results do not depend on
// timing.  Every wait is bounded (a.wait SM cycles): past it the status is set, an abort flag
// lets every CTA leave.  Bound by HBM and dp4a together at large orders (14 bytes and 34 dp4a
// per complex entry), by the barriers (about 1 us each) and FP64 latencies at small ones.
// Measured per step (one item, averaged over a reduction): order 832 real 13.0 us, 2808 real
// 15.8, 2496 complex 22.1, 4992 complex 40.9 (the digit product: 2.3, 4.8, 8.2, 25.0).
template <typename T>
struct PanelSmem {
  static constexpr bool CPX = sizeof(T) == 16;
  static constexpr int NP = CPX ? 4 : 1, NL = kMaxLevel + 1, NPL = CPX ? 2 * kDig : kDig;
  static constexpr int STG = 3, TILE4 = 32 * NPL;  // ring stages per warp, 16-byte words per tile
  static constexpr int RING = 8 * STG * TILE4 * 16;
  static constexpr int ACC = NP * NL * 8 * 32 * 4;   // [product, level][warp][row]
  static constexpr int LVL = NL * 32 * (int)sizeof(T);  // [level][row] 64-bit sums, Re then Im
  static constexpr int UB = 8 * 2 * NPL * 16;
  static constexpr int VEC = 4 * (kPanelMax + 1) * (int)sizeof(T);
  static constexpr int TOTAL = RING + ACC + LVL + UB + VEC;
  static_assert(TOTAL <= 226 * 1024, "shared memory of the panel kernel");
};
constexpr int kPanelThreads = 384;

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release(unsigned* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(p) : "memory");
}
template <int ID, int N>
__device__ __forceinline__ void bar_named() {
  asm volatile("bar.sync %0, %1;\n" ::"n"(ID), "n"(N) : "memory");
}
// One thread per CTA (which has arrived on *cnt): wait for target arrivals; false on abort or
// timeout.
__device__ __forceinline__ bool grid_wait(unsigned* cnt, unsigned target, unsigned* abortf, long long limit) {
  const long long t0 = clock64();
  for (unsigned n = 1; (int)(ld_acquire(cnt) - target) < 0; n++) {
    if (n & 63u) continue;
    if (*(volatile unsigned*)abortf) return false;
    if (clock64() - t0 > limit) {
      atomicExch(abortf, 1u);
      return false;
    }
  }
  return true;
}

// The same over the CTAs of a cluster: an mbarrier of G arrivals in every CTA.  Lanes below G
// arrive on the barrier of CTA `lane`; a thread waits for its own CTA's phase.  Consecutive
// phases alternate between two mbarriers: an arrival names no sender and arrivals at different
// CTAs are not ordered, so that on one mbarrier a CTA that has seen phase n could arrive for n + 1
// at a CTA where another's arrival for n is still on its way, and complete n there in its place.
// With two, an arrival for n + 2 on the mbarrier of n follows everyone's for n + 1, which
// follow their completions of n.
__device__ __forceinline__ void cluster_arrive(uint64_t* bar, int cta) {
  asm volatile(
      "{\n .reg .b32 ra;\n mapa.shared::cluster.u32 ra, %0, %1;\n"
      " mbarrier.arrive.release.cluster.shared::cluster.b64 _, [ra];\n}\n" ::"r"(
          (unsigned)__cvta_generic_to_shared(bar)),
      "r"(cta)
      : "memory");
}
__device__ __forceinline__ bool cluster_wait(uint64_t* bar, unsigned parity, long long limit) {
  const long long t0 = clock64();
  unsigned ok = 0;
  while (true) {
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"((unsigned)__cvta_generic_to_shared(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > limit) return false;
  }
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Runs of digit tiles: T = R C tiles of order j (T G < 2^31 at every supported order), CTA b
// of G has [run0(b), run0(b + 1)).
struct PanelRuns {
  unsigned C, R, T, G;
  __device__ PanelRuns(int j, int G_) : C((j + 15) >> 4), R((j + 31) >> 5), T(R * C), G(G_) {}
  __device__ int run0(int b) const { return (int)((unsigned)b * T / G); }
  __device__ int owner(int t) const { return (int)((((unsigned)t + 1u) * G - 1u) / T); }  // run holding tile t
};

template <typename T, bool CL>
__global__ void __launch_bounds__(kPanelThreads, 1) hetrd_panel_kernel(const PanelArgs<T> a, int maxseg) {
  using SM = PanelSmem<T>;
  constexpr bool CPX = SM::CPX;
  constexpr int NP = SM::NP, NL = SM::NL, NPL = SM::NPL, STG = SM::STG, TILE4 = SM::TILE4;
  extern __shared__ __align__(128) unsigned char psm[];
  uint4* ring_all = reinterpret_cast<uint4*>(psm);
  auto accs = reinterpret_cast<int(*)[8][32]>(psm + SM::RING);
  long long* lvl = reinterpret_cast<long long*>(psm + SM::RING + SM::ACC);
  unsigned char* ubuf = psm + SM::RING + SM::ACC + SM::LVL;
  T* y1s = reinterpret_cast<T*>(psm + SM::RING + SM::ACC + SM::LVL + SM::UB);
  T* y2s = y1s + (kPanelMax + 1);
  T* ujs = y2s + (kPanelMax + 1);
  T* qjs = ujs + (kPanelMax + 1);
  __shared__ T s_inv, s_upiv, s_sub, s_pj, s_us[64];
  __shared__ double s_tau, s_kq, s_red[12];
  __shared__ __align__(8) uint64_t s_bar[4];  // cluster form: two for all threads, two for the vector warps
  __shared__ int s_fu, s_ok, s_abort, s_rede[12];

  const int z = blockIdx.y, b = blockIdx.x, G = gridDim.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int lda = a.lda, ldu = a.ldu;
  T* A = a.A + z * a.sA;
  T* U = a.U + z * a.sU;
  T* Q = a.Q + z * a.sU;
  T* arow2 = a.arow + z * 2 * a.sv;
  T* part = a.part + (long long)z * a.gs * (2 * kPanelMax);
  T* y = a.y + (long long)z * (2 * kPanelMax);
  T* P = a.P + z * a.sP;
  double* dot = a.dot + (long long)z * a.gs;
  double* nrm = a.nrm + (long long)z * a.gs;
  int* mex = a.mex + (long long)z * a.gs;
  double* tau = a.tau + z * a.stau;
  unsigned* bar = a.bar + 4 * z;
  const unsigned long long* rmax = a.hd.rmax + (size_t)z * a.hd.ldd;
  const uint4* D = reinterpret_cast<const uint4*>(a.hd.D + z * a.hd.sD);
  const int ldc = a.hd.ldd >> 4;  // tiles per row tile
  const int cs = (a.jh + G - 1) / G, c0 = b * cs, c1 = min(c0 + cs, a.jh);  // this CTA's rows
  // targets of the two counters (cluster form: phases passed)
  unsigned arrived = CL ? 0u : a.base, arrivedv = CL ? 0u : a.basev;
  constexpr int NOEXP = -100000;

  // shares of the next reflector's norm (over the entries before the pivot) and scale
  auto put_norm = [&](double n2, int e, bool groups) {
    if (groups) {  // one value per 8 lanes
      n2 += __shfl_xor_sync(0xffffffffu, n2, 8);
      n2 += __shfl_xor_sync(0xffffffffu, n2, 16);
    } else {
      n2 = warp_sum(n2);
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) {
      s_red[warp] = n2;
      s_rede[warp] = e;
    }
    __syncthreads();
    if (warp == 0) {
      double t = lane < 12 ? s_red[lane] : 0.0;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      const int m = __reduce_max_sync(0xffffffffu, lane < 12 ? s_rede[lane] : NOEXP);
      if (lane == 0) {
        nrm[b] = t;
        mex[b] = m;
      }
    }
  };
  auto scale_of = [&](T v, int d) -> int {  // d: the entry's equilibration exponent
    const unsigned long long mb = maxbits(v);
    return mb ? bscale(mb) + d : NOEXP;
  };
  // full barrier over the item's CTAs; false once any wait expired (uniform over the CTA)
  auto barrier = [&]() -> bool {
    __syncthreads();
    arrived += CL ? 1u : (unsigned)G;
    if (CL) {
      if (warp == 0) {
        uint64_t* sb = &s_bar[(arrived - 1) & 1u];
        if (lane < G) cluster_arrive(sb, lane);
        if (lane == 0 && !cluster_wait(sb, ((arrived - 1) >> 1) & 1u, a.wait)) s_abort = 1;
      }
    } else if (tid == 0) {
      red_release(bar);
      if (!grid_wait(bar, arrived, bar + 2, a.wait)) s_abort = 1;
    }
    __syncthreads();
    return s_abort == 0;
  };
  uint4* ring = ring_all + warp * (STG * TILE4);
  // stage i % STG <- the warp's i-th tile of the run of step j
  auto issue = [&](int C, int t, int t1, int i) {  // t: the tile, of the run that ends at t1
    if (t < t1) {
      const int r = t / C, cb = t - r * C;
      const uint4* src = D + ((size_t)r * ldc + cb) * TILE4 + lane;
      uint4* st = ring + (i % STG) * TILE4 + lane;
#pragma unroll
      for (int q = 0; q < NPL; q++) cp_async16(st + 32 * q, src + 32 * q);
    }
    cp_async_commit();
  };

  // y and row j-1 of U and Q (their earlier steps) into shared memory, threads t of nt
  int j = a.jh, k = 0;
  auto load_panel_vectors = [&](int t, int nt) {
    for (int s = t; s < k; s += nt) {
      y1s[s] = ldcg(y + s);
      y2s[s] = ldcg(y + k + s);
      ujs[s] = ldcg(U + (size_t)(j - 1) * ldu + s);
      qjs[s] = ldcg(Q + (size_t)(j - 1) * ldu + s);
    }
  };
  // one earlier step's share of U y1 + Q y2 and of row j-1's updates
  auto correct = [&](T& corr, T& rs, T u, T q, int s) {
    mac(corr, u, y1s[s]);
    mac(corr, q, y2s[s]);
    mac(rs, ujs[s], conjg(q));
    mac(rs, qjs[s], conjg(u));
  };

  if (tid == 0) s_abort = 0;
  if (CL) {
    if (tid == 0) {
      for (int q = 0; q < 4; q++)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"((unsigned)__cvta_generic_to_shared(&s_bar[q])),
                     "r"(q < 2 ? G : G + a.late));
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    cluster_sync_all();
  }
  {
    T* ar = arow2 + (j & 1) * a.sv;
    double n2 = 0.0;
    int e = NOEXP;
    for (int c = c0 + tid; c < c1; c += kPanelThreads) {
      const T v = A[(size_t)j * lda + c];
      ar[c] = v;
      if (c < j - 1) {
        n2 += abs2(v);
        e = max(e, scale_of(v, deq(rmax[c])));
      }
    }
    __syncthreads();
    put_norm(n2, e, false);
    if (warp < 8) {
      const PanelRuns pr(j, G);
      const int t0 = pr.run0(b), t1 = pr.run0(b + 1);
#pragma unroll
      for (int i = 0; i < STG - 1; i++) issue(pr.C, t0 + warp + 8 * i, t1, i);
    }
  }
  bool live = barrier();

  for (; j >= a.jl && live; j--) {
    k = a.jh - j;
    const T* ar = arow2 + (j & 1) * a.sv;
    // the entry of a whose digits this lane makes for the warp's next tile: column lane & 15, Re
    // (lanes 0-15) or Im (lanes 16-31), loaded a tile ahead (the first one before the scalars)
    const PanelRuns pr(j, G);
    const int t0 = pr.run0(b), t1 = pr.run0(b + 1);
    T araw = zero<T>();
    unsigned long long rraw = 0ull;
    auto vfetch = [&](int t) {
      const int c = 16 * (t % (int)pr.C) + (lane & 15);
      if (t < t1 && c < j) {
        araw = ldcg(ar + c);
        rraw = rmax[c];
      }
    };
    const int vt = tid - 256, ce = min(c1, j);
    T apre = zero<T>();  // the vector warps' rows of a
    if (warp < 8) vfetch(t0 + warp);
    else if (vt < 64 && c0 + vt < ce) apre = ldcg(ar + c0 + vt);
    if (warp == 0) {
      double tail = 0.0;
      int e = NOEXP;
      const T alpha = conjg(ldcg(ar + j - 1));
      const int dpiv = deq(rmax[j - 1]);
      for (int g = lane; g < G; g += 32) {
        tail += __ldcg(nrm + g);
        e = max(e, __ldcg(mex + g));
      }
      tail = warp_sum(tail);
      e = __reduce_max_sync(0xffffffffu, e);
      // |a| and |alpha| in two lanes, then the three reciprocals in three lanes: one square
      // root and one division deep.  u = alpha + ph |a| at the pivot, tau = 1 + |alpha| / |a|.
      const double a2 = abs2(alpha), sq = sqrt(lane & 1 ? a2 : tail + a2);
      const double xn = __shfl_sync(0xffffffffu, sq, 0), aa = __shfl_sync(0xffffffffu, sq, 1);
      const double rc = recip(lane == 0 ? aa : lane == 1 ? aa + xn : xn);
      const double raa = __shfl_sync(0xffffffffu, rc, 0), rsum = __shfl_sync(0xffffffffu, rc, 1);
      const double rxn = __shfl_sync(0xffffffffu, rc, 2);
      if (lane == 0) {
        if (!(tail > 0.0)) {  // nothing to annihilate: P_j = I
          s_ok = 0;
          s_inv = s_upiv = from_real<T>(1.0);
          s_sub = conjg(alpha);
          s_tau = 0.0;
          e = scale_of(from_real<T>(1.0), dpiv);
        } else {
          const T ph = aa > 0.0 ? alpha * raa : from_real<T>(1.0);
          const T upiv = ph * (aa + xn);
          s_ok = 1;
          s_upiv = upiv;
          s_inv = conjg(ph) * rsum;
          s_sub = conjg(ph) * (-xn);  // lower-storage sub-diagonal
          s_tau = (aa + xn) * rxn;
          e = max(e, scale_of(upiv, dpiv));
        }
        s_fu = e;
        if (b == 0) tau[j] = s_tau;
      }
    }
    __syncthreads();
    const T inv = s_inv;
    const bool refl = s_ok != 0;

    if (warp < 8) {
      // ---- matrix-vector product over the CTA's run of tiles
      const int fu = s_fu;
      int acc[NP][NL];
#pragma unroll
      for (int q = 0; q < NP; q++)
#pragma unroll
        for (int L = 0; L < NL; L++) acc[q][L] = 0;
      double d0 = 0.0;  // u^H p_raw (real: the block is Hermitian)
      int i = 0;
      const int C = pr.C;
      for (int seg = 0, r = t0 / C; t0 < t1 && r * C < t1; r++, seg++) {
        const int te = min(t1, (r + 1) * C), row = 32 * r + lane;
        T arow = zero<T>();
        int drow = 0;
        if (warp == 0 && row < j) {
          arow = ldcg(ar + row);
          drow = deq(rmax[row]);
        }
        for (int t = t0 + warp + 8 * i; t < te; t += 8, i++) {
          double xv = 0.0;
          int xe = 0;
          {
            const int c = 16 * (t - r * C) + (lane & 15);
            if (c < j) {
              const T v = c == j - 1 ? s_upiv : (refl ? conjg(araw) : zero<T>());
              xv = lane < 16 ? re(v) : im(v);
              xe = fu - deq(rraw);
            }
          }
          vfetch(t + 8);
          const unsigned long long d = digit_bytes(xv, xe);
          unsigned char* ub = ubuf + (warp * 2 + (i & 1)) * (NPL * 16);
          if (CPX || lane < 16) {
#pragma unroll
            for (int q = 0; q < kDig; q++)
              ub[((lane >> 4) * kDig + q) * 16 + (lane & 15)] = (unsigned char)(d >> (8 * (kDig - 1 - q)));
          }
          __syncwarp();  // the digits are written, and every lane is done with the stage refilled next
          issue(C, t + 8 * (STG - 1), t1, i + STG - 1);
          cp_async_wait<STG - 1>();
          __syncwarp();
          const uint4* st = ring + (i % STG) * TILE4 + lane;
          const uint4* uq = reinterpret_cast<const uint4*>(ub);
          uint4 av[NPL];
#pragma unroll
          for (int q = 0; q < NPL; q++) av[q] = st[32 * q];
#pragma unroll
          for (int w = 0; w < kDig; w++) {
            const uint4 ur = uq[w];
            uint4 ui;
            if constexpr (CPX) ui = uq[kDig + w];
#pragma unroll
            for (int q = 0; q < kDig && q + w <= kMaxLevel; q++) {
              acc[0][q + w] = dp4x4(av[q], ur, acc[0][q + w]);
              if constexpr (CPX) {
                acc[1][q + w] = dp4x4(av[kDig + q], ui, acc[1][q + w]);
                acc[2][q + w] = dp4x4(av[q], ui, acc[2][q + w]);
                acc[3][q + w] = dp4x4(av[kDig + q], ur, acc[3][q + w]);
              }
            }
          }
        }
        // the row tile's sums: over the warps exactly, one level per warp; then the eight levels
        // as two 64-bit integers (|sums| < 2^37), weighted in FP64
#pragma unroll
        for (int q = 0; q < NP; q++)
#pragma unroll
          for (int L = 0; L < NL; L++) {
            accs[q * NL + L][warp][lane] = acc[q][L];
            acc[q][L] = 0;
          }
        bar_named<1, 256>();
        {
          long long s0 = 0, s1 = 0, s2 = 0, s3 = 0;
#pragma unroll
          for (int w = 0; w < 8; w++) {
            s0 += accs[warp][w][lane];
            if constexpr (CPX) {
              s1 += accs[NL + warp][w][lane];
              s2 += accs[2 * NL + warp][w][lane];
              s3 += accs[3 * NL + warp][w][lane];
            }
          }
          lvl[warp * 32 + lane] = s0 - s1;
          if constexpr (CPX) lvl[(NL + warp) * 32 + lane] = s2 + s3;
        }
        bar_named<1, 256>();
        if (warp == 0 && row < j) {
          const int E = drow + fu - 12;
          // 2^{E - 24} (sum_L S_L 2^{24 - 8L}, levels 0-3) + 2^{E - 56} (levels 4-7)
          auto levels = [&](const long long* sl) -> double {
            long long h = 0, l = 0;
#pragma unroll
            for (int L = 0; L < 4; L++) {
              h = (h << 8) + sl[L * 32 + lane];
              l = (l << 8) + sl[(4 + L) * 32 + lane];
            }
            const double v = fma((double)l, 0x1p-32, (double)h);
            const int be = E - 24 + 1023;
            return be > 0 && be < 2047 ? v * __longlong_as_double((long long)be << 52) : ldexp(v, E - 24);
          };
          T pv;
          if constexpr (CPX) pv = inv * T{levels(lvl), levels(lvl + NL * 32)};
          else pv = inv * levels(lvl);
          P[((size_t)b * maxseg + seg) * 32 + lane] = pv;
          const T ur = row == j - 1 ? from_real<T>(1.0) : (refl ? conjg(arow) * inv : zero<T>());
          d0 = fma(re(ur), re(pv), d0);
          if constexpr (CPX) d0 = fma(im(ur), im(pv), d0);
        }
      }
      if (warp == 0) {
        d0 = warp_sum(d0);
        if (lane == 0) dot[b] = d0;
      }
      if (j > a.jl) {  // the next step's first tiles
        const PanelRuns pn(j - 1, G);
        const int n0 = pn.run0(b), n1 = pn.run0(b + 1);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < STG - 1; q++) issue(pn.C, n0 + warp + 8 * q, n1, q);
      }
    } else {
      // ---- u' for this CTA's rows, and their shares of Q^H u (entries 0..k-1) and U^H u
      T ya[2] = {zero<T>(), zero<T>()}, yb[2] = {zero<T>(), zero<T>()};  // even and odd rows
      for (int r0 = c0; r0 < ce; r0 += 64) {
        const int nr = min(64, ce - r0);
        bar_named<2, 128>();
        if (vt < nr) {
          const int c = r0 + vt;
          const T av = r0 == c0 ? apre : ldcg(ar + c);
          const T uv = c == j - 1 ? from_real<T>(1.0) : (refl ? conjg(av) * inv : zero<T>());
          s_us[vt] = uv;
          U[(size_t)c * ldu + k] = uv;
          A[(size_t)j * lda + c] = c == j - 1 ? s_sub : (refl ? uv : av);
        }
        bar_named<2, 128>();
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const int en = vt + 128 * h;
          if (en >= 2 * k) break;
          const T* src = (en < k ? Q + en : U + (en - k)) + (size_t)r0 * ldu;
          for (int r = 0; r < nr; r += 8) {  // eight rows' loads in flight
            T v[8];
#pragma unroll
            for (int q = 0; q < 8; q++)
              v[q] = r + q < nr ? src[(size_t)(r + q) * ldu] : zero<T>();
#pragma unroll
            for (int q = 0; q < 8; q++)
              if (r + q < nr) macc(q & 1 ? yb[h] : ya[h], v[q], s_us[r + q]);
          }
        }
      }
      // barrier of the vector warps over the item's CTAs
      auto vbarrier = [&]() {
        bar_named<2, 128>();
        arrivedv += CL ? 1u : (unsigned)G;
        if (CL) {
          uint64_t* sb = &s_bar[2 + ((arrivedv - 1) & 1u)];
          if (warp == 8 && lane < G) cluster_arrive(sb, lane);
          if (vt == 0 && !cluster_wait(sb, ((arrivedv - 1) >> 1) & 1u, a.wait)) s_abort = 1;
        } else if (vt == 0) {
          red_release(bar + 1);
          if (!grid_wait(bar + 1, arrivedv, bar + 2, a.wait)) s_abort = 1;
        }
        bar_named<2, 128>();
      };
      if (k > 0) {
#pragma unroll
        for (int h = 0; h < 2; h++)
          if (vt + 128 * h < 2 * k) part[(size_t)b * (2 * kPanelMax) + vt + 128 * h] = ya[h] + yb[h];
        vbarrier();
        // LG lanes per entry, 32 / LG entries per warp at a time
        const int LG = G > 16 ? 32 : G > 8 ? 16 : 8, per = 32 / LG, sub = lane / LG, sl = lane % LG;
        for (int e0 = (warp - 8) * per; b + G * e0 < 2 * k; e0 += 4 * per) {
          const int en = b + G * (e0 + sub);
          T v = zero<T>();
          if (en < 2 * k)
            for (int g = sl; g < G; g += LG) v += ldcg(part + (size_t)g * (2 * kPanelMax) + en);
          for (int o = LG >> 1; o > 0; o >>= 1) v += shfl_xor(v, o);
          if (sl == 0 && en < 2 * k) y[en] = v;
        }
      }
      if (a.early) {
        if (k > 0) {
          vbarrier();
          load_panel_vectors(vt, 128);
          bar_named<2, 128>();
        }
        // groups of 8 lanes, one row each (16 rows at a time): U y1 + Q y2 into Q's new column
        // (replaced by q below), row j-1 with the earlier updates into the next row's buffer
        const int grp = vt >> 3, gl = vt & 7;
        T* an = arow2 + ((j - 1) & 1) * a.sv;
        for (int base = c0; base < ce; base += 16) {
          const int c = base + grp;
          T corr = zero<T>(), rs = zero<T>();
          if (c < ce) {
            const T* Uc = U + (size_t)c * ldu;
            const T* Qc = Q + (size_t)c * ldu;
            for (int s0 = gl; s0 < k; s0 += 32) {  // four steps' loads in flight
              T u0[4], q0[4];
#pragma unroll
              for (int q = 0; q < 4; q++) {
                const int sq = min(s0 + 8 * q, k - 1);
                u0[q] = Uc[sq];
                q0[q] = Qc[sq];
              }
#pragma unroll
              for (int q = 0; q < 4; q++)
                if (s0 + 8 * q < k) correct(corr, rs, u0[q], q0[q], s0 + 8 * q);
            }
          }
          corr = group8_sum(corr);
          rs = group8_sum(rs);
          if (c < ce && gl == 0) {
            Q[(size_t)c * ldu + k] = corr;
            if (j > a.jl) an[c] = A[(size_t)(j - 1) * lda + c] - rs;
          }
        }
      }
    }
    // where the partial products of this lane's first row of the next part lie (the integer
    // divisions before the barrier)
    // (16 lanes per row where one pass of 20 rows does, else 8 and passes of 40)
    const int lr = ce - c0 <= 20 ? 4 : 3, LR = 1 << lr, RP = 320 >> lr;
    const int grp = tid >> lr, gl = tid & (LR - 1);
    const int prow = warp < 10 ? c0 + grp : j - 1, pl = warp < 10 ? gl : lane, pn = warp < 10 ? LR : 32;
    int pb0 = 0, pb1 = -1, pg0 = 0, pg1 = 0;
    if (warp < 10 ? prow < ce : warp == 11) {
      pb0 = pr.owner((prow >> 5) * pr.C) + pl;
      pb1 = pr.owner(((prow >> 5) + 1) * pr.C - 1);
      if (pb0 <= pb1) {
        pg0 = pr.run0(pb0);
        pg1 = pr.run0(pb0 + 1);
        pg0 = pg0 < pg1 ? (prow >> 5) - pg0 / (int)pr.C : -1;  // the run's segment, -1: empty run
      }
    }
    if (!barrier()) break;

    // ---- p, q, and row j-1 with the panel's updates
    const bool rowupd = j > a.jl;
    const double t = s_tau;
    auto p_from = [&](int row, int g, int b1, int nl) -> T {  // runs g, g + nl .. b1 of the row
      const int r = row >> 5;
      T v = zero<T>();
      for (; g <= b1; g += nl) {
        const int g0 = pr.run0(g);
        if (g0 < pr.run0(g + 1)) v += ldcg(P + ((size_t)g * maxseg + (r - g0 / (int)pr.C)) * 32 + (row & 31));
      }
      return v;
    };
    // groups of LR lanes of warps 0-9, one row each; kq and row j-1's p on the other two warps;
    // the first rows' loads go out before y arrives
    T* an = arow2 + ((j - 1) & 1) * a.sv;
    const int ke = a.early ? 0 : k;  // steps of the corrections still to do
    T pv0 = zero<T>(), u0[4], q0[4];
    double dsum = 0.0;
    if (warp < 10) {
      if (c0 + grp < ce) {
        const T* Uc = U + (size_t)(c0 + grp) * ldu;
        const T* Qc = Q + (size_t)(c0 + grp) * ldu;
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const int sq = max(min(gl + LR * q, ke - 1), 0);
          u0[q] = ke > 0 ? Uc[sq] : zero<T>();
          q0[q] = ke > 0 ? Qc[sq] : zero<T>();
        }
      }
    } else if (warp == 10) {
      for (int g = lane; g < G; g += 32) dsum += __ldcg(dot + g);
    }
    if (pb0 <= pb1) {
      if (pg0 >= 0) pv0 = ldcg(P + ((size_t)pb0 * maxseg + pg0) * 32 + (prow & 31));
      if (pb0 + pn <= pb1) pv0 += p_from(prow, pb0 + pn, pb1, pn);
    }
    if (!a.early) load_panel_vectors(tid, kPanelThreads);
    __syncthreads();
    if (warp == 10) {  // kq = (tau / 2) u^H p = (tau^2 / 2) (u^H p_raw - 2 Re y2^H y1)
      for (int s = lane; s < k; s += 32) {
        dsum = fma(-2.0 * re(y2s[s]), re(y1s[s]), dsum);
        if constexpr (CPX) dsum = fma(-2.0 * im(y2s[s]), im(y1s[s]), dsum);
      }
      dsum = warp_sum(dsum);
      if (lane == 0) s_kq = (0.5 * t) * (t * dsum);
    } else if (warp == 11 && rowupd) {  // p[j-1] - U y1 - Q y2 of row j-1
      for (int s = lane; s < k; s += 32) {
        mac(pv0, -ujs[s], y1s[s]);
        mac(pv0, -qjs[s], y2s[s]);
      }
      pv0 = warp_sum(pv0);
      if (lane == 0) s_pj = pv0;
    }
    double n2 = 0.0;
    int ex = NOEXP;
    bool synced = false;
    for (int base = c0; base < ce || !synced; base += RP) {
      const int c = base + grp;
      const bool ok = c < ce && warp < 10;
      T pv = pv0, corr = zero<T>(), rs = zero<T>(), uc = zero<T>(), aold = zero<T>();
      int dc = 0;
      if (ok) {
        const T* Uc = U + (size_t)c * ldu;
        const T* Qc = Q + (size_t)c * ldu;
        if (synced) pv = p_from(c, pr.owner((c >> 5) * pr.C) + gl, pr.owner(((c >> 5) + 1) * pr.C - 1), LR);
        if (gl == 0) {
          uc = ldcg(Uc + k);
          if (a.early) corr = ldcg(Qc + k);
          if (rowupd) {
            aold = a.early ? ldcg(an + c) : A[(size_t)(j - 1) * lda + c];
            dc = deq(rmax[c]);
          }
        }
        for (int s0 = gl; s0 < ke; s0 += 4 * LR) {  // four steps' loads in flight
          if (synced || s0 > gl) {
#pragma unroll
            for (int q = 0; q < 4; q++) {
              const int sq = min(s0 + LR * q, ke - 1);
              u0[q] = Uc[sq];
              q0[q] = Qc[sq];
            }
          }
#pragma unroll
          for (int q = 0; q < 4; q++) {
            const int sq = s0 + LR * q;
            if (sq < ke) correct(corr, rs, u0[q], q0[q], sq);
          }
        }
      }
      if (warp < 10) {
        pv = pv - corr;
        const bool upd = ke > 0 && rowupd;
        if (LR == 16) {
          pv += shfl_xor(pv, 8);
          if (upd) rs += shfl_xor(rs, 8);
        }
        pv = group8_sum(pv);
        if (upd) rs = group8_sum(rs);
      }
      if (!synced) {  // kq and row j-1's share
        __syncthreads();
        synced = true;
      }
      if (ok && gl == 0) {
        const double kq = s_kq;
        const T qc = t * pv - kq * uc;
        Q[(size_t)c * ldu + k] = qc;
        if (rowupd) {
          const T qj = t * s_pj - from_real<T>(kq);  // u'[j-1] = 1
          rs += conjg(qc);
          mac(rs, qj, conjg(uc));
          const T an_c = aold - rs;
          if (c == j - 1) {
            A[(size_t)(j - 1) * lda + c] = an_c;
          } else {
            an[c] = an_c;
            if (c < j - 2) {
              n2 += abs2(an_c);
              ex = max(ex, scale_of(an_c, dc));
            }
          }
        }
      }
    }
    if (!rowupd) break;
    put_norm(n2, ex, true);
    live = barrier();
  }
  cp_async_wait<0>();
  if (CL) cluster_sync_all();  // no CTA leaves while another may still arrive on its barriers
  if (s_abort && tid == 0) set_status(a.st ? a.st + z : nullptr, ST_ETIMEOUT, -3);
}

// CTAs per item: as many as leave each at most kPanelTiles digit tiles and kPanelRows<T> rows
// (the split of its FP64 corrections), up to the SMs.  Twice as many (12 tiles, 8 / 4 rows) is
// 2 % faster for one problem (order 1152 real: 20.0 against 20.6 ms the whole call) but leaves
// no SMs to other streams' reductions: eight uneven systems of order 208 to 1144 on eight
// streams 57 ms against 43; half as many 36 ms, and one problem 4 % slower.  The count depends
// on the problem alone, so a solve in a batch gives the bits of the solve by itself.
constexpr int kPanelTiles = 24;
template <typename T>
constexpr int kPanelRows = sizeof(T) == 16 ? 8 : 16;
// Per device, found once: the value of `find` for the current device (kernel attributes are
// per device too).
template <typename F>
static int per_device(std::atomic<int> (&known)[64], F find) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 64) return find(dev);
  int v = known[dev].load();  // value + 1
  if (v == 0) known[dev].store(v = find(dev) + 1);
  return v - 1;
}
template <typename T>
static int panel_capacity() {
  static std::atomic<int> known[64];
  return per_device(known, [](int dev) {
    int sms = 0, per = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(hetrd_panel_kernel<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         PanelSmem<T>::TOTAL);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, hetrd_panel_kernel<T, false>, kPanelThreads,
                                                  PanelSmem<T>::TOTAL);
    cudaGetLastError();
    return sms * (per > 0 ? 1 : 0);
  });
}
// Clusters of c panel CTAs (c = 16, 8, 4, 2, 1) that are resident at once, attributes set.
template <typename T, int c>
static int panel_clusters() {
  static std::atomic<int> known[64];
  return per_device(known, [](int) {
    auto k = hetrd_panel_kernel<T, true>;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, PanelSmem<T>::TOTAL);
    cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = c;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(kPanelThreads);
    cfg.dynamicSmemBytes = PanelSmem<T>::TOTAL;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n > 0) return n;
    cudaGetLastError();
    return 0;
  });
}

template <typename T>
static int hetrd_panel_ctas(int jh, int items) {
  const int top = std::min(panel_capacity<T>() / items, kPanelCtas);
  const long long tiles = (long long)((jh + 31) / 32) * ((jh + 15) / 16);
  return (int)std::min<long long>(
      top, std::max<long long>((tiles + kPanelTiles - 1) / kPanelTiles, (jh + kPanelRows<T> - 1) / kPanelRows<T>));
}

// The cluster form: one cluster of up to 16 CTAs per item, barriers through shared-memory
// mbarriers, no co-residency of the whole grid needed.  It pays at the smallest orders only
// (16 SMs do the FP64 corrections: order 640 real 20 us per step against 12.7 us on 80 CTAs).
// The largest cluster of which the GPU holds one per item: a step of these orders is latency,
// and waves of clusters repeat it.  All panels of a call, clusters of 16 in waves / this rule:
// order 104 complex, 8 items 2.77 / 1.58 ms, 64 items 13.9 / 2.9, 512 items 105 / 14; order 40
// real, 1000 items 48.8 / 3.2 (two launches per step in FP64: 3.8).
constexpr long long kClusterTiles = 64;
static bool panel_in_cluster(int jh) {
  return (long long)((jh + 31) / 32) * ((jh + 15) / 16) <= kClusterTiles;
}
template <typename T>
static int panel_cluster_ctas(int items) {
  if (panel_clusters<T, 16>() >= items) return 16;
  if (panel_clusters<T, 8>() >= items) return 8;
  if (panel_clusters<T, 4>() >= items) return 4;
  if (panel_clusters<T, 2>() >= items) return 2;
  return panel_clusters<T, 1>() > 0 ? 1 : 0;
}

template <typename T>
int hetrd_panel_items(int jh, int items) {
  if (panel_in_cluster(jh) && panel_cluster_ctas<T>(items) > 0) return items;
  while (items > 1 && panel_capacity<T>() < items) items = (items + 1) / 2;
  return items;
}

template <typename T>
constexpr int kEarlyTiles = sizeof(T) == 16 ? 60 : 150;
template <typename T>
bool hetrd_panel(PanelArgs<T> a, int items, unsigned* base, unsigned* basev, cudaStream_t s) {
  const int cl = panel_in_cluster(a.jh) ? panel_cluster_ctas<T>(items) : 0;
  const int G = cl > 0 ? cl : std::min(a.gs, hetrd_panel_ctas<T>(a.jh, items));
  if (G < 1) return false;
  int maxseg = (a.jh + 31) / 32 / G + 2;
  const int steps = a.jh - a.jl + 1;
  // U y1 + Q y2 behind the product from kEarlyTiles tiles per CTA up
  a.early = (long long)((a.jh + 31) / 32) * ((a.jh + 15) / 16) >= (long long)kEarlyTiles<T> * G;
  a.base = *base;
  a.basev = *basev + a.late;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  cfg.gridDim = dim3(G, items);
  cfg.blockDim = dim3(kPanelThreads);
  cfg.dynamicSmemBytes = PanelSmem<T>::TOTAL;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  count_launch();
  if (cl > 0) {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = G;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    return cudaLaunchKernelEx(&cfg, hetrd_panel_kernel<T, true>, a, maxseg) == cudaSuccess;
  }
  *base += 2u * steps * G;
  *basev += (a.early ? 2u : 1u) * (unsigned)(steps - 1) * G;
  cudaFuncSetAttribute(hetrd_panel_kernel<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, PanelSmem<T>::TOTAL);
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  return cudaLaunchKernelEx(&cfg, hetrd_panel_kernel<T, false>, a, maxseg) == cudaSuccess;
}

// d_i = Re A_ii, e_i = |A_{i+1,i}|, ph_0 = 1, ph_{i+1} = ph_i A_{i+1,i}/|A_{i+1,i}|.  One CTA
// per item; the phases are a scan of products: a run of rows per thread, the runs' products
// over the block, then every row of the run.  (One thread walking the rows took 4.5 ms at
// order 4992.)
template <typename T>
__global__ void __launch_bounds__(1024) hetrd_finish_kernel(const T* A, int lda, long long sA, int m, double* d,
                                                            double* e, long long sde, T* ph, long long sph) {
  __shared__ T run[1024];
  const int z = blockIdx.x, tid = threadIdx.x;
  A += z * sA;
  d += z * sde;
  e += z * sde;
  ph += z * sph;
  const int per = (m + 1023) / 1024, i0 = tid * per, i1 = min(m, i0 + per);
  auto unit = [&](int i) -> T {  // phase of A_{i+1,i} (1 where it is zero)
    const T s = A[(size_t)(i + 1) * lda + i];
    const double a = sqrt(abs2(s));
    return a > 0.0 ? s * (1.0 / a) : from_real<T>(1.0);
  };
  T prod = from_real<T>(1.0);
  for (int i = i0; i < i1; i++) {
    d[i] = re(A[(size_t)i * lda + i]);
    if (i + 1 < m) {
      e[i] = sqrt(abs2(A[(size_t)(i + 1) * lda + i]));
      const T w = unit(i);
      ph[i + 1] = w;  // the row's own factor, replaced below
      prod = prod * w;
    }
  }
  run[tid] = prod;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {  // inclusive scan
    const T v = tid >= o ? run[tid - o] : from_real<T>(1.0);
    __syncthreads();
    run[tid] = v * run[tid];
    __syncthreads();
  }
  T cur = tid > 0 ? run[tid - 1] : from_real<T>(1.0);
  if (tid == 0) ph[0] = cur;
  for (int i = i0; i < i1 && i + 1 < m; i++) {
    cur = cur * ph[i + 1];
    ph[i + 1] = cur;
  }
}

__device__ __forceinline__ double widen(double a) { return a; }
__device__ __forceinline__ double widen(float a) { return (double)a; }
__device__ __forceinline__ zc widen(zc a) { return a; }
__device__ __forceinline__ zc widen(cf a) { return zc{(double)a.x, (double)a.y}; }

// V[:, c] = u'_{j1-c} (rows 0..j1-1), tb[c] = tau[j1-c].  Reflectors stored in single
// precision (the mixed-precision path) are widened exactly to FP64.
template <typename T, typename TV>
__global__ void gather_reflectors_kernel(const T* A, int lda, long long sA, const double* tau, long long stau,
                                         int j0, int j1, TV* V, int ldv, long long sV, double* tb, long long stb) {
  const int z = blockIdx.z;
  A += z * sA;
  tau += z * stau;
  V += z * sV;
  tb += z * stb;
  const int nbb = j1 - j0 + 1;
  for (int i = blockIdx.y; i < j1; i += gridDim.y)
    for (int c = threadIdx.x; c < nbb; c += blockDim.x) {
      int jj = j1 - c;
      TV v = zero<TV>();
      if (i < jj - 1) v = widen(A[(size_t)jj * lda + i]);
      else if (i == jj - 1) v = from_real<TV>(1.0);
      V[(size_t)i * ldv + c] = v;
      if (i == 0) tb[c] = tau[jj];
    }
}

template <typename T>
void hetrd_reflector(T* A, int lda, long long sA, int j, T* u, long long sv, double* tau, long long stau, int count,
                     cudaStream_t s, double* uw) {
  count_launch();
  hetrd_reflector_kernel<T><<<count, 256, 0, s>>>(A, lda, sA, j, u, sv, tau, stau, uw);
}

template <typename T>
void hetrd_digits(const T* A, int lda, long long sA, int n, const HemvDigits& hd, int count, cudaStream_t s) {
  if (n <= 0) return;
  cudaMemsetAsync(hd.rmax, 0, sizeof(unsigned long long) * hd.ldd * count, s);
  count_launch(2);
  hetrd_dmax_kernel<T><<<dim3((n + 63) / 64, (n + 63) / 64, count), 256, 0, s>>>(A, lda, sA, n, hd.rmax, hd.ldd);
  const int nt = ((n + 15) / 16 * 16 + 31) / 32;
  hetrd_digits_kernel<T><<<dim3(nt, nt, count), 64, 0, s>>>(A, lda, sA, n, hd);
}

void hetrd_sums(const zc* A, int lda, long long sA, int n, double* Sg, int count, cudaStream_t s) {
  if (n <= 0) return;
  dim3 grid((n + 255) / 256 < 16 ? (n + 255) / 256 : 16, n < 4096 ? n : 4096, count);
  count_launch();
  hetrd_sums_kernel<<<grid, 256, 0, s>>>(A, lda, sA, n, Sg);
}

template <typename T>
void hetrd_phemv(const T* A, int lda, long long sA, int j, const T* u, T* p, long long sv, const double* tau,
                 long long stau, const T* U, const T* Q, int ldu, long long sU, int k, T* part, long long spart,
                 T* y, long long sy, int* ticket, int count, cudaStream_t s, const double* Sg, const double* uw) {
  count_launch();
  if ((long long)((j + 63) / 64) * count >= 4 * 152)
    hetrd_phemv_kernel<T, 64><<<dim3((j + 63) / 64, count), 256, 0, s>>>(A, lda, sA, j, u, p, sv, tau, stau, U, Q,
                                                                         ldu, sU, k, part, spart, y, sy, ticket, Sg,
                                                                         uw);
  else
    hetrd_phemv_kernel<T, 16><<<dim3((j + 15) / 16, count), 256, 0, s>>>(A, lda, sA, j, u, p, sv, tau, stau, U, Q,
                                                                         ldu, sU, k, part, spart, y, sy, ticket, Sg,
                                                                         uw);
}

template <typename T>
void hetrd_pupdate(T* A, int lda, long long sA, int j, T* u, const T* p, long long sv, double* tau, long long stau,
                   T* U, T* Q, int ldu, long long sU, int k, const T* y, long long sy, int rowupd, int* ticket,
                   int count, cudaStream_t s, double* uw) {
  const int sm = (int)(4 * sizeof(T) * (ldu + 1));
  if (sm > 48 * 1024) cudaFuncSetAttribute(hetrd_pupdate_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  count_launch();
  hetrd_pupdate_kernel<T><<<dim3((j + 63) / 64, count), 256, sm, s>>>(A, lda, sA, j, u, p, sv, tau, stau, U, Q, ldu,
                                                                      sU, k, y, sy, rowupd, ticket, uw);
}

template <typename T>
void hetrd_finish(const T* A, int lda, long long sA, int m, double* d, double* e, long long sde, T* ph,
                  long long sph, int count, cudaStream_t s) {
  count_launch();
  hetrd_finish_kernel<T><<<count, 1024, 0, s>>>(A, lda, sA, m, d, e, sde, ph, sph);
}

template <typename T, typename TV>
void gather_reflectors(const T* A, int lda, long long sA, const double* tau, long long stau, int j0, int j1,
                       TV* V, int ldv, long long sV, double* tb, long long stb, int count, cudaStream_t s) {
  dim3 grid(1, j1 < 2048 ? j1 : 2048, count);
  count_launch();
  gather_reflectors_kernel<T, TV><<<grid, 64, 0, s>>>(A, lda, sA, tau, stau, j0, j1, V, ldv, sV, tb, stb);
}

// ph (FP64 type) from the single-precision phases of the mixed-precision path.
template <typename T, typename TV>
__global__ void widen_kernel(const T* src, TV* dst, long long n) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    dst[t] = widen(src[t]);
}

template <typename T, typename TV>
void widen_copy(const T* src, TV* dst, long long n, cudaStream_t s) {
  if (n <= 0) return;
  count_launch();
  const long long b = (n + 255) / 256;
  widen_kernel<T, TV><<<(int)(b < 4096 ? b : 4096), 256, 0, s>>>(src, dst, n);
}

// W = [U 2^h | Q 2^-h | U 2^h] (n rows of 3 kp), h per column the power of two that brings
// the column's largest entries of U and Q together: the deferred update U Q^H + Q U^H is then
// one product W[:, 0:2kp] W[:, kp:3kp]^H.  A row of W has one scale, so both parts are truncated
// below the larger of the two balanced ones (two products scale them apart): normwise the same,
// |W|^2 = |U| |Q| columnwise.  On matrices D B D graded over 6 and 10 decades either way (order 200
// complex, B of condition 6) the small eigenvalues come out as with two products: worst relative
// error 3.1e-12 against 2.9e-12 in the direction that keeps them, norm error 7e-16 against 1.4e-15.
// CTAs of 32 bytes of a row; the second reading comes from L2.  HBM-bound (5 entries moved per
// entry of U); the update's reconstruction and C traffic halve: reduction of order 4992 complex
// 235.7 -> 229.5 ms, four of 1625 54.6 -> 52.5, order 2808 real 50.3 -> 48.8.
constexpr int kPackThreads = 1024;
template <typename T>
__global__ void __launch_bounds__(kPackThreads) panel_pack_kernel(const T* U, const T* Q, int ldu, long long sU, int n,
                                                                  int kp, T* W, long long sW) {
  constexpr int C = 32 / sizeof(T);
  __shared__ int top[2][C];
  const int z = blockIdx.y, c = threadIdx.x % C, k = blockIdx.x * C + c, r0 = threadIdx.x / C;
  U += z * sU;
  Q += z * sU;
  W += z * sW;
  if (threadIdx.x < 2 * C) (&top[0][0])[threadIdx.x] = 0;
  __syncthreads();
  auto mag = [](T v) { return max(__double2hiint(fabs(re(v))), __double2hiint(fabs(im(v)))); };
  if (k < kp) {
    int mu = 0, mq = 0;
#pragma unroll 8
    for (int r = r0; r < n; r += kPackThreads / C) {
      mu = max(mu, mag(U[(size_t)r * ldu + k]));
      mq = max(mq, mag(Q[(size_t)r * ldu + k]));
    }
    atomicMax(&top[0][c], mu);
    atomicMax(&top[1][c], mq);
  }
  __syncthreads();
  if (k >= kp) return;
  const int eu = top[0][c] >> 20, eq = top[1][c] >> 20;  // 0: zero or subnormal, 2047: not finite
  const int h = eu == 0 || eq == 0 || eu == 2047 || eq == 2047 ? 0 : (eq - eu) >> 1;
  const double su = __hiloint2double((1023 + h) << 20, 0), sq = __hiloint2double((1023 - h) << 20, 0);
#pragma unroll 4
  for (int r = r0; r < n; r += kPackThreads / C) {
    const T u = su * U[(size_t)r * ldu + k], q = sq * Q[(size_t)r * ldu + k];
    T* w = W + (size_t)r * 3 * kp + k;
    w[0] = u;
    w[kp] = q;
    w[2 * kp] = u;
  }
}

template <typename T>
void panel_pack(const T* U, const T* Q, int ldu, long long sU, int n, int kp, T* W, long long sW, int count,
                cudaStream_t s) {
  constexpr int C = 32 / sizeof(T);
  count_launch();
  panel_pack_kernel<T><<<dim3((kp + C - 1) / C, count), kPackThreads, 0, s>>>(U, Q, ldu, sU, n, kp, W, sW);
}

// Lower triangle of the FP64 A (lda, sA) rounded into the single-precision B (ldb, sB).
template <typename T, typename TL>
__global__ void narrow_lower_kernel(const T* A, int lda, long long sA, TL* B, int ldb, long long sB, int n) {
  const int z = blockIdx.z;
  A += z * sA;
  B += z * sB;
  for (int i = blockIdx.y; i < n; i += gridDim.y)
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j <= i; j += gridDim.x * blockDim.x) {
      const T a = A[(size_t)i * lda + j];
      TL b;
      if constexpr (sizeof(T) == 16) b = TL{(float)re(a), (float)im(a)};
      else b = (TL)re(a);
      B[(size_t)i * ldb + j] = b;
    }
}

template <typename T, typename TL>
void narrow_lower(const T* A, int lda, long long sA, TL* B, int ldb, long long sB, int n, int count, cudaStream_t s) {
  if (n <= 0) return;
  dim3 grid((n + 255) / 256 < 16 ? (n + 255) / 256 : 16, n < 2048 ? n : 2048, count);
  count_launch();
  narrow_lower_kernel<T, TL><<<grid, 256, 0, s>>>(A, lda, sA, B, ldb, sB, n);
}

#define INST(T)                                                                                            \
  template void hetrd_reflector<T>(T*, int, long long, int, T*, long long, double*, long long, int,         \
                                   cudaStream_t, double*);                                                 \
  template void hetrd_phemv<T>(const T*, int, long long, int, const T*, T*, long long, const double*,        \
                               long long, const T*, const T*, int, long long, int, T*, long long, T*, long long, \
                               int*, int, cudaStream_t, const double*, const double*);                     \
  template void hetrd_pupdate<T>(T*, int, long long, int, T*, const T*, long long, double*, long long, T*,  \
                                 T*, int, long long, int, const T*, long long, int, int*, int, cudaStream_t, \
                                 double*);                                                                \
  template void hetrd_finish<T>(const T*, int, long long, int, double*, double*, long long, T*, long long,   \
                                int, cudaStream_t);                                                        \
  template void gather_reflectors<T, T>(const T*, int, long long, const double*, long long, int, int, T*,    \
                                        int, long long, double*, long long, int, cudaStream_t);               \
  template void hetrd_digits<T>(const T*, int, long long, int, const HemvDigits&, int, cudaStream_t);           \
  template void panel_pack<T>(const T*, const T*, int, long long, int, int, T*, long long, int, cudaStream_t);    \
  template int hetrd_panel_items<T>(int, int);                                                             \
  template bool hetrd_panel<T>(PanelArgs<T>, int, unsigned*, unsigned*, cudaStream_t);
INST(double)
INST(zc)
#undef INST
#define INST(T)                                                                                            \
  template void hetrd_reflector<T>(T*, int, long long, int, T*, long long, double*, long long, int,         \
                                   cudaStream_t, double*);                                                 \
  template void hetrd_phemv<T>(const T*, int, long long, int, const T*, T*, long long, const double*,        \
                               long long, const T*, const T*, int, long long, int, T*, long long, T*, long long, \
                               int*, int, cudaStream_t, const double*, const double*);                     \
  template void hetrd_pupdate<T>(T*, int, long long, int, T*, const T*, long long, double*, long long, T*,  \
                                 T*, int, long long, int, const T*, long long, int, int*, int, cudaStream_t, \
                                 double*);                                                                \
  template void hetrd_finish<T>(const T*, int, long long, int, double*, double*, long long, T*, long long,   \
                                int, cudaStream_t);
INST(float)
INST(cf)
template void gather_reflectors<float, double>(const float*, int, long long, const double*, long long, int, int,
                                               double*, int, long long, double*, long long, int, cudaStream_t);
template void gather_reflectors<cf, zc>(const cf*, int, long long, const double*, long long, int, int, zc*, int,
                                        long long, double*, long long, int, cudaStream_t);
template void widen_copy<float, double>(const float*, double*, long long, cudaStream_t);
template void widen_copy<cf, zc>(const cf*, zc*, long long, cudaStream_t);
template void narrow_lower<double, float>(const double*, int, long long, float*, int, long long, int, int,
                                          cudaStream_t);
template void narrow_lower<zc, cf>(const zc*, int, long long, cf*, int, long long, int, int, cudaStream_t);

}  // namespace gks
