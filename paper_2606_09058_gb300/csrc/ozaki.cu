// FP64-accurate GEMM from exact bf16 tensor-core products, in two forms: residues modulo 16
// coprime moduli and the Chinese remainder theorem (the default; Ozaki, Uchino and Imamura),
// described at the moduli below, and digit pairs (Ozaki, Ogita, Oishi and Rump's error-free
// splitting):
//
// Each row i of op(A) is scaled by 2^-e_i (e_i = 1 + floor(log2 max_k |a_ik|), so every
// entry is below 1 in magnitude) and cut into S digits of 6 bits, truncating toward zero:
//   a_ik = 2^e_i * sum_{s=1..S} d_s(i,k) 2^{-6s} + r,  |d_s| <= 63,  |r| < 2^{e_i - 6S}.
// Columns of op(B) are cut the same way.  Every digit is an integer of at most 6 bits, so
// it is exact in bf16 and every digit product (< 2^12) and every sum of up to 4096 of them
// is exact in the FP32 accumulator of the bf16 mma.  The kernel multiplies the digit pairs
// with s + t <= S + 1 (the dropped pairs are below 2^{-6(S+1)}), drains each exact chunk
// into an FP64 accumulator scaled by 2^{-6(s+t)}, and applies 2^{e_i + f_j} at the end.
// With S = 9 the digits carry 54 bits below each row's largest entry.  (S <= 10 keeps the
// digit integer within 60 bits.)
//
// Complex products use a real embedding that keeps (Re, Im) of one output next to each
// other: A' = [Re a, Im a] interleaved along k, B' column 2j = (Re b, -Im b) interleaved,
// column 2j+1 = (Im b, Re b); then (A' B')[i][2j] = Re c_ij and [i][2j+1] = Im c_ij.
//
// On GB300 the bf16 tensor cores (tcgen05) run the 45 digit products of S = 9 at an
// FP64-equivalent rate of 18 TFLOP/s and the 16 residue products at 73 TFLOP/s on a complex
// product of order 4096, against 1.06 TFLOP/s for the FP64 pipe.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <mutex>
#include <type_traits>

#include "dense.h"
#include "tcgen05.cuh"

namespace gks {

static constexpr int OZ_BITS = 6;
static constexpr int OZ_KSTEP = 64;   // k per pipeline step
static constexpr int OZ_CHUNK = 4096; // exact FP32 accumulation length (63*63*4096 < 2^24)

// ------------------------------------------------------------------ splitting

// ------------------------------------------------------------------ residue moduli
// Pairwise coprime moduli up to 256 (2^8, 3*5*17, 11*23, 251, 13*19, 241, 239, 233, 229,
// 227, 223, 7*31, 211, 199, 197, 193), largest first: a residue in symmetric form has
// |r| <= 128, an integer exact in bf16, and a product of two is at most 2^14.
static constexpr int CRT_MAXMOD = 16;
__host__ __device__ constexpr uint32_t crt_mod(int l) {
  return l == 0 ? 256u : l == 1 ? 255u : l == 2 ? 253u : l == 3 ? 251u : l == 4 ? 247u : l == 5 ? 241u
       : l == 6 ? 239u : l == 7 ? 233u : l == 8 ? 229u : l == 9 ? 227u : l == 10 ? 223u : l == 11 ? 217u
       : l == 12 ? 211u : l == 13 ? 199u : l == 14 ? 197u : 193u;
}

// Per-vector scale codes: 0 for a zero vector, e + kExpBias for entries below 2^e in
// magnitude, kExpNan for a vector with a non-finite entry (its products are NaN, as on the
// FP64 pipe).  Codes order like the magnitudes, so chunks of a vector combine by atomicMax.
static constexpr int kExpBias = 2048, kExpNan = 1 << 20;
__device__ __forceinline__ int exp_of(int code) { return code ? code - kExpBias : 0; }

// x - m round(x / m) for an integer-valued float |x| <= 2^24: the quotient is rounded with
// the 1.5 * 2^23 shift (|x / m| < 2^22), and the fused multiply-add is exact because the
// result is a small integer.
__device__ __forceinline__ float crt_fold(float x, float m, float inv) {
  const float q = __fsub_rn(__fmaf_rn(x, inv, 12582912.0f), 12582912.0f);
  return __fmaf_rn(-q, m, x);
}

// The split values of one element x of a vector whose entries are below 2^e in magnitude,
// into o[0..S); sh = 6S - e (digits) or p - e (residues).  Integer and FP32 operations only
// (the FP64 pipe takes 1.7 operations per SM clock): u = trunc(|x| 2^sh) is the significand
// shifted by the exponent difference.
// cs = 1 or -1 is a further sign (the conjugation's).
// Digits (RES false): the S base-64 digits of u, most significant first, with x's sign.
// Residues (RES true): u < 2^62 in 21-bit limbs, reduced modulo each of the first S moduli by
// Horner's rule in exact FP32 steps (|r| 2^7 + |limb| < 2^22), the limbs with x's sign:
// symmetric residues |r| <= 128.  11 FP32 operations per modulus in place of five 32-bit integer
// remainders by a constant.
// With wt (operand B) the residues are those of y_l times the integer, y_l = (M / m_l)^-1 mod
// m_l in symmetric form: the product's residues then carry the weights of the
// reconstruction, one multiplication per operand entry instead of one per output.
struct CrtWeights {
  float y[CRT_MAXMOD];
};
template <bool RES>
__device__ __forceinline__ void split_vals(double x, int sh, int S, float cs, float (&o)[16], const CrtWeights* wt) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int xe = (int)((bits >> 52) & 0x7ff);
  const unsigned long long m = xe == 0x7ff ? 0ull : (bits & 0xfffffffffffffull) | (xe ? (1ull << 52) : 0ull);
  const int s = (xe ? xe : 1) - 1075 + sh;
  const unsigned long long u = s >= 0 ? (s < 64 ? m << s : 0ull) : (s > -64 ? m >> -s : 0ull);
  const float sg = (bits >> 63) ? -cs : cs;
  if constexpr (RES) {
    const float a0 = sg * (float)(uint32_t)(u & 0x1fffffull), a1 = sg * (float)(uint32_t)((u >> 21) & 0x1fffffull),
                a2 = sg * (float)(uint32_t)(u >> 42);
#pragma unroll
    for (int l = 0; l < CRT_MAXMOD; l++) {
      constexpr uint32_t lim = 1u << 21;
      const uint32_t mi = crt_mod(l), wi = lim % mi;
      const float mf = (float)mi, inv = 1.0f / mf, w = 2u * wi > mi ? (float)wi - mf : (float)wi;
      const float r2 = crt_fold(a2, mf, inv);
      const float r1 = crt_fold(__fmaf_rn(r2, w, a1), mf, inv);
      o[l] = crt_fold(__fmaf_rn(r1, w, a0), mf, inv);
      if (wt) o[l] = crt_fold(o[l] * wt->y[l], mf, inv);
    }
  } else {
#pragma unroll
    for (int t = 0; t < 16; t++)
      o[t] = t < S ? sg * (float)((u >> (OZ_BITS * max(S - 1 - t, 0))) & 63) : 0.0f;
  }
}

// Two consecutive embedded positions of S planes, one 4-byte store per plane.
__device__ __forceinline__ void store_pair(const float (&o0)[16], const float (&o1)[16], float s1, __nv_bfloat16* dst,
                                           long long sstride, int S) {
#pragma unroll
  for (int s = 0; s < 16; s++)
    if (s < S)
      *reinterpret_cast<__nv_bfloat162*>(dst + s * sstride) = __floats2bfloat162_rn(o0[s], s1 * o1[s]);
}

// One operand of a split product: vector v is row v of op(A) (role 0) or column v of op(B)
// (role 1) of the stored matrix X (row-major, ld); op(A)_{v,k} = X[v][k] (N), X[k][v] (T),
// conj X[k][v] (C);  op(B)_{k,v} = X[k][v] (N), X[v][k] (T), conj X[v][k] (C).  Batch item z
// at item_off(z, sX, sX2, nb2); ksc (nullable, stride sks) scales element k first.
template <typename T>
struct SplitOp {
  const T* X;
  int ld, role, op, nvec, nvp;  // nvp: vectors with the padding (complex B: half the embedded rows)
  long long sX, sX2;
  int* ex;                      // scale codes, stride sE per item
  long long sE;
  const double* ksc;
  long long sks;
  __nv_bfloat16* D;             // planes [S][rows][Kp], item stride sD, plane stride sstride
  long long sstride, sD;
  __device__ bool contig() const { return (role == 0) == (op == OP_N); }  // k contiguous in memory
  // element k of vector v, up to signs (KS: scaled by kz)
  template <bool KS>
  __device__ T at(const T* Xz, const double* kz, int v, int k) const {
    T x = contig() ? Xz[(size_t)v * ld + k] : Xz[(size_t)k * ld + v];
    if constexpr (KS) x = x * kz[k];
    return x;
  }
  // the sign of the imaginary part that the conjugation asks for: 1 or -1
  __device__ float conj_sign() const { return op == OP_C ? -1.0f : 1.0f; }
};
// f<true>() with a scaled operand, f<false>() without: the FP64 multiplications (and the
// conjugation's, moved to the split values' signs) do not reach the unscaled path, whose
// reading they bound: scale pass of a complex 4096^2 pair 227 us with them, 92 us without.
template <typename F>
__device__ __forceinline__ void scaled_or_not(const double* kz, F f) {
  if (kz) f(std::true_type{});
  else f(std::false_type{});
}
template <typename T>
struct SplitPair {
  SplitOp<T> o[2];
  int n0;  // blockIdx.x below n0: operand 0
};

// Ordering key of |x|: the top word of its bits (1 for values below 2^-1042).
__device__ __forceinline__ uint32_t mag_key(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  return hi ? hi : (__double2loint(x) ? 1u : 0u);
}
__device__ __forceinline__ uint32_t mag_key(zc x) { return max(mag_key(x.x), mag_key(x.y)); }

__device__ __forceinline__ int exp_code(uint32_t m) {
  return m == 0 ? 0 : m >= 0x7ff00000u ? kExpNan : (int)(m >> 20) - 1022 + kExpBias;
}

// The planes of two embedded positions of vector v: the complex element k0 + lane (x0), or
// the real elements k0 + 2 lane and the next (x0, x1).
template <typename T, bool RES>
__device__ __forceinline__ void emit_pair(const SplitOp<T>& q, __nv_bfloat16* D, int v, int k0, int lane, T x0, T x1,
                                          int code, int Kp, int S, int p, const CrtWeights& y) {
  const int sh = code == kExpNan ? -4096 : (RES ? p : OZ_BITS * S) - exp_of(code);
  const CrtWeights* wt = q.role ? &y : nullptr;
  float o0[16], o1[16];
  if constexpr (sizeof(T) == 16) {
    split_vals<RES>(x0.x, sh, S, 1.0f, o0, wt);
    split_vals<RES>(x0.y, sh, S, q.conj_sign(), o1, wt);
    const size_t k = 2 * ((size_t)k0 + lane);
    if (q.role == 0) {
      store_pair(o0, o1, 1.0f, D + (size_t)v * Kp + k, q.sstride, S);
    } else {  // column 2v = (Re, -Im), column 2v + 1 = (Im, Re) along k
      store_pair(o0, o1, -1.0f, D + (size_t)(2 * v) * Kp + k, q.sstride, S);
      store_pair(o1, o0, 1.0f, D + (size_t)(2 * v + 1) * Kp + k, q.sstride, S);
    }
  } else {
    split_vals<RES>(x0, sh, S, 1.0f, o0, wt);
    split_vals<RES>(x1, sh, S, 1.0f, o1, wt);
    store_pair(o0, o1, 1.0f, D + (size_t)v * Kp + k0 + 2 * lane, q.sstride, S);
  }
}

// Pass 1, both operands in one launch: scale codes of 32 vectors over a chunk of kScaleK
// elements per CTA (grid x: vectors of A then of B, y: k chunks, z: items), combined by
// atomicMax into codes cleared beforehand.  Bound by reading the operands once; the chunks
// keep the GPU filled for thin operands (512 vectors of length 5000: 16 CTAs without them).
static constexpr int kScaleK = 512;
template <typename T>
__global__ void __launch_bounds__(256) oz_scale_kernel(const SplitPair<T> sp, int K, int nb2, const int* kdev) {
  __shared__ uint32_t pm[8][32];
  const bool second = (int)blockIdx.x >= sp.n0;
  const SplitOp<T>& q = sp.o[second];
  const int v0 = ((int)blockIdx.x - (second ? sp.n0 : 0)) * 32, z = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (kdev) K = min(K, max(0, kdev[z]));
  const int k0 = blockIdx.y * kScaleK, k1 = min(K, k0 + kScaleK);
  if (k0 >= k1) return;
  const T* X = q.X + item_off(z, q.sX, q.sX2, nb2);
  const double* kz = q.ksc ? q.ksc + z * q.sks : nullptr;
  int* ex = q.ex + z * q.sE;
  auto put = [&](int v, uint32_t m) {
    if (m) atomicMax(ex + v, exp_code(m));
  };
  if (q.contig()) {
    for (int vv = warp; vv < 32; vv += 8) {
      const int v = v0 + vv;
      if (v >= q.nvec) break;
      uint32_t m = 0;
      scaled_or_not(kz, [&](auto ks) {
        for (int k = k0 + lane; k < k1; k += 128) {  // four loads in flight per lane
          T x[4];
#pragma unroll
          for (int t = 0; t < 4; t++) x[t] = k + 32 * t < k1 ? q.template at<decltype(ks)::value>(X, kz, v, k + 32 * t) : zero<T>();
#pragma unroll
          for (int t = 0; t < 4; t++) m = max(m, mag_key(x[t]));
        }
      });
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) put(v, m);
    }
  } else {
    uint32_t m = 0;
    const int v = v0 + lane;
    if (v < q.nvec)
      scaled_or_not(kz, [&](auto ks) {
        for (int k = k0 + warp; k < k1; k += 64) {  // eight loads in flight per lane
          T x[8];
#pragma unroll
          for (int t = 0; t < 8; t++) x[t] = k + 8 * t < k1 ? q.template at<decltype(ks)::value>(X, kz, v, k + 8 * t) : zero<T>();
#pragma unroll
          for (int t = 0; t < 8; t++) m = max(m, mag_key(x[t]));
        }
      });
    pm[warp][lane] = m;
    __syncthreads();
    if (warp == 0 && v < q.nvec) {
#pragma unroll
      for (int w = 1; w < 8; w++) m = max(m, pm[w][lane]);
      put(v, m);
    }
  }
}

// Pass 2, both operands in one launch: one CTA (256 threads) per tile of 32 vectors x 64
// embedded positions (64 k real, 32 k complex; grid x: vectors of A then of B, y: k, z:
// items) over the padded planes.  The tile is staged through shared memory (read along the
// contiguous direction), then its S digits or residues are written with lanes along k, two
// positions (4 bytes) per lane: full 128-byte lines per plane and vector.  Padding vectors
// and k beyond K (the item's, after kdev) up to the last k block read get zeros, so the
// planes need no clearing.
template <typename T, bool RES>
__global__ void __launch_bounds__(256) oz_split_kernel(const SplitPair<T> sp, int K, int Kp, int S, int p, int nb2,
                                                       const int* kdev, const CrtWeights y) {
  constexpr bool CPX = sizeof(T) == 16;
  constexpr int TK = CPX ? 32 : 64;
  __shared__ T tile[TK][33];
  const bool second = (int)blockIdx.x >= sp.n0;
  const SplitOp<T>& q = sp.o[second];
  const int v0 = ((int)blockIdx.x - (second ? sp.n0 : 0)) * 32, k0 = blockIdx.y * TK, z = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (kdev) {
    K = min(K, max(0, kdev[z]));
    if (k0 >= (K + TK - 1) / TK * TK) return;  // k blocks the product kernel does not read
  }
  const T* X = q.X + item_off(z, q.sX, q.sX2, nb2);
  const double* kz = q.ksc ? q.ksc + z * q.sks : nullptr;
  const int* ex = q.ex + z * q.sE;
  __nv_bfloat16* D = q.D + z * q.sD;
  scaled_or_not(kz, [&](auto ks) {
    if (q.contig()) {  // lanes along k
#pragma unroll
      for (int w = 0; w < 4; w++) {
        const int vv = warp + 8 * w, v = v0 + vv;
#pragma unroll
        for (int t = 0; t < TK; t += 32) {
          const int k = k0 + t + lane;
          tile[t + lane][vv] = (v < q.nvec && k < K) ? q.template at<decltype(ks)::value>(X, kz, v, k) : zero<T>();
        }
      }
    } else {  // lanes along the vectors
#pragma unroll
      for (int w = 0; w < TK / 8; w++) {
        const int kk = warp + 8 * w, k = k0 + kk, v = v0 + lane;
        tile[kk][lane] = (k < K && v < q.nvec) ? q.template at<decltype(ks)::value>(X, kz, v, k) : zero<T>();
      }
    }
  });
  __syncthreads();
#pragma unroll 1
  for (int vv = warp; vv < 32; vv += 8) {
    const int v = v0 + vv;
    if (v >= q.nvp) break;
    const T* t = &tile[0][vv];
    emit_pair<T, RES>(q, D, v, k0, lane, CPX ? t[33 * lane] : t[66 * lane], CPX ? zero<T>() : t[66 * lane + 33],
                      v < q.nvec ? ex[v] : 0, Kp, S, p, y);
  }
}

// Both passes in one launch where 8 vectors fit in shared memory (padded K' up to kFusedK):
// a warp per vector finds its scale code and writes its planes, so the operands are read
// once and thin products (the panel updates) save two of five launches.
static constexpr int kFusedK = 1024;
template <typename T>
static constexpr int fused_ld(int kpl) { return (kpl + 15) / 16 * 16 + 4; }  // 8 vectors x 4 k on distinct banks
template <typename T, bool RES>
__global__ void __launch_bounds__(256) oz_fused_kernel(const SplitPair<T> sp, int K, int Kp, int S, int p, int nb2,
                                                       const int* kdev, const CrtWeights y, int ldk) {
  constexpr bool CPX = sizeof(T) == 16;
  extern __shared__ __align__(16) unsigned char fused_raw[];
  T* rows = reinterpret_cast<T*>(fused_raw);  // [8][ldk]
  const bool second = (int)blockIdx.x >= sp.n0;
  const SplitOp<T>& q = sp.o[second];
  const int v0 = ((int)blockIdx.x - (second ? sp.n0 : 0)) * 8, z = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, kpl = CPX ? Kp / 2 : Kp;
  if (kdev) K = min(K, max(0, kdev[z]));
  const T* X = q.X + item_off(z, q.sX, q.sX2, nb2);
  const double* kz = q.ksc ? q.ksc + z * q.sks : nullptr;
  scaled_or_not(kz, [&](auto ks) {
    if (q.contig()) {
      const int v = v0 + warp;
#pragma unroll 4
      for (int k = lane; k < kpl; k += 32)
        rows[warp * ldk + k] = (v < q.nvec && k < K) ? q.template at<decltype(ks)::value>(X, kz, v, k) : zero<T>();
    } else {
      const int v = v0 + (tid & 7);
#pragma unroll 4
      for (int k = tid >> 3; k < kpl; k += 32)
        rows[(tid & 7) * ldk + k] = (v < q.nvec && k < K) ? q.template at<decltype(ks)::value>(X, kz, v, k) : zero<T>();
    }
  });
  __syncthreads();
  const int v = v0 + warp;
  if (v >= q.nvp) return;
  const T* row = rows + warp * ldk;
  uint32_t m = 0;
  for (int k = lane; k < kpl; k += 32) m = max(m, mag_key(row[k]));
  m = __reduce_max_sync(0xffffffffu, m);
  const int code = exp_code(m);
  if (lane == 0 && v < q.nvec) q.ex[z * q.sE + v] = code;
  __nv_bfloat16* D = q.D + z * q.sD;
#pragma unroll 1
  for (int k0 = 0; k0 < kpl; k0 += CPX ? 32 : 64)
    emit_pair<T, RES>(q, D, v, k0, lane, CPX ? row[k0 + lane] : row[k0 + 2 * lane],
                      CPX ? zero<T>() : row[k0 + 2 * lane + 1], code, Kp, S, p, y);
}

// ------------------------------------------------------------------ product kernel

static constexpr int OZ_BM = 128, OZ_BN = 128;  // output tile of the product kernel

struct OzArgs {
  const __nv_bfloat16* Ad;  // [S][Mp][Kp]
  const __nv_bfloat16* Bd;  // [S][Np][Kp]   (embedded columns, K-major)
  const int* ea;            // scale codes of the M rows
  const int* eb;            // scale codes of the logical N columns
  void* C;
  int ldc;
  int M, N;                 // logical output (N complex columns when cplx)
  int Mp, Np, Kp;           // padded digit shapes (Np = embedded columns)
  int S;
  int cplx, lower;
  double alpha, beta;
  long long sAd, sBd;       // slice strides (elements)
  long long zAd, zBd, zEa, zEb, zC;  // batch item strides of the digits, exponents and C
  long long zC2;            // two-level batch (nb2 > 0): C of item z at (z / nb2) zC + (z % nb2) zC2
  int nb2;
  const int* kdev;          // optional per-item K read on the device (logical, <= K)
  long long wait;           // bound of every mbarrier wait, in SM clock cycles
  long long skip_copy;      // test hook: the producer leaves out this copy (-1 = none)
};

// ------------------------------------------------------------------ tcgen05 product kernel
//
// The same digit products on the 5th-generation tensor cores.  One CTA owns a 128 x 128
// output tile (of the embedded product) and walks the units in level order: a unit is a
// level L = s + t and a K chunk short enough that the sum over all pairs of the level,
// (L - 1) 63^2 chunk, stays within 2^24, so one FP32 accumulation holds every pair of the
// level exactly and a single drain (scale 2^{-6L}) serves them all.  Warp 0 streams
// 128 x 64 digit tiles of A slice s and B slice t into a
// ring of shared-memory stages with TMA (128-byte swizzle), one thread of warp 1 issues
// tcgen05.mma (M = N = 128, K = 16) into one of two FP32 accumulators in tensor memory,
// and eight epilogue warps read the finished accumulator with tcgen05.ld, scale it by
// 2^{-6L} and add it into FP64 registers (thread = one tile row x 64 columns), while
// the tensor cores fill the other accumulator.  Every wait is bounded: past the limit
// the CTA raises an abort flag and a timeout status, lets its copies and products land,
// frees its tensor memory and exits.
namespace tcg {
// k blocks per unit of level L: (L - 1) pairs, digit products up to 63^2.
__device__ __forceinline__ int level_blocks(int L) {
  const int cb = (int)((1u << 24) / ((unsigned)(L - 1) * 3969u * (unsigned)BK));
  return min(cb, OZ_CHUNK / BK);
}

// x 2^-s as a double, for x an integer-valued float (the exact unit sums): built from the
// float's bits with integer operations (sign, exponent shifted by 896 - s, mantissa moved
// up by 29 bits), so the drain spends one FP64 add per element and no FP64 conversion.
__device__ __forceinline__ double exact_scaled(uint32_t b, uint32_t s) {
  const uint32_t e = (b >> 23) & 0xffu;
  const uint32_t hi = (b & 0x80000000u) | ((e + 896u - s) << 20) | ((b & 0x7fffffu) >> 3);
  const uint32_t lo = b << 29;
  return e ? __hiloint2double((int)hi, (int)lo) : 0.0;
}
}  // namespace tcg

__global__ void __launch_bounds__(tcg::THREADS, 1)
    oz_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, OzArgs a,
                 DevStatus* status) {
  using namespace tcg;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2], done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  unsigned char* ring = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // grouped tile order: consecutive CTAs walk 8 row tiles of one column tile, then the next
  // column tile, so the CTAs resident together share both operands' digit tiles in L2
  int m0, n0;
  {
    constexpr int G = 8;
    const int ntn = gridDim.x, ntm = gridDim.y;
    const int bid = blockIdx.y * ntn + blockIdx.x, per = G * ntn;
    const int fm = (bid / per) * G, gs = min(ntm - fm, G), r = bid % per;
    m0 = (fm + r % gs) * BM;
    n0 = (r / gs) * BN;
  }
  const int z = blockIdx.z;
  const int ncol0 = a.cplx ? n0 / 2 : n0;
  if (a.lower && m0 + BM - 1 < ncol0) return;  // whole tile above the diagonal (uniform)

  const int S = a.S;
  int kblocks = a.Kp / BK;
  if (a.kdev) {
    const int ke = min(a.Kp, max(0, a.kdev[z]) * (a.cplx ? 2 : 1));
    kblocks = (ke + BK - 1) / BK;
  }

  if (tid == 0) {
    for (int i = 0; i < STAGES; i++) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int b = 0; b < 2; b++) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], EPI_WARPS);
    }
    mbar_init(&done, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  volatile int* abort = &abort_flag;

  double acc[64];
#pragma unroll
  for (int i = 0; i < 64; i++) acc[i] = 0.0;

  if (warp == 0) {
    if (lane == 0) {
      // producer: digit tiles of A slice s and B slice t, k block kb, in unit order
      long long q = 0;
      for (int L = 2; L <= S + 1 && !*abort; L++) {
        const int cb = level_blocks(L);
        for (int c0 = 0; c0 < kblocks && !*abort; c0 += cb) {
          const int c1 = min(kblocks, c0 + cb);
          for (int si = 1; si < L && !*abort; si++) {
            const int ya = (z * S + si - 1) * a.Mp + m0, yb = (z * S + (L - si) - 1) * a.Np + n0;
            for (int kb = c0; kb < c1; kb++, q++) {
              const int stg = (int)(q % STAGES);
              const uint32_t ph = (uint32_t)((q / STAGES) & 1);
              if (!mbar_wait(&empty[stg], ph ^ 1u, abort, a.wait)) break;
              if (q == a.skip_copy) continue;  // test hook: this stage never fills
              unsigned char* sa = ring + (size_t)stg * STAGE_BYTES;
              mbar_expect_tx(&full[stg], STAGE_BYTES);
              tma_load_2d(sa, &mapA, &full[stg], kb * BK, ya);
              tma_load_2d(sa + TILE_BYTES, &mapB, &full[stg], kb * BK, yb);
            }
          }
        }
      }
      // let every issued copy land before the CTA can leave
      for (long long r = (q > STAGES ? q - STAGES : 0); r < q; r++)
        if (r != a.skip_copy) mbar_drain(&full[r % STAGES], (uint32_t)((r / STAGES) & 1), a.wait);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // MMA issuer
      long long q = 0;
      int u = 0;
      bool ok = true;
      for (int L = 2; L <= S + 1 && ok; L++) {
        const int cb = level_blocks(L);
        for (int c0 = 0; c0 < kblocks && ok; c0 += cb, u++) {
          const int c1 = min(kblocks, c0 + cb);
          const int b = u & 1;
          const uint32_t uph = (uint32_t)((u >> 1) & 1);
          if (!mbar_wait(&tempty[b], uph ^ 1u, abort, a.wait)) {
            ok = false;
            break;
          }
          tc_fence_after();
          uint32_t accum = 0;
          for (int si = 1; si < L && ok; si++) {
            for (int kb = c0; kb < c1; kb++, q++) {
              const int stg = (int)(q % STAGES);
              const uint32_t ph = (uint32_t)((q / STAGES) & 1);
              if (!mbar_wait(&full[stg], ph, abort, a.wait)) {
                ok = false;
                break;
              }
              tc_fence_after();
              const uint32_t sa = smem_u32(ring + (size_t)stg * STAGE_BYTES);
              const uint64_t da = sw128_desc(sa), db = sw128_desc(sa + TILE_BYTES);
#pragma unroll
              for (int kk = 0; kk < BK / 16; kk++) {
                umma(tmem + (uint32_t)(b * BN), da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), accum);
                accum = 1u;
              }
              umma_commit(&empty[stg]);
            }
          }
          if (!ok) break;
          umma_commit(&tfull[b]);
        }
      }
      // all issued products complete before tensor memory is released
      umma_commit(&done);
      mbar_drain(&done, 0, a.wait);
    }
  } else {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31, column half (w - 2) / 4
    const int lq = warp & 3, ch = (warp - 2) >> 2;
    int u = 0;
    bool ok = true;
    for (int L = 2; L <= S + 1 && ok; L++) {
      const int cb = level_blocks(L);
      const uint32_t sh = (uint32_t)(OZ_BITS * L);
      for (int c0 = 0; c0 < kblocks; c0 += cb, u++) {
        const int b = u & 1;
        const uint32_t uph = (uint32_t)((u >> 1) & 1);
        if (!mbar_wait(&tfull[b], uph, abort, a.wait)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t taddr = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(b * BN + ch * 64);
        uint32_t v[32];
        tmem_ld32(taddr, v);
#pragma unroll
        for (int i = 0; i < 32; i++) acc[i] += exact_scaled(v[i], sh);
        tmem_ld32(taddr + 32, v);
#pragma unroll
        for (int i = 0; i < 32; i++) acc[32 + i] += exact_scaled(v[i], sh);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[b]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS));
  }
  if (*abort) {
    if (tid == 0) set_status(status, ST_ETIMEOUT, -2);
    return;
  }
  if (warp < 2) return;
  // C = alpha 2^{e_i + f_j} acc + beta C for this thread's row and 64 embedded columns
  const int lq = warp & 3, ch = (warp - 2) >> 2;
  const int i = m0 + lq * 32 + lane;
  if (i >= a.M) return;
  const long long zz = z;
  const int* ea = a.ea + zz * a.zEa;
  const int* eb = a.eb + zz * a.zEb;
  if (a.cplx) {
    zc* C = static_cast<zc*>(a.C) + item_off(z, a.zC, a.zC2, a.nb2);
    const int j0 = n0 / 2 + ch * 32;
#pragma unroll
    for (int jj = 0; jj < 32; jj++) {
      const int j = j0 + jj;
      if (j >= a.N || (a.lower && j > i)) continue;
      const bool bad = ea[i] == kExpNan || eb[j] == kExpNan;
      const int ee = exp_of(ea[i]) + exp_of(eb[j]);
      zc v{ldexp(bad ? nan("") : acc[2 * jj], ee) * a.alpha, ldexp(bad ? nan("") : acc[2 * jj + 1], ee) * a.alpha};
      zc* cp = C + (size_t)i * a.ldc + j;
      if (a.beta != 0.0) v = v + a.beta * (*cp);
      *cp = v;
    }
  } else {
    double* C = static_cast<double*>(a.C) + item_off(z, a.zC, a.zC2, a.nb2);
    const int j0 = n0 + ch * 64;
#pragma unroll
    for (int jj = 0; jj < 64; jj++) {
      const int j = j0 + jj;
      if (j >= a.N || (a.lower && j > i)) continue;
      const bool bad = ea[i] == kExpNan || eb[j] == kExpNan;
      double v = ldexp(bad ? nan("") : acc[jj], exp_of(ea[i]) + exp_of(eb[j])) * a.alpha;
      double* cp = C + (size_t)i * a.ldc + j;
      if (a.beta != 0.0) v += a.beta * (*cp);
      *cp = v;
    }
  }
}

// ------------------------------------------------------------------ residue products
//
// The modular form of the split product (the integer-modular scheme of Ozaki, Uchino and
// Imamura, here on the bf16 tensor cores).  Row i of op(A) is scaled by 2^{p - e_i} and
// truncated to integers A'_ik (|A'_ik| < 2^p), column j of op(B) the same, and the integer
// product X = A'B' is recovered from its residues modulo n pairwise coprime m_l by the
// Chinese remainder theorem, since |X| < Kp 2^{2p} <= M / 2 with M = m_1 ... m_n.  For each
// modulus the kernel multiplies the residue planes of A' and B' over K: symmetric residues
// are bf16-exact integers of magnitude <= 128, so a k chunk of 1024 sums exactly in the
// FP32 accumulator (<= 2^24).  Eight epilogue warps fold each chunk into a residue kept
// in FP32 registers (x - m round(x / m), exact on integers) while the tensor cores fill the
// other accumulator, and write the symmetric residue of every element as one byte when the
// modulus ends.  B' enters as the residues of y_l B', y_l = (M / m_l)^-1 mod m_l, so what is
// stored is already the weighted residue of the reconstruction.  One product per modulus: 16
// moduli keep p = 55 bits for K up to 16384, where nine 6-bit digits keep 54 bits with 45
// digit-pair products.  crt_recon_kernel rebuilds X and scales it back by 2^{e_i + f_j - 2p}.
//
// Measured (832 x 832 x 64 real, one product, CUDA events): 95 us with weights and range
// corrections in the epilogue, all moduli of a tile in one CTA and 16 elements per
// reconstruction thread; 52 us with the forms below (13 us product kernel, 19 us
// reconstruction, 6 us splitting).  Complex 4992 x 4992 x 512: 3.17 -> 2.00 ms.
constexpr int CRT_CHUNK_BLOCKS = 16;  // k blocks per exact chunk: 16 * 64 * 128^2 = 2^24

struct CrtArgs {
  const __nv_bfloat16* Ad;  // [count][n][Mp][Kp] residue planes of A'
  const __nv_bfloat16* Bd;  // [count][n][Np][Kp] residue planes of B' (embedded columns, K-major)
  uint8_t* R;               // [count][n][Mp][Np] residues of X
  int Mp, Np, Kp, n, cplx, lower;
  int ng;                   // CTAs per tile: CTA g takes moduli [g n / ng, (g + 1) n / ng)
  long long zR;             // item stride of R (bytes)
  const int* kdev;          // optional per-item K read on the device (logical, <= K)
  long long wait;           // bound of every mbarrier wait, in SM clock cycles
  long long skip_copy;      // test hook: the producer leaves out this copy (-1 = none)
};

// Tile of the residue kernel: 128 x 256 outputs per CTA (the B operand tile twice as wide as
// the digit-pair kernel's, so each A tile fetched into shared memory serves twice the MMA
// work), four stages of 48 KB, and two 256-column FP32 accumulators filling the 512 columns
// of tensor memory.
namespace crtc {
constexpr int BN = 256;
constexpr int STAGES = 4;
constexpr int B_BYTES = BN * tcg::BK * 2;
constexpr int STAGE_BYTES = tcg::TILE_BYTES + B_BYTES;
constexpr int TMEM_COLS = 2 * BN;
constexpr int OUT_BYTES = 32 * 128;  // an epilogue warp's 32 rows x 128 residues
constexpr int SMEM = STAGES * STAGE_BYTES + tcg::EPI_WARPS * OUT_BYTES + 1024;
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                           ((uint32_t)(tcg::BM >> 4) << 24);
static_assert(SMEM <= 227 * 1024, "shared memory of the residue kernel");
}  // namespace crtc

// Whether one fold of a chunk sum (|x| <= 2^24) fits the stored byte.  The quotient may miss by
// one next to a half (1 / m is rounded: an error up to 0.004 at |x / m| = 65793), which leaves
// |r| = (m + 1) / 2: 127 at most from modulus 253 down, but 128 for 255, where the byte stands
// for -128, congruent modulo 256 only.  Modulus 256 divides exactly.  A second fold (|x| < 2^14)
// has the exact quotient.
__host__ __device__ constexpr bool crt_one_fold(int l) { return crt_mod(l) == 256u || crt_mod(l) <= 253u; }

// Four symmetric residues as bytes r + 128 (r = 128, modulus 256 only, wraps to -128): adding
// 1.5 * 2^23 leaves r in the low bits of the float, so no conversion instruction is needed.
__device__ __forceinline__ uint32_t crt_bytes(float r0, float r1, float r2, float r3) {
  const uint32_t b0 = __float_as_uint(__fadd_rn(r0, 12582912.0f)), b1 = __float_as_uint(__fadd_rn(r1, 12582912.0f));
  const uint32_t b2 = __float_as_uint(__fadd_rn(r2, 12582912.0f)), b3 = __float_as_uint(__fadd_rn(r3, 12582912.0f));
  return __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410) ^ 0x80808080u;
}

__global__ void __launch_bounds__(tcg::THREADS, 1)
    crt_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, CrtArgs a,
                  DevStatus* status) {
  using namespace tcg;
  using crtc::BN;
  using crtc::STAGE_BYTES;
  using crtc::STAGES;
  using crtc::TMEM_COLS;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2], done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  unsigned char* ring = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int m0, n0;  // grouped tile order, as in oz_tc_kernel
  {
    constexpr int G = 8;
    const int ntn = gridDim.x, ntm = gridDim.y;
    const int bid = blockIdx.y * ntn + blockIdx.x, per = G * ntn;
    const int fm = (bid / per) * G, gs = min(ntm - fm, G), r = bid % per;
    m0 = (fm + r % gs) * BM;
    n0 = (r / gs) * BN;
  }
  const int z = blockIdx.z / a.ng, grp = blockIdx.z % a.ng;
  const int ncol0 = a.cplx ? n0 / 2 : n0;
  if (a.lower && m0 + BM - 1 < ncol0) return;  // whole tile above the diagonal (uniform)

  const int n = a.n, l0 = grp * n / a.ng, l1 = (grp + 1) * n / a.ng;
  int kblocks = a.Kp / BK;
  if (a.kdev) {
    const int ke = min(a.Kp, max(0, a.kdev[z]) * (a.cplx ? 2 : 1));
    kblocks = (ke + BK - 1) / BK;
  }
  const int nchunk = (kblocks + CRT_CHUNK_BLOCKS - 1) / CRT_CHUNK_BLOCKS;

  if (tid == 0) {
    for (int i = 0; i < STAGES; i++) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int b = 0; b < 2; b++) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], EPI_WARPS);
    }
    mbar_init(&done, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  volatile int* abort = &abort_flag;

  if (warp == 0) {
    if (lane == 0) {
      // producer: residue tiles of A' and B' for modulus l, k block kb
      long long q = 0;
      for (int l = l0; l < l1 && !*abort; l++) {
        const int ya = (z * n + l) * a.Mp + m0, yb = (z * n + l) * a.Np + n0;
        for (int kb = 0; kb < kblocks; kb++, q++) {
          const int stg = (int)(q % STAGES);
          const uint32_t ph = (uint32_t)((q / STAGES) & 1);
          if (!mbar_wait(&empty[stg], ph ^ 1u, abort, a.wait)) break;
          if (q == a.skip_copy) continue;  // test hook: this stage never fills
          unsigned char* sa = ring + (size_t)stg * STAGE_BYTES;
          mbar_expect_tx(&full[stg], STAGE_BYTES);
          tma_load_2d(sa, &mapA, &full[stg], kb * BK, ya);
          tma_load_2d(sa + TILE_BYTES, &mapB, &full[stg], kb * BK, yb);
        }
      }
      for (long long r = (q > STAGES ? q - STAGES : 0); r < q; r++)
        if (r != a.skip_copy) mbar_drain(&full[r % STAGES], (uint32_t)((r / STAGES) & 1), a.wait);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // MMA issuer: one accumulator per (modulus, k chunk)
      long long q = 0;
      int u = 0;
      bool ok = true;
      for (int l = l0; l < l1 && ok; l++) {
        for (int c = 0; c < nchunk && ok; c++, u++) {
          const int b = u & 1;
          const uint32_t uph = (uint32_t)((u >> 1) & 1);
          if (!mbar_wait(&tempty[b], uph ^ 1u, abort, a.wait)) {
            ok = false;
            break;
          }
          tc_fence_after();
          uint32_t accum = 0;
          const int kb1 = min(kblocks, (c + 1) * CRT_CHUNK_BLOCKS);
          for (int kb = c * CRT_CHUNK_BLOCKS; kb < kb1; kb++, q++) {
            const int stg = (int)(q % STAGES);
            const uint32_t ph = (uint32_t)((q / STAGES) & 1);
            if (!mbar_wait(&full[stg], ph, abort, a.wait)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t sa = smem_u32(ring + (size_t)stg * STAGE_BYTES);
            const uint64_t da = sw128_desc(sa), db = sw128_desc(sa + TILE_BYTES);
#pragma unroll
            for (int kk = 0; kk < BK / 16; kk++) {
              tcg::umma<crtc::IDESC>(tmem + (uint32_t)(b * BN), da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2),
                                     accum);
              accum = 1u;
            }
            umma_commit(&empty[stg]);
          }
          if (!ok) break;
          umma_commit(&tfull[b]);
        }
      }
      umma_commit(&done);
      mbar_drain(&done, 0, a.wait);
    }
  } else {
    // epilogue: warp w owns TMEM lanes 32 (w % 4) .. +31 (tile rows) and column half
    // (w - 2) / 4 (128 columns)
    const int lq = warp & 3, ch = (warp - 2) >> 2;
    uint4* out = reinterpret_cast<uint4*>(ring + (size_t)STAGES * STAGE_BYTES + (warp - 2) * crtc::OUT_BYTES);
    auto flush = [&](int l) {
      __syncwarp();
      uint8_t* dst = a.R + z * a.zR + ((size_t)l * a.Mp + m0 + lq * 32) * a.Np + n0 + ch * 128;
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int r = 4 * q + (lane >> 3), w = lane & 7;
        __stcs(reinterpret_cast<uint4*>(dst + (size_t)r * a.Np + 16 * w), out[r * 8 + (w ^ (r & 7))]);
      }
      __syncwarp();
    };
    int u = 0;
    bool ok = true;
    for (int l = l0; l < l1 && ok; l++) {
      const float mf = (float)crt_mod(l), inv = __frcp_rn(mf);
      // the thread's row of residues goes to shared memory in 16-byte words (word w of row r at
      // w ^ (r & 7): distinct banks), and from there in full 128-byte lines, 4 rows per warp store
      auto put = [&](int word, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
        out[lane * 8 + (word ^ (lane & 7))] = make_uint4(w0, w1, w2, w3);
      };
      if (nchunk == 1 && crt_one_fold(l)) {  // K' <= 1024: the accumulator folds straight to its bytes
        const int b = u & 1;
        const uint32_t uph = (uint32_t)((u >> 1) & 1);
        u++;
        if (!mbar_wait(&tfull[b], uph, abort, a.wait)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t taddr = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(b * BN + ch * 128);
#pragma unroll
        for (int g = 0; g < 4; g++) {
          uint32_t v[32];
          tmem_ld32(taddr + 32 * g, v);
          if (g == 3) {  // the last read: the accumulator is free before its bytes are formed
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[b]);
          }
          uint32_t w[8];
#pragma unroll
          for (int t = 0; t < 8; t++)
            w[t] = crt_bytes(crt_fold(__uint_as_float(v[4 * t]), mf, inv), crt_fold(__uint_as_float(v[4 * t + 1]), mf, inv),
                             crt_fold(__uint_as_float(v[4 * t + 2]), mf, inv),
                             crt_fold(__uint_as_float(v[4 * t + 3]), mf, inv));
          put(2 * g, w[0], w[1], w[2], w[3]);
          put(2 * g + 1, w[4], w[5], w[6], w[7]);
        }
        flush(l);
        continue;
      }
      float acc[128];
#pragma unroll
      for (int t = 0; t < 128; t++) acc[t] = 0.0f;
      for (int c = 0; c < nchunk; c++, u++) {
        const int b = u & 1;
        const uint32_t uph = (uint32_t)((u >> 1) & 1);
        if (!mbar_wait(&tfull[b], uph, abort, a.wait)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t taddr = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(b * BN + ch * 128);
#pragma unroll
        for (int g = 0; g < 4; g++) {
          uint32_t v[32];
          tmem_ld32(taddr + 32 * g, v);
#pragma unroll
          for (int t = 0; t < 32; t++) acc[32 * g + t] += crt_fold(__uint_as_float(v[t]), mf, inv);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[b]);
      }
      if (!ok) break;
#pragma unroll
      for (int q = 0; q < 8; q++) {
        uint32_t w[4];
#pragma unroll
        for (int t = 0; t < 4; t++) {
          const float* x = acc + 16 * q + 4 * t;
          w[t] = crt_bytes(crt_fold(x[0], mf, inv), crt_fold(x[1], mf, inv), crt_fold(x[2], mf, inv),
                           crt_fold(x[3], mf, inv));
        }
        put(q, w[0], w[1], w[2], w[3]);
      }
      flush(l);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS));
  }
  if (*abort && tid == 0) set_status(status, ST_ETIMEOUT, -2);
}

// Constants of the reconstruction for n moduli: X = sum_l t_l (M / m_l) mod M with the
// weighted symmetric residues t_l = (X y_l) mod m_l that the product kernel stores as bytes
// t_l + 128.  Moduli are taken in groups of three, v_g = sum_l byte_l m_a m_b (the other two
// of the group; below 2^26), and S = E + sum_g v_g M / (m_a m_b m_c) with E = -128 sum_l
// M / m_l mod M, so that S is non-negative, congruent to X and below 32 M.
constexpr int CRT_GROUPS = 6;
struct CrtRecon {
  uint32_t cf[CRT_MAXMOD];         // product of the other moduli of the group (0 from n up)
  uint32_t Ng[CRT_GROUPS][4];      // M / (product of the group), 32-bit limbs, least first
  uint32_t E[4];
  unsigned long long Mv[2];        // M
  float inv_mf;                    // 2^{32 b} / M
  int b;                           // limb at which the quotient estimate starts: max(0, top limb of M - 1)
  int n;
};

// 128-bit magnitude (w3 the top word) times 2^e to the nearest double (ties to even), from its
// bits: h the 64 bits from the leading one, l what is left of them, the 53-bit mantissa's
// leading one and a rounding carry added into the exponent (through ldexp only where the
// result leaves the normal range).  Most values fill the top word.
__device__ __forceinline__ double u128_scaled(uint32_t w3, uint32_t w2, uint32_t w1, uint32_t w0, bool neg, int e) {
  uint32_t h1, h0, l = 0;
  int lz;
  if (w3) {
    lz = __clz((int)w3);
    h1 = __funnelshift_l(w2, w3, lz);
    h0 = __funnelshift_l(w1, w2, lz);
    l = __funnelshift_l(w0, w1, lz) | (w0 << lz);
  } else if (w2) {
    lz = __clz((int)w2);
    h1 = __funnelshift_l(w1, w2, lz);
    h0 = __funnelshift_l(w0, w1, lz);
    l = w0 << lz;
    lz += 32;
  } else if (w1) {
    lz = __clz((int)w1);
    h1 = __funnelshift_l(w0, w1, lz);
    h0 = w0 << lz;
    lz += 64;
  } else {
    if (!w0) return 0.0;
    lz = __clz((int)w0);
    h1 = w0 << lz;
    h0 = 0;
    lz += 96;
  }
  const uint32_t rest = ((h0 & 0x7ffu) << 1) | (l != 0u), odd = (h0 >> 11) & 1u;
  const unsigned long long mant = (((unsigned long long)(h1 >> 11) << 32) | __funnelshift_r(h0, h1, 11)) +
                                  (rest + odd > 0x800u ? 1ull : 0ull);
  const int be = 127 - lz + 1022;  // the exponent field below the leading one of mant
  const unsigned long long sgn = neg ? 1ull << 63 : 0ull;
  if ((unsigned)(be + e) < 2046u) return __longlong_as_double((long long)(sgn | (((unsigned long long)(be + e) << 52) + mant)));
  return ldexp(__longlong_as_double((long long)(sgn | (((unsigned long long)be << 52) + mant))), e);
}

// The signed integer X of the bytes of element el, as a double times 2^e.  S is
// accumulated in four 64-bit limbs without carries (v_g limb < 2^58, six of them); with |X|
// <= (1/2 - 2^-10) M the quotient round(S / M) is exact from a single-precision estimate
// (S / M < 32, relative error below 2^-20), and X = S - q M in 128-bit two's complement from
// the table of q M.  About 150 integer operations per element: bound by the integer pipe.
__device__ __forceinline__ double crt_value(const uint32_t (&w)[CRT_MAXMOD][2], int el, const CrtRecon& cr,
                                            const ulonglong2* qM, int e) {
  unsigned long long c0 = cr.E[0], c1 = cr.E[1], c2 = cr.E[2], c3 = cr.E[3];
#pragma unroll
  for (int g = 0; g < CRT_GROUPS; g++) {
    uint32_t v = 0;
#pragma unroll
    for (int l = 3 * g; l < 3 * g + 3 && l < CRT_MAXMOD; l++)
      v += ((w[l][el >> 2] >> (8 * (el & 3))) & 0xffu) * cr.cf[l];
    c0 += (unsigned long long)v * cr.Ng[g][0];
    c1 += (unsigned long long)v * cr.Ng[g][1];
    c2 += (unsigned long long)v * cr.Ng[g][2];
    c3 += (unsigned long long)v * cr.Ng[g][3];
  }
  c1 += c0 >> 32;
  c2 += c1 >> 32;
  c3 += c2 >> 32;
  const uint32_t s0 = (uint32_t)c0, s1 = (uint32_t)c1, s2 = (uint32_t)c2, s3 = (uint32_t)c3;
  const uint32_t s4 = (uint32_t)(c3 >> 32);
  const uint32_t a2 = cr.b == 0 ? s2 : cr.b == 1 ? s3 : s4;
  const uint32_t a1 = cr.b == 0 ? s1 : cr.b == 1 ? s2 : s3;
  const uint32_t a0 = cr.b == 0 ? s0 : cr.b == 1 ? s1 : s2;
  const float sf = __fmaf_rn((float)a2, 18446744073709551616.0f, __fmaf_rn((float)a1, 4294967296.0f, (float)a0));
  const uint32_t q = __float_as_uint(__fmaf_rn(sf, cr.inv_mf, 12582912.0f)) & 31u;  // nearest integer
  const ulonglong2 m = qM[q];
  unsigned long long lo = ((unsigned long long)s1 << 32) | s0, hi = ((unsigned long long)s3 << 32) | s2;
  hi -= m.y + (lo < m.x ? 1ull : 0ull);
  lo -= m.x;
  const bool neg = (hi >> 63) != 0ull;
  if (neg) {
    lo = 0ull - lo;
    hi = ~hi + (lo == 0ull ? 1ull : 0ull);
  }
  return u128_scaled((uint32_t)(hi >> 32), (uint32_t)hi, (uint32_t)(lo >> 32), (uint32_t)lo, neg, e);
}

// C = alpha 2^{e_i + f_j - 2p} X + beta C for the logical outputs (lower: j <= i only).
// A thread takes 8 consecutive embedded columns of a row: one 8-byte load per modulus (the
// residue planes are Np bytes per row, Np a multiple of 256), then the 8 values (4 complex).
// The CTA's 128 such runs are numbered row by row over the ncg runs per row, so that narrow
// outputs fill the CTAs too, and the values go through shared memory so that C is read and
// written with consecutive lanes on consecutive elements.
template <typename T>
__global__ void __launch_bounds__(128) crt_recon_kernel(const uint8_t* R, long long zR, int Mp, int Np, int M, int N,
                                                        int ncg, const int* ea, const int* eb, long long zEa,
                                                        long long zEb, int sc, const CrtRecon cr, T* C, int ldc,
                                                        long long zC, long long zC2, int nb2, double alpha,
                                                        double beta, int lower) {
  constexpr bool CPX = sizeof(T) == 16;
  constexpr int PER = CPX ? 4 : 8;  // logical columns per thread
  __shared__ T val[128][PER + 1];
  __shared__ ulonglong2 qM[32];
  __shared__ int srow[128], scol[128];  // first column, N + PER where the thread has nothing
  const int z = blockIdx.z, tid = threadIdx.x;
  const long long plane = (long long)Mp * Np, t0 = (long long)blockIdx.x * 128 + tid;
  const int i = (int)(t0 / ncg), j0 = (int)(t0 % ncg) * PER;
  const bool ok = i < M && !(lower && j0 > i);
  srow[tid] = i;
  scol[tid] = ok ? j0 : N + PER;
  if (tid < 32) {  // q M in 128 bits
    const unsigned __int128 v = (((unsigned __int128)cr.Mv[1] << 64) | cr.Mv[0]) * (unsigned)tid;
    qM[tid] = make_ulonglong2((unsigned long long)v, (unsigned long long)(v >> 64));
  }
  __syncthreads();
  if (ok) {
    const uint8_t* Rz = R + z * zR + (size_t)i * Np + (CPX ? 2 * j0 : j0);
    uint32_t w[CRT_MAXMOD][2];
#pragma unroll
    for (int l = 0; l < CRT_MAXMOD; l++) {
      uint2 v = make_uint2(0u, 0u);
      if (l < cr.n) v = __ldcs(reinterpret_cast<const uint2*>(Rz + l * plane));
      w[l][0] = v.x;
      w[l][1] = v.y;
    }
    const int ci = ea[z * zEa + i], ei = exp_of(ci) + sc;
#pragma unroll
    for (int q = 0; q < PER; q++) {
      const int j = j0 + q;
      if (j >= N) break;
      const int cj = eb[z * zEb + j], e = ei + exp_of(cj);
      if (ci == kExpNan || cj == kExpNan) {
        if constexpr (CPX) val[tid][q] = zc{nan(""), nan("")};
        else val[tid][q] = nan("");
      } else if constexpr (CPX) {
        val[tid][q] = zc{crt_value(w, 2 * q, cr, qM, e), crt_value(w, 2 * q + 1, cr, qM, e)};
      } else {
        val[tid][q] = crt_value(w, q, cr, qM, e);
      }
    }
  }
  __syncthreads();
  T* Cz = C + item_off(z, zC, zC2, nb2);
#pragma unroll
  for (int q = 0; q < PER; q++) {
    const int idx = q * 128 + tid, o = idx / PER, r = srow[o], j = scol[o] + idx % PER;
    if (j >= N || (lower && j > r)) continue;
    T* cp = Cz + (size_t)r * ldc + j;
    T v = val[o][idx % PER];
    if (alpha == -1.0) v = -v;
    else if (alpha != 1.0) v = alpha * v;
    if (beta == 1.0) v = v + *cp;
    else if (beta != 0.0) v = v + beta * (*cp);
    *cp = v;
  }
}

// ---- tensor maps (driver entry point looked up once through the runtime)
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static std::once_flag once;
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    cudaGetLastError();
  });
  return fn;
}

// 2-D bf16 map over rows x Kp (row stride Kp), box 64 (k) x 128 (rows), 128-byte swizzle.
static bool digit_map(CUtensorMap* m, const void* base, long long rows, int Kp, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)Kp, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)Kp * 2};
  cuuint32_t box[2] = {(cuuint32_t)tcg::BK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ------------------------------------------------------------------ host

static int round_up(int x, int m) { return (x + m - 1) / m * m; }

// Digit planes of an item: the same padded shapes ozaki_gemm uses (K = 0 still takes one
// 64-wide k block of zero digits, so that the product kernel computes C = beta C).
static int padded_k(int K, bool cplx) {
  const int Ke = cplx ? 2 * K : K;
  return round_up(Ke > 0 ? Ke : 1, OZ_KSTEP);
}

// Residue plan for padded length Kp and at least `bits` bits per operand: moduli n whose
// product M satisfies 2 Kp 2^{2p} <= M with p >= bits (p as large as M allows, at most 62),
// and the reconstruction constants.  FP64-accurate products (bits >= 54) take all 16 moduli:
// p = 59 at Kp = 64 and 57 at 1024, against 54 with the 15 that would do up to Kp = 256, so
// that thin products, which would otherwise run on the FP64 kernel, keep several bits below
// the FP64 rounding of their largest terms for 1/15 more work.  Fewer bits (the mixed
// path's back-transform): the fewest moduli.  False if 16 moduli fall short.
struct CrtPlan {
  int n, p;
  CrtRecon cr;
  CrtWeights wt;
};
static bool crt_plan(int Kp, int bits, CrtPlan* pl) {
  typedef unsigned __int128 u128;
  u128 M = 1;
  for (int n = 1; n <= CRT_MAXMOD; n++) {
    M *= crt_mod(n - 1);
    // 2^{2p} <= room, with the 2^-9 margin that makes the reconstruction's quotient exact
    const u128 room = (M - (M >> 9)) / ((u128)2 * (u128)Kp);
    int lg = -1;
    for (u128 t = room; t; t >>= 1) lg++;
    const int p = lg < 0 ? -1 : std::min(lg / 2, 62);
    if (p < bits || (bits >= 54 && n < CRT_MAXMOD)) continue;
    pl->n = n;
    pl->p = p;
    CrtRecon& c = pl->cr;
    c = CrtRecon{};
    pl->wt = CrtWeights{};
    c.n = n;
    const int top = (int)(M >> 96) ? 3 : (int)(M >> 64) ? 2 : (M >> 32) ? 1 : 0;
    c.Mv[0] = (unsigned long long)M;
    c.Mv[1] = (unsigned long long)(M >> 64);
    c.b = std::max(0, top - 1);
    c.inv_mf = (float)(std::ldexp(1.0, 32 * c.b) / (double)M);
    u128 off = 0;  // 128 sum_l M / m_l mod M
    for (int l = 0; l < n; l++) {
      const uint32_t m = crt_mod(l);
      const u128 Nl = M / m;
      for (int t = 0; t < 128; t++) off = (off + Nl) % M;
      const uint32_t r = (uint32_t)(Nl % m);
      uint32_t y = 1;
      while ((r * y) % m != 1u) y++;  // r is coprime to m
      pl->wt.y[l] = 2 * y > m ? (float)y - (float)m : (float)y;
    }
    const u128 E = off ? M - off : 0;
    for (int t = 0; t < 4; t++) c.E[t] = (uint32_t)(E >> (32 * t));
    for (int g = 0; g < CRT_GROUPS && 3 * g < n; g++) {
      const int e = std::min(n, 3 * g + 3);
      uint32_t P = 1;
      for (int l = 3 * g; l < e; l++) P *= crt_mod(l);
      for (int l = 3 * g; l < e; l++) c.cf[l] = P / crt_mod(l);
      const u128 Ng = M / P;
      for (int t = 0; t < 4; t++) c.Ng[g][t] = (uint32_t)(Ng >> (32 * t));
    }
    return true;
  }
  return false;
}

// S > 0: S digits of 6 bits (digit-pair products); S < 0: residues carrying at least 6|S|
// bits (digit pairs again when 16 moduli cannot).
static bool residue_form(int S, int Kp, CrtPlan* pl) { return S < 0 && crt_plan(Kp, OZ_BITS * -S, pl); }

// Embedded output columns padded to the product kernel's tile width.
static int padded_n(int N, bool cplx, bool res) { return round_up(cplx ? 2 * N : N, res ? crtc::BN : OZ_BN); }

size_t ozaki_workspace_bytes(int M, int N, int K, bool cplx, int S) {
  const int Kp = padded_k(K, cplx);
  CrtPlan pl;
  const bool res = residue_form(S, Kp, &pl);
  const int Mp = round_up(M, OZ_BM), Np = padded_n(N, cplx, res);
  size_t b;
  if (res)
    b = (size_t)pl.n * (((size_t)Mp + Np) * Kp * 2 + (size_t)Mp * Np);
  else
    b = (size_t)std::abs(S) * ((size_t)Mp + Np) * Kp * 2;
  b += sizeof(int) * ((size_t)Mp + Np) + 1024;
  return (b + 255) & ~size_t(255);
}

// count items, item z at A + z sA, B + z sB, C + z sC.  work holds, for all items, the A
// planes [count][P][Mp][Kp], then the B planes [count][P][Np][Kp] (P = S digits or n
// residues), then (residues) the residues of the product [count][n][Mp][Np] as bytes, then
// the exponents [count][Mp] and [count][Np] (within count * ozaki_workspace_bytes).
template <typename T>
bool ozaki_gemm(int opA, int opB, int M, int N, int K, double alpha, const T* A, int lda, long long sA, const T* B,
                int ldb, long long sB, double beta, T* C, int ldc, long long sC, int count, int lower, int S,
                void* work, DevStatus* status, cudaStream_t s, const double* kscale, long long sks,
                const int* kdev, long long wait_cycles, long long skip_copy, long long sA2, long long sB2,
                long long sC2, int nb2) {
  if (M <= 0 || N <= 0 || count <= 0) return true;
  const bool cplx = sizeof(T) == 16;
  const int Kp = padded_k(K, cplx);
  CrtPlan pl;
  const bool res = residue_form(S, Kp, &pl);
  const int Mp = round_up(M, OZ_BM), Np = padded_n(N, cplx, res);
  const int P = res ? pl.n : std::abs(S);  // planes per operand
  const long long zA = (long long)P * Mp * Kp, zB = (long long)P * Np * Kp;
  const long long zR = res ? (long long)P * Mp * Np : 0;
  __nv_bfloat16* Ad = static_cast<__nv_bfloat16*>(work);
  __nv_bfloat16* Bd = Ad + zA * count;
  uint8_t* R = reinterpret_cast<uint8_t*>(Bd + zB * count);
  int* ea = reinterpret_cast<int*>(R + zR * count);
  int* eb = ea + (size_t)Mp * count;
  SplitPair<T> sp;
  sp.o[0] = SplitOp<T>{A, lda, 0, opA, M, Mp, sA, sA2, ea, Mp, kscale, sks, Ad, (long long)Mp * Kp, zA};
  sp.o[1] = SplitOp<T>{B, ldb, 1, opB, N, cplx ? Np / 2 : Np, sB, sB2, eb, Np, nullptr, 0, Bd, (long long)Np * Kp, zB};
  const int bits = res ? pl.p : 0;
  if (Kp <= kFusedK) {
    sp.n0 = Mp / 8;
    const int ldk = fused_ld<T>(cplx ? Kp / 2 : Kp), sm = 8 * ldk * (int)sizeof(T);
    const dim3 grid(sp.n0 + sp.o[1].nvp / 8, 1, count);
    count_launch();
    if (res) {
      cudaFuncSetAttribute(oz_fused_kernel<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
      oz_fused_kernel<T, true><<<grid, 256, sm, s>>>(sp, K, Kp, P, bits, nb2, kdev, pl.wt, ldk);
    } else {
      cudaFuncSetAttribute(oz_fused_kernel<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
      oz_fused_kernel<T, false><<<grid, 256, sm, s>>>(sp, K, Kp, P, bits, nb2, kdev, CrtWeights{}, ldk);
    }
  } else {
    // the scale codes start at 0 (the zero vector)
    cudaMemsetAsync(ea, 0, sizeof(int) * ((size_t)Mp + Np) * count, s);
    sp.n0 = (M + 31) / 32;
    count_launch(2);
    oz_scale_kernel<T><<<dim3(sp.n0 + (N + 31) / 32, (K + kScaleK - 1) / kScaleK, count), 256, 0, s>>>(sp, K, nb2,
                                                                                                      kdev);
    sp.n0 = Mp / 32;
    const dim3 tiles(sp.n0 + (sp.o[1].nvp + 31) / 32, Kp / 64, count);
    if (res) oz_split_kernel<T, true><<<tiles, 256, 0, s>>>(sp, K, Kp, P, bits, nb2, kdev, pl.wt);
    else oz_split_kernel<T, false><<<tiles, 256, 0, s>>>(sp, K, Kp, P, bits, nb2, kdev, CrtWeights{});
  }
  const long long wait = wait_cycles > 0 ? wait_cycles : (1ll << 32);
  // Moduli of a tile over ng CTAs when the tiles alone leave SMs idle: the rounds of 152 CTAs
  // times the moduli per CTA (one more for its prologue) is least.  The residues, and so the
  // result, do not depend on ng.
  int ng = 1;
  if (res) {
    const long long mt = Mp / OZ_BM, nt = Np / crtc::BN;
    const long long tl = std::max<long long>(1, (lower ? (mt * nt + mt) / 2 : mt * nt) * count);
    long long best = -1;
    for (int g = 1; g <= P && (long long)count * g <= 65535; g++) {
      const long long cost = ((tl * g + 151) / 152) * ((P + g - 1) / g + 1);
      if (best < 0 || cost < best) {
        best = cost;
        ng = g;
      }
    }
  }
  dim3 grid(Np / (res ? crtc::BN : OZ_BN), Mp / OZ_BM, count * ng);
  CUtensorMap ma, mb;
  if (!digit_map(&ma, Ad, (long long)count * P * Mp, Kp, tcg::BM) ||
      !digit_map(&mb, Bd, (long long)count * P * Np, Kp, res ? crtc::BN : tcg::BN))
    return false;
  if (res) {
    CrtArgs ca;
    ca.Ad = Ad;
    ca.Bd = Bd;
    ca.R = R;
    ca.Mp = Mp;
    ca.Np = Np;
    ca.Kp = Kp;
    ca.n = P;
    ca.ng = ng;
    ca.cplx = cplx ? 1 : 0;
    ca.lower = lower;
    ca.zR = zR;
    ca.kdev = kdev;
    ca.wait = wait;
    ca.skip_copy = skip_copy;
    cudaFuncSetAttribute(crt_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, crtc::SMEM);
    count_launch(2);
    crt_tc_kernel<<<grid, tcg::THREADS, crtc::SMEM, s>>>(ma, mb, ca, status);
    const int ncg = (N + (cplx ? 3 : 7)) / (cplx ? 4 : 8);
    crt_recon_kernel<T><<<dim3((unsigned)(((long long)M * ncg + 127) / 128), 1, count), 128, 0, s>>>(
        R, zR, Mp, Np, M, N, ncg, ea, eb, Mp, Np, -2 * pl.p, pl.cr, C, ldc, sC, sC2, nb2, alpha, beta, lower);
    return true;
  }
  OzArgs oa;
  oa.Ad = Ad;
  oa.Bd = Bd;
  oa.ea = ea;
  oa.eb = eb;
  oa.C = C;
  oa.ldc = ldc;
  oa.M = M;
  oa.N = N;
  oa.Mp = Mp;
  oa.Np = Np;
  oa.Kp = Kp;
  oa.S = P;
  oa.cplx = cplx ? 1 : 0;
  oa.lower = lower;
  oa.alpha = alpha;
  oa.beta = beta;
  oa.sAd = (long long)Mp * Kp;
  oa.sBd = (long long)Np * Kp;
  oa.zAd = zA;
  oa.zBd = zB;
  oa.zEa = Mp;
  oa.zEb = Np;
  oa.zC = sC;
  oa.zC2 = sC2;
  oa.nb2 = nb2;
  oa.kdev = kdev;
  oa.wait = wait;
  oa.skip_copy = skip_copy;
  cudaFuncSetAttribute(oz_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tcg::SMEM);
  count_launch();
  oz_tc_kernel<<<grid, tcg::THREADS, tcg::SMEM, s>>>(ma, mb, oa, status);
  return true;
}

template bool ozaki_gemm<double>(int, int, int, int, int, double, const double*, int, long long, const double*, int,
                                 long long, double, double*, int, long long, int, int, int, void*, DevStatus*,
                                 cudaStream_t, const double*, long long, const int*, long long, long long,
                                 long long, long long, long long, int);
template bool ozaki_gemm<zc>(int, int, int, int, int, double, const zc*, int, long long, const zc*, int, long long,
                             double, zc*, int, long long, int, int, int, void*, DevStatus*, cudaStream_t,
                             const double*, long long, const int*, long long, long long, long long, long long,
                             long long, int);

}  // namespace gks
