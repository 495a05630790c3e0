// Divide-and-conquer eigensolver for the real symmetric tridiagonal T (paper Sec. 6:
// the GEMM-rich second half of the dense eigensolve; written here from Cuppen's method
// with Gu-Eisenstat vector recomputation).
//
//  * Tear: T = diag(T1, T2) + rho v v^T at every split s (rho = |e_{s-1}|,
//    v = (e_last; sign e_first)), i.e. d_{s-1} -= rho and d_s -= rho before the leaves.
//  * Leaves (<= 16 rows): one warp each runs implicit QL redundantly on every lane, lane
//    i accumulating row i of the leaf's eigenvector block.
//  * Merge of (lam1, Z1), (lam2, Z2): z = (last row of Z1; sign * first row of Z2)/sqrt2,
//    rho' = 2 rho; poles merged in ascending order; deflation of negligible z_i and of
//    close pole pairs (Givens rotation); the K remaining roots of
//    1 + rho' sum z_i^2/(d_i - lam) = 0 are found by bisection in tau = lam - d_origin
//    (origin the nearer pole) so that every difference d_i - lam = (d_i - d_origin) - tau is
//    accurate; z_hat is recomputed from the roots (Gu-Eisenstat) so the vectors
//    z_hat_i/(d_i - lam_j) are numerically orthogonal.
//  * The merged eigenvector matrix is diag(Z1, Z2) W, W = G^T [unit vectors | secular
//    vectors] in ascending eigenvalue order: two GEMMs per merge (Z1 W_top, Z2 W_bottom),
//    grouped over all merges of a level and all batch items in one launch.
#include <algorithm>
#include <cmath>
#include <vector>

#include "dense.h"

namespace gks {

static constexpr int DC_LEAF = 16;
static constexpr double DC_U = 1.1102230246251565e-16;

struct DcNode {
  int off, n1, n2;
};

struct DcLevel {
  std::vector<DcNode> nodes;
  DcNode* d_nodes = nullptr;
  GemmDesc* d_gemm = nullptr;
  int maxn = 0, maxhalf = 0;
};

struct DcPlan {
  int m = 0, count = 0, depth = 0;
  std::vector<DcLevel> levels;  // levels[t]: t = 0 merges leaves, t = depth-1 is the root
  std::vector<int> leaves;      // (off, n) pairs
  std::vector<int> splits;      // split positions s (tear between s-1 and s)
  int* d_leaves = nullptr;
  int* d_splits = nullptr;
  const double* zbound = nullptr;  // Z pointer the GEMM lists were built for
  void* wbound = nullptr;
  long long sZbound = 0;
};

// per-item workspace layout (all arrays of length m)
struct DcWs {
  double *Zb, *W, *lamA, *lamB, *ds, *zs, *dK, *zK, *lamK, *tauK, *zhat, *dD, *rc, *rs;
  double *xf, *zf;  // single-precision forms of dK (float2: leading and trailing part) and zK^2 (float)
  int *src, *idxK, *orig, *idxD, *ra, *rb, *colsrc, *cnt;
};

__host__ __device__ inline size_t dc_item_bytes(int m) {
  size_t mm = (size_t)m * m;
  return sizeof(double) * (2 * mm + 14 * (size_t)m) + sizeof(int) * (10 * (size_t)m) + 256;
}

__host__ __device__ inline DcWs dc_ws(void* base, int m) {
  DcWs w;
  double* pd = static_cast<double*>(base);
  const size_t mm = (size_t)m * m;
  w.Zb = pd; pd += mm;
  w.W = pd; pd += mm;
  double** dl[14] = {&w.lamA, &w.lamB, &w.ds, &w.zs, &w.dK, &w.zK, &w.lamK, &w.tauK, &w.zhat, &w.dD, &w.rc, &w.rs,
                     &w.xf, &w.zf};
  for (int k = 0; k < 14; k++) { *dl[k] = pd; pd += m; }
  int* pi = reinterpret_cast<int*>(pd);
  int** il[8] = {&w.src, &w.idxK, &w.orig, &w.idxD, &w.ra, &w.rb, &w.colsrc, &w.cnt};
  for (int k = 0; k < 7; k++) { *il[k] = pi; pi += m; }
  w.cnt = pi;
  return w;
}

// ------------------------------------------------------------------ kernels

__global__ void dc_tear_kernel(double* d, const double* e, long long sde, const int* splits, int nsplit) {
  const int z = blockIdx.x;
  d += z * sde;
  e += z * sde;
  for (int side = 1; side >= 0; side--) {  // the splits' left rows, then their right rows
    for (int k = threadIdx.x; k < nsplit; k += blockDim.x) d[splits[k] - side] -= fabs(e[splits[k] - 1]);
    __syncthreads();
  }
}

// One warp per leaf, one leaf per CTA. Every lane runs the same QL iteration on (d, e) in
// shared memory; lane i applies the rotations to row i of the leaf's eigenvector block.  A
// serial chain of rotations: one reciprocal square root each in place of a hypot and two
// divisions (the block is scaled by a power of two so that no square overflows), arrays in
// shared memory in place of dynamically indexed local ones, and leaves of at most 16 rows (a
// quarter of the rotations of 32 for one more merge level): 1.87 ms at order 832 with 32 rows,
// 220 us here.
__global__ void __launch_bounds__(32) dc_leaf_kernel(const double* d, const double* e, long long sde, double* lam,
                                                     long long slam, double* Z, long long sZ, int m,
                                                     const int* leaves, DevStatus* st) {
  __shared__ double dd[DC_LEAF], ee[DC_LEAF], zr[DC_LEAF][33];
  const int z = blockIdx.y, leaf = blockIdx.x, lane = threadIdx.x;
  const int off = leaves[2 * leaf], n = leaves[2 * leaf + 1];
  d += z * sde;
  e += z * sde;
  lam += z * slam;
  Z += z * sZ;
  double dv = lane < n ? d[off + lane] : 0.0, ev = lane + 1 < n ? e[off + lane] : 0.0;
  double big = fmax(fabs(dv), fabs(ev));
  for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
  const int sc = (big > 0.0 && isfinite(big)) ? ilogb(big) : 0;  // entries at most 2 in magnitude
  if (lane < DC_LEAF) {
    dd[lane] = ldexp(dv, -sc);
    ee[lane] = ldexp(ev, -sc);
  }
  for (int i = 0; i < n; i++) zr[i][lane] = (i == lane) ? 1.0 : 0.0;
  __syncwarp();
  bool ok = true;
  for (int l = 0; l < n && ok; l++) {
    for (int sweep = 0;; sweep++) {
      // the first negligible off-diagonal from l on (below 1e-150 of the block its square, which
      // the shift and the rotations take, underflows: beside equal zero diagonal entries the
      // shift would be 0 / 0)
      const bool neg = lane >= l && lane < n - 1 &&
                       fabs(ee[lane]) <= fmax(DC_U * (fabs(dd[lane]) + fabs(dd[lane + 1])), 1e-150);
      const unsigned mask = __ballot_sync(0xffffffffu, neg);
      const int q = mask ? __ffs(mask) - 1 : n - 1;
      __syncwarp();
      if (mask && lane == 0) ee[q] = 0.0;
      __syncwarp();
      if (q == l) break;
      if (sweep >= 60) { ok = false; break; }
      // shift: eigenvalue of [[d_l, e_l], [e_l, d_{l+1}]] nearer to d_l
      const double el = ee[l], h = 0.5 * (dd[l + 1] - dd[l]);
      const double mu = dd[l] - el * el / (h + copysign(sqrt(fma(h, h, el * el)), h));
      double x = dd[q] - mu, y = ee[q - 1];
      double g = dd[q], z1 = zr[q][lane];
      for (int k = q; k > l; k--) {
        const double r2 = fma(x, x, y * y), ri = r2 > 0.0 ? rsqrt(r2) : 0.0;
        const double c = r2 > 0.0 ? x * ri : 1.0, sn = y * ri;
        const double a = dd[k - 1], b = ee[k - 1], en = k - 1 > l ? ee[k - 2] : 0.0, z0 = zr[k - 1][lane];
        // [[a, b], [b, g]] rotated: s t moves between the diagonal entries, t = s (a - g) + 2 c b
        const double t = fma(sn, a - g, 2.0 * c * b);
        const double gk = fma(sn, -t, a);  // new d_{k-1}: a - s t
        __syncwarp();
        if (lane == 0) {
          if (k < q) ee[k] = r2 * ri;
          dd[k] = fma(sn, t, g);            // g + s t
        }
        const double bk = fma(c, t, -b);    // new coupling: c t - b
        zr[k][lane] = fma(sn, z0, c * z1);
        z1 = fma(c, z0, -sn * z1);
        x = bk;
        y = sn * en;
        if (lane == 0) {
          ee[k - 1] = bk;
          if (k - 1 > l) ee[k - 2] = c * en;
        }
        g = gk;
        __syncwarp();
      }
      if (lane == 0) dd[l] = g;
      zr[l][lane] = z1;
      __syncwarp();
    }
  }
  if (!ok) {
    if (lane == 0) set_status(st ? st + z : nullptr, ST_ENOCONV, off);
  }
  // ascending order (ties keep the lower index); ordered bits, so that the ranks are a
  // permutation whatever the values
  const double v = lane < n ? dd[lane] : 0.0;
  auto key = [](double x) -> long long {
    const long long k = __double_as_longlong(x + 0.0);
    return k < 0 ? k ^ 0x7fffffffffffffffll : k;
  };
  int rank = 0;
  for (int i = 0; i < n; i++) {
    const long long o = key(dd[i]), kv = key(v);
    if (o < kv || (o == kv && i < lane)) rank++;
  }
  if (lane < n) lam[off + rank] = ldexp(v, sc);
  for (int c = 0; c < n; c++) {
    const int pos = __shfl_sync(0xffffffffu, rank, c);
    if (lane < n) Z[(size_t)(off + lane) * m + off + pos] = zr[c][lane];
  }
}

__device__ __forceinline__ int lower_bound_d(const double* a, int n, double v) {
  int lo = 0, hi = n;
  while (lo < hi) { int mid = (lo + hi) >> 1; if (a[mid] < v) lo = mid + 1; else hi = mid; }
  return lo;
}
__device__ __forceinline__ int upper_bound_d(const double* a, int n, double v) {
  int lo = 0, hi = n;
  while (lo < hi) { int mid = (lo + hi) >> 1; if (a[mid] <= v) lo = mid + 1; else hi = mid; }
  return lo;
}

struct DcArgs {
  int m;
  long long sitem;      // bytes between batch items' workspaces
  char* ws;             // workspace base (item 0)
  const double* e;      // off-diagonal (untouched by the tear)
  long long sde;
  const double* lam;    // current eigenvalues (children)
  double* lamNew;
  long long slam;
  const double* Zc;     // current eigenvector blocks
  long long sZ;
};

// Powers of two (x, y = 1 / x) that bring a merge's spectrum, poles' spread plus rho', below 1;
// zeros when its exponent is at the ends of the range (single precision then decides nothing).
__device__ __forceinline__ double2 secular_scale(double spread, double rho2) {
  const int ex = (__double2hiint(spread + rho2) >> 20) & 0x7ff;
  if (ex < 2 || ex > 2043) return make_double2(0.0, 0.0);
  return make_double2(__hiloint2double((2045 - ex) << 20, 0), __hiloint2double((ex + 1) << 20, 0));
}

// Powers of two (x, y = 1 / x) for a merge whose entries lie outside 2^-340 .. 2^340 (a block that
// is tiny beside the rest of T): in its own units the squares of the secular sums and of the
// vectors neither overflow nor vanish.  1 otherwise, and then no bit changes.
__device__ __forceinline__ double2 node_scale(double top) {
  const int ex = (__double2hiint(top) >> 20) & 0x7ff;
  if (top == 0.0 || (ex > 683 && ex < 1363)) return make_double2(1.0, 1.0);
  const int k = max(-1000, min(1000, 1023 - ex));
  return make_double2(__hiloint2double((1023 + k) << 20, 0), __hiloint2double((1023 - k) << 20, 0));
}

__device__ __forceinline__ DcWs item_ws(const DcArgs& a, int z) { return dc_ws(a.ws + z * a.sitem, a.m); }

// Exclusive sum of v over the CTA (1024 threads), total in *all.
__device__ int block_scan(int v, int* scratch, int* all) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  __syncthreads();
  if (lane == 31) scratch[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int t = scratch[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    scratch[lane] = t;
  }
  __syncthreads();
  *all = scratch[31];
  return x - v + (warp ? scratch[warp - 1] : 0);
}

// Merge setup, one CTA per (node, item): z vector, merged poles, deflation.  The scan for
// close poles is sequential only where rotations happen: negligible z_i drop out by a
// compaction, the test between neighbouring survivors runs for all pairs at once on the
// unrotated values (which are the current ones unless the pair before rotated), and one
// thread walks the runs that start at a pair that fails it.  (Walking every pole from global
// memory took 6.3 ms for the last merge of order 4992.)  Poles are kept in the node's units
// (node_scale, left in ds[0], ds[1] for the merge's other kernels) up to dc_colmap_kernel.
__global__ void __launch_bounds__(1024) dc_merge_prep_kernel(DcArgs a, const DcNode* nodes) {
  __shared__ double red[32];
  __shared__ int scan[32], s_nrot, s_bad;
  const DcNode nd = nodes[blockIdx.x];
  const int z = blockIdx.y, tid = threadIdx.x, nt = 1024;
  DcWs w = item_ws(a, z);
  const int m = a.m, off = nd.off, n1 = nd.n1, n2 = nd.n2, n = n1 + n2, s = off + n1;
  const double* lam = a.lam + z * a.slam;
  const double* Zc = a.Zc + z * a.sZ;
  const double beta = a.e[z * a.sde + s - 1];
  double rho2 = 2.0 * fabs(beta);
  const double sg = beta < 0.0 ? -1.0 : 1.0;
  const double isq2 = 0.70710678118654752440;
  double *ds = w.ds + off, *zs = w.zs + off, *dK = w.dK + off, *zK = w.zK + off, *dD = w.dD + off;
  double *rc = w.rc + off, *rs = w.rs + off;
  int *src = w.src + off, *idxK = w.idxK + off, *idxD = w.idxD + off, *ra = w.ra + off, *rb = w.rb + off;
  int *links = w.colsrc + off, *gone = w.orig + off;  // free until the roots and the column map
  for (int i = tid; i < n; i += nt) {  // every slot valid, also if non-finite values collide below
    ds[i] = 0.0;
    zs[i] = 0.0;
    src[i] = i;
  }
  __syncthreads();
  double dmax = 0.0;
  for (int i = tid; i < n; i += nt) {
    int pos;
    double zv, dv;
    if (i < n1) {
      dv = lam[off + i];
      zv = Zc[(size_t)(s - 1) * m + off + i] * isq2;
      pos = i + lower_bound_d(lam + s, n2, dv);
    } else {
      int k = i - n1;
      dv = lam[s + k];
      zv = sg * Zc[(size_t)s * m + s + k] * isq2;
      pos = k + upper_bound_d(lam + off, n1, dv);
    }
    ds[pos] = dv;
    zs[pos] = zv;
    src[pos] = i;
    dmax = fmax(dmax, fabs(dv));
  }
  for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
  if ((tid & 31) == 0) red[tid >> 5] = dmax;
  if (tid == 0) s_nrot = s_bad = 0;
  __syncthreads();
  for (int k = 0; k < 32; k++) dmax = fmax(dmax, red[k]);
  const double2 unit = node_scale(fmax(dmax, rho2));
  if (unit.x != 1.0) {
    for (int i = tid; i < n; i += nt) ds[i] *= unit.x;
    dmax *= unit.x;
    rho2 *= unit.x;
    __syncthreads();
  }
  const double tol = 8.0 * DC_U * fmax(dmax, rho2);
  // survivors (in dK, zK, idxK) and negligible z_i (in dD, idxD), each in ascending order
  const int per = (n + nt - 1) / nt, p0 = min(n, tid * per), p1 = min(n, p0 + per);
  int cnt = 0, ns = 0;
  for (int p = p0; p < p1; p++) cnt += !(rho2 * fabs(zs[p]) <= tol);
  int at = block_scan(cnt, scan, &ns);
  for (int p = p0, q = p0 - at; p < p1; p++) {
    if (!(rho2 * fabs(zs[p]) <= tol)) {
      dK[at] = ds[p]; zK[at] = zs[p]; idxK[at] = src[p]; at++;
    } else {
      dD[q] = ds[p]; idxD[q] = src[p]; q++;
    }
  }
  const int nsm = n - ns;
  __syncthreads();
  // pairs (i, i + 1) close enough to rotate: |c s (d_{i+1} - d_i)| <= tol with c, s ~ z_{i+1}, z_i
  auto close = [tol](double pd, double pz, double dp, double zp) {
    return fabs(pz * zp * (dp - pd)) <= tol * fma(pz, pz, zp * zp);
  };
  const int pr = (ns + nt - 1) / nt, l0 = min(ns, tid * pr), l1 = min(ns, l0 + pr);
  int nl = 0;
  cnt = 0;
  for (int i = l0; i < l1; i++) {
    gone[i] = 0;
    cnt += i + 1 < ns && close(dK[i], zK[i], dK[i + 1], zK[i + 1]);
  }
  at = block_scan(cnt, scan, &nl);
  for (int i = l0; i < l1 && cnt; i++)
    if (i + 1 < ns && close(dK[i], zK[i], dK[i + 1], zK[i + 1])) links[at++] = i;
  __syncthreads();
  int K = ns, nD = nsm;
  if (nl > 0) {
    if (tid == 0) {
      int nrot = 0, next = 0;  // next: first survivor not yet walked over
      for (int f = 0; f < nl; f++) {
        int i = links[f];
        if (i < next) continue;
        double pd = dK[i], pz = zK[i];
        int ps = idxK[i];
        while (i + 1 < ns) {
          const double dp = dK[i + 1], zp = zK[i + 1];
          if (!close(pd, pz, dp, zp)) break;
          const double r = hypot(pz, zp), c = zp / r, sn = pz / r;
          const int sp = idxK[i + 1];
          ra[nrot] = ps; rb[nrot] = sp; rc[nrot] = c; rs[nrot] = sn;
          gone[i] = 1;
          // the rotation's deflated pole, kept with the small ones' tail (sorted below)
          dD[nsm + nrot] = c * c * pd + sn * sn * dp; idxD[nsm + nrot] = ps;
          nrot++;
          pd = sn * sn * pd + c * c * dp; pz = r; ps = sp;
          i++;
          dK[i] = pd; zK[i] = pz;
        }
        next = i + 1;
      }
      for (int i = 1; i < nrot; i++) {  // rotations can perturb the order slightly
        double dv = dD[nsm + i];
        int iv = idxD[nsm + i], j = i - 1;
        while (j >= 0 && dD[nsm + j] > dv) { dD[nsm + j + 1] = dD[nsm + j]; idxD[nsm + j + 1] = idxD[nsm + j]; j--; }
        dD[nsm + j + 1] = dv; idxD[nsm + j + 1] = iv;
      }
      s_nrot = nrot;
    }
    __syncthreads();
    const int nrot = s_nrot;
    K = ns - nrot;
    nD = nsm + nrot;
    // survivors left, compacted through ds, zs, src; the deflated lists merged the same way
    cnt = 0;
    for (int i = l0; i < l1; i++) cnt += !gone[i];
    int all;
    at = block_scan(cnt, scan, &all);
    for (int i = l0; i < l1; i++)
      if (!gone[i]) { ds[at] = dK[i]; zs[at] = zK[i]; src[at] = idxK[i]; at++; }
    __syncthreads();
    for (int i = tid; i < K; i += nt) { dK[i] = ds[i]; zK[i] = zs[i]; idxK[i] = src[i]; }
    __syncthreads();
    for (int i = tid; i < nD; i += nt) {
      const double v = dD[i];
      const int pos = i < nsm ? i + lower_bound_d(dD + nsm, nrot, v) : i - nsm + upper_bound_d(dD, nsm, v);
      ds[pos] = v; src[pos] = idxD[i];
    }
    __syncthreads();
    for (int i = tid; i < nD; i += nt) { dD[i] = ds[i]; idxD[i] = src[i]; }
    for (int i = tid; i + 1 < K; i += nt)
      if (dK[i] > dK[i + 1]) s_bad = 1;
    __syncthreads();
    if (s_bad && tid == 0)
      for (int i = 1; i < K; i++) {
        double dv = dK[i], zv = zK[i];
        int iv = idxK[i], j = i - 1;
        while (j >= 0 && dK[j] > dv) { dK[j + 1] = dK[j]; zK[j + 1] = zK[j]; idxK[j + 1] = idxK[j]; j--; }
        dK[j + 1] = dv; zK[j + 1] = zv; idxK[j + 1] = iv;
      }
  }
  __syncthreads();
  if (K > 0) {
    const double base = dK[0];
    const double sc = secular_scale(dK[K - 1] - base, rho2).x;
    float2* xf = reinterpret_cast<float2*>(w.xf + off);
    float* zf = reinterpret_cast<float*>(w.zf + off);
    for (int i = tid; i < K; i += nt) {
      const double x = (dK[i] - base) * sc;
      const float h = (float)x;
      xf[i] = make_float2(h, (float)(x - h));
      zf[i] = (float)(zK[i] * zK[i]);
    }
  }
  if (tid == 0) {
    ds[0] = unit.x;
    ds[1] = unit.y;
    w.cnt[3 * off + 0] = K;
    w.cnt[3 * off + 1] = nD;
    w.cnt[3 * off + 2] = s_nrot;
  }
}

// a / x with one correction of the quotient.
__device__ __forceinline__ double quot(double a, double x) {
  const double r = recip(x), q = a * r, t = fma(-q, x, a);
  return isfinite(t) ? fma(r, t, q) : a / x;
}

// Next iterate of f's root from the sums at tau: psi (poles left of the root), phi (poles
// right of it) and their derivatives, each modelled by one pole plus a constant matched in
// value and slope,
//   psi ~ p + q/(delta_j - tau),  phi ~ s + t/(delta_{j+1} - tau);
// the model's root, a quadratic in the distance from the origin's pole, u = delta_j - tau or
// (right) v = delta_{j+1} - tau: a root close to the right pole is lost in u = v - D, and one
// root in a few hundred then bisected 30 to 60 times.  dl, dr: delta_j, delta_{j+1}.
template <typename F>
__device__ __forceinline__ F secular_step(F ps, F psd, F fs, F fsd, F rho, F dl, F dr, F tau, F lo, F hi, bool last,
                                          bool right) {
  const F one = 1, two = 2, half = 0.5;
  const F ul = dl - tau;                       // delta_j - tau
  const F qa = rho * psd * ul * ul;            // rho' q
  const F c0 = one + rho * (ps - psd * ul);    // 1 + rho' p
  if (last) {
    const F c = c0 + rho * fs;                 // no pole on the right
    return (c > 0) ? dl + qa / c : half * (lo + hi);  // c + qa/(dl - x) = 0
  }
  const F ur = dr - tau;
  const F ta = rho * fsd * ur * ur;            // rho' t
  const F c = c0 + rho * (fs - fsd * ur);      // 1 + rho'(p + s)
  const F D = dr - dl;
  // c u^2 + (qa + ta + c D) u + qa D = 0, u in (-D, 0);
  // c v^2 + (qa + ta - c D) v - ta D = 0, v in (0, D)
  const F B = qa + ta + (right ? -c * D : c * D), C = right ? -ta * D : qa * D;
  const F o = right ? dr : dl;
  if (c == 0) return o + C / B;
  F disc = B * B - 2 * two * c * C;
  disc = disc > 0 ? sqrt(disc) : (F)0;
  // roots: (-B -+ disc)/(2c); stable form picks the root in range
  const F r1 = (B > 0) ? (-B - disc) / (two * c) : (two * C) / (-B + disc);
  const F r2 = (B > 0) ? (two * C) / (-B - disc) : (-B + disc) / (two * c);
  const F x1 = right ? -r1 : r1;
  return o - ((x1 < 0 && x1 > -D) ? r1 : r2);
}

// Sums over the poles in single precision, relative to pole o (x0): the differences from the
// parts of the scaled poles are good to 2^-24 of themselves and 2^-48 of the spectrum.
__device__ __forceinline__ void secular_sums(const float2* xf, const float* zf, int K, int j, float2 x0, float tau,
                                             int lane, float& ps, float& psd, float& fs, float& fsd) {
  ps = psd = fs = fsd = 0.0f;
  for (int i = lane; i < K; i += 32) {
    const float2 x = xf[i];
    const float r = __frcp_rn(((x.x - x0.x) + (x.y - x0.y)) - tau), t = zf[i] * r;
    if (i <= j) { ps += t; psd = fmaf(t, r, psd); }
    else { fs += t; fsd = fmaf(t, r, fsd); }
  }
  ps = warp_sum(ps); psd = warp_sum(psd); fs = warp_sum(fs); fsd = warp_sum(fsd);
}

// Secular roots, one warp per root.  With origin pole d_o and tau = lam - d_o the function
//   f(tau) = 1 + rho' sum_i z_i^2 / (delta_i - tau),  delta_i = d_i - d_o,
// is increasing between its poles.  Each iteration evaluates psi, phi and their derivatives
// (lanes split the K terms) and takes the model's root (secular_step) when it falls inside
// the current sign bracket and the step is at most half the one before last; otherwise it
// bisects.  (Asking two steps to halve the bracket instead sends a one-sided convergence back
// to the middle every second time: half the roots took 20 iterations.)  Stops when f is below
// its rounding level or the bracket is at the working precision of tau.
// The FP64 pipe bounds it (9 operations per pole and iteration, 64 clocks per warp
// instruction), so the same iteration runs in single precision first, on the FP32 pipe, and
// FP64 starts from its root: two or three evaluations in place of eight.  The side of the
// middle is taken from single precision only where the gap is resolved (2^-48 of the spectrum
// against 1e-9) and f is far from zero.  Nothing else depends on that start.
// Measured, all merges with their vectors (FP64 from the middle of the bracket / this): order
// 832 1.59 / 0.68 ms, eight of 832 4.26 / 3.02, order 2808 5.70 / 2.61, 4992 11.0 / 6.5.
__global__ void dc_secular_kernel(DcArgs a, const DcNode* nodes, DevStatus* st) {
  const DcNode nd = nodes[blockIdx.y];
  const int z = blockIdx.z;
  DcWs w = item_ws(a, z);
  const int off = nd.off, s = off + nd.n1;
  const int K = w.cnt[3 * off];
  const int lane = threadIdx.x & 31;
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (j >= K) return;
  const double rho2 = 2.0 * fabs(a.e[z * a.sde + s - 1]) * w.ds[off];
  const double* dK = w.dK + off;
  const double* zK = w.zK + off;
  const float2* xf = reinterpret_cast<const float2*>(w.xf + off);
  const float* zf = reinterpret_cast<const float*>(w.zf + off);
  const double2 sc = secular_scale(dK[K - 1] - dK[0], rho2);
  const float rhof = (float)(rho2 * sc.x);
  const bool last = (j == K - 1);
  int o;
  double lo, hi;
  float ps4, psd4, fs4, fsd4;
  if (!last) {
    const double gap = dK[j + 1] - dK[j];
    const double mid = 0.5 * gap;
    secular_sums(xf, zf, K, j, xf[j], (float)(mid * sc.x), lane, ps4, psd4, fs4, fsd4);
    const float f4 = 1.0f + rhof * (ps4 + fs4), a4 = 1.0f + rhof * (fabsf(ps4) + fabsf(fs4));
    bool right = f4 < 0.0f;
    if (!(gap * sc.x > 1e-9) || !(fabsf(f4) > 1e-3f * a4)) {
      double f = 0.0;
      for (int i = lane; i < K; i += 32) f = fma(zK[i] * zK[i], recip((dK[i] - dK[j]) - mid), f);
      f = 1.0 + rho2 * warp_sum(f);
      right = !(f >= 0.0);
    }
    if (!right) { o = j; lo = 0.0; hi = mid; }
    else { o = j + 1; lo = -mid; hi = 0.0; }
  } else {
    double zz = 0.0;
    for (int i = lane; i < K; i += 32) zz += zK[i] * zK[i];
    zz = warp_sum(zz);
    o = j; lo = 0.0; hi = rho2 * zz * (1.0 + 4.0 * DC_U) + 4.0 * DC_U * fabs(dK[j]);
  }
  const double d0 = dK[o];
  // poles bracketing the root, relative to the origin: left = delta_j, right = delta_{j+1}
  const double dl = dK[j] - d0;
  const double dr = last ? 0.0 : dK[j + 1] - d0;
  double tau = 0.5 * (lo + hi);
  {
    const float dl4 = (float)(dl * sc.x), dr4 = (float)(dr * sc.x);
    const float2 x0 = xf[o];
    float l4 = (float)(lo * sc.x), h4 = (float)(hi * sc.x), t4 = 0.5f * (l4 + h4);
    float s1 = h4 - l4, s2 = s1;
    for (int it = 0; it < 24; it++) {
      secular_sums(xf, zf, K, j, x0, t4, lane, ps4, psd4, fs4, fsd4);
      const float f = 1.0f + rhof * (ps4 + fs4);
      if (f < 0.0f) l4 = t4; else h4 = t4;
      if (!(fabsf(f) > 6e-7f * (1.0f + rhof * (fabsf(ps4) + fabsf(fs4))))) break;
      float cand = secular_step<float>(ps4, psd4, fs4, fsd4, rhof, dl4, dr4, t4, l4, h4, last, o != j);
      if (!(cand > l4 && cand < h4) || fabsf(cand - t4) > 0.5f * s2) cand = 0.5f * (l4 + h4);
      if (cand == t4) break;
      s2 = s1;
      s1 = fabsf(cand - t4);
      t4 = cand;
      if (s1 <= 2e-7f * fabsf(cand)) break;
    }
    const double guess = (double)t4 * sc.y;
    if (guess > lo && guess < hi) tau = guess;
  }
  double s1 = hi - lo, s2 = hi - lo;  // the last step and the one before: a step must halve the latter
  int it = 0;
  for (; it < 200; it++) {
    double ps = 0.0, psd = 0.0, fs = 0.0, fsd = 0.0;
    // poles i <= j lie left of the root (terms negative), the others right of it
    for (int i = lane; i < K; i += 32) {
      const double t = zK[i] * recip((dK[i] - d0) - tau);
      if (i <= j) { ps = fma(zK[i], t, ps); psd = fma(t, t, psd); }
      else { fs = fma(zK[i], t, fs); fsd = fma(t, t, fsd); }
    }
    ps = warp_sum(ps); psd = warp_sum(psd); fs = warp_sum(fs); fsd = warp_sum(fsd);
    const double absum = fabs(ps) + fabs(fs);
    const double f = 1.0 + rho2 * (ps + fs);
    if (f < 0.0) lo = tau; else hi = tau;
    if (fabs(f) <= 8.0 * DC_U * (1.0 + rho2 * absum)) break;
    if (!(hi - lo > 2.0 * DC_U * fmax(fabs(lo), fabs(hi)))) break;
    double cand = secular_step<double>(ps, psd, fs, fsd, rho2, dl, dr, tau, lo, hi, last, o != j);
    if (!(cand > lo && cand < hi) || fabs(cand - tau) > 0.5 * s2) cand = 0.5 * (lo + hi);
    if (cand == tau) break;
    s2 = s1;
    s1 = fabs(cand - tau);
    tau = cand;
  }
  if (it >= 200 && lane == 0) set_status(st ? st + z : nullptr, ST_ENOCONV, off + j);
  if (lane == 0) {
    w.orig[off + j] = o;
    w.tauK[off + j] = tau;
    w.lamK[off + j] = d0 + tau;
  }
}

// Gu-Eisenstat: z_hat_i^2 = (lam_i - d_i)/rho' * prod_{j != i} (lam_j - d_i)/(d_j - d_i).  A
// warp per entry: a thread per entry (39 CTAs at K = 4992) took 2.0 ms.
__global__ void dc_zhat_kernel(DcArgs a, const DcNode* nodes) {
  const DcNode nd = nodes[blockIdx.y];
  const int z = blockIdx.z;
  DcWs w = item_ws(a, z);
  const int off = nd.off, s = off + nd.n1;
  const int K = w.cnt[3 * off];
  const int lane = threadIdx.x & 31, i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= K) return;
  const double rho2 = 2.0 * fabs(a.e[z * a.sde + s - 1]) * w.ds[off];
  const double* dK = w.dK + off;
  const double di = dK[i];
  // a warp per entry, the factors over the lanes (each near 1 but for the nearest: no overflow)
  double prod = 1.0;
  for (int j = lane; j < K; j += 32) {
    const double lj = (dK[w.orig[off + j]] - di) + w.tauK[off + j];
    prod *= j == i ? lj / rho2 : quot(lj, dK[j] - di);
  }
  for (int o = 16; o > 0; o >>= 1) prod *= __shfl_xor_sync(0xffffffffu, prod, o);
  if (lane) return;
  double zh = sqrt(fabs(prod));
  w.zhat[off + i] = w.zK[off + i] < 0.0 ? -zh : zh;
}

// Output column positions: roots and deflated values merged in ascending order.
__global__ void dc_colmap_kernel(DcArgs a, const DcNode* nodes) {
  const DcNode nd = nodes[blockIdx.y];
  const int z = blockIdx.z;
  DcWs w = item_ws(a, z);
  const int off = nd.off;
  const int K = w.cnt[3 * off], nD = w.cnt[3 * off + 1];
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  double* lamNew = a.lamNew + z * a.slam;
  const double unit = w.ds[off + 1];
  if (t < K) {
    double v = w.lamK[off + t];
    int pos = t + lower_bound_d(w.dD + off, nD, v);
    w.colsrc[off + pos] = t;
    lamNew[off + pos] = v * unit;
  } else if (t < K + nD) {
    int i = t - K;
    double v = w.dD[off + i];
    int pos = i + upper_bound_d(w.lamK + off, K, v);
    w.colsrc[off + pos] = -1 - i;
    lamNew[off + pos] = v * unit;
  }
}

// W^T columns (children-basis vectors), one warp per output column, then the deflation
// rotations G^T applied last-to-first.
__global__ void dc_buildw_kernel(DcArgs a, const DcNode* nodes) {
  const DcNode nd = nodes[blockIdx.y];
  const int z = blockIdx.z;
  DcWs w = item_ws(a, z);
  const int m = a.m, off = nd.off, n = nd.n1 + nd.n2;
  const int K = w.cnt[3 * off], nrot = w.cnt[3 * off + 2];
  const int lane = threadIdx.x & 31;
  const int pos = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (pos >= n) return;
  double* col = w.W + (size_t)(off + pos) * m + off;
  for (int r = lane; r < n; r += 32) col[r] = 0.0;
  __syncwarp();
  const int nD = w.cnt[3 * off + 1];
  const int src = w.colsrc[off + pos];
  if (src >= K || src < -nD) return;  // only reachable on non-finite input: leave the column zero
  if (src >= 0) {
    const int j = src;
    const double* dK = w.dK + off;
    const double dj = dK[w.orig[off + j]], tj = w.tauK[off + j];
    double s2 = 0.0;
    for (int i = lane; i < K; i += 32) {
      double v = w.zhat[off + i] * recip((dK[i] - dj) - tj);
      s2 += v * v;
    }
    s2 = warp_sum(s2);
    const double inv = 1.0 / sqrt(s2);
    for (int i = lane; i < K; i += 32) col[w.idxK[off + i]] = w.zhat[off + i] * recip((dK[i] - dj) - tj) * inv;
  } else {
    if (lane == 0) col[w.idxD[off + (-1 - src)]] = 1.0;
  }
  __syncwarp();
  if (lane == 0) {
    for (int r = nrot - 1; r >= 0; r--) {
      const int ia = w.ra[off + r], ib = w.rb[off + r];
      const double c = w.rc[off + r], sn = w.rs[off + r];
      const double xa = col[ia], xb = col[ib];
      col[ia] = c * xa + sn * xb;
      col[ib] = -sn * xa + c * xb;
    }
  }
}

// ------------------------------------------------------------------ host side

static void build_tree(DcPlan* p) {
  int m = p->m, depth = 0;
  while (((m + (1 << depth) - 1) >> depth) > DC_LEAF) depth++;
  p->depth = depth;
  // nodes per depth from the root down
  std::vector<std::vector<std::pair<int, int>>> seg(depth + 1);
  seg[0].push_back({0, m});
  for (int l = 0; l < depth; l++)
    for (auto& sg : seg[l]) {
      int n1 = sg.second / 2;
      seg[l + 1].push_back({sg.first, n1});
      seg[l + 1].push_back({sg.first + n1, sg.second - n1});
      p->splits.push_back(sg.first + n1);
    }
  for (auto& sg : seg[depth]) { p->leaves.push_back(sg.first); p->leaves.push_back(sg.second); }
  p->levels.resize(depth);
  for (int t = 0; t < depth; t++) {
    int l = depth - 1 - t;  // depth of the parents merged at step t
    DcLevel& L = p->levels[t];
    for (auto& sg : seg[l]) {
      int n1 = sg.second / 2;
      L.nodes.push_back({sg.first, n1, sg.second - n1});
      L.maxn = std::max(L.maxn, sg.second);
      L.maxhalf = std::max(L.maxhalf, sg.second - n1);
    }
  }
  std::sort(p->splits.begin(), p->splits.end());
}

DcPlan* dc_plan_create(int m, int count) {
  DcPlan* p = new DcPlan();
  p->m = m;
  p->count = count;
  build_tree(p);
  cudaMalloc(&p->d_leaves, sizeof(int) * std::max<size_t>(1, p->leaves.size()));
  cudaMemcpy(p->d_leaves, p->leaves.data(), sizeof(int) * p->leaves.size(), cudaMemcpyHostToDevice);
  cudaMalloc(&p->d_splits, sizeof(int) * std::max<size_t>(1, p->splits.size()));
  if (!p->splits.empty())
    cudaMemcpy(p->d_splits, p->splits.data(), sizeof(int) * p->splits.size(), cudaMemcpyHostToDevice);
  for (auto& L : p->levels) {
    cudaMalloc(&L.d_nodes, sizeof(DcNode) * L.nodes.size());
    cudaMemcpy(L.d_nodes, L.nodes.data(), sizeof(DcNode) * L.nodes.size(), cudaMemcpyHostToDevice);
    cudaMalloc(&L.d_gemm, sizeof(GemmDesc) * 2 * L.nodes.size() * count);
  }
  return p;
}

void dc_plan_destroy(DcPlan* p) {
  if (!p) return;
  cudaFree(p->d_leaves);
  cudaFree(p->d_splits);
  for (auto& L : p->levels) { cudaFree(L.d_nodes); cudaFree(L.d_gemm); }
  delete p;
}

size_t dc_workspace_bytes(const DcPlan* p) { return dc_item_bytes(p->m) * p->count; }

// Z buffer used at merge step t (input) is buf[t % 2]; leaves write buf[0]; the root
// writes buf[depth % 2], chosen to be the caller's Z.
static void build_gemm_lists(DcPlan* p, double* Z, long long sZ, void* work) {
  const int m = p->m;
  const size_t item = dc_item_bytes(m);
  for (int t = 0; t < p->depth; t++) {
    DcLevel& L = p->levels[t];
    std::vector<GemmDesc> h;
    for (int z = 0; z < p->count; z++) {
      DcWs w = dc_ws(static_cast<char*>(work) + z * item, m);
      double* buf[2];
      buf[p->depth % 2] = Z + z * sZ;
      buf[(p->depth + 1) % 2] = w.Zb;
      const double* in = buf[t % 2];
      double* out = buf[(t + 1) % 2];
      for (auto& nd : L.nodes) {
        const int off = nd.off, n = nd.n1 + nd.n2, s = off + nd.n1;
        GemmDesc g1{in + (size_t)off * m + off, w.W + (size_t)off * m + off, out + (size_t)off * m + off, nullptr,
                    nd.n1, n, nd.n1, m, m, m};
        GemmDesc g2{in + (size_t)s * m + s, w.W + (size_t)off * m + s, out + (size_t)s * m + off, nullptr, nd.n2, n,
                    nd.n2, m, m, m};
        h.push_back(g1);
        h.push_back(g2);
      }
    }
    cudaMemcpy(L.d_gemm, h.data(), sizeof(GemmDesc) * h.size(), cudaMemcpyHostToDevice);
  }
  p->zbound = Z;
  p->wbound = work;
  p->sZbound = sZ;
}

size_t dc_split_item_bytes(const DcPlan* p, int min_half, int S) {
  size_t b = 0;
  for (auto& L : p->levels)
    if (L.maxhalf >= min_half)
      for (auto& nd : L.nodes) {
        const int n = nd.n1 + nd.n2;
        b = std::max(b, ozaki_workspace_bytes(nd.n1, n, nd.n1, false, S));
        b = std::max(b, ozaki_workspace_bytes(nd.n2, n, nd.n2, false, S));
      }
  return b;
}

void dc_solve(DcPlan* p, double* d, double* e, long long sde, double* lam, double* Z, long long sZ, void* work,
              DevStatus* st, cudaStream_t s, Prof* prof, const DcSplit* sp) {
  const int m = p->m, cnt = p->count;
  if (p->zbound != Z || p->wbound != work || p->sZbound != sZ) {
    if (p->zbound) cudaStreamSynchronize(s);  // work in flight may still read the lists
    build_gemm_lists(p, Z, sZ, work);
  }
  const size_t item = dc_item_bytes(m);
  DcWs w0 = dc_ws(work, m);
  // lam ping-pong: leaves write lamA (item stride = item bytes / 8 doubles)
  const long long slam = (long long)(item / sizeof(double));
  double* lamBuf[2] = {w0.lamA, w0.lamB};
  double* zbuf0 = (p->depth % 2 == 0) ? Z : w0.Zb;
  const long long sZ0 = (p->depth % 2 == 0) ? sZ : slam;
  int tok = prof->begin();
  count_launch();
  dc_tear_kernel<<<cnt, 256, 0, s>>>(d, e, sde, p->d_splits, (int)p->splits.size());
  const int nleaves = (int)p->leaves.size() / 2;
  count_launch();
  dc_leaf_kernel<<<dim3(nleaves, cnt), 32, 0, s>>>(d, e, sde, lamBuf[0], slam, zbuf0, sZ0, m, p->d_leaves, st);
  prof->end(tok, PC_DC_LEAF, 0.0, 0.0);
  for (int t = 0; t < p->depth; t++) {
    DcLevel& L = p->levels[t];
    const int nn = (int)L.nodes.size();
    DcArgs a;
    a.m = m;
    a.sitem = (long long)item;
    a.ws = static_cast<char*>(work);
    a.e = e;
    a.sde = sde;
    a.lam = lamBuf[t % 2];
    a.lamNew = lamBuf[(t + 1) % 2];
    a.slam = slam;
    const bool in_is_Z = ((t % 2) == (p->depth % 2));
    a.Zc = in_is_Z ? Z : w0.Zb;
    a.sZ = in_is_Z ? sZ : slam;
    tok = prof->begin();
    count_launch();
    dc_merge_prep_kernel<<<dim3(nn, cnt), 1024, 0, s>>>(a, L.d_nodes);
    dim3 g1((L.maxn + 127) / 128, nn, cnt);
    count_launch();
    dc_secular_kernel<<<dim3((L.maxn + 7) / 8, nn, cnt), 256, 0, s>>>(a, L.d_nodes, st);
    count_launch();
    dc_zhat_kernel<<<dim3((L.maxn + 7) / 8, nn, cnt), 256, 0, s>>>(a, L.d_nodes);
    count_launch();
    dc_colmap_kernel<<<g1, 128, 0, s>>>(a, L.d_nodes);
    count_launch();
    dc_buildw_kernel<<<dim3((L.maxn + 7) / 8, nn, cnt), 256, 0, s>>>(a, L.d_nodes);
    prof->end(tok, PC_DC_SECULAR, 0.0, 0.0);
    double gfl = 0.0, gby = 0.0;
    for (auto& nd : L.nodes) {
      const double nn1 = nd.n1, nn2 = nd.n2, n = nn1 + nn2;
      gfl += 2.0 * (nn1 * nn1 + nn2 * nn2) * n;
      gby += 8.0 * (nn1 * nn1 + nn2 * nn2 + 2.0 * n * n);
    }
    if (sp && sp->per > 0 && L.maxhalf >= sp->min_half) {
      // large merges: per node, exact split-bf16 products batched over the items
      tok = prof->begin();
      const long long sin = in_is_Z ? sZ : slam, sout = in_is_Z ? slam : sZ;
      double* in0 = in_is_Z ? Z : w0.Zb;
      double* out0 = in_is_Z ? w0.Zb : Z;
      bool ok = true;
      for (auto& nd : L.nodes) {
        const int off = nd.off, n = nd.n1 + nd.n2, sft = off + nd.n1;
        for (int z0 = 0; z0 < cnt && ok; z0 += sp->per) {
          const int c = std::min(sp->per, cnt - z0);
          const DcWs wz = dc_ws(static_cast<char*>(work) + (size_t)z0 * item, m);
          const long long iz = (long long)z0 * sin, oz = (long long)z0 * sout;
          ok = ozaki_gemm<double>(OP_N, OP_T, nd.n1, n, nd.n1, 1.0, in0 + iz + (size_t)off * m + off, m, sin,
                                  wz.W + (size_t)off * m + off, m, slam, 0.0, out0 + oz + (size_t)off * m + off, m,
                                  sout, c, 0, sp->S, sp->work, st, s, nullptr, 0, nullptr, sp->wait) &&
               ozaki_gemm<double>(OP_N, OP_T, nd.n2, n, nd.n2, 1.0, in0 + iz + (size_t)sft * m + sft, m, sin,
                                  wz.W + (size_t)off * m + sft, m, slam, 0.0, out0 + oz + (size_t)sft * m + off, m,
                                  sout, c, 0, sp->S, sp->work, st, s, nullptr, 0, nullptr, sp->wait);
        }
      }
      prof->end(tok, PC_OZAKI, gfl * cnt, gby * cnt);
      if (ok) continue;
    }
    tok = prof->begin();
    GemmBatch gb{};
    gb.list = L.d_gemm;
    gb.count = 2 * nn * cnt;
    gb.opA = OP_N;
    gb.opB = OP_T;
    gb.alpha = 1.0;
    gb.beta = 0.0;
    gemm<double>(gb, L.maxhalf, L.maxn, s);
    prof->end(tok, PC_DC_GEMM, gfl * cnt, gby * cnt);
  }
  // final eigenvalues
  double* lamFinal = lamBuf[p->depth % 2];
  copy2d<double>(lam, m, sde, lamFinal, m, slam, 1, m, cnt, s);
}

}  // namespace gks
