// Fermi-Dirac occupations, chemical potential and band energy (paper Sec. 3.1 Part 3,
// Sec. 3.2 Part 4; occupation f_i of Sec. 2).
//
//   f(x) = 1 / (1 + e^x),  x = (eps - mu) / kT, evaluated as e^-x/(1+e^-x) for x > 0;
//   N(mu) = sum_k w_k g_s sum_i f((eps_ki - mu)/kT) is increasing in mu, and mu solves
//   N(mu) = n_elec by bisection on [min eps - 1, max eps + 1] (stop when the bracket is
//   below 4u max(1, |mu|), at most 200 halvings);
//   E_band = sum_k w_k g_s sum_i f_ki eps_ki.
// Also writes kscale = g_s f (zero where f < f_cut) and n_rho(k) = #{i : f_ki >= f_cut},
// the leading columns kept in rho (eps ascending, so f is non-increasing in i).
#include <algorithm>

#include "dense.h"

namespace gks {

__device__ __forceinline__ double fermi_fn(double x) {
  if (x > 0.0) {
    double t = exp(-x);
    return t / (1.0 + t);
  }
  return 1.0 / (1.0 + exp(x));
}

// One cluster of kOccC CTAs x 128 threads per system; system q owns k-points [q*nk, (q+1)*nk).
// The FP64 pipe bounds an evaluation of N(mu) (about 40 operations per eigenvalue and SM with
// 1.7 per clock), so it is spread over the cluster's SMs, and eigenvalues more than 40 kT
// below mu (f = 1 exactly) or 60 kT above (f < 1e-26) take no exponential.  The sum is the one
// of 1024 threads in one CTA (thread tid of rank r stands for thread 128 r + tid, their 32 warp
// sums combined in one shuffle tree), so the halvings do not depend on the cluster.  The
// halvings far from mu need no FP64 sum: N is evaluated in single precision first (three
// FP64 operations per eigenvalue), and where that differs from n_elec by more than its error
// bound it decides.  Then Newton's iteration finds the root to its rounding, and a halving
// point further from it than that is decided by the side it lies on (N is increasing); where
// N is too flat for that (mu in a gap) every halving is evaluated.  6656 eigenvalues: 3.9 ms on
// one CTA, 0.47 ms on the cluster with every halving in FP64, 0.20 ms here.
constexpr int kOccC = 8, kOccT = 128;
__device__ __forceinline__ void occ_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// Every warp's value into slot 4 rank + warp of all CTAs of the cluster.
template <bool BAR = true>
__device__ __forceinline__ void occ_share(double* slots, int rank, double v) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane < kOccC)
    asm volatile(
        "{\n .reg .b32 ra;\n mapa.shared::cluster.u32 ra, %0, %1;\n st.shared::cluster.f64 [ra], %2;\n}\n" ::"r"(
            (unsigned)__cvta_generic_to_shared(slots + 4 * rank + warp)),
        "r"(lane), "d"(v)
        : "memory");
  if (BAR) occ_barrier();
}

__global__ void __launch_bounds__(kOccT) fermi_mu_kernel(const double* eps, int m, int nk, const double* w, double gs,
                                                         double kT, double n_elec, double f_cut, double* occ,
                                                         double* kscale, double* mu_out, double* e_band, int* nrho,
                                                         DevStatus* st) {
  __shared__ double slots[2][32], slots2[32];
  const int q = blockIdx.y, rank = blockIdx.x, lane = threadIdx.x & 31;
  const int tid = rank * kOccT + threadIdx.x;
  constexpr int nt = kOccC * kOccT;
  const long long base = (long long)q * nk * m;
  eps += base;
  occ += base;
  kscale += base;
  const long long tot = (long long)nk * m;
  double lo, hi;
  {
    double vmin = 1e300, vmax = -1e300;
    for (long long t = tid; t < tot; t += nt) { vmin = fmin(vmin, eps[t]); vmax = fmax(vmax, eps[t]); }
    for (int o = 16; o > 0; o >>= 1) {
      vmin = fmin(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
      vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
    }
    occ_barrier();  // every CTA of the cluster runs
    occ_share(slots[0], rank, vmin);
    occ_share(slots[1], rank, vmax);
    vmin = slots[0][lane];
    vmax = slots[1][lane];
    for (int o = 16; o > 0; o >>= 1) {
      vmin = fmin(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
      vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
    }
    lo = vmin - 1.0;
    hi = vmax + 1.0;
    occ_barrier();  // the slots have been read
  }
  double wsum = 0.0;
  for (int k = 0; k < nk; k++) wsum += w[k];
  const bool bad = !(kT > 0.0) || !(n_elec > 0.0) || !(n_elec < gs * m * wsum) || !isfinite(lo) || !isfinite(hi);
  if (bad) {  // the same in every CTA
    if (tid == 0) set_status(st, ST_EINVAL, 0);
    return;
  }
  const int k0 = tid / m, dk = nt / m, r0 = tid % m, dr = nt % m;  // k-point and row of t = tid + i nt
  // sum over the system of fn(t, k), by every thread
  int phase = 0;
  auto total = [&](auto fn, double* second = nullptr) -> double {  // second: a sum fn keeps itself
    double s = 0.0;
    int k = k0, r = r0;
    for (long long t = tid; t < tot; t += nt) {
      s += fn(t, k);
      k += dk;
      r += dr;
      if (r >= m) {
        r -= m;
        k++;
      }
    }
    s = warp_sum(s);
    phase ^= 1;
    if (second) {
      occ_barrier();  // its slots have been read
      occ_share<false>(slots2, rank, warp_sum(*second));
    }
    occ_share(slots[phase], rank, s);
    if (second) *second = warp_sum(slots2[lane]);
    return warp_sum(slots[phase][lane]);
  };
  const double u = 1.1102230246251565e-16;
  // |error| of the single-precision N: f within 2e-7 each (the argument's rounding included:
  // |x| f (1 - f) 2^-24 < 0.3 2^-24), their sum within 100 additions' roundings per lane
  const double rkT = 1.0 / kT;
  double far = 1e-4 * gs * m * wsum;
  double root = 0.0, near = 1e300;  // halving points further than near from root need no sum
  for (int it = 0; it < 200; it++) {
    double mid = 0.5 * (lo + hi);
    if (hi - lo <= 4.0 * u * fmax(1.0, fabs(mid))) break;
    if (far > 0.0) {
      const double s = gs * total([&](long long t, int k) -> double {
        return w[k] * (double)(1.0f / (1.0f + __expf((float)((eps[t] - mid) * rkT))));
      });
      if (s < n_elec - far) { lo = mid; continue; }
      if (s > n_elec + far) { hi = mid; continue; }
      far = 0.0;  // closer than that from here on
      double x = mid, dx = hi - lo;
      for (int nt2 = 0; nt2 < 6 && x > lo && x < hi; nt2++) {
        double d = 0.0;
        const double s2 = total([&](long long t, int k) -> double {
          const double f = fermi_fn((eps[t] - x) * rkT);
          d += w[k] * f * (1.0 - f);
          return w[k] * f;
        }, &d);
        const double slope = gs * d * rkT, noise = 64.0 * u * n_elec / slope;  // sums round by u n_elec
        const double step = (n_elec - gs * s2) / slope;
        x += step;
        dx = fabs(step);
        if (!(dx > 4.0 * noise + 4.0 * u)) {
          const double reach = 4.0 * (dx + noise) + 16.0 * u * fmax(1.0, fabs(x));
          if (x > lo && x < hi && reach < 0.125 * (hi - lo)) {
            root = x;
            near = reach;
          }
          break;
        }
      }
    }
    if (fabs(mid - root) > near) {
      if (mid < root) lo = mid;
      else hi = mid;
      continue;
    }
    const double one = mid - 40.0 * kT, none = mid + 60.0 * kT;
    const double s = gs * total([&](long long t, int k) -> double {
      const double e = eps[t];
      return e < one ? w[k] : e > none ? 0.0 : w[k] * fermi_fn((e - mid) / kT);
    });
    if (s < n_elec) lo = mid;
    else hi = mid;
  }
  const double mu = 0.5 * (lo + hi);
  const double eb = total([&](long long t, int k) -> double {
    const double f = fermi_fn((eps[t] - mu) / kT);
    occ[t] = f;
    kscale[t] = (f >= f_cut) ? gs * f : 0.0;
    return w[k] * gs * f * eps[t];
  });
  if (tid == 0) {
    mu_out[q] = mu;
    e_band[q] = eb;
  }
  for (int k = tid; k < nk; k += nt) {
    // f non-increasing along the ascending eigenvalues: binary search for the last kept
    // (written by this cluster before the barrier of the last sum)
    const double* fk = occ + (long long)k * m;
    int lo_i = 0, hi_i = m;
    while (lo_i < hi_i) {
      int mid = (lo_i + hi_i) >> 1;
      if (__ldcg(fk + mid) >= f_cut) lo_i = mid + 1;
      else hi_i = mid;
    }
    nrho[(long long)q * nk + k] = lo_i;
  }
  occ_barrier();  // no CTA leaves while another may still write to its slots
}

void fermi_mu(const double* eps, int m, int nk, const double* w, double gs, double kT, double n_elec, double f_cut,
              double* occ, double* kscale, double* mu, double* e_band, int* nrho, DevStatus* st, int nsys,
              cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  cfg.gridDim = dim3(kOccC, nsys);
  cfg.blockDim = dim3(kOccT);
  cfg.stream = s;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = kOccC;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  count_launch();
  cudaLaunchKernelEx(&cfg, fermi_mu_kernel, eps, m, nk, w, gs, kT, n_elec, f_cut, occ, kscale, mu, e_band, nrho, st);
}

__global__ void expand_weights_kernel(const double* w, int nk, int rep, double* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nk * rep) return;
  const int k = t / rep;
  out[t] = w ? w[k] : 1.0 / nk;
}

void expand_weights(const double* w, int nk, int rep, double* out, cudaStream_t s) {
  count_launch();
  expand_weights_kernel<<<(nk * rep + 255) / 256, 256, 0, s>>>(w, nk, rep, out);
}

__global__ void clamp_nrho_kernel(int* nrho, int nk, int cols, DevStatus* st, int st_stride) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nk) return;
  if (nrho[k] > cols) {
    set_status(st ? st + (long long)k * st_stride : nullptr, ST_EINVAL, nrho[k]);
    nrho[k] = cols;
  }
}

void clamp_nrho(int* nrho, int nk, int cols, DevStatus* st, int st_stride, cudaStream_t s) {
  count_launch();
  clamp_nrho_kernel<<<(nk + 255) / 256, 256, 0, s>>>(nrho, nk, cols, st, st_stride);
}

__global__ void mul_elem_kernel(const double* a, const double* b, double* out, long long n) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = a[t] * b[t];
}

void mul_elem(const double* a, const double* b, double* out, long long n, cudaStream_t s) {
  count_launch();
  const long long blocks = std::min<long long>((n + 255) / 256, 4096);
  mul_elem_kernel<<<(int)std::max<long long>(blocks, 1), 256, 0, s>>>(a, b, out, n);
}

}  // namespace gks
