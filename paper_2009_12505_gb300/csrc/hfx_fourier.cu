// The two steps next to the exchange build, in FP64 on CUDA cores:
//
// Real-space density matrix from Kohn-Sham eigenvectors (Eq. DM_realspace).
// With the block key (K, L, n) = sites (K, 0) and (L, n), so that
// R_K - R_L = -R_n,
//   D_{Kk,Ll}(n) = (1/N_k) sum_q sum_b f_qb c_q[Kk][b] conj(c_q[Ll][b])
//                  exp(2 pi i kappa_q . n),
// kappa_q the q-th k point in fractional reciprocal coordinates.  D is real
// when the k set and the eigenvectors are time-reversal symmetric; the largest
// |imaginary part| is reported so a caller can check that.
//
// Exchange matrix at k points (Eq. Ham_rs2kspace):
//   Sigma_{Ii,Jj}(k) = sum_{keys (I, J, n)} exp(2 pi i kappa . n) Sigma(I, J, n)_{ij}.
//
// Both are gathers: each output element is a fixed-order sum, so results are
// deterministic.  The phases come from sincospi of 2 kappa . n, computed once
// per (k point, key) in shared memory: in FP64 (1/64 of the FP32 rate here) one
// sincospi costs about twenty multiply-adds.
#include <cuda_runtime.h>

#include "hfx_internal.h"

namespace {

constexpr int DN_BANDS = 16;           // bands staged at a time
constexpr int DN_STR = DN_BANDS + 1;   // staged row stride: rows start in different banks

// One block per group: an atom pair (K, L), K <= L, and up to DENSITY_IMAGES
// of its keys.  The band sum z_q[k][l] = sum_b f c_K conj(c_L) does not depend
// on n, so it is formed once per k point and turned by each key's phase; a key
// (L, K, n) takes conj(z)^T.  It is bound by the FP64 units: 4 nbands + 4
// images multiply-adds per element and k point, from shared memory, where one
// block per key took 6 nbands for every key.  64-atom Si-like cell (832
// orbitals, 160 bands, 8 k points, 7872 keys): the whole call 27.4 ms before
// (kernel 20.7 ms), 5.65 ms now.
__global__ void __launch_bounds__(256) k_density(
    int nk, const double *__restrict__ kfrac, int nb, int nbands,
    const double2 *__restrict__ coef, const double *__restrict__ occ,
    const DensityGroup *__restrict__ groups, const DensityKey *__restrict__ dkeys,
    const int32_t *__restrict__ aoff, const int32_t *__restrict__ nao, double *__restrict__ out,
    unsigned long long *__restrict__ maxim) {
  __shared__ double2 sK[HFX_MAX_NAO * DN_STR], sL[HFX_MAX_NAO * DN_STR];
  __shared__ double2 sph[2][DENSITY_IMAGES];
  const DensityGroup gr = groups[blockIdx.x];
  const int nK = nao[gr.K], nL = nao[gr.L];
  const int64_t aK = aoff[gr.K], aL = aoff[gr.L];
  const double inv = 1.0 / nk;
  unsigned long long mx = 0;
  for (int t0 = 0; t0 < nK * nL; t0 += blockDim.x) {
    const int t = t0 + threadIdx.x;
    const bool live = t < nK * nL;
    const int k = live ? t / nL : 0, l = live ? t - k * nL : 0;
    double re[DENSITY_IMAGES], im[DENSITY_IMAGES];
#pragma unroll
    for (int j = 0; j < DENSITY_IMAGES; ++j) re[j] = im[j] = 0.0;
    for (int q = 0; q < nk; ++q) {
      // written two k points after the last read of this half: a barrier lies between
      if (threadIdx.x < gr.count) {
        const DensityKey &e = dkeys[gr.first + threadIdx.x];
        double s, c;
        sincospi(2.0 * (kfrac[3 * q] * e.n[0] + kfrac[3 * q + 1] * e.n[1] +
                        kfrac[3 * q + 2] * e.n[2]), &s, &c);
        sph[q & 1][threadIdx.x] = make_double2(c, e.tr ? -s : s);
      }
      double zr = 0.0, zi = 0.0;
      for (int b0 = 0; b0 < nbands; b0 += DN_BANDS) {
        __syncthreads();
        for (int i = threadIdx.x; i < (nK + nL) * DN_BANDS; i += blockDim.x) {
          const int r = i / DN_BANDS, b = i - r * DN_BANDS;
          const bool isK = r < nK;
          double2 v = make_double2(0.0, 0.0);
          if (b0 + b < nbands) {
            v = coef[((int64_t)q * nb + (isK ? aK + r : aL + r - nK)) * nbands + b0 + b];
            if (isK) {
              const double f = occ[(int64_t)q * nbands + b0 + b];
              v.x *= f;
              v.y *= f;
            }
          }
          (isK ? sK + r * DN_STR : sL + (r - nK) * DN_STR)[b] = v;
        }
        __syncthreads();
        if (live) {
#pragma unroll
          for (int b = 0; b < DN_BANDS; ++b) {
            const double2 x = sK[k * DN_STR + b], y = sL[l * DN_STR + b];
            zr = fma(x.x, y.x, zr);
            zi = fma(x.y, y.x, zi);
            zr = fma(x.y, y.y, zr);
            zi = fma(-x.x, y.y, zi);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < DENSITY_IMAGES; ++j)
        if (j < gr.count) {
          // a transposed key has conj(z) e^{i phi}: its conjugate is z e^{-i phi}
          const double2 ph = sph[q & 1][j];
          re[j] += zr * ph.x - zi * ph.y;
          im[j] += zr * ph.y + zi * ph.x;
        }
    }
#pragma unroll
    for (int j = 0; j < DENSITY_IMAGES; ++j)
      if (live && j < gr.count) {
        const DensityKey &e = dkeys[gr.first + j];
        out[e.off + (e.tr ? l * nK + k : t)] = re[j] * inv;
        mx = max(mx, (unsigned long long)__double_as_longlong(fabs(im[j] * inv)));
      }
    __syncthreads();
  }
  // nonnegative doubles order as their bit patterns, with NaN (an overflowed
  // sum) above them all
  for (int o = 16; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) atomicMax(maxim, mx);
}

constexpr int SK_KEYS = 256;  // keys whose phases are held at a time

// One block per (k point, I, J); the keys of (I, J) are the sorted range
// [lower_bound(I, J), ...) of the build's key list.  Per element two
// multiply-adds a key: the phases (one sincospi per key, not per element and
// key) come from shared memory.  64-atom cell with 8 k points: the whole call
// 26.2 ms before (kernel 1.51 ms, most of it copies in the binding), 4.96 ms
// now.
__global__ void __launch_bounds__(256) k_sigma_k(
    int nk, const double *__restrict__ kfrac, int natoms, const int32_t *__restrict__ aoff,
    const int32_t *__restrict__ nao, int64_t nkeys, const uint64_t *__restrict__ skeys,
    const int64_t *__restrict__ soffs, const double *__restrict__ sigma, int64_t nb,
    double2 *__restrict__ out) {
  __shared__ double2 ph[SK_KEYS];
  const int64_t bid = blockIdx.x;
  const int q = (int)(bid / ((int64_t)natoms * natoms));
  const int64_t ij = bid - (int64_t)q * natoms * natoms;
  const int I = (int)(ij / natoms), J = (int)(ij - (int64_t)I * natoms);
  // the keys of (I, J): [lo, end)
  auto bound = [&](uint64_t k) {
    int64_t lo = 0, hi = nkeys;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (skeys[mid] < k) lo = mid + 1; else hi = mid;
    }
    return lo;
  };
  const int64_t lo = bound(hk_pack(I, J, -128, -128, -128));
  const int64_t end = bound(hk_pack(I, J, -128, -128, -128) + (1ull << 24));
  const int nI = nao[I], nJ = nao[J], n = nI * nJ;
  const double kx = kfrac[3 * q], ky = kfrac[3 * q + 1], kz = kfrac[3 * q + 2];
  const int64_t s0 = lo < end ? soffs[lo] : 0;  // blocks of one pair are consecutive
  for (int t0 = 0; t0 < n; t0 += blockDim.x) {
    const int t = t0 + threadIdx.x;
    double re = 0.0, im = 0.0;
    for (int64_t e0 = lo; e0 < end; e0 += SK_KEYS) {
      const int m = (int)min((int64_t)SK_KEYS, end - e0);
      __syncthreads();
      if (threadIdx.x < m) {
        int32_t k[5];
        hk_unpack(skeys[e0 + threadIdx.x], k);
        double s, c;
        sincospi(2.0 * (kx * k[2] + ky * k[3] + kz * k[4]), &s, &c);
        ph[threadIdx.x] = make_double2(c, s);
      }
      __syncthreads();
      if (t < n) {
        const double *v = sigma + s0 + (e0 - lo) * n + t;
#pragma unroll 4
        for (int e = 0; e < m; ++e) {
          const double x = v[(int64_t)e * n];
          re += x * ph[e].x;
          im += x * ph[e].y;
        }
      }
    }
    if (t < n) {
      const int i = t / nJ, j = t - i * nJ;
      out[((int64_t)q * nb + aoff[I] + i) * nb + aoff[J] + j] = make_double2(re, im);
    }
  }
}

}  // namespace

cudaError_t launch_density(int nk, const double *kfrac, int nb, int nbands, const double *coef,
                           const double *occ, int64_t ngroups, const DensityGroup *groups,
                           const DensityKey *dkeys, const int32_t *aoff, const int32_t *nao,
                           double *out, unsigned long long *maxim, cudaStream_t st) {
  if (ngroups <= 0) return cudaSuccess;
  k_density<<<(unsigned)ngroups, 256, 0, st>>>(nk, kfrac, nb, nbands,
                                               reinterpret_cast<const double2 *>(coef), occ,
                                               groups, dkeys, aoff, nao, out, maxim);
  return cudaGetLastError();
}

cudaError_t launch_sigma_k(int nk, const double *kfrac, int natoms, const int32_t *aoff,
                           const int32_t *nao, int64_t nkeys, const uint64_t *skeys,
                           const int64_t *soffs, const double *sigma, int64_t nb, double *out,
                           cudaStream_t st) {
  const int64_t nblk = (int64_t)nk * natoms * natoms;
  if (nblk <= 0) return cudaSuccess;
  k_sigma_k<<<(unsigned)nblk, 256, 0, st>>>(nk, kfrac, natoms, aoff, nao, nkeys, skeys, soffs,
                                            sigma, nb, reinterpret_cast<double2 *>(out));
  return cudaGetLastError();
}
