// Power spectrum and normalised descriptor (Eq. 09 and Sec. I), one warp per atom.
//   p[c1][c2][l] = sum_{m=-l..l} c[c1][lm] c[c2][lm]   (real Y_lm: same value as Eq. 09)
//   packed entry (c1 <= c2, l) = p times sqrt(2) when c1 != c2;  q = p / |p|.
#include <algorithm>

#include "internal.h"
#include "size_rules.h"

// Shared-memory reads bound this kernel, so channel rows are padded to 16-byte steps (an odd
// number of them) and read 16 bytes at a time: the lanes of a warp hold up to 32 channel pairs
// but only a few distinct rows, so one such read costs the wavefronts of its distinct rows (3 for
// both rows at 10 channels) instead of one per 4-byte read (8 for the same data).  The products
// of one l are summed in the order of m as two partial sums, even and odd.  100,000 atoms, 10
// channels, l_max 10: 334 -> 320 us; the 256-structure batch: 210 -> 181 us (L1 wavefronts 72 % on 16,000
// atoms of the first recipe, 63 % on 64 structures of the second).
template <typename T> struct Vec16;
template <> struct Vec16<float> { using type = float4; static constexpr int N = 4; };
template <> struct Vec16<double> { using type = double2; static constexpr int N = 2; };

// LC: the basis class's bound on l_max (the (l, m) loops unrolled to it, l_max <= LC at run time)
//
// Optional GAP operand of the mixed path (op.a16 set): u = (q - qbar) / |q - qbar| in FP16 ([hi]
// or [hi | hi | lo] by op.terms), |q - qbar| and qbar.(q - qbar), summed in the operation order
// of prep_atoms_kernel (gap_tc.cu) while q passes, q - qbar kept in shared memory for u.
template <typename T, int LC>
__global__ void powspec_kernel(const T* __restrict__ c, int n_atoms, int nch, int lmax,
                               int per_warp, T* q, T* pnorm, GapOperand op) {
  pdl_begin();
  // one warp per atom: c staged in shared memory, each lane owns whole channel pairs
  // (c1 <= c2) and all their l, the unnormalised p stays in shared memory until |p| is known
  using V = Vec16<T>;
  constexpr int VN = V::N;
  constexpr int LT = (LC + 1) * (LC + 1);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  T* cs = reinterpret_cast<T*>(smem_raw) + (size_t)warp * per_warp;
  const int L = (lmax + 1) * (lmax + 1), RS = powspec_row(L, sizeof(T));
  const int lp1 = lmax + 1;
  const int npair = nch * (nch + 1) / 2;
  const int D = npair * lp1;
  T* ps = cs + nch * RS;
  const T SQRT2 = (T)1.4142135623730951;
  const int wpb = blockDim.x >> 5;
  for (int atom = blockIdx.x * wpb + warp; atom < n_atoms; atom += gridDim.x * wpb) {
    const T* ci = c + (size_t)atom * nch * L;
    __syncwarp();
#pragma unroll 2
    for (int ch = 0; ch < nch; ++ch) {
#pragma unroll
      for (int k = 0; k < (LT + 31) / 32; ++k)
        if (lane + 32 * k < L) cs[ch * RS + lane + 32 * k] = __ldg(ci + ch * L + lane + 32 * k);
    }
    __syncwarp();
    T ss = 0;
    for (int pc = lane; pc < npair; pc += 32) {
      int c1 = 0, rem = pc;
      while (rem >= nch - c1) {
        rem -= nch - c1;
        ++c1;
      }
      const int c2 = c1 + rem;
      const typename V::type* a = reinterpret_cast<const typename V::type*>(cs + c1 * RS);
      const typename V::type* b = reinterpret_cast<const typename V::type*>(cs + c2 * RS);
      const T f = c1 != c2 ? SQRT2 : T(1);
      T* out = ps + pc * lp1;
      T av[VN], bv[VN];
#pragma unroll
      for (int l = 0; l <= LC; ++l) {
        if (l <= lmax) {
          T v0 = 0, v1 = 0;
#pragma unroll
          for (int m = 0; m <= 2 * l; ++m) {
            const int lm = l * l + m;
            if (lm % VN == 0) {
              *reinterpret_cast<typename V::type*>(av) = a[lm / VN];
              *reinterpret_cast<typename V::type*>(bv) = b[lm / VN];
            }
            if (m & 1) v1 = fma(av[lm % VN], bv[lm % VN], v1);
            else v0 = fma(av[lm % VN], bv[lm % VN], v0);
          }
          const T v = (v0 + v1) * f;
          out[l] = v;
          ss += v * v;
        }
      }
    }
    ss = warp_sum(ss);
    const T norm = sqrt(ss);
    if (lane == 0) pnorm[atom] = norm;
    const T inv = T(1) / norm;
    __syncwarp();
    T* qi = q + (size_t)atom * D;
    if (sizeof(T) == 4 && op.a16) {
      float s2 = 0.f, dq = 0.f;
      for (int k = lane; k < D; k += 32) {
        const T v = ps[k] * inv;
        qi[k] = v;
        const float qb = op.qbar[k], t = (float)v - qb;
        s2 = fmaf(t, t, s2);
        dq = fmaf(t, qb, dq);
        ps[k] = (T)t;
      }
      s2 = warp_sum(s2);
      dq = warp_sum(dq);
      const float nn = sqrtf(s2);
      const float iv = nn > 0.f ? 1.f / nn : 0.f;
      __syncwarp();
      __half* row = op.a16 + (size_t)atom * op.terms * op.dp;
      for (int k = 2 * lane; k < op.dp; k += 64) {  // (dp is even: a multiple of 64)
        const float u0 = k < D ? (float)ps[k] * iv : 0.f, u1 = k + 1 < D ? (float)ps[k + 1] * iv : 0.f;
        const __half2 hi = __floats2half2_rn(u0, u1);
        *reinterpret_cast<__half2*>(row + k) = hi;
        if (op.terms == 3) {
          *reinterpret_cast<__half2*>(row + op.dp + k) = hi;
          *reinterpret_cast<__half2*>(row + 2 * op.dp + k) =
              __floats2half2_rn(u0 - __low2float(hi), u1 - __high2float(hi));
        }
      }
      if (lane == 0) {
        op.nrm[atom] = nn;
        op.uq[atom] = dq;
      }
    } else {
      for (int k = lane; k < D; k += 32) qi[k] = ps[k] * inv;
    }
  }
}

template <typename T, int LC>
static cudaError_t launch_powspec(const T* c, int n_atoms, int nch, int lmax, T* q, T* pnorm, cudaStream_t st,
                                  const GapOperand& op) {
  if (n_atoms == 0) return cudaSuccess;
  const PowspecShape y = powspec_shape(nch, lmax, sizeof(T));
  const int wpb = y.warps, per_warp = y.per_warp;
  if (wpb < 1) return cudaErrorInvalidConfiguration;
  const size_t smem = (size_t)per_warp * sizeof(T) * wpb;
  auto kern = powspec_kernel<T, LC>;
  cudaError_t e = sg_set_smem<powspec_kernel<T, LC>>(smem);
  if (e != cudaSuccess) return e;
  const int sms = sg_sm_count(), per_sm = sg_blocks_per_sm<powspec_kernel<T, LC>>(wpb * 32, smem);
  long long grid = (long long)sms * per_sm;
  const long long need = (n_atoms + wpb - 1) / wpb;
  if (grid > need) grid = need;
  sg_launch(kern, (unsigned)grid, wpb * 32, smem, st, c, n_atoms, nch, lmax, per_warp, q, pnorm, op);
  ++sg_kernel_launches;
  return cudaGetLastError();
}

template <typename T>
cudaError_t sg_power_spectrum(const T* c, int n_atoms, int nch, int lmax, int lc, T* q, T* pnorm, cudaStream_t st,
                              const GapOperand& op) {
  if (lmax > lc) return cudaErrorInvalidValue;
  switch (lc) {
    case 6: return launch_powspec<T, 6>(c, n_atoms, nch, lmax, q, pnorm, st, op);
    case 8: return launch_powspec<T, 8>(c, n_atoms, nch, lmax, q, pnorm, st, op);
    case 10: return launch_powspec<T, 10>(c, n_atoms, nch, lmax, q, pnorm, st, op);
    case 12: return launch_powspec<T, 12>(c, n_atoms, nch, lmax, q, pnorm, st, op);
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t sg_power_spectrum<float>(const float*, int, int, int, int, float*, float*, cudaStream_t,
                                              const GapOperand&);
template cudaError_t sg_power_spectrum<double>(const double*, int, int, int, int, double*, double*, cudaStream_t,
                                               const GapOperand&);
