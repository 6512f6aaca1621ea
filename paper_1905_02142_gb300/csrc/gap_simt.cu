// GAP model on CUDA cores (FP64 path, and the FP32 reference variant of the mixed path).
//   S = Q Qs^T,  eps_i = sum_s alpha_s S_is^zeta   (Sec. IV.A, SOAP kernel of Sec. I)
//   kp_is = zeta alpha_s S_is^(zeta-1),  g = kp Qs = dE/dq   (adjoint of the above)
// Register-tiled GEMM.  FP64 instructions bound it (about two lanes per SM and clock), so a
// call's time is that of the SM with the most output elements: 64 x 64 tiles where they fill
// the GPU evenly, 32 x 32 or 32 x 16 where few 64 x 64 tiles would leave SMs without work
// (1000 atoms x 500 rows, D = 324: forward 365 -> 308 us, backward 526 -> 335 us; 310 us of
// FP64 pipe each).
#include "internal.h"
#include "size_rules.h"

#define GB_K 16

template <typename T> static SimtTile pick_tile(int n, int m) {
  if (sizeof(T) == 4) return {64, 64};  // (FP32: the allocation-free entry point's fixed layout)
  return simt_tile_f64(n, m, sg_sm_count());
}

template <typename T> int sg_gap_tiles(int n, int m) {
  const SimtTile t = pick_tile<T>(n, m);
  return (m + t.n - 1) / t.n;
}
template int sg_gap_tiles<float>(int, int);
template int sg_gap_tiles<double>(int, int);

template <typename T> __device__ __forceinline__ T kpow(T s, int izeta, T zeta) {
  if (izeta > 0) {
    T o = s;
    for (int k = 1; k < izeta; ++k) o *= s;
    return o;
  }
  return pow(s > T(0) ? s : T(0), zeta);
}

// MODE 0: C = A B^T (A [M,K], B [N,K]) with the GAP forward epilogue
// MODE 1: C = A B   (A [M,K], B [K,N]) plain store
template <typename T, int MODE, int TM, int TN, int RM, int RN>
__global__ void __launch_bounds__(TM / RM * (TN / RN))
gemm_kernel(const T* __restrict__ A, const T* __restrict__ B, int M, int N, int K,
            const T* __restrict__ alpha, int izeta, T zeta, T* eps_part, int n_tiles, T* out,
            int ldo) {
  pdl_begin();
  constexpr int TX = TN / RN, TY = TM / RM, THREADS = TX * TY;
  static_assert(TX == 16 || TX == 8, "the row sums shuffle over the TX threads of a row");
  __shared__ T As[GB_K][TM + 4];
  __shared__ T Bs[GB_K][TN + 4];
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int row0 = blockIdx.y * TM, col0 = blockIdx.x * TN;
  T acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = 0;
  for (int k0 = 0; k0 < K; k0 += GB_K) {
#pragma unroll
    for (int e = tid; e < TM * GB_K; e += THREADS) {  // A tile: TM rows x 16 k
      const int r = e >> 4, kk = e & 15, gr = row0 + r, gk = k0 + kk;
      As[kk][r] = (gr < M && gk < K) ? A[(size_t)gr * K + gk] : T(0);
    }
#pragma unroll
    for (int e = tid; e < TN * GB_K; e += THREADS) {
      if (MODE == 0) {  // B tile: TN rows x 16 k
        const int r = e >> 4, kk = e & 15, gc = col0 + r, gk = k0 + kk;
        Bs[kk][r] = (gc < N && gk < K) ? B[(size_t)gc * K + gk] : T(0);
      } else {          // B tile: 16 k x TN columns
        const int kb = e / TN, c = e % TN, gkb = k0 + kb, gc = col0 + c;
        Bs[kb][c] = (gkb < K && gc < N) ? B[(size_t)gkb * N + gc] : T(0);
      }
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GB_K; ++kk) {
      T a[RM], b[RN];
#pragma unroll
      for (int i = 0; i < RM; ++i) a[i] = As[kk][ty + TY * i];
#pragma unroll
      for (int j = 0; j < RN; ++j) b[j] = Bs[kk][tx + TX * j];
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  if (MODE == 0) {
#pragma unroll
    for (int i = 0; i < RM; ++i) {
      const int gr = row0 + ty + TY * i;
      T part = 0;
#pragma unroll
      for (int j = 0; j < RN; ++j) {
        const int gc = col0 + tx + TX * j;
        if (gr < M && gc < N) {
          const T s = acc[i][j], al = alpha[gc];
          const T sz1 = (izeta == 1) ? T(1) : kpow(s, izeta > 0 ? izeta - 1 : 0, zeta - T(1));
          const T sz = (izeta > 0) ? sz1 * s : kpow(s, 0, zeta);
          part += al * sz;
          if (out) out[(size_t)gr * ldo + gc] = zeta * al * sz1;
        }
      }
      // reduce over the TX threads of this row (tx = lane mod TX)
#pragma unroll
      for (int o = TX / 2; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      if (tx == 0 && gr < M) eps_part[(size_t)gr * n_tiles + blockIdx.x] = part;
    }
  } else {
#pragma unroll
    for (int i = 0; i < RM; ++i) {
      const int gr = row0 + ty + TY * i;
#pragma unroll
      for (int j = 0; j < RN; ++j) {
        const int gc = col0 + tx + TX * j;
        if (gr < M && gc < N) out[(size_t)gr * ldo + gc] = acc[i][j];
      }
    }
  }
}

template <typename T, int MODE>
static cudaError_t launch_gemm(const T* A, const T* B, int M, int N, int K, const T* alpha, int izeta, T zeta,
                               T* eps_part, int n_tiles, T* out, int ldo, cudaStream_t st) {
  const SimtTile t = pick_tile<T>(M, N);
  const dim3 grid((N + t.n - 1) / t.n, (M + t.m - 1) / t.m);
  if (t.m == 64) {
    sg_launch(gemm_kernel<T, MODE, 64, 64, 4, 4>, grid, 256, 0, st, A, B, M, N, K, alpha, izeta, zeta, eps_part, n_tiles, out, ldo);
    ++sg_kernel_launches;
    return cudaGetLastError();
  }
  if constexpr (sizeof(T) == 8) {
    if (t.n == 32)
      sg_launch(gemm_kernel<T, MODE, 32, 32, 2, 2>, grid, 256, 0, st, A, B, M, N, K, alpha, izeta, zeta, eps_part, n_tiles, out, ldo);
    else
      sg_launch(gemm_kernel<T, MODE, 32, 16, 2, 2>, grid, 128, 0, st, A, B, M, N, K, alpha, izeta, zeta, eps_part, n_tiles, out, ldo);
  }
  ++sg_kernel_launches;
  return cudaGetLastError();
}

template <typename T>
cudaError_t sg_gap_forward_simt(const T* q, const T* qs, const T* alpha, int n, int m, int d,
                                double zeta, T* eps_part, int n_tiles, T* kp, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const int iz = (zeta >= 1.0 && zeta == (double)(int)zeta) ? (int)zeta : 0;
  return launch_gemm<T, 0>(q, qs, n, m, d, alpha, iz, (T)zeta, eps_part, n_tiles, kp, m, st);
}

template <typename T>
cudaError_t sg_gap_backward_simt(const T* kp, const T* qs, int n, int m, int d, T* g,
                                 cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  return launch_gemm<T, 1>(kp, qs, n, d, m, nullptr, 0, T(0), nullptr, 0, g, d, st);
}

template cudaError_t sg_gap_forward_simt<float>(const float*, const float*, const float*, int, int,
                                                int, double, float*, int, float*, cudaStream_t);
template cudaError_t sg_gap_forward_simt<double>(const double*, const double*, const double*, int,
                                                 int, int, double, double*, int, double*, cudaStream_t);
template cudaError_t sg_gap_backward_simt<float>(const float*, const float*, int, int, int, float*,
                                                 cudaStream_t);
template cudaError_t sg_gap_backward_simt<double>(const double*, const double*, int, int, int,
                                                  double*, cudaStream_t);
