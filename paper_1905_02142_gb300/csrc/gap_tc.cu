// GAP model on the tensor cores (mixed-precision path): tcgen05.mma with FP16 operands
// staged by TMA in 128B-swizzled shared memory and FP32 accumulators in tensor memory.
//
//   eps_i = sum_s alpha_s (q_i . q_s)^zeta      (Sec. IV.A with the SOAP kernel of Sec. I)
//   g_i   = dE/dq_i = sum_s zeta alpha_s (q_i . q_s)^(zeta-1) q_s
//
// The dot products q_i.q_s lie close together (0.86..1.0 on carbon-like boxes) and the
// alpha_s have random signs, so eps_i is a strong cancellation: plain BF16 operands lose
// ~6e-2 of it and plain FP16 ~5e-3.  The products are therefore split as
//   q = qbar + n u,  qbar = mean of the sparse rows, n = |q - qbar|, |u| = 1,
//   q_i.q_s = qbar.qbar + qbar.(q_i - qbar) + qbar.(q_s - qbar) + n_i n_s (u_i . u_s),
// with the rank-one terms in FP32 and only u_i.u_s on the tensor cores, either as one FP16
// product hi*hi (K = D) or as the split hi*hi + hi*lo + lo*hi (one GEMM over K = 3 D:
// A = [hi|hi|lo], B = [hi|lo|hi]; relative error ~1e-7 on eps).  How much one product loses
// depends on the model (a few 1e-6 on carbon-like boxes with thousands of sparse rows, above
// 1e-4 with a dozen): the library measures it per model and picks the number of products.
// The backward product needs less: g_i = r_i qbar + kappa kp'_i U with
// r_i = sum_s zeta alpha_s S^(zeta-1) in FP32, kp'_is = zeta alpha_s n_s S^(zeta-1) / kappa in
// FP16 and U the unit sparse rows in FP16 (single pass).
#include <cuda.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "tcgen05.cuh"

namespace {

constexpr int BM = 128, BK = 64;

using namespace tc5;

// Columns an epilogue takes per TMEM read: Epi::CHUNK (24 or 32) if declared, else 32.
template <class E, class = void> struct EpiChunk { static constexpr int value = 32; };
template <class E> struct EpiChunk<E, std::void_t<decltype(E::CHUNK)>> { static constexpr int value = E::CHUNK; };
// Epilogues with Epi::STAGED write a 32 x 32 FP16 output box per chunk through shared memory
// and a TMA store (two 2 KB staging buffers per epilogue warp).
template <class E, class = void> struct EpiStaged { static constexpr bool value = false; };
template <class E> struct EpiStaged<E, std::void_t<decltype(E::STAGED)>> { static constexpr bool value = E::STAGED; };

// ------------------------------------------------------------------ epilogues
struct EpiStore {  // C = A B^T (diagnostic)
  int rows, cols;
  float* c;
  __device__ void begin(int) {}
  __device__ void apply(int row, int col0, const uint32_t* v) {
    if (row >= rows) return;
    for (int j = 0; j < 32; ++j)
      if (col0 + j < cols) c[(size_t)row * cols + col0 + j] = __uint_as_float(v[j]);
  }
  __device__ void end(int, int) {}
};

// s^(Z-1) for a compile-time integer Z >= 1
template <int Z>
__device__ __forceinline__ float pow_zm1(float s) {
  float o = 1.f;
#pragma unroll
  for (int k = 1; k < Z; ++k) o *= s;
  return o;
}

struct EpiGapFwd {
  static constexpr bool STAGED = true;  // kp through shared memory and TMA stores
  int rows, ld_kp, n_tiles, izeta;
  float zeta;
  const float *u, *nrm;              // [N]
  const float4* col;                 // [Mp] (qbar.qbar + qbar.(q_s-qbar), n_s, alpha_s, f_s)
  float *eps_part, *r_part;          // [N][n_tiles]
  __half* kp;                        // [N][ld_kp] or null
  float eps, r, ui, ni;
  __device__ void begin(int row) {
    eps = 0.f;
    r = 0.f;
    ui = row < rows ? u[row] : 0.f;
    ni = row < rows ? nrm[row] : 0.f;
  }
  // S^(zeta-1) for one output, zeta fixed at compile time (Z > 0) or general (Z = 0)
  template <int Z>
  __device__ __forceinline__ void run(int col0, const uint32_t* v, uint32_t* out) {
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
      float kv[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 c = __ldg(col + col0 + j + h);
        const float S = fmaf(ni * c.y, __uint_as_float(v[j + h]), ui + c.x);
        const float sz1 = Z > 0 ? pow_zm1<Z>(S) : powf(fmaxf(S, 0.f), zeta - 1.f);
        eps = fmaf(c.z, sz1 * S, eps);
        r = fmaf(zeta * c.z, sz1, r);
        kv[h] = c.w * sz1;
      }
      const __half2 h2 = __floats2half2_rn(kv[0], kv[1]);
      out[j / 2] = *reinterpret_cast<const uint32_t*>(&h2);
    }
  }
  // S-dependent sums of one row's 32 columns; out: their 32 FP16 kernel derivatives in pairs
  __device__ __forceinline__ void row_chunk(int col0, const uint32_t* v, uint32_t* out) {
    switch (izeta) {
      case 1: run<1>(col0, v, out); break;
      case 2: run<2>(col0, v, out); break;
      case 3: run<3>(col0, v, out); break;
      case 4: run<4>(col0, v, out); break;
      default: run<0>(col0, v, out); break;
    }
  }
  // The warp's 32 rows (row0 ..) x 32 columns (col0 ..): sums in registers; with kp, the
  // kernel derivatives go to this warp's staging buffer `buf` (64 B per row) and one lane
  // stores the 32 x 32 box with TMA (rows past the end are clipped by the tensor map).
  __device__ void apply_staged(int row, int row0, int col0, const uint32_t* v, unsigned char* stage, int& buf,
                               const CUtensorMap* map) {
    const int lane = threadIdx.x & 31;
    uint32_t out[16];
    if (row < rows) {
      row_chunk(col0, v, out);
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k) out[k] = 0u;
    }
    if (!kp) return;
    if (lane == 0) bulk_wait_read1();  // the store of two chunks ago has read this buffer
    __syncwarp();
    unsigned char* sb = stage + buf * 2048;
    uint4* dst = reinterpret_cast<uint4*>(sb + lane * 64);
#pragma unroll
    for (int k = 0; k < 4; ++k) dst[k] = make_uint4(out[4 * k], out[4 * k + 1], out[4 * k + 2], out[4 * k + 3]);
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) {
      if (row0 < rows) tma_store_2d(map, col0, row0, sb);  // (a box wholly past the end: nothing)
      bulk_commit();
    }
    buf ^= 1;
  }
  __device__ void end(int row, int slot) {
    if (row >= rows) return;
    eps_part[(size_t)row * n_tiles + slot] = eps;
    r_part[(size_t)row * n_tiles + slot] = r;
  }
};

// The gradient rows leave through the warp's 32 x 32 shared-memory box (as EpiKernelRows): one
// store instruction writes 128 contiguous bytes of one row instead of 4 bytes of 32 rows
// (D is not a multiple of 4, so a TMA store cannot write them).  100,000 x 605, K = 4096: 574
// -> 403 us; 4096 x 1224, K = 2048: 62 -> 35 us.
struct EpiGapBwd {
  static constexpr bool STAGED = true;
  int rows, d, n_tiles;
  float kappa;
  const float* qbar;    // [Dp]
  const float* r_part;  // [N][n_tiles]
  float* g;             // [N][d]
  float r;              // of the lane's row
  __device__ void begin(int row) {
    r = 0.f;
    if (row < rows) {
#pragma unroll 4
      for (int t = 0; t < n_tiles; ++t) r += r_part[(size_t)row * n_tiles + t];
    }
  }
  __device__ void apply_staged(int, int row0, int col0, const uint32_t* v, unsigned char* stage, int&,
                               const CUtensorMap*) {
    const int lane = threadIdx.x & 31, k = col0 + lane;
    float* box = reinterpret_cast<float*>(stage);
    __syncwarp();  // the previous box has been read
#pragma unroll
    for (int j = 0; j < 32; ++j) box[lane * 32 + (j ^ lane)] = __uint_as_float(v[j]);
    __syncwarp();
    const float qb = k < d ? __ldg(qbar + k) : 0.f;
    const int n = min(32, rows - row0);
#pragma unroll 4
    for (int t = 0; t < n; ++t) {
      const float rt = __shfl_sync(0xffffffffu, r, t);
      if (k < d) g[(size_t)(row0 + t) * d + k] = fmaf(rt, qb, kappa * box[t * 32 + (lane ^ t)]);
    }
  }
  __device__ void end(int, int) {}
};

// Kernel rows of the fitting matrices (atoms x sparse set): k(i, s) = S^zeta, and for the
// force rows the weight w = zeta S^(zeta-1) / |p_i|; S as in EpiGapFwd.
// Bound by its output stores (64 MB for 4000 x 4000 rows against 0.03 ms of MMAs).  A TMEM
// read leaves one row per lane, and storing from there writes 32 rows x 4 bytes per
// instruction: the 32 x 32 box is turned through the warp's 4 KB of shared memory instead
// (column c of row r at r 32 + (c ^ r): conflict-free both ways, no padding), so each store
// instruction writes 128 contiguous bytes of one row, for any row stride m.  4000 x 4000 rows,
// K = 1920: 208 -> 65 us; 10,000 x 1000 with the weights, K = 1152: 206 -> 43 us.
struct EpiKernelRows {
  static constexpr bool STAGED = true;
  int rows, m, ldw, izeta;
  float zeta;
  const float *u, *nrm, *pnorm;      // [N]
  const float4* col;                 // [Mp] as in EpiGapFwd
  float* k;                          // [N][m]
  float* w;                          // [N][ldw] or null
  float ui, ni, ip;                  // of the lane's row
  __device__ void begin(int row) {
    ui = row < rows ? u[row] : 0.f;
    ni = row < rows ? nrm[row] : 0.f;
    ip = (row < rows && w) ? 1.f / pnorm[row] : 0.f;
  }
  template <int Z>
  __device__ __forceinline__ void run(int row0, int s, const float* box) {
    const int lane = threadIdx.x & 31;
    const float4 c = __ldg(col + s);
    const int n = min(32, rows - row0);
#pragma unroll 4
    for (int r = 0; r < n; ++r) {
      const float nr = __shfl_sync(0xffffffffu, ni, r), ur = __shfl_sync(0xffffffffu, ui, r);
      const float S = fmaf(nr * c.y, box[r * 32 + (lane ^ r)], ur + c.x);
      const float sz1 = Z > 0 ? pow_zm1<Z>(S) : powf(fmaxf(S, 0.f), zeta - 1.f);
      if (s < m) k[(size_t)(row0 + r) * m + s] = Z > 0 ? sz1 * S : powf(fmaxf(S, 0.f), zeta);
      if (w) w[(size_t)(row0 + r) * ldw + s] = zeta * sz1 * __shfl_sync(0xffffffffu, ip, r);
    }
  }
  __device__ void apply_staged(int, int row0, int col0, const uint32_t* v, unsigned char* stage, int&,
                               const CUtensorMap*) {
    const int lane = threadIdx.x & 31;
    float* box = reinterpret_cast<float*>(stage);
    __syncwarp();  // the previous box has been read
#pragma unroll
    for (int j = 0; j < 32; ++j) box[lane * 32 + (j ^ lane)] = __uint_as_float(v[j]);
    __syncwarp();
    switch (izeta) {
      case 1: run<1>(row0, col0 + lane, box); break;
      case 2: run<2>(row0, col0 + lane, box); break;
      case 3: run<3>(row0, col0 + lane, box); break;
      case 4: run<4>(row0, col0 + lane, box); break;
      default: run<0>(row0, col0 + lane, box); break;
    }
  }
  __device__ void end(int, int) {}
};

// Force rows of the fitting matrices: rows = sparse environments s, columns = projected
// descriptor Jacobian columns J' (see design.cu) ordered by target atom.  With the sparse
// operand [kd (q_s - qbar) | kd | kd] and the column [2^e J' | hi | lo of 2^e qbar.J'], the
// accumulator is kd 2^e q_s.J', and the contribution of a column (owner o, target t,
// component a = col mod 3) is w_os 2^-e / kd times it.  The running sums of one target are
// added to dk[t][a][s] when the target changes (a target's columns are contiguous).
// Tiles of 192 columns are read 24 at a time, so every chunk starts at a column triple (the
// three components of one pair or self slot: one owner, one target, one scale).
struct EpiDesignGrad {
  static constexpr int CHUNK = 24;
  int m, ldw, ncols;
  float inv_kd;
  const int2* col_at;                // [ncols] (owner, target)
  const float4* col_v;               // [ncols] .z = 2^-e of the column's triple
  const float* w;                    // [N][ldw] w_os
  float* dk;                         // [N][3][m]
  int target;
  float acc0, acc1, acc2;
  __device__ void flush(int row) {
    if (target >= 0) {
      float* o = dk + (size_t)target * 3 * m + row;
      if (acc0 != 0.f) atomicAdd(o, acc0);
      if (acc1 != 0.f) atomicAdd(o + m, acc1);
      if (acc2 != 0.f) atomicAdd(o + 2 * m, acc2);
    }
    acc0 = acc1 = acc2 = 0.f;
  }
  __device__ void begin(int) {
    target = -1;
    acc0 = acc1 = acc2 = 0.f;
  }
  // Lane 3t reads the record of triple t (coalesced); owner, target and scale reach every
  // lane by shuffles, and the 8 owners' weights at this row are requested before the first
  // use.  All lanes take part (rows past m compute but do not write).
  __device__ void apply(int row, int col0, const uint32_t* v) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool live = row < m;
    const int mine = col0 + lane;
    int2 at_l = make_int2(-1, -1);
    float cz_l = 0.f;
    if (lane < CHUNK && lane % 3 == 0 && mine < ncols) {
      at_l = __ldg(col_at + mine);
      cz_l = __ldg(&col_v[mine].z);
    }
    float wk[CHUNK / 3];
    int tg[CHUNK / 3];
#pragma unroll
    for (int t = 0; t < CHUNK / 3; ++t) {
      const int o = __shfl_sync(FULL, at_l.x, 3 * t);
      const float cz = __shfl_sync(FULL, cz_l, 3 * t);
      tg[t] = __shfl_sync(FULL, at_l.y, 3 * t);
      wk[t] = (live && o >= 0) ? __ldg(w + (size_t)o * ldw + row) * (cz * inv_kd) : 0.f;
    }
#pragma unroll
    for (int t = 0; t < CHUNK / 3; ++t) {
      if (tg[t] < 0) continue;  // past the last column (same for every lane)
      if (tg[t] != target) {
        if (live) flush(row);
        target = tg[t];
      }
      acc0 = fmaf(wk[t], __uint_as_float(v[3 * t]), acc0);
      acc1 = fmaf(wk[t], __uint_as_float(v[3 * t + 1]), acc1);
      acc2 = fmaf(wk[t], __uint_as_float(v[3 * t + 2]), acc2);
    }
  }
  __device__ void end(int row, int) {
    if (row < m) flush(row);
  }
  // The same over a group of 48 columns whose tile stays while the rows pass
  // (force_rows_kernel).  What the 16 triples of the group need is the same for every row, so it
  // is worked out once per column tile: the warp's table holds each owner's weight-row offset,
  // scale and target, and a mask says before which triples the target changes.  Per row tile that
  // leaves 16 weight loads (requested one tile ahead), 16 multiplications and 48 FMAs.
  struct Table {
    uint32_t off[16];
    float scale[16];
    int target[16];
  };
  // returns the change mask (bit t: triple t has another target than triple t - 1)
  __device__ uint32_t fill(Table& tb, int col0) const {
    const int lane = threadIdx.x & 31, t = lane & 15;
    const int c = min(col0 + 3 * t, ncols - 3);  // past the end: the last triple with scale 0
    const int2 at = __ldg(col_at + c);
    const int before = __shfl_up_sync(0xffffffffu, at.y, 1);
    __syncwarp();  // the previous table has been read
    if (lane < 16) {
      tb.off[t] = (uint32_t)at.x * (uint32_t)ldw;
      tb.scale[t] = col0 + 3 * t < ncols ? __ldg(&col_v[c].z) * inv_kd : 0.f;
      tb.target[t] = at.y;
    }
    __syncwarp();
    return __ballot_sync(0xffffffffu, lane > 0 && lane < 16 && at.y != before);
  }
  __device__ __forceinline__ void weights(const Table& tb, int row, float (&wk)[16]) const {
    const float* wr = w + row;  // (row < ldw: the weights are padded as the sparse operand)
#pragma unroll
    for (int t = 0; t < 16; t += 4) {
      const uint4 o = *reinterpret_cast<const uint4*>(tb.off + t);
      wk[t] = __ldg(wr + o.x);
      wk[t + 1] = __ldg(wr + o.y);
      wk[t + 2] = __ldg(wr + o.z);
      wk[t + 3] = __ldg(wr + o.w);
    }
  }
  __device__ __forceinline__ void add_to(int tg, int row) {
    if (row < m) {
      float* o = dk + (size_t)tg * 3 * m + row;
      atomicAdd(o, acc0);
      atomicAdd(o + m, acc1);
      atomicAdd(o + 2 * m, acc2);
    }
    acc0 = acc1 = acc2 = 0.f;
  }
  template <int C>
  __device__ __forceinline__ void chunk(const Table& tb, uint32_t mask, int row, const float (&wk)[16], const uint32_t* v) {
#pragma unroll
    for (int t = 0; t < 8; t += 4) {
      const float4 sc = *reinterpret_cast<const float4*>(tb.scale + 8 * C + t);
      const float s4[4] = {sc.x, sc.y, sc.z, sc.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int k = 8 * C + t + u;
        if (k > 0 && ((mask >> k) & 1u)) add_to(tb.target[k - 1], row);
        const float s = s4[u] * wk[k];
        acc0 = fmaf(s, __uint_as_float(v[3 * (t + u)]), acc0);
        acc1 = fmaf(s, __uint_as_float(v[3 * (t + u) + 1]), acc1);
        acc2 = fmaf(s, __uint_as_float(v[3 * (t + u) + 2]), acc2);
      }
    }
  }
};

// ------------------------------------------------------------------ the GEMM
// Persistent, warp-specialised: one CTA per SM walks the output tiles (row-major over
// [M/BM] x [N/BN], so CTAs running together share A rows in L2).
//   warp 0, lane 0 : TMA producer, STAGES-deep ring of A/B tiles (full/empty mbarriers)
//   warp 1, lane 0 : MMA issuer, accumulates each tile into one of two TMEM buffers
//   warps 2..      : epilogue, EPI_WARPS warps; warp w reads TMEM lanes 32*(w%4) .. +31 and
//                    a 1/(EPI_WARPS/4) share of the columns; it releases the buffer when done
// so the epilogue of one tile overlaps the MMAs of the next.
// MFAST walks the tiles column-major instead ([N/BN] x [M/BM], m fastest): for a B far
// larger than A, CTAs running together then share B tiles and B is read from memory once.
template <int BN, int STAGES, int EPI_WARPS, class Epi, bool MFAST = false>
__global__ void __launch_bounds__(32 * (2 + EPI_WARPS), 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmC, int num_kb, int m_tiles, int n_tiles, Epi epi, int* err) {
  pdl_begin();
  constexpr uint32_t A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2;
  constexpr int HALVES = EPI_WARPS / 4;           // column groups per tile
  constexpr int COLS = BN / HALVES;               // columns per epilogue warp
  constexpr int CH = EpiChunk<Epi>::value;        // columns per TMEM read
  static_assert((CH == 32 || CH == 24) && COLS % CH == 0, "epilogue chunking");
  // TMEM is allocated in powers of two (>= 32 columns): room for two BN-wide accumulators
  constexpr uint32_t TMEM_COLS = 2 * BN <= 32 ? 32 : 2 * BN <= 64 ? 64 : 2 * BN <= 128 ? 128 : 2 * BN <= 256 ? 256 : 512;
  static_assert(2 * BN <= 512, "two accumulators must fit in tensor memory");
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * A_BYTES;
  __shared__ __align__(8) uint64_t full_bar[STAGES];
  __shared__ __align__(8) uint64_t empty_bar[STAGES];
  __shared__ __align__(8) uint64_t tfull_bar[2];
  __shared__ __align__(8) uint64_t tempty_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total = m_tiles * n_tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull_bar[b], 1);
      mbar_init(&tempty_bar[b], EPI_WARPS);
    }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      int issued[STAGES];
      for (int s = 0; s < STAGES; ++s) issued[s] = 0;
      for (int t = blockIdx.x; t < total && !abort_flag; t += gridDim.x) {
        const int m0 = (MFAST ? t % m_tiles : t / n_tiles) * BM, n0 = (MFAST ? t / m_tiles : t % n_tiles) * BN;
        for (int kb = 0; kb < num_kb; ++kb, ++it) {
          const int s = it % STAGES, round = it / STAGES;
          if (round > 0 && !mbar_wait(&empty_bar[s], (round - 1) & 1)) {
            abort_flag = 1;
            break;
          }
          mbar_expect_tx(&full_bar[s], A_BYTES + B_BYTES);
          tma_load_2d(sA + s * A_BYTES, &tmA, kb * BK, m0, &full_bar[s]);
          tma_load_2d(sB + s * B_BYTES, &tmB, kb * BK, n0, &full_bar[s]);
          ++issued[s];
        }
      }
      // every copy started here has landed before the block may exit
      for (int s = 0; s < STAGES; ++s)
        if (issued[s] > 0 && !mbar_wait(&full_bar[s], (issued[s] - 1) & 1)) abort_flag = 1;
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      // One thread issues every MMA, so its own instructions are on the critical path (an MMA of
      // 192 columns lasts 96 cycles): descriptors are formed once and advanced by constants
      // (32 bytes of K are 2 in a descriptor's address field), the ring stage is a counter
      // (100,000 x 4096, K = 1920: 1092 -> 1040 us).
      constexpr uint32_t idesc = idesc_f16(BM, BN);
      const uint64_t da0 = sw128_desc(smem_u32(sA)), db0 = sw128_desc(smem_u32(sB));
      int s = 0, lt = 0;
      uint32_t par = 0;  // parity of the ring's round
      for (int t = blockIdx.x; t < total && !abort_flag; t += gridDim.x, ++lt) {
        const int b = lt & 1, use = lt >> 1;
        if (use > 0 && !mbar_wait(&tempty_bar[b], (use - 1) & 1)) {
          abort_flag = 1;
          break;
        }
        fence_after();
        const uint32_t acc = tmem + (uint32_t)(b * BN);
        bool ok = true;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!mbar_wait_quick(&full_bar[s], par)) {
            ok = false;
            break;
          }
          fence_after();
          const uint64_t da = da0 + (uint32_t)s * (A_BYTES >> 4), db = db0 + (uint32_t)s * (B_BYTES >> 4);
          mma_f16(acc, da, db, idesc, kb != 0);
#pragma unroll
          for (int k = 1; k < BK / 16; ++k) mma_f16(acc, da + 2 * k, db + 2 * k, idesc, 1);
          mma_commit(&empty_bar[s]);
          if (++s == STAGES) {
            s = 0;
            par ^= 1;
          }
        }
        if (!ok) {
          abort_flag = 1;
          break;
        }
        mma_commit(&tfull_bar[b]);
      }
    }
    __syncwarp();
  } else {
    const int ew = warp - 2;                 // 0 .. EPI_WARPS-1
    const int lg = warp & 3;                 // TMEM lane group this warp may access
    const int half = ew / 4;                 // column group
    unsigned char* stage = sB + STAGES * B_BYTES + ew * 4096;  // staged epilogues only
    int buf = 0;
    int lt = 0;
    for (int t = blockIdx.x; t < total; t += gridDim.x, ++lt) {
      const int b = lt & 1, use = lt >> 1;
      const bool ready = __all_sync(0xffffffffu, mbar_wait(&tfull_bar[b], use & 1) && !abort_flag);
      if (!ready) {
        if (lane == 0) {
          abort_flag = 1;
          atomicOr(err, SG_ERR_TIMEOUT);
        }
        break;
      }
      fence_after();
      const int m0 = (MFAST ? t % m_tiles : t / n_tiles) * BM, n0 = (MFAST ? t / m_tiles : t % n_tiles) * BN;
      const int row = m0 + lg * 32 + lane;
      epi.begin(row);
#pragma unroll 1
      for (int c = 0; c < COLS / CH; ++c) {
        uint32_t v[CH];
        const int col = half * COLS + c * CH;
        const uint32_t ta = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(b * BN + col);
        if constexpr (CH == 32) {
          tmem_ld32(ta, v);
        } else {
          tmem_ld16_nw(ta, v);
          tmem_ld8_nw(ta + 16, v + 16);
          tmem_wait();
        }
        if constexpr (EpiStaged<Epi>::value) epi.apply_staged(row, m0 + lg * 32, n0 + col, v, stage, buf, &tmC);
        else epi.apply(row, n0 + col, v);
      }
      epi.end(row, (MFAST ? t / m_tiles : t % n_tiles) * HALVES + half);
      fence_before();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty_bar[b])) : "memory");
    }
    if constexpr (EpiStaged<Epi>::value) {
      if (lane == 0) bulk_wait_all();  // every TMA store of this warp has completed
      __syncwarp();
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS)
                 : "memory");
}

// The force-row GEMM: the B tile (192 Jacobian columns) kept in shared memory while every row
// tile of A (the sparse operand, which stays in L2) passes.  One CTA takes column tiles
// blockIdx.x, + gridDim.x, ..; barriers per B block let the next column tile's block load as
// soon as the last row tile has consumed it.  The streaming GEMM reloads B for every row tile (15
// GB of L2 reads for 1.53 M columns) and its epilogue is a chain of column record -> owner's
// weight -> accumulator; here the records are read once per column tile and the weights
// requested ahead.  1.53 M columns, K = 384, 1024 rows: 1455 -> 1344 us (without the epilogue
// 1087; the MMAs alone would take 500: the A ring's 64 KB in flight bound it).  ksteps: MMA
// steps of 16 in K that hold data (the padding of the last block is not multiplied).
template <int STAGES, int KB_MAX>
__global__ void __launch_bounds__(32 * (2 + 16), 1)
force_rows_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int num_kb,
                     int ksteps, int m_tiles, int n_tiles, EpiDesignGrad epi, int* err) {
  pdl_begin();
  constexpr int BN = 192, EPI_WARPS = 16, COLS = BN / (EPI_WARPS / 4);
  static_assert(COLS == 48, "two chunks of 24 columns per epilogue warp");
  constexpr uint32_t A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sB = smem;                       // [num_kb] blocks of the current column tile
  uint8_t* sA = smem + num_kb * B_BYTES;    // ring
  __shared__ __align__(8) uint64_t afull[STAGES], aempty[STAGES], bfull[KB_MAX], bempty[KB_MAX];
  __shared__ __align__(8) uint64_t tfull_bar[2], tempty_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], 1);
    }
    for (int k = 0; k < KB_MAX; ++k) {
      mbar_init(&bfull[k], 1);
      mbar_init(&bempty[k], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull_bar[b], 1);
      mbar_init(&tempty_bar[b], EPI_WARPS);
    }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&tmem_slot, 512);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int it = 0, ct = 0, a_issued[STAGES], b_issued = 0;
      for (int s = 0; s < STAGES; ++s) a_issued[s] = 0;
      for (int nt = blockIdx.x; nt < n_tiles && !abort_flag; nt += gridDim.x, ++ct) {
        for (int mt = 0; mt < m_tiles && !abort_flag; ++mt) {
          for (int kb = 0; kb < num_kb; ++kb, ++it) {
            if (mt == 0) {
              if (ct > 0 && !mbar_wait(&bempty[kb], (ct - 1) & 1)) {
                abort_flag = 1;
                break;
              }
              mbar_expect_tx(&bfull[kb], B_BYTES);
              tma_load_2d(sB + kb * B_BYTES, &tmB, kb * BK, nt * BN, &bfull[kb]);
              b_issued = ct * num_kb + kb + 1;
            }
            const int s = it % STAGES, round = it / STAGES;
            if (round > 0 && !mbar_wait(&aempty[s], (round - 1) & 1)) {
              abort_flag = 1;
              break;
            }
            mbar_expect_tx(&afull[s], A_BYTES);
            tma_load_2d(sA + s * A_BYTES, &tmA, kb * BK, mt * BM, &afull[s]);
            ++a_issued[s];
          }
        }
      }
      // every copy started here has landed before the block may exit
      for (int s = 0; s < STAGES; ++s)
        if (a_issued[s] > 0 && !mbar_wait(&afull[s], (a_issued[s] - 1) & 1)) abort_flag = 1;
      for (int kb = 0; kb < num_kb; ++kb) {
        const int loads = (b_issued - kb + num_kb - 1) / num_kb;  // of this block
        if (loads > 0 && !mbar_wait(&bfull[kb], (loads - 1) & 1)) abort_flag = 1;
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_f16(BM, BN);
      const uint64_t da0 = sw128_desc(smem_u32(sA)), db0 = sw128_desc(smem_u32(sB));
      const int last = ksteps - (num_kb - 1) * (BK / 16);  // steps of the last block
      int s = 0, ct = 0, lt = 0;
      uint32_t par = 0;
      bool ok = true;
      for (int nt = blockIdx.x; nt < n_tiles && ok && !abort_flag; nt += gridDim.x, ++ct) {
        for (int mt = 0; mt < m_tiles && ok; ++mt, ++lt) {
          const int b = lt & 1, use = lt >> 1;
          if (use > 0 && !mbar_wait(&tempty_bar[b], (use - 1) & 1)) {
            ok = false;
            break;
          }
          fence_after();
          const uint32_t acc = tmem + (uint32_t)(b * 256);
          for (int kb = 0; kb < num_kb; ++kb) {
            if ((mt == 0 && !mbar_wait_quick(&bfull[kb], ct & 1)) || !mbar_wait_quick(&afull[s], par)) {
              ok = false;
              break;
            }
            fence_after();
            const uint64_t da = da0 + (uint32_t)s * (A_BYTES >> 4), db = db0 + (uint32_t)kb * (B_BYTES >> 4);
            mma_f16(acc, da, db, idesc, kb != 0);
#pragma unroll
            for (int k = 1; k < BK / 16; ++k)
              if (kb + 1 < num_kb || k < last) mma_f16(acc, da + 2 * k, db + 2 * k, idesc, 1);
            mma_commit(&aempty[s]);
            if (mt == m_tiles - 1) mma_commit(&bempty[kb]);
            if (++s == STAGES) {
              s = 0;
              par ^= 1;
            }
          }
          if (ok) mma_commit(&tfull_bar[b]);
        }
      }
      if (!ok) abort_flag = 1;
    }
    __syncwarp();
  } else {
    const int ew = warp - 2, lg = warp & 3, half = ew / 4;
    int lt = 0;
    bool ready = true;
    // two tables per warp: this column tile's, and the next one's, filled while this one runs
    EpiDesignGrad::Table* tables =
        reinterpret_cast<EpiDesignGrad::Table*>(smem + (size_t)KB_MAX * B_BYTES + STAGES * A_BYTES) + 2 * ew;
    int cur = 0;
    uint32_t mask = epi.fill(tables[0], (int)blockIdx.x * BN + half * COLS), next_mask = 0;
    const int row0 = lg * 32 + lane;
    float wk[16], wn[16];
    epi.weights(tables[0], row0, wk);
    for (int nt = blockIdx.x; nt < n_tiles && ready; nt += gridDim.x) {
      const EpiDesignGrad::Table& tb = tables[cur];
      const bool more = nt + (int)gridDim.x < n_tiles;
      if (more) next_mask = epi.fill(tables[cur ^ 1], (nt + (int)gridDim.x) * BN + half * COLS);
      for (int mt = 0; mt < m_tiles; ++mt, ++lt) {
        const int b = lt & 1, use = lt >> 1;
        const int row = mt * BM + row0;
        // the next tile's weights, in flight while this one's accumulators are awaited and used
        if (mt + 1 < m_tiles) epi.weights(tb, row + BM, wn);
        else if (more) epi.weights(tables[cur ^ 1], row0, wn);
        ready = __all_sync(0xffffffffu, mbar_wait(&tfull_bar[b], use & 1) && !abort_flag);
        if (!ready) {
          if (lane == 0) {
            abort_flag = 1;
            atomicOr(err, SG_ERR_TIMEOUT);
          }
          break;
        }
        fence_after();
        epi.begin(row);
        const uint32_t ta = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(b * 256 + half * COLS);
        uint32_t v[24];
        tmem_ld16_nw(ta, v);
        tmem_ld8_nw(ta + 16, v + 16);
        tmem_wait();
        epi.chunk<0>(tb, mask, row, wk, v);
        tmem_ld16_nw(ta + 24, v);
        tmem_ld8_nw(ta + 40, v + 16);
        tmem_wait();
        fence_before();
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty_bar[b])) : "memory");
        epi.chunk<1>(tb, mask, row, wk, v);
        epi.add_to(tb.target[15], row);
#pragma unroll
        for (int t = 0; t < 16; ++t) wk[t] = wn[t];
      }
      cur ^= 1;
      mask = next_mask;
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

template <int BN, int STAGES, int EPI_WARPS = 0, bool STAGED = false>
constexpr size_t smem_bytes() {
  return (size_t)STAGES * (BM * BK * 2 + BN * BK * 2) + 1024 + (STAGED ? (size_t)EPI_WARPS * 4096 : 0);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// 2D FP16 row-major matrix [rows][cols] (cols a multiple of 64) with row stride ld elements
// (ld = cols when 0), tiles of box_rows x 64.
bool make_map(CUtensorMap* m, const void* base, int rows, int cols, int box_rows, int ld = 0) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld > 0 ? ld : cols) * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2D FP16 output [rows][cols] (row stride cols) written in boxes of 32 x 32 by TMA stores
bool make_store_map(CUtensorMap* m, void* base, int rows, int cols) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {32, 32};
  cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

// C = A B^T over K = k; lda, ldb: row strides of A and B in elements (k when 0)
template <int BN, int STAGES, int EPI_WARPS, bool MFAST = false, class Epi>
cudaError_t launch_gemm(const void* A, int a_rows, const void* B, int b_rows, int k, Epi epi, int* err,
                        cudaStream_t st, int lda = 0, int ldb = 0, const CUtensorMap* mc = nullptr) {
  if (k % BK != 0 || a_rows <= 0 || b_rows <= 0) return cudaErrorInvalidValue;
  if ((lda > 0 && lda < k) || (ldb > 0 && ldb < k)) return cudaErrorInvalidValue;
  CUtensorMap ma, mb;
  if (!make_map(&ma, A, a_rows, k, BM, lda) || !make_map(&mb, B, b_rows, k, BN, ldb))
    return cudaErrorInvalidValue;
  auto kern = tc_gemm_kernel<BN, STAGES, EPI_WARPS, Epi, MFAST>;
  constexpr size_t smem = smem_bytes<BN, STAGES, EPI_WARPS, EpiStaged<Epi>::value>();
  static_assert(smem <= 227 * 1024, "shared memory per block");
  cudaError_t e = sg_set_smem<tc_gemm_kernel<BN, STAGES, EPI_WARPS, Epi, MFAST>>(smem);
  if (e != cudaSuccess) return e;
  const int sms = sg_sm_count();
  const int m_tiles = (a_rows + BM - 1) / BM, n_tiles = (b_rows + BN - 1) / BN;
  if ((long long)m_tiles * n_tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  const int grid = std::min(sms, m_tiles * n_tiles);
  sg_launch(kern, grid, 32 * (2 + EPI_WARPS), smem, st, ma, mb, mc ? *mc : ma, k / BK, m_tiles, n_tiles, epi, err);
  ++sg_kernel_launches;
  return cudaGetLastError();
}

// K = k, of which the first k_used hold data; false if the B tile of this K does not fit beside
// an A ring of STAGES blocks.
template <int STAGES, int KB_MAX>
bool launch_force_rows(const void* A, int a_rows, const void* B, int b_rows, int k, int k_used,
                       const EpiDesignGrad& epi, int* err, cudaStream_t st, cudaError_t* e) {
  const int num_kb = k / BK;
  if (k % BK != 0 || num_kb > KB_MAX) return false;
  constexpr size_t smem = (size_t)KB_MAX * 192 * BK * 2 + (size_t)STAGES * BM * BK * 2 + 1024 +
                          2 * 16 * sizeof(EpiDesignGrad::Table);
  static_assert(smem <= 227 * 1024, "shared memory per block");
  CUtensorMap ma, mb;
  *e = cudaErrorInvalidValue;
  if (!make_map(&ma, A, a_rows, k, BM, 0) || !make_map(&mb, B, b_rows, k, 192, 0)) return true;
  *e = sg_set_smem<force_rows_kernel<STAGES, KB_MAX>>(smem);
  if (*e != cudaSuccess) return true;
  const int m_tiles = (a_rows + BM - 1) / BM, n_tiles = (b_rows + 191) / 192;
  *e = sg_launch(force_rows_kernel<STAGES, KB_MAX>, std::min(sg_sm_count(), n_tiles), 32 * (2 + 16), smem, st, ma, mb,
                 num_kb, (k_used + 15) / 16, m_tiles, n_tiles, epi, err);
  ++sg_kernel_launches;
  return true;
}

// ------------------------------------------------------------------ operand preparation
// one warp per atom: u = (q - qbar)/|q - qbar| in FP16, A row = [hi] (TERMS = 1, row
// stride dp) or the split [hi | hi | lo] (TERMS = 3, row stride 3 dp)
template <int TERMS>
__global__ void prep_atoms_kernel(const float* __restrict__ q, int n, int d, int dp,
                                  const float* __restrict__ qbar, __half* A, float* nrm, float* uq) {
  pdl_begin();
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  const float* qi = q + (size_t)i * d;
  float ss = 0.f, dq = 0.f;
  for (int k = lane; k < d; k += 32) {
    const float t = qi[k] - qbar[k];
    ss = fmaf(t, t, ss);
    dq = fmaf(t, qbar[k], dq);
  }
  ss = warp_sum(ss);
  dq = warp_sum(dq);
  const float nn = sqrtf(ss);
  const float inv = nn > 0.f ? 1.f / nn : 0.f;
  __half* row = A + (size_t)i * TERMS * dp;
  for (int k = lane; k < dp; k += 32) {
    const float uk = k < d ? (qi[k] - qbar[k]) * inv : 0.f;
    const __half hi = __float2half_rn(uk);
    row[k] = hi;
    if (TERMS == 3) {
      row[dp + k] = hi;
      row[2 * dp + k] = __float2half_rn(uk - __half2float(hi));
    }
  }
  if (lane == 0) {
    nrm[i] = nn;
    uq[i] = dq;
  }
}

}  // namespace

// Tile configurations of the two GAP products.  Each is a (columns per tile BN, pipeline
// stages, epilogue warps) instance of tc_gemm_kernel; configuration 0 is chosen from the
// product's shape, the others are fixed (the autotuner times all of them):
//   forward  0: by shape   1: (128, 6, 4)   2: (128, 6, 8)
//   backward 0: by shape   1: (128, 6, 4)   2: (192, 5, 4)   3: (256, 4, 4)   4: (160, 5, 4)
// The forward's columns are the sparse set padded to 256 (every BN divides it); the
// backward's, the descriptor padded to 64 (ragged last tiles read TMA's zero fill).
// By shape: the BN with the fewest waves of tiles over the SMs, weighted by the cost of one
// tile (proportional to BN + 64: the A tile and the epilogue's fixed part).  Large batches
// take the widest tiles; a product with fewer wide tiles than SMs takes narrow ones.  The
// forward's choices, (256, 4, 8) and (128, 6, 4), both sum 128 columns per slot in the same
// order, and the backward's outputs do not depend on the tile: every choice by shape gives
// the same bits.  1000 atoms x 500 sparse rows, D = 324: forward 14.8 -> 13.0 us, backward
// (64 columns) 25 -> 8.5 us.
static int pick_bn(int n, int cols, const int* bns, int count) {
  const int sms = sg_sm_count(), m_tiles = (n + BM - 1) / BM;
  int best = bns[0];
  long long best_cost = -1;
  for (int k = 0; k < count; ++k) {
    const long long tiles = (long long)m_tiles * ((cols + bns[k] - 1) / bns[k]);
    const long long cost = (tiles + sms - 1) / sms * (bns[k] + 64);
    if (best_cost < 0 || cost < best_cost) {
      best = bns[k];
      best_cost = cost;
    }
  }
  return best;
}
static int fwd_bn(int mp, int cfg, int n) {
  static const int bns[2] = {256, 128};
  return cfg == 0 ? pick_bn(n, mp, bns, 2) : 128;
}
static int bwd_bn(int dp, int cfg, int n) {
  static const int bns[5] = {256, 224, 160, 128, 64};
  static const int fixed[5] = {0, 128, 192, 256, 160};
  return cfg == 0 ? pick_bn(n, dp, bns, 5) : fixed[cfg];
}
// column groups of a forward tile: 8 epilogue warps take half of its columns each
static int fwd_halves(int bn, int cfg) { return bn == 256 || cfg == 2 ? 2 : 1; }

// partial-sum slots per row of the forward epilogue: one per column group of every tile
int sg_gap_tc_tiles(int mp, int fwd_cfg, int n) {
  const int bn = fwd_bn(mp, fwd_cfg, n);
  return mp / bn * fwd_halves(bn, fwd_cfg);
}
int sg_gap_tc_tiles_max(int mp) { return mp / 64; }

cudaError_t sg_gap_tc_prepare(const float* q, int n, int d, int dp, const float* qbar, __half* A, float* nrm,
                              float* uq, int terms, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if (terms == 1)
    sg_launch(prep_atoms_kernel<1>, (n * 32 + 127) / 128, 128, 0, st, q, n, d, dp, qbar, A, nrm, uq);
  else if (terms == 3)
    sg_launch(prep_atoms_kernel<3>, (n * 32 + 127) / 128, 128, 0, st, q, n, d, dp, qbar, A, nrm, uq);
  else
    return cudaErrorInvalidValue;
  ++sg_kernel_launches;
  return cudaGetLastError();
}

cudaError_t sg_gap_tc_forward(const GapTcModel& md, int terms, const __half* A, const float* nrm,
                              const float* uq, int n, float* eps_part, float* r_part, __half* kp, int* err,
                              cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if (terms != 1 && terms != 3) return cudaErrorInvalidValue;
  EpiGapFwd e{};
  e.rows = n;
  e.ld_kp = md.mp;
  e.n_tiles = sg_gap_tc_tiles(md.mp, md.fwd_cfg, n);
  e.izeta = md.izeta;
  e.zeta = md.zeta;
  e.u = uq;
  e.nrm = nrm;
  e.col = md.col;
  e.eps_part = eps_part;
  e.r_part = r_part;
  e.kp = kp;
  // one FP16 product hi.hi: A rows [hi] against the first dp columns of the sparse rows
  // [hi | lo | hi]; three: A rows [hi | hi | lo] against the whole rows
  const int k = terms * md.dp, lda = terms * md.dp, ldb = 3 * md.dp;
  // the kernel derivatives [n][mp] leave through shared memory in 32 x 32 TMA stores
  CUtensorMap mc;
  if (kp && !make_store_map(&mc, kp, n, md.mp)) return cudaErrorInvalidValue;
  const CUtensorMap* pmc = kp ? &mc : nullptr;
  if (md.fwd_cfg < 0 || md.fwd_cfg >= SG_GAP_FWD_CFGS) return cudaErrorInvalidValue;
  if (fwd_bn(md.mp, md.fwd_cfg, n) == 256)
    return launch_gemm<256, 4, 8>(A, n, md.B, md.mp, k, e, err, st, lda, ldb, pmc);
  if (md.fwd_cfg == 2) return launch_gemm<128, 6, 8>(A, n, md.B, md.mp, k, e, err, st, lda, ldb, pmc);
  return launch_gemm<128, 6, 4>(A, n, md.B, md.mp, k, e, err, st, lda, ldb, pmc);
}

cudaError_t sg_gap_tc_backward(const GapTcModel& md, const __half* kp, const float* r_part, int n, float* g,
                               int* err, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  EpiGapBwd e{};
  e.rows = n;
  e.d = md.d;
  e.n_tiles = sg_gap_tc_tiles(md.mp, md.fwd_cfg, n);  // the forward's partial-sum layout
  e.kappa = md.kappa;
  e.qbar = md.qbar;
  e.r_part = r_part;
  e.g = g;
  if (md.bwd_cfg < 0 || md.bwd_cfg >= SG_GAP_BWD_CFGS) return cudaErrorInvalidValue;
  switch (bwd_bn(md.dp, md.bwd_cfg, n)) {
    case 256: return launch_gemm<256, 4, 4>(kp, n, md.BT, md.dp, md.mp, e, err, st);
    case 224: return launch_gemm<224, 4, 4>(kp, n, md.BT, md.dp, md.mp, e, err, st);
    case 192: return launch_gemm<192, 5, 4>(kp, n, md.BT, md.dp, md.mp, e, err, st);
    case 160: return launch_gemm<160, 5, 4>(kp, n, md.BT, md.dp, md.mp, e, err, st);
    case 128: return launch_gemm<128, 6, 4>(kp, n, md.BT, md.dp, md.mp, e, err, st);
    default: return launch_gemm<64, 8, 4>(kp, n, md.BT, md.dp, md.mp, e, err, st);
  }
}

cudaError_t sg_tc_gemm_store(const __half* A, int m, const __half* B, int nn, int k, float* C, int* err,
                             cudaStream_t st) {
  EpiStore e{m, nn, C};
  return launch_gemm<128, 6, 4>(A, m, B, nn, k, e, err, st);
}

cudaError_t sg_tc_kernel_rows(const GapTcModel& md, const __half* A, const float* nrm, const float* uq, int n,
                              int m, const float* pnorm, float* k, float* w, int* err, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  EpiKernelRows e{};
  e.rows = n;
  e.m = m;
  e.ldw = md.mp;
  e.izeta = md.izeta;
  e.zeta = md.zeta;
  e.u = uq;
  e.nrm = nrm;
  e.pnorm = pnorm;
  e.col = md.col;
  e.k = k;
  e.w = w;
  // tiles by shape (each output depends on its row and column alone)
  static const int bns[3] = {256, 128, 64};
  switch (pick_bn(n, md.mp, bns, 3)) {
    case 256: return launch_gemm<256, 4, 8>(A, n, md.B, md.mp, 3 * md.dp, e, err, st);
    case 128: return launch_gemm<128, 6, 8>(A, n, md.B, md.mp, 3 * md.dp, e, err, st);
    default: return launch_gemm<64, 8, 4>(A, n, md.B, md.mp, 3 * md.dp, e, err, st);
  }
}

cudaError_t sg_tc_design_grad(const GapTcModel& md, int n_atoms, int m, const __half* J, long long ncols, const int2* col_at,
                              const float4* col_v, const float* w, float* dk, int* err, cudaStream_t st) {
  if (ncols == 0) return cudaSuccess;
  if (ncols > 0x7fffffffLL - 256) return cudaErrorInvalidValue;
  EpiDesignGrad e{};
  e.m = m;
  e.ldw = md.mp;
  e.ncols = (int)ncols;
  e.inv_kd = 1.f / md.kd;
  e.col_at = col_at;
  e.col_v = col_v;
  e.w = w;
  e.dk = dk;
  // A = the scaled centred sparse rows with their two unit columns, K = dpd.  B stationary where
  // it fits (D <= 446) and the column tiles give every SM several; else the streaming GEMM.
  cudaError_t rc = cudaSuccess;
  if (ncols >= 192LL * 4 * sg_sm_count() && (unsigned long long)n_atoms * md.mp < (1ull << 32) &&
      (launch_force_rows<4, 6>(md.Ad, md.mp, J, (int)ncols, md.dpd, md.d + 2, e, err, st, &rc) ||
       launch_force_rows<2, 7>(md.Ad, md.mp, J, (int)ncols, md.dpd, md.d + 2, e, err, st, &rc)))
    return rc;
  return launch_gemm<192, 5, 16, true>(md.Ad, md.mp, J, (int)ncols, md.dpd, e, err, st);
}
