// Dense matrix products of the exact local solver (Sec. 3: the exact patch
// inverse A_v^-1 as the variant the paper compares against): for a run of
// patches sharing one boundary-type combination, the patch tensors gathered as
// the columns of R (m^d x cnt) are multiplied by the dense inverse,
//
//   Y = alpha * A R,   A: m^d x m^d symmetric;  R, Y: m^d x cnt, column-major,
//
// with m^d = 729, 1331, 2197 for 3D k = 5, 6, 7.
//
// FP64: emulated on the FP16 tensor cores by splitting the operands into
// integer slices (an error-free splitting of the Ozaki type).  Every row of A
// and every column of R is scaled by a power of two into (-1, 1) and split into
// kSlices balanced digits of kSliceBits bits: x = 2^e sum_i x_i 2^(-6 (i+1)), x_i
// an integer with |x_i| <= 32 (64 for the first), exact in FP16.  A product of
// slices is an integer, and so is the sum of the products of all slice pairs of
// one level i + j = l < kSlices: at most K (2 * 64 * 32 + 7 * 32^2) = 11,264 K,
// below 2^24 for K <= 1,472, so the tensor cores' FP32 accumulation of a whole
// level over that inner length is exact (longer ones are taken in parts).  The
// nine levels are combined as integers, four or five to a 48-bit number, and
// those in FP64: two FP64 FMAs per output and part instead of 45, which had
// taken as long as the slice products.  The dropped pairs and the split's
// remainder are below 2^(-6 kSlices) relative to the row and column maxima:
// 2^-54 for 9 slices, the FP64 significand.  The bound is relative to the
// maxima, so fewer slices fail where a row of the inverse spans a wide range (8
// slices: 2.5e-10 on one exact step of the single 3D k = 7 patch of level 1,
// against 1e-10 asked).  FP16 mma.sync runs at 600 TFLOP/s on GB300 against 1.1
// for the FP64 tensor instruction (measured), so the 45 slice products of the
// emulation beat the FP64 product several times over.
//
// A color's patches of all boundary-type combinations are one launch: most
// combinations have a handful of patches, and a launch for each of the 27 (with
// its gather, split and scatter) had run 6 to 18 blocks at a time: one MVS step
// of Q5 on 16^3 cells took 118 ms that way, 4.7 ms in one launch per color.  There
// the 16 residuals take a third of the step and the tensor pipe is bound by the
// tiles of one to ten patches; on large runs the HMMA rate is the bound.
//
// FP32 (the mixed forms): FFMA with 8 x 8 outputs per thread, a 128 x 128 tile
// per block of 256 threads, 128-bit shared-memory operand loads, k-panels of 8,
// double-buffered.
#include <cuda_runtime.h>

#include <cuda_fp16.h>

#include <algorithm>
#include <cstdint>

#include "fx.cuh"
#include "kernels.cuh"
#include "ops.h"

namespace bh {
namespace {

__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void async_wait_group() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---- FP64 by FP16 slices ----------------------------------------------------
// One warp per column n of X (rows x cols, column-major, leading dimension
// rows): F[n] = e with max_k |X(k, n)| < 2^e, slices Xs[i][n][k] (leading
// dimension ldk >= rows, a multiple of 8; zero for k in [rows, ldk)).  The digits
// are taken from the value as a 54-bit integer: with 32 added to every digit
// they are its 6-bit fields.  A column with a value that is not finite becomes
// NaN.
__global__ void __launch_bounds__(256) slice_cols_kernel(const double* __restrict__ X, int rows,
                                                         int cols, int ldk, __half* __restrict__ Xs,
                                                         int* __restrict__ F) {
  const int col = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (col >= cols) return;
  const double* x = X + (int64_t)col * rows;
  unsigned mag = 0u;
  for (int k = lane; k < rows; k += 32) mag = max(mag, fx_mag(x[k]));
  mag = __reduce_max_sync(0xffffffffu, mag);
  const bool tiny = mag < (64u << 20);  // near the denormals: scaled by 2^200 first
  if (tiny) {
    mag = 0u;
    for (int k = lane; k < rows; k += 32) mag = max(mag, fx_mag(x[k] * 0x1p200));
    mag = __reduce_max_sync(0xffffffffu, mag);
  }
  const bool finite = mag < (0x7ffu << 20);
  const int e = mag ? (int)(mag >> 20) - 1022 : 0;
  if (lane == 0) F[col] = tiny ? e - 200 : e;
  const int64_t plane = (int64_t)cols * ldk;
  constexpr long long kOff = 0x820820820820ll;  // 32 in each of the eight digits below the first
  auto digits = [&](int k) -> long long {
    if (k >= rows) return kOff;
    const double v = tiny ? x[k] * 0x1p200 : x[k];
    return ((fx_from_double(v, fx_base(e, kSlices * kSliceBits + 1)) + 1) >> 1) + kOff;
  };
  for (int k = 2 * lane; k < ldk; k += 64) {
    const long long d0 = digits(k), d1 = digits(k + 1);
    __half* o = Xs + (int64_t)col * ldk + k;
#pragma unroll
    for (int i = 0; i < kSlices; ++i) {
      const int sh = kSliceBits * (kSlices - 1 - i);
      // a digit as the FP16 number 1536 + digit (units of one there)
      const int q0 = (int)(d0 >> sh), q1 = (int)(d1 >> sh);
      const int h0 = 0x6600 + (i == 0 ? q0 : (q0 & 63) - 32);
      const int h1 = 0x6600 + (i == 0 ? q1 : (q1 & 63) - 32);
      __half2_raw r;
      r.x = (unsigned short)(finite ? h0 : 0x7fff);
      r.y = (unsigned short)(finite ? h1 : 0x7fff);
      const __half2 v = __hsub2(__half2(r), __half2half2(__ushort_as_half(0x6600)));
      *reinterpret_cast<__half2*>(o + i * plane) = v;
    }
  }
}

struct SlicedCfg {
  static constexpr int BM = 64, BN = 32, BK = 16, THREADS = 256, STAGES = 2;
  static constexpr int LD = BK + 8;  // halves per shared-memory row (48 bytes: the eight rows
                                     // of an ldmatrix fall in distinct 16-byte banks)
  static constexpr int PART = 1472 / BK;  // inner panels whose level sums stay below 2^24
  static constexpr int SMEM = STAGES * kSlices * (BM + BN) * LD * 2;
};

__device__ __forceinline__ void async_copy16(void* dst, const void* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}

__device__ __forceinline__ void hmma_16x8x16(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t* r, const void* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}

// Y = alpha A R from the slices: As[slot][i][m][k] and Ea[slot][m] of the rows of
// the inverses, Rs[j][n][k] and Fr[n] of the columns of R (leading dimension ldk).
// A block computes the 64 x 32 tile of 64 rows and the columns of one GemmTile
// (one inverse) with 8 warps of 16 x 16, all slices of an inner panel of 16 in
// shared memory at once: each A fragment is loaded once and multiplied with the
// nine B slices held in registers, the products of a level in one accumulator.
__global__ void __launch_bounds__(SlicedCfg::THREADS, 2) gemm_sliced_kernel(
    int md, int cnt, int ldk, double alpha, const __half* __restrict__ As,
    const int* __restrict__ Ea, const __half* __restrict__ Rs, const int* __restrict__ Fr,
    const GemmTile* __restrict__ tiles, double* __restrict__ Y) {
  using C = SlicedCfg;
  constexpr int S = kSlices;
  extern __shared__ __align__(16) unsigned char gemm_smem[];
  __half* smem = reinterpret_cast<__half*>(gemm_smem);  // [stage][slice][BM + BN][LD]
  const GemmTile tile = tiles[blockIdx.y];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = (warp & 3) * 16, wn = (warp >> 2) * 16;
  const int bm0 = blockIdx.x * C::BM, bn0 = tile.col;
  const int nk = (ldk + C::BK - 1) / C::BK;
  const int64_t aplane = (int64_t)md * ldk, rplane = (int64_t)cnt * ldk;
  As += tile.slot * S * aplane;
  Ea += (int64_t)tile.slot * md;
  auto load = [&](int kt) {
    __half* st = smem + (kt % C::STAGES) * S * (C::BM + C::BN) * C::LD;
    for (int q = tid; q < S * (C::BM + C::BN) * 2; q += C::THREADS) {
      const int c = q & 1, row = q >> 1, sl = row / (C::BM + C::BN), r = row - sl * (C::BM + C::BN);
      const int gk = kt * C::BK + 8 * c;
      const bool isA = r < C::BM;
      const bool in = gk < ldk && (isA ? bm0 + r < md : r - C::BM < tile.cols);
      const __half* src = isA ? As + sl * aplane + (int64_t)(bm0 + r) * ldk
                              : Rs + sl * rplane + (int64_t)(bn0 + r - C::BM) * ldk;
      async_copy16(st + row * C::LD + 8 * c, in ? src + gk : As, in);
    }
    async_commit();
  };
  float acc[S][2][4];  // per level, 8-column half
  double out[2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      out[h][c] = 0.0;
#pragma unroll
      for (int l = 0; l < S; ++l) acc[l][h][c] = 0.f;
    }
  load(0);
  for (int kt = 0; kt < nk; ++kt) {
    if (kt + 1 < nk) {
      load(kt + 1);
      async_wait_group<1>();
    } else {
      async_wait_group<0>();
    }
    __syncthreads();
    const __half* st = smem + (kt % C::STAGES) * S * (C::BM + C::BN) * C::LD;
    // fragments: A rows wm + (lane % 16), columns 8 (lane / 16); B as the four 8 x 8
    // blocks (columns 0-7, 8-15) x (k 0-7, 8-15)
    const __half* pa = st + (wm + (lane & 15)) * C::LD + 8 * (lane >> 4);
    const __half* pb =
        st + (C::BM + wn + (lane & 7) + 8 * (lane >> 4)) * C::LD + 8 * ((lane >> 3) & 1);
    uint32_t b[S][4];
#pragma unroll
    for (int j = 0; j < S; ++j) ldmatrix_x4(b[j], pb + j * (C::BM + C::BN) * C::LD);
#pragma unroll
    for (int i = 0; i < S; ++i) {
      uint32_t a[4];
      ldmatrix_x4(a, pa + i * (C::BM + C::BN) * C::LD);
#pragma unroll
      for (int j = 0; i + j < S; ++j) {
        hmma_16x8x16(acc[i + j][0], a, b[j]);
        hmma_16x8x16(acc[i + j][1], a, b[j] + 2);
      }
    }
    __syncthreads();  // the stage is overwritten by the copy two panels ahead
    if (kt == nk - 1 || (kt + 1) % C::PART == 0) {  // exact integers so far
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          // levels 0..3 in units of level 3, 4..8 in units of level 8
          long long hi = 0, lo = 0;
          bool nan = false;
#pragma unroll
          for (int l = 0; l < S; ++l) {
            const float f = acc[l][h][c];
            nan |= !(f == f);
            if (l < 4)
              hi = hi * (1 << kSliceBits) + __float2int_rn(f);
            else
              lo = lo * (1 << kSliceBits) + __float2int_rn(f);
            acc[l][h][c] = 0.f;
          }
          // level l counts 2^(-6 (l + 2))
          out[h][c] = fma((double)hi, 0x1p-30, out[h][c]);
          out[h][c] = fma((double)lo, 0x1p-60, out[h][c]);
          if (nan) out[h][c] = __longlong_as_double(0x7ff8000000000000ll);
        }
    }
  }
  // D fragment c: row g (+ 8 for c >= 2), column 2t + (c & 1)
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int gm = bm0 + wm + g + (c >= 2 ? 8 : 0);
      const int ln = wn + 8 * h + 2 * t + (c & 1);
      if (gm < md && ln < tile.cols)
        Y[(int64_t)(bn0 + ln) * md + gm] = alpha * ldexp(out[h][c], Ea[gm] + Fr[bn0 + ln]);
    }
}

// ---- FP32: FFMA, 8 x 8 per thread --------------------------------------------
struct GemmF32Cfg {
  static constexpr int BM = 128, BN = 128, BK = 8, PAD = 4, THREADS = 256;
  static constexpr int LDA = BM + PAD, LDB = BN + PAD;
};

__global__ void __launch_bounds__(GemmF32Cfg::THREADS) gemm_f32_kernel(int md, int cnt,
                                                                       float alpha,
                                                                       const float* __restrict__ A,
                                                                       const float* __restrict__ R,
                                                                       float* __restrict__ Y) {
  using C = GemmF32Cfg;
  __shared__ __align__(16) float As[2][C::BK][C::LDA];
  __shared__ __align__(16) float Bs[2][C::BK][C::LDB];
  const int tid = threadIdx.x;
  const int tm = tid & 15, tn = tid >> 4;  // rows 4 tm + {0..3} and 64 + 4 tm + {0..3}; same for n
  const int bm0 = blockIdx.x * C::BM, bn0 = blockIdx.y * C::BN;
  const int nk = (md + C::BK - 1) / C::BK;

  auto load = [&](int s, int k0) {
    for (int e = tid; e < C::BK * C::BM; e += C::THREADS) {
      const int k = e / C::BM, m = e % C::BM;
      const int gm = bm0 + m, gk = k0 + k;
      const bool in = gm < md && gk < md;
      async_copy_or_zero(&As[s][k][m], A + (in ? (int64_t)gk * md + gm : 0), in);
    }
    for (int e = tid; e < C::BK * C::BN; e += C::THREADS) {
      const int k = e % C::BK, n = e / C::BK;
      const int gk = k0 + k, gn = bn0 + n;
      const bool in = gk < md && gn < cnt;
      async_copy_or_zero(&Bs[s][k][n], R + (in ? (int64_t)gn * md + gk : 0), in);
    }
    async_commit();
  };

  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;

  load(0, 0);
  for (int kt = 0; kt < nk; ++kt) {
    const int s = kt & 1;
    if (kt + 1 < nk) {
      load(s ^ 1, (kt + 1) * C::BK);
      async_wait_group<1>();
    } else {
      async_wait_group<0>();
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < C::BK; ++k) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[s][k][4 * tm]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[s][k][64 + 4 * tm]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[s][k][4 * tn]);
      const float4 b1 = *reinterpret_cast<const float4*>(&Bs[s][k][64 + 4 * tn]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int gm = bm0 + (i < 4 ? 4 * tm + i : 64 + 4 * tm + i - 4);
    if (gm >= md) continue;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int gn = bn0 + (j < 4 ? 4 * tn + j : 64 + 4 * tn + j - 4);
      if (gn < cnt) Y[(int64_t)gn * md + gm] = alpha * acc[i][j];
    }
  }
}

}  // namespace

int slice_ld(int rows) { return (rows + 7) / 8 * 8; }

cudaError_t slice_cols(const double* X, int rows, int cols, uint16_t* Xs, int* F,
                       cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return cudaSuccess;
  const int64_t threads = (int64_t)cols * 32;
  slice_cols_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(
      X, rows, cols, slice_ld(rows), reinterpret_cast<__half*>(Xs), F);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

int gemm_tile_cols() { return SlicedCfg::BN; }

cudaError_t gemm_f64_sliced(int md, int cnt, double alpha, const uint16_t* As, const int* Ea,
                            const uint16_t* Rs, const int* Fr, const GemmTile* tiles, int ntiles,
                            double* Y, cudaStream_t st) {
  if (md <= 0 || cnt <= 0 || ntiles <= 0) return cudaSuccess;
  using C = SlicedCfg;
  static const cudaError_t attr = cudaFuncSetAttribute(
      gemm_sliced_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (attr != cudaSuccess) return attr;
  for (int t0 = 0; t0 < ntiles; t0 += 65535) {
    const dim3 grid((unsigned)((md + C::BM - 1) / C::BM), (unsigned)std::min(ntiles - t0, 65535));
    gemm_sliced_kernel<<<grid, C::THREADS, C::SMEM, st>>>(
        md, cnt, slice_ld(md), alpha, reinterpret_cast<const __half*>(As), Ea,
        reinterpret_cast<const __half*>(Rs), Fr, tiles + t0, Y);
    g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  }
  return cudaGetLastError();
}

cudaError_t gemm_f32(int md, int cnt, float alpha, const float* A, const float* R, float* Y,
                     cudaStream_t st) {
  if (md <= 0 || cnt <= 0) return cudaSuccess;
  using C = GemmF32Cfg;
  const dim3 grid((unsigned)((md + C::BM - 1) / C::BM), (unsigned)((cnt + C::BN - 1) / C::BN));
  if (grid.y > 65535u) return cudaErrorInvalidValue;
  gemm_f32_kernel<<<grid, C::THREADS, 0, st>>>(md, cnt, alpha, A, R, Y);
  g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

}  // namespace bh
