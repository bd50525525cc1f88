// Plain FP32 CUDA-core gemm, the reference form of C = alpha * A * B + beta * C
// (the kind of kernel the paper generates for its GPU target, Section V-B).
//
// Two-level tiling: 128 x 128 output tiles per CTA (64 x 64 when those would
// leave SMs without work), a 16-deep k-slice staged in shared memory (double
// buffered, next slice prefetched into registers while the current one is
// consumed), and register blocking of 8 x 8 (8 x 4) outputs per thread, two
// neighbouring columns per packed FP32 multiply-add (fma.rn.f32x2: the two
// roundings of two fmaf, in half the instructions; storing one operand twice
// in shared memory, to save the register copies that make a pair of one
// value, was bound by the extra reads: 1024^3 79 us against 60).  Full tiles (all 128 rows and columns in range, k-slice
// complete) take unpredicated, vectorised loads when the leading dimensions
// allow it; partial tiles predicate every access.  The full/partial choice is
// uniform per CTA, so it introduces no divergence.  TA / TB: A stored K x M
// (lda >= M), B stored N x K (ldb >= K); the slices are loaded along the
// stored rows and land in the same shared-memory layout, so the arithmetic
// (and its order) is that of the untransposed kernel.
#include <cuda_runtime.h>

#include "internal.h"

namespace gb {

namespace {

// Bound by instruction issue: a thread's 8 x 4 columns take 16 packed
// multiply-adds a k, beside three shared-memory reads and the copies that pair
// up A's values.  1024^3: 102.5 us with 128 x 128 tiles and single
// multiply-adds (64 CTAs), 59.4 with 64 x 64 tiles and packed ones (256 CTAs);
// 4096 x 4096 x 2048 46.8 -> 56.8 TFLOP/s.  Prefetching two slices instead of
// one changed nothing.
// (a 16-deep slice reads 64 contiguous bytes of each row of A: 8192^3 ran 5 %
// faster than with an 8-deep one)
constexpr int BKs = 16;

// Square tiles of TILE outputs a side; a thread holds 8 rows x TN columns.
template <int TILE>
struct SimtCfg {
  static constexpr int TN = TILE == 128 ? 8 : 4;
  static constexpr int THREADS = (TILE / 8) * (TILE / TN);
  static constexpr int CTAS = TILE == 128 ? 2 : 4;   // a SM, by registers
  static constexpr int LQ = TILE / 4;                // threads along a row of 4-float loads
  static_assert(THREADS == 8 * LQ && THREADS == 2 * TILE, "slice loads: 8 floats a thread");
};

// (a.x b.x + c.x, a.y b.y + c.y), each rounded once, to nearest even.
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
  return d;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

struct Frag {
  float a[8];
  float b[8];
};

// Four consecutive floats of a stored row (row r, columns c..c+3), in range
// when r < rows and c + i < cols.
template <bool FULL, bool VEC>
__device__ __forceinline__ void load4(float* v, const float* __restrict__ X, int64_t ld,
                                      int64_t r, int64_t c, int64_t rows, int64_t cols) {
  if (FULL && VEC) {
    const float4 q = *reinterpret_cast<const float4*>(X + r * ld + c);
    v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
  } else if (FULL) {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = X[r * ld + c + i];
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = (r < rows && c + i < cols) ? X[r * ld + c + i] : 0.0f;
  }
}

// Load the A slice (TILE rows x 16 k) and B slice (16 k x TILE cols) of one
// k-step into registers, along the stored rows.  A row-major: thread t loads
// row t/2, k (t%2)*8..+7; A stored K x M: k-rows t/LQ and t/LQ + 8, m
// (t%LQ)*4..+3.  B row-major: k-rows t/LQ and t/LQ + 8, columns
// (t%LQ)*4..+3; B stored N x K: column t/2, k (t%2)*8..+7.
template <int TILE, bool FULL, bool VEC, bool TA, bool TB>
__device__ __forceinline__ void load_slice(Frag& f, const float* __restrict__ A, int64_t lda,
                                           const float* __restrict__ B, int64_t ldb, int64_t M,
                                           int64_t N, int64_t K, int64_t m0, int64_t n0,
                                           int64_t k0, int tid) {
  const int hi2 = tid >> 1, lo2 = (tid & 1) * 8;
  const int hi32 = tid / SimtCfg<TILE>::LQ, lo32 = (tid % SimtCfg<TILE>::LQ) * 4;
  if (TA) {
    load4<FULL, VEC>(f.a, A, lda, k0 + hi32, m0 + lo32, K, M);
    load4<FULL, VEC>(f.a + 4, A, lda, k0 + hi32 + 8, m0 + lo32, K, M);
  } else {
    load4<FULL, VEC>(f.a, A, lda, m0 + hi2, k0 + lo2, M, K);
    load4<FULL, VEC>(f.a + 4, A, lda, m0 + hi2, k0 + lo2 + 4, M, K);
  }
  if (TB) {
    load4<FULL, VEC>(f.b, B, ldb, n0 + hi2, k0 + lo2, N, K);
    load4<FULL, VEC>(f.b + 4, B, ldb, n0 + hi2, k0 + lo2 + 4, N, K);
  } else {
    load4<FULL, VEC>(f.b, B, ldb, k0 + hi32, n0 + lo32, K, N);
    load4<FULL, VEC>(f.b + 4, B, ldb, k0 + hi32 + 8, n0 + lo32, K, N);
  }
}

// Into shared memory, As[k][m] and Bs[k][n] whatever the stored layout.
template <int TILE, bool TA, bool TB>
__device__ __forceinline__ void store_slice(const Frag& f, float (*As)[TILE], float (*Bs)[TILE],
                                            int tid) {
  const int hi2 = tid >> 1, lo2 = (tid & 1) * 8;
  const int hi32 = tid / SimtCfg<TILE>::LQ, lo32 = (tid % SimtCfg<TILE>::LQ) * 4;
  if (TA) {
    *reinterpret_cast<float4*>(&As[hi32][lo32]) = make_float4(f.a[0], f.a[1], f.a[2], f.a[3]);
    *reinterpret_cast<float4*>(&As[hi32 + 8][lo32]) = make_float4(f.a[4], f.a[5], f.a[6], f.a[7]);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) As[lo2 + i][hi2] = f.a[i];
  }
  if (TB) {
#pragma unroll
    for (int i = 0; i < 8; ++i) Bs[lo2 + i][hi2] = f.b[i];
  } else {
    *reinterpret_cast<float4*>(&Bs[hi32][lo32]) = make_float4(f.b[0], f.b[1], f.b[2], f.b[3]);
    *reinterpret_cast<float4*>(&Bs[hi32 + 8][lo32]) = make_float4(f.b[4], f.b[5], f.b[6], f.b[7]);
  }
}

// As, Bs: the kernel's double-buffered shared slices ([2][BKs][TILE] each),
// declared once for both tile paths.
template <int TILE, bool FULL, bool VEC, bool TA, bool TB>
__device__ __forceinline__ void gemm_tile(int64_t M, int64_t N, int64_t K, float alpha,
                                          const float* __restrict__ A, int64_t lda,
                                          const float* __restrict__ B, int64_t ldb, float beta,
                                          float* __restrict__ C, int64_t ldc, int64_t m0,
                                          int64_t n0, bool cvec, float (*As)[BKs][TILE],
                                          float (*Bs)[BKs][TILE]) {
  constexpr int TN = SimtCfg<TILE>::TN;
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  unsigned long long acc[8][TN / 2];   // two columns each
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;

  const int64_t kfull = K / BKs;          // complete k-slices
  const int64_t ksteps = (K + BKs - 1) / BKs;
  Frag f;
  auto load = [&](int64_t ks) {
    if (ks < kfull)
      load_slice<TILE, FULL, VEC, TA, TB>(f, A, lda, B, ldb, M, N, K, m0, n0, ks * BKs, tid);
    else
      load_slice<TILE, false, false, TA, TB>(f, A, lda, B, ldb, M, N, K, m0, n0, ks * BKs, tid);
  };
  load(0);
  store_slice<TILE, TA, TB>(f, As[0], Bs[0], tid);
  __syncthreads();

  for (int64_t ks = 0; ks < ksteps; ++ks) {
    const int cur = ks & 1;
    if (ks + 1 < ksteps) load(ks + 1);
#pragma unroll
    for (int k = 0; k < BKs; ++k) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[cur][k][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[cur][k][TILE / 2 + ty * 4]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      unsigned long long bv[TN / 2];
#pragma unroll
      for (int h = 0; h < TN / 4; ++h) {
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(&Bs[cur][k][h * (TILE / 2) + tx * 4]);
        bv[2 * h] = b.x, bv[2 * h + 1] = b.y;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const unsigned long long aa = pack2(av[i], av[i]);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = fma2(aa, bv[j], acc[i][j]);
      }
    }
    if (ks + 1 < ksteps) {
      store_slice<TILE, TA, TB>(f, As[cur ^ 1], Bs[cur ^ 1], tid);
      __syncthreads();
    }
  }

  // epilogue: rows ty*4+i (+TILE/2), columns tx*4+j (+TILE/2)
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int64_t row = m0 + (i < 4 ? ty * 4 + i : TILE / 2 + ty * 4 + (i - 4));
    if (!FULL && row >= M) continue;
    float* crow = C + row * ldc;
#pragma unroll
    for (int h = 0; h < TN / 4; ++h) {
      const int64_t col = n0 + h * (TILE / 2) + tx * 4;
      const float2 lo = unpack2(acc[i][2 * h]), hi = unpack2(acc[i][2 * h + 1]);
      const float a4[4] = {lo.x, lo.y, hi.x, hi.y};
      if (FULL && cvec) {
        float4* cp = reinterpret_cast<float4*>(crow + col);
        float4 o;
        if (beta != 0.0f) {
          const float4 old = *cp;
          o = make_float4(fmaf(alpha, a4[0], beta * old.x), fmaf(alpha, a4[1], beta * old.y),
                          fmaf(alpha, a4[2], beta * old.z), fmaf(alpha, a4[3], beta * old.w));
        } else {
          o = make_float4(alpha * a4[0], alpha * a4[1], alpha * a4[2], alpha * a4[3]);
        }
        *cp = o;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (FULL || col + j < N) {
            float* cp = crow + col + j;
            *cp = beta != 0.0f ? fmaf(alpha, a4[j], beta * *cp) : alpha * a4[j];
          }
        }
      }
    }
  }
}

template <int TILE, bool VEC, bool TA, bool TB>
__global__ void __launch_bounds__(SimtCfg<TILE>::THREADS, SimtCfg<TILE>::CTAS)
    simt_gemm_kernel(int64_t M, int64_t N, int64_t K, float alpha, const float* A, int64_t lda, const float* B,
                     int64_t ldb, float beta, float* C, int64_t ldc, bool cvec) {
  __shared__ __align__(16) float As[2][BKs][TILE];
  __shared__ __align__(16) float Bs[2][BKs][TILE];
  const int64_t m0 = static_cast<int64_t>(blockIdx.y) * TILE;
  const int64_t n0 = static_cast<int64_t>(blockIdx.x) * TILE;
  if (m0 + TILE <= M && n0 + TILE <= N)
    gemm_tile<TILE, true, VEC, TA, TB>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, m0, n0, cvec, As, Bs);
  else
    gemm_tile<TILE, false, VEC, TA, TB>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, m0, n0, cvec, As, Bs);
}

template <int TILE, bool TA, bool TB>
cudaError_t simt_launch_tile(bool vec, int64_t M, int64_t N, int64_t K, float alpha, const float* A, int64_t lda,
                             const float* B, int64_t ldb, float beta, float* C, int64_t ldc, bool cvec,
                             cudaStream_t s) {
  const dim3 grid(static_cast<unsigned>((N + TILE - 1) / TILE), static_cast<unsigned>((M + TILE - 1) / TILE));
  constexpr int THREADS = SimtCfg<TILE>::THREADS;
  if (vec)
    simt_gemm_kernel<TILE, true, TA, TB><<<grid, THREADS, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, cvec);
  else
    simt_gemm_kernel<TILE, false, TA, TB><<<grid, THREADS, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, cvec);
  return cudaGetLastError();
}

template <bool TA, bool TB>
cudaError_t simt_launch(bool small, bool vec, int64_t M, int64_t N, int64_t K, float alpha, const float* A,
                        int64_t lda, const float* B, int64_t ldb, float beta, float* C, int64_t ldc, bool cvec,
                        cudaStream_t s) {
  return small ? simt_launch_tile<64, TA, TB>(vec, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, cvec, s)
               : simt_launch_tile<128, TA, TB>(vec, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, cvec, s);
}

__global__ void scale_c_kernel(int64_t M, int64_t N, float beta, float* C, int64_t ldc) {
  const int64_t total = M * N;
  for (int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; idx < total;
       idx += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    float* cp = C + (idx / N) * ldc + idx % N;
    *cp = beta != 0.0f ? beta * *cp : 0.0f;
  }
}

}  // namespace

cudaError_t simt_gemm_launch(int64_t M, int64_t N, int64_t K, float alpha, const float* A,
                             int64_t lda, const float* B, int64_t ldb, float beta, float* C,
                             int64_t ldc, int sms, cudaStream_t s, bool transA, bool transB) {
  if ((M + 127) / 128 > 65535) return cudaErrorInvalidConfiguration;
  // 64 x 64 tiles when the fullest SM then has fewer outputs to compute.
  // Their operand traffic a multiply-add is twice as high: a tenth more work
  // with 16-byte loads, 1.6 times as much with 4-byte ones (unaligned rows:
  // at 1.1, 4099 x 1001 x 700 took 203 us against 164 with 128 x 128 tiles).
  const int64_t t128 = ((M + 127) / 128) * ((N + 127) / 128), t64 = ((M + 63) / 64) * ((N + 63) / 64);
  const int64_t w128 = (t128 + sms - 1) / sms * 128 * 128, w64 = (t64 + sms - 1) / sms * 64 * 64;
  const bool vec = (lda % 4 == 0) && (ldb % 4 == 0) &&
                   (reinterpret_cast<uintptr_t>(A) % 16 == 0) &&
                   (reinterpret_cast<uintptr_t>(B) % 16 == 0);
  const bool small = w64 * (vec ? 11 : 16) < w128 * 10 && (M + 63) / 64 <= 65535;
  const bool cvec = (ldc % 4 == 0) && (reinterpret_cast<uintptr_t>(C) % 16 == 0);
  if (transA && transB) return simt_launch<true, true>(small, vec, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, cvec, s);
  if (transA) return simt_launch<true, false>(small, vec, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, cvec, s);
  if (transB) return simt_launch<false, true>(small, vec, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, cvec, s);
  return simt_launch<false, false>(small, vec, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, cvec, s);
}

cudaError_t scale_c_launch(int64_t M, int64_t N, float beta, float* C, int64_t ldc, cudaStream_t s) {
  const int64_t total = M * N;
  int64_t blocks = (total + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  scale_c_kernel<<<static_cast<int>(blocks), 256, 0, s>>>(M, N, beta, C, ldc);
  return cudaGetLastError();
}

}  // namespace gb
