// Split-precision gemm without a packing pass: C = alpha * op(A) * op(B) +
// beta * C in BF16X3, one launch, for tall thin products and small ones.
//
// The packed path reads A, writes its planes and reads them again: on 50176 x
// 64 x 576 its two kernels take 41 + 28 us for operands that cross HBM in 19.
// Here TMA brings 32-deep FP32 items of both operands into a staging ring, the
// split warps write them as hi and lo parts in the unswizzled core-matrix
// layout, and the MMAs read those:
//   * an operand whose stored rows run along K (A, or B given transposed) is
//     written K-major, one whose rows run along M or N (B, or A given
//     transposed) MN-major: the same code, as a 16-byte chunk of eight
//     neighbouring stored values is a row of a core matrix either way, and no
//     transpose is ever done;
//   * the products, their order and the folds out of tensor memory are the
//     packed kernel's, so the results of unscaled operands are the same bits; a
//     plan takes this kernel for the calls whose rows TMA can load and the packed
//     path for the others.
//
// Turned tiles: the last rows of A, at most 64, may be computed transposed (see
// direct_grid): the operands change places, the products keep their order, and the
// sums leave along the rows of C.
//
// Scaling: a tile covers all of K, so its split warps see the maximum of its
// 128 rows of A and BN columns of B; if either lies outside the unscaled range
// the tile is computed once more with the exponents (nothing has been stored
// by then), its values read straight from global memory, so that the ring's
// loads for the next tile stay where they are.  (1024^3 with all of A out of the
// range takes 53 us for 19, packed 53; with one block of 128 rows 53, packed 42.)
//
// Bounded by shared-memory bandwidth (an item of a 128 x 64 tile crosses it four
// times: copied in, read, written as parts, read by the MMAs, about 850 cycles;
// 1050 measured) and next by HBM.  50176 x 64 x 576: 72.6 -> 35.7 us a call.
// Register-staged plain loads instead of TMA took 55 us there (latency),
// cp.async by the split warps 77 (their proxy fence waits for the copies in
// flight).
//
// Roles (768 threads): warps 0..15 split (four groups of four, each taking every
// fourth item: a group's reads, conversions and writes are a chain of latencies,
// and with two groups the tall thin product above took 42 us), 16..19 epilogue,
// 20 MMAs and tensor memory, 21 loads (22 and 23 only give their registers).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "epilogue.cuh"
#include "internal.h"
#include "ptx.cuh"
#include "scale.cuh"
#include "split_arith.cuh"

namespace gb {

namespace {

constexpr int kDirThreads = 768;
constexpr int kGroups = 4, kSplitThreads = 128;   // split groups, threads of one
constexpr int kEpiWarp0 = 16, kMmaWarp = 20, kLoadWarp = 21;
// registers a thread: the launch's 80 x 768, shared out by warpgroup
constexpr int kRegsSplit = 80, kRegsEpi = 120, kRegsCtrl = 40;
static_assert(kGroups * kRegsSplit + kRegsEpi + kRegsCtrl <= 6 * 80, "register split");
constexpr int kKI = 32;                    // K of an item
constexpr int kStages = kGroups, kDirSlots = kGroups;   // a group's items all pass through the same of each
constexpr int kVerdicts = 16;
// bytes between 16-byte chunks of an item, 32 modulo 128: the stores of eight
// lanes (four chunks of two stored rows) fall into different banks
constexpr int kChbK = 128 * 16 + 32;       // K-major A: chunks of 8 k, 128 rows
constexpr int kChbMn = kKI * 16 + 32;      // MN-major: chunks of 8 rows, 32 k

template <int BN>
struct DirCfg {
  static constexpr int CHB_BK = BN * 16 + 32;                 // K-major B
  static constexpr int A_PLANE = 8704;                        // 16 chunks of kChbMn, 4 of kChbK
  static constexpr int B_PLANE = (BN / 8 * kChbMn + 127) / 128 * 128;
  static constexpr int SLOT = 2 * (A_PLANE + B_PLANE);
  static constexpr int ITEM_A = 128 * kKI * 4, ITEM = (128 + BN) * kKI * 4;   // FP32 bytes
  static constexpr int EPI_PITCH = 33;
  static constexpr int EPI_BYTES = 4 * 32 * EPI_PITCH * 4;
  static constexpr int OFF_SLOT = kStages * ITEM;
  static constexpr int OFF_EPI = OFF_SLOT + kDirSlots * SLOT;
  static constexpr int OFF_BAR = (OFF_EPI + EPI_BYTES + 127) / 128 * 128;
  static constexpr int SMEM = OFF_BAR + 512 + 1024;
  static constexpr int NACC = 4, TMEM_COLS = NACC * BN;
  static_assert(16 * kChbMn <= A_PLANE && 4 * kChbK <= A_PLANE && 4 * CHB_BK <= B_PLANE &&
                    (BN / 8) * kChbMn <= B_PLANE && A_PLANE % 128 == 0 && B_PLANE % 128 == 0,
                "slot");
  static_assert(SMEM <= 231424 && ITEM % 1024 == 0, "shared memory");
};

// A staged operand is a run of 128-byte rows of 32 neighbouring stored values
// (K-major: the operand's rows; MN-major: piece by piece of 32 rows, its k), in
// the 128-byte swizzle.  A split thread's unit n is the quarter row t + 128 n:
// eight values, read as two 16-byte accesses free of bank conflicts, which
// become a 16-byte chunk of each plane.
struct Units {
  uint32_t src0;         // the first half's place; unit n is 4096 n bytes on
  uint32_t dst0, step;   // unit n's chunk: dst0 + n * step
};
__device__ __forceinline__ Units make_units(bool mn, uint32_t chb_k, int t) {
  Units u;
  const int r = t / 4, j = t % 4;
  u.src0 = r * 128 + ((2 * j) ^ (r & 7)) * 16;
  u.dst0 = j * (mn ? kChbMn : chb_k) + r * 16;
  u.step = mn ? 4 * kChbMn : 32 * 16;
  return u;
}

template <int N>
__device__ __forceinline__ void read_units(float (&v)[N][8], const uint8_t* src, const Units& u) {
#pragma unroll
  for (int n = 0; n < N; ++n) {
    const float4 a = *reinterpret_cast<const float4*>(src + (u.src0 + 4096 * n));
    const float4 b = *reinterpret_cast<const float4*>(src + ((u.src0 ^ 16u) + 4096 * n));
    v[n][0] = a.x, v[n][1] = a.y, v[n][2] = a.z, v[n][3] = a.w;
    v[n][4] = b.x, v[n][5] = b.y, v[n][6] = b.z, v[n][7] = b.w;
  }
}

// The units' values from global memory, zero outside the operand: row r0 and
// k-range from k0 on of X (stored K x rows if mn).
template <int N>
__device__ __forceinline__ void fetch_units(float (&v)[N][8], const float* X, int64_t ld, int rows, int K, bool mn,
                                            int r0, int k0, int t) {
#pragma unroll
  for (int n = 0; n < N; ++n) {
    const int o = (mn ? k0 : r0 + 32 * n) + t / 4, in = (mn ? r0 + 32 * n : k0) + t % 4 * 8;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      v[n][e] = o < (mn ? K : rows) && in + e < (mn ? rows : K) ? X[static_cast<int64_t>(o) * ld + in + e] : 0.0f;
  }
}

template <int N>
__device__ __forceinline__ float max_units(const float (&v)[N][8]) {
  float m = 0.0f;
#pragma unroll
  for (int n = 0; n < N; ++n)
#pragma unroll
    for (int k = 0; k < 8; ++k) m = fmaxf(m, fabsf(v[n][k]));
  return m;
}

// Splits the units' values (times sf; m: their maximum) into hi parts at dst and
// lo parts `plane` bytes further on.
template <int N>
__device__ __forceinline__ void write_units(float (&v)[N][8], float m, const Units& u, uint8_t* dst, uint32_t plane,
                                            float sf) {
  if (sf != 1.0f) {
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
      for (int k = 0; k < 8; ++k) v[n][k] *= sf;
  }
  const bool finite = m < __uint_as_float(0x7F800000u);
#pragma unroll
  for (int n = 0; n < N; ++n) {
    uint4 h, l;
    split_chunk_bf16(v[n], finite, h, l);
    *reinterpret_cast<uint4*>(dst + (u.dst0 + n * u.step)) = h;
    *reinterpret_cast<uint4*>(dst + (u.dst0 + n * u.step) + plane) = l;
  }
}

// Epilogue of a turned tile: this thread's sums are those of column col of C, in
// rows row0 .. row0 + BN - 1; a warp's accesses are 128 contiguous bytes of a row.
template <int BN>
__device__ __forceinline__ void store_turned(float (&S)[BN], const DirectArgs& a, int e, int row0, int col) {
  const int rows = col < a.N ? a.M - row0 : 0;
  float alpha = a.alpha;
  if (e != 0) {   // (as epilogue_store)
#pragma unroll
    for (int i = 0; i < BN; ++i) S[i] = scale_pow2(alpha * S[i], e);
    alpha = 1.0f;
  }
  const float* in = a.C + static_cast<int64_t>(row0) * a.ldc + col;
  float* out = const_cast<float*>(in);
#pragma unroll
  for (int j = 0; j < BN; j += 8) {
    float old[8];
    if (a.beta != 0.0f) {
#pragma unroll
      for (int k = 0; k < 8; ++k, in += a.ldc) old[k] = j + k < rows ? *in : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k, out += a.ldc)
      if (j + k < rows) *out = a.beta != 0.0f ? fmaf(alpha, S[j + k], a.beta * old[k]) : alpha * S[j + k];
  }
}

// TURN: launches with turned tiles.
template <int BN, bool TURN>
__global__ void __launch_bounds__(kDirThreads, 1)
    tc_direct_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const DirectArgs a) {
  using Cfg = DirCfg<BN>;
  constexpr int NACC = Cfg::NACC;
  constexpr int BOX_A = TURN ? BN : 128;   // rows of a K-major box of the operand in A's place
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t sbase = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (sbase - raw);
  const uint32_t bar0 = sbase + Cfg::OFF_BAR;
  auto sfull = [&](int i) { return bar0 + 8u * i; };
  auto sempty = [&](int i) { return bar0 + 8u * (kStages + i); };
  constexpr int B1 = 2 * kStages;
  auto full = [&](int i) { return bar0 + 8u * (B1 + i); };
  auto empty = [&](int i) { return bar0 + 8u * (B1 + kDirSlots + i); };
  constexpr int B2 = B1 + 2 * kDirSlots;
  auto accf = [&](int i) { return bar0 + 8u * (B2 + i); };
  auto acce = [&](int i) { return bar0 + 8u * (B2 + NACC + i); };
  auto vbar = [&](int i) { return bar0 + 8u * (B2 + 2 * NACC + i); };
  const uint32_t drain_bar = bar0 + 8u * (B2 + 2 * NACC + kVerdicts);
  constexpr int NBAR = B2 + 2 * NACC + kVerdicts + 1;
  static_assert(8 * NBAR + 16 + 8 * kVerdicts <= 512, "barrier block");
  unsigned* const vmax = reinterpret_cast<unsigned*>(smem + Cfg::OFF_BAR + 8 * NBAR);   // [kVerdicts][2]
  uint32_t* const tmem_slot = vmax + 2 * kVerdicts;
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* const err = a.err;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) mbar_init(sfull(i), 1), mbar_init(sempty(i), 4);
    for (int i = 0; i < kDirSlots; ++i) mbar_init(full(i), 4), mbar_init(empty(i), 1);
    for (int i = 0; i < NACC; ++i) mbar_init(accf(i), 1), mbar_init(acce(i), 4);
    for (int i = 0; i < kVerdicts; ++i) mbar_init(vbar(i), 4 * kGroups), vmax[2 * i] = vmax[2 * i + 1] = 0u;
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(smem_u32(tmem_slot), Cfg::TMEM_COLS);
    tmem_relinquish();
  }
  if (warp == kLoadWarp && lane == 0) {      // kernel parameters: fetched meanwhile
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  griddep_wait();                     // the operands may be the previous kernel's output
  griddep_launch_dependents();

  const int items = (a.K + kKI - 1) / kKI;
  const int plain = a.tiles_m * a.tiles_n;
  const int units = plain + (TURN ? a.turned : 0);
  const int fold = a.fold * (64 / kKI);
  // tile of unit u: rows fastest, so that CTAs running together share columns of B.
  // Returns whether it is turned: 128 columns of B from m0 on take A's place and
  // the last rows of A, from n0 on, take B's (the product transposed).
  auto tile = [&](int u, int& m0, int& n0) {
    if (TURN && u >= plain) {
      m0 = (u - plain) * 128, n0 = a.tiles_m * 128;
      return true;
    }
    const int tn = u / a.tiles_m;
    m0 = (u - tn * a.tiles_m) * 128, n0 = tn * BN;
    return false;
  };
  // whether the operand in A's (B's) place runs along M or N in its rows
  auto mn_a = [&](bool turned) { return turned ? a.transB == 0 : a.transA != 0; };
  auto mn_b = [&](bool turned) { return turned ? a.transA != 0 : a.transB == 0; };
  // a unit's exponents, once its maxima are known (seq: the CTA's unit count)
  auto exponents = [&](int seq, int& eA, int& eB) {
    const volatile unsigned* v = vmax + 2 * (seq % kVerdicts);
    eA = block_exponent(v[0]), eB = block_exponent(v[1]);
  };

  if (warp >= kMmaWarp) {
    warpgroup_regs_dec<kRegsCtrl>();
  if (warp == kLoadWarp) {
    // ----------------------------------------------------------------- loads
    if (elect_one()) {
      uint32_t it = 0;
      bool ok = true;
      for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
        int m0, n0;
        const bool turned = tile(u, m0, n0);
        const bool mnA = mn_a(turned), mnB = mn_b(turned);
        const CUtensorMap* const mapA = turned ? &tmB : &tmA;
        const CUtensorMap* const mapB = turned ? &tmA : &tmB;
        for (int c = 0; c < items; ++c, ++it) {
          const uint32_t s = it % kStages;
          if (!(ok = mbar_wait(sempty(s), ((it / kStages) & 1u) ^ 1u, abort_flag, err))) break;
          const uint32_t dst = sbase + s * Cfg::ITEM;
          mbar_arrive_expect_tx(sfull(s), Cfg::ITEM);
          // boxes of 32 stored values: the operand's rows, or pieces of 32 rows of k
          if (mnA) {
#pragma unroll
            for (int b = 0; b < 4; ++b) tma_load_3d(dst + b * 4096, mapA, sfull(s), m0 + 32 * b, kKI * c, 0);
          } else {
#pragma unroll
            for (int b = 0; b < 128; b += BOX_A)
              tma_load_3d(dst + b * 128, mapA, sfull(s), kKI * c, m0 + b, 0);
          }
          if (!mnB) {
            tma_load_3d(dst + Cfg::ITEM_A, mapB, sfull(s), kKI * c, n0, 0);
          } else {
#pragma unroll
            for (int b = 0; b < BN / 32; ++b)
              tma_load_3d(dst + Cfg::ITEM_A + b * 4096, mapB, sfull(s), n0 + 32 * b, kKI * c, 0);
          }
        }
      }
      if (!ok) {
        // abort: let the copies issued land before shared memory is released
        for (uint32_t k = it > kStages ? it - kStages : 0; k < it; ++k)
          mbar_wait_drain(sfull(k % kStages), (k / kStages) & 1u);
      }
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------ MMA issuer
    if (elect_one()) {
      const uint32_t s0 = sbase + Cfg::OFF_SLOT;
      constexpr uint32_t loA = Cfg::A_PLANE >> 4, loB = Cfg::B_PLANE >> 4;
      uint32_t idesc, stepA, stepB, a1, b1, a2, b2;
      uint64_t dA0, dB0;
      auto set_roles = [&](bool turned) {
        const bool mnA = mn_a(turned), mnB = mn_b(turned);
        idesc = idesc_f32acc(false, 128, BN) | (mnA ? 1u << 15 : 0u) | (mnB ? 1u << 16 : 0u);
        dA0 = mnA ? sdesc_plain(s0, 128, kChbMn) : sdesc_plain(s0, kChbK, 128);
        dB0 = mnB ? sdesc_plain(s0 + 2 * Cfg::A_PLANE, 128, kChbMn)
                  : sdesc_plain(s0 + 2 * Cfg::A_PLANE, Cfg::CHB_BK, 128);
        stepA = (mnA ? 256 : 2 * kChbK) >> 4, stepB = (mnB ? 256 : 2 * Cfg::CHB_BK) >> 4;
        // the packed kernel's products in its order: lo*hi, hi*lo, hi*hi (of A and B)
        a1 = turned ? 0 : loA, b1 = turned ? loB : 0, a2 = turned ? loA : 0, b2 = turned ? 0 : loB;
      };
      set_roles(false);
      uint32_t it = 0, ab = 0, aph = 0;
      int seq = 0;
      bool ok = true, any = false;
      for (int u = blockIdx.x; ok && u < units; u += gridDim.x, ++seq) {
        const bool turned = TURN && u >= plain;
        if (TURN) set_roles(turned);
        for (int pass = 0; ok && pass < 2; ++pass) {
          for (int c0 = 0; ok && c0 < items; c0 += fold) {
            const int c1 = min(c0 + fold, items);
            if (!(ok = mbar_wait(acce(ab), aph ^ 1u, abort_flag, err))) break;
            const uint32_t d = tmem_base + ab * BN;
            for (int c = c0; c < c1; ++c, ++it) {
              const uint32_t s = it % kDirSlots;
              if (!(ok = mbar_wait(full(s), (it / kDirSlots) & 1u, abort_flag, err))) break;
              tc_fence_after();
              uint64_t da = dA0 + s * (Cfg::SLOT >> 4), db = dB0 + s * (Cfg::SLOT >> 4);
#pragma unroll
              for (int kk = 0; kk < kKI / 16; ++kk) {
                umma_bf16(d, da + a1, db + b1, idesc, c > c0 || kk > 0 ? 1u : 0u);
                umma_bf16(d, da + a2, db + b2, idesc, 1u);
                umma_bf16(d, da, db, idesc, 1u);
                da += stepA, db += stepB;
              }
              any = true;
              umma_commit(empty(s));
            }
            if (!ok) break;
            umma_commit(accf(ab));
            if (++ab == NACC) ab = 0, aph ^= 1u;
          }
          if (!ok || pass == 1) break;
          if (!(ok = mbar_wait(vbar(seq % kVerdicts), (seq / kVerdicts) & 1u, abort_flag, err))) break;
          int eA, eB;
          exponents(seq, eA, eB);
          if ((eA | eB) == 0) break;       // the usual case: no second pass
        }
      }
      if (any) {
        umma_commit(drain_bar);
        mbar_wait_drain(drain_bar, 0);
      }
    }
    __syncwarp();
  }
  } else if (warp >= kEpiWarp0) {
    // -------------------------------------------------------------- epilogue
    warpgroup_regs_inc<kRegsEpi>();
    const int q = warp & 3;
    float* const buf = reinterpret_cast<float*>(smem + Cfg::OFF_EPI) + q * 32 * Cfg::EPI_PITCH;
    uint32_t ab = 0, aph = 0;
    int seq = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < units; u += gridDim.x, ++seq) {
      int m0, n0;
      const bool turned = tile(u, m0, n0);
      if (!turned) {
        const int row = m0 + q * 32 + lane;
        if (a.beta != 0.0f && row < a.M) {
          const float* rp = a.C + static_cast<int64_t>(row) * a.ldc + n0;
          const int ncols = min(BN, a.N - n0);
#pragma unroll
          for (int j = 0; j < BN; j += 32)
            if (j < ncols) prefetch_l2(rp + j);
          prefetch_l2(rp + ncols - 1);
        }
      }
      float S[BN];
      int e = 0;
      for (int pass = 0; ok && pass < 2; ++pass) {
        for (int c0 = 0; c0 < items; c0 += fold) {
          const bool waited = mbar_wait(accf(ab), aph, abort_flag, err);
          if (!__all_sync(0xffffffffu, waited)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + ab * BN;
#pragma unroll
          for (int j = 0; j < BN; j += 16) {
            uint32_t x[16];
            tmem_ld_32x32b_x16(taddr + j, x);
            tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float v = __uint_as_float(x[k]);
              S[j + k] = c0 == 0 ? v : S[j + k] + v;
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acce(ab));
          if (++ab == NACC) ab = 0, aph ^= 1u;
        }
        if (!ok || pass == 1) break;
        const bool known = mbar_wait(vbar(seq % kVerdicts), (seq / kVerdicts) & 1u, abort_flag, err);
        if (!__all_sync(0xffffffffu, known)) {
          ok = false;
          break;
        }
        int eA, eB;
        exponents(seq, eA, eB);
        e = eA + eB;
        if ((eA | eB) == 0) break;
      }
      if (!ok) break;
      if (turned) {
        store_turned<BN>(S, a, e, n0, m0 + q * 32 + lane);
        continue;
      }
      EpiView v;
      v.M = a.M, v.N = a.N, v.C = a.C, v.ldc = a.ldc, v.alpha = a.alpha, v.beta = a.beta;
      v.amaxA = v.amaxB = nullptr, v.partial = nullptr, v.split_k = 1, v.amaxA_stride = 0;
      epilogue_store<BN, Cfg::EPI_PITCH>(S, v, e, 0, m0 + q * 32, n0, lane, buf);
    }
  } else {
    // ----------------------------------------------------------------- split
    constexpr int NA = 4, NB = BN / 32;                // eight-value units of a thread
    const int t = threadIdx.x % kSplitThreads;
    const uint32_t g = warp >> 2;                      // group: items g, g + 4, ... of the CTA's run
    Units ua = make_units(mn_a(false), kChbK, t), ub = make_units(mn_b(false), Cfg::CHB_BK, t);
    uint32_t it = 0, st = 0;                           // items written to slots, items staged
    int seq = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < units; u += gridDim.x, ++seq) {
      int m0, n0;
      const bool turned = tile(u, m0, n0);
      if (TURN) ua = make_units(mn_a(turned), kChbK, t), ub = make_units(mn_b(turned), Cfg::CHB_BK, t);
      float sfA = 1.0f, sfB = 1.0f;
      float mA = 0.0f, mB = 0.0f;
      for (int pass = 0; ok && pass < 2; ++pass) {
        for (int c = static_cast<int>((g - it) % kGroups); c < items; c += kGroups) {
          const uint32_t ic = it + c, s = ic % kDirSlots, sc = st + c, sg = sc % kStages;
          float va[NA][8], vb[NB][8];
          if (pass == 0) {
            const bool in = mbar_wait(sfull(sg), (sc / kStages) & 1u, abort_flag, err);
            if (!__all_sync(0xffffffffu, in)) {
              ok = false;
              break;
            }
            read_units<NA>(va, smem + sg * Cfg::ITEM, ua);
            read_units<NB>(vb, smem + sg * Cfg::ITEM + Cfg::ITEM_A, ub);
          } else {
            int tt = turned;   // (opaque: selected here, not held in registers through the loop)
            asm volatile("" : "+r"(tt));
            const bool tu = tt != 0;
            fetch_units<NA>(va, tu ? a.B : a.A, tu ? a.ldb : a.lda, tu ? a.N : a.M, a.K, mn_a(tu), m0, kKI * c, t);
            fetch_units<NB>(vb, tu ? a.A : a.B, tu ? a.lda : a.ldb, tu ? a.M : a.N, a.K, mn_b(tu), n0, kKI * c, t);
          }
          const float uA = max_units<NA>(va), uB = max_units<NB>(vb);
          mA = fmaxf(mA, uA), mB = fmaxf(mB, uB);
          if (pass == 0) {
            // The stage is free once every lane has its values: each lane orders
            // its reads before the next copy into it (another proxy's writes; an
            // arrival right behind the reads let the copy overtake some of them).
            // The fence costs 2 to 3 %.  Given back behind the parts' fence alone,
            // the stage is late for operands that come from HBM: 50176 x 64 x 576
            // 40.7 us against 35.7, 512^3 on cold inputs 16.4 against 14.4 (9.8
            // against 10.4 where L2 holds them).
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(sempty(sg));
          }
          const bool free = mbar_wait(empty(s), ((ic / kDirSlots) & 1u) ^ 1u, abort_flag, err);
          if (!__all_sync(0xffffffffu, free)) {
            ok = false;
            break;
          }
          uint8_t* slot = smem + Cfg::OFF_SLOT + s * Cfg::SLOT;
          write_units<NA>(va, uA, ua, slot, Cfg::A_PLANE, sfA);
          write_units<NB>(vb, uB, ub, slot + 2 * Cfg::A_PLANE, Cfg::B_PLANE, sfB);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(full(s));
        }
        it += items;
        if (pass == 0) st += items;
        if (!ok || pass == 1) break;
        const int vs = seq % kVerdicts;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          mA = fmaxf(mA, __shfl_xor_sync(0xffffffffu, mA, o));
          mB = fmaxf(mB, __shfl_xor_sync(0xffffffffu, mB, o));
        }
        if (lane == 0) {
          atomicMax(&vmax[2 * vs], __float_as_uint(mA));
          atomicMax(&vmax[2 * vs + 1], __float_as_uint(mB));
          // the entry six tiles on (ten back) is read by nobody any more: every role is
          // at most eight tiles behind this one (four slots, four accumulators)
          const int old = (seq + 6) % kVerdicts;
          if (warp == 0) vmax[2 * old] = vmax[2 * old + 1] = 0u;
          mbar_arrive(vbar(vs));
        }
        const bool known = mbar_wait(vbar(vs), (seq / kVerdicts) & 1u, abort_flag, err);
        if (!__all_sync(0xffffffffu, known)) {
          ok = false;
          break;
        }
        int eA, eB;
        exponents(seq, eA, eB);
        if ((eA | eB) == 0) break;
        sfA = pow2f(-eA), sfB = pow2f(-eB);   // once more, scaled
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, Cfg::TMEM_COLS);
  }
}

template <int BN, bool TURN>
cudaError_t direct_variant(bool launch, const CUtensorMap* tmA, const CUtensorMap* tmB, const DirectArgs& a, int grid,
                           cudaStream_t s) {
  using Cfg = DirCfg<BN>;
  static thread_local int configured_device = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (configured_device != dev) {
    e = cudaFuncSetAttribute(tc_direct_kernel<BN, TURN>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM);
    if (e != cudaSuccess) return e;
    configured_device = dev;
  }
  if (!launch) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kDirThreads);
  cfg.dynamicSmemBytes = Cfg::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, tc_direct_kernel<BN, TURN>, *tmA, *tmB, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t direct_dispatch(bool launch, int bn, const CUtensorMap* tmA, const CUtensorMap* tmB, const DirectArgs& a,
                            int grid, cudaStream_t s) {
  if (bn == 32) return direct_variant<32, false>(launch, tmA, tmB, a, grid, s);
  if (bn == 64 && a.turned) return direct_variant<64, true>(launch, tmA, tmB, a, grid, s);
  if (bn == 64) return direct_variant<64, false>(launch, tmA, tmB, a, grid, s);
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t direct_prepare(int bn, bool turned) {
  DirectArgs a{};
  a.turned = turned;
  return direct_dispatch(false, bn, nullptr, nullptr, a, 0, nullptr);
}

// A turned tile covers 64 rows x 128 columns where a plain one covers 128 x 64, so
// where at most 64 rows are left after the whole row tiles, turned ones need half
// as many tiles for them.  They are used where that saves a wave: 1060^3 has 9 x 17
// = 153 plain tiles on 152 SMs, or 8 x 17 + 9 = 145.
DirectGrid direct_grid(int bn, int64_t M, int64_t N, int sms) {
  DirectGrid g{(M + 127) / 128, (N + bn - 1) / bn, 0};
  const int64_t rest = M % 128;
  if (bn == 64 && rest > 0 && rest <= 64) {
    const DirectGrid t{M / 128, g.tiles_n, (N + 127) / 128};
    if ((t.units() + sms - 1) / sms < (g.units() + sms - 1) / sms) return t;
  }
  return g;
}

cudaError_t direct_launch(int bn, const CUtensorMap& tmA, const CUtensorMap& tmB, DirectArgs a, int sms,
                          cudaStream_t s) {
  const DirectGrid g = direct_grid(bn, a.M, a.N, sms);
  a.tiles_m = static_cast<int>(g.tiles_m);
  a.tiles_n = static_cast<int>(g.tiles_n);
  a.turned = static_cast<int>(g.turned);
  return direct_dispatch(true, bn, &tmA, &tmB, a, static_cast<int>(std::min<int64_t>(g.units(), sms)), s);
}

}  // namespace gb
