// Direct convolution from halo tiles in shared memory (odd R x S filter,
// stride 1, same zero padding, NHWC image, C a multiple of 16): the packed
// convolution's default kernel for the two-plane modes (BF16X3, TF32X3).
//
// The im2col kernel (tc_conv_kernel) loads every input value once per filter
// tap, from planes that a pass of their own has written: on the paper's layer
// (32 x 512 x 512 x 16 -> 16, 3 x 3) the split pass moved 1.07 GB (172 us) and
// the main kernel waited on chains of im2col loads (721 us; tensor pipe, L2
// and DRAM all below 30 %).  Here the image is read once, as FP32:
//   * a unit is a block of 16 output rows x 8 T output columns (T MMA tiles of
//     16 rows x 8 columns) times KN output features;
//   * for each group of 16 input channels one TMA tile load brings the unit's
//     halo, (16 + R - 1) x (8 T + S - 1) pixels of FP32 (zero outside the
//     image), into a staging buffer; the split warps write it as hi and lo
//     parts into a slot of 16-byte channel chunks: chunk j of pixel q lies at
//     j CHB + 16 q, the layout of an unswizzled K-major operand whose 8-row
//     groups are image rows;
//   * an MMA tile's A operand for filter tap (r, s) is then the same slot read
//     from (r BW + s) pixels further on: nothing is copied per tap;
//   * the filter comes as 128-byte k-chunks of its packed planes (hi rows, then
//     lo rows, one operand of 2 KN rows): x_hi x [w_hi | w_lo] is ONE MMA of
//     width 2 KN, x_lo x w_hi one of width KN into the second half, so that
//     hi*hi accumulates apart from the two smaller products (between folds at
//     most 44 MMAs of it and 88 of those; the im2col kernel takes 48 of all
//     three into one sum) and A's hi part is read once for two products.
// The filter's K order is (channel group, tap, channel), so that a slot serves
// all its taps before the next group's; the pack permutes the rows.
//
// What bounds it: shared-memory bandwidth.  A unit of 512 pixels of the paper's
// layer (3 x 3, 16 -> 16) reads its A rows for 72 MMAs (2736 cycles at 128
// bytes a cycle, with B), and the halo's arrival, its two passes of the split
// and the staged outputs add about 1500; 108 units a SM.  Measured: paper's
// layer 963 -> 281 us a call (split pass, its rescale pass, filter pack and
// main kernel before; DRAM floor 158), 8 x 256 x 256 x 64 -> 64 202 -> 101 us.
//
// Whole-image exponent: beta == 0 runs unscaled at once while the split warps
// fold max |x|, and a second launch repeats the convolution scaled only when
// that maximum lies outside the unscaled range (it exits at once otherwise; such
// an image takes twice the time: the paper's layer 529 us against 1245 of the
// im2col path, 1 x 224 x 224 x 128 -> 128 83 against 64, where a scan of the
// image first would cost every call 3 us of 48);
// with beta != 0 (C is read, so a second pass could not start over) the
// maximum is taken before, by the preparing launch.
//
// Roles (512 threads): warp 0 loads halos, warps 1 and 3 issue MMAs (warp 3 owns
// tensor memory), warp 2 loads filter chunks; warps 4..11 epilogue (two
// warpgroups, alternating tiles); warps 12..15 split.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "ptx.cuh"
#include "scale.cuh"
#include "split_arith.cuh"
#include "tile_order.cuh"

namespace gb {

namespace {

constexpr int kThreads = 512;
constexpr int kEpiWarp0 = 4, kEpiWarps = 8;
constexpr int kSplitWarp0 = 12, kSplitWarps = 4;
constexpr int kMaxRing = 8;               // most buffers of any ring
constexpr int kBarBytes = 1024;
constexpr int kOutBytes = kEpiWarps * 4096;   // an epilogue warp's output staging
constexpr int kSmemMax = 231424;           // dynamic shared memory (the kernel has a few static bytes too)

// Channel chunks (16 bytes) of a 16-channel group per plane.
constexpr int chunks_of(bool tf32) { return tf32 ? 4 : 2; }

// Bytes between channel chunks of a slot: 128 / chunks modulo 128, so that the
// split warps' 16-byte stores (eight lanes: consecutive chunks, then pixels)
// fall into different banks.
inline int chunk_stride(int px, bool tf32) {
  return (px * 16 + 127) / 128 * 128 + 128 / chunks_of(tf32);
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ float4 ld_shared_v4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

// One 16-byte chunk of hi and of lo parts from its FP32 values (finite: none
// of them is Inf or NaN; the bits are those of split_bf16 / split_tf32).
template <bool TF32>
__device__ __forceinline__ void split_chunk(const float* x, bool finite, uint4& hv, uint4& lv) {
  if constexpr (TF32) {
    (void)finite;
    unsigned h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float a, b;
      split_tf32(x[k], a, b);
      h[k] = __float_as_uint(a), l[k] = __float_as_uint(b);
    }
    hv = make_uint4(h[0], h[1], h[2], h[3]);
    lv = make_uint4(l[0], l[1], l[2], l[3]);
  } else {
    split_chunk_bf16(x, finite, hv, lv);
  }
}

// Position of unit u: output-feature block fastest, then column block, row
// block, image (units running together share halos and rows in L2).
struct UnitPos {
  int n, h0, w0, k0;
};

template <bool TF32, int KN, int T>
__global__ void __launch_bounds__(kThreads, 1)
    conv_halo_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmB,
                     const __grid_constant__ CUtensorMap tmO, const HaloArgs a) {
  constexpr int NJ = chunks_of(TF32);     // 16-byte chunks of a group and plane
  constexpr int KS = NJ / 2;              // k-steps (32 bytes of K) of a group and tap
  constexpr int ACC = T * 2 * KN;         // TMEM columns of one accumulator buffer
  constexpr int NACC = 2;
  constexpr int TMEM_COLS = NACC * ACC < 32 ? 32 : NACC * ACC;
  constexpr int WCHUNK = 2 * KN * 128;    // bytes of one filter chunk (4 k-steps)
  static_assert(TMEM_COLS <= 512 && (TMEM_COLS & (TMEM_COLS - 1)) == 0, "tensor memory");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t sbase = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (sbase - raw);
  // filter ring | output staging | image staging ring | slot ring | barriers
  const uint32_t off_out = a.nw * WCHUNK;
  const uint32_t off_stage = off_out + kOutBytes;
  const uint32_t off_slot = off_stage + a.nstage * a.stage_bytes;
  const uint32_t off_bar = a.off_bar;
  const uint32_t bar0 = sbase + off_bar;
  auto wfull = [&](int i) { return bar0 + 8u * i; };
  auto wempty = [&](int i) { return bar0 + 8u * (kMaxRing + i); };
  auto sfull = [&](int i) { return bar0 + 8u * (2 * kMaxRing + i); };
  auto sempty = [&](int i) { return bar0 + 8u * (3 * kMaxRing + i); };
  auto hfull = [&](int i) { return bar0 + 8u * (4 * kMaxRing + i); };
  auto hempty = [&](int i) { return bar0 + 8u * (5 * kMaxRing + i); };
  auto accf = [&](int i) { return bar0 + 8u * (6 * kMaxRing + i); };
  auto acce = [&](int i) { return bar0 + 8u * (6 * kMaxRing + NACC + i); };
  auto drain_bar = [&](int i) { return bar0 + 8u * (6 * kMaxRing + 2 * NACC + i); };
  auto cbar = [&](int i) { return bar0 + 8u * (6 * kMaxRing + 2 * NACC + 2 + i); };   // two an epilogue warp
  constexpr int NBAR = 6 * kMaxRing + 2 * NACC + 2 + 2 * kEpiWarps;
  static_assert(8 * NBAR + 8 <= kBarBytes, "barrier block");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + off_bar + 8 * NBAR);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* const err = a.err;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (a.pass == kHaloRescale) {
    // launched after the unscaled pass: nothing to do unless the image needs
    // its exponent (uniform over the grid)
    griddep_wait();
    if (block_exponent(*reinterpret_cast<const volatile unsigned*>(a.amaxA)) == 0) {
      griddep_launch_dependents();
      clear_execution_state(a.state, a.state_words);
      return;
    }
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < kMaxRing; ++i) {
      mbar_init(wfull(i), 1);
      mbar_init(wempty(i), 2);       // the two MMA issuers' commits
      mbar_init(sfull(i), 1);
      mbar_init(sempty(i), kSplitWarps);
      mbar_init(hfull(i), kSplitWarps);
      mbar_init(hempty(i), 2);
    }
    for (int i = 0; i < NACC; ++i) {
      mbar_init(accf(i), 2);
      mbar_init(acce(i), kEpiWarps);
    }
    for (int i = 0; i < 2 * kEpiWarps; ++i) mbar_init(cbar(i), 1);
    mbar_init(drain_bar(0), 1);
    mbar_init(drain_bar(1), 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 3) {
    tmem_alloc(smem_u32(tmem_slot), TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // The unscaled pass follows a packing kernel that touches only the filter,
  // and all of whose CTAs have passed their own wait for the stream's earlier
  // work when this launch starts: the image may be loaded and split at once.
  // Everything else waits for that kernel.
  const bool early = a.pass == kHaloFirst && (warp == 0 || warp >= kSplitWarp0);
  if (!early) griddep_wait();
  griddep_launch_dependents();

  const int nunits = a.units;
  auto pos = [&](int u) {
    UnitPos p;
    const int t0 = u / a.nb;
    p.k0 = (u - t0 * a.nb) * KN;
    const int t1 = t0 / a.wb;
    p.w0 = (t0 - t1 * a.wb) * (8 * T);
    p.n = t1 / a.hb;
    p.h0 = (t1 - p.n * a.hb) * 16;
    return p;
  };
  const int G = a.groups;
  const int taps = a.R * a.S;
  const int steps = a.steps;              // k-steps of a unit: G x taps x KS

  if (warp == 0) {
    // ------------------------------------------------------- halo loads
    if (elect_one()) {
      tma_prefetch_desc(&tmX);
      uint32_t st = 0, ph = 0;
      uint32_t used = 0, par = 0;
      bool ok = true;
      for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x) {
        const UnitPos p = pos(u);
        for (int g = 0; g < G; ++g) {
          if (!mbar_wait(sempty(st), ph ^ 1u, abort_flag, err)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(sfull(st), a.load_bytes);
          tma_load_4d(sbase + off_stage + st * a.stage_bytes, &tmX, sfull(st), 16 * g, p.w0 - a.S / 2,
                      p.h0 - a.R / 2, p.n);
          used |= 1u << st;
          par = (par & ~(1u << st)) | (ph << st);
          if (++st == static_cast<uint32_t>(a.nstage)) st = 0, ph ^= 1u;
        }
      }
      if (!ok)
        for (int i = 0; i < a.nstage; ++i)
          if (used & (1u << i)) mbar_wait_drain(sfull(i), (par >> i) & 1u);
    }
  } else if (warp == 2) {
    // ----------------------------------------------------- filter loads
    if (elect_one()) {
      tma_prefetch_desc(&tmB);
      uint32_t st = 0, ph = 0;
      uint32_t used = 0, par = 0;
      bool ok = true;
      for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x) {
        const UnitPos p = pos(u);
        for (int c = 0; c < a.chunks; ++c) {
          if (!mbar_wait(wempty(st), ph ^ 1u, abort_flag, err)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(wfull(st), WCHUNK);
          const uint32_t dst = sbase + st * WCHUNK;
          tma_load_3d(dst, &tmB, wfull(st), c * (TF32 ? 32 : 64), p.k0, 0);
          tma_load_3d(dst + KN * 128, &tmB, wfull(st), c * (TF32 ? 32 : 64), p.k0, 1);
          used |= 1u << st;
          par = (par & ~(1u << st)) | (ph << st);
          if (++st == static_cast<uint32_t>(a.nw)) st = 0, ph ^= 1u;
        }
      }
      if (!ok)
        for (int i = 0; i < a.nw; ++i)
          if (used & (1u << i)) mbar_wait_drain(wfull(i), (par >> i) & 1u);
    }
  } else if (warp == 1 || warp == 3) {
    // ------------------------------------------------------ MMA issuers
    // Two threads, each for every other tile (their accumulators are their
    // own).  A chunk's four k-steps are straight-line code: on one thread a
    // taken branch costs about as much as an MMA of width 32, and a loop with
    // its waits and wraps at every step issued 72 MMAs in 5700 cycles that
    // run in 2900.
    if (elect_one()) {
      constexpr uint32_t idesc2 = idesc_f32acc(TF32, 128, 2 * KN);
      constexpr uint32_t idesc1 = idesc_f32acc(TF32, 128, KN);
      const int is = warp >> 1;
      // descriptors move by adding 16-byte units to their address field
      const uint64_t slot0 = sdesc_plain(sbase + off_slot + is * 128, a.chb, a.bw * 16);
      const uint64_t w0 = sdesc_k_sw128(sbase);
      const uint32_t slot_units = a.slot_bytes >> 4, sub_units = a.chb >> 3, lo_units = (NJ * a.chb) >> 4;
      const uint32_t row_units = a.bw - a.S;   // from a filter row's last column to the next row's first
      const int S = a.S, gsteps = taps * KS;
      uint32_t wst = 0, wph = 0, hst = 0, hph = 0, ab = 0, aph = 0;
      bool ok = true, any = false;
      for (int u = blockIdx.x; u < nunits; u += gridDim.x) {
        if (!(ok = mbar_wait(hfull(hst), hph, abort_flag, err))) break;
        uint64_t da = slot0 + hst * slot_units, da_next = 0;
        int s = 0, sub = 0, tleft = gsteps, block_left = 0;
        uint32_t d0 = 0, acc = 0;
        for (int i = 0; i < steps; i += 4) {
          if (block_left == 0) {                // a new accumulation block (a multiple of 4 steps)
            if (!(ok = mbar_wait(acce(ab), aph ^ 1u, abort_flag, err))) break;
            block_left = a.steps_per_block;
            d0 = tmem_base + ab * ACC + is * 2 * KN;
            acc = 0;
          }
          const int nv = min(4, steps - i);
          const bool group_end = tleft <= nv;   // (a group has at least 9 steps)
          if (group_end && i + tleft < steps) { // this chunk, or the next, goes on in the next group's slot
            const bool wrap = hst + 1 == static_cast<uint32_t>(a.nslot);
            const uint32_t nst = wrap ? 0u : hst + 1;
            if (!(ok = mbar_wait(hfull(nst), wrap ? hph ^ 1u : hph, abort_flag, err))) break;
            da_next = slot0 + nst * slot_units;
          }
          if (!(ok = mbar_wait(wfull(wst), wph, abort_flag, err))) break;
          tc_fence_after();
          const uint64_t db = w0 + wst * (WCHUNK >> 4);
          auto step = [&](int k) {
            const uint64_t dh = KS == 1 ? da : da + sub * sub_units;
#pragma unroll
            for (int t = 0; t < T / 2; ++t) {
              const uint32_t d = d0 + t * 4 * KN;
              if constexpr (TF32) {
                umma_tf32(d, dh + 16 * t, db + 2 * k, idesc2, acc);
                umma_tf32(d + KN, dh + 16 * t + lo_units, db + 2 * k, idesc1, 1u);
              } else {
                umma_bf16(d, dh + 16 * t, db + 2 * k, idesc2, acc);
                umma_bf16(d + KN, dh + 16 * t + lo_units, db + 2 * k, idesc1, 1u);
              }
            }
            acc = 1;
            // the next step's tap (selects, no branches)
            const bool tap_end = KS == 1 || sub == KS - 1;
            sub = tap_end ? 0 : sub + 1;
            s = tap_end ? s + 1 : s;
            da += tap_end ? 1u : 0u;
            const bool row_end = s == S;
            s = row_end ? 0 : s;
            da += row_end ? row_units : 0u;
            const bool end = --tleft == 0;
            tleft = end ? gsteps : tleft;
            da = end ? da_next : da;
          };
          if (nv == 4) {
#pragma unroll
            for (int k = 0; k < 4; ++k) step(k);
          } else {
            for (int k = 0; k < nv; ++k) step(k);
          }
          any = true;
          umma_commit(wempty(wst));
          if (++wst == static_cast<uint32_t>(a.nw)) wst = 0, wph ^= 1u;
          if (group_end) {
            umma_commit(hempty(hst));
            if (++hst == static_cast<uint32_t>(a.nslot)) hst = 0, hph ^= 1u;
          }
          block_left -= nv;
          if (block_left == 0 || i + 4 >= steps) {
            umma_commit(accf(ab));
            if (++ab == NACC) ab = 0, aph ^= 1u;
          }
        }
        if (!ok) break;
      }
      if (any) {
        umma_commit(drain_bar(is));
        mbar_wait_drain(drain_bar(is), 0);
      }
    }
    __syncwarp();
  } else if (warp >= kEpiWarp0 && warp < kEpiWarp0 + kEpiWarps) {
    // --------------------------------------------------------- epilogue
    constexpr int TW = T / 2;             // tiles of a warpgroup
    // Staged outputs: CB columns of the warp's 4 x 8 pixels at a time go
    // through shared memory (swizzled: eight lanes' 16-byte stores in different
    // banks) and out by TMA, so that whole lines are written and the stores
    // take no load/store cycles from the split warps, which share that path
    // (32-byte stores straight from registers: 316 us against 279 on the paper's
    // layer); with beta != 0 the old values come in the same way, ahead of the
    // accumulator.
    constexpr int CB = KN < 32 ? KN : 32;
    constexpr int PIECE = 32 * CB * 4;    // bytes of one staged piece
    constexpr int NBUF = 4096 / PIECE;
    constexpr int NP = TW * KN / CB;      // pieces of a unit
    // The pieces take the buffers in turn, and only those that are stored: the
    // wait for all but the newest NBUF - 1 stores then covers the buffer's own.
    // (Counting skipped pieces too, a unit at the right edge handed the buffer
    // of the newest store to the next unit, unwaited.)
    static_assert(TW == 1 || KN == CB, "the pieces inside the output come first");
    const int ew = warp - kEpiWarp0;
    const int q = warp & 3;
    const int wg = ew >> 2;
    const uint32_t buf0 = sbase + off_out + ew * 4096;
    const int eA = a.pass == kHaloFirst ? 0 : block_exponent(*a.amaxA);
    uint32_t ab = 0, aph = 0, obuf = 0;
    uint32_t cpar = 0, pending = 0;       // per buffer: parity of its next load, a load in flight
    bool ok = true;
    const int nblk = (steps + a.steps_per_block - 1) / a.steps_per_block;
    for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x) {
      const UnitPos p = pos(u);
      const int e = eA + block_exponent(a.amaxB[p.k0 / kScaleBlock]);
      const int hw = p.h0 + q * 4;
      const int ncol = min(KN, a.K - p.k0);
      // piece i: tile i / (KN / CB), columns from CB (i mod KN / CB) on
      auto piece_in = [&](int i) {
        return hw < a.H && p.w0 + (2 * (i / (KN / CB)) + wg) * 8 < a.W && (i % (KN / CB)) * CB < ncol;
      };
      auto load_old = [&](int i) {        // piece i's old values into its buffer
        if (!piece_in(i)) return;
        const uint32_t b = (obuf + i) % NBUF;   // (all pieces before it are inside as well)
        if (lane == 0) {
          bulk_wait_read<0>();            // the buffer's last store has read it
          mbar_arrive_expect_tx(cbar(2 * ew + b), PIECE);
          tma_load_4d(buf0 + b * PIECE, &tmO, cbar(2 * ew + b), p.k0 + (i % (KN / CB)) * CB,
                      p.w0 + (2 * (i / (KN / CB)) + wg) * 8, hw, p.n);
        }
        pending |= 1u << b;
      };
      if (a.staged && a.beta != 0.0f) {
#pragma unroll
        for (int i = 0; i < (NP < NBUF ? NP : NBUF); ++i) load_old(i);
      }
      float S[TW][KN];
      for (int b = 0; b < nblk; ++b) {
        const bool waited = mbar_wait(accf(ab), aph, abort_flag, err);
        if (!__all_sync(0xffffffffu, waited)) {
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int t = 0; t < TW; ++t) {
          const uint32_t taddr =
              tmem_base + (static_cast<uint32_t>(q * 32) << 16) + ab * ACC + (2 * t + wg) * 2 * KN;
#pragma unroll
          for (int j = 0; j < KN; j += 16) {
            uint32_t x[16], y[16];
            tmem_ld_32x32b_x16(taddr + j, x);
            tmem_ld_32x32b_x16(taddr + KN + j, y);
            tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float v = __uint_as_float(x[k]) + __uint_as_float(y[k]);
              S[t][j + k] = b == 0 ? v : S[t][j + k] + v;
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce(ab));
        if (++ab == NACC) ab = 0, aph ^= 1u;
      }
      if (!ok) break;
      // undo the scaling: alpha comes before the power of two, so that a
      // result in range is not lost to an overflow of the unscaled sum
      float alpha = a.alpha;
      if (e != 0) {
#pragma unroll
        for (int t = 0; t < TW; ++t)
#pragma unroll
          for (int k = 0; k < KN; ++k) S[t][k] = scale_pow2(alpha * S[t][k], e);
        alpha = 1.0f;
      }
      if (a.staged) {
        uint32_t stored = 0;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          if (!piece_in(i)) continue;     // (uniform over the warp)
          ++stored;
          const uint32_t b = (obuf + i) % NBUF;
          const uint32_t buf = buf0 + b * PIECE;
          if (a.beta != 0.0f) {
            const bool waited = mbar_wait(cbar(2 * ew + b), (cpar >> b) & 1u, abort_flag, err);
            if (!__all_sync(0xffffffffu, waited)) {
              ok = false;
              break;
            }
            cpar ^= 1u << b;
            pending &= ~(1u << b);
          } else {
            if (lane == 0) bulk_wait_read<NBUF - 1>();
            __syncwarp();
          }
#pragma unroll
          for (int k = 0; k < CB; k += 4) {
            // lane = pixel: tile row q * 4 + lane / 8, column lane % 8
            const uint32_t unit = CB == 16 ? (k / 4) ^ ((lane >> 1) & 3) : (k / 4) ^ (lane & 7);
            const uint32_t at = buf + lane * CB * 4 + unit * 16;
            const float* sv = &S[i / (KN / CB)][(i % (KN / CB)) * CB + k];
            float4 v;
            if (a.beta != 0.0f) {
              const float4 c = ld_shared_v4(at);
              v = make_float4(fmaf(alpha, sv[0], a.beta * c.x), fmaf(alpha, sv[1], a.beta * c.y),
                              fmaf(alpha, sv[2], a.beta * c.z), fmaf(alpha, sv[3], a.beta * c.w));
            } else {
              v = make_float4(alpha * sv[0], alpha * sv[1], alpha * sv[2], alpha * sv[3]);
            }
            st_shared_v4(at, v);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_4d(&tmO, buf, p.k0 + (i % (KN / CB)) * CB, p.w0 + (2 * (i / (KN / CB)) + wg) * 8, hw, p.n);
            bulk_commit();
          }
          if (a.beta != 0.0f && i + NBUF < NP) load_old(i + NBUF);
        }
        obuf = (obuf + stored) % NBUF;
        continue;
      }
      // features not a multiple of 4, or a misaligned output: straight stores,
      // 16 columns' old values read before any is overwritten
      const int h = hw + (lane >> 3);
#pragma unroll
      for (int t = 0; t < TW; ++t) {
        const int w = p.w0 + (2 * t + wg) * 8 + (lane & 7);
        if (h >= a.H || w >= a.W) continue;
        float* o = a.out + ((static_cast<int64_t>(p.n) * a.H + h) * a.W + w) * a.K + p.k0;
#pragma unroll
        for (int j = 0; j < KN; j += 16) {
          if (j >= ncol) break;
          float c[16];
          if (a.beta != 0.0f) {
#pragma unroll
            for (int k = 0; k < 16; ++k) c[k] = j + k < ncol ? o[j + k] : 0.0f;
          }
#pragma unroll
          for (int k = 0; k < 16; ++k)
            if (j + k < ncol) o[j + k] = a.beta != 0.0f ? fmaf(alpha, S[t][j + k], a.beta * c[k]) : alpha * S[t][j + k];
        }
      }
    }
    // every load has landed and every store has read shared memory and is done
    for (uint32_t b = 0; b < NBUF; ++b)
      if (pending & (1u << b)) mbar_wait_drain(cbar(2 * ew + b), (cpar >> b) & 1u);
    if (a.staged && lane == 0) bulk_wait<0>();
  } else if (warp >= kSplitWarp0) {
    // ------------------------------------------------------------ split
    const int ct = threadIdx.x - kSplitWarp0 * 32;
    const float sf = a.pass == kHaloFirst ? 1.0f : pow2f(-block_exponent(*a.amaxA));
    const int n = a.px * NJ;              // 16-byte output chunks of a plane
    const uint32_t lo_off = NJ * a.chb;
    uint32_t st = 0, sph = 0, hs = 0, hph = 0;
    unsigned m = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < nunits; u += gridDim.x) {
      for (int g = 0; g < G; ++g) {
        int w_ok = 1;
        if (lane == 0)
          w_ok = mbar_wait(sfull(st), sph, abort_flag, err) && mbar_wait(hempty(hs), hph ^ 1u, abort_flag, err);
        if (!__shfl_sync(0xffffffffu, w_ok, 0)) {
          ok = false;
          break;
        }
        __syncwarp();   // lane 0's waits order the other lanes' accesses
        const uint8_t* src = smem + off_stage + st * a.stage_bytes;
        uint8_t* dst = smem + off_slot + hs * a.slot_bytes;
        // four output chunks a thread at a time: all reads first (a store to
        // the slot would keep the compiler from moving later reads up)
        constexpr int U = 4, NT = 32 * kSplitWarps;
        constexpr int EL = 16 / NJ;                    // values of a chunk: 8 (bf16) or 4 (tf32)
        // (bf16: a lane's two 16-byte reads in an order that keeps eight
        // lanes in different banks)
        const int sw = TF32 ? 0 : ((lane >> 2) & 1) * 16;
        for (int i0 = ct; i0 < n; i0 += U * NT) {
          float x[U][EL];
          unsigned bm = 0;
#pragma unroll
          for (int k = 0; k < U; ++k) {
            const int i = min(i0 + k * NT, n - 1);     // (past the end: the last chunk again, not stored)
            const uint8_t* p = src + i * (EL * 4);
            const float4 p0 = *reinterpret_cast<const float4*>(p + sw);
            float4 v0 = p0;
            if constexpr (!TF32) {
              const float4 p1 = *reinterpret_cast<const float4*>(p + (sw ^ 16));
              v0 = sw ? p1 : p0;
              const float4 v1 = sw ? p0 : p1;
              x[k][4] = v1.x, x[k][5] = v1.y, x[k][6] = v1.z, x[k][7] = v1.w;
            }
            x[k][0] = v0.x, x[k][1] = v0.y, x[k][2] = v0.z, x[k][3] = v0.w;
          }
#pragma unroll
          for (int k = 0; k < U; ++k)
#pragma unroll
            for (int l = 0; l < EL; ++l) {
              bm = max(bm, abs_bits(x[k][l]));
              x[k][l] *= sf;
            }
          m = max(m, bm);
          const bool finite = bm < 0x7F800000u;        // else hi = x, lo = 0 for Inf and NaN
#pragma unroll
          for (int k = 0; k < U; ++k) {
            const int i = i0 + k * NT;
            if (i >= n) break;
            uint8_t* d = dst + (i & (NJ - 1)) * a.chb + (i / NJ) * 16;
            uint4 hv, lv;
            split_chunk<TF32>(x[k], finite, hv, lv);
            *reinterpret_cast<uint4*>(d) = hv;
            *reinterpret_cast<uint4*>(d + lo_off) = lv;
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(hfull(hs));
          mbar_arrive(sempty(st));
        }
        if (++st == static_cast<uint32_t>(a.nstage)) st = 0, sph ^= 1u;
        if (++hs == static_cast<uint32_t>(a.nslot)) hs = 0, hph ^= 1u;
      }
    }
    if (a.pass == kHaloFirst) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0 && m) atomicMax(a.amaxA, m);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 3) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
  // (the unscaled pass leaves the state to the launch that follows it)
  clear_execution_state(a.state, a.state_words);
}

template <bool TF32, int KN, int T>
cudaError_t halo_variant(bool launch, const HaloArgs* a, int grid, const CUtensorMap* tmX, const CUtensorMap* tmB,
                         const CUtensorMap* tmO, cudaStream_t s) {
  static thread_local int configured_device = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (configured_device != dev) {
    e = cudaFuncSetAttribute(conv_halo_kernel<TF32, KN, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return e;
    configured_device = dev;
  }
  if (!launch) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = static_cast<size_t>(a->off_bar) + kBarBytes + 1024;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, conv_halo_kernel<TF32, KN, T>, *tmX, *tmB, *tmO, *a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <bool TF32>
cudaError_t halo_dispatch(bool launch, const HaloArgs& a, int grid, const CUtensorMap* tmX,
                          const CUtensorMap* tmB, const CUtensorMap* tmO, cudaStream_t s) {
  if (a.kn == 16 && a.tiles == 4) return halo_variant<TF32, 16, 4>(launch, &a, grid, tmX, tmB, tmO, s);
  if (a.kn == 16 && a.tiles == 2) return halo_variant<TF32, 16, 2>(launch, &a, grid, tmX, tmB, tmO, s);
  if (a.kn == 32 && a.tiles == 4) return halo_variant<TF32, 32, 4>(launch, &a, grid, tmX, tmB, tmO, s);
  if (a.kn == 32 && a.tiles == 2) return halo_variant<TF32, 32, 2>(launch, &a, grid, tmX, tmB, tmO, s);
  if (a.kn == 64 && a.tiles == 2) return halo_variant<TF32, 64, 2>(launch, &a, grid, tmX, tmB, tmO, s);
  return cudaErrorInvalidValue;
}

}  // namespace

// Longest chain of k-steps one accumulator takes before it is folded into
// FP32 registers (the tensor core's FP32 sum does not round to nearest).  The
// im2col kernel folds every 16 k-steps of three products, 48 MMAs into one
// accumulator; here hi*hi has an accumulator of its own, one MMA a k-step, and
// the two small products share the other, two a k-step.  With 48 k-steps a fold
// the TF32X3 errors were a little above the im2col kernel's (128 -> 64 features,
// 3 x 3, 144 k-steps: 9.27e-7 against 9.10e-7); with 44 they are below it on every
// shape tried (7.04e-7 there, 8.4e-7 against 9.0e-7 at 64 -> 64, 7 x 7), in BF16X3
// 3.80e-6 against 3.85e-6.  The one more fold costs 0.3 to 0.9 % there and nothing
// elsewhere; 40 would cost 1 % at 9 x 9.
constexpr int kHaloFold = 44;

// Whether the halo kernel is the faster one: its estimate against that of the im2col
// kernel with tiles of 128 x bn, ctas of them at a time on a SM.  Both in
// microseconds: a constant, and waves of units (tiles) at what a group of 16 channels
// of one takes: here the split of its halo's pixels and its MMAs (taps x tiles), there
// loads and MMAs of its taps.  Fitted to 1152 shapes (9 to 500 pixels a side, 1 to 200
// images, 16 to 128 channels and 16 to 192 features, 3 x 3 to 11 x 11, both betas; rms
// 4 to 8 %).  Blocks that are mostly padding, or a last wave that the im2col tiles do
// not need, make it the slower one.  The im2col kernel then folds twice as often as by
// default, for errors no larger than this one's, which costs it up to 8 %: hence the
// margin.  64 images of 17 x 17 x 64 -> 64, 11 x 11: 140 -> 89 us; 16 of 56 x 56 x 128 ->
// 128, 3 x 3 in TF32X3: 122 -> 106; the 58 shapes sent away 1.20 times as fast on average,
// none slower.
bool halo_pays(Prec prec, const HaloArgs& a, int64_t batch, int bn, int ctas, int sms) {
  struct Cost {
    double fixed, tap;   // halo: per 1000 pixels, per tap and tile; im2col: per group, per tap
  };
  static constexpr Cost kHalo[2][3] = {{{0.60, 0.046}, {0.96, 0.050}, {1.04, 0.060}},     // 16, 32, 64 features a unit
                                       {{1.39, 0.100}, {3.42, 0.096}, {4.59, 0.109}}};
  static constexpr Cost kIm2col[2][3] = {{{0.22, 0.219}, {0.17, 0.140}, {0.64, 0.150}},   // tiles 32, 64, 128 wide
                                         {{0.73, 0.377}, {0.42, 0.307}, {0.93, 0.313}}};
  const int tf32 = prec == Prec::TF32, taps = a.R * a.S;
  const Cost h = kHalo[tf32][a.kn == 16 ? 0 : a.kn == 32 ? 1 : 2], i = kIm2col[tf32][bn == 32 ? 0 : bn == 64 ? 1 : 2];
  const int64_t slots = static_cast<int64_t>(sms) * ctas;
  const int64_t tiles = ((batch * a.H * a.W + 127) / 128) * ((a.K + bn - 1) / bn);
  const double hwaves = static_cast<double>((a.units + sms - 1) / sms);
  const double iwaves = static_cast<double>((tiles + slots - 1) / slots);
  const double halo = 16.0 + hwaves * a.groups * (h.fixed * a.px / 1000.0 + h.tap * taps * a.tiles);
  const double im2col = 22.0 + (iwaves - 0.2) * a.groups * (i.fixed + i.tap * taps);
  return halo <= (tf32 ? 1.08 : 1.11) * im2col;
}

bool halo_geometry(Prec prec, int64_t batch, int64_t H, int64_t W, int64_t C, int64_t K, int R, int S,
                   HaloArgs* out) {
  // (a filter chunk of four k-steps meets at most one group's end with nine taps or more)
  if ((prec != Prec::BF16 && prec != Prec::TF32) || C % 16 != 0 || R * S < 9) return false;
  const bool tf32 = prec == Prec::TF32;
  HaloArgs a{};
  a.H = static_cast<int>(H), a.W = static_cast<int>(W), a.K = static_cast<int>(K);
  a.R = R, a.S = S;
  a.groups = static_cast<int>(C / 16);
  a.kn = K <= 16 ? 16 : K <= 32 ? 32 : 64;
  a.steps = a.groups * R * S * (chunks_of(tf32) / 2);
  a.chunks = (a.steps + 3) / 4;
  const int nblk = (a.steps + kHaloFold - 1) / kHaloFold;
  a.steps_per_block = ((a.steps + nblk - 1) / nblk + 3) / 4 * 4;   // whole filter chunks
  const int wchunk = 2 * a.kn * 128;
  // as many tiles a unit (less halo per output) as leave room for two buffers
  // of each ring, then more buffers: staging first (bytes in flight).  The
  // widest filters on two tiles may leave room for one staging buffer only
  // (their groups multiply for ten times as long as they load).
  const int room = kSmemMax - 1024 - kBarBytes;
  auto bytes = [&] { return a.nw * wchunk + kOutBytes + a.nstage * a.stage_bytes + a.nslot * a.slot_bytes; };
  for (a.tiles = a.kn == 64 ? 2 : 4; a.tiles >= 2; a.tiles /= 2) {
    a.bw = 8 * a.tiles + S - 1;
    a.px = a.bw * (16 + R - 1);
    a.load_bytes = a.px * 64;
    a.stage_bytes = (a.load_bytes + 127) / 128 * 128;
    a.chb = chunk_stride(a.px, tf32);
    a.slot_bytes = 2 * chunks_of(tf32) * a.chb;
    a.nstage = 2, a.nslot = 2, a.nw = std::min(4, std::max(2, a.chunks));
    if (bytes() > room && a.tiles == 2) a.nstage = 1, a.nw = 2;
    if (bytes() > room) continue;
    for (int* n : {&a.nstage, &a.nslot, &a.nstage})
      if (++*n, bytes() > room) --*n;
    a.off_bar = (bytes() + 127) / 128 * 128;
    if (a.off_bar > room) continue;
    a.hb = static_cast<int>((H + 15) / 16);
    a.wb = static_cast<int>((W + 8 * a.tiles - 1) / (8 * a.tiles));
    a.nb = static_cast<int>((K + a.kn - 1) / a.kn);
    // Above 64 features the halo is split again for each block of 64: then
    // the blocks must not be mostly padding (128 -> 128 features, 3 x 3,
    // against the im2col kernel: 16 images of 50 x 50, blocks 61 % full,
    // 0.95-0.97x; 2 of 130 x 260 at 5 x 5, 86 % full, 1.03x; 1 of 224 x 224,
    // 1.21x.  Of 140 shapes, 28 to 260 pixels a side, 16 to 256 channels, 3 x 3
    // to 11 x 11, that first one alone was slower by more than 1 %.)
    if (a.nb > 1 && 10 * H * W < 7 * (16LL * a.hb) * (8LL * a.tiles * a.wb)) return false;
    const int64_t units = batch * a.hb * a.wb * a.nb;
    if (units > INT32_MAX) return false;
    a.units = static_cast<int>(units);
    *out = a;
    return true;
  }
  return false;
}

cudaError_t halo_prepare(Prec prec, const HaloArgs& a) {
  return prec == Prec::TF32 ? halo_dispatch<true>(false, a, 0, nullptr, nullptr, nullptr, nullptr)
                            : halo_dispatch<false>(false, a, 0, nullptr, nullptr, nullptr, nullptr);
}

cudaError_t halo_launch(Prec prec, const HaloArgs& a, int grid, const CUtensorMap& tmX, const CUtensorMap& tmB,
                        const CUtensorMap& tmO, cudaStream_t s) {
  return prec == Prec::TF32 ? halo_dispatch<true>(true, a, grid, &tmX, &tmB, &tmO, s)
                            : halo_dispatch<false>(true, a, grid, &tmX, &tmB, &tmO, s);
}

}  // namespace gb
