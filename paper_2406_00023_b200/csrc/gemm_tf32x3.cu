// Grouped GEMMs of the fp32 expert FFN on the 5th-generation tensor cores.  Operands and results are fp32;
// every operand value v is split into hi = v rounded to tf32 and lo = (v - hi) rounded to tf32, and a product
// is taken as hi*hi + (hi*lo + lo*hi): the products are exact in fp32, what is dropped is lo*lo (below 2^-22
// of a product) and the rounding of lo (2^-23).
//
// The tensor core's fp32 accumulator drops the bits that do not fit instead of rounding them, an error that
// always points towards zero and would add up over a long contraction.  So a chain of MMAs is never longer
// than one K block (32 values: four MMAs): hi*hi and the cross terms of such a chain go to accumulators of
// their own in tensor memory, and the epilogue warps add each chain to running sums in registers with rounded
// fp32 additions while the next one is multiplied.  Even so a contraction of positive products comes out 1.2e-7 short,
// where fp32 FMAs are off by 1.2e-7 at 64 values and 4.3e-7 at 1024 (products of either sign: 1.4e-7 against 1.4e-7 to
// 5.7e-7), and in a layer of short contractions these add up with what the scores are short by (weight gradients of
// T 512, d 256, h 512: 8.0e-7, with the CUDA-core GEMMs 7.0e-7).  Contractions over at most 384 columns or 256 rows
// therefore end a chain after two MMAs: 0.6e-7 short, that layer 7.1e-7, 158 -> 161 us.  (For all of them that would be
// 651 -> 739 us at T 1531, d 768, h 1000; four MMAs are already below the FMAs there.  Chains of eight: 2.0e-7.)
//
// One persistent kernel serves the six contractions (the three weight gradients in one launch).  Roles in a CTA of 640 threads:
//   warp 0       TMA: a K block arrives as plain fp32 in the place of its hi tiles
//   warp 1       issues the MMAs (kind::tf32, 128 x 2 BN and 128 x BN, 8 values of K each)
//   warps 4-11   split a block into hi (in place) and lo, both K-major with the 128-byte swizzle, in two groups of
//                four warps that take alternate blocks, so that the load latency and the fence of one block pass
//                under the arithmetic of the other.  An operand whose contraction index is not contiguous in
//                memory is turned on the way (4 x 4 blocks in registers).
//   warps 12-19  add the chunks' accumulators, then SwiGLU / its derivative / plain stores
// Registers are split unevenly (setmaxnreg): the epilogue holds 64 running sums per thread.
// What bounds it is shared memory: 12 KiB and 8 KiB of operands per pair of MMAs, 32 KiB in by TMA, 32 KiB read and
// 64 KiB written by the split, about 1600 cycles of its port per K block at BN = 128, of about 1850 that a block
// takes (the MMAs alone: 940).  An fp32 step of T 1531, d 768, h 1000, 12 experts: 2.8 ms with the CUDA-core kernels,
// 0.65 ms with these.
// A tile is 128 x BN, BN = 128, or 64 where 128 would leave SMs without a tile.  All waits are bounded; on
// expiry the kernel leaves 0x7c0a in etr_stats.error_word, frees its tensor memory and returns.
#include <algorithm>

#include "common.cuh"
#include "tcgen05_ptx.cuh"

namespace etr {

constexpr int F3_BM = 128;
constexpr int F3_BK = 32;                        // floats per K block: one 128-byte swizzle row
template <int BN> struct F3Ring { static constexpr int STAGES = BN == 128 ? 3 : 4; };      // 192 KiB either way
constexpr int F3_THREADS = 640;
// registers per thread by role; 640 threads are launched with 96 each (61440), the split takes 60416
constexpr int F3_REGS_LAUNCH = 96, F3_REGS_IO = 40, F3_REGS_CONV = 88, F3_REGS_EPI = 128;
static_assert(128 * F3_REGS_IO + 256 * F3_REGS_CONV + 256 * F3_REGS_EPI <= F3_THREADS * F3_REGS_LAUNCH, "register split");
// Contractions of at most so many values end a chain of MMAs after 16 values instead of 32.
constexpr int F3_SHORT_WIDTH = 384, F3_SHORT_ROWS = 256;
constexpr int F3_SCRATCH = 32 * 80;              // per epilogue warp: 32 rows of 64 bytes, 16 bytes of pad each

// F3_WGRAD: the three weight gradients in one launch (plain stores; M = d and N = h of the first, exchanged for the others).
enum { F3_STORE = 0, F3_SWIGLU = 1, F3_DSWIGLU = 2, F3_WGRAD = 3 };

struct F3Params {
  int two_k;               // the first half of the K blocks from (A0, B0), the rest from (A1, B1); both ranges are K long
  int M, N, K, E;          // per-expert extents
  int dyn_m;               // rows are the expert's (M = C_stride bounds them); otherwise K is the expert's row count
  const int32_t* counts;
  float* out0; float* out1; float* out2;
  const float* in0; const float* in1;
  long long out_bs;
  int ld_out;
  etr_stats* stats;
  long long wait_limit;
};

struct F3Tile { int e, m0, n0, K, kblocks, m_lim, N, which; };      // which: the gradient, 0 where there is one output

__device__ __forceinline__ void f3_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void f3_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// v -> (hi, lo), both tf32 values (round to nearest, on the integer image: a cvt per value costs twice the time),
// hi + lo = v up to 2^-23 |v|; the tensor core does not read the low 13 bits of lo.  Values that rounding would carry past
// the largest finite one are cut; an infinity or NaN is hi (lo then holds nothing of use).  minus_zero is -0.0 in a register
// that the compiler knows nothing about: the addition leaves every number as it is and makes any NaN the canonical one
// (a payload in the bits that are cut would leave an infinity; a test and an OR instead took 5 % of a layer).
__device__ __forceinline__ void f3_split(float v, float minus_zero, float& hi, float& lo) {
  v += minus_zero;
  uint32_t u = __float_as_uint(v);
  if (fabsf(v) < __uint_as_float(0x7f7ff000u)) u += 0x1000u;
  hi = __uint_as_float(u & 0xffffe000u);
  lo = __uint_as_float(__float_as_uint(v - hi) + 0x1000u);
}
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 f3_pair(uint32_t x, uint32_t y) { return (f32x2)y << 32 | x; }
__device__ __forceinline__ f32x2 f3_add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 f3_zero_times(f32x2 a, f32x2 c) {      // 0 * a + c: c, or NaN where a is infinite or NaN
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(0ull), "l"(c));
  return d;
}
// x, or the largest finite value of its sign where x is infinite or NaN.
__device__ __forceinline__ uint32_t f3_finite(uint32_t x) {
  float d;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(d) : "f"(__uint_as_float(x)), "f"(3.402823466e38f));
  return __float_as_uint(d);
}
// sum[i] += hh[i] + xx[i].  Where an operand is infinite the cross terms hold inf * 0 or inf - inf; hi*hi alone then has the
// value that fp32 products would give, an infinity or NaN, which no finite number added to it changes.  Chains of four MMAs:
// one test for the sixteen columns.  Of two, where the epilogue is the longest stage: no test, whose latency counts twice
// as often, but every cross term made finite (fp32 step of T 1531: 880 us with the test, 739 without).
template <int CHAIN>
__device__ __forceinline__ void f3_add16(f32x2* sum, const uint32_t* hh, const uint32_t* xx) {
  bool all_finite = false;
  if (CHAIN == 4) {
    f32x2 odd[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      odd[i] = f3_zero_times(f3_pair(xx[4 * i], xx[4 * i + 1]), f3_zero_times(f3_pair(xx[4 * i + 2], xx[4 * i + 3]), 0ull));
    const f32x2 o2 = f3_add2(f3_add2(odd[0], odd[1]), f3_add2(odd[2], odd[3]));
    const float o = __uint_as_float((uint32_t)o2) + __uint_as_float((uint32_t)(o2 >> 32));
    all_finite = o == o;
  }
  if (CHAIN == 4 && all_finite) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      sum[i] = f3_add2(sum[i], f3_add2(f3_pair(hh[2 * i], hh[2 * i + 1]), f3_pair(xx[2 * i], xx[2 * i + 1])));
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      sum[i] = f3_add2(sum[i], f3_add2(f3_pair(hh[2 * i], hh[2 * i + 1]), f3_pair(f3_finite(xx[2 * i]), f3_finite(xx[2 * i + 1]))));
  }
}

__device__ __forceinline__ int f3_mtiles(const F3Params& p, int n_e) {
  return p.dyn_m ? (min((n_e + 127) & ~127, p.M) + F3_BM - 1) / F3_BM : (p.M + F3_BM - 1) / F3_BM;
}
// Tiles of an expert.
template <int EPI>
__device__ __forceinline__ int f3_tiles(const F3Params& p, int n_e, int cols) {
  if (EPI != F3_WGRAD) return f3_mtiles(p, n_e) * ((p.N + cols - 1) / cols);
  return (p.M + F3_BM - 1) / F3_BM * ((p.N + cols - 1) / cols) + 2 * ((p.N + F3_BM - 1) / F3_BM) * ((p.M + cols - 1) / cols);
}
template <int EPI>
__device__ __forceinline__ bool f3_tile(const F3Params& p, const int* prefix, const int* counts, int tile, int& e_cur,
                                        int cols, F3Tile& t) {
  if (tile >= prefix[p.E]) return false;
  while (tile >= prefix[e_cur + 1]) ++e_cur;
  int local = tile - prefix[e_cur], mt;
  const int n_e = counts[e_cur];
  t.e = e_cur;
  t.which = 0;
  t.N = p.N;
  if (EPI == F3_WGRAD) {
    const int first = (p.M + F3_BM - 1) / F3_BM * ((p.N + cols - 1) / cols);
    const int other = (p.N + F3_BM - 1) / F3_BM * ((p.M + cols - 1) / cols);
    if (local >= first) {
      local -= first;
      t.which = local < other ? 1 : 2;
      if (local >= other) local -= other;
      t.N = p.M;
    }
    t.m_lim = t.which ? p.N : p.M;
    mt = (t.m_lim + F3_BM - 1) / F3_BM;
  } else {
    mt = f3_mtiles(p, n_e);
    t.m_lim = p.dyn_m ? min((n_e + 127) & ~127, p.M) : p.M;
  }
  t.m0 = (local % mt) * F3_BM;
  t.n0 = (local / mt) * cols;
  t.K = p.dyn_m ? p.K : n_e;
  t.kblocks = (t.K + F3_BK - 1) / F3_BK * (p.two_k ? 2 : 1);
  return true;
}

// One box (32 operand rows x 32 values of K, 4 KiB) split by one warp, raw values in `hi`.  K-major: a lane takes
// 16-byte pieces lane, lane + 32, ... in memory order, rewritten where they were.  MN-major: the raw box is 32 rows
// of K x 32 operand rows, the same 4 KiB; a lane takes operand rows 4 q .. 4 q + 3 at four consecutive k, twice,
// and turns the 4 x 4 blocks.  16-byte chunk c of row r lies at r * 128 + ((c ^ r % 8) * 16); the eight lanes of a
// shared-memory phase write eight different chunks (and read four, twice).
// klim: rows of K that exist in this block (MN-major; what lies behind them is not an operand value).
template <bool MN>
__device__ __forceinline__ void f3_split_box(uint8_t* hi, uint8_t* lo, int klim, int lane) {
  float mz;
  asm volatile("mov.b32 %0, 0x80000000;" : "=f"(mz));
  float4 v[8];
  const int q = (lane >> 3) * 2 + ((lane >> 2) & 1), c0 = lane & 3;          // MN: quad of rows, chunk of K of the first block
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if (!MN) {
      v[j] = *reinterpret_cast<const float4*>(hi + 16 * (lane + 32 * j));
    } else {
      const int k = 4 * (c0 + (j & 4)) + (j & 3);
      v[j] = k < klim ? *reinterpret_cast<const float4*>(hi + k * 128 + ((q ^ (k & 7)) << 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  if (MN) __syncwarp();                                                      // the whole box has been read
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    int off;
    float4 x;
    if (!MN) {
      off = 16 * (lane + 32 * j);
      x = v[j];
    } else {
      const int r = 4 * q + (j & 3);
      off = r * 128 + (((c0 + (j & 4)) ^ (r & 7)) << 4);
      const float4* b = v + (j & 4);
      auto at = [&](const float4& y) { return (j & 3) == 0 ? y.x : (j & 3) == 1 ? y.y : (j & 3) == 2 ? y.z : y.w; };
      x = make_float4(at(b[0]), at(b[1]), at(b[2]), at(b[3]));
    }
    float4 h, l;
    f3_split(x.x, mz, h.x, l.x); f3_split(x.y, mz, h.y, l.y); f3_split(x.z, mz, h.z, l.z); f3_split(x.w, mz, h.w, l.w);
    *reinterpret_cast<float4*>(hi + off) = h;
    *reinterpret_cast<float4*>(lo + off) = l;
  }
}

// The TMA boxes of one operand tile of ROWS rows: one box of 32 values of K x ROWS (K-major), or a box of 32 rows of
// K x 32 operand rows for every 32 of them (MN-major).
template <bool MN, int ROWS>
__device__ __forceinline__ void f3_fetch(uint32_t dst, const CUtensorMap* map, uint32_t bar, int row0, int k0, int e) {
  if (!MN) {
    tma_load_3d(dst, map, bar, k0, row0, e);
  } else {
#pragma unroll
    for (int j = 0; j < ROWS; j += 32) tma_load_3d(dst + j * 128, map, bar, row0 + j, k0, e);
  }
}

// A 32-row x 16-column block (lane = row) stored through the warp's scratch: 64 contiguous bytes of a row per
// four lanes.  ncols: columns that exist (a multiple of 4, may exceed 16).
__device__ __forceinline__ void f3_store16(uint8_t* scratch, int lane, int nvalid, int ncols, float* dst, int ld,
                                           const float* v) {
  float4* mine = reinterpret_cast<float4*>(scratch + lane * 80);
#pragma unroll
  for (int q = 0; q < 4; ++q) mine[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  __syncwarp();
  const int sub = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = (lane >> 2) + 8 * i;
    const float4 w = *reinterpret_cast<const float4*>(scratch + row * 80 + sub * 16);
    if (row < nvalid && 4 * sub < ncols) *reinterpret_cast<float4*>(dst + (long long)row * ld + 4 * sub) = w;
  }
  __syncwarp();
}

template <int EPI, bool A_MN, bool B_MN, int BN, int CHAIN>
__global__ void __launch_bounds__(F3_THREADS, 1)
tf32x3_gemm_kernel(const __grid_constant__ CUtensorMap mapA0, const __grid_constant__ CUtensorMap mapA1,
                   const __grid_constant__ CUtensorMap mapB0, const __grid_constant__ CUtensorMap mapB1,
                   const __grid_constant__ CUtensorMap mapA2, const F3Params p, uint32_t idesc) {
  constexpr int F3_STAGES = F3Ring<BN>::STAGES;
  constexpr int COLS = EPI == F3_SWIGLU ? BN / 2 : BN;               // output columns of a tile
  constexpr uint32_t A_BYTES = F3_BM * 128, B_BYTES = BN * 128;      // one of hi, lo
  constexpr uint32_t STAGE = 2 * A_BYTES + 2 * B_BYTES;
  constexpr int F3_ACC = 256 / BN;                                   // accumulator stages of hi*hi and cross terms
  constexpr uint32_t TMEM_COLS = F3_ACC * 2 * BN;
  constexpr int GW = BN / 4;                                         // columns of a thread's two groups

  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[3 * F3_STAGES + 2 * F3_ACC];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag_s;
  __shared__ int tile_prefix[257];
  __shared__ int s_counts[256];

  volatile int* abort_flag = &abort_flag_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint8_t* tiles = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t tiles_base = smem_u32(tiles);
  const uint32_t full_bar = smem_u32(&bars[0]);                      // [STAGES] the TMA boxes have landed
  const uint32_t conv_bar = smem_u32(&bars[F3_STAGES]);              // [STAGES] both operands are split
  const uint32_t empty_bar = smem_u32(&bars[2 * F3_STAGES]);         // [STAGES] the MMAs have read the stage
  const uint32_t tfull_bar = smem_u32(&bars[3 * F3_STAGES]);         // [ACC] a chain's accumulators are complete
  const uint32_t tempty_bar = smem_u32(&bars[3 * F3_STAGES + F3_ACC]);      // [ACC] they have been read

  if (tid == 0) {
    abort_flag_s = 0;
    for (int s = 0; s < F3_STAGES; ++s) {
      mbar_init(full_bar + 8 * s, 1); mbar_init(conv_bar + 8 * s, 4); mbar_init(empty_bar + 8 * s, 1);
    }
    for (int a = 0; a < F3_ACC; ++a) { mbar_init(tfull_bar + 8 * a, 1); mbar_init(tempty_bar + 8 * a, 8); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  grid_wait();
  if (warp == 2) {
    tile_prefix_warp(tile_prefix, s_counts, p.counts, p.E, lane, [&](int n_e) { return f3_tiles<EPI>(p, n_e, COLS); });
  }
  tc_fence_before();
  __syncthreads();
  grid_release();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(F3_REGS_IO));
    if (warp == 0) {
      // ---- TMA producer --------------------------------------------------------------------------------------
      constexpr int B_ROWS = EPI == F3_SWIGLU ? BN / 2 : BN;         // SwiGLU: half of the tile's rows from each weight
      int e_cur = 0, stage = 0;
      uint32_t phase = 0;
      F3Tile t;
      bool ok = true;
      for (int tile = blockIdx.x; ok && f3_tile<EPI>(p, tile_prefix, s_counts, tile, e_cur, COLS, t); tile += gridDim.x) {
        const int kb1 = p.two_k ? t.kblocks / 2 : t.kblocks;
        for (int kb = 0; kb < t.kblocks; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait(empty_bar + 8 * stage, phase ^ 1u, abort_flag, p.wait_limit));
          if (!ok) break;
          if (elect_one()) {
            const bool second = kb >= kb1;
            const int k0 = (second ? kb - kb1 : kb) * F3_BK;
            const uint32_t sa = tiles_base + stage * STAGE, sb = sa + 2 * A_BYTES, bar = full_bar + 8 * stage;
            mbar_expect_tx(bar, A_BYTES + B_BYTES);
            const bool alt = EPI == F3_WGRAD ? t.which != 0 : second;
            f3_fetch<A_MN, F3_BM>(sa, EPI == F3_WGRAD && t.which == 2 ? &mapA2 : alt ? &mapA1 : &mapA0, bar, t.m0, k0, t.e);
            f3_fetch<B_MN, B_ROWS>(sb, alt ? &mapB1 : &mapB0, bar, t.n0, k0, t.e);
            if (EPI == F3_SWIGLU) f3_fetch<B_MN, B_ROWS>(sb + B_BYTES / 2, &mapB1, bar, t.n0, k0, t.e);
          }
          __syncwarp();
          if (++stage == F3_STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    } else if (warp == 1) {
      // ---- MMA issuer ----------------------------------------------------------------------------------------
      const uint32_t idesc_wide = (idesc & ~(0x3fu << 17)) | ((uint32_t)(2 * BN >> 3) << 17);
      int e_cur = 0, stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      F3Tile t;
      bool ok = true;
      for (int tile = blockIdx.x; ok && f3_tile<EPI>(p, tile_prefix, s_counts, tile, e_cur, COLS, t); tile += gridDim.x) {
        for (int kb = 0; kb < t.kblocks; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait(conv_bar + 8 * stage, phase, abort_flag, p.wait_limit));
          const uint32_t a_hi = tiles_base + stage * STAGE, a_lo = a_hi + A_BYTES, b_hi = a_hi + 2 * A_BYTES;
#pragma unroll
          for (int k0 = 0; k0 < F3_BK / 8; k0 += CHAIN) {
            ok = ok && __all_sync(0xffffffffu, mbar_wait(tempty_bar + 8 * acc, acc_phase ^ 1u, abort_flag, p.wait_limit));
            if (!ok) break;
            tc_fence_after();
            if (elect_one()) {
              const uint32_t d_tmem = tmem_base + (uint32_t)(acc * 2 * BN);
              // hi and lo of B lie one behind the other: A_hi x [B_hi; B_lo]^T is one MMA of 2 BN columns (hi*hi in the
              // first BN, hi*lo in the others), and A_lo x B_hi^T adds lo*hi to the latter
#pragma unroll
              for (int kk = k0; kk < k0 + CHAIN; ++kk)
                f3_mma(d_tmem, make_smem_desc(a_hi + 32 * kk, 16u, 1024u), make_smem_desc(b_hi + 32 * kk, 16u, 1024u),
                       idesc_wide, kk > k0 ? 1u : 0u);
#pragma unroll
              for (int kk = k0; kk < k0 + CHAIN; ++kk)
                f3_mma(d_tmem + BN, make_smem_desc(a_lo + 32 * kk, 16u, 1024u), make_smem_desc(b_hi + 32 * kk, 16u, 1024u),
                       idesc, 1u);
              if (k0 + CHAIN == F3_BK / 8) tc_commit(empty_bar + 8 * stage);
              tc_commit(tfull_bar + 8 * acc);
            }
            __syncwarp();
            if (++acc == F3_ACC) { acc = 0; acc_phase ^= 1u; }
          }
          if (!ok) break;
          if (++stage == F3_STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp < 12) {
    // ---- converter warps: group g takes blocks g, g + 2, ... of the CTA's sequence ----------------------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(F3_REGS_CONV));
    const int group = (warp - 4) >> 2;
    int e_cur = 0, stage = 0, turn = 0;
    uint32_t phase = 0;
    F3Tile t;
    bool ok = true;
    for (int tile = blockIdx.x; ok && f3_tile<EPI>(p, tile_prefix, s_counts, tile, e_cur, COLS, t); tile += gridDim.x) {
      for (int kb = 0; kb < t.kblocks; ++kb) {
        if (turn == group) {
          // With an odd number of stages the use of this stage before this one is the other group's, and the parity of a
          // barrier tells its last two uses apart only: were that block still on its way (behind the one after it), the
          // wait for this one would pass on the parity of the use before.  So that use has to be split first.
          if (F3_STAGES % 2 != 0)
            ok = __all_sync(0xffffffffu, mbar_wait(conv_bar + 8 * stage, phase ^ 1u, abort_flag, p.wait_limit));
          ok = ok && __all_sync(0xffffffffu, mbar_wait(full_bar + 8 * stage, phase, abort_flag, p.wait_limit));
          if (!ok) break;
          uint8_t* st = tiles + (size_t)stage * STAGE;
          uint8_t* sb = st + 2 * A_BYTES;
          // rows of K behind the contraction's end: TMA has filled those outside the tensor with zeros, but an
          // expert's row count ends inside its buffer
          const int klim = p.dyn_m ? F3_BK : t.K - kb * F3_BK;
          const int w = (warp - 4) & 3;
          f3_split_box<A_MN>(st + 4096 * w, st + A_BYTES + 4096 * w, klim, lane);
          if (BN == 128 || w >= 2) {
            const int o = 4096 * (BN == 128 ? w : w - 2);
            f3_split_box<B_MN>(sb + o, sb + B_BYTES + o, klim, lane);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // generic writes -> the MMA's reads
          __syncwarp();
          if (lane == 0) mbar_arrive(conv_bar + 8 * stage);
        }
        turn ^= 1;
        if (++stage == F3_STAGES) { stage = 0; phase ^= 1u; }
      }
    }
  } else {
    // ---- epilogue warps: running sums of 2 GW columns of one row per thread -----------------------------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(F3_REGS_EPI));
    const int q = warp & 3, half = (warp - 12) >> 2;
    uint8_t* scratch = tiles + (size_t)F3_STAGES * STAGE + (warp - 12) * F3_SCRATCH;
    const int g0 = EPI == F3_SWIGLU ? half * GW : half * 2 * GW;     // first columns of the two groups in the tile
    const int g1 = EPI == F3_SWIGLU ? BN / 2 + half * GW : g0 + GW;
    int e_cur = 0, acc = 0;
    uint32_t acc_phase = 0;
    F3Tile t;
    bool ok = true;
    for (int tile = blockIdx.x; ok && f3_tile<EPI>(p, tile_prefix, s_counts, tile, e_cur, COLS, t); tile += gridDim.x) {
      f32x2 run[GW];                                                 // 2 GW running sums
#pragma unroll
      for (int i = 0; i < GW; ++i) run[i] = 0ull;
      // first column in the tile of the j-th sixteen sums
      auto col = [&](int j) { return (uint32_t)(16 * j < GW ? g0 + 16 * j : g1 + 16 * j - GW); };
      for (int chain = 0; chain < t.kblocks * (F3_BK / 8 / CHAIN); ++chain) {
        ok = __all_sync(0xffffffffu, mbar_wait(tfull_bar + 8 * acc, acc_phase, abort_flag, p.wait_limit));
        if (!ok) break;
        tc_fence_after();
        const uint32_t taddr = tmem_base + (uint32_t)(acc * 2 * BN) + ((uint32_t)(32 * q) << 16);
#pragma unroll
        for (int j = 0; j < GW / 8; ++j) {
          uint32_t hh[16], xx[16];
          f3_ld16(taddr + col(j), hh);
          f3_ld16(taddr + BN + col(j), xx);
          tc_wait_ld();
          f3_add16<CHAIN>(run + 8 * j, hh, xx);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty_bar + 8 * acc);
        if (++acc == F3_ACC) { acc = 0; acc_phase ^= 1u; }
      }
      if (!ok) break;
      const int row0 = t.m0 + 32 * q, nvalid = min(32, t.m_lim - row0);
      const int ld_out = EPI == F3_WGRAD ? t.N : p.ld_out;
      float* const out = EPI == F3_WGRAD && t.which ? (t.which == 1 ? p.out1 : p.out2) : p.out0;
      const long long wb = (long long)t.e * p.out_bs + (long long)row0 * ld_out;
      float sum[2][GW];
#pragma unroll
      for (int i = 0; i < GW; ++i) {
        sum[i / (GW / 2)][2 * i % GW] = __uint_as_float((uint32_t)run[i]);
        sum[i / (GW / 2)][2 * i % GW + 1] = __uint_as_float((uint32_t)(run[i] >> 32));
      }
      __syncwarp();
      if (EPI == F3_SWIGLU) {
#pragma unroll
        for (int c = 0; c < GW; c += 16) {
          const int n = t.n0 + g0 + c;
          if (n >= p.N) break;
          float hv[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float g = sum[0][c + i];
            hv[i] = g / (1.0f + expf(-g)) * sum[1][c + i];
          }
          f3_store16(scratch, lane, nvalid, p.N - n, p.out0 + wb + n, p.ld_out, &sum[0][c]);
          f3_store16(scratch, lane, nvalid, p.N - n, p.out1 + wb + n, p.ld_out, &sum[1][c]);
          f3_store16(scratch, lane, nvalid, p.N - n, p.out2 + wb + n, p.ld_out, hv);
        }
      } else {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
#pragma unroll
          for (int c = 0; c < GW; c += 16) {
            const int n = t.n0 + (g ? g1 : g0) + c;
            if (n >= t.N) break;
            if (EPI == F3_DSWIGLU) {
              float du[16];
              const float4* G = reinterpret_cast<const float4*>(p.in0 + wb + (long long)lane * p.ld_out + n);
              const float4* U = reinterpret_cast<const float4*>(p.in1 + wb + (long long)lane * p.ld_out + n);
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                float4 gq = make_float4(0.f, 0.f, 0.f, 0.f), uq = gq;
                if (lane < nvalid && n + 4 * v < p.N) { gq = G[v]; uq = U[v]; }
                const float gg[4] = {gq.x, gq.y, gq.z, gq.w}, uu[4] = {uq.x, uq.y, uq.z, uq.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const float dh = sum[g][c + 4 * v + i], s = 1.0f / (1.0f + expf(-gg[i]));
                  sum[g][c + 4 * v + i] = dh * uu[i] * s * (1.0f + gg[i] * (1.0f - s));
                  du[4 * v + i] = dh * gg[i] * s;
                }
              }
              f3_store16(scratch, lane, nvalid, p.N - n, p.out1 + wb + n, p.ld_out, du);
            }
            f3_store16(scratch, lane, nvalid, t.N - n, out + wb + n, ld_out, &sum[g][c]);
          }
        }
      }
    }
  }

  // ---- teardown ---------------------------------------------------------------------------------------
  __syncwarp();
  if (*abort_flag) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }      // copies and MMAs still in flight end before the memory is released
    if (tid == 0 && p.stats != nullptr) atomicExch(&p.stats->error_word, 0x7c0a);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// Row-major fp32 tensor [E, rows, cols] as a 3-D map (cols, rows, E), boxes of 32 columns x box_rows, 128-byte swizzle.
static etr_status f3_map(CUtensorMap* m, const void* base, int cols, int rows, int E, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return ETR_ERR_CUDA;
  const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)E};
  const cuuint64_t strides[2] = {(cuuint64_t)cols * 4, (cuuint64_t)cols * 4 * (cuuint64_t)rows};
  const cuuint32_t box[3] = {(cuuint32_t)F3_BK, (cuuint32_t)box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? ETR_OK : ETR_ERR_CUDA;
}

// A row-major [E, rows, cols] operand.  K-major: the columns are the contraction; MN-major: the rows are.
struct F3Operand { const void* ptr; int cols, rows; };

template <int EPI, bool A_MN, bool B_MN, int BN, int CHAIN>
static etr_status f3_launch_bn(const char* name, const F3Operand* A, const F3Operand* B, const F3Params& p,
                               int max_tiles, cudaStream_t st) {
  constexpr size_t smem = (size_t)F3Ring<BN>::STAGES * (2 * F3_BM + 2 * BN) * 128 + 1024 + 8 * F3_SCRATCH;
  auto k = tf32x3_gemm_kernel<EPI, A_MN, B_MN, BN, CHAIN>;
  static std::atomic<unsigned long long> attr_done{0};      // one bit per device
  if (!ensure_dyn_smem(k, smem, attr_done)) return ETR_ERR_CUDA;
  uint32_t idesc = 0;
  idesc |= 1u << 4;                        // accumulator fp32
  idesc |= 2u << 7;                        // A tf32
  idesc |= 2u << 10;                       // B tf32, both K-major in shared memory
  idesc |= (uint32_t)(BN >> 3) << 17;
  idesc |= (uint32_t)(F3_BM >> 4) << 24;
  CUtensorMap a[2], b[2];
  for (int i = 0; i < 2; ++i) {
    const F3Operand &oa = A[i].ptr ? A[i] : A[0], &ob = B[i].ptr ? B[i] : B[0];
    ETR_TRY(f3_map(&a[i], oa.ptr, oa.cols, oa.rows, p.E, A_MN ? F3_BK : F3_BM));
    ETR_TRY(f3_map(&b[i], ob.ptr, ob.cols, ob.rows, p.E, B_MN ? F3_BK : (EPI == F3_SWIGLU ? BN / 2 : BN)));
  }
  CUtensorMap a2 = a[0];
  if (EPI == F3_WGRAD) ETR_TRY(f3_map(&a2, A[2].ptr, A[2].cols, A[2].rows, p.E, F3_BK));
  ETR_TIME_BEGIN(name);
  launch_kernel(k, std::max(1, std::min(max_tiles, current_sm_count())), F3_THREADS, smem, st, 1, a[0], a[1], b[0], b[1], a2, p, idesc);
  ETR_LAUNCH_CHECK();
  return ETR_OK;
}
// k_max: the longest contraction that the launch can hold.
template <int EPI, bool A_MN, bool B_MN>
static etr_status f3_launch(const char* name, const F3Operand* A, const F3Operand* B, const F3Params& p,
                            int tiles_m, int k_max, cudaStream_t st) {
  // 128-column tiles unless they leave SMs without one
  constexpr int C128 = EPI == F3_SWIGLU ? 64 : 128, C64 = C128 / 2;
  int t128 = tiles_m * ceil_div(p.N, C128), t64 = tiles_m * ceil_div(p.N, C64);
  if (EPI == F3_WGRAD) {
    t128 += 2 * p.E * ceil_div(p.N, F3_BM) * ceil_div(p.M, C128);
    t64 += 2 * p.E * ceil_div(p.N, F3_BM) * ceil_div(p.M, C64);
  }
  const bool wide = t128 >= current_sm_count();
  if (k_max <= (p.dyn_m ? F3_SHORT_WIDTH : F3_SHORT_ROWS))
    return wide ? f3_launch_bn<EPI, A_MN, B_MN, 128, 2>(name, A, B, p, t128, st)
                : f3_launch_bn<EPI, A_MN, B_MN, 64, 2>(name, A, B, p, t64, st);
  return wide ? f3_launch_bn<EPI, A_MN, B_MN, 128, 4>(name, A, B, p, t128, st)
              : f3_launch_bn<EPI, A_MN, B_MN, 64, 4>(name, A, B, p, t64, st);
}

static F3Params f3_params(const etr_config* c, const etr_route* rt, etr_stats* stats) {
  F3Params p = {};
  p.E = c->E; p.counts = rt->counts; p.stats = stats;
  p.wait_limit = c->wait_limit_cycles > 0 ? (long long)c->wait_limit_cycles : ETR_WAIT_LIMIT_CYCLES;
  return p;
}

etr_status tf32x3_ffn_forward(const etr_config* c, const etr_route* rt, const void* Xp, const void* W1g,
                              const void* W1u, const void* W2, void* G, void* U, void* H, void* O,
                              etr_stats* stats, cudaStream_t st) {
  const int d = c->d, h = c->h, Cs = c_stride_of(c), mt = c->E * (Cs / F3_BM);
  const long long ldx = (long long)Cs * d, lhx = (long long)Cs * h;
  {  // G, U, H = SwiGLU(Xp W1g^T, Xp W1u^T)
    F3Params p = f3_params(c, rt, stats);
    const F3Operand A[2] = {{Xp, d, Cs}, {}}, B[2] = {{W1g, d, h}, {W1u, d, h}};
    p.M = Cs; p.N = h; p.K = d; p.dyn_m = 1;
    p.out0 = (float*)G; p.out1 = (float*)U; p.out2 = (float*)H; p.out_bs = lhx; p.ld_out = h;
    ETR_TRY((f3_launch<F3_SWIGLU, false, false>("tf32x3_gemm_swiglu", A, B, p, mt, d, st)));
  }
  F3Params p = f3_params(c, rt, stats);      // O = H W2^T
  const F3Operand A[2] = {{H, h, Cs}, {}}, B[2] = {{W2, h, d}, {}};
  p.M = Cs; p.N = d; p.K = h; p.dyn_m = 1; p.out0 = (float*)O; p.out_bs = ldx; p.ld_out = d;
  return f3_launch<F3_STORE, false, false>("tf32x3_gemm_down", A, B, p, mt, h, st);
}

etr_status tf32x3_ffn_backward(const etr_config* c, const etr_route* rt, const void* dO, const void* Xp,
                               const void* G, const void* U, const void* H, const void* W1g, const void* W1u,
                               const void* W2, void* dG, void* dU, void* dXp, void* dW1g, void* dW1u, void* dW2,
                               etr_stats* stats, cudaStream_t st) {
  const int d = c->d, h = c->h, Cs = c_stride_of(c), E = c->E, mt = E * (Cs / F3_BM);
  const long long ldx = (long long)Cs * d, lhx = (long long)Cs * h, w = (long long)h * d;
  {  // dH = dO W2, then dG, dU
    F3Params p = f3_params(c, rt, stats);
    const F3Operand A[2] = {{dO, d, Cs}, {}}, B[2] = {{W2, h, d}, {}};
    p.M = Cs; p.N = h; p.K = d; p.dyn_m = 1;
    p.out0 = (float*)dG; p.out1 = (float*)dU; p.in0 = (const float*)G; p.in1 = (const float*)U;
    p.out_bs = lhx; p.ld_out = h;
    ETR_TRY((f3_launch<F3_DSWIGLU, false, true>("tf32x3_gemm_dswiglu", A, B, p, mt, d, st)));
  }
  {  // dXp = dG W1g + dU W1u
    F3Params p = f3_params(c, rt, stats);
    const F3Operand A[2] = {{dG, h, Cs}, {dU, h, Cs}}, B[2] = {{W1g, d, h}, {W1u, d, h}};
    p.two_k = 1; p.M = Cs; p.N = d; p.K = h; p.dyn_m = 1; p.out0 = (float*)dXp; p.out_bs = ldx; p.ld_out = d;
    ETR_TRY((f3_launch<F3_STORE, false, true>("tf32x3_gemm_dxp", A, B, p, mt, 2 * h, st)));
  }
  // dW2 = dO^T H, dW1g = dG^T Xp, dW1u = dU^T Xp over the expert's rows, one launch: a launch each left its last (at 512 tokens
  // its only) round of tiles part-filled and paid the head and the tail of a tile's chain three times.  30 -> 21 us at T 512, d 256,
  // h 512, E 8; 152 -> 128 at T 1531, d 768, h 1000, E 12 (tiles of 64 columns up to two rounds of 128: the same).
  F3Params p = f3_params(c, rt, stats);
  const F3Operand A[3] = {{dO, d, Cs}, {dG, h, Cs}, {dU, h, Cs}}, B[2] = {{H, h, Cs}, {Xp, d, Cs}};
  p.M = d; p.N = h; p.out0 = (float*)dW2; p.out1 = (float*)dW1g; p.out2 = (float*)dW1u; p.out_bs = w;
  return f3_launch<F3_WGRAD, true, true>("tf32x3_gemm_dw", A, B, p, E * ceil_div(d, F3_BM), c->capacity, st);
}

}  // namespace etr
