// Grouped GEMMs of the expert FFN on the 5th-generation tensor cores (bf16 in, fp32
// accumulate in tensor memory).  One persistent, warp-specialised design serves all six
// contractions of the forward and backward pass, in four tile forms (and one more kernel):
//
//   tc_grouped_gemm_kernel            one CTA per 128 x 256 tile (cta_group::1), 4-stage ring
//   tc_grouped_gemm_pair_kernel       a cluster of two CTAs per 256 x 256 tile (cta_group::2),
//                                     6-stage ring, two accumulator stages
//   tc_grouped_gemm_pair_wide_kernel  a cluster of two CTAs per 256 x 512 tile: two accumulators
//                                     share the A operand, 4-stage ring, halves released separately
//   tc_grouped_gemm_swap_kernel       the pair form with the operands exchanged: 256 rows of the weights are M, up
//                                     to 256 tokens (a multiple of 16) are N (contractions over d or h)
//   tc_wgrad_pair_kernel              the pair form's weight gradients, all three in one launch
//
//   warp 0      TMA producer: 64x64-element boxes (128-byte swizzle) into the ring
//   warp 1      allocates tensor memory, issues tcgen05.mma (the pair's leader CTA only)
//   warps 2-9   epilogue: tcgen05.ld of the fp32 accumulator, fused SwiGLU / its derivative,
//               bf16 stores (two warps per 32-lane quarter of tensor memory, half of the
//               columns each); it overlaps the next tile's MMAs
//
// Every operand is fetched as 64x64 boxes of its row-major tensor, so one tensor map per
// tensor serves both uses of it: "K-major" (the contraction index is contiguous in memory)
// and "MN-major" (the output index is contiguous: weight-gradient GEMMs, which contract over
// rows, and the data-gradient GEMMs, which read the weights transposed).  Only the
// shared-memory matrix descriptor differs.
//
// Tiles never straddle experts: the per-expert row count is read from `counts` on the
// device, and tiles are dealt round-robin to the CTAs of a persistent grid.  All waits on
// mbarriers are bounded; on expiry the kernel records a code in etr_stats.error_word,
// stops issuing work, releases its tensor memory and returns.
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "tcgen05_ptx.cuh"

namespace etr {

constexpr int TC_BM = 128;
constexpr int TC_BK = 64;
constexpr int TC_STAGES = 4;
constexpr int TC_THREADS = 320;        // TMA warp, MMA warp, 8 epilogue warps
constexpr uint32_t TC_BOX_BYTES = 64 * 64 * 2;
constexpr long long TC_WAIT_LIMIT_CYCLES = ETR_WAIT_LIMIT_CYCLES;

enum { TC_EPI_STORE = 0, TC_EPI_SWIGLU = 1, TC_EPI_DSWIGLU = 2, TC_EPI_DSWIGLU_BOX = 3 };      // the last: pair form only
enum { TC_DYN_M = 1, TC_DYN_K = 2 };

struct TcParams {
  int a_mn, b_mn;        // 1: operand is MN-major in memory
  int dual_b;            // SwiGLU: accumulator columns [0,128) from B0, [128,256) from B1
  int k1_blocks;         // > 0: K blocks [0,k1) use (A0,B0), the rest (A1,B1)
  int M, N, K;           // per-expert extents (DYN_M: M = C_stride cap; DYN_K: K unused)
  int dyn, E;
  const int32_t* counts;
  __nv_bfloat16* out0; __nv_bfloat16* out1; __nv_bfloat16* out2;
  const __nv_bfloat16* in0; const __nv_bfloat16* in1;
  long long out_bs;      // elements between experts in the outputs (and in0/in1)
  int ld_out;
  uint32_t idesc;
  etr_stats* stats;
  // Row gather (token rearrangement fused into the operand fetch): the rows of one operand are
  // rows of the token matrix X named by slot_token, fetched four at a time by TMA gather.
  // gather 1: the A operand's rows (row r of expert e is token slot_token[e*gather_ld + r]);
  // gather 2: the B operand's K rows (contractions over the expert's rows).  Slots holding -1 fetch
  // row gather_oob, which lies outside X and reads as zeros.  The gathered operand's map is mapA0
  // (gather 1) or mapB0 (gather 2), a 2-D map of X with a one-row box.
  int gather;
  int gather_ld, gather_oob;
  const int32_t* gather_idx;
  // Combine folded into the plain-store epilogue (Top-1 token choice: a token has at most one row, so
  // its output is that row times its gate and needs no sum): besides out0, row r of expert e also goes,
  // scaled, to row sc_tok[e*M + r] of sc_out (skipped where the slot holds -1).  sc_out == nullptr: off.
  const int32_t* sc_tok; const float* sc_gate; __nv_bfloat16* sc_out; int sc_ld;
  long long wait_limit;  // bound of every mbarrier wait, in SM clock cycles
  int out_f32;           // plain-store epilogue: out0 is fp32 (weight gradients with grad_fp32)
};

// ---- PTX wrappers (mbarrier helpers and the bounded wait: common.cuh) ---------------------------
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ void load32(const __nv_bfloat16* src, float* v) {
  const uint4* p = reinterpret_cast<const uint4*>(src);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint4 w = p[q];
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[8 * q + 2 * i] = __uint_as_float(u[i] << 16);
      v[8 * q + 2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
    }
  }
}

// last_kk: 16-wide MMA steps of the last K block that hold rows in use (contractions over an expert's
// rows: the steps beyond multiply pad rows, which are zero, and are skipped)
struct TileCoord { int e, m0, n0, kblocks, m_lim, last_kk; };

// Warp-cooperative store of a 32-row x 32-column bf16 block whose row `lane` is held by lane
// `lane` as 32 floats.  Written directly, every store instruction would touch 32 rows with 16
// bytes each (half a sector per row).  Instead the block is turned in a per-warp shared-memory
// scratch (32 rows x 80 bytes: the 16-byte pad makes both phases bank-conflict free) so that an
// instruction writes 8 rows x 64 contiguous bytes: whole sectors, half as many of them.
constexpr int TC_SCRATCH_ROW_BYTES = 80;
constexpr int TC_SCRATCH_BYTES = 32 * TC_SCRATCH_ROW_BYTES;      // per epilogue warp
__device__ __forceinline__ void store32_warp(uint8_t* scratch, int lane, int nvalid, __nv_bfloat16* dst,
                                             int ld_out, const float* v) {
  uint4* mine = reinterpret_cast<uint4*>(scratch + lane * TC_SCRATCH_ROW_BYTES);
#pragma unroll
  for (int q = 0; q < 4; ++q)
    mine[q] = make_uint4(pack_bf16(v[8 * q], v[8 * q + 1]), pack_bf16(v[8 * q + 2], v[8 * q + 3]),
                         pack_bf16(v[8 * q + 4], v[8 * q + 5]), pack_bf16(v[8 * q + 6], v[8 * q + 7]));
  __syncwarp();
  const int sub = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = (lane >> 2) + 8 * i;
    const uint4 w = *reinterpret_cast<const uint4*>(scratch + row * TC_SCRATCH_ROW_BYTES + sub * 16);
    if (row < nvalid) *reinterpret_cast<uint4*>(dst + (long long)row * ld_out + sub * 8) = w;
  }
  __syncwarp();
}

// The same turn for 16 raw 32-bit words per lane (64 bytes of a row): a 32 x 32 block already packed
// to bf16, or half of a 32 x 32 block of fp32.  dst is the first row's address, rows ld_bytes apart.
__device__ __forceinline__ void store_rows64(uint8_t* scratch, int lane, int nvalid, char* dst,
                                             long long ld_bytes, const uint32_t* w16) {
  uint4* mine = reinterpret_cast<uint4*>(scratch + lane * TC_SCRATCH_ROW_BYTES);
#pragma unroll
  for (int q = 0; q < 4; ++q) mine[q] = make_uint4(w16[4 * q], w16[4 * q + 1], w16[4 * q + 2], w16[4 * q + 3]);
  __syncwarp();
  const int sub = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = (lane >> 2) + 8 * i;
    const uint4 w = *reinterpret_cast<const uint4*>(scratch + row * TC_SCRATCH_ROW_BYTES + sub * 16);
    if (row < nvalid) *reinterpret_cast<uint4*>(dst + row * ld_bytes + sub * 16) = w;
  }
  __syncwarp();
}
__device__ __forceinline__ void store32_warp_packed(uint8_t* scratch, int lane, int nvalid, __nv_bfloat16* dst,
                                                    int ld_out, const uint32_t* w16) {
  store_rows64(scratch, lane, nvalid, reinterpret_cast<char*>(dst), 2ll * ld_out, w16);
}
// A 32 x 32 block of fp32 accumulators (lane = row, 32 raw words) stored as fp32: two 64-byte halves.
__device__ __forceinline__ void store32_warp_f32(uint8_t* scratch, int lane, int nvalid, float* dst, int ld_out,
                                                 const uint32_t* r32) {
  store_rows64(scratch, lane, nvalid, reinterpret_cast<char*>(dst), 4ll * ld_out, r32);
  store_rows64(scratch, lane, nvalid, reinterpret_cast<char*>(dst) + 64, 4ll * ld_out, r32 + 16);
}
// The combine of a Top-1 layer in the epilogue: the 32 x 32 block just stored (packed bf16, w16 of this
// lane's row) scaled by the row's gate and written to the row of the token the slot holds.  The value
// is formed exactly as the separate kernels would: the stored bf16 output widened, times the gate in
// fp32, rounded to bf16.  Rows turn through the scratch like any store; the token of a row comes from
// the lane that owns it.
__device__ __forceinline__ void scatter32_warp(uint8_t* scratch, int lane, int tok, float gate,
                                               __nv_bfloat16* out, int ld, int col, const uint32_t* w16) {
  uint4* mine = reinterpret_cast<uint4*>(scratch + lane * TC_SCRATCH_ROW_BYTES);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t w = w16[4 * q + i];
      y[i] = pack_bf16(gate * __uint_as_float(w << 16), gate * __uint_as_float(w & 0xffff0000u));
    }
    mine[q] = make_uint4(y[0], y[1], y[2], y[3]);
  }
  __syncwarp();
  const int sub = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = (lane >> 2) + 8 * i;
    const int t = __shfl_sync(0xffffffffu, tok, row);
    const uint4 w = *reinterpret_cast<const uint4*>(scratch + row * TC_SCRATCH_ROW_BYTES + sub * 16);
    if (t >= 0) *reinterpret_cast<uint4*>(out + (long long)t * ld + col + sub * 8) = w;
  }
  __syncwarp();
}
// Zeros to a 32-row x 32-column block of the output (nothing to contract): wbase is the element offset of its first
// row and column.  Like any store, 8 rows of 64 bytes per instruction.
__device__ __forceinline__ void store_zero_block(const TcParams& p, long long wbase, int lane, int nvalid) {
  const uint4 z = make_uint4(0, 0, 0, 0);
  const int sub = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = (lane >> 2) + 8 * i;
    if (row >= nvalid) continue;
    const long long o = wbase + (long long)row * p.ld_out;
    if (p.out_f32) {
      float* q = reinterpret_cast<float*>(p.out0) + o + sub * 4;
      *reinterpret_cast<uint4*>(q) = z;
      *reinterpret_cast<uint4*>(q + 16) = z;
    } else {
      *reinterpret_cast<uint4*>(p.out0 + o + sub * 8) = z;
    }
  }
}

// The reverse turn for the saved activations the SwiGLU derivative reads: fetched as 8 rows x
// 64 contiguous bytes per instruction (regs `t`), later handed to the lane that owns the row.
__device__ __forceinline__ void load32_warp_issue(const __nv_bfloat16* src, int ld, int lane, int nvalid,
                                                  uint4 (&t)[4]) {
  const int sub = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = (lane >> 2) + 8 * i;
    t[i] = row < nvalid ? *reinterpret_cast<const uint4*>(src + (long long)row * ld + sub * 8)
                        : make_uint4(0, 0, 0, 0);
  }
}
__device__ __forceinline__ void load32_warp_turn(uint8_t* scratch, int lane, const uint4 (&t)[4],
                                                 uint4 (&mine)[4]) {
  const int sub = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    *reinterpret_cast<uint4*>(scratch + ((lane >> 2) + 8 * i) * TC_SCRATCH_ROW_BYTES + sub * 16) = t[i];
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 4; ++q)
    mine[q] = *reinterpret_cast<const uint4*>(scratch + lane * TC_SCRATCH_ROW_BYTES + q * 16);
  __syncwarp();
}

// dG and dU of two adjacent elements, in the place of the bf16 pairs of G and U.
__device__ __forceinline__ void dswiglu_pair(float dh0, float dh1, uint32_t& gw, uint32_t& uw) {
  const float dh[2] = {dh0, dh1};
  const float g[2] = {__uint_as_float(gw << 16), __uint_as_float(gw & 0xffff0000u)};
  const float u[2] = {__uint_as_float(uw << 16), __uint_as_float(uw & 0xffff0000u)};
  float dg[2], du[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float sgm = __fdividef(1.0f, 1.0f + __expf(-g[k]));
    dg[k] = dh[k] * u[k] * sgm * (1.0f + g[k] * (1.0f - sgm));
    du[k] = dh[k] * g[k] * sgm;
  }
  gw = pack_bf16(dg[0], dg[1]);
  uw = pack_bf16(du[0], du[1]);
}

// The epilogue of one accumulator tile for one warp: `nch` chunks of 32 columns starting at
// chunk c_beg, read from tensor memory at taddr and stored (or fused with SwiGLU / its
// derivative) at row offset obase.  pg/pu hold the prefetched G and U of the first chunk.
template <int EPI, int BN>
__device__ __forceinline__ void epilogue_chunks(const TcParams& p, int n0, uint32_t taddr, long long obase,
                                                bool row_ok, int c_beg, int nch, uint4 (&pg)[4],
                                                uint4 (&pu)[4], uint8_t* scratch, int lane, int nvalid,
                                                int sc_t = -1, float sc_g = 0.f) {
  const long long wbase = obase - (long long)lane * p.ld_out;     // row 0 of this warp's 32 rows
#pragma unroll 1
  for (int c = c_beg; c < c_beg + nch; ++c) {
    if (n0 + 32 * c >= p.N) break;
    __syncwarp();               // tcgen05.ld is warp-collective: reconverge after masked stores
    uint32_t r0[32];
    float v[32];
    tc_ld32(taddr + 32 * c, r0);
    if (EPI == TC_EPI_SWIGLU) {
      uint32_t r1[32];
      tc_ld32(taddr + BN / 2 + 32 * c, r1);
      tc_wait_ld();
      float hv[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float g = __uint_as_float(r0[i]), u = __uint_as_float(r1[i]);
        hv[i] = __fdividef(g, 1.0f + __expf(-g)) * u;
        v[i] = g;
      }
      store32_warp(scratch, lane, nvalid, p.out0 + wbase + 32 * c, p.ld_out, v);
      store32_warp(scratch, lane, nvalid, p.out2 + wbase + 32 * c, p.ld_out, hv);
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r1[i]);
      store32_warp(scratch, lane, nvalid, p.out1 + wbase + 32 * c, p.ld_out, v);
    } else if (EPI == TC_EPI_DSWIGLU) {
      uint4 cg[4], cu[4];
      load32_warp_turn(scratch, lane, pg, cg);
      load32_warp_turn(scratch, lane, pu, cu);
      if (c + 1 < c_beg + nch && n0 + 32 * (c + 1) < p.N) {
        load32_warp_issue(p.in0 + wbase + 32 * (c + 1), p.ld_out, lane, nvalid, pg);
        load32_warp_issue(p.in1 + wbase + 32 * (c + 1), p.ld_out, lane, nvalid, pu);
      }
      tc_wait_ld();
      {
        float dg[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const uint32_t wg = reinterpret_cast<const uint32_t*>(cg)[i >> 1];
          const uint32_t wu = reinterpret_cast<const uint32_t*>(cu)[i >> 1];
          const float g = (i & 1) ? __uint_as_float(wg & 0xffff0000u) : __uint_as_float(wg << 16);
          const float u = (i & 1) ? __uint_as_float(wu & 0xffff0000u) : __uint_as_float(wu << 16);
          const float dh = __uint_as_float(r0[i]);
          const float sgm = __fdividef(1.0f, 1.0f + __expf(-g));
          dg[i] = dh * u * sgm * (1.0f + g * (1.0f - sgm));
          v[i] = dh * g * sgm;
        }
        store32_warp(scratch, lane, nvalid, p.out0 + wbase + 32 * c, p.ld_out, dg);
        store32_warp(scratch, lane, nvalid, p.out1 + wbase + 32 * c, p.ld_out, v);
      }
    } else {
      tc_wait_ld();
      if (p.out_f32) {
        store32_warp_f32(scratch, lane, nvalid, reinterpret_cast<float*>(p.out0) + wbase + 32 * c, p.ld_out, r0);
      } else if (p.sc_out == nullptr) {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r0[i]);
        store32_warp(scratch, lane, nvalid, p.out0 + wbase + 32 * c, p.ld_out, v);
      } else {
        uint32_t pk[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) pk[i] = pack_bf16(__uint_as_float(r0[2 * i]), __uint_as_float(r0[2 * i + 1]));
        store32_warp_packed(scratch, lane, nvalid, p.out0 + wbase + 32 * c, p.ld_out, pk);
        scatter32_warp(scratch, lane, sc_t, sc_g, p.sc_out, p.sc_ld, n0 + 32 * c, pk);
      }
    }
  }
}



// Tile index -> coordinates.  tile_prefix[e] = first tile of expert e.
__device__ __forceinline__ bool tile_coord(const TcParams& p, const int* tile_prefix, const int* counts_s,
    int tile, int& e_cur,
                                           int n_tile_cols, TileCoord& tc) {
  if (tile >= tile_prefix[p.E]) return false;
  while (tile >= tile_prefix[e_cur + 1]) ++e_cur;
  const int local = tile - tile_prefix[e_cur];
  const int n_e = counts_s[e_cur];
  int mt_count;
  if (p.dyn == TC_DYN_M) {
    mt_count = (min(n_e, p.M) + TC_BM - 1) / TC_BM;
    tc.kblocks = (p.K + TC_BK - 1) / TC_BK;
    tc.last_kk = TC_BK / 16;
    tc.m_lim = mt_count * TC_BM;
  } else {
    mt_count = (p.M + TC_BM - 1) / TC_BM;
    tc.kblocks = (n_e + TC_BK - 1) / TC_BK;
    tc.last_kk = n_e > 0 ? ((n_e - 1) % TC_BK) / 16 + 1 : TC_BK / 16;
    tc.m_lim = p.M;
  }
  tc.e = e_cur;
  tc.m0 = (local % mt_count) * TC_BM;
  tc.n0 = (local / mt_count) * n_tile_cols;
  (void)n_tile_cols;
  return true;
}

template <int BN, int EPI>
__global__ void __launch_bounds__(TC_THREADS, 1)
tc_grouped_gemm_kernel(const __grid_constant__ CUtensorMap mapA0, const __grid_constant__ CUtensorMap mapA1,
                       const __grid_constant__ CUtensorMap mapB0, const __grid_constant__ CUtensorMap mapB1,
                       const TcParams p) {
  constexpr int B_BOXES = BN / 64;
  constexpr uint32_t STAGE_BYTES = (2 + B_BOXES) * TC_BOX_BYTES;
  constexpr int N_TILE_COLS = (EPI == TC_EPI_SWIGLU) ? BN / 2 : BN;
  constexpr uint32_t TMEM_COLS = 512;

  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * TC_STAGES + 4];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag_s;
  __shared__ int tile_prefix[257];
  __shared__ int s_counts[256];      // the experts' row counts, read from global memory once

  volatile int* abort_flag = &abort_flag_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t full_bar = smem_u32(&bars[0]);                   // [TC_STAGES]
  const uint32_t empty_bar = smem_u32(&bars[TC_STAGES]);          // [TC_STAGES]
  const uint32_t tfull_bar = smem_u32(&bars[2 * TC_STAGES]);      // [2]
  const uint32_t tempty_bar = smem_u32(&bars[2 * TC_STAGES + 2]); // [2]

  // ---- set-up ---------------------------------------------------------------------------------
  if (tid == 0) {
    abort_flag_s = 0;
    for (int s = 0; s < TC_STAGES; ++s) { mbar_init(full_bar + 8 * s, 1); mbar_init(empty_bar + 8 * s, 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar + 8 * a, 1); mbar_init(tempty_bar + 8 * a, 8); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  grid_wait();
  if (warp == 2) {
    const int nt = (p.N + N_TILE_COLS - 1) / N_TILE_COLS;
    tile_prefix_warp(tile_prefix, s_counts, p.counts, p.E, lane, [&](int n_e) {
      return nt * (p.dyn == TC_DYN_M ? (min(n_e, p.M) + TC_BM - 1) / TC_BM : (p.M + TC_BM - 1) / TC_BM);
    });
  }
  tc_fence_before();
  __syncthreads();
  grid_release();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;

  if (warp == 0) {
    // ---- TMA producer ---------------------------------------------------------------------------
    if (lane == 0) {
      int e_cur = 0, stage = 0;
      uint32_t phase = 0;
      TileCoord tc;
      bool ok = true;
      for (int tile = blockIdx.x; ok && tile_coord(p, tile_prefix, s_counts, tile, e_cur, N_TILE_COLS, tc); tile += gridDim.x) {
        for (int kb = 0; kb < tc.kblocks; ++kb) {
          if (!mbar_wait(empty_bar + 8 * stage, phase ^ 1u, abort_flag, p.wait_limit)) { ok = false; break; }
          const uint32_t fb = full_bar + 8 * stage;
          mbar_expect_tx(fb, STAGE_BYTES);
          const bool second = p.k1_blocks > 0 && kb >= p.k1_blocks;
          const int k0 = (second ? kb - p.k1_blocks : kb) * TC_BK;
          const CUtensorMap* ma = second ? &mapA1 : &mapA0;
          const uint32_t sa = tiles_base + stage * STAGE_BYTES;
          const uint32_t sb = sa + 2 * TC_BOX_BYTES;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            if (p.a_mn) tma_load_3d(sa + j * TC_BOX_BYTES, ma, fb, tc.m0 + 64 * j, k0, tc.e);
            else        tma_load_3d(sa + j * TC_BOX_BYTES, ma, fb, k0, tc.m0 + 64 * j, tc.e);
          }
#pragma unroll
          for (int j = 0; j < B_BOXES; ++j) {
            const CUtensorMap* mb = &mapB0;
            int nn = tc.n0 + 64 * j;
            if (p.dual_b) {
              if (j >= B_BOXES / 2) { mb = &mapB1; nn = tc.n0 + 64 * (j - B_BOXES / 2); }
            } else if (second) {
              mb = &mapB1;
            }
            if (p.b_mn) tma_load_3d(sb + j * TC_BOX_BYTES, mb, fb, nn, k0, tc.e);
            else        tma_load_3d(sb + j * TC_BOX_BYTES, mb, fb, k0, nn, tc.e);
          }
          if (++stage == TC_STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer ------------------------------------------------------------------------------
    if (lane == 0) {
      int e_cur = 0, stage = 0, acc_stage = 0;
      uint32_t phase = 0, acc_phase = 0;
      TileCoord tc;
      bool ok = true;
      const uint32_t a_lbo = p.a_mn ? TC_BOX_BYTES : 16u, b_lbo = p.b_mn ? TC_BOX_BYTES : 16u;
      const uint32_t a_kstep = p.a_mn ? 2048u : 32u, b_kstep = p.b_mn ? 2048u : 32u;
      for (int tile = blockIdx.x; ok && tile_coord(p, tile_prefix, s_counts, tile, e_cur, N_TILE_COLS, tc); tile += gridDim.x) {
        if (tc.kblocks == 0) continue;
        if (!mbar_wait(tempty_bar + 8 * acc_stage, acc_phase ^ 1u, abort_flag, p.wait_limit)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc_stage * 256);
        for (int kb = 0; kb < tc.kblocks; ++kb) {
          if (!mbar_wait(full_bar + 8 * stage, phase, abort_flag, p.wait_limit)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = tiles_base + stage * STAGE_BYTES;
          const uint32_t sb = sa + 2 * TC_BOX_BYTES;
#pragma unroll
          for (int kk = 0; kk < TC_BK / 16; ++kk) {
            const uint64_t ad = make_smem_desc(sa + kk * a_kstep, a_lbo, 1024u);
            const uint64_t bd = make_smem_desc(sb + kk * b_kstep, b_lbo, 1024u);
            tc_mma(d_tmem, ad, bd, p.idesc, (kb > 0 || kk > 0) ? 1u : 0u);
          }
          tc_commit(empty_bar + 8 * stage);          // frees the stage when these MMAs retire
          if (++stage == TC_STAGES) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        tc_commit(tfull_bar + 8 * acc_stage);        // accumulator complete
        if (++acc_stage == 2) { acc_stage = 0; acc_phase ^= 1u; }
      }
    }
  } else {
    // ---- epilogue warps ---------------------------------------------------------------------------
    const int q = warp & 3;                        // quarter of tensor memory this warp may read
    uint8_t* scratch = smem_raw + (tiles_base - smem_u32(smem_raw)) + TC_STAGES * STAGE_BYTES + (warp - 2) * TC_SCRATCH_BYTES;
    const int half = (warp - 2) >> 2;              // which half of the tile's columns it handles
    constexpr int NCH = N_TILE_COLS / 32 / 2;      // 32-column chunks per warp
    const int row_in_tile = 32 * q + lane;
    int e_cur = 0, acc_stage = 0;
    uint32_t acc_phase = 0;
    TileCoord tc;
    bool ok = true;
    for (int tile = blockIdx.x; ok && tile_coord(p, tile_prefix, s_counts, tile, e_cur, N_TILE_COLS, tc); tile += gridDim.x) {
      const int grow = tc.m0 + row_in_tile;
      const bool row_ok = grow < tc.m_lim;
      const int c_beg = half * NCH;
      const long long obase = (long long)tc.e * p.out_bs + (long long)grow * p.ld_out + tc.n0;
      if (tc.kblocks == 0) {        // nothing to contract: the block of the output is zero
        const int nz = min(32, max(0, tc.m_lim - (grow - lane)));
        for (int c = c_beg; c < c_beg + NCH && tc.n0 + 32 * c < p.N; ++c)
          store_zero_block(p, obase - (long long)lane * p.ld_out + 32 * c, lane, nz);
        continue;
      }
      // SwiGLU derivative: the saved G and U of the first chunk are fetched before the
      // accumulator is ready, those of chunk c+1 while chunk c is processed
      uint4 pg[4], pu[4];
      const int nvalid = min(32, max(0, tc.m_lim - (grow - lane)));
      if (EPI == TC_EPI_DSWIGLU && tc.n0 + 32 * c_beg < p.N) {
        const long long wb = obase - (long long)lane * p.ld_out + 32 * c_beg;
        load32_warp_issue(p.in0 + wb, p.ld_out, lane, nvalid, pg);
        load32_warp_issue(p.in1 + wb, p.ld_out, lane, nvalid, pu);
      }
      if (!mbar_wait(tfull_bar + 8 * acc_stage, acc_phase, abort_flag, p.wait_limit)) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + (uint32_t)(acc_stage * 256) + ((uint32_t)(32 * q) << 16);
      int sc_t = -1;
      float sc_g = 0.f;
      if (EPI == TC_EPI_STORE && p.sc_out != nullptr && row_ok && grow < p.M) {
        sc_t = p.sc_tok[(long long)tc.e * p.M + grow];
        sc_g = p.sc_gate[(long long)tc.e * p.M + grow];
      }
      epilogue_chunks<EPI, BN>(p, tc.n0, taddr, obase, row_ok, c_beg, NCH, pg, pu, scratch, lane, nvalid, sc_t, sc_g);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty_bar + 8 * acc_stage);
      if (++acc_stage == 2) { acc_stage = 0; acc_phase ^= 1u; }
    }
  }

  // ---- teardown -----------------------------------------------------------------------------------
  __syncwarp();
  if (*abort_flag) {
    // give copies that are still in flight time to land before the CTA's memory is released
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }
    if (tid == 0) atomicExch(&p.stats->error_word, 0x7c05);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// ---- two-CTA form ---------------------------------------------------------------------------------
// The same pipeline on CTA pairs (thread-block cluster of 2, tcgen05 cta_group::2): one MMA covers
// 256 x 256 x 16, each CTA holding its own 128 rows of A, half of the B tile (128 of the 256
// columns) and the accumulator of its 128 rows.  Per CTA and K block only 32 KiB enter shared
// memory instead of 48 KiB, and the tensor core reads half of B from the peer, which takes
// pressure off the shared-memory port; six stages fit.  Only the leader CTA (cluster rank 0)
// issues MMAs.  Both CTAs' TMA loads complete on the leader's "full" barrier; the leader's
// commits are multicast to both CTAs' "empty" and "accumulator full" barriers; the epilogue
// warps of both CTAs arrive on the leader's "accumulator empty" barrier.  No load is multicast.
constexpr int TC2_STAGES = 6;
constexpr uint32_t TC2_STAGE_BYTES = 4 * TC_BOX_BYTES;       // per CTA: 2 boxes of A, 2 of B

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_id_x() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_count_x() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t smem_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                                  long long limit_cycles) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const long long t0 = clock64();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((it & 255u) == 0u) {
      if (*abort_flag) return false;
      if (clock64() - t0 > limit_cycles) { *abort_flag = 1; return false; }
    }
  }
}
// TMA load into this CTA's shared memory whose completion is counted on a barrier of the pair
// (cluster address); not a multicast.
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar_cluster,
                                                 int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar_cluster), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
// Four rows of a 2-D tensor (one-row box of 64 columns), 4 x 128 bytes written consecutively.
__device__ __forceinline__ void tma_gather4_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar_cluster,
                                                 int col, int4 rows) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes.cta_group::2"
      " [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar_cluster), "r"(col), "r"(rows.x), "r"(rows.y), "r"(rows.z), "r"(rows.w)
      : "memory");
}
// Token ids of four consecutive slots, -1 replaced by the out-of-range row.
__device__ __forceinline__ int4 gather_rows(const int32_t* idx, int oob) {
  int4 r = *reinterpret_cast<const int4*>(idx);
  r.x = r.x < 0 ? oob : r.x; r.y = r.y < 0 ? oob : r.y; r.z = r.z < 0 ? oob : r.z; r.w = r.w < 0 ? oob : r.w;
  return r;
}
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {      // arrives on `bar` in both CTAs
  const uint16_t mask = 3;
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask) : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}

// Pair-tile index -> coordinates (256 rows per pair tile).
__device__ __forceinline__ bool tile_coord_pair(const TcParams& p, const int* tile_prefix, const int* counts_s,
    int tile, int& e_cur,
                                                int n_tile_cols, TileCoord& tc) {
  if (tile >= tile_prefix[p.E]) return false;
  while (tile >= tile_prefix[e_cur + 1]) ++e_cur;
  const int local = tile - tile_prefix[e_cur];
  const int n_e = counts_s[e_cur];
  int mt_count;
  if (p.dyn == TC_DYN_M) {
    mt_count = (min(n_e, p.M) + 255) / 256;
    tc.kblocks = (p.K + TC_BK - 1) / TC_BK;
    tc.last_kk = TC_BK / 16;
    tc.m_lim = (min(n_e, p.M) + TC_BM - 1) / TC_BM * TC_BM;
  } else {
    mt_count = (p.M + 255) / 256;
    tc.kblocks = (n_e + TC_BK - 1) / TC_BK;
    tc.last_kk = n_e > 0 ? ((n_e - 1) % TC_BK) / 16 + 1 : TC_BK / 16;
    tc.m_lim = p.M;
  }
  tc.e = e_cur;
  tc.m0 = (local % mt_count) * 256;
  tc.n0 = (local / mt_count) * n_tile_cols;
  return true;
}

// GATHER is TcParams::gather, and CFG the operand modes (bit 0 a_mn, 1 b_mn, 2 dual_b, 3 two K ranges), as
// compile-time constants: the single-lane producer and MMA loops are on the kernel's critical path,
// and run-time branches cost there even when not taken (6-8 % of a GEMM for the operand modes,
// 10 % per gather branch).
// A second epilogue of the SwiGLU derivative (TC_EPI_DSWIGLU_BOX): G and U of a chunk of 32 columns come by TMA into a box of
// the warp's own (32 rows of 64 bytes each, 64-byte swizzle), a lane turns its row into dG and dU in place, and TMA stores the
// boxes.  Two boxes of each per warp: a chunk's load passes under the chunk before.  The other one fetches and stores through a
// scratch, two more passes over shared memory for each of the four tensors, and 3000 cycles a chunk.  The boxes cost a stage of the
// ring (five instead of six), which long contractions miss more than they gain (fetching bounds them: three stages 279, four 250,
// five 234 us against 223 with the scratch and six at d 2048, E 128, h 768).  So below d = 2048: 89 -> 68 us at d 1024 (E 16, h 2816, 512
// rows), 60 -> 48 at d 1088, 20 -> 17 and 17 -> 14 at d 512; at d 2048 (h 1408) 177 -> 179 with 1024 rows, 170 -> 169 with 769.
constexpr int DSW_BOX_MAX_K = 2048;
constexpr uint32_t DSW_BOX = 32 * 64, DSW_SLOT = 2 * DSW_BOX;      // G and U of a chunk
struct DswMaps { CUtensorMap G, U, dG, dU; };
// Ring and epilogue space of the pair form, and behind them what would otherwise be static shared memory.  The swizzled boxes
// want a multiple of 1024: the kernel declares its dynamic block so, instead of rounding the address up as the other forms do,
// for which five stages, the boxes and this leave no room.
template <int EPI> struct PairRing {
  static constexpr int STAGES = EPI == TC_EPI_DSWIGLU_BOX ? 5 : TC2_STAGES;
  static constexpr uint32_t TAIL = STAGES * TC2_STAGE_BYTES + (EPI == TC_EPI_DSWIGLU_BOX ? 8 * 2 * DSW_SLOT : 8 * TC_SCRATCH_BYTES);
};
struct PairShared {
  uint64_t bars[30];         // 2 STAGES + 4, the boxes' 16 more
  uint32_t tmem_base_slot;
  int abort_flag;
  int tile_prefix[257];
  int counts[256];           // the experts' row counts, read from global memory once
};
__device__ __forceinline__ uint32_t dsw_addr(uint32_t box, int lane, int c) {      // 16-byte piece c of this lane's row
  return box + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4);
}
__device__ __forceinline__ void dsw_load(const DswMaps& m, uint32_t slot, uint32_t bar, int col, int row, int e) {      // one lane
  mbar_expect_tx(bar, DSW_SLOT);
  tma_load_3d(slot, &m.G, bar, col, row, e);
  tma_load_3d(slot + DSW_BOX, &m.U, bar, col, row, e);
}
__device__ __forceinline__ void dsw_store(const DswMaps& m, uint32_t slot, int col, int row, int e) {                   // one lane
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(&m.dG), "r"(slot), "r"(col), "r"(row), "r"(e) : "memory");
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(&m.dU), "r"(slot + DSW_BOX), "r"(col), "r"(row), "r"(e) : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void lds128(uint32_t a, uint32_t* w) {
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t a, const uint32_t* w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
}

template <int EPI, int GATHER, int CFG>
__global__ void __launch_bounds__(TC_THREADS, 1)
tc_grouped_gemm_pair_kernel(const __grid_constant__ CUtensorMap mapA0, const __grid_constant__ CUtensorMap mapA1,
                            const __grid_constant__ CUtensorMap mapB0, const __grid_constant__ CUtensorMap mapB1,
                            const TcParams p, const __grid_constant__ DswMaps em) {
  constexpr int BN = 256;
  constexpr int N_TILE_COLS = (EPI == TC_EPI_SWIGLU) ? BN / 2 : BN;
  constexpr uint32_t TMEM_COLS = 512;
  constexpr int STAGES = PairRing<EPI>::STAGES;
  constexpr bool A_MN = (CFG & 1) != 0, B_MN = (CFG & 2) != 0, DUAL_B = (CFG & 4) != 0, TWO_K = (CFG & 8) != 0;

  extern __shared__ __align__(1024) uint8_t pair_smem[];
  const uint32_t tiles_base = smem_u32(pair_smem);
  PairShared& sh = *reinterpret_cast<PairShared*>(pair_smem + PairRing<EPI>::TAIL);
  uint64_t* bars = sh.bars;
  uint32_t& tmem_base_slot = sh.tmem_base_slot;
  int& abort_flag_s = sh.abort_flag;
  int* tile_prefix = sh.tile_prefix;
  int* s_counts = sh.counts;

  volatile int* abort_flag = &abort_flag_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = (int)cluster_id_x(), npairs = (int)cluster_count_x();
  const uint32_t full_bar = smem_u32(&bars[0]);                    // [STAGES]  used in the leader
  const uint32_t empty_bar = smem_u32(&bars[STAGES]);          // [STAGES]  in each CTA
  const uint32_t tfull_bar = smem_u32(&bars[2 * STAGES]);      // [2]           in each CTA
  const uint32_t tempty_bar = smem_u32(&bars[2 * STAGES + 2]); // [2]           used in the leader

  if (tid == 0) {
    abort_flag_s = 0;
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar + 8 * s, 1); mbar_init(empty_bar + 8 * s, 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar + 8 * a, 1); mbar_init(tempty_bar + 8 * a, 16); }
    if (EPI == TC_EPI_DSWIGLU_BOX)
      for (int b = 0; b < 16; ++b) mbar_init(smem_u32(&bars[2 * STAGES + 4 + b]), 1);      // a box pair has landed, two per epilogue warp
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  __syncwarp();
  cluster_sync_all();                 // both CTAs' barriers exist before any remote arrive
  grid_wait();
  if (warp == 2) {
    const int nt = (p.N + N_TILE_COLS - 1) / N_TILE_COLS;
    tile_prefix_warp(tile_prefix, s_counts, p.counts, p.E, lane, [&](int n_e) {
      return nt * (p.dyn == TC_DYN_M ? (min(n_e, p.M) + 255) / 256 : (p.M + 255) / 256);
    });
  }
  tc_fence_before();
  __syncthreads();
  grid_release();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  const uint32_t leader_full = map_to_cta(full_bar, 0);
  const uint32_t leader_tempty = map_to_cta(tempty_bar, 0);

  if (warp == 0) {
    // ---- TMA producer (both CTAs) ---------------------------------------------------------------
    // Without a gather lane 0 works alone.  With one, the whole warp walks the loop: lane l
    // fetches rows 4l..4l+3 of the gathered operand's 128 (gather 1) or, for the two 64-column
    // boxes of a K block, rows 4(l%16)..+3 of box l/16 (gather 2); lane 0 issues the rest.
    if (lane == 0 || GATHER) {
      int e_cur = 0, stage = 0;
      uint32_t phase = 0;
      TileCoord tc;
      bool ok = true;
      for (int tile = pair; ok && tile_coord_pair(p, tile_prefix, s_counts, tile, e_cur, N_TILE_COLS, tc); tile += npairs) {
        const int m0c = tc.m0 + 128 * (int)rank;
        const int32_t* gidx = p.gather_idx + (size_t)tc.e * p.gather_ld;
        int4 rows_a = make_int4(0, 0, 0, 0), rows_b = make_int4(0, 0, 0, 0);
        if (GATHER == 1)      // a CTA's 128 rows lie inside the expert's C_stride slots or all past them
          rows_a = m0c < p.M ? gather_rows(gidx + m0c + 4 * lane, p.gather_oob)
                             : make_int4(p.gather_oob, p.gather_oob, p.gather_oob, p.gather_oob);
        if (GATHER == 2 && tc.kblocks > 0) rows_b = gather_rows(gidx + 4 * (lane & 15), p.gather_oob);
        for (int kb = 0; kb < tc.kblocks; ++kb) {
          int4 rows_next = rows_b;
          if (GATHER == 2 && kb + 1 < tc.kblocks)
            rows_next = gather_rows(gidx + (kb + 1) * TC_BK + 4 * (lane & 15), p.gather_oob);
          if (!mbar_wait_cluster(empty_bar + 8 * stage, phase ^ 1u, abort_flag, p.wait_limit)) { ok = false; break; }
          if (rank == 0 && lane == 0) mbar_expect_tx(full_bar + 8 * stage, 2 * TC2_STAGE_BYTES);
          const uint32_t fb = leader_full + 8 * stage;
          const bool second = TWO_K && kb >= p.k1_blocks;
          const int k0 = (second ? kb - p.k1_blocks : kb) * TC_BK;
          const CUtensorMap* ma = second ? &mapA1 : &mapA0;
          const CUtensorMap* mb = DUAL_B ? (rank ? &mapB1 : &mapB0) : (second ? &mapB1 : &mapB0);
          const int nb = DUAL_B ? tc.n0 : tc.n0 + 128 * (int)rank;
          const uint32_t sa = tiles_base + stage * TC2_STAGE_BYTES;
          const uint32_t sb = sa + 2 * TC_BOX_BYTES;
          if (GATHER == 1) tma_gather4_pair(sa + 512u * lane, &mapA0, fb, k0, rows_a);
          if (GATHER == 2)
            tma_gather4_pair(sb + (lane >> 4) * TC_BOX_BYTES + 512u * (lane & 15), &mapB0, fb,
                             nb + 64 * (lane >> 4), rows_b);
          if (lane == 0) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              if (GATHER != 1) {
                if (A_MN) tma_load_3d_pair(sa + j * TC_BOX_BYTES, ma, fb, m0c + 64 * j, k0, tc.e);
                else        tma_load_3d_pair(sa + j * TC_BOX_BYTES, ma, fb, k0, m0c + 64 * j, tc.e);
              }
              if (GATHER != 2) {
                if (B_MN) tma_load_3d_pair(sb + j * TC_BOX_BYTES, mb, fb, nb + 64 * j, k0, tc.e);
                else        tma_load_3d_pair(sb + j * TC_BOX_BYTES, mb, fb, k0, nb + 64 * j, tc.e);
              }
            }
          }
          rows_b = rows_next;
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer (leader CTA only) --------------------------------------------------------------
    if (lane == 0 && rank == 0) {
      int e_cur = 0, stage = 0, acc_stage = 0;
      uint32_t phase = 0, acc_phase = 0;
      TileCoord tc;
      bool ok = true;
      const uint32_t a_lbo = A_MN ? TC_BOX_BYTES : 16u, b_lbo = B_MN ? TC_BOX_BYTES : 16u;
      const uint32_t a_kstep = A_MN ? 2048u : 32u, b_kstep = B_MN ? 2048u : 32u;
      for (int tile = pair; ok && tile_coord_pair(p, tile_prefix, s_counts, tile, e_cur, N_TILE_COLS, tc); tile += npairs) {
        if (tc.kblocks == 0) continue;
        if (!mbar_wait_cluster(tempty_bar + 8 * acc_stage, acc_phase ^ 1u, abort_flag, p.wait_limit)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc_stage * 256);
        // A contraction over the expert's rows (operand modes 3, or the generic form) ends in a K block
        // whose last 16-wide steps may hold pad rows only: that block is peeled off the loop and runs
        // just the steps with rows in use (the skipped ones would add zeros).  The loop itself stays
        // free of the test: anything extra in it shows in the GEMM time.
        constexpr bool PEEL = CFG == 3;
        const int nloop = PEEL ? tc.kblocks - 1 : tc.kblocks;
        for (int kb = 0; kb < nloop; ++kb) {
          if (!mbar_wait_cluster(full_bar + 8 * stage, phase, abort_flag, p.wait_limit)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = tiles_base + stage * TC2_STAGE_BYTES;
          const uint32_t sb = sa + 2 * TC_BOX_BYTES;
#pragma unroll
          for (int kk = 0; kk < TC_BK / 16; ++kk) {
            const uint64_t ad = make_smem_desc(sa + kk * a_kstep, a_lbo, 1024u);
            const uint64_t bd = make_smem_desc(sb + kk * b_kstep, b_lbo, 1024u);
            tc_mma_pair(d_tmem, ad, bd, p.idesc, (kb > 0 || kk > 0) ? 1u : 0u);
          }
          tc_commit_pair(empty_bar + 8 * stage);      // frees the stage in both CTAs
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (PEEL && ok) {
          if (!mbar_wait_cluster(full_bar + 8 * stage, phase, abort_flag, p.wait_limit)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = tiles_base + stage * TC2_STAGE_BYTES;
          const uint32_t sb = sa + 2 * TC_BOX_BYTES;
#pragma unroll
          for (int kk = 0; kk < TC_BK / 16; ++kk) {
            if (kk < tc.last_kk) {
              const uint64_t ad = make_smem_desc(sa + kk * a_kstep, a_lbo, 1024u);
              const uint64_t bd = make_smem_desc(sb + kk * b_kstep, b_lbo, 1024u);
              tc_mma_pair(d_tmem, ad, bd, p.idesc, (nloop > 0 || kk > 0) ? 1u : 0u);
            }
          }
          tc_commit_pair(empty_bar + 8 * stage);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        tc_commit_pair(tfull_bar + 8 * acc_stage);    // accumulators complete in both CTAs
        if (++acc_stage == 2) { acc_stage = 0; acc_phase ^= 1u; }
      }
    }
  } else {
    // ---- epilogue warps (both CTAs, own 128 rows) -----------------------------------------------------
    const int q = warp & 3;
    uint8_t* scratch = pair_smem + STAGES * TC2_STAGE_BYTES + (warp - 2) * TC_SCRATCH_BYTES;
    const int half = (warp - 2) >> 2;
    constexpr int NCH = N_TILE_COLS / 32 / 2;
    const int row_in_tile = 128 * (int)rank + 32 * q + lane;
    int e_cur = 0, acc_stage = 0;
    uint32_t acc_phase = 0, box_phase = 0;
    TileCoord tc;
    bool ok = true;
    for (int tile = pair; ok && tile_coord_pair(p, tile_prefix, s_counts, tile, e_cur, N_TILE_COLS, tc); tile += npairs) {
      const int grow = tc.m0 + row_in_tile;
      const bool row_ok = grow < tc.m_lim;
      const int c_beg = half * NCH;
      const long long obase = (long long)tc.e * p.out_bs + (long long)grow * p.ld_out + tc.n0;
      if (tc.kblocks == 0) {
        const int nz = min(32, max(0, tc.m_lim - (grow - lane)));
        for (int c = c_beg; c < c_beg + NCH && tc.n0 + 32 * c < p.N; ++c)
          store_zero_block(p, obase - (long long)lane * p.ld_out + 32 * c, lane, nz);
        continue;
      }
      const int nvalid = min(32, max(0, tc.m_lim - (grow - lane)));
      if constexpr (EPI == TC_EPI_DSWIGLU_BOX) {
        const int row = grow - lane, col = tc.n0 + 32 * c_beg;
        // Chunks of this warp, none where its rows or its half of the columns are past the edge (N - col is then as low as
        // -64, at N = 64 mod 256): never negative, the accumulator is given back below for none and at the last one else.
        const int nch = nvalid > 0 ? min(NCH, (max(0, p.N - col) + 31) / 32) : 0;
        const uint32_t slots = tiles_base + STAGES * TC2_STAGE_BYTES + (uint32_t)(warp - 2) * 2 * DSW_SLOT;
        const uint32_t lbar = smem_u32(&bars[2 * STAGES + 4 + 2 * (warp - 2)]);
        if (lane == 0) {
          asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");      // the last tile's boxes have been read
          for (int c = 0; c < min(nch, 2); ++c) dsw_load(em, slots + c * DSW_SLOT, lbar + 8 * c, col + 32 * c, row, tc.e);
        }
        __syncwarp();
        ok = __all_sync(0xffffffffu, mbar_wait_cluster(tfull_bar + 8 * acc_stage, acc_phase, abort_flag, p.wait_limit));
        if (!ok) break;
        tc_fence_after();
        const uint32_t taddr = tmem_base + (uint32_t)(acc_stage * 256 + 32 * c_beg) + ((uint32_t)(32 * q) << 16);
        for (int c = 0; c < nch; ++c) {
          const int b = c & 1;
          const uint32_t slot = slots + b * DSW_SLOT;
          uint32_t r0[32], gw[16], uw[16];
          tc_ld32(taddr + 32 * c, r0);
          ok = __all_sync(0xffffffffu, mbar_wait(lbar + 8 * b, (box_phase >> b) & 1u, abort_flag, p.wait_limit));
          if (!ok) break;
          box_phase ^= 1u << b;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            lds128(dsw_addr(slot, lane, i), gw + 4 * i);
            lds128(dsw_addr(slot + DSW_BOX, lane, i), uw + 4 * i);
          }
          tc_wait_ld();
          if (c + 1 == nch) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * acc_stage);
          }
#pragma unroll
          for (int i = 0; i < 16; ++i)
            dswiglu_pair(__uint_as_float(r0[2 * i]), __uint_as_float(r0[2 * i + 1]), gw[i], uw[i]);
          if (c >= 1 && c + 1 < nch && lane == 0) {      // the other slot has been stored a chunk ago
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            dsw_load(em, slots + (b ^ 1) * DSW_SLOT, lbar + 8 * (b ^ 1), col + 32 * (c + 1), row, tc.e);
          }
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            sts128(dsw_addr(slot, lane, i), gw + 4 * i);
            sts128(dsw_addr(slot + DSW_BOX, lane, i), uw + 4 * i);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) dsw_store(em, slot, col + 32 * c, row, tc.e);
        }
        if (!ok) break;
        if (nch == 0) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * acc_stage);
        }
        if (++acc_stage == 2) { acc_stage = 0; acc_phase ^= 1u; }
        continue;
      }
      uint4 pg[4], pu[4];
      if (EPI == TC_EPI_DSWIGLU && tc.n0 + 32 * c_beg < p.N) {
        const long long wb = obase - (long long)lane * p.ld_out + 32 * c_beg;
        load32_warp_issue(p.in0 + wb, p.ld_out, lane, nvalid, pg);
        load32_warp_issue(p.in1 + wb, p.ld_out, lane, nvalid, pu);
      }
      if (!mbar_wait_cluster(tfull_bar + 8 * acc_stage, acc_phase, abort_flag, p.wait_limit)) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + (uint32_t)(acc_stage * 256) + ((uint32_t)(32 * q) << 16);
      int sc_t = -1;
      float sc_g = 0.f;
      if (EPI == TC_EPI_STORE && p.sc_out != nullptr && row_ok && grow < p.M) {
        sc_t = p.sc_tok[(long long)tc.e * p.M + grow];
        sc_g = p.sc_gate[(long long)tc.e * p.M + grow];
      }
      if (EPI == TC_EPI_STORE && CFG == 3) {
        // Weight gradients: a tile of a few rows' contraction is all epilogue, so the accumulators are read in one go
        // (four loads in flight instead of a wait per chunk) and released before the stores.
        constexpr int NC = EPI == TC_EPI_STORE ? NCH : 1;
        uint32_t r[NC][32];
#pragma unroll
        for (int c = 0; c < NC; ++c) tc_ld32(taddr + 32 * (c_beg + c), r[c]);
        tc_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * acc_stage);
        const long long wb = obase - (long long)lane * p.ld_out + 32 * c_beg;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          if (tc.n0 + 32 * (c_beg + c) >= p.N) break;
          if (p.out_f32) {
            store32_warp_f32(scratch, lane, nvalid, reinterpret_cast<float*>(p.out0) + wb + 32 * c, p.ld_out, r[c]);
          } else {
            uint32_t pk[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) pk[i] = pack_bf16(__uint_as_float(r[c][2 * i]), __uint_as_float(r[c][2 * i + 1]));
            store32_warp_packed(scratch, lane, nvalid, p.out0 + wb + 32 * c, p.ld_out, pk);
          }
        }
      } else {
        epilogue_chunks<EPI, BN>(p, tc.n0, taddr, obase, row_ok, c_beg, NCH, pg, pu, scratch, lane, nvalid, sc_t, sc_g);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * acc_stage);
      }
      if (++acc_stage == 2) { acc_stage = 0; acc_phase ^= 1u; }
    }
    if (EPI == TC_EPI_DSWIGLU_BOX && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }

  // ---- teardown: neither CTA leaves while the other may still touch its barriers or memory -------
  __syncwarp();
  if (*abort_flag) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }
    if (tid == 0) atomicExch(&p.stats->error_word, 0x7c06);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
  cluster_sync_all();                 // the next kernel's blocks may start on an SM as soon as its CTA is gone
}

// ---- CTA-pair kernel, two output tiles per pass ------------------------------------------------------
// Same pair as above, but one pass covers 256 rows x 2 adjacent column tiles: the A boxes of a K
// block are fetched once and multiplied into two accumulators (tensor-memory columns [0,256) and
// [256,512)), so a K block moves 48 KiB per CTA for twice the flops of the 32 KiB above: a
// quarter less operand traffic from L2 per flop.  The price is that all of tensor memory is one
// tile's accumulator: the next tile's MMAs wait for the epilogue.  To hide most of that, the
// epilogue drains and releases the two halves separately, and the MMA warp runs the first K
// blocks of the next tile into half 0 alone (those stages stay held) until half 1 is free.
constexpr int TCW_STAGES = 4;
constexpr uint32_t TCW_STAGE_BYTES = 6 * TC_BOX_BYTES;       // per CTA: 2 boxes of A, 2 + 2 of B
constexpr int TCW_LEAD = TCW_STAGES - 1;                     // K blocks half 0 may run ahead of half 1

__device__ __forceinline__ bool tile_coord_wide(const TcParams& p, const int* tile_prefix, const int* counts_s,
    int tile, int& e_cur,
                                                int n_tile_cols, TileCoord& tc) {
  if (tile >= tile_prefix[p.E]) return false;
  while (tile >= tile_prefix[e_cur + 1]) ++e_cur;
  const int local = tile - tile_prefix[e_cur];
  const int n_e = counts_s[e_cur];
  int mt_count;
  if (p.dyn == TC_DYN_M) {
    mt_count = (min(n_e, p.M) + 255) / 256;
    tc.kblocks = (p.K + TC_BK - 1) / TC_BK;
    tc.last_kk = TC_BK / 16;
    tc.m_lim = (min(n_e, p.M) + TC_BM - 1) / TC_BM * TC_BM;
  } else {
    mt_count = (p.M + 255) / 256;
    tc.kblocks = (n_e + TC_BK - 1) / TC_BK;
    tc.last_kk = n_e > 0 ? ((n_e - 1) % TC_BK) / 16 + 1 : TC_BK / 16;
    tc.m_lim = p.M;
  }
  tc.e = e_cur;
  tc.m0 = (local % mt_count) * 256;
  tc.n0 = (local / mt_count) * 2 * n_tile_cols;
  return true;
}

template <int EPI, int GATHER, int CFG>
__global__ void __launch_bounds__(TC_THREADS, 1)
tc_grouped_gemm_pair_wide_kernel(const __grid_constant__ CUtensorMap mapA0, const __grid_constant__ CUtensorMap mapA1,
                                 const __grid_constant__ CUtensorMap mapB0, const __grid_constant__ CUtensorMap mapB1,
                                 const TcParams p) {
  constexpr int BN = 256;
  constexpr int N_TILE_COLS = (EPI == TC_EPI_SWIGLU) ? BN / 2 : BN;
  constexpr uint32_t TMEM_COLS = 512;
  constexpr bool A_MN = (CFG & 1) != 0, B_MN = (CFG & 2) != 0, DUAL_B = (CFG & 4) != 0, TWO_K = (CFG & 8) != 0;

  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * TCW_STAGES + 3];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag_s;
  __shared__ int tile_prefix[257];
  __shared__ int s_counts[256];      // the experts' row counts, read from global memory once

  volatile int* abort_flag = &abort_flag_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = (int)cluster_id_x(), npairs = (int)cluster_count_x();
  const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t full_bar = smem_u32(&bars[0]);                    // [TCW_STAGES]  used in the leader
  const uint32_t empty_bar = smem_u32(&bars[TCW_STAGES]);          // [TCW_STAGES]  in each CTA
  const uint32_t tfull_bar = smem_u32(&bars[2 * TCW_STAGES]);      // [1]           in each CTA
  const uint32_t tempty_bar = smem_u32(&bars[2 * TCW_STAGES + 1]); // [2]           used in the leader

  if (tid == 0) {
    abort_flag_s = 0;
    for (int s = 0; s < TCW_STAGES; ++s) { mbar_init(full_bar + 8 * s, 1); mbar_init(empty_bar + 8 * s, 1); }
    mbar_init(tfull_bar, 1);
    for (int a = 0; a < 2; ++a) mbar_init(tempty_bar + 8 * a, 16);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  __syncwarp();
  cluster_sync_all();                 // both CTAs' barriers exist before any remote arrive
  grid_wait();
  if (warp == 2) {
    const int nt = (p.N + 2 * N_TILE_COLS - 1) / (2 * N_TILE_COLS);
    tile_prefix_warp(tile_prefix, s_counts, p.counts, p.E, lane, [&](int n_e) {
      return nt * (p.dyn == TC_DYN_M ? (min(n_e, p.M) + 255) / 256 : (p.M + 255) / 256);
    });
  }
  tc_fence_before();
  __syncthreads();
  grid_release();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  const uint32_t leader_full = map_to_cta(full_bar, 0);
  const uint32_t leader_tempty = map_to_cta(tempty_bar, 0);

  if (warp == 0) {
    // ---- TMA producer (both CTAs) ---------------------------------------------------------------
    // Lane 0 alone, or with a gathered A operand the whole warp (lane l fetches rows 4l..4l+3 of
    // the CTA's 128 rows of A; lane 0 also issues the B boxes).
    if (lane == 0 || GATHER) {
      int e_cur = 0, stage = 0;
      uint32_t phase = 0;
      TileCoord tc;
      bool ok = true;
      for (int tile = pair; ok && tile_coord_wide(p, tile_prefix, s_counts, tile, e_cur, N_TILE_COLS, tc); tile += npairs) {
        const int m0c = tc.m0 + 128 * (int)rank;
        const bool two = tc.n0 + N_TILE_COLS < p.N;
        int4 rows_a = make_int4(0, 0, 0, 0);
        if (GATHER == 1)
          rows_a = m0c < p.M ? gather_rows(p.gather_idx + (size_t)tc.e * p.gather_ld + m0c + 4 * lane, p.gather_oob)
                             : make_int4(p.gather_oob, p.gather_oob, p.gather_oob, p.gather_oob);
        for (int kb = 0; kb < tc.kblocks; ++kb) {
          if (!mbar_wait_cluster(empty_bar + 8 * stage, phase ^ 1u, abort_flag, p.wait_limit)) { ok = false; break; }
          if (rank == 0 && lane == 0) mbar_expect_tx(full_bar + 8 * stage, 2 * (two ? 6 : 4) * TC_BOX_BYTES);
          const uint32_t fb = leader_full + 8 * stage;
          const bool second = TWO_K && kb >= p.k1_blocks;
          const int k0 = (second ? kb - p.k1_blocks : kb) * TC_BK;
          const CUtensorMap* ma = second ? &mapA1 : &mapA0;
          const CUtensorMap* mb = DUAL_B ? (rank ? &mapB1 : &mapB0) : (second ? &mapB1 : &mapB0);
          const uint32_t sa = tiles_base + stage * TCW_STAGE_BYTES;
          if (GATHER == 1) tma_gather4_pair(sa + 512u * lane, &mapA0, fb, k0, rows_a);
          if (lane == 0) {
            if (GATHER != 1) {
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                if (A_MN) tma_load_3d_pair(sa + j * TC_BOX_BYTES, ma, fb, m0c + 64 * j, k0, tc.e);
                else        tma_load_3d_pair(sa + j * TC_BOX_BYTES, ma, fb, k0, m0c + 64 * j, tc.e);
              }
            }
            for (int hf = 0; hf < (two ? 2 : 1); ++hf) {
              const uint32_t sb = sa + (2 + 2 * hf) * TC_BOX_BYTES;
              const int nh = tc.n0 + hf * N_TILE_COLS;
              const int nb = DUAL_B ? nh : nh + 128 * (int)rank;
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                if (B_MN) tma_load_3d_pair(sb + j * TC_BOX_BYTES, mb, fb, nb + 64 * j, k0, tc.e);
                else        tma_load_3d_pair(sb + j * TC_BOX_BYTES, mb, fb, k0, nb + 64 * j, tc.e);
              }
            }
          }
          if (++stage == TCW_STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer (leader CTA only) --------------------------------------------------------------
    if (lane == 0 && rank == 0) {
      int e_cur = 0, stage = 0;
      uint32_t phase = 0, acc_phase = 0;
      TileCoord tc;
      bool ok = true;
      const uint32_t a_lbo = A_MN ? TC_BOX_BYTES : 16u, b_lbo = B_MN ? TC_BOX_BYTES : 16u;
      const uint32_t a_kstep = A_MN ? 2048u : 32u, b_kstep = B_MN ? 2048u : 32u;
      // one K block of one half: 4 MMAs of 256 x 256 x 16
      auto issue = [&](int st, int hf, bool first_block) {
        const uint32_t sa = tiles_base + st * TCW_STAGE_BYTES;
        const uint32_t sb = sa + (2 + 2 * hf) * TC_BOX_BYTES;
#pragma unroll
        for (int kk = 0; kk < TC_BK / 16; ++kk) {
          const uint64_t ad = make_smem_desc(sa + kk * a_kstep, a_lbo, 1024u);
          const uint64_t bd = make_smem_desc(sb + kk * b_kstep, b_lbo, 1024u);
          tc_mma_pair(tmem_base + (uint32_t)(hf * 256), ad, bd, p.idesc, (!first_block || kk > 0) ? 1u : 0u);
        }
      };
      for (int tile = pair; ok && tile_coord_wide(p, tile_prefix, s_counts, tile, e_cur, N_TILE_COLS, tc); tile += npairs) {
        if (tc.kblocks == 0) continue;
        const bool two = tc.n0 + N_TILE_COLS < p.N;
        if (!mbar_wait_cluster(tempty_bar, acc_phase ^ 1u, abort_flag, p.wait_limit)) { ok = false; break; }
        tc_fence_after();
        // Lead-in: half 0 of the first K blocks while the epilogue still drains half 1.
        const int lead = two ? min(TCW_LEAD, tc.kblocks) : 0;
        int st = stage;
        uint32_t ph = phase;
        for (int kb = 0; kb < lead; ++kb) {
          if (!mbar_wait_cluster(full_bar + 8 * st, ph, abort_flag, p.wait_limit)) { ok = false; break; }
          tc_fence_after();
          issue(st, 0, kb == 0);
          if (++st == TCW_STAGES) { st = 0; ph ^= 1u; }
        }
        if (!ok) break;
        if (!mbar_wait_cluster(tempty_bar + 8, acc_phase ^ 1u, abort_flag, p.wait_limit)) { ok = false; break; }
        tc_fence_after();
        for (int kb = 0; kb < tc.kblocks; ++kb) {
          if (kb >= lead) {
            if (!mbar_wait_cluster(full_bar + 8 * stage, phase, abort_flag, p.wait_limit)) { ok = false; break; }
            tc_fence_after();
            issue(stage, 0, kb == 0);
          }
          if (two) issue(stage, 1, kb == 0);
          tc_commit_pair(empty_bar + 8 * stage);      // frees the stage in both CTAs
          if (++stage == TCW_STAGES) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        tc_commit_pair(tfull_bar);                    // both accumulators complete in both CTAs
        acc_phase ^= 1u;
      }
    }
  } else {
    // ---- epilogue warps (both CTAs, own 128 rows) -----------------------------------------------------
    const int q = warp & 3;
    uint8_t* scratch = smem_raw + (tiles_base - smem_u32(smem_raw)) + TCW_STAGES * TCW_STAGE_BYTES + (warp - 2) * TC_SCRATCH_BYTES;
    const int half = (warp - 2) >> 2;
    constexpr int NCH = N_TILE_COLS / 32 / 2;
    const int row_in_tile = 128 * (int)rank + 32 * q + lane;
    int e_cur = 0;
    uint32_t acc_phase = 0;
    TileCoord tc;
    bool ok = true;
    for (int tile = pair; ok && tile_coord_wide(p, tile_prefix, s_counts, tile, e_cur, N_TILE_COLS, tc); tile += npairs) {
      const int grow = tc.m0 + row_in_tile;
      const bool row_ok = grow < tc.m_lim;
      const int c_beg = half * NCH;
      const bool two = tc.n0 + N_TILE_COLS < p.N;
      const long long obase = (long long)tc.e * p.out_bs + (long long)grow * p.ld_out + tc.n0;
      if (tc.kblocks == 0) {
        const int nz = min(32, max(0, tc.m_lim - (grow - lane)));
        for (int hf = 0; hf < (two ? 2 : 1); ++hf)
          for (int c = c_beg; c < c_beg + NCH && tc.n0 + hf * N_TILE_COLS + 32 * c < p.N; ++c)
            store_zero_block(p, obase - (long long)lane * p.ld_out + hf * N_TILE_COLS + 32 * c, lane, nz);
        continue;
      }
      uint4 pg[4], pu[4];
      const int nvalid = min(32, max(0, tc.m_lim - (grow - lane)));
      if (EPI == TC_EPI_DSWIGLU && tc.n0 + 32 * c_beg < p.N) {
        const long long wb = obase - (long long)lane * p.ld_out + 32 * c_beg;
        load32_warp_issue(p.in0 + wb, p.ld_out, lane, nvalid, pg);
        load32_warp_issue(p.in1 + wb, p.ld_out, lane, nvalid, pu);
      }
      int sc_t = -1;
      float sc_g = 0.f;
      if (EPI == TC_EPI_STORE && p.sc_out != nullptr && row_ok && grow < p.M) {
        sc_t = p.sc_tok[(long long)tc.e * p.M + grow];
        sc_g = p.sc_gate[(long long)tc.e * p.M + grow];
      }
      if (!mbar_wait_cluster(tfull_bar, acc_phase, abort_flag, p.wait_limit)) { ok = false; break; }
      tc_fence_after();
      if (EPI == TC_EPI_STORE && !p.out_f32) {
        // Plain stores: empty each half into registers (packed bf16) and release it at once;
        // the turn through the scratch and the global stores follow while the MMAs run on.
        static_assert(EPI != TC_EPI_STORE || NCH == 4, "four chunks of 32 columns per warp and half");
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t pk[NCH][16];
          const int n0h = tc.n0 + hf * N_TILE_COLS;
          const bool live = hf == 0 || two;
          if (live) {
            const uint32_t taddr = tmem_base + (uint32_t)(hf * 256) + ((uint32_t)(32 * q) << 16);
            uint32_t r[NCH][32];
#pragma unroll
            for (int c = 0; c < NCH; ++c) tc_ld32(taddr + 32 * (c_beg + c), r[c]);
            tc_wait_ld();
#pragma unroll
            for (int c = 0; c < NCH; ++c)
#pragma unroll
              for (int i = 0; i < 16; ++i)
                pk[c][i] = pack_bf16(__uint_as_float(r[c][2 * i]), __uint_as_float(r[c][2 * i + 1]));
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * hf);
          if (live) {
            const long long wb = obase - (long long)lane * p.ld_out + hf * N_TILE_COLS;
#pragma unroll
            for (int c = 0; c < NCH; ++c)
              if (n0h + 32 * (c_beg + c) < p.N)
              {
                store32_warp_packed(scratch, lane, nvalid, p.out0 + wb + 32 * (c_beg + c), p.ld_out, pk[c]);
                if (p.sc_out != nullptr)
                  scatter32_warp(scratch, lane, sc_t, sc_g, p.sc_out, p.sc_ld, n0h + 32 * (c_beg + c), pk[c]);
              }
          }
        }
      } else if (EPI == TC_EPI_SWIGLU) {
        // Fused SwiGLU: G and U of a half are read, H computed, and all three packed to bf16 in
        // registers before the half is released; the stores follow.
        static_assert(EPI != TC_EPI_SWIGLU || NCH == 2, "two chunks of 32 gate columns per warp and half");
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t pk[NCH][3][16];
          const int n0h = tc.n0 + hf * N_TILE_COLS;
          const bool live = hf == 0 || two;
          if (live) {
            const uint32_t taddr = tmem_base + (uint32_t)(hf * 256) + ((uint32_t)(32 * q) << 16);
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
              uint32_t r0[32], r1[32];
              tc_ld32(taddr + 32 * (c_beg + c), r0);
              tc_ld32(taddr + BN / 2 + 32 * (c_beg + c), r1);
              tc_wait_ld();
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const float g0 = __uint_as_float(r0[2 * i]), g1 = __uint_as_float(r0[2 * i + 1]);
                const float u0 = __uint_as_float(r1[2 * i]), u1 = __uint_as_float(r1[2 * i + 1]);
                pk[c][0][i] = pack_bf16(g0, g1);
                pk[c][1][i] = pack_bf16(u0, u1);
                pk[c][2][i] = pack_bf16(__fdividef(g0, 1.0f + __expf(-g0)) * u0, __fdividef(g1, 1.0f + __expf(-g1)) * u1);
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * hf);
          if (live) {
            const long long wb = obase - (long long)lane * p.ld_out + hf * N_TILE_COLS;
#pragma unroll
            for (int c = 0; c < NCH; ++c)
              if (n0h + 32 * (c_beg + c) < p.N) {
                store32_warp_packed(scratch, lane, nvalid, p.out0 + wb + 32 * (c_beg + c), p.ld_out, pk[c][0]);
                store32_warp_packed(scratch, lane, nvalid, p.out2 + wb + 32 * (c_beg + c), p.ld_out, pk[c][2]);
                store32_warp_packed(scratch, lane, nvalid, p.out1 + wb + 32 * (c_beg + c), p.ld_out, pk[c][1]);
              }
          }
        }
      } else {
        for (int hf = 0; hf < 2; ++hf) {
          if (hf == 0 || two) {
            const int n0h = tc.n0 + hf * N_TILE_COLS;
            const long long ob = obase + hf * N_TILE_COLS;
            if (EPI == TC_EPI_DSWIGLU && hf == 1 && n0h + 32 * c_beg < p.N) {
              const long long wb = ob - (long long)lane * p.ld_out + 32 * c_beg;
              load32_warp_issue(p.in0 + wb, p.ld_out, lane, nvalid, pg);
              load32_warp_issue(p.in1 + wb, p.ld_out, lane, nvalid, pu);
            }
            const uint32_t taddr = tmem_base + (uint32_t)(hf * 256) + ((uint32_t)(32 * q) << 16);
            epilogue_chunks<EPI, BN>(p, n0h, taddr, ob, row_ok, c_beg, NCH, pg, pu, scratch, lane, nvalid, sc_t, sc_g);
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * hf);
        }
      }
      acc_phase ^= 1u;
    }
  }

  // ---- teardown: neither CTA leaves while the other may still touch its barriers or memory -------
  __syncwarp();
  if (*abort_flag) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }
    if (tid == 0) atomicExch(&p.stats->error_word, 0x7c07);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
  cluster_sync_all();                 // the next kernel's blocks may start on an SM as soon as its CTA is gone
}

// ---- CTA-pair kernel, operands exchanged ---------------------------------------------------------------
// The contractions whose rows are the expert's tokens, with the weights as the M operand (256 rows of them per
// pair, always full) and the tokens as N: N may be any multiple of 16 up to 256, so an expert's n rows are cut
// into ceil(n / 256) tiles of equal size and only the last 16-row step is padded, where the forms above compute
// whole tiles of 256 (or 128) token rows.  With few rows per expert (decoding) an MMA costs next to nothing and
// the kernel is a stream of the weights.
//
//   out[t][n] = sum_k tokens[t][k] * weights[n][k]:  accumulator lane = n, column = token
//
// The epilogue turns the 32 x 32 blocks (lane = output column) through the warp's scratch with transposing stmatrix
// (16-bit stores instead made the fused epilogues the bound of contractions over 1024 or less).
// SwiGLU: the 128 rows of a CTA are 64 rows of W1g and the same 64 of W1u; the warps that hold U hand it, in
// fp32, to the warps that hold G through shared memory.  Ring, roles, waits and teardown are those of the pair form.
constexpr uint32_t TCS_XBUF_BYTES = 16 * 32 * 4;      // per pair of epilogue warps: U of 16 tokens x 32 columns

struct SwapParams {
  int two_k;             // the first half of the K blocks from (A0, B0), the rest from (A1, B1)
  int M, N, K, E;        // M: C_stride (bound of an expert's rows), N: output columns, K: of one range
  int tok_box;           // rows of a token box (8, 16, 32 or 64)
  const int32_t* counts;
  __nv_bfloat16* out0; __nv_bfloat16* out1; __nv_bfloat16* out2;
  const __nv_bfloat16* in0; const __nv_bfloat16* in1;
  etr_stats* stats;
  const int32_t* sc_tok; const float* sc_gate; __nv_bfloat16* sc_out; int sc_ld;      // as in TcParams
  long long wait_limit;
};
struct SwapTile { int e, n0, t0, nt, rows, kblocks; };      // nt: tokens of the tile (a multiple of 16)

__device__ __forceinline__ int swap_tile_rows(int n) {      // tokens per tile of an expert with n > 0 rows
  const int parts = (n + 255) / 256;
  return ((n + parts - 1) / parts + 15) & ~15;
}
__device__ __forceinline__ bool swap_tile(const SwapParams& p, const int* tile_prefix, const int* counts_s, int tile,
                                          int& e_cur, int cols, SwapTile& t) {
  if (tile >= tile_prefix[p.E]) return false;
  while (tile >= tile_prefix[e_cur + 1]) ++e_cur;
  const int local = tile - tile_prefix[e_cur], n = min(counts_s[e_cur], p.M);
  const int size = swap_tile_rows(n), parts = (n - 1) / size + 1;
  t.e = e_cur;
  t.rows = n;
  t.t0 = (local % parts) * size;
  t.nt = min(size, (n - t.t0 + 15) & ~15);
  t.n0 = (local / parts) * cols;
  t.kblocks = (p.K + TC_BK - 1) / TC_BK * (p.two_k ? 2 : 1);
  return true;
}

// A 32 x 32 block of accumulators (lanes = output columns, columns = tokens) as matrix fragments: two loads of
// 16 lanes, each thread lane t / 4 (and + 8) at the token pair 2 (t % 4) of every eight tokens.  Value index
// 16 * (lane half) + 4 * (eight tokens) + 2 * (+ 8 lanes) + (token of the pair): the fragment of stmatrix and
// ldmatrix, whose transposing forms turn the block to and from row-major bf16.
__device__ __forceinline__ void tc_ld_block(uint32_t taddr, uint32_t* r) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t* p = r + 16 * h;
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(p[0]), "=r"(p[1]), "=r"(p[2]), "=r"(p[3]), "=r"(p[4]), "=r"(p[5]), "=r"(p[6]), "=r"(p[7]),
          "=r"(p[8]), "=r"(p[9]), "=r"(p[10]), "=r"(p[11]), "=r"(p[12]), "=r"(p[13]), "=r"(p[14]), "=r"(p[15])
        : "r"(taddr + ((uint32_t)(16 * h) << 16)));
  }
}
// Address of this lane's row of the 8 x 8 matrices of eight tokens (i): token row, 16 bytes per 8 output columns.
__device__ __forceinline__ uint32_t turn_addr(const uint8_t* scratch, int lane, int i) {
  return smem_u32(scratch) + (8 * i + (lane & 7)) * TC_SCRATCH_ROW_BYTES + (lane >> 3) * 16;
}
// Such a block, rounded to bf16, to rows 0 .. nrows - 1 of dst (first row, first of the 32 columns).
__device__ __forceinline__ void store_turned(uint8_t* scratch, int lane, int nrows, __nv_bfloat16* dst, int ld,
                                             const float* v) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};"
                 ::"r"(turn_addr(scratch, lane, i)), "r"(pack_bf16(v[4 * i], v[4 * i + 1])),
                 "r"(pack_bf16(v[4 * i + 2], v[4 * i + 3])), "r"(pack_bf16(v[16 + 4 * i], v[16 + 4 * i + 1])),
                 "r"(pack_bf16(v[16 + 4 * i + 2], v[16 + 4 * i + 3])) : "memory");
  __syncwarp();
  const int sub = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = (lane >> 2) + 8 * i;
    const uint4 w = *reinterpret_cast<const uint4*>(scratch + row * TC_SCRATCH_ROW_BYTES + sub * 16);
    if (row < nrows) *reinterpret_cast<uint4*>(dst + (long long)row * ld + sub * 8) = w;
  }
  __syncwarp();
}
// The block just stored once more, scaled, to the rows of its tokens (Top-1 combine, see scatter32_warp); the
// scratch still holds it.
__device__ __forceinline__ void scatter_turned(const uint8_t* scratch, int lane, int nrows, const int32_t* tok,
                                               const float* gate, __nv_bfloat16* out, int ld) {
  const int sub = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = (lane >> 2) + 8 * i;
    if (row >= nrows) continue;
    const int t = tok[row];
    if (t < 0) continue;
    const float g = gate[row];
    const uint4 w = *reinterpret_cast<const uint4*>(scratch + row * TC_SCRATCH_ROW_BYTES + sub * 16);
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
    uint32_t y[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) y[k] = pack_bf16(g * __uint_as_float(u[k] << 16), g * __uint_as_float(u[k] & 0xffff0000u));
    *reinterpret_cast<uint4*>(out + (long long)t * ld + sub * 8) = make_uint4(y[0], y[1], y[2], y[3]);
  }
  __syncwarp();
}
// The reverse: a 32-row x 32-column block fetched by load32_warp_issue, as fragments of bf16 pairs (word
// 4 * (eight tokens) + matrix, the pairs that store_turned packs).
__device__ __forceinline__ void load_turned(uint8_t* scratch, int lane, const uint4 (&t)[4], uint32_t* w) {
  const int sub = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    *reinterpret_cast<uint4*>(scratch + ((lane >> 2) + 8 * i) * TC_SCRATCH_ROW_BYTES + sub * 16) = t[i];
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 4; ++i)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w[4 * i]), "=r"(w[4 * i + 1]), "=r"(w[4 * i + 2]), "=r"(w[4 * i + 3])
                 : "r"(turn_addr(scratch, lane, i)) : "memory");
  __syncwarp();
}
// Zeros to rows r0 .. r1 - 1 of a 32-column block (the pad rows behind an expert's last tile), 8 rows at a time.
__device__ __forceinline__ void zero_rows32(__nv_bfloat16* dst, int ld, int r0, int r1, int lane) {
  for (int r = r0 + (lane >> 2); r < r1; r += 8)
    *reinterpret_cast<uint4*>(dst + (long long)r * ld + (lane & 3) * 8) = make_uint4(0, 0, 0, 0);
}

template <int EPI, bool A_MN>
__global__ void __launch_bounds__(TC_THREADS, 1)
tc_grouped_gemm_swap_kernel(const __grid_constant__ CUtensorMap mapA0, const __grid_constant__ CUtensorMap mapA1,
                            const __grid_constant__ CUtensorMap mapB0, const __grid_constant__ CUtensorMap mapB1,
                            const SwapParams p, uint32_t idesc) {
  constexpr bool DUAL = EPI == TC_EPI_SWIGLU;
  constexpr int COLS = DUAL ? 128 : 256;           // output columns of a pair tile
  constexpr uint32_t TMEM_COLS = 512;              // two accumulator stages of 256 tokens

  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * TC2_STAGES + 4 + 8];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag_s;
  __shared__ int tile_prefix[257];
  __shared__ int s_counts[256];

  volatile int* abort_flag = &abort_flag_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = (int)cluster_id_x(), npairs = (int)cluster_count_x();
  const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t full_bar = smem_u32(&bars[0]);                    // [TC2_STAGES]  used in the leader
  const uint32_t empty_bar = smem_u32(&bars[TC2_STAGES]);          // [TC2_STAGES]  in each CTA
  const uint32_t tfull_bar = smem_u32(&bars[2 * TC2_STAGES]);      // [2]           in each CTA
  const uint32_t tempty_bar = smem_u32(&bars[2 * TC2_STAGES + 2]); // [2]           used in the leader
  const uint32_t xfull_bar = smem_u32(&bars[2 * TC2_STAGES + 4]);  // [4]  SwiGLU: U is in the exchange buffer
  const uint32_t xempty_bar = smem_u32(&bars[2 * TC2_STAGES + 8]); // [4]  ... and has been read

  if (tid == 0) {
    abort_flag_s = 0;
    for (int s = 0; s < TC2_STAGES; ++s) { mbar_init(full_bar + 8 * s, 1); mbar_init(empty_bar + 8 * s, 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar + 8 * a, 1); mbar_init(tempty_bar + 8 * a, 16); }
    for (int x = 0; x < 4; ++x) { mbar_init(xfull_bar + 8 * x, 1); mbar_init(xempty_bar + 8 * x, 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  __syncwarp();
  cluster_sync_all();                 // both CTAs' barriers exist before any remote arrive
  grid_wait();
  if (warp == 2) {
    const int nc = (p.N + COLS - 1) / COLS;
    tile_prefix_warp(tile_prefix, s_counts, p.counts, p.E, lane, [&](int n_e) {
      const int n = min(n_e, p.M);
      return n > 0 ? nc * ((n - 1) / swap_tile_rows(n) + 1) : 0;
    });
  }
  tc_fence_before();
  __syncthreads();
  grid_release();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  const uint32_t leader_full = map_to_cta(full_bar, 0);
  const uint32_t leader_tempty = map_to_cta(tempty_bar, 0);

  if (warp == 0) {
    // ---- TMA producer (both CTAs) ---------------------------------------------------------------
    int e_cur = 0, stage = 0;
    uint32_t phase = 0;
    SwapTile t;
    bool ok = true;
    for (int tile = pair; ok && swap_tile(p, tile_prefix, s_counts, tile, e_cur, COLS, t); tile += npairs) {
      const int kb1 = p.two_k ? t.kblocks / 2 : t.kblocks;
      const int tr0 = t.t0 + (int)rank * (t.nt / 2), boxes = (t.nt / 2 + p.tok_box - 1) / p.tok_box;
      const uint32_t box_bytes = (uint32_t)p.tok_box * 128u;
      for (int kb = 0; kb < t.kblocks; ++kb) {
        ok = __all_sync(0xffffffffu, mbar_wait_cluster(empty_bar + 8 * stage, phase ^ 1u, abort_flag, p.wait_limit));
        if (!ok) break;
        if (elect_one()) {
          if (rank == 0) mbar_expect_tx(full_bar + 8 * stage, 2 * (2 * TC_BOX_BYTES + boxes * box_bytes));
          const uint32_t fb = leader_full + 8 * stage;
          const bool second = kb >= kb1;
          const int k0 = (second ? kb - kb1 : kb) * TC_BK;
          const uint32_t sa = tiles_base + stage * TC2_STAGE_BYTES, sb = sa + 2 * TC_BOX_BYTES;
          const CUtensorMap* ma = second ? &mapA1 : &mapA0;
          const CUtensorMap* mb = second ? &mapB1 : &mapB0;
          if (DUAL) {
            tma_load_3d_pair(sa, &mapA0, fb, k0, t.n0 + 64 * (int)rank, t.e);
            tma_load_3d_pair(sa + TC_BOX_BYTES, &mapA1, fb, k0, t.n0 + 64 * (int)rank, t.e);
          } else {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              const int n = t.n0 + 128 * (int)rank + 64 * j;
              if (A_MN) tma_load_3d_pair(sa + j * TC_BOX_BYTES, ma, fb, n, k0, t.e);
              else      tma_load_3d_pair(sa + j * TC_BOX_BYTES, ma, fb, k0, n, t.e);
            }
          }
          for (int i = 0; i < boxes; ++i) tma_load_3d_pair(sb + i * box_bytes, mb, fb, k0, tr0 + i * p.tok_box, t.e);
        }
        __syncwarp();
        if (++stage == TC2_STAGES) { stage = 0; phase ^= 1u; }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer (leader CTA only) --------------------------------------------------------------
    if (rank == 0) {
      int e_cur = 0, stage = 0, acc_stage = 0;
      uint32_t phase = 0, acc_phase = 0;
      SwapTile t;
      bool ok = true;
      constexpr uint32_t a_lbo = A_MN ? TC_BOX_BYTES : 16u, a_kstep = A_MN ? 2048u : 32u;
      for (int tile = pair; ok && swap_tile(p, tile_prefix, s_counts, tile, e_cur, COLS, t); tile += npairs) {
        ok = __all_sync(0xffffffffu, mbar_wait_cluster(tempty_bar + 8 * acc_stage, acc_phase ^ 1u, abort_flag, p.wait_limit));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc_stage * 256);
        const uint32_t id = idesc | ((uint32_t)(t.nt >> 3) << 17);
        for (int kb = 0; kb < t.kblocks; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait_cluster(full_bar + 8 * stage, phase, abort_flag, p.wait_limit));
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint32_t sa = tiles_base + stage * TC2_STAGE_BYTES, sb = sa + 2 * TC_BOX_BYTES;
#pragma unroll
            for (int kk = 0; kk < TC_BK / 16; ++kk)
              tc_mma_pair(d_tmem, make_smem_desc(sa + kk * a_kstep, a_lbo, 1024u), make_smem_desc(sb + kk * 32u, 16u, 1024u),
                          id, (kb > 0 || kk > 0) ? 1u : 0u);
            tc_commit_pair(empty_bar + 8 * stage);                       // frees the stage in both CTAs
            if (kb + 1 == t.kblocks) tc_commit_pair(tfull_bar + 8 * acc_stage);      // accumulators complete in both CTAs
          }
          __syncwarp();
          if (++stage == TC2_STAGES) { stage = 0; phase ^= 1u; }
        }
        if (++acc_stage == 2) { acc_stage = 0; acc_phase ^= 1u; }
      }
    }
  } else {
    // ---- epilogue warps (both CTAs, own 128 lanes) -----------------------------------------------------
    const int q = warp & 3, half = (warp - 2) >> 2;
    uint8_t* scratch = smem_raw + (tiles_base - smem_u32(smem_raw)) + TC2_STAGES * TC2_STAGE_BYTES + (warp - 2) * TC_SCRATCH_BYTES;
    const int x = 2 * half + (q & 1);               // SwiGLU: the exchange this warp takes part in
    const bool is_u = DUAL && q >= 2;
    float* xbuf = reinterpret_cast<float*>(smem_raw + (tiles_base - smem_u32(smem_raw)) + TC2_STAGES * TC2_STAGE_BYTES +
                                           8 * TC_SCRATCH_BYTES + x * TCS_XBUF_BYTES);
    uint32_t x_phase = 0;
    int e_cur = 0, acc_stage = 0;
    uint32_t acc_phase = 0;
    SwapTile t;
    bool ok = true;
    for (int tile = pair; ok && swap_tile(p, tile_prefix, s_counts, tile, e_cur, COLS, t); tile += npairs) {
      const int nb = DUAL ? t.n0 + 64 * (int)rank + 32 * (q & 1) : t.n0 + 128 * (int)rank + 32 * q;      // first column
      const bool live = nb < p.N;
      const long long row0 = (long long)t.e * p.M + t.t0;
      const int chunks = (t.nt + 31) / 32;
      const long long ob = row0 * p.N + nb;
      uint4 pg[4], pu[4];
      if (EPI == TC_EPI_DSWIGLU) {                   // G and U of the warp's part of the NEXT tile, towards L2
        SwapTile tn;
        int e_next = e_cur;
        if (swap_tile(p, tile_prefix, s_counts, tile + npairs, e_next, COLS, tn)) {
          const int nn = tn.n0 + 128 * (int)rank + 32 * q;
          for (int r = 32 * half + lane; nn < p.N && r < tn.nt; r += 64) {
            const long long o = ((long long)tn.e * p.M + tn.t0 + r) * p.N + nn;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p.in0 + o));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p.in1 + o));
          }
        }
      }
      if (EPI == TC_EPI_DSWIGLU && live && half < chunks) {      // the saved G and U of the first chunk
        const int nv = min(32, t.nt - 32 * half);
        load32_warp_issue(p.in0 + ob + (long long)(32 * half) * p.N, p.N, lane, nv, pg);
        load32_warp_issue(p.in1 + ob + (long long)(32 * half) * p.N, p.N, lane, nv, pu);
      }
      ok = __all_sync(0xffffffffu, mbar_wait_cluster(tfull_bar + 8 * acc_stage, acc_phase, abort_flag, p.wait_limit));
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + (uint32_t)(acc_stage * 256) + ((uint32_t)(32 * q) << 16);
      for (int c = half; c < chunks; c += 2) {
        const int nv = min(32, t.nt - 32 * c);                   // rows of this chunk (columns past nt hold nothing of use)
        const long long cb = ob + (long long)(32 * c) * p.N;
        __syncwarp();
        uint32_t r[32];
        tc_ld_block(taddr + 32 * c, r);
        tc_wait_ld();
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
        if (EPI == TC_EPI_SWIGLU) {
          if (is_u) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
              ok = __all_sync(0xffffffffu, mbar_wait(xempty_bar + 8 * x, x_phase ^ 1u, abort_flag, p.wait_limit));
              if (!ok) break;
#pragma unroll
              for (int j = 0; j < 16; ++j) xbuf[32 * j + lane] = v[16 * s + j];
              __syncwarp();
              if (lane == 0) mbar_arrive(xfull_bar + 8 * x);
              x_phase ^= 1u;
            }
            if (!ok) break;
            if (live) store_turned(scratch, lane, nv, p.out1 + cb, p.N, v);
          } else {
            float hv[32];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
              ok = __all_sync(0xffffffffu, mbar_wait(xfull_bar + 8 * x, x_phase, abort_flag, p.wait_limit));
              if (!ok) break;
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const float g = v[16 * s + j];
                hv[16 * s + j] = __fdividef(g, 1.0f + __expf(-g)) * xbuf[32 * j + lane];
              }
              __syncwarp();
              if (lane == 0) mbar_arrive(xempty_bar + 8 * x);
              x_phase ^= 1u;
            }
            if (!ok) break;
            if (live) {
              store_turned(scratch, lane, nv, p.out0 + cb, p.N, v);
              store_turned(scratch, lane, nv, p.out2 + cb, p.N, hv);
            }
          }
        } else if (EPI == TC_EPI_DSWIGLU) {
          if (live) {
            uint32_t gw[16], uw[16];
            float g[32];
            load_turned(scratch, lane, pg, gw);
            load_turned(scratch, lane, pu, uw);
            if (c + 2 < chunks) {
              const int nx = min(32, t.nt - 32 * (c + 2));
              load32_warp_issue(p.in0 + cb + 64ll * p.N, p.N, lane, nx, pg);
              load32_warp_issue(p.in1 + cb + 64ll * p.N, p.N, lane, nx, pu);
            }
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const int k = 4 * ((j & 15) >> 2) + 2 * (j >> 4) + ((j >> 1) & 1);      // value j is half (j & 1) of word k
              const float gj = __uint_as_float((j & 1) ? gw[k] & 0xffff0000u : gw[k] << 16);
              const float uj = __uint_as_float((j & 1) ? uw[k] & 0xffff0000u : uw[k] << 16);
              const float dh = v[j], sgm = __fdividef(1.0f, 1.0f + __expf(-gj));
              g[j] = dh * uj * sgm * (1.0f + gj * (1.0f - sgm));
              v[j] = dh * gj * sgm;
            }
            store_turned(scratch, lane, nv, p.out0 + cb, p.N, g);
            store_turned(scratch, lane, nv, p.out1 + cb, p.N, v);
          }
        } else if (live) {
          store_turned(scratch, lane, nv, p.out0 + cb, p.N, v);
          if (p.sc_out != nullptr)
            scatter_turned(scratch, lane, nv, p.sc_tok + row0 + 32 * c, p.sc_gate + row0 + 32 * c, p.sc_out + nb, p.sc_ld);
        }
      }
      if (!ok) break;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * acc_stage);
      if (++acc_stage == 2) { acc_stage = 0; acc_phase ^= 1u; }
      if (live && t.t0 + t.nt >= t.rows) {           // the expert's last tile: its pad rows, half of them per warp
        const int z0 = t.t0 + t.nt, z1 = min((t.rows + TC_BM - 1) / TC_BM * TC_BM, p.M);
        if (z0 < z1) {
          const int zm = z0 + (z1 - z0) / 2, a = half ? zm : z0, b = half ? z1 : zm;
          const long long eb = (long long)t.e * p.M * p.N + nb;
          if (EPI == TC_EPI_SWIGLU) {
            if (is_u) {
              zero_rows32(p.out1 + eb, p.N, a, b, lane);
            } else {
              zero_rows32(p.out0 + eb, p.N, a, b, lane);
              zero_rows32(p.out2 + eb, p.N, a, b, lane);
            }
          } else {
            zero_rows32(p.out0 + eb, p.N, a, b, lane);
            if (EPI == TC_EPI_DSWIGLU) zero_rows32(p.out1 + eb, p.N, a, b, lane);
          }
        }
      }
    }
  }

  // ---- teardown: neither CTA leaves while the other may still touch its barriers or memory -------
  __syncwarp();
  if (*abort_flag) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }
    if (tid == 0) atomicExch(&p.stats->error_word, 0x7c0b);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
  cluster_sync_all();                 // the next kernel's blocks may start on an SM as soon as its CTA is gone
}

// ---- weight gradients ------------------------------------------------------------------------------------
// dW2 = dO^T H, dW1g = dG^T Xp and dW1u = dU^T Xp of every expert in ONE launch: contractions over the expert's rows, both
// operands MN-major, CTA pairs on tiles of 256 x up to 256 (the last column tile has 128 columns where that is all that is
// left).  What bounds it: with many rows per expert the tensor pipe and the operands' way into the SMs; with few (one to
// four K blocks a tile) the stream of outputs to HBM.  For the latter the epilogue writes nothing itself: it packs 64
// columns of its 32 rows into a swizzled box in shared memory and hands that to TMA.  A tile's way through it is a chain
// of latencies all the same (in cycles: 1300 to 4400 for 128 columns of tensor memory while all warps read, 240 to release them, twice
// 700 for a box), so there are two sets of eight epilogue warps that take alternate tiles, one per accumulator stage.
// Measured, the three gradients: one launch each, warps turning 32 x 32 blocks and storing 64-byte row pieces; one launch,
// boxes, eight warps; this.  10 rows per expert (E 32, d 2048, h 4096) 500, 385, 292 us (5.5 TB/s of outputs); 112 rows (E 16,
// h 2816) 195, 176, 139; 512 rows (E 16, d 1024, h 2816) 147, 120, 121; 1024 rows (E 32, d 2048, h 1408) 486, 457, 449; 722 rows
// (E 64, d 4096, h 2048) 1880, 1815, 1767.  No gain: columns of tiles first, two or four boxes per warp; three stages: 15 % slower.
constexpr int WG_STAGES = 5;
constexpr uint32_t WG_STAGE_BYTES = 4 * TC_BOX_BYTES;        // per CTA: 128 columns of A, 128 of B, 64 rows each
constexpr uint32_t WG_BOX_BYTES = 32 * 128;                  // an output box: 32 rows of 128 bytes
constexpr int WG_EPI_WARPS = 16, WG_THREADS = 64 + 32 * WG_EPI_WARPS;
constexpr size_t WG_SMEM = WG_STAGES * WG_STAGE_BYTES + WG_EPI_WARPS * WG_BOX_BYTES + 1024;

struct WgradParams {
  int d, h, E;
  int nout;              // 3: dW2, dW1g, dW1u; 1: dW2 alone (dW1 gathers its rows elsewhere)
  int krows;             // rows of a K block: 64, or 16 or 32 where the capacity is no larger
  int out_f32;
  const int32_t* counts;
  etr_stats* stats;
  long long wait_limit;
  uint32_t idesc;        // without N
};
struct WgradMaps { CUtensorMap dO, H, dG, dU, Xp, W2, W1g, W1u; };
// The tiles of a pair, every npairs-th: of an expert those of dW2, then dW1g, then dW1u, row tiles first.
struct WgradTiles {
  int e, which, m0, n0, nt, M, N, rows;      // the current tile; nt: its columns, 128 or 256
  int in_e, per, step_e, step_i;
  __device__ __forceinline__ bool first(const WgradParams& p, const int* counts_s, int tile, int step) {
    per = ((p.d + 255) >> 8) * ((p.h + 255) >> 8);
    const int all = p.nout * per;
    e = tile / all; in_e = tile - e * all;
    step_e = step / all; step_i = step - step_e * all;
    return set(p, counts_s);
  }
  __device__ __forceinline__ bool next(const WgradParams& p, const int* counts_s) {
    e += step_e; in_e += step_i;
    if (in_e >= p.nout * per) { in_e -= p.nout * per; ++e; }
    return set(p, counts_s);
  }
  __device__ __forceinline__ bool set(const WgradParams& p, const int* counts_s) {
    if (e >= p.E) return false;
    which = (in_e >= per) + (in_e >= 2 * per);
    M = which ? p.h : p.d;
    N = which ? p.d : p.h;
    const int local = in_e - which * per, tm = (M + 255) >> 8, tn = local / tm;
    m0 = (local - tn * tm) * 256;
    n0 = tn * 256;
    nt = N - n0 > 128 ? 256 : 128;
    rows = counts_s[e];
    return true;
  }
};

__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar_cluster, int c0, int c1,
                                                 int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar_cluster), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
// 32 words of this lane's row (128 bytes) into the swizzled box at buf, then the whole box to (col, row, e) of the output.
__device__ __forceinline__ void wgrad_store_box(uint32_t buf, int lane, const uint32_t* w, const CUtensorMap* map, int col,
                                                int row, int e) {
  if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");      // the last box has been read
  __syncwarp();
#pragma unroll
  for (int c = 0; c < 8; ++c)
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(buf + lane * 128 + ((c ^ (lane & 7)) << 4)), "r"(w[4 * c]),
                 "r"(w[4 * c + 1]), "r"(w[4 * c + 2]), "r"(w[4 * c + 3]) : "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (lane == 0) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"(map), "r"(buf), "r"(col), "r"(row), "r"(e) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
}

__global__ void __launch_bounds__(WG_THREADS, 1)
tc_wgrad_pair_kernel(const __grid_constant__ WgradMaps maps, const WgradParams p) {
  constexpr uint32_t TMEM_COLS = 512;              // two accumulator stages
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * WG_STAGES + 4];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag_s;
  __shared__ int s_counts[256];

  volatile int* abort_flag = &abort_flag_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = (int)cluster_id_x(), npairs = (int)cluster_count_x();
  const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t full_bar = smem_u32(&bars[0]);                    // [WG_STAGES]  used in the leader
  const uint32_t empty_bar = smem_u32(&bars[WG_STAGES]);           // [WG_STAGES]  in each CTA
  const uint32_t tfull_bar = smem_u32(&bars[2 * WG_STAGES]);       // [2]          in each CTA
  const uint32_t tempty_bar = smem_u32(&bars[2 * WG_STAGES + 2]);  // [2]          used in the leader

  if (tid == 0) {
    abort_flag_s = 0;
    for (int s = 0; s < WG_STAGES; ++s) { mbar_init(full_bar + 8 * s, 1); mbar_init(empty_bar + 8 * s, 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar + 8 * a, 1); mbar_init(tempty_bar + 8 * a, 16); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  __syncwarp();
  cluster_sync_all();                 // both CTAs' barriers exist before any remote arrive
  grid_wait();
  for (int e = tid; e < p.E; e += WG_THREADS) s_counts[e] = p.counts[e];
  tc_fence_before();
  __syncthreads();
  grid_release();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  const uint32_t leader_full = map_to_cta(full_bar, 0);
  const uint32_t leader_tempty = map_to_cta(tempty_bar, 0);
  const uint32_t blk = (uint32_t)p.krows * 128u;   // bytes of 64 columns of a K block

  if (warp == 0) {
    // ---- TMA producer (both CTAs) ---------------------------------------------------------------
    int stage = 0;
    uint32_t phase = 0;
    WgradTiles t;
    bool ok = true;
    for (bool more = t.first(p, s_counts, pair, npairs); ok && more; more = t.next(p, s_counts)) {
      const CUtensorMap* ma = t.which == 0 ? &maps.dO : t.which == 1 ? &maps.dG : &maps.dU;
      const CUtensorMap* mb = t.which == 0 ? &maps.H : &maps.Xp;
      const int ca = (t.m0 + 128 * (int)rank) >> 6, cb = (t.n0 + (t.nt >> 1) * (int)rank) >> 6;      // in blocks of 64 columns
      for (int k0 = 0; k0 < t.rows; k0 += p.krows) {
        ok = __all_sync(0xffffffffu, mbar_wait_cluster(empty_bar + 8 * stage, phase ^ 1u, abort_flag, p.wait_limit));
        if (!ok) break;
        if (elect_one()) {
          if (rank == 0) mbar_expect_tx(full_bar + 8 * stage, 8 * blk);
          const uint32_t fb = leader_full + 8 * stage, sa = tiles_base + stage * WG_STAGE_BYTES;
          tma_load_4d_pair(sa, ma, fb, 0, k0, ca, t.e);
          tma_load_4d_pair(sa + 2 * TC_BOX_BYTES, mb, fb, 0, k0, cb, t.e);      // of a tile of 128 columns, half is not used
        }
        __syncwarp();
        if (++stage == WG_STAGES) { stage = 0; phase ^= 1u; }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer (leader CTA only) --------------------------------------------------------------
    if (rank == 0) {
      int stage = 0, acc_stage = 0;
      uint32_t phase = 0, acc_phase = 0;
      WgradTiles t;
      bool ok = true;
      for (bool more = t.first(p, s_counts, pair, npairs); ok && more; more = t.next(p, s_counts)) {
        if (t.rows == 0) continue;
        ok = __all_sync(0xffffffffu, mbar_wait_cluster(tempty_bar + 8 * acc_stage, acc_phase ^ 1u, abort_flag, p.wait_limit));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc_stage * 256);
        const uint32_t id = p.idesc | ((uint32_t)(t.nt >> 3) << 17);
        auto mma = [&](int kk, bool first) {
          const uint32_t sa = tiles_base + stage * WG_STAGE_BYTES;
          tc_mma_pair(d_tmem, make_smem_desc(sa + kk * 2048u, blk, 1024u),
                      make_smem_desc(sa + 2 * TC_BOX_BYTES + kk * 2048u, blk, 1024u), id, first ? 0u : 1u);
        };
        auto block = [&](int steps, bool first, bool last) {      // one K block; false: a wait ran out
          if (!__all_sync(0xffffffffu, mbar_wait_cluster(full_bar + 8 * stage, phase, abort_flag, p.wait_limit))) return false;
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < TC_BK / 16; ++kk)
              if (steps == TC_BK / 16 || kk < steps) mma(kk, first && kk == 0);
            tc_commit_pair(empty_bar + 8 * stage);                       // frees the stage in both CTAs
            if (last) tc_commit_pair(tfull_bar + 8 * acc_stage);         // accumulators complete in both CTAs
          }
          __syncwarp();
          if (++stage == WG_STAGES) { stage = 0; phase ^= 1u; }
          return true;
        };
        // The last K block is peeled off: it runs only the 16-row steps that hold rows in use (the others would add the
        // zeros of pad rows), and a test in the loop costs more than it saves.
        const int nloop = (t.rows - 1) / p.krows;
        if (p.krows == TC_BK) {
          for (int kb = 0; ok && kb < nloop; ++kb) ok = block(TC_BK / 16, kb == 0, false);
        } else {
          for (int kb = 0; ok && kb < nloop; ++kb) ok = block(p.krows / 16, kb == 0, false);
        }
        ok = ok && block((t.rows - nloop * p.krows + 15) >> 4, nloop == 0, true);
        if (!ok) break;
        if (++acc_stage == 2) { acc_stage = 0; acc_phase ^= 1u; }
      }
    }
  } else {
    // ---- epilogue warps (both CTAs, own 128 rows; 128 of the tile's columns each) -------------------------
    const int q = warp & 3, half = ((warp - 2) >> 2) & 1, mine = (warp - 2) >> 3;
    const uint32_t box = tiles_base + WG_STAGES * WG_STAGE_BYTES + (uint32_t)(warp - 2) * WG_BOX_BYTES;
    int turn = 0, empties = 0;                       // which set takes the next tile with rows, and without
    uint32_t acc_phase = 0;
    WgradTiles t;
    for (bool more = t.first(p, s_counts, pair, npairs); more; more = t.next(p, s_counts)) {
      const CUtensorMap* mo = t.which == 0 ? &maps.W2 : t.which == 1 ? &maps.W1g : &maps.W1u;
      const int row = t.m0 + 128 * (int)rank + 32 * q, col = t.n0 + 128 * half;
      int& whose = t.rows == 0 ? empties : turn;
      const bool own = whose == mine;
      whose ^= 1;
      if (!own) continue;
      const uint32_t taddr = tmem_base + (uint32_t)(mine * 256 + 128 * half) + ((uint32_t)(32 * q) << 16);
      if (t.rows > 0) {
        if (!__all_sync(0xffffffffu, mbar_wait_cluster(tfull_bar + 8 * mine, acc_phase, abort_flag, p.wait_limit))) break;
        acc_phase ^= 1u;
        tc_fence_after();
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {                  // 64 columns at a time
        uint32_t r[2][32];
        if (t.rows == 0) {                           // nothing to contract: zeros
#pragma unroll
          for (int i = 0; i < 32; ++i) r[0][i] = r[1][i] = 0u;
        } else {
          tc_ld32(taddr + 64 * c, r[0]);
          tc_ld32(taddr + 64 * c + 32, r[1]);
          tc_wait_ld();
          if (c == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * mine);
          }
        }
        if (row >= t.M || col + 64 * c >= t.N) continue;
        if (p.out_f32) {
#pragma unroll
          for (int u = 0; u < 2; ++u) wgrad_store_box(box, lane, r[u], mo, col + 64 * c + 32 * u, row, t.e);
        } else {
          uint32_t w[32];
#pragma unroll
          for (int i = 0; i < 32; ++i)
            w[i] = pack_bf16(__uint_as_float(r[i >> 4][2 * (i & 15)]), __uint_as_float(r[i >> 4][2 * (i & 15) + 1]));
          wgrad_store_box(box, lane, w, mo, col + 64 * c, row, t.e);
        }
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");      // every box is in the output
  }

  // ---- teardown: neither CTA leaves while the other may still touch its barriers or memory -------
  __syncwarp();
  if (*abort_flag) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }
    if (tid == 0) atomicExch(&p.stats->error_word, 0x7c0c);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
  cluster_sync_all();                 // the next kernel's blocks may start on an SM as soon as its CTA is gone
}

// ---- host side --------------------------------------------------------------------------------------
// Row-major bf16 tensor [E, rows, cols] as a 3-D map (cols, rows, E), boxes of 64 columns x box_rows, 128-byte swizzle.
static etr_status make_map(CUtensorMap* m, const void* base, int cols, int rows, int E, int box_rows = 64) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return ETR_ERR_CUDA;
  const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)E};
  const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)cols * 2 * (cuuint64_t)rows};
  const cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
                        estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? ETR_OK : ETR_ERR_CUDA;
}

// Row-major bf16 token matrix [T, d] as a 2-D map (d, T) with a one-row box of 64 columns, for row
// gathers; rows at or past T read as zeros.
static etr_status make_gather_map(CUtensorMap* m, const void* base, int cols, int rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return ETR_ERR_CUDA;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  const cuuint32_t box[2] = {64, 1};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                        estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? ETR_OK : ETR_ERR_CUDA;
}

// Row-major bf16 tensor [E, rows, cols] in boxes of 32 rows x 32 columns, 64-byte swizzle.
static etr_status make_map_chunks(CUtensorMap* m, const void* base, int cols, int rows, int E) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return ETR_ERR_CUDA;
  const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)E};
  const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)cols * 2 * (cuuint64_t)rows};
  const cuuint32_t box[3] = {32, 32, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? ETR_OK : ETR_ERR_CUDA;
}

static uint32_t make_idesc(int a_mn, int b_mn, int n, int m_instr = TC_BM) {
  uint32_t d = 0;
  d |= 1u << 4;                     // accumulator fp32
  d |= 1u << 7;                     // A bf16
  d |= 1u << 10;                    // B bf16
  d |= (uint32_t)(a_mn ? 1 : 0) << 15;
  d |= (uint32_t)(b_mn ? 1 : 0) << 16;
  d |= (uint32_t)(n >> 3) << 17;
  d |= (uint32_t)(m_instr >> 4) << 24;
  return d;
}

static int sm_count() { return current_sm_count(); }

template <int BN, int EPI>
static etr_status tc_launch(const char* name, const CUtensorMap& a0, const CUtensorMap& a1,
                            const CUtensorMap& b0, const CUtensorMap& b1, TcParams p, int max_tiles,
                            cudaStream_t st) {
  constexpr size_t smem = (size_t)TC_STAGES * (2 + BN / 64) * TC_BOX_BYTES + 1024 + 8 * TC_SCRATCH_BYTES;
  auto k = tc_grouped_gemm_kernel<BN, EPI>;
  static std::atomic<unsigned long long> attr_done{0};      // one bit per device
  if (!ensure_dyn_smem(k, smem, attr_done)) return ETR_ERR_CUDA;
  p.idesc = make_idesc(p.a_mn, p.b_mn, BN);
  const int grid = max_tiles < sm_count() ? (max_tiles < 1 ? 1 : max_tiles) : sm_count();
  ETR_TIME_BEGIN(name);
  launch_kernel(k, grid, TC_THREADS, smem, st, 1, a0, a1, b0, b1, p);
  ETR_LAUNCH_CHECK();
  return ETR_OK;
}

template <int EPI, int GATHER, int CFG>
static etr_status tc_launch_pair_cfg(const char* name, const CUtensorMap& a0, const CUtensorMap& a1,
                                 const CUtensorMap& b0, const CUtensorMap& b1, TcParams p, int max_tiles,
                                 cudaStream_t st) {
  constexpr size_t smem = PairRing<EPI>::TAIL + sizeof(PairShared);
  static_assert(smem <= 232448 && 2 * PairRing<EPI>::STAGES + 4 + (EPI == TC_EPI_DSWIGLU_BOX ? 16 : 0) <= 30, "shared memory of a CTA");
  auto k = tc_grouped_gemm_pair_kernel<EPI, GATHER, CFG>;
  static std::atomic<unsigned long long> attr_done{0};      // one bit per device
  if (!ensure_dyn_smem(k, smem, attr_done)) return ETR_ERR_CUDA;
  p.idesc = make_idesc(p.a_mn, p.b_mn, 256, 256);
  DswMaps em;
  memset(&em, 0, sizeof(em));
  if (EPI == TC_EPI_DSWIGLU_BOX) {
    ETR_TRY(make_map_chunks(&em.G, p.in0, p.N, p.M, p.E));
    ETR_TRY(make_map_chunks(&em.U, p.in1, p.N, p.M, p.E));
    ETR_TRY(make_map_chunks(&em.dG, p.out0, p.N, p.M, p.E));
    ETR_TRY(make_map_chunks(&em.dU, p.out1, p.N, p.M, p.E));
  }
  const int pairs_max = sm_count() / 2;
  const int pairs = max_tiles < pairs_max ? (max_tiles < 1 ? 1 : max_tiles) : pairs_max;
  ETR_TIME_BEGIN(name);
  launch_kernel(k, 2 * pairs, TC_THREADS, smem, st, 2, a0, a1, b0, b1, p, em);
  ETR_LAUNCH_CHECK();
  return ETR_OK;
}

template <int EPI, int GATHER, int CFG>
static etr_status tc_launch_pair_wide_cfg(const char* name, const CUtensorMap& a0, const CUtensorMap& a1,
                                      const CUtensorMap& b0, const CUtensorMap& b1, TcParams p, int max_tiles,
                                      cudaStream_t st) {
  constexpr size_t smem = (size_t)TCW_STAGES * TCW_STAGE_BYTES + 1024 + 8 * TC_SCRATCH_BYTES;
  auto k = tc_grouped_gemm_pair_wide_kernel<EPI, GATHER, CFG>;
  static std::atomic<unsigned long long> attr_done{0};      // one bit per device
  if (!ensure_dyn_smem(k, smem, attr_done)) return ETR_ERR_CUDA;
  p.idesc = make_idesc(p.a_mn, p.b_mn, 256, 256);
  const int pairs_max = sm_count() / 2;
  const int pairs = max_tiles < pairs_max ? (max_tiles < 1 ? 1 : max_tiles) : pairs_max;
  ETR_TIME_BEGIN(name);
  launch_kernel(k, 2 * pairs, TC_THREADS, smem, st, 2, a0, a1, b0, b1, p);
  ETR_LAUNCH_CHECK();
  return ETR_OK;
}


// An instantiation for each set of operand modes that an epilogue is used with: one of SwiGLU and its derivative; of plain
// stores the down GEMM, dXp, and weight gradients (of gathered rows in the pair form, forced by gemm_impl in the wide one).
static int tc_cfg(const TcParams& p) { return (p.a_mn ? 1 : 0) | (p.b_mn ? 2 : 0) | (p.dual_b ? 4 : 0) | (p.k1_blocks > 0 ? 8 : 0); }
template <int EPI, int GATHER>
static etr_status tc_launch_pair(const char* name, const CUtensorMap& a0, const CUtensorMap& a1,
                                 const CUtensorMap& b0, const CUtensorMap& b1, const TcParams& p, int max_tiles,
                                 cudaStream_t st) {
  constexpr int C0 = EPI == TC_EPI_SWIGLU ? 4 : EPI != TC_EPI_STORE ? 2 : GATHER == 2 ? 3 : 0;
  constexpr int C1 = EPI == TC_EPI_STORE && GATHER == 0 ? 10 : C0;
  const int cfg = tc_cfg(p);
  if (cfg == C0) return tc_launch_pair_cfg<EPI, GATHER, C0>(name, a0, a1, b0, b1, p, max_tiles, st);
  if (cfg == C1) return tc_launch_pair_cfg<EPI, GATHER, C1>(name, a0, a1, b0, b1, p, max_tiles, st);
  return ETR_ERR_UNSUPPORTED;
}
template <int EPI, int GATHER>
static etr_status tc_launch_pair_wide(const char* name, const CUtensorMap& a0, const CUtensorMap& a1,
                                      const CUtensorMap& b0, const CUtensorMap& b1, const TcParams& p, int max_tiles,
                                      cudaStream_t st) {
  constexpr int C0 = EPI == TC_EPI_SWIGLU ? 4 : EPI != TC_EPI_STORE ? 2 : 0;
  constexpr int C1 = EPI == TC_EPI_STORE ? 10 : C0, C2 = EPI == TC_EPI_STORE ? 3 : C0;
  const int cfg = tc_cfg(p);
  if (cfg == C0) return tc_launch_pair_wide_cfg<EPI, GATHER, C0>(name, a0, a1, b0, b1, p, max_tiles, st);
  if (cfg == C1) return tc_launch_pair_wide_cfg<EPI, GATHER, C1>(name, a0, a1, b0, b1, p, max_tiles, st);
  if (cfg == C2) return tc_launch_pair_wide_cfg<EPI, GATHER, C2>(name, a0, a1, b0, b1, p, max_tiles, st);
  return ETR_ERR_UNSUPPORTED;
}

// The three forms of one contraction; max_tiles is an upper bound counted in 128-row tiles of one
// column tile (it only caps the grid for small problems).
enum TcForm { TC_FORM_SINGLE, TC_FORM_PAIR, TC_FORM_PAIR_WIDE };

// Which form runs a contraction that the exchanged form (use_swap) does not take.  A forced gemm_impl decides alone.
// AUTO: weight gradients (short contractions over the expert's rows, large outputs) and the SwiGLU derivative (its epilogue
// also fetches G and U) on 256 x 256 pair tiles.  Plain stores come here with fewer than three rounds of pair tiles:
// 128-row tiles on single CTAs balance better and pad the expert's rows to 128 instead of 256.  SwiGLU: pair tiles; with
// gathered rows (fuse_dispatch), which the exchanged form has no producer for, the wide form where its saving in operand
// traffic outweighs its exposed epilogue, i.e. at 48 K blocks or more and four rounds of wide tiles per CTA pair.
static TcForm tc_form_of(const etr_config* c, int epi, const TcParams& p) {
  if (p.gather) {      // the pair kernels fetch gathered rows; wide only where it is chosen anyway
    if (c->gemm_impl == ETR_GEMM_TCGEN05_2CTA_WIDE && p.gather == 1) return TC_FORM_PAIR_WIDE;
    if (c->gemm_impl != ETR_GEMM_AUTO || p.gather == 2) return TC_FORM_PAIR;
  }
  if (c->gemm_impl == ETR_GEMM_TCGEN05) return TC_FORM_SINGLE;
  if (c->gemm_impl == ETR_GEMM_TCGEN05_2CTA) return TC_FORM_PAIR;
  if (c->gemm_impl == ETR_GEMM_TCGEN05_2CTA_WIDE) return TC_FORM_PAIR_WIDE;
  if (p.dyn != TC_DYN_M || epi == TC_EPI_DSWIGLU) return TC_FORM_PAIR;
  if (epi == TC_EPI_STORE) return TC_FORM_SINGLE;
  const long long wide_tiles = (long long)p.E * ceil_div(p.M, 256) * ceil_div(p.N, 256);
  return ceil_div(p.K, TC_BK) >= 48 && wide_tiles >= 4ll * (sm_count() / 2) ? TC_FORM_PAIR_WIDE : TC_FORM_PAIR;
}
template <int EPI>
static etr_status tc_run(TcForm form, const char* name, const CUtensorMap& a0, const CUtensorMap& a1,
                         const CUtensorMap& b0, const CUtensorMap& b1, const TcParams& p, int max_tiles,
                         cudaStream_t st) {
  // gathered operands exist for the SwiGLU GEMM (A rows) and the plain-store weight gradients (K rows)
  if (form == TC_FORM_PAIR_WIDE) {
    if (EPI == TC_EPI_SWIGLU && p.gather == 1)
      return tc_launch_pair_wide<EPI, EPI == TC_EPI_SWIGLU ? 1 : 0>(name, a0, a1, b0, b1, p, (max_tiles + 1) / 2, st);
    if (p.gather) return ETR_ERR_UNSUPPORTED;
    return tc_launch_pair_wide<EPI, 0>(name, a0, a1, b0, b1, p, (max_tiles + 1) / 2, st);
  }
  if (form == TC_FORM_PAIR) {
    if (EPI == TC_EPI_SWIGLU && p.gather == 1)
      return tc_launch_pair<EPI, EPI == TC_EPI_SWIGLU ? 1 : 0>(name, a0, a1, b0, b1, p, (max_tiles + 1) / 2, st);
    if (EPI == TC_EPI_STORE && p.gather == 2)
      return tc_launch_pair<EPI, EPI == TC_EPI_STORE ? 2 : 0>(name, a0, a1, b0, b1, p, (max_tiles + 1) / 2, st);
    if (p.gather) return ETR_ERR_UNSUPPORTED;
    if (EPI == TC_EPI_DSWIGLU && p.K < DSW_BOX_MAX_K)
      return tc_launch_pair<EPI == TC_EPI_DSWIGLU ? TC_EPI_DSWIGLU_BOX : EPI, 0>(name, a0, a1, b0, b1, p, (max_tiles + 1) / 2, st);
    return tc_launch_pair<EPI, 0>(name, a0, a1, b0, b1, p, (max_tiles + 1) / 2, st);
  }
  if (p.gather) return ETR_ERR_UNSUPPORTED;
  return tc_launch<256, EPI>(name, a0, a1, b0, b1, p, max_tiles, st);
}

// ---- exchanged operands: host side ----------------------------------------------------------------------
// Rows of a token box: half of a tile's tokens at most, so that a layer with few rows per expert fetches few.
static int swap_tok_box(const etr_config* c) {
  const int half = std::min(64, ceil_div(std::min(c->capacity, 256), 16) * 8);
  return half <= 8 ? 8 : half <= 16 ? 16 : half <= 32 ? 32 : 64;
}
// Where the exchanged form runs (gemm_impl AUTO; the other forms otherwise).  Measured against the form that
// tc_form_of takes, same box, in us:
//   capacity <= 192: a 256-row tile would be padding by a quarter or more.  8 rows per expert (E 13, d 1216,
//     h 6144): SwiGLU 92 -> 86, down 56 -> 48, derivative 80 -> 52, dXp 95 -> 75.
//   plain stores with at least three rounds of tiles: down 153 -> 139 and dXp 258 -> 244 at 1024 rows (E 32, d 2048,
//     h 1408), 147 -> 127 and 248 -> 223 at 769 rows of 1280, 656 -> 582 and 1183 -> 1117 at 717 rows (E 64, d 4096,
//     h 2048).  With fewer rounds the last one weighs more than the padding saved: 54 -> 59 and 91 -> 99 at 512
//     rows (E 16, d 1024, h 2816; 2.2 rounds).  (Tiles of 128 tokens there: 64 and 109.)
//   the fused epilogues are longer here (an exchange, a transposed read), so they need a longer contraction:
//     SwiGLU from K = 2048 (365 -> 348 at E 128, d 2048, h 768; 97 -> 105 at d 1024), its derivative from
//     K = 4096 (702 -> 668 at d 4096; 183 -> 219 at d 2048).  Between the measured lines (E 32, h 1408): SwiGLU at d 1536
//     222 -> 228 with 1024 rows, 119 -> 121 with 512, 213 -> 203 with 769 of 1280, 113 -> 103 with 300 of 1024;
//     derivative at d 3072 278 -> 281, 158 -> 162, 269 -> 236, 152 -> 130.  So at the line the two forms are even on full
//     buffers, and rows in use well below the capacity, which the host does not know, favour the exchanged form.
static bool use_swap(const etr_config* c, int epi) {
  if (c->gemm_impl != ETR_GEMM_AUTO) return false;
  if (c->capacity <= 192) return true;
  if (epi == TC_EPI_SWIGLU) return c->d >= 2048;
  if (epi == TC_EPI_DSWIGLU) return c->d >= 4096;
  return (long long)c->E * ceil_div(c->capacity, 256) * ceil_div(c->d, 256) >= 3 * (sm_count() / 2);
}
static SwapParams swap_params(const etr_config* c, const etr_route* rt, etr_stats* stats) {
  SwapParams p = {};
  p.M = c_stride_of(c); p.E = c->E; p.tok_box = swap_tok_box(c); p.counts = rt->counts; p.stats = stats;
  p.wait_limit = c->wait_limit_cycles > 0 ? (long long)c->wait_limit_cycles : TC_WAIT_LIMIT_CYCLES;
  return p;
}
template <int EPI, bool A_MN>
static etr_status swap_launch(const char* name, const CUtensorMap& a0, const CUtensorMap& a1, const CUtensorMap& b0,
                              const CUtensorMap& b1, const SwapParams& p, cudaStream_t st) {
  constexpr size_t smem = (size_t)TC2_STAGES * TC2_STAGE_BYTES + 1024 + 8 * TC_SCRATCH_BYTES + 4 * TCS_XBUF_BYTES;
  auto k = tc_grouped_gemm_swap_kernel<EPI, A_MN>;
  static std::atomic<unsigned long long> attr_done{0};      // one bit per device
  if (!ensure_dyn_smem(k, smem, attr_done)) return ETR_ERR_CUDA;
  const long long tiles = (long long)p.E * ceil_div(p.M, 256) * ceil_div(p.N, EPI == TC_EPI_SWIGLU ? 128 : 256);
  const int pairs = (int)std::max(1ll, std::min(tiles, (long long)(sm_count() / 2)));
  ETR_TIME_BEGIN(name);
  launch_kernel(k, 2 * pairs, TC_THREADS, smem, st, 2, a0, a1, b0, b1, p, make_idesc(A_MN, 0, 0, 256));
  ETR_LAUNCH_CHECK();
  return ETR_OK;
}

// ---- weight gradients: host side ------------------------------------------------------------------------
// Row-major bf16 tensor [E, rows, cols] as a 4-D map (64 columns, rows, blocks of 64 columns, E): a box of 64 columns x
// box_rows x 2 blocks is 128 columns, each block of 64 with its 128-byte swizzle.  cols is a multiple of 64.
static etr_status make_map_blocks(CUtensorMap* m, const void* base, int cols, int rows, int E, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return ETR_ERR_CUDA;
  const cuuint64_t dims[4] = {64, (cuuint64_t)rows, (cuuint64_t)(cols / 64), (cuuint64_t)E};
  const cuuint64_t strides[3] = {(cuuint64_t)cols * 2, 128, (cuuint64_t)cols * 2 * (cuuint64_t)rows};
  const cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 2, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? ETR_OK : ETR_ERR_CUDA;
}
// Row-major output [E, rows, cols], bf16 or fp32, stored in boxes of 128 bytes x 32 rows.
static etr_status make_map_out(CUtensorMap* m, void* base, int cols, int rows, int E, bool f32) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return ETR_ERR_CUDA;
  const cuuint64_t eb = f32 ? 4 : 2;
  const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)E};
  const cuuint64_t strides[2] = {cols * eb, cols * eb * (cuuint64_t)rows};
  const cuuint32_t box[3] = {f32 ? 32u : 64u, 32, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides,
                        box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? ETR_OK : ETR_ERR_CUDA;
}
// Xp == nullptr: dW2 alone.
static etr_status wgrad_launch(const etr_config* c, const etr_route* rt, const void* dO, const void* Xp, const void* H,
                               const void* dG, const void* dU, void* dW1g, void* dW1u, void* dW2, etr_stats* stats,
                               cudaStream_t st) {
  const int d = c->d, h = c->h, Cs = c_stride_of(c), E = c->E;
  WgradParams p = {};
  p.d = d; p.h = h; p.E = E; p.nout = Xp ? 3 : 1;
  p.krows = c->capacity <= 16 ? 16 : c->capacity <= 32 ? 32 : TC_BK;      // the rows behind are not even fetched
  p.out_f32 = c->grad_fp32 != 0;
  p.counts = rt->counts; p.stats = stats;
  p.wait_limit = c->wait_limit_cycles > 0 ? (long long)c->wait_limit_cycles : TC_WAIT_LIMIT_CYCLES;
  p.idesc = make_idesc(1, 1, 0, 256);
  WgradMaps m;
  ETR_TRY(make_map_blocks(&m.dO, dO, d, Cs, E, p.krows));
  ETR_TRY(make_map_blocks(&m.H, H, h, Cs, E, p.krows));
  ETR_TRY(make_map_out(&m.W2, dW2, h, d, E, p.out_f32));
  m.dG = m.dU = m.Xp = m.dO; m.W1g = m.W1u = m.W2;
  if (Xp) {
    ETR_TRY(make_map_blocks(&m.dG, dG, h, Cs, E, p.krows));
    ETR_TRY(make_map_blocks(&m.dU, dU, h, Cs, E, p.krows));
    ETR_TRY(make_map_blocks(&m.Xp, Xp, d, Cs, E, p.krows));
    ETR_TRY(make_map_out(&m.W1g, dW1g, d, h, E, p.out_f32));
    ETR_TRY(make_map_out(&m.W1u, dW1u, d, h, E, p.out_f32));
  }
  static std::atomic<unsigned long long> attr_done{0};      // one bit per device
  if (!ensure_dyn_smem(tc_wgrad_pair_kernel, WG_SMEM, attr_done)) return ETR_ERR_CUDA;
  const long long tiles = (long long)E * p.nout * ceil_div(d, 256) * ceil_div(h, 256);
  const int pairs = (int)std::min(tiles, (long long)(sm_count() / 2));
  ETR_TIME_BEGIN("tc_gemm_dw");
  launch_kernel(tc_wgrad_pair_kernel, 2 * pairs, WG_THREADS, WG_SMEM, st, 2, m, p);
  ETR_LAUNCH_CHECK();
  return ETR_OK;
}

static TcParams tc_params(const etr_config* c) {
  TcParams p = {};
  p.wait_limit = c->wait_limit_cycles > 0 ? (long long)c->wait_limit_cycles : TC_WAIT_LIMIT_CYCLES;
  return p;
}

size_t tc_workspace_bytes(const etr_config*) { return 0; }
bool tc_available() { return true; }

etr_status tc_ffn_forward(const etr_config* c, const etr_route* rt, const void* Xp, const void* Xtok, const void* W1g,
                          const void* W1u, const void* W2, void* G, void* U, void* H, void* O,
                          etr_stats* stats, void*, void* Y_top1, cudaStream_t st) {
  const int d = c->d, h = c->h, Cs = c_stride_of(c), E = c->E;
  CUtensorMap mXp, mW1g, mW1u, mW2, mH;
  if (Xtok) ETR_TRY(make_gather_map(&mXp, Xtok, d, c->T));
  else ETR_TRY(make_map(&mXp, Xp, d, Cs, E));
  ETR_TRY(make_map(&mW1g, W1g, d, h, E));
  ETR_TRY(make_map(&mW1u, W1u, d, h, E));
  ETR_TRY(make_map(&mW2, W2, h, d, E));
  ETR_TRY(make_map(&mH, H, h, Cs, E));
  const int mt = Cs / TC_BM;
  // G, U, H = SwiGLU(Xp W1g^T, Xp W1u^T)
  if (!Xtok && use_swap(c, TC_EPI_SWIGLU)) {
    SwapParams p = swap_params(c, rt, stats);
    ETR_TRY(make_map(&mXp, Xp, d, Cs, E, p.tok_box));
    p.N = h; p.K = d;
    p.out0 = (__nv_bfloat16*)G; p.out1 = (__nv_bfloat16*)U; p.out2 = (__nv_bfloat16*)H;
    ETR_TRY((swap_launch<TC_EPI_SWIGLU, false>("tc_gemm_swiglu", mW1g, mW1u, mXp, mXp, p, st)));
  } else {
    TcParams p = tc_params(c);
    if (Xtok) { p.gather = 1; p.gather_ld = Cs; p.gather_oob = c->T; p.gather_idx = rt->slot_token; }
    p.dual_b = 1; p.M = Cs; p.N = h; p.K = d; p.dyn = TC_DYN_M; p.E = E; p.counts = rt->counts;
    p.out0 = (__nv_bfloat16*)G; p.out1 = (__nv_bfloat16*)U; p.out2 = (__nv_bfloat16*)H;
    p.out_bs = (long long)Cs * h; p.ld_out = h; p.stats = stats;
    ETR_TRY((tc_run<TC_EPI_SWIGLU>(tc_form_of(c, TC_EPI_SWIGLU, p), "tc_gemm_swiglu", mXp, mXp, mW1g, mW1u, p,
                                           E * mt * ceil_div(h, 128), st)));
  }
  // O = H W2^T.  Y_top1 (Top-1): the combine in this epilogue (the caller has zeroed the rows of unrouted tokens)
  if (use_swap(c, TC_EPI_STORE)) {
    SwapParams p = swap_params(c, rt, stats);
    ETR_TRY(make_map(&mH, H, h, Cs, E, p.tok_box));
    p.N = d; p.K = h; p.out0 = (__nv_bfloat16*)O;
    if (Y_top1) { p.sc_tok = rt->slot_token; p.sc_gate = rt->gate; p.sc_out = (__nv_bfloat16*)Y_top1; p.sc_ld = d; }
    ETR_TRY((swap_launch<TC_EPI_STORE, false>("tc_gemm_down", mW2, mW2, mH, mH, p, st)));
  } else {
    TcParams p = tc_params(c);
    p.M = Cs; p.N = d; p.K = h; p.dyn = TC_DYN_M; p.E = E; p.counts = rt->counts;
    p.out0 = (__nv_bfloat16*)O; p.out_bs = (long long)Cs * d; p.ld_out = d; p.stats = stats;
    if (Y_top1) {
      p.sc_tok = rt->slot_token; p.sc_gate = rt->gate; p.sc_out = (__nv_bfloat16*)Y_top1; p.sc_ld = d;
    }
    ETR_TRY((tc_run<TC_EPI_STORE>(tc_form_of(c, TC_EPI_STORE, p), "tc_gemm_down", mH, mH, mW2, mW2, p, E * mt * ceil_div(d, 256), st)));
  }
  return ETR_OK;
}

etr_status tc_ffn_backward(const etr_config* c, const etr_route* rt, const void* dO, const void* Xp,
                           const void* Xtok, const void* G, const void* U, const void* H, const void* W1g,
                           const void* W1u, const void* W2, void* dG, void* dU, void* dXp, void* dW1g,
                           void* dW1u, void* dW2, etr_stats* stats, void*, cudaStream_t st) {
  const int d = c->d, h = c->h, Cs = c_stride_of(c), E = c->E;
  CUtensorMap mdO, mXp, mH, mdG, mdU, mW1g, mW1u, mW2;
  ETR_TRY(make_map(&mdO, dO, d, Cs, E));
  if (Xtok) ETR_TRY(make_gather_map(&mXp, Xtok, d, c->T));
  else ETR_TRY(make_map(&mXp, Xp, d, Cs, E));
  ETR_TRY(make_map(&mH, H, h, Cs, E));
  ETR_TRY(make_map(&mdG, dG, h, Cs, E));
  ETR_TRY(make_map(&mdU, dU, h, Cs, E));
  ETR_TRY(make_map(&mW1g, W1g, d, h, E));
  ETR_TRY(make_map(&mW1u, W1u, d, h, E));
  ETR_TRY(make_map(&mW2, W2, h, d, E));
  const int mt = Cs / TC_BM;
  // dH = dO W2 (W2 read with its output index contiguous), then dG, dU
  if (use_swap(c, TC_EPI_DSWIGLU)) {
    SwapParams p = swap_params(c, rt, stats);
    CUtensorMap t;
    ETR_TRY(make_map(&t, dO, d, Cs, E, p.tok_box));
    p.N = h; p.K = d;
    p.out0 = (__nv_bfloat16*)dG; p.out1 = (__nv_bfloat16*)dU;
    p.in0 = (const __nv_bfloat16*)G; p.in1 = (const __nv_bfloat16*)U;
    ETR_TRY((swap_launch<TC_EPI_DSWIGLU, true>("tc_gemm_dswiglu", mW2, mW2, t, t, p, st)));
  } else {
    TcParams p = tc_params(c);
    p.b_mn = 1; p.M = Cs; p.N = h; p.K = d; p.dyn = TC_DYN_M; p.E = E; p.counts = rt->counts;
    p.out0 = (__nv_bfloat16*)dG; p.out1 = (__nv_bfloat16*)dU;
    p.in0 = (const __nv_bfloat16*)G; p.in1 = (const __nv_bfloat16*)U;
    p.out_bs = (long long)Cs * h; p.ld_out = h; p.stats = stats;
    ETR_TRY((tc_run<TC_EPI_DSWIGLU>(tc_form_of(c, TC_EPI_DSWIGLU, p), "tc_gemm_dswiglu", mdO, mdO, mW2, mW2, p,
                                            E * mt * ceil_div(h, 256), st)));
  }
  // dXp = dG W1g + dU W1u: one contraction over 2h
  if (use_swap(c, TC_EPI_STORE)) {
    SwapParams p = swap_params(c, rt, stats);
    CUtensorMap tg, tu;
    ETR_TRY(make_map(&tg, dG, h, Cs, E, p.tok_box));
    ETR_TRY(make_map(&tu, dU, h, Cs, E, p.tok_box));
    p.N = d; p.K = h; p.two_k = 1; p.out0 = (__nv_bfloat16*)dXp;
    ETR_TRY((swap_launch<TC_EPI_STORE, true>("tc_gemm_dxp", mW1g, mW1u, tg, tu, p, st)));
  } else {
    TcParams p = tc_params(c);
    p.b_mn = 1; p.k1_blocks = ceil_div(h, TC_BK); p.M = Cs; p.N = d; p.K = 2 * h; p.dyn = TC_DYN_M;
    p.E = E; p.counts = rt->counts;
    p.out0 = (__nv_bfloat16*)dXp; p.out_bs = (long long)Cs * d; p.ld_out = d; p.stats = stats;
    ETR_TRY((tc_run<TC_EPI_STORE>(tc_form_of(c, TC_EPI_STORE, p), "tc_gemm_dxp", mdG, mdU, mW1g, mW1u, p,
                                          E * mt * ceil_div(d, 256), st)));
  }
  // Weight gradients, contractions over the expert's rows.  The pair form takes all three in one launch; the forms that
  // gemm_impl forces, and rows gathered from X (fuse_dispatch), run them one by one.
  TcParams dw2 = tc_params(c);
  dw2.a_mn = 1; dw2.b_mn = 1; dw2.M = d; dw2.N = h; dw2.dyn = TC_DYN_K; dw2.E = E; dw2.counts = rt->counts;
  dw2.out0 = (__nv_bfloat16*)dW2; dw2.out_bs = (long long)d * h; dw2.ld_out = h; dw2.stats = stats;
  dw2.out_f32 = c->grad_fp32 != 0;
  const TcForm form = tc_form_of(c, TC_EPI_STORE, dw2);
  if (form == TC_FORM_PAIR) {
    ETR_TRY(wgrad_launch(c, rt, dO, Xtok ? nullptr : Xp, H, dG, dU, dW1g, dW1u, dW2, stats, st));
    if (!Xtok) return ETR_OK;
  } else {
    ETR_TRY((tc_run<TC_EPI_STORE>(form, "tc_gemm_dw2", mdO, mdO, mH, mH, dw2, E * ceil_div(d, TC_BM) * ceil_div(h, 256), st)));
  }
  for (int which = 0; which < 2; ++which) {  // dW1g = dG^T Xp, dW1u = dU^T Xp
    TcParams p = dw2;
    p.M = h; p.N = d; p.ld_out = d; p.out0 = (__nv_bfloat16*)(which ? dW1u : dW1g);
    if (Xtok) { p.gather = 2; p.gather_ld = Cs; p.gather_oob = c->T; p.gather_idx = rt->slot_token; }
    const CUtensorMap& ma = which ? mdU : mdG;
    ETR_TRY((tc_run<TC_EPI_STORE>(tc_form_of(c, TC_EPI_STORE, p), "tc_gemm_dw1", ma, ma, mXp, mXp, p,
                                          E * ceil_div(h, TC_BM) * ceil_div(d, 256), st)));
  }
  return ETR_OK;
}

// The pipeline's bounded wait exercised on its own: thread 0 waits on an mbarrier that nothing ever
// arrives on (no TMA, no tensor memory, nothing in flight), gives up after `limit` cycles and leaves
// the code 0x7c08 in error_word, exactly as a GEMM kernel would; the kernel then returns normally.
__global__ void __launch_bounds__(32) tc_wait_selftest_kernel(etr_stats* stats, long long limit) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag_s;
  if (threadIdx.x == 0) {
    abort_flag_s = 0;
    mbar_init(smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (threadIdx.x == 0 && !mbar_wait(smem_u32(&bar), 0u, &abort_flag_s, limit))
    atomicExch(&stats->error_word, 0x7c08);
}

etr_status tc_wait_selftest(etr_stats* stats, long long limit, cudaStream_t st) {
  ETR_TIME_BEGIN("tc_wait_selftest_kernel");
  tc_wait_selftest_kernel<<<1, 32, 0, st>>>(stats, limit);
  ETR_LAUNCH_CHECK();
  return ETR_OK;
}

}  // namespace etr
