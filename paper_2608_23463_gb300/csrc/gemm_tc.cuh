// tcgen05 / TMEM / TMA GEMM for sm_103a with fused epilogues.
//
//   D[M, N] = sum_k A[m, k] * B[n, k]     (bf16 operands, fp32 accumulation)
//
// A is K-major (stored [M, K]) or MN-major (stored [K, M]); likewise B ([N, K]
// or [K, N]).  Every contraction of the layer (compression, proxy Q/K/V/O,
// decompression, and all of their weight / input gradients) is one of these.
//
// Persistent: one CTA per SM walks the 128 x BN output tiles tile = blockIdx.x
// + k * gridDim.x (N fastest, so co-running CTAs share A panels and all of B
// in L2; M fastest when A has at most 16 row tiles and B is wider than the
// grid, so co-running CTAs share B tiles).  With BN = 256 the kernel also runs
// on CTA pairs (clusters of two; gemm_plan chooses): a pair owns a 256 x 256 tile,
// rank 0 issues tcgen05.mma.cta_group::2 (M = 256) and each CTA stages its 128
// rows of A and half of B, so a stage is 32 KB instead of 48 and 7 fit where 4 did (6
// beside a fused epilogue's X, 5 beside the affine one's): the deeper ring hides the HBM
// latency of the streamed operand (a mainloop measured at ~680 cycles per 64-deep K block
// with 4 stages runs at ~525 with 6, the MMAs' own time being 512).  Roles:
//   warp 0   : TMA producer (one thread): STAGES-deep ring of 128B-swizzled
//              64-wide K slices of A and B, continuing across tiles
//   warp 1   : TMEM allocator + MMA issuer (one elected lane): tcgen05.mma
//              M=128 (a pair: 256), N=BN, K=16 into one of two TMEM
//              accumulators (2*BN columns), tcgen05.commit frees smem stages
//              and hands a finished accumulator to the epilogue (a pair: to
//              both CTAs; both CTAs' stage loads complete on rank 0's full
//              barriers, and rank 1's MMA warp has nothing to issue)
//   warps 2-9: epilogue: tcgen05.ld 32 columns at a time (warp w reads TMEM
//              lanes 32*(w%4).. and half of the tile's columns), fused
//              epilogue functor, global stores.  While they drain
//              accumulator i, the MMA warp fills the other.
// Epilogues that read tensors shaped like the output (kRows: the local stream
// X for injection, the direct gradient for dX) give lane (sr, sp) = (lane / 4,
// lane % 4) four columns pairs or eight columns of rows sr, sr + 8, sr + 16, sr
// + 24 of a 32 x 32 chunk, straight from TMEM.  The chunk of X comes by
// cp.async into a ring of 2 KB slots a warp, results leave as 64 contiguous
// bytes a row, and the per-column parameters sit in registers.  Two forms:
//   kDirect (two outputs, K-major B): the rows of B are loaded in the order that
//            puts 8 consecutive columns of a row into one lane, which reads only
//            its own 16 bytes of X and stores both outputs from registers; the
//            reordered loads (four boxes for one) cost the mainloop 15%
//   else     MMA fragments (column pairs), X by ldmatrix, the output over it by
//            stmatrix and out; any B; a second output would go the same way
//            (injection 448 us so, 417 direct), one output is faster (cross_out,
//            M 131072, N = K = 1024: 175 us so, 189 direct)
// What bounds these kernels besides the MMAs is shared memory, its bandwidth
// and its size, and the lines that a store instruction touches (with 32 bytes a
// row injection takes 615 us).  An epilogue whose lanes own rows (X tile by TMA
// in 64 KB, four broadcast parameters a column, outputs staged) took 7k of the
// 16.8k cycles of a 128 x 256 x 1024 tile in shared memory and left room for a
// three-stage ring; these take 1-2k and leave a CTA pair six stages.
// Measured, before and after: injection of the 262144-token layer (M 32768, N
// 8192, K 1024) 487 -> 417 us, its dX 342 -> 330; of the 65536-token layer 152
// -> 122 and 109 -> 99; affine injection of four 512 x 512 images (M 16384, N
// 65536, K 512) 1317 -> 1100, their dX 577 -> 491; cross_out 266 -> 175.
// Every mbarrier wait is bounded (common.cuh); on a timeout the kernel flags
// the error, drains its own copies and MMAs (bounded), frees TMEM and returns.
#pragma once

#include "common.cuh"

namespace pf {

constexpr int GEMM_BM = 128;
constexpr int GEMM_BK = 64;
constexpr int GEMM_EPI_WARPS = 8;  // two per TMEM lane quarter, each owning half the columns
constexpr int GEMM_THREADS = 64 + 32 * GEMM_EPI_WARPS;

// PAIR: the tile is shared by a CTA pair, each CTA staging half of B.
// SB: bytes of shared memory the epilogue stages its output in (0: none).
constexpr uint32_t GEMM_SMEM_MAX = 232448;  // dynamic shared memory per CTA (227 KB)
template <int BN, bool PAIR, uint32_t SB>
struct GemmCfg {
  static constexpr int B_ROWS = PAIR ? BN / 2 : BN;            // B rows staged by one CTA
  static constexpr uint32_t A_BYTES = GEMM_BM * GEMM_BK * 2;  // 16 KB
  static constexpr uint32_t B_BYTES = B_ROWS * GEMM_BK * 2;   // 16/32 KB
  static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr uint32_t FIXED_BYTES = 1024 /*align*/ + 256 /*barriers*/ + SB;
  static constexpr int FIT = (int)((GEMM_SMEM_MAX - FIXED_BYTES) / STAGE_BYTES);
  static constexpr int MOST = PAIR ? 7 : (BN == 256 ? 4 : 6);
  static constexpr int STAGES = FIT < MOST ? FIT : MOST;
  static constexpr uint32_t SMEM_BYTES = STAGES * STAGE_BYTES + FIXED_BYTES;
  static_assert(SMEM_BYTES <= GEMM_SMEM_MAX, "shared memory");
  static_assert(2 * STAGES + 6 <= 31, "barrier region");
};

// Barrier of the epilogue threads (named barrier 1) that also ANDs a predicate
// across them, so that every epilogue thread takes the same branch.
__device__ __forceinline__ bool epi_bar_and(bool p) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred pi, po;\n\t"
      "setp.ne.u32 pi, %1, 0;\n\t"
      "bar.red.and.pred po, 1, %2, pi;\n\t"
      "selp.u32 %0, 1, 0, po;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)p), "n"(32 * GEMM_EPI_WARPS)
      : "memory");
  return r != 0;
}

// A warp's 32 x 32 fp32 stage: row r's 16-byte piece p (columns 4p..) sits at
// piece p ^ (r & 7) of its 128 bytes, so that neither the row-per-lane writes
// nor reads of whole rows (8 lanes a row) or of 8-column segments (4 lanes a
// row) meet in a bank.
constexpr uint32_t GEMM_STG_BYTES = GEMM_EPI_WARPS * 4096;
__device__ __forceinline__ float4* stg_ptr(float* s, int r, int p) {
  return reinterpret_cast<float4*>(s + r * 32 + ((p ^ (r & 7)) << 2));
}
__device__ __forceinline__ void stg_put_row(float* s, int r, const float* v) {
#pragma unroll
  for (int p = 0; p < 8; ++p)
    *stg_ptr(s, r, p) = make_float4(v[4 * p], v[4 * p + 1], v[4 * p + 2], v[4 * p + 3]);
}
__device__ __forceinline__ void stg_get8(float* s, int r, int p8, float* f) {
  const float4 a = *stg_ptr(s, r, 2 * p8), b = *stg_ptr(s, r, 2 * p8 + 1);
  f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
  f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}
// 16 bytes from global to shared memory, past L1: the rows of a chunk are k1 * d
// elements apart, powers of two of which meet in a few sets of the little L1
// that the stage ring leaves (X through registers: 754 us).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ld8_f32(const float* p, float* v) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(p));
  const float4 b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ uint4 pack8_bf16(const float* v) {
  return make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]),
                    pack_bf16(v[6], v[7]));
}

// Shared memory of the epilogue: a kRows one has xd slots of X a warp.
template <class Epi>
constexpr int gemm_xd(bool pair) {
  return pair ? Epi::kPairDepth : 2;
}
template <class Epi>
constexpr uint32_t gemm_slot_bytes() {
  return 2048 + Epi::kParBytes;
}
template <class Epi>
constexpr uint32_t gemm_stage_bytes(bool pair) {
  return Epi::kRows ? (uint32_t)(GEMM_EPI_WARPS * gemm_xd<Epi>(pair)) * gemm_slot_bytes<Epi>()
                    : Epi::kStageBytes;
}

template <int BN, bool A_MN, bool B_MN, class Epi, bool PAIR = false>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmT, int tail, int M, int N, int K,
                   int splits, Epi epi) {
  static_assert(!PAIR || BN == 256, "CTA pairs use 256-wide tiles");
  static_assert(!Epi::kDirect || !B_MN, "direct epilogues need a K-major B");
  constexpr uint32_t SB = gemm_stage_bytes<Epi>(PAIR);
  using Cfg = GemmCfg<BN, PAIR, SB>;
  constexpr int STAGES = Cfg::STAGES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  // output staging of the epilogue warps (kStageBytes), then the barriers:
  // full[S], empty[S], tfull[2], tempty[2], done
  uint8_t* const epi_smem = smem + STAGES * Cfg::STAGE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(epi_smem + SB);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 6);
  __shared__ uint32_t s_consumed;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // a pair (cluster of two CTAs) works on one tile of 2 x 128 rows: `unit` is
  // the pair (or the lone CTA), `rank` this CTA's half of the rows
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
  const int unit = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const int n_units = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  constexpr int TILE_M = PAIR ? 2 * GEMM_BM : GEMM_BM;
  const int num_n = (N + BN - 1) / BN, num_m = (M + TILE_M - 1) / TILE_M;
  const int mn_tiles = num_m * num_n;
  // N fastest keeps the co-running CTAs on one A panel with all of B in L2;
  // when A is a few row tiles and B is wider than the grid, M fastest instead
  // lets the co-running CTAs share each B tile (B is then read once)
  const bool m_fast = num_m <= 16 && num_n > n_units;
  const int tiles = mn_tiles * splits;
  const int num_k = (K + GEMM_BK - 1) / GEMM_BK;
  const int kps = (num_k + splits - 1) / splits;  // K tiles per split
  // tile t -> split t / mn_tiles (slowest), then M, then N (fastest); m0 is
  // this CTA's first row
#define PF_TILE_DECODE(t)                                                        \
  const int sp = (t) / mn_tiles, rem = (t) % mn_tiles;                           \
  const int m0 = (m_fast ? rem % num_m : rem / num_n) * TILE_M + (int)rank * GEMM_BM; \
  const int n0 = (m_fast ? rem / num_m : rem % num_n) * BN;                      \
  const int kb = sp * kps, ke = min(num_k, kb + kps);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES);
  const uint32_t tfull0 = smem_u32(bars + 2 * STAGES), tempty0 = tfull0 + 16;
  const uint32_t done = tfull0 + 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull0 + 8 * b, 1);
      // one arrival per epilogue warp (of both CTAs of a pair, on rank 0)
      mbar_init(tempty0 + 8 * b, PAIR ? 2 * GEMM_EPI_WARPS : GEMM_EPI_WARPS);
    }
    mbar_init(done, 1);
    fence_barrier_init();
    s_consumed = 0;
  }
  if (warp == 1) {
    if (PAIR) {
      tmem_alloc_pair(smem_u32(tmem_slot), 2 * BN);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(tmem_slot), 2 * BN);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();  // both CTAs' barriers exist before any remote arrival
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // the setup above overlaps the kernel before this one; every address that is read
  // follows from the tile, and with it from the wait
  const int first = unit + pdl_enter();
  uint32_t issued = 0;

  if (warp == 0 && lane == 0) {
    // ---------------------------------------------------------- producer
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
    // test hook: arm no stage and issue no load, so that nothing is ever in
    // flight and the MMA warp's first wait runs out
    const bool skip_loads = *(volatile int*)&g_debug_skip_loads != 0;
    uint32_t it = 0;
    bool ok = true;
    for (int tile = first; tile < tiles && ok; tile += n_units) {
      PF_TILE_DECODE(tile)
      (void)sp;
      for (int kt = kb; kt < ke; ++kt, ++it) {
        const int s = it % STAGES;
        const uint32_t ph = (it / STAGES) & 1;
        if (!mbar_wait(empty0 + 8 * s, ph ^ 1)) {
          ok = false;
          break;
        }
        if (skip_loads) continue;
        // a pair: both CTAs' loads complete on rank 0's full barrier, which
        // rank 0 arms for the two CTAs' bytes
        const uint32_t fb = PAIR ? smem_map_rank(full0 + 8 * s, 0) : full0 + 8 * s;
        if (!PAIR || rank == 0)
          mbar_arrive_expect_tx(full0 + 8 * s, (PAIR ? 2u : 1u) * Cfg::STAGE_BYTES);
        auto ld = [&](uint32_t dst, const CUtensorMap* map, int c0, int c1) {
          if (PAIR)
            tma_load_2d_pair(dst, map, fb, c0, c1);
          else
            tma_load_2d(dst, map, fb, c0, c1);
        };
        const uint32_t a_dst = smem_u32(smem + s * Cfg::STAGE_BYTES);
        const uint32_t b_dst = a_dst + Cfg::A_BYTES;
        const int k0 = kt * GEMM_BK;
        // columns below `tail` of the operand that ends inside a row (A or B, by the
        // majors) go through their own map
        if (!A_MN) {
          ld(a_dst, !B_MN && !Epi::kRows && k0 < tail ? &tmT : &tmA, k0, m0);
        } else {
          ld(a_dst, &tmA, m0, k0);
          ld(a_dst + 8192, &tmA, m0 + 64, k0);
        }
        // this CTA's B rows: all of them, or (a pair) its half of the columns
        if (Epi::kDirect) {
          // box row 32 g + 2 s + e of a 128-row box holds B row 8 s + 2 g + e
          constexpr int JB = Cfg::B_ROWS / 128;
#pragma unroll
          for (int j = 0; j < JB; ++j) {
            const int s8 = epi.b_row(n0, j + (int)rank * JB) >> 3;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              if (PAIR)
                tma_load_4d_pair(b_dst + j * 16384 + g * 4096, &tmB, fb, k0, 0, g, s8);
              else
                tma_load_4d(b_dst + j * 16384 + g * 4096, &tmB, fb, k0, 0, g, s8);
            }
          }
        } else if (!B_MN) {
          constexpr int JB = Cfg::B_ROWS / 128;
#pragma unroll
          for (int j = 0; j < JB; ++j)
            ld(b_dst + j * 16384, &tmB, k0, epi.b_row(n0, j + (int)rank * JB));
        } else {
          constexpr int JB = Cfg::B_ROWS / 64;
#pragma unroll
          for (int j = 0; j < JB; ++j) {
            const int n = n0 + 64 * (j + (int)rank * JB);
            ld(b_dst + j * 8192, A_MN && n < tail ? &tmT : &tmB, n, k0);
          }
        }
        issued = it + 1;
      }
    }
  } else if (warp == 1 && PAIR && rank == 1) {
    // rank 1 of a pair: rank 0 issues the MMAs for both CTAs
  } else if (warp == 1) {
    // ---------------------------------------------------------- MMA issuer
    // The whole warp runs the loop; one elected lane issues and commits.
    constexpr uint32_t idesc = idesc_bf16_f32(TILE_M, BN, A_MN ? 1 : 0, B_MN ? 1 : 0);
    uint32_t it = 0, lt = 0;
    bool ok = true;
    for (int tile = first; tile < tiles && ok; tile += n_units, ++lt) {
      const uint32_t buf = lt & 1, use = lt >> 1;
      if (!mbar_wait_warp(tempty0 + 8 * buf, (use & 1) ^ 1)) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem + buf * BN;
      PF_TILE_DECODE(tile)
      (void)sp;
      (void)m0;
      (void)n0;
      for (int kt = kb; kt < ke; ++kt, ++it) {
        const int s = it % STAGES;
        const uint32_t ph = (it / STAGES) & 1;
        if (!mbar_wait_warp(full0 + 8 * s, ph)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t a_base = smem_u32(smem + s * Cfg::STAGE_BYTES);
        const uint32_t b_base = a_base + Cfg::A_BYTES;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < GEMM_BK / 16; ++kk) {
            // K-major: 16 K-elements = 32 bytes along the swizzled 128-byte row,
            //          8-row groups 1024 bytes apart (SBO).
            // MN-major: 16 K-rows = 2048 bytes; 64-wide MN slabs 8192 bytes apart
            //          (LBO), 8-row K groups 1024 bytes apart (SBO).
            const uint64_t ad = A_MN ? smem_desc_sw128(a_base + kk * 2048, 8192, 1024)
                                     : smem_desc_sw128(a_base + kk * 32, 16, 1024);
            const uint64_t bd = B_MN ? smem_desc_sw128(b_base + kk * 2048, 8192, 1024)
                                     : smem_desc_sw128(b_base + kk * 32, 16, 1024);
            if (PAIR)
              tc_mma_f16_pair(d_tmem, ad, bd, idesc, (kt != kb || kk != 0) ? 1u : 0u);
            else
              tc_mma_f16(d_tmem, ad, bd, idesc, (kt != kb || kk != 0) ? 1u : 0u);
          }
          if (PAIR)
            tc_commit_pair(empty0 + 8 * s);
          else
            tc_commit(empty0 + 8 * s);
        }
        __syncwarp();
      }
      if (elect_one()) {
        if (PAIR)
          tc_commit_pair(tfull0 + 8 * buf);
        else
          tc_commit(tfull0 + 8 * buf);
      }
      __syncwarp();
    }
    if (lane == 0) s_consumed = it;
    if (elect_one()) {
      if (PAIR)
        tc_commit_pair(done);
      else
        tc_commit(done);
    }
    __syncwarp();
  } else if (warp >= 2) {
    // ---------------------------------------------------------- epilogue
    const int q = warp & 3;                               // TMEM lane quarter
    const int c_begin = ((warp - 2) >> 2) * (BN / 2);     // this warp's column half
    // the accumulator has been read: rank 0's MMA warp may fill it again
    auto release = [&](uint32_t buf) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (PAIR && rank == 1)
          mbar_arrive_remote_relaxed(smem_map_rank(tempty0 + 8 * buf, 0));
        else
          mbar_arrive(tempty0 + 8 * buf);
      }
    };
    uint32_t lt = 0;
    if constexpr (Epi::kRows) {
      // No barrier couples the warps: one that sees a wait run out leaves alone.
      constexpr int NCH = Epi::kPaired ? BN / 128 : BN / 64;  // 32-column chunks per warp
      constexpr int XD = gemm_xd<Epi>(PAIR), AHEAD = XD - 1 < NCH ? XD - 1 : NCH;
      const int cb = Epi::kPaired ? c_begin / 2 : c_begin;
      const int sr = lane >> 2, sp = lane & 3;
      typename Epi::Rows rows, nrows;
      // A slot holds the chunk's 32 rows x 64 bytes of X.  Lane (sr, sp) copies
      // pieces sp (16 bytes) of rows sr + 8 it to `mine`.  Fragments: row r's piece
      // p sits at piece p ^ (r / 2 % 4), so that neither a matrix's eight rows nor
      // the lanes' pieces meet in a bank; lane names row lane % 8 of matrix lane / 8.
      constexpr uint32_t SLOT = gemm_slot_bytes<Epi>();
      uint8_t* const slots = epi_smem + (warp - 2) * (XD * SLOT);
      const uint32_t slots0 = smem_u32(slots);
      const uint32_t mine = Epi::kDirect ? lane * 16 : sr * 64 + ((sp ^ ((sr >> 1) & 3)) << 4);
      const uint32_t mrow = (lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) << 4);
      auto info = [&](int t, typename Epi::Rows& r) -> int {  // rows of tile t; returns its n0
        const int rem = t % mn_tiles;
        const int m0 = (m_fast ? rem % num_m : rem / num_n) * TILE_M + (int)rank * GEMM_BM;
        const int n0 = (m_fast ? rem / num_m : rem % num_n) * BN;
        epi.rows_info(r, m0 + q * 32 + sr, n0);
        return n0;
      };
      auto load = [&](uint32_t trow, int c, uint32_t* r) {
        if constexpr (Epi::kDirect) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int g = 0; g < 4; ++g)
              tmem_ld_16x8_async(trow + ((uint32_t)(16 * h) << 16) +
                                     (uint32_t)((c & ~127) + 32 * g + ((c & 127) >> 2)),
                                 r + 16 * h + 4 * g);
        } else {
          tmem_ld_frag_async(trow + (uint32_t)c, r);
          tmem_ld_frag_async(trow + (16u << 16) + (uint32_t)c, r + 16);
        }
        tmem_wait_ld(r);
      };
      uint32_t put = 0, get = 0;  // pieces of how many chunks were requested / used
      // Pieces past the last row or token are not read: their slot holds what it held, and
      // their results are not stored.  (All read from X's first 16 bytes instead, 208 such
      // rows of 1024 x 12288 took 60 of 90 us in one L2 slice.)
      auto fetch = [&](const typename Epi::Rows& r, int n0, int ci) {
        const int c = cb + 32 * ci;
        if (n0 + c < N) {  // uniform
#pragma unroll
          for (int it = 0; it < 4; ++it)
            if (const bf16* x = epi.src(r, it, n0, c + 8 * sp))
              cp_async16(slots0 + (put % XD) * SLOT + it * 512 + mine, x);
          if constexpr (Epi::kParBytes > 0)
            if (lane * 16 < (int)Epi::kParBytes)
              cp_async16(slots0 + (put % XD) * SLOT + 2048 + lane * 16, epi.par_src(r, c, lane));
        }
      };
      int n0 = 0, nn0 = 0;
      if (first < tiles) {
        n0 = info(first, rows);
#pragma unroll
        for (int ci = 0; ci < AHEAD; ++ci, ++put) {
          fetch(rows, n0, ci);
          cp_async_commit();
        }
      }
      for (int tile = first; tile < tiles; tile += n_units, ++lt) {
        const uint32_t buf = lt & 1, use = lt >> 1;
        const bool more = tile + n_units < tiles;
        if (more) {
          nn0 = info(tile + n_units, nrows);
        }
        if (!mbar_wait_warp(tfull0 + 8 * buf, use & 1)) break;
        tc_fence_after();
        const uint32_t trow = tmem + buf * BN + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
        for (int ci = 0; ci < NCH; ++ci, ++put, ++get) {
          const int c = cb + 32 * ci;
          const bool live = n0 + c < N;  // uniform
          typename Epi::Par par;
          if constexpr (Epi::kParBytes > 0) {
            __syncwarp();  // the slot's last reader is done
          } else {
            if (live) epi.params(par, n0, c + (Epi::kDirect ? 8 : 2) * sp);
          }
          // the pieces of the chunk AHEAD of this one
          if (ci + AHEAD < NCH)
            fetch(rows, n0, ci + AHEAD);
          else if (more)
            fetch(nrows, nn0, ci + AHEAD - NCH);
          cp_async_commit();
          // r[16 h + 4 g + 2 k + e]: row sr + 16 h + 8 k, column 8 g + 2 sp + e (direct:
          // column 8 sp + 2 g + e)
          const uint32_t slot = (get % XD) * SLOT;
          uint32_t r[32];
          load(trow, c, r);
          if constexpr (Epi::kDirect) {
            uint32_t r2[32];
            if (Epi::kPaired) load(trow, c + BN / 2, r2);  // belong to columns c..
            if (ci == NCH - 1) release(buf);
            cp_async_wait<AHEAD>();  // this chunk's pieces have landed
            if constexpr (Epi::kParBytes > 0) {
              __syncwarp();
              if (live) epi.params(par, slots + slot + 2048, sp);
            }
            if (live) {
#pragma unroll
              for (int it = 0; it < 4; ++it) {
                float f[8], ft[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const int i = 16 * (it >> 1) + 4 * (j >> 1) + 2 * (it & 1) + (j & 1);
                  f[j] = __uint_as_float(r[i]);
                  if (Epi::kPaired) ft[j] = __uint_as_float(r2[i]);
                }
                const uint4 x = *reinterpret_cast<const uint4*>(slots + slot + it * 512 + mine);
                if constexpr (Epi::kPaired)
                  epi.apply(rows, par, it, n0, c + 8 * sp, f, ft, x);
                else
                  epi.apply(rows, par, it, n0, c + 8 * sp, f, x);
              }
            }
          } else {
            if (ci == NCH - 1) release(buf);
            cp_async_wait<AHEAD>();
            __syncwarp();  // the warp's pieces of this chunk have landed
            uint32_t o[4][4];
#pragma unroll
            for (int it = 0; it < 4; ++it) {
              uint32_t x[4];
              ldmatrix_x4(slots0 + slot + it * 512 + mrow, x);
              const uint32_t* a = r + 16 * (it >> 1) + 2 * (it & 1);
#pragma unroll
              for (int g = 0; g < 4; ++g)
                o[it][g] = epi.apply(
                    make_float2(__uint_as_float(a[4 * g]), __uint_as_float(a[4 * g + 1])), x[g]);
            }
            __syncwarp();  // the slot's readers are done: the output takes its place
#pragma unroll
            for (int it = 0; it < 4; ++it) stmatrix_x4(slots0 + slot + it * 512 + mrow, o[it]);
            __syncwarp();
            if (live) {
#pragma unroll
              for (int it = 0; it < 4; ++it) {
                const uint4 w = *reinterpret_cast<const uint4*>(slots + slot + it * 512 + mine);
                if (bf16* d = epi.dst(rows, it, n0, c + 8 * sp)) *reinterpret_cast<uint4*>(d) = w;
              }
            }
          }
        }
        rows = nrows;
        n0 = nn0;
      }
      cp_async_wait<0>();
    } else {
      for (int tile = first; tile < tiles; tile += n_units, ++lt) {
        PF_TILE_DECODE(tile)
        const bool no_k = ke <= kb;
        const uint32_t buf = lt & 1, use = lt >> 1;
        const bool ok = mbar_wait(tfull0 + 8 * buf, use & 1);
        tc_fence_after();
        const int rl = q * 32 + lane;
        // split-K partial epilogues address row (split * M + row); -1 = out of range
        const int erow = Epi::kSplitRows ? (m0 + rl < M ? sp * M + m0 + rl : -1) : m0 + rl;
        const typename Epi::Row ri = epi.row_info(erow, n0);
        const uint32_t trow = tmem + buf * BN + ((uint32_t)(q * 32) << 16);
        // 32-column chunks, the TMEM load of chunk i+1 in flight while chunk i
        // is processed
        constexpr int NCH = BN / 64;
        auto run = [&](uint32_t* r, int c) {
          if (no_k) {  // uniform: a split with no K blocks
#pragma unroll
            for (int i = 0; i < 32; ++i) r[i] = 0u;
          }
          float v[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
          epi.apply(ri, erow, n0 + c, v, epi_smem, rl);
        };
        uint32_t ra[32], rb[32];
        tmem_ld32_async(trow + (uint32_t)c_begin, ra);
        tmem_wait_ld(ra);
#pragma unroll 1
        for (int ci = 0; ci < NCH; ci += 2) {
          const int c = c_begin + ci * 32;
          tmem_ld32_async(trow + (uint32_t)(c + 32), rb);
          run(ra, c);
          tmem_wait_ld(rb);
          if (ci + 2 < NCH) tmem_ld32_async(trow + (uint32_t)(c + 64), ra);
          run(rb, c + 32);
          if (ci + 2 < NCH) tmem_wait_ld(ra);
        }
        release(buf);
        // leave together if any epilogue thread saw a wait run out
        if (!epi_bar_and(ok)) break;
      }
    }
  }
  tc_fence_before();
  if (__syncthreads_or(*(volatile int*)&g_dev_error != 0)) {
    // error path: let in-flight TMA copies and MMAs land before TMEM/smem go.
    if (warp == 0 && lane == 0) {
      if (PAIR && rank == 1) {
        // its loads complete on rank 0's barriers: give them a bounded time
        // (far above a load's latency) to land before the CTA goes
        const unsigned long long t0 = globaltimer();
        while (globaltimer() - t0 < 50000ull) {
        }
      } else {
        for (uint32_t it = s_consumed; it < issued; ++it)
          mbar_wait_drain(full0 + 8 * (it % STAGES), (it / STAGES) & 1);
      }
    }
    if (warp == 1 && lane == 0) mbar_wait_drain(done, 0);
    __syncthreads();
  } else if (warp == 1 && lane == 0) {
    mbar_wait(done, 0);
  }
  __syncthreads();
  // a pair: neither CTA leaves (or frees TMEM) while the other may still use
  // its shared memory or TMEM
  if (PAIR) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    if (PAIR)
      tmem_dealloc_pair(tmem, 2 * BN);
    else
      tmem_dealloc(tmem, 2 * BN);
  }
}

// ------------------------------------------------------------------ epilogues
// Row-per-lane epilogues: row_info(row, n0) is evaluated once per tile and
// output row; apply(ri, row, col, v, stg, rl) then receives 32 consecutive
// accumulator columns [col, col+32) of that row (rl: the row inside the tile).
// kRows epilogues: rows_info(r, row, n0) describes a lane's rows row, row + 8,
// row + 16, row + 24 of the tile that starts at output column n0; src(r, it, n0,
// c) is the address of the 16 bytes that its it-th row needs for columns n0 + c
// .. + 7, or null for a row or token past the end: nothing is copied then, x is what the
// slot held before, and what is made of it must not be stored.  kDirect: params(par,
// n0, c) reads the parameters of columns n0 + c .. + 7 and apply(r, par, it, n0, c, f, x)
// stores them (kPaired: with columns c + BN/2 in ft).  Else apply(f, x) gives an output
// pair and dst the address of 8 output columns of a row, or null.  b_row(n0, j) is the first
// row of B (K-major) loaded for 128-row box j of the tile starting at output
// column n0.  N is a multiple of 32.
struct EpiBase {
  static constexpr uint32_t kParBytes = 0;  // kRows: parameters of a 32-column chunk, beside its X
  static constexpr bool kRows = false;
  static constexpr bool kDirect = false;
  static constexpr int kPairDepth = 0;
  static constexpr bool kPaired = false;
  static constexpr bool kSplitRows = false;
  // shared memory for staging the output (0: the epilogue stores from registers)
  static constexpr uint32_t kStageBytes = 0;
  __device__ __forceinline__ int b_row(int n0, int j) const { return n0 + 128 * j; }
};
// n / d and n % d for 0 <= n < 2^31 by a multiplication with ceil(2^(31 + l) / d), l =
// ceil(log2 d) (Granlund and Montgomery, 1994): a tile's rows take eight divisions a lane.
struct FastDiv {
  uint32_t d, mul, sh;
  explicit FastDiv(int dv) : d((uint32_t)dv), mul(0), sh(0) {
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;
    if (l > 0) {
      mul = (uint32_t)(((1ull << (31 + l)) + d - 1) / d);
      sh = l - 1;
    }
  }
  __device__ __forceinline__ int div(int n) const {
    return d == 1 ? n : (int)(__umulhi((uint32_t)n, mul) >> sh);
  }
};

struct EpiRowsBase : EpiBase {
  static constexpr bool kRows = true;
  static constexpr int kPairDepth = 2;  // gemm_xd of a CTA pair
  struct Par {};
  __device__ __forceinline__ void params(Par&, int, int) const {}
  // acc + X (the sums of a product and a bf16 matrix)
  __device__ __forceinline__ uint32_t apply(float2 f, uint32_t x) const {
    const float2 a = unpack_bf16(x);
    return pack_bf16(f.x + a.x, f.y + a.y);
  }
};

// v = acc (+ bias[col]) (+ addend[row, col]); stored as fp32 and/or bf16.
struct EpiLinear : EpiBase {
  struct Row {
    bool ok;
  };
  int M, N;
  const float* bias;
  const float* addend;
  long ld_add;
  float* out_f32;
  long ld_f32;
  bf16* out_bf16;
  long ld_bf16;
  int act_silu;
  bf16* pre_bf16;
  long ld_pre;
  const bf16* dsilu_of;
  long ld_dsilu;
  __device__ __forceinline__ Row row_info(int row, int) const { return Row{row < M}; }
  __device__ __forceinline__ void apply(const Row& ri, int row, int col, float* v, uint8_t*,
                                        int) const {
    if (!ri.ok || col >= N) return;
    if (bias) {
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        float4 b = *reinterpret_cast<const float4*>(bias + col + i);
        v[i] += b.x; v[i + 1] += b.y; v[i + 2] += b.z; v[i + 3] += b.w;
      }
    }
    if (addend) {
      const float* a = addend + (long)row * ld_add + col;
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        float4 b = *reinterpret_cast<const float4*>(a + i);
        v[i] += b.x; v[i + 1] += b.y; v[i + 2] += b.z; v[i + 3] += b.w;
      }
    }
    if (pre_bf16) {
      bf16* o = pre_bf16 + (long)row * ld_pre + col;
#pragma unroll
      for (int i = 0; i < 32; i += 8) store8_bf16(o + i, v + i);
    }
    if (act_silu) {
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = v[i] / (1.f + __expf(-v[i]));
    }
    if (dsilu_of) {
      const bf16* u = dsilu_of + (long)row * ld_dsilu + col;
#pragma unroll
      for (int i = 0; i < 32; i += 8) {
        const uint4 q = *reinterpret_cast<const uint4*>(u + i);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 f = unpack_bf16(w[j]);
          const float s0 = 1.f / (1.f + __expf(-f.x)), s1 = 1.f / (1.f + __expf(-f.y));
          v[i + 2 * j] *= s0 * (1.f + f.x * (1.f - s0));
          v[i + 2 * j + 1] *= s1 * (1.f + f.y * (1.f - s1));
        }
      }
    }
    if (out_f32) {
      float* o = out_f32 + (long)row * ld_f32 + col;
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        *reinterpret_cast<float4*>(o + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
    if (out_bf16) {
      bf16* o = out_bf16 + (long)row * ld_bf16 + col;
#pragma unroll
      for (int i = 0; i < 32; i += 8) store8_bf16(o + i, v + i);
    }
  }
};

// A linear epilogue (v = acc + bias, fp32 and / or bf16 out) that stores
// whole rows: each warp stages its 32 x 32 chunk in shared memory and writes
// it back row by row, 128 contiguous bytes of fp32 per row.  Used where the
// output is large next to the contraction (short K), so that the stores from
// one row per lane would bound the epilogue.
struct EpiLinearStaged : EpiBase {
  static constexpr uint32_t kStageBytes = GEMM_STG_BYTES;
  struct Row {
    bool ok;
  };
  int M, N;
  const float* bias;
  float* out_f32;
  long ld_f32;
  bf16* out_bf16;
  long ld_bf16;
  __device__ __forceinline__ Row row_info(int row, int) const { return Row{row < M}; }
  __device__ __forceinline__ void apply(const Row&, int row, int col, float* v, uint8_t* stg,
                                        int rl) const {
    if (col >= N) return;  // uniform across the warp
    const int lane = threadIdx.x & 31, ew = (threadIdx.x >> 5) - 2;
    float* s = reinterpret_cast<float*>(stg) + ew * 1024;
    if (bias) {
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        const float4 b = *reinterpret_cast<const float4*>(bias + col + i);
        v[i] += b.x; v[i + 1] += b.y; v[i + 2] += b.z; v[i + 3] += b.w;
      }
    }
    stg_put_row(s, lane, v);
    __syncwarp();
    const int rfirst = row - (rl & 31);
    if (out_f32) {  // 8 lanes per row, 4 rows per instruction
#pragma unroll
      for (int it = 0; it < 8; ++it) {
        const int rr = it * 4 + (lane >> 3), p = lane & 7;
        const float4 val = *stg_ptr(s, rr, p);
        if (rfirst + rr < M)
          *reinterpret_cast<float4*>(out_f32 + (long)(rfirst + rr) * ld_f32 + col + 4 * p) = val;
      }
    }
    if (out_bf16) {  // 4 lanes per row (8 values each), 8 rows per instruction
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        const int rr = it * 8 + (lane >> 2), p = lane & 3;
        float f[8];
        stg_get8(s, rr, p, f);
        if (rfirst + rr < M)
          *reinterpret_cast<uint4*>(out_bf16 + (long)(rfirst + rr) * ld_bf16 + col + 8 * p) =
              pack8_bf16(f);
      }
    }
    __syncwarp();  // the staging is reused by the next chunk
  }
};

// out = acc + add, bf16, row strides ld and ld_add (the residual and direct
// gradient sums of the cross injection).
struct EpiAddRows : EpiRowsBase {
  struct Rows {
    int row;
  };
  int M, N;
  const bf16* add;
  long ld_add;
  bf16* out;
  long ld;
  __device__ __forceinline__ void rows_info(Rows& r, int row, int) const { r.row = row; }
  __device__ __forceinline__ const bf16* src(const Rows& r, int it, int n0, int c) const {
    const int row = r.row + 8 * it;
    return row < M ? add + (long)row * ld_add + n0 + c : nullptr;
  }
  __device__ __forceinline__ bf16* dst(const Rows& r, int it, int n0, int c) const {
    const int row = r.row + 8 * it;
    return row < M ? out + (long)row * ld + n0 + c : nullptr;
  }
};

// Last decompression level of a 1D layer fused with routing and injection.
// GEMM rows are proxy-order rows r = (b*m + i)*k2 + a (proxy i of sequence b,
// level-1 row a); columns c in [0, k1*d) are (token c/d of the k1-group,
// channel c%d).  D = acc + b_d1 is saved in that layout; it is injected into
// block i + shift (shift = 1: causal routing, 0: bidirectional) at token
// (i+shift)*P + a*k1 + c/d:
//   gated: X_out = X + sigmoid(w_x X + w_dlt D + b_g) D    (Eq. inj-gate)
//   add:   X_out = X + D                                    (Eq. inj-add)
// With shift = 1 the last proxy of a sequence feeds no block; its rows copy
// the sequence's block 0, which receives nothing, X_out = X.
struct EpiInject1D : EpiRowsBase {
  static constexpr bool kDirect = true;
  struct Rows {
    long off[4];  // element offset of the row's first token in X and X_out
    int lim[4];   // columns < lim belong to tokens < L of the row's block (0: none)
    int row;
    uint32_t copy;  // bit it: row it copies block 0
  };
  struct Par {
    float b[8], wx[8], wd[8], bg[8];
  };
  int M, N;
  const float* bias;
  bf16* D_save;
  const bf16* X;
  bf16* X_out;
  const float *w_x, *w_dlt, *b_g;
  int d, k1, k2, m, L, shift, gated;
  FastDiv dk2, dm, dd;  // by k2, m, d
  __device__ __forceinline__ void rows_info(Rows& r, int row, int) const {
    r.row = row;
    r.copy = 0;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int rr = row + 8 * it;
      const int prox = dk2.div(rr), a = rr - prox * k2;
      const int b = dm.div(prox), i = prox - b * m;
      int blk = i + shift;
      if (blk >= m) {
        blk = 0;
        r.copy |= 1u << it;
      }
      const long tok0 = (long)blk * (k1 * k2) + (long)a * k1;
      const long lim = (L - tok0) * d;
      r.off[it] = ((long)b * L + tok0) * d;
      r.lim[it] = rr < M && lim > 0 ? (lim < N ? (int)lim : N) : 0;
    }
  }
  __device__ __forceinline__ const bf16* src(const Rows& r, int it, int n0, int c) const {
    return n0 + c < r.lim[it] ? X + r.off[it] + n0 + c : nullptr;
  }
  __device__ __forceinline__ void params(Par& p, int n0, int c) const {
    const int col = n0 + c;
    ld8_f32(bias + col, p.b);
    if (gated) {
      const int ch = col - dd.div(col) * d;
      ld8_f32(w_x + ch, p.wx);
      ld8_f32(w_dlt + ch, p.wd);
      ld8_f32(b_g + ch, p.bg);
    }
  }
  // the gate arithmetic runs on column pairs with packed fp32x2 FMAs (each
  // lane an IEEE fp32 FMA, as the scalar form)
  __device__ __forceinline__ void apply(const Rows& r, const Par& p, int it, int n0, int c,
                                        const float* f, uint4 x) const {
    const int col = n0 + c;
    const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
    uint32_t ow[4], dw[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = 2 * j;
      const float2 x2 = unpack_bf16(xw[j]);
      const float2 d2 = __fadd2_rn(make_float2(f[k], f[k + 1]), make_float2(p.b[k], p.b[k + 1]));
      float2 o2;
      if (gated) {
        const float2 g2 = __ffma2_rn(make_float2(p.wx[k], p.wx[k + 1]), x2,
                                     __ffma2_rn(make_float2(p.wd[k], p.wd[k + 1]), d2,
                                                make_float2(p.bg[k], p.bg[k + 1])));
        const float2 hg = __fmul2_rn(g2, make_float2(0.5f, 0.5f));
        const float2 t2 = make_float2(tanh_approx(hg.x), tanh_approx(hg.y));
        const float2 s2 = __ffma2_rn(make_float2(0.5f, 0.5f), t2, make_float2(0.5f, 0.5f));
        o2 = __ffma2_rn(s2, d2, x2);
      } else {
        o2 = __fadd2_rn(x2, d2);
      }
      ow[j] = pack_bf16(o2.x, o2.y);
      dw[j] = pack_bf16(d2.x, d2.y);
    }
    if (col < r.lim[it])
      *reinterpret_cast<uint4*>(X_out + r.off[it] + col) =
          (r.copy >> it) & 1u ? x : make_uint4(ow[0], ow[1], ow[2], ow[3]);
    const int row = r.row + 8 * it;
    if (D_save && row < M)
      *reinterpret_cast<uint4*>(D_save + (long)row * N + col) =
          make_uint4(dw[0], dw[1], dw[2], dw[3]);
  }
};

// First compression level's input gradient added to the direct injection
// gradient that dX already holds: rows r = (b*m + i)*k2 + a, columns (token
// c/d of the group, channel c%d) -> token i*P + a*k1 + c/d of sequence b.
// Each element of dX is read and written by one lane.
struct EpiDX1D : EpiRowsBase {
  struct Rows {
    long off[4];
    int lim[4];
  };
  int M, N;
  bf16* dX;
  int d, k1, L;
  FastDiv dper;  // by the rows of a sequence, m k2
  __device__ __forceinline__ void rows_info(Rows& r, int row, int) const {
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int rr = row + 8 * it, b = dper.div(rr);
      const long tok0 = (long)(rr - b * (int)dper.d) * k1, lim = (L - tok0) * d;
      r.off[it] = ((long)b * L + tok0) * d;
      r.lim[it] = rr < M && lim > 0 ? (lim < N ? (int)lim : N) : 0;
    }
  }
  __device__ __forceinline__ const bf16* src(const Rows& r, int it, int n0, int c) const {
    return dst(r, it, n0, c);
  }
  __device__ __forceinline__ bf16* dst(const Rows& r, int it, int n0, int c) const {
    return n0 + c < r.lim[it] ? dX + r.off[it] + n0 + c : nullptr;
  }
};

// KV append (Sec. 3.8): rows are sequences b, columns [0, 2d) the proxy's key
// and value rows W_kh H and W_vh H, written as bf16 at cache row n_proxy[b] of
// the sequences whose open block is full and whose cache has room; without n_proxy,
// row by row.
struct EpiAppendKV : EpiBase {
  struct Row {
    bool ok;
    long off;
  };
  int M, N;
  bf16 *K, *V;
  const int *n_open, *n_proxy;
  int d, P, cap;
  __device__ __forceinline__ Row row_info(int row, int) const {
    Row r{false, 0};
    if (row < M && !n_proxy) {
      r.ok = true;
      r.off = (long)row * d;
    } else if (row < M) {
      const int np = n_proxy[row];
      r.ok = n_open[row] == P && np >= 0 && np < cap;
      r.off = ((long)row * cap + (r.ok ? np : 0)) * d;
    }
    return r;
  }
  __device__ __forceinline__ void apply(const Row& ri, int, int col, float* v, uint8_t*,
                                        int) const {
    if (!ri.ok || col >= N) return;
    bf16* o = col < d ? K + ri.off + col : V + ri.off + (col - d);
#pragma unroll
    for (int i = 0; i < 32; i += 8) store8_bf16(o + i, v + i);
  }
};

// Decompression of the 2D layer fused with affine injection (Eq. inj-affine):
// X_out = (1 + s) * LayerNorm(X) + t.  GEMM rows are patches r = (b, by, bx);
// W_d1 [2*P*d, d] holds s for token p of a patch at rows [2pd, 2pd+d) and t at
// [2pd+d, 2(p+1)d).  Output tile n0 = 256*nt covers token p = nt / (d/128) and
// channels [cb, cb+128), cb = 128 * (nt % (d/128)): its B rows are loaded as
// s (columns 0..127) then t (128..255), so each lane holds matching s and t.
// LayerNorm statistics per token from `stats` (mean, 1/std).  s is saved in
// patch order [B*m, P*d] for the backward.
struct EpiAffine2D : EpiRowsBase {
  static constexpr bool kDirect = true;
  static constexpr bool kPaired = true;
  // two chunks ahead of X (K = d <= 512: the epilogue, not the ring, bounds it), the
  // chunk's biases with it: 16384 patches of 64 tokens, d = 512, take 973 us, with
  // their loads in the open and eight divisions a row 1110
  static constexpr int kPairDepth = 3;
  static constexpr uint32_t kParBytes = 256;
  struct Rows {
    long off[4];  // element offset of (token, channel cb) in X and X_out
    float2 st[4];
    int row;
    int pcol, pbias;  // p d + cb and 2 p d + cb
  };
  struct Par {
    float bs[8], bt[8];
  };
  int M;
  const float* bias;
  bf16* S_save;
  const bf16* X;
  bf16* X_out;
  const float* stats;
  int d, patch, gh, gw, m;
  FastDiv dm, dnpw, dpatch, dch;  // by m, patches per row, patch, 128-channel slices of d
  __device__ __forceinline__ int ptok(int n0) const { return dch.div(n0 >> 8); }
  __device__ __forceinline__ int cbase(int n0) const {
    return ((n0 >> 8) - ptok(n0) * (int)dch.d) << 7;
  }
  __device__ __forceinline__ int b_row(int n0, int j) const {
    return ptok(n0) * 2 * d + j * d + cbase(n0);
  }
  __device__ __forceinline__ void rows_info(Rows& r, int row, int n0) const {
    const int p = ptok(n0), py = dpatch.div(p), px = p - py * patch, cb = cbase(n0);
    r.row = row;
    r.pcol = p * d + cb;
    r.pbias = r.pcol + p * d;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int rr = row + 8 * it;
      r.off[it] = 0;
      r.st[it] = make_float2(0.f, 0.f);
      if (rr < M) {
        const int b = dm.div(rr), pr = rr - b * m, by = dnpw.div(pr), bx = pr - by * (int)dnpw.d;
        const long tok = (long)b * gh * gw + (long)(by * patch + py) * gw + bx * patch + px;
        r.off[it] = tok * d + cb;
        r.st[it] = __ldg(reinterpret_cast<const float2*>(stats) + tok);
      }
    }
  }
  __device__ __forceinline__ const bf16* src(const Rows& r, int it, int, int c) const {
    return r.row + 8 * it < M ? X + r.off[it] + c : nullptr;
  }
  // piece `lane` of a chunk's 32 biases of s, then 32 of t; a lane's columns of it
  __device__ __forceinline__ const float* par_src(const Rows& r, int c, int lane) const {
    return bias + r.pbias + (lane & 8 ? d : 0) + c + 4 * (lane & 7);
  }
  __device__ __forceinline__ void params(Par& p, const uint8_t* par, int sp) const {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      *reinterpret_cast<float4*>(p.bs + 4 * i) =
          *reinterpret_cast<const float4*>(par + sp * 32 + 16 * i);
      *reinterpret_cast<float4*>(p.bt + 4 * i) =
          *reinterpret_cast<const float4*>(par + 128 + sp * 32 + 16 * i);
    }
  }
  __device__ __forceinline__ void apply(const Rows& r, const Par& p, int it, int, int c, float* fs,
                                        const float* ft, uint4 x) const {
    const int row = r.row + 8 * it;
    if (row >= M) return;
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
    float o[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float2 x2 = unpack_bf16(w[j >> 1]);
      const float xe = j & 1 ? x2.y : x2.x;
      const float sv = fs[j] + p.bs[j];
      fs[j] = sv;
      o[j] = fmaf(1.f + sv, (xe - r.st[it].x) * r.st[it].y, ft[j] + p.bt[j]);
    }
    *reinterpret_cast<uint4*>(X_out + r.off[it] + c) = pack8_bf16(o);
    const long pd = (long)patch * patch * d;
    *reinterpret_cast<uint4*>(S_save + (long)row * pd + r.pcol + c) = pack8_bf16(fs);
  }
};

// Compression input gradient of the 2D layer: rows are patches, columns
// (token p = c / d of the patch, channel c % d); the direct gradient comes from
// dXd (same patch order) and the sum is written to dX at the token's raster
// position (a 32-column chunk is 32 channels of one token: d % 32 == 0).
struct EpiDX2D : EpiRowsBase {
  struct Rows {
    long base[4];  // offset of the patch's top-left token in dX
    int row;
  };
  int M, N;
  const bf16* dXd;
  bf16* dX;
  int d, patch, gh, gw, m;
  FastDiv dm, dnpw, dpatch, dd;  // by m, patches per row, patch, d
  __device__ __forceinline__ void rows_info(Rows& r, int row, int) const {
    r.row = row;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int rr = row + 8 * it;
      const int b = dm.div(rr), pr = rr - b * m, by = dnpw.div(pr), bx = pr - by * (int)dnpw.d;
      r.base[it] = ((long)b * gh * gw + (long)by * patch * gw + bx * patch) * d;
    }
  }
  __device__ __forceinline__ const bf16* src(const Rows& r, int it, int n0, int c) const {
    const int row = r.row + 8 * it;
    return row < M ? dXd + (long)row * N + n0 + c : nullptr;
  }
  __device__ __forceinline__ bf16* dst(const Rows& r, int it, int n0, int c) const {
    const int col = n0 + c, p = dd.div(col), py = dpatch.div(p);
    const long ofs = ((long)py * gw + (p - py * patch)) * d + (col - p * d);
    return r.row + 8 * it < M ? dX + r.base[it] + ofs : nullptr;
  }
};

// Split-K partial: raw fp32 accumulator of split s written to
// part[(s * M + row) * N + col]; a reduce kernel applies the linear epilogue.
struct EpiPartial : EpiBase {
  static constexpr bool kSplitRows = true;
  struct Row {
    long off;
  };
  int N;
  float* part;
  __device__ __forceinline__ Row row_info(int erow, int) const {
    return Row{erow < 0 ? -1L : (long)erow * N};
  }
  __device__ __forceinline__ void apply(const Row& ri, int, int col, float* v, uint8_t*,
                                        int) const {
    if (ri.off < 0 || col >= N) return;
    float* o = part + ri.off + col;
#pragma unroll
    for (int i = 0; i < 32; i += 4)
      *reinterpret_cast<float4*>(o + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
  }
};

}  // namespace pf
