// Host side of the tcgen05 GEMM: TMA tensor maps, tile-width choice and the
// instantiations used by the layer (see gemm_tc.cuh for the kernel).
#include <cudaTypedefs.h>

#include <algorithm>

#include "gemm_tc.cuh"
#include "kernels.h"

namespace pf {

int take_dev_error_gemm() { return take_dev_error_tu(); }
int set_wait_limit_gemm(unsigned long long ns) { return set_wait_limit_tu(ns); }
int set_debug_skip_loads_gemm(int on) {
  return cudaMemcpyToSymbol(g_debug_skip_loads, &on, sizeof(on)) == cudaSuccess ? 0 : -1;
}

int num_sms() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 148;
  }
  return n;
}

namespace {

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (fn == nullptr) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// 2D bf16 map over a row-major [outer, inner] matrix with `ld` elements per
// row, 128-byte swizzle, zero fill outside the matrix.
bool make_map(CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer, uint64_t ld,
              uint32_t box_inner, uint32_t box_outer) {
  auto fn = encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {ld * 2};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// rows = M (for A) or N (for B).
bool make_operand_map(CUtensorMap* m, const Operand& op, int rows, int K) {
  // whole rows only; with none of them, the tail's map, which is zero past the tail
  const bool cut = op.full >= 0, none = op.full == 0;
  const uint64_t in = (uint64_t)(op.mn ? rows : K), out = (uint64_t)(op.mn ? K : rows);
  return make_map(m, op.ptr, none ? (uint64_t)op.tail : in,
                  none ? 1 : cut ? (uint64_t)op.full : out, (uint64_t)op.ld, 64, op.mn ? 64 : 128);
}

// The first `tail` columns of a matrix that ends inside a row: they have one row
// more than the others.
bool make_tail_map(CUtensorMap* m, const Operand& op) {
  return make_map(m, op.ptr, (uint64_t)op.tail, (uint64_t)op.full + 1, (uint64_t)op.ld, 64,
                  op.mn ? 64 : 128);
}

// The maps of a product: A, B, and of the one operand that ends inside a row (A if
// both are K-major, B if both are MN-major) the columns below `tail`.
struct Maps {
  CUtensorMap a, b, t;
  int tail;
};
// B of a direct epilogue: row n = 8 s + 2 g + e as dimensions (k, e, g, s); a box
// holds 32 rows of one g.
bool make_segment_map(CUtensorMap* m, const Operand& op, int rows, int K) {
  auto fn = encode_fn();
  if (fn == nullptr || op.mn || rows % 8 != 0) return false;
  const cuuint64_t row = (cuuint64_t)op.ld * 2;
  cuuint64_t dims[4] = {(cuuint64_t)K, 2, 4, (cuuint64_t)rows / 8};
  cuuint64_t strides[3] = {row, 2 * row, 8 * row};
  cuuint32_t box[4] = {64, 2, 1, 16};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(op.ptr), dims, strides, box,
            es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_maps(Maps* m, bool direct, int M, int N, int K, const Operand& A, const Operand& B) {
  if ((A.full >= 0 && (A.mn || B.mn)) || (B.full >= 0 && !(A.mn && B.mn)) || A.tail % 64 != 0 ||
      B.tail % 64 != 0 || (A.full == 0 && A.tail == 0) || (B.full == 0 && B.tail == 0))
    return false;
  if (!make_operand_map(&m->a, A, M, K) ||
      !(direct ? make_segment_map(&m->b, B, N, K) : make_operand_map(&m->b, B, N, K)))
    return false;
  const Operand& op = A.full > 0 ? A : B;
  m->tail = op.full > 0 ? op.tail : 0;
  m->t = m->a;  // unused below column 0
  return m->tail == 0 || make_tail_map(&m->t, op);
}

// Co-resident CTA pairs of the pair kernel (at most half the SMs).
template <class Kern>
int max_pairs(Kern kern, int threads, int smem) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (num_sms() / 2));
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    return 0;
  }
  return std::min(n, num_sms() / 2);
}

// How an M x N x K product is tiled: 128- or 256-wide tiles, on CTA pairs or
// not, K in S slices.
struct Plan {
  int bn = 128, S = 1;
  bool pair = false;
};

// Cycles of a plan, from measured rates: one 64-deep K block of a 128 x 128 tile
// takes a CTA 552 cycles, of a 128 x 256 tile 770, of a pair's 256 x 256 tile 656
// (the pair reads half as much shared memory per MMA and its ring is deeper); a
// wave of tiles costs about 1200 more to fill and hand over, and slices a pass of
// S + 1 fp32 matrices at 3300 bytes a cycle after another launch.  The split
// products of the 65536-token layer (M = N = 1024, K = 65536) take 124 + 10 us
// on 7 slices of 128-wide tiles, 90 + 11 on 9 of a pair's; M 4096, N 1024, K 8192
// takes 57 us on 128 single CTAs, 50 on 64 pairs.
constexpr int kPlanSms = 152;  // planning target (GB300); fixed so sizes are device-independent
double plan_cost(int M, int N, int K, int bn, bool pair, int S) {
  const long tm = pair ? 2 * GEMM_BM : GEMM_BM;
  const long tiles = ((N + bn - 1) / bn) * ((M + tm - 1) / tm) * S;
  const long units = pair ? kPlanSms / 2 : kPlanSms, waves = (tiles + units - 1) / units;
  const long nk = (K + GEMM_BK - 1) / GEMM_BK, kb = (nk + S - 1) / S;
  const double c = bn == 128 ? 552. : pair ? 656. : 770.;
  const double red = S > 1 ? 5000. + 4.0 * M * (double)N * (S + 1) / 3300. : 0.;
  return waves * (kb * c + 1200.) + red;
}

// K slices of at least 16 blocks that fill the SMs with 128 x 128 tiles (1: the tiles
// alone do).
int fill_slices(int M, int N, int K) {
  const long tiles = (long)((N + 127) / 128) * ((M + GEMM_BM - 1) / GEMM_BM);
  const int num_k = (K + GEMM_BK - 1) / GEMM_BK;
  if (tiles >= kPlanSms || num_k < 32) return 1;
  int best = 1;
  double best_eff = (double)tiles / kPlanSms;
  for (int S = 2; S <= 16 && num_k / S >= 16; ++S) {
    const long t = tiles * S;
    const double eff = (double)t / (((t + kPlanSms - 1) / kPlanSms) * kPlanSms);
    if (eff > best_eff + 1e-9) {
      best = S;
      best_eff = eff;
    }
  }
  return best;
}

// The cheapest plan whose slices' partial sums fit `bytes`: slices are at least
// 16 K blocks deep and must promise a tenth, since a last wave that is partly
// empty costs less than the model says (weight gradients of the 262144-token
// layer, 128 pair tiles in two waves: 320 us, on four slices 321 + 33).  If it has fewer
// than min_S slices, min_S on 128 x 128 tiles.
// Why min_S: each MMA cuts its 16 products' sum off at the accumulator's last bit, so a
// slice's error grows with its depth (2-norm, about 2^-26 of the result an MMA).  Where
// inputs are rounded to bf16 or the result is, that is lost beside 1e-3; in the proxies
// of a one-level compression nothing else is: 2565 patches of 24576 values, d = 384, are
// 8.9e-6 off float64 on three slices, 2.0e-6 on twelve.  Why 128 x 128 tiles then: the
// model leaves out the partial sums' stores, which short slices of wider tiles do not hide
// (product and sum, M 3624, N 512, K 16384: thirteen slices of 128-wide tiles 92 us, fifteen
// of a pair's 101).
Plan gemm_plan(int M, int N, int K, size_t bytes, int min_S) {
  Plan best;
  const long nk = (K + GEMM_BK - 1) / GEMM_BK;
  double cost = 1e300;
  for (int v = 0; v < 3; ++v) {
    const int bn = v == 0 ? 128 : 256;
    const bool pair = v == 2;
    if (v > 0 && N < 256) continue;
    for (int S = 1; S <= 32 && (S == 1 || (nk / S >= 16 && v != 1)); ++S) {
      if (S > 1 && (N % 4 != 0 || (size_t)S * M * N * sizeof(float) > bytes)) break;
      const double c = plan_cost(M, N, K, bn, pair, S) * (S > 1 ? 1.0 / 0.9 : 1.0);
      if (c < cost) {
        cost = c;
        best.bn = bn;
        best.pair = pair;
        best.S = S;
      }
    }
  }
  while (min_S > 1 && (N % 4 != 0 || (size_t)min_S * M * N * sizeof(float) > bytes)) --min_S;
  if (best.S < min_S) {
    best.bn = 128;
    best.pair = false;
    best.S = min_S;
  }
  return best;
}

template <int BN, bool AMN, bool BMN, class Epi>
cudaError_t launch(int M, int N, int K, const Maps& tm, const Epi& epi, cudaStream_t st,
                   const Plan& plan) {
  const int splits = plan.S;
  if constexpr (BN == 256) {  // CTA pairs: 256 x 256 tiles, half of B per CTA
    auto kern2 = gemm_tc_kernel<BN, AMN, BMN, Epi, true>;
    constexpr int smem2 = GemmCfg<BN, true, gemm_stage_bytes<Epi>(true)>::SMEM_BYTES;
    if (plan.pair) {
      cudaError_t e = cudaFuncSetAttribute(kern2, cudaFuncAttributeMaxDynamicSharedMemorySize, smem2);
      if (e != cudaSuccess) return e;
      static const int pairs = max_pairs(kern2, GEMM_THREADS, smem2);
      const long pair_tiles =
          (long)((N + BN - 1) / BN) * ((M + 2 * GEMM_BM - 1) / (2 * GEMM_BM)) * splits;
      if (pairs > 0)
        return launch_clusters(2, kern2, 2 * (unsigned)std::min<long>(pair_tiles, pairs),
                               GEMM_THREADS, smem2, st, tm.a, tm.b, tm.t, tm.tail, M, N, K, splits,
                               epi);
    }
  }
  auto kern = gemm_tc_kernel<BN, AMN, BMN, Epi>;
  constexpr int smem = GemmCfg<BN, false, gemm_stage_bytes<Epi>(false)>::SMEM_BYTES;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const long tiles = (long)((N + BN - 1) / BN) * ((M + GEMM_BM - 1) / GEMM_BM) * splits;
  const int grid = (int)std::min<long>(tiles, num_sms());
  return launch_kernel(kern, grid, GEMM_THREADS, smem, st, tm.a, tm.b, tm.t, tm.tail, M, N, K, splits,
                       epi);
}

// Operand majors that the epilogue's callers use: all four for the linear
// ones, K-major A (and for a direct one K-major B) for the fused ones.
template <int BN, class Epi>
cudaError_t launch_majors(int M, int N, int K, const Operand& A, const Operand& B, const Maps& tm,
                          const Epi& epi, cudaStream_t st, const Plan& plan) {
  if (!A.mn && !B.mn) return launch<BN, false, false>(M, N, K, tm, epi, st, plan);
  if constexpr (!Epi::kDirect)
    if (!A.mn && B.mn) return launch<BN, false, true>(M, N, K, tm, epi, st, plan);
  if constexpr (!Epi::kRows) {
    if (A.mn && B.mn) return launch<BN, true, true>(M, N, K, tm, epi, st, plan);
    return launch<BN, true, false>(M, N, K, tm, epi, st, plan);
  }
  return cudaErrorInvalidValue;
}

bool operand_ok(const Operand& op) {
  return op.ptr != nullptr && (reinterpret_cast<uintptr_t>(op.ptr) & 15) == 0 && op.ld > 0 &&
         (op.ld * 2) % 16 == 0;
}

template <class Epi>
cudaError_t gemm_dispatch(int M, int N, int K, Operand A, Operand B, const Epi& epi,
                          cudaStream_t st) {
  if (M <= 0 || N <= 0 || N % 32 != 0 || K < 0 || !operand_ok(A) || !operand_ok(B))
    return cudaErrorInvalidValue;
  Maps tm;
  if (!make_maps(&tm, Epi::kDirect, M, N, K, A, B)) return cudaErrorInvalidValue;
  LaunchTimer lt(gemm_tag_label(), st, 2.0 * M * N * (double)K,
                 2.0 * ((double)M * K + (double)N * K) + gemm_tag_bytes());
  Plan plan = gemm_plan(M, N, K, 0, 1);
  if constexpr (Epi::kPaired) {
    plan.bn = 256;
    plan.pair = plan_cost(M, N, K, 256, true, 1) <= plan_cost(M, N, K, 256, false, 1);
  } else if (plan.bn == 128) {
    return launch_majors<128>(M, N, K, A, B, tm, epi, st, plan);
  }
  return launch_majors<256>(M, N, K, A, B, tm, epi, st, plan);
}

// out = sum_s part[s] (+ bias) (+ addend) -> fp32 and/or bf16, 4 columns per thread.
__global__ void splitk_reduce_kernel(const float* __restrict__ part, int S, int M, int N,
                                     EpiLinearArgs e) {
  const int pz = pdl_enter();
  const long i = ((long)blockIdx.x * blockDim.x + threadIdx.x + pz) * 4;
  if (i >= (long)M * N) return;
  const long row = i / N;
  const int col = (int)(i % N);
  float4 v = *reinterpret_cast<const float4*>(part + i);
#pragma unroll 8
  for (int s = 1; s < S; ++s) {
    const float4 w = *reinterpret_cast<const float4*>(part + (long)s * M * N + i);
    v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
  }
  if (e.bias) {
    const float4 b = *reinterpret_cast<const float4*>(e.bias + col);
    v.x += b.x; v.y += b.y; v.z += b.z; v.w += b.w;
  }
  if (e.addend) {
    const float4 a = *reinterpret_cast<const float4*>(e.addend + row * e.ld_add + col);
    v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
  }
  if (e.add_bf16) {
    const uint2 u = *reinterpret_cast<const uint2*>(e.add_bf16 + row * e.ld_add_bf16 + col);
    const float2 a0 = unpack_bf16(u.x), a1 = unpack_bf16(u.y);
    v.x += a0.x; v.y += a0.y; v.z += a1.x; v.w += a1.y;
  }
  if (e.out_f32) *reinterpret_cast<float4*>(e.out_f32 + row * e.ld_f32 + col) = v;
  if (e.out_bf16)
    *reinterpret_cast<uint2*>(e.out_bf16 + row * e.ld_bf16 + col) =
        make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
}

}  // namespace

bool tmap_bf16_2d(CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer, uint64_t ld,
                  uint32_t box_inner, uint32_t box_outer) {
  return make_map(m, base, inner, outer, ld, box_inner, box_outer);
}

bool tmap_bf16_seq(CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer, uint64_t n_seq,
                   uint64_t ld, uint32_t box_inner, uint32_t box_outer) {
  auto fn = encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[3] = {inner, outer, n_seq};
  cuuint64_t strides[2] = {ld * 2, outer * ld * 2};
  cuuint32_t box[3] = {box_inner, box_outer, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t splitk_scratch_bytes(int M, int N, int K, int exact_in) {
  const int S = gemm_plan(M, N, K, ~size_t(0), exact_in ? fill_slices(M, N, K) : 1).S;
  return S > 1 ? (size_t)S * M * N * sizeof(float) : 0;
}
size_t splitk_scratch_bytes(int M, int N, int K) { return splitk_scratch_bytes(M, N, K, 0); }

size_t splitk_scratch_least(int M, int N, int K) {
  const int S = fill_slices(M, N, K);
  return S > 1 ? (size_t)S * M * N * sizeof(float) : 0;
}

cudaError_t gemm_linear(int M, int N, int K, Operand A, Operand B, const EpiLinearArgs& e,
                        cudaStream_t st) {
  Plan plan;
  if (e.splitk_scratch && !e.act_silu && !e.pre_bf16 && !e.dsilu_of)
    plan = gemm_plan(M, N, K, e.splitk_bytes, e.exact_in ? fill_slices(M, N, K) : 1);
  const int S = plan.S;
  if (S > 1) {
    // deterministic split-K: raw partials, then one reduce applying the epilogue
    if (M <= 0 || N % 32 != 0 || !operand_ok(A) || !operand_ok(B)) return cudaErrorInvalidValue;
    Maps tm;
    if (!make_maps(&tm, false, M, N, K, A, B)) return cudaErrorInvalidValue;
    EpiPartial epi{{}, N, e.splitk_scratch};
    {
      LaunchTimer lt(gemm_tag_label(), st, 2.0 * M * N * (double)K,
                     2.0 * ((double)M * K + (double)N * K) + 4.0 * S * M * N);
      const cudaError_t err =
          plan.bn == 256 ? launch_majors<256>(M, N, K, A, B, tm, epi, st, plan)
                         : launch_majors<128>(M, N, K, A, B, tm, epi, st, plan);
      if (err != cudaSuccess) return err;
    }
    LaunchTimer lt("splitk_reduce", st, (double)S * M * N, 4.0 * (S + 1.0) * M * N);
    const long quads = (long)M * N / 4;
    return launch_kernel(splitk_reduce_kernel, (unsigned)((quads + 255) / 256), 256, 0, st,
                         e.splitk_scratch, S, M, N, e);
  }
  if (e.add_bf16) {  // bf16 sum of the product and a bf16 matrix, nothing else
    if (((uintptr_t)e.add_bf16 & 15) || e.ld_add_bf16 % 8 || !e.out_bf16 || e.ld_bf16 % 8 ||
        e.bias || e.addend || e.out_f32 || e.act_silu || e.pre_bf16 || e.dsilu_of || A.mn)
      return cudaErrorInvalidValue;
    EpiAddRows epi{{}, M, N, e.add_bf16, e.ld_add_bf16, e.out_bf16, e.ld_bf16};
    return gemm_dispatch(M, N, K, A, B, epi, st);
  }
  if ((e.pre_bf16 && ((uintptr_t)e.pre_bf16 & 15 || e.ld_pre % 8)) ||
      (e.dsilu_of && ((uintptr_t)e.dsilu_of & 15 || e.ld_dsilu % 8)))
    return cudaErrorInvalidValue;
  // a short contraction with a plain (bias) epilogue stores whole rows from a
  // shared-memory stage: its output, not its mainloop, would bound it
  if (K <= 2048 && !e.addend && !e.act_silu && !e.pre_bf16 && !e.dsilu_of &&
      (e.out_f32 == nullptr || e.ld_f32 % 4 == 0) && (e.out_bf16 == nullptr || e.ld_bf16 % 8 == 0)) {
    EpiLinearStaged epi{{}, M, N, e.bias, e.out_f32, e.ld_f32, e.out_bf16, e.ld_bf16};
    return gemm_dispatch(M, N, K, A, B, epi, st);
  }
  EpiLinear epi{{},         M,          N,          e.bias,      e.addend,  e.ld_add,
                e.out_f32,  e.ld_f32,   e.out_bf16, e.ld_bf16,   e.act_silu, e.pre_bf16,
                e.ld_pre,   e.dsilu_of, e.ld_dsilu};
  return gemm_dispatch(M, N, K, A, B, epi, st);
}

cudaError_t gemm_inject1d(int M, int N, int K, Operand A, Operand B, const EpiInjectArgs& e,
                          cudaStream_t st) {
  EpiInject1D epi{{}, M, N, e.bias, e.D_save, e.X, e.X_out, e.w_x, e.w_dlt, e.b_g,
                  e.d, e.k1, e.k2, e.m, e.L, e.shift, e.gated, FastDiv(e.k2), FastDiv(e.m), FastDiv(e.d)};
  if (A.mn || B.mn || e.d % 32 != 0) return cudaErrorInvalidValue;
  return gemm_dispatch(M, N, K, A, B, epi, st);
}

cudaError_t gemm_dx1d(int M, int N, int K, Operand A, Operand B, const EpiDXArgs& e,
                      cudaStream_t st) {
  EpiDX1D epi{{}, M, N, e.dX, e.d, e.k1, e.L, FastDiv(e.m * e.k2)};
  if (A.mn || !B.mn || e.d % 8 != 0) return cudaErrorInvalidValue;
  return gemm_dispatch(M, N, K, A, B, epi, st);
}

cudaError_t gemm_append_kv(int M, int N, int K, Operand A, Operand B, const EpiAppendArgs& e,
                           cudaStream_t st) {
  EpiAppendKV epi{{}, M, N, e.K, e.V, e.n_open, e.n_proxy, e.d, e.P, e.cap};
  if (A.mn || B.mn) return cudaErrorInvalidValue;
  return gemm_dispatch(M, N, K, A, B, epi, st);
}

cudaError_t gemm_affine2d(int M, int N, int K, Operand A, Operand B, const EpiAffine2DArgs& e,
                          cudaStream_t st) {
  EpiAffine2D epi{{}, M, e.bias, e.S_save, e.X, e.X_out, e.stats, e.d, e.patch, e.gh, e.gw, e.m,
                  FastDiv(e.m), FastDiv(e.gw / e.patch), FastDiv(e.patch), FastDiv(e.d >> 7)};
  if (A.mn || B.mn || e.d % 128 != 0) return cudaErrorInvalidValue;
  return gemm_dispatch(M, N, K, A, B, epi, st);
}

cudaError_t gemm_dx2d(int M, int N, int K, Operand A, Operand B, const EpiDX2DArgs& e,
                      cudaStream_t st) {
  EpiDX2D epi{{},   M,     N,    e.dXd,        e.dX,
              e.d,  e.patch, e.gh, e.gw,         e.m,
              FastDiv(e.m), FastDiv(e.gw / e.patch), FastDiv(e.patch), FastDiv(e.d)};
  if (A.mn || !B.mn || e.d % 32 != 0) return cudaErrorInvalidValue;
  return gemm_dispatch(M, N, K, A, B, epi, st);
}

}  // namespace pf
