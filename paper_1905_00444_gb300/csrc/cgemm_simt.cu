// One contraction step as a complex FP32 GEMM on the FMA pipes (the plain path): one
// launch per step, one CTA per output tile (tile body in cgemm_tile.cuh).  Two CTAs per SM
// (at most 128 registers a thread): against one CTA with 8 x 8 outputs a thread, K = N = 256
// over 2^19 columns went from 4.96 to 4.64 ms (55.4 to 59.2 TFLOP/s) and K = N = 64 over 2^21
// columns from 1.63 to 1.25 ms (42 to 55).
#include <cuda_runtime.h>

#include <cstdio>

#include "cgemm_tile.cuh"
#include "launch.cuh"
#include "qfx_internal.h"

namespace qfx {
namespace {
using namespace simt;

__device__ __forceinline__ void simt_cp_async8(float2* smem, const float2* gmem) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gmem));
}

template <int BM, int BJ, int TM, int TJ, bool KMODE>
__global__ void __launch_bounds__(256, 2) cgemm_step_kernel(const StepArgs a) {
  launch_wait();
  launch_next();
  extern __shared__ float4 smem_raw[];
  cgemm_tile<BM, BJ, TM, TJ, KMODE>(a, blockIdx.x, blockIdx.y, smem_raw);
}

// A grid of at most one CTA per SM asks for more than half of an SM's shared memory, so that no two
// of its CTAs share an SM.  Such a grid is chosen for it (fill_variant), but CTAs that start early
// take the slots that the kernel before leaves, two on some SMs, and then the step takes twice its
// time: K = 128, N = 64 over 16384 columns in 128 CTAs behind K = 64 in 256 47 us, and 26 so; a call of
// 6x5x(1+28+1) 923 us and 684.
constexpr size_t kOwnSm = 116 << 10;

// Shared-memory opt-in of one tile kernel, once per device (also called ahead of a graph
// capture, which must not be the first launch to set it).
template <int BM, int BJ, int TM, int TJ, bool KMODE>
int ensure_attr() {
  static_assert(Cfg<BM, BJ, TM, TJ, KMODE>::SMEM <= kOwnSm, "a tile fits its request");
  static int attr_done[64] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && !attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(cgemm_step_kernel<BM, BJ, TM, TJ, KMODE>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOwnSm);
    if (e != cudaSuccess) return (int)e;
    attr_done[dev] = 1;
  }
  return 0;
}

template <int BM, int BJ, int TM, int TJ, bool KMODE>
int launch_cfg(const StepArgs& a, int batch, cudaStream_t stream) {
  using C_ = Cfg<BM, BJ, TM, TJ, KMODE>;
  auto kern = cgemm_step_kernel<BM, BJ, TM, TJ, KMODE>;
  if (int e = ensure_attr<BM, BJ, TM, TJ, KMODE>()) return e;
  const int64_t NT = (a.N + BM - 1) / BM;
  const int64_t JT = (a.J + BJ - 1) / BJ;
  const int64_t blocks = NT * JT;
  if (blocks > 0x7fffffffLL || batch > 65535) return (int)cudaErrorInvalidConfiguration;
  count_launch();
  const size_t smem = blocks * batch <= num_sms() ? kOwnSm : C_::SMEM;
  return (int)launch_early(kern, dim3((unsigned)blocks, batch), dim3(256), smem, stream, a);
}

// Chunk products of a split-K contraction with a small result: part c is the N x Sd product
// (at most kPartsOut outputs) of rows [c * chunk, (c + 1) * chunk) of S and B.  A thread owns one
// output and walks its chunk's k in order, with the operations of the step tiles, so the
// result is theirs bit for bit.  The step tiles would fill a row of 512 columns with Sd of them
// (N = Sd = 8, 2048 chunks of 1024: 1.50 ms; here 0.11); a block takes kPartsOut / (N * Sd)
// chunks, and slabs of KB rows of both operands arrive by cp.async in two buffers.  The floor is
// their reading (268 MB, 40 us); the chain of a chunk's k adds to it.
constexpr int kPartsOut = 256;
__global__ void __launch_bounds__(kPartsOut) small_parts_kernel(const float2* S, const float2* B, float2* part, int chunk,
                                                               int64_t parts, int N, int Sd, int KB) {
  launch_wait();
  launch_next();
  extern __shared__ __align__(16) float2 slab[];
  const int out = N * Sd, per_block = kPartsOut / out, row = N + Sd;
  const int own = threadIdx.x / out, e = threadIdx.x - own * out, n = e / Sd, s = e - n * Sd;
  const int64_t c0 = (int64_t)blockIdx.x * per_block;
  const int here = (int)min((int64_t)per_block, parts - c0);
  // buffer: per chunk of the block, KB rows of S, then KB rows of B
  auto fetch = [&](int k0, int buf) {
    float2* dst = slab + (int64_t)buf * per_block * KB * row;
    const int rows = min(KB, chunk - k0);
    for (int w = 0; w < here; ++w) {
      const int64_t k = (c0 + w) * chunk + k0;
      for (int i = threadIdx.x; i < rows * N; i += kPartsOut)
        simt_cp_async8(dst + (int64_t)w * KB * row + i, S + k * N + i);
      for (int i = threadIdx.x; i < rows * Sd; i += kPartsOut)
        simt_cp_async8(dst + (int64_t)w * KB * row + KB * N + i, B + k * Sd + i);
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  float re = 0.f, im = 0.f;
  fetch(0, 0);
  for (int k0 = 0, buf = 0; k0 < chunk; k0 += KB, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;\n" ::);
    __syncthreads();   // this slab landed for every thread; the other buffer is free
    if (k0 + KB < chunk) fetch(k0 + KB, buf ^ 1);
    if (own < here) {
      const float2* Sk = slab + ((int64_t)buf * per_block + own) * KB * row;
      const float2* Bk = Sk + KB * N;
      const int rows = min(KB, chunk - k0);
#pragma unroll 8
      for (int k = 0; k < rows; ++k) {
        const float2 a = Sk[k * N + n], b = Bk[k * Sd + s];
        re = fmaf(a.x, b.x, re);
        re = fmaf(-a.y, b.y, re);
        im = fmaf(a.x, b.y, im);
        im = fmaf(a.y, b.x, im);
      }
    }
  }
  if (own < here) part[(c0 + own) * out + e] = make_float2(re, im);
}

// Split-K sum of a chunked contraction.  A block covers E consecutive outputs with kRedL lanes
// each: lane l of an output adds chunks l, l + kRedL, ... in FP64, then lane 0 adds the lanes'
// sums in lane order and rounds once to FP32.  FP64 conversions and additions run at two lanes
// a clock on an SM, so few outputs take blocks of 4 of them, spread over the SMs (64 outputs
// of 2048 chunks: 42 us, against 78 in blocks of 32); many take 32, whose warps read longer runs.
constexpr int kRedL = 8;
template <int E>
__global__ void __launch_bounds__(E * kRedL) reduce_parts_kernel(const float2* part,
                                                                 int64_t part_stride, int64_t parts,
                                                                 int64_t out, float2* C, int64_t c_stride) {
  launch_wait();
  launch_next();
  __shared__ double2 lanes[kRedL][E];
  const int el = threadIdx.x % E, lane = threadIdx.x / E;
  const int64_t e = (int64_t)blockIdx.x * E + el;
  const float2* pp = part + (int64_t)blockIdx.y * part_stride;
  double re = 0.0, im = 0.0;
  if (e < out) {
#pragma unroll 8
    for (int64_t c = lane; c < parts; c += kRedL) {
      const float2 v = pp[c * out + e];
      re += (double)v.x;
      im += (double)v.y;
    }
  }
  lanes[lane][el] = make_double2(re, im);
  __syncthreads();
  if (lane == 0 && e < out) {
    for (int l = 1; l < kRedL; ++l) {
      re += lanes[l][el].x;
      im += lanes[l][el].y;
    }
    C[(int64_t)blockIdx.y * c_stride + e] = make_float2((float)re, (float)im);
  }
}

}  // namespace

int launch_reduce_parts(const void* part, int64_t part_stride, int64_t parts, int64_t out, void* C,
                        int64_t c_stride, int batch, void* stream) {
  if (parts < 1 || out < 1 || batch < 1 || batch > 65535) return (int)cudaErrorInvalidValue;
  const bool few = out <= 32 * (int64_t)num_sms();
  const int64_t blocks = few ? (out + 3) / 4 : (out + 31) / 32;
  if (blocks > 0x7fffffffLL) return (int)cudaErrorInvalidConfiguration;
  auto kern = few ? reduce_parts_kernel<4> : reduce_parts_kernel<32>;
  count_launch();
  return (int)launch_early(kern, dim3((unsigned)blocks, (unsigned)batch), dim3((few ? 4 : 32) * kRedL), 0,
                           (cudaStream_t)stream, (const float2*)part, part_stride, parts, out, (float2*)C, c_stride);
}

// Whether launch_small_parts takes a split-K contraction of this result.
bool small_parts_fit(int64_t N, int64_t Sd) { return N * Sd <= kPartsOut; }

int launch_small_parts(const void* S, const void* B, void* part, int64_t chunk, int64_t parts, int64_t N,
                       int64_t Sd, void* stream) {
  if (!small_parts_fit(N, Sd) || chunk < 1 || chunk > (1 << 20) || parts < 1) return (int)cudaErrorInvalidValue;
  const int per_block = kPartsOut / (int)(N * Sd);
  const int64_t blocks = (parts + per_block - 1) / per_block;
  if (blocks > 0x7fffffffLL) return (int)cudaErrorInvalidConfiguration;
  // rows per slab: two buffers in at most 40 KB (N + Sd <= 257 and per_block = 1 at the widest)
  const int row = (int)(N + Sd) * per_block * 8;
  int KB = 64;
  while (KB > 1 && 2 * KB * row > (40 << 10)) KB /= 2;
  count_launch();
  return (int)launch_early(small_parts_kernel, dim3((unsigned)blocks), dim3(kPartsOut), (size_t)2 * KB * row,
                           (cudaStream_t)stream, (const float2*)S, (const float2*)B, (float2*)part, (int)chunk,
                           parts, (int)N, (int)Sd, KB);
}

int simt_prepare_attributes() {
#define QFX_ATTR(V, BM, BJ, TM, TJ, KM) \
  if (int e = ensure_attr<BM, BJ, TM, TJ, KM>()) return e;
  QFX_SIMT_VARIANTS(QFX_ATTR)
  QFX_SIMT_FILL_VARIANTS(QFX_ATTR)
#undef QFX_ATTR
  return 0;
}

// Tile variants (QFX_SIMT_VARIANTS): 0..4 stream B along s in column pairs (JMODE), 5..9 take
// any Sd.  N >= 64 takes the 64-row tile also where 128 rows fit: it re-reads B from L2 and
// still runs at 59.1 TFLOP/s against 57.4 at K = N = 256 (the 128-row tile, left to the
// autotuner, has half as many columns in flight).
int pick_variant(int64_t N, int64_t Sd) {
  int base = N >= 64 ? 1 : N >= 32 ? 2 : N >= 16 ? 3 : 4;
  return base + ((Sd % 2) ? 5 : 0);
}

int num_sms() {
  static int n[64] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 64) dev = 63;
  if (!n[dev]) cudaDeviceGetAttribute(&n[dev], cudaDevAttrMultiProcessorCount, dev);
  return n[dev] > 0 ? n[dev] : 1;
}

// Variants 0..9 keep their tile when its grid gives more than three CTAs to two SMs (8 x 4096
// columns, K = N = 64, 256 CTAs: 25.9 us, 26.0 with 64 x 64).  A smaller grid is bound by the latency
// of a tile's k loop, and the CTAs that share an SM take about as long as one after another: the
// step takes the tile of least time.  A tile's times, alone on its SM and for each of those that
// share one, are relative to 64 x 64 alone (105 us at K = 1024 and even Sd, 117 odd), for even and for
// odd Sd; they are fitted to 1300 steps of K = 16 to 1024, N = 2 to 512, 64 to 80000 columns.  The
// choice is 0.2% slower than each step's fastest tile on geometric mean, and 11% faster than the
// first tile that gives more CTAs than SMs (852 columns of K = 1024, N = 512: 106 us with 32 x 128 and
// 112 CTAs, 136 with 16 x 128 and 224).  Where K < 32 loads and stores count more than the loop, and
// CTAs that share an SM hide one another's: their times count 0.65 (all amplitudes of 4x4x(1+16+1)
// 110.7 us, 113.4 without; measured with slabs of 8 rows k in all tiles).
// Every tile sums an output's k terms in the same order, so the choice never changes a result.
int fill_variant(int variant, int64_t K, int64_t N, int64_t J, int batch) {
  struct Tile { int bm, bj, alone[2], shared[2]; };
  static const Tile base[5] = {{128, 64, {180, 220}, {172, 172}}, {64, 128, {180, 220}, {172, 172}},
                               {32, 256, {217, 217}, {200, 200}}, {16, 256, {120, 140}, {125, 125}},
                               {8, 512, {145, 193}, {180, 180}}};
  static const Tile fill[5] = {{64, 64, {100, 100}, {97, 97}}, {32, 128, {102, 102}, {107, 107}},    // 20..24, 25..29
                               {16, 128, {72, 72}, {74, 68}}, {8, 256, {73, 94}, {80, 80}},
                               {8, 128, {44, 44}, {46, 46}}};
  if (variant < 0 || variant > 9 || batch < 1) return variant;
  const int64_t sms = num_sms();
  const int odd = variant >= 5;
  auto ctas = [&](const Tile& t) { return ((N + t.bm - 1) / t.bm) * ((J + t.bj - 1) / t.bj) * batch; };
  auto time = [&](const Tile& t) {
    const int64_t on_sm = (ctas(t) + sms - 1) / sms;
    return on_sm == 1 ? (int64_t)t.alone[odd] : on_sm * t.shared[odd] * (K < 32 ? 65 : 100) / 100;
  };
  const Tile& own = base[variant % 5];
  int64_t least = time(own);
  if (2 * ctas(own) > 3 * sms) return variant;
  int best = variant;
  for (int i = 0; i < 5; ++i) {
    if (fill[i].bm > own.bm || time(fill[i]) >= least) continue;
    least = time(fill[i]);
    best = 20 + i + 5 * odd;
  }
  return best;
}

bool simt_variant_valid(int variant, int64_t Sd) {
  const bool jmode = (variant >= 0 && variant < 5) || (variant >= 20 && variant < 25);
  const bool kmode = (variant >= 5 && variant < 10) || (variant >= 25 && variant < 30);
  return (jmode && Sd % 2 == 0) || kmode;
}

int launch_step(const void* S, int64_t s_stride, const void* B, int64_t b_stride, void* C,
                int64_t c_stride, int64_t P, int64_t K, int64_t N, int64_t NL, int64_t Sd,
                int batch, int variant, int precision, void* stream, int beta) {
  (void)precision;
  StepArgs a{(const float2*)S, s_stride, (const float2*)B, b_stride, (float2*)C, c_stride,
             P, K, N, NL, Sd, P * Sd, beta};
  if (variant < 0) variant = pick_variant(N, Sd);
  if (!simt_variant_valid(variant, Sd)) return (int)cudaErrorInvalidValue;  // JMODE needs even Sd
  cudaStream_t st = (cudaStream_t)stream;
  switch (variant) {
#define QFX_CASE(V, BM, BJ, TM, TJ, KM) \
  case V: return launch_cfg<BM, BJ, TM, TJ, KM>(a, batch, st);
    QFX_SIMT_VARIANTS(QFX_CASE)
    QFX_SIMT_FILL_VARIANTS(QFX_CASE)
#undef QFX_CASE
    default: return (int)cudaErrorInvalidValue;
  }
}

}  // namespace qfx
