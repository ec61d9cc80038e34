// One contraction step on the 5th-generation tensor cores (tcgen05, TMEM accumulators),
// with complex FP32 operands split into lower-precision terms.
//
//   C[nh][p][nl][s] = sum_k S[k][nh*NL + nl] * B[p][k][s]     (Sec. III.E, Eq. 1)
//
// The paper ran this product as complex FP32 CGEMM without tensor cores, because FP16
// inputs lose too much precision (Sec. III.E).  Here each FP32 real operand x is split
// into terms of a tensor-core type and the complex product is formed from real products
// (4M: Re = Ar Sr - Ai Si, Im = Ar Si + Ai Sr), each real product being the sum of the
// cross products of the terms whose magnitude is above FP32 rounding:
//   BF16x3: x = h + m + l (successive round-to-nearest residuals), products
//           hh, hm, mh, hl, lh, mm  (error ~2^-24 relative);
//   TF32x3: x = b + s, products bb, bs, sb  (error ~2^-21 relative).
// Accumulation is FP32 in TMEM.
//
// Tiles: the boundary tensor B is the A operand (rows j), the site matrix S the B operand
// (rows n), pre-split once per step by split_site_kernel into the shared-memory image of its
// term planes.  Default tiles are 256 rows j by Nt <= 128 columns n on a pair of CTAs
// (cgemm_pair_kernel), or for short contractions 128 rows on one CTA (cgemm_cta_kernel), with
// split accumulators in TMEM: hi x hi products go to "main" accumulators, every cross-term
// product to "small" ones, added in the epilogue, so that the large accumulators see two
// additions per k-step.  There the complex product is embedded in N: S is held per term as planes
// Sr, Si, -Sr, and one MMA of N = 2 Nt takes Ar x [Sr; Si] into (re, im) and another
// -Ai x [Si; -Sr], so each MMA reads A once for both halves.
// QFX_TC_FAST_ACCUMULATION tiles (cgemm_cta_kernel too) are 128 x 256 with one accumulator pair
// (re [0,256), im [256,512)) and four real products per term pair (4M).
// The kernels are persistent: producer warps split FP32 rows of B into term planes (K-major,
// no-swizzle core-matrix layout), one thread issues the MMAs, others stream the site image with
// bulk copies and, for default tiles, the rows of B with tensor-map copies into staging buffers
// when the shape allows it, and epilogue warps drain TMEM into C.
// Rings of shared-memory stages are guarded by mbarriers.  Every wait has a deadline;
// on expiry the kernel records an error, drains its own copies and MMAs, frees TMEM and
// returns (the host reports QFX_ETIMEOUT).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>

#include "launch.cuh"
#include "ptx_async.cuh"
#include "qfx_internal.h"

namespace qfx {

__device__ unsigned int g_tc_status = 0;

namespace {

using namespace ptx;

constexpr int kRows = 128;        // UMMA M
constexpr int kPlaneA = kRows * 32;   // bytes of one A term plane per stage
constexpr unsigned long long kWaitNs = 1000000000ull;   // 1 s per wait

template <int MODE>
struct Mode;
template <>
struct Mode<QFX_PREC_C3M_BF16X3> {
  static constexpr int TERMS = 3, KS = 16, NPROD = 6;
  static constexpr uint32_t FMT = 1;   // BF16
  __device__ static constexpr int ta(int i) { return i == 0 ? 1 : i == 1 ? 0 : i == 2 ? 2 : i == 3 ? 0 : i == 4 ? 1 : 0; }
  __device__ static constexpr int tb(int i) { return i == 0 ? 1 : i == 1 ? 2 : i == 2 ? 0 : i == 3 ? 1 : i == 4 ? 0 : 0; }
};
template <>
struct Mode<QFX_PREC_C3M_BF16X2> {
  static constexpr int TERMS = 2, KS = 16, NPROD = 3;
  static constexpr uint32_t FMT = 1;   // BF16: h, m with products hm, mh, hh (~2^-16)
  __device__ static constexpr int ta(int i) { return i == 0 ? 0 : i == 1 ? 1 : 0; }
  __device__ static constexpr int tb(int i) { return i == 0 ? 1 : i == 1 ? 0 : 0; }
};
template <>
struct Mode<QFX_PREC_C3M_TF32X3> {
  static constexpr int TERMS = 2, KS = 8, NPROD = 3;
  static constexpr uint32_t FMT = 2;   // TF32
  __device__ static constexpr int ta(int i) { return i == 0 ? 0 : i == 1 ? 1 : 0; }
  __device__ static constexpr int tb(int i) { return i == 0 ? 1 : i == 1 ? 0 : 0; }
};

// ---- term splitting ------------------------------------------------------------
// T BF16 terms of two numbers, packed (x0 in the low half): each the round-to-nearest of what
// the previous ones left
template <int T>
__device__ __forceinline__ void split_bf16x2(float x0, float x1, uint32_t t[T]) {
#pragma unroll
  for (int i = 0; i < T; ++i) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(t[i]) : "f"(x1), "f"(x0));
    if (i + 1 < T) {
      x0 -= __uint_as_float(t[i] << 16);
      x1 -= __uint_as_float(t[i] & 0xffff0000u);
    }
  }
}
__device__ __forceinline__ uint32_t to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void split_tf32x2(float x, uint32_t t[2]) {
  t[0] = to_tf32(x);
  t[1] = to_tf32(x - __uint_as_float(t[0]));
}

// Writes the KS values of one row (component c of `v`) as TERMS planes of 32 bytes each.
// Row r of a plane lives at (r/8)*256 + kc*128 + (r%8)*16 (8x16-byte core matrices;
// kc = which 16-byte half of the row).
template <int MODE>
__device__ __forceinline__ void store_row_terms(char* plane0, int plane_bytes, int row,
                                                const float* x) {
  using M_ = Mode<MODE>;
  const int base = (row >> 3) * 256 + (row & 7) * 16;
  if constexpr (M_::FMT == 1) {   // BF16 terms, 16 per row
    constexpr int T = M_::TERMS;
    uint32_t w[T][8];
#pragma unroll
    for (int k = 0; k < 16; k += 2) {
      uint32_t a[T];
      split_bf16x2<T>(x[k], x[k + 1], a);
#pragma unroll
      for (int t = 0; t < T; ++t) w[t][k / 2] = a[t];
    }
#pragma unroll
    for (int t = 0; t < T; ++t) {
      char* pl = plane0 + t * plane_bytes + base;
      *reinterpret_cast<uint4*>(pl) = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
      *reinterpret_cast<uint4*>(pl + 128) = make_uint4(w[t][4], w[t][5], w[t][6], w[t][7]);
    }
  } else {
    uint32_t w[2][8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      uint32_t a[2];
      split_tf32x2(x[k], a);
      w[0][k] = a[0];
      w[1][k] = a[1];
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      char* pl = plane0 + t * plane_bytes + base;
      *reinterpret_cast<uint4*>(pl) = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
      *reinterpret_cast<uint4*>(pl + 128) = make_uint4(w[t][4], w[t][5], w[t][6], w[t][7]);
    }
  }
  (void)sizeof(M_);
}

// One 16-byte half (kc) of a row's KS values as TERMS planes, for producers that share a row.
template <int MODE>
__device__ __forceinline__ void store_half_terms(char* plane0, int row, int kc, const float* x) {
  constexpr int T = Mode<MODE>::TERMS;
  char* pl = plane0 + (row >> 3) * 256 + kc * 128 + (row & 7) * 16;
  uint32_t w[T][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t t[T];
    if constexpr (Mode<MODE>::FMT == 1) split_bf16x2<T>(x[2 * i], x[2 * i + 1], t);
    else split_tf32x2(x[i], t);
#pragma unroll
    for (int q = 0; q < T; ++q) w[q][i] = t[q];
  }
#pragma unroll
  for (int q = 0; q < T; ++q)
    *reinterpret_cast<uint4*>(pl + q * kPlaneA) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
}

// ---- PTX helpers -----------------------------------------------------------------
// Bounded wait: false if the deadline passed or another role gave up.  Roles off the
// critical path pass sleep_ns > 0 so that their polling does not take issue slots from
// the producers.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort,
                                          unsigned sleep_ns = 0) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long deadline = globaltimer() + kWaitNs;
  while (!mbar_try(bar, parity)) {
    if (*abort) return false;
    if (globaltimer() > deadline) {
      *abort = 1;
      atomicOr(&g_tc_status, 1u);
      return false;
    }
    if (sleep_ns) __nanosleep(sleep_ns);
  }
  return true;
}
// Waits for work already in flight (copies, MMAs), whatever the abort flag says: after a timeout
// it is still on its way, and neither TMEM nor the CTA may go before it has ended.
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity, unsigned long long limit_ns,
                                           unsigned sleep_ns = 0) {
  if (mbar_try(bar, parity)) return;
  const unsigned long long deadline = globaltimer() + limit_ns;
  while (!mbar_try(bar, parity) && globaltimer() < deadline)
    if (sleep_ns) __nanosleep(sleep_ns);
}
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  // K-major, no swizzle: LBO = 128 B (next core matrix along K), SBO = 256 B (next
  // 8-row group); bits 46-48 = 0b001; base offset 0; layout type 0.
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(128 >> 4) << 16) |
         ((uint64_t)(256 >> 4) << 32) | (1ull << 46);
}
template <int MODE>
__device__ __forceinline__ uint32_t instr_desc(int n, bool neg_a) {
  // D = F32 (bits 4-5 = 1), A/B format (bits 7-9, 10-12), negate A (bit 13),
  // both K-major (bits 15, 16 = 0), N >> 3 (bits 17-22), M >> 4 (bits 24-28).
  return (1u << 4) | (Mode<MODE>::FMT << 7) | (Mode<MODE>::FMT << 10) | ((neg_a ? 1u : 0u) << 13) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
}
template <int MODE>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if constexpr (Mode<MODE>::FMT == 1) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
  } else {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
  }
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}


__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// ---- CTA pairs -------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// every thread of both CTAs, at points that each reaches (all waits before them are bounded)
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// Arrives on the barrier at this shared-memory offset in CTA 0 of the pair.  The planes that it
// stands for are ordered by their writers' proxy fences, the TMEM reads by the tcgen05 fence.  Its
// own order is the default one, a release within the CTA: that the other CTA sees what lies before
// it rests on the customary use of this form for CTA pairs and on tests that compare every bit, not
// on the memory model's words.  Release and acquire at cluster scope wait for the thread's other
// stores, those of C among them.  us with the default / with cluster scope in the producers / in all
// arrivals and waits: BF16x3 K = N = 256 over 2^19 columns 876 / 928 / 978, K = N = 64 over 2^21 406 /
// 528 / 548, TF32x3 K = N = 256 866 / 970 / 1002, a BF16x2 chunk of K = 1024 473 / 781 / 790.
__device__ __forceinline__ void mbar_arrive_leader(uint32_t bar) {
  asm volatile(
      "{\n.reg .b32 r;\nmapa.shared::cluster.u32 r, %0, 0;\n"
      "mbarrier.arrive.shared::cluster.b64 _, [r];\n}" ::"r"(bar) : "memory");
}
template <int MODE>
__device__ __forceinline__ uint32_t instr_desc_pair(int n, bool neg_a) {   // M = 256 over both CTAs
  return instr_desc<MODE>(n, neg_a) + ((uint32_t)(kRows >> 4) << 24);
}
template <int MODE>
__device__ __forceinline__ void mma_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if constexpr (Mode<MODE>::FMT == 1) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
  } else {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
  }
}
// one arrival on the barrier at this offset in both CTAs once the MMAs issued so far are done
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"((uint16_t)3) : "memory");
}

// x / d and x % d in 32 bits where they hold it (a 64-bit division takes over a hundred clocks)
__device__ __forceinline__ void divmod(int64_t x, int64_t d, int64_t& q, int64_t& r) {
  if (((uint64_t)x | (uint64_t)d) >> 32) {
    q = x / d;
    r = x - q * d;
  } else {
    const uint32_t q32 = (uint32_t)x / (uint32_t)d;
    q = q32;
    r = (uint32_t)x - q32 * (uint32_t)d;
  }
}

struct TcArgs {
  const float2* B; int64_t b_stride;
  float2* C; int64_t c_stride;
  const char* simage; int64_t img_stride;   // pre-split S, per item
  int64_t P, K, N, NL, Sd, J;
  int Nt;            // columns n per tile (<= 128 split accumulators, <= 256 single)
  int NHt;           // tiles along n per 128-row tile
  int64_t JT;        // 128-row tiles per item (256-row ones for pairs)
  int64_t tiles;     // total tiles (items x JT x NHt)
  int sd_shift;      // log2 Sd where Sd is a power of two, else -1
  int withhold_s;    // test hook: never stream S, so the bounded waits expire
  int use_tma;       // pair tiles: producers read FP32 rows staged by tensor-map copies
  int stages, nbuf;  // pair tiles: operand stages and staging buffers
  int box_s, box_p;  // tensor-map box: box_s consecutive s (columns), box_p values of p
  int beta;          // 1: add the product into C (a chunk of a long contraction)
};

// Operand stages start on 128-byte boundaries (tensor-map copies land there; the dynamic
// window itself is only 16-byte aligned behind the static shared variables).
constexpr uint32_t kAlignPad = 128;

// Tile t -> (item g, 128-row tile jt, column tile nh).  Within an item the column tiles
// come in bands of kBand; inside a band the column tile runs fastest, so the tiles in
// flight at once (one per CTA) share a few column slices of the S image and a few row
// tiles of B in L2 (with N = 8192 one k-chunk of the S image alone is 151 MB).  With
// NHt <= kBand this is the plain order, column tile fastest.
constexpr int64_t kBand = 8;
__device__ __forceinline__ void tile_coords(const TcArgs& a, int64_t t, int64_t& g, int64_t& jt,
                                            int64_t& nh) {
  int64_t r = t, band;
  g = 0;
  if (a.tiles > a.JT * a.NHt) divmod(t, a.JT * a.NHt, g, r);
  int64_t n0 = 0, w = a.NHt;
  if (a.NHt > kBand) {
    divmod(r, kBand * a.JT, band, r);
    n0 = band * kBand;
    w = a.NHt - n0 < kBand ? a.NHt - n0 : kBand;
  }
  jt = r;
  nh = n0;
  if (w > 1) {
    divmod(r, w, jt, r);
    nh = n0 + r;
  }
}
// row index j = p * Sd + s
__device__ __forceinline__ void split_row(const TcArgs& a, int64_t j, int64_t& p, int64_t& s) {
  if (a.sd_shift >= 0) {
    p = j >> a.sd_shift;
    s = j & (a.Sd - 1);
  } else {
    divmod(j, a.Sd, p, s);
  }
}

// ---- tiles on one CTA -------------------------------------------------------------------
// 128 rows j on one CTA per SM.  SPLIT: default accumulation of steps of few k-steps
// (takes_cta_tile), Nt <= 128, main accumulators in TMEM columns [0, 2 Nt), small ones in [256,
// 256 + 2 Nt), each re then im.  Otherwise fast accumulation, Nt <= 256: re in [0, Nt), im in [256,
// 256 + Nt).  Warps: 0-3 producers, 4-11 epilogue (two per TMEM lane quarter, each half the
// columns), 12 TMEM owner + MMA issuer, 13 site stream and tensor-map copies.
template <int MODE, bool SPLIT>
struct CtaCfg {
  using M_ = Mode<MODE>;
  static constexpr int NT_MAX = SPLIT ? 128 : 256;
  static constexpr int PLANES = 2 * M_::TERMS;             // planes of B per stage
  static constexpr int SPLANES = SPLIT ? 3 * M_::TERMS : PLANES;   // and of S
  static constexpr int STAGES = SPLIT ? (M_::TERMS == 3 ? 3 : 4) : 3;
  static constexpr int STAGE_A = PLANES * kPlaneA;
  static constexpr int STAGE_IN = kRows * M_::KS * 8;
  // staging buffers of tensor-map copies; the operand ring of the fast tile leaves no room for them
  static constexpr int NBUF = SPLIT ? (M_::KS == 16 ? 2 : 4) : 0;
  static constexpr int THREADS = 14 * 32;
  static size_t smem(int nt) {
    return kAlignPad + (size_t)STAGES * (STAGE_A + SPLANES * nt * 32) + (size_t)NBUF * STAGE_IN +
           (3 * STAGES + 3 + 2 * NBUF) * sizeof(uint64_t);
  }
};

template <int MODE, bool SPLIT>
__global__ void __launch_bounds__(CtaCfg<MODE, SPLIT>::THREADS, 1)
    cgemm_cta_kernel(const TcArgs a, const __grid_constant__ CUtensorMap tmA) {
  using M_ = Mode<MODE>;
  using CF = CtaCfg<MODE, SPLIT>;
  constexpr int TERMS = M_::TERMS, KS = M_::KS, STAGES = CF::STAGES;
  extern __shared__ __align__(16) char smem_raw[];
  char* smem = smem_raw + ((kAlignPad - (smem_u32(smem_raw) & (kAlignPad - 1))) & (kAlignPad - 1));
  const int stageA = CF::STAGE_A;
  const int planeS = a.Nt * 32;
  const int stageS = CF::SPLANES * planeS;
  char* sA = smem;
  char* sS = smem + STAGES * stageA;
  char* sIn = sS + STAGES * stageS;                 // NBUF x [box_p][KS][box_s] float2
  uint64_t* bars = reinterpret_cast<uint64_t*>(sIn + CF::NBUF * CF::STAGE_IN);
  // bars: fullA[S], fullS[S], empty[S], acc_full, tmem_free, done, in_full[NBUF], in_empty[NBUF]
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t KT = a.K / KS;

  auto fullA = [&](int s) { return smem_u32(&bars[s]); };
  auto fullS = [&](int s) { return smem_u32(&bars[STAGES + s]); };
  auto empty = [&](int s) { return smem_u32(&bars[2 * STAGES + s]); };
  const uint32_t acc_full = smem_u32(&bars[3 * STAGES]);
  const uint32_t tmem_free = smem_u32(&bars[3 * STAGES + 1]);
  const uint32_t done = smem_u32(&bars[3 * STAGES + 2]);
  auto in_full = [&](int b) { return smem_u32(&bars[3 * STAGES + 3 + b]); };
  auto in_empty = [&](int b) { return smem_u32(&bars[3 * STAGES + 3 + CF::NBUF + b]); };

  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(fullA(s), kRows);
      mbar_init(fullS(s), 1);
      mbar_init(empty(s), 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(tmem_free, 8);
    mbar_init(done, 1);
    for (int b = 0; b < CF::NBUF; ++b) {
      mbar_init(in_full(b), 1);
      mbar_init(in_empty(b), kRows);
    }
    mbar_init_fence();
  }
  launch_wait();       // the site image is written; before the TMEM, which an earlier kernel may hold
  launch_next();
  __syncwarp();
  if (warp == 12) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_base_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base_slot;
  volatile int* abort = &abort_flag;

  if (warp < 4) {
    // ---- producers: split 128 rows of B per k-stage into term planes -------------------
    // Rows arrive through tensor-map copies staged NBUF k-stages ahead (issued by warp 13), or
    // through loads issued one k-stage ahead into registers, so that their latency overlaps the
    // split and the wait for a free operand stage.
    int64_t t = blockIdx.x, it = 0, q = 0;
    if (CF::NBUF > 0 && a.use_tma) {
      constexpr int NB = CF::NBUF > 0 ? CF::NBUF : 1;
      const int ps = tid / a.box_s, ss = tid % a.box_s;     // this row inside the box
      while (t < a.tiles && !*abort) {
        const int b = (int)(q % NB);
        if (!mbar_wait(in_full(b), (uint32_t)((q / NB) & 1), abort)) break;
        const float2* in = reinterpret_cast<const float2*>(sIn + b * CF::STAGE_IN);
        float re[KS], im[KS];
#pragma unroll
        for (int kk = 0; kk < KS; ++kk) {
          const float2 v = in[(ps * KS + kk) * a.box_s + ss];
          re[kk] = v.x;
          im[kk] = v.y;
        }
        // the next tensor-map copy rewrites this buffer through the async proxy: order these
        // generic reads before it
        fence_async_smem();
        mbar_arrive(in_empty(b));
        const int s = (int)(q % STAGES);
        if (q >= STAGES && !mbar_wait(empty(s), (uint32_t)((q / STAGES - 1) & 1), abort)) break;
        char* st = sA + s * stageA;
        store_row_terms<MODE>(st, kPlaneA, tid, re);
        store_row_terms<MODE>(st + TERMS * kPlaneA, kPlaneA, tid, im);
        fence_async_smem();
        mbar_arrive(fullA(s));
        ++q;
        if (++it == KT) { it = 0; t += gridDim.x; }
      }
    } else {
    auto row_ptr = [&](int64_t tt, int64_t& pofs) -> const float2* {
      int64_t g, jt, nh;
      tile_coords(a, tt, g, jt, nh);
      const int64_t jg = jt * kRows + tid;
      int64_t p, sidx;
      split_row(a, jg, p, sidx);
      pofs = jg < a.J ? p * a.K * a.Sd + sidx : -1;
      return a.B + g * a.b_stride;
    };
    float2 nxt[KS];
    auto fetch = [&](int64_t tt, int64_t ii) {
      int64_t pofs;
      const float2* Bg = row_ptr(tt, pofs);
#pragma unroll
      for (int kk = 0; kk < KS; ++kk)
        nxt[kk] = pofs >= 0 ? Bg[pofs + (ii * KS + kk) * a.Sd] : make_float2(0.f, 0.f);
    };
    if (t < a.tiles) fetch(t, 0);
    while (t < a.tiles && !*abort) {
      float re[KS], im[KS];
#pragma unroll
      for (int kk = 0; kk < KS; ++kk) { re[kk] = nxt[kk].x; im[kk] = nxt[kk].y; }
      int64_t nt = t, ni = it + 1;
      if (ni == KT) { nt = t + gridDim.x; ni = 0; }
      if (nt < a.tiles) fetch(nt, ni);
      const int s = (int)(q % STAGES);
      if (q >= STAGES && !mbar_wait(empty(s), (uint32_t)((q / STAGES - 1) & 1), abort)) break;
      char* st = sA + s * stageA;
      store_row_terms<MODE>(st, kPlaneA, tid, re);
      store_row_terms<MODE>(st + TERMS * kPlaneA, kPlaneA, tid, im);
      fence_async_smem();
      mbar_arrive(fullA(s));
      ++q;
      t = nt;
      it = ni;
    }
    }
  } else if (warp == 13) {
    // ---- S image stream ------------------------------------------------------------
    if (lane == 0) {
      int64_t q = 0, issued = 0;
      bool ok = !a.withhold_s;
      for (int64_t t = blockIdx.x; t < a.tiles && ok; t += gridDim.x) {
        int64_t g, jt, nh;
        tile_coords(a, t, g, jt, nh);
        const char* img = a.simage + g * a.img_stride;
        for (int64_t it = 0; it < KT; ++it, ++q) {
          const int s = (int)(q % STAGES);
          if (q >= STAGES && !mbar_wait(empty(s), (uint32_t)((q / STAGES - 1) & 1), abort, 32)) { ok = false; break; }
          mbar_arrive_tx(fullS(s), (uint32_t)stageS);
          bulk_copy(smem_u32(sS + s * stageS), img + (it * a.NHt + nh) * stageS, (uint32_t)stageS, fullS(s));
          issued = q + 1;
        }
      }
      // drain: every issued copy must land before the CTA exits
      for (int64_t i = (issued > STAGES ? issued - STAGES : 0); i < issued; ++i) {
        mbar_drain(fullS((int)(i % STAGES)), (uint32_t)((i / STAGES) & 1), kWaitNs);
      }
    } else if (lane == 1 && CF::NBUF > 0 && a.use_tma) {
      // ---- FP32 rows of B: one tensor-map copy per (tile, k-stage) into staging --------
      constexpr int NB = CF::NBUF > 0 ? CF::NBUF : 1;
      int64_t q = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < a.tiles && ok; t += gridDim.x) {
        int64_t g, jt, nh, p, sidx;
        tile_coords(a, t, g, jt, nh);
        split_row(a, jt * kRows, p, sidx);
        for (int64_t it = 0; it < KT; ++it, ++q) {
          const int b = (int)(q % NB);
          if (q >= NB && !mbar_wait(in_empty(b), (uint32_t)((q / NB - 1) & 1), abort, 32)) { ok = false; break; }
          mbar_arrive_tx(in_full(b), (uint32_t)CF::STAGE_IN);
          tma_load_4d(smem_u32(sIn + b * CF::STAGE_IN), &tmA, (int)sidx, (int)(it * KS), (int)p, (int)g, in_full(b));
        }
      }
      for (int64_t i = (q > NB ? q - NB : 0); i < q; ++i)
        mbar_drain(in_full((int)(i % NB)), (uint32_t)((i / NB) & 1), kWaitNs);
    }
  } else if (warp == 12) {
    // ---- MMA issue -----------------------------------------------------------------
    if (lane == 0) {
      int64_t q = 0, tc = 0;
      bool ok = true;
      const int n_mma = SPLIT ? 2 * a.Nt : a.Nt;
      const uint32_t idesc_p = instr_desc<MODE>(n_mma, false), idesc_n = instr_desc<MODE>(n_mma, true);
      for (int64_t t = blockIdx.x; t < a.tiles && ok; t += gridDim.x, ++tc) {
        if (tc > 0 && !mbar_wait(tmem_free, (uint32_t)((tc - 1) & 1), abort)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        bool started[2] = {false, false};
        for (int64_t it = 0; it < KT; ++it, ++q) {
          const int s = (int)(q % STAGES);
          const uint32_t par = (uint32_t)((q / STAGES) & 1);
          if (!mbar_wait(fullA(s), par, abort) || !mbar_wait(fullS(s), par, abort)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a0 = smem_u32(sA + s * stageA), b0 = smem_u32(sS + s * stageS);
          if constexpr (SPLIT) {
            // Ar x [Sr; Si] -> (re, im) += (Ar Sr, Ar Si);  (-Ai) x [Si; -Sr] -> += (-Ai Si, Ai Sr)
#pragma unroll
            for (int ca = 0; ca < 2; ++ca) {
#pragma unroll
              for (int pi = 0; pi < M_::NPROD; ++pi) {
                const int acc = M_::ta(pi) == 0 && M_::tb(pi) == 0 ? 0 : 1;   // hi x hi products: main
                const uint64_t ad = smem_desc(a0 + (ca * TERMS + M_::ta(pi)) * kPlaneA);
                const uint64_t bd = smem_desc(b0 + (3 * M_::tb(pi) + ca) * planeS);
                mma<MODE>(tmem + (uint32_t)(acc * 256), ad, bd, ca ? idesc_n : idesc_p, started[acc] ? 1u : 0u);
                started[acc] = true;
              }
            }
          } else {   // 4M with re in TMEM columns [0, Nt) and im in [256, 256 + Nt)
#pragma unroll
            for (int rp = 0; rp < 4; ++rp) {
              const int ca = (rp == 0 || rp == 2) ? 0 : 1;          // Ar, Ai, Ar, Ai
              const int cb = (rp == 0 || rp == 3) ? 0 : 1;          // Sr, Si, Si, Sr
              const int to_im = rp >= 2 ? 1 : 0;
              const uint32_t idesc = rp == 1 ? idesc_n : idesc_p;   // - Ai Si
#pragma unroll
              for (int pi = 0; pi < M_::NPROD; ++pi) {
                const uint64_t ad = smem_desc(a0 + (ca * TERMS + M_::ta(pi)) * kPlaneA);
                const uint64_t bd = smem_desc(b0 + (cb * TERMS + M_::tb(pi)) * planeS);
                mma<MODE>(tmem + (uint32_t)(to_im * 256), ad, bd, idesc, started[to_im] ? 1u : 0u);
                started[to_im] = true;
              }
            }
          }
          mma_commit(empty(s));
        }
        if (ok) mma_commit(acc_full);
      }
      mma_commit(done);
    }
  } else {
    // ---- epilogue (warps 4-11): TMEM -> C ----------------------------------------------
    const int quarter = warp & 3, half = (warp - 4) >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    // 16-column chunks alternate between the two warps of a lane quarter
    const int nchunks = a.Nt / 16;
    const int my_last = ((nchunks - 1 - half) >= 0) ? (nchunks - 1 - ((nchunks - 1 - half) & 1)) : -1;
    int64_t tc = 0;
    for (int64_t t = blockIdx.x; t < a.tiles; t += gridDim.x, ++tc) {
      const bool ok = __all_sync(0xffffffffu, mbar_wait(acc_full, (uint32_t)(tc & 1), abort, 256) && !*abort);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      int64_t g, jt, nh;
      tile_coords(a, t, g, jt, nh);
      const int64_t jg = jt * kRows + row;
      const bool valid = jg < a.J;
      float2* Cg = a.C + g * a.c_stride;
      int64_t p, sidx;
      split_row(a, jg, p, sidx);
      const int64_t jofs = p * a.NL * a.Sd + sidx;
      const int64_t strideNH = a.P * a.NL * a.Sd;
      if (my_last < 0) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(tmem_free);
      }
      for (int ci = half; ci < nchunks; ci += 2) {
        const int c0 = ci * 16;
        float vr[16], vi[16];
        if (SPLIT) {
          float sr[16], si[16];
          tmem_ld16(tmem + lane_base + c0, vr);
          tmem_ld16(tmem + lane_base + a.Nt + c0, vi);
          tmem_ld16(tmem + lane_base + 256 + c0, sr);
          tmem_ld16(tmem + lane_base + 256 + a.Nt + c0, si);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int i = 0; i < 16; ++i) { vr[i] += sr[i]; vi[i] += si[i]; }
        } else {
          tmem_ld16(tmem + lane_base + c0, vr);
          tmem_ld16(tmem + lane_base + 256 + c0, vi);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        }
        if (ci == my_last) {
          // last TMEM read of this tile by this warp: hand the columns back to the MMA
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(tmem_free);
        }
        if (valid) {
          // one division per chunk, then step along n with a carry into nh (a 64-bit
          // division per element cost more than the MMAs of the tile)
          const int n0 = (int)nh * a.Nt + c0, NL = (int)a.NL;
          int nl = n0 % NL;
          float2* dst = Cg + (int64_t)(n0 / NL) * strideNH + (int64_t)nl * a.Sd + jofs;
          if (!a.beta) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              *dst = make_float2(vr[i], vi[i]);
              dst += a.Sd;
              if (++nl == NL) { nl = 0; dst += strideNH - (int64_t)NL * a.Sd; }
            }
          } else {   // a chunk of a long contraction: add into C
            // all 16 reads first: one memory latency per chunk, not one per element
            float2 o[16];
            float2* d = dst;
            int l = nl;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              o[i] = __ldcg(d);
              d += a.Sd;
              if (++l == NL) { l = 0; d += strideNH - (int64_t)NL * a.Sd; }
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              *dst = make_float2(vr[i] + o[i].x, vi[i] + o[i].y);
              dst += a.Sd;
              if (++nl == NL) { nl = 0; dst += strideNH - (int64_t)NL * a.Sd; }
            }
          }
        }
      }
    }
  }

  if (warp == 12) mbar_drain(done, 0, kWaitNs, 256);   // last MMAs finished before freeing TMEM
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 12) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// ---- default tiles on CTA pairs ------------------------------------------------------
// Two CTAs of a cluster (the two SMs of a TPC) compute 256 rows j x Nt columns n together:
// one tcgen05.mma.cta_group::2 of M = 256 takes 128 rows of B from each CTA and half of the
// 2 Nt rows of the embedded site operand from each, so an SM's shared memory holds and feeds
// its tensor core half of that operand (Sr and Si in CTA 0, Si and -Sr in CTA 1), where a
// CTA by itself reads all of it for every MMA.  Per BF16x3 k-step and SM at Nt = 128 that is
//   MMA reads 12 x (4 + 4) KB, site stream 24 KB, term planes 24 KB, staging 2 x 16 KB:
//   176 KB = 1375 clk at 128 B/clk against 1638 clk of MMA at the measured rate,
// where a single CTA moves 236 KB = 1844 clk.  Measured against such a single CTA (K = N = 256,
// 2^19 columns): one cool launch takes 0.82 ms (0.83 of the tensor probe) against 0.98; run
// for seconds both are held by the 1400 W limit, 0.96 against 1.07 ms for BF16x3 and 0.91
// against 1.02 for TF32x3; BF16x2 at K = N = 1024 over 2^15 columns went from 0.67 to 0.50 ms.
//
// With 4 Nt <= 256 the accumulators of two tiles fit the TMEM (the halves of its 512
// columns): the MMAs of a tile run while the epilogue stores the one before.  At Nt = 128
// they take turns, and the MMAs wait until the epilogue has read them.  Its stores back up
// (100 clk for each of 256 bytes, with every SM storing at once), so it reads ahead of them:
// with registers taken over from the other roles it holds 5 chunks of 8 columns beside the one
// it stores, and hands the TMEM back after the third of its 8 chunks.
//
// Roles, in each CTA on its own 128 rows: warps 0-7 producers, 8 TMEM owner and MMA issuer, 9
// site stream, 10 tensor-map copies, 12-19 epilogue (two per TMEM lane quarter).  CTA 0 (the
// leader) issues every MMA; its barriers collect the arrivals of both CTAs, and the commits
// arrive on the barriers of both.  Warp 8 of CTA 1 passes the arrival of its site copies on to
// the leader.
// A CTA leaves only after the cluster barrier at the end, when nothing refers to it any more.
template <int MODE>
struct PairCfg {
  using M_ = Mode<MODE>;
  static constexpr int NT_MAX = 128;
  // k-steps (of one MMA per product) in an operand stage: the fence, arrivals and waits of a
  // stage cost its roles 500 to 800 clk, which the 6 MMAs of a two-term k-step (819 clk) barely
  // cover.  Two k-steps of TF32 take the bytes of one of BF16 (K = N = 256 over 2^19 columns:
  // 984 -> 903 us when it was chosen); two of BF16x2 leave room for two stages only (490 -> 515
  // us at K = 1024).
  static constexpr int SUB = M_::KS == 8 ? 2 : 1;
  static constexpr int PLANES = 2 * M_::TERMS;              // planes of each operand per k-step
  static constexpr int STAGE_A = SUB * PLANES * kPlaneA;
  static constexpr int STAGE_IN = kRows * SUB * M_::KS * 8;
  static constexpr int MAX_STAGES = 8, MAX_BUF = 8;
  static constexpr int NBARS = 3 * MAX_STAGES + 5 + 2 * MAX_BUF;
  static constexpr int THREADS = 20 * 32;
  static size_t smem(int nt, int stages, int nbuf) {
    return kAlignPad + (size_t)stages * (STAGE_A + SUB * PLANES * nt * 32) + (size_t)nbuf * STAGE_IN +
           NBARS * sizeof(uint64_t);
  }
};

// Position in a ring of `n` slots and the parity of its current pass.
struct Ring {
  int i = 0;
  uint32_t pass = 0;
  __device__ __forceinline__ void step(int n) {
    if (++i == n) { i = 0; pass ^= 1u; }
  }
};
template <int N>
__device__ __forceinline__ void reg_release() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void reg_take() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
// Barrier of the 8 producer warps; true for all of them where `p` holds for any.
__device__ __forceinline__ bool producers_any(bool p) {
  uint32_t r;
  __syncwarp();
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred q, 1, 256, p;\nselp.u32 %0, 1, 0, q;\n}"
      : "=r"(r) : "r"((uint32_t)p) : "memory");
  return r != 0;
}
// Registers per thread of the roles' warpgroups; the launch gives each of the five 96.
constexpr int kRegLaunch = 96, kRegProd = 72, kRegCtl = 48, kRegEpi = 144;
static_assert(2 * kRegProd + kRegCtl + 2 * kRegEpi <= 5 * kRegLaunch, "the roles share the launch's registers");

template <int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PairCfg<MODE>::THREADS, 1)
    cgemm_pair_kernel(const TcArgs a, const __grid_constant__ CUtensorMap tmA) {
  using M_ = Mode<MODE>;
  using CF = PairCfg<MODE>;
  constexpr int TERMS = M_::TERMS, KS = M_::KS, SUB = CF::SUB;
  extern __shared__ __align__(16) char smem_raw[];
  char* smem = smem_raw + ((kAlignPad - (smem_u32(smem_raw) & (kAlignPad - 1))) & (kAlignPad - 1));
  const int planeS = a.Nt * 32;
  const int stepS = CF::PLANES * planeS, stageS = SUB * stepS;
  const int stages = a.stages, nbuf = a.nbuf;
  char* sA = smem;
  char* sS = smem + stages * CF::STAGE_A;
  char* sIn = sS + stages * stageS;                 // nbuf x [box_p][SUB * KS][box_s] float2
  uint64_t* bars = reinterpret_cast<uint64_t*>(sIn + nbuf * CF::STAGE_IN);
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;
  __shared__ int site_pos, site_pass, site_issued;   // of the site stream at its end
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();
  const int k_steps = (int)(a.K / KS);                // the last stage of a tile may have fewer
  const int KT = (k_steps + SUB - 1) / SUB;
  const int n_acc = 4 * a.Nt <= 256 ? 2 : 1;         // tiles whose accumulators fit the TMEM

  const uint32_t bar0 = smem_u32(bars);
  auto full = [&](int s) { return bar0 + 8 * s; };                         // leader's: stage s of both CTAs
  auto fullS = [&](int s) { return bar0 + 8 * (CF::MAX_STAGES + s); };     // CTA 1's: its site copies
  auto empty = [&](int s) { return bar0 + 8 * (2 * CF::MAX_STAGES + s); };
  auto acc_full = [&](int c) { return bar0 + 8 * (3 * CF::MAX_STAGES + c); };
  auto tmem_free = [&](int c) { return bar0 + 8 * (3 * CF::MAX_STAGES + 2 + c); };   // leader's: both epilogues
  const uint32_t done = bar0 + 8 * (3 * CF::MAX_STAGES + 4);
  auto in_full = [&](int b) { return bar0 + 8 * (3 * CF::MAX_STAGES + 5 + b); };
  auto in_empty = [&](int b) { return bar0 + 8 * (3 * CF::MAX_STAGES + 5 + CF::MAX_BUF + b); };

  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < stages; ++s) {
      mbar_init(full(s), 4);         // the producers and the site copies of each CTA
      mbar_init(fullS(s), 1);
      mbar_init(empty(s), 1);
    }
    for (int c = 0; c < 2; ++c) {
      mbar_init(acc_full(c), 1);
      mbar_init(tmem_free(c), 16);   // 8 epilogue warps of each CTA
    }
    mbar_init(done, 1);
    for (int b = 0; b < nbuf; ++b) {
      mbar_init(in_full(b), 1);
      mbar_init(in_empty(b), 1);
    }
    mbar_init_fence();
  }
  __syncwarp();
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_base_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_barrier();   // barriers of both CTAs initialised, TMEM allocated in both
  launch_wait();       // the site image is written
  launch_next();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base_slot;
  volatile int* abort = &abort_flag;
  const int64_t pair0 = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  // tile t of the pair: a.JT counts 256-row tiles, this CTA has rows [128 jt, 128 jt + 128)
  auto coords = [&](int64_t t, int64_t& g, int64_t& jt, int64_t& nh) {
    tile_coords(a, t, g, jt, nh);
    jt = 2 * jt + rank;
  };

  if (warp < 8) {
    // ---- producers: split 128 rows of B per k-stage into term planes -------------------
    reg_release<kRegProd>();
    // Two threads share a row, each half of its k.  A barrier among the producers collects a
    // stage's reads and writes, and one thread's proxy fence behind it orders them all: the
    // operand planes before the MMAs that read them, the staging buffer's reads before the copy
    // that reuses it.  A fence in every warp held up the SM's other memory instructions, the
    // epilogue's stores above all (K = N = 256 over 2^19 columns, TF32x3: 1.02 -> 0.91 ms).
    constexpr int KH = KS / 2;
    const int prow = tid & (kRows - 1), kh = tid >> 7;
    const int64_t n_stages = pair0 < a.tiles ? ((a.tiles - pair0 + pairs - 1) / pairs) * KT : 0;
    Ring op;                    // operand stages
    float re[SUB][KH], im[SUB][KH];
    // re, im into the next operand stage, unless a wait ran out (`ok` false): then, at once for
    // all producers, false
    auto put = [&](bool ok) -> bool {
      if (ok) ok = mbar_wait(empty(op.i), op.pass ^ 1u, abort);
      if (ok) {
        char* st = sA + op.i * CF::STAGE_A;
#pragma unroll
        for (int u = 0; u < SUB; ++u) {
          store_half_terms<MODE>(st + u * CF::PLANES * kPlaneA, prow, kh, re[u]);
          store_half_terms<MODE>(st + (u * CF::PLANES + TERMS) * kPlaneA, prow, kh, im[u]);
        }
      }
      if (producers_any(!ok)) return false;
      if (tid == 0) {
        fence_async_smem();
        mbar_arrive_leader(full(op.i));
      }
      op.step(stages);
      return true;
    };
    if (a.use_tma) {
      const int ps = prow / a.box_s, ss = prow % a.box_s;     // this row inside the box
      const int in_ofs = (ps * SUB * KS + kh * KH) * a.box_s + ss;
      Ring in;
      for (int64_t q = 0; q < n_stages; ++q) {
        const bool ok = mbar_wait(in_full(in.i), in.pass, abort);
        if (ok) {
          const float2* src = reinterpret_cast<const float2*>(sIn + in.i * CF::STAGE_IN) + in_ofs;
#pragma unroll
          for (int u = 0; u < SUB; ++u)
#pragma unroll
            for (int kk = 0; kk < KH; ++kk) {   // rows past K arrive as zeros
              const float2 v = src[(u * KS + kk) * a.box_s];
              re[u][kk] = v.x;
              im[u][kk] = v.y;
            }
        }
        if (!put(ok)) break;
        if (tid == 0) mbar_arrive(in_empty(in.i));
        in.step(nbuf);
      }
    } else {
      // rows that no tensor map describes: loads issued one k-stage ahead into registers (not
      // the read-only path: the kernel that writes B may still run when this one starts)
      float2 nxt[SUB][KH];
      int64_t t = pair0;
      int it = 0;
      bool inside = false;
      const float2* src = nullptr;
      auto fetch = [&]() {
        if (it == 0) {
          int64_t g, jt, nh, p, sidx;
          coords(t, g, jt, nh);
          const int64_t jg = jt * kRows + prow;
          inside = jg < a.J;
          split_row(a, jg, p, sidx);
          src = a.B + g * a.b_stride + p * a.K * a.Sd + sidx + (int64_t)(kh * KH) * a.Sd;
        }
#pragma unroll
        for (int u = 0; u < SUB; ++u)
#pragma unroll
          for (int kk = 0; kk < KH; ++kk)
            nxt[u][kk] = inside && it * SUB + u < k_steps ? src[(u * KS + kk) * a.Sd] : make_float2(0.f, 0.f);
        src += SUB * KS * a.Sd;
        if (++it == KT) { it = 0; t += pairs; }
      };
      if (n_stages > 0) fetch();
      for (int64_t q = 0; q < n_stages; ++q) {
#pragma unroll
        for (int u = 0; u < SUB; ++u)
#pragma unroll
          for (int kk = 0; kk < KH; ++kk) { re[u][kk] = nxt[u][kk].x; im[u][kk] = nxt[u][kk].y; }
        if (q + 1 < n_stages) fetch();
        if (!put(true)) break;
      }
    }
  } else if (warp < 12) {
    reg_release<kRegCtl>();
    if (warp == 9 && lane == 0) {
      // ---- site image stream: per term the two planes of this CTA's half ---------------
      Ring st;
      int issued = 0;           // stages whose latest copy is this role's
      bool ok = !a.withhold_s;
      for (int64_t t = pair0; t < a.tiles && ok; t += pairs) {
        int64_t g, jt, nh;
        coords(t, g, jt, nh);
        const char* src = a.simage + g * a.img_stride + nh * (3 * TERMS) * planeS + rank * planeS;
        for (int it = 0; it < KT; ++it) {
          if (!mbar_wait(empty(st.i), st.pass ^ 1u, abort)) { ok = false; break; }
          const uint32_t bar = rank == 0 ? full(st.i) : fullS(st.i);
          const int subs = k_steps - it * SUB < SUB ? k_steps - it * SUB : SUB;
          mbar_arrive_tx(bar, (uint32_t)(subs * stepS));
          for (int u = 0; u < subs; ++u) {
#pragma unroll
            for (int tm = 0; tm < TERMS; ++tm)
              bulk_copy(smem_u32(sS + st.i * stageS + u * stepS + tm * 2 * planeS), src + (int64_t)tm * 3 * planeS,
                        (uint32_t)(2 * planeS), bar);
            src += (int64_t)a.NHt * (3 * TERMS) * planeS;
          }
          st.step(stages);
          if (issued < stages) ++issued;
        }
      }
      site_pos = st.i;
      site_pass = (int)st.pass;
      site_issued = issued;
    } else if (warp == 10 && lane == 0 && a.use_tma) {
      // ---- FP32 rows of B: one tensor-map copy per (tile, k-stage) into staging --------
      Ring in;
      int64_t issued = 0;
      bool ok = true;
      for (int64_t t = pair0; t < a.tiles && ok; t += pairs) {
        int64_t g, jt, nh, p, sidx;
        coords(t, g, jt, nh);
        split_row(a, jt * kRows, p, sidx);
        for (int it = 0; it < KT; ++it) {
          if (!mbar_wait(in_empty(in.i), in.pass ^ 1u, abort)) { ok = false; break; }
          mbar_arrive_tx(in_full(in.i), (uint32_t)CF::STAGE_IN);
          tma_load_4d(smem_u32(sIn + in.i * CF::STAGE_IN), &tmA, (int)sidx, it * SUB * KS, (int)p, (int)g, in_full(in.i));
          in.step(nbuf);
          ++issued;
        }
      }
      for (int64_t i = 0; i < (issued < nbuf ? issued : nbuf); ++i) {   // newest first
        in.i = in.i == 0 ? nbuf - 1 : in.i - 1;
        if (in.i == nbuf - 1) in.pass ^= 1u;
        mbar_drain(in_full(in.i), in.pass, kWaitNs);
      }
    } else if (warp == 8 && lane == 0 && rank == 0) {
      // ---- MMA issue -------------------------------------------------------------------
      Ring st, acc;
      bool ok = true;
      const uint32_t idesc_p = instr_desc_pair<MODE>(2 * a.Nt, false), idesc_n = instr_desc_pair<MODE>(2 * a.Nt, true);
      const uint32_t small = (uint32_t)(n_acc == 2 ? 2 * a.Nt : 256);
      for (int64_t t = pair0; t < a.tiles && ok; t += pairs) {
        if (!mbar_wait(tmem_free(acc.i), acc.pass ^ 1u, abort)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d0 = tmem + (uint32_t)(acc.i * 256);
        bool started[2] = {false, false};
        for (int it = 0; it < KT; ++it) {
          if (!mbar_wait(full(st.i), st.pass, abort)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int u = 0; u < SUB; ++u) {
            if (u > 0 && it * SUB + u >= k_steps) break;
            const uint32_t a0 = smem_u32(sA + st.i * CF::STAGE_A) + u * CF::PLANES * kPlaneA;
            const uint32_t b0 = smem_u32(sS + st.i * stageS) + u * stepS;
            // Ar x [Sr; Si] -> (re, im) += (Ar Sr, Ar Si);  (-Ai) x [Si; -Sr] -> += (-Ai Si, Ai Sr)
#pragma unroll
            for (int ca = 0; ca < 2; ++ca) {
#pragma unroll
              for (int pi = 0; pi < M_::NPROD; ++pi) {
                const int k = M_::ta(pi) == 0 && M_::tb(pi) == 0 ? 0 : 1;   // hi x hi products: main
                const uint64_t ad = smem_desc(a0 + (ca * TERMS + M_::ta(pi)) * kPlaneA);
                const uint64_t bd = smem_desc(b0 + (2 * M_::tb(pi) + ca) * planeS);
                mma_pair<MODE>(d0 + (k ? small : 0u), ad, bd, ca ? idesc_n : idesc_p, started[k] ? 1u : 0u);
                started[k] = true;
              }
            }
          }
          mma_commit_pair(empty(st.i));
          st.step(stages);
        }
        if (ok) mma_commit_pair(acc_full(acc.i));
        acc.step(n_acc);
      }
      mma_commit_pair(done);
    } else if (warp == 8 && lane == 0) {
      // ---- CTA 1: its site copies have landed ------------------------------------------
      Ring st;
      bool ok = true;
      for (int64_t t = pair0; t < a.tiles && ok; t += pairs)
        for (int it = 0; it < KT; ++it) {
          if (!mbar_wait(fullS(st.i), st.pass, abort)) { ok = false; break; }
          mbar_arrive_leader(full(st.i));
          st.step(stages);
        }
    }
    __syncwarp();
  } else {
    // ---- epilogue: TMEM -> C -----------------------------------------------------------
    reg_take<kRegEpi>();
    const int quarter = warp & 3, half = (warp - 12) >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    // 8-column chunks alternate between the two warps of a lane quarter: chunks half, half + 2,
    // ..., AHEAD of them in registers before the first is stored
    constexpr int MOST = CF::NT_MAX / 16, AHEAD = 5, RING = AHEAD + 1;
    const int mine = a.Nt / 16;
    const int N = (int)a.N, NL = (int)a.NL;
    const int64_t wrap = a.P * a.NL * a.Sd - (int64_t)NL * a.Sd;   // from the end of one nh to the next
    Ring acc;
    for (int64_t t = pair0; t < a.tiles; t += pairs) {
      // addresses first, while the MMAs of the tile run
      int64_t g, jt, nh, p, sidx;
      coords(t, g, jt, nh);
      const int64_t jg = jt * kRows + row;
      const bool valid = jg < a.J;
      split_row(a, jg, p, sidx);
      float2* Cj = a.C + g * a.c_stride + p * a.NL * a.Sd + sidx;
      if (!__all_sync(0xffffffffu, mbar_wait(acc_full(acc.i), acc.pass, abort))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t main0 = tmem + (uint32_t)(acc.i * 256) + lane_base;
      const uint32_t small0 = main0 + (uint32_t)(n_acc == 2 ? 2 * a.Nt : 256);
      float vr[RING][8], vi[RING][8];
      auto load = [&](int i, int buf) {   // main + small of this warp's chunk i
        const uint32_t c0 = (uint32_t)((half + 2 * i) * 8);
        float sr[8], si[8];
        tmem_ld8(main0 + c0, vr[buf]);
        tmem_ld8(main0 + a.Nt + c0, vi[buf]);
        tmem_ld8(small0 + c0, sr);
        tmem_ld8(small0 + a.Nt + c0, si);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int e = 0; e < 8; ++e) { vr[buf][e] += sr[e]; vi[buf][e] += si[e]; }
        if (i + 1 == mine) {   // this warp has read the accumulators: back to the MMAs
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive_leader(tmem_free(acc.i));
        }
      };
#pragma unroll
      for (int i = 0; i < AHEAD; ++i)
        if (i < mine) load(i, i);
#pragma unroll
      for (int i = 0; i < MOST; ++i) {
        if (i + AHEAD < MOST && i + AHEAD < mine) load(i + AHEAD, (i + AHEAD) % RING);
        if (i < mine && valid) {
          const int buf = i % RING;
          // columns n0 .. n0 + 7 of S: one division (none where n does not split) and, where the
          // chunk crosses from one nh to the next, a carry
          const int n0 = (int)nh * a.Nt + (half + 2 * i) * 8;
          const int nh0 = NL == N ? 0 : n0 / NL;
          int left = (nh0 + 1) * NL - n0;   // columns to the end of this nh
          float2* dst = Cj + nh0 * wrap + (int64_t)n0 * a.Sd;
          if (a.beta) {   // a chunk of a long contraction: add into C
            // all 8 reads first: one memory latency per chunk, not one per element.  Not the
            // read-only path, which is for memory that nothing writes during the kernel: this
            // kernel writes C, and the one of the chunk before may end after this one's start
            float2 o[8];
            const float2* d = dst;
            int l = left;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              o[e] = __ldcg(d);
              d += a.Sd;
              if (--l == 0) { l = NL; d += wrap; }
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) { vr[buf][e] += o[e].x; vi[buf][e] += o[e].y; }
          }
          if (left >= 8) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              *dst = make_float2(vr[buf][e], vi[buf][e]);
              dst += a.Sd;
            }
          } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              *dst = make_float2(vr[buf][e], vi[buf][e]);
              dst += a.Sd;
              if (--left == 0) { left = NL; dst += wrap; }
            }
          }
        }
      }
      acc.step(n_acc);
    }
  }

  __syncwarp();
  if (warp == 8 && rank == 0) mbar_drain(done, 0, kWaitNs, 256);   // last MMAs finished before freeing TMEM
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_barrier();   // the roles of both CTAs and all MMAs have ended
  if (warp == 9 && lane == 0 && *abort) {
    // after a timeout some site copies may have no MMA that waited for them
    Ring st{site_pos, (uint32_t)site_pass};
    for (int i = 0; i < site_issued; ++i) {   // newest first
      st.i = st.i == 0 ? stages - 1 : st.i - 1;
      if (st.i == stages - 1) st.pass ^= 1u;
      mbar_drain(rank == 0 ? full(st.i) : fullS(st.i), st.pass, kWaitNs / 100);
    }
  }
  if (warp == 8) {
    mbar_drain(done, 0, kWaitNs, 256);   // CTA 1: the last commit has arrived here as well
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
  cluster_barrier();   // neither CTA leaves while the other still frees its half or awaits an arrival
}

// Pre-split of the site matrix S[k][n] into the per-stage shared-memory image, per
// (stage ks, n tile), each plane [row n within the tile][32 bytes]:
//   EMB (default tiles): per term t the planes Sr_t, Si_t, -Sr_t, so that [Sr_t; Si_t]
//     and [Si_t; -Sr_t] are contiguous 2 Nt-row operands (complex product embedded in N);
//   otherwise: Sr terms then Si terms.
template <int MODE, bool EMB>
__global__ void __launch_bounds__(128) split_site_kernel(const float2* S, int64_t s_stride,
                                                          int K, int N, int Nt, char* image,
                                                          int64_t img_stride) {
  using M_ = Mode<MODE>;
  constexpr int TERMS = M_::TERMS, KS = M_::KS;
  launch_wait();
  launch_next();
  const int n = blockIdx.x * 128 + threadIdx.x;
  const int ks = blockIdx.y;
  const int g = blockIdx.z;
  if (n >= N) return;
  const float2* Sg = S + (int64_t)g * s_stride;
  float re[KS], im[KS];
#pragma unroll
  for (int kk = 0; kk < KS; ++kk) {
    const int k = ks * KS + kk;
    float2 v = make_float2(0.f, 0.f);
    if (k < K) v = Sg[(int64_t)k * N + n];
    re[kk] = v.x;
    im[kk] = v.y;
  }
  const int planeS = Nt * 32;
  const int nht = N / Nt, nh = n / Nt, r = n % Nt;
  constexpr int SPL = EMB ? 3 * TERMS : 2 * TERMS;
  char* st = image + (int64_t)g * img_stride + ((int64_t)ks * nht + nh) * SPL * planeS;
  if constexpr (EMB) {
    store_row_terms<MODE>(st, 3 * planeS, r, re);
    store_row_terms<MODE>(st + planeS, 3 * planeS, r, im);
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) re[kk] = -re[kk];
    store_row_terms<MODE>(st + 2 * planeS, 3 * planeS, r, re);
  } else {
    store_row_terms<MODE>(st, planeS, r, re);
    store_row_terms<MODE>(st + TERMS * planeS, planeS, r, im);
  }
}

// Whether tiles of 128 rows do not straddle p unevenly and the inner extent of a tensor map's box
// is at least 16 bytes.
bool rows_fit_map(int64_t Sd) { return Sd >= 2 && (Sd % 128 == 0 || 128 % Sd == 0); }

// Tensor map over B viewed as (s, k, p, item) 8-byte elements, box (box_s, ks, box_p, 1)
// = one 128-row, ks-deep k-stage of a tile.  False if the shape does not allow it.
bool make_b_map(CUtensorMap* map, const void* B, int64_t b_stride, int batch, int64_t P, int64_t K,
                int64_t Sd, int ks, int* box_s, int* box_p) {
  auto enc = tensor_map_encoder();
  if (!enc || !rows_fit_map(Sd)) return false;
  const int bs = (int)(Sd < 128 ? Sd : 128), bp = 128 / bs;
  const cuuint64_t dims[4] = {(cuuint64_t)Sd, (cuuint64_t)K, (cuuint64_t)P, (cuuint64_t)batch};
  const cuuint64_t item = (cuuint64_t)(batch > 1 ? b_stride : P * K * Sd) * 8;
  const cuuint64_t strides[3] = {(cuuint64_t)Sd * 8, (cuuint64_t)(K * Sd) * 8, item};
  const cuuint32_t box[4] = {(cuuint32_t)bs, (cuuint32_t)ks, (cuuint32_t)bp, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  if (((uintptr_t)B & 15) || (item & 15)) return false;
  const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, const_cast<void*>(B), dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  *box_s = bs;
  *box_p = bp;
  return true;
}

// Staging buffers (16 KB each) of a pair tile, and as many operand stages as the rest of the
// shared memory holds: 3 buffers, but 2 for TF32, whose 64 KB stages then number 3 at Nt = 128
// instead of 2 (K = N = 256 over 2^19 columns: 903 us against 946; BF16x3 927 with 2 buffers and
// 926 with 3, at K = N = 64 over 2^21 columns 446 and 433).
constexpr int kMaxSmem = 227 << 10;   // per CTA, the kernels' static variables included
constexpr int kStaticSmem = 64;
template <int MODE>
void pair_rings(int nt, int* stages, int* nbuf) {
  using PC = PairCfg<MODE>;
  *nbuf = PC::SUB == 1 ? 3 : 2;
  *stages = 2;
  while (*stages < PC::MAX_STAGES && PC::smem(nt, *stages + 1, *nbuf) + kStaticSmem <= kMaxSmem) ++*stages;
}

// Shared-memory opt-in of the tensor-core kernels of a mode, once per device (also called
// ahead of a graph capture).
template <int MODE>
int ensure_tc_attr() {
  static int attr_done[64] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && !attr_done[dev]) {
    using FC = CtaCfg<MODE, false>;
    using SC = CtaCfg<MODE, true>;
    cudaError_t e = cudaFuncSetAttribute(cgemm_cta_kernel<MODE, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)FC::smem(FC::NT_MAX));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(cgemm_cta_kernel<MODE, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)SC::smem(SC::NT_MAX));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(cgemm_pair_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               kMaxSmem - kStaticSmem);
    if (e != cudaSuccess) return (int)e;
    // the roles' shares are drawn from what the launch gives: with fewer registers than that
    // (another compiler's choice) the epilogue's warps would wait for theirs without end
    cudaFuncAttributes fa{};
    if ((e = cudaFuncGetAttributes(&fa, cgemm_pair_kernel<MODE>)) != cudaSuccess) return (int)e;
    if (fa.numRegs < kRegLaunch) return (int)cudaErrorLaunchOutOfResources;
    attr_done[dev] = 1;
  }
  return 0;
}

// Whether a default step takes tiles on one CTA.  With few k-steps a tile ends before the pair's
// handshakes do (arrivals and commits that cross to the other SM, behind that tile's stores), and
// the smaller tile without them is faster; with more, the pair's halved operand reads win.  us on
// pairs / on one CTA, for about 10^6 columns in rows that a tensor map describes:
//   TF32x3 K = 8, N = 32 143 / 71; K = 32, N = 64 207 / 165, N = 128 270 / 243; K = 48, N = 64 213 / 210,
//     N = 128 286 / 289;
//   BF16x2 K = 16, N = 64 163 / 105; K = 32, N = 64 169 / 133, N = 128 236 / 202; K = 48, N = 32 129 / 142;
//   BF16x3 K = 16, N = 32 132 / 79, N = 128 240 / 201; K = 32, N = 64 183 / 149, N = 128 245 / 245; K = 48,
//     N = 32 149 / 156;
// and for 7 x 10^5 columns whose rows the producers load themselves, where a pair's 16 warps have
// more loads in flight:
//   TF32x3 K = 8, N = 32 96 / 61; K = 16, N = 16 87 / 88, N = 64 135 / 114; K = 24, N = 32 107 / 133;
//   BF16x2 K = 16, N = 64 116 / 91; K = 32, N = 32 103 / 119; BF16x3 K = 16, N = 32 94 / 76, N = 128 177 / 179;
//     K = 32, N = 32 107 / 113.
template <int MODE>
bool takes_cta_tile(int64_t K, int Nt, bool mapped) {
  if (!mapped || K <= 16) return K <= 16;
  return K <= 32 && (Mode<MODE>::TERMS == 2 || Nt <= 64);
}

template <int MODE>
int launch_tc_mode(bool fast, const void* S, int64_t s_stride, const void* B, int64_t b_stride, void* C,
                   int64_t c_stride, int64_t P, int64_t K, int64_t N, int64_t NL, int64_t Sd,
                   int batch, char* scratch, int64_t scratch_stride, int withhold, bool no_tma, int beta,
                   cudaStream_t st) {
  using M_ = Mode<MODE>;
  using FC = CtaCfg<MODE, false>;
  using SC = CtaCfg<MODE, true>;
  using PC = PairCfg<MODE>;
  const int64_t nt_max = fast ? FC::NT_MAX : PC::NT_MAX;
  const int Nt = (int)(N < nt_max ? N : nt_max);   // N % 16 == 0
  const int KT = (int)(K / M_::KS);
  if (int err = ensure_tc_attr<MODE>()) return err;
  dim3 sg((unsigned)((N + 127) / 128), KT, batch);
  auto split = fast ? split_site_kernel<MODE, false> : split_site_kernel<MODE, true>;
  cudaError_t e = launch_early(split, sg, dim3(128), 0, st, (const float2*)S, s_stride, (int)K, (int)N, Nt, scratch,
                               scratch_stride);
  count_launch();
  if (e != cudaSuccess) return (int)e;
  const bool mapped = !fast && !no_tma && rows_fit_map(Sd);
  const bool pair = !fast && !takes_cta_tile<MODE>(K, Nt, mapped);
  TcArgs a{};
  a.B = (const float2*)B; a.b_stride = b_stride;
  a.C = (float2*)C; a.c_stride = c_stride;
  a.simage = scratch; a.img_stride = scratch_stride;
  a.P = P; a.K = K; a.N = N; a.NL = NL; a.Sd = Sd; a.J = P * Sd;
  a.Nt = Nt;
  a.NHt = (int)(N / Nt);
  const int rows = pair ? 2 * kRows : kRows;
  a.JT = (a.J + rows - 1) / rows;
  a.tiles = (int64_t)batch * a.JT * a.NHt;
  a.sd_shift = -1;
  for (int b = 0; b < 62; ++b)
    if (Sd == int64_t(1) << b) a.sd_shift = b;
  a.withhold_s = withhold;
  a.beta = beta;
  alignas(64) CUtensorMap tmA;
  std::memset(&tmA, 0, sizeof(tmA));
  a.use_tma = mapped && make_b_map(&tmA, B, b_stride, batch, P, K, Sd, pair ? PC::SUB * M_::KS : M_::KS, &a.box_s, &a.box_p);
  // the kernels start while split_site_kernel runs, so that barriers and launch latency (and for
  // pairs the TMEM) are out of the way
  if (pair) {
    const int64_t pairs = std::min<int64_t>(a.tiles, num_sms() / 2);
    pair_rings<MODE>(Nt, &a.stages, &a.nbuf);
    e = launch_early(cgemm_pair_kernel<MODE>, dim3((unsigned)(2 * pairs)), dim3(PC::THREADS),
                     PC::smem(Nt, a.stages, a.nbuf), st, a, tmA);
  } else {
    const unsigned grid = (unsigned)std::min<int64_t>(a.tiles, num_sms());
    e = fast ? launch_early(cgemm_cta_kernel<MODE, false>, dim3(grid), dim3(FC::THREADS), FC::smem(Nt), st, a, tmA)
             : launch_early(cgemm_cta_kernel<MODE, true>, dim3(grid), dim3(SC::THREADS), SC::smem(Nt), st, a, tmA);
  }
  count_launch();
  return (int)e;
}

// ---- tensor-core rate probe -------------------------------------------------------
// One CTA per SM (its shared-memory request leaves room for no second one) issues `iters`
// MMAs of the mode's operand kind, M = 128, N = 256, one K step, from fixed pseudo-random
// shared-memory operands into two alternating TMEM accumulators, committing every 256
// MMAs.  The host times the launch: dense tensor flop/s of that kind as this code issues it.
constexpr size_t kProbeSmem = 128 << 10;
template <int MODE>
__global__ void __launch_bounds__(128, 1) tc_probe_kernel(int64_t iters) {
  extern __shared__ __align__(16) char probe_raw[];
  char* sm = probe_raw + ((128u - (smem_u32(probe_raw) & 127u)) & 127u);
  char* sA = sm;               // 128 rows x 32 B
  char* sB = sm + kPlaneA;     // 256 rows x 32 B
  __shared__ uint64_t bars[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int tid = threadIdx.x;
  // operands: 12 KB of small pseudo-random values of the mode's type
  for (int i = tid; i < 3 * kPlaneA / 4; i += blockDim.x) {
    uint32_t h = (uint32_t)i * 2654435761u + 0x9e3779b9u * (blockIdx.x + 1);
    h ^= h >> 15;
    const float x = (float)(h & 0xffff) * (1.0f / 65536.0f) - 0.5f;
    uint32_t w;
    if constexpr (Mode<MODE>::FMT == 1) {
      const uint32_t b = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x));
      w = b | (b << 16);
    } else {
      w = __float_as_uint(x) & 0xffffe000u;   // TF32: 10 explicit mantissa bits
    }
    reinterpret_cast<uint32_t*>(sm)[i] = w;
  }
  fence_async_smem();
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(smem_u32(&bars[0]), 1);
    mbar_init(smem_u32(&bars[1]), 1);
    mbar_init_fence();
  }
  if (tid < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  if (tid < 32) {
    // warp-uniform loop; lane 0 issues 16 MMAs per iteration (a thread issuing one MMA per
    // loop iteration kept the tensor pipe about half idle)
    volatile int* abort = &abort_flag;
    const uint64_t ad = smem_desc(smem_u32(sA)), bd = smem_desc(smem_u32(sB));
    const uint32_t idesc = instr_desc<MODE>(256, false);
    // commit groups of 256 MMAs alternate between two barriers (a barrier never has two
    // commits outstanding); group g completes phase g / 2 of barrier g % 2
    auto wait_group = [&](int64_t g) {
      return mbar_wait(smem_u32(&bars[g & 1]), (uint32_t)((g >> 1) & 1), abort);
    };
    int64_t groups = 0;
    bool ok = true;
    for (int64_t i0 = 0; i0 < iters && ok; i0 += 16) {   // iters is a multiple of 256
      if (tid == 0) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
          mma<MODE>(tmem + (uint32_t)((u & 1) * 256), ad, bd, idesc, (i0 + u) >= 2 ? 1u : 0u);
      }
      if (((i0 + 15) & 255) == 255) {
        if (tid == 0) mma_commit(smem_u32(&bars[groups & 1]));
        __syncwarp();
        if (groups > 0) ok = wait_group(groups - 1);   // at most two groups in flight
        ++groups;
      }
    }
    if (ok && groups > 0) wait_group(groups - 1);   // the last group covers every MMA
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid < 32) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

template <int MODE>
int run_tc_probe(int64_t iters, double* tflops, cudaStream_t st) {
  auto kern = tc_probe_kernel<MODE>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kProbeSmem);
  if (e != cudaSuccess) return (int)e;
  const int grid = num_sms();
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return (int)cudaErrorUnknown;
  iters = (iters + 255) / 256 * 256;
  kern<<<grid, 128, kProbeSmem, st>>>((iters / 8 + 255) / 256 * 256);   // warm-up
  cudaEventRecord(e0, st);
  kern<<<grid, 128, kProbeSmem, st>>>(iters);
  cudaEventRecord(e1, st);
  count_launch(2);
  e = cudaEventSynchronize(e1);
  float ms = 0.f;
  if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (e != cudaSuccess) return (int)e;
  const double flop_per_mma = 2.0 * kRows * 256 * Mode<MODE>::KS;
  *tflops = (double)grid * (double)iters * flop_per_mma / (ms * 1e-3) / 1e12;
  return 0;
}

}  // namespace

bool tc_eligible(int precision, int64_t K, int64_t N, int64_t J, int flags) {
  // default tiles are 128 columns wide (N <= 128 or whole 128-column tiles); fast ones
  // 256 (N <= 256 or whole 256-column tiles)
  const int64_t nt = (flags & kTcFast) ? 256 : 128;
  const bool n_ok = N % 16 == 0 && (N <= nt || N % nt == 0);
  if (precision == QFX_PREC_C3M_BF16X3 || precision == QFX_PREC_C3M_BF16X2)
    return n_ok && K % 16 == 0 && J >= kRows;
  if (precision == QFX_PREC_C3M_TF32X3) return n_ok && K % 8 == 0 && J >= kRows;
  return false;
}

uint64_t tc_scratch_bytes(int precision, int64_t K, int64_t N) {
  // per k-stage and column n: 3 planes per term (the embedded layout of default tiles)
  if (precision == QFX_PREC_C3M_BF16X3) return (uint64_t)(K / 16) * 9 * (uint64_t)N * 32;
  if (precision == QFX_PREC_C3M_BF16X2) return (uint64_t)(K / 16) * 6 * (uint64_t)N * 32;
  if (precision == QFX_PREC_C3M_TF32X3) return (uint64_t)(K / 8) * 6 * (uint64_t)N * 32;
  return 0;
}

int launch_step_tc(const void* S, int64_t s_stride, const void* B, int64_t b_stride, void* C,
                   int64_t c_stride, int64_t P, int64_t K, int64_t N, int64_t NL, int64_t Sd,
                   int batch, int precision, char* scratch, int64_t scratch_stride, void* stream,
                   int flags) {
  cudaStream_t st = (cudaStream_t)stream;
  const int beta = (flags & kTcBeta) ? 1 : 0;
  const bool fast = (flags & kTcFast) != 0;
  const int withhold = (flags & kTcWithhold) ? 1 : 0;
  const bool no_tma = (flags & kTcNoTma) != 0;
  if (precision == QFX_PREC_C3M_BF16X3)
    return launch_tc_mode<QFX_PREC_C3M_BF16X3>(fast, S, s_stride, B, b_stride, C, c_stride, P, K, N, NL, Sd, batch,
                                               scratch, scratch_stride, withhold, no_tma, beta, st);
  if (precision == QFX_PREC_C3M_BF16X2)
    return launch_tc_mode<QFX_PREC_C3M_BF16X2>(fast, S, s_stride, B, b_stride, C, c_stride, P, K, N, NL, Sd, batch,
                                               scratch, scratch_stride, withhold, no_tma, beta, st);
  if (precision == QFX_PREC_C3M_TF32X3)
    return launch_tc_mode<QFX_PREC_C3M_TF32X3>(fast, S, s_stride, B, b_stride, C, c_stride, P, K, N, NL, Sd, batch,
                                               scratch, scratch_stride, withhold, no_tma, beta, st);
  return (int)cudaErrorInvalidValue;
}

int tc_probe(int precision, int64_t iters, double* tflops, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  if (precision == QFX_PREC_C3M_BF16X3 || precision == QFX_PREC_C3M_BF16X2)
    return run_tc_probe<QFX_PREC_C3M_BF16X3>(iters, tflops, st);
  if (precision == QFX_PREC_C3M_TF32X3) return run_tc_probe<QFX_PREC_C3M_TF32X3>(iters, tflops, st);
  return (int)cudaErrorInvalidValue;
}

int tc_prepare_attributes() {
  (void)tensor_map_encoder();   // resolve the driver entry point outside any capture
  int e = 0;
  if (!e) e = ensure_tc_attr<QFX_PREC_C3M_BF16X3>();
  if (!e) e = ensure_tc_attr<QFX_PREC_C3M_BF16X2>();
  if (!e) e = ensure_tc_attr<QFX_PREC_C3M_TF32X3>();
  return e;
}

int tc_take_status() {
  unsigned int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_tc_status, sizeof(v)) != cudaSuccess) return -1;
  if (v) {
    const unsigned int z = 0;
    cudaMemcpyToSymbol(g_tc_status, &z, sizeof(z));
  }
  return (int)v;
}

}  // namespace qfx
