// Tile body of the FP32 SIMT contraction step, shared by the per-step kernels
// (cgemm_simt.cu) and the persistent batch scheduler (batch.cu).
//
//   C[nh][p][nl][s] = sum_k S[k][nh*NL + nl] * B[p][k][s]
//
// is the TTGT contraction of Sec. III.E with the transposes folded into the addressing:
// rows are n (M = N), columns are j = p*Sd + s (J = P*Sd), the reduction is k.  Eq. 1
// counts 8*N*J*K flops; each complex multiply-add is 4 real FMAs (the paper's complex
// FP32 CGEMM, without tensor cores).
//
// Tiling: one CTA computes BM x BJ outputs with NTH threads, each thread TM x TJ.  The k
// loop moves slabs of S and B (8 rows k, or 16) through two shared-memory buffers; the slab after the
// next waits in registers meanwhile.  B is stored with the real parts of two neighbouring
// columns side by side and then their imaginary parts, so that a 16-byte read gives two
// operands of the packed FP32 FMA (two columns per instruction); the entries of S become
// pairs in registers.  The register file bounds this loop, not the FMA pipe: an outer
// product on registers alone runs at 64 TFLOP/s row by row and at 71 when each row walks
// back over the columns that the one before ended on, of 80.5; with the reads of shared
// memory and the duplications it stays at about 60.  Tiles of at most 128 registers a thread
// leave room for two CTAs on an SM, so that one's start and end hide behind the other's
// loop: K = N = 256 runs at the same rate with one CTA of 8 x 8 outputs a thread, but K = 64,
// with 8 slabs to a tile, gains most of its time from the second one.
//
// JMODE loads two columns as one 16-byte vector (Sd even).  KMODE takes any Sd: for Sd = 1
// (the last site of a line) a column is contiguous in k and 8 lanes (or 16) read its slab; otherwise
// the lanes run along s with 8-byte loads.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace qfx {
namespace simt {

struct StepArgs {
  const float2* S; int64_t s_stride;
  const float2* B; int64_t b_stride;
  float2* C; int64_t c_stride;
  int64_t P, K, N, NL, Sd, J;
  int32_t beta;   // 1: add the product into C (a chunk of a long contraction), 0: write it
};

template <int BM, int BJ, int TM, int TJ, bool KMODE, int NTH = 256>
struct Cfg {
  // Rows k of a slab.  The fill tiles of 8 rows move 8 bytes for 64 FMAs and are bound by what they
  // have in flight: a slab of 16 takes 1024 x 8 over 50000 columns from 151 to 122 us (Sd = 64) and 185
  // to 144 (Sd = 1).  8 x 512 has no room for it beside a second CTA.
  static constexpr int BK = BM == 8 && BJ <= 256 ? 16 : 8;
  static constexpr int TYN = BM / TM, TXN = BJ / TJ;
  static constexpr int LDA = BM + 2, LDB = BJ + 2;   // float2 per row; rows are 16-byte multiples
  static constexpr int A_IT = (BK * BM + NTH - 1) / NTH;
  static constexpr int B_IT = (BK * BJ) / (2 * NTH);   // column pairs per thread and slab
  static constexpr size_t SMEM = (size_t)2 * BK * (LDA + LDB) * sizeof(float2);
  static_assert(TYN * TXN == NTH, "one thread per TM x TJ outputs");
  static_assert(TM % 2 == 0 && TJ % 2 == 0, "even thread tiles");
  static_assert((BK * BJ) % (2 * NTH) == 0, "B loader coverage");
  static_assert(NTH % (BJ / 2) == 0 && NTH % BM == 0, "a thread's columns are fixed");
};

// Two FP32 numbers in one 64-bit register pair, and the packed FMA on them: each half is one
// round-to-nearest FMA, bit for bit that of fmaf.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
// volatile: the compiler keeps the order in which they are written (see above)
__device__ __forceinline__ void fma2(f32x2& c, f32x2 a, f32x2 b) {
  asm volatile("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

// x / d and x % d of a column index: in 32 bits where they hold it (a 64-bit division takes
// as long as several k slabs)
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

// One BM x BJ output tile of the step; `tile` enumerates (n tile, j tile) with the n tile
// fastest, `item` selects the batch entry.  NTH threads; `smem_raw` holds Cfg::SMEM bytes.
// Every output accumulates its k terms in the same order whatever the tile shape, so all
// variants give bit-identical results.
template <int BM, int BJ, int TM, int TJ, bool KMODE, int NTH = 256>
__device__ __forceinline__ void cgemm_tile(const StepArgs& a, int64_t tile, int64_t item,
                                           float4* smem_raw) {
  using C_ = Cfg<BM, BJ, TM, TJ, KMODE, NTH>;
  constexpr int BK = C_::BK, TXN = C_::TXN, LDA = C_::LDA, LDB = C_::LDB, TQ = TJ / 2;
  float2* As = reinterpret_cast<float2*>(smem_raw);
  float2* Bs = As + 2 * BK * LDA;

  const int tid = threadIdx.x;
  const int tx = tid % TXN, ty = tid / TXN;
  int64_t jt, nt;
  divmod(tile, (a.N + BM - 1) / BM, jt, nt);
  const int n0 = (int)(nt * BM);
  const int64_t j0 = jt * BJ;
  // plain loads: in the batch scheduler S and B were written earlier in the same launch, which
  // the read-only path may not see
  const float2* S = a.S + item * a.s_stride;
  const float2* B = a.B + item * a.b_stride;
  float2* C = a.C + item * a.c_stride;
  const int64_t Sd = a.Sd, J = a.J;
  const int N = (int)a.N;
  const int KT = (int)((a.K + BK - 1) / BK);             // slabs, and rows k of the last one
  const int klast = (int)(a.K - (int64_t)(KT - 1) * BK);

  // this thread's B elements of a slab.  Along s: the column pair jj, rows kk0 + i * KSTEP.
  // Along k (KMODE, Sd = 1): row kk0, the columns jj + i * JSTEP.
  constexpr int KSTEP = NTH / (BJ / 2), JSTEP = NTH / BK;
  const bool along_k = KMODE && Sd == 1;
  const int kk0 = along_k ? tid % BK : tid / (BJ / 2);
  const int jj = along_k ? tid / BK : (tid % (BJ / 2)) * 2;
  const float2* bp;
  int64_t next = 1;        // KMODE: from column jj to the one after it
  bool ok0, ok1 = false;   // those columns exist
  {
    int64_t p, s;
    const int64_t j = j0 + jj;
    divmod(j, Sd, p, s);
    bp = B + p * a.K * Sd + s + (int64_t)kk0 * Sd;
    ok0 = j < J;
    if (KMODE) {
      ok1 = j + 1 < J;
      if (s + 1 == Sd) next = a.K * Sd - s;
    }
  }
  // and its entries of S: column n0 + tid % BM, rows tid / BM + i * ASTEP
  constexpr int ASTEP = NTH / BM;
  const bool nin = n0 + tid % BM < N;
  const float2* sp = S + (int64_t)(tid / BM) * N + n0 + tid % BM;
  float4 rb[C_::B_IT];
  float2 ra[C_::A_IT];
  auto fetch = [&](int kt) {   // slab kt into registers
    const int krows = kt + 1 < KT ? BK : klast;
#pragma unroll
    for (int i = 0; i < C_::A_IT; ++i) {
      const int e = tid + i * NTH;
      const int kk = e / BM;
      ra[i] = make_float2(0.f, 0.f);
      if ((BK * BM % NTH == 0 || e < BK * BM) && kk < krows && nin)
        ra[i] = sp[(int64_t)(i * ASTEP) * N];
    }
    if (KMODE && along_k) {
      const bool kin = kk0 < krows;
#pragma unroll
      for (int i = 0; i < C_::B_IT; ++i) {
        float2 v[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (kin && j0 + jj + (2 * i + h) * JSTEP < J) v[h] = bp[(int64_t)(2 * i + h) * JSTEP * a.K];
        rb[i] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
      }
    } else {
#pragma unroll
      for (int i = 0; i < C_::B_IT; ++i) {
        rb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        const float2* src = bp + (int64_t)i * KSTEP * Sd;
        if (kk0 + i * KSTEP < krows) {
          if (!KMODE) {
            if (ok0) rb[i] = *reinterpret_cast<const float4*>(src);
          } else {
            if (ok0) { const float2 v = *src; rb[i].x = v.x; rb[i].y = v.y; }
            if (ok1) { const float2 v = src[next]; rb[i].z = v.x; rb[i].w = v.y; }
          }
        }
      }
    }
    bp += BK * Sd;
    sp += BK * (int64_t)N;
  };
  auto store = [&](int buf) {   // registers into buffer `buf`
#pragma unroll
    for (int i = 0; i < C_::A_IT; ++i) {
      const int e = tid + i * NTH;
      if (BK * BM % NTH == 0 || e < BK * BM) As[(buf * BK + e / BM) * LDA + e % BM] = ra[i];
    }
    if (KMODE && along_k) {
      float* row = reinterpret_cast<float*>(Bs + (buf * BK + kk0) * LDB);
#pragma unroll
      for (int i = 0; i < C_::B_IT; ++i) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int c = jj + (2 * i + h) * JSTEP;
          row[(c >> 1) * 4 + (c & 1)] = h ? rb[i].z : rb[i].x;
          row[(c >> 1) * 4 + (c & 1) + 2] = h ? rb[i].w : rb[i].y;
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < C_::B_IT; ++i)
        *reinterpret_cast<float4*>(Bs + (buf * BK + kk0 + i * KSTEP) * LDB + jj) =
            make_float4(rb[i].x, rb[i].z, rb[i].y, rb[i].w);
    }
  };

  f32x2 cr[TM][TQ], ci[TM][TQ];   // real and imaginary parts of column pairs
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int q = 0; q < TQ; ++q) { cr[i][q] = 0; ci[i][q] = 0; }

  fetch(0);
  store(0);
  if (KT > 1) fetch(1);
  __syncthreads();
  for (int kt = 0; kt < KT; ++kt) {
    const int buf = kt & 1;
    const float2* Ak = As + buf * BK * LDA + ty * TM;
    const float2* Bk = Bs + buf * BK * LDB + tx * 2;
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      // the padding of every tile ends at a multiple of 8
      if (BK == 16 && kk == 8 && kt + 1 == KT && klast <= 8) break;
      float2 sv[TM];
      f32x2 br[TQ], bi[TQ];
#pragma unroll
      for (int i = 0; i < TM / 2; ++i) {
        const float4 t = *reinterpret_cast<const float4*>(Ak + kk * LDA + 2 * i);
        sv[2 * i] = make_float2(t.x, t.y);
        sv[2 * i + 1] = make_float2(t.z, t.w);
      }
#pragma unroll
      for (int q = 0; q < TQ; ++q) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(Bk + kk * LDB + q * 2 * TXN);
        br[q] = t.x;
        bi[q] = t.y;
      }
      // per output re += sr br, then re += (-si) bi; im += sr bi, then im += si br
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const f32x2 sr = pack2(sv[i].x, sv[i].x), si = pack2(sv[i].y, sv[i].y), ns = pack2(-sv[i].y, -sv[i].y);
#pragma unroll
        for (int z = 0; z < TQ; ++z) {
          const int q = i & 1 ? TQ - 1 - z : z;
          fma2(ci[i][q], sr, bi[q]);
          fma2(cr[i][q], sr, br[q]);
        }
#pragma unroll
        for (int z = 0; z < TQ; ++z) {
          const int q = i & 1 ? z : TQ - 1 - z;
          fma2(ci[i][q], si, br[q]);
        }
#pragma unroll
        for (int z = 0; z < TQ; ++z) {
          const int q = i & 1 ? TQ - 1 - z : z;
          fma2(cr[i][q], ns, bi[q]);
        }
      }
      // the other buffer's readers passed the barrier at the end of the last slab; its loads
      // have had half a slab, and the next ones start as early as their registers are free
      if (kk == BK / 2 - 1 && kt + 1 < KT) store(buf ^ 1);
      if (kk == BK / 2 && kt + 2 < KT) fetch(kt + 2);
    }
    __syncthreads();
  }

  // epilogue: C[nh][p][nl][s]
  const int NL = (int)a.NL;
  const int64_t strideNH = a.P * a.NL * Sd;
  // (nh, nl) of this thread's first row once; the rows below step with a carry (a division
  // per element is a large share of the epilogue)
  const int nfirst = n0 + ty * TM;
  const int nh_first = nfirst / NL, nl_first = nfirst % NL;
#pragma unroll
  for (int q = 0; q < TQ; ++q) {
    const int64_t j = j0 + q * 2 * TXN + tx * 2;
    if (j >= J) continue;
    int64_t p, s;
    divmod(j, Sd, p, s);
    float2* dst = C + nh_first * strideNH + p * (NL * Sd) + nl_first * Sd + s;
    const int64_t step1 = s + 1 == Sd ? NL * Sd - s : 1;   // to column j + 1
    int nl = nl_first;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      if (nfirst + i >= N) break;
      const float2 re = unpack2(cr[i][q]), im = unpack2(ci[i][q]);
      if (!KMODE) {
        float4 w = make_float4(re.x, im.x, re.y, im.y);
        if (a.beta) {
          const float4 o = *reinterpret_cast<const float4*>(dst);
          w.x += o.x; w.y += o.y; w.z += o.z; w.w += o.w;
        }
        *reinterpret_cast<float4*>(dst) = w;
      } else {
        float2 w0 = make_float2(re.x, im.x);
        if (a.beta) { const float2 o = *dst; w0.x += o.x; w0.y += o.y; }
        *dst = w0;
        if (j + 1 < J) {
          float2 w1 = make_float2(re.y, im.y);
          if (a.beta) { const float2 o = dst[step1]; w1.x += o.x; w1.y += o.y; }
          dst[step1] = w1;
        }
      }
      dst += Sd;
      if (++nl == NL) { nl = 0; dst += strideNH - NL * Sd; }
    }
  }
}

// Tile variants: 0..4 stream B along s (JMODE), 5..9 the same tiles for any Sd.  Rows:
// 128, 64, 32, 16, 8.
#define QFX_SIMT_VARIANTS(X)        \
  X(0, 128, 64, 4, 8, false)        \
  X(1, 64, 128, 4, 8, false)        \
  X(2, 32, 256, 4, 8, false)        \
  X(3, 16, 256, 4, 4, false)        \
  X(4, 8, 512, 4, 4, false)         \
  X(5, 128, 64, 4, 8, true)         \
  X(6, 64, 128, 4, 8, true)         \
  X(7, 32, 256, 4, 8, true)         \
  X(8, 16, 256, 4, 4, true)         \
  X(9, 8, 512, 4, 4, true)

// Fill variants: smaller tiles for grids that the tiles above would leave with fewer CTAs than
// SMs (fill_variant picks them at launch time; the batch scheduler keeps 0..9).
#define QFX_SIMT_FILL_VARIANTS(X)   \
  X(20, 64, 64, 4, 4, false)        \
  X(21, 32, 128, 4, 4, false)       \
  X(22, 16, 128, 2, 4, false)       \
  X(23, 8, 256, 2, 4, false)        \
  X(24, 8, 128, 2, 2, false)        \
  X(25, 64, 64, 4, 4, true)         \
  X(26, 32, 128, 4, 4, true)        \
  X(27, 16, 128, 2, 4, true)        \
  X(28, 8, 256, 2, 4, true)         \
  X(29, 8, 128, 2, 2, true)

}  // namespace simt
}  // namespace qfx
