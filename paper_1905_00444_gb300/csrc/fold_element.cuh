// Per-element time fold of one site tensor (Sec. III, Fig. 3), shared by fold.cu and the
// batch scheduler.  See fold.cu for the method.
#pragma once
#include <cuda_runtime.h>

#include "qfx_internal.h"

namespace qfx {
namespace foldk {

// Float-float ("double-single") arithmetic: a real value is the unevaluated sum hi + lo
// of two FP32 numbers with |lo| <= ulp(hi)/2, about 48 significant bits, on the FP32
// pipes (this GPU runs FP64 at 1/64 of the FP32 rate).  Built from two error-free
// transformations: Knuth's TwoSum (s + e = a + b exactly) and the product's exact error
// by a fused multiply-add (a*b - fl(a*b), Dekker's TwoProduct with FMA); the sum and
// product below follow Dekker's double-length algorithms (1971).  Every step is an
// explicit round-to-nearest intrinsic, which the compiler never contracts or reorders, so
// every caller rounds exactly alike: the group fold relies on it to reproduce the
// per-element fold bit for bit.
struct ff {
  float hi, lo;
};
struct cff {
  ff re, im;
};
__device__ __forceinline__ ff two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ ff fast_two_sum(float a, float b) {   // needs |a| >= |b| or a = 0
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  const ff s = two_sum(a.hi, b.hi);
  return two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ ff ff_neg(ff a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = __fmul_rn(a.hi, b.hi);
  const float e = __fmaf_rn(a.hi, b.hi, -p);   // exact: a.hi * b.hi = p + e
  return fast_two_sum(p, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e)));
}
__device__ __forceinline__ cff cmul(cff a, cff b) {
  return {ff_add(ff_mul(a.re, b.re), ff_neg(ff_mul(a.im, b.im))),
          ff_add(ff_mul(a.re, b.im), ff_mul(a.im, b.re))};
}
__device__ __forceinline__ cff cadd(cff a, cff b) { return {ff_add(a.re, b.re), ff_add(a.im, b.im)}; }
__device__ __forceinline__ float ff_round(ff a) { return __fadd_rn(a.hi, a.lo); }
__device__ __forceinline__ cff cff_zero() { return {{0.f, 0.f}, {0.f, 0.f}}; }
__device__ __forceinline__ cff cff_one() { return {{1.f, 0.f}, {0.f, 0.f}}; }

// Bond values (up, left, right, down, each plus its cut offset for slice `sid`) and the x
// value of element i of site `st`; the output bitstring x1w is given as words (qubit q is
// bit q % 64 of word q / 64).
struct FoldCoord {
  uint64_t val[4];
  int xv;
};
__device__ __forceinline__ int64_t take_bits(int64_t& r, int32_t dim) {   // r mod dim; r /= dim
  const int64_t v = r & (int64_t)(dim - 1);
  r >>= 31 - __clz(dim);
  return v;
}
__device__ __forceinline__ FoldCoord fold_coord(const FoldSite& st, const CutDev* __restrict__ cuts, int n_cuts,
                                                const uint64_t* x1w, int64_t sid, int64_t i) {
  int64_t off[4] = {0, 0, 0, 0};
  for (int c = 0; c < n_cuts; ++c) {
    const CutDev cd = cuts[c];
    const int64_t digit = (sid / cd.suffix) % cd.radix;
#pragma unroll
    for (int s = 0; s < 4; ++s)
      if (st.edge[s] == cd.edge) off[s] = digit * cd.size;
  }
  // every local dimension is a power of two (2^bits of a bond, halved by cuts)
  int64_t r = i;
  const int64_t vd = take_bits(r, st.dim[4]), vr = take_bits(r, st.dim[3]), vx = take_bits(r, st.dim[2]);
  const int64_t vl = take_bits(r, st.dim[1]), vu = r;
  FoldCoord fc;
  fc.val[0] = (uint64_t)(vu + off[0]);
  fc.val[1] = (uint64_t)(vl + off[1]);
  fc.val[2] = (uint64_t)(vr + off[2]);
  fc.val[3] = (uint64_t)(vd + off[3]);
  fc.xv = st.x_open ? (int)vx : (int)((x1w[st.qubit >> 6] >> (st.qubit & 63)) & 1ull);
  return fc;
}

// Events of one site's time line staged in shared memory: what each one is (kind, slot and bit
// packed) and its matrix, 16 floats (a (hi, lo) pair per FP64 real of the 2x2 complex matrix,
// row-major; a general gate's four blocks stay in global memory, at `block`).  Read from global
// memory, an event costs every thread two dependent loads, more than its arithmetic.
constexpr int kFoldStage = 64;
struct FoldStage {
  float4 mat[kFoldStage][4];
  int32_t what[kFoldStage];
  int32_t block[kFoldStage];
};
__device__ __forceinline__ int32_t pack_event(const FoldEvent& ev) { return ev.kind | (ev.slot << 4) | (ev.bit << 8); }
// events [e0, e0 + n), n <= kFoldStage, by `threads` threads of index `tid` (a barrier follows)
__device__ __forceinline__ void stage_events(FoldStage& sm, const FoldEvent* __restrict__ events,
                                             const float* __restrict__ matsf, int e0, int n, int tid, int threads) {
  for (int i = tid; i < 4 * n; i += threads) {
    const FoldEvent ev = events[e0 + (i >> 2)];
    sm.mat[i >> 2][i & 3] = reinterpret_cast<const float4*>(matsf + 16 * (int64_t)ev.mat)[i & 3];
    if ((i & 3) == 0) {
      sm.what[i >> 2] = pack_event(ev);
      sm.block[i >> 2] = ev.mat;
    }
  }
}

// The bond bits an event reads for an element (0 for a one-qubit gate): one bit for a
// diagonal two-qubit gate, two (k = 2*o0 + i0) for a general one.
__device__ __forceinline__ int event_key(int32_t what, const FoldCoord& fc) {
  const int kind = what & 15, slot = (what >> 4) & 15, bit = what >> 8;
  if (kind == EV_GATE) return 0;
  const uint64_t bv = slot == 0 ? fc.val[0] : slot == 1 ? fc.val[1] : slot == 2 ? fc.val[2] : fc.val[3];
  const uint64_t mask = (kind == EV_PROJ || kind == EV_DIAG) ? 1ull : 3ull;
  return (int)((bv >> bit) & mask);
}

// One event on the site's 2-vector (v0, v1), for bond bits k: a one-qubit gate; the
// projector on q0 or the diagonal on q1 of a diagonal two-qubit gate; |o0><i0| on q0 or
// the 2x2 block B_k on q1 of a general one.  `m` is the event's matrix (a block's own one).
__device__ __forceinline__ cff entry4(float4 v) { return {{v.x, v.y}, {v.z, v.w}}; }
__device__ __forceinline__ void apply_event(int kind, const float4* m, int k, cff& v0, cff& v1) {
  if (kind == EV_GATE || kind == EV_BLOCK) {
    const cff n0 = cadd(cmul(entry4(m[0]), v0), cmul(entry4(m[1]), v1));
    const cff n1 = cadd(cmul(entry4(m[2]), v0), cmul(entry4(m[3]), v1));
    v0 = n0;
    v1 = n1;
  } else if (kind == EV_PROJ) {
    if (k) v0 = cff_zero();
    else   v1 = cff_zero();
  } else if (kind == EV_DIAG) {
    v0 = cmul(v0, entry4(m[2 * k]));
    v1 = cmul(v1, entry4(m[2 * k + 1]));
  } else {   // EV_ELEM: |o0><i0|
    const cff src = (k & 1) ? v1 : v0;
    v0 = (k >> 1) ? cff_zero() : src;
    v1 = (k >> 1) ? src : cff_zero();
  }
}

// Elements i0 .. i0 + G - 1 of site `st` for slice `sid`: float-float evolution of their
// 2-vectors through the site's time line from |0>.  Consecutive elements differ only in the low
// bits of the innermost bond (its latest gates), so up to the first event that reads one of
// those bits they share one 2-vector, computed once with the operations of each element's
// own fold (the results do not depend on G); from there on each element has its own.
template <int G>
struct FoldState {
  FoldCoord fc[G];
  cff v0[G], v1[G];
  bool split;
  __device__ __forceinline__ void begin(const FoldSite& st, const CutDev* __restrict__ cuts, int n_cuts,
                                        const uint64_t* x1w, int64_t sid, int64_t i0) {
#pragma unroll
    for (int q = 0; q < G; ++q) fc[q] = fold_coord(st, cuts, n_cuts, x1w, sid, i0 + q);
    v0[0] = cff_one();
    v1[0] = cff_zero();
    split = G == 1;
  }
  // the staged events [0, n)
  __device__ __forceinline__ void run(const FoldStage& sm, const float* __restrict__ matsf, int n) {
    for (int e = 0; e < n; ++e) {
      const int32_t what = sm.what[e];
      const int kind = what & 15;
      int k[G];
#pragma unroll
      for (int q = 0; q < G; ++q) k[q] = event_key(what, fc[q]);
      if constexpr (G > 1) {
        if (!split) {
          bool same = true;
#pragma unroll
          for (int q = 1; q < G; ++q) same = same && k[q] == k[0];
          if (same) {
            apply(sm, matsf, e, kind, k[0], v0[0], v1[0]);
            continue;
          }
          fan_out();
        }
      }
#pragma unroll
      for (int q = 0; q < G; ++q) apply(sm, matsf, e, kind, k[q], v0[q], v1[q]);
    }
  }
  __device__ __forceinline__ float2 result(int q) const {   // rounded once to complex64
    const cff res = fc[q].xv ? v1[q] : v0[q];
    return make_float2(ff_round(res.re), ff_round(res.im));
  }
  __device__ __forceinline__ void end() {
    if constexpr (G > 1)
      if (!split) fan_out();
  }

 private:
  __device__ __forceinline__ void fan_out() {
#pragma unroll
    for (int q = 1; q < G; ++q) { v0[q] = v0[0]; v1[q] = v1[0]; }
    split = true;
  }
  __device__ __forceinline__ void apply(const FoldStage& sm, const float* __restrict__ matsf, int e, int kind, int k,
                                        cff& a, cff& b) {
    if (kind == EV_BLOCK)
      apply_event(kind, reinterpret_cast<const float4*>(matsf + 16 * ((int64_t)sm.block[e] + k)), k, a, b);
    else
      apply_event(kind, sm.mat[e], k, a, b);
  }
};

}  // namespace foldk
}  // namespace qfx
