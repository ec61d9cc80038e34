// Site-tensor builder (time-first folding), per-site power-of-two normalisation, and the
// FP64 sum of slice contributions.
//
// Fold (Sec. III, Fig. 3): for grid site q, the gates on its time line are applied to
// |0> in order; a diagonal two-qubit gate D between q0 and q1 is split as
// D(b0, b1) = sum_k delta(b0, k) D(k, b1), so q0 applies the projector |k><k| and q1
// applies diag(D(k,0), D(k,1)), with k one bit (leg) of the bond between them.  The
// tensor element T[up][left][x][right][down] is <x| ... |0> for the leg bits that its
// bond values carry.  Each element is evolved in float-float arithmetic (FP32 pairs,
// about 48 significant bits; see fold_element.cuh) and rounded once to complex64.  The events
// and their matrices come from shared memory.  Where the elements are many, a thread takes 4
// consecutive ones, which share the arithmetic of most events; where they would leave SMs idle,
// one, whose chain of events is shorter.  The sites of one item of 4x4x(1+16+1) (16 of at most
// 512 elements, about 26 events): 12 us, against 35 with 4 elements a thread and events from
// global memory; 37 items of 6x6x(1+24+1): 0.60 ms against 0.71.
//
// Normalisation (Sec. III.E: inputs normalised, outputs renormalised, to keep FP32
// away from underflow): each site is scaled by 2^-e with e chosen so that its largest
// |re| or |im| lies in [1/2, 1); the exponents are summed per work item and undone in
// FP64 when the slice contributions are added (Sec. III.A: sum over paths).
#include <cuda_runtime.h>

#include "fold_element.cuh"
#include "launch.cuh"
#include "qfx_internal.h"

namespace qfx {
namespace {

constexpr int kThreads = 256;

template <int G>
__global__ void __launch_bounds__(kThreads) fold_kernel(
    const FoldSite* __restrict__ sites, const FoldEvent* __restrict__ events,
    const float* __restrict__ matsf, const CutDev* __restrict__ cuts, int n_cuts,
    const uint64_t* x1, int x1_words, int64_t n_batch, int64_t slice_begin,
    int64_t item0, char* hdr, uint64_t hdr_stride, char* items, uint64_t item_bytes,
    uint64_t sites_off, int n_sites) {
  launch_wait();
  launch_next();
  __shared__ foldk::FoldStage sm;
  const FoldSite st = sites[blockIdx.y];
  const int g = blockIdx.z;
  const int64_t i0 = ((int64_t)blockIdx.x * kThreads + threadIdx.x) * G;
  if ((int64_t)blockIdx.x * kThreads * G >= st.size) return;   // block-uniform
  const int64_t item = item0 + g;
  const int64_t b = item % n_batch;
  const int64_t sid = slice_begin + item / n_batch;
  foldk::FoldState<G> f;
  f.begin(st, cuts, n_cuts, x1 + b * x1_words, sid, i0 < st.size ? i0 : 0);
  for (int e0 = st.ev_begin; e0 < st.ev_end; e0 += foldk::kFoldStage) {
    const int n = min(foldk::kFoldStage, st.ev_end - e0);
    if (e0 > st.ev_begin) __syncthreads();   // the last stage's readers are done
    foldk::stage_events(sm, events, matsf, e0, n, threadIdx.x, kThreads);
    __syncthreads();
    f.run(sm, matsf, n);
  }
  f.end();
  float mx = 0.f;
  float2* T = reinterpret_cast<float2*>(items + (uint64_t)g * item_bytes + sites_off) + st.offset;
#pragma unroll
  for (int q = 0; q < G; ++q)
    if (i0 + q < st.size) {
      const float2 v = f.result(q);
      T[i0 + q] = v;
      mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
  // non-negative floats order like their bit patterns
  const unsigned bits = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
  if ((threadIdx.x & 31) == 0 && bits) {
    unsigned* maxabs = reinterpret_cast<unsigned*>(hdr + (uint64_t)g * hdr_stride);
    atomicMax(maxabs + blockIdx.y, bits);
  }
}

// Fold and scale in one launch for sites of at most kSmallSite elements: a block per site and
// item, an element per thread.  The block knows its site's largest entry, so the header needs
// no clearing and the site no second pass (4x4x(1+16+1): three calls fewer of 21).
constexpr int kSmallSite = 1024;
__global__ void __launch_bounds__(kSmallSite) fold_scale_kernel(
    const FoldSite* __restrict__ sites, const FoldEvent* __restrict__ events,
    const float* __restrict__ matsf, const CutDev* __restrict__ cuts, int n_cuts,
    const uint64_t* x1, int x1_words, int64_t n_batch, int64_t slice_begin,
    int64_t item0, char* hdr, uint64_t hdr_stride, char* items, uint64_t item_bytes,
    uint64_t sites_off, int n_sites) {
  launch_wait();
  launch_next();
  __shared__ foldk::FoldStage sm;
  __shared__ unsigned largest;
  const FoldSite st = sites[blockIdx.x];
  const int g = blockIdx.y, i = threadIdx.x;
  if (i == 0) largest = 0u;
  const int64_t item = item0 + g;
  const int64_t b = item % n_batch;
  const int64_t sid = slice_begin + item / n_batch;
  foldk::FoldState<1> f;
  f.begin(st, cuts, n_cuts, x1 + b * x1_words, sid, i < st.size ? i : 0);
  for (int e0 = st.ev_begin; e0 < st.ev_end; e0 += foldk::kFoldStage) {
    const int n = min(foldk::kFoldStage, st.ev_end - e0);
    if (e0 > st.ev_begin) __syncthreads();
    foldk::stage_events(sm, events, matsf, e0, n, i, blockDim.x);
    __syncthreads();
    f.run(sm, matsf, n);
  }
  float2 v = f.result(0);
  // an entry that is no number counts as 0, as in fold_kernel: the others keep their scale
  const float mx = i < st.size ? fmaxf(0.f, fmaxf(fabsf(v.x), fabsf(v.y))) : 0.f;
  const unsigned bits = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
  __syncthreads();   // `largest` is cleared (also where a site has no events)
  if ((i & 31) == 0 && bits) atomicMax(&largest, bits);
  __syncthreads();
  const float m = __uint_as_float(largest);
  int e = 0;
  if (m > 0.f) frexpf(m, &e);
  if (i == 0) reinterpret_cast<int*>(hdr + (uint64_t)g * hdr_stride)[n_sites + blockIdx.x] = e;
  if (i >= st.size) return;
  if (e != 0) {
    const float sc = ldexpf(1.0f, -e);
    v.x *= sc;
    v.y *= sc;
  }
  (reinterpret_cast<float2*>(items + (uint64_t)g * item_bytes + sites_off) + st.offset)[i] = v;
}

__global__ void __launch_bounds__(kThreads) scale_kernel(
    const FoldSite* __restrict__ sites, char* hdr, uint64_t hdr_stride, char* items,
    uint64_t item_bytes, uint64_t sites_off, int n_sites) {
  launch_wait();
  launch_next();
  const FoldSite st = sites[blockIdx.y];
  const int g = blockIdx.z;
  const unsigned* maxabs = reinterpret_cast<const unsigned*>(hdr + (uint64_t)g * hdr_stride);
  const float m = __uint_as_float(maxabs[blockIdx.y]);
  int e = 0;
  if (m > 0.f) frexpf(m, &e);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    int* exps = reinterpret_cast<int*>(hdr + (uint64_t)g * hdr_stride) + n_sites;
    exps[blockIdx.y] = e;
  }
  const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (i >= st.size || e == 0) return;
  const float sc = ldexpf(1.0f, -e);
  float2* T = reinterpret_cast<float2*>(items + (uint64_t)g * item_bytes + sites_off) + st.offset;
  float2 v = T[i];
  v.x *= sc;
  v.y *= sc;
  T[i] = v;
}

__global__ void __launch_bounds__(kThreads) accumulate_kernel(
    const int32_t* __restrict__ open_perm, int n_open, int n_sites, int64_t n_batch,
    int64_t item0, int items, const char* hdr, uint64_t hdr_stride, const char* itemsp,
    uint64_t item_bytes, uint64_t final_off, double* out) {
  launch_wait();
  launch_next();
  const int64_t per = int64_t(1) << n_open;
  const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (t >= n_batch * per) return;
  const int64_t b = t / per, o = t % per;
  int64_t f = 0;
  for (int i = 0; i < n_open; ++i) f |= ((o >> i) & 1) << open_perm[i];
  // items of this chunk with batch index b, in increasing slice order
  int64_t first = item0 + ((b - item0 % n_batch) % n_batch + n_batch) % n_batch;
  // a row starts with its item of the first slice, so `out` needs no clearing
  const bool start = first < n_batch;
  double re = 0.0, im = 0.0;
  if (!start && first < item0 + items) {
    re = out[2 * t];
    im = out[2 * t + 1];
  }
  bool any = false;
  for (int64_t item = first; item < item0 + items; item += n_batch) {
    const int g = (int)(item - item0);
    const int* exps = reinterpret_cast<const int*>(hdr + (uint64_t)g * hdr_stride) + n_sites;
    int E = 0;
    for (int s = 0; s < n_sites; ++s) E += exps[s];
    const float2 c = reinterpret_cast<const float2*>(itemsp + (uint64_t)g * item_bytes + final_off)[f];
    re += ldexp((double)c.x, E);
    im += ldexp((double)c.y, E);
    any = true;
  }
  if (any) {
    out[2 * t] = re;
    out[2 * t + 1] = im;
  }
}

}  // namespace

static int launch_fold(const DeviceTables& t, int n_sites, int64_t max_site_size, int n_cuts,
                const uint64_t* x1, int x1_words, int64_t n_batch, int64_t slice_begin,
                int64_t item0, int items, char* hdr, uint64_t hdr_stride, char* itemsp,
                uint64_t item_bytes, uint64_t sites_off, void* stream) {
  // groups of 4 once they give every SM four blocks
  const int64_t grouped = (max_site_size + 4 * kThreads - 1) / (4 * kThreads) * n_sites * items;
  const int G = grouped >= 4 * (int64_t)num_sms() ? 4 : 1;
  const int64_t per_block = (int64_t)kThreads * G;
  dim3 grid((unsigned)((max_site_size + per_block - 1) / per_block), n_sites, items);
  auto kern = G == 4 ? fold_kernel<4> : fold_kernel<1>;
  count_launch();
  return (int)launch_early(kern, grid, dim3(kThreads), 0, (cudaStream_t)stream, t.sites, t.events, t.matsf, t.cuts,
                           n_cuts, x1, x1_words, n_batch, slice_begin, item0, hdr, hdr_stride, itemsp, item_bytes,
                           sites_off, n_sites);
}

static int launch_scale(const DeviceTables& t, int n_sites, int64_t max_site_size, int items,
                 char* hdr, uint64_t hdr_stride, char* itemsp, uint64_t item_bytes,
                 uint64_t sites_off, void* stream) {
  dim3 grid((unsigned)((max_site_size + kThreads - 1) / kThreads), n_sites, items);
  count_launch();
  return (int)launch_early(scale_kernel, grid, dim3(kThreads), 0, (cudaStream_t)stream, t.sites, hdr, hdr_stride,
                           itemsp, item_bytes, sites_off, n_sites);
}

int launch_sites(const DeviceTables& t, int n_sites, int64_t max_site_size, int n_cuts,
                 const uint64_t* x1, int x1_words, int64_t n_batch, int64_t slice_begin,
                 int64_t item0, int items, char* hdr, uint64_t hdr_stride, char* itemsp,
                 uint64_t item_bytes, uint64_t sites_off, void* stream) {
  // (with many items the grouped fold does less arithmetic, and its launches do not show)
  if (max_site_size <= kSmallSite && (int64_t)n_sites * items <= 8 * (int64_t)num_sms()) {
    count_launch();
    return (int)launch_early(fold_scale_kernel, dim3(n_sites, items), dim3((unsigned)((max_site_size + 31) / 32 * 32)),
                             0, (cudaStream_t)stream, t.sites, t.events, t.matsf, t.cuts, n_cuts, x1, x1_words,
                             n_batch, slice_begin, item0, hdr, hdr_stride, itemsp, item_bytes, sites_off, n_sites);
  }
  for (int g = 0; g < items; g += hdr_stride ? items : 1) {   // per-site maxima, from zero
    const cudaError_t e = cudaMemsetAsync(hdr + (uint64_t)g * hdr_stride, 0,
                                          hdr_stride ? (size_t)items * hdr_stride : (size_t)n_sites * 8,
                                          (cudaStream_t)stream);
    if (e != cudaSuccess) return (int)e;
  }
  const int err = launch_fold(t, n_sites, max_site_size, n_cuts, x1, x1_words, n_batch, slice_begin, item0, items,
                              hdr, hdr_stride, itemsp, item_bytes, sites_off, stream);
  return err ? err : launch_scale(t, n_sites, max_site_size, items, hdr, hdr_stride, itemsp, item_bytes, sites_off, stream);
}

int launch_accumulate(const DeviceTables& t, int n_sites, int n_open, int64_t n_batch,
                      int64_t item0, int items, const char* hdr, uint64_t hdr_stride,
                      const char* itemsp, uint64_t item_bytes, uint64_t final_off, double* out,
                      void* stream) {
  const int64_t total = n_batch << n_open;
  const unsigned blocks = (unsigned)((total + kThreads - 1) / kThreads);
  count_launch();
  return (int)launch_early(accumulate_kernel, dim3(blocks), dim3(kThreads), 0, (cudaStream_t)stream, t.open_perm,
                           n_open, n_sites, n_batch, item0, items, hdr, hdr_stride, itemsp, item_bytes, final_off,
                           out);
}

}  // namespace qfx
