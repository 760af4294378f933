// Projection of dense 3x3 kernels onto the PCONV constraint set (pattern per kernel + a keep rate
// over kernels): what turns trained weights into weights that pconv_pack accepts.  All on the device:
// per kernel the pattern that retains the largest sum of squares; the k-th largest retained sum by a
// radix select on the bits of the (non-negative) fp32 sums, 11 + 11 + 10 bits; masking.
//
// The weights are read twice (the second time partly from L2) and written once: 35 us at the copy rate for
// 4096x512 kernels, of which it takes 101 us -- scoring 35, masking 35, digits 24, ids 7.  What the scoring and
// masking passes spend the rest on has not been shown; ~200 instructions a kernel are 11 us of issue.  Five
// launches: the first digit's histogram is taken where the sums are formed, and the block that finishes a
// histogram last picks the digit, so no launch exists for the picks.
#include <algorithm>
#include <cstring>

#include "pconv_internal.h"

namespace pconv {
namespace {

constexpr int kThreads = 256;
constexpr int kBlockKernels = 1024;      // 3x3 kernels that a block stages at a time (36 KB)
constexpr int kBins = 2048;

struct PatternSet {
  int n;
  uint16_t mask[PCONV_MAX_PATTERNS];
};

struct SelectState {
  unsigned int prefix;        // the bits of the threshold found so far (higher digits)
  unsigned int remaining;     // rank (from the top, 1-based) still to be found inside the prefix; 0 = not begun
  unsigned int done[3];       // blocks that have added their histogram of a pass
  unsigned int hist[3][kBins];
};

__device__ __forceinline__ void dependents_and_wait() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Adds the block's histogram to the pass's; the block that is the last to do so picks the digit whose
// bucket holds the wanted rank, counting from the largest digit down.
__device__ __forceinline__ void finish_pass(const unsigned int* h, SelectState* st, int pass, int shift, unsigned int rank) {
  __shared__ unsigned int warp_sum[kThreads / 32];
  __shared__ bool last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __syncthreads();
  for (int b = tid; b < kBins; b += kThreads)
    if (h[b]) atomicAdd(&st->hist[pass][b], h[b]);
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(&st->done[pass], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  // thread t sums the eight bins below 2048 - 8 t
  constexpr int kPer = kBins / kThreads;
  unsigned int v[kPer], sum = 0;
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    v[i] = __ldcg(&st->hist[pass][kBins - 1 - (tid * kPer + i)]);
    sum += v[i];
  }
  unsigned int before = sum;               // inclusive, then exclusive prefix over the threads
#pragma unroll
  for (int d = 1; d < 32; d *= 2) {
    const unsigned int o = __shfl_up_sync(0xffffffffu, before, d);
    if (lane >= d) before += o;
  }
  if (lane == 31) warp_sum[warp] = before;
  __syncthreads();
  for (int w = 0; w < warp; ++w) before += warp_sum[w];
  before -= sum;
  const unsigned int want = pass == 0 ? rank : st->remaining;
  __syncthreads();
  if (before < want && want <= before + sum) {
    unsigned int left = want - before;
    int i = 0;
    for (; i < kPer - 1 && left > v[i]; ++i) left -= v[i];
    st->prefix = (pass == 0 ? 0u : st->prefix) | (unsigned int)(kBins - 1 - (tid * kPer + i)) << shift;
    st->remaining = left;
  }
}

// Retained sum of squares under every pattern; the first maximum wins.  Separate multiply and add
// in ascending tap order: the decision must not depend on how the compiler contracts the sum.  The
// weights pass through shared memory: 16-byte loads, and rows of nine words have no bank conflicts
// (straight from global memory every load touches nine lines a warp).
__global__ void __launch_bounds__(kThreads) score_kernel(const float* __restrict__ w, long long n, PatternSet ps,
                                                         float* __restrict__ best, signed char* __restrict__ pid,
                                                         SelectState* st, unsigned int rank) {
  __shared__ __align__(16) float tile[kBlockKernels * 9];
  __shared__ unsigned int h[kBins];
  dependents_and_wait();
  for (int b = threadIdx.x; b < kBins; b += kThreads) h[b] = 0;
  const bool aligned = (reinterpret_cast<uintptr_t>(w) & 15u) == 0;
  for (long long k0 = (long long)blockIdx.x * kBlockKernels; k0 < n; k0 += (long long)gridDim.x * kBlockKernels) {
    const int kn = (int)(n - k0 < kBlockKernels ? n - k0 : kBlockKernels);
    const float* src = w + k0 * 9;
    __syncthreads();
    if (aligned && kn == kBlockKernels) {
#pragma unroll
      for (int i = 0; i < kBlockKernels * 9 / 4 / kThreads; ++i)
        reinterpret_cast<float4*>(tile)[threadIdx.x + i * kThreads] =
            __ldg(reinterpret_cast<const float4*>(src) + threadIdx.x + i * kThreads);
    } else {
      for (int i = threadIdx.x; i < kn * 9; i += kThreads) tile[i] = __ldg(src + i);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kn; k += kThreads) {
      float sq[9];
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        const float v = tile[k * 9 + t];
        sq[t] = __fmul_rn(v, v);
      }
      float top = -1.f;
      int arg = 0;
      for (int p = 0; p < ps.n; ++p) {
        float s = 0.f;
#pragma unroll
        for (int t = 0; t < 9; ++t)
          if (ps.mask[p] >> t & 1) s = __fadd_rn(s, sq[t]);
        if (s > top) {
          top = s;
          arg = p;
        }
      }
      best[k0 + k] = top;
      pid[k0 + k] = (signed char)arg;
      atomicAdd(&h[__float_as_uint(top) >> 21], 1u);
    }
  }
  finish_pass(h, st, 0, 21, rank);
}

// A later digit: histogram of the values whose higher digits are those found so far.
__global__ void __launch_bounds__(kThreads) digit_kernel(const float* __restrict__ best, long long n, int pass, int shift,
                                                         int bits, SelectState* st) {
  __shared__ unsigned int h[kBins];
  dependents_and_wait();
  for (int b = threadIdx.x; b < kBins; b += kThreads) h[b] = 0;
  __syncthreads();
  const unsigned int prefix = st->prefix, high = 0xFFFFFFFFu << (shift + bits), low = (1u << bits) - 1u;
  auto count = [&](float f) {
    const unsigned int b = __float_as_uint(f);
    if ((b & high) == (prefix & high)) atomicAdd(&h[b >> shift & low], 1u);
  };
  const long long n4 = n / 4;
  for (long long i = blockIdx.x * (long long)kThreads + threadIdx.x; i < n4; i += (long long)gridDim.x * kThreads) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(best) + i);
    count(v.x);
    count(v.y);
    count(v.z);
    count(v.w);
  }
  if (blockIdx.x == 0 && threadIdx.x < n - 4 * n4) count(best[4 * n4 + threadIdx.x]);
  finish_pass(h, st, pass, shift, 0);
}

// Masks the flat array, V values a thread (4: 16-byte accesses).  `out` may be `w` itself (in-place
// use), so neither pointer is declared restrict; a value is read by the thread that writes it.
template <int V>
__global__ void __launch_bounds__(kThreads) mask_kernel(const float* w, long long n, PatternSet ps,
                                                        const float* __restrict__ best,
                                                        const SelectState* __restrict__ st, int keep_none, float* out,
                                                        const signed char* __restrict__ pid) {
  __shared__ unsigned int mask_s[PCONV_MAX_PATTERNS];
  if (threadIdx.x < PCONV_MAX_PATTERNS) mask_s[threadIdx.x] = ps.mask[threadIdx.x];
  dependents_and_wait();
  __syncthreads();
  const unsigned int limit = st->prefix;
  const long long all = n * 9;
  for (long long e = (blockIdx.x * (long long)kThreads + threadIdx.x) * V; e < all;
       e += (long long)gridDim.x * kThreads * V) {
    const long long k = e / 9;
    const int t0 = (int)(e - k * 9);
    // the masks of the (at most two) kernels these values belong to, one after the other
    unsigned int bits = 0;
#pragma unroll
    for (int j = 0; j < (V > 1 ? 2 : 1); ++j)
      if (k + j < n && (j == 0 || t0 + V > 9)) {
        const bool kept = !keep_none && __float_as_uint(__ldg(best + k + j)) >= limit;   // ties with the k-th stay
        if (kept) bits |= mask_s[__ldg(pid + k + j)] << (9 * j);
      }
    bits >>= t0;
    if (V == 4 && e + 4 <= all) {
      float4 v = *reinterpret_cast<const float4*>(w + e);
      v.x = (bits & 1u) ? v.x : 0.f;
      v.y = (bits & 2u) ? v.y : 0.f;
      v.z = (bits & 4u) ? v.z : 0.f;
      v.w = (bits & 8u) ? v.w : 0.f;
      *reinterpret_cast<float4*>(out + e) = v;
    } else {
      for (int i = 0; i < V && e + i < all; ++i) out[e + i] = (bits >> i & 1u) ? w[e + i] : 0.f;
    }
  }
}

// Pattern ids of the kernels that went.
__global__ void __launch_bounds__(kThreads) drop_kernel(const float* __restrict__ best, long long n,
                                                        const SelectState* __restrict__ st, int keep_none,
                                                        signed char* __restrict__ pid) {
  dependents_and_wait();
  const unsigned int limit = st->prefix;
  for (long long i = blockIdx.x * (long long)kThreads + threadIdx.x; i < n; i += (long long)gridDim.x * kThreads)
    if (keep_none || __float_as_uint(__ldg(best + i)) < limit) pid[i] = -1;
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace
}  // namespace pconv

using namespace pconv;

extern "C" pconv_status pconv_project_workspace_bytes(long long n_kernels, size_t* bytes) {
  if (!bytes) return PCONV_ERR_NULL;
  if (n_kernels < 0) return PCONV_ERR_SHAPE;
  *bytes = align256((size_t)n_kernels * 4) + align256(sizeof(SelectState));
  return PCONV_OK;
}

extern "C" pconv_status pconv_project(const float* w_dev, long long n_kernels,
                                      const uint16_t* patterns, int n_patterns, double keep,
                                      float* w_out_dev, signed char* pattern_id_dev, void* ws_dev,
                                      size_t ws_bytes, void* stream_v) {
  if (!w_dev || !patterns || !w_out_dev || !pattern_id_dev || !ws_dev) return PCONV_ERR_NULL;
  if (n_kernels < 0 || !(keep >= 0.0 && keep <= 1.0)) return PCONV_ERR_SHAPE;
  if (n_patterns < 1 || n_patterns > PCONV_MAX_PATTERNS) return PCONV_ERR_PATTERN_SET;
  PatternSet ps;
  std::memset(&ps, 0, sizeof(ps));
  ps.n = n_patterns;
  for (int p = 0; p < n_patterns; ++p) {
    if (patterns[p] >= 512 || __builtin_popcount(patterns[p]) != 4) return PCONV_ERR_PATTERN_SET;
    for (int q = 0; q < p; ++q)
      if (patterns[q] == patterns[p]) return PCONV_ERR_PATTERN_SET;
    ps.mask[p] = patterns[p];
  }
  size_t need = 0;
  pconv_project_workspace_bytes(n_kernels, &need);
  if (ws_bytes < need) return PCONV_ERR_WORKSPACE;
  if (((uintptr_t)ws_dev & 255u) || ((uintptr_t)w_dev & 3u) || ((uintptr_t)w_out_dev & 3u)) return PCONV_ERR_ALIGN;
  if (n_kernels == 0) return PCONV_OK;
  cudaStream_t stream = (cudaStream_t)stream_v;
  float* best = (float*)ws_dev;
  SelectState* st = (SelectState*)((char*)ws_dev + align256((size_t)n_kernels * 4));
  long long k = (long long)(keep * (double)n_kernels + 0.5);
  if (k > n_kernels) k = n_kernels;
  const int keep_none = k == 0;
  if (n_kernels > 0xFFFFFFFFll) return PCONV_ERR_SHAPE;
  const long long blocks = (n_kernels + kBlockKernels - 1) / kBlockKernels;
  if (blocks > 0x7FFFFFFF) return PCONV_ERR_SHAPE;
  if (cudaMemsetAsync(st, 0, sizeof(SelectState), stream) != cudaSuccess) {
    cudaGetLastError();
    return PCONV_ERR_CUDA;
  }
  const long long sms = device_sm_count();
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto grid = [&](long long want, long long per_sm) {
    cfg.gridDim = dim3((unsigned)std::max<long long>(1, std::min(want, sms * per_sm)), 1, 1);
  };
  grid(blocks, 5);
  cudaError_t e = cudaLaunchKernelEx(&cfg, score_kernel, w_dev, n_kernels, ps, best, pattern_id_dev, st,
                                     (unsigned int)(k > 0 ? k : 1));
  grid((n_kernels + 4 * kThreads - 1) / (4 * kThreads), 4);
  if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, digit_kernel, (const float*)best, n_kernels, 1, 10, 11, st);
  if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, digit_kernel, (const float*)best, n_kernels, 2, 0, 10, st);
  const bool wide = (((uintptr_t)w_dev | (uintptr_t)w_out_dev) & 15u) == 0;
  grid((n_kernels * 9 + 4 * kThreads - 1) / (4 * kThreads), 32);
  if (e == cudaSuccess)
    e = wide ? cudaLaunchKernelEx(&cfg, mask_kernel<4>, w_dev, n_kernels, ps, (const float*)best,
                                  (const SelectState*)st, keep_none, w_out_dev, (const signed char*)pattern_id_dev)
             : cudaLaunchKernelEx(&cfg, mask_kernel<1>, w_dev, n_kernels, ps, (const float*)best,
                                  (const SelectState*)st, keep_none, w_out_dev, (const signed char*)pattern_id_dev);
  grid((n_kernels + kThreads - 1) / kThreads, 8);
  if (e == cudaSuccess)
    e = cudaLaunchKernelEx(&cfg, drop_kernel, (const float*)best, n_kernels, (const SelectState*)st, keep_none,
                           pattern_id_dev);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return PCONV_ERR_CUDA;
  }
  return PCONV_OK;
}
