// Threshold calibration (App. A.2, "Threshold Calibration"): the similarity of every benign pair, the nearest-rank
// percentile of those similarities, and the capped threshold min(cap, percentile).
//
//   pair_sim_kernel   one warp per pair: fp32 dot of two bf16 rows (16-byte loads, each lane's chunks in order,
//                     butterfly sum). HBM-bound: 4d bytes per pair.
//   select_*          the exact k-th smallest similarity by a three-pass radix select (11, 11, 10 bits) over the
//                     similarities mapped to order-preserving unsigned integers. Up to kClusterMax similarities one
//                     launch does all of it (select_cluster: one CTA, or a cluster of eight, holding the values in
//                     registers); more take, per pass, a count over all CTAs (shared histograms, warp-aggregated
//                     adds) into a global histogram, then a one-CTA pick.
#include <math.h>

#include "internal.cuh"

namespace lc {
namespace {

constexpr int kPairWarps = 8;

__device__ __forceinline__ float dot8(const uint4& u, const uint4& v, float acc) {
  const __nv_bfloat162* a = reinterpret_cast<const __nv_bfloat162*>(&u);
  const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 x = __bfloat1622float2(a[e]);
    const float2 y = __bfloat1622float2(b[e]);
    acc = fmaf(x.x, y.x, acc);
    acc = fmaf(x.y, y.y, acc);
  }
  return acc;
}

__global__ void __launch_bounds__(kPairWarps * 32)
    pair_sim_kernel(const uint4* __restrict__ x, const uint4* __restrict__ y, int64_t n, int d,
                    float* __restrict__ sims) {
  // select_cluster may be scheduled now: it waits for this grid before reading the similarities
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * kPairWarps + (threadIdx.x >> 5);
  if (i >= n) return;
  const int v = d / 8;
  float acc = 0.f;
  for (int c = lane; c < v; c += 32) acc = dot8(__ldg(x + i * v + c), __ldg(y + i * v + c), acc);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) sims[i] = acc;
}

// Exact k-th smallest similarity: a radix select over the order-preserving integer image of the floats, 11, 11
// and 10 bits per pass. Each pass counts, over all CTAs, the elements whose higher bits equal the prefix chosen so
// far; a one-CTA kernel then picks the bin that holds the rank and narrows the prefix.
constexpr int kBins = 2048;
constexpr int kCountThreads = 1024;
constexpr int kPerThread = 8;

struct SelectState {
  uint32_t prefix;
  uint32_t mask;
  int64_t rank;   // rank still to find among the elements matching prefix under mask (0-based)
};

__device__ __forceinline__ unsigned int* ws_hist(void* ws) { return static_cast<unsigned int*>(ws); }
__device__ __forceinline__ SelectState* ws_state(void* ws) {
  return reinterpret_cast<SelectState*>(static_cast<unsigned char*>(ws) + kBins * 4);
}

__global__ void select_init(void* ws, int64_t rank) {
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) ws_hist(ws)[b] = 0;
  if (threadIdx.x == 0) *ws_state(ws) = SelectState{0u, 0u, rank};
}

__global__ void __launch_bounds__(kCountThreads)
    select_count(const float* __restrict__ sims, int64_t n, void* ws, int shift, uint32_t bin_mask) {
  __shared__ unsigned int hist[kBins];
  const int lane = threadIdx.x & 31;
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) hist[b] = 0;
  __syncthreads();
  const SelectState st = *ws_state(ws);
  const int64_t step = (int64_t)gridDim.x * blockDim.x * kPerThread;
  const int64_t n_round = (n + step - 1) / step * step;   // uniform trip count: every lane reaches __match_any_sync
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x * kPerThread; base < n_round; base += step) {
    float v[kPerThread];
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) {
      const int64_t i = base + (int64_t)u * blockDim.x + threadIdx.x;
      v[u] = i < n ? __ldg(sims + i) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) {
      const int64_t i = base + (int64_t)u * blockDim.x + threadIdx.x;
      uint32_t bin = kBins;   // not counted
      if (i < n) {
        const uint32_t o = score_order(v[u]);
        if ((o & st.mask) == st.prefix) bin = (o >> shift) & bin_mask;
      }
      const unsigned peers = __match_any_sync(0xffffffffu, bin);
      if (bin < kBins && lane == __ffs(peers) - 1) atomicAdd(&hist[bin], __popc(peers));
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kBins; b += blockDim.x)
    if (hist[b]) atomicAdd(&ws_hist(ws)[b], hist[b]);
}

// One CTA of kBins / 2 threads: exclusive scan of the histogram, the bin holding the rank, the narrowed prefix;
// the histogram is cleared for the next pass. After the last pass the prefix is the value itself.
__global__ void __launch_bounds__(kBins / 2)
    select_pick(void* ws, int shift, uint32_t bin_mask, float cap, float* __restrict__ out, int last) {
  __shared__ unsigned long long part[kBins / 2];
  __shared__ int s_bin;
  __shared__ unsigned long long s_below;
  unsigned int* gh = ws_hist(ws);
  SelectState* st = ws_state(ws);
  const int t = threadIdx.x;
  const unsigned long long c0 = gh[2 * t], c1 = gh[2 * t + 1];
  part[t] = c0 + c1;
  __syncthreads();
  for (int off = 1; off < kBins / 2; off <<= 1) {   // inclusive scan (Hillis-Steele)
    const unsigned long long add = t >= off ? part[t - off] : 0;
    __syncthreads();
    part[t] += add;
    __syncthreads();
  }
  const unsigned long long before = t ? part[t - 1] : 0;
  const unsigned long long r = (unsigned long long)st->rank;
  if (r >= before && r < before + c0 + c1) {
    const bool first = r < before + c0;
    s_bin = 2 * t + (first ? 0 : 1);
    s_below = first ? before : before + c0;
  }
  __syncthreads();
  gh[2 * t] = 0;
  gh[2 * t + 1] = 0;
  if (t == 0) {
    SelectState nx = *st;
    nx.prefix |= (uint32_t)s_bin << shift;
    nx.mask |= bin_mask << shift;
    nx.rank = (int64_t)(r - s_below);
    *st = nx;
    if (last) {
      const float value = score_of_order(nx.prefix);
      out[0] = value;
      out[1] = fminf(cap, value);
    }
  }
}

// The whole select in one launch of one cluster of G CTAs: thread t of the cluster holds the similarities t, t + T,
// t + 2 T, ... (T threads in all, at most kPer each). Each pass counts into the CTA's own shared histogram; after a
// cluster barrier every CTA adds up all G histograms (through distributed shared memory) and picks the same bin.
// Bound by latency. A call (similarities included), against separate kernels for the set-up and for each pass's count
// and pick (us, calls back to back, before / after): 500 pairs x 1024 39.0 / 10.7, 5,000 x 384 41.0 / 12.3, 16,384 x 768
// 45.1 / 24.7, 60,000 x 384 53.3 / 41.0, 131,072 x 768 98.4 / 95.5. Past that the values no longer fit the cluster's
// registers, and counting on all SMs is as fast.
constexpr int kSelThreads = 1024;
constexpr int kPer = 16;
constexpr int kSelCluster = 8;
constexpr int64_t kCtaMax = (int64_t)kSelThreads * kPer;           // one CTA
constexpr int64_t kClusterMax = kCtaMax * kSelCluster;             // a cluster
static_assert(kBins == 2 * kSelThreads, "two bins per thread");

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// The word at the same shared-memory address in CTA `rank` of the cluster.
__device__ __forceinline__ unsigned int ld_cluster(const unsigned int* p, uint32_t rank) {
  uint32_t addr, v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(addr)
               : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

template <int G>
__global__ void __launch_bounds__(kSelThreads)
    select_cluster(const float* __restrict__ sims, int n, int rank, float cap, float* __restrict__ out) {
  __shared__ unsigned int hist[kBins];
  __shared__ unsigned int warp_sum[kSelThreads / 32];
  __shared__ int s_bin, s_below;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int first = blockIdx.x * kSelThreads + t;
  hist[2 * t] = hist[2 * t + 1] = 0;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  uint32_t v[kPer];
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const int i = first + u * G * kSelThreads;
    v[u] = i < n ? score_order(__ldcg(sims + i)) : 0u;
  }
  uint32_t prefix = 0, mask = 0;
#pragma unroll
  for (int pass = 0; pass < 3; ++pass) {
    const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0;
    const uint32_t bin_mask = pass == 2 ? 0x3FFu : 0x7FFu;
    __syncthreads();   // the histogram is clear
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      if (u * G * kSelThreads >= n) break;   // the same for every thread
      const bool counted = first + u * G * kSelThreads < n && (v[u] & mask) == prefix;
      const uint32_t bin = counted ? (v[u] >> shift) & bin_mask : (uint32_t)kBins;
      const unsigned peers = __match_any_sync(0xffffffffu, bin);
      if (counted && lane == __ffs(peers) - 1) atomicAdd(&hist[bin], __popc(peers));
    }
    // bins 2t and 2t + 1 over the cluster, and the counts below them (an inclusive scan over warps, then their totals)
    unsigned int c0 = 0, c1 = 0;
    if constexpr (G > 1) {
      cluster_barrier();
      for (uint32_t g = 0; g < (uint32_t)G; ++g) {
        c0 += ld_cluster(hist + 2 * t, g);
        c1 += ld_cluster(hist + 2 * t + 1, g);
      }
      cluster_barrier();   // every CTA has read the histograms before they are cleared (and before any CTA exits)
    } else {
      __syncthreads();
      c0 = hist[2 * t];
      c1 = hist[2 * t + 1];
    }
    hist[2 * t] = hist[2 * t + 1] = 0;
    unsigned int before = c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int x = __shfl_up_sync(0xffffffffu, before, o);
      if (lane >= o) before += x;
    }
    if (lane == 31) warp_sum[warp] = before;
    __syncthreads();
    before -= c0 + c1;
    unsigned int total = lane < warp ? warp_sum[lane] : 0u;
    before += __reduce_add_sync(0xffffffffu, total);
    if ((unsigned)rank >= before && (unsigned)rank < before + c0 + c1) {
      const bool lo = (unsigned)rank < before + c0;
      s_bin = 2 * t + (lo ? 0 : 1);
      s_below = (int)(lo ? before : before + c0);
    }
    __syncthreads();
    prefix |= (uint32_t)s_bin << shift;
    mask |= bin_mask << shift;
    rank -= s_below;
  }
  if (blockIdx.x == 0 && t == 0) {
    const float value = score_of_order(prefix);
    out[0] = value;
    out[1] = fminf(cap, value);
  }
}

template <int G>
cudaError_t launch_select_cluster(const float* sims, int n, int rank, float cap, float* out, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(kSelThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = G;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = G > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, select_cluster<G>, sims, n, rank, cap, out);
}

}  // namespace

size_t calibrate_workspace_bytes() { return kBins * 4 + sizeof(SelectState); }

cudaError_t launch_calibrate(const void* x, const void* y, int64_t n, int d, int64_t rank, float cap, float* sims,
                             float* result, void* ws, int num_sms, cudaStream_t st) {
  const int64_t blocks = (n + kPairWarps - 1) / kPairWarps;
  pair_sim_kernel<<<(unsigned)blocks, kPairWarps * 32, 0, st>>>(static_cast<const uint4*>(x),
                                                                 static_cast<const uint4*>(y), n, d, sims);
  if (n <= kClusterMax) {
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return n <= kCtaMax ? launch_select_cluster<1>(sims, (int)n, (int)rank, cap, result, st)
                        : launch_select_cluster<kSelCluster>(sims, (int)n, (int)rank, cap, result, st);
  }
  select_init<<<1, 1024, 0, st>>>(ws, rank);
  const int64_t want = (n + (int64_t)kCountThreads * kPerThread - 1) / ((int64_t)kCountThreads * kPerThread);
  const int grid = (int)(want < 2 * num_sms ? want : 2 * num_sms);
  const int shifts[3] = {21, 10, 0};
  const uint32_t masks[3] = {0x7FFu, 0x7FFu, 0x3FFu};
  for (int pass = 0; pass < 3; ++pass) {
    select_count<<<grid, kCountThreads, 0, st>>>(sims, n, ws, shifts[pass], masks[pass]);
    select_pick<<<1, kBins / 2, 0, st>>>(ws, shifts[pass], masks[pass], cap, result, pass == 2);
  }
  return cudaGetLastError();
}

}  // namespace lc

extern "C" size_t lacache_calibrate_workspace_bytes(void) { return lc::calibrate_workspace_bytes(); }

extern "C" lacache_status lacache_calibrate(int64_t n, int32_t d, const void* x_dev, const void* y_dev,
                                            double percentile, float cap, float* sims_dev, float* result_dev,
                                            void* workspace_dev, void* cuda_stream) {
  lc::NvtxRange nvtx("lacache_calibrate");
  if (n < 1 || n > (int64_t)INT32_MAX || d <= 0 || !x_dev || !y_dev || !sims_dev || !result_dev || !workspace_dev)
    return LACACHE_ERR_INVALID_ARG;
  if (!(percentile >= 0.0 && percentile <= 100.0) || isnan(cap)) return LACACHE_ERR_INVALID_ARG;
  if (d % 8 != 0 || d > lc::kMaxD) return LACACHE_ERR_UNSUPPORTED;
  if (((uintptr_t)x_dev & 15u) || ((uintptr_t)y_dev & 15u) || ((uintptr_t)workspace_dev & 15u))
    return LACACHE_ERR_INVALID_ARG;
  // nearest rank: ceil(percentile / 100 * n), at least 1 and at most n; the kernels take it 0-based
  int64_t rank = (int64_t)ceil(percentile / 100.0 * (double)n);
  if (rank < 1) rank = 1;
  if (rank > n) rank = n;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return LACACHE_ERR_CUDA;
  return lc::launch_calibrate(x_dev, y_dev, n, d, rank - 1, cap, sims_dev, result_dev, workspace_dev, sms,
                              (cudaStream_t)cuda_stream) == cudaSuccess
             ? LACACHE_OK
             : LACACHE_ERR_CUDA;
}
