// Per-layer top-k anchors by radix select, plus MinMax normalisation (Section 3.2; Appendix A.1).
// One thread-block cluster per (layer, request) segment, a contiguous slice of the segment per block: radix passes of
// 11, 11 and 10 bits that find the k-th largest score exactly, then an index-ordered compaction so that equal scores go
// to the lower position and the anchors come out ascending.
#include "common.cuh"
#include "select.cuh"
#include "sm100_ptx.cuh"
#include <algorithm>

namespace relaxkv {

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelBins = 2048;                  // bins of a radix pass (the last one uses half)
constexpr int kSelKeysMax = 24576;              // keys of a block's slice kept in shared memory (96 KB)

// Monotone map float -> uint32 (larger float, larger key), and back.
__device__ __forceinline__ uint32_t order_key(float x) {
  const uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float order_value(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t cluster_addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_addr) : "memory");
  return v;
}
__device__ __forceinline__ uint2 ld_cluster_u32x2(uint32_t cluster_addr) {
  uint2 v;
  asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(cluster_addr) : "memory");
  return v;
}

// Exclusive prefix over the block of one counter per thread (one barrier; `warp_tot` is overwritten).
__device__ __forceinline__ int block_prefix(int v, int* warp_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  const int w = lane < warp ? warp_tot[lane] : 0;        // every warp adds up the totals before it
  return warp_reduce_sum(w) + inc - v;
}

// What bounds this kernel is latency: a segment is 4 KB to 256 KB, and the passes over it depend on one another.  One
// block per segment spent 16 us on 1 K scores (one thread walking 256 bins four times) and 32 / 72 / 124 us on segments
// of 16 K / 32 K / 64 K scores (each pass a block-wide walk through L2).  Here a slice's keys are read once and stay in
// shared memory (slices above kSelKeysMax keys are read again from L2 in each pass), the histograms of a
// cluster's blocks are added through distributed shared memory by every block for itself, and the bin is found by a
// block-wide prefix: 4.5 us, and 10.1 / 13.5 (15.7 for 40 segments) / 15.6 us.
template <int NS>                                          // slices = blocks of a cluster
__global__ void __launch_bounds__(kSelThreads)
select_topk_kernel(ReqTable rt, int n_layers, int keys_cap, const float* raw, float* norm, int* anchors, DeviceStatus* st) {
  extern __shared__ uint32_t s_keys[];                     // [keys_cap]
  __shared__ __align__(16) uint32_t s_hist[3][kSelBins];
  __shared__ int s_tot[3][kSelWarps], s_cnt[2][kSelWarps];
  __shared__ uint32_t s_lo[kSelWarps], s_hi[kSelWarps];
  __shared__ uint32_t s_found[3][2];                       // bin, how many are still needed from it
  __shared__ uint32_t s_pub[4];                            // read by the cluster: slice minimum, maximum; counts > and ==
  const int B = rt.n_req;
  const int slice = (int)blockIdx.x % NS, seg = (int)blockIdx.x / NS;
  const int l = seg / B, b = seg % B;
  const int T = rt.ctx_len[b];
  const int k = rt.k[b];
  const long long sum_t = rt.ctx_cu[B];
  const int per = ((T + NS - 1) / NS + 31) & ~31;
  const int i0 = min(T, slice * per), n = min(T, i0 + per) - i0;
  const float* x = raw + (long long)l * sum_t + rt.ctx_cu[b] + i0;
  int* out = anchors + (long long)l * rt.k_cu[B] + rt.k_cu[b];
  const bool cached = per <= keys_cap;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto key_at = [&](int i) -> uint32_t { return cached ? s_keys[i] : order_key(x[i]); };
  auto all_sync = [] { if (NS > 1) ptx::cluster_sync(); else __syncthreads(); };

  for (int i = threadIdx.x; i < 3 * kSelBins; i += kSelThreads) (&s_hist[0][0])[i] = 0u;
  griddep_launch();
  griddep_wait();
  __syncthreads();

  // ---- keys, slice minimum / maximum (in key order: the order of the floats), first histogram --------------------------
  uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += kSelThreads) {
    const uint32_t key = order_key(x[i]);
    if (cached) s_keys[i] = key;
    if (norm != nullptr) {
      const float v = order_value(key);
      if (v == v) { lo = min(lo, key); hi = max(hi, key); }      // a NaN takes no part in the range, as with fminf / fmaxf
    }
    atomicAdd(&s_hist[0][key >> 21], 1u);
  }
  if (norm != nullptr) {
    lo = __reduce_min_sync(0xffffffffu, lo); hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) { s_lo[warp] = lo; s_hi[warp] = hi; }
    __syncthreads();
    if (warp == 0) {
      lo = __reduce_min_sync(0xffffffffu, s_lo[lane]); hi = __reduce_max_sync(0xffffffffu, s_hi[lane]);
      if (lane == 0) { s_pub[0] = lo; s_pub[1] = hi; }
    }
  }

  // ---- the k-th largest key: 11 + 11 + 10 bits ---------------------------------------------------------------------------
  uint32_t prefix = 0u;
  int need = k;
#pragma unroll
  for (int pass = 0; pass < 3; ++pass) {
    const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0), below = pass == 0 ? 32 : (pass == 1 ? 21 : 10);
    const uint32_t bin_mask = pass == 2 ? 1023u : 2047u;
    if (pass > 0) {
#pragma unroll 4
      for (int i = threadIdx.x; i < n; i += kSelThreads) {
        const uint32_t key = key_at(i);
        if ((key >> below) == prefix) atomicAdd(&s_hist[pass][(key >> shift) & bin_mask], 1u);
      }
    }
    all_sync();                                            // every slice's histogram is complete
    // thread t looks at bins 2047 - 2t and 2046 - 2t: prefixes run from the largest key down
    const int b0 = kSelBins - 1 - 2 * (int)threadIdx.x;
    const uint2 own = *reinterpret_cast<const uint2*>(&s_hist[pass][b0 - 1]);
    uint2 other[NS];
    const uint32_t hist_addr = ptx::smem_u32(&s_hist[pass][b0 - 1]);
#pragma unroll
    for (int r = 1; r < NS; ++r) other[r] = ld_cluster_u32x2(ptx::mapa_shared(hist_addr, (uint32_t)((slice + r) % NS)));
    int c0 = (int)own.y, c1 = (int)own.x;
#pragma unroll
    for (int r = 1; r < NS; ++r) { c0 += (int)other[r].y; c1 += (int)other[r].x; }
    const int before = block_prefix(c0 + c1, s_tot[pass]);
    if (before < need && need <= before + c0 + c1) {       // exactly one thread
      const bool second = need > before + c0;
      s_found[pass][0] = (uint32_t)(second ? b0 - 1 : b0);
      s_found[pass][1] = (uint32_t)(need - before - (second ? c0 : 0));
    }
    __syncthreads();
    prefix = (prefix << (below - shift)) | s_found[pass][0];
    need = (int)s_found[pass][1];
  }
  const uint32_t tau = prefix;             // key of the k-th largest score
  const int need_eq = need;                // how many elements equal to it are selected (lowest positions), >= 1

  // ---- ordered compaction: a contiguous run of the slice per warp -----------------------------------------------------------
  const int run = ((n + kSelWarps - 1) / kSelWarps + 31) & ~31;
  const int r0 = min(n, warp * run), r1 = min(n, r0 + run);
  int ngt = 0, neq = 0;
#pragma unroll 4
  for (int i = r0 + lane; i < r1; i += 32) { const uint32_t key = key_at(i); ngt += (key > tau); neq += (key == tau); }
  ngt = warp_reduce_sum(ngt); neq = warp_reduce_sum(neq);
  if (lane == 0) { s_cnt[0][warp] = ngt; s_cnt[1][warp] = neq; }
  __syncthreads();
  const int cg = s_cnt[0][lane], ce = s_cnt[1][lane];
  int egt = warp_reduce_sum(lane < warp ? cg : 0), eeq = warp_reduce_sum(lane < warp ? ce : 0);
  if (NS > 1) {
    if (warp == 0) {
      const int tg = warp_reduce_sum(cg), te = warp_reduce_sum(ce);
      if (lane == 0) { s_pub[2] = (uint32_t)tg; s_pub[3] = (uint32_t)te; }
    }
    all_sync();
    uint32_t g = 0u, e = 0u;                                // lane r fetches the counts of slice r
    if (lane < slice) {
      g = ld_cluster_u32(ptx::mapa_shared(ptx::smem_u32(&s_pub[2]), (uint32_t)lane));
      e = ld_cluster_u32(ptx::mapa_shared(ptx::smem_u32(&s_pub[3]), (uint32_t)lane));
    }
    egt += warp_reduce_sum((int)g); eeq += warp_reduce_sum((int)e);
  }
  const uint32_t below_lane = (1u << lane) - 1u;
  for (int i = r0; i < r1; i += 32) {                       // whole warps: r1 may cut the last one
    const bool in = i + lane < r1;
    const uint32_t key = in ? key_at(i + lane) : 0u;
    const uint32_t mgt = __ballot_sync(0xffffffffu, in && key > tau), meq = __ballot_sync(0xffffffffu, in && key == tau);
    const int my_gt = egt + __popc(mgt & below_lane), my_eq = eeq + __popc(meq & below_lane);
    if (in && (key > tau || (key == tau && my_eq < need_eq))) {
      const int o = my_gt + min(my_eq, need_eq);
      if (o < k) out[o] = i0 + i + lane; else report(st, RELAXKV_ERR_BAD_INDEX, KID_SELECT, o, k);
    }
    egt += __popc(mgt); eeq += __popc(meq);
  }

  // ---- MinMax ---------------------------------------------------------------------------------------------------------------
  if (norm != nullptr) {                                    // s_pub[0..1] of every slice: complete since the first pass
    uint32_t klo = 0xffffffffu, khi = 0u;
    if (lane < NS) {
      klo = ld_cluster_u32(ptx::mapa_shared(ptx::smem_u32(&s_pub[0]), (uint32_t)lane));
      khi = ld_cluster_u32(ptx::mapa_shared(ptx::smem_u32(&s_pub[1]), (uint32_t)lane));
    }
    klo = __reduce_min_sync(0xffffffffu, klo); khi = __reduce_max_sync(0xffffffffu, khi);
    const float vlo = klo <= khi ? order_value(klo) : INFINITY, vhi = klo <= khi ? order_value(khi) : -INFINITY;
    const float range = vhi - vlo;
    float* nb = norm + (long long)l * sum_t + rt.ctx_cu[b] + i0;
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kSelThreads) nb[i] = (range > 0.f) ? (order_value(key_at(i)) - vlo) / range : 0.f;
  }
  if (NS > 1) ptx::cluster_sync();                    // nobody leaves while a peer may still read its words
}

// g[i] = (1/L) * sum over layers (in layer order) of scores[l, i]   (Appendix B, global repair target sweep)
__global__ void mean_scores_kernel(int n_layers, long long sum_t, const float* __restrict__ scores, float* __restrict__ g) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= sum_t) return;
  float a = 0.f;
  for (int l = 0; l < n_layers; ++l) a += scores[(long long)l * sum_t + i];
  g[i] = a / (float)n_layers;
}

// scores[i] *= factor   (combining the per-shard mean scores of a head-sharded layout: mean over shards)
__global__ void scale_scores_kernel(long long n, float factor, float* __restrict__ scores) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) scores[i] *= factor;
}

// Blocks per segment, by the longest segment of the call and by what the GPU holds at once: a block of 1024 threads has an SM
// to itself, 32 clusters of four run together (36 take two waves: 11 -> 21 us at 16 K keys) and eight or nine of eight do (ten
// take two: 17 -> 22 us at 64 K).  Measured in us, by slices:
//   segments x keys     1      2      4      8        segments x keys     1      2      4      8
//    1 x  6 K          7.4    8.2    8.8   11.6        12 x 32 K         25.1   15.6   12.6   22.7
//    1 x  8 K          8.1    8.6    9.3   11.8        28 x 32 K         25.0   15.6   13.2   26.8
//    1 x 12 K         10.4   10.1   10.0   12.1        40 x 32 K           -    15.7   25.4   40.4
//    1 x 16 K         12.6   10.7   10.1   12.6         1 x 48 K         40.9   19.8   14.7   15.0
//    8 x 16 K         12.8   11.0   10.3   14.1         1 x 64 K         65.1   39.3   17.1   15.6
//    1 x 32 K         24.7   15.4   12.3   13.5        64 x 64 K         78.5   40.4   35.8   58.5
// (scores spread over many bins).  Equal leading bits make the histogram's additions queue up, the longer the more keys a block has: scores of 16 query
// rows over 6719 keys took 4.6 us more in one block than in two.  So slices of at most 4 K keys, up to eight, but fewer where they would not
// all run at once; and more again, two waves of them, rather than slices too long for shared memory.
static int select_slices(const ReqTable& rt, long long n_seg, int sms) {
  int t_max = 1, s = 1;
  for (int b = 0; b < rt.n_req; ++b) t_max = std::max(t_max, rt.ctx_len[b]);
  const int want = t_max <= 4096 ? 1 : (t_max <= 8192 ? 2 : (t_max <= 16384 ? 4 : 8));
  auto together = [&](int n) { return n == 8 ? n_seg * 16 <= sms : n_seg * n * 8 <= 7ll * sms; };
  while (s < want && together(2 * s)) s *= 2;
  while (s < 8 && t_max > kSelKeysMax * s && n_seg * (2 * s) <= 2ll * sms) s *= 2;
  return s;
}

template <int NS>
static relaxkv_status launch_select_slices(const ReqTable& rt, int n_layers, const float* raw, float* norm, int* anchors,
                                           DeviceStatus* st, int dev, cudaStream_t stream) {
  static std::atomic<int> attr_done[kMaxDevices];
  if (!attr_done[dev].load(std::memory_order_acquire)) {
    if (cudaFuncSetAttribute(select_topk_kernel<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelKeysMax * 4) != cudaSuccess)
      return RELAXKV_ERR_CUDA;
    attr_done[dev].store(1, std::memory_order_release);
  }
  int cap = 0;                                              // the longest slice that is kept in shared memory
  for (int b = 0; b < rt.n_req; ++b) {
    const int per = ((rt.ctx_len[b] + NS - 1) / NS + 31) & ~31;
    if (per <= kSelKeysMax) cap = std::max(cap, per);
  }
  return cuda_ok(launch_chained_clusters(NS, select_topk_kernel<NS>, dim3((unsigned)(n_layers * rt.n_req * NS)),
                                         dim3(kSelThreads), (size_t)cap * 4, stream, rt, n_layers, cap, raw, norm, anchors, st));
}

relaxkv_status launch_select(const ReqTable& rt, int n_layers, const float* raw, float* norm, int* anchors,
                             cudaStream_t stream) {
  DeviceStatus* st = status_word();
  const int sms = sm_count_of_current_device();
  int dev = 0;
  if (!st || sms <= 0 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return RELAXKV_ERR_CUDA;
  switch (select_slices(rt, (long long)n_layers * rt.n_req, sms)) {
    case 1: return launch_select_slices<1>(rt, n_layers, raw, norm, anchors, st, dev, stream);
    case 2: return launch_select_slices<2>(rt, n_layers, raw, norm, anchors, st, dev, stream);
    case 4: return launch_select_slices<4>(rt, n_layers, raw, norm, anchors, st, dev, stream);
    default: return launch_select_slices<8>(rt, n_layers, raw, norm, anchors, st, dev, stream);
  }
}

}  // namespace relaxkv

using namespace relaxkv;

extern "C" relaxkv_status relaxkv_select_topk(const relaxkv_shape* shape, int32_t n_layers, const int32_t* h_k,
                                              const float* raw_scores, float* norm_scores_out, int32_t* anchors_out,
                                              relaxkv_stream stream) {
  RELAXKV_RANGE("relaxkv_select_topk");
  relaxkv_status rc = check_shape(shape);
  if (rc != RELAXKV_OK) return rc;
  if (n_layers < 1 || !h_k || !raw_scores || !anchors_out) return RELAXKV_ERR_INVALID_ARG;
  for (int b = 0; b < shape->n_req; ++b)
    if (h_k[b] < 1 || h_k[b] > shape->h_ctx_len[b]) return RELAXKV_ERR_INVALID_ARG;
  ReqTable rt;
  fill_req_table(rt, shape, nullptr, h_k);
  return launch_select(rt, n_layers, raw_scores, norm_scores_out, anchors_out, static_cast<cudaStream_t>(stream));
}

extern "C" relaxkv_status relaxkv_mean_scores(const relaxkv_shape* shape, int32_t n_layers, const float* scores,
                                              float* mean_out, relaxkv_stream stream) {
  RELAXKV_RANGE("relaxkv_mean_scores");
  relaxkv_status rc = check_shape(shape);
  if (rc != RELAXKV_OK) return rc;
  if (n_layers < 1 || !scores || !mean_out) return RELAXKV_ERR_INVALID_ARG;
  long long sum_t = 0;
  for (int b = 0; b < shape->n_req; ++b) sum_t += shape->h_ctx_len[b];
  mean_scores_kernel<<<(unsigned)((sum_t + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(n_layers, sum_t, scores, mean_out);
  return launch_ok();
}

extern "C" relaxkv_status relaxkv_scale_scores(const relaxkv_shape* shape, int32_t n_layers, float* scores, float factor,
                                               relaxkv_stream stream) {
  RELAXKV_RANGE("relaxkv_scale_scores");
  relaxkv_status rc = check_shape(shape);
  if (rc != RELAXKV_OK) return rc;
  if (n_layers < 1 || !scores || !(factor > 0.f)) return RELAXKV_ERR_INVALID_ARG;
  long long n = 0;
  for (int b = 0; b < shape->n_req; ++b) n += shape->h_ctx_len[b];
  n *= n_layers;
  scale_scores_kernel<<<(unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(n, factor, scores);
  return launch_ok();
}
