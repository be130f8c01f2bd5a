// Repair schedule: highest selected layer h_i, sorted union U, position->rank map and the per-layer
// active targets R_l as ranks into U (Section 3.2; Algorithm 1, steps 6-12).  Integer work only.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace relaxkv {

// The four kernels of a schedule take a few microseconds each and depend on one another: they are launched chained, so
// that each one's launch and ramp-up run under its predecessor.  Everything a predecessor writes is read through plain
// pointers after griddep_wait().
constexpr int kSetThreads = 1024;
constexpr int kSetWarps = kSetThreads / 32;
constexpr int kSetSlices = 8;                    // blocks of the cluster that writes one list

__global__ void __launch_bounds__(256) fill_i32_kernel(int* p, long long n, int v) {
  griddep_launch();
  griddep_wait();
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

// h[i] = max layer that selected position i.
__global__ void __launch_bounds__(256) highest_layer_kernel(ReqTable rt, int n_layers, const int* anchors, int* h, DeviceStatus* st) {
  griddep_launch();
  griddep_wait();
  const int sum_k = rt.k_cu[rt.n_req];
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)n_layers * sum_k) return;
  const int l = (int)(idx / sum_k);
  const int j = (int)(idx - (long long)l * sum_k);
  const int b = find_segment(rt.k_cu, rt.n_req, j);
  const int pos = anchors[idx];
  if (pos < 0 || pos >= rt.ctx_len[b]) { report(st, RELAXKV_ERR_BAD_INDEX, KID_SETS, (int)idx, pos); return; }
  atomicMax(&h[rt.ctx_cu[b] + pos], l);
}

// Block (b, s): s == 0 counts |U_b|; s = l+1 counts |R_{l,b}|.  counts[b] and counts[B + l*B + b].
__global__ void __launch_bounds__(kSetThreads) count_sets_kernel(ReqTable rt, int n_layers, const int* h, int* counts) {
  griddep_launch();
  griddep_wait();
  const int B = rt.n_req;
  const int b = blockIdx.x % B, s = blockIdx.x / B;
  const int T = rt.ctx_len[b];
  const int* hb = h + rt.ctx_cu[b];
  const int thr = (s == 0) ? 0 : (s - 1);
  int n = 0;
#pragma unroll 8
  for (int i = threadIdx.x; i < T; i += kSetThreads) n += (hb[i] >= thr) ? 1 : 0;
  __shared__ int red[kSetWarps];
  n = warp_reduce_sum(n);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x < 32) {
    int v = red[threadIdx.x];
    v = warp_reduce_sum(v);
    if (threadIdx.x == 0) counts[s == 0 ? b : B + (s - 1) * B + b] = v;
  }
}

// Cluster (b, 0) writes u_pos / u_rank, cluster (b, l+1) the ranks of R_{l,b}; each block takes a contiguous slice of the
// positions.  Where a list starts is the sum of the counts before it, which every block adds up for itself (u_cu and r_cu
// are those sums).  One block per list took 20 / 77 / 149 us for segments of 16 K / 32 K / 64 K positions (a thread walked
// 64 consecutive positions, one dependent uncoalesced load and store after the other), and a launch of its own for the
// prefix of the counts another 4 us; now 7 / 20 / 24 us including what overlaps the kernels before it.
__global__ void __launch_bounds__(kSetThreads) write_sets_kernel(ReqTable rt, int n_layers, const int* h, const int* counts,
                                                                 int* u_pos, int* u_cu, int* u_rank, int* r_rank, int* r_cu,
                                                                 int* host_counts) {
  __shared__ int s_u[kSetWarps], s_r[kSetWarps], s_base[kSetWarps];
  __shared__ int s_pub[2];                                    // this slice's totals, read by the cluster
  const int B = rt.n_req;
  const int slice = (int)blockIdx.x % kSetSlices, list = (int)blockIdx.x / kSetSlices;
  const int b = list % B, s = list / B;
  const int T = rt.ctx_len[b];
  const int* hb = h + rt.ctx_cu[b];
  const int thr = (s == 0) ? 0 : (s - 1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = ((T + kSetSlices - 1) / kSetSlices + 31) & ~31;
  const int p0 = min(T, slice * per), p1 = min(T, p0 + per);
  const int run = ((p1 - p0 + kSetWarps - 1) / kSetWarps + 31) & ~31;      // a contiguous run of positions per warp
  const int i0 = min(p1, p0 + warp * run), i1 = min(p1, i0 + run);
  griddep_launch();
  griddep_wait();
  int nu = 0, nr = 0;
#pragma unroll 8
  for (int i = i0 + lane; i < i1; i += 32) { const int v = hb[i]; nu += (v >= 0); nr += (v >= thr); }
  // the list's place: counts of the lists before it
  const int* cnt = s == 0 ? counts : counts + B;
  const int idx = s == 0 ? b : (s - 1) * B + b;
  int base = 0;
  for (int i = threadIdx.x; i < idx; i += kSetThreads) base += cnt[i];
  nu = warp_reduce_sum(nu); nr = warp_reduce_sum(nr); base = warp_reduce_sum(base);
  if (lane == 0) { s_u[warp] = nu; s_r[warp] = nr; s_base[warp] = base; }
  __syncthreads();
  const int wu = s_u[lane], wr = s_r[lane];
  base = warp_reduce_sum(s_base[lane]);
  int eu = warp_reduce_sum(lane < warp ? wu : 0), er = warp_reduce_sum(lane < warp ? wr : 0);
  if (warp == 0) {
    const int tu = warp_reduce_sum(wu), tr = warp_reduce_sum(wr);
    if (lane == 0) { s_pub[0] = tu; s_pub[1] = tr; }
  }
  ptx::cluster_sync();
  int gu = 0, gr = 0;                                         // lane r fetches the totals of slice r
  if (lane < slice) {
    gu = ptx::ld_cluster_s32(ptx::mapa_shared(ptx::smem_u32(&s_pub[0]), (uint32_t)lane));
    gr = ptx::ld_cluster_s32(ptx::mapa_shared(ptx::smem_u32(&s_pub[1]), (uint32_t)lane));
  }
  eu += warp_reduce_sum(gu); er += warp_reduce_sum(gr);

  if (slice == 0 && threadIdx.x == 0) {
    const int n = cnt[idx];
    if (s == 0) { u_cu[b] = base; if (b == B - 1) u_cu[B] = base + n; }
    else { r_cu[idx] = base; if (idx == n_layers * B - 1) r_cu[idx + 1] = base + n; }
  }
  if (host_counts != nullptr && blockIdx.x == 0)
    for (int i = threadIdx.x; i < B + n_layers * B; i += kSetThreads) host_counts[i] = counts[i];
  const uint32_t below = (1u << lane) - 1u;
  int* ur = u_rank + rt.ctx_cu[b];
  int* dst = s == 0 ? u_pos + base : r_rank + base;
  for (int i = i0; i < i1; i += 32) {
    const bool in = i + lane < i1;
    const int v = in ? hb[i + lane] : -1;
    const uint32_t mu = __ballot_sync(0xffffffffu, v >= 0), mr = __ballot_sync(0xffffffffu, in && v >= thr);
    const int rank = eu + __popc(mu & below);                 // members of U before this position
    if (s == 0) {
      if (v >= 0) dst[rank] = i + lane;
      if (in) ur[i + lane] = v >= 0 ? rank : -1;
    } else if (in && v >= thr) {
      dst[er + __popc(mr & below)] = rank;
    }
    eu += __popc(mu); er += __popc(mr);
  }
  ptx::cluster_sync();                                        // nobody leaves while a peer may still read its totals
}

}  // namespace relaxkv

using namespace relaxkv;

// The launch sequence both entry points share: `counts` (device int32 [B + n_layers*B]) is the only scratch.
static relaxkv_status build_sets(const relaxkv_shape* shape, int32_t n_layers, const int32_t* h_k, const int32_t* anchors,
                                 int32_t* highest_layer_out, int32_t* u_pos_out, int32_t* u_cu_out, int32_t* u_rank_out,
                                 int32_t* r_rank_out, int32_t* r_cu_out, int32_t* h_counts_pinned, int* counts,
                                 cudaStream_t stream) {
  DeviceStatus* st = status_word();
  if (!st) return RELAXKV_ERR_CUDA;
  ReqTable rt;
  fill_req_table(rt, shape, nullptr, h_k);
  const int B = shape->n_req;
  const long long sum_t = rt.ctx_cu[B];
  // The caller's counts are written by the last kernel where the device can reach them (pinned memory: a copy behind it
  // would cost another 8 us of a schedule's 15), else by a copy.
  int* host_counts = nullptr;
  if (h_counts_pinned) {
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, h_counts_pinned) != cudaSuccess) (void)cudaGetLastError();
    else if (attr.type == cudaMemoryTypeHost) host_counts = static_cast<int*>(attr.devicePointer);
  }
  // Nothing in `counts` has to start at zero: count_sets_kernel overwrites every entry that write_sets_kernel and the
  // copy below read.
  const long long n_anchor = (long long)n_layers * rt.k_cu[B];
  const unsigned lists = (unsigned)(B * (n_layers + 1));
  cudaError_t e = launch_chained(fill_i32_kernel, dim3((unsigned)((sum_t + 255) / 256)), dim3(256), 0, stream,
                                 highest_layer_out, sum_t, -1);
  if (e == cudaSuccess)
    e = launch_chained(highest_layer_kernel, dim3((unsigned)((n_anchor + 255) / 256)), dim3(256), 0, stream, rt, n_layers,
                       anchors, highest_layer_out, st);
  if (e == cudaSuccess)
    e = launch_chained(count_sets_kernel, dim3(lists), dim3(kSetThreads), 0, stream, rt, n_layers, highest_layer_out, counts);
  if (e == cudaSuccess)
    e = launch_chained_clusters(kSetSlices, write_sets_kernel, dim3(lists * kSetSlices), dim3(kSetThreads), 0, stream, rt,
                                n_layers, highest_layer_out, counts, u_pos_out, u_cu_out, u_rank_out, r_rank_out, r_cu_out, host_counts);
  relaxkv_status rc = cuda_ok(e);
  if (rc != RELAXKV_OK) return rc;
  if (h_counts_pinned && !host_counts)
    rc = cuda_ok(cudaMemcpyAsync(h_counts_pinned, counts, sizeof(int) * (size_t)(B + n_layers * B),
                                 cudaMemcpyDeviceToHost, stream));
  return rc;
}

static relaxkv_status check_sets_args(const relaxkv_shape* shape, int32_t n_layers, const int32_t* h_k,
                                      const int32_t* anchors, const int32_t* highest_layer_out, const int32_t* u_pos_out,
                                      const int32_t* u_cu_out, const int32_t* u_rank_out, const int32_t* r_rank_out,
                                      const int32_t* r_cu_out) {
  relaxkv_status rc = check_shape(shape);
  if (rc != RELAXKV_OK) return rc;
  if (n_layers < 1 || n_layers > 65535 || !h_k || !anchors || !highest_layer_out || !u_pos_out || !u_cu_out ||
      !u_rank_out || !r_rank_out || !r_cu_out)
    return RELAXKV_ERR_INVALID_ARG;
  for (int b = 0; b < shape->n_req; ++b)
    if (h_k[b] < 1 || h_k[b] > shape->h_ctx_len[b]) return RELAXKV_ERR_INVALID_ARG;
  return RELAXKV_OK;
}

extern "C" relaxkv_status relaxkv_build_active_sets(
    const relaxkv_shape* shape, int32_t n_layers, const int32_t* h_k, const int32_t* anchors,
    int32_t* highest_layer_out, int32_t* u_pos_out, int32_t* u_cu_out, int32_t* u_rank_out,
    int32_t* r_rank_out, int32_t* r_cu_out, int32_t* h_counts_pinned,
    void* workspace, size_t workspace_bytes, relaxkv_stream stream_) {
  RELAXKV_RANGE("relaxkv_build_active_sets");
  relaxkv_status rc = check_sets_args(shape, n_layers, h_k, anchors, highest_layer_out, u_pos_out, u_cu_out, u_rank_out,
                                      r_rank_out, r_cu_out);
  if (rc != RELAXKV_OK) return rc;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return RELAXKV_ERR_INVALID_ARG;
  const WsLayout ws = ws_layout(shape, n_layers);
  if (workspace_bytes < ws.total) return RELAXKV_ERR_WORKSPACE_TOO_SMALL;
  int* counts = reinterpret_cast<int*>(static_cast<char*>(workspace) + ws.counts);
  return build_sets(shape, n_layers, h_k, anchors, highest_layer_out, u_pos_out, u_cu_out, u_rank_out, r_rank_out, r_cu_out,
                    h_counts_pinned, counts, static_cast<cudaStream_t>(stream_));
}

// ---- variant whose scratch lives in the library image ------------------------------------------
// Some hosts of this library own every byte of device memory themselves and give an extension no
// way to ask for more: an inference-server plug-in that is handed its input and output tensors and
// nothing else, or an embedded runtime whose memory pool is sealed once start-up ends.  Such a
// caller cannot provide the `workspace` that relaxkv_build_active_sets needs.  For them the set
// counts are kept in this fixed array, which every GPU that loads the library holds until exit.
constexpr int kStaticCountsMax = 8192;           // ints: B + n_layers*B must fit
static __device__ __align__(256) int g_static_counts[kStaticCountsMax];

// Device address of g_static_counts on the current device.  In host code the array's name is only a
// handle; the address a kernel can use comes from cudaGetSymbolAddress, once per device, with that
// device current.
static relaxkv_status static_counts_ptr(int** out) {
  static std::atomic<int*> cached[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return RELAXKV_ERR_CUDA;
  int* p = cached[dev].load(std::memory_order_acquire);
  if (!p) {
    if (cudaGetSymbolAddress((void**)&p, g_static_counts) != cudaSuccess || p == nullptr) return RELAXKV_ERR_CUDA;
    cached[dev].store(p, std::memory_order_release);
  }
  *out = p;
  return RELAXKV_OK;
}

extern "C" relaxkv_status relaxkv_build_active_sets_static(
    const relaxkv_shape* shape, int32_t n_layers, const int32_t* h_k, const int32_t* anchors,
    int32_t* highest_layer_out, int32_t* u_pos_out, int32_t* u_cu_out, int32_t* u_rank_out,
    int32_t* r_rank_out, int32_t* r_cu_out, int32_t* h_counts_pinned, relaxkv_stream stream_) {
  RELAXKV_RANGE("relaxkv_build_active_sets_static");
  relaxkv_status rc = check_sets_args(shape, n_layers, h_k, anchors, highest_layer_out, u_pos_out, u_cu_out, u_rank_out,
                                      r_rank_out, r_cu_out);
  if (rc != RELAXKV_OK) return rc;
  const int B = shape->n_req;
  if ((long long)B + (long long)n_layers * B > kStaticCountsMax) return RELAXKV_ERR_UNSUPPORTED_SHAPE;
  int* counts = nullptr;
  if ((rc = static_counts_ptr(&counts)) != RELAXKV_OK) return rc;
  return build_sets(shape, n_layers, h_k, anchors, highest_layer_out, u_pos_out, u_cu_out, u_rank_out, r_rank_out, r_cu_out,
                    h_counts_pinned, counts, static_cast<cudaStream_t>(stream_));
}
