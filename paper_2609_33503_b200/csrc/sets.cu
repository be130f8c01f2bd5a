// Repair schedule: highest selected layer h_i, sorted union U, position->rank map and the per-layer
// active targets R_l as ranks into U (Section 3.2; Algorithm 1, steps 6-12).  Integer work only.
#include "common.cuh"
#include "sm100_ptx.cuh"
#include <algorithm>
#include <atomic>

namespace relaxkv {

// The four kernels of a schedule take a few microseconds each and depend on one another: they are launched chained, so
// that each one's launch and ramp-up run under its predecessor.  Everything a predecessor writes is read through plain
// pointers after griddep_wait().
constexpr int kSetThreads = 1024;
constexpr int kSetWarps = kSetThreads / 32;
constexpr int kSetSlices = 8;                    // blocks of a cluster that writes one list, at most

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

// Cluster (b, 0) writes u_pos / u_rank, cluster (b, l+1) the ranks of R_{l,b}; each of its NS blocks takes a contiguous slice of the
// positions (set_slices).  Where a list starts is the sum of the counts before it, which every block adds up for itself (u_cu and r_cu
// are those sums).  One block per list took 20 / 77 / 149 us for segments of 16 K / 32 K / 64 K positions (a thread walked
// 64 consecutive positions, one dependent uncoalesced load and store after the other), and a launch of its own for the
// prefix of the counts another 4 us; the whole schedule of 40 layers now takes 12 / 14 / 21 us.
template <int NS>                                 // slices = blocks of a cluster
__global__ void __launch_bounds__(kSetThreads) write_sets_kernel(ReqTable rt, int n_layers, const int* h, const int* counts,
                                                                 int* u_pos, int* u_cu, int* u_rank, int* r_rank, int* r_cu,
                                                                 int* host_counts) {
  __shared__ int s_u[kSetWarps], s_r[kSetWarps], s_base[kSetWarps];
  __shared__ int s_pub[2];                                    // this slice's totals, read by the cluster
  const int B = rt.n_req;
  const int slice = (int)blockIdx.x % NS, list = (int)blockIdx.x / NS;
  const int b = list % B, s = list / B;
  const int T = rt.ctx_len[b];
  const int* hb = h + rt.ctx_cu[b];
  const int thr = (s == 0) ? 0 : (s - 1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = ((T + NS - 1) / NS + 31) & ~31;
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
  if (NS > 1) {
    if (warp == 0) {
      const int tu = warp_reduce_sum(wu), tr = warp_reduce_sum(wr);
      if (lane == 0) { s_pub[0] = tu; s_pub[1] = tr; }
    }
    ptx::cluster_sync();
    int gu = 0, gr = 0;                                       // lane r fetches the totals of slice r
    if (lane < slice) {
      gu = ptx::ld_cluster_s32(ptx::mapa_shared(ptx::smem_u32(&s_pub[0]), (uint32_t)lane));
      gr = ptx::ld_cluster_s32(ptx::mapa_shared(ptx::smem_u32(&s_pub[1]), (uint32_t)lane));
    }
    eu += warp_reduce_sum(gu); er += warp_reduce_sum(gr);
  }

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
  if (NS > 1) ptx::cluster_sync();                            // nobody leaves while a peer may still read its totals
}

// The whole schedule of ONE request in one launch: a cluster whose blocks each hold a contiguous slice of the positions in
// shared memory.  Every block reads all anchors and keeps the layers of its own positions; the blocks' counts per layer meet
// through distributed shared memory, which gives every list's place; a warp then writes one list of its block's slice, or a run
// of it.  Four dependent launches become one, for work that is mostly their latency: positions of a slice times lists up to
// kOneWorkMax.  Launched call by call the host's time decides (16 us for four launches, 8 for one), replayed from a graph the GPU's.
// Four launches / one, us, call by call and (from a graph): 1 K positions and 1 layer 14.1 / 6.5 (6.1 / 4.2), 32 layers 14.7 / 7.4
// (6.7 / 6.2); 8 K and 1 layer 14.0 / 6.7 (7.9 / 5.1), 5 layers 14.6 / 8.8 (8.6 / 7.3), 6 layers, work 7168, 14.7 / 10.6 (8.2 / 9.1); 16 K and 3
// layers, the line, 14.4 / 11.0 (9.3 / 9.5); past it 16 K and 12 layers 10.6 / 18.0 on the GPU.  The line is drawn for calls (the counts are
// read by the host behind this one); from 6144 to it a replay loses up to 1 us, with a hundred lists and more up to 3.
constexpr int kOneWorkMax = 8192;
constexpr int kOneLayersMax = kOneWorkMax / 32;  // a slice is at least 32 positions

__global__ void __launch_bounds__(kSetThreads) schedule_one_kernel(int T, int k, int n_layers, const int* anchors, int* h, int* u_pos,
                                                                   int* u_cu, int* u_rank, int* r_rank, int* r_cu, int* counts,
                                                                   int* host_counts, DeviceStatus* st) {
  extern __shared__ int s_h[];                                // highest layer of the slice's positions
  __shared__ int s_hist[kOneLayersMax], s_cnt[kOneLayersMax]; // positions whose highest layer is / is at least l; s_cnt is read by the cluster
  __shared__ int s_run_u[kSetWarps], s_run_r[kSetWarps];
  __shared__ int s_tot[kOneLayersMax], s_before[kOneLayersMax], s_base[kOneLayersMax];
  const int slice = (int)blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = ((T + kSetSlices - 1) / kSetSlices + 31) & ~31;
  const int p0 = min(T, slice * per), n = min(T, p0 + per) - p0;
  for (int i = tid; i < n; i += kSetThreads) s_h[i] = -1;
  for (int l = tid; l < n_layers; l += kSetThreads) s_hist[l] = 0;
  griddep_launch();
  griddep_wait();
  __syncthreads();
  const int n_anchors = n_layers * k;
#pragma unroll 8
  for (int idx = tid; idx < n_anchors; idx += kSetThreads) {
    const int pos = anchors[idx];
    if ((unsigned)(pos - p0) < (unsigned)n) atomicMax(&s_h[pos - p0], idx / k);
    else if (slice == 0 && (pos < 0 || pos >= T)) report(st, RELAXKV_ERR_BAD_INDEX, KID_SETS, idx, pos);
  }
  __syncthreads();
  for (int i0 = warp * 32; i0 < n; i0 += kSetThreads) {
    const int v = i0 + lane < n ? s_h[i0 + lane] : -1;
    if (i0 + lane < n) h[p0 + i0 + lane] = v;
    const unsigned same = __match_any_sync(0xffffffffu, v);   // few layers: many lanes count into one word
    if (v >= 0 && lane == __ffs(same) - 1) atomicAdd(&s_hist[v], __popc(same));
  }
  __syncthreads();
  if (tid < n_layers) {
    int c = 0;
    for (int l = tid; l < n_layers; ++l) c += s_hist[l];
    s_cnt[tid] = c;
  }
  ptx::cluster_sync();
  if (tid < n_layers) {
    int tot = 0, before = 0;
#pragma unroll
    for (int r = 0; r < kSetSlices; ++r) {
      const int c = ptx::ld_cluster_s32(ptx::mapa_shared(ptx::smem_u32(&s_cnt[tid]), (uint32_t)r));
      tot += c;
      if (r < slice) before += c;
    }
    s_tot[tid] = tot; s_before[tid] = before;
  }
  __syncthreads();
  if (tid < n_layers) {
    int base = 0;
    for (int l = 0; l < tid; ++l) base += s_tot[l];
    s_base[tid] = base + s_before[tid];
    if (slice == 0) {
      r_cu[tid] = base;
      counts[1 + tid] = s_tot[tid];
      if (host_counts) host_counts[1 + tid] = s_tot[tid];
      if (tid == n_layers - 1) r_cu[n_layers] = base + s_tot[tid];
      if (tid == 0) { u_cu[0] = 0; u_cu[1] = s_tot[0]; counts[0] = s_tot[0]; if (host_counts) host_counts[0] = s_tot[0]; }
    }
  }
  __syncthreads();
  // with few lists several warps share one: a run of the slice each, behind the counts of the runs before it
  int share = 1;
  while (2 * share * (n_layers + 1) <= kSetWarps) share *= 2;
  const int run = ((n + share - 1) / share + 31) & ~31;
  const int i0 = min(n, (warp % share) * run), i1 = min(n, i0 + run);
  int du = 0, dr = 0;
  if (share > 1) {
    const int thr = max(0, warp / share - 1);
    for (int i = i0 + lane; i < i1; i += 32) { const int v = s_h[i]; du += (v >= 0); dr += (v >= thr); }
    du = warp_reduce_sum(du); dr = warp_reduce_sum(dr);
    if (lane == 0) { s_run_u[warp] = du; s_run_r[warp] = dr; }
    __syncthreads();
    du = 0; dr = 0;
    for (int w = warp - warp % share; w < warp; ++w) { du += s_run_u[w]; dr += s_run_r[w]; }
  }
  const uint32_t below = (1u << lane) - 1u;
  for (int list = warp / share; list <= n_layers; list += kSetWarps / share) {      // 0: U, l + 1: R_l
    const int thr = list == 0 ? 0 : list - 1;
    int eu = s_before[0] + du, er = list == 0 ? 0 : s_base[thr] + dr;
#pragma unroll 4
    for (int i = i0 + lane; i - lane < i1; i += 32) {
      const int v = i < i1 ? s_h[i] : -1;
      const uint32_t mu = __ballot_sync(0xffffffffu, v >= 0), mr = __ballot_sync(0xffffffffu, v >= thr);
      const int rank = eu + __popc(mu & below);
      if (list == 0) {
        if (v >= 0) u_pos[rank] = p0 + i;
        if (i < i1) u_rank[p0 + i] = v >= 0 ? rank : -1;
      } else if (v >= thr) {
        r_rank[er + __popc(mr & below)] = rank;
      }
      eu += __popc(mu); er += __popc(mr);
    }
  }
  ptx::cluster_sync();                                        // nobody leaves while a peer may still read its counts
}

}  // namespace relaxkv

using namespace relaxkv;

// Blocks that share one list (1, 2, 4 or 8): the count with the least waves x (wave + slice).  A wave of two blocks of 1024 threads
// per SM takes about 3 us, 4 / 4.5 / 5.5 as clusters of 2 / 4 / 8, and a block about 0.3 us per 1 K positions of its slice.  Long
// lists want many blocks: 9 lists of 200 K positions 86 / 57 / 38 / 30 us with 1 / 2 / 4 / 8, one request of 64 K x 40 layers 31 / 23 / 21 / 24.
// Many lists want one each: 64 requests of 1 K x 40 layers 48 / 101 / 188 / 432 us, 8 of 8 K x 40 17 / 24 / 35 / 63, 8 of 32 K x 40 42 / 46 / 56 / 89
// (the whole schedule; eight blocks for every list took 2.6 M threads for 2624 lists).
static int set_slices(const ReqTable& rt, long long lists, int sms) {
  int t_max = 1, best = 1;
  for (int b = 0; b < rt.n_req; ++b) t_max = std::max(t_max, rt.ctx_len[b]);
  const double wave_us[4] = {3.0, 4.0, 4.5, 5.5};
  double best_cost = 0.0;
  for (int i = 0, ns = 1; ns <= kSetSlices; ++i, ns *= 2) {
    const double cost = (double)((lists * ns + 2 * sms - 1) / (2 * sms)) * (wave_us[i] + 3e-4 * t_max / ns);
    if (ns == 1 || cost < best_cost) { best_cost = cost; best = ns; }
  }
  return best;
}

// The launch sequence both entry points share: `counts` (device int32 [B + n_layers*B]) is the only scratch.
static relaxkv_status build_sets(const relaxkv_shape* shape, int32_t n_layers, const int32_t* h_k, const int32_t* anchors,
                                 int32_t* highest_layer_out, int32_t* u_pos_out, int32_t* u_cu_out, int32_t* u_rank_out,
                                 int32_t* r_rank_out, int32_t* r_cu_out, int32_t* h_counts_pinned, int* counts,
                                 cudaStream_t stream) {
  DeviceStatus* st = status_word();
  const int sms = sm_count_of_current_device();
  if (!st || sms <= 0) return RELAXKV_ERR_CUDA;
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
  const long long n_anchor = (long long)n_layers * rt.k_cu[B];
  const long long slice_len = ((sum_t + kSetSlices - 1) / kSetSlices + 31) & ~31ll;
  if (B == 1 && slice_len * (n_layers + 1) <= kOneWorkMax) {           // one request, little work: everything in one launch
    const relaxkv_status rc1 = cuda_ok(launch_chained_clusters(
        kSetSlices, schedule_one_kernel, dim3(kSetSlices), dim3(kSetThreads), (size_t)slice_len * 4, stream, rt.ctx_len[0], rt.k[0], n_layers,
        anchors, highest_layer_out, u_pos_out, u_cu_out, u_rank_out, r_rank_out, r_cu_out, counts, host_counts, st));
    if (rc1 != RELAXKV_OK || !h_counts_pinned || host_counts) return rc1;
    return cuda_ok(cudaMemcpyAsync(h_counts_pinned, counts, sizeof(int) * (size_t)(1 + n_layers), cudaMemcpyDeviceToHost, stream));
  }
  // Nothing in `counts` has to start at zero: count_sets_kernel overwrites every entry that write_sets_kernel and the
  // copy below read.
  const unsigned lists = (unsigned)(B * (n_layers + 1));
  cudaError_t e = launch_chained(fill_i32_kernel, dim3((unsigned)((sum_t + 255) / 256)), dim3(256), 0, stream,
                                 highest_layer_out, sum_t, -1);
  if (e == cudaSuccess)
    e = launch_chained(highest_layer_kernel, dim3((unsigned)((n_anchor + 255) / 256)), dim3(256), 0, stream, rt, n_layers,
                       anchors, highest_layer_out, st);
  if (e == cudaSuccess)
    e = launch_chained(count_sets_kernel, dim3(lists), dim3(kSetThreads), 0, stream, rt, n_layers, highest_layer_out, counts);
  if (e == cudaSuccess) {
    auto write = [&](auto* kernel, int slices) {
      return launch_chained_clusters(slices, kernel, dim3(lists * (unsigned)slices), dim3(kSetThreads), 0, stream, rt, n_layers,
                                     highest_layer_out, counts, u_pos_out, u_cu_out, u_rank_out, r_rank_out, r_cu_out, host_counts);
    };
    switch (set_slices(rt, lists, sms)) {
      case 1: e = write(write_sets_kernel<1>, 1); break;
      case 2: e = write(write_sets_kernel<2>, 2); break;
      case 4: e = write(write_sets_kernel<4>, 4); break;
      default: e = write(write_sets_kernel<8>, 8);
    }
  }
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
