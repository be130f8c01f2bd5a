// y = x W^T (+ residual) for at most 128 rows of x: the query's own tokens going through the block (Section 2 of the
// paper: the query pass that yields the scores, and the query prefill that closes the time-to-first-token region) and the
// decoded tokens of a batch.  The work is streaming the weight matrix once, so the weights are the M side of the MMA:
// a tile is 128 weight rows (TMEM lanes = output features) against all rows of x (N = 16 ... 128 columns, the row count
// rounded up to 16), and a thread block holds half an SM's shared memory as a TMA ring of 64-wide K blocks (a
// whole SM's above 64 rows, where x takes as much of a stage as the weights, and from 33 rows on for few tiles).  128 to 192 KB of weights per SM are in
// flight, and x rows that do not exist are neither multiplied nor, past the 16
// granularity, staged.  A thread-block CLUSTER of S blocks shares a tile and splits K: block r multiplies K blocks
// [r n_k / S, (r + 1) n_k / S) into its own TMEM accumulator, writes the partial tile into its own shared memory and
// pushes to every other block, in one bulk copy each, the features that one owns (128 / S); every block then sums the S
// partials of its own features in rank order, adds the residual and writes bf16.  A fixed order: results
// do not depend on timing.  No scratch in global memory.  Up to four rows (a decoded batch) K is always summed in eight parts, each
// in TMEM columns of its own where a block has several: the bits then depend on K alone, not on how many blocks share a tile, so a
// projection gives the same bits stacked with others and by itself.
// Up to three output segments (feature ranges going to different buffers) serve the fused Q/K/V projection; the fused
// gate/up projection takes 64 gate rows and their 64 up rows as one tile and applies the activation in the epilogue.
// Bound by HBM (N K 2 bytes); with 128 rows of x as the M side, one block per SM and plain launches, four rows of a decode
// step went through the FMA pipe (gate/up 34816 x 5120 77 us, 5120 x 17408 40 us, 6144 x 4096 13.6 us; now 55, 32 and 12.3:
// 6.5, 5.6 and 4.1 TB/s), 57 rows took 65 / 36 / 16.2 us (now 56 / 32.5 / 12.3) and 128 rows 65 / 37.7 / 17.2 us (60.5 / 35.9 /
// 15.5, and 2 to 3 us less behind a short kernel, where the start is hidden).  What is left above the bytes is about 4 us of a launch: the first
// products 3 us behind the wait, the exchange of the partial tiles and the hand-over to the next kernel behind the last.
// Launched chained: barriers, tensor memory and an L2 prefetch of the ring's first weight tiles come before the wait for
// the kernels in front (a prefetch only: the weights are read after the wait, whoever wrote them).
// The cluster barriers have no time limit, so every thread executes all of them whatever its (bounded) waits on the
// mbarriers have returned, and no block leaves before its peers have read its partial tile.
#include "common.cuh"
#include "gemm_skinny.cuh"
#include "gemv.cuh"
#include "sm100_ptx.cuh"
#include <algorithm>
#include <atomic>

namespace relaxkv {

using namespace ptx;

bool make_map_3d(CUtensorMap* m, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint64_t stride1_bytes,
                 uint64_t stride2_bytes, uint32_t b1, uint32_t b2);          // attention_sm100.cu

__host__ __device__ constexpr int sk_threads(int epi) { return 64 + 32 * epi; }
constexpr int kSkManyRows = 32;                                            // whole tiles: rows from which eight warps write them
constexpr int kSkDeepK = 8192;                                             // few rows: K from which eight blocks share a tile
constexpr int kSkParts = 8, kSkPartCols = 16;                               // few rows: parts of K, MMA columns of each
constexpr int kSkBars = 2 * kSkStagesMax + 2;                              // full, empty per stage; accumulator full; partial tiles received
constexpr int kSkTail = 8 * kSkBars + 16 + 1024;                           // barriers, slots, alignment
static_assert(sk_exchange_fits(1, 1, kSkinnyMaxRows, false, kSkinnyMaxRows, sk_stages(kSkinnyMaxRows, false)), "a tile of its own reuses the TMA ring");

// S blocks per tile; a block's share of K is PL parts, each summed in an accumulator of its own (PL > 1: n_cols is kSkPartCols).
template <int S, int PL, int E>
__global__ void __launch_bounds__(64 + 32 * E, 2)
gemm_skinny_sm100_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x,
                         int M, int n_cols, int n_stages, int n_feat, int K, int swiglu, const __grid_constant__ SkinnyOut outs,
                         DeviceStatus* st) {
  const uint32_t rank = (S > 1) ? cluster_ctarank() : 0u;
  const int tile = (int)(blockIdx.x / S);
  const int n_k = (K + kSkBK - 1) / kSkBK;
  auto part_begin = [&](int j) { return (int)((long long)j * n_k / (S * PL)); };       // first K block of part j (of all ranks)
  const int k0 = part_begin((int)rank * PL), k1 = part_begin(((int)rank + 1) * PL);
  // the weight rows of this tile: two boxes of 64
  const int f0 = swiglu ? tile * (kSkFeat / 2) : tile * kSkFeat;            // first output feature
  const int r0 = swiglu ? (f0 / 128) * 256 + f0 % 128 : f0, r1 = swiglu ? r0 + 128 : r0 + kSkFeat / 2;

  // of the tile's features, in groups of four, block r of the cluster adds up and writes [r all / S, (r + 1) all / S)
  const int all_quads = sk_quads(swiglu != 0);
  const int own_q0 = sk_quad((int)rank, S, swiglu != 0), own_quads = sk_quad((int)rank + 1, S, swiglu != 0) - own_q0;

  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t stage_bytes = (uint32_t)(kSkWBytes + n_cols * kSkBK * 2), ring = stage_bytes * (uint32_t)n_stages;
  const uint32_t bar0 = base + ring;
  const uint32_t bar_full = bar0, bar_empty = bar0 + 8 * kSkStagesMax, bar_acc = bar0 + 16 * kSkStagesMax, bar_recv = bar_acc + 8;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + ring + 8 * kSkBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(const_cast<uint32_t*>(tmem_slot) + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tmem_cols = n_cols * PL <= 32 ? 32u : (n_cols * PL <= 64 ? 64u : 128u);

  if (threadIdx.x == 0) {
    for (int s = 0; s < n_stages; ++s) { mbar_init(bar_full + 8 * s, 1); mbar_init(bar_empty + 8 * s, 1); }
    mbar_init(bar_acc, 1);
    mbar_init(bar_recv, 1);
    *abort_flag = 0;
    fence_barrier_init();
    if (S > 1) mbar_expect_tx(bar_recv, (uint32_t)((S - 1) * PL * M * (swiglu ? 2 : 1) * own_quads * 16));
    fence_proxy_async_smem();
  }
  if (warp == 4 && lane == 0) {
    prefetch_tensormap(&tm_w); prefetch_tensormap(&tm_x);
    for (int kt = k0; kt < min(k1, k0 + n_stages); ++kt) {
      tma_prefetch_3d(&tm_w, kt * kSkBK, r0, 0);
      if (swiglu || r1 < n_feat) tma_prefetch_3d(&tm_w, kt * kSkBK, r1, 0);
    }
  }
  if (warp == 5) { tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), tmem_cols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // Only now that this block has its tensor memory may the next kernel's blocks come (they allocate some themselves).
  // All blocks of a one-wave launch are resident by then, so the next kernel only takes room that is left over.
  griddep_launch();
  griddep_wait();
  // After an expired wait elsewhere the tensor-core kernels write nothing until the status word has been read.  The word is
  // fetched here and looked at before the outputs are written: waiting for it first would cost a memory latency, and
  // everything up to there stays inside the block and its cluster.
  const int status = *reinterpret_cast<volatile int*>(&st->status);
  bool ok = true;
  if (warp == 4) {
    // ---- TMA producer ----
    if (lane == 0) {
      for (int kt = k0, it = 0, s = 0, ph = 0; kt < k1; ++kt, ++it) {
        if (it >= n_stages && !mbar_wait(bar_empty + 8 * s, (uint32_t)(ph ^ 1), abort_flag)) break;
        const uint32_t dst = base + (uint32_t)s * stage_bytes;
        mbar_expect_tx(bar_full + 8 * s, stage_bytes);
        tma_load_3d(dst, &tm_w, bar_full + 8 * s, kt * kSkBK, r0, 0);
        tma_load_3d(dst + kSkWBytes / 2, &tm_w, bar_full + 8 * s, kt * kSkBK, r1, 0);
        tma_load_3d(dst + kSkWBytes, &tm_x, bar_full + 8 * s, kt * kSkBK, 0, 0);
        if (++s == n_stages) { s = 0; ph ^= 1; }
      }
    }
  } else if (warp == 5) {
    // ---- MMA issuer ----
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16_f32(kSkFeat, n_cols, 0);
      bool go = true;
      int s = 0, ph = 0;
      for (int i = 0; go && i < PL; ++i) {
        const int kb = part_begin((int)rank * PL + i), ke = part_begin((int)rank * PL + i + 1);
        for (int kt = kb; kt < ke; ++kt) {
          if (!(go = mbar_wait(bar_full + 8 * s, (uint32_t)ph, abort_flag))) break;
          tc_fence_after();
          const uint32_t sw = base + (uint32_t)s * stage_bytes;
          mma_ss_4steps(tmem_base + (uint32_t)(i * n_cols), desc_lo(sw, 16), desc_lo(sw + kSkWBytes, 16), desc_hi_sw128(1024), idesc,
                        kt > kb ? 1u : 0u);
          mma_commit(bar_empty + 8 * s);
          if (++s == n_stages) { s = 0; ph ^= 1; }
        }
      }
      if (go) mma_commit(bar_acc);
    }
  } else {
    // ---- epilogue warps (thread = weight row = TMEM lane): this block's partial tile -> its own shared memory, the features of each
    // block of the cluster behind one another: [block][gate, up][row of x][feature] fp32.  The MMAs have completed by then, so the TMA
    // ring is free to hold it, here (said to the cluster by the arrival below) and behind it what the other blocks send. ----
    // (What does not depend on the products comes before the wait for them: the divisions and the residual's first rows.)
    const int halves = swiglu ? 2 : 1;
    const int tl = (warp & 3) * 32 + lane, up = swiglu ? tl / (kSkFeat / 2) : 0, f_st = tl - up * (kSkFeat / 2);
    const int r_st = S > 1 ? (((f_st >> 2) + 1) * S - 1) / all_quads : 0, q_st = r_st * all_quads / S;
    const int w_st = ((r_st + 1) * all_quads / S - q_st) * 4;    // features of the block that this thread's feature goes to
    float* stage = reinterpret_cast<float*>(base_ptr) + PL * M * (halves * 4 * q_st + up * w_st) + f_st - 4 * q_st;
    // this block's run of the tile's features, four features of one row of x per thread and round
    const int et = warp < 4 ? (int)threadIdx.x : (int)threadIdx.x - 64;
    const int rows = 32 * E / own_quads, m0 = et / own_quads, q = et % own_quads;               // rows of x per round
    const int col0 = f0 + (own_q0 + q) * 4;
    // which output buffer these features go to (segment boundaries are multiples of 8)
    int sg = 0;
    while (sg + 1 < outs.n && col0 >= outs.col0[sg + 1]) ++sg;
    const int width = outs.col0[sg + 1] - outs.col0[sg];
    uint16_t* y = outs.y[sg] + (col0 - outs.col0[sg]);
    const uint16_t* res = outs.residual[sg] ? outs.residual[sg] + (col0 - outs.col0[sg]) : nullptr;
    const bool mine = m0 < rows && col0 < n_feat && status != RELAXKV_ERR_TIMEOUT;
    constexpr int R = PL > 1 ? 1 : 4;                            // rounds whose loads are in flight together (up to four rows: one in all)
    uint2 r[R];
    auto load_residual = [&](int mb) {
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const int m = mb + j * rows;
        r[j] = (res != nullptr && mine && m < M) ? *reinterpret_cast<const uint2*>(res + (long long)m * width) : make_uint2(0u, 0u);
      }
    };
    load_residual(m0);

    ok = mbar_wait(bar_acc, 0, abort_flag);
    ok = __all_sync(0xffffffffu, ok);
    if (S > 1) cluster_arrive();
    tc_fence_after();
    if (ok) {
      const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
      for (int c = warp < 4 ? 0 : 32; c < (PL > 1 ? PL * kSkPartCols : M); c += 8 * E) {
        uint32_t v[32];
        tmem_ld32(t_lane + c, v);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; ++i) {                           // staged: the rows of x of one part behind the other
          const int m = PL > 1 ? i % kSkPartCols : c + i, part = PL > 1 ? c / kSkPartCols + i / kSkPartCols : 0;
          if (m < M) stage[(part * M + m) * w_st] = __uint_as_float(v[i]);
        }
      }
    }
    if (S > 1) {
      fence_proxy_async_smem();
      cluster_wait();                                            // every block's ring is free
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * E) : "memory");    // the partial tile is in place
    const int sent = PL * M * halves * own_quads * 4;            // floats of one block's contribution to this one
    if (S > 1) {
      // One bulk copy to every other block of the cluster.  (Each block reading its share of every peer, and its own, through ld.shared::cluster and
      // two whole cluster barriers took 4 of the 14.3 us of a projection of 57 rows by 5120 x 5120 in six blocks per tile; now 12.9.)
      if ((int)threadIdx.x < S && threadIdx.x != rank && !*abort_flag) {
        const int to = (int)threadIdx.x, q0 = to * all_quads / S, quads = (to + 1) * all_quads / S - q0;
        const uint32_t per = (uint32_t)(PL * M * halves * 16);   // bytes per group of four features
        bulk_push(mapa_shared(base + sk_part_bytes(PL * M) + rank * (per * (uint32_t)quads), (uint32_t)to), base + per * (uint32_t)q0,
                  per * (uint32_t)quads, mapa_shared(bar_recv, (uint32_t)to));
      }
      if (ok) ok = mbar_wait_cluster(bar_recv, 0, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      cluster_arrive();                                          // nothing is on its way to this block any more
    }
    const float* recv = reinterpret_cast<const float*>(base_ptr + sk_part_bytes(PL * M)) + q * 4;
    const float* own = reinterpret_cast<const float*>(base_ptr) + PL * M * halves * 4 * own_q0 + q * 4;
    auto sum4 = [&](int m, int half) {
      float4 v[S * PL];
#pragma unroll
      for (int src = 0; src < S * PL; ++src)
        v[src] = *reinterpret_cast<const float4*>((src / PL == (int)rank ? own : recv + src / PL * sent) + (half * PL * M + src % PL * M + m) * own_quads * 4);
      float4 f = v[0];
#pragma unroll
      for (int src = 1; src < S * PL; ++src) {                   // order of K: the same sum whatever the timing
        f.x += v[src].x; f.y += v[src].y; f.z += v[src].z; f.w += v[src].w;
      }
      return f;
    };
    if (ok && mine) {
      for (int mb = m0; mb < M; mb += R * rows) {
        float4 f[R], u[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int m = min(mb + j * rows, M - 1);
          f[j] = sum4(m, 0);
          if (swiglu) u[j] = sum4(m, 1);
        }
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int m = mb + j * rows;
          if (m >= M) break;
          float4 v = f[j];
          if (swiglu) {                                          // one rounding, after the activation
            v.x = v.x / (1.f + __expf(-v.x)) * u[j].x; v.y = v.y / (1.f + __expf(-v.y)) * u[j].y;
            v.z = v.z / (1.f + __expf(-v.z)) * u[j].z; v.w = v.w / (1.f + __expf(-v.w)) * u[j].w;
          }
          if (res != nullptr) {
            v.x += __uint_as_float(r[j].x << 16); v.y += __uint_as_float(r[j].x & 0xffff0000u);
            v.z += __uint_as_float(r[j].y << 16); v.w += __uint_as_float(r[j].y & 0xffff0000u);
          }
          __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
          *reinterpret_cast<uint2*>(y + (long long)m * width) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
        }
        if (mb + R * rows < M) load_residual(mb + R * rows);
      }
    }
  }
  if (S > 1) {
    __syncwarp();
    if (warp == 4 || warp == 5) { cluster_arrive(); cluster_wait(); cluster_arrive(); }
    cluster_wait();                             // nobody leaves while its partial tile is on its way to a peer
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) report(st, RELAXKV_ERR_TIMEOUT, KID_GEMM_SM100, (int)blockIdx.x, 1);
    const uint64_t tw = global_timer_ns();
    while (global_timer_ns() - tw < 200000ull) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == 5) { tc_fence_after(); tmem_dealloc(tmem_base, tmem_cols); }
}

struct SkinnyPlan {
  int n_rows, n_cols, n_stages, n_feat, n_in, swiglu, tiles, dev, sms;
  bool whole_sm;                                                            // one block per SM, twice the stages
  size_t smem;
  DeviceStatus* st;
  cudaStream_t stream;
};

template <int S, int PL, int E>
static bool opt_in_smem(int dev) {
  static std::atomic<int> attr_done[kMaxDevices];
  if (!attr_done[dev].load(std::memory_order_acquire)) {
    if (cudaFuncSetAttribute(gemm_skinny_sm100_kernel<S, PL, E>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSkRing1 + kSkTail) != cudaSuccess)
      return false;
    attr_done[dev].store(1, std::memory_order_release);
  }
  return true;
}

// Clusters of S blocks, one block per SM, that can be resident at once (per device, looked up once: a GPC's SMs are not a
// multiple of every S).  0: error.
template <int S>
static int max_clusters(int dev, int sms) {
  static std::atomic<int> cached[kMaxDevices];
  int n = S == 1 ? sms : cached[dev].load(std::memory_order_acquire);
  if (n == 0) {
    if (!opt_in_smem<S, 1, 4>(dev)) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(sms / S * S));
    cfg.blockDim = dim3(sk_threads(4));
    cfg.dynamicSmemBytes = kSkRing1 + kSkTail;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)S; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_skinny_sm100_kernel<S, 1, 4>, &cfg) != cudaSuccess || n < 1) n = std::max(1, sms / S / 2);
    cached[dev].store(n, std::memory_order_release);
  }
  return n;
}

// Launches with clusters of S blocks if that is one wave of resident blocks that have two K blocks each (or S is 1).
template <int S, int PL = 1, int E = 4>
static bool try_launch(const SkinnyPlan& p, const CUtensorMap& tm_w, const CUtensorMap& tm_x, const SkinnyOut& outs, relaxkv_status* rc) {
  const int n_k = (p.n_in + kSkBK - 1) / kSkBK;
  if (S > 1 && n_k < 2 * S) return false;
  if (S > 1 && !sk_exchange_fits(S, PL, p.n_rows, p.swiglu != 0, p.n_cols, p.n_stages)) return false;
  // with two blocks per SM an even cluster sits on S / 2 SMs (the occupancy query itself counts one block per SM)
  const int resident = p.whole_sm ? max_clusters<S>(p.dev, p.sms) : (S % 2 ? 2 * max_clusters<S>(p.dev, p.sms) : max_clusters<(S + 1) / 2>(p.dev, p.sms));
  if (resident < 1 || !opt_in_smem<S, PL, E>(p.dev)) { *rc = RELAXKV_ERR_CUDA; return true; }
  if (S > 1 && p.tiles > resident) return false;
  *rc = cuda_ok(launch_chained_clusters(S, gemm_skinny_sm100_kernel<S, PL, E>, dim3((unsigned)(p.tiles * S)), dim3(sk_threads(E)), p.smem,
                                        p.stream, tm_w, tm_x, p.n_rows, p.n_cols, p.n_stages, p.n_feat, p.n_in, p.swiglu, outs, p.st));
  return true;
}

relaxkv_status launch_gemm_skinny(const void* x, const void* weight, const SkinnyOut& outs, int n_rows, int n_out, int n_in,
                                  int swiglu, cudaStream_t stream) {
  RELAXKV_RANGE("gemm_skinny_sm100_kernel");
  SkinnyPlan p = {};
  p.n_rows = n_rows; p.n_in = n_in; p.swiglu = swiglu; p.stream = stream;
  p.n_cols = (n_rows + 15) & ~15;                                            // N of the MMA
  p.n_feat = swiglu ? n_out / 2 : n_out;
  p.tiles = (n_out + kSkFeat - 1) / kSkFeat;                                 // also of the fused gate/up projection
  CUtensorMap tm_w, tm_x;
  if (!make_map_3d(&tm_w, weight, (uint64_t)n_in, (uint64_t)n_out, 1, (uint64_t)n_in * 2, (uint64_t)n_in * 2 * (uint64_t)n_out, kSkFeat / 2, 1) ||
      !make_map_3d(&tm_x, x, (uint64_t)n_in, (uint64_t)n_rows, 1, (uint64_t)n_in * 2, (uint64_t)n_in * 2 * (uint64_t)n_rows, (uint32_t)p.n_cols, 1))
    return RELAXKV_ERR_CUDA;
  p.st = status_word();
  if (!p.st || cudaGetDevice(&p.dev) != cudaSuccess || p.dev < 0 || p.dev >= kMaxDevices) return RELAXKV_ERR_CUDA;
  p.sms = sm_count_of_current_device();
  if (p.sms <= 0) return RELAXKV_ERR_CUDA;
  // Above 64 rows two blocks of an SM would have three stages each; with no more tiles than SMs one block with six is
  // faster (128 rows, 5120 x 17408: 38 against 43 us), with more tiles two (34816 x 5120: 63 against 73 us).  From 33 rows on
  // clusters of at least four blocks also want an SM per block, which all of them get where the tiles are a quarter of the SMs
  // (64 rows, two blocks / one: 2048 x 2048 8.4 / 6.9 us, 3072 x 2048 9.8 / 7.6, 4096 x 4096 12.9 / 10.7, 4096 x 14336 25.9 / 24.1; 33 rows 6.8 / 6.2,
  // 7.8 / 7.1, 11.0 / 10.2, 24.0 / 23.5; 40 tiles of 5120 x 5120 14.4 / 13.8 and 13.2 / 13.1; 17 rows, 2048 x 4096 7.4 / 7.8).
  p.whole_sm = (p.n_cols > kSkCols2 && p.tiles <= p.sms) || (p.n_cols > 32 && p.tiles * 4 <= p.sms);
  p.n_stages = sk_stages(p.n_cols, p.whole_sm);
  p.smem = (size_t)p.n_stages * sk_stage_bytes(p.n_cols) + kSkTail;
  relaxkv_status rc = RELAXKV_OK;
  // The largest cluster that fits.  A projection of up to four rows is always summed over K in kSkParts parts, however many blocks
  // share them, so that it has the same bits stacked with others and by itself.
  // Eight blocks where K is long, or where each gets an SM: else they fill the SMs that the next kernel's blocks would start on.
  if (n_rows <= kGemvMaxRows && !swiglu && (n_in + kSkBK - 1) / kSkBK >= kSkParts) {
    const bool eight = n_in >= kSkDeepK || p.tiles * 8 <= p.sms;
    if ((eight && try_launch<8, 1>(p, tm_w, tm_x, outs, &rc)) || try_launch<4, 2>(p, tm_w, tm_x, outs, &rc) || try_launch<2, 4>(p, tm_w, tm_x, outs, &rc))
      return rc;
    try_launch<1, 8>(p, tm_w, tm_x, outs, &rc);
    return rc;
  }
  if (try_launch<8>(p, tm_w, tm_x, outs, &rc) || try_launch<7>(p, tm_w, tm_x, outs, &rc) || try_launch<6>(p, tm_w, tm_x, outs, &rc) ||
      try_launch<5>(p, tm_w, tm_x, outs, &rc) || try_launch<4>(p, tm_w, tm_x, outs, &rc) || try_launch<3>(p, tm_w, tm_x, outs, &rc) ||
      try_launch<2>(p, tm_w, tm_x, outs, &rc))
    return rc;
  // A block with a tile of its own adds nothing up but writes every feature of it: eight warps for many rows (28672 x 4096 gate/up: 57 rows
  // 42.7 us with four, 41.9, 128 rows 47.4 / 45.7).  In a cluster four are enough, and more cost their start (5120 x 5120: 57 rows 13.0 / 13.8).
  if (p.n_rows > kSkManyRows) try_launch<1, 1, 8>(p, tm_w, tm_x, outs, &rc);
  else try_launch<1>(p, tm_w, tm_x, outs, &rc);
  return rc;
}

}  // namespace relaxkv
