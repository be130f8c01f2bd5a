// Sparse-context repair attention on the Blackwell tensor cores (Section 3.3; Algorithm 1, steps 16-19).
//
// One CTA owns a pair of tiles of 128 query rows = (floor(256/G) consecutive active targets) x (the G query
// heads of one KV head), so every K/V tile it stages is shared by the whole GQA group.  It walks the
// context prefix a tile can see in 128-key tiles of the materialised mixed context:
//   TMA (128B swizzle)  ->  S = Q K^T  (tcgen05.mma, fp32 accumulator in TMEM)
//   softmax warps: tcgen05.ld S, position-based causal mask on the staircase edge, online max/sum with
//                  lazy rescaling, P -> bf16 back into TMEM (over S)
//   O += P V            (tcgen05.mma, A operand = P from TMEM, B = V tile MN-major from shared memory)
// A CTA runs the TWO tiles (A, B) in ping-pong: while the softmax warps of one tile work, the
// tensor pipe runs the other tile's MMAs; both tiles share every K/V tile staged in shared memory.
// Warp roles: warps 0-3 softmax/epilogue of tile A, warps 4-7 of tile B (thread = query row = TMEM
// lane), warp 8 TMA producer, warp 9 MMA issuer and TMEM owner, warp 10 a helper for cache-only calls.  K/V tiles
// move through a 5-slot ring in the order K_0 V_0 K_1 V_1 ... and are signalled in pairs (V_j, K_{j+1}) - what
// step j of the MMA warp consumes.
// When a call has too few query tiles to fill the GPU, grid.y splits every pair's context; the blocks leave
// normalised partial results that combine_splits_kernel merges by their log-sum-exp.  Of a call over lists that
// has pairs enough but none to follow its longest ones, only those are cut (attention_pieces.cuh).  The K/V tensor maps
// cover either the materialised mixed context (the repair calls) or the cache itself (relaxkv_cache_attention).
// Calls over short gathered contexts (at most 128 key tiles, one split) take attention_persist_kernel below: one
// block per SM walks the same list of (tile pair, KV head) items and overlaps each turn-over with its neighbours.
// Every wait is bounded; an expired wait raises the block's abort flag, records RELAXKV_ERR_TIMEOUT in the
// device status word and the block tears down normally.
#include "attention_common.cuh"
#include "attention_pieces.cuh"
#include "decode_attention.cuh"
#include "sm100_ptx.cuh"
#include <algorithm>
#include <atomic>

namespace relaxkv {

using namespace ptx;

constexpr float kLog2eA = 1.4426950408889634f;
constexpr float kLn2A = 0.6931471805599453f;
constexpr float kRescaleThreshold = 8.0f;     // log2 units: rescale O only when the row max grew by more

constexpr int kBM = 128;                      // query rows per tile (TMEM lanes)
constexpr int kBN = 128;                      // keys per context tile
constexpr int kHalfBytes = 128 * 128;         // 128 rows x 64 bf16: one 128B-swizzled half tile
// P of a tile is handed to the MMA warp in two groups: its first 32 * kPLo keys, then the rest.  96 + 32 against 64 + 64 keys, us per call
// of one layer with every entry repaired: 24 K entries, 40 / 8 heads 5350 / 5440, 32 / 8 heads of dim 64 3155 / 3150; 6 K entries, 32 / 8
// heads of dim 64 212 / 214: one value for both head dims.
constexpr int kPLo = 3;
constexpr int kRing = 5;                      // K/V tile buffers, used in the order K0 V0 K1 V1 ...
constexpr int kNoLimit = 0x7fffffff;          // causal limit of a row that nobody reads: no tile is masked for it
constexpr int kL2Tiles = 5;                     // query calls: key tiles of a block requested into L2 before its wait
constexpr int kPersistMaxTiles = 128;          // contexts up to this many key tiles take the persistent form
constexpr int kAttnThreads = 384;             // 2 x 4 softmax warps + a control warpgroup (TMA warp, MMA warp, 2 idle)

template <int D>
struct AttnSmem {
  static constexpr int kHalves = D / 64;
  static constexpr int kTileBytes = kHalves * kHalfBytes;
  static constexpr int kQ = 0;                                  // two query tiles
  static constexpr int kKV = kQ + 2 * kTileBytes;               // ring of kRing K/V tiles
  static constexpr int kBar = kKV + kRing * kTileBytes;         // mbarriers (8 B each)
  static constexpr int kPairBars = 3;                           // (V_j, K_{j+1}) pairs in flight: full and empty barriers
  static constexpr int kNumBars = 1 + 8 + 2 * kPairBars + 2;
  static constexpr int kMisc = kBar + 8 * kNumBars;             // tmem address, abort flag
  static constexpr int kTotal = kMisc + 16;
  static constexpr int kDynamic = kTotal + 1024;                // slack to align the base to 1024 B
};

// P of keys [32 C0, 32 C1) of a row's tile: p = 2^(s * scale - m), row sums, bf16 into TMEM over S.  The scaling and the sums use packed
// fp32 pairs.
template <int C0, int C1>
__device__ __forceinline__ void softmax_keys(uint32_t t_s, const uint32_t* s, float scale_log2, float neg_m, float& zs0, float& zs1,
                                             float& zs2, float& zs3) {
#pragma unroll
  for (int c = C0; c < C1; ++c) {
    uint32_t pk[16];
#pragma unroll
    for (int i = 0; i < 32; i += 8) {
      float x[8], p[8];
#pragma unroll
      for (int e = 0; e < 8; e += 2)
        fma2(x[e], x[e + 1], __uint_as_float(s[c * 32 + i + e]), __uint_as_float(s[c * 32 + i + e + 1]), scale_log2, scale_log2, neg_m, neg_m);
#pragma unroll
      for (int e = 0; e < 8; ++e) p[e] = fast_exp2(x[e]);
      add2(zs0, zs1, p[0], p[1]); add2(zs2, zs3, p[2], p[3]);
      add2(zs0, zs1, p[4], p[5]); add2(zs2, zs3, p[6], p[7]);
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        __nv_bfloat162 h = __floats2bfloat162_rn(p[e], p[e + 1]);
        pk[(i + e) >> 1] = *reinterpret_cast<uint32_t*>(&h);
      }
    }
    tmem_st16(t_s + c * 16, pk);
  }
}

// 16 bf16 values of an output row; as one sector where the output is 32-byte aligned (the call asks for 16).
__device__ __forceinline__ void store_16(uint16_t* p, const uint32_t* w, bool sectors) {
  if (sectors) {
    st_global_32b(p, w);
  } else {
    reinterpret_cast<uint4*>(p)[0] = make_uint4(w[0], w[1], w[2], w[3]);
    reinterpret_cast<uint4*>(p)[1] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// One step of a query row's online softmax (thread = query row = TMEM lane): S_x(j) is read from TMEM, the keys
// past the row's limit (counted from the tile's first key) are masked on the tiles that straddle the staircase,
// the running maximum m and sum z are updated (O_x is rescaled only when the maximum grew by more than the
// threshold), and P is written over S as bf16 in two column groups, each handed to the MMA warp (bar_p_lo,
// bar_p_hi) as soon as it is stored.  m starts at -1e30, so that a row whose first tile is fully masked keeps a finite reference.
// The step is a link of the chain S -> P -> P V -> next S that bounds the kernel.  The maximum comes first.  Exponentials begun with the
// tile before's reference are no faster where both tiles of a pair keep the SM busy (8 K stack 8.12 ms either way, 12 layers of 40 / 8
// heads at 32 K 35.8; ragged query passes of one to 25 rows per tile 1 to 3 % faster), and where maxima grow along the context they have
// to be done again, four warps waiting for the slowest of them (6 K entries, 32 / 8 heads, keys that grow thirtyfold: 397 us against 321
// with the maximum first; of dim 64 333 against 229).
template <int D>
__device__ __forceinline__ void softmax_step(uint32_t t_s, uint32_t t_o, int limit, bool first, float scale_log2,
                                             float& m, float& z, uint32_t bar_p_lo, uint32_t bar_p_hi) {
  uint32_t s[kBN];
#pragma unroll
  for (int c = 0; c < kBN / 32; ++c) tmem_ld32(t_s + c * 32, &s[c * 32]);
  tmem_wait_ld();
  if (limit < kBN - 1) {
#pragma unroll
    for (int i = 0; i < kBN; ++i)
      if (i > limit) s[i] = 0xff800000u;                      // -inf
  }
  float mx8[8];                         // eight independent chains instead of one 128-deep dependency chain
#pragma unroll
  for (int e = 0; e < 8; ++e) mx8[e] = fmaxf(__uint_as_float(s[2 * e]), __uint_as_float(s[2 * e + 1]));
#pragma unroll
  for (int i = 16; i < kBN; i += 2) mx8[(i >> 1) & 7] = fmax3(mx8[(i >> 1) & 7], __uint_as_float(s[i]), __uint_as_float(s[i + 1]));
  const float m_new =
      fmax3(fmax3(mx8[0], mx8[1], mx8[2]), fmax3(mx8[3], mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7])) * scale_log2;
  const float m_old = m;
  const bool need = m_new > m + kRescaleThreshold;
  if (need) m = m_new;
  // S_x(j) is complete, hence so is O_x += P_x V_{j-1}: O_x may be rescaled here (nothing lies in it before the first tile)
  if (__any_sync(0xffffffffu, need) && !first) {
    const float alpha = fast_exp2(m_old - m);
    z *= alpha;
#pragma unroll 1
    for (int c = 0; c < D / 32; ++c) {
      uint32_t o[32];
      tmem_ld32(t_o + c * 32, o);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
      tmem_st32(t_o + c * 32, o);
    }
  }
  float zs0 = 0.f, zs1 = 0.f, zs2 = 0.f, zs3 = 0.f;
  softmax_keys<0, kPLo>(t_s, s, scale_log2, -m, zs0, zs1, zs2, zs3);
  tmem_wait_st();
  tc_fence_before();
  mbar_arrive(bar_p_lo);                  // the first keys are done: hand them to the MMA warp early
  softmax_keys<kPLo, kBN / 32>(t_s, s, scale_log2, -m, zs0, zs1, zs2, zs3);
  z += (zs0 + zs1) + (zs2 + zs3);
  tmem_wait_st();
  tc_fence_before();
  mbar_arrive(bar_p_hi);
}

template <int D>
__global__ void __launch_bounds__(kAttnThreads, 1)
attention_sm100_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                       const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_k_new,
                       const __grid_constant__ CUtensorMap tm_v_new, int all_fresh, const __grid_constant__ ReqTable rt,
                       const __grid_constant__ PieceTable pt, int mode, int allow_empty, int head_inner, int dense_ctx, int H, int Hkv, int pair_targets, float scale_log2,
                       const int* u_pos, const int* u_cu, const int* r_rank, const int* r_cu,
                       long long n_target_rows, uint16_t* __restrict__ out, float* __restrict__ lse_out,
                       float* __restrict__ part_o, float* __restrict__ part_lse, DeviceStatus* st) {
  using L = AttnSmem<D>;
  constexpr int kHalves = L::kHalves;
  constexpr uint32_t kTmemCols = 512;          // S_A | S_B | O_A | O_B, 128 columns each (O uses D of them)

  // ---- which pair of query tiles ------------------------------------------------------------------
  // rt.tile_cu counts tile PAIRS per request (from the host bounds); pairs are walked from the end of
  // the target list (longest context first).  Tile A = the earlier targets, tile B = the later ones.
  const int B = rt.n_req;
  const int G = H / Hkv;
  const int n_pairs_total = rt.tile_cu[B];
  // ---- shared memory -----------------------------------------------------------------------------
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t q_smem = base + L::kQ, kv_smem = base + L::kKV;
  const uint32_t bar0 = base + L::kBar;
  const uint32_t bar_q = bar0;
  const uint32_t bar_sfull = bar0 + 8;          // [2]
  const uint32_t bar_pfull = bar0 + 24;         // [2] first 32 kPLo keys of P ready
  const uint32_t bar_pfull_hi = bar0 + 40;      // [2] the other keys of P ready
  const uint32_t bar_ofinal = bar0 + 56;        // [2]
  const uint32_t bar_full = bar0 + 72;          // [kPairBars] pair p = (V_{p-1}, K_p) has landed
  const uint32_t bar_empty = bar_full + 8 * L::kPairBars;   // [kPairBars] pair p has been consumed by both tiles
  const uint32_t bar_vreq = bar_empty + 8 * L::kPairBars;   // the request's last V tile has landed (MMA warp -> helper warp)
  const uint32_t bar_vfix = bar_vreq + 8;                   // its rows past the request's end are zeroed (helper -> MMA warp)
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + L::kMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + L::kMisc + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // Barriers, tensor memory, zeroed padding: this block's own.  A call without lists, whose every block has work, sets them up while the
  // kernels in front finish; with lists a block may turn out to have none (loose host bounds), so it looks first.
  auto set_up = [&]() {
    if (threadIdx.x == 0) {
      mbar_init(bar_q, 1);
      for (int x = 0; x < 2; ++x) { mbar_init(bar_sfull + 8 * x, 1); mbar_init(bar_pfull + 8 * x, 128); mbar_init(bar_pfull_hi + 8 * x, 128); mbar_init(bar_ofinal + 8 * x, 1); }
      for (int s = 0; s < L::kPairBars; ++s) { mbar_init(bar_full + 8 * s, 1); mbar_init(bar_empty + 8 * s, 1); }
      mbar_init(bar_vreq, 1);
      mbar_init(bar_vfix, 32);
      *abort_flag = 0;
      fence_barrier_init();
      fence_proxy_async_smem();
    }
    if (warp == 9) {
      tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), kTmemCols);
      tmem_relinquish();
    }
    // rows of the Q tiles that no (target, head) pair fills: zero them (they feed unused MMA rows)
    {
      const int used = pair_targets * G;
      const int n_pad = 2 * kBM - used;
      for (int i = threadIdx.x; i < n_pad * 8 * kHalves; i += kAttnThreads) {
        const int piece = i & 7, r = (i >> 3) % n_pad, hf = (i >> 3) / n_pad;
        *reinterpret_cast<uint4*>(base_ptr + L::kQ + hf * 2 * kHalfBytes + (used + r) * 128 + piece * 16) = make_uint4(0, 0, 0, 0);
      }
      fence_proxy_async_smem();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  };
  const bool early = r_cu == nullptr;
  auto give_back = [&]() {                                          // of a block that leaves with what it has set up
    if (!early) return;
    __syncthreads();
    if (warp == 9) { tc_fence_after(); tmem_dealloc(*tmem_slot, kTmemCols); }
  };
  if (threadIdx.x == 256) { prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_k); prefetch_tensormap(&tm_v); }
  // Block order.  Large contexts: KV head outermost, so one head's K/V stays in L2 while its tiles run.
  // Contexts that fit L2 whole (head_inner): tile pair outermost, so the longest tiles of every head start first.
  const int hd = head_inner ? (int)(blockIdx.x % Hkv) : (int)(blockIdx.x / n_pairs_total);
  const int tt = head_inner ? (int)(blockIdx.x / Hkv) : (int)(blockIdx.x - hd * n_pairs_total);
  const int b = find_segment(rt.tile_cu, B, tt);
  // Context split: this block walks the context tiles [j0, j0 + chunk) of its pair and leaves a normalised partial result + its log-sum-exp.
  // Either all pairs alike (gridDim.y, used when there are too few query tiles to fill the GPU) or the longest pairs of a request in pieces (pt).
  int p_rev = tt - rt.tile_cu[b], n_splits = (int)gridDim.y, split = (int)blockIdx.y, slot0 = 0;
  if (pt.most > 0) {
    split = unit_piece(p_rev, rt.tile_cu[b + 1] - rt.tile_cu[b], pt.pieces[b], pt.long_pairs[b], &p_rev);
    n_splits = split < 0 ? 1 : pt.pieces[b];
    split = max(split, 0);
    slot0 = pt.slot_cu[b] + p_rev * pair_targets;
  }
  if (early) set_up();
  if (early && threadIdx.x == 256) {
    // the first K/V tiles into L2 (a prefetch only: they are read after the wait)
    const int nr = rt.q_len[b], last = min(nr, ((nr + pair_targets - 1) / pair_targets - p_rev) * pair_targets) - 1;
    const int n = (rt.ctx_len[b] - nr + last) / kBN + 1, chunk = (n + (int)gridDim.y - 1) / (int)gridDim.y, t0 = (int)blockIdx.y * chunk;
    for (int t = t0; t < min(n, t0 + min(chunk, kL2Tiles)); ++t)
      for (int hf = 0; hf < kHalves; ++hf) {
        tma_prefetch_3d(&tm_k, hf * 64, hd, (int)rt.tok_off[b] + t * kBN);
        tma_prefetch_3d(&tm_v, hf * 64, hd, (int)rt.tok_off[b] + t * kBN);
      }
  }
  griddep_wait();
  const int status = *reinterpret_cast<volatile int*>(&st->status);       // (fetched beside the lists)
  // no lists (r_cu == NULL): the targets are the last q_len tokens of every request
  const int row_b = r_cu ? r_cu[b] : rt.q_cu[b];
  const int nr = r_cu ? r_cu[b + 1] - row_b : rt.q_len[b];
  const long long row0 = r_cu ? (long long)row_b - r_cu[0] : row_b;
  const int first_pos = rt.ctx_len[b] - nr;
  // dense_ctx: the context is the cache itself (every position of the request), a target's limit is its position
  const int nu = dense_ctx ? rt.ctx_len[b] : (u_cu[b + 1] - u_cu[b]);
  const int n_pairs_true = (nr + pair_targets - 1) / pair_targets;
  if (p_rev >= n_pairs_true) { give_back(); return; }
  // a true count above its host bound, or more target rows than q_new / out hold: report, touch nothing
  if (nr > rt.bound_a[b] || (mode == RELAXKV_CTX_UNION && nu > rt.bound_b[b]) ||
      row0 + nr > n_target_rows) {
    if (threadIdx.x == 0) report(st, RELAXKV_ERR_BAD_INDEX, KID_ATTN_SM100, nr, nu);
    give_back();
    return;
  }
  // After a timeout nothing is written.  (Without lists to wait for, the word is looked at where the outputs are written.)
  if (!early && status == RELAXKV_ERR_TIMEOUT) return;
  const int pair = n_pairs_true - 1 - p_rev;
  const int rho0 = pair * pair_targets;                       // first target of tile A
  const int ctx_len_b = (mode == RELAXKV_CTX_UNION) ? nu : rt.ctx_len[b];
  const long long ctx_base = dense_ctx ? rt.tok_off[b] : ((mode == RELAXKV_CTX_UNION) ? (long long)u_cu[b] : rt.ctx_cu[b]);
  const int q_row_base = (int)row0 + rho0;                    // (offsets of the lists are 32-bit)
  // targets of the pair, context tiles of each query tile
  const int n_tgt = min(pair_targets, nr - rho0);
  int n_kv[2];
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    n_kv[x] = 0;
    if (n_tgt * G > x * kBM) {
      const int rho_last = rho0 + (min(n_tgt * G, (x + 1) * kBM) - 1) / G;
      const int c = r_cu ? r_rank[row_b + rho_last] : first_pos + rho_last;
      const int cc = min(max(c, 0), max(nu - 1, 0));
      int lim_last = (mode == RELAXKV_CTX_UNION) ? cc : u_pos[u_cu[b] + cc];
      lim_last = min(max(lim_last, 0), ctx_len_b - 1);
      n_kv[x] = lim_last / kBN + 1;
    }
  }
  const int n_kv_max = max(n_kv[0], n_kv[1]);
  // slot of the pair's first row in the workspace (which holds some ten thousand); -1: the only piece, written to the output
  const int slot_base = n_splits == 1 ? -1 : (pt.most > 0 ? split * pt.slot_cu[B] + slot0 : split * (int)n_target_rows + q_row_base);
  const int chunk = (n_kv_max + n_splits - 1) / n_splits;
  const int j0 = split * chunk;
  int n_my[2];
#pragma unroll
  for (int x = 0; x < 2; ++x) n_my[x] = max(0, min(n_kv[x], j0 + chunk) - j0);
  const int n_my_max = max(n_my[0], n_my[1]);
  if (n_my_max == 0) {                        // nothing of this pair's context falls into this split
    if (slot_base >= 0 && threadIdx.x < 2 * kBM) {
      const int row = threadIdx.x, t_local = row / G;
      if (t_local < n_tgt) {
        part_lse[(long long)(slot_base + t_local) * H + hd * G + (row - t_local * G)] = -INFINITY;
      }
    }
    give_back();
    return;
  }

  // Cache-only calls read K/V tiles straight from the cache: the last tile of a request may reach past the request's
  // final token into rows that belong to nobody.  Their keys are masked, but their V rows would still meet a zero
  // probability on the tensor core (0 x NaN = NaN), so a helper warp zeroes those V rows once the tile has landed.
  const int v_fix_tile = (dense_ctx && (ctx_len_b % kBN) != 0) ? (ctx_len_b / kBN - j0) : -1;
  const bool need_v_fix = v_fix_tile >= 0 && v_fix_tile < n_my_max;

  if (!early) set_up();
  const uint32_t tmem_base = *tmem_slot;

  // Register budget: the control warpgroup gives registers to the two softmax warpgroups
  // (12 warps x 168 at launch = 8 x 224 + 4 x 56).
  if (warp >= 8) {
  reg_dealloc<56>();
  if (warp == 8) {
    // ================= TMA producer =================
    if (lane == 0) {
      mbar_expect_tx(bar_q, (uint32_t)(kHalves * pair_targets * G * 128));
      for (int hf = 0; hf < kHalves; ++hf)
        tma_load_3d(q_smem + hf * 2 * kHalfBytes, &tm_q, bar_q, hf * 64, hd * G, q_row_base);
      // The tiles travel in the order K_0 V_0 K_1 V_1 ... through the ring slots u % kRing (u = 2j for K_j, 2j + 1
      // for V_j; j counted from j0).  They are signalled in PAIRS p = (V_{p-1}, K_p): step j of the MMA warp needs
      // exactly pair j + 1 (V_j for P V, K_{j+1} for the next Q K^T), so it waits once and frees once per step.
      const bool fresh = all_rows_fresh(all_fresh, u_cu, r_cu);
      const CUtensorMap *map_k = fresh ? &tm_k_new : &tm_k, *map_v = fresh ? &tm_v_new : &tm_v;
      auto load_tile = [&](int u, uint32_t bar) {
        const int s = u % kRing;
        const int row = (int)(ctx_base + (long long)(j0 + (u >> 1)) * kBN);
        const CUtensorMap* tm = (u & 1) ? map_v : map_k;
        for (int hf = 0; hf < kHalves; ++hf)
          tma_load_3d(kv_smem + s * L::kTileBytes + hf * kHalfBytes, tm, bar, hf * 64, hd, row);
      };
      for (int pr = 0; pr <= n_my_max; ++pr) {                  // pair pr: V_{pr-1} (if pr > 0) and K_pr (if pr < n)
        const uint32_t bar = bar_full + 8 * (pr % L::kPairBars);
        const bool has_v = pr > 0, has_k = pr < n_my_max;
        // slot of V_{pr-1} was last used by K_{pr-3} (pair pr-3), slot of K_pr by V_{pr-3} (pair pr-2)
        if (pr >= 3 && !mbar_wait(bar_empty + 8 * ((pr - 3) % L::kPairBars), (uint32_t)((pr - 3) / L::kPairBars) & 1, abort_flag)) break;
        mbar_expect_tx(bar, (uint32_t)((has_v ? L::kTileBytes : 0) + (has_k ? L::kTileBytes : 0)));
        if (has_v) load_tile(2 * pr - 1, bar);
        if (has_k) {
          if (pr >= 3 && !mbar_wait(bar_empty + 8 * ((pr - 2) % L::kPairBars), (uint32_t)((pr - 2) / L::kPairBars) & 1, abort_flag)) break;
          load_tile(2 * pr, bar);
        }
      }
    }
  } else if (warp == 9) {
    // ================= MMA issuer =================
    if (lane == 0) {
      constexpr uint32_t idesc_qk = idesc_bf16_f32(kBM, kBN, 0);
      constexpr uint32_t idesc_pv = idesc_bf16_f32(kBM, D, 1);
      bool ok = mbar_wait(bar_q, 0, abort_flag);
      // This lane issues every MMA, and each instruction it executes in between delays the next one (measured: the
      // step got 1 % shorter when the ring-slot and barrier arithmetic below replaced a modulo and a division per
      // use).  So the positions are carried along and advanced once per step: ring slot of the step's V tile and of
      // the K tile behind it, and the pair barrier (byte offset, phase) that covers the two.
      uint32_t sv = 1, sk = 2, pk = 8, pph = 0;
      const int n0 = n_my[0], n1 = n_my[1];
      auto issue_qk = [&](int x, uint32_t slot) {                   // S_x = Q_x K^T with the K tile in `slot` -> bar_sfull[x]
        mma_ss_kloop<kHalves>(tmem_base + x * 128, desc_lo(q_smem + x * kHalfBytes, 16),
                              desc_lo(kv_smem + slot * L::kTileBytes, 16), desc_hi_sw128(1024), idesc_qk);
        mma_commit(bar_sfull + 8 * x);
      };
      // O_x += P_x V   (P_x read from TMEM where the softmax warps left it, over S_x; V in slot sv)
      auto issue_pv = [&](int x, uint32_t par, uint32_t acc) -> bool {
        const uint32_t v_lo = desc_lo(kv_smem + sv * L::kTileBytes, kHalfBytes);
        if (!mbar_wait(bar_pfull + 8 * x, par, abort_flag)) return false;
        tc_fence_after();
        mma_ts_steps<2 * kPLo>(tmem_base + 256 + x * 128, tmem_base + x * 128, v_lo, desc_hi_sw128(1024), idesc_pv, acc);
        // the last keys of P arrive while the first 32 * kPLo are being multiplied
        if (!mbar_wait(bar_pfull_hi + 8 * x, par, abort_flag)) return false;
        tc_fence_after();
        mma_ts_steps<8 - 2 * kPLo>(tmem_base + 256 + x * 128, tmem_base + x * 128 + 16 * kPLo, v_lo + 256 * kPLo, desc_hi_sw128(1024),
                                   idesc_pv, 1u);
        return true;
      };
      // pair 0 = K_0 alone
      if (ok) ok = mbar_wait(bar_full, 0, abort_flag);
      if (ok) {
        tc_fence_after();
        if (n0 > 0) issue_qk(0, 0);
        if (n1 > 0) issue_qk(1, 0);
        mma_commit(bar_empty);
      }
      for (int j = 0; ok && j < n_my_max; ++j) {                // j counted from j0; this step consumes pair j + 1
        if (!(ok = mbar_wait(bar_full + pk, pph, abort_flag))) break;
        if (need_v_fix && j == v_fix_tile) {                    // V_j reaches past the request's end: have those rows zeroed
          mbar_arrive(bar_vreq);
          if (!(ok = mbar_wait(bar_vfix, 0, abort_flag))) break;
        }
        tc_fence_after();
        const uint32_t par = (uint32_t)j & 1u, acc = j > 0 ? 1u : 0u;
        if (j < n0) {
          if (!(ok = issue_pv(0, par, acc))) break;
          if (j == n0 - 1) mma_commit(bar_ofinal);
          if (j + 1 < n0) issue_qk(0, sk);
        }
        if (j < n1) {
          if (!(ok = issue_pv(1, par, acc))) break;
          if (j == n1 - 1) mma_commit(bar_ofinal + 8);
          if (j + 1 < n1) issue_qk(1, sk);
        }
        mma_commit(bar_empty + pk);                             // V_j and K_{j+1}: free once both tiles are through
        sv += 2; if (sv >= kRing) sv -= kRing;
        sk += 2; if (sk >= kRing) sk -= kRing;
        pk += 8; if (pk == 8 * L::kPairBars) { pk = 0; pph ^= 1u; }
      }
    }
  } else if (warp == 10 && need_v_fix) {
    // ================= helper: zero the V rows past the request's last token (cache-only calls) =================
    if (mbar_wait(bar_vreq, 0, abort_flag)) {                   // raised by the MMA warp once that tile has landed
      const int first = ctx_len_b % kBN;                        // first foreign row of the tile
      uint8_t* vt = base_ptr + L::kKV + ((2 * v_fix_tile + 1) % kRing) * L::kTileBytes;
      for (int i = lane; i < (kBN - first) * 8 * kHalves; i += 32) {
        const int piece = i & 7, r = first + ((i >> 3) % (kBN - first)), hf = (i >> 3) / (kBN - first);
        *reinterpret_cast<uint4*>(vt + hf * kHalfBytes + r * 128 + piece * 16) = make_uint4(0, 0, 0, 0);
      }
      fence_proxy_async_smem();
    }
    mbar_arrive(bar_vfix);
  }
  } else {
    reg_alloc<224>();
    // ================= softmax + epilogue: thread = query row = TMEM lane =================
    const int x = warp >> 2;                                    // 0: tile A, 1: tile B
    const int t_local = (int)threadIdx.x / G, j_head = (int)threadIdx.x - t_local * G;      // flat rows of the pair: tile A, then B
    bool row_valid = t_local < n_tgt;
    const int rho_t = rho0 + t_local;
    // Rows without a target (one of 256 with five heads per KV head; three of 128 when a target's heads had to share a tile) and rows of an empty context see every key: what they
    // hold is not stored (an empty context's row is written as zeros), and a limit below the tile sends their whole warp through the
    // masking of every tile, 1.0 k clk of a 3.5 k step (12 layers of 40 / 8 heads at 32 K, repaired: 40.7 -> 37.3 ms; every row used,
    // 32 / 8 heads at 8 K: 8.42 -> 8.37).
    int limit = kNoLimit;
    bool row_empty = false;                                     // explicit lists: a target that sees no context entry
    if (row_valid) {
      const int c = r_cu ? r_rank[row_b + rho_t] : first_pos + rho_t;
      if (c == -1 && allow_empty) {
        row_empty = true;
      } else if (c < 0 || c >= nu) {
        report(st, RELAXKV_ERR_BAD_INDEX, KID_ATTN_SM100, c, nu);
        limit = 0;
      } else {
        limit = (mode == RELAXKV_CTX_UNION) ? c : u_pos[u_cu[b] + c];
        if (limit < 0 || limit >= ctx_len_b) { report(st, RELAXKV_ERR_BAD_INDEX, KID_ATTN_SM100, limit, ctx_len_b); limit = 0; }
      }
    }
    const uint32_t lane_base = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t t_s = lane_base + x * 128, t_o = lane_base + 256 + x * 128;
    const uint32_t my_sfull = bar_sfull + 8 * x, my_pfull = bar_pfull + 8 * x;
    const int my_n = n_my[x];
    limit -= j0 * kBN;                                          // counted from the split's first tile
    float m = -1.0e30f, z = 0.f;
    bool ok = true;
    for (int j = 0; j < my_n; ++j) {
      ok = mbar_wait(my_sfull, j & 1, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      softmax_step<D>(t_s, t_o, limit - j * kBN, j == 0, scale_log2, m, z, my_pfull, bar_pfull_hi + 8 * x);
    }
    if (ok && my_n > 0) {
      ok = mbar_wait(bar_ofinal + 8 * x, 0, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
    }
    row_valid = row_valid && status != RELAXKV_ERR_TIMEOUT;
    if (ok && my_n > 0) {
      tc_fence_after();
      const bool none = row_empty || !(z > 0.f);                // an empty context is defined as a zero output row
      const float inv = none ? 0.f : 1.f / z;
      const float lse = none ? -INFINITY : (m + log2f(z)) * kLn2A;
      const int orow = q_row_base + t_local;
      if (slot_base < 0) {
        uint16_t* optr = out + ((long long)orow * H + hd * G + j_head) * D;
        const bool sectors = (reinterpret_cast<uintptr_t>(out) & 31u) == 0;
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t o[32];
          tmem_ld32(t_o + c * 32, o);
          tmem_wait_ld();
          if (row_valid) {
#pragma unroll
            for (int i = 0; i < 32; i += 16) {
              uint32_t w[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(o[i + 2 * e]) * inv, __uint_as_float(o[i + 2 * e + 1]) * inv);
                // a row of an empty context is zero whatever the keys gave it (0 x NaN is not)
                w[e] = row_empty ? 0u : *reinterpret_cast<uint32_t*>(&h2);
              }
              store_16(optr + c * 32 + i, w, sectors);
            }
          }
        }
        if (row_valid && lse_out) lse_out[(long long)(hd * G + j_head) * n_target_rows + orow] = lse;
      } else {
        // partial result of this split: fp32, normalised by this split's own sum
        const long long slot = (long long)(slot_base + t_local) * H + hd * G + j_head;
        float* optr = part_o + slot * D;
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t o[32];
          tmem_ld32(t_o + c * 32, o);
          tmem_wait_ld();
          if (row_valid) {
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * inv);
#pragma unroll
            for (int i = 0; i < 32; i += 8) st_global_32b(optr + c * 32 + i, o + i);      // (the workspace is 256-byte aligned)
          }
        }
        if (row_valid) part_lse[slot] = lse;
      }
    } else if (ok && my_n == 0 && slot_base >= 0 && row_valid) {
      // this tile's context ends before the split begins (the pair's other tile still has work here)
      part_lse[(long long)(slot_base + t_local) * H + hd * G + j_head] = -INFINITY;
    }
  }

  // ---- teardown ------------------------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  griddep_launch();                         // behind the barrier: one thread that calls it early speaks for its block
  if (*abort_flag) {
    if (threadIdx.x == 0) report(st, RELAXKV_ERR_TIMEOUT, KID_ATTN_SM100, pair, hd);
    // give copies and MMAs still in flight time to land before shared memory and TMEM are released
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 200000ull) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ---------------------------------------------------------------------------------------------------------------------
// Persistent form of the kernel above, for calls whose blocks are short (a context of at most 128 tiles): one block
// per SM walks work items (pair of query tiles x KV head, the same list in the same longest-first order) that its
// producer lane claims from a global counter a few steps before the current item ends.  Barriers, tensor memory and
// the K/V ring live across items; the next item's first K tile travels with the current item's last V tile, its Q
// tiles are loaded as soon as the current item's last Q K^T has completed, and its first Q K^T is issued right behind
// the current item's last P V, so a block turn-over costs about 5 k clk instead of about 14 k.  Items reach the other
// roles as 64-byte records in a two-slot mailbox in shared memory.  One split only, gathered contexts only (the
// cache-only calls keep the kernel above).  Same arithmetic per row, hence the same bits.
// ---------------------------------------------------------------------------------------------------------------------
template <int D>
struct PersistSmem {
  static constexpr int kHalves = D / 64;
  static constexpr int kTileBytes = kHalves * kHalfBytes;
  static constexpr int kQ = 0;
  static constexpr int kKV = kQ + 2 * kTileBytes;
  static constexpr int kBar = kKV + kRing * kTileBytes;
  static constexpr int kPairBars = 3;
  // q | s, p, p_hi, ofinal x2 | pairs full/empty | qfree | odrained x2 | item full x2 | item free x2
  static constexpr int kNumBars = 1 + 8 + 2 * kPairBars + 1 + 2 + 2 + 2;
  static constexpr int kMisc = kBar + 8 * kNumBars;                     // tmem address, abort flag, two item records
  static constexpr int kTotal = kMisc + 8 + 2 * 64;
  static constexpr int kDynamic = kTotal + 1024;
};

// One work item as every role needs it; 16 ints so that it travels through shared memory as four 16-byte pieces.
struct WorkItem {
  int work;            // 1: work, -1: the list is exhausted
  int n_max, n_my0, n_my1;
  int n_tgt, pad0, hd, q_row_base;
  int nu, ctx_len_b, r_base, rho0;      // r_base = r_cu[b]
  int u_base, ctx_base, b, pad;         // u_base = u_cu[b]
  __device__ __forceinline__ int n_my(int x) const { return x ? n_my1 : n_my0; }
};
__device__ __forceinline__ void item_store(int4* rec, const WorkItem& it) {
  rec[0] = make_int4(it.work, it.n_max, it.n_my0, it.n_my1);
  rec[1] = make_int4(it.n_tgt, 0, it.hd, it.q_row_base);
  rec[2] = make_int4(it.nu, it.ctx_len_b, it.r_base, it.rho0);
  rec[3] = make_int4(it.u_base, it.ctx_base, it.b, 0);
}
__device__ __forceinline__ void item_load_head(const int4* rec, WorkItem& it) {      // what the MMA issuer needs
  const int4 a = rec[0];
  it.work = a.x; it.n_max = a.y; it.n_my0 = a.z; it.n_my1 = a.w;
}
__device__ __forceinline__ void item_load(const int4* rec, WorkItem& it) {
  item_load_head(rec, it);
  const int4 b = rec[1], c = rec[2], d = rec[3];
  it.n_tgt = b.x; it.pad0 = 0; it.hd = b.z; it.q_row_base = b.w;
  it.nu = c.x; it.ctx_len_b = c.y; it.r_base = c.z; it.rho0 = c.w;
  it.u_base = d.x; it.ctx_base = d.y; it.b = d.z; it.pad = 0;
}

__device__ __forceinline__ WorkItem decode_item(int id, const ReqTable& rt, int head_inner, int G, int Hkv, int mode, int pair_targets,
                                                const int* u_pos, const int* u_cu, const int* r_rank, const int* r_cu,
                                                long long n_target_rows, DeviceStatus* st) {
  WorkItem it;
  it.work = 0; it.pad = it.pad0 = 0;
  const int B = rt.n_req;
  const int n_pairs_total = rt.tile_cu[B];
  it.hd = head_inner ? (id % Hkv) : (id / n_pairs_total);
  const int tt = head_inner ? (id / Hkv) : (id - it.hd * n_pairs_total);
  const int b = find_segment(rt.tile_cu, B, tt);
  it.b = b;
  const int p_rev = tt - rt.tile_cu[b];
  it.r_base = r_cu[b]; it.u_base = u_cu[b];
  const int nr = r_cu[b + 1] - it.r_base;
  const int nu = u_cu[b + 1] - it.u_base;
  it.nu = nu;
  const int n_pairs_true = (nr + pair_targets - 1) / pair_targets;
  it.n_max = 0; it.n_my0 = it.n_my1 = 0; it.n_tgt = 0;
  it.rho0 = 0; it.ctx_len_b = 0; it.ctx_base = 0; it.q_row_base = 0;
  if (p_rev >= n_pairs_true) return it;
  if (nr > rt.bound_a[b] || (mode == RELAXKV_CTX_UNION && nu > rt.bound_b[b]) || (long long)(r_cu[b + 1] - r_cu[0]) > n_target_rows) {
    report(st, RELAXKV_ERR_BAD_INDEX, KID_ATTN_SM100, nr, nu);
    return it;
  }
  const int pair = n_pairs_true - 1 - p_rev;
  it.rho0 = pair * pair_targets;
  it.ctx_len_b = (mode == RELAXKV_CTX_UNION) ? nu : rt.ctx_len[b];
  it.ctx_base = (int)((mode == RELAXKV_CTX_UNION) ? (long long)it.u_base : rt.ctx_cu[b]);
  it.q_row_base = (it.r_base - r_cu[0]) + it.rho0;
  it.n_tgt = min(pair_targets, nr - it.rho0);
  int nm[2] = {0, 0};
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    if (it.n_tgt * G > x * kBM) {
      const int c = r_rank[it.r_base + it.rho0 + (min(it.n_tgt * G, (x + 1) * kBM) - 1) / G];
      const int cc = min(max(c, 0), max(nu - 1, 0));
      int lim_last = (mode == RELAXKV_CTX_UNION) ? cc : u_pos[it.u_base + cc];
      lim_last = min(max(lim_last, 0), it.ctx_len_b - 1);
      nm[x] = lim_last / kBN + 1;
    }
  }
  it.n_my0 = nm[0]; it.n_my1 = nm[1];
  it.n_max = max(nm[0], nm[1]);
  it.work = it.n_max > 0;
  return it;
}

template <int D>
__global__ void __launch_bounds__(kAttnThreads, 1)
attention_persist_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                         const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_k_new,
                         const __grid_constant__ CUtensorMap tm_v_new, int all_fresh, const __grid_constant__ ReqTable rt,
                         int mode, int allow_empty, int head_inner, int H, int Hkv, int pair_targets, float scale_log2,
                         const int* u_pos, const int* u_cu, const int* r_rank, const int* r_cu,
                         long long n_target_rows, uint16_t* __restrict__ out, float* __restrict__ lse_out,
                         int total_items, int* __restrict__ work_counter, DeviceStatus* st) {
  using L = PersistSmem<D>;
  constexpr int kHalves = L::kHalves;
  constexpr uint32_t kTmemCols = 512;
  const int G = H / Hkv;
  if (threadIdx.x == 256) { prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_k); prefetch_tensormap(&tm_v); }
  griddep_wait();
  if (*reinterpret_cast<volatile int*>(&st->status) == RELAXKV_ERR_TIMEOUT) return;

  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t q_smem = base + L::kQ, kv_smem = base + L::kKV;
  const uint32_t bar0 = base + L::kBar;
  const uint32_t bar_q = bar0;
  const uint32_t bar_sfull = bar0 + 8, bar_pfull = bar0 + 24, bar_pfull_hi = bar0 + 40, bar_ofinal = bar0 + 56;
  const uint32_t bar_full = bar0 + 72, bar_empty = bar_full + 8 * L::kPairBars;
  const uint32_t bar_qfree = bar_empty + 8 * L::kPairBars;
  const uint32_t bar_odrained = bar_qfree + 8;          // [2]
  const uint32_t bar_item = bar_odrained + 16;          // [2]
  const uint32_t bar_itemfree = bar_item + 16;          // [2]
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + L::kMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + L::kMisc + 4);
  int4* item_rec = reinterpret_cast<int4*>(base_ptr + L::kMisc + 8 + 8);   // two records of 64 bytes, 16-byte aligned
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    mbar_init(bar_q, 1);
    for (int x = 0; x < 2; ++x) { mbar_init(bar_sfull + 8 * x, 1); mbar_init(bar_pfull + 8 * x, 128); mbar_init(bar_pfull_hi + 8 * x, 128); mbar_init(bar_ofinal + 8 * x, 1); }
    for (int s = 0; s < L::kPairBars; ++s) { mbar_init(bar_full + 8 * s, 1); mbar_init(bar_empty + 8 * s, 1); }
    mbar_init(bar_qfree, 1);
    for (int x = 0; x < 2; ++x) { mbar_init(bar_odrained + 8 * x, 128); mbar_init(bar_item + 8 * x, 1); mbar_init(bar_itemfree + 8 * x, 2 * kBM + 1); }
    *abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == 9) { tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), kTmemCols); tmem_relinquish(); }
  {
    const int used = pair_targets * G;
    const int n_pad = 2 * kBM - used;
    for (int i = threadIdx.x; i < n_pad * 8 * kHalves; i += kAttnThreads) {
      const int piece = i & 7, r = (i >> 3) % n_pad, hf = (i >> 3) / n_pad;
      *reinterpret_cast<uint4*>(base_ptr + L::kQ + hf * 2 * kHalfBytes + (used + r) * 128 + piece * 16) = make_uint4(0, 0, 0, 0);
    }
    fence_proxy_async_smem();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // The k-th published record sits in slot k & 1 (phase k >> 1).  A reader copies it and arrives on the slot's
  // "free" barrier; the producer overwrites a slot only after all 257 readers of its previous record have done so.
  auto read_item = [&](int k, WorkItem& it, bool head_only) -> bool {
    if (!mbar_wait(bar_item + 8 * (k & 1), (uint32_t)(k >> 1) & 1, abort_flag)) return false;
    if (head_only) item_load_head(item_rec + 4 * (k & 1), it); else item_load(item_rec + 4 * (k & 1), it);
    mbar_arrive(bar_itemfree + 8 * (k & 1));
    return true;
  };

  if (warp >= 8) {
  reg_dealloc<56>();
  if (warp == 8) {
    // ================= producer: work items, Q tiles, K/V tiles =================
    if (lane == 0) {
      int n_fetched = 0, n_pub = 0;
      bool ok = true;
      auto fetch_work = [&](WorkItem& it) -> bool {          // next item that has work; false when the list is exhausted
        for (;;) {
          const int id = (n_fetched == 0) ? (int)blockIdx.x : (int)gridDim.x + atomicAdd(work_counter, 1);
          ++n_fetched;
          if (id >= total_items) { it.work = -1; return false; }
          it = decode_item(id, rt, head_inner, G, Hkv, mode, pair_targets, u_pos, u_cu, r_rank, r_cu, n_target_rows, st);
          if (it.work) return true;
        }
      };
      auto publish = [&](const WorkItem& it) -> bool {
        const int k = n_pub;
        if (k >= 2 && !mbar_wait(bar_itemfree + 8 * (k & 1), (uint32_t)((k - 2) >> 1) & 1, abort_flag)) return false;
        item_store(item_rec + 4 * (k & 1), it);
        mbar_arrive(bar_item + 8 * (k & 1));
        ++n_pub;
        return true;
      };
      auto load_q = [&](const WorkItem& it) {
        mbar_expect_tx(bar_q, (uint32_t)(kHalves * pair_targets * G * 128));
        for (int hf = 0; hf < kHalves; ++hf) tma_load_3d(q_smem + hf * 2 * kHalfBytes, &tm_q, bar_q, hf * 64, it.hd * G, it.q_row_base);
      };
      const bool fresh = all_rows_fresh(all_fresh, u_cu, r_cu);
      const CUtensorMap *map_k = fresh ? &tm_k_new : &tm_k, *map_v = fresh ? &tm_v_new : &tm_v;
      auto load_tile = [&](int u, const WorkItem& it, int j, uint32_t bar) {      // u = 2 g for K of global tile g, 2 g + 1 for V
        const int s = u % kRing;
        const int row = it.ctx_base + j * kBN;
        const CUtensorMap* tm = (u & 1) ? map_v : map_k;
        for (int hf = 0; hf < kHalves; ++hf) tma_load_3d(kv_smem + s * L::kTileBytes + hf * kHalfBytes, tm, bar, hf * 64, it.hd, row);
      };
      WorkItem cur, nxt;
      fetch_work(cur);
      ok = publish(cur);
      if (ok && cur.work > 0) {
        load_q(cur);
        int Gt = 0;                                                  // tile index, counted over the items, of cur's tile 0
        int cw = 0;                                                  // work items done so far
        for (;;) {
          bool have_nxt = false, fetched = false;
          for (int j = 0; ok && j <= cur.n_max; ++j) {               // pair g = (V_{g-1}, K_g)
            if (!fetched && j >= cur.n_max - 2) {                    // claim the next item late (the list balances the SMs
                                                                     // only if nobody holds work long before starting it),
                                                                     // yet a few steps before the readers ask for it
              have_nxt = fetch_work(nxt);
              fetched = true;
              if (!(ok = publish(nxt))) break;
            }
            if (j == 0 && cw > 0) continue;                          // loaded as the trailing pair of the previous item
            const int g = Gt + j;
            const bool has_v = j > 0;
            const bool has_k = (j < cur.n_max) || have_nxt;
            if (!has_v && !has_k) continue;
            const uint32_t bar = bar_full + 8 * (uint32_t)(g % L::kPairBars);
            if (g >= 3 && !(ok = mbar_wait(bar_empty + 8 * (uint32_t)((g - 3) % L::kPairBars), (uint32_t)((g - 3) / L::kPairBars) & 1, abort_flag))) break;
            mbar_expect_tx(bar, (uint32_t)((has_v ? L::kTileBytes : 0) + (has_k ? L::kTileBytes : 0)));
            if (has_v) load_tile(2 * g - 1, cur, j - 1, bar);
            if (has_k) {
              if (g >= 3 && !(ok = mbar_wait(bar_empty + 8 * (uint32_t)((g - 2) % L::kPairBars), (uint32_t)((g - 2) / L::kPairBars) & 1, abort_flag))) break;
              if (j < cur.n_max) load_tile(2 * g, cur, j, bar); else load_tile(2 * g, nxt, 0, bar);
            }
          }
          if (!ok || !have_nxt) break;
          // every Q K^T of cur has completed: the Q tiles may be replaced
          if (!(ok = mbar_wait(bar_qfree, (uint32_t)cw & 1, abort_flag))) break;
          load_q(nxt);
          Gt += cur.n_max; cur = nxt; ++cw;
        }
      }
    }
  } else if (warp == 9) {
    // ================= MMA issuer =================
    // One lane issues every MMA; each of its instructions delays the next one, so the loop over an item's inner steps
    // holds nothing but the waits and the issues, and the item's first and last step (which also look at the previous
    // item's epilogue and at the next item) run through a separate, general copy of the step.
    if (lane == 0) {
      constexpr uint32_t idesc_qk = idesc_bf16_f32(kBM, kBN, 0);
      constexpr uint32_t idesc_pv = idesc_bf16_f32(kBM, D, 1);
      bool ok = true;
      uint32_t k = 0;                       // index of the current item
      uint32_t sp0 = 0, sp1 = 0;            // parity of each tile's next P (its S / P barriers complete once per step)
      uint32_t op0 = 0, op1 = 0;            // epilogues of each tile so far (parity of its "O drained" barrier)
      // running positions, advanced once per step: ring slot of the step's V tile and of the K tile behind it, and the
      // pair barrier (offset, phase) that covers the two
      uint32_t sv = 1, sk = 2, pk = 8;
      uint32_t pph = 0;
      auto issue_qk = [&](int x, uint32_t slot) {                   // S_x = Q_x K^T with the K tile in `slot`
        mma_ss_kloop<kHalves>(tmem_base + x * 128, desc_lo(q_smem + x * kHalfBytes, 16), desc_lo(kv_smem + slot * L::kTileBytes, 16),
                              desc_hi_sw128(1024), idesc_qk);
        mma_commit(bar_sfull + 8 * x);
      };
      auto issue_pv = [&](int x, uint32_t par, uint32_t acc) -> bool {   // O_x (+)= P_x V with the V tile in slot sv
        const uint32_t v_lo = desc_lo(kv_smem + sv * L::kTileBytes, kHalfBytes);
        if (!mbar_wait(bar_pfull + 8 * x, par, abort_flag)) return false;
        tc_fence_after();
        mma_ts_steps<2 * kPLo>(tmem_base + 256 + x * 128, tmem_base + x * 128, v_lo, desc_hi_sw128(1024), idesc_pv, acc);
        if (!mbar_wait(bar_pfull_hi + 8 * x, par, abort_flag)) return false;
        tc_fence_after();
        mma_ts_steps<8 - 2 * kPLo>(tmem_base + 256 + x * 128, tmem_base + x * 128 + 16 * kPLo, v_lo + 256 * kPLo, desc_hi_sw128(1024),
                                   idesc_pv, 1u);
        return true;
      };
      auto advance = [&]() {
        mma_commit(bar_empty + pk);
        sv += 2; if (sv >= kRing) sv -= kRing;
        sk += 2; if (sk >= kRing) sk -= kRing;
        pk += 8; if (pk == 8 * L::kPairBars) { pk = 0; pph ^= 1u; }
      };
      WorkItem cur, nxt;
      cur.work = 0; nxt.work = 0; nxt.n_max = nxt.n_my0 = nxt.n_my1 = 0;
      ok = read_item(0, cur, true);
      if (ok && cur.work > 0) {
        ok = mbar_wait(bar_q, 0, abort_flag);
        if (ok) ok = mbar_wait(bar_full, 0, abort_flag);
        if (ok) {
          tc_fence_after();
          if (cur.n_my0 > 0) issue_qk(0, 0);
          if (cur.n_my1 > 0) issue_qk(1, 0);
          if (cur.n_max == 1) mma_commit(bar_qfree);
          mma_commit(bar_empty);
        }
        while (ok) {
          const int n0 = cur.n_my0, n1 = cur.n_my1, n_max = cur.n_max;
          bool have_nxt = false;
          // the general step: j = 0 and j = n_max - 1
          auto edge_step = [&](int j) -> bool {
            if (!mbar_wait(bar_full + pk, pph, abort_flag)) return false;
            const bool last = (j == n_max - 1);
            if (last) {                                             // the next item's record: shown early in cur
              if (!read_item((int)k + 1, nxt, true)) return false;
              have_nxt = nxt.work > 0;
            }
            tc_fence_after();
            bool q_ready = false;
            if (j < n0) {
              if (j == 0 && op0 > 0) {                              // O_0 of the previous item must have been read out
                if (!mbar_wait(bar_odrained, (op0 - 1) & 1u, abort_flag)) return false;
                tc_fence_after();
              }
              if (!issue_pv(0, (sp0 + (uint32_t)j) & 1u, j > 0 ? 1u : 0u)) return false;
              if (j == n0 - 1) mma_commit(bar_ofinal);
              if (j + 1 < n0) issue_qk(0, sk);
            }
            if (last && have_nxt && mbar_try_wait(bar_q, (k + 1) & 1u)) {   // the next item's Q tiles have landed already
              q_ready = true;
              tc_fence_after();
              if (nxt.n_my0 > 0) issue_qk(0, sk);
            }
            if (j < n1) {
              if (j == 0 && op1 > 0) {
                if (!mbar_wait(bar_odrained + 8, (op1 - 1) & 1u, abort_flag)) return false;
                tc_fence_after();
              }
              if (!issue_pv(1, (sp1 + (uint32_t)j) & 1u, j > 0 ? 1u : 0u)) return false;
              if (j == n1 - 1) mma_commit(bar_ofinal + 8);
              if (j + 1 < n1) issue_qk(1, sk);
            }
            if (last && have_nxt) {
              if (!q_ready) {
                if (!mbar_wait(bar_q, (k + 1) & 1u, abort_flag)) return false;
                tc_fence_after();
                if (nxt.n_my0 > 0) issue_qk(0, sk);
              }
              if (nxt.n_my1 > 0) issue_qk(1, sk);
              if (nxt.n_max == 1) mma_commit(bar_qfree);
            }
            advance();
            return true;
          };
          if (!(ok = edge_step(0))) break;
          // inner steps 1 .. n_max - 2
          for (int j = 1; j < n_max - 1; ++j) {
            if (!(ok = mbar_wait(bar_full + pk, pph, abort_flag))) break;
            tc_fence_after();
            if (j < n0) {
              if (!(ok = issue_pv(0, (sp0 + (uint32_t)j) & 1u, 1u))) break;
              if (j == n0 - 1) mma_commit(bar_ofinal);
              if (j + 1 < n0) issue_qk(0, sk);
            }
            if (j < n1) {
              if (!(ok = issue_pv(1, (sp1 + (uint32_t)j) & 1u, 1u))) break;
              if (j == n1 - 1) mma_commit(bar_ofinal + 8);
              if (j + 1 < n1) issue_qk(1, sk);
            }
            advance();
          }
          if (!ok) break;
          if (n_max >= 2) {
            mma_commit(bar_qfree);                                  // the last Q K^T of cur has been issued
            if (!(ok = edge_step(n_max - 1))) break;
          }
          sp0 += (uint32_t)n0; sp1 += (uint32_t)n1;
          op0 += (n0 > 0) ? 1u : 0u; op1 += (n1 > 0) ? 1u : 0u;
          if (!have_nxt) break;
          cur = nxt; ++k;
        }
      }
    }
  }
  } else {
    reg_alloc<224>();
    // ================= softmax + epilogue =================
    const int x = warp >> 2;
    const int t_local = (int)threadIdx.x / G, j_head = (int)threadIdx.x - t_local * G;      // flat rows of the pair: tile A, then B
    const uint32_t lane_base = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t t_s = lane_base + x * 128, t_o = lane_base + 256 + x * 128;
    const uint32_t my_sfull = bar_sfull + 8 * x, my_pfull = bar_pfull + 8 * x;
    const uint32_t rec_smem = smem_u32(item_rec);
    // One register of phase state: bit 0 = parity of this tile's next S, bit 1 = parity of its next final O,
    // bits 2.. = index of the current item.  The item's record stays in shared memory (its slot is released only
    // after the epilogue), so that little of it has to live in registers across the key loop.
    uint32_t ph = 0;
    auto rec_ld = [&](uint32_t k, int piece) -> int4 {
      int4 v;
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(rec_smem + (k & 1u) * 64u + piece * 16u));
      return v;
    };
    auto wait_rec = [&](uint32_t k) -> bool { return mbar_wait(bar_item + 8 * (k & 1u), (k >> 1) & 1u, abort_flag); };
    // this thread's row of item k: validity and the load of its context rank
    auto row_rank = [&](uint32_t k, bool& valid) -> int {
      const int4 a = rec_ld(k, 0), b = rec_ld(k, 1), cc = rec_ld(k, 2);
      valid = a.x > 0 && t_local < b.x;
      return valid ? r_rank[cc.z + cc.w + t_local] : 0;
    };
    bool ok = wait_rec(0);
    bool row_valid = false;
    int c = ok ? row_rank(0, row_valid) : 0;
    while (ok) {
      const uint32_t k = ph >> 2;
      int limit = kNoLimit, my_n;
      bool row_empty = false;
      {
        const int4 a = rec_ld(k, 0);
        if (a.x <= 0) { mbar_arrive(bar_itemfree + 8 * (k & 1u)); break; }
        my_n = x ? a.w : a.z;
        if (row_valid) {
          const int4 cc = rec_ld(k, 2), d = rec_ld(k, 3);
          const int nu = cc.x, ctx_len_b = cc.y;
          if (c == -1 && allow_empty) {
            row_empty = true;
          } else if (c < 0 || c >= nu) {
            report(st, RELAXKV_ERR_BAD_INDEX, KID_ATTN_SM100, c, nu);
            limit = 0;
          } else {
            limit = (mode == RELAXKV_CTX_UNION) ? c : u_pos[d.x + c];
            if (limit < 0 || limit >= ctx_len_b) { report(st, RELAXKV_ERR_BAD_INDEX, KID_ATTN_SM100, limit, ctx_len_b); limit = 0; }
          }
        }
      }
      float m = -1.0e30f, z = 0.f;
      for (int j = 0; j < my_n; ++j) {
        ok = mbar_wait(my_sfull, (ph + (uint32_t)j) & 1u, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        softmax_step<D>(t_s, t_o, limit - j * kBN, j == 0, scale_log2, m, z, my_pfull, bar_pfull_hi + 8 * x);
      }
      if (!ok) break;
      // the next item's record (shown long ago) and this thread's row of it: the load travels under the epilogue
      ok = wait_rec(k + 1);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      bool nrow_valid;
      const int nc = row_rank(k + 1, nrow_valid);
      if (my_n > 0) {
        ok = mbar_wait(bar_ofinal + 8 * x, (ph >> 1) & 1u, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const bool none = row_empty || !(z > 0.f);
        const float inv = none ? 0.f : 1.f / z;
        const float lse = none ? -INFINITY : (m + log2f(z)) * kLn2A;
        const int4 b = rec_ld(k, 1);
        const int hd = b.z;
        const long long orow = (long long)b.w + t_local;
        uint16_t* optr = out + ((long long)orow * H + hd * G + j_head) * D;
        const bool sectors = (reinterpret_cast<uintptr_t>(out) & 31u) == 0;
#pragma unroll
        for (int cc = 0; cc < D / 32; ++cc) {
          uint32_t o[32];
          tmem_ld32(t_o + cc * 32, o);
          tmem_wait_ld();
          if (row_valid) {
#pragma unroll
            for (int i = 0; i < 32; i += 16) {
              uint32_t w[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(o[i + 2 * e]) * inv, __uint_as_float(o[i + 2 * e + 1]) * inv);
                // a row of an empty context is zero whatever the keys gave it (0 x NaN is not)
                w[e] = row_empty ? 0u : *reinterpret_cast<uint32_t*>(&h2);
              }
              store_16(optr + cc * 32 + i, w, sectors);
            }
          }
        }
        if (row_valid && lse_out) lse_out[(long long)(hd * G + j_head) * n_target_rows + orow] = lse;
        tc_fence_before();
        mbar_arrive(bar_odrained + 8 * x);
        ph ^= 2u;
      }
      mbar_arrive(bar_itemfree + 8 * (k & 1u));                     // this thread is through with item k's record
      ph = ((ph + (uint32_t)my_n) & 1u) | (ph & 2u) | ((k + 1) << 2);
      c = nc; row_valid = nrow_valid;
    }
  }

  tc_fence_before();
  __syncthreads();
  griddep_launch();                         // behind the barrier: one thread that calls it early speaks for its block
  if (*abort_flag) {
    if (threadIdx.x == 0) report(st, RELAXKV_ERR_TIMEOUT, KID_ATTN_SM100, (int)blockIdx.x, -2);
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 200000ull) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == 9) { tc_fence_after(); tmem_dealloc(tmem_base, kTmemCols); }
}

// Explicit lists (the paper's controlled configurations): per target the index of the last context entry
// at or before its position (-1: none), per context entry the row of the fresh K/V that replaces it (-1:
// cached).  rt.tile_cu = prefix of the host bounds on the target counts, rt.bound_b = bounds on the context.
__global__ void build_list_maps_kernel(ReqTable rt, const int* __restrict__ ctx_pos, const int* __restrict__ ctx_cu,
                                       const int* __restrict__ tgt_pos, const int* __restrict__ tgt_cu,
                                       long long ctx_bound_total, int* __restrict__ limit, int* __restrict__ fresh_row,
                                       DeviceStatus* st) {
  const int B = rt.n_req;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long n_tgt_slots = rt.tile_cu[B];
  if (i < n_tgt_slots) {
    const int b = find_segment(rt.tile_cu, B, (int)i);
    const int rho = (int)i - rt.tile_cu[b];
    const int t0 = tgt_cu[b], nt = tgt_cu[b + 1] - t0;
    if (rho == 0 && (nt > rt.bound_a[b] || tgt_cu[0] != 0)) report(st, RELAXKV_ERR_BAD_INDEX, KID_ATTN_SM100, nt, tgt_cu[0]);
    if (rho < nt) {
      const int p = tgt_pos[t0 + rho];
      const int c0 = ctx_cu[b], nc = ctx_cu[b + 1] - c0;
      int lo = 0, hi = nc;                                   // first context entry with position > p
      while (lo < hi) { const int mid = (lo + hi) >> 1; if (ctx_pos[c0 + mid] <= p) lo = mid + 1; else hi = mid; }
      if (p < 0 || p >= rt.ctx_len[b]) { report(st, RELAXKV_ERR_BAD_INDEX, KID_ATTN_SM100, p, rt.ctx_len[b]); lo = 1; }
      limit[t0 + rho] = lo - 1;
    }
  } else if (i < n_tgt_slots + ctx_bound_total) {
    const long long x = i - n_tgt_slots;
    if (x < ctx_cu[B]) {
      int b = 0;
      while (b + 1 < B && x >= ctx_cu[b + 1]) ++b;
      const int p = ctx_pos[x];
      const int t0 = tgt_cu[b], nt = tgt_cu[b + 1] - t0;
      int lo = 0, hi = nt;
      while (lo < hi) { const int mid = (lo + hi) >> 1; if (tgt_pos[t0 + mid] < p) lo = mid + 1; else hi = mid; }
      fresh_row[x] = (lo < nt && tgt_pos[t0 + lo] == p) ? (t0 + lo) : -1;
    }
  }
}

// Test utility: one thread waits (bounded) on an mbarrier that nothing ever completes.  Exercises the
// give-up path of every kernel's waits without hanging anything: the wait expires after the limit,
// the abort flag is raised and RELAXKV_ERR_TIMEOUT lands in the device status word.
__global__ void wait_timeout_probe_kernel(DeviceStatus* st) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ volatile int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    mbar_init(smem_u32(&bar), 1);
    fence_barrier_init();
    const bool ok = mbar_wait(smem_u32(&bar), 0, &abort_flag);
    if (!ok && abort_flag) report(st, RELAXKV_ERR_TIMEOUT, KID_ATTN_SM100, -1, -1);
  }
}

constexpr int kCombineThreads = 128;
constexpr long long kCombineFewWarps = 64;
constexpr int kMaxCombineSplits = 1024;       // four warps x 4 KB of weights

// Merges the partial results of a context split: out = sum_s w_s O_s / sum_s w_s with w_s = exp(lse_s - max lse).
// One warp per (target row, query head), U partial results of it in flight.  Rows past the true target count, the rows of requests that the
// blocks in front refused (marked, kRefusedLse) and, after an expired wait, all rows are left alone: there are no partial results of them.
// ROWS: the rows of the call.  PIECES: the slots of the pairs that were cut (pt); what was refused is said per request.  LISTS: the rows of a call that
// no gather went before, whose counts are held against the bounds here.
// The loads are asked for side by side and whether a row is written is looked at last: a return before the sums lets the compiler move the
// loads behind it (attention of four requests of 700 to 1300 tokens, in pieces, 30.9 us a call / 27.8).
enum MergeForm { ROWS, PIECES, LISTS };
template <int U, MergeForm FORM>
__global__ void __launch_bounds__(kCombineThreads)
combine_splits_kernel(const float* part_o, const float* part_lse, int n_splits,
                      long long n_target_rows, int H, int D, const int* r_cu, const int* refused, int n_req,
                      uint16_t* __restrict__ out, float* __restrict__ lse_out, const __grid_constant__ PieceTable pt, int pair_targets,
                      DeviceStatus* st) {
  // the splits' weights of this warp's (row, head): the lanes fetch the log-sum-exps side by side (a serial walk over
  // the splits would pay one memory latency per split), the sums below still run in split order
  __shared__ float wgt_s[kCombineThreads / 32][kMaxCombineSplits];
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long w = (long long)blockIdx.x * (kCombineThreads / 32) + wib;
  const long long slot = w / H, slot_rows = FORM == PIECES ? pt.slot_cu[n_req] : n_target_rows;
  const int h = (int)(w - slot * H);
  const bool mine = slot < slot_rows;
  int b = 0;
  if (FORM == PIECES) {
    while (b + 1 < n_req && slot >= pt.slot_cu[b + 1]) ++b;
    n_splits = pt.pieces[b];
  }
  const int per = D / 32;                       // 2 or 4 consecutive floats per lane
  const float* o = part_o + (slot * H + h) * D + lane * per;
  const long long sp_stride = slot_rows * H * D;
  auto load = [&](int sp) -> float4 {
    if (per == 4) return *reinterpret_cast<const float4*>(o + sp * sp_stride);
    const float2 v = *reinterpret_cast<const float2*>(o + sp * sp_stride);
    return make_float4(v.x, v.y, 0.f, 0.f);
  };
  griddep_launch();
  griddep_wait();                               // the partial results come from the kernel before
  if (!mine) return;
  // A launch of a few rows is a chain of memory latencies, so the first partial results, the log-sum-exps and the row
  // count are fetched side by side (what rows past the true count or empty splits hold is not used), and each further
  // group of partial results while the one before is added up.
  const int status = *reinterpret_cast<volatile int*>(&st->status);
  float4 v[U];
#pragma unroll
  for (int u = 0; u < U; ++u) v[u] = u < n_splits ? load(u) : make_float4(0.f, 0.f, 0.f, 0.f);
  long long row = slot;
  bool here = true;                             // rows past the true counts (and requests that were refused) hold nothing
  if (FORM == PIECES) {
    const int c0 = r_cu[0], cb = r_cu[b], nr = r_cu[b + 1] - cb, rel = (int)slot - pt.slot_cu[b], p_rev = rel / pair_targets;
    const int rho = ((nr + pair_targets - 1) / pair_targets - 1 - p_rev) * pair_targets + rel - p_rev * pair_targets;
    row = (long long)(cb - c0) + rho;
    here = rho >= 0 && rho < nr && nr <= pt.bound[b] && (long long)(cb - c0) + nr <= n_target_rows && refused[b] == 0;
  } else {
    here = slot < (r_cu ? min((long long)(r_cu[n_req] - r_cu[0]), n_target_rows) : n_target_rows);
  }
  float mx = -INFINITY;
  for (int sp = lane; sp < n_splits; sp += 32) {
    const float l = part_lse[((long long)sp * slot_rows + slot) * H + h];
    wgt_s[wib][sp] = l;
    mx = fmaxf(mx, l);
  }
  mx = warp_reduce_max(mx);
  __syncwarp();
  for (int sp = lane; sp < n_splits; sp += 32) {
    const float l = wgt_s[wib][sp];
    wgt_s[wib][sp] = (l == -INFINITY || mx == -INFINITY) ? 0.f : __expf(l - mx);
  }
  __syncwarp();
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  float den = 0.f;
  for (int s0 = 0; s0 < n_splits; s0 += U) {    // fixed order: reproducible
    float4 nx[U];
#pragma unroll
    for (int u = 0; u < U; ++u) nx[u] = s0 + U + u < n_splits ? load(s0 + U + u) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float wgt = s0 + u < n_splits ? wgt_s[wib][s0 + u] : 0.f;
      const bool live = wgt > 0.f;                // an empty split wrote no partial output: whatever is there is ignored
      den += wgt;
      acc[0] = fmaf(wgt, live ? v[u].x : 0.f, acc[0]); acc[1] = fmaf(wgt, live ? v[u].y : 0.f, acc[1]);
      acc[2] = fmaf(wgt, live ? v[u].z : 0.f, acc[2]); acc[3] = fmaf(wgt, live ? v[u].w : 0.f, acc[3]);
      v[u] = nx[u];
    }
  }
  if (FORM == LISTS) {
    while (b + 1 < n_req && slot >= r_cu[b + 1] - r_cu[0]) ++b;
    here = here && r_cu[b + 1] - r_cu[b] <= pt.bound[b] && r_cu[b + 1] - r_cu[0] <= n_target_rows;
  }
  if (!here || mx == __uint_as_float(kRefusedLse) || status == RELAXKV_ERR_TIMEOUT) return;
  const float inv = den > 0.f ? 1.f / den : 0.f;
  uint16_t* optr = out + (row * H + h) * D + lane * per;
  __nv_bfloat162 h01 = __floats2bfloat162_rn(acc[0] * inv, acc[1] * inv);
  *reinterpret_cast<uint32_t*>(optr) = *reinterpret_cast<uint32_t*>(&h01);
  if (per == 4) {
    __nv_bfloat162 h23 = __floats2bfloat162_rn(acc[2] * inv, acc[3] * inv);
    *reinterpret_cast<uint32_t*>(optr + 2) = *reinterpret_cast<uint32_t*>(&h23);
  }
  if (lane == 0 && lse_out) lse_out[(long long)h * n_target_rows + row] = den > 0.f ? mx + logf(den) : -INFINITY;
}

relaxkv_status launch_combine_splits(const float* part_o, const float* part_lse, int n_splits, long long n_target_rows, int H,
                                     int D, const int32_t* r_cu, int n_req, long long rows_bound, void* out, float* lse_out,
                                     DeviceStatus* st, cudaStream_t stream) {
  const long long warps = rows_bound * H;
  if (warps <= 0) return RELAXKV_OK;
  if (n_splits > kMaxCombineSplits) return RELAXKV_ERR_UNSUPPORTED_SHAPE;
  constexpr int wpb = kCombineThreads / 32;
  // A decoded row whose context one wave of blocks shares (18 splits with eight KV heads): all of them in one go, one memory latency less (12 layers of a
  // decode step at 32 K 1985 us, 1970 so).  Up to eight splits the small form: with the registers of the large one beside it the next projection's
  // blocks come later (16 layers of four requests 1969 / 2017).
  auto kern = n_splits > 8 && warps <= kCombineFewWarps ? combine_splits_kernel<20, ROWS> : combine_splits_kernel<8, ROWS>;
  return cuda_ok(launch_chained(kern, (unsigned)((warps + wpb - 1) / wpb), kCombineThreads, 0, stream, part_o,
                                part_lse, n_splits, (long long)n_target_rows, H, D, r_cu, nullptr, n_req, static_cast<uint16_t*>(out), lse_out, PieceTable{}, 0, st));
}

// ---- host side ---------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static std::atomic<EncodeTiledFn> cached{nullptr};
  EncodeTiledFn fn = cached.load(std::memory_order_acquire);
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess) {
      fn = reinterpret_cast<EncodeTiledFn>(p);
      cached.store(fn, std::memory_order_release);
    }
  }
  return fn;
}

// bf16 tensor [d2, d1, d0] with d0 contiguous; box {64, b1, b2}; 128-byte swizzle; out-of-range reads give zeros.
bool make_map_3d(CUtensorMap* m, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint64_t stride1_bytes,
                 uint64_t stride2_bytes, uint32_t b1, uint32_t b2) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {d0, d1, d2};
  const cuuint64_t strides[2] = {stride1_bytes, stride2_bytes};
  const cuuint32_t box[3] = {64u, b1, b2};
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D>
static relaxkv_status launch_attention(const relaxkv_shape* shape, int mode, AttnPlan& plan, const void* q_new,
                                       const int32_t* u_pos, const int32_t* u_cu, const int32_t* r_rank,
                                       const int32_t* r_cu_layer, long long n_target_rows, void* out, float* lse_out,
                                       cudaStream_t stream, int allow_empty = 0) {
  const int H = shape->n_q_heads, Hkv = shape->n_kv_heads, G = H / Hkv;
  // A pair of query tiles is 256 rows: whole targets with the G heads of a KV head each, the one in the middle with heads in both tiles
  // where 128 is no multiple of G.  Five heads: 51 targets; with 25 in each tile, 2 % more pairs, 12 repaired layers of 40 / 8 heads at
  // 32 K took 36.09 ms, now 35.71, four of eight requests of 8 to 64 K 49.65 / 49.04.
  const int pair_targets = 2 * kBM / G;
  const int B = shape->n_req;
  for (int b = 0; b < B; ++b)     // tile_cu counts the launch units per request: PAIRS of query tiles
    plan.rt.tile_cu[b + 1] = plan.rt.tile_cu[b] + (plan.rt.bound_a[b] + pair_targets - 1) / pair_targets;
  const long long grid = (long long)plan.rt.tile_cu[B] * Hkv;
  if (grid == 0) return RELAXKV_OK;
  if (grid > 0x7fffffffLL) return RELAXKV_ERR_UNSUPPORTED_SHAPE;
  CUtensorMap tm_q, tm_k, tm_v;
  const uint64_t row_q = (uint64_t)H * D * 2, row_kv = (uint64_t)Hkv * D * 2;
  if (!make_map_3d(&tm_q, q_new, D, H, (uint64_t)n_target_rows, (uint64_t)D * 2, row_q, (uint32_t)G, (uint32_t)pair_targets) ||
      !make_map_3d(&tm_k, plan.k_base, D, Hkv, (uint64_t)plan.ctx_rows, plan.kv_head_stride_bytes, plan.kv_token_stride_bytes, 1u,
                   (uint32_t)kBN) ||
      !make_map_3d(&tm_v, plan.v_base, D, Hkv, (uint64_t)plan.ctx_rows, plan.kv_head_stride_bytes, plan.kv_token_stride_bytes, 1u,
                   (uint32_t)kBN))
    return RELAXKV_ERR_CUDA;
  // The fresh rows as a context (rows past the last read as zeros, as the materialised context's do).
  CUtensorMap tm_k_new = tm_k, tm_v_new = tm_v;
  if (plan.all_fresh > 0 &&
      (!make_map_3d(&tm_k_new, plan.k_new, D, Hkv, (uint64_t)plan.all_fresh, (uint64_t)D * 2, row_kv, 1u, (uint32_t)kBN) ||
       !make_map_3d(&tm_v_new, plan.v_new, D, Hkv, (uint64_t)plan.all_fresh, (uint64_t)D * 2, row_kv, 1u, (uint32_t)kBN)))
    return RELAXKV_ERR_CUDA;
  DeviceStatus* st = status_word();
  if (!st) return RELAXKV_ERR_CUDA;
  // the materialised context (K and V, all heads) against the 126 MB L2
  long long ctx_rows_used = 0;
  for (int b = 0; b < B; ++b) ctx_rows_used += plan.rt.bound_b[b];
  const int head_inner = (ctx_rows_used * (long long)row_kv * 2 <= (40ll << 20)) ? 1 : 0;
  const int sms = sm_count_of_current_device();
  if (sms <= 0) return RELAXKV_ERR_CUDA;
  // Context split.  A block's work is its pair's context length; with fewer blocks than a few waves of SMs (a query
  // prefill, a decode step, a layer with few targets, a short context) the longest pairs would run alone at the end,
  // so every pair's context is cut into pieces of at least four tiles until the launch has about four blocks per SM, one with fewer pairs than SMs.
  // A query's own rows (no lists) see their whole context and are few: as many pieces as there are SMs, of one tile if need be; the merge
  // takes as long as about three tiles, so up to four are left whole.  Pieces of four tiles at least as against one, us: 64 rows over 2 K 18.0 / 16.2,
  // 30 rows over 2 K with 8 / 2 heads 13.9 / 10.3, 100 rows over 5 K 17.9 / 15.7, 32 rows over 1 K with 4 / 1 heads of dim 64 10.5 / 8.6, requests of 512 and
  // 900 17.4 / 12.3; 57 rows over 8 K (of the 15 pieces asked for, 13 of five tiles; now 16 of four) 22.7 / 21.4.  Targets along the context
  // have shorter pairs and more rows to merge: 16 layers over 836 tokens, repaired, 503 / 511.
  long long max_tiles = 1;
  for (int b = 0; b < B; ++b) max_tiles = std::max<long long>(max_tiles, (plan.rt.bound_b[b] + kBN - 1) / kBN);
  long long n_splits = 1;
  const int forced = (shape->h_tuning && shape->h_tuning->attention_ctx_splits > 0) ? shape->h_tuning->attention_ctx_splits : 0;
  if (forced > 0) {
    n_splits = forced;
  } else if (grid < 4ll * sms) {
    n_splits = grid < sms && !r_cu_layer
                   ? std::min<long long>(sms / grid, max_tiles > 4 ? max_tiles : 1)
                   : std::min<long long>(std::max<long long>(1, (grid < sms ? sms : 4ll * sms) / grid), std::max<long long>(1, max_tiles / 4));
  }
  n_splits = std::min<long long>(n_splits, kMaxCtxSplits);
  n_splits = std::min<long long>(n_splits, kSplitRowsCap / n_target_rows);   // partial slots: [split][row of the call]
  if (n_splits < 1) n_splits = 1;
  // Or only the longest pairs of the call, in pieces.  Decided without a look at attention_persistent, whose settings have the same bits; a number of
  // blocks asked for is one of the persistent form, which has no pieces.
  PieceTable pt{};
  const bool automatic = forced == 0 && (!shape->h_tuning || shape->h_tuning->attention_grid_blocks <= 0);
  if (automatic && r_cu_layer && !plan.dense_ctx && grid <= 4ll * sms) {
    int tiles[kMaxReqInline], pairs[kMaxReqInline];
    double steps = 0.0;
    for (int b = 0; b < B; ++b) {
      tiles[b] = (plan.rt.bound_b[b] + kBN - 1) / kBN;
      pairs[b] = tiles[b] > 0 ? plan.rt.tile_cu[b + 1] - plan.rt.tile_cu[b] : 0;
      steps += 0.5 * tiles[b] * (pairs[b] + 1) * (pairs[b] > 0);
    }
    const double per_sm = steps * Hkv / sms;
    const double bytes = 2.0 * n_splits * plan.sum_targets * H * D * 4;
    const double uncut = std::max((double)max_tiles / (double)n_splits, 1.05 * per_sm) + (n_splits > 1 ? kPieceMergeSteps + bytes / kPieceBytesPerStep : 0.0);
    pt = plan_pieces(tiles, pairs, plan.rt.bound_a, B, pair_targets, Hkv, (long long)H * D * 4, split_rows_cap(shape), sms, uncut);
  }
  if (pt.most > 0) {
    n_splits = 1;
    int cu = 0;
    for (int b = 0; b < B; ++b) {
      cu += (plan.rt.bound_a[b] + pair_targets - 1) / pair_targets + pt.long_pairs[b] * (pt.pieces[b] - 1);
      plan.rt.tile_cu[b + 1] = cu;
    }
  }
  const long long units = (long long)plan.rt.tile_cu[B] * Hkv;
  auto kern = attention_sm100_kernel<D>;
  static std::atomic<int> attr_done[kMaxDevices];          // per device: the opt-in to > 48 KB of dynamic shared memory
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return RELAXKV_ERR_CUDA;
  if (!attr_done[dev].load(std::memory_order_acquire)) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnSmem<D>::kDynamic) != cudaSuccess)
      return RELAXKV_ERR_CUDA;
    attr_done[dev].store(1, std::memory_order_release);
  }
  // Persistent form: where a block's work is short the turn-over between blocks is what there is to save (measured
  // 3 % at an 8K context; nothing at 32K, where the chip runs at its power cap either way).
  const relaxkv_tuning* tun = shape->h_tuning;
  const int want_persist = tun ? tun->attention_persistent : 0;
  if (n_splits == 1 && pt.most == 0 && !plan.dense_ctx && (want_persist == 1 || (want_persist == 0 && max_tiles <= kPersistMaxTiles && grid > sms))) {
    auto pk = attention_persist_kernel<D>;
    static std::atomic<int> pattr_done[kMaxDevices];
    if (!pattr_done[dev].load(std::memory_order_acquire)) {
      if (cudaFuncSetAttribute(pk, cudaFuncAttributeMaxDynamicSharedMemorySize, PersistSmem<D>::kDynamic) != cudaSuccess)
        return RELAXKV_ERR_CUDA;
      pattr_done[dev].store(1, std::memory_order_release);
    }
    int* counter = reinterpret_cast<int*>(plan.split_o);            // unused by a one-split call; zeroed by the gather
    long long pgrid = std::min<long long>(grid, sms);
    if (tun && tun->attention_grid_blocks > 0) pgrid = std::min<long long>(grid, tun->attention_grid_blocks);
    RELAXKV_RANGE("attention_persist_kernel");
    return cuda_ok(launch_chained(pk, (unsigned)pgrid, kAttnThreads, PersistSmem<D>::kDynamic, stream,
        tm_q, tm_k, tm_v, tm_k_new, tm_v_new, plan.all_fresh, plan.rt, mode, allow_empty, head_inner, H, Hkv, pair_targets, shape->softmax_scale * kLog2eA,
        u_pos, u_cu, r_rank, r_cu_layer, n_target_rows, static_cast<uint16_t*>(out), lse_out, (int)grid, counter, st));
  }
  RELAXKV_RANGE("attention_sm100_kernel");
  relaxkv_status rc = cuda_ok(launch_chained(kern, dim3((unsigned)units, (unsigned)n_splits), kAttnThreads, AttnSmem<D>::kDynamic, stream,
      tm_q, tm_k, tm_v, tm_k_new, tm_v_new, plan.all_fresh, plan.rt, pt, mode, allow_empty, head_inner, plan.dense_ctx, H, Hkv, pair_targets, shape->softmax_scale * kLog2eA,
      u_pos, u_cu, r_rank, r_cu_layer, n_target_rows, static_cast<uint16_t*>(out), lse_out, plan.split_o, plan.split_lse, st));
  if (rc != RELAXKV_OK || (n_splits == 1 && pt.most == 0)) return rc;
  const bool own_counts = plan.dense_ctx && r_cu_layer;      // (no gather has marked what is refused)
  if (pt.most == 0 && !own_counts)
    return launch_combine_splits(plan.split_o, plan.split_lse, (int)n_splits, n_target_rows, H, D, r_cu_layer, B, plan.sum_targets, out, lse_out, st, stream);
  if (own_counts) std::copy_n(plan.rt.bound_a, B, pt.bound);
  const long long warps = (own_counts ? plan.sum_targets : pt.slot_cu[B]) * H;
  constexpr int wpb = kCombineThreads / 32;
  auto merge = own_counts ? combine_splits_kernel<8, LISTS> : combine_splits_kernel<8, PIECES>;
  return cuda_ok(launch_chained(merge, (unsigned)((warps + wpb - 1) / wpb), kCombineThreads, 0, stream, plan.split_o, plan.split_lse,
                                own_counts ? (int)n_splits : pt.most, n_target_rows, H, D, r_cu_layer, plan.refused, B, static_cast<uint16_t*>(out), lse_out, pt, pair_targets, st));
}

}  // namespace relaxkv

using namespace relaxkv;

extern "C" relaxkv_status relaxkv_sparse_ctx_attention(
    const relaxkv_shape* shape, relaxkv_ctx_mode mode, const relaxkv_cache_view* cache,
    const void* q_new, const void* k_new, const void* v_new,
    const int32_t* u_pos, const int32_t* u_cu, const int32_t* r_rank, const int32_t* r_cu_layer,
    int64_t n_target_rows, const int32_t* h_max_targets, const int32_t* h_max_ctx,
    void* out, float* lse_out, void* workspace, size_t workspace_bytes, relaxkv_stream stream_) {
  RELAXKV_RANGE("relaxkv_sparse_ctx_attention");
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  // The fresh rows may be read while outputs are written, unless a caller has the outputs take their place.
  bool fresh_in_place = false;
  if (shape && n_target_rows > 0) {
    auto apart = [&](const void* x, const void* y, long long y_bytes) {
      const uintptr_t x0 = reinterpret_cast<uintptr_t>(x), y0 = reinterpret_cast<uintptr_t>(y);
      const uintptr_t x_bytes = (uintptr_t)n_target_rows * shape->n_kv_heads * shape->head_dim * 2;
      return y == nullptr || x0 + x_bytes <= y0 || y0 + (uintptr_t)y_bytes <= x0;
    };
    const long long o_bytes = (long long)n_target_rows * shape->n_q_heads * shape->head_dim * 2, l_bytes = (long long)n_target_rows * shape->n_q_heads * 4;
    fresh_in_place = apart(k_new, out, o_bytes) && apart(v_new, out, o_bytes) && apart(k_new, lse_out, l_bytes) && apart(v_new, lse_out, l_bytes);
  }
  AttnPlan plan;
  relaxkv_status rc = prepare_attention(shape, mode, cache, q_new, k_new, v_new, u_pos, u_cu, r_rank, r_cu_layer,
                                        n_target_rows, h_max_targets, h_max_ctx, out, workspace, workspace_bytes,
                                        stream, plan, nullptr, fresh_in_place);
  if (rc != RELAXKV_OK) return rc;
  if (shape->head_dim == 128)
    return launch_attention<128>(shape, mode, plan, q_new, u_pos, u_cu, r_rank, r_cu_layer, n_target_rows, out, lse_out, stream);
  return launch_attention<64>(shape, mode, plan, q_new, u_pos, u_cu, r_rank, r_cu_layer, n_target_rows, out, lse_out, stream);
}

extern "C" relaxkv_status relaxkv_debug_wait_timeout(relaxkv_stream stream) {
  RELAXKV_RANGE("relaxkv_debug_wait_timeout");
  DeviceStatus* st = status_word();
  if (!st) return RELAXKV_ERR_CUDA;
  wait_timeout_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(st);
  return launch_ok();
}

extern "C" relaxkv_status relaxkv_list_attention(
    const relaxkv_shape* shape, const relaxkv_cache_view* cache,
    const void* q_new, const void* k_new, const void* v_new,
    const int32_t* ctx_pos, const int32_t* ctx_cu, const int32_t* tgt_pos, const int32_t* tgt_cu,
    int64_t n_target_rows, const int32_t* h_max_targets, const int32_t* h_max_ctx,
    void* out, float* lse_out, void* workspace, size_t workspace_bytes, relaxkv_stream stream_) {
  RELAXKV_RANGE("relaxkv_list_attention");
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  relaxkv_status rc = check_shape(shape);
  if (rc != RELAXKV_OK) return rc;
  if (!ctx_pos || !ctx_cu || !tgt_pos || !tgt_cu || !h_max_targets || !h_max_ctx || !workspace)
    return RELAXKV_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return RELAXKV_ERR_INVALID_ARG;
  const WsLayout ws = ws_layout(shape, 1);
  if (workspace_bytes < ws.total) return RELAXKV_ERR_WORKSPACE_TOO_SMALL;
  int* limit = reinterpret_cast<int*>(static_cast<char*>(workspace) + ws.list_limit);
  int* fresh = reinterpret_cast<int*>(static_cast<char*>(workspace) + ws.list_fresh);
  // 1. the two maps
  ReqTable rt;
  fill_req_table(rt, shape, nullptr, nullptr);
  long long tgt_total = 0, ctx_total = 0;
  for (int b = 0; b < shape->n_req; ++b) {
    if (h_max_targets[b] < 0 || h_max_targets[b] > shape->h_ctx_len[b] || h_max_ctx[b] < 0 ||
        h_max_ctx[b] > shape->h_ctx_len[b])
      return RELAXKV_ERR_INVALID_ARG;
    rt.bound_a[b] = h_max_targets[b];
    rt.bound_b[b] = h_max_ctx[b];
    tgt_total += h_max_targets[b];
    ctx_total += h_max_ctx[b];
    rt.tile_cu[b + 1] = (int)tgt_total;
  }
  if (tgt_total + ctx_total > 0x7fffffffLL) return RELAXKV_ERR_UNSUPPORTED_SHAPE;
  DeviceStatus* st = status_word();
  if (!st) return RELAXKV_ERR_CUDA;
  if (tgt_total + ctx_total > 0) {
    const long long n = tgt_total + ctx_total;
    build_list_maps_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(rt, ctx_pos, ctx_cu, tgt_pos, tgt_cu, ctx_total,
                                                                          limit, fresh, st);
    if ((rc = launch_ok()) != RELAXKV_OK) return rc;
  }
  // 2. gather (fresh rows resolved through the map) and 3. the attention kernel with the limits as "ranks"
  AttnPlan plan;
  rc = prepare_attention(shape, RELAXKV_CTX_UNION, cache, q_new, k_new, v_new, ctx_pos, ctx_cu, limit, tgt_cu, n_target_rows,
                         h_max_targets, h_max_ctx, out, workspace, workspace_bytes, stream, plan, fresh);
  if (rc != RELAXKV_OK) return rc;
  if (shape->head_dim == 128)
    return launch_attention<128>(shape, RELAXKV_CTX_UNION, plan, q_new, ctx_pos, ctx_cu, limit, tgt_cu, n_target_rows, out,
                                 lse_out, stream, 1);
  return launch_attention<64>(shape, RELAXKV_CTX_UNION, plan, q_new, ctx_pos, ctx_cu, limit, tgt_cu, n_target_rows, out,
                              lse_out, stream, 1);
}

// Attention of given token positions over the cache's own causal prefix (cache only, no gather): the tensor maps
// cover the cache, a target's causal limit is its position.
extern "C" relaxkv_status relaxkv_cache_attention(
    const relaxkv_shape* shape, const relaxkv_cache_view* cache, const void* q_new,
    const int32_t* tgt_pos, const int32_t* tgt_cu, int64_t n_target_rows, const int32_t* h_max_targets,
    void* out, float* lse_out, void* workspace, size_t workspace_bytes, relaxkv_stream stream) {
  RELAXKV_RANGE("relaxkv_cache_attention");
  if (!tgt_pos || !tgt_cu) return RELAXKV_ERR_INVALID_ARG;
  return relaxkv::cache_attention(shape, cache, q_new, tgt_pos, tgt_cu, n_target_rows, h_max_targets, out, lse_out, workspace,
                                  workspace_bytes, static_cast<cudaStream_t>(stream));
}

// No lists (both NULL): the targets are the last shape->h_q_len[b] tokens of every request, known to the kernels without a
// launch that writes them down.
relaxkv_status relaxkv::cache_attention(
    const relaxkv_shape* shape, const relaxkv_cache_view* cache, const void* q_new,
    const int32_t* tgt_pos, const int32_t* tgt_cu, int64_t n_target_rows, const int32_t* h_max_targets,
    void* out, float* lse_out, void* workspace, size_t workspace_bytes, cudaStream_t stream) {
  relaxkv_status rc = check_shape(shape);
  if (rc != RELAXKV_OK) return rc;
  if ((rc = check_cache(shape, cache, true)) != RELAXKV_OK) return rc;
  if (!q_new || !out || !h_max_targets || !workspace) return RELAXKV_ERR_INVALID_ARG;
  if (!aligned16(q_new) || !aligned16(out) || n_target_rows < 1) return RELAXKV_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return RELAXKV_ERR_INVALID_ARG;
  const WsLayout ws = ws_layout(shape, 1);
  if (workspace_bytes < ws.total) return RELAXKV_ERR_WORKSPACE_TOO_SMALL;
  AttnPlan plan;
  fill_req_table(plan.rt, shape, cache, nullptr);
  plan.sum_targets = 0;
  long long cache_rows = 0;
  for (int b = 0; b < shape->n_req; ++b) {
    if (h_max_targets[b] < 0 || h_max_targets[b] > shape->h_ctx_len[b]) return RELAXKV_ERR_INVALID_ARG;
    plan.rt.bound_a[b] = h_max_targets[b];
    plan.rt.bound_b[b] = shape->h_ctx_len[b];
    plan.sum_targets += h_max_targets[b];
    cache_rows = std::max<long long>(cache_rows, (long long)cache->h_req_token_offset[b] + shape->h_ctx_len[b]);
  }
  if (plan.sum_targets > 0x7fffffffLL || cache_rows > 0x7fffffffLL) return RELAXKV_ERR_UNSUPPORTED_SHAPE;
  char* base = static_cast<char*>(workspace);
  plan.kctx = nullptr; plan.vctx = nullptr;
  plan.split_o = reinterpret_cast<float*>(base + ws.split_o);
  plan.split_lse = reinterpret_cast<float*>(base + ws.split_lse);
  plan.k_base = cache->k; plan.v_base = cache->v;
  plan.kv_head_stride_bytes = (unsigned long long)cache->head_stride * 2;
  plan.kv_token_stride_bytes = (unsigned long long)cache->token_stride * 2;
  plan.ctx_rows = cache_rows;
  plan.dense_ctx = 1;
  // one target per request at most (a decode step): the streaming kernel
  bool one_each = true;
  for (int b = 0; b < shape->n_req; ++b) one_each = one_each && h_max_targets[b] <= 1;
  if (one_each) return launch_decode_attention(shape, plan, q_new, tgt_pos, tgt_cu, n_target_rows, out, lse_out, stream);
  // lists: targets by position (their "rank" in the dense context), counts from tgt_cu; u_pos / u_cu are not read
  if (shape->head_dim == 128)
    return launch_attention<128>(shape, RELAXKV_CTX_UNION, plan, q_new, nullptr, nullptr, tgt_pos, tgt_cu, n_target_rows, out,
                                 lse_out, stream);
  return launch_attention<64>(shape, RELAXKV_CTX_UNION, plan, q_new, nullptr, nullptr, tgt_pos, tgt_cu, n_target_rows, out,
                              lse_out, stream);
}
