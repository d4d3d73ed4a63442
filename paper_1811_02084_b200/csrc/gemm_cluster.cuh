// Contractions with too few 256-row output tiles to fill the chip: the same bf16 x bf16 -> fp32 product as
// gemm_tcgen05_kernel on 128 x BN tiles, one tile per CTA (not persistent, two CTAs fit an SM so that one loads while the
// other writes its result, and a dependent launch finds room to set itself up), and K cut over the CTAs of a cluster:
// each accumulates its range of k-blocks in its tensor memory, leaves the fp32 tile in shared memory, and finishes
// 1 / split of the rows: it adds the cluster's parts through distributed shared memory in ascending order of K and runs
// the component-wise stages on the sum, a 16-byte piece per thread, rows contiguous across lanes.
//
// The slices that a layout cuts M, N and the batch dimensions into do not appear here: every output element is one sum
// over all of K whoever owns it, so tiles run across slice boundaries and no slice edge is padded to a tile.
// Bound: at these sizes a fixed part (set-up, first loads, exchange, stores: 2.5 - 5 us) and 0.18 us (BN 64) or 0.20 us (BN 128) per
// 64-deep k-block of a CTA alone on its SM, which is what two loading threads in turn need for one (330 - 390 cycles).
// Measured against 256-row tiles with the whole of K on one pair: the feed-forward block (forward and backward) on 128 tokens,
// 1024 x 4096, 116 -> 48.6 us; the decoder layer's forward pass on 512 tokens 103 -> 57.4 us; the attention block on
// 3 x 200 tokens 118 -> 48.2 us (its core included).  These are passes over tensors that change from one to the next; over the same ones, which then lie in
// L2, 44.7, 51.6 and 47.6, and replayed from a graph 42.7, 49.0 and 44.3.
// Included by gemm_tcgen05.cu, whose wrappers, bounded waits and status word it uses.

struct ClusterArgs {
  int M, N;
  int n_outer;
  int outer_size[3];
  long long outer_sC[3];
  int a_mn_major, b_mn_major;
  long long ldc;
  int m_tiles, n_tiles;
  int tiles_group;           // tiles of one problem of a grouped launch
  int kb_term, kb_total;     // k-blocks of one product, of all products of a multi-term launch
  int grouped;
  int late_wait;
  void* C[3];
  int c_bf16;
  int c_wide;                // f32 rows (and outputs) start on 32 bytes
  const void* bias;
  int bias_bf16, bias_along_m;
  const void* mask;
  int mask_bf16;
  const void* resid;
  int resid_bf16;
  float scale[3];            // per problem of a grouped launch
  int relu;
  int k_from_row;            // the terms with k below the tile's first row are zero and are left out (one batch dimension's causal sums)
  float* rsum;               // column sums: added to the zeroed output, unless
  int rsum_store;            // ... one CTA has all rows: it stores them
  int rsum_gather;           // ... one cluster has all rows: its first CTA adds them up in order
  float* rsum_partial;       // not NULL: [row group][N], finished in order by a launch behind this one
};

constexpr int kClProducers = 2;
constexpr int kClThreads = 256;
constexpr int kClRingBytes = 96 * 1024;        // 4 stages of 24 KB (BN = 64) or 3 of 32 KB (BN = 128); the fp32 tile lies in the same bytes
constexpr int kClSmemBytes = kClRingBytes + 1024;

__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 ld_cluster(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ float ld_cluster1(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}

// four consecutive elements at `off` of a bf16 or f32 array (8- or 16-byte aligned)
__device__ __forceinline__ float4 ld_quad(const void* p, int bf16, long long off) {
  if (!bf16) return *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p) + off);
  const uint2 u = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(p) + off);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
}

// The fp32 tile in shared memory: 16-byte piece p of row r lies in slot q = p / 2 + (p mod 2) BN / 8 of the row, at
// r * 4 BN + ((q ^ (r mod 8)) * 16): the pieces that a warp reads together (even ones of neighbouring columns, then odd
// ones) and the ones it writes together (one piece of 32 rows) fall into different banks.
template <int BN>
__device__ __forceinline__ uint32_t tile_at(int row, int piece) {
  const uint32_t q = (uint32_t)(piece >> 1) + (uint32_t)(piece & 1) * (BN / 8);
  return (uint32_t)row * (BN * 4) + ((q ^ (uint32_t)(row & 7)) << 4);
}

// The component-wise stages on eight consecutive columns of one row, and the store.
template <bool kEpi>
__device__ __forceinline__ void finish_eight(const ClusterArgs& a, void* C, float scale, float* v, long long off, int m, bool second, const float* bias8, float* cs) {
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] *= scale;
  if (kEpi) {
    if (a.bias) {
      if (a.bias_along_m) {
        const float b = a.bias_bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(a.bias)[m]) : reinterpret_cast<const float*>(a.bias)[m];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += b;
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += bias8[j];
      }
    }
    if (a.relu) {
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = fmaxf(v[j], 0.f);
    }
    if (a.mask) {
      const float4 x = ld_quad(a.mask, a.mask_bf16, off), y = second ? ld_quad(a.mask, a.mask_bf16, off + 4) : x;
      const float k[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = k[j] > 0.f ? v[j] : 0.f;
    }
    if (a.rsum) {
#pragma unroll
      for (int j = 0; j < 8; ++j) cs[j] += v[j];
    }
    if (a.resid) {
      const float4 x = ld_quad(a.resid, a.resid_bf16, off), y = second ? ld_quad(a.resid, a.resid_bf16, off + 4) : x;
      v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w; v[4] += y.x; v[5] += y.y; v[6] += y.z; v[7] += y.w;
    }
  }
  if (a.c_bf16) {
    *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(C) + off) =
        make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
  } else if (a.c_wide && second) {   // a whole 32-byte sector an instruction (f32 4096 x 1024 from K = 128, twice in a feed-forward block on 128 tokens: the block 48.6 -> 45.2 us)
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(reinterpret_cast<float*>(C) + off), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
  } else {
    float4* const c = reinterpret_cast<float4*>(reinterpret_cast<float*>(C) + off);
    c[0] = make_float4(v[0], v[1], v[2], v[3]);
    if (second) c[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
}

// kSplit CTAs share a tile's K; kEpi: any stage beyond a scale
template <int BN, int kSplit, bool kEpi>
__global__ void __launch_bounds__(kClThreads, 2)
gemm_cluster_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const __grid_constant__ ExtraMaps extra,
                    const __grid_constant__ ClusterArgs a) {
  constexpr int kStageB = BN * BK * 2, kStage = kAStageBytes + kStageB, kStages = kClRingBytes / kStage;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t bars[2 * kStages + 1];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_word;
  __shared__ float col_part[kEpi ? 8 : 1][BN];
  const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
  volatile int* const abort_flag = &abort_word;
  auto full_bar = [&](int s) { return smem_u32(bars + s); };
  auto empty_bar = [&](int s) { return smem_u32(bars + kStages + s); };
  const uint32_t done_bar = smem_u32(bars + 2 * kStages);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  const int part = (int)(blockIdx.x % kSplit);
  int t = (int)(blockIdx.x / kSplit);
  const int group = t / a.tiles_group;
  t -= group * a.tiles_group;
  const int mt = t % a.m_tiles; t /= a.m_tiles;        // (neighbours share the tile of B)
  const int nt = t % a.n_tiles; t /= a.n_tiles;
  int o[3] = {0, 0, 0};
  long long c_off = 0;
  int row_block = 0;                                   // index of this tile's rows among all blocks of rows
  {
    int w = t;
    for (int j = a.n_outer - 1; j >= 0; --j) { o[j] = w % a.outer_size[j]; w /= a.outer_size[j]; c_off += (long long)o[j] * a.outer_sC[j]; }
    row_block = t * a.m_tiles + mt;
  }
  const int m0 = mt * BM, n0 = nt * BN;
  const int kb_first = a.k_from_row ? min(m0 / BK, a.kb_total - 1) : 0, kb_count = a.kb_total - kb_first;
  const int kb0 = kb_first + (int)((long long)kb_count * part / kSplit), kb1 = kb_first + (int)((long long)kb_count * (part + 1) / kSplit);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(done_bar, 1);
    abort_word = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_a) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_b) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(BN) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem = tmem_slot;
  if (!a.late_wait) asm volatile("griddepcontrol.wait;" ::: "memory");       // (see gemm_tcgen05_kernel)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // Two threads load, taking turns: a wait, the barrier's byte count and the copies of a k-block take one thread 560 - 680 cycles, however many
  // stages the ring has, and the MMAs 200 - 260.  128 x 1024 x 4096 unsplit 19.8 us with one, 14.3 with two; a third changes nothing.
  if (warp != 1 && warp <= kClProducers) {
    if (mtf::elect_one()) {
      const int first = warp ? warp - 1 : 0;
      int stage = first;
      uint32_t phase = 0;
      for (int kb = kb0 + first; kb < kb1; kb += kClProducers) {
        const int term = kb / a.kb_term, k0 = (kb - term * a.kb_term) * BK;
        const int sel = a.grouped ? group : term;
        const CUtensorMap* const pa = sel == 0 ? &map_a : &extra.m[2 * (sel - 1)];
        const CUtensorMap* const pb = sel == 0 ? &map_b : &extra.m[2 * (sel - 1) + 1];
        if (!mbar_wait(empty_bar(stage), phase ^ 1u, 0xA00 + stage, abort_flag)) break;
        const uint32_t fb = full_bar(stage), sa = ring + stage * kStage, sb = sa + kAStageBytes;
        mbar_expect_tx(fb, (uint32_t)kStage);
        if (a.a_mn_major) {
          tma_load_5d<false>(sa, pa, fb, m0, k0, o[2], o[1], o[0]);
          tma_load_5d<false>(sa + 8192, pa, fb, m0 + 64, k0, o[2], o[1], o[0]);
        } else {
          tma_load_5d<false>(sa, pa, fb, k0, m0, o[2], o[1], o[0]);
        }
        if (a.b_mn_major) {
#pragma unroll
          for (int j = 0; j < BN / 64; ++j) tma_load_5d<false>(sb + 8192 * j, pb, fb, n0 + 64 * j, k0, o[2], o[1], o[0]);
        } else {
          tma_load_5d<false>(sb, pb, fb, k0, n0, o[2], o[1], o[0]);
        }
        if ((stage += kClProducers) >= kStages) { stage -= kStages; phase ^= 1u; }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (mtf::elect_one()) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a.a_mn_major << 15) | ((uint32_t)a.b_mn_major << 16) |
                             ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
      const uint32_t a_step = a.a_mn_major ? 2048u : 32u, b_step = a.b_mn_major ? 2048u : 32u;
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!(ok = mbar_wait(full_bar(stage), phase, 0xA10 + stage, abort_flag))) break;
        tcgen05_fence_after();
        const uint32_t sa = ring + stage * kStage, sb = sa + kAStageBytes;
        const uint64_t da = make_smem_desc(sa, a.a_mn_major), db = make_smem_desc(sb, a.b_mn_major);
#pragma unroll
        for (int k = 0; k < BK / 16; ++k) umma_bf16<false>(tmem, da + k * (a_step >> 4), db + k * (b_step >> 4), idesc, (kb > kb0 || k) ? 1u : 0u);
        umma_commit<false>(empty_bar(stage), 0);
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
      if (ok) umma_commit<false>(done_bar, 0);
    }
    __syncwarp();
  }

  // ---- this CTA's part of the sum: tensor memory -> shared memory, two warps per lane quarter ----
  if (__all_sync(0xffffffffu, mbar_wait(done_bar, 0u, 0xA20, abort_flag))) {
    tcgen05_fence_after();
    const int row = (warp & 3) * 32 + lane;
#pragma unroll
    for (int c = 0; c < BN / 2; c += 32) {
      const int col = (warp >> 2) * (BN / 2) + c;
      uint32_t v[32];
      tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)col, v);
      tmem_ld_wait();
      if (kb0 == kb1) {              // (k_from_row: the last rows' few k-blocks may not reach every part)
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = 0u;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) st_shared_v4(ring + tile_at<BN>(row, col / 4 + j), v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
    }
  }
  tcgen05_fence_before();
  if (kSplit > 1) cluster_sync();
  else __syncthreads();

  // ---- sum over the cluster and the component-wise stages: a lane owns eight columns of a row ----
  constexpr int kLanesRow = BN / 8, kRowsPass = 32 / kLanesRow, kRowsWarp = BM / kSplit / 8;
  constexpr int kPasses = kRowsWarp > kRowsPass ? kRowsWarp / kRowsPass : 1;
  const bool lane_on = lane / kLanesRow < kRowsWarp;             // (split 8, BN 64: two rows a warp, half of a pass)
  const int piece = 2 * (lane % kLanesRow), n = n0 + 4 * piece;
  const int row0 = part * (BM / kSplit) + warp * kRowsWarp + lane / kLanesRow;
  const bool on = lane_on && n < a.N, second = n + 4 < a.N;
  void* const C = a.C[group];
  const float scale = a.scale[group];
  float bias8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, cs[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (kEpi && a.bias && !a.bias_along_m && on) {
    const float4 x = ld_quad(a.bias, a.bias_bf16, n), y = second ? ld_quad(a.bias, a.bias_bf16, n + 4) : x;
    bias8[0] = x.x; bias8[1] = x.y; bias8[2] = x.z; bias8[3] = x.w; bias8[4] = y.x; bias8[5] = y.y; bias8[6] = y.z; bias8[7] = y.w;
  }
  long long off = c_off + (long long)(m0 + row0) * a.ldc + n;
  if (kSplit > 1) {
    float s[kPasses][8];
#pragma unroll
    for (int i = 0; i < kPasses; ++i) {
      const uint32_t at0 = ring + tile_at<BN>(row0 + i * kRowsPass, piece), at1 = ring + tile_at<BN>(row0 + i * kRowsPass, piece + 1);
      if (on && m0 + row0 + i * kRowsPass < a.M) {
        float4 x[kSplit], y[kSplit];
#pragma unroll
        for (int q = 0; q < kSplit; ++q) { x[q] = ld_cluster(peer_addr(at0, q)); y[q] = second ? ld_cluster(peer_addr(at1, q)) : x[q]; }
        float* const v = s[i];
        v[0] = x[0].x; v[1] = x[0].y; v[2] = x[0].z; v[3] = x[0].w; v[4] = y[0].x; v[5] = y[0].y; v[6] = y[0].z; v[7] = y[0].w;
#pragma unroll
        for (int q = 1; q < kSplit; ++q) {
          v[0] += x[q].x; v[1] += x[q].y; v[2] += x[q].z; v[3] += x[q].w; v[4] += y[q].x; v[5] += y[q].y; v[6] += y[q].z; v[7] += y[q].w;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kPasses; ++i, off += kRowsPass * a.ldc)
      if (on && m0 + row0 + i * kRowsPass < a.M) finish_eight<kEpi>(a, C, scale, s[i], off, m0 + row0 + i * kRowsPass, second, bias8, cs);
    // With its reads done a CTA lets the rest of the cluster end (a peer's shared memory is gone once it has).  They are done here:
    // only what a store of this lane needs was read (no row past M, no piece past N), and the stores have taken it.  Nothing is
    // published, and a releasing arrive costs 0.3 us in front of the stores and 0.5 us behind them.
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  } else {
#pragma unroll 2
    for (int i = 0; i < kPasses; ++i, off += kRowsPass * a.ldc) {
      const int r = row0 + i * kRowsPass;
      if (!on || m0 + r >= a.M) continue;
      const uint4 x = ld_shared_v4(ring + tile_at<BN>(r, piece)), y = ld_shared_v4(ring + tile_at<BN>(r, piece + 1));
      float v[8] = {__uint_as_float(x.x), __uint_as_float(x.y), __uint_as_float(x.z), __uint_as_float(x.w),
                    __uint_as_float(y.x), __uint_as_float(y.y), __uint_as_float(y.z), __uint_as_float(y.w)};
      finish_eight<kEpi>(a, C, scale, v, off, m0 + r, second, bias8, cs);
    }
  }
  if (kEpi && a.rsum) {              // fused reduce_sum over this CTA's rows, in a fixed order
#pragma unroll
    for (int d = kLanesRow; d < 32; d <<= 1) {
#pragma unroll
      for (int j = 0; j < 8; ++j) cs[j] += __shfl_xor_sync(0xffffffffu, cs[j], d);
    }
    if (lane < kLanesRow) {
      *reinterpret_cast<float4*>(&col_part[warp][4 * piece]) = make_float4(cs[0], cs[1], cs[2], cs[3]);
      *reinterpret_cast<float4*>(&col_part[warp][4 * piece + 4]) = make_float4(cs[4], cs[5], cs[6], cs[7]);
    }
    __syncthreads();
    const int c = threadIdx.x;
    if (c < BN && n0 + c < a.N) {
      float x = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) x += col_part[w][c];
      if (a.rsum_gather) col_part[0][c] = x;
      else if (a.rsum_partial) a.rsum_partial[(size_t)(row_block * kSplit + part) * a.N + n0 + c] = x;
      else if (a.rsum_store) a.rsum[n0 + c] = x;
      else atomicAdd(a.rsum + n0 + c, x);
    }
    if (kSplit > 1 && a.rsum_gather) {
      __syncwarp();                  // (the aligned barriers take whole warps)
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
      cluster_sync();
      if (part == 0 && c < BN && n0 + c < a.N) {
        float x = 0.f;
#pragma unroll
        for (int q = 0; q < kSplit; ++q) x += ld_cluster1(peer_addr(smem_u32(&col_part[0][c]), q));
        a.rsum[n0 + c] = x;
      }
      __syncwarp();
      asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");      // (the store has taken what was read)
    }
  }
  if (*abort_flag)
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);      // failure path: copies and MMAs in flight land before the resources go away
  __syncwarp();
  if (kSplit > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");      // the cluster has read this CTA's part
  __syncthreads();
  if (a.late_wait) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (warp == 1) {
    __syncwarp();
    tcgen05_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN) : "memory");
  }
}

// How a launch runs here; split 0: not at all (gemm_tcgen05_kernel takes it).
struct ClusterPick { int bn, split; };
