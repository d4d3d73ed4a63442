// Attention core of the Transformer layout (Section 9: every (batch, head) pair is an independent problem) by rows: a CTA
// owns 128 query positions of one pair and walks the pair's keys in blocks of 128, so rows may have any length (a multiple
// of 8) and heads 64 or 128 columns.  Two launches of this shape, forward and backward:
//
//   forward   logits[l, m] = scale q[l] . kk[m]  (causal: m <= l);  P = softmax_m (bf16, written once);  o[l] = sum_m P[l, m] vv[m]
//   backward  D[l] = sum_m dP[l, m] P[l, m],  dP[l, m] = do[l] . vv[m];  dS[l, m] = P[l, m] (dP[l, m] - D[l]) (bf16, written
//             once);  dq[l] = scale sum_m dS[l, m] kk[m]
//
// Forward: the keys are walked twice.  The first walk leaves every row's maximum and sum of exponentials, the second forms
// the normalised weights, rounds them into a shared-memory tile that is both the source of the store to HBM and the A
// operand of O += P_j V_j.  Three blocks of fp32 logits fit tensor memory beside O, so rows of at most 384 keys keep them
// there and compute them once; longer rows compute them again, which costs d multiply-adds a logit on a pipe that waits for
// the exponentials anyway and saves the 8 bytes a logit of a trip through memory.
// Backward: also two walks.  The first one is the MMA thread's alone: D[l] = sum_v do[l, v] O[l, v] with O = P vv kept in
// fp32.  (From the stored, rounded o the row term is off by up to 0.1 of dS's rms on causal rows.)  The second forms dP,
// and dS over the tile of P it was made from.  dkk = dS^T q and dvv = P^T do sum over queries: a grouped contraction behind
// this launch reads dS and P.
// Blocks that lie wholly right of the diagonal are not computed; their weights are stored from a tile of zeros.
//
// Measured: 32 pairs of 1024 causal positions, heads of 128: forward 34 us against 105 us for logits, softmax and P . V as
// three launches; backward 32 + 26 us against 158 us for five.  24 pairs of 200 positions, heads of 64: the attention block
// forward and backward 71 -> 53 us.  Not used for heads of 64 with 128, 256, 384 or 512 positions, whose kernels keep a pair's
// keys on the chip: 256 pairs of 512 positions take 96 us here and 77 us there (forward), 168 and 156 us (backward).
//
// Bound: the special-function unit (16 exponentials a clock and SM) and the hand-overs between the MMA thread and the
// warps.  Warp roles (608 threads): 0 TMA loads, 1 MMA issue, 2 TMA stores, 3-18 arithmetic (four warps per tensor-memory
// lane quarter, each owns 32 of a block's 128 columns).  Row values that span the four warps of a quarter meet at a named
// barrier of its 128 threads.  Every mbarrier wait is bounded; on expiry a code is recorded, a CTA-wide flag is raised, the
// remaining waits return at once, work is skipped, and all roles leave through the teardown.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "launch.cuh"
#include "mtf_internal.h"

namespace {

constexpr int kWarps = 16;                        // arithmetic warps
constexpr int kThreads = 96 + 32 * kWarps;
constexpr uint32_t kBox = 128 * 64 * 2;           // 128 rows x 64 bf16 columns (128-byte rows, 128B swizzle)
constexpr int kSlots = 3;                         // ring of key-side blocks (K_j or V_j)
constexpr long long kWaitCycles = 4000000000LL;

__device__ int g_rows_status = 0;

struct RowArgs {
  int B, H, L;
  int causal;
  int q_tiles;
  int zeros;                     // also store zeros right of the diagonal
  float scale;
  __nv_bfloat16* out;            // o (forward) or dq (backward), [B, L, H, D]
};

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mb_init(uint32_t bar, uint32_t count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory"); }
__device__ __forceinline__ void mb_expect(uint32_t bar, uint32_t bytes) { asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory"); }
__device__ __forceinline__ void mb_arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }
__device__ __forceinline__ bool mb_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __noinline__ bool mb_wait_slow(uint32_t bar, uint32_t parity, int code, volatile int* abort_flag) {
  const long long t0 = clock64();
  while (true) {
    for (int i = 0; i < 64; ++i)
      if (mb_try(bar, parity)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > kWaitCycles) {
      atomicCAS(&g_rows_status, 0, code);
      *abort_flag = 1;
      return false;
    }
  }
}
__device__ __forceinline__ bool mb_wait(uint32_t bar, uint32_t parity, int code, volatile int* abort_flag) {
  for (int i = 0; i < 16; ++i)
    if (mb_try(bar, parity)) return true;
  return mb_wait_slow(bar, parity, code, abort_flag);
}
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
               ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_store(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(map), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void umma(uint32_t tmem_c, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(tmem_c), "l"(da), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Shared-memory matrix descriptor of a 128B-swizzled bf16 tile with rows of 128 bytes: K-major (a row holds 64 k-elements of
// one m/n index), or MN-major (64 m/n-elements of one k index; the next 64 m/n-elements one box further on).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, int mn_major) {
  const uint64_t lbo = mn_major ? (uint64_t)(kBox >> 4) : 1u;
  return (uint64_t)((addr & 0x3FFFF) >> 4) | (lbo << 16) | ((uint64_t)(1024u >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ uint32_t idesc_of(int b_mn, int n) {      // M = 128, A K-major
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)b_mn << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// 16-deep step ks of a K-major operand made of 64-wide boxes, in descriptor units
__device__ __forceinline__ uint64_t k_step(int ks) { return (uint64_t)((ks >> 2) * (int)(kBox >> 4) + (ks & 3) * 2); }
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h2);
}
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ uint4 lds_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void sts_v4(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

// Shared memory from a 1024-byte aligned base, D columns a head: the CTA's own rows (q, or do) | ring of key-side blocks |
// two 128 x 128 tiles (P, or P then dS) | a box of zeros | row exchange | barriers
template <int D>
struct Lay {
  static constexpr uint32_t own = 0, ring = own + (D / 64) * kBox, slot = (D / 64) * kBox, tile = ring + kSlots * slot, zero = tile + 4 * kBox,
                            xch = zero + kBox, bars = xch + 2 * 4 * 128 * 4, end = bars + 32 * 8 + 64;
};
enum { B_OWN = 0, B_KV_FULL, B_KV_EMPTY = B_KV_FULL + kSlots, B_S_FULL = B_KV_EMPTY + kSlots /*3*/, B_S_EMPTY = B_S_FULL + 3 /*3*/, B_T_LOAD = B_S_EMPTY + 3 /*2, backward: P has arrived*/,
       B_T_FULL = B_T_LOAD + 2 /*2: the warps have written a tile*/, B_T_EMPTY = B_T_FULL + 2 /*2*/, B_ACC = B_T_EMPTY + 2 /*2: O, dq complete*/, B_COUNT = B_ACC + 2 };

template <int D, bool kBwd>
__global__ void __launch_bounds__(kThreads, 1)
attention_rows_kernel(const __grid_constant__ CUtensorMap map_own, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                      const __grid_constant__ CUtensorMap map_p, const __grid_constant__ CUtensorMap map_ds, const RowArgs a) {
  using S = Lay<D>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = s_u32(smem_raw), base = (raw + 1023u) & ~1023u;
  const uint32_t bar0 = base + S::bars;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + (base - raw) + S::bars + 32 * 8);
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int L = a.L, units = a.B * a.H, n_blocks = (L + 127) / 128;
  // the longest rows first: the blocks that follow fill in behind them
  const int qt = a.q_tiles - 1 - (int)(blockIdx.x / (unsigned)units), u = (int)(blockIdx.x % (unsigned)units);
  const int b = u / a.H, h = u % a.H, row0 = qt * 128;
  const int nk = a.causal ? min(qt + 1, n_blocks) : n_blocks;      // key blocks with live columns
  const bool twice = nk > 3;                                       // forward: the logits of the second walk are computed again

  if (threadIdx.x == 0) {
    for (int i = 0; i < B_COUNT; ++i) mb_init(bar(i), 1);
    for (int i = 0; i < 3; ++i) mb_init(bar(B_S_EMPTY + i), kWarps);
    for (int i = 0; i < 2; ++i) { mb_init(bar(B_T_FULL + i), kWarps); mb_init(bar(B_T_EMPTY + i), 2); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_own) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_p) : "memory");
    if (kBwd) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_ds) : "memory");
  }
  if (a.zeros && nk < n_blocks)
    for (uint32_t i = threadIdx.x; i < kBox / 16; i += kThreads) sts_v4(base + S::zero + 16u * i, 0u, 0u, 0u, 0u);
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot, tmem_acc = tmem + 384u;        // three blocks of logits (or dP), then O / dq
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    // ------------------------------- TMA loads ----------------------------------
    if (mtf::elect_one()) {
      bool ok = true;
      int seq = 0, tiles = 0;
      auto block = [&](const CUtensorMap* map, int j) {
        const int s = seq % kSlots;
        if (!ok || !(ok = mb_wait(bar(B_KV_EMPTY + s), ((uint32_t)(seq / kSlots) & 1u) ^ 1u, 0xD01, abort_flag))) return;
        mb_expect(bar(B_KV_FULL + s), S::slot);
        for (int c = 0; c < D / 64; ++c) tma_load(base + S::ring + (uint32_t)s * S::slot + (uint32_t)c * kBox, map, bar(B_KV_FULL + s), c * 64, j * 128, h, b);
        ++seq;
      };
      auto tile_p = [&](int j) {
        const int s = tiles & 1;
        if (!ok || !(ok = mb_wait(bar(B_T_EMPTY + s), ((uint32_t)(tiles >> 1) & 1u) ^ 1u, 0xD02, abort_flag))) return;
        mb_expect(bar(B_T_LOAD + s), 2 * kBox);
        for (int c = 0; c < 2; ++c) tma_load(base + S::tile + (uint32_t)(2 * s + c) * kBox, &map_p, bar(B_T_LOAD + s), j * 128 + c * 64, row0, h, b);
        ++tiles;
      };
      mb_expect(bar(B_OWN), S::slot);
      for (int c = 0; c < D / 64; ++c) tma_load(base + S::own + (uint32_t)c * kBox, &map_own, bar(B_OWN), c * 64, row0, h, b);
      if (kBwd) {
        for (int j = 0; j < nk; ++j) { tile_p(j); block(&map_v, j); }
        for (int j = 0; j <= nk; ++j) {            // in the order the MMA thread wants them: dP_j, then dq of the block before
          if (j < nk) { block(&map_v, j); }
          if (j > 0) block(&map_k, j - 1);
          if (j < nk) tile_p(j);
        }
      } else {
        for (int j = 0; j < nk; ++j) block(&map_k, j);
        for (int j = 0; j <= nk; ++j) {
          if (twice && j < nk) block(&map_k, j);
          if (j > 0) block(&map_v, j - 1);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------- MMA issue ----------------------------------
    if (mtf::elect_one()) {
      const uint32_t id_s = idesc_of(0, 128), id_acc = idesc_of(1, D);
      const uint64_t d_own = smem_desc(base + S::own, 0);
      int seq = 0, sbuf = 0;                       // key-side blocks taken, logits (dP) blocks issued
      bool ok = mb_wait(bar(B_OWN), 0u, 0xD10, abort_flag);
      auto slot_in = [&]() -> uint32_t {           // the next key-side block
        const int s = seq % kSlots;
        ok = ok && mb_wait(bar(B_KV_FULL + s), (uint32_t)(seq / kSlots) & 1u, 0xD11, abort_flag);
        return base + S::ring + (uint32_t)s * S::slot;
      };
      auto slot_out = [&]() { umma_commit(bar(B_KV_EMPTY + seq % kSlots)); ++seq; };
      auto issue_s = [&]() {                       // own rows . block^T -> 128 x 128
        const uint32_t blk = slot_in();
        const int n = sbuf % 3;
        ok = ok && mb_wait(bar(B_S_EMPTY + n), ((uint32_t)(sbuf / 3) & 1u) ^ 1u, 0xD12, abort_flag);
        if (!ok) return;
        fence_after();
        const uint64_t db = smem_desc(blk, 0);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) umma(tmem + (uint32_t)n * 128u, d_own + k_step(ks), db + k_step(ks), id_s, ks != 0);
        umma_commit(bar(B_S_FULL + n));
        slot_out();
        ++sbuf;
      };
      auto issue_acc = [&](int tile, bool first) {      // tile (128 x 128 keys) . block -> O or dq
        const uint32_t blk = slot_in();
        if (!ok) return;
        fence_after();
        const uint64_t da = smem_desc(base + S::tile + (uint32_t)(2 * (tile & 1)) * kBox, 0), db = smem_desc(blk, 1);
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) umma(tmem_acc, da + k_step(ks), db + (uint64_t)(ks * (2048 >> 4)), id_acc, !first || ks != 0);
        umma_commit(bar(B_T_EMPTY + (tile & 1)));
        slot_out();
      };
      int tile = 0;
      if (kBwd) {
        for (int j = 0; j < nk && ok; ++j, ++tile) {       // O += P_j V_j
          ok = ok && mb_wait(bar(B_T_LOAD + (tile & 1)), (uint32_t)(tile >> 1) & 1u, 0xD13, abort_flag);
          issue_acc(tile, j == 0);
          if (ok) umma_commit(bar(B_T_EMPTY + (tile & 1)));      // (this walk's tiles have no store: both arrivals are the MMAs')
        }
        if (ok) umma_commit(bar(B_ACC));
      } else {
        for (int j = 0; j < nk && ok; ++j) issue_s();
      }
      for (int j = 0; j <= nk && ok; ++j) {
        if ((kBwd || twice) && j < nk) issue_s();          // the next block's logits / dP while the warps work on this one's
        if (j > 0 && ok) {
          ok = mb_wait(bar(B_T_FULL + (tile & 1)), (uint32_t)((j - 1) >> 1) & 1u, 0xD14, abort_flag);      // (the second walk's tiles only)
          if (ok) issue_acc(tile, j == 1);
          ++tile;
        }
      }
      if (ok) umma_commit(bar(B_ACC + 1));
    }
  } else if (warp == 2) {
    // ------------------------------- TMA stores ---------------------------------
    if (mtf::elect_one()) {
      const CUtensorMap* const map = kBwd ? &map_ds : &map_p;
      if (a.zeros)
        for (int j = nk; j < n_blocks; ++j)
          for (int c = 0; c < 2; ++c)
            if (j * 128 + c * 64 < L) tma_store(map, base + S::zero, j * 128 + c * 64, row0, h, b);
      const int first = kBwd ? nk & 1 : 0;         // parity of the tile the second walk begins with
      for (int j = 0; j < nk; ++j) {
        const int s = (first + j) & 1;
        if (!mb_wait(bar(B_T_FULL + s), (uint32_t)(j >> 1) & 1u, 0xD20, abort_flag)) break;
        for (int c = 0; c < 2; ++c)
          if (j * 128 + c * 64 < L) tma_store(map, base + S::tile + (uint32_t)(2 * s + c) * kBox, j * 128 + c * 64, row0, h, b);
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        mb_arrive(bar(B_T_EMPTY + s));
      }
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
  } else {
    // ------------------------------- arithmetic ---------------------------------
    const int q = warp & 3, part = (warp - 3) >> 2;        // lane quarter; which 32 of a block's 128 columns
    const int row_l = q * 32 + lane, row = row0 + row_l;
    const uint32_t lanes = (uint32_t)(q * 32) << 16;
    const uint32_t sw = (uint32_t)(row_l & 7);
    const uint32_t in_tile = (uint32_t)(part >> 1) * kBox + (uint32_t)row_l * 128u;        // this thread's four pieces of a tile
    auto piece = [&](int i) { return in_tile + ((((uint32_t)(part & 1) * 4u + (uint32_t)i) ^ sw) << 4); };
    bool ok = true;
    auto wait = [&](int i, uint32_t parity, int code) { ok = __all_sync(0xffffffffu, ok && mb_wait(bar(i), parity, code, abort_flag)); };
    // a value of every row from each of the quarter's four warps
    auto meet = [&](int plane, float mine, float* all) {
      const uint32_t x = base + S::xch + (uint32_t)plane * 2048u + 4u * (uint32_t)row_l;
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(x + 512u * (uint32_t)part), "f"(mine) : "memory");
      asm volatile("bar.sync %0, 128;" ::"r"(1 + q) : "memory");
#pragma unroll
      for (int p = 0; p < 4; ++p) asm volatile("ld.shared.f32 %0, [%1];" : "=f"(all[p]) : "r"(x + 512u * (uint32_t)p) : "memory");
    };
    uint32_t v[32];
    if (!kBwd) {
      const float sl2 = a.scale * 1.4426950408889634f;     // logits in units of log 2
      const int lim = a.causal ? min(L, row + 1) : L;      // columns [0, lim) take part
      const int lim_warp = __shfl_sync(0xffffffffu, lim, 31), lim_all = __shfl_sync(0xffffffffu, lim, 0);
      float mx = -INFINITY, sum = 0.f;
      for (int j = 0; j < nk; ++j) {
        const int c0 = j * 128 + part * 32;
        wait(B_S_FULL + j % 3, (uint32_t)(j / 3) & 1u, 0xD30);
        fence_after();
        const bool live = ok && c0 < lim_warp;
        if (live) {
          tmem_ld32(tmem + lanes + (uint32_t)((j % 3) * 128 + part * 32), v);
          tmem_ld_wait();
        }
        if (twice) {
          fence_before();
          __syncwarp();
          if (lane == 0) mb_arrive(bar(B_S_EMPTY + j % 3));
        }
        if (!live) continue;
        if (c0 + 32 > lim_all) {
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (c0 + i >= lim) v[i] = 0xff800000u;         // -inf
        }
        float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int i = 0; i < 32; ++i) m4[i & 3] = fmaxf(m4[i & 3], __uint_as_float(v[i]));
        const float m2 = fmaxf(mx, fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])));
        if (m2 == -INFINITY) {                             // no column above -inf yet; a NaN among them (fmaxf drops it) stays in the sum
          float t = 0.f;
#pragma unroll
          for (int i = 0; i < 32; ++i) t += __uint_as_float(v[i]);
          if (t != t) sum = t;
          continue;
        }
        const float off = m2 * sl2;
        float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 32; ++i) s4[i & 3] += ex2(fmaf(__uint_as_float(v[i]), sl2, -off));
        sum = sum * ex2(fmaf(mx, sl2, -off)) + ((s4[0] + s4[1]) + (s4[2] + s4[3]));
        mx = m2;
      }
      float ms[4], ss[4];
      meet(0, mx, ms);
      meet(1, sum, ss);
      const float top = fmaxf(fmaxf(ms[0], ms[1]), fmaxf(ms[2], ms[3])), off = top * sl2;
      float total = 0.f;
#pragma unroll
      for (int p = 0; p < 4; ++p) total += ms[p] == -INFINITY ? ss[p] : ss[p] * ex2(fmaf(ms[p], sl2, -off));
      const float inv = 1.f / total;
      for (int j = 0; j < nk; ++j) {
        const int c0 = j * 128 + part * 32, n = twice ? nk + j : j;
        if (twice) {
          wait(B_S_FULL + n % 3, (uint32_t)(n / 3) & 1u, 0xD31);
          fence_after();
        }
        const bool live = ok && c0 < lim_warp;
        if (live) {
          tmem_ld32(tmem + lanes + (uint32_t)((n % 3) * 128 + part * 32), v);
          tmem_ld_wait();
        }
        if (twice) {
          fence_before();
          __syncwarp();
          if (lane == 0) mb_arrive(bar(B_S_EMPTY + n % 3));
        }
        uint32_t pk[16];
        if (!live) {
#pragma unroll
          for (int i = 0; i < 16; ++i) pk[i] = 0u;
        } else if (c0 + 32 <= lim_all) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            pk[i] = pack2(ex2(fmaf(__uint_as_float(v[2 * i]), sl2, -off)) * inv, ex2(fmaf(__uint_as_float(v[2 * i + 1]), sl2, -off)) * inv);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            pk[i] = pack2(c0 + 2 * i < lim ? ex2(fmaf(__uint_as_float(v[2 * i]), sl2, -off)) * inv : 0.f,
                          c0 + 2 * i + 1 < lim ? ex2(fmaf(__uint_as_float(v[2 * i + 1]), sl2, -off)) * inv : 0.f);
        }
        wait(B_T_EMPTY + (j & 1), ((uint32_t)(j >> 1) & 1u) ^ 1u, 0xD32);
        const uint32_t tile = base + S::tile + (uint32_t)(2 * (j & 1)) * kBox;
        if (ok) {
#pragma unroll
          for (int i = 0; i < 4; ++i) sts_v4(tile + piece(i), pk[4 * i], pk[4 * i + 1], pk[4 * i + 2], pk[4 * i + 3]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mb_arrive(bar(B_T_FULL + (j & 1)));
      }
    } else {
      // D of this thread's row: its quarter of the columns of O against do (boxes of 64 columns, swizzled like every tile)
      wait(B_OWN, 0u, 0xD33);
      wait(B_ACC, 0u, 0xD34);
      fence_after();
      constexpr int kCols = D / 4;
      float dot = 0.f;
      if (ok) {
        if (kCols == 32) tmem_ld32(tmem_acc + lanes + (uint32_t)(part * kCols), v);
        else tmem_ld16(tmem_acc + lanes + (uint32_t)(part * kCols), v);
        uint4 w[kCols / 8];
#pragma unroll
        for (int i = 0; i < kCols / 8; ++i) {
          const int p = part * (kCols / 8) + i;            // 16-byte piece of the row
          w[i] = lds_v4(base + S::own + (uint32_t)(p >> 3) * kBox + (uint32_t)row_l * 128u + ((((uint32_t)p & 7u) ^ sw) << 4));
        }
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < kCols / 8; ++i) {
          const uint32_t ww[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            dot = fmaf(bf_lo(ww[e]), __uint_as_float(v[8 * i + 2 * e]), dot);
            dot = fmaf(bf_hi(ww[e]), __uint_as_float(v[8 * i + 2 * e + 1]), dot);
          }
        }
      }
      fence_before();
      float ds[4];
      meet(0, dot, ds);
      const float Dl = (ds[0] + ds[1]) + (ds[2] + ds[3]);
      for (int j = 0; j < nk; ++j) {
        const int t = nk + j;                              // tiles and their loads are counted through both walks
        const uint32_t tile = base + S::tile + (uint32_t)(2 * (t & 1)) * kBox;
        wait(B_S_FULL + j % 3, (uint32_t)(j / 3) & 1u, 0xD35);
        fence_after();
        if (ok) tmem_ld32(tmem + lanes + (uint32_t)((j % 3) * 128 + part * 32), v);
        wait(B_T_LOAD + (t & 1), (uint32_t)(t >> 1) & 1u, 0xD36);
        uint4 w[4];
        if (ok) {
#pragma unroll
          for (int i = 0; i < 4; ++i) w[i] = lds_v4(tile + piece(i));
        }
        tmem_ld_wait();
        fence_before();
        __syncwarp();
        if (lane == 0) mb_arrive(bar(B_S_EMPTY + j % 3));
        if (ok) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint32_t ww[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
            uint32_t r[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              r[e] = pack2(bf_lo(ww[e]) * (__uint_as_float(v[8 * i + 2 * e]) - Dl), bf_hi(ww[e]) * (__uint_as_float(v[8 * i + 2 * e + 1]) - Dl));
            sts_v4(tile + piece(i), r[0], r[1], r[2], r[3]);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mb_arrive(bar(B_T_FULL + (t & 1)));
      }
    }
    // O or dq: a quarter of the columns per warp
    wait(B_ACC + 1, 0u, 0xD37);
    fence_after();
    if (ok) {
      constexpr int kCols = D / 4;
      if (kCols == 32) tmem_ld32(tmem_acc + lanes + (uint32_t)(part * kCols), v);
      else tmem_ld16(tmem_acc + lanes + (uint32_t)(part * kCols), v);
      tmem_ld_wait();
      if (row < L) {
        const float s = kBwd ? a.scale : 1.f;
        uint4* const dst = reinterpret_cast<uint4*>(a.out + (((long long)b * L + row) * a.H + h) * D + part * kCols);
#pragma unroll
        for (int i = 0; i < kCols / 8; ++i)
          dst[i] = make_uint4(pack2(__uint_as_float(v[8 * i]) * s, __uint_as_float(v[8 * i + 1]) * s), pack2(__uint_as_float(v[8 * i + 2]) * s, __uint_as_float(v[8 * i + 3]) * s),
                              pack2(__uint_as_float(v[8 * i + 4]) * s, __uint_as_float(v[8 * i + 5]) * s), pack2(__uint_as_float(v[8 * i + 6]) * s, __uint_as_float(v[8 * i + 7]) * s));
      }
    }
  }

  // ------------------------------- teardown --------------------------------------
  __syncwarp();
  if (*abort_flag)
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);      // copies and MMAs in flight get time to land
  fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encoder() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qr) == cudaSuccess && qr == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// bf16 tensor as a 4-d map of boxes of 64 x 128: [d3][d2][d1][d0], d0 contiguous, strides of d1 .. d3 in elements
mtf_status box_map(CUtensorMap* m, const void* p, int64_t d0, int64_t d1, int64_t d2, int64_t d3, int64_t s1, int64_t s2, int64_t s3) {
  EncodeTiledFn enc = encoder();
  if (!enc) return mtf::fail(MTF_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
  const cuuint64_t d[4] = {(cuuint64_t)d0, (cuuint64_t)d1, (cuuint64_t)d2, (cuuint64_t)d3};
  const cuuint64_t s[3] = {(cuuint64_t)s1 * 2, (cuuint64_t)s2 * 2, (cuuint64_t)s3 * 2};
  const cuuint32_t box[4] = {64, 128, 1, 1}, es[4] = {1, 1, 1, 1};
  const CUresult r = mtf::in_context([&] { return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(p), d, s, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE); });
  return r == CUDA_SUCCESS ? MTF_OK : mtf::fail(MTF_ERR_CUDA, "cuTensorMapEncodeTiled failed with %d", (int)r);
}

template <int D, bool kBwd>
mtf_status launch_rows(const void* own, const void* kk, const void* vv, const void* weights, const void* ds, const RowArgs& a, cudaStream_t st) {
  const int64_t L = a.L, H = a.H, B = a.B;
  CUtensorMap mo, mk, mv, mp, md;
  mtf_status s;
  const void* const rows[3] = {own, kk, vv};
  CUtensorMap* const maps[3] = {&mo, &mk, &mv};
  for (int i = 0; i < 3; ++i)
    if ((s = box_map(maps[i], rows[i], D, L, H, B, H * D, D, L * H * D)) != MTF_OK) return s;
  if ((s = box_map(&mp, weights, L, L, H, B, L, L * L, H * L * L)) != MTF_OK) return s;
  if ((s = box_map(&md, ds ? ds : weights, L, L, H, B, L, L * L, H * L * L)) != MTF_OK) return s;
  constexpr size_t smem = 1024 + Lay<D>::end;
  cudaError_t e = cudaFuncSetAttribute(attention_rows_kernel<D, kBwd>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return mtf::fail(MTF_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3((unsigned)(B * H * a.q_tiles), 1, 1); cfg.blockDim = dim3(kThreads, 1, 1); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cfg.attrs = at; cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, attention_rows_kernel<D, kBwd>, mo, mk, mv, mp, md, a);
  if (e != cudaSuccess) return mtf::fail(MTF_ERR_CUDA, "attention_rows_kernel: %s", cudaGetErrorString(e));
  mtf::count_launch();
  return MTF_OK;
}

}  // namespace

namespace mtf {

bool attention_rows_supported(int64_t B, int64_t H, int64_t L, int64_t d_k, int64_t d_v) {
  return d_k == d_v && (d_k == 64 || d_k == 128) && L >= 8 && L % 8 == 0 && L <= 0x7fffff && B * H * ((L + 127) / 128) <= 0x7fffffffLL;
}

// own: q (forward) or do (backward) [B, L, H, D]; kk, vv [B, L, H, D]; weights [B, H, L, L] (written / read); ds [B, H, L, L] (backward only, written); out: o or
// dq.  All bf16, dense, 16-byte aligned.  `zeros`: positions right of the diagonal's blocks are written too (the weights always).
mtf_status launch_attention_rows(bool backward, const void* own, const void* kk, const void* vv, const void* weights, void* ds, void* out, int64_t B, int64_t H,
                                 int64_t L, int64_t D, float scale, int causal, int zeros, void* stream) {
  if (!attention_rows_supported(B, H, L, D, D)) return fail(MTF_ERR_UNSUPPORTED, "attention by rows: length %lld, head size %lld", (long long)L, (long long)D);
  if (!(scale > 0.f)) return fail(MTF_ERR_UNSUPPORTED, "attention by rows needs a positive scale");
  for (const void* p : {own, kk, vv, weights, (const void*)out, backward ? (const void*)ds : own})
    if (!p || (reinterpret_cast<uintptr_t>(p) & 15)) return fail(MTF_ERR_INVALID_ARG, "attention by rows: NULL or misaligned tensor");
  if (B * H <= 0) return MTF_OK;
  RowArgs a;
  a.B = (int)B; a.H = (int)H; a.L = (int)L; a.causal = causal ? 1 : 0; a.q_tiles = (int)((L + 127) / 128); a.zeros = zeros; a.scale = scale;
  a.out = reinterpret_cast<__nv_bfloat16*>(out);
  cudaStream_t st = (cudaStream_t)stream;
  if (D == 64) return backward ? launch_rows<64, true>(own, kk, vv, weights, ds, a, st) : launch_rows<64, false>(own, kk, vv, weights, nullptr, a, st);
  return backward ? launch_rows<128, true>(own, kk, vv, weights, ds, a, st) : launch_rows<128, false>(own, kk, vv, weights, nullptr, a, st);
}

mtf_status read_attention_rows_status(int* code) {
  int v = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_rows_status, sizeof(int));
  if (e != cudaSuccess) return fail(MTF_ERR_CUDA, "cudaMemcpyFromSymbol: %s", cudaGetErrorString(e));
  if (v) { int z = 0; cudaMemcpyToSymbol(g_rows_status, &z, sizeof(int)); }
  *code = v;
  return MTF_OK;
}

}  // namespace mtf
