// f32 einsums of matrix-product form (see F32Params) on the bf16 tensor cores, without giving up bits: 2^16 times an f32 value below
// 2^111 is the exact sum of three bf16 values, 2^16 a = a1 + a2 + a3 (a1 = bf16(2^16 a), a2 = bf16(2^16 a - a1), a3 = 2^16 a - a1 - a2), and
//   2^32 a b  =  a1 b1  +  (a1 b2 + a2 b1)  +  (a1 b3 + a2 b2 + a3 b1)  +  terms below 2^-25 |2^32 a b|,
// six exact products (the splitting of Henry, Tang and Heinecke, "Leveraging the bfloat16 Artificial Intelligence Datatype For
// Higher-Precision Computations", 2019).  The 2^16 puts the last bit of f32's smallest values, 2^-149, on bf16's, 2^-133: without it values below
// 2^-110 would lose bits, and a product below 2^-126 would too; what now leaves the range below is under 2^-155 a term, less than one f32
// addition drops there.  A value or a sum that leaves it above comes out infinite or NaN.  What limits the sums is the accumulator in tensor memory, which rounds towards zero on every addition.  So
// the large products never meet there: each 16-deep step of a1 b1 has an accumulator block of its own (one instruction, nothing added
// to it), the threads add the four blocks of a 64-deep stage pairwise and then to a running f32 sum, rounding to nearest; the small products stay
// in two more blocks (their rounding is 2^-8 of the large ones') and are added once at the end.
// Outputs that come out infinite or NaN (an infinity or NaN among their operands, a value from 2^111 or a sum from 2^96 on) are computed
// again by the warp that owns them, in plain f32 over the same part of K.
//
// A block of 512 threads owns a 128 x 64 tile: all threads load f32 (two stages ahead, in registers), split, and write the pieces into
// 128-byte-swizzled K- or MN-major boxes, whichever way the operand lies in memory; one thread issues a stage's 16 MMAs and they
// run while the block splits the next one.  Few tiles: K over up to 8 blocks of a cluster, whose parts are added in ascending order
// through distributed shared memory.  (Warps of their own for splitting, adding and issuing: 2048^3 228 us where this took 175, and 1 us
// more for a small product.)
// Bound: a stage takes 1.3 us (2500 cycles) and no unit is full in it: issue slots 53 %, shared memory's wavefronts 41 %, tensor pipe 28 % of the
// active cycles (2048 x 2048 x 1024).  Its steps follow one another: split and store, wait for the stage before, read its accumulators, barrier, issue; the
// tensor core idles from that wait to the issue, since a second set of a stage's a1 b1 blocks would need 640 of 512 columns (two sets of half a stage 384: not written).  A small product is the chain of
// launch, first loads, one stage and stores (4.5 us).
// Measured against plain FP32 arithmetic on the 64 x 64 tiles of einsum_f32.cu: 1024 x 1024 x 256 22.2 -> 9.5 us, 1024 x 256 x 1024 23.3 ->
// 11.2, 2048^3 503 -> 170, 128^3 6.1 -> 5.2, 8 x 256 x 64 4.8 -> 4.5; error against 64 bits (2-norm, normal values) 1.5e-7 -> 6.4e-8 at K = 256,
// 4.1e-7 -> 1.2e-7 at K = 2048, 6.0e-8 -> 4.8e-8 or less at K = 16.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "launch.cuh"
#include "mtf_internal.h"

namespace {

constexpr int kTM = 128, kTN = 64;      // rows and columns of C per block
constexpr int kBK = 64;                 // k of a stage
constexpr int kThreads = 512;
constexpr int kRing = 2;
constexpr uint32_t kPieceA = kTM * kBK * 2, kPieceB = kTN * kBK * 2, kStage = 3 * (kPieceA + kPieceB);
constexpr uint32_t kSmemBytes = kRing * kStage + 1024;
static_assert(32768 + kThreads / 32 * 32 * 53 * 4 <= kRing * kStage, "a stage per warp past the tile");
constexpr int kTmemCols = 512;          // four blocks of a1 b1, two of the small products, 64 columns each (allocations are powers of two)
constexpr long long kWaitCycles = 4000000000LL;
constexpr float kMost = 3.402823466e38f;                  // the largest f32
constexpr float kUp = 65536.f, kDown = 2.3283064365386962891e-10f;      // 2^16 on every operand, 2^-32 on the sums

__device__ int g_f32_status = 0;

struct F32TcArgs {
  F32Params p;
  int vecA, vecB;                   // 16-byte global loads are aligned
  int m_tiles, n_tiles, split;
  const float* A;
  const float* B;
  void* C;
  const void* bias;
  const void* mask;
  const void* resid;
  float* rsum;
  float* bsum;                      // not NULL: the sums over k of B's columns (of the blocks with the first rows)
  int late_wait;                    // this launch touches nothing that the launch before it touches: it waits for that one at its end
  int c_bf16, bias_bf16, mask_bf16, resid_bf16, relu;
  int rsum_mode;                    // 0: added to the zeroed output; 1: one block has all rows; 2: one cluster has
  float scale;
};

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mb_init(uint32_t bar, uint32_t count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory"); }
__device__ __forceinline__ void umma_commit(uint32_t bar) { asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory"); }
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
      atomicCAS(&g_f32_status, 0, code);
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
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void umma(uint32_t tmem_c, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
               ::"r"(tmem_c), "l"(da), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// 128B-swizzled boxes: K-major (a row of 128 bytes holds 64 k of one m|n), or MN-major (64 m|n of one k; the next 64 m|n 8 KB on)
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, int mn_major) {
  const uint64_t lbo = mn_major ? (8192u >> 4) : 1u;
  return (uint64_t)((addr & 0x3FFFF) >> 4) | (lbo << 16) | ((uint64_t)(1024u >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h2);
}
__device__ __forceinline__ float lo_of(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_of(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ float ld_any(const void* p, int bf16, long long off) {
  return bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[off]) : reinterpret_cast<const float*>(p)[off];
}
__device__ __forceinline__ float4 ld_peer(uint32_t addr, uint32_t rank) {
  float4 v;
  asm volatile(
      "{\n\t.reg .b32 ra;\n\t"
      "mapa.shared::cluster.u32 ra, %4, %5;\n\t"
      "ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [ra];\n\t}"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr), "r"(rank) : "memory");
  return v;
}
// the same piece of kParts blocks, added in ascending order (all loads before the first addition)
template <int kParts>
__device__ __forceinline__ float4 sum_parts(uint32_t addr) {
  float4 x[kParts];
#pragma unroll
  for (int q = 0; q < kParts; ++q) x[q] = ld_peer(addr, (uint32_t)q);
#pragma unroll
  for (int q = 1; q < kParts; ++q) { x[0].x += x[q].x; x[0].y += x[q].y; x[0].z += x[q].z; x[0].w += x[q].w; }
  return x[0];
}
// `nv` (1 to 4) consecutive values of a bf16 or f32 array
__device__ __forceinline__ float4 ld4_any(const void* p, int bf16, long long off, int nv) {
  if (!bf16) {
    const float* const f = reinterpret_cast<const float*>(p) + off;
    if (nv == 4 && !(reinterpret_cast<uintptr_t>(f) & 15)) return *reinterpret_cast<const float4*>(f);
  }
  float4 v = make_float4(ld_any(p, bf16, off), 0.f, 0.f, 0.f);
  if (nv > 1) v.y = ld_any(p, bf16, off + 1);
  if (nv > 2) v.z = ld_any(p, bf16, off + 2);
  if (nv > 3) v.w = ld_any(p, bf16, off + 3);
  return v;
}
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();                      // (the aligned barrier takes whole warps)
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Two f32 at a time
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair(float x, float y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ f32x2 pair_bits(uint32_t x, uint32_t y) { return pair(__uint_as_float(x), __uint_as_float(y)); }
__device__ __forceinline__ void unpair(f32x2 v, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// This thread's 16-byte pieces of a kRows x 64 operand tile.  Along k (s_k == 1): piece i is row tid / 16 + 32 i, k 4 (tid mod 16);
// otherwise along m|n: row 4 (tid mod (kRows / 4)), k tid / (kRows / 4) + (2048 / kRows) i.  Either way a thread's pieces lie at one
// swizzled address of the tile plus a multiple of whole 8-row groups.
template <int kRows, bool kAlongK>
struct Pieces {
  static constexpr int kN = kRows * kBK / 4 / kThreads, kPerK = kRows / 4, kStepK = kThreads / kPerK;
  static constexpr uint32_t kStepBytes = kAlongK ? 32 * 128 : kStepK * 128;
  const float* base;
  int off;                     // element offset of the first piece in the first stage
  int off_step, stage_step;    // what a piece and a stage add to it
  int mn, mn_end, k, s_mn;
  uint32_t at;                 // the first piece in the tile
  bool whole;                  // every piece lies inside the rows and is aligned
  __device__ __forceinline__ void init(const float* b, int smn, int sk, int v, int mn0, int rows_end) {
    const int tid = threadIdx.x;
    base = b; s_mn = smn; mn_end = rows_end;
    const int r = kAlongK ? tid >> 4 : 4 * (tid % kPerK);
    k = kAlongK ? 4 * (tid & 15) : tid / kPerK;
    mn = mn0 + r;
    whole = v != 0 && mn0 + kRows <= rows_end;
    off = min(mn, rows_end - 1) * smn + k * sk;          // (a row past the end is not read; its offset need not fit)
    off_step = kAlongK ? 32 * smn : kStepK * sk;
    stage_step = kBK * sk;
    at = kAlongK ? (uint32_t)r * 128u + ((((uint32_t)k >> 3) ^ ((uint32_t)r & 7u)) << 4) + ((uint32_t)k & 4u) * 2u
                 : ((uint32_t)r >> 6) * 8192u + (uint32_t)k * 128u + (((((uint32_t)r & 63u) >> 3) ^ ((uint32_t)k & 7u)) << 4) + ((uint32_t)r & 4u) * 2u;
  }
  __device__ __forceinline__ void load(int stage, int K, int vec, float4* r) const {
    const float* const first = base + (off + stage * stage_step);
    if (whole && (stage + 1) * kBK <= K) {
#pragma unroll
      for (int i = 0; i < kN; ++i) r[i] = __ldg(reinterpret_cast<const float4*>(first + i * off_step));
      return;
    }
#pragma unroll
    for (int i = 0; i < kN; ++i) {
      r[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      const int left = K - (stage * kBK + k + (kAlongK ? 0 : i * kStepK)), rows_left = mn_end - (mn + (kAlongK ? 32 * i : 0));
      if (left <= 0 || rows_left <= 0) continue;
      const float* const q = first + i * off_step;
      const int in = kAlongK ? left : rows_left, s = kAlongK ? 1 : s_mn;
      if (vec && in >= 4) { r[i] = __ldg(reinterpret_cast<const float4*>(q)); continue; }
      r[i].x = __ldg(q);
      if (in > 1) r[i].y = __ldg(q + s);
      if (in > 2) r[i].z = __ldg(q + 2 * s);
      if (in > 3) r[i].w = __ldg(q + 3 * s);
    }
  }
  // the three bf16 pieces of every value, times 2^16, into three tiles, `piece_bytes` apart
  template <uint32_t kPieceBytes>
  __device__ __forceinline__ void store(uint8_t* tile, const float4* r) const {
#pragma unroll
    for (int i = 0; i < kN; ++i) {
      f32x2 xy = mul2(pair(r[i].x, r[i].y), pair(kUp, kUp)), zw = mul2(pair(r[i].z, r[i].w), pair(kUp, kUp));
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        float x, y, z, w;
        unpair(xy, x, y); unpair(zw, z, w);
        const uint32_t p = pack2(x, y), s = pack2(z, w);
        *reinterpret_cast<uint2*>(tile + at + (q * kPieceBytes + i * kStepBytes)) = make_uint2(p, s);
        if (q < 2) { xy = sub2(xy, pair(lo_of(p), hi_of(p))); zw = sub2(zw, pair(lo_of(s), hi_of(s))); }
      }
    }
  }
};

// Plain f32 for the outputs of one warp's 32 rows x 16 columns that came out infinite or NaN: k from k0 to k1 in order, 32 at a time through the
// warp's own `stage`, loaded by lanes that lie side by side in memory.  `out`: this lane's row of the tile; piece q of its columns at 16 (q ^ sw).
// Bound: issue, about half of it multiply-adds.  All NaN, beside ordinary values and beside einsum_f32.cu (which takes the same time for either): 1024 x 1024 x 256
// 42.6, 9.5 and 22.2 us; 2048^3 1132, 170 and 503.  One NaN, which costs the warps of its row: 33 and 278.
constexpr int kStageA = 33, kStageB = 20, kStageFloats = 32 * (kStageA + kStageB);      // rows of A 33 words apart: no bank conflicts; of B 20: 16-byte pieces
__device__ __noinline__ void redo_plain(uint8_t* out, uint32_t sw, uint32_t q0, float* stage, const float* A, const float* B, int sAm, int sAk, int sBn, int sBk, int rows, int cols, int k0,
                                        int k1) {
  const int lane = threadIdx.x & 31, hi = lane >> 4, lo = lane & 15;
  const bool along_a = sAk == 1, along_b = sBk == 1;
  // this lane's values: along k, row (column) i at k = lane; otherwise row lane at k = i, column lo at k = 2 i + hi
  const float* pa = A + (along_a ? lane : lane * sAm);
  const float* pb = B + (along_b ? lane : lo * sBn + hi * sBk);
  const int step_a = along_a ? sAm : sAk, step_b = along_b ? sBn : 2 * sBk;
  float* const sa = stage + (along_a ? lane * kStageA : lane);
  float* const sb = stage + 32 * kStageA;
  float* const sb0 = sb + (along_b ? lane * kStageB : hi * kStageB + lo);
  const int put_a = along_a ? 1 : kStageA, put_b = along_b ? 1 : 2 * kStageB;
  float sum[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) sum[j] = 0.f;
  pa += (long long)k0 * sAk;
  pb += (long long)k0 * sBk;
#pragma unroll 1
  for (int left = k1 - k0; left > 0; left -= 32, pa += 32 * sAk, pb += 32 * sBk) {
    const int na = along_a ? (lane < left ? rows : 0) : (lane < rows ? left : 0), nb = along_b ? (lane < left ? cols : 0) : (lo < cols ? (left - hi + 1) / 2 : 0);
    float x[32], y[16];
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = i < na ? __ldg(pa + i * step_a) : 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) y[i] = i < nb ? __ldg(pb + i * step_b) : 0.f;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 32; ++i) sa[i * put_a] = x[i];
#pragma unroll
    for (int i = 0; i < 16; ++i) sb0[i * put_b] = y[i];
    __syncwarp();
#pragma unroll 4
    for (int k = 0; k < min(left, 32); ++k) {
      const float v = stage[k * kStageA + lane];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 b = *reinterpret_cast<const float4*>(sb + k * kStageB + 4 * q);
        sum[4 * q] = fmaf(v, b.x, sum[4 * q]);
        sum[4 * q + 1] = fmaf(v, b.y, sum[4 * q + 1]);
        sum[4 * q + 2] = fmaf(v, b.z, sum[4 * q + 2]);
        sum[4 * q + 3] = fmaf(v, b.w, sum[4 * q + 3]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    float* const o = reinterpret_cast<float*>(out + (((q0 + j / 4) ^ sw) << 4)) + (j & 3);
    if (!(fabsf(*o) <= kMost)) *o = sum[j];
  }
}

template <bool kAlongA, bool kAlongB>
__global__ void __launch_bounds__(kThreads, 1) einsum_f32_tc_kernel(const __grid_constant__ F32TcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t done_word;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_word;
  __shared__ float col_part[kTN];
  const uint32_t base = (s_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* const ring = smem_raw + (base - s_u32(smem_raw));
  const uint32_t done = s_u32(&done_word);
  volatile int* const abort_flag = &abort_word;
  const F32Params& p = a.p;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int part = (int)(blockIdx.x % (unsigned)a.split);       // this block's part of K (= its rank in the cluster)
  long long t = blockIdx.x / (unsigned)a.split;
  const int nt = (int)(t % a.n_tiles); t /= a.n_tiles;
  const int mt = (int)(t % a.m_tiles); t /= a.m_tiles;
  long long offA = 0, offB = 0, offC = 0;
  for (int j = p.n_outer - 1; j >= 0; --j) {
    const long long i = t % p.outer_size[j];
    t /= p.outer_size[j];
    offA += i * p.outer_sA[j]; offB += i * p.outer_sB[j]; offC += i * p.outer_sC[j];
  }
  const int m0 = mt * kTM, n0 = nt * kTN;
  const int M = (int)p.M, N = (int)p.N, K = (int)p.K;
  const int all = (K + kBK - 1) / kBK;
  const int s0 = (int)((long long)all * part / a.split), s1 = (int)((long long)all * (part + 1) / a.split);
  const float* const A = a.A + offA;
  const float* const B = a.B + offB;

  if (tid == 0) {
    mb_init(done, 1);
    abort_word = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(&tmem_slot)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;
  // the launch before this one on the stream may have written the operands; the next one may set itself up
  if (!a.late_wait) asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  const int row = (warp & 3) * 32 + lane, col = (warp >> 2) * 16;       // a row of the tile, 16 of its columns
  const uint32_t mine = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)col;
  bool ok = true;
  f32x2 sum2[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) sum2[j] = 0ull;
  auto add_up = [&](int s) {         // the blocks of stage s pairwise, then into the running sum
    ok = __all_sync(0xffffffffu, ok && mb_wait(done, (uint32_t)(s - s0) & 1u, 0xE01, abort_flag));
    if (!ok) return;
    fence_after();
    uint32_t x[16], y[16];
    if ((s + 1) * kBK <= K) {
      f32x2 h[8];
      tmem_ld16(mine, x);
      tmem_ld16(mine + 64u, y);
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < 8; ++j) h[j] = add2(pair_bits(x[2 * j], x[2 * j + 1]), pair_bits(y[2 * j], y[2 * j + 1]));
      tmem_ld16(mine + 128u, x);
      tmem_ld16(mine + 192u, y);
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < 8; ++j)
        sum2[j] = add2(sum2[j], add2(h[j], add2(pair_bits(x[2 * j], x[2 * j + 1]), pair_bits(y[2 * j], y[2 * j + 1]))));
    } else {                         // (the last stage: 1 to 4 blocks)
      const int steps = (K - s * kBK + 15) / 16;
#pragma unroll 1
      for (int k = 0; k < steps; ++k) {
        tmem_ld16(mine + 64u * (uint32_t)k, x);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 8; ++j) sum2[j] = add2(sum2[j], pair_bits(x[2 * j], x[2 * j + 1]));
      }
    }
    fence_before();
  };
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((kAlongA ? 0u : 1u) << 15) | ((kAlongB ? 0u : 1u) << 16) | ((uint32_t)(kTM >> 4) << 24);
  const uint32_t id64 = idesc | ((64u >> 3) << 17), id128 = idesc | ((128u >> 3) << 17);
  const uint32_t ka = kAlongA ? 32u : 2048u, kb = kAlongB ? 32u : 2048u;      // bytes of a 16-deep step
  auto issue = [&](int s, int u) {
    const uint32_t sa = base + (uint32_t)u * kStage, sb = sa + 3 * kPieceA;
    // (straight code: with a run-time trip count the thread needs 100 cycles to issue what the tensor core does in 56)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (s * kBK + 16 * k >= K) break;
      const uint64_t a0 = smem_desc(sa + k * ka, !kAlongA), b0 = smem_desc(sb + k * kb, !kAlongB);
      const uint64_t a1 = a0 + (kPieceA >> 4), a2 = a0 + (kPieceA >> 3), b1 = b0 + (kPieceB >> 4);
      umma(tmem + 64u * (uint32_t)k, a0, b0, id64, 0u);
      umma(tmem + 256u, a0, b1, id128, (s > s0 || k) ? 1u : 0u);        // a1 b2 | a1 b3
      umma(tmem + 256u, a1, b0, id128, 1u);                             // a2 b1 | a2 b2
      umma(tmem + 320u, a2, b0, id64, 1u);                              //         a3 b1
    }
    umma_commit(done);
  };
  Pieces<kTM, kAlongA> pa;
  Pieces<kTN, kAlongB> pb;
  pa.init(A, (int)p.sAm, (int)p.sAk, a.vecA, m0, M);
  pb.init(B, (int)p.sBn, (int)p.sBk, a.vecB, n0, N);
  float4 ra[2][Pieces<kTM, kAlongA>::kN], rb[2][Pieces<kTN, kAlongB>::kN];
  pa.load(s0, K, a.vecA, ra[0]);
  pb.load(s0, K, a.vecB, rb[0]);
  if (s0 + 1 < s1) { pa.load(s0 + 1, K, a.vecA, ra[1]); pb.load(s0 + 1, K, a.vecB, rb[1]); }
  // (a thread's values of B are the same four columns at every k.  Both operands along M and N, as in the weight gradients, has this code; a variant of its own
  // for the one launch that wants it cost that launch 1.7 us of instruction fetches, and in the other orders it cost the loop 1 %)
  constexpr bool kSumsB = !kAlongA && !kAlongB;
  const bool sums_b = kSumsB && a.bsum && mt == 0;
  float4 b_sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int s = s0; s < s1; s += 2) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int c = s + u;
      if (c >= s1) break;
      uint8_t* const sa = ring + (uint32_t)u * kStage;           // (free: the stage two back is complete, add_up waited for it)
      pa.template store<kPieceA>(sa, ra[u]);
      pb.template store<kPieceB>(sa + 3 * kPieceA, rb[u]);
      if (kSumsB && sums_b) {
        static_assert(Pieces<kTN, kAlongB>::kN % 2 == 0, "pairs");
#pragma unroll
        for (int i = 0; i < Pieces<kTN, kAlongB>::kN; i += 2) {
          const float4 p = rb[u][i], q = rb[u][i + 1];
          b_sum.x += p.x + q.x; b_sum.y += p.y + q.y; b_sum.z += p.z + q.z; b_sum.w += p.w + q.w;
        }
      }
      if (c + 2 < s1) { pa.load(c + 2, K, a.vecA, ra[u]); pb.load(c + 2, K, a.vecB, rb[u]); }
      if (c > s0) add_up(c - 1);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      if (warp == 0) {
        fence_after();
        if (mtf::elect_one()) issue(c, u);
        __syncwarp();
      }
    }
  }
  add_up(s1 - 1);
  if (ok) {                          // (the last stage's signal came behind every MMA)
    uint32_t x[16], y[16];
    tmem_ld16(mine + 256u, x);
    tmem_ld16(mine + 320u, y);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 8; ++j)
      sum2[j] = mul2(add2(sum2[j], add2(pair_bits(x[2 * j], x[2 * j + 1]), pair_bits(y[2 * j], y[2 * j + 1]))), pair(kDown, kDown));
  }
  // this block's part of the tile: 16-byte piece q of row r at r * 256 + ((q ^ (r mod 8)) * 16); every MMA has read the ring
  f32x2 odd2 = 0ull;                 // zero times every value: NaN if one is infinite or NaN
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float v[4];
    unpair(sum2[2 * q], v[0], v[1]);
    unpair(sum2[2 * q + 1], v[2], v[3]);
    odd2 = fma2(sum2[2 * q], 0ull, fma2(sum2[2 * q + 1], 0ull, odd2));
    *reinterpret_cast<float4*>(ring + row * 256 + (((col / 4 + q) ^ (row & 7)) << 4)) = make_float4(v[0], v[1], v[2], v[3]);
  }
  float odd_x, odd_y;
  unpair(odd2, odd_x, odd_y);
  if (__builtin_expect(__any_sync(0xffffffffu, ok && !(odd_x + odd_y == 0.f) && m0 + row < M && n0 + col < N), 0)) {      // (past the tile there is room for every warp's stage)
    const int m = m0 + row - lane, n = n0 + col;
    redo_plain(ring + row * 256, (uint32_t)(row & 7), (uint32_t)col / 4, reinterpret_cast<float*>(ring + 32768) + warp * kStageFloats, A + (long long)m * p.sAm,
               B + (long long)n * p.sBn, (int)p.sAm, (int)p.sAk, (int)p.sBn, (int)p.sBk, M - m, N - n, s0 * kBK, min(K, s1 * kBK));
  }
  fence_before();
  if (a.split > 1) cluster_sync();
  else __syncthreads();

  // the cluster's parts in ascending order, the component-wise stages, the store.  (One copy of this code: a launch runs it four times at
  // most, and fetching four copies cost it 0.6 us.)
  const int rows = kTM / a.split;                   // rows this block finishes: [part * rows, (part + 1) * rows)
  const int c4 = (tid & 15) * 4, n = n0 + c4, nv = min(4, N - n);
  float4 col_sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int i = tid >> 4; i < rows; i += kThreads / 16) {
    const int tr = part * rows + i, m = m0 + tr;
    if (m >= M || nv <= 0) continue;
    const uint32_t at = (uint32_t)tr * 256u + (((uint32_t)(tid & 15) ^ ((uint32_t)tr & 7u)) << 4);
    const float4 s = a.split == 1 ? *reinterpret_cast<const float4*>(ring + at) : a.split == 2 ? sum_parts<2>(base + at) : a.split == 4 ? sum_parts<4>(base + at) : sum_parts<8>(base + at);
    const long long off = offC + (long long)m * p.ldc + n;
    float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] *= a.scale;
    if (a.bias) {
      const float4 b = p.bias_along_m ? ld4_any(a.bias, a.bias_bf16, m, 1) : ld4_any(a.bias, a.bias_bf16, n, nv);
      const bool one = p.bias_along_m;
      v[0] += b.x; v[1] += one ? b.x : b.y; v[2] += one ? b.x : b.z; v[3] += one ? b.x : b.w;
    }
    if (a.relu) {
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = fmaxf(v[j], 0.f);
    }
    if (a.mask) {
      const float4 k = ld4_any(a.mask, a.mask_bf16, off, nv);
      v[0] = k.x > 0.f ? v[0] : 0.f; v[1] = k.y > 0.f ? v[1] : 0.f; v[2] = k.z > 0.f ? v[2] : 0.f; v[3] = k.w > 0.f ? v[3] : 0.f;
    }
    col_sum.x += v[0]; col_sum.y += v[1]; col_sum.z += v[2]; col_sum.w += v[3];      // (a column past N is not stored)
    if (a.resid) {
      const float4 r = ld4_any(a.resid, a.resid_bf16, off, nv);
      v[0] += r.x; v[1] += r.y; v[2] += r.z; v[3] += r.w;
    }
    if (a.c_bf16) {
      __nv_bfloat16* const c = reinterpret_cast<__nv_bfloat16*>(a.C) + off;
      if (nv == 4 && !(reinterpret_cast<uintptr_t>(c) & 7)) {
        *reinterpret_cast<uint2*>(c) = make_uint2(pack2(v[0], v[1]), pack2(v[2], v[3]));
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (j < nv) c[j] = __float2bfloat16_rn(v[j]);
      }
    } else {
      float* const c = reinterpret_cast<float*>(a.C) + off;
      if (nv == 4 && !(reinterpret_cast<uintptr_t>(c) & 15)) {
        *reinterpret_cast<float4*>(c) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (j < nv) c[j] = v[j];
      }
    }
  }
  // fused reduce_sum (over the rows of C), or the sums over k of B's columns: the 32 threads of a column piece, in a fixed order; the cluster's
  // parts in ascending order
  if (a.rsum || sums_b) {
    float* const to = sums_b ? a.bsum : a.rsum;
    const int mode = sums_b ? (a.split > 1 ? 2 : 1) : a.rsum_mode;
    const float4 mine4 = sums_b ? b_sum : col_sum;
    const uint32_t cs = base + 32768u;              // (past the tile: the rest of the cluster may still read it)
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(cs + (uint32_t)(tid >> 4) * 256u + (uint32_t)c4 * 4u), "f"(mine4.x), "f"(mine4.y), "f"(mine4.z),
                 "f"(mine4.w) : "memory");
    __syncthreads();
    float x = 0.f;
    if (tid < kTN) {
      float x4[4] = {0.f, 0.f, 0.f, 0.f};           // (four runs of eight: fewer roundings on the way)
#pragma unroll 8
      for (int i = 0; i < kThreads / 16; ++i) {
        float y;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(y) : "r"(cs + (uint32_t)i * 256u + (uint32_t)tid * 4u) : "memory");
        x4[i & 3] += y;
      }
      x = (x4[0] + x4[1]) + (x4[2] + x4[3]);
    }
    if (mode == 2) {
      if (tid < kTN) col_part[tid] = x;
      cluster_sync();
      if (part == 0 && tid < kTN && n0 + tid < N) {
        x = 0.f;
        for (int q = 0; q < a.split; ++q) {
          float y;
          asm volatile("{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %1, %2;\n\tld.shared::cluster.f32 %0, [ra];\n\t}"
                       : "=f"(y) : "r"(s_u32(&col_part[tid])), "r"(q) : "memory");
          x += y;
        }
        to[n0 + tid] = x;
      }
    } else if (tid < kTN && n0 + tid < N) {
      if (mode == 1) to[n0 + tid] = x;
      else atomicAdd(to + n0 + tid, x);
    }
  }
  __syncwarp();
  if (*abort_flag)
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);      // failure path: MMAs in flight land before the resources go away
  if (a.split > 1) cluster_sync();                  // the cluster may still read this block's part
  else __syncthreads();
  if (a.late_wait) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (warp == 0) {
    __syncwarp();
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

}  // namespace

namespace mtf {

static int64_t tiles_of(const F32Params& p) {
  int64_t tiles = ((p.M + kTM - 1) / kTM) * ((p.N + kTN - 1) / kTN);
  for (int j = 0; j < p.n_outer; ++j) tiles *= p.outer_size[j];
  return tiles;
}

// One block an SM; K is split over a cluster while that adds no wave and leaves every block a stage.
static int split_of(int64_t tiles, int64_t K) {
  int split = 1;
  const int64_t stages = (K + kBK - 1) / kBK;
  while (split < 8 && tiles * split * 2 <= (int64_t)device_sm_count() && stages >= 2 * split) split *= 2;
  return split;
}

// Is this kernel the shorter one for a product that einsum_f32.cu's tiles would take?  Microseconds, fitted to 900 drawn products on both
// (f32_tile_us is that kernel's estimate; a batch counts 0.2 more a round: its tiles are mostly padding when they are cheap; of the 900 none then takes over 1.03 times its time there).  It stays there for K up to about 32, where three pieces of a mostly empty stage are no gain (256 x 64 x 8: 3.9 us there,
// 4.7 here), and for batches of a few rows, where a 128-row tile is mostly padding (250 x [16 x 50 x 393]: 44 and 72).
bool f32_tensor_cores_pay(const F32Params& p) {
  const int64_t tiles = tiles_of(p);
  const int split = split_of(tiles, p.K);
  if (tiles * split > 0x7fffffffLL) return false;
  const int64_t part = ((p.K + kBK - 1) / kBK + split - 1) / split, sms = device_sm_count();
  const double rounds = (double)((tiles * split + sms - 1) / sms);
  return (split > 1 ? 0.5 : 0.0) + rounds * ((p.n_outer ? 4.0 : 3.8) + 1.5 * (double)part) < f32_tile_us(p);
}

bool f32_tc_sums_b(const F32Params& p, bool other_sums) { return !other_sums && !p.swapped && !p.n_outer && p.sAk != 1 && p.sBn == 1 && p.sBk != 1; }

template <bool kAlongA, bool kAlongB>
static mtf_status launch_orders(const F32TcArgs& a, int64_t blocks, cudaStream_t st) {
  // the opt-in to the shared memory is a property of a device
  constexpr int kMaxDevices = 64;
  static std::once_flag once[kMaxDevices];
  static cudaError_t attr[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return fail(MTF_ERR_CUDA, "cudaGetDevice");
  std::call_once(once[dev], [dev] { attr[dev] = cudaFuncSetAttribute(einsum_f32_tc_kernel<kAlongA, kAlongB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes); });
  if (attr[dev] != cudaSuccess) return fail(MTF_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(attr[dev]));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)a.split; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)blocks, 1, 1); cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes; cfg.stream = st; cfg.attrs = at; cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, einsum_f32_tc_kernel<kAlongA, kAlongB>, a);
  return e == cudaSuccess ? MTF_OK : fail(MTF_ERR_CUDA, "einsum_f32_tc_kernel: %s", cudaGetErrorString(e));
}

mtf_status launch_f32_tc(const F32Params& p, const void* A, const void* B, void* C, int dtC, const void* bias, int dtBias, const void* mask, int dtMask,
                         const void* resid, int dtRes, float scale, int relu, float* rsum, void* stream, bool late, float* bsum) {
  F32TcArgs a;
  a.p = p;
  if (p.swapped) std::swap(A, B);
  a.A = reinterpret_cast<const float*>(A); a.B = reinterpret_cast<const float*>(B);
  a.C = C; a.bias = bias; a.mask = mask; a.resid = resid; a.rsum = rsum;
  a.bsum = bsum; a.late_wait = late ? 1 : 0;
  if (bsum && !f32_tc_sums_b(p, rsum != nullptr)) return fail(MTF_ERR_UNSUPPORTED, "f32 product: column sums of B need operands contiguous along M and N, no batch and no other column sums");
  a.c_bf16 = dtC == MTF_BF16; a.bias_bf16 = dtBias == MTF_BF16; a.mask_bf16 = dtMask == MTF_BF16; a.resid_bf16 = dtRes == MTF_BF16;
  a.relu = relu; a.scale = scale;
  auto vec = [&](const void* base, int64_t s_mn, int64_t s_k, const int64_t* outer) {
    bool ok = !(reinterpret_cast<uintptr_t>(base) & 15) && (s_k == 1 ? s_mn % 4 == 0 : (s_mn == 1 && s_k % 4 == 0));
    for (int j = 0; j < p.n_outer; ++j) ok = ok && outer[j] % 4 == 0;
    return ok ? 1 : 0;
  };
  a.vecA = vec(A, p.sAm, p.sAk, p.outer_sA);
  a.vecB = vec(B, p.sBn, p.sBk, p.outer_sB);
  a.m_tiles = (int)((p.M + kTM - 1) / kTM);
  a.n_tiles = (int)((p.N + kTN - 1) / kTN);
  const int64_t tiles = tiles_of(p);
  a.split = split_of(tiles, p.K);
  if (tiles * a.split > 0x7fffffffLL) return fail(MTF_ERR_UNSUPPORTED, "output too large for the f32 kernel's grid");
  note_contraction(kTM, a.split);
  a.rsum_mode = tiles == a.n_tiles ? (a.split == 1 ? 1 : 2) : 0;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e;
  if (rsum && !a.rsum_mode && (e = cudaMemsetAsync(rsum, 0, (size_t)p.N * sizeof(float), st)) != cudaSuccess)
    return fail(MTF_ERR_CUDA, "cudaMemsetAsync: %s", cudaGetErrorString(e));
  const bool ka = p.sAk == 1, kb = p.sBk == 1;
  const mtf_status s = ka ? (kb ? launch_orders<true, true>(a, tiles * a.split, st) : launch_orders<true, false>(a, tiles * a.split, st))
                          : (kb ? launch_orders<false, true>(a, tiles * a.split, st) : launch_orders<false, false>(a, tiles * a.split, st));
  if (s != MTF_OK) return s;
  count_launch();
  return MTF_OK;
}

mtf_status read_f32_status(int* code) {
  int v = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_f32_status, sizeof(int));
  if (e != cudaSuccess) return fail(MTF_ERR_CUDA, "cudaMemcpyFromSymbol: %s", cudaGetErrorString(e));
  if (v) { int z = 0; cudaMemcpyToSymbol(g_f32_status, &z, sizeof(int)); }
  *code = v;
  return MTF_OK;
}

}  // namespace mtf
