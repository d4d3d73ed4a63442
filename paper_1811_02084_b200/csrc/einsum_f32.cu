// f32 einsums with the structure of a (batched) matrix product: C[o..][m][n] = sum_k A[o..][m][k] B[o..][k][n], each of
// M, N, K one merged strided dimension, up to three batch dimensions.  Plain FP32 arithmetic, for products of short K and
// batches of a few rows; the others run on the tensor cores in pieces (einsum_f32_tc.cu).  Component-wise
// stages of Section 6 / Section 7 run on the sum before the store, as in the generic kernel.
//
// Bound: the FP32 pipe at large sizes, launch and load latency at small ones.  A block of 256 threads owns a 64 x 64
// tile; its four groups of 64 threads take every fourth run of 8 of a 32-deep k-block, 8 x 8 outputs per thread (four
// 16-byte shared loads feed 32 packed multiply-adds).  Small tiles, so that few outputs still fill the chip, and where
// they do not, up to 8 blocks of a cluster share one tile's K and add their parts through distributed shared memory.
// The split of K over groups and blocks also shortens every chain of additions, so the sums are no less exact than one
// thread's sequential loop over K (all of K is walked in ascending order inside each part, parts are added in ascending
// order).  Two thirds of the instructions are not multiply-adds (the doubling of A's values, the staging): staging A doubled
// takes six shared loads a step instead of four and measured 210 us where this takes 149, plain multiply-adds 169.
// Measured against one thread per output element (the generic kernel), with every product of a block on this kernel: the feed-forward block
// forward and backward on 1024 tokens, 256 x 1024 hidden, 4804 -> 149 us (22 of 75 TFLOP/s); on 8 tokens, 64 x 256 hidden, 179 ->
// 33 us (six launches); its error against 64 bits there 5.3e-7 -> 2.0e-7.  Most of those products run in pieces now (70 and 28.9 us).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "mtf_internal.h"

namespace {

constexpr int kTile = 64;           // rows and columns of C per block
constexpr int kBK = 32;             // k-block
constexpr int kThreads = 256;
constexpr int kGroups = 4;          // groups of 64 threads, each with its own quarter of every k-block
constexpr int kBufFloats = 2 * kBK * kTile;                        // one stage: A and B tiles, [k][m|n]
constexpr int kSmemBytes = kGroups * kTile * kTile * 4;            // the groups' partial tiles; the two stages (32 KB) lie in the same bytes

struct F32Args {
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
  int c_bf16, bias_bf16, mask_bf16, resid_bf16, relu, rsum_store;
  float scale;
};

__device__ __forceinline__ float ld_any(const void* p, int bf16, long long off) {
  return bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[off]) : reinterpret_cast<const float*>(p)[off];
}

__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long twice(float x) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}

// Column c of row k of a staged tile lives at column c ^ 4 ((k / 4) mod 8): the exchange keeps 16-byte pieces whole and
// spreads the transposing stores of a K-contiguous operand over the banks.
__device__ __forceinline__ int swz(int k, int c) { return c ^ (((k >> 2) & 7) << 2); }
__device__ __forceinline__ int at(int k, int c) { return k * kTile + swz(k, c); }

// This thread's two 16-byte pieces of a 64 x 32 operand tile.  Along k (s_k == 1): piece f is row f / 8, k 4 (f mod 8);
// otherwise along m|n: piece f is k f / 16, column 4 (f mod 16).
struct Pieces {
  const float* base;
  int off[2];                  // element offset of the piece in the first k-block
  int step;                    // ... and what a k-block adds
  int s_mn, k_at[2], mn_left[2];      // first k of the piece inside a k-block, columns of it inside the tensor
  bool along_k, vec;
  __device__ __forceinline__ void init(const float* b, int smn, int sk, int v, int mn0, int mn_end) {
    base = b; s_mn = smn; along_k = sk == 1; vec = v != 0; step = kBK * sk;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int f = threadIdx.x + i * kThreads;
      const int mn = mn0 + (along_k ? f >> 3 : 4 * (f & 15));
      k_at[i] = along_k ? 4 * (f & 7) : f >> 4;
      mn_left[i] = mn_end - mn;
      off[i] = mn * smn + k_at[i] * sk;
    }
  }
  __device__ __forceinline__ void load(int kb, int K, float4* r) const {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      r[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      const int left = K - (kb * kBK + k_at[i]);
      if (left <= 0 || mn_left[i] <= 0) continue;
      const float* const q = base + (off[i] + kb * step);
      const int in = along_k ? left : mn_left[i], s = along_k ? 1 : s_mn;
      if (vec && in >= 4) { r[i] = __ldg(reinterpret_cast<const float4*>(q)); continue; }
      r[i].x = __ldg(q);
      if (in > 1) r[i].y = __ldg(q + s);
      if (in > 2) r[i].z = __ldg(q + 2 * s);
      if (in > 3) r[i].w = __ldg(q + 3 * s);
    }
  }
  __device__ __forceinline__ void store(float* tile, const float4* r) const {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int f = threadIdx.x + i * kThreads;
      if (along_k) {
        const int mn = f >> 3, k = 4 * (f & 7);
        tile[at(k, mn)] = r[i].x; tile[at(k + 1, mn)] = r[i].y; tile[at(k + 2, mn)] = r[i].z; tile[at(k + 3, mn)] = r[i].w;
      } else {
        *reinterpret_cast<float4*>(tile + at(f >> 4, 4 * (f & 15))) = r[i];
      }
    }
  }
};

__device__ __forceinline__ float4 ld_peer(uint32_t addr, uint32_t rank) {
  float4 v;
  asm volatile(
      "{\n\t.reg .b32 ra;\n\t"
      "mapa.shared::cluster.u32 ra, %4, %5;\n\t"
      "ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [ra];\n\t}"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr), "r"(rank) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();                      // (the aligned barrier takes whole warps; lanes leave the loops before it one by one)
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __launch_bounds__(kThreads, 2) einsum_f32_kernel(const __grid_constant__ F32Args a) {
  extern __shared__ __align__(16) float smem[];
  __shared__ float col_part[4][kTile];
  const F32Params& p = a.p;
  const int tid = threadIdx.x;
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
  const int m0 = mt * kTile, n0 = nt * kTile;
  const int M = (int)p.M, N = (int)p.N, K = (int)p.K;
  const int kb_all = (K + kBK - 1) / kBK;
  const int kb0 = (int)((long long)kb_all * part / a.split), kb1 = (int)((long long)kb_all * (part + 1) / a.split);
  const bool alongA = p.sAk == 1, alongB = p.sBk == 1;
  const float* const A = a.A + offA;
  const float* const B = a.B + offB;
  // the launch before this one on the stream may have written the operands; the next one may set itself up
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  const int g = tid >> 6, tx = tid & 7, ty = (tid >> 3) & 7;
  unsigned long long acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  Pieces pa, pb;
  pa.init(A, (int)p.sAm, (int)p.sAk, a.vecA, m0, M);
  pb.init(B, (int)p.sBn, (int)p.sBk, a.vecB, n0, N);
  float4 ra[2], rb[2];
  if (kb0 < kb1) {
    pa.load(kb0, K, ra);
    pb.load(kb0, K, rb);
    pa.store(smem, ra);
    pb.store(smem + kBK * kTile, rb);
  }
  __syncthreads();
#pragma unroll 1
  for (int kb = kb0; kb < kb1; ++kb) {
    const float* const sa = smem + ((kb - kb0) & 1) * kBufFloats;
    const float* const sb = sa + kBK * kTile;
    const bool more = kb + 1 < kb1;
    if (more) {
      pa.load(kb + 1, K, ra);
      pb.load(kb + 1, K, rb);
    }
#pragma unroll 1
    for (int k4 = 0; k4 < kBK / kGroups; k4 += 4) {
      const int k0 = g * (kBK / kGroups) + k4;
      const float* const ka = sa + at(k0, 4 * ty);                 // (columns 32 further on lie 32 floats on, the next k 64 floats on)
      const float* const kbp = sb + at(k0, 4 * tx);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const float4 a0 = *reinterpret_cast<const float4*>(ka + kk * kTile), a1 = *reinterpret_cast<const float4*>(ka + kk * kTile + 32);
        const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(kbp + kk * kTile), b1 = *reinterpret_cast<const ulonglong2*>(kbp + kk * kTile + 32);
        const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const unsigned long long d = twice(av[i]);
          fma2(acc[i][0], d, b0.x); fma2(acc[i][1], d, b0.y); fma2(acc[i][2], d, b1.x); fma2(acc[i][3], d, b1.y);
        }
      }
    }
    if (more) {                                     // (the other stage: its last readers passed the barrier at the end of the round before)
      float* const nsa = smem + ((kb + 1 - kb0) & 1) * kBufFloats;
      pa.store(nsa, ra);
      pb.store(nsa + kBK * kTile, rb);
    }
    __syncthreads();
  }

  // the four groups' parts, then (split > 1) the cluster's, in ascending order
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float* const row = smem + g * kTile * kTile + ((i < 4 ? 4 * ty + i : 28 + 4 * ty + i)) * kTile;
    *reinterpret_cast<ulonglong2*>(row + 4 * tx) = make_ulonglong2(acc[i][0], acc[i][1]);
    *reinterpret_cast<ulonglong2*>(row + 32 + 4 * tx) = make_ulonglong2(acc[i][2], acc[i][3]);
  }
  __syncthreads();
  const int rows = kTile / a.split;                 // rows this block finishes: [part * rows, (part + 1) * rows)
  auto local_sum = [&](int e) {                     // piece e of the tile, summed over the groups
    float4 s = *reinterpret_cast<const float4*>(smem + 4 * e);
#pragma unroll
    for (int q = 1; q < kGroups; ++q) {
      const float4 x = *reinterpret_cast<const float4*>(smem + q * kTile * kTile + 4 * e);
      s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
    }
    return s;
  };
  if (a.split > 1) {
    for (int e = tid; e < kTile * kTile / 4; e += kThreads) {
      const float4 s = local_sum(e);
      *reinterpret_cast<float4*>(smem + 4 * e) = s;
    }
    cluster_sync();
  }
  const uint32_t smem_addr = (uint32_t)__cvta_generic_to_shared(smem);
  const int c4 = (tid & 15) * 4;
  float4 col_sum = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int r = tid >> 4; r < rows; r += kThreads / 16) {
    const int row = part * rows + r, e = row * (kTile / 4) + (tid & 15);
    float4 s;
    if (a.split > 1) {
      s = ld_peer(smem_addr + 16u * (uint32_t)e, 0u);
      for (int q = 1; q < a.split; ++q) {
        const float4 x = ld_peer(smem_addr + 16u * (uint32_t)e, (uint32_t)q);
        s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
      }
    } else {
      s = local_sum(e);
    }
    const int m = m0 + row, n = n0 + c4;
    if (m >= M || n >= N) continue;
    float v[4] = {s.x, s.y, s.z, s.w};
    const long long off = offC + (long long)m * p.ldc + n;
    const int nv = N - n < 4 ? N - n : 4;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (j >= nv) { v[j] = 0.f; continue; }
      float x = v[j] * a.scale;
      if (a.bias) x += ld_any(a.bias, a.bias_bf16, p.bias_along_m ? m : n + j);
      if (a.relu) x = fmaxf(x, 0.f);
      if (a.mask && !(ld_any(a.mask, a.mask_bf16, off + j) > 0.f)) x = 0.f;
      v[j] = x;
    }
    col_sum.x += v[0]; col_sum.y += v[1]; col_sum.z += v[2]; col_sum.w += v[3];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < nv && a.resid) v[j] += ld_any(a.resid, a.resid_bf16, off + j);
    if (a.c_bf16) {
      __nv_bfloat16* const c = reinterpret_cast<__nv_bfloat16*>(a.C) + off;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j < nv) c[j] = __float2bfloat16_rn(v[j]);
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
  if (a.rsum) {                                     // fused reduce_sum: 16 threads of a column piece, in a fixed order
    __syncthreads();
    float* const cs = smem + kTile * kTile;         // (the groups' parts 1 .. 3 have been read; part 0 may still be read by the cluster)
    *reinterpret_cast<float4*>(cs + (tid >> 4) * kTile + c4) = col_sum;
    __syncthreads();
    const int c = tid & 63, q = tid >> 6;
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) s += cs[(q * 4 + i) * kTile + c];
    col_part[q][c] = s;
    __syncthreads();
    if (tid < kTile && n0 + tid < N) {
      const float x = (col_part[0][tid] + col_part[1][tid]) + (col_part[2][tid] + col_part[3][tid]);
      if (a.rsum_store) a.rsum[n0 + tid] = x;
      else atomicAdd(a.rsum + n0 + tid, x);
    }
  }
  if (a.split > 1) cluster_sync();                  // the cluster may still read this block's part
}

}  // namespace

namespace mtf {

static int64_t tiles_of(const F32Params& p) {
  int64_t tiles = ((p.M + kTile - 1) / kTile) * ((p.N + kTile - 1) / kTile);
  for (int j = 0; j < p.n_outer; ++j) tiles *= p.outer_size[j];
  return tiles;
}

// Two blocks fit an SM.  K is split over a cluster while that does not add a wave and leaves every block at least
// two k-blocks (one to load while the other is worked on).
static int split_of(int64_t tiles, int64_t K) {
  int split = 1;
  const int64_t kb = (K + kBK - 1) / kBK;
  while (split < 8 && tiles * split * 2 <= 2 * (int64_t)device_sm_count() && kb >= 4 * split) split *= 2;
  return split;
}

// Is this kernel the shorter one?  A tile costs the same however few of its 64 x 64 outputs exist, so batches of small
// products, single rows or columns and short K stay with one thread per output: 100000 products of 1 x 1 take 3.4 us there
// and 1469 here, 4096 of 4 x 4 x 4 3.6 and 62, 1000000 x 1 x 1 14 and 260; 8 x 256 x 64 takes 23 and 5.  Microseconds, fitted to
// 4400 drawn products on both: there a start, and the chain of K loads (the first ones cold) or the outputs and multiply-adds
// of a full chip, whichever is longer; here the k-blocks of one block on an SM, or rounds of two.  29 drawn products take more
// than 1.05 times their time on the generic kernel, 1.1 us at most, which this kernel's early set-up behind the launch before
// it makes up (the 8-token block: 31 us so, 36 with its two 8-deep products there); on average they are 0.5 % from the better.
double f32_tile_us(const F32Params& p) {
  const int64_t tiles = tiles_of(p), sms = device_sm_count();
  const int split = split_of(tiles, p.K);
  const int64_t kb = ((p.K + kBK - 1) / kBK + split - 1) / split;
  const double rounds = (double)((tiles * split + 2 * sms - 1) / (2 * sms));
  return (split > 1 ? 1.0 : 0.0) + (tiles * split <= sms ? 2.2 + 1.6 * (double)kb : 0.5 + rounds * (2.2 + 2.1 * (double)kb));
}
bool f32_tiles_pay(const F32Params& p) {
  const int64_t tiles = tiles_of(p);
  if (tiles * split_of(tiles, p.K) > 0x7fffffffLL) return false;
  double outputs = (double)p.M * (double)p.N;
  for (int j = 0; j < p.n_outer; ++j) outputs *= (double)p.outer_size[j];
  const double there = 2.0 + std::max(0.15 * (double)p.K + 0.12 * (double)std::min<int64_t>(p.K, 16), outputs / 130e3 + outputs * (double)p.K / 600e3);
  return f32_tile_us(p) < there;
}

mtf_status launch_f32(const F32Params& p, const void* A, const void* B, void* C, int dtC, const void* bias, int dtBias, const void* mask, int dtMask,
                      const void* resid, int dtRes, float scale, int relu, float* rsum, void* stream) {
  F32Args a;
  a.p = p;
  if (p.swapped) std::swap(A, B);
  a.A = reinterpret_cast<const float*>(A); a.B = reinterpret_cast<const float*>(B);
  a.C = C; a.bias = bias; a.mask = mask; a.resid = resid; a.rsum = rsum;
  a.c_bf16 = dtC == MTF_BF16; a.bias_bf16 = dtBias == MTF_BF16; a.mask_bf16 = dtMask == MTF_BF16; a.resid_bf16 = dtRes == MTF_BF16;
  a.relu = relu; a.scale = scale;
  auto vec = [&](const void* base, int64_t s_mn, int64_t s_k, const int64_t* outer) {
    bool ok = !(reinterpret_cast<uintptr_t>(base) & 15) && (s_k == 1 ? s_mn % 4 == 0 : (s_mn == 1 && s_k % 4 == 0));
    for (int j = 0; j < p.n_outer; ++j) ok = ok && outer[j] % 4 == 0;
    return ok ? 1 : 0;
  };
  a.vecA = vec(A, p.sAm, p.sAk, p.outer_sA);
  a.vecB = vec(B, p.sBn, p.sBk, p.outer_sB);
  a.m_tiles = (int)((p.M + kTile - 1) / kTile);
  a.n_tiles = (int)((p.N + kTile - 1) / kTile);
  const int64_t tiles = tiles_of(p);
  a.split = split_of(tiles, p.K);
  if (tiles * a.split > 0x7fffffffLL) return fail(MTF_ERR_UNSUPPORTED, "output too large for the f32 kernel's grid");
  note_contraction(kTile, a.split);
  a.rsum_store = rsum && tiles == a.n_tiles && a.split == 1;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e;
  if (rsum && !a.rsum_store && (e = cudaMemsetAsync(rsum, 0, (size_t)p.N * sizeof(float), st)) != cudaSuccess)
    return fail(MTF_ERR_CUDA, "cudaMemsetAsync: %s", cudaGetErrorString(e));
  // the opt-in to 64 KB of shared memory is a property of a device
  constexpr int kMaxDevices = 64;
  static std::once_flag once[kMaxDevices];
  static cudaError_t attr[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return fail(MTF_ERR_CUDA, "cudaGetDevice");
  std::call_once(once[dev], [dev] { attr[dev] = cudaFuncSetAttribute(einsum_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes); });
  if (attr[dev] != cudaSuccess) return fail(MTF_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(attr[dev]));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)a.split; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(tiles * a.split), 1, 1); cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes; cfg.stream = st; cfg.attrs = at; cfg.numAttrs = 2;
  if ((e = cudaLaunchKernelEx(&cfg, einsum_f32_kernel, a)) != cudaSuccess) return fail(MTF_ERR_CUDA, "einsum_f32_kernel: %s", cudaGetErrorString(e));
  count_launch();
  return MTF_OK;
}

}  // namespace mtf
