// The f32 feed-forward block on a few tokens, one launch forward and one backward instead of two and four:
//   forward    h = relu(x.w + bias),  y = h.v
//   backward   dhp = (dy.v^T) * [h > 0],  dbias = sum_tokens dhp,  dx = dhp.w^T,  dv = h^T.dy,  dw = x^T.dhp
// A cluster of eight blocks, each the owner of an eighth of the hidden units (the paper's split of d_ff over processors, Section
// 8.2): everything a block needs of w and v is its own, h, dhp, dw, dv and dbias of its hidden units need no other block, and the one sum over all of
// them (y, dx) is the Allreduce, taken through distributed shared memory in block order.
//
// All operands are copied to shared memory at once (4-byte asynchronous copies: any alignment, one wait).  Products run from there: a thread
// owns four rows by two columns, sums four terms in f32 and the fours in f64, K over several threads where outputs are few; their parts and the blocks'
// parts are added in f64 too, and every result is rounded once, so that no sum is less exact than one on the matrix kernels.  2-norm errors against 64 bits
// in 1e-8, launch by launch | in eights | in fours:
//   8 tokens, 64 x 256    h 5.6 | 6.0 | 4.8   y 8.2 | 7.8 | 6.4   dx 7.7 | 7.7 | 6.2   dw 6.6 | 7.3 | 6.4   dv 7.0 | 7.3 | 6.4
//   64 tokens, 40 x 72    h 5.1 | 5.9 | 4.7   y 7.0 | 7.6 | 6.2   dx 6.6 | 7.7 | 6.3   dw 6.2 | 7.7 | 6.3   dv 6.6 | 7.7 | 6.2
//
// Bound: latency (launch, one round of loads, two barriers of the cluster) and, towards the limits below, the copies and the shared-memory reads of eight
// SMs.  The block at 8 tokens, 64 x 256, forward and backward: 28.5 -> 15.3 us (launch by launch six dependent launches of 4 - 5 us; sums of eight
// terms in f32 instead of four 15.1).
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "launch.cuh"
#include "mtf_internal.h"

namespace {

constexpr int kBlocks = 8, kThreads = 512;
constexpr int kRed = 8 * kThreads;                // f64 parts of sums that several threads share
constexpr size_t kMaxSmem = 200 * 1024;

struct SmallArgs {
  int T, D, F, E;                                 // tokens, width in, hidden units, width out
  const float *x, *w, *bias, *v, *h, *dy;
  float *h_out, *y, *dx, *dw, *dbias, *dv, *dhp;  // (dhp: NULL unless asked for)
};

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__host__ __device__ __forceinline__ int odd(int n) { return n | 1; }             // row stride of w and v: neither a row nor a column of them meets a bank twice
__host__ __device__ __forceinline__ int up4(int n) { return (n + 3) & ~3; }      // row stride and rows of the others

// rows x cols at src (row stride ss) -> dst (row stride ds)
__device__ __forceinline__ void stage(float* dst, int ds, const float* src, int ss, int rows, int cols) {
  if (cols <= 0) return;
  const int step_r = kThreads / cols, step_c = kThreads % cols;
  int r = (int)threadIdx.x / cols, c = (int)threadIdx.x % cols;
  while (r < rows) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s_u32(dst + r * ds + c)), "l"(src + (long long)r * ss + c) : "memory");
    r += step_r; c += step_c;
    if (c >= cols) { c -= cols; ++r; }
  }
}
__device__ __forceinline__ void stage_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
}

// out(m, n, sum_k A(m, k) B[k sBk + n sBn]), operands in shared memory; the whole block calls it.  A(m, k) is A[m lda + k] (kAlongK) or
// A[k lda + m], with lda a multiple of four and rows (columns) up to the next multiple of four there, whatever they hold.
template <bool kAlongK, typename Out>
__device__ __forceinline__ void product(int M, int N, int K, const float* A, int lda, const float* B, int sBk, int sBn, double* red, Out out) {
  const int nh = (N + 1) / 2, tasks = (M + 3) / 4 * nh;
  if (tasks == 0) return;
  int parts = 1;
  while (2 * parts * tasks <= kThreads && K >= 16 * parts) parts *= 2;
  const int len = ((K + parts - 1) / parts + 3) / 4 * 4;
  const int part = parts > 1 ? (int)threadIdx.x / tasks : 0;
  for (int task = (int)threadIdx.x - part * tasks; task < tasks && part < parts; task += kThreads) {
    const int m0 = task / nh * 4, n0 = task % nh, n1 = n0 + nh;
    int k = part * len;
    const int k1 = min(K, k + len);
    const float* a = kAlongK ? A + m0 * lda + k : A + k * lda + m0;
    const float* b0 = B + n0 * sBn + k * sBk;
    const float* b1 = B + min(n1, N - 1) * sBn + k * sBk;
    double acc[4][2] = {};
#pragma unroll 1                                  // (short code: it is fetched cold; unrolled twice 4 % of the launch)
    for (; k < k1; k += 4) {
      float s[4][2] = {};
      if (k + 4 <= k1) {                         // four 16-byte reads of A, which every lane of a row shares
        float f[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 q = *reinterpret_cast<const float4*>(a + i * lda);
          const float r[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
          for (int t = 0; t < 4; ++t) (kAlongK ? f[i][t] : f[t][i]) = r[t];      // f[row][k]
        }
        a += kAlongK ? 4 : 4 * lda;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const float p = *b0, q = *b1;
          b0 += sBk; b1 += sBk;
#pragma unroll
          for (int i = 0; i < 4; ++i) { s[i][0] = fmaf(f[i][t], p, s[i][0]); s[i][1] = fmaf(f[i][t], q, s[i][1]); }
        }
      } else {
#pragma unroll 1
        for (int t = k; t < k1; ++t) {
          const float p = *b0, q = *b1;
          b0 += sBk; b1 += sBk;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float f = kAlongK ? a[i * lda] : a[i];
            s[i][0] = fmaf(f, p, s[i][0]);
            s[i][1] = fmaf(f, q, s[i][1]);
          }
          a += kAlongK ? 1 : lda;
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) { acc[i][0] += (double)s[i][0]; acc[i][1] += (double)s[i][1]; }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (parts > 1) {
        red[(part * 8 + 2 * i) * tasks + task] = acc[i][0];
        red[(part * 8 + 2 * i + 1) * tasks + task] = acc[i][1];
      } else if (m0 + i < M) {
        out(m0 + i, n0, acc[i][0]);
        if (n1 < N) out(m0 + i, n1, acc[i][1]);
      }
    }
  }
  if (parts == 1) return;
  __syncthreads();
  for (int i = (int)threadIdx.x; i < 8 * tasks; i += kThreads) {
    const int j = i / tasks, task = i - j * tasks, m = task / nh * 4 + j / 2, n = task % nh + (j & 1) * nh;
    if (m >= M || n >= N) continue;
    double s = 0.0, s1 = 0.0;                     // (parts is a power of two above one: two chains)
#pragma unroll 1                                  // (as above: 1 %)
    for (int q = 0; q < parts; q += 2) { s += red[q * 8 * tasks + i]; s1 += red[(q + 1) * 8 * tasks + i]; }
    out(m, n, s + s1);
  }
  __syncthreads();                                // (the next product may use `red`)
}

// (aligned barriers take whole warps; a product in one part ends in a loop that lanes leave at different turns, and nothing else brings them together)
__device__ __forceinline__ void cluster_arrive() { __syncwarp(); asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { __syncwarp(); asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// out[i] = the sum over the cluster's blocks of part[i], each block an eighth of the elements
__device__ __forceinline__ void add_blocks(const double* part, int n, int rank, float* out) {
  const uint32_t base = s_u32(part);
  for (int i = rank * kThreads + (int)threadIdx.x; i < n; i += kBlocks * kThreads) {
    double x[kBlocks];
#pragma unroll
    for (int q = 0; q < kBlocks; ++q)
      asm volatile("{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %1, %2;\n\tld.shared::cluster.f64 %0, [ra];\n\t}" : "=d"(x[q]) : "r"(base + 8u * (uint32_t)i), "r"(q) : "memory");
#pragma unroll
    for (int q = 1; q < kBlocks; ++q) x[0] += x[q];
    out[i] = (float)x[0];
  }
}

// f64 first: parts of sums and this block's part of y (dx); then the tiles
struct Carve {
  uint8_t* p;
  __device__ double* f64(int n) { double* r = reinterpret_cast<double*>(p); p += (size_t)n * 8; return r; }
  __device__ float* f32(int n) { float* r = reinterpret_cast<float*>(p); p += (size_t)n * 4; return r; }
};

__global__ void __cluster_dims__(kBlocks, 1, 1) __launch_bounds__(kThreads, 1) ffn_small_forward_kernel(const SmallArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int per = (a.F + kBlocks - 1) / kBlocks, rank = (int)blockIdx.x, f0 = min(rank * per, a.F), n = min(per, a.F - f0);
  const int rows = up4(a.T), ld = up4(a.D), lf = up4(per), sw = odd(per), sv = odd(a.E);
  Carve c{smem};
  double* const red = c.f64(kRed);
  double* const part = c.f64(up4(a.T * a.E));
  float *const x = c.f32(rows * ld), *const h = c.f32(rows * lf), *const w = c.f32(a.D * sw), *const v = c.f32(per * sv), *const bias = c.f32(per);
  mtf::chain_wait();
  stage(x, ld, a.x, a.D, a.T, a.D);
  stage(w, sw, a.w + f0, a.F, a.D, n);
  if (a.bias) stage(bias, per, a.bias + f0, per, 1, n);
  stage(v, sv, a.v + (long long)f0 * a.E, a.E, n, a.E);
  stage_wait();
  product<true>(a.T, n, a.D, x, ld, w, sw, 1, red, [&](int t, int f, double s) {
    const float r = fmaxf((float)(a.bias ? s + (double)bias[f] : s), 0.f);
    h[t * lf + f] = r;
    a.h_out[(long long)t * a.F + f0 + f] = r;
  });
  __syncthreads();
  product<true>(a.T, a.E, n, h, lf, v, sv, 1, red, [&](int t, int e, double s) { part[t * a.E + e] = s; });
  cluster_arrive();
  cluster_wait();
  add_blocks(part, a.T * a.E, rank, a.y);
  cluster_arrive();                               // (the cluster may still read this block's part)
  cluster_wait();
}

__global__ void __cluster_dims__(kBlocks, 1, 1) __launch_bounds__(kThreads, 1) ffn_small_backward_kernel(const SmallArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int per = (a.F + kBlocks - 1) / kBlocks, rank = (int)blockIdx.x, f0 = min(rank * per, a.F), n = min(per, a.F - f0);
  const int rows = up4(a.T), ld = up4(a.D), lf = up4(per), le = up4(a.E), sw = odd(per), sv = odd(a.E);
  Carve c{smem};
  double* const red = c.f64(kRed);
  double* const part = c.f64(up4(a.T * a.D));
  float *const x = c.f32(rows * ld), *const h = c.f32(rows * lf), *const dy = c.f32(rows * le), *const dhp = c.f32(rows * lf), *const w = c.f32(a.D * sw), *const v = c.f32(per * sv);
  mtf::chain_wait();
  stage(dy, le, a.dy, a.E, a.T, a.E);
  stage(v, sv, a.v + (long long)f0 * a.E, a.E, n, a.E);
  stage(h, lf, a.h + f0, a.F, a.T, n);
  stage(w, sw, a.w + f0, a.F, a.D, n);
  stage(x, ld, a.x, a.D, a.T, a.D);
  stage_wait();
  product<true>(a.T, n, a.E, dy, le, v, 1, sv, red, [&](int t, int f, double s) {
    const float r = h[t * lf + f] > 0.f ? (float)s : 0.f;
    dhp[t * lf + f] = r;
    if (a.dhp) a.dhp[(long long)t * a.F + f0 + f] = r;
  });
  __syncthreads();
  product<true>(a.T, a.D, n, dhp, lf, w, 1, sw, red, [&](int t, int d, double s) { part[t * a.D + d] = s; });
  cluster_arrive();                               // (the results that are this block's alone while the others get there)
  product<false>(n, a.E, a.T, h, lf, dy, le, 1, red, [&](int f, int e, double s) { a.dv[(long long)(f0 + f) * a.E + e] = (float)s; });
  product<false>(a.D, n, a.T, x, ld, dhp, lf, 1, red, [&](int d, int f, double s) { a.dw[(long long)d * a.F + f0 + f] = (float)s; });
  if (a.dbias)
    for (int f = (int)threadIdx.x; f < n; f += kThreads) {
      double s = 0.0;
      for (int t = 0; t < a.T; ++t) s += (double)dhp[t * lf + f];
      a.dbias[f0 + f] = (float)s;
    }
  cluster_wait();
  add_blocks(part, a.T * a.D, rank, a.dx);
  cluster_arrive();
  cluster_wait();
}

size_t smem_bytes(int64_t T, int64_t D, int64_t F, int64_t E, bool backward) {
  const int64_t per = (F + kBlocks - 1) / kBlocks, rows = up4((int)T), ld = up4((int)D), lf = up4((int)per), le = up4((int)E);
  const int64_t tiles = rows * (ld + lf + (backward ? le + lf : 0)) + D * odd((int)per) + per * odd((int)E) + (backward ? 0 : per);
  return (size_t)(8 * (kRed + up4((int)(T * (backward ? D : E)))) + 4 * tiles);
}

mtf_status launch(void (*kernel)(SmallArgs), std::once_flag* once, cudaError_t* attr, size_t smem, const SmallArgs& a, void* stream) {
  constexpr int kMaxDevices = 64;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return mtf::fail(MTF_ERR_CUDA, "cudaGetDevice");
  std::call_once(once[dev], [&] { attr[dev] = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem); });
  if (attr[dev] != cudaSuccess) return mtf::fail(MTF_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(attr[dev]));
  mtf::launch_chained(kernel, kBlocks, kThreads, smem, (cudaStream_t)stream, a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return mtf::fail(MTF_ERR_CUDA, "f32 feed-forward block on a few tokens: %s", cudaGetErrorString(e));
  mtf::count_launch();
  return MTF_OK;
}

}  // namespace

namespace mtf {

// Whether a direction runs here, or as one launch per einsum: forward up to 3 x 2^17 multiply-adds a product; backward up to 2^20, where the products over at most 32 tokens
// are no work for the tensor cores, else as many as forward; fewer where much of w and v has to be copied.  us, here and launch by launch (graphs of ten passes):
//   tokens x width x hidden   8 x 64 x 256  16 x 64 x 512  4 x 128 x 512  64 x 40 x 72  128 x 40 x 72  48 x 64 x 256  16 x 128 x 512  8 x 128 x 1024  1 x 48 x 2048
//   forward                     6.6   9.2      9.1   9.4      8.8   9.8     6.9   9.7     9.6  10.2     9.9   9.9      13.0  10.2     14.1  11.4       9.7  14.1
//   backward                    8.6  17.0     12.6  17.6     12.0  19.4    10.7  14.3    14.5  15.1    16.9  14.4      18.9  18.8     22.1  20.1      14.7  21.5
// The forward limit of 65536 weights is a cautious one: with up to 8 tokens the launch is the shorter one up to 131072 (2 x 40 x 3000 11.4 and 17.3, 4 x 48 x 2048
// 9.9 and 13.9, 8 x 48 x 2048 12.5 and 14.2), which runs launch by launch.
bool ffn_small_pays(int64_t T, int64_t D, int64_t F, int64_t E, bool backward) {
  if (T <= 0 || D <= 0 || F <= 0 || E <= 0 || T > 4096 || D > 8192 || F > 65536 || E > 8192) return false;
  const int64_t weights = F * std::max(D, E), work = T * weights;
  const int64_t most = !backward || T > 32 ? 3 << 17 : weights > 65536 ? 1 << 19 : 1 << 20;
  if (work > most || weights > (backward ? 131072 : 65536)) return false;
  return smem_bytes(T, D, F, E, backward) <= kMaxSmem;
}

mtf_status launch_ffn_small_forward(int64_t T, int64_t D, int64_t F, int64_t E, const float* x, const float* w, const float* bias, const float* v, float* h, float* y,
                                    void* stream) {
  static std::once_flag once[64];
  static cudaError_t attr[64];
  SmallArgs a = {(int)T, (int)D, (int)F, (int)E, x, w, bias, v, nullptr, nullptr, h, y, nullptr, nullptr, nullptr, nullptr, nullptr};
  return launch(ffn_small_forward_kernel, once, attr, smem_bytes(T, D, F, E, false), a, stream);
}

mtf_status launch_ffn_small_backward(int64_t T, int64_t D, int64_t F, int64_t E, const float* x, const float* w, const float* v, const float* h, const float* dy,
                                     float* dx, float* dw, float* dbias, float* dv, float* dhp, void* stream) {
  static std::once_flag once[64];
  static cudaError_t attr[64];
  SmallArgs a = {(int)T, (int)D, (int)F, (int)E, x, w, nullptr, v, h, dy, nullptr, nullptr, dx, dw, dbias, dv, dhp};
  return launch(ffn_small_backward_kernel, once, attr, smem_bytes(T, D, F, E, true), a, stream);
}

}  // namespace mtf
