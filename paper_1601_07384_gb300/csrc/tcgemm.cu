// Dense products of the learned preconditioner's layers on the tensor cores (tcgen05, kind::f16):
//   D(m, n) = Sum_k A(m, k) B(n, k) + bias(n) (+ Sum_k A2(m, k) B2(n, k))
// with the operands rounded to bfloat16, each product accumulated in binary32, followed by ReLU with the
// pre-activation kept.  One CTA (8 warps) owns a tile of 128 rows of D and all N <= 256
// columns; its accumulator lives in tensor memory (128 lanes x N columns).  One thread issues the MMAs
// (M = 128, K = 16 each) of every 64-wide slice of K and commits them to the mbarrier of the slice's
// buffer; after the last slice every warp reads its 32 lanes of the accumulator.  A second grid
// dimension splits K into ranges written to separate output slices (weight gradients: partial sums
// over chunks of tets, reduced afterwards in a fixed order).
//
// What bounds it: the operands are binary32 (activations) with arbitrary leading dimensions, so they
// are converted on the way into shared memory, and at these sizes (K <= 180, a few dozen CTAs) the time
// is the latency of that staging, not the tensor pipe.  So a thread stages 8 consecutive k of one row at
// a time: two 16-byte loads where the rows are 16-byte aligned (8 strided ones, coalesced over the
// lanes' consecutive rows, for an operand that is contiguous along its rows), all loads of a slice in
// flight before the first conversion, one 16-byte store into the K-major core-matrix layout; and a slice
// is staged while the tensor cores work on the slice before it (two buffers).  6,000 x 64 x 64 in the
// network: 6-9 us per product, against 65 us with element-wise staging, one buffer and 128 threads.
#include <cuda_bf16.h>

#include "solver.h"
#include "tc_ptx.cuh"

namespace stdg {


constexpr int kTcRows = 128;                 // M of one MMA and of the CTA tile
constexpr int kTcKC = 64;                    // K slice staged at a time (4 MMAs of K = 16)
constexpr int kTcThreads = 256;
constexpr long kTcSpin = 4000;               // bounded waits (each try suspends up to 1 ms)

// byte offset of element (r, k) of a K-major tile with kTcKC columns: core matrix (r / 8, k / 8) at
// ((r / 8) (kTcKC / 8) + k / 8) 128, row r % 8 at 16 (r % 8), element k % 8 at 2 (k % 8)
__device__ __forceinline__ uint32_t tc_off(int r, int k) {
  return (uint32_t)((((r >> 3) * (kTcKC / 8) + (k >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1));
}

__device__ __forceinline__ float tc_val(const float* p) { return *p; }
__device__ __forceinline__ float tc_val(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ uint4 tc_pack(const float (&v)[8]) {
  uint4 o;
  __nv_bfloat162 h;
  h = __floats2bfloat162_rn(v[0], v[1]); o.x = *reinterpret_cast<uint32_t*>(&h);
  h = __floats2bfloat162_rn(v[2], v[3]); o.y = *reinterpret_cast<uint32_t*>(&h);
  h = __floats2bfloat162_rn(v[4], v[5]); o.z = *reinterpret_cast<uint32_t*>(&h);
  h = __floats2bfloat162_rn(v[6], v[7]); o.w = *reinterpret_cast<uint32_t*>(&h);
  return o;
}

// Stages rows [r0, r0 + rows) and k [k0, k0 + 64) of an operand X(r, k) as bfloat16, zero outside R rows
// and past kend (rows a multiple of 16).  KMAJ: X(r, k) at X[r ld + k], else at X[k ld + r].  ones: row
// R - 1 is all ones (the bias column of a weight gradient).
template <typename T, bool KMAJ>
__device__ __forceinline__ void tc_stage(unsigned char* dst, const T* __restrict__ X, int64_t ld, int r0, int rows, int R,
                                         int k0, int kend, bool ones) {
  constexpr int U = 4;                       // 8-element pieces in flight per thread
  const int npc = rows * (kTcKC / 8);
  // 16-byte loads of 8 consecutive k: rows and base 16-byte aligned (k0 is a multiple of 64 from an
  // operand start, and 8 elements are 16 or 32 bytes)
  const bool vec = KMAJ && ((ld * sizeof(T)) & 15) == 0 && (reinterpret_cast<uintptr_t>(X + k0) & 15) == 0;
  for (int base = threadIdx.x; base < npc; base += U * kTcThreads) {
    float v[U][8];
    int off[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int pc = base + u * kTcThreads;
      off[u] = -1;
#pragma unroll
      for (int e = 0; e < 8; ++e) v[u][e] = 0.0f;
      if (pc >= npc) continue;
      // 8 consecutive lanes take 8 consecutive rows: the 16-byte pieces of one core matrix, so the
      // stores are free of bank conflicts; each lane reads whole 32-byte sectors of its row
      // (k-contiguous operand) or the lanes read consecutive addresses (row-contiguous operand)
      const int r = KMAJ ? ((pc >> 6) << 3) | (pc & 7) : pc % rows, kc = KMAJ ? (pc >> 3) & 7 : pc / rows;
      const int k = k0 + 8 * kc, row = r0 + r;
      off[u] = (int)tc_off(r, 8 * kc);
      if (row >= R || k >= kend) continue;
      if (ones && row == R - 1) {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[u][e] = k + e < kend ? 1.0f : 0.0f;
      } else if (KMAJ && vec && k + 8 <= kend) {
        const T* p = X + (int64_t)row * ld + k;
        if constexpr (sizeof(T) == 4) {
          const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
          v[u][0] = a.x; v[u][1] = a.y; v[u][2] = a.z; v[u][3] = a.w;
          v[u][4] = b.x; v[u][5] = b.y; v[u][6] = b.z; v[u][7] = b.w;
        } else {
          const uint4 a = *reinterpret_cast<const uint4*>(p);
          const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            v[u][2 * e] = __uint_as_float(w[e] << 16);
            v[u][2 * e + 1] = __uint_as_float(w[e] & 0xFFFF0000u);
          }
        }
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (k + e < kend) v[u][e] = tc_val(KMAJ ? X + (int64_t)row * ld + k + e : X + (int64_t)(k + e) * ld + row);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (off[u] >= 0) *reinterpret_cast<uint4*>(dst + off[u]) = tc_pack(v[u]);
  }
}

// tensor-memory columns of an accumulator with Np columns: a power of two, at least 32
__host__ __device__ constexpr uint32_t tc_cols(int Np) {
  uint32_t c = 32;
  while ((int)c < Np) c <<= 1;
  return c;
}

template <typename TB, bool AK, bool BK>
__global__ void __launch_bounds__(kTcThreads) k_tc_gemm(TcGemmArgs a) {
  extern __shared__ __align__(1024) unsigned char tsm[];
  const int Np = (a.N + 15) & ~15;           // the MMA's N: a multiple of 16 for M = 128
  const uint32_t abytes = kTcRows * kTcKC * 2, bbytes = (uint32_t)Np * kTcKC * 2;
  unsigned char* As = tsm;                   // 2 x (128 x 64) bfloat16
  unsigned char* Bs = tsm + 2 * abytes;      // 2 x (Np x 64) bfloat16
  uint64_t* bar = reinterpret_cast<uint64_t*>(Bs + 2 * bbytes);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 2);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * kTcRows;
  const int kbeg = blockIdx.y * a.ksplit, kend = min(a.K, kbeg + a.ksplit);
  const int nsl1 = (kend - kbeg + kTcKC - 1) / kTcKC;
  const int nsl = nsl1 + (a.A2 ? (a.K2 + kTcKC - 1) / kTcKC : 0);
  uint32_t ncols = tc_cols(Np);
  // the second product has its own accumulator (added in binary32 after the first one and the bias)
  // while both fit in 256 columns
  const uint32_t acc2 = a.A2 && ncols <= 128 ? ncols : 0;
  ncols += acc2;
  if (warp == 0) tc_alloc(tslot, ncols);
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  const uint32_t idesc = tc_idesc_bf16(kTcRows, Np);
  bool bad = false;
  // the phase in which use number `use` of a buffer completes
  auto wait_use = [&](int buf, int use) {
    long spins = 0;
    while (!mbar_wait_hint(&bar[buf], (uint32_t)(use & 1)))
      if (++spins > kTcSpin) { bad = true; break; }
  };
  int sl = 0;
  for (; sl < nsl; ++sl) {
    const int buf = sl & 1;
    if (sl >= 2) wait_use(buf, (sl >> 1) - 1);   // the MMAs have read this buffer before it is rewritten
    unsigned char* Ab = As + buf * abytes;
    unsigned char* Bb = Bs + buf * bbytes;
    if (sl < nsl1) {
      const int k0 = kbeg + sl * kTcKC;
      tc_stage<float, AK>(Ab, a.A, a.lda, m0, kTcRows, a.M, k0, kend, false);
      tc_stage<TB, BK>(Bb, static_cast<const TB*>(a.B), a.ldb, 0, Np, a.N, k0, kend, a.b_ones_last != 0);
    } else {
      const int k0 = (sl - nsl1) * kTcKC;
      tc_stage<float, AK>(Ab, a.A2, a.lda2, m0, kTcRows, a.M, k0, a.K2, false);
      tc_stage<TB, BK>(Bb, static_cast<const TB*>(a.B2), a.ldb2, 0, Np, a.N, k0, a.K2, false);
    }
    fence_async_smem();                      // generic stores -> the tensor cores' (async) reads
    if (__syncthreads_or(bad)) { bad = true; break; }
    if (tid == 0) {
      tc_fence_after();
#pragma unroll
      for (int ks = 0; ks < kTcKC / 16; ++ks) {
        // K = 16 per MMA: two core matrices along K (lbo 128 bytes), 8-row groups 1024 bytes apart
        const uint64_t ad = tc_smem_desc(smem_u32(Ab) + ks * 256, 128, (kTcKC / 8) * 128);
        const uint64_t bd = tc_smem_desc(smem_u32(Bb) + ks * 256, 128, (kTcKC / 8) * 128);
        tc_mma_bf16(tmem + (sl >= nsl1 ? acc2 : 0u), ad, bd, idesc, ks > 0 || (sl > 0 && !(acc2 && sl == nsl1)) ? 1u : 0u);
      }
      tc_commit(&bar[buf]);
    }
  }
  // the last use of each buffer (sl: slices issued), the MMAs complete in order
  for (int q = max(0, sl - 2); q < sl; ++q) wait_use(q & 1, q >> 1);
  bad = __syncthreads_or(bad) != 0;
  tc_fence_after();
  if (bad) {
    if (tid == 0) atomicExch(a.err, 1);
  } else {
    const bool any = nsl > 0;                // no K range: the product is 0
    const int row = m0 + (warp & 3) * 32 + lane;   // a warp reads the lanes of its quarter
    float* Dz = a.D + (int64_t)blockIdx.y * a.dsplit;
    const bool vec = (a.ldd & 3) == 0 && (reinterpret_cast<uintptr_t>(Dz) & 15) == 0 &&
                     (!a.pre || (reinterpret_cast<uintptr_t>(a.pre) & 15) == 0);
    for (int c0 = (warp >> 2) * 8; c0 < Np; c0 += 16) {
      float v[8];
      tc_ld8(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
      float w[8];
      if (acc2) tc_ld8(tmem + acc2 + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, w);
      if (row >= a.M) continue;
      const int64_t idx = (int64_t)row * a.ldd + c0;
#pragma unroll
      for (int j = 0; j < 8; ++j)
        v[j] = (any ? v[j] : 0.0f) + (a.bias && c0 + j < a.N ? a.bias[c0 + j] : 0.0f);
      if (acc2) {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += w[j];
      }
      if (vec && c0 + 8 <= a.N) {
        if (a.relu) {
          if (a.pre) {
            *reinterpret_cast<float4*>(a.pre + idx) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(a.pre + idx + 4) = make_float4(v[4], v[5], v[6], v[7]);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = fmaxf(v[j], 0.0f);
        }
        *reinterpret_cast<float4*>(Dz + idx) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(Dz + idx + 4) = make_float4(v[4], v[5], v[6], v[7]);
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (c0 + j >= a.N) break;
          float o = v[j];
          if (a.relu) {
            if (a.pre) a.pre[idx + j] = o;
            o = fmaxf(o, 0.0f);
          }
          Dz[idx + j] = o;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tc_dealloc(tmem, ncols);
}

template <typename TB, bool AK, bool BK>
static cudaError_t tc_launch(const TcGemmArgs& a, size_t smem, dim3 grid, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_tc_gemm<TB, AK, BK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_tc_gemm<TB, AK, BK><<<grid, kTcThreads, smem, st>>>(a);
  return cudaGetLastError();
}

// Launch: D = A B^T over all of K (ksplit <= 0) or in K ranges of ksplit, a multiple of 64 (grid.y
// ranges, outputs dsplit apart).  Tensor memory is 512 columns per SM: the shared memory asked for
// leaves room for two CTAs with 256 columns, three with 128, and at most seven below that.
cudaError_t launch_tc_gemm(TcGemmArgs a, cudaStream_t st) {
  if (a.N < 1 || a.N > 256 || a.M < 1) return cudaErrorInvalidValue;
  if (a.ksplit <= 0) a.ksplit = a.K > 0 ? a.K : 1;
  const int Np = (a.N + 15) & ~15;
  const size_t need = 2 * ((size_t)kTcRows * kTcKC * 2 + (size_t)Np * kTcKC * 2) + 64;
  const uint32_t cols = tc_cols(Np) * (a.A2 && Np <= 128 ? 2 : 1);
  const size_t floor_b = cols > 128 ? 100 * 1024 : cols > 64 ? 58 * 1024 : 0;
  const size_t smem = need > floor_b ? need : floor_b;
  const int nsplit = a.K > 0 ? (a.K + a.ksplit - 1) / a.ksplit : 1;
  dim3 grid((a.M + kTcRows - 1) / kTcRows, nsplit);
  if (a.b_bf16) {
    if (!a.a_kmajor) return cudaErrorInvalidValue;
    return a.b_kmajor ? tc_launch<__nv_bfloat16, true, true>(a, smem, grid, st)
                      : tc_launch<__nv_bfloat16, true, false>(a, smem, grid, st);
  }
  if (a.a_kmajor != a.b_kmajor) return cudaErrorInvalidValue;
  return a.a_kmajor ? tc_launch<float, true, true>(a, smem, grid, st) : tc_launch<float, false, false>(a, smem, grid, st);
}

}  // namespace stdg

using namespace stdg;

// Test entry of the tensor-core product (binary32 A, B rounded to bfloat16, binary32 result):
// D[m * ldd + n] = Sum_k A[m * lda + k] B[n * ldb + k], 1 <= N <= 256.
extern "C" stdg_status stdg_tc_gemm_bf16(const float* A_dev, int64_t lda, const float* B_dev, int64_t ldb,
                                         float* D_dev, int64_t ldd, int M, int N, int K, void* stream) {
  if (!A_dev || !B_dev || !D_dev || M < 1 || N < 1 || N > 256 || K < 1) {
    set_error("stdg_tc_gemm_bf16: invalid argument (1 <= N <= 256)");
    return STDG_EINVAL;
  }
  int* err = nullptr;
  if (cudaMalloc(&err, sizeof(int)) != cudaSuccess) { set_error("stdg_tc_gemm_bf16: cudaMalloc failed"); return STDG_ENOMEM; }
  cudaStream_t st = (cudaStream_t)stream;
  cudaMemsetAsync(err, 0, sizeof(int), st);
  TcGemmArgs a{};
  a.M = M; a.N = N; a.K = K; a.ksplit = 0;
  a.A = A_dev; a.lda = lda; a.a_kmajor = 1;
  a.B = B_dev; a.ldb = ldb; a.b_kmajor = 1; a.b_bf16 = 0;
  a.D = D_dev; a.ldd = ldd; a.dsplit = 0;
  a.err = err;
  cudaError_t e = launch_tc_gemm(a, st);
  int herr = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(err);
  if (e != cudaSuccess) { set_error("stdg_tc_gemm_bf16: %s", cudaGetErrorString(e)); return STDG_ECUDA; }
  if (herr) { set_error("stdg_tc_gemm_bf16: a bounded wait for the tensor cores gave up"); return STDG_ETIMEOUT; }
  return STDG_OK;
}
