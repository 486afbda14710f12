// Operand preparation of the GEMM family: row-major FP32 matrices to the
// tensor-core operand formats, A row-major as it is, B transposed to K-major.
//
// Bound: HBM (one FP32 read, one operand write; FP8 reads twice, the scale
// needs the maximum first).  Both operands go through one launch, so a small
// product pays one launch instead of two, and every thread has four 16-byte
// loads in flight and writes four elements at a time.  Measured for A and B
// together, calls in a row in a graph, against one element per thread and store
// in a launch per operand:
//   BF16  8192^3   246 -> 112 us (7.2 TB/s)    4096^3   67 ->  29 us
//   FP32  8192^3   358 -> 237 us (6.8 TB/s)    4096^3   92 ->  59 us
//   FP8   8192^3   390 -> 173 us               4096^3  113 ->  41 us
//   BF16  8192 x 8191 x 4096 (N odd)  127 -> 58 us
// FP8 at 8192^3 is the time of two reads and one write at 7 TB/s.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <algorithm>

#include "pm_internal.cuh"

namespace pm {

__device__ __forceinline__ float tf32_rn(float x) {
  // round to nearest even at mantissa bit 13 (finite inputs)
  uint32_t b = __float_as_uint(x);
  if ((b & 0x7f800000u) == 0x7f800000u) return x;
  b = (b + 0xfffu + ((b >> 13) & 1u)) & 0xffffe000u;
  return __uint_as_float(b);
}

__device__ __forceinline__ float fp8_scale_of(unsigned int amax_bits) {
  const float amax = __uint_as_float(amax_bits);
  return amax > 0.f ? 448.f / amax : 1.f;
}

// One launch prepares both operands: blocks [0, a_blocks) convert A, the rest
// transpose and convert B, kPrepBlock elements each.
struct PrepArgs {
  const float* A;
  const float* B;
  void* A_op;
  void* B_op;
  int64_t nA;                      // elements of A (0: only B)
  int K, N;                        // B is K x N
  unsigned int a_blocks, n_tiles;  // blocks of A; 64-column tiles of B per 64-row band
  unsigned int* amax;              // FP8: |max| bits of A and of B
  float* scales;                   // FP8: s_A and s_B are written here
  int a_vec;                       // A, A_op (both planes) allow 4-element vectors
  int b_vec_in, b_vec_out;         // B rows / B_op rows (both planes) allow them
};

constexpr int kPrepThreads = 256;
constexpr int kPrepVec = 4;                                    // float4 loads in flight per thread
constexpr int kPrepBlock = kPrepThreads * kPrepVec * 4;        // 4096 elements = one 64 x 64 tile of B
constexpr int kPrepTile = 64;

template <int MODE>
__device__ __forceinline__ void prep_store1(void* y, int64_t i, int64_t lo_off, float v, float s) {
  if constexpr (MODE == PM_BF16) {
    static_cast<__nv_bfloat16*>(y)[i] = __float2bfloat16_rn(v);
  } else if constexpr (MODE == PM_FP8E4M3) {
    static_cast<__nv_fp8_storage_t*>(y)[i] = __nv_cvt_float_to_fp8(v * s, __NV_SATFINITE, __NV_E4M3);
  } else {
    const float hi = tf32_rn(v);
    static_cast<float*>(y)[i] = hi;
    static_cast<float*>(y)[i + lo_off] = tf32_rn(v - hi);
  }
}

// Elements i .. i+3 (i a multiple of 4, y aligned to four elements).
template <int MODE>
__device__ __forceinline__ void prep_store4(void* y, int64_t i, int64_t lo_off, float4 v, float s) {
  if constexpr (MODE == PM_BF16) {
    __nv_bfloat162 p[2] = {__floats2bfloat162_rn(v.x, v.y), __floats2bfloat162_rn(v.z, v.w)};
    *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(y) + i) = *reinterpret_cast<const uint2*>(p);
  } else if constexpr (MODE == PM_FP8E4M3) {
    const uint32_t a = __nv_cvt_float2_to_fp8x2(make_float2(v.x * s, v.y * s), __NV_SATFINITE, __NV_E4M3);
    const uint32_t b = __nv_cvt_float2_to_fp8x2(make_float2(v.z * s, v.w * s), __NV_SATFINITE, __NV_E4M3);
    *reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(y) + i) = a | (b << 16);
  } else {
    const float4 hi = make_float4(tf32_rn(v.x), tf32_rn(v.y), tf32_rn(v.z), tf32_rn(v.w));
    *reinterpret_cast<float4*>(static_cast<float*>(y) + i) = hi;
    *reinterpret_cast<float4*>(static_cast<float*>(y) + i + lo_off) =
        make_float4(tf32_rn(v.x - hi.x), tf32_rn(v.y - hi.y), tf32_rn(v.z - hi.z), tf32_rn(v.w - hi.w));
  }
}

// Clears the |max| words ahead of amax_kernel.  A kernel and not a memset, so that
// amax_kernel is set up and reads during it.  FP8 preparations in a captured graph,
// 512^3 8.2 -> 3.9 us, 2048^3 12.3 -> 8.8, 4096^3 44.7 -> 41.0; called one by one, each
// with its GEMM, 2048^3 22.9 -> 21.2, 4096^3 102.3 -> 101.4, below 1024^3 bound by the
// host's calls on either side.
__global__ void amax_clear_kernel(unsigned int* amax_bits) {
  grid_dependents_launch();
  if (threadIdx.x < 2) amax_bits[threadIdx.x] = 0u;
}

// Per-tensor |max| of A and B (FP8), one launch: blocks [0, a_blocks) read A,
// the rest B, in kPrepBlock pieces with four 16-byte loads in flight per thread;
// one atomic per block.
__global__ void __launch_bounds__(kPrepThreads) amax_kernel(const float* __restrict__ A, int64_t nA,
                                                            unsigned int a_blocks, const float* __restrict__ B,
                                                            int64_t nB, int a_vec, int b_vec,
                                                            unsigned int* __restrict__ amax_bits) {
  grid_dependents_launch();                      // the conversion may be set up (it waits for this grid)
  const bool is_a = blockIdx.x < a_blocks;
  const float* x = is_a ? A : B;
  const int64_t n = is_a ? nA : nB;
  const unsigned int first = is_a ? blockIdx.x : blockIdx.x - a_blocks;
  const unsigned int step = is_a ? a_blocks : gridDim.x - a_blocks;
  const bool vec = (is_a ? a_vec : b_vec) != 0;
  float m = 0.f;
  for (int64_t base = (int64_t)first * kPrepBlock; base < n; base += (int64_t)step * kPrepBlock) {
    if (vec && base + kPrepBlock <= n) {
      const float4* p = reinterpret_cast<const float4*>(x + base) + threadIdx.x;
      float4 v[kPrepVec];
#pragma unroll
      for (int u = 0; u < kPrepVec; ++u) v[u] = __ldg(p + u * kPrepThreads);
#pragma unroll
      for (int u = 0; u < kPrepVec; ++u)
        m = fmaxf(fmaxf(fmaxf(m, fabsf(v[u].x)), fmaxf(fabsf(v[u].y), fabsf(v[u].z))), fabsf(v[u].w));
    } else {
      const int64_t end = min(base + (int64_t)kPrepBlock, n);
      for (int64_t i = base + threadIdx.x; i < end; i += kPrepThreads) m = fmaxf(m, fabsf(__ldg(x + i)));
    }
  }
  __shared__ float wm[kPrepThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kPrepThreads / 32; ++w) m = fmaxf(m, wm[w]);
    grid_dependency_wait();                      // after amax_clear_kernel; A and B are older than that
    atomicMax(amax_bits + (is_a ? 0 : 1), __float_as_uint(m));
  }
}

// Plain loads: A and B may be the results of the kernel that this one overlaps
// (grid_dependency_wait).  Vector accesses are used where the pointers and the row lengths allow them
// (a_vec, b_vec_in, b_vec_out: four elements of the type, checked on the
// host); otherwise, and in partial blocks, one element at a time.  A 64 x 64
// tile of B goes through shared memory with rows of 65 words: four k of one
// column per thread, eight lanes along k, read without bank conflicts and
// written as full 32-byte sectors in every type.
template <int MODE>
__global__ void __launch_bounds__(kPrepThreads) prep_kernel(const PrepArgs p) {
  __shared__ float tile[kPrepTile * (kPrepTile + 1)];
  const int tid = threadIdx.x;
  grid_dependents_launch();                      // a GEMM on these operands may be set up
  grid_dependency_wait();                        // what the previous kernel of the stream wrote or still read is settled
  // FP8: the maximum pass read A and B at once, each front to back; walking the
  // blocks from the end starts with what it read last of B, which is still in L2
  const unsigned int blk = MODE == PM_FP8E4M3 ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
  float s = 1.f;
  if constexpr (MODE == PM_FP8E4M3) {
    s = fp8_scale_of(p.amax[blk < p.a_blocks ? 0 : 1]);
    if (tid == 0 && blk == 0 && p.a_blocks) p.scales[0] = s;
    if (tid == 0 && blk == p.a_blocks) p.scales[1] = s;
  }
  if (blk < p.a_blocks) {
    const int64_t base = (int64_t)blk * kPrepBlock;
    if (p.a_vec && base + kPrepBlock <= p.nA) {
      const float4* x = reinterpret_cast<const float4*>(p.A + base) + tid;
      float4 v[kPrepVec];
#pragma unroll
      for (int u = 0; u < kPrepVec; ++u) v[u] = x[u * kPrepThreads];
#pragma unroll
      for (int u = 0; u < kPrepVec; ++u)
        prep_store4<MODE>(p.A_op, base + 4 * (tid + u * kPrepThreads), p.nA, v[u], s);
    } else {
      // eight loads ahead of their stores (for all the compiler knows the stores go to where the loads read)
      const float* x = p.A + base;
      const int left = (int)min((int64_t)kPrepBlock, p.nA - base);
      for (int j0 = tid; j0 < left; j0 += 8 * kPrepThreads) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = j0 + u * kPrepThreads < left ? x[j0 + u * kPrepThreads] : 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (j0 + u * kPrepThreads < left) prep_store1<MODE>(p.A_op, base + j0 + u * kPrepThreads, p.nA, v[u], s);
      }
    }
    return;
  }
  const unsigned int bt = blk - p.a_blocks;
  const int k0 = (int)(bt / p.n_tiles) * kPrepTile, n0 = (int)(bt % p.n_tiles) * kPrepTile;
  constexpr int S = kPrepTile + 1;
  if (p.b_vec_in && k0 + kPrepTile <= p.K && n0 + kPrepTile <= p.N) {
    const int r0 = tid >> 4, c = (tid & 15) * 4;
    float4 v[kPrepVec];
#pragma unroll
    for (int u = 0; u < kPrepVec; ++u)
      v[u] = *reinterpret_cast<const float4*>(p.B + (size_t)(k0 + r0 + 16 * u) * p.N + n0 + c);
#pragma unroll
    for (int u = 0; u < kPrepVec; ++u) {
      float* t = tile + (r0 + 16 * u) * S + c;
      t[0] = v[u].x; t[1] = v[u].y; t[2] = v[u].z; t[3] = v[u].w;
    }
  } else {
    const int r0 = tid >> 6, c = tid & 63;
    const bool in = n0 + c < p.N;
    float v[kPrepTile / 4];
#pragma unroll
    for (int u = 0; u < kPrepTile / 4; ++u) {
      const int k = k0 + r0 + 4 * u;
      v[u] = (in && k < p.K) ? p.B[(size_t)k * p.N + n0 + c] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kPrepTile / 4; ++u) tile[(r0 + 4 * u) * S + c] = v[u];
  }
  __syncthreads();
  const int64_t lo = (int64_t)p.N * p.K;
  if (p.b_vec_out) {
    // four k per thread, eight lanes along k (bank 4 kq + n: no conflicts),
    // four columns per warp and pass
    const int kq = tid & 7, nn = tid >> 3;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int kk = 4 * (kq + 8 * (u & 1)), n = nn + 32 * (u >> 1);
      if (k0 + kk >= p.K || n0 + n >= p.N) continue;
      const float* t = tile + kk * S + n;
      prep_store4<MODE>(p.B_op, (int64_t)(n0 + n) * p.K + k0 + kk, lo, make_float4(t[0], t[S], t[2 * S], t[3 * S]), s);
    }
  } else {
    const int kk = tid & 63;
    for (int n = tid >> 6; n < kPrepTile; n += 4)
      if (k0 + kk < p.K && n0 + n < p.N)
        prep_store1<MODE>(p.B_op, (int64_t)(n0 + n) * p.K + k0 + kk, lo, tile[kk * S + n], s);
  }
}

// Launches the operand preparation of A (rows x K, or none: A == nullptr) and
// B (K x N, or none) on stream s.  FP8: scales[2..3] collect the |max| bits
// (cleared here if clear is set, else by the caller before the first operand),
// scales[0..1] the scales.
static pm_status prepare_on(int dt, const float* A, int64_t rows, const float* B, int K, int N, void* A_op, void* B_op,
                            float* scales, bool clear, cudaStream_t s) {
  PrepArgs p = {};
  const int e = dt == PM_FP32 ? 4 : (dt == PM_BF16 ? 2 : 1);
  auto aligned = [](const void* x, int bytes) { return ((uintptr_t)x & (uintptr_t)(bytes - 1)) == 0; };
  p.A = A;
  p.B = B;
  p.A_op = A_op;
  p.B_op = B_op;
  p.nA = A ? rows * K : 0;
  p.K = K;
  p.N = N;
  p.a_vec = aligned(A, 16) && aligned(A_op, 4 * e) && (dt != PM_FP32 || p.nA % 4 == 0);
  p.b_vec_in = aligned(B, 16) && N % 4 == 0;
  p.b_vec_out = aligned(B_op, 4 * e) && K % 4 == 0;
  const int64_t nB = B ? (int64_t)K * N : 0;
  const int64_t a_blocks = (p.nA + kPrepBlock - 1) / kPrepBlock;
  p.n_tiles = (unsigned int)((N + kPrepTile - 1) / kPrepTile);
  const int64_t blocks = a_blocks + (B ? (int64_t)((K + kPrepTile - 1) / kPrepTile) * p.n_tiles : 0);
  PM_REQUIRE(blocks < (1ll << 31), PM_EINVAL, "operands too large for one preparation launch");
  p.a_blocks = (unsigned int)a_blocks;
  if (dt == PM_FP8E4M3) {
    p.scales = scales;
    p.amax = reinterpret_cast<unsigned int*>(scales + 2);
    // eight resident blocks per SM, shared between the matrices by their size
    const int64_t cap = (int64_t)std::max(1, sm_count()) * 8;
    const int64_t pieces_b = (nB + kPrepBlock - 1) / kPrepBlock;
    int64_t ga = a_blocks, gb = pieces_b;
    if (ga + gb > cap) {
      ga = A ? std::max<int64_t>(1, cap * a_blocks / (a_blocks + pieces_b)) : 0;
      gb = B ? std::max<int64_t>(1, cap - ga) : 0;
    }
    if (clear) {
      amax_clear_kernel<<<1, 32, 0, s>>>(p.amax);
      pm_status st = launch_status("amax_clear_kernel");
      if (st != PM_OK) return st;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned int)(ga + gb));
    cfg.blockDim = dim3(kPrepThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = clear ? 1 : 0;                // only amax_clear_kernel may still run beside it
    cudaError_t e1 = cudaLaunchKernelEx(&cfg, amax_kernel, A, p.nA, (unsigned int)ga, B, nB, (int)aligned(A, 16),
                                        (int)aligned(B, 16), p.amax);
    if (e1 != cudaSuccess) return cuda_fail(e1, "cudaLaunchKernelEx(amax_kernel)");
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned int)blocks);
  cfg.blockDim = dim3(kPrepThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto kern = dt == PM_FP8E4M3 ? prep_kernel<PM_FP8E4M3> : (dt == PM_BF16 ? prep_kernel<PM_BF16> : prep_kernel<PM_FP32>);
  cudaError_t e2 = cudaLaunchKernelEx(&cfg, kern, (const PrepArgs)p);
  if (e2 != cudaSuccess) return cuda_fail(e2, "cudaLaunchKernelEx(prep_kernel)");
  return PM_OK;
}

pm_status launch_prepare(int dt, const float* A, int64_t rows, const float* B, int K, int N, void* A_op, void* B_op,
                         float* scales, cudaStream_t s) {
  return prepare_on(dt, A, rows, B, K, N, A_op, B_op, scales, false, s);
}

}  // namespace pm

extern "C" pm_status pm_gemm_prepare(int32_t dtype, const float* A_dev, const float* B_dev, int32_t M, int32_t N,
                                     int32_t K, void* A_op_dev, void* B_op_dev, float* scales_dev, void* stream) {
  PM_REQUIRE(dtype >= 0 && dtype <= 2 && M > 0 && N > 0 && K > 0, PM_EINVAL, "bad dtype or shape");
  PM_REQUIRE(A_dev && B_dev && A_op_dev && B_op_dev, PM_EINVAL, "null pointer");
  PM_REQUIRE(dtype != PM_FP8E4M3 || scales_dev, PM_EINVAL, "FP8 needs scales_dev (4 floats)");
  PM_REQUIRE(K <= pm::kPrepareMaxK, PM_EINVAL, "K %d is above %d", K, pm::kPrepareMaxK);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return pm::prepare_on(dtype, A_dev, M, B_dev, K, N, A_op_dev, B_op_dev, scales_dev, true, s);
}

