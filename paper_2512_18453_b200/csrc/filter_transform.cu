// Filter transform U = G g G^T of the half pipeline (Section 2.1 step 2 in its 2-D nested form, Appendix B.5),
// evaluated in float and rounded once to half.  g [K,R,R,C] -> U [n*n][K][C].
//
// What bounds it: the stores of U, n*n / (R*R) times the bytes of g.  A thread owns one filter, four consecutive
// channels (eight-byte accesses, a warp's store 256 contiguous bytes) and two rows of the n x n frequencies, so that
// a small layer still spreads over the SMs, or all rows, so that the taps of a large one are read once (see the launcher).
// Launched as a programmatic dependent: a plain launch costs the host up to twice as much and nothing of it overlaps.
// Against one thread per channel pair and whole filter, launched plainly: F(6,3) 512 x 512 (38 MB) 7.5 -> 7.2 us back to
// back, 64 x 64 3.4 -> 2.1; F(8,3) 512 x 512 (57 MB) 10.9 -> 9.9; per call 11.2 -> 6.0 us wherever the host is the bound.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "nova_internal.h"
#include "sm100.cuh"
#include "tma_host.h"
#include "transform_math.cuh"

namespace nova {
namespace {
using namespace xf;

constexpr int kFtThreads = 256;

template <int N, int R, int ROWS>
__global__ void __launch_bounds__(kFtThreads)
filter_transform_half_kernel(const __grid_constant__ Coefs cf, const __half* __restrict__ g, __half* __restrict__ U, int K, int C) {
  sm100::pdl_wait();
  sm100::pdl_launch_dependents();
  const unsigned c4 = (unsigned)C >> 2;
  const unsigned long long idx = (unsigned long long)blockIdx.x * kFtThreads + threadIdx.x;
  const unsigned k = (unsigned)(idx / c4);
  if (k >= (unsigned)K) return;
  const int c = (int)(idx % c4) * 4;
  float2 gg[2][R][R];                               // [channel pair][a][b]
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(g + ((size_t)(k * R + a) * R + b) * C + c));
      gg[0][a][b] = __half22float2(*reinterpret_cast<const __half2*>(&v.x));
      gg[1][a][b] = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
    }
  const size_t f_stride = (size_t)K * C;
  __half* dst = U + (size_t)k * C + c;
#pragma unroll 2
  for (int e = 0; e < ROWS; ++e) {
    const int p = ROWS * (int)blockIdx.y + e;
    float2 t[2][R];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int b = 0; b < R; ++b) {
        t[h][b] = mul2(cf.G[p][0], gg[h][0][b]);
#pragma unroll
        for (int a = 1; a < R; ++a) t[h][b] = fma2(cf.G[p][a], gg[h][a][b], t[h][b]);
      }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      uint2 o;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float2 s = mul2(cf.G[q][0], t[h][0]);
#pragma unroll
        for (int b = 1; b < R; ++b) s = fma2(cf.G[q][b], t[h][b], s);
        const __half2 r = __floats2half2_rn(s.x, s.y);
        (h ? o.y : o.x) = *reinterpret_cast<const uint32_t*>(&r);
      }
      *reinterpret_cast<uint2*>(dst + (size_t)(p * N + q) * f_stride) = o;
    }
  }
}

template <int N, int R, int ROWS>
int start(const nova_plan* plan, const void* g, int K, int C, void* U, cudaStream_t s) {
  const long long work = (long long)K * (C / 4);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((work + kFtThreads - 1) / kFtThreads), N / ROWS);
  cfg.blockDim = dim3(kFtThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return (int)cudaLaunchKernelEx(&cfg, filter_transform_half_kernel<N, R, ROWS>, plan->kcoefs, (const __half*)g, (__half*)U, K, C);
}

// All n rows per thread from 2^17 threads on, where they fill the chip by themselves.  Two rows / all rows: 3 x 3, 1024 x
// 1024: F(2,3) 9.3 / 7.8 us, F(4,3) 19.0 / 15.7, F(6,3) 28.6 / 26.3; 2048 x 2048: F(6,3) 111 / 98, F(6,5) 246 / 215; 1024 x 512:
// F(6,3) 13.5 / 11.9, F(8,3) 21.5 / 19.1.  Below: 512 x 512 F(6,3) 7.6 / 8.7, F(8,3) 10.3 / 13.5; 64 x 64 F(6,5) 6.5 / 7.8.
template <int N, int R>
int go(const nova_plan* plan, const void* g, int K, int C, void* U, cudaStream_t s) {
  return (long long)K * (C / 4) >= 1 << 17 ? start<N, R, N>(plan, g, K, C, U, s) : start<N, R, 2>(plan, g, K, C, U, s);
}

}  // namespace

int launch_filter_transform(const nova_plan* plan, const void* g, int K, int C, void* U, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  if (plan->mode == NOVA_FP32) return (int)cudaErrorInvalidValue;      // the fp32 mode has its own transforms
  if (plan->r == 3) switch (plan->n) {
      case 4: return go<4, 3>(plan, g, K, C, U, s);
      case 6: return go<6, 3>(plan, g, K, C, U, s);
      case 8: return go<8, 3>(plan, g, K, C, U, s);
      case 10: return go<10, 3>(plan, g, K, C, U, s);
    }
  if (plan->r == 5) switch (plan->n) {
      case 6: return go<6, 5>(plan, g, K, C, U, s);
      case 8: return go<8, 5>(plan, g, K, C, U, s);
      case 10: return go<10, 5>(plan, g, K, C, U, s);
    }
  return (int)cudaErrorInvalidValue;
}

}  // namespace nova
