// Input-tile transform for tiles of 4 points (Section 2.1 step 1 in its 2-D nested form, Appendix B.5):
// V = B^T d B in half mode for F(2,3), on CUDA cores.
//
// What bounds it: the bytes.  A tile has 16 points and a handful of additions per point, so the tensor-core
// kernel spends its time on fixed costs per (tile, 64 channels); here a thread owns one tile and four
// consecutive channels, keeps the whole patch in registers and does 16 eight-byte loads and 16 eight-byte stores,
// each of a warp 256 contiguous bytes at 128 channels.  The four patches that share an input pixel are those of
// neighbouring threads' tiles and find it in the L1.
// A CTA waits for the preceding kernel and lets the following one be scheduled like the other transforms.
// Whole call, against the tensor-core kernel (C >= 64) and the two-channel CUDA-core kernel (below): 32 x 56 x 56,
// 128 -> 128: 158.6 -> 117 us; 32 x 28 x 28, 512 -> 256: 121 -> 83; 2 x 14 x 14, 512 -> 128: 11.1 -> 9.9; 8 x 28 x 28,
// 32 -> 64: 11.6 -> 9.4; 32 x 56 x 56, 24 -> 64: 54.6 -> 50.4; 8 x 56 x 56, 64 -> 64 unchanged at 18.8.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "nova_internal.h"
#include "sm100.cuh"
#include "tma_host.h"
#include "transform_math.cuh"

namespace nova {
namespace {
using namespace xf;

constexpr int kN4Threads = 128;

__device__ __forceinline__ float2 lo2(uint2 v) { return __half22float2(*reinterpret_cast<const __half2*>(&v.x)); }
__device__ __forceinline__ float2 hi2(uint2 v) { return __half22float2(*reinterpret_cast<const __half2*>(&v.y)); }
__device__ __forceinline__ uint32_t pack2(float2 v) {
  const __half2 h = __floats2half2_rn(v.x, v.y);
  return *reinterpret_cast<const uint32_t*>(&h);
}

template <bool SYM>
__global__ void __launch_bounds__(kN4Threads)
input_transform_n4_kernel(const __grid_constant__ Coefs cf, const __half* __restrict__ x, __half* __restrict__ V, int H, int W,
                          int C, int ldv, int Th, int Tw, long long p0, int pc, int pc_pad) {
  constexpr int N = 4;
  sm100::pdl_wait();
  sm100::pdl_launch_dependents();
  const unsigned c4 = (unsigned)C >> 2;
  const unsigned long long idx = (unsigned long long)blockIdx.x * kN4Threads + threadIdx.x;
  const unsigned pl = (unsigned)(idx / c4);
  if (pl >= (unsigned)pc) return;
  const int c = (int)(idx % c4) * 4;
  const unsigned long long p = (unsigned long long)p0 + pl;
  const int tw = (int)(p % (unsigned)Tw);
  const unsigned long long q = p / (unsigned)Tw;
  const int th = (int)(q % (unsigned)Th);
  const long long img = (long long)(q / (unsigned)Th);
  const int h0 = 2 * th - 1, w0 = 2 * tw - 1;
  const __half* base = x + ((img * H + h0) * (long long)W + w0) * C + c;
  uint2 d[N][N];
#pragma unroll
  for (int a = 0; a < N; ++a)
#pragma unroll
    for (int b = 0; b < N; ++b) {
      d[a][b] = make_uint2(0u, 0u);
      if ((unsigned)(h0 + a) < (unsigned)H && (unsigned)(w0 + b) < (unsigned)W)
        d[a][b] = __ldg(reinterpret_cast<const uint2*>(base + ((long long)a * W + b) * C));
    }
  // columns first (index a), then rows (index b), as the other transforms: half the channels at a time
  uint32_t o[2][N][N];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    float2 t[N][N];
#pragma unroll
    for (int a = 0; a < N; ++a) {
      float2 in[N], out[N];
#pragma unroll
      for (int b = 0; b < N; ++b) in[b] = e ? hi2(d[a][b]) : lo2(d[a][b]);
      bt_all_rows<N, SYM>(cf, in, out);
#pragma unroll
      for (int b = 0; b < N; ++b) t[b][a] = out[b];
    }
#pragma unroll
    for (int nu = 0; nu < N; ++nu) {
      float2 out[N];
      bt_all_rows<N, SYM>(cf, t[nu], out);
#pragma unroll
      for (int xi = 0; xi < N; ++xi) o[e][xi][nu] = pack2(out[xi]);
    }
  }
  const size_t f_stride = (size_t)pc_pad * ldv;
  __half* dst = V + (size_t)pl * ldv + c;
#pragma unroll
  for (int xi = 0; xi < N; ++xi)
#pragma unroll
    for (int nu = 0; nu < N; ++nu)
      *reinterpret_cast<uint2*>(dst + (size_t)(xi * N + nu) * f_stride) = make_uint2(o[0][xi][nu], o[1][xi][nu]);
}

}  // namespace

int launch_input_transform_n4(const nova_plan* plan, const Geom& g, const void* x, void* V, long long p0, int pc, int pc_pad,
                              void* stream) {
  const long long work = (long long)pc * (g.C / 4);
  const int grid = (int)((work + kN4Threads - 1) / kN4Threads);
  cudaStream_t s = (cudaStream_t)stream;
  return (int)(plan->symmetric
                   ? launch_overlapped(input_transform_n4_kernel<true>, grid, kN4Threads, 0, s, plan->kcoefs, (const __half*)x,
                                       (__half*)V, g.H, g.W, g.C, g.ldv, g.Th, g.Tw, p0, pc, pc_pad)
                   : launch_overlapped(input_transform_n4_kernel<false>, grid, kN4Threads, 0, s, plan->kcoefs, (const __half*)x,
                                       (__half*)V, g.H, g.W, g.C, g.ldv, g.Th, g.Tw, p0, pc, pc_pad));
}

}  // namespace nova
