// Section 2.1 steps 2-4 of the fp32 mode in ONE kernel (tiles of up to 8 points): V = B^T d B, M[f] =
// V[f] U[f]^T and Y = A^T M A for a block of 8 tiles and up to 32 filters at a time, V and M never leaving
// the SM.  Sums are carried in double; V and y are rounded once to float, M is not rounded at all.
//
// What bounds it: the double-precision pipe (64 multiply-adds per clock and SM, as DFMA and as DMMA), which
// a product of n*n * C * K multiply-adds per tile fills whatever the layout; so the float operands are
// fetched and widened as little as possible and no pass over V or M is left.  The three kernels this one
// replaced widened every operand at every use and were several times off that bound; figures at
// choose_blocks.
//
// Roles (warpgroups, registers split by setmaxnreg):
//   product warps    warp (nu, h) owns the n frequencies (., nu) and its share of the filters: the sums of
//                    8 tiles x 8 * nb filters x n rows xi live in its registers while the loop over the
//                    channels runs (mma.sync m8n8k4 f64).  A thread's operands of a row are 16 CONSECUTIVE
//                    bytes of channels, which only permutes the order of the contraction.  After the last
//                    chunk: A^T along xi in registers, the n columns meet in shared memory (kZRows output
//                    rows at a time), A^T along nu, y.
//   transform warps  V of the next chunk from the patches of x; a thread owns one (tile, channel), reads
//                    its patch once and produces V row pair by row pair.  With eight warps the row pairs of
//                    a patch are shared out to two threads.
//   producer warps   TMA: U, one box of n frequencies x filters per row xi; x, one box per tile
//                    (out-of-range pixels and channels read as 0).
// With `split` > 1 the channel chunks of a block are dealt to the CTAs of a cluster, which add their sums
// through distributed shared memory (A^T along xi is linear, so it comes first).
// Every wait is bounded by the clock; after one has expired no role waits any more and all run to their end.
#include <cuda_runtime.h>

#include "nova_internal.h"
#include "sm100.cuh"
#include "tma_host.h"
#include "transform_math.cuh"

namespace nova {
namespace {
using namespace sm100;
using namespace xf;

constexpr int kTiles = 8;                // tiles of a block: the rows of one mma
constexpr int kProducerWarps = 4;
constexpr int kChunk = 16;               // channels per chunk
constexpr int kRowBytes = 4 * kChunk;
constexpr int kRecRing = 8;              // tile records: the producer is at most five blocks ahead of the stores

// ROWS: the end of a block that exchanges one output row at a time (see kZRows), whatever the tile
template <int M, int R, bool ROWS>
struct Fc32 {
  static constexpr int N = M + R - 1, PAD = (R - 1) / 2, NF = N * N;
  static constexpr int NH = (N == 8) ? 1 : 2;                      // warps that share a column nu
  static constexpr int NB = (N == 8) ? 4 : 2;                      // 8-filter blocks of a warp, at most
  static constexpr int F = 8 * NB * NH;                            // filters of a block, at most: 32
  static constexpr int kProductWarps = N * NH;                     // 8, 12, 8
  static constexpr int kProductThreads = 32 * kProductWarps;
  static constexpr int kShares = (N == 8) ? 1 : 2;                 // threads per (tile, channel) of the transform
  static constexpr int kTransformWarps = 4 * kShares;
  static constexpr int kThreads = kProductThreads + 32 * (kTransformWarps + kProducerWarps);
  static constexpr int kStages = (N == 6) ? 6 : 4;                 // ring of U
  static_assert(N % kStages == 0, "a row always uses the same stage");
  static constexpr int kXTile = NF * kRowBytes;
  static constexpr int kXBytes = kTiles * kXTile;
  static constexpr int kVRow = N * kTiles * kRowBytes;
  static constexpr int kVBytes = N * kVRow;
  static constexpr int kStage = N * F * kRowBytes;
  static constexpr int kZRow = N * kTiles * F * 8;
  // Output rows that meet in shared memory at a time.  Row by row, in two buffers in turn, most product warps wait at a barrier
  // per row: a block's end took as long as one of its chunks.  Whole call, row by row / this: F(4,3) 8 x 56 x 56, 64 -> 64 34.6 / 33.9 us,
  // 3 x 46 x 46, 32 -> 32 9.9 / 9.1; F(6,3) 61 x 107, 32 -> 256 28.3 / 26.9.  Two output rows stay with it: 8 x 56 x 56, 64 -> 64, F(2,3) 55.8 / 58.7.
  // A kernel compiled with this end is the slower one where a cluster splits the channels, although that path's source is the same: six
  // points, 1 x 40 x 40, 112 -> 8 9.11 / 9.37, 9 x 24 x 15, 224 -> 8 12.57 / 12.85, 2 x 101 x 32, 224 -> 16 17.9 / 18.3; such calls keep a
  // kernel with the row-by-row end (eight points gain either way: 2 x 7 x 30, 48 -> 8, asymmetric 24.5 / 21.1).
  static constexpr int kZRows = (M == 2 || ROWS) ? 1 : (N == 8) ? 2 : M;
  static_assert(M % kZRows == 0, "");
  static constexpr int kOffX = 0;
  static constexpr int kOffV = kOffX + kXBytes;
  static constexpr int kOffU = kOffV + 2 * kVBytes;
  static constexpr int kOffZ = kOffU + kStages * kStage;
  static constexpr int kOffRec = kOffZ + (kZRows == 1 ? 2 : kZRows) * kZRow;
  static constexpr int kOffBar = kOffRec + kRecRing * kTiles * 16;
  static constexpr int kTotal = kOffBar + 8 * (2 * kStages + 2 + 4) + 16 + 128;
  static_assert(kTotal <= 227 * 1024, "shared memory of one CTA");
  static_assert(M * kZRow <= kOffRec, "the exchange of a split block fits over the operand buffers");
  static_assert(kXTile % 128 == 0 && kStage % 128 == 0 && kVRow % 128 == 0, "");
  // registers per thread; their sum must not exceed what the block is launched with
  static constexpr int kLaunchRegs = (65536 / kThreads) / 8 * 8;
  static constexpr int kProductRegs = (N == 8) ? 160 : (N == 6) ? 88 : 104;
  static constexpr int kTransformRegs = (N == 8) ? 168 : (N == 6) ? 88 : 80;
  static constexpr int kProducerRegs = 24;
  static_assert(kProductRegs * kProductThreads + kTransformRegs * 32 * kTransformWarps + kProducerRegs * 32 * kProducerWarps <=
                kLaunchRegs * kThreads, "register split");
};

struct FcRec {            // where a tile's outputs go; rows = 0 for a tile past the end
  long long ybase;        // element offset of pixel (0, 0), filter 0 of the tile
  int rows, cols;
};
struct FcArgs {
  int H, W, K, Th, Tw;
  long long P;
  int chunks, num_kb, nb, split, relu;
  unsigned blocks;
};

__device__ __forceinline__ void fc_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_test(bar, parity)) return;
  if (*abort_flag) return;
  if (!mbar_wait(bar, parity, abort_flag)) *abort_flag = 1;
}
__device__ __forceinline__ float4 lds_f4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ float lds_f1(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts_f1(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void sts_d2(uint32_t a, Dbl2 v) { asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory"); }
__device__ __forceinline__ Dbl2 lds_d2(uint32_t a) {
  Dbl2 v;
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
  return v;
}
// the double pair at a shared::cluster address (another CTA's shared memory)
__device__ __forceinline__ Dbl2 lds_peer_d2(uint32_t a) {
  Dbl2 v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// The barriers below are aligned ones: a warp comes to them as a whole, after stores that only some of its threads did.
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mma884(Dbl2& d, float a, float b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
               : "+d"(d.x), "+d"(d.y) : "d"((double)a), "d"((double)b));
}

// Rows 0 and n-1 first, then the pairs: the order in which the transform produces them.
template <int N>
__host__ __device__ constexpr int row_of(int step) { return step == 0 ? 0 : step == 1 ? N - 1 : step - 1; }

// Steps 2G and 2G + 1 (rows) of V for one (tile, channel) from its patch, to shared memory.
template <int N, bool SYM, int G>
__device__ __forceinline__ void v_row_pair(const CoefsD& cf, const float (&raw)[N * N], uint32_t dst, int row_bytes) {
  double ta[N], tb[N], o[N];
#pragma unroll
  for (int b = 0; b < N; ++b) {
    double in[N];
#pragma unroll
    for (int a = 0; a < N; ++a) in[a] = (double)raw[a * N + b];
    bt_two_rows<N, SYM, G>(cf, in, ta[b], tb[b]);
  }
  bt_all_rows<N, SYM>(cf, ta, o);
#pragma unroll
  for (int nu = 0; nu < N; ++nu) sts_f1(dst + 2 * G * row_bytes + nu * kTiles * kRowBytes, (float)o[nu]);
  bt_all_rows<N, SYM>(cf, tb, o);
#pragma unroll
  for (int nu = 0; nu < N; ++nu) sts_f1(dst + (2 * G + 1) * row_bytes + nu * kTiles * kRowBytes, (float)o[nu]);
}

// Output row i of one (tile, filter pair).
template <int M>
__device__ __forceinline__ void put_row(int i, const Dbl2 (&v)[M], float* yt, const FcRec& rec, const FcArgs& a) {
  if (i >= rec.rows) return;
  float* p = yt + (long long)i * a.W * a.K;
#pragma unroll
  for (int j = 0; j < M; ++j)
    if (j < rec.cols) {
      float2 f = make_float2((float)v[j].x, (float)v[j].y);
      if (a.relu) f = make_float2(f.x < 0.f ? 0.f : f.x, f.y < 0.f ? 0.f : f.y);       // NaN and +inf pass
      __stcs(reinterpret_cast<float2*>(p + (long long)j * a.K), f);
    }
}

template <int M, int R, bool SYM, bool ROWS>
__global__ void __launch_bounds__(Fc32<M, R, ROWS>::kThreads, 1)
fused_fp32_kernel(const __grid_constant__ CoefsD cf, const __grid_constant__ CUtensorMap tmX,
                  const __grid_constant__ CUtensorMap tmU, float* __restrict__ y, const __grid_constant__ FcArgs args,
                  int* __restrict__ status) {
  using Cfg = Fc32<M, R, ROWS>;
  constexpr int N = Cfg::N, NB = Cfg::NB, ST = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
  FcRec* rec = reinterpret_cast<FcRec*>(smem + Cfg::kOffRec);
  uint64_t* u_full = reinterpret_cast<uint64_t*>(smem + Cfg::kOffBar);
  uint64_t* u_free = u_full + ST;
  uint64_t* x_full = u_free + ST;
  uint64_t* x_free = x_full + 1;
  uint64_t* v_full = x_free + 1;          // [2]
  uint64_t* v_free = v_full + 2;          // [2]
  volatile int* abort_flag = reinterpret_cast<volatile int*>(v_free + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = args.split;
  const unsigned rank = split > 1 ? blockIdx.x % (unsigned)split : 0u;      // the CTA's rank in its cluster
  const unsigned first = blockIdx.x / (unsigned)split, stride = gridDim.x / (unsigned)split;
  const int my_chunks = (args.chunks - (int)rank + split - 1) / split;
  const int f_run = 8 * args.nb * Cfg::NH;

  if (threadIdx.x == 32) { tma_prefetch(&tmX); tma_prefetch(&tmU); }
  if (threadIdx.x == 0) {
    for (int i = 0; i < ST; ++i) { mbar_init(&u_full[i], 1); mbar_init(&u_free[i], Cfg::kProductWarps); }
    mbar_init(x_full, 1);
    mbar_init(x_free, Cfg::kTransformWarps);
    for (int i = 0; i < 2; ++i) { mbar_init(&v_full[i], Cfg::kTransformWarps); mbar_init(&v_free[i], Cfg::kProductWarps); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  pdl_wait();
  pdl_launch_dependents();

  if (warp < Cfg::kProductWarps) {
    // ================= product warps
    if constexpr (Cfg::kProductRegs > Cfg::kLaunchRegs) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(Cfg::kProductRegs));
    const int nu = warp % N, h = warp / N;
    const int g = lane >> 2, t = lane & 3;
    const uint32_t va = smem_u32(smem + Cfg::kOffV) + (uint32_t)((nu * kTiles + g) * kRowBytes + t * 16);
    const uint32_t ua = smem_u32(smem + Cfg::kOffU) + (uint32_t)((nu * f_run + h * 8 * args.nb + g) * kRowBytes + t * 16);
    const uint32_t zb = smem_u32(smem + Cfg::kOffZ);
    uint32_t q = 0, it = 0;
    for (unsigned blk = first; blk < args.blocks; blk += stride, ++it) {
      Dbl2 acc[N][NB];
#pragma unroll
      for (int a = 0; a < N; ++a)
#pragma unroll
        for (int c = 0; c < NB; ++c) acc[a][c] = Dbl2{0.0, 0.0};
      for (int c = 0; c < my_chunks; ++c, ++q) {
        fc_wait(&v_full[q & 1], (q >> 1) & 1, abort_flag);
#pragma unroll
        for (int s = 0; s < N; ++s) {
          constexpr int kPer = N / ST;
          const int xi = row_of<N>(s), stage = s % ST;
          fc_wait(&u_full[stage], (q * kPer + s / ST) & 1, abort_flag);
          const float4 A = lds_f4(va + (q & 1) * Cfg::kVBytes + s * Cfg::kVRow);
          const uint32_t us = ua + stage * Cfg::kStage;
#pragma unroll
          for (int nb = 0; nb < NB; ++nb) {
            if (nb >= args.nb) break;
            const float4 B = lds_f4(us + nb * 8 * kRowBytes);
            mma884(acc[xi][nb], A.x, B.x);
            mma884(acc[xi][nb], A.y, B.y);
            mma884(acc[xi][nb], A.z, B.z);
            mma884(acc[xi][nb], A.w, B.w);
          }
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(&u_free[stage]);
            if (s == N - 1) mbar_arrive(&v_free[q & 1]);
          }
        }
      }
      // A^T along xi: sums of frequencies (., nu) -> column nu of the m output rows, in place
#pragma unroll
      for (int nb = 0; nb < NB; ++nb) {
        Dbl2 in[N], z[M];
#pragma unroll
        for (int a = 0; a < N; ++a) in[a] = acc[a][nb];
        at_apply<M, SYM, Dbl2, N>(cf, in, z);
#pragma unroll
        for (int i = 0; i < M; ++i) acc[i][nb] = z[i];
      }
      // row i of the columns: [nu][tile][filter], the 8-filter block XORed with the tile modulo 4 (banks)
      auto put_columns = [&](uint32_t base, int i) {
#pragma unroll
        for (int nb = 0; nb < NB; ++nb)
          if (nb < args.nb)
            sts_d2(base + (uint32_t)((nu * kTiles + g) * Cfg::F + ((((h * args.nb + nb) * 8) ^ ((g & 3) << 3)) + 2 * t)) * 8, acc[i][nb]);
      };
      auto product_sync = [] {
        __syncwarp();
        asm volatile("bar.sync 1, %0;" ::"n"(Cfg::kProductThreads) : "memory");
      };
      const int kb = (int)(blk % (unsigned)args.num_kb);
      const int fp_log = 31 - __clz(f_run >> 1);
      const int pairs = kTiles * (f_run >> 1);
      const FcRec* rc = rec + (it % kRecRing) * kTiles;
      if (split == 1) {
        if constexpr (Cfg::kZRows == 1) {
          static_assert(kTiles * Cfg::F / 2 <= Cfg::kProductThreads, "one (tile, filter pair) per thread");
          const int tl = threadIdx.x >> fp_log, fc = (threadIdx.x & ((f_run >> 1) - 1)) * 2;
          const int k = kb * f_run + fc;
#pragma unroll
          for (int i = 0; i < M; ++i) {
            const uint32_t zr = zb + (i & 1) * Cfg::kZRow;
            put_columns(zr, i);
            product_sync();
            if ((int)threadIdx.x < pairs && k < args.K) {
              const FcRec rt = rc[tl];
              Dbl2 in[N], yv[M];
#pragma unroll
              for (int a = 0; a < N; ++a) in[a] = lds_d2(zr + (uint32_t)((a * kTiles + tl) * Cfg::F + (fc ^ ((tl & 3) << 3))) * 8);
              at_apply<M, SYM, Dbl2, N>(cf, in, yv);
              put_row<M>(i, yv, y + rt.ybase + k, rt, args);
            }
          }
        } else {
#pragma unroll
          for (int i0 = 0; i0 < M; i0 += Cfg::kZRows) {
            product_sync();         // the rows before have been read
#pragma unroll
            for (int r = 0; r < Cfg::kZRows; ++r) put_columns(zb + r * Cfg::kZRow, i0 + r);
            product_sync();
            for (int u = threadIdx.x; u < pairs * Cfg::kZRows; u += Cfg::kProductThreads) {
              const int r = u >> (fp_log + 3), idx = u & (pairs - 1);
              const int tl = idx >> fp_log, fc = (idx & ((f_run >> 1) - 1)) * 2;
              const int k = kb * f_run + fc;
              if (k >= args.K) continue;
              const FcRec rt = rc[tl];
              Dbl2 in[N], yv[M];
#pragma unroll
              for (int a = 0; a < N; ++a)
                in[a] = lds_d2(zb + (uint32_t)r * Cfg::kZRow + (uint32_t)((a * kTiles + tl) * Cfg::F + (fc ^ ((tl & 3) << 3))) * 8);
              at_apply<M, SYM, Dbl2, N>(cf, in, yv);
              put_row<M>(i0 + r, yv, y + rt.ybase + k, rt, args);
            }
          }
        }
      } else {
        // the cluster's CTAs hold the sums of different channels: all rows to shared memory (over the operand
        // buffers, which no one reads any more), then each CTA adds and finishes its share of the outputs
        const uint32_t z0 = smem_u32(smem);
        product_sync();
#pragma unroll
        for (int i = 0; i < M; ++i) put_columns(z0 + i * Cfg::kZRow, i);
        cluster_sync();
        const int units = pairs * M;
        for (int u = (int)rank * Cfg::kProductThreads + threadIdx.x; u < units; u += split * Cfg::kProductThreads) {
          const int i = u / pairs, idx = u % pairs;
          const int tl = idx >> fp_log, fc = (idx & ((f_run >> 1) - 1)) * 2;
          const int k = kb * f_run + fc;
          if (k >= args.K) continue;
          const FcRec rt = rc[tl];
          Dbl2 in[N], yv[M];
#pragma unroll
          for (int a = 0; a < N; ++a) in[a] = Dbl2{0.0, 0.0};
          for (int s = 0; s < split; ++s) {
            const uint32_t pz = peer_addr(z0 + (uint32_t)i * Cfg::kZRow + (uint32_t)(tl * Cfg::F + (fc ^ ((tl & 3) << 3))) * 8, (uint32_t)s);
#pragma unroll
            for (int a = 0; a < N; ++a) in[a] = vadd(in[a], lds_peer_d2(pz + (uint32_t)(a * kTiles * Cfg::F) * 8));
          }
          at_apply<M, SYM, Dbl2, N>(cf, in, yv);
          put_row<M>(i, yv, y + rt.ybase + k, rt, args);
        }
        cluster_sync();                    // nobody leaves while another CTA still reads its sums
      }
    }
  } else if (warp < Cfg::kProductWarps + Cfg::kTransformWarps) {
    // ================= transform warps
    if constexpr (Cfg::kTransformRegs > Cfg::kLaunchRegs) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(Cfg::kTransformRegs));
    else asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Cfg::kTransformRegs));
    const int tid = (threadIdx.x - Cfg::kProductThreads) & 127;
    const int share = (threadIdx.x - Cfg::kProductThreads) >> 7;
    const int ch = tid & 15, tl = tid >> 4, odd = tl & 1;
    uint32_t q = 0;
    for (unsigned blk = first; blk < args.blocks; blk += stride)
      for (int c = 0; c < my_chunks; ++c, ++q) {
        fc_wait(x_full, q & 1, abort_flag);
        // the two tiles of a warp lie a multiple of 128 bytes apart: the upper half warp reads the
        // columns of a pair in the other order, so that the halves use different banks
        const uint32_t xe = smem_u32(smem + Cfg::kOffX) + (uint32_t)(tl * Cfg::kXTile + ch * 4 + odd * kRowBytes);
        const uint32_t xo = xe - 2 * odd * kRowBytes;
        float raw[N * N];
#pragma unroll
        for (int a = 0; a < N; ++a)
#pragma unroll
          for (int b = 0; b < N; b += 2) {
            const float w0 = lds_f1(xe + (a * N + b) * kRowBytes), w1 = lds_f1(xo + (a * N + b + 1) * kRowBytes);
            raw[a * N + b] = odd ? w1 : w0;
            raw[a * N + b + 1] = odd ? w0 : w1;
          }
        __syncwarp();
        if (lane == 0) mbar_arrive(x_free);
        fc_wait(&v_free[q & 1], ((q >> 1) & 1) ^ 1, abort_flag);
        const uint32_t dst = smem_u32(smem + Cfg::kOffV) + (q & 1) * Cfg::kVBytes + (uint32_t)(tl * kRowBytes + ch * 4);
        if (Cfg::kShares == 1 || share == 0) {
          v_row_pair<N, SYM, 0>(cf, raw, dst, Cfg::kVRow);
          if constexpr (N == 8) v_row_pair<N, SYM, 1>(cf, raw, dst, Cfg::kVRow);
        }
        if (Cfg::kShares == 1 || share == 1) {
          if constexpr (N < 8) v_row_pair<N, SYM, 1>(cf, raw, dst, Cfg::kVRow);
          if constexpr (N >= 6) v_row_pair<N, SYM, 2>(cf, raw, dst, Cfg::kVRow);
          if constexpr (N >= 8) v_row_pair<N, SYM, 3>(cf, raw, dst, Cfg::kVRow);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&v_full[q & 1]);
      }
    if (split > 1) { cluster_sync(); cluster_sync(); }
  } else {
    // ================= producer warps
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Cfg::kProducerRegs));
    const int pw = warp - Cfg::kProductWarps - Cfg::kTransformWarps;
    if (pw == 0) {
      uint32_t q = 0;
      const uint32_t bytes = (uint32_t)(N * f_run * kRowBytes);
      for (unsigned blk = first; blk < args.blocks; blk += stride) {
        const int kb = (int)(blk % (unsigned)args.num_kb);
        for (int c = 0; c < my_chunks; ++c, ++q) {
          const int c0 = ((int)rank + c * split) * kChunk;
#pragma unroll 1
          for (int s = 0; s < N; ++s) {
            constexpr int kPer = N / ST;
            const int stage = s % ST;
            fc_wait(&u_free[stage], ((q * kPer + s / ST) & 1) ^ 1, abort_flag);
            if (lane == 0 && !*abort_flag) {
              mbar_expect_tx(&u_full[stage], bytes);
              tma_load_3d(smem + Cfg::kOffU + stage * Cfg::kStage, &tmU, &u_full[stage], c0, kb * f_run, row_of<N>(s) * N);
            }
            __syncwarp();
          }
        }
      }
    } else if (pw == 1) {
      uint32_t q = 0, it = 0;
      for (unsigned blk = first; blk < args.blocks; blk += stride, ++it) {
        const long long pb = (long long)(blk / (unsigned)args.num_kb) * kTiles;
        const bool live = lane < kTiles && pb + lane < args.P;
        const uint32_t p = (uint32_t)(pb + lane);                // 2^32 tiles of 8 channels do not fit any memory
        const uint32_t tw = p % (uint32_t)args.Tw, r = p / (uint32_t)args.Tw, th = r % (uint32_t)args.Th, img = r / (uint32_t)args.Th;
        const int n_live = (int)(args.P - pb < kTiles ? args.P - pb : kTiles);
        for (int c = 0; c < my_chunks; ++c, ++q) {
          const int c0 = ((int)rank + c * split) * kChunk;
          fc_wait(x_free, (q & 1) ^ 1, abort_flag);
          if (c == 0 && lane < kTiles) {
            FcRec o = {0, 0, 0};
            if (live) {
              const int h0 = M * (int)th, w0 = M * (int)tw;
              o.ybase = (((long long)img * args.H + h0) * args.W + w0) * args.K;
              o.rows = min(M, args.H - h0);
              o.cols = min(M, args.W - w0);
            }
            rec[(it % kRecRing) * kTiles + lane] = o;
          }
          __syncwarp();
          const bool go = !*abort_flag;
          if (lane == 0 && go) mbar_expect_tx(x_full, (uint32_t)(n_live * Cfg::kXTile));
          __syncwarp();
          if (live && go)
            tma_load_4d(smem + Cfg::kOffX + lane * Cfg::kXTile, &tmX, x_full, c0, M * (int)tw - Cfg::PAD, M * (int)th - Cfg::PAD, (int)img);
          __syncwarp();
        }
      }
    }
    if (split > 1) { cluster_sync(); cluster_sync(); }
  }
  if (*abort_flag) {
    if (lane == 0) atomicExch(status, NOVA_ERR_DEVICE_TIMEOUT);
    settle_after_timeout();
  }
}

// Tiles whose split blocks have a kernel of their own (see kZRows).
template <int M, int R>
constexpr bool split_by_rows() { return M + R - 1 == 6 && M > 2; }

// setmaxnreg draws on the registers the block was launched with: a build whose register count is not what the split was
// computed for does without this kernel.
template <int M, int R, bool SYM, bool ROWS = false>
bool built() {
  static const int regs = [] {
    cudaFuncAttributes at;
    return cudaFuncGetAttributes(&at, fused_fp32_kernel<M, R, SYM, ROWS>) == cudaSuccess ? at.numRegs : 0;
  }();
  if constexpr (split_by_rows<M, R>() && !ROWS)
    if (!built<M, R, SYM, true>()) return false;
  return regs >= Fc32<M, R, ROWS>::kLaunchRegs;
}

template <int M, int R, bool SYM, bool ROWS>
int go(const nova_plan* plan, const Geom& g, const void* x, const void* U, void* y, int relu, int nb, int split,
       cudaStream_t stream) {
  using Cfg = Fc32<M, R, ROWS>;
  EncodeTiledFn enc = tensor_map_encoder();
  if (!enc) return (int)cudaErrorUnknown;
  auto kernel = fused_fp32_kernel<M, R, SYM, ROWS>;
  if (!built<M, R, SYM, ROWS>()) return (int)cudaErrorInvalidConfiguration;
  const int f_run = 8 * nb * Cfg::NH;
  CUtensorMap tmX, tmU;
  cuuint32_t estr[4] = {1, 1, 1, 1};
  {
    cuuint64_t dims[4] = {(cuuint64_t)g.C, (cuuint64_t)g.W, (cuuint64_t)g.H, (cuuint64_t)g.N};
    cuuint64_t strides[3] = {(cuuint64_t)g.C * 4, (cuuint64_t)g.W * g.C * 4, (cuuint64_t)g.H * g.W * g.C * 4};
    cuuint32_t box[4] = {kChunk, (cuuint32_t)Cfg::N, (cuuint32_t)Cfg::N, 1};
    if (enc(&tmX, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void*>(x), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return (int)cudaErrorUnknown;
  }
  {
    cuuint64_t dims[3] = {(cuuint64_t)g.C, (cuuint64_t)g.K, (cuuint64_t)Cfg::NF};
    cuuint64_t strides[2] = {(cuuint64_t)g.C * 4, (cuuint64_t)g.K * g.C * 4};
    cuuint32_t box[3] = {kChunk, (cuuint32_t)f_run, (cuuint32_t)Cfg::N};
    if (enc(&tmU, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(U), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return (int)cudaErrorUnknown;
  }
  if (cudaError_t e = allow_dynamic_smem<Cfg::kTotal>(kernel); e != cudaSuccess) return (int)e;
  FcArgs a;
  a.H = g.H; a.W = g.W; a.K = g.K; a.Th = g.Th; a.Tw = g.Tw;
  a.P = g.P;
  a.chunks = (g.C + kChunk - 1) / kChunk;
  a.num_kb = (g.K + f_run - 1) / f_run;
  a.nb = nb; a.split = split; a.relu = relu;
  a.blocks = (unsigned)((g.P + kTiles - 1) / kTiles * a.num_kb);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(split > 1 ? a.blocks * split : (a.blocks < (unsigned)plan->sm_count ? a.blocks : (unsigned)plan->sm_count));
  cfg.blockDim = dim3(Cfg::kThreads);
  cfg.dynamicSmemBytes = Cfg::kTotal;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)split;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = split > 1 ? 2 : 1;
  return (int)cudaLaunchKernelEx(&cfg, kernel, plan->kcoefs_d, tmX, tmU, (float*)y, a, plan->status_dev);
}

// Filters per block and channel split.  Wide blocks transform x less often, narrow ones and clusters reach
// more SMs; the estimate is rounds of blocks x (chunks x time per chunk + time for the end of a block), in
// units of 10 ns fitted to B200 timings of 12 layers, with the end of a block by single rows.  With the present one the
// choice is still within 2 % of the best of all in 90 of 94 random layers, 4 % in 92 (the others: F(2,3) 2 x 12 x 28, 184 -> 248 34.7 / 31.9
// us, F(6,3), asymmetric, 5 x 15 x 28, 24 -> 80 22.0 / 17.5).  Clusters of 4: 33 fit the chip at once; of 8, fewer than 16
// do, and they lost on every layer tried (14 x 14, 256 -> 256, F(4,3): 13.5 us with 4, 27.7 us with 8).
// Measured against the three kernels before, whole call: F(4,3) 8 images 56 x 56, 64 -> 64: 82.5 -> 33.9 us;
// F(2,3) 16 x 16, 8 -> 8: 10.6 -> 3.4; F(6,3) 112 x 112, 64 -> 64: 49.3 -> 24.6; F(4,3) 14 x 14, 512 -> 512:
// 113 -> 29.5; F(6,3), asymmetric set, 2 x 28 x 28, 128 -> 128: 33.6 -> 31.8.
void choose_blocks(int n, const Geom& g, int sms, int* nb_out, int* split_out) {
  struct Cost { int chunk, end; };
  static const Cost kCost[3][3] = {{{83, 30}, {106, 40}, {0, 0}},          // n = 4: 8-filter blocks per warp 1, 2
                                   {{161, 166}, {213, 190}, {0, 0}},       // n = 6
                                   {{240, 400}, {280, 500}, {350, 700}}};  // n = 8: 1, 2, 4
  const int nh = n == 8 ? 1 : 2;
  const long long chunks = (g.C + kChunk - 1) / kChunk, tiles = (g.P + kTiles - 1) / kTiles;
  long long best = -1;
  for (int split = 1; split <= 4; split *= 2) {
    if (split > chunks) break;
    long long slots = split == 1 ? sms : split == 2 ? sms / 2 - 2 : sms / 4 - 4;
    if (slots < 1) slots = 1;
    for (int e = 0; e < (n == 8 ? 3 : 2); ++e) {
      const int f = (8 << e) * nh;
      const long long blocks = tiles * ((g.K + f - 1) / f);
      const Cost& c = kCost[n / 2 - 2][e];
      const long long t = (blocks + slots - 1) / slots * ((chunks + split - 1) / split * c.chunk + c.end + (split > 1 ? 60 * split : 0));
      if (best < 0 || t < best) { best = t; *nb_out = 1 << e; *split_out = split; }
    }
  }
}

}  // namespace

bool fused_fp32_applies(const nova_plan* plan) {
  if (plan->mode != NOVA_FP32 || plan->n > 8) return false;
  if (plan->device < 0) return true;                   // plans made without a device only answer questions
  const int key = plan->r * 10 + plan->m;
  const bool sym = plan->symmetric != 0;
  switch (key) {
    case 32: return sym ? built<2, 3, true>() : built<2, 3, false>();
    case 34: return sym ? built<4, 3, true>() : built<4, 3, false>();
    case 36: return sym ? built<6, 3, true>() : built<6, 3, false>();
    case 52: return sym ? built<2, 5, true>() : built<2, 5, false>();
    case 54: return sym ? built<4, 5, true>() : built<4, 5, false>();
  }
  return false;
}

int launch_fused_fp32(const nova_plan* plan, const Geom& g, const void* x, const void* U, void* y, int relu, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  int nb = 1, split = 1;
  choose_blocks(plan->n, g, plan->sm_count, &nb, &split);
#define NOVA_FC32(MV, RV)                                                                                            \
  do {                                                                                                                 \
    if constexpr (split_by_rows<MV, RV>())                                                                             \
      if (split > 1)                                                                                                   \
        return plan->symmetric ? go<MV, RV, true, true>(plan, g, x, U, y, relu, nb, split, s)                          \
                               : go<MV, RV, false, true>(plan, g, x, U, y, relu, nb, split, s);                        \
    return plan->symmetric ? go<MV, RV, true, false>(plan, g, x, U, y, relu, nb, split, s)                             \
                           : go<MV, RV, false, false>(plan, g, x, U, y, relu, nb, split, s);                           \
  } while (0)
  if (plan->r == 3) {
    if (plan->m == 2) NOVA_FC32(2, 3);
    if (plan->m == 4) NOVA_FC32(4, 3);
    if (plan->m == 6) NOVA_FC32(6, 3);
  } else if (plan->r == 5) {
    if (plan->m == 2) NOVA_FC32(2, 5);
    if (plan->m == 4) NOVA_FC32(4, 5);
  }
#undef NOVA_FC32
  return (int)cudaErrorInvalidValue;
}

}  // namespace nova
