// Layers of few tiles and few channels in half mode, where three dependent kernels cost their two boundaries and little else:
//   few_tiles_kernel      product and output transform (Section 2.1 steps 3 and 4) in one kernel after the input transform;
//   few_tiles_n4_kernel   with 4 points (F(2,3)) the input transform too.
// A CTA owns 16 tiles x KB filters and ALL frequencies of them: warp (xi, h) the row xi of frequencies for its share of the
// filters.  No CTA waits for another one, and M goes no further than registers and shared memory.
//
// What bounds it: latency.  A warp's step (64 channels of one frequency: ldmatrix, 4 to 16 mma.sync, the copies of a later
// step) is a chain that one or two warps per scheduler do not hide: F(4,3), 8 x 56 x 56, 64 -> 64, 12.0 us by itself with 45 % of the
// issue slots and 12 % of the tensor pipe used; a contraction of nothing but such steps makes some 270 multiply-adds per clock
// and SM, where tcgen05 makes 4096.  And U, which every block of 16 tiles fetches again.  So it is for layers whose work per
// CTA is a few dozen of these steps; which ones, and figures: see few_tiles_blocks.
//
// V and U are contracted in the same groups of 16 channels as by tcgen05.mma.  Nothing documented says that both instructions
// add such a group alike; on every input tried they do, to the bit (unit normals, values spread over 18 powers of two,
// subnormals, cancelling channels: the tests).  The transforms' arithmetic and its order are the three-kernel path's.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "nova_internal.h"
#include "output_math.cuh"
#include "sm100.cuh"
#include "tma_host.h"
#include "transform_math.cuh"

namespace nova {
namespace {
using namespace sm100;
using namespace xf;

constexpr int kT = 16;                 // tiles of a block: the rows of one mma
constexpr int kRow = 128;              // bytes of a row of operands: 64 channels

struct FtRec {                         // a tile: where its patch and its outputs are, which rows and columns exist
  long long xbase, ybase;
  int yrows, ycols;                    // outputs inside the image; yrows = 0 for a tile past the end
  unsigned xrows, xcols;               // patch rows and columns inside the image, as bits
};
struct FtArgs {
  int H, W, C, K, Th, Tw, relu, num_kb, pc, pc_pad;
  long long p0;
};

template <int M, int R, int HW, int NB>
struct FtCfg {
  static constexpr int N = M + R - 1;
  static constexpr int KB = 8 * NB * HW;                   // filters of a block
  static constexpr int kThreads = 32 * N * HW;
  static constexpr int kStage = (kT + 8 * NB) * kRow;      // V and U of one frequency and 64 channels
  static constexpr int kStages = 4;
  static constexpr int kZPitch = KB + 8;                   // floats; a quarter of the banks from row to row
  static constexpr int kZPlane = kT * kZPitch * 4;
  static constexpr int kZBytes = N * M * kZPlane;
  static constexpr int kRing = N * HW * kStages * kStage;
  static constexpr int kOffRec = kRing > kZBytes ? kRing : kZBytes;
  static constexpr int kTotal = kOffRec + kT * (int)sizeof(FtRec) + 128;
  static_assert(kTotal <= 227 * 1024, "shared memory of one CTA");
};

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix4(uint32_t a, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldmatrix2(uint32_t a, uint32_t& r0, uint32_t& r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(a) : "memory");
}
// 16 bytes to shared memory, or 16 zero bytes (nothing is read then)
__device__ __forceinline__ void copy16(uint32_t d, const void* p, bool there) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(p), "r"(there ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory"); }
__device__ __forceinline__ void sts_f32x2(uint32_t a, float2 v) { asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory"); }
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

template <int M, int R>
__device__ __forceinline__ void make_record(FtRec* rec, const FtArgs& a, int t0) {
  constexpr int N = M + R - 1, PAD = (R - 1) / 2;
  if (threadIdx.x >= kT) return;
  FtRec o = {0, 0, 0, 0, 0u, 0u};
  if (t0 + (int)threadIdx.x < a.pc) {
    const unsigned p = (unsigned)(a.p0 + t0 + threadIdx.x), tw = p % (unsigned)a.Tw, q = p / (unsigned)a.Tw;
    const unsigned th = q % (unsigned)a.Th, img = q / (unsigned)a.Th;
    const int h0 = M * (int)th, w0 = M * (int)tw;
    o.xbase = (((long long)img * a.H + (h0 - PAD)) * a.W + (w0 - PAD)) * a.C;
    if (a.relu & 2) {                  // y is [N, H/2, W/2, K]
      o.ybase = (((long long)img * (a.H >> 1) + (h0 >> 1)) * (a.W >> 1) + (w0 >> 1)) * a.K;
      o.yrows = (a.H >> 1) - (h0 >> 1);
      o.ycols = (a.W >> 1) - (w0 >> 1);
    } else {
      o.ybase = (((long long)img * a.H + h0) * a.W + w0) * a.K;
      o.yrows = a.H - h0;
      o.ycols = a.W - w0;
    }
    for (int i = 0; i < N; ++i) {
      o.xrows |= (unsigned)(h0 - PAD + i) < (unsigned)a.H ? 1u << i : 0u;
      o.xcols |= (unsigned)(w0 - PAD + i) < (unsigned)a.W ? 1u << i : 0u;
    }
  }
  rec[threadIdx.x] = o;
}

// The operands of one frequency and 64 channels (rows of 128 bytes, the 16-byte piece XORed with the row modulo 8)
// into the sums of 16 tiles x 8 * NB filters.
template <int NB>
__device__ __forceinline__ void contract(float (&acc)[NB][4], uint32_t v, uint32_t u) {
  const int lane = threadIdx.x & 31;
  const uint32_t x = (uint32_t)(lane & 7), ha = (uint32_t)(lane >> 4), hb = (uint32_t)((lane >> 3) & 1);
  const uint32_t va = v + (uint32_t)(lane & 15) * kRow, ua = u + (uint32_t)((lane & 7) + (NB > 1 ? (lane >> 4) << 3 : 0)) * kRow;
  uint32_t A[4][4], B[4][NB][2];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    ldmatrix4(va + (((2 * s + ha) ^ x) << 4), A[s][0], A[s][1], A[s][2], A[s][3]);
    if constexpr (NB == 1) {
      ldmatrix2(ua + (((2 * s + hb) ^ x) << 4), B[s][0][0], B[s][0][1]);
    } else {
#pragma unroll
      for (int k = 0; k < NB; k += 2)
        ldmatrix4(ua + (uint32_t)k * 8 * kRow + (((2 * s + hb) ^ x) << 4), B[s][k][0], B[s][k][1], B[s][k + 1][0], B[s][k + 1][1]);
    }
  }
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int k = 0; k < NB; ++k) mma16816(acc[k], A[s], B[s][k][0], B[s][k][1]);
}

// z_xi[j] of one (tile, filter pair)
template <int M, int R, int KB>
struct ZRows {
  static constexpr int kPlane = kT * (KB + 8) * 4;
  uint32_t base;
  template <int XI, int J>
  __device__ __forceinline__ void fill(float2 (&z)[M]) const {
    if constexpr (J < M) {
      z[J] = lds_f32x2<(XI * M + J) * kPlane>(base);
      fill<XI, J + 1>(z);
    }
  }
  template <int XI>
  __device__ __forceinline__ void row(float2 (&z)[M]) const { fill<XI, 0>(z); }
};

// A^T along nu on a warp's row of sums, the rows meet in shared memory (over the operands, which no one reads any more),
// A^T along xi, y.
template <int M, int R, bool SYM, int HW, int NB>
__device__ __forceinline__ void finish(const Coefs& cf, const float (&acc)[M + R - 1][NB][4], uint32_t sz, int xi, int h, const FtRec* rec, int kb,
                                       __half* y, const FtArgs& a) {
  using Cfg = FtCfg<M, R, HW, NB>;
  constexpr int N = Cfg::N, KB = Cfg::KB;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NB; ++k)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float2 in[N], z[M];
#pragma unroll
      for (int nu = 0; nu < N; ++nu) in[nu] = make_float2(acc[nu][k][2 * e], acc[nu][k][2 * e + 1]);
      at_apply<M, SYM, float2, N>(cf, in, z);
      const uint32_t d = sz + (uint32_t)((xi * M * kT + e * 8 + g) * Cfg::kZPitch + (h * NB + k) * 8 + 2 * t) * 4;
#pragma unroll
      for (int j = 0; j < M; ++j) sts_f32x2(d + j * Cfg::kZPlane, z[j]);
    }
  __syncthreads();
  for (int i = threadIdx.x; i < kT * KB / 2; i += Cfg::kThreads) {
    const int tl = i / (KB / 2), fl = i % (KB / 2) * 2, k = kb * KB + fl;
    const FtRec r = rec[tl];
    if (k >= a.K || r.yrows == 0) continue;
    float2 Y[M][M];
    accumulate_rows<M, SYM, float2, N>(cf, ZRows<M, R, KB>{sz + (uint32_t)(tl * Cfg::kZPitch + fl) * 4}, Y);
    if (a.relu & 2)
      store_tile_pooled<M, __half>(Y, y + r.ybase + k, (size_t)(a.W >> 1) * a.K, a.K, r.yrows, r.ycols, a.relu & 1);
    else
      store_tile<M, __half>(Y, y + r.ybase + k, (size_t)a.W * a.K, a.K, r.yrows, r.ycols, a.relu & 1);
  }
}

// Product and output transform.  Each warp has a ring of its own, which it fills and reads: no barrier in the loop.
template <int M, int R, bool SYM, int NB>
__global__ void __launch_bounds__(FtCfg<M, R, 1, NB>::kThreads, 1)
few_tiles_kernel(const __grid_constant__ Coefs cf, const __half* V, const __half* U, __half* y, const __grid_constant__ FtArgs a) {
  using Cfg = FtCfg<M, R, 1, NB>;
  constexpr int N = Cfg::N, S = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
  FtRec* rec = reinterpret_cast<FtRec*>(smem + Cfg::kOffRec);
  const int xi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kb = (int)(blockIdx.x % (unsigned)a.num_kb), t0 = (int)(blockIdx.x / (unsigned)a.num_kb) * kT;
  const uint32_t ring = smem_u32(smem) + (uint32_t)(xi * (S * Cfg::kStage));
  const int chunks = (a.C + 63) >> 6, steps = N * chunks;
  // loads: 4 rows x 8 pieces of 16 bytes per instruction
  constexpr int LV = kT / 4, LU = 2 * NB;
  const int lr = lane >> 3, lc = lane & 7, kw = kb * Cfg::KB;
  const size_t ufs = (size_t)a.K * a.C * 2, vfs = (size_t)a.pc_pad * a.C * 2;          // from frequency to frequency
  const char* pv = reinterpret_cast<const char*>(V + (size_t)(xi * N) * a.pc_pad * a.C + (size_t)(t0 + lr) * a.C + lc * 8);
  const char* pu = reinterpret_cast<const char*>(U + (size_t)(xi * N) * a.K * a.C + (size_t)(kw + lr) * a.C + lc * 8);
  const size_t row4 = (size_t)a.C * 8;                                                 // four rows
  const uint32_t d0 = ring + lr * kRow + (uint32_t)((lc ^ lr) << 4), d1 = ring + lr * kRow + (uint32_t)((lc ^ (lr + 4)) << 4);
  uint32_t okv = 0, oku = 0;
#pragma unroll
  for (int i = 0; i < LV; ++i) okv |= (t0 + i * 4 + lr < a.pc ? 1u : 0u) << i;
#pragma unroll
  for (int i = 0; i < LU; ++i) oku |= (kw + i * 4 + lr < a.K ? 1u : 0u) << i;
  const int c_end = a.C - (chunks - 1) * 64 > lc * 8 ? chunks : chunks - 1;            // chunks in which this lane's piece exists
  auto fetch_v = [&](const char* p, bool okc, uint32_t st) {
#pragma unroll
    for (int i = 0; i < LV; ++i) {
      const bool ok = okc && (okv >> i & 1u);
      copy16(((i & 1) ? d1 : d0) + st + i * 512, ok ? p + i * row4 : (const char*)V, ok);
    }
  };
  auto fetch_u = [&](const char* p, bool okc, uint32_t st) {
#pragma unroll
    for (int i = 0; i < LU; ++i) {
      const bool ok = okc && (oku >> i & 1u);
      copy16(((i & 1) ? d1 : d0) + st + kT * kRow + i * 512, ok ? p + i * row4 : (const char*)U, ok);
    }
  };
  make_record<M, R>(rec, a, t0);
  // The first stages' U does not wait for the input transform, which lets this kernel start only after its own wait, when
  // everything before it has completed.
  {
    int c = 0;
    const char *q0 = pu, *q = pu;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      if (s < steps) fetch_u(q, c < c_end, s * Cfg::kStage);
      q += kRow;
      if (++c == chunks) { c = 0; q0 += ufs; q = q0; }
    }
  }
  pdl_launch_dependents();
  pdl_wait();
  int fc = 0;                                              // the next load: its chunk, its addresses
  const char *qv0 = pv, *qu0 = pu, *qv = pv, *qu = pu;
  auto advance = [&] {
    qv += kRow;
    qu += kRow;
    if (++fc == chunks) { fc = 0; qv0 += vfs; qu0 += ufs; qv = qv0; qu = qu0; }
  };
#pragma unroll
  for (int s = 0; s < S; ++s) {
    if (s < steps) fetch_v(qv, fc < c_end, s * Cfg::kStage);
    copy_commit();
    advance();
  }
  float acc[N][NB][4];
  int left = steps - S;
  uint32_t st = 0;
#pragma unroll
  for (int nu = 0; nu < N; ++nu) {
#pragma unroll
    for (int k = 0; k < NB; ++k)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[nu][k][e] = 0.f;
#pragma unroll 1
    for (int c = 0; c < chunks; ++c) {
      copy_wait<S - 1>();                                  // a group per step, in order
      __syncwarp();
      contract<NB>(acc[nu], ring + st, ring + st + kT * kRow);
      __syncwarp();
      if (left > 0) { fetch_u(qu, fc < c_end, st); fetch_v(qv, fc < c_end, st); }
      copy_commit();
      --left;
      advance();
      st = st == (S - 1) * Cfg::kStage ? 0u : st + Cfg::kStage;
    }
  }
  copy_wait<0>();
  finish<M, R, SYM, 1, NB>(cf, acc, smem_u32(smem), xi, 0, rec, kb, y, a);
}

// F(2,3): the input transform too.  A warp transforms two tiles of 64 channels at a time, a lane two channels, as
// input_transform_n4.cu does; the next 64 channels' patches are fetched while these are contracted.
template <int NB>
struct N4Cfg : FtCfg<2, 3, 2, NB> {
  using Base = FtCfg<2, 3, 2, NB>;
  static constexpr int kVF = kT * kRow;                    // V of one frequency
  static constexpr int kUF = 8 * NB * kRow;                // a warp's U of one frequency
  static constexpr int kOffU = 16 * kVF;
  static constexpr int kOffRec = kOffU + 8 * 4 * kUF;
  static constexpr int kTotal = kOffRec + kT * (int)sizeof(FtRec) + 128;
  static_assert(Base::kZBytes <= kOffRec, "the rows of sums fit over the operands");
};

// 128 registers, so that two CTAs share an SM, cost the kernel of 32 filters a block 76 bytes of spills (120 with dense transforms).
template <bool SYM, int NB>
__global__ void __launch_bounds__(256, 2)
few_tiles_n4_kernel(const __grid_constant__ Coefs cf, const __half* x, const __half* U, __half* y, const __grid_constant__ FtArgs a) {
  using Cfg = N4Cfg<NB>;
  constexpr int N = 4;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
  FtRec* rec = reinterpret_cast<FtRec*>(smem + Cfg::kOffRec);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int xi = warp & 3, h = warp >> 2;
  const int kb = (int)(blockIdx.x % (unsigned)a.num_kb), t0 = (int)(blockIdx.x / (unsigned)a.num_kb) * kT;
  const uint32_t sv = smem_u32(smem), su = sv + Cfg::kOffU + warp * (4 * Cfg::kUF);
  make_record<2, 3>(rec, a, t0);
  __syncthreads();
  pdl_wait();
  pdl_launch_dependents();

  // U: a group of copies per frequency of the row
  const int lr = lane >> 3, lc = lane & 7, kw = kb * Cfg::KB + h * 8 * NB;
  const size_t ufs = (size_t)a.K * a.C;
  const __half* pu = U + (size_t)(xi * N) * ufs + (size_t)(kw + lr) * a.C + lc * 8;
  auto fetch_u = [&](int nu, int c0) {
#pragma unroll
    for (int i = 0; i < 2 * NB; ++i) {
      const bool ok = kw + i * 4 + lr < a.K && c0 + lc * 8 < a.C;
      copy16(su + nu * Cfg::kUF + (uint32_t)((i * 4 + lr) * kRow + ((lc ^ ((i * 4 + lr) & 7)) << 4)),
             ok ? pu + nu * ufs + (size_t)(i * 4) * a.C + c0 : U, ok);
    }
    copy_commit();
  };
  uint32_t d[2][N][N];
  auto fetch_x = [&](int c0) {
    const int c = c0 + 2 * lane;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const FtRec r = rec[warp + 8 * e];
      const __half* p = x + r.xbase + c;
#pragma unroll
      for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) {
          d[e][i][j] = 0u;
          if (c < a.C && (r.xrows >> i & 1u) && (r.xcols >> j & 1u))
            d[e][i][j] = *reinterpret_cast<const uint32_t*>(p + ((long long)i * a.W + j) * a.C);
        }
    }
  };
  fetch_x(0);
#pragma unroll
  for (int nu = 0; nu < N; ++nu) fetch_u(nu, 0);
  float acc[N][NB][4];
#pragma unroll
  for (int nu = 0; nu < N; ++nu)
#pragma unroll
    for (int k = 0; k < NB; ++k)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[nu][k][e] = 0.f;
#pragma unroll 1
  for (int c0 = 0; c0 < a.C; c0 += 64) {
    if (c0) __syncthreads();                               // V of the previous channels has been read
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float2 t[N][N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        float2 in[N], out[N];
#pragma unroll
        for (int j = 0; j < N; ++j) in[j] = __half22float2(*reinterpret_cast<const __half2*>(&d[e][i][j]));
        bt_all_rows<N, SYM>(cf, in, out);
#pragma unroll
        for (int j = 0; j < N; ++j) t[j][i] = out[j];
      }
      const int tl = warp + 8 * e;
      const uint32_t dst = sv + (uint32_t)(tl * kRow + (((lane >> 2) ^ (tl & 7)) << 4) + (lane & 3) * 4);
#pragma unroll
      for (int nu = 0; nu < N; ++nu) {
        float2 out[N];
        bt_all_rows<N, SYM>(cf, t[nu], out);
#pragma unroll
        for (int q = 0; q < N; ++q) {
          const __half2 o = __floats2half2_rn(out[q].x, out[q].y);
          sts_u32(dst + (q * N + nu) * Cfg::kVF, *reinterpret_cast<const uint32_t*>(&o));
        }
      }
    }
    __syncthreads();
    const bool more = c0 + 64 < a.C;
    if (more) fetch_x(c0 + 64);
#pragma unroll
    for (int nu = 0; nu < N; ++nu) {
      copy_wait<N - 1>();                                  // a group per frequency, in order
      __syncwarp();
      contract<NB>(acc[nu], sv + (xi * N + nu) * Cfg::kVF, su + nu * Cfg::kUF);
      __syncwarp();
      if (more) fetch_u(nu, c0 + 64);
      else copy_commit();
    }
  }
  copy_wait<0>();
  finish<2, 3, SYM, 2, NB>(cf, acc, sv, xi, h, rec, kb, y, a);
}

FtArgs make_args(const Geom& g, long long p0, int pc, int pc_pad, int relu, int KB) {
  FtArgs a;
  a.H = g.H; a.W = g.W; a.C = g.C; a.K = g.K; a.Th = g.Th; a.Tw = g.Tw;
  a.relu = relu; a.num_kb = (g.K + KB - 1) / KB; a.pc = pc; a.pc_pad = pc_pad; a.p0 = p0;
  return a;
}

constexpr int kOwnSm = 120 * 1024;
// Shared memory that keeps two CTAs off one SM while another SM has none.  Without it CTAs that become resident while the
// input transform still runs share SMs: F(4,3), 4 x 97 x 37, 184 -> 16 21.1 / 12.9 us, 8 x 30 x 26, 176 -> 16 15.7 / 10.0, 8 x 28 x 28, 64 -> 64
// 7.7 / 7.0; F(6,3) 2 x 30 x 30, 64 -> 64 and F(2,3) 2 x 24 x 24, 128 -> 136 6.7 and 6.8 either way.
int own_sm(int bytes, int grid, int sms) { return bytes < kOwnSm && grid <= sms ? kOwnSm : bytes; }

template <int M, int R, bool SYM, int NB>
int go(const nova_plan* plan, const Geom& g, const void* V, const void* U, void* y, long long p0, int pc, int pc_pad, int relu, cudaStream_t s) {
  using Cfg = FtCfg<M, R, 1, NB>;
  const auto kernel = few_tiles_kernel<M, R, SYM, NB>;
  const FtArgs a = make_args(g, p0, pc, pc_pad, relu, Cfg::KB);
  const int grid = (pc + kT - 1) / kT * a.num_kb, smem = own_sm(Cfg::kTotal, grid, plan->sm_count);
  if (cudaError_t e = allow_dynamic_smem<(Cfg::kTotal > kOwnSm ? Cfg::kTotal : kOwnSm)>(kernel); e != cudaSuccess) return (int)e;
  return (int)launch_overlapped(kernel, grid, Cfg::kThreads, smem, s, plan->kcoefs, (const __half*)V, (const __half*)U, (__half*)y, a);
}
template <bool SYM, int NB>
int go_n4(const nova_plan* plan, const Geom& g, const void* x, const void* U, void* y, int relu, cudaStream_t s) {
  using Cfg = N4Cfg<NB>;
  const auto kernel = few_tiles_n4_kernel<SYM, NB>;
  if (cudaError_t e = allow_dynamic_smem<Cfg::kTotal>(kernel); e != cudaSuccess) return (int)e;
  const FtArgs a = make_args(g, 0, (int)g.P, (int)g.P, relu, Cfg::KB);
  const int grid = ((int)g.P + kT - 1) / kT * a.num_kb;
  return (int)launch_overlapped(kernel, grid, Cfg::kThreads, Cfg::kTotal, s, plan->kcoefs, (const __half*)x, (const __half*)U, (__half*)y, a);
}
template <int M, int R, int NB>
int go_sym(const nova_plan* plan, const Geom& g, const void* V, const void* U, void* y, long long p0, int pc, int pc_pad, int relu, cudaStream_t s) {
  return plan->symmetric ? go<M, R, true, NB>(plan, g, V, U, y, p0, pc, pc_pad, relu, s) : go<M, R, false, NB>(plan, g, V, U, y, p0, pc, pc_pad, relu, s);
}
template <int M, int R>
int go_nb(int nb, const nova_plan* plan, const Geom& g, const void* V, const void* U, void* y, long long p0, int pc, int pc_pad, int relu, cudaStream_t s) {
  switch (nb) {
    case 1: return go_sym<M, R, 1>(plan, g, V, U, y, p0, pc, pc_pad, relu, s);
    case 2: return go_sym<M, R, 2>(plan, g, V, U, y, p0, pc, pc_pad, relu, s);
    case 4: return go_sym<M, R, 4>(plan, g, V, U, y, p0, pc, pc_pad, relu, s);
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace

// The block of filters, in eights (1, 2 or 4), where these kernels are the faster ones; plus 10 where the input transform is in
// them; 0 elsewhere.  The line lies at the number of CTAs and ks = 64-channel pieces, which are steps of each warp.
// Whole call, kernels without a merged product / this rule, geometric mean over the layers that the rule takes of 220 random ones
// each, 1 .. 32 images of 7 .. 112 pixels with 16 .. 512 channels: n = 4 1.56x (147 layers, none slower), n = 6 1.32x (155, none
// slower), n = 8 1.28x (128, two slower: 100 tiles 80 -> 64 10.0 / 10.2, 50 tiles 120 -> 256 9.9 / 10.4).  Some of them (us):
//   n = 4, input transform included   100 tiles 32 -> 8 9.0 / 4.0, 684 tiles 64 -> 32 8.7 / 4.8, 2040 tiles 48 -> 64 11.5 / 7.2
//     up to 12 MB of M, which is product_output.cu's line (and none beyond it, should that kernel not be there): 5016 tiles 64 -> 32
//     15.1 / 10.1, 16 tiles 64 -> 8192 13.2 / 7.3, 182 tiles 64 -> 768 11.0 / 6.9
//     up to 16 filters in blocks of 16 however many tiles, three kernels / blocks of 32 / blocks of 16: 2808 tiles 24 -> 8 10.7 / 7.2 / 5.6,
//     7050 tiles 64 -> 16 17.3 / 10.4 / 8.8, 16896 tiles 56 -> 8 32.4 / 26.4 / 21.6
//     not where ragged rows of x are transformed densely for each of many blocks, more of them than two per SM: 361 tiles 56 -> 512
//     11.7 / 13.0, 960 tiles 40 -> 192 12.1 / 12.6, 648 tiles 24 -> 256 11.9 / 12.2; the same with symmetric points 11.6 / 11.4, 11.8 / 11.3,
//     11.7 / 10.8; 1406 tiles 56 -> 128 14.2 / 13.0; 160 tiles 24 -> 1024 12.3 / 11.7
//   n = 4, more channels              180 tiles 192 -> 32 9.0 / 6.5, 252 tiles 256 -> 16 8.9 / 7.1, 870 tiles 256 -> 72 12.7 / 12.7 (not taken)
//   n = 6, ks = 1                     36 tiles 64 -> 16 9.1 / 6.6, 1568 tiles 64 -> 64 14.1 / 12.2, 480 tiles 16 -> 512 19.1 / 21.3 (not taken)
//     between one and two blocks of 32 filters per SM, three kernels / blocks of 16 / blocks of 32: 3600 tiles 16 -> 16 18.2 / 11.1 / 15.0, 1404 tiles
//     32 -> 48 13.7 / 9.9 / 13.8, 1444 tiles 48 -> 64 14.4 / 13.1 / 14.4, 2312 tiles 16 -> 64 16.8 / 14.9 / 14.7, 528 tiles 32 -> 256 14.6 / 13.2 / 12.8,
//     2256 tiles 64 -> 64 16.4 / 14.3 / 14.2; ragged rows: 1250 tiles 40 -> 64 14.1 / 13.4 / 14.5, 2312 tiles 40 -> 64 19.9 / 18.1 / 17.6,
//     4416 tiles 56 -> 32 22.0 / 20.6 / 19.7, not taken 1764 tiles 24 -> 64 16.1 / 16.6 / 16.9, 363 tiles 24 -> 256 13.0 / 13.9 / 13.4, 1458 tiles
//     56 -> 64 14.3 / 16.3 / 15.5
//   n = 6, ks = 3                     200 tiles 176 -> 88 10.5 / 9.2, 1012 tiles 192 -> 16 13.6 / 11.1, 256 tiles 160 -> 64 9.8 / 9.3; ragged rows:
//     16 tiles 152 -> 256 9.0 / 8.2, 196 tiles 136 -> 16 9.9 / 9.5, 512 tiles 152 -> 16 11.4 / 10.9, 256 tiles 184 -> 32 9.8 / 10.1 (not taken), 98 tiles 184 -> 96 9.4 / 9.8 (not
//     taken): the three kernels pay for a third block of 128 tiles from 257 tiles on
//   n = 6, ks = 2                     60 tiles 128 -> 32 9.4 / 6.8, 513 tiles 128 -> 64 11.8 / 9.3, 828 tiles 104 -> 128 15.4 / 20.8 (not taken)
//   n = 8                             72 tiles 64 -> 24 9.1 / 6.5, 950 tiles 32 -> 32 14.8 / 10.6, 360 tiles 136 -> 32 14.5 / 15.4 (not taken)
//     two pieces of channels: 40 tiles 128 -> 256 10.1 / 8.4, 98 tiles 96 -> 32 9.0 / 8.7, 952 tiles 112 -> 24 17.0 / 14.5; ragged rows from 257 tiles on,
//     where the three kernels pay for a third block of 128, with many filters and up to 8 tiles: 288 tiles 120 -> 32 11.8 / 11.7, 676 tiles 104 -> 24
//     15.0 / 13.3, 98 tiles 104 -> 160 11.9 / 10.9, 25 tiles 88 -> 400 11.3 / 10.0, 4 tiles 104 -> 40 9.8 / 8.4; not taken 42 tiles 120 -> 48
//     9.1 / 10.2, 100 tiles 88 -> 32 9.0 / 9.5, 256 tiles 104 -> 64 10.8 / 11.2
// With 10 points a CTA's steps are too many (16 tiles 56 -> 80 10.6 / 10.8).
int few_tiles_blocks(const nova_plan* plan, const Geom& g) {
  if (plan->mode != NOVA_FP16_F32ACC || plan->n > 8 || !plan->status_dev || plan->sm_count < 64 || g.P > (1 << 20)) return 0;
  const long long sms = plan->sm_count, tb = (g.P + kT - 1) / kT;
  const int ks = (g.C + 63) / 64;
  const bool ragged = g.C % 16 != 0;                     // rows of channels that are not whole sectors of 32 bytes
  const long long c8 = tb * ((g.K + 7) / 8), c16 = tb * ((g.K + 15) / 16), c32 = tb * ((g.K + 31) / 32);
  if (plan->n == 4) {
    if (ks == 1) {
      if (64e-6 * (double)g.P * g.K >= 12) return 0;
      if (g.K <= 16 || c16 <= sms) return 11;
      return ragged && !plan->symmetric && c32 > 2 * sms && g.K > 128 && g.K < 1024 ? 0 : 12;
    }
    if (ks == 2) return c16 <= sms / 2 ? 11 : c32 <= sms ? 4 : 0;
    if (ks <= 4) return c16 <= sms ? 2 : c32 <= sms / 2 ? 4 : 0;
    return ks <= 6 && c8 <= sms / 2 ? 1 : 0;
  }
  if (plan->n == 6) {
    if (ks <= 2 && c8 <= sms / 2) return 1;
    if (ks <= 2 && (c16 <= sms || c32 <= sms)) return c16 <= sms ? 2 : 4;
    if (ks == 1 && c32 <= 2 * sms) {
      // two CTAs of 16 filters on an SM against one of 32
      const bool halves = c16 <= sms * 8 / 3;
      if (c16 <= 2 * sms) return 2;
      if (ragged && g.K > 40) return g.C > 40 ? 0 : halves && g.K <= 128 ? 2 : c32 > sms * 5 / 3 ? 4 : 0;
      return halves || g.C == 64 ? 2 : 4;
    }
    if (ks == 3) return c8 <= (!ragged || tb > 16 ? sms : tb <= 5 || g.C < 144 ? sms / 2 : 16) ? 1 : 0;
    return 0;
  }
  if (ks > 2 || (ks == 2 && ragged && tb <= 16 && g.P > 8 && (g.K < 160 || c8 < 64))) return 0;
  return c8 <= sms ? 1 : c16 <= sms ? 2 : ks == 1 && c32 <= sms ? 4 : 0;
}

int launch_few_tiles(const nova_plan* plan, const Geom& g, const void* V, const void* U, void* y, long long p0, int pc, int pc_pad, int relu,
                     int blocks8, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  switch (plan->r * 10 + plan->m) {
    case 32: return go_nb<2, 3>(blocks8, plan, g, V, U, y, p0, pc, pc_pad, relu, s);
    case 34: return go_nb<4, 3>(blocks8, plan, g, V, U, y, p0, pc, pc_pad, relu, s);
    case 36: return go_nb<6, 3>(blocks8, plan, g, V, U, y, p0, pc, pc_pad, relu, s);
    case 52: return go_nb<2, 5>(blocks8, plan, g, V, U, y, p0, pc, pc_pad, relu, s);
    case 54: return go_nb<4, 5>(blocks8, plan, g, V, U, y, p0, pc, pc_pad, relu, s);
  }
  return (int)cudaErrorInvalidValue;
}

int launch_few_tiles_n4(const nova_plan* plan, const Geom& g, const void* x, const void* U, void* y, int relu, int blocks8, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  if (blocks8 == 1) return plan->symmetric ? go_n4<true, 1>(plan, g, x, U, y, relu, s) : go_n4<false, 1>(plan, g, x, U, y, relu, s);
  return plan->symmetric ? go_n4<true, 2>(plan, g, x, U, y, relu, s) : go_n4<false, 2>(plan, g, x, U, y, relu, s);
}

}  // namespace nova
