// Section 2.1 steps 3 and 4 in ONE kernel for tiles of 4, 6 or 8 points: the transformed-domain product M[f] = V[f]
// U[f]^T on the tensor cores and the output transform Y = A^T M A, with M never leaving the chip.  Half operands, or
// the int8 pipeline's bytes (I8: int32 sums, dequantised before the transform).
//
// Why: M is n*n floats per (tile, filter); written and read back it is the largest tensor of the three-kernel
// pipeline, several times the L2 on the large layers and a kernel boundary on the small ones.  The n*n sums of 128
// tiles x 64 filters do not fit one SM's tensor memory, but those of one ROW xi of frequencies do: n accumulators of
// 64 columns.  So a cluster of n CTAs takes a block of 128 tiles x F filters, CTA xi computes the frequencies (xi, .),
// applies A^T along nu to them (n values become m), and the rows meet through distributed shared memory: the CTA
// that owns a group of 8 tiles receives their row results from all n CTAs, applies A^T along xi and stores y.
//
// What bounds it: the loads of V and U, n * (128 + F) * C elements per block and CTA (V is fetched once per F filters,
// which is why wide layers stay with the three kernels), and the exchange, 128 * F * m floats per CTA, (n-1)/n of it to
// other SMs.  Which layers take it, and figures: see use_product_output.
//
// Roles of a CTA (20, 24 or 28 warps at 8, 6 or 4 points, registers split by setmaxnreg):
//   warps 0, 3    TMA producers: [128 tiles][64 channels] boxes of V and [F filters][64 channels] boxes of U into a ring
//   warps 1, 2    tcgen05.mma (M = 128, N = F), accumulator nu at column nu * F; two sets of accumulators where 512
//                 columns hold them
//   warps 4-11    row transform, two groups that take alternate slices of 16 filters: tcgen05.ld of the n
//                 accumulators, A^T along nu, stores into the owner CTA's exchange buffers (two or four, in turn)
//   the rest      finish, two groups that take alternate slices, a warp per 4 of the CTA's own tiles: A^T along xi, y (or the
//                 pooled y)
// The arithmetic and its order are the three-kernel path's, so the results are the same bits.
// Every wait is bounded by the clock; after one has expired no role of the CTA waits any more and all run to their end.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "nova_internal.h"
#include "output_math.cuh"
#include "sm100.cuh"
#include "tma_host.h"

namespace nova {
namespace {
using namespace sm100;
using namespace xf;

constexpr int kRows = 128;             // tiles of a block: TMEM lanes
constexpr int kRowBytes = 128;         // one swizzle row of channels per stage: 64 halves or 128 int8
constexpr int kUmmaBytes = 32;
constexpr int kSliceF = 16;            // filters exchanged at a time
constexpr int kVBytes = kRows * kRowBytes;

template <int M, int R>
struct PoCfg {
  static constexpr int N = M + R - 1;
  static constexpr int kOct = (16 + N - 1) / N;                  // groups of 8 tiles a CTA owns, at most
  static constexpr int kSrc = kOct * M * 4 * 128;                // bytes one CTA sends another per slice
  static constexpr int kBuf = N * kSrc;
  static constexpr int kFinish = 2 * kOct;                       // finish warps per exchange buffer: one per 4 tiles
  static constexpr int kThreads = 32 * (4 + 8 + 2 * kFinish);    // 896, 768, 640
  // registers per thread; the split must not exceed what the block is launched with
  static constexpr int kLaunchRegs = (65536 / kThreads) / 8 * 8; // 72, 80, 96
  static constexpr int kIssueRegs = 40;
  static constexpr int kRowRegs = (N == 4) ? 72 : 88;
  static constexpr int kFinishRegs = (N == 4) ? 72 : (N == 6) ? 80 : 128;
  static_assert(128 * kIssueRegs + 256 * kRowRegs + 64 * kFinish * kFinishRegs <= kThreads * kLaunchRegs, "register split");
  static constexpr int kOffZ = 0;
  static_assert(2 * kBuf % 1024 == 0, "swizzled operands");
  // A stage holds the operands of two columns nu, one per MMA issuer; each issuer uses every stage, so that no one
  // gets two phases ahead of a barrier that it waits on by parity.
  static constexpr int stage_bytes(int F) { return 2 * (kVBytes + F * kRowBytes); }
  static constexpr int stages(int F, int bufs) {
    return (232448 - bufs * kBuf - 2048) / stage_bytes(F) < 4 ? (232448 - bufs * kBuf - 2048) / stage_bytes(F) : 4;
  }
  static constexpr int total(int F, int bufs) { return bufs * kBuf + stages(F, bufs) * stage_bytes(F) + 256 + 1024; }
  static constexpr int kMaxF = (N == 4) ? 64 : 32;               // see block_filters
  static constexpr int kMaxTotal = 227 * 1024;                   // stages() fills up to it, whatever F and the buffers
  static_assert(total(kMaxF, 2) <= kMaxTotal && total(kMaxF, 4) <= kMaxTotal && total(16, 2) <= kMaxTotal && total(16, 4) <= kMaxTotal &&
                total(32, 2) <= kMaxTotal && total(32, 4) <= kMaxTotal && stages(kMaxF, 2) >= 2, "shared memory of one CTA");
  // Exchange buffers: four for few channels, where the ring of operands can spare a stage.  With two, a row group waits for the
  // buffer that it filled a slice ago to be read in all CTAs.  Whole call, two / four: F(2,3) 32 x 56 x 56, 128 -> 128 75.1 / 69.8 us,
  // 32 x 112 x 112, 64 -> 64 135.7 / 131.9; F(4,3) 32 x 112 x 112, 64 -> 128 152.7 / 148.0, 64 -> 64 93.3 / 92.3, 8 x 112 x 112, 64 -> 256 73.6 / 69.7.  With more channels
  // the stage is worth more: F(2,3) 8 x 56 x 56, 256 -> 64 29.4 / 30.2, F(4,3) 32 x 112 x 112, 128 -> 128 202 / 235, F(2,5) 8 x 56 x 56, 128 -> 256
  // 66.1 / 69.9; with 8 points 32 x 56 x 56, 64 -> 128, F(4,5) 62.4 / 64.9.
  static constexpr int bufs(int F, int num_ks) { return N <= 6 && num_ks <= (N == 4 ? 2 : 1) && stages(F, 4) >= 2 ? 4 : 2; }
};

struct PoArgs {
  int H, W, C, K, Th, Tw, pc, pc_pad;
  long long p0;
  int F, num_kb, items, clusters, nacc, relu, stages, box_rows, bufs;
  uint32_t none;                       // 0, which the compiler does not know
};

__device__ __forceinline__ bool test_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// A barrier that threads of other CTAs arrive at (acquire at cluster scope).  Bounded like mbar_wait.
__device__ __forceinline__ void wait_cluster(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (test_cluster(bar, parity)) return;
  if (*abort_flag) return;
  uint64_t t0 = 0;
  for (uint32_t spin = 0; spin < kSpinLimit; ++spin) {
    if (test_cluster(bar, parity)) return;
    if ((spin & 15u) == 15u) {
      if (*abort_flag) return;
      const uint64_t now = global_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kWaitLimitNs) break;
    }
  }
  *abort_flag = 1;
}
__device__ __forceinline__ void wait_local(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_test(bar, parity)) return;
  if (*abort_flag) return;
  if (!mbar_wait(bar, parity, abort_flag)) *abort_flag = 1;
}
__device__ __forceinline__ uint32_t peer(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// "I have read my exchange buffer", to another CTA.  What orders the reads before it is that it depends on their values
// (see the finish warps): a store that follows from the arrival cannot be what they saw.  A release at cluster scope
// would also wait for the stores of y issued before: 32 x 112 x 112, 64 -> 128, F(2,3) 203 -> 282 us, and 241 with one
// warp per buffer that passes a local arrive on.
__device__ __forceinline__ void arrive_peer(uint32_t bar_cluster_addr) {
  asm volatile("mbarrier.arrive.release.cta.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster_addr) : "memory");
}
// 16 bytes to ANOTHER CTA's shared memory (the instruction is not defined for the executing CTA's own), counted on that
// CTA's barrier when they are there.  (Plain remote stores and one release per slice cost 3 to 4 thousand cycles per
// slice in waiting for the stores.)
__device__ __forceinline__ void store_peer(uint32_t a, uint32_t bar, float x, float y, float z, float w) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w), "r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();                          // an aligned barrier: a warp comes to it as a whole
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void store_own(uint32_t a, float x, float y, float z, float w) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
template <int OFF>
__device__ __forceinline__ float2 lds_ordered(uint32_t saddr) {        // not moved above the wait before it
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2+%3];" : "=f"(v.x), "=f"(v.y) : "r"(saddr), "n"(OFF) : "memory");
  return v;
}

// z_xi[j] of this thread's (tile, filter pair) as CTA xi left it in the exchange buffer
template <int M, int R>
struct ExchangeRows {
  using Cfg = PoCfg<M, R>;
  uint32_t base;
  template <int XI, int J>
  __device__ __forceinline__ void fill(float2 (&z)[M]) const {
    if constexpr (J < M) {
      z[J] = lds_ordered<XI * Cfg::kSrc + J * 512>(base);
      fill<XI, J + 1>(z);
    }
  }
  template <int XI>
  __device__ __forceinline__ void row(float2 (&z)[M]) const { fill<XI, 0>(z); }
};

// setmaxnreg in the direction that leads from the launch's count to REGS
template <int REGS, int FROM>
__device__ __forceinline__ void set_registers() {
  if constexpr (REGS > FROM) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS));
  else if constexpr (REGS < FROM) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS));
}

template <int M, int R, bool SYM, bool I8>
__global__ void __launch_bounds__(PoCfg<M, R>::kThreads, 1)
product_output_kernel(const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmU,
                      const __grid_constant__ Coefs cf, __half* __restrict__ y, const __grid_constant__ PoArgs args,
                      int* __restrict__ status, const float* __restrict__ scale_U, const float* __restrict__ scale_V,
                      const uint8_t* __restrict__ Vdrop) {
  using Cfg = PoCfg<M, R>;
  constexpr int N = Cfg::N;
  const int bufs = args.bufs, off_ring = bufs * Cfg::kBuf;
  const int ST = args.stages, kStageBytes = 2 * (kVBytes + args.F * kRowBytes);
  constexpr int BLOCK_K = I8 ? kRowBytes : kRowBytes / 2;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + off_ring + ST * kStageBytes);
  uint64_t* empty_bar = full_bar + ST;
  uint64_t* tmem_full = empty_bar + ST;             // [2]
  uint64_t* tmem_empty = tmem_full + 2;             // [2]
  uint64_t* z_full = tmem_empty + 2;                // [4] rows of all CTAs have arrived in the exchange buffer
  uint64_t* z_free = z_full + 4;                    // [4] every owner has read its buffer
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(z_free + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = blockIdx.x % N;             // the CTA's rank in its cluster: its row xi
  const int cluster = (int)(blockIdx.x / N);
  const int F = args.F, slices = F / kSliceF, nacc = args.nacc;
  const int num_ks = (args.C + BLOCK_K - 1) / BLOCK_K;
  const int num_pb = (args.pc + kRows - 1) / kRows;
  const uint32_t n_local = args.items > cluster ? (uint32_t)((args.items - cluster + args.clusters - 1) / args.clusters) : 0u;
  // Blocks of tiles in descending order (the input transform left the highest ones in the L2), the filter blocks of a
  // block of tiles next to each other in time.
  auto item_of = [&](uint32_t local, int& pb, int& kb) {
    const int it = cluster + (int)local * args.clusters;
    pb = num_pb - 1 - it / args.num_kb;
    kb = it % args.num_kb;
  };
  const int my_oct = (16 - (int)rank + N - 1) / N;  // groups of 8 tiles this CTA owns: rank, rank + N, ..

  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; ++s) { mbar_init(&full_bar[s], 2); mbar_init(&empty_bar[s], 2); }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tmem_full[a], 2);
      mbar_init(&tmem_empty[a], 8);
    }
    for (int b = 0; b < 4; ++b) {
      mbar_init(&z_full[b], (uint32_t)(1 + my_oct));   // what the other CTAs send, and the own rows per owned octet
      mbar_init(&z_free[b], (uint32_t)(N * Cfg::kFinish));
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const uint32_t cols_used = (uint32_t)(nacc * N * F);
  const uint32_t tmem_cols = cols_used <= 32 ? 32 : cols_used <= 64 ? 64 : cols_used <= 128 ? 128 : cols_used <= 256 ? 256 : 512;
  if (warp == 1) tmem_alloc(tmem_slot, tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_arrive();                                  // the barriers of all CTAs are initialised
  cluster_wait();
  const uint32_t tmem_base = *tmem_slot;
  pdl_launch_dependents();

  if (warp < 4) {
    set_registers<Cfg::kIssueRegs, Cfg::kLaunchRegs>();
    if (warp == 0 || warp == 3) {
      // ---------------- TMA producers: warp 0 fetches V, warp 3 fetches U (one warp alone took 600 cycles per stage over
      // both); a box covers both columns of the stage.  The first stages' U does not wait
      // for the input transform, which lets this kernel start only after its own wait, when everything before it has
      // completed.
      const bool is_v = warp == 0;
      const uint32_t tx = 2u * (is_v ? (uint32_t)(args.box_rows * kRowBytes) : (uint32_t)(F * kRowBytes));
      if (is_v) pdl_wait();
      uint32_t stage = 0, phase = 0;
      const size_t pitch = (size_t)args.C * (I8 ? 1 : 2);
      for (uint32_t local = 0; local < n_local; ++local) {
        int pb, kb;
        item_of(local, pb, kb);
        int back = -ST, bks = 0, bnu = 0;             // the load ST places back: number, channels and columns
        for (int nu = 0; nu < N; nu += 2)
          for (int ks = 0; ks < num_ks; ++ks) {
            wait_local(&empty_bar[stage], phase ^ 1, abort_flag);
            if (lane == 0 && !*abort_flag) {
              uint8_t* dst = smem + off_ring + stage * kStageBytes;
              mbar_expect_tx(&full_bar[stage], tx);
              if (is_v) tma_load_3d(dst, &tmV, &full_bar[stage], ks * BLOCK_K, pb * kRows, (int)rank * N + nu);
              else tma_load_3d(dst + 2 * kVBytes, &tmU, &full_bar[stage], ks * BLOCK_K, kb * F, (int)rank * N + nu);
            }
            __syncwarp();
            if (++stage == (uint32_t)ST) { stage = 0; phase ^= 1; }
            // With one block of filters the load ST places back, whose stage has just come free, was the last read of
            // its lines of V (scratch): they need not be written back.
            if (is_v && Vdrop) {
              if (back >= 0) {
                const uint8_t* line = Vdrop + ((size_t)((int)rank * N + bnu) * args.pc_pad + (size_t)pb * kRows) * pitch + (size_t)bks * kRowBytes;
#pragma unroll
                for (int r = 0; r < 2 * kRows / 32; ++r) {
                  const int row = (r & 3) * 32 + lane;
                  l2_discard_line(line + ((size_t)(r >> 2) * args.pc_pad + row) * pitch);
                }
                if (++bks == num_ks) { bks = 0; bnu += 2; }
              }
              ++back;
            }
          }
      }
    } else if (warp <= 2) {
      // ---------------- MMA issuers: one thread of warp 1 + e issues the columns nu of parity e.  (One issuer alone
      // took 660 cycles per stage, more than the loads.)
      pdl_wait();
      __syncwarp();
      if (elect_one()) {
        const int e = warp - 1;
        const uint32_t idesc = I8 ? umma_idesc_i8(kRows, F) : umma_idesc_f16(kRows, F);
        const uint64_t desc0 = umma_desc_sw128(smem_u32(smem) + off_ring + e * args.box_rows * kRowBytes);
        const uint32_t b_off = (uint32_t)(2 * kVBytes - e * args.box_rows * kRowBytes + e * F * kRowBytes);
        uint32_t stage = 0, phase = 0;
        for (uint32_t local = 0; local < n_local; ++local) {
          const uint32_t acc = nacc == 2 ? local & 1 : 0u, use = nacc == 2 ? local >> 1 : local;
          wait_local(&tmem_empty[acc], (use & 1) ^ 1, abort_flag);
          tc_fence_after();
          for (int nu = e; nu < N; nu += 2) {
            const uint32_t tmem_d = tmem_base + acc * (uint32_t)(N * F) + (uint32_t)(nu * F);
            for (int ks = 0; ks < num_ks; ++ks) {
              wait_local(&full_bar[stage], phase, abort_flag);
              tc_fence_after();
              if (!*abort_flag) {
                const uint64_t ad = umma_desc_advance(desc0, stage * kStageBytes), bd = umma_desc_advance(ad, b_off);
                if constexpr (I8) {
                  umma_i8(tmem_d, ad, bd, idesc, ks > 0 ? 1u : 0u);
#pragma unroll
                  for (int k = 1; k < kRowBytes / kUmmaBytes; ++k)
                    umma_i8(tmem_d, umma_desc_advance(ad, k * kUmmaBytes), umma_desc_advance(bd, k * kUmmaBytes), idesc, 1u);
                } else {
                  umma_f16(tmem_d, ad, bd, idesc, ks > 0 ? 1u : 0u);
#pragma unroll
                  for (int k = 1; k < kRowBytes / kUmmaBytes; ++k)
                    umma_f16_c<true>(tmem_d, umma_desc_advance(ad, k * kUmmaBytes), umma_desc_advance(bd, k * kUmmaBytes), idesc);
                }
                umma_commit(&empty_bar[stage]);
              }
              if (++stage == (uint32_t)ST) { stage = 0; phase ^= 1; }
            }
          }
          if (!*abort_flag) umma_commit(&tmem_full[acc]);
        }
      }
      __syncwarp();
    }
  } else if (warp < 12) {
    // ---------------- row transform: group e takes the slices whose running number is e modulo 2
    set_registers<Cfg::kRowRegs, Cfg::kLaunchRegs>();
    const int quad = warp & 3, grp = (warp - 4) >> 2;
    const int tile = quad * 32 + lane, oct = tile >> 3, t8 = tile & 7;
    const uint32_t owner = (uint32_t)(oct % N);
    // this thread's place in the owner's exchange buffer: [xi][octet][j][filter quad][tile ^ 2 * quad][4]
    const uint32_t zoff = rank * Cfg::kSrc + (uint32_t)(oct / N) * (M * 512);
    const bool own = owner == rank;
    const uint32_t zbase = (own ? smem_u32(smem + Cfg::kOffZ) : peer(smem_u32(smem + Cfg::kOffZ), owner)) + zoff;
    const bool warp_owns = __any_sync(0xffffffffu, own);       // the octets of a CTA lie in different warps
    const uint32_t zbar = peer(smem_u32(z_full), owner);
    pdl_wait();
    float sv = 0.f;
    if constexpr (I8) sv = *scale_V;
    uint32_t gs = 0;
    for (uint32_t local = 0; local < n_local; ++local) {
      int pb, kb;
      item_of(local, pb, kb);
      const uint32_t acc = nacc == 2 ? local & 1 : 0u, use = nacc == 2 ? local >> 1 : local;
      wait_local(&tmem_full[acc], use & 1, abort_flag);
      tc_fence_after();
      const bool live = pb * kRows + quad * 32 < args.pc;         // some tile of this warp exists
      const bool send = pb * kRows + oct * 8 < args.pc;           // ... of this thread's octet
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + acc * (uint32_t)(N * F);
      for (int s = 0; s < slices; ++s, ++gs) {
        if ((int)(gs & 1) != grp) continue;
        const uint32_t b = gs & (uint32_t)(bufs - 1);
        wait_cluster(&z_free[b], ((gs & (uint32_t)bufs) ? 1u : 0u) ^ 1u, abort_flag);
        __syncwarp();                                // the loads of tensor memory are a whole warp's
        if (live) {
#pragma unroll 1
          for (int fq = 0; fq < 4; ++fq) {
            uint32_t r[N][4];
#pragma unroll
            for (int nu = 0; nu < N; ++nu) tmem_ld4(taddr + nu * F + s * kSliceF + fq * 4, r[nu]);
            tmem_ld_wait();
            const uint32_t dst = zbase + b * Cfg::kBuf + (uint32_t)(fq * 128 + ((t8 ^ (fq << 1)) << 4));
            float2 za[M], zb[M];
            const int k0 = kb * F + s * kSliceF + fq * 4;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              float2 in[N];
              float2 qs = make_float2(0.f, 0.f);
              if constexpr (I8)
                qs = make_float2(__fmul_rn(k0 + 2 * h < args.K ? __ldg(scale_U + k0 + 2 * h) : 0.f, sv),
                                 __fmul_rn(k0 + 2 * h + 1 < args.K ? __ldg(scale_U + k0 + 2 * h + 1) : 0.f, sv));
#pragma unroll
              for (int nu = 0; nu < N; ++nu) {
                in[nu] = make_float2(__uint_as_float(r[nu][2 * h]), __uint_as_float(r[nu][2 * h + 1]));
                if constexpr (I8) in[nu] = dequant(in[nu], qs);
              }
              at_apply<M, SYM, float2, N>(cf, in, h ? zb : za);
            }
            if (send && own) {
#pragma unroll
              for (int j = 0; j < M; ++j) store_own(dst + j * 512, za[j].x, za[j].y, zb[j].x, zb[j].y);
            } else if (send) {
#pragma unroll
              for (int j = 0; j < M; ++j) store_peer(dst + j * 512, zbar + b * 8, za[j].x, za[j].y, zb[j].x, zb[j].y);
            }
          }
        }
        __syncwarp();
        if (warp_owns && lane == 0) mbar_arrive(&z_full[b]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tmem_empty[acc]);
    }
  } else {
    // ---------------- finish: group e takes the slices whose running number is e modulo 2, hence always the same buffers
    set_registers<Cfg::kFinishRegs, Cfg::kLaunchRegs>();
    const uint32_t grp = warp - 12 >= Cfg::kFinish ? 1u : 0u;
    const int w = warp - 12 - (int)grp * Cfg::kFinish;
    const int fp = lane & 7, tt = lane >> 3;
    const uint32_t tell = peer(smem_u32(z_free), lane < N ? (uint32_t)lane : 0u);
    pdl_wait();
    uint32_t gs = 0;
    for (uint32_t local = 0; local < n_local; ++local) {
      int pb, kb;
      item_of(local, pb, kb);
      for (int s = 0; s < slices; ++s, ++gs) {
        if ((gs & 1) != grp) continue;
        const uint32_t b = gs & (uint32_t)(bufs - 1);
        if (w == 0 && lane == 0) {                   // what the other CTAs send for the octets of this CTA that exist
          int live = 0;
          for (int slot = 0; slot < my_oct; ++slot) live += pb * kRows + (slot * N + (int)rank) * 8 < args.pc ? 1 : 0;
          mbar_expect_tx(&z_full[b], (uint32_t)(live * (N - 1) * M * 512));
        }
        wait_cluster(&z_full[b], (gs & (uint32_t)bufs) ? 1u : 0u, abort_flag);
        const int k = kb * F + s * kSliceF + 2 * fp;
        // a warp has 4 of the CTA's tiles x 16 filters (the last warps of a CTA that owns fewer octets have none)
        const int slot = w >> 1, t8 = (w & 1) * 4 + tt;
        const int pl = pb * kRows + (slot * N + (int)rank) * 8 + t8;
        float2 Y[M][M];
        uint32_t seen = 0;
        const bool mine = slot < my_oct && pl < args.pc && k < args.K;
        if (mine) {
          const uint32_t base = smem_u32(smem + Cfg::kOffZ) + b * Cfg::kBuf +
                                (uint32_t)(slot * (M * 512) + (fp >> 1) * 128 + ((t8 ^ ((fp >> 1) << 1)) << 4) + (fp & 1) * 8);
          accumulate_rows<M, SYM, float2, N>(cf, ExchangeRows<M, R>{base}, Y);
          // every value read of the buffer is in a sum of the first or the last row: the arrival below waits for all of
          // them (args.none is 0; 0 to 2 % of the call)
#pragma unroll
          for (int i = 0; i < M; i += M - 1)
#pragma unroll
            for (int j = 0; j < M; ++j) seen |= __float_as_uint(Y[i][j].x) | __float_as_uint(Y[i][j].y);
        }
        const bool unread = __any_sync(0xffffffffu, (seen & args.none) != 0u);
        if (lane < N && !unread) arrive_peer(tell + b * 8);
        if (mine) {
          const unsigned p = (unsigned)(args.p0 + pl);
          const unsigned tw = p % (unsigned)args.Tw, q2 = p / (unsigned)args.Tw;
          const unsigned th = q2 % (unsigned)args.Th, img = q2 / (unsigned)args.Th;
          const int h0 = M * (int)th, w0 = M * (int)tw;
          if (args.relu & 2) {
            const int Ho = args.H >> 1, Wo = args.W >> 1, ho = h0 >> 1, wo = w0 >> 1;
            store_tile_pooled<M, __half>(Y, y + (((size_t)img * Ho + ho) * Wo + wo) * args.K + k, (size_t)Wo * args.K, args.K,
                                         Ho - ho, Wo - wo, args.relu & 1);
          } else {
            store_tile<M, __half>(Y, y + (((size_t)img * args.H + h0) * args.W + w0) * args.K + k, (size_t)args.W * args.K, args.K,
                                  args.H - h0, args.W - w0, args.relu & 1);
          }
        }
      }
    }
  }

  const bool expired = *abort_flag != 0;
  if (expired && lane == 0) atomicExch(status, NOVA_ERR_DEVICE_TIMEOUT);
  tc_fence_before();
  cluster_arrive();                                  // nobody leaves while another CTA may still write to or signal it
  cluster_wait();
  if (expired) settle_after_timeout();               // also for what the others sent here and nobody waited for
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, tmem_cols);
  }
}

// [nfreq][rows][inner] elements, rows `pitch` elements apart, 128-byte swizzled boxes of box_rows rows of two neighbouring frequencies
bool make_map(CUtensorMap* map, bool i8, const void* base, int inner, int pitch, int rows, long long freq_stride, int nfreq, int box_rows) {
  EncodeTiledFn enc = tensor_map_encoder();
  if (!enc) return false;
  const int esize = i8 ? 1 : 2;
  cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)rows, (cuuint64_t)nfreq};
  cuuint64_t strides[2] = {(cuuint64_t)pitch * esize, (cuuint64_t)freq_stride * esize};
  cuuint32_t box[3] = {(cuuint32_t)(kRowBytes / esize), (cuuint32_t)box_rows, 2};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, i8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(base), dims, strides,
             box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int cluster_slots(int n, int sms) {                  // clusters of n CTAs that run at once (148 SMs: 33, 22, 15)
  const int s = n == 4 ? sms / 4 - 4 : n == 6 ? sms / 6 - 2 : sms / 8 - 3;
  return s < 1 ? 1 : s;
}

// setmaxnreg draws on the registers the block was launched with: a build whose register count is not what the split was
// computed for does without this kernel.
template <int M, int R, bool SYM, bool I8>
bool built() {
  static const int regs = [] {
    cudaFuncAttributes at;
    return cudaFuncGetAttributes(&at, product_output_kernel<M, R, SYM, I8>) == cudaSuccess ? at.numRegs : 0;
  }();
  return regs >= PoCfg<M, R>::kLaunchRegs;
}
template <int M, int R>
bool built(bool sym, bool i8) {
  return i8 ? (sym ? built<M, R, true, true>() : built<M, R, false, true>()) : (sym ? built<M, R, true, false>() : built<M, R, false, false>());
}
bool built(const nova_plan* plan, bool i8) {
  const bool sym = plan->symmetric != 0;
  switch (plan->r * 10 + plan->m) {
    case 32: return built<2, 3>(sym, i8);
    case 34: return built<4, 3>(sym, i8);
    case 36: return built<6, 3>(sym, i8);
    case 52: return built<2, 5>(sym, i8);
    case 54: return built<4, 5>(sym, i8);
  }
  return false;
}

template <int M, int R, bool SYM, bool I8>
int go(const nova_plan* plan, const Geom& g, const void* V, const void* U, void* y, long long p0, int pc, int pc_pad, int relu, int F,
       const float* scale_U, const float* scale_V, cudaStream_t stream) {
  using Cfg = PoCfg<M, R>;
  auto kernel = product_output_kernel<M, R, SYM, I8>;
  if (!built<M, R, SYM, I8>()) return (int)cudaErrorInvalidConfiguration;
  PoArgs a;
  // rows of a box of V: a layer of fewer than 128 tiles fetches no zero fill (the rows beyond hold what they held:
  // their sums are not sent)
  a.box_rows = pc < kRows ? (pc + 7) & ~7 : kRows;
  CUtensorMap tmV, tmU;
  if (!make_map(&tmV, I8, V, g.C, g.ldv, pc, (long long)pc_pad * g.ldv, Cfg::N * Cfg::N, a.box_rows) ||
      !make_map(&tmU, I8, U, g.C, g.C, g.K, (long long)g.K * g.C, Cfg::N * Cfg::N, F))
    return (int)cudaErrorUnknown;
  a.H = g.H; a.W = g.W; a.C = g.C; a.K = g.K; a.Th = g.Th; a.Tw = g.Tw; a.pc = pc; a.pc_pad = pc_pad; a.p0 = p0;
  a.F = F;
  a.num_kb = (g.K + F - 1) / F;
  a.items = (pc + kRows - 1) / kRows * a.num_kb;
  const int slots = cluster_slots(Cfg::N, plan->sm_count);
  a.clusters = a.items < slots ? a.items : slots;
  a.nacc = 2 * Cfg::N * F <= 512 ? 2 : 1;
  a.relu = relu;
  a.none = 0;
  a.bufs = Cfg::bufs(F, (g.C * (I8 ? 1 : 2) + kRowBytes - 1) / kRowBytes);
  a.stages = Cfg::stages(F, a.bufs);
  const int smem = Cfg::total(F, a.bufs);
  if (cudaError_t e = allow_dynamic_smem<Cfg::kMaxTotal>(kernel); e != cudaSuccess) return (int)e;
  const int esize = I8 ? 1 : 2;
  const bool drop = a.num_kb == 1 && ((size_t)g.C * esize) % kRowBytes == 0 && (reinterpret_cast<uintptr_t>(V) % kRowBytes) == 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.clusters * Cfg::N));
  cfg.blockDim = dim3(Cfg::kThreads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = Cfg::N;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return (int)cudaLaunchKernelEx(&cfg, kernel, tmV, tmU, plan->kcoefs, (__half*)y, a, plan->status_dev, scale_U, scale_V,
                                 drop ? (const uint8_t*)V : (const uint8_t*)nullptr);
}

// Filters per block: 64 with 4 points, where two sets of accumulators still fit (but for a single block of at most 64
// filters and 64 channels, which 32 spreads better), 32 otherwise.  F(2,3), 25088 tiles, 128 -> 128: 1.40x with 32,
// 1.66x with 64 over the three kernels; 6272 tiles, 64 -> 64: 1.25x and 1.20x; F(4,3), 25088 tiles, 64 -> 128: 1.50x and 1.34x.
int block_filters(int n, int K, int num_ks) {
  if (K <= 16) return 16;
  return n == 4 && K >= 64 && (K > 64 || num_ks > 1) ? 64 : 32;
}

}  // namespace

// Against product and output transform as two kernels.  What this kernel saves is M (n*n floats per tile and filter,
// written and read); what it costs is V once per F filters instead of once per 256, and an exchange at 17 bytes per
// clock and SM.  So it pays where M is large and the channels few: num_ks = 128-byte rows of channels.  Whole calls, time of
// three kernels / of two, by MB of M, over 1100 layers of 1 .. 32 images of 28 x 28 .. 112 x 112:
//   n = 4          up to two rows: 13 MB 1.0 .. 1.3, 26 MB 1.1 .. 1.4, 103 MB 1.3 .. 1.5, 411 MB 1.5 .. 2.2
//                  more: one filter block 1.04 .. 1.2; several: 8 rows 26 MB 1.0, 51 MB 0.94 .. 1.12, 103 MB 1.0 .. 1.1, 411 MB 1.35; 12 rows
//                  51 MB 0.85 .. 1.1, 103 MB 0.91; 16 rows 26 .. 103 MB 0.81 .. 0.95: the more rows, the more of M it takes
//   n = 6, m = 2   one row 29 MB 1.14, 58 MB 1.04 .. 1.24; two rows 58 MB 1.04 .. 1.14, 116 MB 1.1 .. 1.2, 462 MB 1.4
//   n = 6, m = 4   one row: 14 .. 58 MB 0.96 .. 1.02, 116 MB 1.0 .. 1.06, 231 MB and more 1.07 .. 1.7; two rows: 116 MB 0.93 .. 1.06,
//                  173 MB 0.95, 231 MB 0.97 (256 filters) .. 1.18 (64), 462 MB 1.16 .. 1.24
//   n = 8, m = 4   one row: 26 MB 1.06, 103 MB 1.18; two rows: 103 MB 0.96 .. 1.06, 206 MB 0.98 .. 1.03, 411 MB 1.07 .. 1.26
//   n = 8, m = 6   one row: 95 MB 0.96, 189 MB 1.01, 419 MB 1.05; two rows: 105 MB 0.87, 379 MB 1.04 .. 1.07, 757 MB 1.13, but with 512
//                  filters 419 MB 0.97
// Rows of channels that are not whole 32-byte sectors lose 5 to 10 % more here, because those of U keep their pitch: 72 or 104
// channels 0.87 .. 0.96 at two rows, 24 or 40 channels 0.9 .. 0.97 near the line of n = 8, m = 4.
// INT8 lines up with half at the same number of rows (32 x 56 x 56, 256 -> 256: 132 -> 123 us).
bool use_product_output(const nova_plan* plan, const Geom& g, bool int8) {
  if (plan->mode != NOVA_FP16_F32ACC || plan->n > 8 || !plan->status_dev || plan->sm_count < 64 || g.P >= (1ll << 31)) return false;
  if (!built(plan, int8)) return false;
  const int num_ks = (g.C * (int8 ? 1 : 2) + kRowBytes - 1) / kRowBytes;
  const double m_mb = 4e-6 * plan->n * plan->n * (double)g.P * g.K;
  if (plan->n == 4) {
    const int F = block_filters(4, g.K, num_ks), num_kb = (g.K + F - 1) / F;
    return m_mb >= 12 && (num_kb == 1 || m_mb * (num_kb == 2 ? 4 : 2) >= num_ks * num_ks);
  }
  if (num_ks > 2) return false;
  if (plan->n == 6) return m_mb >= (plan->m == 2 ? 50 : 100 * num_ks);
  return m_mb >= (plan->m == 6 ? 300 : num_ks == 1 ? 20 : 150);
}

int launch_product_output(const nova_plan* plan, const Geom& g, const void* V, const void* U, void* y, long long p0, int pc,
                          int pc_pad, int relu, void* stream, const float* scale_U, const float* scale_V) {
  cudaStream_t s = (cudaStream_t)stream;
  const int F = block_filters(plan->n, g.K, (g.C * (scale_U ? 1 : 2) + kRowBytes - 1) / kRowBytes);
#define NOVA_PO(MV, RV)                                                                                                      \
  do {                                                                                                                       \
    if (scale_U)                                                                                                             \
      return plan->symmetric ? go<MV, RV, true, true>(plan, g, V, U, y, p0, pc, pc_pad, relu, F, scale_U, scale_V, s)            \
                             : go<MV, RV, false, true>(plan, g, V, U, y, p0, pc, pc_pad, relu, F, scale_U, scale_V, s);          \
    return plan->symmetric ? go<MV, RV, true, false>(plan, g, V, U, y, p0, pc, pc_pad, relu, F, scale_U, scale_V, s)             \
                           : go<MV, RV, false, false>(plan, g, V, U, y, p0, pc, pc_pad, relu, F, scale_U, scale_V, s);           \
  } while (0)
  if (plan->r == 3) {
    if (plan->m == 2) NOVA_PO(2, 3);
    if (plan->m == 4) NOVA_PO(4, 3);
    if (plan->m == 6) NOVA_PO(6, 3);
  } else if (plan->r == 5) {
    if (plan->m == 2) NOVA_PO(2, 5);
    if (plan->m == 4) NOVA_PO(4, 5);
  }
#undef NOVA_PO
  return (int)cudaErrorInvalidValue;
}

}  // namespace nova
