// Step 3 for up to 8 tokens: the product as a stream of packed weights through warp-level MMAs.
//   w4a4_gemm_stream_kernel   INT4 tokens: mma.sync m16n8k32, s8 x s8 -> s32 (exact)
//   wo_gemm_stream_kernel     fp16 tokens (weight-only variant): mma.sync m16n8k16, fp32 accumulation
//
// With so few tokens a layer is its weights' trip through the chip, and then what follows the tokens' arrival.  The
// tensor-memory kernels hold 128 KB of weights on each of 112 to 128 SMs ahead of the tokens, half of a 29 MB layer, and stream
// the rest afterwards; here every SM holds up to 200 KB.  The weights go from shared memory to registers, where the nibbles are
// widened, and on to the MMA: no operand ring and no hand-overs between roles, one wait per 256 channels.  What follows the
// tokens is bound by the widening (logic pipe, half rate) and the latency of its chain with four warps per scheduler: 8 x 8192
// -> 28672 in fp16 34 us, 42 % of the issue slots.  Layers: 1 x 4096 -> 14336 10.4 -> 9.6 us, 1 x 14336 -> 4096 13.8 -> 11.5, 8 x
// 4096 -> 4096 8.0 -> 7.0; weight-only 1 x 4096 -> 14336 18.5 -> 13.2, 2 x 8192 -> 8192 24.7 -> 16.4, 8 x 4096 -> 11008 14.9 ->
// 12.5.  16 tokens were tried too: INT4 12.1 us a layer against 11.7, fp16 17.3 and 16.6 (twice the MMAs and token fragments).
// Both kernels are at 96 registers, all that 18 warps (allocated as 20) leave a thread; the fp16 one spills ten words there, and
// was tried for 16 tokens under that limit.
//
// A block takes a tile of up to 128 output channels, as many as give every SM the same share; its sixteen warps split K, and the
// channels where there are more than 32, and add up at the end.  The weights are the A operand (16 channels x 32 or 16 of K), the
// tokens B.  K is walked in 16-byte pieces of a weight row: lane 4 g + t takes piece t of row g, so that the MMA's idea of which
// k is which is a permutation -- the same one for weights and tokens.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "sq_internal.h"
#include "sq_ptx.cuh"

namespace sq {
namespace {

constexpr int SM_WARPS = 16;                         // consumers; one warp each for the weight and the token loads besides
constexpr int SM_THREADS = (SM_WARPS + 2) * 32;
constexpr int SM_MAX_ROWS = 128;                     // output channels of a tile
constexpr int SM_MAX_STAGES = 32;                    // one per lane of a loading warp
constexpr int SM_FLIGHT = 128 * 1024;                // bytes of weights requested and not landed, per SM

enum StreamSite : uint32_t { SM_W_FULL = 96, SM_X_FULL, SM_EMPTY_W, SM_EMPTY_X };

struct StreamLayout {
  int rows;             // output channels per tile
  int wr, nb;           // groups of warps along the channels (the others split K), blocks of 16 channels each at most
  int stages, flight;   // ring depth, stages in flight
  int w_st, x_st;       // bytes of a stage: 256 channels of `rows` weight rows, and of the tokens
  int off_x, off_red, off_bar, total;
};

// `red`: bytes for the sums; `overlay`: they take the place of the ring, which has been read by then.
__host__ __device__ inline StreamLayout stream_layout(int rows, int x_st, int red, bool overlay) {
  StreamLayout L;
  L.rows = rows;
  L.wr = rows > 32 ? 2 : 1;
  L.nb = ((rows + 15) / 16 + L.wr - 1) / L.wr;
  L.w_st = (rows * 128 + 1023) / 1024 * 1024;
  L.x_st = x_st;
  const int bars = 3 * SM_MAX_STAGES * 8;
  const int room = 227 * 1024 - 1024 - (overlay ? 0 : red) - bars;
  int s = room / (L.w_st + L.x_st);
  s = s > SM_MAX_STAGES ? SM_MAX_STAGES : s;
  const int lap = SM_WARPS / L.wr / 2;               // stages that the warps work on side by side
  L.stages = s / lap * lap;
  // Whole laps, one at least: block it - flight then is the same warps' as block it, see stream_loads.
  const int f = SM_FLIGHT / L.w_st / lap * lap;
  L.flight = f < lap ? lap : (f > L.stages ? L.stages : f);
  const int ring = L.stages * (L.w_st + L.x_st);       // (a ragged last block's fragments reach into the next stage, or the tokens')
  L.off_x = L.stages * L.w_st;
  L.off_red = overlay ? 0 : ring;
  L.off_bar = overlay ? (ring > red ? ring : (red + 15) / 16 * 16) : ring + red;
  L.total = L.off_bar + bars;
  return L;
}

// The loading warps' walk over blocks 0 .. total - 1: lane s owns the ring's stage s.  One thread that issues every load takes
// some 0.2 us over each; the lanes of a warp issue theirs together.  `issue(it)` requests block `it`; `first`: blocks below it
// have been requested already; `landed_bars`: no more than L.flight blocks are on their way (the weights), else null.
template <typename Issue>
__device__ __forceinline__ void stream_loads(const StreamLayout& L, int total, int first, uint64_t* empty, uint64_t* landed_bars,
                                             uint32_t site, uint32_t limit, Issue issue) {
  const int lane = threadIdx.x & 31;
  int it = lane < first ? lane + L.stages : lane;
  uint32_t ph = it < L.stages ? 1u : 0u;             // parity of the phase of `empty` that this lane waits for
  bool left = lane < L.stages && it < total;
  bool landed = landed_bars == nullptr;
  uint32_t idle = 0;
  while (__any_sync(0xFFFFFFFFu, left)) {
    bool go = left && (it < L.stages || mbar_test_wait(&empty[lane], ph));
    // Block f = it - flight, which this lane looks at once it has issued block it - stages, is read by the same warps as block
    // `it` (the flight is whole laps), after block it - stages or being that block.  So its stage is not free for a refill before
    // this lane looks; and the tests of a pass come before its loads.  The phase cannot be missed, however far apart the warps are.
    // (With flights of other lengths -- 9 of 12 stages -- a pair of warps a ring behind the others left this lane waiting for good.)
    if (left && !landed) {
      const int f = it - L.flight;
      landed = mbar_test_wait(&landed_bars[f % L.stages], (f / L.stages) & 1);
    }
    go = go && landed;
    __syncwarp();
    if (go) {
      issue(it);
      it += L.stages;
      ph ^= 1;
      landed = landed_bars == nullptr;
      left = it < total;
    }
    if (__any_sync(0xFFFFFFFFu, go)) {
      idle = 0;
    } else {
      __nanosleep(100);                              // the consumers need the issue slots
      if (++idle <= limit / 8) continue;
      if (lane == 0) atomicCAS(&g_device_status, 0u, (site << 8) | 1u);
      break;
    }
  }
}

__device__ __forceinline__ void mma_s8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void red_add_shared(int* p, int v) {
  asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
// In program order: the compiler would bring all of a stage's fragments forward, and spill.
__device__ __forceinline__ uint4 lds128(const void* p) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(smem_u32(p)));
  return v;
}
__device__ __forceinline__ uint32_t even_codes(uint32_t w) { return (w << 4) & 0xF0F0F0F0u; }
__device__ __forceinline__ uint32_t odd_codes(uint32_t w) { return w & 0xF0F0F0F0u; }
__device__ __forceinline__ uint32_t word_of(const uint4& v, int i) { return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w)); }
// Row of a block of eight behind MMA row g: with rows g and g + 4 next to each other the sixteen-byte pieces that a quarter of
// a warp reads out of the swizzled stage lie in different banks.
__device__ __forceinline__ int frag_row(int g) { return (g >> 1) | ((g & 1) << 2); }

constexpr int SM_NT = 8, SM_RP8 = 136;              // W4A4: tokens of a tile; pitch of the sums, 8 banks from token to token

__global__ void __launch_bounds__(SM_THREADS, 1)
w4a4_gemm_stream_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
                        const __grid_constant__ StreamLayout L, const __half* __restrict__ sx, const __half* __restrict__ sw,
                        int M, int N, int K, __half* __restrict__ Y, int32_t* __restrict__ accdbg) {
  griddep_launch_dependents();                       // a rotate kernel launched behind this one may set itself up
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  uint64_t* w_full = reinterpret_cast<uint64_t*>(smem + L.off_bar);
  uint64_t* x_full = w_full + SM_MAX_STAGES;
  uint64_t* empty = x_full + SM_MAX_STAGES;
  int* red = reinterpret_cast<int*>(smem + L.off_red);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int num_sb = (K + 255) / 256;
  const int tiles = (N + L.rows - 1) / L.rows;
  const int cta = static_cast<int>(blockIdx.x), ncta = static_cast<int>(gridDim.x);
  const int my_tiles = cta < tiles ? (tiles - cta + ncta - 1) / ncta : 0;
  const int total = my_tiles * num_sb;
  const uint32_t limit = wait_limit();

  auto issue_w = [&](int it) {
    const int s = it % L.stages;
    mbar_arrive_expect_tx(&w_full[s], static_cast<uint32_t>(L.rows * 128));
    tma_load_2d(smem + s * L.w_st, &tmap_w, &w_full[s], it % num_sb * 128, (cta + it / num_sb * ncta) * L.rows);
  };
  const int first = min(L.flight, total);
  if (warp == SM_WARPS) {
    // The weights do not depend on the kernel before this one: they go out before anything else is set up.
    if (lane < L.stages) mbar_init(&w_full[lane], 1);
    mbar_fence_init();
    __syncwarp();
    if (lane < first) issue_w(lane);
    if (lane < L.stages) {
      mbar_init(&x_full[lane], 1);
      mbar_init(&empty[lane], static_cast<uint32_t>(2 * L.wr));
    }
    mbar_fence_init();
  }
  for (int i = threadIdx.x; i < SM_NT * SM_RP8; i += SM_THREADS) red[i] = 0;
  __syncthreads();

  if (warp == SM_WARPS) {
    stream_loads(L, total, first, empty, w_full, SM_EMPTY_W, limit, issue_w);
  } else if (warp == SM_WARPS + 1) {
    griddep_wait();                                  // Xq may come from the kernel launched before this one
    stream_loads(L, total, 0, empty, nullptr, SM_EMPTY_X, limit, [&](int it) {
      const int s = it % L.stages;
      mbar_arrive_expect_tx(&x_full[s], static_cast<uint32_t>(L.x_st));
      tma_load_2d(smem + L.off_x + s * L.x_st, &tmap_x, &x_full[s], it % num_sb * 128, 0);
    });
  } else {
    const int g = lane >> 2, t = lane & 3, pg = frag_row(g);
    const int kgs = SM_WARPS / L.wr;                 // groups along K: two share a stage, half of its channels each
    const int kg = warp % kgs, rg = warp / kgs;
    const int q0 = kg >> 1, qn = kgs >> 1;
    const int blocks = (L.rows + 15) / 16, first_block = rg * L.nb;            // of 16 channels
    const uint32_t frag = pg * 128 + (((4 * (kg & 1) + t) ^ pg) << 4);
    const unsigned char *wf = smem + first_block * 2048 + frag, *xf = smem + L.off_x + frag;
    const int rp = threadIdx.x & 63, tk = threadIdx.x >> 6;          // epilogue: a pair of channels of one token
    griddep_wait();                                  // the token steps come from the kernel before, which may still read Y
    const float sxv = tk < M ? __half2float(__ushort_as_half(__ldcg(reinterpret_cast<const unsigned short*>(sx) + tk))) : 0.0f;
    auto consume = [&](auto blocks_of_warp) {
      constexpr int NB = decltype(blocks_of_warp)::value;
      bool ok = true;
      int it = q0, s = q0;                             // this warp's next block and its stage
      uint32_t ph = 0;
      for (int tl = 0, tile = cta; tl < my_tiles; ++tl, tile += ncta) {
        const int ch = tile * L.rows + 2 * rp;
        const bool live = 2 * rp < L.rows && ch < N;
        const __half2 swv = live ? *reinterpret_cast<const __half2*>(sw + ch) : __floats2half2_rn(0.0f, 0.0f);
        int acc[NB][4];
  #pragma unroll
        for (int b = 0; b < NB; ++b)
  #pragma unroll
          for (int e = 0; e < 4; ++e) acc[b][e] = 0;
        const int end = (tl + 1) * num_sb;
        for (; it < end && ok; it += qn) {
          ok = mbar_wait(&w_full[s], ph, SM_W_FULL, limit);
          if (!ok) break;
          const unsigned char *wp = wf + s * L.w_st, *xp = xf + s * L.x_st;
          // All fragments first, then the steps of 32 channels with the blocks side by side: a chain of MMAs into one
          // accumulator takes 21 cycles a link and up, the tensor pipe 8.
          uint4 u[NB], v[NB];
  #pragma unroll
          for (int b = 0; b < NB; ++b) {
            u[b] = *reinterpret_cast<const uint4*>(wp + b * 2048);
            v[b] = *reinterpret_cast<const uint4*>(wp + b * 2048 + 1024);
          }
          ok = mbar_wait(&x_full[s], ph, SM_X_FULL, limit);
          if (!ok) break;
          const uint4 x = *reinterpret_cast<const uint4*>(xp);
  #pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint32_t b0 = even_codes(word_of(x, i)), b1 = odd_codes(word_of(x, i));
  #pragma unroll
            for (int b = 0; b < NB; ++b) {
              const uint32_t p = word_of(u[b], i), q = word_of(v[b], i);
              mma_s8(acc[b], even_codes(p), even_codes(q), odd_codes(p), odd_codes(q), b0, b1);
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&empty[s]);
          s += qn;                                     // the depth is a multiple of qn: a warp meets every phase of its stages
          if (s >= L.stages) { s -= L.stages; ph ^= 1; }
        }
        // The warps' sums over K meet in shared memory (integers: in any order).
  #pragma unroll
        for (int b = 0; b < NB; ++b) {
          int* r0 = red + (first_block + b) * 16 + pg;
  #pragma unroll
          for (int e = 0; e < 4; ++e)                  // e & 1: token t or t + 4, e >> 1: the block's second eight rows
            red_add_shared(r0 + (t + 4 * (e & 1)) * SM_RP8 + 8 * (e >> 1), acc[b][e]);
        }
        named_barrier(1, SM_WARPS * 32);
        if (live && tk < M) {
          int2 a = *reinterpret_cast<const int2*>(red + tk * SM_RP8 + 2 * rp);
          a.x >>= 8;                                   // exact: the sum is 256 * acc
          a.y >>= 8;
          const __half2 h = __floats2half2_rn((__int_as_float(0x4B400000 + a.x) - 12582912.0f) * (sxv * __low2float(swv)),
                                              (__int_as_float(0x4B400000 + a.y) - 12582912.0f) * (sxv * __high2float(swv)));
          *reinterpret_cast<__half2*>(Y + static_cast<size_t>(tk) * N + ch) = h;
          if (accdbg) *reinterpret_cast<int2*>(accdbg + static_cast<size_t>(tk) * N + ch) = a;
        }
        if (tl + 1 < my_tiles) {
          named_barrier(1, SM_WARPS * 32);
          for (int i = threadIdx.x; i < SM_NT * SM_RP8; i += SM_WARPS * 32) red[i] = 0;
          named_barrier(1, SM_WARPS * 32);
        }
      }
    };
    switch (min(L.nb, blocks - first_block)) {
      case 1: consume(std::integral_constant<int, 1>()); break;
      case 2: consume(std::integral_constant<int, 2>()); break;
      case 3: consume(std::integral_constant<int, 3>()); break;
      default: consume(std::integral_constant<int, 4>());
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Weight-only: the tokens are fp16, four times the bytes, and every block reads those of its share of K.  Where that is more
// than the weights (few channels, long K), K is split over a cluster: its blocks work on one tile of up to 128 channels.
// ---------------------------------------------------------------------------------------------
constexpr int SM_RPF = 132;                          // pitch of the sums: 8 banks between a lane's token pairs
constexpr int SM_PART = SM_NT * SM_RPF;              // floats of one set of partial sums

__global__ void __launch_bounds__(SM_THREADS, 1)
wo_gemm_stream_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_z,
                      const __grid_constant__ StreamLayout L, const __half* __restrict__ sw, int M, int N, int K, int splits,
                      __half* __restrict__ Y) {
  griddep_launch_dependents();                       // a rotate kernel launched behind this one may set itself up
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  uint64_t* w_full = reinterpret_cast<uint64_t*>(smem + L.off_bar);
  uint64_t* x_full = w_full + SM_MAX_STAGES;
  uint64_t* empty = x_full + SM_MAX_STAGES;
  float* part = reinterpret_cast<float*>(smem + L.off_red);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int crank = splits > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int num_sb = (K + 255) / 256;
  const int sb0 = crank * num_sb / splits, nsb = (crank + 1) * num_sb / splits - sb0;      // this block's share of K
  const int tiles = (N + L.rows - 1) / L.rows;
  const int cid = static_cast<int>(blockIdx.x) / splits, ncl = static_cast<int>(gridDim.x) / splits;
  const int my_tiles = cid < tiles ? (tiles - cid + ncl - 1) / ncl : 0;
  const int total = my_tiles * nsb;
  const uint32_t limit = wait_limit();

  auto issue_w = [&](int it) {
    const int s = it % L.stages;
    mbar_arrive_expect_tx(&w_full[s], static_cast<uint32_t>(L.rows * 128));
    tma_load_2d(smem + s * L.w_st, &tmap_w, &w_full[s], (sb0 + it % nsb) * 128, (cid + it / nsb * ncl) * L.rows);
  };
  const int first = min(L.flight, total);
  if (warp == SM_WARPS) {
    if (lane < L.stages) mbar_init(&w_full[lane], 1);
    mbar_fence_init();
    __syncwarp();
    if (lane < first) issue_w(lane);
    if (lane < L.stages) {
      mbar_init(&x_full[lane], 1);
      mbar_init(&empty[lane], static_cast<uint32_t>(2 * L.wr));
    }
    mbar_fence_init();
  }
  __syncthreads();

  if (warp == SM_WARPS) {
    stream_loads(L, total, first, empty, w_full, SM_EMPTY_W, limit, issue_w);
  } else if (warp == SM_WARPS + 1) {
    griddep_wait();                                  // Z16 may come from the kernel launched before this one
    stream_loads(L, total, 0, empty, nullptr, SM_EMPTY_X, limit, [&](int it) {
      const int s = it % L.stages;
      mbar_arrive_expect_tx(&x_full[s], static_cast<uint32_t>(L.x_st));
#pragma unroll
      for (int b = 0; b < 4; ++b)                    // 64 channels each
        tma_load_2d(smem + L.off_x + s * L.x_st + b * (SM_NT * 128), &tmap_z, &x_full[s], (sb0 + it % nsb) * 256 + b * 64, 0);
    });
  } else {
    const int g = lane >> 2, t = lane & 3, pg = frag_row(g);
    const int kgs = SM_WARPS / L.wr;                 // groups along K: two share a stage, half of its channels each
    const int kg = warp % kgs, rg = warp / kgs;
    const int q0 = kg >> 1, qn = kgs >> 1;
    const int blocks = (L.rows + 15) / 16, first_block = rg * L.nb;            // of 16 channels
    const unsigned char* wf = smem + first_block * 2048 + pg * 128 + (((4 * (kg & 1) + t) ^ pg) << 4);
    const unsigned char* xf = smem + L.off_x + (2 * (kg & 1) + (t >> 1)) * (SM_NT * 128) + g * 128;
    const uint32_t xc = static_cast<uint32_t>((4 * (t & 1)) ^ g) << 4;      // piece t: half of a token row of 64 channels
    const int rp = threadIdx.x & 63, tk = threadIdx.x >> 6;          // epilogue: a pair of channels of one token
    const int rpp = (L.rows / 2 + splits - 1) / splits;              // channel pairs that a block of the cluster finishes
    griddep_wait();                                  // the kernel before this one may still read Y
    const WidenConsts wk = widen_consts();
    auto consume = [&](auto blocks_of_warp) {
      constexpr int NB = decltype(blocks_of_warp)::value;
      bool ok = true;
      int it = q0, s = q0;                           // this warp's next block and its stage
      uint32_t ph = 0;
      for (int tl = 0, tile = cid; tl < my_tiles; ++tl, tile += ncl) {
        const int ch = tile * L.rows + 2 * rp;
        const bool live = 2 * rp < L.rows && ch < N && tk < M;
        const float2 swv = live ? __half22float2(*reinterpret_cast<const __half2*>(sw + ch)) : make_float2(0.0f, 0.0f);
        float acc[NB][4];
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[b][e] = 0.0f;
        const int end = (tl + 1) * nsb;
        for (; it < end && ok; it += qn) {
          ok = mbar_wait(&w_full[s], ph, SM_W_FULL, limit) && mbar_wait(&x_full[s], ph, SM_X_FULL, limit);
          if (!ok) break;
          const unsigned char *wp = wf + s * L.w_st, *xp = xf + s * L.x_st;
#pragma unroll
          for (int b0 = 0; b0 < NB; b0 += 2) {       // two blocks at a time: the registers hold no more
            uint4 u[2], v[2];
#pragma unroll
            for (int b = 0; b < 2; ++b) {
              if (b0 + b < NB) {
                u[b] = lds128(wp + (b0 + b) * 2048);
                v[b] = lds128(wp + (b0 + b) * 2048 + 1024);
              }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint4 x = lds128(xp + (xc ^ (i << 4)));
#pragma unroll
              for (int b = 0; b < 2; ++b) {
                if (b0 + b < NB) {
                  const uint4 p = widen_word(word_of(u[b], i), wk), q = widen_word(word_of(v[b], i), wk);
                  mma_f16(acc[b0 + b], p.x, q.x, p.y, q.y, x.x, x.y);
                  mma_f16(acc[b0 + b], p.z, q.z, p.w, q.w, x.z, x.w);
                }
              }
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&empty[s]);
          s += qn;                                   // the depth is a multiple of qn: a warp meets every phase of its stages
          if (s >= L.stages) { s -= L.stages; ph ^= 1; }
        }
        // Sums over K, always in the same order: the upper half of the groups along K hands its own to the lower half, whose
        // four (or eight, with one group of warps along the channels) are added up one by one.
        if (L.off_red == 0) named_barrier(1, SM_WARPS * 32);         // the ring has been read
        float* mine = part + (kg & (kgs / 2 - 1)) * SM_PART + first_block * 16 + pg;
#pragma unroll
        for (int upper = 1; upper >= 0; --upper) {
          if ((kg >= kgs / 2) == (upper == 1)) {
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
              for (int e = 0; e < 4; ++e) {          // e & 1: token 2 t or 2 t + 1, e >> 1: the block's second eight rows
                float* p = mine + (2 * t + (e & 1)) * SM_RPF + b * 16 + 8 * (e >> 1);
                *p = upper ? acc[b][e] : acc[b][e] + *p;
              }
          }
          named_barrier(1, SM_WARPS * 32);
        }
        float* sums = part + tk * SM_RPF + 2 * rp;
        __half2* y = reinterpret_cast<__half2*>(Y + static_cast<size_t>(tk) * N + ch);
        if (live) {
          float2 a = make_float2(0.0f, 0.0f);
          for (int k = 0; k < kgs / 2; ++k) {
            const float2 b = *reinterpret_cast<const float2*>(sums + k * SM_PART);
            a.x += b.x;
            a.y += b.y;
          }
          if (splits > 1) *reinterpret_cast<float2*>(sums) = a;      // the first set's place: this thread alone reads it here
          else *y = __floats2half2_rn(a.x * swv.x, a.y * swv.y);
        }
        if (splits > 1) {
          // One tile per cluster then.  Block r of it finishes the channel pairs [r rpp, (r + 1) rpp).
          __syncwarp();
          cluster_arrive_release();
          cluster_wait_acquire();
          if (live && rp / rpp == crank) {
            float2 a = make_float2(0.0f, 0.0f);
            for (int r = 0; r < splits; ++r) {
              float2 b;
              asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(b.x), "=f"(b.y)
                           : "r"(cluster_map(sums, static_cast<uint32_t>(r))) : "memory");
              a.x += b.x;
              a.y += b.y;
            }
            *y = __floats2half2_rn(a.x * swv.x, a.y * swv.y);
          }
        } else if (tl + 1 < my_tiles) {
          named_barrier(1, SM_WARPS * 32);           // the sums have been read
        }
      }
    };
    switch (min(L.nb, blocks - first_block)) {
      case 1: consume(std::integral_constant<int, 1>()); break;
      case 2: consume(std::integral_constant<int, 2>()); break;
      case 3: consume(std::integral_constant<int, 3>()); break;
      default: consume(std::integral_constant<int, 4>());
    }
  }
  if (splits > 1) {
    // Every thread of the cluster's blocks arrives twice: nobody leaves while another block reads its sums.
    __syncwarp();
    if (warp >= SM_WARPS || my_tiles == 0) {
      cluster_arrive_release();
      cluster_wait_acquire();
    }
    cluster_arrive_release();
    cluster_wait_acquire();
  }
}

sq_status_t launch_w4a4_stream(const StreamLayout& L, const void* Xq, const void* sx, const void* Wq, const void* sw, int M, int N,
                               int K, void* Y, int32_t* accdbg, int grid, cudaStream_t s) {
  auto kern = w4a4_gemm_stream_kernel;
  const int smem = L.total + 1024;
  if (!ensure_dyn_smem(reinterpret_cast<const void*>(kern), smem)) return SQ_ERR_CUDA;
  CUtensorMap mw, mx;
  if (!make_packed_map(&mw, Wq, N, K / 2, L.rows) || !make_packed_map(&mx, Xq, M, K / 2, SM_NT)) return SQ_ERR_CUDA;
  const cudaError_t err = launch_maybe_pdl(kern, dim3(static_cast<unsigned>(grid)), dim3(SM_THREADS), static_cast<size_t>(smem), s,
                                           mw, mx, L, static_cast<const __half*>(sx), static_cast<const __half*>(sw), M, N, K,
                                           static_cast<__half*>(Y), accdbg);
  count_launch();
  return err == cudaSuccess ? SQ_OK : SQ_ERR_CUDA;
}

// Clusters of `s` blocks of the weight-only kernel that the device holds at once (its shared memory leaves one block per SM).
int wo_stream_clusters(int s) {
  static std::atomic<int> cache[64][4];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  const int slot = s == 2 ? 1 : (s == 4 ? 2 : 3);
  int v = cache[dev][slot].load(std::memory_order_relaxed);
  if (v != 0) return v > 0 ? v : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(sm_count() / s * s));
  cfg.blockDim = dim3(SM_THREADS);
  cfg.dynamicSmemBytes = 227 * 1024;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(s);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (!ensure_dyn_smem(reinterpret_cast<const void*>(wo_gemm_stream_kernel), 227 * 1024) ||
      cudaOccupancyMaxActiveClusters(&n, wo_gemm_stream_kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  cache[dev][slot].store(n > 0 ? n : -1, std::memory_order_relaxed);
  return n;
}

sq_status_t launch_wo_stream(int rows, int splits, int blocks, const void* Z16, const void* Wq, const void* sw, int M, int N, int K,
                             void* Y, cudaStream_t s) {
  const int tiles = (N + rows - 1) / rows, ncl = std::min(tiles, blocks);
  const StreamLayout L = stream_layout(rows, SM_NT * 512, 8 / (rows > 32 ? 2 : 1) * SM_PART * 4, tiles <= blocks);
  auto kern = wo_gemm_stream_kernel;
  const int smem = L.total + 1024;
  if (!ensure_dyn_smem(reinterpret_cast<const void*>(kern), smem)) return SQ_ERR_CUDA;
  EncodeTiledFn enc = get_encode_fn();
  if (!enc) return SQ_ERR_CUDA;
  CUtensorMap mz, mw;
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(M)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(K) * 2};
  const cuuint32_t box[2] = {64, SM_NT};
  const cuuint32_t estr[2] = {1, 1};
  if (enc(&mz, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(Z16), dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return SQ_ERR_CUDA;
  if (!make_packed_map(&mw, Wq, N, K / 2, rows)) return SQ_ERR_CUDA;
  const cudaError_t err = launch_cluster_maybe_pdl(kern, dim3(static_cast<unsigned>(ncl * splits)), dim3(SM_THREADS),
                                                   static_cast<size_t>(smem), s, static_cast<unsigned>(splits), mw, mz, L,
                                                   static_cast<const __half*>(sw), M, N, K, splits, static_cast<__half*>(Y));
  count_launch();
  return err == cudaSuccess ? SQ_OK : SQ_ERR_CUDA;
}

// SMs for the product: the others are left to the tokens' rotation.  The next layer's may set itself up there, and none of this
// layer's keeps a block of the product off its SM.
int stream_blocks(int sms, int M) { return std::max(1, sms - std::min(M, 16)); }

// Channels per tile, even: as many as give every block the same share.
int stream_rows(int N, int blocks) {
  const int waves = (N + blocks * SM_MAX_ROWS - 1) / (blocks * SM_MAX_ROWS);
  const int rows = (N + blocks * waves - 1) / (blocks * waves);
  return std::max(8, (rows + 1) / 2 * 2);
}

}  // namespace

// Against the kernels that took these calls before: layers over 31 shapes, K 256 to 28672, 1 / 2 / 4 / 8 tokens, 1.07 / 1.12 / 1.15 /
// 1.31 on the geometric mean.  What stays with them, in us a layer, theirs and this kernel's:
//   one token, every warp of the dot products one task (N of 32 to 64 channels per SM), K from 2048 to 7168: all or most of the weights
//     are in registers before the token exists.  4096 x 8192 7.92 and 8.69, 4096 x 9472 7.40 and 8.85, 3072 x 5120 6.69 and 7.09,
//     6144 x 7168 9.09 and 9.99; beside it 4096 x 4096 6.70 and 6.58, 4096 x 10240 9.67 and 8.42, 8192 x 8192 12.1 and 11.6
//   two tokens likewise, K from 3072 to 4096: 4096 x 7104 7.60 and 8.58, 4096 x 5328 7.46 and 8.04 (N of whole 512 within 5 % either way)
//   one or two tokens, K beyond 16384, where the 33 to 48 channels of a tile are three blocks for two groups of warps:
//     28672 x 6144 23.1 and 25.9; x 4096 20.8 and 20.0, x 8192 32.7 and 27.2
//   three tokens and more, K beyond 16384 and N up to 8192, or K beyond 12288 and N up to 1024: every SM reads all the tokens, and
//     the decode kernel splits K over a cluster.  28672 x 1024 13.8 and 17.9, 20480 x 4096 15.1 and 16.3, 14336 x 1024 10.0 and 10.6;
//     beside it 28672 x 10240 34.7 and 30.7, 16384 x 4096 12.7 and 12.6, 14336 x 2048 11.5 and 10.7
static bool stream_yields(int64_t M, int64_t N, int64_t K) {
  const int64_t sms = sm_count();
  if (M > 2) return gemm_decode_supported(M, N, K) && (K > 16384 ? N <= 8192 : K > 12288 && N <= 1024);
  if (!gemv_supported(M, N, K) || N <= 32 * sms || N > 64 * sms) return false;
  if (K > 16384) return N <= 48 * sms;
  return M == 1 ? K >= 2048 && K <= 7168 : K >= 3072 && K <= 4096;
}

bool w4a4_stream_supported(int64_t M, int64_t N, int64_t K) {
  return M >= 1 && M <= SM_NT && N >= 128 && N % 2 == 0 && K % 32 == 0 && K >= 256 && !stream_yields(M, N, K);
}

// The product of a batch's last 1 to 8 tokens behind another product: launch, start and end, the walk along K, the weights.  (By
// itself it takes some 0.6 us less, within a tenth for K up to 14336; the rest is for what the two-pass choice also costs.)
double gemm_stream_estimate_us(int64_t N, int64_t K) { return 2.2 + 0.04 * ((K + 255) / 256) + 0.15e-6 * (0.5 * N * K); }

sq_status_t launch_w4a4_gemm_stream(const void* Xq, const void* sx, const void* Wq, const void* sw, int M, int N, int K, void* Y,
                                    int32_t* accdbg, cudaStream_t s) {
  const int sms = sm_count();
  if (sms <= 0) return SQ_ERR_CUDA;
  const int blocks = stream_blocks(sms, M), rows = stream_rows(N, blocks);
  const StreamLayout L = stream_layout(rows, SM_NT * 128, SM_NT * SM_RP8 * 4, false);
  const int grid = std::min((N + rows - 1) / rows, blocks);
  return launch_w4a4_stream(L, Xq, sx, Wq, sw, M, N, K, Y, accdbg, grid, s);
}

// Likewise (1 / 2 / 4 / 8 tokens: 1.24 / 1.35 / 1.34 / 1.34).  Small layers of one token stay with the dot products: 512 x 2048
// 4.46 us against 4.81, 1024 x 4096 5.20 and 5.47, 2048 x 3072 6.90 and 7.16; beside them 2048 x 4096 7.23 and 7.15, and however few the
// channels of longer rows 2560 x 1024 8.88 and 6.92, 8192 x 128 14.2 and 8.2, 14336 x 512 21.4 and 10.1.
bool wo_stream_supported(int64_t M, int64_t N, int64_t K) {
  return M >= 1 && M <= SM_NT && N >= 128 && N % 2 == 0 && K % 32 == 0 && K >= 256 && (M > 1 || K > 2048 || N * K / 2 >= 4000000);
}

sq_status_t launch_wo_gemm_stream(const void* Z16, const void* Wq, const void* sw, int M, int N, int K, void* Y, cudaStream_t s) {
  const int sms = sm_count();
  if (sms <= 0) return SQ_ERR_CUDA;
  const int num_sb = (K + 255) / 256, blocks = stream_blocks(sms, M);
  // Cycles of a block's share: its stages at some 40 bytes of weights and tokens a cycle (their MMAs, 32 per 16 channels, take
  // less), and what the cluster's exchange costs.  8 x 14336 -> 4096 with K in 1 / 2 / 4 / 8: 20.0 / 19.5 / 18.8 / 20.0 us,
  // 8 x 8192 -> 1024: 12.6 / 10.7 / 9.7 / 10.2.
  auto cost = [](int rows, int waves, int sbs, int splits) {
    return waves * sbs * (rows * 128.0 + SM_NT * 512.0) / 40.0 + (splits > 1 ? 1500.0 : 0.0);
  };
  int rows = stream_rows(N, blocks), splits = 1, clusters = blocks;
  double best = cost(rows, (N + rows * blocks - 1) / (rows * blocks), num_sb, 1);
  for (int sp = 2; sp <= 8 && num_sb / sp >= 2; sp *= 2) {
    const int ncl = std::min(wo_stream_clusters(sp), blocks / sp);
    if (ncl < 1 || N > ncl * SM_MAX_ROWS) continue;
    const int r = stream_rows(N, ncl);
    const double c = cost(r, 1, (num_sb + sp - 1) / sp, sp);
    if (c < best) {
      best = c;
      rows = r;
      splits = sp;
      clusters = ncl;
    }
  }
  return launch_wo_stream(rows, splits, clusters, Z16, Wq, sw, M, N, K, Y, s);
}

}  // namespace sq
