// Steps 1+2 on the tensor cores (sm_100a): Z_t = R1^T X~_t R2 (Eq. "eq18"), per-token absmax,
// INT4 quantisation (Section 3.2) and packing, one fused kernel.
//
// Both small contractions run as tcgen05.mma kind::f16 with fp32 accumulation in TMEM, with the
// operands split so that the result keeps fp32 accuracy:
//   stage 1  D1[p'][q]  = sum_p R1[p][p'] X~[p][q]     A = R1^T (shared memory, fp16 hi + lo),
//                                                      B = X~   (the TMA tile as it lands, used as
//                                                               an MN-major operand; exact fp16)
//   stage 2  D2[p'][q'] = sum_q D1[p'][q] R2[q][q']    A = D1   (TMEM, fp16 hi + lo, per-lane
//                                                               power-of-two scale),
//                                                      B = R2^T (shared memory, fp16 hi + lo)
// (hi*hi + lo*hi + hi*lo; the lo*lo term is below fp32 resolution).  TMEM lanes are the p' index,
// so a thread of the epilogue owns n2 CONSECUTIVE channels of one token (half of them where two warps
// share a lane): it packs them in registers and writes whole 32-byte sectors of the packed row straight
// to global memory (16 bytes where it has 32 channels), and a warp's stores are contiguous.
// 128 / LS tokens share one accumulator (LS = lanes per token, a power of two >= n1).  Stage 1 of all of them is one instruction
// of the weight-stationary form: R1^T's LS rows times the tokens side by side, whose columns it lays on successive lane ranges.
// (Before it each token took MMAs of its own, with R1^T's image shifted to its lanes and zero rows elsewhere: two or four times
// as many to issue and to run.
// Same bits; 11008 x 4096 37.4 -> 33.6 us, 2048 x 4096 11.2 -> 10.2, 777 x 4096 7.1 -> 6.1, fp16 rows 41.3 -> 36.6, 11.6 -> 9.7,
// 7.7 -> 6.6; packing 11008 x 4096 39.4 -> 35.5.)  Four tokens with n2 = 128 (n1 <= 32) have more columns than the 256 it takes:
// one instruction for the first 64 columns of each and one for the others (2048 x 3072 12.1 -> 11.6, fp16 rows 11.2 -> 10.5).  The
// zero rows let an infinity into the tokens beside its own, as NaN; now it stays in its row.  Both factors are stored
// pre-multiplied by 2^10 to keep
// the lo parts out of the fp16 subnormal range; every power-of-two factor is divided out exactly.
//
// Warp roles: warp 0 lane 0 = TMA producer, warp 1 lane 0 = MMA issuer, then the warps of the S
// accumulator slots: four each, or eight, two per lane quarter with half of the columns each (more
// warps to issue from while others wait).  Slot w handles the token groups w, w + S, ...: its warps
// convert D1 in place to fp16 hi/lo, and after stage 2 reduce the absmax, quantise, pack and store.
// While one slot waits for its MMAs the others compute.  Forms (launch_rotate_quant_tc):
//   n2 = 64    two CTAs per SM with two slots of four warps; one CTA with four slots where the images
//              leave no room for that
//   n2 = 128   one CTA per SM, two slots of eight warps
//   few tokens one slot of eight warps, one token at a time
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "sq_internal.h"
#include "sq_ptx.cuh"

namespace sq {
namespace {

constexpr float kFactorScale = 1024.0f;           // 2^10 applied to R1 and R2 in the images
constexpr int kFactorScaleLog2 = 10;
constexpr int kMaxDynSmem = 227 * 1024;
constexpr int kHalfDynSmem = 113 * 1024;        // two CTAs per SM

enum RqSite : uint32_t { RQ_X_EMPTY = 16, RQ_X_FULL, RQ_D_FREE, RQ_A2_READY, RQ_D1_FULL, RQ_D2_FULL, RQ_IMG };

// Byte offset of element (row r, k) inside a K-major tile with 128-byte rows and 128-byte swizzle.
inline size_t sw128_offset(int r, int k) { return static_cast<size_t>(r) * 128 + ((((k >> 3) ^ (r & 7))) << 4) + (k & 7) * 2; }

struct RqLayout {
  int LS, G, N1, KA1, XQ, S, XS, rowsA;
  int a1_tile, a1_part, a1_bytes, b2_tile, b2_part, b2_bytes, x_tile, x_token, x_bytes;
  int off_a1, off_b2, off_x, off_misc, total;
  int parts;            // instructions per step of stage 1 when several tokens share an accumulator
};

// `one_token`: one token per accumulator (the other lanes stay zero) instead of as many as fit.
__host__ __device__ inline RqLayout rq_layout(int n1, int n2, int budget = kMaxDynSmem, bool one_token = false) {
  RqLayout L;
  L.LS = n1 <= 32 ? 32 : (n1 <= 64 ? 64 : 128);   // TMEM lanes per token
  L.G = one_token ? 1 : 128 / L.LS;               // tokens per accumulator
  L.parts = L.G * n2 <= 256 ? 1 : 2;              // the N of one is 256 at most
  L.N1 = (n1 + 15) & ~15;                         // K of stage 1, padded to the MMA's K = 16
  L.KA1 = (L.N1 + 63) / 64;                       // 64-wide K atoms of stage 1
  L.XQ = n2 / 64;                                 // 64-wide column blocks of a token
  L.S = 256 / n2;                                 // accumulator slots
  L.rowsA = 256 - L.LS;
  L.a1_tile = L.rowsA * 128;
  L.a1_part = L.KA1 * L.a1_tile;
  L.a1_bytes = 2 * L.a1_part;
  L.b2_tile = n2 * 128;
  L.b2_part = L.XQ * L.b2_tile;
  L.b2_bytes = 2 * L.b2_part;
  L.x_tile = L.N1 * 128;
  L.x_token = L.XQ * L.x_tile;
  L.x_bytes = L.G * L.x_token;
  L.off_a1 = 0;
  L.off_b2 = L.off_a1 + L.a1_bytes;
  L.off_x = L.off_b2 + L.b2_bytes;
  // per-lane absmax swap of the forms with eight warps per slot: [slots][2][128 lanes] floats, behind the barriers
  const int extra = one_token ? 1024 : (n2 == 128 ? 2048 : 0);
  const int room = budget - 1024 - 512 - extra - L.off_x;
  const int xs = room / L.x_bytes;
  L.XS = xs > 4 ? 4 : xs;                         // X ring depth
  L.off_misc = L.off_x + L.XS * L.x_bytes;
  L.total = L.off_misc + 512 + extra;
  return L;
}

// Shared-memory descriptor of an MN-major operand with the 128-byte swizzle: 64 elements along
// N are contiguous (one 128-byte row), 8 consecutive K rows form a 1024-byte atom, `lbo_bytes`
// separates successive groups of 64 along N.
__device__ __forceinline__ uint64_t umma_desc_sw128_mn(uint32_t smem_addr, uint32_t lbo_bytes) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>(1024 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

// Untiled bulk copy global -> shared, completion counted on an mbarrier (16-byte aligned, size a
// multiple of 16).
__device__ __forceinline__ void bulk_load_1d(void* smem_dst, const void* gmem_src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(gmem_src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ uint32_t pack_half2(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// Eight consecutive codes -> one packed word.  u_i = floor(t_i) + 8 is taken from the low bits of
// t_i + (2^23 + 8) rounded towards -inf (no conversion instruction); the words' common high bits
// cancel in `kBias`; flipping bit 3 of every nibble turns the offset code into two's complement.
__device__ __forceinline__ uint32_t join8_codes(const float* u) {
  constexpr uint32_t kBias = 0x4B000000u * 0x11111111u;
  uint32_t w = __float_as_uint(u[7]);
#pragma unroll
  for (int i = 6; i >= 0; --i) w = w * 16u + __float_as_uint(u[i]);
  return (w - kBias) ^ 0x88888888u;
}
__device__ __forceinline__ uint32_t pack8_codes(const float* t) {
  float u[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) u[i] = __fadd_rd(t[i], 8388616.0f);
  return join8_codes(u);
}

// Two fp32 numbers in a register pair: one instruction works on both, each rounded as the scalar form rounds it.  The warps
// of these kernels issued on 64 % of the cycles with scalar steps (11008 x 4096, 47 us) and do on 51 % with these (37 us).
using F2 = unsigned long long;

__device__ __forceinline__ F2 f2_pack(float a, float b) {
  F2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ void f2_unpack(F2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  F2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ F2 f2_add_rd(F2 a, F2 b) {
  F2 d;
  asm("add.rm.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) {
  F2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float absmax3(float a, float b, float c) {
  float d;
  asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// One whole 32-byte sector per lane: the lanes of a warp write rows that are 32 bytes (packed codes) to 256 bytes (fp16)
// apart, and sectors written in two halves cost twice.  The buffers are only promised to be 16-byte aligned.
__device__ __forceinline__ void store_sector(void* p, const uint32_t* v, bool aligned32) {
  if (aligned32) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
                 "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
  } else {
    static_cast<uint4*>(p)[0] = make_uint4(v[0], v[1], v[2], v[3]);
    static_cast<uint4*>(p)[1] = make_uint4(v[4], v[5], v[6], v[7]);
  }
}

// Eight rotated values -> one packed word: code = floor(z / Delta + 1/2), product and sum rounded on their own.  The sum is
// taken one by one: as a pair behind the pair product it was contracted into a fused multiply-add for all its ".rn", and
// one code in some 5e7 came out one lower.
template <bool CLAMP>
__device__ __forceinline__ uint32_t codes8(const float* z, F2 inv2) {
  const F2 magic2 = f2_pack(8388616.0f, 8388616.0f);
  float u[8];
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    float a, b;
    f2_unpack(f2_mul(f2_pack(z[e], z[e + 1]), inv2), a, b);
    a = __fadd_rn(a, 0.5f);
    b = __fadd_rn(b, 0.5f);
    if (CLAMP) {
      a = fminf(fmaxf(a, -8.0f), 7.5f);
      b = fminf(fmaxf(b, -8.0f), 7.5f);
    }
    f2_unpack(f2_add_rd(f2_pack(a, b), magic2), u[e], u[e + 1]);
  }
  return join8_codes(u);
}

// 32 rotated values -> 16 packed bytes.
template <bool CLAMP>
__device__ __forceinline__ void codes32(const float* z, F2 inv2, uint32_t* pk) {
#pragma unroll
  for (int e = 0; e < 4; ++e) pk[e] = codes8<CLAMP>(z + 8 * e, inv2);
}

// max |D| over the HC columns of a lane from TMEM column `d` on (four independent chains).  `r` keeps the last 32 columns:
// the pass that follows starts with those and reads the others once more.
template <int HC>
__device__ __forceinline__ float lane_absmax(uint32_t d, uint32_t (&r)[32]) {
  float m[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int c = 0; c < HC / 32; ++c) {
    tmem_ld_32x32b_x32(d + 32 * c, r);
    tmem_wait_ld();
#pragma unroll
    for (int e = 0; e < 32; e += 8)
#pragma unroll
      for (int x = 0; x < 4; ++x)
        m[x] = absmax3(m[x], __uint_as_float(r[e + 2 * x]), __uint_as_float(r[e + 2 * x + 1]));
  }
  return fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
}

// The lane's power-of-two scale `sc`, chosen so that its largest entry lands in [2^13, 2^14), and `un`, which divides it
// and the two factor scales out again exactly: z = D2 * 2^-(k + 20).
__device__ __forceinline__ void lane_scale(float m, float& sc, float& un) {
  const int ebits = static_cast<int>((__float_as_uint(m) >> 23) & 0xFF);
  int k = 13 - (ebits - 127);
  if (m == 0.0f) k = 0;
  k = max(-126, min(127, k));
  sc = __uint_as_float(static_cast<uint32_t>(k + 127) << 23);
  const int uexp = -(k + 2 * kFactorScaleLog2) + 127;
  un = (uexp >= 1) ? __uint_as_float(static_cast<uint32_t>(min(uexp, 254)) << 23) : 0.0f;
}

// D1 -> fp16 hi + lo of D1 * sc in place: 16 fp32 columns become 8 columns of hi and 8 of lo.  `r` holds the last 32
// columns.  (v sc is exact unless it underflows, and then hi is 0: the difference is what the fused form would give.)
template <int HC>
__device__ __forceinline__ void split_in_place(uint32_t d1, uint32_t (&r)[32], float sc) {
  const F2 sc2 = f2_pack(sc, sc);
#pragma unroll
  for (int c = HC / 32 - 1; c >= 0; --c) {
    uint32_t o[32];
    if (c < HC / 32 - 1) {
      tmem_ld_32x32b_x32(d1 + 32 * c, r);
      tmem_wait_ld();
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const F2 v = f2_mul(f2_pack(__uint_as_float(r[16 * h + 2 * e]), __uint_as_float(r[16 * h + 2 * e + 1])), sc2);
        float a, b;
        f2_unpack(v, a, b);
        const __half2 hh = __floats2half2_rn(a, b);
        const float2 hf = __half22float2(hh);
        f2_unpack(f2_sub(v, f2_pack(hf.x, hf.y)), a, b);
        o[16 * h + e] = *reinterpret_cast<const uint32_t*>(&hh);
        o[16 * h + 8 + e] = pack_half2(a, b);
      }
    tmem_st_32x32b_x32(d1 + 32 * c, o);
  }
}

// The lane's HC columns of D2, times `un`, as fp16 (the weight-only variant: nothing is quantised).
template <int HC>
__device__ __forceinline__ void store_rotated_f16(uint32_t d2, float un, __half* __restrict__ zrow, bool live) {
  const F2 un2 = f2_pack(un, un);
  const bool aligned32 = (reinterpret_cast<uintptr_t>(zrow) & 31) == 0;
#pragma unroll
  for (int c = 0; c < HC / 32; ++c) {
    uint32_t r[32], o[16];
    tmem_ld_32x32b_x32(d2 + 32 * c, r);
    tmem_wait_ld();
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      float a, b;
      f2_unpack(f2_mul(f2_pack(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1])), un2), a, b);
      o[e] = pack_half2(a, b);
    }
    if (live) {
      store_sector(zrow + 32 * c, o, aligned32);
      store_sector(zrow + 32 * c + 16, o + 8, aligned32);
    }
  }
}

// Quantises, packs and stores the lane's HC columns of D2.  `r` holds the last 32 columns; `inv_un` = un / Delta (exact, a
// power of two times 1 / Delta).  Delta >= 2^-14 (a normal fp16) bounds |z / Delta| by 7 (1 + 2^-11): no clamp is needed then.
template <int HC>
__device__ __forceinline__ void store_codes(uint32_t d2, uint32_t (&r)[32], __half delta, float inv_un, float un, bool live,
                                            uint8_t* __restrict__ orow, float* __restrict__ zrow) {
  const F2 inv2 = f2_pack(inv_un, inv_un);
  const bool aligned32 = (reinterpret_cast<uintptr_t>(orow) & 31) == 0;
  uint32_t pk[HC / 8];
  const bool clamp = __half2float(delta) < 6.103515625e-05f;
#pragma unroll
  for (int c = HC / 32 - 1; c >= 0; --c) {
    if (c < HC / 32 - 1) {
      tmem_ld_32x32b_x32(d2 + 32 * c, r);
      tmem_wait_ld();
    }
    const float* z = reinterpret_cast<const float*>(r);
    if (clamp) codes32<true>(z, inv2, pk + 4 * c);
    else codes32<false>(z, inv2, pk + 4 * c);
    if (live) {
      if (zrow) {
#pragma unroll
        for (int e = 0; e < 32; e += 4)
          *reinterpret_cast<float4*>(zrow + 32 * c + e) = make_float4(z[e] * un, z[e + 1] * un, z[e + 2] * un, z[e + 3] * un);
      }
    }
  }
  if (live) {
    if constexpr (HC == 32) {
      *reinterpret_cast<uint4*>(orow) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    } else {
#pragma unroll
      for (int c = 0; c < HC / 64; ++c) store_sector(orow + 32 * c, pk + 8 * c, aligned32);
    }
  }
}

// Shared memory that a launch asks for.  Forms that want an SM of their own ask for more than half of it.  No form asks for so
// little that a CTA-pair rotation (142 KB and more) fits beside it: dependents may start before a CTA has allocated its tensor
// memory, one that took all 512 columns first would leave it waiting, and then wait for it.
constexpr int kAloneSmem = 120 * 1024, kLeastSmem = 88 * 1024;
inline int rq_smem(const RqLayout& L, int ctas_per_sm) { return std::max(L.total + 1024, ctas_per_sm == 1 ? kAloneSmem : kLeastSmem); }

// The kernel's body, for CTA `cta` of `ncta` that share the token groups (the fused decode kernel of
// sq_linear_fused.cu runs it in its first CTAs, with more warps in the block than the roles below use).
// `TOKENS`: one token per accumulator (1) or several (2), where that is known when the kernel is compiled; 0: by the layout.  With
// the choice left to the kernel the MMA issuer lost time over it: 1 x 4096 3.65 us against 3.55, 50 x 14336 (112 x 128) 5.85
// against 5.68, 2048 x 14336 32.8 against 31.1; three MLP layers of 50 tokens 49.8 against 47.9.
template <int N2, int S, int CW = 1, bool F16OUT = false, int TOKENS = 0>
__device__ __forceinline__ void rotate_quant_tc_body(const CUtensorMap& tmap_x, const RqLayout& L,
                                                     const unsigned char* __restrict__ a1_img,
                                                     const unsigned char* __restrict__ b2_img, int n1, int rows,
                                                     uint8_t* __restrict__ Xq, __half* __restrict__ scales,
                                                     float* __restrict__ Zdbg, int cta, int ncta) {
  constexpr int TM_COLS = S * 2 * N2;             // 256 or 512
  constexpr int XQ = N2 / 64;
  constexpr int SLOT_COLS = 2 * N2;              // D1 (N2 columns) + D2 (N2 columns)
  // The layout comes from the host (the same rq_layout call that sized the shared memory); group
  // counts are 32-bit: the set-up is on the critical path of a decode step.
  const int n = n1 * N2;
  const int G = TOKENS == 1 ? 1 : L.G, LS = L.LS;

  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  unsigned char* a1s = smem + L.off_a1;
  unsigned char* b2s = smem + L.off_b2;
  unsigned char* xs = smem + L.off_x;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.off_misc);
  uint64_t* x_full = bars;             // [4]
  uint64_t* x_empty = bars + 4;        // [4]
  uint64_t* d1_full = bars + 8;        // [4]
  uint64_t* a2_ready = bars + 12;      // [4]
  uint64_t* d2_full = bars + 16;       // [4]
  uint64_t* img_full = bars + 24;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 25);
  float* amax_x = reinterpret_cast<float*>(bars + 26);      // [S groups][2 parities][4 warps]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ngroups = (rows + G - 1) / G;
  const int my_groups = (ngroups > cta) ? (ngroups - cta + ncta - 1) / ncta : 0;
  const uint32_t limit = wait_limit();

  // One X tile set per token group: G tokens, XQ 64-column blocks each.
  auto load_group = [&](int i, int s) {                  // group i -> ring stage s
    const int g = cta + i * ncta;
    mbar_arrive_expect_tx(&x_full[s], static_cast<uint32_t>(L.x_bytes));
    for (int tk = 0; tk < G; ++tk)
      for (int a = 0; a < XQ; ++a)
        tma_load_3d(xs + s * L.x_bytes + tk * L.x_token + a * L.x_tile, &tmap_x, &x_full[s], a * 64, 0,
                    g * G + tk);
  };
  const int preload = my_groups < L.XS ? my_groups : L.XS;

  if (threadIdx.x == 0) {
    // The first loads go out before anything else is set up: the factor images (they belong to the
    // handle, so they may be fetched while the kernel before this one in the stream still runs), then,
    // once that kernel has completed (it may have produced X, and may still be reading the buffers this
    // one writes), the whole X ring.  Every store of this kernel depends on X having landed.  Only the
    // barriers the loads complete on exist at that point; nobody else touches a barrier before the
    // __syncthreads below.
    for (int b = 0; b < 4; ++b) mbar_init(&x_full[b], 1);
    mbar_init(img_full, 1);
    mbar_fence_init();
    mbar_arrive_expect_tx(img_full, static_cast<uint32_t>(L.a1_bytes + L.b2_bytes));
    for (int o = 0; o < L.a1_bytes; o += 16384)
      bulk_load_1d(a1s + o, a1_img + o, static_cast<uint32_t>(min(16384, L.a1_bytes - o)), img_full);
    for (int o = 0; o < L.b2_bytes; o += 16384)
      bulk_load_1d(b2s + o, b2_img + o, static_cast<uint32_t>(min(16384, L.b2_bytes - o)), img_full);
    griddep_wait();
    // Only now may a GEMM launched behind this kernel start: it requests its weights before it waits for
    // this kernel, and whatever precedes this kernel (sq_pack_weight, say) may have been writing them.
    // (Not later either: behind the tensor memory's allocation, 4 x 11008 -> 4096 took 11.3 us instead of 10.8.)
    griddep_launch_dependents();
    for (int i = 0; i < preload; ++i) load_group(i, i);
    for (int b = 0; b < 4; ++b) {
      mbar_init(&x_empty[b], 1);
      mbar_init(&d1_full[b], 1);
      mbar_init(&a2_ready[b], 4 * CW);
      mbar_init(&d2_full[b], 1);
    }
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, TM_COLS);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------ producer: keeps the X ring full -------------------------------------
    if (lane == 0) {
      int s = 0;                                       // preload == XS here: ring stage and phase are counted along
      uint32_t ph = 0;
      for (int i = preload; i < my_groups; ++i) {
        if (!mbar_wait(&x_empty[s], ph, RQ_X_EMPTY, limit)) break;
        load_group(i, s);
        if (++s == L.XS) {
          s = 0;
          ph ^= 1;
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------------------------------
    if (elect_one()) {
      // stage 1: A K-major (shared), B MN-major (bit 16); stage 2: A from TMEM, B K-major
      const uint32_t idesc1 = umma_idesc(/*c=f32*/ 1, /*a=f16*/ 0, /*b=f16*/ 0, 128, N2) | (1u << 16);
      const uint32_t idesc2 = umma_idesc(/*c=f32*/ 1, /*a=f16*/ 0, /*b=f16*/ 0, 128, N2);
      // weight-stationary: M = LS rows, N = the columns of G tokens, whose tiles follow one another at the stride of a column block,
      // or 64 columns of each at the stride of a token
      const bool halves = N2 == 128 && TOKENS != 1 && L.parts == 2;
      const uint32_t idesc_ws = umma_idesc(1, 0, 0, static_cast<uint32_t>(LS), static_cast<uint32_t>((halves ? 64 : N2) * G)) | (1u << 16);
      const uint64_t a1_desc0 = umma_desc_sw128(smem_u32(a1s)), b2_desc0 = umma_desc_sw128(smem_u32(b2s));
      const uint64_t x_desc0 = umma_desc_sw128_mn(smem_u32(xs), static_cast<uint32_t>(halves ? L.x_token : L.x_tile));
      const int ksteps1 = L.N1 / 16;                 // K = p, 16 per MMA
      bool ok = mbar_wait(img_full, 0, RQ_IMG, limit);
      auto stage1 = [&](int i, int xs_i) {
        const int slot = i % S;
        tc_fence_after_sync();
        const uint32_t d1 = tmem_base + slot * SLOT_COLS;
        // descriptors differ only in their start-address field (16-byte units, no carry out of it)
        const uint64_t ad = a1_desc0 + (((128 - LS) * 128) >> 4), bd0 = x_desc0 + ((xs_i * L.x_bytes) >> 4);
        if (TOKENS == 2 || (TOKENS == 0 && G > 1)) {
          auto steps = [&](uint32_t d, uint64_t bd) {
            uint32_t acc = 0;
#pragma unroll 2                                       // 333 x 4096 4.76 us, 4.86 with the compiler's four
            for (int ks = 0; ks < ksteps1; ++ks, bd += 2048 >> 4) {
              const uint64_t ah = ad + (((ks >> 2) * L.a1_tile + (ks & 3) * 32) >> 4);
              umma_f16_ws(d, ah, bd, idesc_ws, acc);                       // hi
              umma_f16_ws(d, ah + (L.a1_part >> 4), bd, idesc_ws, 1u);     // lo
              acc = 1;
            }
          };
          steps(d1, bd0);
          if (halves) steps(d1 + 64, bd0 + (L.x_tile >> 4));
        } else {
          uint64_t bd = bd0;
          uint32_t acc = 0;
          for (int ks = 0; ks < ksteps1; ++ks, bd += 2048 >> 4) {
            const uint64_t ah = ad + (((ks >> 2) * L.a1_tile + (ks & 3) * 32) >> 4);
            umma_f16(d1, ah, bd, idesc1, acc);
            umma_f16(d1, ah + (L.a1_part >> 4), bd, idesc1, 1u);
            acc = 1;
          }
        }
        umma_commit(&x_empty[xs_i]);
        umma_commit(&d1_full[slot]);
      };
      auto stage2 = [&](int i) {
        const int slot = i % S;
        tc_fence_after_sync();
        const uint32_t d1 = tmem_base + slot * SLOT_COLS, d2 = d1 + N2;
#pragma unroll
        for (int j = 0; j < N2 / 16; ++j) {
          const uint64_t bh = b2_desc0 + (((j >> 2) * L.b2_tile + (j & 3) * 32) >> 4), bl = bh + (L.b2_part >> 4);
          umma_f16_ts(d2, d1 + 16 * j, bh, idesc2, j > 0 ? 1u : 0u);      // hi * hi
          umma_f16_ts(d2, d1 + 16 * j + 8, bh, idesc2, 1u);               // lo * hi
          umma_f16_ts(d2, d1 + 16 * j, bl, idesc2, 1u);                   // hi * lo
        }
        umma_commit(&d2_full[slot]);
      };
      // Whichever is ready goes: stage 1 of the next group whose X tile has landed and whose slot's D1
      // columns are free, and stage 2 of the oldest group whose operand has been converted.  D1 is free
      // as soon as stage 2 of the slot's previous group has completed (it was that stage's A operand),
      // so stage 1 of the next group runs while the previous one is still being quantised out of the D2
      // columns; D2 is not written again before the group's warps have finished reading it, because
      // they convert the next group (which is what lets its stage 2 go) only after that.
      // (Ring stage and phase of X are counted along: XS is a run-time number, and a division per poll cost more than what
      // it polled for.)
      int i1 = 0, i2 = 0, xr = 0;
      uint32_t xph = 0;
      uint32_t idle = 0;
      while (ok && i2 < my_groups) {
        bool did = false;
        if (i1 < my_groups && i1 < i2 + S &&
            mbar_test_wait(&x_full[xr], xph) &&
            mbar_test_wait(&d2_full[i1 % S], ((i1 / S) & 1) ^ 1)) {
          stage1(i1++, xr);
          if (++xr == L.XS) {
            xr = 0;
            xph ^= 1;
          }
          did = true;
        }
        if (i2 < i1 && mbar_test_wait(&a2_ready[i2 % S], (i2 / S) & 1)) {
          stage2(i2++);
          did = true;
        }
        if (did) {
          idle = 0;
        } else if (++idle > limit) {
          atomicCAS(&g_device_status, 0u, (static_cast<uint32_t>(RQ_A2_READY) << 8) | 1u);
          ok = false;
        }
      }
    }
  } else if (warp < 2 + 4 * S * CW) {
    // ------------------------------ compute groups ------------------------------------------------
    // CW warps per lane quarter: warp (quarter, cp) owns columns [cp * HC, (cp + 1) * HC) of it.
    constexpr int HC = N2 / CW;                    // columns per warp
    const int gi = (warp - 2) >> 2;
    const int w = gi / CW, cp = gi % CW;           // accumulator slot of this group
    const int quarter = warp & 3;                  // TMEM lane quarter this warp may touch
    const int lane_g = quarter * 32 + lane;        // accumulator lane = token-in-group * LS + p'
    const int tk = lane_g / LS, pp = lane_g % LS;
    const uint32_t lane_addr = static_cast<uint32_t>(quarter * 32) << 16;
    const uint32_t d1 = tmem_base + w * SLOT_COLS + lane_addr + cp * HC, d2 = d1 + N2;
    const int wpt = LS / 32;                       // lane quarters that share a token
    const int q0 = (quarter / wpt) * wpt;
    float* lane_m = reinterpret_cast<float*>(smem + L.off_misc + 512);       // CW == 2: [S][2][128 lanes]
    bool ok = true;
    for (int i = w; i < my_groups && ok; i += S) {
      const int g = cta + i * ncta;
      const long long token = static_cast<long long>(g) * G + tk;
      const uint32_t ph = (i / S) & 1;
      const bool live = (pp < n1) && (tk < G) && (token < rows);
      uint32_t r[32];

      // ---- D1 -> fp16 hi/lo in place, with a per-lane power-of-two scale --------------------------
      ok = mbar_wait(&d1_full[w], ph, RQ_D1_FULL, limit);
      if (!ok) break;
      tc_fence_after_sync();
      float m = lane_absmax<HC>(d1, r);
      if constexpr (CW == 2) {
        // The lane's scale must be the same in the two warps that share the lane.
        lane_m[(w * 2 + cp) * 128 + lane_g] = m;
        named_barrier(1 + w, 256);
        m = fmaxf(m, lane_m[(w * 2 + (cp ^ 1)) * 128 + lane_g]);
      }
      float sc, un;
      lane_scale(m, sc, un);
      split_in_place<HC>(d1, r, sc);
      tmem_wait_st();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&a2_ready[w]);

      // ---- D2: absmax over the token, quantise, pack, store ------------------------------------------
      ok = mbar_wait(&d2_full[w], ph, RQ_D2_FULL, limit);
      if (!ok) break;
      tc_fence_after_sync();
      if constexpr (F16OUT) {
        store_rotated_f16<HC>(d2, un, reinterpret_cast<__half*>(Xq) + token * n + pp * N2 + cp * HC, live);
        continue;
      }
      float zm = lane_absmax<HC>(d2, r) * un;        // lanes of padding rows hold exact zeros
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) zm = fmaxf(zm, __shfl_xor_sync(0xffffffffu, zm, o));
      float* amax_w = amax_x + (w * 2 + ph) * 4 * CW;
      if (lane == 0) amax_w[quarter * CW + cp] = zm;
      named_barrier(1 + w, 128 * CW);
      float amax = amax_w[q0 * CW];
      for (int x = 1; x < wpt * CW; ++x) amax = fmaxf(amax, amax_w[q0 * CW + x]);
      __half delta;
      float inv;
      row_scale(amax, delta, inv);
      store_codes<HC>(d2, r, delta, inv * un, un, live, Xq + token * (n / 2) + pp * (N2 / 2) + cp * (HC / 2),
                      (Zdbg != nullptr && live) ? Zdbg + token * n + pp * N2 + cp * HC : nullptr);
      if (live && pp == 0 && cp == 0) scales[token] = delta;
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, TM_COLS);
  }
}

// S accumulator slots (= compute groups) per CTA.  With S * 2 * N2 = 256 TMEM columns two CTAs share
// an SM (each with its own producer and MMA issuer); with 512 a CTA has the SM to itself.
template <int N2, int S, int CW = 1, bool F16OUT = false, int TOKENS = 0>
__global__ void __launch_bounds__((2 + 4 * S * CW) * 32, (CW == 1 && S * 2 * N2 <= 256) ? 2 : 1)
rotate_quant_tc_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ RqLayout L,
                       const unsigned char* __restrict__ a1_img, const unsigned char* __restrict__ b2_img, int n1,
                       int rows, uint8_t* __restrict__ Xq, __half* __restrict__ scales, float* __restrict__ Zdbg) {
  rotate_quant_tc_body<N2, S, CW, F16OUT, TOKENS>(tmap_x, L, a1_img, b2_img, n1, rows, Xq, scales, Zdbg, static_cast<int>(blockIdx.x),
                              static_cast<int>(gridDim.x));
}

// ---------------------------------------------------------------------------------------------
// Host: factor images (the exact shared-memory bytes: fp16 hi/lo, 2^10 pre-scale, swizzled)
// ---------------------------------------------------------------------------------------------
void split_half(float v, __half& hi, __half& lo) {
  hi = __float2half_rn(v);
  lo = __float2half_rn(v - __half2float(hi));
}

void put_half(std::vector<unsigned char>& img, size_t off, __half h) {
  const unsigned short u = __half_as_ushort(h);
  img[off] = static_cast<unsigned char>(u & 0xFF);
  img[off + 1] = static_cast<unsigned char>(u >> 8);
}

}  // namespace

bool rotate_quant_tc_supported(int n1, int n2) {
  if (n2 != 64 && n2 != 128) return false;
  if (n1 < 1 || n1 > 128) return false;
  return rq_layout(n1, n2).XS >= 2;
}

// Builds and uploads the two images for a handle.  Returns false on a CUDA failure.
bool rotate_quant_tc_prepare(sq_rotation* h) {
  const int n1 = h->n1, n2 = h->n2;
  const RqLayout L = rq_layout(n1, n2);
  std::vector<unsigned char> a1(L.a1_bytes, 0), b2(L.b2_bytes, 0);
  // A1 (stage-1 A operand): rows = lanes, K = p.  R1^T sits at rows [128 - LS, 128 - LS + n1) of a (256 - LS)-row image.  A
  // single token takes 128 rows from there on, which leaves zeros on the lanes behind its own; several tokens side by side take
  // LS.  (The zero rows ahead of R1^T belong to images shifted to the other tokens' lanes, which nothing uses any more; they
  // are still copied into every CTA, and room for X is lost to them.)
  for (int pp = 0; pp < n1; ++pp)
    for (int p = 0; p < n1; ++p) {
      __half hi, lo;
      split_half(kFactorScale * h->R1[static_cast<size_t>(p) * n1 + pp], hi, lo);
      const size_t off = static_cast<size_t>(p / 64) * L.a1_tile + sw128_offset(128 - L.LS + pp, p % 64);
      put_half(a1, off, hi);
      put_half(a1, static_cast<size_t>(L.a1_part) + off, lo);
    }
  // B2 (stage-2 B operand): rows q', K = q, value 2^10 * R2[q][q']
  for (int qp = 0; qp < n2; ++qp)
    for (int q = 0; q < n2; ++q) {
      __half hi, lo;
      split_half(kFactorScale * h->R2[static_cast<size_t>(q) * n2 + qp], hi, lo);
      const size_t off = static_cast<size_t>(q / 64) * L.b2_tile + sw128_offset(qp, q % 64);
      put_half(b2, off, hi);
      put_half(b2, static_cast<size_t>(L.b2_part) + off, lo);
    }
  if (cudaMalloc(&h->dA1img, a1.size()) != cudaSuccess || cudaMalloc(&h->dB2img, b2.size()) != cudaSuccess ||
      cudaMemcpy(h->dA1img, a1.data(), a1.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(h->dB2img, b2.data(), b2.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  h->tc_ready = true;
  return true;
}

sq_status_t launch_rotate_quant_tc(const sq_rotation* h, const void* X, int64_t rows, void* Xq, void* scales,
                                   float* Zdbg, cudaStream_t s, bool f16out) {
  const int n1 = h->n1, n2 = h->n2;
  if (rows > 0x7FFFFFFF) return SQ_ERR_UNSUPPORTED;   // the kernel counts token groups in 32 bits
  // n2 = 64 with images small enough: two CTAs per SM, two accumulator slots each.
  const RqLayout Lh = rq_layout(n1, n2, kHalfDynSmem);
  const bool dual = (n2 == 64) && Lh.XS >= 2;
  // A handful of tokens: latency is all there is.  One token per accumulator (a group's stage 1 is half or a quarter as
  // long) and eight warps on it also with n2 = 64; the sums are the same, in the same order.  16 x 4096 (64 x 64): 4.57 ->
  // 3.86 us, layer to 14336 11.5 -> 10.7.
  // The quantising form asks for an SM of its own (120 KB: the layer for one token 11.1 us without, 9.9 with) and keeps the
  // product's CTA off it.  Hence no more than 16 tokens: many layers have 128 such CTAs in clusters, and beyond 20 tokens the
  // last of them wait for the rotation to end (32 x 4096 -> 4096 10.2 us, 9.1 in the other form; 32 x 8192 -> 4096 12.9 and
  // 11.8; against that 24 x 8192 -> 1024 9.9 and 10.2).  The fp16 form shares its SM (18.4 us, alone on it 25: the
  // dot-product kernel behind it then doubles up on another SM) and goes up to 32.
  const bool few = rows <= (f16out ? 32 : 16);
  const RqLayout L = few ? rq_layout(n1, n2, kMaxDynSmem, true) : (dual ? Lh : rq_layout(n1, n2));
  EncodeTiledFn enc = get_encode_fn();
  if (!enc) return SQ_ERR_CUDA;
  CUtensorMap mx;
  const cuuint64_t dims[3] = {static_cast<cuuint64_t>(n2), static_cast<cuuint64_t>(n1), static_cast<cuuint64_t>(rows)};
  const cuuint64_t strides[2] = {static_cast<cuuint64_t>(n2) * 2, static_cast<cuuint64_t>(n1) * n2 * 2};
  const cuuint32_t box[3] = {64, static_cast<cuuint32_t>(L.N1), 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  if (enc(&mx, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(X), dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return SQ_ERR_CUDA;
  const int sms = sm_count();
  if (sms <= 0) return SQ_ERR_CUDA;
  const long long ngroups = (rows + L.G - 1) / L.G;
  const unsigned char* a1 = static_cast<const unsigned char*>(h->dA1img);
  const unsigned char* b2 = static_cast<const unsigned char*>(h->dB2img);
  auto launch = [&](auto n2_c, auto slots_c, auto cw_c, auto f16_c, int ctas_per_sm) -> bool {
    constexpr int N2 = decltype(n2_c)::value, S = decltype(slots_c)::value, CW = decltype(cw_c)::value;
    constexpr bool F16 = decltype(f16_c)::value;
    auto kern = rotate_quant_tc_kernel<N2, S, CW, F16, 1>;
    if constexpr (S == 2) {                          // one slot is one token at a time; four are for n1 > 64
      if (L.G > 1) kern = rotate_quant_tc_kernel<N2, S, CW, F16, 2>;
    }
    const int smem = rq_smem(L, ctas_per_sm);
    if (!ensure_dyn_smem(reinterpret_cast<const void*>(kern), smem)) return false;
    const unsigned grid = static_cast<unsigned>(std::min<long long>(ngroups, static_cast<long long>(sms) * ctas_per_sm));
    return launch_dependent(kern, dim3(grid), dim3((2 + 4 * S * CW) * 32), static_cast<size_t>(smem), s, mx, L, a1, b2, n1,
                            static_cast<int>(rows), static_cast<uint8_t*>(Xq), static_cast<__half*>(scales),
                            Zdbg) == cudaSuccess;
  };
  // n2 = 128 (one CTA per SM, two slots): eight warps per slot, 18 in all instead of 10 -- measured 10 %
  // faster on 4096 x 8192 (39.7 -> 35.5 us) and 0.8 us on the decode batches (6.6 -> 5.8 us).  With n2 = 64
  // and two CTAs per SM the same split leaves 56 registers per thread and was slower (12.0 -> 15.9 us).
  using std::integral_constant;
  auto form = [&](auto f16) -> bool {                // rotation only: Xq receives the rotated rows as fp16, `scales` is not touched
    const integral_constant<int, 64> c64;
    const integral_constant<int, 128> c128;
    const integral_constant<int, 1> one;
    const integral_constant<int, 2> two;
    if (few) return n2 == 64 ? launch(c64, one, two, f16, f16 ? 2 : 1) : launch(c128, one, two, f16, f16 ? 2 : 1);
    if (n2 == 128) return launch(c128, two, two, f16, 1);
    return dual ? launch(c64, two, one, f16, 2) : launch(c64, integral_constant<int, 4>(), one, f16, 1);
  };
  const bool ok = f16out ? form(std::true_type()) : form(std::false_type());
  if (!ok) return SQ_ERR_CUDA;
  count_launch();
  return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ERR_CUDA;
}

}  // namespace sq
