// Steps 1+2 on warp-level tensor instructions: factor pairs with n2 = 32 (n1 <= 128), any number of rows.
//
// The tcgen05 kernels want n2 = 64 or 128; the narrow layers of small models (512, 1024, 2048 channels) went through the
// fp32 kernel, which is bound by its multiply-adds.  Here a warp carries 16 columns q' of a token through both stages:
//
//   stage 1  T^T[q'][p]  = sum_q R2^T[q'][q] X^T[q][p]    A = R2^T (shared memory, fp16 hi + lo), B = X^T: the token's
//                                                         rows as they lie in memory, 16 bytes per lane, exact fp16
//   stage 2  Z^T[q'][p'] = sum_p T^T[q'][p] R1[p][p']     A = T^T: the accumulators of stage 1 are in the layout of
//                                                         this operand (fp16 hi + lo, one power-of-two scale),
//                                                         B = R1 (shared memory, fp16 hi + lo)
// with the split, the passes (hi*hi + lo*hi + hi*lo) and the 2^10 pre-scale of the factors as in the tcgen05 kernel: the
// result keeps fp32 accuracy.  For n1 > 64 the p axis is cut over two warps: each makes its part of T and of Z, and the
// fp16 operand of stage 2 goes through shared memory once.  A CTA (two or four warps) owns a token at a time; its warps
// meet for the absmax.
//
// Operand order.  k-slots may stand for any channel as long as A and B agree: lane (g, c) loads q = 8 c .. 8 c + 7 of row
// p = 8 t + g, and the eight halves are the b registers of both k-steps; the image of R2^T is stored in that order.  Rows
// g and g + 8 of the m16 tile stand for q' = 2 g and 2 g + 1, so that a thread holds the two codes of a byte; three
// shuffles turn eight lanes' bytes into eight-byte pieces of the packed row.
//
// Bound by latency at these sizes (one token is 0.1 to 0.3 us of products).  Measured against the fp32 kernel, back-to-back
// launches: 64 x 512 (16 x 32) 4.8 -> 1.7 us, 1024 x 2048 (64 x 32) 20.6 -> 5.9 us, 2048 x 4096 (128 x 32) 113 -> 26 us;
// fp16 rows out 64 x 512 7.2 -> 1.5 us.
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "sq_internal.h"
#include "sq_ptx.cuh"

namespace sq {
namespace {

enum RmSite : uint32_t { RM_B1 = 112 };

__device__ __forceinline__ void mma_f16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Token bytes the kernel before this one may just have written: past the L1 cache.
__device__ __forceinline__ uint4 ld_token16(const void* p) { return __ldcg(static_cast<const uint4*>(p)); }

// Eight lanes (g = lane / 4, same lane % 4) each hold eight bytes, byte i meant for lane g = i: lane g gets the
// eight bytes meant for it, in the order of their source lanes.  Three exchanges, halving what travels together.
__device__ __forceinline__ uint2 transpose_bytes_8(uint32_t w0, uint32_t w1, int g) {
  const bool h2 = g & 4, h1 = g & 2, h0 = g & 1;
  uint32_t keep = h2 ? w1 : w0, recv = __shfl_xor_sync(0xFFFFFFFFu, h2 ? w0 : w1, 16);
  const uint32_t p = h2 ? recv : keep, q = h2 ? keep : recv;               // from source lanes with bit 2 clear, set
  keep = __byte_perm(p, q, h1 ? 0x7632 : 0x5410);
  recv = __shfl_xor_sync(0xFFFFFFFFu, __byte_perm(p, q, h1 ? 0x5410 : 0x7632), 8);
  uint32_t s0 = h1 ? recv : keep, s1 = h1 ? keep : recv;                   // from source bit 1 clear, set
  const uint32_t pp = __byte_perm(s0, s1, 0x5410), qq = __byte_perm(s0, s1, 0x7632);
  keep = __byte_perm(pp, qq, h0 ? 0x7531 : 0x6420);
  recv = __shfl_xor_sync(0xFFFFFFFFu, __byte_perm(pp, qq, h0 ? 0x6420 : 0x7531), 4);
  s0 = h0 ? recv : keep;
  s1 = h0 ? keep : recv;
  return make_uint2(__byte_perm(s0, s1, 0x5140), __byte_perm(s0, s1, 0x7362));
}

// Tiles of eight p per warp (NT) and warps per q' slice (PW) for n1; the padded n1 is 8 * NT * PW.
struct RmShape { int NT, PW; };
inline RmShape rm_shape(int n1) {
  if (n1 <= 16) return {2, 1};
  if (n1 <= 32) return {4, 1};
  if (n1 <= 48) return {6, 1};
  if (n1 <= 64) return {8, 1};
  if (n1 <= 80) return {5, 2};
  if (n1 <= 96) return {6, 2};
  if (n1 <= 112) return {7, 2};
  return {8, 2};
}

constexpr int RM_N2 = 32, RM_SLICES = RM_N2 / 16;      // q' slices of a token, PW warps each

// Shared memory: [R1 operand][R2^T operand][T operand, PW > 1: slice x (hi, lo) x k-step x half x lane x 8 B][maxima, barrier].
constexpr int RM_A2_SLICE = RM_N2 / 16 * 1024;
constexpr int rm_smem(int NT, int PW) {
  const int ntt = NT * PW;
  return ntt / 2 * ntt * 512 + RM_SLICES * RM_A2_SLICE + (PW > 1 ? RM_SLICES * 2 * (ntt / 2) * 512 : 0) + 128;
}

// Tokens cta, cta + ncta, ... of `rows`: how many there are.  Unsigned, since rows goes up to 2^31 - 1 and the token behind
// the last one may lie beyond that.
__host__ __device__ inline int rm_tokens(int cta, int ncta, int rows) {
  return rows > cta ? static_cast<int>((static_cast<unsigned>(rows - cta) + static_cast<unsigned>(ncta - 1)) / static_cast<unsigned>(ncta)) : 0;
}

template <int NT, int PW>
__global__ void __launch_bounds__(RM_SLICES * PW * 32, 3)
rotate_quant_mma_kernel(const uint4* __restrict__ a2_img, const uint4* __restrict__ b1_img, int n1, int rows,
                        const __half* __restrict__ X, uint8_t* __restrict__ Xq, __half* __restrict__ scales,
                        float* __restrict__ Zdbg, bool f16out) {
  constexpr int N2 = RM_N2, WARPS = RM_SLICES * PW;
  constexpr int NTT = NT * PW, KJ = NTT / 2;           // p tiles, k-steps of stage 2
  static_assert(NTT % 2 == 0, "whole k-steps");
  constexpr int B1_BYTES = KJ * NTT * 512, A2_BYTES = RM_SLICES * RM_A2_SLICE;
  constexpr int T_BYTES = PW > 1 ? RM_SLICES * 2 * KJ * 512 : 0;
  extern __shared__ __align__(128) unsigned char rm_smem_raw[];
  uint4* b1s = reinterpret_cast<uint4*>(rm_smem_raw);
  unsigned char* a2s = rm_smem_raw + B1_BYTES;
  uint2* ts = reinterpret_cast<uint2*>(a2s + A2_BYTES);                    // [slice][hi, lo][k-step][half][lane]
  float* zmax = reinterpret_cast<float*>(a2s + A2_BYTES + T_BYTES);        // [2][WARPS]: of the token
  float* tmax = zmax + 16;                                                 // [WARPS]: of T (PW > 1)
  uint64_t* bar = reinterpret_cast<uint64_t*>(zmax + 28);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int m = warp / PW, part = warp % PW;           // q' slice, part of the p axis
  const int n = n1 * N2;
  const uint32_t limit = wait_limit();

  // The factors belong to the handle: fetched while the kernel before this one still runs.
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    mbar_fence_init();
    mbar_arrive_expect_tx(bar, B1_BYTES + A2_BYTES);
    bulk_load_1d(a2s, a2_img, A2_BYTES, bar);
    for (int o = 0; o < B1_BYTES; o += 16384)
      bulk_load_1d(rm_smem_raw + o, reinterpret_cast<const unsigned char*>(b1_img) + o,
                   static_cast<uint32_t>(B1_BYTES - o < 16384 ? B1_BYTES - o : 16384), bar);
  }
  griddep_wait();
  griddep_launch_dependents();                         // not earlier: see the tcgen05 kernel
  __syncthreads();                                     // the barrier exists
  uint4 x[NT];
  auto load_x = [&](long long token) {
    const __half* xt = X + token * n + c * 8;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int p = (part * NT + t) * 8 + g;
      x[t] = p < n1 ? ld_token16(xt + p * N2) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  const uint4* a2 = reinterpret_cast<const uint4*>(a2s + m * RM_A2_SLICE) + lane;
  int par = 0;
  load_x(blockIdx.x);
  const bool ok = mbar_wait(bar, 0, RM_B1, limit);
  long long token = blockIdx.x;
  for (int left = rm_tokens(blockIdx.x, gridDim.x, rows); left > 0; --left, token += gridDim.x, par ^= 1) {
    // ---- stage 1 ------------------------------------------------------------------------------------------
    float T[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) T[t][e] = 0.0f;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const uint4 h4 = a2[(s * 2 + 0) * 32], l4 = a2[(s * 2 + 1) * 32];
      const uint32_t h[4] = {h4.x, h4.y, h4.z, h4.w}, l[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
      for (int t = 0; t < NT; ++t) mma_f16_16816(T[t], h, s ? x[t].z : x[t].x, s ? x[t].w : x[t].y);
#pragma unroll
      for (int t = 0; t < NT; ++t) mma_f16_16816(T[t], l, s ? x[t].z : x[t].x, s ? x[t].w : x[t].y);
    }
    if (left > 1) load_x(token + gridDim.x);      // the next token's rows
    // ---- T -> fp16 hi + lo, scaled so that the slice's largest entry lands in [2^13, 2^14) ----------------------
    float tm = 0.0f;
#pragma unroll
    for (int t = 0; t < NT; ++t)
      tm = fmaxf(tm, fmaxf(fmaxf(fabsf(T[t][0]), fabsf(T[t][1])), fmaxf(fabsf(T[t][2]), fabsf(T[t][3]))));
    tm = warp_max(tm);
    if constexpr (PW > 1) {
      if (lane == 0) tmax[warp] = tm;
      named_barrier(1 + m, PW * 32);
#pragma unroll
      for (int w = 0; w < PW; ++w) tm = fmaxf(tm, tmax[m * PW + w]);
    }
    int k = 13 - (static_cast<int>((__float_as_uint(tm) >> 23) & 0xFF) - 127);
    if (tm == 0.0f) k = 0;
    k = max(-126, min(127, k));
    const float sc = __uint_as_float(static_cast<uint32_t>(k + 127) << 23);
    const int uexp = -(k + 2 * kFactorScaleLog2) + 127;        // z = result * 2^-(k + 20), exactly
    const float un = (uexp >= 1) ? __uint_as_float(static_cast<uint32_t>(min(uexp, 254)) << 23) : 0.0f;
    uint32_t th[NT][2], tl[NT][2];
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float v0 = T[t][2 * r], v1 = T[t][2 * r + 1];
        const __half2 hh = __floats2half2_rn(v0 * sc, v1 * sc);
        const float2 hf = __half22float2(hh);
        th[t][r] = *reinterpret_cast<const uint32_t*>(&hh);
        tl[t][r] = pack_half2(fmaf(v0, sc, -hf.x), fmaf(v1, sc, -hf.y));
      }
    if constexpr (PW > 1) {
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const int tg = part * NT + t;                  // k-step tg / 2, half tg % 2 of it
        ts[((m * 2 + 0) * KJ * 2 + tg) * 32 + lane] = make_uint2(th[t][0], th[t][1]);
        ts[((m * 2 + 1) * KJ * 2 + tg) * 32 + lane] = make_uint2(tl[t][0], tl[t][1]);
      }
      named_barrier(1 + m, PW * 32);
    }
    // ---- stage 2 ------------------------------------------------------------------------------------------
    float z[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) z[t][e] = 0.0f;
    const uint4* bj = b1s + part * NT * 32 + lane;
#pragma unroll(PW > 1 ? 1 : KJ)
    for (int j = 0; j < KJ; ++j) {
      uint32_t h[4], l[4];
      if constexpr (PW > 1) {
        const uint2 h01 = ts[((m * 2 + 0) * KJ * 2 + 2 * j) * 32 + lane], h23 = ts[((m * 2 + 0) * KJ * 2 + 2 * j + 1) * 32 + lane];
        const uint2 l01 = ts[((m * 2 + 1) * KJ * 2 + 2 * j) * 32 + lane], l23 = ts[((m * 2 + 1) * KJ * 2 + 2 * j + 1) * 32 + lane];
        h[0] = h01.x; h[1] = h01.y; h[2] = h23.x; h[3] = h23.y;
        l[0] = l01.x; l[1] = l01.y; l[2] = l23.x; l[3] = l23.y;
      } else {
        h[0] = th[2 * j][0]; h[1] = th[2 * j][1]; h[2] = th[2 * j + 1][0]; h[3] = th[2 * j + 1][1];
        l[0] = tl[2 * j][0]; l[1] = tl[2 * j][1]; l[2] = tl[2 * j + 1][0]; l[3] = tl[2 * j + 1][1];
      }
      uint4 b[NT];
#pragma unroll
      for (int t = 0; t < NT; ++t) b[t] = bj[(j * NTT + t) * 32];
#pragma unroll
      for (int t = 0; t < NT; ++t) mma_f16_16816(z[t], h, b[t].x, b[t].y);      // hi * hi
#pragma unroll
      for (int t = 0; t < NT; ++t) mma_f16_16816(z[t], l, b[t].x, b[t].y);      // lo * hi
#pragma unroll
      for (int t = 0; t < NT; ++t) mma_f16_16816(z[t], h, b[t].z, b[t].w);      // hi * lo
    }
    // z[t][e], z[t][2 + e]: channels q' = 16 m + 2 g, + 1 of row p' = 8 (part NT + t) + 2 c + e.
    if (f16out) {                                      // rotation only: fp16 rows out
      __half* zrow = reinterpret_cast<__half*>(Xq) + token * n + m * 16 + 2 * g;
#pragma unroll
      for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int p = (part * NT + t) * 8 + 2 * c + e;
          if (p < n1 && ok) *reinterpret_cast<uint32_t*>(zrow + p * N2) = pack_half2(z[t][e] * un, z[t][2 + e] * un);
        }
      if constexpr (PW > 1) __syncthreads();           // the T operand has been read
      continue;
    }
    float zm = 0.0f;
#pragma unroll
    for (int t = 0; t < NT; ++t)
      zm = fmaxf(zm, fmaxf(fmaxf(fabsf(z[t][0]), fabsf(z[t][1])), fmaxf(fabsf(z[t][2]), fabsf(z[t][3]))));
    zm = warp_max(zm * un);                            // padding rows hold exact zeros
    float* zp = zmax + par * WARPS;                    // two sets in turn: one barrier per token is enough
    if (lane == 0) zp[warp] = zm;
    __syncthreads();
    float amax = zp[0];
#pragma unroll
    for (int w = 1; w < WARPS; ++w) amax = fmaxf(amax, zp[w]);
    __half delta;
    float inv;
    row_scale(amax, delta, inv);
    const float inv_un = inv * un;                     // exact: un is a power of two
    // Delta >= 2^-14 (a normal fp16) bounds |z / Delta| by 7 (1 + 2^-11): no clamp is needed then.
    const bool clamp = __half2float(delta) < 6.103515625e-05f;
    uint8_t* orow = Xq + token * (n / 2) + m * 8;
#pragma unroll
    for (int gr = 0; gr < (NT + 3) / 4; ++gr) {
      uint32_t w[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float tt[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int t = 4 * gr + 2 * h + (i >> 1), e = i & 1;
#pragma unroll
          for (int o = 0; o < 2; ++o) {
            float v = t < NT ? __fadd_rn(__fmul_rn(z[t < NT ? t : 0][2 * o + e], inv_un), 0.5f) : 0.0f;
            if (clamp) v = fminf(fmaxf(v, -8.0f), 7.5f);
            tt[2 * i + o] = v;
          }
        }
        w[h] = pack8_codes(tt);
      }
      const uint2 out = transpose_bytes_8(w[0], w[1], g);
      const int t = 4 * gr + (g >> 1), p = (part * NT + t) * 8 + 2 * c + (g & 1);
      if (t < NT && p < n1 && ok) *reinterpret_cast<uint2*>(orow + p * (N2 / 2)) = out;
    }
    if (Zdbg != nullptr) {
      float* zrow = Zdbg + token * n + m * 16 + 2 * g;
#pragma unroll
      for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int p = (part * NT + t) * 8 + 2 * c + e;
          if (p < n1) *reinterpret_cast<float2*>(zrow + p * N2) = make_float2(z[t][e] * un, z[t][2 + e] * un);
        }
    }
    if (threadIdx.x == 0 && ok) scales[token] = delta;
  }
}

template <int NT, int PW>
sq_status_t launch_rm(const sq_rotation* h, const void* X, int64_t rows, void* Xq, void* scales, float* Zdbg, bool f16out,
                      cudaStream_t s) {
  const int sms = sm_count();
  if (sms <= 0) return SQ_ERR_CUDA;
  auto kern = rotate_quant_mma_kernel<NT, PW>;
  constexpr int smem = rm_smem(NT, PW);
  if (!ensure_dyn_smem(reinterpret_cast<const void*>(kern), smem)) return SQ_ERR_CUDA;
  // Tokens in equal runs over the CTAs that are resident at once.
  const long long cap = static_cast<long long>(sms) * std::min(PW == 2 ? 3 : (NT <= 4 ? 8 : 5), 220 * 1024 / (smem + 1024));
  const long long per = (rows + cap - 1) / cap;
  const uint4* b1 = static_cast<const uint4*>(h->dMmaImg);
  const uint4* a2 = b1 + static_cast<size_t>(NT * PW / 2) * (NT * PW) * 32;
  const cudaError_t err = launch_dependent(kern, dim3(static_cast<unsigned>((rows + per - 1) / per)), dim3(RM_SLICES * PW * 32),
                                           static_cast<size_t>(smem), s, a2, b1, static_cast<int>(h->n1), static_cast<int>(rows),
                                           static_cast<const __half*>(X), static_cast<uint8_t*>(Xq),
                                           static_cast<__half*>(scales), Zdbg, f16out);
  count_launch();
  return err == cudaSuccess ? SQ_OK : SQ_ERR_CUDA;
}

}  // namespace

bool rotate_quant_mma_supported(int n1, int n2) { return n1 >= 1 && n1 <= 128 && n2 == RM_N2; }

// Uploads the two operand images in fragment order: R1 as [k-step][tile][lane] {b0 hi, b1 hi, b0 lo, b1 lo}, then R2^T as
// [q' slice][k-step][hi, lo][lane] {a0 .. a3}.
bool rotate_quant_mma_prepare(sq_rotation* h) {
  const int n1 = h->n1, n2 = h->n2;
  const RmShape sh = rm_shape(n1);
  const int ntt = sh.NT * sh.PW, kj = ntt / 2;
  const size_t b1_words = static_cast<size_t>(kj) * ntt * 128, a2_words = static_cast<size_t>(n2 / 16) * (n2 / 16) * 256;
  std::vector<uint32_t> img(b1_words + a2_words, 0u);
  auto split_word = [](float v0, float v1, uint32_t& hi, uint32_t& lo) {
    __half h0, l0, h1, l1;
    split_half(v0, h0, l0);
    split_half(v1, h1, l1);
    hi = __half_as_ushort(h0) | static_cast<uint32_t>(__half_as_ushort(h1)) << 16;
    lo = __half_as_ushort(l0) | static_cast<uint32_t>(__half_as_ushort(l1)) << 16;
  };
  auto r1 = [&](int p, int pp) { return p < n1 && pp < n1 ? kFactorScale * h->R1[static_cast<size_t>(p) * n1 + pp] : 0.0f; };
  auto r2 = [&](int q, int qp) { return kFactorScale * h->R2[static_cast<size_t>(q) * n2 + qp]; };
  for (int j = 0; j < kj; ++j)
    for (int t = 0; t < ntt; ++t)
      for (int lane = 0; lane < 32; ++lane) {
        const int g = lane >> 2, c = lane & 3;
        uint32_t* w = img.data() + (static_cast<size_t>(j * ntt + t) * 32 + lane) * 4;
        for (int r = 0; r < 2; ++r)
          split_word(r1(16 * j + 8 * r + 2 * c, 8 * t + g), r1(16 * j + 8 * r + 2 * c + 1, 8 * t + g), w[r], w[2 + r]);
      }
  for (int m = 0; m < n2 / 16; ++m)
    for (int s = 0; s < n2 / 16; ++s)
      for (int lane = 0; lane < 32; ++lane) {
        const int g = lane >> 2, c = lane & 3;
        uint32_t* w = img.data() + b1_words + (static_cast<size_t>((m * (n2 / 16) + s) * 2) * 32 + lane) * 4;
        for (int r = 0; r < 4; ++r) {
          const int q = 32 * (s >> 1) + 8 * c + 4 * (s & 1) + 2 * (r >> 1), qp = 16 * m + 2 * g + (r & 1);
          split_word(r2(q, qp), r2(q + 1, qp), w[r], w[128 + r]);
        }
      }
  if (cudaMalloc(&h->dMmaImg, img.size() * 4) != cudaSuccess ||
      cudaMemcpy(h->dMmaImg, img.data(), img.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

sq_status_t launch_rotate_quant_mma(const sq_rotation* h, const void* X, int64_t rows, void* Xq, void* scales, float* Zdbg,
                                    cudaStream_t s, bool f16out) {
  if (rows > 0x7FFFFFFF) return SQ_ERR_UNSUPPORTED;
  const RmShape sh = rm_shape(h->n1);
  if (sh.PW == 1) {
    if (sh.NT == 2) return launch_rm<2, 1>(h, X, rows, Xq, scales, Zdbg, f16out, s);
    if (sh.NT == 4) return launch_rm<4, 1>(h, X, rows, Xq, scales, Zdbg, f16out, s);
    if (sh.NT == 6) return launch_rm<6, 1>(h, X, rows, Xq, scales, Zdbg, f16out, s);
    return launch_rm<8, 1>(h, X, rows, Xq, scales, Zdbg, f16out, s);
  }
  if (sh.NT == 5) return launch_rm<5, 2>(h, X, rows, Xq, scales, Zdbg, f16out, s);
  if (sh.NT == 6) return launch_rm<6, 2>(h, X, rows, Xq, scales, Zdbg, f16out, s);
  if (sh.NT == 7) return launch_rm<7, 2>(h, X, rows, Xq, scales, Zdbg, f16out, s);
  return launch_rm<8, 2>(h, X, rows, Xq, scales, Zdbg, f16out, s);
}

}  // namespace sq
