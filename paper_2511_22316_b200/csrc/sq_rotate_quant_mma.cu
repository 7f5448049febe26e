// Steps 1+2 on warp-level tensor instructions in float64: factor pairs with n2 = 32 (n1 <= 128), any number of rows.
//
// The tcgen05 kernels want n2 = 64 or 128; the narrow layers of small models (512, 1024, 2048 channels) went through the
// fp32 kernel, which is bound by its multiply-adds.  Here a warp carries 16 columns q' of a token through both stages:
//
//   stage 1  T^T[q'][p]  = sum_q R2^T[q'][q] X^T[q][p]    A = R2^T (shared memory), B = X^T: the token's rows as they lie
//                                                         in memory, 16 bytes per lane
//   stage 2  Z^T[q'][p'] = sum_p T^T[q'][p] R1[p][p']     A = T^T: the accumulators of stage 1 as they are (through
//                                                         shared memory), B = R1 (shared memory, as fp32)
// Both are mma.sync m16n8k16 in float64, rounded once to fp32 at the end.  The unit runs at half the fp32 rate, which these
// sizes do not feel, and it takes any fp32 factor and passes infinities and NaN on as the fp32 kernel does.  Operands split
// into two fp16 numbers (the tcgen05 kernels' way) were faster on many rows, 2048 x 4096 in 26 us, but two to three times as
// far from float64 as the fp32 kernel, NaN for factors beyond 64, and finite codes for tokens with infinities.
// The p axis is cut over two or four warps: each makes its part of T and of Z, and the operand of stage 2 goes through
// shared memory once.  A CTA (four or eight warps) owns a token at a time; its warps meet for the absmax.
//
// Operand order.  k-slots may stand for any channel as long as A and B agree: lane (g, c) loads q = 8 c .. 8 c + 7 of row
// p = 8 t + g, and the eight halves are the b registers of both k-steps; the image of R2^T is stored in that order.  Rows
// g and g + 8 of the m16 tile stand for q' = 2 g and 2 g + 1, so that a thread holds the two codes of a byte; three
// shuffles turn eight lanes' bytes into eight-byte pieces of the packed row.
//
// Few rows are bound by the latency of a token's products, many by the float64 unit: 8192 x 4096 (128 x 32) runs it at
// 16.2 TFMA/s, 87 % of its 64 per cycle and SM.  Measured against the fp32 kernel, back-to-back launches: 64 x 512
// (16 x 32) 5.0 -> 1.9 us, 300 x 2048 (64 x 32) 11.3 -> 7.0 us, 2048 x 4096 (128 x 32) 111 -> 84 us; fp16 rows out 64 x 512
// 7.4 -> 1.7 us.  Distance of z from float64: 2.5e-8 of it (the one rounding), the fp32 kernel's 1.0e-7 to 2.6e-7.
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "sq_internal.h"
#include "sq_ptx.cuh"

namespace sq {
namespace {

enum RmSite : uint32_t { RM_B1 = 112 };

// Fragments: a[2 i], a[2 i + 1] rows g and g + 8 of k = c + 4 i; b[i] column g of k = c + 4 i; d rows g, g + 8 (d[2], d[3]),
// columns 2 c, 2 c + 1.
__device__ __forceinline__ void mma_f64_16816(double (&d)[4], const double (&a)[8], const double (&b)[4]) {
  asm("mma.sync.aligned.m16n8k16.row.col.f64.f64.f64.f64 {%0, %1, %2, %3}, {%4, %5, %6, %7, %8, %9, %10, %11}, "
      "{%12, %13, %14, %15}, {%0, %1, %2, %3};"
      : "+d"(d[0]), "+d"(d[1]), "+d"(d[2]), "+d"(d[3])
      : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(a[4]), "d"(a[5]), "d"(a[6]), "d"(a[7]), "d"(b[0]), "d"(b[1]), "d"(b[2]),
        "d"(b[3]));
}
__device__ __forceinline__ void halves_to_f64(uint32_t w0, uint32_t w1, double (&b)[4]) {
  const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&w0)), f1 = __half22float2(*reinterpret_cast<const __half2*>(&w1));
  b[0] = f0.x; b[1] = f0.y; b[2] = f1.x; b[3] = f1.y;
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

// Tiles of eight p per warp (NT) and warps per q' slice (PW) for n1; the padded n1 is 8 * NT * PW.  Few tiles per warp and
// more warps, as far as the padding stays small: with few rows a token's chain of products is all there is (one token of
// 64 x 32: 5.8 us with eight tiles and one warp, 3.4 with two and four).
struct RmShape { int NT, PW; };
inline RmShape rm_shape(int n1) {
  if (n1 <= 16) return {1, 2};
  if (n1 <= 32) return {2, 2};
  if (n1 <= 48) return {3, 2};
  if (n1 <= 64) return {2, 4};
  if (n1 <= 80) return {5, 2};
  if (n1 <= 96) return {3, 4};
  if (n1 <= 112) return {7, 2};
  return {4, 4};
}
// Blocks that share an SM: what the registers allow, or fewer where that measured faster.
constexpr int rm_ctas(int NT, int PW) { return PW == 4 ? (NT == 4 ? 2 : 3) : (NT == 1 ? 8 : (NT <= 3 ? 4 : 3)); }

constexpr int RM_N2 = 32, RM_SLICES = RM_N2 / 16;      // q' slices of a token, PW warps each

// Shared memory: [R1 operand, fp32][R2^T operand][T operand: slice x tile x half x lane x 16 B][maxima, barrier].
constexpr int RM_A2_SLICE = RM_N2 * 32 / 4 * 16;
constexpr int rm_smem(int NT, int PW) {
  const int ntt = NT * PW;
  return ntt / 2 * ntt * 512 + RM_SLICES * RM_A2_SLICE + RM_SLICES * ntt * 1024 + 128;
}

// Tokens cta, cta + ncta, ... of `rows`: how many there are.  Unsigned, since rows goes up to 2^31 - 1 and the token behind
// the last one may lie beyond that.
__host__ __device__ inline int rm_tokens(int cta, int ncta, int rows) {
  return rows > cta ? static_cast<int>((static_cast<unsigned>(rows - cta) + static_cast<unsigned>(ncta - 1)) / static_cast<unsigned>(ncta)) : 0;
}

template <int NT, int PW>
__global__ void __launch_bounds__(RM_SLICES * PW * 32, rm_ctas(NT, PW))
rotate_quant_mma_kernel(const double2* __restrict__ a2_img, const float4* __restrict__ b1_img, int n1, int rows,
                        const __half* __restrict__ X, uint8_t* __restrict__ Xq, __half* __restrict__ scales,
                        float* __restrict__ Zdbg, bool f16out) {
  constexpr int N2 = RM_N2, WARPS = RM_SLICES * PW;
  constexpr int NTT = NT * PW, KJ = NTT / 2;           // p tiles, k-steps of stage 2
  static_assert(NTT % 2 == 0, "whole k-steps");
  constexpr int B1_BYTES = KJ * NTT * 512, A2_BYTES = RM_SLICES * RM_A2_SLICE;
  constexpr int T_BYTES = RM_SLICES * NTT * 1024;
  extern __shared__ __align__(128) unsigned char rm_smem_raw[];
  const float4* b1s = reinterpret_cast<const float4*>(rm_smem_raw);
  unsigned char* a2s = rm_smem_raw + B1_BYTES;
  double2* ts = reinterpret_cast<double2*>(a2s + A2_BYTES);                // [slice][tile][even, odd p][lane]
  float* zmax = reinterpret_cast<float*>(a2s + A2_BYTES + T_BYTES);        // [2][WARPS]: of the token
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
  const double2* a2 = reinterpret_cast<const double2*>(a2s + m * RM_A2_SLICE) + lane;
  int par = 0;
  load_x(blockIdx.x);
  const bool ok = mbar_wait(bar, 0, RM_B1, limit);
  long long token = blockIdx.x;
  for (int left = rm_tokens(blockIdx.x, gridDim.x, rows); left > 0; --left, token += gridDim.x, par ^= 1) {
    // ---- stage 1 ------------------------------------------------------------------------------------------
    double T[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) T[t][e] = 0.0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      double a[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const double2 v = a2[(4 * s + i) * 32];
        a[2 * i] = v.x;
        a[2 * i + 1] = v.y;
      }
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        double b[4];
        halves_to_f64(s ? x[t].z : x[t].x, s ? x[t].w : x[t].y, b);
        mma_f64_16816(T[t], a, b);
      }
    }
    if (left > 1) load_x(token + gridDim.x);      // the next token's rows
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      double2* o = ts + ((m * NTT + part * NT + t) * 2) * 32 + lane;
      o[0] = make_double2(T[t][0], T[t][2]);
      o[32] = make_double2(T[t][1], T[t][3]);
    }
    named_barrier(1 + m, PW * 32);
    // ---- stage 2 ------------------------------------------------------------------------------------------
    double zd[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) zd[t][e] = 0.0;
    const float4* bj = b1s + part * NT * 32 + lane;
#pragma unroll(KJ > 4 ? 1 : KJ)
    for (int j = 0; j < KJ; ++j) {
      double a[8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {                    // tile 2 j + h: even rows p, odd rows p
        const double2* o = ts + ((m * NTT + 2 * j + h) * 2) * 32 + lane;
        const double2 v0 = o[0], v1 = o[32];
        a[4 * h + 0] = v0.x; a[4 * h + 1] = v0.y; a[4 * h + 2] = v1.x; a[4 * h + 3] = v1.y;
      }
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const float4 v = bj[(j * NTT + t) * 32];
        const double b[4] = {v.x, v.y, v.z, v.w};
        mma_f64_16816(zd[t], a, b);
      }
    }
    float z[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) z[t][e] = static_cast<float>(zd[t][e]);
    // z[t][e], z[t][2 + e]: channels q' = 16 m + 2 g, + 1 of row p' = 8 (part NT + t) + 2 c + e.
    if (f16out) {                                      // rotation only: fp16 rows out
      __half* zrow = reinterpret_cast<__half*>(Xq) + token * n + m * 16 + 2 * g;
#pragma unroll
      for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int p = (part * NT + t) * 8 + 2 * c + e;
          if (p < n1 && ok) *reinterpret_cast<uint32_t*>(zrow + p * N2) = pack_half2(z[t][e], z[t][2 + e]);
        }
      __syncthreads();                                 // the T operand has been read
      continue;
    }
    float zm = 0.0f;
#pragma unroll
    for (int t = 0; t < NT; ++t)
      zm = fmaxf(zm, fmaxf(fmaxf(fabsf(z[t][0]), fabsf(z[t][1])), fmaxf(fabsf(z[t][2]), fabsf(z[t][3]))));
    zm = warp_max(zm);                                 // padding rows hold zeros, or NaN, which a maximum passes over
    float* zp = zmax + par * WARPS;                    // two sets in turn: one barrier per token is enough
    if (lane == 0) zp[warp] = zm;
    __syncthreads();
    float amax = zp[0];
#pragma unroll
    for (int w = 1; w < WARPS; ++w) amax = fmaxf(amax, zp[w]);
    __half delta;
    float inv;
    row_scale(amax, delta, inv);
    // A finite Delta >= 2^-14 (a normal fp16) bounds |z / Delta| by 7 (1 + 2^-11): no clamp is needed then.  A token with an
    // infinity has an infinite Delta, one with a NaN has 0; its codes are 0.
    const bool clamp = !(__half2float(delta) >= 6.103515625e-05f && __half2float(delta) <= 65504.0f);
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
            float v = t < NT ? __fadd_rn(__fmul_rn(z[t < NT ? t : 0][2 * o + e], inv), 0.5f) : 0.0f;
            if (clamp) v = v == v ? fminf(fmaxf(v, -8.0f), 7.5f) : 0.5f;
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
          if (p < n1) *reinterpret_cast<float2*>(zrow + p * N2) = make_float2(z[t][e], z[t][2 + e]);
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
  const int resident = std::min(rm_ctas(NT, PW), 220 * 1024 / (smem + 1024));
  const long long grid = std::min<long long>(rows, static_cast<long long>(sms) * resident);
  const float4* b1 = static_cast<const float4*>(h->dMmaImg);
  const double2* a2 = reinterpret_cast<const double2*>(b1 + static_cast<size_t>(NT * PW / 2) * (NT * PW) * 32);
  const cudaError_t err = launch_dependent(kern, dim3(static_cast<unsigned>(grid)), dim3(RM_SLICES * PW * 32),
                                           static_cast<size_t>(smem), s, a2, b1, static_cast<int>(h->n1), static_cast<int>(rows),
                                           static_cast<const __half*>(X), static_cast<uint8_t*>(Xq),
                                           static_cast<__half*>(scales), Zdbg, f16out);
  count_launch();
  return err == cudaSuccess ? SQ_OK : SQ_ERR_CUDA;
}

}  // namespace

bool rotate_quant_mma_supported(int n1, int n2) { return n1 >= 1 && n1 <= 128 && n2 == RM_N2; }

// Uploads the two operand images in fragment order: R1 in fp32 as [k-step][tile][lane] {b0 .. b3}, then R2^T in float64 as
// [q' slice][k-slot of a lane][lane] {rows g, g + 8}.
bool rotate_quant_mma_prepare(sq_rotation* h) {
  const int n1 = h->n1, n2 = h->n2;
  const RmShape sh = rm_shape(n1);
  const int ntt = sh.NT * sh.PW, kj = ntt / 2;
  const size_t b1_bytes = static_cast<size_t>(kj) * ntt * 512;
  std::vector<unsigned char> img(b1_bytes + static_cast<size_t>(RM_SLICES) * RM_A2_SLICE, 0);
  float* b1 = reinterpret_cast<float*>(img.data());
  double* a2 = reinterpret_cast<double*>(img.data() + b1_bytes);
  for (int j = 0; j < kj; ++j)
    for (int t = 0; t < ntt; ++t)
      for (int lane = 0; lane < 32; ++lane)
        for (int i = 0; i < 4; ++i) {
          const int p = 16 * j + 8 * (i >> 1) + 2 * (lane & 3) + (i & 1), pp = 8 * t + (lane >> 2);
          if (p < n1 && pp < n1) b1[(static_cast<size_t>(j * ntt + t) * 32 + lane) * 4 + i] = h->R1[static_cast<size_t>(p) * n1 + pp];
        }
  for (int m = 0; m < RM_SLICES; ++m)
    for (int k = 0; k < 8; ++k)
      for (int lane = 0; lane < 32; ++lane)
        for (int r = 0; r < 2; ++r)
          a2[((m * 8 + k) * 32 + lane) * 2 + r] = h->R2[static_cast<size_t>(8 * (lane & 3) + k) * n2 + 16 * m + 2 * (lane >> 2) + r];
  if (cudaMalloc(&h->dMmaImg, img.size()) != cudaSuccess ||
      cudaMemcpy(h->dMmaImg, img.data(), img.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

sq_status_t launch_rotate_quant_mma(const sq_rotation* h, const void* X, int64_t rows, void* Xq, void* scales, float* Zdbg,
                                    cudaStream_t s, bool f16out) {
  if (rows > 0x7FFFFFFF) return SQ_ERR_UNSUPPORTED;
  const RmShape sh = rm_shape(h->n1);
  if (sh.PW == 4) {
    if (sh.NT == 2) return launch_rm<2, 4>(h, X, rows, Xq, scales, Zdbg, f16out, s);
    if (sh.NT == 3) return launch_rm<3, 4>(h, X, rows, Xq, scales, Zdbg, f16out, s);
    return launch_rm<4, 4>(h, X, rows, Xq, scales, Zdbg, f16out, s);
  }
  if (sh.NT == 1) return launch_rm<1, 2>(h, X, rows, Xq, scales, Zdbg, f16out, s);
  if (sh.NT == 2) return launch_rm<2, 2>(h, X, rows, Xq, scales, Zdbg, f16out, s);
  if (sh.NT == 3) return launch_rm<3, 2>(h, X, rows, Xq, scales, Zdbg, f16out, s);
  if (sh.NT == 5) return launch_rm<5, 2>(h, X, rows, Xq, scales, Zdbg, f16out, s);
  return launch_rm<7, 2>(h, X, rows, Xq, scales, Zdbg, f16out, s);
}

}  // namespace sq
