// Online activation decomposition kernels.
//   INT8  (Sec. 3.2, Eqs. alpha..x2; Alg. 1 lines 1-5): one CTA per row, 128-bit BF16 loads, row maximum by warp
//          shuffles, the rounded IEEE quotients without a division per value (quant.cuh), 8 codes per store.
//   MXFP4 (Sec. 3.2.1, Alg. 2, on the E2M1 grid): one thread per 32-element block - the block maximum needs
//          no cross-thread reduction and beta follows from alpha by a shift.
#include <cuda_bf16.h>
#include <cuda_fp4.h>

#include <cstdlib>

#include "host_common.h"
#include "quant.cuh"
#include "sm100.cuh"

namespace msd {

// Bound by issue slots and latency (4096 rows of 4096, 67 MB: 27 us with launch, 21 instructions per value, of which 5 are the row
// maximum's reductions and divisions; 59 us and 32 instructions with one value at a time and a check on each).  The row is read twice: the first pass takes the maximum, the second
// quantises (its reads hit the L1 cache; a thread's first two units of 8 values stay in registers, which is all there is
// at decode widths).  The second pass is a loop that is NOT unrolled and keeps two units in flight: with four unrolled
// copies of the quantisation the kernel spent most of its time waiting for instructions, and with a register limit of 40
// the spills cost more (38 us) than the warps gained.
template <int kThreads>
__global__ void __launch_bounds__(kThreads, kThreads == 1024 ? 1 : 1280 / kThreads)
decompose_int8_kernel(const uint16_t* __restrict__ x, int64_t ldx, int K, int8_t* __restrict__ q1,
                      int8_t* __restrict__ q2, float* __restrict__ alpha_out, float* __restrict__ beta_out,
                      float c1, float c2) {
  // x may be the output of the preceding kernel, q1 / q2 its input.  Only then may the GEMM launched behind this kernel as
  // its programmatic dependent become resident: it asks for weights at once, and they too may have been written by what
  // precedes this kernel.  (Letting it in before the wait gained 1.5 us at 4096 x 4096 and nothing on larger weights.)
  pdl_wait_primary();
  pdl_launch_dependents();
  const int row = blockIdx.x;
  const uint4* xr = reinterpret_cast<const uint4*>(x + static_cast<int64_t>(row) * ldx);
  const int units = K >> 3;
  const int u0 = threadIdx.x;
  const uint4 zero = make_uint4(0, 0, 0, 0);
  uint4 cur = u0 < units ? __ldg(xr + u0) : zero;
  uint4 next = u0 + kThreads < units ? __ldg(xr + u0 + kThreads) : zero;
  float m = 0.0f;
#pragma unroll 4
  for (int u = u0 + 2 * kThreads; u < units; u += kThreads) m = fmaxf(m, unit_absmax(__ldg(xr + u)));
  m = fmaxf(m, fmaxf(unit_absmax(cur), unit_absmax(next)));

  __shared__ float warp_max[kThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
  __syncthreads();
  m = warp_max[threadIdx.x & (kThreads / 32 - 1)];
#pragma unroll
  for (int o = kThreads / 64; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));

  const float alpha = __fdiv_rn(m, c1);            // Eq. alpha (c1 = 127, or 127.49 with fractional scaling, Sec. 3.3)
  const float beta = __fdiv_rn(alpha, c2);         // Eq. beta  (c2 = 254, or 254.98)
  // reciprocals only steer the fast path of the quantisation
  const float inv_alpha = alpha > 0.0f ? __frcp_rn(alpha) : 0.0f;
  const float inv_beta = beta > 0.0f ? __frcp_rn(beta) : 0.0f;
  if (threadIdx.x == 0) {
    alpha_out[row] = alpha;
    beta_out[row] = beta;
  }
  if (unit_scales_ok(alpha, beta)) {
    uint2* o1 = reinterpret_cast<uint2*>(q1 + static_cast<int64_t>(row) * K);
    uint2* o2 = reinterpret_cast<uint2*>(q2 + static_cast<int64_t>(row) * K);
#pragma unroll 1
    for (int u = u0; u < units; u += kThreads) {
      uint4 after = zero;
      if (u + 2 * kThreads < units) after = __ldg(xr + u + 2 * kThreads);
      uint2 r1, r2;
      unit_quantize(cur, alpha, beta, inv_alpha, inv_beta, r1, r2);
      o1[u] = r1;
      o2[u] = r2;
      cur = next;
      next = after;
    }
  } else {
    // a zero row, or scales outside the range the fast path is proven for: value by value, with true divisions
#pragma unroll 1
    for (int k = threadIdx.x; k < K; k += kThreads) {
      const float v = __uint_as_float(static_cast<uint32_t>(__ldg(reinterpret_cast<const uint16_t*>(xr) + k)) << 16);
      int a = 0, b = 0;
      if (alpha > 0.0f) {
        a = quant_i8(v, alpha, inv_alpha);                               // Eq. x1
        const float r = __fmaf_rn(-alpha, static_cast<float>(a), v);     // Eq. residual, exact
        if (beta > 0.0f) b = quant_i8(r, beta, inv_beta);                // Eq. x2
      }
      q1[static_cast<int64_t>(row) * K + k] = static_cast<int8_t>(a);
      q2[static_cast<int64_t>(row) * K + k] = static_cast<int8_t>(b);
    }
  }
}

// ---- MXFP4 ------------------------------------------------------------------------------------------------------
constexpr int kMxThreads = 256;

// 2^e as an FP32 number for e in [-126, 127]
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float(static_cast<uint32_t>(e + 127) << 23); }

// The first `rl.blocks` CTAs do the (independent) scale relayout `rl`, the others the decomposition, 256 consecutive
// 32-element blocks (row-major) per CTA and round.
__global__ void __launch_bounds__(kMxThreads)
decompose_mxfp4_kernel(const uint16_t* __restrict__ x, int64_t ldx, int64_t M, int K, uint8_t* __restrict__ q1,
                       uint8_t* __restrict__ q2, uint8_t* __restrict__ e1, uint8_t* __restrict__ e2, int sf_kgroups,
                       const SfRelayout rl, const RowGroups rg) {
  pdl_wait_primary();            // as in decompose_int8_kernel
  pdl_launch_dependents();
  const int kblocks = K >> 5;
  const int64_t nblocks = M * kblocks;
  if (static_cast<int>(blockIdx.x) < rl.blocks) {
    __shared__ uint32_t sm_rl[kSfRelayoutSmemWords];
    sf_relayout(rl, blockIdx.x, rl.blocks, sm_rl);
    return;
  }
  const int64_t units = (nblocks + kMxThreads - 1) / kMxThreads;
  // whole warps of valid blocks and word-aligned scale positions (the scale arrays are then 4-byte aligned as well)
  const bool pack4 = (kblocks & 3) == 0 && ((reinterpret_cast<uintptr_t>(e1) | reinterpret_cast<uintptr_t>(e2)) & 3) == 0;
  for (int64_t u = blockIdx.x - rl.blocks; u < units; u += gridDim.x - rl.blocks) {
    const int64_t b = u * kMxThreads + threadIdx.x;
    const unsigned lanes = __ballot_sync(0xffffffffu, b < nblocks);      // the lanes of this warp that have a block
    if (b < nblocks) {
    const int64_t row_in = b / kblocks;
    const int kb = static_cast<int>(b - row_in * kblocks);
    const uint4* src = reinterpret_cast<const uint4*>(x + row_in * ldx + kb * 32);
    int64_t row = row_in, srow = row_in;    // where the row's first component and its scales go
    int second = rg.second;                 // rows from there to the second component's
    if (rg.n > 0) {
      int g = 0;
      for (int step = kMaxRowGroups / 2; step > 0; step >>= 1)
        if (g + step < rg.n && row_in >= rg.off[g + step]) g += step;
      row = static_cast<int64_t>(g) * rg.rows + (row_in - rg.off[g]);
      srow = static_cast<int64_t>(g) * rg.srows + (row_in - rg.off[g]);
      if (rg.stacked) second = (rg.off[g + 1] - rg.off[g] + 7) & ~7;
    }
    uint32_t w[16];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint4 t = __ldg(src + i);
      w[4 * i] = t.x; w[4 * i + 1] = t.y; w[4 * i + 2] = t.z; w[4 * i + 3] = t.w;
    }
    uint32_t m2 = 0;       // maximum of |x| as BF16 bits (monotone in the value for finite inputs), both halves at once
#pragma unroll
    for (int i = 0; i < 16; ++i) m2 = __vmaxu2(m2, w[i] & 0x7FFF7FFFu);
    const uint32_t mbits = max(m2 & 0xFFFFu, m2 >> 16);
    const int expf = static_cast<int>(mbits >> 7);
    int a = -123;
    if (expf > 0) a = max(-123, (expf - 127) - 2 + (((mbits & 0x7Fu) > 0x10u) ? 1 : 0));
    a = min(a, 127);
    const int bexp = a - 4;                                   // beta = alpha / 16
    // x / alpha and r / beta are exact multiplications by a power of two: a is in [-123, 126] for finite BF16 inputs
    // (largest exponent 127, minus 2, plus at most 1), so 2^-a and 2^(4-a) are normal FP32 numbers
    const float sa = pow2f(max(-a, -126)), sb = pow2f(-bexp);
    const float alpha = pow2f(a);
    uint32_t o1[4] = {0, 0, 0, 0}, o2[4] = {0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float v0 = bf16lo(w[i]), v1 = bf16hi(w[i]);
      const __nv_fp4x2_storage_t c1 =
          __nv_cvt_float2_to_fp4x2(make_float2(v0 * sa, v1 * sa), __NV_E2M1, cudaRoundNearest);
      const float2 d1 = __half22float2(__half2(__nv_cvt_fp4x2_to_halfraw2(c1, __NV_E2M1)));
      const float r0 = __fmaf_rn(-alpha, d1.x, v0), r1 = __fmaf_rn(-alpha, d1.y, v1);   // exact residuals
      const __nv_fp4x2_storage_t c2 =
          __nv_cvt_float2_to_fp4x2(make_float2(r0 * sb, r1 * sb), __NV_E2M1, cudaRoundNearest);
      o1[i >> 2] |= static_cast<uint32_t>(c1) << (8 * (i & 3));
      o2[i >> 2] |= static_cast<uint32_t>(c2) << (8 * (i & 3));
    }
    *reinterpret_cast<uint4*>(q1 + row * (K >> 1) + kb * 16) = make_uint4(o1[0], o1[1], o1[2], o1[3]);
    *reinterpret_cast<uint4*>(q2 + (row + second) * (K >> 1) + kb * 16) = make_uint4(o2[0], o2[1], o2[2], o2[3]);
    // sf_kgroups == 0: row-major [M, K/32]; otherwise the 512-byte blocks (128 rows x 4 scales) the block-scaled
    // MMA's shared-memory -> TMEM scale copy expects: block (row/128, kb/4), byte (row%32)*16 + ((row/32)%4)*4 + kb%4
    auto scale_at = [&](int64_t r) {
      return sf_kgroups == 0 ? r * kblocks + kb : ((r >> 7) * sf_kgroups + (kb >> 2)) * 512 + (r & 31) * 16 + ((r >> 5) & 3) * 4 + (kb & 3);
    };
    const int64_t so1 = scale_at(srow), so2 = scale_at(srow + second);
    if (pack4) {
      // four neighbouring lanes hold the four scales of one aligned 32-bit word (kblocks is a multiple of 4)
      uint32_t w1 = static_cast<uint32_t>(a + 127) << (8 * (threadIdx.x & 3)), w2 = static_cast<uint32_t>(bexp + 127) << (8 * (threadIdx.x & 3));
      w1 |= __shfl_xor_sync(lanes, w1, 1); w2 |= __shfl_xor_sync(lanes, w2, 1);
      w1 |= __shfl_xor_sync(lanes, w1, 2); w2 |= __shfl_xor_sync(lanes, w2, 2);
      if ((threadIdx.x & 3) == 0) {
        *reinterpret_cast<uint32_t*>(e1 + so1) = w1;
        *reinterpret_cast<uint32_t*>(e2 + so2) = w2;
      }
    } else {
      e1[so1] = static_cast<uint8_t>(a + 127);
      e2[so2] = static_cast<uint8_t>(bexp + 127);
    }
    // A K that ends halfway through a 256-element block leaves it a group of four scales that the MMAs take with operands of zeros: they
    // must be numbers (0xFF is NaN), whatever the workspace held.
    if (sf_kgroups > (kblocks >> 2) && kb + 4 >= kblocks) e1[so1 + 512] = e2[so2 + 512] = 0;
    }
  }
}

msd_status_t launch_decompose_int8(const void* x_bf16, int64_t M, int64_t K, int64_t ldx, int8_t* q1, int8_t* q2,
                                   float* alpha, float* beta, float c1, float c2, cudaStream_t stream) {
  if (M == 0) return MSD_OK;
  // A programmatic dependent of whatever precedes it (in a chain of layers: the previous layer's GEMM), so that its launch
  // and the launch of the GEMM behind it are over when that kernel ends; launched plainly, 4 to 5 us passed between two
  // GEMMs in which no weights moved (16 tokens, 4096 x 4096: 14.9 us a call launched plainly, 13.2 as a dependent; 1 token, 14336 x 4096:
  // 18.6 and 16.9).
  // Few rows: the kernel sits on the critical path of the GEMM behind it, and more threads per row mean a shorter
  // latency.  Many rows: throughput counts, so a thread takes several units and many rows share an SM.  Whole calls, us with 128 / 256 /
  // 512 / 1024 threads a row: 160 rows, 4096 x 4096 21.0 / 18.5 / 17.7 / 18.9; 400, 24.9 with 256 and 24.7 with 512; 1000, 35.1 / 32.7 /
  // 34.2 / 39.5; 129 rows, 4096 x 14336 48.1 / 39.6 / 36.2 / 34.3; 600, 102.9 / 88.7 / 84.8 / 87.2; 2500, 231 / 221 / 242 / 258; 1000 rows,
  // 2048 x 1024 14.4 / 14.7 / 17.0 / 22.0.
  int threads = K >= 8192 ? 1024 : (K >= 2048 ? 512 : 256);
  if (M > 448) threads /= 2;
  if (M > 800 && threads == 512) threads = 256;
  auto kernel = threads == 1024 ? decompose_int8_kernel<1024>
              : threads == 512 ? decompose_int8_kernel<512>
              : threads == 256 ? decompose_int8_kernel<256> : decompose_int8_kernel<128>;
  const cudaError_t err = launch_pdl(kernel, dim3(static_cast<unsigned>(M)), dim3(static_cast<unsigned>(threads)), 0, stream, option(OPT_NO_PDL) <= 0,
                                     static_cast<const uint16_t*>(x_bf16), ldx, static_cast<int>(K), q1, q2, alpha, beta, c1, c2);
  return err == cudaSuccess ? MSD_OK : MSD_ERR_CUDA;
}

msd_status_t launch_decompose_mxfp4(const void* x_bf16, int64_t M, int64_t K, int64_t ldx, uint8_t* q1, uint8_t* q2,
                                    uint8_t* e1, uint8_t* e2, int sf_kgroups, cudaStream_t stream, SfRelayout* relayout,
                                    const RowGroups* groups) {
  if (M == 0) return MSD_OK;
  const int per_sm = 32, rl_per_sm = (relayout && relayout->matrices > 1) ? 16 : 4;
  SfRelayout rl = {};
  if (relayout) {
    rl = *relayout;
    const int64_t rb = static_cast<int64_t>(rl.row_blocks) * ((rl.sf_kgroups + 31) / 32) * (rl.matrices > 1 ? rl.matrices : 1);   // units
    rl.blocks = static_cast<int>(rb < rl_per_sm * sm_count() ? rb : rl_per_sm * sm_count());
    relayout->blocks = rl.blocks;
  }
  RowGroups rg = {};
  if (groups) rg = *groups;
  const int64_t nblocks = M * (K >> 5);
  const int64_t want = (nblocks + kMxThreads - 1) / kMxThreads;
  const int64_t cap = static_cast<int64_t>(sm_count()) * per_sm;
  const unsigned grid = static_cast<unsigned>(want < cap ? want : cap) + static_cast<unsigned>(rl.blocks);
  static DeviceOnce once;
  once([] { return cudaFuncSetAttribute(decompose_mxfp4_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) == cudaSuccess; });
  const cudaError_t err = launch_pdl(decompose_mxfp4_kernel, dim3(grid), dim3(kMxThreads), 0, stream, option(OPT_NO_PDL) <= 0,
                                     static_cast<const uint16_t*>(x_bf16), ldx, M, static_cast<int>(K), q1, q2, e1, e2, sf_kgroups, rl, rg);
  return err == cudaSuccess ? MSD_OK : MSD_ERR_CUDA;
}

}  // namespace msd

extern "C" {

msd_status_t msd_decompose_int8_ex(const void* x_bf16, int64_t M, int64_t K, int64_t ldx, int8_t* q1, int8_t* q2,
                                   float* alpha, float* beta, msd_scaling_t scaling, void* stream) {
  if (scaling != MSD_SCALING_DEFAULT && scaling != MSD_SCALING_FRACTIONAL) return MSD_ERR_UNSUPPORTED;
  if (M < 0 || K <= 0 || K % 16 != 0 || ldx < K || ldx % 8 != 0 || M > 0x7FFFFFFF || K > 0x7FFFFFF0) return MSD_ERR_BAD_SHAPE;
  if (M == 0) return MSD_OK;
  if (!x_bf16 || !q1 || !q2 || !alpha || !beta) return MSD_ERR_NULL_POINTER;
  if (!msd::aligned(x_bf16, 16) || !msd::aligned(q1, 16) || !msd::aligned(q2, 16) || !msd::aligned(alpha, 4) ||
      !msd::aligned(beta, 4))
    return MSD_ERR_BAD_ALIGNMENT;
  return msd::launch_decompose_int8(x_bf16, M, K, ldx, q1, q2, alpha, beta, msd::scaling_c1(scaling), msd::scaling_c2(scaling),
                                    static_cast<cudaStream_t>(stream));
}

msd_status_t msd_decompose_int8(const void* x_bf16, int64_t M, int64_t K, int64_t ldx, int8_t* q1, int8_t* q2,
                                float* alpha, float* beta, void* stream) {
  return msd_decompose_int8_ex(x_bf16, M, K, ldx, q1, q2, alpha, beta, MSD_SCALING_DEFAULT, stream);
}

msd_status_t msd_decompose_mxfp4(const void* x_bf16, int64_t M, int64_t K, int64_t ldx, uint8_t* q1, uint8_t* q2,
                                 uint8_t* e8m0_1, uint8_t* e8m0_2, void* stream) {
  if (M < 0 || K <= 0 || K % 32 != 0 || ldx < K || ldx % 8 != 0 || K > 0x7FFFFFE0) return MSD_ERR_BAD_SHAPE;
  if (M == 0) return MSD_OK;
  if (!x_bf16 || !q1 || !q2 || !e8m0_1 || !e8m0_2) return MSD_ERR_NULL_POINTER;
  if (!msd::aligned(x_bf16, 16) || !msd::aligned(q1, 16) || !msd::aligned(q2, 16)) return MSD_ERR_BAD_ALIGNMENT;
  return msd::launch_decompose_mxfp4(x_bf16, M, K, ldx, q1, q2, e8m0_1, e8m0_2, 0, static_cast<cudaStream_t>(stream));
}

}  // extern "C"
