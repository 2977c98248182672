// rotate_quant_8bit.cu -- the quantizers of the 8-bit linears (main results
// table, 4-8-x rows; appendix "Latency measurement on GPU", FP8 setting):
// the online rotation x R (Sec. 3.1, skipped when there is none) followed by
//
//   kFmtInt8Planes  Eq. 1 with N = 8 (per token): code c = q (symmetric) or
//                   u - 128 (asymmetric), stored as the two E4M3 planes the
//                   W4A8 GEMM reads: row [2K] bytes, byte k = E4M3(16 (c >> 4)),
//                   byte K + k = E4M3(c & 15) (both exact);
//   kFmtE4M3        per-row FP8: alpha = clip max|x| / 448, code =
//                   E4M3(x / alpha) rounded to nearest even, saturating;
//   kFmtInt4Bytes   Eq. 1 with N = 4, symmetric per output channel (weights of
//                   the W4A8 linear): each 4-bit code stored as one E4M3 byte,
//                   plus the row sum of the codes.
//
// One CTA of 256 threads per row (persistent over rows), the row transformed
// in shared memory as fp32, or kept in registers without a rotation
// (row_transform.cuh).  GB300: the activations of 2048 x 4096 without a
// rotation 8.4 -> 4.5 us (FP8) and 9.7 -> 6.7 us (planes), 2048 x 8192 with
// H_8192 91.8 -> 20.3 us (FP8), 4096 x 14336 INT4_BYTES weights merged with
// H_28 (x) H_512 401 -> 99 us.
// Codes are taken on the unnormalised row; alpha and beta carry 1/sqrt(K).
#include <cuda_fp16.h>

#include "launch_util.h"
#include "row_transform.cuh"
#include "spinq_device.cuh"
#include "spinq_internal.h"

namespace spinq {
namespace {

constexpr int kThreads = kRowThreads;

__device__ __forceinline__ uint32_t e4m3x2(float lo, float hi) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return r;
}

// NS: order of the small factor; 0: no rotation, the row in CPT chunks per
// thread.
template <int FMT, bool SYM, bool CLAMP, int NS, int CPT>
__global__ void __launch_bounds__(kThreads, NS > 1 ? 3 : CPT > 8 ? 2 : 4) rq8_rows_kernel(Rq8Args a) {
  extern __shared__ __align__(16) float s[];
  __shared__ float red[2 * kThreads / 32];
  __shared__ int red_sum[kThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K = (int)a.K;
  const __half* __restrict__ x = reinterpret_cast<const __half*>(a.x);
  pdl_wait();
  pdl_trigger();

  for (int64_t row = blockIdx.x; row < a.rows; row += gridDim.x) {
    uint4 plain[CPT];
    RowRange<SYM> range;
    if constexpr (NS == 0) {
      range = row_plain<CPT, SYM>(x + row * a.ldx, K, plain, red);
    } else {
      if (row + gridDim.x < a.rows) row_prefetch(x + (row + gridDim.x) * a.ldx, K);
      range = row_transform<NS, SYM>(x + row * a.ldx, nullptr, s, K, a.n_pow2, red);
    }
    const float hi = range.hi, lo = range.lo;
    // per-row constants (unnormalised row)
    float inv, off = 0.f, alpha, beta = 0.f;
    if (FMT == kFmtE4M3) {
      const float m = a.clip * hi;
      alpha = m * (1.f / 448.f);
      inv = m > 0.f ? 448.f / m : 0.f;
    } else {
      const float qmax = FMT == kFmtInt8Planes ? 127.f : 7.f;
      if (SYM) {
        const float m = a.clip * hi;
        alpha = m / qmax;
        inv = m > 0.f ? qmax / m : 0.f;
      } else {
        const float h2 = a.clip * hi, l2 = a.clip * lo;
        alpha = (h2 - l2) / 255.f;
        inv = h2 > l2 ? 255.f / (h2 - l2) : 0.f;
        beta = l2;
        off = -l2 * inv;
      }
    }
    int csum = 0;
    uint8_t* out = a.codes + row * (FMT == kFmtInt8Planes ? 2 * a.K : a.K);
    auto quant8 = [&](int c, const float (&v)[8]) {
      uint32_t w0[2] = {0, 0}, w1[2] = {0, 0};
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        float t0 = fmaf(v[e], inv, off), t1 = fmaf(v[e + 1], inv, off);
        uint32_t b0, b1;
        if (FMT == kFmtE4M3) {
          b0 = e4m3x2(t0, t1);   // both bytes at once: lo element in the low byte
          b1 = 0;
        } else {
          if (FMT == kFmtInt8Planes) {
            if (CLAMP) {
              t0 = SYM ? fminf(fmaxf(t0, -128.f), 127.f) : fminf(fmaxf(t0, 0.f), 255.f);
              t1 = SYM ? fminf(fmaxf(t1, -128.f), 127.f) : fminf(fmaxf(t1, 0.f), 255.f);
            }
            const int c0 = __float2int_rn(t0) - (SYM ? 0 : 128), c1 = __float2int_rn(t1) - (SYM ? 0 : 128);
            b0 = e4m3x2((float)(16 * (c0 >> 4)), (float)(16 * (c1 >> 4)));
            b1 = e4m3x2((float)(c0 & 15), (float)(c1 & 15));
          } else {   // kFmtInt4Bytes: symmetric 4-bit codes, one per byte
            if (CLAMP) {
              t0 = fminf(fmaxf(t0, -8.f), 7.f);
              t1 = fminf(fmaxf(t1, -8.f), 7.f);
            }
            const int c0 = __float2int_rn(t0), c1 = __float2int_rn(t1);
            csum += c0 + c1;
            b0 = e4m3x2((float)c0, (float)c1);
            b1 = 0;
          }
        }
        w0[e >> 2] |= b0 << (8 * (e & 3));
        w1[e >> 2] |= b1 << (8 * (e & 3));
      }
      *reinterpret_cast<uint2*>(out + 8 * c) = make_uint2(w0[0], w0[1]);
      if (FMT == kFmtInt8Planes) *reinterpret_cast<uint2*>(out + a.K + 8 * c) = make_uint2(w1[0], w1[1]);
    };
    float v[8];
    if constexpr (NS == 0) {
#pragma unroll
      for (int i = 0; i < CPT; ++i) {
        if (tid + kThreads * i >= K / 8) break;
        row_get8(plain[i], v);
        quant8(tid + kThreads * i, v);
      }
    } else {
      for (int c = tid; c < K / 8; c += kThreads) {
        row_get8(s, c, v);
        quant8(c, v);
      }
    }
    if (FMT == kFmtInt4Bytes) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) csum += __shfl_xor_sync(0xffffffffu, csum, o);
      if (lane == 0) red_sum[warp] = csum;
    }
    __syncthreads();
    if (tid == 0) {
      a.scale[row] = alpha * a.norm;
      if (!SYM && FMT == kFmtInt8Planes) a.zero[row] = beta * a.norm;
      if (FMT == kFmtInt4Bytes && a.rowsum) {
        int tot = 0;
        for (int w = 0; w < kThreads / 32; ++w) tot += red_sum[w];
        a.rowsum[row] = tot;
      }
    }
    __syncthreads();
  }
}

template <int FMT, bool SYM, bool CLAMP, int NS, int CPT>
cudaError_t launch_ns(const Rq8Args& a, cudaStream_t stream) {
  const size_t smem = NS == 0 ? 0 : sizeof(float) * (size_t)a.K;
  auto kern = rq8_rows_kernel<FMT, SYM, CLAMP, NS, CPT>;
  int per_sm = 0;
  cudaError_t e = prepare_launch(kern, kThreads, smem, &per_sm);
  if (e != cudaSuccess) return e;
  const int64_t cap = NS == 0 ? INT32_MAX : (int64_t)device_sm_count() * per_sm;
  const int64_t grid = a.rows < cap ? a.rows : cap;
  e = launch_pdl(kern, dim3((unsigned)grid), dim3(kThreads), smem, stream, 1, a);
  return e;
}

template <int FMT, bool SYM, bool CLAMP>
cudaError_t launch_t(const Rq8Args& a, cudaStream_t stream) {
  switch (a.n_small) {
    case 0:
      return with_row_chunks(a.K, [&](auto cpt) { return launch_ns<FMT, SYM, CLAMP, 0, cpt()>(a, stream); });
    case 12: return launch_ns<FMT, SYM, CLAMP, 12, 1>(a, stream);
    case 20: return launch_ns<FMT, SYM, CLAMP, 20, 1>(a, stream);
    case 28: return launch_ns<FMT, SYM, CLAMP, 28, 1>(a, stream);
  }
  return launch_ns<FMT, SYM, CLAMP, 1, 1>(a, stream);
}

template <int FMT>
cudaError_t launch_fmt(const Rq8Args& a, cudaStream_t stream) {
  const bool clamp = a.clip < 1.0f;
  if (a.symmetric) return clamp ? launch_t<FMT, true, true>(a, stream) : launch_t<FMT, true, false>(a, stream);
  if constexpr (FMT == kFmtInt8Planes)   // the only asymmetric format
    return clamp ? launch_t<FMT, false, true>(a, stream) : launch_t<FMT, false, false>(a, stream);
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_rotate_quant_8bit(const Rq8Args& a, cudaStream_t stream) {
  if (a.rows == 0) return cudaSuccess;
  // a Paley rotation with the unclipped activation formats: the Paley kernel
  bool handled = false;
  const cudaError_t ep = launch_rotate_quant_8bit_paley(a, stream, &handled);
  if (ep != cudaSuccess || handled) return ep;
  switch (a.format) {
    case kFmtInt8Planes: return launch_fmt<kFmtInt8Planes>(a, stream);
    case kFmtE4M3: return launch_fmt<kFmtE4M3>(a, stream);
    case kFmtInt4Bytes: return launch_fmt<kFmtInt4Bytes>(a, stream);
  }
  return cudaErrorNotSupported;
}

}  // namespace spinq
