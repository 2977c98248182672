// rotate_quant_rows.cu -- one CTA per row: rotation x R (Sec. 3.1, R4 and the
// weight merge W' = W R) followed by the Eq. 1 quantizer of the whole row.
//
// The row is transformed in shared memory as fp32 (row_transform.cuh; K <=
// 32768 -> 128 KB).  The 1/sqrt(K) normalization is not applied to the
// elements: Eq. 1 codes do not change when a row is scaled, so only alpha and
// beta are multiplied by it.  Without a rotation the row stays in registers.
// GB300, 4-bit weights: 4096 x 14336 merged with H_28 (x) H_512 675 -> 99 us
// (56 % of the FP32 pipe, whose additions alone take 54 us), 3072 x 8192 with
// H_8192 124 -> 33 us, 28672 x 4096 without a rotation 98 -> 66 us (0.65 of
// HBM).
//
// This kernel serves the offline weight path (any supported size) and every
// activation shape that the specialised kernel does not cover.
#include <cuda_fp16.h>

#include "launch_util.h"
#include "row_transform.cuh"
#include "spinq_device.cuh"
#include "spinq_internal.h"

namespace spinq {
namespace {

constexpr int kThreads = kRowThreads;

__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// NS: order of the small factor; 0: no rotation, the row in CPT chunks per
// thread.
template <int NS, int CPT, bool SYM, bool ROWSUM, bool CLAMP>
__global__ void __launch_bounds__(kThreads, NS > 1 ? 3 : CPT > 8 ? 2 : 4) rotate_quant_rows_kernel(RotQuantArgs a) {
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
      range = row_transform<NS, SYM>(x + row * a.ldx, a.signs, s, K, a.n_pow2, red);
    }
    const float hi = range.hi, lo = range.lo;
    // Eq. 1 on the unnormalised row; alpha and beta carry the normalisation.
    float inv, off, alpha, beta = 0.f;
    if (SYM) {
      const float m = a.clip * hi;
      alpha = m / 7.f;
      inv = m > 0.f ? 7.f / m : 0.f;
      off = 0.f;
    } else {
      const float h2 = a.clip * hi, l2 = a.clip * lo;
      alpha = (h2 - l2) / 15.f;
      inv = h2 > l2 ? 15.f / (h2 - l2) : 0.f;
      beta = l2;
      off = -l2 * inv;
    }

    int csum = 0;
    uint32_t* out = reinterpret_cast<uint32_t*>(a.codes + row * (a.K / 2));
    auto quant8 = [&](int c, const float (&v)[8]) {
      uint32_t r[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float t = fmaf(v[e], inv, off);
        if (CLAMP) t = SYM ? fminf(fmaxf(t, -8.f), 7.f) : fminf(fmaxf(t, 0.f), 15.f);
        r[e] = round_bits(t);
        if (ROWSUM) csum += (int)(r[e] - __float_as_uint(kRoundMagic));
      }
      out[c] = pack8_nibbles(r);
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
    if (ROWSUM) {
      csum = warp_sum(csum);
      if (lane == 0) red_sum[warp] = csum;
    }
    __syncthreads();
    if (tid == 0) {
      a.scale[row] = alpha * a.norm;
      if (!SYM) a.zero[row] = beta * a.norm;
      if (ROWSUM) {
        int tot = 0;
        for (int w = 0; w < kThreads / 32; ++w) tot += red_sum[w];
        a.rowsum[row] = tot;
      }
    }
    __syncthreads();
  }
}

template <int NS, int CPT, bool SYM, bool ROWSUM, bool CLAMP>
cudaError_t launch_ns(const RotQuantArgs& a, cudaStream_t stream) {
  const size_t smem = NS == 0 ? 0 : sizeof(float) * (size_t)a.K;
  auto kern = rotate_quant_rows_kernel<NS, CPT, SYM, ROWSUM, CLAMP>;
  int per_sm = 0;
  cudaError_t e = prepare_launch(kern, kThreads, smem, &per_sm);
  if (e != cudaSuccess) return e;
  // Rotated rows: one resident wave, so that a CTA can bring its next row
  // into L2 while it transforms this one (119 -> 99 us at 4096 x 14336 with
  // the compile-time column addresses).  A CTA per row without a rotation:
  // there the loads of many short rows have to be in flight together
  // (28672 x 4096: 98 -> 66 us).
  const int64_t cap = NS == 0 ? INT32_MAX : (int64_t)device_sm_count() * per_sm;
  const int64_t grid = a.rows < cap ? a.rows : cap;
  e = launch_pdl(kern, dim3((unsigned)grid), dim3(kThreads), smem, stream, 1, a);
  return e;
}

template <bool SYM, bool ROWSUM, bool CLAMP>
cudaError_t launch_t(const RotQuantArgs& a, cudaStream_t stream) {
  switch (a.n_small) {
    case 0:
      return with_row_chunks(a.K, [&](auto cpt) { return launch_ns<0, cpt(), SYM, ROWSUM, CLAMP>(a, stream); });
    case 12: return launch_ns<12, 1, SYM, ROWSUM, CLAMP>(a, stream);
    case 20: return launch_ns<20, 1, SYM, ROWSUM, CLAMP>(a, stream);
    case 28: return launch_ns<28, 1, SYM, ROWSUM, CLAMP>(a, stream);
  }
  return launch_ns<1, 1, SYM, ROWSUM, CLAMP>(a, stream);
}

}  // namespace

cudaError_t launch_rotate_quant_rows(const RotQuantArgs& a, cudaStream_t stream) {
  if (a.rows == 0) return cudaSuccess;
  bool handled = false;
  cudaError_t e = launch_rotate_quant_act_fast(a, stream, &handled);
  if (handled || e != cudaSuccess) return e;
  e = launch_rotate_quant_act_paley(a, stream, &handled);
  if (handled || e != cudaSuccess) return e;
  const bool clamp = a.clip < 1.0f;
  if (a.symmetric) {
    if (a.rowsum) return clamp ? launch_t<true, true, true>(a, stream) : launch_t<true, true, false>(a, stream);
    return clamp ? launch_t<true, false, true>(a, stream) : launch_t<true, false, false>(a, stream);
  }
  if (a.rowsum) return cudaErrorInvalidValue;
  return clamp ? launch_t<false, false, true>(a, stream) : launch_t<false, false, false>(a, stream);
}

}  // namespace spinq
