// row_transform.cuh -- one row of a rotation x (H_s (x) H_P) by one CTA, fp32
// in shared memory; shared by the row kernels of the 4-bit and the 8-bit
// quantizers (weights of every size, and the activations that no specialised
// kernel takes).
//
// The arithmetic is the radix-2 one: butterflies (u + w, u - w) over the bits
// of the fast index from the lowest to the highest, then for every column the
// sum over the slow index i' = 0, 1, .. of +-x[i'] in that order, starting at
// zero.  Every addition is rounded to fp32, so the order fixes the results.
//
// What bounds it: the additions themselves.  A row of H_28 (x) H_512 takes 9 +
// 28 additions per element, 14336 * 37 / 128 lanes = 4144 cycles per SM; one
// stage per CTA barrier and a runtime-indexed column kept that pipe idle
// (a shared-memory round trip per stage, the column in local memory).  Here:
//   - a thread loads 32 consecutive elements and takes the first five stages
//     in registers, then up to four stages per shared-memory pass on 16 x 2
//     elements (two neighbouring columns as a packed pair);
//   - the small factor's signs are compile-time constants, a thread owns two
//     neighbouring columns and every addition is one packed instruction.
// 4096 x 14336 weights with H_28 (x) H_512: 675 us before, 99 us now.
#pragma once

#include <cuda_fp16.h>
#include <float.h>

#include <type_traits>

#include "spinq_device.cuh"

namespace spinq {

constexpr int kRowThreads = 256;

// Paley I signs at compile time (the construction of hadamard_tables.cu):
// true where H_n[r][c] = -1.
template <int N>
struct PaleySigns {
  bool neg[N][N];
  constexpr PaleySigns() : neg() {
    constexpr int q = N - 1;
    bool square[N] = {};
    for (int a = 1; a < q; ++a) square[mul(a, a)] = true;
    for (int r = 0; r < N; ++r)
      for (int c = 0; c < N; ++c)
        neg[r][c] = r == c || r == 0 ? false : c == 0 ? true : !square[sub(r - 1, c - 1)];
  }
  static constexpr int sub(int a, int b) {
    constexpr int q = N - 1;
    if (q != 27) return (a - b + q) % q;
    return (a % 3 - b % 3 + 3) % 3 + 3 * ((a / 3 % 3 - b / 3 % 3 + 3) % 3) + 9 * ((a / 9 - b / 9 + 3) % 3);
  }
  static constexpr int mul(int a, int b) {
    constexpr int q = N - 1;
    if (q != 27) return a * b % q;
    const int x[3] = {a % 3, a / 3 % 3, a / 9}, y[3] = {b % 3, b / 3 % 3, b / 9};
    int z[5] = {};
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) z[i + j] += x[i] * y[j];
    // over GF(3): t^4 = t^2 + 2 t, t^3 = t + 2
    z[2] += z[4], z[1] += 2 * z[4] + z[3], z[0] += 2 * z[3];
    return z[0] % 3 + 3 * (z[1] % 3) + 9 * (z[2] % 3);
  }
};

// Where element a of the row lives in shared memory: the 16-byte chunk bits
// 2..4 are XOR-ed with higher bits, so that the first stage's stores (32
// consecutive elements per thread), the passes (neighbouring pairs across the
// lanes) and the quantizer's loads (8 consecutive elements per thread) meet
// no bank conflict.  Linear over XOR: phys(a ^ b) = phys(a) ^ phys(b).
__host__ __device__ constexpr uint32_t row_phys(uint32_t a) {
  const uint32_t h = (a >> 5) & 31u;
  return a ^ ((h & 3u) << 2) ^ (((h ^ (h >> 1) ^ (h >> 2) ^ (h >> 3) ^ (h >> 4)) & 1u) << 4);
}

// Running range of a thread's final values.
template <bool SYM>
struct RowRange {
  float hi = SYM ? 0.f : -FLT_MAX, lo = FLT_MAX;
  __device__ __forceinline__ void add(float a, float b) {   // 3-input max / min
    if (SYM) {
      asm("max.f32 %0, %0, %1, %2;" : "+f"(hi) : "f"(fabsf(a)), "f"(fabsf(b)));
    } else {
      asm("max.f32 %0, %0, %1, %2;" : "+f"(hi) : "f"(a), "f"(b));
      asm("min.f32 %0, %0, %1, %2;" : "+f"(lo) : "f"(a), "f"(b));
    }
  }
  __device__ __forceinline__ void add(F2 v) {
    float a, b;
    f2_split(v, a, b);
    add(a, b);
  }
};

// Loads the row (fp16, K % 32 == 0), applies the random signs and stages
// 0 .. G0 - 1, and stores it as fp32.
template <int G0, bool SYM>
__device__ __forceinline__ void row_load(const __half* xr, const uint8_t* signs, float* s, int K, bool last,
                                         RowRange<SYM>& range) {
  for (int c = threadIdx.x; c < K / 32; c += kRowThreads) {
    F2 f[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint4 v = __ldg(reinterpret_cast<const uint4*>(xr) + 4 * c + q);
      if (signs) {   // bit e: element 8 (4 c + q) + e
        const uint32_t sb = signs[4 * c + q];
        v.x ^= ((sb << 15) & 0x8000u) | ((sb << 30) & 0x80000000u);
        v.y ^= ((sb << 13) & 0x8000u) | ((sb << 28) & 0x80000000u);
        v.z ^= ((sb << 11) & 0x8000u) | ((sb << 26) & 0x80000000u);
        v.w ^= ((sb << 9) & 0x8000u) | ((sb << 24) & 0x80000000u);
      }
      const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 t = __half22float2(h[e]);
        f[4 * q + e] = f2_make(t.x, t.y);
      }
    }
#pragma unroll
    for (int p = 0; p < 16; ++p) f2_bfly_inner(f[p]);
#pragma unroll
    for (int d = 1; d < (1 << (G0 - 1)); d <<= 1)
#pragma unroll
      for (int p = 0; p < 16; ++p)
        if (!(p & d)) f2_bfly(f[p], f[p | d]);
    if (last) {
#pragma unroll
      for (int p = 0; p < 16; ++p) range.add(f[p]);
    }
    const uint32_t pb = row_phys(32u * (uint32_t)c);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      float4 o;
      f2_split(f[2 * q], o.x, o.y);
      f2_split(f[2 * q + 1], o.z, o.w);
      *reinterpret_cast<float4*>(s + (pb ^ (4u * q))) = o;
    }
  }
}

// Stages LH .. LH + R - 1 of every block of 2^(LH + R) elements.
template <int LH, int R, bool SYM>
__device__ __forceinline__ void row_pass(float* s, int K, bool last, RowRange<SYM>& range) {
  for (int p = threadIdx.x; p < K >> (R + 1); p += kRowThreads) {
    const uint32_t l = 2u * (p & ((1u << (LH - 1)) - 1u)), rest = (uint32_t)p >> (LH - 1);
    const uint32_t pb = row_phys((rest << (LH + R)) | l);
    F2 v[1 << R];
    // the element's own bits are added, only the bank bits need an XOR
    auto at = [&](int k) -> float2* {
      const uint32_t off = (uint32_t)k << LH;
      return reinterpret_cast<float2*>(s + (pb ^ (row_phys(off) ^ off)) + off);
    };
#pragma unroll
    for (int k = 0; k < 1 << R; ++k) {
      const float2 t = *at(k);
      v[k] = f2_make(t.x, t.y);
    }
#pragma unroll
    for (int d = 1; d < 1 << R; d <<= 1)
#pragma unroll
      for (int k = 0; k < 1 << R; ++k)
        if (!(k & d)) f2_bfly(v[k], v[k | d]);
#pragma unroll
    for (int k = 0; k < 1 << R; ++k) {
      float2 t;
      f2_split(v[k], t.x, t.y);
      *at(k) = t;
      if (last) range.add(v[k]);
    }
  }
}

template <int LH, bool SYM>
__device__ __forceinline__ void row_passes(float* s, int K, int r, bool last, RowRange<SYM>& range) {
  switch (r) {
    case 1: return row_pass<LH, 1>(s, K, last, range);
    case 2: return row_pass<LH, 2>(s, K, last, range);
    case 3: return row_pass<LH, 3>(s, K, last, range);
    default: return row_pass<LH, 4>(s, K, last, range);
  }
}

// acc +- t.  Volatile, so that the sums stay in program order: shared prefixes
// of the sums, kept for later outputs, would cost the registers that hold the
// columns (228 bytes of spills at three CTAs per SM).
__device__ __forceinline__ void f2_accumulate(F2& acc, F2 t, bool neg) {
  if (neg) {
    asm volatile("sub.rn.f32x2 %0, %0, %1;" : "+l"(acc.u) : "l"(t.u));
  } else {
    asm volatile("add.rn.f32x2 %0, %0, %1;" : "+l"(acc.u) : "l"(t.u));
  }
}

// y[i][j] = sum_i' x[i'][j] H_s[i'][i] over the slow index, in place (a thread
// owns the columns j, j + 1).  PC: the block size P at compile time, so that
// the column's addresses are immediate offsets; 0: P at run time.
template <int NS, int PC, bool SYM>
__device__ __forceinline__ void row_small_factor(float* s, int P, RowRange<SYM>& range) {
  constexpr PaleySigns<NS> H{};
  const F2 zero = f2_make(0.f, 0.f);
  if (PC) P = PC;
  for (int j = 2 * threadIdx.x; j < P; j += 2 * kRowThreads) {
    const uint32_t pj = row_phys((uint32_t)j);
    // the block's bits are disjoint from the column's; added (an immediate) where
    // they also lie above the bank bits that row_phys changes
    auto at = [&](int i) -> float2* {
      const uint32_t off = (uint32_t)(i * P);
      if constexpr (PC >= 32) return reinterpret_cast<float2*>(s + (pj ^ (row_phys(off) ^ off)) + off);
      return reinterpret_cast<float2*>(s + (pj ^ row_phys(off)));
    };
    F2 t[NS];
#pragma unroll
    for (int ip = 0; ip < NS; ++ip) {
      const float2 v = *at(ip);
      t[ip] = f2_make(v.x, v.y);
    }
#pragma unroll
    for (int i = 0; i < NS; i += 2) {
      F2 acc[2] = {zero, zero};
#pragma unroll
      for (int ip = 0; ip < NS; ++ip)
#pragma unroll
        for (int u = 0; u < 2; ++u) f2_accumulate(acc[u], t[ip], H.neg[ip][i + u]);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        range.add(acc[u]);
        float2 o;
        f2_split(acc[u], o.x, o.y);
        *at(i + u) = o;
      }
    }
  }
}

// Brings the row at xr into L2 (the CTA's next row, while this one is
// transformed).
__device__ __forceinline__ void row_prefetch(const __half* xr, int K) {
  for (int c = threadIdx.x; c < K / 64; c += kRowThreads)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(xr + 64 * c));
}

// Combines the CTA's ranges.  `red`: 2 * kRowThreads / 32 floats.
template <bool SYM>
__device__ __forceinline__ void row_block_range(RowRange<SYM>& range, float* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    range.hi = fmaxf(range.hi, __shfl_xor_sync(0xffffffffu, range.hi, o));
    if (!SYM) range.lo = fminf(range.lo, __shfl_xor_sync(0xffffffffu, range.lo, o));
  }
  if (lane == 0) {
    red[warp] = range.hi;
    red[kRowThreads / 32 + warp] = range.lo;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kRowThreads / 32; ++w) {
    range.hi = fmaxf(range.hi, red[w]);
    if (!SYM) range.lo = fminf(range.lo, red[kRowThreads / 32 + w]);
  }
}

// The whole transform of one row: fp16 in global memory to fp32 in `s`
// (element a at row_phys(a)), with the CTA's range of the final values.
// `red`: 2 * kRowThreads / 32 floats.  Ends with every thread past a barrier
// that follows all stores to s.
template <int NS, bool SYM>
__device__ __forceinline__ RowRange<SYM> row_transform(const __half* xr, const uint8_t* signs, float* s, int K,
                                                       int P, float* red) {
  RowRange<SYM> range;
  const int lg = 31 - __clz(P);
  if (lg >= 5) {
    row_load<5>(xr, signs, s, K, NS == 1 && lg == 5, range);
  } else if (lg == 4) {
    row_load<4>(xr, signs, s, K, NS == 1, range);
  } else {   // 8, the smallest block (K % 32 == 0)
    row_load<3>(xr, signs, s, K, NS == 1, range);
  }
  __syncthreads();
  if (lg > 5) {
    row_passes<5>(s, K, lg - 5 < 4 ? lg - 5 : 4, NS == 1 && lg <= 9, range);
    __syncthreads();
  }
  if (lg > 9) {
    row_passes<9>(s, K, lg - 9 < 4 ? lg - 9 : 4, NS == 1 && lg <= 13, range);
    __syncthreads();
  }
  if (lg > 13) {   // 16384, the largest
    row_pass<13, 1>(s, K, NS == 1, range);
    __syncthreads();
  }
  if constexpr (NS > 1) {
    if (P == 512) {
      row_small_factor<NS, 512>(s, P, range);
    } else if (P == 256) {
      row_small_factor<NS, 256>(s, P, range);
    } else {
      row_small_factor<NS, 0>(s, P, range);
    }
    __syncthreads();
  }
  row_block_range(range, red);
  return range;
}

// The 8 consecutive elements 8 c .. 8 c + 7 of the transformed row.
__device__ __forceinline__ void row_get8(const float* s, int c, float (&v)[8]) {
  const uint32_t pb = row_phys(8u * (uint32_t)c);
  const float4 a = *reinterpret_cast<const float4*>(s + pb), b = *reinterpret_cast<const float4*>(s + (pb ^ 4u));
  v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
}

// A row without a rotation stays in registers: up to CPT 16-byte chunks (8
// elements) per thread, chunk tid + kRowThreads v in c[v].
template <int CPT, bool SYM>
__device__ __forceinline__ RowRange<SYM> row_plain(const __half* xr, int K, uint4 (&c)[CPT], float* red) {
  RowRange<SYM> range;
#pragma unroll
  for (int v = 0; v < CPT; ++v) {
    const int ch = threadIdx.x + kRowThreads * v;
    c[v] = make_uint4(0u, 0u, 0u, 0u);
    if (ch < K / 8) c[v] = __ldg(reinterpret_cast<const uint4*>(xr) + ch);
  }
#pragma unroll
  for (int v = 0; v < CPT; ++v) {
    if ((int)threadIdx.x + kRowThreads * v >= K / 8) break;
    const __half2* h = reinterpret_cast<const __half2*>(&c[v]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 t = __half22float2(h[e]);
      range.add(t.x, t.y);
    }
  }
  row_block_range(range, red);
  return range;
}

__device__ __forceinline__ void row_get8(const uint4& c, float (&v)[8]) {
  const __half2* h = reinterpret_cast<const __half2*>(&c);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 t = __half22float2(h[e]);
    v[2 * e] = t.x, v[2 * e + 1] = t.y;
  }
}

// Runs f with the compile-time chunk count (2, 4, 8 or 16) that holds a plain
// row of K <= 32768 elements.
template <typename F>
cudaError_t with_row_chunks(int64_t K, F f) {
  const int64_t n = (K / 8 + kRowThreads - 1) / kRowThreads;
  if (n <= 2) return f(std::integral_constant<int, 2>{});
  if (n <= 4) return f(std::integral_constant<int, 4>{});
  if (n <= 8) return f(std::integral_constant<int, 8>{});
  return f(std::integral_constant<int, 16>{});
}

}  // namespace spinq
