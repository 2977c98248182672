// cayley_step.cu -- spinq_cayley_step: one Cayley SGD update of a batch of
// n x n rotations (Sec. 3.2), n in {16, 32, 64, 128} (R2 is head_dim x
// head_dim, one per layer), one CTA or one cluster of CTAs per rotation.
//
//   G_hat = G R^T - 1/2 R R^T G R^T,   Y = G_hat - G_hat^T,
//   R' = (I - a/2 Y)^-1 (I + a/2 Y) R  by the fixed-point iteration
//   R'_0 = R + a Y R,  R'_{k+1} = R + (a/2) Y (R + R'_k).
//
// G is the negative of the loss gradient the caller passes (the printed update
// with G = +grad climbs the loss; the cited Cayley SGD forms G_hat from the
// negative gradient).  With D_k = R'_k - R the iteration reads
// D_0 = M = a Y R, D_{k+1} = M + (a/2) Y D_k, and R' = R + D_iters: M stays in
// registers, so three n x n fp32 buffers in shared memory suffice
// (3 * 128 * 132 * 4 = 203 KB at n = 128):
//
//   buf0 = R^T, buf1 = -grad         (loaded)
//   buf2 = A = G R^T                 [G buf1, R^T buf0]
//   buf1 = C = R^T A                 [R^T buf0, A buf2]
//   buf2 = G_hat = A - 1/2 R C       [R = buf0 read transposed, C buf1]
//   buf1 = Y = G_hat - G_hat^T;  buf0 transposed in place to R
//   M = a Y R (registers), buf2 = D_0 = M
//   D_{k+1} = M + (a/2) Y D_k        ping-pong between buf0 and buf2
//   R_out = R + D_iters              (R re-read from global memory)
//
// Thread (rg, cg) owns rows i0 = TR rg .. and columns 4 cg .. 4 cg + 3 and
// N/2 + 4 cg .. + 3 of every product (so that the 16-byte operand loads of a
// quarter warp are contiguous); the products run on packed fp32 pairs
// (fma.rn.f32x2), the column pairs of a row in one register pair.
#include <cuda_runtime.h>

#include <atomic>

#include "launch_util.h"
#include "spinq_device.cuh"
#include "spinq_internal.h"

namespace spinq {
namespace {

template <int N>
struct CayleyShape {
  static_assert(N == 16 || N == 128, "the other sizes take cayley_cluster_kernel");
  static constexpr int TR = N == 128 ? 4 : 1;                   // rows per thread
  static constexpr int CG = N / 8;                              // column groups of 8
  static constexpr int RG = N / TR;                             // row groups
  static constexpr int THREADS = CG * RG;
  static constexpr int S = N + 4;                               // row stride in floats
  static constexpr int BUF = N * S;
  static constexpr int BYTES = 3 * BUF * 4;
  static_assert(THREADS <= 1024 && THREADS % 32 == 0, "block shape");
};

template <int N>
using Acc = F2[CayleyShape<N>::TR][4];

// acc[r][c] += sum_k X(i0 + r, k) * B[k][col 2c, 2c + 1 of the thread], with
// X(i, k) = X[i][k], or X[k][i] when XT.
template <int N, bool XT>
__device__ __forceinline__ void mm_acc(const float* X, const float* B, int i0, int ja, int jb, Acc<N>& acc) {
  using S = CayleyShape<N>;
#pragma unroll 1
  for (int k0 = 0; k0 < N; k0 += 4) {
    float xv[4][S::TR];   // four k at a time: one 16-byte load per row
    if (!XT) {
#pragma unroll
      for (int r = 0; r < S::TR; ++r) {
        const float4 t = *reinterpret_cast<const float4*>(X + (i0 + r) * S::S + k0);
        xv[0][r] = t.x, xv[1][r] = t.y, xv[2][r] = t.z, xv[3][r] = t.w;
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = k0 + q;
      if (XT) {
        if constexpr (S::TR == 4) {
          const float4 t = *reinterpret_cast<const float4*>(X + k * S::S + i0);
          xv[q][0] = t.x, xv[q][1] = t.y, xv[q][2] = t.z, xv[q][3] = t.w;
        } else {
          xv[q][0] = X[k * S::S + i0];
        }
      }
      const float4 b0 = *reinterpret_cast<const float4*>(B + k * S::S + ja);
      const float4 b1 = *reinterpret_cast<const float4*>(B + k * S::S + jb);
      const F2 bp[4] = {f2_make(b0.x, b0.y), f2_make(b0.z, b0.w), f2_make(b1.x, b1.y), f2_make(b1.z, b1.w)};
#pragma unroll
      for (int r = 0; r < S::TR; ++r) {
        const F2 xx = f2_make(xv[q][r], xv[q][r]);
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = f2_fma(xx, bp[c], acc[r][c]);
      }
    }
  }
}

template <int N>
__device__ __forceinline__ void acc_zero(Acc<N>& acc) {
#pragma unroll
  for (int r = 0; r < CayleyShape<N>::TR; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = f2_make(0.f, 0.f);
}

template <int N>
__device__ __forceinline__ void tile_store(float* dst, int i0, int ja, int jb, const Acc<N>& acc) {
  using S = CayleyShape<N>;
#pragma unroll
  for (int r = 0; r < S::TR; ++r) {
    float v[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) f2_split(acc[r][c], v[2 * c], v[2 * c + 1]);
    *reinterpret_cast<float4*>(dst + (i0 + r) * S::S + ja) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(dst + (i0 + r) * S::S + jb) = make_float4(v[4], v[5], v[6], v[7]);
  }
}

template <int N>
__global__ void __launch_bounds__(CayleyShape<N>::THREADS, 1)
    cayley_step_kernel(const float* __restrict__ R, const float* __restrict__ grad, float alpha, int iters,
                       float* R_out, float* Y_out) {
  using S = CayleyShape<N>;
  extern __shared__ __align__(16) float sm[];
  float* buf0 = sm;
  float* buf1 = sm + S::BUF;
  float* buf2 = sm + 2 * S::BUF;
  const int tid = threadIdx.x;
  const int cg = tid % S::CG, rg = tid / S::CG;
  // columns 4 cg .. + 3 and N/2 + 4 cg .. + 3: the 16-byte operand loads of
  // a quarter warp (cg = 0..7, one rg) cover 128 contiguous bytes
  const int i0 = rg * S::TR, ja = 4 * cg, jb = N / 2 + 4 * cg;
  const size_t base = (size_t)blockIdx.x * N * N;
  pdl_wait();
  pdl_trigger();

  // buf0 = R^T, buf1 = G = -grad
#pragma unroll
  for (int r = 0; r < S::TR; ++r) {
    const float4 a0 = *reinterpret_cast<const float4*>(R + base + (size_t)(i0 + r) * N + ja);
    const float4 a1 = *reinterpret_cast<const float4*>(R + base + (size_t)(i0 + r) * N + jb);
    const float v[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
    for (int c = 0; c < 8; ++c) buf0[(c < 4 ? ja + c : jb + c - 4) * S::S + i0 + r] = v[c];
    const float4 g0 = *reinterpret_cast<const float4*>(grad + base + (size_t)(i0 + r) * N + ja);
    const float4 g1 = *reinterpret_cast<const float4*>(grad + base + (size_t)(i0 + r) * N + jb);
    *reinterpret_cast<float4*>(buf1 + (i0 + r) * S::S + ja) = make_float4(-g0.x, -g0.y, -g0.z, -g0.w);
    *reinterpret_cast<float4*>(buf1 + (i0 + r) * S::S + jb) = make_float4(-g1.x, -g1.y, -g1.z, -g1.w);
  }
  __syncthreads();

  Acc<N> acc;
  // A = G R^T -> buf2
  acc_zero<N>(acc);
  mm_acc<N, false>(buf1, buf0, i0, ja, jb, acc);
  tile_store<N>(buf2, i0, ja, jb, acc);
  __syncthreads();
  // C = R^T A -> buf1
  acc_zero<N>(acc);
  mm_acc<N, false>(buf0, buf2, i0, ja, jb, acc);
  tile_store<N>(buf1, i0, ja, jb, acc);
  __syncthreads();
  // G_hat = A - 1/2 R C -> buf2
  acc_zero<N>(acc);
  mm_acc<N, true>(buf0, buf1, i0, ja, jb, acc);
  const F2 mhalf = f2_make(-0.5f, -0.5f);
#pragma unroll
  for (int r = 0; r < S::TR; ++r) {
    const float* at = buf2 + (i0 + r) * S::S;   // this thread's own tile of A
    const float4 t0 = *reinterpret_cast<const float4*>(at + ja);
    const float4 t1 = *reinterpret_cast<const float4*>(at + jb);
    const F2 av[4] = {f2_make(t0.x, t0.y), f2_make(t0.z, t0.w), f2_make(t1.x, t1.y), f2_make(t1.z, t1.w)};
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = f2_fma(acc[r][c], mhalf, av[c]);
  }
  tile_store<N>(buf2, i0, ja, jb, acc);
  __syncthreads();
  // Y = G_hat - G_hat^T -> buf1 (and Y_out); buf0 transposed in place to R
#pragma unroll
  for (int r = 0; r < S::TR; ++r) {
    const int i = i0 + r;
    float y[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int j = c < 4 ? ja + c : jb + c - 4;
      y[c] = buf2[i * S::S + j] - buf2[j * S::S + i];
      buf1[i * S::S + j] = y[c];
      if (i < j) {
        const float t = buf0[i * S::S + j];
        buf0[i * S::S + j] = buf0[j * S::S + i];
        buf0[j * S::S + i] = t;
      }
    }
    if (Y_out) {
      *reinterpret_cast<float4*>(Y_out + base + (size_t)i * N + ja) = make_float4(y[0], y[1], y[2], y[3]);
      *reinterpret_cast<float4*>(Y_out + base + (size_t)i * N + jb) = make_float4(y[4], y[5], y[6], y[7]);
    }
  }
  __syncthreads();
  // M = a Y R (registers), D_0 = M -> buf2
  Acc<N> m;
  acc_zero<N>(acc);
  mm_acc<N, false>(buf1, buf0, i0, ja, jb, acc);
  const F2 a2 = f2_make(alpha, alpha), h2 = f2_make(0.5f * alpha, 0.5f * alpha), zero2 = f2_make(0.f, 0.f);
#pragma unroll
  for (int r = 0; r < S::TR; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) m[r][c] = f2_fma(acc[r][c], a2, zero2);
  if (iters > 0) tile_store<N>(buf2, i0, ja, jb, m);
  // D_{k+1} = M + (a/2) Y D_k, left in acc (D_0 = M when iters = 0)
  float* cur = buf2;
  float* nxt = buf0;
  for (int k = 0; k < iters; ++k) {
    __syncthreads();
    acc_zero<N>(acc);
    mm_acc<N, false>(buf1, cur, i0, ja, jb, acc);
#pragma unroll
    for (int r = 0; r < S::TR; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[r][c] = f2_fma(acc[r][c], h2, m[r][c]);
    if (k + 1 < iters) tile_store<N>(nxt, i0, ja, jb, acc);
    float* t = cur;
    cur = nxt;
    nxt = t;
  }
  if (iters == 0) {
#pragma unroll
    for (int r = 0; r < S::TR; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[r][c] = m[r][c];
  }
  // R' = R + D
#pragma unroll
  for (int r = 0; r < S::TR; ++r) {
    const size_t off = base + (size_t)(i0 + r) * N;
    const float4 a0 = *reinterpret_cast<const float4*>(R + off + ja);
    const float4 a1 = *reinterpret_cast<const float4*>(R + off + jb);
    float v[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) f2_split(acc[r][c], v[2 * c], v[2 * c + 1]);
    *reinterpret_cast<float4*>(R_out + off + ja) = make_float4(a0.x + v[0], a0.y + v[1], a0.z + v[2], a0.w + v[3]);
    *reinterpret_cast<float4*>(R_out + off + jb) = make_float4(a1.x + v[4], a1.y + v[5], a1.z + v[6], a1.w + v[7]);
  }
}

// ---------------------------------------------------------------------------
// The same step with a cluster of C CTAs per rotation, for batches that leave
// SMs idle.  CTA r owns the columns J = [r N / C, (r + 1) N / C) of every
// product.  With R and G whole in each CTA, A = G R^T, C = R^T A and
// G_hat = A - 1/2 R C need column slabs only; one exchange through distributed
// shared memory gives every CTA the whole G_hat, hence Y, and the update
// D_{k+1} = M + (a/2) Y D_k is column-local again.  A thread owns 4 rows x 4
// columns.  Each output is the same chain of fused multiply-adds over
// k = 0, 1, .. as in the kernel above, so the results are bit-identical.
//
// What bounds it: the FP32 pipe and, next to it, issue (a product of 128 x 128
// x 32 per CTA is 4096 cycles of FMAs; the operands come as 16-byte loads of
// four k at a time, 8 loads for 64 FMAs).  32 rotations of 128 x 128, two
// iterations: 86 us with one CTA each, 29 us with four (12 us of it FMAs; the
// 16-byte shared-memory loads take about three wavefronts each and set the
// pace, then about 8 us of loads, exchange and transposes).
// ---------------------------------------------------------------------------
template <int N, int C>
struct CayleySlab {
  static constexpr int W = N / C;                 // columns per CTA
  static constexpr int CG = W / 4;                // column groups of 4
  static constexpr int THREADS = (N / 4) * CG;
  static constexpr int S = N + 4;                 // row stride of the whole matrices
  static constexpr int SW = W + 4;                // row stride of the slabs
  static constexpr int FULL = N * S, SLAB = N * SW;
  static constexpr int BYTES = (2 * FULL + 2 * SLAB) * 4;
  static_assert(W % 4 == 0 && THREADS % 32 == 0 && THREADS <= 1024, "block shape");
};

using Acc4 = F2[4][2];   // 4 rows x 2 column pairs

// acc[r][c] += sum_k X(i0 + RS r, k) B[k][j0 + 2c, j0 + 2c + 1], k ascending; X
// is N x N with row stride S (XT: its transpose is stored, RS = 1), B has row
// stride SB.  RS = N / 4 puts the rows of a warp's threads next to each other:
// their 16-byte loads along k fall in different banks (RS = 1 had 2-way
// conflicts).
template <int N, bool XT, int RS, int S, int SB>
__device__ __forceinline__ void slab_mm(const float* X, const float* B, int i0, int j0, Acc4& acc) {
#pragma unroll
  for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = f2_make(0.f, 0.f);
#pragma unroll 2
  for (int k = 0; k < N; k += 4) {
    float x[4][4];   // [row][k]
    float4 b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 t = *reinterpret_cast<const float4*>(XT ? X + (k + q) * S + i0 : X + (i0 + RS * q) * S + k);
      if (XT) {
        x[0][q] = t.x, x[1][q] = t.y, x[2][q] = t.z, x[3][q] = t.w;
      } else {
        x[q][0] = t.x, x[q][1] = t.y, x[q][2] = t.z, x[q][3] = t.w;
      }
      b[q] = *reinterpret_cast<const float4*>(B + (k + q) * SB + j0);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const F2 b0 = f2_make(b[q].x, b[q].y), b1 = f2_make(b[q].z, b[q].w);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const F2 xx = f2_make(x[r][q], x[r][q]);
        acc[r][0] = f2_fma(xx, b0, acc[r][0]);
        acc[r][1] = f2_fma(xx, b1, acc[r][1]);
      }
    }
  }
}

template <int RS, int SB>
__device__ __forceinline__ void slab_store(float* dst, int i0, int j0, const Acc4& acc) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    float4 v;
    f2_split(acc[r][0], v.x, v.y);
    f2_split(acc[r][1], v.z, v.w);
    *reinterpret_cast<float4*>(dst + (i0 + RS * r) * SB + j0) = v;
  }
}

__device__ __forceinline__ void copy_async16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ float4 ld_shared_cluster_v4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];\n"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

template <int N, int C>
__global__ void __launch_bounds__(CayleySlab<N, C>::THREADS, 1)
    cayley_cluster_kernel(const float* R, const float* __restrict__ grad, float alpha, int iters, float* R_out,
                          float* Y_out) {
  using L = CayleySlab<N, C>;
  constexpr int S = L::S, SW = L::SW, W = L::W, T = L::THREADS;
  extern __shared__ __align__(16) float sm[];
  float* bR = sm;               // R, row-major
  float* bG = sm + L::FULL;     // grad, then G_hat, then Y
  float* bP = bG + L::FULL;     // R^T slab, C, the iterates
  float* bQ = bP + L::SLAB;     // A, G_hat slab, the iterates
  const int tid = threadIdx.x;
  const int rank = C > 1 ? (int)cluster_ctarank() : 0;
  const int J0 = rank * W;
  constexpr int RS = N / 4;
  const int i0 = tid / L::CG, j0 = 4 * (tid % L::CG);   // rows i0 + RS r
  const size_t base = (size_t)(blockIdx.x / C) * N * N;
  pdl_wait();
  pdl_trigger();

  // R and grad as they are, every copy in flight at once
#pragma unroll 8
  for (int e = tid; e < N * N / 4; e += T) {
    const int i = e / (N / 4), j = 4 * (e % (N / 4));
    copy_async16(bR + i * S + j, R + base + (size_t)i * N + j);
    copy_async16(bG + i * S + j, grad + base + (size_t)i * N + j);
  }
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  // bP = R^T[:, J], 4 x 4 blocks transposed in registers
  for (int e = tid; e < (N / 4) * (W / 4); e += T) {
    const int k = 4 * (e % (N / 4)), j = 4 * (e / (N / 4));
    float v[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 t = *reinterpret_cast<const float4*>(bR + (J0 + j + q) * S + k);
      v[q][0] = t.x, v[q][1] = t.y, v[q][2] = t.z, v[q][3] = t.w;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      *reinterpret_cast<float4*>(bP + (k + q) * SW + j) = make_float4(v[0][q], v[1][q], v[2][q], v[3][q]);
  }
  __syncthreads();

  Acc4 acc;
  // A = G R^T with G = -grad: the negated product of grad (rounding is
  // symmetric, so the same bits)
  slab_mm<N, false, RS, S, SW>(bG, bP, i0, j0, acc);
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) acc[r][c].u ^= 0x8000000080000000ull;
  slab_store<RS, SW>(bQ, i0, j0, acc);
  __syncthreads();
  slab_mm<N, true, 1, S, SW>(bR, bQ, 4 * i0, j0, acc);    // C = R^T A
  slab_store<1, SW>(bP, 4 * i0, j0, acc);
  __syncthreads();
  slab_mm<N, false, RS, S, SW>(bR, bP, i0, j0, acc);   // G_hat = A - 1/2 R C
  const F2 mhalf = f2_make(-0.5f, -0.5f);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float4 t = *reinterpret_cast<const float4*>(bQ + (i0 + RS * r) * SW + j0);   // this thread's own tile of A
    acc[r][0] = f2_fma(acc[r][0], mhalf, f2_make(t.x, t.y));
    acc[r][1] = f2_fma(acc[r][1], mhalf, f2_make(t.z, t.w));
  }
  slab_store<RS, SW>(bQ, i0, j0, acc);
  // every CTA's slab of G_hat is in place; G (bG) has been read
  if constexpr (C > 1) {
    cluster_sync_all();
  } else {
    __syncthreads();
  }
  // the loads of eight elements in flight together
  constexpr int NG = N * N / 4 / T < 8 ? N * N / 4 / T : 8;
  static_assert(N * N / 4 % (T * NG) == 0, "whole batches of loads");
  for (int e0 = tid; e0 < N * N / 4; e0 += T * NG) {
    float4 v[NG];
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const int e = e0 + q * T, i = e / (N / 4), j = 4 * (e % (N / 4));
      const float* own = bQ + i * SW + j % W;
      if constexpr (C > 1) {
        v[q] = ld_shared_cluster_v4(mapa_shared(smem_u32(own), (uint32_t)(j / W)));
      } else {
        v[q] = *reinterpret_cast<const float4*>(own);
      }
    }
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const int e = e0 + q * T, i = e / (N / 4), j = 4 * (e % (N / 4));
      *reinterpret_cast<float4*>(bG + i * S + j) = v[q];
    }
  }
  // no CTA overwrites its slab or leaves before every CTA has read it
  if constexpr (C > 1) {
    cluster_sync_all();
  } else {
    __syncthreads();
  }
  // Y = G_hat - G_hat^T in place, 4 x 4 blocks (bi, bj) and (bj, bi) together
  constexpr int NB = N / 4;
  for (int e = tid; e < NB * NB; e += T) {
    const int bi = e / NB, bj = e % NB;
    if (bi > bj) continue;
    float u[4][4], l[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 a = *reinterpret_cast<const float4*>(bG + (4 * bi + r) * S + 4 * bj);
      const float4 b = *reinterpret_cast<const float4*>(bG + (4 * bj + r) * S + 4 * bi);
      u[r][0] = a.x, u[r][1] = a.y, u[r][2] = a.z, u[r][3] = a.w;
      l[r][0] = b.x, l[r][1] = b.y, l[r][2] = b.z, l[r][3] = b.w;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      *reinterpret_cast<float4*>(bG + (4 * bi + r) * S + 4 * bj) =
          make_float4(u[r][0] - l[0][r], u[r][1] - l[1][r], u[r][2] - l[2][r], u[r][3] - l[3][r]);
      if (bi != bj)
        *reinterpret_cast<float4*>(bG + (4 * bj + r) * S + 4 * bi) =
            make_float4(l[r][0] - u[0][r], l[r][1] - u[1][r], l[r][2] - u[2][r], l[r][3] - u[3][r]);
    }
  }
  __syncthreads();
  if (Y_out) {   // this CTA's rows J0 .. J0 + W - 1
    for (int e = tid; e < W * N / 4; e += T) {
      const int i = J0 + e / (N / 4), j = 4 * (e % (N / 4));
      *reinterpret_cast<float4*>(Y_out + base + (size_t)i * N + j) = *reinterpret_cast<const float4*>(bG + i * S + j);
    }
  }
  // M = a Y R (registers), D_0 = M
  slab_mm<N, false, RS, S, S>(bG, bR + J0, i0, j0, acc);
  const F2 a2 = f2_make(alpha, alpha), h2 = f2_make(0.5f * alpha, 0.5f * alpha), zero2 = f2_make(0.f, 0.f);
  Acc4 m;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) acc[r][c] = m[r][c] = f2_fma(acc[r][c], a2, zero2);
  float *cur = bP, *nxt = bQ;
  if (iters > 0) slab_store<RS, SW>(cur, i0, j0, m);
  for (int k = 0; k < iters; ++k) {
    __syncthreads();
    slab_mm<N, false, RS, S, SW>(bG, cur, i0, j0, acc);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c) acc[r][c] = f2_fma(acc[r][c], h2, m[r][c]);
    if (k + 1 < iters) slab_store<RS, SW>(nxt, i0, j0, acc);
    float* t = cur;
    cur = nxt;
    nxt = t;
  }
  // R' = R + D
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float4 a = *reinterpret_cast<const float4*>(bR + (i0 + RS * r) * S + J0 + j0);
    float4 d;
    f2_split(acc[r][0], d.x, d.y);
    f2_split(acc[r][1], d.z, d.w);
    *reinterpret_cast<float4*>(R_out + base + (size_t)(i0 + RS * r) * N + J0 + j0) =
        make_float4(a.x + d.x, a.y + d.y, a.z + d.z, a.w + d.w);
  }
}

// (n = 16, and n = 128 for batches that fill the SMs)
template <int N>
cudaError_t launch_cayley_n(const CayleyArgs& a, cudaStream_t stream) {
  using S = CayleyShape<N>;
  auto kern = cayley_step_kernel<N>;
  int per_sm = 0;
  cudaError_t e = prepare_launch(kern, S::THREADS, S::BYTES, &per_sm);
  if (e != cudaSuccess) return e;
  e = launch_pdl(kern, dim3((unsigned)a.batch), dim3(S::THREADS), S::BYTES, stream, 1, a.R, a.grad, a.alpha,
                 a.iters, a.R_out, a.Y_out);
  return e;
}

template <int N, int C>
cudaError_t launch_cayley_cluster(const CayleyArgs& a, cudaStream_t stream) {
  using L = CayleySlab<N, C>;
  auto kern = cayley_cluster_kernel<N, C>;
  int per_sm = 0;
  cudaError_t e = prepare_launch(kern, L::THREADS, L::BYTES, &per_sm);
  if (e != cudaSuccess) return e;
  e = launch_pdl(kern, dim3((unsigned)(a.batch * C)), dim3(L::THREADS), L::BYTES, stream, C, a.R, a.grad, a.alpha,
                 a.iters, a.R_out, a.Y_out);
  return e;
}

// Clusters of this kernel that can be resident at once, asked once per device
// (0 if the device answers with an error).
template <int N, int C>
int64_t max_clusters() {
  using L = CayleySlab<N, C>;
  static std::atomic<int> cache[64];   // clusters + 1; 0: not asked yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int n = cache[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    auto kern = cayley_cluster_kernel<N, C>;
    int per_sm = 0, clusters = 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(L::THREADS);
    cfg.dynamicSmemBytes = L::BYTES;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (prepare_launch(kern, L::THREADS, L::BYTES, &per_sm) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess) {
      cudaGetLastError();
      clusters = 0;
    }
    n = clusters + 1;
    cache[dev].store(n, std::memory_order_relaxed);
  }
  return n - 1;
}

// One rotation of 128 x 128 takes 84 us on one CTA, 47, 29 and 21 us on a
// cluster of 2, 4 and 8 (two iterations); a batch runs in waves of the
// clusters that can be resident.  E.g. 32 rotations: clusters of 4 (29 us), 76:
// of 2 (47 us), from 77 on one CTA each.  64 x 64: 9.7 us on two CTAs against
// 14 us on one, as long as every CTA has an SM of its own.
cudaError_t launch_cayley_128(const CayleyArgs& a, cudaStream_t stream) {
  const int64_t sms = device_sm_count();
  const struct {
    int64_t resident;
    double us;
  } form[4] = {{sms, 84.0}, {max_clusters<128, 2>(), 47.0}, {max_clusters<128, 4>(), 29.0}, {max_clusters<128, 8>(), 21.0}};
  int best = 0;
  double best_us = 0;
  for (int f = 0; f < 4; ++f) {
    if (form[f].resident < 1) continue;
    const double us = (double)((a.batch + form[f].resident - 1) / form[f].resident) * form[f].us;
    if (f == 0 || us < best_us) {
      best = f;
      best_us = us;
    }
  }
  switch (best) {
    case 1: return launch_cayley_cluster<128, 2>(a, stream);
    case 2: return launch_cayley_cluster<128, 4>(a, stream);
    case 3: return launch_cayley_cluster<128, 8>(a, stream);
  }
  return launch_cayley_n<128>(a, stream);
}

}  // namespace

cudaError_t launch_cayley_step(const CayleyArgs& a, cudaStream_t stream) {
  switch (a.n) {
    case 16: return launch_cayley_n<16>(a, stream);
    case 32: return launch_cayley_cluster<32, 1>(a, stream);
    case 64:
      return 2 * a.batch <= device_sm_count() ? launch_cayley_cluster<64, 2>(a, stream)
                                              : launch_cayley_cluster<64, 1>(a, stream);
    case 128: return launch_cayley_128(a, stream);
  }
  return cudaErrorNotSupported;
}

}  // namespace spinq
