// rotate_quant_kv.cu -- R3 on Q and K over head_dim followed by the 4-bit
// asymmetric KV-cache quantizer (Sec. 3.1 R3; Eq. 1; appendix "Quantization
// choice").  V is quantized without rotation (R2 merged into W_v / W_o).
//
// Work unit: one warp, 8 rows of D elements (D = 64 or 128) of one tensor.
// A quad of lanes (g = lane/4 picks the row, c = lane%4) owns one row; lane c
// loads the 8*V consecutive elements [8Vc, 8Vc + 8V) as V 16-byte chunks
// (V = D/32).  Element index bits: e (3 bits, inside a chunk), v (log2 V
// bits, chunk within the lane), c (2 bits, the lane in the quad).
//
// Stage 1 runs on the tensor core, on the raw fp16 input: one m16n8k16 MMA
// per chunk with B = the 16-point Sylvester matrix contracts the 4 bits
// {e0, e2, c0, c1} (k = 2c + e0 + 8 e2); the two A rows g and g+8 carry e1 = 0
// and e1 = 1.  The outputs land in the lane that supplied the inputs, at the
// same element positions, already in fp32 (entries are +-1, so the products
// are exact and the sums are fp32 sums of 16 fp16 values).  The remaining
// bits (e1 and v) are radix-2 butterflies inside the lane.  For V the same
// MMA with B = I16 only widens fp16 to fp32 (exactly).
//
// Eq. 1 on the unnormalised rotated row: the codes do not depend on the
// 1/sqrt(D) factor, which is applied to alpha and beta (and to Q's output).
#include <cuda_fp16.h>
#include <float.h>

#include "launch_util.h"
#include "spinq_device.cuh"
#include "spinq_internal.h"

namespace spinq {
namespace {

constexpr int kWarps = 8;

// RoPE kernel: warps per SM (registers and shared memory allow 16).
constexpr int kRopeWarpsPerSm = 16;
// Row stages of a warp's copy ring (4 KB): two steps of 2 KB, four of 1 KB.
// Measured at 8 x 4096 tokens: D = 128 with 2 / 3 / 4 stages 128 / 132 / 134 us,
// D = 64 with 2 / 3 / 4 stages 111 / 98 / 98 us.
constexpr int rope_stages(int D) { return D == 128 ? 2 : 4; }

__device__ __forceinline__ uint32_t h16_pair(int k0, int k1, int n, bool hadamard) {
  float v0, v1;
  if (hadamard) {
    v0 = (__popc(k0 & n) & 1) ? -1.f : 1.f;
    v1 = (__popc(k1 & n) & 1) ? -1.f : 1.f;
  } else {
    v0 = k0 == n ? 1.f : 0.f;
    v1 = k1 == n ? 1.f : 0.f;
  }
  return pack_half2_bits(v0, v1);
}

// B fragments of a lane for the MMA's n-tiles 0 (n = g) and 1 (n = g + 8):
// the 16-point Hadamard matrix and the identity.
struct BFrags {
  uint32_t h[2][2], i[2][2];
  __device__ __forceinline__ BFrags(int g, int c) {
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const int n = g + 8 * nt;
      h[nt][0] = h16_pair(2 * c, 2 * c + 1, n, true);
      h[nt][1] = h16_pair(2 * c + 8, 2 * c + 9, n, true);
      i[nt][0] = h16_pair(2 * c, 2 * c + 1, n, false);
      i[nt][1] = h16_pair(2 * c + 8, 2 * c + 9, n, false);
    }
  }
};

// Rotation (Q, K) and output of one row per quad: KIND 0 = Q, 1 = K, 2 = V;
// `in` the lane's 16-byte chunks of the row (fp16, after RoPE).  Works on
// packed pairs of neighbouring elements.
template <int D, bool CLAMP, int KIND>
__device__ __forceinline__ void finish_row(const KVArgs& a, const BFrags& B, int64_t row, bool valid, int c,
                                           const uint4 (&in)[D / 32]) {
  constexpr int V = D / 32;
  F2 y[V][4];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    // the chunk's words are the A fragment as they are: k = e0 + 2c + 8 e2,
    // row g + 8 e1 (no register moves), so the MMA contracts {e0, e2, c}
    const uint32_t A[4] = {in[v].x, in[v].y, in[v].z, in[v].w};
    if constexpr (KIND == 2) {
      mma_16816_f16_f32_pairs(y[v][0], y[v][1], A, B.i[0][0], B.i[0][1]);
      mma_16816_f16_f32_pairs(y[v][2], y[v][3], A, B.i[1][0], B.i[1][1]);
    } else {
      mma_16816_f16_f32_pairs(y[v][0], y[v][1], A, B.h[0][0], B.h[0][1]);
      mma_16816_f16_f32_pairs(y[v][2], y[v][3], A, B.h[1][0], B.h[1][1]);
    }
  }

  if constexpr (KIND != 2) {
#pragma unroll
    for (int v = 0; v < V; ++v) {   // e1, the bit the MMA leaves
      f2_bfly(y[v][0], y[v][1]);
      f2_bfly(y[v][2], y[v][3]);
    }
#pragma unroll
    for (int bit = 1; bit < V; bit <<= 1)
#pragma unroll
      for (int v = 0; v < V; ++v)
        if (!(v & bit)) {
#pragma unroll
          for (int e = 0; e < 4; ++e) f2_bfly(y[v][e], y[v | bit][e]);
        }
  }

  if constexpr (KIND == 0) {
    if (valid) {
      uint4* q = reinterpret_cast<uint4*>(reinterpret_cast<__half*>(a.q_out) + row * D) + c * V;
      const F2 norm = f2_make(a.norm, a.norm);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float lo, hi;
          f2_split(f2_mul(y[v][e], norm), lo, hi);
          o[e] = pack_half2_bits(lo, hi);
        }
        q[v] = make_uint4(o[0], o[1], o[2], o[3]);
      }
    }
  } else {
  // asymmetric Eq. 1 over the row (quad reduction)
  float hi = -FLT_MAX, lo = FLT_MAX;
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float x0, x1;
      f2_split(y[v][e], x0, x1);
      asm("max.f32 %0, %0, %1, %2;" : "+f"(hi) : "f"(x0), "f"(x1));
      asm("min.f32 %0, %0, %1, %2;" : "+f"(lo) : "f"(x0), "f"(x1));
    }
  hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, 1));
  hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, 2));
  lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, 1));
  lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, 2));
  const float h2 = a.clip * hi, l2 = a.clip * lo;
  const float inv = h2 > l2 ? 15.f / (h2 - l2) : 0.f;
  const float off = -l2 * inv;
  const F2 inv2 = f2_make(inv, inv), off2 = f2_make(off, off), magic2 = f2_make(kRoundMagic, kRoundMagic);
  uint32_t words[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    uint32_t b[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      F2 t = f2_fma(y[v][e], inv2, off2);
      float t0, t1;
      if (CLAMP) {
        f2_split(t, t0, t1);
        t = f2_make(fminf(fmaxf(t0, 0.f), 15.f), fminf(fmaxf(t1, 0.f), 15.f));
      }
      f2_split(f2_add(t, magic2), t0, t1);
      b[2 * e] = __float_as_uint(t0);
      b[2 * e + 1] = __float_as_uint(t1);
    }
    words[v] = pack8_nibbles(b);
  }
  if (valid) {
    const float nrm = KIND == 1 ? a.norm : 1.f;
    uint8_t* codes = KIND == 1 ? a.k_codes : a.v_codes;
    uint32_t* dst = reinterpret_cast<uint32_t*>(codes + row * (D / 2)) + c * V;
    if (V == 4) {
      *reinterpret_cast<uint4*>(dst) = make_uint4(words[0], words[1], words[2 % V], words[3 % V]);
    } else {
      *reinterpret_cast<uint2*>(dst) = make_uint2(words[0], words[1 % V]);
    }
    if (c == 0) {
      (KIND == 1 ? a.k_scale : a.v_scale)[row] = (h2 - l2) / 15.f * nrm;
      (KIND == 1 ? a.k_zero : a.v_zero)[row] = l2 * nrm;
    }
  }
  }
}

// Without RoPE: a warp takes 8 consecutive rows of one tensor at a time.
// Bound by HBM: 8 x 4096 tokens of 32 + 8 + 8 heads (709 MB) 114 us, 0.92 of the
// copy rate.
template <int D, bool CLAMP>
__global__ void __launch_bounds__(kWarps * 32, 4) rotate_quant_kv_kernel(KVArgs a) {
  constexpr int V = D / 32;  // 16-byte chunks per lane
  const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int warp = threadIdx.x >> 5;
  const BFrags B(g, c);
  pdl_wait();
  pdl_trigger();
  const int64_t gq = (a.rows_q + 7) / 8, gk = (a.rows_kv + 7) / 8;
  const int64_t total = gq + 2 * gk;
  const int64_t stride = (int64_t)gridDim.x * kWarps;
  for (int64_t G = (int64_t)blockIdx.x * kWarps + warp; G < total; G += stride) {
    const int kind = G < gq ? 0 : G < gq + gk ? 1 : 2;
    const int64_t row = (kind == 0 ? G : kind == 1 ? G - gq : G - gq - gk) * 8 + g;
    const bool valid = row < (kind == 0 ? a.rows_q : a.rows_kv);
    const __half* src = reinterpret_cast<const __half*>(kind == 0 ? a.q_in : kind == 1 ? a.k_in : a.v_in);
    const uint4* p = reinterpret_cast<const uint4*>(src + row * D) + c * V;
    uint4 in[V];
#pragma unroll
    for (int v = 0; v < V; ++v) in[v] = valid ? __ldg(p + v) : make_uint4(0, 0, 0, 0);
    if (kind == 0) {
      finish_row<D, CLAMP, 0>(a, B, row, valid, c, in);
    } else if (kind == 1) {
      finish_row<D, CLAMP, 1>(a, B, row, valid, c, in);
    } else {
      finish_row<D, CLAMP, 2>(a, B, row, valid, c, in);
    }
  }
}

// ---------------------------------------------------------------------------
// With RoPE ahead of R3.  A warp takes 8 consecutive tokens (lane group g its
// token t0 + g) and walks a range of heads of Q, K and V, so that a token's
// (cos, sin) row is fetched once for all of them: it lies in the warp's own
// shared memory, where the lanes' 16-byte reads are free of bank conflicts.
// The rows stream through a ring of cp.async stages, one head of 8 tokens each.
//
// What bounds it: issue slots (55 % active) next to HBM.  With 8 rows of one
// tensor per step (the layout above) every row read its 512-byte table row
// again through L1 and divided its row number by the head count: 664 warp
// instructions per 8 rows and 6 of 9 stall cycles on loads (ncu); now 390, and
// the partner's half comes from the staged row instead of 16 shuffles.
// 8 x 4096 tokens of 32 + 8 + 8 heads (D = 128): 187 -> 128 us (0.82 of the copy
// rate); 48 + 12 + 12 heads of 64: 128 -> 98 us; 77 tokens: 3.5 -> 2.7 us.
// ---------------------------------------------------------------------------
template <int D>
struct RopeTable {
  // the table rows of 8 tokens: D/2 (cos, sin) pairs each, the second half and
  // every next token skewed by 16 and 32 bytes
  static constexpr int HALF = D / 4 * 8 + 16;
  static constexpr int ROW = 2 * HALF;
  static constexpr int WARP = 8 * ROW;
};

struct RopePlan {
  int64_t tokens;   // B * S
  int64_t items;    // token blocks * parts
  int parts;        // head ranges per token block
  int heads;        // heads per range (of Hq + 2 Hkv)
};

__device__ __forceinline__ void copy_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}

// Where a warp's copies (and, NST - 1 steps later, its arithmetic)
// stand: head h of [.., h1) for the 8 tokens from tok of `item`.
struct RopeCursor {
  int64_t item, tok;
  int h, h1;
  __device__ __forceinline__ void open(const RopePlan& p, int total) {
    const int64_t tb = item / p.parts;
    h = (int)(item - tb * p.parts) * p.heads;
    h1 = min(h + p.heads, total);
    tok = tb * 8;
  }
};

// XOR on the chunk's two low bits (see the stage layout): for lanes (g, c) with
// chunks (D / 32) c + v the 8 lanes of a quarter warp fall in 8 bank groups.
template <int D>
__device__ __forceinline__ int rope_swizzle(int r, int ch) {
  return D == 128 ? (ch >> 3) | ((r & 1) << 1) : (r >> 0) & 1;
}

// W: warps per CTA.
template <int D, bool CLAMP, int W>
__global__ void __launch_bounds__(W * 32, kRopeWarpsPerSm / W)
    rope_rotate_quant_kv_kernel(KVArgs a, RopePlan plan) {
  constexpr int V = D / 32, NST = rope_stages(D);
  using Tab = RopeTable<D>;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);   // uniform for the compiler too
  const BFrags B(g, c);
  const int Hq = (int)a.Hq, Hkv = (int)a.Hkv, total = Hq + 2 * Hkv;
  unsigned char* tab = smem + warp * (Tab::WARP + NST * D * 16) + g * Tab::ROW;
  const unsigned char* tl = tab + (c & 1) * Tab::HALF;
  // A stage holds the 8 rows of a step (CPR 16-byte chunks each, chunk ch of
  // row r at ch ^ rope_swizzle): the copies take whole rows, two or four per
  // instruction, the reads 4 lanes' pieces of 8 rows, without bank conflicts.
  constexpr int CPR = D / 8, STAGE = 8 * CPR * 16;
  const uint32_t ring = smem_u32(smem + warp * (Tab::WARP + NST * STAGE) + Tab::WARP);
  const int lr = lane / CPR, lc = lane % CPR;   // row (of 32 / CPR) and chunk of the lane's copies
  // the partner's value enters with sign -1 in the first half and +1 in the
  // second: y = x cos + (-+x') sin, the sign flipped on its fp16 bits
  const uint32_t nsign = c < 2 ? 0x80008000u : 0u;
  const int64_t stride = (int64_t)gridDim.x * W;
  pdl_wait();
  pdl_trigger();

  RopeCursor ld, cur;   // the copies' and the arithmetic's place
  ld.item = cur.item = (int64_t)blockIdx.x * W + warp;
  if (cur.item >= plan.items) return;
  ld.open(plan, total);
  cur.open(plan, total);
  int ls = 0, cs = 0;   // their stages
  auto issue = [&]() {
    if (ld.item < plan.items) {
      const int h = ld.h;
      const __half* src = reinterpret_cast<const __half*>(h < Hq ? a.q_in : h < Hq + Hkv ? a.k_in : a.v_in);
      const int H = h < Hq ? Hq : Hkv, hh = h < Hq ? h : h < Hq + Hkv ? h - Hq : h - Hq - Hkv;
      const uint32_t dst = ring + ls * STAGE;
#pragma unroll
      for (int k = 0; k < 8 * CPR / 32; ++k) {
        const int r = lr + 32 / CPR * k;
        const int64_t tok = min(ld.tok + r, plan.tokens - 1);
        copy_async16(dst + 16 * (r * CPR + (lc ^ rope_swizzle<D>(r, lc))), src + (tok * H + hh) * D + 8 * lc);
      }
      if (++ld.h == ld.h1) {
        ld.item += stride;
        if (ld.item < plan.items) ld.open(plan, total);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");   // an empty group past the end keeps the count uniform
    ls = ls + 1 == NST ? 0 : ls + 1;
  };
#pragma unroll
  for (int s = 0; s < NST - 1; ++s) issue();

  while (true) {
    const bool valid = cur.tok + g < plan.tokens;
    const int64_t tok = valid ? cur.tok + g : plan.tokens - 1;   // the quad's token
    if (cur.h < Hq + Hkv) {
      // this quad's token: D / 4 chunks of 16 bytes (two pairs)
      int64_t pos = a.positions[tok];
      pos = pos < 0 ? 0 : (pos >= a.max_pos ? a.max_pos - 1 : pos);
      const float4* src = reinterpret_cast<const float4*>(a.cos_sin + pos * D);
      float4 t[D / 16];
#pragma unroll
      for (int k = 0; k < D / 16; ++k) t[k] = __ldg(src + c + 4 * k);
      __syncwarp();   // the last item's reads are done
#pragma unroll
      for (int k = 0; k < D / 16; ++k) {
        const int ch = c + 4 * k;
        *reinterpret_cast<float4*>(tab + 16 * ch + (ch >= D / 8 ? 16 : 0)) = t[k];
      }
      __syncwarp();
    }
#pragma unroll 1
    for (; cur.h < cur.h1; ++cur.h) {
      issue();
      asm volatile("cp.async.wait_group %0;\n" ::"n"(NST - 1) : "memory");
      __syncwarp();   // every lane's copies have landed
      const uint32_t st = ring + cs * STAGE + 16 * g * CPR;
      auto chunk = [&](int ch) { return lds128(st + 16 * (ch ^ rope_swizzle<D>(g, ch))); };
      uint4 in[V];
#pragma unroll
      for (int v = 0; v < V; ++v) in[v] = chunk(V * c + v);
      if (cur.h >= Hq + Hkv) {
        finish_row<D, CLAMP, 2>(a, B, tok * Hkv + (cur.h - Hq - Hkv), valid, c, in);
        cs = cs + 1 == NST ? 0 : cs + 1;
        __syncwarp();   // the stage has been read
        continue;
      }
      // Rotary embedding (rotate-half form), in fp32 from the caller's
      // (cos, sin) table, rounded back to fp16 like the model's activations:
      // y_i = x_i cos - x_{i+D/2} sin and y_{i+D/2} = x_i sin + x_{i+D/2} cos.
      // The partner i +- D/2 is read from the stage (chunks of lane c ^ 2);
      // both products of an element are one packed multiplication, the pair
      // (x, -+x') times (cos, sin).
#pragma unroll
      for (int v = 0; v < V; ++v) {
        uint32_t w[4] = {in[v].x, in[v].y, in[v].z, in[v].w};
        const uint4 pv = chunk(V * (c ^ 2) + v);
        const uint32_t pws[4] = {pv.x, pv.y, pv.z, pv.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t pw = pws[j] ^ nsign;
          const float4 t = *reinterpret_cast<const float4*>(tl + 8 * (8 * v + 2 * j));
          const float2 x = __half22float2(*reinterpret_cast<const __half2*>(&w[j]));
          const float2 o = __half22float2(*reinterpret_cast<const __half2*>(&pw));
          float p0, p1, q0, q1;
          f2_split(f2_mul(f2_make(x.x, o.x), f2_make(t.x, t.y)), p0, p1);
          f2_split(f2_mul(f2_make(x.y, o.y), f2_make(t.z, t.w)), q0, q1);
          w[j] = pack_half2_bits(__fadd_rn(p0, p1), __fadd_rn(q0, q1));
        }
        in[v] = make_uint4(w[0], w[1], w[2], w[3]);
      }
      cs = cs + 1 == NST ? 0 : cs + 1;
      __syncwarp();   // the stage has been read
      if (cur.h < Hq) {
        finish_row<D, CLAMP, 0>(a, B, tok * Hq + cur.h, valid, c, in);
      } else {
        finish_row<D, CLAMP, 1>(a, B, tok * Hkv + (cur.h - Hq), valid, c, in);
      }
    }
    cur.item += stride;
    if (cur.item >= plan.items) break;
    cur.open(plan, total);
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

template <int D, bool CLAMP>
cudaError_t launch_plain(const KVArgs& a, cudaStream_t stream) {
  const int64_t groups = (a.rows_q + 7) / 8 + 2 * ((a.rows_kv + 7) / 8);
  const int sms = device_sm_count();
  int64_t blocks = (groups + kWarps - 1) / kWarps;
  const int64_t cap = (int64_t)sms * 16;  // persistent-style cap: 16 blocks of 8 warps per SM
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  const cudaError_t e =
      launch_pdl(rotate_quant_kv_kernel<D, CLAMP>, dim3((unsigned)blocks), dim3(kWarps * 32), 0, stream, 1, a);
  return e;
}

// Head ranges for `tokens`: enough items for every resident warp, ranges long
// enough that fetching the table (about one head's time) is shared, and as
// little of a last partial wave as possible: the number of waves w that
// minimises w * (heads per range + 1).
RopePlan plan_rope(int64_t tokens, int total, int64_t warps) {
  const int64_t blocks = (tokens + 7) / 8;
  RopePlan best{tokens, blocks, 1, total};
  int64_t best_cost = INT64_MAX;
  for (int64_t w = 1; w <= 64; ++w) {
    int64_t parts = warps * w / blocks;
    if (parts < 1) continue;
    if (parts > total) parts = total;
    const int heads = (int)((total + parts - 1) / parts);
    if (w * (heads + 1) < best_cost) {
      best_cost = w * (heads + 1);
      best.heads = heads;
      best.parts = (total + heads - 1) / heads;
      best.items = blocks * best.parts;
    }
    if (parts == total) break;
  }
  if (best_cost == INT64_MAX) {   // more token blocks than 64 waves of warps
    best.heads = total;
    best.parts = 1;
    best.items = blocks;
  }
  return best;
}

template <int D, bool CLAMP, int W>
cudaError_t launch_rope_w(const KVArgs& a, const RopePlan& plan, cudaStream_t stream) {
  auto kern = rope_rotate_quant_kv_kernel<D, CLAMP, W>;
  const size_t smem = W * (RopeTable<D>::WARP + rope_stages(D) * D * 16);
  int per_sm = 0;
  cudaError_t e = prepare_launch(kern, W * 32, smem, &per_sm);
  if (e != cudaSuccess) return e;
  int64_t blocks = (plan.items + W - 1) / W;
  const int64_t cap = (int64_t)device_sm_count() * per_sm;
  if (blocks > cap) blocks = cap;
  e = launch_pdl(kern, dim3((unsigned)blocks), dim3(W * 32), smem, stream, 1, a, plan);
  return e;
}

// CTAs of 8 warps where every resident warp has work (2048 tokens of 48 heads:
// 13.4 us against 14.1 with 4 warps, 8 x 4096: 128 against 132), else of 4, so
// that the few items spread over more SMs (77 tokens: 2.7 against 3.3 us).
template <int D, bool CLAMP>
cudaError_t launch_rope(const KVArgs& a, cudaStream_t stream) {
  const int64_t tokens = a.Hq > 0 ? a.rows_q / a.Hq : a.rows_kv / a.Hkv;
  const int total = (int)(a.Hq + 2 * a.Hkv);
  const int64_t warps = (int64_t)device_sm_count() * kRopeWarpsPerSm;
  const RopePlan plan = plan_rope(tokens, total, warps);
  return (tokens + 7) / 8 * total >= warps ? launch_rope_w<D, CLAMP, 8>(a, plan, stream)
                                           : launch_rope_w<D, CLAMP, 4>(a, plan, stream);
}

template <int D>
cudaError_t launch_d(const KVArgs& a, cudaStream_t stream) {
  const bool clamp = a.clip < 1.0f;
  if (a.positions) return clamp ? launch_rope<D, true>(a, stream) : launch_rope<D, false>(a, stream);
  return clamp ? launch_plain<D, true>(a, stream) : launch_plain<D, false>(a, stream);
}

}  // namespace

cudaError_t launch_rotate_quant_kv(const KVArgs& a, cudaStream_t stream) {
  if (a.rows_q == 0 && a.rows_kv == 0) return cudaSuccess;
  if (a.D == 128) return launch_d<128>(a, stream);
  if (a.D == 64) return launch_d<64>(a, stream);
  return cudaErrorInvalidValue;
}

}  // namespace spinq
