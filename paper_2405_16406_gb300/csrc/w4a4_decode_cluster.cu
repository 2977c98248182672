// w4a4_decode_cluster.cu -- W4A4 linear for up to 128 tokens whose K range is
// split over the CTAs of a cluster (see w4a4_gemm.cu for the codes as E4M3
// values, the exactness of the accumulator and the epilogue formula).
//
// The weight tile is the MMA's M side (128 output channels per cluster), the
// tokens its N side (mn = M rounded up to 16); CTA `rank` of a cluster of C
// takes K steps of 128 from rank / C of the range on.  Each leaves its exact
// partial sums S 2^18 - 8 sum u_a in its own shared memory, over the operand
// stages, and after a cluster barrier the CTAs share the tokens: a warp adds
// the C float4s of a token's row over distributed shared memory, takes
// 8 rowsum_n off and writes y.
//
// Warp roles (448 threads, one CTA per SM):
//   warp 0       TMA producer, 8 packed stages of one K step
//   warp 1       TMEM allocation, MMA issue, two operand stages
//   warps 2..5   token scales, then the partial sums
//   warps 6..13  unpack, two groups of four with one operand stage each, in
//                turn; then the partial sums
//
// What bounds it: a CTA's K step (0.42 us at 77 tokens: unpacking 128 weight
// rows and the tokens, 32 KB of shared-memory stores and the barriers between
// the roles; two groups in turn overlap one group's waits with the other's
// work) and about 6 us of start-up, first copies and last sums.  The split-K
// kernel of w4a4_gemm.cu adds its partial sums by atomics in global memory and
// lets the last slice of a tile convert them, 1.8 + 0.089 M us; over the
// cluster that part is one pass over shared memory.  77 tokens, 4096 -> 4096,
// with the quantizer: 23.0 us there, 11.6 here (clusters of 4); 14336 -> 4096:
// 35.1 and 20.3 (30 MB, 4.3 us of HBM).  The row sum correction takes
// w_rowsum instead of counting the weights again, which leaves their unpacking
// to masks and stores.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>

#include "../../include/spinq.h"
#include "launch_util.h"
#include "spinq_device.cuh"
#include "spinq_internal.h"
#include "tensor_map.h"

namespace spinq {
namespace {

constexpr int kThreads = 448;
constexpr int kFirstUnpackWarp = 6;
constexpr int kGroupThreads = 128;
constexpr int NP = 8;   // packed stages (even: a stage always belongs to the same group, which sees each of its phases)
constexpr int kMaxCluster = kDecodeMaxCluster;
constexpr uint64_t kWaitLimitNs = 2000000000ull;
__device__ uint64_t g_wait_ns = kWaitLimitNs;

struct DecodeParams {
  GemmArgs a;
  int* status;
  int mn;        // tokens rounded up to 16
  int ksteps;    // K / 128
  int cluster;   // CTAs per 128 channels
  int tmem_cols;
};

// Shared memory (from a 1024-byte boundary): unpacked weights [2][128][128],
// unpacked tokens [2][mn][128], packed weights [NP][128][64], packed tokens
// [NP][mn][64], barriers and per-token values.  The partial sums [mn][128]
// fp32 lie over the stages.
struct Layout {
  uint32_t ua, pw, pa, bars, misc, rsa, tal, tbp, total;
  __host__ __device__ explicit Layout(int mn) {
    ua = 2 * 16384;
    pw = ua + 2 * mn * 128;
    pa = pw + NP * 8192;
    bars = pa + NP * mn * 64;
    misc = bars + (2 * NP + 8) * 8;   // 2 NP + 7 barriers; tensor-memory address, abort flag, scratch word
    rsa = misc + 16;                      // [2][mn], one per group
    tal = rsa + 2 * mn * 4;
    tbp = tal + mn * 4;
    total = tbp + mn * 4;
  }
};

__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status,
                                         int site) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (globaltimer_ns() - t0 > g_wait_ns) {
      if (status && atomicCAS(status, 0, (int)SPINQ_ETIMEOUT) == 0) atomicExch(status + 1, site);
      *abort_flag = 1;
      return false;
    }
  }
}
// By all lanes of a warp, with one answer for all of them.
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status,
                                          int site) {
  return __all_sync(0xffffffffu, wait_bar(bar, parity, abort_flag, status, site));
}

// 32 packed codes -> 32 unsigned E4M3 bytes, even and odd codes of each byte
__device__ __forceinline__ void unpack16(const uint4 w, uint32_t x, uint4& lo, uint4& hi) {
  uint32_t t;
  t = w.x ^ x; lo.x = t & 0x0F0F0F0Fu; hi.x = (t >> 4) & 0x0F0F0F0Fu;
  t = w.y ^ x; lo.y = t & 0x0F0F0F0Fu; hi.y = (t >> 4) & 0x0F0F0F0Fu;
  t = w.z ^ x; lo.z = t & 0x0F0F0F0Fu; hi.z = (t >> 4) & 0x0F0F0F0Fu;
  t = w.w ^ x; lo.w = t & 0x0F0F0F0Fu; hi.w = (t >> 4) & 0x0F0F0F0Fu;
}

__device__ __forceinline__ float4 ld_cluster_v4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];\n"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
// Barrier of all threads of the cluster that does not ask for converged warps.
__device__ __forceinline__ void cluster_sync_threads() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}

// TA: 16-byte token chunks per unpack thread and K step, at most.
template <int TA, bool ASYM, bool ACC_OUT>
__global__ void __launch_bounds__(kThreads, 1)
    w4a4_decode_cluster_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmA,
                               const DecodeParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int mn = p.mn;
  const Layout L(mn);
  uint64_t* full_p = reinterpret_cast<uint64_t*>(base + L.bars);
  uint64_t* empty_p = full_p + NP;
  uint64_t* full_u = empty_p + NP;
  uint64_t* empty_u = full_u + 2;
  uint64_t* acc_full = empty_u + 2;
  uint64_t* rs_full = acc_full + 1;
  uint64_t* drain = rs_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + L.misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base + L.misc + 4);
  volatile uint32_t* scratch = reinterpret_cast<volatile uint32_t*>(base + L.misc + 8);   // see wait_loaded
  int* rsa = reinterpret_cast<int*>(base + L.rsa);
  float* tal = reinterpret_cast<float*>(base + L.tal);
  float* tbp = reinterpret_cast<float*>(base + L.tbp);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int C = p.cluster, rank = blockIdx.x;   // gridDim.x is the cluster
  const int n0 = blockIdx.y * 128;
  const int k_begin = rank * p.ksteps / C;      // ksteps <= 512
  const int nk = (rank + 1) * p.ksteps / C - k_begin;

  if (tid == 0) {
    for (int i = 0; i < NP; ++i) {
      mbar_init(&full_p[i], 1);
      mbar_init(&empty_p[i], 4);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&full_u[i], 4);
      mbar_init(&empty_u[i], 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(rs_full, 8);
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tmW);
    prefetch_tmap(&tmA);
  }
  // This CTA's slice of the weights (up to 16 K steps) into L2 while the
  // previous kernel finishes: L2 is coherent with its stores and nothing
  // reaches registers or shared memory.
  if (warp >= 2 && warp < 6 && n0 + tid - 64 < p.a.N) {
    const uint8_t* w = p.a.w_codes + (size_t)(n0 + tid - 64) * (size_t)(p.a.K / 2) + k_begin * 64;
    for (int off = 0; off < 64 * nk && off < 1024; off += 128) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(w + off));
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, (uint32_t)p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();
  pdl_trigger();

  int issued = 0;   // copies the producer issued (for the drain after an abort)
  if (warp == 0) {
    if (lane == 0) {
      for (int it = 0; it < nk && !p.a.debug_stall; ++it) {
        const int s = it & (NP - 1);
        if (!wait_bar(&empty_p[s], (uint32_t)(it / NP) & 1u ^ 1u, abort_flag, p.status, 61)) break;
        mbar_arrive_expect_tx(&full_p[s], (uint32_t)(128 + mn) * 64);
        tma_load_2d(base + L.pw + s * 8192, &tmW, &full_p[s], (k_begin + it) * 64, n0);
        tma_load_2d(base + L.pa + s * mn * 64, &tmA, &full_p[s], (k_begin + it) * 64, 0);
        issued = it + 1;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = umma_idesc_e4m3_f32(128, mn);
      for (int it = 0; it < nk; ++it) {
        const int su = it & 1;
        if (!wait_bar(&full_u[su], (uint32_t)(it >> 1) & 1u, abort_flag, p.status, 62)) break;
        tc_fence_after();
        const uint64_t w0 = umma_desc_sw128(smem_u32(base) + su * 16384);
        const uint64_t a0 = umma_desc_sw128(smem_u32(base) + L.ua + su * mn * 128);
        // K slices of 32: the descriptors' start address advances by 32 bytes
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) tc_mma_f8f6f4(tmem, w0 + kk * 2, a0 + kk * 2, idesc, (it | kk) != 0);
        tc_commit(&empty_u[su]);
      }
      tc_commit(acc_full);
      tc_commit(drain);
      const uint64_t t0 = globaltimer_ns();
      while (!mbar_try_wait(drain, 0) && globaltimer_ns() - t0 < kWaitLimitNs) {
      }
    }
  } else if (warp >= kFirstUnpackWarp) {
    const int group = (warp - kFirstUnpackWarp) >> 2;
    const int u = tid - (kFirstUnpackWarp + 4 * group) * 32;   // 0 .. 127
    const uint32_t xa = ASYM ? 0u : 0x88888888u;
    const uint32_t sbase = smem_u32(base);
    // 16-byte chunk i = u + 128 j of a packed tile is chunk i % 4 of row i / 4;
    // its codes go to chunks 2 (i % 4) and + 1 of the swizzled tile's row.  j
    // adds 32 rows, four 8-row groups.
    const int r0 = u >> 2;
    const uint32_t dst = (uint32_t)((r0 >> 3) * 1024 + (r0 & 7) * 128 + (((2 * (u & 3)) ^ (r0 & 7)) << 4));
    const uint32_t UW = sbase + (uint32_t)(group * 16384) + dst;
    const uint32_t UA = sbase + L.ua + (uint32_t)(group * mn * 128) + dst;
    const uint32_t PW = sbase + L.pw + (uint32_t)(u * 16), PA = sbase + L.pa + (uint32_t)(u * 16);
    const int chunks = mn * 4;
    int sa[TA];
#pragma unroll
    for (int j = 0; j < TA; ++j) sa[j] = 0;
    int s = group, ph = 0;
    for (int it = group; it < nk; it += 2) {
      if (!wait_warp(&full_p[s], (uint32_t)ph, abort_flag, p.status, 63)) break;
      uint4 ww[4], wa[TA];
#pragma unroll
      for (int j = 0; j < 4; ++j) ww[j] = lds128(PW + s * 8192 + 2048 * j);
#pragma unroll
      for (int j = 0; j < TA; ++j)
        wa[j] = u + kGroupThreads * j < chunks ? lds128(PA + s * mn * 64 + 2048 * j) : make_uint4(0, 0, 0, 0);
      // packed stage consumed, once every lane's loads have read it
      wait_loaded(ww, scratch);
      wait_loaded(wa, scratch);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty_p[s]);
      if (!wait_warp(&empty_u[group], ((uint32_t)(it >> 1) & 1u) ^ 1u, abort_flag, p.status, 64)) break;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint4 lo, hi;
        unpack16(ww[j], 0x88888888u, lo, hi);
        sts128(UW + 4096 * j, lo);
        sts128((UW ^ 16u) + 4096 * j, hi);
      }
#pragma unroll
      for (int j = 0; j < TA; ++j) {
        if (u + kGroupThreads * j < chunks) {
          uint4 lo, hi;
          unpack16(wa[j], xa, lo, hi);
          sa[j] = (int)__dp4a(lo.x + lo.y + lo.z + lo.w + hi.x + hi.y + hi.z + hi.w, 0x01010101u, (unsigned)sa[j]);
          sts128(UA + 4096 * j, lo);
          sts128((UA ^ 16u) + 4096 * j, hi);
        }
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full_u[group]);
      if ((s += 2) >= NP) s = group, ph ^= 1;
    }
    __syncwarp();
    // token sums over this group's steps: 4 lanes share a row
#pragma unroll
    for (int j = 0; j < TA; ++j) {
      sa[j] += __shfl_xor_sync(0xffffffffu, sa[j], 1);
      sa[j] += __shfl_xor_sync(0xffffffffu, sa[j], 2);
      const int r = r0 + 32 * j;
      if ((u & 3) == 0 && r < mn) rsa[group * mn + r] = sa[j];
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(rs_full);
  } else {
    // the tokens' scales, staged while the main loop runs
    for (int m = tid - 64; m < mn; m += 128) {
      const float alpha = m < p.a.M ? __ldg(p.a.a_scale + m) : 0.f;
      tal[m] = alpha;
      tbp[m] = ASYM && m < p.a.M ? __ldg(p.a.a_zero + m) + 8.f * alpha : 0.f;
    }
  }
  __syncwarp();

  // the channels' constants for the last part: 4 per lane
  const int n = n0 + 4 * lane;
  float4 sn = make_float4(0.f, 0.f, 0.f, 0.f);
  int4 rwi = make_int4(0, 0, 0, 0);
  if (n < p.a.N) {
    sn = __ldg(reinterpret_cast<const float4*>(p.a.w_scale + n));
    rwi = __ldg(reinterpret_cast<const int4*>(p.a.w_rowsum + n));
  }
  float* part = reinterpret_cast<float*>(base);
  if (warp >= 2) {
    // ---------------- this slice's exact sums: every stage has been read
    const bool ok = wait_warp(acc_full, 0, abort_flag, p.status, 65) && wait_warp(rs_full, 0, abort_flag, p.status, 66);
    __syncwarp();
    tc_fence_after();
    const int q = warp & 3, nl = 32 * q + lane;
    if (ok) {
      for (int c0 = 16 * ((warp - 2) >> 2); c0 < mn; c0 += 48) {
        uint32_t r[16];
        tmem_ld_32x32b_x16(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c0, r);
        tmem_ld_wait(r);
#pragma unroll
        for (int e = 0; e < 16; ++e)
          part[(c0 + e) * 128 + nl] =
              fmaf(__uint_as_float(r[e]), 262144.0f, -8.f * (float)(rsa[c0 + e] + rsa[mn + c0 + e]));
      }
    }
    tc_fence_before();
  }
  __syncwarp();
  cluster_sync_threads();   // (a cluster of one CTA: its threads)
  // ---------------- this CTA's tokens rank, rank + C, ..: sum of the slices, y
  if (!*abort_flag) {
    const float4 rw = make_float4((float)rwi.x, (float)rwi.y, (float)rwi.z, (float)rwi.w);
    for (int m = rank + C * warp; m < p.a.M; m += C * (kThreads / 32)) {
      const uint32_t at = smem_u32(part + m * 128 + 4 * lane);
      float4 v[kMaxCluster];
#pragma unroll
      for (int c = 0; c < kMaxCluster; ++c)
        if (c < C) v[c] = ld_cluster_v4(mapa_shared(at, (uint32_t)c));
      float4 t = v[0];
#pragma unroll
      for (int c = 1; c < kMaxCluster; ++c)
        if (c < C) t.x += v[c].x, t.y += v[c].y, t.z += v[c].z, t.w += v[c].w;
      const float al = tal[m], bp = tbp[m];
      const float a0 = t.x - 8.f * rw.x, a1 = t.y - 8.f * rw.y, a2 = t.z - 8.f * rw.z, a3 = t.w - 8.f * rw.w;
      if (n < p.a.N) {
        const size_t at_y = (size_t)m * p.a.N + n;
        *reinterpret_cast<uint2*>(reinterpret_cast<__half*>(p.a.y) + at_y) =
            make_uint2(pack_half2_bits(sn.x * fmaf(al, a0, bp * rw.x), sn.y * fmaf(al, a1, bp * rw.y)),
                       pack_half2_bits(sn.z * fmaf(al, a2, bp * rw.z), sn.w * fmaf(al, a3, bp * rw.w)));
        if (ACC_OUT)
          *reinterpret_cast<int4*>(p.a.acc_out + at_y) =
              make_int4(__float2int_rn(a0), __float2int_rn(a1), __float2int_rn(a2), __float2int_rn(a3));
      }
    }
  }
  __syncwarp();
  cluster_sync_threads();   // no CTA leaves while another reads its partial sums
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, (uint32_t)p.tmem_cols);
  }
  // The abort flag is final here: after an abort let the producer's last
  // copies land before the CTA and its shared memory go away.
  if (warp == 0 && lane == 0 && *abort_flag)
    for (int j = issued - NP < 0 ? 0 : issued - NP; j < issued; ++j) {
      const uint64_t t0 = globaltimer_ns();
      while (!mbar_try_wait(&full_p[j & (NP - 1)], (uint32_t)(j / NP) & 1u) && globaltimer_ns() - t0 < kWaitLimitNs) {
      }
    }
}

// One CTA per SM: more than half of an SM's shared memory.  Two share it worse
// (a cluster's CTAs are packed in pairs while other SMs idle): 77 tokens,
// 4096 -> 4096, clusters of 4, 15.0 us against 11.7 with the quantizer.
constexpr size_t kMinSmem = 118 * 1024;

template <int TA, bool ASYM, bool ACC_OUT>
cudaError_t launch_t(const GemmArgs& a, int cluster, cudaStream_t stream) {
  const int mn = (int)((a.M + 15) / 16 * 16), tmem_cols = mn <= 32 ? 32 : mn <= 64 ? 64 : 128;
  const size_t smem = std::max<size_t>(Layout(mn).total + 1024, kMinSmem);
  CUtensorMap tmW, tmA;
  if (!encode_packed_map(&tmW, a.w_codes, a.N, a.K, 128) || !encode_packed_map(&tmA, a.a_codes, a.M, a.K, mn))
    return cudaErrorNotSupported;
  auto kern = w4a4_decode_cluster_kernel<TA, ASYM, ACC_OUT>;
  int per_sm = 0;
  cudaError_t e = prepare_launch(kern, kThreads, smem, &per_sm);
  if (e != cudaSuccess) return e;
  const int ksteps = (int)(a.K / 128);
  if (cluster < 1 || cluster > kMaxCluster || cluster > ksteps) return cudaErrorInvalidValue;
  DecodeParams p{a, device_status_word(), mn, ksteps, cluster, tmem_cols};
  p.a.debug_stall = take_debug_stall() ? 1 : 0;
  e = launch_pdl(kern, dim3((unsigned)cluster, (unsigned)((a.N + 127) / 128)), dim3(kThreads), smem, stream, cluster,
                 tmW, tmA, p);
  return e;
}

template <bool ASYM, bool ACC_OUT>
cudaError_t launch_m(const GemmArgs& a, int cluster, cudaStream_t stream) {
  if (a.M <= 32) return launch_t<1, ASYM, ACC_OUT>(a, cluster, stream);
  if (a.M <= 64) return launch_t<2, ASYM, ACC_OUT>(a, cluster, stream);
  if (a.M <= 96) return launch_t<3, ASYM, ACC_OUT>(a, cluster, stream);
  return launch_t<4, ASYM, ACC_OUT>(a, cluster, stream);
}

}  // namespace

cudaError_t set_wait_limit_decode_cluster(uint64_t ns) { return cudaMemcpyToSymbol(g_wait_ns, &ns, sizeof(ns)); }

int w4a4_decode_clusters(int cluster) {
  static std::atomic<int> cache[64][kMaxCluster + 1];   // clusters + 1; 0: not asked yet
  int dev = 0;
  if (cluster < 1 || cluster > kMaxCluster || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int n = cache[dev][cluster].load(std::memory_order_relaxed);
  if (n == 0) {
    auto kern = w4a4_decode_cluster_kernel<1, true, false>;   // every shape takes one CTA per SM
    int per_sm = 0, clusters = 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)cluster);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kMinSmem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cluster == 1) {
      clusters = device_sm_count();
    } else if (prepare_launch(kern, kThreads, kMinSmem, &per_sm) != cudaSuccess ||
               cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess) {
      cudaGetLastError();
      clusters = 0;
    }
    n = clusters + 1;
    cache[dev][cluster].store(n, std::memory_order_relaxed);
  }
  return n - 1;
}

cudaError_t launch_w4a4_decode_cluster(const GemmArgs& a, int cluster, cudaStream_t stream) {
  const bool acc = a.acc_out != nullptr;
  if (a.a_zero) return acc ? launch_m<true, true>(a, cluster, stream) : launch_m<true, false>(a, cluster, stream);
  return acc ? launch_m<false, true>(a, cluster, stream) : launch_m<false, false>(a, cluster, stream);
}

}  // namespace spinq
