// Pieces shared by the LSTM recurrence kernels: launch arguments, cluster addressing, asynchronous stores into a peer CTA's shared
// memory that count bytes on the peer's mbarrier, bounded cluster waits, the fast activations and the exact 3-way bf16 split
// of an fp32 value.
#pragma once
#include <cuda.h>
#include "common.cuh"
#include "kernels.h"

namespace kve {

constexpr int RNN_WARPS = 8;
constexpr int RNN_THREADS = RNN_WARPS * 32;

struct RnnArgs {
  int seq_base;            // the layer's first sequence in the tensor maps over the bf16 summaries (the inputs x_t = [Kbar_t ; Vbar_t])
  const uint16_t* W_ih;    // bf16 [4 d_g][256]
  const float* b_ih;       // [4 d_g]
  const float* b_hh;
  float* H;                // [S * n_range][d_g / 8]: partial sums of w_s . h_t
  const uint16_t* W_hh;    // bf16 [4 d_g][d_g]
  const float* w_s;        // [d_g]
  float b_s;
  float* scores;           // [S][max_chunks]
  float* lstm_h;           // [S][d_g]
  float* lstm_c;
  int32_t* status;
  int32_t* n_listed;       // set to list_cut if that is not negative
  int list_cut;
  int S, max_chunks, t0, n_range, reset;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t smem_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
  return r;
}
// 16 bytes into a peer's shared memory (addresses from mapa), counted on the peer's barrier
__device__ __forceinline__ void st_async_cluster(uint32_t dst, const uint4& v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w), "r"(bar)
               : "memory");
}
// box of a tensor map (dimensions x, y, z) into this CTA's shared memory, bytes counted on `bar`.  No multicast.
__device__ __forceinline__ void tma_load_3d(uint32_t dst_smem, const CUtensorMap* tm, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst_smem),
      "l"(tm), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
      : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded: gives up `deadline_ns` (one second unless told otherwise) after the quick polls ran out, then false
__device__ __forceinline__ bool mbar_wait_cluster_bounded(uint64_t* bar, uint32_t parity,
                                                          unsigned long long deadline_ns = 1000000000ull) {
  for (int i = 0; i < 4096; ++i)
    if (mbar_try_wait_cluster(bar, parity)) return true;
  unsigned long long t_start, t_now;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_start));
  do {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    __nanosleep(128);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_now));
  } while (t_now - t_start < deadline_ns);
  return false;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ float fast_sigmoid(float x) { return __fdividef(1.f, 1.f + __expf(-x)); }
__device__ __forceinline__ float fast_tanh(float x) { return 2.f * fast_sigmoid(2.f * x) - 1.f; }
// Two LSTM cells at once, in packed operations where there are any: pre-activations in the order i, f, g, o; updates c, returns h.
// With E(x) = 2^(-x log2 e):
//   c = f c + i g = [c (1 + E_i)(1 + E_2g) + (1 - E_2g)(1 + E_f)] / [(1 + E_f)(1 + E_i)(1 + E_2g)],  h = (1 - E_2c) / [(1 + E_o)(1 + E_2c)]
// five exponentials and two reciprocals per cell.  The exponents stop at 40 (a sigmoid of 1e-12), which keeps the products finite.
__device__ __forceinline__ float2 lstm_cell_pair(const float2 (&pre)[4], float2& c) {
  constexpr float L2E = 1.44269504088896340736f;
  const float2 one = make_float2(1.f, 1.f);
  auto e = [](float2 x, float scale) {      // 2^(-x scale), at most 2^40; NaN stays NaN
    const float2 y = mul2(x, make_float2(-scale, -scale));
    float2 z;
    asm("min.NaN.f32 %0, %1, 0f42200000;" : "=f"(z.x) : "f"(y.x));
    asm("min.NaN.f32 %0, %1, 0f42200000;" : "=f"(z.y) : "f"(y.y));
    return make_float2(ex2_fast(z.x), ex2_fast(z.y));
  };
  auto minus = [&](float2 x) { return add2(one, make_float2(-x.x, -x.y)); };
  const float2 ei = add2(one, e(pre[0], L2E)), ef = add2(one, e(pre[1], L2E));
  const float2 g2 = e(pre[2], 2.f * L2E), eo = add2(one, e(pre[3], L2E));
  const float2 ig = mul2(ei, add2(one, g2));
  const float2 num = fma2(c, ig, mul2(minus(g2), ef)), den = mul2(ef, ig);
  c = make_float2(__fdividef(num.x, den.x), __fdividef(num.y, den.y));
  const float2 c2 = e(c, 2.f * L2E);
  const float2 top = minus(c2), low = mul2(eo, add2(one, c2));
  return make_float2(__fdividef(top.x, low.x), __fdividef(top.y, low.y));
}
// four 8 x 8 b16 blocks of shared memory as mma fragments (lane l gives the address of row l & 7 of block l >> 3)
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

// exact 3-way split of an fp32 value into bf16 pieces: x = p0 + p1 + p2
__device__ __forceinline__ void split3(float x, uint32_t (&p)[3]) {
  p[0] = f32_to_bf16_bits(x);
  const float r1 = x - __uint_as_float(p[0] << 16);
  p[1] = f32_to_bf16_bits(r1);
  const float r2 = r1 - __uint_as_float(p[1] << 16);
  p[2] = f32_to_bf16_bits(r2);
}

}  // namespace kve
