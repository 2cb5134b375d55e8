// kvE_summarize_chunks kernels (Eq. 2): per (sequence, chunk) the mean of the chunk's C key rows and
// of its C value rows, then (AGG_MLP) a 2-layer GELU MLP on each mean.
//
// chunk_mean: HBM-bound.  One warp per page (K or V of a (sequence, chunk) unit): 8 bytes per lane and row, 32 rows in flight,
// added in temporal order in fp32 (so the sum has the same rounding as a plain sequential loop), divided by C with an
// IEEE division.  Two-warp CTAs, dealt out by the hardware: a few units spread over all SMs, and many need no common wave.
//   Measured (chains of launches, DRAM): 8 sequences x 28 chunks of 64 tokens 12.3 -> 3.3 us, 128 x 1 (one trigger) 10.3 -> 3.0,
//   512 x 12 of 128 tokens 95 -> 62 us (6.5 TB/s), 512 x 121 of 128 tokens 672 -> 614 us (6.6 TB/s).  (Before: a warp per
//   unit, 16 bytes per lane, 8 rows in flight, one resident wave striding over the units, launched behind a drained GPU.)
// The kernel wants the L1 that attention, with its 200 KB of shared memory per SM, takes away: CTAs that land beside it keep
// the SM in that split for as long as any of them is there, and 32 rows in flight per lane do not fit (4 GB: 720 us).  Large
// launches therefore ask for the large L1 (an SM drains before its first CTA); small ones start at once.
#include "common.cuh"
#include "kernels.h"
#include "umma.cuh"
#include "gelu.cuh"

namespace kve {

constexpr int MEAN_WARPS = 2;
constexpr int MEAN_UNROLL = 32;                       // rows in flight
constexpr long long MEAN_LARGE_ROWS = 1LL << 16;      // K (or V) rows from which a launch asks for the large L1: 32 MB

// POOL_MAX: element-wise maximum of the chunk instead of its mean (the "pooling" aggregator of Sec. 3.1)
template <bool POOL_MAX>
__global__ void __launch_bounds__(MEAN_WARPS * 32) kve_chunk_mean_kernel(LayerView v, int t0, int n_range, FastDiv by_range,
                                                                        int final_output, int dev_window, int list_cut) {
  pdl_launch_dependents();
  pdl_wait();
  if (list_cut >= 0 && blockIdx.x == 0 && threadIdx.x == 0) *v.n_listed = list_cut;
  if (dev_window >= 0) {      // one chunk per sequence, found on the device
    const NextChunk nx = next_chunk(v.n_listed, v.seq_len, v.C, dev_window, v.max_chunks);
    if (!nx.due) return;
    t0 = nx.t;
  }
  const int lane = threadIdx.x & 31, is_v = threadIdx.x >> 5, unit = (int)blockIdx.x;
  const int s = (int)by_range.div((uint32_t)unit), t = t0 + (unit - s * n_range);
  const long long page = v.page_table[(long long)s * v.max_chunks + t];
  if (page < 0 || page >= v.n_pages) {
    if (lane == 0) set_status(v.status, ERR_CAPACITY);
    return;
  }
  const uint2* src = reinterpret_cast<const uint2*>((is_v ? v.v_pages : v.k_pages) + page * v.C * D) + lane;
  float acc[4];
#pragma unroll
  for (int x = 0; x < 4; ++x) acc[x] = POOL_MAX ? -INFINITY : 0.f;
  auto take = [&](const uint2& w) {      // the next row
    const float f[4] = {bf16lo(w.x), bf16hi(w.x), bf16lo(w.y), bf16hi(w.y)};
#pragma unroll
    for (int x = 0; x < 4; ++x) acc[x] = POOL_MAX ? fmaxf(acc[x], f[x]) : acc[x] + f[x];
  };
  int j = 0;
  for (; j + MEAN_UNROLL <= v.C; j += MEAN_UNROLL) {
    uint2 w[MEAN_UNROLL];
#pragma unroll
    for (int u = 0; u < MEAN_UNROLL; ++u) w[u] = __ldcs(src + (j + u) * (D / 4));
#pragma unroll
    for (int u = 0; u < MEAN_UNROLL; ++u) take(w[u]);
  }
  if (j < v.C) {      // the rest of the chunk, in flight together too
    uint2 w[MEAN_UNROLL];
#pragma unroll
    for (int u = 0; u < MEAN_UNROLL; ++u)
      if (j + u < v.C) w[u] = __ldcs(src + (j + u) * (D / 4));
#pragma unroll
    for (int u = 0; u < MEAN_UNROLL; ++u)
      if (j + u < v.C) take(w[u]);
  }
  if (!POOL_MAX) {
    const float fc = (float)v.C;
#pragma unroll
    for (int x = 0; x < 4; ++x) acc[x] = __fdiv_rn(acc[x], fc);
  }
  const long long o = ((long long)s * v.max_chunks + t) * D + lane * 4;
  *reinterpret_cast<float4*>((is_v ? v.vsum_f32 : v.ksum_f32) + o) = make_float4(acc[0], acc[1], acc[2], acc[3]);
  if (final_output)
    *reinterpret_cast<uint2*>((is_v ? v.vsum_bf16 : v.ksum_bf16) + o) = make_uint2(pack_bf16x2(acc[0], acc[1]), pack_bf16x2(acc[2], acc[3]));
}

// ---- the same mean over short chunks ---------------------------------------------------------------------------------
// With few rows per page a CTA per unit spends its time starting up (and the summaries, 1536 bytes a unit, become the larger
// part of the traffic).  Here a warp takes a unit, K in its lower and V in its upper lanes, 16 bytes each, SHORT_ROWS rows in flight, or
// (MULTI) as many units of up to four rows as make up that number; eight warps to a CTA.
//   us, a CTA per unit -> this: 128 sequences x 4160 tokens in chunks of 1, 4, 8, 16, 24 tokens 962 -> 165, 270 -> 74, 144 -> 57, 74 -> 45,
//   55 -> 42; 60 x 2000 in chunks of 1, 4, 8 204 -> 39, 52 -> 15, 29 -> 11.  From 9 tokens on a launch that leaves SMs without work is
//   better off with all rows of a page in flight: 8 x 2048 in chunks of 24 6.1 us this way, 4.0 the other; 60 x 2000 14.8 and 12.8.
constexpr int SHORT_WARPS = 8, SHORT_ROWS = 8;

template <bool POOL_MAX, bool MULTI>
__global__ void __launch_bounds__(SHORT_WARPS * 32, 4) kve_chunk_mean_short_kernel(LayerView v, int t0, int n_range, FastDiv by_range, int n_units,
                                                                                  int final_output, int dev_window, int list_cut) {
  pdl_launch_dependents();
  pdl_wait();
  if (list_cut >= 0 && blockIdx.x == 0 && threadIdx.x == 0) *v.n_listed = list_cut;
  if (dev_window >= 0) {      // one chunk per sequence, found on the device
    const NextChunk nx = next_chunk(v.n_listed, v.seq_len, v.C, dev_window, v.max_chunks);
    if (!nx.due) return;
    t0 = nx.t;
  }
  const int lane = threadIdx.x & 31, is_v = lane >> 4, l16 = lane & 15;
  const int per_warp = MULTI ? SHORT_ROWS / v.C : 1;
  const long long unit0 = ((long long)blockIdx.x * SHORT_WARPS + (threadIdx.x >> 5)) * per_warp;
  const int n_mine = (int)min((long long)per_warp, n_units - unit0);
  if (n_mine <= 0) return;
  // lane u keeps the page and the summary row of unit u
  int page = -1;
  long long row_of = 0;
  if (lane < n_mine) {
    const int unit = (int)unit0 + lane, s = (int)by_range.div((uint32_t)unit);
    row_of = (long long)s * v.max_chunks + t0 + (unit - s * n_range);
    page = v.page_table[row_of];
    if (page < 0 || page >= v.n_pages) {
      set_status(v.status, ERR_CAPACITY);
      page = -1;
    }
  }
  const uint4* pool = reinterpret_cast<const uint4*>(is_v ? v.v_pages : v.k_pages) + l16;
  float acc[8];
  auto clear = [&]() {
#pragma unroll
    for (int x = 0; x < 8; ++x) acc[x] = POOL_MAX ? -INFINITY : 0.f;
  };
  auto take = [&](const uint4& w) {      // the next row
    const float f[8] = {bf16lo(w.x), bf16hi(w.x), bf16lo(w.y), bf16hi(w.y), bf16lo(w.z), bf16hi(w.z), bf16lo(w.w), bf16hi(w.w)};
#pragma unroll
    for (int x = 0; x < 8; ++x) acc[x] = POOL_MAX ? fmaxf(acc[x], f[x]) : acc[x] + f[x];
  };
  auto finish = [&](int u) {
    const long long o = __shfl_sync(0xffffffffu, row_of, u) * D + l16 * 8;
    if (__shfl_sync(0xffffffffu, page, u) < 0) return;
    const float fc = (float)v.C;
#pragma unroll
    for (int x = 0; x < 8; ++x)
      if (!POOL_MAX) acc[x] = __fdiv_rn(acc[x], fc);
    float4* out = reinterpret_cast<float4*>((is_v ? v.vsum_f32 : v.ksum_f32) + o);
    out[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    out[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    if (final_output)
      *reinterpret_cast<uint4*>((is_v ? v.vsum_bf16 : v.ksum_bf16) + o) =
          make_uint4(pack_bf16x2(acc[0], acc[1]), pack_bf16x2(acc[2], acc[3]), pack_bf16x2(acc[4], acc[5]), pack_bf16x2(acc[6], acc[7]));
  };
  uint4 w[SHORT_ROWS];
  clear();
  if constexpr (MULTI) {
    int u = 0, row = 0;
#pragma unroll
    for (int x = 0; x < SHORT_ROWS; ++x) {
      const int p = __shfl_sync(0xffffffffu, page, u);
      if (p >= 0) w[x] = __ldcs(pool + ((long long)p * v.C + row) * 16);      // (lanes without a unit hold -1)
      if (++row == v.C) { row = 0; ++u; }
    }
    u = row = 0;
#pragma unroll
    for (int x = 0; x < SHORT_ROWS; ++x) {
      if (u >= n_mine) break;
      take(w[x]);
      if (++row == v.C) {
        finish(u);
        clear();
        row = 0;
        ++u;
      }
    }
  } else {
    const int p = __shfl_sync(0xffffffffu, page, 0);
    if (p < 0) return;
    const uint4* src = pool + (long long)p * v.C * 16;
    for (int j = 0; j < v.C; j += SHORT_ROWS) {
#pragma unroll
      for (int x = 0; x < SHORT_ROWS; ++x)
        if (j + x < v.C) w[x] = __ldcs(src + (j + x) * 16);
#pragma unroll
      for (int x = 0; x < SHORT_ROWS; ++x)
        if (j + x < v.C) take(w[x]);
    }
    finish(0);
  }
}

static cudaError_t launch_chunk_mean_short(const LayerView& v, int t0, int n_range, long long n_units, bool final_output, bool pool_max,
                                           cudaStream_t st, int dev_window, int list_cut) {
  const bool multi = 2 * v.C <= SHORT_ROWS && n_units * v.C / SHORT_ROWS > 16LL * sm_count();      // (16 warps for every SM first)
  const long long per_cta = (long long)SHORT_WARPS * (multi ? SHORT_ROWS / v.C : 1);
  const dim3 grid((unsigned)((n_units + per_cta - 1) / per_cta)), block(SHORT_WARPS * 32);
  const FastDiv by_range = fast_div((uint32_t)n_range);
  auto* kernel = pool_max ? (multi ? kve_chunk_mean_short_kernel<true, true> : kve_chunk_mean_short_kernel<true, false>)
                          : (multi ? kve_chunk_mean_short_kernel<false, true> : kve_chunk_mean_short_kernel<false, false>);
  return launch_pdl(kernel, grid, block, 0, st, v, t0, n_range, by_range, (int)n_units, pool_max || final_output ? 1 : 0, dev_window, list_cut);
}

cudaError_t launch_chunk_mean(const LayerView& v, int t0, int t1, bool final_output, bool pool_max, cudaStream_t st, int dev_window, int list_cut) {
  const int n_range = dev_window >= 0 ? 1 : t1 - t0;
  const long long n_units = (long long)v.S * n_range;
  if (n_units <= 0) return cudaSuccess;
  if (n_units >= (1LL << 31)) return cudaErrorInvalidValue;
  if (v.C <= SHORT_ROWS || (v.C < 32 && n_units > 64LL * sm_count())) return launch_chunk_mean_short(v, t0, n_range, n_units, final_output, pool_max, st, dev_window, list_cut);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  attr[1].val.sharedMemCarveout = cudaSharedmemCarveoutMaxL1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)n_units);
  cfg.blockDim = dim3(MEAN_WARPS * 32);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = n_units * v.C >= MEAN_LARGE_ROWS ? 2 : 1;
  const FastDiv by_range = fast_div((uint32_t)n_range);
  return pool_max ? cudaLaunchKernelEx(&cfg, kve_chunk_mean_kernel<true>, v, t0, n_range, by_range, 1, dev_window, list_cut)
                  : cudaLaunchKernelEx(&cfg, kve_chunk_mean_kernel<false>, v, t0, n_range, by_range, final_output ? 1 : 0, dev_window, list_cut);
}

// ---- the same mean for a launch that runs beside the gate recurrence -----------------------------------------------
// The recurrence leaves an SM 4 K to 25 K of its registers and about two thirds of its shared memory (two CTAs of this kernel), so the rows on their way wait there: a
// warp's pages come in bulk copies of 16 rows, eight of them in flight, and are added up row by row as above (the same rounding).
// A CTA takes several units in a row, so that the copies of the next one are under way while the last is added up.
// 512 sequences, pages of 128 tokens: 92 chunks of the gate (203 us alone) and the means of 29 (142 us alone) take 272 us together; with three
// planes 86 chunks (239 us) and 35 (172 us) 325 us.  (Beside the recurrence of before, without the projection: 4.1 TB/s, the recurrence 22 % longer; the
// kernel above, its rows in registers: 3 TB/s.)  Fewer rows in flight were slower for the whole step (eight pieces of 8 rows +1 %, four +9 %), asynchronous
// 16-byte copies +0.6 %; 256 rows per CTA +1 %, 512 +2 %, and a CTA per page +4 % with pages of 32 tokens.
constexpr int MB_ROWS = 16, MB_STAGES = 8;
constexpr int MB_CTA_ROWS = 128;                      // rows of K (or V) that a CTA takes, about
constexpr int MB_STAGE_BYTES = MB_ROWS * D * 2;
constexpr int MB_SMEM_BAR = MEAN_WARPS * MB_STAGES * MB_STAGE_BYTES;
constexpr int MB_SMEM_BYTES = MB_SMEM_BAR + MEAN_WARPS * MB_STAGES * 8;

template <bool POOL_MAX>
__global__ void __launch_bounds__(MEAN_WARPS * 32, 65536 / MEAN_BESIDE_REGS) kve_chunk_mean_beside_kernel(LayerView v, int t0, int n_range, FastDiv by_range, int n_units,
                                                                               int units_per_cta, int final_output) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  pdl_launch_dependents();
  if (blockIdx.x == gridDim.x - 1) {      // an extra CTA, the last to be placed: this launch is not over before the one it runs beside
    pdl_wait();
    return;
  }
  const int lane = threadIdx.x & 31, is_v = threadIdx.x >> 5;
  const int unit0 = (int)blockIdx.x * units_per_cta, n_mine = min(units_per_cta, n_units - unit0);      // 1 .. 32
  // lane u keeps the page and the summary row of unit u
  long long page = -1, row_of = 0;
  if (lane < n_mine) {
    const int s = (int)by_range.div((uint32_t)(unit0 + lane)), t = t0 + (unit0 + lane - s * n_range);
    row_of = (long long)s * v.max_chunks + t;
    page = v.page_table[row_of];
    if (page < 0 || page >= v.n_pages) {
      set_status(v.status, ERR_CAPACITY);
      page = -1;
    }
  }
  unsigned char* ring = smem_raw + is_v * MB_STAGES * MB_STAGE_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw + MB_SMEM_BAR) + is_v * MB_STAGES;
  const uint16_t* pool = is_v ? v.v_pages : v.k_pages;
  const int per_unit = (v.C + MB_ROWS - 1) / MB_ROWS;      // pieces of a page; one without a page has none
  int f_unit = 0, f_piece = 0, n_fetched = 0;              // the next piece to fetch (the same in all lanes)
  auto fetch = [&]() {
    long long p = -1;
    while (f_unit < n_mine && (p = __shfl_sync(0xffffffffu, page, f_unit)) < 0) ++f_unit;
    if (f_unit >= n_mine) return;
    if (lane == 0) {
      const uint32_t bytes = (uint32_t)min(MB_ROWS, v.C - f_piece * MB_ROWS) * D * 2;
      uint64_t* bar = &full[n_fetched % MB_STAGES];
      mbar_arrive_expect_tx(bar, bytes);
      bulk_g2s(ring + (n_fetched % MB_STAGES) * MB_STAGE_BYTES, pool + (p * v.C + f_piece * MB_ROWS) * D, bytes, bar);
    }
    ++n_fetched;
    if (++f_piece == per_unit) { f_piece = 0; ++f_unit; }
  };
  if (lane == 0) {
    for (int i = 0; i < MB_STAGES; ++i) mbar_init(&full[i], 1);
    mbar_fence_init();
  }
  __syncwarp();
  for (int i = 0; i < MB_STAGES; ++i) fetch();
  bool ok = true;
  int i = 0;                                               // the next piece to add up
  for (int u = 0; u < n_mine && ok; ++u) {
    if (__shfl_sync(0xffffffffu, page, u) < 0) continue;
    float acc[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) acc[x] = POOL_MAX ? -INFINITY : 0.f;
    auto take = [&](const uint2& w) {
      const float f[4] = {bf16lo(w.x), bf16hi(w.x), bf16lo(w.y), bf16hi(w.y)};
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[x] = POOL_MAX ? fmaxf(acc[x], f[x]) : acc[x] + f[x];
    };
    for (int p = 0; p < per_unit; ++p, ++i) {
      ok = __all_sync(0xffffffffu, mbar_wait_bounded(&full[i % MB_STAGES], (uint32_t)((i / MB_STAGES) & 1)));
      if (!ok) break;
      const uint2* row = reinterpret_cast<const uint2*>(ring + (i % MB_STAGES) * MB_STAGE_BYTES) + lane;
      const int rows = min(MB_ROWS, v.C - p * MB_ROWS);
      if (rows == MB_ROWS) {
#pragma unroll
        for (int j = 0; j < MB_ROWS; ++j) take(row[j * (D / 4)]);
      } else {
        for (int j = 0; j < rows; ++j) take(row[j * (D / 4)]);
      }
      __syncwarp();
      fetch();
    }
    if (!ok) break;
    if (!POOL_MAX) {
      const float fc = (float)v.C;
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[x] = __fdiv_rn(acc[x], fc);
    }
    const long long o = __shfl_sync(0xffffffffu, row_of, u) * D + lane * 4;
    *reinterpret_cast<float4*>((is_v ? v.vsum_f32 : v.ksum_f32) + o) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    if (final_output)
      *reinterpret_cast<uint2*>((is_v ? v.vsum_bf16 : v.ksum_bf16) + o) = make_uint2(pack_bf16x2(acc[0], acc[1]), pack_bf16x2(acc[2], acc[3]));
  }
  if (!ok) {      // a wait ran out: the other copies under way are still waited for
    if (lane == 0) set_status(v.status, ERR_TIMEOUT);
    for (++i; i < n_fetched; ++i) mbar_wait_bounded(&full[i % MB_STAGES], (uint32_t)((i / MB_STAGES) & 1));
  }
}

cudaError_t launch_chunk_mean_beside(const LayerView& v, int t0, int t1, bool final_output, bool pool_max, cudaStream_t st) {
  const int n_range = t1 - t0;
  const long long n_units = (long long)v.S * n_range;
  if (n_units <= 0 || n_units >= (1LL << 31) - 64) return cudaErrorInvalidValue;
  static DeviceFlags opted, opted_max;
  const cudaError_t e = pool_max ? smem_opt_in(opted_max, kve_chunk_mean_beside_kernel<true>, MB_SMEM_BYTES)
                                 : smem_opt_in(opted, kve_chunk_mean_beside_kernel<false>, MB_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  int per_cta = v.C < MB_CTA_ROWS ? MB_CTA_ROWS / v.C : 1;
  if (per_cta > 32) per_cta = 32;
  while (per_cta > 1 && n_units / per_cta < 4 * sm_count()) per_cta /= 2;
  const dim3 grid((unsigned)((n_units + per_cta - 1) / per_cta) + 1), block(MEAN_WARPS * 32);
  const FastDiv by_range = fast_div((uint32_t)n_range);
  return pool_max ? launch_pdl(kve_chunk_mean_beside_kernel<true>, grid, block, MB_SMEM_BYTES, st, v, t0, n_range, by_range, (int)n_units, per_cta, 1)
                  : launch_pdl(kve_chunk_mean_beside_kernel<false>, grid, block, MB_SMEM_BYTES, st, v, t0, n_range, by_range, (int)n_units, per_cta,
                               final_output ? 1 : 0);
}

// ---- aggregator MLP (Eq. 2 read as mean -> d_sum -> d, exact-erf GELU), fp32 FMA ------------------
// A CTA takes MLP_ROWS (sequence, chunk) units of one side (blockIdx.y: 0 = keys, 1 = values).
// The unit's mean sits in ksum_f32 / vsum_f32 (written by chunk_mean); the MLP output overwrites it
// and its bf16 rounding goes to ksum_bf16 / vsum_bf16.
constexpr int MLP_ROWS = 32;
constexpr int MLP_THREADS = 256;

__device__ __forceinline__ float gelu_erf(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752440f)); }

__device__ __forceinline__ void unpack8(const uint4& w, float (&f)[8]) {
  f[0] = bf16lo(w.x); f[1] = bf16hi(w.x); f[2] = bf16lo(w.y); f[3] = bf16hi(w.y);
  f[4] = bf16lo(w.z); f[5] = bf16hi(w.z); f[6] = bf16lo(w.w); f[7] = bf16hi(w.w);
}

__global__ void __launch_bounds__(MLP_THREADS) kve_chunk_mlp_kernel(LayerView v, int t0, int n_range, long long n_units,
                                                                   MlpWeights w, int d_sum, int dev_window) {
  pdl_launch_dependents();
  pdl_wait();
  if (dev_window >= 0) {      // one chunk per sequence, found on the device
    const NextChunk nx = next_chunk(v.n_listed, v.seq_len, v.C, dev_window, v.max_chunks);
    if (!nx.due) return;
    t0 = nx.t;
  }
  extern __shared__ __align__(16) float smem[];
  float* Xs = smem;                    // [MLP_ROWS][128]
  float* Hs = smem + MLP_ROWS * D;     // [MLP_ROWS][d_sum]
  const int tid = threadIdx.x;
  const int side = blockIdx.y;
  const uint16_t* W1 = side ? w.W1V : w.W1K;
  const uint16_t* W2 = side ? w.W2V : w.W2K;
  const float* b1 = side ? w.b1V : w.b1K;
  const float* b2 = side ? w.b2V : w.b2K;
  float* sum_f32 = side ? v.vsum_f32 : v.ksum_f32;
  uint16_t* sum_b16 = side ? v.vsum_bf16 : v.ksum_bf16;
  const long long unit0 = (long long)blockIdx.x * MLP_ROWS;

  // stage the means
  for (int i = tid; i < MLP_ROWS * (D / 4); i += MLP_THREADS) {
    const int r = i / (D / 4), c4 = i % (D / 4);
    const long long unit = unit0 + r;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (unit < n_units) {
      const int s = (int)(unit / n_range);
      const int t = t0 + (int)(unit - (long long)s * n_range);
      x = *reinterpret_cast<const float4*>(sum_f32 + ((long long)s * v.max_chunks + t) * D + c4 * 4);
    }
    reinterpret_cast<float4*>(Xs)[i] = x;
  }
  __syncthreads();

  // layer 1: thread owns hidden unit u, accumulates all rows
  for (int u = tid; u < d_sum; u += MLP_THREADS) {
    float acc[MLP_ROWS];
    const float bias = b1[u];
#pragma unroll
    for (int r = 0; r < MLP_ROWS; ++r) acc[r] = bias;
    const uint4* wrow = reinterpret_cast<const uint4*>(W1 + (long long)u * D);
    for (int x8 = 0; x8 < D / 8; ++x8) {
      float wf[8];
      unpack8(__ldg(wrow + x8), wf);
#pragma unroll
      for (int r = 0; r < MLP_ROWS; ++r) {
        const float4 a = *reinterpret_cast<const float4*>(Xs + r * D + x8 * 8);
        const float4 b = *reinterpret_cast<const float4*>(Xs + r * D + x8 * 8 + 4);
        acc[r] = fmaf(wf[0], a.x, acc[r]); acc[r] = fmaf(wf[1], a.y, acc[r]);
        acc[r] = fmaf(wf[2], a.z, acc[r]); acc[r] = fmaf(wf[3], a.w, acc[r]);
        acc[r] = fmaf(wf[4], b.x, acc[r]); acc[r] = fmaf(wf[5], b.y, acc[r]);
        acc[r] = fmaf(wf[6], b.z, acc[r]); acc[r] = fmaf(wf[7], b.w, acc[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < MLP_ROWS; ++r) Hs[r * d_sum + u] = gelu_erf(acc[r]);
  }
  __syncthreads();

  // layer 2: thread owns output dim x for half of the rows
  {
    const int x = tid & (D - 1);
    const int r0 = (tid >> 7) * (MLP_ROWS / 2);
    float acc[MLP_ROWS / 2];
    const float bias = b2[x];
#pragma unroll
    for (int r = 0; r < MLP_ROWS / 2; ++r) acc[r] = bias;
    const uint4* wrow = reinterpret_cast<const uint4*>(W2 + (long long)x * d_sum);
    for (int u8 = 0; u8 < d_sum / 8; ++u8) {
      float wf[8];
      unpack8(__ldg(wrow + u8), wf);
#pragma unroll
      for (int r = 0; r < MLP_ROWS / 2; ++r) {
        const float4 a = *reinterpret_cast<const float4*>(Hs + (r0 + r) * d_sum + u8 * 8);
        const float4 b = *reinterpret_cast<const float4*>(Hs + (r0 + r) * d_sum + u8 * 8 + 4);
        acc[r] = fmaf(wf[0], a.x, acc[r]); acc[r] = fmaf(wf[1], a.y, acc[r]);
        acc[r] = fmaf(wf[2], a.z, acc[r]); acc[r] = fmaf(wf[3], a.w, acc[r]);
        acc[r] = fmaf(wf[4], b.x, acc[r]); acc[r] = fmaf(wf[5], b.y, acc[r]);
        acc[r] = fmaf(wf[6], b.z, acc[r]); acc[r] = fmaf(wf[7], b.w, acc[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < MLP_ROWS / 2; ++r) {
      const long long unit = unit0 + r0 + r;
      if (unit < n_units) {
        const int s = (int)(unit / n_range);
        const int t = t0 + (int)(unit - (long long)s * n_range);
        const long long o = ((long long)s * v.max_chunks + t) * D + x;
        sum_f32[o] = acc[r];
        sum_b16[o] = (uint16_t)f32_to_bf16_bits(acc[r]);
      }
    }
  }
}

// ---- the same MLP on the 5th-generation tensor cores (d_sum a multiple of 64, at most 256) ----------------
// Both layers are GEMMs over a tile of 128 (sequence, chunk) units:
//   H = M W1^T  (128 x d_sum, K = 128),   Y = gelu(H + b1) W2^T  (128 x 128, K = d_sum).
// The left operands (the chunk means, the activations) are fp32.  Each is split exactly into three
// bf16 planes (x = p0 + p1 + p2), the weights are bf16 by definition, so every product the tensor
// core forms is exact and the result differs from a plain fp32 loop only in summation order.
//  * A CTA serves one side (keys or values) and keeps that side's W1 and W2 (64 KB each, K-major,
//    128-byte swizzle) in shared memory for all its tiles.
//  * Warps 8-15 load the means of a tile, split them and store the planes as the A operand of layer 1 (96 KB); later they take
//    Y of the tile before out of tensor memory, add b2 and write the fp32 summary and its bf16 rounding.
//  * Warp 16 (one thread) issues the MMAs: layer 1 in halves of 128 hidden units into two accumulators, layer 2 in slices of
//    32 units into Y - whichever has its inputs ready.
//  * Warps 0-7, two groups of four, take the slices in turn: 32 hidden units of a row per thread out of tensor memory, b1, GELU,
//    split, and back into TENSOR memory as the A operand of layer 2 (shared memory is full).  One group's slice is
//    multiplied while the other's is worked out.
// So layer 1 of a tile, its activations, layer 2 and the output of the tile before overlap.  Per tile the MMAs now take
// ~13000 cycles (the ones with their left operand in tensor memory 130 to 180 each, the others 85) and the activations
// ~9000 per warp; with all sixteen warps going through the phases together a tile took 22500 cycles.  512 x 121 chunks:
// 96 -> 88 us; the second layer alone on 256 x 56 chunks 25 -> 15 us; small launches (256 x 56 chunks: 33 us) are the weights'
// way into shared memory and the latency of one or two tiles, and did not change.
// POOLED: the second layer alone, on the pooled activations hid [2][n_units][d_sum] of the per-token aggregator.  Its small
// planes have an accumulator of their own (in the columns that layer 1 leaves free): the tensor core cuts off what lies
// below the last bit of the accumulator at each of its steps, so the large sum takes d_sum / 16 of them, not three times that
// (rms error of the
// summaries against 64 bits on 256 x 56 chunks: keys 3.7e-7 -> 1.3e-7, values 2.4e-7 -> 0.7e-7; fp32 loops: 1.4e-7, 1.0e-7).
// Every mbarrier wait is bounded; on give-up the status word gets KVE_ERR_TIMEOUT.
constexpr int MT_M = 128;
constexpr int MT_GELU_WARPS = 8, MT_IO_WARPS = 8;
constexpr int MT_MMA_WARP = MT_GELU_WARPS + MT_IO_WARPS;
constexpr int MT_THREADS = (MT_MMA_WARP + 1) * 32;
constexpr int MT_MAX_DSUM = 256;
constexpr int MT_SLICE = 32;                                              // hidden units per layer-2 slice
constexpr int MT_PLANE_KB_BYTES = MT_M * umma::KBLOCK_ROW_BYTES;          // 16 KB: one plane, one K-block of 64
constexpr int MT_SMEM_A = 0;                                              // 96 KB: 3 planes x 2 K-blocks
constexpr int MT_SMEM_W1 = MT_SMEM_A + 6 * MT_PLANE_KB_BYTES;
constexpr int MT_SMEM_W2 = MT_SMEM_W1 + MT_MAX_DSUM * D * 2;
constexpr int MT_SMEM_B1 = MT_SMEM_W2 + D * MT_MAX_DSUM * 2;
constexpr int MT_SMEM_B2 = MT_SMEM_B1 + MT_MAX_DSUM * 4;
constexpr int MT_SMEM_BAR = MT_SMEM_B2 + D * 4;
constexpr int MT_SMEM_BYTES = MT_SMEM_BAR + 128 + 1024;                   // + slack to reach a 1024-byte boundary
static_assert(MT_SMEM_BYTES <= 227 * 1024, "shared memory of one CTA");
constexpr int MT_TMEM_COLS = 512;      // H halves: columns 0 and 128; Y: 256; activations of the two groups: 384, 432 (3 planes x 16)
constexpr int MT_TMEM_YLO = 0;         // POOLED: sum of the two small planes, where H would be
constexpr int MT_TMEM_Y = 256, MT_TMEM_ACT = 384, MT_ACT_COLS = 3 * MT_SLICE / 2;

// 8 consecutive floats: one 32-byte access (a whole sector) where the array starts on such a boundary, two of 16 bytes otherwise
__device__ __forceinline__ void load8(const float* p, float (&x)[8], bool wide) {
  if (wide) {
    asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7])
                 : "l"(p)
                 : "memory");
  } else {
    const float4 lo = *reinterpret_cast<const float4*>(p), hi = *reinterpret_cast<const float4*>(p + 4);
    x[0] = lo.x; x[1] = lo.y; x[2] = lo.z; x[3] = lo.w;
    x[4] = hi.x; x[5] = hi.y; x[6] = hi.z; x[7] = hi.w;
  }
}
__device__ __forceinline__ void store8(float* p, const float (&x)[8], bool wide) {
  if (wide) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(x[4]),
                 "f"(x[5]), "f"(x[6]), "f"(x[7])
                 : "memory");
  } else {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
    *reinterpret_cast<float4*>(p + 4) = make_float4(x[4], x[5], x[6], x[7]);
  }
}
// splits 8 consecutive fp32 values and stores the three 16-byte pieces at dst + pl * plane_stride
__device__ __forceinline__ void store_split8(const float (&x)[8], unsigned char* dst, int plane_stride) {
  uint32_t w[4][3];
#pragma unroll
  for (int e = 0; e < 4; ++e) split3_pair(x[2 * e], x[2 * e + 1], w[e]);
#pragma unroll
  for (int pl = 0; pl < 3; ++pl)
    *reinterpret_cast<uint4*>(dst + pl * plane_stride) = make_uint4(w[0][pl], w[1][pl], w[2][pl], w[3][pl]);
}

template <bool POOLED>
__global__ void __launch_bounds__(MT_THREADS, 1) kve_chunk_mlp_tc_kernel(LayerView v, int t0, int n_range, FastDiv by_range, int n_units,
                                                                         MlpWeights w, int d_sum, int dev_window,
                                                                         const float* __restrict__ hid) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* As = smem + MT_SMEM_A;
  unsigned char* W1s = smem + MT_SMEM_W1;
  unsigned char* W2s = smem + MT_SMEM_W2;
  float* b1s = reinterpret_cast<float*>(smem + MT_SMEM_B1);
  float* b2s = reinterpret_cast<float*>(smem + MT_SMEM_B2);
  uint64_t* a_full = reinterpret_cast<uint64_t*>(smem + MT_SMEM_BAR);      // planes of a tile's means stored
  uint64_t* a_free = a_full + 1;                                            // ... read (layer 1 done)
  uint64_t* h_full = a_free + 1;                                            // [2] accumulator of a half written
  uint64_t* h_free = h_full + 2;                                            // [2] ... read
  uint64_t* act_full = h_free + 2;                                          // [2] a group's slice of activations stored
  uint64_t* act_free = act_full + 2;                                        // [2] ... multiplied
  uint64_t* y_full = act_free + 2;                                          // Y of a tile complete
  uint64_t* y_free = y_full + 1;                                            // ... read
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(y_free + 1);

  pdl_launch_dependents();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int side = blockIdx.y;
  const uint16_t* W1 = side ? w.W1V : w.W1K;
  const uint16_t* W2 = side ? w.W2V : w.W2K;
  float* sum_f32 = side ? v.vsum_f32 : v.ksum_f32;
  uint16_t* sum_b16 = side ? v.vsum_bf16 : v.ksum_bf16;

  // ---- one-time set-up -----------------------------------------------------------------------------
  for (int i = tid; !POOLED && i < d_sum * 16; i += MT_THREADS) {   // W1 [d_sum][128]: rows of 16 pieces, 2 K-blocks
    const int r = i >> 4, p = i & 15;
    cp_async16(W1s + (p >> 3) * (d_sum * umma::KBLOCK_ROW_BYTES) + umma::piece_offset(r, p & 7),
               reinterpret_cast<const uint4*>(W1 + (long long)r * D) + p, true);
  }
  const int w2_pieces = d_sum / 8;
  for (int i = tid; i < D * w2_pieces; i += MT_THREADS) {           // W2 [128][d_sum]: K-blocks of 16 KB
    const int r = i / w2_pieces, p = i - r * w2_pieces;
    cp_async16(W2s + (p >> 3) * MT_PLANE_KB_BYTES + umma::piece_offset(r, p & 7),
               reinterpret_cast<const uint4*>(W2 + (long long)r * d_sum) + p, true);
  }
  for (int i = tid; !POOLED && i < d_sum; i += MT_THREADS) b1s[i] = (side ? w.b1V : w.b1K)[i];
  for (int i = tid; i < D; i += MT_THREADS) b2s[i] = (side ? w.b2V : w.b2K)[i];
  if (warp == MT_MMA_WARP) umma::tmem_alloc(tmem_slot, MT_TMEM_COLS);
  if (tid == 0) {
    mbar_init(a_full, MT_IO_WARPS);
    mbar_init(a_free, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&h_full[i], 1);
      mbar_init(&h_free[i], MT_GELU_WARPS);
      mbar_init(&act_full[i], MT_GELU_WARPS / 2);
      mbar_init(&act_free[i], 1);
    }
    mbar_init(y_full, 1);
    mbar_init(y_free, MT_IO_WARPS);
    mbar_fence_init();
  }
  cp_async_wait_all();
  umma::fence_smem_to_async();
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tmem = *tmem_slot;

  pdl_wait();      // weights, barriers and tensor memory are set up; the chunk means come from the previous kernel
  int n_tiles = (n_units + MT_M - 1) / MT_M;
  if (dev_window >= 0) {      // one chunk per sequence, found on the device
    const NextChunk nx = next_chunk(v.n_listed, v.seq_len, v.C, dev_window, v.max_chunks);
    if (!nx.due) n_tiles = 0;
    t0 = nx.t;
  }
  const int my_tiles = n_tiles > (int)blockIdx.x ? (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
  const int n_halves = (d_sum + 127) / 128, n_slices = d_sum / MT_SLICE;
  auto summary_row = [&](int unit) -> long long {
    const int s = (int)by_range.div((uint32_t)unit);
    return (long long)s * v.max_chunks + t0 + (unit - s * n_range);
  };
  const uint32_t lane_bits = (uint32_t)((warp & 3) * 32) << 16;      // the tensor-memory lanes of this warp
  const int row = (warp & 3) * 32 + lane;                             // row of the tile = tensor-memory lane
  bool ok = true;

  if (warp < MT_GELU_WARPS) {
    // ================= activations =================
    const int group = warp >> 2;
    const uint32_t act = tmem + MT_TMEM_ACT + group * MT_ACT_COLS + lane_bits;
    int n_act = 0;                                        // slices of this group so far
    for (int k = 0; k < my_tiles && ok; ++k) {
      const int unit = (blockIdx.x + k * gridDim.x) * MT_M + row;
      for (int j = group; j < n_slices && ok; j += 2, ++n_act) {
        const int half = k * n_halves + (j >> 2), hb = half & 1;      // running number of the half, its accumulator
        if constexpr (!POOLED) {
          if ((j & 3) == group) ok = __all_sync(0xffffffffu, mbar_wait_bounded(&h_full[hb], (uint32_t)((half >> 1) & 1)));
          if (!ok) break;
          umma::fence_after_sync();
        }
        uint32_t p[3][16];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          float h[16];
          if constexpr (POOLED) {
            const float* src = hid + ((long long)side * n_units + unit) * d_sum + j * MT_SLICE + q * 16;
#pragma unroll
            for (int e = 0; e < 16; ++e) h[e] = 0.f;
            if (unit < n_units) {
              load8(src, reinterpret_cast<float(&)[8]>(h[0]), true);      // (workspace)
              load8(src + 8, reinterpret_cast<float(&)[8]>(h[8]), true);
            }
          } else {
            umma::tmem_ld16(tmem + hb * 128 + (j & 3) * MT_SLICE + q * 16 + lane_bits, h);
          }
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            float2 y = make_float2(h[2 * e], h[2 * e + 1]);
            if constexpr (!POOLED) y = gelu2(add2(y, *reinterpret_cast<const float2*>(b1s + j * MT_SLICE + q * 16 + 2 * e)));
            uint32_t s3[3];
            split3_pair(y.x, y.y, s3);
#pragma unroll
            for (int pl = 0; pl < 3; ++pl) p[pl][q * 8 + e] = s3[pl];
          }
        }
        if (!POOLED && (j + 2 >= n_slices || (j & 3) >= 2)) {      // this group's last slice of the half
          umma::fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&h_free[hb]);
        }
        // the group's slice before has been multiplied
        if (n_act > 0) ok = __all_sync(0xffffffffu, mbar_wait_bounded(&act_free[group], (uint32_t)((n_act - 1) & 1)));
        if (!ok) break;
        umma::fence_after_sync();
#pragma unroll
        for (int pl = 0; pl < 3; ++pl) umma::tmem_st16_nowait(act + pl * (MT_SLICE / 2), p[pl]);
        umma::tmem_st_wait();
        umma::fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&act_full[group]);
      }
    }
    if (!ok && lane == 0) set_status(v.status, ERR_TIMEOUT);
  } else if (warp < MT_MMA_WARP) {
    // ================= means in, summaries out =================
    const int c0 = ((warp - MT_GELU_WARPS) >> 2) * 64;      // this thread's 64 columns of its row: K-block c0 / 64
    const bool wide = (reinterpret_cast<uintptr_t>(sum_f32) & 31) == 0;      // the caller's buffer: 16 bytes are enough
    // a thread keeps its 32-byte column and walks down 8 rows, so that a warp's load covers whole rows
    const int io = tid - MT_GELU_WARPS * 32, pc = io & 15;
    for (int k = POOLED ? 0 : -1; k < my_tiles && ok; ++k) {      // round k: the means of tile k + 1 in, then the summaries of tile k out
      if (!POOLED && k + 1 < my_tiles) {
        const int unit0 = (blockIdx.x + (k + 1) * gridDim.x) * MT_M + (io >> 4);
        float x[8][8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int unit = unit0 + 16 * i;
#pragma unroll
          for (int e = 0; e < 8; ++e) x[i][e] = 0.f;
          if (unit < n_units) load8(sum_f32 + summary_row(unit) * D + pc * 8, x[i], wide);
        }
        if (k >= 0) ok = __all_sync(0xffffffffu, mbar_wait_bounded(a_free, (uint32_t)(k & 1)));
        if (!ok) break;
#pragma unroll
        for (int i = 0; i < 8; ++i)      // plane pl, K-block kb at (pl * 2 + kb) * 16 KB
          store_split8(x[i], As + (pc >> 3) * MT_PLANE_KB_BYTES + umma::piece_offset((io >> 4) + 16 * i, pc & 7), 2 * MT_PLANE_KB_BYTES);
        umma::fence_smem_to_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(a_full);
      }
      if (k < 0) continue;
      ok = __all_sync(0xffffffffu, mbar_wait_bounded(y_full, (uint32_t)(k & 1)));
      if (!ok) break;
      umma::fence_after_sync();
      float y[2][32];
      umma::tmem_ld32(tmem + MT_TMEM_Y + c0 + lane_bits, y[0]);
      umma::tmem_ld32(tmem + MT_TMEM_Y + c0 + 32 + lane_bits, y[1]);
      if constexpr (POOLED) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float lo[16];
          umma::tmem_ld16(tmem + MT_TMEM_YLO + c0 + 16 * q + lane_bits, lo);
#pragma unroll
          for (int e = 0; e < 16; ++e) y[q >> 1][(q & 1) * 16 + e] += lo[e];
        }
      }
      umma::fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(y_free);
      const int unit = (blockIdx.x + k * gridDim.x) * MT_M + row;
      if (unit < n_units) {
        const long long o = summary_row(unit) * D + c0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          float z[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) z[e] = y[q >> 2][(q & 3) * 8 + e] + b2s[c0 + q * 8 + e];
          store8(sum_f32 + o + q * 8, z, wide);
          *reinterpret_cast<uint4*>(sum_b16 + o + q * 8) =
              make_uint4(pack_bf16x2(z[0], z[1]), pack_bf16x2(z[2], z[3]), pack_bf16x2(z[4], z[5]), pack_bf16x2(z[6], z[7]));
        }
      }
    }
    if (!ok && lane == 0) set_status(v.status, ERR_TIMEOUT);
  } else if (lane == 0) {
    // ================= MMA issue (one thread) =================
    const uint32_t a_base = smem_u32(As), w1_base = smem_u32(W1s), w2_base = smem_u32(W2s);
    constexpr uint32_t idesc2 = umma::instr_desc_bf16(MT_M, D);
    const int n_l1 = POOLED ? 0 : my_tiles * n_halves, n_l2 = my_tiles * n_slices;
    int l1 = 0, l2 = 0, l1_tile = 0, l1_half = 0, l2_tile = 0, l2_slice = 0;
    uint32_t idle = 0;
    while (l2 < n_l2) {
      bool progress = false;
      // layer 1: a half of a tile's hidden units into accumulator l1 & 1, once that has been read
      if (l1 < n_l1 && mbar_test_wait(a_full, (uint32_t)(l1_tile & 1)) &&
          (l1 < 2 || mbar_test_wait(&h_free[l1 & 1], (uint32_t)(((l1 >> 1) - 1) & 1)))) {
        umma::fence_after_sync();
        const int width = d_sum - l1_half * 128 < 128 ? 64 : 128;
        const uint32_t idesc1 = umma::instr_desc_bf16(MT_M, width);
        bool acc = false;
#pragma unroll 1
        for (int pl = 2; pl >= 0; --pl)                 // smallest plane first
#pragma unroll 1
          for (int kb = 0; kb < 2; ++kb)
#pragma unroll
            for (int s = 0; s < 4; ++s) {
              umma::mma_bf16(tmem + (l1 & 1) * 128, umma::smem_desc(a_base + (pl * 2 + kb) * MT_PLANE_KB_BYTES + s * 32),
                             umma::smem_desc(w1_base + kb * (d_sum * umma::KBLOCK_ROW_BYTES) + l1_half * 128 * umma::KBLOCK_ROW_BYTES + s * 32), idesc1, acc);
              acc = true;
            }
        umma::commit(&h_full[l1 & 1]);
        ++l1;
        if (++l1_half == n_halves) { l1_half = 0; ++l1_tile; umma::commit(a_free); }
        progress = true;
      }
      // layer 2: 32 hidden units; the first slice of a tile overwrites Y, once that has been read
      if (mbar_test_wait(&act_full[l2_slice & 1], (uint32_t)(((l2_tile * n_slices + l2_slice) >> 1) & 1)) &&
          (l2_slice > 0 || l2_tile == 0 || mbar_test_wait(y_free, (uint32_t)((l2_tile - 1) & 1)))) {
        umma::fence_after_sync();
        const uint32_t act = tmem + MT_TMEM_ACT + (l2_slice & 1) * MT_ACT_COLS;
        const uint32_t wb = w2_base + (l2_slice >> 1) * MT_PLANE_KB_BYTES + (l2_slice & 1) * 64;
#pragma unroll 1
        for (int pl = 2; pl >= 0; --pl)
#pragma unroll
          for (int s = 0; s < 2; ++s)
            umma::mma_bf16_ts(tmem + (POOLED && pl ? MT_TMEM_YLO : MT_TMEM_Y), act + pl * (MT_SLICE / 2) + s * 8, umma::smem_desc(wb + s * 32),
                              idesc2, !(l2_slice == 0 && s == 0 && (pl == 2 || (POOLED && pl == 0))));
        umma::commit(&act_free[l2_slice & 1]);
        ++l2;
        if (++l2_slice == n_slices) { l2_slice = 0; ++l2_tile; umma::commit(y_full); }
        progress = true;
      }
      if (progress) idle = 0;
      else if (++idle > (1u << 24)) { set_status(v.status, ERR_TIMEOUT); break; }
      else if (idle > 4096) __nanosleep(64);
    }
  }

  umma::fence_before_sync();
  __syncthreads();
  if (warp == MT_MMA_WARP) umma::tmem_dealloc(tmem, MT_TMEM_COLS);
}

cudaError_t launch_pooled_out(const LayerView& v, int t0, int t1, const MlpWeights& w, int d_sum, const float* hid, cudaStream_t st) {
  const int n_range = t1 - t0;
  const long long n_units = (long long)v.S * n_range;
  if (d_sum % 64 != 0 || d_sum > MT_MAX_DSUM || n_units + MT_M >= (1LL << 31) || (long long)v.S * v.max_chunks >= (1LL << 31))
    return cudaErrorInvalidValue;
  static DeviceFlags opted;
  const cudaError_t e = smem_opt_in(opted, kve_chunk_mlp_tc_kernel<true>, MT_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const long long n_tiles = (n_units + MT_M - 1) / MT_M, half = sm_count() / 2;
  return launch_pdl(kve_chunk_mlp_tc_kernel<true>, dim3((unsigned)(n_tiles < half ? n_tiles : half), 2), dim3(MT_THREADS), MT_SMEM_BYTES, st, v,
                    t0, n_range, fast_div((uint32_t)n_range), (int)n_units, w, d_sum, -1, hid);
}

cudaError_t launch_chunk_mlp(const LayerView& v, int t0, int t1, const MlpWeights& w, int d_sum, cudaStream_t st, int dev_window) {
  const int n_range = dev_window >= 0 ? 1 : t1 - t0;
  const long long n_units = (long long)v.S * n_range;
  if (n_units <= 0) return cudaSuccess;
  if (d_sum % 64 == 0 && d_sum <= MT_MAX_DSUM && n_units + MT_M < (1LL << 31) &&
      (long long)v.S * v.max_chunks < (1LL << 31)) {
    static DeviceFlags opted_tc;
    {
      cudaError_t e = smem_opt_in(opted_tc, kve_chunk_mlp_tc_kernel<false>, MT_SMEM_BYTES);
      if (e != cudaSuccess) return e;
    }
    const long long n_tiles = (n_units + MT_M - 1) / MT_M;
    const long long half = sm_count() / 2;
    const long long per_side = n_tiles < half ? n_tiles : half;  // one CTA per SM: half of the SMs per side
    dim3 grid((unsigned)per_side, 2);
    return launch_pdl(kve_chunk_mlp_tc_kernel<false>, grid, dim3(MT_THREADS), MT_SMEM_BYTES, st, v, t0, n_range, fast_div((uint32_t)n_range), (int)n_units, w, d_sum, dev_window,
                      nullptr);
  }
  const size_t smem = sizeof(float) * (size_t)MLP_ROWS * (D + d_sum);
  static DeviceFlags opted;
  {
    cudaError_t e = smem_opt_in(opted, kve_chunk_mlp_kernel, (int)(sizeof(float) * MLP_ROWS * (D + 1024)));
    if (e != cudaSuccess) return e;
  }
  dim3 grid((unsigned)((n_units + MLP_ROWS - 1) / MLP_ROWS), 2);
  // Launched behind its predecessor, not beside it: its few CTAs then find SMs of their own (8 x 27 chunks, d_sum 512: 109 us, 74 so)
  kve_chunk_mlp_kernel<<<grid, dim3(MLP_THREADS), smem, st>>>(v, t0, n_range, n_units, w, d_sum, dev_window);
  return cudaGetLastError();
}

}  // namespace kve
