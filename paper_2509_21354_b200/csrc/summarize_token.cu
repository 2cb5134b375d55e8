// KVE_AGG_TOKEN_MLP: Eq. 2 with the MLP acting on every token of the chunk, the C outputs mean-pooled:
//   Kbar = (1/C) sum_j [ W2 gelu(W1 k_j + b1) + b2 ]  =  W2 [ (1/C) sum_j gelu(W1 k_j + b1) ] + b2
// (the last layer is affine and the mean is linear, so the activations are pooled and the second layer
// runs once per chunk, in summarize.cu).
//
//  kve_token_mlp_pool_kernel - the contraction W1 [d_sum, 128] x [128, tokens] over EVERY stale token on the
//    5th-generation tensor cores, activation and pooling in the epilogue, one pass over the stale KV.
//    * A CTA serves one side (keys or values) and keeps that side's W1 (d_sum x 128 bf16, K-major, 128-byte swizzle) in
//      shared memory: the A operand, in slabs of 128 hidden units.
//    * Tile = 128 consecutive tokens of one sequence's stale range (one or several whole chunks, or a
//      128-token slice of a longer chunk).  The token rows are bf16 already, so they are the B operand as
//      they stand: 16-byte asynchronous copies put a page's rows straight into the swizzled layout; 8 tcgen05.mma
//      (M 128, N 128, K 16 each) per slab accumulate the pre-activations in tensor memory, hidden unit = lane,
//      token = column.  A thread of the sixteen warps therefore holds many tokens of ONE hidden unit: its bias is a
//      constant, and the sum over a chunk's tokens stays in registers.  (With tokens as lanes the same kernel needed 31
//      shuffles and as many selects per 32 activations, a bias load each and an atomic per sum: 38 instructions per
//      activation, 690 us for 256 sequences x 56 chunks x 64 tokens x 2 sides x 256 units; now MEASURED.)
//    * Two token buffers and two accumulators, one CTA-wide barrier per tile: behind it the tensor core works on tile i + 1 and
//      the copies of tile i + 2 are under way while the warps go through tile i.
//    * The pooled activations (1/C) sum_j gelu(...) go to a scratch row per (side, sequence, chunk).
//    Bound by the activation arithmetic (14 fp32 operations, 4 of the integer pipe and an exponential per activation).
// The only wait (on the MMA commit) is bounded; on give-up the status word gets KVE_ERR_TIMEOUT.
#include "common.cuh"
#include "kernels.h"
#include "umma.cuh"
#include "gelu.cuh"

namespace kve {

constexpr int TM_N = 128;                                   // tokens per tile
constexpr int TM_SLAB = 128;                                // hidden units per MMA
constexpr int TM_THREADS = 512;                             // 16 warps: four per scheduler hide the latency of the activation chains
constexpr int TM_MAX_DSUM = 256;
constexpr int TM_KB_BYTES = TM_N * umma::KBLOCK_ROW_BYTES;  // 16 KB: 128 rows x 64 head dims
constexpr int TM_SMEM_W1 = 0;                               // 2 K-blocks of [d_sum rows][64]: up to 64 KB
constexpr int TM_SMEM_X = TM_SMEM_W1 + 2 * TM_MAX_DSUM * umma::KBLOCK_ROW_BYTES;   // 2 buffers x 2 K-blocks: 64 KB
constexpr int TM_SMEM_POOL = TM_SMEM_X + 2 * 2 * TM_KB_BYTES;          // [2 tile parities][4 groups of 32 tokens][d_sum] sums
constexpr int TM_SMEM_BAR = TM_SMEM_POOL + 2 * 4 * TM_MAX_DSUM * 4;
constexpr int TM_SMEM_BYTES = TM_SMEM_BAR + 32 + 1024;      // + slack to reach a 1024-byte boundary
constexpr int TM_TMEM_COLS = 512;                           // two accumulators of up to two slabs x 128 columns
static_assert(TM_SMEM_BYTES > 116 * 1024, "one CTA per SM: each allocates all of tensor memory");

struct TokenMlpArgs {
  LayerView v;
  int t0, n_range;           // chunks [t0, t0 + n_range) of every sequence
  FastDiv by_range;
  int tiles_per_item;        // max(1, C / 128): 128-token tiles of one chunk
  int units_per_item;        // max(1, 128 / C): chunks in one tile
  int n_units, n_items;
  MlpWeights w;
  float* hid;                // [2][n_units][d_sum] pooled activations (side, unit = s * n_range + (t - t0))
};

template <int DSUM>
__global__ void __launch_bounds__(TM_THREADS, 1) kve_token_mlp_pool_kernel(TokenMlpArgs a) {
  constexpr int SLABS = DSUM / TM_SLAB;
  constexpr int COLS = TM_N * SLABS / 4;       // tokens a thread goes through per tile: 64 or 32
  constexpr int GROUPS = COLS / 32;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* W1s = smem + TM_SMEM_W1;
  unsigned char* Xs = smem + TM_SMEM_X;
  float* pool = reinterpret_cast<float*>(smem + TM_SMEM_POOL);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + TM_SMEM_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + TM_SMEM_BAR + 8);

  pdl_launch_dependents();
  const LayerView& v = a.v;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int side = blockIdx.y;
  const uint16_t* W1 = side ? a.w.W1V : a.w.W1K;
  const uint16_t* pages = side ? v.v_pages : v.k_pages;

  // ---- one-time set-up: W1 of this side, tensor memory, barrier --------------------------------------------
  for (int i = tid; i < DSUM * 16; i += TM_THREADS) {              // W1 [DSUM][128]: rows of 16 pieces, 2 K-blocks
    const int r = i >> 4, p = i & 15;
    cp_async16(W1s + (p >> 3) * (DSUM * umma::KBLOCK_ROW_BYTES) + umma::piece_offset(r, p & 7),
               reinterpret_cast<const uint4*>(W1 + (long long)r * D) + p, true);
  }
  if (warp == 0) umma::tmem_alloc(tmem_slot, TM_TMEM_COLS);
  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_fence_init();
  }
  const uint32_t x_base = smem_u32(Xs), w1_base = smem_u32(W1s);
  constexpr uint32_t idesc = umma::instr_desc_bf16(TM_SLAB, TM_N);

  // this thread's hidden unit and tokens: tensor-memory lane 32 (warp & 3) + lane of slab `slab`, columns [col0, col0 + COLS)
  const int lg = warp & 3, quarter = warp >> 2;
  const int slab = SLABS == 2 ? quarter >> 1 : 0, col0 = (SLABS == 2 ? quarter & 1 : quarter) * COLS;
  const int unit = slab * TM_SLAB + lg * 32 + lane;
  const float b1_scaled = (side ? a.w.b1V : a.w.b1K)[unit] * GELU_SCALE;
  const uint32_t tmem_off = (uint32_t)(slab * TM_N + col0) + ((uint32_t)(lg * 32) << 16);

  // A CTA walks whole items (a chunk longer than a tile keeps all its 128-token slices on one CTA, in a row).  What this
  // thread copies of a tile: the 16-byte piece p of the rows r0 + 32 i.
  const int p16 = tid & 15, r0 = tid >> 4;
  int src_item = blockIdx.x, src_slice = 0;                         // the tile the next look-up is for
  int page[TM_N / 32], page_slice = 0;                              // its pages (-1: no row) and slice
  auto look_up = [&]() {
#pragma unroll
    for (int i = 0; i < TM_N / 32; ++i) {
      const int r = r0 + 32 * i;
      const int u_in = a.units_per_item > 1 ? r / v.C : 0;
      const int u = src_item * a.units_per_item + u_in;
      page[i] = -1;
      if (src_item < a.n_items && u < a.n_units) {
        const int s = (int)a.by_range.div((uint32_t)u);
        const int t = a.t0 + (u - s * a.n_range);
        page[i] = max(v.page_table[(long long)s * v.max_chunks + t], -2);      // below -1: a bad entry, flagged when it is used
        if (page[i] == -1) page[i] = -2;
      }
    }
    page_slice = src_slice;
    if (++src_slice == a.tiles_per_item) { src_slice = 0; src_item += gridDim.x; }
  };
  // copies of the tile looked up last, zeros where there is no row
  auto gather = [&](int buf) {
    unsigned char* dst0 = Xs + buf * 2 * TM_KB_BYTES + (p16 >> 3) * TM_KB_BYTES;
#pragma unroll
    for (int i = 0; i < TM_N / 32; ++i) {
      const int r = r0 + 32 * i;
      const bool live = page[i] >= 0 && page[i] < v.n_pages;
      if (!live && page[i] != -1) set_status(v.status, ERR_CAPACITY);
      const int r_in = (a.units_per_item > 1 ? r % v.C : r) + page_slice * TM_N;
      cp_async16(dst0 + umma::piece_offset(r, p16 & 7), pages + (live ? ((long long)page[i] * v.C + r_in) * D : 0) + p16 * 8, live);
    }
  };
  auto issue_mma = [&](uint32_t tmem_acc, int buf) {
    umma::fence_after_sync();
#pragma unroll
    for (int sl = 0; sl < SLABS; ++sl)
#pragma unroll
      for (int kb = 0; kb < 2; ++kb)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          umma::mma_bf16(tmem_acc + sl * TM_N, umma::smem_desc(w1_base + kb * (DSUM * umma::KBLOCK_ROW_BYTES) + sl * (TM_SLAB * umma::KBLOCK_ROW_BYTES) + k * 32),
                         umma::smem_desc(x_base + (buf * 2 + kb) * TM_KB_BYTES + k * 32), idesc, (kb | k) != 0);
    umma::commit(bar);
  };
  // the finished sums of a tile (its last slice): pooled activations out
  const float inv_c = 1.f / (float)v.C;
  const int groups_per_chunk = (v.C < TM_N ? v.C : TM_N) / 32;
  auto write_pooled = [&](int item, int parity) {
    const float* pl = pool + parity * 4 * TM_MAX_DSUM;
    for (int i = tid; i < a.units_per_item * DSUM; i += TM_THREADS) {
      const int u_in = i / DSUM, col = i - u_in * DSUM, u = item * a.units_per_item + u_in;
      float sum = 0.f;
      for (int g = 0; g < groups_per_chunk; ++g) sum += pl[(u_in * groups_per_chunk + g) * TM_MAX_DSUM + col];
      if (u < a.n_units) a.hid[((long long)side * a.n_units + u) * DSUM + col] = sum * inv_c;
    }
  };

  pdl_wait();      // W1 is on its way; the pages come from earlier kernels
  const int my_items = a.n_items > (int)blockIdx.x ? (a.n_items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
  const long long n_tiles = (long long)my_items * a.tiles_per_item;      // of this CTA
  look_up();
  if (n_tiles > 0) gather(0);
  look_up();
  cp_async_wait_all();
  umma::fence_smem_to_async();
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tmem_d = *tmem_slot;
  if (n_tiles > 0 && tid == 0) issue_mma(tmem_d, 0);
  if (n_tiles > 1) gather(1);
  look_up();

  float2 relu_sum[GROUPS], tail_sum[GROUPS];      // per 32 tokens: sum of max(u, 0) and of the tails
#pragma unroll
  for (int g = 0; g < GROUPS; ++g) relu_sum[g] = tail_sum[g] = make_float2(0.f, 0.f);
  int item = blockIdx.x, slice = 0, done_item = -1;      // done_item: its sums wait in the other parity's pool
  for (long long tile = 0; tile < n_tiles; ++tile) {
    const int sel = (int)(tile & 1);
    const bool ok = mbar_wait_bounded(bar, (uint32_t)sel);      // this tile's MMAs are done: its token buffer is free
    cp_async_wait_all();                                        // the next tile's rows are in place
    umma::fence_smem_to_async();
    umma::fence_before_sync();
    if (__syncthreads_or(!ok)) {      // also: the other accumulator and the other pool were left a tile ago
      if (tid == 0) set_status(v.status, ERR_TIMEOUT);
      break;
    }
    umma::fence_after_sync();
    if (tile + 1 < n_tiles && tid == 0) issue_mma(tmem_d + (uint32_t)(sel ^ 1) * (SLABS * TM_N), sel ^ 1);
    if (tile + 2 < n_tiles) {
      gather(sel);
      look_up();      // the page ids arrive while this tile is worked through
    }
    if (done_item >= 0) write_pooled(done_item, sel ^ 1);
    done_item = -1;
#pragma unroll
    for (int g = 0; g < GROUPS; ++g) {
      float h[32];
      umma::tmem_ld32(tmem_d + (uint32_t)sel * (SLABS * TM_N) + tmem_off + (uint32_t)(g * 32), h);
#pragma unroll
      for (int e = 0; e < 32; e += 2) {
        float2 relu, ea;
        const float2 u = fma2(make_float2(h[e], h[e + 1]), make_float2(GELU_SCALE, GELU_SCALE), make_float2(b1_scaled, b1_scaled));
        const float2 p = gelu_tail2(u, relu, ea);
        tail_sum[g] = fma2(ea, p, tail_sum[g]);
        relu_sum[g] = add2(relu_sum[g], relu);
      }
    }
    if (++slice == a.tiles_per_item) {      // the chunk(s) of this item are complete
#pragma unroll
      for (int g = 0; g < GROUPS; ++g) {
        pool[(sel * 4 + col0 / 32 + g) * TM_MAX_DSUM + unit] = (relu_sum[g].x + relu_sum[g].y) * (1.f / GELU_SCALE) - (tail_sum[g].x + tail_sum[g].y);
        relu_sum[g] = tail_sum[g] = make_float2(0.f, 0.f);
      }
      done_item = item;
      slice = 0;
      item += gridDim.x;
    }
  }
  umma::fence_before_sync();
  __syncthreads();
  if (done_item >= 0) write_pooled(done_item, (int)((n_tiles - 1) & 1));
  if (warp == 0) umma::tmem_dealloc(tmem_d, TM_TMEM_COLS);
}

bool token_mlp_supported(int C, int d_sum) {
  if (d_sum <= 0 || d_sum % 128 != 0 || d_sum > TM_MAX_DSUM) return false;      // the epilogue hands out 32-column groups
  if (C < 32 || C % 32 != 0) return false;
  return C <= 128 ? (128 % C == 0) : (C % 128 == 0);
}

template <int DSUM>
static cudaError_t launch_pool(const TokenMlpArgs& a, dim3 grid, cudaStream_t st) {
  static DeviceFlags opted;
  const cudaError_t e = smem_opt_in(opted, kve_token_mlp_pool_kernel<DSUM>, TM_SMEM_BYTES);
  return e == cudaSuccess ? launch_pdl(kve_token_mlp_pool_kernel<DSUM>, grid, dim3(TM_THREADS), TM_SMEM_BYTES, st, a) : e;
}

cudaError_t launch_chunk_token_mlp(const LayerView& v, int t0, int t1, const MlpWeights& w, int d_sum, float* hid, cudaStream_t st) {
  const int n_range = t1 - t0;
  const long long n_units = (long long)v.S * n_range;
  if (n_units <= 0) return cudaSuccess;
  if (!token_mlp_supported(v.C, d_sum) || n_units >= (1LL << 31)) return cudaErrorInvalidValue;
  TokenMlpArgs a;
  a.v = v; a.t0 = t0; a.n_range = n_range; a.by_range = fast_div((uint32_t)n_range);
  a.tiles_per_item = v.C > TM_N ? v.C / TM_N : 1;
  a.units_per_item = v.C < TM_N ? TM_N / v.C : 1;
  a.n_units = (int)n_units;
  a.n_items = (a.n_units + a.units_per_item - 1) / a.units_per_item;
  a.w = w; a.hid = hid;
  // one CTA per SM, half of the SMs per side; a CTA walks whole items (all 128-token slices of a chunk in a row)
  long long per_side = sm_count() / 2;
  if (per_side > a.n_items) per_side = a.n_items;
  if (per_side < 1) per_side = 1;
  const dim3 grid((unsigned)per_side, 2);
  const cudaError_t e = d_sum == 256 ? launch_pool<256>(a, grid, st) : launch_pool<128>(a, grid, st);
  return e == cudaSuccess ? launch_pooled_out(v, t0, t1, w, d_sum, hid, st) : e;
}

}  // namespace kve
