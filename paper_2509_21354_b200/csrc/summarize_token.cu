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
//      activation, 690 us for 256 sequences x 56 chunks x 64 tokens x 2 sides x 256 units; 250 us so.)
//    * Warp roles around a ring of four token buffers and two accumulators (four with 128 hidden units): four copy warps (two tiles under
//      way behind the newest), one MMA thread, sixteen epilogue warps.  With two buffers and one CTA-wide barrier per tile the kernel took 522 us
//      where it now takes 223.
//    * Each accumulator has epilogue warps of its own, and a thread goes through all 128 tokens of its hidden unit: one hand-over, one first load
//      from tensor memory per 128 activations, no sums that meet in shared memory.  (All sixteen warps on every tile, 64 or 32 tokens a
//      thread: 256 sequences x 56 chunks x 64 tokens x 256 units 254 us with the second layer, 238 so; 128 units 160 and 145 us; 64 x 30 x 128
//      tokens 82 and 75 us.)  Items (chunks or groups of chunks) go through the accumulators in turn, so that the slices of a long chunk
//      stay with the same threads.  A CTA with few items has all sixteen warps on every tile all the same (SHARED): the bits are those of the other
//      way, the sums of 32 tokens are added up in the same order.
//    * The exponentials of eight tokens are taken beside the polynomial of the next eight.
//    * The pooled activations (1/C) sum_j gelu(...) go to a scratch row per (side, sequence, chunk).
//    Bound by the activation arithmetic: 20 issue slots per pair of activations (18.6 cycles of the fp32 pipe, 16 of the exponentials'), 65 %
//    of the schedulers' slots used.
// Every mbarrier wait is bounded; on give-up the status word gets KVE_ERR_TIMEOUT.
#include "common.cuh"
#include "kernels.h"
#include "umma.cuh"
#include "gelu.cuh"

namespace kve {

constexpr int TM_N = 128;                                   // tokens per tile
constexpr int TM_SLAB = 128;                                // hidden units per MMA
constexpr int TM_EPI_WARPS = 16;                            // four per scheduler hide the latency of the activation chains
constexpr int TM_COPY_WARPS = 4;
constexpr int TM_MMA_WARP = TM_EPI_WARPS + TM_COPY_WARPS;
constexpr int TM_THREADS = (TM_MMA_WARP + 1) * 32;
constexpr int TM_MAX_DSUM = 256;
constexpr int TM_KB_BYTES = TM_N * umma::KBLOCK_ROW_BYTES;  // 16 KB: 128 rows x 64 head dims
constexpr int TM_SMEM_W1 = 0;                               // 2 K-blocks of [d_sum rows][64]: up to 64 KB
constexpr int TM_XBUFS = 4;                                  // token buffers
constexpr int TM_LAG = 2;                                    // tiles whose copies are under way behind the newest
constexpr int TM_SMEM_X = TM_SMEM_W1 + 2 * TM_MAX_DSUM * umma::KBLOCK_ROW_BYTES;   // 4 buffers x 2 K-blocks: 128 KB
constexpr int TM_TMEM_COLS = 512;                           // accumulators: one slab x 128 columns (four) or two (two)
constexpr int TM_MAX_ACC = TM_TMEM_COLS / TM_N;
constexpr int TM_SMEM_POOL = TM_SMEM_X + TM_XBUFS * 2 * TM_KB_BYTES;          // [2 items][4 groups of 32 tokens][d_sum] sums
constexpr int TM_SMEM_BAR = TM_SMEM_POOL + 2 * 4 * TM_MAX_DSUM * 4;
constexpr int TM_SMEM_BYTES = TM_SMEM_BAR + (2 * TM_XBUFS + 2 * TM_MAX_ACC) * 8 + 16 + 1024;      // + slack to reach a 1024-byte boundary
static_assert(TM_SMEM_BYTES > 116 * 1024, "one CTA per SM: each allocates all of tensor memory");

struct TokenMlpArgs {
  LayerView v;
  int t0, n_range;           // chunks [t0, t0 + n_range) of every sequence
  FastDiv by_range;
  int tiles_per_item;        // max(1, C / 128): 128-token tiles of one chunk
  int units_per_item;        // max(1, 128 / C): chunks in one tile
  int n_units, n_items;
  int list_cut;              // >= 0: the keep list covers no more than that from now on
  MlpWeights w;
  float* hid;                // [2][n_units][d_sum] pooled activations (side, unit = s * n_range + (t - t0))
};

// The order in which a CTA goes through its tiles.  Items side by side, as many as there are accumulators, slice by slice; or (SHARED) one item
// after the other, the accumulators in turn.
template <int ACCS, bool SHARED>
struct TileWalk {
  int my_items, tiles_per_item;      // items of this CTA: blockIdx.x + k gridDim.x
  int k0 = 0, slice = 0, acc = 0;    // this tile: slice `slice` of item k0 + acc (SHARED: k0), in accumulator `acc`
  int turns = 0;                     // SHARED: completed rounds through the accumulators
  __device__ __forceinline__ bool done() const { return k0 >= my_items; }
  __device__ __forceinline__ int item() const { return (int)blockIdx.x + (SHARED ? k0 : k0 + acc) * (int)gridDim.x; }
  __device__ __forceinline__ int turn() const { return SHARED ? turns : k0 / ACCS * tiles_per_item + slice; }      // of the accumulator: 0, 1, ..
  __device__ __forceinline__ void next() {
    if constexpr (SHARED) {
      if (++acc == ACCS) { acc = 0; ++turns; }
      if (++slice < tiles_per_item) return;
      slice = 0;
      ++k0;
    } else {
      if (++acc < ACCS && k0 + acc < my_items) return;
      acc = 0;
      if (++slice < tiles_per_item) return;
      slice = 0;
      k0 += ACCS;
    }
  }
};

// The activations of GROUPS x 32 tokens (columns from `cols` on) of a thread's hidden unit, added to `sum` 32 by 32; frees the accumulator.
template <int GROUPS>
__device__ __forceinline__ void pool_tile(uint32_t cols, float b1, float (&sum)[GROUPS], uint64_t* acc_free) {
  constexpr float G6[7] = KVE_GELU_TAIL6;
  umma::fence_after_sync();
  uint32_t h[2][16];                              // 16 columns in work, 16 on their way
  umma::tmem_ld16_nowait(cols, h[0]);
#pragma unroll
  for (int g = 0; g < GROUPS; ++g) {
    // 32 tokens, eight at a time; the exponentials of the block before go out between the polynomial steps of this one
    float2 relu_sum = make_float2(0.f, 0.f), tail_sum = make_float2(0.f, 0.f), abs_before[4], p_before[4];
#pragma unroll
    for (int blk = 0; blk <= 4; ++blk) {
      float2 abs_x[4], p[4];
      if (blk < 4) {
        const int q = blk >> 1;
        if (blk % 2 == 0) {
          umma::tmem_ld_wait16(h[q]);
          if (blk == 0 || g < GROUPS - 1) umma::tmem_ld16_nowait(cols + (uint32_t)(g * 32 + (q + 1) * 16), h[q ^ 1]);
          else {
            umma::fence_before_sync();
            __syncwarp();
            if ((threadIdx.x & 31) == 0) mbar_arrive(acc_free);
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int e = (blk & 1) * 8 + 2 * i;
          const float2 x = add2(make_float2(__uint_as_float(h[q][e]), __uint_as_float(h[q][e + 1])), make_float2(b1, b1));
          abs_x[i] = make_float2(fminf(fabsf(x.x), 6.f), fminf(fabsf(x.y), 6.f));
          relu_sum = add2(relu_sum, make_float2(relu_nan(x.x), relu_nan(x.y)));
          p[i] = make_float2(G6[6], G6[6]);
        }
      }
      float2 tail[4];
#pragma unroll
      for (int y = 0; y < 8; ++y) {      // an exponential of the block before, three steps of this one
        if (blk > 0) {
          if (y & 1) tail[y >> 1].y = ex2_fast(p_before[y >> 1].y);
          else tail[y >> 1].x = ex2_fast(p_before[y >> 1].x);
        }
        if (blk < 4)
#pragma unroll
          for (int z = 3 * y; z < 3 * y + 3; ++z) p[z & 3] = fma2(p[z & 3], abs_x[z & 3], make_float2(G6[5 - z / 4], G6[5 - z / 4]));
      }
      if (blk > 0)
#pragma unroll
        for (int i = 0; i < 4; ++i) tail_sum = fma2(abs_before[i], tail[i], tail_sum);
#pragma unroll
      for (int i = 0; i < 4; ++i) { abs_before[i] = abs_x[i]; p_before[i] = p[i]; }
    }
    const float got = (relu_sum.x + relu_sum.y) - (tail_sum.x + tail_sum.y);
    sum[g] += got;
  }
}

template <int DSUM, bool SHARED>
__global__ void __launch_bounds__(TM_THREADS, 1) kve_token_mlp_pool_kernel(TokenMlpArgs a) {
  constexpr int SLABS = DSUM / TM_SLAB;
  constexpr int ACCS = TM_TMEM_COLS / (TM_N * SLABS);          // accumulators, each with its own epilogue warps
  constexpr int ACC_WARPS = TM_EPI_WARPS / ACCS;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* W1s = smem + TM_SMEM_W1;
  unsigned char* Xs = smem + TM_SMEM_X;
  uint64_t* x_full = reinterpret_cast<uint64_t*>(smem + TM_SMEM_BAR);      // [4] token buffer filled by the copy warps
  uint64_t* x_free = x_full + TM_XBUFS;                                     // [4] token buffer read (MMA commit)
  uint64_t* acc_full = x_free + TM_XBUFS;                                   // [ACCS] accumulator written (MMA commit)
  uint64_t* acc_free = acc_full + TM_MAX_ACC;                               // [ACCS] accumulator read by its epilogue warps
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_free + TM_MAX_ACC);

  pdl_launch_dependents();
  const LayerView& v = a.v;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int side = blockIdx.y;

  // ---- one-time set-up: W1 of this side, tensor memory, barriers -------------------------------------------
  const uint16_t* W1 = side ? a.w.W1V : a.w.W1K;
  for (int i = tid; i < DSUM * 16; i += TM_THREADS) {              // W1 [DSUM][128]: rows of 16 pieces, 2 K-blocks
    const int r = i >> 4, p = i & 15;
    cp_async16(W1s + (p >> 3) * (DSUM * umma::KBLOCK_ROW_BYTES) + umma::piece_offset(r, p & 7),
               reinterpret_cast<const uint4*>(W1 + (long long)r * D) + p, true);
  }
  if (warp == TM_MMA_WARP) umma::tmem_alloc(tmem_slot, TM_TMEM_COLS);
  if (tid == 0) {
    for (int i = 0; i < TM_XBUFS; ++i) {
      mbar_init(&x_full[i], TM_COPY_WARPS * 32);
      mbar_init(&x_free[i], 1);
    }
    for (int i = 0; i < ACCS; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_free[i], SHARED ? TM_EPI_WARPS : ACC_WARPS);
    }
    mbar_fence_init();
  }
  cp_async_wait_all();
  umma::fence_smem_to_async();
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tmem_d = *tmem_slot;
  pdl_wait();      // the pages come from earlier kernels
  if (a.list_cut >= 0 && blockIdx.x == 0 && side == 0 && tid == 0) *v.n_listed = a.list_cut;

  // A CTA walks whole items (a chunk longer than a tile keeps all its 128-token slices on one CTA, in a row)
  const int my_items = a.n_items > (int)blockIdx.x ? (a.n_items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
  const int n_tiles = my_items * a.tiles_per_item;      // of this CTA
  TileWalk<ACCS, SHARED> walk{my_items, a.tiles_per_item};
  const int chunk_shift = v.C >= TM_N ? 7 : (v.C == 64 ? 6 : 5);      // row r of a tile: chunk r >> chunk_shift

  if (warp >= TM_EPI_WARPS && warp < TM_MMA_WARP) {
    // ================= copy warps: the tile's rows into the swizzled layout =================
    const int ct = tid - TM_EPI_WARPS * 32, p16 = ct & 15, r0 = ct >> 4;      // the 16-byte piece p16 of the rows r0 + 8 i
    const uint16_t* pages = (side ? v.v_pages : v.k_pages) + p16 * 8;
    unsigned char* dst0 = Xs + (p16 >> 3) * TM_KB_BYTES;
    int page[4];                                       // of the (up to four) chunks of the tile to come, looked up a tile ahead
    auto look_up = [&]() {
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int u = walk.item() * a.units_per_item + x;
        page[x] = -1;
        if (x < a.units_per_item && !walk.done() && u < a.n_units) {
          const int s = (int)a.by_range.div((uint32_t)u);
          page[x] = v.page_table[(long long)s * v.max_chunks + a.t0 + (u - s * a.n_range)];
        }
      }
    };
    look_up();
    bool ok = true;
    for (int tile = 0; tile < n_tiles + TM_LAG && ok; ++tile) {
      if (tile < n_tiles) {
        const int buf = tile % TM_XBUFS;
        if (tile >= TM_XBUFS) ok = mbar_wait_bounded(&x_free[buf], (uint32_t)((tile / TM_XBUFS - 1) & 1));
        long long src[4];                              // element offset of the first row taken from each chunk; -1: zeros
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const bool live = page[x] >= 0 && page[x] < v.n_pages;
          if (!live && x < a.units_per_item && walk.item() * a.units_per_item + x < a.n_units) set_status(v.status, ERR_CAPACITY);
          src[x] = live ? ((long long)page[x] * v.C + walk.slice * TM_N) * D : -1;
        }
        walk.next();
        look_up();
#pragma unroll
        for (int i = 0; i < TM_N / 8; ++i) {
          const long long base = chunk_shift == 7 ? src[0] : (chunk_shift == 6 ? src[i >> 3] : src[i >> 2]);
          const int r = r0 + 8 * i, r_in = r & ((1 << chunk_shift) - 1);
          cp_async16(dst0 + buf * 2 * TM_KB_BYTES + umma::piece_offset(r, p16 & 7), pages + (base < 0 ? 0 : base + r_in * D), base >= 0);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");      // (an empty group at the end keeps the count)
      if (tile >= TM_LAG) {
        asm volatile("cp.async.wait_group %0;" ::"n"(TM_LAG) : "memory");
        umma::fence_smem_to_async();
        mbar_arrive(&x_full[(tile - TM_LAG) % TM_XBUFS]);
      }
    }
    if (!ok) set_status(v.status, ERR_TIMEOUT);
    cp_async_wait_all();
  } else if (warp == TM_MMA_WARP) {
    // ================= MMA issue (one thread) =================
    if (lane == 0) {
      constexpr uint32_t idesc = umma::instr_desc_bf16(TM_SLAB, TM_N);
      const uint32_t x_base = smem_u32(Xs), w1_base = smem_u32(W1s);
      for (int tile = 0; tile < n_tiles; ++tile, walk.next()) {
        const int buf = walk.acc, turn = walk.turn(), xb = tile % TM_XBUFS;
        if (!mbar_wait_bounded(&x_full[xb], (uint32_t)((tile / TM_XBUFS) & 1)) ||
            (turn > 0 && !mbar_wait_bounded(&acc_free[buf], (uint32_t)((turn - 1) & 1)))) {
          set_status(v.status, ERR_TIMEOUT);
          break;
        }
        umma::fence_after_sync();
#pragma unroll
        for (int sl = 0; sl < SLABS; ++sl)
#pragma unroll
          for (int kb = 0; kb < 2; ++kb)
#pragma unroll
            for (int k = 0; k < 4; ++k)
              umma::mma_bf16(tmem_d + (uint32_t)(buf * SLABS + sl) * TM_N,
                             umma::smem_desc(w1_base + kb * (DSUM * umma::KBLOCK_ROW_BYTES) + sl * (TM_SLAB * umma::KBLOCK_ROW_BYTES) + k * 32),
                             umma::smem_desc(x_base + (xb * 2 + kb) * TM_KB_BYTES + k * 32), idesc, (kb | k) != 0);
        umma::commit(&x_free[xb]);
        umma::commit(&acc_full[buf]);
      }
    }
  } else {
    // ================= epilogue warps =================
    // this thread's hidden unit: tensor-memory lane 32 (warp & 3) + lane of slab `slab`.  All 128 tokens of the tiles in accumulator
    // warp / ACC_WARPS, or (SHARED) that share of the tokens of every tile
    const int buf = warp / ACC_WARPS, lg = warp & 3, slab = SLABS == 2 ? (warp >> 2) & 1 : 0;
    const int unit = slab * TM_SLAB + lg * 32 + lane;
    const float b1 = (side ? a.w.b1V : a.w.b1K)[unit];
    const uint32_t lanes = tmem_d + ((uint32_t)(lg * 32) << 16);
    const float inv_c = 1.f / (float)v.C;
    if constexpr (SHARED) {
      constexpr int GROUPS = TM_N / 32 / ACCS;
      float* pool = reinterpret_cast<float*>(smem + TM_SMEM_POOL);      // [2][4][DSUM]: the sums of 32 tokens each of an item
      float* hid = a.hid + (long long)side * a.n_units * DSUM;
      const int unit_shift = a.units_per_item == 4 ? 0 : (a.units_per_item == 2 ? 1 : 2), unit_groups = 1 << unit_shift;      // sums that make up a chunk
      bool alive = true;      // a warp whose wait ran out goes on without: the others meet it at the barrier below
      int acc = 0, turn = 0;
      for (int k = 0; k < my_items; ++k) {
        float sum[GROUPS];
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) sum[g] = 0.f;
        for (int slice = 0; slice < a.tiles_per_item; ++slice) {
          if (alive && !__all_sync(0xffffffffu, mbar_wait_bounded(&acc_full[acc], (uint32_t)(turn & 1)))) {
            alive = false;
            if (lane == 0) set_status(v.status, ERR_TIMEOUT);
          }
          if (alive) pool_tile<GROUPS>(lanes + (uint32_t)((acc * SLABS + slab) * TM_N + buf * GROUPS * 32), b1, sum, &acc_free[acc]);
          if (++acc == ACCS) { acc = 0; ++turn; }
        }
        const int first = ((int)blockIdx.x + k * (int)gridDim.x) * a.units_per_item;
        if (unit_groups <= GROUPS) {      // whole chunks
#pragma unroll
          for (int g = 0; g < GROUPS; ++g) {
            if (g & (unit_groups - 1)) continue;
            const int u = first + ((buf * GROUPS + g) >> unit_shift);
            if (u < a.n_units) hid[(long long)u * DSUM + unit] = (unit_groups == 2 ? sum[g] + sum[(g + 1) % GROUPS] : sum[g]) * inv_c;
          }
          continue;
        }
        float* pl = pool + (k & 1) * 4 * DSUM;
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) pl[(buf * GROUPS + g) * DSUM + unit] = sum[g];
        asm volatile("bar.sync 1, %0;" ::"n"(TM_EPI_WARPS * 32) : "memory");      // the other half keeps the next item apart
        for (int i = tid; i < a.units_per_item * DSUM; i += TM_EPI_WARPS * 32) {
          const int x = i / DSUM, col = i % DSUM;
          float total = pl[(x << unit_shift) * DSUM + col];
          for (int g = 1; g < unit_groups; ++g) total += pl[((x << unit_shift) + g) * DSUM + col];
          if (first + x < a.n_units) hid[(long long)(first + x) * DSUM + col] = total * inv_c;
        }
      }
    } else {
      const uint32_t cols = lanes + (uint32_t)((buf * SLABS + slab) * TM_N);
      float* hid = a.hid + (long long)side * a.n_units * DSUM + unit;
      int turn = 0;
      for (int k = buf; k < my_items; k += ACCS) {
        float sum[4] = {0.f, 0.f, 0.f, 0.f};              // per 32 tokens (of all slices of a long chunk)
        bool alive = true;
        for (int slice = 0; slice < a.tiles_per_item && alive; ++slice, ++turn) {
          alive = __all_sync(0xffffffffu, mbar_wait_bounded(&acc_full[buf], (uint32_t)(turn & 1)));
          if (!alive) {
            if (lane == 0) set_status(v.status, ERR_TIMEOUT);
            break;
          }
          pool_tile<4>(cols, b1, sum, &acc_free[buf]);
        }
        if (!alive) break;
        // the chunk(s) of this item are complete
        const int first = ((int)blockIdx.x + k * (int)gridDim.x) * a.units_per_item;
        if (a.units_per_item == 1) {
          hid[(long long)first * DSUM] = (((sum[0] + sum[1]) + sum[2]) + sum[3]) * inv_c;
        } else if (a.units_per_item == 2) {
          if (first < a.n_units) hid[(long long)first * DSUM] = (sum[0] + sum[1]) * inv_c;
          if (first + 1 < a.n_units) hid[(long long)(first + 1) * DSUM] = (sum[2] + sum[3]) * inv_c;
        } else {
  #pragma unroll
          for (int x = 0; x < 4; ++x)
            if (first + x < a.n_units) hid[(long long)(first + x) * DSUM] = sum[x] * inv_c;
        }
      }
    }
  }
  umma::fence_before_sync();
  __syncthreads();
  if (warp == TM_MMA_WARP) umma::tmem_dealloc(tmem_d, TM_TMEM_COLS);
}

bool token_mlp_supported(int C, int d_sum) {
  if (d_sum <= 0 || d_sum % 128 != 0 || d_sum > TM_MAX_DSUM) return false;      // the epilogue hands out 32-column groups
  if (C < 32 || C % 32 != 0) return false;
  return C <= 128 ? (128 % C == 0) : (C % 128 == 0);
}

template <int DSUM, bool SHARED>
static cudaError_t launch_pool(const TokenMlpArgs& a, dim3 grid, cudaStream_t st) {
  static DeviceFlags opted;
  const cudaError_t e = smem_opt_in(opted, kve_token_mlp_pool_kernel<DSUM, SHARED>, TM_SMEM_BYTES);
  return e == cudaSuccess ? launch_pdl(kve_token_mlp_pool_kernel<DSUM, SHARED>, grid, dim3(TM_THREADS), TM_SMEM_BYTES, st, a) : e;
}

cudaError_t launch_chunk_token_mlp(const LayerView& v, int t0, int t1, const MlpWeights& w, int d_sum, float* hid, int list_cut, cudaStream_t st) {
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
  a.w = w; a.hid = hid; a.list_cut = list_cut;
  // one CTA per SM, half of the SMs per side; a CTA walks whole items (all 128-token slices of a chunk in a row)
  long long per_side = sm_count() / 2;
  if (per_side > a.n_items) per_side = a.n_items;
  if (per_side < 1) per_side = 1;
  const dim3 grid((unsigned)per_side, 2);
  // All epilogue warps on every tile where a CTA has few of them: with one item the warps of one accumulator would have all the work (74 units of
  // 128 tokens, d_sum 128: 12.1 us a call, 11.6 so; of 384 tokens 16.7 and 14.8), with many the sums that meet in shared memory cost more than
  // an uneven end.  Lines where both meet, items a CTA: 3 with chunks of 32 (8 x 75: 16.9 and 16.5 us), where nothing has to meet; d_sum 128: 2 (148 x
  // 64 tokens 15.9 and 15.7; 175 x 64 16.8 and 16.9); d_sum 256, where a thread has 64 tokens of a tile: 5 with chunks of 64 (600 x 64 26.3 and
  // 26.1; 800 x 64 28.8 and 28.9), 1 with chunks of 128 (140 x 128 19.6 and 19.7), 3 with longer ones (200 x 384 36.4 and 35.0; 260 x 384 41.3 and 41.8).
  const int shared_items = v.C == 32 ? 3 : (d_sum == 128 ? 2 : (v.C == 64 ? 5 : (v.C > TM_N ? 3 : 1)));
  const bool shared = (a.n_items + per_side - 1) / per_side <= shared_items;
  const cudaError_t e = d_sum == 256 ? (shared ? launch_pool<256, true>(a, grid, st) : launch_pool<256, false>(a, grid, st))
                                     : (shared ? launch_pool<128, true>(a, grid, st) : launch_pool<128, false>(a, grid, st));
  return e == cudaSuccess ? launch_pooled_out(v, t0, t1, w, d_sum, hid, st) : e;
}

}  // namespace kve
