// Gate input projection (Eq. 3, the W_ih x_t term for all chunks at once):
//   P[s, t, :] = W_ih [Kbar_t ; Vbar_t] + b_ih + b_hh      a GEMM [S * n_range, 256] x [256, 4 d_g]
// stored with the four gates of a hidden unit side by side (column 4 u + gate)
// bf16 operands (the rounded summaries and bf16 weights, so every product is exact), fp32
// accumulation in tensor memory (tcgen05.mma, M = 128, N = 128 per instruction), bias fused in the
// epilogue.
//
//  * A CTA owns one 128-column slice of W_ih^T for its whole life: the slice (64 KB, K-major,
//    128-byte swizzle) goes to shared memory once, by cp.async.
//  * It then walks over 128-row tiles of X.  Four copy warps gather the rows straight from the summary store
//    (columns 0..127 of a row from ksum_bf16, 128..255 from vsum_bf16) into a ring of eight swizzled K-blocks
//    ([128 rows][64], 16 KB), four of them in flight; one thread issues the four MMAs of a K-block as it arrives.
//  * Two accumulators in tensor memory: while eight epilogue warps read tile i out of one (warp w: lanes
//    32 (w % 4) .., column half w / 4), add the bias and store P, the MMAs of tile i + 1 run into the other.  The epilogue
//    turns each 32 x 32 block through shared memory so that a store instruction writes whole 128-byte row segments.
//  * 256-column slices (128 KB of weights) left room for one tile of X, whose gather, MMAs and store then followed one
//    another: 5.0 us per 128 x 256 tile.  512 sequences x 121 chunks (254 MB of P) 74 us, 70 us this way; 256 x 56
//    26.7 us, 25.0; 8 x 28 at d_g = 128 12.3 us, 10.8 (event pairs).  Bound by shared memory: writing and reading
//    the tiles of X and turning P take about 2500 of the 3800 cycles of a tile.
//  * Every wait is bounded; on give-up the status word gets KVE_ERR_TIMEOUT.
#include "common.cuh"
#include "kernels.h"
#include "umma.cuh"

namespace kve {

constexpr int PJ_M = 128, PJ_N = 128, PJ_K = 2 * D;
constexpr int PJ_KB = PJ_K / umma::KBLOCK_ELEMS;               // 4 K-blocks of 64
constexpr int PJ_EPI_WARPS = 8, PJ_COPY_WARPS = 4;
constexpr int PJ_MMA_WARP = PJ_EPI_WARPS + PJ_COPY_WARPS;
constexpr int PJ_THREADS = (PJ_MMA_WARP + 1) * 32;
constexpr int PJ_SLOTS = 8, PJ_LAG = 4;                        // K-blocks in the ring; copies under way behind the newest
constexpr int PJ_KB_BYTES = PJ_M * umma::KBLOCK_ROW_BYTES;     // 16 KB, for rows of X and of W_ih alike
constexpr int PJ_SMEM_B = 0;
constexpr int PJ_SMEM_A = PJ_SMEM_B + PJ_KB * PJ_KB_BYTES;     // 64 KB
constexpr int PJ_SMEM_STG = PJ_SMEM_A + PJ_SLOTS * PJ_KB_BYTES;   // +128 KB; per epilogue warp: a 32 x 32 fp32 block on its way out
constexpr int PJ_SMEM_BIAS = PJ_SMEM_STG + PJ_EPI_WARPS * 4096;
constexpr int PJ_SMEM_BAR = PJ_SMEM_BIAS + PJ_N * 4;
constexpr int PJ_SMEM_BYTES = PJ_SMEM_BAR + (2 * PJ_SLOTS + 4) * 8 + 16 + 1024;   // + slack to reach a 1024-byte boundary
static_assert(PJ_SMEM_BYTES <= 227 * 1024 && PJ_M == PJ_N, "shared memory of one CTA");
constexpr int PJ_TMEM_COLS = 2 * PJ_N;

__global__ void __launch_bounds__(PJ_THREADS, 1) kve_gate_proj_kernel(LayerView v, int t0, int n_range, FastDiv by_range, int n_rows,
                                                                      const uint16_t* __restrict__ W_ih,
                                                                      const float* __restrict__ b_ih,
                                                                      const float* __restrict__ b_hh, int n_cols,
                                                                      float* __restrict__ P, int list_cut) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* Bs = smem + PJ_SMEM_B;
  unsigned char* As = smem + PJ_SMEM_A;
  float* bias = reinterpret_cast<float*>(smem + PJ_SMEM_BIAS);
  uint64_t* a_full = reinterpret_cast<uint64_t*>(smem + PJ_SMEM_BAR);      // [8] K-block filled by the copy warps
  uint64_t* a_free = a_full + PJ_SLOTS;                                     // [8] K-block multiplied (MMA commit)
  uint64_t* acc_full = a_free + PJ_SLOTS;                                   // [2] accumulator written (MMA commit)
  uint64_t* acc_free = acc_full + 2;                                        // [2] accumulator read by the epilogue warps
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_free + 2);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int col0 = blockIdx.x * PJ_N;
  const int n_tiles = (n_rows + PJ_M - 1) / PJ_M;
  const int my_tiles = n_tiles > (int)blockIdx.y ? (n_tiles - (int)blockIdx.y + (int)gridDim.y - 1) / (int)gridDim.y : 0;

  // ---- one-time set-up: weight slice, bias, tensor memory, barriers ---------------------------------
  for (int i = tid; i < PJ_N * 32; i += PJ_THREADS) {
    const int r = i >> 5, p = i & 31;                 // p: 16-byte piece of the 512-byte weight row
    // column c of P holds gate c & 3 of hidden unit c >> 2 (the four pre-activations of a unit side by side: the
    // recurrence fetches them with one 16-byte load): row (c & 3) d_g + (c >> 2) of W_ih
    const int c = col0 + r, d_g = n_cols >> 2;
    cp_async16(Bs + (p >> 3) * PJ_KB_BYTES + umma::piece_offset(r, p & 7),
               reinterpret_cast<const uint4*>(W_ih + (long long)((c & 3) * d_g + (c >> 2)) * PJ_K) + p, true);
  }
  for (int i = tid; i < PJ_N; i += PJ_THREADS) {
    const int c = col0 + i, row = (c & 3) * (n_cols >> 2) + (c >> 2);
    bias[i] = b_ih[row] + b_hh[row];
  }
  if (warp == PJ_MMA_WARP) umma::tmem_alloc(tmem_slot, PJ_TMEM_COLS);
  if (tid == 0) {
    for (int i = 0; i < PJ_SLOTS; ++i) {
      mbar_init(&a_full[i], PJ_COPY_WARPS * 32);
      mbar_init(&a_free[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_free[i], PJ_EPI_WARPS);
    }
    mbar_fence_init();
  }
  cp_async_wait_all();
  umma::fence_smem_to_async();
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tmem = *tmem_slot;

  pdl_wait();      // the summaries come from the previous kernel
  pdl_launch_dependents();      // the recurrence's CTAs have nothing to do before that and take up room (8 sequences x 28 chunks: a step 0.6 us shorter)
  if (list_cut >= 0 && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *v.n_listed = list_cut;

  if (warp < PJ_EPI_WARPS) {
    // ================= epilogue: accumulator + bias -> P =================
    float* stg = reinterpret_cast<float*>(smem + PJ_SMEM_STG) + warp * 1024;
    const int lg = warp & 3, half = warp >> 2;
    for (int k = 0; k < my_tiles; ++k) {
      const int buf = k & 1, row0 = ((int)blockIdx.y + k * (int)gridDim.y) * PJ_M + lg * 32;
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&acc_full[buf], (uint32_t)((k >> 1) & 1)))) {
        if (lane == 0) set_status(v.status, ERR_TIMEOUT);
        break;
      }
      umma::fence_after_sync();
      const uint32_t acc_addr = tmem + (uint32_t)(buf * PJ_N + half * 64) + ((uint32_t)(lg * 32) << 16);
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
        const int c = half * 64 + cc * 32;
        float acc[32];
        umma::tmem_ld32(acc_addr + (uint32_t)(cc * 32), acc);
        if (cc == 1) {
          umma::fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_free[buf]);
        }
        // tcgen05.ld hands a thread one row (32 columns); the block is turned through the staging area (16-byte groups, group q
        // of row r at position q ^ (r & 7): conflict-free both ways) so that a store instruction covers four rows with
        // 128 contiguous bytes each
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 b = *reinterpret_cast<const float4*>(bias + c + 4 * q);
          *reinterpret_cast<float4*>(stg + lane * 32 + ((q ^ (lane & 7)) << 2)) =
              make_float4(acc[4 * q] + b.x, acc[4 * q + 1] + b.y, acc[4 * q + 2] + b.z, acc[4 * q + 3] + b.w);
        }
        __syncwarp();
        const int q = lane & 7;
        float* out = P + (long long)row0 * n_cols + col0 + c + q * 4;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int rr = i * 4 + (lane >> 3);
          const float4 val = *reinterpret_cast<const float4*>(stg + rr * 32 + ((q ^ (rr & 7)) << 2));
          if (row0 + rr < n_rows) *reinterpret_cast<float4*>(out + (long long)rr * n_cols) = val;
        }
        __syncwarp();
      }
    }
  } else if (warp < PJ_MMA_WARP) {
    // ================= copy warps: K-blocks of X =================
    const int ct = tid - PJ_EPI_WARPS * 32, p = ct & 7, r0 = ct >> 3;      // the 16-byte piece p of the rows r0 + 16 i
    const int n_blocks = my_tiles * PJ_KB;
    int row_of[PJ_M / 16];      // summary row of this thread's rows of the tile, -1 beyond the last one
    bool ok = true;
    for (int n = 0; n < n_blocks + PJ_LAG && ok; ++n) {
      if (n < n_blocks) {
        const int slot = n % PJ_SLOTS, kb = n % PJ_KB;
        if (kb == 0) {
          const int base = ((int)blockIdx.y + n / PJ_KB * (int)gridDim.y) * PJ_M + r0;
#pragma unroll
          for (int i = 0; i < PJ_M / 16; ++i) {
            const int gr = base + 16 * i, s = (int)by_range.div((uint32_t)gr);
            row_of[i] = gr < n_rows ? s * v.max_chunks + t0 + (gr - s * n_range) : -1;
          }
        }
        if (n >= PJ_SLOTS) ok = mbar_wait_bounded(&a_free[slot], (uint32_t)((n / PJ_SLOTS - 1) & 1));
        const uint16_t* src = (kb < PJ_KB / 2 ? v.ksum_bf16 : v.vsum_bf16) + (kb & 1) * umma::KBLOCK_ELEMS + p * 8;
        unsigned char* dst = As + slot * PJ_KB_BYTES;
#pragma unroll
        for (int i = 0; i < PJ_M / 16; ++i)
          cp_async16(dst + umma::piece_offset(r0 + 16 * i, p), src + (long long)max(row_of[i], 0) * D, row_of[i] >= 0);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");      // (an empty group at the end keeps the count)
      if (n >= PJ_LAG) {
        asm volatile("cp.async.wait_group %0;" ::"n"(PJ_LAG) : "memory");
        umma::fence_smem_to_async();
        mbar_arrive(&a_full[(n - PJ_LAG) % PJ_SLOTS]);
      }
    }
    if (!ok) set_status(v.status, ERR_TIMEOUT);
    cp_async_wait_all();
  } else if (lane == 0) {
    // ================= MMA issue (one thread) =================
    const uint32_t a_base = smem_u32(As), b_base = smem_u32(Bs);
    constexpr uint32_t idesc = umma::instr_desc_bf16(PJ_M, PJ_N);
    bool ok = true;
    for (int n = 0; n < my_tiles * PJ_KB && ok; ++n) {
      const int slot = n % PJ_SLOTS, kb = n % PJ_KB, tile = n / PJ_KB, buf = tile & 1;
      ok = mbar_wait_bounded(&a_full[slot], (uint32_t)((n / PJ_SLOTS) & 1));
      if (kb == 0 && tile >= 2) ok = ok && mbar_wait_bounded(&acc_free[buf], (uint32_t)(((tile >> 1) - 1) & 1));
      if (!ok) break;
      umma::fence_after_sync();
#pragma unroll
      for (int k = 0; k < 4; ++k)
        umma::mma_bf16(tmem + (uint32_t)(buf * PJ_N), umma::smem_desc(a_base + slot * PJ_KB_BYTES + k * 32),
                       umma::smem_desc(b_base + kb * PJ_KB_BYTES + k * 32), idesc, (kb | k) != 0);
      umma::commit(&a_free[slot]);
      if (kb == PJ_KB - 1) umma::commit(&acc_full[buf]);
    }
    if (!ok) set_status(v.status, ERR_TIMEOUT);
  }

  umma::fence_before_sync();
  __syncthreads();
  if (warp == PJ_MMA_WARP) umma::tmem_dealloc(tmem, PJ_TMEM_COLS);
}

cudaError_t launch_gate_proj(const LayerView& v, int t0, int t1, const uint16_t* W_ih, const float* b_ih,
                             const float* b_hh, int d_g, float* P, int list_cut, cudaStream_t st) {
  const int n_range = t1 - t0;
  const long long n_rows = (long long)v.S * n_range;
  if (n_rows <= 0) return cudaSuccess;
  const int n_cols = 4 * d_g;                     // 256, 512 or 1024: whole 128-column slices
  if (n_cols % PJ_N != 0) return cudaErrorInvalidValue;
  if (n_rows + PJ_M >= (1LL << 31) || (long long)v.S * v.max_chunks >= (1LL << 31)) return cudaErrorInvalidValue;
  static DeviceFlags opted;
  {
    cudaError_t e = smem_opt_in(opted, kve_gate_proj_kernel, PJ_SMEM_BYTES);
    if (e != cudaSuccess) return e;
  }
  const int col_slices = n_cols / PJ_N;
  const long long n_tiles = (n_rows + PJ_M - 1) / PJ_M;
  long long row_ctas = sm_count() / col_slices;          // one CTA per SM (shared memory), every slice equally served
  if (row_ctas > n_tiles) row_ctas = n_tiles;
  if (row_ctas < 1) row_ctas = 1;
  dim3 grid((unsigned)col_slices, (unsigned)row_ctas);
  return launch_pdl(kve_gate_proj_kernel, grid, dim3(PJ_THREADS), PJ_SMEM_BYTES, st, v, t0, n_range, fast_div((uint32_t)n_range), (int)n_rows, W_ih, b_ih, b_hh, n_cols, P, list_cut);
}

}  // namespace kve
