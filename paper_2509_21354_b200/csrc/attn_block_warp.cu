// Attention of a block of at most 32 query rows (query tokens x heads of a KV head) over the retained set (Sec. 3.3, softmax of Eq. 1),
// out[r] = softmax(q[r] K'^T * scale) V', with both products on warp-level tensor-core MMAs.
//
// HBM-bound: every retained K/V row is fetched once per KV sequence.  A 64-row tile of K and V (32 KB) takes an SM ~1200 cycles to
// receive; its 256 MMAs (m16n8k16, 16 query rows each) take ~512.  What the tile must not meet on its way is a chain of hand-overs:
//  * grid = (splits, KV sequences), one CTA per SM.  A producer warp fetches the tiles by tiled copies (TMA, 128-byte swizzle) into a ring.
//  * Eight consumer warps in two groups that take tiles in turn; a warp owns 16 of the tile's keys for all query rows and keeps its
//    own running maximum, sum and accumulator O [32][128] in registers: nothing is exchanged between warps before the end.
//    S = Q K^T with the queries as the M side (fragments in registers for the whole kernel), so its accumulators are, rounded to
//    bf16, at once the left operand of O += P V.  (Rounding p moves an output by at most 2^-8 sum p |v| / sum p.)
//  * The reference of the exponentials follows a row's maximum lazily: only when one has grown by more than 8 (log2 units) are
//    O and the sums rescaled, so p stays below 2^8.
//  * At the end the eight states meet in shared memory (the ring is free) and a warp merges a row at a time.  Splits leave
//    records in the workspace; the last CTA of a sequence to finish (ticket, nobody spins) merges them, four rows of a warp side by side
//    (record after record and row after row, each a trip to L2: 64 sequences x 4099 rows in 2 splits 34.9 us, 30.0 so; 8 x 2000 in 16
//    splits 17.7 and 12.7).
// Measured (28 query rows; before: on tcgen05, the block replicated down its 128 lanes): 128 sequences x 1084 rows 21.4 -> 18.4 us,
// 64 x 4099 40.1 -> 30.0 us, 128 x 4000 (32 rows) 54.9 -> 45.2 us = 6.5 TB/s less ~5 us of start and merge.  The stream alone, without
// arithmetic, takes 16.4 us of the first.
// Every mbarrier wait is bounded; on give-up the status word gets KVE_ERR_TIMEOUT.
#include "attn_block.cuh"

namespace kve {

constexpr int BW_STAGES = 6;                           // even: a stage belongs to one group, which waits for its phases in order
constexpr int BW_CWARPS = 8, BW_GWARPS = 4;            // consumer warps; warps of a group
constexpr int BW_THREADS = (BW_CWARPS + 4) * 32;       // and a warpgroup with the producer (registers move between warpgroups)
constexpr int BW_REGS = 232, BW_PRODUCER_REGS = 40, BW_LAUNCH_REGS = 168;
static_assert(3 * BW_LAUNCH_REGS == 2 * BW_REGS + BW_PRODUCER_REGS, "the warpgroups ask for exactly what the launch has");
constexpr int BW_XP = 136;                             // floats per row of the exchange area: acc[128], m, l, and no bank conflicts
constexpr int BW_OFF_Q = BW_STAGES * BK_STAGE_BYTES;   // [32 rows][128] bf16 as two K-blocks of 4 KB
constexpr int BW_OFF_BAR = BW_OFF_Q + 32 * ROW_BYTES;
constexpr int BW_SMEM_BYTES = BW_OFF_BAR + 2 * BW_STAGES * 8 + 16 + 1024;      // + slack to reach a 1024-byte boundary
static_assert(BW_STAGES % 2 == 0, "a group that came ahead of the other would take a phase that has not begun for a complete one");
static_assert(BW_SMEM_BYTES <= 227 * 1024 && BW_CWARPS * 32 * BW_XP * 4 <= BW_OFF_Q, "shared memory of one CTA; the exchange area fits the ring");
constexpr float BW_RESCALE_STEP = 8.f;                 // log2 units a row's maximum may run ahead of the reference

__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void consumers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(BW_CWARPS * 32) : "memory"); }

// MT: 16-row tiles of the query block
template <int MT>
__global__ void __maxnreg__(BW_LAUNCH_REGS)
kve_decode_attn_block_warp_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                                  const __grid_constant__ CUtensorMap tmKs, const __grid_constant__ CUtensorMap tmVs, BlockArgs a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* ring = smem;
  unsigned char* Qs = smem + BW_OFF_Q;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + BW_OFF_BAR);
  uint64_t* empty = full + BW_STAGES;
  int* flag = reinterpret_cast<int*>(empty + BW_STAGES);
  volatile int* issued = flag + 1;       // tiles that the producer has issued when it is through, -1 before

  pdl_launch_dependents();
  const LayerView& v = a.v;
  const int s = blockIdx.y, split = blockIdx.x;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

  // what the first look-ups after the wait will need, pulled into L2 meanwhile
  if (warp == BW_CWARPS) {
    const int raw0 = (a.mode == ATTN_DENSE) ? 0 : a.n_chunks * v.C, chunk0 = (int)a.by_c.div((uint32_t)(raw0 + split * a.rows_per_split));
    if (lane == 0) prefetch_l2(v.seq_len + a.by_h.div((uint32_t)s));
    if (lane == 1) prefetch_l2(v.keep_cnt + s);
    if (lane == 2 && chunk0 < v.max_chunks) prefetch_l2(v.page_table + (long long)s * v.max_chunks + chunk0);
  } else if (warp == 0) {
    for (int r = lane; r < 2 * a.R; r += 32) prefetch_l2(a.q + q_row_offset(a, s, r >> 1) + (r & 1) * 64);
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < BW_STAGES; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], BW_GWARPS);
    }
    mbar_fence_init();
    *issued = -1;
  }
  __syncthreads();

  if (warp >= BW_CWARPS) {
    // ================= producer warp =================
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(BW_PRODUCER_REGS));
    if (warp > BW_CWARPS) return;
    pdl_wait();      // lengths, keep lists and summaries come from earlier kernels
    const int first = first_pages(a, s, split, lane);
    const BlockGeom gm = block_geometry(a, s, split);
    // the sequence has outgrown what this launch was sized for (a replayed launch): rows would be dropped
    if (gm.outgrown && split == 0 && lane == 0) set_status(v.status, ERR_CAPACITY);
    if (split < gm.n_splits) {
      const int n = block_producer<BW_STAGES, 0>(a, gm, s, lane, &tmK, &tmV, &tmKs, &tmVs, first, ring, full, empty);
      if (lane == 0) *issued = n;
    }
    return;
  }

  // ================= consumer warps =================
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(BW_REGS));
  pdl_wait();
  const BlockGeom gm = block_geometry(a, s, split);
  if (split >= gm.n_splits) return;      // nothing for this CTA
  const int group = warp >> 2, gw = warp & 3, g = lane >> 2, tig = lane & 3;

  // ---- the query block as the left operand, fragments in registers ----
  for (int idx = threadIdx.x; idx < MT * 16 * 16; idx += BW_CWARPS * 32) {
    const int r = idx >> 4, p16 = idx & 15;
    uint4 val = make_uint4(0u, 0u, 0u, 0u);
    if (r < a.R) val = *reinterpret_cast<const uint4*>(a.q + q_row_offset(a, s, r) + p16 * 8);
    *reinterpret_cast<uint4*>(Qs + r * ROW_BYTES + ((p16 ^ (r & 7)) << 4)) = val;
  }
  consumers_sync();
  uint32_t Q[MT][8][4];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int kt = 0; kt < 8; ++kt) {      // matrices: rows 0-7 / 8-15, then the same at the upper 8 of the 16 head dims
      const int r = mt * 16 + ((lane >> 3) & 1) * 8 + (lane & 7), p16 = kt * 2 + (lane >> 4);
      ldsm_x4(Q[mt][kt], smem_u32(Qs) + r * ROW_BYTES + ((p16 ^ (r & 7)) << 4));
    }
  // what a lane holds: query rows 16 mt + g + 8 e, as C fragments
  float O[MT][16][4], m_ref[MT][2], l_run[MT][2];
  int tok[MT][2];      // query token of each row
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
    for (int x = 0; x < 16; ++x)
#pragma unroll
      for (int e = 0; e < 4; ++e) O[mt][x][e] = 0.f;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      m_ref[mt][e] = -INFINITY;
      l_run[mt][e] = 0.f;
      tok[mt][e] = (int)a.by_g.div((uint32_t)min(mt * 16 + e * 8 + g, a.R - 1));
    }
  }
  const float sl2 = a.scale * 1.44269504088896340736f;      // logits in log2 units
  // this lane's row of the matrices that it addresses: K rows (keys 0-7 twice, 8-15 twice), V rows (keys 0-7, 8-15, twice)
  const int k_row = gw * 16 + (lane >> 4) * 8 + (lane & 7), v_row = gw * 16 + ((lane >> 3) & 1) * 8 + (lane & 7);

  for (int i = group; i < gm.n_tiles; i += 2) {
    const int stage = i % BW_STAGES;
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full[stage], (uint32_t)((i / BW_STAGES) & 1)))) {
      // copies into the ring may be under way: this warp meets the others, which use the ring for something else then, when they have landed
      // (the producer comes to an end, too, if it waits for us)
      if (lane == 0) set_status(v.status, ERR_TIMEOUT);
      for (int k = 0; k < (1 << 20) && *issued < 0; ++k) __nanosleep(2048);
      ring_drain<BW_STAGES>(full, *issued);
      break;
    }
    const int row0 = gm.r_begin + i * BK_TILE;
    const int valid = gm.rows_valid(row0);
    if (gw * 16 < valid) {
      unsigned char* kt_base = ring + stage * BK_STAGE_BYTES;
      const uint32_t kb = smem_u32(kt_base), vb = kb + BK_TILE_BYTES;
      // ---- S = Q K^T for the warp's 16 keys ----
      float S[MT][2][4];
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) S[mt][nt][e] = 0.f;
#pragma unroll
      for (int kt = 0; kt < 8; ++kt) {
        uint32_t K[4];
        ldsm_x4(K, kb + tile_piece(k_row, kt * 2 + ((lane >> 3) & 1)));
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          mma_bf16_16816(S[mt][0], Q[mt][kt], K[0], K[1]);
          mma_bf16_16816(S[mt][1], Q[mt][kt], K[2], K[3]);
        }
      }
      // ---- logits in log2 units; columns that a row may not use are -inf ----
      // causal blocks: query token t sees the cache up to its own position, i.e. all but the last T - 1 - t rows of the raw tail
      // (the block's own tokens are the newest rows of the tail)
      const bool edge = a.causal && row0 < gm.tail_pad && row0 + BK_TILE > gm.n_tail - (a.T - 1);
      float mx[MT][2];
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) { S[mt][nt][2 * e] *= sl2; S[mt][nt][2 * e + 1] *= sl2; }
          if (edge || gw * 16 + 16 > valid) {
            const int visible = (edge ? min(valid, gm.n_tail - (a.T - 1 - tok[mt][e]) - row0) : valid) - gw * 16 - tig * 2;
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
              if (nt * 8 >= visible) S[mt][nt][2 * e] = -INFINITY;
              if (nt * 8 + 1 >= visible) S[mt][nt][2 * e + 1] = -INFINITY;
            }
          }
          mx[mt][e] = fmaxf(fmaxf(S[mt][0][2 * e], S[mt][0][2 * e + 1]), fmaxf(S[mt][1][2 * e], S[mt][1][2 * e + 1]));
        }
      // ---- the reference follows the maximum ----
      bool grown = false;
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int e = 0; e < 2; ++e) grown |= mx[mt][e] > m_ref[mt][e] + BW_RESCALE_STEP;
      if (__any_sync(0xffffffffu, grown)) {      // (always on the warp's first tile with something to see: the reference is -inf)
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            float m = mx[mt][e];
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
            const float m_new = fmaxf(m_ref[mt][e], m);
            const float f = (m_ref[mt][e] == -INFINITY) ? 0.f : ex2_fast(m_ref[mt][e] - m_new);      // nothing accumulated yet: O is 0
            m_ref[mt][e] = m_new;
            l_run[mt][e] *= f;
#pragma unroll
            for (int x = 0; x < 16; ++x) { O[mt][x][2 * e] *= f; O[mt][x][2 * e + 1] *= f; }
          }
      }
      // ---- p, its bf16 rounding as the left operand of O += P V ----
      uint32_t P[MT][4];
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          // (a row that has not seen a single column yet has m_ref = -inf: its p are 0, not exp2(-inf + inf))
          const float neg_m = (m_ref[mt][e] == -INFINITY) ? 0.f : -m_ref[mt][e];
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) {
            const float p0 = ex2_fast(S[mt][nt][2 * e] + neg_m), p1 = ex2_fast(S[mt][nt][2 * e + 1] + neg_m);
            l_run[mt][e] += p0 + p1;
            P[mt][nt * 2 + e] = pack_bf16x2(p0, p1);
          }
        }
      if (gw * 16 + 16 > valid) {
        // stale V rows of a partial tile are cleared: 0 * NaN would stay in O
        for (int idx = lane; idx < (gw * 16 + 16 - valid) * 16; idx += 32)
          *reinterpret_cast<uint4*>(kt_base + BK_TILE_BYTES + tile_piece(valid + (idx >> 4), idx & 15)) = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // before the next copy into this stage
        __syncwarp();
      }
#pragma unroll
      for (int dt = 0; dt < 8; ++dt) {
        uint32_t V[4];
        ldsm_x4_trans(V, vb + tile_piece(v_row, dt * 2 + (lane >> 4)));
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          mma_bf16_16816(O[mt][2 * dt], P[mt], V[0], V[1]);
          mma_bf16_16816(O[mt][2 * dt + 1], P[mt], V[2], V[3]);
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[stage]);
  }

  // ---- the eight states (m_ref, l, O) meet in shared memory: [warp][row][BW_XP] from the start of the ring ----
  float* xch = reinterpret_cast<float*>(smem);
  consumers_sync();      // every tile has been read, or a warp has given up and seen the copies land
  float* mine = xch + warp * 32 * BW_XP;
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float l = l_run[mt][e];
      l += __shfl_xor_sync(0xffffffffu, l, 1);
      l += __shfl_xor_sync(0xffffffffu, l, 2);
      float* row = mine + (mt * 16 + e * 8 + g) * BW_XP;
#pragma unroll
      for (int x = 0; x < 16; ++x) *reinterpret_cast<float2*>(row + x * 8 + tig * 2) = make_float2(O[mt][x][2 * e], O[mt][x][2 * e + 1]);
      if (tig == 0) *reinterpret_cast<float2*>(row + 128) = make_float2(m_ref[mt][e], l);
    }
  consumers_sync();
  const bool direct = gm.n_splits == 1;
  for (int r = warp; r < a.R; r += BW_CWARPS) {
    float2 ml[BW_CWARPS];
    float mC = -INFINITY, lC = 0.f;
#pragma unroll
    for (int w = 0; w < BW_CWARPS; ++w) {
      ml[w] = *reinterpret_cast<const float2*>(xch + (w * 32 + r) * BW_XP + 128);
      mC = fmaxf(mC, ml[w].x);
    }
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < BW_CWARPS; ++w) {
      const float f = (ml[w].x == -INFINITY) ? 0.f : exp2f(ml[w].x - mC);
      lC = fmaf(ml[w].y, f, lC);
      const float4 o = *reinterpret_cast<const float4*>(xch + (w * 32 + r) * BW_XP + lane * 4);
      acc = make_float4(fmaf(o.x, f, acc.x), fmaf(o.y, f, acc.y), fmaf(o.z, f, acc.z), fmaf(o.w, f, acc.w));
    }
    if (direct) {
      write_block_out(a, s, r, lane, acc, mC, lC);
    } else {
      float* rec = a.partials + (((long long)s * a.max_splits + split) * a.rec_rows + r) * BK_REC;
      *reinterpret_cast<float4*>(rec + lane * 4) = acc;
      if (lane == 0) *reinterpret_cast<float2*>(rec + 128) = make_float2(mC, lC);
    }
  }
  if (direct) return;
  block_merge_splits(a, s, gm.n_splits, flag, warp, lane, BW_CWARPS, consumers_sync);
}

template <int MT>
static cudaError_t launch_warp(const CUtensorMap* tm, const BlockArgs& a, dim3 grid, cudaStream_t st) {
  static DeviceFlags opted;
  const cudaError_t e = smem_opt_in(opted, kve_decode_attn_block_warp_kernel<MT>, BW_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  return launch_pdl(kve_decode_attn_block_warp_kernel<MT>, grid, dim3(BW_THREADS), BW_SMEM_BYTES, st, tm[0], tm[1], tm[2], tm[3], a);
}

cudaError_t launch_attn_block_warp(const CUtensorMap* tm, const BlockArgs& a, dim3 grid, cudaStream_t st) {
  return a.R <= 16 ? launch_warp<1>(tm, a, grid, st) : launch_warp<2>(tm, a, grid, st);
}

}  // namespace kve
