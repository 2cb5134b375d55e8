// Pieces shared by the block-of-queries attention kernels: launch arguments, the geometry of a
// sequence's padded logical rows, the TMA producer warp and the merge of split records.
//
// Logical rows of a sequence: the raw tail (padded up to whole 64-row tiles), then the kept rows
// (summary rows, or the raw rows of kept chunks), so a tile is either all tail or all kept rows.  A
// tile lands in shared memory as K tile then V tile, each two K-blocks [64 rows][64 bf16] with the
// 128-byte swizzle (what a tensor copy with that swizzle mode writes): the 16-byte piece c of row r
// of a K-block sits at r * 128 + ((c ^ (r & 7)) << 4).
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "kernels.h"

namespace kve {

constexpr int BK_TILE = ATTN_TILE_ROWS;         // 64 rows per stage
constexpr int BK_KBLOCK_BYTES = BK_TILE * 128;  // one K-block: 64 rows x 64 bf16
constexpr int BK_TILE_BYTES = 2 * BK_KBLOCK_BYTES;        // K (or V) tile, 16 KB
constexpr int BK_STAGE_BYTES = 2 * BK_TILE_BYTES;         // K tile then V tile
constexpr int BK_SUM_BOX = ATTN_BLOCK_SUM_BOX;   // rows per tensor-copy box over the compacted kept summary rows
constexpr int BK_REC = ATTN_PARTIAL_FLOATS;     // floats per (query row) record: acc[128], m, l, pad

struct BlockArgs {
  LayerView v;
  FastDiv by_c, by_h, by_g, by_split;      // by the chunk size, KV heads, query heads per KV head, rows per split
  int mode, n_chunks, rows_per_split, max_splits;
  int T, G, R;              // query tokens, query heads per KV head, T * G
  int rec_rows;             // query-row records per (sequence, split) in `partials`
  int causal;               // query token t sees the cache up to its own position only
  int hp;                   // rows per page box
  long long sum_row0;       // first row of this layer in the tensor maps over the compacted kept summary rows
  const uint16_t* q;        // [B][T][Hq][128]
  uint16_t* out;            // [B][T][Hq][128]
  float* lse;               // [B][T][Hq] or null
  float scale;
  float* partials;          // [S][max_splits][rec_rows][BK_REC]
  int32_t* counters;        // [S], zero between launches
};

struct BlockGeom {
  int raw0, n_tail, tail_pad, n_rows, n_splits, r_begin, r_end, n_tiles;
  bool outgrown;      // the sequence needs more splits than the launch has: rows beyond the grid are dropped (flagged)
  // valid rows of the tile that starts at padded row `row0`
  __device__ __forceinline__ int rows_valid(int row0) const {
    return row0 < tail_pad ? min(BK_TILE, n_tail - row0) : min(BK_TILE, n_rows - row0);
  }
};

__device__ __forceinline__ BlockGeom block_geometry(const BlockArgs& a, int s, int split) {
  const LayerView& v = a.v;
  BlockGeom g;
  int n = v.seq_len[a.by_h.div((uint32_t)s)];
  n = min(max(n, 0), v.max_tokens);
  const int M = (a.mode == ATTN_DENSE) ? 0 : min(max(v.keep_cnt[s], 0), a.n_chunks);
  g.raw0 = (a.mode == ATTN_DENSE) ? 0 : a.n_chunks * v.C;
  const int n_lead = (a.mode == ATTN_RAW) ? M * v.C : M;
  g.n_tail = max(0, n - g.raw0);
  g.tail_pad = (g.n_tail + BK_TILE - 1) / BK_TILE * BK_TILE;
  g.n_rows = g.tail_pad + n_lead;
  g.n_splits = max(1, (int)a.by_split.div((uint32_t)(g.n_rows + a.rows_per_split - 1)));
  // a replayed launch the sequence has outgrown: the splits that exist still merge and the ticket
  // counter still returns to zero; the caller learns about the dropped rows from the status word
  g.outgrown = g.n_splits > (int)gridDim.x;
  g.n_splits = min(g.n_splits, (int)gridDim.x);
  g.r_begin = split * a.rows_per_split;
  g.r_end = min(g.n_rows, g.r_begin + a.rows_per_split);
  g.n_tiles = (max(g.r_end - g.r_begin, 0) + BK_TILE - 1) / BK_TILE;
  return g;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst_smem, const CUtensorMap* tm, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
          dst_smem),
      "l"(tm), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

// byte offset of the 16-byte piece p16 (0..15 along the 128 head dims) of tile row `row`
__device__ __forceinline__ uint32_t tile_piece(int row, int p16) {
  return (uint32_t)((p16 >> 3) * BK_KBLOCK_BYTES + row * 128 + (((p16 & 7) ^ (row & 7)) << 4));
}

// element offset of query / output row r of KV sequence s in the [B][T][Hq][128] layout
__device__ __forceinline__ long long q_row_offset(const BlockArgs& a, int s, int r) {
  const int b = (int)a.by_h.div((uint32_t)s), h = s - b * a.v.H;
  const int t = (int)a.by_g.div((uint32_t)r), g = r - t * a.G;
  return ((((long long)b * a.T + t) * (a.G * a.v.H)) + h * a.G + g) * D;
}

// A granule is what one page box covers: hp rows of a page (a tile has 64 / hp of them; hp is a power of two, so 32 granules are
// whole tiles).  Page ids of a split's first 32 granules, one per lane, looked up as if all were raw tail: where those lie follows
// from the launch arguments, so the look-ups need not wait for the stored length.
__device__ __forceinline__ int first_pages(const BlockArgs& a, int s, int split, int lane) {
  const int raw0 = (a.mode == ATTN_DENSE) ? 0 : a.n_chunks * a.v.C;
  const int chunk = (int)a.by_c.div((uint32_t)(raw0 + split * a.rows_per_split + lane * a.hp));
  return chunk < a.v.max_chunks ? a.v.page_table[(long long)s * a.v.max_chunks + chunk] : -1;
}

// Producer warp: fetches the CTA's tiles with 2-D tensor copies into the ring `ring` (STAGES stages), arming full[stage] with the
// byte count and waiting (bounded) on empty[stage] before a stage is reused.  Returns the tiles issued; their
// copies may still be under way, and a CTA of which anybody gives up a wait has to see them land (ring_drain) before it leaves.  Page ids are looked up 32 granules at a time, a
// batch ahead, and looked at only when a copy needs them: a look-up is a trip to L2, and one per tile in the producer's way made 128
// sequences x 1084 rows 18.5 us, 18.1 so (64 x 4099 35.2 and 34.6).  What a lane fetches for a tile: up to two boxes (K and V each, both 64-column halves):
//   page tiles:    lane j < granules: hp rows of a page to tile row j * hp
//   summary tiles: lane j < ceil(valid / 16): 16 kept summary rows (compacted by kvE_compact)
// FILL_PAUSE_NS: pause between the tiles of the first filling of the ring.  Asked for all at once they land at about the same time, and the first
// lands late: where a tile takes longer to work on than to fetch (the tcgen05 kernel: five hand-overs) that is the launch's start.  128 rows x 256
// sequences x 300 rows 26.7 us without, 25.7 with 250 ns, 25.6 with 500; 64 rows x 128 x 1084 22.2, 21.6, 21.7; the kernel on
// warp MMAs, which keeps up with the copies, loses (28 rows x 128 x 1084 16.5 and 16.9).
template <int STAGES, int FILL_PAUSE_NS>
__device__ __forceinline__ int block_producer(const BlockArgs& a, const BlockGeom& gm, int s, int lane,
                                               const CUtensorMap* tmK, const CUtensorMap* tmV, const CUtensorMap* tmKs,
                                               const CUtensorMap* tmVs, int first, unsigned char* ring, uint64_t* full,
                                               uint64_t* empty) {
  const LayerView& v = a.v;
  const long long sb = (long long)s * v.max_chunks;
  const int per_tile = BK_TILE / a.hp;
  // page of the granule that starts at padded row `row` of the sequence (-1: none); `known`: its page if it lies in the raw tail
  auto look_up = [&](int row, bool use_known, int known) -> int {
    if (row < gm.tail_pad) {
      if (use_known) return known;
      const int chunk = (int)a.by_c.div((uint32_t)(gm.raw0 + row));
      return row < gm.n_tail ? v.page_table[sb + chunk] : -1;
    }
    if (a.mode != ATTN_RAW || row >= gm.r_end) return -1;
    const int chunk = v.keep_idx[sb + (int)a.by_c.div((uint32_t)(row - gm.tail_pad))];
    return (chunk >= 0 && chunk < a.n_chunks) ? v.page_table[sb + chunk] : -1;
  };
  int pages = look_up(gm.r_begin + lane * a.hp, true, first);
  int pages_next = look_up(gm.r_begin + (32 + lane) * a.hp, false, -1);
  int i = 0;
  for (; i < gm.n_tiles; ++i) {
    const int stage = i % STAGES, round = i / STAGES;
    const int granule = i * per_tile;
    if (i > 0 && granule % 32 == 0) {
      pages = pages_next;
      pages_next = look_up(gm.r_begin + (granule + 32 + lane) * a.hp, false, -1);
    }
    const int row0 = gm.r_begin + i * BK_TILE;
    const int valid = gm.rows_valid(row0);
    const bool from_pages = row0 < gm.tail_pad || a.mode == ATTN_RAW;
    int src = -1;
    if (from_pages) {
      int page = __shfl_sync(0xffffffffu, pages, (granule + lane) % 32);
      if (lane * a.hp < valid) {
        const int pos = (row0 < gm.tail_pad ? gm.raw0 + row0 : row0 - gm.tail_pad) + lane * a.hp;
        if (page < 0 || page >= v.n_pages) { set_status(v.status, ERR_CAPACITY); page = 0; }
        src = (int)((long long)page * v.C + (pos - (int)a.by_c.div((uint32_t)pos) * v.C));
      }
    } else if (lane * BK_SUM_BOX < valid) {
      // kept summary rows sit compacted, one contiguous run per sequence: boxes of BK_SUM_BOX rows, lane j the j-th
      src = (int)(a.sum_row0 + sb + (row0 - gm.tail_pad) + lane * BK_SUM_BOX);
    }
    if (round > 0 && !__all_sync(0xffffffffu, mbar_wait_bounded(&empty[stage], (round - 1) & 1))) {
      if (lane == 0) set_status(v.status, ERR_TIMEOUT);
      break;
    }
    const int box = from_pages ? a.hp : BK_SUM_BOX;
    if (lane == 0) mbar_arrive_expect_tx(&full[stage], (uint32_t)((valid + box - 1) / box * box) * 2u * ROW_BYTES);
    __syncwarp();
    if (src >= 0) {
      // rows beyond the kept count inside the last summary box are older kept rows or zeros (finite), masked by the row count
      const CUtensorMap *mk = from_pages ? tmK : tmKs, *mv = from_pages ? tmV : tmVs;
      const uint32_t kdst = smem_u32(ring + stage * BK_STAGE_BYTES) + (uint32_t)(lane * box) * 128u, vdst = kdst + BK_TILE_BYTES;
      tma_load_2d(kdst, mk, 0, src, &full[stage]);
      tma_load_2d(kdst + BK_KBLOCK_BYTES, mk, 64, src, &full[stage]);
      tma_load_2d(vdst, mv, 0, src, &full[stage]);
      tma_load_2d(vdst + BK_KBLOCK_BYTES, mv, 64, src, &full[stage]);
    }
    if (FILL_PAUSE_NS > 0 && i < STAGES - 1) __nanosleep(FILL_PAUSE_NS);
  }
  return i;
}

// normalises one query row's columns 4 c4 .. +3 and writes them (bf16) and, from c4 == 0, the row's lse
__device__ __forceinline__ void write_block_out(const BlockArgs& a, int s, int row, int c4, const float4& acc, float mC,
                                                float lC) {
  if (row >= a.R) return;
  const float inv = (lC > 0.f) ? (1.f / lC) : 0.f;
  const long long off = q_row_offset(a, s, row);
  uint2 w;
  w.x = pack_bf16x2(acc.x * inv, acc.y * inv);
  w.y = pack_bf16x2(acc.z * inv, acc.w * inv);
  *reinterpret_cast<uint2*>(a.out + off + c4 * 4) = w;
  if (a.lse && c4 == 0) a.lse[off / D] = (lC > 0.f) ? (mC + log2f(lC)) * 0.69314718055994530942f : -INFINITY;
}

// After the n_warps warps of a CTA have written its split's records: takes a ticket; the last CTA of the sequence merges all splits'
// records and writes the output.  `flag`: an int in shared memory; `sync`: barrier of those warps.
// A record is a trip to L2 away: the (m, l) pairs of a warp's rows come side by side, a split per lane (there are at most 32), then the
// accumulators of four rows at a time: 8 sequences x 9000 rows x 128 queries in 18 splits 85.9 us with a row and a record after the other, 48.5 so;
// 64 x 4099 x 64 in 2 splits 49.0 and 41.1.
template <typename Sync>
__device__ __forceinline__ void block_merge_splits(const BlockArgs& a, int s, int n_splits, int* flag, int warp, int lane, int n_warps, Sync sync) {
  sync();
  // the ticket publishes this CTA's records (release, cumulative over the barrier) and shows the last arriver the others'
  if (warp == 0 && lane == 0) {
    int ticket;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(ticket) : "l"(a.counters + s) : "memory");
    *flag = ticket == n_splits - 1;
  }
  sync();
  if (*flag == 0) return;        // somebody else finishes later and merges
  const float* base = a.partials + (long long)s * a.max_splits * a.rec_rows * BK_REC;
  const long long stride = (long long)a.rec_rows * BK_REC;
#pragma unroll 1
  for (int r0 = warp; r0 < a.R; r0 += 4 * n_warps) {
    float m[4], l[4], f[4];      // rows r0 + x n_warps; f: weight of split `lane`
    float4 acc[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int r = r0 + x * n_warps;
      const float2 ml = r < a.R && lane < n_splits ? __ldcg(reinterpret_cast<const float2*>(base + lane * stride + r * BK_REC + 128)) : make_float2(-INFINITY, 0.f);
      m[x] = ml.x;
      l[x] = ml.y;
      acc[x] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const float mine = m[x];
      m[x] = warp_max(mine);
      f[x] = mine == -INFINITY ? 0.f : exp2f(mine - m[x]);
      l[x] = warp_sum(l[x] * f[x]);
    }
#pragma unroll 2
    for (int k = 0; k < n_splits; ++k)
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int r = r0 + x * n_warps;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < a.R) o = __ldcg(reinterpret_cast<const float4*>(base + k * stride + r * BK_REC) + lane);
        const float w = __shfl_sync(0xffffffffu, f[x], k);
        acc[x] = make_float4(fmaf(o.x, w, acc[x].x), fmaf(o.y, w, acc[x].y), fmaf(o.z, w, acc[x].z), fmaf(o.w, w, acc[x].w));
      }
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (r0 + x * n_warps < a.R) write_block_out(a, s, r0 + x * n_warps, lane, acc[x], m[x], l[x]);
  }
  if (warp == 0 && lane == 0) a.counters[s] = 0;      // leave the ticket counter clean for the next launch
}

}  // namespace kve
