// Flash-decode over the retained set (Sec. 3.3, softmax of Eq. 1):
//   out = softmax(q K'^T * scale) V',  rows of K', V' = [raw tail] ++ [kept chunks, oldest first]
// and, with mode = DENSE, Eq. 1 over every stored token (the full-cache baseline).
//
// HBM-bound: every retained K and V row (256 bytes each) is read exactly once, so the kernel is built
// to keep every SM streaming from its first microsecond to its last:
//  * A sequence's rows form 64-row tiles (raw tail first, kept chunks after it).  The host picks k,
//    the number of equal parts every sequence is cut into, so that the S k parts divide evenly over
//    the CTAs of one resident wave (two per SM); CTA c takes parts [c S k / G, (c + 1) S k / G): a
//    contiguous run that may span several sequences.  Its pipeline runs across sequence boundaries
//    without draining, every CTA moves nearly the same number of bytes whatever S is, and where a
//    part begins follows from the launch arguments, the stored length and one keep count, so the
//    first copies leave two dependent loads after the kernel starts.
//  * Warp 8 (producer) turns tiles into copies (TMA engine, global -> shared, mbarrier byte counting): one K and one V copy per
//    chunk that a tile touches (kept summary rows sit compacted in one run per sequence: one copy), into a 3-stage ring
//    of 64-row tiles.  The query row of a sequence travels with the first tile of that sequence.  Up to 32 tiles are worked
//    out side by side, one per lane (page ids included), and the lanes take turns at issuing theirs: a tile costs the
//    waits and the copies.  With the work done tile by tile the warp needed 1700 cycles a tile (divisions by the chunk
//    size, shuffles, 64-bit addresses) and held everything back: 8 layers of 128 sequences x 330 rows 9.75 us a
//    layer, 8.75 us so.  (With the page of every ROW looked up, 512 sequences x 1100 rows took 56.7 us, 5.0 TB/s;
//    49.8 us now.)
//  * While the predecessor on the stream still runs, a warp goes through the CTA's first tiles on what the tables hold (a
//    guess, which tells the producer after its wait where to look) and others pull the guessed rows of two tiles into L2:
//    12.7 -> 11.4 us a layer in that setting.
//  * Warps 0-7 (consumers) are two groups of four that take tiles in turn, 16 rows per warp.  (One group: 8.75 us a layer, two:
//    8.2 us - a tile is ~1400 cycles of dependent steps, and two of them now run at a time.)  The logits q.k are eight
//    warp-level MMAs (the rows are the M side, q fills the N side: bf16 products, fp32 sums), which leaves a group of
//    four lanes with the logits of two rows; online
//    softmax with warp shuffles, then p.V in fp32 with half a warp per row and 8 output dims per lane.  When a CTA's run
//    leaves a sequence, the consumers drop their (m, l, acc) into a double-buffered exchange area and carry on with the
//    next sequence.
//  * Warp 9 (merger) folds the eight consumer states of a finished sequence (or part of one), and
//    either writes the output (this CTA had the whole sequence) or a partial record plus an atomic
//    ticket; the CTA that draws a sequence's last ticket merges its records by log-sum-exp.  Nobody
//    spins on another CTA.
//  * Fused append (kvE_decode_step): the step's new token need not be in its page yet.  Its row is streamed from the
//    caller's buffer as the last row of the raw tail, the CTA that streams it also stores it in the page, and the stored
//    length is advanced once every CTA has read the old one: one launch per decode step and layer instead of two.
// Every mbarrier wait is bounded; on give-up the status word gets KVE_ERR_TIMEOUT.
#include "common.cuh"
#include "kernels.h"

namespace kve {

// Optional per-CTA time stamps (build with -DKVE_ATTN_STAMPS, see attn_stamps.py): where a launch's time goes.
// Slots: 0 kernel entry, 1 after the wait for the predecessor, 2 first copy issued, 3 first tile landed,
// 4 last tile consumed, 5 merger warp done, 6 producer warp done.  Compiled out of the product library.
#ifdef KVE_ATTN_STAMPS
constexpr int STAMP_CTAS = 2048, STAMP_SLOTS = 8;
__device__ unsigned long long g_attn_stamps[STAMP_CTAS * STAMP_SLOTS];
__device__ __forceinline__ void stamp(int slot) {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  if (blockIdx.x < STAMP_CTAS) g_attn_stamps[blockIdx.x * STAMP_SLOTS + slot] = t;
}
#define KVE_STAMP(cond, slot) do { if (cond) stamp(slot); } while (0)
#else
#define KVE_STAMP(cond, slot) do { } while (0)
#endif

constexpr int AT_TILE = ATTN_TILE_ROWS;       // rows per stage
constexpr int AT_STAGES = 3;
constexpr int AT_CGROUPS = 2;                 // consumer groups, which take tiles in turn
constexpr int AT_GWARPS = 4;                  // warps of a group
constexpr int AT_CWARPS = AT_CGROUPS * AT_GWARPS;
constexpr int AT_SUB = AT_TILE / AT_GWARPS;   // 16 rows per warp per tile: the rows of one m16n8k16 MMA
constexpr int AT_PRODUCER = AT_CWARPS;        // warp ids
constexpr int AT_GUESSER = 4;                 // consumer that guesses the first plan: the producer's scheduler, and no tile to prefetch
constexpr int AT_THREADS = (AT_CWARPS + 2) * 32;
constexpr int AT_STAGE_ELEMS = AT_TILE * D;   // bf16 elements of one K (or V) tile
constexpr int AT_LANE_SEGS = 3;               // chunks a tile may touch for one lane to issue its copies
constexpr int AT_SHORT_CHUNK = AT_TILE / (AT_LANE_SEGS - 1);      // that holds for all tiles with chunks of 32 tokens and more
constexpr int AT_PREFETCH_TILES = 2;          // most tiles a CTA pulls into L2 before its predecessor has finished
static_assert(AT_GUESSER % 4 == AT_PRODUCER % 4 && AT_GUESSER >= AT_PREFETCH_TILES && AT_GUESSER < AT_CWARPS, "the guessing warp");
static_assert(AT_SUB == 16, "the logits of a warp's rows are one m16n8k16 tile");

// shared-memory carve-up (bytes)
constexpr int AT_OFF_K = 0;
constexpr int AT_OFF_V = AT_OFF_K + AT_STAGES * AT_STAGE_ELEMS * 2;
constexpr int AT_OFF_Q = AT_OFF_V + AT_STAGES * AT_STAGE_ELEMS * 2;                 // [stages][128] bf16
constexpr int AT_OFF_COMB = AT_OFF_Q + AT_STAGES * ROW_BYTES;                       // [2][consumer warps][132] fp32
constexpr int AT_OFF_INFO = AT_OFF_COMB + 2 * AT_CWARPS * ATTN_PARTIAL_FLOATS * 4;  // [stages] int4
constexpr int AT_OFF_FINFO = AT_OFF_INFO + AT_STAGES * 16;                          // [2] int4
constexpr int AT_OFF_BAR = AT_OFF_FINFO + 2 * 16;                                   // full[3], empty[3], ffull[2], fempty[2]
constexpr int AT_OFF_GUESS = AT_OFF_BAR + (2 * AT_STAGES + 4) * 8;                  // [32] int4: the guessed first plan; its barrier
constexpr int AT_SMEM_BYTES = AT_OFF_GUESS + 32 * 16 + 16;
static_assert(AT_OFF_COMB % 16 == 0 && AT_OFF_INFO % 16 == 0 && AT_OFF_BAR % 8 == 0 && AT_OFF_GUESS % 16 == 0, "alignment of the carve-up");

int attn_smem_bytes() { return AT_SMEM_BYTES; }

// tile flags handed from the producer to the consumers
constexpr int TF_NEW = 1;      // first tile of a (sequence, list) in this CTA: fresh softmax state, query row in the stage
constexpr int TF_FLUSH = 2;    // last tile of a (sequence, list) in this CTA: hand the state to the merger afterwards
constexpr int TF_END = 4;      // no tile: the CTA's work is done

struct AttnArgs {
  LayerView v;
  FastDiv by_c, by_k;          // by the chunk size, by k
  int mode;
  int n_chunks;                // the host's count of chunks under the keep list: a prefetch hint; the kernel reads the device's
  int k;                       // parts per sequence
  const uint16_t* q;
  uint16_t* out;
  float* lse;
  float scale;
  const uint16_t* kkept;       // [S][max_chunks][128] kept summary rows, compacted (SUMMARY mode)
  const uint16_t* vkept;
  float* partials;             // [S + G][132]: the record of (sequence s, CTA c) sits at s + c
  int32_t* counters;           // [S], zero between launches
  // fused append (kvE_decode_step): one new token per sequence, placed at the length the device holds
  const uint16_t* k_new;       // [S][128] or null
  const uint16_t* v_new;
  int32_t* ticket;             // last CTA to finish publishes the new length
};

// what every role derives from the launch arguments and the stored length
struct AttnGeo {
  int n_tail, raw0, TT, per;   // tail rows / tiles per sequence; rows a kept chunk contributes
  int n;                       // tokens attended to (the new one included when one is being appended)
  int n_chunks;                // chunks the keep list covers (0 for full-cache attention)
  bool appending;              // the last tail row of every sequence is the new token, taken from k_new / v_new
};

// CTA c of P takes parts [c I / P, (c + 1) I / P); CTAs c >= P take none.  32-bit arithmetic (64-bit division
// would sit on the path to the first copy): the host keeps I * G below 2^32.
__device__ __forceinline__ uint32_t piece_begin(uint32_t c, uint32_t I, uint32_t P) { return c >= P ? I : (c * I) / P; }
// the CTA that holds part x
__device__ __forceinline__ uint32_t piece_of(uint32_t x, uint32_t I, uint32_t P) { return ((x + 1u) * P - 1u) / I; }

// bulk prefetch into L2 (16-byte aligned, a multiple of 16 bytes)
__device__ __forceinline__ void prefetch_l2_bulk(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
// read from L2 (never from a line that L1 may hold from before the predecessor finished)
__device__ __forceinline__ int load_hint(const int32_t* p) { return *reinterpret_cast<const volatile int32_t*>(p); }

// Pulls what the producer will look up for sequence s into L2 (fire and forget: the keep count, the page ids
// of the raw tail, the head of the kept-chunk list), so that the dependent look-ups that follow cost an L2 hit each.
__device__ __forceinline__ void prefetch_sequence_metadata(const AttnArgs& a, int s, int lane) {
  const LayerView& v = a.v;
  if (s < 0 || s >= v.S) return;
  const long long sb = (long long)s * v.max_chunks;
  const int first_tail_chunk = (a.mode == ATTN_DENSE) ? 0 : a.n_chunks;
  if (lane == 0) prefetch_l2(v.keep_cnt + s);
  // page ids of the tail: 32 entries per 128-byte line; up to 8 lines (256 chunks) ahead
  if (lane < 8 && first_tail_chunk + lane * 32 < v.max_chunks) prefetch_l2(v.page_table + sb + first_tail_chunk + lane * 32);
  if (a.mode == ATTN_RAW && lane == 8) prefetch_l2(v.keep_idx + sb);
}

// rows the kept chunks of sequence s contribute
__device__ __forceinline__ int lead_rows_from(const AttnArgs& a, const AttnGeo& g, int keep_cnt) {
  if (a.mode == ATTN_DENSE || g.n_chunks <= 0) return 0;
  return min(max(keep_cnt, 0), g.n_chunks) * g.per;
}
// up to 32 tiles of one sequence as the producer sees them, one per lane
struct TilePlan {
  int n, s;                         // tiles of the batch, their sequence (the same in every lane)
  int list, rows, flags;            // list 0: raw tail, 1: kept chunks
  int row0, c0, n_seg;              // first row in the list; its chunk (kept chunks: position in the keep list); chunks the tile touches
  int page[AT_LANE_SEGS];           // their pages (-1: none), when there are no more than that
  int i_new, new_page;              // the tile that ends with the token being appended (-1: none), that token's page
  uint4 new_row;                    // this lane's 16 bytes of it
};

// The rows of a tile that lie in one chunk: `pos` is the chunk (raw tail) or the index in the keep list (kept chunks at full
// resolution), `r` the first row inside it, `len` how many, `dst` where they go in the tile.
struct TileSegment { int pos, r, len, dst; };
__device__ __forceinline__ TileSegment tile_segment(int row0, int rows, int C, int pos) {
  TileSegment g;
  g.pos = pos;
  const int lo = max(row0, g.pos * C), hi = min(row0 + rows, g.pos * C + C);
  g.r = lo - g.pos * C;
  g.len = max(hi - lo, 0);
  g.dst = lo - row0;
  return g;
}

__device__ __forceinline__ AttnGeo make_geometry(const AttnArgs& a, int n, int listed) {
  AttnGeo g;
  n = min(max(n, 0), a.v.max_tokens);
  g.appending = a.k_new != nullptr && n < a.v.max_tokens;
  if (g.appending) n += 1;
  g.n = n;
  g.n_chunks = (a.mode == ATTN_DENSE) ? 0 : min(max(listed, 0), a.v.max_chunks);
  g.raw0 = g.n_chunks * a.v.C;
  g.n_tail = max(0, n - g.raw0);
  g.TT = (g.n_tail + AT_TILE - 1) / AT_TILE;
  g.per = (a.mode == ATTN_RAW) ? a.v.C : 1;
  return g;
}

// What the CTA will stream first, pulled into L2 while the predecessor on the stream is still running: lengths, keep lists and
// page ids are read before they are final, but only to guess addresses (checked against the pools), and a prefetch returns
// nothing - a wrong guess costs a few lines of L2, a right one (the decode loop: the same layer a token ago) takes the cold
// look-ups and the first rows off the path.  Warp w takes every AT_CWARPS-th of the CTA's first tiles in its first sequence.
__device__ __forceinline__ void prefetch_first_tiles(const AttnArgs& a, uint32_t i0, uint32_t i1, int warp, int lane) {
  const LayerView& v = a.v;
  const uint32_t uk = (uint32_t)a.k;
  const int s = (int)(i0 / uk);
  const AttnGeo g = make_geometry(a, load_hint(v.seq_len), a.mode == ATTN_DENSE ? 0 : load_hint(v.n_listed));
  const int keep = a.mode == ATTN_DENSE ? 0 : load_hint(v.keep_cnt + s);
  const int lead = min(max(keep, 0), g.n_chunks) * g.per;
  const int tiles = g.TT + (lead + AT_TILE - 1) / AT_TILE;
  const uint32_t p_lo = i0 - (uint32_t)s * uk, p_hi = min(i1 - (uint32_t)s * uk, uk);
  const int j0 = (int)((p_lo * (uint32_t)tiles) / uk), j1 = min((int)((p_hi * (uint32_t)tiles) / uk), j0 + AT_PREFETCH_TILES);
  const long long sb = (long long)s * v.max_chunks;
  for (int j = j0 + warp; j < j1; j += AT_CWARPS) {
    const bool tail = j < g.TT;
    const int jj = tail ? j : j - g.TT, rows = min(AT_TILE, (tail ? g.n_tail : lead) - jj * AT_TILE);
    if (!tail && a.mode == ATTN_SUMMARY) {
      if (lane < 2) prefetch_l2_bulk((lane ? a.vkept : a.kkept) + (sb + jj * AT_TILE) * D, (uint32_t)rows * ROW_BYTES);
      continue;
    }
    const int row0 = (tail ? g.raw0 : 0) + jj * AT_TILE;
    const TileSegment sg = tile_segment(row0, rows, v.C, (int)a.by_c.div((uint32_t)row0) + lane);
    if (sg.len <= 0 || sg.pos >= v.max_chunks) continue;
    const int chunk = tail ? sg.pos : load_hint(v.keep_idx + sb + sg.pos);
    if (chunk < 0 || chunk >= v.max_chunks) continue;
    const long long page = load_hint(v.page_table + sb + chunk);
    if (page < 0 || page >= v.n_pages) continue;
    const long long off = (page * v.C + sg.r) * D;
    prefetch_l2_bulk(v.k_pages + off, (uint32_t)sg.len * ROW_BYTES);
    prefetch_l2_bulk(v.v_pages + off, (uint32_t)sg.len * ROW_BYTES);
  }
}

// SHORT: chunks below 32 tokens, of which a tile may touch more than AT_LANE_SEGS
template <bool SHORT>
__global__ void __launch_bounds__(AT_THREADS, 2) kve_decode_attn_kernel(AttnArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  uint16_t* Ks = reinterpret_cast<uint16_t*>(smem + AT_OFF_K);
  uint16_t* Vs = reinterpret_cast<uint16_t*>(smem + AT_OFF_V);
  uint16_t* Qs = reinterpret_cast<uint16_t*>(smem + AT_OFF_Q);
  float* comb = reinterpret_cast<float*>(smem + AT_OFF_COMB);
  int4* info = reinterpret_cast<int4*>(smem + AT_OFF_INFO);
  int4* finfo = reinterpret_cast<int4*>(smem + AT_OFF_FINFO);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + AT_OFF_BAR);
  uint64_t* empty = full + AT_STAGES;
  uint64_t* ffull = empty + AT_STAGES;
  uint64_t* fempty = ffull + 2;
  int4* guess = reinterpret_cast<int4*>(smem + AT_OFF_GUESS);
  uint64_t* guessed = reinterpret_cast<uint64_t*>(guess + 32);

  pdl_launch_dependents();
  const LayerView& v = a.v;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  KVE_STAMP(threadIdx.x == 0, 0);
  // this CTA's parts follow from the launch arguments alone
  const uint32_t c = blockIdx.x, uk = (uint32_t)a.k;
  const uint32_t n_items = (uint32_t)v.S * uk, n_pieces = min(gridDim.x, n_items);
  const uint32_t i0 = piece_begin(c, n_items, n_pieces), i1 = piece_begin(c + 1, n_items, n_pieces);
  if (i0 < i1 && warp == AT_PRODUCER) prefetch_sequence_metadata(a, (int)(i0 / uk), lane);
  if (threadIdx.x == 0) {
    mbar_init(guessed, 1);
    for (int i = 0; i < AT_STAGES; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], AT_CWARPS);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&ffull[i], AT_CWARPS);
      mbar_init(&fempty[i], 1);
    }
    mbar_fence_init();
  }
  __syncthreads();
  if (warp == AT_PRODUCER || warp == AT_GUESSER) {
    // ================= producer warp (and, up to the first plan, a consumer that has nothing to do yet) =================
    // walks the CTA's parts in order, sequence by sequence; within a sequence the tiles [j, j_hi) that its parts in this CTA
    // cover (part p of a sequence with T tiles: tiles [p T / k, (p + 1) T / k))
    const int s_first = (int)(i0 / uk), s_last = i0 < i1 ? (int)((i1 - 1u) / uk) : s_first;
    AttnGeo g;
    int s = s_first, j = 0, j_hi = 0, lt_rows = 0, keep_next = 0;
    bool fresh = true, done = i0 >= i1;
    auto enter_sequence = [&](int keep_cnt) {
      lt_rows = lead_rows_from(a, g, keep_cnt);
      const uint32_t tiles = (uint32_t)(g.TT + (lt_rows + AT_TILE - 1) / AT_TILE);
      // part p of the sequence's tiles: [p tiles / k, (p + 1) tiles / k); p <= 32 and tiles < 2^20, so 32 bits do
      const uint32_t p_lo = (s == s_first) ? i0 - (uint32_t)s * uk : 0u;
      const uint32_t p_hi = (s == s_last) ? i1 - (uint32_t)s * uk : uk;
      j = (int)a.by_k.div(p_lo * tiles);
      j_hi = (int)a.by_k.div(p_hi * tiles);
      fresh = true;
      if (s < s_last) {      // the next one's look-ups: its keep count now, the rest into L2
        keep_next = (a.mode == ATTN_DENSE) ? 0 : load_hint(v.keep_cnt + s + 1);
        prefetch_sequence_metadata(a, s + 1, lane);
      }
    };
    auto page_of = [&](int seq, int list, int pos) -> int {      // -1: names nothing
      const long long sb = (long long)seq * v.max_chunks;
      int chunk = pos;
      if (list != 0) chunk = pos < v.max_chunks ? load_hint(v.keep_idx + sb + pos) : -1;
      return (chunk >= 0 && chunk < (list != 0 ? g.n_chunks : v.max_chunks)) ? load_hint(v.page_table + sb + chunk) : -1;
    };
    // The next tiles of a sequence, up to 32, worked out side by side: lane i holds tile i and will issue its copies.  `guess`: a
    // plan whose page ids are taken over where it looked at the same tail chunks.
    auto make_plan = [&](TilePlan& p, const TilePlan* guess) {
      p.n = 0;
      p.i_new = -1;
      if (done) return;
      const int left = j_hi - j, idx = j + lane;
      p.n = min(32, max(left, 1));       // parts without a tile: an empty one keeps the bookkeeping uniform
      p.s = s;
      p.list = idx >= g.TT ? 1 : 0;
      const int jj = p.list ? idx - g.TT : idx;
      p.rows = lane < left ? min(AT_TILE, (p.list ? lt_rows : g.n_tail) - jj * AT_TILE) : 0;
      p.flags = (fresh && lane == 0 ? TF_NEW : 0) | (idx + 1 >= j_hi ? TF_FLUSH : 0);
      p.row0 = (p.list ? 0 : g.raw0) + jj * AT_TILE;
      p.c0 = (int)a.by_c.div((uint32_t)p.row0);
      p.n_seg = (p.rows > 0 && (p.list == 0 || a.mode == ATTN_RAW)) ? (int)a.by_c.div((uint32_t)(p.row0 + p.rows - 1)) - p.c0 + 1 : 0;
      if (p.n_seg <= AT_LANE_SEGS) {
        const bool known = guess != nullptr && p.list == 0 && guess->list == 0 && guess->c0 == p.c0 && guess->n_seg >= p.n_seg;
#pragma unroll
        for (int x = 0; x < AT_LANE_SEGS; ++x) p.page[x] = known ? guess->page[x] : (x < p.n_seg ? page_of(s, p.list, p.c0 + x) : -1);
      }
      // fused append: the last row of the tail is the new token; whoever streams it also stores it in its page (lanes 0-15 the K
      // row, 16-31 the V row, 16 bytes each)
      const int i_new = g.TT - 1 - j;
      if (g.appending && i_new >= 0 && i_new < min(32, left)) {
        p.i_new = i_new;
        p.new_page = page_of(s, 0, (int)a.by_c.div((uint32_t)(g.n - 1)));
        p.new_row = __ldcg(reinterpret_cast<const uint4*>((lane >> 4 ? a.v_new : a.k_new) + (long long)s * D) + (lane & 15));
      }
      j += p.n;
      fresh = false;
      if (j >= j_hi) {
        if (s == s_last) done = true;
        else { ++s; enter_sequence(keep_next); }
      }
    };

    // The first tiles are worked out twice: by a consumer warp from what the tables hold while the predecessor still runs - only
    // a guess at where to look, and a way to have the code at hand - and by the producer from the real values, when the look-ups
    // of the length, the coverage, the keep count and the guessed page ids go out together.  Without a predecessor there is no
    // guess yet when the producer comes by, and it does not wait for one.  (The producer guessing first, in
    // front of its own wait, and the rows' prefetch in front of the barrier below: 8 sequences behind a kernel of another library 8.4 us,
    // 6.6 so; 128 x 330 rows 8.4 and 6.6; in chains of decode steps 0.1 us for it.)
    TilePlan cur, nxt;
    nxt.n = 0;
    const bool real = warp == AT_PRODUCER;
    if (real) {
      pdl_wait();      // lengths, keep lists, summaries and the new token come from earlier kernels
      KVE_STAMP(lane == 0, 1);
    }
    const int len_stored = load_hint(v.seq_len);
    // chunks the keep list covers: the device's own count, so that a launch replayed from a CUDA graph follows the
    // gate triggers that happened since it was captured (the launch argument is only the host's view at capture time)
    const int listed = (a.mode == ATTN_DENSE) ? 0 : load_hint(v.n_listed);
    const int keep_cnt = (a.mode == ATTN_DENSE || done) ? 0 : load_hint(v.keep_cnt + s_first);
    if (real && !done && __all_sync(0xffffffffu, mbar_test_wait(guessed, 0))) {
      const int4 gs = guess[lane];
      nxt.n = 1;
      nxt.list = gs.x; nxt.c0 = gs.y; nxt.n_seg = gs.z;
#pragma unroll
      for (int x = 0; x < AT_LANE_SEGS; ++x) nxt.page[x] = (nxt.list == 0 && x < nxt.n_seg) ? page_of(s_first, 0, nxt.c0 + x) : -1;
    }
    g = make_geometry(a, len_stored, listed);
    if (!done) enter_sequence(keep_cnt);
    make_plan(cur, nxt.n > 0 ? &nxt : nullptr);
    if (!real) {
      if (cur.n > 0) {
        guess[lane] = make_int4(cur.list, cur.c0, cur.n_seg, 0);
        __syncwarp();
        if (lane == 0) mbar_arrive(guessed);      // release
      }
    } else {
      if (a.k_new != nullptr && !g.appending && blockIdx.x == 0 && lane == 0) set_status(v.status, ERR_CAPACITY);   // cache full

      // The copies of tile i of the batch: lane i waits for the stage, publishes the tile's description and issues one K and one V
      // copy per chunk the tile touches, all from its own registers; the lanes take turns.  Chunks so short that a tile may
      // have more than AT_LANE_SEGS of them: the whole warp, 32 chunks at a time, their pages `pg` looked up a tile ahead, and chunks
      // that follow one another in the pool (pages dealt out in order) in one copy.  (One copy per chunk, looked up when its
      // turn came: 60 sequences x 2000 rows in chunks of one token 48.8 us, 17.5 so with the pages in order, 43.3 scattered; 128 x 4160 in
      // chunks of 4 and 16 tokens 71 -> 66 and 51 -> 48.)  False on a timed-out wait.
      auto look_up = [&](const TilePlan& p, int i, int (&pg)[2]) {
        const int n_seg = __shfl_sync(0xffffffffu, p.n_seg, i), c0 = __shfl_sync(0xffffffffu, p.c0, i), list = __shfl_sync(0xffffffffu, p.list, i);
#pragma unroll
        for (int h = 0; h < 2; ++h) pg[h] = n_seg > AT_LANE_SEGS && lane + 32 * h < n_seg ? page_of(p.s, list, c0 + lane + 32 * h) : -1;
      };
      int it = 0;
      auto issue = [&](const TilePlan& p, int i, const int (&pg)[2]) -> bool {
        const int stage = it % AT_STAGES, round = it / AT_STAGES;
        ++it;
        uint16_t *kd = Ks + stage * AT_STAGE_ELEMS, *vd = Vs + stage * AT_STAGE_ELEMS;
        const bool with_new = i == p.i_new;
        bool ok = true;
        if (lane == i) {
          ok = round == 0 || mbar_wait_bounded(&empty[stage], (round - 1) & 1);
          if (ok) {
            info[stage] = make_int4(p.s, p.rows, p.flags, p.list);
            const bool with_q = (p.flags & TF_NEW) != 0;
            mbar_arrive_expect_tx(&full[stage], (uint32_t)p.rows * 2u * ROW_BYTES + (with_q ? (uint32_t)ROW_BYTES : 0u));      // release: whoever sees the phase sees the description
            if (p.n_seg > 0 && p.n_seg <= AT_LANE_SEGS) {
              int r = p.row0 - p.c0 * v.C, dst = 0, rest = p.rows - (with_new ? 1 : 0);
#pragma unroll
              for (int x = 0; x < AT_LANE_SEGS; ++x) {
                const int len = min(v.C - r, rest);
                if (len > 0) {
                  int page = p.page[x];
                  if (page < 0 || page >= v.n_pages) { set_status(v.status, ERR_CAPACITY); page = 0; }
                  const long long off = ((long long)page * v.C + r) * D;
                  bulk_g2s(kd + dst * D, v.k_pages + off, (uint32_t)len * ROW_BYTES, &full[stage]);
                  bulk_g2s(vd + dst * D, v.v_pages + off, (uint32_t)len * ROW_BYTES, &full[stage]);
                }
                dst += len; rest -= len; r = 0;
              }
            } else if (p.n_seg == 0 && p.rows > 0) {      // kept summary rows: one contiguous run per sequence
              const long long off = ((long long)p.s * v.max_chunks + p.row0) * D;
              bulk_g2s(kd, a.kkept + off, (uint32_t)p.rows * ROW_BYTES, &full[stage]);
              bulk_g2s(vd, a.vkept + off, (uint32_t)p.rows * ROW_BYTES, &full[stage]);
            }
            if (with_new) {
              bulk_g2s(kd + (p.rows - 1) * D, a.k_new + (long long)p.s * D, ROW_BYTES, &full[stage]);
              bulk_g2s(vd + (p.rows - 1) * D, a.v_new + (long long)p.s * D, ROW_BYTES, &full[stage]);
            }
            if (with_q) bulk_g2s(Qs + stage * D, a.q + (long long)p.s * D, ROW_BYTES, &full[stage]);
          } else {
            set_status(v.status, ERR_TIMEOUT);
          }
        }
        ok = __shfl_sync(0xffffffffu, (int)ok, i) != 0;
        if constexpr (SHORT) {
          const int n_seg = __shfl_sync(0xffffffffu, p.n_seg, i);
          if (ok && n_seg > AT_LANE_SEGS) {
            const int row0 = __shfl_sync(0xffffffffu, p.row0, i), c0 = __shfl_sync(0xffffffffu, p.c0, i);
            const int rows = __shfl_sync(0xffffffffu, p.rows, i) - (with_new ? 1 : 0);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (32 * h >= n_seg) break;
              TileSegment sg = tile_segment(row0, rows, v.C, c0 + lane + 32 * h);
              if (lane + 32 * h >= n_seg) sg.len = 0;
              int page = pg[h];
              if (sg.len > 0 && (page < 0 || page >= v.n_pages)) { set_status(v.status, ERR_CAPACITY); page = 0; }
              const long long row = (long long)page * v.C + sg.r;      // of the pool
              const long long end = row + sg.len, end_before = __shfl_up_sync(0xffffffffu, end, 1);
              const bool head = sg.len > 0 && (lane == 0 || row != end_before);
              const unsigned heads = __ballot_sync(0xffffffffu, head), live = __ballot_sync(0xffffffffu, sg.len > 0);      // live: the first lanes
              const unsigned above = lane == 31 ? 0u : heads & ~((2u << lane) - 1u);
              const int last = (above ? __ffs(above) - 1 : __popc(live)) - 1;      // last chunk of the run that starts here
              const int run = __shfl_sync(0xffffffffu, sg.dst + sg.len, last & 31) - sg.dst;
              if (head) {
                bulk_g2s(kd + sg.dst * D, v.k_pages + row * D, (uint32_t)run * ROW_BYTES, &full[stage]);
                bulk_g2s(vd + sg.dst * D, v.v_pages + row * D, (uint32_t)run * ROW_BYTES, &full[stage]);
              }
            }
            __syncwarp();
          }
        }
        return ok;
      };
      bool ok = true;
      int pg[2] = {-1, -1}, pg_next[2] = {-1, -1};
      if (SHORT && cur.n > 0) look_up(cur, 0, pg);
      while (ok && cur.n > 0) {
        for (int i = 0; ok && i < cur.n; ++i) {
          if (i == cur.n - 1) make_plan(nxt, nullptr);      // its look-ups run while this batch's last copies are issued
          if constexpr (SHORT) {
            if (i < cur.n - 1) look_up(cur, i + 1, pg_next);
            else if (nxt.n > 0) look_up(nxt, 0, pg_next);
          }
          ok = issue(cur, i, pg);
          if constexpr (SHORT) { pg[0] = pg_next[0]; pg[1] = pg_next[1]; }
          KVE_STAMP(it == 1 && lane == 0, 2);
        }
        if (cur.i_new >= 0) {
          if (cur.new_page >= 0 && cur.new_page < v.n_pages)
            *(reinterpret_cast<uint4*>((lane >> 4 ? v.v_pages : v.k_pages) + ((long long)cur.new_page * v.C + (g.n - 1 - (int)a.by_c.div((uint32_t)(g.n - 1)) * v.C)) * D) + (lane & 15)) = cur.new_row;
          else if (lane == 0) set_status(v.status, ERR_CAPACITY);
        }
        cur = nxt;
      }
      // a description without a tile takes a stage of its own (no copies): that is how the consumers learn that they are done
      if (ok && lane == 0) {
        const int stage = it % AT_STAGES, round = it / AT_STAGES;
        if (round == 0 || mbar_wait_bounded(&empty[stage], (round - 1) & 1)) {
          info[stage] = make_int4(-1, 0, TF_END, 0);
          mbar_arrive(&full[stage]);
        } else {
          set_status(v.status, ERR_TIMEOUT);
        }
      }
      // Fused append: the length advances as soon as every CTA has read the old one, which is what the tickets count (nothing else
      // in the launch reads it; later launches wait for this one to complete).
      if (g.appending) {
        __syncwarp();
        int last = 0;
        if (lane == 0) {
          int arrived;
          asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(arrived) : "l"(a.ticket) : "memory");
          last = arrived == (int)gridDim.x - 1;
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last) {
          for (int b = lane; b < v.B; b += 32) v.seq_len[b] = g.n;
          if (lane == 0) *a.ticket = 0;      // clean for the next launch
        }
      }
      KVE_STAMP(lane == 0, 6);
    }
  }
  if (warp < AT_CWARPS) {
    // ================= consumer warps =================
    if (i0 < i1) prefetch_first_tiles(a, i0, i1, warp, lane);
    pdl_wait();
    const float sl2 = a.scale * 1.44269504088896340736f;   // logits kept in log2 units
    const int gwarp = warp % AT_GWARPS;
    const int g8 = lane >> 2, tig = lane & 3, odd = g8 & 1;              // MMA fragment coordinates: rows g8 and g8 + 8 of the warp's 16
    const int half = lane >> 4, l16 = lane & 15;           // p.V: rows 2 i + half, head dims 8 l16 .. + 7
    uint4 qf[4];                                           // q as the B operand (the same in all eight columns): 8 dims from 8 (tig + 4 j)
#pragma unroll
    for (int j = 0; j < 4; ++j) qf[j] = make_uint4(0u, 0u, 0u, 0u);
    float2 acc[4];
    float m = -INFINITY, l = 0.f;                          // l: this lane's rows only (replicated over tig), added up at the flush
#pragma unroll
    for (int x = 0; x < 4; ++x) acc[x] = make_float2(0.f, 0.f);
    int n_flush = 0;
    for (int i = 0;; ++i) {
      const int stage = i % AT_STAGES, round = i / AT_STAGES;
      if (!mbar_wait_bounded(&full[stage], round & 1)) {
        if (lane == 0) set_status(v.status, ERR_TIMEOUT);
        break;
      }
      const int4 ti = info[stage];                 // (sequence, rows, flags, list)
      KVE_STAMP(i == 0 && warp == 0 && lane == 0, 3);
      if (ti.z & TF_END) {
        KVE_STAMP(warp == 0 && lane == 0, 4);
        // tell the merger that nothing more comes
        const int fb = n_flush & 1;
        if (n_flush >= 2 && !mbar_wait_bounded(&fempty[fb], ((n_flush >> 1) - 1) & 1)) {
          if (lane == 0) set_status(v.status, ERR_TIMEOUT);
          break;
        }
        if (warp == 0 && lane == 0) finfo[fb] = make_int4(-1, 0, 0, 0);
        __syncwarp();
        if (lane == 0) mbar_arrive(&ffull[fb]);
        break;
      }
      if (ti.z & TF_NEW) {
#pragma unroll
        for (int j = 0; j < 4; ++j) qf[j] = *(reinterpret_cast<const uint4*>(Qs + stage * D) + tig + 4 * (j ^ odd));
        m = -INFINITY; l = 0.f;
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[x] = make_float2(0.f, 0.f);
      }
      const int nvalid = i % AT_CGROUPS == warp / AT_GWARPS ? min(max(ti.y - gwarp * AT_SUB, 0), AT_SUB) : 0;      // the other groups' tiles: only their flags
      if (nvalid > 0) {
        // ---- q.k of the warp's 16 rows: eight MMAs.  A lane fetches 8 consecutive head dims of a row at once; they feed the k
        // positions of two MMAs, for K and q alike (a contraction does not notice the order).  Odd rows and odd columns go through
        // the dims in another order than even ones, so that a quarter warp's two rows (256 bytes apart) lie in different banks:
        // of the eight columns, all of which hold q, those of the row's own parity are its logit.
        const uint4* kt = reinterpret_cast<const uint4*>(Ks + stage * AT_STAGE_ELEMS + (gwarp * AT_SUB) * D) + g8 * 16 + tig;
        // Every MMA starts from zero and the sums of 16 products are added up here: the tensor core cuts off what lies below the
        // last bit of its accumulator, an ordinary addition rounds.  (Two chains of four MMAs: a logit
        // of N(0, 1) rows off by 7.3e-8 rms and biased towards zero by 2.9e-8, 6.1e-8 and no bias so; 8 layers of 128 sequences x 330
        // rows 7.04 and 7.17 us a layer.)
        float2 d0[4], d1[4];      // rows g8, g8 + 8: both parities
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
          const uint4 ra = kt[4 * (j ^ odd)], rb = kt[4 * (j ^ odd) + 8 * 16];
          const uint32_t A0[4] = {ra.x, rb.x, ra.y, rb.y}, A1[4] = {ra.z, rb.z, ra.w, rb.w};
          mma_bf16_16816(c0, A0, qf[j].x, qf[j].y);
          mma_bf16_16816(c1, A1, qf[j].z, qf[j].w);
          d0[j] = add2(make_float2(c0[0], c0[1]), make_float2(c1[0], c1[1]));
          d1[j] = add2(make_float2(c0[2], c0[3]), make_float2(c1[2], c1[3]));
        }
        const float2 l0 = add2(add2(d0[0], d0[1]), add2(d0[2], d0[3])), l1 = add2(add2(d1[0], d1[1]), add2(d1[2], d1[3]));
        // ---- online softmax ----
        const float s0 = (g8 < nvalid) ? (odd ? l0.y : l0.x) * sl2 : -INFINITY;
        const float s1 = (g8 + 8 < nvalid) ? (odd ? l1.y : l1.x) * sl2 : -INFINITY;
        float mx = fmaxf(s0, s1);
#pragma unroll
        for (int o = 4; o <= 16; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float m_new = fmaxf(m, mx);
        // (logits of -inf only, so far: their weights are 0, not exp2(-inf + inf))
        const float m_sub = m_new == -INFINITY ? 0.f : m_new;
        const float p0 = ex2_fast(s0 - m_sub), p1 = ex2_fast(s1 - m_sub);
        const float alpha = ex2_fast(m - m_sub);
        l = fmaf(l, alpha, p0 + p1);
        m = m_new;
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[x] = mul2(acc[x], make_float2(alpha, alpha));
        // ---- p.V: half a warp per row, 16 bytes per lane ----
        const uint4* vt = reinterpret_cast<const uint4*>(Vs + stage * AT_STAGE_ELEMS + (gwarp * AT_SUB) * D) + half * 16 + l16;
#pragma unroll
        for (int i2 = 0; i2 < 8; ++i2) {
          const float pr = __shfl_sync(0xffffffffu, i2 < 4 ? p0 : p1, ((2 * i2 + half) & 7) * 4);
          if (2 * i2 + half < nvalid) {            // rows beyond the tile's last one hold stale bytes
            const uint4 w = vt[i2 * 32];
            const float2 pp = make_float2(pr, pr);
            acc[0] = fma2(pp, make_float2(bf16lo(w.x), bf16hi(w.x)), acc[0]);
            acc[1] = fma2(pp, make_float2(bf16lo(w.y), bf16hi(w.y)), acc[1]);
            acc[2] = fma2(pp, make_float2(bf16lo(w.z), bf16hi(w.z)), acc[2]);
            acc[3] = fma2(pp, make_float2(bf16lo(w.w), bf16hi(w.w)), acc[3]);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[stage]);
      if (ti.z & TF_FLUSH) {
        // hand (m, l, acc) of this (sequence, list) to the merger; the exchange area is double-buffered
        const int fb = n_flush & 1;
        if (n_flush >= 2 && !mbar_wait_bounded(&fempty[fb], ((n_flush >> 1) - 1) & 1)) {
          if (lane == 0) set_status(v.status, ERR_TIMEOUT);
          break;
        }
        float* cw = comb + (fb * AT_CWARPS + warp) * ATTN_PARTIAL_FLOATS;
        float tot[8], lt = l;
#pragma unroll
        for (int x = 0; x < 4; ++x) {      // even + odd rows
          tot[2 * x] = acc[x].x + __shfl_xor_sync(0xffffffffu, acc[x].x, 16);
          tot[2 * x + 1] = acc[x].y + __shfl_xor_sync(0xffffffffu, acc[x].y, 16);
        }
#pragma unroll
        for (int o = 4; o <= 16; o <<= 1) lt += __shfl_xor_sync(0xffffffffu, lt, o);
        *reinterpret_cast<float4*>(cw + l16 * 8 + half * 4) = half ? make_float4(tot[4], tot[5], tot[6], tot[7]) : make_float4(tot[0], tot[1], tot[2], tot[3]);
        if (lane == 0) { cw[128] = m; cw[129] = lt; }
        if (warp == 0 && lane == 0) finfo[fb] = make_int4(ti.x, ti.w, 0, 0);
        __syncwarp();
        if (lane == 0) mbar_arrive(&ffull[fb]);      // release
        ++n_flush;
      }
    }
  } else if (warp > AT_PRODUCER) {
    // ================= merger warp =================
    pdl_wait();
    for (int f = 0;; ++f) {
      const int fb = f & 1;
      if (!mbar_wait_bounded(&ffull[fb], (f >> 1) & 1)) {
        if (lane == 0) set_status(v.status, ERR_TIMEOUT);
        break;
      }
      const int4 fi = finfo[fb];                   // (sequence, -, -, -); sequence < 0: no more work
      const int s = fi.x;
      if (s < 0) break;
      // ---- the consumer states -> one ----
      const float* cb = comb + fb * AT_CWARPS * ATTN_PARTIAL_FLOATS;
      float mC = -INFINITY;
#pragma unroll
      for (int w = 0; w < AT_CWARPS; ++w) mC = fmaxf(mC, cb[w * ATTN_PARTIAL_FLOATS + 128]);
      float lC = 0.f, accC[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int w = 0; w < AT_CWARPS; ++w) {
        const float mw = cb[w * ATTN_PARTIAL_FLOATS + 128];
        const float sc = (mw == -INFINITY) ? 0.f : exp2f(mw - mC);
        lC = fmaf(cb[w * ATTN_PARTIAL_FLOATS + 129], sc, lC);
        const float4 av = *reinterpret_cast<const float4*>(cb + w * ATTN_PARTIAL_FLOATS + lane * 4);
        accC[0] = fmaf(av.x, sc, accC[0]); accC[1] = fmaf(av.y, sc, accC[1]);
        accC[2] = fmaf(av.z, sc, accC[2]); accC[3] = fmaf(av.w, sc, accC[3]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&fempty[fb]);     // the exchange buffer may be refilled

      // ---- which CTAs hold parts of sequence s ----
      const uint32_t c0 = piece_of((uint32_t)s * uk, n_items, n_pieces), c1 = piece_of((uint32_t)(s + 1) * uk - 1u, n_items, n_pieces);
      const int n_parts = (int)(c1 - c0 + 1u);
      if (n_parts > 1) {
        float* mine = a.partials + (long long)(s + c) * ATTN_PARTIAL_FLOATS;
        *reinterpret_cast<float4*>(mine + lane * 4) = make_float4(accC[0], accC[1], accC[2], accC[3]);
        if (lane == 0) { mine[128] = mC; mine[129] = lC; }
        // The ticket is an acquire-release atomic at device scope: taken by lane 0 after the warp has synchronised, it
        // publishes the whole warp's record (release is cumulative over what the barrier ordered before it) and, for the
        // last arriver, makes the other CTAs' records visible to the warp once it has synchronised again - one round
        // trip to L2 instead of fence, atomic, fence.
        __syncwarp();
        int ticket = 0;
        if (lane == 0)
          asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(ticket) : "l"(a.counters + s) : "memory");
        ticket = __shfl_sync(0xffffffffu, ticket, 0);
        if (ticket != n_parts - 1) continue;       // somebody else finishes later and merges
        __syncwarp();
        // records of sequence s: CTAs c0 .. c1, at s + c0 .. s + c1; lanes fetch the (m, l) pairs side by side
        const float* base = a.partials + (long long)(s + c0) * ATTN_PARTIAL_FLOATS;
        mC = -INFINITY;
        for (int p = lane; p < n_parts; p += 32) mC = fmaxf(mC, __ldcg(base + (long long)p * ATTN_PARTIAL_FLOATS + 128));
        mC = warp_max(mC);
        lC = 0.f;
        for (int p = lane; p < n_parts; p += 32) {
          const float mw = __ldcg(base + (long long)p * ATTN_PARTIAL_FLOATS + 128);
          const float sc = (mw == -INFINITY) ? 0.f : exp2f(mw - mC);
          lC = fmaf(__ldcg(base + (long long)p * ATTN_PARTIAL_FLOATS + 129), sc, lC);
        }
        lC = warp_sum(lC);
        accC[0] = accC[1] = accC[2] = accC[3] = 0.f;
#pragma unroll 4
        for (int p = 0; p < n_parts; ++p) {
          const float* ps = base + (long long)p * ATTN_PARTIAL_FLOATS;
          const float mw = __ldcg(ps + 128);
          const float4 av = __ldcg(reinterpret_cast<const float4*>(ps + lane * 4));
          const float sc = (mw == -INFINITY) ? 0.f : exp2f(mw - mC);
          accC[0] = fmaf(av.x, sc, accC[0]); accC[1] = fmaf(av.y, sc, accC[1]);
          accC[2] = fmaf(av.z, sc, accC[2]); accC[3] = fmaf(av.w, sc, accC[3]);
        }
        if (lane == 0) a.counters[s] = 0;          // leave the ticket counter clean for the next launch
      }
      const float inv = (lC > 0.f) ? (1.f / lC) : 0.f;
      uint2 o;
      o.x = pack_bf16x2(accC[0] * inv, accC[1] * inv);
      o.y = pack_bf16x2(accC[2] * inv, accC[3] * inv);
      *reinterpret_cast<uint2*>(a.out + (long long)s * D + lane * 4) = o;
      if (a.lse && lane == 0) a.lse[s] = (lC > 0.f) ? (mC + log2f(lC)) * 0.69314718055994530942f : -INFINITY;
    }
    KVE_STAMP(lane == 0, 5);
  }
}

cudaError_t launch_attn(const LayerView& v, AttnMode mode, int n_chunks, int parts_per_seq, int grid, const void* q, void* out,
                        float* lse, float scale, const void* kkept, const void* vkept, float* partials, int32_t* counters,
                        const void* k_new, const void* v_new, int32_t* ticket, cudaStream_t st) {
  if (v.S <= 0) return cudaSuccess;
  const bool is_short = v.C < AT_SHORT_CHUNK;
  static DeviceFlags opted, opted_short;
  {
    const cudaError_t e = is_short ? smem_opt_in(opted_short, kve_decode_attn_kernel<true>, AT_SMEM_BYTES)
                                   : smem_opt_in(opted, kve_decode_attn_kernel<false>, AT_SMEM_BYTES);
    if (e != cudaSuccess) return e;
  }
  AttnArgs a;
  a.by_c = fast_div((uint32_t)v.C); a.by_k = fast_div((uint32_t)(parts_per_seq < 1 ? 1 : parts_per_seq));
  a.v = v; a.mode = (int)mode; a.n_chunks = n_chunks; a.k = parts_per_seq < 1 ? 1 : parts_per_seq;
  a.q = static_cast<const uint16_t*>(q); a.out = static_cast<uint16_t*>(out); a.lse = lse; a.scale = scale;
  a.kkept = static_cast<const uint16_t*>(kkept); a.vkept = static_cast<const uint16_t*>(vkept);
  a.partials = partials; a.counters = counters;
  a.k_new = static_cast<const uint16_t*>(k_new); a.v_new = static_cast<const uint16_t*>(v_new); a.ticket = ticket;
  return launch_pdl(is_short ? kve_decode_attn_kernel<true> : kve_decode_attn_kernel<false>, dim3((unsigned)(grid < 1 ? 1 : grid)), dim3(AT_THREADS), AT_SMEM_BYTES, st, a);
}

}  // namespace kve

#ifdef KVE_ATTN_STAMPS
// instrumented build only: copy the stamps of the last launch to the host / clear them
extern "C" int kve_attn_stamps_read(unsigned long long* host, int n) {
  return (int)cudaMemcpyFromSymbol(host, kve::g_attn_stamps, sizeof(unsigned long long) * n);
}
extern "C" int kve_attn_stamps_clear() {
  void* p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, kve::g_attn_stamps);
  if (e == cudaSuccess) e = cudaMemset(p, 0, sizeof(kve::g_attn_stamps));
  return (int)e;
}
#endif
