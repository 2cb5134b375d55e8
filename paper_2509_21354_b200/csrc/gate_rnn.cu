// The gate (Eq. 3): input projection, LSTM recurrence and score head, for every sequence, chunks oldest first:
//   pre_t = W_ih [Kbar_t ; Vbar_t] + b_ih + b_hh + W_hh h_{t-1};  i,f,o = sigmoid, g = tanh;  c_t = f c_{t-1} + i g;  h_t = o tanh(c_t)
//   s_t   = sigmoid(w_s . h_t + b_s)
//
// The chain over t is strictly sequential, so the kernel is built for latency per step:
//  * A thread-block cluster of CL CTAs owns NG groups of 8 sequences for all steps (NG = 2 when one
//    group per cluster would not fit the GPU in one wave: the groups are independent pipelines, and a
//    warp handles them one after the other, so one group's exchange overlaps the other's arithmetic).  Each CTA owns 64 hidden
//    units, i.e. 256 rows of W_hh; eight warps own 8 units each and keep their rows in REGISTERS as mma A fragments
//    for the whole kernel (128 registers per thread at d_g = 256).  (Sixteen warps, eight per group, with ten of the sixteen k
//    tiles' fragments read from shared memory because 128 registers do not hold them: 330 us on 512 sequences x 121
//    chunks, 347 us with the groups taking turns at the tensor cores, against 285 us then.)
//  * Per step the CTA computes its rows of W_hh h with warp-level tensor-core MMAs (m16n8k16, bf16 x bf16 -> fp32).  W_hh is
//    bf16 by definition; the fp32 state h enters as PL = 2 bf16 planes by default (h = hi + lo up to 2^-17 |h|: 16 of its 24
//    significant bits; a third plane makes the products exact, moves the scores by 1e-7 - far below what the fast
//    exponentials of the cell update contribute, 5e-5 - and costs a third more MMAs).  Each plane has its own
//    accumulators (as many independent MMA chains), added smallest plane first at the end.  128 MMAs per scheduler and round take
//    ~1000 cycles of ~2400, whether one warp or two issue them, and in as many chains as one likes: that is their rate.
//  * MMA rows are ordered so that one thread ends up holding the i, f, g, o pre-activations of the
//    same (hidden unit, sequence): the cell update is thread-local, c lives in registers.  The cells of two sequences are updated side by side
//    in packed operations (256 x 56 75.1 -> 74.3 us).  f, i and g share one reciprocal
//    and o and tanh(c) another (five exponentials and two reciprocals per element instead of five and five: the
//    special-function unit is what the cell update waits for).
//  * Input projection: a warp of a third warpgroup multiplies W_ih x_t a batch of GX_ROUNDS rounds (step, group) ahead on tcgen05.  The
//    CTA's 256 rows of W_ih are the left operand and stay in TENSOR memory (half of it); a batch's summary rows, 64 columns
//    of the product, come as four tiled copies (8 or 16 sequences x 8 or 4 consecutive chunks of 64 elements each); the two sets of
//    accumulators fill the other half.  Rows of W_ih are placed so that tcgen05.ld in its 16-lane shape hands a thread its own four
//    pre-activations of two sequences in the layout of the MMA fragments: two instructions a round.  As a kernel of its own
//    (a GEMM over all chunks, P = 254 MB on 512 sequences x 121 chunks written and read again) it took 70 us there, 25 us on 256 x 56, 11 us on
//    8 x 28 at d_g = 128; here it adds what the issue of its MMAs (32 a batch, ~68 cycles each whatever the columns) takes away from the
//    recurrence's warps: 3 us on 256 x 56 (77.5 us without them, 3 more if one warp issues all).  A chain of 300 chunks of 8 sequences pays more for that than the
//    GEMM cost it (348 -> 354 us; 8 x 400 at d_g = 128 315 -> 323), all others gain.  Issued by the recurrence's own warps it cost another 2 to 4 us and, with the branches
//    around it, 10 % of a round.
//  * Exchange of h_t: a warp writes the planes of its 8 hidden units into its own CTA's double-buffered h planes (two units per
//    4-byte word, after one shuffle), and sends them from there to every other CTA of the cluster in 16-byte asynchronous stores that
//    count their bytes on an mbarrier there, so a step costs one one-way transfer and no cluster-wide barrier.  (By bulk copies, with the proxy
//    fence that they need: 82 us on 256 sequences x 56 chunks, 80 so; 512 x 121 293 and 279 us.)  A CTA can only be sent step t+1 data after it has
//    itself sent step t data, i.e. after all its warps have finished reading the buffer that is being overwritten.
//  * The score head is not part of the chain: a warp leaves the products of w_s and h_t in shared memory, another warp of the third
//    warpgroup adds up its 8 units (d_g / 8 partial sums per (s, t) go to memory: an eighth of the bytes of h_t) and announces the bytes of
//    the next exchange, and when the chain is through the cluster adds the partial sums up in a fixed order.  (Both by the recurrence's
//    warps: 77 us on 60 sequences x 80 chunks at d_g = 128, 73.6 so.)
//  Measured, the whole gate: 512 sequences x 121 chunks 319 -> 264 us, 256 x 56 86.9 -> 73.4 us, 32 x 250 297.2 -> 296.2 us, 8 x 28 at d_g = 128
//  30 to 32 -> 27.0 us, 60 x 80 74.2 -> 69.4 us, 60 x 5 12.2 -> 8.8 us (before: projection and recurrence as two kernels, back to back).
//  Slower, with the kernels of that time: waiting for the CTA's own planes and the peers' apart, with the own units' MMAs in between (255 -> 261 us a step
//  on 256 sequences), the two warps of a scheduler taking turns at the tensor cores (512 x 121 279 -> 317 us), and the sums of the even and the
//  odd k tiles in accumulators of their own (286 -> 308 us).
// Every mbarrier wait is bounded (one second); on give-up the status word gets KVE_ERR_TIMEOUT and
// the CTA stops sending, which lets its peers run into their own limits and leave as well.
#include "gate_rnn.cuh"
#include "tensor_map.h"
#include "umma.cuh"

namespace kve {

// the input projection: rounds (step, group) of a batch, 8 columns of the product each; shared and tensor memory
constexpr int GX_ROUNDS = 8;
constexpr int GX_N = GX_ROUNDS * 8;                          // columns of a batch: (step, group, sequence)
constexpr int GX_KB = 2 * D / umma::KBLOCK_ELEMS;            // K-blocks of 64: keys' summary, values' summary
constexpr int GX_KB_BYTES = GX_N * umma::KBLOCK_ROW_BYTES;   // 8 KB
constexpr int GX_BYTES = GX_KB * GX_KB_BYTES;                // 32 KB
constexpr int GX_TMEM_W = 0;                                 // two tiles of 128 rows of W_ih, 128 columns (256 bf16) each
constexpr int GX_TMEM_ACC = 2 * D;                           // [batch & 1][tile][GX_N]
constexpr int GX_TMEM_COLS = 512;
static_assert(GX_TMEM_ACC + 4 * GX_N == GX_TMEM_COLS, "tensor memory");
// two warpgroups of the recurrence and a third with the projectors and the score warp (a warpgroup, because registers move
// between whole warpgroups: with 9 warps of equal shares the recurrence would have 168 registers)
constexpr int GATE_THREADS = RNN_THREADS + 128;
// registers per thread of the recurrence and of the third warpgroup, which share out those of the launch.  As few as none of them spills:
// what a launch leaves of an SM's registers is where the means of kvE_refresh's second range run (three planes at d_g = 256 with 232 and 40
// left room for none of their CTAs: kvE_refresh of 512 sequences x 121 chunks of 128, MLP, 1041 us, 926 so)
template <int DG, int PL>
constexpr int RNN_REGS = DG == 256 ? (PL == 3 ? 224 : 208) : (DG == 128 ? (PL == 3 ? 192 : 184) : 136);
template <int DG, int PL>
constexpr int PROJ_REGS = DG == 256 && PL == 3 ? 32 : (DG == 128 && PL == 3 ? 48 : 40);
template <int DG, int PL>
constexpr int GATE_REGS = (2 * RNN_REGS<DG, PL> + PROJ_REGS<DG, PL>) / 3;

// Optional cycle budget of one recurrence step (build with -DKVE_RNN_STAMPS, see rnn_stamps.py): warp 0 of CTA 0 adds
// up, over all steps and groups, the clock64 cycles between five points of a step - 0: waiting for the peers' h,
// 1: fragment loads + MMA chain, 2: start of a round (pre-activations asked for), 3: cell update, 4: splitting and sending h,
// 6: the rest of a round - and
// slot 5 counts the (step, group) rounds.  The marks are contiguous: the slots add up to the whole step loop.  Compiled out of the product library.
#ifdef KVE_RNN_STAMPS
__device__ unsigned long long g_rnn_cycles[8];
#define KVE_RNN_MARK(slot)                                                                   \
  do {                                                                                       \
    if (blockIdx.x == 0 && warp == 0 && lane == 0) {                                         \
      const long long now_ = clock64();                                                      \
      atomicAdd(&g_rnn_cycles[slot], (unsigned long long)(now_ - mark_));                    \
      mark_ = now_;                                                                          \
    }                                                                                        \
  } while (0)
#define KVE_RNN_MARK_BEGIN() long long mark_ = clock64()
__device__ unsigned long long g_rnn_once[8];
#define KVE_RNN_ONCE(slot)                                                                   \
  do {                                                                                       \
    if (blockIdx.x == 0 && threadIdx.x == 0) {                                               \
      unsigned long long t_;                                                                 \
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_));                                 \
      g_rnn_once[slot] = t_;                                                                 \
    }                                                                                        \
  } while (0)
#else
#define KVE_RNN_MARK(slot) do { } while (0)
#define KVE_RNN_MARK_BEGIN() do { } while (0)
#define KVE_RNN_ONCE(slot) do { } while (0)
#endif

// bytes in front of the summary rows: h buffers, products of the score, barriers
template <int DG, int NG, int PL>
constexpr int RNN_SMEM_X = NG * 2 * (DG / 8) * PL * 8 * 8 * 2 + NG * 2 * RNN_WARPS * 64 * 4 + (2 * NG + 5) * 8 + 8;

template <int DG, int CL, int NG, int PL, bool MANY>
__global__ void __cluster_dims__(CL, 1, 1) __maxnreg__((GATE_REGS<DG, PL>))
    kve_gate_rnn_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, RnnArgs a) {
  constexpr int HU = DG / CL;            // hidden units owned by this CTA
  constexpr int KT = DG / 16;            // k tiles
  constexpr int NS = 8;                  // sequences per group: the n of the m16n8k16 MMA
  constexpr int KBLK = PL * NS * 8;                     // bf16 elements of one k-block (8 units): [plane][sequence][8]
  constexpr int HS_BUF = (DG / 8) * KBLK;               // bf16 elements per h buffer
  constexpr uint32_t H_BYTES = PL * NS * (DG - HU) * 2; // bytes of h planes a CTA receives from its peers per step and group
  constexpr int OFF_PROD = NG * 2 * HS_BUF * 2;
  constexpr int PROD_BUF = RNN_WARPS * 8 * NS;          // floats: w_s h of a round, [warp][sequence & 1][sequence / 2][8 units]
  constexpr int OFF_BARS = OFF_PROD + NG * 2 * PROD_BUF * 4;
  constexpr int T = GX_ROUNDS / NG;                     // steps of a batch of the input projection
  constexpr bool P_LATE = DG < 256;                     // pre-activations fetched behind the MMAs, not in front: 77 us, 79 (60 sequences x 80 chunks, d_g = 128)
  constexpr bool PACE_BY_SENDS = DG == 256 && NG == 1;  // where in a round the projector's MMAs go out
  constexpr int SENDS = ((CL - 1) * PL * NS + 31) / 32;         // 16-byte messages to the peers per lane, step and group
  static_assert(HU == 8 * RNN_WARPS && KT % 2 == 0, "one pair of m16 tiles (8 units x 4 gates) per warp");
  // what the warpgroups ask for is exactly what the launch has, or the last one to ask would wait for good
  static_assert(3 * GATE_REGS<DG, PL> == 2 * RNN_REGS<DG, PL> + PROJ_REGS<DG, PL> && GATE_REGS<DG, PL> % 8 == 0 && RNN_REGS<DG, PL> % 8 == 0, "register split");
  static_assert(GATE_THREADS * GATE_REGS<DG, PL> + 2 * MEAN_BESIDE_REGS <= 65536, "two CTAs of kve_chunk_mean_beside_kernel fit beside this one");
  static_assert(OFF_BARS % 16 == 0, "16-byte pieces");

  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint16_t* hs = reinterpret_cast<uint16_t*>(smem_raw);                          // [NG][2][DG / 8][PL][NS][8]
  float* prod = reinterpret_cast<float*>(smem_raw + OFF_PROD);                   // [NG][2][PROD_BUF]
  uint64_t* hbar = reinterpret_cast<uint64_t*>(smem_raw + OFF_BARS);             // [NG][2] h planes landed
  uint64_t* x_full = hbar + 2 * NG;                                              // rows of a batch landed
  uint64_t* x_done = x_full + 1;                                                 // [2] pre-activations of a batch computed
  uint64_t* x_read = x_done + 2;                                                 // [2] ... and read by all warps
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(x_read + 2);
  volatile int* rounds_done = reinterpret_cast<volatile int*>(tmem_slot + 1);    // rounds of which warp 0 has its MMAs (or its sends) behind it
  // [GX_KB] K-blocks of summary rows, on a 1024-byte boundary
  unsigned char* xs = smem_raw + ((smem_u32(smem_raw) + RNN_SMEM_X<DG, NG, PL> + 1023u) & ~1023u) - smem_u32(smem_raw);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);      // (the same in all lanes, for the compiler to see)
  const int g = lane >> 2, tig = lane & 3;
  const uint32_t rank = cluster_rank();
  // A cluster takes a set of NS NG sequences, or (MANY) one set after the other: group gi owns sequences seq0 + 8 gi .. + 7
  int seq0 = (blockIdx.x / CL) * NS * NG;
  const int seq_step = MANY ? (int)(gridDim.x / CL) * NS * NG : 0;
  const int ug = (int)rank * HU + warp * 8 + g;                // this thread's hidden unit

  KVE_RNN_ONCE(0);
  if (tid == 0) {
    for (int i = 0; i < 2 * NG; ++i) mbar_init(&hbar[i], RNN_WARPS + 1);
    *rounds_done = 0;
    mbar_init(x_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&x_done[i], 2);
      mbar_init(&x_read[i], RNN_WARPS);
    }
    mbar_fence_init();
  }
  if (warp == 0) umma::tmem_alloc(tmem_slot, GX_TMEM_COLS);
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tmem = *tmem_slot;

  const int n_batches = (a.n_range + T - 1) / T;
  // what the barriers have seen of earlier sets: batches of the projection, exchanges through buffer b of h (bit b: an odd number)
  int batches_before = 0, exchanged = 0;
  auto next_set = [&]() {      // false: that was the last one
    if (!MANY || (seq0 += seq_step) >= a.S) return false;
    batches_before += n_batches;
    exchanged ^= ((a.n_range - 1) / 2 & 1) | (a.n_range / 2 & 1) << 1;
    return true;
  };
  // a warp's worth of partial sums from the products of a round: lane = (warp, sequence / 2), for both halves of the sequences
  auto put_scores = [&](int gi, int step) {
    const float* src = prod + (gi * 2 + (step & 1)) * PROD_BUF;
    const int w = lane & 7, pair = lane >> 3;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float4 x = *reinterpret_cast<const float4*>(src + ((w * 2 + e) * 4 + pair) * 8), y = *reinterpret_cast<const float4*>(src + ((w * 2 + e) * 4 + pair) * 8 + 4);
      const int s = seq0 + gi * NS + pair * 2 + e;
      if (s < a.S) a.H[(long long)(s * a.n_range + step) * (DG / 8) + rank * RNN_WARPS + w] = ((x.x + x.y) + (x.z + x.w)) + ((y.x + y.y) + (y.z + y.w));
    }
  };
  if (warp >= RNN_WARPS) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"((PROJ_REGS<DG, PL>)));
    // ================= projector warps =================
    // Pre-activations W_ih x_t a batch of GX_ROUNDS rounds ahead of the recurrence.  Each of the two issues the MMAs of one tile: every
    // issue holds up the other warps of its scheduler for some 45 cycles, wherever in the round it falls, and this way two schedulers
    // share them (256 sequences x 56 chunks 78.5 -> 76.9 us, 32 x 250 320 -> 312).
    pdl_wait();      // the summaries come from earlier kernels
    __syncthreads();      // W_ih is in tensor memory, and xs, its staging area, is free
    umma::fence_after_sync();
    bool ok = true;      // (a CTA that has given up takes part in the meetings of the cluster until the last set)
    do {
      cluster_arrive();      // the recurrence's first meeting, which this warp has nothing to wait for
      int n_fetched = 0, n_begun = 0;
      if ((warp == RNN_WARPS || warp == RNN_WARPS + 2) && lane == 0 && ok) {
        const int tile = warp == RNN_WARPS ? 0 : 1;
        asm volatile("fence.proxy.async.global;" ::: "memory");
        for (int b = 0; b < n_batches && ok; ++b) {
          const int run = batches_before + b, buf = run & 1;
          // the rows of all steps and sequences of the batch: a copy per K-block, zeros beyond the store (what it brings beyond the range
          // or from another layer goes into columns that nobody reads)
          if (tile == 0) {
            mbar_arrive_expect_tx(x_full, GX_BYTES);
#pragma unroll
            for (int kb = 0; kb < GX_KB; ++kb)
              tma_load_3d(smem_u32(xs) + kb * GX_KB_BYTES, kb < GX_KB / 2 ? &map_k : &map_v, (kb & 1) * umma::KBLOCK_ELEMS, a.seq_base + seq0, a.t0 + b * T, x_full);
          }
          n_fetched = run + 1;
          ok = mbar_wait_bounded(x_full, (uint32_t)(run & 1)) && (run < 2 || mbar_wait_bounded(&x_read[buf], (uint32_t)(((run >> 1) - 1) & 1)));
          if (!ok) break;
          umma::fence_after_sync();
          n_begun = run + 1;
          const uint32_t acc = tmem + GX_TMEM_ACC + (uint32_t)((buf * 2 + tile) * GX_N);
          // A K-block at a time, when warp 0 reports the right moment of a round (for the pace only: the wait gives up soon): behind its
          // sends at d_g = 256, where the recurrence then waits for its peers (32 x 250 312 -> 303 us), behind its MMAs below (8 x 400 at
          // d_g = 128 333 -> 321.5).  With two groups there is always somebody at work: a tile at a time (512 x 121 285 -> 277 us).
#pragma unroll 1
          for (int kb = 0; kb < GX_KB; ++kb) {
            const int due = NG == 1 ? (b - 1) * GX_ROUNDS + 1 + 2 * kb : (b - 1) * GX_ROUNDS + 2 + 3 * tile;
            if (b > 0 && (NG == 1 || kb == 0))
              for (int poll = 0; poll < 2048 && *rounds_done < due; ++poll) __nanosleep(30);
#pragma unroll
            for (int k = 0; k < 4; ++k)
              umma::mma_bf16_ts(acc, tmem + GX_TMEM_W + (uint32_t)(tile * D + kb * 32 + k * 8), umma::smem_desc(smem_u32(xs) + kb * GX_KB_BYTES + k * 32),
                                umma::instr_desc_bf16(128, GX_N), (kb | k) != 0);
          }
          umma::commit(&x_done[buf]);
          ok = mbar_wait_bounded(&x_done[buf], (uint32_t)((run >> 1) & 1));      // the rows may be overwritten
        }
        if (!ok) {      // nothing is under way any more when the CTA leaves
          set_status(a.status, ERR_TIMEOUT);
          mbar_wait_bounded(x_full, (uint32_t)((n_fetched - 1) & 1));
          if (n_begun > 0) mbar_wait_bounded(&x_done[(n_begun - 1) & 1], (uint32_t)(((n_begun - 1) >> 1) & 1));
        }
      }
      if (warp == RNN_WARPS + 1) {
        // ================= score warp =================
        // Announces the bytes of every exchange, and adds up what the warps leave of w_s . h_t when it is through (eight units in pairs;
        // the warps' sums go to memory).  Its arrival for the next exchange says that it has read what that one will overwrite.
        for (int step = 0; step + 1 < a.n_range && ok; ++step) {
          const int buf = (step + 1) & 1;
          if (lane < NG) {
            if (CL > 1) mbar_arrive_expect_tx(&hbar[2 * lane + buf], H_BYTES);
            else mbar_arrive(&hbar[2 * lane + buf]);
          }
          for (int gi = 0; gi < NG && ok; ++gi) {
            ok = __all_sync(0xffffffffu, mbar_wait_cluster_bounded(&hbar[2 * gi + buf], (uint32_t)(((exchanged >> buf) + (step >> 1)) & 1)));
            if (ok) put_scores(gi, step);
          }
          __syncwarp();      // all lanes have read: an arrival orders only what its own lane has done
        }
        if (!ok && lane == 0) set_status(a.status, ERR_TIMEOUT);
      }
      __syncwarp();
      cluster_wait();
      cluster_sync_all();
    } while (next_set());
    return;
  }

  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(RNN_REGS<DG, PL>));
  // ---- W_ih rows of this CTA into tensor memory, the left operand of the input projection ------------------------
  // Tile w / 4, lanes 32 (w % 4) .. are the rows of warp w in the order of its MMA fragments: lane l = row (l & 7) of gate l >> 3.
  // A K-block (32 rows x 128 bytes) at a time through the warp's share of the X area.
  const uint32_t tmem_mine = tmem + ((uint32_t)(warp & 3) << 21);      // this warp's quarter of the lanes
  unsigned char* w_stage = xs + warp * (32 * umma::KBLOCK_ROW_BYTES);
  auto fetch_w_ih = [&](int kb) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = i * 4 + (lane >> 3), p = lane & 7;
      cp_async16(w_stage + umma::piece_offset(r, p),
                 a.W_ih + ((long long)(r >> 3) * DG + (int)rank * HU + warp * 8 + (r & 7)) * (2 * D) + kb * umma::KBLOCK_ELEMS + p * 8, true);
    }
  };
  auto store_w_ih = [&](int kb) {
    cp_async_wait_all();
    __syncwarp();
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      uint32_t r[16];
#pragma unroll
      for (int p = 0; p < 4; ++p)
        *reinterpret_cast<uint4*>(&r[4 * p]) = *reinterpret_cast<const uint4*>(w_stage + umma::piece_offset(lane, half * 4 + p));
      umma::tmem_st16_nowait(tmem_mine + GX_TMEM_W + (uint32_t)((warp >> 2) * D + kb * 32 + half * 16), r);
    }
    __syncwarp();      // read by all lanes: the next K-block may come
  };

  // ---- W_hh rows of this CTA as A fragments ---------------------------------------------------------------------
  // Register j of the fragment of k tile kt holds the two bf16 at k = 16 kt + 8 (j >> 1) + 2 tig of row (j & 1): word
  // 8 kt + 4 (j >> 1) + tig of the row.  The four lanes of a group (equal g) fetch 16 consecutive words of the row with one
  // 16-byte load each (lane tig: words 4 tig ..) and turn the 4 x 4 block among themselves with shuffles, so that lane tig
  // ends up with words tig, 4 + tig, 8 + tig, 12 + tig: a quarter of the load instructions of word-by-word fetches (5 -> 2 us).
  // A pair of k tiles for both m tiles at a time:
  auto load_pair = [&](int kp, uint32_t (&f)[2][2][4]) {      // f[m tile][k tile of the pair]
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int rs = 0; rs < 2; ++rs) {
        const uint4 w = __ldg(reinterpret_cast<const uint4*>(a.W_hh + ((long long)(mt * 2 + rs) * DG + ug) * DG) + kp * 4 + tig);
        const bool hi = (tig & 2) != 0, lo = (tig & 1) != 0;
        // lanes t and t ^ 2 swap halves: afterwards y0, y1 come from lane (t & 1), y2, y3 from lane (t & 1) + 2, words 2 hi, 2 hi + 1
        const uint32_t r0 = __shfl_xor_sync(0xffffffffu, hi ? w.x : w.z, 2), r1 = __shfl_xor_sync(0xffffffffu, hi ? w.y : w.w, 2);
        const uint32_t y0 = hi ? r0 : w.x, y1 = hi ? r1 : w.y, y2 = hi ? w.z : r0, y3 = hi ? w.w : r1;
        // lanes t and t ^ 1 swap the word the other one wants
        const uint32_t u0 = __shfl_xor_sync(0xffffffffu, lo ? y0 : y1, 1), u1 = __shfl_xor_sync(0xffffffffu, lo ? y2 : y3, 1);
        const uint32_t k0 = lo ? y1 : y0, k1 = lo ? y3 : y2;
        f[mt][0][rs] = lo ? u0 : k0;              // word tig of the lane group's 16
        f[mt][0][rs + 2] = lo ? k0 : u0;          // word 4 + tig
        f[mt][1][rs] = lo ? u1 : k1;              // word 8 + tig
        f[mt][1][rs + 2] = lo ? k1 : u1;          // word 12 + tig
      }
  };
  uint32_t A[KT / 2][2][2][4];
#pragma unroll
  for (int kb = 0; kb < GX_KB; ++kb) {
    fetch_w_ih(kb);
#pragma unroll
    for (int kp = kb * KT / 2 / GX_KB; kp < (kb + 1) * KT / 2 / GX_KB; ++kp) load_pair(kp, A[kp]);
    store_w_ih(kb);
  }
  const float w_score = __ldg(a.w_s + ug);
  float bias[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) bias[q] = __ldg(a.b_ih + q * DG + ug) + __ldg(a.b_hh + q * DG + ug);
  umma::tmem_st_wait();

  KVE_RNN_ONCE(1);
  pdl_wait();      // the weights are in place; the carried state comes from earlier kernels
  // only now, when all earlier work is complete: a launch may run beside this kernel without waiting for anything (kvE_refresh)
  pdl_launch_dependents();
  if (a.list_cut >= 0 && blockIdx.x == 0 && tid == 0) *a.n_listed = a.list_cut;
  KVE_RNN_ONCE(2);
  umma::fence_smem_to_async();
  umma::fence_before_sync();
  __syncthreads();      // W_ih is in tensor memory: the projector may start
  bool alive = true;
  do {
    if (MANY && tid == 0) *rounds_done = 0;
    // ---- initial state: every CTA needs the full h of its sequences as planes in buffer 0 of each group -------------
    for (int i = tid; i < NG * NS * (DG / 2); i += RNN_THREADS) {
      const int js = i / (DG / 2), k2 = i % (DG / 2);      // js: sequence of the cluster, 0 .. 8 NG - 1
      const int j = js % NS, s = seq0 + js;
      float h0 = 0.f, h1 = 0.f;
      if (!a.reset && s < a.S) {
        const float2 hv = *reinterpret_cast<const float2*>(a.lstm_h + (long long)s * DG + k2 * 2);
        h0 = hv.x; h1 = hv.y;
      }
      uint32_t p0[3], p1[3];      // the leading PL pieces are used
      split3(h0, p0);
      split3(h1, p1);
#pragma unroll
      for (int pl = 0; pl < PL; ++pl)
        *reinterpret_cast<uint32_t*>(hs + js / NS * 2 * HS_BUF + (k2 >> 2) * KBLK + (pl * NS + j) * 8 + (k2 & 3) * 2) = p0[pl] | (p1[pl] << 16);
    }
    // state of the sequences 2 tig, 2 tig + 1 of every group
    float2 c[NG], hlast[NG];
#pragma unroll
    for (int gi = 0; gi < NG; ++gi) {
      const int s = seq0 + gi * NS + tig * 2;
      const bool even = !a.reset && s < a.S, odd = !a.reset && s + 1 < a.S;
      const long long at = (long long)s * DG + ug;
      c[gi] = make_float2(even ? a.lstm_c[at] : 0.f, odd ? a.lstm_c[at + DG] : 0.f);
      hlast[gi] = make_float2(even ? a.lstm_h[at] : 0.f, odd ? a.lstm_h[at + DG] : 0.f);
    }

    // message m of a warp goes to peer (rank + 1 + m / rows of a block): row m % rows of that CTA's buffers, as an address in the cluster window
    uint32_t peer_hs[SENDS > 0 ? SENDS : 1];
#pragma unroll
    for (int x = 0; x < SENDS; ++x)
      peer_hs[x] = map_to_rank(smem_u32(hs), (rank + 1 + (lane + 32 * x) / (PL * NS)) % CL) + (lane + 32 * x) % (PL * NS) * 16;

    // barriers initialised and buffer 0 filled in every CTA before anyone sends
    KVE_RNN_ONCE(3);
    cluster_sync_all();
    KVE_RNN_ONCE(4);

    KVE_RNN_MARK_BEGIN();
    for (int batch = 0; batch < n_batches && alive; ++batch) {
      // ---- the pre-activations of the next T steps' inputs
      const int run = batches_before + batch;
      alive = __all_sync(0xffffffffu, mbar_wait_bounded(&x_done[run & 1], (uint32_t)((run >> 1) & 1)));
      if (!alive) {
        if (lane == 0) set_status(a.status, ERR_TIMEOUT);
        break;
      }
      umma::fence_after_sync();
      uint32_t acc_x = tmem_mine + GX_TMEM_ACC + (uint32_t)(((run & 1) * 2 + (warp >> 2)) * GX_N);
      const int step_end = min(batch * T + T, a.n_range);
      for (int step = batch * T; step < step_end; ++step) {
        const int buf = step & 1;
        const bool send_h = step + 1 < a.n_range;
#pragma unroll
        for (int gi = 0; gi < NG; ++gi) {
          uint16_t* hs_g = hs + gi * 2 * HS_BUF;
          uint64_t* hbar_g = hbar + 2 * gi;
          // pre-activations of the round's inputs, in the layout of the MMA accumulators
          uint32_t pin[2][4];
          auto ask_pin = [&]() {
            umma::tmem_ld_frag_nowait(acc_x, pin[0]);
            umma::tmem_ld_frag_nowait(acc_x + (16u << 16), pin[1]);
            acc_x += 8;
          };
          if (!P_LATE) ask_pin();
          KVE_RNN_MARK(2);
          // ---- h_{t-1} from every CTA of the cluster (each buffer completes once per two steps) -----------------------------
          if (step > 0) {
            // (one poll usually waits long enough: it is the only thing in the way then)
            const uint32_t parity = ((exchanged >> buf) + ((step - 1) >> 1)) & 1;
            if (!__all_sync(0xffffffffu, mbar_try_wait_cluster(&hbar_g[buf], parity))) {
              alive = __all_sync(0xffffffffu, mbar_wait_cluster_bounded(&hbar_g[buf], parity));
              if (!alive) {
                if (lane == 0) set_status(a.status, ERR_TIMEOUT);
                break;
              }
            }
          }
          KVE_RNN_MARK(0);

          // ---- W_hh h_{t-1} on the tensor cores: one accumulator set per plane ---------------------------------------------
          float acc[PL][2][4];
#pragma unroll
          for (int pl = 0; pl < PL; ++pl)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
              for (int e = 0; e < 4; ++e) acc[pl][mt][e] = 0.f;
          // B fragments: one ldmatrix.x4 brings the 8 sequences x 32 k-values of a plane (two k tiles);
          // lane l addresses row (l & 7) of the 8 x 8 block (l >> 3).
          const uint32_t hb_lane = smem_u32(hs_g + buf * HS_BUF + (lane >> 3) * KBLK + (lane & 7) * 8);
          uint32_t bf[2][PL][4];
          auto load_b = [&](int kp) {
#pragma unroll
            for (int pl = 0; pl < PL; ++pl) ldmatrix_x4(bf[kp & 1][pl], hb_lane + (uint32_t)((kp * 4 * KBLK + pl * NS * 8) * 2));
          };
          load_b(0);
#pragma unroll
          for (int kp = 0; kp < KT / 2; ++kp) {
            if (kp + 1 < KT / 2) load_b(kp + 1);      // a pair of k tiles ahead
#pragma unroll
            for (int half = 0; half < 2; ++half)
#pragma unroll
              for (int pl = 0; pl < PL; ++pl)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) mma_bf16_16816(acc[pl][mt], A[kp][mt][half], bf[kp & 1][pl][2 * half], bf[kp & 1][pl][2 * half + 1]);
          }
          if (!PACE_BY_SENDS && tid == 0) *rounds_done = step * NG + gi + 1;
          KVE_RNN_MARK(1);

          // (the vote is a scheduling fence: without it the compiler draws what follows into the MMA chain, 10 % of a step)
          if (!__all_sync(0xffffffffu, alive)) break;
          if (P_LATE) ask_pin();
          umma::tmem_ld_wait_frags(pin[0], pin[1]);
          // ---- cell update (thread-local), planes of h_t into this CTA's buffer ---------------------
          float2 pre[4];       // both sequences: 0 = i, 1 = f (tile 0, rows g / g+8), 2 = g, 3 = o (tile 1)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int mt = q >> 1, ai = (q & 1) * 2;
            float2 sum = make_float2(acc[PL - 1][mt][ai], acc[PL - 1][mt][ai + 1]);      // smallest plane first
#pragma unroll
            for (int pl = PL - 2; pl >= 0; --pl) sum = add2(sum, make_float2(acc[pl][mt][ai], acc[pl][mt][ai + 1]));
            pre[q] = add2(sum, add2(make_float2(__uint_as_float(pin[mt][ai]), __uint_as_float(pin[mt][ai + 1])), make_float2(bias[q], bias[q])));
          }
          const float2 hv = lstm_cell_pair(pre, c[gi]);
          hlast[gi] = hv;
          KVE_RNN_MARK(3);
          // products of the score: nothing of the chain waits for their sum
          {
            float* mine = prod + (gi * 2 + buf) * PROD_BUF + (warp * 2 * 4 + tig) * 8 + g;
            mine[0] = w_score * hv.x;
            mine[4 * 8] = w_score * hv.y;
          }
          // ---- the warp's k-block (8 units: [plane][sequence][8], contiguous) to every CTA of the cluster ----
          if (send_h) {
            const uint32_t off = (uint32_t)(((gi * 2 + (buf ^ 1)) * HS_BUF + ((int)rank * RNN_WARPS + warp) * KBLK) * 2);
            // lanes g and g ^ 1 hold neighbouring units: an even g takes both units of sequence 2 tig, an odd one those of 2 tig + 1, and
            // a warp's store instruction is a whole plane of the block: 128 bytes in a row
            const bool odd = (g & 1) != 0;
            unsigned char* mine = reinterpret_cast<unsigned char*>(hs) + off + (tig * 2 + (g & 1)) * 16 + (g >> 1) * 4;
            uint32_t pl[3];      // planes of both sequences, the even one below
            split3_pair(hv.x, hv.y, pl);
            const uint32_t h0 = __byte_perm(pl[0], pl[1], 0x5410), h1 = __byte_perm(pl[0], pl[1], 0x7632);      // two planes of a sequence
            const uint32_t keep = odd ? h1 : h0, got = __shfl_xor_sync(0xffffffffu, odd ? h0 : h1, 4);
            *reinterpret_cast<uint32_t*>(mine) = __byte_perm(odd ? got : keep, odd ? keep : got, 0x5410);
            *reinterpret_cast<uint32_t*>(mine + NS * 16) = __byte_perm(odd ? got : keep, odd ? keep : got, 0x7632);
            if constexpr (PL == 3) {
              const uint32_t got2 = __shfl_xor_sync(0xffffffffu, pl[2], 4);
              *reinterpret_cast<uint32_t*>(mine + 2 * NS * 16) = __byte_perm(odd ? got2 : pl[2], odd ? pl[2] : got2, odd ? 0x7632 : 0x5410);
            }
            __syncwarp();
            // peers: 16-byte rows out of the own block, each counted in bytes on the receiver's barrier; lane l sends message l, l + 32 ..
#pragma unroll
            for (int x = 0; x < SENDS; ++x) {
              const uint4 row = *reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned char*>(hs) + off + (lane + 32 * x) % (PL * NS) * 16);
              if (x * 32 + lane < (CL - 1) * PL * NS)
                st_async_cluster(peer_hs[x] + off, row, peer_hs[x] - (lane + 32 * x) % (PL * NS) * 16 + OFF_BARS + (2 * gi + (buf ^ 1)) * 8);
            }
            if (lane == 0) mbar_arrive(&hbar_g[buf ^ 1]);     // release: this warp's own pieces are in place
          }
          if (PACE_BY_SENDS && tid == 0) *rounds_done = step + 1;
          KVE_RNN_MARK(4);
#ifdef KVE_RNN_STAMPS
          if (blockIdx.x == 0 && tid == 0) atomicAdd(&g_rnn_cycles[5], 1ull);
#endif
          KVE_RNN_MARK(6);
        }
        if (!alive) break;
      }
      umma::fence_before_sync();      // this warp's loads out of the accumulators come before what the projector writes there next
      __syncwarp();
      if (lane == 0) mbar_arrive(&x_read[run & 1]);
    }

    KVE_RNN_ONCE(5);
    // ---- carried state out ---------------------------------------------------------------------------
#pragma unroll
    for (int gi = 0; gi < NG; ++gi)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int s = seq0 + gi * NS + tig * 2 + e;
        if (s < a.S && alive) {
          a.lstm_c[(long long)s * DG + ug] = e ? c[gi].y : c[gi].x;
          a.lstm_h[(long long)s * DG + ug] = e ? hlast[gi].y : hlast[gi].x;
        }
      }
    // (the last step's products, which no exchange follows)
    asm volatile("bar.sync 1, %0;" ::"n"(RNN_THREADS) : "memory");
    if (warp < NG && alive) put_scores(warp, a.n_range - 1);
    // nobody leaves while a peer may still be sending into its shared memory; the partial sums of all CTAs are in place behind it
    cluster_sync_all();
    KVE_RNN_ONCE(6);
    if (!MANY && warp == 0) umma::tmem_dealloc(tmem, GX_TMEM_COLS);
    // ---- score head: s_t = sigmoid(w_s . h_t + b_s); a row's d_g / 8 partial sums lie side by side and are added in order -----------
    const int n_seq = min(NS * NG, a.S - seq0);
    for (int i = (int)rank * RNN_THREADS + tid; i < n_seq * a.n_range; i += CL * RNN_THREADS) {
      const float4* src = reinterpret_cast<const float4*>(a.H + ((long long)seq0 * a.n_range + i) * (DG / 8));
      float sum = 0.f;
#pragma unroll
      for (int q = 0; q < DG / 32; ++q) {
        const float4 x = __ldcg(src + q);
        sum += x.x; sum += x.y; sum += x.z; sum += x.w;
      }
      const int s = i / a.n_range;
      a.scores[(long long)(seq0 + s) * a.max_chunks + a.t0 + (i - s * a.n_range)] = 1.f / (1.f + expf(-(sum + a.b_s)));
    }
  } while (next_set());
  if (MANY && warp == 0) umma::tmem_dealloc(tmem, GX_TMEM_COLS);
}

// Clusters that the current device holds at a time
template <int DG, int CL, int NG, int PL, bool MANY>
static cudaError_t resident_clusters(cudaLaunchConfig_t cfg, int* most) {
  static std::atomic<int> known[MAX_DEVICES];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  *most = known[dev].load(std::memory_order_acquire);
  if (*most > 0) return cudaSuccess;
  cudaLaunchAttribute shape[1];
  shape[0].id = cudaLaunchAttributeClusterDimension;
  shape[0].val.clusterDim.x = CL;
  shape[0].val.clusterDim.y = shape[0].val.clusterDim.z = 1;
  cfg.attrs = shape;
  cfg.numAttrs = 1;
  e = cudaOccupancyMaxActiveClusters(most, kve_gate_rnn_kernel<DG, CL, NG, PL, MANY>, &cfg);
  if (e == cudaSuccess && *most < 1) e = cudaErrorInvalidConfiguration;
  if (e == cudaSuccess) known[dev].store(*most, std::memory_order_release);
  return e;
}

template <int DG, int CL, int NG, int PL, bool MANY = false>
static cudaError_t launch_rnn_t(const RnnArgs& a, const CUtensorMap* maps, cudaStream_t st) {
  constexpr int smem = RNN_SMEM_X<DG, NG, PL> + GX_BYTES + 1024;      // + slack to reach a 1024-byte boundary
  static DeviceFlags opted;
  {
    cudaError_t e = smem_opt_in(opted, kve_gate_rnn_kernel<DG, CL, NG, PL, MANY>, smem);
    if (e != cudaSuccess) return e;
  }
  int clusters = (a.S + 8 * NG - 1) / (8 * NG);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  // an SM keeps its division of shared memory and L1 as long as a CTA is there: all of it shared, for what may run beside this kernel
  attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  attr[1].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * CL);
  cfg.blockDim = dim3(GATE_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  if (MANY) {      // as few sets one after the other as all clusters at a time need
    int most = 0;
    const cudaError_t e = resident_clusters<DG, CL, NG, PL, MANY>(cfg, &most);
    if (e != cudaSuccess) return e;
    const int sets = (clusters + most - 1) / most;
    clusters = (clusters + sets - 1) / sets;
    cfg.gridDim = dim3(clusters * CL);
  }
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kve_gate_rnn_kernel<DG, CL, NG, PL, MANY>, maps[0], maps[1], a);
}

// CTAs of a cluster; two groups of 8 sequences per cluster once one group per cluster would need more than one wave of clusters
static int cluster_ctas(int d_g) { return d_g / 64; }
static bool two_groups(int S, int d_g) { return (S + 7) / 8 > sm_count() / cluster_ctas(d_g); }

// Microseconds per chunk (two planes of h, d_g = 256): 1.22 with one group of sequences per cluster, 2.28 with two, as measured when kvE_refresh's rule was
// fitted to them (1.18 and 2.18 now)
double gate_rnn_us_per_chunk(int S, int d_g, int planes) {
  const bool two = two_groups(S, d_g);
  const int clusters = (S + (two ? 15 : 7)) / (two ? 16 : 8), wave = sm_count() / cluster_ctas(d_g);
  return (two ? 2.28 : 1.22) * (planes == 3 ? 1.25 : 1.0) * ((clusters + wave - 1) / wave);
}

// More sequences than the clusters of one wave hold, and few chunks: the clusters of one wave go through several sets of sequences, because what a
// cluster does before its first round (weights into registers and tensor memory, 4 us) would be most of the launch.  us, a wave of new
// clusters for every set -> one wave: 4096 sequences x 1 chunk at d_g = 64, 128, 256 14.0 -> 11.0, 31.2 -> 20.2, 76.4 -> 45.1; 1200 x 16 at d_g = 128
// 59.9 -> 56.7, 2400 x 16 at d_g = 64 43.3 -> 43.0, 600 x 4 at d_g = 256 27.9 -> 26.6.  With more chunks the rounds of that instance, 5 % longer at d_g = 256
// and 2 % at 64, outweigh it: 600 x 8 at d_g = 256 44.0 -> 44.7, 2400 x 28 at d_g = 64 68.3 -> 69.3.
template <int DG>
constexpr int MANY_CHUNKS = DG == 256 ? 4 : 16;

template <int DG, int PL>
static cudaError_t launch_rnn_planes(const RnnArgs& a, const CUtensorMap* maps, cudaStream_t st) {
  constexpr int CL = DG / 64;
  if (!two_groups(a.S, DG)) return launch_rnn_t<DG, CL, 1, PL>(a, maps, st);
  const bool many = (a.S + 15) / 16 > sm_count() / CL && a.n_range <= MANY_CHUNKS<DG>;
  return many ? launch_rnn_t<DG, CL, 2, PL, true>(a, maps, st) : launch_rnn_t<DG, CL, 2, PL>(a, maps, st);
}

cudaError_t encode_gate_maps(void* maps, const void* ksum, const void* vsum, long long n_seq, int max_chunks, int S, int d_g) {
  static_assert(sizeof(CUtensorMap) == GATE_MAP_BYTES, "tensor map size");
  const int ng = two_groups(S, d_g) ? 2 : 1;
  for (int i = 0; i < 2; ++i) {
    // element, sequence, chunk: a box holds the sequences of a cluster at GX_ROUNDS / ng consecutive chunks
    const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)n_seq, (cuuint64_t)max_chunks};
    const cuuint64_t strides[2] = {(cuuint64_t)max_chunks * ROW_BYTES, (cuuint64_t)ROW_BYTES};
    const cuuint32_t box[3] = {(cuuint32_t)umma::KBLOCK_ELEMS, (cuuint32_t)(8 * ng), (cuuint32_t)(GX_ROUNDS / ng)};
    const cudaError_t e = encode_bf16_map(static_cast<CUtensorMap*>(maps) + i, i ? vsum : ksum, 3, dims, strides, box);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_gate_rnn(const LayerView& v, const void* maps, int seq_base, int t0, int t1, const uint16_t* W_ih, const uint16_t* W_hh, const float* b_ih, const float* b_hh,
                            const float* w_s, float b_s, int d_g, float* H, bool reset_state, int planes, int list_cut, cudaStream_t st) {
  if (t1 <= t0 || v.S <= 0) return cudaSuccess;
  if ((long long)v.S * (t1 - t0) >= (1LL << 31) - 128) return cudaErrorInvalidValue;
  const CUtensorMap* tm = static_cast<const CUtensorMap*>(maps);
  RnnArgs a;
  a.seq_base = seq_base; a.W_ih = W_ih; a.b_ih = b_ih; a.b_hh = b_hh;
  a.n_listed = v.n_listed; a.list_cut = list_cut;
  a.H = H; a.W_hh = W_hh; a.w_s = w_s; a.b_s = b_s;
  a.scores = v.scores; a.lstm_h = v.lstm_h; a.lstm_c = v.lstm_c; a.status = v.status;
  a.S = v.S; a.max_chunks = v.max_chunks; a.t0 = t0; a.n_range = t1 - t0; a.reset = reset_state ? 1 : 0;
  switch (d_g) {
    case 256: return planes == 3 ? launch_rnn_planes<256, 3>(a, tm, st) : launch_rnn_planes<256, 2>(a, tm, st);
    case 128: return planes == 3 ? launch_rnn_planes<128, 3>(a, tm, st) : launch_rnn_planes<128, 2>(a, tm, st);
    case 64:  return planes == 3 ? launch_rnn_planes<64, 3>(a, tm, st) : launch_rnn_planes<64, 2>(a, tm, st);
    default:  return cudaErrorInvalidValue;
  }
}

}  // namespace kve

#ifdef KVE_RNN_STAMPS
// instrumented build only: read and clear the cycle sums
extern "C" int kve_rnn_once_read(unsigned long long* host) {
  return (int)cudaMemcpyFromSymbol(host, kve::g_rnn_once, sizeof(kve::g_rnn_once));
}
extern "C" int kve_rnn_cycles_read(unsigned long long* host) {
  cudaError_t e = cudaMemcpyFromSymbol(host, kve::g_rnn_cycles, sizeof(kve::g_rnn_cycles));
  void* p = nullptr;
  if (e == cudaSuccess) e = cudaGetSymbolAddress(&p, kve::g_rnn_cycles);
  if (e == cudaSuccess) e = cudaMemset(p, 0, sizeof(kve::g_rnn_cycles));
  return (int)e;
}
#endif
