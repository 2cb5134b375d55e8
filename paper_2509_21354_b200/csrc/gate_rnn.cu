// LSTM recurrence + score head of the gate (Eq. 3): for every sequence, chunks oldest first,
//   pre_t = P_t + W_hh h_{t-1};  i,f,o = sigmoid, g = tanh;  c_t = f c_{t-1} + i g;  h_t = o tanh(c_t)
//   s_t   = sigmoid(w_s . h_t + b_s)
// P_t (= W_ih x_t + b_ih + b_hh) comes from the projection GEMM.
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
//    accumulators (as many independent MMA chains), added smallest plane first at the end.
//  * MMA rows are ordered so that one thread ends up holding the i, f, g, o pre-activations of the
//    same (hidden unit, sequence): the cell update is thread-local, c lives in registers.  f, i and g share one reciprocal
//    and o and tanh(c) another (five exponentials and two reciprocals per element instead of five and five: the
//    special-function unit is what the cell update waits for).
//  * Exchange of h_t: a warp writes the planes of its 8 hidden units into its own CTA's double-buffered h planes (two units per
//    4-byte word, after one shuffle); from there bulk copies put the block into those of every other CTA of the cluster and count
//    their bytes on an mbarrier there, so a step costs one one-way transfer and no cluster-wide barrier.  (With the planes
//    gathered in a staging area in 2-byte stores and copied to the own buffer from there: 8.6 us more on 512 sequences x 121 chunks,
//    1.5 us on 256 x 56, 0.8 us on 8 x 28 at d_g = 128.)  A CTA can only be sent step t+1 data after it has itself sent step t data, i.e. after all its warps have finished
//    reading the buffer that is being overwritten.
//  * P_{t+1} is fetched a round ahead: the projection kernel stores the four pre-activations of a hidden unit side by side, so a
//    thread takes them with one 16-byte load.
//  * The score head is not part of the chain: a warp leaves its 8 units' share of w_s . h_t per sequence (d_g / 8 partial sums
//    per (s, t): an eighth of the bytes of h_t), and when the chain is through the cluster adds them up in a fixed order.
//  Measured, recurrence and score head: 512 sequences x 121 chunks 314 -> 276 us, 256 x 56 92.5 -> 79 us, 8 x 28 at
//  d_g = 128 51.6 -> 32 us (there a cluster of two CTAs halves the MMA chain: one CTA held all of W_hh).  Slower: waiting for the
//  CTA's own planes and the peers' apart, with the own units' MMAs in between (255 -> 261 us a step on 256 sequences), and
//  the score's shuffles between the MMAs (248 -> 255 us).
// Every mbarrier wait is bounded (one second); on give-up the status word gets KVE_ERR_TIMEOUT and
// the CTA stops sending, which lets its peers run into their own limits and leave as well.
#include "gate_rnn.cuh"

namespace kve {

// Optional cycle budget of one recurrence step (build with -DKVE_RNN_STAMPS, see rnn_stamps.py): warp 0 of CTA 0 adds
// up, over all steps and groups, the clock64 cycles between five points of a step - 0: waiting for the peers' h,
// 1: fragment loads + MMA chain, 2: prefetch of the next step's P, 3: cell update and plane split, 4: sending h,
// 6: from the end of one round to the start of the next (the loaded P moves into place, barrier bookkeeping) - and
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

template <int DG, int CL, int NG, int PL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(RNN_THREADS, 1) kve_gate_rnn_kernel(RnnArgs a) {
  constexpr int HU = DG / CL;            // hidden units owned by this CTA
  constexpr int KT = DG / 16;            // k tiles
  constexpr int NS = 8;                  // sequences per group: the n of the m16n8k16 MMA
  constexpr int KBLK = PL * NS * 8;                     // bf16 elements of one k-block (8 units): [plane][sequence][8]
  constexpr int HS_BUF = (DG / 8) * KBLK;               // bf16 elements per h buffer
  constexpr uint32_t H_BYTES = PL * NS * (DG - HU) * 2; // bytes of h planes a CTA receives from its peers per step and group
  constexpr int OFF_BARS = NG * 2 * HS_BUF * 2;
  constexpr int BULK_PENDING = 2 * NG - 1;              // a group's copies of two steps ago: all but the newest 2 NG - 1 commits
  static_assert(HU == 8 * RNN_WARPS && KT % 2 == 0, "one pair of m16 tiles (8 units x 4 gates) per warp");
  static_assert(OFF_BARS % 16 == 0, "16-byte pieces");

  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint16_t* hs = reinterpret_cast<uint16_t*>(smem_raw);                          // [NG][2][DG / 8][PL][NS][8]
  uint64_t* hbar = reinterpret_cast<uint64_t*>(smem_raw + OFF_BARS);             // [NG][2] h planes landed

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = tid >> 5;
  const int g = lane >> 2, tig = lane & 3;
  const uint32_t rank = cluster_rank();
  const int seq0 = (blockIdx.x / CL) * NS * NG;      // group gi owns sequences seq0 + 8 gi .. + 7
  const int ug = (int)rank * HU + warp * 8 + g;                // this thread's hidden unit

  KVE_RNN_ONCE(0);
  if (tid == 0) {
    for (int i = 0; i < 2 * NG; ++i) mbar_init(&hbar[i], RNN_WARPS + (CL > 1 ? 1 : 0));
    mbar_fence_init();
  }

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
  for (int kp = 0; kp < KT / 2; ++kp) load_pair(kp, A[kp]);
  const float w_score = __ldg(a.w_s + ug);

  KVE_RNN_ONCE(1);
  pdl_wait();      // W_hh is in place; the carried state and P come from earlier kernels
  // only now, when all earlier work is complete: a launch may run beside this kernel without waiting for anything (kvE_refresh)
  pdl_launch_dependents();
  KVE_RNN_ONCE(2);
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
  float c[NG][2], hlast[NG][2];
#pragma unroll
  for (int gi = 0; gi < NG; ++gi)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int s = seq0 + gi * NS + tig * 2 + e;
      const bool carried = !a.reset && s < a.S;
      c[gi][e] = carried ? a.lstm_c[(long long)s * DG + ug] : 0.f;
      hlast[gi][e] = carried ? a.lstm_h[(long long)s * DG + ug] : 0.f;
    }
  // the four pre-activations of a unit lie side by side in P: one 16-byte load
  const float4* p_unit = reinterpret_cast<const float4*>(a.P) + ug;
  auto load_p = [&](int gi, int step, float4 (&pv)[2]) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int s = seq0 + gi * NS + tig * 2 + e;
      const bool there = s < a.S && step < a.n_range;
      const float4* p = p_unit + (long long)(s * a.n_range + step) * DG;
      pv[e] = there ? __ldcs(p) : make_float4(0.f, 0.f, 0.f, 0.f);
      // the 8 lanes of a group cover one 128-byte line of the row after it: one of them asks L2 for it
      if (s < a.S && step + 1 < a.n_range && g == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + DG));
    }
  };
  float4 pin[2];
  load_p(0, 0, pin);
  float* part_out = a.H + rank * RNN_WARPS + warp;

  // lane r < CL feeds peer r: that CTA's h buffers and barriers, as addresses in the cluster window
  const uint32_t peer_hs = map_to_rank(smem_u32(hs), lane < CL ? lane : 0);
  const uint32_t peer_bar = map_to_rank(smem_u32(&hbar[0]), lane < CL ? lane : 0);

  // barriers initialised and buffer 0 filled in every CTA before anyone sends
  KVE_RNN_ONCE(3);
  cluster_sync_all();
  KVE_RNN_ONCE(4);

  bool alive = true;
  KVE_RNN_MARK_BEGIN();
  for (int step = 0; step < a.n_range && alive; ++step) {
    const int buf = step & 1;
    const bool send_h = step + 1 < a.n_range;
    // this step's sends of the cluster land in buffer buf^1 of each group: announce the bytes
    if (CL > 1 && send_h && tid == 0) {
#pragma unroll
      for (int gi = 0; gi < NG; ++gi) mbar_arrive_expect_tx(&hbar[2 * gi + (buf ^ 1)], H_BYTES);
    }
#pragma unroll
    for (int gi = 0; gi < NG; ++gi) {
      uint16_t* hs_g = hs + gi * 2 * HS_BUF;
      uint64_t* hbar_g = hbar + 2 * gi;
      // P of the next round, used there: requested before the wait (one group), while the MMAs drain (two, where nothing waits)
      float4 pv[2];
      if (NG == 1) load_p(0, step + 1, pv);
      KVE_RNN_MARK(2);
      // ---- h_{t-1} from every CTA of the cluster (each buffer completes once per two steps) -----------------------------
      if (step > 0) {
        if (!mbar_wait_cluster_bounded(&hbar_g[buf], ((step - 1) >> 1) & 1)) {
          if (lane == 0) set_status(a.status, ERR_TIMEOUT);
          alive = false;
        }
        alive = __all_sync(0xffffffffu, alive);
        if (!alive) break;
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
      KVE_RNN_MARK(1);

      if (NG > 1) {
        // (the vote is a scheduling fence: without it the compiler spreads the loads' address arithmetic over the MMA chain)
        if (!__all_sync(0xffffffffu, alive)) break;
        load_p((gi + 1) % NG, step + (gi + 1) / NG, pv);
      }
      // ---- cell update (thread-local), planes of h_t into this CTA's buffer ---------------------
      // the copies from there two steps ago have been read: those of the group's last step may still be under way
      if (CL > 1) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(BULK_PENDING) : "memory");
      __syncwarp();
      uint32_t split[2][3];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float pre[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {   // q: 0 = i, 1 = f (tile 0, rows g / g+8), 2 = g, 3 = o (tile 1)
          const int mt = q >> 1, ai = (q & 1) * 2 + e;
          float sum = acc[PL - 1][mt][ai];      // smallest plane first
#pragma unroll
          for (int pl = PL - 2; pl >= 0; --pl) sum += acc[pl][mt][ai];
          pre[q] = sum + (q == 0 ? pin[e].x : (q == 1 ? pin[e].y : (q == 2 ? pin[e].z : pin[e].w)));
        }
        const float hv = lstm_cell(pre, c[gi][e]);
        hlast[gi][e] = hv;
        split3(hv, split[e]);
      }
      KVE_RNN_MARK(3);
      // ---- the warp's k-block (8 units: [plane][sequence][8], contiguous) to every CTA of the cluster ----
      if (send_h) {
        const uint32_t off = (uint32_t)(((gi * 2 + (buf ^ 1)) * HS_BUF + ((int)rank * RNN_WARPS + warp) * KBLK) * 2);
        // lanes g and g ^ 1 hold neighbouring units: an even g takes both units of sequence 2 tig, an odd one those of 2 tig + 1, and
        // a warp's store instruction is a whole plane of the block: 128 bytes in a row
        const bool odd = (g & 1) != 0;
        unsigned char* mine = reinterpret_cast<unsigned char*>(hs) + off + (tig * 2 + (g & 1)) * 16 + (g >> 1) * 4;
        const uint32_t keep = odd ? split[1][0] | split[1][1] << 16 : split[0][0] | split[0][1] << 16;
        const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? split[0][0] | split[0][1] << 16 : split[1][0] | split[1][1] << 16, 4);
        *reinterpret_cast<uint32_t*>(mine) = __byte_perm(odd ? got : keep, odd ? keep : got, 0x5410);
        *reinterpret_cast<uint32_t*>(mine + NS * 16) = __byte_perm(odd ? got : keep, odd ? keep : got, 0x7632);
        if constexpr (PL == 3) {
          const uint32_t keep2 = odd ? split[1][2] : split[0][2], got2 = __shfl_xor_sync(0xffffffffu, odd ? split[0][2] : split[1][2], 4);
          *reinterpret_cast<uint32_t*>(mine + 2 * NS * 16) = (odd ? got2 : keep2) | (odd ? keep2 : got2) << 16;
        }
        if (CL > 1) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // visible to the bulk copies
        __syncwarp();
        if (CL > 1) {
          // peers: one bulk copy each out of the own buffer, its bytes counted on the receiver's barrier
          if (lane < CL && lane != (int)rank)
            bulk_s2cluster(peer_hs + off, smem_u32(hs) + off, KBLK * 2, peer_bar + (2 * gi + (buf ^ 1)) * 8);
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        if (lane == 0) mbar_arrive(&hbar_g[buf ^ 1]);     // release: this warp's own pieces are in place
      }
      KVE_RNN_MARK(4);
      // ---- this warp's share of the score, behind the sends: lane group g = 0 ends up with sequence 2 tig, g = 1 with 2 tig + 1 ----
      {
        const bool odd = (g & 1) != 0;
        const float d0 = w_score * hlast[gi][0], d1 = w_score * hlast[gi][1];
        float d = (odd ? d1 : d0) + __shfl_xor_sync(0xffffffffu, odd ? d0 : d1, 4);
        d += __shfl_xor_sync(0xffffffffu, d, 8);
        d += __shfl_xor_sync(0xffffffffu, d, 16);
        const int s = seq0 + gi * NS + tig * 2 + (g & 1);
        if (g < 2 && s < a.S) part_out[(long long)(s * a.n_range + step) * (DG / 8)] = d;
      }
#ifdef KVE_RNN_STAMPS
      if (blockIdx.x == 0 && tid == 0) atomicAdd(&g_rnn_cycles[5], 1ull);
#endif
      pin[0] = pv[0];
      pin[1] = pv[1];
      KVE_RNN_MARK(6);
    }
  }

  KVE_RNN_ONCE(5);
  // ---- carried state out ---------------------------------------------------------------------------
#pragma unroll
  for (int gi = 0; gi < NG; ++gi)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int s = seq0 + gi * NS + tig * 2 + e;
      if (s < a.S && alive) {
        a.lstm_c[(long long)s * DG + ug] = c[gi][e];
        a.lstm_h[(long long)s * DG + ug] = hlast[gi][e];
      }
    }
  // nobody leaves while a peer may still be sending into its shared memory; the partial sums of all CTAs are in place behind it
  cluster_sync_all();
  KVE_RNN_ONCE(6);
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
}

template <int DG, int CL, int NG, int PL>
static cudaError_t launch_rnn_t(const RnnArgs& a, cudaStream_t st) {
  constexpr int KBLK_BYTES = PL * 8 * 8 * 2;
  constexpr int smem = NG * 2 * (DG / 8) * KBLK_BYTES + NG * 2 * 8;
  static DeviceFlags opted;
  {
    cudaError_t e = smem_opt_in(opted, kve_gate_rnn_kernel<DG, CL, NG, PL>, smem);
    if (e != cudaSuccess) return e;
  }
  const int clusters = (a.S + 8 * NG - 1) / (8 * NG);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  // an SM keeps its division of shared memory and L1 as long as a CTA is there: all of it shared, for what may run beside this kernel
  attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  attr[1].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * CL);
  cfg.blockDim = dim3(RNN_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kve_gate_rnn_kernel<DG, CL, NG, PL>, a);
}

// CTAs of a cluster; two groups of 8 sequences per cluster once one group per cluster would need more than one wave of clusters
static int cluster_ctas(int d_g) { return d_g / 64; }
static bool two_groups(int S, int d_g) { return (S + 7) / 8 > sm_count() / cluster_ctas(d_g); }

// Microseconds per chunk as measured (two planes of h, d_g = 256): 1.22 with one group of sequences per cluster, 2.28 with two
double gate_rnn_us_per_chunk(int S, int d_g, int planes) {
  const bool two = two_groups(S, d_g);
  const int clusters = (S + (two ? 15 : 7)) / (two ? 16 : 8), wave = sm_count() / cluster_ctas(d_g);
  return (two ? 2.28 : 1.22) * (planes == 3 ? 1.25 : 1.0) * ((clusters + wave - 1) / wave);
}

template <int PL>
static cudaError_t launch_rnn_planes(const RnnArgs& a, int d_g, cudaStream_t st) {
  const bool two = two_groups(a.S, d_g);
  switch (d_g) {
    case 256: return two ? launch_rnn_t<256, 4, 2, PL>(a, st) : launch_rnn_t<256, 4, 1, PL>(a, st);
    case 128: return two ? launch_rnn_t<128, 2, 2, PL>(a, st) : launch_rnn_t<128, 2, 1, PL>(a, st);
    case 64:  return two ? launch_rnn_t<64, 1, 2, PL>(a, st) : launch_rnn_t<64, 1, 1, PL>(a, st);
    default:  return cudaErrorInvalidValue;
  }
}

cudaError_t launch_gate_rnn(const LayerView& v, int t0, int t1, const uint16_t* W_hh, const float* w_s, float b_s,
                            int d_g, const float* P, float* H, bool reset_state, int planes, cudaStream_t st) {
  if (t1 <= t0 || v.S <= 0) return cudaSuccess;
  RnnArgs a;
  a.P = P; a.H = H; a.W_hh = W_hh; a.w_s = w_s; a.b_s = b_s;
  a.scores = v.scores; a.lstm_h = v.lstm_h; a.lstm_c = v.lstm_c; a.status = v.status;
  a.S = v.S; a.max_chunks = v.max_chunks; a.t0 = t0; a.n_range = t1 - t0; a.reset = reset_state ? 1 : 0;
  return planes == 3 ? launch_rnn_planes<3>(a, d_g, st) : launch_rnn_planes<2>(a, d_g, st);
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
