// kvE_selftest_timeout: makes the bounded-wait helpers of the library run out on purpose, safely.
// Every kernel of the library waits on mbarriers (copies landing, tensor-core commits, peers of a cluster) through
// mbar_wait_bounded / mbar_wait_cluster_bounded; when such a wait gives up, the kernel records KVE_ERR_TIMEOUT in the
// status word and leaves in order.  Here a barrier is armed with bytes (or an arrival) that nothing ever delivers and
// the wait limit is a few thousand polls / two milliseconds: the kernel must return, the status word must read
// KVE_ERR_TIMEOUT, and the context must stay usable.  Nothing faults, traps or spins without a bound.
#include "gate_rnn.cuh"

namespace kve {

// which 0: a CTA waits for 16 bytes of a bulk copy that is never issued (the wait of the copy pipelines)
__global__ void __launch_bounds__(32) kve_selftest_cta_wait_kernel(int32_t* status) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
    mbar_arrive_expect_tx(&bar, 16);      // the arrival is there, the bytes never come: the phase cannot complete
  }
  __syncwarp();
  const bool ok = mbar_wait_bounded(&bar, 0, 4096);
  if (!ok && threadIdx.x == 0) set_status(status, ERR_TIMEOUT);
}

// which 1: the two CTAs of a cluster each wait for an arrival from the peer that the peer never sends (the wait of the
// recurrence kernel); both give up after two milliseconds, then leave together like that kernel does
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(32) kve_selftest_cluster_wait_kernel(int32_t* status) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
  }
  cluster_sync_all();
  const bool ok = mbar_wait_cluster_bounded(&bar, 0, 2000000ull);
  if (!ok && threadIdx.x == 0) set_status(status, ERR_TIMEOUT);
  cluster_sync_all();      // nobody leaves while a peer could still address its shared memory
}

// which 2: a ring of copies whose reader gives up.  Four stages are armed, three of them get their copies; the wait for the first, whose copy
// is never issued, runs out, and the ring is drained as the copy pipelines do it.  The other copies must have landed by then: the
// status word reads KVE_ERR_CAPACITY instead of KVE_ERR_TIMEOUT if a byte of them is missing.
__global__ void __launch_bounds__(32) kve_selftest_ring_kernel(const uint4* src, int32_t* status) {
  constexpr int STAGES = 4, PIECES = SELFTEST_RING_BYTES / STAGES / 16;
  __shared__ __align__(128) uint4 ring[STAGES][PIECES];
  __shared__ __align__(8) uint64_t full[STAGES];
  for (int i = threadIdx.x; i < STAGES * PIECES; i += 32) (&ring[0][0])[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) mbar_init(&full[i], 1);
    mbar_fence_init();
    for (int i = 0; i < STAGES; ++i) {
      mbar_arrive_expect_tx(&full[i], PIECES * 16);
      if (i > 0) bulk_g2s(ring[i], src + i * PIECES, PIECES * 16, &full[i]);
    }
  }
  __syncwarp();
  const bool ok = mbar_wait_bounded(&full[0], 0, 4096);
  ring_drain<STAGES>(full, STAGES);
  bool landed = true;
  for (int i = PIECES + threadIdx.x; i < STAGES * PIECES; i += 32) {
    const uint4 x = (&ring[0][0])[i], y = src[i];
    landed = landed && x.x == y.x && x.y == y.y && x.z == y.z && x.w == y.w;
  }
  if (!__all_sync(0xffffffffu, landed)) {
    if (threadIdx.x == 0) set_status(status, ERR_CAPACITY);
  } else if (!ok && threadIdx.x == 0) {
    set_status(status, ERR_TIMEOUT);
  }
}

cudaError_t launch_selftest_timeout(int which, const void* src, int32_t* status, cudaStream_t st) {
  if (which == 0) kve_selftest_cta_wait_kernel<<<1, 32, 0, st>>>(status);
  else if (which == 2) kve_selftest_ring_kernel<<<1, 32, 0, st>>>(static_cast<const uint4*>(src), status);
  else kve_selftest_cluster_wait_kernel<<<2, 32, 0, st>>>(status);
  return cudaGetLastError();
}

}  // namespace kve
