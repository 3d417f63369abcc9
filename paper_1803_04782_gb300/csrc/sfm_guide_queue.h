// sfm_guide_queue.h -- the queue of tiles from which the CTAs of k_guidance
// (sfm_kernels.cu) take their work.  Plain functions on shared words, one
// atomic each, compiled for the device and for the host, so that their
// interleavings can be run through on a CPU as well.
//
// Entry `pos` of the run (0, 1, ...) sits in ring[pos mod ntiles].  A tile is in
// the queue at most once (`queued`), so at most ntiles entries are untaken; but
// they need not be the ntiles youngest: a CTA that has claimed a position and not
// yet looked at the slot is passed by others, whose tiles are queued again.  So
// a slot is handed over explicitly: its word says whose turn it is, an entry is
// put in only once the slot's last one has been taken, and is taken by position.
//
// No wait here can be circular: an entry waits for the taker of the one ntiles
// positions before it, which has been claimed (else more than ntiles tiles would
// be untaken) by a CTA that waits for that entry alone, and so on down to the
// first ntiles, which wait for nothing.
#pragma once

#ifdef __CUDACC__
#define SFM_HD __host__ __device__ __forceinline__
#else
#define SFM_HD inline
#endif

namespace sfm {

typedef unsigned long long guide_word;

struct GuideQueue {
  // entries made so far (low half), and tiles queued or being relaxed (high
  // half), so that one atomic makes an entry's place and keeps the run alive
  guide_word work;
  unsigned head, pad;  // positions claimed
};
// zero at first
struct GuideTiles {
  GuideQueue* q;
  // state << 32 | tile; state 2 L: free for the slot's use L = pos / ntiles,
  // 2 L + 1: holds that use's tile
  guide_word* ring;
  int* queued;
  int ntiles;
};
constexpr int kGuideQueueInts = (int)(sizeof(GuideQueue) / sizeof(int));
constexpr int kGuideTileInts = 3;  // ints a tile

SFM_HD GuideTiles guide_tiles(int* scratch, int ntiles) {
  GuideTiles t;
  t.q = reinterpret_cast<GuideQueue*>(scratch);
  t.ring = reinterpret_cast<guide_word*>(t.q + 1);
  t.queued = reinterpret_cast<int*>(t.ring + ntiles);
  t.ntiles = ntiles;
  return t;
}

// false: the tile is in the queue already (and its taker will see what the
// caller has written before)
SFM_HD bool guide_mark(const GuideTiles& gt, int t) {
#ifdef __CUDA_ARCH__
  return atomicExch(&gt.queued[t], 1) == 0;
#else
  return __atomic_exchange_n(&gt.queued[t], 1, __ATOMIC_SEQ_CST) == 0;
#endif
}
// the position of a marked tile's entry
SFM_HD unsigned guide_position(const GuideTiles& gt) {
  const guide_word one = (1ull << 32) + 1ull;
#ifdef __CUDA_ARCH__
  return (unsigned)atomicAdd(&gt.q->work, one);
#else
  return (unsigned)__atomic_fetch_add(&gt.q->work, one, __ATOMIC_SEQ_CST);
#endif
}
// false: the slot's last entry has not been taken yet
SFM_HD bool guide_publish(const GuideTiles& gt, unsigned pos, int t) {
  const unsigned n = (unsigned)gt.ntiles;
  const guide_word free = (guide_word)(pos / n * 2u) << 32, full = (free + (1ull << 32)) | (unsigned)t;
#ifdef __CUDA_ARCH__
  return atomicCAS(&gt.ring[pos % n], free, full) == free;
#else
  guide_word was = free;
  return __atomic_compare_exchange_n(&gt.ring[pos % n], &was, full, false, __ATOMIC_SEQ_CST, __ATOMIC_SEQ_CST);
#endif
}
SFM_HD unsigned guide_claim(const GuideTiles& gt) {
#ifdef __CUDA_ARCH__
  return atomicAdd(&gt.q->head, 1u);
#else
  return __atomic_fetch_add(&gt.q->head, 1u, __ATOMIC_SEQ_CST);
#endif
}
// the tile of a claimed position, -1 while its entry is not there
SFM_HD int guide_take(const GuideTiles& gt, unsigned pos) {
  const unsigned n = (unsigned)gt.ntiles, full = pos / n * 2u + 1u;
  volatile guide_word* slot = &gt.ring[pos % n];
  const guide_word v = *slot;
  if ((unsigned)(v >> 32) != full) return -1;
  *slot = (guide_word)(full + 1u) << 32;
  return (int)(unsigned)v;
}
// from here on the tile may be queued again
SFM_HD void guide_unmark(const GuideTiles& gt, int t) {
#ifdef __CUDA_ARCH__
  atomicExch(&gt.queued[t], 0);
#else
  __atomic_exchange_n(&gt.queued[t], 0, __ATOMIC_SEQ_CST);
#endif
}
SFM_HD guide_word guide_work(const GuideTiles& gt) {
  return *reinterpret_cast<volatile guide_word*>(&gt.q->work);
}
SFM_HD bool guide_over(guide_word work) { return (work >> 32) == 0; }
// a tile that was taken is relaxed, and what it changed is queued
SFM_HD void guide_done(const GuideTiles& gt) {
#ifdef __CUDA_ARCH__
  atomicAdd(&gt.q->work, ~0ull << 32);
#else
  __atomic_fetch_add(&gt.q->work, ~0ull << 32, __ATOMIC_SEQ_CST);
#endif
}

}  // namespace sfm
