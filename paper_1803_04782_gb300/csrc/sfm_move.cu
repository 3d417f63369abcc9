// sfm_move.cu -- decide, vote and commit of a crowded single lattice, a block
// a bin (sfm_move.cuh).
#include <cuda_runtime.h>
#include <stdint.h>

#include "sfm_internal.h"
#include "sfm_move.cuh"

namespace sfm {

namespace {

template <int T>
__global__ void __launch_bounds__(T, 1024 / T)
    k_decide_bins(Geo g, const int32_t* bin_start, uint32_t* rec, const int32_t* rec_id,
                  const uint8_t* goal, const uint8_t* ocls, const int32_t* D, const float* F, float beta,
                  const float* own, const float* dirdot, uint8_t* choice, WalkPeriods wp,
                  Counters* ctr) {
  __shared__ DecideTile t;
  const int b = blockIdx.x, first = bin_start[b], end = bin_start[b + 1];
  if (first >= end) return;
  unsigned decided = 0, ties = 0;
  decide_bin<T, true>(t, g, b % g.nbx, b / g.nbx, first, end, rec, rec_id, goal, ocls, D, F, beta, own,
                   dirdot, choice, wp, wp.period ? ctr->t : 0, decided, ties);
  decided = __reduce_add_sync(0xffffffffu, decided);
  ties = __reduce_add_sync(0xffffffffu, ties);
  if ((threadIdx.x & 31) == 0 && decided) {
    atomicAdd(&ctr->decided, (unsigned long long)decided);
    if (ties) atomicAdd(&ctr->near_ties, (unsigned long long)ties);
  }
}

// ... and choice = won = 0 for the pedestrians that are not alive, as in k_vote
template <int T>
__global__ void __launch_bounds__(T, 1024 / T)
    k_vote_bins(int n, Geo g, const int32_t* bin_start, uint32_t* rec, const int32_t* rec_id,
                const uint8_t* alive, uint8_t* choice, const int32_t* occ, uint64_t seed, Counters* ctr,
                uint8_t* won, const int32_t* gid) {
  __shared__ VoteTile t;
  const int b = blockIdx.x, first = bin_start[b], end = bin_start[b + 1];
  for (int i = b * T + threadIdx.x; i < n; i += gridDim.x * T)
    if (!alive[i]) {
      choice[i] = 0;
      won[i] = 0;
    }
  if (first >= end) return;
  count_votes(ctr, vote_bin<T>(t, g, b % g.nbx, b / g.nbx, first, end, rec, rec_id, choice, occ, seed,
                            ctr->t, 0, gid, won));
}

template <int T>
__global__ void __launch_bounds__(T)
    k_commit_bins(Geo g, const int32_t* bin_start, const uint32_t* rec, const int32_t* rec_id, int2* xy,
                  uint8_t* alive, uint8_t* heading, const uint8_t* cell, int32_t* occ, uint8_t* ocls,
                  Counters* ctr) {
  const int b = blockIdx.x, first = bin_start[b], last = bin_start[b + 1];
  const bool whole = !(ctr->err & kErrTimeout);  // as in k_commit
  const int end = whole ? last : first;
  unsigned nm = 0, nl = 0;
  for (int i = first + threadIdx.x; i < end; i += T) {
    const uint32_t rc = rec[i];
    if (!(rc >> kRecWon & 1u)) continue;
    bool left;
    commit_record(rc, rec_id[i], g, b % g.nbx, b / g.nbx, xy, alive, heading, cell, occ, ocls, left);
    ++nm;
    nl += left;
  }
  __syncwarp();
  count_moves(ctr, nm, nl);
  if (b == 0 && threadIdx.x == 0 && whole) ctr->t += 1;
}

// few bins: at most two for each SM
bool few_bins(const Geo& g) { return g.nbx * g.nby <= 2 * device_sm_count(); }

}  // namespace

// k<T><<<a block a bin, T threads>>>(args...)
#define SFM_BINS(k, ...)                                                                  \
  do {                                                                                    \
    if (few_bins(g))                                                                      \
      k<kMoveThreadsFew><<<g.nbx * g.nby, kMoveThreadsFew, 0, s>>>(__VA_ARGS__);          \
    else                                                                                  \
      k<kMoveThreads><<<g.nbx * g.nby, kMoveThreads, 0, s>>>(__VA_ARGS__);                \
  } while (0)

void launch_decide_bins(const Geo& g, const int32_t* bin_start, uint32_t* rec, const int32_t* rec_id,
                        const uint8_t* goal, const uint8_t* ocls, const int32_t* D, const float* F,
                        float beta, const Tables& tb, uint8_t* choice, cudaStream_t s,
                        const WalkPeriods& wp, Counters* ctr) {
  SFM_BINS(k_decide_bins, g, bin_start, rec, rec_id, goal, ocls, D, F, beta, tb.own, tb.dirdot, choice,
           wp, ctr);
}

void launch_vote_bins(int n, const Geo& g, const int32_t* bin_start, uint32_t* rec,
                      const int32_t* rec_id, const uint8_t* alive, uint8_t* choice, const int32_t* occ,
                      uint64_t seed, Counters* ctr, uint8_t* won, cudaStream_t s, const int32_t* gid) {
  SFM_BINS(k_vote_bins, n, g, bin_start, rec, rec_id, alive, choice, occ, seed, ctr, won, gid);
}

void launch_commit_bins(const Geo& g, const int32_t* bin_start, const uint32_t* rec,
                        const int32_t* rec_id, int2* xy, uint8_t* alive, uint8_t* heading,
                        const uint8_t* cell, int32_t* occ, uint8_t* ocls, Counters* ctr,
                        cudaStream_t s) {
  SFM_BINS(k_commit_bins, g, bin_start, rec, rec_id, xy, alive, heading, cell, occ, ocls, ctr);
}
#undef SFM_BINS

}  // namespace sfm
