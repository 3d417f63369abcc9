// sfm_move.cuh -- the per-pedestrian stages (S3 decide, S4 vote, S5 commit)
// bin by bin, for crowds: one block takes a bin's records and what its su and
// their neighbours hold in shared memory.  Same decisions, elections and moves
// as decide_one, vote_one and commit_one (sfm_device.cuh), which take a
// pedestrian at a time.  Shared by the single lattice (sfm_move.cu) and the
// batch (sfm_batch.cu).
//
// The stages are bound by requests to memory, not by bytes: a pedestrian's own
// arrays are read in bin order, a 32-byte sector for each value, and decide_one
// reads 27 neighbours, vote_one 8 and then each occupied one's choice.  Here a
// record carries the position and heading from the binning on, the choice from
// the decision on and the win from the vote on, and a neighbour is read once
// for its whole bin. 
// Decide, vote and commit of 500 000 pedestrians on 1000 x 1000 (one-pass
// ncu, caches flushed): 19, 23 and 16 us against 22, 33 and 21 (256 threads a
// block); a whole tick at r = 3 99.5 -> 72.6 us, at a density of 0.8 124.8 ->
// 85.0.
#pragma once
#include "sfm_device.cuh"

namespace sfm {

// Threads of a block, T: 128, or 512 for a lattice with few bins.  A tick of
// 1000 x 1000 half full at r = 3 takes 72.6 us with 128, 77.9 with 256 and 87.7
// with 512; of 300 x 300 (100 bins) 55.5, 48.2 and 45.9.
constexpr int kMoveThreads = 128, kMoveThreadsFew = 512;
// a record's bits: column | row << 8 | heading class << 16, and
constexpr int kRecChoice = 20, kRecWon = 24;

// su (x0 + i % SIDE, y0 + i / SIDE) of a square of SIDE su, wrapped; false
// outside the lattice (or the square)
template <int SIDE>
__device__ __forceinline__ bool square_su(const Geo& g, int x0, int y0, bool inside, int i, int& x,
                                          int& y) {
  x = x0 + i % SIDE;
  y = y0 + i / SIDE;
  return i < SIDE * SIDE && (inside || (wrap_coord(x, g.W, g.px, x) & wrap_coord(y, g.H, g.py, y)));
}
// the whole square lies in the lattice (the same for the block: no wrapping)
template <int SIDE>
__device__ __forceinline__ bool square_inside(const Geo& g, int x0, int y0) {
  return x0 >= 0 && y0 >= 0 && x0 + SIDE <= g.W && y0 + SIDE <= g.H;
}

constexpr int kDecideSide = kBin + 2, kVoteSide = kBin + 4;

struct DecideTile {
  float f[kDecideSide * kDecideSide];
  int32_t d[kDecideSide * kDecideSide];
  float own[81], dirdot[81];
  uint8_t o[kDecideSide * kDecideSide];
};

// Decisions of the records [first, end) of bin (bx, by); all threads of the
// block call it, first < end.
template <int T, bool TIE>
__device__ __forceinline__ void decide_bin(DecideTile& t, const Geo& g, int bx, int by, int first,
                                           int end, uint32_t* rec, const int32_t* rec_id,
                                           const uint8_t* goal, const uint8_t* ocls,
                                           const int32_t* D, const float* F, float beta,
                                           const float* own, const float* dirdot, uint8_t* choice,
                                           const WalkPeriods& wp, long long tick,
                                           unsigned& decided, unsigned& ties) {
  constexpr int S = kDecideSide, K = (S * S + T - 1) / T;
  const int tid = threadIdx.x, x0 = bx * kBin - 1, y0 = by * kBin - 1;
  const bool inside = square_inside<S>(g, x0, y0);
  int i = first + tid, p = 0, gl = 0;
  uint32_t rc = 0;
  if (i < end) {
    rc = rec[i];
    p = rec_id[i];
  }
  float f[K];
  int32_t d[K];
  uint8_t o[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    int x, y;
    f[k] = 0.f;
    d[k] = 0;
    o[k] = 1;  // outside the lattice: not admissible
    if (square_su<S>(g, x0, y0, inside, tid + k * T, x, y)) {
      f[k] = F[(size_t)y * g.W + x];
      d[k] = D[(size_t)y * g.W + x];
      o[k] = ocls[(size_t)y * g.opitch + x];
    }
  }
  if (i < end) gl = goal[p];
  if (tid < 81) {
    t.own[tid] = own[tid];
    t.dirdot[tid] = dirdot[tid];
  }
  static_assert(T >= 81, "a thread each for the 81 entries");
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (tid + k * T < S * S) {
      t.f[tid + k * T] = f[k];
      t.d[tid + k * T] = d[k];
      t.o[tid + k * T] = o[k];
    }
  __syncthreads();
  const bool in[3] = {true, true, true};
  while (i < end) {
    int k = 0;
    if (!(wp.period && tick % wp.period[p] != wp.phase[p])) {
      const int c = ((int)((rc >> 8) & 0xffu) + 1) * S + (int)(rc & 0xffu) + 1;
      float nf[9];
      int32_t nd[9];
      uint8_t no[9];
#pragma unroll
      for (int m = 0; m < 9; ++m) {
        const int n = c + move_dy(m) * S + move_dx(m);
        nf[m] = t.f[n];
        nd[m] = t.d[n];
        no[m] = t.o[n];
      }
      bool tie = false;
      k = pick_move<false, TIE>(nf, nd, no, in, in, (int)((rc >> 16) & 0xfu), gl, beta, t.own, t.dirdot,
                                nullptr, nullptr, &tie);
      ++decided;
      ties += tie ? 1u : 0u;
    }
    choice[p] = (uint8_t)k;
    rec[i] = rc | (uint32_t)k << kRecChoice;
    i += T;
    if (i < end) {
      rc = rec[i];
      p = rec_id[i];
      gl = goal[p];
    }
  }
}

struct VoteTile {
  int32_t occ[kVoteSide * kVoteSide];
  uint8_t ch[kVoteSide * kVoteSide];
};

// Elections of the movers among the records [first, end) of bin (bx, by) (all
// threads of the block; first < end).  Returns the thread's largest registrant
// count of a target.
template <int T>
__device__ __forceinline__ int vote_bin(VoteTile& t, const Geo& g, int bx, int by, int first, int end,
                                        uint32_t* rec, const int32_t* rec_id, const uint8_t* choice,
                                        const int32_t* occ, uint64_t seed, long long tick, int ped_off,
                                        const int32_t* gid, uint8_t* won) {
  constexpr int S = kVoteSide, K = (S * S + T - 1) / T;
  const int tid = threadIdx.x, x0 = bx * kBin - 2, y0 = by * kBin - 2;
  const bool inside = square_inside<S>(g, x0, y0);
  int o[K];
  uint8_t ch[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    int x, y;
    o[k] = square_su<S>(g, x0, y0, inside, tid + k * T, x, y) ? occ[(size_t)y * g.W + x] : -1;
  }
#pragma unroll
  for (int k = 0; k < K; ++k) ch[k] = o[k] >= 0 ? choice[o[k]] : (uint8_t)0;
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (tid + k * T < S * S) {
      t.occ[tid + k * T] = o[k];
      t.ch[tid + k * T] = ch[k];
    }
  __syncthreads();
  const uint64_t st = splitmix_nth(seed, (uint64_t)tick + 1);
  int most = 0;
  for (int i = first + tid; i < end; i += T) {
    const uint32_t rc = rec[i];
    const int p = rec_id[i], k = (int)(rc >> kRecChoice) & 0xf;
    bool win = false;
    if (k) {
      const int target = ((int)((rc >> 8) & 0xffu) + 2 + c_dy[k]) * S + (int)(rc & 0xffu) + 2 + c_dx[k];
      const long long idp = gid ? (long long)gid[p] : (long long)(p - ped_off);
      const uint64_t mine = splitmix_nth(st, (uint64_t)idp + 1);
      int regs = 1;
      win = true;
#pragma unroll
      for (int j = 1; j <= 8; ++j) {
        constexpr int opp[9] = {0, 5, 6, 7, 8, 1, 2, 3, 4};
        const int n = target + move_dy(j) * S + move_dx(j);
        if (t.ch[n] != opp[j] || k == opp[j]) continue;  // no move to the target, or p's own
        ++regs;
        const int r = t.occ[n];
        const long long ido = gid ? (long long)gid[r] : (long long)(r - ped_off);
        const uint64_t po = splitmix_nth(st, (uint64_t)ido + 1);
        if (po < mine || (po == mine && ido < idp)) win = false;
      }
      most = max(most, regs);
    }
    won[p] = win ? 1 : 0;
    if (win) rec[i] = rc | 1u << kRecWon;
  }
  return most;
}

// Move of record rc (pedestrian p) of bin (bx, by), which won its target.
__device__ __forceinline__ void commit_record(uint32_t rc, int p, const Geo& g, int bx, int by,
                                              int2* xy, uint8_t* alive, uint8_t* heading,
                                              const uint8_t* cell, int32_t* occ, uint8_t* ocls,
                                              bool& left) {
  const int k = (int)(rc >> kRecChoice) & 0xf;
  const int x = bx * kBin + (int)(rc & 0xffu), y = by * kBin + (int)((rc >> 8) & 0xffu);
  int tx, ty;
  wrap_coord(x + c_dx[k], g.W, g.px, tx);
  wrap_coord(y + c_dy[k], g.H, g.py, ty);
  const size_t c1 = (size_t)ty * g.W + tx;
  left = cell[c1] == kExit;
  occ[(size_t)y * g.W + x] = -1;
  ocls[(size_t)y * g.opitch + x] = 0;
  if (left) {
    alive[p] = 0;
  } else {
    occ[c1] = p;
    ocls[(size_t)ty * g.opitch + tx] = (uint8_t)(1 + k);
  }
  xy[p] = make_int2(tx, ty);
  heading[p] = (uint8_t)k;
}

// the counters of a block's votes and moves, one atomic a warp (all threads)
__device__ __forceinline__ void count_votes(Counters* ctr, int most) {
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) == 0) {
    if (most > 2) atomicMax(&ctr->max_registrants, most);
    if (most > 8) atomicOr(&ctr->err, kErrEnroll);
  }
}
__device__ __forceinline__ void count_moves(Counters* ctr, unsigned moved, unsigned left) {
  moved = __reduce_add_sync(0xffffffffu, moved);
  left = __reduce_add_sync(0xffffffffu, left);
  if ((threadIdx.x & 31) == 0) {
    if (moved) atomicAdd(&ctr->moved, (unsigned long long)moved);
    if (left) atomicAdd(&ctr->exited, (unsigned long long)left);
  }
}

}  // namespace sfm
