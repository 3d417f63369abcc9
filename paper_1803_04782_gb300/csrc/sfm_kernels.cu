// sfm_kernels.cu -- sm_103a kernels of one tick of the discrete social-field
// pedestrian model (Alg. 1 of the paper: k-5 field superposition, k-2 decision,
// k-3 vote, k-4 commit), re-designed as gathers so that no step needs atomics
// on the field (Sec. 3.1 s-1 avoids them with fan-out caches instead).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "sfm_gather.cuh"
#include "sfm_guide_queue.h"
#include "sfm_internal.h"

namespace sfm {

static inline int cdiv(int a, int b) { return (a + b - 1) / b; }

// ------------------------------------------------------------------ tables
// Kernel values are evaluated once per scene in FP64 and rounded to FP32.
// Latency of the FP64 powers bounds it, so a thread takes one, in small blocks
// (blockIdx.y: the crowd's law, WALL's, EXIT's): 31 -> 16 us at r = 40.
constexpr int kTabThreads = 64;
__global__ void __launch_bounds__(kTabThreads)
    k_tables(int r, double kP, double aP, double gamma, double kO, double aO, double kE, double aE,
             float* T0, float* TX, float* TY, float* KO, float* KE, float* own, float* dirdot,
             float2* hvec) {
  const int S = 2 * r + 1, n = S * S;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, law = blockIdx.y;
  if (i < n) {
    const int dx = i % S - r, dy = i / S - r;
    const bool centre = dx == 0 && dy == 0;
    const double d = centre ? 1.0 : sqrt((double)(dx * dx + dy * dy));
    const double base = (law == 0 ? kP : law == 1 ? kO : kE) * pow(d, law == 0 ? aP : law == 1 ? aO : aE);
    if (law == 0) {
      T0[i] = centre ? 0.f : (float)base;
      TX[i] = centre ? 0.f : (float)(base * gamma * dx / d);
      TY[i] = centre ? 0.f : (float)(base * gamma * dy / d);
    } else {
      (law == 1 ? KO : KE)[i] = centre ? 0.f : (float)base;
    }
  }
  if (law) return;
  if (i < 81) {
    const int h = i / 9, k = i % 9;
    double hx = 0.0, hy = 0.0;
    if (h > 0) {
      const double nh = sqrt((double)(c_dx[h] * c_dx[h] + c_dy[h] * c_dy[h]));
      hx = c_dx[h] / nh;
      hy = c_dy[h] / nh;
    }
    double o = 0.0;
    if (k > 0 && r >= 1) {
      const double d = sqrt((double)(c_dx[k] * c_dx[k] + c_dy[k] * c_dy[k]));
      o = kP * pow(d, aP) * (1.0 + gamma * (hx * c_dx[k] + hy * c_dy[k]) / d);
    }
    own[i] = (float)o;
    dirdot[i] = (float)(c_dx[k] * hx + c_dy[k] * hy);
    if (k == 0) hvec[h] = make_float2((float)hx, (float)hy);
  }
}

void launch_tables(int r, const sfm_params& p, float* T0, float* TX, float* TY, float* KO,
                   float* KE, float* own, float* dirdot, float2* hvec, cudaStream_t s) {
  const int n = (2 * r + 1) * (2 * r + 1);
  const int total = n > 81 ? n : 81;
  k_tables<<<dim3(cdiv(total, kTabThreads), 3), kTabThreads, 0, s>>>(
      r, p.kP, p.aP, p.gamma, p.kO, p.aO, p.kE, p.aE, T0, TX, TY, KO, KE, own, dirdot, hvec);
}

// ------------------------------------------------------------ static field
// F_static(c) = sum over WALL / EXIT su o within the window of K_O / K_E(c - o),
// a dense window gather over a shared-memory copy of the cell tile and its
// r-halo; compensated (Kahan) FP32 accumulation because up to (2r+1)^2 - 1
// terms enter one su.  Computed once per scene.
__global__ void __launch_bounds__(kFieldThreads)
    k_static_field(Geo g, const uint8_t* __restrict__ cell, const float* __restrict__ KO,
                   const float* __restrict__ KE, float* __restrict__ Fs) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int r = g.r, S = 2 * r + 1, nT = S * S, HW = kTile + 2 * r;
  float* sKO = reinterpret_cast<float*>(smem);
  float* sKE = sKO + nT;
  uint8_t* sC = reinterpret_cast<uint8_t*>(sKE + nT);
  const int tid = threadIdx.x;
  const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile;
  for (int i = tid; i < nT; i += blockDim.x) {
    sKO[i] = KO[i];
    sKE[i] = KE[i];
  }
  for (int i = tid; i < HW * HW; i += blockDim.x) {
    const int hx = i % HW, hy = i / HW;
    int gx, gy;
    uint8_t v = kFree;
    if (wrap_coord(x0 - r + hx, g.W, g.px, gx) && wrap_coord(y0 - r + hy, g.H, g.py, gy))
      v = cell[(size_t)gy * g.W + gx];
    sC[i] = v;
  }
  __syncthreads();
  const int lane = tid & 31, w = tid >> 5;
  float sum[kRowsPerThread], comp[kRowsPerThread];
#pragma unroll
  for (int j = 0; j < kRowsPerThread; ++j) sum[j] = comp[j] = 0.f;
  for (int dy = -r; dy <= r; ++dy) {
    for (int dx = -r; dx <= r; ++dx) {
      const int ti = (dy + r) * S + (dx + r);
      const float ko = sKO[ti], ke = sKE[ti];
      const uint8_t* col = sC + (lane - dx + r);
#pragma unroll
      for (int j = 0; j < kRowsPerThread; ++j) {
        const uint8_t b = col[(4 * w + j - dy + r) * HW];
        const float v = (b == kWall) ? ko : ((b == kExit) ? ke : 0.f);
        const float yk = v - comp[j];
        const float tk = sum[j] + yk;
        comp[j] = (tk - sum[j]) - yk;
        sum[j] = tk;
      }
    }
  }
  const int x = x0 + lane;
#pragma unroll
  for (int j = 0; j < kRowsPerThread; ++j) {
    const int y = y0 + 4 * w + j;
    if (x < g.W && y < g.H) Fs[(size_t)y * g.W + x] = sum[j];
  }
}

// From radius 12 on, the product of the wall and exit planes with the two
// laws' tables (sfm_product.cu; every entry as close to its law as FP32, the sum
// rounded once, like the compensated sum above).  The dense gather reads
// (2r + 1)^2 cells a su.  Set-up by the host's clock, product against gather: a
// 2048 x 2048 lattice 2.10 ms against 2.76 at radius 12 and 2.32 against 9.73 at
// 40; a 512 x 512 one 596 us against 591 and 753 against 1137; a 100 x 100 one,
// where the tables and a tile's start show, 309 against 277 and 464 against 574
// (320 both at 18).  The rule looks at the radius and the laws alone, so a
// lattice, its row bands and a batch round alike; the line lies where large
// lattices gain more than small ones lose.  (The cells' second limbs take a
// second table, for their precision: set-up of a 2048 x 2048 floor at radius 40
// 1350 -> 1481 us.)
constexpr int kStaticProductRadius = 12;
static bool static_product(int r, const sfm_params& prm, ProductScales* sc) {
  return r >= kStaticProductRadius && product_cell_scales(r, prm, sc);
}

size_t static_tmp_bytes(int r) {
  return r >= kStaticProductRadius && r <= kProductMaxRadius ? product_table_bytes(r, kCellPlanes) : 0;
}

void launch_static_field(const Geo& g, const uint8_t* cell, const Tables& tb, const sfm_params& prm,
                         float* Fs, void* tmp, Counters* ctr, cudaStream_t s) {
  ProductScales sc;
  if (static_product(g.r, prm, &sc)) {
    launch_limb_tables(g.r, prm, sc, kCellPlanes, static_cast<uint8_t*>(tmp), s);
    ProductArgs a;
    product_layout(g.r, &a);
    a.nch = kCellPlanes;
    a.ctr = ctr;
    a.store_hi = g.H;
    a.one.src = cell;
    a.one.spitch = g.W;
    a.one.out = Fs;
    a.one.tab = static_cast<const uint8_t*>(tmp);
    a.one.W = g.W;
    a.one.H = g.H;
    a.one.px = g.px;
    a.one.py = g.py;
    a.one.r = g.r;
    a.one.ntx = product_tiles_x(g.W);
    a.one.c0 = (float)(1.0 / sc.s0);
    a.one.c1 = (float)(1.0 / (sc.s0 * sc.s1));
    launch_product(a, s);
    return;
  }
  const int S = 2 * g.r + 1, HW = kTile + 2 * g.r;
  const size_t smem = (size_t)2 * S * S * sizeof(float) + (size_t)HW * HW;
  constexpr int kMaxS = 2 * SFM_MAX_RADIUS + 1, kMaxHW = kTile + 2 * SFM_MAX_RADIUS;
  allow_shared(k_static_field, (size_t)2 * kMaxS * kMaxS * sizeof(float) + (size_t)kMaxHW * kMaxHW);
  dim3 grid(cdiv(g.W, kTile), cdiv(g.H, kTile));
  k_static_field<<<grid, kFieldThreads, smem, s>>>(g, cell, tb.KO, tb.KE, Fs);
}

// --------------------------------------------------------------- guidance
// Chamfer (5, 7) geodesic distance to the nearest EXIT through non-WALL su
// (kDInf where none is reachable, kDWall on WALL su), the fixed point of
// D(c) = min_k D(c + Delta_k) + w_k.  The fixed point is unique and every
// update only lowers values towards it, so the result is exact whatever the
// order of the updates.
//
// Tiles of 32 x 32 su are relaxed in shared memory by persistent CTAs that
// take them from a queue, without rounds: a tile whose border a CTA lowers
// puts the neighbours that see it into the queue.  The time is the chain of
// tiles from an exit to the farthest su, so what matters is one tile's
// latency: a thread a su, a row looked at again only after it or the row
// above or below changed, and distances carried along a whole row or column
// by one scan, so a front crosses a tile in a few steps.  A 2048 x 2048 floor
// takes 563 us (one-pass ncu); a launch a round, with the host asking for the
// outcome of each, took 35 rounds of 36 us and their round trips: 1.9 ms
// (scene set-up 2.90 against 1.61 ms).  256 threads a tile, eight CTAs an SM:
// 878 us; without the scan down the columns 642.
constexpr int kGuideThreads = kTile * kTile;
// A wait lasts for a second at most, or this many looks.  It is one for one
// position: an idle CTA's comes nearer with every tile that is queued, each
// well under a millisecond after the last, so the wait covers a few hundred
// tiles however long the chain is (52 000 tiles in a row, the most before the
// distances end at 2^23: 0.28 s).
constexpr int kGuideSpins = 1 << 23;

__device__ __forceinline__ void guide_push(const GuideTiles& gt, int t, Counters* ctr) {
  if (!guide_mark(gt, t)) return;
  const unsigned pos = guide_position(gt);
  unsigned long long t0 = 0;
  for (int i = 0; !guide_publish(gt, pos, t); ++i) {
    if (i == kGuideSpins || second_is_over(i, t0)) {
      atomicOr(&ctr->err, kErrTimeout);
      return;
    }
    __nanosleep(100);
  }
}

// the next tile of the queue, -1 when no tile is left (or the wait ran out)
__device__ int guide_pop(const GuideTiles& gt, Counters* ctr) {
  const unsigned pos = guide_claim(gt);
  unsigned long long t0 = 0;
  for (int i = 0; i < kGuideSpins && !second_is_over(i, t0); ++i) {
    const int t = guide_take(gt, pos);
    if (t >= 0) {
      guide_unmark(gt, t);
      __threadfence();  // its values are read after that
      return t;
    }
    if (guide_over(guide_work(gt))) return -1;
    __nanosleep(100);
  }
  atomicOr(&ctr->err, kErrTimeout);
  return -1;
}

// neighbour (dx, dy) of tile (tx, ty), wrapped in periodic dimensions; -1: none
__device__ __forceinline__ int guide_neighbour(const Geo& g, int ntx, int nty, int tx, int ty, int dx, int dy) {
  int nx = tx + dx, ny = ty + dy;
  if (g.px) nx = (nx + ntx) % ntx;
  if (g.py) ny = (ny + nty) % nty;
  return nx >= 0 && nx < ntx && ny >= 0 && ny < nty ? ny * ntx + nx : -1;
}

// start values, and the tiles that see an exit into the queue (test: and one
// that no CTA will ever finish)
__global__ void __launch_bounds__(1024)
    k_guidance_init(Geo g, const uint8_t* __restrict__ cell, int32_t* __restrict__ D, GuideTiles gt,
                    Counters* ctr, int unfinished) {
  const int ntx = (g.W + kTile - 1) / kTile, nty = (g.H + kTile - 1) / kTile;
  const int tx = blockIdx.x % ntx, ty = blockIdx.x / ntx;
  const int x = tx * kTile + (threadIdx.x & 31), y = ty * kTile + (threadIdx.x >> 5);
  bool source = false;
  if (x < g.W && y < g.H) {
    const size_t c = (size_t)y * g.W + x;
    const uint8_t v = cell[c];
    source = v == kExit;
    D[c] = source ? 0 : (v == kWall ? kDWall : kDInf);
  }
  if (unfinished && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&gt.q->work, 1ull << 32);
  if (__syncthreads_or(source) && threadIdx.x < 9) {
    const int t = guide_neighbour(g, ntx, nty, tx, ty, (int)threadIdx.x % 3 - 1, (int)threadIdx.x / 3 - 1);
    if (t >= 0) guide_push(gt, t, ctr);
  }
}

// the exported form: WALL su read kDInf, like unreachable ones
__global__ void k_guidance_export(int32_t* __restrict__ D, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    if (D[i] == kDWall) D[i] = kDInf;
}

// the imported form: WALL su carry kDWall whatever the caller gave there
__global__ void k_guidance_import(const uint8_t* __restrict__ cell, int32_t* __restrict__ D, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    if (cell[i] == kWall) D[i] = kDWall;
}

// Distances carried along a line of 32 su (a lane a su), 5 a step, to the
// walls on either side (`open`: the line's su without walls), where some su
// lies more than a step above its neighbour.
__device__ __forceinline__ int guide_scan(int v, uint32_t open, int lane) {
  const bool mine = (open >> lane) & 1u;
  const int l1 = __shfl_up_sync(0xffffffffu, v, 1), r1 = __shfl_down_sync(0xffffffffu, v, 1);
  if (!__any_sync(0xffffffffu, mine && ((lane > 0 && v > l1 + 5) || (lane < 31 && v > r1 + 5)))) return v;
  // open su next to this one on either side
  const uint32_t below = ~open & ((1u << lane) - 1u), above = lane == 31 ? 0u : ~open >> (lane + 1);
  const int runl = mine ? (below ? lane - 32 + __clz(below) : lane) : 0;
  const int runr = mine ? (above ? __ffs(above) - 1 : 31 - lane) : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, v, o);
    if (runl >= o) v = min(v, u + 5 * o);
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_down_sync(0xffffffffu, v, o);
    if (runr >= o) v = min(v, u + 5 * o);
  }
  return v;
}

__global__ void __launch_bounds__(kGuideThreads, 2)
    k_guidance(Geo g, int32_t* __restrict__ D, GuideTiles gt, Counters* ctr) {
  // odd pitch: columns are read without bank conflicts too
  __shared__ int sD[kTile + 2][kTile + 3];
  __shared__ uint32_t s_open[kTile];               // su of a row that are inside and no walls
  __shared__ int s_row[kTile + 2], s_col[kTile];   // last step that changed a row, a column
  __shared__ int s_tile;
  __shared__ uint32_t s_edge;
  const int ntx = (g.W + kTile - 1) / kTile, nty = (g.H + kTile - 1) / kTile;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;  // lane: column, w: row (and column w of a scan)
  for (;;) {
    if (tid == 0) {
      s_tile = guide_pop(gt, ctr);
      s_edge = 0u;
    }
    __syncthreads();
    const int tile = s_tile;
    if (tile < 0) break;
    const int tx = tile % ntx, ty = tile / ntx, x0 = tx * kTile, y0 = ty * kTile;
    const int gx = x0 + lane, gy = y0 + w;
    // other CTAs lower these values meanwhile: read past L1.  Where a last
    // tile is cut short by a periodic lattice's end, the su just beyond it is
    // the one on the other side.
    int wx, wy;
    int32_t first = kDWall;
    if (gx <= g.W && gy <= g.H && wrap_coord(gx, g.W, g.px, wx) && wrap_coord(gy, g.H, g.py, wy))
      first = __ldcg(&D[(size_t)wy * g.W + wx]);
    sD[w + 1][lane + 1] = first;
    const uint32_t open = __ballot_sync(0xffffffffu, gx < g.W && gy < g.H && first != kDWall);
    if (lane == 0) s_open[w] = open;
    if (tid < kTile + 2) s_row[tid] = -1;
    if (tid < kTile) s_col[tid] = -1;
    if (tid < 4 * kTile + 4) {
      // the ring of su around the tile: two rows of 34, then two columns of 32
      int hx, hy;
      if (tid < 2 * (kTile + 2)) {
        hy = tid < kTile + 2 ? 0 : kTile + 1;
        hx = tid % (kTile + 2);
      } else {
        const int k = tid - 2 * (kTile + 2);
        hx = k < kTile ? 0 : kTile + 1;
        hy = 1 + k % kTile;
      }
      sD[hy][hx] = wrap_coord(x0 - 1 + hx, g.W, g.px, wx) && wrap_coord(y0 - 1 + hy, g.H, g.py, wy)
                       ? __ldcg(&D[(size_t)wy * g.W + wx])
                       : kDInf;
    }
    __syncthreads();
    const uint32_t copen = __ballot_sync(0xffffffffu, (s_open[lane] >> w) & 1u);  // column w
    volatile int(*vD)[kTile + 3] = sD;
    volatile int *vrow = s_row, *vcol = s_col;
    for (int step = 0; step < 4 * kTile * kTile; ++step) {
      bool changed = false;
      // rows: the eight neighbours, then along the row
      if (step == 0 || vrow[w] >= step - 1 || vrow[w + 1] >= step - 1 || vrow[w + 2] >= step - 1) {
        const int cur = vD[w + 1][lane + 1];
        int best = cur;
        if ((open >> lane) & 1u) {
          best = min(best, min(vD[w][lane + 1], vD[w + 2][lane + 1]) + 5);
          best = min(best, min(vD[w + 1][lane], vD[w + 1][lane + 2]) + 5);
          best = min(best, min(vD[w][lane], vD[w][lane + 2]) + 7);
          best = min(best, min(vD[w + 2][lane], vD[w + 2][lane + 2]) + 7);
        }
        best = guide_scan(best, open, lane);
        if (best < cur) {
          vD[w + 1][lane + 1] = best;
          vrow[w + 1] = step;
          vcol[lane] = step;
          changed = true;
        }
      }
      __syncthreads();
      // columns that changed: along the column
      if (vcol[w] == step) {
        const int cur = vD[lane + 1][w + 1], best = guide_scan(cur, copen, lane);
        if (best < cur) {
          vD[lane + 1][w + 1] = best;
          vrow[lane + 1] = step;
        }
      }
      if (!__syncthreads_or(changed)) break;
    }
    // what this CTA lowered (another one may be at the same tile: the smaller
    // value stays), and which neighbours see it: bit (dy + 1) * 3 + (dx + 1)
    uint32_t edge = 0u;
    const int v = vD[w + 1][lane + 1];
    if (v < first && gx < g.W && gy < g.H) {
      atomicMin(&D[(size_t)gy * g.W + gx], v);
      const bool l = lane == 0, r = lane == kTile - 1 || gx == g.W - 1;
      const bool t = w == 0, b = w == kTile - 1 || gy == g.H - 1;
      edge = (l ? 1u << 3 : 0u) | (r ? 1u << 5 : 0u) | (t ? 1u << 1 : 0u) | (b ? 1u << 7 : 0u) |
             (l && t ? 1u : 0u) | (r && t ? 1u << 2 : 0u) | (l && b ? 1u << 6 : 0u) | (r && b ? 1u << 8 : 0u);
    }
    edge = __reduce_or_sync(0xffffffffu, edge);
    if (lane == 0 && edge) atomicOr(&s_edge, edge);
    __threadfence();
    __syncthreads();
    if (tid < 32) {
      if (tid < 9 && ((s_edge >> tid) & 1u)) {
        const int t = guide_neighbour(g, ntx, nty, tx, ty, tid % 3 - 1, tid / 3 - 1);
        if (t >= 0) guide_push(gt, t, ctr);
      }
      __syncwarp();
      if (tid == 0) guide_done(gt);
    }
    __syncthreads();
  }
}

int device_sm_count() {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  if (!cached[dev]) {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    cached[dev] = n > 0 ? n : 1;
  }
  return cached[dev];
}

size_t guidance_scratch_ints(const Geo& g) {
  const size_t ntiles = (size_t)cdiv(g.W, kTile) * cdiv(g.H, kTile);
  return kGuideQueueInts + kGuideTileInts * ntiles;
}

void launch_guidance(const Geo& g, const uint8_t* cell, int32_t* D, int* scratch, Counters* ctr,
                     cudaStream_t s, bool unfinished) {
  const int ntiles = cdiv(g.W, kTile) * cdiv(g.H, kTile);
  const GuideTiles gt = guide_tiles(scratch, ntiles);
  cudaMemsetAsync(scratch, 0, guidance_scratch_ints(g) * sizeof(int), s);
  k_guidance_init<<<ntiles, 1024, 0, s>>>(g, cell, D, gt, ctr, unfinished);
  // CTAs wait for what running ones put into the queue or take out of it
  const int fit = 2 * device_sm_count();
  const int blocks = ntiles < fit ? ntiles : fit;
  k_guidance<<<blocks, kGuideThreads, 0, s>>>(g, D, gt, ctr);
}

void launch_guidance_export(int32_t* D, size_t n, cudaStream_t s) {
  if (!n) return;
  int blocks = (int)((n + 255) / 256);
  if (blocks > device_sm_count() * 64) blocks = device_sm_count() * 64;
  k_guidance_export<<<blocks, 256, 0, s>>>(D, n);
}

void launch_guidance_import(const uint8_t* cell, int32_t* D, size_t n, cudaStream_t s) {
  if (!n) return;
  int blocks = (int)((n + 255) / 256);
  if (blocks > device_sm_count() * 64) blocks = device_sm_count() * 64;
  k_guidance_import<<<blocks, 256, 0, s>>>(cell, D, n);
}

// ------------------------------------------------------------- placement
__global__ void k_place_clear(int n, const int2* __restrict__ xy, const uint8_t* __restrict__ alive,
                              Geo g, int32_t* __restrict__ occ, uint8_t* __restrict__ ocls,
                              Sizes sz) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n || !alive[p]) return;
  const int2 q = xy[p];
  const int a = sz.w ? sz.w[p] >> 1 : 0, b = sz.w ? sz.h[p] >> 1 : 0;
  for (int j = -b; j <= b; ++j)
    for (int i = -a; i <= a; ++i) {
      size_t s;
      if (rect_su(g, q.x, q.y, i, j, s)) occ[s] = -1;
    }
  ocls[(size_t)q.y * g.opitch + q.x] = 0;
}

__global__ void k_place_scatter(int n, const int2* __restrict__ xy,
                                const uint8_t* __restrict__ heading,
                                const uint8_t* __restrict__ goal, const uint8_t* __restrict__ alive,
                                const uint8_t* __restrict__ cell, Geo g, int32_t* __restrict__ occ,
                                uint8_t* __restrict__ ocls, Counters* ctr, Sizes sz) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  if (heading[p] > 8 || goal[p] > 8) atomicOr(&ctr->err, kErrPlaceRange);
  if (!alive[p]) return;
  const int2 q = xy[p];
  if (q.x < 0 || q.x >= g.W || q.y < 0 || q.y >= g.H) {
    atomicOr(&ctr->err, kErrPlaceRange);
    return;
  }
  const size_t c = (size_t)q.y * g.W + q.x;
  if (cell[c] != kFree) atomicOr(&ctr->err, kErrPlaceConflict);
  // the rectangle (1 x 1 without sizes): inside, off walls, on nobody else
  const int a = sz.w ? sz.w[p] >> 1 : 0, b = sz.w ? sz.h[p] >> 1 : 0;
  for (int j = -b; j <= b; ++j)
    for (int i = -a; i <= a; ++i) {
      size_t s;
      if (!rect_su(g, q.x, q.y, i, j, s)) {
        atomicOr(&ctr->err, kErrPlaceConflict);
        continue;
      }
      if (cell[s] == kWall || atomicCAS(&occ[s], -1, p) != -1)
        atomicOr(&ctr->err, kErrPlaceConflict);
    }
  ocls[(size_t)q.y * g.opitch + q.x] = (uint8_t)(1 + (heading[p] > 8 ? 0 : heading[p]));
}

void launch_place_clear(int n, const int2* xy, const uint8_t* alive, const Geo& g, int32_t* occ,
                        uint8_t* ocls, cudaStream_t s, const Sizes& sz) {
  if (n <= 0) return;
  k_place_clear<<<cdiv(n, 256), 256, 0, s>>>(n, xy, alive, g, occ, ocls, sz);
}

// A placement of as many 1 x 1 pedestrians into the same arrays (the tick
// graphs are kept).  Only pedestrians whose su or alive flag changes leave
// (leave_su) and claim (claim_su, with the checks of k_place_scatter)
// occupancy-grid entries, in two launches so that a su vacated by one may be
// claimed by another; a pedestrian that keeps its su only rewrites its class
// entry when its heading changed.  The entries of the others are already
// right: the previous placement validated them and every tick keeps the grids
// in step with the pedestrians.

// Pedestrian p, alive at q before the placement, is placed at v (alive: a):
// frees q unless it stays there.
__device__ __forceinline__ void leave_su(int2 q, int2 v, uint8_t a, const Geo& g,
                                         int32_t* __restrict__ occ, uint8_t* __restrict__ ocls) {
  if (a && q.x == v.x && q.y == v.y) return;
  occ[(size_t)q.y * g.W + q.x] = -1;
  ocls[(size_t)q.y * g.opitch + q.x] = 0;
}

// Live pedestrian p placed at v with heading hp; before the placement it was
// at q (if a_old) with heading h_old.
__device__ __forceinline__ void claim_su(int p, int2 v, uint8_t hp, bool a_old, int2 q,
                                         uint8_t h_old, const uint8_t* __restrict__ cell,
                                         const Geo& g, int32_t* __restrict__ occ,
                                         uint8_t* __restrict__ ocls, Counters* ctr) {
  const uint8_t cls = (uint8_t)(1 + (hp > 8 ? 0 : hp));
  if (a_old && q.x == v.x && q.y == v.y) {
    if (hp != h_old) ocls[(size_t)v.y * g.opitch + v.x] = cls;
    return;
  }
  if (v.x < 0 || v.x >= g.W || v.y < 0 || v.y >= g.H) {
    atomicOr(&ctr->err, kErrPlaceRange);
    return;
  }
  const size_t c = (size_t)v.y * g.W + v.x;
  if (cell[c] != kFree || atomicCAS(&occ[c], -1, p) != -1) atomicOr(&ctr->err, kErrPlaceConflict);
  ocls[(size_t)v.y * g.opitch + v.x] = cls;
}

// From copies: xy_prev / alive_prev / heading_prev hold the state before the
// placement, xy / heading / goal / alive the new one.
__global__ void k_place_diff_clear(int n, const int2* __restrict__ xy_prev,
                                   const uint8_t* __restrict__ alive_prev,
                                   const int2* __restrict__ xy, const uint8_t* __restrict__ alive,
                                   Geo g, int32_t* __restrict__ occ, uint8_t* __restrict__ ocls) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n || !alive_prev[p]) return;
  leave_su(xy_prev[p], xy[p], alive[p], g, occ, ocls);
}

__global__ void k_place_diff_claim(int n, const int2* __restrict__ xy_prev,
                                   const uint8_t* __restrict__ alive_prev,
                                   const uint8_t* __restrict__ heading_prev,
                                   const int2* __restrict__ xy, const uint8_t* __restrict__ heading,
                                   const uint8_t* __restrict__ goal, const uint8_t* __restrict__ alive,
                                   const uint8_t* __restrict__ cell, Geo g, int32_t* __restrict__ occ,
                                   uint8_t* __restrict__ ocls, Counters* ctr) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const uint8_t hp = heading[p];
  if (hp > 8 || goal[p] > 8) atomicOr(&ctr->err, kErrPlaceRange);
  if (!alive[p]) return;
  claim_su(p, xy[p], hp, alive_prev[p] != 0, xy_prev[p], heading_prev[p], cell, g, occ, ocls, ctr);
}

// The same placement read in place from the caller's buffers (device memory
// or pinned host memory mapped into the device's address space; a NULL
// heading, goal or alive array stands for 0, 0, 1): the first launch stages
// the new state in st_* and clears the su of the pedestrians that leave
// theirs; the second claims the su of those that take a new one (the checks
// of k_place_scatter), rewrites the class entry of those that turn in place,
// and installs the new state with cleared decisions.
__global__ void k_place_direct_stage(int n, const int2* __restrict__ src_xy,
                                     const uint8_t* __restrict__ src_h,
                                     const uint8_t* __restrict__ src_g,
                                     const uint8_t* __restrict__ src_a, int2* __restrict__ st_xy,
                                     uint8_t* __restrict__ st_h, uint8_t* __restrict__ st_g,
                                     uint8_t* __restrict__ st_a, const int2* __restrict__ xy,
                                     const uint8_t* __restrict__ alive, Geo g,
                                     int32_t* __restrict__ occ, uint8_t* __restrict__ ocls) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int2 v = src_xy[p];
  const uint8_t a = src_a ? src_a[p] : 1;
  st_xy[p] = v;
  st_h[p] = src_h ? src_h[p] : 0;
  st_g[p] = src_g ? src_g[p] : 0;
  st_a[p] = a;
  if (alive[p]) leave_su(xy[p], v, a, g, occ, ocls);
}

__global__ void k_place_direct_claim(int n, const int2* __restrict__ st_xy,
                                     const uint8_t* __restrict__ st_h,
                                     const uint8_t* __restrict__ st_g,
                                     const uint8_t* __restrict__ st_a, int2* __restrict__ xy,
                                     uint8_t* __restrict__ heading, uint8_t* __restrict__ goal,
                                     uint8_t* __restrict__ alive, uint8_t* __restrict__ choice,
                                     uint8_t* __restrict__ won, const uint8_t* __restrict__ cell,
                                     Geo g, int32_t* __restrict__ occ, uint8_t* __restrict__ ocls,
                                     Counters* ctr) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int2 v = st_xy[p], q = xy[p];
  const uint8_t hp = st_h[p], gp = st_g[p], ap = st_a[p], a_old = alive[p], h_old = heading[p];
  xy[p] = v;
  heading[p] = hp;
  goal[p] = gp;
  alive[p] = ap;
  choice[p] = 0;
  won[p] = 0;
  if (hp > 8 || gp > 8) atomicOr(&ctr->err, kErrPlaceRange);
  if (ap) claim_su(p, v, hp, a_old != 0, q, h_old, cell, g, occ, ocls, ctr);
}

void launch_place_direct(int n, const int2* src_xy, const uint8_t* src_h, const uint8_t* src_g,
                         const uint8_t* src_a, int2* st_xy, uint8_t* st_h, uint8_t* st_g,
                         uint8_t* st_a, int2* xy, uint8_t* heading, uint8_t* goal, uint8_t* alive,
                         uint8_t* choice, uint8_t* won, const uint8_t* cell, const Geo& g,
                         int32_t* occ, uint8_t* ocls, Counters* ctr, cudaStream_t s) {
  if (n <= 0) return;
  // one pedestrian a thread: many small reads in flight move pinned host
  // buffers faster than fewer, wider ones (measured: 4 a thread with 16-byte
  // accesses slowed the read-back from 0.078 to 0.126 ms for 10^6)
  k_place_direct_stage<<<cdiv(n, 256), 256, 0, s>>>(n, src_xy, src_h, src_g, src_a, st_xy, st_h, st_g,
                                                    st_a, xy, alive, g, occ, ocls);
  k_place_direct_claim<<<cdiv(n, 256), 256, 0, s>>>(n, st_xy, st_h, st_g, st_a, xy, heading, goal,
                                                    alive, choice, won, cell, g, occ, ocls, ctr);
}

// Pedestrian state written in place into the caller's buffers (any may be
// NULL; device memory or mapped pinned host memory), one pedestrian a thread.
__global__ void k_read_peds(int n, const int2* __restrict__ xy, const uint8_t* __restrict__ heading,
                            const uint8_t* __restrict__ alive, int2* __restrict__ dxy,
                            uint8_t* __restrict__ dh, uint8_t* __restrict__ da) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  if (dxy) dxy[p] = xy[p];
  if (dh) dh[p] = heading[p];
  if (da) da[p] = alive[p];
}

void launch_read_peds(int n, const int2* xy, const uint8_t* heading, const uint8_t* alive, int2* dxy,
                      uint8_t* dh, uint8_t* da, cudaStream_t s) {
  if (n <= 0) return;
  k_read_peds<<<cdiv(n, 256), 256, 0, s>>>(n, xy, heading, alive, dxy, dh, da);
}

void launch_place_diff(int n, const int2* xy_prev, const uint8_t* alive_prev,
                       const uint8_t* heading_prev, const int2* xy, const uint8_t* heading,
                       const uint8_t* goal, const uint8_t* alive, const uint8_t* cell, const Geo& g,
                       int32_t* occ, uint8_t* ocls, Counters* ctr, cudaStream_t s) {
  if (n <= 0) return;
  k_place_diff_clear<<<cdiv(n, 256), 256, 0, s>>>(n, xy_prev, alive_prev, xy, alive, g, occ, ocls);
  k_place_diff_claim<<<cdiv(n, 256), 256, 0, s>>>(n, xy_prev, alive_prev, heading_prev, xy, heading,
                                                  goal, alive, cell, g, occ, ocls, ctr);
}

// per-placement counters and flags back to zero (the tick counter stays)
__global__ void k_reset_counters(Counters* ctr) {
  ctr->moved = 0;
  ctr->exited = 0;
  ctr->max_registrants = 0;
  ctr->err = 0;
  ctr->decided = 0;
  ctr->near_ties = 0;
}

void launch_reset_counters(Counters* ctr, cudaStream_t s) { k_reset_counters<<<1, 1, 0, s>>>(ctr); }

void launch_place_scatter(int n, const int2* xy, const uint8_t* heading, const uint8_t* goal,
                          const uint8_t* alive, const uint8_t* cell, const Geo& g, int32_t* occ,
                          uint8_t* ocls, Counters* ctr, cudaStream_t s, const Sizes& sz) {
  if (n <= 0) return;
  k_place_scatter<<<cdiv(n, 256), 256, 0, s>>>(n, xy, heading, goal, alive, cell, g, occ, ocls,
                                               ctr, sz);
}

// --------------------------------------------------------- S1: binning
// Counting sort of the live pedestrians into 32 x 32-su bins, read off the
// per-su occupancy-class grid so that the order inside a bin is row-major
// and therefore deterministic; one warp a bin.
constexpr int kBinWarps = 4;  // bins a block: small blocks spread a small lattice's bins over the SMs

__global__ void k_bin_count(Geo g, const uint8_t* ocls, int32_t* count) {
  tick_kernel_begin();
  const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (b >= g.nbx * g.nby) return;
  const int c = bin_count_one(g, ocls, b % g.nbx, b / g.nbx, lane);
  if (lane == 0) count[b] = c;
}

// launches of launch_scan: two passes, or one when a block covers all n
static int scan_launches(int n) { return scan_tmp_elems(n) == 1 ? 1 : 2; }

// SCANNED: a scan has put the bins' first slots into `start`; else a block adds
// up the counts of the bins before its own and writes its part of `start`.
template <bool SCANNED>
__global__ void __launch_bounds__(32 * kBinWarps)
    k_bin_fill(Geo g, const uint8_t* ocls, const int32_t* occ, const int32_t* count, int32_t* start,
               uint32_t* rec, int32_t* rec_id) {
  tick_kernel_begin();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nbins = g.nbx * g.nby, b0 = blockIdx.x * kBinWarps, b = b0 + warp;
  int first = 0;
  if (SCANNED) {
    if (b < nbins) first = start[b];
  } else {
    __shared__ int sBefore[kBinWarps], sMine[kBinWarps];
    int before = 0;
#pragma unroll 8
    for (int i = threadIdx.x; i < b0; i += 32 * kBinWarps) before += count[i];
    const int mine = b < nbins ? count[b] : 0;
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) {
      sBefore[warp] = before;
      sMine[warp] = mine;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kBinWarps; ++w) first += sBefore[w] + (w < warp ? sMine[w] : 0);
    if (lane == 0 && b < nbins) {
      start[b] = first;
      if (b == nbins - 1) start[nbins] = first + mine;
    }
  }
  if (b >= nbins) return;
  bin_fill_one(g, ocls, occ, first, rec, rec_id, b % g.nbx, b / g.nbx, lane);
}

// Launches, not work, are what binning a small lattice costs, so its scan is
// part of the fill: a tick of a 100 x 100 lattice took 24.3 us with a scan of
// its own and 21.4 without, one of 512 x 512 34.6 and 32.3, one of 2048 x 2048
// (4096 bins, as many as the one-launch scan takes; a block then adds up 16 KB
// of counts at most) 112.3 and 110.4.  Counting in the fill as well, each
// block the bins before its own, gained nothing (21.5 us with 16 bins, 35.8
// against 29.7 with 64).
int launch_bins_from_grid(const Geo& g, const uint8_t* ocls, const int32_t* occ, int32_t* count,
                          int32_t* start, int32_t* scan_tmp, uint32_t* rec, int32_t* rec_id,
                          cudaStream_t s, bool early) {
  const int nbins = g.nbx * g.nby, blocks = cdiv(nbins, kBinWarps), threads = 32 * kBinWarps;
  launch_tick_kernel(k_bin_count, blocks, threads, 0, s, early, g, ocls, count);
  if (nbins <= kBinsPrefix) {
    launch_tick_kernel(k_bin_fill<false>, blocks, threads, 0, s, early, g, ocls, occ,
                       count, start, rec, rec_id);
    return 2;
  }
  launch_scan(count, start, nbins, scan_tmp, s);
  launch_tick_kernel(k_bin_fill<true>, blocks, threads, 0, s, early, g, ocls, occ, count,
                     start, rec, rec_id);
  return 2 + scan_launches(nbins);
}

// The same records driven by the pedestrian list, for sparse crowds where
// reading the whole class grid costs more than the pedestrians: count with
// atomics (each pedestrian keeps its arrival slot), scan, scatter each
// pedestrian's su key (row << 5 | column inside the bin) to its slot, then
// rank: a pedestrian's place in its bin is the number of smaller keys there
// (keys are unique, one pedestrian per su), which is the row-major order of
// the grid path.  Work per pedestrian is the size of its bin.
__device__ __forceinline__ int ped_bin(const Geo& g, int2 q) {
  return (q.y / kBin) * g.nbx + q.x / kBin;
}

__global__ void k_binp_count(int n, Geo g, const int2* __restrict__ xy,
                             const uint8_t* __restrict__ alive, int32_t* __restrict__ count,
                             int32_t* __restrict__ slot) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n || !alive[p]) return;
  slot[p] = atomicAdd(&count[ped_bin(g, xy[p])], 1);
}

__global__ void k_binp_scatter(int n, Geo g, const int2* __restrict__ xy,
                               const uint8_t* __restrict__ alive, const int32_t* __restrict__ slot,
                               const int32_t* __restrict__ start, uint32_t* __restrict__ key) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n || !alive[p]) return;
  const int2 q = xy[p];
  key[start[ped_bin(g, q)] + slot[p]] = (uint32_t)((q.y % kBin) << 5 | (q.x % kBin));
}

__global__ void k_binp_rank(int n, Geo g, const int2* __restrict__ xy,
                            const uint8_t* __restrict__ alive, const uint8_t* __restrict__ heading,
                            const int32_t* __restrict__ start, const uint32_t* __restrict__ key,
                            uint32_t* __restrict__ rec, int32_t* __restrict__ rec_id) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n || !alive[p]) return;
  const int2 q = xy[p];
  const int b = ped_bin(g, q);
  const int s = start[b], e = start[b + 1];
  const int col = q.x % kBin, row = q.y % kBin;
  const uint32_t mine = (uint32_t)(row << 5 | col);
  int rank = 0;
  for (int i = s; i < e; ++i) rank += key[i] < mine;
  const uint32_t cls = heading[p] > 8 ? 0u : heading[p];
  rec[s + rank] = (uint32_t)col | ((uint32_t)row << 8) | (cls << 16);
  rec_id[s + rank] = p;
}

int launch_bins_from_peds(const Geo& g, int n, const int2* xy, const uint8_t* alive,
                          const uint8_t* heading, int32_t* count, int32_t* start,
                          int32_t* scan_tmp, int32_t* slot, uint32_t* key, uint32_t* rec,
                          int32_t* rec_id, cudaStream_t s) {
  const int nbins = g.nbx * g.nby;
  cudaMemsetAsync(count, 0, (size_t)nbins * sizeof(int32_t), s);
  if (n > 0) k_binp_count<<<cdiv(n, 256), 256, 0, s>>>(n, g, xy, alive, count, slot);
  launch_scan(count, start, nbins, scan_tmp, s);
  if (n <= 0) return scan_launches(nbins);
  k_binp_scatter<<<cdiv(n, 256), 256, 0, s>>>(n, g, xy, alive, slot, start, key);
  k_binp_rank<<<cdiv(n, 256), 256, 0, s>>>(n, g, xy, alive, heading, start, key, rec, rec_id);
  return 3 + scan_launches(nbins);
}

// ------------------------------------------------------------------ scan
// Exclusive prefix sum of n int32 into out[0..n] (out[n] = total), two passes:
// per-block totals, and the final one, in which a block adds up the totals
// before it (a pass of its own for them took 2.5 us); only the final one when a
// block covers all n.
constexpr int kScanThreads = 1024, kScanItems = 4, kScanChunk = kScanThreads * kScanItems;

__device__ int block_exclusive_scan(int v, int* sWarp, int& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) sWarp[w] = inc;
  __syncthreads();
  if (w == 0) {
    int s = lane < nw ? sWarp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += t;
    }
    if (lane < nw) sWarp[lane] = s;
  }
  __syncthreads();
  total = sWarp[nw - 1];
  const int excl = inc - v + (w > 0 ? sWarp[w - 1] : 0);
  __syncthreads();
  return excl;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_totals(const int32_t* __restrict__ in, int n,
                                                              int32_t* __restrict__ totals) {
  __shared__ int sWarp[32];
  const int base = blockIdx.x * kScanChunk + threadIdx.x * kScanItems;
  int s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k)
    if (base + k < n) s += in[base + k];
  int total;
  block_exclusive_scan(s, sWarp, total);
  if (threadIdx.x == 0) totals[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_final(const int32_t* __restrict__ in, int n,
                                                             const int32_t* __restrict__ totals,
                                                             int32_t* __restrict__ out) {
  __shared__ int sWarp[32];
  const int i0 = blockIdx.x * kScanChunk + threadIdx.x * kScanItems;
  int v[kScanItems], s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    v[k] = (i0 + k < n) ? in[i0 + k] : 0;
    s += v[k];
  }
  int total, before = 0;
  if (totals) {  // of the blocks before this one
    int t = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += kScanThreads) t += totals[b];
    block_exclusive_scan(t, sWarp, before);
  }
  int e = block_exclusive_scan(s, sWarp, total) + before;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    if (i0 + k < n) out[i0 + k] = e;
    e += v[k];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1) out[n] = e;
}

int scan_tmp_elems(int n) { return cdiv(n > 0 ? n : 1, kScanChunk); }

void launch_scan(const int32_t* in, int32_t* out, int n, int32_t* block_tmp, cudaStream_t s) {
  const int nb = scan_tmp_elems(n);
  if (nb > 1) k_scan_totals<<<nb, kScanThreads, 0, s>>>(in, n, block_tmp);
  k_scan_final<<<nb, kScanThreads, 0, s>>>(in, n, nb > 1 ? block_tmp : nullptr, out);
}

// ------------------------------------ S2: field gather for radius > 50
// Used where the heading-class tables would not fit in shared memory (the
// class-table gather in sfm_field.cu covers radius <= 50).  Each CTA owns a
// 32 x 32 su tile.  The pedestrians of the bins that overlap
// the tile's r-halo are staged in shared memory in chunks of at most `cap`
// records (the bounded multi-step sum of Alg. 3 / Eq. 1: the per-su sum is
// split into a fixed number of partial passes), every lane accumulates the
// kernel-table value of each staged pedestrian inside its window for its 4
// rows, and the tile is written once as F = F_static + sum.
struct HaloBin {
  int start, count, xoff, yoff;
};
constexpr int kMaxImages = 24;

// Bins (one dimension) overlapping the halo [lo, hi]; returns entries (bin,
// offset of the bin origin relative to the tile origin).
__device__ int halo_list(int lo, int hi, int n, int periodic, int nbins, int t0, int* bin,
                         int* off) {
  int cnt = 0;
  if (!periodic) {
    if (lo < 0) lo = 0;
    if (hi > n - 1) hi = n - 1;
    for (int b = lo / kBin; lo <= hi && b <= hi / kBin; ++b) {
      if (cnt < kMaxImages) { bin[cnt] = b; off[cnt] = b * kBin - t0; }
      ++cnt;
    }
    return cnt;
  }
  const int k0 = floor_div(lo, n), k1 = floor_div(hi, n);
  for (int k = k0; k <= k1; ++k) {
    int a = lo - k * n, z = hi - k * n;
    if (a < 0) a = 0;
    if (z > n - 1) z = n - 1;
    for (int b = a / kBin; a <= z && b <= z / kBin; ++b) {
      if (cnt < kMaxImages) { bin[cnt] = b; off[cnt] = b * kBin + k * n - t0; }
      ++cnt;
    }
  }
  (void)nbins;
  return cnt;
}

__global__ void __launch_bounds__(kFieldThreads)
    k_field(Geo g, const int32_t* __restrict__ bin_start, const uint32_t* __restrict__ rec,
            Tables tb, const float* __restrict__ Fs, float* __restrict__ out, int out_row0,
            int ty0, int store_lo, int store_hi, int cap, Counters* ctr) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ HaloBin sBins[kMaxImages * kMaxImages];
  __shared__ int sPref[kMaxImages * kMaxImages + 1];
  __shared__ int sNB;
  const int r = g.r, S = 2 * r + 1, nT = S * S;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  int4* sPed = reinterpret_cast<int4*>(smem);
  float* sT0 = reinterpret_cast<float*>(sPed + cap);
  float* sTX = sT0 + nT;
  float* sTY = sTX + nT;
  const int x0 = blockIdx.x * kTile, y0 = (ty0 + blockIdx.y) * kTile;

  for (int i = tid; i < nT; i += blockDim.x) {
    sT0[i] = tb.T0[i];
    sTX[i] = tb.TX[i];
    sTY[i] = tb.TY[i];
  }
  if (tid == 0) {
    int bxs[kMaxImages], xo[kMaxImages], bys[kMaxImages], yo[kMaxImages];
    const int nxl = halo_list(x0 - r, x0 + kTile - 1 + r, g.W, g.px, g.nbx, x0, bxs, xo);
    const int nyl = halo_list(y0 - r, y0 + kTile - 1 + r, g.H, g.py, g.nby, y0, bys, yo);
    int nb = 0;
    if (nxl > kMaxImages || nyl > kMaxImages) {
      atomicOr(&ctr->err, kErrHalo);
    } else {
      for (int a = 0; a < nyl; ++a)
        for (int b = 0; b < nxl; ++b) {
          sBins[nb].start = bys[a] * g.nbx + bxs[b];  // bin id for now
          sBins[nb].xoff = xo[b];
          sBins[nb].yoff = yo[a];
          ++nb;
        }
    }
    sNB = nb;
  }
  __syncthreads();
  const int nb = sNB;
  for (int i = tid; i < nb; i += blockDim.x) {
    const int id = sBins[i].start;
    const int s0 = bin_start[id];
    sBins[i].start = s0;
    sBins[i].count = bin_start[id + 1] - s0;
  }
  __syncthreads();
  if (tid == 0) {
    int acc = 0;
    for (int i = 0; i < nb; ++i) {
      sPref[i] = acc;
      acc += sBins[i].count;
    }
    sPref[nb] = acc;
  }
  __syncthreads();
  const int total = sPref[nb];

  float acc[kRowsPerThread];
#pragma unroll
  for (int j = 0; j < kRowsPerThread; ++j) acc[j] = 0.f;
  const int rowb = kRowsPerThread * w;  // first row of this warp inside the tile

  for (int base = 0; base < total; base += cap) {
    const int cnt = min(cap, total - base);
    for (int i = tid; i < cnt; i += blockDim.x) {
      const int q = base + i;
      int lo = 0, hi = nb;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (sPref[mid] <= q) lo = mid; else hi = mid;
      }
      const uint32_t rc = rec[sBins[lo].start + (q - sPref[lo])];
      const int cls = (rc >> 16) & 0xf;
      const float2 h = tb.hvec[cls];
      sPed[i] = make_int4(sBins[lo].xoff + (int)(rc & 0xff), sBins[lo].yoff + (int)((rc >> 8) & 0xff),
                          __float_as_int(h.x), __float_as_int(h.y));
    }
    __syncthreads();
    for (int i = 0; i < cnt; ++i) {
      const int4 pd = sPed[i];
      const int dyb = rowb - pd.y;  // dy of this warp's first row
      if (dyb + kRowsPerThread - 1 < -r || dyb > r) continue;    // warp-uniform
      if (kTile - 1 - pd.x < -r || -pd.x > r) continue;          // warp-uniform
      const int dx = lane - pd.x;
      if ((unsigned)(dx + r) > (unsigned)(2 * r)) continue;
      const float hx = __int_as_float(pd.z), hy = __int_as_float(pd.w);
#pragma unroll
      for (int j = 0; j < kRowsPerThread; ++j) {
        const int dy = dyb + j;
        if ((unsigned)(dy + r) <= (unsigned)(2 * r)) {
          const int ti = (dy + r) * S + (dx + r);
          acc[j] += fmaf(hy, sTY[ti], fmaf(hx, sTX[ti], sT0[ti]));
        }
      }
    }
    __syncthreads();
  }
  const int x = x0 + lane;
#pragma unroll
  for (int j = 0; j < kRowsPerThread; ++j) {
    const int y = y0 + rowb + j;
    if (x < g.W && y < g.H && y >= store_lo && y < store_hi) {
      const size_t c = (size_t)y * g.W + x;
      out[(size_t)(y - out_row0) * g.W + x] = Fs[c] + acc[j];
    }
  }
}

constexpr size_t kFieldBudget = 200 * 1024;
static_assert((size_t)3 * (2 * SFM_MAX_RADIUS + 1) * (2 * SFM_MAX_RADIUS + 1) * sizeof(float) +
                      256 * sizeof(int4) <= kFieldBudget, "tables and a chunk fit at any radius");
static int field_cap(int r, size_t* smem_out) {
  const int S = 2 * r + 1;
  const size_t tables = (size_t)3 * S * S * sizeof(float);
  int cap = kStageCap;
  while (cap > 256 && tables + (size_t)cap * sizeof(int4) > kFieldBudget) cap >>= 1;
  *smem_out = tables + (size_t)cap * sizeof(int4);
  return cap;
}

cudaError_t launch_field_v1(const Geo& g, const int32_t* bin_start, const uint32_t* rec,
                            const Tables& tb, const float* Fs, float* out, int out_row0,
                            int store_lo, int store_hi, Counters* ctr, cudaStream_t s) {
  const int ty0 = store_lo / kTile, ty1 = (store_hi + kTile - 1) / kTile;
  if (ty1 <= ty0) return cudaSuccess;
  size_t smem;
  const int cap = field_cap(g.r, &smem);
  allow_shared(k_field, kFieldBudget);
  dim3 grid(cdiv(g.W, kTile), ty1 - ty0);
  k_field<<<grid, kFieldThreads, smem, s>>>(g, bin_start, rec, tb, Fs, out, out_row0, ty0,
                                            store_lo, store_hi, cap, ctr);
  return cudaPeekAtLastError();
}

__global__ void k_class_tables(int r, int SP, double kP, double aP, double gamma, double taper_in,
                               float* __restrict__ T) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < class_table_entries(r, SP)) class_table_entry(i, r, SP, kP, aP, gamma, taper_in, T);
}

int class_table_stride(int r) { return class_table_stride_of(r); }

size_t class_table_floats(int r) { return class_table_floats_of(r); }

static void class_tables(int r, int sp, const sfm_params& p, float* T, cudaStream_t s, double taper_in) {
  if (!sp) return;
  k_class_tables<<<cdiv(class_table_entries(r, sp), 128), 128, 0, s>>>(r, sp, p.kP, p.aP, p.gamma, taper_in,
                                                                       T);
}

void launch_class_tables(int r, const sfm_params& p, float* T, cudaStream_t s, double taper_in) {
  class_tables(r, class_table_stride(r), p, T, s, taper_in);
}

// in the layout of the row-trimmed gather
void launch_class_tables3(int r, const sfm_params& p, float* T, cudaStream_t s) {
  class_tables(r, field3_stride(r), p, T, s, 1e30);
}

// --------------------------------------------------------- S3: decide
// Per live pedestrian (visited in bin order, so neighbouring threads read
// neighbouring su): E over the 9 candidates (stay + 8 neighbours), admissible
// iff inside, not WALL and unoccupied at tick start; select of the minimum
// with ties to the smallest class.
__global__ void __launch_bounds__(256, 4) k_decide(const int32_t* __restrict__ rec_id, const int32_t* __restrict__ bin_start,
                         int b_lo, int b_hi, const int2* __restrict__ xy,
                         const uint8_t* __restrict__ heading, const uint8_t* __restrict__ goal,
                         const uint8_t* __restrict__ ocls, const int32_t* __restrict__ D,
                         const float* __restrict__ F, int main_off,
                         int lo_row, int hi_row, int hi_off, int y_lo, int y_hi, Geo g,
                         float beta, const float* __restrict__ own,
                         const float* __restrict__ dirdot, uint8_t* __restrict__ choice,
                         WalkPeriods wp, Counters* __restrict__ ctr, int ring) {
  let_next_start();  // the next band's gather copies its tables on the SMs that are done
  // grid-stride over the records of bins [b_lo, b_hi): a band's launch needs
  // no more blocks than the GPU holds, whatever its share of the crowd.  The
  // records are taken from the last backwards: the gather wrote the band's
  // bottom rows last, so the first blocks find their field rows still in L2
  // (0.199 -> 0.195 ms a banded floor tick).
  const int end = bin_start[b_hi];
  const long long t = wp.period ? wp.ctr->t : 0;
  const int cnt = end - bin_start[b_lo];
  unsigned decided = 0, ties = 0;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < cnt; k += gridDim.x * blockDim.x) {
    const int p = rec_id[end - 1 - k];
    if (wp.period && t % wp.period[p] != wp.phase[p]) {
      choice[p] = 0;  // not this pedestrian's tick: it stays
      continue;
    }
    bool tie = false;
    choice[p] = decide_one<true>(p, g, xy, heading, goal, ocls, D, F, main_off, lo_row,
                                 hi_row, hi_off, y_lo, y_hi, beta, own, dirdot, &tie, ring);
    ++decided;
    ties += tie ? 1u : 0u;
  }
  // decisions and near ties, one atomic per warp
  decided = __reduce_add_sync(0xffffffffu, decided);
  ties = __reduce_add_sync(0xffffffffu, ties);
  if (ctr && (threadIdx.x & 31) == 0 && decided) {
    atomicAdd(&ctr->decided, (unsigned long long)decided);
    if (ties) atomicAdd(&ctr->near_ties, (unsigned long long)ties);
  }
}

// Multi-su pedestrians, kQuad lanes each, which share the su that it may enter:
// the chains of dependent reads bound these stages (55 000 pedestrians of 3 x 3
// su on 1000 x 1000: decide 22 -> 18 us and vote 29 -> 19, against a thread a
// pedestrian that tests the su of each move one after the other).
constexpr int kQuad = 4;

__global__ void __launch_bounds__(256, 4)
    k_decide_sized(const int32_t* __restrict__ rec_id, const int32_t* __restrict__ bin_start, int b_lo,
                   int b_hi, const int2* __restrict__ xy, const uint8_t* __restrict__ heading,
                   const uint8_t* __restrict__ goal, const uint8_t* __restrict__ cell,
                   const int32_t* __restrict__ D, const float* __restrict__ F, int main_off, int lo_row,
                   int hi_row, int hi_off, int y_lo, int y_hi, Geo g, float beta,
                   const float* __restrict__ own, const float* __restrict__ dirdot,
                   uint8_t* __restrict__ choice, WalkPeriods wp, Sizes sz,
                   const int32_t* __restrict__ occ, Counters* __restrict__ ctr, int ring) {
  const int end = bin_start[b_hi], cnt = end - bin_start[b_lo];
  const long long t = wp.period ? wp.ctr->t : 0;
  const int sub = threadIdx.x % kQuad, step = gridDim.x * blockDim.x / kQuad;
  unsigned decided = 0, ties = 0;
  for (int k0 = blockIdx.x * blockDim.x / kQuad; k0 < cnt; k0 += step) {
    const int k = k0 + threadIdx.x / kQuad;
    const int p = k < cnt ? rec_id[end - 1 - k] : -1;
    const bool walks = p >= 0 && !(wp.period && t % wp.period[p] != wp.phase[p]);
    uint32_t blocked = 0;
    if (walks) {
      const int2 q = xy[p];
      blocked = blocked_moves<kQuad>(g, cell, occ, q.x, q.y, sz.w[p] >> 1, sz.h[p] >> 1, sub);
    }
#pragma unroll
    for (int o = 1; o < kQuad; o <<= 1) blocked |= __shfl_xor_sync(0xffffffffu, blocked, o);
    if (p < 0 || sub) continue;
    bool tie = false;
    choice[p] = walks ? decide_one<true, true>(p, g, xy, heading, goal, nullptr, D, F, main_off,
                                               lo_row, hi_row, hi_off, y_lo, y_hi, beta, own, dirdot,
                                               &tie, ring, blocked)
                      : (uint8_t)0;
    decided += walks;
    ties += tie ? 1u : 0u;
  }
  __syncwarp();
  decided = __reduce_add_sync(0xffffffffu, decided);
  ties = __reduce_add_sync(0xffffffffu, ties);
  if (ctr && (threadIdx.x & 31) == 0 && decided) {
    atomicAdd(&ctr->decided, (unsigned long long)decided);
    if (ties) atomicAdd(&ctr->near_ties, (unsigned long long)ties);
  }
}

void launch_decide(int n, const int32_t* rec_id, const int32_t* bin_start, int b_lo, int b_hi,
                   const int2* xy, const uint8_t* heading, const uint8_t* goal,
                   const uint8_t* cell, const uint8_t* ocls, const int32_t* D, const float* F,
                   int main_off, int lo_row, int hi_row, int hi_off, int y_lo, int y_hi,
                   const Geo& g, float beta, const Tables& tb, uint8_t* choice, cudaStream_t s,
                   const WalkPeriods& wp, const Sizes& sz, const int32_t* occ,
                   Counters* ctr, int ring) {
  if (n <= 0 || b_hi <= b_lo) return;
  static int max_blocks = 0;
  if (!max_blocks) {
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    max_blocks = (nsm > 0 ? nsm : 1) * 8;  // two rounds of the 4 blocks of 256 an SM holds (64 registers)
  }
  if (sz.w) {
    const int blocks = cdiv(n, 256 / kQuad) < max_blocks ? cdiv(n, 256 / kQuad) : max_blocks;
    k_decide_sized<<<blocks, 256, 0, s>>>(rec_id, bin_start, b_lo, b_hi, xy, heading, goal, cell, D, F,
                                          main_off, lo_row, hi_row, hi_off, y_lo, y_hi, g, beta, tb.own,
                                          tb.dirdot, choice, wp, sz, occ, ctr, ring);
    return;
  }
  const int blocks = cdiv(n, 256) < max_blocks ? cdiv(n, 256) : max_blocks;
  k_decide<<<blocks, 256, 0, s>>>(rec_id, bin_start, b_lo, b_hi, xy, heading, goal, ocls, D, F, main_off,
                                  lo_row, hi_row, hi_off, y_lo, y_hi, g, beta, tb.own, tb.dirdot, choice,
                                  wp, ctr, ring);
}

// ------------------------------------------------------------ S4: vote
// The election of sub-job k-3 (vote_one), over the live pedestrians in bin
// order; and choice = won = 0 for the pedestrians that are not alive, which
// nothing else here reads or writes (a launch of its own for them, before the
// binning, took 2-3 us a tick).
__global__ void k_vote(int n, const int32_t* __restrict__ rec_id,
                       const int32_t* __restrict__ bin_start, int nbins,
                       const int2* __restrict__ xy, const uint8_t* __restrict__ alive,
                       uint8_t* __restrict__ choice, const int32_t* __restrict__ occ, Geo g,
                       uint64_t seed, Counters* ctr, uint8_t* __restrict__ won,
                       const int32_t* __restrict__ gid) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && !alive[i]) {
    choice[i] = 0;
    won[i] = 0;
  }
  if (i >= bin_start[nbins]) return;
  const int regs = vote_one(rec_id[i], 0, g, xy, choice, occ, seed, ctr->t, won, gid);
  if (regs > 2) atomicMax(&ctr->max_registrants, regs);
  if (regs > 8) atomicOr(&ctr->err, kErrEnroll);
}

__global__ void __launch_bounds__(256, 2)
    k_vote_sized(int n, const int32_t* __restrict__ rec_id, const int32_t* __restrict__ bin_start,
                 int nbins, const int2* __restrict__ xy, const uint8_t* __restrict__ alive,
                 uint8_t* __restrict__ choice, const int32_t* __restrict__ occ, Geo g, uint64_t seed,
                 Counters* ctr, uint8_t* __restrict__ won, Sizes sz) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) / kQuad, sub = threadIdx.x % kQuad;
  if (sub == 0 && i < n && !alive[i]) {
    choice[i] = 0;
    won[i] = 0;
  }
  const int p = i < bin_start[nbins] ? rec_id[i] : -1;
  bool win = false;
  int regs = 0;
  if (p >= 0)
    regs = vote_one_sized<kQuad>(p, g, xy, choice, occ, sz.w, sz.h, seed, ctr->t, sub, win);
#pragma unroll
  for (int o = 1; o < kQuad; o <<= 1) {
    regs = max(regs, __shfl_xor_sync(0xffffffffu, regs, o));
    win = win & __shfl_xor_sync(0xffffffffu, win, o);
  }
  if (p < 0 || sub) return;
  won[p] = win ? 1 : 0;
  if (regs > 2) atomicMax(&ctr->max_registrants, regs);
  if (regs > 8) atomicOr(&ctr->err, kErrEnroll);
}

void launch_vote(int n, const int32_t* rec_id, const int32_t* bin_start, const int2* xy,
                 const uint8_t* alive, uint8_t* choice, const int32_t* occ, const Geo& g,
                 uint64_t seed, Counters* ctr, uint8_t* won, cudaStream_t s, const Sizes& sz,
                 const int32_t* gid) {
  if (n <= 0) return;
  const int nbins = g.nbx * g.nby;
  if (sz.w)
    k_vote_sized<<<cdiv(n, 256 / kQuad), 256, 0, s>>>(n, rec_id, bin_start, nbins, xy, alive, choice, occ,
                                                      g, seed, ctr, won, sz);
  else
    k_vote<<<cdiv(n, 256), 256, 0, s>>>(n, rec_id, bin_start, nbins, xy, alive, choice, occ, g, seed, ctr,
                                        won, gid);
}

// ---------------------------------------------------------- S5: commit
__global__ void k_commit(const int32_t* __restrict__ rec_id, const int32_t* __restrict__ bin_start,
                         int nbins, int2* __restrict__ xy, uint8_t* __restrict__ alive,
                         uint8_t* __restrict__ heading, const uint8_t* __restrict__ choice,
                         const uint8_t* __restrict__ won, const uint8_t* __restrict__ cell,
                         int32_t* __restrict__ occ, uint8_t* __restrict__ ocls, Geo g,
                         Counters* ctr, Sizes sz) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, nrec = bin_start[nbins];
  const bool whole = !(ctr->err & kErrTimeout);  // else nobody moves, on a field that is not
  bool moved = false, left = false;
  if (i < nrec && whole) {
    if (sz.w)
      commit_one_sized(rec_id[i], g, xy, alive, heading, choice, won, cell, occ, ocls, sz.w, sz.h,
                       moved, left);
    else
      commit_one(rec_id[i], g, xy, alive, heading, choice, won, cell, occ, ocls, moved, left);
  }
  const unsigned nm = __popc(__ballot_sync(0xffffffffu, moved));
  const unsigned nl = __popc(__ballot_sync(0xffffffffu, left));
  if ((threadIdx.x & 31) == 0) {
    if (nm) atomicAdd(&ctr->moved, (unsigned long long)nm);
    if (nl) atomicAdd(&ctr->exited, (unsigned long long)nl);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && whole) ctr->t += 1;
}

void launch_commit(int n, const int32_t* rec_id, const int32_t* bin_start, int2* xy,
                   uint8_t* alive, uint8_t* heading, const uint8_t* choice, const uint8_t* won,
                   const uint8_t* cell, int32_t* occ, uint8_t* ocls, const Geo& g, Counters* ctr,
                   cudaStream_t s, const Sizes& sz) {
  const int blocks = n > 0 ? cdiv(n, 256) : 1;
  k_commit<<<blocks, 256, 0, s>>>(rec_id, bin_start, g.nbx * g.nby, xy, alive, heading, choice,
                                  won, cell, occ, ocls, g, ctr, sz);
}

// ------------------------------------------------- S3 - S5 in one block
// Decide, vote and commit of up to 1024 pedestrian slots, a thread each, with
// a block barrier where the single stages have a launch.  Bound by the chain of
// dependent reads (record, position, neighbourhood, rivals), which the stages
// have as well; with two launches less, the shorter binning and the early
// starts a tick of the 100 x 100 room with 200 pedestrians went from 32 to 21 us.
__global__ void __launch_bounds__(kMoveMaxPeds)
    k_move(int n, const int32_t* rec_id, const int32_t* bin_start, int nbins, int2* xy,
           uint8_t* alive, uint8_t* heading, const uint8_t* __restrict__ goal,
           const uint8_t* __restrict__ cell, int32_t* occ, uint8_t* ocls,
           const int32_t* __restrict__ D, const float* F, Geo g, float beta, uint64_t seed,
           const float* __restrict__ own, const float* __restrict__ dirdot, uint8_t* choice,
           uint8_t* won, Counters* ctr, WalkPeriods wp, const int32_t* __restrict__ gid) {
  // by pedestrian: the choices and wins of the stages before, not read back
  // from memory
  __shared__ uint8_t s_choice[kMoveMaxPeds], s_won[kMoveMaxPeds];
  tick_kernel_begin();
  const int i = threadIdx.x;
  const long long t = ctr->t;
  const bool whole = !(ctr->err & kErrTimeout);  // as in k_commit
  const int p = i < bin_start[nbins] ? rec_id[i] : -1;
  if (i < n && !alive[i]) {
    choice[i] = 0;
    won[i] = 0;
  }
  bool decided = false, tie = false;
  if (p >= 0) {
    decided = !(wp.period && t % wp.period[p] != wp.phase[p]);
    const uint8_t k = decided ? decide_one<true>(p, g, xy, heading, goal, ocls, D, F, 0, -1, -1, 0, 0, g.H,
                                                 beta, own, dirdot, &tie)
                              : (uint8_t)0;
    s_choice[p] = choice[p] = k;
  }
  __syncthreads();
  int regs = 0;
  if (p >= 0) {
    regs = vote_one(p, 0, g, xy, s_choice, occ, seed, t, s_won, gid);
    won[p] = s_won[p];
  }
  __syncthreads();
  bool moved = false, left = false;
  if (p >= 0 && whole) commit_one(p, g, xy, alive, heading, s_choice, s_won, cell, occ, ocls, moved, left);
  const unsigned nd = __popc(__ballot_sync(0xffffffffu, decided));
  const unsigned nt = __popc(__ballot_sync(0xffffffffu, tie));
  const unsigned nm = __popc(__ballot_sync(0xffffffffu, moved));
  const unsigned nl = __popc(__ballot_sync(0xffffffffu, left));
  regs = __reduce_max_sync(0xffffffffu, regs);
  if ((i & 31) == 0) {
    if (nd) atomicAdd(&ctr->decided, (unsigned long long)nd);
    if (nt) atomicAdd(&ctr->near_ties, (unsigned long long)nt);
    if (nm) atomicAdd(&ctr->moved, (unsigned long long)nm);
    if (nl) atomicAdd(&ctr->exited, (unsigned long long)nl);
    if (regs > 2) atomicMax(&ctr->max_registrants, regs);
    if (regs > 8) atomicOr(&ctr->err, kErrEnroll);
  }
  if (i == 0 && whole) ctr->t = t + 1;
}

void launch_move(int n, const int32_t* rec_id, const int32_t* bin_start, int2* xy, uint8_t* alive,
                 uint8_t* heading, const uint8_t* goal, const uint8_t* cell, int32_t* occ,
                 uint8_t* ocls, const int32_t* D, const float* F, const Geo& g, float beta,
                 uint64_t seed, const Tables& tb, uint8_t* choice, uint8_t* won, Counters* ctr,
                 cudaStream_t s, const WalkPeriods& wp, const int32_t* gid, bool early) {
  launch_tick_kernel(k_move, 1, 32 * cdiv(n, 32), 0, s, early, n, rec_id, bin_start, g.nbx * g.nby, xy, alive,
                     heading, goal, cell, occ, ocls, D, F, g, beta, seed, tb.own, tb.dirdot, choice, won, ctr,
                     wp, gid);
}

}  // namespace sfm
