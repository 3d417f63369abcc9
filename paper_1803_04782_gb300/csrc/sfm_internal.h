// sfm_internal.h -- device data layout and kernel launchers shared by the
// C-ABI host code (sfm_api.cu) and the kernels (sfm_kernels.cu, sfm_field.cu,
// sfm_batch.cu, sfm_surrogate.cu, sfm_noalloc.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sfm.h"
#include "sfm_limbs.h"

namespace sfm {

// streaming multiprocessors of the current device (its attribute, cached)
int device_sm_count();

constexpr int kFree = 0, kWall = 1, kExit = 2;
constexpr int32_t kDInf = 1 << 23;  // guidance distance of unreachable su (and WALL su, as exported)
// the guidance array's value on WALL su inside the library: it marks the su
// inadmissible, so a decision needs no read of the cell grid; exported as kDInf
constexpr int32_t kDWall = kDInf + 1;

// Three-component field gather (radius > 50): a CTA owns a 32 x 32 su tile;
// warp w owns rows 4w..4w+3 of it, lane l owns column l.
constexpr int kTile = 32;
// Rows of the band buffer beyond a band's: the row above the band and the
// next band's first tile row (the ring of run_tick's banded field)
constexpr int kBandExtraRows = kTile + 1;
constexpr int kFieldThreads = 256;
constexpr int kRowsPerThread = kTile / (kFieldThreads / 32);  // 4
constexpr int kStageCap = 2048;    // pedestrians staged in shared memory per chunk
constexpr int kMaxHaloBins = 128;  // bins touched by one tile's halo (checked)
constexpr int kBin = 32;           // side of a pedestrian bin (one warp column per su)
// class-table gather: a warp owns a 16 x 16 su footprint (half-warp h = rows
// 8h..8h+7, lane = column) or a 32 x 16 one (lane = column, 16 rows), 32
// warps per CTA.  The 4 heading-class tables sit in shared memory with row
// stride SP = 2 (mod 4), which puts the two half-warps' rows (8 SP apart) on
// disjoint banks.  A "wide" stride leaves >= 31 zero columns after each row's
// 2r + 1, so a lane outside a pedestrian's reach reads a zero and no lane
// needs a range test; the narrow stride 102 (radius 42..50, where wide tables
// would not fit in shared memory) keeps the test.
constexpr int kV2Rows = 8;         // rows per lane of the 16 x 16 footprint
constexpr int kFieldPadRows = 15;  // zero rows above/below each class table
constexpr int kV2Threads = 1024;
constexpr int kTableGuard = 32;    // zero floats in front of the tables in shared memory
constexpr int kNarrowStride = 102;
constexpr int kNumStrideClasses = 7;  // the wide strides 34, 50, ..., 114, then 102
constexpr int kMaxTableRadius = 50;   // largest radius of the class-table gather
constexpr int kMaxTableStride = 114;

constexpr int stride_of_class(int ci) { return ci < 6 ? 34 + 16 * ci : kNarrowStride; }
constexpr int class_of_stride(int sp) { return sp == kNarrowStride ? 6 : (sp - 34) / 16; }
constexpr bool wide_stride(int sp) { return sp != kNarrowStride; }

// Row stride of the class tables for radius r (0: beyond the gather).
constexpr int class_table_stride_of(int r) {
  if (r < 0 || r > kMaxTableRadius) return 0;
  for (int ci = 0; ci < 6; ++ci)
    if (stride_of_class(ci) >= 2 * r + 32) return stride_of_class(ci);
  return kNarrowStride;  // 2r + 1 <= 101
}
constexpr size_t class_table_floats_of(int r) {
  return class_table_stride_of(r)
             ? (size_t)4 * (2 * r + 1 + 2 * kFieldPadRows) * class_table_stride_of(r)
             : 0;
}
constexpr size_t max_class_table_floats(int rmax) {
  size_t m = 0;
  for (int r = 0; r <= rmax; ++r) m = class_table_floats_of(r) > m ? class_table_floats_of(r) : m;
  return m;
}
// shared memory of a gather CTA: guard, tables, per-warp record scratch
static_assert((kTableGuard + max_class_table_floats(kMaxTableRadius)) * 4 +
                      kV2Threads / 32 * 32 * 8 <= 227 * 1024 - 1024,
              "class tables exceed shared memory");

// Row-trimmed class-table gather (sfm_field3.cu): 32 x 32 su footprints,
// blocks of 16 columns x 16 rows.  Fifteen zero rows above and below each window
// (a visit reads whole blocks) and at least 15 zero columns after each row; the
// row stride is one of a few compile-time classes.  Radius 1..40.
constexpr int kField3PadRows = 15;
static_assert(kField3PadRows == kFieldPadRows, "one table kernel writes both layouts");
constexpr int kField3Threads = 896;
constexpr int kShape16x16 = 0, kShape32x16 = 1, kShape32x32 = 2;
constexpr int field3_stride(int r) {
  // >= 2r + 16: zero columns for the 16 of a block
  if (r < 1 || r > 40) return 0;
  for (int sp = 48; sp <= 112; sp += 32)
    if (sp >= 2 * r + 16) return sp;
  return 0;
}
constexpr size_t field3_table_floats(int r) {
  return field3_stride(r) ? (size_t)4 * (2 * r + 1 + 2 * kField3PadRows) * field3_stride(r) : 0;
}
constexpr size_t max_field3_table_floats() {
  size_t m = 0;
  for (int r = 0; r <= kMaxTableRadius; ++r)
    m = field3_table_floats(r) > m ? field3_table_floats(r) : m;
  return m;
}
static_assert((kTableGuard + max_field3_table_floats()) * 4 + kField3Threads / 32 * 32 * 8 <=
                  227 * 1024,
              "row-trimmed gather tables exceed shared memory");
// Dynamic shared memory that `k` may be launched with: a limit of the whole
// device context, so it is always the most that any launch of k asks for, never
// what one launch needs (which another host thread's launch, or another
// context's captured one, may exceed).
template <class K>
inline cudaError_t allow_shared(K* k, size_t most) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}
// ... of a gather's CTA of `threads` at any radius up to kMaxTableRadius
constexpr size_t max_gather_shared(int threads) {
  return (kTableGuard + max_class_table_floats(kMaxTableRadius)) * sizeof(float) +
         (size_t)threads * sizeof(int2);
}

// the row-trimmed footprint `shape` can run at radius r
constexpr bool field3_shape_ok(int shape, int r) {
  return field3_stride(r) != 0 && shape == kShape32x32;
}

// device error flags (sticky until read by a synchronising call)
enum : uint32_t {
  kErrPlaceConflict = 1u,  // two pedestrians on one su, or on a WALL/EXIT su
  kErrPlaceRange = 2u,     // off-lattice position or class > 8
  kErrEnroll = 4u,         // more than 8 registrants for one su (impossible by construction)
  kErrHalo = 8u,           // a tile's halo touched more bins than kMaxHaloBins
  kErrTimeout = 16u,       // a bounded device wait gave up; the crowd stays where it is
};

struct Counters {
  unsigned long long moved;
  unsigned long long exited;
  int max_registrants;
  uint32_t err;
  long long t;  // tick counter read by the vote and advanced by the commit
  // the class-table gather's footprint tickets: next ticket, CTAs done; zero
  // between launches (the launch's last CTA puts them back), so launches
  // sharing one context's counters run one at a time, in stream order
  unsigned int field_tickets[2];
  // decisions taken since the placement, and those among them whose best
  // and second-best admissible energies lie within 1e-5 of their magnitude
  // (near ties, which a differently rounded field may break the other way)
  unsigned long long decided;
  unsigned long long near_ties;
};

// Multi-su pedestrians (Sec. 2): pedestrian p occupies the w[p] x h[p]
// rectangle (odd sides) centred on its centre su; occ holds p on every su of
// it.  w == nullptr: every pedestrian is 1 x 1 (the plain model).
struct Sizes {
  const uint8_t* w = nullptr;
  const uint8_t* h = nullptr;
};
constexpr int kMaxPedSide = 15;  // largest width / height of a pedestrian

// Geometry and model constants passed by value to every kernel.
struct Geo {
  int W, H, px, py;
  int r;
  int nbx, nby;  // bins per row / column
  int opitch;    // row pitch (bytes) of the occupancy-class grid, a multiple of 128
};

// A far part added by the class-table gather's epilogue (the learned
// surrogate): F = (Fs + near sum) + scale * Y~, Y~ the bilinear interpolation
// of an Hc x Wc grid of s x s cells between cell centres (wrapped in periodic
// dimensions, clamped otherwise).  Y == nullptr: no far part.
struct FarPart {
  const float* Y = nullptr;
  int s = 1, Hc = 0, Wc = 0;
  float scale = 0.f;
  float inv_s = 1.f;  // 1 / s
};

struct Tables {
  const float* T0;      // (2r+1)^2: kP d^aP          (pedestrian, isotropic part)
  const float* TX;      // (2r+1)^2: kP d^aP gamma dx/d
  const float* TY;      // (2r+1)^2: kP d^aP gamma dy/d
  const float* KO;      // (2r+1)^2: kO d^aO
  const float* KE;      // (2r+1)^2: kE d^aE
  const float* own;     // [9 heading][9 move]: K_P(Delta_move; h)
  const float* dirdot;  // [9 goal][9 move]: Delta_move . u_goal
  const float2* hvec;   // [9]: unit heading vectors
  const float* CT;      // 4 padded heading-class tables of the v2 gather (or NULL)
  const float* CT3 = nullptr;  // the same in the row-trimmed gather's layout (or NULL)
  int shape = 0;        // class-table gather footprint: kShape16x16 .. kShape32x32
};

// Footprint of the class-table gather used when none has been tuned; W x H: the
// su of a launch (a band's rows).  32 x 32 from 16 an SM on (2432 on 152 SMs):
// up to there the 16 x 16 ones' four times as many make two rounds of the warps,
// then three.  16 x 16 over 32 x 32, a tick, at a pedestrian on every 50th su and
// at three on ten: r = 7 2401 footprints 0.95 and 0.83, 2500 1.02 and 0.96; r = 20
// 0.96 and 0.90, 1.06 and 1.04; r = 36 0.95 and 0.92, 1.03 and 1.05 (in bands of
// 2048 columns 2304 0.93 and 0.91, 2560 1.10 and 1.08 at r = 20; 1024 0.65 and
// 0.55).  Beyond the 32 x 32's radii, 32 x 16 at r = 45: 1250^2 (3160) 89 us
// against 112, but 1000^2 (2016) 78 and 68.
inline int default_field_shape(int r, int W, int H) {
  const int64_t nx = (W + 31) / 32, enough = 16 * (int64_t)device_sm_count() + 1;
  if (field3_stride(r)) return nx * ((H + 31) / 32) >= enough ? kShape32x32 : kShape16x16;
  return r > 30 && nx * ((H + 15) / 16) >= enough ? kShape32x16 : kShape16x16;
}

// ---- crowded lattices (sfm_product.cu) ----
// Largest radius of the tensor-core product: the sums over a full window of
// (2r + 1)^2 - 1 su stay below 2^24 with 23 bits and more to a table entry,
// and a plane and two table stages fit in shared memory.
constexpr int kProductMaxRadius = 44;
// A lattice is crowded, and its field summed by the product and not by a
// gather, from 9 pedestrians on 20 su.  The product is the faster way from
// far fewer (its time does not depend on the crowd: bins and field of a 1000 x
// 1000 lattice half full take 599 us by the gather at radius 38, 173 by the
// product, and at radius 3 66 and 39), but the two round differently,
// and in a run of many ticks one decision in 10^5 that falls the other way
// moves its neighbours: the line lies above the room, corridor and batch
// workloads (at most 2 su in 5), whose runs stay bit for bit what they were.
//
// A lattice no larger than the window either way is summed by the gather where
// that is clearly the faster way: its launch lasts as long as one footprint's
// chain of visits, 45 ns each in a context (107 beyond the wide strides' radii)
// and about twice that in a batch, which has to decide alike; the product's
// lasts as long as its start and a plane's products.  Ticks by product and
// gather at a density of 0.46: 20 x 20 at r = 38 62 and 20 us, 300 x 7 at r = 30
// 54 and 27, 3000 x 10 at r = 30 82 and 33; but 40 x 40 at r = 20 39 and 43, 64 x
// 64 at r = 38 69 and 84, at r = 44 73 and 211.
inline bool lattice_crowded(int W, int H, int r, int64_t n) {
  if (20 * n < 9 * (int64_t)W * H) return false;
  if (W > 2 * r && H > 2 * r) return true;
  const double seen = 2.0 * r + 16;  // su a side that a 16 x 16 footprint's window spans
  const double visits = (double)n / ((double)W * H) * (W < seen ? W : seen) * (H < seen ? H : seen);
  const double products = seen * ((2 * r + 8 + 15) / 16);  // a plane's, 128 clocks each
  return 25.0 + products * 128.0 / 2070.0 < 12.0 + visits * (r > 41 ? 0.2 : 0.1);
}

// Planes (and their tables): a crowd's presence and four heading axes; a cell
// grid's walls and exits, twice each (sfm_limbs.h)
constexpr int kCrowdPlanes = 5, kCellPlanes = 4;

// One lattice of a product launch: the source bytes (class grid or cell
// grid), the limb tables of its radius, and where the sums go.
struct ProductLattice {
  const uint8_t* src = nullptr;
  const float* Fs = nullptr;   // added to the sum (NULL: nothing)
  float* out = nullptr;        // W x H field (a launch may give its own)
  const uint8_t* tab = nullptr;
  int W = 0, H = 0, px = 0, py = 0, r = 0;
  int spitch = 0;  // bytes of a source row
  int ntx = 0;     // tiles a row
  float c0 = 0.f, c1 = 0.f;  // weights of the two limbs' sums
};
struct ProductArgs {
  ProductLattice one;                        // the lattice, when `lattices` is NULL
  const ProductLattice* lattices = nullptr;  // a batch's
  const int2* tiles = nullptr;               // a batch's tiles (lattice, tile), costly ones first
  int tile0 = 0, ntiles = 0;  // of `one`: set by launch_product from the rows to store
  int nch = kCrowdPlanes;     // or kCellPlanes
  // sums of split tiles, product_scratch_floats() a tile, zero between
  // launches (NULL: no tile is split)
  float* scratch = nullptr;
  int* tick = nullptr;        // arrivals of each split tile, zero between launches
  float* out = nullptr;       // overrides the lattice's own
  int out_row0 = 0, store_lo = 0, store_hi = 0, ring = 0;  // as launch_field's
  int plane_bytes = 0, stage_bytes = 0, nplanes = 0, nstages = 0, smem_bytes = 0;
  Counters* ctr = nullptr;
  int missing = 0;  // a test's: builders of planes that are waited for and do not exist
};
// Fixed-point scales of the limb tables (sfm_limbs.h).  false: the radius or the
// law's range over the window is beyond them.
bool product_crowd_scales(int r, const sfm_params& p, ProductScales* out);
bool product_cell_scales(int r, const sfm_params& p, ProductScales* out);
size_t product_table_bytes(int r, int nch);
void launch_limb_tables(int r, const sfm_params& p, const ProductScales& sc, int nch, uint8_t* tab,
                        cudaStream_t s);
void product_layout(int rmax, ProductArgs* a);  // shared-memory split for radii up to rmax
int product_tiles_x(int W);
int product_tiles_y(int H);
size_t product_scratch_floats();
cudaError_t launch_product(ProductArgs a, cudaStream_t s);

// ---- launchers (sfm_kernels.cu) ----
void launch_tables(int r, const sfm_params& p, float* T0, float* TX, float* TY, float* KO,
                   float* KE, float* own, float* dirdot, float2* hvec, cudaStream_t s);
// tmp: static_tmp_bytes() of device memory, 16-byte aligned, overwritten (limb
// tables).  ctr: error flags of a bounded wait.
size_t static_tmp_bytes(int r);
void launch_static_field(const Geo& g, const uint8_t* cell, const Tables& tb, const sfm_params& prm,
                         float* Fs, void* tmp, Counters* ctr, cudaStream_t s);
// Guidance distances; scratch: guidance_scratch_ints() ints of device memory,
// overwritten.  A bounded wait that runs out sets kErrTimeout in ctr.
size_t guidance_scratch_ints(const Geo& g);
// unfinished: a test's, with a tile that is never taken.
void launch_guidance(const Geo& g, const uint8_t* cell, int32_t* D, int* scratch, Counters* ctr,
                     cudaStream_t s, bool unfinished = false);
void launch_guidance_export(int32_t* D, size_t n, cudaStream_t s);
void launch_guidance_import(const uint8_t* cell, int32_t* D, size_t n, cudaStream_t s);

void launch_place_clear(int n, const int2* xy, const uint8_t* alive, const Geo& g, int32_t* occ,
                        uint8_t* ocls, cudaStream_t s, const Sizes& sz = Sizes());
void launch_place_scatter(int n, const int2* xy, const uint8_t* heading, const uint8_t* goal,
                          const uint8_t* alive, const uint8_t* cell, const Geo& g, int32_t* occ,
                          uint8_t* ocls, Counters* ctr, cudaStream_t s, const Sizes& sz = Sizes());
// placement of as many 1 x 1 pedestrians: grid entries of the changed ones only
// (from the previous state kept in *_prev, or read in place from the caller's
// device-visible buffers and staged in st_*)
void launch_place_direct(int n, const int2* src_xy, const uint8_t* src_h, const uint8_t* src_g,
                         const uint8_t* src_a, int2* st_xy, uint8_t* st_h, uint8_t* st_g,
                         uint8_t* st_a, int2* xy, uint8_t* heading, uint8_t* goal, uint8_t* alive,
                         uint8_t* choice, uint8_t* won, const uint8_t* cell, const Geo& g,
                         int32_t* occ, uint8_t* ocls, Counters* ctr, cudaStream_t s);
void launch_read_peds(int n, const int2* xy, const uint8_t* heading, const uint8_t* alive, int2* dxy,
                      uint8_t* dh, uint8_t* da, cudaStream_t s);
void launch_place_diff(int n, const int2* xy_prev, const uint8_t* alive_prev,
                       const uint8_t* heading_prev, const int2* xy, const uint8_t* heading,
                       const uint8_t* goal, const uint8_t* alive, const uint8_t* cell, const Geo& g,
                       int32_t* occ, uint8_t* ocls, Counters* ctr, cudaStream_t s);

// `early`: launched while the kernel before it in the stream still runs
// (programmatic dependent launch; launch_tick_kernel below).
void launch_scan(const int32_t* in, int32_t* out, int n, int32_t* block_tmp, cudaStream_t s);
int scan_tmp_elems(int n);
// Records of each bin in row-major su order, and the pedestrian id of each
// record (the per-pedestrian stages walk pedestrians in this spatial order),
// from the class grid or from the pedestrian list.  Returns the kernels launched.
int launch_bins_from_grid(const Geo& g, const uint8_t* ocls, const int32_t* occ, int32_t* count,
                          int32_t* start, int32_t* scan_tmp, uint32_t* rec, int32_t* rec_id,
                          cudaStream_t s, bool early = false);
int launch_bins_from_peds(const Geo& g, int n, const int2* xy, const uint8_t* alive,
                          const uint8_t* heading, int32_t* count, int32_t* start,
                          int32_t* scan_tmp, int32_t* slot, uint32_t* key, uint32_t* rec,
                          int32_t* rec_id, cudaStream_t s);
// lattices of at most this many bins: binned from the class grid by two
// launches instead of a count, a scan and a fill
constexpr int kBinsPrefix = 4096;
void launch_reset_counters(Counters* ctr, cudaStream_t s);

// Field gather; stores lattice rows y in [store_lo, store_hi) at
// out[(y - out_row0) * W + x].  Every su is summed in the same order whatever
// the row range, so banded and unbanded passes agree bit for bit.
// the three-component gather (radius > 50), called by launch_field
cudaError_t launch_field_v1(const Geo& g, const int32_t* bin_start, const uint32_t* rec, const Tables& tb,
                     const float* Fs, float* out, int out_row0, int store_lo, int store_hi,
                     Counters* ctr, cudaStream_t s);
// ring > 0: out is a ring of `ring` rows, row y stored at (y - out_row0) mod
// ring (y - out_row0 < 2 ring); only the row-trimmed gather takes one
// (launch_field_v3 returns false otherwise)
// returns the launch's status: a tick stops where its field was refused
cudaError_t launch_field(const Geo& g, const int32_t* bin_start, const uint32_t* rec, const Tables& tb,
                  const float* Fs, float* out, int out_row0, int store_lo, int store_hi,
                  Counters* ctr, cudaStream_t s, const FarPart& far = FarPart(), int ring = 0,
                  bool early = false);
int class_table_stride(int r);
size_t class_table_floats(int r);
// taper_in < r: entries weighted by 1 up to Euclidean distance taper_in and
// a raised cosine down to 0 at r (the surrogate's near part); default none
void launch_class_tables(int r, const sfm_params& p, float* T, cudaStream_t s,
                         double taper_in = 1e30);
// the row-trimmed gather (sfm_field3.cu): false (nothing launched) when the
// radius, the tables or the footprint do not select it
bool launch_field_v3(const Geo& g, const int32_t* bin_start, const uint32_t* rec,
                     const Tables& tb, const float* Fs, float* out, int out_row0, int store_lo,
                     int store_hi, unsigned int* tickets, bool sorted, cudaStream_t s, int ring,
                     bool early, cudaError_t* launched);
void launch_class_tables3(int r, const sfm_params& p, float* T, cudaStream_t s);

// The per-pedestrian stages visit the live pedestrians of bins [b_lo, b_hi)
// through rec_id (n bounds the launch).  F rows: lattice rows [y_lo, y_hi) at
// buffer row (y - y_lo + main_off), lattice row lo_row at buffer row 0 and
// hi_row at buffer row hi_off.
// Walk periods (Sec. 2): pedestrian p may move only on ticks t with
// t mod period[p] = phase[p] (t = ctr->t, read on the device); period ==
// nullptr: every pedestrian is active.
struct WalkPeriods {
  const uint8_t* period = nullptr;
  const uint8_t* phase = nullptr;
  const Counters* ctr = nullptr;
};

void launch_decide(int n, const int32_t* rec_id, const int32_t* bin_start, int b_lo, int b_hi,
                   const int2* xy, const uint8_t* heading, const uint8_t* goal,
                   const uint8_t* cell, const uint8_t* ocls, const int32_t* D, const float* F,
                   int main_off, int lo_row, int hi_row, int hi_off, int y_lo, int y_hi,
                   const Geo& g, float beta, const Tables& tb, uint8_t* choice, cudaStream_t s,
                   const WalkPeriods& wp = WalkPeriods(), const Sizes& sz = Sizes(),
                   const int32_t* occ = nullptr, Counters* ctr = nullptr, int ring = 0);
// The vote also sets choice = won = 0 for pedestrians that are not alive.
void launch_vote(int n, const int32_t* rec_id, const int32_t* bin_start, const int2* xy,
                 const uint8_t* alive, uint8_t* choice, const int32_t* occ, const Geo& g,
                 uint64_t seed, Counters* ctr, uint8_t* won, cudaStream_t s,
                 const Sizes& sz = Sizes(), const int32_t* gid = nullptr);
void launch_commit(int n, const int32_t* rec_id, const int32_t* bin_start, int2* xy,
                   uint8_t* alive, uint8_t* heading, const uint8_t* choice, const uint8_t* won,
                   const uint8_t* cell, int32_t* occ, uint8_t* ocls, const Geo& g, Counters* ctr,
                   cudaStream_t s, const Sizes& sz = Sizes());
// Decide, vote and commit of a whole lattice (F: its rows) of n <=
// kMoveMaxPeds pedestrian slots of 1 x 1 su in one launch.
constexpr int kMoveMaxPeds = 1024;
// One block saves two launches, but its reads are those of one SM.  A tick by it
// and by three launches: 256 pedestrians on 300 x 300 19.8 and 22.6 us, 512 23.3
// both, 1024 31.1 and 23.5; 384 on 2000 x 2000 32.0 and 31.9; where many share a
// su's surroundings later: 768 on 100 x 100 27.8 and 28.6, 1024 29.6 and 27.4, on
// 40 x 40 45.7 and 49.0.  Beside a gather of large tables the block has little
// L1: 617 x 477 at r = 45, 128 pedestrians 24.1 and 25.3, 200 27.8 and 26.3, 256 31.0
// and 27.2 (at r = 30 22.5 and 25.5).  Rectangles read their whole rings: always slower.
inline bool move_in_one(int W, int H, int r, int n, bool sized) {
  const int64_t su = (int64_t)W * H;
  return !sized && n > 0 && n <= (r > 33 ? 192 : su > 128 * 128 ? 384 : su > 64 * 64 ? 768 : kMoveMaxPeds);
}
void launch_move(int n, const int32_t* rec_id, const int32_t* bin_start, int2* xy, uint8_t* alive,
                 uint8_t* heading, const uint8_t* goal, const uint8_t* cell, int32_t* occ,
                 uint8_t* ocls, const int32_t* D, const float* F, const Geo& g, float beta,
                 uint64_t seed, const Tables& tb, uint8_t* choice, uint8_t* won, Counters* ctr,
                 cudaStream_t s, const WalkPeriods& wp, const int32_t* gid, bool early);

// The same stages of a whole lattice of 1 x 1 pedestrians, a block a bin
// (sfm_move.cu): the choice and the win are kept in the records as well.
// From a pedestrian on every tenth su on: a tick at r = 3 of 2048 x 2048 takes
// 142 us by bins against 150 by pedestrian at a density of 1/8, but 100 against
// 93 at 1/16 (1000 x 1000: 52 and 54, 40 and 41).
inline bool move_by_bins(int W, int H, int n) { return (int64_t)n * 10 >= (int64_t)W * H; }
void launch_decide_bins(const Geo& g, const int32_t* bin_start, uint32_t* rec, const int32_t* rec_id,
                        const uint8_t* goal, const uint8_t* ocls, const int32_t* D, const float* F,
                        float beta, const Tables& tb, uint8_t* choice, cudaStream_t s,
                        const WalkPeriods& wp, Counters* ctr);
void launch_vote_bins(int n, const Geo& g, const int32_t* bin_start, uint32_t* rec,
                      const int32_t* rec_id, const uint8_t* alive, uint8_t* choice, const int32_t* occ,
                      uint64_t seed, Counters* ctr, uint8_t* won, cudaStream_t s, const int32_t* gid);
void launch_commit_bins(const Geo& g, const int32_t* bin_start, const uint32_t* rec,
                        const int32_t* rec_id, int2* xy, uint8_t* alive, uint8_t* heading,
                        const uint8_t* cell, int32_t* occ, uint8_t* ocls, Counters* ctr,
                        cudaStream_t s);

// k<<<grid, block, smem, s>>>(args...), with `early` as a programmatic
// dependent launch: its blocks start once every block of the kernel before it
// has called tick_kernel_begin() (or ended), and its own tick_kernel_begin()
// waits for that kernel's completion.  Every thread of a kernel launched so
// calls it before it reads or writes anything that changes from tick to tick,
// so a kernel that has passed it has all the work before it behind it.
template <class... P, class... A>
inline cudaError_t launch_tick_kernel(void (*k)(P...), int grid, int block, size_t smem,
                                      cudaStream_t s, bool early, const A&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)grid);
  c.blockDim = dim3((unsigned)block);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&c, k, P(args)...);
}

}  // namespace sfm
