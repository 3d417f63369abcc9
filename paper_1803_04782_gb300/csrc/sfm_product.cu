// sfm_product.cu -- the field of a crowded lattice as a matrix product on the
// 5th-generation tensor cores (S2, k-5 of the paper's Alg. 1): where at least
// 9 of 20 su hold a pedestrian, one table word read from shared memory for
// every (su, pedestrian) pair costs far more than a dense convolution of the
// occupancy with the kernel window.
//
// Arithmetic.  A crowd is five planes of {-1, 0, +1}: occupancy and the four
// heading axes (E-W, N-S, NE-SW, NW-SE), and K_P is the sum of five window
// tables, one a plane.  Each table entry is held in fixed point as two
// integers of FP16 ("limbs"): T = L0 / s0 + L1 / (s0 s1) (sfm_limbs.h).
// Products with {-1, 0, +1} and every partial sum are integers below 2^24 in
// magnitude, so the FP32 accumulators hold them exactly: a sum is the same
// whatever the order, the tile or the split, and is rounded once, when the
// limbs are joined.  Against 64 bits the field of a periodic 1000 x 1000
// lattice half full at radius 38 is off by 3.0e-8 (2-norm), the gathers' FP32
// sums by 8.6e-7.  A cell grid (the static field) is its walls and exits, two
// planes each.
//
// The product.  A tile is 64 x 256 su = 8 x 16 blocks of 8 x 16 su.  D[m][n]
// = sum_k A[m][k] B[n][k]: m a block, n a su of the block and a limb, k a su
// of the block's window, 2r + 16 rows of 16 C >= 2r + 8 columns.  A is the
// plane itself, FP16 in shared memory: 8 blocks side by side are 64
// consecutive su, one 128-byte core matrix, and the next 8 columns of the
// window start 16 bytes on (the no-swizzle descriptor's offset between the
// halves of K), so no im2col copy exists.  B is Toeplitz in y: stored by the
// difference j = (su row) - (window row), so a window row is a shift of the
// start address.  Both limbs ride in one M = 128, N = 256 product, which
// reads A once and keeps the pipe busy for 128 clocks, so the tensor pipe
// bounds a launch with many tiles.  The 1000 x 1000 lattice has 64 tiles for
// 152 SMs: at radius 38 their planes are split over two CTAs a tile (the pipe
// is busy for 69 % of the SMs' active clocks; the longest CTA has three planes,
// the mean 2.1), at radius 3 a tile is one CTA's and latency bounds it (21 %;
// six windows' reads, 220 products).  Measured there (ncu, cold): 168 us at
// radius 38 and 31 at radius 3; bins and field together took 599 and 66 us by
// the gathers and take 173 and 39; a plane rebuilt from memory each time took
// 233 and 63.
//
// Roles of a CTA, one an SM: warp 0 copies tables (one plane's 16 window
// columns a stage), warp 1 issues the products, the others build planes from
// the class grid and write results.  Every wait is bounded (about a second);
// one that runs out raises kErrTimeout, the roles run through without
// waiting, and what is in flight is waited for before TMEM is freed.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "sfm_umma.cuh"

namespace sfm {

namespace {

constexpr int kTW = 64, kTH = 256;     // su of a tile
constexpr int kFirst = 4;              // warps 4.. build planes and write results
constexpr int kWorkers = 16;
constexpr int kProdThreads = 32 * (kFirst + kWorkers);
constexpr int kHeadBytes = 256;        // mbarriers and words
constexpr size_t kScratchFloats = (size_t)kTW * kTH * 2;  // a split tile's sums
constexpr int kSmem = 227 * 1024;

__host__ __device__ constexpr int chunks_of(int r) { return (2 * r + 8 + 15) / 16; }
__host__ __device__ constexpr int pitch_of(int r) { return (kTW - 8 + 16 * chunks_of(r)) * 2; }
__host__ __device__ constexpr int rows_of(int r) { return kTH + 2 * r; }
__host__ __device__ constexpr int plane_bytes_of(int r) { return (rows_of(r) * pitch_of(r) + 127) / 128 * 128; }
__host__ __device__ constexpr int stage_bytes_of(int r) { return (2 * r + 31) * 512; }
// chunks of 8 su of a plane a worker thread holds, at most
constexpr int kMaxChunks =
    (rows_of(kProductMaxRadius) * pitch_of(kProductMaxRadius) / 16 + kWorkers * 32 - 1) / (kWorkers * 32);
static_assert(pitch_of(kProductMaxRadius) % 16 == 0, "a row is a whole number of chunks");
static_assert(kTW * 2 == 128, "8 blocks side by side are one core matrix");
static_assert(kWorkers % 4 == 0, "the workers cover the four TMEM lane quarters alike");
static_assert(kHeadBytes + plane_bytes_of(kProductMaxRadius) + 2 * stage_bytes_of(kProductMaxRadius) <= kSmem,
              "a plane and two table stages must fit");

// kind::f16: FP32 accumulators, FP16 operands, M = 128, N = 256
constexpr uint32_t kIdesc = (1u << 4) | ((256u >> 3) << 17) | ((128u >> 4) << 24);

// 8 source bytes at columns x .. x + 7 of a row of W (0 outside a closed lattice)
__device__ __forceinline__ uint2 source8(const uint8_t* __restrict__ row, int x, int W, int px) {
  if (px && (x < 0 || x >= W)) {
    x %= W;
    if (x < 0) x += W;
  }
  if (x >= 0 && x + 8 <= W) {
    // the aligned words that hold the 8 bytes (each holds at least one of them)
    const uintptr_t p = reinterpret_cast<uintptr_t>(row + x);
    const uint32_t* q = reinterpret_cast<const uint32_t*>(p & ~(uintptr_t)3);
    const int sh = (int)(p & 3) * 8;
    const uint32_t a = __ldg(q), b = __ldg(q + 1), c = sh ? __ldg(q + 2) : 0u;
    return make_uint2(__funnelshift_r(a, b, sh), __funnelshift_r(b, c, sh));
  }
  // across an edge: byte by byte, all reads in flight
  uint32_t v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    int xx = x + e;
    if (px) xx = xx < W ? xx : (xx - W < W ? xx - W : xx % W);
    v[e] = xx >= 0 && xx < W ? row[xx] : 0u;
  }
  return make_uint2(v[0] | v[1] << 8 | v[2] << 16 | v[3] << 24, v[4] | v[5] << 8 | v[6] << 16 | v[7] << 24);
}

// Four source bytes as four FP16 of +1 (bytes that equal `pos`, or with pos 0
// all but 0), -1 (those that equal `neg`) or 0.
__device__ __forceinline__ uint2 signs4(uint32_t v, uint32_t pos, uint32_t neg) {
  const uint32_t p = pos ? __vcmpeq4(v, pos) : __vcmpne4(v, 0u);
  uint32_t hi = p & 0x3C3C3C3Cu;                            // the high byte of 1.0
  if (neg) hi |= __vcmpeq4(v, neg) & 0xBCBCBCBCu;           // and of -1.0
  return make_uint2(__byte_perm(hi, 0u, 0x1404), __byte_perm(hi, 0u, 0x3424));
}

// Slices that `rest` (< G) tiles are split into: whichever count makes least
// of the clocks of a CTA's share -- `plane` a plane, 35 000 for the sums that
// go through memory (clock64 on the 1000 x 1000 lattice: 8 000 to add them,
// 3 000 for the arrival, 22 000 for the last CTA to join them).
__device__ __forceinline__ int slices_of(int rest, int nch, int G, int plane) {
  int S = 1, best = nch * plane * ((rest + G - 1) / G);
  for (int s = 2; s <= nch; ++s) {
    const int c = ((nch + s - 1) / s * plane + 11000) * ((rest * s + G - 1) / G) + 24000;
    if (c < best) {
      best = c;
      S = s;
    }
  }
  return S;
}

__global__ void __launch_bounds__(kProdThreads, 1) k_product(const __grid_constant__ ProductArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, me = blockIdx.x;
  const uint32_t bar = (uint32_t)__cvta_generic_to_shared(smem);
  // mbarriers: stage full / empty (up to 8 stages), plane full / empty (2),
  // accumulators full / empty (2); then the words below
  auto sfull = [&](int i) { return bar + 8 * i; };
  auto sempty = [&](int i) { return bar + 64 + 8 * i; };
  auto pfull = [&](int i) { return bar + 128 + 8 * i; };
  auto pempty = [&](int i) { return bar + 144 + 8 * i; };
  auto afull = [&](int i) { return bar + 160 + 8 * i; };
  auto aempty = [&](int i) { return bar + 176 + 8 * i; };
  volatile int* word = reinterpret_cast<volatile int*>(smem + 192);
  // word[0] TMEM address, [1], [2] planes that hold something (their sequence
  // number), [3], [4] accumulator sets that were written, [5] copies issued,
  // [6] stages handed back by the issuer, [7] last arrival of a split tile
  const uint32_t plane0 = bar + kHeadBytes;
  const uint32_t stage0 = plane0 + (uint32_t)(a.nplanes * a.plane_bytes);
  if (tid == 0) {
    for (int i = 0; i < a.nstages; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(sfull(i)));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(sempty(i)));
    }
    for (int i = 0; i < 2; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(pfull(i)), "r"(kWorkers + a.missing));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(pempty(i)));
      // the issuer's own arrival (it publishes word[3 + i]) and its commit
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 2;\n" ::"r"(afull(i)));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(aempty(i)), "r"(kWorkers));
    }
    for (int i = 1; i < 8; ++i) word[i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(bar + 192));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = (uint32_t)word[0];

  // Units.  Whole multiples of G tiles go out one a CTA (back and forth, so a
  // cost-sorted list balances); the planes of the rest are split over the
  // CTAs that would idle, the integer sums added up in `scratch` and joined
  // by the last CTA of the tile.
  const int nch = a.nch, T = a.ntiles, whole = T / G, rest = T - whole * G;
  // the clocks of a plane of the rest's first tile, the largest radius in it:
  // 128 a product, and its plane to build (by the last one's, a batch's few
  // tiles of radius 44 beside others of 3 were not split and took 190 us)
  int S;
  {
    const int r = a.lattices ? a.lattices[a.tiles[rest ? whole * G : 0].x].r : a.one.r;
    S = a.scratch ? slices_of(rest, nch, G, (2 * r + 16) * chunks_of(r) * 128 + 2000) : 1;
  }
  const int units = whole + (rest * S) / G + (me < rest * S % G ? 1 : 0);
  struct Unit {
    int rank, slice, c0, c1;  // tile, its split slot (-1: not split), planes [c0, c1)
  };
  auto unit = [&](int i) {
    Unit u;
    u.slice = -1;
    u.c0 = 0;
    u.c1 = nch;
    if (i < whole) {
      u.rank = i * G + ((i & 1) ? G - 1 - me : me);
    } else {
      const int v = (i - whole) * G + me, s = v % S;
      u.rank = whole * G + v / S;
      if (S > 1) {
        u.slice = v / S;
        u.c0 = s * nch / S;
        u.c1 = (s + 1) * nch / S;
      }
    }
    return u;
  };
  auto lattice = [&](int rank, int& tx, int& ty) -> const ProductLattice& {
    const int2 lt = a.tiles ? a.tiles[rank] : make_int2(0, a.tile0 + rank);
    const ProductLattice& l = a.lattices ? a.lattices[lt.x] : a.one;
    tx = lt.y % l.ntx;
    ty = lt.y / l.ntx;
    return l;
  };

  bool failed = false;
  auto wait = [&](uint32_t b, uint32_t parity) {
    if (!failed && !mbar_wait(b, parity)) failed = true;
  };
  const int nplanes = a.nplanes, nstages = a.nstages;
  const uint32_t plane_bytes = (uint32_t)a.plane_bytes, stage_bytes = (uint32_t)a.stage_bytes;
  int n_stage = 0, n_plane = 0, n_unit = 0;  // running counts, each role its own
  if (warp == 0) {
    if (lane == 0) {
      for (int i = 0; i < units && !failed; ++i) {
        const Unit u = unit(i);
        int tx, ty;
        const ProductLattice& l = lattice(u.rank, tx, ty);
        const int C = chunks_of(l.r);
        const uint8_t* const tab = l.tab;
        const uint32_t bytes = (uint32_t)stage_bytes_of(l.r);
        for (int k = u.c0 * C; k < u.c1 * C; ++k, ++n_stage) {
          const int st = n_stage % nstages;
          wait(sempty(st), ((uint32_t)(n_stage / nstages) & 1u) ^ 1u);
          if (failed) break;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(sfull(st)), "r"(bytes)
                       : "memory");
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                  stage0 + (uint32_t)st * stage_bytes),
              "l"(tab + (size_t)k * bytes), "r"(bytes), "r"(sfull(st))
              : "memory");
          word[5] = n_stage + 1;
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      for (int i = 0; i < units && !failed; ++i, ++n_unit) {
        const Unit u = unit(i);
        int tx, ty;
        const int r = lattice(u.rank, tx, ty).r;
        const int C = chunks_of(r), P = pitch_of(r), K = 2 * r + 16;
        const int set = n_unit & 1;
        const uint32_t d = tmem + (uint32_t)(set * 256);
        uint32_t acc = 0;
        wait(aempty(set), ((uint32_t)(n_unit >> 1) & 1u) ^ 1u);
        for (int ch = u.c0; ch < u.c1 && !failed; ++ch, ++n_plane) {
          const int pb = nplanes == 2 ? n_plane & 1 : 0;
          wait(pfull(pb), (uint32_t)(n_plane / nplanes) & 1u);
          const bool some = word[1 + pb] == n_plane + 1;  // an empty plane adds nothing
          for (int c = 0; c < C && !failed; ++c, ++n_stage) {
            const int st = n_stage % nstages;
            wait(sfull(st), (uint32_t)(n_stage / nstages) & 1u);
            if (failed) break;
            if (some) {
              asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
              uint64_t ad = umma_desc(plane0 + (uint32_t)pb * plane_bytes + (uint32_t)(c * 32), 16,
                                    (uint32_t)(16 * P));
              uint64_t bd = umma_desc(stage0 + (uint32_t)st * stage_bytes + (uint32_t)((K - 1) * 512), 128, 256);
              for (int ky = 0; ky < K; ++ky) {
                umma_f16(d, ad, bd, kIdesc, acc);
                acc = 1;
                ad += (uint64_t)(P >> 4);
                bd -= (uint64_t)(512 >> 4);
              }
              umma_commit(sempty(st));
            } else {
              mbar_arrive(sempty(st));
            }
            word[6] = n_stage + 1;
          }
          if (some)
            umma_commit(pempty(pb));
          else
            mbar_arrive(pempty(pb));
        }
        word[3 + set] = (int)acc;
        mbar_arrive(afull(set));
        if (acc)
          umma_commit(afull(set));
        else
          mbar_arrive(afull(set));
      }
    }
    __syncwarp();
  } else if (warp >= kFirst) {
    const int w = warp - kFirst;
    // A unit's source bytes stay in registers for all its planes: chunk t of
    // a plane (8 su, 16 bytes of FP16; a row is a whole number of them) is
    // worker thread t mod 512's, so a plane costs conversions and stores only.
    uint2 raw[kMaxChunks];
    int nraw = 0;
    auto fetch = [&](const Unit& u) {
      int tx, ty;
      const ProductLattice& l = lattice(u.rank, tx, ty);
      const uint8_t* const src = l.src;
      const int W = l.W, H = l.H, px = l.px, py = l.py, pitch = l.spitch, r = l.r;
      const int x0 = tx * kTW - r, y0 = ty * kTH - r;
      const int per = pitch_of(r) / 16, need = kTW + 2 * r, n = rows_of(r) * per;
      const int me = w * 32 + lane, di = kWorkers * 32 / per, dq = kWorkers * 32 % per;
      int row = me / per, q = me % per;
      nraw = (n - me + kWorkers * 32 - 1) / (kWorkers * 32);
#pragma unroll
      for (int e = 0; e < kMaxChunks; ++e) {
        raw[e] = make_uint2(0u, 0u);
        int y;
        if (e < nraw && 8 * q < need && wrap_coord(y0 + row, H, py, y))
          raw[e] = source8(src + (size_t)y * pitch, x0 + 8 * q, W, px);
        row += di;
        q += dq;
        if (q >= per) {
          q -= per;
          ++row;
        }
      }
    };
    auto build = [&](int ch) {
      const int pb = nplanes == 2 ? n_plane & 1 : 0;
      wait(pempty(pb), ((uint32_t)(n_plane / nplanes) & 1u) ^ 1u);
      // class values 1 + heading: E 2, NE 3, N 4, NW 5, then W 6, SW 7, S 8,
      // SE 9; a cell grid's 1 (wall) and 2 (exit) are two planes each
      const bool cells = nch == kCellPlanes;
      const int v = cells ? 1 + (ch >> 1) : (ch == 0 ? 0 : (ch == 1 ? 2 : (ch == 2 ? 4 : (ch == 3 ? 3 : 5))));
      const uint32_t pos = (uint32_t)v * 0x01010101u;
      const uint32_t neg = cells || ch == 0 ? 0u : (uint32_t)(v + 4) * 0x01010101u;
      const uint32_t dst = plane0 + (uint32_t)pb * plane_bytes + (uint32_t)(w * 32 + lane) * 16;
      uint32_t any = 0;
#pragma unroll
      for (int e = 0; e < kMaxChunks; ++e) {
        if (e < nraw) {
          const uint2 a2 = signs4(raw[e].x, pos, neg), b2 = signs4(raw[e].y, pos, neg);
          any |= a2.x | a2.y | b2.x | b2.y;
          asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(dst + (uint32_t)(e * kWorkers * 512)),
                       "r"(a2.x), "r"(a2.y), "r"(b2.x), "r"(b2.y)
                       : "memory");
        }
      }
      if (__any_sync(0xffffffffu, any != 0) && lane == 0) word[1 + pb] = n_plane + 1;
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(pfull(pb));
      ++n_plane;
    };
    // this thread's block (bx, by): lane m of the accumulators
    const int quad = warp & 3, by = 4 * quad + (lane >> 3), bx = lane & 7;
    auto finish = [&](const Unit& u) {
      const int set = n_unit & 1;
      int tx, ty;
      const ProductLattice& l = lattice(u.rank, tx, ty);
      const int x = tx * kTW + 8 * bx, yb = ty * kTH + 16 * by, W = l.W;
      const int y_lo = max(yb, a.store_lo), y_hi = x < W ? min(l.H, a.store_hi) : 0;
      const float c0 = l.c0, c1 = l.c1;
      const float* const Fs = l.Fs;
      float* const out = a.out ? a.out : l.out;
      // the static field of this thread's su of a row (16-byte accesses where
      // the rows' alignment allows), and the row's results
      const bool wide = (W & 3) == 0 && x + 8 <= W &&
                        ((reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(Fs)) & 15) == 0;
      auto base = [&](int y, float (&f)[8]) {
#pragma unroll
        for (int e = 0; e < 8; ++e) f[e] = 0.f;
        if (!Fs || y < y_lo || y >= y_hi) return;
        const float* p = Fs + (size_t)y * W + x;
        if (wide) {
          const float4 lo = __ldg(reinterpret_cast<const float4*>(p));
          const float4 hi = __ldg(reinterpret_cast<const float4*>(p) + 1);
          f[0] = lo.x, f[1] = lo.y, f[2] = lo.z, f[3] = lo.w;
          f[4] = hi.x, f[5] = hi.y, f[6] = hi.z, f[7] = hi.w;
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (x + e < W) f[e] = __ldg(p + e);
        }
      };
      auto emit = [&](int y, const float (&f)[8], const float (&v)[8]) {
        int row = y - a.out_row0;
        if (a.ring && row >= a.ring) row -= a.ring;
        float* o = out + (size_t)row * W + x;
        if (wide) {
          reinterpret_cast<float4*>(o)[0] = make_float4(f[0] + v[0], f[1] + v[1], f[2] + v[2], f[3] + v[3]);
          reinterpret_cast<float4*>(o)[1] = make_float4(f[4] + v[4], f[5] + v[5], f[6] + v[6], f[7] + v[7]);
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (x + e < W) o[e] = f[e] + v[e];
        }
      };
      float* const part =
          u.slice < 0 ? nullptr : a.scratch + (size_t)u.slice * kScratchFloats + (size_t)(8 * by + bx) * 16;
      constexpr int kRowsEach = 16 / (kWorkers / 4);
      float f[2][8];  // the next row's static field is read ahead
      if (!part) base(yb + (w >> 2), f[0]);
      wait(afull(set), (uint32_t)(n_unit >> 1) & 1u);
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const bool written = word[3 + set] != 0;
#pragma unroll
      for (int t = 0; t < kRowsEach; ++t) {
        const int ny = (w >> 2) + t * (kWorkers / 4);
        if (!part && t + 1 < kRowsEach) base(yb + ny + kWorkers / 4, f[(t + 1) & 1]);
        uint32_t v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = 0u;
        if (written) {
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
              "%12, %13, %14, %15}, [%16];\n"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
                "=r"(v[14]), "=r"(v[15])
              : "r"(tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(set * 256 + ny * 16)));
          asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        }
        const int y = yb + ny;
        const bool here = y >= y_lo && y < y_hi;
        if (here && !part) {
          float o[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) o[e] = fmaf(__uint_as_float(v[e]), c0, __uint_as_float(v[8 + e]) * c1);
          emit(y, f[t & 1], o);
        } else if (here && written) {
          float* p = part + (size_t)ny * 128 * 16;
#pragma unroll
          for (int e = 0; e < 16; e += 4)
            asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(p + e),
                         "f"(__uint_as_float(v[e])), "f"(__uint_as_float(v[e + 1])),
                         "f"(__uint_as_float(v[e + 2])), "f"(__uint_as_float(v[e + 3]))
                         : "memory");
        }
        __syncwarp();  // the next tcgen05.ld takes the whole warp
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(aempty(set));
      if (part) {
        // the last slice of the tile joins the limbs and leaves zeros
        __threadfence();
        asm volatile("bar.sync 1, %0;\n" ::"n"(kWorkers * 32) : "memory");
        if (w == 0 && lane == 0) {
          int* tick = a.tick + u.slice;
          const int last = atomicAdd(tick, 1) == S - 1;
          if (last) *tick = 0;
          __threadfence();
          word[7] = last;
        }
        asm volatile("bar.sync 1, %0;\n" ::"n"(kWorkers * 32) : "memory");
        if (word[7]) {
          __threadfence();
          // two rows' sums and static field in flight together
#pragma unroll
          for (int t = 0; t < kRowsEach; t += 2) {
            float4 h[2][4];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const int ny = (w >> 2) + (t + k) * (kWorkers / 4), y = yb + ny;
              const float4* p = reinterpret_cast<const float4*>(part + (size_t)ny * 128 * 16);
#pragma unroll
              for (int e = 0; e < 4; ++e)
                h[k][e] = y >= y_lo && y < y_hi ? __ldcg(p + e) : make_float4(0.f, 0.f, 0.f, 0.f);
              base(y, f[k]);
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const int ny = (w >> 2) + (t + k) * (kWorkers / 4), y = yb + ny;
              if (y < y_lo || y >= y_hi) continue;
              float4* p = reinterpret_cast<float4*>(part + (size_t)ny * 128 * 16);
#pragma unroll
              for (int e = 0; e < 4; ++e) p[e] = make_float4(0.f, 0.f, 0.f, 0.f);
              const float4 h0 = h[k][0], h1 = h[k][1], l0 = h[k][2], l1 = h[k][3];
              const float o[8] = {fmaf(h0.x, c0, l0.x * c1), fmaf(h0.y, c0, l0.y * c1),
                                  fmaf(h0.z, c0, l0.z * c1), fmaf(h0.w, c0, l0.w * c1),
                                  fmaf(h1.x, c0, l1.x * c1), fmaf(h1.y, c0, l1.y * c1),
                                  fmaf(h1.z, c0, l1.z * c1), fmaf(h1.w, c0, l1.w * c1)};
              emit(y, f[k], o);
            }
          }
        }
        // word[7] is rewritten by the next split unit only after all read it
        asm volatile("bar.sync 1, %0;\n" ::"n"(kWorkers * 32) : "memory");
      }
      ++n_unit;
    };
    // a unit's results are written after the next unit's first plane is
    // built, so that plane's products run meanwhile
    Unit last{};
    for (int i = 0; i < units; ++i) {
      const Unit u = unit(i);
      fetch(u);
      for (int ch = u.c0; ch < u.c1; ++ch) {
        build(ch);
        if (ch == u.c0 && i > 0) finish(last);
      }
      last = u;
    }
    if (units > 0) finish(last);
  }

  // after a failed wait: the copies and products in flight are waited for
  if (__syncthreads_or(failed ? 1 : 0) && tid == 0) {
    const int issued = word[5], back = word[6];
    for (int st = 0; st < nstages; ++st) {
      if (issued <= st) continue;
      const int i = issued - 1 - (issued - 1 - st) % nstages;
      mbar_wait(sfull(st), (uint32_t)(i / nstages) & 1u);
    }
    if (back > 0) mbar_wait(sempty((back - 1) % nstages), (uint32_t)((back - 1) / nstages) & 1u);
    atomicOr(&a.ctr->err, kErrTimeout);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

// Entry [plane][chunk][j][limb][half of the 16 window columns][su column]
// [window column]: the kernel at dy = j - r - 15, dx = su column - window
// column + r, evaluated in FP64, zero outside the window.  A thread takes an
// entry (dx, dy) of the kernel and writes it wherever it stands, for up to eight
// su columns and all channels: FP64 powers bound it (a thread a limb pair, one
// for each, took 33 us at r = 40; now 13, and 20 for the cells' two laws).
__global__ void k_limb_tables(int r, int nch, double k0, double a0, double k1, double a1, double gamma,
                              double s0, double s1, __half* __restrict__ tab) {
  const int C = chunks_of(r), J = 2 * r + 31, E = 16 * C + 7;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= E * J) return;
  const int e = i % E, j = i / E;
  const int dy = j - r - 15, dx = r + 7 - e;  // = su column - window column + r
  const bool in = dx >= -r && dx <= r && dy >= -r && dy <= r && (dx | dy) != 0;
  const double d = in ? sqrt((double)(dx * dx + dy * dy)) : 1.0;
  const bool cells = nch == kCellPlanes;
  const double p0 = in ? pow(d, a0) : 0.0, p1 = !cells ? 0.0 : a1 == a0 ? p0 : in ? pow(d, a1) : 0.0;
  const double v0 = in ? k0 * p0 : 0.0, v1 = in ? k1 * p1 : 0.0;
  for (int ch = 0; ch < nch; ++ch) {
    const double v = cells ? (ch < 2 ? v0 : v1) : crowd_entry(v0, gamma, dx, dy, d, ch);
    const double first = limb16(v * s0), rest = (v * s0 - first) * s1, whole = rint(rest);
    // a cell plane's second table: what FP16 leaves of the second limb
    const bool second = cells && (ch & 1);
    const __half hi = __double2half(second ? 0.0 : first);
    const __half lo = __double2half(!cells ? limb16(rest) : second ? whole - limb16(whole) : limb16(whole));
#pragma unroll
    for (int nx = 0; nx < 8; ++nx) {
      const int w = nx - 7 + e;  // the window column
      if (w < 0 || w >= 16 * C) continue;
      __half* o = tab + ((size_t)(ch * C + w / 16) * J + j) * 256 + (w >> 3 & 1) * 64 + nx * 8 + (w & 7);
      o[0] = hi;
      o[128] = lo;
    }
  }
}

}  // namespace

bool product_crowd_scales(int r, const sfm_params& p, ProductScales* out) {
  return r >= 1 && r <= kProductMaxRadius && crowd_limb_scales(r, p.kP, p.aP, p.gamma, out);
}

bool product_cell_scales(int r, const sfm_params& p, ProductScales* out) {
  return r >= 1 && r <= kProductMaxRadius && cell_limb_scales(r, p.kO, p.aO, p.kE, p.aE, out);
}

size_t product_table_bytes(int r, int nch) { return (size_t)nch * chunks_of(r) * stage_bytes_of(r); }

void launch_limb_tables(int r, const sfm_params& p, const ProductScales& sc, int nch, uint8_t* tab,
                        cudaStream_t s) {
  const int n = (16 * chunks_of(r) + 7) * (2 * r + 31);
  const bool crowd = nch == kCrowdPlanes;
  k_limb_tables<<<(n + 63) / 64, 64, 0, s>>>(r, nch, crowd ? p.kP : p.kO, crowd ? p.aP : p.aO, p.kE,
                                                p.aE, p.gamma, sc.s0, sc.s1, reinterpret_cast<__half*>(tab));
}

void product_layout(int rmax, ProductArgs* a) {
  a->plane_bytes = plane_bytes_of(rmax);
  a->stage_bytes = stage_bytes_of(rmax);
  // a second plane where three stages still fit beside it, then as many
  // stages (up to 8) as the rest takes
  const int room = kSmem - kHeadBytes;
  a->nplanes = 2 * a->plane_bytes + 3 * a->stage_bytes <= room ? 2 : 1;
  a->nstages = (room - a->nplanes * a->plane_bytes) / a->stage_bytes;
  if (a->nstages > 8) a->nstages = 8;
  a->smem_bytes = kHeadBytes + a->nplanes * a->plane_bytes + a->nstages * a->stage_bytes;
}

int product_tiles_x(int W) { return (W + kTW - 1) / kTW; }
int product_tiles_y(int H) { return (H + kTH - 1) / kTH; }
size_t product_scratch_floats() { return kScratchFloats; }

cudaError_t launch_product(ProductArgs a, cudaStream_t s) {
  if (!a.lattices) {
    // the tile rows that hold rows [store_lo, store_hi)
    const int ty0 = a.store_lo / kTH, ty1 = (a.store_hi + kTH - 1) / kTH;
    a.tile0 = ty0 * a.one.ntx;
    a.ntiles = (ty1 - ty0) * a.one.ntx;
  }
  if (a.ntiles <= 0) return cudaSuccess;
  const cudaError_t e = allow_shared(k_product, kSmem);
  if (e != cudaSuccess) return e;
  return launch_tick_kernel(k_product, device_sm_count(), kProdThreads, a.smem_bytes, s, false, a);
}

}  // namespace sfm
