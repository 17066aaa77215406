// CUDA kernels of the GB300 TSDF library (sm_103a).
//
//  band_alloc_kernel  Sec. IV-B first step: one CTA per pixel tile; every
//                     valid pixel's ray segment inside the truncation band is
//                     walked through the block grid (Amanatides & Woo
//                     traversal) and its blocks recorded in a CTA-local set
//                     in shared memory; the tile's distinct blocks are then
//                     claimed in the open-addressing hash (atomicCAS on the
//                     packed key), given a pool block if new, and get the
//                     frame's bit; the first bit on a block appends it to
//                     the batch work list.
//  patch_alloc_kernel the same blocks for larger pinhole launches: one pixel
//                     of every 4 x 4 patch is walked, and the others only
//                     where a conservative test cannot show that their
//                     blocks are known already.
//  integrate_kernel   Sec. IV-B second step (Eq. 1-3 and the update
//                     functors: TSDF, occupancy, colour): the warps of a
//                     persistent grid take quarters of work-list blocks, 4
//                     voxels per thread held in registers across every frame
//                     of the batch that met the block, one coalesced read
//                     and write per block and batch.
//  query_kernel,      point -> voxel lookup through the hash.
//  query_color_kernel
//  decay_kernel       occupancy decay over every allocated block (Sec. V-E).
//
// Discrete decisions use explicit round-to-nearest intrinsics in a fixed
// order (no contraction) so that they are reproducible on a CPU.
#include <algorithm>
#include <atomic>
#include <cfloat>
#include <cmath>

#include "tsdf_internal.cuh"

namespace gbt {
namespace {

constexpr float kPiF = (float)3.14159265358979323846;
constexpr float kHalfPiF = (float)(3.14159265358979323846 / 2);

// Approximate reciprocal (within 1 ulp; 0 gives +-inf).
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// IEEE round-to-nearest reciprocal of a decision input.  FAST: the hardware
// approximation (within 1 ulp) refined by one Newton step with fused
// multiply-adds, e = 1 - x y, y' = y + y e (Markstein's method), which equals
// __frcp_rn(x) bit for bit for |x| in [2^-126, 2^126] (checked over all
// 4,227,858,434 such inputs).  The host selects FAST kernels only for
// batches whose inverted values all lie in that range or are zero (zero is
// never inverted), see fast_rcp_ok in the host code.
template <bool FAST>
__device__ __forceinline__ float rcp_dec(float x) {
  if (!FAST) return __frcp_rn(x);
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  const float e = __fmaf_rn(-x, y, 1.0f);
  return __fmaf_rn(y, e, y);
}

// rcp_dec<true> of a pair: the two refinement steps on the paired FP32
// operations (per component the same round-to-nearest result).
__device__ __forceinline__ float2 rcp_dec2(float a, float b) {
  float2 y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(a));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(b));
  const float2 e = __ffma2_rn(make_float2(-a, -b), y, make_float2(1.0f, 1.0f));
  return __ffma2_rn(y, e, y);
}

// ------------------------------------------------------------------ hash

__device__ __forceinline__ int hash_insert(const MapDev& m, unsigned long long key, bool& inserted) {
  uint32_t slot = hash_key(key) & m.cap_mask;
  inserted = false;
  // one atomic per probed slot: it inserts into an empty slot and reports
  // the slot's key otherwise (a single L2 round trip when the key is found)
  for (uint32_t probe = 0; probe <= m.cap_mask; ++probe) {
    const unsigned long long old = atomicCAS(m.keys + slot, kEmptyKey, key);
    if (old == kEmptyKey) {
      inserted = true;
      return (int)slot;
    }
    if (old == key) return (int)slot;
    slot = (slot + 1) & m.cap_mask;
  }
  return -1;
}

// ------------------------------------------------- block-grid traversal

__device__ __forceinline__ void claim_block(const MapDev& m, unsigned long long key, int bit) {
  bool ins;
  const int slot = hash_insert(m, key, ins);
  if (slot < 0) {
    atomicOr(m.counters + kCntStatus, (unsigned long long)kStHashFull);
    return;
  }
  if (ins) {
    const unsigned long long p = atomicAdd(m.counters + kCntBlocks, 1ull);
    if (p < (unsigned long long)m.max_blocks) {
      m.vals[slot] = -(int)p - 2;
      m.block_keys[p] = key;
    } else {
      m.vals[slot] = -1;
      atomicOr(m.counters + kCntStatus, (unsigned long long)kStPoolFull);
    }
  }
  if (atomicOr(m.mask + slot, 1u << bit) == 0u) {
    const uint32_t idx = atomicAdd(m.ctl, 1u);
    if (idx < m.list_cap) m.list[idx] = (uint32_t)slot;
    else atomicOr(m.counters + kCntStatus, (unsigned long long)kStListFull);
  }
}

// Walk in anchor-relative cell coordinates with a 32-bit key
// (cx + 512) | (cy + 512) << 10 | (cz + 512) << 20; used when the segment
// starts within kRelStart cells of the anchor, so that every cell of the walk
// (at most kMaxCells steps) stays inside the 10-bit fields.  The decisions
// are the prescribed FP32 sequence of the traversal, cell for cell.
constexpr int kRelBias = 512;
constexpr float kRelStart = 470.0f;
constexpr uint32_t kEmptyRel = 0xFFFFFFFFu;

// The sensor origin o is not stored: it is frame-wide (uniform across the
// CTA) and passed to every step, which keeps the per-lane state small (the
// allocator is compiled for 32 registers a thread: 8 CTAs of 256 threads per
// SM; measured faster than 40 registers without spills at 6 CTAs).
struct Walk32 {
  uint32_t key;
  uint32_t kx, ky, kz;  // key change of one step along each axis (+unit, -unit, 0)
  float bx, by, bz;     // next boundary per axis (+inf for an axis the ray does not cross)
  float ix, iy, iz;      // reciprocal direction per axis
  float s1;
  int n;

  // t of an axis is always (b - o) * inv; an axis with zero direction has
  // b = +inf and inv = 1, so its t is +inf.
  template <bool FAST>
  __device__ __forceinline__ void axis(float d, float fl, uint32_t unit, uint32_t& k, float& inv, float& b) {
    const bool pos = d > 0.0f, neg = d < 0.0f;
    k = pos ? unit : (neg ? 0u - unit : 0u);
    inv = (pos || neg) ? rcp_dec<FAST>(d) : 1.0f;
    b = pos ? fl + 1.0f : (neg ? fl : __int_as_float(0x7f800000));
  }
  template <bool FAST>
  __device__ __forceinline__ void start(float px, float py, float pz, float dx, float dy, float dz,
                                        float s1_, int bx0, int by0, int bz0, uint32_t flag) {
    const float flx = floorf(px), fly = floorf(py), flz = floorf(pz);
    key = ((uint32_t)((int)flx - bx0 + kRelBias) | ((uint32_t)((int)fly - by0 + kRelBias) << 10) |
           ((uint32_t)((int)flz - bz0 + kRelBias) << 20)) | flag;
    axis<FAST>(dx, flx, 1u, kx, ix, bx);
    axis<FAST>(dy, fly, 1u << 10, ky, iy, by);
    axis<FAST>(dz, flz, 1u << 20, kz, iz, bz);
    s1 = s1_;
    n = 1;
  }
  // The crossing parameters are recomputed from the boundaries at every
  // step, not carried: they are dead while the cell's key is recorded (at 32
  // registers a thread, carrying them spilled 88 bytes; 94.6 against 97.7 us
  // per 32-frame launch).  CAP: stop after kMaxCells cells; without it the
  // host has proved that every segment of the batch ends sooner (the cell
  // count then needs no register and no test).
  template <bool CAP>
  __device__ __forceinline__ bool next(float ox, float oy, float oz) {
    const float tx = __fmul_rn(__fsub_rn(bx, ox), ix);
    const float ty = __fmul_rn(__fsub_rn(by, oy), iy);
    const float tz = __fmul_rn(__fsub_rn(bz, oz), iz);
    const bool sy_ = ty < tx;
    const float t01 = fminf(tx, ty);
    const bool sz_ = tz < t01;
    const float t = fminf(t01, tz);
    if (!(t <= s1) || (CAP && n == kMaxCells)) return false;
    const bool sx_ = !sz_ && !sy_, syy = !sz_ && sy_;
    const uint32_t dk = sz_ ? kz : (sy_ ? ky : kx);
    key += dk;
    // the boundary moves by +1 or -1 along the stepped axis: the sign of its
    // key change (never 0: an axis the ray does not cross has t = +inf)
    const float f = __uint_as_float((dk & 0x80000000u) | 0x3f800000u);
    // predicated additions (an unconditional add of 0 costs a select more)
    if (sx_) bx = __fadd_rn(bx, f);
    if (syy) by = __fadd_rn(by, f);
    if (sz_) bz = __fadd_rn(bz, f);
    if (CAP) ++n;
    return true;
  }
};

__device__ __forceinline__ unsigned long long rel_to_key(uint32_t r, const int* a, int bx0 = 0,
                                                         int by0 = 0, int bz0 = 0) {
  return pack_key(a[0] + bx0 + (int)(r & 1023u) - kRelBias,
                  a[1] + by0 + (int)((r >> 10) & 1023u) - kRelBias,
                  a[2] + bz0 + (int)((r >> 20) & 1023u) - kRelBias);
}
constexpr uint32_t kFarFlag = 1u << 30;  // key counted from the segment's own start cell

// CTA-local set of relative block keys (open addressing in shared memory):
// `set` holds kSetSize slots, `keys` receives each key when it first enters
// the set (appended at *nkeys), so the tile's distinct blocks need no scan of
// the slots afterwards.  Returns false when the key could not be placed
// within kSetProbes slots, or is a far segment's key (bit 30: counted from
// the segment's own start cell, never in the set; it cannot match a slot,
// which holds a near key or kEmptyRel, so it always reaches the slow path);
// the caller then claims it globally itself.  The probing loop is inlined:
// at the allocator's 32 registers a call's saves and restores cost more
// than the larger code (measured 5 % slower as a call).
__device__ __forceinline__ bool set_insert_slow(uint32_t* set, uint32_t* keys, uint32_t* nkeys,
                                                uint32_t key, uint32_t h);

__device__ __forceinline__ bool set_insert(uint32_t* set, uint32_t* keys, uint32_t* nkeys, uint32_t key) {
  const uint32_t h = (key * 0x9E3779B1u) >> (32 - kSetBits);
  // common case: the key is already at its home slot
  if (((volatile uint32_t*)set)[h] == key) return true;
  return set_insert_slow(set, keys, nkeys, key, h);
}

__device__ __forceinline__ bool set_insert_slow(uint32_t* set, uint32_t* keys, uint32_t* nkeys,
                                                uint32_t key, uint32_t h) {
  if (key & kFarFlag) return false;
  volatile uint32_t* vs = set;
#pragma unroll 1
  for (int probe = 0; probe < kSetProbes; ++probe) {
    const uint32_t cur = vs[h];
    if (cur == key) return true;
    if (cur == kEmptyRel) {
      const uint32_t old = atomicCAS(set + h, kEmptyRel, key);
      if (old == kEmptyRel) {
        keys[atomicAdd(nkeys, 1u)] = key;  // at most kSetSize distinct keys
        return true;
      }
      if (old == key) return true;
    }
    h = (h + 1) & (kSetSize - 1);
  }
  return false;
}

// Band segment of pixel (i, j) (Sec. IV-B ray through the block grid): ray
// direction in anchor-relative block units per unit of depth (camera) or
// range (LiDAR) and the band [max(d - tau, 0), d + tau].  False if the pixel
// is outside the image or its depth is invalid.  A pinhole pixel outside the
// image was given depth 0, which is invalid; its ray is computed and unused.
// Pinhole rays: d = (fma(M0, rx, c0), fma(M3, rx, c1), fma(M6, rx, c2)) with
// the row's c = fma(M[3k+1], ry, M[3k+2]) staged once per tile row.
template <bool PINHOLE_ONLY>
__device__ __forceinline__ bool pixel_segment(const FrameDev& F, const MapDev& m,
                                              const float* s_ray, int i, int j, int lane, int ty,
                                              float d, float& dx, float& dy, float& dz, float& s0,
                                              float& s1) {
  bool valid;
  if (PINHOLE_ONLY || F.kind == kSensorPinhole) {
    valid = d > 0.0f && d <= FLT_MAX;
    const float rx = s_ray[lane];
    const float4 c = reinterpret_cast<const float4*>(s_ray + kTileW)[ty];
    dx = __fmaf_rn(F.M[0], rx, c.x);
    dy = __fmaf_rn(F.M[3], rx, c.y);
    dz = __fmaf_rn(F.M[6], rx, c.z);
  } else {
    if (i >= F.width || j >= F.height) return false;
    valid = d >= F.min_range && d <= F.max_range;
    const float2 az = __ldg(reinterpret_cast<const float2*>(F.tab) + i);
    const float2 el = __ldg(reinterpret_cast<const float2*>(F.tab) + F.width + j);
    const float bx = __fmul_rn(el.y, az.x), by = __fmul_rn(el.y, az.y), bz = el.x;
    dx = __fmaf_rn(F.M[0], bx, __fmaf_rn(F.M[1], by, __fmul_rn(F.M[2], bz)));
    dy = __fmaf_rn(F.M[3], bx, __fmaf_rn(F.M[4], by, __fmul_rn(F.M[5], bz)));
    dz = __fmaf_rn(F.M[6], bx, __fmaf_rn(F.M[7], by, __fmul_rn(F.M[8], bz)));
  }
  s0 = fmaxf(__fsub_rn(d, m.tau), 0.0f);
  s1 = __fadd_rn(d, m.tau);
  return valid;
}

// Shared memory of one allocation tile.
template <int TH>
struct AllocSmem {
  uint32_t set[kSetSize];   // CTA-local set of relative block keys
  uint32_t keys[kSetSize];  // the set's keys, in order of first insertion
  uint32_t nkeys;
  // pinhole: rx = (i - cu) / fu per column, then per row the three
  // fma(M[3k+1], ry, M[3k+2]) with ry = (j - cv) / fv (and one pad word)
  __align__(16) float ray[kTileW + 4 * TH];
};

// Frame of allocation tile `cta`: tiles are numbered frame by frame,
// FrameDev::blk_begin being a frame's first.
template <int NF, int NM>
__device__ __forceinline__ int tile_frame(const BatchParams<NF, NM>& p, int cta) {
  int f = 0;  // the last frame whose first tile is <= cta
  for (int lo = 1, hi = p.n_frames - 1; lo <= hi;) {
    const int mid = (lo + hi) >> 1;
    if (cta >= p.fr[mid].blk_begin) {
      f = mid;
      lo = mid + 1;
    } else {
      hi = mid - 1;
    }
  }
  return f;
}

// Allocation tile `cta` of the batch, a tile of frame f, run by all
// kAllocThreads threads of a CTA.  With p.overlap the stream's next kernel may be
// scheduled once the walks are done.
template <int NF, int NM, int TH, bool PINHOLE_ONLY, bool STATS, bool FAST, bool CAP>
__device__ __forceinline__ void alloc_tile(const BatchParams<NF, NM>& p, int f, int cta, AllocSmem<TH>& sm,
                                           bool wait) {
  constexpr int kRows = TH * kTileW / kAllocThreads;  // pixel rows per thread
  uint32_t segs = 0, cells = 0;                        // walk statistics
  uint32_t* s_set = sm.set;
  uint32_t* s_keys = sm.keys;
  float* s_ray = sm.ray;
  __syncthreads();  // a previous tile of this CTA is done with the shared arrays
  for (int i = threadIdx.x; i < kSetSize; i += kAllocThreads) s_set[i] = kEmptyRel;
  if (threadIdx.x == 0) sm.nkeys = 0;
  const FrameDev& F = p.fr[f];
  // with one map its fields are constant operands, not indexed loads
  const MapDev& m = NM == 1 ? p.maps[0] : p.maps[F.map];
  const int tiles_x = (F.width + kTileW - 1) / kTileW;
  const int tile = cta - F.blk_begin;
  const int x0 = (tile % tiles_x) * kTileW, y0 = (tile / tiles_x) * TH;
  const int lane = threadIdx.x % kTileW, wy = threadIdx.x / kTileW;
  if (PINHOLE_ONLY || F.kind == kSensorPinhole) {
    if (threadIdx.x < kTileW)
      s_ray[threadIdx.x] = __fdiv_rn(__fsub_rn((float)(x0 + (int)threadIdx.x), F.cu), F.fu);
    else if (threadIdx.x < kTileW + TH) {
      const float ry = __fdiv_rn(__fsub_rn((float)(y0 + (int)threadIdx.x - kTileW), F.cv), F.fv);
      reinterpret_cast<float4*>(s_ray + kTileW)[threadIdx.x - kTileW] =
          make_float4(__fmaf_rn(F.M[1], ry, F.M[2]), __fmaf_rn(F.M[4], ry, F.M[5]),
                      __fmaf_rn(F.M[7], ry, F.M[8]), 0.0f);
    }
  }
  // nothing above reads memory that the stream's previous kernel may write
  if (wait) wait_prev_grid();
  // all of this thread's depths are requested before any is used
  float dep[kRows];
#pragma unroll
  for (int q = 0; q < kRows; ++q) {
    const int i = x0 + lane, j = y0 + wy + q * (kAllocThreads / kTileW);
    dep[q] = (i < F.width && j < F.height) ? __ldg(F.depth + (size_t)j * F.width + i) : 0.0f;
  }
  __syncthreads();

#pragma unroll
  for (int q = 0; q < kRows; ++q) {
    const int ty = wy + q * (kAllocThreads / kTileW);
    bool live = false;
    Walk32 wk;
    wk.key = kEmptyRel;
    int b0x = 0, b0y = 0, b0z = 0;  // key origin of a far segment
    float dx, dy, dz, s0, s1;
    if (pixel_segment<PINHOLE_ONLY>(F, m, s_ray, x0 + lane, y0 + ty, lane, ty, dep[q], dx, dy, dz, s0, s1)) {
      const float px = __fmaf_rn(s0, dx, F.o[0]), py = __fmaf_rn(s0, dy, F.o[1]),
                  pz = __fmaf_rn(s0, dz, F.o[2]);
      if (fabsf(px) < kRelStart && fabsf(py) < kRelStart && fabsf(pz) < kRelStart) {
        wk.start<FAST>(px, py, pz, dx, dy, dz, s1, 0, 0, 0, 0u);
        live = true;
      } else if (fabsf(px) < 262144.0f && fabsf(py) < 262144.0f && fabsf(pz) < 262144.0f) {
        // far from the sensor's block (long range or small voxels): count
        // cells from the start cell and claim them globally one by one
        b0x = (int)floorf(px);
        b0y = (int)floorf(py);
        b0z = (int)floorf(pz);
        wk.start<FAST>(px, py, pz, dx, dy, dz, s1, b0x, b0y, b0z, kFarFlag);
        live = true;
      }
    }
    segs += live ? 1u : 0u;
    while (__any_sync(0xffffffffu, live)) {
      if (live) {
        ++cells;
        if (!set_insert(s_set, s_keys, &sm.nkeys, wk.key)) {
          if (wk.key & kFarFlag)
            claim_block(m, rel_to_key(wk.key & ~kFarFlag, F.a, b0x, b0y, b0z), F.bit);
          else
            claim_block(m, rel_to_key(wk.key, F.a), F.bit);
        }
        live = wk.template next<CAP>(F.o[0], F.o[1], F.o[2]);
      }
    }
  }
  if (p.overlap) allow_next_grid();
  __syncthreads();
  // the tile's distinct blocks, claimed one per thread
  const uint32_t nk = sm.nkeys;
  for (uint32_t i = threadIdx.x; i < nk; i += kAllocThreads) claim_block(m, rel_to_key(s_keys[i], F.a), F.bit);
  if (STATS) {
    for (int o = 16; o > 0; o >>= 1) {
      segs += __shfl_down_sync(0xffffffffu, segs, o);
      cells += __shfl_down_sync(0xffffffffu, cells, o);
    }
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(m.counters + kCntSegments, (unsigned long long)segs);
      atomicAdd(m.counters + kCntCells, (unsigned long long)cells);
    }
  }
}

// One CTA per kTileW x TH pixel tile of one frame.  Each warp walks the
// band segments of one pixel row at a time and records the blocks met in a
// CTA-local set; then the tile's distinct blocks are claimed in the global
// hash.  Segments that start far from the sensor's block count cells from
// their own start cell and claim their blocks directly.  PINHOLE_ONLY: every
// frame of the batch is a pinhole camera (the LiDAR code is left out);
// STATS: count band segments and walked cells (a diagnostic, 5 % slower);
// FAST: reciprocals by rcp_dec<true> (the host checked their range); CAP:
// walks stop after kMaxCells cells (without it the host proved them shorter).
template <int NF, int NM, int TH, bool PINHOLE_ONLY, bool STATS, bool FAST, bool CAP>
__global__ void __launch_bounds__(kAllocThreads, 7)
    band_alloc_kernel(const __grid_constant__ BatchParams<NF, NM> p) {
  __shared__ AllocSmem<TH> sm;
  const int f = tile_frame(p, (int)blockIdx.x);
  alloc_tile<NF, NM, TH, PINHOLE_ONLY, STATS, FAST, CAP>(p, f, (int)blockIdx.x, sm, p.overlap != 0);
}

// ------------------------------------------- pinhole tiles by pixel patches
//
// A tile's pixels see few blocks (a 64 x 64 pixel tile of a 2 cm map meets 30
// to 150 of them, each from hundreds of pixels), so most walks find nothing
// new.  patch_tile walks one pixel of every 4 x 4 patch, then asks of each
// patch whether all its pixels' walks could only meet blocks that the tile
// has already, and walks the pixels of those patches where the answer is no.
//
// Walking every pixel is issue-bound (about 340 warp instructions per 32
// pixels); here about a sixth of the pixels are walked (5 to 13 % of them
// after the test) and a patch's test costs about one walk.  Measured per
// launch, walking every pixel against this: 32 frames of 640x480 at 2 cm 98.9
// -> 47.6 us, 24 frames of 1280x720 at 5 cm 184 -> 61 us.  48 registers, 5
// CTAs of 256 threads per SM (60 registers and 4 CTAs were slower); tiles of
// 32 x 32 pixels were slower at every size (89 us for the 32 frames).
//
// The test is conservative and never decides a block: a bundle of pixels has
// ray directions within [dmin, dmax] per axis (the FP32 direction is monotone
// in the pixel's column and row, so the corner pixels bound it) and depths
// within [a0, b1] along them; every block the FP32 walks of these pixels can
// meet contains, inflated by s1 (dmax - dmin) / 2 + kBundleMargin per axis,
// a point of the central ray (the walk's roundings move a crossing by less
// than 4 ulp of the coordinate, 2.3e-4 blocks at |coordinate| < 960).  The blocks
// met by the inflated central ray are looked up row by row (a row = 32 blocks
// along x = one word of the tile's bitmap).
constexpr int kWin = 32;                  // bitmap window edge, blocks
constexpr float kBundleMargin = 1e-3f;    // blocks
constexpr int kPatchKeys = 512;           // distinct blocks a tile lists; more are claimed one by one
constexpr int kMaxRows = 16;              // bitmap rows one bundle test looks at
constexpr int kOutBits = 9;               // slots for claimed blocks outside the window: 512
// key field pattern of a cell inside the window: field = cell - window base + kRelBias
constexpr uint32_t kWinMask = ~(31u | (31u << 10) | (31u << 20));
constexpr uint32_t kWinPattern = (uint32_t)kRelBias | ((uint32_t)kRelBias << 10) | ((uint32_t)kRelBias << 20);

// A patch tile is kPatchTile x kPatchTile pixels, one thread per 4 x 4 patch.
constexpr int kPatchesX = kPatchTile / 4;
static_assert(kPatchesX * kPatchesX == kAllocThreads, "one thread per patch");

struct PatchSmem {
  __align__(16) uint32_t bm[kWin * kWin];  // bit x of word y + 32 z: the block is in the tile's set
  uint32_t keys[kPatchKeys];            // the set's keys in order of insertion
  __align__(8) uint32_t out[1 << kOutBits];  // claimed keys outside the window (claimed_outside)
  __align__(16) float4 row[kPatchTile]; // fma(M[3k+1], ry, M[3k+2]) per pixel row
  float rx[kPatchTile];                 // (i - cu) / fu per pixel column
  uint32_t nkeys, lo;                   // lo, hi: the tile's depth range (depth_range)
  int hi;
  uint32_t n[2];                        // patches, strips that the test left open
  // the open patches, then from kAllocThreads on the open strips: column / 4 | row << 8
  uint16_t open[5 * kAllocThreads];
};

// Record a walk's cell in the tile's bitmap; false if it must be claimed by
// the caller (outside the window, or the key list is full).
__device__ __forceinline__ bool bitmap_insert(uint32_t* bm, uint32_t* keys, uint32_t* nkeys, uint32_t key) {
  if ((key & kWinMask) != kWinPattern) return false;
  uint32_t* w = bm + (((key >> 10) & 31u) | ((key >> 15) & 0x3E0u));
  const uint32_t bit = 1u << (key & 31u);
  if (*(volatile uint32_t*)w & bit) return true;
  if (!(atomicOr(w, bit) & bit)) {
    const uint32_t i = atomicAdd(nkeys, 1u);
    if (i >= (uint32_t)kPatchKeys) return false;
    keys[i] = key;
  }
  return true;
}

// Whether the tile has claimed the block already, for blocks that the bitmap
// does not hold: the last key claimed at each of a few hashed slots.  Two
// threads that write a slot at once, or a key that another replaced, only
// claim again, which changes nothing; the slot is written by the thread that
// claims.  A tile that sees a near and a far surface has most of its cells
// outside the window, and claiming each in the global hash as it was walked
// cost more than walking by rows (32 frames of 640x480 at 1 cm: rows 107 us,
// 133 without the slots, 85 with them; 16 frames of 1280x720 at 7.5 mm: 145,
// 171, 119).  Tiles whose cells are all inside never come here: 32 frames at 2
// cm 65 us with and without.
__device__ __forceinline__ bool claimed_outside(uint32_t* out, uint32_t key) {
  volatile uint32_t* slot = out + ((key * 0x9E3779B1u) >> (32 - kOutBits));
  if (*slot == key) return true;
  *slot = key;
  return false;
}

// Whether every block that the bundle can meet is in the bitmap.  ow: sensor
// origin minus the window's base, in blocks.
__device__ __forceinline__ bool bundle_covered(const uint32_t* bm, const float* ow, const float* dmin,
                                               const float* dmax, float a0, float b1) {
  int lo[3], hi[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    lo[k] = __float2int_rd(__fmaf_rn(dmin[k] >= 0.0f ? a0 : b1, dmin[k], ow[k] - kBundleMargin));
    hi[k] = __float2int_rd(__fmaf_rn(dmax[k] >= 0.0f ? b1 : a0, dmax[k], ow[k] + kBundleMargin));
  }
  if (((lo[0] | lo[1] | lo[2] | hi[0] | hi[1] | hi[2]) & ~31) != 0) return false;  // not inside the window
  const int ny = hi[1] - lo[1] + 1, rows = ny * (hi[2] - lo[2] + 1);
  if (rows > kMaxRows) return false;
  const uint32_t full = (0xFFFFFFFFu << lo[0]) & (0xFFFFFFFFu >> (31 - hi[0]));
  // the central ray and the half width of the bundle around it
  float dc[3], e[3], inv[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    dc[k] = 0.5f * (dmin[k] + dmax[k]);
    e[k] = __fmaf_rn(b1 * 0.5f, dmax[k] - dmin[k], kBundleMargin);
    inv[k] = rcp_approx(dc[k]);
  }
  int y = lo[1], z = lo[2];
  for (int r = 0; r < rows; ++r) {
    const uint32_t missing = full & ~bm[y + kWin * z];
    if (missing) {
      // the part of the central ray inside the row's slabs, then its x range
      const float fy = (float)y - ow[1], fz = (float)z - ow[2];
      const float ya = (fy - e[1]) * inv[1], yb = (fy + (1.0f + e[1])) * inv[1];
      const float za = (fz - e[2]) * inv[2], zb = (fz + (1.0f + e[2])) * inv[2];
      const float t0 = fmaxf(fmaxf(a0, fminf(ya, yb)), fminf(za, zb));
      const float t1 = fminf(fminf(b1, fmaxf(ya, yb)), fmaxf(za, zb));
      if (t0 <= t1) {
        const float xa = __fmaf_rn(t0, dc[0], ow[0]), xb = __fmaf_rn(t1, dc[0], ow[0]);
        const int xl = max(__float2int_rd(fminf(xa, xb) - e[0]), lo[0]);
        const int xh = min(__float2int_rd(fmaxf(xa, xb) + e[0]), hi[0]);
        if (xl <= xh && (missing & (0xFFFFFFFFu << xl) & (0xFFFFFFFFu >> (31 - xh)))) return false;
      }
    }
    if (++y > hi[1]) {
      y = lo[1];
      ++z;
    }
  }
  return true;
}

// Depth of pixel (i, j), 0 outside the image.
__device__ __forceinline__ float pixel_depth(const FrameDev& F, int i, int j) {
  return (i < F.width && j < F.height) ? __ldg(F.depth + (size_t)j * F.width + i) : 0.0f;
}

// Four depths of a row from column i (a multiple of 4), 0 outside the image;
// one 16-byte load where the image allows it (FrameDev::vec4).
__device__ __forceinline__ float4 strip_depths(const FrameDev& F, int i, int j) {
  if (F.vec4) {
    if (i < F.width && j < F.height)
      return __ldg(reinterpret_cast<const float4*>(F.depth + (size_t)j * F.width + i));
    return make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
  return make_float4(pixel_depth(F, i, j), pixel_depth(F, i + 1, j), pixel_depth(F, i + 2, j),
                     pixel_depth(F, i + 3, j));
}

// Depth range of valid depths (0 < d <= FLT_MAX) over their bits: a valid
// depth's bits minus 1 are below 0x7F7FFFFF, and every other value's are not
// (unsigned), so the unsigned minimum ignores the invalid ones; the signed
// maximum ignores 0 and negative values, and reports infinities and NaN as
// 0x7F800000 or more.
constexpr uint32_t kNoDepth = 0x7F7FFFFFu;
__device__ __forceinline__ void depth_range(const float4& d, uint32_t& lo, int& hi) {
  const uint32_t a = __float_as_uint(d.x), b = __float_as_uint(d.y), c = __float_as_uint(d.z),
                 e = __float_as_uint(d.w);
  lo = min(lo, min(min(a - 1u, b - 1u), min(c - 1u, e - 1u)));
  hi = max(hi, max(max((int)a, (int)b), max((int)c, (int)e)));
}
__device__ __forceinline__ bool depth_ok(float d) { return __float_as_uint(d) - 1u < kNoDepth; }

template <int NF, int NM>
__device__ __forceinline__ void patch_tile(const BatchParams<NF, NM>& p, const FrameDev& F, const MapDev& m,
                                           int tile, PatchSmem& sm) {
  constexpr int NT = kAllocThreads;
  const int t = threadIdx.x;
  const int tiles_x = (F.width + kPatchTile - 1) / kPatchTile;
  const int x0 = (tile % tiles_x) * kPatchTile, y0 = (tile / tiles_x) * kPatchTile;
  const int px = (t % kPatchesX) * 4, py = (t / kPatchesX) * 4;  // this thread's patch in the tile
  static_assert(kWin * kWin == 4 * NT && (1 << kOutBits) == 2 * NT, "one store each per thread");
  reinterpret_cast<uint4*>(sm.bm)[t] = make_uint4(0u, 0u, 0u, 0u);
  reinterpret_cast<uint2*>(sm.out)[t] = make_uint2(kEmptyRel, kEmptyRel);
  for (int i = t; i < 2 * kPatchTile; i += NT) {
    if (i < kPatchTile) {
      sm.rx[i] = __fdiv_rn(__fsub_rn((float)(x0 + i), F.cu), F.fu);
    } else {
      const float ry = __fdiv_rn(__fsub_rn((float)(y0 + i - kPatchTile), F.cv), F.fv);
      sm.row[i - kPatchTile] = make_float4(__fmaf_rn(F.M[1], ry, F.M[2]), __fmaf_rn(F.M[4], ry, F.M[5]),
                                           __fmaf_rn(F.M[7], ry, F.M[8]), 0.0f);
    }
  }
  if (t == 0) {
    sm.nkeys = 0u;
    sm.lo = 0xFFFFFFFFu;
    sm.hi = 0;
    sm.n[0] = sm.n[1] = 0u;
  }
  if (p.overlap) wait_prev_grid();  // nothing above reads memory that the previous kernel may write
  float4 d[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) d[r] = strip_depths(F, x0 + px, y0 + py + r);
  uint32_t plo = 0xFFFFFFFFu;
  int phi = 0;
#pragma unroll
  for (int r = 0; r < 4; ++r) depth_range(d[r], plo, phi);
  // the pixel walked for the patch: one of the middle four
  float seed = d[1].y;
  int sx = px + 1, sy = py + 1;
  if (!depth_ok(seed)) { seed = d[2].z; sx = px + 2; sy = py + 2; }
  if (!depth_ok(seed)) { seed = d[1].z; sx = px + 2; sy = py + 1; }
  if (!depth_ok(seed)) { seed = d[2].y; sx = px + 1; sy = py + 2; }
  __syncthreads();
  const uint32_t wlo = __reduce_min_sync(0xffffffffu, plo);
  const int whi = __reduce_max_sync(0xffffffffu, phi);
  if ((t & 31) == 0) {
    atomicMin(&sm.lo, wlo);
    atomicMax(&sm.hi, whi);
  }
  __syncthreads();
  if (sm.lo >= kNoDepth) {  // no valid pixel
    if (p.overlap) allow_next_grid();
    return;
  }
  // the window's base: the middle of the tile's depth range on its central
  // ray; around the sensor where that is far off (the test then fails and
  // the walks claim what lies outside)
  int w[3];
  float ow[3];
  {
    const float mid = 0.5f * (__uint_as_float(sm.lo + 1u) + __int_as_float(min(sm.hi, 0x7F7FFFFF)));
    const float rx = sm.rx[kPatchTile / 2];
    const float4 c = sm.row[kPatchTile / 2];
    const float q[3] = {__fmaf_rn(mid, __fmaf_rn(F.M[0], rx, c.x), F.o[0]),
                        __fmaf_rn(mid, __fmaf_rn(F.M[3], rx, c.y), F.o[1]),
                        __fmaf_rn(mid, __fmaf_rn(F.M[6], rx, c.z), F.o[2])};
    const bool near = fabsf(q[0]) < 440.0f && fabsf(q[1]) < 440.0f && fabsf(q[2]) < 440.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      w[k] = (near ? __float2int_rd(q[k]) : 0) - kWin / 2;
      ow[k] = F.o[k] - (float)w[k];
    }
  }

  for (int stage = 0;; ++stage) {
    // walks: stage 0 one pixel per patch, stage 1 the pixels of the strips
    // that the test left open
    const int n = stage == 0 ? NT : 4 * (int)sm.n[1];
    for (int i = t; (i & ~31) < n; i += NT) {
      int lx = sx, ly = sy;
      float dep = seed;
      if (stage) {
        dep = 0.0f;
        if (i < n) {
          const int s = sm.open[NT + (i >> 2)];
          lx = (s & 255) * 4 + (i & 3);
          ly = s >> 8;
          dep = pixel_depth(F, x0 + lx, y0 + ly);
        }
      }
      bool live = false;
      Walk32 wk;
      wk.key = 0u;
      int b0x = 0, b0y = 0, b0z = 0;  // key origin of a far segment
      if (depth_ok(dep)) {
        const float rx = sm.rx[lx];
        const float4 c = sm.row[ly];
        const float dx = __fmaf_rn(F.M[0], rx, c.x), dy = __fmaf_rn(F.M[3], rx, c.y), dz = __fmaf_rn(F.M[6], rx, c.z);
        const float s0 = fmaxf(__fsub_rn(dep, m.tau), 0.0f), s1 = __fadd_rn(dep, m.tau);
        const float qx = __fmaf_rn(s0, dx, F.o[0]), qy = __fmaf_rn(s0, dy, F.o[1]), qz = __fmaf_rn(s0, dz, F.o[2]);
        if (fabsf(qx - (float)w[0]) < kRelStart && fabsf(qy - (float)w[1]) < kRelStart &&
            fabsf(qz - (float)w[2]) < kRelStart) {
          wk.start<true>(qx, qy, qz, dx, dy, dz, s1, w[0], w[1], w[2], 0u);
          live = true;
        } else if (fabsf(qx) < 262144.0f && fabsf(qy) < 262144.0f && fabsf(qz) < 262144.0f) {
          b0x = (int)floorf(qx);
          b0y = (int)floorf(qy);
          b0z = (int)floorf(qz);
          wk.start<true>(qx, qy, qz, dx, dy, dz, s1, b0x, b0y, b0z, kFarFlag);
          live = true;
        }
      }
      while (__any_sync(0xffffffffu, live)) {
        if (live) {
          // a far segment's key has bit 30 set and never has the window's pattern
          if (!bitmap_insert(sm.bm, sm.keys, &sm.nkeys, wk.key)) {
            if (wk.key & kFarFlag)
              claim_block(m, rel_to_key(wk.key & ~kFarFlag, F.a, b0x, b0y, b0z), F.bit);
            else if (!claimed_outside(sm.out, wk.key))
              claim_block(m, rel_to_key(wk.key, F.a, w[0], w[1], w[2]), F.bit);
          }
          live = wk.template next<false>(F.o[0], F.o[1], F.o[2]);
        }
      }
    }
    if (stage) break;
    __syncthreads();
    // the test: level 0 the 4 x 4 patches, level 1 the 4 x 1 strips of the
    // patches that it left open
    for (int level = 0; level < 2; ++level) {
      const int nb = level == 0 ? NT : 4 * (int)sm.n[0];
      for (int i = t; i < nb; i += NT) {
        int lx = px, ly = py, rows = 3;
        uint32_t lo = plo;
        int hi = phi;
        if (level) {
          const int patch = sm.open[i >> 2];
          lx = (patch & 255) * 4;
          ly = (patch >> 8) + (i & 3);
          rows = 0;
          lo = 0xFFFFFFFFu;
          hi = 0;
          depth_range(strip_depths(F, x0 + lx, y0 + ly), lo, hi);
        }
        if (lo >= kNoDepth) continue;  // no valid depth
        bool covered = false;
        if (hi <= 0x7F7FFFFF) {
          const float a0 = fmaxf(__fsub_rn(__uint_as_float(lo + 1u), m.tau), 0.0f);
          const float b1 = __fadd_rn(__int_as_float(hi), m.tau);
          const float ra = sm.rx[lx], rb = sm.rx[lx + 3];
          const float4 ca = sm.row[ly], cb = sm.row[ly + rows];
          float dmin[3], dmax[3];
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const float c0 = k == 0 ? ca.x : (k == 1 ? ca.y : ca.z), c1 = k == 0 ? cb.x : (k == 1 ? cb.y : cb.z);
            const float mk = F.M[3 * k];
            const float v0 = __fmaf_rn(mk, ra, c0), v1 = __fmaf_rn(mk, rb, c0), v2 = __fmaf_rn(mk, ra, c1),
                        v3 = __fmaf_rn(mk, rb, c1);
            dmin[k] = fminf(fminf(v0, v1), fminf(v2, v3));
            dmax[k] = fmaxf(fmaxf(v0, v1), fmaxf(v2, v3));
          }
          covered = bundle_covered(sm.bm, ow, dmin, dmax, a0, b1);
        }
        if (!covered) sm.open[(level ? NT : 0) + atomicAdd(&sm.n[level], 1u)] = (uint16_t)(lx >> 2 | ly << 8);
      }
      __syncthreads();
    }
  }
  if (p.overlap) allow_next_grid();
  __syncthreads();
  // the tile's distinct blocks, claimed one per thread
  const uint32_t nk = min(sm.nkeys, (uint32_t)kPatchKeys);
  for (uint32_t i = t; i < nk; i += NT) claim_block(m, rel_to_key(sm.keys[i], F.a, w[0], w[1], w[2]), F.bit);
}

union PatchOrRowSmem {
  PatchSmem patch;
  AllocSmem<kTileHTiny> row;
};

// Allocation of a batch whose frames all pass the host's reciprocal and
// segment-length checks: pinhole frames by patch_tile, LiDAR frames (MIXED)
// by alloc_tile.
template <int NF, int NM, bool MIXED>
__global__ void __launch_bounds__(kAllocThreads, 5)
    patch_alloc_kernel(const __grid_constant__ BatchParams<NF, NM> p) {
  const int f = tile_frame(p, (int)blockIdx.x);
  const FrameDev& F = p.fr[f];
  const MapDev& m = NM == 1 ? p.maps[0] : p.maps[F.map];
  if (MIXED) {
    __shared__ PatchOrRowSmem sm;
    if (F.kind != kSensorPinhole)
      alloc_tile<NF, NM, kTileHTiny, false, false, true, false>(p, f, (int)blockIdx.x, sm.row, p.overlap != 0);
    else
      patch_tile(p, F, m, (int)blockIdx.x - F.blk_begin, sm.patch);
  } else {
    __shared__ PatchSmem sm;
    patch_tile(p, F, m, (int)blockIdx.x - F.blk_begin, sm);
  }
}

// ------------------------------------------------ per-voxel projection

// FP32 atan2 for decisions: octant reduction, the half-angle identity
// atan t = 2 atan(t / (1 + sqrt(1 + t^2))) applied twice (|t| <= tan(pi/16)),
// then the Maclaurin series of atan through t^13.
__device__ __forceinline__ float atan2_dec(float y, float x) {
  const float ax = fabsf(x), ay = fabsf(y);
  const float mx = fmaxf(ax, ay), mn = fminf(ax, ay);
  if (mx == 0.0f) return 0.0f;
  const float t = __fdiv_rn(mn, mx);
  const float t1 = __fdiv_rn(t, __fadd_rn(1.0f, __fsqrt_rn(__fmaf_rn(t, t, 1.0f))));
  const float t2 = __fdiv_rn(t1, __fadd_rn(1.0f, __fsqrt_rn(__fmaf_rn(t1, t1, 1.0f))));
  const float z = __fmul_rn(t2, t2);
  float q = 1.0f / 13.0f;
  q = __fmaf_rn(q, z, -(1.0f / 11.0f));
  q = __fmaf_rn(q, z, 1.0f / 9.0f);
  q = __fmaf_rn(q, z, -(1.0f / 7.0f));
  q = __fmaf_rn(q, z, 1.0f / 5.0f);
  q = __fmaf_rn(q, z, -(1.0f / 3.0f));
  q = __fmaf_rn(q, z, 1.0f);
  float a = __fmul_rn(4.0f, __fmul_rn(t2, q));
  if (ay > ax) a = __fsub_rn(kHalfPiF, a);
  if (x < 0.0f) a = __fsub_rn(kPiF, a);
  if (y < 0.0f) a = -a;
  return a;
}

// The pair forms below take the same decisions as atan2_dec and __fsqrt_rn
// with two voxels per instruction.  A LiDAR projection takes six divisions and
// six square roots; the library's routines made it 450 issue slots a voxel
// (52 us for a 1024x64 scan of 8,227 blocks).

// Square roots: the hardware reciprocal root and one residual step on the
// root, d = x - g g, g' = g + d (y / 2) (Markstein's method).  Equal to
// __fsqrt_rn for every x in [2^-60, 2^100) (checked over all of them).
__device__ __forceinline__ float2 sqrt2_dec(float2 x) {
  float2 y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(x.x));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(x.y));
  const float2 g = __fmul2_rn(x, y), h = __fmul2_rn(y, make_float2(0.5f, 0.5f));
  const float2 d = __ffma2_rn(make_float2(-g.x, -g.y), g, x);
  return __ffma2_rn(d, h, g);
}

// t / (1 + sqrt(1 + t^2)) for t in [0, 1]: as a function of t alone it was
// compared with the IEEE operations over every t in [2^-60, 1] (below, both
// are t / 2), so the quotient needs no refined reciprocal.
__device__ __forceinline__ float2 half_tan2(float2 t) {
  const float2 one = make_float2(1.0f, 1.0f);
  const float2 b = __fadd2_rn(one, sqrt2_dec(__ffma2_rn(t, t, one)));
  float2 y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(b.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(b.y));
  const float2 q = __fmul2_rn(t, y);
  return __ffma2_rn(__ffma2_rn(make_float2(-b.x, -b.y), q, t), y, q);
}

// atan2_dec of two voxels whose larger magnitude is in [2^-30, 2^31] and whose
// smaller one is 0 or at least 2^-80: the quotient mn / mx by the correctly
// rounded reciprocal and one residual step (as div_voxel; nothing underflows
// in this range).
// mx, mn: the larger and smaller magnitude; Y_POSITIVE: y >= 0.
template <bool Y_POSITIVE>
__device__ __forceinline__ float2 atan2_dec2(float2 y, float2 x, float2 mx, float2 mn) {
  const float2 r = rcp_dec2(mx.x, mx.y);
  const float2 q0 = __fmul2_rn(mn, r);
  const float2 t = __ffma2_rn(__ffma2_rn(make_float2(-mx.x, -mx.y), q0, mn), r, q0);
  const float2 t2 = half_tan2(half_tan2(t));
  const float2 z = __fmul2_rn(t2, t2);
  float2 q = make_float2(1.0f / 13.0f, 1.0f / 13.0f);
  q = __ffma2_rn(q, z, make_float2(-(1.0f / 11.0f), -(1.0f / 11.0f)));
  q = __ffma2_rn(q, z, make_float2(1.0f / 9.0f, 1.0f / 9.0f));
  q = __ffma2_rn(q, z, make_float2(-(1.0f / 7.0f), -(1.0f / 7.0f)));
  q = __ffma2_rn(q, z, make_float2(1.0f / 5.0f, 1.0f / 5.0f));
  q = __ffma2_rn(q, z, make_float2(-(1.0f / 3.0f), -(1.0f / 3.0f)));
  q = __ffma2_rn(q, z, make_float2(1.0f, 1.0f));
  float2 a = __fmul2_rn(make_float2(4.0f, 4.0f), __fmul2_rn(t2, q));
  if (fabsf(y.x) > fabsf(x.x)) a.x = __fsub_rn(kHalfPiF, a.x);
  if (fabsf(y.y) > fabsf(x.y)) a.y = __fsub_rn(kHalfPiF, a.y);
  if (x.x < 0.0f) a.x = __fsub_rn(kPiF, a.x);
  if (x.y < 0.0f) a.y = __fsub_rn(kPiF, a.y);
  if (!Y_POSITIVE && y.x < 0.0f) a.x = -a.x;
  if (!Y_POSITIVE && y.y < 0.0f) a.y = -a.y;
  return a;
}

// LiDAR projection of a voxel centre in the sensor's frame (Eq. 3): range,
// azimuth and polar angle.
__device__ __noinline__ float3 lidar_angles(float x, float y, float z) {
  const float rr = __fsqrt_rn(__fmaf_rn(x, x, __fmaf_rn(y, y, __fmul_rn(z, z))));
  const float rho = __fsqrt_rn(__fmaf_rn(x, x, __fmul_rn(y, y)));
  return make_float3(rr, atan2_dec(y, x), atan2_dec(rho, z));
}

// lidar_angles of two points (x, y, z): by the pair forms if both lie in their
// range (all three magnitudes at least 2^-80, the larger of |x| and |y| at
// least 2^-30, all at most 2^30), else one by one.
__device__ __forceinline__ void lidar_angles2(float2 x, float2 y, float2 z, float2& rr, float2& th, float2& ph) {
  const float2 mx = make_float2(fmaxf(fabsf(x.x), fabsf(y.x)), fmaxf(fabsf(x.y), fabsf(y.y)));
  const float2 mn = make_float2(fminf(fabsf(x.x), fabsf(y.x)), fminf(fabsf(x.y), fabsf(y.y)));
  const float low = fminf(fminf(mn.x, mn.y), fminf(fabsf(z.x), fabsf(z.y)));
  const float high = fmaxf(fmaxf(mx.x, mx.y), fmaxf(fabsf(z.x), fabsf(z.y)));
  if (low >= 0x1p-80f && fminf(mx.x, mx.y) >= 0x1p-30f && high <= 0x1p30f) {
    rr = sqrt2_dec(__ffma2_rn(x, x, __ffma2_rn(y, y, __fmul2_rn(z, z))));
    const float2 rho = sqrt2_dec(__ffma2_rn(x, x, __fmul2_rn(y, y)));
    th = atan2_dec2<false>(y, x, mx, mn);
    ph = atan2_dec2<true>(rho, z, make_float2(fmaxf(rho.x, fabsf(z.x)), fmaxf(rho.y, fabsf(z.y))),
                          make_float2(fminf(rho.x, fabsf(z.x)), fminf(rho.y, fabsf(z.y))));
  } else {
    const float3 a = lidar_angles(x.x, y.x, z.x), b = lidar_angles(x.y, y.y, z.y);
    rr = make_float2(a.x, b.x);
    th = make_float2(a.y, b.y);
    ph = make_float2(a.z, b.z);
  }
}

// min / max that return NaN if either operand is one.
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// Azimuth column k in [-1, naz] wrapped into [0, naz).
__device__ __forceinline__ int wrap_az(int k, int naz) {
  return k < 0 ? k + naz : (k >= naz ? k - naz : k);
}

__device__ __forceinline__ bool lidar_valid(const FrameDev& F, float d) {
  return d >= F.min_range && d <= F.max_range;
}

// TSDF update functor (Sec. IV-B): weighted running average, the average
// taken with the unclamped weight sum, then weights capped; a zero weight on
// an unobserved voxel changes nothing.
__device__ __forceinline__ void fuse(float& D, float& W, float s, float w, float wmax) {
  const float wn = W + w;
  if (!(wn > 0.0f)) return;
  D = D + __fdividef(w * (s - D), wn);
  W = fminf(wn, wmax);
}

// Weight f_w(d_p) (Sec. IV-B: constant or from the sensor's error model):
// 1, times 1 / d_v^2 for inverse-square weighting, times a linear drop-off
// from 1 at d_p = -dropoff to 0 at d_p = -tau behind the surface.
__device__ __forceinline__ float weight(const MapDev& m, float dv, float dp) {
  float w = 1.0f;
  if (m.weighting & 1) w = __fdividef(1.0f, dv * dv);
  if ((m.weighting & 2) && dp < -m.dropoff) w *= __fdividef(m.tau + dp, m.tau - m.dropoff);
  return w;
}

// Update functor of a voxel that passed the projection test, d_p >= -tau:
// the TSDF average, or for an occupancy layer (Sec. IV-B, second functor)
// the running addition of l_free in front of the surface (d_p > 0) and
// l_occ otherwise.
// WEIGHTED: the map uses a non-constant weighting function (the constant
// weight 1 keeps the update short: fewer instructions in the unrolled loops).
template <int STORAGE, bool WEIGHTED>
__device__ __forceinline__ void apply(const MapDev& m, float& D, float& W, float dv, float dp) {
  if (STORAGE == kStorageOcc) {
    D += dp > 0.0f ? m.l_free : m.l_occ;
  } else if (WEIGHTED) {
    fuse(D, W, fminf(dp, m.tau), weight(m, dv, dp), m.wmax);
  } else {
    const float wn = W + 1.0f;
    D = D + __fdividef(fminf(dp, m.tau) - D, wn);
    W = fminf(wn, m.wmax);
  }
}

// Colour functor: the running average of the pixel's r, g, b with weight 1
// per frame (the TSDF average applied per channel), weights capped.
__device__ __forceinline__ void apply_color(const MapDev& m, float& R, float& G, float& B, float& W,
                                            uint32_t c) {
  const float wn = W + 1.0f;
  const float iw = __frcp_rn(wn);
  R = __fmaf_rn(__fsub_rn((float)(c & 255u), R), iw, R);
  G = __fmaf_rn(__fsub_rn((float)((c >> 8) & 255u), G), iw, G);
  B = __fmaf_rn(__fsub_rn((float)((c >> 16) & 255u), B), iw, B);
  W = fminf(wn, m.wmax);
}

// A thread's four voxels: (x, y, z), (x, y, z + 1), (x + 1, y, z) and
// (x + 1, y, z + 1), as global voxel indices in FP32 (exact: below 2^23 + 8
// in magnitude), and the index `at` of the first two's x pair in its block
// (x / 2 + 4 y + 32 z).  A warp holds two z layers, 8 x 8 voxels each, and its
// lanes look one layer up at a time: a gather of depths then touches fewer
// image rows than with four voxels along x per thread (two layers at a time).
struct VoxelQuad {
  float x, y, z;
  int at;
};

// The voxels in registers: D and W (TSDF distance and weight, occupancy
// log-odds, or colour red and weight) and, for colour only, G and B.
template <int STORAGE>
struct Voxels4;

template <>
struct Voxels4<kStorageF32> {
  __device__ __forceinline__ static void load(const MapDev& m, int pool, int at, float* D, float* W,
                                              float* G, float* B) {
    const float4* src = reinterpret_cast<const float4*>(m.pool) + (size_t)pool * 256 + at;
    const float4 a = src[0], b = src[32];
    D[0] = a.x; W[0] = a.y; D[2] = a.z; W[2] = a.w;
    D[1] = b.x; W[1] = b.y; D[3] = b.z; W[3] = b.w;
  }
  __device__ __forceinline__ static void store(const MapDev& m, int pool, int at, const float* D,
                                               const float* W, const float* G, const float* B) {
    float4* dst = reinterpret_cast<float4*>(m.pool) + (size_t)pool * 256 + at;
    dst[0] = make_float4(D[0], W[0], D[2], W[2]);
    dst[32] = make_float4(D[1], W[1], D[3], W[3]);
  }
};

template <>
struct Voxels4<kStorageOcc> {
  __device__ __forceinline__ static void load(const MapDev& m, int pool, int at, float* D, float* W,
                                              float* G, float* B) {
    const float2* src = reinterpret_cast<const float2*>(m.pool) + (size_t)pool * 256 + at;
    const float2 a = src[0], b = src[32];
    D[0] = a.x; D[2] = a.y; D[1] = b.x; D[3] = b.y;
    W[0] = W[1] = W[2] = W[3] = 0.0f;
  }
  __device__ __forceinline__ static void store(const MapDev& m, int pool, int at, const float* D,
                                               const float* W, const float* G, const float* B) {
    float2* dst = reinterpret_cast<float2*>(m.pool) + (size_t)pool * 256 + at;
    dst[0] = make_float2(D[0], D[2]);
    dst[32] = make_float2(D[1], D[3]);
  }
};

// 16-bit storages: one word per voxel.
template <int STORAGE>
__device__ __forceinline__ void unpack16(const MapDev& m, uint32_t w, float& D, float& W) {
  if (STORAGE == kStorageF16) {
    const __half2 h = *reinterpret_cast<const __half2*>(&w);
    D = __low2float(h) * m.tau;
    W = __high2float(h);
  } else {
    D = x16_dist(w, m.x16_unit);
    W = x16_weight(w);
  }
}
template <int STORAGE>
__device__ __forceinline__ uint32_t pack16(const MapDev& m, float D, float W) {
  if (STORAGE == kStorageF16) {
    const __half2 h = __floats2half2_rn(D * m.inv_tau, W);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
  return x16_pack(D, W, m.x16_scale);
}
template <int STORAGE>
struct Voxels4Word {
  __device__ __forceinline__ static void load(const MapDev& m, int pool, int at, float* D, float* W,
                                              float* G, float* B) {
    const uint2* src = reinterpret_cast<const uint2*>(m.pool) + (size_t)pool * 256 + at;
    const uint2 a = src[0], b = src[32];
    unpack16<STORAGE>(m, a.x, D[0], W[0]);
    unpack16<STORAGE>(m, a.y, D[2], W[2]);
    unpack16<STORAGE>(m, b.x, D[1], W[1]);
    unpack16<STORAGE>(m, b.y, D[3], W[3]);
  }
  __device__ __forceinline__ static void store(const MapDev& m, int pool, int at, const float* D,
                                               const float* W, const float* G, const float* B) {
    uint2* dst = reinterpret_cast<uint2*>(m.pool) + (size_t)pool * 256 + at;
    dst[0] = make_uint2(pack16<STORAGE>(m, D[0], W[0]), pack16<STORAGE>(m, D[2], W[2]));
    dst[32] = make_uint2(pack16<STORAGE>(m, D[1], W[1]), pack16<STORAGE>(m, D[3], W[3]));
  }
};
template <>
struct Voxels4<kStorageF16> : Voxels4Word<kStorageF16> {};
template <>
struct Voxels4<kStorageX16> : Voxels4Word<kStorageX16> {};

template <>
struct Voxels4<kStorageColor> {
  __device__ __forceinline__ static void load(const MapDev& m, int pool, int at, float* D, float* W,
                                              float* G, float* B) {
    const float4* src = reinterpret_cast<const float4*>(m.pool) + (size_t)pool * 512 + 2 * at;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 a = src[(i & 1) * 64 + (i >> 1)];
      D[i] = a.x; G[i] = a.y; B[i] = a.z; W[i] = a.w;
    }
  }
  __device__ __forceinline__ static void store(const MapDev& m, int pool, int at, const float* D,
                                               const float* W, const float* G, const float* B) {
    float4* dst = reinterpret_cast<float4*>(m.pool) + (size_t)pool * 512 + 2 * at;
#pragma unroll
    for (int i = 0; i < 4; ++i) dst[(i & 1) * 64 + (i >> 1)] = make_float4(D[i], G[i], B[i], W[i]);
  }
};

// Voxel centres in frame F's sensor frame (Eq. 1), in the FP32 decision
// sequence p_i = fma(R_i0, qx, fma(R_i1, qy, fma(R_i2, qz, t_i))).
__device__ __forceinline__ void quad_points(const FrameDev& F, float v, const VoxelQuad& r,
                                            float* px, float* py, float* pz) {
  // anchor-relative voxel indices: exact in FP32 (|index| < 2^24)
  const float rx = __fsub_rn(r.x, (float)(F.a[0] * 8)), ry = __fsub_rn(r.y, (float)(F.a[1] * 8)),
              rz = __fsub_rn(r.z, (float)(F.a[2] * 8));
  const float qy = __fmul_rn(__fadd_rn(ry, 0.5f), v);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float qz = __fmul_rn(__fadd_rn(rz, (float)k + 0.5f), v);
    const float cx = __fmaf_rn(F.Rcl[1], qy, __fmaf_rn(F.Rcl[2], qz, F.tloc[0]));
    const float cy = __fmaf_rn(F.Rcl[4], qy, __fmaf_rn(F.Rcl[5], qz, F.tloc[1]));
    const float cz = __fmaf_rn(F.Rcl[7], qy, __fmaf_rn(F.Rcl[8], qz, F.tloc[2]));
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float qx = __fmul_rn(__fadd_rn(rx, (float)j + 0.5f), v);
      px[2 * j + k] = __fmaf_rn(F.Rcl[0], qx, cx);
      py[2 * j + k] = __fmaf_rn(F.Rcl[3], qx, cy);
      pz[2 * j + k] = __fmaf_rn(F.Rcl[6], qx, cz);
    }
  }
}

// A pinhole frame's projection constants, staged in shared memory once per
// CTA: 16-byte loads in the voxel loop instead of one constant-bank load per
// field (the frame index is not known at compile time, so the fields cannot
// be instruction operands).  What multiplies voxel pairs is stored twice, as
// the paired operations read it.
struct __align__(16) FrameProj {
  float2 r0x, r1x, r2x, r0y, r1y, r2y, r0z, r1z, r2z;  // R_CL, duplicated
  float2 t0, t1, t2, nfu, nfv, cu, cv;                 // t_loc; -fu, -fv
  float ax, ay, az;                                    // 8 a: the anchor block's first voxel
  int width;
  const float* depth;
  int height, unused;
};

__device__ __forceinline__ float2 twice(float x) { return make_float2(x, x); }

__device__ __forceinline__ void stage_frame(const FrameDev& F, FrameProj& S) {
  S.r0x = twice(F.Rcl[0]); S.r1x = twice(F.Rcl[3]); S.r2x = twice(F.Rcl[6]);
  S.r0y = twice(F.Rcl[1]); S.r1y = twice(F.Rcl[4]); S.r2y = twice(F.Rcl[7]);
  S.r0z = twice(F.Rcl[2]); S.r1z = twice(F.Rcl[5]); S.r2z = twice(F.Rcl[8]);
  S.t0 = twice(F.tloc[0]); S.t1 = twice(F.tloc[1]); S.t2 = twice(F.tloc[2]);
  S.nfu = twice(-F.fu); S.nfv = twice(-F.fv);
  S.cu = twice(F.cu); S.cv = twice(F.cv);
  S.ax = (float)(F.a[0] * 8); S.ay = (float)(F.a[1] * 8); S.az = (float)(F.a[2] * 8);
  S.width = F.width;
  S.height = F.height;
  S.depth = F.depth;
}

// -1 / z of a voxel pair, the negative of rcp_dec<FAST> (rounding is
// symmetric in sign): e = 1 + z y with y ~ -1/z, then y + y e.
template <bool FAST>
__device__ __forceinline__ float2 neg_rcp2(float2 z) {
  if (!FAST) return make_float2(-__frcp_rn(z.x), -__frcp_rn(z.y));
  const float2 y = make_float2(rcp_approx(-z.x), rcp_approx(-z.y));
  return __ffma2_rn(y, __ffma2_rn(z, y, twice(1.0f)), y);
}

// floor(u) by a round-down addition: the low bits of u + 1.5 * 2^23 hold it
// for |u| < 2^22, and for any other u (NaN included) the difference from
// kFloorBits is, unsigned, at least 2^22.  (A conversion instruction runs at an
// eighth of the rate, on the unit that also serves the reciprocals.)
constexpr float kFloorMagic = 12582912.0f;
constexpr uint32_t kFloorBits = 0x4B400000u;

// The constant-weight TSDF update (apply) of a voxel pair, selected per voxel:
// D + (s - D) / (W + 1), rounded once after the product with the reciprocal.
// (As the addition of a product it was contracted to this by the compiler.)
__device__ __forceinline__ void update_pair(const MapDev& m, float* D, float* W, float2 dp, bool ok0, bool ok1) {
  const float2 wn = __fadd2_rn(make_float2(W[0], W[1]), twice(1.0f));
  const float2 D2 = make_float2(D[0], D[1]);
  const float2 diff = __ffma2_rn(D2, twice(-1.0f), make_float2(fminf(dp.x, m.tau), fminf(dp.y, m.tau)));
  const float2 dn = __ffma2_rn(diff, make_float2(rcp_approx(wn.x), rcp_approx(wn.y)), D2);
  if (ok0) { D[0] = dn.x; W[0] = fminf(wn.x, m.wmax); }
  if (ok1) { D[1] = dn.y; W[1] = fminf(wn.y, m.wmax); }
}

// NQ consecutive pinhole frames of the batch: phase 1 projects every voxel
// into every frame (Eq. 2, nearest pixel) and issues all depth loads (and
// colour loads for a colour layer), phase 2 applies the updates in frame
// order.  An out-of-image projection reads no pixel and yields d = 0, which
// is invalid like a missing depth.  A colour layer updates only voxels within
// tau of the surface on both sides.  Voxel pairs share the paired FP32
// operations (per component the same round-to-nearest result), and the
// constant-weight update is computed for every voxel and selected, not
// branched to, so the four voxels' chains overlap.
template <int NQ, int STORAGE, bool WEIGHTED, bool FAST, class P>
__device__ __forceinline__ void fuse_pinhole(const P& p, const FrameProj* s_fp, const int (&fq)[2],
                                             const MapDev& m, const VoxelQuad& r, float* D, float* W,
                                             float* G, float* B, uint32_t& upd) {
  float d[NQ][4], z[NQ][4];
  uint32_t c[NQ][4];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const FrameProj& S = s_fp[fq[q]];
    const float* depth = S.depth;
    const int width = S.width, height = S.height;
    // voxel centres in the sensor frame (quad_points with staged constants),
    // as pairs along z
    const float2 qy = twice(__fmul_rn(__fadd_rn(__fsub_rn(r.y, S.ay), 0.5f), m.v));
    const float2 qz = __fmul2_rn(__fadd2_rn(twice(__fsub_rn(r.z, S.az)), make_float2(0.5f, 1.5f)), twice(m.v));
    const float2 cx = __ffma2_rn(S.r0y, qy, __ffma2_rn(S.r0z, qz, S.t0));
    const float2 cy = __ffma2_rn(S.r1y, qy, __ffma2_rn(S.r1z, qz, S.t1));
    const float2 cz = __ffma2_rn(S.r2y, qy, __ffma2_rn(S.r2z, qz, S.t2));
    const float fx = __fsub_rn(r.x, S.ax);
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const float2 qx = twice(__fmul_rn(__fadd_rn(fx, (float)(i / 2) + 0.5f), m.v));
      const float2 x = __ffma2_rn(S.r0x, qx, cx), y = __ffma2_rn(S.r1x, qx, cy), zz = __ffma2_rn(S.r2x, qx, cz);
      const float2 niz = neg_rcp2<FAST>(zz);
      // u = x / z fu + cu + 1/2 as (x (-1/z)) (-fu) + cu + 1/2
      const float2 u = __fadd2_rn(__ffma2_rn(__fmul2_rn(x, niz), S.nfu, S.cu), twice(0.5f));
      const float2 v = __fadd2_rn(__ffma2_rn(__fmul2_rn(y, niz), S.nfv, S.cv), twice(0.5f));
      z[q][i] = zz.x;
      z[q][i + 1] = zz.y;
      if (FAST) {
        // pixel = floor(u), valid iff 0 <= u < W: one unsigned comparison of
        // the floored value per axis (the host checked W, H <= 2^22; z > 0
        // implies z >= 2^-126 in FAST batches, so 1 / z is finite)
        const float2 tu = __fadd2_rd(u, twice(kFloorMagic)), tv = __fadd2_rd(v, twice(kFloorMagic));
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const uint32_t iu = __float_as_uint(k ? tu.y : tu.x) - kFloorBits;
          const uint32_t iv = __float_as_uint(k ? tv.y : tv.x) - kFloorBits;
          const bool in = z[q][i + k] > 0.0f && iu < (uint32_t)width && iv < (uint32_t)height;
          const int pix = (int)iv * width + (int)iu;
          d[q][i + k] = in ? __ldg(depth + pix) : 0.0f;
          if (STORAGE == kStorageColor) c[q][i + k] = in ? __ldg(p.fr[fq[q]].rgba + pix) : 0u;
        }
      } else {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float uk = k ? u.y : u.x, vk = k ? v.y : v.x;
          const bool in = z[q][i + k] > 0.0f && uk >= 0.0f && uk < (float)width && vk >= 0.0f && vk < (float)height;
          const int pix = (int)vk * width + (int)uk;
          d[q][i + k] = in ? __ldg(depth + pix) : 0.0f;
          if (STORAGE == kStorageColor) c[q][i + k] = in ? __ldg(p.fr[fq[q]].rgba + pix) : 0u;
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q)
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const float2 dp = __ffma2_rn(make_float2(z[q][i], z[q][i + 1]), twice(-1.0f),
                                   make_float2(d[q][i], d[q][i + 1]));  // d - z, rounded once
      // a valid depth, 0 < d <= FLT_MAX: one unsigned comparison of its bits
      const bool ok0 = depth_ok(d[q][i]) && !(dp.x < -m.tau), ok1 = depth_ok(d[q][i + 1]) && !(dp.y < -m.tau);
      if (STORAGE == kStorageColor) {
        if (ok0 && !(dp.x > m.tau)) {
          apply_color(m, D[i], G[i], B[i], W[i], c[q][i]);
          ++upd;
        }
        if (ok1 && !(dp.y > m.tau)) {
          apply_color(m, D[i + 1], G[i + 1], B[i + 1], W[i + 1], c[q][i + 1]);
          ++upd;
        }
      } else if (STORAGE == kStorageOcc || WEIGHTED) {
        if (ok0) apply<STORAGE, WEIGHTED>(m, D[i], W[i], z[q][i], dp.x);
        if (ok1) apply<STORAGE, WEIGHTED>(m, D[i + 1], W[i + 1], z[q][i + 1], dp.y);
        upd += (ok0 ? 1u : 0u) + (ok1 ? 1u : 0u);
      } else {
        update_pair(m, D + i, W + i, dp, ok0, ok1);
        upd += (ok0 ? 1u : 0u) + (ok1 ? 1u : 0u);
      }
    }
}

// A LiDAR frame (Eq. 1 and 3): phase 1 finds every voxel's beam cell and
// issues its range loads (the four around it, or the nearest one), phase 2
// applies the guarded bilinear sample and the updates.  A voxel at the
// sensor origin, outside the elevation rows or with an invalid sample is not
// updated; azimuth wraps.  Colour layers take pinhole frames only.
//
// FAST (constant weight, at most 2^21 columns and rows, the host checks):
// voxel pairs throughout, cells floored by the round-down addition (kFloorMagic),
// and the sample and update only where a pair has a valid cell (about a third
// of the voxels of an outdoor scan's band do).  A 1024x64 scan's launch 43.3 ->
// 39.4 us; 32 mixed frames over 16 maps 88.8 -> 80.8.
template <int STORAGE, bool WEIGHTED, bool FAST>
__device__ __forceinline__ void fuse_lidar(const FrameDev& F, const MapDev& m, const VoxelQuad& r,
                                           float* D, float* W, uint32_t& upd) {
  if (STORAGE == kStorageColor) return;
  float px[4], py[4], pz[4];
  quad_points(F, m.v, r, px, py, pz);
  const int naz = F.width, nel = F.height;
  float2 rr[2], th[2], ph[2];
#pragma unroll
  for (int k = 0; k < 2; ++k)
    lidar_angles2(make_float2(px[2 * k], px[2 * k + 1]), make_float2(py[2 * k], py[2 * k + 1]),
                  make_float2(pz[2 * k], pz[2 * k + 1]), rr[k], th[k], ph[k]);
  if (FAST && !WEIGHTED && !m.lidar_nearest) {
    float2 fx[2], fy[2], d00[2], d10[2], d01[2], d11[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      // u = (theta - theta_start) alpha, rounded before 1/2 is taken off.  (The
      // compiler contracts a paired addition of the product, even one written
      // as add.rn.f32x2; this form it leaves alone, which the tests watch by
      // comparing with the scalar form below.)
      const float2 uu = __ffma2_rn(__fmul2_rn(__fadd2_rn(th[k], twice(-F.theta_start)), twice(F.alpha)), twice(1.0f), twice(-0.5f));
      const float2 vv = __ffma2_rn(__fmul2_rn(__fadd2_rn(ph[k], twice(-F.phi_start)), twice(F.beta)), twice(1.0f), twice(-0.5f));
      const float2 tu = __fadd2_rd(uu, twice(kFloorMagic)), tv = __fadd2_rd(vv, twice(kFloorMagic));
      fx[k] = __ffma2_rn(__fadd2_rn(tu, twice(-kFloorMagic)), twice(-1.0f), uu);  // uu - floor(uu), exact floor
      fy[k] = __ffma2_rn(__fadd2_rn(tv, twice(-kFloorMagic)), twice(-1.0f), vv);
      float q[2][4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k0 = (int)(__float_as_uint(h ? tu.y : tu.x) - kFloorBits);
        const int j0 = (int)(__float_as_uint(h ? tv.y : tv.x) - kFloorBits);
        const bool ok = (h ? rr[k].y : rr[k].x) > 0.0f && (uint32_t)j0 < (uint32_t)(nel - 1) &&
                        (uint32_t)(k0 + 1) <= (uint32_t)(naz + 1);
        q[h][0] = q[h][1] = q[h][2] = q[h][3] = __int_as_float(0x7fc00000);  // no cell: not valid
        if (ok) {
          const int c0 = wrap_az(k0, naz), c1 = c0 + 1 == naz ? 0 : c0 + 1;
          const float* row0 = F.depth + j0 * naz;
          const float* row1 = row0 + naz;
          q[h][0] = __ldg(row0 + c0);
          q[h][1] = __ldg(row0 + c1);
          q[h][2] = __ldg(row1 + c0);
          q[h][3] = __ldg(row1 + c1);
        }
      }
      d00[k] = make_float2(q[0][0], q[1][0]);
      d10[k] = make_float2(q[0][1], q[1][1]);
      d01[k] = make_float2(q[0][2], q[1][2]);
      d11[k] = make_float2(q[0][3], q[1][3]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      bool ok[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float a = h ? d00[k].y : d00[k].x, b = h ? d10[k].y : d10[k].x, c = h ? d01[k].y : d01[k].x,
                    e = h ? d11[k].y : d11[k].x;
        const float hi = max_nan(max_nan(a, b), max_nan(c, e)), lo = min_nan(min_nan(a, b), min_nan(c, e));
        ok[h] = lo >= F.min_range && hi <= F.max_range && !(__fsub_rn(hi, lo) > m.guard);
      }
      if (!(ok[0] || ok[1])) continue;
      const float2 top = __ffma2_rn(fx[k], __ffma2_rn(d00[k], twice(-1.0f), d10[k]), d00[k]);
      const float2 bot = __ffma2_rn(fx[k], __ffma2_rn(d01[k], twice(-1.0f), d11[k]), d01[k]);
      const float2 d = __ffma2_rn(fy[k], __ffma2_rn(top, twice(-1.0f), bot), top);
      const float2 dp = __ffma2_rn(rr[k], twice(-1.0f), d);
      ok[0] = ok[0] && !(dp.x < -m.tau);
      ok[1] = ok[1] && !(dp.y < -m.tau);
      const int i = 2 * k;
      if (STORAGE == kStorageOcc) {
        if (ok[0]) apply<STORAGE, false>(m, D[i], W[i], rr[k].x, dp.x);
        if (ok[1]) apply<STORAGE, false>(m, D[i + 1], W[i + 1], rr[k].y, dp.y);
      } else {
        update_pair(m, D + i, W + i, dp, ok[0], ok[1]);
      }
      upd += (ok[0] ? 1u : 0u) + (ok[1] ? 1u : 0u);
    }
    return;
  }
  float fx[4], fy[4], d00[4], d10[4], d01[4], d11[4];
  bool ok[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float rri = (i & 1) ? rr[i >> 1].y : rr[i >> 1].x;
    const float u = __fmul_rn(__fsub_rn((i & 1) ? th[i >> 1].y : th[i >> 1].x, F.theta_start), F.alpha);
    const float v = __fmul_rn(__fsub_rn((i & 1) ? ph[i >> 1].y : ph[i >> 1].x, F.phi_start), F.beta);
    ok[i] = rri > 0.0f;
    d00[i] = d10[i] = d01[i] = d11[i] = 0.0f;
    if (m.lidar_nearest) {
      const float ku = floorf(u), jv = floorf(v);
      fx[i] = fy[i] = 0.0f;
      ok[i] = ok[i] && jv >= 0.0f && jv <= (float)(nel - 1) && ku >= -1.0f && ku <= (float)naz;
      if (ok[i]) d00[i] = __ldg(F.depth + (int)jv * naz + wrap_az((int)ku, naz));
    } else {
      const float uu = __fsub_rn(u, 0.5f), vv = __fsub_rn(v, 0.5f);
      const float k0f = floorf(uu), j0f = floorf(vv);
      fx[i] = __fsub_rn(uu, k0f);
      fy[i] = __fsub_rn(vv, j0f);
      ok[i] = ok[i] && j0f >= 0.0f && j0f <= (float)(nel - 2) && k0f >= -1.0f && k0f <= (float)naz;
      if (ok[i]) {
        const int k0 = wrap_az((int)k0f, naz), k1 = k0 + 1 == naz ? 0 : k0 + 1;
        const float* row0 = F.depth + (int)j0f * naz;
        const float* row1 = row0 + naz;
        d00[i] = __ldg(row0 + k0);
        d10[i] = __ldg(row0 + k1);
        d01[i] = __ldg(row1 + k0);
        d11[i] = __ldg(row1 + k1);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (!ok[i]) continue;
    const float rri = (i & 1) ? rr[i >> 1].y : rr[i >> 1].x;
    float d;
    if (m.lidar_nearest) {
      d = d00[i];
      if (!lidar_valid(F, d)) continue;
    } else {
      if (!(lidar_valid(F, d00[i]) && lidar_valid(F, d10[i]) && lidar_valid(F, d01[i]) &&
            lidar_valid(F, d11[i])))
        continue;
      const float hi = fmaxf(fmaxf(d00[i], d10[i]), fmaxf(d01[i], d11[i]));
      const float lo = fminf(fminf(d00[i], d10[i]), fminf(d01[i], d11[i]));
      if (__fsub_rn(hi, lo) > m.guard) continue;
      const float top = __fmaf_rn(fx[i], __fsub_rn(d10[i], d00[i]), d00[i]);
      const float bot = __fmaf_rn(fx[i], __fsub_rn(d11[i], d01[i]), d01[i]);
      d = __fmaf_rn(fy[i], __fsub_rn(bot, top), top);
    }
    const float dp = __fsub_rn(d, rri);
    if (dp < -m.tau) continue;
    apply<STORAGE, WEIGHTED>(m, D[i], W[i], rri, dp);
    ++upd;
  }
}

// Shared memory of the integration workers of a CTA.
constexpr int kRing = 8;  // entries in hand
template <int NF, int NM>
struct IntegSmem {
  uint32_t begin[NM + 1];         // first entry of each map's list in the batch's work
  unsigned long long upd[NM];     // voxel updates per map
  unsigned long long pairs[NM];   // (block, frame) pairs per map
  uint32_t ticket;                // slabs handed out
  uint32_t seq[kRing];            // sequence number of the entry in a ring slot
  uint32_t entry[kRing];
  uint32_t done[kRing];           // slabs finished in the slot's entries, all together
  FrameProj fp[NF];
};

// Wait until *a == value (a shared-memory word that another warp of the CTA
// sets without waiting for this one); false after 2^22 polls.
__device__ __forceinline__ bool poll_shared(const uint32_t* a, uint32_t value) {
  for (int i = 0; i < (1 << 22); ++i)
    if (*(const volatile uint32_t*)a == value) {
      __threadfence_block();
      return true;
    }
  return false;
}

// Entry metadata: COHERENT loads bypass L1, for a kernel that reads
// metadata that other CTAs of the same launch wrote.
template <bool COHERENT, class T>
__device__ __forceinline__ T meta_load(const T* a) {
  if (COHERENT) return __ldcg(a);
  return *a;
}

// The integration of a batch's work list: every entry is a hash slot met by
// some frames of the batch; its block's 512 voxels are held in registers (4
// per thread) across those frames, in batch order, and written back once.
//
// A block is four slabs of 128 voxels, one per warp, and warps take slabs by
// ticket: four consecutive tickets are one entry, so a block's slabs run on
// one SM at about the same time (their depth gathers share L1 lines), and no
// warp waits for another to finish a block (a CTA barrier per entry cost 16 %
// of the warps' time).  The warp that takes an entry's first slab fetches the
// next entry (handed out dynamically: blocks differ in their frame counts)
// into a ring of kRing slots; a slot is free once the four slabs of its last
// entry are done.  Tickets go out in order and an entry's slabs depend on no
// later one, so both waits end; they are bounded all the same (BatchParams::
// wait_extra withholds the first entry to see that).  The warp that finishes
// an entry's last slab clears its mask (every slab has read it by then).  The
// last CTA to finish resets every map's work list.
template <int NF, int NM, bool COHERENT, int STORAGE, bool PINHOLE_ONLY, bool WEIGHTED, bool FAST>
__device__ __forceinline__ void integrate_entries(const BatchParams<NF, NM>& p, IntegSmem<NF, NM>& sm,
                                                  bool wait) {
  if (threadIdx.x < NM) sm.upd[threadIdx.x] = sm.pairs[threadIdx.x] = 0ull;
  for (int f = threadIdx.x; f < p.n_frames; f += blockDim.x)
    if (p.fr[f].kind == kSensorPinhole) stage_frame(p.fr[f], sm.fp[f]);
  if (threadIdx.x < kRing) {
    sm.seq[threadIdx.x] = threadIdx.x || p.wait_extra ? 0xFFFFFFFFu : 0u;
    sm.entry[threadIdx.x] = blockIdx.x;
    sm.done[threadIdx.x] = 0u;
  }
  // nothing above reads memory that the stream's previous kernel may write
  if (wait) wait_prev_grid();
  if (threadIdx.x == 0) {
    sm.ticket = 0u;
    // the batch's work = the concatenation of every map's list
    uint32_t acc = 0;
    for (int k = 0; k < p.n_maps; ++k) {
      sm.begin[k] = acc;
      acc += min(__ldcg(p.maps[k].ctl), p.maps[k].list_cap);
    }
    sm.begin[p.n_maps] = acc;
  }
  __syncthreads();
  const uint32_t n = sm.begin[p.n_maps];
  // a CTA's first entry is its own index: one beyond the list has none and is
  // not counted below (CTA 0 always is).  A CTA that starts late may read the
  // list as already reset: then it was not counted either.  (In the fused
  // kernel every CTA is counted: the reset ends the grid wait's count, so it
  // has to come after every CTA has left the wait.)
  if (!COHERENT && blockIdx.x >= n && blockIdx.x != 0) return;
  const uint32_t ctas = COHERENT ? gridDim.x : max(1u, min(n, gridDim.x));
  const int lane = threadIdx.x & 31;

  for (;;) {
    uint32_t k = 0, e = 0;
    bool ok = true;
    if (lane == 0) {
      k = atomicAdd(&sm.ticket, 1u);
      ok = poll_shared(&sm.seq[(k >> 2) % kRing], k >> 2);
      e = *(const volatile uint32_t*)&sm.entry[(k >> 2) % kRing];
    }
    k = __shfl_sync(0xffffffffu, k, 0);
    e = __shfl_sync(0xffffffffu, e, 0);
    const uint32_t seq = k >> 2, next = seq + 1;
    // the next entry, asked for now and published once this one's voxels are requested
    uint32_t fetched = e;
    if ((k & 3u) == 0u && lane == 0 && e < n) fetched = gridDim.x + atomicAdd(p.maps[0].ctl + 2, 1u);
    int mi = 0, pool = -1;
    uint32_t slot = 0, bits = 0;
    float D[4], W[4], G4[4], B[4];
    VoxelQuad vq;
    const bool work = e < n && __all_sync(0xffffffffu, ok);
    // this thread's voxels: x = 2 (lane & 3) and the next, y = lane >> 2, z = 2 slab and the next
    vq.at = (int)(k & 3u) * 64 + lane;
    if (work) {
      if (NM > 1)
        while (mi + 1 < p.n_maps && e >= sm.begin[mi + 1]) ++mi;
      const MapDev& m = NM == 1 ? p.maps[0] : p.maps[mi];
      slot = meta_load<COHERENT>(m.list + (e - sm.begin[mi]));
      const int val = meta_load<COHERENT>(m.vals + slot);
      bits = meta_load<COHERENT>(m.mask + slot);
      const unsigned long long slot_key = meta_load<COHERENT>(m.keys + slot);
      pool = val <= -2 ? -val - 2 : val;
      if (val < 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) { D[i] = 0.0f; W[i] = 0.0f; G4[i] = 0.0f; B[i] = 0.0f; }
      } else {
        Voxels4<STORAGE>::load(m, pool, vq.at, D, W, G4, B);
      }
      vq.x = (float)(key_coord(slot_key, 0) * 8 + 2 * (lane & 3));
      vq.y = (float)(key_coord(slot_key, 1) * 8 + (lane >> 2));
      vq.z = (float)(key_coord(slot_key, 2) * 8 + 2 * (int)(k & 3u));
    }
    if ((k & 3u) == 0u && lane == 0) {
      if (!poll_shared(&sm.done[next % kRing], 4u * (next / kRing))) ok = false;
      sm.entry[next % kRing] = fetched;
      __threadfence_block();
      *(volatile uint32_t*)&sm.seq[next % kRing] = next;
    }
    if (!__all_sync(0xffffffffu, ok)) {
      // some of the batch's entries are left out, whichever map they are in
      if (lane == 0)
        for (int i = 0; i < p.n_maps; ++i) atomicOr(p.maps[i].counters + kCntStatus, (unsigned long long)kStTimeout);
      break;
    }
    if (!work) break;
    const MapDev& m = NM == 1 ? p.maps[0] : p.maps[mi];
    uint32_t my_upd = 0;
    if (pool >= 0) {
      while (bits) {
        // bit k of the mask is frame k of the batch; frames apply in batch
        // order.  Two consecutive pinhole frames issue all their depth loads
        // before the first update (longer runs measured slower: the unrolled
        // code outgrows the instruction cache).
        int fq[2];
        int nq = 0;
        bool go = true;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          fq[q] = -1;
          if (go && bits) {
            const int f = __ffs(bits) - 1;
            if (PINHOLE_ONLY || p.fr[f].kind == kSensorPinhole) {
              fq[q] = f;
              ++nq;
              bits &= bits - 1u;
            } else {
              go = false;
            }
          }
        }
        if (NF > 1 && nq == 2)
          fuse_pinhole<2, STORAGE, WEIGHTED, FAST>(p, sm.fp, fq, m, vq, D, W, G4, B, my_upd);
        else if (nq >= 1)
          fuse_pinhole<1, STORAGE, WEIGHTED, FAST>(p, sm.fp, fq, m, vq, D, W, G4, B, my_upd);
        else if (!PINHOLE_ONLY) {
          const int f = __ffs(bits) - 1;  // a LiDAR frame
          bits &= bits - 1u;
          fuse_lidar<STORAGE, WEIGHTED, FAST>(p.fr[f], m, vq, D, W, my_upd);
        }
      }
      Voxels4<STORAGE>::store(m, pool, vq.at, D, W, G4, B);
    }
    // per-map update count; the entry's last slab clears its metadata
    my_upd = __reduce_add_sync(0xffffffffu, my_upd);
    if (lane == 0) {
      if (my_upd) atomicAdd(&sm.upd[mi], (unsigned long long)my_upd);
      __threadfence_block();
      if (atomicAdd(&sm.done[seq % kRing], 1u) == 4u * (seq / kRing) + 3u) {
        atomicAdd(&sm.pairs[mi], (unsigned long long)__popc(meta_load<COHERENT>(m.mask + slot)));
        m.mask[slot] = 0u;
        if (pool >= 0) {
          m.vals[slot] = pool;  // no longer new
          if (m.dirty) m.dirty[pool] = kDirtyEsdf | kDirtyMesh;
        }
      }
    }
  }
  if (p.overlap) allow_next_grid();
  __syncthreads();
  if (threadIdx.x < p.n_maps && sm.upd[threadIdx.x])
    atomicAdd(p.maps[threadIdx.x].counters + kCntUpdates, sm.upd[threadIdx.x]);
  if (threadIdx.x < p.n_maps && sm.pairs[threadIdx.x])
    atomicAdd(p.maps[threadIdx.x].counters + kCntPairs, sm.pairs[threadIdx.x]);
  // the last CTA to finish resets every map's work list for the next batch
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned done = atomicAdd(p.maps[0].ctl + 1, 1u);
    if (done == ctas - 1) {
      for (int k = 0; k < p.n_maps; ++k) {
        atomicAdd(p.maps[k].counters + kCntVisits, (unsigned long long)(sm.begin[k + 1] - sm.begin[k]));
        atomicAdd(p.maps[k].counters + kCntLaunches, 1ull);
        p.maps[k].ctl[0] = 0u;
      }
      p.maps[0].ctl[1] = 0u;
      p.maps[0].ctl[2] = 0u;
      p.maps[0].ctl[3] = 0u;  // the fused kernel's barrier count
    }
  }
}

template <int NF, int NM, int STORAGE, bool PINHOLE_ONLY, bool WEIGHTED, bool FAST = false>
__global__ void __launch_bounds__(kIntegrateThreads, STORAGE == kStorageColor ? 6 : 7)
    integrate_kernel(const __grid_constant__ BatchParams<NF, NM> p) {
  __shared__ IntegSmem<NF, NM> sm;
  integrate_entries<NF, NM, false, STORAGE, PINHOLE_ONLY, WEIGHTED, FAST>(p, sm, p.overlap != 0);
}

// ------------------------------------------- one launch per batch (fused)

// Bounded waits give up after this many nanoseconds of the global timer.
constexpr unsigned long long kWaitLimitNs = 1000000000ull;

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned int load_acquire(const unsigned int* a) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}

// Grid-wide barrier of a cooperative launch (all CTAs resident): thread 0 of
// every CTA arrives on *count, then waits until `expected` CTAs have arrived,
// for at most kWaitLimitNs.  A wait that runs out sets kStTimeout in *status
// (the map's sticky status) and makes the CTA return false.
__device__ __noinline__ bool grid_wait(unsigned int* count, unsigned int expected, unsigned long long* status) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(count, 1u);
    const unsigned long long t0 = global_ns();
    int ok = 1;
    while (load_acquire(count) < expected) {
      if (global_ns() - t0 > kWaitLimitNs) {
        atomicOr(status, (unsigned long long)kStTimeout);
        ok = 0;
        break;
      }
      __nanosleep(128);
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

constexpr int kFusedThreads = kAllocThreads;

template <int NF, int NM, int TH>
union FusedSmem {
  AllocSmem<TH> a;
  IntegSmem<NF, NM> i;
};

// Allocation and integration of one batch in one persistent, cooperative
// launch: the CTAs walk every allocation tile of the batch (grid-stride),
// meet at a bounded grid-wide wait (the integration reads the work list,
// slot masks and pool indices that every tile wrote), then integrate the
// work list.  Single-map
// batches, TSDF storage, constant weighting, no walk statistics.
// Four resident CTAs per SM (64 registers): the rig's fused step measured
// 16.1 ms per 1,000 frames against 18.2 ms with three.
template <int NF, int NM, int TH, int STORAGE, bool PINHOLE_ONLY, bool FAST>
__global__ void __launch_bounds__(kFusedThreads, 4)
    fused_kernel(const __grid_constant__ BatchParams<NF, NM> p) {
  __shared__ FusedSmem<NF, NM, TH> sm;
  for (int cta = blockIdx.x; cta < p.alloc_ctas; cta += gridDim.x)
    alloc_tile<NF, NM, TH, PINHOLE_ONLY, false, FAST, true>(p, tile_frame(p, cta), cta, sm.a, false);
  if (!grid_wait(p.maps[0].ctl + 3, gridDim.x + (unsigned)p.wait_extra, p.maps[0].counters + kCntStatus))
    return;  // timed out: integration skipped, the map reports TSDF_ERR_TIMEOUT
  __syncthreads();  // the tiles' shared memory is free for the integration
  integrate_entries<NF, NM, true, STORAGE, PINHOLE_ONLY, false, FAST>(p, sm.i, false);
}

template <int STORAGE>
__global__ void __launch_bounds__(kPointThreads)
    query_kernel(const MapDev m, const float* __restrict__ pts, int64_t n, float inv_v, bool vec,
                 float* __restrict__ dist, float* __restrict__ weight) {
  const int64_t i = (int64_t)blockIdx.x * kPointThreads + threadIdx.x;
  wait_prev_grid();
  allow_next_grid();
  if (kPointsPerThread * i >= n) return;
  float c[3 * kPointsPerThread], D[kPointsPerThread], W[kPointsPerThread];
  int pool[kPointsPerThread], l[kPointsPerThread];
  load_points(pts, i, n, vec, c);
  find_points(m, inv_v, c, pool, l);
#pragma unroll
  for (int k = 0; k < kPointsPerThread; ++k) {
    D[k] = W[k] = 0.0f;
    if (pool[k] < 0) continue;
    const size_t at = (size_t)pool[k] * 512 + l[k];
    if (STORAGE == kStorageOcc) {
      D[k] = reinterpret_cast<const float*>(m.pool)[at];
    } else if (STORAGE == kStorageF32) {
      const float2 v = reinterpret_cast<const float2*>(m.pool)[at];
      D[k] = v.x;
      W[k] = v.y;
    } else if (STORAGE == kStorageX16) {
      const uint32_t w = reinterpret_cast<const uint32_t*>(m.pool)[at];
      D[k] = x16_dist(w, m.x16_unit);
      W[k] = x16_weight(w);
    } else {
      const __half2 h = reinterpret_cast<const __half2*>(m.pool)[at];
      D[k] = __low2float(h) * m.tau;
      W[k] = __high2float(h);
    }
  }
  store_points(dist, i, n, vec, D);
  store_points(weight, i, n, vec, W);
}

// Colour of the voxel holding each point: r, g, b and the colour weight;
// zeros where no block or no colour update exists.
__global__ void __launch_bounds__(kPointThreads)
    query_color_kernel(const MapDev m, const float* __restrict__ pts, int64_t n, float inv_v, bool vec,
                       float* __restrict__ rgb, float* __restrict__ weight) {
  const int64_t i = (int64_t)blockIdx.x * kPointThreads + threadIdx.x;
  wait_prev_grid();
  allow_next_grid();
  if (kPointsPerThread * i >= n) return;
  float c[3 * kPointsPerThread], W[kPointsPerThread];
  float4 out[kPointsPerThread];
  int pool[kPointsPerThread], l[kPointsPerThread];
  load_points(pts, i, n, vec, c);
  find_points(m, inv_v, c, pool, l);
#pragma unroll
  for (int k = 0; k < kPointsPerThread; ++k) {
    out[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (pool[k] >= 0) out[k] = reinterpret_cast<const float4*>(m.pool)[(size_t)pool[k] * 512 + l[k]];
    W[k] = out[k].w;
  }
  if (vec && kPointsPerThread * (i + 1) <= n) {
    float4* o = reinterpret_cast<float4*>(rgb) + 3 * i;
    __stcs(o, make_float4(out[0].x, out[0].y, out[0].z, out[1].x));
    __stcs(o + 1, make_float4(out[1].y, out[1].z, out[2].x, out[2].y));
    __stcs(o + 2, make_float4(out[2].z, out[3].x, out[3].y, out[3].z));
  } else {
#pragma unroll
    for (int k = 0; k < kPointsPerThread; ++k)
      if (kPointsPerThread * i + k < n) {
        float* o = rgb + 3 * (kPointsPerThread * i + k);
        o[0] = out[k].x;
        o[1] = out[k].y;
        o[2] = out[k].z;
      }
  }
  store_points(weight, i, n, vec, W);
}

// Occupancy decay over every allocated block: log-odds above 0 drop by
// d_occ, below 0 rise by d_free, neither crossing 0.  The pool's first
// min(blocks, max_blocks) blocks are exactly the allocated ones; a thread
// handles four voxels (one 16-byte word) per step of a grid-stride loop.
__global__ void decay_kernel(const MapDev m, float d_occ, float d_free) {
  wait_prev_grid();
  allow_next_grid();
  const unsigned long long nb =
      min((unsigned long long)m.max_blocks, __ldcg(m.counters + kCntBlocks));
  const size_t n4 = (size_t)nb * 128;
  float4* pool = reinterpret_cast<float4*>(m.pool);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
       i += (size_t)gridDim.x * blockDim.x) {
    float4 l = pool[i];
    const float4 before = l;
    float* c = &l.x;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      c[k] = c[k] > 0.0f ? fmaxf(c[k] - d_occ, 0.0f) : (c[k] < 0.0f ? fminf(c[k] + d_free, 0.0f) : c[k]);
    pool[i] = l;
    // a changed block is due for the next ESDF update and mesh extraction
    // (all writers of a block's flag byte set the same bits)
    if (m.dirty && (l.x != before.x || l.y != before.y || l.z != before.z || l.w != before.w))
      m.dirty[i / 128] |= kDirtyEsdf | kDirtyMesh;
  }
}

// Empty a map: hash slots, every mask set, changed flags, counters and
// control words in one launch, four slots or 16 flags per thread and step in
// 16-byte stores.  One kernel and three memsets before cost a step over 16
// maps four launches a map (85 us of its 1,040 us).
__global__ void reset_kernel(const MapDev m, uint32_t cap, const MoreSets more) {
  const uint32_t first = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  const uint4 ones = make_uint4(~0u, ~0u, ~0u, ~0u), zero = make_uint4(0u, 0u, 0u, 0u);
  static_assert(kEmptyKey == ~0ull, "an empty key is all ones");
  wait_prev_grid();
  allow_next_grid();
  for (uint32_t i = first; i < cap / 4; i += step) {
    reinterpret_cast<uint4*>(m.keys)[2 * i] = ones;
    reinterpret_cast<uint4*>(m.keys)[2 * i + 1] = ones;
    reinterpret_cast<uint4*>(m.vals)[i] = ones;  // -1 each
    reinterpret_cast<uint4*>(m.mask)[i] = zero;
#pragma unroll
    for (int k = 0; k < kSets - 1; ++k) reinterpret_cast<uint4*>(more.mask[k])[i] = zero;
  }
  for (uint32_t i = cap / 4 * 4 + first; i < cap; i += step) {  // a table of two slots
    m.keys[i] = kEmptyKey;
    m.vals[i] = -1;
    m.mask[i] = 0u;
    for (int k = 0; k < kSets - 1; ++k) more.mask[k][i] = 0u;
  }
  const uint32_t nd = (uint32_t)m.max_blocks;
  for (uint32_t i = first; i < nd / 16; i += step) reinterpret_cast<uint4*>(m.dirty)[i] = zero;
  for (uint32_t i = nd / 16 * 16 + first; i < nd; i += step) m.dirty[i] = 0;
  if (first < kNumCounters) m.counters[first] = 0ull;
  if (first < 4) {
    m.ctl[first] = 0u;
    for (int k = 0; k < kSets - 1; ++k) more.ctl[k][first] = 0u;
  }
}

}  // namespace

// True when every frame of the batch is a pinhole camera: the kernels are
// then launched without their LiDAR code (smaller, fewer branches).
template <int NF, int NM>
bool pinhole_only(const BatchParams<NF, NM>& p) {
  for (int f = 0; f < p.n_frames; ++f)
    if (p.fr[f].kind != kSensorPinhole) return false;
  return true;
}

// Every frame's band segments meet fewer than kMaxCells blocks (host check).
template <int NF, int NM>
bool short_walks(const BatchParams<NF, NM>& p) {
  for (int f = 0; f < p.n_frames; ++f)
    if (!p.fr[f].short_walks) return false;
  return true;
}

// Launch kernel k; with p.overlap as a programmatic dependent launch.
template <class P>
cudaError_t launch_k(void (*k)(P), dim3 g, dim3 b, cudaStream_t s, const P& p) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = g;
  cfg.blockDim = b;
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = p.overlap ? at : nullptr;
  cfg.numAttrs = p.overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, p);
}

// Patch tiles where every frame passes the host's checks and the launch has
// enough pixels to fill the chip with them.  A patch tile's stages (walk, two
// tests, walk, claim) run one after the other, so a launch takes at least
// about 20 us: one 640x480 frame 22 us against 12 us by rows, eight frames 28
// against 32, 32 frames 48 against 99, 24 frames of 1280x720 at 5 cm voxels
// 61 against 184; the lines cross near kPatchPixels.
//
// And where a patch's pixels mostly share their blocks: `span` is the pixels
// that a voxel covers at one metre, |f| v.  Below 5 the test fails nearly
// everywhere at room distances, and below 1 cm a tile's window (32 blocks,
// 2.6 m) does not hold a room's depths either, so that only large images or
// launches gain (us, rows against patches; 32 frames of 640x480 unless said):
//   1 cm     107 /  86     320x240 at 1.25 cm  45 /  55     at 1 cm  44 / 64
//   7.5 mm   118 / 141     1280x720 x 16      145 / 118
//   5 mm     131 / 213     1280x720 x 16      155 / 196
//                          1920x1080 x 8      161 / 150     one      32 / 60
//                          3840x2160 x 2      154 / 120     one      81 / 78
//   3 mm                   3840x2160 x 2      163 / 156     one      88 / 101
// Scenes deeper than a room at fine voxels still lose (2 cm, an open lot to 20
// m: 96 / 130): the host does not see depths.
constexpr float kFineVoxel = 0.0099f;   // m
constexpr float kPatchSpan = 5.0f;      // least span of voxels from kFineVoxel up,
constexpr float kFineSpan = 15.0f;      // of finer ones,
constexpr float kFineSpanLarge = 7.5f;  // of finer ones in launches of kFinePixels or more
constexpr int64_t kFinePixels = 10000000;
inline bool patches_share_blocks(float span, float v, int64_t pixels) {
  if (v >= kFineVoxel) return span >= kPatchSpan;
  return span >= (pixels >= kFinePixels ? kFineSpanLarge : kFineSpan);
}

template <int NF, int NM>
AllocShape pick_alloc_shape(const BatchParams<NF, NM>& p, int tile_h) {
  bool pinhole = false, ok = true;
  int64_t pixels = 0, tiny_tiles = 0;
  for (int k = 0; k < p.n_maps; ++k) ok = ok && !p.maps[k].walk_stats;
  for (int f = 0; f < p.n_frames; ++f) {
    const FrameDev& F = p.fr[f];
    ok = ok && F.fast_rcp && F.short_walks;
    pinhole = pinhole || F.kind == kSensorPinhole;
    pixels += (int64_t)F.width * F.height;
    tiny_tiles += (int64_t)((F.width + kTileW - 1) / kTileW) * ((F.height + kTileHTiny - 1) / kTileHTiny);
  }
  bool patches = ok && pinhole && (tile_h ? tile_h == kTileHBig : pixels >= kPatchPixels);
  for (int f = 0; patches && !tile_h && f < p.n_frames; ++f) {
    const FrameDev& F = p.fr[f];
    const float v = p.maps[NM == 1 ? 0 : F.map].v;
    if (F.kind == kSensorPinhole) patches = patches_share_blocks(std::min(std::fabs(F.fu), std::fabs(F.fv)) * v, v, pixels);
  }
  if (patches) return AllocShape{kPatchTile, kTileHTiny};
  const bool big = tile_h ? tile_h == kTileHBig : pixels >= kBigTilePixels;
  // Tiles of 8 rows walk one pixel per thread instead of two: less latency
  // where they still fit one wave (a 64x48 call 16.5 -> 14.5 us, 640x480
  // calls 119 -> 116 us for eight, a 1024x64 scan 57.4 -> 53.1), more claims
  // per pixel where they do not (848x480: 80 -> 88 us for four calls).
  if (ok && !tile_h && tiny_tiles <= kOneWave) return AllocShape{0, kTileHTiny};
  return AllocShape{0, big ? kTileHBig : kTileHSmall};
}

template <int NF, int NM>
cudaError_t launch_band_alloc(const BatchParams<NF, NM>& p, int n_ctas, AllocShape shape, cudaStream_t s) {
  if (n_ctas <= 0) return cudaSuccess;
  const bool ph = pinhole_only(p);
  const dim3 g(n_ctas), b(kAllocThreads);
  if (shape.patch)
    return ph ? launch_k(patch_alloc_kernel<NF, NM, false>, g, b, s, p)
              : launch_k(patch_alloc_kernel<NF, NM, true>, g, b, s, p);
  const bool big = shape.row_h == kTileHBig;
  bool st = false;
  for (int k = 0; k < p.n_maps; ++k) st = st || p.maps[k].walk_stats != 0;
  if (st)  // diagnostics: one generic variant per tile height
    return big ? launch_k(band_alloc_kernel<NF, NM, kTileHBig, false, true, false, true>, g, b, s, p)
               : launch_k(band_alloc_kernel<NF, NM, kTileHSmall, false, true, false, true>, g, b, s, p);
  if (!short_walks(p))  // segments that may reach the cap: one generic variant per tile height
    return big ? launch_k(band_alloc_kernel<NF, NM, kTileHBig, false, false, false, true>, g, b, s, p)
               : launch_k(band_alloc_kernel<NF, NM, kTileHSmall, false, false, false, true>, g, b, s, p);
  const bool fast = p.fast_rcp != 0;
  if (shape.row_h == kTileHTiny)  // every frame passed the host's checks (pick_alloc_shape)
    return ph ? launch_k(band_alloc_kernel<NF, NM, kTileHTiny, true, false, true, false>, g, b, s, p)
              : launch_k(band_alloc_kernel<NF, NM, kTileHTiny, false, false, true, false>, g, b, s, p);
  if (big) {
    if (ph) return fast ? launch_k(band_alloc_kernel<NF, NM, kTileHBig, true, false, true, false>, g, b, s, p)
                        : launch_k(band_alloc_kernel<NF, NM, kTileHBig, true, false, false, false>, g, b, s, p);
    return fast ? launch_k(band_alloc_kernel<NF, NM, kTileHBig, false, false, true, false>, g, b, s, p)
                : launch_k(band_alloc_kernel<NF, NM, kTileHBig, false, false, false, false>, g, b, s, p);
  }
  if (ph) return fast ? launch_k(band_alloc_kernel<NF, NM, kTileHSmall, true, false, true, false>, g, b, s, p)
                      : launch_k(band_alloc_kernel<NF, NM, kTileHSmall, true, false, false, false>, g, b, s, p);
  return fast ? launch_k(band_alloc_kernel<NF, NM, kTileHSmall, false, false, true, false>, g, b, s, p)
              : launch_k(band_alloc_kernel<NF, NM, kTileHSmall, false, false, false, false>, g, b, s, p);
}

// Launch integration kernel k on a persistent grid: per_sm CTAs per SM (the
// map's knob), or if that is 0 as many as can be resident with this variant's
// registers, at most `limit` (0: no limit).  Pinhole launches (not colour) are
// limited.  In a batch of many frames an entry is long work, and with every SM
// full of entries half of them are started at once and the chip drains
// unevenly (32 frames of 640x480, us per launch with 3, 4, 5, 7 and 9 CTAs per
// SM: 56.6, 55.1, 55.3, 61.8, 61.4); a single frame's launch leaves room for the
// next call's allocation, which starts while it drains (eight 640x480 calls,
// us in all with 3, 4, 5, 6, 7: 126.5, 120.1, 120.4, 123.8, 125.5).  LiDAR scans
// want every warp (four scans with 4, 5, 6, 7: 271, 252, 242, 231 us), and so do
// maps of fine voxels, whose lists are ten thousand entries and more (with 5 and
// 7, us: 32 frames of 640x480 at 1.25 cm 109 and 109, at 1 cm 147 and 143, at 5
// mm 686 and 650; one 1920x1080 frame at 1.25 cm 18 and 18, at 1 cm 22 and 19, at 5
// mm 75 and 61).
constexpr int kPinholePerSm = 5;
constexpr float kLimitVoxel = 0.011f;  // least voxel edge with the limit, m
template <class P>
cudaError_t launch_persistent(void (*k)(P), int per_sm, int limit, cudaStream_t s, const P& p,
                              std::atomic<int>& fit) {
  int n = fit.load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, kIntegrateThreads, 0) != cudaSuccess || n <= 0) {
      cudaGetLastError();
      n = 4;
    }
    fit.store(n, std::memory_order_relaxed);
  }
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return cudaGetLastError();
  if (per_sm > 0) n = std::min(n, per_sm);
  else if (limit > 0) n = std::min(n, limit);
  return launch_k(k, dim3(std::max(1, sms) * n), dim3(kIntegrateThreads), s, p);
}

template <int NF, int NM, int STORAGE, bool PINHOLE_ONLY, bool WEIGHTED, bool FAST>
cudaError_t launch_variant(const BatchParams<NF, NM>& p, int per_sm, int limit, cudaStream_t s) {
  static std::atomic<int> fit{0};  // resident CTAs per SM of this variant (all devices are alike here)
  return launch_persistent(integrate_kernel<NF, NM, STORAGE, PINHOLE_ONLY, WEIGHTED, FAST>, per_sm, limit, s, p, fit);
}

template <int NF, int NM>
cudaError_t launch_integrate(const BatchParams<NF, NM>& p, int per_sm, cudaStream_t s) {
  // all maps of a batch share one storage type (checked by the host API)
  // colour maps take pinhole frames only (checked by the host API)
  const bool ph = pinhole_only(p);
  const int st = p.maps[0].storage;
  // the weighted update with weighting 0 is the constant-weight update, so
  // one weighted map selects the weighted kernel for the whole batch
  bool wt = false;
  for (int k = 0; k < p.n_maps; ++k) wt = wt || p.maps[k].weighting != 0;
  // FAST: pinhole reciprocals by rcp_dec<true> (the host checked their range)
  const bool fast = p.fast_rcp != 0;
  float v = p.maps[0].v;
  for (int k = 1; k < p.n_maps; ++k) v = std::min(v, p.maps[k].v);
  const int limit = ph && st != kStorageColor && v >= kLimitVoxel ? kPinholePerSm : 0;
#define GBT_INTEG(ST, PH) \
  (fast ? launch_variant<NF, NM, ST, PH, false, true>(p, per_sm, limit, s) \
        : launch_variant<NF, NM, ST, PH, false, false>(p, per_sm, limit, s))
  // weighted maps: pinhole batches with fast reciprocals leave the LiDAR code
  // and the IEEE reciprocals out too (24 frames of 1280x720: 39.0 -> 34.2 us)
#define GBT_WEIGHTED(ST) \
  (ph && fast ? launch_variant<NF, NM, ST, true, true, true>(p, per_sm, limit, s) \
              : launch_variant<NF, NM, ST, false, true, false>(p, per_sm, limit, s))
  if (st == kStorageColor) return GBT_INTEG(kStorageColor, true);
  if (st == kStorageOcc) return ph ? GBT_INTEG(kStorageOcc, true) : GBT_INTEG(kStorageOcc, false);
  if (st == kStorageX16) {
    if (wt) return GBT_WEIGHTED(kStorageX16);
    return ph ? GBT_INTEG(kStorageX16, true) : GBT_INTEG(kStorageX16, false);
  }
  if (st == kStorageF16) {
    if (wt) return GBT_WEIGHTED(kStorageF16);
    return ph ? GBT_INTEG(kStorageF16, true) : GBT_INTEG(kStorageF16, false);
  }
  if (wt) return GBT_WEIGHTED(kStorageF32);
  return ph ? GBT_INTEG(kStorageF32, true) : GBT_INTEG(kStorageF32, false);
#undef GBT_INTEG
#undef GBT_WEIGHTED
}

// The fused kernel of a tile height for a storage and sensor mix, launched
// cooperatively with as many CTAs as can be resident at once.
template <int NF, int NM, int TH>
cudaError_t launch_fused_th(const BatchParams<NF, NM>& p, int st, bool ph, cudaStream_t s) {
  void (*k)(BatchParams<NF, NM>) = nullptr;
  const bool fast = p.fast_rcp != 0;
#define GBT_FUSED(ST) \
  (ph ? (fast ? fused_kernel<NF, NM, TH, ST, true, true> : fused_kernel<NF, NM, TH, ST, true, false>) \
      : (fast ? fused_kernel<NF, NM, TH, ST, false, true> : fused_kernel<NF, NM, TH, ST, false, false>))
  int si = 0;
  if (st == kStorageF32) {
    k = GBT_FUSED(kStorageF32);
    si = 0;
  } else if (st == kStorageF16) {
    k = GBT_FUSED(kStorageF16);
    si = 1;
  } else {
    k = GBT_FUSED(kStorageX16);
    si = 2;
  }
#undef GBT_FUSED
  static int per_sm[3][2][2] = {};  // resident CTAs per SM of each variant (all devices are alike here)
  int& n = per_sm[si][ph ? 1 : 0][fast ? 1 : 0];
  if (n == 0 && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, kFusedThreads, 0) != cudaSuccess) {
    n = 0;
    return cudaGetLastError();
  }
  if (n <= 0) return cudaErrorNotSupported;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return cudaGetLastError();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n * sms);
  cfg.blockDim = dim3(kFusedThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;  // every CTA resident: the grid-wide wait can complete
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, p);
}

template <int NF, int NM>
cudaError_t launch_fused(const BatchParams<NF, NM>& p, int tile_h, cudaStream_t s) {
  const MapDev& m0 = p.maps[0];
  if (NM != 1 || p.n_maps != 1 || p.overlap || m0.walk_stats || m0.weighting != 0) return cudaErrorNotSupported;
  const int st = m0.storage;
  if (st != kStorageF32 && st != kStorageF16 && st != kStorageX16) return cudaErrorNotSupported;
  if (p.alloc_ctas <= 0) return cudaErrorNotSupported;
  const bool ph = pinhole_only(p);
  return tile_h == kTileHBig ? launch_fused_th<NF, NM, kTileHBig>(p, st, ph, s)
                             : launch_fused_th<NF, NM, kTileHSmall>(p, st, ph, s);
}

template cudaError_t launch_fused<kMaxFrames, 1>(const BatchParams<kMaxFrames, 1>&, int, cudaStream_t);
template AllocShape pick_alloc_shape<1, 1>(const BatchParams<1, 1>&, int);
template AllocShape pick_alloc_shape<kMaxFrames, 1>(const BatchParams<kMaxFrames, 1>&, int);
template AllocShape pick_alloc_shape<kMaxFrames, kMaxMaps>(const BatchParams<kMaxFrames, kMaxMaps>&, int);
template cudaError_t launch_band_alloc<1, 1>(const BatchParams<1, 1>&, int, AllocShape, cudaStream_t);
template cudaError_t launch_band_alloc<kMaxFrames, kMaxMaps>(const BatchParams<kMaxFrames, kMaxMaps>&,
                                                             int, AllocShape, cudaStream_t);
template cudaError_t launch_integrate<1, 1>(const BatchParams<1, 1>&, int, cudaStream_t);
template cudaError_t launch_band_alloc<kMaxFrames, 1>(const BatchParams<kMaxFrames, 1>&, int, AllocShape,
                                                     cudaStream_t);
template cudaError_t launch_integrate<kMaxFrames, 1>(const BatchParams<kMaxFrames, 1>&, int, cudaStream_t);
template cudaError_t launch_integrate<kMaxFrames, kMaxMaps>(const BatchParams<kMaxFrames, kMaxMaps>&,
                                                            int, cudaStream_t);

cudaError_t launch_query(const MapDev& m, const float* pts, int64_t n, float* dist, float* weight,
                         cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const PointLaunch q = point_launch(m.v, n, pts, dist, weight);
  const auto k = m.storage == kStorageOcc   ? query_kernel<kStorageOcc>
                 : m.storage == kStorageF16 ? query_kernel<kStorageF16>
                 : m.storage == kStorageX16 ? query_kernel<kStorageX16>
                                            : query_kernel<kStorageF32>;
  return launch_dependent(k, q.blocks, kPointThreads, s, m, pts, n, q.inv_v, q.vec, dist, weight);
}

cudaError_t launch_query_color(const MapDev& m, const float* pts, int64_t n, float* rgb, float* weight,
                               cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const PointLaunch q = point_launch(m.v, n, pts, rgb, weight);
  return launch_dependent(query_color_kernel, q.blocks, kPointThreads, s, m, pts, n, q.inv_v, q.vec, rgb, weight);
}

cudaError_t launch_decay(const MapDev& m, float d_occ, float d_free, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return launch_dependent(decay_kernel, sms * 8, 256, s, m, d_occ, d_free);
}

cudaError_t launch_reset(const MapDev& m, uint32_t cap, const MoreSets& more, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned need = std::max((cap / 4 + 255) / 256, ((unsigned)m.max_blocks / 16 + 255) / 256);
  return launch_dependent(reset_kernel, std::max(1u, std::min(need, (unsigned)sms * 8)), 256, s, m, cap, more);
}

}  // namespace gbt
