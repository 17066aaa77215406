// Internal device-side data layout of the GB300 TSDF library (not part of the
// C ABI).  One map = a block hash (Sec. IV-A: integer block coordinates ->
// 8x8x8-voxel block) plus a pool of blocks stored contiguously in HBM.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace gbt {

constexpr int kBlockVoxels = 512;      // 8 x 8 x 8, x fastest
constexpr int kMaxCells = 32;          // cap on blocks met by one band segment
constexpr int kMaxFrames = 32;         // frames per batch (one bit each in the slot mask)
constexpr int kMaxMaps = 16;           // maps per batch
constexpr unsigned long long kEmptyKey = ~0ull;
constexpr int kAllocThreads = 256;     // threads per allocation CTA
constexpr int kTileW = 32;             // allocation CTA = one 32 x (16 or 32) pixel tile
constexpr int kTileHTiny = 8;          // launches whose tiles then fit one wave, LiDAR frames beside patch tiles
constexpr int kOneWave = 8 * 152;      // allocation CTAs resident at once on GB300's 152 SMs
constexpr int kTileHSmall = 16;        // small launches: more CTAs
constexpr int kTileHBig = 32;          // large launches: fewer, fuller CTAs
constexpr int kBigTilePixels = 1 << 21;  // pixels per launch from which big tiles are used
constexpr int kPatchTile = 64;           // patch tiles: 64 x 64 pixels (pick_alloc_shape)
constexpr int kPatchPixels = 3 << 19;    // pixels per launch from which patch tiles are used
constexpr int kSetBits = 10;           // CTA-local block-key set: 1024 slots
constexpr int kSetSize = 1 << kSetBits;
constexpr int kSetProbes = 32;
constexpr int kIntegrateThreads = 128; // 4 voxels per thread

// Per-map u64 counters.
enum : int {
  kCntBlocks = 0,   // pool blocks handed out (may exceed max_blocks when full)
  kCntUpdates = 1,  // voxel updates
  kCntStatus = 2,   // sticky status bits
  kCntVisits = 3,   // work-list entries consumed by integration launches
  kCntLaunches = 4, // integration launches
  kCntSegments = 5, // band segments walked by the allocator (valid pixels in range)
  kCntCells = 6,    // cells emitted by those walks (with repeats across pixels)
  kCntPairs = 7,    // (block, frame) pairs integrated: 512 voxel projections each
  kNumCounters = 8
};
// Sticky status bits.
enum : unsigned long long { kStPoolFull = 1, kStHashFull = 2, kStListFull = 4, kStTimeout = 8 };

enum : int { kSensorPinhole = 0, kSensorLidar = 1 };
// Voxel storage: TSDF {D, W} as FP32, as FP16 (D / tau) or as 16-bit fixed
// point (D / tau) with an FP16 weight, occupancy log-odds as one FP32 value,
// or colour {r, g, b, W} as four FP32 values.  The first three codes are the
// ABI's TSDF_STORAGE_* values.
enum : int { kStorageF32 = 0, kStorageF16 = 1, kStorageX16 = 2, kStorageOcc = 3, kStorageColor = 4 };

// 16-bit fixed-point TSDF voxel (one 32-bit word): D / tau as a signed
// fraction with kX16Steps steps per tau in the low half (round to nearest,
// saturating at +-tau), W as an FP16 number in the high half.
constexpr float kX16Steps = 32767.0f;
__host__ __device__ __forceinline__ float x16_dist(uint32_t word, float unit) {
  return (float)(int16_t)(uint16_t)(word & 0xFFFFu) * unit;
}
__host__ __device__ __forceinline__ float x16_weight(uint32_t word) {
  __half_raw r;
  r.x = (unsigned short)(word >> 16);
  return __half2float(__half(r));
}
__device__ __forceinline__ uint32_t x16_pack(float D, float W, float scale) {
  const float q = fminf(fmaxf(__fmul_rn(D, scale), -kX16Steps), kX16Steps);
  const int qi = __float2int_rn(q);
  const __half h = __float2half_rn(W);
  return ((uint32_t)qi & 0xFFFFu) | ((uint32_t)__half_as_ushort(h) << 16);
}

// Device view of one map.  The work list holds the hash slots met by the
// frames of the batch in flight; the integration launch consumes it and its
// last CTA resets the list length.  vals[slot]: pool index >= 0; -1 = no pool block
// (pool was full); <= -2 = block allocated by the current batch, pool index
// -v - 2, contents not yet initialised.
struct MapDev {
  unsigned long long* keys;       // [cap] packed block keys, kEmptyKey = free
  int32_t* vals;                  // [cap]
  uint32_t* mask;                 // [cap] frames of the current batch meeting the block
  void* pool;                     // [max_blocks][512] float2 {D, W}, __half2 {D/tau, W} or
                                  // fixed-point words (x16_pack)
  unsigned long long* block_keys; // [max_blocks] key of each pool block
  unsigned long long* counters;   // [kNumCounters]; kCntSegments and kCntCells are
                                  // written only when walk_stats != 0
  int32_t walk_stats;             // count band segments and cells (diagnostic)
  uint32_t* list;                 // [list_cap] slots met by the current batch
  unsigned int* ctl;              // [0] list length, [1] finished integration CTAs,
                                  // [2] entries handed out (first map of a batch)
  uint32_t list_cap;
  uint32_t cap_mask;              // hash capacity - 1 (power of two)
  int32_t max_blocks;
  int32_t storage;
  int32_t lidar_nearest;
  float v;                        // voxel edge (m)
  float tau;                      // truncation distance, (float)(trunc * (double)v)
  float inv_tau;
  float x16_scale, x16_unit;      // fixed-point storage: steps per metre, metres per step
  float wmax;
  float guard;                    // LiDAR bilinear guard (m)
  float l_occ, l_free;            // occupancy layer: log-odds added per update
  int32_t weighting;              // TSDF weight: bit 0 inverse square depth, bit 1 drop-off
  float dropoff;                  // drop-off start behind the surface (m)
  uint8_t* dirty;                 // [max_blocks] kDirtyEsdf / kDirtyMesh: changed since the
                                  // last ESDF update / mesh extraction (may be null)
};
// A map has kSets mask / work-list / control sets: the allocation of up to
// kSets - 1 sub-batches can run ahead of the integration.  The first is
// MapDev's own.  With two sets the allocation of the next sub-batch waited for
// the integration before last and the SMs idled through every integration's
// tail: the 300-frame 640x480 sequence 1,112 us with two sets, 979 with four.
constexpr int kSets = 4;
struct MoreSets {
  uint32_t* mask[kSets - 1];
  uint32_t* list[kSets - 1];
  unsigned int* ctl[kSets - 1];
};
// kDirtyNbr: a face neighbour changed (occupancy ESDF sites read across faces)
enum : uint8_t { kDirtyEsdf = 1, kDirtyMesh = 2, kDirtyNbr = 4 };

// ESDF layer of a map (Sec. IV-C), indexed like the pool.  State word per
// voxel: parent offset x, y, z as 9-bit two's complement in bits 0-8, 9-17,
// 18-26; kEsdfObs, kEsdfSite, kEsdfPar (has a parent), kEsdfInside.
constexpr uint32_t kEsdfObs = 1u << 27, kEsdfSite = 1u << 28, kEsdfPar = 1u << 29,
                   kEsdfInside = 1u << 30;
constexpr uint32_t kEsdfOffMask = (1u << 27) - 1u;
constexpr int kEsdfBitWords = (1 << 16) / 32;
constexpr int kEsdfCounts = 16;
// Words of EsdfDev::cnt: update set and lost-site sizes of the mark and clear
// stages, the three exchange-set sizes in rotation, the grid barrier's
// arrivals, and what the host reads: iterations run, a barrier timed out.
enum : int { kEcUpdate = 0, kEcLost = 2, kEcExchange = 3, kEcBarrier = 6, kEcIterations = 7, kEcTimeout = 8 };
struct EsdfDev {
  uint32_t* st;         // [max_blocks][512] voxel states
  uint32_t* st2;        // [max_blocks][512] states produced by a face exchange
  uint32_t* list;       // [max_blocks] update set of the mark and clear stages
  uint32_t* tlist[2];   // [max_blocks] update set and its face neighbours (alternate
                        // iterations use alternate lists)
  uint32_t* clist;      // [max_blocks] blocks where a site disappeared
  uint32_t* stamp_s;    // [max_blocks] generation that put the block in an update set
  uint32_t* stamp_t;    // [max_blocks] generation that put the block in a tlist
  uint32_t* ver;        // [max_blocks] generation of the block's last rewrite << 1 | buffer
                        // holding it (0: st, 1: st2; 0 between updates)
  int32_t* nbr;         // [max_blocks][6] pool index of each face neighbour (-x, +x, -y,
                        // +y, -z, +z), -1 if none; rebuilt by every update
  uint32_t* bits;       // [2][kEsdfBitWords] hashed bitmaps of the clist blocks and of their
                        // coarse cells, rebuilt by every update
  uint32_t* cnt;        // [kEsdfCounts] set sizes and barrier of the update in flight (kEc*)
  unsigned long long* stats;    // [0] voxels whose parent stopped being a site, [1] lowering
                                // iterations, [2] blocks swept, [3] blocks in face exchanges
  float site_eps, min_weight;
  int32_t max_dist;     // voxels, <= 255
};

// One frame as the kernels see it.  Geometry is anchor-relative: a is the
// block holding the sensor origin; Rcl, tloc map anchor-local voxel centres
// into the sensor frame; M, o map sensor rays into anchor-relative block
// units.  All FP32 values are rounded once from FP64 on the host.
struct FrameDev {
  int32_t kind, map, width, height;
  const float* depth;
  const uint32_t* rgba;  // colour layer: registered colour image (r in the low byte)
  const float* tab;      // LiDAR: cos/sin of beam azimuths [2*n_az], then polar [2*n_el]
  float fu, fv, cu, cv;  // pinhole
  float theta_start, phi_start, alpha, beta, min_range, max_range;  // LiDAR
  float Rcl[9], tloc[3];
  float M[9], o[3];
  int32_t a[3];
  int32_t blk_begin;     // first allocation CTA of this frame
  int32_t bit;           // bit of this frame in the slot masks = its index in the batch
  int32_t fast_rcp;      // host check: this frame's inverted decision values are in [2^-126, 2^126]
  int32_t short_walks;   // host check: this frame's band segments meet fewer than kMaxCells blocks
  int32_t vec4;          // depth rows can be read as 16-byte words (aligned base, width a multiple of 4)
};

// Tiles of an allocation launch: pinhole frames in patch x patch pixel tiles
// (0: in rows like LiDAR frames), the others in kTileW x row_h tiles.
struct AllocShape {
  int patch, row_h;
};

template <int NF, int NM>
struct BatchParams {
  int32_t n_frames;
  int32_t n_maps;
  int32_t overlap;     // launched as a programmatic dependent of the stream's previous kernel
  int32_t alloc_ctas;  // allocation tiles of the batch (the fused kernel loops over them)
  int32_t wait_extra;  // test hook: the fused kernel's grid wait expects this many extra CTAs; in an
                       // integration launch, if not 0, no warp gets an entry
  int32_t fast_rcp;    // every reciprocal of the batch's decisions lies in [2^-126, 2^126] or is not taken
  MapDev maps[NM];
  FrameDev fr[NF];
};

// Block key: three 21-bit fields holding coordinate + 2^20 (x lowest), so a
// unit step along an axis is a plain add of 1 << (21 * axis) to the key.
// Bit 63 is always 0, so no key equals kEmptyKey.
constexpr int kKeyBias = 1 << 20;
__host__ __device__ __forceinline__ constexpr unsigned long long pack_key(int x, int y, int z) {
  return (unsigned long long)(unsigned)(x + kKeyBias) |
         ((unsigned long long)(unsigned)(y + kKeyBias) << 21) |
         ((unsigned long long)(unsigned)(z + kKeyBias) << 42);
}
__host__ __device__ __forceinline__ int key_coord(unsigned long long k, int axis) {
  return (int)((k >> (21 * axis)) & 0x1FFFFF) - kKeyBias;
}
// 64-bit finaliser (MurmurHash3 fmix64) for slot selection.
__host__ __device__ __forceinline__ uint32_t hash_key(unsigned long long k) {
  k ^= k >> 33;
  k *= 0xff51afd7ed558ccdull;
  k ^= k >> 33;
  k *= 0xc4ceb9fe1a85ec53ull;
  k ^= k >> 33;
  return (uint32_t)k;
}

// Launchers (kernels.cu).
// Slot of `key` in the hash, or -1 (linear probing, bounded by the table size).
__device__ __forceinline__ int hash_find(const MapDev& m, unsigned long long key) {
  uint32_t slot = hash_key(key) & m.cap_mask;
  for (uint32_t probe = 0; probe <= m.cap_mask; ++probe) {
    const unsigned long long k = m.keys[slot];
    if (k == key) return (int)slot;
    if (k == kEmptyKey) return -1;
    slot = (slot + 1) & m.cap_mask;
  }
  return -1;
}

// Programmatic dependent launch: a kernel launched with BatchParams::overlap
// may be scheduled while the stream's previous kernel is still running; it
// stages what its parameters give (sensor constants, empty shared sets), then
// waits here, before its first global memory access, until that kernel has
// completed and its writes are visible.  Such a kernel lets the next one be
// scheduled once its CTAs have done their main work.  Ordinary launches skip
// both instructions.
__device__ __forceinline__ void wait_prev_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_next_grid() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launch a kernel that begins with wait_prev_grid() as a programmatic
// dependent of the stream's previous kernel: short kernels (queries, resets,
// decay) then pay no launch gap, and by allow_next_grid() at their start
// neither does what follows them.
template <class... P, class... A>
cudaError_t launch_dependent(void (*k)(P...), unsigned blocks, unsigned threads, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

// ----------------------------------------------------------- point lookup
//
// The query kernels look up kPointsPerThread consecutive points per thread.
// Points usually come in order (a grid, a ray, the voxels of a block), so
// neighbours share a block: a point in its predecessor's block takes its
// pool index, and the other points' probes are all issued before any is
// used.  One point per thread waited on point -> key -> slot -> value chains:
// 5.9 M voxel centres of a 5 cm map 41.5 us, four per thread 26.1 us (28
// bytes a point; the 300-frame room's 10 M points 95 -> 57 us).
constexpr int kPointsPerThread = 4;

// Quotients of the points by the voxel edge, rounded to nearest as x / v is:
// by the correctly rounded reciprocal and one residual step (Markstein's
// method; equal to the division on the 93 M quotients that lie closest to a
// rounding boundary, within 31 / 2^24 of a last place, for every odd divisor
// significand) where nothing underflows, else by division.  inv_v = 0 selects
// division (set by the host for extreme voxel edges).
__device__ __forceinline__ float div_voxel(float x, float v, float inv_v) {
  if (fabsf(x) < 0x1p-60f || inv_v == 0.0f) return __fdiv_rn(x, v);
  const float q = __fmul_rn(x, inv_v);
  return __fmaf_rn(__fmaf_rn(-v, q, x), inv_v, q);
}

// Coordinates of points 4 i .. 4 i + 3 of n (0 beyond n): three 16-byte loads
// when the array allows them.
__device__ __forceinline__ void load_points(const float* __restrict__ pts, int64_t i, int64_t n, bool vec,
                                            float (&c)[3 * kPointsPerThread]) {
  const int64_t first = kPointsPerThread * i;
  if (vec && first + kPointsPerThread <= n) {
    const float4* p = reinterpret_cast<const float4*>(pts) + 3 * i;
    const float4 a = __ldcs(p), b = __ldcs(p + 1), d = __ldcs(p + 2);
    c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w;
    c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
    c[8] = d.x; c[9] = d.y; c[10] = d.z; c[11] = d.w;
  } else {
#pragma unroll
    for (int k = 0; k < 3 * kPointsPerThread; ++k) c[k] = 3 * first + k < 3 * n ? pts[3 * first + k] : 0.0f;
  }
}

// Store four values of points 4 i .. 4 i + 3 of n.
__device__ __forceinline__ void store_points(float* __restrict__ out, int64_t i, int64_t n, bool vec,
                                             const float (&v)[kPointsPerThread]) {
  const int64_t first = kPointsPerThread * i;
  if (vec && first + kPointsPerThread <= n) {
    __stcs(reinterpret_cast<float4*>(out) + i, make_float4(v[0], v[1], v[2], v[3]));
  } else {
#pragma unroll
    for (int k = 0; k < kPointsPerThread; ++k)
      if (first + k < n) out[first + k] = v[k];
  }
}

// For each point its block's pool index (-1 where there is none) and the
// voxel's index in the block.
__device__ __forceinline__ void find_points(const MapDev& m, float inv_v, const float (&c)[3 * kPointsPerThread],
                                            int (&pool)[kPointsPerThread], int (&voxel)[kPointsPerThread]) {
  unsigned long long key[kPointsPerThread], seen[kPointsPerThread];
  uint32_t slot[kPointsPerThread];
  const float lim = 8.0f * 1048576.0f;
#pragma unroll
  for (int k = 0; k < kPointsPerThread; ++k) {
    const float gx = floorf(div_voxel(c[3 * k], m.v, inv_v)), gy = floorf(div_voxel(c[3 * k + 1], m.v, inv_v)),
                gz = floorf(div_voxel(c[3 * k + 2], m.v, inv_v));
    key[k] = kEmptyKey;  // no block has this key
    voxel[k] = 0;
    if (fabsf(gx) < lim && fabsf(gy) < lim && fabsf(gz) < lim) {
      const int ix = (int)gx, iy = (int)gy, iz = (int)gz;
      key[k] = pack_key(ix >> 3, iy >> 3, iz >> 3);
      voxel[k] = (ix & 7) + 8 * (iy & 7) + 64 * (iz & 7);
    }
  }
#pragma unroll
  for (int k = 0; k < kPointsPerThread; ++k) {
    seen[k] = kEmptyKey;
    pool[k] = -1;
    if (key[k] != kEmptyKey && (k == 0 || key[k] != key[k > 0 ? k - 1 : 0])) {
      slot[k] = hash_key(key[k]) & m.cap_mask;
      seen[k] = m.keys[slot[k]];
      pool[k] = m.vals[slot[k]];
    }
  }
#pragma unroll
  for (int k = 0; k < kPointsPerThread; ++k) {
    if (k > 0 && key[k] == key[k > 0 ? k - 1 : 0]) {
      pool[k] = pool[k > 0 ? k - 1 : 0];
      continue;
    }
    if (seen[k] != key[k] || key[k] == kEmptyKey) {  // not at its home slot: probe on
      pool[k] = -1;
      for (uint32_t probe = 0; seen[k] != kEmptyKey && probe < m.cap_mask; ++probe) {
        slot[k] = (slot[k] + 1) & m.cap_mask;
        seen[k] = m.keys[slot[k]];
        if (seen[k] == key[k]) {
          pool[k] = m.vals[slot[k]];
          break;
        }
      }
    }
    pool[k] = pool[k] >= 0 ? pool[k] : -1;
  }
}

// Tiles for a batch; tile_h: the map's knob (0 = chosen from the batch's pixels).
template <int NF, int NM>
AllocShape pick_alloc_shape(const BatchParams<NF, NM>& p, int tile_h);
template <int NF, int NM>
cudaError_t launch_band_alloc(const BatchParams<NF, NM>& p, int n_ctas, AllocShape shape, cudaStream_t s);
template <int NF, int NM>
cudaError_t launch_integrate(const BatchParams<NF, NM>& p, int per_sm, cudaStream_t s);
// Allocation and integration of one batch in a single cooperative launch;
// cudaErrorNotSupported for batches it does not cover (the caller then
// launches the two kernels).
template <int NF, int NM>
cudaError_t launch_fused(const BatchParams<NF, NM>& p, int tile_h, cudaStream_t s);
// Launch shape of the query kernels for n points, the reciprocal for
// div_voxel, and whether all of the arrays are 16-byte aligned.
struct PointLaunch {
  unsigned blocks;
  float inv_v;
  bool vec;
};
constexpr int kPointThreads = 128;
inline PointLaunch point_launch(float v, int64_t n, const void* a, const void* b, const void* c) {
  const int64_t per = (int64_t)kPointThreads * kPointsPerThread;
  const uintptr_t bits = (uintptr_t)a | (uintptr_t)b | (uintptr_t)c;
  return {(unsigned)((n + per - 1) / per), v >= 0x1p-40f && v <= 0x1p40f ? 1.0f / v : 0.0f, (bits & 15u) == 0};
}
cudaError_t launch_query_color(const MapDev& m, const float* pts, int64_t n, float* rgb, float* weight,
                               cudaStream_t s);
cudaError_t launch_query(const MapDev& m, const float* pts, int64_t n, float* dist, float* weight,
                         cudaStream_t s);
cudaError_t launch_reset(const MapDev& m, uint32_t cap, const MoreSets& more, cudaStream_t s);
cudaError_t launch_decay(const MapDev& m, float d_occ, float d_free, cudaStream_t s);
// Forget the ESDF states of the map's blocks; before launch_reset, which
// forgets how many there are.
cudaError_t launch_esdf_reset(const MapDev& m, const EsdfDev& e, cudaStream_t s);
// ESDF stages (esdf.cu).
cudaError_t launch_esdf_mark(const MapDev& m, const EsdfDev& e, uint32_t gen, cudaStream_t s);
cudaError_t launch_esdf_clear(const MapDev& m, const EsdfDev& e, uint32_t gen, cudaStream_t s);
cudaError_t launch_esdf_lower(const MapDev& m, const EsdfDev& e, uint32_t gen, unsigned wait_extra, cudaStream_t s);
cudaError_t launch_esdf_query(const MapDev& m, const EsdfDev& e, const float* pts, int64_t n,
                              float* dist, cudaStream_t s);
cudaError_t launch_import(const MapDev& m, const int32_t* keys, const float* D, const float* W,
                          int64_t n, cudaStream_t s);

// Marching-cubes case table: triangles (edge numbers) of each inside mask.
struct MeshTable {
  uint8_t count[256];
  int8_t edges[256][15];
};
// Meshing scratch of a map, allocated by the first extraction.
struct MeshDev {
  uint32_t* list;     // [max_blocks] blocks to mesh
  uint32_t* stamp;    // [max_blocks] generation that listed the block
  unsigned long long* cnt;  // [0] list size, [1] triangles produced
  unsigned long long* host; // pinned copy of cnt
};
cudaError_t launch_mesh(const MapDev& m, const MeshDev& md, const MeshTable& table, int changed_only,
                        uint32_t gen, float min_weight, float* pos, int32_t* keys, int32_t* cubes,
                        int64_t cap, cudaStream_t s);

}  // namespace gbt
