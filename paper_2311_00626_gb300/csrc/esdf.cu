// ESDF layer kernels (Sec. IV-C) and the map import kernel, sm_103a.
//
// The ESDF layer is indexed like the TSDF pool: block p of the pool has the
// 512 voxel state words st[p * 512 ..].  One update runs the stages of
// Sec. IV-C in order:
//
//   esdf_mark_kernel   mark sites in the blocks changed since the last
//                      update (the dirty flags the integration sets) and
//                      reset voxels whose site status, observation or side
//                      changed; collect the update set and the blocks where
//                      a site disappeared (occupancy layers: the face-
//                      neighbour table first, then esdf_occ_spread_kernel
//                      and esdf_occ_mark_kernel, whose site test reads
//                      across block faces)
//   esdf_clear_kernel  in every block near one of the latter, drop parents
//                      that are no longer sites
//   esdf_lower_kernel  one cooperative launch: the face-neighbour table of
//                      every block, then the lowering iterations until no
//                      block changes.  An iteration is six in-block sweeps
//                      (+x, -x, +y, -y, +z, -z) of every block of the update
//                      set, then an exchange in which the set and its
//                      existing face neighbours try, on their faces, the
//                      parents of the adjacent voxels across the faces, all
//                      reading the states as they were before the exchange;
//                      the blocks that changed are the next update set.
//
// All distance arithmetic is on integer offsets (squared lengths), so the
// result is exact and does not depend on the order in which CTAs run.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "tsdf_internal.cuh"

namespace gbt {
namespace {

constexpr int kEsdfThreads = 128;  // threads per CTA (4 voxels each, or 4 warps of 16)

__device__ __forceinline__ int off_comp(uint32_t s, int axis) {
  const int raw = (int)((s >> (9 * axis)) & 511u);
  return raw >= 256 ? raw - 512 : raw;
}

__device__ __forceinline__ int dist2(uint32_t s) {
  const int x = off_comp(s, 0), y = off_comp(s, 1), z = off_comp(s, 2);
  return x * x + y * y + z * z;
}

__device__ __forceinline__ uint32_t n_blocks(const MapDev& m) {
  return (uint32_t)min((unsigned long long)m.max_blocks, __ldcg(m.counters + kCntBlocks));
}

// Pool index of the block with coordinates (x, y, z), or -1.
__device__ __forceinline__ int pool_of(const MapDev& m, int x, int y, int z) {
  const int slot = hash_find(m, pack_key(x, y, z));
  if (slot < 0) return -1;
  const int val = m.vals[slot];
  return val >= 0 ? val : -1;
}

// Append block p to an update set (list, size) unless this generation has it already.
__device__ __forceinline__ void add_update(const EsdfDev& e, uint32_t* list, uint32_t* size,
                                           uint32_t p, uint32_t gen) {
  if (atomicExch(e.stamp_s + p, gen) != gen) list[atomicAdd(size, 1u)] = p;
}

// Hashed bitmaps of the blocks where a site disappeared (lost-site blocks)
// and of their coarse cells (cubes of G = R + 1 blocks, R the reach of a
// parent in blocks), written by the mark stage for the clear stage.
constexpr int kNearBits = kEsdfBitWords * 32;
constexpr int kCoordBias = 1 << 21;  // block coordinates + bias >= 0

__device__ __forceinline__ uint32_t near_bit(int cx, int cy, int cz) {
  return ((uint32_t)cx * 73856093u ^ (uint32_t)cy * 19349663u ^ (uint32_t)cz * 83492791u) & (kNearBits - 1);
}

__device__ __forceinline__ int parent_reach(const EsdfDev& e) { return (e.max_dist + 7) / 8 + 1; }

__device__ __forceinline__ bool bit_set(const uint32_t* bits, uint32_t b) {
  return (__ldg(bits + (b >> 5)) >> (b & 31)) & 1u;
}

// ------------------------------------------------------------- mark sites

// New state of a voxel from its observation, site and side: a new site
// takes itself as parent; a voxel that stops being a site, becomes
// observed or changes sides loses its parent (lost: a site disappeared).
__device__ __forceinline__ uint32_t marked_state(uint32_t old, bool obs, bool site, bool inside, bool& lost) {
  if (site) return kEsdfObs | kEsdfSite | kEsdfPar | (inside ? kEsdfInside : 0u);
  if (old & kEsdfSite) {
    lost = true;
    return obs ? (kEsdfObs | (inside ? kEsdfInside : 0u)) : 0u;
  }
  if (!obs) return 0u;
  if (!(old & kEsdfObs) || ((old & kEsdfInside) != 0u) != inside) return kEsdfObs | (inside ? kEsdfInside : 0u);
  return old;
}

// Update-set and lost-site bookkeeping of a marked block (lane 0).
__device__ __forceinline__ void mark_done(const MapDev& m, const EsdfDev& e, uint32_t p, uint32_t gen, bool any,
                                          bool lost) {
  if (any) add_update(e, e.list, e.cnt + kEcUpdate, p, gen);
  if (lost) {
    e.clist[atomicAdd(e.cnt + kEcLost, 1u)] = p;
    const unsigned long long key = m.block_keys[p];
    const int G = parent_reach(e) + 1;
    const int cx = key_coord(key, 0) + kCoordBias, cy = key_coord(key, 1) + kCoordBias,
              cz = key_coord(key, 2) + kCoordBias;
    const uint32_t l = near_bit(cx, cy, cz), c = near_bit(cx / G, cy / G, cz / G);
    atomicOr(e.bits + (l >> 5), 1u << (l & 31));
    atomicOr(e.bits + kEsdfBitWords + (c >> 5), 1u << (c & 31));
  }
}

// One warp per pool block, 16 voxels per lane (voxels 128 j + 4 lane + i),
// read and written as 16-byte vectors.
__global__ void __launch_bounds__(kEsdfThreads)
    esdf_mark_kernel(const MapDev m, const EsdfDev e, uint32_t gen) {
  constexpr int kWarps = kEsdfThreads / 32;
  const uint32_t nb = n_blocks(m);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (uint32_t p = blockIdx.x * kWarps + warp; p < nb; p += gridDim.x * kWarps) {
    if (!(m.dirty[p] & kDirtyEsdf)) continue;  // same value for every lane
    uint4* stb = reinterpret_cast<uint4*>(e.st + (size_t)p * 512) + lane;
    bool any = false, lost = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float D[4], W[4];
      if (m.storage == kStorageF16) {
        const uint4 raw = reinterpret_cast<const uint4*>(m.pool)[(size_t)p * 128 + 32 * j + lane];
        const uint32_t w4[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const __half2 h = *reinterpret_cast<const __half2*>(&w4[i]);
          D[i] = __low2float(h) * m.tau;
          W[i] = __high2float(h);
        }
      } else if (m.storage == kStorageX16) {
        const uint4 raw = reinterpret_cast<const uint4*>(m.pool)[(size_t)p * 128 + 32 * j + lane];
        const uint32_t w4[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          D[i] = x16_dist(w4[i], m.x16_unit);
          W[i] = x16_weight(w4[i]);
        }
      } else {
        const float4* src = reinterpret_cast<const float4*>(m.pool) + (size_t)p * 256 + 64 * j + 2 * lane;
        const float4 a = src[0], b = src[1];
        D[0] = a.x; W[0] = a.y; D[1] = a.z; W[1] = a.w;
        D[2] = b.x; W[2] = b.y; D[3] = b.z; W[3] = b.w;
      }
      const uint4 o4 = stb[32 * j];
      const uint32_t old[4] = {o4.x, o4.y, o4.z, o4.w};
      uint32_t nw[4];
      bool changed = false;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool obs = W[i] >= e.min_weight;
        nw[i] = marked_state(old[i], obs, obs && fabsf(D[i]) <= e.site_eps, obs && D[i] < 0.0f, lost);
        changed = changed || nw[i] != old[i];
      }
      if (changed) stb[32 * j] = make_uint4(nw[0], nw[1], nw[2], nw[3]);
      any = any || changed;
    }
    any = __any_sync(0xffffffffu, any);  // also: every lane has read dirty[p]
    lost = __any_sync(0xffffffffu, lost);
    if (lane == 0) {
      m.dirty[p] &= (uint8_t)~kDirtyEsdf;
      mark_done(m, e, p, gen, any, lost);
    }
  }
}

// Occupancy layers (Sec. IV-C: an occupancy voxel is a site if it is
// adjacent to free voxels).  Log-odds l > 0 is occupied, l < 0 free, l = 0
// unknown (never observed, or decayed back to probability 1/2); observed =
// occupied or free, inside = occupied, site = occupied with a free voxel
// among its six face neighbours.  Neighbours across a block face are read
// through the face-neighbour table (a missing block is unknown), so a block
// is marked when it changed or one of its face neighbours did.

// Flag the face neighbours of every changed block.  Every writer of a byte
// here sets the same bit, so the unsynchronised read-modify-writes agree.
__global__ void esdf_occ_spread_kernel(const MapDev m, const EsdfDev e) {
  const uint32_t nb = n_blocks(m);
  for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < nb; p += gridDim.x * blockDim.x) {
    if (!(m.dirty[p] & kDirtyEsdf)) continue;
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const int q = e.nbr[6 * p + f];
      if (q >= 0) m.dirty[q] |= kDirtyNbr;
    }
  }
}

// One warp per flagged block: the block's log-odds staged in shared memory,
// 16 voxels per lane (voxels 128 j + 4 lane + i) as in esdf_mark_kernel.
__global__ void __launch_bounds__(kEsdfThreads)
    esdf_occ_mark_kernel(const MapDev m, const EsdfDev e, uint32_t gen) {
  constexpr int kWarps = kEsdfThreads / 32;
  __shared__ __align__(16) float s_l[kWarps][512];
  const uint32_t nb = n_blocks(m);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* pool = reinterpret_cast<const float*>(m.pool);
  float* sl = s_l[warp];
  for (uint32_t p = blockIdx.x * kWarps + warp; p < nb; p += gridDim.x * kWarps) {
    if (!(m.dirty[p] & (kDirtyEsdf | kDirtyNbr))) continue;  // same value for every lane
#pragma unroll
    for (int j = 0; j < 4; ++j)
      reinterpret_cast<float4*>(sl)[32 * j + lane] = reinterpret_cast<const float4*>(pool)[(size_t)p * 128 + 32 * j + lane];
    const int mine = lane < 6 ? e.nbr[6 * p + lane] : -1;
    int q[6];  // face neighbours -x, +x, -y, +y, -z, +z
#pragma unroll
    for (int f = 0; f < 6; ++f) q[f] = __shfl_sync(0xffffffffu, mine, f);
    __syncwarp();
    uint4* stb = reinterpret_cast<uint4*>(e.st + (size_t)p * 512) + lane;
    bool any = false, lost = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint4 o4 = stb[32 * j];
      const uint32_t old[4] = {o4.x, o4.y, o4.z, o4.w};
      uint32_t nw[4];
      bool changed = false;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int l = 128 * j + 4 * lane + i;
        const int c[3] = {l & 7, (l >> 3) & 7, l >> 6};
        const float v = sl[l];
        bool free_nbr = false;
#pragma unroll
        for (int f = 0; f < 6; ++f) {
          const int axis = f >> 1, d = (f & 1) ? 1 : -1, stride = axis == 0 ? 1 : (axis == 1 ? 8 : 64);
          const int cn = c[axis] + d;
          float w;
          if (cn >= 0 && cn < 8) w = sl[l + d * stride];
          else w = q[f] >= 0 ? pool[(size_t)q[f] * 512 + l - d * 7 * stride] : 0.0f;
          free_nbr = free_nbr || w < 0.0f;
        }
        const bool obs = v != 0.0f, inside = v > 0.0f;
        nw[i] = marked_state(old[i], obs, inside && free_nbr, inside, lost);
        changed = changed || nw[i] != old[i];
      }
      if (changed) stb[32 * j] = make_uint4(nw[0], nw[1], nw[2], nw[3]);
      any = any || changed;
    }
    any = __any_sync(0xffffffffu, any);  // also: every lane is done with sl and dirty[p]
    lost = __any_sync(0xffffffffu, lost);
    if (lane == 0) {
      m.dirty[p] &= (uint8_t)~(kDirtyEsdf | kDirtyNbr);
      mark_done(m, e, p, gen, any, lost);
    }
  }
}

// ---------------------------------------------------------- clear invalid

// Between updates every parent is a site, and sites disappear only in the
// lost-site blocks.  A block is checked if a marked coarse cell is among the
// 27 around its own (every block within R of a lost-site block is), and in
// it a parent is looked up only if its block's bit is set.  Bitmap
// collisions only add checks of parents that are still sites, which change
// nothing.
// One warp per pool block, 16 voxels per lane (voxels 128 j + 4 lane + i).
__global__ void __launch_bounds__(kEsdfThreads)
    esdf_clear_kernel(const MapDev m, const EsdfDev e, uint32_t gen) {
  constexpr int kWarps = kEsdfThreads / 32;
  const uint32_t nc = __ldcg(e.cnt + kEcLost);
  if (nc == 0) return;
  const uint32_t nb = n_blocks(m);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = parent_reach(e) + 1;  // coarse cell edge in blocks
  const uint32_t* lost_bits = e.bits;
  const uint32_t* cell_bits = e.bits + kEsdfBitWords;
  unsigned long long my_cleared = 0;
  for (uint32_t p = blockIdx.x * kWarps + warp; p < nb; p += gridDim.x * kWarps) {
    const unsigned long long key = m.block_keys[p];
    const int bx = key_coord(key, 0), by = key_coord(key, 1), bz = key_coord(key, 2);
    bool near = false;
    if (lane < 27) {
      const uint32_t b = near_bit((bx + kCoordBias) / G + lane % 3 - 1, (by + kCoordBias) / G + (lane / 3) % 3 - 1,
                                  (bz + kCoordBias) / G + lane / 9 - 1);
      near = bit_set(cell_bits, b);
    }
    if (!__any_sync(0xffffffffu, near)) continue;
    uint4* blk = reinterpret_cast<uint4*>(e.st + (size_t)p * 512) + lane;
    uint32_t v[16];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint4 a = blk[32 * j];
      v[4 * j] = a.x; v[4 * j + 1] = a.y; v[4 * j + 2] = a.z; v[4 * j + 3] = a.w;
    }
    bool any = false;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int l = 128 * j + 4 * lane + i;
        const uint32_t s = v[4 * j + i];
        if (!(s & kEsdfPar) || (s & kEsdfSite)) continue;
        // parent voxel in global voxel coordinates, then its block and index
        const int gx = 8 * bx + (l & 7) + off_comp(s, 0);
        const int gy = 8 * by + ((l >> 3) & 7) + off_comp(s, 1);
        const int gz = 8 * bz + (l >> 6) + off_comp(s, 2);
        const int pbx = gx >> 3, pby = gy >> 3, pbz = gz >> 3;
        const uint32_t lb = near_bit(pbx + kCoordBias, pby + kCoordBias, pbz + kCoordBias);
        if (!bit_set(lost_bits, lb)) continue;  // its block lost no site
        const int pp = (pbx == bx && pby == by && pbz == bz) ? (int)p : pool_of(m, pbx, pby, pbz);
        const bool ok = pp >= 0 &&
                        (e.st[(size_t)pp * 512 + (gx & 7) + 8 * (gy & 7) + 64 * (gz & 7)] & kEsdfSite);
        if (!ok) {
          e.st[(size_t)p * 512 + l] = s & ~(kEsdfPar | kEsdfOffMask);
          ++my_cleared;
          any = true;
        }
      }
    if (__any_sync(0xffffffffu, any) && lane == 0) add_update(e, e.list, e.cnt + kEcUpdate, p, gen);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) my_cleared += __shfl_down_sync(0xffffffffu, my_cleared, o);
  if (lane == 0 && my_cleared) atomicAdd(e.stats, my_cleared);
}

// ------------------------------------------------------------ lower ESDF

// Face-neighbour table of every pool block (the block set does not change
// during an update).
__device__ __forceinline__ void neighbour_table(const MapDev& m, const EsdfDev& e) {
  const uint32_t nb = n_blocks(m);
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < 6u * nb; k += gridDim.x * blockDim.x) {
    const uint32_t p = k / 6u;
    const int f = (int)(k - 6u * p);
    const unsigned long long key = m.block_keys[p];
    const int d = (f & 1) ? 1 : -1;
    e.nbr[k] = pool_of(m, key_coord(key, 0) + (f >> 1 == 0 ? d : 0), key_coord(key, 1) + (f >> 1 == 1 ? d : 0),
                       key_coord(key, 2) + (f >> 1 == 2 ? d : 0));
  }
}
__global__ void esdf_nbr_kernel(const MapDev m, const EsdfDev e) { neighbour_table(m, e); }

// In-block sweeps keep the block in shared memory padded to 9 words per
// x-row and 72 per z-slice, so that the lines of every axis are read with at
// most two-way bank conflicts.
constexpr int kSweepRow = 9, kSweepSlice = 72;
constexpr int kSweepWords = 7 + 7 * kSweepRow + 7 * kSweepSlice + 1;

__device__ __forceinline__ int sweep_idx(int l) {
  return (l & 7) + kSweepRow * ((l >> 3) & 7) + kSweepSlice * (l >> 6);
}

// In shared memory a voxel is two words.  The first is its state with each
// offset component biased by 256 (its 9-bit two's complement field with the
// top bit flipped), so that a step along an axis is an addition in the field.
// The second is its cost: the squared offset length of its parent (0 for a
// site), max_dist^2 + 1 without a parent, kNoCost unobserved.  With them one
// comparison decides a relaxation: a candidate must be shorter than the
// voxel's cost, which a site's never is, a candidate past max_dist cannot be,
// and a voxel without a parent cannot offer (its offset field is 0, so its
// candidate costs max_dist^2 + 2).  Only unobserved voxels need a test of
// their own.  kEsdfPar is not kept up to date there; it is set on the way out
// where the cost is at most max_dist^2.  (Testing flags, range and parents one
// by one took 16 instructions a step instead of 9: 48 frames of a room mapped
// and their distances updated twice 533 -> 491 us.)
constexpr uint32_t kOffBias = 0x100u | (0x100u << 9) | (0x100u << 18);
constexpr int kNoCost = 1 << 28;

__device__ __forceinline__ int voxel_cost(uint32_t state, int max2) {
  return (state & kEsdfPar) ? dist2(state) : ((state & kEsdfObs) ? max2 + 1 : kNoCost);
}

// The squared length of neighbour q's parent offset seen from one step back
// along AXIS (q = p + D): |o|^2 + 2 D o + 1, o its biased component - 256.
template <int AXIS, int D>
__device__ __forceinline__ int step_cost(uint32_t qw, int qc) {
  const int f2 = AXIS == 0 ? (int)((qw << 1) & 0x3FEu) : (int)((qw >> (9 * AXIS - 1)) & 0x3FEu);
  return D > 0 ? qc + f2 + (1 - 512) : qc - f2 + (1 + 512);
}

// Voxel p (word, cost) tries the parent of its neighbour q at p + D.
template <int AXIS, int D>
__device__ __forceinline__ bool relax_step(uint32_t& pw, int& pc, uint32_t qw, int qc) {
  const int c = step_cost<AXIS, D>(qw, qc);
  if (!(c < pc && (pw & kEsdfObs))) return false;
  pw = ((qw + ((uint32_t)D << (9 * AXIS))) & kEsdfOffMask) | (pw & ~kEsdfOffMask);
  pc = c;
  return true;
}

// Both sweeps along AXIS of two lines of eight voxels (first i = 1 .. 7, each
// voxel trying its predecessor's parent, then i = 6 .. 0, each trying its
// successor's), in registers; two lines per lane overlap their chains.
template <int AXIS>
__device__ __forceinline__ void sweep_lines(uint32_t* s, int* s2, int base0, int base1) {
  constexpr int stride = AXIS == 0 ? 1 : (AXIS == 1 ? kSweepRow : kSweepSlice);
  uint32_t w0[8], w1[8];
  int d0[8], d1[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    w0[i] = s[base0 + stride * i];
    d0[i] = s2[base0 + stride * i];
    w1[i] = s[base1 + stride * i];
    d1[i] = s2[base1 + stride * i];
  }
#pragma unroll
  for (int i = 1; i < 8; ++i) {
    relax_step<AXIS, -1>(w0[i], d0[i], w0[i - 1], d0[i - 1]);
    relax_step<AXIS, -1>(w1[i], d1[i], w1[i - 1], d1[i - 1]);
  }
#pragma unroll
  for (int i = 6; i >= 0; --i) {
    relax_step<AXIS, 1>(w0[i], d0[i], w0[i + 1], d0[i + 1]);
    relax_step<AXIS, 1>(w1[i], d1[i], w1[i + 1], d1[i + 1]);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    s[base0 + stride * i] = w0[i];
    s2[base0 + stride * i] = d0[i];
    s[base1 + stride * i] = w1[i];
    s2[base1 + stride * i] = d1[i];
  }
}

constexpr int kLowerThreads = 256;
constexpr int kLowerWarps = kLowerThreads / 32;

// One warp's block in shared memory: words and costs.
struct LowerBlock {
  uint32_t s[kSweepWords];
  int s2[kSweepWords];
};

// Grid-wide barrier `k` (0, 1, ...) of a cooperative launch: every CTA is
// resident, so the wait ends; after a second of the global timer it gives up
// all the same, flags it and returns false to the whole CTA.  extra (a test
// hook): from barrier kWaitTestBarrier on, CTAs expected that do not exist.
constexpr unsigned kWaitTestBarrier = 4;  // after phase 3: a few exchange generations are stamped
__device__ __forceinline__ bool grid_barrier(const EsdfDev& e, unsigned k, unsigned extra, bool* s_ok) {
  const unsigned expected = (k + 1u) * gridDim.x + (k >= kWaitTestBarrier ? extra : 0u);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(e.cnt + kEcBarrier, 1u);
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    bool ok = true;
    for (;;) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(e.cnt + kEcBarrier) : "memory");
      if (v >= expected) break;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t - t0 > 1000000000ull) {
        ok = false;
        atomicOr(e.cnt + kEcTimeout, 1u);
        break;
      }
      __nanosleep(32);
    }
    __threadfence();
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok;
}

// The current block's sweeps, by its warp.
__device__ __forceinline__ void sweep_block(LowerBlock& b, int lane) {
  const int a = lane & 7, c = lane >> 3;  // lines (a, c) and (a, c + 4) on the two other axes, in axis order
  __syncwarp();
  sweep_lines<0>(b.s, b.s2, kSweepRow * a + kSweepSlice * c, kSweepRow * a + kSweepSlice * (c + 4));
  __syncwarp();
  sweep_lines<1>(b.s, b.s2, a + kSweepSlice * c, a + kSweepSlice * (c + 4));
  __syncwarp();
  sweep_lines<2>(b.s, b.s2, a + kSweepRow * c, a + kSweepRow * (c + 4));
  __syncwarp();
}

// Block states between global and shared memory, 16-byte vectors (voxels
// 128 j + 4 lane + i).  Global accesses bypass L1: other SMs wrote the block
// earlier in this launch.
__device__ __forceinline__ void load_block(LowerBlock& b, const uint32_t* g, int lane, int max2) {
  uint4 v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = __ldcg(reinterpret_cast<const uint4*>(g) + 32 * j + lane);
  __syncwarp();  // the previous block's reads are done
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t w[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int at = sweep_idx(128 * j + 4 * lane + i);
      b.s[at] = w[i] ^ kOffBias;
      b.s2[at] = voxel_cost(w[i], max2);
    }
  }
}
__device__ __forceinline__ void store_block(const LowerBlock& b, uint32_t* g, int lane, int max2) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int at = sweep_idx(128 * j + 4 * lane + i);
      w[i] = (b.s[at] ^ kOffBias) | (b.s2[at] <= max2 ? kEsdfPar : 0u);
    }
    __stcg(reinterpret_cast<uint4*>(g) + 32 * j + lane, make_uint4(w[0], w[1], w[2], w[3]));
  }
}

// The block and its existing face neighbours join the exchange set of
// generation gen (lanes 0 .. 6; nbr: the lane's neighbour, or the block).
__device__ __forceinline__ void join_exchange(const EsdfDev& e, int nbr, uint32_t gen, uint32_t* list, uint32_t* size,
                                              int lane) {
  if (lane < 7 && nbr >= 0 && atomicExch(e.stamp_t + nbr, gen) != gen) list[atomicAdd(size, 1u)] = (uint32_t)nbr;
}

// The lowering iterations in one cooperative launch.
//
// A block belongs to one warp at a time.  Phase 0 sweeps the update set that
// the mark and clear stages left; phase k >= 1 is the exchange of iteration
// k - 1 fused with the sweeps of iteration k: a warp takes a block of the
// exchange set, tries its six faces, and if the block changed sweeps it right
// away (sweeps read nothing else) and puts it and its neighbours in the next
// exchange set.  The exchange must read every neighbour as it was before the
// phase, so a block is rewritten in the other of two buffers (st, st2):
// ver[p] = generation of its last rewrite << 1 | buffer, and a reader that
// finds the present generation there reads the other buffer, which no one
// writes in this phase.  One grid barrier per iteration; the last step copies
// the blocks that ended in st2 back.
//
// Three kernels per iteration and a read-back of the set size every four cost
// the 16 iterations of a room map of 40 frames from scratch and its update
// after 8 more 470 us of kernels and six host round trips; this launch takes
// 122 + 60 us.  The sweeps' instructions bound the first phases, the latency
// of a block's dependent steps and of the barriers the small ones.
__global__ void __launch_bounds__(kLowerThreads, 3)
    esdf_lower_kernel(const MapDev m, const EsdfDev e, uint32_t gen, int with_table, unsigned wait_extra) {
  __shared__ LowerBlock blocks[kLowerWarps];
  __shared__ bool s_ok;
  const int lane = threadIdx.x & 31;
  LowerBlock& b = blocks[threadIdx.x >> 5];
  // warps numbered across the CTAs first, so that a short list spreads over the SMs
  const uint32_t warp = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, warps = gridDim.x * kLowerWarps;
  const int max2 = e.max_dist * e.max_dist;
  const uint32_t n0 = __ldcg(e.cnt + kEcUpdate);
  if (n0 == 0) return;  // nothing marked: the same for every CTA
  unsigned barrier = 0;
  if (with_table) {
    neighbour_table(m, e);
    if (!grid_barrier(e, barrier++, wait_extra, &s_ok)) return;
  }
  const uint32_t my_face = lane < 6 ? (uint32_t)lane : 0u;
  // phase 0: sweep the update set in place
  for (uint32_t k = warp; k < n0; k += warps) {
    const uint32_t p = __ldcg(e.list + k);
    int nbr = __ldcg(e.nbr + 6 * (size_t)p + my_face);
    if (lane == 6) nbr = (int)p;
    uint32_t* g = e.st + (size_t)p * 512;
    load_block(b, g, lane, max2);
    sweep_block(b, lane);
    store_block(b, g, lane, max2);
    join_exchange(e, nbr, gen, e.tlist[1], e.cnt + kEcExchange + 1, lane);
  }
  uint32_t swept = n0, pulled = 0, k = 1;
  for (;; ++k) {
    if (!grid_barrier(e, barrier++, wait_extra, &s_ok)) return;
    const uint32_t n = __ldcg(e.cnt + kEcExchange + k % 3);
    if (n == 0) break;
    const uint32_t* list = (k & 1u) ? e.tlist[1] : e.tlist[0];
    uint32_t* next = (k & 1u) ? e.tlist[0] : e.tlist[1];
    uint32_t* next_size = e.cnt + kEcExchange + (k + 1) % 3;
    if (blockIdx.x == 0 && threadIdx.x == 0) e.cnt[kEcExchange + (k + 2) % 3] = 0u;  // last read in the phase before
    pulled += n;
    const uint32_t now = (gen + k - 1u) & 0x7FFFFFFFu;  // this phase's generation in ver
    for (uint32_t i = warp; i < n; i += warps) {
      const uint32_t p = __ldcg(list + i);
      int nbr = __ldcg(e.nbr + 6 * (size_t)p + my_face);
      if (lane == 6) nbr = (int)p;
      // buffer of this block (lane 6) and of each neighbour (lanes 0 .. 5)
      uint32_t ver = lane < 7 && nbr >= 0 ? __ldcg(e.ver + nbr) : 0u;
      uint32_t buf = ver & 1u;
      if (lane < 6 && (ver >> 1) == now) buf ^= 1u;
      const uint32_t mine = __shfl_sync(0xffffffffu, buf, 6);
      // the voxels across the six faces, two per lane and face (u, v: the
      // face's coordinates, v = 2 (lane >> 4) ... in steps of 32 voxels)
      uint32_t q[6][2];
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        const int nb = __shfl_sync(0xffffffffu, nbr, f);
        const uint32_t nbuf = __shfl_sync(0xffffffffu, buf, f);
        const uint32_t* src = (nbuf ? e.st2 : e.st) + (size_t)(nb >= 0 ? nb : 0) * 512;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int u = lane & 7, v = (lane >> 3) + 4 * h, far = (f & 1) ? 0 : 7;  // the neighbour's facing layer
          const int l = f < 2 ? far + 8 * u + 64 * v : (f < 4 ? u + 8 * far + 64 * v : u + 8 * v + 64 * far);
          q[f][h] = nb >= 0 ? __ldcg(src + l) : 0u;
        }
      }
      load_block(b, (mine ? e.st2 : e.st) + (size_t)p * 512, lane, max2);
      bool any = false;
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int u = lane & 7, v = (lane >> 3) + 4 * h, near = (f & 1) ? 7 : 0;
          const int at = f < 2 ? near + kSweepRow * u + kSweepSlice * v
                               : (f < 4 ? u + kSweepRow * near + kSweepSlice * v : u + kSweepRow * v + kSweepSlice * near);
          if (!(q[f][h] & kEsdfPar)) continue;
          uint32_t w = b.s[at];
          int c = b.s2[at];
          const uint32_t qw = q[f][h] ^ kOffBias;
          const int qc = dist2(q[f][h]);
          const bool take = f == 0   ? relax_step<0, -1>(w, c, qw, qc)
                            : f == 1 ? relax_step<0, 1>(w, c, qw, qc)
                            : f == 2 ? relax_step<1, -1>(w, c, qw, qc)
                            : f == 3 ? relax_step<1, 1>(w, c, qw, qc)
                            : f == 4 ? relax_step<2, -1>(w, c, qw, qc)
                                     : relax_step<2, 1>(w, c, qw, qc);
          if (take) {
            b.s[at] = w;
            b.s2[at] = c;
            any = true;
          }
        }
      }
      if (!__any_sync(0xffffffffu, any)) continue;
      sweep_block(b, lane);
      store_block(b, (mine ? e.st : e.st2) + (size_t)p * 512, lane, max2);
      if (lane == 0) {
        __stcg(e.ver + p, (now << 1) | (mine ^ 1u));
        atomicAdd(e.stats + 2, 1ull);
      }
      join_exchange(e, nbr, gen + k, next, next_size, lane);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    atomicAdd(e.stats + 1, (unsigned long long)(k - 1));
    atomicAdd(e.stats + 2, (unsigned long long)swept);
    atomicAdd(e.stats + 3, (unsigned long long)pulled);
    e.cnt[kEcIterations] = k - 1;
  }
  // every block's states in st again
  const uint32_t nb = n_blocks(m);
  for (uint32_t p = warp; p < nb; p += warps) {
    if (!(__ldcg(e.ver + p) & 1u)) continue;  // the same for every lane
    const uint4* src = reinterpret_cast<const uint4*>(e.st2 + (size_t)p * 512) + lane;
    uint4* dst = reinterpret_cast<uint4*>(e.st + (size_t)p * 512) + lane;
    uint4 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = __ldcg(src + 32 * j);
#pragma unroll
    for (int j = 0; j < 4; ++j) dst[32 * j] = v[j];
    __syncwarp();
    if (lane == 0) e.ver[p] &= ~1u;
  }
}

// Only the map's own blocks have states (a pool block gets its first ones when
// it is marked, after it was handed out), so a reset clears those and not the
// whole pool: 128 MiB for 2^16 pool blocks, about 25 us, of which a room fills
// a tenth.  An update that gave up at a barrier leaves more behind: blocks in
// their second buffer, and stamps of generations that the host never learned
// of and will give out again.
__global__ void esdf_reset_kernel(const MapDev m, const EsdfDev e) {
  const size_t n = (size_t)n_blocks(m) * 128;
  uint4* st = reinterpret_cast<uint4*>(e.st);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    st[i] = make_uint4(0u, 0u, 0u, 0u);
  for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < n / 128; p += (size_t)gridDim.x * blockDim.x)
    e.ver[p] = e.stamp_s[p] = e.stamp_t[p] = 0u;
  if (blockIdx.x == 0 && threadIdx.x < 4) e.stats[threadIdx.x] = 0ull;
}

// ---------------------------------------------------------------- query

// Signed distance (m) at each point: the parent offset's length times the
// voxel size, negative inside; max_dist for an observed voxel without a
// parent; NaN for an unknown voxel or a point outside every block.
__global__ void __launch_bounds__(kPointThreads)
    esdf_query_kernel(const MapDev m, const EsdfDev e, const float* __restrict__ pts, int64_t n, float inv_v,
                      bool vec, float* __restrict__ dist) {
  const int64_t i = (int64_t)blockIdx.x * kPointThreads + threadIdx.x;
  wait_prev_grid();
  allow_next_grid();
  if (kPointsPerThread * i >= n) return;
  float c[3 * kPointsPerThread], out[kPointsPerThread];
  int pool[kPointsPerThread], l[kPointsPerThread];
  load_points(pts, i, n, vec, c);
  find_points(m, inv_v, c, pool, l);
  uint32_t st[kPointsPerThread];
#pragma unroll
  for (int k = 0; k < kPointsPerThread; ++k) st[k] = pool[k] >= 0 ? e.st[(size_t)pool[k] * 512 + l[k]] : 0u;
#pragma unroll
  for (int k = 0; k < kPointsPerThread; ++k) {
    out[k] = __int_as_float(0x7fc00000);
    if (st[k] & kEsdfObs) {
      const float d = (st[k] & kEsdfPar) ? sqrtf((float)dist2(st[k])) : (float)e.max_dist;
      out[k] = ((st[k] & kEsdfInside) ? -d : d) * m.v;
    }
  }
  store_points(dist, i, n, vec, out);
}

// ---------------------------------------------------------------- import

// One CTA per input block: find or insert its key (a new key takes the next
// pool block), write its voxels in the map's storage, mark it changed.
__global__ void __launch_bounds__(kEsdfThreads)
    import_kernel(const MapDev m, const int32_t* __restrict__ keys, const float* __restrict__ D,
                  const float* __restrict__ W, int64_t n) {
  __shared__ int s_pool;
  const int t = threadIdx.x;
  for (int64_t b = blockIdx.x; b < n; b += gridDim.x) {
    __syncthreads();
    if (t == 0) {
      const unsigned long long key = pack_key(keys[3 * b], keys[3 * b + 1], keys[3 * b + 2]);
      int pool = -1;
      uint32_t slot = hash_key(key) & m.cap_mask;
      for (uint32_t probe = 0; probe <= m.cap_mask; ++probe) {
        const unsigned long long old = atomicCAS(m.keys + slot, kEmptyKey, key);
        if (old == kEmptyKey) {
          const unsigned long long q = atomicAdd(m.counters + kCntBlocks, 1ull);
          if (q < (unsigned long long)m.max_blocks) {
            m.block_keys[q] = key;
            m.vals[slot] = (int)q;
            pool = (int)q;
          } else {
            m.vals[slot] = -1;
            atomicOr(m.counters + kCntStatus, (unsigned long long)kStPoolFull);
          }
          break;
        }
        if (old == key) {
          pool = m.vals[slot];
          break;
        }
        slot = (slot + 1) & m.cap_mask;
        if (probe == m.cap_mask) atomicOr(m.counters + kCntStatus, (unsigned long long)kStHashFull);
      }
      s_pool = pool;
    }
    __syncthreads();
    const int pool = s_pool;
    if (pool < 0) continue;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int l = 4 * t + i;
      const float d = D[b * 512 + l], w = W[b * 512 + l];
      if (m.storage == kStorageOcc) {
        reinterpret_cast<float*>(m.pool)[(size_t)pool * 512 + l] = d;
      } else if (m.storage == kStorageF16) {
        reinterpret_cast<__half2*>(m.pool)[(size_t)pool * 512 + l] = __floats2half2_rn(d * m.inv_tau, w);
      } else if (m.storage == kStorageX16) {
        reinterpret_cast<uint32_t*>(m.pool)[(size_t)pool * 512 + l] = x16_pack(d, w, m.x16_scale);
      } else {
        reinterpret_cast<float2*>(m.pool)[(size_t)pool * 512 + l] = make_float2(d, w);
      }
    }
    if (t == 0 && m.dirty) m.dirty[pool] = kDirtyEsdf | kDirtyMesh;
  }
}

int grid_for(int per_sm) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return std::max(1, sms) * per_sm;
}

}  // namespace

cudaError_t launch_esdf_mark(const MapDev& m, const EsdfDev& e, uint32_t gen, cudaStream_t s) {
  if (m.storage == kStorageOcc) {
    // occupancy sites read across block faces: the neighbour table first
    esdf_nbr_kernel<<<grid_for(4), 256, 0, s>>>(m, e);
    esdf_occ_spread_kernel<<<grid_for(4), 256, 0, s>>>(m, e);
    esdf_occ_mark_kernel<<<grid_for(16), kEsdfThreads, 0, s>>>(m, e, gen);
  } else {
    esdf_mark_kernel<<<grid_for(16), kEsdfThreads, 0, s>>>(m, e, gen);
  }
  return cudaGetLastError();
}

cudaError_t launch_esdf_clear(const MapDev& m, const EsdfDev& e, uint32_t gen, cudaStream_t s) {
  esdf_clear_kernel<<<grid_for(10), kEsdfThreads, 0, s>>>(m, e, gen);  // 48 registers: 10 CTAs per SM
  return cudaGetLastError();
}

cudaError_t launch_esdf_reset(const MapDev& m, const EsdfDev& e, cudaStream_t s) {
  esdf_reset_kernel<<<grid_for(4), 256, 0, s>>>(m, e);
  return cudaGetLastError();
}

// The lowering iterations, launched cooperatively with every CTA that can be
// resident.  A stream may have fewer SMs than the device (an MPS share, a
// green context): a launch that is refused as too large is made with half the
// CTAs, down to one, which meets only itself at the barriers and needs no
// cooperative launch.  Exchange generations start at gen.  The neighbour table
// is built here unless the mark stage of an occupancy layer built it.
// wait_extra: the barriers' test hook.
cudaError_t launch_esdf_lower(const MapDev& m, const EsdfDev& e, uint32_t gen, unsigned wait_extra, cudaStream_t s) {
  static std::atomic<int> fit{0};  // resident CTAs per SM (all devices are alike here)
  int n = fit.load(std::memory_order_relaxed);
  if (n == 0) {
    const cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, esdf_lower_kernel, kLowerThreads, 0);
    if (err != cudaSuccess) return err;
    if (n <= 0) return cudaErrorNotSupported;
    fit.store(n, std::memory_order_relaxed);
  }
  const int with_table = m.storage == kStorageOcc ? 0 : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kLowerThreads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;  // every CTA resident: the grid barriers can complete
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  for (int ctas = grid_for(n); ctas > 1; ctas /= 2) {
    cfg.gridDim = dim3(ctas);
    const cudaError_t err = cudaLaunchKernelEx(&cfg, esdf_lower_kernel, m, e, gen, with_table, wait_extra);
    if (err != cudaErrorCooperativeLaunchTooLarge && err != cudaErrorNotSupported) return err;
    cudaGetLastError();
  }
  cfg.gridDim = dim3(1);
  cfg.numAttrs = 0;
  return cudaLaunchKernelEx(&cfg, esdf_lower_kernel, m, e, gen, with_table, wait_extra);
}

cudaError_t launch_esdf_query(const MapDev& m, const EsdfDev& e, const float* pts, int64_t n,
                              float* dist, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const PointLaunch q = point_launch(m.v, n, pts, dist, nullptr);
  return launch_dependent(esdf_query_kernel, q.blocks, kPointThreads, s, m, e, pts, n, q.inv_v, q.vec, dist);
}

cudaError_t launch_import(const MapDev& m, const int32_t* keys, const float* D, const float* W,
                          int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  import_kernel<<<grid_for(8), kEsdfThreads, 0, s>>>(m, keys, D, W, n);
  return cudaGetLastError();
}

}  // namespace gbt
