// Marching-cubes meshing of TSDF blocks (Sec. IV-B: updated blocks are
// meshed with a parallel Marching Cubes), sm_103a.
//
//  mesh_list_kernel  the blocks to mesh: every block, or every block changed
//                    since the last extraction together with the seven
//                    blocks whose cubes reach into it (-x, -y, -z sides)
//  mesh_kernel       one warp per listed block: the 9 x 9 rows of nine voxels
//                    along x that its cubes read (the last of each axis from
//                    the neighbours) are staged in the warp's part of shared
//                    memory, the values and per row two 9-bit masks, inside
//                    and observed; each lane finds the cubes with triangles
//                    of two lines along x from four rows' masks; the warp
//                    reserves the block's output with one atomic and emits
//                    its triangles one per lane, staged so that the stores
//                    are contiguous
//
// A cube joins voxel centres g .. g + (1, 1, 1) and belongs to the block
// holding g; it is meshed only if its eight corners exist and are observed.
// Vertices are interpolated in FP32 on the edge from its lower corner.
#include "tsdf_internal.cuh"

namespace gbt {
namespace {

constexpr int kMeshWarps = 4;   // blocks meshed at once per CTA
constexpr int kRow = 12;        // words per staged row of nine values (16-byte aligned)
constexpr int kRows = 9 * 9;    // rows (y, z), y fastest
constexpr int kChunkTris = 32 * 5;  // triangles of 32 cubes, at most

__device__ __forceinline__ int pool_at(const MapDev& m, int x, int y, int z) {
  const int slot = hash_find(m, pack_key(x, y, z));
  if (slot < 0) return -1;
  const int val = m.vals[slot];
  return val >= 0 ? val : -1;
}

__device__ __forceinline__ void add_block(const MeshDev& md, uint32_t p, uint32_t gen) {
  if (atomicExch(md.stamp + p, gen) != gen) md.list[atomicAdd(md.cnt, 1ull)] = p;
}

__global__ void mesh_list_kernel(const MapDev m, const MeshDev md, int changed_only, uint32_t gen) {
  const uint32_t nb = (uint32_t)min((unsigned long long)m.max_blocks, __ldcg(m.counters + kCntBlocks));
  for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < nb; p += gridDim.x * blockDim.x) {
    if (!changed_only) {
      add_block(md, p, gen);
      continue;
    }
    if (!(m.dirty[p] & kDirtyMesh)) continue;
    m.dirty[p] &= (uint8_t)~kDirtyMesh;
    const unsigned long long key = m.block_keys[p];
    const int bx = key_coord(key, 0), by = key_coord(key, 1), bz = key_coord(key, 2);
    for (int c = 0; c < 8; ++c) {
      const int q = c == 0 ? (int)p : pool_at(m, bx - (c & 1), by - ((c >> 1) & 1), bz - ((c >> 2) & 1));
      if (q >= 0) add_block(md, (uint32_t)q, gen);
    }
  }
}

// TSDF voxel of a storage word: value, and whether it is observed.
__device__ __forceinline__ void word_voxel(const MapDev& m, uint32_t w, float min_weight, float& d, bool& ok) {
  if (m.storage == kStorageF16) {
    const __half2 h = *reinterpret_cast<const __half2*>(&w);
    d = __low2float(h) * m.tau;
    ok = __high2float(h) >= min_weight;
  } else {
    d = x16_dist(w, m.x16_unit);
    ok = x16_weight(w) >= min_weight;
  }
}

// Row r = y + 8 z of pool block q (eight voxels along x) and voxel r of block
// qx, its first along x, as the row's ninth: values to d, masks returned
// (inside bits 0 .. 8, observed bits 16 .. 24).  A missing block (negative) is
// unobserved.
__device__ __forceinline__ uint32_t load_row(const MapDev& m, int q, int qx, int r, float min_weight, float (&d)[9]) {
  uint32_t mask = 0u;
#pragma unroll
  for (int x = 0; x < 9; ++x) d[x] = 0.0f;
  if (m.storage == kStorageF32) {
    if (q >= 0) {
      const float4* src = reinterpret_cast<const float4*>(m.pool) + (size_t)q * 256 + 4 * r;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 v = src[k];
        d[2 * k] = v.x;
        d[2 * k + 1] = v.z;
        mask |= (v.y >= min_weight ? 1u << (16 + 2 * k) : 0u) | (v.w >= min_weight ? 2u << (16 + 2 * k) : 0u);
      }
    }
    if (qx >= 0) {
      const float2 v = reinterpret_cast<const float2*>(m.pool)[(size_t)qx * 512 + 8 * r];
      d[8] = v.x;
      mask |= v.y >= min_weight ? 1u << 24 : 0u;
    }
  } else {
    if (q >= 0) {
      const uint4* src = reinterpret_cast<const uint4*>(m.pool) + (size_t)q * 128 + 2 * r;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const uint4 v = src[k];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          bool ok;
          word_voxel(m, w[i], min_weight, d[4 * k + i], ok);
          mask |= ok ? 1u << (16 + 4 * k + i) : 0u;
        }
      }
    }
    if (qx >= 0) {
      bool ok;
      word_voxel(m, reinterpret_cast<const uint32_t*>(m.pool)[(size_t)qx * 512 + 8 * r], min_weight, d[8], ok);
      mask |= ok ? 1u << 24 : 0u;
    }
  }
#pragma unroll
  for (int x = 0; x < 9; ++x) mask |= d[x] < 0.0f ? 1u << x : 0u;
  return mask;
}

// One warp's block in shared memory.
struct MeshBlock {
  __align__(16) float d[kRow * kRows];  // value at (x, y, z): x + kRow (y + 9 z)
  uint32_t mask[kRows];
  uint16_t cube[512];         // the block's cubes with triangles, in order of their lanes
  uint8_t tri[kChunkTris];    // triangles of 32 cubes: cube in the chunk | number << 5
  __align__(16) float out[32 * 12];  // 32 triangles' positions, keys or cubes
};

// Masks of the four rows around line (y, z) of cubes.
struct LineMasks {
  uint32_t r0, r1, r2, r3;
  __device__ __forceinline__ LineMasks(const MeshBlock& b, int y, int z)
      : r0(b.mask[y + 9 * z]), r1(b.mask[y + 1 + 9 * z]), r2(b.mask[y + 9 * (z + 1)]), r3(b.mask[y + 1 + 9 * (z + 1)]) {}
  // cubes whose eight corners are observed and not all on one side
  __device__ __forceinline__ uint32_t surface() const {
    const uint32_t all = r0 & r1 & r2 & r3, any = r0 | r1 | r2 | r3;
    const uint32_t both = all & (all >> 1);  // bits 16 ..: observed; bits 0 ..: all corners inside
    return (both >> 16) & (any | (any >> 1)) & ~both & 0xFFu;
  }
  // case of cube x: corner c = x + 2 y + 4 z
  __device__ __forceinline__ int cube_case(int x) const {
    return (int)(((r0 >> x) & 3u) | (((r1 >> x) & 3u) << 2) | (((r2 >> x) & 3u) << 4) | (((r3 >> x) & 3u) << 6));
  }
};

// Copy a warp's n staged words to out.
__device__ __forceinline__ void copy_out(const float* stage, float* out, int n, int lane) {
  __syncwarp();
  for (int i = lane; i < n; i += 32) __stcs(out + i, stage[i]);
  __syncwarp();
}

// Reading every cube's corners and flags one by one (144 shared loads a lane)
// and storing each lane's triangles a word at a time (24 scattered stores a
// triangle) took 97.6 us for the blocks of 64 frames of the room; this takes
// 72.5.  Six CTAs per SM (32 KB of shared memory each) leave a warp about two
// blocks, so what remains is mostly the latency of a block's chain: list, key,
// neighbours, rows, reservation, triangles.
__global__ void __launch_bounds__(kMeshWarps * 32, 6)
    mesh_kernel(const MapDev m, const MeshDev md, const __grid_constant__ MeshTable tab, float min_weight,
                float* __restrict__ out_pos, int32_t* __restrict__ out_keys,
                int32_t* __restrict__ out_cube, int64_t cap) {
  __shared__ MeshBlock s_block[kMeshWarps];
  __shared__ uint8_t s_count[256];
  __shared__ int8_t s_edges[256 * 15];
  {
    const uint8_t* src = reinterpret_cast<const uint8_t*>(&tab);
    for (int i = threadIdx.x; i < 256; i += blockDim.x) s_count[i] = src[i];
    for (int i = threadIdx.x; i < 256 * 15; i += blockDim.x) s_edges[i] = (int8_t)src[256 + i];
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  MeshBlock& b = s_block[warp];
  const uint32_t n = (uint32_t)__ldcg(md.cnt);
  for (uint32_t k = warp * gridDim.x + blockIdx.x; k < n; k += gridDim.x * kMeshWarps) {
    const uint32_t p = md.list[k];
    const unsigned long long key = m.block_keys[p];
    const int bx = key_coord(key, 0), by = key_coord(key, 1), bz = key_coord(key, 2);
    // pool block of the block (lane 0) and of its neighbour at offset
    // (lane & 1, lane >> 1 & 1, lane >> 2) for lanes 1 .. 7
    const int nbq = lane == 0 ? (int)p
                    : (lane < 8 ? pool_at(m, bx + (lane & 1), by + ((lane >> 1) & 1), bz + (lane >> 2)) : -1);
    int nb[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) nb[i] = __shfl_sync(0xffffffffu, nbq, i);
    __syncwarp();  // the previous block's reads of the staging are done
    // rows (y, z) of the block, two per lane; then the rows at y = 8 (lanes
    // 0 .. 7), z = 8 (lanes 8 .. 15) and both (lane 16)
#pragma unroll
    for (int it = 0; it < 3; ++it) {
      int q = nb[0], qx = nb[1], r = lane + 32 * it, at = (r & 7) + 9 * (r >> 3);
      if (it == 2) {
        q = lane < 8 ? nb[2] : (lane < 16 ? nb[4] : nb[6]);
        qx = lane < 8 ? nb[3] : (lane < 16 ? nb[5] : nb[7]);
        r = lane < 8 ? 8 * lane : (lane < 16 ? lane - 8 : 0);
        at = lane < 8 ? 8 + 9 * lane : (lane < 16 ? lane - 8 + 72 : 80);
        if (lane > 16) break;
      }
      float d[9];
      const uint32_t mask = load_row(m, q, qx, r, min_weight, d);
      float4* dst = reinterpret_cast<float4*>(b.d + kRow * at);
      dst[0] = make_float4(d[0], d[1], d[2], d[3]);
      dst[1] = make_float4(d[4], d[5], d[6], d[7]);
      b.d[kRow * at + 8] = d[8];
      b.mask[at] = mask;
    }
    __syncwarp();
    // cubes with triangles on the lane's lines (y, z) = (lane & 7, lane >> 3)
    // and (lane & 7, 4 + (lane >> 3))
    int mine = 0, busy = 0;  // the lane's triangles and cubes with triangles
    uint32_t surf[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const LineMasks line(b, lane & 7, (lane >> 3) + 4 * j);
      surf[j] = line.surface();
      busy += __popc(surf[j]);
      for (uint32_t w = surf[j]; w; w &= w - 1u) mine += s_count[line.cube_case(__ffs(w) - 1)];
    }
    // one output reservation per block; an inclusive scan of the cube counts
    const int total = __reduce_add_sync(0xffffffffu, mine);
    if (total == 0) continue;
    int incl = busy;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int ncubes = __shfl_sync(0xffffffffu, incl, 31);
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(md.cnt + 1, (unsigned long long)total);
    int slot = incl - busy;
#pragma unroll
    for (int j = 0; j < 2; ++j)
      for (uint32_t w = surf[j]; w; w &= w - 1u)
        b.cube[slot++] = (uint16_t)((__ffs(w) - 1) + 8 * (lane & 7) + 64 * ((lane >> 3) + 4 * j));
    base = __shfl_sync(0xffffffffu, base, 0);
    __syncwarp();
    // 32 cubes at a time: their triangles listed, then emitted one per lane
    for (int e = 0; e < ncubes; e += 32) {
      int ent = 0, nt = 0;  // this lane's cube | case << 9, and its triangles
      if (e + lane < ncubes) {
        const int c = b.cube[e + lane];
        const LineMasks line(b, (c >> 3) & 7, c >> 6);
        const int ci = line.cube_case(c & 7);
        ent = c | (ci << 9);
        nt = s_count[ci];
      }
      int end = nt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, end, o);
        if (lane >= o) end += y;
      }
      const int tris = __shfl_sync(0xffffffffu, end, 31);
      for (int i = 0; i < nt; ++i) b.tri[end - nt + i] = (uint8_t)(lane | (i << 5));
      __syncwarp();
      for (int t0 = 0; t0 < tris; t0 += 32) {
        const int code = t0 + lane < tris ? b.tri[t0 + lane] : 0;
        const int te = __shfl_sync(0xffffffffu, ent, code & 31);
        const int cube = te & 511, ci = te >> 9, tr = code >> 5;
        const int x = cube & 7, y = (cube >> 3) & 7, z = cube >> 6;
        const int gx = 8 * bx + x, gy = 8 * by + y, gz = 8 * bz + z;
        const float* corner = b.d + x + kRow * (y + 9 * z);  // corner 0
        int g[3][3], axes[3];
        float* o = b.out + 9 * lane;
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          const int ed = s_edges[15 * ci + 3 * tr + v];
          const int axis = ed >> 2, u = ed & 1, w = (ed >> 1) & 1;
          // lower corner of edge ed: bit `axis` clear, the other two axes u, w
          const int o1 = axis == 0 ? 1 : 0, o2 = axis == 2 ? 1 : 2;
          const int lo = (u << o1) | (w << o2);
          const float* c0 = corner + (lo & 1) + kRow * (((lo >> 1) & 1) + 9 * (lo >> 2));
          const float dlo = c0[0], dhi = c0[axis == 0 ? 1 : (axis == 1 ? kRow : 9 * kRow)];
          const float tt = __fdiv_rn(dlo, __fsub_rn(dlo, dhi));
          g[v][0] = gx + (lo & 1);
          g[v][1] = gy + ((lo >> 1) & 1);
          g[v][2] = gz + (lo >> 2);
          axes[v] = axis;
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            float cf = __fadd_rn((float)g[v][a], 0.5f);
            if (a == axis) cf = __fadd_rn(cf, tt);
            o[3 * v + a] = __fmul_rn(cf, m.v);
          }
        }
        // the 32 triangles' words are contiguous in each output
        const long long room = (long long)cap - (long long)base;
        const int count = (int)max(0ll, min((long long)min(32, tris - t0), room));
        copy_out(b.out, out_pos + 9 * base, 9 * count, lane);
        if (out_keys) {
          int* ko = reinterpret_cast<int*>(b.out) + 12 * lane;
#pragma unroll
          for (int v = 0; v < 3; ++v)
            *reinterpret_cast<int4*>(ko + 4 * v) = make_int4(g[v][0], g[v][1], g[v][2], axes[v]);
          copy_out(b.out, reinterpret_cast<float*>(out_keys) + 12 * base, 12 * count, lane);
        }
        if (out_cube) {
          int* co = reinterpret_cast<int*>(b.out) + 3 * lane;
          co[0] = gx;
          co[1] = gy;
          co[2] = gz;
          copy_out(b.out, reinterpret_cast<float*>(out_cube) + 3 * base, 3 * count, lane);
        }
        base += (unsigned long long)min(32, tris - t0);
      }
      __syncwarp();  // the chunk's triangle list is used up
    }
  }
}

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

}  // namespace

cudaError_t launch_mesh(const MapDev& m, const MeshDev& md, const MeshTable& table, int changed_only,
                        uint32_t gen, float min_weight, float* pos, int32_t* keys, int32_t* cubes,
                        int64_t cap, cudaStream_t s) {
  const int sms = sm_count();
  mesh_list_kernel<<<sms * 2, 256, 0, s>>>(m, md, changed_only, gen);
  mesh_kernel<<<sms * 6, kMeshWarps * 32, 0, s>>>(m, md, table, min_weight, pos, keys, cubes, cap);
  return cudaGetLastError();
}

}  // namespace gbt
