// rads.cu -- radiodensity-aware dual sampling (RADS, Sec. 3.3): the initial
// point cloud of a DDGS model from a CT volume.
//
//   P^mc  marching-cubes points of the isolevel (min + max) / 2 (Sec. 4.1):
//         one point on every grid edge whose two end voxels lie on opposite
//         sides of it, at the linear interpolation along the edge; n1 of them
//         kept uniformly without replacement (the n1 smallest counter-based
//         keys), in edge order.
//   P^dw  n2 voxel centres drawn with probability proportional to HU - min.
//   Scales: the 3D Gaussian splatting default, the root mean squared distance
//         to the 3 nearest other points.
//
// Every pass over the volume is a memory-bound sweep: blocks own chunks of
// 4096 consecutive voxels; a warp walks 512 of them lane-interleaved (voxel
// base + 32 i + lane), so each load of the voxel and of its +x/+y/+z
// neighbours is one coalesced 64-byte request, and the per-warp crossing
// order is the global edge order. The crossing list is sized by one host
// synchronisation; the n1-th smallest key is found by a radix select and the
// kept crossings are compacted in order. The neighbour search runs on a grid of
// cells over the volume.
#include <algorithm>
#include <climits>
#include <cmath>

#include "ddgs_internal.cuh"

namespace ddgs {
namespace {

constexpr int RT = 256;         // threads per block of the sweeps
constexpr int RI = 16;          // voxels (keys) per lane
constexpr int RCH = RT * RI;    // voxels (keys) per block: 4096
constexpr int SUB = 32 * RI;    // voxels per warp (sub-chunk): 512
constexpr int NSUB = RT / 32;   // sub-chunks per chunk
constexpr int SEL_BITS = 11, SEL_BINS = 1 << SEL_BITS;  // radix select: digits of a pass
constexpr int SEL_CAND = 4096;  // keys that the select's last step orders in one block
constexpr int KNN_CELLS = 32768;  // most cells of the neighbour search's grid
constexpr int KNN_NEAR = 1;     // rings of cells searched by eight lanes a point, then by a warp
constexpr int KNN_T = 256;      // threads per block of the search
constexpr uint32_t CROWD_SPREAD = 16;  // see knn_crowded
constexpr int CROWD_TILE = 1024;  // points staged at a time for those in crowded cells

// Output number i + 1 of SplitMix64 (Steele, Lea and Flood, OOPSLA 2014)
// seeded with `seed`: the state after i + 1 golden-gamma steps, finalised.
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t i) {
  uint64_t z = seed + (i + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

struct RadsState {
  int32_t hu_min, hu_max;
  uint64_t prefix;   // radix select: the wanted key's digits found so far
  uint64_t rank;     // its rank among the keys sharing that prefix
  uint32_t done;     // blocks finished in the current select pass
  uint32_t n_cand;   // keys sharing the prefix found so far
  uint32_t n_far;    // points whose neighbours lie beyond KNN_NEAR cells
  uint32_t n_crowd;  // points in crowded cells
  uint32_t hist[SEL_BINS];
};

// The grid of the neighbour search: cells of equal size over the volume's box,
// which holds every point.
struct KnnGrid {
  float lo[3], inv[3], size[3], slack[3];  // cell of x: (x - lo) inv; size: of a cell; slack: rounding
  int32_t n[3];
  __device__ __forceinline__ int axis(int a, float x) const {
    return min(max((int)((x - lo[a]) * inv[a]), 0), n[a] - 1);
  }
  __device__ __forceinline__ int cell(float x, float y, float z) const {
    return (axis(2, z) * n[1] + axis(1, y)) * n[0] + axis(0, x);
  }
};

struct Vol {
  const int16_t *hu;
  int32_t nx, ny, nz;
  int64_t nvox;
  float sx, sy, sz, ox, oy, oz;
};

template <class Tv>
__device__ __forceinline__ Tv warp_sum(Tv x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
template <class Tv>
__device__ __forceinline__ Tv warp_incl_scan(Tv x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const Tv y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// ---- pass 1: min and max of the volume ----
// Bound by DRAM (one read of the volume): four 16-byte loads in flight per
// thread and packed 16-bit min / max, two voxels an instruction (512^3: 64 ->
// 60 us, 4.5 TB/s).
__global__ void __launch_bounds__(RT) rads_minmax_kernel(Vol v, RadsState *st) {
  after_previous();
  const int64_t n8 = v.nvox / 8, stride = (int64_t)gridDim.x * blockDim.x;
  const uint4 *p = reinterpret_cast<const uint4 *>(v.hu);  // 8 voxels, little-endian
  uint32_t lo2 = 0x7fff7fffu, hi2 = 0x80008000u;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  auto take = [&](const uint4 &q) {
    lo2 = __vmins2(__vmins2(lo2, __vmins2(q.x, q.y)), __vmins2(q.z, q.w));
    hi2 = __vmaxs2(__vmaxs2(hi2, __vmaxs2(q.x, q.y)), __vmaxs2(q.z, q.w));
  };
  for (; i + 3 * stride < n8; i += 4 * stride) {
    const uint4 q0 = p[i], q1 = p[i + stride], q2 = p[i + 2 * stride], q3 = p[i + 3 * stride];
    take(q0);
    take(q1);
    take(q2);
    take(q3);
  }
  for (; i < n8; i += stride) take(p[i]);
  int lo = min((int)(int16_t)(lo2 & 0xffffu), (int)(int16_t)(lo2 >> 16));
  int hi = max((int)(int16_t)(hi2 & 0xffffu), (int)(int16_t)(hi2 >> 16));
  for (int64_t j = n8 * 8 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < v.nvox; j += stride) {
    const int a = v.hu[j];
    lo = min(lo, a);
    hi = max(hi, a);
  }
  // one atomic pair per block: a pair per warp queued 20,000 of them on two words
  __shared__ int s_lo[RT / 32], s_hi[RT / 32];
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0) {
    s_lo[threadIdx.x >> 5] = lo;
    s_hi[threadIdx.x >> 5] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < RT / 32; ++w) {
      lo = min(lo, s_lo[w]);
      hi = max(hi, s_hi[w]);
    }
    atomicMin(&st->hu_min, lo);
    atomicMax(&st->hu_max, hi);
  }
}

// Lane-interleaved walk of one warp's 512 voxels: voxel c0 + 32 i + lane.
struct VoxelWalk {
  int64_t v;
  int32_t x, y, z;
  __device__ __forceinline__ VoxelWalk(const Vol &vol, int64_t first) : v(first) {
    const int64_t plane = (int64_t)vol.nx * vol.ny;
    z = (int32_t)(first / plane);
    const int64_t r = first - (int64_t)z * plane;
    y = (int32_t)(r / vol.nx);
    x = (int32_t)(r - (int64_t)y * vol.nx);
  }
  __device__ __forceinline__ void advance(const Vol &vol) {
    v += 32;
    x += 32;
    while (x >= vol.nx) {
      x -= vol.nx;
      if (++y == vol.ny) { y = 0; ++z; }
    }
  }
};

// Crossing edges (bit a = edge to the +a neighbour) of a voxel inside the
// volume; a voxel is above the isolevel when 2 HU > lam2 = min + max.
__device__ __forceinline__ uint32_t crossing_bits(const Vol &vol, const VoxelWalk &w, int lam2,
                                                  int &hu) {
  hu = vol.hu[w.v];
  const bool a = 2 * hu > lam2;
  uint32_t bits = 0;
  if (w.x + 1 < vol.nx) bits |= (uint32_t)((2 * (int)vol.hu[w.v + 1] > lam2) != a);
  if (w.y + 1 < vol.ny) bits |= (uint32_t)((2 * (int)vol.hu[w.v + vol.nx] > lam2) != a) << 1;
  if (w.z + 1 < vol.nz)
    bits |= (uint32_t)((2 * (int)vol.hu[w.v + (int64_t)vol.nx * vol.ny] > lam2) != a) << 2;
  return bits;
}

// 8 consecutive voxels of one row (rows are a multiple of 8 voxels on the
// vector path): int16 values from one 16-byte load, little-endian.
__device__ __forceinline__ void unpack8(const uint4 q, int h[8]) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    h[2 * k] = (int)(int16_t)(w[k] & 0xffffu);
    h[2 * k + 1] = (int)(int16_t)(w[k] >> 16);
  }
}

// Which of 8 voxels lie above the isolevel (2 HU > lam2, i.e. HU >= t with t =
// floor(lam2 / 2) + 1): voxel j in bit 8 j + 7, voxel 4 + j in bit 8 j + 6.
// With u = HU + 32768 and kc = 65536 - (t + 32768), u >= t + 32768 is the carry
// out of u + kc; the halving add (x & y) + ((x ^ y) >> 1) leaves it in the top
// bit of each 16-bit half, so that a word of two voxels takes four instructions.
// (kc fits 16 bits: t > min >= -32768.)
__device__ __forceinline__ uint32_t above2(uint32_t w, uint32_t kc2) {
  const uint32_t x = w ^ 0x80008000u;
  return (x & kc2) + (((x ^ kc2) & 0xfffefffeu) >> 1);
}
__device__ __forceinline__ uint32_t above8(const uint4 q, uint32_t kc2) {
  // the high bytes of the four halves
  const uint32_t lo = __byte_perm(above2(q.x, kc2), above2(q.y, kc2), 0x7531);
  const uint32_t hi = __byte_perm(above2(q.z, kc2), above2(q.w, kc2), 0x7531);
  return (lo & 0x80808080u) | ((hi >> 1) & 0x40404040u);
}
__device__ __forceinline__ uint32_t above_carry(int lam2) {  // kc in both halves
  const int t = (lam2 >> 1) + 1;                             // arithmetic shift: floor
  const uint32_t kc = (uint32_t)(65536 - (t + 32768)) & 0xffffu;
  return kc | (kc << 16);
}

// x and row y + z ny of voxel v0.
struct GroupAt {
  uint32_t x, y, z;
  // voxel counts stay below 2^32 (edge ids fit 32 bits): 32-bit division
  __device__ __forceinline__ GroupAt(const Vol &vol, uint32_t v0) {
    const uint32_t plane = (uint32_t)vol.nx * (uint32_t)vol.ny;
    z = v0 / plane;
    const uint32_t r = v0 - z * plane;
    y = r / (uint32_t)vol.nx;
    x = r - y * (uint32_t)vol.nx;
  }
  __device__ __forceinline__ void advance(const Vol &vol, uint32_t by) {
    x += by;
    while (x >= (uint32_t)vol.nx) {
      x -= (uint32_t)vol.nx;
      if (++y == (uint32_t)vol.ny) {
        y = 0;
        ++z;
      }
    }
  }
};

// Crossings of voxels v0 .. v0 + 7 (v0 a multiple of 8, nx a multiple of 8), in
// above8's bit order: edges to the +x, +y and +z neighbours in bx, by, bz. All
// lanes of a warp take part, lane l with the group after lane l - 1's (a lane
// past the volume with live = false).
struct GroupCross {
  uint32_t bx, by, bz;
  uint4 own;
  __device__ __forceinline__ GroupCross(const Vol &vol, int64_t v0, const GroupAt &at, bool live, uint32_t kc2) {
    const uint4 *p = reinterpret_cast<const uint4 *>(vol.hu);
    own = live ? p[v0 >> 3] : make_uint4(0u, 0u, 0u, 0u);
    uint4 qy = own, qz = own;
    if (live && at.y + 1 < (uint32_t)vol.ny) qy = p[(v0 + vol.nx) >> 3];
    if (live && at.z + 1 < (uint32_t)vol.nz) qz = p[(v0 + (int64_t)vol.nx * vol.ny) >> 3];
    const bool hx = at.x + 8 < (uint32_t)vol.nx;
    const uint32_t a = above8(own, kc2);
    by = a ^ above8(qy, kc2);
    bz = a ^ above8(qz, kc2);
    // voxel 8 is the next lane's first
    uint32_t na = __shfl_down_sync(0xffffffffu, a, 1) & 0x80u;
    if ((threadIdx.x & 31) == 31 && live && hx)
      na = (above2((uint32_t)(uint16_t)vol.hu[v0 + 8], kc2) & 0x8000u) >> 8;
    bx = (a ^ (a >> 8)) & 0x00c0c0c0u;             // j against j + 1, j = 0..2 and 4..6
    bx |= (a ^ (a << 25)) & 0x80000000u;           // 3 against 4
    if (hx) bx |= (a ^ (na << 23)) & 0x40000000u;  // 7 against 8
    if (!live) bx = by = bz = 0u;
  }
  __device__ __forceinline__ uint32_t count() const { return __popc(bx) + __popc(by) + __popc(bz); }
  // bit 3 j + a for voxel j and axis a: the edge id is 3 v0 + bit
  __device__ __forceinline__ uint32_t edge_bits() const {
    uint32_t bits = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int at = j < 4 ? 8 * j + 7 : 8 * (j - 4) + 6;
      bits |= (((bx >> at) & 1u) << (3 * j)) | (((by >> at) & 1u) << (3 * j + 1)) |
              (((bz >> at) & 1u) << (3 * j + 2));
    }
    return bits;
  }
  // sum of HU - mn over the 8 voxels
  __device__ __forceinline__ uint32_t weight(int mn) const {
    int h = __dp2a_lo((int)own.x, 0x0101, 0);  // both 16-bit halves times 1
    h = __dp2a_lo((int)own.y, 0x0101, h);
    h = __dp2a_lo((int)own.z, 0x0101, h);
    h = __dp2a_lo((int)own.w, 0x0101, h);
    return (uint32_t)(h - 8 * mn);
  }
};

// ---- pass 2: crossings and weight per warp sub-chunk (512 voxels) ----
// Bound by L2 reads (each voxel is read as itself and as the +z neighbour; the
// +y one mostly hits L1), packed compares of two voxels an instruction: 512^3
// 168 -> 127 us. (Resident warps that go from sub-chunk to sub-chunk: 161 us.)
template <bool VEC>
__global__ void __launch_bounds__(RT) rads_count_kernel(Vol vol, const RadsState *st, uint32_t *csub,
                                                        uint64_t *wsub) {
  after_previous();
  const int lane = threadIdx.x & 31;
  const int mn = st->hu_min, lam2 = st->hu_min + st->hu_max;
  const uint32_t kc2 = above_carry(lam2);
  const int64_t sub = (int64_t)blockIdx.x * NSUB + (threadIdx.x >> 5);
  const int64_t sub0 = sub * SUB;
  uint32_t c = 0;
  uint32_t ws = 0;  // at most 16 x 65,535 a lane
  if (VEC) {
    GroupAt at(vol, (uint32_t)sub0 + 8 * lane);
#pragma unroll
    for (int i = 0; i < SUB / 256; ++i) {
      if (i) at.advance(vol, 256);
      const int64_t v0 = sub0 + 256 * i + 8 * lane;
      const bool live = v0 < vol.nvox;
      const GroupCross g(vol, v0, at, live, kc2);
      c += g.count();
      if (live) ws += g.weight(mn);
    }
  } else if (sub0 + lane < vol.nvox) {
    VoxelWalk w(vol, sub0 + lane);
    for (int i = 0; i < RI && w.v < vol.nvox; ++i, w.advance(vol)) {
      int hu;
      c += __popc(crossing_bits(vol, w, lam2, hu));
      ws += (uint32_t)(hu - mn);
    }
  }
  c = __reduce_add_sync(0xffffffffu, c);
  ws = __reduce_add_sync(0xffffffffu, ws);
  if (lane == 0) {
    csub[sub] = c;
    wsub[sub] = ws;
  }
}

// ---- exclusive scans of per-chunk values over many blocks: a[] (uint32)
// and optionally b[] (uint64) into ao[0..n], bo[0..n] (ao[n], bo[n] = totals).
// Local scans of 1024 entries, a one-block scan of their totals, then the add.
constexpr int SCAN_T = 1024;

__device__ __forceinline__ uint64_t block_excl_scan64(uint64_t x, uint64_t *s_w, uint64_t &total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint64_t inc = warp_incl_scan(x);
  __syncthreads();
  if (lane == 31) s_w[wid] = inc;
  __syncthreads();
  if (wid == 0) s_w[lane] = warp_incl_scan(lane < (int)(blockDim.x >> 5) ? s_w[lane] : 0ull);
  __syncthreads();
  total = s_w[(blockDim.x >> 5) - 1];
  return (wid ? s_w[wid - 1] : 0ull) + inc - x;
}

// Entry i of a (and of b) is the sum of `per` consecutive values.
__global__ void __launch_bounds__(SCAN_T) rads_scan_local_kernel(const uint32_t *a, const uint64_t *b, int per,
                                                                 int64_t n, uint64_t *ao, uint64_t *bo,
                                                                 uint64_t *tops) {
  after_previous();
  __shared__ uint64_t s_w[32];
  const int64_t i = (int64_t)blockIdx.x * SCAN_T + threadIdx.x;
  uint64_t ta, tb;
  uint64_t xa = 0, xb = 0;
  if (i < n)
    for (int k = 0; k < per; ++k) {
      xa += a[i * per + k];
      if (b) xb += b[i * per + k];
    }
  const uint64_t ea = block_excl_scan64(xa, s_w, ta);
  if (i < n) ao[i] = ea;
  if (b) {
    const uint64_t eb = block_excl_scan64(xb, s_w, tb);
    if (i < n) bo[i] = eb;
  }
  if (threadIdx.x == 0) {
    tops[2 * blockIdx.x] = ta;
    tops[2 * blockIdx.x + 1] = b ? tb : 0ull;
  }
}

// Every block sums the local totals before its own; the last one also writes
// the grand totals.
__global__ void __launch_bounds__(SCAN_T) rads_scan_add_kernel(const uint64_t *tops, int64_t n,
                                                               uint64_t *ao, uint64_t *bo) {
  after_previous();
  __shared__ uint64_t s_a[32], s_b[32];
  const int t = threadIdx.x;  // gridDim.x <= SCAN_T
  const bool before = t < (int)blockIdx.x;
  const uint64_t xa = warp_sum(before ? tops[2 * t] : 0ull), xb = warp_sum(before ? tops[2 * t + 1] : 0ull);
  if ((t & 31) == 0) {
    s_a[t >> 5] = xa;
    s_b[t >> 5] = xb;
  }
  __syncthreads();
  uint64_t pa = 0, pb = 0;
  for (int w = 0; w < 32; ++w) {
    pa += s_a[w];
    pb += s_b[w];
  }
  const int64_t i = (int64_t)blockIdx.x * SCAN_T + t;
  if (i < n) {
    ao[i] += pa;
    if (bo) bo[i] += pb;
  }
  if (blockIdx.x == gridDim.x - 1 && t == 0) {
    ao[n] = pa + tops[2 * blockIdx.x];
    if (bo) bo[n] = pb + tops[2 * blockIdx.x + 1];
  }
}

__device__ __forceinline__ uint64_t edge_key(uint64_t seed, uint64_t e) {
  return ((splitmix64(seed, e) >> 32) << 32) | e;
}

// ---- pass 3: the keys of every crossing, in edge order. A warp without
// crossings (most of the volume) returns at once; the others know where their
// keys start from the counts of pass 2 (512^3: 182 -> 72 us; resident warps that
// look at 32 sub-chunks at a time and go through the non-empty ones 114, as these
// lie together). ----
template <bool VEC>
__global__ void __launch_bounds__(RT) rads_emit_kernel(Vol vol, const RadsState *st,
                                                       const uint64_t *coff, const uint32_t *csub,
                                                       uint64_t seed, uint64_t *keys, uint64_t cap) {
  after_previous();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t cs = lane < NSUB ? csub[(int64_t)blockIdx.x * NSUB + lane] : 0u;
  if (__shfl_sync(0xffffffffu, cs, wid) == 0) return;  // nothing for this warp to write
  uint64_t run = coff[blockIdx.x] + warp_sum(lane < wid ? cs : 0u);
  const int lam2 = st->hu_min + st->hu_max;
  const int64_t sub0 = (int64_t)blockIdx.x * RCH + wid * SUB;
  constexpr int NIT = VEC ? SUB / 256 : RI;
  uint32_t bits[NIT];
#pragma unroll
  for (int i = 0; i < NIT; ++i) bits[i] = 0;
  if (VEC) {
    const uint32_t kc2 = above_carry(lam2);
    GroupAt at(vol, (uint32_t)sub0 + 8 * lane);
#pragma unroll
    for (int i = 0; i < NIT; ++i) {
      if (i) at.advance(vol, 256);
      const int64_t v0 = sub0 + 256 * i + 8 * lane;
      bits[i] = GroupCross(vol, v0, at, v0 < vol.nvox, kc2).edge_bits();
    }
  } else if (sub0 + lane < vol.nvox) {
    VoxelWalk w(vol, sub0 + lane);
#pragma unroll
    for (int i = 0; i < NIT; ++i) {
      if (w.v < vol.nvox) {
        int hu;
        bits[i] = crossing_bits(vol, w, lam2, hu);
        w.advance(vol);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < NIT; ++i) {
    const uint32_t n = __popc(bits[i]);
    const uint32_t incl = warp_incl_scan(n);
    uint64_t o = run + (incl - n);
    // first edge id of this lane's voxels in iteration i: 3 v0 (+ bit index)
    const uint64_t e0 = VEC ? 3ull * (uint64_t)(sub0 + 256 * i + 8 * lane)
                            : 3ull * (uint64_t)(sub0 + 32 * i + lane);
    uint32_t b = bits[i];
    while (b) {
      const int k = __ffs(b) - 1;
      b &= b - 1;
      if (o < cap) keys[o] = edge_key(seed, e0 + (uint64_t)k);
      ++o;
    }
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
}

// ---- radix select of the rank-th smallest key: 11-bit digits from the top,
// the last block of each pass picks the digit, until about SEL_CAND / 2 keys can
// share the prefix (one pass up to 4 M crossings: the keys' top bits are a
// hash); the last step gathers the keys that do and its last block finds the
// rank among them. (Six digit passes over all keys and an
// initialisation took 60 us at 0.8 M crossings, these two 22.) ----
constexpr int SEL_T = 1024;
__global__ void __launch_bounds__(SEL_T) rads_select_pass_kernel(const uint64_t *keys, int64_t m,
                                                                 RadsState *st, int shift, int64_t rank0) {
  after_previous();
  __shared__ uint32_t h[SEL_BINS];
  __shared__ uint32_t s_w[32];
  __shared__ bool s_last;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  for (int k = t; k < SEL_BINS; k += SEL_T) h[k] = 0;
  __syncthreads();
  const uint64_t mask = shift + SEL_BITS >= 64 ? 0ull : (~0ull << (shift + SEL_BITS));
  const uint64_t prefix = st->prefix;
  for (int64_t i = (int64_t)blockIdx.x * SEL_T + t; i < m; i += (int64_t)gridDim.x * SEL_T) {
    const uint64_t k = keys[i];
    if ((k & mask) == prefix) atomicAdd(&h[(uint32_t)(k >> shift) & (SEL_BINS - 1)], 1u);
  }
  __syncthreads();
  for (int k = t; k < SEL_BINS; k += SEL_T)
    if (h[k]) atomicAdd(&st->hist[k], h[k]);
  __threadfence();
  __syncthreads();
  if (t == 0) s_last = atomicAdd(&st->done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // the last block: the digit whose count interval holds the rank
  constexpr int PER = SEL_BINS / SEL_T;
  uint32_t hv[PER], sum = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    hv[k] = __ldcg(&st->hist[t * PER + k]);
    sum += hv[k];
  }
  const uint64_t rank = rank0 >= 0 ? (uint64_t)rank0 : st->rank;  // rank0: the first pass
  const uint32_t inc = warp_incl_scan(sum);
  if (lane == 31) s_w[wid] = inc;
  __syncthreads();
  uint64_t excl = inc - sum;
  for (int w = 0; w < wid; ++w) excl += s_w[w];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    if (hv[k] && excl <= rank && rank < excl + hv[k]) {
      st->prefix = prefix | ((uint64_t)(t * PER + k) << shift);
      st->rank = rank - excl;
    }
    excl += hv[k];
  }
  for (int k = 0; k < PER; ++k) st->hist[t * PER + k] = 0;
  if (t == 0) st->done = 0;
}

// The rank-th smallest of the keys that share the prefix (the bits above
// `shift`): gathered into cand, or, where more than SEL_CAND share it, read
// again from the list by the last block, one pass per bit.
__global__ void __launch_bounds__(1024) rads_select_last_kernel(const uint64_t *keys, int64_t m,
                                                                RadsState *st, int shift, uint64_t *cand) {
  after_previous();
  __shared__ uint32_t s_n;
  __shared__ bool s_last;
  __shared__ uint64_t s_key[SEL_CAND];
  const int t = threadIdx.x;
  const uint64_t mask = ~0ull << shift;
  uint64_t prefix = st->prefix;
  for (int64_t i = (int64_t)blockIdx.x * 1024 + t; i < m; i += (int64_t)gridDim.x * 1024) {
    const uint64_t k = keys[i];
    if ((k & mask) == prefix) {
      const uint32_t at = atomicAdd(&st->n_cand, 1u);
      if (at < SEL_CAND) cand[at] = k;
    }
  }
  __threadfence();
  __syncthreads();
  if (t == 0) s_last = atomicAdd(&st->done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const uint32_t n = __ldcg(&st->n_cand);
  const bool fits = n <= SEL_CAND;
  if (fits)
    for (uint32_t i = t; i < n; i += 1024) s_key[i] = __ldcg(&cand[i]);
  uint64_t rank = st->rank;
  if (n <= 1024) {  // the usual case: every key counts the smaller ones (keys are unique)
    __syncthreads();
    if ((uint32_t)t < n) {
      const uint64_t k = s_key[t];
      uint32_t less = 0;
      for (uint32_t i = 0; i < n; ++i) less += s_key[i] < k;
      if (less == rank) st->prefix = k;
    }
    return;
  }
  for (int bit = shift - 1; bit >= 0; --bit) {  // is the wanted key's bit 0 or 1?
    if (t == 0) s_n = 0;
    __syncthreads();
    uint32_t zeros = 0;
    const uint64_t want = prefix >> bit;
    if (fits) {
      for (uint32_t i = t; i < n; i += 1024) zeros += (s_key[i] >> bit) == want;
    } else {
      for (int64_t i = t; i < m; i += 1024) zeros += (keys[i] >> bit) == want;
    }
    zeros = warp_sum(zeros);
    if ((t & 31) == 0 && zeros) atomicAdd(&s_n, zeros);
    __syncthreads();
    const uint32_t z = s_n;
    if (rank >= z) {
      rank -= z;
      prefix |= 1ull << bit;
    }
    __syncthreads();
  }
  if (t == 0) st->prefix = prefix;
}

// ---- compaction of the kept crossings (key <= limit), in edge order ----
__global__ void __launch_bounds__(RT) rads_keep_count_kernel(const uint64_t *keys, int64_t m,
                                                             const RadsState *st, int all,
                                                             uint32_t *cnt) {
  after_previous();
  __shared__ uint32_t s_c[RT / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint64_t limit = all ? ~0ull : st->prefix;
  const int64_t first = (int64_t)blockIdx.x * RCH + wid * (32 * RI) + lane;
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < RI; ++i) {
    const int64_t j = first + 32 * i;
    c += (j < m && keys[j] <= limit) ? 1u : 0u;
  }
  c = warp_sum(c);
  if (lane == 0) s_c[wid] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int k = 0; k < RT / 32; ++k) t += s_c[k];
    cnt[blockIdx.x] = t;
  }
}

// off null: every block sums the counts of the blocks before it, so that no
// scan is launched for up to KEEP_SUM of them. Each point is also counted in its
// cell of the neighbour search's grid.
constexpr int KEEP_SUM = 2048;
__global__ void __launch_bounds__(RT) rads_keep_emit_kernel(Vol vol, const uint64_t *keys,
                                                            int64_t m, const RadsState *st,
                                                            int all, const uint32_t *cnt,
                                                            const uint64_t *off, int64_t n_out, float *means,
                                                            int64_t *kept_edges, KnnGrid grid,
                                                            uint32_t *cells, uint32_t *place) {
  after_previous();
  __shared__ uint32_t s_c[RT / 32];
  __shared__ uint64_t s_b[RT / 32];
  uint64_t before = 0;
  if (off) before = threadIdx.x == 0 ? off[blockIdx.x] : 0;
  else
    for (int64_t j = threadIdx.x; j < blockIdx.x; j += RT) before += cnt[j];
  before = warp_sum(before);
  if ((threadIdx.x & 31) == 0) s_b[threadIdx.x >> 5] = before;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint64_t limit = all ? ~0ull : st->prefix;
  const int lam2 = st->hu_min + st->hu_max;
  const int64_t first = (int64_t)blockIdx.x * RCH + wid * (32 * RI) + lane;
  uint32_t sel = 0;  // bit i: this lane's key of iteration i is kept
#pragma unroll
  for (int i = 0; i < RI; ++i) {
    const int64_t j = first + 32 * i;
    if (j < m && keys[j] <= limit) sel |= 1u << i;
  }
  const uint32_t wc = warp_sum((uint32_t)__popc(sel));
  if (lane == 0) s_c[wid] = wc;
  __syncthreads();
  uint64_t run = 0;
  for (int k = 0; k < RT / 32; ++k) run += s_b[k];
  for (int k = 0; k < wid; ++k) run += s_c[k];
  const uint32_t plane = (uint32_t)vol.nx * (uint32_t)vol.ny;  // edge ids fit 32 bits
  for (int i = 0; i < RI; ++i) {
    const bool kept = (sel >> i) & 1u;
    const uint32_t bal = __ballot_sync(0xffffffffu, kept);
    if (kept) {
      const uint64_t o = run + __popc(bal & ((1u << lane) - 1u));
      if (o < (uint64_t)n_out) {
        const uint32_t e = (uint32_t)keys[first + 32 * i];
        const uint32_t v = e / 3u;
        const int axis = (int)(e - 3u * v);
        const uint32_t z = v / plane, r = v - z * plane, y = r / (uint32_t)vol.nx, x = r - y * (uint32_t)vol.nx;
        const uint32_t step = axis == 0 ? 1u : (axis == 1 ? (uint32_t)vol.nx : plane);
        const float f0 = (float)vol.hu[v], f1 = (float)vol.hu[(int64_t)v + step];
        const float t = (0.5f * (float)lam2 - f0) / (f1 - f0);
        float c[3] = {(float)x, (float)y, (float)z};
        c[axis] += t;
        const float px = fmaf(vol.sx, c[0], vol.ox), py = fmaf(vol.sy, c[1], vol.oy),
                    pz = fmaf(vol.sz, c[2], vol.oz);
        means[3 * o] = px;
        means[3 * o + 1] = py;
        means[3 * o + 2] = pz;
        place[o] = atomicAdd(&cells[grid.cell(px, py, pz)], 1u);
        if (kept_edges) kept_edges[o] = (int64_t)e;
      }
    }
    run += __popc(bal);
  }
}

// ---- P^dw: one warp per draw ----
template <bool VEC>
__global__ void __launch_bounds__(RT) rads_draw_kernel(Vol vol, const RadsState *st,
                                                       const uint64_t *woff, const uint64_t *wsub,
                                                       int64_t nblk, int32_t n2, uint64_t seed,
                                                       int64_t row0, float *means,
                                                       int64_t *draw_voxels, KnnGrid grid,
                                                       uint32_t *cells, uint32_t *place) {
  after_previous();
  const int lane = threadIdx.x & 31;
  const int64_t j = (int64_t)blockIdx.x * (RT / 32) + (threadIdx.x >> 5);
  if (j >= n2) return;  // warp-uniform
  const uint64_t total = woff[nblk];
  const uint64_t target = __umul64hi(splitmix64(~seed, (uint64_t)j), total);
  // the chunk whose weight interval [woff[c], woff[c+1]) holds the target
  // (the last c with woff[c] <= target), 32 places at a time
  int64_t lo = 0, hi = nblk;  // woff[lo] <= target < woff[hi]
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) / 32, at = lo + lane * step;
    const uint32_t le = __ballot_sync(0xffffffffu, at < hi && woff[at] <= target);  // lane 0 always
    lo += (31 - __clz(le)) * step;
    hi = min(hi, lo + step);
  }
  uint64_t rem = target - woff[lo];
  // then the warp sub-chunk (512 voxels) inside it
  const uint64_t wsl = lane < NSUB ? wsub[lo * NSUB + lane] : 0ull;
  const uint64_t winc = warp_incl_scan(wsl);
  const uint32_t sub_past = __ballot_sync(0xffffffffu, lane < NSUB && winc > rem);
  const int s = sub_past ? __ffs(sub_past) - 1 : NSUB - 1;
  rem -= __shfl_sync(0xffffffffu, winc - wsl, s);
  const int64_t sub0 = lo * RCH + (int64_t)s * SUB;
  const int mn = st->hu_min;
  uint64_t run = 0;
  int64_t found = -1;
  if (VEC) {
    const uint4 *p = reinterpret_cast<const uint4 *>(vol.hu);
    for (int i = 0; i < SUB / 256; ++i) {
      const int64_t v0 = sub0 + 256 * i + 8 * lane;
      int h[8];
      uint64_t wl = 0;
      if (v0 < vol.nvox) {
        unpack8(p[v0 >> 3], h);
#pragma unroll
        for (int k = 0; k < 8; ++k) wl += (uint64_t)(h[k] - mn);
      }
      const uint64_t incl = warp_incl_scan(wl);
      const uint32_t past = __ballot_sync(0xffffffffu, run + incl > rem);
      if (past) {
        const int L = __ffs(past) - 1;
        int64_t f = -1;
        if (lane == L) {
          uint64_t acc = run + incl - wl;
          for (int k = 0; k < 8; ++k) {
            acc += (uint64_t)(h[k] - mn);
            if (acc > rem) { f = v0 + k; break; }
          }
        }
        found = __shfl_sync(0xffffffffu, f, L);
        break;
      }
      run += __shfl_sync(0xffffffffu, incl, 31);
    }
  } else {
    for (int i = 0; i < SUB / 32; ++i) {
      const int64_t v = sub0 + 32 * i + lane;
      const uint64_t w = v < vol.nvox ? (uint64_t)((int)vol.hu[v] - mn) : 0ull;
      const uint64_t incl = warp_incl_scan(w);
      const uint32_t past = __ballot_sync(0xffffffffu, run + incl > rem);
      if (past) {
        found = sub0 + 32 * i + (__ffs(past) - 1);
        break;
      }
      run += __shfl_sync(0xffffffffu, incl, 31);
    }
  }
  if (lane != 0 || found < 0) return;  // found < 0 cannot happen while target < total
  const uint64_t plane = (uint64_t)vol.nx * vol.ny;
  const uint64_t z = (uint64_t)found / plane, r = (uint64_t)found - z * plane;
  const uint64_t y = r / vol.nx, x = r - y * vol.nx;
  const int64_t o = row0 + j;
  const float px = fmaf(vol.sx, (float)x, vol.ox), py = fmaf(vol.sy, (float)y, vol.oy),
              pz = fmaf(vol.sz, (float)z, vol.oz);
  means[3 * o] = px;
  means[3 * o + 1] = py;
  means[3 * o + 2] = pz;
  place[o] = atomicAdd(&cells[grid.cell(px, py, pz)], 1u);
  if (draw_voxels) draw_voxels[j] = found;
}

// ---- scales: the 3 nearest other points, found on the grid. Every list keeps
// the 4 smallest squared distances, the point itself included (it contributes
// exactly one 0, the smallest value), so no per-pair self test is needed. ----
__device__ __forceinline__ void insert4(float d2, float &b0, float &b1, float &b2, float &b3) {
  if (d2 < b3) {
    if (d2 < b2) {
      b3 = b2;
      if (d2 < b1) {
        b2 = b1;
        if (d2 < b0) { b1 = b0; b0 = d2; } else { b1 = d2; }
      } else {
        b2 = d2;
      }
    } else {
      b3 = d2;
    }
  }
}

// Cell counts to cell starts (one block).
__global__ void __launch_bounds__(1024) rads_knn_scan_kernel(uint32_t *cells, int n_cells) {  // cells: 16-byte aligned
  after_previous();
  __shared__ uint32_t s_w[32];
  constexpr int PER = KNN_CELLS / 1024;
  static_assert(PER % 4 == 0, "cells in vectors of four");
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  uint32_t x[PER], sum = 0;
  uint4 *mine = reinterpret_cast<uint4 *>(cells) + t * (PER / 4);  // zeros past n_cells
#pragma unroll
  for (int k = 0; k < PER / 4; ++k) {
    const uint4 v = t * PER < n_cells ? mine[k] : make_uint4(0u, 0u, 0u, 0u);
    x[4 * k] = v.x;
    x[4 * k + 1] = v.y;
    x[4 * k + 2] = v.z;
    x[4 * k + 3] = v.w;
    sum += v.x + v.y + v.z + v.w;
  }
  const uint32_t inc = warp_incl_scan(sum);
  if (lane == 31) s_w[wid] = inc;
  __syncthreads();
  if (wid == 0) s_w[lane] = warp_incl_scan(s_w[lane]);
  __syncthreads();
  uint32_t run = (wid ? s_w[wid - 1] : 0u) + inc - sum;
  // entries from n_cells on get the number of all points
#pragma unroll
  for (int k = 0; k < PER / 4; ++k) {
    uint4 v;
    v.x = run;
    v.y = v.x + x[4 * k];
    v.z = v.y + x[4 * k + 1];
    v.w = v.z + x[4 * k + 2];
    run = v.w + x[4 * k + 3];
    mine[k] = v;
  }
  if (t == 1023) cells[KNN_CELLS] = run;
}

__global__ void rads_knn_sort_kernel(const float *means, int64_t n, KnnGrid grid, const uint32_t *cells,
                                     const uint32_t *place, float4 *pts) {
  after_previous();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float x = means[3 * i], y = means[3 * i + 1], z = means[3 * i + 2];
  pts[cells[grid.cell(x, y, z)] + place[i]] = make_float4(x, y, z, __uint_as_float((uint32_t)i));
}

// The 4 smallest of two ascending lists of 4, ascending.
__device__ __forceinline__ void merge4(float b[4], const float o[4]) {
  float m0 = fminf(b[0], o[3]), m1 = fminf(b[1], o[2]), m2 = fminf(b[2], o[1]), m3 = fminf(b[3], o[0]);
  // (m0 .. m3) is bitonic
  const float l0 = fminf(m0, m2), h0 = fmaxf(m0, m2), l1 = fminf(m1, m3), h1 = fmaxf(m1, m3);
  b[0] = fminf(l0, l1);
  b[1] = fmaxf(l0, l1);
  b[2] = fminf(h0, h1);
  b[3] = fmaxf(h0, h1);
}

// Squared distance of two points: the brute-force search's, bit for bit.
__device__ __forceinline__ float distance2(const float4 &c, const float4 &q) {
  const float dx = c.x - q.x, dy = c.y - q.y, dz = c.z - q.z;
  return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}

// The 4 smallest over a group of LANES lanes, each with its own list.
template <int LANES>
__device__ __forceinline__ void merge_group(uint32_t group, float m[4]) {
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) {
    float t[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) t[k] = __shfl_xor_sync(group, m[k], o);
    merge4(m, t);
  }
}
template <int LANES>
__device__ __forceinline__ uint32_t lane_group() {
  return LANES == 32 ? 0xffffffffu : ((1u << (LANES & 31)) - 1u) << ((threadIdx.x & 31) / LANES * LANES);
}

// log s of sorted point q: b[0] is the point itself (0), the others are the
// nearest other points.
__device__ __forceinline__ void knn_scale(const float4 &q, int64_t n, const float b[4], float *log_scales) {
  const int kk = n - 1 < 3 ? (int)(n - 1) : 3;
  float m = 0.f;
  if (kk >= 1) m += b[1];
  if (kk >= 2) m += b[2];
  if (kk >= 3) m += b[3];
  m = kk > 0 ? m / (float)kk : 0.f;
  const float ls = 0.5f * logf(fmaxf(m, 1e-7f));
  const int64_t o = __float_as_uint(q.w);
  log_scales[3 * o] = ls;
  log_scales[3 * o + 1] = ls;
  log_scales[3 * o + 2] = ls;
}

// Points of a crowd (the n_crowd last entries of `far`, backwards): a block compares
// 32 of them, one a lane, with every point, CROWD_TILE at a time in shared memory,
// of which each warp takes its share. The grid spares such a point nothing, and its
// scan costs more a pair (40,216 points in one cell: the whole call 912 us, with the
// grid alone 2,062, with a search over all pairs in place of the grid 937; two points
// a lane 934, eight or sixteen lanes a point 987-1,115, tiles of 256 points 1,015).
// A point is of a crowd when more than seven in eight of all points are in its first
// ring, and no axis of cells has one in CROWD_SPREAD of these on both its sides: there
// the points further out see fewer, stay with the grid, and both searches are paid for
// one after the other (the 19,600 points of a box of 40^3 voxels in a 512^3 volume:
// call 662 us, 523 with this rule; lines at a half and a third of the points were
// slower still). y and z are looked at, whose rows have been counted.
__device__ __forceinline__ void knn_crowded(const float4 *pts, int64_t n, int64_t n_crowd, const uint32_t *far,
                                            float4 *s_p, float *log_scales) {
  constexpr int NW = KNN_T / 32;
  static_assert(NW * 32 <= CROWD_TILE, "the warps' results take the tile's place");
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const float inf = __int_as_float(0x7f800000);
  for (int64_t first = (int64_t)blockIdx.x * 32; first < n_crowd; first += (int64_t)gridDim.x * 32) {
    const float4 q = pts[far[n - 1 - min(first + lane, n_crowd - 1)]];
    float b[4] = {inf, inf, inf, inf};
    for (int64_t t0 = 0; t0 < n; t0 += CROWD_TILE) {
      const int cnt = (int)min((int64_t)CROWD_TILE, n - t0);
      __syncthreads();
      for (int k = threadIdx.x; k < cnt; k += KNN_T) s_p[k] = pts[t0 + k];
      __syncthreads();
#pragma unroll 4
      for (int k = w; k < cnt; k += NW) insert4(distance2(s_p[k], q), b[0], b[1], b[2], b[3]);
    }
    __syncthreads();
    s_p[w * 32 + lane] = make_float4(b[0], b[1], b[2], b[3]);
    __syncthreads();
    if (w == 0 && first + lane < n_crowd) {
      for (int k = 1; k < NW; ++k) {
        const float4 v = s_p[k * 32 + lane];
        const float o[4] = {v.x, v.y, v.z, v.w};
        merge4(b, o);
      }
      knn_scale(q, n, b, log_scales);
    }
  }
}

// LANES lanes per point. The cells within r of the point's own form a box;
// once the 4th smallest distance found in it is no larger than the distance to
// the box's faces (less a slack for the rounding of the cell assignment), no
// point outside can be nearer. The rows of cells along x are stretches of
// consecutive points. Points that need more than KNN_NEAR cells (isolated ones:
// hundreds of rows, mostly empty) are left to a second launch with a warp for
// each, which starts again, and so are those of a crowd (knn_crowded). (Brute force
// over all pairs: 344 us for the 25,000 points of a 512^3 volume; grid and search 65.
// All rows shared by eight lanes 143, a lane per row from the second ring on 96, KNN_NEAR = 2 and 3 20 and 35
// more than 1.) A stretch of a crowded cell is long, and its scan waits for its
// loads: with three in flight in place of one, the 20,800 points of two bright boxes
// of 30^3 voxels in a 512^3 volume take 228 us in place of 302. Six blocks per SM (39
// registers): five (48 registers) 174 us there, but the search of a 301 x 277 x 190
// volume's points, 782 blocks, then needs a second wave (the whole call 221 -> 224 us).
template <int LANES, bool FAR>
__global__ void __launch_bounds__(KNN_T, FAR ? 1 : 6)
rads_knn_kernel(const float4 *pts, int64_t n, KnnGrid grid, const uint32_t *cells, RadsState *st, uint32_t *far,
                float *log_scales) {
  after_previous();
  const int sub = threadIdx.x & (LANES - 1);
  const uint32_t group = lane_group<LANES>();
  const float inf = __int_as_float(0x7f800000);
  const int64_t count = FAR ? (int64_t)st->n_far : n;
  for (int64_t item = ((int64_t)blockIdx.x * KNN_T + threadIdx.x) / LANES; item < count;
       item += (int64_t)gridDim.x * KNN_T / LANES) {
    const int64_t i = FAR ? (int64_t)far[item] : item;
    const float4 q = pts[i];
    const int cx = grid.axis(0, q.x), cy = grid.axis(1, q.y), cz = grid.axis(2, q.z);
    float b[4] = {inf, inf, inf, inf};
    bool found = false, left = false, crowded = false;
    for (int r = 1; !found; ++r) {
      const int x0 = max(cx - r, 0), x1 = min(cx + r, grid.n[0] - 1), y0 = max(cy - r, 0),
                y1 = min(cy + r, grid.n[1] - 1), z0 = max(cz - r, 0), z1 = min(cz + r, grid.n[2] - 1);
      float m[4] = {inf, inf, inf, inf};  // this lane's share of the new cells
      auto scan = [&](uint32_t p, uint32_t p1, uint32_t step) {
        for (; p < p1; p += step) insert4(distance2(pts[p], q), m[0], m[1], m[2], m[3]);
      };
      if (r == 1) {  // nine rows, often full: the lanes share each. Lane t has row t's stretch (and t + LANES's)
        auto stretch = [&](int t, uint32_t &p0, uint32_t &p1) {
          const int z = cz + t / 3 - 1, y = cy + t % 3 - 1;
          p0 = p1 = 0;
          if (t < 9 && z >= z0 && z <= z1 && y >= y0 && y <= y1) {
            const int row = (z * grid.n[1] + y) * grid.n[0];
            p0 = cells[row + x0];
            p1 = cells[row + x1 + 1];
          }
        };
        uint32_t p0, p1, e0 = 0, e1 = 0;
        stretch(sub, p0, p1);
        if (LANES < 9) stretch(sub + LANES, e0, e1);
        if (!FAR) {
          auto group_sum = [&](uint32_t x) {
#pragma unroll
            for (int o = LANES / 2; o > 0; o >>= 1) x += __shfl_xor_sync(group, x, o);
            return x;
          };
          const uint32_t own = p1 - p0, ninth = e1 - e0;  // the points of row sub, and (first lane) of row 8
          const uint32_t c = group_sum(own + ninth);
          if (8 * (uint64_t)c > 7 * (uint64_t)n) {  // nearly all points: a crowd? (knn_crowded)
            const uint32_t zl = group_sum(sub < 3 ? own : 0u), zh = group_sum((sub >= 6 ? own : 0u) + ninth);
            const uint32_t yl = group_sum(sub % 3 == 0 ? own : 0u), yh = group_sum((sub % 3 == 2 ? own : 0u) + ninth);
            crowded = max(min(zl, zh), min(yl, yh)) <= c / CROWD_SPREAD;
            if (crowded) break;
          }
        }
#pragma unroll 1
        for (int t = 0; t < 9; ++t) {
          const uint32_t a = __shfl_sync(group, t < LANES ? p0 : e0, t % LANES, LANES),
                         z = __shfl_sync(group, t < LANES ? p1 : e1, t % LANES, LANES);
          uint32_t p = a + sub;
          if (!FAR)
            for (; p + 2 * LANES < z; p += 3 * LANES) {  // three loads in flight
              const float4 c0 = pts[p], c1 = pts[p + LANES], c2 = pts[p + 2 * LANES];
              insert4(distance2(c0, q), m[0], m[1], m[2], m[3]);
              insert4(distance2(c1, q), m[0], m[1], m[2], m[3]);
              insert4(distance2(c2, q), m[0], m[1], m[2], m[3]);
            }
          scan(p, z, LANES);
        }
      } else {  // many rows, mostly empty (else the search had ended): a lane per row
        const int ny = y1 - y0 + 1, rows = ny * (z1 - z0 + 1);
        for (int t = sub; t < rows; t += LANES) {
          const int z = z0 + t / ny, y = y0 + t % ny, row = (z * grid.n[1] + y) * grid.n[0];
          if (z == cz - r || z == cz + r || y == cy - r || y == cy + r) {
            scan(cells[row + x0], cells[row + x1 + 1], 1);
          } else {  // the middle of the row was searched before
            if (cx - r >= 0) scan(cells[row + cx - r], cells[row + cx - r + 1], 1);
            if (cx + r < grid.n[0]) scan(cells[row + cx + r], cells[row + cx + r + 1], 1);
          }
        }
      }
      merge_group<LANES>(group, m);
      merge4(b, m);
      // distance to the nearest face of the box that has cells behind it
      float d = inf;
      const float at[3] = {q.x, q.y, q.z};
      const int lo[3] = {x0, y0, z0}, hi[3] = {x1, y1, z1};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float rel = at[a] - grid.lo[a];
        if (lo[a] > 0) d = fminf(d, rel - (float)lo[a] * grid.size[a] - grid.slack[a]);
        if (hi[a] < grid.n[a] - 1) d = fminf(d, (float)(hi[a] + 1) * grid.size[a] - rel - grid.slack[a]);
      }
      // d is infinite when every cell was searched; a NaN or negative d goes on
      found = d == inf || (d > 0.f && b[3] <= d * d * 0.9999f);
      if (!FAR && r == KNN_NEAR) {
        left = !found;
        break;
      }
    }
    if (sub != 0) continue;
    if (left) {
      far[atomicAdd(&st->n_far, 1u)] = (uint32_t)i;
      continue;
    }
    if (crowded) {
      far[n - 1 - atomicAdd(&st->n_crowd, 1u)] = (uint32_t)i;
      continue;
    }
    knn_scale(q, n, b, log_scales);
  }
  if constexpr (FAR) {
    __shared__ float4 s_p[CROWD_TILE];
    knn_crowded(pts, n, (int64_t)st->n_crowd, far, s_p, log_scales);
  }
}

}  // namespace
}  // namespace ddgs

#define RCK(call)                                                  \
  do {                                                             \
    cudaError_t e_ = (call);                                       \
    if (e_ != cudaSuccess) return ddgs::cuda_status(e_, #call);    \
  } while (0)

namespace {

// Reallocate the workspace buffer p (a field of the workspace) for `need`
// bytes. Its capacity is zeroed first, so an allocation that fails leaves the
// buffer marked empty and the next call retries it.
template <class Tp>
ddgs_status grow_bytes(Tp *&p, int64_t &cap, int64_t need) {
  if (need <= cap && p) return DDGS_OK;
  cap = 0;
  if (p) RCK(cudaFree(p));
  p = nullptr;
  const int64_t c = need + need / 4 + 4096;
  RCK(cudaMalloc(reinterpret_cast<void **>(&p), (size_t)c));
  cap = c;
  return DDGS_OK;
}

int64_t align256(int64_t x) { return (x + 255) & ~int64_t(255); }

// Exclusive scans of n per-chunk sums of `per` values (a, and b if not null) with totals at
// [n]; n <= 1024 * 1024.
void scan_chunks(const uint32_t *a, const uint64_t *b, int per, int64_t n, uint64_t *ao, uint64_t *bo,
                 uint64_t *tops, cudaStream_t st) {
  using namespace ddgs;
  const int64_t nt = (n + SCAN_T - 1) / SCAN_T;
  {
    LaunchScope ls(KID_RADS_SCAN, st);
    launch_next(rads_scan_local_kernel, (unsigned)nt, SCAN_T, 0, st, a, b, per, n, ao, bo, tops);
  }
  {
    LaunchScope ls(KID_RADS_SCAN, st);
    launch_next(rads_scan_add_kernel, (unsigned)nt, SCAN_T, 0, st, tops, n, ao, bo);
  }
}

// Cells of the neighbour search: about two per point, cubes where the box's
// sides allow, at most KNN_CELLS. (The points fill a part of the box only, so
// that an occupied cell holds a few.)
ddgs::KnnGrid knn_grid(const ddgs::Vol &v, int64_t n) {
  ddgs::KnnGrid g{};
  const int32_t vox[3] = {v.nx, v.ny, v.nz};
  const float s[3] = {v.sx, v.sy, v.sz}, o[3] = {v.ox, v.oy, v.oz};
  double ext[3], vol = 1.0;
  int axes = 0;
  for (int a = 0; a < 3; ++a) {
    ext[a] = (double)s[a] * (vox[a] - 1);  // a negative spacing runs downwards
    g.lo[a] = (float)(ext[a] < 0 ? o[a] + ext[a] : o[a]);
    ext[a] = std::fabs(ext[a]);
    if (!(ext[a] < 1e30)) ext[a] = 0.0;  // not finite: one cell
    if (ext[a] > 0) { vol *= ext[a]; ++axes; }
  }
  const double want = (double)std::max<int64_t>(1, std::min<int64_t>(2 * n, ddgs::KNN_CELLS));
  double edge = axes ? std::pow(vol / want, 1.0 / axes) : 1.0;
  for (;;) {
    int64_t cells = 1;
    for (int a = 0; a < 3; ++a) {
      const double k = edge > 0 ? std::floor(ext[a] / edge) : 0.0;
      g.n[a] = (int32_t)std::max(1.0, std::min(k, (double)ddgs::KNN_CELLS));
      cells *= g.n[a];
    }
    if (cells <= ddgs::KNN_CELLS) break;
    edge *= 1.05;
  }
  for (int a = 0; a < 3; ++a) {
    g.inv[a] = ext[a] > 0 ? (float)(g.n[a] / ext[a]) : 0.f;
    g.size[a] = ext[a] > 0 ? (float)(ext[a] / g.n[a]) : 0.f;
    // far above the rounding of x - lo, of the product and of a face's position
    g.slack[a] = (float)(1e-5 * (ext[a] + std::fabs((double)g.lo[a])));
  }
  return g;
}

}  // namespace

extern "C" ddgs_status ddgs_rads(const ddgs_volume *vol, int32_t n1, int32_t n2, uint64_t seed,
                                 ddgs_workspace *ws, float *means, float *log_scales,
                                 int64_t *kept_edges, int64_t *draw_voxels, int64_t *counts,
                                 void *stream) {
  using namespace ddgs;
  if (!vol || !ws || !counts || !vol->hu || n1 < 0 || n2 < 0) return DDGS_ERR_INVALID_ARG;
  int dev = -1;  // the workspace's buffers live on the device current at its creation
  if (cudaGetDevice(&dev) != cudaSuccess || dev != ws->device) return DDGS_ERR_INVALID_ARG;
  if (vol->nx < 1 || vol->ny < 1 || vol->nz < 1) return DDGS_ERR_INVALID_ARG;
  const int64_t nvox = (int64_t)vol->nx * vol->ny * vol->nz;
  if (nvox * 3 >= (int64_t(1) << 32)) return DDGS_ERR_INVALID_ARG;  // edge ids fill the key's low word
  if ((reinterpret_cast<uintptr_t>(vol->hu) & 15u) != 0) return DDGS_ERR_INVALID_ARG;
  if ((int64_t)n1 + n2 > 0 && (!means || !log_scales)) return DDGS_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Vol v{vol->hu, vol->nx, vol->ny, vol->nz, nvox, vol->spacing[0], vol->spacing[1],
        vol->spacing[2], vol->origin[0], vol->origin[1], vol->origin[2]};
  const int64_t nblk = (nvox + RCH - 1) / RCH;
  const bool vec = vol->nx % 8 == 0;  // rows of whole 16-byte vectors
  const int64_t n_max = (int64_t)n1 + n2;
  const KnnGrid grid = knn_grid(v, n_max);
  const int n_cells = grid.n[0] * grid.n[1] * grid.n[2];

  // scratch: cells u32[KNN_CELLS + 1] | state | csub u32[8 nblk] | wsub u64[8 nblk] | coff u64[nblk+1] |
  //          woff u64[nblk+1] | scan tops u64[2][1024] | select candidates u64[SEL_CAND] |
  //          place u32[n1+n2] | far u32[n1+n2] | sorted points f32x4[n1+n2]
  const int64_t o_state = align256(4 * (KNN_CELLS + 1)), o_cs = o_state + align256(sizeof(RadsState)),
                o_ws = o_cs + align256(4 * NSUB * nblk), o_coff = o_ws + align256(8 * NSUB * nblk),
                o_woff = o_coff + align256(8 * (nblk + 1)), o_tops = o_woff + align256(8 * (nblk + 1)),
                o_cand = o_tops + align256(16 * SCAN_T), o_place = o_cand + align256(8 * SEL_CAND),
                o_far = o_place + align256(4 * n_max), o_pts = o_far + align256(4 * n_max),
                bytes = o_pts + align256(16 * std::max<int64_t>(n_max, 1));
  ddgs_status s;
  if ((s = grow_bytes(ws->rads_buf, ws->rads_buf_cap, bytes))) return s;
  unsigned char *b = ws->rads_buf;
  uint32_t *cells = reinterpret_cast<uint32_t *>(b);
  RadsState *state = reinterpret_cast<RadsState *>(b + o_state);
  uint32_t *csub = reinterpret_cast<uint32_t *>(b + o_cs);
  uint64_t *wsub = reinterpret_cast<uint64_t *>(b + o_ws);
  uint64_t *tops = reinterpret_cast<uint64_t *>(b + o_tops);
  uint64_t *coff = reinterpret_cast<uint64_t *>(b + o_coff);
  uint64_t *woff = reinterpret_cast<uint64_t *>(b + o_woff);
  uint64_t *cand = reinterpret_cast<uint64_t *>(b + o_cand);
  uint32_t *place = reinterpret_cast<uint32_t *>(b + o_place);
  uint32_t *far = reinterpret_cast<uint32_t *>(b + o_far);
  float4 *pts = reinterpret_cast<float4 *>(b + o_pts);

  RCK(cudaMemsetAsync(b, 0, (size_t)o_cs, st));  // cells and state
  RCK(cudaMemsetAsync(&state->hu_min, 0x7f, sizeof(int32_t), st));  // > any int16
  RCK(cudaMemsetAsync(&state->hu_max, 0x80, sizeof(int32_t), st));  // < any int16
  {
    LaunchScope ls(KID_RADS_MINMAX, st);
    const int64_t want = (nvox / 8 + RT - 1) / RT;
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, 8 * device_sms()));
    launch_next(rads_minmax_kernel, blocks, RT, 0, st, v, state);
  }
  {
    LaunchScope ls(KID_RADS_COUNT, st);
    auto k = vec ? rads_count_kernel<true> : rads_count_kernel<false>;
    launch_next(k, (unsigned)nblk, RT, 0, st, v, state, csub, wsub);
  }
  scan_chunks(csub, wsub, NSUB, nblk, coff, woff, tops, st);
  RCK(cudaGetLastError());
  uint64_t tot[2] = {0, 0};
  RCK(cudaMemcpyAsync(&tot[0], coff + nblk, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
  RCK(cudaMemcpyAsync(&tot[1], woff + nblk, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
  RCK(cudaStreamSynchronize(st));
  const int64_t M = (int64_t)tot[0];
  const int64_t m1 = std::min<int64_t>(n1, M), m2 = tot[1] > 0 ? n2 : 0;

  if (m1 > 0) {
    // keys u64[M] | off u64[nkb+1] | cnt u32[nkb]
    const int64_t nkb = (M + RCH - 1) / RCH;
    const int64_t k_off = align256(8 * M), k_cnt = k_off + align256(8 * (nkb + 1)),
                  kbytes = k_cnt + align256(4 * nkb);
    if ((s = grow_bytes(ws->rads_keys, ws->rads_key_cap, kbytes))) return s;
    unsigned char *kb = reinterpret_cast<unsigned char *>(ws->rads_keys);
    uint64_t *keys = ws->rads_keys;
    uint64_t *koff = nkb > KEEP_SUM ? reinterpret_cast<uint64_t *>(kb + k_off) : nullptr;
    uint32_t *kcnt = reinterpret_cast<uint32_t *>(kb + k_cnt);
    {
      LaunchScope ls(KID_RADS_EMIT, st);
      auto k = vec ? rads_emit_kernel<true> : rads_emit_kernel<false>;
      launch_next(k, (unsigned)nblk, RT, 0, st, v, state, coff, csub, seed, keys, (uint64_t)M);
    }
    const int all = M <= n1 ? 1 : 0;
    if (!all) {
      const unsigned hg = (unsigned)std::max<int64_t>(1, std::min<int64_t>((M + SEL_T - 1) / SEL_T, device_sms()));
      int shift = 64;
      do {
        shift -= SEL_BITS;
        LaunchScope ls(KID_RADS_SELECT, st);
        launch_next(rads_select_pass_kernel, hg, SEL_T, 0, st, keys, M, state, shift,
                    shift == 64 - SEL_BITS ? (int64_t)n1 - 1 : (int64_t)-1);
      } while ((M >> (64 - shift)) > SEL_CAND / 2 && shift > SEL_BITS);
      LaunchScope ls(KID_RADS_SELECT, st);
      launch_next(rads_select_last_kernel, hg, SEL_T, 0, st, keys, M, state, shift, cand);
    }
    {
      LaunchScope ls(KID_RADS_SELECT, st);
      launch_next(rads_keep_count_kernel, (unsigned)nkb, RT, 0, st, keys, M, state, all, kcnt);
    }
    if (koff) scan_chunks(kcnt, nullptr, 1, nkb, koff, nullptr, tops, st);
    {
      LaunchScope ls(KID_RADS_SELECT, st);
      launch_next(rads_keep_emit_kernel, (unsigned)nkb, RT, 0, st, v, keys, M, state, all, kcnt, koff, m1, means,
                  kept_edges, grid, cells, place);
    }
    RCK(cudaGetLastError());
  }
  if (m2 > 0) {
    LaunchScope ls(KID_RADS_DRAW, st);
    const unsigned g = (unsigned)((m2 + RT / 32 - 1) / (RT / 32));
    auto k = vec ? rads_draw_kernel<true> : rads_draw_kernel<false>;
    launch_next(k, g, RT, 0, st, v, state, woff, wsub, nblk, (int32_t)m2, seed, m1, means, draw_voxels, grid, cells,
                place);
    RCK(cudaGetLastError());
  }
  const int64_t n = m1 + m2;
  if (n > 0) {
    {
      LaunchScope ls(KID_RADS_KNN, st);
      launch_next(rads_knn_scan_kernel, 1u, 1024u, 0, st, cells, n_cells);
    }
    {
      LaunchScope ls(KID_RADS_KNN, st);
      launch_next(rads_knn_sort_kernel, (unsigned)((n + 255) / 256), 256u, 0, st, means, n, grid, cells, place, pts);
    }
    {
      LaunchScope ls(KID_RADS_KNN, st);
      launch_next(rads_knn_kernel<8, false>, (unsigned)((n * 8 + KNN_T - 1) / KNN_T), KNN_T, 0, st, pts, n, grid, cells,
                  state, far, log_scales);
    }
    {
      LaunchScope ls(KID_RADS_KNN, st);
      const unsigned g = (unsigned)std::min<int64_t>((n * 32 + KNN_T - 1) / KNN_T, 8 * device_sms());
      launch_next(rads_knn_kernel<32, true>, g, KNN_T, 0, st, pts, n, grid, cells, state, far, log_scales);
    }
    RCK(cudaGetLastError());
  }
  counts[0] = m1;
  counts[1] = m2;
  counts[2] = M;
  return DDGS_OK;
}
