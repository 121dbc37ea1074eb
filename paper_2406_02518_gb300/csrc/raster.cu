// raster.cu -- per-tile front-to-back blending (Eq. 1) and its backward pass.
//
// Persistent kernels: every warp takes a (tile, pixel region) item from a work
// queue ordered by list length, stages the tile's list 32 entries at a time in
// its own slice of shared memory and never waits for another warp. A region is
// 8 x 8 pixels, two per lane (the pixel-pair kernels), or 8 x 4 pixels, one per
// lane, for renders of few regions. Staging is a gather by Gaussian index from
// the per-view records, which is why it uses plain vector loads rather than a
// bulk tensor copy.
//
// Forward per pixel p, over the list in ascending depth (Eq. 1):
//   q = (p - mu-hat)^T conic (p - mu-hat); skip if q > q_max;
//   sigma = min(alpha_max, alpha exp(-q/2)); skip if sigma < alpha_min;
//   T' = T (1 - sigma); stop (without adding) if T' < t_min;
//   C += c sigma T; T = T'.
// Backward per pixel, over the same list from the last added Gaussian to the
// first, recovering T before each Gaussian as T' / (1 - sigma) and carrying
// the suffix sum S = sum over later Gaussians of c sigma T:
//   dC/dc = sigma T,  dC/dsigma = c T - S / (1 - sigma),
//   dsigma/dalpha = G and dsigma/dq = -alpha G / 2 unless sigma was clamped.
// The per-pixel 2D gradients of one Gaussian are summed over the region in
// registers (a lane per entry) and reach global memory with one vector atomic
// per (region, Gaussian).
//
// The tile edge T fixes the lists, not the regions: in tiles of 16 or 32 pixels
// most entries of a list miss a given region, so the entries that cover a pixel
// of it are collected first (EntryStream, Picker) and a batch is 32 of those.
// (Blocks of T x T threads that staged 128 to 512 entries for all their warps,
// each warp testing every entry against its four 4 x 2 quarters, were the former
// default for these tiles: 100k Gaussians, three 375 x 501 views at T = 16:
// forward 176 -> 112, backward 358 -> 190 us. The staging depth a caller asks
// for no longer selects a kernel.)
//
// PIX = true renders the Eq. 3 variant whose ray angles are each pixel's own:
// a record then carries (a, h) instead of a colour, and the pair's colour is
// c = sigmoid(a + Y_1(d_p) . h) with d_p the pixel ray's unit direction. The
// backward pass sums dL/dz (z the logit) and dL/dh per (region, Gaussian) and
// adds the pose gradient through each pixel's ray.
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "ddgs_internal.cuh"

namespace ddgs {
namespace {

struct RasterArgs {
  RenderShape s;
  RasterParams P;
  const float4 *rec;  // two float4 per record
  const uint32_t *vals;  // tile lists: Gaussian indices in depth order
  const uint2 *ranges;
  float4 *grad2d;
  float *image, *t_final;
  uint32_t *n_last;
  const float *dL_dimage, *t_final_in;
  const uint32_t *n_last_in;
  const uint32_t *order;     // global tiles, longest list first
  uint32_t *counter;         // work-queue head (zero at launch)
  unsigned long long *req_end;  // [R]: latest %globaltimer of a finished tile, or null
  // per-pixel ray angles only
  const float4 *rec2;        // (a, h_0, h_1, h_2) per record
  float4 *grad_h;            // dL/dh per record
  const float *world_to_cam, *detector;
  float *pose_grad;          // [V][12] or null
  ZeroList zero;             // backward: the summed gradients that the next kernel adds to
};

__device__ __forceinline__ float sigmoid_r(float x) { return rcp_approx(1.f + __expf(-x)); }

// The ray through pixel centre (px, py) of a view: rc = ((px - c_u) pitch_u,
// (py - c_v) pitch_v, sdd) in camera coordinates, world direction d = W^T rc,
// and Y_1 of d / |d| (real harmonics of degree 1: sqrt(3/(4 pi)) (-y, z, -x)).
struct PixRay {
  float rc[3], dh[3], inv, Y[3];
};

__device__ __forceinline__ void pixel_ray(const float *pose, const float *det, int H, int W,
                                          float px, float py, PixRay &r) {
  const float cu = 0.5f * (float)W + det[3], cv = 0.5f * (float)H + det[4];
  r.rc[0] = (px - cu) * det[1];
  r.rc[1] = (py - cv) * det[2];
  r.rc[2] = det[0];
  float d[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) d[c] = pose[c] * r.rc[0] + pose[4 + c] * r.rc[1] + pose[8 + c] * r.rc[2];
  r.inv = 1.f / sqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
#pragma unroll
  for (int c = 0; c < 3; ++c) r.dh[c] = d[c] * r.inv;
  r.Y[0] = -SH_C1 * r.dh[1];
  r.Y[1] = SH_C1 * r.dh[2];
  r.Y[2] = -SH_C1 * r.dh[0];
}

__device__ __forceinline__ float pixel_colour(const PixRay &r, float4 z) {
  return sigmoid_r(fmaf(r.Y[2], z.w, fmaf(r.Y[1], z.z, fmaf(r.Y[0], z.y, z.x))));
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Pixel-space box of the q <= q_max ellipse: the record's packed
// half-extents (computed from the 2D covariance by the preprocess).
__device__ __forceinline__ float4 ellipse_box(float4 r0, float4 r1) {
  const float2 e = unpack_halfwidths(r1.w);
  return make_float4(r0.x - e.x, r0.x + e.x, r0.y - e.y, r0.y + e.y);
}

constexpr int WARPS = 8;  // warps per block of the 8 x 4 kernels

__device__ __forceinline__ uint32_t warp_next_item(uint32_t *counter) {
  uint32_t it = 0;
  if ((threadIdx.x & 31) == 0) it = atomicAdd(counter, 1u);
  return __shfl_sync(0xffffffffu, it, 0);
}

// ---- per-lane walks ----
// Lane l owns pixel (l & 7, l >> 3) of the warp's 8 x 4 region. Every staged
// entry turns its ellipse box into a 32-bit mask of the region's pixels whose
// centres it covers; a bit-matrix transpose across the warp then gives each
// lane the staged entries covering its own pixel, and each lane walks only
// those (in list order). A lane evaluates far fewer entries than a group of
// lanes sharing one walk would, and no lane waits for a group.

// Warp-wide transpose of a 32 x 32 bit matrix: lane r holds row r on entry;
// on return lane c holds column c (bit r = bit c of row r). Five rounds of
// block swaps (16, 8, 4, 2, 1).
__device__ __forceinline__ uint32_t transpose32(uint32_t x) {
  const int lane = threadIdx.x & 31;
  constexpr uint32_t LO[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
#pragma unroll
  for (int r = 0; r < 5; ++r) {
    const int d = 16 >> r;
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, d);
    x = (lane & d) ? ((x & ~LO[r]) | ((y >> d) & LO[r])) : ((x & LO[r]) | ((y << d) & ~LO[r]));
  }
  return x;
}

// A tile list (or its first n entries) in walk order, 32 entries at a time: front
// to back, or back to front (BACK). Lane l holds the record of walk index j + l;
// the ids one chunk ahead and the records of the chunk held are in flight while
// earlier ones are used.
constexpr uint32_t NO_ENTRY = 0xffffffffu;
template <bool BACK>
struct EntryStream {
  const uint32_t *vals;
  const float4 *rec;
  int64_t n_req;
  uint32_t n, j;
  uint32_t id, id_next;
  float4 r0, r1;
  __device__ __forceinline__ uint32_t load_id(uint32_t i) const {
    return i < n ? vals[BACK ? n - 1u - i : i] : NO_ENTRY;
  }
  // an id past n_req: no entry, or garbage after a capacity overflow
  __device__ __forceinline__ bool valid(uint32_t i) const { return (int64_t)i < n_req; }
  __device__ __forceinline__ void load_rec() {
    if (valid(id)) {
      r0 = rec[2 * (int64_t)id];
      r1 = rec[2 * (int64_t)id + 1];
    }
  }
  __device__ __forceinline__ EntryStream(const uint32_t *list, uint32_t len, const float4 *records, int64_t nr)
      : vals(list), rec(records), n_req(nr), n(len), j(0) {
    const uint32_t lane = threadIdx.x & 31;
    id = load_id(lane);
    id_next = load_id(32u + lane);
    r0 = r1 = make_float4(0.f, 0.f, 0.f, 0.f);
    load_rec();
  }
  __device__ __forceinline__ bool more() const { return j < n; }
  __device__ __forceinline__ void next() {
    j += 32u;
    id = id_next;
    id_next = load_id(j + 32u + (threadIdx.x & 31));
    load_rec();
  }
};

// Collects 32 entries whose cover of the region is not empty from a stream
// (fewer at its end). An entry that no longer fits the batch stays with its
// lane for the next one. PICK = false: every entry is taken (8 x 8 regions of
// T = 8 lists, where nearly all cover the region), and slot k of batch b is
// walk index 32 b + k.
template <bool PICK>
struct Picker {
  float4 c0, c1;
  uint32_t id, j, cover;
  __device__ __forceinline__ Picker() : id(NO_ENTRY), j(0), cover(0) {}
  // stage(slot, r0, r1, id, j) writes an entry; cov(r0, r1) is its cover mask;
  // s_cover, s_j: [32]. Returns the number of slots filled; `mask` is the cover
  // of slot `lane`.
  template <class Stream, class Cov, class Stage>
  __device__ __forceinline__ int fill(Stream &st, uint32_t *s_cover, uint32_t *s_j, Cov cov,
                                      Stage stage, uint32_t &mask) {
    const uint32_t lane = threadIdx.x & 31;
    mask = 0;
    if constexpr (!PICK) {
      const int cnt = (int)min(32u, st.n - st.j);
      const uint32_t i = st.id, w = st.j + lane;
      const float4 r0 = st.r0, r1 = st.r1;
      st.next();
      if (st.valid(i)) {
        stage((int)lane, r0, r1, i, w);
        mask = cov(r0, r1);
      }
      __syncwarp();
      return cnt;
    } else {
      int n = 0;
      for (;;) {
        const uint32_t bal = __ballot_sync(0xffffffffu, cover != 0);
        if (bal == 0) {
          if (!st.more()) break;
          id = st.id;
          j = st.j + lane;
          c0 = st.r0;
          c1 = st.r1;
          st.next();
          cover = st.valid(id) ? cov(c0, c1) : 0u;
          continue;
        }
        const int dst = n + __popc(bal & ((1u << lane) - 1u));
        if (cover != 0 && dst < 32) {
          stage(dst, c0, c1, id, j);
          s_cover[dst] = cover;
          s_j[dst] = j;
          cover = 0;
        }
        n += __popc(bal);
        if (n >= 32) {
          n = 32;
          break;
        }
      }
      __syncwarp();
      if ((int)lane < n) mask = s_cover[lane];
      return n;
    }
  }
  __device__ __forceinline__ bool left() const { return PICK && __any_sync(0xffffffffu, cover != 0); }
};

// Slots of a picked batch (walk indices s_j, ascending, cnt of them) that come
// before walk index `first`.
__device__ __forceinline__ int slots_before(const uint32_t *s_j, int cnt, uint32_t first) {
  int k = 0;
#pragma unroll
  for (int step = 16; step > 0; step >>= 1)
    if (k + step <= cnt && s_j[k + step - 1] < first) k += step;
  if (k < cnt && s_j[k] < first) ++k;
  return k;
}

// Pixels of an 8 x 4 region whose centres lie in the box (x0, x1, y0, y1):
// bit y * 8 + x for pixel centre (cx + x, cy + y). ROWS: by row pairs (rows 0, 1
// and 2, 3 together), the entries that a pixel sees in the pixel-pair kernels.
template <bool ROWS>
__device__ __forceinline__ uint32_t region_cover(float4 b, float cx, float cy) {
  const int x0 = max(0, __float2int_ru(b.x - cx)), x1 = min(7, __float2int_rd(b.y - cx));
  const int y0 = max(0, __float2int_ru(b.z - cy)), y1 = min(3, __float2int_rd(b.w - cy));
  if (x0 > x1 || y0 > y1) return 0u;
  const uint32_t row = (0xffu >> (7 - x1)) & (0xffu << x0);
  const uint32_t rows = (0xffffffffu >> (8 * (3 - (ROWS ? y1 | 1 : y1)))) &
                        (0xffffffffu << (8 * (ROWS ? y0 & ~1 : y0)));
  return (row * 0x01010101u) & rows;
}

// The 8 x 4 pixel region of a work item, lane l at pixel (l & 7, l >> 3).
struct Region {
  int v, H, W, wx0, wy0, px, py;
  bool inside;
  int64_t rec_base, img_off, n_req;
  // tile edge T (8, 16 or 32): T / 8 regions per tile row
  __device__ __forceinline__ Region(const RenderShape &s, int64_t gt, int region, int T) {
    v = find_view(s.view, s.V, gt);
    const ViewTab vt = s.view[v];
    H = vt.H;
    W = vt.W;
    rec_base = vt.rec_off;
    img_off = vt.img_off;
    n_req = s.req[vt.req].n;
    const int64_t local = gt - vt.tile_base;
    const int tyi = (int)(local / vt.tiles_x), txi = (int)(local - (int64_t)tyi * vt.tiles_x);
    const int WX = T / 8;
    wx0 = txi * T + (region % WX) * 8;
    wy0 = tyi * T + (region / WX) * 4;
    const int lane = threadIdx.x & 31;
    px = wx0 + (lane & 7);
    py = wy0 + (lane >> 3);
    inside = px < W && py < H;
  }
  __device__ __forceinline__ int64_t pixel() const { return img_off + (int64_t)py * W + px; }
};

struct LaneFwdSmem {
  float4 a[32], b[32];
};

template <bool ROWS>
__device__ __forceinline__ void fwd_lane_item(const RasterArgs &a, int64_t gt, int region, LaneFwdSmem &sm) {
  const Region rg(a.s, gt, region, a.s.tile);
  const uint2 range = a.ranges[gt];
  const float px = rg.px + 0.5f, py = rg.py + 0.5f;
  const float cx = rg.wx0 + 0.5f, cy = rg.wy0 + 0.5f;
  float Tr = 1.f, C = 0.f;
  uint32_t last = 0;
  bool done = !rg.inside;
  EntryStream<false> st(a.vals + range.x, range.y - range.x, a.rec + 2 * rg.rec_base, rg.n_req);
  Picker<false> pk;
  for (uint32_t b0 = 0; st.more(); b0 += 32) {
    if (__all_sync(0xffffffffu, done)) break;
    uint32_t cover;
    pk.fill(st, nullptr, nullptr,
            [&](float4 r0, float4 r1) { return region_cover<ROWS>(ellipse_box(r0, r1), cx, cy); },
            [&](int k, float4 r0, float4 r1, uint32_t, uint32_t) { sm.a[k] = r0; sm.b[k] = r1; }, cover);
    uint32_t mine = transpose32(cover);  // staged entries covering this lane's pixel
    if (done) mine = 0;
    const int trips = (int)__reduce_max_sync(0xffffffffu, (uint32_t)__popc(mine));
    for (int t = 0; t < trips; ++t) {
      if (mine == 0) continue;
      const int k = __ffs(mine) - 1;
      mine &= mine - 1;
      const float4 A = sm.a[k], B = sm.b[k];
      PairEval e;
      if (!eval_pair(A.x, A.y, A.z, A.w, B.x, B.y, px, py, a.P, e)) continue;
      const float Tn = __fmaf_rn(-Tr, e.sigma, Tr);  // T (1 - sigma)
      if (Tn < a.P.t_min) {
        done = true;
        mine = 0;
        continue;
      }
      C = fmaf(B.z * e.sigma, Tr, C);
      Tr = Tn;
      last = b0 + (uint32_t)k + 1u;
    }
    __syncwarp();  // the slice is rewritten by the next batch
  }
  if (rg.inside) {
    const int64_t pix = rg.pixel();
    a.image[pix] = C;
    a.t_final[pix] = Tr;
    a.n_last[pix] = last;
  }
}

// Five resident blocks per SM (48 registers): these renders have few items per
// warp slot, and a warp with more registers finishes an item sooner (one 512^2
// view, 0.069 ms against 0.078 at eight blocks). Picking the covering entries of
// T = 16 lists first, as the pair kernels do, only lengthens a warp's serial
// chain here (100k Gaussians, one 128^2 view: 91 -> 100 us).
// ROWS: the backward of this render takes pixel pairs. The box only culls (q <=
// q_max decides), but for ellipses so thin that rounding could pass a pixel
// outside the box both passes must look at the same pixels.
template <bool ROWS>
__global__ void __launch_bounds__(WARPS * 32, 5) raster_fwd_lane_kernel(RasterArgs a) {
  const uint32_t nw = (uint32_t)(a.s.tile * a.s.tile / 32);
  __shared__ LaneFwdSmem sm[WARPS];
  const uint64_t n_items = (uint64_t)a.s.total_tiles * nw;
  after_previous();
  for (;;) {
    const uint32_t item = warp_next_item(a.counter);
    if (item >= n_items) break;
    const int64_t gt = a.order[item / nw];
    fwd_lane_item<ROWS>(a, gt, (int)(item % nw), sm[threadIdx.x >> 5]);
    if (a.req_end && (threadIdx.x & 31) == 0)
      atomicMax(a.req_end + a.s.view[find_view(a.s.view, a.s.V, gt)].req, global_ns());
  }
}

// Backward of one (tile, region) item in two phases per staged batch of 32
// entries (back to front):
//  1. every lane walks the entries covering its pixel, from the last one the
//     forward pass added, recovering T and the suffix sum S, and stores two
//     numbers per (pixel, entry) it adds: A = dL/dsigma * G (0 where sigma
//     was clamped) and Bc = dL/dc = g sigma T;
//  2. after a transpose of the (pixel, entry) bits, lane e sums entry e's
//     numbers over its pixels in registers: sum A, sum Bc and the moments
//     sum A x, A y, A x^2, A x y, A y^2 of the pixel offsets (x, y) in the
//     region. With u' = u - (region origin), dx = u' - x, dy = v' - y and
//     dL/dq = -alpha A / 2, the sums of dL/dq dx, dL/dq dy, dL/dq dx^2, ...
//     that the mean and conic gradients need follow from those moments.
// No lane reduces another lane's values and no shared-memory atomic is used.
constexpr int AB_STRIDE = 32;  // float2 per pixel row of the (pixel, entry) table
// Warps per block of the per-lane backward: 77 KB, two blocks per SM. Three (a
// batch's covers and walk indices in the table's place make room for them) are no
// faster: these renders have few items, and a warp that shares its SM with more of
// them finishes the longest list later (raster_bwd, 100k Gaussians, one view at tile
// 8: 256^2 63 and 63 us, 300^2 60 and 79, 360^2 68 and 75; 340^2 at tile 32 86 and 110).
constexpr int LANE_WARPS = 8;

struct LaneBwdSmem {
  float4 a[33], b[33];  // entry 32: a sentinel that no pixel adds
  uint32_t id[32], cover[32], j[32];
  float2 ab[32 * AB_STRIDE];  // [pixel][entry ^ pixel]: (A, Bc)
};

template <int T>
__device__ __forceinline__ void bwd_lane_item(const RasterArgs &a, int64_t gt, int region, LaneBwdSmem &sm) {
  constexpr bool PICK = T > 8;
  const int lane = threadIdx.x & 31;
  const Region rg(a.s, gt, region, T);
  const uint2 range = a.ranges[gt];
  const float px = rg.px + 0.5f, py = rg.py + 0.5f;
  const float cx = rg.wx0 + 0.5f, cy = rg.wy0 + 0.5f;
  float Tr = 1.f, g = 0.f;
  uint32_t last = 0;
  if (rg.inside) {
    const int64_t pix = rg.pixel();
    Tr = a.t_final_in[pix];
    last = a.n_last_in[pix];
    g = a.dL_dimage[pix];
  }
  if (g == 0.f) last = 0;  // nothing to propagate from this pixel
  if (last > range.y - range.x) last = range.y - range.x;  // never read past the list
  if (lane == 0) {  // q' = -inf at every pixel
    sm.a[32] = make_float4(3.0e38f, 3.0e38f, -1.f, 0.f);
    sm.b[32] = make_float4(-1.f, 0.f, 0.f, 0.f);
  }
  // the walk carries g T and g S (Tr, S), so that g drops out of the per-pair
  // products: g dC/dsigma = c gT - gS / (1 - sigma), g dC/dc = sigma gT
  Tr *= g;
  const uint32_t max_last = __reduce_max_sync(0xffffffffu, last);
  const uint32_t first = max_last - last;  // this pixel's first walk index
  float S = 0.f;
  EntryStream<true> st(a.vals + range.x, max_last, a.rec + 2 * rg.rec_base, rg.n_req);
  Picker<PICK> pk;
  for (uint32_t b0 = 0; st.more() || pk.left(); b0 += 32) {
    uint32_t cover;
    const int cnt = pk.fill(
        st, sm.cover, sm.j,
        [&](float4 r0, float4 r1) { return region_cover<false>(ellipse_box(r0, r1), cx, cy); },
        [&](int k, float4 r0, float4 r1, uint32_t id, uint32_t) { sm.a[k] = r0; sm.b[k] = r1; sm.id[k] = id; },
        cover);
    uint32_t mine = transpose32(cover);
    // the first staged entries may lie past this pixel's last added Gaussian
    int skip = 0;
    if (PICK) {
      if (cnt > 0 && first > sm.j[0]) skip = slots_before(sm.j, cnt, first);
    } else {
      skip = first > b0 ? (int)min(first - b0, 32u) : 0;
    }
    mine &= skip >= 32 ? 0u : (0xffffffffu << skip);
    uint32_t used = 0;
    const int trips = (int)__reduce_max_sync(0xffffffffu, (uint32_t)__popc(mine));
    // one entry per trip, written without branches (a lane past its last
    // entry evaluates the sentinel entry 32, whose q' is -inf, so that no
    // flag of its own is needed: 2.87 -> 2.84 ms): eval_pair's decisions, in
    // the same arithmetic. (Two entries per trip paid while the walk branched;
    // without branches the odd trip's padding costs more than the overlap
    // gives: 2.95 -> 2.93 ms.)
    // the next entry's record is read from shared memory while this one is
    // evaluated (2.92 -> 2.91 ms); the entry's own bit (the lowest of mine)
    // marks it walked and added (2.84 -> 2.83 ms)
    uint32_t bn = mine & (0u - mine);  // the next entry's bit (0 past the last)
    int kn = __popc(bn - 1u);          // its index: 32, the sentinel, past the last
    float4 An = sm.a[kn], Bn = sm.b[kn];
    for (int t = 0; t < trips; ++t) {
      const int k = kn;
      const uint32_t bit = bn;
      const float4 A = An, B = Bn;
      mine ^= bit;
      bn = mine & (0u - mine);
      kn = __popc(bn - 1u);
      An = sm.a[kn];
      Bn = sm.b[kn];
      const float dx = __fsub_rn(A.x, px), dy = __fsub_rn(A.y, py);
      const float tq = __fmaf_rn(A.w, dy, __fmul_rn(A.z, dx));
      const float q = __fmaf_rn(__fmul_rn(B.x, dy), dy, __fmul_rn(dx, tq));
      const float G = exp2_approx(q), aG = __fmul_rn(B.y, G), sigma = fminf(a.P.alpha_max, aG);
      const bool ok = !(q < a.P.q_lim || q > 0.f) && sigma >= a.P.alpha_min;
      // 1 / (1 - sigma) with sigma <= alpha_max < 1: the fast reciprocal's
      // relative error (~1 ulp) is far inside the gradient tolerance
      const float inv_om = rcp_approx(__fsub_rn(1.f, sigma));
      const float Tn = Tr * inv_om;
      const float g_dC = fmaf(B.z, Tn, -S * inv_om);  // g dC/dsigma
      const float sT = sigma * Tn;  // g dC/dc, shared with S's update (2.83 -> 2.81 ms)
      const float Sn = fmaf(B.z, sT, S);
      const float gA = (aG > a.P.alpha_max) ? 0.f : g_dC * G;
      if (ok) sm.ab[lane * AB_STRIDE + (k ^ lane)] = make_float2(gA, sT);
      Tr = ok ? Tn : Tr;
      S = ok ? Sn : S;
      used |= ok ? bit : 0u;
    }
    __syncwarp();
    uint32_t pm = transpose32(used);  // lane e: the pixels that added entry e
    if (pm) {
      float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f, s4 = 0.f, s5 = 0.f, s6 = 0.f;
      do {  // two pixels per trip: half the loop overhead, two loads in flight
        const int p = __ffs(pm) - 1;
        pm &= pm - 1;
        const bool two = pm != 0;
        const int q = two ? __ffs(pm) - 1 : p;
        pm &= pm - 1;
        const float2 ab = sm.ab[p * AB_STRIDE + (lane ^ p)];
        float2 cd = sm.ab[q * AB_STRIDE + (lane ^ q)];
        if (!two) cd = make_float2(0.f, 0.f);
        // pixel offsets in the region by conversion (a table in shared memory
        // cost bank conflicts: 2.91 -> 2.89 ms without it)
        const float x = (float)(p & 7), y = (float)(p >> 3);
        const float x2 = (float)(q & 7), y2 = (float)(q >> 3);
        const float ax = ab.x * x, ay = ab.x * y, cx2 = cd.x * x2, cy2 = cd.x * y2;
        s0 += ab.x + cd.x;
        s1 += ax + cx2;
        s2 += ay + cy2;
        s3 = fmaf(ax, x, fmaf(cx2, x2, s3));
        s4 = fmaf(ax, y, fmaf(cx2, y2, s4));
        s5 = fmaf(ay, y, fmaf(cy2, y2, s5));
        s6 += ab.y + cd.y;
      } while (pm);
      const float4 A = sm.a[lane], B = sm.b[lane];
      const float u = A.x - cx, v = A.y - cy;  // mean relative to pixel (0, 0)
      // sums over the entry's pixels of A dx, A dy, A dx^2, A dx dy, A dy^2
      const float sdx = fmaf(u, s0, -s1), sdy = fmaf(v, s0, -s2);
      const float sxx = fmaf(u, fmaf(u, s0, -2.f * s1), s3);
      const float sxy = fmaf(u, fmaf(v, s0, -s2), fmaf(-v, s1, s4));
      const float syy = fmaf(v, fmaf(v, s0, -2.f * s2), s5);
      const float hq = -0.5f * B.y;  // dL/dq = -alpha A / 2
      // dq/du = 2 (a dx + b dy), dq/dv = 2 (b dx + c dy), dq/db = 2 dx dy;
      // the record holds (a', 2b', c') = CONIC_SCALE (a, 2b, c) in A.z, A.w, B.x
      const float hk = hq * INV_CONIC_SCALE;
      const float gx = hk * sdx, gy = hk * sdy;
      const float du = fmaf(2.f * A.z, gx, A.w * gy);
      const float dv = fmaf(A.w, gx, 2.f * B.x * gy);
      float4 *dst = a.grad2d + 2 * (rg.rec_base + sm.id[lane]);
      atomicAdd(dst, make_float4(du, dv, hq * sxx, 2.f * hq * sxy));
      atomicAdd(dst + 1, make_float4(hq * syy, s0, s6, 0.f));
    }
    __syncwarp();  // the slice is rewritten by the next batch
  }
}

template <int T>
__global__ void __launch_bounds__(LANE_WARPS * 32, 3) raster_bwd_lane_kernel(RasterArgs a) {
  constexpr int NW = T * T / 32;
  extern __shared__ __align__(16) unsigned char lane_smem[];
  LaneBwdSmem &sm = reinterpret_cast<LaneBwdSmem *>(lane_smem)[threadIdx.x >> 5];
  const uint64_t n_items = (uint64_t)a.s.total_tiles * NW;
  after_previous();
  a.zero.clear();
  for (;;) {
    const uint32_t item = warp_next_item(a.counter);
    if (item >= n_items) break;
    const int64_t gt = a.order[item / NW];
    bwd_lane_item<T>(a, gt, (int)(item % NW), sm);
    if (a.req_end && (threadIdx.x & 31) == 0)
      atomicMax(a.req_end + a.s.view[find_view(a.s.view, a.s.V, gt)].req, global_ns());
  }
}

constexpr size_t LANE_BWD_SMEM = LANE_WARPS * sizeof(LaneBwdSmem);

// ---- pixel pairs: an 8 x 8 region per warp, two pixels per lane ----
// Lane l owns the pixels (l & 7, 2 (l >> 3)) and the one below it. An entry
// staged once serves 64 pixels instead of 32, a list of 8 x 8 tiles has no
// entry that misses the region, and neighbouring pixels mostly share their
// entries, so that a warp takes 10.4 trips per 32 entries of a tile where its
// two 8 x 4 halves took 16.9, and the backward's sums per entry 6.0 where they
// took 14.5 (CPU count over the benchmark's lists). The two pixels' chains are
// independent, and most of their arithmetic is done on binary32 pairs (add,
// mul and fma .rn.f32x2: one instruction, each half rounded as the scalar
// operation is). sigma is carried negated (max(-alpha_max, -alpha G)), which turns
// 1 - sigma and T (1 - sigma) into an add and an fma; every decision is the
// one eval_pair takes, bit for bit.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t p) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(p));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// A staged entry: mean, a', 2b', c', -alpha, colour. The pair kernels are bound by
// issue slots and by shared memory, whose pipe was busy 84 % forward and 86 %
// backward when each lane loaded 48 bytes a trip, the values duplicated for the
// packed units (now 68 and 76 %, issue 81 and 70 %). So an
// entry is two 16-byte pieces, in arrays of their own so that eight consecutive
// entries meet no bank conflict; duplicating in registers is cheaper (raster_fwd
// and raster_bwd at 64 views of 256^2: 1068 -> 1008 and 2168 -> 2078 us, 2M
// Gaussians on 8 of 1024^2 1418 -> 1310 and 2950 -> 2834). Smaller pieces take
// fewer cycles of the pipe but more instructions (8 bytes 1018 and 2082, 4 bytes
// 1020 and 2106), and so does q' in scalar operations (1044 and 2105).
struct PairEntry {
  float u, v, a, b, c, na, col;
};
template <int N>
struct PairSlots {
  float4 f[2][N];
  __device__ __forceinline__ void put(int k, const PairEntry &e) {
    f[0][k] = make_float4(e.u, e.v, e.a, e.b);
    f[1][k] = make_float4(e.c, e.na, e.col, 0.f);
  }
  __device__ __forceinline__ PairEntry get(int k) const {
    const float4 x = f[0][k], y = f[1][k];
    return {x.x, x.y, x.z, x.w, y.x, y.y, y.z};
  }
};

__device__ __forceinline__ PairEntry pair_entry(float4 r0, float4 r1) {
  return {r0.x, r0.y, r0.z, r0.w, r1.x, -r1.y, r1.z};
}

// q' at both pixels (eval_pair's operations); npy = (-py, -(py + 1)).
__device__ __forceinline__ uint64_t pair_q(const PairEntry &s, float px, uint64_t npy) {
  const float dx = __fsub_rn(s.u, px), m = __fmul_rn(s.a, dx);
  const uint64_t dy = add2(pack2(s.v, s.v), npy);
  const uint64_t t = fma2(pack2(s.b, s.b), dy, pack2(m, m));
  return fma2(mul2(pack2(s.c, s.c), dy), dy, mul2(pack2(dx, dx), t));
}

// The 8 x 8 pixel region of a work item.
struct PairRegion {
  int v, H, W, wx0, wy0, px, py;
  bool in0, in1;
  int64_t rec_base, img_off, n_req;
  __device__ __forceinline__ PairRegion(const RenderShape &s, int64_t gt, int region, int T) {
    v = find_view(s.view, s.V, gt);
    const ViewTab vt = s.view[v];
    H = vt.H;
    W = vt.W;
    rec_base = vt.rec_off;
    img_off = vt.img_off;
    n_req = s.req[vt.req].n;
    const int64_t local = gt - vt.tile_base;
    const int tyi = (int)(local / vt.tiles_x), txi = (int)(local - (int64_t)tyi * vt.tiles_x);
    const int WX = T / 8;
    wx0 = txi * T + (region % WX) * 8;
    wy0 = tyi * T + (region / WX) * 8;
    const int lane = threadIdx.x & 31;
    px = wx0 + (lane & 7);
    py = wy0 + 2 * (lane >> 3);
    in0 = px < W && py < H;
    in1 = px < W && py + 1 < H;
  }
  __device__ __forceinline__ int64_t pixel() const { return img_off + (int64_t)py * W + px; }
};

// Pairs of an 8 x 8 region that the box (x0, x1, y0, y1) covers a pixel centre
// of: bit 8 r + x for column x and rows 2 r, 2 r + 1.
__device__ __forceinline__ uint32_t pair_cover(float4 b, float cx, float cy) {
  const int x0 = max(0, __float2int_ru(b.x - cx)), x1 = min(7, __float2int_rd(b.y - cx));
  const int y0 = max(0, __float2int_ru(b.z - cy)), y1 = min(7, __float2int_rd(b.w - cy));
  if (x0 > x1 || y0 > y1) return 0u;
  const uint32_t row = (0xffu >> (7 - x1)) & (0xffu << x0);
  const uint32_t rows = (0xffffffffu >> (8 * (3 - (y1 >> 1)))) & (0xffffffffu << (8 * (y0 >> 1)));
  return (row * 0x01010101u) & rows;
}

// Forward of one item. Two batches of 32 entries are staged at a time: a lane
// that has walked its entries of the older batch goes on with the newer one
// instead of waiting for the busiest lane, whose share of the older batch sets
// the number of trips (7.7 trips per batch instead of 10.4 at the benchmark).
// T is negated once a pixel has stopped (every later T (1 - sigma) is then
// below t_min), and from the start outside the image.
template <bool PIX>
struct PairFwdSmem {
  PairSlots<64> slot;
  uint32_t j[64], cover[32];
  float4 z[PIX ? 64 : 1];  // (a, h_0, h_1, h_2)
};

template <int T, bool PIX>
__device__ __forceinline__ void fwd_pair_item(const RasterArgs &a, int64_t gt, int region, PairFwdSmem<PIX> &sm) {
  constexpr bool PICK = T > 8;
  const PairRegion rg(a.s, gt, region, T);
  const uint2 range = a.ranges[gt];
  const float px = rg.px + 0.5f;
  const uint64_t npy = pack2(-(rg.py + 0.5f), -(rg.py + 1.5f));
  const float cx = rg.wx0 + 0.5f, cy = rg.wy0 + 0.5f;
  const float namax = -a.P.alpha_max, namin = -a.P.alpha_min;
  PixRay ray0, ray1;
  if (PIX) {
    pixel_ray(a.world_to_cam + 12 * rg.v, a.detector + 5 * rg.v, rg.H, rg.W, px, rg.py + 0.5f, ray0);
    pixel_ray(a.world_to_cam + 12 * rg.v, a.detector + 5 * rg.v, rg.H, rg.W, px, rg.py + 1.5f, ray1);
  }
  float T0 = rg.in0 ? 1.f : -1.f, T1 = rg.in1 ? 1.f : -1.f, C0 = 0.f, C1 = 0.f;
  uint32_t last0 = 0, last1 = 0;
  bool done = !rg.in0;  // in1 implies in0
  EntryStream<false> st(a.vals + range.x, range.y - range.x, a.rec + 2 * rg.rec_base, rg.n_req);
  Picker<PICK> pk;
  uint32_t m = 0, nx = 0;         // entries left of the older and of the newer batch
  uint32_t slot = 0, pos = 1;     // first slot and first 1-based list position of m's batch
  for (uint32_t b0 = 0;; b0 += 32) {
    if (__all_sync(0xffffffffu, done)) break;
    // everything before the batch at b0 - 32 is walked
    const uint32_t half = b0 & 32u;
    if (m == 0) {
      m = nx;
      slot = half ^ 32u;
      pos = b0 - 31u;
    }
    nx = 0;
    const int trips = (int)__reduce_max_sync(0xffffffffu, (uint32_t)__popc(m));
    if (st.more() || pk.left()) {
      uint32_t cover;
      pk.fill(st, sm.cover, sm.j + half,
              [&](float4 r0, float4 r1) { return pair_cover(ellipse_box(r0, r1), cx, cy); },
              [&](int k, float4 r0, float4 r1, uint32_t id, uint32_t) {
                sm.slot.put(half + k, pair_entry(r0, r1));
                if (PIX) sm.z[half + k] = a.rec2[rg.rec_base + id];
              },
              cover);
      nx = transpose32(cover);
      if (done) nx = 0;
    } else if (trips == 0) {
      break;
    }
    uint32_t add0 = 0, add1 = 0;  // PICK: 1 + slot of the last entry added
    for (int t = 0; t < trips; ++t) {
      if (m == 0) {
        m = nx;
        nx = 0;
        slot ^= 32u;
        pos += 32u;
      }
      if (m == 0) continue;
      const uint32_t k = (uint32_t)__ffs(m) - 1u;
      m &= m - 1;
      const PairEntry s = sm.slot.get(slot + k);
      const uint64_t q = pair_q(s, px, npy);
      const float2 qf = unpack2(q);
      const float2 ng = make_float2(__fmul_rn(s.na, exp2_approx(qf.x)), __fmul_rn(s.na, exp2_approx(qf.y)));
      const float ns0 = fmaxf(namax, ng.x), ns1 = fmaxf(namax, ng.y);  // -sigma
      const bool ok0 = !(qf.x < a.P.q_lim || qf.x > 0.f) && ns0 <= namin;
      const bool ok1 = !(qf.y < a.P.q_lim || qf.y > 0.f) && ns1 <= namin;
      const uint64_t ns = pack2(ns0, ns1), Tr = pack2(T0, T1);
      const float2 Tn = unpack2(fma2(Tr, ns, Tr));  // T (1 - sigma)
      const bool st0 = ok0 && Tn.x < a.P.t_min, st1 = ok1 && Tn.y < a.P.t_min;
      // C - (colour (-sigma)) T
      float2 col = make_float2(s.col, s.col);
      if (PIX && (ok0 || ok1)) {
        const float4 z = sm.z[slot + k];
        col = make_float2(pixel_colour(ray0, z), pixel_colour(ray1, z));
      }
      const float2 w = make_float2(__fmul_rn(col.x, ns0), __fmul_rn(col.y, ns1));
      const uint32_t p = PICK ? slot + k + 1u : pos + k;
      if (ok0 && !st0) {
        C0 = fmaf(-w.x, T0, C0);
        T0 = Tn.x;
        (PICK ? add0 : last0) = p;
      }
      if (ok1 && !st1) {
        C1 = fmaf(-w.y, T1, C1);
        T1 = Tn.y;
        (PICK ? add1 : last1) = p;
      }
      if (st0 || st1) {
        if (st0) T0 = -fabsf(T0);
        if (st1) T1 = -fabsf(T1);
        if (T0 < 0.f && T1 < 0.f) {
          done = true;
          m = nx = 0;
        }
      }
    }
    if (PICK) {
      if (add0) last0 = sm.j[add0 - 1u] + 1u;
      if (add1) last1 = sm.j[add1 - 1u] + 1u;
    }
    __syncwarp();  // the older half is rewritten by the next batch
  }
  if (rg.in0) {
    const int64_t pix = rg.pixel();
    a.image[pix] = C0;
    a.t_final[pix] = fabsf(T0);
    a.n_last[pix] = last0;
    if (rg.in1) {
      a.image[pix + rg.W] = C1;
      a.t_final[pix + rg.W] = fabsf(T1);
      a.n_last[pix + rg.W] = last1;
    }
  }
}

// 32 warps per SM at 64 registers (40 at 48: 1.09 -> 1.15 ms at 64 poses, 24 at
// 80: 1.20); blocks of four warps spread a small render over more SMs than
// blocks of eight. The picking and the per-pixel instances keep more state and
// take 80 registers (100k Gaussians, 4 x 256^2 at T = 16: 71 us at 72, 66 at 80;
// per-pixel rays, 200k, 8 x 256^2 at T = 8: 154, and 165 at 96).
constexpr int PAIR_FWD_WARPS = 4, PAIR_FWD_BLOCKS = 8;
template <int T, bool PIX>
__global__ void __launch_bounds__(PAIR_FWD_WARPS * 32, PIX || T > 8 ? 6 : PAIR_FWD_BLOCKS)
raster_fwd_pair_kernel(RasterArgs a) {
  constexpr int NW = T * T / 64;
  __shared__ PairFwdSmem<PIX> sm[PAIR_FWD_WARPS];
  const uint64_t n_items = (uint64_t)a.s.total_tiles * NW;
  after_previous();
  for (;;) {
    const uint32_t item = warp_next_item(a.counter);
    if (item >= n_items) break;
    const int64_t gt = a.order[item / NW];
    fwd_pair_item<T, PIX>(a, gt, (int)(item % NW), sm[threadIdx.x >> 5]);
    if (a.req_end && (threadIdx.x & 31) == 0)
      atomicMax(a.req_end + a.s.view[find_view(a.s.view, a.s.V, gt)].req, global_ns());
  }
}

// Backward of one item, the two phases of bwd_lane_item on pixel pairs. Phase
// 1 stores, per (pair, entry) with a pixel it adds, S = A_0 + A_1, D = A_1 (A
// of the lower pixel) and the sum of -dL/dc over the pair; with x the pair's
// column and y its upper row, phase 2 gets every moment of the pixel offsets
// from sums over pairs: sum A = sum S, A x = S x, A y = S y + D, A x^2 = S x^2,
// A x y = (S y + D) x, A y^2 = S y^2 + D (2 y + 1). With per-pixel rays the
// table holds dL/dz of both pixels instead, for the sums of dL/dz and dL/dz Y.
//
// A pair adds few of a batch's 32 entries (4.4 in a regular view of 500k
// Gaussians, 11.2 in a dense fit). With per-pixel rays, whose table is twice as
// wide, a lane therefore keeps what it stores one after the other, PAIR_KEEP
// entries at most: entry e of pair p is the popc of the pair's added entries
// below e, and a longer walk is done in stretches, each with its own sums. So
// sixteen warps fit per SM, not ten (200k Gaussians on 8 views of 256^2:
// raster_bwd 347 -> 297 us; keeping 12 gives the same, 8 is 7 % slower). Without rays the [pair][entry] table stays: the
// look-ups and the second set of atomics cost more than the warps give (64 views
// of 256^2 2168 -> 2278 us, 100k Gaussians on one 512^2 view 88 -> 119).
constexpr int PAIR_KEEP = 16;
template <bool PIX>
struct PairBwdSmem {
  PairSlots<33> slot;  // entry 32: a sentinel that no pixel adds
  float4 z[PIX ? 33 : 1];   // (a, h_0, h_1, h_2)
  float4 y[PIX ? 64 : 1];   // Y_1 of the rays of the upper and of the lower pixels
  uint32_t used[PIX ? 32 : 1];  // the entries that each pair added
  uint32_t id[32], cover[32], j[32];
  static constexpr int KEEP = PIX ? PAIR_KEEP : 32;  // a lane's entries in the tables
  float2 sd[KEEP * 32];  // [pair][entry ^ pair], with rays [stored][pair]: (S, D)
  float2 dz[PIX ? KEEP * 32 : 1];  // the same: dL/dz of the two pixels
  float nb[PIX ? 1 : KEEP * 32];   // the same: -sum of dL/dc
};
// Blocks of four warps and 55 KB (45 KB with rays), sixteen warps per SM.
template <bool PIX>
struct PairBwd {
  static constexpr int WARPS = 4, BLOCKS = 4;
  static constexpr size_t SMEM = WARPS * sizeof(PairBwdSmem<PIX>);
};

template <int T, bool PIX>
__device__ __forceinline__ void bwd_pair_item(const RasterArgs &a, int64_t gt, int region, PairBwdSmem<PIX> &sm) {
  constexpr bool PICK = T > 8;
  const int lane = threadIdx.x & 31;
  const PairRegion rg(a.s, gt, region, T);
  const uint2 range = a.ranges[gt];
  const float px = rg.px + 0.5f;
  const uint64_t npy = pack2(-(rg.py + 0.5f), -(rg.py + 1.5f));
  const float cx = rg.wx0 + 0.5f, cy = rg.wy0 + 0.5f;
  const float namax = -a.P.alpha_max, namin = -a.P.alpha_min;
  const uint32_t len = range.y - range.x;
  float T0 = 0.f, T1 = 0.f;
  uint32_t last0 = 0, last1 = 0;
  if (rg.in0) {
    const int64_t pix = rg.pixel();
    const float g = a.dL_dimage[pix];
    T0 = a.t_final_in[pix] * g;  // the walk carries g T and g S
    last0 = g == 0.f ? 0u : min(a.n_last_in[pix], len);  // never read past the list
    if (rg.in1) {
      const float h = a.dL_dimage[pix + rg.W];
      T1 = a.t_final_in[pix + rg.W] * h;
      last1 = h == 0.f ? 0u : min(a.n_last_in[pix + rg.W], len);
    }
  }
  PixRay ray0, ray1;
  float gY0[3] = {0.f, 0.f, 0.f}, gY1[3] = {0.f, 0.f, 0.f};  // dL/dY_1 of the pixels' rays
  if (PIX) {
    pixel_ray(a.world_to_cam + 12 * rg.v, a.detector + 5 * rg.v, rg.H, rg.W, px, rg.py + 0.5f, ray0);
    pixel_ray(a.world_to_cam + 12 * rg.v, a.detector + 5 * rg.v, rg.H, rg.W, px, rg.py + 1.5f, ray1);
    sm.y[lane] = make_float4(ray0.Y[0], ray0.Y[1], ray0.Y[2], 0.f);
    sm.y[32 + lane] = make_float4(ray1.Y[0], ray1.Y[1], ray1.Y[2], 0.f);
  }
  if (lane == 0) {  // q' = -inf at every pixel
    sm.slot.put(32, {3.0e38f, 3.0e38f, -1.f, 0.f, -1.f, 0.f, 0.f});
    if (PIX) sm.z[32] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const uint32_t max_last = __reduce_max_sync(0xffffffffu, max(last0, last1));
  const uint32_t first0 = max_last - last0, first1 = max_last - last1;  // the pixels' first walk indices
  uint64_t nS = 0;  // -g S of both pixels
  uint64_t Tr = pack2(T0, T1);
  const uint64_t one = pack2(1.f, 1.f);
  EntryStream<true> st(a.vals + range.x, max_last, a.rec + 2 * rg.rec_base, rg.n_req);
  Picker<PICK> pk;
  for (uint32_t b0 = 0; st.more() || pk.left(); b0 += 32) {
    uint32_t cover;
    const int cnt = pk.fill(
        st, sm.cover, sm.j,
        [&](float4 r0, float4 r1) { return pair_cover(ellipse_box(r0, r1), cx, cy); },
        [&](int k, float4 r0, float4 r1, uint32_t id, uint32_t) {
          sm.slot.put(k, pair_entry(r0, r1));
          sm.id[k] = id;
          if (PIX) sm.z[k] = a.rec2[rg.rec_base + id];
        },
        cover);
    uint32_t mine = transpose32(cover);
    // the first staged entries may lie past a pixel's last added Gaussian
    int skip0, skip1;
    if (PICK) {
      skip0 = cnt > 0 && first0 > sm.j[0] ? slots_before(sm.j, cnt, first0) : 0;
      skip1 = cnt > 0 && first1 > sm.j[0] ? slots_before(sm.j, cnt, first1) : 0;
    } else {
      skip0 = first0 > b0 ? (int)min(first0 - b0, 32u) : 0;
      skip1 = first1 > b0 ? (int)min(first1 - b0, 32u) : 0;
    }
    const int skip = min(skip0, skip1);
    mine &= skip >= 32 ? 0u : (0xffffffffu << skip);
    int trips = (int)__reduce_max_sync(0xffffffffu, (uint32_t)__popc(mine));
    uint32_t bn = mine & (0u - mine);  // the next entry's bit (0 past the last)
    int kn = __popc(bn - 1u);          // its index: 32, the sentinel, past the last
    PairEntry sn = sm.slot.get(kn);
    while (trips > 0) {
      uint32_t used = 0;
      int next = lane;  // with rays: where the next stored entry goes
      for (int t = PIX ? min(trips, sm.KEEP) : trips; t > 0; --t) {
        const int k = kn;
        const uint32_t bit = bn;
        const PairEntry s = sn;
        mine ^= bit;
        bn = mine & (0u - mine);
        kn = __popc(bn - 1u);
        sn = sm.slot.get(kn);
        const float2 qf = unpack2(pair_q(s, px, npy));
        const float g0 = exp2_approx(qf.x), g1 = exp2_approx(qf.y);
        const uint64_t G = pack2(g0, g1);
        const float2 ng = make_float2(__fmul_rn(s.na, g0), __fmul_rn(s.na, g1));
        const float ns0 = fmaxf(namax, ng.x), ns1 = fmaxf(namax, ng.y);  // -sigma
        const bool ok0 = !(qf.x < a.P.q_lim || qf.x > 0.f) && ns0 <= namin && k >= skip0;
        const bool ok1 = !(qf.y < a.P.q_lim || qf.y > 0.f) && ns1 <= namin && k >= skip1;
        const uint64_t ns = pack2(ns0, ns1);
        // 1 / (1 - sigma) with sigma <= alpha_max < 1: the fast reciprocal's
        // relative error (~1 ulp) is far inside the gradient tolerance
        const float2 om = unpack2(add2(one, ns));
        const uint64_t inv = pack2(rcp_approx(om.x), rcp_approx(om.y));
        const uint64_t Tn = mul2(Tr, inv);
        uint64_t col = pack2(s.col, s.col);
        float4 z;
        float2 cf;
        if (PIX) {
          z = sm.z[k];
          cf = make_float2(pixel_colour(ray0, z), pixel_colour(ray1, z));
          col = pack2(cf.x, cf.y);
        }
        const uint64_t gdC = fma2(col, Tn, mul2(nS, inv));  // g dC/dsigma
        const uint64_t nsT = mul2(ns, Tn);                  // -g dC/dc
        const uint64_t nSn = fma2(col, nsT, nS);
        const float2 gA = unpack2(mul2(gdC, G)), nb = unpack2(nsT);
        const float A0 = ok0 && !(ng.x < namax) ? gA.x : 0.f, A1 = ok1 && !(ng.y < namax) ? gA.y : 0.f;
        const float b0_ = ok0 ? nb.x : 0.f, b1_ = ok1 ? nb.y : 0.f;
        if (ok0 || ok1) {
          const int at = PIX ? next : lane * 32 + (k ^ lane);
          sm.sd[at] = make_float2(A0 + A1, A1);
          if (PIX) {
            const float z0 = -b0_ * cf.x * (1.f - cf.x), z1 = -b1_ * cf.y * (1.f - cf.y);
            sm.dz[at] = make_float2(ok0 ? z0 : 0.f, ok1 ? z1 : 0.f);
            if (ok0) {
              gY0[0] = fmaf(z0, z.y, gY0[0]);
              gY0[1] = fmaf(z0, z.z, gY0[1]);
              gY0[2] = fmaf(z0, z.w, gY0[2]);
            }
            if (ok1) {
              gY1[0] = fmaf(z1, z.y, gY1[0]);
              gY1[1] = fmaf(z1, z.z, gY1[1]);
              gY1[2] = fmaf(z1, z.w, gY1[2]);
            }
          } else {
            sm.nb[at] = b0_ + b1_;
          }
          used |= bit;
          next += 32;
        }
        const float2 To = unpack2(Tr), Tv = unpack2(Tn), So = unpack2(nS), Sv = unpack2(nSn);
        Tr = pack2(ok0 ? Tv.x : To.x, ok1 ? Tv.y : To.y);
        nS = pack2(ok0 ? Sv.x : So.x, ok1 ? Sv.y : So.y);
      }
      trips = PIX ? trips - sm.KEEP : 0;
      if (PIX) sm.used[lane] = used;
      __syncwarp();
      uint32_t pm = transpose32(used);  // lane e: the pairs that added entry e
      const uint32_t below = (1u << lane) - 1u;
      if (pm) {
        uint64_t sd = 0, sdx = 0, sdy = 0;  // sums of (S, D), (S, D) x, (S, D) y
        float sxx = 0.f, sxy = 0.f, syy = 0.f, sb = 0.f, sh[3] = {0.f, 0.f, 0.f};
        do {  // two pairs per trip: half the loop overhead, two loads in flight
          const int p = __ffs(pm) - 1;
          pm &= pm - 1;
          const bool two = pm != 0;
          const int q = two ? __ffs(pm) - 1 : p;
          pm &= pm - 1;
          const int ip = PIX ? p + 32 * __popc(sm.used[p] & below) : p * 32 + (lane ^ p);
          const int iq = PIX ? q + 32 * __popc(sm.used[q] & below) : q * 32 + (lane ^ q);
          const float2 u = sm.sd[ip];
          float2 v = sm.sd[iq];
          if (!two) v = make_float2(0.f, 0.f);
          if (PIX) {
            const float2 zu = sm.dz[ip];
            float2 zv = sm.dz[iq];
            if (!two) zv = make_float2(0.f, 0.f);
            sb += (zu.x + zu.y) + (zv.x + zv.y);
            const float4 yu0 = sm.y[p], yu1 = sm.y[32 + p], yv0 = sm.y[q], yv1 = sm.y[32 + q];
            sh[0] = fmaf(zu.x, yu0.x, fmaf(zu.y, yu1.x, fmaf(zv.x, yv0.x, fmaf(zv.y, yv1.x, sh[0]))));
            sh[1] = fmaf(zu.x, yu0.y, fmaf(zu.y, yu1.y, fmaf(zv.x, yv0.y, fmaf(zv.y, yv1.y, sh[1]))));
            sh[2] = fmaf(zu.x, yu0.z, fmaf(zu.y, yu1.z, fmaf(zv.x, yv0.z, fmaf(zv.y, yv1.z, sh[2]))));
          } else {
            const float ub = sm.nb[ip], vb = sm.nb[iq];
            sb -= ub + (two ? vb : 0.f);
          }
          const float x = (float)(p & 7), y = (float)((p >> 2) & 6);
          const float x2 = (float)(q & 7), y2 = (float)((q >> 2) & 6);
          const uint64_t up = pack2(u.x, u.y), vp = pack2(v.x, v.y);
          sd = add2(sd, add2(up, vp));
          sdx = fma2(up, pack2(x, x), fma2(vp, pack2(x2, x2), sdx));
          sdy = fma2(up, pack2(y, y), fma2(vp, pack2(y2, y2), sdy));
          const float ax = u.x * x, ax2 = v.x * x2;
          sxx = fmaf(ax, x, fmaf(ax2, x2, sxx));
          sxy = fmaf(ax, y, fmaf(ax2, y2, sxy));
          syy = fmaf(u.x * y, y, fmaf(v.x * y2, y2, syy));
        } while (pm);
        const float2 fd = unpack2(sd), fx = unpack2(sdx), fy = unpack2(sdy);
        const float s0 = fd.x, s1 = fx.x, s2 = fy.x + fd.y, s4 = sxy + fx.y,
                    s5 = syy + fmaf(2.f, fy.y, fd.y);
        const PairEntry sl = sm.slot.get(lane);
        const float ca = sl.a, cb2 = sl.b, cc = sl.c;
        const float u = sl.u - cx, v = sl.v - cy;  // mean relative to pixel (0, 0)
        // sums over the entry's pixels of A dx, A dy, A dx^2, A dx dy, A dy^2
        const float sdx1 = fmaf(u, s0, -s1), sdy1 = fmaf(v, s0, -s2);
        const float gxx = fmaf(u, fmaf(u, s0, -2.f * s1), sxx);
        const float gxy = fmaf(u, fmaf(v, s0, -s2), fmaf(-v, s1, s4));
        const float gyy = fmaf(v, fmaf(v, s0, -2.f * s2), s5);
        const float hq = 0.5f * sl.na;  // dL/dq = -alpha A / 2
        // dq/du = 2 (a dx + b dy), dq/dv = 2 (b dx + c dy), dq/db = 2 dx dy;
        // the record holds (a', 2b', c') = CONIC_SCALE (a, 2b, c)
        const float hk = hq * INV_CONIC_SCALE;
        const float gx = hk * sdx1, gy = hk * sdy1;
        const float du = fmaf(2.f * ca, gx, cb2 * gy);
        const float dv = fmaf(cb2, gx, 2.f * cc * gy);
        const int64_t r = rg.rec_base + sm.id[lane];
        atomicAdd(a.grad2d + 2 * r, make_float4(du, dv, hq * gxx, 2.f * hq * gxy));
        atomicAdd(a.grad2d + 2 * r + 1, make_float4(hq * gyy, s0, sb, 0.f));
        if (PIX) atomicAdd(a.grad_h + r, make_float4(sh[0], sh[1], sh[2], 0.f));
      }
      __syncwarp();  // the sums of the next stretch use the same table
    }
    __syncwarp();  // the slice is rewritten by the next batch, also after one without a trip
  }
  if (PIX && a.pose_grad) {
    // Y_1(d / |d|), d = W^T rc: dL/dW[r][c] = rc[r] dL/dd[c], summed over the warp
    float w9[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) w9[i] = 0.f;
    auto add = [&](const PixRay &ray, const float gY[3]) {
      if (gY[0] == 0.f && gY[1] == 0.f && gY[2] == 0.f) return;
      const float ddh[3] = {-SH_C1 * gY[2], -SH_C1 * gY[0], SH_C1 * gY[1]};
      const float dot = ddh[0] * ray.dh[0] + ddh[1] * ray.dh[1] + ddh[2] * ray.dh[2];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float dd = (ddh[c] - ray.dh[c] * dot) * ray.inv;
#pragma unroll
        for (int r = 0; r < 3; ++r) w9[3 * r + c] = fmaf(ray.rc[r], dd, w9[3 * r + c]);
      }
    };
    add(ray0, gY0);
    add(ray1, gY1);
    const bool mine = (w9[0] != 0.f) | (w9[1] != 0.f) | (w9[2] != 0.f) | (w9[3] != 0.f) | (w9[4] != 0.f) |
                      (w9[5] != 0.f) | (w9[6] != 0.f) | (w9[7] != 0.f) | (w9[8] != 0.f);
    if (__any_sync(0xffffffffu, mine)) {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w9[i] += __shfl_xor_sync(0xffffffffu, w9[i], o);
      }
      if (lane < 9) {
        float x = w9[0];
#pragma unroll
        for (int i = 1; i < 9; ++i) if (lane == i) x = w9[i];
        if (x != 0.f) atomicAdd(a.pose_grad + 12 * (int64_t)rg.v + 4 * (lane / 3) + lane % 3, x);
      }
    }
  }
}

template <int T, bool PIX>
__global__ void __launch_bounds__(PairBwd<PIX>::WARPS * 32, PairBwd<PIX>::BLOCKS) raster_bwd_pair_kernel(RasterArgs a) {
  constexpr int NW = T * T / 64;
  extern __shared__ __align__(16) unsigned char lane_smem[];
  PairBwdSmem<PIX> &sm = reinterpret_cast<PairBwdSmem<PIX> *>(lane_smem)[threadIdx.x >> 5];
  const uint64_t n_items = (uint64_t)a.s.total_tiles * NW;
  after_previous();
  a.zero.clear();
  for (;;) {
    const uint32_t item = warp_next_item(a.counter);
    if (item >= n_items) break;
    const int64_t gt = a.order[item / NW];
    bwd_pair_item<T, PIX>(a, gt, (int)(item % NW), sm);
    if (a.req_end && (threadIdx.x & 31) == 0)
      atomicMax(a.req_end + a.s.view[find_view(a.s.view, a.s.V, gt)].req, global_ns());
  }
}

// ---- work order: all tiles by descending list length (four buckets per
// factor of two), so that the longest lists start first and the persistent
// warps finish together. Within a bucket the tiles stay roughly in order, view
// by view. (Ordering every view by itself, log2 buckets: 24 uneven requests
// raster_fwd 0.243 -> 0.193, raster_bwd 0.501 -> 0.439 ms; 100k Gaussians on
// one 512^2 view 0.065 -> 0.059 and 0.095 -> 0.088; 64 equal views of 256^2
// 1.087 -> 1.071 and 2.148 -> 2.173.) The binning's offsets kernel has counted
// the buckets; a block takes 1,024 tiles and reserves their places per bucket
// with one atomic each. ----
__global__ void __launch_bounds__(1024) tile_order_kernel(int64_t n_tiles, const uint2 *ranges,
                                                          uint32_t *lpt, uint32_t *order) {
  __shared__ uint32_t s_cnt[LPT_BUCKETS], s_w[32];
  static_assert(LPT_BUCKETS <= 1024, "one thread per bucket");
  const int t = threadIdx.x, lane = t & 31;
  const int64_t gt = (int64_t)blockIdx.x * 1024 + t;
  after_previous();
  if (t < LPT_BUCKETS) s_cnt[t] = 0;
  // longer buckets come first: thread t has bucket LPT_BUCKETS - 1 - t
  const int b = LPT_BUCKETS - 1 - t;
  const uint32_t c = b >= 0 ? lpt[b] : 0;
  uint32_t inc = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_w[t >> 5] = inc;
  __syncthreads();
  int mine = 0;
  uint32_t rank = 0;
  if (gt < n_tiles) {
    mine = lpt_bucket(ranges[gt]);
    rank = atomicAdd(&s_cnt[mine], 1u);
  }
  __syncthreads();
  if (b >= 0 && s_cnt[b]) {
    uint32_t start = inc - c + atomicAdd(&lpt[LPT_BUCKETS + b], s_cnt[b]);
    for (int w = 0; w < t >> 5; ++w) start += s_w[w];
    s_cnt[b] = start;
  }
  __syncthreads();
  if (gt < n_tiles) order[s_cnt[mine] + rank] = (uint32_t)gt;
}

// Resident blocks per SM of a kernel, cached per (device, kernel); the query
// is not a stream operation, so it is also legal while a stream is captured.
int blocks_per_sm(void (*k)(RasterArgs), int threads, size_t dyn_smem) {
  static std::mutex mu;
  static std::map<std::pair<int, const void *>, int> cache;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  const auto key = std::make_pair(dev, reinterpret_cast<const void *>(k));
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, dyn_smem) != cudaSuccess || n < 1) n = 1;
  cache[key] = n;
  return n;
}

// Pixel pairs (8 x 8 regions) where there are enough of them: with few items
// the serial walk of the longest one sets the time, and a region of half the
// pixels walks it faster. Measured fwd / bwd in us, pairs against 8 x 4
// regions, at tile 8: 256 regions (100k Gaussians, 128^2) 68.6 / 68.2 against
// 62.6 / 59.6; 1,024 (500k, 256^2) 76 / 83 against 70 / 84; 3,200 (100k, 2 x
// 320^2) 62 / 83 against 72 / 107; 8,192 (500k, 8 x 256^2) 192 / 315 against
// 223 / 379. Crowded views (depth slices) have lists so long that the forward
// needs an item for every warp slot: 4,096 regions (500k, 64 x 64^2) 922 / 920
// against 704 / 1,029, 9,216 (64 x 96^2) 428 / 677 against 439 / 862.
constexpr int64_t PAIR_MIN_ITEMS = 2048;
bool bwd_pairs(const RenderShape &s) {
  return s.total_tiles * (int64_t)(s.tile * s.tile / 64) >= PAIR_MIN_ITEMS;
}
bool fwd_pairs(const RenderShape &s) {
  const int64_t slots = (int64_t)PAIR_FWD_WARPS * PAIR_FWD_BLOCKS * device_sms();
  return bwd_pairs(s) && (!s.sliced || s.total_tiles * (int64_t)(s.tile * s.tile / 64) >= slots);
}

// A persistent grid: every resident block, at most one warp per item.
template <class Kernel>
void launch_items(Kernel k, int kid, const RasterArgs &a, int regions, int warps, size_t dyn, cudaStream_t st) {
  const int64_t need = (a.s.total_tiles * regions + warps - 1) / warps;
  const int64_t grid = std::min<int64_t>((int64_t)blocks_per_sm(k, warps * 32, dyn) * device_sms(), need);
  LaunchScope ls((KernelId)kid, st);
  launch_next(k, (unsigned)grid, (unsigned)warps * 32, dyn, st, a);
}

template <int T, bool PIX>
void launch_fwd_t(const RasterArgs &a, cudaStream_t st) {
  if (PIX || fwd_pairs(a.s)) {
    launch_items(raster_fwd_pair_kernel<T, PIX>, KID_RASTER_FWD, a, T * T / 64, PAIR_FWD_WARPS, 0, st);
    return;
  }
  auto k = bwd_pairs(a.s) ? raster_fwd_lane_kernel<true> : raster_fwd_lane_kernel<false>;
  launch_items(k, KID_RASTER_FWD, a, T * T / 32, WARPS, 0, st);
}

template <int T, bool PIX>
void launch_bwd_t(const RasterArgs &a, cudaStream_t st) {
  if (prepare_raster_kernels() != cudaSuccess) return;  // surfaces via cudaGetLastError
  if (PIX || bwd_pairs(a.s))
    launch_items(raster_bwd_pair_kernel<T, PIX>, KID_RASTER_BWD, a, T * T / 64, PairBwd<PIX>::WARPS,
                 PairBwd<PIX>::SMEM, st);
  else
    launch_items(raster_bwd_lane_kernel<T>, KID_RASTER_BWD, a, T * T / 32, LANE_WARPS, LANE_BWD_SMEM, st);
}

template <bool PIX>
void fwd_dispatch(const RasterArgs &a, int tile, cudaStream_t st) {
  if (a.s.total_tiles <= 0) return;
  switch (tile) {
    case 8: launch_fwd_t<8, PIX>(a, st); break;
    case 16: launch_fwd_t<16, PIX>(a, st); break;
    default: launch_fwd_t<32, PIX>(a, st); break;
  }
}

template <bool PIX>
void bwd_dispatch(const RasterArgs &a, int tile, cudaStream_t st) {
  if (a.s.total_tiles <= 0) return;
  switch (tile) {
    case 8: launch_bwd_t<8, PIX>(a, st); break;
    case 16: launch_bwd_t<16, PIX>(a, st); break;
    default: launch_bwd_t<32, PIX>(a, st); break;
  }
}

}  // namespace

void launch_tile_order(const RenderShape &s, ddgs_workspace &ws, cudaStream_t st) {
  if (s.total_tiles <= 0) return;
  LaunchScope ls(KID_TILE_ORDER, st);
  launch_next(tile_order_kernel, (unsigned)((s.total_tiles + 1023) / 1024), 1024u, 0, st, s.total_tiles, ws.ranges,
              ws.head->counters + LIST_CLASSES, ws.order);
}

void launch_raster_fwd(const RenderShape &s, const RasterParams &p, ddgs_workspace &ws,
                       float *image, float *t_final, uint32_t *n_last, const PixelRays *pr,
                       cudaStream_t st) {
  RasterArgs a{};
  a.s = s;
  a.P = p;
  a.rec = ws.rec;
  a.vals = ws.vals;
  a.ranges = ws.ranges;
  a.image = image;
  a.t_final = t_final;
  a.n_last = n_last;
  a.order = ws.order;
  a.counter = &ws.head->queue[0];
  a.req_end = ws.req_time ? ws.req_time + 1 : nullptr;
  if (pr) {  // per-pixel ray angles
    a.rec2 = ws.rec2;
    a.world_to_cam = pr->world_to_cam;
    a.detector = pr->detector;
    fwd_dispatch<true>(a, s.tile, st);
  } else {
    fwd_dispatch<false>(a, s.tile, st);
  }
}

void launch_raster_bwd(const RenderShape &s, const RasterParams &p, ddgs_workspace &ws,
                       const float *dL_dimage, const float *t_final, const uint32_t *n_last,
                       const PixelRays *pr, const ZeroList &zero, cudaStream_t st) {
  RasterArgs a{};
  a.s = s;
  a.P = p;
  a.rec = ws.rec;
  a.vals = ws.vals;
  a.ranges = ws.ranges;
  a.grad2d = ws.grad2d;
  a.dL_dimage = dL_dimage;
  a.t_final_in = t_final;
  a.n_last_in = n_last;
  a.order = ws.order;
  a.counter = &ws.head->queue[1];
  a.zero = zero;
  a.req_end = ws.req_time ? ws.req_time + 1 + s.R : nullptr;
  if (pr) {  // per-pixel ray angles
    a.rec2 = ws.rec2;
    a.grad_h = ws.grad_h;
    a.world_to_cam = pr->world_to_cam;
    a.detector = pr->detector;
    a.pose_grad = pr->pose_grad;
    bwd_dispatch<true>(a, s.tile, st);
  } else {
    bwd_dispatch<false>(a, s.tile, st);
  }
}

cudaError_t prepare_raster_kernels() {
  // the backward kernels keep their (pixel, entry) tables in dynamic shared
  // memory beyond the default 48 KiB; set once per device, outside any capture
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
  const struct { void (*k)(RasterArgs); size_t smem; } big[] = {
      {raster_bwd_lane_kernel<8>, LANE_BWD_SMEM}, {raster_bwd_lane_kernel<16>, LANE_BWD_SMEM},
      {raster_bwd_lane_kernel<32>, LANE_BWD_SMEM},
      {raster_bwd_pair_kernel<8, false>, PairBwd<false>::SMEM}, {raster_bwd_pair_kernel<16, false>, PairBwd<false>::SMEM},
      {raster_bwd_pair_kernel<32, false>, PairBwd<false>::SMEM},
      {raster_bwd_pair_kernel<8, true>, PairBwd<true>::SMEM}, {raster_bwd_pair_kernel<16, true>, PairBwd<true>::SMEM},
      {raster_bwd_pair_kernel<32, true>, PairBwd<true>::SMEM}};
  for (const auto &x : big) {
    e = cudaFuncSetAttribute(x.k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)x.smem);
    if (e != cudaSuccess) return e;
  }
  if (dev >= 0 && dev < 64) done[dev] = true;
  return cudaSuccess;
}

// Streaming multiprocessors of the current device (cached per device).
int device_sms() {
  static int sms[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return 152;
  if (!sms[dev]) {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    sms[dev] = n > 0 ? n : 152;
  }
  return sms[dev];
}

}  // namespace ddgs
