// Screen-space photon splat: the renderer's "splat/gather" step of Fig. 2.
// The paper only cites its splatting method, so this is a plain radius
// kernel, evaluated as a gather.  k_view_count casts one primary ray per pixel
// through the scene's BVH (visible point, normal facing the camera,
// primitive).  The photons are sorted by the cells of a grid over space (count with
// ranks, scan, place), skipping those whose kernel cube reaches the near plane.
// k_gather and k_gather_dense then take the pixels in tiles of 8 x 4 and give each
// the photons of the cells around its visible point p: every photon x with
// energy E arriving on the visible side and s = |p - x| / r < 1 adds
// rho/pi E 2 (1 - s^2) / (pi r^2).  Each pixel is written once, without
// atomics, and the work per pixel is bounded by the photons near it, not by
// how many pixels a photon's footprint covers.
#include <algorithm>
#include <cmath>

#include "pv_scene.h"

using namespace pvk;

namespace {

struct Cam {
  float3 pos, f, r, u;       // centre, forward, right, up (unit)
  float tx, ty;              // tan of the half field of view, horizontal and vertical
  uint32_t W, H;
  float znear;               // photons whose kernel cube reaches closer are skipped
};

struct GPixel {              // 32 bytes per pixel
  float4 p;                  // visible point, w = primitive id bits (-1: background)
  float4 n;                  // normal facing the camera
};

// Grid over space: cells of edge radius / kCellsPerRadius.  A photon within ``radius`` of a point lies at most
// kReach cells from the point's cell along every axis.  Cells next to each other
// in x are next to each other in the sorted photons, so the cells around points in
// a box are a few ranges (rows).
//
// Where the scene's extent has few enough cells, axes wrap around after nx, ny, nz
// cells, numbered with x fastest; each axis has at least 2 kReach + 2 cells, so the
// cells around a point are distinct and hold every photon once.  Otherwise (small
// radii) there is one row of nx = ``cells`` (a power of two) places around which
// cell (x, y, z) lies at x + sy y + sz z: the rows of a group of points are
// distinct (rows_distinct), and photons on a plane or in a box spread over all
// places as a hash spreads them.  (Axes that wrap earlier instead lay the cells of
// a plane on each other: 2.5M photon places over a floor, 700 x 500 points, r = 2 mm
// 813 us, 147 in one row; r = 20 mm 330 and 101; the 1M-path city at 1920 x 1080
// 1149 and 966 us at 2 mm, 541 and 529 at 0.1 m.)  Points far apart may share a
// place: such photons fail the distance test.
constexpr int kCellsPerRadius = 1;
constexpr int kReach = kCellsPerRadius;
constexpr int kSpread = 2;         // cells between points gathered together (k_gather); city, four warps: 1 0.51 ms, 2 0.47, 3 0.51, 4 0.60

struct Grid {
  float inv_edge;
  int nx, ny, nz;
  uint32_t cells;
  uint32_t sy, sz;             // sy = 0: axes wrap by themselves
};

// sy and sz of ``cells`` places: the two-dimensional low-discrepancy sequence of the
// plastic number p = 1.3247 (1/p and 1/p^2 of the places).
constexpr uint32_t stride_y(uint32_t cells) { return (uint32_t)(0.7548776662466927 * cells) | 1u; }
constexpr uint32_t stride_z(uint32_t cells) { return (uint32_t)(0.5698402909980532 * cells) | 1u; }

// Whether the rows around a group of points, at most 2 (kSpread + kReach) apart in y
// and in z and one more cell long, never overlap.
constexpr bool rows_distinct(uint32_t cells) {
  constexpr int kSpan = 2 * (kSpread + kReach);
  for (int dy = -kSpan; dy <= kSpan; ++dy)
    for (int dz = 0; dz <= kSpan; ++dz) {
      if (dz == 0 && dy <= 0) continue;
      const uint32_t d = ((uint32_t)dy * stride_y(cells) + (uint32_t)dz * stride_z(cells)) & (cells - 1u);
      if (d < kSpan + 1u || cells - d < kSpan + 1u) return false;
    }
  return true;
}
constexpr uint32_t kMinCells = 2048, kMaxCells = 1u << 30;
constexpr bool all_rows_distinct() {
  for (uint32_t c = kMinCells; c <= kMaxCells; c <<= 1)
    if (!rows_distinct(c)) return false;
  return true;
}
static_assert(all_rows_distinct(), "a photon would be met twice");

__device__ __forceinline__ int3 grid_cell(const Grid& g, float3 x) {
  const float lim = 1.0e9f;
  return make_int3((int)fminf(fmaxf(floorf(x.x * g.inv_edge), -lim), lim),
                   (int)fminf(fmaxf(floorf(x.y * g.inv_edge), -lim), lim),
                   (int)fminf(fmaxf(floorf(x.z * g.inv_edge), -lim), lim));
}

__device__ __forceinline__ int wrap(int c, int n) {
  const int m = c % n;
  return m < 0 ? m + n : m;
}

// First place of the row of cells (., cy, cz) where axes wrap by themselves.
__device__ __forceinline__ uint32_t grid_row(const Grid& g, int cy, int cz) {
  return ((uint32_t)wrap(cz, g.nz) * g.ny + (uint32_t)wrap(cy, g.ny)) * g.nx;
}

// Place of a cell in a grid of one row.
__device__ __forceinline__ uint32_t row_place(const Grid& g, int cx, int cy, int cz) {
  return ((uint32_t)cx + g.sy * (uint32_t)cy + g.sz * (uint32_t)cz) & (g.cells - 1u);
}

__device__ __forceinline__ uint32_t grid_index(const Grid& g, int3 c) {
  return g.sy ? row_place(g, c.x, c.y, c.z) : grid_row(g, c.y, c.z) + (uint32_t)wrap(c.x, g.nx);
}

// One primary ray per pixel, a warp per 8 x 4 pixels (its rays then visit much
// the same nodes: city at 1920 x 1080 0.277 ms in rows of 32 pixels, 0.232 ms in
// tiles, 0.222 ms with five blocks per SM asked of the register allocator; six
// take 0.237 ms).
__device__ __forceinline__ void gbuffer_tile(const SceneView& sv, const Cam& c, GPixel* g, uint32_t tile) {
  const uint32_t tiles_x = (c.W + 15u) / 16u;
  const uint32_t w = threadIdx.x >> 5, l = threadIdx.x & 31u;
  const uint32_t i = (tile % tiles_x) * 16u + (w & 1u) * 8u + (l & 7u);
  const uint32_t j = (tile / tiles_x) * 16u + (w >> 1) * 4u + (l >> 3);
  if (i >= c.W || j >= c.H) return;
  const float x = (2.0f * ((float)i + 0.5f) / (float)c.W - 1.0f) * c.tx;
  const float y = (1.0f - 2.0f * ((float)j + 0.5f) / (float)c.H) * c.ty;
  const float3 d = normalize(c.f + x * c.r + y * c.u);
  const Ray r = make_ray(c.pos, d, 0.0f);
  Hit h;
  Work wk;
  GPixel o;
  o.p = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
  o.n = make_float4(0.f, 0.f, 0.f, 0.f);
  const int root = *sv.root;
  if (closest_hit<kStack, true>(sv, root, r, -1, h, wk)) {
    const Tri T = load_tri(sv.tris, h.tri);
    const float3 p = make_float3(fmaf(h.t, d.x, c.pos.x), fmaf(h.t, d.y, c.pos.y), fmaf(h.t, d.z, c.pos.z));
    float3 nn = normalize(cross(f3(T.e1), f3(T.e2)));
    if (dot(nn, d) > 0.0f) nn = -1.0f * nn;
    o.p = make_float4(p.x, p.y, p.z, T.v0.w);
    o.n = make_float4(nn.x, nn.y, nn.z, 0.f);
  }
  g[(size_t)j * c.W + i] = o;
}

// A photon takes part when every corner of its kernel cube lies beyond the
// near plane (its screen footprint is then bounded).
__device__ __forceinline__ bool in_front(const Cam& c, float3 x, float radius) {
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float3 cor = make_float3(x.x + ((q & 1) ? radius : -radius), x.y + ((q & 2) ? radius : -radius),
                                   x.z + ((q & 4) ? radius : -radius));
    if (!(dot(cor - c.pos, c.f) > c.znear)) return false;
  }
  return true;
}

// The photons that take part, sorted by cell: position, the segment they
// arrive along (position minus the path's previous vertex) and energy.
struct Photons {
  float4* xd;                  // pairs: position, w = energy.x; arriving segment, w = energy.y
  float* e;                    // energy.z
};

constexpr uint32_t kSkipped = 0xFFFFFFFFu;

// The paths whose photons are sorted and gathered in one pass: all of them, or a
// part in a workspace that does not hold all (SplatLayout).
struct PathRange {
  uint32_t first, count;
};

// Count the photons per cell; rank[k count + i] = the rank within its cell of
// photon k of the range's path i, so that placing needs no second round of atomics.  A thread per path,
// which has the loads (and then the atomics) of kRowsAtOnce rows in flight.
// (Measured on the city, 2.0M photons, as kernels of their own: count 54 us and
// place 73 us at 2 rows, 57 and 85 us at 4, 49 and 110 us one at a time; a thread
// per photon, exiting where a path is shorter, 57 and 107 us.)
constexpr uint32_t kRowsAtOnce = 2;

__device__ __forceinline__ void count_photons(const Cam& c, const Grid& g, float radius, PathRange R, uint32_t n,
                                              uint32_t B, const uint32_t* info, const float4* pa, uint32_t* counts,
                                              uint32_t* rank, uint32_t i) {
  if (i >= R.count) return;
  const uint32_t p = R.first + i;
  const uint32_t L = min(info_nseg(info[p]), B);
  for (uint32_t k0 = 0; k0 < L; k0 += kRowsAtOnce) {
    float4 x[kRowsAtOnce];
    uint32_t r[kRowsAtOnce];
#pragma unroll
    for (uint32_t q = 0; q < kRowsAtOnce; ++q)
      if (k0 + q < L) x[q] = pa[(size_t)(k0 + q) * n + p];
#pragma unroll
    for (uint32_t q = 0; q < kRowsAtOnce; ++q) {
      r[q] = kSkipped;
      if (k0 + q < L && in_front(c, f3(x[q]), radius)) r[q] = atomicAdd(counts + grid_index(g, grid_cell(g, f3(x[q]))), 1u);
    }
#pragma unroll
    for (uint32_t q = 0; q < kRowsAtOnce; ++q)
      if (k0 + q < L) rank[(size_t)(k0 + q) * R.count + i] = r[q];
  }
}

// Place the photons (starts: exclusive prefix of the counts).
__global__ void __launch_bounds__(256) k_photon_place(Grid g, PathRange R, uint32_t n, uint32_t B, const uint32_t* info,
                                                      const float* origin, const float4* pa, const float4* pb,
                                                      const uint32_t* starts, const uint32_t* rank, Photons out) {
  grid_dependency_wait();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, p = R.first + i;
  if (i >= R.count) return;
  const uint32_t L = min(info_nseg(info[p]), B);
  if (L == 0) return;
  float3 prev = make_float3(origin[p], origin[n + p], origin[2 * (size_t)n + p]);
  for (uint32_t k0 = 0; k0 < L; k0 += kRowsAtOnce) {
    float4 x[kRowsAtOnce], e[kRowsAtOnce];
    uint32_t r[kRowsAtOnce];
#pragma unroll
    for (uint32_t q = 0; q < kRowsAtOnce; ++q) {
      r[q] = kSkipped;
      if (k0 + q < L) {
        x[q] = pa[(size_t)(k0 + q) * n + p];
        e[q] = pb[(size_t)(k0 + q) * n + p];
        r[q] = rank[(size_t)(k0 + q) * R.count + i];
      }
    }
#pragma unroll
    for (uint32_t q = 0; q < kRowsAtOnce; ++q)
      if (r[q] != kSkipped) r[q] += starts[grid_index(g, grid_cell(g, f3(x[q])))];
#pragma unroll
    for (uint32_t q = 0; q < kRowsAtOnce; ++q) {
      if (k0 + q >= L) break;
      if (r[q] != kSkipped) {
        const float3 d = f3(x[q]) - prev;
        out.xd[2 * (size_t)r[q]] = make_float4(x[q].x, x[q].y, x[q].z, e[q].x);
        out.xd[2 * (size_t)r[q] + 1] = make_float4(d.x, d.y, d.z, e[q].y);
        out.e[r[q]] = e[q].z;
      }
      prev = f3(x[q]);
    }
  }
}

// Primary rays and the count of the photons need nothing of each other and are one
// launch: the count's waits on memory and atomics are hidden behind the rays (a room
// at 641 x 361 68 -> 62 us; on the city, where both fill the chip, 9 us less.
// Placing the photons beside half of the rays in the same way gained nothing more).
// Two kinds of blocks in one grid, the fewer ones at every stride-th place.
struct Mix {
  uint32_t few, stride, total;
  bool photons_few;
};

Mix mix_blocks(uint32_t photon_blocks, uint32_t pixel_blocks) {
  Mix m;
  m.photons_few = photon_blocks <= pixel_blocks;
  m.few = std::min(photon_blocks, pixel_blocks);
  m.total = photon_blocks + pixel_blocks;
  m.stride = m.few ? m.total / m.few : 1u;
  return m;
}

// Whether block b is one of the photons' blocks; index: which one of its kind.
__device__ __forceinline__ bool mix_photons(const Mix& m, uint32_t b, uint32_t& index) {
  const uint32_t before = min((b + m.stride - 1u) / m.stride, m.few);    // of the fewer kind
  const bool few = before < m.few && b == before * m.stride;
  index = few ? before : b - before;
  return few == m.photons_few;
}

__global__ void __launch_bounds__(256, 5) k_view_count(Mix m, SceneView sv, Cam c, Grid g, float radius, PathRange R,
                                                       uint32_t n, uint32_t B, const uint32_t* info, const float4* pa,
                                                       uint32_t* counts, uint32_t* rank, GPixel* gb) {
  grid_dependency_wait();
  uint32_t i;
  if (mix_photons(m, blockIdx.x, i)) count_photons(c, g, radius, R, n, B, info, pa, counts, rank, i * 256u + threadIdx.x);
  else gbuffer_tile(sv, c, gb, i);
}

// Exclusive scan of m = tiles * 4096 counters: tile sums, their scan, then
// each tile's own scan plus its offset.
__global__ void __launch_bounds__(1024) k_tile_sums(const uint32_t* v, uint32_t* sums) {
  grid_dependency_wait();
  __shared__ uint32_t w[32];
  const uint4 x = reinterpret_cast<const uint4*>(v)[(size_t)blockIdx.x * 1024 + threadIdx.x];
  uint32_t t = __reduce_add_sync(0xffffffffu, x.x + x.y + x.z + x.w);
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x < 32) {
    t = __reduce_add_sync(0xffffffffu, w[threadIdx.x]);
    if (threadIdx.x == 0) sums[blockIdx.x] = t;
    if (blockIdx.x == 0 && threadIdx.x < 2) sums[gridDim.x + 1 + threadIdx.x] = 0u;    // the dense tiles' counters
  }
}

__global__ void __launch_bounds__(1024) k_tile_scan(uint32_t* v, const uint32_t* offs) {
  grid_dependency_wait();
  __shared__ uint32_t w[32];
  uint4* p = reinterpret_cast<uint4*>(v) + (size_t)blockIdx.x * 1024 + threadIdx.x;
  const uint4 x = *p;
  const uint32_t own = x.x + x.y + x.z + x.w;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) w[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    uint32_t s = w[lane], si = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, si, o);
      if (lane >= o) si += y;
    }
    w[lane] = si - s;
  }
  __syncthreads();
  const uint32_t base = offs[blockIdx.x] + w[wid] + incl - own;
  *p = make_uint4(base, base + x.x, base + x.x + x.y, base + x.x + x.y + x.z);
}

// Packed single-precision operations of sm_100 and later, each half rounded as
// the scalar instruction rounds it.
__device__ __forceinline__ unsigned long long pack2(float2 v) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(v.x), "f"(v.y));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long r) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
  return v;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)), "l"(pack2(c)));
  return unpack2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
  return unpack2(r);
}
// (a, a) - b
__device__ __forceinline__ float2 sub2(float a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(make_float2(a, a))), "l"(pack2(make_float2(-b.x, -b.y))));
  return unpack2(r);
}

// Order-preserving map of floats to integers, for warp-wide minima and maxima.
__device__ __forceinline__ int ordered(float f) {
  const int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7FFFFFFF;
}
__device__ __forceinline__ float unordered(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7FFFFFFF); }
__device__ __forceinline__ float warp_min(float f) { return unordered(__reduce_min_sync(0xffffffffu, ordered(f))); }
__device__ __forceinline__ float warp_max(float f) { return unordered(__reduce_max_sync(0xffffffffu, ordered(f))); }

// Every visible pixel gathers the photons around its visible point, a warp for
// 8 x 4 pixels, which mostly see points close to each other.  The warp looks up the
// rows of cells around the box of these points (a lane per row), deals their
// photons out to its lanes 32 at a time (coalesced loads), keeps those within the
// radius of the box in shared memory, and walks the kept ones with all lanes
// together: every photon is a broadcast read and a test against each lane's pixel.
// Where the points spread over more than kSpread cells beyond the first one (an
// edge in depth), the warp takes them group by group.  The kept photons lie word by
// word, so that four of them are tested with packed arithmetic (fma.rn.f32x2) on
// 16-byte reads.
//
// A tile that meets more than kDenseAt photons (under a lamp, or with many groups)
// is left to k_gather_dense, where a block of kDenseParts warps deals its photons
// out.  Photons per tile differ by a thousand times within one image: with one
// warp for every tile the densest finish long after the others, with several the
// look-up of the rows, which each of them repeats, is most of the light tiles' time.
//
// Bound by issue: on the 1M-path city at 1920 x 1080 and r = 0.3 m (2.0M photons)
// the two take 0.34 ms (one warp for every tile 0.61 ms, two 0.45, four 0.43; one
// photon at a time and four warps 0.46).  With 100k paths 0.105 ms (four warps
// 0.264), r = 0.15 m 0.215 ms (0.402), at 960 x 360 0.256 ms (0.331), 300k paths of a
// smaller district at 1076 x 704 0.137 ms (0.151), a room at 641 x 361 31 us (34).
// A thread per pixel walking 27 hashed cells, which read each photon's
// previous vertex from the path buffers, took 3.57 ms on the city (1.14 ms with
// cells sorted by row and the segment in the record: long waits on loads at 12 of
// 32 lanes); two pixels per lane and cells of half the radius were slower than one
// and the whole radius (0.58 and 0.63 against 0.47 ms, four warps).
// Photons met (city, room and the district at 1076 x 704, us): 512 348, 31, 141; 1024
// 341, 31, 137; 1536 349, 31, 138; 2048 358, 31, 147.  Warps, at 1024: 4 358, 31, 140;
// 16 381, 31, 145.
constexpr uint32_t kDenseAt = 1024;
constexpr int kDenseParts = 8;
constexpr uint32_t kAloneMet = 32;   // walk_alone

// What the gather reads and writes.  The dense tiles are listed in the unused
// words of the visible points' normals (a tile has at least one pixel), which
// k_gather itself never reads; their number and a ticket follow the photons' total.
struct Gather {
  Cam c;
  Grid g;
  float radius;
  GPixel* gb;
  const uint32_t* starts;
  Photons ph;
  uint32_t* dense;                 // number of dense tiles, ticket
  float* image;
  bool add;                        // onto the image of the passes before
};

// Each pixel's photons by its own lane, for tiles whose points lie apart: at radii
// small against the scene every pixel is a group of its own, and a warp that takes
// 32 groups one after the other looks up nine rows for a handful of photons each
// time.  False, with the sums spoilt, once some pixel has met more than kAloneMet
// photons; the tile's groups are then gathered as usual.
// 1M-path city at 1920 x 1080, r = 1 mm: 975 -> 570 us (hashed cells, a thread a
// pixel: 768); 100k paths 744 -> 345 (560); a room at 641 x 361, r = 0.1 mm 118 -> 63
// (88).  Taken where a tile's first pixel and its last are groups of their own, in grids
// of one row only: taken at groups of up to 4, 8 or 16 pixels and up to 64 or 256
// photons met it is faster still at such radii, but what the tiles that give up have
// spent costs the city image 2 to 25 % at r = 0.1 to 0.4 m; on the first pixel alone it
// cost small images of districts at such radii 2 to 8 %.
__device__ __forceinline__ bool walk_alone(const Gather& G, bool todo, int3 cell, float3 P, float3 N, float2 (&sum)[3]) {
  const Grid& g = G.g;
  const uint32_t* const starts = G.starts;
  const float inv_r2 = 1.0f / (G.radius * G.radius);
  constexpr int kSide = 2 * kReach + 1;
  uint32_t met = 0;
#pragma unroll 1
  for (int r = 0; r < kSide * kSide; ++r) {
    uint32_t beg = 0, cnt = 0, beg2 = 0, cnt2 = 0;   // where the row wraps, the rest of it at its start
    if (todo) {
      const uint32_t x = row_place(g, cell.x - kReach, cell.y - kReach + r % kSide, cell.z - kReach + r / kSide);
      const uint32_t end = x + kSide;
      beg = starts[x];
      cnt = starts[min(end, g.cells)] - beg;
      if (end > g.cells) {
        beg2 = starts[0];
        cnt2 = starts[end - g.cells] - beg2;
      }
      met += cnt + cnt2;
    }
    if (__any_sync(0xffffffffu, met > kAloneMet)) return false;
    for (uint32_t k = 0; k < cnt + cnt2; ++k) {      // at most kAloneMet
      const uint32_t i = k < cnt ? beg + k : beg2 + (k - cnt);
      const float4 x = __ldg(G.ph.xd + 2 * (size_t)i);
      const float dx = P.x - x.x, dy = P.y - x.y, dz = P.z - x.z;
      const float w = fmaf(-inv_r2, fmaf(dz, dz, fmaf(dy, dy, dx * dx)), 1.0f);
      if (w > 0.0f) {
        const float4 d = __ldg(G.ph.xd + 2 * (size_t)i + 1);
        if (fmaf(N.x, d.x, fmaf(N.y, d.y, N.z * d.z)) < 0.0f) {
          sum[0].x = fmaf(x.w, w, sum[0].x);
          sum[1].x = fmaf(d.w, w, sum[1].x);
          sum[2].x = fmaf(__ldg(G.ph.e + i), w, sum[2].x);
        }
      }
    }
    __syncwarp();
  }
  return true;
}

// One tile, by kParts warps of which this is number ``part``.  With kParts = 1 a
// tile that meets more than kDenseAt photons is listed instead.
template <int kParts, bool kOneRow>
__device__ __forceinline__ void gather_tile(const SceneView& sv, const Gather& G, uint32_t tile, int part) {
  const Cam& c = G.c;
  const Grid& g = G.g;
  const float radius = G.radius;
  const GPixel* const gb = G.gb;
  const uint32_t* const starts = G.starts;
  const Photons& ph = G.ph;
  constexpr int kBuf = 64;         // photons kept before they are tested: at most 32 left over plus 32 new
  enum { kX, kY, kZ, kDx, kDy, kDz, kEx, kEy, kEz, kWords };
  __shared__ __align__(16) float s_ph[kParts][kWords][kBuf];
  __shared__ float s_acc[kParts > 1 ? kParts : 1][3][32];
  const int lane = threadIdx.x & 31;
  const uint32_t tiles_x = (c.W + 7u) / 8u;
  const uint32_t pi = (tile % tiles_x) * 8u + (lane & 7), pj = (tile / tiles_x) * 4u + (lane >> 3);
  const bool inside = pi < c.W && pj < c.H;
  const float inv_r2 = 1.0f / (radius * radius);
  const float away = 3.0e18f;      // beyond every photon's radius
  float3 P = make_float3(0.f, 0.f, 0.f), nrm = P, Q = P, N = P;   // Q, N: P and nrm within the group
  int prim = -1;
  if (inside) {
    const GPixel* q = gb + ((size_t)pj * c.W + pi);
    const float4 p = q->p;
    prim = __float_as_int(p.w);
    if (prim >= 0) {
      P = f3(p);
      const float2 nxy = *reinterpret_cast<const float2*>(&q->n);    // not n.w, which other warps write (Gather)
      nrm = make_float3(nxy.x, nxy.y, q->n.z);
    }
  }
  const int3 cell = grid_cell(g, P);
  bool todo = prim >= 0;
  uint32_t met = 0;                // photons in the rows of cells so far
  uint32_t kept = 0;               // photons in the buffer
  float2 sum[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  float(&ph_s)[kWords][kBuf] = s_ph[part];
  bool odd = false;                // some photon of the buffer has an energy that is not finite
  auto test_kept = [&]() {
    const uint32_t n4 = (kept + 3u) & ~3u;
    if (kept + lane < n4)              // filled up with photons that light no side
#pragma unroll
      for (int k = 0; k < kWords; ++k) ph_s[k][kept + lane] = 0.f;
    __syncwarp();
    for (uint32_t i = 0; i < n4; i += 4) {
      const auto word = [&](int k) { return *reinterpret_cast<const float4*>(&ph_s[k][i]); };
      const float4 x = word(kX), y = word(kY), z = word(kZ);
      float2 w[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 dx = sub2(Q.x, h ? make_float2(x.z, x.w) : make_float2(x.x, x.y));
        const float2 dy = sub2(Q.y, h ? make_float2(y.z, y.w) : make_float2(y.x, y.y));
        const float2 dz = sub2(Q.z, h ? make_float2(z.z, z.w) : make_float2(z.x, z.y));
        w[h] = fma2(make_float2(-inv_r2, -inv_r2), fma2(dz, dz, fma2(dy, dy, mul2(dx, dx))), make_float2(1.f, 1.f));
      }
      if (!(fmaxf(fmaxf(w[0].x, w[0].y), fmaxf(w[1].x, w[1].y)) > 0.0f)) continue;
      const float4 sx = word(kDx), sy = word(kDy), sz = word(kDz), ex = word(kEx), ey = word(kEy), ez = word(kEz);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        // a photon counts within the radius, and where it arrives on the visible side
        const float2 side = fma2(make_float2(N.x, N.x), h ? make_float2(sx.z, sx.w) : make_float2(sx.x, sx.y),
                                 fma2(make_float2(N.y, N.y), h ? make_float2(sy.z, sy.w) : make_float2(sy.x, sy.y),
                                      mul2(make_float2(N.z, N.z), h ? make_float2(sz.z, sz.w) : make_float2(sz.x, sz.y))));
        const float2 v = make_float2(side.x < 0.0f ? fmaxf(w[h].x, 0.0f) : 0.0f, side.y < 0.0f ? fmaxf(w[h].y, 0.0f) : 0.0f);
        float2 a = h ? make_float2(ex.z, ex.w) : make_float2(ex.x, ex.y);
        float2 b = h ? make_float2(ey.z, ey.w) : make_float2(ey.x, ey.y);
        float2 c = h ? make_float2(ez.z, ez.w) : make_float2(ez.x, ez.y);
        if (odd) {                     // infinity times a weight of 0 would not be nothing
          if (!(v.x > 0.0f)) a.x = b.x = c.x = 0.0f;
          if (!(v.y > 0.0f)) a.y = b.y = c.y = 0.0f;
        }
        sum[0] = fma2(a, v, sum[0]);
        sum[1] = fma2(b, v, sum[1]);
        sum[2] = fma2(c, v, sum[2]);
      }
    }
    __syncwarp();
    kept = 0;
    odd = false;
  };
  // the group of the first pixel left: those within kSpread cells of it
  const auto group = [&](unsigned left, int3& c0) {
    const int src = __ffs(left) - 1;
    c0 = make_int3(__shfl_sync(0xffffffffu, cell.x, src), __shfl_sync(0xffffffffu, cell.y, src),
                   __shfl_sync(0xffffffffu, cell.z, src));
    return todo && abs(cell.x - c0.x) <= kSpread && abs(cell.y - c0.y) <= kSpread && abs(cell.z - c0.z) <= kSpread;
  };
  if (kParts == 1 && kOneRow) {
    const unsigned left = __ballot_sync(0xffffffffu, todo);
    int3 c0;
    const auto single = [&](unsigned from) { return __popc(__ballot_sync(0xffffffffu, group(from, c0))) == 1; };
    if (left && single(left) && single(0x80000000u >> __clz(left))) {       // the first pixel and the last
      if (walk_alone(G, todo, cell, P, nrm, sum)) todo = false;
      else sum[0] = sum[1] = sum[2] = make_float2(0.f, 0.f);
    }
  }
  for (;;) {
    const unsigned left = __ballot_sync(0xffffffffu, todo);
    if (!left) break;
    int3 c0;
    const bool in = group(left, c0);
    todo = todo && !in;
    Q = in ? P : make_float3(away, away, away);
    N = in ? nrm : make_float3(0.f, 0.f, 0.f);
    const int3 lo = make_int3(__reduce_min_sync(0xffffffffu, in ? cell.x : c0.x),
                              __reduce_min_sync(0xffffffffu, in ? cell.y : c0.y),
                              __reduce_min_sync(0xffffffffu, in ? cell.z : c0.z));
    const int3 hi = make_int3(__reduce_max_sync(0xffffffffu, in ? cell.x : c0.x),
                              __reduce_max_sync(0xffffffffu, in ? cell.y : c0.y),
                              __reduce_max_sync(0xffffffffu, in ? cell.z : c0.z));
    float3 bl = make_float3(warp_min(in ? P.x : away), warp_min(in ? P.y : away), warp_min(in ? P.z : away));
    float3 bh = make_float3(warp_max(in ? P.x : -away), warp_max(in ? P.y : -away), warp_max(in ? P.z : -away));
    // the box grown by the radius, and by what rounding may take off its corners and the distances
    const float mag = fmaxf(fmax3(fabsf(bl.x), fabsf(bl.y), fabsf(bl.z)), fmax3(fabsf(bh.x), fabsf(bh.y), fabsf(bh.z)));
    const float grow = radius * 1.00001f + mag * 4.0e-7f;
    bl = make_float3(bl.x - grow, bl.y - grow, bl.z - grow);
    bh = make_float3(bh.x + grow, bh.y + grow, bh.z + grow);
    // rows of cells around the group (each axis at most once around the grid); a row is two ranges where it wraps
    const int ny = min(hi.y - lo.y + 1 + 2 * kReach, g.ny), nz = min(hi.z - lo.z + 1 + 2 * kReach, g.nz);
    const int len = min(hi.x - lo.x + 1 + 2 * kReach, g.nx);
    const int rows = ny * nz;
    int x0 = 0, over = 0;                        // the rows' first cell, and how many lie beyond its end
    const uint32_t place = kOneRow ? row_place(g, lo.x - kReach, lo.y - kReach, lo.z - kReach) : 0u;   // of row 0
    const int whole = (rows + 31) & ~31;         // in one row some rows may wrap: their second ranges follow from here
    if (!kOneRow) {
      x0 = wrap(lo.x - kReach, g.nx);
      over = x0 + len - g.nx;
    }
    int ranges = over > 0 ? 2 * rows : rows;
    for (int r0 = 0; r0 < ranges; r0 += 32) {
      uint32_t beg = 0, cnt = 0;
      if (kOneRow) {
        const bool second = r0 >= whole;
        const int r = r0 + lane - (second ? whole : 0);
        bool wraps = false;
        if (r < rows) {
          const uint32_t x = (place + g.sy * (uint32_t)(r % ny) + g.sz * (uint32_t)(r / ny)) & (g.cells - 1u);
          const uint32_t end = x + len;
          wraps = end > g.cells;
          beg = starts[second ? 0u : x];
          cnt = starts[!second ? min(end, g.cells) : wraps ? end - g.cells : 0u] - beg;
        }
        if (__any_sync(0xffffffffu, wraps)) ranges = whole + rows;
      } else if (r0 + lane < ranges) {
        const bool second = r0 + lane >= rows;
        const int r = second ? r0 + lane - rows : r0 + lane;
        const uint32_t row = grid_row(g, lo.y - kReach + r % ny, lo.z - kReach + r / ny);
        beg = starts[row + (second ? 0 : x0)];
        cnt = starts[row + (second ? over : min(x0 + len, g.nx))] - beg;
      }
      uint32_t incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
      const uint32_t shift = beg - (incl - cnt);             // the photon of rank t, if in this lane's range: shift + t
      met += total;
      if (kParts == 1 && met > kDenseAt) {
        if (lane == 0) G.gb[atomicAdd(G.dense, 1u)].n.w = __uint_as_float(tile);
        return;
      }
      for (uint32_t t0 = 32u * part; t0 < total; t0 += 32u * kParts) {
        const uint32_t t = t0 + lane;
        int row = 0;                                         // the range that holds rank t: the first with incl > t
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          if (__shfl_sync(0xffffffffu, incl, row + o - 1) <= t) row += o;
        const uint32_t i = __shfl_sync(0xffffffffu, shift, row) + t;
        bool keep = false;
        float4 x;
        if (t < total) {
          x = __ldg(ph.xd + 2 * (size_t)i);
          keep = x.x >= bl.x && x.x <= bh.x && x.y >= bl.y && x.y <= bh.y && x.z >= bl.z && x.z <= bh.z;
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        bool finite = true;
        if (keep) {
          const uint32_t at = kept + __popc(m & ((1u << lane) - 1u));
          const float4 d = __ldg(ph.xd + 2 * (size_t)i + 1);
          ph_s[kX][at] = x.x;
          ph_s[kY][at] = x.y;
          ph_s[kZ][at] = x.z;
          ph_s[kDx][at] = d.x;
          ph_s[kDy][at] = d.y;
          ph_s[kDz][at] = d.z;
          ph_s[kEx][at] = x.w;
          ph_s[kEy][at] = d.w;
          const float ez = __ldg(ph.e + i);
          ph_s[kEz][at] = ez;
          finite = isfinite(x.w) && isfinite(d.w) && isfinite(ez);
        }
        odd |= !__all_sync(0xffffffffu, finite);
        kept += __popc(m);
        if (kept > 32u) test_kept();
      }
    }
    if (kept) test_kept();
  }
  // the parts of a pixel's sum meet in shared memory
  float3 acc = make_float3(sum[0].x + sum[0].y, sum[1].x + sum[1].y, sum[2].x + sum[2].y);
  if (kParts > 1) {
    s_acc[part][0][lane] = acc.x;
    s_acc[part][1][lane] = acc.y;
    s_acc[part][2][lane] = acc.z;
    __syncthreads();
    if (part > 0) return;
#pragma unroll
    for (int q = 1; q < kParts; ++q)
      acc = acc + make_float3(s_acc[q][0][lane], s_acc[q][1][lane], s_acc[q][2][lane]);
  }
  if (!inside) return;
  float* o = G.image + 3 * ((size_t)pj * c.W + pi);
  if (prim < 0) {                  // nothing seen: zero also where the normalisation overflows
    if (!G.add) o[0] = o[1] = o[2] = 0.0f;
    return;
  }
  const float norm = 2.0f / (3.14159265f * radius * radius) / 3.14159265f;   // kernel normalisation and 1/pi
  const float4 alb = __ldg(sv.prim_alb + prim);
  acc = make_float3(alb.x * acc.x * norm, alb.y * acc.y * norm, alb.z * acc.z * norm);
  if (G.add) acc = acc + make_float3(o[0], o[1], o[2]);
  o[0] = acc.x;
  o[1] = acc.y;
  o[2] = acc.z;
}

template <bool kOneRow>
__global__ void __launch_bounds__(32, 32) k_gather(SceneView sv, Gather G) {
  grid_dependency_wait();
  gather_tile<1, kOneRow>(sv, G, blockIdx.x, 0);
}

template <bool kOneRow>
__global__ void __launch_bounds__(32 * kDenseParts, 32 / kDenseParts) k_gather_dense(SceneView sv, Gather G) {
  grid_dependency_wait();
  __shared__ uint32_t s_next;
  const uint32_t n = G.dense[0];
  for (;;) {
    if (threadIdx.x == 0) s_next = atomicAdd(G.dense + 1, 1u);
    __syncthreads();
    const uint32_t k = s_next;
    if (k >= n) break;
    gather_tile<kDenseParts, kOneRow>(sv, G, __float_as_uint(G.gb[k].n.w), threadIdx.x >> 5);
    __syncthreads();               // s_next and the parts' sums have been read
  }
}

Cam make_cam(const pv_scene* s, const pv_camera* cam) {
  double pos[3], tg[3], up[3], f[3], r[3], u[3];
  for (int k = 0; k < 3; ++k) {
    pos[k] = cam->pos[k];
    tg[k] = cam->target[k];
    up[k] = cam->up[k];
    f[k] = tg[k] - pos[k];
  }
  auto nrm = [](double* v) {
    const double l = std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    for (int k = 0; k < 3; ++k) v[k] /= l;
  };
  nrm(f);
  r[0] = f[1] * up[2] - f[2] * up[1];
  r[1] = f[2] * up[0] - f[0] * up[2];
  r[2] = f[0] * up[1] - f[1] * up[0];
  nrm(r);
  u[0] = r[1] * f[2] - r[2] * f[1];
  u[1] = r[2] * f[0] - r[0] * f[2];
  u[2] = r[0] * f[1] - r[1] * f[0];
  const double ty = std::tan(0.5 * (double)cam->fov_y);
  Cam c;
  c.pos = make_float3((float)pos[0], (float)pos[1], (float)pos[2]);
  c.f = make_float3((float)f[0], (float)f[1], (float)f[2]);
  c.r = make_float3((float)r[0], (float)r[1], (float)r[2]);
  c.u = make_float3((float)u[0], (float)u[1], (float)u[2]);
  c.ty = (float)ty;
  c.tx = (float)(ty * (double)cam->width / (double)cam->height);
  c.W = cam->width;
  c.H = cam->height;
  c.znear = 1e-3f * s->diag;
  return c;
}

bool camera_ok(const pv_camera* c) {
  if (!c || c->width == 0 || c->height == 0 || c->width > 16384 || c->height > 16384) return false;
  if (!(c->fov_y > 0.0f && c->fov_y < 3.1f)) return false;
  const double f[3] = {(double)c->target[0] - c->pos[0], (double)c->target[1] - c->pos[1],
                       (double)c->target[2] - c->pos[2]};
  const double cr[3] = {f[1] * c->up[2] - f[2] * c->up[1], f[2] * c->up[0] - f[0] * c->up[2],
                        f[0] * c->up[1] - f[1] * c->up[0]};
  return f[0] * f[0] + f[1] * f[1] + f[2] * f[2] > 0.0 && cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2] > 0.0;
}

// Workspace layout: G-buffer, photons per cell (padded to whole scan
// tiles), tile sums, photon ranks, sorted photons: 40 bytes a photon place, and 4 to
// 8 for the cells.  A workspace of 32 bytes a place (least_bytes) does as well: half
// the cells, and the paths in two passes (1M-path city at 1920 x 1080 380 MB, 648 us, and 324 MB, 769 us).
struct SplatLayout {
  size_t gbuf, counts, sums, rank, xd, e, bytes;
  uint32_t cells;                                   // most cells a grid may have
  uint32_t paths;                                   // most paths a pass may have
  SplatLayout(uint32_t n, uint32_t B, uint32_t width, uint32_t height) {
    const uint64_t photons = (uint64_t)n * B;
    cells = full_cells(photons);
    paths = n;
    gbuf = 0;
    counts = up((size_t)width * height * sizeof(GPixel));
    sums = up(counts + (size_t)tiles(cells) * 4096 * sizeof(uint32_t));
    rank = up(sums + (size_t)(tiles(cells) + 3) * sizeof(uint32_t));
    xd = up(rank + (size_t)photons * sizeof(uint32_t));
    e = up(xd + 2 * (size_t)photons * sizeof(float4));
    bytes = up(e + (size_t)photons * sizeof(float));
  }
  // Squeeze into ``room`` (at least least_bytes, fewer than ``bytes``).
  void squeeze(uint32_t n, uint32_t B, size_t room) {
    cells /= 2;
    sums = counts + (size_t)tiles(cells) * 4096 * sizeof(uint32_t);
    xd = (sums + (size_t)(tiles(cells) + 3) * sizeof(uint32_t) + 15) & ~(size_t)15;
    paths = (uint32_t)std::min<size_t>((room - xd) / (2 * sizeof(float4) + sizeof(float) + sizeof(uint32_t)) / B, n);
    e = xd + 2 * (size_t)paths * B * sizeof(float4);
    rank = e + (size_t)paths * B * sizeof(float);
    bytes = rank + (size_t)paths * B * sizeof(uint32_t);
  }
  static size_t least_bytes(uint32_t n, uint32_t B, uint32_t width, uint32_t height) {
    const uint64_t photons = (uint64_t)n * B;
    const size_t c = full_cells(photons);
    return up(up(up((size_t)width * height * sizeof(GPixel)) + c * sizeof(uint32_t)) + (c / 4096 + 1) * sizeof(uint32_t)) +
           up((size_t)photons * 2 * sizeof(float4));
  }
  static uint32_t full_cells(uint64_t photons) {     // a power of two >= the photons, at least one scan tile
    uint32_t c = 4096;
    while (c < photons && c < kMaxCells) c <<= 1;
    return c;
  }
  // scan tiles over the counters of a grid of c cells and the total behind them
  static uint32_t tiles(uint32_t c) { return (uint32_t)(((uint64_t)c + 1 + 4095) / 4096); }
  static size_t up(size_t x) { return (x + 255) & ~(size_t)255; }
};

// Cells of edge radius / kCellsPerRadius over the scene's extent, each axis
// with at least 2 kReach + 2 cells; one row of ``most`` places (a power of two)
// where that is more than ``most`` cells, of half as many where it is not twice as
// many (clearing and summing up the counters then takes half as long: district of
// 300k paths, 700 x 500, r = 0.12 139 -> 124 us).
Grid make_grid(const pv_scene* s, float radius, uint32_t most) {
  Grid g;
  g.inv_edge = (float)kCellsPerRadius / radius;
  int n[3];
  for (int k = 0; k < 3; ++k) {
    const double c = ((double)s->box_hi[k] - s->box_lo[k]) * g.inv_edge + 2.0;
    n[k] = c < 1048576.0 ? std::max((int)c, 2 * kReach + 2) : 1048576;      // NaN: the most
  }
  const uint64_t all = (uint64_t)n[0] * n[1] * n[2];
  const bool fits = all <= most;
  const uint32_t row = all <= 2 * (uint64_t)most && most > kMinCells ? most / 2 : most;
  g.nx = fits ? n[0] : (int)row;
  g.ny = fits ? n[1] : 1 << 30;
  g.nz = fits ? n[2] : 1 << 30;
  g.cells = fits ? (uint32_t)all : row;
  g.sy = fits ? 0u : stride_y(row);
  g.sz = fits ? 0u : stride_z(row);
  return g;
}

}  // namespace

extern "C" size_t pv_splat_workspace_bytes(const pv_scene* s, uint32_t width, uint32_t height) {
  if (!s) return 0;
  return SplatLayout(s->n_paths_total, s->B, width, height).bytes;
}

extern "C" int pv_splat(pv_scene* s, const pv_paths* paths, const pv_camera* cam, float radius, float* d_image,
                        void* d_work, size_t work_bytes, void* stream) {
  const int rc = pvh::check_paths(s, paths);
  if (rc != PV_OK) return rc;
  if (!camera_ok(cam) || !d_image || !d_work || !(radius > 0.0f)) return PV_ERR_ARG;
  if (paths->n > (1u << 27)) return PV_ERR_LIMIT;            // photon ranks are 32-bit
  const uint32_t n = paths->n;
  SplatLayout lay(n, s->B, cam->width, cam->height);
  if (reinterpret_cast<uintptr_t>(d_work) & 255u) return PV_ERR_ARG;
  if (work_bytes < lay.bytes) {
    if (work_bytes < SplatLayout::least_bytes(n, s->B, cam->width, cam->height)) return PV_ERR_ARG;
    lay.squeeze(n, s->B, work_bytes);
  }
  cudaStream_t st = (cudaStream_t)stream;
  s->last_stream = st;
  const Cam c = make_cam(s, cam);
  const Grid g = make_grid(s, radius, lay.cells);
  char* w = static_cast<char*>(d_work);
  GPixel* gbuf = reinterpret_cast<GPixel*>(w + lay.gbuf);
  uint32_t* counts = reinterpret_cast<uint32_t*>(w + lay.counts);
  uint32_t* sums = reinterpret_cast<uint32_t*>(w + lay.sums);
  uint32_t* rank = reinterpret_cast<uint32_t*>(w + lay.rank);
  const Photons ph = {reinterpret_cast<float4*>(w + lay.xd), reinterpret_cast<float*>(w + lay.e)};
  const pvk::SceneView sv = pvh::view(s);
  // after the memset, the kernels are dependent launches: short kernels had a launch's latency between them
  const uint32_t tiles = SplatLayout::tiles(g.cells);
  const float4* pa = reinterpret_cast<const float4*>(paths->pa);
  const float4* pb = reinterpret_cast<const float4*>(paths->pb);
  const uint32_t gather_tiles = ((c.W + 7) / 8) * ((c.H + 3) / 4);
  const uint32_t dense_blocks = std::min<uint32_t>(gather_tiles, 32u / kDenseParts * (uint32_t)s->num_sms);
  PathRange R = {0, std::min(n, lay.paths)};
  do {
    const uint32_t photon_blocks = (R.count + 255) / 256;
    const uint32_t views = R.first == 0 ? ((c.W + 15) / 16) * ((c.H + 15) / 16) : 0u;
    const Mix m = mix_blocks(photon_blocks, views);
    PV_CHECK(cudaMemsetAsync(counts, 0, (size_t)tiles * 4096 * sizeof(uint32_t), st));
    pvh::launch_dependent(k_view_count, m.total, 256, 0, st, m, sv, c, g, radius, R, n, s->B, paths->info, pa, counts,
                          rank, gbuf);
    pvh::launch_dependent(k_tile_sums, tiles, 1024, 0, st, counts, sums);
    pvh::exclusive_scan(sums, tiles, st);
    pvh::launch_dependent(k_tile_scan, tiles, 1024, 0, st, counts, sums);
    if (R.count)
      pvh::launch_dependent(k_photon_place, photon_blocks, 256, 0, st, g, R, n, s->B, paths->info, paths->origin, pa, pb,
                            counts, rank, ph);
    const Gather G = {c, g, radius, gbuf, counts, ph, sums + tiles + 1, d_image, R.first > 0};
    pvh::launch_dependent(g.sy ? k_gather<true> : k_gather<false>, gather_tiles, 32, 0, st, sv, G);
    pvh::launch_dependent(g.sy ? k_gather_dense<true> : k_gather_dense<false>, dense_blocks, 32 * kDenseParts, 0, st, sv,
                          G);
    R.first += R.count;
    R.count = std::min(n - R.first, lay.paths);
  } while (R.first < n);
  return pvh::cuda_status(cudaGetLastError());
}
