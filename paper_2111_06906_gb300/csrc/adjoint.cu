// Differentiable deposit model, its adjoint, and budgeted re-trace lists.
//
// The paper has no gradients.  This model ranks the paths to re-trace when a
// ray budget cannot cover every path the Eq. 2 test invalidated.  Each stored
// path keeps its triangles and sampled directions; under parameters theta
//   - the emission follows the light: a point light at p re-aims from p
//     along the stored first segment; a rectangle keeps the stored point
//     (alpha, beta) and direction (ell) in its frame, with the tangent t
//     fixed and the normal n free: o = p + alpha t + beta (n x t) and
//     d0 = ell.x t + ell.y (n x t) + ell.z n;
//   - photon k is re-found on its triangle's plane (unit normal nu_k through
//     the stored photon, translated with its dynamic object) along the stored
//     incoming direction: x_k = x_{k-1} + d nu.(q_k - x_{k-1}) / (nu.d);
//   - energies scale with the light's intensity factor;
//   - photons splat with the uniform cubic B-spline over 4 x 4 texels
//     (C2, texel centres at half-integers, texels outside dropped).
// theta = per light [pos 3, normal 3, scale 1], then per dynamic object in
// slot order [translation 3].  At the current pose the model reproduces the
// stored photons.  The adjoint runs the chain backwards per path:
//   dx_k/dx_{k-1} = I - d nu^T/(nu.d),  dx_k/dq_k = d nu^T/(nu.d),
//   dx_1/do = I - d0 nu^T/(nu.d0),      dx_1/dd0 = tau_1 (I - d0 nu^T/(nu.d0)).
#include <algorithm>
#include <cstring>

#include "pv_scene.h"

using namespace pvk;

namespace {

constexpr int kMaxTheta = 7 * PV_MAX_LIGHTS + 3 * kMaxDyn;

struct ModelArgs {
  uint32_t n, n_lights, n_theta;
  const uint32_t* info;
  const float* origin;
  const float4* pa;
  const float4* pb;
  const float* theta;           // device [n_theta]
  uint32_t W, H;
  float x0, z0, x1, z1;
  float cur_t[kMaxDyn][3];      // current translation of each dynamic slot
};

struct Emission {
  float3 o, d0, t, ell;
  float beta;
  bool rect;
};

__device__ __forceinline__ float3 load3(const float* p) { return make_float3(p[0], p[1], p[2]); }

// Emission of the model path under the light's parameters tl (shared memory).
__device__ __forceinline__ Emission model_emission(const LightPose& Lp, const float* tl, const ModelArgs& A,
                                                   uint32_t p, float3 x10) {
  Emission e;
  const float3 o0 = make_float3(A.origin[p], A.origin[A.n + p], A.origin[2 * (size_t)A.n + p]);
  const float3 d00 = x10 - o0;
  e.t = Lp.t;
  e.rect = Lp.type != PV_LIGHT_POINT;
  if (!e.rect) {
    e.o = load3(tl);
    e.d0 = d00;
    e.beta = 0.f;
    e.ell = make_float3(0.f, 0.f, 0.f);
  } else {
    const float3 rel = o0 - Lp.pos;
    const float alpha = dot(Lp.t, rel);
    e.beta = dot(Lp.b, rel);
    e.ell = make_float3(dot(Lp.t, d00), dot(Lp.b, d00), dot(Lp.n, d00));
    const float3 nl = load3(tl + 3);
    const float3 bl = cross(nl, Lp.t);
    e.o = load3(tl) + alpha * Lp.t + e.beta * bl;
    e.d0 = e.ell.x * Lp.t + e.ell.y * bl + e.ell.z * nl;
  }
  return e;
}

// Unit normal of stored photon v's triangle and its dynamic slot (-1: static).
__device__ __forceinline__ float3 photon_normal(const SceneView& sv, float4 v, int& slot) {
  const int prim = __float_as_int(v.w);
  const uint32_t sl = slot_of(sv, prim);
  slot = sl == 255u ? -1 : (int)sl;
  return normalize(prim_normal(sv, prim, false));
}

// Plane point of stored photon v, moved with its object's translation.
__device__ __forceinline__ float3 photon_point(const ModelArgs& A, const float* s_th, float4 v, int slot) {
  float3 q = f3(v);
  if (slot >= 0) {
    const float* tt = s_th + 7 * A.n_lights + 3 * slot;
    q = q + make_float3(tt[0] - A.cur_t[slot][0], tt[1] - A.cur_t[slot][1], tt[2] - A.cur_t[slot][2]);
  }
  return q;
}

// Uniform cubic B-spline footprint of (x, z): with u = (x - x0) W/(x1 - x0) - 1/2
// (texel-centre coordinate), i0 = floor(u) and f = u - i0, texels i0-1 .. i0+2
// get the cardinal weights (1-f)^3/6, (3f^3 - 6f^2 + 4)/6,
// (-3f^3 + 3f^2 + 3f + 1)/6, f^3/6 (derivatives -(1-f)^2/2, (3f^2 - 4f)/2,
// (-3f^2 + 2f + 1)/2, f^2/2); the 2-D weight is the product over x and z.
struct Spline {
  int i0, j0;                 // texel of tap 0 in x and z
  float wx[4], dx[4], wz[4], dz[4];
  float sx, sz;
};

__device__ __forceinline__ void bspline1(float f, float* w, float* d) {
  const float g = 1.f - f, f2 = f * f, f3 = f2 * f;
  w[0] = g * g * g * (1.f / 6.f);
  w[1] = (3.f * f3 - 6.f * f2 + 4.f) * (1.f / 6.f);
  w[2] = (-3.f * f3 + 3.f * f2 + 3.f * f + 1.f) * (1.f / 6.f);
  w[3] = f3 * (1.f / 6.f);
  d[0] = -0.5f * g * g;
  d[1] = 0.5f * (3.f * f2 - 4.f * f);
  d[2] = 0.5f * (-3.f * f2 + 2.f * f + 1.f);
  d[3] = 0.5f * f2;
}

__device__ __forceinline__ Spline spline(const ModelArgs& A, float x, float z) {
  Spline b;
  b.sx = (float)A.W / (A.x1 - A.x0);
  b.sz = (float)A.H / (A.z1 - A.z0);
  const float u = (x - A.x0) * b.sx - 0.5f, v = (z - A.z0) * b.sz - 0.5f;
  const float fi = floorf(u), fj = floorf(v);
  bspline1(u - fi, b.wx, b.dx);
  bspline1(v - fj, b.wz, b.dz);
  // far outside: keep the indices representable (every tap is dropped)
  b.i0 = (int)fmaxf(fminf(fi, 1e9f), -1e9f) - 1;
  b.j0 = (int)fmaxf(fminf(fj, 1e9f), -1e9f) - 1;
  return b;
}

// Four floats added at p (16-byte aligned), nothing returned.
__device__ __forceinline__ void add4(float4* p, const float (&v)[4]) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3])
               : "memory");
}

__device__ __forceinline__ void stage_theta(const ModelArgs& A, float* s_th) {
  for (uint32_t j = threadIdx.x; j < A.n_theta; j += blockDim.x) s_th[j] = A.theta[j];
}

// Shared memory of one warp of 32 consecutive paths: per photon (row k, lane of
// its path, arrays [B][32]) two or three words, and the list of the warp's photons.
//
// The chain of a path is serial, but what costs is the 4 x 4 texels of each of
// its photons.  With a thread per path the rounds over photons run until the
// warp's longest path ends (two of up to seven photons on average), 8 to 11 of
// 32 lanes active.  So each lane first walks its path's chain and leaves its
// photons' x and z here, and then the warp's photons are dealt out to the lanes
// through the list.  (Dealing out their normals as well took 14-24 % longer: six
// more words a photon leave room for fewer warps.)
struct PhotonSmem {
  float* a;                    // x, then the adjoint's dL/dx
  float* b;                    // z, then the adjoint's dL/dz
  float* c;                    // the adjoint's dL/d(intensity)
  uint16_t* list;              // [32 B] lane | row << 5
};

// A row of four RGB taps is 12 consecutive floats at any multiple of 4 bytes.  It
// is read and added through the 16-byte chunks that hold it: four of them from
// the last 16-byte boundary at or before the row, which starts o = 0..3 floats
// behind (the fourth holds none of it when o = 0); widths chosen by alignment
// made the lanes take turns.  k_model_deposit gives the chunks to four lanes next
// to each other, so that a row is one request to L2; a lane per photon made four.
// Each lane leaves its photon's taps here, then each four lanes take a photon's rows.
struct TapSmem {
  float p[32][19];             // energy x wx of the 12 floats from [3] on, zeros around them (odd stride: no conflicts)
  float wz[32][5];
  size_t first[32];            // float index of row 0 (wraps below zero for a row outside)
  uint32_t rows[32];           // bit r: row r goes by chunks
};
static_assert(sizeof(TapSmem) % 8 == 0 && 4 * (sizeof(TapSmem) + 32 * PV_MAX_BOUNCES * 10) <= 46 * 1024, "shared memory of a block");

// Bytes a warp needs: ``taps`` of them for its taps, then kWords words a photon and the list.
template <uint32_t kWords>
__host__ __device__ __forceinline__ uint32_t warp_smem_bytes(uint32_t B, uint32_t taps) {
  return taps + ((32u * B * (4u * kWords + 2u) + 7u) & ~7u);
}

template <uint32_t kWords>
__device__ __forceinline__ PhotonSmem photon_smem(unsigned char* warp, uint32_t B) {
  float* f = reinterpret_cast<float*>(warp);
  return {f, f + 32 * B, f + 64 * B, reinterpret_cast<uint16_t*>(f + 32 * B * kWords)};
}

// What a path's chain leaves with its lane.
struct Chain {
  uint32_t nseg, light;
  float sc, tau1;
  Emission e;
};

// Walk the chain of path p (>= A.n: no path): photon k's model position into
// row k of the warp's shared memory, and the warp's photons into its list;
// returns their number.  All lanes call.
__device__ __forceinline__ uint32_t walk_chain(const SceneView& sv, const FrameLights& L, const ModelArgs& A,
                                               const float* s_th, uint32_t p, const PhotonSmem& S, Chain& c) {
  const int lane = threadIdx.x & 31;
  c.nseg = 0;
  c.light = 0;
  c.sc = c.tau1 = 0.f;
  if (p < A.n) {
    const uint32_t w = A.info[p];
    c.nseg = min(info_nseg(w), sv.B);
    c.light = info_light(w);
  }
  uint32_t at = c.nseg;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, at, o);
    if (lane >= o) at += y;
  }
  const uint32_t total = __shfl_sync(0xffffffffu, at, 31);
  at -= c.nseg;
  if (c.nseg > 0) {
    float4 v = A.pa[p];
    c.e = model_emission(L.cur[c.light], s_th + 7 * c.light, A, p, f3(v));
    c.sc = s_th[7 * c.light + 6];
    float3 prev = c.e.o, dir = c.e.d0;
    for (uint32_t k = 0; k < c.nseg; ++k) {
      const float4 vn = k + 1 < c.nseg ? A.pa[(size_t)(k + 1) * A.n + p] : v;
      int slot;
      const float3 nu = photon_normal(sv, v, slot);
      const float3 q = photon_point(A, s_th, v, slot);
      const float tau = dot(nu, q - prev) / dot(nu, dir);
      if (k == 0) c.tau1 = tau;
      const float3 x = prev + tau * dir;
      S.a[32 * k + lane] = x.x;
      S.b[32 * k + lane] = x.z;
      S.list[at + k] = (uint16_t)(lane | (k << 5));
      dir = f3(vn) - f3(v);                       // stored direction of the next segment
      v = vn;
      prev = x;
    }
  }
  __syncwarp();
  return total;
}

// This lane's photon into the warp's taps; returns the rows that go by chunks
// (inside the atlas in x, their 16 floats inside the array, which is 16-byte
// aligned if ``vec_ok``).
__device__ __forceinline__ uint32_t tap_store(TapSmem& T, int lane, const ModelArgs& A, const Spline& b, float3 E,
                                              bool vec_ok) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    T.p[lane][3 + 3 * q] = E.x * b.wx[q];
    T.p[lane][4 + 3 * q] = E.y * b.wx[q];
    T.p[lane][5 + 3 * q] = E.z * b.wx[q];
    T.wz[lane][q] = b.wz[q];
  }
  const size_t floats = 3 * (size_t)A.W * A.H;
  const size_t first = 3 * ((size_t)(int64_t)b.j0 * A.W + (size_t)(int64_t)b.i0);
  T.first[lane] = first;
  uint32_t rows = 0;
  if (vec_ok && b.i0 >= 0 && b.i0 + 3 < (int)A.W)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int tj = b.j0 + r;
      if (tj >= 0 && tj < (int)A.H && first + 3 * (size_t)A.W * r + 16 <= floats) rows |= 1u << r;
    }
  return T.rows[lane] = rows;
}

// Forward splat.  Bound by the atomics' requests in L2.  City, 2.0M photons into
// 1024 x 1024 texels: 249 us with a thread per path and access widths by
// alignment, 217 us with the photons dealt out a lane each, 141 us with four lanes
// a photon (16 lanes: 142 us, a quarter more instructions).
__global__ void __launch_bounds__(128) k_model_deposit(SceneView sv, FrameLights L, ModelArgs A, float* atlas) {
  grid_dependency_wait();
  __shared__ float s_th[kMaxTheta];
  extern __shared__ __align__(16) unsigned char s_photons[];
  stage_theta(A, s_th);
  __syncthreads();
  const bool vec_ok = (reinterpret_cast<uintptr_t>(atlas) & 15u) == 0;
  unsigned char* const mine = s_photons + (threadIdx.x >> 5) * warp_smem_bytes<2>(sv.B, sizeof(TapSmem));
  TapSmem& T = *reinterpret_cast<TapSmem*>(mine);
  const PhotonSmem S = photon_smem<2>(mine + sizeof(TapSmem), sv.B);
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 19; ++i)
    if (i < 3 || i > 14) T.p[lane][i] = 0.f;
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x, p0 = p - lane;
  Chain c;
  const uint32_t total = walk_chain(sv, L, A, s_th, p, S, c);
  const size_t stride = 3 * (size_t)A.W;
  for (uint32_t t0 = 0; t0 < total; t0 += 32) {
    const bool has = t0 + lane < total;
    const uint32_t id = S.list[has ? t0 + lane : t0], own = id & 31u, k = id >> 5;
    const float sc = __shfl_sync(0xffffffffu, c.sc, own);
    if (has) {
      const float3 E = sc * f3(A.pb[(size_t)k * A.n + p0 + own]);
      const Spline b = spline(A, S.a[32 * k + own], S.b[32 * k + own]);
      const uint32_t rows = tap_store(T, lane, A, b, E, vec_ok);
      if (rows != 15u)                            // at the atlas' edges, or an unaligned atlas: texel by texel
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int tj = b.j0 + r;
          if (((rows >> r) & 1u) || tj < 0 || tj >= (int)A.H) continue;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int ti = b.i0 + q;
            if (ti < 0 || ti >= (int)A.W) continue;
            float* t = atlas + 3 * ((size_t)tj * A.W + ti);
            const float wc = b.wx[q] * b.wz[r];
            atomicAdd(t + 0, E.x * wc);
            atomicAdd(t + 1, E.y * wc);
            atomicAdd(t + 2, E.z * wc);
          }
        }
    }
    __syncwarp();
    const uint32_t n = min(32u, total - t0);
    const int q = lane & 3;
    for (uint32_t j = lane >> 2; j < n; j += 8) {
      const uint32_t rows = T.rows[j];
      size_t first = T.first[j];
      uint32_t o = (uint32_t)first & 3u;
      const float* w = &T.p[j][3 + 4 * q - (int)o];
      float v[4] = {w[0], w[1], w[2], w[3]};
#pragma unroll
      for (int r = 0; r < 4; ++r, first += stride) {
        if (r > 0 && (A.W & 3u)) {                // rows of another alignment
          o = (uint32_t)first & 3u;
          w = &T.p[j][3 + 4 * q - (int)o];
#pragma unroll
          for (int i = 0; i < 4; ++i) v[i] = w[i];
        }
        if (!((rows >> r) & 1u) || (q == 3 && o == 0u)) continue;
        const float wz = T.wz[j][r];
        const float u[4] = {v[0] * wz, v[1] * wz, v[2] * wz, v[3] * wz};
        add4(reinterpret_cast<float4*>(atlas + (first - o)) + q, u);
      }
    }
    __syncwarp();
  }
}

// w[o .. o + 11] into v, o = 0..3.
__device__ __forceinline__ void shift_down(const float (&w)[16], uint32_t o, float (&v)[12]) {
  const bool s1 = o & 1u, s2 = o & 2u;
  float t[13];
#pragma unroll
  for (int i = 0; i < 13; ++i) t[i] = s2 ? w[i + 2] : w[i];
#pragma unroll
  for (int i = 0; i < 12; ++i) v[i] = s1 ? t[i + 1] : t[i];
}

// Reverse mode: the chain forward, the splat gradient of every photon (only x
// and z are nonzero) and its share of the intensity's, dealt out over the warp,
// then the chain backward, which reloads the planes and directions.  dtheta is
// reduced per block in shared memory, then added to the global vector.
// Bound by L1's wavefronts (65 %) and the chains' loads.  City, 2.0M photons:
// 258 us with a thread per path and 48 scalar reads of the gradient a photon,
// 166 us with the photons dealt out a lane each and four wide reads a row.  (Four
// lanes a photon, one request a row, 228 us and 16 lanes 316 us: what they save in
// L1 they spend on summing up and on shared memory.)
__global__ void __launch_bounds__(128) k_adjoint(SceneView sv, FrameLights L, ModelArgs A, const float* G,
                                                 float* dtheta, float* score) {
  grid_dependency_wait();
  __shared__ float s_th[kMaxTheta];
  __shared__ float s_acc[kMaxTheta];
  extern __shared__ __align__(16) unsigned char s_photons[];
  stage_theta(A, s_th);
  for (uint32_t j = threadIdx.x; j < A.n_theta; j += blockDim.x) s_acc[j] = 0.f;
  __syncthreads();
  const bool vec_ok = (reinterpret_cast<uintptr_t>(G) & 15u) == 0;
  const size_t floats = 3 * (size_t)A.W * A.H;
  const PhotonSmem S = photon_smem<3>(s_photons + (threadIdx.x >> 5) * warp_smem_bytes<3>(sv.B, 0), sv.B);
  const int lane = threadIdx.x & 31;
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x, p0 = p - lane;
  float lc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // this path's light gradient
  Chain c;
  const uint32_t total = walk_chain(sv, L, A, s_th, p, S, c);
  for (uint32_t t0 = 0; t0 < total; t0 += 32) {
    const bool has = t0 + lane < total;
    const uint32_t id = S.list[has ? t0 + lane : t0], own = id & 31u, k = id >> 5;
    const float sc = __shfl_sync(0xffffffffu, c.sc, own);
    if (!has) continue;
    const float3 E0 = f3(A.pb[(size_t)k * A.n + p0 + own]);
    const Spline b = spline(A, S.a[32 * k + own], S.b[32 * k + own]);
    const bool inside = vec_ok && b.i0 >= 0 && b.i0 + 3 < (int)A.W;
    float2 g = make_float2(0.f, 0.f);
    float gscale = 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int tj = b.j0 + r;
      if (tj < 0 || tj >= (int)A.H) continue;
      float gr = 0.f, gdx = 0.f;                  // row sums of ge weighted by wx, dx
      auto tap = [&](int q, float r0, float r1, float r2) {
        const float ge = r0 * E0.x + r1 * E0.y + r2 * E0.z;
        gr = fmaf(ge, b.wx[q], gr);
        gdx = fmaf(ge, b.dx[q], gdx);
      };
      const size_t first = 3 * ((size_t)tj * A.W + (size_t)(int64_t)b.i0);
      if (inside && first + 16 <= floats) {
        const uint32_t o = (uint32_t)first & 3u;
        const float4* at = reinterpret_cast<const float4*>(G + (first - o));
        float w[16], v[12];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 x = q < 3 || o ? __ldg(at + q) : make_float4(0.f, 0.f, 0.f, 0.f);
          w[4 * q] = x.x;
          w[4 * q + 1] = x.y;
          w[4 * q + 2] = x.z;
          w[4 * q + 3] = x.w;
        }
        shift_down(w, o, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) tap(q, v[3 * q], v[3 * q + 1], v[3 * q + 2]);
      } else {
        // texels outside are left out, not taken as zero: the energy or the weight may be infinite
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int ti = b.i0 + q;
          if (ti < 0 || ti >= (int)A.W) continue;
          const float* t = G + 3 * ((size_t)tj * A.W + ti);
          tap(q, __ldg(t), __ldg(t + 1), __ldg(t + 2));
        }
      }
      g.x = fmaf(gdx, b.wz[r], g.x);
      g.y += gr * b.dz[r];
      gscale = fmaf(gr, b.wz[r], gscale);
    }
    S.a[32 * k + own] = g.x * (sc * b.sx);
    S.b[32 * k + own] = g.y * (sc * b.sz);
    S.c[32 * k + own] = gscale;
  }
  __syncwarp();
  if (c.nseg > 0) {
    const Emission& e = c.e;
    float gscale = 0.f;
    float3 g = make_float3(0.f, 0.f, 0.f);
    float4 vk = A.pa[(size_t)(c.nseg - 1) * A.n + p];
    for (uint32_t k = c.nseg; k >= 1; --k) {
      g.x += S.a[32 * (k - 1) + lane];
      g.z += S.b[32 * (k - 1) + lane];
      gscale += S.c[32 * (k - 1) + lane];
      const float4 vp = k == 1 ? vk : A.pa[(size_t)(k - 2) * A.n + p];
      int slot;
      const float3 nu = photon_normal(sv, vk, slot);
      const float3 d = k == 1 ? e.d0 : f3(vk) - f3(vp);
      const float r = dot(d, g) / dot(nu, d);
      if (slot >= 0) {
        float* a = s_acc + 7 * A.n_lights + 3 * slot;
        atomicAdd(a + 0, nu.x * r);
        atomicAdd(a + 1, nu.y * r);
        atomicAdd(a + 2, nu.z * r);
      }
      g = g - r * nu;
      vk = vp;
    }
    // light: g is now the gradient with respect to o; d0 receives tau_1 g
    lc[0] = g.x;
    lc[1] = g.y;
    lc[2] = g.z;
    lc[6] = gscale;
    if (e.rect) {
      const float3 gd = c.tau1 * g;
      const float3 gn = e.beta * cross(e.t, g) + e.ell.y * cross(e.t, gd) + e.ell.z * gd;
      lc[3] = gn.x;
      lc[4] = gn.y;
      lc[5] = gn.z;
    }
  }
  if (score && p < A.n) score[p] = fabsf(c.sc * lc[6]);
  // light entries: summed over the warp per light, one shared atomic per entry
  for (uint32_t ll = 0; ll < A.n_lights; ++ll) {
    const bool mine = c.nseg > 0 && c.light == ll;
    if (!__any_sync(0xffffffffu, mine)) continue;
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      float v = mine ? lc[q] : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0 && v != 0.f) atomicAdd(&s_acc[7 * ll + q], v);
    }
  }
  __syncthreads();
  for (uint32_t j = threadIdx.x; j < A.n_theta; j += blockDim.x)
    if (s_acc[j] != 0.f) atomicAdd(dtheta + j, s_acc[j]);
}

// ---- ray budget: the ``budget`` listed paths of largest score by radix select
// A listed path's key is its score's bits if the score is positive, else 0 (NaN,
// zero and negatives rank last); equal keys rank by their place in the list.  Three
// histograms of 11, 11 and 9 key bits, each over the keys that share the bits
// picked so far, give the key T of the last path kept and how many paths of key
// T are kept; then the paths above T, and the first of those at T, are marked.
// Sorting all n slots on 32 bits instead took 12 launches, four of them a scan by
// one block: 151 us for 400k paths, where these five take 22 us.
constexpr uint32_t kBudgetThreads = 256, kBudgetBins = 2048, kBudgetItems = 8;
constexpr uint32_t kBudgetStep = kBudgetThreads * kBudgetItems;
constexpr uint32_t kNoKey = 0xFFFFFFFFu;     // an id out of range

// What a level has picked: the key bits so far and how many paths of those bits are still to be kept.
struct BudgetState {
  uint32_t prefix, want;
};

// Workspace (32-bit words): three histograms, three states, ties per tile.
struct BudgetWork {
  uint32_t hist[3][kBudgetBins];
  BudgetState state[3];
  uint32_t ties[pvh::kBudgetTiles];
};
static_assert(sizeof(BudgetWork) <= pvh::kBudgetWords * sizeof(uint32_t), "workspace of the ray budget");

// The highest bin b whose count, with the counts of all bins above it, reaches
// ``want`` (> 0, at most the total); want becomes what bin b has to give.  All
// threads of the block call; ``sh``: 10 words.
__device__ __forceinline__ uint32_t budget_pick(const uint32_t* hist, uint32_t& want, uint32_t* sh) {
  constexpr uint32_t kPer = kBudgetBins / kBudgetThreads;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t top = kBudgetBins - 1u - kPer * threadIdx.x;
  uint32_t v[kPer], own = 0;
#pragma unroll
  for (uint32_t k = 0; k < kPer; ++k) own += v[k] = hist[top - k];
  uint32_t incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if ((int)lane >= o) incl += y;
  }
  if (lane == 31u) sh[warp] = incl;
  __syncthreads();
  uint32_t above = incl - own;
  for (uint32_t w = 0; w < warp; ++w) above += sh[w];
#pragma unroll
  for (uint32_t k = 0; k < kPer; ++k) {
    if (above < want && want <= above + v[k]) {
      sh[8] = top - k;
      sh[9] = want - above;
    }
    above += v[k];
  }
  __syncthreads();
  const uint32_t bin = sh[8];
  want = sh[9];
  return bin;
}

// Level kLevel (0, 1, 2): pick the bin of the level before and count this
// level's bins over the keys that match.  Level 0 also makes the keys and
// clears the marks.
template <int kLevel>
__global__ void __launch_bounds__(kBudgetThreads) k_budget_hist(const uint32_t* list, const uint32_t* count,
                                                                const float* score, uint32_t n, uint32_t budget,
                                                                uint32_t* keys, uint32_t* marks, BudgetWork* W) {
  grid_dependency_wait();
  __shared__ uint32_t s_hist[kBudgetBins];
  __shared__ uint32_t sh[10];
  constexpr uint32_t kShift = kLevel == 0 ? 20u : kLevel == 1 ? 9u : 0u;      // lowest bit of this level
  constexpr uint32_t kMask = kLevel == 2 ? 511u : 2047u;
  constexpr uint32_t kAbove = kLevel == 1 ? 20u : 9u;                         // lowest bit of the levels before
  for (uint32_t i = threadIdx.x; i < kBudgetBins; i += kBudgetThreads) s_hist[i] = 0u;
  BudgetState st = {0u, 0u};
  if (kLevel > 0) {
    if (kLevel == 1) {
      uint32_t total = 0;                      // paths in range
      for (uint32_t i = threadIdx.x & 31u; i < kBudgetBins; i += 32u) total += W->hist[0][i];
      st.want = min(budget, __reduce_add_sync(0xffffffffu, total));
    } else {
      st = W->state[kLevel - 2];
    }
    if (st.want) st.prefix = st.prefix * kBudgetBins + budget_pick(W->hist[kLevel - 1], st.want, sh);
    if (blockIdx.x == 0 && threadIdx.x == 0) W->state[kLevel - 1] = st;
    if (!st.want) return;
  }
  __syncthreads();
  const uint32_t m = min(*count, n);
  const uint32_t end = kLevel == 0 ? n : m;
  for (uint32_t i = blockIdx.x * kBudgetThreads + threadIdx.x; i < end; i += gridDim.x * kBudgetThreads) {
    uint32_t key = kNoKey;
    if (kLevel == 0) {
      marks[i] = 0u;
      if (i >= m) continue;
      const uint32_t id = list[i];
      if (id < n) {
        const float s = score[id];
        key = s > 0.f ? __float_as_uint(s) : 0u;
      }
      keys[i] = key;
      if (key != kNoKey) atomicAdd(s_hist + (key >> kShift), 1u);
    } else {
      key = keys[i];
      if (key != kNoKey && key >> kAbove == st.prefix) atomicAdd(s_hist + ((key >> kShift) & kMask), 1u);
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < kBudgetBins; i += kBudgetThreads)
    if (s_hist[i]) atomicAdd(&W->hist[kLevel][i], s_hist[i]);
}

// The last key T, and the paths of key T in every tile of the list (a block per tile).
__global__ void __launch_bounds__(kBudgetThreads) k_budget_ties(const uint32_t* count, uint32_t n, uint32_t tile,
                                                                const uint32_t* keys, BudgetWork* W) {
  grid_dependency_wait();
  __shared__ uint32_t sh[10];
  BudgetState st = W->state[1];
  if (st.want) st.prefix = st.prefix * 512u + budget_pick(W->hist[2], st.want, sh);
  if (blockIdx.x == 0 && threadIdx.x == 0) W->state[2] = st;
  if (!st.want) return;
  const uint64_t b = (uint64_t)blockIdx.x * tile;
  const uint32_t m = min(*count, n), e = (uint32_t)min(b + tile, (uint64_t)m);
  uint32_t ties = 0;
  for (uint64_t i = b + threadIdx.x; i < e; i += kBudgetThreads) ties += keys[i] == st.prefix ? 1u : 0u;
  ties = __reduce_add_sync(0xffffffffu, ties);
  __syncthreads();
  if ((threadIdx.x & 31u) == 0u) sh[threadIdx.x >> 5] = ties;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (uint32_t w = 0; w < kBudgetThreads / 32u; ++w) t += sh[w];
    W->ties[blockIdx.x] = t;
  }
}

// Mark (bit 30, as in the info word) the paths above T and the first state.want of those at T.
__global__ void __launch_bounds__(kBudgetThreads) k_budget_mark(const uint32_t* list, const uint32_t* count, uint32_t n,
                                                                uint32_t tile, const uint32_t* keys,
                                                                const BudgetWork* W, uint32_t* marks) {
  grid_dependency_wait();
  __shared__ uint32_t sh[kBudgetThreads / 32u + 1u];
  const BudgetState st = W->state[2];
  if (!st.want) return;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  uint32_t before = 0;                         // ties in the tiles before this one
  for (uint32_t t = lane; t < blockIdx.x; t += 32u) before += W->ties[t];
  before = __reduce_add_sync(0xffffffffu, before);
  const uint64_t b = (uint64_t)blockIdx.x * tile;
  const uint32_t m = min(*count, n), e = (uint32_t)min(b + tile, (uint64_t)m);
  for (uint64_t i0 = b; i0 < e; i0 += kBudgetThreads) {
    const uint64_t i = i0 + threadIdx.x;
    const uint32_t key = i < e ? keys[i] : kNoKey;
    const bool tie = key == st.prefix;
    const unsigned tm = __ballot_sync(0xffffffffu, tie);
    if (lane == 0) sh[warp] = __popc(tm);
    __syncthreads();
    uint32_t rank = before + __popc(tm & ((1u << lane) - 1u)), all = 0;
    for (uint32_t w = 0; w < kBudgetThreads / 32u; ++w) {
      if (w < warp) rank += sh[w];
      all += sh[w];
    }
    before += all;
    if (key != kNoKey && (key > st.prefix || (tie && rank < st.want))) marks[list[i]] = PV_INFO_REPLACE;
    __syncthreads();
  }
}

int model_args(const pv_scene* s, const pv_paths* p, const float* theta, uint32_t width, uint32_t height,
               const float* rect, ModelArgs& A) {
  if (!theta || !rect || width == 0 || height == 0 || width > (1u << 20) || height > (1u << 20)) return PV_ERR_ARG;
  if (!(rect[2] > rect[0]) || !(rect[3] > rect[1])) return PV_ERR_ARG;
  std::memset(&A, 0, sizeof A);
  A.n = p->n;
  A.n_lights = s->n_lights;
  A.n_theta = 7 * s->n_lights + 3 * s->n_dyn;
  A.info = p->info;
  A.origin = p->origin;
  A.pa = reinterpret_cast<const float4*>(p->pa);
  A.pb = reinterpret_cast<const float4*>(p->pb);
  A.theta = theta;
  A.W = width;
  A.H = height;
  A.x0 = rect[0];
  A.z0 = rect[1];
  A.x1 = rect[2];
  A.z1 = rect[3];
  for (uint32_t sl = 0; sl < s->n_dyn; ++sl)
    for (int k = 0; k < 3; ++k) A.cur_t[sl][k] = s->h_xf_new[12 * sl + 4 * k + 3];
  return PV_OK;
}

}  // namespace

extern "C" int pv_theta_size(const pv_scene* s) {
  if (!s) return PV_ERR_ARG;
  return (int)(7 * s->n_lights + 3 * s->n_dyn);
}

extern "C" int pv_theta_current(const pv_scene* s, float* h_theta) {
  if (!s || !h_theta) return PV_ERR_ARG;
  for (uint32_t l = 0; l < s->n_lights; ++l) {
    for (int k = 0; k < 3; ++k) {
      h_theta[7 * l + k] = s->lights_new[l].pos[k];
      h_theta[7 * l + 3 + k] = s->lights_new[l].normal[k];
    }
    h_theta[7 * l + 6] = 1.0f;
  }
  for (uint32_t sl = 0; sl < s->n_dyn; ++sl)
    for (int k = 0; k < 3; ++k) h_theta[7 * s->n_lights + 3 * sl + k] = s->h_xf_new[12 * sl + 4 * k + 3];
  return PV_OK;
}

extern "C" int pv_model_deposit(pv_scene* s, const pv_paths* paths, const float* d_theta, float* d_atlas,
                                uint32_t width, uint32_t height, const float* rect, void* stream) {
  int rc = pvh::check_paths(s, paths);
  if (rc != PV_OK) return rc;
  if (!d_atlas) return PV_ERR_ARG;
  ModelArgs A;
  if ((rc = model_args(s, paths, d_theta, width, height, rect, A)) != PV_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  s->last_stream = st;
  // 128 threads a block at most 40 KB of shared memory (15 photons a path)
  constexpr uint32_t kThreads = 128;
  if (paths->n)
    pvh::launch_dependent(k_model_deposit, (paths->n + kThreads - 1) / kThreads, kThreads,
                          kThreads / 32 * warp_smem_bytes<2>(s->B, sizeof(TapSmem)), st, pvh::view(s), pvh::frame_lights(s), A,
                          d_atlas);
  return pvh::cuda_status(cudaGetLastError());
}

extern "C" int pv_adjoint_deposit(pv_scene* s, const pv_paths* paths, const float* d_theta, const float* d_grad_atlas,
                                  uint32_t width, uint32_t height, const float* rect, float* d_dtheta, float* d_score,
                                  void* stream) {
  int rc = pvh::check_paths(s, paths);
  if (rc != PV_OK) return rc;
  if (!d_grad_atlas || !d_dtheta) return PV_ERR_ARG;
  ModelArgs A;
  if ((rc = model_args(s, paths, d_theta, width, height, rect, A)) != PV_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  s->last_stream = st;
  constexpr uint32_t kThreads = 128;
  if (paths->n)
    pvh::launch_dependent(k_adjoint, (paths->n + kThreads - 1) / kThreads, kThreads,
                          kThreads / 32 * warp_smem_bytes<3>(s->B, 0), st, pvh::view(s), pvh::frame_lights(s), A, d_grad_atlas,
                          d_dtheta, d_score);
  return pvh::cuda_status(cudaGetLastError());
}

extern "C" int pv_budget_list(pv_scene* s, const uint32_t* d_list, const uint32_t* d_count, const float* d_score,
                              uint32_t budget, uint32_t* d_out, uint32_t* d_out_count, void* stream) {
  if (!s || !d_list || !d_count || !d_score || !d_out || !d_out_count) return PV_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  s->last_stream = st;
  const uint32_t n = s->n_paths_total;
  if (n == 0) return pvh::cuda_status(cudaMemsetAsync(d_out_count, 0, sizeof(uint32_t), st));
  BudgetWork* W = reinterpret_cast<BudgetWork*>(s->b_work);
  uint32_t* const keys = s->b_keys;
  pvh::ClearSet C;
  C.add(W, sizeof W->hist / sizeof(uint32_t));
  C.add(s->ws_tiles, pvh::compact_words(n));
  pvh::launch_clear(s, C, st);
  const uint32_t blocks = std::min((n + kBudgetStep - 1) / kBudgetStep, 4u * (uint32_t)s->num_sms);
  pvh::launch_dependent(k_budget_hist<0>, blocks, kBudgetThreads, 0, st, d_list, d_count, d_score, n, budget, keys, s->ws_mask, W);
  pvh::launch_dependent(k_budget_hist<1>, blocks, kBudgetThreads, 0, st, d_list, d_count, d_score, n, budget, keys, s->ws_mask, W);
  pvh::launch_dependent(k_budget_hist<2>, blocks, kBudgetThreads, 0, st, d_list, d_count, d_score, n, budget, keys, s->ws_mask, W);
  // tiles of whole steps, at most kBudgetTiles of them
  const uint32_t tile = std::max<uint32_t>((n / pvh::kBudgetTiles / kBudgetStep + 1u) * kBudgetStep, kBudgetStep);
  const uint32_t tiles = (n + tile - 1) / tile;
  pvh::launch_dependent(k_budget_ties, tiles, kBudgetThreads, 0, st, d_count, n, tile, keys, W);
  pvh::launch_dependent(k_budget_mark, tiles, kBudgetThreads, 0, st, d_list, d_count, n, tile, keys, W, s->ws_mask);
  pvh::launch_compact(s, s->ws_mask, n, d_out, d_out_count, nullptr, st, 0, false);
  return pvh::cuda_status(cudaGetLastError());
}
