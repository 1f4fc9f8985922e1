// Analytic-scene ray-caster: the rendering step that fills the per-pixel buffers of
// Eq. 2 (range, strength, angles, velocity; Section II renders them with the light at
// the Tx and the camera at the Rx).  See include/rsim.h for the geometry and the
// definition of each output.
//
// One kernel, rc_render, one thread per pixel of a tile of the image (32 x 8,
// narrower and higher where that pads fewer columns): the ray
// direction from the tile's angles, the first positive hit over all primitives, then normal,
// Lambert strength and closing speed at the hit point.  The FP64 angle of a column or row
// and its sine and cosine are computed once per tile (40 of each instead of 512: FP64 runs
// at 1/64 of the FP32 rate), and up to kRcByValue primitives travel in the kernel's
// arguments instead of a copy ahead of it.  A primitive whose bounding sphere the ray stays
// clear of is skipped after an FP32 test.
// Per call, before and after: 600 x 600 pixels, 100 primitives 165 -> 75 us (FP32), 4423 ->
// 692 us (FP64); 512 x 512, 20 primitives 39 -> 21 us; 256 x 256, 12 primitives 25 -> 20 us
// (FP32, bound by the host's call), 134 -> 49 us (FP64); the same bits.  The primitives are
// staged in shared memory in tiles of 64, each thread of a block deriving one primitive's constants (unit normal,
// the dual basis of a plane, the unit-sphere frame of an ellipsoid, the constant terms
// of the quadratics) in the compute precision T = float for FP32 buffers, double for
// FP64 buffers.  A plane's in-plane coordinates use the dual basis b* = (c x n) / |n|^2,
// c* = (n x b) / |n|^2 (n = b x c), which needs no Gram determinant.
// Every curved surface is met as a sphere in some frame (the end caps as they are, the
// cylinder in the plane across its axis, the ellipsoid in its unit-sphere frame).  The
// roots of |f + t u|^2 = rr (u a unit vector) take the discriminant from the distance
// of the centre to the ray's line, rr - |f - (f . u) u|^2, and the near root as c / q,
// which keeps FP32 precision for rays that graze a surface (Haines, Guenther and
// Akenine-Moller, "Precision Improvements for Ray/Sphere Intersection", Ray Tracing
// Gems, 2019).
#include <math.h>

#include <cmath>
#include <string>

#include "rsim_ctx.h"
#include "rsim_internal.h"

namespace rsim {
namespace {

constexpr int kRcTile = 64;  // primitives per shared-memory tile
constexpr int kRcThreads = 256;
constexpr int kRcByValue = 24;  // 3,840 bytes of kernel arguments

// N primitives in the kernel's arguments; more than kRcByValue come from device memory, and
// their launch carries one (unread) instead of 3,840 bytes.
template <int N>
struct RcArgs {
  rsim_primitive p[N];
};

template <typename T>
struct RcPrim {
  int kind;
  T a[3], v[3], om[3], rho;
  // plane:     e0 = b*, e1 = c* (dual basis: (x - a) = s b + u c gives s = (x - a) . b*,
  //            u = (x - a) . c*), e2 = unit normal; k0 = a . e2
  // capsule:   e0 = b - a (axis), e1 = ap (the origin's offset from the axis line, across
  //            it), e2 = b; k0 = |ap|^2 - r^2, k1 = |a|^2 - r^2, k2 = |b|^2 - r^2, k3 = 1 / |axis|^2
  // ellipsoid: e0, e1, e2 = e_i / |e_i|^2 (the unit-sphere frame); (k0, k1, k2) = s0 = -a . w_i,
  //            k3 = |s0|^2 - 1
  T e0[3], e1[3], e2[3];
  T k0, k1, k2, k3;
  T rr;  // capsule: r^2
  float m[3], reach;  // a sphere that holds the primitive, its radius widened for FP32 rounding
};

template <typename T>
__device__ __forceinline__ T dot3t(const T* x, const T* y) {
  return x[0] * y[0] + x[1] * y[1] + x[2] * y[2];
}

template <typename T>
__device__ __forceinline__ void cross3(const T* x, const T* y, T* z) {
  z[0] = x[1] * y[2] - x[2] * y[1];
  z[1] = x[2] * y[0] - x[0] * y[2];
  z[2] = x[0] * y[1] - x[1] * y[0];
}

// The per-primitive constants of the intersection test, in T.
template <typename T>
__device__ void derive(const rsim_primitive& p, RcPrim<T>& q) {
  T a[3], b[3], c[3], d[3];
  for (int i = 0; i < 3; ++i) {
    a[i] = (T)p.a[i];
    b[i] = (T)p.b[i];
    c[i] = (T)p.c[i];
    d[i] = (T)p.d[i];
    q.a[i] = a[i];
    q.v[i] = (T)p.vel[i];
    q.om[i] = (T)p.omega[i];
  }
  q.kind = p.kind;
  q.rho = (T)p.rho;
  q.k0 = q.k1 = q.k2 = q.k3 = (T)0;
  q.rr = (T)1;
  if (p.kind == RSIM_PRIM_PLANE) {
    T n[3], cn[3], nb[3];
    cross3(b, c, n);
    const T nn = dot3t(n, n), ln = sqrt(nn);
    cross3(c, n, cn);
    cross3(n, b, nb);
    for (int i = 0; i < 3; ++i) {
      q.e0[i] = cn[i] / nn;
      q.e1[i] = nb[i] / nn;
      q.e2[i] = n[i] / ln;
    }
    q.k0 = dot3t(a, q.e2);
  } else if (p.kind == RSIM_PRIM_CAPSULE) {
    const T r = c[0];
    T ax[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
    const T h2 = dot3t(ax, ax);
    const T f = -dot3t(a, ax) / h2;  // (origin - a) . axis / h2
    for (int i = 0; i < 3; ++i) {
      q.e0[i] = ax[i];
      q.e1[i] = -a[i] - f * ax[i];
      q.e2[i] = b[i];
    }
    q.rr = r * r;
    q.k0 = dot3t(q.e1, q.e1) - q.rr;
    q.k1 = dot3t(a, a) - q.rr;
    q.k2 = dot3t(b, b) - q.rr;
    q.k3 = (T)1 / h2;
  } else {  // ellipsoid
    const T* E[3] = {b, c, d};
    T* W[3] = {q.e0, q.e1, q.e2};
    T s0[3];
    for (int i = 0; i < 3; ++i) {
      const T ee = dot3t(E[i], E[i]);
      for (int j = 0; j < 3; ++j) W[i][j] = E[i][j] / ee;
      s0[i] = -dot3t(a, W[i]);
    }
    q.k0 = s0[0];
    q.k1 = s0[1];
    q.k2 = s0[2];
    q.k3 = dot3t(s0, s0) - (T)1;
  }
}

// The sphere about the primitive, in FP32: the middle of the parallelogram, the capsule's
// axis or the ellipsoid, and a radius widened by a thousandth and by 1e-4 of the distance
// (hundreds of times the rounding of the test below and of hit()).  Primitives at distances
// whose square leaves FP32's range get an infinite one.
template <typename T>
__device__ __forceinline__ void bound(const rsim_primitive& p, RcPrim<T>& q) {
  float b[3], c[3], rad;
  for (int i = 0; i < 3; ++i) {
    b[i] = (float)(p.kind == RSIM_PRIM_CAPSULE ? p.b[i] - p.a[i] : p.b[i]);
    c[i] = (float)p.c[i];
    q.m[i] = (float)p.a[i];
  }
  const float bb = dot3t(b, b), cc = dot3t(c, c), bc = dot3t(b, c);
  if (p.kind == RSIM_PRIM_PLANE) {
    for (int i = 0; i < 3; ++i) q.m[i] += 0.5f * (b[i] + c[i]);
    rad = 0.5f * sqrtf(bb + cc + 2.f * fabsf(bc));
  } else if (p.kind == RSIM_PRIM_CAPSULE) {
    for (int i = 0; i < 3; ++i) q.m[i] += 0.5f * b[i];
    rad = 0.5f * sqrtf(bb) + c[0];
  } else {
    const float d[3] = {(float)p.d[0], (float)p.d[1], (float)p.d[2]};
    rad = sqrtf(fmaxf(bb, fmaxf(cc, dot3t(d, d))));
  }
  const float mm = dot3t(q.m, q.m), reach = rad * 1.001f + 1e-4f * sqrtf(mm);
  q.reach = mm > 1e-20f && mm < 1e30f && rad < 1e15f ? reach : INFINITY;
}

// Whether the ray along d (unit, FP32) stays clear of that sphere, or has it behind.
template <typename T>
__device__ __forceinline__ bool clear_of(const RcPrim<T>& q, const float* d) {
  const float b = dot3t(q.m, d);
  const float g[3] = {q.m[0] - b * d[0], q.m[1] - b * d[1], q.m[2] - b * d[2]};
  return dot3t(g, g) > q.reach * q.reach || b < -q.reach;
}

template <typename T>
__device__ __forceinline__ T t_inf() {
  return (T)INFINITY;
}

// The two roots t1 <= t2 of |f + t u|^2 = rr for a unit vector u, with c = |f|^2 - rr;
// false when the line misses the sphere.
template <typename T>
__device__ __forceinline__ bool sphere_roots(const T* f, const T* u, T rr, T c, T& t1, T& t2) {
  const T b = dot3t(f, u);
  const T g[3] = {f[0] - b * u[0], f[1] - b * u[1], f[2] - b * u[2]};
  const T disc = rr - dot3t(g, g);
  if (!(disc >= (T)0)) return false;
  const T q = -b - copysign(sqrt(disc), b);  // |q| = |b| + sqrt(disc): no cancellation
  t1 = q;
  t2 = (q != (T)0) ? c / q : q;
  if (t1 > t2) {
    const T x = t1;
    t1 = t2;
    t2 = x;
  }
  return true;
}

// Smallest positive root of |f + t u|^2 = rr, +inf if none.
template <typename T>
__device__ __forceinline__ T sphere_first(const T* f, const T* u, T rr, T c) {
  T t1, t2;
  if (!sphere_roots(f, u, rr, c, t1, t2)) return t_inf<T>();
  return t1 > (T)0 ? t1 : (t2 > (T)0 ? t2 : t_inf<T>());
}

// Distance along the unit ray d to the primitive (+inf if it misses).
template <typename T>
__device__ T hit(const RcPrim<T>& p, const T* d) {
  if (p.kind == RSIM_PRIM_PLANE) {
    const T dn = dot3t(d, p.e2);
    if (dn == (T)0) return t_inf<T>();
    const T t = p.k0 / dn;
    if (!(t > (T)0)) return t_inf<T>();
    T x[3] = {t * d[0] - p.a[0], t * d[1] - p.a[1], t * d[2] - p.a[2]};
    const T s = dot3t(x, p.e0), u = dot3t(x, p.e1);
    return (s >= (T)0 && s <= (T)1 && u >= (T)0 && u <= (T)1) ? t : t_inf<T>();
  }
  if (p.kind == RSIM_PRIM_CAPSULE) {
    // lateral surface: in the plane across the axis the ray is t dp (dp = d across the
    // axis) from the offset ap, a circle of radius r about the axis; keep the hits whose
    // foot on the axis lies between a and b
    T best = t_inf<T>();
    const T da = dot3t(d, p.e0);
    const T dp[3] = {d[0] - da * p.k3 * p.e0[0], d[1] - da * p.k3 * p.e0[1], d[2] - da * p.k3 * p.e0[2]};
    const T lp = sqrt(dot3t(dp, dp));
    if (lp > (T)0) {
      const T u[3] = {dp[0] / lp, dp[1] / lp, dp[2] / lp};
      T s1, s2;
      if (sphere_roots(p.e1, u, p.rr, p.k0, s1, s2)) {
        const T aax = dot3t(p.a, p.e0);
        const T ts[2] = {s1 / lp, s2 / lp};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const T t = ts[i];
          const T foot = (t * da - aax) * p.k3;
          if (t > (T)0 && foot >= (T)0 && foot <= (T)1 && t < best) best = t;
        }
      }
    }
    // the end spheres about a and b, seen from the origin: f = -a, -b
    const T fa[3] = {-p.a[0], -p.a[1], -p.a[2]};
    const T fb[3] = {-p.e2[0], -p.e2[1], -p.e2[2]};
    const T ta = sphere_first(fa, d, p.rr, p.k1);
    const T tb = sphere_first(fb, d, p.rr, p.k2);
    return fmin(best, fmin(ta, tb));
  }
  // ellipsoid: the unit sphere |s0 + t sd|^2 = 1 in its frame, t = tau / |sd|
  const T sd[3] = {dot3t(d, p.e0), dot3t(d, p.e1), dot3t(d, p.e2)};
  const T ls = sqrt(dot3t(sd, sd));
  const T u[3] = {sd[0] / ls, sd[1] / ls, sd[2] / ls};
  const T s0[3] = {p.k0, p.k1, p.k2};
  return sphere_first(s0, u, (T)1, p.k3) / ls;
}

template <typename T>
__device__ void normal_at(const RcPrim<T>& p, const T* x, T* n) {
  if (p.kind == RSIM_PRIM_PLANE) {
    n[0] = p.e2[0];
    n[1] = p.e2[1];
    n[2] = p.e2[2];
  } else if (p.kind == RSIM_PRIM_CAPSULE) {
    const T xa[3] = {x[0] - p.a[0], x[1] - p.a[1], x[2] - p.a[2]};
    T f = dot3t(xa, p.e0) * p.k3;
    f = f < (T)0 ? (T)0 : (f > (T)1 ? (T)1 : f);
    for (int i = 0; i < 3; ++i) n[i] = xa[i] - f * p.e0[i];
  } else {
    const T xa[3] = {x[0] - p.a[0], x[1] - p.a[1], x[2] - p.a[2]};
    const T s[3] = {dot3t(xa, p.e0), dot3t(xa, p.e1), dot3t(xa, p.e2)};
    for (int i = 0; i < 3; ++i) n[i] = s[0] * p.e0[i] + s[1] * p.e1[i] + s[2] * p.e2[i];
  }
}

template <typename T>
__device__ __forceinline__ void sin_cos(T x, T* s, T* c) {
  if constexpr (sizeof(T) == 4)
    sincosf(x, s, c);
  else
    sincos(x, s, c);
}

// `prims`: the primitives in device memory, or NULL when they are in `byval`.
template <typename T, int N>
__global__ void __launch_bounds__(kRcThreads)
rc_render(const __grid_constant__ RcArgs<N> byval, const rsim_primitive* __restrict__ prims, int n_prims, int n_az,
          int n_el, int tw, int tiles_x, double az0, double az1, double el0, double el1, int falloff, T* __restrict__ R,
          T* __restrict__ sre, T* __restrict__ sim, T* __restrict__ az_out, T* __restrict__ el_out,
          T* __restrict__ vel) {
  __shared__ RcPrim<T> tile[kRcTile];
  // the tile's angles, tw columns then th rows, their sines and cosines (tw + th <= 257)
  __shared__ T ang[kRcThreads + 1], sn[kRcThreads + 1], cs[kRcThreads + 1];
  __shared__ __align__(16) rsim_primitive raw[N];
  const int th = kRcThreads / tw;
  const int i0 = (int)(blockIdx.x % (unsigned)tiles_x) * tw, j0 = (int)(blockIdx.x / (unsigned)tiles_x) * th;
  const int tid = threadIdx.x, tx = tid % tw, ty = tid / tw;
  // in FP64 in the order of the cell-centred grid formula, unfused; from the second warp on,
  // while the first derives primitives
  for (int q = (tid + kRcThreads - 32) % kRcThreads; q < tw + th; q += kRcThreads) {
    const bool is_az = q < tw;
    const double lo = is_az ? az0 : el0, hi = is_az ? az1 : el1;
    const int at = is_az ? i0 + q : j0 + (q - tw), n = is_az ? n_az : n_el;
    const T x = (T)__dadd_rn(lo, __ddiv_rn(__dmul_rn((double)at + 0.5, __dsub_rn(hi, lo)), (double)n));
    ang[q] = x;
    sin_cos(x, &sn[q], &cs[q]);
  }
  if (N > 1 && !prims) {
    const uint32_t* from = reinterpret_cast<const uint32_t*>(&byval);
    uint32_t* to = reinterpret_cast<uint32_t*>(raw);
    for (int w = tid; w < n_prims * (int)(sizeof(rsim_primitive) / 4); w += kRcThreads) to[w] = from[w];
  }
  const rsim_primitive* src = prims ? prims : raw;
  wait_prior_grid();
  __syncthreads();
  const int i = i0 + tx, j = j0 + ty;
  const bool live = i < n_az && j < n_el;
  const int64_t p = (int64_t)j * n_az + i;
  const T a = ang[tx], e = ang[tw + ty];
  const T sa = sn[tx], ca = cs[tx], se = sn[tw + ty], ce = cs[tw + ty];
  const T d[3] = {ce * sa, ce * ca, se};
  const float df[3] = {(float)d[0], (float)d[1], (float)d[2]};
  T best = t_inf<T>();
  int which = -1;
  for (int k0 = 0; k0 < n_prims; k0 += kRcTile) {
    const int nt = min(kRcTile, n_prims - k0);
    __syncthreads();
    for (int k = threadIdx.x; k < nt; k += blockDim.x) {
      derive(src[k0 + k], tile[k]);
      bound(src[k0 + k], tile[k]);
    }
    __syncthreads();
    if (live) {
      for (int k = 0; k < nt; ++k) {
        if (clear_of(tile[k], df)) continue;
        const T t = hit(tile[k], d);
        if (t < best) {  // strict: a tie keeps the primitive listed first
          best = t;
          which = k0 + k;
        }
      }
    }
  }
  if (!live) return;
  T r = t_inf<T>(), s = (T)0, w = (T)0;
  if (which >= 0) {
    RcPrim<T> q;
    if (n_prims <= kRcTile)
      q = tile[which];  // the only tile is still staged
    else
      derive(src[which], q);
    r = best;
    const T x[3] = {r * d[0], r * d[1], r * d[2]};
    T n[3];
    normal_at(q, x, n);
    const T cosi = fabs(dot3t(n, d)) / sqrt(dot3t(n, n));
    s = q.rho * cosi;
    if (falloff) s = s / (r * r);
    const T xa[3] = {x[0] - q.a[0], x[1] - q.a[1], x[2] - q.a[2]};
    const T u[3] = {q.v[0] + q.om[1] * xa[2] - q.om[2] * xa[1], q.v[1] + q.om[2] * xa[0] - q.om[0] * xa[2],
                    q.v[2] + q.om[0] * xa[1] - q.om[1] * xa[0]};
    w = -dot3t(u, d);
  }
  R[p] = r;
  sre[p] = s;
  sim[p] = (T)0;
  az_out[p] = a;
  el_out[p] = e;
  vel[p] = w;
}

bool finite3(const double* x) { return std::isfinite(x[0]) && std::isfinite(x[1]) && std::isfinite(x[2]); }
double hdot(const double* x, const double* y) { return x[0] * y[0] + x[1] * y[1] + x[2] * y[2]; }

// Argument checks of one primitive (the conditions rsim.h lists); "" when valid.
std::string check_prim(const rsim_primitive& p) {
  if (p.kind != RSIM_PRIM_PLANE && p.kind != RSIM_PRIM_CAPSULE && p.kind != RSIM_PRIM_ELLIPSOID)
    return "unknown primitive kind";
  if (!finite3(p.a) || !finite3(p.b) || !finite3(p.c) || !finite3(p.d) || !finite3(p.vel) ||
      !finite3(p.omega) || !std::isfinite(p.rho))
    return "non-finite primitive field";
  if (p.kind == RSIM_PRIM_PLANE) {
    const double bb = hdot(p.b, p.b), cc = hdot(p.c, p.c), bc = hdot(p.b, p.c);
    if (!(bb > 0 && cc > 0 && bb * cc - bc * bc > 1e-12 * bb * cc)) return "plane edges are zero or (nearly) parallel";
  } else if (p.kind == RSIM_PRIM_CAPSULE) {
    if (!(p.c[0] > 0)) return "capsule radius must be > 0";
    const double ax[3] = {p.b[0] - p.a[0], p.b[1] - p.a[1], p.b[2] - p.a[2]};
    if (!(hdot(ax, ax) > 0)) return "capsule ends coincide";
  } else {
    const double* E[3] = {p.b, p.c, p.d};
    for (int i = 0; i < 3; ++i)
      if (!(hdot(E[i], E[i]) > 0)) return "ellipsoid semi-axis is zero";
    for (int i = 0; i < 3; ++i)
      for (int j = i + 1; j < 3; ++j)
        if (std::fabs(hdot(E[i], E[j])) > 1e-9 * std::sqrt(hdot(E[i], E[i]) * hdot(E[j], E[j])))
          return "ellipsoid semi-axes are not orthogonal";
  }
  return "";
}

// Columns of a block's image tile: 32 (whole 128-byte runs of the FP32 arrays), or the power
// of two that holds a narrower image.  Where more than an eighth of the columns would be padding,
// 16 or 8, as long as that pads less: 33 x 3000 pixels, one primitive, FP64 52 -> 34 us (43 with
// pixels numbered in a line), 65 x 400 with 100 264 -> 182; FP32 14 -> 11.5 and 43 -> 37.
int rc_tile_width(int n_az) {
  int w = 1;
  while (w < 32 && w < n_az) w *= 2;
  auto padded = [n_az](int64_t x) { return (n_az + x - 1) / x * x; };
  while (w > 8 && padded(w) > (int64_t)n_az + n_az / 8 && padded(w / 2) < padded(w)) w /= 2;
  return w;
}

// Tiles along the columns, and in all: 64-bit, a side may be as long as an int holds.
int64_t rc_tiles_x(const rsim_camera& cam) {
  const int64_t w = rc_tile_width(cam.n_az);
  return (cam.n_az + w - 1) / w;
}
int64_t rc_tiles(const rsim_camera& cam) {
  const int64_t h = kRcThreads / rc_tile_width(cam.n_az);
  return rc_tiles_x(cam) * ((cam.n_el + h - 1) / h);
}

template <typename T, int N>
cudaError_t launch_raycast(const rsim_primitive* host, const rsim_primitive* dev, int n, const rsim_camera& cam,
                           const rsim_pixel_out& out, cudaStream_t st) {
  RcArgs<N> byval;
  if (!dev)
    for (int i = 0; i < n; ++i) byval.p[i] = host[i];
  return launch_dependent(rc_render<T, N>, dim3((unsigned)rc_tiles(cam)), dim3(kRcThreads), 0, st, byval, dev, n,
                          cam.n_az, cam.n_el, rc_tile_width(cam.n_az), (int)rc_tiles_x(cam), cam.az_min, cam.az_max,
                          cam.el_min, cam.el_max, (cam.flags & RSIM_RC_NO_FALLOFF) ? 0 : 1, (T*)out.range,
                          (T*)out.sigma_re, (T*)out.sigma_im, (T*)out.az, (T*)out.el, (T*)out.vel);
}

}  // namespace
}  // namespace rsim

using namespace rsim;

extern "C" rsim_status rsim_raycast(rsim_ctx* ctx, const rsim_camera* cam, const rsim_primitive* prims,
                                    int32_t n_prims, const rsim_pixel_out* out, rsim_stream stream) {
  if (!ctx || !cam || !out) return fail(RSIM_ERR_INVALID_ARG, "NULL argument");
  if (n_prims < 0 || (n_prims > 0 && !prims)) return fail(RSIM_ERR_INVALID_ARG, "bad primitive array");
  if (cam->n_az < 1 || cam->n_el < 1) return fail(RSIM_ERR_INVALID_ARG, "n_az and n_el must be >= 1");
  if (!std::isfinite(cam->az_min) || !std::isfinite(cam->az_max) || !std::isfinite(cam->el_min) ||
      !std::isfinite(cam->el_max))
    return fail(RSIM_ERR_INVALID_ARG, "non-finite camera angle");
  if (cam->flags & ~RSIM_RC_NO_FALLOFF) return fail(RSIM_ERR_INVALID_ARG, "unknown camera flag bits");
  if (out->P != (int64_t)cam->n_az * cam->n_el) return fail(RSIM_ERR_INVALID_ARG, "out->P != n_az * n_el");
  if (out->dtype != RSIM_F32 && out->dtype != RSIM_F64) return fail(RSIM_ERR_INVALID_ARG, "unknown dtype");
  if (!out->range || !out->sigma_re || !out->sigma_im || !out->az || !out->el || !out->vel)
    return fail(RSIM_ERR_INVALID_ARG, "NULL output array");
  if (rc_tiles(*cam) > 0x7fffffffll) return fail(RSIM_ERR_OVERFLOW, "too many pixels");
  for (int k = 0; k < n_prims; ++k) {
    const std::string why = check_prim(prims[k]);
    if (!why.empty()) return fail(RSIM_ERR_INVALID_ARG, "primitive " + std::to_string(k) + ": " + why);
  }
  cudaSetDevice(ctx->device);
  cudaStream_t st = (cudaStream_t)stream;
  const rsim_primitive* raw = nullptr;
  cudaError_t e = cudaSuccess;
  if (n_prims > kRcByValue) {
    const size_t raw_bytes = ((sizeof(rsim_primitive) * (size_t)n_prims + 255) / 256) * 256;
    rsim_status s = ensure_workspace(ctx, raw_bytes + 256, st);
    if (s != RSIM_OK) return s;
    e = cudaMemcpyAsync(ctx->ws, prims, sizeof(rsim_primitive) * (size_t)n_prims, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return cuda_fail(e, "upload of the primitives");
    raw = (const rsim_primitive*)ctx->ws;
  }
  auto launch = out->dtype == RSIM_F32 ? (raw ? launch_raycast<float, 1> : launch_raycast<float, kRcByValue>)
                                       : (raw ? launch_raycast<double, 1> : launch_raycast<double, kRcByValue>);
  e = launch(prims, raw, n_prims, *cam, *out, st);
  if (e != cudaSuccess) return cuda_fail(e, "ray-caster kernels");
  return RSIM_OK;
}
