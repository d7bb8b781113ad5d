// Scene-partition kernels (paper Sec. 4.1 airspace-aware visibility, Sec. 4.3 seamless merging).
//
//  - Airspace boxes: per cell, min / max of the points' x and z and max of y, by block
//    reductions and order-preserving integer atomics (one launch per 256 cells, chunks of 4K points).
//  - Visibility: one thread per (camera, cell) pair, in double-floats: the area of the projected box inside the
//    image rectangle over the image area, as edge integrals: of the silhouette for a box in front of
//    the near plane, of the faces turned away (clipped by it) for one that the plane cuts.  Where the
//    faces have no orientation (a singular camera) or the magnitudes are extreme the box is clipped in FP64,
//    projected, its convex hull (monotone chain) clipped to the image rectangle (Sutherland-Hodgman),
//    and the shoelace area taken.
//  - Merge: one pass over all cells' Gaussians.  Blocks take 1,024 Gaussians in ticket order, test
//    the region, find their output offset by a decoupled look-back over the blocks before them,
//    and copy the kept Gaussians' parameters straight into the merged arrays.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <vector>

#include "doublefloat.cuh"
#include "internal.h"
#include "vg_common.cuh"
#include "vgpartition.h"

namespace vg {
namespace {

// ---------------------------------------------------------------- airspace boxes

// Order-preserving map of a float to an unsigned integer (so atomicMin / atomicMax order floats).
__device__ __forceinline__ unsigned f2ord(float f) {
  const unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(unsigned o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

// Points per block: 16K made 1,232 blocks of the 20M points of 16 cells, one wave of 8 an SM and a second
// wave of 16 blocks (53 us); short chunks even that out.
constexpr int kBoxChunk = 1 << 12;
constexpr int kBoxCellsPerLaunch = 256;

// Chunk table of one launch: cell c of the launch owns blocks [chunk[c], chunk[c+1]) and points
// [first[c], first[c] + count[c]).
struct BoxJob {
  int n;
  int chunk[kBoxCellsPerLaunch + 1];
  long long first[kBoxCellsPerLaunch];
  long long count[kBoxCellsPerLaunch];
};

__global__ void box_init(unsigned* ob, int n_cells) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n_cells) return;
  for (int a = 0; a < 3; ++a) {
    ob[6 * k + a] = 0xFFFFFFFFu;   // running minima start at the largest ordinal
    ob[6 * k + 3 + a] = 0u;        // running maxima at the smallest
  }
}

__global__ void __launch_bounds__(256) box_reduce(const float* __restrict__ pts, const BoxJob job, unsigned* ob) {
  __shared__ unsigned sm[6][8];
  int lo_c = 0, hi_c = job.n - 1;   // this block's cell: the last c with chunk[c] <= blockIdx.x
  while (lo_c < hi_c) {
    const int mid = (lo_c + hi_c + 1) >> 1;
    if (job.chunk[mid] <= (int)blockIdx.x) lo_c = mid; else hi_c = mid - 1;
  }
  const int c = lo_c;
  unsigned v[6] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0u, 0u, 0u};
  const long long lo = (long long)(blockIdx.x - job.chunk[c]) * kBoxChunk;
  const int n = (int)(lo + kBoxChunk < job.count[c] ? kBoxChunk : job.count[c] - lo);
  const float* p = pts + 3 * (job.first[c] + lo);
  auto put = [&](int a, float f) {
    const unsigned o = f2ord(f);
    v[a] = min(v[a], o);
    v[3 + a] = max(v[3 + a], o);
  };
  // four points are three 16-byte words once the address allows (a multiple of 4 bytes plus 12 k, so
  // after at most three points); the points before that and after the last four by scalar loads
  int head = 0;
  while (head < n && head < 4 && (reinterpret_cast<uintptr_t>(p + 3 * head) & 15u)) ++head;
  const int quads = (n - head) / 4, tail = head + 4 * quads;
  const int loose = head + (n - tail);
  if ((int)threadIdx.x < loose) {
    const int i = (int)threadIdx.x < head ? (int)threadIdx.x : tail + ((int)threadIdx.x - head);
#pragma unroll
    for (int a = 0; a < 3; ++a) put(a, __ldg(p + 3 * i + a));
  }
  const float4* w = reinterpret_cast<const float4*>(p + 3 * head);
#pragma unroll 4
  for (int i = threadIdx.x; i < quads; i += blockDim.x) {
    const float4 x = __ldg(w + 3 * i), y = __ldg(w + 3 * i + 1), z = __ldg(w + 3 * i + 2);
    put(0, x.x); put(1, x.y); put(2, x.z);
    put(0, x.w); put(1, y.x); put(2, y.y);
    put(0, y.z); put(1, y.w); put(2, z.x);
    put(0, z.y); put(1, z.z); put(2, z.w);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      const unsigned w = __shfl_xor_sync(0xffffffffu, v[a], o);
      v[a] = a < 3 ? min(v[a], w) : max(v[a], w);
    }
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int a = 0; a < 6; ++a) sm[a][wp] = v[a];
  __syncthreads();
  if (threadIdx.x < 6) {
    const int a = threadIdx.x;
    unsigned r = sm[a][0];
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) r = a < 3 ? min(r, sm[a][k]) : max(r, sm[a][k]);
    unsigned* dst = ob + 6 * (size_t)c;
    if (a < 3) atomicMin(dst + a, r); else atomicMax(dst + a, r);
  }
}

// ordinals -> floats; y starts at the ground plane
__global__ void box_finish(unsigned* ob, int n_cells, float ground_y) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n_cells) return;
  float* f = reinterpret_cast<float*>(ob);
  float v[6];
  for (int a = 0; a < 6; ++a) v[a] = ord2f(ob[6 * k + a]);
  const bool empty = ob[6 * k] == 0xFFFFFFFFu;    // no point was reduced into this cell
  if (empty) {
    v[0] = v[1] = v[2] = INFINITY;
    v[3] = v[4] = v[5] = -INFINITY;
  } else {
    v[1] = ground_y;
  }
  for (int a = 0; a < 6; ++a) f[6 * k + a] = v[a];
}

// ---------------------------------------------------------------- visibility

constexpr int kMaxPoly = 32;   // >= 2 x 16 (the hull stack) and >= 16 + 4 (four clips of a convex hull)

struct D2 {
  double x, y;
};

__device__ __forceinline__ double cross3(const D2& o, const D2& a, const D2& b) {
  return (a.x - o.x) * (b.y - o.y) - (a.y - o.y) * (b.x - o.x);
}

// Convex hull of p[0..n) (n <= 16) by the monotone chain, counter-clockwise, into h; returns its size.
__device__ int hull(D2* p, int n, D2* h) {
  for (int i = 1; i < n; ++i) {   // insertion sort by (x, y)
    const D2 q = p[i];
    int j = i - 1;
    while (j >= 0 && (p[j].x > q.x || (p[j].x == q.x && p[j].y > q.y))) {
      p[j + 1] = p[j];
      --j;
    }
    p[j + 1] = q;
  }
  if (n <= 2) {
    for (int i = 0; i < n; ++i) h[i] = p[i];
    return n;
  }
  int k = 0;
  for (int i = 0; i < n; ++i) {
    while (k >= 2 && cross3(h[k - 2], h[k - 1], p[i]) <= 0.0) --k;
    h[k++] = p[i];
  }
  for (int i = n - 2, t = k + 1; i >= 0; --i) {
    while (k >= t && cross3(h[k - 2], h[k - 1], p[i]) <= 0.0) --k;
    h[k++] = p[i];
  }
  return k - 1;
}

// Sutherland-Hodgman clip of poly[0..n) by the half-plane (coordinate `axis` >= or <= bound).
__device__ int clip_poly(const D2* in, int n, D2* out, int axis, double bound, bool keep_greater) {
  int m = 0;
  for (int k = 0; k < n; ++k) {
    const D2 a = in[k], b = in[(k + 1) % n];
    const double av = axis ? a.y : a.x, bv = axis ? b.y : b.x;
    const bool ina = keep_greater ? av >= bound : av <= bound;
    const bool inb = keep_greater ? bv >= bound : bv <= bound;
    if (ina && m < kMaxPoly) out[m++] = a;
    if (ina != inb && m < kMaxPoly) {
      const double t = (bound - av) / (bv - av);
      out[m++] = D2{a.x + t * (b.x - a.x), a.y + t * (b.y - a.y)};
    }
  }
  return m;
}

__device__ double box_visibility(const float* box, const vg_camera& cam) {
  double R[9], t[3];
  for (int r = 0; r < 3; ++r) {
    for (int c = 0; c < 3; ++c) R[3 * r + c] = (double)cam.world_to_cam[4 * r + c];
    t[r] = (double)cam.world_to_cam[4 * r + 3];
  }
  double c[8][3];
  for (int k = 0; k < 8; ++k) {
    const double w[3] = {(double)box[(k & 1) ? 3 : 0], (double)box[((k >> 1) & 1) ? 4 : 1],
                         (double)box[((k >> 2) & 1) ? 5 : 2]};
    for (int r = 0; r < 3; ++r) c[k][r] = R[3 * r] * w[0] + R[3 * r + 1] * w[1] + R[3 * r + 2] * w[2] + t[r];
  }
  const double near = (double)cam.near_plane;
  // the box clipped to z >= near: its inside corners and its edges' crossings of the plane (a
  // plane crosses at most 6 edges of a box, and then at most 7 corners are inside: <= 13 points)
  double q[16][3];
  int nq = 0;
  for (int k = 0; k < 8; ++k)
    if (c[k][2] >= near) {
      q[nq][0] = c[k][0]; q[nq][1] = c[k][1]; q[nq][2] = c[k][2];
      ++nq;
    }
  const int edges[12][2] = {{0, 1}, {2, 3}, {4, 5}, {6, 7}, {0, 2}, {1, 3}, {4, 6}, {5, 7}, {0, 4}, {1, 5}, {2, 6}, {3, 7}};
  for (int e = 0; e < 12; ++e) {
    const double* a = c[edges[e][0]];
    const double* b = c[edges[e][1]];
    if ((a[2] - near) * (b[2] - near) < 0.0) {
      const double s = (near - a[2]) / (b[2] - a[2]);
      for (int r = 0; r < 3; ++r) q[nq][r] = a[r] + s * (b[r] - a[r]);
      ++nq;
    }
  }
  if (nq == 0) return 0.0;
  D2 p[16], h[kMaxPoly], g[kMaxPoly];
  const double fx = cam.fx, fy = cam.fy, cx = cam.cx, cy = cam.cy;
  for (int k = 0; k < nq; ++k) p[k] = D2{fx * q[k][0] / q[k][2] + cx, fy * q[k][1] / q[k][2] + cy};
  int n = hull(p, nq, h);
  if (n < 3) return 0.0;
  const double W = cam.width, H = cam.height;
  n = clip_poly(h, n, g, 0, -0.5, true);
  if (n < 3) return 0.0;
  n = clip_poly(g, n, h, 0, W - 0.5, false);
  if (n < 3) return 0.0;
  n = clip_poly(h, n, g, 1, -0.5, true);
  if (n < 3) return 0.0;
  n = clip_poly(g, n, h, 1, H - 0.5, false);
  if (n < 3) return 0.0;
  double a2 = 0.0;
  for (int k = 0; k < n; ++k) {
    const D2& a = h[k];
    const D2& b = h[(k + 1) % n];
    a2 += a.x * b.y - a.y * b.x;
  }
  return 0.5 * fabs(a2) / (W * H);
}

// Silhouette of a box by which of its faces are turned away from the camera: bit 2a + side for the
// face of axis a on its lower (0) or upper (1) side.  An edge along axis a, on side kb of axis b and kc
// of axis c (a, b, c cyclic), lies on the silhouette if just one of its two faces is turned away, and
// runs along that face's boundary as seen from outside: upwards for face (b, kb) if kb == kc.  Corner k
// has its x, y, z sides in bits 0, 1, 2.
struct Silhouette {
  unsigned char n[64];
  unsigned char edge[64][6];      // first corner | second corner << 3
};
constexpr Silhouette make_silhouettes() {
  Silhouette t{};
  for (int mask = 0; mask < 64; ++mask) {
    int n = 0;
    unsigned char e[12] = {};
    for (int a = 0; a < 3; ++a)
      for (int q = 0; q < 4; ++q) {
        const int b = (a + 1) % 3, c = (a + 2) % 3, kb = q & 1, kc = q >> 1;
        const bool away_b = (mask >> (2 * b + kb)) & 1, away_c = (mask >> (2 * c + kc)) & 1;
        if (away_b == away_c) continue;
        const int base = (kb << b) | (kc << c), top = base | (1 << a);
        const bool up = (kb == kc) == away_b;
        e[n++] = (unsigned char)(up ? base | (top << 3) : top | (base << 3));
      }
    // the faces of one axis are never both turned towards a camera outside: other masks are rounding
    const bool seen = (mask & 3) != 0 && (mask & 12) != 0 && (mask & 48) != 0 && n <= 6;
    t.n[mask] = (unsigned char)(seen ? n : 0);
    for (int k = 0; k < 6; ++k) t.edge[mask][k] = seen && k < n ? e[k] : 0;
  }
  return t;
}
__constant__ Silhouette c_silhouette = make_silhouettes();

__device__ __forceinline__ dd dd_clamp(dd v, float lo, float hi) {
  return v < dd(lo) ? dd(lo) : dd(hi) < v ? dd(hi) : v;
}

// Signed area between the image of the edge p -> n (camera coordinates, both in front) and the image's left
// side, with x clamped to [-1/2, W - 1/2] and y to [-1/2, H - 1/2]: the integral of clamp(x(y)) + 1/2 over
// the edge's y.  Summed over a closed polygon's edges it is the signed area of its intersection with that
// rectangle, and exactly 0 for a polygon beside the image: above and below no edge has a y in range, on the
// left every x is clamped to 0, and on the right (where the dy would only cancel up to rounding) no edge
// sets `within`, which says that some of it has an x left of the right side.  The bounds of y are met in
// space, where they are linear, not on the image, where the end of an edge beside the camera lies a
// million pixels off and takes the digits with it.
__device__ __forceinline__ dd edge_area(const dd* p, const dd* n, const vg_camera& cam, bool& within) {
  const float width = (float)cam.width, yh = (float)cam.height - 0.5f;
  const dd fx(cam.fx), fy(cam.fy), cx = dd(cam.cx) + dd(0.5f), cy(cam.cy), below = cy + dd(0.5f), above = dd(yh) - cy;
  const dd ph = fy * p[1], nh = fy * n[1];
  const dd lo0 = ph + below * p[2], lo1 = nh + below * n[2];       // >= 0: at or above the lower bound
  const dd hi0 = above * p[2] - ph, hi1 = above * n[2] - nh;       // >= 0: at or below the upper bound
  if ((lo0.h <= 0.f && lo1.h <= 0.f) || (hi0.h <= 0.f && hi1.h <= 0.f)) return dd(0.f);
  auto at = [&](const dd* e, dd eh, dd lo, dd hi, dd& x, dd& y) {
    dd q0 = e[0], q2 = e[2];
    const bool under = lo.h < 0.f, over = hi.h < 0.f;
    if (under || over) {
      const dd t = under ? lo0 / (lo0 - lo1) : hi0 / (hi0 - hi1);
      q0 = p[0] + t * (n[0] - p[0]);
      q2 = p[2] + t * (n[2] - p[2]);
    }
    x = fx * q0 / q2 + cx;
    y = under ? dd(-0.5f) : over ? dd(yh) : eh / q2 + cy;
  };
  dd xa, ya, xb, yb;
  at(p, ph, lo0, hi0, xa, ya);
  at(n, nh, lo1, hi1, xb, yb);
  const dd dy = yb - ya, ca = dd_clamp(xa, 0.f, width), cb = dd_clamp(xb, 0.f, width);
  within = within || !(ca == dd(width) && cb == dd(width));
  if (ca == cb) return dy * ca;
  const dd mean = dd(0.5f) * (ca + cb);
  if (ca == xa && cb == xb) return dy * mean;
  // constant before x enters the range at ca and after it leaves at cb; as ca plus a part of cb - ca, so
  // that an end a million pixels off does not cancel against itself
  return dy * (ca + (cb - ca) * ((xb - mean) / (xb - xa)));
}

// A box in camera coordinates: the lower corner and the edges; which faces are turned away (bits as in
// Silhouette, 0 if that has no meaning here: a singular camera, or magnitudes that double-floats or
// the areas formed from them would not hold).
struct CamBox {
  dd c0[3], e[3][3];
  int away;
  bool thin;        // a line or a point
};
constexpr float kFarBox = 1e9f, kNearest = 1e-6f, kLongest = 1e7f;   // metres, metres, pixels
__device__ __forceinline__ CamBox cam_box(const float* __restrict__ box, const vg_camera& cam) {
  CamBox q;
  dd lo[3], len[3];
  float R[3][3], top = 0.f;
  int flat = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float u = fminf(box[a], box[a + 3]), v = fmaxf(box[a], box[a + 3]);
    lo[a] = dd(u);
    len[a] = dd(v) - dd(u);
    top = fmaxf(top, fmaxf(fabsf(u), fabsf(v)));
    flat += u == v ? 1 : 0;
  }
  bool ok = top < kFarBox && cam.near_plane > kNearest && cam.fx < kLongest && cam.fy < kLongest &&
            fabsf(cam.cx) < kLongest && fabsf(cam.cy) < kLongest;
#pragma unroll
  for (int a = 0; a < 6; ++a) ok = ok && fabsf(box[a]) < kFarBox;     // false for a NaN
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    dd t(cam.world_to_cam[4 * r + 3]);
    ok = ok && fabsf(t.h) < kFarBox;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      R[a][r] = cam.world_to_cam[4 * r + a];
      ok = ok && fabsf(R[a][r]) < 1e3f;
      t = t + dd(R[a][r]) * lo[a];
      q.e[a][r] = dd(R[a][r]) * len[a];
    }
    q.c0[r] = t;
  }
  // the camera (the origin) against the planes of each axis's two faces, normal R_b x R_c (so that a
  // flat box has two faces too, one of them turned away)
  q.away = 0;
  q.thin = flat >= 2;
  dd det(0.f);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float* f = R[(a + 1) % 3];
    const float* g = R[(a + 2) % 3];
    dd n[3];
#pragma unroll
    for (int r = 0; r < 3; ++r)
      n[r] = dd(f[(r + 1) % 3]) * dd(g[(r + 2) % 3]) - dd(f[(r + 2) % 3]) * dd(g[(r + 1) % 3]);
    if (a == 0) det = dd(R[0][0]) * n[0] + dd(R[0][1]) * n[1] + dd(R[0][2]) * n[2];
    const dd s = q.c0[0] * n[0] + q.c0[1] * n[1] + q.c0[2] * n[2], u = s + len[a] * det;
    const bool lower = det.h > 0.f ? s.h <= 0.f : s.h >= 0.f, upper = det.h > 0.f ? u.h >= 0.f : u.h <= 0.f;
    q.away |= (lower ? 1 : 0) << (2 * a) | (upper ? 2 : 0) << (2 * a);
  }
  if (!ok || !(fabsf(det.h) > 1e-6f)) q.away = 0;
  return q;
}
__device__ __forceinline__ void cam_corner(const CamBox& q, int k, dd* p) {
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    dd v = q.c0[r];
    if (k & 1) v = v + q.e[0][r];
    if (k & 2) v = v + q.e[1][r];
    if (k & 4) v = v + q.e[2][r];
    p[r] = v;
  }
}
// Signed image area of face `face` (2 axis + side) of a box, clipped by the near plane, if it is turned
// away from the camera, else 0.  The faces turned away tile the silhouette whether or not the near plane
// cuts it: what the plane uncovers is seen from inside.
__device__ dd face_area(const CamBox& q, int face, const vg_camera& cam) {
  if (!((q.away >> face) & 1)) return dd(0.f);
  const int b = 1 << ((face >> 1) + 1) % 3, c = 1 << ((face >> 1) + 2) % 3, base = (face & 1) << (face >> 1);
  const dd near(cam.near_plane);
  // corners in the order b, c: counter-clockwise from outside on the upper face, clockwise on the lower
  const int around[4] = {base, base | b, base | b | c, base | c};
  dd p[3], area(0.f), out[3], in[3];
  bool cuts = false, within = false;
  cam_corner(q, around[3], p);
#pragma unroll 1
  for (int k = 0; k < 4; ++k) {
    dd n[3];
    cam_corner(q, around[k], n);
    const bool in0 = !(p[2] < near), in1 = !(n[2] < near);
    if (in0 || in1) {
      dd u[3] = {p[0], p[1], p[2]}, v[3] = {n[0], n[1], n[2]};
      if (in0 != in1) {
        const dd s = (near - p[2]) / (n[2] - p[2]);
        const dd w[3] = {p[0] + s * (n[0] - p[0]), p[1] + s * (n[1] - p[1]), near};
        cuts = true;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          if (in0) v[r] = out[r] = w[r];
          else u[r] = in[r] = w[r];
        }
      }
      area = area + edge_area(u, v, cam, within);
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) p[r] = n[r];
  }
  if (cuts) area = area + edge_area(out, in, cam, within);       // along the near plane
  return !within ? dd(0.f) : (face & 1) ? area : -area;
}

// Bound by instruction issue.  A box wholly in front of the near plane (most) takes no arrays, sorts or
// hull: eight corners, three cross products, at most six edge integrals.  Boxes that the near plane cuts
// are gathered, and a block's threads take one face of one of them each, since one such lane would
// hold up its warp.  All in double-floats: 4,000 cameras x 16 cells took 188 us on the general path in
// FP64, and 295 us on these paths in FP64 (about 1,000 instructions a pair at 16 clocks a warp).
constexpr int kVisThreads = 128;
__global__ void __launch_bounds__(kVisThreads) visibility_kernel(const float* __restrict__ boxes, int n_cells,
                                                                 const vg_camera* __restrict__ cams, int n_cams,
                                                                 double threshold, float* out_vis, uint8_t* out_sel) {
  __shared__ float2 s_p[8][3][kVisThreads];     // corners (boxes in front)
  __shared__ float2 s_area[6 * kVisThreads];    // faces (boxes that the near plane cuts)
  __shared__ int s_cut[kVisThreads];
  __shared__ int s_ncut;
  if (threadIdx.x == 0) s_ncut = 0;
  __syncthreads();
  const long long first = (long long)blockIdx.x * kVisThreads, idx = first + threadIdx.x;
  const long long pairs = (long long)n_cams * n_cells;
  auto put = [&](long long i, double v) {
    if (out_vis) out_vis[i] = (float)v;
    if (out_sel) out_sel[i] = v > threshold ? 1 : 0;
  };
  auto share = [](dd a, const vg_camera& cam) {
    return fabs((double)a.h + (double)a.l) / ((double)cam.width * (double)cam.height);
  };
  if (idx < pairs) {
    const vg_camera& cam = cams[idx / n_cells];
    const float* box = boxes + 6 * (idx % n_cells);
    const CamBox q = cam_box(box, cam);
    int in = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      dd p[3];
      cam_corner(q, k, p);
      in += p[2] < dd(cam.near_plane) ? 0 : 1;
#pragma unroll
      for (int r = 0; r < 3; ++r) s_p[k][r][threadIdx.x] = make_float2(p[r].h, p[r].l);
    }
    const int edges = c_silhouette.n[q.away];
    if (q.away == 0) {
      put(idx, box_visibility(box, cam));
    } else if (in == 0 || q.thin) {      // thin: no area, and its edges' would cancel only up to rounding
      put(idx, 0.0);
    } else if (in == 8 && edges > 0) {
      dd area(0.f);
      bool within = false;
#pragma unroll 1
      for (int k = 0; k < edges; ++k) {
        const int w = c_silhouette.edge[q.away][k];
        dd p[3], n[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const float2 a = s_p[w & 7][r][threadIdx.x], b = s_p[w >> 3][r][threadIdx.x];
          p[r] = dd(a.x, a.y);
          n[r] = dd(b.x, b.y);
        }
        area = area + edge_area(p, n, cam, within);
      }
      put(idx, within ? share(area, cam) : 0.0);
    } else {
      s_cut[atomicAdd(&s_ncut, 1)] = threadIdx.x;
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int t = threadIdx.x; t < 6 * s_ncut; t += kVisThreads) {
    const long long i = first + s_cut[t / 6];
    const vg_camera& cam = cams[i / n_cells];
    const dd a = face_area(cam_box(boxes + 6 * (i % n_cells), cam), t % 6, cam);
    s_area[t] = make_float2(a.h, a.l);
  }
  __syncthreads();
  if ((int)threadIdx.x < s_ncut) {
    const long long i = first + s_cut[threadIdx.x];
    dd area(0.f);
    for (int f = 0; f < 6; ++f) area = area + dd(s_area[6 * threadIdx.x + f].x, s_area[6 * threadIdx.x + f].y);
    put(i, share(area, cams[i / n_cells]));
  }
}

// ---------------------------------------------------------------- merge

struct MCell {
  const float* means;
  const float* ls;
  const float* q;
  const float* lg;
  const float* sh;
  long long offset;   // first merged-input index of this cell
  float x0, x1, z0, z1;
};

struct MergeOut {
  float *means, *ls, *q, *lg, *sh;
  long long* n;
};

__device__ __forceinline__ int find_cell(const MCell* cells, int n_cells, long long i) {
  int lo = 0, hi = n_cells - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (cells[mid].offset <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Bound by HBM: 12 bytes of every mean, 236 read and written of every kept Gaussian at degree 3.  A
// block lists its kept Gaussians in shared memory and copies their rows together (copy_rows); one
// thread copying its own Gaussian's rows reached 0.47 of the measured HBM rate (20M Gaussians of 16
// cells: 1,942 us), its 16-byte stores 192 bytes apart.  Four Gaussians a thread make a quarter of
// the blocks that look back one after another.
constexpr int kMergeItems = 4, kMergeTile = 256 * kMergeItems;
template <int F>
__global__ void __launch_bounds__(256, 8) merge_kernel(const MCell* __restrict__ cells, int n_cells, long long total,
                                                    unsigned* ticket, unsigned long long* status, MergeOut out,
                                                    unsigned* timeout) {
  __shared__ unsigned s_blk, s_base;
  __shared__ unsigned s_sm[8];
  __shared__ uint2 s_row[kMergeTile];     // (cell, index in it) of each kept Gaussian
  if (threadIdx.x == 0) s_blk = atomicAdd(ticket, 1u);
  __syncthreads();
  const unsigned blk = s_blk;
  // a thread takes consecutive Gaussians, so that one scan gives the output order
  const long long i0 = (long long)blk * kMergeTile + (long long)threadIdx.x * kMergeItems;
  uint2 row[kMergeItems];
  unsigned keep = 0;
  int k = i0 < total ? find_cell(cells, n_cells, i0) : 0;
#pragma unroll
  for (int j = 0; j < kMergeItems; ++j) {
    const long long i = i0 + j;
    if (i >= total) continue;
    while (k + 1 < n_cells && cells[k + 1].offset <= i) ++k;
    const MCell& c = cells[k];
    const long long li = i - c.offset;
    row[j] = make_uint2((unsigned)k, (unsigned)li);
    const float x = __ldg(c.means + 3 * li), z = __ldg(c.means + 3 * li + 2);
    if (x >= c.x0 && x < c.x1 && z >= c.z0 && z < c.z1) keep |= 1u << j;
  }
  unsigned tot;
  unsigned at = block_exclusive_scan((unsigned)__popc(keep), &tot, s_sm);
#pragma unroll
  for (int j = 0; j < kMergeItems; ++j)
    if (keep >> j & 1u) s_row[at++] = row[j];
  if (threadIdx.x < 32) {
    const unsigned excl = lookback(status, blk, tot, timeout);
    if (threadIdx.x == 0) {
      s_base = excl;
      if (blk == gridDim.x - 1) {
        __threadfence();
        *out.n = atomicOr(timeout, 0u) ? -1ll : (long long)(excl + tot);
      }
    }
  }
  __syncthreads();
  const size_t o = s_base;
  auto none = [](int) { return false; };
  auto from = [&](const float* MCell::*a, int w) {
    return [=](int r) { const uint2 g = s_row[r]; return cells[g.x].*a + (size_t)g.y * w; };
  };
  copy_rows<F, F % 4 == 0>(out.sh + o * F, (int)tot, from(&MCell::sh, F), none);
  copy_rows<4, true>(out.q + o * 4, (int)tot, from(&MCell::q, 4), none);
  copy_rows<3, false>(out.means + o * 3, (int)tot, from(&MCell::means, 3), none);
  copy_rows<3, false>(out.ls + o * 3, (int)tot, from(&MCell::ls, 3), none);
  copy_rows<1, false>(out.lg + o, (int)tot, from(&MCell::lg, 1), none);
}

struct MergeLayout {
  size_t cells, ticket, status, total;
};

MergeLayout merge_layout(int n_cells, long long total) {
  MergeLayout L{};
  size_t o = 0;
  auto take = [&](size_t b) { size_t at = o; o = align_up(o + b); return at; };
  L.cells = take(sizeof(MCell) * (size_t)n_cells);
  L.ticket = take(2 * sizeof(unsigned));   // ticket, timeout flag
  L.status = take(sizeof(unsigned long long) * (size_t)((total + kMergeTile - 1) / kMergeTile + 1));
  L.total = o;
  return L;
}

bool valid_cam(const vg_camera& c) {
  return c.width >= 1 && c.width <= 16384 && c.height >= 1 && c.height <= 16384 && c.fx > 0.f && c.fy > 0.f &&
         c.near_plane > 0.f;
}

bool aligned256(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 255u) == 0; }

}  // namespace
}  // namespace vg

using namespace vg;

extern "C" vg_status vg_airspace_boxes(const float* points, const int64_t* cell_offsets, int32_t n_cells,
                                       float ground_y, float* out_boxes, vg_stream stream) {
  if (!points || !cell_offsets || !out_boxes || n_cells < 1) return VG_ERR_INVALID;
  for (int k = 0; k < n_cells; ++k)
    if (cell_offsets[k] < 0 || cell_offsets[k + 1] < cell_offsets[k]) return VG_ERR_INVALID;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  unsigned* ob = reinterpret_cast<unsigned*>(out_boxes);
  box_init<<<(n_cells + 127) / 128, 128, 0, s>>>(ob, n_cells);
  int launches = 2;
  // one launch per group of up to 256 cells; a block reduces 4K points of one cell
  for (int k0 = 0; k0 < n_cells; k0 += kBoxCellsPerLaunch) {
    BoxJob job{};
    job.n = n_cells - k0 < kBoxCellsPerLaunch ? n_cells - k0 : kBoxCellsPerLaunch;
    long long blocks = 0;
    for (int c = 0; c < job.n; ++c) {
      job.chunk[c] = (int)blocks;
      job.first[c] = cell_offsets[k0 + c];
      job.count[c] = cell_offsets[k0 + c + 1] - cell_offsets[k0 + c];
      blocks += (job.count[c] + kBoxChunk - 1) / kBoxChunk;
    }
    job.chunk[job.n] = (int)blocks;
    if (blocks == 0) continue;
    if (blocks > 0x7FFFFFFFll) return VG_ERR_INVALID;
    box_reduce<<<(unsigned)blocks, 256, 0, s>>>(points, job, ob + 6 * (size_t)k0);
    ++launches;
  }
  box_finish<<<(n_cells + 127) / 128, 128, 0, s>>>(ob, n_cells, ground_y);
  note_launches(launches);
  return cudaGetLastError() == cudaSuccess ? VG_OK : VG_ERR_CUDA;
}

extern "C" size_t vg_visibility_workspace_bytes(int32_t n_cams) {
  if (n_cams < 1) return 0;
  return align_up(sizeof(vg_camera) * (size_t)n_cams);
}

extern "C" vg_status vg_camera_visibility(const float* boxes, int32_t n_cells, const vg_camera* cams, int32_t n_cams,
                                          float threshold, void* workspace, size_t workspace_bytes,
                                          float* out_visibility, uint8_t* out_selected, vg_stream stream) {
  if (!boxes || !cams || !workspace || n_cells < 1 || n_cams < 1 || (!out_visibility && !out_selected))
    return VG_ERR_INVALID;
  for (int i = 0; i < n_cams; ++i)
    if (!valid_cam(cams[i])) return VG_ERR_INVALID;
  if (!aligned256(workspace)) return VG_ERR_INVALID;
  if (workspace_bytes < vg_visibility_workspace_bytes(n_cams)) return VG_ERR_CAPACITY;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  vg_camera* dcams = static_cast<vg_camera*>(workspace);
  if (cudaMemcpyAsync(dcams, cams, sizeof(vg_camera) * (size_t)n_cams, cudaMemcpyHostToDevice, s) != cudaSuccess)
    return VG_ERR_CUDA;
  const long long pairs = (long long)n_cams * n_cells;
  visibility_kernel<<<(unsigned)((pairs + kVisThreads - 1) / kVisThreads), kVisThreads, 0, s>>>(
      boxes, n_cells, dcams, n_cams, (double)threshold, out_visibility, out_selected);
  note_launches(1);
  return cudaGetLastError() == cudaSuccess ? VG_OK : VG_ERR_CUDA;
}

extern "C" size_t vg_merge_workspace_bytes(const vg_gaussians* cells, int32_t n_cells) {
  if (!cells || n_cells < 1) return 0;
  long long total = 0;
  for (int k = 0; k < n_cells; ++k) {
    if (cells[k].n < 0) return 0;
    total += cells[k].n;
  }
  return merge_layout(n_cells, total).total;
}

extern "C" vg_status vg_merge_cells(const vg_gaussians* cells, const float* regions, int32_t n_cells, void* workspace,
                                    size_t workspace_bytes, float* out_means, float* out_log_scales, float* out_quats,
                                    float* out_opacity_logits, float* out_sh, int64_t* out_n, vg_stream stream) {
  if (!cells || !regions || !workspace || n_cells < 1 || !out_means || !out_log_scales || !out_quats ||
      !out_opacity_logits || !out_sh || !out_n)
    return VG_ERR_INVALID;
  const int deg = cells[0].sh_degree;
  if (deg < 0 || deg > 3) return VG_ERR_INVALID;
  std::vector<MCell> host(n_cells);
  long long total = 0;
  for (int k = 0; k < n_cells; ++k) {
    const vg_gaussians& g = cells[k];
    if (g.sh_degree != deg || g.n < 0 || g.n > 0x7FFFFFFFll) return VG_ERR_INVALID;
    if (g.n > 0 && (!g.means || !g.log_scales || !g.quats || !g.opacity_logits || !g.sh)) return VG_ERR_INVALID;
    if (g.n > 0 && ((reinterpret_cast<uintptr_t>(g.quats) & 15u) ||
                    ((deg == 1 || deg == 3) && (reinterpret_cast<uintptr_t>(g.sh) & 15u))))
      return VG_ERR_INVALID;
    host[k] = MCell{g.means, g.log_scales, g.quats, g.opacity_logits, g.sh, total,
                    regions[4 * k], regions[4 * k + 1], regions[4 * k + 2], regions[4 * k + 3]};
    total += g.n;
  }
  if (total > 0x7FFFFFFFll) return VG_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(out_quats) & 15u) ||
      ((deg == 1 || deg == 3) && (reinterpret_cast<uintptr_t>(out_sh) & 15u)))
    return VG_ERR_INVALID;
  if (!aligned256(workspace)) return VG_ERR_INVALID;
  const MergeLayout L = merge_layout(n_cells, total);
  if (workspace_bytes < L.total) return VG_ERR_CAPACITY;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(workspace);
  if (total == 0) {
    if (cudaMemsetAsync(out_n, 0, sizeof(int64_t), s) != cudaSuccess) return VG_ERR_CUDA;
    return VG_OK;
  }
  if (cudaMemcpyAsync(ws + L.cells, host.data(), sizeof(MCell) * host.size(), cudaMemcpyHostToDevice, s) != cudaSuccess)
    return VG_ERR_CUDA;
  const unsigned blocks = (unsigned)((total + kMergeTile - 1) / kMergeTile);
  if (cudaMemsetAsync(ws + L.ticket, 0, 2 * sizeof(unsigned), s) != cudaSuccess ||
      cudaMemsetAsync(ws + L.status, 0, sizeof(unsigned long long) * blocks, s) != cudaSuccess)
    return VG_ERR_CUDA;
  const MergeOut out{out_means, out_log_scales, out_quats, out_opacity_logits, out_sh,
                     reinterpret_cast<long long*>(out_n)};
  const MCell* dc = reinterpret_cast<const MCell*>(ws + L.cells);
  unsigned* ticket = reinterpret_cast<unsigned*>(ws + L.ticket);
  unsigned long long* status = reinterpret_cast<unsigned long long*>(ws + L.status);
  switch (deg) {
    case 0: merge_kernel<3><<<blocks, 256, 0, s>>>(dc, n_cells, total, ticket, status, out, ticket + 1); break;
    case 1: merge_kernel<12><<<blocks, 256, 0, s>>>(dc, n_cells, total, ticket, status, out, ticket + 1); break;
    case 2: merge_kernel<27><<<blocks, 256, 0, s>>>(dc, n_cells, total, ticket, status, out, ticket + 1); break;
    default: merge_kernel<48><<<blocks, 256, 0, s>>>(dc, n_cells, total, ticket, status, out, ticket + 1); break;
  }
  note_launches(1);
  return cudaGetLastError() == cudaSuccess ? VG_OK : VG_ERR_CUDA;
}
