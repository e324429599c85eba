// Device geometry of the reverted Monte-Carlo trace: random numbers, cosine
// sampling, ray / triangle tests and the heightfield march over a pyramid of bounding planes.
//
// Every operation whose result decides an integer (hit or miss, hit triangle,
// hit pixel, shadow visibility) is written with explicitly rounded FP32
// intrinsics (__fmul_rn, __fadd_rn, ...), which the compiler never fuses, so
// that the decision is a fixed function of the FP32 inputs.
//
// Coordinates: "grid" space, vertex (i, j) at (x, y, z) = (j, i, depth[i*W+j]);
// a world direction (dx, dy, dz) maps to (W dx, W dy, dz) (pixel pitch 1/W).
// Cell (cy, cx) holds triangles T0 = {(cy,cx), (cy,cx+1), (cy+1,cx+1)} and
// T1 = {(cy,cx), (cy+1,cx+1), (cy+1,cx)} with index 2*(cy*(W-1)+cx) + {0,1}.
#pragma once

#include <cstdint>
#include <math.h>
#include <cuda_runtime.h>

namespace irtps {

constexpr int kMaxLevels = 16;

__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }

struct F3 {
  float x, y, z;
};

__device__ __forceinline__ F3 f3sub(F3 a, F3 b) { return {rsub(a.x, b.x), rsub(a.y, b.y), rsub(a.z, b.z)}; }
__device__ __forceinline__ F3 f3cross(F3 a, F3 b) {
  return {rsub(rmul(a.y, b.z), rmul(a.z, b.y)), rsub(rmul(a.z, b.x), rmul(a.x, b.z)),
          rsub(rmul(a.x, b.y), rmul(a.y, b.x))};
}
__device__ __forceinline__ float f3dot(F3 a, F3 b) {
  return radd(radd(rmul(a.x, b.x), rmul(a.y, b.y)), rmul(a.z, b.z));
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k.x += 0x9E3779B9u;
      k.y += 0xBB67AE85u;
    }
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}

// 24-bit uniform in [0, 1), exact in FP32.
__device__ __forceinline__ float u24(uint32_t x) { return __uint2float_rn(x >> 8) * 5.9604644775390625e-08f; }

// cos(2 pi u), sin(2 pi u) for a 24-bit u: quadrant reduction (exact) and Taylor
// polynomials on [0, pi/4], every step rounded to FP32 on its own.
__device__ __forceinline__ void sincos_turn(float u, float &c, float &s) {
  const float v = rmul(u, 4.0f);
  const int q = (int)v;
  const float f = rsub(v, (float)q);
  const bool swap = f > 0.5f;
  const float g = swap ? rsub(1.0f, f) : f;
  const float x = rmul(g, (float)M_PI_2);
  const float x2 = rmul(x, x);
  float ps = 1.0f / 362880.0f;
  ps = rmul(ps, x2);
  ps = radd(-(1.0f / 5040.0f), ps);
  ps = rmul(ps, x2);
  ps = radd(1.0f / 120.0f, ps);
  ps = rmul(ps, x2);
  ps = radd(-(1.0f / 6.0f), ps);
  ps = rmul(ps, x2);
  ps = radd(1.0f, ps);
  const float sx = rmul(x, ps);
  float pc = -(1.0f / 3628800.0f);
  pc = rmul(pc, x2);
  pc = radd(1.0f / 40320.0f, pc);
  pc = rmul(pc, x2);
  pc = radd(-(1.0f / 720.0f), pc);
  pc = rmul(pc, x2);
  pc = radd(1.0f / 24.0f, pc);
  pc = rmul(pc, x2);
  pc = radd(-0.5f, pc);
  pc = rmul(pc, x2);
  const float cx = radd(1.0f, pc);
  const float st = swap ? cx : sx;
  const float ct = swap ? sx : cx;
  switch (q & 3) {
    case 0: c = ct; s = st; break;
    case 1: c = -st; s = ct; break;
    case 2: c = -ct; s = -st; break;
    default: c = st; s = -ct; break;
  }
}

// Cosine-weighted direction about the unit normal n (Malley's method) in the
// orthonormal basis of Duff et al., "Building an Orthonormal Basis, Revisited".
__device__ __forceinline__ F3 cosine_dir(F3 n, uint32_t x0, uint32_t x1) {
  const float u1 = u24(x0), u2 = u24(x1);
  const float r = __fsqrt_rn(u1);
  float c, s;
  sincos_turn(u2, c, s);
  const float lx = rmul(r, c), ly = rmul(r, s);
  const float lz = __fsqrt_rn(rsub(1.0f, u1));
  const float sign = copysignf(1.0f, n.z);
  const float a = __fdiv_rn(-1.0f, radd(sign, n.z));
  const float b = rmul(rmul(n.x, n.y), a);
  const F3 b1 = {radd(1.0f, rmul(rmul(rmul(sign, n.x), n.x), a)), rmul(sign, b), rmul(-sign, n.x)};
  const F3 b2 = {b, radd(sign, rmul(rmul(n.y, n.y), a)), -n.y};
  return {radd(radd(rmul(lx, b1.x), rmul(ly, b2.x)), rmul(lz, n.x)),
          radd(radd(rmul(lx, b1.y), rmul(ly, b2.y)), rmul(lz, n.y)),
          radd(radd(rmul(lx, b1.z), rmul(ly, b2.z)), rmul(lz, n.z))};
}

// Moeller-Trumbore, two-sided, closed barycentric bounds, hit iff t > 0.
__device__ __forceinline__ bool tri_hit(F3 o, F3 d, F3 v0, F3 v1, F3 v2, float &t_out) {
  const F3 e1 = f3sub(v1, v0);
  const F3 e2 = f3sub(v2, v0);
  const F3 pv = f3cross(d, e2);
  const float det = f3dot(e1, pv);
  if (det == 0.0f) return false;
  const float inv = __frcp_rn(det);
  const F3 tv = f3sub(o, v0);
  const float u = rmul(f3dot(tv, pv), inv);
  if (u < 0.0f || u > 1.0f) return false;
  const F3 qv = f3cross(tv, e1);
  const float v = rmul(f3dot(d, qv), inv);
  if (v < 0.0f || radd(u, v) > 1.0f) return false;
  const float t = rmul(f3dot(e2, qv), inv);
  if (!(t > 0.0f)) return false;
  t_out = t;
  return true;
}

// Heightfield + pyramids as the kernels see them.  The level table (offsets and
// row widths) lives in shared memory, filled by each block before use, so that
// a lane-dependent level index does not force it into local memory.
struct Field {
  const float *depth;       // H*W
  const float *pmax;        // maxima, all levels, level l at off[l], row-major lw[l] wide
  const uint2 *planes;      // upper bounding planes of the same nodes (see plane_pack)
  int H, W, Wc, Hc;         // Wc = W-1, Hc = H-1 cells
  int levels;               // levels the march uses (the top one may hold several nodes)
  int top_off;              // offset of the single node of the full pyramid (the surface maximum)
  int off[kMaxLevels];
  int lw[kMaxLevels];
};

struct LevelTable {
  int2 ol[kMaxLevels];  // per level: offset of its nodes in the pyramid arrays, row width
  const uint2 *planes;  // the object's planes (batched launches read them here)
  float zmax_margin;    // (max height) + 1e-4: above it a rising ray can hit nothing
  float dz;             // node-skip margin on heights, 1e-5 (1 + |max height|)
  int top;              // top level of the march
  int pad;
};

// Height bounds of a surface from its top pyramid node.
__device__ __forceinline__ void set_height_bounds(const Field &f, LevelTable *t) {
  const float zmax = __ldg(f.pmax + f.top_off);
  t->zmax_margin = zmax + 1e-4f;
  t->dz = 1e-5f * (1.0f + fabsf(zmax));
  t->planes = f.planes;
  t->top = f.levels - 1;
}

// Copy the level table of f into shared memory and derive the height bounds from
// the top pyramid node (whole block; ends with a barrier).
__device__ __forceinline__ void load_levels(const Field &f, LevelTable *t) {
  if (threadIdx.x < kMaxLevels) t->ol[threadIdx.x] = make_int2(f.off[threadIdx.x], f.lw[threadIdx.x]);
  if (threadIdx.x == 0) set_height_bounds(f, t);
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Upper bounding plane of a pyramid node: surface(x, y) <= gx x + gy y + c over
// the node's rectangle, x and y in grid units.  The slopes are BF16 pairs (any
// slopes bound the surface once c is chosen for them), c is FP32 and rounded up,
// so that a node takes one 8-byte load.  The stored c is raised by plane_slack,
// which covers the rounding of the march's evaluation: at most 40 roundings of
// terms up to |gx| W + |gy| H (about 2.4e-6 of their sum).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float plane_slack(float gx, float gy, float W, float H) {
  return __fmul_ru(3e-6f, __fadd_ru(__fmul_ru(fabsf(gx), W), __fmul_ru(fabsf(gy), H)));
}
__device__ __forceinline__ float bf16_round(float v) {  // to the nearest BF16 (ties away), finite values
  return __uint_as_float((__float_as_uint(v) + 0x8000u) & 0xffff0000u);
}
__device__ __forceinline__ uint2 plane_pack(float gx, float gy, float c) {
  return make_uint2(__float_as_uint(gx) | (__float_as_uint(gy) >> 16), __float_as_uint(c));
}
__device__ __forceinline__ void plane_unpack(uint2 v, float &gx, float &gy, float &c) {
  gx = __uint_as_float(v.x & 0xffff0000u);
  gy = __uint_as_float(v.x << 16);
  c = __uint_as_float(v.y);
}

// Work counters of one thread (pyramid nodes / cells examined, triangle tests, sampled directions).
struct Work {
  uint32_t nodes = 0, tris = 0, draws = 0;
};

constexpr float kHitMargin = 1e-4f;   // entry beyond best hit by this: stop
constexpr float kCorner = 1e-5f;      // near-vertex crossing: test both side cells

// Both triangles of cell (cy, cx).  This is the Moeller-Trumbore test above
// written out for the cell's vertices, whose x and y are consecutive integers:
// every product with an edge component of 0 or 1 is exact, so dropping it leaves
// each remaining rounding, and hence every result bit, unchanged.  The
// rejections are evaluated as one predicate per triangle (straight-line code).
__device__ __forceinline__ void test_cell(const Field &f, int cy, int cx, F3 o, F3 d, float &bt, int &btri, Work &w) {
  w.tris += 2;
  const float *r0 = f.depth + (size_t)cy * f.W + cx;
  const float h00 = __ldg(r0), h01 = __ldg(r0 + 1), h10 = __ldg(r0 + f.W), h11 = __ldg(r0 + f.W + 1);
  const int base = 2 * (cy * f.Wc + cx);
  // shared by both triangles: v0 = (cx, cy, h00), tv = o - v0
  const F3 tv = {rsub(o.x, (float)cx), rsub(o.y, (float)cy), rsub(o.z, h00)};
  const float e11 = rsub(h11, h00);  // z of v11 - v0 (edge to the far corner)
  // T0 = (v00, v01, v11): e1 = (1, 0, h01 - h00), e2 = (1, 1, h11 - h00)
  float t0;
  bool hit0;
  {
    const float e1z = rsub(h01, h00);
    const F3 pv = {rsub(rmul(d.y, e11), d.z), rsub(d.z, rmul(d.x, e11)), rsub(d.x, d.y)};
    const float det = radd(pv.x, rmul(e1z, pv.z));
    const float inv = __frcp_rn(det);
    const float u = rmul(f3dot(tv, pv), inv);
    const F3 qv = {rmul(tv.y, e1z), rsub(tv.z, rmul(tv.x, e1z)), -tv.y};
    const float v = rmul(f3dot(d, qv), inv);
    t0 = rmul(radd(radd(qv.x, qv.y), rmul(e11, qv.z)), inv);
    hit0 = det != 0.0f && u >= 0.0f && u <= 1.0f && v >= 0.0f && radd(u, v) <= 1.0f && t0 > 0.0f;
  }
  // T1 = (v00, v11, v10): e1 = (1, 1, h11 - h00), e2 = (0, 1, h10 - h00)
  float t1;
  bool hit1;
  {
    const float e2z = rsub(h10, h00);
    const F3 pv = {rsub(rmul(d.y, e2z), d.z), -rmul(d.x, e2z), d.x};
    const float det = radd(radd(pv.x, pv.y), rmul(e11, pv.z));
    const float inv = __frcp_rn(det);
    const float u = rmul(f3dot(tv, pv), inv);
    const F3 qv = {rsub(rmul(tv.y, e11), tv.z), rsub(tv.z, rmul(tv.x, e11)), rsub(tv.x, tv.y)};
    const float v = rmul(f3dot(d, qv), inv);
    t1 = rmul(radd(qv.y, rmul(e2z, qv.z)), inv);
    hit1 = det != 0.0f && u >= 0.0f && u <= 1.0f && v >= 0.0f && radd(u, v) <= 1.0f && t1 > 0.0f;
  }
  if (hit0 && (btri < 0 || t0 < bt || (t0 == bt && base < btri))) {
    bt = t0;
    btri = base;
  }
  if (hit1 && (btri < 0 || t1 < bt || (t1 == bt && base + 1 < btri))) {
    bt = t1;
    btri = base + 1;
  }
}

// Incremental heightfield march.  The leaf steps are those of a plain 2D cell
// walk: the grid line X is crossed at parameter e(X) = (X - o) * (1/d) (one
// rounding per operation), lines are crossed in order of e, ties on both axes
// together (a diagonal step), and both side cells are tested at a near-vertex
// crossing.  Whole pyramid nodes that the ray passes above are skipped.
//
// The march stands on a node (nx, ny) of level lv, entered at parameter te: the
// state of the plain walk once every line with e <= te is crossed.  A skip
// crosses the node's exit line at its own e, so it needs no cell index; only a
// descent asks which child holds the ray, and that is whether the middle line is
// crossed (e(mid) <= te).  The leaf cells reached are therefore exactly those of
// the plain walk, and every hit is the plain walk's.
//
// Both axes are mirrored so that the ray moves toward +x and +y: x' = -x and node
// index n' = ~n where d.x < 0 (mask mx = -1).  Negation is exact, so every e keeps
// its bits, and the steps need no direction signs.  The start cell holds the
// origin, on the side the ray moves toward when the origin is on a grid line; a
// ray running exactly along a grid line walks the cells on both sides (up to four
// walks), its traversal origin moved off the line by one ulp toward the walk's
// side (1/0 = inf then orders every line of that axis correctly).
//
// A node is passed when the ray stays above its bounding plane (plane_pack) by the
// margin dz from entry to exit.  Against a constant bound (the node's maximum),
// which a ray leaving a slope clears only after several nodes of every level, the
// planes cut the node visits per segment from 30.1 to 14.3 and the tested cells from 2.7 to 0.9 on a 2048 x 2048
// scene of 200 bumps (7.9 to 4.2 and 1.0 to 0.3 at 512 x 512 with 20; climbs and start level included).  The
// 512 x 512, K = 12, 256-spp trace went from 167 to 131 ms, the 2048 x 2048, K = 16, 16-spp one from 805 to 487 ms.
struct Walker {
  float ox, oy, oz;  // traversal origin: x, y mirrored, z lowered by the node-skip margin
  float dx, dy, dz;  // direction, x and y mirrored (|d.x|, |d.y|)
  float ax, ay;      // 1 / dx, 1 / dy
  int mx, my;        // -1 where the axis is mirrored, else 0
  int nx, ny, lv;    // current node (mirrored index) and its level
  float te;          // entry parameter
  float t_end;       // the walk is over once te lies beyond it: outside the grid, past the best hit (plus
                     // a margin), or, rising, above every vertex (plus a margin)
  float bt;
  int btri;
  int flags;  // bit 0: any-hit; bits 1, 2: a second walk in x, in y; bits 3-4: current walk index; 5-6: see
              // walker_leaf_step; 7, 8: sign bits of the direction's x and y
};

// The true direction (signs of zeros too).
__device__ __forceinline__ F3 walker_dir(const Walker &m) {
  return {__int_as_float(__float_as_int(m.dx) | ((m.flags << 24) & (int)0x80000000)),
          __int_as_float(__float_as_int(m.dy) | ((m.flags << 23) & (int)0x80000000)), m.dz};
}

// (float)(n + 1) of a node index by a magic addition (no conversion unit); |n| < 2^22, and the pyramid's 16 levels hold
// the sides to 2^15 cells.
__device__ __forceinline__ float node_edge(int n) {
  return __fsub_rn(__int_as_float(n + 0x4B400000), 12582911.0f);
}
// Crossing parameter of the line k * s (both exact in FP32): one rounding each for the difference and the product.
__device__ __forceinline__ float line_e(float k, float s, float o, float inv) {
  return rmul(__fmaf_rn(k, s, -o), inv);
}

// v moved by one ulp, up or down.
__device__ __forceinline__ float off_line(float v, bool up) {
  const int i = __float_as_int(v);
  if (v == 0.0f) return __int_as_float(up ? 1 : (int)0x80000001);
  return __int_as_float(i + ((i >= 0) == up ? 1 : -1));
}

// Start cell of walk `wi` (see above).  Returns false when it lies outside the grid.
__device__ __forceinline__ bool walker_begin_walk(Walker &m, const Field &f, F3 o, int wi) {
  int cx = (int)floorf(o.x), cy = (int)floorf(o.y);
  if ((float)cx == o.x && m.mx) --cx;
  if ((float)cy == o.y && m.my) --cy;
  if (m.flags & 6) {  // along a grid line: the second walk one column / row back, the origin off the line
    const int wx = (m.flags & 2) ? wi & 1 : 0, wy = (m.flags & 2) ? wi >> 1 : wi;
    cx -= wx;
    cy -= wy;
    if (m.flags & 2) m.ox = off_line(o.x, wx == 0);
    if (m.flags & 4) m.oy = off_line(o.y, wy == 0);
    m.flags = (m.flags & ~(3 << 3)) | (wi << 3);
  }
  m.nx = cx ^ m.mx;
  m.ny = cy ^ m.my;
  m.lv = 0;
  m.te = 0.0f;
  return (unsigned)cx < (unsigned)f.Wc && (unsigned)cy < (unsigned)f.Hc;
}

// Set up a ray.  Returns true when its walk is over at once (it starts outside the grid).
__device__ __forceinline__ bool walker_init(Walker &m, const Field &f, const LevelTable &lt, F3 o, F3 d, bool any) {
  m.mx = d.x < 0.0f ? -1 : 0;
  m.my = d.y < 0.0f ? -1 : 0;
  m.ox = m.mx ? -o.x : o.x;
  m.oy = m.my ? -o.y : o.y;
  m.oz = o.z - lt.dz;
  m.dx = fabsf(d.x);
  m.dy = fabsf(d.y);
  m.dz = d.z;
  m.ax = __frcp_rn(m.dx);
  m.ay = __frcp_rn(m.dy);
  const bool on_x = floorf(o.x) == o.x, on_y = floorf(o.y) == o.y;
  m.flags = (any ? 1 : 0) | ((on_x && d.x == 0.0f) ? 2 : 0) | ((on_y && d.y == 0.0f) ? 4 : 0) |
            (int)(((__float_as_uint(d.x) >> 31) << 7) | ((__float_as_uint(d.y) >> 31) << 8));
  m.bt = __int_as_float(0x7f800000);
  m.btri = -1;
  // a rising ray is above every vertex (by the margin) beyond this parameter; any rounding of it
  // only moves the end of the walk within the margin, where no triangle can be hit
  const float t_top = d.z > 0.0f ? __fdividef(lt.zmax_margin - o.z, d.z) : __int_as_float(0x7f800000);
  const bool in = walker_begin_walk(m, f, o, 0);
  // the grid is left at its far lines' e (above 0 when `in`); te reaching it ends the walk (te > the float
  // below it); an axis along which the ray does not move has none
  const float inf = __int_as_float(0x7f800000);
  const float gx = (m.flags & 2) ? inf : line_e(m.mx ? 0.0f : (float)f.Wc, 1.0f, m.ox, m.ax);
  const float gy = (m.flags & 4) ? inf : line_e(m.my ? 0.0f : (float)f.Hc, 1.0f, m.oy, m.ay);
  m.t_end = fminf(t_top, __int_as_float(__float_as_int(fminf(gx, gy)) - 1));
  return !in;
}

// The end of a walk: ends the march, or moves to the next walk of a grid-line ray.
// Returns true when the march is over.
__device__ __forceinline__ bool walker_finish_walk(Walker &m, const Field &f, F3 o) {
  if ((m.flags & 6) == 0 || ((m.flags & 1) && m.btri >= 0)) return true;
  const int walks = ((m.flags & 2) ? 2 : 1) * ((m.flags & 4) ? 2 : 1);
  for (int wi = ((m.flags >> 3) & 3) + 1; wi < walks; ++wi)
    if (walker_begin_walk(m, f, o, wi)) return false;
  return true;
}

// Cross the exit lines at tx, ty (the earlier one; both on a tie) and climb, by up to kClimb levels, to
// the largest node whose border that crosses: the bits of the indexes that the step changes say how many
// levels it leaves.
#ifndef IRTPS_CLIMB
#define IRTPS_CLIMB 2
#endif
constexpr int kClimb = IRTPS_CLIMB;
constexpr int kStartLevel = 3;  // level of a primary ray's march after a quick start
__device__ __forceinline__ void walker_cross(Walker &m, float tx, float ty, int top) {
  const int nx = m.nx + (tx <= ty ? 1 : 0), ny = m.ny + (ty <= tx ? 1 : 0);
  m.te = fminf(tx, ty);
  const int up = min(min(31 - __clz((nx ^ m.nx) | (ny ^ m.ny) | 1), kClimb), top - m.lv);
  m.nx = nx >> up;
  m.ny = ny >> up;
  m.lv += up;
}

// The march advances in two kinds of steps.  A node step examines the node: it
// passes over it, descends to the child the ray enters, or - at level 0, when the
// ray is not above the cell - leaves the walker waiting for a leaf step, which
// tests the cell's triangles and takes the plain walk's step to the next cell.
// Keeping the two apart lets a warp run the expensive leaf step for many lanes at once.

// Node step.  Returns true when the walk is over; sets at_leaf when the walker waits for a leaf step.
// The multiply-adds of the plane test run on the FMA pipes, which the march otherwise leaves idle (the
// integer and compare pipe is its bound), and the node's edges come from a magic addition.
__device__ __forceinline__ bool walker_node_step(Walker &m, const uint2 *__restrict__ planes, const LevelTable &lt,
                                                 int top, bool &at_leaf, Work &w) {
  if (m.te > m.t_end) return true;
  ++w.nodes;
  const int2 ol = lt.ol[m.lv];
  const uint2 pv = __ldg(planes + (ol.x + (m.ny ^ m.my) * ol.y + (m.nx ^ m.mx)));
  const float s = __int_as_float(m.lv * (1 << 23) + 0x3f800000);  // 2^lv
  const float fx = node_edge(m.nx), fy = node_edge(m.ny);
  const float tx = line_e(fx, s, m.ox, m.ax), ty = line_e(fy, s, m.oy, m.ay);
  const float t_exit = fminf(tx, ty);
  // clearance above the plane (margin included in oz), linear in t: least at entry or exit
  const float gx = __uint_as_float((pv.x & 0xffff0000u) ^ ((unsigned)m.mx & 0x80000000u));
  const float gy = __uint_as_float((pv.x << 16) ^ ((unsigned)m.my & 0x80000000u));
  const float A = fmaf(-gx, m.ox, fmaf(-gy, m.oy, m.oz - __uint_as_float(pv.y)));
  const float B = fmaf(-gx, m.dx, fmaf(-gy, m.dy, m.dz));
  if (fminf(fmaf(m.te, B, A), fmaf(t_exit, B, A)) > 0.0f) {
    walker_cross(m, tx, ty, top);
  } else if (m.lv > 0) {
    const float h = 0.5f * s;
    const bool far_x = line_e(fx + fx - 1.0f, h, m.ox, m.ax) <= m.te;
    const bool far_y = line_e(fy + fy - 1.0f, h, m.oy, m.ay) <= m.te;
    m.nx = 2 * m.nx + (far_x ? 1 : 0);
    m.ny = 2 * m.ny + (far_y ? 1 : 0);
    --m.lv;
  } else {
    at_leaf = true;
  }
  return false;
}

// Leaf step: both triangles of the current cell, then the plain walk's step.  At a
// near-vertex crossing the two cells beside the vertex are tested too, each by a leaf step of
// its own (flag bits 5-6), so that the test stands in the code once.
enum : int { LEAF_ON = 0, LEAF_OVER = 1, LEAF_AGAIN = 2 };  // walk on, walk over, another leaf step first
__device__ __forceinline__ int walker_leaf_step(Walker &m, const Field &f, F3 o, int top, Work &w) {
  const float inf = __int_as_float(0x7f800000);
  const F3 d = walker_dir(m);
  const int side = (m.flags >> 5) & 3;  // 0: the cell, 1: the one beside it in x, 2: in y
  const int cx = (m.nx + (side == 1 ? 1 : 0)) ^ m.mx, cy = (m.ny + (side == 2 ? 1 : 0)) ^ m.my;
  if ((unsigned)cx < (unsigned)f.Wc && (unsigned)cy < (unsigned)f.Hc) test_cell(f, cy, cx, o, d, m.bt, m.btri, w);
  const float tx = line_e(node_edge(m.nx), 1.0f, m.ox, m.ax);
  const float ty = line_e(node_edge(m.ny), 1.0f, m.oy, m.ay);
  if (fmaxf(tx, ty) < inf && fabsf(rsub(tx, ty)) <= rmul(kCorner, fmaxf(tx, ty)) && side < 2) {
    m.flags += 1 << 5;
    return LEAF_AGAIN;
  }
  m.flags &= ~(3 << 5);
  if (m.btri >= 0) {
    if (m.flags & 1) return LEAF_OVER;
    m.t_end = fminf(m.t_end, radd(m.bt, kHitMargin));  // later cells may only hold closer hits
  }
  if (fminf(tx, ty) == inf) return LEAF_OVER;
  walker_cross(m, tx, ty, top);
  return LEAF_ON;
}

// Step over the first cell of a primary ray (it starts at a vertex: the cell's lines lie at 1 * (1/d)), on to
// level kStartLevel at once: most rays that clear their first cell clear the nodes around it too.
__device__ __forceinline__ void walker_start_next(Walker &m, int top) {
  const int lv = min(kStartLevel, top);
  m.nx = (m.nx + (m.ax <= m.ay ? 1 : 0)) >> lv;
  m.ny = (m.ny + (m.ay <= m.ax ? 1 : 0)) >> lv;
  m.te = fminf(m.ax, m.ay);
  m.lv = lv;
}

// Blocking march (probes, render): steps until done or until `budget` steps are used.
__device__ __forceinline__ bool march(const Field &f, const LevelTable &lt, F3 o, F3 d, bool any, float &t, int &tri,
                                     int &budget, Work &w) {
  Walker m;
  bool over = walker_init(m, f, lt, o, d, any);
  while (!(over && walker_finish_walk(m, f, o))) {
    bool at_leaf = false;
    over = walker_node_step(m, f.planes, lt, f.levels - 1, at_leaf, w);
    while (at_leaf) {
      const int st = walker_leaf_step(m, f, o, f.levels - 1, w);
      over = st == LEAF_OVER;
      at_leaf = st == LEAF_AGAIN;
    }
    if (--budget < 0) break;
  }
  t = m.bt;
  tri = m.btri;
  return m.btri >= 0;
}

// ---------------------------------------------------------------------------
// Quick start of primary rays.  A primary ray leaves the pixel's own vertex p,
// lifted by a little, into one cell; a, b, c are the heights of that cell's other
// vertices above p's (across x, across y, across both, in the mirrored axes).  True when
// neither triangle of the cell can be hit in FP32, so that the cell's test is skipped:
//  - a triangle whose plane holds p is missed by a ray steeper than the plane
//    (the plane is met at t < 0: the lift is positive and exact to 2^-22 of the edges);
//  - where the diagonal does not meet p, the far triangle's plane passes k = a + b - c
//    above p; the ray is steeper than it too and, for k > 0, meets it before the
//    diagonal (by 2^-8 of the way), outside the triangle.
// The slope margin 2^-10 bounds the determinants away from zero, so that the test's
// barycentric coordinates are off by at most 2^-11.  Not taken near the cell's far
// corner, where the walk would test the side cells too.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool start_cell_clear(const Walker &m, float lift, float a, float b, float c) {
  const float e = fmaxf(fabsf(a), fmaxf(fabsf(b), fabsf(c)));
  const float sum = m.dx + m.dy;
  const float margin = 9.765625e-4f * fmaf(sum, e, fabsf(m.dz));
  const bool through = m.mx == m.my;  // the diagonal meets p
  const float s1 = fmaf(m.dx, a, m.dy * (through ? c - a : b));
  const float s2 = fmaf(m.dx, c - b, m.dy * (through ? b : c - a));
  const float q1 = m.dz - s1, q2 = m.dz - s2;
  const bool before = through || (a + b - c) * sum <= 0.99609375f * q2;
  return q1 > margin && q2 > margin && before && lift >= 9.5367431640625e-7f * e &&
         fabsf(m.ax - m.ay) > kCorner * fmaxf(m.ax, m.ay);
}

// ---------------------------------------------------------------------------
// Early escape of primary rays.  For every pixel vertex p and each of the eight
// octants of azimuth (signs of the grid direction's x and y, and whether |y|
// exceeds |x|; the diagonals belong to both neighbours), hz bounds from above
// the slope (height per grid unit) under which the terrain is seen from p:
//   hz = max over cells c meeting the closed octant wedge at p, c not touching p,
//        of (max height of c - H_p) / (distance from p to c).
// A rising ray leaving p's lifted vertex with slope above hz is at every cell c of
// the wedge above c's highest vertex (its height there is at least
// H_p + dist * slope), so it can hit nothing beyond the cell it starts in.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int octant_of(float gx, float gy) {
  return (gx < 0.0f ? 1 : 0) | (gy < 0.0f ? 2 : 0) | (fabsf(gy) > fabsf(gx) ? 4 : 0);
}

// Whether the rectangle [a1, a2] x [b1, b2] (relative to p) meets the closed wedge of octant o.
__device__ __forceinline__ bool wedge_meets(int o, int a1, int a2, int b1, int b2) {
  int A1 = a1, A2 = a2, B1 = b1, B2 = b2;
  if (o & 1) { A1 = -a2; A2 = -a1; }
  if (o & 2) { B1 = -b2; B2 = -b1; }
  if (o & 4) {
    int t = A1; A1 = B1; B1 = t;
    t = A2; A2 = B2; B2 = t;
  }
  return A2 >= 0 && B2 >= 0 && max(B1, 0) <= A2;
}

// Nearest vertex index of a hit coordinate, ties to the lower index.
__device__ __forceinline__ int nearest_index(float q, int n) {
  const int v = (int)ceilf(rsub(q, 0.5f));
  return min(n - 1, max(0, v));
}

}  // namespace irtps
