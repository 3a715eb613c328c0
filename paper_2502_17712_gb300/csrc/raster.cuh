// Visibility: depth pre-pass and "<=" marking pass (Sec. 5.1; App. A "Detecting
// Visible Triangles") as a software rasterizer.
//
// Per triangle (one thread, warps over 32 consecutive triangles so that the
// visible bits of a warp form one VT word):
//   transform (pinned fp32) -> trivial reject when all three vertices are outside
//   one side plane or behind the near plane -> Sutherland-Hodgman against the
//   near plane and the guard band |x|,|y| <= 64 w, only when a vertex is outside
//   -> project, snap to 1/256 px (round half even) -> fan sub-triangles -> cull
//   A <= 0 -> pixel-centre samples with the top-left rule -> z/w interpolated by
//   ((E0 z0 + E1 z1) + E2 z2) * (1/A), kept when -1 <= d <= 1.
// Sub-triangles whose clamped pixel box has more than kSmallMaxPix pixels are
// queued (pass 0) and rasterized by a warp per 16x16 tile in a second kernel.
//
// Kernels: k_raster_front (the per-triangle front end above; it also clears the
// per-frame state for the kernels after it), k_raster_exact (the exact set-up of
// the survivors; small sub-triangles rasterized in-thread, or by a group of 16
// lanes each when the survivors are few for the grid), k_raster_depth_big (the larger
// ones) and k_raster_mark (the visible bits; it also lists the 1024-triangle tiles
// that hold a visible triangle for the chart passes).  Two forms of the last three:
// "winners" (the default; below), where the depth pass keeps each pixel's triangle (with
// conservative marking k_raster_mark_cons then tests what the samples left unmarked),
// and two rasterizations (the tile-depth option), where the exact pass keeps a 48-byte
// record of each small sub-triangle and the marking pass rasterizes the queued tiles and
// the records again.  Edge values that stay below 2^24
// over a box are there stepped as exact fp32 integers.
#pragma once
#include "fa_internal.cuh"

namespace fa {
namespace rs {
namespace {

struct CV {
  float x, y, z, w;
};

struct SV {
  int64_t X, Y;
  float zn;
};

__device__ __forceinline__ float plane_dist(const CV& c, int pl) {
  switch (pl) {
    case 0: return __fadd_rn(c.z, c.w);
    case 1: return __fsub_rn(__fmul_rn(kGuard, c.w), c.x);
    case 2: return __fadd_rn(__fmul_rn(kGuard, c.w), c.x);
    case 3: return __fsub_rn(__fmul_rn(kGuard, c.w), c.y);
    default: return __fadd_rn(__fmul_rn(kGuard, c.w), c.y);
  }
}

__device__ __forceinline__ CV intersect(const CV& a, const CV& b, float da, float db) {
  float t = __fdiv_rn(da, __fsub_rn(da, db));
  CV r;
  r.x = __fadd_rn(a.x, __fmul_rn(t, __fsub_rn(b.x, a.x)));
  r.y = __fadd_rn(a.y, __fmul_rn(t, __fsub_rn(b.y, a.y)));
  r.z = __fadd_rn(a.z, __fmul_rn(t, __fsub_rn(b.z, a.z)));
  r.w = __fadd_rn(a.w, __fmul_rn(t, __fsub_rn(b.w, a.w)));
  return r;
}

constexpr int kMaxPoly = 16;

// Full Sutherland-Hodgman sequence (near, then the four guard planes).  A convex
// triangle gains at most one vertex per plane (<= 8); rounding on nearly
// plane-aligned input could add more, so the buffer holds kMaxPoly and an overflow
// is reported (returns -1) instead of being truncated.
__device__ __forceinline__ int clip_polygon(CV* poly, int n) {
  CV tmp[kMaxPoly];
  for (int pl = 0; pl < 5 && n >= 3; ++pl) {
    int m = 0;
    for (int i = 0; i < n; ++i) {
      const CV c = poly[i];
      const CV nx = poly[(i + 1) % n];
      float dc = plane_dist(c, pl), dn = plane_dist(nx, pl);
      bool ic = dc >= 0.0f, in_ = dn >= 0.0f;
      if (m + 2 > kMaxPoly) return -1;
      if (ic) tmp[m++] = c;
      if (ic != in_) tmp[m++] = ic ? intersect(c, nx, dc, dn) : intersect(nx, c, dn, dc);
    }
    for (int i = 0; i < m; ++i) poly[i] = tmp[i];
    n = m;
  }
  return n;
}

__device__ __forceinline__ SV project(const CV& c, float hx, float hy) {
  float nx = __fdiv_rn(c.x, c.w), ny = __fdiv_rn(c.y, c.w), zn = __fdiv_rn(c.z, c.w);
  float xs = __fmul_rn(__fadd_rn(nx, 1.0f), hx);
  float ys = __fmul_rn(__fadd_rn(ny, 1.0f), hy);
  SV s;
  // |xs * 256| < 2^28 inside the guard band |x|, |y| <= 64 w, so the rounded value
  // fits an int32 (and the 32-bit conversion avoids the fp64 units)
  s.X = __float2int_rn(__fmul_rn(xs, 256.0f));
  s.Y = __float2int_rn(__fmul_rn(ys, 256.0f));
  s.zn = zn;
  return s;
}


// Setup of one sub-triangle: area, 1/A, clamped pixel box.
struct Setup {
  int64_t A;
  int px0, py0, px1, py1;
};

__device__ __forceinline__ Setup setup(const SV& a, const SV& b, const SV& c, int W, int H, bool cons) {
  Setup s;
  s.A = (b.X - a.X) * (c.Y - a.Y) - (c.X - a.X) * (b.Y - a.Y);
  int64_t xmn = min(a.X, min(b.X, c.X)), xmx = max(a.X, max(b.X, c.X));
  int64_t ymn = min(a.Y, min(b.Y, c.Y)), ymx = max(a.Y, max(b.Y, c.Y));
  // sample rule: first / last pixel whose centre 256 p + 128 lies in [min, max];
  // conservative marking: first / last pixel whose square [256 p, 256 p + 256] meets it
  int64_t px0 = -((128 - xmn) >> 8), px1 = (xmx - 128) >> 8;
  int64_t py0 = -((128 - ymn) >> 8), py1 = (ymx - 128) >> 8;
  if (cons) {
    px0 = -((-xmn) >> 8) - 1;
    px1 = xmx >> 8;
    py0 = -((-ymn) >> 8) - 1;
    py1 = ymx >> 8;
  }
  s.px0 = (int)(px0 > 0 ? px0 : 0);
  s.py0 = (int)(py0 > 0 ? py0 : 0);
  s.px1 = (int)(px1 < W - 1 ? px1 : W - 1);
  s.py1 = (int)(py1 < H - 1 ? py1 : H - 1);
  return s;
}

// Edge functions of a sub-triangle at the sample of pixel (px, py) and their steps
// per pixel in x and y (exact int64; E is affine in the sample position).
struct Edges {
  int64_t e[3];   // E0 (edge b->c), E1 (c->a), E2 (a->b) at the sample
  int64_t dx[3];  // change per +1 pixel in x
  int64_t dy[3];  // change per +1 pixel in y
  bool tl[3];
};

__device__ __forceinline__ Edges edges_at(const SV& a, const SV& b, const SV& c, int px, int py) {
  Edges E;
  const int64_t sx = (int64_t)px * 256 + 128, sy = (int64_t)py * 256 + 128;
  const SV* v0[3] = {&b, &c, &a};
  const SV* v1[3] = {&c, &a, &b};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int64_t ex = v1[i]->X - v0[i]->X, ey = v1[i]->Y - v0[i]->Y;
    E.e[i] = ex * (sy - v0[i]->Y) - ey * (sx - v0[i]->X);
    E.dx[i] = -ey * 256;
    E.dy[i] = ex * 256;
    E.tl[i] = ey < 0 || (ey == 0 && ex < 0);
  }
  return E;
}

// Test and shade one pixel with edge values e at its sample.  PASS 0: covered (top-
// left rule) with a depth in [-1, 1]: atomicMin the depth key.  PASS 1: the same
// test, return key <= zbuf.  PASS 2 (conservative marking, App. A): the pixel's
// closed square meets the closed triangle (each edge function is >= 0 at the
// square corner where it is largest: e + (|dx| + |dy|) / 2, a half pixel each way);
// the depth is the sample's where the sample rule covers the centre, else the plane
// at the centre clamped to [zmin, zmax]; return key <= zbuf when it is in [-1, 1].
template <int PASS>
__device__ __forceinline__ bool sample(const Edges& E, const int64_t* e, const SV& a, const SV& b, const SV& c,
                                       float invA, uint32_t* __restrict__ z, float zmin = 0.0f,
                                       float zmax = 0.0f) {
  const bool in = (e[0] > 0 || (e[0] == 0 && E.tl[0])) && (e[1] > 0 || (e[1] == 0 && E.tl[1])) &&
                  (e[2] > 0 || (e[2] == 0 && E.tl[2]));
  if (PASS == 2) {
    bool meets = true;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int64_t ax = E.dx[i] < 0 ? -E.dx[i] : E.dx[i], ay = E.dy[i] < 0 ? -E.dy[i] : E.dy[i];
      meets = meets && (e[i] + ((ax + ay) >> 1) >= 0);
    }
    if (!meets) return false;
  } else if (!in) {
    return false;
  }
  float s = __fmul_rn(ll2float_rn(e[0]), a.zn);
  s = __fadd_rn(s, __fmul_rn(ll2float_rn(e[1]), b.zn));
  s = __fadd_rn(s, __fmul_rn(ll2float_rn(e[2]), c.zn));
  float d = __fmul_rn(s, invA);
  if (PASS == 2 && !in) d = fminf(fmaxf(d, zmin), zmax);
  if (!(d >= -1.0f && d <= 1.0f)) return false;
  const uint32_t key = ordered(d);
  if (PASS == 0) {
    atomicMin(z, key);  // result unused: a fire-and-forget reduction
    return false;
  }
  return key <= __ldcg(z);
}

// Visit the samples of a sub-triangle over pixel rect [px0..px1] x [py0..py1],
// stepping the edge functions.  PASS 1 returns true at the first visible sample.
// sample() on edge values held exactly as floats (integers below 2^24), PASS 0 or 1.
template <int PASS>
__device__ __forceinline__ bool sample_f(float e0, float e1, float e2, const bool* tl, float z0, float z1,
                                         float z2, float invA, uint32_t* __restrict__ z) {
  const bool in = (e0 > 0.0f || (e0 == 0.0f && tl[0])) && (e1 > 0.0f || (e1 == 0.0f && tl[1])) &&
                  (e2 > 0.0f || (e2 == 0.0f && tl[2]));
  if (!in) return false;
  float s = __fmul_rn(e0, z0);
  s = __fadd_rn(s, __fmul_rn(e1, z1));
  s = __fadd_rn(s, __fmul_rn(e2, z2));
  const float d = __fmul_rn(s, invA);
  if (!(d >= -1.0f && d <= 1.0f)) return false;
  const uint32_t key = ordered(d);
  if (PASS == 0) {
    atomicMin(z, key);  // result unused: a fire-and-forget reduction
    return false;
  }
  return key <= __ldcg(z);
}

// raster_rect for boxes whose edge values all stay below 2^24 in magnitude (checked
// by the caller): those integers are exact in fp32, so the edge functions are kept
// and stepped as floats (every sum is again such an integer, hence exact), the
// coverage tests compare the same values and the depth multiplies the same
// correctly rounded conversions as sample() does: the same samples and keys, with
// no 64-bit arithmetic or conversion per sample.  PASS 0 or 1.
template <int PASS>
__device__ __forceinline__ bool raster_rect_f32(const Edges& E, const SV& a, const SV& b, const SV& c, float invA,
                                                int px0, int py0, int px1, int py1, uint32_t* __restrict__ zbuf,
                                                int W) {
  float er[3], fdx[3], fdy[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    er[i] = (float)(int32_t)E.e[i];
    fdx[i] = (float)(int32_t)E.dx[i];
    fdy[i] = (float)(int32_t)E.dy[i];
  }
  bool vis = false;  // PASS 1 stops at the first sample that passes the depth test
  for (int py = py0; py <= py1; ++py) {
    float e0 = er[0], e1 = er[1], e2 = er[2];
    uint32_t* zrow = zbuf + (size_t)py * W;
#pragma unroll 2
    for (int px = px0; px <= px1; ++px) {
      vis |= sample_f<PASS>(e0, e1, e2, E.tl, a.zn, b.zn, c.zn, invA, zrow + px);
      if (PASS == 1 && vis) break;
      e0 = __fadd_rn(e0, fdx[0]);
      e1 = __fadd_rn(e1, fdx[1]);
      e2 = __fadd_rn(e2, fdx[2]);
    }
    if (PASS == 1 && vis) break;
    er[0] = __fadd_rn(er[0], fdy[0]);
    er[1] = __fadd_rn(er[1], fdy[1]);
    er[2] = __fadd_rn(er[2], fdy[2]);
  }
  return vis;
}

template <int PASS>
__device__ bool raster_rect(const SV& a, const SV& b, const SV& c, float invA, int px0, int py0,
                            int px1, int py1, uint32_t* __restrict__ zbuf, int W) {
  const Edges E = edges_at(a, b, c, px0, py0);
  if (PASS != 2 && px1 >= px0 && py1 >= py0) {
    // |E| over the box <= |E(px0, py0)| + |dx| (px1 - px0) + |dy| (py1 - py0)
    bool small = true;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int64_t ax = E.dx[i] < 0 ? -E.dx[i] : E.dx[i], ay = E.dy[i] < 0 ? -E.dy[i] : E.dy[i];
      const int64_t ae = E.e[i] < 0 ? -E.e[i] : E.e[i];
      small = small && ax < (1ll << 24) && ay < (1ll << 24) &&
              ae + ax * (int64_t)(px1 - px0) + ay * (int64_t)(py1 - py0) < (1ll << 24);
    }
    if (small) return raster_rect_f32<PASS>(E, a, b, c, invA, px0, py0, px1, py1, zbuf, W);
  }
  const float zmin = fminf(a.zn, fminf(b.zn, c.zn)), zmax = fmaxf(a.zn, fmaxf(b.zn, c.zn));
  int64_t er[3] = {E.e[0], E.e[1], E.e[2]};
  bool vis = false;  // PASS 1: no early exit, so the depth loads can overlap
  for (int py = py0; py <= py1; ++py) {
    int64_t e[3] = {er[0], er[1], er[2]};
    uint32_t* zrow = zbuf + (size_t)py * W;
#pragma unroll 2
    for (int px = px0; px <= px1; ++px) {
      vis |= sample<PASS>(E, e, a, b, c, invA, zrow + px, zmin, zmax);
      e[0] += E.dx[0];
      e[1] += E.dx[1];
      e[2] += E.dx[2];
    }
    er[0] += E.dy[0];
    er[1] += E.dy[1];
    er[2] += E.dy[2];
  }
  return vis;
}

// One small sub-triangle that passed the depth pre-pass set-up: its snapped
// vertices, depths and clamped pixel box, kept so that the marking pass does not
// redo the set-up.  48 bytes: {X0, Y0, X1, Y1}, {X2, Y2, px0 | py0 << 16,
// px1 | py1 << 16}, {z0, z1, z2, triangle}.
struct CandTri {
  int4 a;
  int4 b;
  float4 c;
};
static_assert(sizeof(CandTri) == 48, "CandTri is 48 bytes");

constexpr int kFrontThreads = 512;

struct RasterArgs {
  Mat4 M;
  int cons;  // conservative marking (FA_VIS_CONSERVATIVE): conservative pixel boxes
  const float* Mdev;  // when set, the matrix is read here on the device instead of M
  const float* pos;
  const uint32_t* idx;
  uint32_t T;
  int W, H;
  float hx, hy;
  uint32_t* zbuf;
  BigTri* queue;
  uint32_t queue_cap;
  uint32_t* tile_owner;  // queue record of each reserved tile
  uint32_t tile_cap;
  CandTri* cand;
  uint32_t cand_cap;
  uint32_t* surv;  // triangles that need the exact set-up, one region per front block
  uint32_t* surv_count;  // [front_blocks] survivors per region
  uint32_t surv_per_block;
  uint32_t front_blocks;
  uint32_t clip_base;  // first candidate slot of the clipped path
  float4* surv_clip;  // [T][3] their clip coordinates
  uint32_t* tile_flag;  // per 1024-triangle tile: listed in tile_list
  uint32_t* tile_list;
  uint32_t* clip_count;  // [front_blocks] clipped triangles per region of `clip`
  uint32_t* blockcnt;    // per-tile counts of the chart passes (cleared here)
  uint32_t* viscnt;
  uint32_t ntiles;
  int reset_status;      // the front end clears the device status word first
  int32_t* tri_chart;    // when set, the front end sets it to -1 (the chart pass writes visible ones)
  uint32_t* partial_clear;  // when set, the front end also clears these ceil(T/32) words
  uint32_t mid_max_pix;     // boxes up to this size may be rasterized in-thread (<= kSmallMaxPix: off)
  uint32_t* zmax;           // [ztx * ceil(H / 16)] largest depth key of each 16x16 pixel tile, or
                            // null: no tile-depth pass (FA_RASTER_HIZ off)
  int ztx;                  // tiles per row, ceil(W / 16)
  uint32_t* clip;  // triangles that need clipping, one region per front block like surv
  DevCounters* ctr;
  uint32_t* vt;
  // single-pass visibility (see "winners" below): the depth buffer holds key << 32 | triangle
  int win;
  unsigned long long* zid;  // [W * H], the same memory as zbuf
  uint4* ties;              // [kTies] (pixel, key, triangle, triangle) of equal keys
  uint32_t mid_blocks, mid_lists, mid_per_block;  // exact pass's blocks, mid-size lists, slots per block
};

__device__ __forceinline__ CandTri make_cand(const SV& a, const SV& b, const SV& c, const Setup& s, uint32_t t) {
  CandTri r;
  r.a = make_int4((int)a.X, (int)a.Y, (int)b.X, (int)b.Y);
  r.b = make_int4((int)c.X, (int)c.Y, s.px0 | (s.py0 << 16), s.px1 | (s.py1 << 16));
  r.c = make_float4(a.zn, b.zn, c.zn, __uint_as_float(t));
  return r;
}

__device__ __forceinline__ void store_cand(const RasterArgs& A, uint32_t slot, const CandTri& r) {
  if (slot < A.cand_cap) {
    float4* d = reinterpret_cast<float4*>(A.cand + slot);
    d[0] = make_float4(__int_as_float(r.a.x), __int_as_float(r.a.y), __int_as_float(r.a.z), __int_as_float(r.a.w));
    d[1] = make_float4(__int_as_float(r.b.x), __int_as_float(r.b.y), __int_as_float(r.b.z), __int_as_float(r.b.w));
    d[2] = r.c;
  } else {
    set_status(A.ctr, FA_E_CAPACITY);
  }
}

// Depth pre-pass of the fan (sv[0], sv[i], sv[i+1]) of one mesh triangle t.  Large
// sub-triangles go to the tile queue; small ones are rasterized here and, when
// `out` is given and the fan has a single sub-triangle, returned for the candidate
// list (otherwise appended one by one).  Returns the number of records in `out`.
__device__ int depth_fan(const RasterArgs& A, uint32_t t, const SV* sv, int n, CandTri* out) {
  int nq = 0;
  uint64_t tiles = 0;
  bool big = false;
  for (int i = 1; i + 1 < n; ++i) {
    Setup s = setup(sv[0], sv[i], sv[i + 1], A.W, A.H, A.cons);
    if (s.A <= 0 || s.px1 < s.px0 || s.py1 < s.py0) continue;
    int w = s.px1 - s.px0 + 1, h = s.py1 - s.py0 + 1;
    if (w * h > kSmallMaxPix) big = true;
    ++nq;
    tiles += (uint64_t)((w + kBigTile - 1) / kBigTile) * (uint64_t)((h + kBigTile - 1) / kBigTile);
  }
  if (nq == 0) return 0;
  if (big) {
    unsigned long long old = atomicAdd(&A.ctr->big, ((unsigned long long)nq << 40) | (unsigned long long)tiles);
    uint64_t e0 = old >> 40, tile = old & ((1ull << 40) - 1);
    if (e0 + nq <= A.queue_cap && tile + tiles <= A.tile_cap) {
      int q = 0;
      for (int i = 1; i + 1 < n; ++i) {
        Setup s = setup(sv[0], sv[i], sv[i + 1], A.W, A.H, A.cons);
        if (s.A <= 0 || s.px1 < s.px0 || s.py1 < s.py0) continue;
        BigTri bt;
        bt.X[0] = (int32_t)sv[0].X; bt.X[1] = (int32_t)sv[i].X; bt.X[2] = (int32_t)sv[i + 1].X;
        bt.Y[0] = (int32_t)sv[0].Y; bt.Y[1] = (int32_t)sv[i].Y; bt.Y[2] = (int32_t)sv[i + 1].Y;
        bt.zn[0] = sv[0].zn; bt.zn[1] = sv[i].zn; bt.zn[2] = sv[i + 1].zn;
        bt.px0 = s.px0; bt.py0 = s.py0; bt.px1 = s.px1; bt.py1 = s.py1;
        bt.tri = t;
        bt.tile0 = (uint32_t)tile;
        bt.pad = 0;
        A.queue[e0 + q] = bt;
        const int w = s.px1 - s.px0 + 1, h = s.py1 - s.py0 + 1;
        const uint64_t nt = (uint64_t)((w + kBigTile - 1) / kBigTile) * (uint64_t)((h + kBigTile - 1) / kBigTile);
        for (uint64_t j = 0; j < nt; ++j) A.tile_owner[tile + j] = (uint32_t)(e0 + q);
        tile += nt;
        ++q;
      }
      return 0;
    }
    // queue or tile table full: the reserved records become empty, the reserved
    // tiles get no owner, and the sub-triangles are handled here instead
    for (uint64_t e = e0; e < e0 + nq && e < A.queue_cap; ++e) {
      BigTri bt = {};
      bt.px0 = 1; bt.px1 = 0; bt.py0 = 1; bt.py1 = 0;
      bt.tile0 = (uint32_t)tile;
      A.queue[e] = bt;
    }
    for (uint64_t j = tile; j < tile + tiles && j < A.tile_cap; ++j) A.tile_owner[j] = 0xFFFFFFFFu;
  }
  int nout = 0;
  for (int i = 1; i + 1 < n; ++i) {
    Setup s = setup(sv[0], sv[i], sv[i + 1], A.W, A.H, A.cons);
    if (s.A <= 0 || s.px1 < s.px0 || s.py1 < s.py0) continue;
    float invA = __fdiv_rn(1.0f, ll2float_rn(s.A));
    raster_rect<0>(sv[0], sv[i], sv[i + 1], invA, s.px0, s.py0, s.px1, s.py1, A.zbuf, A.W);
    const CandTri r = make_cand(sv[0], sv[i], sv[i + 1], s, t);
    if (out && nq == 1) {
      *out = r;
      nout = 1;
    } else {
      store_cand(A, A.clip_base + atomicAdd(&A.ctr->ncand, 1u), r);
    }
  }
  return nout;
}

// Triangles that cross the near plane or the guard band (rare): clip first.
__device__ __noinline__ void depth_clipped(const RasterArgs& A, uint32_t t, float4 c0, float4 c1, float4 c2) {
  CV poly[kMaxPoly];
  poly[0] = CV{c0.x, c0.y, c0.z, c0.w};
  poly[1] = CV{c1.x, c1.y, c1.z, c1.w};
  poly[2] = CV{c2.x, c2.y, c2.z, c2.w};
  int n = clip_polygon(poly, 3);
  if (n < 0) {
    set_status(A.ctr, FA_E_CAPACITY);
    return;
  }
  if (n < 3) return;
  for (int i = 0; i < n; ++i)
    if (!(poly[i].w > 0.0f)) return;
  SV sv[kMaxPoly];
  for (int i = 0; i < n; ++i) sv[i] = project(poly[i], A.hx, A.hy);
  depth_fan(A, t, sv, n, nullptr);
}

// Conservative test on approximate screen positions (correctly rounded 1/w, then
// the same screen mapping): true when the triangle surely covers no sample or is
// surely back-facing.  m bounds, per axis, the distance between the approximate
// position and the exact snapped vertex: 1/512 px of snapping plus
// (|ndc| + 1) * (size / 2) * 2^-20 for the different rounding of x * (1/w) and x / w
// followed by the same +1 and scale.  Both tests only drop triangles the exact path
// would drop, so results are unchanged.
__device__ __forceinline__ bool surely_empty(const RasterArgs& A, const float4& c0, const float4& c1, const float4& c2) {
  const float r0 = __frcp_rn(c0.w), r1 = __frcp_rn(c1.w), r2 = __frcp_rn(c2.w);
  const float nx0 = c0.x * r0, nx1 = c1.x * r1, nx2 = c2.x * r2;
  const float ny0 = c0.y * r0, ny1 = c1.y * r1, ny2 = c2.y * r2;
  const float x0 = (nx0 + 1.0f) * A.hx, x1 = (nx1 + 1.0f) * A.hx, x2 = (nx2 + 1.0f) * A.hx;
  const float y0 = (ny0 + 1.0f) * A.hy, y1 = (ny1 + 1.0f) * A.hy, y2 = (ny2 + 1.0f) * A.hy;
  const float ax = fmaxf(fabsf(nx0), fmaxf(fabsf(nx1), fabsf(nx2))) + 1.0f;
  const float ay = fmaxf(fabsf(ny0), fmaxf(fabsf(ny1), fabsf(ny2))) + 1.0f;
  const float mx = 0.001953125f + ax * A.hx * 9.5367431640625e-7f + 1e-6f;
  const float my = 0.001953125f + ay * A.hy * 9.5367431640625e-7f + 1e-6f;
  // pixel centres p + 0.5 inside the widened box, clamped to the viewport
  const float lo_x = fminf(x0, fminf(x1, x2)) - mx, hi_x = fmaxf(x0, fmaxf(x1, x2)) + mx;
  const float lo_y = fminf(y0, fminf(y1, y2)) - my, hi_y = fmaxf(y0, fmaxf(y1, y2)) + my;
  // (conservative marking: pixels whose squares meet the widened box)
  const float px0 = fmaxf(A.cons ? ceilf(lo_x) - 1.0f : ceilf(lo_x - 0.5f), 0.0f);
  const float px1 = fminf(A.cons ? floorf(hi_x) : floorf(hi_x - 0.5f), (float)(A.W - 1));
  const float py0 = fmaxf(A.cons ? ceilf(lo_y) - 1.0f : ceilf(lo_y - 0.5f), 0.0f);
  const float py1 = fminf(A.cons ? floorf(hi_y) : floorf(hi_y - 0.5f), (float)(A.H - 1));
  if (px0 > px1 || py0 > py1) return true;
  // signed doubled area in px^2 against its error bound
  const float e1x = x1 - x0, e1y = y1 - y0, e2x = x2 - x0, e2y = y2 - y0;
  const float p1 = e1x * e2y, p2 = e1y * e2x;
  const float area = p1 - p2;
  const float m = fmaxf(mx, my);
  const float bound = 2.0f * m * (fabsf(e1x) + fabsf(e1y) + fabsf(e2x) + fabsf(e2y)) + 24.0f * m * m +
                      2.384185791015625e-7f * (fabsf(p1) + fabsf(p2)) + 1e-6f;
  return area < -bound;
}

// Front end of the depth pre-pass for one mesh triangle: transform, trivial reject,
// route to the clipped list, conservative reject.  Returns 1 when the triangle needs
// the exact set-up (unclipped; its clip coordinates are left in c[3]), 2 when it must
// be clipped first, 0 when dropped.
struct TriPos {
  float p[9];  // the three corners' world positions
};

__device__ __forceinline__ uint3 load_tri(const uint32_t* __restrict__ idx, uint32_t t) {
  const uint32_t* f = idx + 3 * (size_t)t;
  return make_uint3(__ldg(f), __ldg(f + 1), __ldg(f + 2));
}

__device__ __forceinline__ TriPos load_pos(const float* __restrict__ pos, uint3 i) {
  TriPos q;
  const uint32_t v[3] = {i.x, i.y, i.z};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float* p = pos + 3 * (size_t)v[k];
    q.p[3 * k] = __ldg(p);
    q.p[3 * k + 1] = __ldg(p + 1);
    q.p[3 * k + 2] = __ldg(p + 2);
  }
  return q;
}

__device__ __forceinline__ int front_triangle(const RasterArgs& A, const Mat4& M, const TriPos& q, float4* c) {
  const float4 c0 = transform(M, q.p[0], q.p[1], q.p[2]), c1 = transform(M, q.p[3], q.p[4], q.p[5]),
               c2 = transform(M, q.p[6], q.p[7], q.p[8]);
  // trivial reject: all vertices outside one side plane, or all behind the near plane
  // (no sample can be covered then: see the design notes on exactness)
  if ((c0.x > c0.w && c1.x > c1.w && c2.x > c2.w) || (c0.x < -c0.w && c1.x < -c1.w && c2.x < -c2.w) ||
      (c0.y > c0.w && c1.y > c1.w && c2.y > c2.w) || (c0.y < -c0.w && c1.y < -c1.w && c2.y < -c2.w) ||
      (__fadd_rn(c0.z, c0.w) < 0.0f && __fadd_rn(c1.z, c1.w) < 0.0f && __fadd_rn(c2.z, c2.w) < 0.0f))
    return 0;
  const CV v0{c0.x, c0.y, c0.z, c0.w}, v1{c1.x, c1.y, c1.z, c1.w}, v2{c2.x, c2.y, c2.z, c2.w};
  bool outside = false;
#pragma unroll
  for (int pl = 0; pl < 5; ++pl)
    outside |= !(plane_dist(v0, pl) >= 0.0f) || !(plane_dist(v1, pl) >= 0.0f) || !(plane_dist(v2, pl) >= 0.0f);
  if (outside) return 2;
  if (!(v0.w > 0.0f) || !(v1.w > 0.0f) || !(v2.w > 0.0f)) return 0;
  if (surely_empty(A, c0, c1, c2)) return 0;
  c[0] = c0;
  c[1] = c1;
  c[2] = c2;
  return 1;
}

// Snapped vertices and set-up of an unclipped triangle from its clip coordinates,
// all in registers (the fan of an unclipped triangle is the triangle itself).
struct Exact {
  SV a, b, c;
  Setup s;
};

__device__ __forceinline__ Exact exact_setup(const RasterArgs& A, const float4& c0, const float4& c1,
                                             const float4& c2) {
  Exact E;
  E.a = project(CV{c0.x, c0.y, c0.z, c0.w}, A.hx, A.hy);
  E.b = project(CV{c1.x, c1.y, c1.z, c1.w}, A.hx, A.hy);
  E.c = project(CV{c2.x, c2.y, c2.z, c2.w}, A.hx, A.hy);
  E.s = setup(E.a, E.b, E.c, A.W, A.H, A.cons);
  return E;
}

// Depth pre-pass, front end: one thread per triangle; survivors go to a compact list
// (warp-aggregated appends) so that the exact set-up runs on full warps.
// Also clears, for the kernels after it, the depth buffer, VT, the counters and the
// per-tile flags and counts of the visible-tile list (none of which it reads).
template <bool DEV_M>
__device__ __forceinline__ void front_body(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  const Mat4 M = DEV_M ? load_mat(A.Mdev) : A.M;
  __shared__ uint32_t s_count, s_nclip;
  if (threadIdx.x == 0) {
    s_count = 0;
    s_nclip = 0;
    if (bid == 0) {
      if (A.reset_status) A.ctr->status = 0;
      A.ctr->big = 0ull;
      A.ctr->ncand = 0u;
      A.ctr->n_vtiles = 0u;
      A.ctr->uf_item = 0u;
      A.ctr->n_ties = 0u;
      A.ctr->cons_item = 0u;
    }
  }
  if (bid == 0 && threadIdx.x < kMidLists) A.ctr->n_mid[threadIdx.x][0] = 0u;
  {
    const uint32_t gstride = nblk * blockDim.x, g0 = bid * blockDim.x + threadIdx.x;
    const uint32_t npix = ((uint32_t)A.W * (uint32_t)A.H) << (A.win ? 1 : 0);  // 32-bit words of the depth buffer
    const uint32_t n4 = npix / 4, nwords = (A.T + 31) / 32;
    uint4* z4 = reinterpret_cast<uint4*>(A.zbuf);
    const uint4 ff = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
    for (uint32_t i = g0; i < n4; i += gstride) z4[i] = ff;
    for (uint32_t i = n4 * 4 + g0; i < npix; i += gstride) A.zbuf[i] = 0xFFFFFFFFu;
    for (uint32_t i = g0; i < nwords; i += gstride) A.vt[i] = 0u;
    for (uint32_t i = g0; i < A.ntiles; i += gstride) {
      A.tile_flag[i] = 0u;
      A.blockcnt[i] = 0u;
      A.viscnt[i] = 0u;
    }
    if (A.partial_clear)
      for (uint32_t i = g0; i < nwords; i += gstride) A.partial_clear[i] = 0u;
    if (A.tri_chart) {
      int4* t4 = reinterpret_cast<int4*>(A.tri_chart);
      for (uint32_t i = g0; i < A.T / 4; i += gstride) t4[i] = make_int4(-1, -1, -1, -1);
      for (uint32_t i = (A.T / 4) * 4 + g0; i < A.T; i += gstride) A.tri_chart[i] = -1;
    }
  }
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31;
  // block b owns survivor slots [b * surv_per_block, (b + 1) * surv_per_block): it sees
  // at most that many triangles, so its region cannot overflow
  const uint32_t region = bid * A.surv_per_block;
  // software pipeline over this thread's triangles t, t + stride, ...: the indices
  // are loaded two iterations ahead and the corner positions one iteration ahead, so
  // that each iteration waits on no dependent load of its own
  const uint32_t stride = nblk * blockDim.x;
  const uint32_t t0 = bid * blockDim.x + threadIdx.x;
  uint3 idx1 = t0 + stride < A.T ? load_tri(A.idx, t0 + stride) : make_uint3(0u, 0u, 0u);
  TriPos pos0 = load_pos(A.pos, t0 < A.T ? load_tri(A.idx, t0) : make_uint3(0u, 0u, 0u));
  for (uint32_t base = bid * blockDim.x; base < A.T; base += stride) {
    const uint32_t t = base + threadIdx.x;
    const TriPos cur = pos0;
    pos0 = load_pos(A.pos, idx1);
    idx1 = t + 2u * stride < A.T ? load_tri(A.idx, t + 2u * stride) : make_uint3(0u, 0u, 0u);
    float4 c[3];
    const int r = t < A.T ? front_triangle(A, M, cur, c) : 0;
    const uint32_t b1 = __ballot_sync(0xFFFFFFFFu, r == 1), b2 = __ballot_sync(0xFFFFFFFFu, r == 2);
    if (b1) {
      uint32_t o = 0;
      if (lane == 0) o = atomicAdd(&s_count, (uint32_t)__popc(b1));
      o = __shfl_sync(0xFFFFFFFFu, o, 0);
      if (r == 1) {
        const uint32_t slot = region + o + __popc(b1 & ((1u << lane) - 1u));
        A.surv[slot] = t;
        float4* sc = A.surv_clip + 3 * (size_t)slot;
        sc[0] = c[0];
        sc[1] = c[1];
        sc[2] = c[2];
      }
    }
    if (b2) {  // rare: the block's clipped region, like the survivors'
      uint32_t o = 0;
      if (lane == 0) o = atomicAdd(&s_nclip, (uint32_t)__popc(b2));
      o = __shfl_sync(0xFFFFFFFFu, o, 0);
      if (r == 2) A.clip[region + o + __popc(b2 & ((1u << lane) - 1u))] = t;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    A.surv_count[bid] = s_count;
    A.clip_count[bid] = s_nclip;
  }
}

// The shared words of region_prefix, one array for all bodies of a kernel.
__device__ __forceinline__ uint32_t* region_pre() {
  __shared__ uint32_t pre[kMaxFrontBlocks + 1];
  return pre;
}

// Exclusive prefix of the front blocks' per-region counts (survivors or clipped
// triangles) into shared memory (front_blocks <= kMaxFrontBlocks); returns the
// total.  Called by every thread of a block of exactly NT threads.
template <int NT>
__device__ uint32_t region_prefix(const RasterArgs& A, const uint32_t* counts, uint32_t* pre) {
  constexpr uint32_t kPer = (kMaxFrontBlocks + NT - 1) / NT;
  __shared__ uint32_t s_warp[NT / 32];
  const uint32_t nb = A.front_blocks, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t c[kPer], sum = 0;
#pragma unroll
  for (uint32_t j = 0; j < kPer; ++j) {
    const uint32_t b = threadIdx.x * kPer + j;
    c[j] = b < nb ? __ldcg(counts + b) : 0u;
    sum += c[j];
  }
  uint32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= (uint32_t)o) inc += y;
  }
  if (lane == 31) s_warp[w] = inc;
  __syncthreads();
  uint32_t wpre = 0, tot = 0;
#pragma unroll
  for (uint32_t k = 0; k < (uint32_t)(NT / 32); ++k) {
    const uint32_t x = s_warp[k];
    wpre += k < w ? x : 0u;
    tot += x;
  }
  uint32_t run = wpre + inc - sum;
#pragma unroll
  for (uint32_t j = 0; j < kPer; ++j) {
    const uint32_t b = threadIdx.x * kPer + j;
    if (b <= nb) pre[b] = run;
    run += c[j];
  }
  __syncthreads();
  return tot;
}
template <int NT>
__device__ __forceinline__ uint32_t surv_prefix(const RasterArgs& A, uint32_t* pre) {
  return region_prefix<NT>(A, A.surv_count, pre);
}

// Survivor slot of dense index v: block b with pre[b] <= v < pre[b + 1].
// Slot of dense index v in the front blocks' regions (survivors or clipped
// triangles, as pre was built): block b with pre[b] <= v < pre[b + 1].  vfirst <=
// v is the warp's first index, the same in every lane: its search reads the same
// shared words in all lanes (broadcasts), and a lane searches on its own only when
// v lies in a later region than vfirst.
__device__ __forceinline__ uint32_t surv_slot(const RasterArgs& A, const uint32_t* pre, uint32_t v,
                                              uint32_t vfirst) {
  uint32_t lo = 0, hi = A.front_blocks;  // pre[lo] <= vfirst < pre[hi]
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (pre[mid] <= vfirst) lo = mid;
    else hi = mid;
  }
  if (v >= pre[lo + 1]) {
    hi = A.front_blocks;
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (pre[mid] <= v) lo = mid;
      else hi = mid;
    }
  }
  return lo * A.surv_per_block + (v - pre[lo]);
}

// The samples of one sub-triangle per group of kRasterGroup lanes: the group's
// leader (its first lane) holds the snapped vertices, area and pixel box, and `go`;
// every lane of the group takes the box's samples sub, sub + kRasterGroup, ...  PASS
// as in sample(): 0 writes the depth keys; 1 and 2 return whether a sample of the
// leader's sub-triangle passed the depth test (in every lane of the group).  All
// lanes of the warp call it.
constexpr uint32_t kRasterGroup = 16;
template <int PASS>
__device__ __forceinline__ bool group_raster(const SV& a0, const SV& b0, const SV& c0, int64_t A0, int qx0, int qy0,
                                             int qx1, int qy1, bool go0, uint32_t* __restrict__ zbuf, int W) {
  const uint32_t lane = threadIdx.x & 31, src = lane & ~(kRasterGroup - 1u), sub = lane - src;
  // every lane of the warp takes part in every shuffle (the groups' leaders differ in
  // `go`, so no shuffle may sit under it)
  const bool go = __shfl_sync(0xFFFFFFFFu, go0, src);
  const SV a{__shfl_sync(0xFFFFFFFFu, (int32_t)a0.X, src), __shfl_sync(0xFFFFFFFFu, (int32_t)a0.Y, src),
             __shfl_sync(0xFFFFFFFFu, a0.zn, src)};
  const SV b{__shfl_sync(0xFFFFFFFFu, (int32_t)b0.X, src), __shfl_sync(0xFFFFFFFFu, (int32_t)b0.Y, src),
             __shfl_sync(0xFFFFFFFFu, b0.zn, src)};
  const SV c{__shfl_sync(0xFFFFFFFFu, (int32_t)c0.X, src), __shfl_sync(0xFFFFFFFFu, (int32_t)c0.Y, src),
             __shfl_sync(0xFFFFFFFFu, c0.zn, src)};
  const int64_t Ar = (int64_t)(((uint64_t)__shfl_sync(0xFFFFFFFFu, (uint32_t)((uint64_t)A0 >> 32), src) << 32) |
                               (uint64_t)__shfl_sync(0xFFFFFFFFu, (uint32_t)A0, src));
  const int px0 = __shfl_sync(0xFFFFFFFFu, qx0, src), py0 = __shfl_sync(0xFFFFFFFFu, qy0, src);
  const int px1 = __shfl_sync(0xFFFFFFFFu, qx1, src), py1 = __shfl_sync(0xFFFFFFFFu, qy1, src);
  bool vis = false;
  if (go) {
    const float invA = __fdiv_rn(1.0f, ll2float_rn(Ar));
    const float zmin = fminf(a.zn, fminf(b.zn, c.zn)), zmax = fmaxf(a.zn, fmaxf(b.zn, c.zn));
    const int w = px1 - px0 + 1, npix = w * (py1 - py0 + 1);
    for (int s = (int)sub; s < npix; s += (int)kRasterGroup) {
      const int px = px0 + s % w, py = py0 + s / w;
      const Edges E = edges_at(a, b, c, px, py);
      vis |= sample<PASS>(E, E.e, a, b, c, invA, zbuf + (size_t)py * W + px, zmin, zmax);
    }
  }
  if (PASS == 0) return false;
  const uint32_t gmask = ((1u << kRasterGroup) - 1u) << src;
  return (__ballot_sync(0xFFFFFFFFu, vis) & gmask) != 0u;
}

// Depth pre-pass, exact part: survivors of the front end.  Survivor i writes its
// candidate record (or an empty marker) at slot i, so no counter is needed; clipped
// triangles append theirs after slot T.
template <bool DEV_M, int NT>
__device__ __forceinline__ void exact_body(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  uint32_t* pre = region_pre();
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t n = surv_prefix<NT>(A, pre);
  const uint32_t stride = nblk * blockDim.x;
  // Few survivors for the grid (a small frame): each gets a group of kRasterGroup
  // lanes, its leader doing the set-up and the group sharing the box's samples, so
  // that the grid's warps are not each waiting on one thread's sample loop.  The
  // same samples get the same keys either way.
  const bool grouped = (uint64_t)n * kRasterGroup <= (uint64_t)stride;
  const uint32_t sub = lane & (kRasterGroup - 1u);
  for (uint32_t wbase = bid * blockDim.x + (threadIdx.x & ~31u); (grouped ? wbase / kRasterGroup : wbase) < n;
       wbase += stride) {
    const uint32_t vfirst = grouped ? wbase / kRasterGroup : wbase;
    // (in a group only the leader sets up; the others take no survivor here)
    const uint32_t v = grouped ? (sub == 0u ? vfirst + lane / kRasterGroup : n) : wbase + lane;
    const uint32_t i = v < n ? surv_slot(A, pre, v, vfirst) : 0u;
    Exact E = {};
    uint32_t t = 0, tiles = 0;
    int kind = 0;  // 0 nothing, 1 small, 2 large
    bool mid = false;  // large, but at most kMidMaxPix pixels
    uint32_t mid_pix = 0, mid_cost = 0;
    if (v < n) {
      const float4* sc = A.surv_clip + 3 * (size_t)i;
      t = __ldcg(A.surv + i);
      E = exact_setup(A, __ldcs(sc), __ldcs(sc + 1), __ldcs(sc + 2));
      if (E.s.A > 0 && E.s.px1 >= E.s.px0 && E.s.py1 >= E.s.py0) {
        const int w = E.s.px1 - E.s.px0 + 1, h = E.s.py1 - E.s.py0 + 1;
        if (w * h > kSmallMaxPix) {
          kind = 2;
          tiles = (uint32_t)(((w + kBigTile - 1) / kBigTile) * ((h + kBigTile - 1) / kBigTile));
          mid = w * h <= (int)A.mid_max_pix;
          if (mid) {
            mid_pix = (uint32_t)(w * h);
            // the tile path: two rows per warp step in each 16-pixel-wide tile
            // column, plus the queue record and its set-up
            mid_cost = kMidStepCost * (uint32_t)((w + kBigTile - 1) / kBigTile) * (uint32_t)((h + 1) / 2) +
                       kMidTriCost;
          }
        } else {
          kind = 1;
        }
      }
    }
    // Mid-size boxes are rasterized in-thread when that is cheaper for the warp: the
    // in-thread loop lasts as long as the warp's largest box (the small boxes' 16
    // samples are paid anyway), the tile path costs each such triangle its tile
    // steps and its queue record.  Either way the same samples get the same keys.
    {
      const uint32_t smax = __reduce_max_sync(0xFFFFFFFFu, mid_pix);
      const uint32_t tsum = __reduce_add_sync(0xFFFFFFFFu, mid_cost);
      if (mid && (smax - (uint32_t)kSmallMaxPix) * kMidSampleCost < tsum) {
        kind = 1;
        tiles = 0;
      }
    }
    // large triangles of the warp reserve queue records and tiles with one atomic
    const uint32_t bigs = __ballot_sync(0xFFFFFFFFu, kind == 2);
    if (bigs) {
      uint32_t tpre = tiles;  // inclusive prefix of tiles over the warp
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, tpre, o);
        if (lane >= (unsigned)o) tpre += y;
      }
      const uint32_t ttot = __shfl_sync(0xFFFFFFFFu, tpre, 31);
      unsigned long long old = 0;
      if (lane == 0)
        old = atomicAdd(&A.ctr->big, ((unsigned long long)__popc(bigs) << 40) | (unsigned long long)ttot);
      old = __shfl_sync(0xFFFFFFFFu, old, 0);
      if (kind == 2) {
        const uint64_t e = (old >> 40) + __popc(bigs & ((1u << lane) - 1u));
        const uint64_t tile = (old & ((1ull << 40) - 1)) + (tpre - tiles);
        if (e < A.queue_cap && tile + tiles <= A.tile_cap) {
          BigTri bt;
          bt.X[0] = (int32_t)E.a.X; bt.X[1] = (int32_t)E.b.X; bt.X[2] = (int32_t)E.c.X;
          bt.Y[0] = (int32_t)E.a.Y; bt.Y[1] = (int32_t)E.b.Y; bt.Y[2] = (int32_t)E.c.Y;
          bt.zn[0] = E.a.zn; bt.zn[1] = E.b.zn; bt.zn[2] = E.c.zn;
          bt.px0 = E.s.px0; bt.py0 = E.s.py0; bt.px1 = E.s.px1; bt.py1 = E.s.py1;
          bt.tri = t;
          bt.tile0 = (uint32_t)tile;
          bt.pad = 0;
          A.queue[e] = bt;
          for (uint32_t j = 0; j < tiles; ++j) A.tile_owner[tile + j] = (uint32_t)e;
          kind = 0;
        } else {
          // queue or tile table full: empty record, no owners, rasterized here
          if (e < A.queue_cap) {
            BigTri bt = {};
            bt.px0 = 1; bt.px1 = 0; bt.py0 = 1; bt.py1 = 0;
            bt.tile0 = (uint32_t)tile;
            A.queue[e] = bt;
          }
          for (uint64_t j = tile; j < tile + tiles && j < A.tile_cap; ++j) A.tile_owner[j] = 0xFFFFFFFFu;
          kind = 1;
        }
      }
    }
    if (v < n) {
      if (kind == 1) {
        if (!grouped) {
          const float invA = __fdiv_rn(1.0f, ll2float_rn(E.s.A));
          raster_rect<0>(E.a, E.b, E.c, invA, E.s.px0, E.s.py0, E.s.px1, E.s.py1, A.zbuf, A.W);
        }
        store_cand(A, i, make_cand(E.a, E.b, E.c, E.s, t));
      } else {
        reinterpret_cast<uint32_t*>(A.cand + i)[6] = 0xFFFFFFFFu;  // empty: px0 = py0 = 0xFFFF
      }
    }
    if (grouped) group_raster<0>(E.a, E.b, E.c, E.s.A, E.s.px0, E.s.py0, E.s.px1, E.s.py1, kind == 1, A.zbuf, A.W);
  }
  // then the (rare) triangles that need clipping, from the front blocks' regions
  __syncthreads();  // pre is reused
  const uint32_t nc = region_prefix<NT>(A, A.clip_count, pre);
  for (uint32_t i = bid * blockDim.x + threadIdx.x; i < nc; i += stride) {
    const uint32_t t = __ldcg(A.clip + surv_slot(A, pre, i, i));
    const uint32_t* f = A.idx + 3 * (size_t)t;
    const Mat4 M = DEV_M ? load_mat(A.Mdev) : A.M;
    const float4 c0 = load_clip(M, A.pos, __ldg(f)), c1 = load_clip(M, A.pos, __ldg(f + 1)),
                 c2 = load_clip(M, A.pos, __ldg(f + 2));
    depth_clipped(A, t, c0, c1, c2);
  }
}

// Occlusion test of the marking pass on the final depth buffer (exact): a
// sub-triangle whose every sample depth is above the largest depth key of every
// 16x16 tile that its pixel box [px0, px1] x [py0, py1] touches cannot mark.  A
// sample depth is the rounded barycentric combination of the vertex depths; it
// lies within 7 * 2^-24 * max |z| of the exact value (three rounded terms, their
// two sums, 1 / A and the product), which lies in [zmin, zmax] (the clamped depth
// of conservative marking too), so zmin - 1e-6 max |z|, rounded down, bounds it
// from below.
__device__ __forceinline__ bool hidden_by_tiles(const RasterArgs& A, float z0, float z1, float z2, int px0, int py0,
                                                int px1, int py1) {
  const float zmin = fminf(z0, fminf(z1, z2));
  const float zabs = fmaxf(fabsf(z0), fmaxf(fabsf(z1), fabsf(z2)));
  const float lo = __fsub_rd(zmin, __fmaf_ru(zabs, 1e-6f, 1e-37f));
  const uint32_t klo = ordered(lo);
  uint32_t zm = 0u;
  for (int ty = py0 >> 4; ty <= (py1 >> 4); ++ty)
    for (int tx = px0 >> 4; tx <= (px1 >> 4); ++tx) zm = max(zm, __ldcg(A.zmax + ty * A.ztx + tx));
  return klo > zm;
}

// The largest depth key of each 16x16 pixel tile of the final depth buffer: a
// warp per tile, a half warp per row.
__device__ __forceinline__ void zmax_body(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t zty = (uint32_t)((A.H + 15) / 16), ntile = (uint32_t)A.ztx * zty;
  const uint32_t nwarps = (nblk * blockDim.x) >> 5;
  for (uint32_t g = (bid * blockDim.x + threadIdx.x) >> 5; g < ntile; g += nwarps) {
    const int x = (int)(g % (uint32_t)A.ztx) * 16 + (int)(lane & 15);
    const int y0 = (int)(g / (uint32_t)A.ztx) * 16 + (int)(lane >> 4);
    uint32_t m = 0u;
    uint32_t k[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int y = y0 + 2 * r;
      k[r] = (x < A.W && y < A.H) ? __ldcg(A.zbuf + (size_t)y * A.W + x) : 0u;
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) m = max(m, k[r]);
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if (lane == 0) A.zmax[g] = m;
  }
}

// The marking pass lists each 1024-triangle tile in which it marks a triangle, once.
__device__ __forceinline__ void note_tile(const RasterArgs& A, uint32_t tile) {
  if (!__ldcg(A.tile_flag + tile) && atomicExch(A.tile_flag + tile, 1u) == 0u)
    A.tile_list[atomicAdd(&A.ctr->n_vtiles, 1u)] = tile;
}

// The depth key of a pixel: the buffer's word, or the upper half of key << 32 | triangle.
template <bool WIN>
__device__ __forceinline__ uint32_t* zword(const RasterArgs& A, size_t pix) {
  return WIN ? reinterpret_cast<uint32_t*>(A.zid) + 2 * pix + 1 : A.zbuf + pix;
}

// One 16x16 tile of a queued record, by a warp, PASS as in sample().
template <int PASS, bool WIN>
__device__ __forceinline__ void raster_tile(const RasterArgs& A, const BigTri& q, uint32_t local) {
  const uint32_t lane = threadIdx.x & 31;
  const int px0 = q.px0, py0 = q.py0, px1 = q.px1, py1 = q.py1;
  // marking: another tile of the sub-triangle may have marked its triangle already
  // (one answer for the warp, which stays together below)
  if (PASS >= 1 && __any_sync(0xFFFFFFFFu, (__ldcg(A.vt + (q.tri >> 5)) >> (q.tri & 31)) & 1u)) return;
  const uint32_t tx_n = (uint32_t)((px1 - px0 + kBigTile) / kBigTile);
  const int bx = px0 + (int)(local % tx_n) * kBigTile, by = py0 + (int)(local / tx_n) * kBigTile;
  if (PASS >= 1 && !WIN && hidden_by_tiles(A, q.zn[0], q.zn[1], q.zn[2], bx, by, min(bx + kBigTile - 1, px1),
                                   min(by + kBigTile - 1, py1)))
    return;
  SV a{q.X[0], q.Y[0], q.zn[0]}, b{q.X[1], q.Y[1], q.zn[1]}, c{q.X[2], q.Y[2], q.zn[2]};
  const int64_t Ar = (b.X - a.X) * (c.Y - a.Y) - (c.X - a.X) * (b.Y - a.Y);
  const float invA = __fdiv_rn(1.0f, ll2float_rn(Ar));
  const float zmin = fminf(a.zn, fminf(b.zn, c.zn)), zmax = fmaxf(a.zn, fmaxf(b.zn, c.zn));
  bool vis = false;
  const int px = bx + (int)(lane % kBigTile), py_first = by + (int)(lane / kBigTile);
  const Edges E = edges_at(a, b, c, px, py_first);
  int64_t e[3] = {E.e[0], E.e[1], E.e[2]};
  // only the tile's rows inside the box (the last tile row of a box is often
  // short); the same trip count in every lane
  const int rows = min(by + kBigTile - 1, py1) - by + 1;
  const int steps = (rows + 32 / kBigTile - 1) / (32 / kBigTile);
#pragma unroll 1
  for (int k = 0; k < steps; ++k) {
    const int py = py_first + k * (32 / kBigTile);
    if (px <= px1 && py <= py1)
      vis |= sample<PASS>(E, e, a, b, c, invA, zword<WIN>(A, (size_t)py * A.W + px), zmin, zmax);
    if (PASS >= 1 && __any_sync(0xFFFFFFFFu, vis)) break;
    e[0] += E.dy[0] * (32 / kBigTile);
    e[1] += E.dy[1] * (32 / kBigTile);
    e[2] += E.dy[2] * (32 / kBigTile);
  }
  if (PASS >= 1) {
    if (__any_sync(0xFFFFFFFFu, vis) && lane == 0) {
      atomicOr(A.vt + (q.tri >> 5), 1u << (q.tri & 31));
      note_tile(A, q.tri >> 10);
    }
  }
}

// Large sub-triangles: one warp per 16x16 tile of a queued record (grid-stride).
template <int PASS>
__device__ __forceinline__ void big_tiles(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warp = ((uint64_t)bid * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)nblk * blockDim.x) >> 5;
  const unsigned long long st = __ldcg(&A.ctr->big);
  const uint64_t n_ent = (st >> 40) < A.queue_cap ? (st >> 40) : A.queue_cap;
  const uint64_t n_tiles = st & ((1ull << 40) - 1);
  if (n_ent == 0) return;
  const uint64_t n_used = n_tiles < A.tile_cap ? n_tiles : A.tile_cap;
  for (uint64_t g = warp; g < n_used; g += nwarps) {
    const uint32_t lo = __ldcg(A.tile_owner + g);
    if (lo >= n_ent) continue;
    const BigTri& q = A.queue[lo];
    const int px0 = q.px0, py0 = q.py0, px1 = q.px1, py1 = q.py1;
    if (px1 < px0 || py1 < py0) continue;
    const uint32_t tx_n = (uint32_t)((px1 - px0 + kBigTile) / kBigTile);
    const uint32_t ty_n = (uint32_t)((py1 - py0 + kBigTile) / kBigTile);
    const uint64_t local = g - q.tile0;
    if (local >= (uint64_t)tx_n * ty_n) continue;
    raster_tile<PASS, false>(A, q, (uint32_t)local);
  }
}

// Marking pass: first the tiles of the large sub-triangles, then the candidate
// list (a record is visible when one of its samples has key <= the depth buffer;
// visible bits are OR-ed per VT word and warp).  One launch for both, so blocks
// that finish their share of the tiles early take candidate records.
template <bool CONS, int NT>
__device__ __forceinline__ void mark_body(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  uint32_t* pre = region_pre();
  __shared__ int32_t s_status;
  if (threadIdx.x == 0) s_status = __ldcg(&A.ctr->status);
  __syncthreads();
  if (s_status != 0) return;
  big_tiles<CONS ? 2 : 1>(A, bid, nblk);
  const uint32_t ns = surv_prefix<NT>(A, pre);
  const uint32_t nc = min(__ldcg(&A.ctr->ncand), A.cand_cap - A.clip_base);
  const uint32_t n = ns + nc;  // survivor records, then the clipped-path records
  const uint32_t stride = nblk * blockDim.x;
  // few records for the grid: a group of kRasterGroup lanes per record (as in the
  // exact pass), its samples tested together instead of one after the other
  const bool grouped = (uint64_t)n * kRasterGroup <= (uint64_t)stride;
  const uint32_t sub = threadIdx.x & (kRasterGroup - 1u);
  for (uint32_t base = bid * blockDim.x; (grouped ? base / kRasterGroup : base) < n; base += stride) {
    const uint32_t wb = base + (threadIdx.x & ~31u);  // the warp's first thread
    const uint32_t kfirst = grouped ? wb / kRasterGroup : wb;
    const uint32_t k = grouped ? (sub == 0u ? kfirst + (threadIdx.x & 31u) / kRasterGroup : n) : base + threadIdx.x;
    bool vis = false, go = false;
    uint32_t t = 0xFFFFFFFFu;
    SV ga{0, 0, 0.0f}, gb{0, 0, 0.0f}, gc{0, 0, 0.0f};
    int64_t gA = 0;
    int gx0 = 0, gy0 = 0, gx1 = -1, gy1 = -1;
    if (k < n) {
      const uint32_t i = k < ns ? surv_slot(A, pre, k, kfirst) : A.clip_base + (k - ns);
      const float4* s = reinterpret_cast<const float4*>(A.cand + i);
      const float4 fb = __ldcs(s + 1);
      const uint32_t b0 = __float_as_uint(fb.z), b1 = __float_as_uint(fb.w);
      if (b0 != 0xFFFFFFFFu) {
        const float4 fa = __ldcs(s), fc = __ldcs(s + 2);
        const SV a{__float_as_int(fa.x), __float_as_int(fa.y), fc.x};
        const SV b{__float_as_int(fa.z), __float_as_int(fa.w), fc.y};
        const SV c{__float_as_int(fb.x), __float_as_int(fb.y), fc.z};
        t = __float_as_uint(fc.w);
        const int px0 = (int)(b0 & 0xFFFFu), py0 = (int)(b0 >> 16), px1 = (int)(b1 & 0xFFFFu), py1 = (int)(b1 >> 16);
        if (!hidden_by_tiles(A, fc.x, fc.y, fc.z, px0, py0, px1, py1)) {
          const int64_t Ar = (b.X - a.X) * (c.Y - a.Y) - (c.X - a.X) * (b.Y - a.Y);
          if (grouped) {
            go = true;
            ga = a;
            gb = b;
            gc = c;
            gA = Ar;
            gx0 = px0;
            gy0 = py0;
            gx1 = px1;
            gy1 = py1;
          } else {
            const float invA = __fdiv_rn(1.0f, ll2float_rn(Ar));
            vis = raster_rect<CONS ? 2 : 1>(a, b, c, invA, px0, py0, px1, py1, A.zbuf, A.W);
          }
        }
      }
    }
    if (grouped) {
      const bool gv = group_raster<CONS ? 2 : 1>(ga, gb, gc, gA, gx0, gy0, gx1, gy1, go, A.zbuf, A.W);
      vis = sub == 0u && k < n && gv;
    }
    const uint32_t word = vis ? (t >> 5) : 0xFFFFFFFFu;
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, word);
    const uint32_t bits = __reduce_or_sync(peers, vis ? (1u << (t & 31)) : 0u);
    if (vis && (__ffs(peers) - 1) == (int)(threadIdx.x & 31)) {
      atomicOr(A.vt + word, bits);
      note_tile(A, word >> 5);
    }
  }
}

// Depth pre-pass of the large sub-triangles.
__device__ __forceinline__ void depth_big_body(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  big_tiles<0>(A, bid, nblk);
}

// ------------------------------------------------------------------ winners
//
// Single-pass visibility (the default).  A sample of the
// marking pass passes "<=" exactly when its key equals the pixel's smallest key, and
// both passes take the same samples, so the triangles to mark are those that own a
// pixel's smallest key: the depth pass keeps key << 32 | triangle per pixel (64-bit
// atomicMin) and the marking pass is one read of that buffer instead of a second
// rasterization.  Two triangles with the same key at a pixel are told by the returned
// old value: the key a pixel ends with stays there once it has arrived, so every later
// triangle with that key sees it and lists the pair; the marking pass marks the pairs
// whose key is still the pixel's.  If the list overflows (coincident geometry), the marking
// pass tests what is not marked against the buffer instead (mark_all).
//
// Three sizes of sub-triangles, so that the lanes of a warp have like work: boxes of at
// most kSmallMaxPix pixels are rasterized where they are set up (exact pass); boxes of
// at most kMidPix are listed and then rasterized by 4 .. 32 lanes each, as many as fill
// the grid, neighbouring lanes taking neighbouring samples; larger ones are 16x16 tiles,
// a warp per tile.  Edge functions of sub-triangles of less than 96 pixels a side fit 32
// bits (twice the product of the sides is 1.21e9; steps past the box's end, 128 rows of
// one pixel at most, add 0.81e9); their conversions to fp32 round as the 64-bit ones do.
// A top-left edge passes at 0, another one from 1, so that with 1 taken from
// the others a sample is covered when no value is negative.
//
// What bounds it: the atomics' round trips and the instructions of the samples (the
// larger boxes of a 3.2M-triangle floor at 1440p issue 60 % of the cycles).  Times of
// that pass: one sample of a lane at a time 851 us; four at once, their returned values
// looked at after the next four, 317 (three 332; six 447; looked at at once 485, which
// is the better way only for the small boxes' four rounds at most, 125 against 160).
// At least four lanes share a box, so that their atomics meet in a sector (one lane
// 446 us, two 384, four 374, eight 420, at three blocks per SM).  A load of the pixel's
// key before the atomic costs more than the atomics it saves (471 us against 379).
// Against two rasterizations, exact + larger boxes + marking: that floor 2475 -> 459
// us, 60 patches at 1080p 247 -> 83, 200 icospheres at 1080p 107 -> 62, one patch of
// 7,938 triangles at 1080p 52 -> 40 (events around each kernel, GB300).
constexpr int kMidPix = 256;  // (512: the same)
constexpr uint32_t kMarkBlocks = 152u * 4u;  // resident blocks of the marking kernel
constexpr uint32_t kMinLanes = 2;  // log2 of the fewest lanes a mid-size box gets
constexpr int kSpan32 = 96 * kSub;  // side of a sub-triangle with 32-bit edge functions

struct Tri32 {
  int X[3], Y[3];
  float z[3];
};

// Snapped vertices, pixel box and size class of one unclipped triangle.
struct WinSetup {
  Tri32 v;
  int px0, py0, px1, py1;
  bool fits;  // 32-bit edge functions
  bool front;  // front facing
  bool live;   // front facing, with a sample in its box
};

__device__ __forceinline__ uint32_t tiles_of(int w, int h) {
  return (uint32_t)((w + kBigTile - 1) / kBigTile) * (uint32_t)((h + kBigTile - 1) / kBigTile);
}

// 32-bit edge functions: the sides are short enough.
__device__ __forceinline__ bool fits32(const Tri32& v) {
  const int xmn = min(v.X[0], min(v.X[1], v.X[2])), xmx = max(v.X[0], max(v.X[1], v.X[2]));
  const int ymn = min(v.Y[0], min(v.Y[1], v.Y[2])), ymx = max(v.Y[0], max(v.Y[1], v.Y[2]));
  return xmx - xmn < kSpan32 && ymx - ymn < kSpan32;
}

__device__ __forceinline__ void project32(const float4& c, float hx, float hy, int& X, int& Y, float& z) {
  const SV s = project(CV{c.x, c.y, c.z, c.w}, hx, hy);
  X = (int)s.X;
  Y = (int)s.Y;
  z = s.zn;
}

__device__ __forceinline__ WinSetup win_setup(const RasterArgs& A, const float4& c0, const float4& c1,
                                              const float4& c2) {
  WinSetup s;
  project32(c0, A.hx, A.hy, s.v.X[0], s.v.Y[0], s.v.z[0]);
  project32(c1, A.hx, A.hy, s.v.X[1], s.v.Y[1], s.v.z[1]);
  project32(c2, A.hx, A.hy, s.v.X[2], s.v.Y[2], s.v.z[2]);
  const int xmn = min(s.v.X[0], min(s.v.X[1], s.v.X[2])), xmx = max(s.v.X[0], max(s.v.X[1], s.v.X[2]));
  const int ymn = min(s.v.Y[0], min(s.v.Y[1], s.v.Y[2])), ymx = max(s.v.Y[0], max(s.v.Y[1], s.v.Y[2]));
  s.px0 = max(-((128 - xmn) >> 8), 0);
  s.px1 = min((xmx - 128) >> 8, A.W - 1);
  s.py0 = max(-((128 - ymn) >> 8), 0);
  s.py1 = min((ymx - 128) >> 8, A.H - 1);
  s.fits = fits32(s.v);
  const int ux = s.v.X[1] - s.v.X[0], uy = s.v.Y[1] - s.v.Y[0], vx = s.v.X[2] - s.v.X[0], vy = s.v.Y[2] - s.v.Y[0];
  s.front = s.fits ? ux * vy - vx * uy > 0 : (int64_t)ux * vy - (int64_t)vx * uy > 0;
  s.live = s.front && s.px1 >= s.px0 && s.py1 >= s.py0;
  return s;
}

// Pixels of the conservative box (as setup's) instead of the samples'; 0: none.
__device__ __forceinline__ int cons_pixels(const RasterArgs& A, WinSetup& s) {
  const int xmn = min(s.v.X[0], min(s.v.X[1], s.v.X[2])), xmx = max(s.v.X[0], max(s.v.X[1], s.v.X[2]));
  const int ymn = min(s.v.Y[0], min(s.v.Y[1], s.v.Y[2])), ymx = max(s.v.Y[0], max(s.v.Y[1], s.v.Y[2]));
  const int px0 = max(-((-xmn) >> 8) - 1, 0), px1 = min(xmx >> 8, A.W - 1);
  const int py0 = max(-((-ymn) >> 8) - 1, 0), py1 = min(ymx >> 8, A.H - 1);
  s.px0 = px0;
  s.py0 = py0;
  s.px1 = px1;
  s.py1 = py1;
  return max(px1 - px0 + 1, 0) * max(py1 - py0 + 1, 0);
}

// Conservative marking takes a sub-triangle whose conservative box has more than kMidPix
// pixels by tiles, so the exact pass queues it with that box (the samples past its own box
// are not covered).  Gives s that box if so.
__device__ __forceinline__ bool cons_queue(const RasterArgs& A, WinSetup& s) {
  if (!s.front) return false;
  WinSetup c = s;
  if (cons_pixels(A, c) <= kMidPix) return false;
  s = c;
  return true;
}

// Set once this block has found the tie list full (cleared before a pass's first sample).
__device__ __forceinline__ volatile uint32_t* ties_full() {
  __shared__ uint32_t full;
  return &full;
}

// Lists a tie.  A block that has found the list full adds no more: the number of ties does
// not matter then, a count that stays below the list's room plus the threads of the grid
// cannot wrap however many samples of a view are equal, and the counter's atomics, all on
// one word, do not hold the samples up (depth pass of eight copies of a patch 303 -> 74
// us).  (The mid-size boxes' loop is sensitive to this function's form: 330 us on a
// 3.2M-triangle floor; with lists by SM and by block, with the flag kept from the compiler
// no longer, with the counter read instead of the flag, 340 to 500.)
__device__ __forceinline__ void note_tie(const RasterArgs& A, uint32_t pix, uint32_t key, uint32_t t0, uint32_t t1) {
  if (*ties_full()) return;
  const uint32_t i = atomicAdd(&A.ctr->n_ties, 1u);
  if (i < kTies) A.ties[i] = make_uint4(pix, key, t0, t1);
  else *ties_full() = 1u;
}

// The samples a thread has put: the returned value of one is looked at when the next
// is on its way.
struct Put {
  unsigned long long old = ~0ull;
  uint32_t key = 0u, pix = 0u;
  __device__ __forceinline__ void check(const RasterArgs& A, uint32_t t) const {
    if ((uint32_t)(old >> 32) == key && (uint32_t)old != t) note_tie(A, pix, key, (uint32_t)old, t);
  }
  __device__ __forceinline__ void put(const RasterArgs& A, uint32_t p, uint32_t k, uint32_t t) {
    const unsigned long long o = atomicMin(A.zid + p, ((unsigned long long)k << 32) | t);
    check(A, t);
    old = o;
    key = k;
    pix = p;
  }
};

// Edge functions at the sample of pixel (px, py), their steps per pixel, and the plane's
// weights of a 32-bit sub-triangle.
struct Edges32 {
  int e[3], dx[3], dy[3], nb[3];  // e: less nb (0: top-left edge, 1: another)
  float invA;
};

__device__ __forceinline__ Edges32 edges32(const Tri32& v, int px, int py) {
  Edges32 E;
  const int sx = px * 256 + 128, sy = py * 256 + 128;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int a = (i + 1) % 3, b = (i + 2) % 3;  // E0: edge v1 -> v2, E1: v2 -> v0, E2: v0 -> v1
    const int ex = v.X[b] - v.X[a], ey = v.Y[b] - v.Y[a];
    E.nb[i] = (ey < 0 || (ey == 0 && ex < 0)) ? 0 : 1;
    E.e[i] = ex * (sy - v.Y[a]) - ey * (sx - v.X[a]) - E.nb[i];
    E.dx[i] = -ey * 256;
    E.dy[i] = ex * 256;
  }
  const int area = (v.X[1] - v.X[0]) * (v.Y[2] - v.Y[0]) - (v.X[2] - v.X[0]) * (v.Y[1] - v.Y[0]);
  E.invA = __fdiv_rn(1.0f, __int2float_rn(area));
  return E;
}

// Depth key of a covered sample with (reduced) edge values e; false outside [-1, 1].
__device__ __forceinline__ bool key32(const Edges32& E, int e0, int e1, int e2, const Tri32& v, uint32_t& key) {
  float s = __fmul_rn(__int2float_rn(e0 + E.nb[0]), v.z[0]);
  s = __fadd_rn(s, __fmul_rn(__int2float_rn(e1 + E.nb[1]), v.z[1]));
  s = __fadd_rn(s, __fmul_rn(__int2float_rn(e2 + E.nb[2]), v.z[2]));
  const float d = __fadd_rn(__fmul_rn(s, E.invA), 0.0f);  // (-0 becomes +0)
  const uint32_t u = __float_as_uint(d);
  key = u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);  // ordered(d)
  return fabsf(d) <= 1.0f;
}

__device__ __forceinline__ uint32_t zkey(const RasterArgs& A, uint32_t pix) {
  return __ldcg(reinterpret_cast<const uint32_t*>(A.zid) + 2 * (size_t)pix + 1);
}

// Puts a thread's N samples (those that are on): their atomics are all on their way
// before the first returned value is looked at.
template <int N>
__device__ __forceinline__ void put_n(const RasterArgs& A, uint32_t t, const bool (&on)[N], const uint32_t (&key)[N],
                                      const uint32_t (&pix)[N]) {
  unsigned long long old[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    old[i] = ~0ull;
    if (on[i]) old[i] = atomicMin(A.zid + pix[i], ((unsigned long long)key[i] << 32) | t);
  }
  bool any = false;
#pragma unroll
  for (int i = 0; i < N; ++i) any |= on[i] && (uint32_t)(old[i] >> 32) == key[i];
  if (!any) return;
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (on[i] && (uint32_t)(old[i] >> 32) == key[i] && (uint32_t)old[i] != t)
      note_tie(A, pix[i], key[i], (uint32_t)old[i], t);
}

// The same with the returned values looked at only when the thread's next N are on their
// way (or at the end): for loops of many rounds, where each would wait for its own.
template <int N>
struct PutN {
  unsigned long long old[N];
  uint32_t key[N], pix[N];
  __device__ __forceinline__ PutN() {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      old[i] = ~0ull;
      key[i] = pix[i] = 0u;
    }
  }
  __device__ __forceinline__ void check(const RasterArgs& A, uint32_t t) const {
#pragma unroll
    for (int i = 0; i < N; ++i)
      if ((uint32_t)(old[i] >> 32) == key[i] && (uint32_t)old[i] != t) note_tie(A, pix[i], key[i], (uint32_t)old[i], t);
  }
  __device__ __forceinline__ void put(const RasterArgs& A, uint32_t t, const bool (&on)[N], const uint32_t (&k)[N],
                                      const uint32_t (&p)[N]) {
    unsigned long long o[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      o[i] = ~0ull;
      if (on[i]) o[i] = atomicMin(A.zid + p[i], ((unsigned long long)k[i] << 32) | t);
    }
    check(A, t);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      old[i] = o[i];
      key[i] = on[i] ? k[i] : 0u;
      pix[i] = p[i];
    }
  }
};

// One of a thread's N samples (those that are on) has the pixel's final key.
template <int N>
__device__ __forceinline__ bool test_n(const RasterArgs& A, const bool (&on)[N], const uint32_t (&key)[N],
                                       const uint32_t (&pix)[N]) {
  uint32_t z[N];
  bool hit = false;
#pragma unroll
  for (int i = 0; i < N; ++i) z[i] = on[i] ? zkey(A, pix[i]) : 0u;
#pragma unroll
  for (int i = 0; i < N; ++i) hit |= on[i] && key[i] <= z[i];
  return hit;
}

// What becomes of the samples: put at once, put with the returned values looked at later,
// or (nothing is written) tested against the final keys.
enum Samples { kPut, kPutLater, kTest };

// Samples first, first + step, .. (row order) of a 32-bit sub-triangle's box, N at a time
// so that their atomics or loads overlap.  step lanes side by side then take neighbouring
// pixels.  kTest: true when one of them has the pixel's final key.
template <int N, Samples DO>
__device__ __forceinline__ bool win_box(const RasterArgs& A, const Tri32& v, uint32_t t, int px0, int py0, int px1,
                                        int py1, int first, int step) {
  const int w = px1 - px0 + 1, n = w * (py1 - py0 + 1);
  if (first >= n) return false;
  const int sy = step == 1 ? (w == 1 ? 1 : 0) : step / w, sx = step - sy * w;  // step = sy rows and sx < w pixels
  const int fy = first / w, fx = first - fy * w;
  const Edges32 E = edges32(v, px0 + fx, py0 + fy);
  // a step inside the row, and one that runs past its end (a row more, w pixels back)
  const int a0 = E.dy[0] * sy + E.dx[0] * sx, a1 = E.dy[1] * sy + E.dx[1] * sx, a2 = E.dy[2] * sy + E.dx[2] * sx;
  const int b0 = a0 + E.dy[0] - E.dx[0] * w, b1 = a1 + E.dy[1] - E.dx[1] * w, b2 = a2 + E.dy[2] - E.dx[2] * w;
  const uint32_t ap = (uint32_t)(A.W * sy + sx), bp = ap + (uint32_t)(A.W - w);
  int e0 = E.e[0], e1 = E.e[1], e2 = E.e[2], col = w - fx;  // col: pixels to the row's end
  uint32_t p = (uint32_t)(py0 + fy) * (uint32_t)A.W + (uint32_t)(px0 + fx);
  PutN<DO == kPutLater ? N : 1> later;
  for (int left = n - 1 - first; left >= 0;) {  // (negative once the box is done)
    uint32_t key[N], pix[N];
    bool on[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      pix[i] = p;
      on[i] = (e0 | e1 | e2 | left) >= 0 && key32(E, e0, e1, e2, v, key[i]);
      col -= sx;
      const bool wrap = col <= 0;
      col += wrap ? w : 0;
      e0 += wrap ? b0 : a0;
      e1 += wrap ? b1 : a1;
      e2 += wrap ? b2 : a2;
      p += wrap ? bp : ap;
      left -= step;
    }
    if constexpr (DO == kPutLater) later.put(A, t, on, key, pix);
    else if constexpr (DO == kPut) put_n(A, t, on, key, pix);
    else if (test_n(A, on, key, pix)) return true;
  }
  if constexpr (DO == kPutLater) later.check(A, t);
  return false;
}

// Any sub-triangle, 64-bit edge functions: samples first, first + step, .. of its box in
// row order.  TEST: nothing is written; true when one of them has the pixel's final key.
template <bool TEST>
__device__ __forceinline__ bool win_rect64(const RasterArgs& A, const SV& a, const SV& b, const SV& c, uint32_t t, int px0,
                                           int py0, int px1, int py1, uint32_t first, uint32_t step) {
  const int64_t Ar = (b.X - a.X) * (c.Y - a.Y) - (c.X - a.X) * (b.Y - a.Y);
  const float invA = __fdiv_rn(1.0f, ll2float_rn(Ar));
  const uint32_t w = (uint32_t)(px1 - px0 + 1), n = w * (uint32_t)(py1 - py0 + 1);
  Put q;
  for (uint32_t s = first; s < n; s += step) {
    const int px = px0 + (int)(s % w), py = py0 + (int)(s / w);
    const Edges E = edges_at(a, b, c, px, py);
    const bool in = (E.e[0] > 0 || (E.e[0] == 0 && E.tl[0])) && (E.e[1] > 0 || (E.e[1] == 0 && E.tl[1])) &&
                    (E.e[2] > 0 || (E.e[2] == 0 && E.tl[2]));
    if (!in) continue;
    float f = __fmul_rn(ll2float_rn(E.e[0]), a.zn);
    f = __fadd_rn(f, __fmul_rn(ll2float_rn(E.e[1]), b.zn));
    f = __fadd_rn(f, __fmul_rn(ll2float_rn(E.e[2]), c.zn));
    const float d = __fmul_rn(f, invA);
    if (!(d >= -1.0f && d <= 1.0f)) continue;
    const uint32_t key = ordered(d), p = (uint32_t)py * (uint32_t)A.W + (uint32_t)px;
    if (TEST) {
      if (key <= zkey(A, p)) return true;
    } else {
      q.put(A, p, key, t);
    }
  }
  if (!TEST) q.check(A, t);
  return false;
}

// Record e of the queue: a large sub-triangle whose tiles are numbered from `tile` on.
// (Records and tiles are reserved by one atomic, so a later record has later tiles.)
__device__ __forceinline__ void win_queue(const RasterArgs& A, const int (&X)[3], const int (&Y)[3],
                                          const float (&z)[3], int px0, int py0, int px1, int py1, bool fits,
                                          uint32_t t, uint32_t e, uint64_t tile) {
  BigTri bt;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    bt.X[i] = X[i];
    bt.Y[i] = Y[i];
    bt.zn[i] = z[i];
  }
  bt.px0 = px0;
  bt.py0 = py0;
  bt.px1 = px1;
  bt.py1 = py1;
  bt.tri = t;
  bt.tile0 = (uint32_t)tile;
  bt.pad = (fits ? 0x80000000u : 0u) | (uint32_t)(tile >> 32);
  A.queue[e] = bt;
}

__device__ __forceinline__ uint64_t first_tile(uint32_t tile0, uint32_t pad) {
  return tile0 | (uint64_t)(pad & 0x7FFFFFFFu) << 32;
}

// Owners of each lane's record's tiles (none: tiles = 0) that the table has room for: few
// by the lane itself, many by the whole warp (the exact pass of a 1080p view with two
// clipped ground triangles: 361 us with every lane on its own, 22 so).  All lanes of the
// warp call it.
__device__ __forceinline__ void own_tiles(const RasterArgs& A, uint32_t e, uint64_t tile, uint32_t tiles) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t j0 = (uint32_t)(tile < A.tile_cap ? tile : A.tile_cap);
  const uint32_t n = tiles < A.tile_cap - j0 ? tiles : A.tile_cap - j0;
  if (n <= 8u)
    for (uint32_t j = 0; j < n; ++j) A.tile_owner[j0 + j] = e;
  for (uint32_t m = __ballot_sync(0xFFFFFFFFu, n > 8u); m; m &= m - 1u) {
    const int src = __ffs(m) - 1;
    const uint32_t we = __shfl_sync(0xFFFFFFFFu, e, src), wj = __shfl_sync(0xFFFFFFFFu, j0, src),
                   wn = __shfl_sync(0xFFFFFFFFu, n, src);
    for (uint32_t j = lane; j < wn; j += 32u) A.tile_owner[wj + j] = we;
  }
}

// The record that tile g belongs to, the last one that starts at or before it: each round
// the lanes look at 32 records evenly apart.
__device__ __forceinline__ uint32_t record_of(const RasterArgs& A, uint32_t n_ent, uint64_t g) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t lo = 0, hi = n_ent;
  while (hi - lo > 1u) {
    const uint32_t step = (hi - lo + 31u) / 32u, i = lo + lane * step;
    bool before = false;
    if (i < hi) {
      const uint2 q = __ldcg(reinterpret_cast<const uint2*>(&A.queue[i].tile0));
      before = first_tile(q.x, q.y) <= g;
    }
    lo += ((uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, before)) - 1u) * step;  // (record lo starts at or before g)
    hi = min(hi, lo + step);
  }
  return lo;
}

// Tile::run(A, record, tile in it) for every tile of the queued records, a warp each; st:
// the queue's counter.  The table holds the owners of the first tile_cap tiles, four for
// each record there is room for.  The tiles past it (of a few triangles that fill the
// view) are taken in runs of neighbours: the first one's record is looked up, the next
// ones' are the same or the next.  (Rasterized by the threads that set them up instead, 40
// triangles that fill a 1080p window take 1.7 s and 40 clipped ones 734 ms; so 0.69 and
// 0.33 ms.)
template <class Tile>
__device__ __forceinline__ void for_tiles(const RasterArgs& A, unsigned long long st, uint32_t bid, uint32_t nblk) {
  const uint32_t warp = (bid * blockDim.x + threadIdx.x) >> 5, nwarps = (nblk * blockDim.x) >> 5;
  const uint32_t n_ent = (uint32_t)min((unsigned long long)A.queue_cap, st >> 40);
  if (n_ent == 0u) return;
  uint64_t n_tiles = st & ((1ull << 40) - 1);
  if ((st >> 40) > A.queue_cap) {  // tiles reserved past the last record belong to no one
    const BigTri& q = A.queue[n_ent - 1u];
    n_tiles = first_tile(q.tile0, q.pad) + tiles_of(q.px1 - q.px0 + 1, q.py1 - q.py0 + 1);
  }
  const uint32_t n_tab = (uint32_t)min(n_tiles, (uint64_t)A.tile_cap);
  const uint64_t rest = n_tiles - n_tab, each = (rest + nwarps - 1u) / nwarps;
  const uint32_t run = each < 1u ? 1u : each > 32u ? 32u : (uint32_t)each;
  const uint64_t runs = (rest + run - 1u) / run;
  for (uint64_t i = warp; i < n_tab + runs; i += nwarps) {
    uint32_t e, k = 1u;
    uint64_t g = i;
    if (i < n_tab) {
      e = __ldcg(A.tile_owner + i);
    } else {
      g = n_tab + (i - n_tab) * run;
      k = (uint32_t)min((uint64_t)run, n_tiles - g);
      e = record_of(A, n_ent, g);
    }
    for (; k; --k, ++g) {
      const BigTri* q = A.queue + e;
      uint64_t local = g - first_tile(q->tile0, q->pad);
      if (local >= tiles_of(q->px1 - q->px0 + 1, q->py1 - q->py0 + 1)) {  // (the run's next record)
        ++q;
        ++e;
        local = 0u;
      }
      Tile::run(A, *q, (uint32_t)local);
    }
  }
}

// A triangle that must be clipped (rare).  Its sub-triangles are rasterized here (small,
// or the queue is full) or queued, their records first .. first + n - 1 returned for their
// tiles' owners.  TEST: those rasterized here, tested as in win_rect64.
struct Fan {
  uint32_t first, n;
};

template <bool TEST>
__device__ __noinline__ bool win_clipped(const RasterArgs& A, uint32_t t, float4 c0, float4 c1, float4 c2, Fan& fan) {
  fan = Fan{0u, 0u};
  CV poly[kMaxPoly];
  poly[0] = CV{c0.x, c0.y, c0.z, c0.w};
  poly[1] = CV{c1.x, c1.y, c1.z, c1.w};
  poly[2] = CV{c2.x, c2.y, c2.z, c2.w};
  const int n = clip_polygon(poly, 3);
  if (n < 0) {
    if (!TEST) set_status(A.ctr, FA_E_CAPACITY);
    return false;
  }
  if (n < 3) return false;
  for (int i = 0; i < n; ++i)
    if (!(poly[i].w > 0.0f)) return false;
  SV sv[kMaxPoly];
  uint32_t nq = 0;
  uint64_t tiles = 0;
  for (int i = 0; i < n; ++i) sv[i] = project(poly[i], A.hx, A.hy);
  if (!TEST) {
    for (int i = 1; i + 1 < n; ++i) {
      const Setup s = setup(sv[0], sv[i], sv[i + 1], A.W, A.H, A.cons);
      const int w = s.px1 - s.px0 + 1, h = s.py1 - s.py0 + 1;
      if (s.A <= 0 || w <= 0 || h <= 0 || w * h <= kSmallMaxPix) continue;
      ++nq;
      tiles += tiles_of(w, h);
    }
  }
  const bool full = TEST && (__ldcg(&A.ctr->big) >> 40) > A.queue_cap;
  uint64_t e = 0, tile = 0;
  if (nq) {
    const unsigned long long old = atomicAdd(&A.ctr->big, ((unsigned long long)nq << 40) | (unsigned long long)tiles);
    e = old >> 40;
    tile = old & ((1ull << 40) - 1);
    if (e < A.queue_cap) fan = Fan{(uint32_t)e, min(nq, A.queue_cap - (uint32_t)e)};
  }
  for (int i = 1; i + 1 < n; ++i) {
    const SV &a = sv[0], &b = sv[i], &c = sv[i + 1];
    const Setup s = setup(a, b, c, A.W, A.H, A.cons);
    const int w = s.px1 - s.px0 + 1, h = s.py1 - s.py0 + 1;
    if (s.A <= 0 || w <= 0 || h <= 0) continue;
    if (TEST) {
      if ((w * h <= kSmallMaxPix || full) && win_rect64<true>(A, a, b, c, t, s.px0, s.py0, s.px1, s.py1, 0u, 1u))
        return true;
      continue;
    }
    if (w * h > kSmallMaxPix) {
      if (e < A.queue_cap) {
        const int X[3] = {(int)a.X, (int)b.X, (int)c.X}, Y[3] = {(int)a.Y, (int)b.Y, (int)c.Y};
        const float z[3] = {a.zn, b.zn, c.zn};
        win_queue(A, X, Y, z, s.px0, s.py0, s.px1, s.py1, false, t, (uint32_t)e, tile);
        ++e;
        tile += tiles_of(w, h);
        continue;
      }
    }
    win_rect64<false>(A, a, b, c, t, s.px0, s.py0, s.px1, s.py1, 0u, 1u);
  }
  return false;
}

// First slot of mid-size list r (its blocks' shares one after the other).
__device__ __forceinline__ uint32_t mid_base(const RasterArgs& A, uint32_t r) {
  return (uint32_t)((uint64_t)r * A.mid_blocks / A.mid_lists) * A.mid_per_block;
}

// Exact set-up of the survivors (as exact_body): small ones rasterized here, mid-size
// ones listed, large ones queued.
// CONS: conservative marking (A.cons) may ask for cons_queue.
template <bool DEV_M, int NT, bool CONS>
__device__ __forceinline__ void exact_win_body(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  uint32_t* pre = region_pre();
  const uint32_t lane = threadIdx.x & 31;
  // (the clipped triangles' counts with the survivors': mostly there are none)
  uint32_t clipped = 0;
  if (threadIdx.x == 0) *ties_full() = 0u;
#pragma unroll
  for (uint32_t j = 0; j < (kMaxFrontBlocks + NT - 1) / NT; ++j)
    if (threadIdx.x + j * NT < A.front_blocks) clipped |= __ldcg(A.clip_count + threadIdx.x + j * NT);
  const uint32_t n = surv_prefix<NT>(A, pre);
  const uint32_t stride = nblk * blockDim.x;
  const bool grouped = (uint64_t)n * kRasterGroup <= (uint64_t)stride;  // few survivors: see exact_body
  const uint32_t sub = lane & (kRasterGroup - 1u);
  const uint32_t list = ((bid + 1u) * A.mid_lists - 1u) / A.mid_blocks;
  const uint32_t lbase = mid_base(A, list), lcap = mid_base(A, list + 1u) - lbase;
  for (uint32_t wbase = bid * blockDim.x + (threadIdx.x & ~31u); (grouped ? wbase / kRasterGroup : wbase) < n;
       wbase += stride) {
    const uint32_t vfirst = grouped ? wbase / kRasterGroup : wbase;
    const uint32_t v = grouped ? (sub == 0u ? vfirst + lane / kRasterGroup : n) : wbase + lane;
    WinSetup E = {};
    uint32_t t = 0, tiles = 0;
    int kind = 0;  // 0 nothing, 1 small, 2 large, 3 mid-size
    if (v < n) {
      const uint32_t i = surv_slot(A, pre, v, vfirst);
      const float4* sc = A.surv_clip + 3 * (size_t)i;
      t = __ldcg(A.surv + i);
      E = win_setup(A, __ldcs(sc), __ldcs(sc + 1), __ldcs(sc + 2));
      if (E.live) {
        const int w = E.px1 - E.px0 + 1, h = E.py1 - E.py0 + 1, pix = w * h;
        kind = !E.fits ? 2 : pix <= kSmallMaxPix ? 1 : pix <= kMidPix ? 3 : 2;
      }
      if (CONS && A.cons && cons_queue(A, E)) kind = 2;
      if (kind == 2) tiles = tiles_of(E.px1 - E.px0 + 1, E.py1 - E.py0 + 1);
    }
    // large triangles of the warp reserve queue records and tiles with one atomic; what
    // finds no record any more is listed as mid-size, or, too large for 32 bits, done here
    const uint32_t bigs = __ballot_sync(0xFFFFFFFFu, kind == 2);
    if (bigs) {
      uint32_t tpre = tiles;  // inclusive prefix of tiles over the warp
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, tpre, o);
        if (lane >= (unsigned)o) tpre += y;
      }
      const uint32_t ttot = __shfl_sync(0xFFFFFFFFu, tpre, 31);
      unsigned long long old = 0;
      if (lane == 0)
        old = atomicAdd(&A.ctr->big, ((unsigned long long)__popc(bigs) << 40) | (unsigned long long)ttot);
      old = __shfl_sync(0xFFFFFFFFu, old, 0);
      const uint64_t e = (old >> 40) + __popc(bigs & ((1u << lane) - 1u));
      const uint64_t tile = (old & ((1ull << 40) - 1)) + (tpre - tiles);
      if (kind == 2 && e < A.queue_cap) {
        win_queue(A, E.v.X, E.v.Y, E.v.z, E.px0, E.py0, E.px1, E.py1, E.fits, t, (uint32_t)e, tile);
      } else {
        tiles = 0;
        if (kind == 2 && E.fits) {
          kind = 3;
        } else if (kind == 2) {
          const SV a{E.v.X[0], E.v.Y[0], E.v.z[0]}, b{E.v.X[1], E.v.Y[1], E.v.z[1]}, c{E.v.X[2], E.v.Y[2], E.v.z[2]};
          win_rect64<false>(A, a, b, c, t, E.px0, E.py0, E.px1, E.py1, 0u, 1u);
        }
      }
      own_tiles(A, (uint32_t)e, tile, tiles);
    }
    const uint32_t mids = __ballot_sync(0xFFFFFFFFu, kind == 3);
    if (mids) {
      uint32_t o = 0;
      if (lane == 0) o = atomicAdd(&A.ctr->n_mid[list][0], (uint32_t)__popc(mids));
      o = __shfl_sync(0xFFFFFFFFu, o, 0) + __popc(mids & ((1u << lane) - 1u));
      if (kind == 3) {
        if (o < lcap) {  // (always: the list has room for every survivor its blocks see)
          float4* d = reinterpret_cast<float4*>(A.cand + lbase + o);
          d[0] = make_float4(__int_as_float(E.v.X[0]), __int_as_float(E.v.Y[0]), __int_as_float(E.v.X[1]),
                             __int_as_float(E.v.Y[1]));
          d[1] = make_float4(__int_as_float(E.v.X[2]), __int_as_float(E.v.Y[2]),
                             __int_as_float(E.px0 | (E.py0 << 16)), __int_as_float(E.px1 | (E.py1 << 16)));
          d[2] = make_float4(E.v.z[0], E.v.z[1], E.v.z[2], __uint_as_float(t));
        } else {
          set_status(A.ctr, FA_E_CAPACITY);
        }
      }
    }
    if (!grouped) {
      if (kind == 1) win_box<4, kPut>(A, E.v, t, E.px0, E.py0, E.px1, E.py1, 0, 1);
    } else {
      // the group's leader holds the triangle; each lane takes one sample of its box
      const uint32_t src = lane & ~(kRasterGroup - 1u);
      Tri32 g;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        g.X[j] = __shfl_sync(0xFFFFFFFFu, E.v.X[j], src);
        g.Y[j] = __shfl_sync(0xFFFFFFFFu, E.v.Y[j], src);
        g.z[j] = __shfl_sync(0xFFFFFFFFu, E.v.z[j], src);
      }
      const int px0 = __shfl_sync(0xFFFFFFFFu, E.px0, src), py0 = __shfl_sync(0xFFFFFFFFu, E.py0, src);
      const int px1 = __shfl_sync(0xFFFFFFFFu, E.px1, src), py1 = __shfl_sync(0xFFFFFFFFu, E.py1, src);
      const uint32_t gt = __shfl_sync(0xFFFFFFFFu, t, src);
      const bool go = __shfl_sync(0xFFFFFFFFu, kind, src) == 1;
      if (go) win_box<1, kPut>(A, g, gt, px0, py0, px1, py1, (int)sub, (int)kRasterGroup);
    }
  }
  // then the (rare) triangles that need clipping, from the front blocks' regions
  if (!__syncthreads_or(clipped != 0u)) return;  // (and pre is reused)
  const uint32_t nc = region_prefix<NT>(A, A.clip_count, pre);
  for (uint32_t base = bid * blockDim.x + (threadIdx.x & ~31u); base < nc; base += stride) {
    const uint32_t i = base + lane;
    Fan fan{0u, 0u};
    if (i < nc) {
      const uint32_t t = __ldcg(A.clip + surv_slot(A, pre, i, i));
      const uint32_t* f = A.idx + 3 * (size_t)t;
      const Mat4 M = DEV_M ? load_mat(A.Mdev) : A.M;
      win_clipped<false>(A, t, load_clip(M, A.pos, __ldg(f)), load_clip(M, A.pos, __ldg(f + 1)),
                         load_clip(M, A.pos, __ldg(f + 2)), fan);
    }
    // a record of each lane's fan after the other
    for (uint32_t q = 0; __any_sync(0xFFFFFFFFu, q < fan.n); ++q) {
      uint32_t tiles = 0;
      uint64_t tile = 0;
      if (q < fan.n) {
        const BigTri& r = A.queue[fan.first + q];
        tile = first_tile(r.tile0, r.pad);
        tiles = tiles_of(r.px1 - r.px0 + 1, r.py1 - r.py0 + 1);
      }
      own_tiles(A, fan.first + q, tile, tiles);
    }
  }
}

// Lanes (their log2) of each of n listed sub-triangles on a grid of `stride` threads.
__device__ __forceinline__ uint32_t mid_lanes(uint32_t n, uint32_t stride) {
  uint32_t lg = kMinLanes;
  while (lg < 5u && ((uint64_t)n << (lg + 1u)) <= stride) ++lg;
  return lg;
}

// The listed record of position i, pre: where each list starts.
__device__ __forceinline__ const float4* mid_record(const RasterArgs& A, const uint32_t* pre, uint32_t i) {
  uint32_t lo = 0, hi = kMidLists;  // pre[lo] <= i < pre[hi]
  while (hi - lo > 1u) {
    const uint32_t mid = (lo + hi) >> 1;
    if (pre[mid] <= i) lo = mid;
    else hi = mid;
  }
  return reinterpret_cast<const float4*>(A.cand + mid_base(A, lo) + (i - pre[lo]));
}

// One 16x16 tile of a queued record, by a warp.
struct PutTile {
  static __device__ __forceinline__ void run(const RasterArgs& A, const BigTri& q, uint32_t local) {
    const uint32_t lane = threadIdx.x & 31;
    const int px1 = q.px1, py1 = q.py1;
    const uint32_t tx_n = (uint32_t)((px1 - q.px0 + kBigTile) / kBigTile);
    const int bx = q.px0 + (int)(local % tx_n) * kBigTile, by = q.py0 + (int)(local / tx_n) * kBigTile;
    const uint32_t t = q.tri;
    const int px = bx + (int)(lane % kBigTile), py_first = by + (int)(lane / kBigTile);
    const int py_last = min(by + kBigTile - 1, py1);
    Put put;
    if (q.pad >> 31) {
      const Tri32 v{{q.X[0], q.X[1], q.X[2]}, {q.Y[0], q.Y[1], q.Y[2]}, {q.zn[0], q.zn[1], q.zn[2]}};
      const Edges32 E = edges32(v, px, py_first);
      int e0 = E.e[0], e1 = E.e[1], e2 = E.e[2];
      PutN<4> later;
      if (px <= px1)
        for (int py = py_first; py <= py_last;) {
          uint32_t key[4], pix[4];
          bool on[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            pix[i] = (uint32_t)py * (uint32_t)A.W + (uint32_t)px;
            on[i] = (e0 | e1 | e2) >= 0 && py <= py_last && key32(E, e0, e1, e2, v, key[i]);
            e0 += E.dy[0] * (32 / kBigTile);
            e1 += E.dy[1] * (32 / kBigTile);
            e2 += E.dy[2] * (32 / kBigTile);
            py += 32 / kBigTile;
          }
          later.put(A, t, on, key, pix);
        }
      later.check(A, t);
    } else {
      const SV a{q.X[0], q.Y[0], q.zn[0]}, b{q.X[1], q.Y[1], q.zn[1]}, c{q.X[2], q.Y[2], q.zn[2]};
      const int64_t Ar = (b.X - a.X) * (c.Y - a.Y) - (c.X - a.X) * (b.Y - a.Y);
      const float invA = __fdiv_rn(1.0f, ll2float_rn(Ar));
      const Edges E = edges_at(a, b, c, px, py_first);
      int64_t e[3] = {E.e[0], E.e[1], E.e[2]};
      if (px <= px1)
#pragma unroll 1
        for (int py = py_first; py <= py_last; py += 32 / kBigTile) {
          const bool in = (e[0] > 0 || (e[0] == 0 && E.tl[0])) && (e[1] > 0 || (e[1] == 0 && E.tl[1])) &&
                          (e[2] > 0 || (e[2] == 0 && E.tl[2]));
          if (in) {
            float s = __fmul_rn(ll2float_rn(e[0]), a.zn);
            s = __fadd_rn(s, __fmul_rn(ll2float_rn(e[1]), b.zn));
            s = __fadd_rn(s, __fmul_rn(ll2float_rn(e[2]), c.zn));
            const float d = __fmul_rn(s, invA);
            if (d >= -1.0f && d <= 1.0f) {
              put.put(A, (uint32_t)py * (uint32_t)A.W + (uint32_t)px, ordered(d), t);
            }
          }
          e[0] += E.dy[0] * (32 / kBigTile);
          e[1] += E.dy[1] * (32 / kBigTile);
          e[2] += E.dy[2] * (32 / kBigTile);
        }
    }
    put.check(A, t);
  }
};

// Where each mid-size list starts, pre[0] .. pre[kMidLists] (seen after a barrier).
__device__ __forceinline__ void mid_prefix(const RasterArgs& A, uint32_t* pre) {
  const uint32_t lane = threadIdx.x & 31;
  __syncthreads();  // pre of an earlier item of the same block is free
  if (threadIdx.x < 32) {
    uint32_t c = 0;
    if (lane < A.mid_lists) c = min(__ldcg(&A.ctr->n_mid[lane][0]), mid_base(A, lane + 1u) - mid_base(A, lane));
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= (unsigned)o) x += y;
    }
    pre[lane + 1] = x;
    if (lane == 0) pre[0] = 0u;
  }
}

// The queued tiles, a warp each, then the mid-size lists.  (No call of a function that is
// not inlined: with one in a branch that is never taken the mid-size boxes of a
// 3.2M-triangle floor take 440 us instead of 330.)
__device__ __forceinline__ void depth_win_body(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  __shared__ uint32_t pre[kMidLists + 1];
  const unsigned long long st = __ldcg(&A.ctr->big);
  if (threadIdx.x == 0) *ties_full() = 0u;
  mid_prefix(A, pre);  // (a barrier)
  for_tiles<PutTile>(A, st, bid, nblk);
  __syncthreads();
  const uint32_t n = pre[kMidLists], stride = nblk * blockDim.x;
  const uint32_t lg = mid_lanes(n, stride), sub = threadIdx.x & ((1u << lg) - 1u);
  for (uint32_t i = (bid * blockDim.x + threadIdx.x) >> lg; i < n; i += stride >> lg) {
    const float4* s = mid_record(A, pre, i);
    const float4 f0 = __ldcs(s), f1 = __ldcs(s + 1), f2 = __ldcs(s + 2);
    const Tri32 v{{__float_as_int(f0.x), __float_as_int(f0.z), __float_as_int(f1.x)},
                  {__float_as_int(f0.y), __float_as_int(f0.w), __float_as_int(f1.y)},
                  {f2.x, f2.y, f2.z}};
    const uint32_t b0 = __float_as_uint(f1.z), b1 = __float_as_uint(f1.w), t = __float_as_uint(f2.w);
    const int px0 = (int)(b0 & 0xFFFFu), py0 = (int)(b0 >> 16), px1 = (int)(b1 & 0xFFFFu), py1 = (int)(b1 >> 16);
    win_box<4, kPutLater>(A, v, t, px0, py0, px1, py1, (int)sub, 1 << lg);
  }
}

// Sets triangle t's visible bit.
__device__ __forceinline__ void win_mark(const RasterArgs& A, uint32_t t) {
  const uint32_t bit = 1u << (t & 31);
  if (__ldcg(A.vt + (t >> 5)) & bit) return;
  atomicOr(A.vt + (t >> 5), bit);
  note_tile(A, t >> 10);
}

// Whether triangle t is marked.
__device__ __forceinline__ bool marked(const RasterArgs& A, uint32_t t) {
  return (__ldcg(A.vt + (t >> 5)) >> (t & 31)) & 1u;
}

// A tile of the marking passes over the final keys.
template <int PASS>
struct MarkTile {
  static __device__ __forceinline__ void run(const RasterArgs& A, const BigTri& q, uint32_t local) {
    raster_tile<PASS, true>(A, q, local);
  }
};

__device__ __noinline__ void mark_tiles(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  for_tiles<MarkTile<1>>(A, __ldcg(&A.ctr->big), bid, nblk);
}

// The listed sub-triangles whose triangles are not marked, against the final keys.
__device__ __noinline__ void mark_mids(const RasterArgs& A, uint32_t bid, uint32_t nblk, const uint32_t* pre) {
  const uint32_t n = pre[kMidLists], stride = nblk * blockDim.x;
  const uint32_t lg = mid_lanes(n, stride), sub = threadIdx.x & ((1u << lg) - 1u);
  for (uint32_t i = (bid * blockDim.x + threadIdx.x) >> lg; i < n; i += stride >> lg) {
    const float4* s = mid_record(A, pre, i);
    const float4 f2 = __ldcs(s + 2);
    const uint32_t t = __float_as_uint(f2.w);
    if (marked(A, t)) continue;
    const float4 f0 = __ldcs(s), f1 = __ldcs(s + 1);
    const Tri32 v{{__float_as_int(f0.x), __float_as_int(f0.z), __float_as_int(f1.x)},
                  {__float_as_int(f0.y), __float_as_int(f0.w), __float_as_int(f1.y)},
                  {f2.x, f2.y, f2.z}};
    const uint32_t b0 = __float_as_uint(f1.z), b1 = __float_as_uint(f1.w);
    if (win_box<4, kTest>(A, v, t, (int)(b0 & 0xFFFFu), (int)(b0 >> 16), (int)(b1 & 0xFFFFu), (int)(b1 >> 16), (int)sub,
                          1 << lg))
      win_mark(A, t);
  }
}

// The marking pass when the tie list overflowed: every sub-triangle whose triangle is not
// marked is tested against the final keys, where the depth pass had it: the queued tiles,
// the mid-size lists, the small ones from their survivors and their clipped fans.
template <int NT>
__device__ __noinline__ void mark_all(const RasterArgs& A, uint32_t bid, uint32_t nblk, uint32_t* pre) {
  __shared__ uint32_t mid_pre[kMidLists + 1];
  mid_prefix(A, mid_pre);
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t n = surv_prefix<NT>(A, pre);  // (a barrier: mid_pre is written)
  mark_tiles(A, bid, nblk);
  mark_mids(A, bid, nblk, mid_pre);
  const uint32_t stride = nblk * blockDim.x;
  const bool full = (__ldcg(&A.ctr->big) >> 40) > A.queue_cap;
  for (uint32_t wbase = bid * blockDim.x + (threadIdx.x & ~31u); wbase < n; wbase += stride) {
    const uint32_t v = wbase + lane;
    if (v >= n) continue;
    const uint32_t i = surv_slot(A, pre, v, wbase);
    const uint32_t t = __ldcg(A.surv + i);
    if (marked(A, t)) continue;
    const float4* sc = A.surv_clip + 3 * (size_t)i;
    const WinSetup E = win_setup(A, __ldcs(sc), __ldcs(sc + 1), __ldcs(sc + 2));
    if (!E.live) continue;
    bool hit = false;
    if (!E.fits) {  // (queued, unless there was no room)
      const SV a{E.v.X[0], E.v.Y[0], E.v.z[0]}, b{E.v.X[1], E.v.Y[1], E.v.z[1]}, c{E.v.X[2], E.v.Y[2], E.v.z[2]};
      hit = full && win_rect64<true>(A, a, b, c, t, E.px0, E.py0, E.px1, E.py1, 0u, 1u);
    } else if ((E.px1 - E.px0 + 1) * (E.py1 - E.py0 + 1) <= kSmallMaxPix) {
      hit = win_box<4, kTest>(A, E.v, t, E.px0, E.py0, E.px1, E.py1, 0, 1);
    }
    if (hit) win_mark(A, t);
  }
  __syncthreads();  // pre is reused
  const uint32_t nc = region_prefix<NT>(A, A.clip_count, pre);
  const Mat4 M = A.Mdev ? load_mat(A.Mdev) : A.M;
  for (uint32_t i = bid * blockDim.x + threadIdx.x; i < nc; i += stride) {
    const uint32_t t = __ldcg(A.clip + surv_slot(A, pre, i, i));
    if (marked(A, t)) continue;
    const uint32_t* f = A.idx + 3 * (size_t)t;
    Fan fan;
    if (win_clipped<true>(A, t, load_clip(M, A.pos, __ldg(f)), load_clip(M, A.pos, __ldg(f + 1)),
                          load_clip(M, A.pos, __ldg(f + 2)), fan))
      win_mark(A, t);
  }
}

// Marking: the triangle of every pixel, then the listed ties whose key is the pixel's.
template <int NT>
__device__ __forceinline__ void mark_win_body(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  uint32_t* pre = region_pre();
  __shared__ int32_t s_status;
  __shared__ uint32_t s_ties;
  __syncthreads();  // the shared words of an earlier item of the same block are free
  if (threadIdx.x == 0) {
    s_status = __ldcg(&A.ctr->status);
    s_ties = __ldcg(&A.ctr->n_ties);
  }
  __syncthreads();
  if (s_status != 0) return;
  // A warp takes 64 x kR pixels, two side by side a thread in each row, the block's warps
  // one below the other.  A pixel whose left or upper neighbour has the same triangle is
  // passed over; what is left is looked up in a table of the triangles (and the tiles) the
  // block marked last, so that a triangle costs one atomic for all its pixels in a block.
  constexpr uint32_t kNone = 0xFFFFFFFFu;
  constexpr uint32_t kR = 4, kSeen = 1024, kSeenTiles = 64;
  __shared__ uint32_t seen[kSeen], seen_tile[kSeenTiles];
  for (uint32_t i = threadIdx.x; i < kSeen; i += blockDim.x) seen[i] = kNone;
  if (threadIdx.x < kSeenTiles) seen_tile[threadIdx.x] = kNone;
  __syncthreads();
  volatile uint32_t* vseen = seen;
  volatile uint32_t* vtile = seen_tile;
  const uint32_t lane = threadIdx.x & 31;
  constexpr uint32_t kRows = kR * (NT / 32);
  const uint32_t cols = ((uint32_t)A.W + 63u) / 64u, bands = ((uint32_t)A.H + kRows - 1u) / kRows;
  for (uint32_t g = bid; g < cols * bands; g += nblk) {
    const uint32_t x = (g % cols) * 64u + 2u * lane, y0 = (g / cols) * kRows + (threadIdx.x >> 5) * kR;
    uint2 q[2 * kR];  // (triangle, key)
#pragma unroll
    for (uint32_t r = 0; r < kR; ++r) {
      const uint2* z = reinterpret_cast<const uint2*>(A.zid) + (size_t)(y0 + r) * A.W + x;
      const bool row = y0 + r < (uint32_t)A.H;
      q[2 * r] = row && x < (uint32_t)A.W ? __ldcg(z) : make_uint2(kNone, kNone);
      q[2 * r + 1] = row && x + 1u < (uint32_t)A.W ? __ldcg(z + 1) : make_uint2(kNone, kNone);
    }
    uint32_t t[2 * kR];
#pragma unroll
    for (uint32_t r = 0; r < kR; ++r) {
      const uint32_t a = q[2 * r].y != kNone ? q[2 * r].x : kNone, b = q[2 * r + 1].y != kNone ? q[2 * r + 1].x : kNone;
      const uint32_t up_a = r && q[2 * r - 2].y != kNone ? q[2 * r - 2].x : kNone;
      const uint32_t up_b = r && q[2 * r - 1].y != kNone ? q[2 * r - 1].x : kNone;
      const uint32_t left = __shfl_up_sync(0xFFFFFFFFu, b, 1);
      t[2 * r] = (lane && left == a) || up_a == a ? kNone : a;
      t[2 * r + 1] = b == a || up_b == b ? kNone : b;
    }
#pragma unroll
    for (uint32_t u = 0; u < 2 * kR; ++u) {
      const uint32_t m = t[u];
      if (m == kNone || vseen[m % kSeen] == m) continue;
      vseen[m % kSeen] = m;
      atomicOr(A.vt + (m >> 5), 1u << (m & 31));
      const uint32_t tile = m >> 10;
      if (vtile[tile % kSeenTiles] == tile) continue;
      vtile[tile % kSeenTiles] = tile;
      note_tile(A, tile);
    }
  }
  if (s_ties > kTies) {
    // (conservative marking tests what is not marked anyway; the blocks of the first wave
    // alone, so that no share of the tests waits for the second)
    const uint32_t share = min(nblk, kMarkBlocks);
    if (!A.cons && bid < share) mark_all<NT>(A, bid, share, pre);
    return;
  }
  const uint32_t stride = nblk * blockDim.x;
  for (uint32_t i = bid * blockDim.x + threadIdx.x; i < s_ties; i += stride) {
    const uint4 e = __ldcg(A.ties + i);
    if (zkey(A, e.x) == e.y) {
      win_mark(A, e.z);
      win_mark(A, e.w);
    }
  }
}

// Conservative marking after the winners': the triangles that the samples marked are
// marked already (a covered centre's depth is the sample's), so only the other survivors
// are tested, each pixel of their conservative boxes against the final keys (as
// sample<2>).  Boxes above kMidPix pixels and clipped triangles' are the queued tiles, a
// warp each, as in two rasterizations: a hidden triangle is looked at whole, and one that
// fills a 1080p window takes a warp 18 ms and, clipped, a thread 0.77 s (by tiles 29 and 33
// us).  Of the others those of at most kSmallMaxPix pixels are tested in-thread and larger
// ones by the warp together when there are many survivors; with few, a warp takes few of
// them, all together.  Edge functions in 32 bits, stepped, as in win_box (an edge's largest
// value over a pixel's square is half a step each way from the centre's: 2 % more).
// (Conservative marking of 60 patches at 1080p 182 us with 64-bit edge functions set up at
// every pixel, 100 so; of 200 icospheres, 4.1M triangles, 216 and 66; a 1,024-thread block
// of the persistent kernel has four pixels' keys on their way, its frame of the latter 466
// -> 424 us.)
__device__ __forceinline__ bool cons_box(const RasterArgs& A, const SV& a, const SV& b, const SV& c, int px0, int py0,
                                         int px1, int py1, uint32_t first, uint32_t step) {
  const int64_t Ar = (b.X - a.X) * (c.Y - a.Y) - (c.X - a.X) * (b.Y - a.Y);
  const float invA = __fdiv_rn(1.0f, ll2float_rn(Ar));
  const float zmin = fminf(a.zn, fminf(b.zn, c.zn)), zmax = fmaxf(a.zn, fmaxf(b.zn, c.zn));
  const uint32_t w = (uint32_t)(px1 - px0 + 1), n = w * (uint32_t)(py1 - py0 + 1);
  for (uint32_t s = first; s < n; s += step) {
    const int px = px0 + (int)(s % w), py = py0 + (int)(s / w);
    const Edges E = edges_at(a, b, c, px, py);
    bool meets = true, in = true;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int64_t ax = E.dx[i] < 0 ? -E.dx[i] : E.dx[i], ay = E.dy[i] < 0 ? -E.dy[i] : E.dy[i];
      meets = meets && E.e[i] + ((ax + ay) >> 1) >= 0;
      in = in && (E.e[i] > 0 || (E.e[i] == 0 && E.tl[i]));
    }
    if (!meets) continue;
    float f = __fmul_rn(ll2float_rn(E.e[0]), a.zn);
    f = __fadd_rn(f, __fmul_rn(ll2float_rn(E.e[1]), b.zn));
    f = __fadd_rn(f, __fmul_rn(ll2float_rn(E.e[2]), c.zn));
    float d = __fmul_rn(f, invA);
    if (!in) d = fminf(fmaxf(d, zmin), zmax);
    if (!(d >= -1.0f && d <= 1.0f)) continue;
    if (ordered(d) <= zkey(A, (uint32_t)py * (uint32_t)A.W + (uint32_t)px)) return true;
  }
  return false;
}

template <int N>
__device__ __forceinline__ bool cons_box32(const RasterArgs& A, const Tri32& v, int px0, int py0, int px1, int py1,
                                           int first, int step) {
  const int w = px1 - px0 + 1, n = w * (py1 - py0 + 1);
  if (first >= n) return false;
  const int sy = step == 1 ? (w == 1 ? 1 : 0) : step / w, sx = step - sy * w;  // step = sy rows and sx < w pixels
  const int fy = first / w, fx = first - fy * w;
  const Edges32 E = edges32(v, px0 + fx, py0 + fy);
  const float zmin = fminf(v.z[0], fminf(v.z[1], v.z[2])), zmax = fmaxf(v.z[0], fmaxf(v.z[1], v.z[2]));
  int e[3], in_row[3], past[3], half[3];  // half: from a centre's (reduced) value to the square's largest
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    e[i] = E.e[i];
    in_row[i] = E.dy[i] * sy + E.dx[i] * sx;
    past[i] = in_row[i] + E.dy[i] - E.dx[i] * w;
    half[i] = ((abs(E.dx[i]) + abs(E.dy[i])) >> 1) + E.nb[i];
  }
  const uint32_t ap = (uint32_t)(A.W * sy + sx), bp = ap + (uint32_t)(A.W - w);
  uint32_t p = (uint32_t)(py0 + fy) * (uint32_t)A.W + (uint32_t)(px0 + fx);
  for (int left = n - 1 - first, col = w - fx; left >= 0;) {
    uint32_t key[N], pix[N];
    bool on[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      pix[i] = p;
      on[i] = ((e[0] + half[0]) | (e[1] + half[1]) | (e[2] + half[2]) | left) >= 0;
      float f = __fmul_rn(__int2float_rn(e[0] + E.nb[0]), v.z[0]);
      f = __fadd_rn(f, __fmul_rn(__int2float_rn(e[1] + E.nb[1]), v.z[1]));
      f = __fadd_rn(f, __fmul_rn(__int2float_rn(e[2] + E.nb[2]), v.z[2]));
      float d = __fmul_rn(f, E.invA);
      if ((e[0] | e[1] | e[2]) < 0) d = fminf(fmaxf(d, zmin), zmax);
      on[i] = on[i] && d >= -1.0f && d <= 1.0f;
      key[i] = ordered(d);
      col -= sx;
      const bool wrap = col <= 0;
      col += wrap ? w : 0;
      p += wrap ? bp : ap;
#pragma unroll
      for (int k = 0; k < 3; ++k) e[k] += wrap ? past[k] : in_row[k];
      left -= step;
    }
    if (test_n(A, on, key, pix)) return true;
  }
  return false;
}

// The sub-triangles of a triangle that must be clipped (rare) that are not queued.
__device__ __noinline__ bool cons_clipped(const RasterArgs& A, float4 c0, float4 c1, float4 c2, bool full) {
  CV poly[kMaxPoly];
  poly[0] = CV{c0.x, c0.y, c0.z, c0.w};
  poly[1] = CV{c1.x, c1.y, c1.z, c1.w};
  poly[2] = CV{c2.x, c2.y, c2.z, c2.w};
  const int n = clip_polygon(poly, 3);
  if (n < 3) return false;
  for (int i = 0; i < n; ++i)
    if (!(poly[i].w > 0.0f)) return false;
  SV sv[kMaxPoly];
  for (int i = 0; i < n; ++i) sv[i] = project(poly[i], A.hx, A.hy);
  for (int i = 1; i + 1 < n; ++i) {
    const Setup s = setup(sv[0], sv[i], sv[i + 1], A.W, A.H, true);
    if (s.A <= 0 || s.px1 < s.px0 || s.py1 < s.py0) continue;
    if (!full && (s.px1 - s.px0 + 1) * (s.py1 - s.py0 + 1) > kSmallMaxPix) continue;
    if (cons_box(A, sv[0], sv[i], sv[i + 1], s.px0, s.py0, s.px1, s.py1, 0u, 1u)) return true;
  }
  return false;
}

template <int NT>
__device__ __forceinline__ void mark_cons_body(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  if (!A.win || !A.cons) return;
  uint32_t* pre = region_pre();
  __shared__ int32_t s_cons_status;
  if (threadIdx.x == 0) s_cons_status = __ldcg(&A.ctr->status);
  __syncthreads();
  if (s_cons_status != 0) return;
  // (a queue that has no more room: large ones that found no record are tested here)
  const bool full = (__ldcg(&A.ctr->big) >> 40) > A.queue_cap;
  const int most = full ? 0x7FFFFFFF : kMidPix;
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t n = surv_prefix<NT>(A, pre);
  const uint32_t stride = nblk * blockDim.x, warp = (bid * blockDim.x + threadIdx.x) >> 5, nwarps = stride >> 5;
  uint32_t per = 32;  // survivors a warp takes at a time
  while (per > 1u && (uint64_t)n * 32u <= (uint64_t)nwarps * per * 16u) per >>= 1;
  // (a warp's first share by its index, the next ones from a counter, claimed ahead: shares
  // differ by an order of magnitude, and a block waits for its slowest warp)
  for (uint32_t share = warp; (uint64_t)share * per < n;) {
    const uint32_t base = share * per, v = base + lane;
    uint32_t claimed = 0;
    if (lane == 0) claimed = atomicAdd(&A.ctr->cons_item, 1u);
    WinSetup E = {};
    uint32_t t = 0;
    bool vis = false, big = false;
    if (lane < per && v < n) {
      const uint32_t i = surv_slot(A, pre, v, base);
      t = __ldcg(A.surv + i);
      if (!marked(A, t)) {
        const float4* sc = A.surv_clip + 3 * (size_t)i;
        E = win_setup(A, __ldcs(sc), __ldcs(sc + 1), __ldcs(sc + 2));
        const int pix = E.front ? cons_pixels(A, E) : 0;
        if (pix > 0 && pix <= most) {
          big = pix > (per < 32u ? 1 : kSmallMaxPix) || !E.fits;
          if (!big) vis = cons_box32<(NT > 256 ? 4 : 1)>(A, E.v, E.px0, E.py0, E.px1, E.py1, 0, 1);
        }
      }
    }
    for (uint32_t m = __ballot_sync(0xFFFFFFFFu, big); m; m &= m - 1u) {  // the warp together
      const int src = __ffs(m) - 1;
      Tri32 q;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        q.X[j] = __shfl_sync(0xFFFFFFFFu, E.v.X[j], src);
        q.Y[j] = __shfl_sync(0xFFFFFFFFu, E.v.Y[j], src);
        q.z[j] = __shfl_sync(0xFFFFFFFFu, E.v.z[j], src);
      }
      const int px0 = __shfl_sync(0xFFFFFFFFu, E.px0, src), py0 = __shfl_sync(0xFFFFFFFFu, E.py0, src);
      const int px1 = __shfl_sync(0xFFFFFFFFu, E.px1, src), py1 = __shfl_sync(0xFFFFFFFFu, E.py1, src);
      bool hit;
      if (fits32(q)) {
        hit = cons_box32<1>(A, q, px0, py0, px1, py1, (int)lane, 32);
      } else {
        const SV a{q.X[0], q.Y[0], q.z[0]}, b{q.X[1], q.Y[1], q.z[1]}, c{q.X[2], q.Y[2], q.z[2]};
        hit = cons_box(A, a, b, c, px0, py0, px1, py1, lane, 32u);
      }
      if (__any_sync(0xFFFFFFFFu, hit) && (int)lane == src) vis = true;
    }
    if (vis) win_mark(A, t);
    share = nwarps + __shfl_sync(0xFFFFFFFFu, claimed, 0);
  }
  __syncthreads();  // pre is reused
  const uint32_t nc = region_prefix<NT>(A, A.clip_count, pre);
  const Mat4 M = A.Mdev ? load_mat(A.Mdev) : A.M;
  for (uint32_t i = bid * blockDim.x + threadIdx.x; i < nc; i += stride) {
    const uint32_t t = __ldcg(A.clip + surv_slot(A, pre, i, i));
    if (marked(A, t)) continue;
    const uint32_t* f = A.idx + 3 * (size_t)t;
    if (cons_clipped(A, load_clip(M, A.pos, __ldg(f)), load_clip(M, A.pos, __ldg(f + 1)),
                     load_clip(M, A.pos, __ldg(f + 2)), full))
      win_mark(A, t);
  }
}

// ... and of the queued tiles.  (A call of it in the body above takes that one's registers:
// in the kernel it is inlined after it, in the persistent kernel a function beside it.)
__device__ __forceinline__ void mark_cons_tiles(const RasterArgs& A, uint32_t bid, uint32_t nblk) {
  if (!A.win || !A.cons || __ldcg(&A.ctr->status) != 0) return;
  for_tiles<MarkTile<2>>(A, __ldcg(&A.ctr->big), bid, nblk);
}

inline void set_raster_mode(RasterArgs& A);

// The arguments of one visibility pass on ctx (host side).  front_blocks blocks of
// `threads` threads run the front end; each owns a survivor region large enough for
// every triangle it can see.
inline RasterArgs make_raster_args(fa_ctx* ctx, const fa_mesh* mesh, const Mat4& M, uint32_t W, uint32_t H,
                                   uint32_t* vt, bool reset_status, const float* Mdev, bool cons,
                                   int32_t* tri_chart_init, uint32_t front_blocks, uint32_t threads) {
  RasterArgs A;
  A.cons = cons ? 1 : 0;
  A.Mdev = Mdev;
  A.M = M;
  A.pos = mesh->pos;
  A.idx = mesh->idx;
  A.T = mesh->T;
  A.W = (int)W;
  A.H = (int)H;
  A.hx = 0.5f * (float)W;
  A.hy = 0.5f * (float)H;
  A.zbuf = ctx->zbuf;
  A.queue = ctx->queue;
  A.queue_cap = ctx->queue_cap;
  A.tile_owner = ctx->tile_owner;
  A.tile_cap = ctx->tile_cap;
  A.cand = reinterpret_cast<CandTri*>(ctx->cand);
  A.cand_cap = ctx->cand_cap;
  A.surv = ctx->surv;
  A.surv_count = ctx->surv_count;
  A.front_blocks = front_blocks;
  {
    const uint32_t iters = (mesh->T + front_blocks * threads - 1) / (front_blocks * threads);
    A.surv_per_block = iters * threads;
  }
  A.clip_base = A.front_blocks * A.surv_per_block;
  A.surv_clip = reinterpret_cast<float4*>(ctx->surv_clip);
  A.tile_flag = ctx->tile_flag;
  A.tile_list = ctx->tile_list;
  A.clip_count = ctx->clip_count;
  A.blockcnt = ctx->blockcnt;
  A.viscnt = ctx->viscnt;
  A.ntiles = (mesh->T + 1023) / 1024;
  A.reset_status = reset_status ? 1 : 0;
  A.tri_chart = tri_chart_init;
  A.partial_clear = nullptr;
  A.mid_max_pix = ctx->mid_max_pix;
  A.zmax = (ctx->raster_flags & FA_RASTER_HIZ) ? ctx->zmax : nullptr;
  A.ztx = (int)((W + 15) / 16);
  A.clip = ctx->clip;
  A.ctr = ctx->ctr;
  A.vt = vt;
  A.zid = reinterpret_cast<unsigned long long*>(ctx->zbuf);
  A.ties = ctx->ties;
  set_raster_mode(A);
  return A;
}

// The tile-depth option belongs to the second rasterization and keeps it.
inline void set_raster_mode(RasterArgs& A) { A.win = A.zmax ? 0 : 1; }

// The exact pass's grid (blocks of `threads` threads), from which the mid-size lists get
// their shares: a block sees at most mid_per_block survivors.
inline void set_exact_grid(RasterArgs& A, uint32_t blocks, uint32_t threads) {
  A.mid_blocks = blocks;
  A.mid_lists = blocks < (uint32_t)kMidLists ? blocks : (uint32_t)kMidLists;
  A.mid_per_block = (uint32_t)(((uint64_t)A.T + (uint64_t)blocks * threads - 1) / ((uint64_t)blocks * threads)) * threads;
}

}  // namespace
}  // namespace rs
}  // namespace fa
