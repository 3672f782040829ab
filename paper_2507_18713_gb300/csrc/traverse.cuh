// traverse.cuh -- per-ray device code shared by the forward and adjoint
// kernels: sensor ray generation (Fig. 2, Sec. V-C), traversal of the sparse
// voxel structure (Sec. III-B), record loads and the local fields of
// Eq. 1, 2, 5, 6.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "salf_internal.h"

namespace salf {

constexpr float kPi = 3.14159265358979323846f;
constexpr float kSH0 = 0.28209479177387814f;  // 1 / (2 sqrt(pi))
constexpr float kSH1 = 0.48860251190291992f;  // sqrt(3) / (2 sqrt(pi))

struct Ray {
  int Oi[3];     // origin, finest-cell units: Oi + Of
  float Of[3];
  float d[3];    // unit direction, world frame
  float tn, tf;  // metres
  float s;       // time fraction (t - t0) / (t1 - t0) of the ray's pose
  bool valid;
};

// Sums and products of floats with their rounding errors (Dekker 1971, Knuth's
// TwoSum): pairs hi + lo carry about 48 bits.  The _rn forms are never contracted.
struct Pair {
  float hi, lo;
};

__device__ __forceinline__ Pair two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  return Pair{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}

__device__ __forceinline__ Pair pair_add(Pair a, Pair b) {
  const Pair s = two_sum(a.hi, b.hi);
  return two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}

__device__ __forceinline__ Pair pair_mul(Pair a, const float b[2]) {
  const float p = __fmul_rn(a.hi, b[0]);
  const float e = __fmaf_rn(a.hi, b[0], -p);
  return two_sum(p, __fmaf_rn(a.hi, b[1], __fmaf_rn(a.lo, b[0], e)));
}

// Cells are counted from a ray's origin, so a box plane's distance from the
// origin's cell has to fit an int whichever way the axis is mirrored: cells end
// there, 2^23 short of the int range (a grid's planes lie within 2^22 of 0).
constexpr int kFarCell = 0x7f800000;

// A pair as an int and a fraction in [0, 1] (1: less than 1 by under 2^-25).
// Where it is beyond kFarCell: there, and no fraction.  `about` is its value to
// one float, which may be infinite (the pair is NaN then).
__device__ __forceinline__ int pair_floor(Pair a, float about, float* frac) {
  if (fabsf(about) >= (float)kFarCell) {
    *frac = 0.f;
    return about < 0.f ? -kFarCell : kFarCell;
  }
  const float f = floorf(a.hi);
  const float r = __fadd_rn(__fsub_rn(a.hi, f), a.lo);
  const float k = floorf(r);  // -1 where hi is whole and lo below it; more from 2^25 on
  *frac = __fsub_rn(r, k);
  return (int)f + (int)k;
}

// Sensor ray of pixel (u, v) / LiDAR (azimuth u, beam v).  EXPL: explicit rays may
// come (their code costs the others registers).
template <bool EXPL = true>
__device__ __forceinline__ void gen_ray(const ReqDev& Q, const DevScene& S, int u, int v,
                                        int ray, Ray& r) {
  r.valid = true;
  if (EXPL && Q.kind == SALF_RAYS_EXPLICIT) {
    const float4* q = reinterpret_cast<const float4*>(Q.rays) + 2 * (size_t)ray;
    float4 a = __ldg(q), b = __ldg(q + 1);
    // origin in finest cells, (o - origin) / edge, to 48 bits
    const float o[3] = {a.x, a.y, a.z};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const Pair d = pair_add(Pair{o[k], 0.f}, Pair{-S.origin2[k][0], -S.origin2[k][1]});
      r.Oi[k] = pair_floor(pair_mul(d, S.isf2), __fmul_rn(d.hi, S.isf2[0]), &r.Of[k]);
    }
    float dx = a.w, dy = b.x, dz = b.y;
    float nn = dx * dx + dy * dy + dz * dz;
    r.valid = nn > 0.f;
    float inv = nn > 0.f ? rsqrtf(nn) : 0.f;
    r.d[0] = dx * inv;
    r.d[1] = dy * inv;
    r.d[2] = dz * inv;
    r.tn = b.z;
    r.tf = b.w > 0.f ? b.w : __int_as_float(0x7f800000);
    r.s = 0.f;
    return;
  }
  float dc[3];
  float s = 0.f;
  if (Q.kind == SALF_LIDAR_SPIN) {
    float e = Q.elev_max - (float)v * Q.elev_step;
    float se, ce, sp, cp;
    sincosf(e, &se, &ce);
    // azimuth 2 pi u / W as sin/cos(pi x) with x = 2u/W: no rounding of 2 pi
    sincospif(2.f * (float)u / (float)Q.W, &sp, &cp);
    dc[0] = ce * cp;
    dc[1] = ce * sp;
    dc[2] = se;
    if (Q.moving) s = (float)u / (float)Q.W;
  } else {
    float px = (float)u + 0.5f, py = (float)v + 0.5f;
    if (Q.kind == SALF_PINHOLE) {
      dc[0] = (px - Q.cx) * Q.inv_fx;
      dc[1] = (py - Q.cy) * Q.inv_fy;
      dc[2] = 1.f;
    } else if (Q.kind == SALF_FISHEYE_EQUIDIST) {
      float mx = (px - Q.cx) * Q.inv_fx, my = (py - Q.cy) * Q.inv_fy;
      float th = sqrtf(mx * mx + my * my);
      r.valid = th <= Q.half_fov;
      float st, ct;
      sincosf(th, &st, &ct);
      float k = th > 0.f ? st / th : 1.f;
      dc[0] = k * mx;
      dc[1] = k * my;
      dc[2] = ct;
    } else {  // equirectangular panorama
      // longitude 2 pi (px / W - 0.5) as sin/cos(pi x): no rounding of 2 pi
      float lat = Q.elev_max - (py / (float)Q.H) * (Q.elev_max - Q.elev_min);
      float sl, cl, sa, ca;
      sincospif(2.f * px / (float)Q.W - 1.f, &sl, &cl);
      sincosf(lat, &sa, &ca);
      dc[0] = ca * sl;
      dc[1] = -sa;
      dc[2] = ca * cl;
    }
    if (Q.moving) s = (float)v / (float)(Q.H - 1);
  }
  float d0 = Q.R0[0] * dc[0] + Q.R0[1] * dc[1] + Q.R0[2] * dc[2];
  float d1 = Q.R0[3] * dc[0] + Q.R0[4] * dc[1] + Q.R0[5] * dc[2];
  float d2 = Q.R0[6] * dc[0] + Q.R0[7] * dc[1] + Q.R0[8] * dc[2];
  if (s > 0.f && Q.rel_angle != 0.f) {
    // Rodrigues rotation by alpha about k: d + sin(a) (k x d) + (1 - cos(a)) k x (k x d)
    const float a = s * Q.rel_angle;
    float sh, ch;
    sincosf(0.5f * a, &sh, &ch);
    const float sa = 2.f * sh * ch, omc = 2.f * sh * sh;
    const float kx = Q.rel_axis[0], ky = Q.rel_axis[1], kz = Q.rel_axis[2];
    const float cx = ky * d2 - kz * d1, cy = kz * d0 - kx * d2, cz = kx * d1 - ky * d0;
    const float ccx = ky * cz - kz * cy, ccy = kz * cx - kx * cz, ccz = kx * cy - ky * cx;
    d0 = fmaf(omc, ccx, fmaf(sa, cx, d0));
    d1 = fmaf(omc, ccy, fmaf(sa, cy, d1));
    d2 = fmaf(omc, ccz, fmaf(sa, cz, d2));
  }
  float inv = rsqrtf(d0 * d0 + d1 * d1 + d2 * d2);
  r.d[0] = d0 * inv;
  r.d[1] = d1 * inv;
  r.d[2] = d2 * inv;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r.Oi[k] = Q.Oi[k];
    r.Of[k] = fmaf(s, Q.dO[k], Q.Of[k]);
  }
  r.tn = Q.t_near;
  r.tf = Q.t_far;
  r.s = s;
}

// gen_ray for a pinhole camera with one pose for the whole frame (no rolling
// shutter): the same arithmetic as gen_ray's pinhole branch, without the other
// sensor kinds' code, for kernels that serve only such cameras.
__device__ __forceinline__ void gen_ray_pinhole(const ReqDev& Q, int u, int v, Ray& r) {
  r.valid = true;
  const float px = (float)u + 0.5f, py = (float)v + 0.5f;
  const float dc0 = (px - Q.cx) * Q.inv_fx, dc1 = (py - Q.cy) * Q.inv_fy, dc2 = 1.f;
  const float d0 = Q.R0[0] * dc0 + Q.R0[1] * dc1 + Q.R0[2] * dc2;
  const float d1 = Q.R0[3] * dc0 + Q.R0[4] * dc1 + Q.R0[5] * dc2;
  const float d2 = Q.R0[6] * dc0 + Q.R0[7] * dc1 + Q.R0[8] * dc2;
  const float inv = rsqrtf(d0 * d0 + d1 * d1 + d2 * d2);
  r.d[0] = d0 * inv;
  r.d[1] = d1 * inv;
  r.d[2] = d2 * inv;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r.Oi[k] = Q.Oi[k];
    r.Of[k] = Q.Of[k];  // fmaf(0, dO, Of) in gen_ray
  }
  r.tn = Q.t_near;
  r.tf = Q.t_far;
  r.s = 0.f;
}

// Debug dump of a generated ray: world origin, unit direction, time, valid.
__device__ __forceinline__ void dump_ray(const ReqDev& Q, const DevScene& S, const Ray& r, int ray) {
  float* p = Q.ray_dump + 8 * (size_t)ray;
  const double sf = 1.0 / S.inv_sfin;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    p[k] = (float)(S.origin[k] + ((double)r.Oi[k] + (double)r.Of[k]) * sf);
    p[3 + k] = r.d[k];
  }
  p[6] = Q.time0 + r.s * (Q.time1 - Q.time0);
  p[7] = r.valid ? 1.f : 0.f;
}

// A ray's direction in finest cells per metre and its interval inside the
// tight box of the voxels (no hit can lie outside it).  Zero direction
// components become 1e-20.
struct RayClip {
  float D[3], invD[3];
  float t0, t1;
};

__device__ __forceinline__ void ray_clip(const DevScene& S, const Ray& r, RayClip& q) {
  const float isf = S.isf2[0];
  q.t0 = r.tn;
  q.t1 = r.tf;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float D = r.d[a] * isf;
    if (fabsf(D) < 1e-20f) D = 1e-20f;
    q.D[a] = D;
    q.invD[a] = 1.f / D;
    const float lo = ((float)(S.bmin[a] - r.Oi[a]) - r.Of[a]) * q.invD[a];
    const float hi = ((float)(S.bmax[a] - r.Oi[a]) - r.Of[a]) * q.invD[a];
    q.t0 = fmaxf(q.t0, fminf(lo, hi));
    q.t1 = fminf(q.t1, fmaxf(lo, hi));
  }
}

// Traversal state of one ray.  Axes along which the ray travels downwards are
// mirrored (plane p -> -p, cell c -> ~c, so the cell between planes c and c + 1
// stays the one between its mirrored planes): every ray then travels upwards
// on all three axes, a box is always left through its upper planes, and no
// step selects planes by sign.  Mirroring negates both the plane offset
// (p - Oi) - Of and 1 / D, so every distance is the unmirrored one bit for
// bit.  Positions are relative to the origin cell Oi, so plane distances are
// small integers minus a fraction.
struct Walk {
  int Oi[3];      // origin cell, mirrored
  float Of[3];    // origin inside it, mirrored
  float D[3];     // |direction| in finest cells per metre
  float invD[3];  // metres per finest cell
  int r[3];       // current finest cell, mirrored, relative to Oi
  unsigned neg;   // bit a: axis a is mirrored
  const unsigned short* skip;  // skip boxes of the ray's octant, at mirrored brick (0, 0, 0)
  unsigned box;   // AHEAD: skip box of the current brick
  uint4 word;     // AHEAD: occupancy word of the current block
  float t;        // entry distance of the current cell
  float tend;     // min(t_far, exit of the voxels' tight box)
  bool alive;
};

// 0 or all ones: axis a of the walk is mirrored.
__device__ __forceinline__ int mirror_mask(const Walk& w, int a) {
  return (int)(w.neg << (31 - a)) >> 31;
}

// x of a mirrored axis is -x.
__device__ __forceinline__ float unmirror(const Walk& w, int a, float x) {
  return __uint_as_float(__float_as_uint(x) ^ ((w.neg << (31 - a)) & 0x80000000u));
}

// Occupancy word of the 4x4x4 block that holds finest cell (ix, iy, iz).
__device__ __forceinline__ uint4 block_word(const DevScene& S, int ix, int iy, int iz) {
  const int k = S.K + 2;
  return __ldg(&S.mask0[(unsigned)(iz >> k) * (unsigned)S.mdim01 +
                        (unsigned)(iy >> k) * (unsigned)S.mdim0 + (unsigned)(ix >> k)]);
}

// The skip box and the occupancy word of the walk's cell, read ahead of its next step.
__device__ __forceinline__ void walk_read_ahead(const DevScene& S, Walk& w) {
  int c[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) c[a] = w.r[a] + w.Oi[a];
  w.box = __ldg(w.skip + ((long long)(c[2] >> S.skip_sz) * S.skip_n01 +
                          ((c[1] >> S.skip_sx) * S.skip_n0 + (c[0] >> S.skip_sx))));
  w.word = block_word(S, c[0] ^ mirror_mask(w, 0), c[1] ^ mirror_mask(w, 1),
                      c[2] ^ mirror_mask(w, 2));
}

// (Re)start a walk at distance t: the cell holding the point there, kept
// inside the tight box of the voxels.  AHEAD (here and below): see next_hit.
template <bool AHEAD = false>
__device__ __forceinline__ void walk_seek(const DevScene& S, Walk& w, float t) {
  w.t = t;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int m = mirror_mask(w, a);
    const int Oi = m ? -w.Oi[a] : w.Oi[a];
    const int q = Oi + __float2int_rd(unmirror(w, a, fmaf(t, w.D[a], w.Of[a])));
    w.r[a] = (min(max(q, S.bmin[a]), max(S.bmax[a] - 1, S.bmin[a])) ^ m) - w.Oi[a];
  }
  if (AHEAD && w.alive) walk_read_ahead(S, w);
}

template <bool AHEAD = false>
__device__ __forceinline__ void walk_init(const DevScene& S, const Ray& r, Walk& w) {
  RayClip q;
  ray_clip(S, r, q);
  w.neg = 0u;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const bool neg = q.D[a] < 0.f;
    w.neg |= neg ? 1u << a : 0u;
    w.Oi[a] = neg ? -r.Oi[a] : r.Oi[a];
    w.Of[a] = neg ? -r.Of[a] : r.Of[a];
    w.D[a] = fabsf(q.D[a]);
    w.invD[a] = fabsf(q.invD[a]);
  }
  w.skip = S.skip_oct[w.neg];
  w.alive = r.valid && (q.t0 < q.t1);
  w.tend = q.t1;
  walk_seek<AHEAD>(S, w, q.t0);
}

__device__ __forceinline__ void prefetch_l1(const void* p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

// The voxel owning finest cell (ix, iy, iz), or -1 if the cell is empty; w is its
// block's word.  *lx, *lz = log2 of the edges (x and y; z), in finest cells, of the
// aligned box around the cell that lies in that voxel or is empty.
__device__ __forceinline__ int find_leaf(const DevScene& S, const uint4 w, int ix, int iy, int iz,
                                         int* lx, int* lz) {
  const int K = S.K;
  const int cx = ix >> K, cy = iy >> K, cz = iz >> K;
  // Morton bit of the cell inside its 4x4x4 block: z1 picks the word, then y1,
  // x1, z0 the nibble of its 2x2x1 square, y0, x0 the bit
  const unsigned half = (cz & 2) ? w.y : w.x;
  const unsigned sh = ((cz & 1) << 2) | ((cx & 2) << 2) | ((cy & 2) << 3);
  const unsigned bit = sh | (cx & 1) | ((cy & 1) << 1);
  if ((half >> bit) & 1u) {
    const unsigned pre = __popc(half & ((1u << bit) - 1u)) + ((cz & 2) ? __popc(w.x) : 0);
    if (w.w != 0xffffffffu) {  // block of level-0 voxels: no cell-table read
      *lx = *lz = K;
      return (int)(w.w + pre);
    }
    const int2 en = __ldg(&S.cells[w.z + pre]);
    int e = en.x;
    int l = K;
    if (en.y) {  // split once: child voxel by rank, no node read
      l = K - 1;
      const unsigned ch = ((ix >> l) & 1) | (((iy >> l) & 1) << 1) | (((iz >> l) & 1) << 2);
      const unsigned cm = (unsigned)en.y;
      e = ((cm >> ch) & 1u) ? e + __popc(cm & ((1u << ch) - 1u)) : -1;
    }
    while (e <= -2) {
      --l;
      const int ch = ((ix >> l) & 1) | (((iy >> l) & 1) << 1) | (((iz >> l) & 1) << 2);
      e = __ldg(&S.nodes[(unsigned)(-2 - e) * 8u + (unsigned)ch]);
    }
    *lx = *lz = l;
    return e;
  }
  *lx = ((half >> sh) & 15u) ? K : K + 1;
  *lz = K;
  // bricks larger than a layer of a block (very large grids) may hold empty blocks
  if (S.skip_coarse && !(w.x | w.y)) *lx = *lz = K + 2;
  return -1;
}

__device__ __forceinline__ int find_leaf(const DevScene& S, int ix, int iy, int iz, int* lx,
                                         int* lz) {
  return find_leaf(S, block_word(S, ix, iy, iz), ix, iy, iz, lx, lz);
}

struct Hit {
  int vox;
  int lo[3];  // min corner, mirrored, relative to the origin cell
  int ls;
  float tin, tout;
};

// Distance at which the ray enters a hit's box, not before t0 (where its walk
// from the start began): the same formula as the entry next_hit reports, but
// independent of where a walk started, so every walk of one ray agrees on it.
__device__ __forceinline__ float hit_entry(const Walk& w, const Hit& h, float t0) {
  float t = t0;
#pragma unroll
  for (int a = 0; a < 3; ++a) t = fmaxf(t, ((float)h.lo[a] - w.Of[a]) * w.invD[a]);
  return t;
}

// Advance `w` by one structure step toward the next voxel crossed with
// positive length; true if this step found it (in h).  The caller's warp
// composites the lanes that found one, then calls again: one step per call
// keeps lanes of different rays in step, so a warp costs about its heaviest
// ray, not the sum of per-round maxima (two or three steps per call measured
// slower, and the loop for them cost 1-3% even when it ran once).
//
// A step reads the skip box of the current brick for the ray's octant (2
// bytes).  An empty brick's box reaches up to 31 x 31 x 63 bricks ahead in the
// ray's own directions; a brick that holds voxels has no box, and the cell is
// located in its block (find_leaf).  Either way the box is left through its
// nearest upper plane; the other coordinates come from the exit point, kept
// inside the box and never moved backwards.
//
// Every step ends inside the skip array: boxes end inside it, the start is
// inside the tight box, and a ray whose exit plane is not before the tight
// box's (te >= tend) takes no further step.  The exit axis always advances, so
// a walk ends after at most the array's cells per axis.
//
// AHEAD: a step ends by reading the next cell's box and word, so the reads run while
// the warp composites the step's hits, for five registers and a few instructions more:
// where the walk waits for memory (the adjoint; frames of few rays: fisheye 1080p 295 ->
// 276 us, camera 640x480 -10 to -17%), not where it is bound by issue (camera 1080p 258
// -> 265) or by registers (LiDAR spans 233 -> 241).
template <int DT, bool AHEAD = false>
__device__ __forceinline__ bool next_hit(const DevScene& S, Walk& w, Hit& h) {
  if (!w.alive) return false;
  int c[3], b[3], e[3], rel[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) c[a] = w.r[a] + w.Oi[a];
  int sx = S.skip_sx, sz = S.skip_sz;
  b[0] = c[0] >> sx;
  b[1] = c[1] >> sx;
  b[2] = c[2] >> sz;
  const unsigned v = AHEAD ? w.box
                           : __ldg(w.skip + ((long long)b[2] * S.skip_n01 +
                                             (b[1] * S.skip_n0 + b[0])));
  // the word is read beside the box, which it does not wait for: two steps in three
  // need it (LiDAR 237 -> 233 us, fisheye 298 -> 292, camera 261 -> 259)
  const int ix = c[0] ^ mirror_mask(w, 0), iy = c[1] ^ mirror_mask(w, 1),
            iz = c[2] ^ mirror_mask(w, 2);
  const uint4 word = AHEAD ? w.word : block_word(S, ix, iy, iz);
  e[0] = v & 31u;
  e[1] = (v >> 5) & 31u;
  e[2] = v >> 10;
  int vox = -1;
  if (v == 0u) {
    vox = find_leaf(S, word, ix, iy, iz, &sx, &sz);
    b[0] = c[0] >> sx;
    b[1] = c[1] >> sx;
    b[2] = c[2] >> sz;
    e[0] = e[1] = e[2] = 1;
  }
  float tx[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    rel[a] = ((b[a] + e[a]) << (a == 2 ? sz : sx)) - w.Oi[a];
    tx[a] = ((float)rel[a] - w.Of[a]) * w.invD[a];
  }
  const float te = fminf(fminf(tx[0], tx[1]), tx[2]);
  bool found = false;
  if (vox >= 0) {
    float tin = w.t;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      h.lo[a] = rel[a] - (1 << sx);
      tin = fmaxf(tin, ((float)h.lo[a] - w.Of[a]) * w.invD[a]);
    }
    h.tin = tin;
    h.tout = fminf(te, w.tend);
    found = h.tout > tin;
    h.vox = vox;
    h.ls = sx;
    // start fetching the voxel's record: it is read right after this step
    prefetch_l1(static_cast<const char*>(S.params) +
                (size_t)vox * (DT == SALF_F32 ? 128u : 64u));
  }
  w.alive = te < w.tend;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int q = max(w.r[a], __viaddmin_s32(rel[a], -1, __float2int_rd(fmaf(te, w.D[a], w.Of[a]))));
    w.r[a] = tx[a] <= te ? rel[a] : q;
  }
  w.t = fmaxf(w.t, te);
  if (AHEAD && w.alive) walk_read_ahead(S, w);
  return found;
}

// ---------------------------------------------------------------- records

template <int DT>
struct Record;  // widened record (BF16 only: FP32 records are read in stages)

// Where a record's 16-byte chunks come from: global memory (read-only path)
// or a copy of the raw record bytes in shared memory.
struct GlobalRec {
  const float4* p;
  __device__ __forceinline__ float4 chunk(int k) const { return __ldg(p + k); }
};
struct SharedRec {
  const float4* p;
  __device__ __forceinline__ float4 chunk(int k) const { return p[k]; }
};

// BF16: 32 bf16 (64 B), widened to FP32 in registers.
template <>
struct Record<SALF_BF16> {
  float v[32];
  template <class Src>
  __device__ __forceinline__ void load(const Src& src) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 c = src.chunk(k);
      const uint4 q = make_uint4(__float_as_uint(c.x), __float_as_uint(c.y), __float_as_uint(c.z),
                                 __float_as_uint(c.w));
      unsigned w4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[8 * k + 2 * j] = __uint_as_float(w4[j] << 16);
        v[8 * k + 2 * j + 1] = __uint_as_float(w4[j] & 0xffff0000u);
      }
    }
  }
};

// Local coordinates of the segment midpoint (distance tm) inside a hit's box:
// x = (p - centre) / (edge / 2).
__device__ __forceinline__ void local_coords(const Walk& w, const Hit& h, float tm, float x[3]) {
  const float E = (float)(1 << h.ls);
  const float inv_half = __int_as_float((128 - h.ls) << 23);  // 2 / E, exact: E = 2^ls
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float p = fmaf(tm, w.D[a], w.Of[a]);  // relative to the origin cell
    const float ctr = (float)h.lo[a] + 0.5f * E;
    x[a] = unmirror(w, a, (p - ctr) * inv_half);
  }
}

__device__ __forceinline__ float sigmoidf_fast(float z) {
  return __fdividef(1.f, 1.f + __expf(-z));
}

// Eq. 1 (EXP) or Eq. 5-6 (SDF) density at x; `lin` = W . [x, 1].
template <int MODE>
__device__ __forceinline__ float density(const float* rec, const float x[3], float* lin) {
  float s = fmaf(rec[0], x[0], fmaf(rec[1], x[1], fmaf(rec[2], x[2], rec[3])));
  *lin = s;
  if (MODE == SALF_FIELD_EXP) return __expf(s);
  float a = rec[25], b = rec[26];
  float e = __expf(-fabsf(s) / b);
  float sg = (s > 0.f) ? 1.f : ((s < 0.f) ? -1.f : 0.f);
  return 0.5f * a + 0.5f * a * sg * (1.f - e);
}

// Eq. 2 colour: c = sigmoid(W_c x + W_sh gamma(d)).
__device__ __forceinline__ void colour(const float* rec, const float x[3], const float gam[4],
                                       float c[3]) {
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    float z = rec[4 + 3 * r] * x[0] + rec[5 + 3 * r] * x[1] + rec[6 + 3 * r] * x[2];
    z = fmaf(rec[13 + 4 * r], gam[0], z);
    z = fmaf(rec[14 + 4 * r], gam[1], z);
    z = fmaf(rec[15 + 4 * r], gam[2], z);
    z = fmaf(rec[16 + 4 * r], gam[3], z);
    c[r] = sigmoidf_fast(z);
  }
}

__device__ __forceinline__ float intensity_field(const float* rec, const float x[3]) {
  float z = fmaf(rec[27], x[0], fmaf(rec[28], x[1], fmaf(rec[29], x[2], rec[30])));
  return sigmoidf_fast(z);
}

__device__ __forceinline__ void sh_basis(const float d[3], float gam[4]) {
  gam[0] = kSH0;
  gam[1] = kSH1 * d[1];
  gam[2] = kSH1 * d[2];
  gam[3] = kSH1 * d[0];
}

// Launch-order tile row k -> tile row: first_row, first_row + 1, first_row - 1,
// first_row + 2, ... (rows past one edge continue on the other side).
__device__ __forceinline__ int zigzag_row(int k, int first, int rows) {
  const int below = rows - 1 - first;  // rows after `first`
  const int m = min(first, below);     // pairs that alternate
  if (k <= 2 * m) return (k & 1) ? first + (k + 1) / 2 : first - k / 2;
  const int rest = k - 2 * m;          // only one side left
  return below > first ? first + m + rest : first - m - rest;
}

// Tile of a warp: (pixel column, pixel row) of its first lane.
__device__ __forceinline__ void tile_origin(const ReqDev& Q, int tile, int* u0, int* v0) {
  const int k = (int)((unsigned)tile / (unsigned)Q.tiles_x);
  *u0 = (tile - k * Q.tiles_x) * Q.tile_w;
  *v0 = zigzag_row(k, Q.first_row, Q.tiles_y) * Q.tile_h;
}

// Local field of one voxel at local coordinates x (Eq. 1 or 5-6, Eq. 2, and
// the intensity field): density, the affine geometry value, colour,
// intensity, and the SDF parameters a, b.
struct Field {
  float sig, lin, c[3], io, a, b;
  float dr;  // sigmoid of the raydrop logit (record slot 31), when asked for
};

__device__ __forceinline__ float sdf_density(float s, float a, float b) {
  const float e = __expf(-fabsf(s) / b);
  const float sg = (s > 0.f) ? 1.f : ((s < 0.f) ? -1.f : 0.f);
  return 0.5f * a + 0.5f * a * sg * (1.f - e);
}

// FP32 records are read in two stages (a compiler barrier keeps the second
// stage's loads below the first stage's arithmetic), so only half of the
// record is live in registers at a time.  Slots: Wsigma 0-3, W_c 4-12 (rows
// r, g, b), W_sh 13-24 (rows r, g, b), a 25, b 26, W_int 27-30.
template <int DT, int MODE, class Src>
__device__ __forceinline__ void field_eval_src(const Src& p, bool want_int, const float x[3],
                                               const float gam[4], Field& f,
                                               bool want_drop = false) {
  if constexpr (DT == SALF_F32) {
    const float4 q0 = p.chunk(0), q1 = p.chunk(1), q2 = p.chunk(2), q3 = p.chunk(3);
    f.lin = fmaf(q0.x, x[0], fmaf(q0.y, x[1], fmaf(q0.z, x[2], q0.w)));
    float zr = q1.x * x[0] + q1.y * x[1] + q1.z * x[2];
    float zg = q1.w * x[0] + q2.x * x[1] + q2.y * x[2];
    float zb = q2.z * x[0] + q2.w * x[1] + q3.x * x[2];
    zr = fmaf(q3.y, gam[0], zr);
    zr = fmaf(q3.z, gam[1], zr);
    zr = fmaf(q3.w, gam[2], zr);
    asm volatile("" ::: "memory");
    const float4 q4 = p.chunk(4), q5 = p.chunk(5), q6 = p.chunk(6);
    zr = fmaf(q4.x, gam[3], zr);
    zg = fmaf(q4.y, gam[0], zg);
    zg = fmaf(q4.z, gam[1], zg);
    zg = fmaf(q4.w, gam[2], zg);
    zg = fmaf(q5.x, gam[3], zg);
    zb = fmaf(q5.y, gam[0], zb);
    zb = fmaf(q5.z, gam[1], zb);
    zb = fmaf(q5.w, gam[2], zb);
    zb = fmaf(q6.x, gam[3], zb);
    f.a = q6.y;
    f.b = q6.z;
    f.sig = MODE == SALF_FIELD_EXP ? __expf(f.lin) : sdf_density(f.lin, f.a, f.b);
    f.c[0] = sigmoidf_fast(zr);
    f.c[1] = sigmoidf_fast(zg);
    f.c[2] = sigmoidf_fast(zb);
    f.io = 0.f;
    f.dr = 0.f;
    if (want_int || want_drop) {
      const float4 q7 = p.chunk(7);
      if (want_int)
        f.io = sigmoidf_fast(fmaf(q6.w, x[0], fmaf(q7.x, x[1], fmaf(q7.y, x[2], q7.z))));
      if (want_drop) f.dr = sigmoidf_fast(q7.w);
    }
  } else {
    Record<DT> rec;
    rec.load(p);
    f.sig = density<MODE>(rec.v, x, &f.lin);
    colour(rec.v, x, gam, f.c);
    f.io = want_int ? intensity_field(rec.v, x) : 0.f;
    f.dr = want_drop ? sigmoidf_fast(rec.v[31]) : 0.f;
    f.a = rec.v[25];
    f.b = rec.v[26];
  }
}

// Record bytes per voxel and the 16-byte chunks of one record.
template <int DT>
struct RecordLayout {
  static constexpr int kChunks = DT == SALF_F32 ? 8 : 4;
};

template <int DT, int MODE>
__device__ __forceinline__ void field_eval(const DevScene& S, int vox, bool want_int,
                                           const float x[3], const float gam[4], Field& f,
                                           bool want_drop = false) {
  const GlobalRec src{reinterpret_cast<const float4*>(S.params) +
                      (size_t)vox * RecordLayout<DT>::kChunks};
  field_eval_src<DT, MODE>(src, want_int, x, gam, f, want_drop);
}

// Front-to-back accumulators of one ray (Eq. 3-4).
struct Accum {
  float T, C0, C1, C2, Dp, Ip;
  int nvis;
  float Rp;  // sum of T_i alpha_i sigmoid(rho_i) (raydrop, when asked for)
};

// Composite one hit voxel of length dl with its field at the segment midpoint
// (distance tm, local coordinates x): alpha = 1 - exp(-sigma delta) (Eq. 4),
// weight T alpha (Eq. 3).  The ray kernel and the tile rasteriser both call
// this, so their arithmetic is the same.  Returns 1 - alpha.
template <int DT, int MODE, class Src>
__device__ __forceinline__ float composite_at(const float x[3], float tm, float dl, const Src& src,
                                             bool want_int, const float gam[4], Accum& A,
                                             bool want_drop = false) {
  Field f;
  field_eval_src<DT, MODE>(src, want_int, x, gam, f, want_drop);
  const float e = __expf(-f.sig * dl);  // 1 - alpha (Eq. 4)
  const float wgt = A.T * (1.f - e);    // T_i alpha_i (Eq. 3)
  A.C0 = fmaf(wgt, f.c[0], A.C0);
  A.C1 = fmaf(wgt, f.c[1], A.C1);
  A.C2 = fmaf(wgt, f.c[2], A.C2);
  A.Dp = fmaf(wgt, tm, A.Dp);
  if (want_int) A.Ip = fmaf(wgt, f.io, A.Ip);
  if (want_drop) A.Rp = fmaf(wgt, f.dr, A.Rp);
  A.T *= e;
  return e;
}

template <int DT, int MODE, class Src>
__device__ __forceinline__ float composite_hit(const Walk& w, const Hit& h, const Src& src,
                                              bool want_int, const float gam[4], Accum& A,
                                              bool want_drop = false) {
  const float tm = 0.5f * (h.tin + h.tout);
  float x[3];
  local_coords(w, h, tm, x);
  return composite_at<DT, MODE>(x, tm, h.tout - h.tin, src, want_int, gam, A, want_drop);
}

// Per-ray outputs of a request (colour premultiplied, background added with
// the final transmittance; opacity 1 - T_end, which the weights sum to).
__device__ __forceinline__ void write_outputs(const ReqDev& Q, int ray, bool valid, const Accum& A,
                                              bool want_drop = false) {
  // raydrop: an escaping ray (T_end) returns nothing
  if (want_drop) Q.raydrop[ray] = valid ? A.Rp + A.T : 0.f;
  if (Q.rgb) {
    float* o = Q.rgb + 3 * (size_t)ray;
    o[0] = valid ? fmaf(A.T, Q.bg[0], A.C0) : 0.f;
    o[1] = valid ? fmaf(A.T, Q.bg[1], A.C1) : 0.f;
    o[2] = valid ? fmaf(A.T, Q.bg[2], A.C2) : 0.f;
  }
  const float Op = 1.f - A.T;  // sum of T_i alpha_i telescopes to 1 - T_end (Eq. 3-4)
  if (Q.depth) Q.depth[ray] = A.Dp;
  if (Q.opacity) Q.opacity[ray] = Op;
  if (Q.intensity) Q.intensity[ray] = A.Ip;
  if (Q.saved) {
    float4* s = reinterpret_cast<float4*>(Q.saved) + 2 * (size_t)ray;
    s[0] = make_float4(A.C0, A.C1, A.C2, A.Dp);
    s[1] = make_float4(Op, A.Ip, A.T, (float)A.nvis);
  }
  if (Q.valid) Q.valid[ray] = valid ? 1 : 0;
}

// Products of the transmittances of the spans of a ray (lanes k = 0..K-1 of a
// group of K): *inc = T_0 ... T_k, *ex = T_0 ... T_k-1 (1 for k = 0).  The
// association order is fixed, so the products only fall as the T_k fall.
__device__ __forceinline__ void span_products(float T, int k, int K, float* inc, float* ex) {
  float p = T;
  for (int off = 1; off < K; off <<= 1) {
    const float y = __shfl_up_sync(0xffffffffu, p, off, K);
    if (k >= off) p *= y;
  }
  const float e = __shfl_up_sync(0xffffffffu, p, 1, K);
  *inc = p;
  *ex = k == 0 ? 1.f : e;
}

// Warp tile -> request, pixel.
__device__ __forceinline__ int find_request(const LaunchParams& P, int warp) {
  int r = 0;
  while (r + 1 < P.n_req && warp >= P.req[r + 1].tile_begin) ++r;
  return r;
}

}  // namespace salf
