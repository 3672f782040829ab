// The traversal header compiled for the host, so that a test can follow a ray's
// walk step by step and see every address it reads (tests/test_walk_far_origins.py).
// Signed arithmetic wraps as on the device (-fwrapv).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <limits>
#include <vector>

using std::max;
using std::min;

namespace {
struct Range {
  const char* p;
  size_t n;
};
std::vector<Range> g_ranges;
long g_outside;  // reads that no buffer holds

template <class T>
T ldg(const T* p) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p);
  for (const Range& r : g_ranges) {
    const uintptr_t b = reinterpret_cast<uintptr_t>(r.p);
    if (a >= b && a + sizeof(T) <= b + r.n) return *p;
  }
  ++g_outside;
  return T{};
}
template <class To, class From>
To bits(From x) {
  To y;
  std::memcpy(&y, &x, 4);
  return y;
}
int to_int(float x) {  // conversions saturate, and NaN becomes 0
  if (!(x == x)) return 0;
  if (x >= 2147483648.f) return 0x7fffffff;
  return x < -2147483648.f ? -0x7fffffff - 1 : (int)x;
}
void sincospi(float x, float* s, float* c) {
  *s = std::sin((float)M_PI * x);
  *c = std::cos((float)M_PI * x);
}
}  // namespace

#define __ldg(p) ldg(p)
#define __popc(x) __builtin_popcount(x)
#define __float2int_rd(x) to_int(std::floor(x))
#define __uint_as_float(x) bits<float>(x)
#define __int_as_float(x) bits<float>(x)
#define __float_as_uint(x) bits<unsigned>(x)
#define __viaddmin_s32(a, b, c) std::min((a) + (b), (c))
#define __fadd_rn(a, b) ((a) + (b))
#define __fsub_rn(a, b) ((a) - (b))
#define __fmul_rn(a, b) ((a) * (b))
#define __fmaf_rn(a, b, c) fmaf(a, b, c)
#define __expf(x) expf(x)
#define __fdividef(a, b) ((a) / (b))
#define __shfl_up_sync(m, v, o, k) (v)
#define rsqrtf(x) (1.f / sqrtf(x))
#define sincospif sincospi

#include "traverse_host.cuh"  // traverse.cuh, its prefetch instruction and narrowing casts replaced

// One explicit ray through a grid of level-0 voxels (K = 0): the reads outside
// the buffers, the steps and hits, and the origin's cell and fraction.
extern "C" long walk_ray(const float* ray, const double* origin, double cell, const int* mdim,
                         const int* n, const int* box, const void* mask0,
                         const unsigned short* skip, int ahead, int max_steps, int* steps,
                         int* hits, int* Oi, float* Of) {
  DevScene S;
  std::memset(&S, 0, sizeof(S));
  S.mask0 = static_cast<const uint4*>(mask0);
  S.mdim0 = mdim[0];
  S.mdim01 = mdim[0] * mdim[1];
  S.skip_n0 = n[0];
  S.skip_n01 = n[0] * n[1];
  S.skip_sx = 2;
  const long long n01 = S.skip_n01;
  for (int o = 0; o < 8; ++o) {  // bricks from 0: a mirrored brick ~b is entry n - 1 - b
    long long off = o * n01 * n[2], stride = 1;
    for (int a = 0; a < 3; ++a) {
      off += stride * ((o >> a) & 1 ? n[a] : 0);
      stride *= n[a];
    }
    S.skip_oct[o] = reinterpret_cast<const unsigned short*>(reinterpret_cast<uintptr_t>(skip) + 2 * off);
  }
  for (int a = 0; a < 3; ++a) {
    S.bmin[a] = box[a];
    S.bmax[a] = box[3 + a];
    S.origin[a] = origin[a];
    S.origin2[a][0] = (float)origin[a];
    S.origin2[a][1] = (float)(origin[a] - (double)(float)origin[a]);
  }
  S.inv_sfin = 1.0 / cell;
  S.isf2[0] = (float)S.inv_sfin;
  S.isf2[1] = (float)(S.inv_sfin - (double)S.isf2[0]);
  g_ranges = {{reinterpret_cast<const char*>(ray), 32},
              {static_cast<const char*>(mask0), sizeof(uint4) * (size_t)S.mdim01 * mdim[2]},
              {reinterpret_cast<const char*>(skip), 16 * (size_t)n01 * n[2]}};
  g_outside = 0;
  ReqDev Q;
  std::memset(&Q, 0, sizeof(Q));
  Q.kind = SALF_RAYS_EXPLICIT;
  Q.rays = ray;
  salf::Ray r;
  salf::gen_ray(Q, S, 0, 0, 0, r);
  salf::Walk w;
  salf::Hit h;
  *steps = *hits = 0;
  if (ahead)
    salf::walk_init<true>(S, r, w);
  else
    salf::walk_init<false>(S, r, w);
  while (w.alive && *steps < max_steps && g_outside == 0) {
    ++*steps;
    *hits += (ahead ? salf::next_hit<SALF_F32, true>(S, w, h)
                    : salf::next_hit<SALF_F32, false>(S, w, h)) ? 1 : 0;
  }
  for (int a = 0; a < 3; ++a) {
    Oi[a] = r.Oi[a];
    Of[a] = r.Of[a];
  }
  return w.alive && *steps >= max_steps ? -1 : g_outside;
}
