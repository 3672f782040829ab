// skip.cu -- the skip boxes of a scene (DevScene::skip): for every empty brick
// of the voxels' tight box and each of the 8 direction octants, an empty box
// that starts at the brick and extends in the octant's directions.
//
//  1. k_skip_occ: per column of bricks (x, y) and 64 layers, its occupied
//     bricks as the bits of one word.
//  2. k_skip_rows, k_skip_rects: the OR of the words of every rectangle of
//     2^i x 2^j columns, i, j = 0..4.
//  3. k_skip_boxes: one thread per column, octant and word, all layers in
//     turn.  For each square of 2^i columns that starts at
//     the brick, the run of empty layers (carried from layer to layer); of
//     these boxes the one with the largest smaller side, a layer counting as 8
//     cells of width (rays in driving scenes are nearly horizontal; 4 and 16
//     gave the same steps).  It is then widened in x and in y by 16, 8, 4, 2, 1
//     columns as long as the same layers stay empty.  Boxes end at the word's
//     64 layers.
//
// A greedy box instead of the largest one: on a driving scene, boxes from
// every square size cut a ray's steps by 4% at most (LiDAR 15.6 -> 14.9 steps
// per ray; the occupancy pyramid and column masks that this replaces took 32).
// Without the widening: 18.3.
#include <algorithm>

#include "salf_internal.h"
#include "skip_shape.h"

namespace {

constexpr int kLevels = kSkipLevels;
constexpr int kPad = kSkipPad;
constexpr int kMaxXY = 31, kMaxZ = 63;          // box sizes a skip entry holds, in bricks
constexpr int kChunk = 8;                       // layers per thread of k_skip_boxes

struct SkipGrid {
  int n[3], base[3];
  int p, q;       // log2 of a brick's edges in level-0 cells
  int words;      // 64-layer words of a column
  int px, py;     // padded table size: n + kPad
  unsigned mdim0, mdim01;
};

// Occupancy words of the brick's cells: blocks of 4x4x4 cells, layer bits
// picked from the Morton order (z1: word, z0: nibbles).
__global__ void __launch_bounds__(256) k_skip_occ(const uint4* __restrict__ mask0, SkipGrid G,
                                                  unsigned long long* __restrict__ occ) {
  const long long i = blockIdx.x * 256LL + threadIdx.x;
  if (i >= (long long)G.px * G.py * G.words) return;
  const int x = (int)(i % G.px) - kPad, y = (int)(i / G.px % G.py) - kPad;
  const int wd = (int)(i / ((long long)G.px * G.py));
  unsigned long long bits = 0;  // 0 in the padding before the grid
  if (x >= 0 && y >= 0) {
    const int nb = 1 << (G.p - 2);  // blocks per brick along x and y
    for (int k = 0; k < 64 && wd * 64 + k < G.n[2];) {
      const int bz = G.base[2] + wd * 64 + k;  // brick
      const int z = bz << G.q;                 // its first cell; q < 2: part of one block
      unsigned lo = 0, hi = 0;
      for (int zb = z >> 2; zb <= ((bz + 1) << G.q) - 1 >> 2; ++zb)
        for (int yb = 0; yb < nb; ++yb)
          for (int xb = 0; xb < nb; ++xb) {
            const uint4 m = __ldg(&mask0[(unsigned)zb * G.mdim01 +
                                         (unsigned)((G.base[1] + y) * nb + yb) * G.mdim0 +
                                         (unsigned)((G.base[0] + x) * nb + xb)]);
            lo |= m.x;
            hi |= m.y;
          }
      if (G.q >= 2) {
        if (lo | hi) bits |= 1ull << k;
        ++k;
        continue;
      }
      // the block's layers, then its bricks (base[2] is block aligned)
      unsigned lay = ((lo & 0x0f0f0f0fu) ? 1u : 0u) | ((lo & 0xf0f0f0f0u) ? 2u : 0u) |
                     ((hi & 0x0f0f0f0fu) ? 4u : 0u) | ((hi & 0xf0f0f0f0u) ? 8u : 0u);
      if (G.q == 1) lay = ((lay & 3u) ? 1u : 0u) | ((lay & 12u) ? 2u : 0u);
      bits |= (unsigned long long)lay << k;
      k += 4 >> G.q;
    }
  }
  occ[i] = bits;
}

// The ORs of 2, 4, ..., 2^(kLevels - 1) words from `in` on, `step` apart, `left`
// of them inside the table (nothing lies beyond it), to out + level,
// out + 2 level, ...; returns the first word.
__device__ __forceinline__ unsigned long long or_runs(const unsigned long long* in, int step,
                                                      int left, unsigned long long* out,
                                                      long long level) {
  const unsigned long long first = __ldg(in);
  unsigned long long m = first;
#pragma unroll
  for (int k = 1; k < kLevels; ++k) {
#pragma unroll
    for (int d = 1 << (k - 1); d < 1 << k; ++d)
      if (d < left) m |= __ldg(in + (long long)d * step);
    out[k * level] = m;
  }
  return first;
}

// Rectangles of 2^i x 1 columns: table i * kLevels.
__global__ void __launch_bounds__(256) k_skip_rows(const unsigned long long* __restrict__ occ,
                                                   SkipGrid G, unsigned long long* __restrict__ rect) {
  const long long i = blockIdx.x * 256LL + threadIdx.x;
  const long long table = (long long)G.px * G.py * G.words;
  if (i >= table) return;
  rect[i] = or_runs(occ + i, 1, G.px - (int)(i % G.px), rect + i, kLevels * table);
}

// Rectangles of 2^i x 2^j columns: table i * kLevels + j.
__global__ void __launch_bounds__(256) k_skip_rects(SkipGrid G, unsigned long long* rect) {
  const long long i = blockIdx.x * 256LL + threadIdx.x;
  const long long table = (long long)G.px * G.py * G.words;
  if (i >= table * kLevels) return;
  const long long at = i % table;
  unsigned long long* t = rect + i / table * (kLevels * table) + at;
  or_runs(t, G.px, G.py - (int)(at / G.px % G.py), t, table);
}

// One thread per column, octant (sx, sy, down; 1: the ray travels downwards),
// word and kChunk of its layers.  A warp takes 32 columns along x, a block the 8
// octants.  Bound by instructions and the table reads (L1).  A 1.27M-voxel scene,
// 177 x 177 x 41 bricks: 213 us with all of a word's layers in one thread, 193 in
// chunks, 158 with 32-bit offsets, 110 with the box kept from layer to layer.  Off:
// the offsets' type (skip_wide_offsets).
template <class Off>
__global__ void __launch_bounds__(256) k_skip_boxes(const unsigned long long* __restrict__ rect,
                                                    SkipGrid G, int tiles_x, int chunks,
                                                    unsigned short* __restrict__ skip) {
  int bid = (int)blockIdx.x;
  const int x = bid % tiles_x * 32 + (threadIdx.x & 31);
  bid /= tiles_x;
  const int l0 = bid % chunks * kChunk;  // first layer of the chunk, in the ray's order
  bid /= chunks;
  const int y = bid % G.n[1], wd = bid / G.n[1];
  const int sx = (threadIdx.x >> 5) & 1, sy = (threadIdx.x >> 6) & 1, down = threadIdx.x >> 7;
  if (x >= G.n[0]) return;
  const Off table = (Off)G.px * G.py * G.words;
  const unsigned long long* here = rect + ((Off)wd * G.px * G.py + (y + kPad) * G.px + (x + kPad));
  // word of the 2^i x 2^j rectangle whose far side lies fx, fy columns ahead
  auto at = [&](int i, int j, int fx, int fy) {
    const int dx = sx ? 1 - fx : fx - (1 << i), dy = sy ? 1 - fy : fy - (1 << j);
    return __ldg(here + skip_rect_offset<Off>(i, j, table, G.px, dy, dx));
  };
  const int room_x = min(kMaxXY, sx ? x + 1 : G.n[0] - x);
  const int room_y = min(kMaxXY, sy ? y + 1 : G.n[1] - y);
  unsigned long long sq[kLevels];
#pragma unroll
  for (int k = 0; k < kLevels; ++k) sq[k] = at(k, k, 1 << k, 1 << k);
  const int layers = min(64, G.n[2] - 64 * wd);
  if (l0 >= layers) return;
  const int mx = sx ? G.n[0] - 1 - x : x, my = sy ? G.n[1] - 1 - y : y;
  const long long n01 = (long long)G.n[0] * G.n[1];
  // empty layers of each square from the current layer on; layers are taken
  // against the ray, so the run of the one before carries over.  It starts with
  // the l0 layers beyond the chunk: below layer l0, or above layers - 1 - l0.
  int run[kLevels];
#pragma unroll
  for (int k = 0; k < kLevels; ++k) {
    if (l0 == 0) {
      run[k] = 0;
    } else if (down) {
      const unsigned long long m = sq[k] << (64 - l0);
      run[k] = min(l0, m ? __clzll((long long)m) : 64);
    } else {
      const unsigned long long m = sq[k] >> (layers - l0);
      run[k] = min(l0, m ? __ffsll((long long)m) - 1 : 64);
    }
  }
  int ex = 0, ey = 0, pk = 0, pz = 0;  // the box of the layer before; 0: none
  unsigned long long region = 0;       // the OR over its columns
  for (int l = l0; l < min(layers, l0 + kChunk); ++l) {
    const int z = down ? l : layers - 1 - l;
    int bk = 0, bz = 0, best = 0;
#pragma unroll
    for (int k = 0; k < kLevels; ++k) {
      run[k] = (sq[k] >> z) & 1ull ? 0 : min(run[k] + 1, kMaxZ);
      const int wide = 4 << k, tall = 8 * run[k];
      const int score = run[k] ? (min(wide, tall) << 16) + (wide + tall) : 0;
      if (score > best) {
        best = score;
        bk = k;
        bz = run[k];
      }
    }
    if (bz == 0) {
      ex = 0;
    } else if (ex == 0 || bk != pk || bz != pz + 1 || ((region >> z) & 1ull)) {
      // the box's layers; bz <= 63
      const unsigned long long zs = ((1ull << bz) - 1ull) << (down ? z - bz + 1 : z);
      const int e = 1 << bk;
      ex = min(e, room_x);
      ey = min(e, room_y);
      if (ex == e)
#pragma unroll
        for (int i = kLevels - 1; i >= 0; --i)
          if (ex + (1 << i) <= room_x && !(at(i, bk, ex + (1 << i), e) & zs)) ex += 1 << i;
      const int kx = 31 - __clz(ex);  // two overlapping rectangles cover ex columns
      if (ey == e)
#pragma unroll
        for (int j = kLevels - 1; j >= 0; --j)
          if (ey + (1 << j) <= room_y && !((at(kx, j, 1 << kx, ey + (1 << j)) |
                                            at(kx, j, ex, ey + (1 << j))) & zs))
            ey += 1 << j;
      const int ky = 31 - __clz(ey);
      region = at(kx, ky, 1 << kx, 1 << ky) | at(kx, ky, ex, 1 << ky) |
               at(kx, ky, 1 << kx, ey) | at(kx, ky, ex, ey);
    }
    // else the layer extends the box before it: every widening that failed there
    // fails again, and those that did not stay inside the box, empty in this layer
    pk = bk;
    pz = bz;
    const unsigned entry =
        ex ? (unsigned)ex | ((unsigned)ey << 5) | ((unsigned)bz << 10) : 0u;
    const int gz = 64 * wd + z, mz = down ? G.n[2] - 1 - gz : gz;
    const int oct = sx | (sy << 1) | (down << 2);
    skip[((long long)oct * G.n[2] + mz) * n01 + (long long)my * G.n[0] + mx] = (unsigned short)entry;
  }
}

}  // namespace

void salf_grid_shape(const int32_t dims[3], int mdim[3], int* p, int* q) {
  // a brick is one layer of a 4x4x4 block; in grids beyond 2^28 such bricks (2^32
  // level-0 cells; 4 GB of skip boxes if the voxels span it all) it grows
  // until they fit, first in z
  int sp = 2, sq = 0;
  auto bricks = [&] {
    double b = 1;
    for (int a = 0; a < 3; ++a) {
      const int s = a == 2 ? sq : sp;
      b *= (double)(((int64_t)dims[a] + (1 << s) - 1) >> s);
    }
    return b;
  };
  while (bricks() > (double)(1 << 28)) {
    if (sq < 2) {
      ++sq;
    } else {
      ++sp;
      ++sq;
    }
  }
  for (int a = 0; a < 3; ++a) {  // whole bricks of blocks
    const int s = a == 2 ? (sq < 2 ? 2 : sq) : sp;
    mdim[a] = (int)((((int64_t)dims[a] + (1 << s) - 1) >> s) << (s - 2));
  }
  *p = sp;
  *q = sq;
}

salf_status salf_build_skip(salf_scene* s, int p, int q, cudaStream_t st) {
  DevScene& D = s->dev;
  SkipGrid G;
  G.p = p;
  G.q = q;
  for (int a = 0; a < 3; ++a) {
    const int sh = a == 2 ? q : p;
    // the first brick, block aligned; bmax > bmin unless the scene is empty
    int lo = (D.bmin[a] >> D.K) >> 2 << 2;
    const int hi = D.bmax[a] > D.bmin[a] ? (D.bmax[a] - 1) >> D.K : lo;
    lo = lo >> sh;
    G.base[a] = lo;
    G.n[a] = (hi >> sh) - lo + 1;
  }
  G.words = (G.n[2] + 63) / 64;
  G.px = G.n[0] + kPad;
  G.py = G.n[1] + kPad;
  G.mdim0 = (unsigned)D.mdim0;
  G.mdim01 = (unsigned)D.mdim01;
  const long long n01 = (long long)G.n[0] * G.n[1];
  const long long table = (long long)G.px * G.py * G.words;
  void* skip = nullptr;
  salf_status rs = salf_scene_dalloc(s, (size_t)n01 * G.n[2] * 8 * sizeof(unsigned short), &skip);
  if (rs != SALF_OK) return rs;
  PoolBuf tmp;
  rs = tmp.get(s->ctx, (size_t)table * (1 + kLevels * kLevels) * 8, st);
  if (rs != SALF_OK) return rs;
  unsigned long long* occ = static_cast<unsigned long long*>(tmp.p);
  unsigned long long* rect = occ + table;
  k_skip_occ<<<(unsigned)((table + 255) / 256), 256, 0, st>>>(D.mask0, G, occ);
  k_skip_rows<<<(unsigned)((table + 255) / 256), 256, 0, st>>>(occ, G, rect);
  k_skip_rects<<<(unsigned)((table * kLevels + 255) / 256), 256, 0, st>>>(G, rect);
  const int tiles_x = (G.n[0] + 31) / 32, chunks = (std::min(64, G.n[2]) + kChunk - 1) / kChunk;
  const auto boxes = skip_wide_offsets(table) ? k_skip_boxes<long long> : k_skip_boxes<int>;
  boxes<<<(unsigned)(tiles_x * G.n[1] * G.words * chunks), 256, 0, st>>>(
      rect, G, tiles_x, chunks, static_cast<unsigned short*>(skip));
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return salf_cuda_fail(e, "skip boxes");
  // brick b of axis a is entry b - base of an octant, mirrored (~b) entry
  // n - 1 - (b - base) = ~b + base + n
  for (int o = 0; o < 8; ++o) {
    long long off = o * n01 * G.n[2], stride = 1;
    for (int a = 0; a < 3; ++a) {
      off += stride * ((o >> a) & 1 ? G.base[a] + G.n[a] : -G.base[a]);
      stride *= G.n[a];
    }
    D.skip_oct[o] = reinterpret_cast<const unsigned short*>(
        reinterpret_cast<uintptr_t>(skip) + (uintptr_t)(off * (long long)sizeof(unsigned short)));
  }
  D.skip_n0 = G.n[0];
  D.skip_n01 = (int)n01;
  D.skip_sx = D.K + p;
  D.skip_sz = D.K + q;
  D.skip_coarse = p > 2 || q > 0;
  return SALF_OK;
}
