// scene_build_gpu.cu -- salf_build_scene for a voxel set already in device
// memory: the steps of the host build (scene_build.cpp) as kernels, giving
// the same acceleration structure (Sec. III-B stand-in for the octree):
//  1. per voxel its sort key (4x4x4 block of level-0 cells, Morton index of
//     the cell in the block, Morton index of the min corner in the cell) and
//     the range checks; a stable radix sort of (key, voxel) gives the voxel
//     order;
//  2. one pass over the voxels in that order: overlaps (they show between
//     neighbours), level-0 occupancy words (each warp ORs its voxels of one
//     block first), each block's first voxel and whether it holds a split cell,
//     the voxel boxes and the tight box; a scan of the words' popcounts gives
//     the cells' ranks;
//  3. the cell table's level-0 voxels, the split cells' first voxels and node
//     budgets, and the records in voxel order; then the host reads the checks,
//     counts and the tight box back, once;
//  4. one thread per split cell builds its subtree of nodes from the cell's
//     voxels (consecutive in the voxel order) into a slice sized by an upper
//     bound, and turns a cell split once into (first child, child mask); the
//     skip boxes (skip.cu).
// Kernels of steps 2 and 3 do nothing once a key was out of range.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <string>

#include "salf_internal.h"
#include "scan.cuh"
#include "sort.cuh"

using namespace salf_scan;
using namespace salf_sort;

namespace {

constexpr int kErrLevel = 1, kErrRange = 2, kErrOverlap = 4;

__device__ __forceinline__ unsigned dmorton6(unsigned x, unsigned y, unsigned z) {
  return (x & 1u) | ((y & 1u) << 1) | ((z & 1u) << 2) | ((x & 2u) << 2) | ((y & 2u) << 3) |
         ((z & 2u) << 4);
}

__device__ __forceinline__ unsigned long long dspread3(unsigned long long x) {
  x &= 0x1fffffULL;
  x = (x | x << 32) & 0x1f00000000ffffULL;
  x = (x | x << 16) & 0x1f0000ff0000ffULL;
  x = (x | x << 8) & 0x100f00f00f00f00fULL;
  x = (x | x << 4) & 0x10c30c30c30c30c3ULL;
  x = (x | x << 2) & 0x1249249249249249ULL;
  return x;
}

struct Grid {
  int K;
  int dims[3];
  int mdim[3];  // level-0 occupancy words per axis
};

__device__ __forceinline__ long long block_of(const Grid& G, long long cx, long long cy,
                                              long long cz) {
  return ((cz >> 2) * G.mdim[1] + (cy >> 2)) * G.mdim[0] + (cx >> 2);
}

// What the build reads back.
struct Report {
  int err;          // error bits
  int bad_voxel;    // smallest offending voxel
  int overlap_at;   // smallest voxel-order position of an overlapping pair
  int status;       // the scene's status word (SDF records)
  int box[6];       // tight box: min corner, max corner (finest cells)
  unsigned n_cells;
  unsigned pad;
  unsigned long long n_nodes;
};

__global__ void k_report_init(Report* R) {
  R->err = 0;
  R->bad_voxel = R->overlap_at = INT_MAX;
  R->status = 0;
  for (int a = 0; a < 3; ++a) {
    R->box[a] = INT_MAX;
    R->box[3 + a] = INT_MIN;
  }
  R->n_cells = 0;
  R->n_nodes = 0;
}

// Counts from the scans' last values, and the status word.
__global__ void k_report(Report* R, const unsigned* __restrict__ rank, const unsigned* __restrict__ cnt,
                         long long nb, const unsigned long long* __restrict__ node_off,
                         const unsigned* __restrict__ budget, long long n,
                         const int* __restrict__ status) {
  R->n_cells = rank[nb - 1] + cnt[nb - 1];
  R->n_nodes = node_off ? node_off[n - 1] + budget[n - 1] : 0ull;
  R->status = *status;
}

__global__ void k_keys(const uint8_t* __restrict__ level, const int* __restrict__ ijk, long long n,
                       Grid G, unsigned long long* __restrict__ keys, unsigned* __restrict__ vals,
                       Report* __restrict__ R) {
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  int l = level[v];
  bool bad = false;
  if (l > G.K) {
    atomicOr(&R->err, kErrLevel);
    bad = true;
    l = 0;
  }
  unsigned long long f[3];
  for (int a = 0; a < 3; ++a) {
    long long c = ijk[3 * v + a];
    if (c < 0 || c >= ((long long)G.dims[a] << l)) {
      atomicOr(&R->err, kErrRange);
      bad = true;
      c = 0;
    }
    f[a] = (unsigned long long)c << (G.K - l);
  }
  if (bad) atomicMin(&R->bad_voxel, (int)v);
  const unsigned long long fine = (1ULL << G.K) - 1ULL;
  const long long blk = block_of(G, (long long)(f[0] >> G.K), (long long)(f[1] >> G.K),
                                 (long long)(f[2] >> G.K));
  keys[v] = ((unsigned long long)blk << (6 + 3 * G.K)) |
            ((unsigned long long)dmorton6((unsigned)(f[0] >> G.K) & 3, (unsigned)(f[1] >> G.K) & 3,
                                          (unsigned)(f[2] >> G.K) & 3)
             << (3 * G.K)) |
            (dspread3(f[0] & fine) | (dspread3(f[1] & fine) << 1) | (dspread3(f[2] & fine) << 2));
  vals[v] = (unsigned)v;
}

// A voxel of level l covers the key range [key, key + 8^(K - l)): in key order
// an overlap always shows between neighbours.  Voxels of one block are
// neighbours too: a warp's lanes of one block OR their occupancy bits before
// the one atomic, and a block of threads reduces its tight box before its six.
// 28 us for the whole pass over 1.27M voxels; with an atomic per voxel the words
// took 31 us and the box, six per voxel, 160 us.
__global__ void __launch_bounds__(256) k_voxels(
    const unsigned long long* __restrict__ keys, const unsigned* __restrict__ order,
    const uint8_t* __restrict__ level, const int* __restrict__ ijk, long long n, int K,
    unsigned long long* __restrict__ m0, unsigned* __restrict__ split,
    unsigned* __restrict__ vfirst, int* __restrict__ order_out, int4* __restrict__ vox_box,
    Report* R) {
  __shared__ int s_box[6];
  if (R->err & (kErrLevel | kErrRange)) return;
  if (threadIdx.x < 6) s_box[threadIdx.x] = threadIdx.x < 3 ? INT_MAX : INT_MIN;
  __syncthreads();
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = p < n;
  const int lane = threadIdx.x & 31;
  int lo[3] = {INT_MAX, INT_MAX, INT_MAX}, hi[3] = {INT_MIN, INT_MIN, INT_MIN};
  unsigned long long blk = ~0ull, key = 0;
  unsigned long long bit = 0;
  unsigned sub = 0;
  if (live) {
    key = keys[p];
    const unsigned v = order[p];
    const int l = level[v];
    blk = key >> (6 + 3 * K);
    bit = 1ull << ((key >> (3 * K)) & 63u);
    sub = l > 0 ? 1u : 0u;
    order_out[p] = (int)v;
    for (int a = 0; a < 3; ++a) {
      lo[a] = ijk[3 * (long long)v + a] << (K - l);
      hi[a] = lo[a] + (1 << (K - l));
    }
    vox_box[p] = make_int4(lo[0], lo[1], lo[2], K - l);
    unsigned long long prev = ~0ull;
    if (p > 0) {
      const unsigned long long pk = keys[p - 1];
      prev = pk >> (6 + 3 * K);
      if (key < pk + (1ull << (3 * (K - level[order[p - 1]])))) {
        atomicOr(&R->err, kErrOverlap);
        atomicMin(&R->overlap_at, (int)p);
      }
    }
    if (prev != blk) vfirst[blk] = (unsigned)p;
  }
  const unsigned peers = __match_any_sync(0xffffffffu, blk);
  const unsigned b0 = __reduce_or_sync(peers, (unsigned)bit);
  const unsigned b1 = __reduce_or_sync(peers, (unsigned)(bit >> 32));
  const unsigned sp = __reduce_or_sync(peers, sub);
  if (live && (peers & ((1u << lane) - 1u)) == 0u) {
    atomicOr(&m0[blk], ((unsigned long long)b1 << 32) | b0);
    if (sp) atomicOr(&split[blk], 1u);
  }
  for (int a = 0; a < 3; ++a) {
    const int mn = __reduce_min_sync(0xffffffffu, lo[a]);
    const int mx = __reduce_max_sync(0xffffffffu, hi[a]);
    if (lane == 0) {
      atomicMin(&s_box[a], mn);
      atomicMax(&s_box[3 + a], mx);
    }
  }
  __syncthreads();
  if (threadIdx.x < 3)
    atomicMin(&R->box[threadIdx.x], s_box[threadIdx.x]);
  else if (threadIdx.x < 6)
    atomicMax(&R->box[threadIdx.x], s_box[threadIdx.x]);
}

__global__ void k_popcounts(const unsigned long long* __restrict__ m0, long long nb,
                            unsigned* __restrict__ cnt) {
  const long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (b < nb) cnt[b] = (unsigned)__popcll(m0[b]);
}

__global__ void k_mask0(const unsigned long long* __restrict__ m0, const unsigned* __restrict__ rank,
                        const unsigned* __restrict__ split, const unsigned* __restrict__ vfirst,
                        long long nb, uint4* __restrict__ mask0) {
  const long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  const unsigned long long m = m0[b];
  mask0[b] = make_uint4((unsigned)(m & 0xffffffffULL), (unsigned)(m >> 32), rank[b],
                        (m && !split[b]) ? vfirst[b] : 0xffffffffu);
}

// Cell table, level-0 voxels; for split cells their first voxel and a node
// budget (1 + sum of (level - 1) over the cell's voxels).
__global__ void k_cells(const unsigned* __restrict__ order, const unsigned long long* __restrict__ keys,
                        const uint8_t* __restrict__ level, long long n, int K,
                        const uint4* __restrict__ mask0, int2* __restrict__ cells,
                        int* __restrict__ cell_first, unsigned* __restrict__ node_budget,
                        const Report* __restrict__ R) {
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n || (R->err & (kErrLevel | kErrRange))) return;
  const int l = level[order[p]];
  const unsigned long long key = keys[p];
  const uint4 w = mask0[key >> (6 + 3 * K)];
  const unsigned long long m = ((unsigned long long)w.y << 32) | w.x;
  const unsigned bit = (unsigned)(key >> (3 * K)) & 63u;
  const unsigned rank = w.z + (unsigned)__popcll(m & ((1ULL << bit) - 1ULL));
  if (l == 0) {
    cells[rank] = make_int2((int)p, 0);
    return;
  }
  const bool first = p == 0 || (keys[p - 1] >> (3 * K)) != (key >> (3 * K));
  if (first) cell_first[rank] = (int)p;
  atomicAdd(&node_budget[rank], (unsigned)(l - 1) + (first ? 1u : 0u));
}

// One thread per split cell: its nodes (the host build's insertion order,
// node ids from the cell's slice), then the once-split form if it applies.
__global__ void k_nodes(const unsigned* __restrict__ order, const unsigned long long* __restrict__ keys,
                        const uint8_t* __restrict__ level, const int* __restrict__ ijk, long long n,
                        int K, const int* __restrict__ cell_first,
                        const unsigned long long* __restrict__ node_off, long long n_cells,
                        int* __restrict__ nodes, int2* __restrict__ cells) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_cells) return;
  const int p0 = cell_first[r];
  if (p0 < 0) return;
  const int base = (int)node_off[r];
  int next = 1;
  const int root = base;
  const int sh = 3 * K;
  const unsigned long long cell = keys[p0] >> sh;
  for (long long p = p0; p < n && (keys[p] >> sh) == cell; ++p) {
    const unsigned v = order[p];
    const int l = level[v];
    const int i = ijk[3 * (long long)v], j = ijk[3 * (long long)v + 1], k = ijk[3 * (long long)v + 2];
    int node = root;
    for (int dl = 1; dl <= l; ++dl) {
      const int s = l - dl;
      const int slot = ((i >> s) & 1) | (((j >> s) & 1) << 1) | (((k >> s) & 1) << 2);
      int* e = &nodes[(size_t)node * 8 + slot];
      if (dl == l) {
        *e = (int)p;
      } else {
        if (*e == -1) *e = -2 - (base + next++);
        node = -2 - *e;
      }
    }
  }
  unsigned cm = 0;
  int first = -1, expect = -1;
  bool flat = true;
  for (int c = 0; c < 8 && flat; ++c) {
    const int e = nodes[(size_t)root * 8 + c];
    if (e == -1) continue;
    if (e < 0 || (expect >= 0 && e != expect)) flat = false;
    if (first < 0) first = e;
    expect = e + 1;
    cm |= 1u << c;
  }
  cells[r] = (flat && cm) ? make_int2(first, (int)cm) : make_int2(-2 - root, 0);
}

int bit_width_ll(unsigned long long x) {
  int b = 0;
  while (x) {
    ++b;
    x >>= 1;
  }
  return b;
}

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

salf_status salf_build_scene_gpu(salf_ctx* ctx, const salf_scene_desc* d, salf_scene** out) {
  const int K = d->max_level;
  const long long n = d->n;
  cudaError_t ce = cudaSetDevice(ctx->device);
  if (ce != cudaSuccess) return salf_cuda_fail(ce, "cudaSetDevice");
  // grid geometry (host): the same level sizes as the host build
  int mdim[3], brick_p, brick_q;
  salf_grid_shape(d->dims, mdim, &brick_p, &brick_q);
  const long long nb0 = (long long)mdim[0] * mdim[1] * mdim[2];
  Grid G;
  G.K = K;
  for (int a = 0; a < 3; ++a) {
    G.dims[a] = d->dims[a];
    G.mdim[a] = mdim[a];
  }
  const long long nn = std::max(n, 1LL);
  const int key_bits = std::max(1, bit_width_ll((unsigned long long)std::max(nb0 - 1, 1LL)) + 6 + 3 * K);
  if (key_bits > 64) {
    salf_set_error("salf_build_scene: grid too large for 64-bit voxel keys");
    return SALF_ERR_INVALID;
  }

  // temporaries; the ones that start at 0 and at all ones are together
  const long long hn = radix_hist_elems(nn);
  const size_t b_k = a256(nn * 8), b_v = a256(nn * 4), b_h = a256(hn * 4),
               b_ht = a256(kRadix * 4), b_m0 = a256(nb0 * 8), b_b = a256(nb0 * 4),
               b_rt = a256(scan_tmp_elems(nb0) * 4), b_c = K > 0 ? a256(nn * 4) : 0,
               b_no = K > 0 ? a256(nn * 8) : 0, b_nt = K > 0 ? a256(scan_tmp_elems(nn) * 8) : 0;
  PoolBuf tmp;
  if (tmp.get(ctx, 2 * b_k + 2 * b_v + 2 * b_h + b_ht + b_m0 + 4 * b_b + b_rt + 2 * b_c + b_no +
                       b_nt + 256, 0) != SALF_OK) {
    salf_set_error("salf_build_scene: out of device memory (build workspace)");
    return SALF_ERR_OOM;
  }
  char* t = static_cast<char*>(tmp.p);
  size_t o = 0;
  auto take = [&](size_t b) { char* q = t + o; o += b; return q; };
  auto* m0 = reinterpret_cast<unsigned long long*>(take(b_m0));
  auto* split = reinterpret_cast<unsigned*>(take(b_b));
  auto* node_budget = reinterpret_cast<unsigned*>(take(b_c));
  const size_t zeros = o;
  auto* vfirst = reinterpret_cast<unsigned*>(take(b_b));
  auto* cell_first = reinterpret_cast<int*>(take(b_c));
  const size_t ones = o - zeros;
  auto* kA = reinterpret_cast<unsigned long long*>(take(b_k));
  auto* kB = reinterpret_cast<unsigned long long*>(take(b_k));
  auto* vA = reinterpret_cast<unsigned*>(take(b_v));
  auto* vB = reinterpret_cast<unsigned*>(take(b_v));
  auto* hist = reinterpret_cast<unsigned*>(take(b_h));
  auto* hoff = reinterpret_cast<unsigned*>(take(b_h));
  auto* htmp = reinterpret_cast<unsigned*>(take(b_ht));
  auto* cnt = reinterpret_cast<unsigned*>(take(b_b));
  auto* rank = reinterpret_cast<unsigned*>(take(b_b));
  auto* rtmp = reinterpret_cast<unsigned*>(take(b_rt));
  auto* node_off = reinterpret_cast<unsigned long long*>(take(b_no));
  auto* ntmp = reinterpret_cast<unsigned long long*>(take(b_nt));
  auto* report = reinterpret_cast<Report*>(take(256));
  cudaStream_t st = 0;
  const auto grid = [](long long m) { return (unsigned)((std::max(m, 1LL) + 255) / 256); };
  int launches = 0;

  salf_scene* s = new salf_scene();
  struct Guard {
    salf_scene* s;
    bool keep = false;
    ~Guard() {
      if (!keep) salf_scene_destroy(s);
    }
  } guard{s};
  salf_scene_hold_ctx(s, ctx);
  s->n = n;
  s->mode = d->mode;
  s->dtype = d->dtype;
  s->K = K;
  for (int a = 0; a < 3; ++a) {
    s->dims[a] = d->dims[a];
    s->origin[a] = d->origin[a];
  }
  s->s0 = d->s0;
  s->sfin = d->s0 / (double)(1 << K);
  DevScene& D = s->dev;
  std::memset(&D, 0, sizeof(D));
  salf_status sst;
  auto alloc = [&](size_t bytes, void** p) { return salf_scene_dalloc(s, bytes, p); };
  // every cell holds a voxel, so n entries are enough for the cell table
  void *pmask0 = nullptr, *pcells = nullptr, *pord = nullptr, *pbox = nullptr, *pstatus = nullptr,
       *params = nullptr;
  const size_t rec_bytes = d->dtype == SALF_F32 ? 128 : 64;
  if ((sst = alloc(nb0 * sizeof(uint4), &pmask0)) != SALF_OK ||
      (sst = alloc(nn * sizeof(int2), &pcells)) != SALF_OK ||
      (sst = salf_scene_block(s, nn * sizeof(int), &pord)) != SALF_OK ||
      (sst = alloc(nn * sizeof(int4), &pbox)) != SALF_OK ||
      (sst = alloc(16, &pstatus)) != SALF_OK ||
      (sst = salf_scene_block(s, nn * rec_bytes, &params)) != SALF_OK)
    return sst;
  uint4* mask0 = static_cast<uint4*>(pmask0);
  int2* cells = static_cast<int2*>(pcells);
  D.mask0 = mask0;
  D.mdim0 = mdim[0];
  D.mdim01 = mdim[0] * mdim[1];
  D.cells = cells;
  D.order = static_cast<int*>(pord);
  D.vox_box = static_cast<int4*>(pbox);
  D.status = static_cast<int*>(pstatus);
  D.params = params;
  for (int a = 0; a < 3; ++a) {
    D.origin[a] = d->origin[a];
    D.Gf[a] = d->dims[a] << K;
  }
  D.inv_sfin = 1.0 / s->sfin;
  salf_view_pairs(&D);
  D.K = K;
  D.mode = d->mode;
  D.dtype = d->dtype;
  D.n = (int)n;
  if ((ce = cudaMemsetAsync(t, 0, zeros, st)) != cudaSuccess ||
      (ce = cudaMemsetAsync(t + zeros, 0xff, ones, st)) != cudaSuccess ||
      (ce = cudaMemsetAsync(pstatus, 0, 16, st)) != cudaSuccess ||
      (n == 0 && ((ce = cudaMemsetAsync(pord, 0, sizeof(int), st)) != cudaSuccess ||
                  (ce = cudaMemsetAsync(pbox, 0, sizeof(int4), st)) != cudaSuccess ||
                  (ce = cudaMemsetAsync(pcells, 0xff, sizeof(int2), st)) != cudaSuccess)))
    return salf_cuda_fail(ce, "build workspace init");
  k_report_init<<<1, 1, 0, st>>>(report);

  // 1. keys and sort; 2. words, boxes, ranks
  const uint8_t* level = d->level;
  const int* ijk = d->ijk;
  unsigned long long* keys = kA;
  unsigned* order = vA;
  if (n > 0) {
    k_keys<<<grid(n), 256, 0, st>>>(level, ijk, n, G, kA, vA, report);
    if ((ce = radix_sort_pairs(kA, vA, kB, vB, n, key_bits, hist, hoff, htmp, st, &launches, &keys,
                               &order)) != cudaSuccess)
      return salf_cuda_fail(ce, "build sort");
    k_voxels<<<grid(n), 256, 0, st>>>(keys, order, level, ijk, n, K, m0, split, vfirst,
                                      static_cast<int*>(pord), static_cast<int4*>(pbox), report);
  }
  k_popcounts<<<grid(nb0), 256, 0, st>>>(m0, nb0, cnt);
  if ((ce = scan_exclusive<unsigned, unsigned>(cnt, nb0, rank, rtmp, st, &launches)) != cudaSuccess)
    return salf_cuda_fail(ce, "build rank scan");
  k_mask0<<<grid(nb0), 256, 0, st>>>(m0, rank, split, vfirst, nb0, mask0);

  // 3. cell table and records, then the read-back
  if (n > 0) {
    k_cells<<<grid(n), 256, 0, st>>>(order, keys, level, n, K, mask0, cells, cell_first,
                                     node_budget, report);
    if (K > 0 && (ce = scan_exclusive<unsigned, unsigned long long>(node_budget, n, node_off, ntmp,
                                                                    st, &launches)) != cudaSuccess)
      return salf_cuda_fail(ce, "build node scan");
    // (the sorted order, which is a permutation also when a key was out of range)
    if ((ce = salf_launch_gather_params(d->params, reinterpret_cast<const int*>(order), params, n,
                                        d->dtype, d->mode, D.status, st)) != cudaSuccess)
      return salf_cuda_fail(ce, "gather params");
  }
  k_report<<<1, 1, 0, st>>>(report, rank, cnt, nb0, n > 0 && K > 0 ? node_off : nullptr,
                            node_budget, n, D.status);
  Report h;
  if ((ce = cudaMemcpyAsync(&h, report, sizeof(h), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
      (ce = cudaStreamSynchronize(st)) != cudaSuccess)
    return salf_cuda_fail(ce, "build checks");
  if (h.err & (kErrLevel | kErrRange)) {
    salf_set_error("salf_build_scene: voxel " + std::to_string(h.bad_voxel) +
                   ((h.err & kErrLevel) ? " has level > max_level" : " outside the grid"));
    return SALF_ERR_INVALID;
  }
  if (h.err & kErrOverlap) {
    unsigned pair[2] = {0, 0};
    cudaMemcpy(pair, order + h.overlap_at - 1, 8, cudaMemcpyDeviceToHost);
    salf_set_error("salf_build_scene: voxels " + std::to_string(pair[0]) + " and " +
                   std::to_string(pair[1]) + " overlap");
    return SALF_ERR_OVERLAP;
  }
  if (h.status & SALF_DEVERR_SDF_AB) {
    salf_set_error("salf_build_scene: SDF records need a > 0 and b > 0 (Eq. 6)");
    return SALF_ERR_INVALID;
  }
  for (int a = 0; a < 3; ++a) {
    D.bmin[a] = n > 0 ? h.box[a] : 0;
    D.bmax[a] = n > 0 ? h.box[3 + a] : 0;
  }
  s->n_cells0 = h.n_cells;
  s->n_nodes = (int64_t)h.n_nodes;

  // 4. nodes and skip boxes
  const size_t nodes_n = std::max<unsigned long long>(h.n_nodes, 1);
  void* pnodes = nullptr;
  if ((sst = alloc(nodes_n * 8 * sizeof(int), &pnodes)) != SALF_OK) return sst;
  D.nodes = static_cast<int*>(pnodes);
  if ((ce = cudaMemsetAsync(pnodes, 0xff, nodes_n * 8 * sizeof(int), st)) != cudaSuccess)
    return salf_cuda_fail(ce, "build nodes init");
  if (h.n_nodes > 0)
    k_nodes<<<grid(h.n_cells), 256, 0, st>>>(order, keys, level, ijk, n, K, cell_first, node_off,
                                             h.n_cells, static_cast<int*>(pnodes), cells);
  if ((sst = salf_build_skip(s, brick_p, brick_q, st)) != SALF_OK) return sst;
  if ((ce = cudaStreamSynchronize(st)) != cudaSuccess) return salf_cuda_fail(ce, "build");
  guard.keep = true;
  *out = s;
  return SALF_OK;
}
