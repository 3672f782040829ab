// refine.cu -- densification and pruning of a scene's voxel set (Sec. III-C).
//
// Plan (one thread per voxel): a voxel whose largest composited alpha is
// below the pruning threshold is removed; otherwise a voxel above the finest
// level whose colour-field gradient L1 norm (record slots 4..12) exceeds the
// split threshold becomes its 8 octree children; the rest are kept.  An
// exclusive scan of the output counts (0, 8 or 1) places every voxel's
// output in input order, children in place of their parent.
// Apply (8 lanes per voxel): writes level, cell and record of each output
// voxel.  A child's record carries its parent's fields exactly: every field
// is affine in the local coordinates and x_parent = (x_child + o) / 2 with
// o in {-1, +1}^3, so the slopes halve and the offsets take W . o / 2 (the
// colour rows have no offset of their own: theirs goes to the SH DC term
// through C0 = 1 / (2 sqrt(pi))).
#include <cstring>
#include <mutex>

#include "scan.cuh"
#include "traverse.cuh"

using namespace salf_scan;

namespace {

constexpr float kSH0 = 0.28209479177387814f;

// In input order, from the scene's keys: neighbouring threads read neighbouring
// rows; the counts are summed over a block before their atomics (1M voxels: 27 us;
// in voxel order with an atomic per warp and count 57).
__global__ void __launch_bounds__(256) k_refine_plan(
    const uint8_t* __restrict__ key_level, int n, int K, const float* __restrict__ grads,
    const float* __restrict__ max_alpha, float split_thr, float prune_alpha,
    unsigned char* __restrict__ action, unsigned* __restrict__ count,
    unsigned long long* __restrict__ stats) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  int act = -1;
  if (v < n) {
    const int level = __ldg(&key_level[v]);
    const float4* g = reinterpret_cast<const float4*>(grads) + (size_t)v * 8;
    const float4 g1 = __ldg(g + 1), g2 = __ldg(g + 2), g3 = __ldg(g + 3);  // slots 4..15
    const float l1 = fabsf(g1.x) + fabsf(g1.y) + fabsf(g1.z) + fabsf(g1.w) + fabsf(g2.x) +
                     fabsf(g2.y) + fabsf(g2.z) + fabsf(g2.w) + fabsf(g3.x);
    const float a = __ldg(&max_alpha[v]);
    act = a < prune_alpha ? 2 : ((level < K && l1 > split_thr) ? 1 : 0);
    action[v] = (unsigned char)act;
    count[v] = act == 0 ? 1u : (act == 1 ? 8u : 0u);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int c = __syncthreads_count(act == k);
    if (threadIdx.x == 0 && c) atomicAdd(&stats[k], (unsigned long long)c);
  }
}

// 8 lanes per voxel, a 16-byte chunk of the record each, so that every row is
// read and written as one 128-byte line; kRows voxels per group, whose loads are
// in flight together.  A child's chunk needs other chunks' colour rows and
// intensity slopes: shuffles inside the 8 lanes; all lanes run the same code (a
// switch over the chunks cost as much as the scattered rows saved).  1M voxels
// in, 1.27M out (310 MB): 59 us; a thread per voxel 101.
constexpr int kRows = 4;

__global__ void __launch_bounds__(256) k_refine_apply(
    const uint8_t* __restrict__ key_level, const int* __restrict__ key_ijk, int n,
    const unsigned char* __restrict__ action, const unsigned long long* __restrict__ offs,
    const float* __restrict__ params, unsigned char* __restrict__ level_out,
    int* __restrict__ ijk_out, float* __restrict__ params_out) {
  const int k = (int)(threadIdx.x & 7);  // chunk: slots 4 k .. 4 k + 3
  const long long v0 = blockIdx.x * (32LL * kRows) + (threadIdx.x >> 3);
  int act[kRows], level[kRows], cell[kRows];  // cell: axis k of ijk on lanes 0..2
  unsigned long long o[kRows];
  float4 rec[kRows];
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
    const long long v = v0 + 32 * j;
    act[j] = v < n ? __ldg(&action[v]) : 2;
    rec[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    o[j] = 0;
    level[j] = cell[j] = 0;
    if (v < n) {
      rec[j] = __ldg(reinterpret_cast<const float4*>(params) + v * 8 + k);
      o[j] = __ldg(&offs[v]);
      level[j] = __ldg(&key_level[v]);
      if (k < 3) cell[j] = __ldg(&key_ijk[3 * v + k]);
    }
  }
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
    const float4 q = rec[j];
    float4* dst = reinterpret_cast<float4*>(params_out) + (size_t)o[j] * 8 + k;
    if (act[j] == 0) {
      *dst = q;
      if (k == 0) level_out[o[j]] = (unsigned char)level[j];
      if (k < 3) ijk_out[3 * o[j] + k] = cell[j];
    }
    if (!__any_sync(0xffffffffu, act[j] == 1)) continue;
    const unsigned full = 0xffffffffu;
    const int ijk[3] = {__shfl_sync(full, cell[j], 0, 8), __shfl_sync(full, cell[j], 1, 8),
                        __shfl_sync(full, cell[j], 2, 8)};
    // slots 4..12 (colour rows) and 27 for every lane of the voxel
    const float c4 = __shfl_sync(full, q.x, 1, 8), c5 = __shfl_sync(full, q.y, 1, 8),
                c6 = __shfl_sync(full, q.z, 1, 8), c7 = __shfl_sync(full, q.w, 1, 8),
                c8 = __shfl_sync(full, q.x, 2, 8), c9 = __shfl_sync(full, q.y, 2, 8),
                c10 = __shfl_sync(full, q.z, 2, 8), c11 = __shfl_sync(full, q.w, 2, 8),
                c12 = __shfl_sync(full, q.x, 3, 8), c27 = __shfl_sync(full, q.w, 6, 8);
    if (act[j] != 1) continue;
    level_out[o[j] + k] = (unsigned char)(level[j] + 1);
#pragma unroll
    for (int a = 0; a < 3; ++a) ijk_out[3 * (o[j] + k) + a] = 2 * ijk[a] + ((k >> a) & 1);
    // slopes halve (hx..hw), and one component of the chunk moves by half of
    // (A, B, C) . s, over C0 where it is an SH DC term
    const bool sh = k >= 3 && k <= 5;
    const float A = k == 0 ? q.x : (k == 3 ? c4 : (k == 4 ? c7 : (k == 5 ? c10 : c27)));
    const float B = k == 0 ? q.y : (k == 3 ? c5 : (k == 4 ? c8 : (k == 5 ? c11 : q.x)));
    const float C = k == 0 ? q.z : (k == 3 ? c6 : (k == 4 ? c9 : (k == 5 ? c12 : q.y)));
    const float hx = sh && k != 3 ? 1.f : (k == 6 ? 1.f : 0.5f);
    const float hy = sh || k == 6 ? 1.f : 0.5f;
    const float hz = sh || k == 6 || k == 7 ? 1.f : 0.5f;
    const float hw = k == 1 || k == 2 || k == 6 ? 0.5f : 1.f;
    const float4 base = make_float4(hx * q.x, hy * q.y, hz * q.z, hw * q.w);
    for (int c = 0; c < 8; ++c) {
      const float s[3] = {(c & 1) ? 1.f : -1.f, (c & 2) ? 1.f : -1.f, (c & 4) ? 1.f : -1.f};
      float t = 0.5f * (A * s[0] + B * s[1] + C * s[2]);
      if (sh) t = t / kSH0;
      float4 out = base;
      if (sh) out.y += t;
      if (k == 0) out.w += t;
      if (k == 7) out.z += t;
      dst[8 * c] = out;
    }
  }
}

// Density of the geometry value g (Eq. 1 or Eq. 6) and its derivatives with
// respect to g, a and b.
template <int MODE>
__device__ __forceinline__ float reg_density(float g, float a, float b, float* d_g, float* d_a,
                                             float* d_b) {
  if (MODE == SALF_FIELD_EXP) {
    const float s = __expf(g);
    *d_g = s;
    *d_a = *d_b = 0.f;
    return s;
  }
  const float e = __expf(-fabsf(g) / b);
  const float sg = g > 0.f ? 1.f : (g < 0.f ? -1.f : 0.f);
  const float s = 0.5f * a + 0.5f * a * sg * (1.f - e);
  *d_g = 0.5f * a * e / b;
  *d_a = s / a;
  *d_b = -0.5f * a * g * e / (b * b);
  return s;
}

// Adds a record's gradient of W (slots 0..3) and, in SDF mode, of a and b (slots
// 25, 26) to its row: one 16-byte vector atomic each when the buffer is 16-byte
// aligned (VEC).
template <int MODE, bool VEC>
__device__ __forceinline__ void reg_add(float* __restrict__ grads, int v, const float g[6]) {
  float* G = grads + (size_t)v * 32;
  if constexpr (VEC) {
    atomicAdd(reinterpret_cast<float4*>(G), make_float4(g[0], g[1], g[2], g[3]));
    if (MODE == SALF_FIELD_SDF)
      atomicAdd(reinterpret_cast<float4*>(G + 24), make_float4(0.f, g[4], g[5], 0.f));
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) atomicAdd(G + q, g[q]);
    if (MODE == SALF_FIELD_SDF) {
      atomicAdd(G + 25, g[4]);
      atomicAdd(G + 26, g[5]);
    }
  }
}

// Eq. 7's L_reg over the face-adjacent pairs, one thread per voxel: across
// each face, the voxel owning the finest cell just outside its min corner is
// the neighbour when it is at least as large (then it covers the whole face).
// At the centre of the shared face: s = W.[x,1], alpha = 1 - exp(-sigma(s) l)
// (l: the smaller edge, m), n = W[0:3] / |W[0:3]|.  The loss counts a pair once,
// at its smaller voxel, or at the one on the - side when both are equal.
//
// Gradients: both voxels of an equal pair work the pair out, each for itself,
// so a voxel gathers its own gradient in registers and adds it with one or two
// vector atomics; only a smaller voxel adds its larger neighbour's part.  (With
// each pair worked out once and both parts added by scalar atomics the kernel
// was bound by them, 12 per pair in SDF mode: 1M voxels, SDF, 216 us.)  The
// loss is summed over a block, then over blocks by k_reg_total, in 64 bits:
// thousands of FP32 atomics on one scalar would round it by 1e-6 and more.
template <int MODE, bool VEC>
__global__ void __launch_bounds__(256) k_reg_loss(const __grid_constant__ DevScene S,
                                                  const float* __restrict__ params, float lam_s,
                                                  float lam_a, float lam_n, float sfin,
                                                  float* __restrict__ loss,
                                                  float* __restrict__ partial,
                                                  float* __restrict__ grads) {
  __shared__ float s_acc[8];
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const float4* rec = reinterpret_cast<const float4*>(params);
  float acc = 0.f;
  if (p < S.n) {
    const int4 bi = __ldg(&S.vox_box[p]);
    const int E = 1 << bi.w;
    const int lo[3] = {bi.x, bi.y, bi.z};
    const int vi = __ldg(&S.order[p]);
    const float4 wi = __ldg(rec + (size_t)vi * 8);
    float4 abi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (MODE == SALF_FIELD_SDF) abi = __ldg(rec + (size_t)vi * 8 + 6);
    const float Wi[4] = {wi.x, wi.y, wi.z, wi.w};
    const float ni = sqrtf(Wi[0] * Wi[0] + Wi[1] * Wi[1] + Wi[2] * Wi[2]);
    const float ell = (float)E * sfin;
    float g[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // own gradient: slots 0..3, a, b
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const int ax = f >> 1;
      const int sgn = (f & 1) ? 1 : -1;
      int c[3] = {lo[0], lo[1], lo[2]};
      c[ax] = sgn > 0 ? lo[ax] + E : lo[ax] - 1;
      if (c[ax] < 0 || c[ax] >= S.Gf[ax]) continue;
      int lsj, lz;
      const int j = salf::find_leaf(S, c[0], c[1], c[2], &lsj, &lz);
      if (j < 0 || lsj < bi.w) continue;
      const bool equal = lsj == bi.w;
      const int vj = __ldg(&S.order[j]);
      const float4 wj = __ldg(rec + (size_t)vj * 8);
      float4 abj = make_float4(0.f, 0.f, 0.f, 0.f);
      if (MODE == SALF_FIELD_SDF) abj = __ldg(rec + (size_t)vj * 8 + 6);
      const float Wj[4] = {wj.x, wj.y, wj.z, wj.w};
      // local coordinates of the face centre: +-1 on the axis in i; in j from its
      // box, the aligned one around the cell (2 / edge is an exact power of two)
      const float Ej = (float)(1 << lsj);
      const float inv_half = __int_as_float((128 - lsj) << 23);
      float xi[3] = {0.f, 0.f, 0.f}, xj[3];
      xi[ax] = (float)sgn;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float X = a == ax ? (float)(sgn > 0 ? lo[a] + E : lo[a]) : (float)lo[a] + 0.5f * E;
        xj[a] = (X - ((float)(c[a] >> lsj << lsj) + 0.5f * Ej)) * inv_half;
      }
      const float si = Wi[ax] * xi[ax] + Wi[3];
      const float sj = Wj[0] * xj[0] + Wj[1] * xj[1] + Wj[2] * xj[2] + Wj[3];
      float gi_g, gi_a, gi_b, gj_g, gj_a, gj_b;
      const float sigi = reg_density<MODE>(si, abi.y, abi.z, &gi_g, &gi_a, &gi_b);
      const float sigj = reg_density<MODE>(sj, abj.y, abj.z, &gj_g, &gj_a, &gj_b);
      const float ei = __expf(-sigi * ell), ej = __expf(-sigj * ell);
      const float ds = si - sj, da = ej - ei;  // alpha_i - alpha_j = e_j - e_i
      const float nj = sqrtf(Wj[0] * Wj[0] + Wj[1] * Wj[1] + Wj[2] * Wj[2]);
      float ui[3] = {0.f, 0.f, 0.f}, uj[3] = {0.f, 0.f, 0.f};
      if (ni > 0.f)
        for (int a = 0; a < 3; ++a) ui[a] = Wi[a] / ni;
      if (nj > 0.f)
        for (int a = 0; a < 3; ++a) uj[a] = Wj[a] / nj;
      const float dot = ui[0] * uj[0] + ui[1] * uj[1] + ui[2] * uj[2];
      if (!equal || sgn > 0) acc += lam_s * fabsf(ds) + lam_a * fabsf(da) + lam_n * (1.f - dot);
      const float cs = lam_s * (ds > 0.f ? 1.f : (ds < 0.f ? -1.f : 0.f));
      const float ca = lam_a * (da > 0.f ? 1.f : (da < 0.f ? -1.f : 0.f));
      // d alpha_k / d sigma_k = exp(-sigma_k l) l
      const float ki = ca * ei * ell, kj = -ca * ej * ell;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        g[a] += cs * xi[a] + ki * gi_g * xi[a];
        if (ni > 0.f) g[a] -= lam_n * (uj[a] - ui[a] * dot) / ni;
      }
      g[3] += cs + ki * gi_g;
      g[4] += ki * gi_a;
      g[5] += ki * gi_b;
      if (!equal) {
        float gj[6];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          gj[a] = -cs * xj[a] + kj * gj_g * xj[a];
          if (nj > 0.f) gj[a] -= lam_n * (ui[a] - uj[a] * dot) / nj;
        }
        gj[3] = -cs + kj * gj_g;
        gj[4] = kj * gj_a;
        gj[5] = kj * gj_b;
        reg_add<MODE, VEC>(grads, vj, gj);
      }
    }
    reg_add<MODE, VEC>(grads, vi, g);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) s_acc[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) sum += s_acc[k];
    if (partial)
      partial[blockIdx.x] = sum;
    else if (sum != 0.f)
      atomicAdd(loss, sum);
  }
}

// The blocks' sums, added to the loss once (4 us).
__global__ void __launch_bounds__(1024) k_reg_total(const float* __restrict__ partial, int n,
                                                    float* __restrict__ loss) {
  __shared__ double s_acc[32];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += 1024) acc += (double)__ldg(&partial[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) s_acc[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc = s_acc[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (threadIdx.x == 0 && acc != 0.0) atomicAdd(loss, (float)acc);
  }
}

template <int MODE, bool VEC>
void launch_reg(const DevScene& D, const float* params, float lam_s, float lam_a, float lam_n,
                float sfin, float* loss, float* partial, float* grads, cudaStream_t st) {
  k_reg_loss<MODE, VEC><<<(unsigned)((D.n + 255) / 256), 256, 0, st>>>(
      D, params, lam_s, lam_a, lam_n, sfin, loss, partial, grads);
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

bool misaligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0; }

}  // namespace

extern "C" salf_status salf_scene_refine_plan(salf_scene* sc, const float* grads,
                                             const float* max_alpha, float split_threshold,
                                             float prune_alpha, salf_refine_counts* counts,
                                             void* stream) {
  SALF_RANGE("salf_scene_refine_plan");
  if (!sc || !grads || !max_alpha || !counts) {
    salf_set_error("salf_scene_refine_plan: null argument");
    return SALF_ERR_INVALID;
  }
  if (misaligned16(grads)) {
    salf_set_error("salf_scene_refine_plan: grads must be 16-byte aligned");
    return SALF_ERR_INVALID;
  }
  cudaError_t e;
  if ((e = cudaSetDevice(sc->device)) != cudaSuccess) return salf_cuda_fail(e, "cudaSetDevice");
  std::lock_guard<std::mutex> lk(sc->refine_mu);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const long long n = sc->n, nn = n > 0 ? n : 1;
  const size_t b_act = align256(nn), b_cnt = align256(nn * 4), b_offs = align256((nn + 1) * 8),
               b_tmp = align256(scan_tmp_elems(nn) * 8), b_stats = 256;
  const size_t need = b_act + b_cnt + b_offs + b_tmp + b_stats;
  if (sc->refine_ws_bytes < need) {
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return salf_cuda_fail(e, "refine sync");
    if (sc->refine_ws) cudaFree(sc->refine_ws);
    sc->refine_ws = nullptr;
    sc->refine_ws_bytes = 0;
    if (salf_dev_malloc(sc->ctx, &sc->refine_ws, need) != cudaSuccess) {
      cudaGetLastError();
      salf_set_error("salf_scene_refine_plan: out of device memory");
      return SALF_ERR_OOM;
    }
    sc->refine_ws_bytes = need;
  }
  if (!sc->refine_host &&
      cudaMallocHost(reinterpret_cast<void**>(&sc->refine_host), 64) != cudaSuccess) {
    cudaGetLastError();
    salf_set_error("salf_scene_refine_plan: cudaMallocHost failed");
    return SALF_ERR_OOM;
  }
  char* w = static_cast<char*>(sc->refine_ws);
  unsigned char* action = reinterpret_cast<unsigned char*>(w);
  unsigned* count = reinterpret_cast<unsigned*>(w + b_act);
  unsigned long long* offs = reinterpret_cast<unsigned long long*>(w + b_act + b_cnt);
  unsigned long long* tmp = reinterpret_cast<unsigned long long*>(w + b_act + b_cnt + b_offs);
  unsigned long long* stats =
      reinterpret_cast<unsigned long long*>(w + b_act + b_cnt + b_offs + b_tmp);
  if ((e = cudaMemsetAsync(stats, 0, 4 * sizeof(unsigned long long), st)) != cudaSuccess)
    return salf_cuda_fail(e, "refine stats");
  if (n > 0) {
    const DevScene& D = sc->dev;
    k_refine_plan<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
        sc->key_level, (int)n, D.K, grads, max_alpha, split_threshold, prune_alpha, action, count,
        stats);
    int launches = 0;
    if ((e = scan_exclusive<unsigned, unsigned long long>(count, n, offs, tmp, st, &launches)) !=
        cudaSuccess)
      return salf_cuda_fail(e, "refine scan");
    k_scan_total<unsigned, unsigned long long><<<1, 1, 0, st>>>(count, n, offs);
    if ((e = cudaMemcpyAsync(stats + 3, offs + n, 8, cudaMemcpyDeviceToDevice, st)) !=
        cudaSuccess)
      return salf_cuda_fail(e, "refine total");
  }
  if ((e = cudaMemcpyAsync(sc->refine_host, stats, 4 * sizeof(unsigned long long),
                           cudaMemcpyDeviceToHost, st)) != cudaSuccess)
    return salf_cuda_fail(e, "refine counts");
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return salf_cuda_fail(e, "refine plan");
  counts->n_kept = (int64_t)sc->refine_host[0];
  counts->n_split = (int64_t)sc->refine_host[1];
  counts->n_pruned = (int64_t)sc->refine_host[2];
  counts->n_new = n > 0 ? (int64_t)sc->refine_host[3] : 0;
  sc->refine_planned = true;
  sc->refine_n_new = counts->n_new;
  return SALF_OK;
}

extern "C" salf_status salf_scene_refine_apply(salf_scene* sc, const float* params,
                                              uint8_t* level_out, int32_t* ijk_out,
                                              float* params_out, void* stream) {
  SALF_RANGE("salf_scene_refine_apply");
  if (!sc || !params) {
    salf_set_error("salf_scene_refine_apply: null argument");
    return SALF_ERR_INVALID;
  }
  std::lock_guard<std::mutex> lk(sc->refine_mu);
  if (!sc->refine_planned) {
    salf_set_error("salf_scene_refine_apply: no plan (call salf_scene_refine_plan first)");
    return SALF_ERR_INVALID;
  }
  if (sc->refine_n_new > 0 && (!level_out || !ijk_out || !params_out)) {
    salf_set_error("salf_scene_refine_apply: null output");
    return SALF_ERR_INVALID;
  }
  if (misaligned16(params) || misaligned16(params_out)) {
    salf_set_error("salf_scene_refine_apply: params and params_out must be 16-byte aligned");
    return SALF_ERR_INVALID;
  }
  cudaError_t e;
  if ((e = cudaSetDevice(sc->device)) != cudaSuccess) return salf_cuda_fail(e, "cudaSetDevice");
  const long long n = sc->n, nn = n > 0 ? n : 1;
  char* w = static_cast<char*>(sc->refine_ws);
  const size_t b_act = align256(nn), b_cnt = align256(nn * 4);
  const unsigned char* action = reinterpret_cast<const unsigned char*>(w);
  const unsigned long long* offs = reinterpret_cast<const unsigned long long*>(w + b_act + b_cnt);
  if (n > 0 && sc->refine_n_new > 0) {
    k_refine_apply<<<(unsigned)((n + 32 * kRows - 1) / (32 * kRows)), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        sc->key_level, sc->key_ijk, (int)n, action, offs, params, level_out, ijk_out, params_out);
    if ((e = cudaGetLastError()) != cudaSuccess) return salf_cuda_fail(e, "refine apply");
  }
  return SALF_OK;
}

extern "C" salf_status salf_scene_reg_loss(salf_scene* sc, const float* params, float lambda_s,
                                          float lambda_alpha, float lambda_n, float* loss,
                                          float* grads, void* stream) {
  SALF_RANGE("salf_scene_reg_loss");
  if (!sc || !params || !loss || !grads) {
    salf_set_error("salf_scene_reg_loss: null argument");
    return SALF_ERR_INVALID;
  }
  if (misaligned16(params)) {
    salf_set_error("salf_scene_reg_loss: params must be 16-byte aligned");
    return SALF_ERR_INVALID;
  }
  cudaError_t e;
  if ((e = cudaSetDevice(sc->device)) != cudaSuccess) return salf_cuda_fail(e, "cudaSetDevice");
  const DevScene& D = sc->dev;
  if (D.n > 0) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool vec = !misaligned16(grads);
    const auto run = D.mode == SALF_FIELD_EXP
                         ? (vec ? launch_reg<SALF_FIELD_EXP, true> : launch_reg<SALF_FIELD_EXP, false>)
                         : (vec ? launch_reg<SALF_FIELD_SDF, true> : launch_reg<SALF_FIELD_SDF, false>);
    // up to 32 blocks add their sums themselves, within 32 roundings; so do more
    // where the device has no room for the sums
    const int blocks = (int)((D.n + 255) / 256);
    PoolBuf part;
    if (blocks > 32) (void)part.get(sc->ctx, (size_t)blocks * 4, st);
    float* partial = static_cast<float*>(part.p);
    run(D, params, lambda_s, lambda_alpha, lambda_n, (float)sc->sfin, loss, partial, grads, st);
    if (partial) k_reg_total<<<1, 1024, 0, st>>>(partial, blocks, loss);
    if ((e = cudaGetLastError()) != cudaSuccess) return salf_cuda_fail(e, "reg loss launch");
  }
  return SALF_OK;
}
