// backward.cu -- hand-written adjoint of the forward ray-cast kernel.
//
// For L with per-ray gradients g = dL/d(rgb, depth, opacity, intensity) the
// kernel re-traverses each ray, recomputes the transmittance front to back
// (nothing per voxel is stored by the forward pass), and uses the saved
// per-ray totals Q = (C, D, O, I) for the suffix sums:
//   w_k = T_k alpha_k,  q_k = (c_k, t_mid,k, 1, iota_k),
//   dL/dtau_k = T_{k+1} (g . q_k) - (g . Q - sum_{j<=k} w_j g . q_j)
//               - T_end (g_rgb . background),     tau_k = sigma_k delta_k,
// then chains through Eq. 1 (d sigma / d W = sigma [x, 1]) or Eq. 5-6
// (d sigma / d s = a e^{-|s|/b} / (2b), d sigma / d a = sigma / a,
//  d sigma / d b = -a s e^{-|s|/b} / (2 b^2)) and Eq. 2 (d c / d z = c (1 - c),
// d z / d W_c = x, d z / d W_sh = gamma).  The raydrop output adds
// q_k = sigmoid(rho_k) and a background of 1 (T_end), and d/d rho_k =
// w_k s (1 - s).  Each round, the lanes with a hit walk their rays in order
// (T, the suffix sums and dL/dtau need it) and queue the hit's coefficients
// in a per-warp ring in shared memory; whenever 32 are queued, the whole warp
// builds their 32-scalar gradient rows and adds them to the caller's
// input-order FP32 buffer with 16-byte vector atomics.  Where 4 or more rows of
// a batch are of one voxel, they are staged in shared memory and summed first,
// so that a buffer's scalar is rounded once per batch, not once per row.
//
// Bound by instruction issue (59% of slots, 24 of 32 lanes) and the waits for
// shared memory and records.  The sums run on the whole warp at once, whatever its
// groups: with barriers inside each group the groups took turns.  Adjoint of 8
// views of 960x640 on 1M voxels (BF16; SDF in F32; a LiDAR of 64x1024 on it), us:
//   groups of 4 or more, one sum a batch   1446   1769   297
//   groups of 3 or more; of 2 or more      1489   1808;  1517   1840
//   groups of 6 or more                    1440   1785
// Without the split into parts the long groups' loops take 1763; with up to 8
// parts instead of 4 it is 1610 (registers).  Each part with atomics of its own
// took 1425 / 1779 / 326, but 2 to 8 roundings per batch: the run-to-run noise of
// gradients doubled, and tripled where voxels are large on the screen.
#include "traverse.cuh"

// warps per block
#ifndef SALF_BWD_WARPS
#define SALF_BWD_WARPS 4
#endif
// Resident blocks per SM: static pinholes 5 (94 to 96 registers; 4: 1557 us for the 8
// views), the rest 4 (114; 5: LiDAR 332 us instead of 307, with spills).
#ifndef SALF_BWD_BLOCKS_LEAN
#define SALF_BWD_BLOCKS_LEAN 5
#endif
#ifndef SALF_BWD_BLOCKS
#define SALF_BWD_BLOCKS 4
#endif

using namespace salf;

// LEAN: every request is a pinhole camera with one pose for the frame and
// asks for neither intensity nor raydrop gradients: only that ray generation
// and no intensity or raydrop terms are compiled in (8-camera training
// adjoint measured 1.5% faster).
template <int DT, int MODE, bool LEAN>
__global__ void __launch_bounds__(32 * SALF_BWD_WARPS,
                                  LEAN ? SALF_BWD_BLOCKS_LEAN : SALF_BWD_BLOCKS)
    k_backward(const __grid_constant__ LaunchParams P) {
  // see next_hit: LiDAR fit 464 -> 443 us, 2400x128 on 1.5M voxels 721 -> 686 (SDF 823 ->
  // 783); training step (cameras) 2640 -> 2615, but for SDF fields 4126 -> 4279
  constexpr bool AHEAD = !LEAN || MODE == SALF_FIELD_EXP;
  const int warp = blockIdx.x * SALF_BWD_WARPS + (threadIdx.x >> 5);
  if (warp >= P.total_tiles) return;
  const int lane = threadIdx.x & 31;
  const ReqDev& Q = P.req[find_request(P, warp)];
  const DevScene& S = P.S;
  const int tile = warp - Q.tile_begin;
  // the actor adjoint takes these tiles
  if (Q.tile_skip && (__ldg(&Q.tile_skip[tile >> 5]) >> (tile & 31)) & 1u) return;
  int u0, v0;
  tile_origin(Q, tile, &u0, &v0);
  const int u = u0 + (lane & (Q.tile_w - 1));
  const int v = v0 + (lane >> Q.tile_ws);
  const bool in_img = (u < Q.W) && (v < Q.H);
  const int ray = v * Q.W + u;

  Ray r;
  Walk w;
  w.alive = false;
  r.valid = false;
  r.d[0] = r.d[1] = r.d[2] = 0.f;
  float g[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float gQ = 0.f, Tend = 1.f, gp = 0.f;
  int nv = 0;
  if (in_img) {
    if (LEAN)
      gen_ray_pinhole(Q, u, v, r);
    else
      gen_ray(Q, S, u, v, ray, r);
    walk_init<AHEAD>(S, r, w);
    const float4* sp = reinterpret_cast<const float4*>(Q.bsaved) + 2 * (size_t)ray;
    const float4 s0 = __ldg(sp), s1 = __ldg(sp + 1);
    if (Q.g_rgb) {
      g[0] = __ldg(Q.g_rgb + 3 * (size_t)ray);
      g[1] = __ldg(Q.g_rgb + 3 * (size_t)ray + 1);
      g[2] = __ldg(Q.g_rgb + 3 * (size_t)ray + 2);
    }
    if (Q.g_depth) g[3] = __ldg(Q.g_depth + ray);
    if (Q.g_opacity) g[4] = __ldg(Q.g_opacity + ray);
    if (Q.g_int && Q.want_int) g[5] = __ldg(Q.g_int + ray);
    gQ = g[0] * s0.x + g[1] * s0.y + g[2] * s0.z + g[3] * s0.w + g[4] * s1.x + g[5] * s1.y;
    Tend = s1.z;
    if (Q.g_raydrop) {  // composited part of the raydrop output: raydrop - T_end
      gp = __ldg(Q.g_raydrop + ray);
      gQ = fmaf(gp, __ldg(Q.b_raydrop + ray) - Tend, gQ);
    }
    nv = (int)s1.w;
    if (!r.valid) nv = 0;
    if (nv == 0) w.alive = false;
  }
  float gam[4];
  sh_basis(r.d, gam);
  const bool want_int = !LEAN && Q.want_int != 0;
  const bool want_drop = !LEAN && Q.g_raydrop != nullptr;
  const float gbg = g[0] * Q.bg[0] + g[1] * Q.bg[1] + g[2] * Q.bg[2] + gp;
  float T = 1.f, Pk = 0.f;
  int k = 0;
  // per-warp ring of pending hits (4 chunks each, padded to 5): each round's
  // hits are queued, and the gradient rows and their atomics run 32 at a time
  // on the whole warp.  A hit: (voxel, x), (geometry, SDF a and b, intensity),
  // (colour factors, raydrop), SH basis.
  // The gradient rows of voxels that many hits share are summed here too.
  constexpr int QN = 64, QW = 5;
  __shared__ float4 s_queue[SALF_BWD_WARPS][QN * QW];
  float4* queue = s_queue[threadIdx.x >> 5];
  int head = 0, tail = 0;  // warp-uniform
  const int nq = (want_int || want_drop) ? 8 : 7;

  // gradient rows of n queued hits (n <= 32), summed per voxel, added to d_params
  auto flush = [&](int n) {
    const bool act = lane < n;
    // (a lane without a hit reads its slot of the ring all the same, and is a group of
    // its own)
    float4* slot = queue + ((head + lane) & (QN - 1)) * QW;
    const float4 i0 = slot[0], i1 = slot[1], i2 = slot[2], i3 = slot[3];
    const int key = act ? __float_as_int(i0.x) : -1 - lane;
    const float x0 = i0.y, x1 = i0.z, x2 = i0.w;
    const float di = want_int ? i1.w : 0.f, dr = want_drop ? i2.w : 0.f;
    // chunk q of the hit's gradient row (gamma_0 is a constant)
    auto chunk = [&](int q) {
      switch (q) {
        case 0: return make_float4(i1.x * x0, i1.x * x1, i1.x * x2, i1.x);
        case 1: return make_float4(i2.x * x0, i2.x * x1, i2.x * x2, i2.y * x0);
        case 2: return make_float4(i2.y * x1, i2.y * x2, i2.z * x0, i2.z * x1);
        case 3: return make_float4(i2.z * x2, i2.x * kSH0, i2.x * i3.x, i2.x * i3.y);
        case 4: return make_float4(i2.x * i3.z, i2.y * kSH0, i2.y * i3.x, i2.y * i3.y);
        case 5: return make_float4(i2.y * i3.z, i2.z * kSH0, i2.z * i3.x, i2.z * i3.y);
        case 6:
          return make_float4(i2.z * i3.z, MODE == SALF_FIELD_EXP ? 0.f : i1.y,
                             MODE == SALF_FIELD_EXP ? 0.f : i1.z, di * x0);
        default: return make_float4(di * x1, di * x2, di, dr);
      }
    };
    float4* dst = reinterpret_cast<float4*>(Q.d_params) + (size_t)key * 8;
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    const int gn = __popc(peers);
    const bool staged = gn >= 4;
    if (act && !staged) {  // few rows of this voxel: their atomics cost less than staging
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q < nq) atomicAdd(dst + q, chunk(q));
    }
    if (__any_sync(0xffffffffu, staged)) {
      // A group's rows in parts by lane, as the bits of `every` pick them: 1 (4-7 rows), 2
      // (8-15) or 4; four lanes to a part, each summing one of its chunks.
      const int rank = __popc(peers & ((1u << lane) - 1u));
      const int parts = gn >= 16 ? 4 : gn >= 8 ? 2 : 1, part = rank >> 2, c = rank & 3;
      const unsigned every = parts == 4 ? 0x11111111u : parts == 2 ? 0x55555555u : 0xffffffffu;
      const unsigned mine = staged && part < parts ? peers & (every << part) : 0u;
      // the lanes 4 and 8 ranks up hold the sums of the next part and of the one after
      unsigned up = peers & ~((2u << lane) - 1u);
#pragma unroll
      for (int k = 0; k < 3; ++k) up &= up - 1u;
      const int up4 = (__ffs(up) - 1) & 31;
#pragma unroll
      for (int k = 0; k < 4; ++k) up &= up - 1u;
      const int up8 = (__ffs(up) - 1) & 31;
      const bool any2 = __any_sync(0xffffffffu, parts >= 2), any4 = __any_sync(0xffffffffu, parts == 4);
      // staged in the rows' own slots of the ring (each lane has read its hit), four
      // chunks at a time
#pragma unroll
      for (int q0 = 0; q0 < 8; q0 += 4) {
        if (staged) {
#pragma unroll
          for (int q = 0; q < 4; ++q) slot[q] = chunk(q0 + q);
        }
        __syncwarp();
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        for (unsigned m = mine; m; m &= m - 1u) {
          const float4 r2 = queue[((head + __ffs(m) - 1) & (QN - 1)) * QW + c];
          sum.x += r2.x;
          sum.y += r2.y;
          sum.z += r2.z;
          sum.w += r2.w;
        }
        auto fold = [&](int from, bool take) {
          const float x = __shfl_sync(0xffffffffu, sum.x, from),
                      y = __shfl_sync(0xffffffffu, sum.y, from),
                      z = __shfl_sync(0xffffffffu, sum.z, from),
                      t = __shfl_sync(0xffffffffu, sum.w, from);
          sum.x += take ? x : 0.f;
          sum.y += take ? y : 0.f;
          sum.z += take ? z : 0.f;
          sum.w += take ? t : 0.f;
        };
        if (any4) fold(up8, parts == 4);  // parts 0 and 1 take 2 and 3
        if (any2) fold(up4, parts >= 2);  // part 0 takes 1
        if (staged && part == 0 && q0 + c < nq) atomicAdd(dst + q0 + c, sum);
        __syncwarp();
      }
    }
    head += n;
    __syncwarp();
  };

  for (;;) {
    Hit h;
    const bool hit = next_hit<DT, AHEAD>(S, w, h);
    if (!__any_sync(0xffffffffu, hit || w.alive)) break;
    const unsigned hit_lanes = __ballot_sync(0xffffffffu, hit);
    if (hit) {
      const float tm = 0.5f * (h.tin + h.tout);
      const float dl = h.tout - h.tin;
      float x[3];
      local_coords(w, h, tm, x);
      Field f;
      field_eval<DT, MODE>(S, h.vox, want_int, x, gam, f, want_drop);
      const float sig = f.sig, lin = f.lin, io = f.io;
      const float* c = f.c;
      const float e = __expf(-sig * dl);
      const float wgt = T * (1.f - e);
      // the intensity and raydrop terms only when asked for (a product with a zero
      // factor is not dropped by the compiler)
      float gq = g[0] * c[0] + g[1] * c[1] + g[2] * c[2] + g[3] * tm + g[4];
      if (want_int) gq += g[5] * io;
      if (want_drop) gq += gp * f.dr;
      Pk = fmaf(wgt, gq, Pk);
      const float Tn = T * e;
      const float dtau = Tn * gq - (gQ - Pk) - Tend * gbg;
      const float dsig = dtau * dl;
      // the hit's coefficients: the gradient row is built from them later
      float4* it = queue + ((tail + __popc(hit_lanes & ((1u << lane) - 1u))) & (QN - 1)) * QW;
      float4 geo = make_float4(dsig * sig, 0.f, 0.f, 0.f);
      if (MODE == SALF_FIELD_SDF) {
        const float a = f.a, b = f.b;
        const float ex = __expf(-fabsf(lin) / b);
        geo.x = dsig * (a / (2.f * b)) * ex;
        geo.y = dsig * sig / a;
        geo.z = -dsig * a * lin * ex / (2.f * b * b);
      }
      if (want_int) geo.w = wgt * g[5] * io * (1.f - io);
      it[0] = make_float4(__int_as_float(__ldg(&S.order[h.vox])), x[0], x[1], x[2]);
      it[1] = geo;
      it[2] = make_float4(wgt * g[0] * c[0] * (1.f - c[0]), wgt * g[1] * c[1] * (1.f - c[1]),
                          wgt * g[2] * c[2] * (1.f - c[2]),
                          want_drop ? wgt * gp * f.dr * (1.f - f.dr) : 0.f);
      it[3] = make_float4(gam[1], gam[2], gam[3], 0.f);
      T = Tn;
      if (++k >= nv) w.alive = false;
    }
    tail += __popc(hit_lanes);
    __syncwarp();
    if (tail - head >= 32) flush(32);
  }
  while (tail - head > 0) flush(min(32, tail - head));
}

template <int DT, int MODE>
static cudaError_t launch_bm(const LaunchParams& P, cudaStream_t st) {
  const int blocks = (P.total_tiles + SALF_BWD_WARPS - 1) / SALF_BWD_WARPS;
  if (blocks == 0) return cudaSuccess;
  bool lean = true;
  for (int i = 0; i < P.n_req; ++i) {
    const ReqDev& q = P.req[i];
    lean = lean && q.kind == SALF_PINHOLE && !q.moving && !q.want_int && !q.g_raydrop;
  }
  if (lean)
    k_backward<DT, MODE, true><<<blocks, 32 * SALF_BWD_WARPS, 0, st>>>(P);
  else
    k_backward<DT, MODE, false><<<blocks, 32 * SALF_BWD_WARPS, 0, st>>>(P);
  return cudaGetLastError();
}

cudaError_t salf_launch_backward(const LaunchParams& P, cudaStream_t st) {
  const int dt = P.S.dtype, md = P.S.mode;
  if (dt == SALF_F32 && md == SALF_FIELD_EXP) return launch_bm<SALF_F32, SALF_FIELD_EXP>(P, st);
  if (dt == SALF_F32 && md == SALF_FIELD_SDF) return launch_bm<SALF_F32, SALF_FIELD_SDF>(P, st);
  if (dt == SALF_BF16 && md == SALF_FIELD_EXP) return launch_bm<SALF_BF16, SALF_FIELD_EXP>(P, st);
  return launch_bm<SALF_BF16, SALF_FIELD_SDF>(P, st);
}
