// The exact update of one narrow problem (d <= NC_MAX_D) as ONE kernel on one cluster of thread blocks.
//
// At these widths a launch of the iteration costs more than its work: 128^3 multiply-adds are 0.1 us of the chip, a launch with
// the load latency of its operands about 6 us, and a step takes three of them and the control decision.  Sixteen CTAs of one
// cluster share the 32 x 32 tiles of every product instead, a cluster barrier stands between the products, and every CTA takes the
// decision itself from the same sums.  An element of a product is the same chain of multiply-adds as in the launches' kernels, and
// the coefficients of a step depend on its place in the plan alone: the same bits wherever the start scale rounds to the same number
// and the decisions agree.  (The squares behind these are added in another grouping, sixteen CTAs' instead of a block's per 1024
// elements or per tile: double sums rounded to fp32, so a last bit may differ.)
// What a step takes (d = 128, SM cycles, clock stamps): products 3 x 4.1 k (a warp's multiply-adds: two cycles each, 16 per k),
// operands from the L2 6 k, barriers 6 k (the stores in front of them have to reach the L2), stores 2.7 k, norms and decision 1.8 k;
// an update of eight steps 116 us.  Whole update of the statistics of 16 d rows once its step count is learnt, from an idle stream,
// graph of launches -> this, us (one B200): d = 16, 8 steps 139 -> 57;  64, 9 steps 194 -> 106;  128, 9 steps 223 -> 136;  160, 12
// steps 258 -> 200;  192 (three tiles a CTA) would take 291 in a row of updates where the launches take 237.
#pragma once
#include <mutex>

#include "../../include/conqur.h"
#include "conqur_simt.cuh"

namespace conqur {

constexpr int NC_MAX_D = 160;                    // one or two tiles a CTA; the operand slabs (d x 32) stay in shared memory
constexpr int NC_THREADS = 256;
constexpr int NC_CTAS = 16;
constexpr int NC_WORK = 64;                       // threads that multiply: a 4 x 4 piece of the tile each
constexpr int NC_LD = 36;                        // slab rows: 32 columns and 4 floats against bank conflicts

struct NcArgs {
  float *M, *R, *Xa, *Xb, *E, *B;
  DevState* st;
  NsControlParams c;
  int d, n_endgame;
  float prior_rel, inv_sqrt_d, margin;
};

inline int nc_smem_bytes(int d) { return (d + 3) / 4 * 4 * 2 * NC_LD * (int)sizeof(float); }

__device__ __forceinline__ void nc_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Four elements P[r][c .. c+3] of a d x d matrix, zeros outside.  Other CTAs of the cluster write these: read from the L2.
__device__ __forceinline__ float4 nc_ld4(const float* P, int d, int r, int c, bool vec) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (r >= d || c >= d) return v;
  const float* p = P + (size_t)r * d + c;
  if (vec) return __ldcg(reinterpret_cast<const float4*>(p));        // d % 4 == 0: whole pieces
  v.x = __ldcg(p);
  if (c + 1 < d) v.y = __ldcg(p + 1);
  if (c + 2 < d) v.z = __ldcg(p + 2);
  if (c + 3 < d) v.w = __ldcg(p + 3);
  return v;
}

// Tile (m0, n0) of sum_k A(m, k) B(k, n), each sum one chain in the order of k as sg_mainloop's: thread t < NC_WORK returns rows
// 4 (t / 8) .. +3 and columns 4 (t % 8) .. +3, and the slabs stay in shared memory (row k: A(m0 .. +31, k), then B(k, n0 .. +31)).
// A(m, k) = A[k][m], or A[m][k] with TRANS.  A 16-byte read takes the shared memory four cycles a warp whatever is equal in it,
// so two warps with 4 x 4 pieces (16 cycles per k, 16 multiply-adds each) are faster than four with 2 x 4 (32).
template <bool TRANS>
__device__ __forceinline__ void nc_tile(const float* A, const float* B, int d, int m0, int n0, bool vec, float* smem, float (&out)[4][4]) {
  const int t = threadIdx.x, kp = (d + 3) / 4 * 4;
  float* sa = smem;
  float* sb = sa + kp * NC_LD;
  for (int e0 = 0; e0 < kp * 8; e0 += 4 * NC_THREADS) {            // four pieces of either slab in flight per thread
    float4 va[4], vb[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = e0 + i * NC_THREADS + t;
      va[i] = vb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e < kp * 8) {
        vb[i] = nc_ld4(B, d, e >> 3, n0 + (e & 7) * 4, vec);
        va[i] = TRANS ? nc_ld4(A, d, m0 + (e & 31), (e >> 5) * 4, vec) : nc_ld4(A, d, e >> 3, m0 + (e & 7) * 4, vec);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = e0 + i * NC_THREADS + t;
      if (e >= kp * 8) continue;
      *reinterpret_cast<float4*>(sb + (e >> 3) * NC_LD + (e & 7) * 4) = vb[i];
      if (TRANS) {
        float* q = sa + (e >> 5) * 4 * NC_LD + (e & 31);
        q[0] = va[i].x; q[NC_LD] = va[i].y; q[2 * NC_LD] = va[i].z; q[3 * NC_LD] = va[i].w;
      } else {
        *reinterpret_cast<float4*>(sa + (e >> 3) * NC_LD + (e & 7) * 4) = va[i];
      }
    }
  }
  __syncthreads();
  if (t < NC_WORK) {
    const float* pa = sa + 4 * (t >> 3);
    const float* pb = sb + 4 * (t & 7);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) out[i][j] = 0.f;
#pragma unroll 8
    for (int k = 0; k < kp; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(pa + k * NC_LD), b = *reinterpret_cast<const float4*>(pb + k * NC_LD);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) out[i][j] = fmaf(av[i], bv[j], out[i][j]);
    }
  }
}

__device__ __forceinline__ void nc_st4(float* P, int d, int r, int c, const float (&v)[4], bool vec, bool mirror) {
  if (r >= d || c >= d) return;
  float* p = P + (size_t)r * d + c;
  if (vec) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (c + j < d) p[j] = v[j];
  }
  if (mirror) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (c + j < d) P[(size_t)(c + j) * d + r] = v[j];
  }
}

// Leaves a value in every CTA of the cluster (slot `from` of `slots`, the same place in each one's shared memory); one warp.
// The cluster barrier that follows publishes it.
__device__ __forceinline__ void nc_tell(double v, double* slots, int from) {
  const int lane = threadIdx.x & 31;
  if (lane < NC_CTAS) {
    uint32_t a, r;
    asm("{ .reg .u64 t; cvta.to.shared.u64 t, %1; cvt.u32.u64 %0, t; }" : "=r"(a) : "l"(slots + from));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(lane));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(r), "d"(v) : "memory");
  }
}
// The sixteen values, added in order (every CTA gets the same sum).
__device__ __forceinline__ double nc_total(const double* slots) {
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < NC_CTAS; ++i) s += slots[i];
  return s;
}

__global__ void __launch_bounds__(NC_THREADS, 1) ns_cluster_kernel(const NcArgs g) {
  extern __shared__ __align__(16) float nc_smem[];
  __shared__ double redd[NC_THREADS / 32];
  __shared__ float redf[NC_THREADS / 32];
  __shared__ double sums[2][NC_CTAS], maxima[2][NC_CTAS];     // what the CTAs tell each other, alternating
  __shared__ float coef[4];
  __shared__ int done_s;
  __shared__ SchedEntry sched[NS_SCHED_MAX];
  const int cta = (int)blockIdx.x, t = threadIdx.x, d = g.d, tiles = (d + 31) / 32;
  const size_t dd = (size_t)d * d;
  const bool vec = (d & 3) == 0;
  DevState* st = g.st;
  for (int i = t; i < g.c.n_sched && i < NS_SCHED_MAX; i += NC_THREADS) sched[i] = g.c.sched[i];
  NsControlParams c = g.c;
  c.sched = sched;
  int slot = 0;
  auto sumsq = [&](float lam) {                  // ||M + lam R||_F^2
    double v = 0.0;
#pragma unroll 4
    for (size_t i = (size_t)cta * NC_THREADS + t; i < dd; i += (size_t)NC_CTAS * NC_THREADS) {
      float m = g.M[i];
      if (lam != 0.f) m = fmaf(lam, g.R[i], m);
      v += (double)m * (double)m;
    }
    const double part = block_sum_d<NC_THREADS>(v, redd);
    if (t < 32) nc_tell(__shfl_sync(0xffffffffu, part, 0), sums[slot], cta);
    nc_cluster_sync();
    const double tot = nc_total(sums[slot]);
    slot ^= 1;
    return tot;
  };
  nc_cluster_sync();                             // every CTA runs before anything is written into its shared memory

  // scale of the first iterate (see ns_setup_kernel)
  double tot = sumsq(0.f);
  float lam = 0.f;
  if (g.prior_rel > 0.f) {
    lam = g.prior_rel * (float)sqrt(tot) * g.inv_sqrt_d;
    tot = sumsq(lam);
  }
  const float fro = (float)sqrt(tot);
  const bool ok = fro > 0.f && fro <= 3.0e38f && __ldcg(&st->N) > 0;
  const float x0_scale = ok ? 1.0f / (fro * (1.0f + g.margin)) : 0.f;
  if (cta == 0 && t == 0) {
    st->lam = lam; st->scale = fro; st->x0_scale = x0_scale;
    ns_arm_lifting(st, c.n_lift_init);
    st->ns_done = ok ? 0 : NS_DONE_FAILED;
    st->ns_steps_used = 0; st->ns_final_buf = 0; st->seg_x = 2; st->seg_e = 3; st->tau = 1.0f;
  }
#pragma unroll 4
  for (size_t i = (size_t)cta * NC_THREADS + t; i < dd; i += (size_t)NC_CTAS * NC_THREADS) g.Xa[i] = fmaf(lam, g.R[i], g.M[i]) * x0_scale;
  nc_cluster_sync();
  NsCtl ctl;                                     // thread 0 of every CTA takes the same decisions
  if (t == 0) {
    ns_ctl_load(ctl, st);
    done_s = ctl.ns_done;
  }
  __syncthreads();
  const int sym_tiles = tiles * (tiles + 1) / 2;
  auto sym_coords = [&](int i, int& tm, int& tn) { tn = 0; while ((tn + 1) * (tn + 2) / 2 <= i) ++tn; tm = i - tn * (tn + 1) / 2; };
  const int r = 4 * (t >> 3), c4 = (t & 7) * 4;  // this thread's piece of a tile (t < NC_WORK)
  const float* const slab_a = nc_smem;
  const float* const slab_b = nc_smem + (d + 3) / 4 * 4 * NC_LD;
  float v[4][4];
  int k = 0, cur = 0;
  for (; done_s == 0; ++k, cur ^= 1) {
    const float* X = cur ? g.Xb : g.Xa;
    float* Xn = cur ? g.Xa : g.Xb;
    // E = X^T X - I and its norms
    float mx = 0.f;
    double sq = 0.0;
    for (int i = cta; i < sym_tiles; i += NC_CTAS) {
      int tm, tn;
      sym_coords(i, tm, tn);
      nc_tile<false>(X, X, d, tm * 32, tn * 32, vec, nc_smem, v);
      if (t < NC_WORK) {
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int row = tm * 32 + r + h, col = tn * 32 + c4;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (row >= d || col + j >= d) continue;
            if (row == col + j) v[h][j] -= 1.f;
            mx = fmaxf(mx, fabsf(v[h][j]));
            sq += (tm != tn ? 2.0 : 1.0) * ((double)v[h][j] * (double)v[h][j]);
          }
          nc_st4(g.E, d, row, col, v[h], vec, tm != tn);
        }
      }
      __syncthreads();                           // the slabs are free
    }
    if (t < NC_WORK) {
      sq = warp_sum_d(sq);
      mx = warp_max(mx);
      if (t == 32) { redd[0] = sq; redf[0] = mx; }
    }
    __syncthreads();
    if (t < 32) {
      nc_tell(sq + redd[0], sums[slot], cta);
      nc_tell((double)fmaxf(mx, redf[0]), maxima[slot], cta);
    }
    nc_cluster_sync();
    if (t == 0) {
      const double tsq = nc_total(sums[slot]);
      double tmx = 0.0;
#pragma unroll
      for (int i = 0; i < NC_CTAS; ++i) tmx = fmax(tmx, maxima[slot][i]);
      const unsigned char entry = ns_control_decide(&ctl, (float)tmx, tsq, 0.0, k, cur, c);
      if (cta == 0 && entry && k < 128) st->seg_log[k] = entry;
#pragma unroll
      for (int j = 0; j < 4; ++j) coef[j] = ctl.coef[j];
      done_s = ctl.ns_done;
    }
    slot ^= 1;
    __syncthreads();
    if (done_s != 0) break;
    // B = beta2 E E + beta1 E
    for (int i = cta; i < sym_tiles; i += NC_CTAS) {
      int tm, tn;
      sym_coords(i, tm, tn);
      nc_tile<false>(g.E, g.E, d, tm * 32, tn * 32, vec, nc_smem, v);
      if (t < NC_WORK) {
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int row = tm * 32 + r + h, col = tn * 32 + c4;
          if (row >= d) continue;
#pragma unroll
          for (int j = 0; j < 4; ++j) v[h][j] = fmaf(coef[2], v[h][j], coef[1] * slab_b[row * NC_LD + c4 + j]);     // E(row, col + j)
          nc_st4(g.B, d, row, col, v[h], vec, tm != tn);
        }
      }
      __syncthreads();
    }
    nc_cluster_sync();
    // X_next = X B + gamma X
    for (int i = cta; i < tiles * tiles; i += NC_CTAS) {
      const int tm = i / tiles, tn = i - tm * tiles;
      nc_tile<true>(X, g.B, d, tm * 32, tn * 32, vec, nc_smem, v);
      if (t < NC_WORK) {
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int row = tm * 32 + r + h, col = tn * 32 + c4;
          if (row >= d) continue;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (col + j < d) v[h][j] = fmaf(coef[0], slab_a[(col + j) * NC_LD + r + h], v[h][j]);                   // X(row, col + j)
          nc_st4(Xn, d, row, col, v[h], vec, false);
        }
      }
      __syncthreads();
    }
    nc_cluster_sync();
  }
  // accept or reject (see ns_commit_kernel, ns_commit_state_kernel)
  if (done_s == NS_DONE_CONVERGED) {
    const float* X = cur ? g.Xb : g.Xa;
#pragma unroll 4
    for (size_t i = (size_t)cta * NC_THREADS + t; i < dd; i += (size_t)NC_CTAS * NC_THREADS) {
      g.R[i] = __ldcg(X + i);
      g.M[i] = 0.f;
    }
  }
  if (cta == 0 && t == 0) {
    ns_ctl_store(ctl, st);
    ns_commit_state(st, g.n_endgame);
  }
  nc_cluster_sync();                             // no CTA leaves while another may still write into its shared memory
}

// Whether a cluster of NC_CTAS can be resident on the device (asked once per device, under a lock).
inline bool nc_available(int dev) {
  static std::mutex mu;
  static int known[64] = {};                     // 0: not asked, 1: yes, 2: no
  if (dev < 0 || dev >= 64) return false;
  std::lock_guard<std::mutex> lock(mu);
  if (known[dev] == 0) {
    int n = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(NC_CTAS); cfg.blockDim = dim3(NC_THREADS); cfg.dynamicSmemBytes = (size_t)nc_smem_bytes(NC_MAX_D);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = NC_CTAS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    const bool yes = cudaFuncSetAttribute(ns_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, nc_smem_bytes(NC_MAX_D)) == cudaSuccess &&
                     cudaFuncSetAttribute(ns_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                     cudaOccupancyMaxActiveClusters(&n, ns_cluster_kernel, &cfg) == cudaSuccess && n > 0;
    if (!yes) cudaGetLastError();
    known[dev] = yes ? 1 : 2;
  }
  return known[dev] == 1;
}
inline int nc_launch(const NcArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(NC_CTAS); cfg.blockDim = dim3(NC_THREADS); cfg.dynamicSmemBytes = (size_t)nc_smem_bytes(a.d); cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = NC_CTAS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ns_cluster_kernel, a) == cudaSuccess ? CONQUR_OK : CONQUR_ERR_CUDA;
}

}  // namespace conqur
