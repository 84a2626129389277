// The exact update of one narrow problem (d <= NC_MAX_D) as ONE kernel on one cluster of thread blocks.
//
// At these widths a launch of the iteration costs more than its work: 128^3 multiply-adds are 0.1 us of the chip, a launch with
// the load latency of its operands about 6 us, and a step takes three of them and the control decision.  Sixteen CTAs of one
// cluster share the 32 x 32 tiles of every product instead, and every CTA takes the decision itself from the same sums.  The matrices
// live in shared memory: a finished tile is written straight into that of the CTAs whose next products read it.  Up to d = 128 a CTA
// waits for the bytes it reads and nothing else (beyond, where there is no room to keep what others still read, for barriers of
// the cluster).  An element of a product is the same chain of multiply-adds as in the launches' kernels, and the coefficients of a
// step depend on its place in the plan alone: the same bits wherever the start scale rounds to the same number and the decisions
// agree.  (The squares behind these are added in another grouping, sixteen CTAs' instead of a block's per 1024 elements or per tile:
// double sums rounded to fp32, so a last bit may differ.)
// What a step takes (d = 128, SM cycles, clock stamps): products 3.3 k each, bound by their reads of shared memory, sending 1.3 k (32 KB a
// CTA at 25 bytes a cycle), the way there 0.6 k, norms 0.4 k; the decision runs beside the next product.  Whole update of given statistics
// once its step count is learnt, from an idle stream, us (one B200): matrices in the L2 between the products -> in shared memory with two
// multiplying warps and cluster barriers -> waiting for bytes -> this, with four warps
//   d = 16, 4 steps 36 -> 26 -> 23 -> 24;  64, 4 steps 49 -> 36 -> 35 -> 34;  128, 4 steps 70 -> 61 -> 59 -> 55;  160, 5 steps 121 -> 110 -> - -> 103
// (as a graph of launches the first took 139, with 8 steps, and 128 with 9 steps 223).  192 has no room for its matrices.
#pragma once
#include <mutex>

#include "../../include/conqur.h"
#include "conqur_simt.cuh"

namespace conqur {

constexpr int NC_MAX_TILES = 5;                  // tiles of 32 along a side: one or two of a product's 25 a CTA
constexpr int NC_MAX_D = 32 * NC_MAX_TILES;
constexpr int NC_SMALL_D = 128;                  // up to here three matrices fit
constexpr int NC_THREADS = 256;
constexpr int NC_CTAS = 16;
constexpr int NC_WORK = 128;                     // threads that multiply: a 2 x 4 piece of the tile each
constexpr int NC_LD_TILE = 36;                   // rows of the tile on its way out: 32 columns and 4 floats against bank conflicts

struct NcArgs {
  float *M, *R;
  DevState* st;
  NsControlParams c;
  int d, n_endgame;
  float prior_rel, inv_sqrt_d, margin;
  long long wait_limit;                          // SM cycles a wait for bytes lasts at most
  int lose;                                      // test hook: CTA `lose % 16` waits in step `lose / 16` for bytes that nobody sends (-1: none)
};

// A matrix in shared memory: 32 T rows of 32 T columns and 4 floats against bank conflicts, zeros past d.  Up to four tiles a side three
// of them fit, and a tile never goes where another CTA still reads.  With five there are two, written in place, and a barrier of the
// cluster stands in front of and behind each write.
__host__ __device__ inline int nc_ld(int tiles) { return 32 * tiles + 4; }
__host__ __device__ inline int nc_matrix_floats(int tiles) { return 32 * tiles * nc_ld(tiles); }
__host__ __device__ inline int nc_matrices(int tiles) { return 32 * tiles <= NC_SMALL_D ? 3 : 2; }
inline int nc_smem_bytes(int d) {
  const int tiles = (d + 31) / 32;
  return (nc_matrices(tiles) * nc_matrix_floats(tiles) + 32 * NC_LD_TILE) * (int)sizeof(float);
}

__device__ __forceinline__ void nc_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Tile (m0, n0) of sum_k A(m, k) B(k, n), each sum one chain in the order of k as sg_mainloop's; k runs to kp, d rounded up to four.
// A(m, k) = A[k][m]: thread t < NC_WORK returns rows 2 (t / 8) and the next; A[m][k] with TRANS: rows t / 8 and + 16 (neighbouring rows of
// A lie four banks apart).  Columns 4 (t % 8) .. +3 either way.  A warp's read of 8 or 16 bytes a lane takes the shared memory two or
// four cycles whatever is equal in it, a packed multiply-add the lanes two: four warps with 2 x 4 pieces need 24 and 8 cycles per k (two
// with 4 x 4 16 of either, and took 26 to 32, with nobody to hide a warp's waits behind).
template <bool TRANS>
__device__ __forceinline__ void nc_tile(const float* A, const float* B, int ld, int kp, int m0, int n0, float (&out)[2][4]) {
  const int ty = (int)threadIdx.x >> 3, tx = (int)threadIdx.x & 7;
  const float* pb = B + n0 + 4 * tx;
  const float* pa = TRANS ? A + (m0 + ty) * ld : A + m0 + 2 * ty;
  unsigned long long acc[2][2] = {};
  // (four k ahead in registers.  The last reads go past the matrix, into its row padding or what lies behind it, and go unused.)
  struct Four { float a[2][4]; float4 b[4]; };   // a[row][k]
  auto fetch = [&](int k, Four& f) {
    if (TRANS) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(pa + 16 * i * ld + k);
        f.a[i][0] = v.x; f.a[i][1] = v.y; f.a[i][2] = v.z; f.a[i][3] = v.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 v = *reinterpret_cast<const float2*>(pa + (k + j) * ld);
        f.a[0][j] = v.x; f.a[1][j] = v.y;
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) f.b[j] = *reinterpret_cast<const float4*>(pb + (k + j) * ld);
  };
  auto multiply = [&](const Four& f) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const unsigned long long b0 = f32x2_pack(f.b[j].x, f.b[j].y), b1 = f32x2_pack(f.b[j].z, f.b[j].w);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const unsigned long long a2 = f32x2_pack(f.a[i][j], f.a[i][j]);
        f32x2_fma(acc[i][0], a2, b0);
        f32x2_fma(acc[i][1], a2, b1);
      }
    }
  };
  Four f0, f1;
  fetch(0, f0);
  int k = 0;
  for (; k + 8 <= kp; k += 8) {
    fetch(k + 4, f1);
    multiply(f0);
    fetch(k + 8, f0);
    multiply(f1);
  }
  if (k < kp) multiply(f0);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      out[i][2 * j] = __uint_as_float((uint32_t)acc[i][j]);
      out[i][2 * j + 1] = __uint_as_float((uint32_t)(acc[i][j] >> 32));
    }
}

// This thread's piece of a tile into the tile's buffer (row r0 + step i).
__device__ __forceinline__ void nc_put(float* tile, int r0, int step, const float (&v)[2][4]) {
#pragma unroll
  for (int i = 0; i < 2; ++i)
    *reinterpret_cast<float4*>(tile + (r0 + step * i) * NC_LD_TILE + 4 * ((int)threadIdx.x & 7)) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
}

__device__ __forceinline__ uint32_t nc_smem_u32(const void* p) {
  uint32_t a;
  asm("{ .reg .u64 t; cvta.to.shared.u64 t, %1; cvt.u32.u64 %0, t; }" : "=r"(a) : "l"(p));
  return a;
}
// The tile (or its transpose) to place (r, c) of `matrix` in every CTA of the mask, 16 bytes at a time: piece p of 256.  The cluster
// barrier that follows publishes it.
__device__ __forceinline__ void nc_send(const float* tile, bool transposed, float* matrix, int ld, int r, int c, uint32_t mask, int p) {
  const int row = p >> 3, col = 4 * (p & 7);
  float4 v;
  if (transposed) {
    v.x = tile[col * NC_LD_TILE + row]; v.y = tile[(col + 1) * NC_LD_TILE + row];
    v.z = tile[(col + 2) * NC_LD_TILE + row]; v.w = tile[(col + 3) * NC_LD_TILE + row];
  } else {
    v = *reinterpret_cast<const float4*>(tile + row * NC_LD_TILE + col);
  }
  const uint32_t here = nc_smem_u32(matrix + (32 * r + row) * ld + 32 * c + col);
  for (; mask; mask &= mask - 1) {
    uint32_t there;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(here), "r"(__ffs((int)mask) - 1));
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(there), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
  }
}

// The same for up to four tiles a side, where nothing but the data itself is waited for: the bytes are counted on a barrier in each CTA that
// gets them.  No copy or barrier of the whole cluster stands between two products then.
__device__ __forceinline__ void nc_send_async(const float* tile, bool transposed, float* matrix, int ld, int r, int c, uint32_t mask, int p,
                                              uint64_t* bar) {
  const int row = p >> 3, col = 4 * (p & 7);
  float4 v;
  if (transposed) {
    v.x = tile[col * NC_LD_TILE + row]; v.y = tile[(col + 1) * NC_LD_TILE + row];
    v.z = tile[(col + 2) * NC_LD_TILE + row]; v.w = tile[(col + 3) * NC_LD_TILE + row];
  } else {
    v = *reinterpret_cast<const float4*>(tile + row * NC_LD_TILE + col);
  }
  const uint32_t here = nc_smem_u32(matrix + (32 * r + row) * ld + 32 * c + col), bar_here = nc_smem_u32(bar);
  for (; mask; mask &= mask - 1) {
    const int to = __ffs((int)mask) - 1;
    uint32_t there, bar_there;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(here), "r"(to));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar_there) : "r"(bar_here), "r"(to));
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(there), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar_there) : "memory");
  }
}
__device__ __forceinline__ void nc_bar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(nc_smem_u32(bar)) : "memory");
}
// The barrier's next phase: `bytes` will come (one thread, and only once the one before is over).
__device__ __forceinline__ void nc_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(nc_smem_u32(bar)), "r"(bytes) : "memory");
}
// Waits for a phase's bytes, for `limit` cycles at most; gave_up ends every wait of the CTA.  Whether they came.
__device__ __forceinline__ bool nc_wait(uint64_t* bar, uint32_t parity, volatile int* gave_up, long long limit) {
  const uint32_t at = nc_smem_u32(bar);
  const long long t0 = clock64();
  for (uint32_t spins = 0;; ++spins) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(at), "r"(parity) : "memory");
    if (ok) return true;
    if ((spins & 255u) == 255u && (*gave_up || clock64() - t0 > limit)) { *gave_up = 1; return false; }
  }
}

// The multiplying warps' sums and maxima.
__device__ __forceinline__ double nc_all_of(const double* s) { return (s[0] + s[1]) + (s[2] + s[3]); }
__device__ __forceinline__ float nc_most_of(const float* m) { return fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])); }

// Leaves a value in every CTA of the cluster (slot `from` of `slots`, the same place in each one's shared memory); one warp.
// The cluster barrier that follows publishes it.
__device__ __forceinline__ void nc_tell(double v, double* slots, int from) {
  const int lane = threadIdx.x & 31;
  if (lane < NC_CTAS) {
    uint32_t r;
    const uint32_t a = nc_smem_u32(slots + from);
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(lane));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(r), "d"(v) : "memory");
  }
}
// Two values, counted on a barrier there.
__device__ __forceinline__ void nc_tell_async(double a, double b, double (*slots)[2], int from, uint64_t* bar) {
  const int lane = threadIdx.x & 31;
  if (lane < NC_CTAS) {
    uint32_t there, bar_there;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(nc_smem_u32(slots + from)), "r"(lane));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar_there) : "r"(nc_smem_u32(bar)), "r"(lane));
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];"
                 ::"r"(there), "d"(a), "d"(b), "r"(bar_there) : "memory");
  }
}
// The sixteen values, added in order (every CTA gets the same sum).
__device__ __forceinline__ double nc_total(const double* slots) {
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < NC_CTAS; ++i) s += slots[i];
  return s;
}

template <bool SMALL>
__global__ void __launch_bounds__(NC_THREADS, 1) ns_cluster_kernel(const NcArgs g) {
  extern __shared__ __align__(16) float nc_smem[];
  __shared__ double redd[NC_THREADS / 32];
  __shared__ float redf[NC_THREADS / 32];
  __shared__ double sums[2][NC_CTAS], maxima[2][NC_CTAS];     // what the CTAs tell each other, alternating
  __shared__ float coef[4];
  __shared__ int done_s;
  __shared__ uint32_t by_col[NC_MAX_TILES], by_row[NC_MAX_TILES], by_factor[NC_MAX_TILES];    // who reads what, see below
  __shared__ SchedEntry sched[NS_SCHED_MAX];
  __shared__ __align__(16) double told[2][NC_CTAS][2];        // SMALL: what the CTAs tell each other, alternating
  __shared__ __align__(8) uint64_t bar_e, bar_b, bar_x, bar_t[2];
  __shared__ int gave_up, lost;                               // this CTA gave a wait up, any CTA did
  const int cta = (int)blockIdx.x, t = threadIdx.x, d = g.d, kp = (d + 3) / 4 * 4;
  const int tiles = (d + 31) / 32, ld = nc_ld(tiles), sym_tiles = tiles * (tiles + 1) / 2;
  float* X = nc_smem;
  float* E = X + nc_matrix_floats(tiles);
  float* Bm = SMALL ? E + nc_matrix_floats(tiles) : E;
  float* const tile = nc_smem + nc_matrices(tiles) * nc_matrix_floats(tiles);
  const size_t dd = (size_t)d * d;
  DevState* st = g.st;
  auto sym_coords = [&](int i, int& tm, int& tn) { tn = 0; while ((tn + 1) * (tn + 2) / 2 <= i) ++tn; tm = i - tn * (tn + 1) / 2; };
  for (int i = t; i < g.c.n_sched && i < NS_SCHED_MAX; i += NC_THREADS) sched[i] = g.c.sched[i];
  NsControlParams c = g.c;
  c.sched = sched;
  for (int i = t; i < nc_matrices(tiles) * nc_matrix_floats(tiles) / 4; i += NC_THREADS)
    reinterpret_cast<float4*>(nc_smem)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (t < tiles) {
    // symmetric products read columns of X or of the residual; the last product rows of X and columns of the polynomial
    uint32_t col = 0, row = 0, factor = 0;
    for (int i = 0; i < sym_tiles; ++i) {
      int tm, tn;
      sym_coords(i, tm, tn);
      if (t == tm || t == tn) col |= 1u << (i % NC_CTAS);
    }
    for (int i = 0; i < tiles * tiles; ++i) {
      if (t == i / tiles) row |= 1u << (i % NC_CTAS);
      if (t == i % tiles) factor |= 1u << (i % NC_CTAS);
    }
    by_col[t] = col; by_row[t] = row; by_factor[t] = factor;
  }
  // this CTA's tiles, and the bytes of a step's residual, polynomial and iterate that come to it
  int tm = 0, tn = 0;
  const bool has_sym = cta < sym_tiles, has_full = cta < tiles * tiles;
  if (has_sym) sym_coords(cta, tm, tn);
  const uint32_t n_cols = has_sym ? (tm == tn ? 1u : 2u) : 0u;
  const uint32_t e_bytes = 4096u * tiles * n_cols, b_bytes = has_full ? 4096u * tiles : 0u;
  const uint32_t x_bytes = e_bytes + (has_full ? 4096u * (tiles - n_cols) : 0u);
  if (t == 0) lost = 0;
  if (SMALL && t == 0) {
    nc_bar_init(&bar_e); nc_bar_init(&bar_b); nc_bar_init(&bar_x); nc_bar_init(&bar_t[0]); nc_bar_init(&bar_t[1]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    nc_expect(&bar_e, e_bytes + (g.lose == cta ? 16u : 0u)); nc_expect(&bar_b, b_bytes); nc_expect(&bar_x, x_bytes);
    nc_expect(&bar_t[0], NC_CTAS * 16u); nc_expect(&bar_t[1], NC_CTAS * 16u);
    gave_up = 0;
  }
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
  // every CTA forms the whole first iterate: it reads most of it, and M and R are in the L2
  if ((d & 3) == 0) {
#pragma unroll 4
    for (int i = t; i < d * (d / 4); i += NC_THREADS) {
      const float4 m = reinterpret_cast<const float4*>(g.M)[i], q = reinterpret_cast<const float4*>(g.R)[i];
      const int r = i / (d / 4), c4 = i - r * (d / 4);
      *reinterpret_cast<float4*>(X + r * ld + 4 * c4) = make_float4(fmaf(lam, q.x, m.x) * x0_scale, fmaf(lam, q.y, m.y) * x0_scale,
                                                                    fmaf(lam, q.z, m.z) * x0_scale, fmaf(lam, q.w, m.w) * x0_scale);
    }
  } else {
#pragma unroll 4
    for (int i = t; i < d * d; i += NC_THREADS) {
      const int r = i / d;
      X[r * ld + i - r * d] = fmaf(lam, g.R[i], g.M[i]) * x0_scale;
    }
  }
  nc_cluster_sync();                             // (the state above is there for all, and nobody's matrices are still being cleared)
  NsCtl ctl;                                     // one thread of every CTA, not one that multiplies, takes the same decisions
  const bool decides = t == NC_WORK;
  if (decides) {
    ns_ctl_load(ctl, st);
    done_s = ctl.ns_done;
  }
  __syncthreads();
  const int r2 = 2 * (t >> 3), c4 = 4 * (t & 7); // this thread's piece of it (t < NC_WORK)
  float v[2][4];
  int k = 0, cur = 0;
  // E = X^T X - I, this thread's piece, and its norms
  auto residual = [&](float& mx, double& sq) {
    nc_tile<false>(X, X, ld, kp, tm * 32, tn * 32, v);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = tm * 32 + r2 + h, col = tn * 32 + c4;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (row >= d || col + j >= d) continue;
        if (row == col + j) v[h][j] -= 1.f;
        mx = fmaxf(mx, fabsf(v[h][j]));
        sq += (tm != tn ? 2.0 : 1.0) * ((double)v[h][j] * (double)v[h][j]);
      }
    }
  };
  auto polynomial = [&] {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j) v[h][j] = fmaf(coef[2], v[h][j], coef[1] * E[(tm * 32 + r2 + h) * ld + tn * 32 + c4 + j]);
  };
  auto next = [&](int f, float (&o)[2][4]) {     // X B + gamma X
    const int fm = f / tiles, fn = f - fm * tiles;
    nc_tile<true>(X, Bm, ld, kp, fm * 32, fn * 32, o);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j) o[h][j] = fmaf(coef[0], X[(fm * 32 + (t >> 3) + 16 * h) * ld + fn * 32 + c4 + j], o[h][j]);
  };
  auto decide = [&](double tsq, double tmx) {
    const unsigned char entry = ns_control_decide(&ctl, (float)tmx, tsq, 0.0, k, cur, c);
    if (cta == 0 && entry && k < 128) st->seg_log[k] = entry;
#pragma unroll
    for (int j = 0; j < 4; ++j) coef[j] = ctl.coef[j];
    done_s = ctl.ns_done;
  };
  // Up to sixteen tiles.  A phase begins when what it reads has come.  What may still be read is not written over: the residual goes where
  // the polynomial before it was, the polynomial where the iterate before that was, the next iterate where the residual was, and whoever
  // sends a tile to one of these places has waited, by way of its operands, for what the receiver made of the tile that stands there (a
  // receiver reads columns tm and tn of X and of the residual, column fn of the polynomial and row fm of X; the products behind a tile of
  // column c have read all of column c, and behind every tile of a step stand all CTAs' norms of that step).  Likewise no phase of a
  // barrier gets bytes of the one after the next, and the norms, which not every tile waits for, alternate between two.  Once a phase is over
  // the deciding thread, whose warp does not multiply, says what the next one expects, unless a wait was given up (by a multiplying thread behind
  // its wait: 56.1 -> 55.1 us at d = 128).
  if constexpr (SMALL) {
    const int fm = cta / tiles, fn = cta - fm * tiles;
    for (; done_s == 0; ++k, cur ^= 1) {
      float mx = 0.f;
      double sq = 0.0;
      if (t < NC_WORK) {
        if (k > 0 && x_bytes) nc_wait(&bar_x, (uint32_t)(k - 1) & 1u, &gave_up, g.wait_limit);
        if (has_sym) residual(mx, sq);
        sq = warp_sum_d(sq);
        mx = warp_max(mx);
        if ((t & 31) == 0) { redd[t >> 5] = sq; redf[t >> 5] = mx; }
      }
      __syncthreads();                           // (and the tile before has been sent)
      if (decides && k > 0 && x_bytes && !gave_up) nc_expect(&bar_x, x_bytes);
      if (has_sym && t < NC_WORK) nc_put(tile, r2, 1, v);
      if (t < 32) nc_tell_async(nc_all_of(redd), (double)nc_most_of(redf), told[k & 1], cta, &bar_t[k & 1]);
      __syncthreads();
      if (has_sym) {
        nc_send_async(tile, false, E, ld, tm, tn, by_col[tn], t, &bar_e);
        if (tm != tn) nc_send_async(tile, true, E, ld, tn, tm, by_col[tm], t, &bar_e);
        if (t < NC_WORK) {
          nc_wait(&bar_e, (uint32_t)k & 1u, &gave_up, g.wait_limit);
          nc_tile<false>(E, E, ld, kp, tm * 32, tn * 32, v);      // does not wait for the decision
        }
      }
      if (decides && nc_wait(&bar_t[k & 1], (uint32_t)(k >> 1) & 1u, &gave_up, g.wait_limit)) {
        nc_expect(&bar_t[k & 1], NC_CTAS * 16u);
        double tsq = 0.0, tmx = 0.0;
#pragma unroll
        for (int i = 0; i < NC_CTAS; ++i) { tsq += told[k & 1][i][0]; tmx = fmax(tmx, told[k & 1][i][1]); }
        decide(tsq, tmx);
      }
      __syncthreads();
      if (done_s != 0 || gave_up) break;
      if (decides && has_sym) nc_expect(&bar_e, e_bytes + (g.lose == cta + NC_CTAS * (k + 1) ? 16u : 0u));
      if (has_sym && t < NC_WORK) { polynomial(); nc_put(tile, r2, 1, v); }
      __syncthreads();
      if (has_sym) {
        nc_send_async(tile, false, Bm, ld, tm, tn, by_factor[tn], t, &bar_b);
        if (tm != tn) nc_send_async(tile, true, Bm, ld, tn, tm, by_factor[tm], t, &bar_b);
      }
      if (has_full && t < NC_WORK) {
        nc_wait(&bar_b, (uint32_t)k & 1u, &gave_up, g.wait_limit);
        next(cta, v);
      }
      __syncthreads();
      if (decides && has_full && !gave_up) nc_expect(&bar_b, b_bytes);
      if (has_full && t < NC_WORK) nc_put(tile, t >> 3, 16, v);
      __syncthreads();
      if (has_full) nc_send_async(tile, false, E, ld, fm, fn, by_col[fn] | by_row[fm], t, &bar_x);
      float* const old = X;
      X = E; E = Bm; Bm = old;
    }
    if (gave_up && t < NC_CTAS) {                // the others may have decided otherwise: tell them
      uint32_t there;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(nc_smem_u32(&lost)), "r"(t));
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(there), "r"(1) : "memory");
    }
  } else {
  for (; done_s == 0; ++k, cur ^= 1) {
    float mx = 0.f;
    double sq = 0.0;
    if (t < NC_WORK) {
      if (has_sym) { residual(mx, sq); nc_put(tile, r2, 1, v); }
      sq = warp_sum_d(sq);
      mx = warp_max(mx);
      if ((t & 31) == 0) { redd[t >> 5] = sq; redf[t >> 5] = mx; }
    }
    __syncthreads();
    if (t < 32) {
      nc_tell(nc_all_of(redd), sums[slot], cta);
      nc_tell((double)nc_most_of(redf), maxima[slot], cta);
    }
    if (has_sym) {
      nc_send(tile, false, E, ld, tm, tn, by_col[tn], t);
      if (tm != tn) nc_send(tile, true, E, ld, tn, tm, by_col[tm], t);
    }
    nc_cluster_sync();
    if (has_sym && t < NC_WORK) nc_tile<false>(E, E, ld, kp, tm * 32, tn * 32, v);      // does not wait for the decision
    if (decides) {
      double tmx = 0.0;
#pragma unroll
      for (int i = 0; i < NC_CTAS; ++i) tmx = fmax(tmx, maxima[slot][i]);
      decide(nc_total(sums[slot]), tmx);
    }
    slot ^= 1;
    __syncthreads();
    if (done_s != 0) break;
    if (has_sym && t < NC_WORK) { polynomial(); nc_put(tile, r2, 1, v); }
    nc_cluster_sync();                           // (the residual has been read everywhere)
    if (has_sym) {
      nc_send(tile, false, Bm, ld, tm, tn, by_factor[tn], t);
      if (tm != tn) nc_send(tile, true, Bm, ld, tn, tm, by_factor[tm], t);
    }
    nc_cluster_sync();
    float w[2][4];                               // a second tile's
    const int f1 = cta + NC_CTAS;
    if (t < NC_WORK) {
      next(cta, v);
      nc_put(tile, t >> 3, 16, v);
      if (f1 < tiles * tiles) next(f1, w);
    }
    nc_cluster_sync();                           // (and so has X)
    {
      const int fm = cta / tiles, fn = cta - fm * tiles;
      nc_send(tile, false, X, ld, fm, fn, by_col[fn] | by_row[fm], t);
    }
    if (f1 < tiles * tiles) {
      const int fm = f1 / tiles, fn = f1 - fm * tiles;
      __syncthreads();
      if (t < NC_WORK) nc_put(tile, t >> 3, 16, w);
      __syncthreads();
      nc_send(tile, false, X, ld, fm, fn, by_col[fn] | by_row[fm], t);
    }
    nc_cluster_sync();
  }
  }
  // From here on nobody writes into another's shared memory, and all know whether a wait was given up: then nothing is committed anywhere.
  nc_cluster_sync();
  if (lost) {
    const long long t0 = clock64();              // (let what is on its way land before the memory goes)
    while (clock64() - t0 < 4000000ll) {}
    if (cta == 0 && decides) {
      st->ns_done = NS_DONE_FAILED;
      st->timeout_site = 50;
      atomicOr(&st->status_flags, STATUS_FLAG_NS_FAILED | STATUS_FLAG_TIMEOUT);
    }
    return;
  }
  // accept or reject (see ns_commit_kernel, ns_commit_state_kernel): each CTA holds the rows of X that its tiles of the last product read
  if (done_s == NS_DONE_CONVERGED) {
    for (int f = cta; f < tiles * tiles; f += NC_CTAS) {
      const int row = (f / tiles) * 32 + (t >> 3), col = (f % tiles) * 32 + c4;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (row < d && col + j < d) {
          g.R[(size_t)row * d + col + j] = X[row * ld + col + j];
          g.M[(size_t)row * d + col + j] = 0.f;
        }
    }
  }
  if (cta == 0 && decides) {
    ns_ctl_store(ctl, st);
    ns_commit_state(st, g.n_endgame);
  }
}

// conqur_set_R's check of one narrow matrix, whose product is the launches' (the same chains), with the copy of what is accepted: one
// kernel where the product, the reduction of its partials and, behind the host's decision, the copy took three launches (whole call at
// d = 128 26 -> 21 us).
inline int nc_check_smem_bytes(int d) {              // (a matrix, and four rows that the product's last reads fetch past it)
  const int tiles = (d + 31) / 32;
  return (nc_matrix_floats(tiles) + 4 * nc_ld(tiles)) * (int)sizeof(float);
}
struct NcCheckArgs { const float* src; float* R; DevState* st; double* out; MailPost post; int d; };
// max|R^T R - I| (which drops NaN) and the sum of squares (which keeps it)
__host__ __device__ inline bool nc_accepts(double mx, double sq) { return (float)mx <= 1e-3f && sq - sq == 0.0; }

__global__ void __launch_bounds__(NC_THREADS, 1) nc_check_kernel(const NcCheckArgs g) {
  extern __shared__ __align__(16) float nc_smem[];
  __shared__ double redd[NC_WORK / 32];
  __shared__ float redf[NC_WORK / 32];
  __shared__ double sums[NC_CTAS], maxima[NC_CTAS];
  const int cta = (int)blockIdx.x, t = threadIdx.x, d = g.d, kp = (d + 3) / 4 * 4;
  const int tiles = (d + 31) / 32, ld = nc_ld(tiles), sym_tiles = tiles * (tiles + 1) / 2;
  float* X = nc_smem;
  for (int i = t; i < nc_matrix_floats(tiles); i += NC_THREADS) {
    const int r = i / ld, col = i - r * ld;
    X[i] = r < d && col < d ? g.src[(size_t)r * d + col] : 0.f;
  }
  __syncthreads();
  float mx = 0.f, v[2][4];
  double sq = 0.0;
  if (cta < sym_tiles && t < NC_WORK) {
    int tn = 0;
    while ((tn + 1) * (tn + 2) / 2 <= cta) ++tn;
    const int tm = cta - tn * (tn + 1) / 2;
    nc_tile<false>(X, X, ld, kp, tm * 32, tn * 32, v);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = tm * 32 + 2 * (t >> 3) + h, col = tn * 32 + 4 * (t & 7);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (row >= d || col + j >= d) continue;
        if (row == col + j) v[h][j] -= 1.f;
        mx = fmaxf(mx, fabsf(v[h][j]));
        sq += (tm != tn ? 2.0 : 1.0) * ((double)v[h][j] * (double)v[h][j]);
      }
    }
  }
  if (t < NC_WORK) {
    sq = warp_sum_d(sq);
    mx = warp_max(mx);
    if ((t & 31) == 0) { redd[t >> 5] = sq; redf[t >> 5] = mx; }
  }
  nc_cluster_sync();                             // (the sums of this CTA, and every CTA runs before anything is written into its memory)
  if (t < 32) {
    nc_tell(nc_all_of(redd), sums, cta);
    nc_tell((double)nc_most_of(redf), maxima, cta);
  }
  nc_cluster_sync();
  const double tsq = nc_total(sums);
  double tmx = 0.0;
#pragma unroll
  for (int i = 0; i < NC_CTAS; ++i) tmx = fmax(tmx, maxima[i]);
  if (cta == 0 && t == 0) {
    ns_arm_check(g.st);
    g.out[0] = tmx; g.out[1] = tsq;
    post_mail(g.post);                           // (the matrix given has been read; what follows is in the stream's order)
  }
  if (nc_accepts(tmx, tsq))
    for (int i = cta * NC_THREADS + t; i < d * d; i += NC_CTAS * NC_THREADS) g.R[i] = X[i / d * ld + i % d];
}
inline int nc_check_launch(const NcCheckArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(NC_CTAS); cfg.blockDim = dim3(NC_THREADS); cfg.dynamicSmemBytes = (size_t)nc_check_smem_bytes(a.d); cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = NC_CTAS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, nc_check_kernel, a) == cudaSuccess ? CONQUR_OK : CONQUR_ERR_CUDA;
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
    const bool yes = cudaFuncSetAttribute(ns_cluster_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, nc_smem_bytes(NC_MAX_D)) == cudaSuccess &&
                     cudaFuncSetAttribute(ns_cluster_kernel<false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                     cudaFuncSetAttribute(ns_cluster_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, nc_smem_bytes(NC_SMALL_D)) == cudaSuccess &&
                     cudaFuncSetAttribute(ns_cluster_kernel<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                     cudaFuncSetAttribute(nc_check_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, nc_check_smem_bytes(NC_MAX_D)) == cudaSuccess &&
                     cudaFuncSetAttribute(nc_check_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                     cudaOccupancyMaxActiveClusters(&n, ns_cluster_kernel<false>, &cfg) == cudaSuccess && n > 0;
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
  return cudaLaunchKernelEx(&cfg, a.d <= NC_SMALL_D ? ns_cluster_kernel<true> : ns_cluster_kernel<false>, a) == cudaSuccess ? CONQUR_OK : CONQUR_ERR_CUDA;
}

}  // namespace conqur
