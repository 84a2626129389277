// The fp32 step's two products on the tensor cores, at no less than fp32's precision.
//
// An fp32 number is the sum of three bf16 numbers of 8 bits each, and products of them are exact; but the tensor cores cut what they
// add toward zero (2^-23 of the sum, once per instruction of 16 terms).  A long sum kept in TMEM loses more than an fp32 chain
// does, and what is lost has the sum's sign, so that it does not average out over a matrix.
//
// Rotate.  The first two pieces of a number are multiples of units that its row of X (its column of R) shares: 2^-7 and 2^-16 of its
// largest number's power of two, at most 256 of them; the third is the rest, rounded.  Products of first pieces then add up exactly in
// one accumulator over 512 terms (at most 2^24 units, as neither side's norm exceeds 1 and its largest number is over 128 units; twice
// that, for a last bit, only where a row is its column), first with second pieces in another, and a third one takes the second with
// second pieces, first with third and second with third, whose sums are 2^-10 of the whole and less.  Eight products; the epilogue
// warps add the three to running fp32 sums, to nearest, every 512 terms.  Objectives of 768 .. 4096 wide rows of the calibration
// recipe lie 2e-9 (at most 9e-9) from 64 bits on either side, chains of fp32 multiply-adds 6e-9 (2e-8), and signs fall the other way half
// as often (pieces of each number's own leading bits, 64 terms an accumulator: fewer signs still, but 6e-8 .. 1.2e-7 low, always).
//
// Accumulate.  Pieces of each number's own leading bits (x = p0 + p1 + p2 exactly) times signs, three products; an accumulator holds 64 terms,
// small pieces first, and is then added to running fp32 sums.  M lies 0.5e-7 .. 1.8e-7 from 64 bits where the chains have 1.1e-7 ..
// 1.3e-6 (from d = 768 on, at no size more than they).
//
// What bounds it: the tensor cores and, with them busy, the board's power, where the CUDA cores' product is bound by its
// shared-memory reads.  1000 x 3072 fp32 rows: rotate 504 -> 110 us (96 tiles of 256 x 128 on 74 pairs, 32 instructions of 64 cycles a k
// block; 149 in two rounds of whole tiles), accumulate 409 -> 51, staging 8 -> 8 + 7 (the second pieces take the first ones' place); the
// whole step 885 -> 181.  (Six products of each number's own pieces, on tiles of 256 x 192: rotate 96, step 158.)
#pragma once
#include "conqur_simt.cuh"
#include "conqur_tc.cuh"

namespace conqur {

enum { SP_EPI_ROTATE = 0, SP_EPI_ROTATE_Q = 1, SP_EPI_ACCUM = 2 };

constexpr int SP_STAGES_MAX = 6;
constexpr int SP_THREADS = 384;                          // a warpgroup that loads and issues, two that add up
constexpr int SP_REGS_ISSUE = 56, SP_REGS_EPI = 208;     // registers a thread (launched with 168: 56 + 2 x 208 <= 3 x 168)
constexpr int SP_RING_BYTES = 196608;                    // operand tiles: two stages of 3 + 3 pieces
constexpr int SP_SMEM_BYTES = SP_RING_BYTES + 1024 + 8 * 4096 + 1024;   // ring, barriers, transposition buffers, alignment slack

struct SpArgs {
  int M, N, K;
  int n_stages, stage_bytes;
  float* outF; long long ldo;                            // Y (quantised targets) or M
  __nv_bfloat16* outS; long long lds;                    // targets
  const float* rs;                                       // 1, or 0 for rows that are left out
  unsigned *rowmax, *rowmin;
  StepSums step;                                         // ACCUM: what the step adds to the running sums
  double* part_d;                                        // objective partials: sixteen per tile (a warp's of either CTA)
  DevState* st;
  // rotate: tiles from `whole` on are shared out over k, `share` accumulators of them in a row to each pair (see sp_share_tail)
  int whole, share;
  float* sums;                                           // a shared part's running sums: HALF x 32 for each of its sixteen warps
  unsigned* arrived;                                     // per shared tile and warp (zero before the launch): parts that have left theirs
};

struct SpAux {
  uint64_t full[SP_STAGES_MAX], empty[SP_STAGES_MAX], tfull[2], tempty[2];
  uint32_t tmem_base;
  int abort_flag;
  double red_d[8];
};
static_assert(sizeof(SpAux) <= 1024, "reserved behind the ring");

namespace ptx {
// box of a 3-D map (column, row, piece) into this CTA's shared memory, its bytes counted on a barrier of the pair
__device__ __forceinline__ void tma_load_3d_pair(void* smem_dst, const CUtensorMap* tmap, uint32_t bar_cluster_addr, int x, int y,
                                                 int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"(tmap), "r"(bar_cluster_addr), "r"(x), "r"(y), "r"(z)
      : "memory");
}
template <int N> __device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
// 32 lanes x 32 consecutive fp32 columns.  The wait is tied to r, so that no use of it can move in front.
__device__ __forceinline__ void tmem_ld32_tied(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                 "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]),
                 "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),
                 "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}
// ... 16 columns
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                 "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
}  // namespace ptx

// Each number's own three bf16 pieces (+ e, a remainder below its last bit), two numbers at a time, packed with the first in the low half.
// A piece below 2^-126 is subnormal, so of values below about 2^-110 the low pieces are cut off at 2^-133 and their products with the
// other side at 2^-126 or so.  A step needs no other path for them: normalised rows have norm 1, so that much lies far below the rounding
// of any sum they enter, except that a feature which is that small in every row gets its row of M to 2^-126 absolutely, not relatively
// (fp32 itself ends at 2^-149).
__device__ __forceinline__ void sp_split2(float a, float b, float e0, float e1, uint32_t& w0, uint32_t& w1, uint32_t& w2) {
  w0 = bf16x2_pack(a, b);
  const float ra = a - __uint_as_float(w0 << 16), rb = b - __uint_as_float(w0 & 0xffff0000u);
  w1 = bf16x2_pack(ra, rb);
  w2 = bf16x2_pack((ra - __uint_as_float(w1 << 16)) + e0, (rb - __uint_as_float(w1 & 0xffff0000u)) + e1);
}
__device__ __forceinline__ void sp_split2(float a, float b, uint32_t& w0, uint32_t& w1, uint32_t& w2) {
  w0 = bf16x2_pack(a, b);
  const float ra = a - __uint_as_float(w0 << 16), rb = b - __uint_as_float(w0 & 0xffff0000u);
  w1 = bf16x2_pack(ra, rb);
  w2 = bf16x2_pack(ra - __uint_as_float(w1 << 16), rb - __uint_as_float(w1 & 0xffff0000u));
}

// A 32 x 32 fp32 block (lane = row) through the warp's transposition buffer to `out`: stored, or added with reductions at the
// L2.  Rows and columns past rows_ok / cols_ok are left out; 16-byte pieces where the block is whole and its rows aligned.
template <bool ADD>
__device__ __forceinline__ void sp_put_block(uint8_t* stg, int lane, const float (&v)[32], float* out, long long ld, int rows_ok,
                                             int cols_ok) {
  if (cols_ok >= 32 && (ld & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
    if (ADD) tc_red_block_f32(stg, lane, v, out, ld, rows_ok); else tc_store_block_f32(stg, lane, v, out, ld, rows_ok);
    return;
  }
#pragma unroll
  for (int p = 0; p < 8; ++p)
    *reinterpret_cast<float4*>(stg + lane * 128 + ((p ^ (lane & 7)) << 4)) = make_float4(v[4 * p], v[4 * p + 1], v[4 * p + 2], v[4 * p + 3]);
  __syncwarp();
  if (lane < cols_ok)
    for (int r = 0; r < rows_ok; ++r) {
      const float t = *reinterpret_cast<const float*>(stg + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4);
      if (ADD) atomicAdd(out + (long long)r * ld + lane, t); else out[(long long)r * ld + lane] = t;
    }
  __syncwarp();
}

// D[m][n] = sum_k A(m, k) B(n, k) on 256 x BN tiles of CTA pairs, operands as stacks of bf16 pieces (3-D maps: column, row,
// piece).  Warp 0 loads, warp 1 issues (CTA 0 for both), warps 4-11 add up the accumulators and write the tile (2 and 3 idle: the
// registers go by warpgroups).  A warp's 128 running sums, a block on its way from TMEM and the write-out's addresses do not all fit 208
// registers: the variants with 128 sums spill up to 20 bytes a thread outside the accumulation loop, the others up to 16 or nothing.
//   ROTATE    A = X (K-major), B = R^T (K-major): targets sgn(y) * rs as pc bf16 pieces, objective partials sum |y| rs
//   ROTATE_Q  the same products, stored as fp32 Y with the row's range
//   ACCUM     A = X, B = targets (both MN-major, contraction over rows): added to M, once per element and launch
template <int BN, int EPI, bool SHARE>
__global__ void __launch_bounds__(SP_THREADS, 1)
sp_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const SpArgs g) {
  constexpr bool MN = EPI == SP_EPI_ACCUM;               // orientation of both operands
  constexpr int PA = 3, PB = MN ? 1 : 3;                 // pieces of either operand
  constexpr int SUMS = MN ? 1 : 3, BUFS = MN ? 2 : 1;    // accumulators of a tile at a time, and sets of them
  constexpr int CHUNK = MN ? 1 : 8;                      // k blocks an accumulator holds
  static_assert(!MN || BN % 128 == 0, "MN-major tiles are 64 columns wide in each CTA of the pair");
  static_assert(SUMS * BUFS * BN <= 512, "TMEM columns");
  constexpr int A_BYTES = TC_BM * TC_BK * 2, B_ROWS = BN / 2, B_BYTES = B_ROWS * TC_BK * 2;
  constexpr int HALF = BN / 2, BLOCKS = HALF / 32;       // columns of the tile a warp adds up
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  SpAux* aux = reinterpret_cast<SpAux*>(smem + SP_RING_BYTES);
  volatile int* abort_flag = &aux->abort_flag;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();
  const int worker = (int)(blockIdx.x >> 1), n_workers = (int)(gridDim.x >> 1);
  const int tiles_m = (g.M + 255) / 256, tiles_n = (g.N + BN - 1) / BN, num_tiles = tiles_m * tiles_n;
  const int num_kb = (g.K + TC_BK - 1) / TC_BK;
  const int whole = SHARE ? g.whole : num_tiles, share = SHARE ? g.share : 1;
  const int chunks = (num_kb + CHUNK - 1) / CHUNK;       // accumulators of a tile
  // This pair's pos-th work item: a whole tile, or what it has of a shared one (k blocks kb0 .. kb1, which begin where an accumulator
  // does).
  struct Item { int tile, kb0, kb1; };
  auto get_item = [&](int pos, Item& w) -> bool {
    w.kb0 = 0; w.kb1 = num_kb;
    w.tile = worker + pos * n_workers;
    if (w.tile < whole) return true;
    if (!SHARE) return false;
    const int i = pos - (whole > worker ? (whole - worker + n_workers - 1) / n_workers : 0);
    const int units = (num_tiles - whole) * chunks, u0 = worker * share, u1 = min(units, u0 + share);
    const int u = i == 0 ? u0 : (u0 / chunks + i) * chunks;
    if (u >= u1) return false;
    const int t = u / chunks, c0 = u - t * chunks, c1 = min(chunks, c0 + u1 - u);
    w.tile = whole + t;
    w.kb0 = c0 * CHUNK; w.kb1 = min(num_kb, c1 * CHUNK);
    return true;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < g.n_stages; ++s) { ptx::mbar_init(&aux->full[s], 1); ptx::mbar_init(&aux->empty[s], 1); }
    for (int b = 0; b < 2; ++b) { ptx::mbar_init(&aux->tfull[b], 1); ptx::mbar_init(&aux->tempty[b], 16); }   // a warp's one arrival, both CTAs
    aux->abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
    ptx::prefetch_tmap(&tmA);
    ptx::prefetch_tmap(&tmB);
  }
  if (warp == 1) { ptx::tmem_alloc_pair(&aux->tmem_base, 512); ptx::tmem_relinquish_pair(); }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync_all();
  ptx::tc_fence_after();
  const uint32_t tmem_base = aux->tmem_base;
  int timeout_site = 0;

  if (warp < 4) {
    ptx::regs_dec<SP_REGS_ISSUE>();
    if (warp == 0 && lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      Item w;
      for (int pos = 0; ok && get_item(pos, w); ++pos) {
        int tm, tn;
        tc_tile_coords<1>(w.tile, tiles_m, tiles_n, 0, tm, tn);
        const int m0 = tm * 256 + (int)rank * TC_BM, n0 = tn * BN + (int)rank * B_ROWS;
        for (int kb = w.kb0; kb < w.kb1; ++kb) {
          if (!tc_wait(&aux->empty[stage], phase ^ 1u, abort_flag)) { ok = false; timeout_site = 1; break; }
          uint8_t* sa = smem + stage * g.stage_bytes;
          uint8_t* sb = sa + PA * A_BYTES;
          const uint32_t bar = ptx::mapa_u32(ptx::smem_u32(&aux->full[stage]), 0);
          if (rank == 0) ptx::mbar_expect_tx(&aux->full[stage], 2 * (PA * A_BYTES + PB * B_BYTES));
          const int k0 = kb * TC_BK;
          for (int p = 0; p < PA; ++p) {
            if (MN) {
#pragma unroll
              for (int h = 0; h < TC_BM / 64; ++h) ptx::tma_load_3d_pair(sa + p * A_BYTES + h * 8192, &tmA, bar, m0 + 64 * h, k0, p);
            } else {
              ptx::tma_load_3d_pair(sa + p * A_BYTES, &tmA, bar, k0, m0, p);
            }
          }
          for (int p = 0; p < PB; ++p) {
            if (MN) {
#pragma unroll
              for (int h = 0; h < B_ROWS / 64; ++h) ptx::tma_load_3d_pair(sb + p * B_BYTES + h * 8192, &tmB, bar, n0 + 64 * h, k0, p);
            } else {
              ptx::tma_load_3d_pair(sb + p * B_BYTES, &tmB, bar, k0, n0, p);
            }
          }
          if (++stage == g.n_stages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok) {                                         // copies in flight are counted in the other CTA: give them a fixed time
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000ll) {}
      }
    } else if (warp == 1 && rank == 0) {
      const uint32_t leader = ptx::elect_one();
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((MN ? 1u : 0u) << 15) | ((MN ? 1u : 0u) << 16) |
                             ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      const uint64_t ab0 = tc_smem_desc(ptx::smem_u32(smem), MN ? 8192 : 16, 1024);      // (addresses in units of 16 bytes)
      constexpr uint32_t STEP = MN ? 2048 / 16 : 32 / 16;
      const uint32_t full0 = ptx::smem_u32(&aux->full[0]);
      const uint32_t empty0 = full0 + (uint32_t)(offsetof(SpAux, empty) - offsetof(SpAux, full));
      const uint32_t tfull0 = full0 + (uint32_t)(offsetof(SpAux, tfull) - offsetof(SpAux, full));
      int stage = 0;
      uint32_t phase = 0, n_acc = 0;
      bool ok = true;
      Item w;
      for (int pos = 0; ok && get_item(pos, w); ++pos) {
        const int n_kb = SHARE ? w.kb1 - w.kb0 : num_kb;
        for (int kb = 0; kb < n_kb; ++kb) {
          const uint32_t buf = n_acc % BUFS;
          const bool first = kb % CHUNK == 0;
          if (first && !tc_wait_warp(&aux->tempty[buf], ((n_acc / BUFS) & 1u) ^ 1u, abort_flag)) { ok = false; timeout_site = 2; break; }
          if (!tc_wait_warp(&aux->full[stage], phase, abort_flag)) { ok = false; timeout_site = 3; break; }
          ptx::tc_fence_after();
          const uint64_t sa = ab0 + ((uint32_t)(stage * g.stage_bytes) >> 4), sb = sa + (uint32_t)(PA * (A_BYTES / 16));
          const uint32_t d_tmem = tmem_base + buf * (uint32_t)(SUMS * BN);
#pragma unroll
          for (int sum = MN ? 2 : 3; sum >= 0; --sum)    // what piece numbers add up to: small products first
#pragma unroll
            for (int i = sum > PB - 1 ? sum - (PB - 1) : 0; i <= (sum < PA - 1 ? sum : PA - 1); ++i) {
              const uint64_t ad = sa + (uint32_t)(i * (A_BYTES / 16)), bd = sb + (uint32_t)((sum - i) * (B_BYTES / 16));
              const bool starts = SUMS == 1 ? sum == 2 : sum == 3 ? i == 1 : sum < 2 && i == 0;
#pragma unroll
              for (int j = 0; j < TC_BK / 16; ++j)
                ptx::umma_bf16_by<true>(leader, d_tmem + (uint32_t)(SUMS == 1 ? 0 : (sum < 2 ? sum : 2) * BN), ad + j * STEP, bd + j * STEP, idesc,
                                        first && starts && j == 0 ? 0u : 1u);
            }
          ptx::umma_commit_by<true>(leader, empty0 + (uint32_t)stage * 8u);
          if (kb % CHUNK == CHUNK - 1 || kb == n_kb - 1) {
            ptx::umma_commit_by<true>(leader, tfull0 + buf * 8u);
            ++n_acc;
          }
          if (++stage == g.n_stages) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else {
    ptx::regs_inc<SP_REGS_EPI>();
    const int q = warp & 3, half = (warp >> 2) - 1, ew = warp - 4;
    uint8_t* stg = smem + SP_RING_BYTES + 1024 + ew * 4096;
    const uint32_t tempty0 = ptx::mapa_u32(ptx::smem_u32(&aux->tempty[0]), 0);
    const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * HALF);
    // (these warps have nothing to add up yet)
    if (MN && worker == 0 && rank == 1)
      finalize_step(g.st, 0, g.step, (int)threadIdx.x - 128, aux->red_d, [] { asm volatile("bar.sync 1, 256;" ::: "memory"); });
    uint32_t n_acc = 0;
    bool ok = true;
    Item w;
    for (int pos = 0; ok && get_item(pos, w); ++pos) {
      int tm, tn;
      tc_tile_coords<1>(w.tile, tiles_m, tiles_n, 0, tm, tn);
      float acc[HALF];
#pragma unroll
      for (int i = 0; i < HALF; ++i) acc[i] = 0.f;
      for (int kb = w.kb0; kb < w.kb1; kb += CHUNK, ++n_acc) {
        const uint32_t buf = n_acc % BUFS;
        // (a lane that gives up takes part in the warp's loads all the same; the vote below ends the loop for all lanes at once)
        if (!tc_wait(&aux->tfull[buf], (n_acc / BUFS) & 1u, abort_flag)) { ok = false; timeout_site = 4; }
        ptx::tc_fence_after();
#pragma unroll
        for (int c = 0; c < BLOCKS; ++c) {
          const uint32_t at = t_lane + buf * (uint32_t)(SUMS * BN) + (uint32_t)(c * 32);
          uint32_t r[32];
          ptx::tmem_ld32_tied(at, r);
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[c * 32 + i] += __uint_as_float(r[i]);
          if (SUMS == 3) {
            uint32_t m[32];
            ptx::tmem_ld32_tied(at + (uint32_t)(SUMS == 3 ? BN : 0), r);
            ptx::tmem_ld32_tied(at + (uint32_t)(SUMS == 3 ? 2 * BN : 0), m);
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[c * 32 + i] += __uint_as_float(r[i]) + __uint_as_float(m[i]);
          }
        }
        ptx::tc_fence_before();
        ok = __all_sync(0xffffffffu, ok);
        if (lane == 0) ptx::mbar_arrive_cluster(tempty0 + buf * (uint32_t)sizeof(uint64_t));
        if (!ok) break;
      }
      if (!ok) break;
      if (SHARE && w.kb1 - w.kb0 < num_kb) {
        // A shared tile: every part leaves its sums, and whichever of them comes last adds them all up in the order of the parts (so the
        // result does not depend on which that is) and goes on with the tile.  Warp by warp: nobody waits.
        const int t = w.tile - whole, first = t * chunks / share, last = ((t + 1) * chunks - 1) / share;      // the pairs that share it
        const int slots = chunks % share ? 2 : 1;        // (a pair has parts of at most two tiles)
        auto sums_of = [&](int pair) {
          const int slot = pair * slots + (pair * share / chunks == t ? 0 : 1);
          return g.sums + ((int64_t)(slot * 2 + (int)rank) * 8 + ew) * (HALF * 32) + lane;
        };
        float* mine = sums_of(worker);
#pragma unroll
        for (int i = 0; i < HALF; ++i) __stcg(mine + i * 32, acc[i]);
        __threadfence();
        __syncwarp();
        unsigned before = 0;
        if (lane == 0) before = atomicAdd(g.arrived + (2 * t + (int)rank) * 8 + ew, 1u);
        if (__shfl_sync(0xffffffffu, before, 0) != (unsigned)(last - first)) continue;
        __threadfence();
        const float* all = sums_of(first);
#pragma unroll
        for (int i = 0; i < HALF; ++i) acc[i] = __ldcg(all + i * 32);
        for (int p = first + 1; p <= last; ++p) {
          all = sums_of(p);
#pragma unroll
          for (int i = 0; i < HALF; ++i) acc[i] += __ldcg(all + i * 32);
        }
      }
      const int wrow0 = tm * 256 + (int)rank * TC_BM + q * 32, row = wrow0 + lane;
      const int rows_ok = min(32, max(0, g.M - wrow0));
      const bool row_ok = row < g.M;
      float rs = 0.f;
      if (EPI != SP_EPI_ACCUM) rs = row_ok ? g.rs[row] : 0.f;
      const uint32_t one = bf16_bits(rs);
      double sum = 0.0;
      float vmax = -3.0e38f, vmin = 3.0e38f;
#pragma unroll
      for (int c = 0; c < BLOCKS; ++c) {
        const int col0 = tn * BN + half * HALF + c * 32;
        if (rows_ok == 0 || col0 >= g.N) continue;       // uniform over the warp
        const int cols_ok = min(32, g.N - col0);
        float v[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = row_ok ? acc[c * 32 + i] : 0.f;
        if (EPI == SP_EPI_ROTATE) {
#pragma unroll
          for (int h = 0; h < 4; ++h) {                  // eight terms in fp32, then in double
            float a = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) a += fabsf(v[h * 8 + i]);
            sum += (double)a;
          }
          uint32_t ws[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float a = v[2 * i], b = v[2 * i + 1];
            const uint32_t lo = (a == 0.f) ? 0u : (one ^ ((__float_as_uint(a) >> 16) & 0x8000u));
            const uint32_t hi = (b == 0.f) ? 0u : (one ^ ((__float_as_uint(b) >> 16) & 0x8000u));
            ws[i] = lo | (hi << 16);
          }
          // (the targets' rows are padded to 64 columns; columns past N hold the zero operand's zeros)
          tc_store_block_bf16(stg, lane, ws, g.outS + (long long)wrow0 * g.lds + col0, g.lds, rows_ok);
        } else if (EPI == SP_EPI_ROTATE_Q) {
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (i < cols_ok) { vmax = fmaxf(vmax, v[i]); vmin = fminf(vmin, v[i]); }
          sp_put_block<false>(stg, lane, v, g.outF + (long long)wrow0 * g.ldo + col0, g.ldo, rows_ok, cols_ok);
        } else {
          sp_put_block<true>(stg, lane, v, g.outF + (long long)wrow0 * g.ldo + col0, g.ldo, rows_ok, cols_ok);
        }
      }
      if (EPI == SP_EPI_ROTATE_Q) {
        if (rs > 0.f) { atomicMax(g.rowmax + row, f2ord(vmax)); atomicMin(g.rowmin + row, f2ord(vmin)); }
      }
      if (EPI == SP_EPI_ROTATE) {
        const double t = warp_sum_d(sum * (double)rs);
        if (lane == 0) g.part_d[(2 * w.tile + (int)rank) * 8 + ew] = t;
      }
    }
  }

  if (timeout_site != 0) {
    atomicOr(&g.st->status_flags, STATUS_FLAG_TIMEOUT);
    g.st->timeout_site = timeout_site;
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync_all();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(tmem_base, 512);
  }
}

// The power of two of max's leading bit; pieces on a grid are multiples of 2^-7 of it (at most 256 of them: 8 bits), then of 2^-16.
__device__ __forceinline__ float sp_grid(float max) { return __uint_as_float(__float_as_uint(max) & 0x7f800000u); }
// Two pieces on the grid and the rest rounded to bf16 (additions of 1.5 2^23 grid units round to whole units; all differences are exact).
__device__ __forceinline__ void sp_split_grid(float v, float rest, float grid, float& p0, float& p1, float& p2) {
  const float c0 = grid * 98304.f, c1 = grid * 192.f;
  p0 = __fadd_rn(__fadd_rn(v, c0), -c0);
  const float r = __fadd_rn(v, -p0);
  p1 = __fadd_rn(__fadd_rn(r, c1), -c1);
  p2 = __fadd_rn(__fadd_rn(r, -p1), rest);
}

constexpr int SP_ARRIVED = 2048;                         // counters: sixteen warps of at most 128 shared tiles

// a1: row norms in fp32, and the normalised rows (the product x * rnorm with its rounding error) as pieces: on the row's grid for the
// rotate product (GRID), which also leaves the norms, or each number's own leading bits for the accumulate product, into the same
// place once the former has run.  Skipped rows are zeros.
// Four warps a row, whose pieces of it stay in the L1 between the two passes (1000 x 3072 fp32 rows: one warp a row 14.1 us).
template <typename TIn, bool GRID>
__global__ void __launch_bounds__(128) sp_stage_kernel(const TIn* __restrict__ X, int64_t n, int d, int64_t ld, float* __restrict__ rnorm,
                                                       float* __restrict__ rs, __nv_bfloat16* __restrict__ Xp, int64_t ldp,
                                                       int64_t piece, DevState* st, unsigned* arrived, unsigned* rowmax,
                                                       unsigned* rowmin) {
  if (GRID && blockIdx.x == 0)                           // (the rotate product that follows counts its shared tiles' parts there)
    for (int i = threadIdx.x; i < SP_ARRIVED; i += 128) arrived[i] = 0u;
  __shared__ float part[8];
  const int64_t row = blockIdx.x;
  const int lane = threadIdx.x & 31;
  const TIn* x = X + row * ld;
  const bool vec = ((d & 3) == 0) && ((reinterpret_cast<uintptr_t>(x) & (sizeof(TIn) * 4 - 1)) == 0);
  auto load = [&](int k, float (&v)[4]) {
    if (vec) {
      ld4_as_float(x + k, v);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = k + j < d ? ld_as_float(x + k + j) : 0.f;
    }
  };
  float r, grid = 0.f;
  if (GRID) {
    float ss = 0.f, mx = 0.f;
#pragma unroll 2
    for (int k = (int)threadIdx.x * 4; k < d; k += 512) {
      float v[4];
      load(k, v);
      ss = fmaf(v[0], v[0], ss); ss = fmaf(v[1], v[1], ss); ss = fmaf(v[2], v[2], ss); ss = fmaf(v[3], v[3], ss);
      mx = fmaxf(fmaxf(mx, fmaxf(fabsf(v[0]), fabsf(v[1]))), fmaxf(fabsf(v[2]), fabsf(v[3])));
    }
    ss = warp_sum(ss);
    mx = warp_max(mx);
    if (lane == 0) { part[threadIdx.x >> 5] = ss; part[4 + (threadIdx.x >> 5)] = mx; }
    __syncthreads();
    ss = (part[0] + part[1]) + (part[2] + part[3]);
    mx = fmaxf(fmaxf(part[4], part[5]), fmaxf(part[6], part[7]));
    const bool good = ss > 0.f && ss <= 3.0e38f;
    r = good ? 1.0f / sqrtf(ss) : 0.f;
    grid = good ? sp_grid(mx * r) : 0.f;                 // (rounding keeps the order: no |x * rnorm| is larger)
    if (threadIdx.x == 0) {
      if (!good) {
        atomicAdd(reinterpret_cast<unsigned long long*>(&st->step_skipped), 1ull);
        if (!(ss == 0.f)) atomicOr(&st->status_flags, STATUS_FLAG_NONFINITE);
      }
      rnorm[row] = r;
      rs[row] = good ? 1.f : 0.f;
      if (rowmax) { rowmax[row] = 0u; rowmin[row] = ~0u; }
    }
  } else {
    r = rnorm[row];
  }
  __nv_bfloat16* dst = Xp + row * ldp;
#pragma unroll 2
  for (int k = (int)threadIdx.x * 4; k < d; k += 512) {  // (rows of Xp are padded to 64 elements)
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (r > 0.f) load(k, v);
    uint2 p[3];
    float t[4], e[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) { t[j] = v[j] * r; e[j] = fmaf(v[j], r, -t[j]); }
    if (GRID) {
      float q[4][3];
#pragma unroll
      for (int j = 0; j < 4; ++j) sp_split_grid(t[j], e[j], grid, q[j][0], q[j][1], q[j][2]);
#pragma unroll
      for (int i = 0; i < 3; ++i) p[i] = make_uint2(bf16x2_pack(q[0][i], q[1][i]), bf16x2_pack(q[2][i], q[3][i]));
    } else {
      sp_split2(t[0], t[1], e[0], e[1], p[0].x, p[1].x, p[2].x);
      sp_split2(t[2], t[3], e[2], e[3], p[0].y, p[1].y, p[2].y);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) *reinterpret_cast<uint2*>(dst + i * piece + k) = p[i];
  }
}

// Largest magnitude of each column of R (cleared by the caller; the bits of numbers without sign are ordered like the numbers).
static __global__ void __launch_bounds__(256) sp_colmax_kernel(const float* __restrict__ R, int d, unsigned* __restrict__ colmax) {
  __shared__ float m[8][32];
  const int n = blockIdx.x * 32 + (threadIdx.x & 31), y = threadIdx.x >> 5;
  const int k0 = (int)((int64_t)d * blockIdx.y / gridDim.y), k1 = (int)((int64_t)d * (blockIdx.y + 1) / gridDim.y);
  float v = 0.f;
  if (n < d) {
#pragma unroll 8
    for (int k = k0 + y; k < k1; k += 8) v = fmaxf(v, fabsf(R[(int64_t)k * d + n]));
  }
  m[y][threadIdx.x & 31] = v;
  __syncthreads();
  if (y == 0 && n < d) {
#pragma unroll
    for (int i = 1; i < 8; ++i) v = fmaxf(v, m[i][threadIdx.x]);
    atomicMax(colmax + n, __float_as_uint(v));
  }
}
// R^T as three pieces (row n, column k), the first two on the grid of R's column n, rows ldp elements long: the rotate product then
// reads both operands along k.
static __global__ void __launch_bounds__(256) sp_split_rt_kernel(const float* __restrict__ R, int d, const unsigned* __restrict__ colmax,
                                                                 __nv_bfloat16* __restrict__ Rp, int64_t ldp, int64_t piece) {
  __shared__ float t[32][33];
  const int k0 = blockIdx.y * 32, n0 = blockIdx.x * 32, x = threadIdx.x & 31, y = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = k0 + y + 8 * i, n = n0 + x;
    t[y + 8 * i][x] = (k < d && n < d) ? R[(int64_t)k * d + n] : 0.f;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int n = n0 + y + 8 * i, k = k0 + x;
    if (n >= d || k >= d) continue;
    float p[3];
    sp_split_grid(t[x][y + 8 * i], 0.f, sp_grid(__uint_as_float(colmax[n])), p[0], p[1], p[2]);
#pragma unroll
    for (int j = 0; j < 3; ++j) Rp[j * piece + (int64_t)n * ldp + k] = __float2bfloat16_rn(p[j]);
  }
}

// Second pass of the two-pass step (see quant_target_kernel): Y -> target pieces, objective partials, diagnostics partials.
static __global__ void __launch_bounds__(256) sp_quant_target_kernel(const float* __restrict__ Y, int64_t n, int d,
                                                                     const float* __restrict__ rnorm, const float* __restrict__ rs,
                                                                     const unsigned* __restrict__ rowmax_ord,
                                                                     const unsigned* __restrict__ rowmin_ord, QuantSpec qs,
                                                                     double* __restrict__ partials, __nv_bfloat16* __restrict__ S,
                                                                     int64_t lds, double* __restrict__ part_diag) {
  const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const bool diag = part_diag != nullptr;
  double contrib = 0.0, dterm[4] = {0.0, 0.0, 0.0, 0.0};
  if (row < n) {
    const float r = rs[row];
    RowQuant rq{0.f, 1.f, 0.f, 0.f};
    if (qs.bits) rq = row_quant(qs, ord2f(rowmax_ord[row]), ord2f(rowmin_ord[row]), r > 0.f);
    const bool live = qs.bits ? (rq.inv > 0.f) : (r > 0.f);
    const float* y = Y + row * (int64_t)d;
    unsigned short* s = reinterpret_cast<unsigned short*>(S) + row * lds;
    float qsum = 0.f;
    RowDiag dg{0.f, 0.f, 0.f, 0.f};
    for (int j = lane; j < d; j += 32) {
      const float sg = second_pass_elem(y[j], r, qs, rq, qsum, diag && live, dg);
      const uint32_t neg = sg < 0.f ? 0x8000u : 0u;
      const bool zero = !live || sg == 0.f;
      s[j] = (unsigned short)(zero ? 0u : (0x3f80u ^ neg));                      // +-1
    }
    qsum = warp_sum(qsum);
    if (live) contrib = (double)(r * rq.delta) * (double)qsum;
    if (diag) row_diag_terms(dg, rnorm[row], d, live, dterm);
  }
  __shared__ double red[8][5];
  if (lane == 0) {
    red[threadIdx.x >> 5][0] = contrib;
    for (int k = 0; k < 4; ++k) red[threadIdx.x >> 5][1 + k] = dterm[k];
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w][threadIdx.x];
    if (threadIdx.x == 0) partials[blockIdx.x] = t;
    else if (diag) part_diag[(int64_t)(threadIdx.x - 1) * gridDim.x + blockIdx.x] = t;
  }
}

// ------------------------------------------------------------------ host side
// Steps that take the pieces.  Whole step, CUDA cores -> this, us (one B200):
//   fp32 rows, d = 768  n = 512 71 -> 49, 2048 157 -> 79;  1024  128 55 -> 45, 256 68 -> 46, 1000 147 -> 59, 8192 806 -> 278;
//              2048  64 82 -> 49, 2048 809 -> 164;  3072  1000 885 -> 181, 2048 1662 -> 321;  4096  32 214 -> 112, 2048 2747 -> 632
//   bf16 rows, d = 768  n = 64 56 -> 43, 2048 177 -> 79;  1024  64 74 -> 43;  3072  2048 1835 -> 320
// (below: too few 256-row tiles to fill the chip, and eight products for one.  Narrower ones would gain up to 1.4 times, but their M came
// out further from 64 bits than the CUDA cores': 384 x 8192 rows 0.9e-7 -> 1.7e-7, 512 x 2048 0.8e-7 -> 1.0e-7; at 768 2.6e-7 -> 1.8e-7)
constexpr int SP_MIN_D = 768;
inline bool sp_takes(int64_t n, int d, bool f32) {
  return d >= SP_MIN_D && (f32 ? n * d >= (d >= 1024 ? (int64_t)1 << 17 : (int64_t)1 << 18) : n >= 64);
}
struct SpLayout {
  int64_t ldp;                                           // row length of all pieces: d rounded up to 64
  size_t Xp, Sp, Rp, rs, colmax, arrived;
  size_t borrowed, borrowed_bytes;                       // what the rows' pieces borrow, all of it (0 bytes: they do not)
};
// Contexts that lay them out: those whose longest step takes them (a shorter one may not, a longer one always does).
inline bool sp_layout_wanted(int d, int P, int64_t n_max, bool f32) { return P == 1 && sp_takes(n_max, d, f32); }

// The rows' pieces borrow `scratch` (the update's matrices: no update runs during a step) where they fit it.  The fp32 target matrix C
// of a step on the CUDA cores shares its place with what a step over pieces writes instead, except where such a step goes through it
// too (fake-quantisation, diagnostics).  A row element costs 4 bytes as without pieces for up to 2.7 d rows, else 8.
template <typename Take>
inline void sp_make_layout(int d, int64_t n, bool through_c, size_t scratch, size_t scratch_bytes, size_t* C, SpLayout* L,
                           Take&& take) {
  L->ldp = ((int64_t)d + 63) / 64 * 64;
  const size_t rows = (size_t)(2 * 3 * n * L->ldp), targets = ((size_t)(2 * n * L->ldp) + 255) / 256 * 256;
  const size_t c_bytes = sizeof(float) * (size_t)n * d;
  const bool borrow = rows <= scratch_bytes;
  const size_t mine = targets + (borrow ? 0 : rows);
  *C = take(through_c || c_bytes > mine ? c_bytes : mine);
  L->Sp = through_c ? take(mine) : *C;
  L->Xp = borrow ? scratch : L->Sp + targets;
  L->Rp = take((size_t)(2 * 3 * d * L->ldp));
  L->rs = take(sizeof(float) * (size_t)n);
  L->colmax = take(sizeof(unsigned) * (size_t)d);
  L->arrived = take(sizeof(unsigned) * SP_ARRIVED);
  L->borrowed = scratch;
  L->borrowed_bytes = borrow ? scratch_bytes : 0;
}

// (column, row, piece) map over `pieces` bf16 matrices of rows x cols, `piece` elements apart; box 64 columns x box_rows.
inline int sp_make_tmap(CUtensorMap* tm, const void* ptr, uint64_t rows, uint64_t cols, uint64_t ld, uint64_t pieces, uint64_t piece,
                        uint32_t box_rows) {
  PFN_encodeTiled fn = tc_encode_fn();
  if (!fn) return CONQUR_ERR_CUDA;
  const cuuint64_t dims[3] = {cols, rows, pieces};
  const cuuint64_t strides[2] = {ld * 2, piece * 2};
  const cuuint32_t box[3] = {64, box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    std::fprintf(stderr, "conqur: cuTensorMapEncodeTiled (pieces) failed (%d)\n", (int)r);
    return CONQUR_ERR_CUDA;
  }
  return CONQUR_OK;
}

// Tile width of the accumulate product of M x N outputs on `pairs` CTA pairs: the one with the least rounds x width.  (The rotate
// product's three accumulators fill the TMEM at 128.)
constexpr int SP_ROT_BN = 128;
inline int sp_pick_bn(int64_t M, int64_t N, int pairs) {
  int best = 256;
  double cost = 1e300;
  for (int bn : {256, 128}) {
    const int64_t tiles = ((M + 255) / 256) * ((N + bn - 1) / bn);
    const double c = (double)((tiles + pairs - 1) / pairs) * (bn + 16);
    if (c < cost) { cost = c; best = bn; }
  }
  return best;
}
inline int64_t sp_tiles(int64_t M, int64_t N, int bn) { return ((M + 255) / 256) * ((N + bn - 1) / bn); }

// The rotate product's last, partial round of tiles is shared out over k: its accumulators (512 terms each), tile by tile, go to the
// pairs in runs of equal length, so that a pair works on parts of at most two tiles.  96 tiles on 74 pairs at d = 3072 are one round of
// six accumulators and 22 tiles in runs of two, 8 accumulator times instead of 12.  Whole step over whole tiles -> this, us, fp32 rows:
//   d = 1024  n = 200 51.3 -> 45.4, 512 55.6 -> 49.5;  2048  64 73.9 -> 49.3, 2048 167 -> 164, 4096 314 -> 301;  3072  64 101 -> 71, 512 131 -> 117,
//   1000 217 -> 181, 4096 660 -> 627;  4096  200 170 -> 132, 2048 668 -> 632
// Returns the length of a run: the tile's own length, with nothing shared (and a kernel without the code for it: 0.7 us of 24), where the
// longest run would be no shorter.  `room`: bytes for the parts' sums, which fewer and longer runs need less of.
inline int sp_share_tail(int64_t tiles, int pairs, int K, size_t room) {
  const int r = (int)(tiles % pairs), chunks = (K + 8 * TC_BK - 1) / (8 * TC_BK);
  if (r == 0 || 16 * r > SP_ARRIVED) return chunks;
  for (int share = (r * chunks + pairs - 1) / pairs; share < chunks; ++share) {
    const size_t runs = (size_t)(r * chunks + share - 1) / share, slots = chunks % share ? 2 : 1;
    if (runs * slots * 256 * SP_ROT_BN * sizeof(float) <= room) return share;
  }
  return chunks;
}

template <int BN, int EPI, bool SHARE = false>
inline int sp_launch_bn(int device, int pairs, cudaStream_t s, const CUtensorMap& a, const CUtensorMap& b, SpArgs g) {
  if constexpr (EPI != SP_EPI_ACCUM && !SHARE) {
    if (g.share < (g.K + 8 * TC_BK - 1) / (8 * TC_BK)) return sp_launch_bn<BN, EPI, true>(device, pairs, s, a, b, g);
  }
  auto kern = sp_gemm_kernel<BN, EPI, SHARE>;
  static std::atomic<unsigned long long> attr_dev_mask{0};
  const unsigned long long dev_bit = 1ull << (device & 63);
  if (!(attr_dev_mask.load(std::memory_order_acquire) & dev_bit)) {
    // the warpgroups' shares of registers come out of what the block is launched with: less, and they would wait for more forever
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess || fa.numRegs * 3 < SP_REGS_ISSUE + 2 * SP_REGS_EPI) return CONQUR_ERR_CUDA;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SP_SMEM_BYTES) != cudaSuccess) return CONQUR_ERR_CUDA;
    attr_dev_mask.fetch_or(dev_bit, std::memory_order_release);
  }
  g.stage_bytes = 3 * (TC_BM * TC_BK * 2) + (EPI == SP_EPI_ACCUM ? 1 : 3) * (BN / 2 * TC_BK * 2);
  g.n_stages = SP_RING_BYTES / g.stage_bytes < SP_STAGES_MAX ? SP_RING_BYTES / g.stage_bytes : SP_STAGES_MAX;
  const int64_t tiles = sp_tiles(g.M, g.N, BN);
  int64_t items = tiles;
  if (SHARE) {
    const int chunks = (g.K + 8 * TC_BK - 1) / (8 * TC_BK);
    g.whole = (int)(tiles - tiles % pairs);
    items = g.whole ? g.whole : (tiles * chunks + g.share - 1) / g.share;      // (runs are no more than pairs)
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (unsigned)(items < pairs ? items : pairs)); cfg.blockDim = dim3(SP_THREADS);
  cfg.dynamicSmemBytes = SP_SMEM_BYTES; cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a, b, g) == cudaSuccess ? CONQUR_OK : CONQUR_ERR_CUDA;
}
}  // namespace conqur
