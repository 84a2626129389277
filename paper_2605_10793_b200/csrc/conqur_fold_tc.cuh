// Block-diagonal weight folds on the tensor cores, at no less than fp32's precision (see conqur_split_tc.cuh for the pieces).
//
//   SIDE 0:  out[:, b] = W[:, b] R_b        SIDE 1:  out[b, :] = R_b^T W[b, :]        blocks of 64 or 128
//
// Both are R^T times W (SIDE 0 of W transposed): the product's first operand is 128 x 128 of blockdiag(R)^T (two 64-blocks and
// zeros), whose three bf16 pieces a CTA keeps in TMEM while it walks 128 x 128 tiles of W.  A tile arrives through the copy engine
// half a k at a time (three 32 KB buffers); eight warps split it into pieces in the swizzled operand layout, one half while the
// products read the other; one warp issues the six products of each half into an accumulator of its own (64 terms, small pieces
// first); eight warps add the two halves in fp32 and write the tile (on SIDE 0 a TMEM lane is a column of the output, so a warp's
// stores are turned into whole 16-byte pieces first).  W is read once and out written once: bound by that (128 KB a tile, 5.7 k cycles of
// an SM's share of the HBM rate; splitting takes 5 k, the products 3.1 k, writing 4.5 k).  A rotation comes through the copy engine into
// the pieces' place, ahead of W, and is split from there in 3 k cycles, once or twice a CTA (with single loads from memory, behind W's
// copies, 11 k).  32 blocks of 128, W 4096 x 4096, whole call: CUDA cores 111 us, this 57.5 (65 with single loads); 64 blocks 4096 wide
// INPUT 66 -> 58, where a thread's 4-byte stores had set the pace.
// Error against 64 bits, in 2^-24 of the result's norm, fp32 chain / this: 128-blocks 3.4 / 1.4, 64-blocks 2.4 / 1.3.
//
// Both operands are split after a multiplication by 2^32, so that no piece of any fp32 number is subnormal (its last bit is worth
// 2^-149 at least), and the sums come back by 2^-64: powers of two, which change no bit.  What is left are values that are not
// finite or so large that scaled sums could overflow; a fold that meets one says so, and the caller runs the CUDA-core kernel instead
// (32 blocks of 128, W 4096 x 4096 with a NaN: 64 -> 157 us; tiny values anywhere: 64).
#pragma once
#include "conqur_split_tc.cuh"
#include "conqur_tc_batched.cuh"

namespace conqur {

namespace ptx {
// 32 lanes x 8 consecutive columns: thread t of the warp writes row (lane base + t); complete after tmem_st_wait.
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&w)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"r"(taddr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}
}  // namespace ptx

constexpr int FB_CONV = 256;                             // splitting threads: two warpgroups; then loading and issuing, then two that write
constexpr int FB_THREADS = FB_CONV + 128 + 256;
constexpr int FB_REGS_CONV = 96, FB_REGS_ISSUE = 40, FB_REGS_EPI = 120;   // (launched with 96: 40 + 2 x 120 <= 3 x 96)
static_assert(FB_REGS_ISSUE + 2 * FB_REGS_EPI <= 3 * FB_REGS_CONV, "registers the block is launched with");
constexpr int FB_PIECE = 128 * 128 * 2;
constexpr int FB_HALF = 128 * 64 * 4, FB_RAW = 3;        // half a tile in fp32, and how many of them
constexpr int FB_TM_A = 256;                             // TMEM: two accumulators, then three pieces of 64 columns
constexpr int FB_SMEM_BYTES = 3 * FB_PIECE + FB_RAW * FB_HALF + 1024 + 8 * 4096 + 1024;
static_assert(FB_SMEM_BYTES <= 232448, "227 KB of dynamic shared memory per CTA");

struct FbArgs {
  const float *W, *R;
  float* out;
  int64_t ldw, ldo;
  int logdb, rows, cols;            // blocks of 1 << logdb
  int n_super, tiles;               // 128-wide groups of blocks; W tiles along the other dimension
  int copied, r_copied;             // 1: W's rows, R suit the copy engine (16-byte aligned)
  int* status;                      // page-locked host memory, two words cleared by the caller: flags, and whether a value was unfit
};
struct FbAux {
  uint64_t raw_full[FB_RAW], raw_free[FB_RAW], full[2], free_[2], tfull, tempty, rfull, rread;
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(FbAux) <= 1024, "reserved behind the operands");

constexpr float FB_UP = 4294967296.f, FB_DOWN = 1.f / FB_UP / FB_UP;     // 2^32, and back (128 products: 2^39 2^16 2^64 2^7 < 2^128)
constexpr float FB_W_LIMIT = 549755813888.f, FB_R_LIMIT = 65536.f;       // 2^39, 2^16
// Largest magnitude of what it is shown; NaN stays.
struct FbRange {
  float hi = 0.f;
  __device__ __forceinline__ void see(float v) { asm("max.NaN.f32 %0, %0, %1;" : "+f"(hi) : "f"(fabsf(v))); }
  __device__ __forceinline__ bool within(float limit) const { return hi < limit; }
};

template <int SIDE>
__global__ void __launch_bounds__(FB_THREADS, 1) fold_blocks_kernel(const __grid_constant__ CUtensorMap tmW,
                                                                     const __grid_constant__ CUtensorMap tmR, const FbArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sW = smem;                                    // pieces: two 64-column chunks of 128 rows x 128 bytes each, swizzled by the row
  uint8_t* sRaw = smem + 3 * FB_PIECE;
  FbAux* aux = reinterpret_cast<FbAux*>(sRaw + FB_RAW * FB_HALF);
  volatile int* abort_flag = &aux->abort_flag;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int total = g.n_super * g.tiles;
  const int t0 = (int)((int64_t)total * blockIdx.x / gridDim.x), t1 = (int)((int64_t)total * (blockIdx.x + 1) / gridDim.x);
  const int folded = SIDE == 0 ? g.cols : g.rows;       // length of the folded dimension
  const int db = 1 << g.logdb;

  // a group's rotation, 64 rows of one block either way, into the pieces' place while that is idle (one thread)
  auto copy_r = [&](int sb) {
    ptx::mbar_expect_tx(&aux->rfull, 2u * 64u * 4u << g.logdb);
#pragma unroll
    for (int h = 0; h < 2; ++h) ptx::tma_load_2d(sW + h * FB_PIECE, &tmR, &aux->rfull, 0, sb * 128 + 64 * h);
  };
  if (threadIdx.x == 0) {
    for (int s = 0; s < FB_RAW; ++s) { ptx::mbar_init(&aux->raw_full[s], 1); ptx::mbar_init(&aux->raw_free[s], FB_CONV / 32); }
    for (int b = 0; b < 2; ++b) { ptx::mbar_init(&aux->full[b], FB_CONV / 32); ptx::mbar_init(&aux->free_[b], 1); }
    ptx::mbar_init(&aux->tfull, 1);
    ptx::mbar_init(&aux->tempty, 8);
    ptx::mbar_init(&aux->rfull, 1);
    ptx::mbar_init(&aux->rread, FB_CONV / 32);
    aux->abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
    if (g.r_copied) copy_r(t0 / g.tiles);                // (the first, before the copies of W fill the queues)
    if (g.copied) ptx::prefetch_tmap(&tmW);
  }
  if (warp == FB_CONV / 32 + 1) { ptx::tmem_alloc(&aux->tmem_base, 512); ptx::tmem_relinquish(); }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = aux->tmem_base;
  int timeout_site = 0;

  if (warp < FB_CONV / 32) {
    // ---- splitting, one half of k after the other (64 rows of the tile on SIDE 1, 64 columns on SIDE 0): 4 elements eight times a thread
    int cur_sb = -1;
    bool bad = false;
    uint32_t n = 0, it = 0, nr = 0;
    bool ok = true;
    for (int t = t0; t < t1 && ok; ++t, ++n) {
      const int sb = t / g.tiles, j = t - sb * g.tiles;
      const uint32_t ph = (n & 1u) ^ 1u;
      if (sb != cur_sb) {
        // R^T into TMEM: lane = its row, two consecutive k per column.  (The products of the tile before read the old one last.)
        if (!tc_wait_warp(&aux->free_[0], ph, abort_flag) || !tc_wait_warp(&aux->free_[1], ph, abort_flag)) { timeout_site = 1; break; }
        ptx::tc_fence_after();
        if (g.r_copied && cur_sb >= 0 && threadIdx.x == 0) copy_r(sb);
        cur_sb = sb;
        FbRange rr;
        // a warp's 32 lanes and half of k lie in one block: its own where their block numbers agree, or there are zeros (two blocks side by
        // side, or one past the last).  Sixteen k at a time (8 columns of each piece), the next sixteen on their way meanwhile.
        const int a = (warp & 3) * 32 + lane, kh = warp >> 2;
        const bool in = sb * 128 + kh * 64 < folded && (kh * 64 >> g.logdb) == ((warp & 3) * 32 >> g.logdb);
        const float* src = (g.r_copied ? reinterpret_cast<const float*>(sW + kh * FB_PIECE) : g.R + ((int64_t)(sb * 128 + kh * 64) << g.logdb)) +
                           (a & (db - 1));
        if (g.r_copied && !tc_wait_warp(&aux->rfull, nr & 1u, abort_flag)) { timeout_site = 7; break; }
        const uint32_t ta = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(FB_TM_A + kh * 32);
        float v[2][16];
        auto fetch = [&](int c, float (&x)[16]) {
#pragma unroll
          for (int i = 0; i < 16; ++i) x[i] = in ? src[(c * 16 + i) << g.logdb] : 0.f;
        };
        auto split = [&](int c, const float (&x)[16]) {
          uint32_t w[3][8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            rr.see(x[2 * i]); rr.see(x[2 * i + 1]);
            sp_split2(x[2 * i] * FB_UP, x[2 * i + 1] * FB_UP, w[0][i], w[1][i], w[2][i]);
          }
#pragma unroll
          for (int p = 0; p < 3; ++p) ptx::tmem_st8(ta + (uint32_t)(p * 64 + c * 8), w[p]);
        };
        fetch(0, v[0]);
#pragma unroll 1
        for (int c = 0; c < 4; c += 2) {
          fetch(c + 1, v[1]);
          split(c, v[0]);
          if (c == 0) fetch(2, v[0]);
          split(c + 1, v[1]);
        }
        bad |= !rr.within(FB_R_LIMIT);
        ptx::tmem_st_wait();
        ptx::tc_fence_before();
        if (g.r_copied) {                                // (nobody's pieces go there before all have read it)
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&aux->rread);
          if (!tc_wait_warp(&aux->rread, nr & 1u, abort_flag)) { timeout_site = 7; break; }
          ++nr;
        }
      }
#pragma unroll 1
      for (int h = 0; h < 2; ++h, ++it) {
        const uint32_t slot = it % FB_RAW;
        if (g.copied && !tc_wait_warp(&aux->raw_full[slot], (it / FB_RAW) & 1u, abort_flag)) { ok = false; timeout_site = 2; break; }
        if (!tc_wait_warp(&aux->free_[h], ph, abort_flag)) { ok = false; timeout_site = 1; break; }
        FbRange rr;
        const int row0 = threadIdx.x >> (SIDE == 0 ? 4 : 5), c4 = threadIdx.x & (SIDE == 0 ? 15 : 31);
        constexpr int ROWS = SIDE == 0 ? 16 : 8;         // from one of a thread's eight pieces to the next
        float4 v[8];                                     // (all on their way before the first is split)
        if (g.copied) {
          const uint8_t* src = sRaw + slot * FB_HALF + row0 * (SIDE == 0 ? 256 : 512) + c4 * 16;
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = *reinterpret_cast<const float4*>(src + i * ROWS * (SIDE == 0 ? 256 : 512));
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int row = row0 + i * ROWS;
            const int gr = (SIDE == 0 ? j * 128 + row : sb * 128 + 64 * h + row), gc = (SIDE == 0 ? sb * 128 + 64 * h : j * 128) + c4 * 4;
            const float* p = g.W + (int64_t)gr * g.ldw + gc;
            const bool in = gr < g.rows;
            v[i].x = in && gc < g.cols ? p[0] : 0.f; v[i].y = in && gc + 1 < g.cols ? p[1] : 0.f;
            v[i].z = in && gc + 2 < g.cols ? p[2] : 0.f; v[i].w = in && gc + 3 < g.cols ? p[3] : 0.f;
          }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int row = row0 + i * ROWS, r = SIDE == 0 ? row : 64 * h + row, u = SIDE == 0 ? 8 * h + (c4 >> 1) : c4 >> 1;
          rr.see(v[i].x); rr.see(v[i].y); rr.see(v[i].z); rr.see(v[i].w);
          uint2 w[3];
          sp_split2(v[i].x * FB_UP, v[i].y * FB_UP, w[0].x, w[1].x, w[2].x);
          sp_split2(v[i].z * FB_UP, v[i].w * FB_UP, w[0].y, w[1].y, w[2].y);
          uint8_t* q = sW + (u >> 3) * 16384 + r * 128 + (((u & 7) ^ (r & 7)) << 4) + (c4 & 1) * 8;
#pragma unroll
          for (int p = 0; p < 3; ++p) *reinterpret_cast<uint2*>(q + p * FB_PIECE) = w[p];
        }
        bad |= !rr.within(FB_W_LIMIT);
        ptx::fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          if (g.copied) ptx::mbar_arrive(&aux->raw_free[slot]);
          ptx::mbar_arrive(&aux->full[h]);
        }
      }
    }
    if (*abort_flag && threadIdx.x == 0) {                 // let the rotation's copy land before the CTA's shared memory goes
      const long long c0 = clock64();
      while (clock64() - c0 < 4000000ll) {}
    }
    if (bad) reinterpret_cast<volatile int*>(g.status)[1] = 1;
  } else if (warp < FB_CONV / 32 + 4) {
    ptx::regs_dec<FB_REGS_ISSUE>();
    if (warp == FB_CONV / 32 && lane == 0 && g.copied) {
      // ---- copies of W, half a k of a tile at a time
      uint32_t it = 0;
      bool ok = true;
      for (int t = t0; t < t1 && ok; ++t) {
        const int sb = t / g.tiles, j = t - sb * g.tiles;
        for (int h = 0; h < 2; ++h, ++it) {
          const uint32_t slot = it % FB_RAW;
          if (!tc_wait(&aux->raw_free[slot], ((it / FB_RAW) & 1u) ^ 1u, abort_flag)) { ok = false; timeout_site = 3; break; }
          ptx::mbar_expect_tx(&aux->raw_full[slot], FB_HALF);
          if (SIDE == 0) ptx::tma_load_2d(sRaw + slot * FB_HALF, &tmW, &aux->raw_full[slot], sb * 128 + 64 * h, j * 128);
          else ptx::tma_load_2d(sRaw + slot * FB_HALF, &tmW, &aux->raw_full[slot], j * 128, sb * 128 + 64 * h);
        }
      }
      if (!ok) {                                         // let the copies in flight land before the CTA's shared memory goes
        const long long c0 = clock64();
        while (clock64() - c0 < 4000000ll) {}
      }
    } else if (warp == FB_CONV / 32 + 1) {
      const uint32_t leader = ptx::elect_one();
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((SIDE == 1 ? 1u : 0u) << 16) | ((uint32_t)(128 >> 3) << 17) |
                             ((uint32_t)(128 >> 4) << 24);
      const uint64_t dW = tc_smem_desc(ptx::smem_u32(sW), SIDE == 1 ? 16384 : 16, 1024);
      uint32_t n = 0;
      bool ok = true;
      for (int t = t0; t < t1 && ok; ++t, ++n) {
        if (!tc_wait_warp(&aux->tempty, (n & 1u) ^ 1u, abort_flag)) { timeout_site = 4; break; }
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {                    // halves of k, an accumulator each
          if (!tc_wait_warp(&aux->full[h], n & 1u, abort_flag)) { ok = false; timeout_site = 5; break; }
          ptx::tc_fence_after();
          uint32_t acc = 0;
#pragma unroll
          for (int sum = 2; sum >= 0; --sum)
#pragma unroll
            for (int i = 0; i <= sum; ++i)               // piece i of R, piece sum - i of W
#pragma unroll
              for (int jj = 0; jj < 4; ++jj) {
                ptx::umma_bf16_ta_by(leader, tmem_base + (uint32_t)(h * 128), tmem_base + (uint32_t)(FB_TM_A + i * 64 + (h * 4 + jj) * 8),
                                     dW + (uint32_t)(((sum - i) * FB_PIECE + (SIDE == 1 ? (h * 4 + jj) * 2048 : h * 16384 + jj * 32)) >> 4),
                                     idesc, acc);
                acc = 1u;
              }
          ptx::umma_commit_by<false>(leader, ptx::smem_u32(&aux->free_[h]));
        }
        if (ok) ptx::umma_commit_by<false>(leader, ptx::smem_u32(&aux->tfull));
      }
    }
  } else {
    ptx::regs_inc<FB_REGS_EPI>();
    // ---- writing: a warp takes 32 TMEM lanes and one half of the columns
    const int ew = warp - (FB_CONV / 32 + 4), q = warp & 3, half = ew >> 2;
    uint8_t* stg = smem + 3 * FB_PIECE + FB_RAW * FB_HALF + 1024 + ew * 4096;
    uint32_t n = 0;
    for (int t = t0; t < t1; ++t, ++n) {
      if (!tc_wait_warp(&aux->tfull, n & 1u, abort_flag)) { timeout_site = 6; break; }
      ptx::tc_fence_after();
      const uint32_t ta = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 64);
      float v[64];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t a[16], b[16];
        ptx::tmem_ld16(ta + (uint32_t)(c * 16), a);
        ptx::tmem_ld16(ta + 128u + (uint32_t)(c * 16), b);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[c * 16 + i] = __uint_as_float(a[i]) + __uint_as_float(b[i]);
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&aux->tempty);
      const int sb = t / g.tiles, j = t - sb * g.tiles;
      // lane: row of the rotation's transpose, i.e. of out (SIDE 1) or column of it (SIDE 0); v: the other coordinate
      const int f = sb * 128 + q * 32 + lane, o0 = j * 128 + half * 64;
      const int other = SIDE == 0 ? g.rows : g.cols;
      if (SIDE == 0) {
        // 32 rows of 32 columns at a time, turned in the warp's buffer into 16-byte pieces of a row where out's rows allow them (64 stores of
        // 4 bytes a thread took 6.3 k cycles a tile and set its pace, sixteen of 16 bytes take 4.5 k)
        const int c0 = sb * 128 + q * 32;
        const bool whole = c0 + 32 <= folded && (g.ldo & 3) == 0 && (reinterpret_cast<uintptr_t>(g.out) & 15) == 0;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int r0 = o0 + c * 32;
          if (whole) {
            float* const sf = reinterpret_cast<float*>(stg);
#pragma unroll
            for (int i = 0; i < 32; ++i) sf[i * 32 + (lane ^ ((i & 7) << 2))] = v[c * 32 + i] * FB_DOWN;
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int r = i * 4 + (lane >> 3), piece = lane & 7;
              const float4 t4 = *reinterpret_cast<const float4*>(sf + r * 32 + ((piece ^ (r & 7)) << 2));
              if (r0 + r < other) __stcs(reinterpret_cast<float4*>(g.out + (int64_t)(r0 + r) * g.ldo + c0 + piece * 4), t4);
            }
            __syncwarp();
          } else if (f < folded) {
            float* p = g.out + (int64_t)r0 * g.ldo + f;
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (r0 + i < other) __stcs(p + (int64_t)i * g.ldo, v[c * 32 + i] * FB_DOWN);
          }
        }
      } else {
        const int m0 = sb * 128 + q * 32, rows_ok = min(32, max(0, g.rows - m0));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float b[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) b[i] = v[c * 32 + i] * FB_DOWN;
          const int cols_ok = min(32, max(0, g.cols - (o0 + c * 32)));
          if (cols_ok > 0) sp_put_block<false>(stg, lane, b, g.out + (int64_t)m0 * g.ldo + o0 + c * 32, g.ldo, rows_ok, cols_ok);
        }
      }
    }
  }
  if (timeout_site != 0) *reinterpret_cast<volatile int*>(g.status) = STATUS_FLAG_TIMEOUT;
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == FB_CONV / 32 + 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, 512);
  }
}

// 2-D fp32 tensor (rows x cols, row stride ld elements); box of box_cols x box_rows, out-of-range elements read as zero.
inline int tc_make_tmap_f32(CUtensorMap* tm, const void* ptr, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_cols, uint32_t box_rows) {
  PFN_encodeTiled fn = tc_encode_fn();
  if (!fn) return CONQUR_ERR_CUDA;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {ld * 4};
  const cuuint32_t box[2] = {box_cols, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    std::fprintf(stderr, "conqur: cuTensorMapEncodeTiled (fp32) failed (%d)\n", (int)r);
    return CONQUR_ERR_CUDA;
  }
  return CONQUR_OK;
}

// Folds that take this kernel: several blocks of 64 or 128, enough of W, and tiles that are not mostly empty (each group of blocks
// costs its rotation's splitting, however short the other side is).  Whole call (as timed in a row), fp32 CUDA cores -> this, us,
// blocks x other side:
//   of 128         8 x 1024 35 -> 33, 64 x 96 35 -> 36, 64 x 512 52 -> 39, 64 x 2048 118 -> 58, 256 x 128 52 -> 40, 1024 x 96 116 -> 75;
//                  not 32 x 160 31.5 -> 34, 64 x 64 30 -> 33, 128 x 32 30 -> 33, 512 x 64 53 -> 55, 1024 x 1 57 -> 82, 1024 x 64 75 -> 91
//   of 64, INPUT   64 x 1024 42 -> 39, 512 x 256 61 -> 49, 1024 x 256 97 -> 65;  not 512 x 160 48 -> 52, 1024 x 1 33 -> 54
//   of 64, OUTPUT  64 x 2048 48 -> 44, 512 x 512 71 -> 58, 256 x 2048 114 -> 77; not 64 x 1024 38 -> 40, 1024 x 256 71 -> 77
// (the shapes that are "not" with the rotation loaded singly: up to a tenth less now, and the line has stayed; the CUDA cores give an
// element the same bits in a call of any shape, this kernel gives it its own)
inline bool fold_blocks_takes(int64_t rows, int64_t cols, int block, int side) {
  const bool in = side == CONQUR_FOLD_INPUT;
  const int64_t folded = in ? cols : rows, other = in ? rows : cols;
  if ((block != 64 && block != 128) || folded < 2 * (int64_t)block) return false;
  const int64_t least = block == 128 ? 96 : in ? 256 : 512, whole = block == 128 ? 60 : in ? 240 : 480;
  return other >= least && rows * cols >= whole * (128 * 128) && ((folded + 127) / 128) * ((other + 127) / 128) < (int64_t)1 << 30;
}
inline int fold_blocks_launch(const float* W, int64_t ldw, int rows, int cols, const float* R, int block, int side, float* out,
                              int64_t ldo, int* status, int dev, int sms, cudaStream_t s) {
  static std::atomic<unsigned long long> attr_dev_mask{0};
  const unsigned long long dev_bit = 1ull << (dev & 63);
  if (!(attr_dev_mask.load(std::memory_order_acquire) & dev_bit)) {
    for (auto kern : {fold_blocks_kernel<0>, fold_blocks_kernel<1>}) {
      // (the warpgroups' shares of registers come out of what the block is launched with)
      cudaFuncAttributes fa;
      if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess || fa.numRegs < FB_REGS_CONV) return CONQUR_ERR_CUDA;
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, FB_SMEM_BYTES) != cudaSuccess) return CONQUR_ERR_CUDA;
    }
    attr_dev_mask.fetch_or(dev_bit, std::memory_order_release);
  }
  FbArgs g{W, R, out, ldw, ldo, block == 64 ? 6 : 7, rows, cols, 0, 0, 0, 0, status};
  const bool in = side == CONQUR_FOLD_INPUT;
  g.n_super = ((in ? cols : rows) + 127) / 128;
  g.tiles = ((in ? rows : cols) + 127) / 128;
  CUtensorMap tm = {};
  if ((ldw & 3) == 0 && ldw < (int64_t)1 << 38 && (reinterpret_cast<uintptr_t>(W) & 15) == 0) {    // (a map's strides end at 2^40 bytes)
    if (tc_make_tmap_f32(&tm, W, (uint64_t)rows, (uint64_t)cols, (uint64_t)ldw, in ? 64 : 128, in ? 128 : 64) != CONQUR_OK) return CONQUR_ERR_CUDA;
    g.copied = 1;
  }
  CUtensorMap tr = {};
  if ((reinterpret_cast<uintptr_t>(R) & 15) == 0) {
    if (tc_make_tmap_f32(&tr, R, (uint64_t)(in ? cols : rows), (uint64_t)block, (uint64_t)block, (uint32_t)block, 64) != CONQUR_OK) return CONQUR_ERR_CUDA;
    g.r_copied = 1;
  }
  const int64_t total = (int64_t)g.n_super * g.tiles;
  const unsigned grid = (unsigned)(total < sms ? total : sms);
  if (in) fold_blocks_kernel<0><<<grid, FB_THREADS, FB_SMEM_BYTES, s>>>(tm, tr, g);
  else fold_blocks_kernel<1><<<grid, FB_THREADS, FB_SMEM_BYTES, s>>>(tm, tr, g);
  return cudaGetLastError() == cudaSuccess ? CONQUR_OK : CONQUR_ERR_CUDA;
}

}  // namespace conqur
