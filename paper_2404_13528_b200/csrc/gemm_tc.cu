// bf16 GEMM on the 5th-generation tensor cores (tcgen05), fp32 accumulation in TMEM.
//
//   out[b, m, n] = epilogue( sum_k A[b, m, k] * B[b, n, k] )
//
// Both operands are read "reduction dimension contiguous" (Section 3.2.2) straight from the
// producer's buffer: the composed index map of an eliminated layout run is affine here, so it
// becomes a TMA tensor map (up to 5-D box) and costs nothing at run time.  An operand whose
// rows -- not its reduction dimension -- are contiguous in the producer's buffer (the NCHW ->
// NHWC case) is loaded as it lies and multiplied through the MN-major operand mode of the
// tensor core, so that transpose disappears as well.
//
// Persistent CTAs (one per SM) of 19 warps: warp 0 issues TMA loads into a 3- to 6-stage shared-memory
// ring (a second producer warp takes the B operand when the reduction is long), warp 1 owns the TMEM
// allocation and issues tcgen05.mma (one thread) into one of two accumulator buffers, warps 2-17 run
// the epilogue of the previous tile meanwhile (TMEM -> registers -> bias / GELU / RoPE / residual ->
// bf16 -> staged whole-row stores, optionally scattering rows through an index map: window reverse +
// reverse cyclic shift folded into the store).
#include <cstring>
#include <mutex>
#include <unordered_map>

#include "gemm_tc.cuh"
#include "ptx.cuh"


namespace smartmem {
namespace {

constexpr int BM = 128;
constexpr int BK = 64;                   // 64 bf16 = 128 bytes = one swizzle row
constexpr int A_STAGE_BYTES = BM * BK * 2;

struct OpCoord {
  int rank, mn_major;
  FastDiv tiles_inner;
  int n_outer;                           // outer row atoms then batch atoms, innermost first
  int n_outer_row;
  FastDiv outer[3];
};

struct GemmArgs {
  int M, N, K;
  int tiles_n, tiles_m, batch;
  FastDiv fd_tiles_n, fd_tiles_m;        // tile index -> (tile_n, tile_m, batch) without hardware division
  OpCoord ca, cb;
  __nv_bfloat16* out;
  long long ldc, out_batch_stride;
  const __nv_bfloat16* bias;
  const __nv_bfloat16* residual;
  int gelu, has_rowmap, b_settled;
  int rope_cols, rope_S, rope_pos0;      // columns [0, rope_cols) are rotated; position = rope_pos0 + row % rope_S
  int rope_half;                         // R / 2: the first R columns of each 128-wide head rotate, pairs (i, i + R/2)
  float rope_c;                          // log2(theta) / (R / 2)
  int seg_cols;                          // > 0: column segment s of a row goes to seg_out[s] + row * seg_ld[s]
  __nv_bfloat16* seg_out[3];
  long long seg_ld[3];
  __nv_bfloat16* out2;                   // second copy of the result, transposed inside groups of out2_S rows (null: none)
  FastDiv fd_out2_S;
  int* status;
  int tma_out;                           // lean epilogue: the output leaves as TMA boxes (tensor map tmC) instead of per-thread stores
  DevMap rowmap;
};

// The two-stage kernel's staging tiles, either as boxes (two of 64 KB) or as rows of 512 bytes, the two tiles' side by side and eight rows
// shifted against one another by 16 bytes (eight threads on eight rows then write distinct banks).
constexpr int kStageBoxBytes = 4 * 32 * 512, kStageBytes = 16 * (8 * 1024 + 112);
static_assert(kStageBytes >= 2 * kStageBoxBytes, "room for either form");
__device__ __forceinline__ uint32_t stage_row_off(int row, uint32_t tile) { return (uint32_t)(row * 1024 + (row >> 3) * 112 + (row & 7) * 16) + tile * 512u; }

// Tile -> TMA coordinates of an operand: row origin inside the innermost row atom and the digits
// of the outer row atoms / batch atoms (every tensor map is padded to rank 5, so all five
// coordinates always exist and stay in registers).
struct TileCoord {
  int row0, o0, o1, o2;
};
__device__ __forceinline__ TileCoord op_coords(const OpCoord& oc, uint32_t tile, uint32_t batch, int tile_rows) {
  uint32_t q = fd_div(tile, oc.tiles_inner);
  TileCoord tc;
  tc.row0 = (int)(tile - q * oc.tiles_inner.d) * tile_rows;
  int o[3] = {0, 0, 0};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (i < oc.n_outer) {
      const bool from_rows = i < oc.n_outer_row;
      const uint32_t src = from_rows ? q : batch;
      const uint32_t qq = fd_div(src, oc.outer[i]);
      o[i] = (int)(src - qq * oc.outer[i].d);
      if (from_rows) q = qq; else batch = qq;
    }
  }
  tc.o0 = o[0]; tc.o1 = o[1]; tc.o2 = o[2];
  return tc;
}
__device__ __forceinline__ void tma_load_op(const OpCoord& oc, void* dst, const CUtensorMap* tm, uint64_t* bar, int k0,
                                            int row0, const TileCoord& tc) {
  ptx::tma_load_5d(dst, tm, bar, oc.mn_major ? row0 : k0, oc.mn_major ? k0 : row0, tc.o0, tc.o1, tc.o2);
}
// CTA pair: the bytes are counted on the even CTA's barrier (a shared::cluster address)
__device__ __forceinline__ void tma_load_op_pair(const OpCoord& oc, void* dst, const CUtensorMap* tm, uint32_t bar_cluster, int k0,
                                                 int row0, const TileCoord& tc) {
  ptx::tma_load_5d_pair(dst, tm, bar_cluster, k0, row0, tc.o0, tc.o1, tc.o2);
}

struct TileIdx {
  uint32_t tile_n, tile_m, batch;
};
__device__ __forceinline__ TileIdx split_tile(uint32_t t, const FastDiv& fn, const FastDiv& fm) {
  const uint32_t r = fd_div(t, fn), b = fd_div(r, fm);
  return {t - r * fn.d, r - b * fm.d, b};
}

// The work items of a kernel: its tiles, and where 256-wide pair tiles leave a last round of which fewer than half the pairs have a
// tile, that round's tiles as two 128-wide halves each.  A half takes 0.56 of a tile's time, so the round ends that much earlier.
struct TileItem {
  TileIdx ti;
  int n_off;                             // first column of the item inside its tile
  bool half;
};
template <bool HALVES>
struct Halves {                          // (only the kernels that take halves pay for the parameter)
  CUtensorMap map;                       // a half's B rows
  uint32_t wide_tiles;                   // tiles from this one on come as halves
};
template <>
struct Halves<false> {};
template <bool HALVES>
__device__ __forceinline__ TileItem tile_item(uint32_t t, const GemmArgs& g, const Halves<HALVES>& hv) {
  if constexpr (HALVES) {
    if (t >= hv.wide_tiles) {
      const uint32_t u = t - hv.wide_tiles;
      return {split_tile(hv.wide_tiles + (u >> 1), g.fd_tiles_n, g.fd_tiles_m), (int)(u & 1) * 128, true};
    }
  }
  return {split_tile(t, g.fd_tiles_n, g.fd_tiles_m), 0, false};
}

constexpr int kEpiWarps = 16;
constexpr int kThreads = 64 + 32 * kEpiWarps + 32;      // + a second TMA producer warp (B operand)

// Persistent kernel: one CTA per SM walks over output tiles (tile = blockIdx.x + i * gridDim.x).
// The shared-memory ring and two TMEM accumulator buffers run across tile boundaries, so the
// loads and MMAs of tile i+1 overlap the epilogue of tile i.
//
// PAIR: the two CTAs of a cluster share one 256 x BN tile (cta_group::2).  Each loads its own 128 rows of A and its own
// half of the B tile's rows -- two thirds of the operand bytes a lone CTA pulls in per product, which is what bounds a
// 128 x 256 tile (48 KB per k-block against the ~64 bytes per clock an SM takes in) -- and keeps its own 128 rows of the
// accumulator, which it drains itself.  The even CTA counts both CTAs' bytes on its `full` barriers, issues the products
// and signals `empty` / `tmem_full` in both CTAs; both CTAs' epilogue warps arrive on its `tmem_empty`.
// LEAN: the epilogue knows bias and GELU only (no rotary embedding or second copy; a residual and a row map only on 128-wide
// tiles), which leaves it the registers to pull its whole accumulator slice out of tensor memory at once and hand the buffer
// back before any arithmetic -- for short reductions, where a tile's products take no longer than its epilogue -- and its rows
// leave as 32 x 32 TMA boxes, or as 32-byte vectors through the row map, without staging a tile.  On single CTAs (us):
// M = 50 176, N = 384, K = 128 16.4 -> 11.1, M = 12 544, N = 768, K = 192 9.5 -> 7.1.
// ROWS: the two-stage kernel's tiles leave a row of 512 bytes at a time instead of in boxes (store_rows).
template <int BN, int STAGES, bool A_MN, bool PAIR, bool LEAN, bool ROWS>
__global__ void __launch_bounds__(kThreads, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmC, const __grid_constant__ GemmArgs g,
               const __grid_constant__ Halves<PAIR && BN == 256> hv) {
  static_assert(!PAIR || ((BN == 256 || BN == 128) && !A_MN), "CTA pairs: 256- or 128-wide tiles, K-major A");
  static_assert(!LEAN || BN % 128 == 0, "the lean epilogue's boxes are 32 columns wide");
  constexpr bool RES = !LEAN || BN == 128;                 // the epilogue can add a residual
  constexpr int BN_CTA = PAIR ? BN / 2 : BN;               // rows of B this CTA loads
  constexpr int B_STAGE_BYTES = BN_CTA * BK * 2;
  constexpr uint32_t ACC_COLS = BN <= 32 ? 32 : BN <= 64 ? 64 : BN <= 128 ? 128 : 256;   // one accumulator buffer
  constexpr uint32_t TMEM_COLS = 2 * ACC_COLS;
  constexpr uint32_t IDESC = ptx::make_idesc_bf16(PAIR ? 2 * BM : BM, BN, A_MN, false);
  constexpr bool HALVES = PAIR && BN == 256;               // the last round's tiles may come as halves
  const CUtensorMap* map_half = &tmB;
  if constexpr (HALVES) map_half = &hv.map;
  constexpr uint32_t IDESC_HALF = ptx::make_idesc_bf16(2 * BM, BN / 2, false, false);

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * A_STAGE_BYTES;
  // lean epilogue: a 32 x 32 output box per epilogue warp (64-byte rows, 64-byte swizzle), right behind the ring
  constexpr int CBOX_BYTES = 32 * 64;
  uint8_t* cstage = sB + STAGES * B_STAGE_BYTES;
  // two-stage kernel: two staging tiles of 128 x 256, each four lane quadrants of four 32 x 64 boxes (128-byte rows and swizzle) or of 32 rows
  constexpr bool QTMA = STAGES == 2;
  uint64_t* full = reinterpret_cast<uint64_t*>(cstage + (LEAN ? kEpiWarps * CBOX_BYTES : QTMA ? kStageBytes : 0));
  uint64_t* empty = full + STAGES;
  uint64_t* tmem_full = empty + STAGES;                      // [2]
  uint64_t* tmem_empty = tmem_full + 2;                      // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tmem_empty + 2);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  uint8_t* stage_base = reinterpret_cast<uint8_t*>(tmem_slot + 4);                      // 16-byte aligned

  const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (warp: provably uniform)
  const int nkb = (g.K + BK - 1) / BK;
  const int last_ksteps = (g.K - (nkb - 1) * BK + 15) / 16;
  const bool two_producers = nkb >= 8;
  const uint32_t tiles = (uint32_t)g.tiles_n * g.tiles_m * g.batch;         // PAIR: tiles_m counts 256-row tiles
  uint32_t total_tiles = tiles;                                             // (work items)
  if constexpr (HALVES) total_tiles = 2 * tiles - hv.wide_tiles;
  const uint32_t rank = PAIR ? ptx::cluster_ctarank() : 0u;                  // which half of the pair's tile
  const bool leader = rank == 0;
  const uint32_t cta_first = PAIR ? blockIdx.x >> 1 : blockIdx.x, cta_step = PAIR ? gridDim.x >> 1 : gridDim.x;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      ptx::mbar_init(&full[s], two_producers ? 2 : 1);  // one arrival per producer warp
      ptx::mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(&tmem_full[b], 1);
      ptx::mbar_init(&tmem_empty[b], PAIR ? 2 * kEpiWarps : kEpiWarps);
    }
    *abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmB);
    if constexpr (HALVES) {
      if (hv.wide_tiles < tiles) ptx::prefetch_tensormap(&hv.map);
    }
    if ((QTMA && !ROWS) || (LEAN && g.tma_out)) ptx::prefetch_tensormap(&tmC);
  }
  if (warp == 1) {
    if constexpr (PAIR) ptx::tmem_alloc_pair(tmem_slot, TMEM_COLS);
    else ptx::tmem_alloc(tmem_slot, TMEM_COLS);
  }
  ptx::tc_fence_before();
  if constexpr (PAIR) {
    __syncwarp();
    ptx::cluster_sync();            // the peer's barriers are initialised before anything of this CTA signals them
  } else {
    __syncthreads();
  }
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // Everything above overlapped the previous kernel's tail, and so does the B operand's first round of the ring where nothing in flight
  // writes it (TcEpilogue::b_settled): its producer waits behind that.  (Not in its ring: a thousand lanes that poll for the length of a kernel
  // slow down those that they wait for.)
  if (warp < 2 + kEpiWarps || !two_producers || !g.b_settled) {
    pdl_wait();
    pdl_launch_dependents();
  }

  if (warp == 0) {
    // The whole warp walks the loop and one elected lane issues (as for the products below): under a branch on one lane every
    // operand of a copy is moved to a uniform register in front of it, about 210 ns per copy instead of 120 -- and a k-block's
    // two copies have less than 270 ns if the products are not to wait for them.
    uint32_t kbg = 0, s = 0, ph = 0;                         // k-block counter across tiles, ring position
    bool ok = true;
    const uint32_t full0 = PAIR ? ptx::mapa(ptx::smem_u32(full), 0) : 0u;     // the even CTA's `full` barriers
    for (uint32_t t = cta_first; t < total_tiles && ok; t += cta_step) {
      const TileItem item = tile_item<HALVES>(t, g, hv);
      const TileIdx ti_ = item.ti;
      const uint32_t tile_n = ti_.tile_n, tile_m = PAIR ? 2 * ti_.tile_m + rank : ti_.tile_m, batch = ti_.batch;
      const TileCoord ta = op_coords(g.ca, tile_m, batch, BM), tb = op_coords(g.cb, tile_n, batch, BN);
      const bool half = HALVES && item.half;
      const int brow0 = tb.row0 + (HALVES ? item.n_off : 0) + (int)rank * (half ? BN_CTA / 2 : BN_CTA);
      const uint32_t b_bytes = half ? B_STAGE_BYTES / 2 : B_STAGE_BYTES;
      const CUtensorMap* mapB = half ? map_half : &tmB;
      for (int kb = 0; kb < nkb; ++kb, ++kbg) {
        ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(&empty[s], ph ^ 1, abort_flag, g.status) ? 1 : 0) != 0;
        if (!ok) break;
        if (ptx::elect_one()) {
          if constexpr (PAIR) {
            if (leader) ptx::mbar_expect_tx(&full[s], 2 * (two_producers ? A_STAGE_BYTES : A_STAGE_BYTES + b_bytes));
            tma_load_op_pair(g.ca, sA + s * A_STAGE_BYTES, &tmA, full0 + s * 8, kb * BK, ta.row0, ta);
            if (!two_producers) tma_load_op_pair(g.cb, sB + s * B_STAGE_BYTES, mapB, full0 + s * 8, kb * BK, brow0, tb);
          } else {
            ptx::mbar_expect_tx(&full[s], two_producers ? A_STAGE_BYTES : A_STAGE_BYTES + B_STAGE_BYTES);
            tma_load_op(g.ca, sA + s * A_STAGE_BYTES, &tmA, &full[s], kb * BK, ta.row0, ta);
            if (A_MN) tma_load_op(g.ca, sA + s * A_STAGE_BYTES + A_STAGE_BYTES / 2, &tmA, &full[s], kb * BK, ta.row0 + 64, ta);
            if (!two_producers) tma_load_op(g.cb, sB + s * B_STAGE_BYTES, &tmB, &full[s], kb * BK, tb.row0, tb);
          }
        }
        __syncwarp();
        if (++s == STAGES) { s = 0; ph ^= 1; }
      }
    }
    if (lane == 0 && *abort_flag) {
      if (PAIR) {
        // unwinding a pair: the copies of the odd CTA are counted on the even CTA's barriers, so each side just gives
        // whatever is in flight a fixed time to land
        const unsigned long long t0 = ptx::globaltimer();
        while (ptx::globaltimer() - t0 < 100000ull) {
        }
      } else {
        // unwinding: give copies already in flight a bounded chance to land before the CTA leaves
        for (uint32_t k = (kbg > (uint32_t)STAGES ? kbg - STAGES : 0); k < kbg; ++k) {
          const unsigned long long t0 = ptx::globaltimer();
          while (!ptx::mbar_try_wait(&full[k % STAGES], (k / STAGES) & 1) && ptx::globaltimer() - t0 < 2000000ull) {
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // The whole warp walks the loop and one elected lane issues: with warp-uniform control flow the descriptors
    // stay in uniform registers (under a branch on lane 0 each operand is moved there in front of every product).
    if (leader) {                                     // (the odd CTA's warp 1 only owns its tensor-memory allocation)
      uint32_t it = 0, s = 0, ph = 0;                 // ring position and its phase carry over tiles
      const uint32_t a_base = ptx::smem_u32(sA), b_base = ptx::smem_u32(sB);
      bool ok = true;
      for (uint32_t t = cta_first; t < total_tiles && ok; t += cta_step, ++it) {
        const uint32_t buf = it & 1, use = it >> 1;
        ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(&tmem_empty[buf], (use & 1) ^ 1, abort_flag, g.status) ? 1 : 0) != 0;   // epilogue drained it
        if (!ok) break;
        ptx::tc_fence_after();
        const uint32_t d_tmem = tmem_base + buf * ACC_COLS;
        uint32_t idesc = IDESC;
        if constexpr (HALVES) idesc = t >= hv.wide_tiles ? IDESC_HALF : IDESC;
        for (int kb = 0; kb < nkb; ++kb) {
          ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(&full[s], ph, abort_flag, g.status) ? 1 : 0) != 0;
          if (!ok) break;
          ptx::tc_fence_after();
          // K-major, 128-byte swizzle: 8-row groups are 1024 bytes apart; one k16 step is 32 bytes
          // along the swizzled row.  MN-major: 64-row chunks are 8192 bytes apart (leading offset),
          // 8-deep k groups 1024 bytes apart, one k16 step is 2048 bytes.  A k16 step only moves the
          // start-address field of the descriptor, so the issuing thread adds a constant per MMA.
          const uint64_t ad0 = A_MN ? ptx::make_smem_desc(a_base + s * A_STAGE_BYTES, A_STAGE_BYTES / 2, 1024)
                                    : ptx::make_smem_desc(a_base + s * A_STAGE_BYTES, 16, 1024);
          const uint64_t bd0 = ptx::make_smem_desc(b_base + s * B_STAGE_BYTES, 16, 1024);
          constexpr uint64_t A_STEP = (A_MN ? 2048 : 32) >> 4, B_STEP = 32 >> 4;
          const bool last_kb = kb == nkb - 1;
          auto mma = [&](uint64_t ad, uint64_t bd, uint32_t acc) {
            if constexpr (PAIR) ptx::tc_mma_bf16_pair(d_tmem, ad, bd, idesc, acc);
            else ptx::tc_mma_bf16(d_tmem, ad, bd, IDESC, acc);
          };
          if (ptx::elect_one()) {
            if (!last_kb || last_ksteps == BK / 16) {
              mma(ad0, bd0, kb ? 1u : 0u);
#pragma unroll
              for (int k = 1; k < BK / 16; ++k) mma(ad0 + k * A_STEP, bd0 + k * B_STEP, 1u);
            } else {
              for (int k = 0; k < last_ksteps; ++k) mma(ad0 + k * A_STEP, bd0 + k * B_STEP, (kb | k) ? 1u : 0u);
            }
            if constexpr (PAIR) {
              ptx::tc_commit_pair(&empty[s], 3);
              if (last_kb) ptx::tc_commit_pair(&tmem_full[buf], 3);
            } else {
              ptx::tc_commit(&empty[s]);
              if (last_kb) ptx::tc_commit(&tmem_full[buf]);
            }
          }
          __syncwarp();
          if (++s == STAGES) { s = 0; ph ^= 1; }
        }
      }
    }
  } else if (warp >= 2 + kEpiWarps) {
    // second producer: the B operand (long reductions only; a short one is
    // cheaper to feed from one thread)
    if (two_producers) {
      uint32_t s = 0, ph = 1;
      bool ok = true, waited = !g.b_settled;
      const uint32_t full0 = PAIR ? ptx::mapa(ptx::smem_u32(full), 0) : 0u;
      for (uint32_t t = cta_first; t < total_tiles && ok; t += cta_step) {
        const TileItem item = tile_item<HALVES>(t, g, hv);
        const uint32_t tile_n = item.ti.tile_n, batch = item.ti.batch;
        const TileCoord tb = op_coords(g.cb, tile_n, batch, BN);
        const bool half = HALVES && item.half;
        const int brow0 = tb.row0 + (HALVES ? item.n_off : 0) + (int)rank * (half ? BN_CTA / 2 : BN_CTA);
        const uint32_t b_bytes = half ? B_STAGE_BYTES / 2 : B_STAGE_BYTES;
        const CUtensorMap* mapB = half ? map_half : &tmB;
        for (int kb = 0; kb < nkb; ++kb) {
          if (!waited && kb == STAGES) {
            pdl_wait();
            waited = true;
          }
          ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(&empty[s], ph, abort_flag, g.status) ? 1 : 0) != 0;
          if (!ok) break;
          if (ptx::elect_one()) {
            if constexpr (PAIR) {
              if (leader) ptx::mbar_expect_tx(&full[s], 2 * b_bytes);
              tma_load_op_pair(g.cb, sB + s * B_STAGE_BYTES, mapB, full0 + s * 8, kb * BK, brow0, tb);
            } else {
              ptx::mbar_expect_tx(&full[s], B_STAGE_BYTES);
              tma_load_op(g.cb, sB + s * B_STAGE_BYTES, &tmB, &full[s], kb * BK, tb.row0, tb);
            }
          }
          __syncwarp();
          if (++s == STAGES) { s = 0; ph ^= 1; }
        }
        if (!waited) pdl_wait();                             // (a reduction no longer than the ring)
        waited = true;
      }
    }
  } else {
    // Epilogue.  Warp (quadrant q, column group grp) owns rows q*32..q*32+31 (one TMEM lane per
    // thread) and CG = BN/4 columns, handled in rounds of RC <= 32 columns:
    //   phase 1 (thread = row): TMEM -> fp32 -> [RoPE] -> +bias -> [GELU] -> [+residual] -> bf16 -> staging row
    //   phase 2 (threads spread along the row): 16-byte stores, RC*2 contiguous bytes per row,
    // so a store instruction writes whole 32-byte sectors and several sectors of one line at once.
    constexpr int CG = BN / 4;
    constexpr bool DIRECT = PAIR || LEAN;                            // rows leave the registers as 32-byte stores: no staging at all
    constexpr bool EARLY = DIRECT && LEAN;                   // accumulator slice to registers first, buffer released at once
    constexpr int RC = (BN == 256 && STAGES == 4 && !PAIR && !LEAN) ? 16 : (CG > 32 ? 32 : CG);   // 4 stages leave less staging room
    constexpr int ROUNDS = CG / RC;
    constexpr int RH = ROUNDS > 1 ? ROUNDS / 2 : 1;
    constexpr int VPR = RC / 8;                              // 16-byte vectors per row per round
    constexpr int STG_ROW = RC * 2 + 16;                     // bytes; the pad keeps phase 1 conflict-free
    const int e = warp - 2;
    const int q = warp & 3;                                  // TMEM lane quadrant this warp may read
    const int grp = e >> 2;
    constexpr bool QSTAGE = !DIRECT && !(BN == 256 && STAGES == 4);  // per-quadrant staging of whole rows
    constexpr bool QBULK = BN == 256 && !A_MN && !QTMA;      // staged rows leave as bulk copies (512-byte rows; not the MN-major-A kernel: 13.1 vs 12.1 us)
    constexpr bool BARE = QTMA;                              // nothing but conversion and store: no bias, GELU, residual, rotation, map or second copy
    constexpr bool ROPE = !LEAN && !BARE && !A_MN && BN >= 128;   // kernels that rotate columns
    constexpr int QROW = BN * 2 + 16;                        // bytes; the pad keeps phase 1 conflict-free
    uint8_t* stage = stage_base + e * (32 * STG_ROW);
    uint8_t* qstage = stage_base + q * (32 * QROW);
    uint32_t it = 0;
    bool ok = true;
    const bool res_wide = (reinterpret_cast<uintptr_t>(g.residual) & 31) == 0;   // (row offsets of a pair's output are multiples of 16 elements)
    const uint32_t tmem_empty0 = PAIR ? ptx::mapa(ptx::smem_u32(tmem_empty), 0) : 0u;   // the even CTA's barriers
    for (uint32_t t = cta_first; t < total_tiles && ok; t += cta_step, ++it) {
      const TileItem item = tile_item<HALVES>(t, g, hv);
      const TileIdx ti_ = item.ti;
      const uint32_t tile_n = ti_.tile_n, tile_m = PAIR ? 2 * ti_.tile_m + rank : ti_.tile_m, batch = ti_.batch;
      const uint32_t buf = it & 1, use = it >> 1;
      const int n0 = tile_n * BN + (HALVES ? item.n_off : 0);
      const bool rope_tile = ROPE && g.rope_cols > 0 && n0 < g.rope_cols;
      if (HALVES && item.half && grp >= 2 && !rope_tile) {   // a half's 128 columns are the first two groups' (of a rotated one, everybody's)
        ok = ptx::mbar_wait(&tmem_full[buf], use & 1, abort_flag, g.status);
        if (!ok) break;
        if (lane == 0) ptx::mbar_arrive_cluster(tmem_empty0 + buf * 8);
        continue;
      }
      const int row = tile_m * BM + q * 32 + lane;
      const bool row_ok = row < g.M;
      long long o2_base = 0;                                 // second copy: row = b * S + s goes to out2[b][col][s]
      if (!LEAN && !BARE && g.out2) {
        const uint32_t b2 = fd_div((uint32_t)row, g.fd_out2_S);
        o2_base = (long long)b2 * g.N * g.fd_out2_S.d + ((uint32_t)row - b2 * g.fd_out2_S.d);
      }
      // column-segmented output: a tile never straddles segments (seg_cols is a multiple of BN), so
      // the whole tile has one base and one pitch; the base is biased by the segment's first column
      __nv_bfloat16* out_t = g.out;
      long long ld_t = g.ldc;
      if (!BARE && g.seg_cols > 0) {
        const int sg = n0 / g.seg_cols;
        out_t = g.seg_out[sg] - (long long)sg * g.seg_cols;
        ld_t = g.seg_ld[sg];
      }
      // Output offset of this thread's row, through the row map where the store is a scatter.  (Requested a tile ahead, with the residual, its
      // registers spill and the kernel is slower.)
      long long off = 0;
      if (!BARE) {                                           // (boxes go by coordinates, rows by their own)
        if (row_ok) off = g.has_rowmap ? devmap_eval_unrolled(g.rowmap, (uint32_t)row) : (long long)row * ld_t;
        off += (long long)batch * g.out_batch_stride;
      }
      const __nv_bfloat16* __restrict__ rrow = (RES && !BARE && g.residual) ? g.residual + off : nullptr;
      auto col_of = [&](int rd) {
        return BN == 256 ? 128 * (grp >> 1) + 32 * (grp & 1) + RC * (rd % RH) + 64 * (rd / RH) : grp * CG;
      };

      uint4 res[VPR];
      auto fetch_res = [&](int c0) {
        if constexpr (DIRECT) {                              // (32-byte aligned rows, N a multiple of 16) whole sectors per load
          if (rrow && row_ok && res_wide) {
#pragma unroll
            for (int v = 0; v < VPR; v += 2) {
              res[v] = res[v + 1] = make_uint4(0, 0, 0, 0);
              if (n0 + c0 + v * 8 < g.N) ptx::ld_global_v8(rrow + n0 + c0 + v * 8, res[v], res[v + 1]);
            }
            return;
          }
        }
#pragma unroll
        for (int v = 0; v < VPR; ++v) {
          res[v] = make_uint4(0, 0, 0, 0);
          if (rrow && row_ok && n0 + c0 + v * 8 + 8 <= g.N) res[v] = *reinterpret_cast<const uint4*>(rrow + n0 + c0 + v * 8);
        }
      };
      if (!BARE) fetch_res(col_of(0));                       // in flight while this tile's MMAs still run

      // Rotated columns: pairs (i, i + R/2) of the first R columns of each 128-wide head (R = 128: the whole head).  A warp takes the 16 pairs
      // i = 16 grp + j of every head of the tile (both halves of a pair, as two blocks of 16 columns), or past R two blocks that stay as they
      // are, so each angle's sine and cosine are worked out once per row and tile, while the products still run.  One element at a time, after
      // them, they were three operations of the special-function unit each, 3 us of a 128 x 256 tile: a layer of 666 rows, hidden 1024, was
      // 4.1 us slower with all columns rotated than with 32 of 128.
      const int rope_blocks = g.rope_half >> 4;              // blocks of 16 columns in half of R: 1, 2 or 4
      const bool rotated = grp < rope_blocks;
      float sn[ROPE ? 16 : 1], cs[ROPE ? 16 : 1];
      if constexpr (ROPE) {
        if (rope_tile && rotated) {
          // angle = position * theta^(-i/(R/2)), reduced mod 2 pi in two steps, then the hardware sine / cosine: no table traffic (a [S, 64]
          // table read 16 bytes per lane per row slowed the whole kernel by a fifth)
          const float pos = (float)(row_ok ? g.rope_pos0 + row % g.rope_S : 0);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float f = ptx::ex2(-(float)(grp * 16 + j) * g.rope_c);
            const float ang = pos * f;
            const float kk = rintf(ang * 0.15915494309189535f);
            float red = fmaf(-kk, 6.2831854820251465f, ang);
            red = fmaf(kk, 1.7484556e-7f, red);
            sn[j] = __sinf(red);
            cs[j] = __cosf(red);
          }
        }
      }
      ok = ptx::mbar_wait(&tmem_full[buf], use & 1, abort_flag, g.status);
      if (!ok) break;
      ptx::tc_fence_after();
      const uint32_t taddr = tmem_base + buf * ACC_COLS + ((uint32_t)(q * 32) << 16);
      uint8_t* qtile = cstage + (it & 1) * kStageBoxBytes + q * (kStageBoxBytes / 4);
      uint8_t* qline = cstage + stage_row_off(q * 32 + lane, it & 1);
      if constexpr (QTMA) {
        // what left this staging tile two tiles ago has been read
        if (lane < 8) ptx::bulk_wait_group_read<1>();
        asm volatile("bar.sync %0, 128;" ::"r"(1 + q) : "memory");
      }
      if constexpr (QSTAGE && QBULK) {
        // the previous tile's row copies have read the staging rows before anyone overwrites them
        if (lane < 8) ptx::bulk_wait_group_read<0>();
        asm volatile("bar.sync %0, 128;" ::"r"(1 + q) : "memory");
      }

      // EARLY: the whole accumulator slice of the thread (ROUNDS x RC values) moves to registers first and the buffer goes
      // back to the issuing warp before any arithmetic or store, so the next tile but one starts as early as it can
      uint32_t rall[EARLY ? ROUNDS : 1][RC];
      if constexpr (EARLY) {
#pragma unroll
        for (int rd = 0; rd < ROUNDS; ++rd) ptx::tmem_ld_cols<RC>(taddr + col_of(rd), rall[rd]);
        ptx::tmem_ld_wait();
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if constexpr (PAIR) ptx::mbar_arrive_cluster(tmem_empty0 + buf * 8);
          else ptx::mbar_arrive(&tmem_empty[buf]);
        }
      }
      if constexpr (ROPE) {
        if (rope_tile) {
          const int b0 = rotated ? grp : grp / rope_blocks * 2 * rope_blocks + grp % rope_blocks;
          auto put = [&](int c0, const uint32_t (&w)[8]) {   // 16 columns of the thread's row
            const uint4 lo = make_uint4(w[0], w[1], w[2], w[3]), hi = make_uint4(w[4], w[5], w[6], w[7]);
            if constexpr (DIRECT) {
              if (row_ok) ptx::st_global_v8(out_t + off + n0 + c0, lo, hi);
            } else if constexpr (QSTAGE) {
              *reinterpret_cast<uint4*>(qstage + lane * QROW + c0 * 2) = lo;
              *reinterpret_cast<uint4*>(qstage + lane * QROW + c0 * 2 + 16) = hi;
            } else {
              *reinterpret_cast<uint4*>(stage + lane * STG_ROW) = lo;
              *reinterpret_cast<uint4*>(stage + lane * STG_ROW + 16) = hi;
              __syncwarp();
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const int rr = (lane + 32 * i) >> 1, seg = lane & 1;
                const long long roff = __shfl_sync(0xFFFFFFFFu, off, rr);
                const int rok = __shfl_sync(0xFFFFFFFFu, (int)row_ok, rr);
                const uint4 pk = *reinterpret_cast<const uint4*>(stage + rr * STG_ROW + seg * 16);
                if (rok) *reinterpret_cast<uint4*>(out_t + roff + n0 + c0 + seg * 8) = pk;
              }
              __syncwarp();
            }
          };
          const int heads = HALVES && item.half ? 1 : BN / 128;
#pragma unroll 1
          for (int h = 0; h < heads; ++h) {
            const int c0 = h * 128 + b0 * 16, c1 = c0 + rope_blocks * 16;
            uint32_t x[16], y[16], w[8];
            ptx::tmem_ld16(taddr + c0, x);
            ptx::tmem_ld16(taddr + c1, y);
            ptx::tmem_ld_wait();
            if (rotated) {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const float a = __uint_as_float(x[j]), b = __uint_as_float(y[j]);
                x[j] = __float_as_uint(a * cs[j] - b * sn[j]);
                y[j] = __float_as_uint(b * cs[j] + a * sn[j]);
              }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) w[j] = float2_to_bf16x2(__uint_as_float(x[2 * j]), __uint_as_float(x[2 * j + 1]));
            put(c0, w);
#pragma unroll
            for (int j = 0; j < 8; ++j) w[j] = float2_to_bf16x2(__uint_as_float(y[2 * j]), __uint_as_float(y[2 * j + 1]));
            put(c1, w);
          }
        }
      }
      if (!rope_tile) {
#pragma unroll
        for (int rd = 0; rd < ROUNDS; ++rd) {
          const int c0 = col_of(rd);
          float acc[RC];
          uint4 bv[VPR];                                       // this round's bias columns: requested before the wait on tensor memory
          if (!BARE && g.bias) {
#pragma unroll
            for (int v = 0; v < VPR; ++v) {
              bv[v] = make_uint4(0, 0, 0, 0);
              if (n0 + c0 + v * 8 + 8 <= g.N) bv[v] = *reinterpret_cast<const uint4*>(g.bias + n0 + c0 + v * 8);
            }
          }
          {
            uint32_t rv_local[EARLY ? 1 : RC];
            uint32_t* rv = EARLY ? rall[EARLY ? rd : 0] : rv_local;
            if constexpr (!EARLY) {
              ptx::tmem_ld_cols<RC>(taddr + c0, rv);
              ptx::tmem_ld_wait();
            }
#pragma unroll
            for (int j = 0; j < RC; ++j) acc[j] = __uint_as_float(rv[j]);
          }
          if (!BARE && g.bias) {
#pragma unroll
            for (int v = 0; v < VPR; ++v) {
              const uint32_t w[4] = {bv[v].x, bv[v].y, bv[v].z, bv[v].w};
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const float2 f = bf16x2_to_float2(w[j]);
                acc[v * 8 + 2 * j] += f.x;
                acc[v * 8 + 2 * j + 1] += f.y;
              }
            }
          }
          if (!BARE && g.gelu) {
#pragma unroll
            for (int j = 0; j < RC; ++j) acc[j] = gelu_tanh(acc[j]);
          }
          if (!BARE && rrow) {
#pragma unroll
            for (int v = 0; v < VPR; ++v) {
              const uint32_t w[4] = {res[v].x, res[v].y, res[v].z, res[v].w};
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const float2 f = bf16x2_to_float2(w[j]);
                acc[v * 8 + 2 * j] += f.x;
                acc[v * 8 + 2 * j + 1] += f.y;
              }
            }
            if (rd + 1 < ROUNDS) fetch_res(col_of(rd + 1));
          }
          if (!LEAN && !BARE && g.out2 && row_ok) {
            // The redundant copy of a producer with consumers of different reduction dimensions: the same values with the
            // row's position inside its group as the contiguous dimension.  A warp's 32 rows write 64 contiguous bytes per column.
#pragma unroll
            for (int j = 0; j < RC; ++j)
              if (n0 + c0 + j < g.N) g.out2[o2_base + (long long)(n0 + c0 + j) * g.fd_out2_S.d] = __float2bfloat16_rn(acc[j]);
          }
          uint4 pk_prev = make_uint4(0, 0, 0, 0);
#pragma unroll
          for (int v = 0; v < VPR; ++v) {
            uint4 pk;
            pk.x = float2_to_bf16x2(acc[v * 8 + 0], acc[v * 8 + 1]);
            pk.y = float2_to_bf16x2(acc[v * 8 + 2], acc[v * 8 + 3]);
            pk.z = float2_to_bf16x2(acc[v * 8 + 4], acc[v * 8 + 5]);
            pk.w = float2_to_bf16x2(acc[v * 8 + 6], acc[v * 8 + 7]);
            if constexpr (DIRECT) {
              // 64 contiguous bytes of the thread's own row per round, as two 32-byte stores: whole sectors, and the
              // shared memory (whose bandwidth the operands need) is left to the ring, which gets six stages
              if (LEAN && g.tma_out) {
                // lean epilogue: the warp's 32 x 32 box goes through its own 2 KB of shared memory and leaves as one TMA
                // store -- a row-per-thread store touches 32 lines per instruction, and those stores and the next tile's
                // operand loads were in each other's way
                if (v == 0) {
                  if (lane == 0) ptx::bulk_wait_group_read<0>();     // the previous round's box has been read
                  __syncwarp();
                }
                *reinterpret_cast<uint4*>(cstage + e * CBOX_BYTES + lane * 64 + ((v ^ ((lane >> 1) & 3)) << 4)) = pk;
                if (v == VPR - 1) {
                  ptx::fence_proxy_async();
                  __syncwarp();
                  if (lane == 0 && (int)tile_m * BM + q * 32 < g.M) {
                    ptx::tma_store_2d(&tmC, cstage + e * CBOX_BYTES, n0 + c0, (int)tile_m * BM + q * 32);
                    ptx::bulk_commit_group();
                  }
                }
              } else if (v & 1) {
                if (row_ok && n0 + c0 + v * 8 < g.N) ptx::st_global_v8(out_t + off + n0 + c0 + (v - 1) * 8, pk_prev, pk);
              } else {
                pk_prev = pk;
              }
            } else if constexpr (QTMA) {
              const int c = c0 + v * 8;
              *reinterpret_cast<uint4*>(ROWS ? qline + c * 2 : qtile + (c >> 6) * 4096 + lane * 128 + ((((c & 63) >> 3) ^ (lane & 7)) << 4)) = pk;
            } else if constexpr (QSTAGE) *reinterpret_cast<uint4*>(qstage + lane * QROW + (c0 + v * 8) * 2) = pk;
            else *reinterpret_cast<uint4*>(stage + lane * STG_ROW + v * 16) = pk;
          }
          if constexpr (!QSTAGE && !DIRECT) {
            __syncwarp();
#pragma unroll
            for (int i = 0; i < VPR; ++i) {
              const int v = lane + 32 * i;
              const int rr = v / VPR, seg = v - rr * VPR;
              const long long roff = __shfl_sync(0xFFFFFFFFu, off, rr);
              const int rok = __shfl_sync(0xFFFFFFFFu, (int)row_ok, rr);
              const uint4 pk = *reinterpret_cast<const uint4*>(stage + rr * STG_ROW + seg * 16);
              if (rok && n0 + c0 + seg * 8 + 8 <= g.N) *reinterpret_cast<uint4*>(out_t + roff + n0 + c0 + seg * 8) = pk;
            }
            __syncwarp();
          }
        }
      }
      // all of this warp's TMEM reads of the buffer have completed (wait::ld above)
      if constexpr (!EARLY) {
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if constexpr (PAIR) ptx::mbar_arrive_cluster(tmem_empty0 + buf * 8);
          else ptx::mbar_arrive(&tmem_empty[buf]);
        }
      }
      if constexpr (QTMA) {
        // Very short reductions (batched q k^T): the tile's store is all there is, and with one staging tile the store path
        // idled while the next tile was converted.  Two tiles, and a warp sends one 32 x 64 box of its quadrant (rows and
        // columns past the edge are clipped): 8 x 16 heads, 1024 x 1024 scores of 64: 72.2 -> 55.7 us in a short stream of calls, 73.4 ->
        // 62.8 in a long one.
        ptx::fence_proxy_async();
        asm volatile("bar.sync %0, 128;" ::"r"(1 + q) : "memory");
        if constexpr (ROWS) {                                // (the lanes that wait for their copies: groups are a thread's own)
          if (lane < 8) {
            const int tr = q * 32 + grp * 8 + lane, orow = (int)tile_m * BM + tr;
            if (orow < g.M)
              ptx::bulk_store(g.out + (long long)batch * g.out_batch_stride + (long long)orow * g.ldc + n0, cstage + stage_row_off(tr, it & 1),
                              (uint32_t)min(g.N - n0, BN) * 2u);
            ptx::bulk_commit_group();
          }
        } else if (lane == 0) {
          if ((int)tile_m * BM + q * 32 < g.M && n0 + grp * 64 < g.N)
            ptx::tma_store_3d(&tmC, qtile + grp * 4096, n0 + grp * 64, (int)tile_m * BM + q * 32, (int)batch);
          ptx::bulk_commit_group();
        }
      } else if constexpr (QSTAGE && QBULK) {
        // the four warps of the quadrant have filled a 32 x 256 staging tile: every 512-byte row leaves as one bulk copy
        // (shared memory -> global), eight rows per warp, so no thread spends instructions on moving the tile.  Measured:
        // the batched q k^T GEMM 78.4 -> 72.6 us; on 192-byte rows (the 96-wide scatter GEMM) the same was slower, 22.3 vs
        // 20.7 us, so narrower tiles keep the vector loop below.
        ptx::fence_proxy_async();
        asm volatile("bar.sync %0, 128;" ::"r"(1 + q) : "memory");
        const int rr = grp * 8 + (lane & 7);
        const long long roff = __shfl_sync(0xFFFFFFFFu, off, rr);
        const int rok = __shfl_sync(0xFFFFFFFFu, (int)row_ok, rr);
        const int ncols = g.N - n0 < BN ? g.N - n0 : BN;
        if (lane < 8) {
          if (rok) ptx::bulk_store(out_t + roff + n0, qstage + rr * QROW, (uint32_t)ncols * 2u);
          ptx::bulk_commit_group();
        }
      } else if constexpr (QSTAGE) {
        // the four warps of the quadrant have filled a 32 x BN staging tile: store whole rows
        constexpr int VR = BN / 8;                           // 16-byte vectors per row
        asm volatile("bar.sync %0, 128;" ::"r"(1 + q) : "memory");
        const int tq = grp * 32 + lane;
#pragma unroll
        for (int i = 0; i < VR / 4; ++i) {
          const int v = tq + 128 * i;
          const int rr = v / VR, seg = v - rr * VR;
          const long long roff = __shfl_sync(0xFFFFFFFFu, off, rr);
          const int rok = __shfl_sync(0xFFFFFFFFu, (int)row_ok, rr);
          const uint4 pk = *reinterpret_cast<const uint4*>(qstage + rr * QROW + seg * 16);
          if (rok && n0 + seg * 8 + 8 <= g.N) *reinterpret_cast<uint4*>(out_t + roff + n0 + seg * 8) = pk;
        }
        asm volatile("bar.sync %0, 128;" ::"r"(1 + q) : "memory");
      }
    }
  }
  ptx::bulk_wait_group_read<0>();   // output boxes of the last tile have been read out of shared memory
  ptx::tc_fence_before();
  if constexpr (PAIR) {
    __syncwarp();
    ptx::cluster_sync();            // neither CTA leaves (or frees tensor memory) while the other may still read or signal it
  } else {
    __syncthreads();
  }
  if (warp == 1) {
    ptx::tc_fence_after();
    if constexpr (PAIR) ptx::tmem_dealloc_pair(tmem_base, TMEM_COLS);
    else ptx::tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------------------
// Host side: tensor maps.
// ---------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// Encoded maps by what they were encoded from; a call looks up three to seven of them, so the key is a flat array of words
// compared and hashed without an allocation.
struct TmKey {
  uint64_t w[12];
  bool operator==(const TmKey& o) const { return memcmp(w, o.w, sizeof(w)) == 0; }
};
struct TmHash {
  size_t operator()(const TmKey& k) const {
    uint64_t h = 0x9E3779B97F4A7C15ull;
    for (uint64_t v : k.w) h = (h ^ v) * 0xBF58476D1CE4E5B9ull, h ^= h >> 29;
    return (size_t)h;
  }
};
std::mutex g_tm_mu;
std::unordered_map<TmKey, CUtensorMap, TmHash> g_tm_cache;

int encode_cached(const void* ptr, int rank, const uint64_t* dims, const uint64_t* strides_b, const uint32_t* box,
                  CUtensorMap* out, int swizzle_bytes = 128) {
  TmKey key;
  memset(&key, 0, sizeof(key));
  key.w[0] = (uint64_t)(uintptr_t)ptr;
  key.w[1] = ((uint64_t)rank << 16) | (uint64_t)swizzle_bytes;
  for (int i = 0; i < rank; ++i) {
    key.w[2 + i] = dims[i];
    if (i < rank - 1) key.w[7 + i] = strides_b[i];
    key.w[11] = key.w[11] << 10 | box[i];            // (a box has at most 256 elements a side)
  }
  {
    std::lock_guard<std::mutex> lk(g_tm_mu);
    auto it = g_tm_cache.find(key);
    if (it != g_tm_cache.end()) {
      *out = it->second;
      return SMARTMEM_OK;
    }
  }
  EncodeTiledFn enc = get_encode();
  if (!enc) return SMARTMEM_ERR_CUDA;
  cuuint64_t d[5], s[4];
  cuuint32_t b[5], es[5];
  for (int i = 0; i < rank; ++i) {
    d[i] = dims[i];
    b[i] = box[i];
    es[i] = 1;
    if (i < rank - 1) s[i] = strides_b[i];
  }
  CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(ptr), d, s, b, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_bytes == 0 ? CU_TENSOR_MAP_SWIZZLE_NONE :
                   swizzle_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return SMARTMEM_ERR_CUDA;
  std::lock_guard<std::mutex> lk(g_tm_mu);
  if (g_tm_cache.size() > 4096) g_tm_cache.clear();
  g_tm_cache[key] = *out;
  return SMARTMEM_OK;
}

// Turns an operand description into a tensor map + the coordinate rule of the kernel.
// `box_rows` rows per copy (a CTA pair fetches a tile of `tile_rows` rows as two boxes, one per CTA).
int build_operand(const TcOperand& op, int tile_rows, int box_rows, CUtensorMap* tm, OpCoord* oc) {
  if (op.n_row_atoms < 1 || op.n_row_atoms + op.n_batch_atoms > 4) return SMARTMEM_ERR_UNSUPPORTED;
  if (((uintptr_t)op.ptr & 15) != 0) return SMARTMEM_ERR_ALIGNMENT;
  const int nr = op.n_row_atoms, nb = op.n_batch_atoms;
  const long long in_ext = op.row_extent[nr - 1], in_str = op.row_stride[nr - 1];
  const bool mn = op.k_stride != 1;
  if (mn && in_str != 1) return SMARTMEM_ERR_UNSUPPORTED;
  if (nr > 1 && in_ext % tile_rows) return SMARTMEM_ERR_UNSUPPORTED;
  uint64_t dims[5], strides[4];
  uint32_t box[5];
  int rank = 0;
  auto push = [&](long long ext, long long str_elems, uint32_t bx) -> bool {
    if (rank > 0) {
      if ((str_elems * 2) % 16 || str_elems <= 0) return false;
      strides[rank - 1] = (uint64_t)str_elems * 2;
    }
    dims[rank] = (uint64_t)ext;
    box[rank] = bx;
    ++rank;
    return true;
  };
  bool ok = true;
  if (!mn) {
    ok = ok && push(op.K, 1, BK) && push(in_ext, in_str, (uint32_t)box_rows);
  } else {
    ok = ok && push(in_ext, 1, 64) && push(op.K, op.k_stride, BK);
  }
  memset(oc, 0, sizeof(*oc));
  for (int i = nr - 2; i >= 0 && ok; --i) {
    ok = push(op.row_extent[i], op.row_stride[i], 1);
    oc->outer[oc->n_outer++] = make_fastdiv((uint32_t)op.row_extent[i]);
    oc->n_outer_row++;
  }
  for (int i = nb - 1; i >= 0 && ok; --i) {
    ok = push(op.batch_extent[i], op.batch_stride[i], 1);
    oc->outer[oc->n_outer++] = make_fastdiv((uint32_t)op.batch_extent[i]);
  }
  if (!ok) return SMARTMEM_ERR_UNSUPPORTED;
  if (rank < 2) return SMARTMEM_ERR_UNSUPPORTED;
  while (rank < 5) {                                   // pad: all kernels issue 5-D loads
    strides[rank - 1] = strides[rank - 2] * dims[rank - 1];
    if (strides[rank - 1] >= (1ull << 40)) strides[rank - 1] = strides[rank - 2];
    dims[rank] = 1;
    box[rank] = 1;
    ++rank;
  }
  oc->rank = rank;
  oc->mn_major = mn ? 1 : 0;
  oc->tiles_inner = make_fastdiv((uint32_t)((in_ext + tile_rows - 1) / tile_rows));
  return encode_cached(op.ptr, rank, dims, strides, box, tm);
}

// every offset the map can produce is a multiple of `q` elements
bool devmap_offsets_multiple_of(const DevMap& m, long long q) {
  if (m.base % q) return false;
  for (int a = 0; a < m.n_atoms; ++a)
    if (m.roll_of[a] < 0 && m.stride[a] % q) return false;
  for (int r = 0; r < m.n_rolls; ++r) {
    if (m.roll_stride[r] % q) return false;
    for (int i = 0; i < m.roll_n_parts[r] && m.roll_n_parts[r] > 1; ++i)
      if (m.roll_part_stride[r][i] % q) return false;
  }
  return true;
}

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 148;
  }
  return n;
}

template <int BN, int STAGES, bool A_MN, bool PAIR = false, bool LEAN = false, bool ROWS = false>
int launch_t(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& tc, const Halves<true>& halves, const GemmArgs& g, cudaStream_t st) {
  constexpr bool QST = !PAIR && !(BN == 256 && STAGES == 4);
  constexpr int RCc = !QST ? 16 : ((BN / 4) > 32 ? 32 : (BN / 4));
  constexpr size_t smem = 1024 + STAGES * (A_STAGE_BYTES + (PAIR ? BN / 2 : BN) * BK * 2) + (2 * STAGES + 4) * 8 + 16 +
                          (LEAN ? kEpiWarps * 32 * 64 : PAIR ? 0 : STAGES == 2 ? kStageBytes : !QST ? kEpiWarps * 32 * (RCc * 2 + 16) : 4 * 32 * (BN * 2 + 16));   // pairs store from registers
  if (ensure_max_dynamic_smem((const void*)gemm_tc_kernel<BN, STAGES, A_MN, PAIR, LEAN, ROWS>, (int)smem) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("gemm_tc", st);
  long long tiles = (long long)g.tiles_n * g.tiles_m * g.batch;
  Halves<PAIR && BN == 256> hv;
  if constexpr (PAIR && BN == 256) {
    hv = halves;
    tiles = 2 * tiles - halves.wide_tiles;
  }
  if constexpr (PAIR) {
    // one cluster of two CTAs per tile of 256 rows; the two CTAs of a cluster are neighbours in blockIdx.x
    const long long pairs = sm_count() / 2;
    const unsigned grid = (unsigned)(2 * (tiles < pairs ? tiles : pairs));
    launch_pdl_cluster(gemm_tc_kernel<BN, STAGES, A_MN, PAIR, LEAN, ROWS>, dim3(grid), dim3(kThreads), smem, st, 2u, ta, tb, tc, g, hv);
  } else {
    const unsigned grid = (unsigned)(tiles < sm_count() ? tiles : sm_count());
    launch_pdl(gemm_tc_kernel<BN, STAGES, A_MN, PAIR, LEAN, ROWS>, dim3(grid), dim3(kThreads), smem, st, ta, tb, tc, g, hv);
  }
  count_launch();
  return cudaGetLastError() == cudaSuccess ? SMARTMEM_OK : SMARTMEM_ERR_CUDA;
}

}  // namespace

int tc_encode_2d(const void* ptr, long long inner, long long outer, long long pitch_elems, int box_inner, int box_outer,
                 CUtensorMap* out) {
  if (((uintptr_t)ptr & 15) || (pitch_elems * 2) % 16) return SMARTMEM_ERR_ALIGNMENT;
  const uint64_t dims[2] = {(uint64_t)inner, (uint64_t)outer};
  const uint64_t strides[1] = {(uint64_t)pitch_elems * 2};
  const uint32_t box[2] = {(uint32_t)box_inner, (uint32_t)box_outer};
  return encode_cached(ptr, 2, dims, strides, box, out);
}

int tc_encode_2d_sw64(const void* ptr, long long inner, long long outer, long long pitch_elems, int box_inner,
                      int box_outer, CUtensorMap* out) {
  if (((uintptr_t)ptr & 15) || (pitch_elems * 2) % 16 || box_inner * 2 != 64) return SMARTMEM_ERR_ALIGNMENT;
  const uint64_t dims[2] = {(uint64_t)inner, (uint64_t)outer};
  const uint64_t strides[1] = {(uint64_t)pitch_elems * 2};
  const uint32_t box[2] = {(uint32_t)box_inner, (uint32_t)box_outer};
  return encode_cached(ptr, 2, dims, strides, box, out, 64);
}

int tc_encode_2d_plain(const void* ptr, long long inner, long long outer, long long pitch_elems, int box_inner, int box_outer,
                       CUtensorMap* out) {
  if (((uintptr_t)ptr & 15) || (pitch_elems * 2) % 16) return SMARTMEM_ERR_ALIGNMENT;
  const uint64_t dims[2] = {(uint64_t)inner, (uint64_t)outer};
  const uint64_t strides[1] = {(uint64_t)pitch_elems * 2};
  const uint32_t box[2] = {(uint32_t)box_inner, (uint32_t)box_outer};
  return encode_cached(ptr, 2, dims, strides, box, out, 0);
}

static int encode_nd(const void* ptr, int rank, const long long* dims, const long long* strides_elems, const int* box, int swizzle_bytes,
                     CUtensorMap* out) {
  if (rank < 2 || rank > 5 || ((uintptr_t)ptr & 15) || box[0] * 2 != swizzle_bytes) return SMARTMEM_ERR_ALIGNMENT;
  uint64_t d[5], sb[4];
  uint32_t b[5];
  for (int i = 0; i < rank; ++i) {
    d[i] = (uint64_t)dims[i];
    b[i] = (uint32_t)box[i];
    if (i > 0) {
      sb[i - 1] = (uint64_t)strides_elems[i - 1] * 2;
      if (sb[i - 1] % 16) return SMARTMEM_ERR_ALIGNMENT;
    }
  }
  return encode_cached(ptr, rank, d, sb, b, out, swizzle_bytes);
}
int tc_encode_nd_sw64(const void* ptr, int rank, const long long* dims, const long long* strides_elems, const int* box,
                      CUtensorMap* out) {
  return encode_nd(ptr, rank, dims, strides_elems, box, 64, out);
}
int tc_encode_nd_sw128(const void* ptr, int rank, const long long* dims, const long long* strides_elems, const int* box,
                       CUtensorMap* out) {
  return encode_nd(ptr, rank, dims, strides_elems, box, 128, out);
}

int tc_encode_2d_blocks(const void* ptr, long long inner, long long outer, long long blocks, long long rows, CUtensorMap* out) {
  const long long dims[3] = {BK, outer, inner / BK}, strides[2] = {inner, BK};
  const int box[3] = {BK, (int)rows, (int)blocks};
  return tc_encode_nd_sw128(ptr, 3, dims, strides, box, out);
}

int tc_sm_count() { return sm_count(); }

namespace {
constexpr int kProbeSmem = 120 * 1024;                   // (two of them do not fit an SM)
__global__ void cluster_probe_kernel() {}                // never launched: asked for its occupancy
constexpr int kMaxDevices = 64, kMaxCluster = 8;
std::mutex g_cluster_mu;
int g_cluster_ctas[kMaxDevices][kMaxCluster + 1];        // 0: not asked yet
}  // namespace

// How the SMs are dealt out to GPCs differs from board to board, so the device is asked, once per size.  (One with 148 SMs said 148, 148,
// 135, 132, 130, 132, 105 and 120 for sizes 1 to 8; what stands in where there is no device to ask, for the host-only calls.)
int tc_cluster_ctas(int size) {
  static const int typical[kMaxCluster + 1] = {0, 148, 148, 135, 132, 130, 132, 105, 120};
  const int guess = typical[size] * sm_count() / 148;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return guess;
  std::lock_guard<std::mutex> lk(g_cluster_mu);
  int& known = g_cluster_ctas[dev][size];
  if (known) return known;
  if (ensure_max_dynamic_smem((const void*)cluster_probe_kernel, kProbeSmem) != SMARTMEM_OK) return guess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)size);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = kProbeSmem;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)size;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, cluster_probe_kernel, &cfg) != cudaSuccess || clusters < 1) {
    cudaGetLastError();                                  // (nothing was launched: the guess serves)
    return guess;
  }
  return known = clusters * size;
}

ClusterCtas tc_cluster_ctas_all() {
  static_assert(kMaxClusterSize == kMaxCluster, "one table");
  static thread_local int table_dev = -1;
  static thread_local ClusterCtas table;
  int dev = -1;
  if (cudaGetDevice(&dev) == cudaSuccess && dev == table_dev) return table;
  ClusterCtas t;
  t.n[0] = 0;
  for (int s = 1; s <= kMaxCluster; ++s) t.n[s] = tc_cluster_ctas(s);
  if (dev < 0 || dev >= kMaxDevices) return t;
  std::lock_guard<std::mutex> lk(g_cluster_mu);
  for (int s = 1; s <= kMaxCluster; ++s)
    if (g_cluster_ctas[dev][s] == 0) return t;           // (a guess: asked again next time)
  table = t;
  table_dev = dev;
  return t;
}

int tc_operand_from_map(const smartmem_index_map_t& m, int n_batch_atoms, int n_row_atoms, const void* ptr,
                        TcOperand* op) {
  if (m.klass == 3 || m.n_rolls > 0) return SMARTMEM_ERR_UNSUPPORTED;
  const int nk = m.n_atoms - n_batch_atoms - n_row_atoms;
  if (nk != 1 || n_row_atoms < 0 || n_row_atoms > 3 || n_batch_atoms > 3) return SMARTMEM_ERR_UNSUPPORTED;
  memset(op, 0, sizeof(*op));
  op->ptr = (const char*)ptr + m.base * 2;
  op->n_batch_atoms = n_batch_atoms;
  op->n_row_atoms = n_row_atoms;
  for (int i = 0; i < n_batch_atoms; ++i) {
    op->batch_extent[i] = m.extent[i];
    op->batch_stride[i] = m.src_stride[i];
  }
  for (int i = 0; i < n_row_atoms; ++i) {
    op->row_extent[i] = m.extent[n_batch_atoms + i];
    op->row_stride[i] = m.src_stride[n_batch_atoms + i];
  }
  op->K = m.extent[m.n_atoms - 1];
  op->k_stride = m.src_stride[m.n_atoms - 1];
  if (n_row_atoms == 0) {                              // one row: the map has no atom for it
    op->n_row_atoms = 1;
    op->row_extent[0] = 1;
    op->row_stride[0] = (op->K + 7) / 8 * 8;
  }
  return SMARTMEM_OK;
}

TcOperand tc_operand_plain(const void* ptr, long long rows, long long K, long long ld) {
  TcOperand op;
  memset(&op, 0, sizeof(op));
  op.ptr = ptr;
  op.n_row_atoms = 1;
  op.row_extent[0] = rows;
  op.row_stride[0] = ld;
  op.K = K;
  op.k_stride = 1;
  return op;
}

// The last round of 256-wide pair tiles in halves: where it is not the first and the halves still make one round.  Measured (us, whole
// tiles -> halves): M = 435, K = 4096, N = 12288 (96 tiles on 74 pairs) 46.3 -> 42.2, M = 1268 (240) 108.8 -> 99.3, M = 2048 (384) 159.4 ->
// 153.7; M = 12544, K = 512, N = 2048 (392) 24.2 -> 23.1; M = 20000, K = 512, N = 1024 21.3 -> 20.0.
static bool tail_halves(long long tiles, long long pairs) { return tiles > pairs && tiles % pairs != 0 && 2 * (tiles % pairs) <= pairs; }

// Whether the two-stage kernel's output leaves as rows of 512 bytes or as boxes of 32 x 64.  A box's rows of 128 bytes touch two lines each where
// the output's rows are not whole lines, and where those are not whole sectors of 32 bytes either, L2 holds half-written sectors until the
// neighbouring box comes: boxes then lose as soon as the stores are what a tile takes, that is where the tiles are full or the output is larger
// than L2.  Us, boxes -> rows, K = 64, B x heads x S: 128 x 1000 59.6 -> 54.7, 128 x 968 60.7 -> 52.4, 128 x 776 44.2 -> 42.4, 32 x 1288 30.6 -> 29.2,
// 30 x 1000 16.5 -> 16.1; but 128 x 616 24.9 -> 25.4, 30 x 712 9.9 -> 11.0, and in whole sectors 128 x 992 48.5 -> 53.4, 30 x 1024 15.2 -> 16.8.
// Two k-blocks (K = 128) keep the ring of two stages from running ahead, and rows, which are one copy where boxes are two lines a row, are the better
// from four tiles an SM on: 128 x 1000 78.1 -> 71.5, 128 x 1024 75.1 -> 71.7, 33 x 768 14.9 -> 14.3; 30 x 512 6.8 -> 7.4, 30 x 648 12.4 -> 12.5.
static bool store_rows(long long tiles, long long batch, long long M, long long N, int nkb) {
  if (nkb == 2) return tiles >= 4ll * tc_sm_count();
  const double bytes = 2.0 * (double)(batch * M) * (double)N;
  return N % 16 != 0 && bytes / ((double)tiles * kStageBoxBytes) + bytes / 4e8 > 1.02;
}

int launch_gemm_tc(const TcOperand& A, const TcOperand& B, const TcEpilogue& ep, long long batch, long long M,
                   long long N, long long K, cudaStream_t st) {
  if (M < 1 || N < 1 || K < 1 || batch < 1 ||  M >= (1ll << 31) || N >= (1ll << 31))
    return SMARTMEM_ERR_UNSUPPORTED;
  if (A.K != K || B.K != K) return SMARTMEM_ERR_SHAPE;
  if (((uintptr_t)ep.out & 15) || ((uintptr_t)ep.residual & 15) || ((uintptr_t)ep.bias & 15) || ep.ldc % 8 ||
      ep.out_batch_stride % 8)
    return SMARTMEM_ERR_ALIGNMENT;
  if (N % 8) return SMARTMEM_ERR_UNSUPPORTED;
  const bool a_mn = A.k_stride != 1;
  if (B.k_stride != 1) return SMARTMEM_ERR_UNSUPPORTED;
  const bool splitk_ok = gemm_splitk_supported(A, B, ep, batch, M, N, K);
  if (ep.rms_gamma) return splitk_ok ? launch_gemm_splitk(A, B, ep, M, N, K, st) : SMARTMEM_ERR_UNSUPPORTED;
  if (ep.rope_cols > 0 && (N % 256 || ep.rope_cols % 256 || ep.rope_S < 1 || a_mn || ep.bias || ep.gelu || ep.residual || ep.out2)) return SMARTMEM_ERR_UNSUPPORTED;
  if (ep.rope_cols > 0 && ep.rope_dim != 0 && ep.rope_dim != 32 && ep.rope_dim != 64 && ep.rope_dim != 128) return SMARTMEM_ERR_UNSUPPORTED;
  if (ep.seg_cols > 0) {
    if (ep.seg_cols % 256 || N > 3ll * ep.seg_cols || ep.rowmap || ep.residual || batch != 1) return SMARTMEM_ERR_UNSUPPORTED;
    for (int i = 0; i * (long long)ep.seg_cols < N; ++i)
      if (!ep.seg_out[i] || ((uintptr_t)ep.seg_out[i] & 15) || ep.seg_ld[i] % 8) return SMARTMEM_ERR_ALIGNMENT;
  }
  const int nkb = (int)((K + BK - 1) / BK);
  const long long tiles_m1 = (M + BM - 1) / BM;
  // CTA pairs (two SMs on one tile of 256 rows): their epilogue writes 32-byte vectors.
  // SMARTMEM_GEMM_PAIR=0 keeps every GEMM on single CTAs (for measuring what pairing buys).
  static const int allow_pair = [] { const char* e = getenv("SMARTMEM_GEMM_PAIR"); return (e && e[0] == '0') ? 0 : 1; }();
  const bool pair_ok = allow_pair && !a_mn && tiles_m1 > 1 && nkb > 4 && N % 256 == 0 && A.n_row_atoms == 1 &&
                       (!ep.rowmap || devmap_offsets_multiple_of(*ep.rowmap, 16)) && ep.seg_cols == 0 && !ep.out2 && ep.ldc % 16 == 0 &&
                       ep.out_batch_stride % 16 == 0 && ((uintptr_t)ep.out & 31) == 0;
  // the lean epilogue on single CTAs: whole rows as TMA boxes, or (128 wide) 32-byte vectors through the row map
  const bool lean_ok = !a_mn && batch == 1 && ep.rope_cols == 0 && ep.seg_cols == 0 && !ep.out2;
  const bool lean256_ok = lean_ok && !ep.rowmap && !ep.residual;
  const bool lean128_ok = lean_ok && (lean256_ok || (N % 16 == 0 && ep.ldc % 16 == 0 && ((uintptr_t)ep.out & 31) == 0 && ((uintptr_t)ep.residual & 31) == 0 &&
                                                      (!ep.rowmap || devmap_offsets_multiple_of(*ep.rowmap, 16))));
  int bn = 128;
  bool pair = false, lean = false, halves = false;
  if (batch == 1) {
    // Tile width, and single CTAs or pairs: the smallest of the times fitted to measurements (us): a fixed part, the k-blocks of
    // the first tile, and for every further wave its k-blocks or, where the reduction is short, its epilogue.  A narrow tile
    // costs more per column but splits the columns over more SMs: M = 666, N = K = 2048 (48 tiles of 128 x 256, 96 of half
    // that) 16.1 us on 256-wide single tiles, 9.6 on 128-wide pairs; M = 196, N = 512, K = 2048 14.1 -> 8.8 us on 64-wide ones.
    // With many waves, narrow pair tiles pay for the operand they read twice: M = 16384, N = 512, K = 1024 17.1 us on four waves of
    // 128-wide pairs, 16.2 on two of 256; M = 12544, K = 2048 23.3 on three, 24.8 on two.
    struct Option { int bn; bool pair, lean; double fixed, per_kb, wave, wave_min; };
    static const Option options[] = {{64, false, false, 2.4, 0.185, 0.55, 0.95}, {96, false, false, 2.9, 0.22, 0.8, 1.2},
                                     {128, false, true, 2.6, 0.26, 0.7, 1.15},   {256, false, true, 3.9, 0.5, -0.2, 1.65},
                                     {128, false, false, 2.6, 0.27, 0.4, 2.8},   {256, false, false, 4.4, 0.36, 0.5, 4.0},
                                     {128, true, false, 3.0, 0.185, 0.6, 2.2},   {256, true, false, 5.4, 0.33, 0.4, 3.0}};
    double best = 0.0;
    for (const Option& o : options) {
      if (o.pair && !pair_ok) continue;
      if (o.lean && !(o.bn == 128 ? lean128_ok : lean256_ok)) continue;
      if (ep.rope_cols > 0 && o.bn < 128) continue;          // rotary pairs stay inside a tile
      if (a_mn && o.bn < 128) continue;                      // MN-major A operands come with 128- and 256-wide tiles only
      if (ep.seg_cols > 0 && ep.seg_cols % o.bn) continue;
      if (B.n_row_atoms > 1 && B.row_extent[B.n_row_atoms - 1] % o.bn) continue;
      const long long tiles = (o.pair ? (tiles_m1 + 1) / 2 : tiles_m1) * ((N + o.bn - 1) / o.bn), slots = tc_sm_count() / (o.pair ? 2 : 1);
      // (64-wide tiles fall behind on long reductions: 161 x 4096 -> 4096 16.4 us on 128 CTAs, 14.9 on as many in 128-wide pairs)
      const double kbs = nkb * o.per_kb + (o.bn == 64 && nkb > 32 ? (nkb - 32) * 0.035 : 0.0), wave = kbs + o.wave > o.wave_min ? kbs + o.wave : o.wave_min;
      double t = o.fixed + kbs + (double)((tiles + slots - 1) / slots - 1) * wave;
      const bool tail = o.pair && o.bn == 256 && tail_halves(tiles, slots);
      if (tail) t -= 0.44 * wave;
      if (best == 0.0 || t < best) { best = t; bn = o.bn; pair = o.pair; lean = o.lean; halves = tail; }
    }
    if (splitk_ok && gemm_splitk_us(M, N, K) < best) return launch_gemm_splitk(A, B, ep, M, N, K, st);
  } else {
    // batched: the widest of {256, 128, 96, 64} that divides N (fewest wasted columns), else 128; 256 or 128, whichever leaves
    // fewer idle SMs in the last wave (time of a wave ~ tile width plus a fixed part), for short reductions only: a 128-wide tile
    // reads as many operand bytes per product as shared memory delivers, so over a long K the wider tile wins even with a
    // ragged last wave (measured at K = 2048)
    // Short reductions are bound by their stores, which the wide tile makes in whole rows, so it takes them whatever N is (128 heads,
    // 1000 x 1000 scores of 64: 89 us in 128-wide tiles, 58 in 256; 704 x 704 55 in 64-wide ones, 34), but for an N that 96-wide tiles fill
    // and 256-wide ones do not: one of those takes as long as 2.05 narrow ones (288 x 288: 10.2 us in three, 14.3 in two; 576 x 576 with
    // 24 heads 7.8 in six, 9.3 in three; 960 x 960 71 in ten, 55 in four).
    const long long wide = (N + 255) / 256;
    const bool fill96 = N % 128 && N % 96 == 0 && 100 * (N / 96) < 205 * wide;
    if (ep.rope_cols > 0) bn = 256;
    else if (nkb <= 2 && N >= 192 && !a_mn && !fill96 && tiles_m1 * batch * wide >= tc_sm_count()) bn = 256;
    else if (N % 256 == 0) {
      const long long tm = tiles_m1 * batch, sms = tc_sm_count();
      const long long w256 = (tm * (N / 256) + sms - 1) / sms, w128 = (tm * (N / 128) + sms - 1) / sms;
      bn = (K <= 1024 && w128 * (128 + 48) < w256 * (256 + 48)) ? 128 : 256;
    } else if (N % 128 == 0) bn = 128;
    else if (N % 96 == 0) bn = 96;
    else if (N % 64 == 0) bn = 64;
    if (a_mn && bn < 128) bn = 128;
    // pairs where the row tiles pair up and there is more than one wave of work for the single-CTA kernel
    pair = pair_ok && bn >= 128 && tiles_m1 % 2 == 0 && tiles_m1 * (N / 256) * batch > tc_sm_count();
    if (pair) {
      const long long pairs = tc_sm_count() / 2, t256 = tiles_m1 / 2 * (N / 256) * batch;
      const long long w256 = (t256 + pairs - 1) / pairs, w128 = (2 * t256 + pairs - 1) / pairs;
      bn = (ep.rope_cols == 0 && w128 * (nkb * 0.21 + 1.2) < w256 * (nkb * 0.33 + 2.2)) ? 128 : 256;
    }
  }
  // single CTAs: 256 wide, short K: wider store rounds instead of a 4th stage.  Narrow tiles: their stages are
  // small, and a tile is consumed faster than a load's latency, so the ring runs several tiles ahead.
  const bool plain_out = !pair && !a_mn && !ep.rowmap && ep.seg_cols == 0 && !ep.out2 && !ep.bias && !ep.gelu && !ep.residual && ep.rope_cols == 0;
  int stages = bn == 256 ? (nkb <= 2 && plain_out ? 2 : nkb <= 4 ? 3 : 4) : bn == 64 ? 8 : bn == 96 ? 7 : 5;
  GemmArgs g;
  memset(&g, 0, sizeof(g));
  CUtensorMap ta, tb;
  int rc = build_operand(A, BM, BM, &ta, &g.ca);
  if (rc != SMARTMEM_OK) return rc;
  rc = build_operand(B, bn, pair ? bn / 2 : bn, &tb, &g.cb);
  if (rc != SMARTMEM_OK) return rc;
  g.M = (int)M; g.N = (int)N; g.K = (int)K;
  g.out = (__nv_bfloat16*)ep.out;
  g.ldc = ep.ldc;
  g.out_batch_stride = ep.out_batch_stride;
  g.bias = (const __nv_bfloat16*)ep.bias;
  g.residual = (const __nv_bfloat16*)ep.residual;
  g.gelu = ep.gelu;
  g.b_settled = ep.b_settled;
  g.has_rowmap = ep.rowmap ? 1 : 0;
  if (ep.rowmap) g.rowmap = *ep.rowmap;
  g.rope_cols = ep.rope_cols;
  g.rope_S = ep.rope_S;
  g.rope_pos0 = ep.rope_pos0;
  g.seg_cols = ep.seg_cols;
  for (int i = 0; i < 3; ++i) { g.seg_out[i] = (__nv_bfloat16*)ep.seg_out[i]; g.seg_ld[i] = ep.seg_ld[i]; }
  const int rope_dim = ep.rope_dim ? ep.rope_dim : 128;
  g.rope_half = rope_dim / 2;
  g.rope_c = ep.rope_log2_theta / (float)(rope_dim / 2);
  if (ep.out2) {
    if (ep.out2_S < 1 || M % ep.out2_S || batch != 1 || ((uintptr_t)ep.out2 & 1)) return SMARTMEM_ERR_UNSUPPORTED;
    g.out2 = (__nv_bfloat16*)ep.out2;
    g.fd_out2_S = make_fastdiv((uint32_t)ep.out2_S);
  }
  g.status = device_status_ptr();
  if (!g.status) return SMARTMEM_ERR_CUDA;
  g.tiles_n = (int)((N + bn - 1) / bn);
  g.tiles_m = (int)(pair ? (tiles_m1 + 1) / 2 : tiles_m1); // pairs walk over tiles of 256 rows
  g.fd_tiles_n = make_fastdiv((uint32_t)g.tiles_n);
  g.fd_tiles_m = make_fastdiv((uint32_t)g.tiles_m);
  g.batch = (int)batch;
  if ((long long)g.tiles_n * g.tiles_m * g.batch >= (1ll << 31)) return SMARTMEM_ERR_UNSUPPORTED;
  const long long all_tiles = (long long)g.tiles_n * g.tiles_m * g.batch;
  Halves<true> hv;
  hv.map = tb;
  hv.wide_tiles = (uint32_t)(halves ? all_tiles - all_tiles % (tc_sm_count() / 2) : all_tiles);
  if (halves) {
    OpCoord same;
    rc = build_operand(B, bn, bn / 4, &hv.map, &same);
    if (rc != SMARTMEM_OK) return rc;
  }
  CUtensorMap tc = ta;                                     // (a valid map for the kernels that store without TMA)
  const bool pair_lean = pair && bn == 256 && nkb <= 16 && ep.rope_cols == 0 && !ep.residual;
  if ((pair_lean || lean) && batch == 1 && !ep.rowmap) {     // output as 32 x 32 boxes of [M, N] with pitch ldc
    const uint64_t dims[2] = {(uint64_t)N, (uint64_t)M}, strides[1] = {(uint64_t)ep.ldc * 2};
    const uint32_t box[2] = {32, 32};
    if (encode_cached(ep.out, 2, dims, strides, box, &tc, 64) == SMARTMEM_OK) g.tma_out = 1;
    else if (lean) return SMARTMEM_ERR_CUDA;
    else tc = ta;
  }
  if (pair_lean) return launch_t<256, 6, false, true, true>(ta, tb, tc, hv, g, st);
  if (lean) return bn == 128 ? launch_t<128, 5, false, false, true>(ta, tb, tc, hv, g, st) : launch_t<256, 4, false, false, true>(ta, tb, tc, hv, g, st);
  if (pair && bn == 256) return launch_t<256, 6, false, true>(ta, tb, tc, hv, g, st);
  if (pair) return launch_t<128, 8, false, true>(ta, tb, tc, hv, g, st);
  if (stages == 2) {
    const uint64_t dims[3] = {(uint64_t)N, (uint64_t)M, (uint64_t)batch};
    const uint64_t strides[2] = {(uint64_t)ep.ldc * 2, (uint64_t)(batch > 1 ? ep.out_batch_stride : ep.ldc * M) * 2};
    const uint32_t box[3] = {64, 32, 1};
    if (store_rows(all_tiles, batch, M, N, nkb)) return launch_t<256, 2, false, false, false, true>(ta, tb, tc, hv, g, st);
    if (encode_cached(ep.out, 3, dims, strides, box, &tc) == SMARTMEM_OK) return launch_t<256, 2, false>(ta, tb, tc, hv, g, st);
    stages = 3;
  }
#define SM_CASE(BN_, ST_, MN_)                                                                  \
  if (bn == BN_ && stages == ST_ && a_mn == MN_) return launch_t<BN_, ST_, MN_>(ta, tb, tc, hv, g, st);
  SM_CASE(256, 3, false) SM_CASE(256, 4, false) SM_CASE(128, 5, false) SM_CASE(96, 7, false) SM_CASE(64, 8, false)
  SM_CASE(256, 3, true) SM_CASE(256, 4, true) SM_CASE(128, 5, true)
#undef SM_CASE
  return SMARTMEM_ERR_UNSUPPORTED;
}

}  // namespace smartmem
