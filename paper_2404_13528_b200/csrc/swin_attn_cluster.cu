// Attention half of a wide bf16 Swin block in one kernel, for blocks of few windows:
//   y = x + unshift(unpartition(proj(window_attention(qkv(LN1(partition(shift(x))))))))        C = 64 NV, NV = 2, 3, 4, 6 or 8, heads of 32
//
// Kernel by kernel this is three or four launches of one wave each (norm, QKV linear, window attention, projection), and what they cost
// is a launch, a dependency, a fill and a drain each, about 5 us, with 1-2 us of work in it.  The weights of a wide block do not fit one
// SM, so a cluster of NV CTAs shares a unit of two windows (2 x 64 rows, tokens past the window's end are zero) and each CTA takes
// two heads:
//   * every CTA gathers and normalises all rows of the unit (from L2: cheaper than exchanging them) straight into the QKV operand,
//     which meets its 192 rows of the QKV weights (32 of q, k and v of two heads) as they come in;
//   * per head, the 128 rows of two windows meet K0 and K1 in products that write the lanes of their own window only (so nothing of one
//     window, an infinity least of all, reaches the other), two threads have a row of the softmax, and P stays in tensor memory as the
//     operand of O = P V, lane by lane alike (as in attn_window_tc.cu, and with the same roundings);
//   * a CTA's O is one 64-column block of the projection's operand: it goes to every other CTA of the cluster as one bulk copy between
//     shared memories, into the memory of the normalised rows, and every CTA projects onto its 64 output columns, adds bias and residual
//     and scatters its 128-byte pieces of the rows through the map.
//
// What bounds it is the chain of phases.  Cycles of a unit at C = 192 / 512 (15 100 / 27 000 in all): rows 2200 / 3400, normalisation 2200 / 5600
// (issue slots, half of what the fp32 pipe needs for it), QKV product 2100 / 4900, conversion 1300, scores 450, softmax 1700, P V 500, O 450,
// exchange and projection 2900 / 7100 (20 bytes a clock and SM; with all CTAs sending to the lowest rank first it was 9300, and starting on
// the projection's blocks as they come is 500 to 1500 of it), output 1000.  Two threads a row in the softmax; with one it was 1500 on half the
// warps, and a bias table built word by word held q, k and v back by 1000.
//
// Warp roles: 0-15 rows, then q, k, v, softmax, O (four warps a head and half: 0-7 q, half of k and the lower keys, 8-15 the other half of k, v and
// the upper keys), output; 16 fetches weights and sends O; 17 owns the tensor memory and issues the products.
#include <cstring>

#include "attn.cuh"
#include "gemm_tc.cuh"
#include "ln_operand.cuh"
#include "ptx.cuh"
#include "tc_tiles.cuh"

namespace smartmem {
namespace {

constexpr int D = 32, TP = 64, HP = 2;                 // head dimension, token slots of a window, heads of a CTA
constexpr int kWorkers = 16, kThreads = 32 * (kWorkers + 2);
constexpr int W_ROWS = HP * 3 * D, W_STAGE = W_ROWS * 128;        // a k-block of the CTA's QKV weights: 24 KB
constexpr int P_ROWS = HP * D, P_BLOCK = P_ROWS * 128;            // a k-block of its rows of the projection's: 8 KB
constexpr int OP_BYTES = 128 * 64, OPS_BYTES = HP * 3 * OP_BYTES; // q, k, v of a head: 128 rows x 64 bytes each
constexpr int BIAS_ROW = 36;                           // 32-bit words per row of a bias table (attn_window_tc.cu)
// tensor memory: q, k, v of head h at 96 h, then P (32 columns: 64 keys as bf16 pairs) and O (32) in the place of q and v; S (64 a head);
// the projection
constexpr uint32_t TM_S = 192, TM_Y = 320, TMEM_COLS = 512;

struct AttnClusterArgs {
  const __nv_bfloat16 *x, *ln_g, *ln_b, *b_qkv, *b_proj;
  const uint16_t* table;
  __nv_bfloat16* y;
  int heads, T, ws, shift, n_windows, nWw, nWh, win_per_img, wide;
  FastDiv fd_wpi, fd_nww;
  float eps, scale;
  int* status;
  DevMap rowmap;
};

// Shared memory.  The QKV weights come through a ring of `stages` k-blocks, all of them up to NV = 4; q, k and v take its place once the
// products are done, and so does the projection's weight where there is no room for it beside (NV = 6, 8): `early` of its k-blocks behind
// q, k, v, the rest over them when they have been used.
template <int NV>
struct Plan {
  static constexpr int stages = NV <= 4 ? NV : NV == 6 ? 4 : 3;
  static constexpr int ring = stages * W_STAGE;
  static constexpr bool beside = NV <= 4;
  static constexpr int early = beside ? NV : (ring - OPS_BYTES) / P_BLOCK < NV ? (ring - OPS_BYTES) / P_BLOCK : NV;
  static_assert(ring >= OPS_BYTES && (NV - early) * P_BLOCK <= OPS_BYTES, "q, k, v and what is left of the projection's weight");
  static constexpr int off_ring = NV * kLnBlockBytes, off_wp = off_ring + (beside ? ring : OPS_BYTES);
  static constexpr int off_tab = off_ring + ring + (beside ? NV * P_BLOCK : 0);
  static constexpr int off_raw = off_tab + HP * TP * BIAS_ROW * 4;          // raw columns of the bias table
  static constexpr int off_ln = off_raw + HP * 256 * 2;                     // gamma, beta, biases of q, k, v (by head) and the projection
  static constexpr int off_offs = off_ln + (2 * 64 * NV + W_ROWS + P_ROWS) * 2;
  static constexpr int off_tyx = off_offs + 128 * 8;
  static constexpr int off_code = off_tyx + TP * 4 + 16;                     // a token's place in the bias table: differences index it
  static constexpr int off_red = off_code + TP * 4;                         // row maxima, then row sums, of the two halves of the keys
  static constexpr int off_bars = off_red + HP * 2 * 128 * 4;
  static constexpr int bytes = 1024 + off_bars + 36 * 8;
  static_assert(bytes <= 227 * 1024, "shared memory");
};

template <int NV>
__global__ void __launch_bounds__(kThreads, 1)
swin_attn_cluster_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmP, const __grid_constant__ AttnClusterArgs g) {
  using L = Plan<NV>;
  constexpr int C = 64 * NV;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sA = smem;                                  // [NV][128 rows x 128 B]: normalised rows, later O
  uint8_t* ring = smem + L::off_ring;
  uint8_t* ops = ring;                                 // [head][q, k, v][128 rows x 64 B]
  uint8_t* wp = smem + L::off_wp;
  uint32_t* bias_t = reinterpret_cast<uint32_t*>(smem + L::off_tab);        // [head][64][36]: bf16 pairs
  uint16_t* raw_s = reinterpret_cast<uint16_t*>(smem + L::off_raw);
  __nv_bfloat16* lng = reinterpret_cast<__nv_bfloat16*>(smem + L::off_ln);
  __nv_bfloat16 *lnb = lng + C, *bq = lnb + C, *bp = bq + W_ROWS;
  long long* offs = reinterpret_cast<long long*>(smem + L::off_offs);       // element offset of a row's token, -1: no token
  int* tyx = reinterpret_cast<int*>(smem + L::off_tyx);                     // [64]: ty << 8 | tx
  uint32_t* kmask = reinterpret_cast<uint32_t*>(tyx + TP);
  int* code = reinterpret_cast<int*>(smem + L::off_code);
  float* red = reinterpret_cast<float*>(smem + L::off_red);                 // [head][half][128]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::off_bars);
  uint64_t *w_full = bars, *w_empty = bars + 4, *a_ready = bars + 8, *qkv_full = bars + 9, *qk_ready = bars + 10, *v_ready = bars + 12, *s_full = bars + 14,
           *p_full = bars + 16, *o_full = bars + 18, *o_ready = bars + 20, *a_free = bars + 21, *wp_early = bars + 22, *wp_late = bars + 23, *y_full = bars + 24,
           *o_in = bars + 25;                          // [NV]: O of the CTA t ranks before this one (0: unused)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 34);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
  const int rank = (int)ptx::cluster_ctarank(), unit = (int)blockIdx.x / NV;
  const int T = g.T, ws = g.ws;

  if (warp == kWorkers) {
    if (ptx::elect_one()) {
      for (int i = 0; i < 4; ++i) {
        ptx::mbar_init(&w_full[i], 1);
        ptx::mbar_init(&w_empty[i], 1);
      }
      ptx::mbar_init(a_ready, kWorkers);
      ptx::mbar_init(qkv_full, 1);
      for (int i = 0; i < HP; ++i) {
        ptx::mbar_init(&qk_ready[i], 8);
        ptx::mbar_init(&v_ready[i], 4);
        ptx::mbar_init(&s_full[i], 1);
        ptx::mbar_init(&p_full[i], 8);
        ptx::mbar_init(&o_full[i], 1);
      }
      ptx::mbar_init(o_ready, kWorkers);
      ptx::mbar_init(a_free, NV);
      for (int t = 1; t < NV; ++t) ptx::mbar_init(&o_in[t], 1);
      ptx::mbar_init(wp_early, 1);
      ptx::mbar_init(wp_late, 1);
      ptx::mbar_init(y_full, 1);
      *abort_flag = 0;
      ptx::fence_barrier_init();
      ptx::fence_proxy_async();
      for (int t = 1; t < NV; ++t) ptx::mbar_expect_tx(&o_in[t], kLnBlockBytes);
    }
    __syncwarp();
  } else if (warp == kWorkers + 1) {
    ptx::tmem_alloc(tmem_slot, TMEM_COLS);
  } else {
    if (tid < 128) {                                   // row w * 64 + i: token i of window 2 unit + w
      const int n = 2 * unit + (tid >> 6), i = tid & 63;
      offs[tid] = i < T && n < g.n_windows ? devmap_eval(g.rowmap, (uint32_t)(n * T + i)) : -1;
    } else if (warp == 4) {
      // tokens, and the keys below / right of the wrap line of a seam window (bit c = key c)
      bool y[2], x[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int c = lane + 32 * k, ty = c / ws, tx = c - ty * ws;
        tyx[c] = ty << 8 | tx;
        code[c] = c < T ? ty * (2 * ws - 1) + tx : 0;
        y[k] = c < T && ty >= ws - g.shift;
        x[k] = c < T && tx >= ws - g.shift;
      }
      const uint32_t m0 = __ballot_sync(0xFFFFFFFFu, y[0]), m1 = __ballot_sync(0xFFFFFFFFu, y[1]);
      const uint32_t m2 = __ballot_sync(0xFFFFFFFFu, x[0]), m3 = __ballot_sync(0xFFFFFFFFu, x[1]);
      if (lane == 0) { kmask[0] = m0; kmask[1] = m1; kmask[2] = m2; kmask[3] = m3; }
    } else if (warp == 5) {
      if (lane < 2 * NV) ptx::prefetch_l2((lane < NV ? g.ln_g : g.ln_b - C) + lane * 64);
    } else if (warp < 6 + NV && ptx::elect_one()) {
      // the weights as far as L2: the kernel in front of this one may still be writing them.  (A warp each: one thread takes 0.15 us a copy.)
      ptx::tma_prefetch_4d(&tmW, (warp - 6) * 64, 0, 0, HP * rank);
      ptx::tma_prefetch_2d(&tmP, (warp - 6) * 64, rank * P_ROWS);
    }
  }
  ptx::tc_fence_before();
  __syncwarp();
  ptx::cluster_sync();                                 // the other CTAs' barriers are set up before anything of this one reaches them
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // Unwinding: whatever is in flight gets a fixed time to land.  The two warps below see to the copies and products that they have issued and,
  // the second one, to those that come in: no CTA of the cluster leaves before both of them have arrived.
  auto settle = [] {
    const unsigned long long t0 = ptx::globaltimer();
    while (ptx::globaltimer() - t0 < 100000ull) {
    }
  };

  // the projection takes the blocks of its operand in the order in which they come: its own, then those of the CTAs before it
  auto ring_block = [&](int t) { return t <= rank ? rank - t : rank - t + NV; };

  if (warp == kWorkers) {
    // ---- weights, and the O of this CTA to the others ----------------------------------------------------------------
    pdl_wait();
    bool ok = true;
    auto wait = [&](uint64_t* b, uint32_t ph) { ok = ok && __all_sync(0xFFFFFFFFu, ptx::mbar_wait<true>(b, ph, abort_flag, g.status) ? 1 : 0) != 0; };
    auto load_wp = [&](uint64_t* bar, int from, int to, uint8_t* dst) {
      if (ptx::elect_one()) {
        ptx::mbar_expect_tx(bar, (uint32_t)(to - from) * P_BLOCK);
#pragma unroll 1
        for (int t = from; t < to; ++t) ptx::tma_load_2d(dst + (t - from) * P_BLOCK, &tmP, bar, ring_block(t) * 64, rank * P_ROWS);
      }
      __syncwarp();
    };
#pragma unroll 1
    for (int kb = 0; kb < NV; ++kb) {
      const int s = kb % L::stages;
      if (kb >= L::stages) wait(&w_empty[s], (uint32_t)(kb / L::stages - 1) & 1u);
      if (!ok) break;
      if (ptx::elect_one()) {
        ptx::mbar_expect_tx(&w_full[s], W_STAGE);
        ptx::tma_load_4d(ring + s * W_STAGE, &tmW, &w_full[s], kb * 64, 0, 0, HP * rank);
      }
      __syncwarp();
    }
    if (L::beside && ok) load_wp(wp_early, 0, NV, wp);
    wait(qkv_full, 0);
    if (ok && lane < NV) ptx::mbar_arrive_cluster(ptx::mapa(ptx::smem_u32(a_free), (uint32_t)lane));     // this CTA's rows have been used
    __syncwarp();
    if (!L::beside && ok) load_wp(wp_early, 0, L::early, wp);
    if (L::early < NV) {
      wait(&o_full[0], 0);
      wait(&o_full[1], 0);
      if (ok) load_wp(wp_late, L::early, NV, ops);
    }
    wait(a_free, 0);
    wait(o_ready, 0);
    if (ok && lane > 0 && lane < NV) {                 // (to the next CTA first, so that no two send to the same one at once)
      const uint32_t to = (uint32_t)(rank + lane < NV ? rank + lane : rank + lane - NV);
      ptx::bulk_copy_cluster(ptx::mapa(ptx::smem_u32(sA + rank * kLnBlockBytes), to), sA + rank * kLnBlockBytes, kLnBlockBytes, ptx::mapa(ptx::smem_u32(&o_in[lane]), to));
    }
    __syncwarp();
    if (!ok) settle();
    ptx::cluster_arrive_relaxed();
  } else if (warp == kWorkers + 1) {
    // ---- products (the whole warp walks, an elected lane issues) ------------------------------------------------------
    const uint32_t a0 = ptx::smem_u32(sA), r0 = ptx::smem_u32(ring), ops0 = ptx::smem_u32(ops), wp0 = ptx::smem_u32(wp);
    bool ok = true;
    auto wait = [&](uint64_t* b, uint32_t ph) { ok = ok && __all_sync(0xFFFFFFFFu, ptx::mbar_wait<true>(b, ph, abort_flag, g.status) ? 1 : 0) != 0; };
    constexpr uint32_t idesc_qkv = ptx::make_idesc_bf16(128, W_ROWS, false, false), idesc_s = ptx::make_idesc_bf16(128, TP, false, false),
                       idesc_pv = ptx::make_idesc_bf16(128, D, false, true), idesc_y = ptx::make_idesc_bf16(128, P_ROWS, false, false);
    wait(a_ready, 0);
#pragma unroll 1
    for (int kb = 0; kb < NV; ++kb) {
      const int s = kb % L::stages;
      wait(&w_full[s], (uint32_t)(kb / L::stages) & 1u);
      if (!ok) break;
      ptx::tc_fence_after();
      const uint64_t ad = ptx::make_smem_desc(a0 + kb * kLnBlockBytes, 16, 1024), bd = ptx::make_smem_desc(r0 + s * W_STAGE, 16, 1024);
      if (ptx::elect_one()) {
#pragma unroll
        for (int k = 0; k < 4; ++k) ptx::tc_mma_bf16(tmem_base, ad + 2 * k, bd + 2 * k, idesc_qkv, (kb | k) ? 1u : 0u);
        if (NV > L::stages) ptx::tc_commit(&w_empty[s]);
        if (kb == NV - 1) ptx::tc_commit(qkv_full);
      }
      __syncwarp();
    }
#pragma unroll 1
    for (int h = 0; h < HP; ++h) {
      wait(&qk_ready[h], 0);
      if (!ok) break;
      ptx::tc_fence_after();
      const uint64_t qd = desc_sw64(ops0 + h * 3 * OP_BYTES), kd = desc_sw64(ops0 + (h * 3 + 1) * OP_BYTES);
      if (ptx::elect_one()) {
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {               // 16 features per step: +32 bytes; steps 2-3: the second window's keys, +4096 bytes
          const uint32_t first = ks < 2 ? 0u : ~0u;
          ptx::tc_mma_bf16_lanes(tmem_base + TM_S + h * TP, qd + 2 * (ks & 1), kd + 2 * (ks & 1) + (ks >> 1) * (4096 >> 4), idesc_s, ks & 1, first, ~first);
        }
        ptx::tc_commit(&s_full[h]);
      }
      __syncwarp();
    }
#pragma unroll 1
    for (int h = 0; h < HP; ++h) {
      wait(&v_ready[h], 0);
      wait(&p_full[h], 0);
      if (!ok) break;
      ptx::tc_fence_after();
      const uint64_t vd = desc_sw64(ops0 + (h * 3 + 2) * OP_BYTES);
      if (ptx::elect_one()) {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {               // 16 keys per step: P +8 packed columns, V +1024 bytes; steps 4-7: the second window
          const uint32_t first = ks < 4 ? 0u : ~0u;
          ptx::tc_mma_bf16_ta_lanes(tmem_base + h * 96 + 64, tmem_base + h * 96 + 8 * (ks & 3), vd + ks * (1024 >> 4), idesc_pv, (ks & 3) ? 1u : 0u, first, ~first);
        }
        ptx::tc_commit(&o_full[h]);
      }
      __syncwarp();
    }
    wait(o_ready, 0);
    wait(wp_early, 0);
#pragma unroll 1
    for (int t = 0; t < NV; ++t) {
      if (t > 0) wait(&o_in[t], 0);
      if (L::early < NV && t == L::early) wait(wp_late, 0);
      if (!ok) break;
      ptx::tc_fence_after();
      const uint64_t ad = ptx::make_smem_desc(a0 + ring_block(t) * kLnBlockBytes, 16, 1024);
      const uint64_t bd = ptx::make_smem_desc(t < L::early ? wp0 + t * P_BLOCK : ops0 + (t - L::early) * P_BLOCK, 16, 1024);
      if (ptx::elect_one()) {
#pragma unroll
        for (int k = 0; k < 4; ++k) ptx::tc_mma_bf16(tmem_base + TM_Y, ad + 2 * k, bd + 2 * k, idesc_y, (t | k) ? 1u : 0u);
        if (t == NV - 1) ptx::tc_commit(y_full);
      }
      __syncwarp();
    }
    wait(y_full, 0);
    if (!ok) settle();
    ptx::cluster_arrive_relaxed();                     // (what the others sent is here; each thread arrives when it is done with the others)
  } else {
    bool ok = true;
    auto wait = [&](uint64_t* b) { ok = ok && __all_sync(0xFFFFFFFFu, ptx::mbar_wait(b, 0, abort_flag, g.status) ? 1 : 0) != 0; };
    pdl_wait();
    pdl_launch_dependents();
    // ---- rows: eight a warp, in registers ------------------------------------------------------------------------------
    // (beyond 256 channels in two passes; all rows are asked for first, by asynchronous copies to where the lane that asked writes them
    // normalised)
    constexpr int LN = NV <= 3 ? 8 : 16, J = NV <= 4 ? LN / 4 : 2, V = 8 * NV / LN, PASSES = LN / 4 / J;
    const int sub = lane % LN, rsub = lane / LN;
    uint4 x[J][V];
    auto place = [&](int row, int k) {
      const int v = sub + LN * k;
      return sA + (v >> 3) * kLnBlockBytes + row * 128 + (((v ^ row) & 7) << 4);
    };
#pragma unroll
    for (int j = 0; j < J * PASSES; ++j) {
      const int row = warp * 8 + j * (32 / LN) + rsub;
      const long long off = offs[row];
#pragma unroll
      for (int k = 0; k < V; ++k) {
        if constexpr (PASSES > 1) {
          if (off >= 0) ptx::cp_async16(place(row, k), g.x + off + (sub + LN * k) * 8);
          else *reinterpret_cast<uint4*>(place(row, k)) = make_uint4(0, 0, 0, 0);
        } else {
          x[j % J][k] = make_uint4(0, 0, 0, 0);
          if (off >= 0) x[j % J][k] = *reinterpret_cast<const uint4*>(g.x + off + (sub + LN * k) * 8);
        }
      }
    }
    if (PASSES > 1) ptx::cp_async_commit();
    // parameters to shared memory, their latency under the rows'
    const int n_table = (2 * ws - 1) * (2 * ws - 1);
    if (tid < 2 * C / 8) {
      *reinterpret_cast<uint4*>(lng + tid * 8) = *reinterpret_cast<const uint4*>((tid < C / 8 ? g.ln_g : g.ln_b - C) + tid * 8);
    } else if (tid < 2 * C / 8 + W_ROWS / 8) {
      const int v = tid - 2 * C / 8, hq = v >> 2, hh = hq / 3, which = hq - 3 * hh;          // four vectors a head and operand
      *reinterpret_cast<uint4*>(bq + v * 8) = *reinterpret_cast<const uint4*>(g.b_qkv + which * C + (HP * rank + hh) * D + (v & 3) * 8);
    } else if (tid < 2 * C / 8 + (W_ROWS + P_ROWS) / 8) {
      const int v = tid - (2 * C + W_ROWS) / 8;
      *reinterpret_cast<uint4*>(bp + v * 8) = *reinterpret_cast<const uint4*>(g.b_proj + rank * P_ROWS + v * 8);
    }
    for (int i = tid; i < HP * n_table; i += 32 * kWorkers) {
      const int hh = i & 1, e = i >> 1;
      raw_s[hh * 256 + e] = g.table[e * g.heads + HP * rank + hh];
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kWorkers) : "memory");
#pragma unroll 1
    for (int pass = 0; pass < PASSES; ++pass) {
      if constexpr (PASSES > 1) {
        ptx::cp_async_wait<0>();
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
          for (int k = 0; k < V; ++k) x[j][k] = *reinterpret_cast<const uint4*>(place(warp * 8 + (pass * J + j) * (32 / LN) + rsub, k));
      }
      ln_rows_to_operand<NV, LN, J, V>(
          x,
          [&](int, int v, ptx::f32x2(&ga)[4], ptx::f32x2(&be)[4]) {
            ln_widen8(*reinterpret_cast<const uint4*>(lng + v * 8), ga);
            ln_widen8(*reinterpret_cast<const uint4*>(lnb + v * 8), be);
          },
          g.eps, sA, warp * 8 + pass * J * (32 / LN), lane, [] { return true; });
    }
    ptx::fence_proxy_async();
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(a_ready);
    // ---- while the product runs: the heads' biases as [T, T] tables of bf16 pairs, -inf for padded keys ----------------
#pragma unroll
    for (int i = tid; i < HP * TP * (TP / 8); i += 32 * kWorkers) {        // eight keys of a row
      const int hh = i >> 9, r = (i >> 3) & 63, c0 = (i & 7) * 8;
      const int4 k0 = *reinterpret_cast<const int4*>(code + c0), k1 = *reinterpret_cast<const int4*>(code + c0 + 4);
      const int kc[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
      const uint16_t* row = raw_s + hh * 256 + code[r] + (ws - 1) * 2 * ws;
      uint32_t word[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t lo = c0 + 2 * k < T ? row[-kc[2 * k]] : 0xFF80u, hi = c0 + 2 * k + 1 < T ? row[-kc[2 * k + 1]] : 0xFF80u;
        word[k] = lo | hi << 16;
      }
      *reinterpret_cast<uint4*>(bias_t + (hh * TP + r) * BIAS_ROW + c0 / 2) = make_uint4(word[0], word[1], word[2], word[3]);
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kWorkers) : "memory");
    // ---- q, k, v of a head: a row per thread, rounded to bf16 as the QKV linear stores them; rows without a token are zero ---------
    const int q = warp & 3, hh = (warp >> 2) & 1, part = warp >> 3, r = q * 32 + lane, w = r >> 6, i = r & 63;
    const uint32_t lane_addr = (uint32_t)(q * 32) << 16, mine = tmem_base + lane_addr + hh * 96;
    const long long off = offs[r];
    uint8_t* my_ops = ops + hh * 3 * OP_BYTES;
    wait(qkv_full);
    ptx::tc_fence_after();
    // sixteen columns `c0` of operand `which`
    auto put = [&](int which, int c0, const uint32_t* v) {
#pragma unroll
      for (int ch = 0; ch < 2; ++ch) {
        const uint4 b4 = *reinterpret_cast<const uint4*>(bq + (hh * 3 + which) * D + c0 + ch * 8);
        const uint32_t bw[4] = {b4.x, b4.y, b4.z, b4.w};
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = bf16x2_to_float2(bw[e]);
          o[e] = float2_to_bf16x2(__uint_as_float(v[ch * 8 + 2 * e]) + f.x, __uint_as_float(v[ch * 8 + 2 * e + 1]) + f.y);
        }
        *reinterpret_cast<uint4*>(my_ops + which * OP_BYTES + sw64_off(r, c0 / 8 + ch)) = off >= 0 ? make_uint4(o[0], o[1], o[2], o[3]) : make_uint4(0, 0, 0, 0);
      }
    };
    uint4 res[2] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
    const int grp = warp >> 2, col = rank * P_ROWS + grp * 16;                   // this thread's sixteen output columns of its row
    if (ok) {
      uint32_t v[48];
      ptx::tmem_ld32(mine + part * 64, v);             // q or v
      ptx::tmem_ld16(mine + 32 + part * 16, v + 32);   // half of k
      ptx::tmem_ld_wait();
      put(1, part * 16, v + 32);
      put(part * 2, 0, v);
      put(part * 2, 16, v + 16);
      ptx::tc_fence_before();
      ptx::fence_proxy_async();
      __syncwarp();
      if (lane == 0) {
        ptx::mbar_arrive(&qk_ready[hh]);
        if (part) ptx::mbar_arrive(&v_ready[hh]);
      }
    }
    // ---- softmax (attn_window_tc.cu): two threads a row, 32 keys each --------------------------------------------------------
    const float LOG2E = 1.4426950408889634f;
    const int n = 2 * unit + w;
    uint32_t diff = 0;                                 // keys of another region than this row
    if (g.shift > 0 && n < g.n_windows) {
      const int wl = n - (int)fd_div((uint32_t)n, g.fd_wpi) * g.win_per_img;
      const int wy = (int)fd_div((uint32_t)wl, g.fd_nww), wx = wl - wy * g.nWw;
      if (wy == g.nWh - 1) diff |= kmask[part] ^ ((tyx[i] >> 8) >= ws - g.shift ? 0xFFFFFFFFu : 0u);
      if (wx == g.nWw - 1) diff |= kmask[2 + part] ^ ((tyx[i] & 255) >= ws - g.shift ? 0xFFFFFFFFu : 0u);
    }
    float sc[32], mx = -INFINITY;
    float* red_h = red + hh * 256 + r;
    wait(&s_full[hh]);
    if (ok) {
      ptx::tc_fence_after();
      uint32_t rv[32];
      ptx::tmem_ld32(tmem_base + lane_addr + TM_S + hh * TP + part * 32, rv);
      ptx::tmem_ld_wait();
      float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      const uint32_t* brow = bias_t + (hh * TP + i) * BIAS_ROW + part * 16;
#pragma unroll
      for (int v8 = 0; v8 < 4; ++v8) {
        const uint4 b4 = *reinterpret_cast<const uint4*>(brow + v8 * 4);              // (-inf behind the last key)
        const uint32_t bw[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int c = v8 * 8 + 2 * j;
          sc[c] = fmaf(__uint_as_float(rv[c]), g.scale, __uint_as_float(bw[j] << 16));
          sc[c + 1] = fmaf(__uint_as_float(rv[c + 1]), g.scale, __uint_as_float(bw[j] & 0xFFFF0000u));
        }
      }
      if (__any_sync(0xFFFFFFFFu, diff != 0)) {        // seam windows only: keys of another region get -100
#pragma unroll
        for (int c = 0; c < 32; ++c)
          if ((diff >> c) & 1u) sc[c] -= 100.f;
      }
#pragma unroll
      for (int c = 0; c < 32; ++c) mx4[c & 3] = fmaxf(mx4[c & 3], sc[c]);
      mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      red_h[part * 128] = mx;
    }
    // The two threads of a row exchange their maxima and then their sums, in memory that no other head writes.  A thread's sum goes to
    // where its partner's maximum was, which it alone has read.  (Every warp comes to the barrier: one of the two may have given up waiting.)
    asm volatile("bar.sync %0, 64;" ::"r"(2 + hh * 4 + q) : "memory");
    if (ok) {
      const float nmx = -fmaxf(mx, red_h[(1 - part) * 128]) * LOG2E;
      float sum4[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t pk[16];
#pragma unroll
      for (int c8 = 0; c8 < 4; ++c8) {
        if (part * 32 + c8 * 8 < T) {                  // (uniform)
#pragma unroll
          for (int c = c8 * 8; c < c8 * 8 + 8; c += 2) {
            const float p0 = ptx::ex2(fmaf(sc[c], LOG2E, nmx)), p1 = ptx::ex2(fmaf(sc[c + 1], LOG2E, nmx));
            sum4[c & 2] += p0;
            sum4[(c & 2) + 1] += p1;
            pk[c / 2] = float2_to_bf16x2(p0, p1);
          }
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) pk[c8 * 4 + e] = 0u;
        }
      }
      const float sum = (sum4[0] + sum4[1]) + (sum4[2] + sum4[3]);
      red_h[(1 - part) * 128] = sum;
      ptx::tmem_st16(mine + part * 16, pk);
      ptx::tmem_st_wait();
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&p_full[hh]);
      if (off >= 0) {
        res[0] = *reinterpret_cast<const uint4*>(g.x + off + col);
        res[1] = *reinterpret_cast<const uint4*>(g.x + off + col + 8);
      }
      wait(&p_full[hh]);                               // (complete by now: orders the partner's sum before the read below)
      wait(&o_full[hh]);
      if (ok) {
        // O of this head: columns 32 hh of the CTA's block of the projection's operand, half of them a thread
        ptx::tc_fence_after();
        const float inv = 1.f / (red_h[0] + red_h[128]);
        uint32_t v[16];
        ptx::tmem_ld16(mine + 64 + part * 16, v);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          uint32_t o[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) o[e] = float2_to_bf16x2(__uint_as_float(v[ch * 8 + 2 * e]) * inv, __uint_as_float(v[ch * 8 + 2 * e + 1]) * inv);
          *reinterpret_cast<uint4*>(sA + rank * kLnBlockBytes + r * 128 + (((hh * 4 + part * 2 + ch) ^ (r & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
        }
        ptx::fence_proxy_async();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(o_ready);
      }
    }
    ptx::cluster_arrive_relaxed();
    // ---- output --------------------------------------------------------------------------------------------------------------
    wait(y_full);
    if (ok) {
      ptx::tc_fence_after();
      uint32_t v[16], o[8];
      ptx::tmem_ld16(tmem_base + lane_addr + TM_Y + grp * 16, v);
      const uint4 b0 = *reinterpret_cast<const uint4*>(bp + grp * 16), b1 = *reinterpret_cast<const uint4*>(bp + grp * 16 + 8);
      const uint32_t bw[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
      const uint32_t rw[8] = {res[0].x, res[0].y, res[0].z, res[0].w, res[1].x, res[1].y, res[1].z, res[1].w};
      ptx::tmem_ld_wait();
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float2 b = bf16x2_to_float2(bw[e]), f = bf16x2_to_float2(rw[e]);
        o[e] = float2_to_bf16x2(__uint_as_float(v[2 * e]) + b.x + f.x, __uint_as_float(v[2 * e + 1]) + b.y + f.y);
      }
      if (off >= 0) ln_store16(g.y + off + col, o, g.wide);
    }
  }
  ptx::tc_fence_before();
  __syncwarp();
  ptx::cluster_wait();                                 // no CTA leaves while its O is still being copied or others still signal it
  if (warp == kWorkers + 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

template <int NV>
int launch(const CUtensorMap& tw, const CUtensorMap& tp, const AttnClusterArgs& g, cudaStream_t st) {
  const auto kernel = swin_attn_cluster_kernel<NV>;
  if (ensure_max_dynamic_smem((const void*)kernel, Plan<NV>::bytes) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("swin_attn_cluster", st);
  const unsigned grid = (unsigned)((g.n_windows + 1) / 2 * NV);
  if (launch_pdl_cluster(kernel, dim3(grid), dim3(kThreads), Plan<NV>::bytes, st, (unsigned)NV, tw, tp, g) != cudaSuccess) return SMARTMEM_ERR_CUDA;
  count_launch();
  return SMARTMEM_OK;
}

}  // namespace

// Where it beats the separate kernels: one wave of clusters (us of an attention half, separate -> this, by rows: C = 128 98 16.1 -> 8.1, 3626
// 14.5 -> 8.3, 7252 16.8 -> 9.4; C = 192 98 12.1 -> 8.8, 3920 16.6 -> 10.2; C = 256 98 12.5 -> 9.7, 3234 17.5 -> 11.5; C = 384 98 14.6 -> 12.7,
// 2156 21.0 -> 15.4; C = 512 196 15.0 -> 15.4, 392 16.4 -> 15.5, 1470 21.6 -> 18.2), and for C = 128 and 192 a second one that is well filled
// (C = 128 9016 17.4 -> 17.3, 10780 21.4 -> 17.7, 14504 24.1 -> 18.7; C = 192 4900 17.6 -> 18.5, 6860 21.4 -> 19.8, 8624 22.9 -> 20.9).  From there
// on a unit at a time loses to kernels that stream: C = 128 21756 29.0 -> 28.0, 29008 32.4 -> 37.2; C = 256 6468 23.4 -> 23.0, 9702 29.1 -> 34.3.
bool swin_attn_cluster_wins(const smartmem_swin_params_t& p) {
  const int nv = p.C / 64, T = p.window * p.window;
  if (p.dtype != SMARTMEM_BF16 || p.C % 64 || p.C != p.heads * D || T > TP || (nv != 2 && nv != 3 && nv != 4 && nv != 6 && nv != 8)) return false;
  const long long windows = (long long)p.B * (p.H / p.window) * (p.W / p.window);
  const long long units = (windows + 1) / 2, wave = tc_cluster_ctas(nv) / nv;
  if (units <= wave) return nv < 8 || units >= 3;
  return nv <= 3 && 10 * units >= (nv == 2 ? 13 : 15) * wave && units <= 2 * wave - 2;
}

int launch_swin_attn_cluster(const smartmem_swin_params_t& p, const DevMap& rowmap, const void* x, void* y, cudaStream_t st) {
  AttnClusterArgs g;
  memset(&g, 0, sizeof(g));
  g.x = (const __nv_bfloat16*)x; g.y = (__nv_bfloat16*)y;
  g.ln_g = (const __nv_bfloat16*)p.ln1_g; g.ln_b = (const __nv_bfloat16*)p.ln1_b;
  g.b_qkv = (const __nv_bfloat16*)p.b_qkv; g.b_proj = (const __nv_bfloat16*)p.b_proj; g.table = (const uint16_t*)p.rel_bias_table;
  g.heads = p.heads; g.ws = p.window; g.T = p.window * p.window; g.shift = p.shift;
  g.nWw = p.W / p.window; g.nWh = p.H / p.window; g.win_per_img = g.nWw * g.nWh; g.n_windows = p.B * g.win_per_img;
  g.fd_wpi = make_fastdiv((uint32_t)g.win_per_img);
  g.fd_nww = make_fastdiv((uint32_t)g.nWw);
  g.eps = p.ln_eps; g.scale = 1.0f / sqrtf((float)D);
  g.wide = ((uintptr_t)y & 31) == 0;
  g.rowmap = rowmap;
  g.status = device_status_ptr();
  if (!g.status) return SMARTMEM_ERR_CUDA;
  CUtensorMap tw, tp;
  // [q, k, v][head][32][C]; a box is a k-block of q, k and v of two heads, head by head
  const long long C = p.C, dims[4] = {C, D, 3, p.heads}, strides[3] = {C, C * C, D * C};
  const int box[4] = {64, D, 3, HP};
  int rc = tc_encode_nd_sw128(p.w_qkv, 4, dims, strides, box, &tw);
  if (rc == SMARTMEM_OK) rc = tc_encode_2d(p.w_proj, C, C, C, 64, P_ROWS, &tp);
  if (rc != SMARTMEM_OK) return rc;
  switch (p.C / 64) {
#define SM_CLUSTER(NV) case NV: return launch<NV>(tw, tp, g, st);
    SM_CLUSTER(2) SM_CLUSTER(3) SM_CLUSTER(4) SM_CLUSTER(6) SM_CLUSTER(8)
#undef SM_CLUSTER
  }
  return SMARTMEM_ERR_UNSUPPORTED;
}

}  // namespace smartmem
