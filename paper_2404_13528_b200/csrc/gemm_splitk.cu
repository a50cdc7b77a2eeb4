// bf16 GEMM for few rows: out[m, n] = epilogue( sum_k X[m, k] W[n, k] ), M small against N and K.
//
// A GEMM with few rows of X is the stream of W through the chip, and what bounds it is how many bytes of W are in flight:
// the tiled kernel gives a 128-row tile of X one CTA per 64-256 columns (64-96 CTAs at N = 4096-12288), each with four
// stages of a latency-bound ring, and most of the A tile is padding.  Here the roles are swapped and the reduction is split:
//   * W is the 128-row operand of the tensor core and X its N-side operand, NB = M rounded up to 16 (at most 256) columns
//     wide, so no product is spent on more than 15 rows of padding and a stage is 16 KB of W plus NB x 128 bytes;
//   * the K range of a 128-column output tile is split over the CTAs of a cluster (up to 8), so that every SM pulls on W;
//     the partial sums meet in distributed shared memory: every CTA leaves its fp32 tile in its own shared memory and
//     finishes a share of the rows, reading the other CTAs' tiles.  No workspace, no atomics, a fixed order of additions;
//   * RMSNorm of X can ride along: x g is rounded to bf16 in shared memory on the way to the tensor core, the sum of squares
//     of each row is collected at the same time, and the epilogue multiplies the fp32 sum by rstd -- one rounding, as when
//     the normalised row itself is stored;
//   * W and X have rings of their own: X comes from L2 and is scaled well ahead of the products, so that a stage of W is
//     only held for its copy and its product (with one ring the scaling's latency came off the depth of W's);
//   * where nothing in flight writes W (TcEpilogue::b_settled) the ring is filled with it before the dependency wait, otherwise the
//     same boxes are only prefetched into L2 there: W may be the second operand of a product, or a weight that the kernel before this
//     one is still writing.
//
// Warp roles (8 warps): 0 TMA producer of W, 1 TMEM owner and MMA issuer, 2-6 scale X (RMSNorm), 7 TMA producer of X, 2-5
// drain the accumulator; all eight finish the rows.
#include <cstring>

#include "gemm_tc.cuh"
#include "ptx.cuh"

namespace smartmem {
namespace {

constexpr int BN_W = 128;                         // rows of W (output columns) per tile
constexpr int BK = 64;
constexpr int W_STAGE = BN_W * BK * 2;            // 16 KB
constexpr int kThreads = 256;
constexpr int kMaxSplits = 8;                     // portable cluster size
constexpr int kMaxStages = 12;
constexpr int kMaxXStages = 8;
constexpr int kScaleWarps = 5;
constexpr int kMaxNormRows = 128;

struct SplitArgs {
  int M, N, NB, splits, nkb, stages, xstages, tiles_m;
  uint32_t x_bytes, tmem_cols;                    // bytes of an X stage
  int x_off, gamma_off, table_off, bar_off;              // byte offsets behind the aligned base
  const __nv_bfloat16* gamma;                     // RMSNorm of X (null: none)
  float eps, invK;
  __nv_bfloat16* out;
  long long ldc;
  const __nv_bfloat16 *bias, *residual;
  int gelu, has_rowmap, w_settled;
  int rope_cols, rope_S, rope_pos0, rope_half;
  float rope_c;
  int seg_cols;
  __nv_bfloat16* seg_out[3];
  long long seg_ld[3];
  int* status;
  DevMap rowmap;
};

__global__ void __launch_bounds__(kThreads, 2)
gemm_splitk_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const __grid_constant__ SplitArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  __nv_bfloat16* gamma_s = reinterpret_cast<__nv_bfloat16*>(smem + g.gamma_off);      // this CTA's K range
  long long* offs = reinterpret_cast<long long*>(smem + g.table_off);                 // [NB] output offset of a row
  float* ss = reinterpret_cast<float*>(offs + g.NB);                                  // [NB] this CTA's sums of squares
  float* ssw = ss + g.NB;                                                             // [kScaleWarps][NB] per warp (RMSNorm only)
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + g.bar_off);
  uint64_t* empty = full + kMaxStages;
  uint64_t* xfull = empty + kMaxStages;
  uint64_t* xready = xfull + kMaxXStages;                                             // X scaled (RMSNorm only)
  uint64_t* xempty = xready + kMaxXStages;
  uint64_t* acc_full = xempty + kMaxXStages;
  uint8_t* sx = smem + g.x_off;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  float* buf = reinterpret_cast<float*>(smem);                                        // [NB][128] fp32, over the drained rings

  const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
  const int S = g.splits;
  const int rank = S > 1 ? (int)ptx::cluster_ctarank() : 0;
  const int tile = (int)blockIdx.x / S;
  const int tile_n = tile / g.tiles_m, tile_m = tile - tile_n * g.tiles_m;            // row tiles that share W are neighbours
  const int n0 = tile_n * BN_W, m0 = tile_m * g.NB;
  const int rows = min(g.NB, g.M - m0);
  const int kb0 = (int)((long long)g.nkb * rank / S), kb1 = (int)((long long)g.nkb * (rank + 1) / S), nk = kb1 - kb0;
  const bool norm = g.gamma != nullptr;

  if (tid == 0) {
    for (int s = 0; s < g.stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < g.xstages; ++s) {
      ptx::mbar_init(&xfull[s], 1);
      ptx::mbar_init(&xready[s], 1);
      ptx::mbar_init(&xempty[s], 1);
    }
    ptx::mbar_init(acc_full, 1);
    *abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
  }
  __syncwarp();
  if (warp == 0) {
    // the ring's first round of W (two loops: with the choice inside the elected branch a copy took longer to issue, 0.4 us a launch)
    const int first = min(g.stages, nk);
    if (g.w_settled) {
#pragma unroll 1
      for (int s = 0; s < first; ++s) {
        if (ptx::elect_one()) {
          ptx::mbar_expect_tx(&full[s], W_STAGE);
          ptx::tma_load_2d(smem + s * W_STAGE, &tmW, &full[s], (kb0 + s) * BK, n0);
        }
        __syncwarp();
      }
    } else {
#pragma unroll 1
      for (int s = 0; s < first; ++s) {
        if (ptx::elect_one()) ptx::tma_prefetch_2d(&tmW, (kb0 + s) * BK, n0);
        __syncwarp();
      }
    }
  }
  if (warp == 1) ptx::tmem_alloc(tmem_slot, g.tmem_cols);
  if (norm)                                         // (a line per k-block)
#pragma unroll 1
    for (int i = tid; i < nk; i += kThreads) ptx::prefetch_l2(g.gamma + (kb0 + i) * BK);
  {
    const int sg = g.seg_cols > 0 ? n0 / g.seg_cols : 0;
    const long long ld = g.seg_cols > 0 ? g.seg_ld[sg] : g.ldc;
    for (int i = tid; i < rows; i += kThreads)
      offs[i] = g.has_rowmap ? devmap_eval(g.rowmap, (uint32_t)(m0 + i)) : (long long)(m0 + i) * ld;
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();
  pdl_launch_dependents();

  if (warp == 0 || warp == 7) {
    // (warp-uniform loops, an elected lane issues: see gemm_tc.cu)
    const bool w_side = warp == 0;
    const int ns = w_side ? g.stages : g.xstages;
    uint64_t* bf = w_side ? full : xfull;
    uint64_t* be = w_side ? empty : xempty;
    const uint32_t bytes = w_side ? (uint32_t)W_STAGE : g.x_bytes;
    uint8_t* ring = w_side ? smem : sx;
    const CUtensorMap* tm = w_side ? &tmW : &tmX;
    const int row0 = w_side ? n0 : m0, first = w_side && g.w_settled ? min(ns, nk) : 0;      // (settled W: the first round is on its way already)
    bool ok = true;
    int issued = first;
    uint32_t s = first == ns ? 0 : (uint32_t)first, ph = first == ns ? 0 : 1;
    for (int kb = first; kb < nk; ++kb) {
      ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(&be[s], ph, abort_flag, g.status) ? 1 : 0) != 0;
      if (!ok) break;
      if (ptx::elect_one()) {
        ptx::mbar_expect_tx(&bf[s], bytes);
        ptx::tma_load_2d(ring + s * bytes, tm, &bf[s], (kb0 + kb) * BK, row0);
      }
      __syncwarp();
      ++issued;
      if (++s == (uint32_t)ns) { s = 0; ph ^= 1; }
    }
    if (*abort_flag && lane == 0) {                 // unwinding: copies in flight get a bounded chance to land
      for (int k = issued > ns ? issued - ns : 0; k < issued; ++k) {
        const unsigned long long t0 = ptx::globaltimer();
        while (!ptx::mbar_try_wait(&bf[k % ns], (k / ns) & 1) && ptx::globaltimer() - t0 < 2000000ull) {
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    const uint32_t idesc = ptx::make_idesc_bf16(BN_W, g.NB, false, false);
    const uint32_t wb = ptx::smem_u32(smem), xb = ptx::smem_u32(sx);
    uint64_t* gate = norm ? xready : xfull;
    bool ok = true;
    uint32_t s = 0, ph = 0, xs = 0, xph = 0;
    for (int kb = 0; kb < nk; ++kb) {
      ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(&gate[xs], xph, abort_flag, g.status) && ptx::mbar_wait(&full[s], ph, abort_flag, g.status) ? 1 : 0) != 0;
      if (!ok) break;
      ptx::tc_fence_after();
      const uint64_t ad = ptx::make_smem_desc(wb + s * W_STAGE, 16, 1024);
      const uint64_t bd = ptx::make_smem_desc(xb + xs * g.x_bytes, 16, 1024);
      if (ptx::elect_one()) {
        ptx::tc_mma_bf16(tmem_base, ad, bd, idesc, kb ? 1u : 0u);
#pragma unroll
        for (int k = 1; k < BK / 16; ++k) ptx::tc_mma_bf16(tmem_base, ad + 2 * k, bd + 2 * k, idesc, 1u);
        ptx::tc_commit(&empty[s]);
        ptx::tc_commit(&xempty[xs]);
        if (kb == nk - 1) ptx::tc_commit(acc_full);
      }
      __syncwarp();
      if (++s == (uint32_t)g.stages) { s = 0; ph ^= 1; }
      if (++xs == (uint32_t)g.xstages) { xs = 0; xph ^= 1; }
    }
  } else {                                          // warps 2-6
    bool ok = true;
    if (norm) {
#pragma unroll 1
      for (int i = tid - 64; i < nk * (BK / 8); i += 32 * kScaleWarps)
        reinterpret_cast<uint4*>(gamma_s)[i] = *reinterpret_cast<const uint4*>(g.gamma + kb0 * BK + i * 8);
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kScaleWarps) : "memory");
      // a warp scales whole stages, always the same ones of the ring, so that it sees every phase of their barriers; lane l
      // owns 16-byte chunk l % 8 of rows l / 8 + 4 i, so its eight gammas are the same for all of them.  Four chunks are
      // loaded before the first is worked on.
      const int w = warp - 2, ch = lane & 7, r0 = lane >> 3, ni = (rows + 3) >> 2;
      float sq[kMaxNormRows / 4];
#pragma unroll
      for (int i = 0; i < kMaxNormRows / 4; ++i) sq[i] = 0.f;
      for (int k0 = 0, ph = 0; k0 < nk && ok; k0 += g.xstages, ph ^= 1)
        for (int s = w; s < g.xstages && k0 + s < nk; s += kScaleWarps) {
          const uint4 gv = *reinterpret_cast<const uint4*>(gamma_s + (k0 + s) * BK + ch * 8);
          ok = ptx::mbar_wait(&xfull[s], (uint32_t)ph, abort_flag, g.status);
          if (!ok) break;
          uint8_t* xt = sx + s * g.x_bytes + r0 * 128;
#pragma unroll
          for (int i0 = 0; i0 < kMaxNormRows / 4; i0 += 4)
            if (i0 < ni) {
              uint4 v[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) v[i] = *reinterpret_cast<const uint4*>(xt + (i0 + i) * 512 + ((ch ^ ((r0 + 4 * i) & 7)) << 4));
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float2 a = bf16x2_to_float2(v[i].x), b = bf16x2_to_float2(v[i].y), c = bf16x2_to_float2(v[i].z), d = bf16x2_to_float2(v[i].w);
                sq[i0 + i] += fmaf(a.x, a.x, a.y * a.y) + fmaf(b.x, b.x, b.y * b.y) + (fmaf(c.x, c.x, c.y * c.y) + fmaf(d.x, d.x, d.y * d.y));
                *reinterpret_cast<uint4*>(xt + (i0 + i) * 512 + ((ch ^ ((r0 + 4 * i) & 7)) << 4)) =
                    make_uint4(ptx::mul_bf16x2(v[i].x, gv.x), ptx::mul_bf16x2(v[i].y, gv.y), ptx::mul_bf16x2(v[i].z, gv.z),
                               ptx::mul_bf16x2(v[i].w, gv.w));
              }
            }
          ptx::fence_proxy_async();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&xready[s]);
        }
#pragma unroll
      for (int i = 0; i < kMaxNormRows / 4; ++i)
        if (i < ni) {
          float v = sq[i];
          v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
          v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
          v += __shfl_xor_sync(0xFFFFFFFFu, v, 4);
          if (ch == 0) ssw[w * g.NB + r0 + 4 * i] = v;
        }
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kScaleWarps) : "memory");
      for (int r = tid - 64; r < rows; r += 32 * kScaleWarps) {
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < kScaleWarps; ++k) v += ssw[k * g.NB + r];
        ss[r] = v;
      }
    }
    if (warp >= 6) ok = false;                       // four warps drain the accumulator: one per tensor-memory lane quadrant
    else ok = ok && ptx::mbar_wait(acc_full, 0, abort_flag, g.status);
    ok = __all_sync(0xFFFFFFFFu, ok ? 1 : 0) != 0;
    if (ok) {
      // accumulator lane = output column, accumulator column = row of X: a store writes 32 consecutive floats
      ptx::tc_fence_after();
      const int q = warp & 3;
      const uint32_t ta = tmem_base + ((uint32_t)(q * 32) << 16);
      float* b = buf + q * 32 + lane;
      for (int c = 0; c < rows; c += 16) {
        uint32_t r[16];
        ptx::tmem_ld16(ta + c, r);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j) b[(c + j) * BN_W] = __uint_as_float(r[j]);
      }
    }
  }
  ptx::tc_fence_before();
  __syncwarp();
  if (S > 1) ptx::cluster_sync(); else __syncthreads();

  // finish this CTA's share of the rows: a warp per row, four columns per lane: two adjacent ones at ca and two at cb
  // (rotary partners of one another where the lane rotates), so that a warp stores 128 contiguous bytes twice
  {
    const int ra = (int)((long long)rows * rank / S), rb = (int)((long long)rows * (rank + 1) / S);
    int ca = 2 * lane, cb = 2 * lane + 64;
    bool rot = false;
    if (n0 < g.rope_cols) {                          // pairs (i, i + R/2) of the head's first R columns; the rest as they lie
      const int h = g.rope_half;
      rot = 2 * lane < h;
      ca = rot ? 2 * lane : 4 * lane;
      cb = rot ? 2 * lane + h : 4 * lane + 2;
    }
    const int na = n0 + ca, nb = n0 + cb;
    const bool oka = na < g.N, okb = nb < g.N;       // (N is even)
    float2 ba = make_float2(0.f, 0.f), bb = ba;
    if (g.bias) {
      if (oka) ba = bf16x2_to_float2(*reinterpret_cast<const uint32_t*>(g.bias + na));
      if (okb) bb = bf16x2_to_float2(*reinterpret_cast<const uint32_t*>(g.bias + nb));
    }
    const int sg = g.seg_cols > 0 ? n0 / g.seg_cols : 0;
    __nv_bfloat16* out = g.seg_cols > 0 ? g.seg_out[sg] - (long long)sg * g.seg_cols : g.out;
    float f0 = 0.f, f1 = 0.f;
    if (rot) {
      f0 = ptx::ex2(-(float)(2 * lane) * g.rope_c);
      f1 = ptx::ex2(-(float)(2 * lane + 1) * g.rope_c);
    }
    auto rotate = [](float ang, float& x, float& y) {
      // (reduced mod 2 pi in two steps, then the hardware sine / cosine)
      const float kk = rintf(ang * 0.15915494309189535f);
      float red = fmaf(-kk, 6.2831854820251465f, ang);
      red = fmaf(kk, 1.7484556e-7f, red);
      const float sn = __sinf(red), cs = __cosf(red), x0 = x;
      x = x0 * cs - y * sn;
      y = y * cs + x0 * sn;
    };
    const uint32_t base = ptx::smem_u32(smem), ss_off = ptx::smem_u32(ss) - base;
    uint32_t peer[kMaxSplits];
#pragma unroll
    for (int r = 0; r < kMaxSplits; ++r) peer[r] = (S > 1 && r < S) ? ptx::mapa(base, (uint32_t)r) : base;
#pragma unroll 2
    for (int m = ra + warp; m < rb; m += kThreads / 32) {
      float2 va[kMaxSplits], vb[kMaxSplits];
      float vs[kMaxSplits];
      if (S == 1) {
        va[0] = *reinterpret_cast<const float2*>(buf + m * BN_W + ca);
        vb[0] = *reinterpret_cast<const float2*>(buf + m * BN_W + cb);
        vs[0] = norm ? ss[m] : 0.f;
      } else {
#pragma unroll
        for (int r = 0; r < kMaxSplits; ++r) {
          va[r] = vb[r] = make_float2(0.f, 0.f);
          vs[r] = 0.f;
          if (r < S) {
            va[r] = ptx::ld_cluster_f32x2(peer[r] + (uint32_t)(m * BN_W + ca) * 4u);
            vb[r] = ptx::ld_cluster_f32x2(peer[r] + (uint32_t)(m * BN_W + cb) * 4u);
            if (norm) vs[r] = ptx::ld_cluster_f32(peer[r] + ss_off + (uint32_t)m * 4u);
          }
        }
#pragma unroll
        for (int r = 1; r < kMaxSplits; ++r) {
          va[0].x += va[r].x; va[0].y += va[r].y;
          vb[0].x += vb[r].x; vb[0].y += vb[r].y;
          vs[0] += vs[r];
        }
      }
      float2 a = va[0], b = vb[0];
      if (norm) {
        const float rstd = rsqrtf(vs[0] * g.invK + g.eps);
        a.x *= rstd; a.y *= rstd;
        b.x *= rstd; b.y *= rstd;
      }
      if (rot) {
        const float pos = (float)(g.rope_pos0 + (g.rope_S > 1 ? (m0 + m) % g.rope_S : 0));
        rotate(pos * f0, a.x, b.x);
        rotate(pos * f1, a.y, b.y);
      }
      a.x += ba.x; a.y += ba.y;
      b.x += bb.x; b.y += bb.y;
      if (g.gelu) { a.x = gelu_tanh(a.x); a.y = gelu_tanh(a.y); b.x = gelu_tanh(b.x); b.y = gelu_tanh(b.y); }
      const long long off = offs[m];
      if (g.residual) {
        if (oka) { const float2 f = bf16x2_to_float2(*reinterpret_cast<const uint32_t*>(g.residual + off + na)); a.x += f.x; a.y += f.y; }
        if (okb) { const float2 f = bf16x2_to_float2(*reinterpret_cast<const uint32_t*>(g.residual + off + nb)); b.x += f.x; b.y += f.y; }
      }
      if (oka) *reinterpret_cast<uint32_t*>(out + off + na) = float2_to_bf16x2(a.x, a.y);
      if (okb) *reinterpret_cast<uint32_t*>(out + off + nb) = float2_to_bf16x2(b.x, b.y);
    }
  }
  __syncwarp();
  if (S > 1) ptx::cluster_sync(); else __syncthreads();   // no CTA leaves while another still reads its shared memory
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, g.tmem_cols);
  }
}

// Rows of a row tile: a multiple of 16, at most 256; the tiles are alike, so the last one may be mostly padding (300 rows in ten tiles of
// 32: 12 of its own).  Where the columns are few, as many row tiles as clusters of eight find room for, one CTA per SM: a CTA's share of
// the exchange shrinks with its tile and nothing else is long (134 x 2048 -> 512: 6.8 us in one row tile, 5.3 in three; 200 x 1536 -> 384
// 8.0, 5.2 in five; 100 x 1024 -> 256 5.6, 4.4 in four).  Not with few rows of a large weight, which every row tile reads (33 x 3072 -> 768
// 5.4, 5.8 in two), and beyond eight only for a reduction that is worth it (480 x 768 -> 8 5.1 in fifteen).
int row_tile(long long M, long long N, long long K, const ClusterCtas& fit) {
  long long room = fit.n[kMaxSplits] / kMaxSplits / ((N + BN_W - 1) / BN_W);
  if (M <= 64 && N * K > (1ll << 21)) room = 1;
  if (K < 1024 && room > 8) room = 8;
  const long long need = (M + 255) / 256, tiles = room > need ? room : need;
  return (int)(((M + tiles - 1) / tiles + 15) / 16 * 16);
}

// Sizes of a launch; returns the bytes of shared memory, 0 if a CTA's part does not fit (with RMSNorm: gamma of its K range lies beside
// the rings).
size_t plan_launch(long long M, long long N, long long K, bool norm, SplitArgs& g) {
  const ClusterCtas fit = tc_cluster_ctas_all();
  g.NB = row_tile(M, N, K, fit);
  g.tiles_m = (int)((M + g.NB - 1) / g.NB);
  if (norm && g.NB > kMaxNormRows) return 0;
  g.nkb = (int)(K / BK);
  const long long tiles = (N + BN_W - 1) / BN_W * g.tiles_m;
  g.x_bytes = (uint32_t)(g.NB * BK * 2);
  // Two CTAs per SM where X is narrow enough to leave each a ring of four or more stages of W.  As many splits as there are
  // CTA slots for: a second wave of clusters costs more than the shorter K ranges gain (N = 12288, K = 4096, 96 tiles:
  // 18.8 us in clusters of 2, 24 us in clusters of 3, 135 of which do not fit).
  const int per_sm = g.NB <= 64 ? 2 : 1;
  int splits = 1;
  for (int s = 2; s <= kMaxSplits && s <= g.nkb; ++s)
    if (tiles * s <= (long long)per_sm * fit.n[s]) splits = s;
  g.splits = splits;
  const int nk_max = (g.nkb + splits - 1) / splits;
  const uint32_t gamma_bytes = norm ? (uint32_t)(nk_max * BK * 2) : 0u;
  const uint32_t rows_bytes = (uint32_t)g.NB * 12u + (norm ? (uint32_t)(kScaleWarps * g.NB * 4) : 0u);
  const uint32_t bar_bytes = (2 * kMaxStages + 3 * kMaxXStages + 1) * 8 + 16;
  const uint32_t space = (per_sm == 2 ? 113u : 226u) * 1024u, fixed = 1024u + gamma_bytes + rows_bytes + bar_bytes + 32;
  if (space < fixed) return 0;
  const uint32_t budget = space - fixed;
  // X comes from L2 and needs less depth than W: a quarter of the space, but three stages at least, and one for each scaling
  // warp
  const int min_x = norm ? kScaleWarps : 3;
  int xstages = (int)(budget / 4 / g.x_bytes);
  xstages = xstages > kMaxXStages ? kMaxXStages : xstages < min_x ? min_x : xstages;
  if (xstages > nk_max) xstages = nk_max;
  if (budget < xstages * g.x_bytes + W_STAGE) return 0;
  int stages = (int)((budget - xstages * g.x_bytes) / W_STAGE);
  if (stages > kMaxStages) stages = kMaxStages;
  if (stages > nk_max) stages = nk_max;
  const uint32_t acc_bytes = (uint32_t)g.NB * BN_W * 4;              // the fp32 tile lies over the drained rings
  uint32_t ring = stages * W_STAGE + xstages * g.x_bytes;
  if (ring < acc_bytes) ring = (acc_bytes + 1023) / 1024 * 1024;
  if (ring > budget) return 0;
  g.stages = stages;
  g.xstages = xstages;
  g.x_off = stages * W_STAGE;
  g.gamma_off = (int)ring;
  g.table_off = (g.gamma_off + (int)gamma_bytes + 15) & ~15;
  g.bar_off = (g.table_off + (int)rows_bytes + 15) & ~15;
  g.tmem_cols = g.NB <= 32 ? 32 : g.NB <= 64 ? 64 : g.NB <= 128 ? 128 : 256;
  return 1024 + g.bar_off + bar_bytes;
}

}  // namespace

bool gemm_splitk_supported(const TcOperand& X, const TcOperand& W, const TcEpilogue& ep, long long batch, long long M, long long N,
                           long long K) {
  return batch == 1 && K % BK == 0 && X.n_row_atoms == 1 && X.n_batch_atoms == 0 && W.n_row_atoms == 1 && W.n_batch_atoms == 0 &&
         X.k_stride == 1 && W.k_stride == 1 && !ep.out2 && N % 8 == 0 && (ep.rope_cols == 0 || (N % BN_W == 0 && ep.rope_cols % BN_W == 0)) &&
         (ep.seg_cols == 0 || ep.seg_cols % BN_W == 0);
}

// Microseconds, fitted to measurements: a fixed part, the exchange of the partial sums (distributed shared memory moves about
// 14 bytes per clock and SM, which is what ends the range at 128 rows where the columns leave room for one row tile only), and the stream of W.  Below 32 rows the tiled kernel's estimate
// does not hold (its copies of a mostly empty A tile are slower than full ones), so the line is drawn by measurement, tiled -> this one:
// a long reduction, 2 rows, N = 4096: K = 512 5.1 -> 4.9, 1024 7.7 -> 5.5, 4096 23.6 -> 10.0; 31 rows, N = 512: K = 512 4.4 -> 4.6, 1024
// 5.9 -> 4.8.  A shorter one only where there are tiles enough for every SM and W is not yet all of the cost: 2 rows, K = 256, N = 1024
// 3.7 -> 4.0, 12288 5.1 -> 4.7, 32768 7.8 -> 5.6, 65536 10.3 -> 10.0, 131072 15.9 -> 18.3; 31 rows, 12288 4.8 -> 5.9, 32768 7.4 -> 6.2,
// 65536 10.0 -> 11.2; K = 128, N = 65536 7.3 -> 8.2.
double gemm_splitk_us(long long M, long long N, long long K) {
  const double nb = (double)((M + 15) / 16 * 16);
  if (M < 32) return K >= (M > 16 ? 768 : 512) || (K >= 256 && N * K >= (1ll << 23) && N < 65536) ? 0.0 : 1e30;
  // Few columns, in several row tiles: bound by the exchange (4.35 us at tiles of 32 rows and K = 768, 5.3 at 48 and 2048, 7.2 at 112 and 2048; the tiled
  // kernel 4.8, 8.7 and 8.7), but drawn by whole blocks of 7 x 7 windows, in which the tiled kernel overlaps more of what it follows: 245 rows of 256
  // channels 20.0 -> 18.7 us, 294 of 384 26.3 -> 25.5, 343 26.3 -> 26.4, 245 of 512 30.5 -> 28.8, 294 30.5 -> 30.4, 343 30.6 -> 31.2.
  if (M > 1024) return 1e30;
  const int tile = row_tile(M, N, K, tc_cluster_ctas_all());
  if (tile < M && (N + BN_W - 1) / BN_W * ((M + tile - 1) / tile) <= 24) return 2.96 + 0.04 * tile + 0.00045 * (double)K;
  return M > 128 ? 1e30 : 3.0 + 0.018 * nb + (double)N * (double)K * 2.0 / 6.2e6 * (1.0 + nb / 260.0);
}

bool gemm_splitk_norm_fits(long long M, long long N, long long K) {
  SplitArgs g;
  return M >= 1 && K % BK == 0 && plan_launch(M, N, K, true, g) != 0;
}

int launch_gemm_splitk(const TcOperand& X, const TcOperand& W, const TcEpilogue& ep, long long M, long long N, long long K, cudaStream_t st) {
  SplitArgs g;
  memset(&g, 0, sizeof(g));
  const size_t smem = plan_launch(M, N, K, ep.rms_gamma != nullptr, g);
  if (smem == 0) return SMARTMEM_ERR_UNSUPPORTED;
  g.M = (int)M; g.N = (int)N;
  g.gamma = (const __nv_bfloat16*)ep.rms_gamma; g.eps = ep.rms_eps; g.invK = 1.0f / (float)K;
  g.out = (__nv_bfloat16*)ep.out; g.ldc = ep.ldc;
  g.bias = (const __nv_bfloat16*)ep.bias; g.residual = (const __nv_bfloat16*)ep.residual; g.gelu = ep.gelu;
  g.w_settled = ep.b_settled;
  g.has_rowmap = ep.rowmap ? 1 : 0;
  if (ep.rowmap) g.rowmap = *ep.rowmap;
  const int rope_dim = ep.rope_dim ? ep.rope_dim : 128;
  g.rope_cols = ep.rope_cols; g.rope_S = ep.rope_S > 0 ? ep.rope_S : 1; g.rope_pos0 = ep.rope_pos0; g.rope_half = rope_dim / 2;
  g.rope_c = ep.rope_log2_theta / (float)(rope_dim / 2);
  g.seg_cols = ep.seg_cols;
  for (int i = 0; i < 3; ++i) { g.seg_out[i] = (__nv_bfloat16*)ep.seg_out[i]; g.seg_ld[i] = ep.seg_ld[i]; }
  g.status = device_status_ptr();
  if (!g.status) return SMARTMEM_ERR_CUDA;
  CUtensorMap tw, tx;
  int rc = tc_encode_2d(W.ptr, K, N, W.row_stride[0], BK, BN_W, &tw);
  if (rc == SMARTMEM_OK) rc = tc_encode_2d(X.ptr, K, M, X.row_stride[0], BK, g.NB, &tx);
  if (rc != SMARTMEM_OK) return rc;
  if (ensure_max_dynamic_smem((const void*)gemm_splitk_kernel, 227 * 1024) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("gemm_splitk", st);
  const unsigned grid = (unsigned)((N + BN_W - 1) / BN_W * g.tiles_m * g.splits);
  if (launch_pdl_cluster(gemm_splitk_kernel, dim3(grid), dim3(kThreads), smem, st, (unsigned)g.splits, tw, tx, g) != cudaSuccess)
    return SMARTMEM_ERR_CUDA;
  count_launch();
  return SMARTMEM_OK;
}

}  // namespace smartmem
