// The two halves of an fp32 Swin block, one kernel each (plain FMAs: a 10-bit-mantissa tensor-core path cannot meet 1e-4).
//
//   attention half: y = x + unshift(unpartition(proj(window_attention(qkv(LN1(partition(shift(x))))))))
//   MLP half:       y = x + fc2(GELU(fc1(LN2(x))))
//
// fp32 blocks are mostly small models at small batches: what bounds them is the chain of launches and of latencies inside each, so
// the seven kernels of the block became two (the MLP half's where it wins at that size; the attention half's at every size measured, 1
// to 64 images of 28 x 28 or 56 x 56 x 16 to 256 channels).  A cluster of CTAs shares one unit of work:
//   * attention: a window per cluster, a head per CTA.  Every CTA gathers and normalises the window's rows (redundantly: they
//     are few), computes q, k, v of its head, the scores, softmax and P v; the heads' outputs are exchanged through
//     distributed shared memory and every CTA projects onto its share of the output columns, adds the residual and scatters.
//     With few windows the tokens are shared out as well: a CTA normalises its own, writes their keys and values into the memory
//     of the others of its head, and goes on with its own queries.
//   * MLP: sixteen rows per cluster, a slice of the hidden features per CTA; the partial results of fc2 are added through
//     distributed shared memory in the order of the CTAs.
// Operands lie in shared memory with rows of K + 4 floats (an odd number of 16-byte vectors: eight lanes on eight rows hit
// distinct banks), a thread computes TM x TN outputs with 16-byte reads along K.
// What bounds the attention half is the length of its phases, one behind the other with a barrier between them, not their arithmetic (clock
// stamps: 20 to 130 thousand cycles a window when it had 256 threads, a warp per row in LayerNorm and softmax, parameters read from
// global memory where they were used, and index arithmetic per score).  So every phase is one round of one small tile a thread (512 threads
// beyond 32 tokens), eight lanes share a row, parameters come to shared memory with the rows, and a token's place in the bias table and its
// region are worked out once, ahead of the dependency wait.  Us of a stream of calls, that version -> this: [1,8,8,32] in 4 x 4 windows,
// two heads of 16 9.3 -> 6.3 (the host's call); [1,28,28,96], 7 x 7, three heads of 32 34.2 -> 16.9; [16,28,28,96] 128 -> 84 (both resident
// twice per SM: 64 registers; with 106 it was 100); [16,28,28,48], 4 x 4, three heads of 16 103 -> 56 (139 with 512 threads a window).
// The MLP half had the same faults: [4,14,14,64] 12.3 -> 10.3, [128,14,14,96] 296 -> 265; one output row by two columns a thread instead of two by four
// there: 307.
#include <cstring>

#include "attn.cuh"
#include "gemm_tc.cuh"
#include "ptx.cuh"

namespace smartmem {
namespace {

constexpr int kThreads = 256;                          // of the MLP half
constexpr int kMaxCluster = 8;

// A product's outputs, mt x nt tiles of TM x TN: a warp takes eight row tiles by four column tiles, a thread the rows tm + i mt and the
// columns tn + j nt of its tile, so that a warp's reads of either operand are eight or four neighbouring rows: one pass over the banks each.
// With the lanes along the columns a read of W was up to four passes: [2,21,14,32] in 7 x 7, heads of 16, 8.8 us -> 8.4 this way, [4,16,16,64] in 8 x 8 with
// its MLP half 32 -> 22.8.  Larger tiles leave too few warps to hide the reads: 8 x 4 and 4 x 4 in place of 4 x 4 and 2 x 4 were a tenth slower.
struct WarpTile {
  int tm, tn;
  bool in;
  __device__ __forceinline__ WarpTile(int w, int mt, int nt) {
    const int wr = (mt + 7) >> 3, wc = w / wr, lane = threadIdx.x & 31;
    tm = (w - wc * wr) * 8 + (lane & 7);
    tn = wc * 4 + (lane >> 3);
    in = tm < mt && tn < nt;
  }
};
// warps a product takes
__device__ __forceinline__ int warp_tiles(int mt, int nt) { return ((mt + 7) >> 3) * ((nt + 3) >> 2); }

// acc(i, j) = sum_k A[r0 + i rs][k] W[c0 + j cs][k], rows and columns clamped to M and N (what lies beyond is not used); K a multiple of 4.
// Even and odd k are summed apart, as the two halves of packed multiply-adds, where the registers allow it.
template <int TM, int TN, bool PACKED = (TM * TN <= 8)>
__device__ __forceinline__ void tile_dot(const float* A, int pa, const float* W, int pw, int M, int N, int K, int r0, int rs, int c0, int cs, float (&acc)[TM][TN]) {
  const float* a[TM];
  const float* w[TN];
#pragma unroll
  for (int i = 0; i < TM; ++i) a[i] = A + min(r0 + i * rs, M - 1) * pa;
#pragma unroll
  for (int j = 0; j < TN; ++j) w[j] = W + min(c0 + j * cs, N - 1) * pw;
  if constexpr (PACKED) {
    ptx::f32x2 s[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) s[i][j] = 0ull;
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
      ulonglong2 av[TM], wv[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const ulonglong2*>(a[i] + k);
#pragma unroll
      for (int j = 0; j < TN; ++j) wv[j] = *reinterpret_cast<const ulonglong2*>(w[j] + k);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) s[i][j] = ptx::fma2(av[i].y, wv[j].y, ptx::fma2(av[i].x, wv[j].x, s[i][j]));
    }
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        float lo, hi;
        ptx::unpack2(s[i][j], lo, hi);
        acc[i][j] = lo + hi;
      }
  } else {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
#pragma unroll 1
    for (int k = 0; k < K; k += 4) {
      float4 av[TM], wv[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const float4*>(a[i] + k);
#pragma unroll
      for (int j = 0; j < TN; ++j) wv[j] = *reinterpret_cast<const float4*>(w[j] + k);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j)
          acc[i][j] = fmaf(av[i].w, wv[j].w, fmaf(av[i].z, wv[j].z, fmaf(av[i].y, wv[j].y, fmaf(av[i].x, wv[j].x, acc[i][j]))));
    }
  }
}
// out(r, c) = sum_k A[r][k] W[c][k] for r < M, c < N; epi(r, c, value)
template <int TM, int TN, typename Epi>
__device__ __forceinline__ void tile_gemm(const float* A, int pa, const float* W, int pw, int M, int N, int K, Epi epi) {
  const int mt = (M + TM - 1) / TM, nt = (N + TN - 1) / TN, n = warp_tiles(mt, nt);
  for (int w = threadIdx.x >> 5; w < n; w += kThreads / 32) {
    const WarpTile t(w, mt, nt);
    float acc[TM][TN];
    tile_dot<TM, TN>(A, pa, W, pw, M, N, K, t.tm, mt, t.tn, nt, acc);
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j)
        if (t.in && t.tm + i * mt < M && t.tn + j * nt < N) epi(t.tm + i * mt, t.tn + j * nt, acc[i][j]);
  }
}

// rows [0, n) of `vpr.d` 16-byte vectors from global memory (row r at src(r)) into shared memory with pitch `pitch`
template <int THREADS, typename Src>
__device__ __forceinline__ void load_rows(float* dst, int pitch, int n, const FastDiv& vpr, Src src) {
#pragma unroll 1                                       // (runs once: the unrolled form costs more in instruction fetches)
  for (int i = threadIdx.x; i < n * (int)vpr.d; i += THREADS) {
    const int r = (int)fd_div((uint32_t)i, vpr), v = i - r * (int)vpr.d;
    ptx::cp_async16(dst + r * pitch + v * 4, src(r) + v * 4);
  }
}
template <int LANES>
__device__ __forceinline__ float lanes_sum(float v) {
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}
// LayerNorm of `n` rows in place, LANES lanes per row (mean, then centred squares); gamma and beta in shared memory
template <int THREADS, int LANES>
__device__ __forceinline__ void norm_rows(float* x, int pitch, int n, int C, const float* g, const float* b, float eps) {
  const int l = threadIdx.x & (LANES - 1);
  const float inv = 1.0f / (float)C;
  for (int r0 = 0; r0 < n; r0 += THREADS / LANES) {    // (all lanes of a warp run all rounds: shuffles)
    const int r = r0 + (int)threadIdx.x / LANES;
    const bool in = r < n;
    float4* p = reinterpret_cast<float4*>(x + min(r, n - 1) * pitch);
    const int nv = C / 4;
    float s = 0.f;
#pragma unroll 2
    for (int c = l; c < nv; c += LANES) { const float4 v = p[c]; s += (v.x + v.y) + (v.z + v.w); }
    const float mean = lanes_sum<LANES>(s) * inv;
    float q = 0.f;
#pragma unroll 2
    for (int c = l; c < nv; c += LANES) {
      const float4 v = p[c];
      const float a0 = v.x - mean, a1 = v.y - mean, a2 = v.z - mean, a3 = v.w - mean;
      q += fmaf(a0, a0, a1 * a1) + fmaf(a2, a2, a3 * a3);
    }
    const float rstd = rsqrtf(lanes_sum<LANES>(q) * inv + eps);
    if (in)
#pragma unroll 2
      for (int c = l; c < nv; c += LANES) {
        const float4 v = p[c], gv = reinterpret_cast<const float4*>(g)[c], bv = reinterpret_cast<const float4*>(b)[c];
        p[c] = make_float4(fmaf((v.x - mean) * rstd, gv.x, bv.x), fmaf((v.y - mean) * rstd, gv.y, bv.y), fmaf((v.z - mean) * rstd, gv.z, bv.z),
                           fmaf((v.w - mean) * rstd, gv.w, bv.w));
      }
  }
}

struct AttnF32Args {
  const float *x, *ln_g, *ln_b, *w_qkv, *b_qkv, *table, *w_proj, *b_proj;
  float* y;
  int C, heads, d, T, ws, shift, H, W, nWw, win_per_img;
  int parts, part_rows;                                // CTAs of a window and head, and the tokens of each (the last one has the rest)
  float eps, scale;
  FastDiv fd_vpr, fd_d, fd_ws;                         // vectors of a row, head dimension, window
  int tp;                                              // pitch of P and of v transposed: T rounded up to an odd number of vectors
  DevMap rowmap;
};

// q, k and v of one head: a TM x TN tile a thread
template <int TM, int TN, bool PACKED, bool PARTS>
__device__ __forceinline__ void qkv_phase(const AttnF32Args& g, const float* xs, int pc, const float* wq, const float* bq, float* q, float* k, float* vt, int pd,
                                          int row0, int rows, int h) {
  const int d = g.d, mt = (rows + TM - 1) / TM, nt = 3 * d / TN;
  const WarpTile t((int)threadIdx.x >> 5, mt, nt);
  float acc[TM][TN];
  if (t.in) tile_dot<TM, TN, PACKED>(xs, pc, wq, pc, rows, 3 * d, g.C, t.tm, mt, t.tn, nt, acc);
  if (PARTS) ptx::cluster_wait();                      // (every part has zeroed its v)
  if (!t.in) return;
#pragma unroll
  for (int j = 0; j < TN; ++j) {
    const int c = t.tn + j * nt, which = c < d ? 0 : c < 2 * d ? 1 : 2, e = c - which * d;
    const float b = bq[c], sc = which == 0 ? g.scale : 1.0f;
    float* dst = which == 0 ? q + t.tm * pd + e : which == 1 ? k + (row0 + t.tm) * pd + e : vt + e * g.tp + row0 + t.tm;
    const int step = (which == 2 ? 1 : pd) * mt;
    if (!PARTS || which == 0) {
#pragma unroll
      for (int i = 0; i < TM; ++i)
        if (t.tm + i * mt < rows) dst[i * step] = (acc[i][j] + b) * sc;
    } else {                                           // keys and values: into every part's memory
#pragma unroll 1
      for (int z = 0; z < g.parts; ++z) {
        const uint32_t peer = ptx::mapa(ptx::smem_u32(dst), (uint32_t)(z * g.heads + h));
#pragma unroll
        for (int i = 0; i < TM; ++i)
          if (t.tm + i * mt < rows) ptx::st_cluster_f32(peer + (uint32_t)(i * step) * 4u, acc[i][j] + b);
      }
    }
  }
}

// THREADS: 256 up to 32 tokens, else 512: one output tile a thread in every phase.  ALONE: no more CTAs than SMs, so a thread may have all
// the registers it can use.
// PARTS: the tokens of a window are shared out as well.
template <int THREADS, bool ALONE, bool PARTS>
__global__ void __launch_bounds__(THREADS, ALONE ? 1 : THREADS == 256 ? 3 : 2) swin_attn_f32_kernel(const __grid_constant__ AttnF32Args g) {
  extern __shared__ __align__(16) float sm[];
  const int C = g.C, d = g.d, T = g.T, pc = C + 4, pd = d + 4, tp = g.tp;
  float* xs = sm;                                      // [T][C]: the normalised rows, later every head's output
  float* wq = xs + T * pc;                             // [3 d][C]
  float* wp = wq + 3 * d * pc;                         // [d][C]
  float* q = wp + d * pc;                              // [T][d]
  float* k = q + T * pd;                               // [T][d]
  float* vt = k + T * pd;                              // [d][T], zero beyond T
  float* P = vt + d * tp;                              // [T][T], zero beyond T
  float* lng = P + T * tp;                             // gamma and beta [C], biases of q, k, v [3 d] and of the projection [d]
  float* lnb = lng + C;
  float* bq = lnb + C;
  float* bp = bq + 3 * d;
  const int nt = (2 * g.ws - 1) * (2 * g.ws - 1);
  float* tab = bp + d;                                 // the head's column of the bias table
  long long* offs = reinterpret_cast<long long*>(tab + ((nt + 3) & ~3));
  int* code = reinterpret_cast<int*>(offs + T);        // a token's place in the bias table (differences index it) and its region
  int* label = code + T;
  const int ctas = PARTS ? g.heads * g.parts : g.heads, cta = ctas > 1 ? (int)ptx::cluster_ctarank() : 0;
  const int z = PARTS ? cta / g.heads : 0, h = cta - z * g.heads;
  const int row0 = PARTS ? z * g.part_rows : 0, rows = PARTS ? min(g.part_rows, T - row0) : T;      // this CTA's tokens
  const int n = (int)blockIdx.x / ctas;                // window
  const int tid = threadIdx.x;

  // The head's weights as far as L2: they may still be written by the kernel before this one.  (A line per 32 floats of a head's rows,
  // which lie one behind the other.)
  for (int i = tid * 32; i < d * C; i += THREADS * 32) {
    for (int which = 0; which < 3; ++which) ptx::prefetch_l2(g.w_qkv + (size_t)(which * C + h * d) * C + i);
    ptx::prefetch_l2(g.w_proj + (size_t)h * d * C + i);
  }
  if (tid < T) {
    offs[tid] = devmap_eval(g.rowmap, (uint32_t)(n * T + tid));
    const int wl = n % g.win_per_img, wy = wl / g.nWw, wx = wl - wy * g.nWw;
    const int ty = (int)fd_div((uint32_t)tid, g.fd_ws), tx = tid - ty * g.ws;
    code[tid] = ty * (2 * g.ws - 1) + tx;
    label[tid] = g.shift > 0 ? region_label2(ty, tx, g.ws, wy, wx, g.H, g.W, g.shift) : 0;
  }
  for (int i = tid; i < d * tp; i += THREADS) vt[i] = 0.f;
  for (int i = tid; i < rows * tp; i += THREADS) P[i] = 0.f;
  if (PARTS) ptx::cluster_arrive();
  __syncthreads();
  pdl_wait();
  pdl_launch_dependents();
  load_rows<THREADS>(xs, pc, rows, g.fd_vpr, [&](int r) { return g.x + offs[row0 + r]; });
  for (int i = tid; i < C / 2; i += THREADS)
    ptx::cp_async16(lng + i * 4, (i < C / 4 ? g.ln_g : g.ln_b - C) + i * 4);
  ptx::cp_async_commit();
  // (rows of q, k, v and of the projection lie one behind the other in shared memory, and so do their biases)
  load_rows<THREADS>(wq, pc, 4 * d, g.fd_vpr, [&](int r) {
    const int which = (int)fd_div((uint32_t)r, g.fd_d), e = h * d + r - which * d;
    return which < 3 ? g.w_qkv + (size_t)(which * C + e) * C : g.w_proj + (size_t)e * C;
  });
  ptx::cp_async_commit();
  for (int i = tid; i < 4 * d + nt; i += THREADS) {
    const int which = (int)fd_div((uint32_t)i, g.fd_d), e = h * d + i - which * d;
    bq[i] = i >= 4 * d ? g.table[(i - 4 * d) * g.heads + h] : which < 3 ? g.b_qkv[which * C + e] : g.b_proj[e];
  }
  ptx::cp_async_wait<1>();
  __syncthreads();
  norm_rows<THREADS, 8>(xs, pc, rows, C, lng, lnb, g.eps);
  ptx::cp_async_wait<0>();
  __syncthreads();
  // the smallest tile that gives no warp two (T at most 64 and d 16 or 32: at most 6 and 12 of the largest)
  const int t2 = (rows + 1) / 2;
  if (warp_tiles(t2, 3 * d / 2) <= THREADS / 32) qkv_phase<2, 2, true, PARTS>(g, xs, pc, wq, bq, q, k, vt, pd, row0, rows, h);
  else if (warp_tiles(t2, 3 * d / 4) <= THREADS / 32) qkv_phase<2, 4, true, PARTS>(g, xs, pc, wq, bq, q, k, vt, pd, row0, rows, h);
  else qkv_phase<4, 4, ALONE, PARTS>(g, xs, pc, wq, bq, q, k, vt, pd, row0, rows, h);
  if (PARTS) { __syncwarp(); ptx::cluster_sync(); } else __syncthreads();
  {
    const int nk = (T + 3) / 4;
    const WarpTile t(tid >> 5, t2, nk);
    if (t.in) {
      float acc[2][4];
      tile_dot<2, 4>(q, pd, k, pd, rows, T, d, t.tm, t2, t.tn, nk, acc);
      const int i0 = t.tm, i1 = min(i0 + t2, rows - 1), mid = (g.ws - 1) * 2 * g.ws;
      const int c0 = code[row0 + i0] + mid, c1 = code[row0 + i1] + mid, l0 = label[row0 + i0], l1 = label[row0 + i1];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int col = t.tn + j * nk;
        if (col < T) {
          const int cc = code[col], lc = label[col];
          P[i0 * tp + col] = acc[0][j] + tab[c0 - cc] - (l0 != lc ? 100.f : 0.f);
          if (i0 + t2 < rows) P[i1 * tp + col] = acc[1][j] + tab[c1 - cc] - (l1 != lc ? 100.f : 0.f);
        }
      }
    }
  }
  __syncthreads();
  {                                                    // softmax: eight lanes per row, eight keys per lane
    const int r = min(tid >> 3, rows - 1), l = tid & 7;
    float* p = P + r * tp;
    float v[8], m = -INFINITY;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      v[j] = l + 8 * j < T ? p[l + 8 * j] : -INFINITY;
      m = fmaxf(m, v[j]);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      v[j] = l + 8 * j < T ? expf(v[j] - m) : 0.f;
      s += v[j];
    }
    const float inv = 1.0f / lanes_sum<8>(s);
    if ((tid >> 3) < rows)
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (l + 8 * j < T) p[l + 8 * j] = v[j] * inv;
  }
  __syncthreads();
  // o of this head goes straight into every CTA's row buffer: column h d + c of all of them.  A thread has the same two rows and two
  // columns of it and of the projection.
  const WarpTile t(tid >> 5, t2, d / 2);
  const int c0 = t.tn, c1 = c0 + d / 2, r0 = t.tm, r1 = r0 + t2;
  const bool in0 = t.in, in1 = t.in && r1 < rows;
  float acc[2][2], res[2][2] = {};
  const long long o0 = in0 ? offs[row0 + r0] + h * d : 0, o1 = in1 ? offs[row0 + r1] + h * d : 0;
  if (in0) { res[0][0] = g.x[o0 + c0]; res[0][1] = g.x[o0 + c1]; }
  if (in1) { res[1][0] = g.x[o1 + c0]; res[1][1] = g.x[o1 + c1]; }
  const bool meet = g.heads > 1 && !PARTS;       // everyone has read its normalised rows (where parts met after q, k and v, it has)
  if (meet) ptx::cluster_arrive();
  if (in0) tile_dot<2, 2>(P, tp, vt, tp, rows, d, (T + 3) & ~3, r0, t2, c0, d / 2, acc);
  if (meet) ptx::cluster_wait();
  if (in0) {
    const uint32_t xa = ptx::smem_u32(xs), o = (uint32_t)(r0 * pc + h * d + c0) * 4u;
#pragma unroll 1
    for (int r = 0; r < g.heads; ++r) {
      const uint32_t peer = (g.heads > 1 ? ptx::mapa(xa, (uint32_t)(z * g.heads + r)) : xa) + o;
      ptx::st_cluster_f32(peer, acc[0][0]);
      ptx::st_cluster_f32(peer + d * 2, acc[0][1]);
      if (in1) {
        ptx::st_cluster_f32(peer + t2 * pc * 4, acc[1][0]);
        ptx::st_cluster_f32(peer + t2 * pc * 4 + d * 2, acc[1][1]);
      }
    }
  }
  if (g.heads > 1) { __syncwarp(); ptx::cluster_sync(); } else __syncthreads();
  if (in0) {
    tile_dot<2, 2>(xs, pc, wp, pc, rows, d, C, r0, t2, c0, d / 2, acc);
    g.y[o0 + c0] = acc[0][0] + bp[c0] + res[0][0];
    g.y[o0 + c1] = acc[0][1] + bp[c1] + res[0][1];
    if (in1) {
      g.y[o1 + c0] = acc[1][0] + bp[c0] + res[1][0];
      g.y[o1 + c1] = acc[1][1] + bp[c1] + res[1][1];
    }
  }
}

struct MlpF32Args {
  const float *x, *ln_g, *ln_b, *w1, *b1, *w2, *b2;
  float* y;
  int M, C, hidden, slice, splits;
  float eps;
  FastDiv fd_vpr, fd_vps, fd_C;                        // vectors of a row, of a slice; floats of a row
};
constexpr int kMlpRows = 16;

__global__ void __launch_bounds__(kThreads) swin_mlp_f32_kernel(const MlpF32Args g) {
  extern __shared__ __align__(16) float sm[];
  const int C = g.C, hs = g.slice, pc = C + 4, ph = hs + 4;
  float* xs = sm;                                      // [16][C]
  float* w1 = xs + kMlpRows * pc;                      // [slice][C]
  float* w2 = w1 + hs * pc;                            // [C][slice]
  float* hid = w2 + C * ph;                            // [16][slice]
  float* part = hid + kMlpRows * ph;                   // [16][C]: this slice's share of fc2
  float* lng = part + kMlpRows * C;                    // gamma, beta, the second bias [C], the first [slice]
  float* lnb = lng + C;
  float* b2 = lnb + C;
  float* b1 = b2 + C;
  const int rank = g.splits > 1 ? (int)ptx::cluster_ctarank() : 0;
  const int m0 = (int)blockIdx.x / g.splits * kMlpRows, rows = min(kMlpRows, g.M - m0);
  load_rows<kThreads>(w1, pc, hs, g.fd_vpr, [&](int r) { return g.w1 + (size_t)(rank * hs + r) * C; });
  load_rows<kThreads>(w2, ph, C, g.fd_vps, [&](int r) { return g.w2 + (size_t)r * g.hidden + rank * hs; });
  const int C4 = C / 4, h4 = hs / 4;
  for (int i = threadIdx.x; i < 3 * C4 + h4; i += kThreads)
    ptx::cp_async16(lng + i * 4, (i < C4 ? g.ln_g : i < 2 * C4 ? g.ln_b - C : i < 3 * C4 ? g.b2 - 2 * C : g.b1 + rank * hs - 3 * C) + i * 4);
  ptx::cp_async_commit();
  pdl_wait();
  pdl_launch_dependents();
  load_rows<kThreads>(xs, pc, rows, g.fd_vpr, [&](int r) { return g.x + (size_t)(m0 + r) * C; });
  ptx::cp_async_commit();
  ptx::cp_async_wait<0>();
  __syncthreads();
  norm_rows<kThreads, 16>(xs, pc, rows, C, lng, lnb, g.eps);
  __syncthreads();
  // (eight outputs a thread, but for the narrowest: latency is all they cost)
  auto gelu_out = [&](int r, int c, float v) { hid[r * ph + c] = gelu_erf(v + b1[c]); };
  if (hs >= 48) tile_gemm<2, 4>(xs, pc, w1, pc, rows, hs, C, gelu_out);
  else tile_gemm<1, 2>(xs, pc, w1, pc, rows, hs, C, gelu_out);
  __syncthreads();
  auto part_out = [&](int r, int c, float v) { part[r * C + c] = v; };
  if (C >= 48) tile_gemm<2, 4>(hid, ph, w2, ph, rows, C, hs, part_out);
  else tile_gemm<1, 2>(hid, ph, w2, ph, rows, C, hs, part_out);
  if (g.splits > 1) ptx::cluster_sync(); else __syncthreads();
  const int ra = rows * rank / g.splits, rb = rows * (rank + 1) / g.splits;            // this CTA finishes a share of the rows
  for (int i = ra * C + (int)threadIdx.x; i < rb * C; i += kThreads) {
    float v = 0.f;
    if (g.splits > 1) {
      float t[kMaxCluster];
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r) t[r] = r < g.splits ? ptx::ld_cluster_f32(ptx::mapa(ptx::smem_u32(part + i), (uint32_t)r)) : 0.f;
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r) v += t[r];
    } else {
      v = part[i];
    }
    const size_t o = (size_t)m0 * C + i;
    g.y[o] = v + b2[i - (int)fd_div((uint32_t)i, g.fd_C) * C] + g.x[o];
  }
  if (g.splits > 1) ptx::cluster_sync();               // no CTA leaves while its share is still being read
}

// floats: n rounded up to an odd number of 16-byte vectors
int pitch_of(int n) { return (((n + 3) >> 2) | 1) << 2; }
size_t attn_f32_smem(int C, int d, int T, int ws) {
  const size_t pc = C + 4, pd = d + 4, tp = pitch_of(T), nt = ((2 * ws - 1) * (2 * ws - 1) + 3) & ~3;
  return (T * pc + 4 * d * pc + 2 * T * pd + d * tp + T * tp + 2 * C + 4 * d + nt) * 4 + (size_t)T * 16;
}
size_t mlp_f32_smem(int C, int slice) {
  return ((size_t)kMlpRows * (C + 4) + (size_t)slice * (C + 4) + (size_t)C * (slice + 4) + (size_t)kMlpRows * (slice + 4) + (size_t)kMlpRows * C + 3 * C + slice) * 4;
}
constexpr size_t kMaxSmem = 227 * 1024;
// the fewest slices of the hidden features (4 or 8) that fit
int mlp_f32_splits(int C, int hidden) {
  for (int s = 4; s <= kMaxCluster; s *= 2)
    if (hidden % (4 * s) == 0 && mlp_f32_smem(C, hidden / s) <= kMaxSmem) return s;
  return 0;
}

}  // namespace

bool swin_attn_f32_supported(int C, int heads, int window) {
  const int d = C / heads, T = window * window;
  return heads <= kMaxCluster && C % 4 == 0 && (d == 16 || d == 32) && T <= 64 && attn_f32_smem(C, d, T, window) <= kMaxSmem;
}
bool swin_mlp_f32_supported(int C, long long hidden) { return C % 4 == 0 && hidden < (1 << 20) && mlp_f32_splits(C, (int)hidden) > 0; }

// Every cluster of sixteen rows loads the weights and walks through its phases on its own, about 0.04 us of a full chip beside its
// products; the tiled kernels spend next to nothing per row but run their products at less than half the rate, and their launches cost
// more.  Both estimates in us, fitted to (cluster / LayerNorm and two linears, hidden = 4 C): 784 x 32 8.2 / 10.5, 3136 x 32 14.4 / 16.2,
// 6272 x 32 25.6 / 24.5, 25088 x 32 86 / 70, 784 x 48 9.4 / 14.3, 25088 x 48 114 / 143, 25088 x 64 133 / 252, 25088 x 96 265 / 553,
// 25088 x 192 1486 / 2165; hidden = C: 1568 x 16 6.2 / 8.6, 3136 x 16 11.3 / 8.1, 25088 x 16 63 / 10, 3136 x 64 14.4 / 16.3, 25088 x 64 84 / 70.
// (Within an eighth of one another the separate kernels keep the block.)
bool swin_mlp_f32_wins(long long M, int C, long long hidden) {
  if (!swin_mlp_f32_supported(C, hidden)) return false;
  const double groups = (double)((M + kMlpRows - 1) / kMlpRows), mflop = 4e-6 * kMlpRows * C * (double)hidden;
  return 4.5 + groups * (0.044 + mflop / 17.0) < 8.0 + groups * (mflop / 6.4);
}

int launch_swin_attn_f32(const smartmem_swin_params_t& p, const DevMap& rowmap, const void* x, void* y, cudaStream_t st) {
  AttnF32Args g;
  memset(&g, 0, sizeof(g));
  g.x = (const float*)x; g.y = (float*)y;
  g.ln_g = (const float*)p.ln1_g; g.ln_b = (const float*)p.ln1_b; g.w_qkv = (const float*)p.w_qkv; g.b_qkv = (const float*)p.b_qkv;
  g.table = (const float*)p.rel_bias_table; g.w_proj = (const float*)p.w_proj; g.b_proj = (const float*)p.b_proj;
  g.C = p.C; g.heads = p.heads; g.d = p.C / p.heads; g.ws = p.window; g.T = p.window * p.window; g.shift = p.shift; g.H = p.H; g.W = p.W;
  g.nWw = p.W / p.window; g.win_per_img = g.nWw * (p.H / p.window);
  g.eps = p.ln_eps; g.scale = 1.0f / sqrtf((float)g.d);
  g.tp = pitch_of(g.T);
  g.fd_vpr = make_fastdiv((uint32_t)g.C / 4);
  g.fd_d = make_fastdiv((uint32_t)g.d);
  g.fd_ws = make_fastdiv((uint32_t)g.ws);
  g.rowmap = rowmap;
  long long ctas = (long long)p.B * g.win_per_img * p.heads;
  // Few windows of more than 32 tokens: two or four CTAs share a window and head.  Us, one -> two -> four: 2 CTAs ([1,7,7,64], heads of 32) 13.4 ->
  // 10.2 -> 8.8, 8 ([2,14,14,32]) 10.3 -> 8.3 -> 7.3, 27 ([3,21,21,32]) 10.3 -> 8.3 -> 8.6, 54 ([3,21,21,64]) 13.5 -> 11.7 -> 13.8; 81 ([3,21,21,96]) 17.2 ->
  // 20.3; heads of 16 27 ([3,21,7,48]) 9.7 -> 7.9, 36 ([3,21,14,32] with its MLP half) 13.2 -> 13.6; windows of 16 tokens are alike to 24 CTAs and lose
  // beyond.
  g.parts = 1;
  if (g.T > 32) {
    if (4 * p.heads <= kMaxCluster && 4 * ctas <= tc_sm_count() / 2) g.parts = 4;
    else if (2 * p.heads <= kMaxCluster && 2 * ctas <= (g.d == 32 ? tc_cluster_ctas(2 * p.heads) : tc_sm_count() * 2 / 5)) g.parts = 2;
  }
  g.part_rows = (g.T + g.parts - 1) / g.parts;
  ctas *= g.parts;
  if (ctas >= (1ll << 31) || (long long)p.B * p.H * p.W >= (1ll << 31)) return SMARTMEM_ERR_UNSUPPORTED;
  const size_t smem = attn_f32_smem(g.C, g.d, g.T, g.ws);
  const bool alone = ctas <= tc_sm_count();
  auto kernel = g.T <= 32 ? (alone ? swin_attn_f32_kernel<256, true, false> : swin_attn_f32_kernel<256, false, false>)
                : g.parts > 1 ? swin_attn_f32_kernel<512, true, true>
                              : (alone ? swin_attn_f32_kernel<512, true, false> : swin_attn_f32_kernel<512, false, false>);
  if (ensure_max_dynamic_smem((const void*)kernel, (int)kMaxSmem) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("swin_attn_f32", st);
  if (launch_pdl_cluster(kernel, dim3((unsigned)ctas), dim3(g.T <= 32 ? 256 : 512), smem, st, (unsigned)(p.heads * g.parts), g) != cudaSuccess) return SMARTMEM_ERR_CUDA;
  count_launch();
  return SMARTMEM_OK;
}

int launch_swin_mlp_f32(const smartmem_swin_params_t& p, const void* x, void* y, long long M, bool settled, cudaStream_t st) {
  MlpF32Args g;
  memset(&g, 0, sizeof(g));
  g.x = (const float*)x; g.y = (float*)y;
  g.ln_g = (const float*)p.ln2_g; g.ln_b = (const float*)p.ln2_b; g.w1 = (const float*)p.w_fc1; g.b1 = (const float*)p.b_fc1;
  g.w2 = (const float*)p.w_fc2; g.b2 = (const float*)p.b_fc2;
  g.M = (int)M; g.C = p.C; g.hidden = p.C * p.mlp_ratio; g.eps = p.ln_eps;
  g.splits = mlp_f32_splits(g.C, g.hidden);
  if (g.splits == 0) return SMARTMEM_ERR_UNSUPPORTED;
  // Few rows: twice the slices, half of the products a CTA (us of a block, four -> eight: 144 rows of 96 17.1 -> 15.9, 144 of 64 13.3 -> 12.2; 196 of 96
  // 19.9 -> 20.4, 1323 of 64 21.0 -> 25.7).
  const long long groups = (M + kMlpRows - 1) / kMlpRows;
  if (g.splits == 4 && g.hidden % (4 * kMaxCluster) == 0 && groups * kMaxCluster <= tc_sm_count() / 2) g.splits = kMaxCluster;
  g.slice = g.hidden / g.splits;
  g.fd_vpr = make_fastdiv((uint32_t)g.C / 4);
  g.fd_vps = make_fastdiv((uint32_t)g.slice / 4);
  g.fd_C = make_fastdiv((uint32_t)g.C);
  const long long ctas = groups * g.splits;
  if (ctas >= (1ll << 31)) return SMARTMEM_ERR_UNSUPPORTED;
  const size_t smem = mlp_f32_smem(g.C, g.slice);
  if (ensure_max_dynamic_smem((const void*)swin_mlp_f32_kernel, (int)kMaxSmem) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("swin_mlp_f32", st);
  if (launch_cluster(swin_mlp_f32_kernel, dim3((unsigned)ctas), dim3(kThreads), smem, st, (unsigned)g.splits, settled, g) != cudaSuccess) return SMARTMEM_ERR_CUDA;
  count_launch();
  return SMARTMEM_OK;
}

}  // namespace smartmem
