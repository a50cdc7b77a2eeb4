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
//   * MLP: sixteen rows per cluster, a slice of the hidden features per CTA; the partial results of fc2 are added through
//     distributed shared memory in the order of the CTAs.
// Operands lie in shared memory with rows of K + 4 floats (an odd number of 16-byte vectors: eight lanes on eight rows hit
// distinct banks), a thread computes TM x TN outputs with 16-byte reads along K.
// [1,8,8,32] attention half (4 windows, 2 heads), us of a stream of calls: four kernels 16.7, one 9.4 (8.9 with the weights fetched
// before the dependency wait, which nothing in front of the call would order).
#include <cstring>

#include "attn.cuh"
#include "gemm_tc.cuh"
#include "ptx.cuh"

namespace smartmem {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxCluster = 8;

// out(r, c) = sum_k A[r][k] W[c][k] for r < M, c < N; K a multiple of 4; epi(r, c, value)
template <int TM, int TN, typename Epi>
__device__ __forceinline__ void tile_gemm(const float* A, int pa, const float* W, int pw, int M, int N, int K, Epi epi) {
  const int mt = (M + TM - 1) / TM, nt = (N + TN - 1) / TN;
  for (int idx = threadIdx.x; idx < mt * nt; idx += kThreads) {
    const int tm = idx / nt, tn = idx - tm * nt;
    const float* a[TM];
    const float* w[TN];
    float acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i) a[i] = A + min(tm * TM + i, M - 1) * pa;
#pragma unroll
    for (int j = 0; j < TN; ++j) w[j] = W + min(tn + j * nt, N - 1) * pw;      // (neighbouring lanes on neighbouring rows)
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
#pragma unroll 2
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
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j)
        if (tm * TM + i < M && tn + j * nt < N) epi(tm * TM + i, tn + j * nt, acc[i][j]);
  }
}
// four rows x four columns per thread where that still gives most threads a tile, else two x two
template <typename Epi>
__device__ __forceinline__ void gemm_any(const float* A, int pa, const float* W, int pw, int M, int N, int K, Epi epi) {
  if (M * N >= 16 * 160) tile_gemm<4, 4>(A, pa, W, pw, M, N, K, epi);
  else tile_gemm<2, 2>(A, pa, W, pw, M, N, K, epi);
}

// rows [0, n) of `vpr.d` 16-byte vectors from global memory (row r at src(r)) into shared memory with pitch `pitch`
template <typename Src>
__device__ __forceinline__ void load_rows(float* dst, int pitch, int n, const FastDiv& vpr, Src src) {
#pragma unroll 1                                       // (runs once: the unrolled form costs more in instruction fetches)
  for (int i = threadIdx.x; i < n * (int)vpr.d; i += kThreads) {
    const int r = (int)fd_div((uint32_t)i, vpr), v = i - r * (int)vpr.d;
    ptx::cp_async16(dst + r * pitch + v * 4, src(r) + v * 4);
  }
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}
// LayerNorm of `n` rows in place (a warp per row; mean, then centred squares)
__device__ __forceinline__ void norm_rows(float* x, int pitch, int n, int C, const float* __restrict__ g, const float* __restrict__ b, float eps) {
  const int lane = threadIdx.x & 31;
  for (int r = threadIdx.x >> 5; r < n; r += kThreads / 32) {
    float* p = x + r * pitch;
    float s = 0.f;
    for (int c = lane; c < C; c += 32) s += p[c];
    const float mean = warp_sum(s) / (float)C;
    float q = 0.f;
    for (int c = lane; c < C; c += 32) q = fmaf(p[c] - mean, p[c] - mean, q);
    const float rstd = rsqrtf(warp_sum(q) / (float)C + eps);
    for (int c = lane; c < C; c += 32) p[c] = fmaf((p[c] - mean) * rstd, g[c], b[c]);
  }
}

struct AttnF32Args {
  const float *x, *ln_g, *ln_b, *w_qkv, *b_qkv, *table, *w_proj, *b_proj;
  float* y;
  int C, heads, d, T, ws, shift, H, W, nWw, win_per_img;
  float eps, scale;
  FastDiv fd_vpr, fd_d;                                // vectors of a row, head dimension
  int tp;                                              // pitch of P and of v transposed: T rounded up to an odd number of vectors
  DevMap rowmap;
};

__global__ void __launch_bounds__(kThreads) swin_attn_f32_kernel(const __grid_constant__ AttnF32Args g) {
  extern __shared__ __align__(16) float sm[];
  const int C = g.C, d = g.d, T = g.T, pc = C + 4, pd = d + 4, tp = g.tp;
  float* xs = sm;                                      // [T][C]: the normalised rows, later every head's output
  float* wq = xs + T * pc;                             // [3 d][C]
  float* wp = wq + 3 * d * pc;                         // [d][C]
  float* q = wp + d * pc;                              // [T][d]
  float* k = q + T * pd;                               // [T][d]
  float* vt = k + T * pd;                              // [d][T], zero beyond T
  float* P = vt + d * tp;                              // [T][T], zero beyond T
  float* tab = P + T * tp;                             // the head's column of the bias table
  long long* offs = reinterpret_cast<long long*>(tab + (((2 * g.ws - 1) * (2 * g.ws - 1) + 3) & ~3));
  const int h = g.heads > 1 ? (int)ptx::cluster_ctarank() : 0;
  const int n = (int)blockIdx.x / g.heads;             // window
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // The head's weights as far as L2: they may still be written by the kernel before this one.  (A line per 32 floats of a head's rows,
  // which lie one behind the other.)
  for (int i = tid * 32; i < d * C; i += kThreads * 32) {
    for (int which = 0; which < 3; ++which) ptx::prefetch_l2(g.w_qkv + (size_t)(which * C + h * d) * C + i);
    ptx::prefetch_l2(g.w_proj + (size_t)h * d * C + i);
  }
  for (int i = tid; i < T; i += kThreads) offs[i] = devmap_eval(g.rowmap, (uint32_t)(n * T + i));
  for (int i = tid; i < d * tp; i += kThreads) vt[i] = 0.f;
  for (int i = tid; i < T * tp; i += kThreads) P[i] = 0.f;
  __syncthreads();
  pdl_wait();
  pdl_launch_dependents();
  load_rows(xs, pc, T, g.fd_vpr, [&](int r) { return g.x + offs[r]; });
  // (rows of q, k, v and of the projection lie one behind the other in shared memory)
  load_rows(wq, pc, 4 * d, g.fd_vpr, [&](int r) {
    const int which = (int)fd_div((uint32_t)r, g.fd_d), e = h * d + r - which * d;
    return which < 3 ? g.w_qkv + (size_t)(which * C + e) * C : g.w_proj + (size_t)e * C;
  });
  ptx::cp_async_commit();
  const int nt = (2 * g.ws - 1) * (2 * g.ws - 1);
  for (int i = tid; i < nt; i += kThreads) tab[i] = g.table[i * g.heads + h];
  ptx::cp_async_wait<0>();
  __syncthreads();
  norm_rows(xs, pc, T, C, g.ln_g, g.ln_b, g.eps);
  __syncthreads();
  gemm_any(xs, pc, wq, pc, T, 3 * d, C, [&](int r, int c, float v) {
    const int which = c / d, e = c - which * d;
    v += g.b_qkv[which * C + h * d + e];
    if (which == 0) q[r * pd + e] = v * g.scale;
    else if (which == 1) k[r * pd + e] = v;
    else vt[e * tp + r] = v;
  });
  __syncthreads();
  const int wl = n % g.win_per_img, wy = wl / g.nWw, wx = wl - wy * g.nWw;
  gemm_any(q, pd, k, pd, T, T, d, [&](int i, int j, float s) {
    const int ty = i / g.ws, tx = i - ty * g.ws, sy = j / g.ws, sx = j - sy * g.ws;
    s += tab[(ty - sy + g.ws - 1) * (2 * g.ws - 1) + tx - sx + g.ws - 1];
    if (g.shift > 0 && region_label2(ty, tx, g.ws, wy, wx, g.H, g.W, g.shift) != region_label2(sy, sx, g.ws, wy, wx, g.H, g.W, g.shift)) s -= 100.f;
    P[i * tp + j] = s;
  });
  __syncthreads();
  for (int i = warp; i < T; i += kThreads / 32) {      // softmax: a warp per row, at most two keys per lane
    float* p = P + i * tp;
    const float a = lane < T ? p[lane] : -INFINITY, b = lane + 32 < T ? p[lane + 32] : -INFINITY;
    float m = fmaxf(a, b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    const float ea = lane < T ? expf(a - m) : 0.f, eb = lane + 32 < T ? expf(b - m) : 0.f;
    const float inv = 1.0f / warp_sum(ea + eb);
    if (lane < T) p[lane] = ea * inv;
    if (lane + 32 < T) p[lane + 32] = eb * inv;
  }
  __syncthreads();
  // o of this head goes straight into every CTA's row buffer: column h d + c of all of them
  uint32_t peer[kMaxCluster];
#pragma unroll
  for (int r = 0; r < kMaxCluster; ++r) peer[r] = r < g.heads ? (g.heads > 1 ? ptx::mapa(ptx::smem_u32(xs), (uint32_t)r) : ptx::smem_u32(xs)) : 0u;
  if (g.heads > 1) ptx::cluster_sync();                // everyone has read its normalised rows
  gemm_any(P, tp, vt, tp, T, d, (T + 3) & ~3, [&](int i, int c, float v) {
    const uint32_t o = (uint32_t)(i * pc + h * d + c) * 4u;
#pragma unroll
    for (int r = 0; r < kMaxCluster; ++r)
      if (r < g.heads) ptx::st_cluster_f32(peer[r] + o, v);
  });
  if (g.heads > 1) ptx::cluster_sync(); else __syncthreads();
  gemm_any(xs, pc, wp, pc, T, d, C, [&](int i, int c, float v) {
    const long long o = offs[i] + h * d + c;
    g.y[o] = v + g.b_proj[h * d + c] + g.x[o];
  });
}

struct MlpF32Args {
  const float *x, *ln_g, *ln_b, *w1, *b1, *w2, *b2;
  float* y;
  int M, C, hidden, slice, splits;
  float eps;
  FastDiv fd_vpr, fd_vps;                              // vectors of a row, of a slice
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
  const int rank = g.splits > 1 ? (int)ptx::cluster_ctarank() : 0;
  const int m0 = (int)blockIdx.x / g.splits * kMlpRows, rows = min(kMlpRows, g.M - m0);
  load_rows(w1, pc, hs, g.fd_vpr, [&](int r) { return g.w1 + (size_t)(rank * hs + r) * C; });
  load_rows(w2, ph, C, g.fd_vps, [&](int r) { return g.w2 + (size_t)r * g.hidden + rank * hs; });
  ptx::cp_async_commit();
  pdl_wait();
  pdl_launch_dependents();
  load_rows(xs, pc, rows, g.fd_vpr, [&](int r) { return g.x + (size_t)(m0 + r) * C; });
  ptx::cp_async_commit();
  ptx::cp_async_wait<0>();
  __syncthreads();
  norm_rows(xs, pc, rows, C, g.ln_g, g.ln_b, g.eps);
  __syncthreads();
  tile_gemm<2, 4>(xs, pc, w1, pc, rows, hs, C, [&](int r, int c, float v) { hid[r * ph + c] = gelu_erf(v + g.b1[rank * hs + c]); });
  __syncthreads();
  tile_gemm<2, 4>(hid, ph, w2, ph, rows, C, hs, [&](int r, int c, float v) { part[r * C + c] = v; });
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
    g.y[o] = v + g.b2[i % C] + g.x[o];
  }
  if (g.splits > 1) ptx::cluster_sync();               // no CTA leaves while its share is still being read
}

// floats: n rounded up to an odd number of 16-byte vectors
int pitch_of(int n) { return (((n + 3) >> 2) | 1) << 2; }
size_t attn_f32_smem(int C, int d, int T, int ws) {
  const size_t pc = C + 4, pd = d + 4, tp = pitch_of(T), nt = ((2 * ws - 1) * (2 * ws - 1) + 3) & ~3;
  return (T * pc + 4 * d * pc + 2 * T * pd + d * tp + T * tp + nt) * 4 + (size_t)T * 8;
}
size_t mlp_f32_smem(int C, int slice) {
  return ((size_t)kMlpRows * (C + 4) + (size_t)slice * (C + 4) + (size_t)C * (slice + 4) + (size_t)kMlpRows * (slice + 4) + (size_t)kMlpRows * C) * 4;
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
  return heads <= kMaxCluster && C % 4 == 0 && d % 4 == 0 && T <= 64 && attn_f32_smem(C, d, T, window) <= kMaxSmem;
}
bool swin_mlp_f32_supported(int C, long long hidden) { return C % 4 == 0 && hidden < (1 << 20) && mlp_f32_splits(C, (int)hidden) > 0; }

// Every cluster of sixteen rows loads the weights and walks through its phases on its own, about 0.055 us of a full chip beside its
// products; the tiled kernels spend next to nothing per row but run their products at less than half the rate, and their launches cost
// more.  Both estimates in us, fitted to (cluster / LayerNorm and two linears, hidden = 4 C): 784 x 32 8.0 / 9.8, 3136 x 32 17.6 / 16.2,
// 25088 x 32 111 / 72, 784 x 48 12.0 / 15.6, 25088 x 48 141 / 147, 25088 x 64 161 / 257, 50176 x 96 554 / 1170, 12544 x 192 802 / 1088,
// 12544 x 256 1935 / 1929; hidden = C: 784 x 16 6.7 / 6.9, 25088 x 16 88 / 11, 25088 x 64 118 / 72.
bool swin_mlp_f32_wins(long long M, int C, long long hidden) {
  if (!swin_mlp_f32_supported(C, hidden)) return false;
  const double groups = (double)((M + kMlpRows - 1) / kMlpRows), mflop = 4e-6 * kMlpRows * C * (double)hidden;
  return 4.5 + groups * (0.055 + mflop / 15.0) < 8.0 + groups * (mflop / 6.4);
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
  g.rowmap = rowmap;
  const long long ctas = (long long)p.B * g.win_per_img * p.heads;
  if (ctas >= (1ll << 31) || (long long)p.B * p.H * p.W >= (1ll << 31)) return SMARTMEM_ERR_UNSUPPORTED;
  const size_t smem = attn_f32_smem(g.C, g.d, g.T, g.ws);
  if (ensure_max_dynamic_smem((const void*)swin_attn_f32_kernel, (int)kMaxSmem) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("swin_attn_f32", st);
  if (launch_pdl_cluster(swin_attn_f32_kernel, dim3((unsigned)ctas), dim3(kThreads), smem, st, (unsigned)p.heads, g) != cudaSuccess) return SMARTMEM_ERR_CUDA;
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
  g.slice = g.hidden / g.splits;
  g.fd_vpr = make_fastdiv((uint32_t)g.C / 4);
  g.fd_vps = make_fastdiv((uint32_t)g.slice / 4);
  const long long ctas = (M + kMlpRows - 1) / kMlpRows * g.splits;
  if (ctas >= (1ll << 31)) return SMARTMEM_ERR_UNSUPPORTED;
  const size_t smem = mlp_f32_smem(g.C, g.slice);
  if (ensure_max_dynamic_smem((const void*)swin_mlp_f32_kernel, (int)kMaxSmem) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("swin_mlp_f32", st);
  if (launch_cluster(swin_mlp_f32_kernel, dim3((unsigned)ctas), dim3(kThreads), smem, st, (unsigned)g.splits, settled, g) != cudaSuccess) return SMARTMEM_ERR_CUDA;
  count_launch();
  return SMARTMEM_OK;
}

}  // namespace smartmem
