// smartmem_attn_decode: one decode step of the decoder attention layer against a key/value cache.
//
// ELIMINATE: RMSNorm -> fused QKV GEMM whose epilogue rotates the q and k columns at position `pos`
// and stores the k and v columns of sequence b straight into row (b, pos) of the token-major caches
// [B, S_max, heads, D] (the Concat is the producer's store) -> decode attention reading head h of the
// cache as a strided slice (head split eliminated) and writing column h*D of [B, hidden] (head merge
// eliminated) -> output projection (+ residual).  No copy kernel.
// EXPLICIT: plain QKV GEMM, head-split copy to [3, B, heads, 1, D], stand-alone rotary pass, append copy
// into the per-head caches [B, heads, S_max, D], the same attention kernel on contiguous per-head
// tensors, output projection.
//
// The attention kernel is bandwidth work: every cached key and value is read once (2 * 256 bytes per
// position and head) and used for one 128-long dot product or one 128-wide axpy, so it runs on the
// ordinary FMA pipe with 16-byte loads; the tensor cores would multiply a one-row query tile.
#include <cuda_bf16.h>

#include <map>
#include <mutex>
#include <tuple>

#include "attn.cuh"
#include "chain_util.hpp"
#include "common.cuh"
#include "gemm_tc.cuh"
#include "ptx.cuh"

#define EXPORT extern "C" __attribute__((visibility("default")))

using namespace smartmem;

namespace {

constexpr int DH = 128;                  // head dimension
constexpr int DEC_WARPS = 8;             // 16 half-warps, four cached positions per half-warp and stage; and a producer warp
constexpr int DEC_THREADS = 32 * (DEC_WARPS + 1);
constexpr int DEC_GROUPS = 2 * DEC_WARPS;
constexpr int DEC_UNROLL = 4;
constexpr int DEC_STEP = DEC_GROUPS * DEC_UNROLL;             // positions per stage
constexpr int DEC_BOX = 32;                                   // rows per TMA box
constexpr int DEC_BOX_BYTES = DEC_BOX * DH * 2;
constexpr int DEC_STAGES = 3;
constexpr int DEC_STAGE_BYTES = 2 * DEC_STEP * DH * 2;        // keys, then values
constexpr int DEC_MAX_S = 16384;
constexpr int DEC_MAX_SPLIT = 8;         // portable cluster size

struct DecodeAttnArgs {
  const __nv_bfloat16* q;  long long q_sb, q_sh;          // q[b, h, :] = q + b*q_sb + h*q_sh
  const __nv_bfloat16* k;  const __nv_bfloat16* v;        // caches as [rows, pitch] matrices: position s of (b, h) is the
  int pitch, rows, rows_b, rows_h, cols_h;                // 128 elements at row b*rows_b + h*rows_h + s, column h*cols_h
  __nv_bfloat16* o;        long long o_sb, o_sh;
  int heads, units, S, split;                                    // S = positions attended (cached + the new one)
  float scale_log2e;                                      // head_dim^-1/2 * log2(e)
  int* status;
};

__device__ __forceinline__ void unpack8(const uint4& u, float (&f)[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    f[2 * j] = __uint_as_float(w[j] << 16);
    f[2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
  }
}

// A cluster of `split` CTAs per (sequence, head), each over a contiguous share of the positions.  What bounds it is bytes in
// flight: the rows come through a ring of three 32 KB stages (64 positions: four boxes of 32 rows of keys or values), two CTAs
// per SM.  (The same loop on loads to registers needs the L1 for its data in flight; behind a GEMM that leaves the SM
// configured for shared memory it ran a tenth slower.)  One pass: sixteen lanes share a row (16 bytes each), a half-warp
// scores four positions per stage and keeps its own running maximum, sum and weighted value sum (8 of the 128 output columns
// per lane); the half-warps' results are merged through shared memory, the CTAs' through distributed shared memory.  With one share per (sequence, head)
// and short contexts the grid is two CTAs per SM and each walks over several, its ring running on from one to the next (64 sequences of
// 100 positions, 32 heads: a CTA for each was 19 us of waves of one load latency each).
// Cached rows do not depend on the kernel before this one: only the stage that holds the new position waits for it.
__global__ void __launch_bounds__(DEC_THREADS, 2)
decode_attn_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ DecodeAttnArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* ring = smem_raw + ((128u - (ptx::smem_u32(smem_raw) & 127u)) & 127u);
  __shared__ uint64_t full[DEC_STAGES], empty[DEC_STAGES];
  __shared__ int abort_flag;
  __shared__ __align__(16) float part[2][DEC_WARPS][DH];                // (alternating: one barrier per unit of work)
  __shared__ float gm[2][DEC_WARPS], gl[2][DEC_WARPS];
  __shared__ float cta_o[DH], cta_ml[2];
  const int unit0 = (int)blockIdx.x / a.split, unit_step = (int)gridDim.x / a.split;
  const int rank = a.split > 1 ? (int)ptx::cluster_ctarank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
  const int l16 = tid & 15, grp = tid >> 4;
  const int s_lo = (int)((long long)a.S * rank / a.split), s_hi = (int)((long long)a.S * (rank + 1) / a.split);
  const int n_st = (s_hi - s_lo + DEC_STEP - 1) / DEC_STEP;
  if (tid == 0) {
    for (int i = 0; i < DEC_STAGES; ++i) {
      ptx::mbar_init(&full[i], 1);
      ptx::mbar_init(&empty[i], DEC_WARPS);
    }
    abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
  }
  __syncthreads();
  if (warp == DEC_WARPS) {
    bool ok = true, waited = false;
    uint32_t s = 0, ph = 1;
    int issued = 0;
    for (int unit = unit0; unit < a.units && ok; unit += unit_step) {
      const int b = unit / a.heads, h = unit - b * a.heads;
      const int row = b * a.rows_b + h * a.rows_h, col = h * a.cols_h;
      for (int i = 0; i < n_st; ++i) {
        const int p0 = s_lo + i * DEC_STEP, np = min(DEC_STEP, s_hi - p0), nbox = (np + DEC_BOX - 1) / DEC_BOX;
        ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(&empty[s], ph, &abort_flag, a.status) ? 1 : 0) != 0;
        if (!ok) break;
        if (!waited && p0 + nbox * DEC_BOX >= a.S) { pdl_wait(); waited = true; }
        if (ptx::elect_one()) {
          uint8_t* st = ring + s * DEC_STAGE_BYTES;
          ptx::mbar_expect_tx(&full[s], (uint32_t)nbox * 2u * DEC_BOX_BYTES);
          for (int x = 0; x < nbox; ++x) {
            ptx::tma_load_2d(st + x * DEC_BOX_BYTES, &tmK, &full[s], col, row + p0 + x * DEC_BOX);
            ptx::tma_load_2d(st + DEC_STAGE_BYTES / 2 + x * DEC_BOX_BYTES, &tmV, &full[s], col, row + p0 + x * DEC_BOX);
          }
        }
        __syncwarp();
        ++issued;
        if (++s == DEC_STAGES) { s = 0; ph ^= 1; }
      }
    }
    if (abort_flag && lane == 0) {                    // unwinding: copies in flight get a bounded chance to land
      for (int k = issued > DEC_STAGES ? issued - DEC_STAGES : 0; k < issued; ++k) {
        const unsigned long long t0 = ptx::globaltimer();
        while (!ptx::mbar_try_wait(&full[k % DEC_STAGES], (k / DEC_STAGES) & 1) && ptx::globaltimer() - t0 < 2000000ull) {
        }
      }
    }
    __syncwarp();
    pdl_wait();
  } else {
    pdl_wait();
    pdl_launch_dependents();
    auto q_of = [&](int unit) {
      const int b = unit / a.heads, h = unit - b * a.heads;
      return unit < a.units ? *reinterpret_cast<const uint4*>(a.q + b * a.q_sb + h * a.q_sh + l16 * 8) : make_uint4(0, 0, 0, 0);
    };
    uint4 q_next = q_of(unit0);
    uint32_t s = 0, ph = 0;
    int pb = 0;
    for (int unit = unit0; unit < a.units; unit += unit_step, pb ^= 1) {
      float qf[8];
      unpack8(q_next, qf);
      q_next = q_of(unit + unit_step);
#pragma unroll
      for (int j = 0; j < 8; ++j) qf[j] *= a.scale_log2e;
      float m = -INFINITY, l = 0.f, acc[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] = 0.f;
      for (int i = 0; i < n_st; ++i) {
        const int np = min(DEC_STEP, s_hi - (s_lo + i * DEC_STEP));
        if (!ptx::mbar_wait(&full[s], ph, &abort_flag, a.status)) break;
        const uint8_t* kt = ring + s * DEC_STAGE_BYTES + grp * (DH * 2) + l16 * 16;
        uint4 kv[DEC_UNROLL], vv[DEC_UNROLL];
#pragma unroll
        for (int u = 0; u < DEC_UNROLL; ++u) {
          kv[u] = *reinterpret_cast<const uint4*>(kt + u * (DEC_GROUPS * DH * 2));
          vv[u] = *reinterpret_cast<const uint4*>(kt + DEC_STAGE_BYTES / 2 + u * (DEC_GROUPS * DH * 2));
        }
        float d[DEC_UNROLL], vf[DEC_UNROLL][8];
#pragma unroll
        for (int u = 0; u < DEC_UNROLL; ++u) {
          float kf[8];
          unpack8(kv[u], kf);
          float d0 = 0.f, d1 = 0.f;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            d0 = fmaf(qf[2 * j], kf[2 * j], d0);
            d1 = fmaf(qf[2 * j + 1], kf[2 * j + 1], d1);
          }
          d[u] = d0 + d1;
          // rows past the share are whatever lay in the ring or behind the cache's last used row: never multiplied
          const bool in = grp + u * DEC_GROUPS < np;
          unpack8(in ? vv[u] : make_uint4(0, 0, 0, 0), vf[u]);
        }
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&empty[s]);
        if (++s == DEC_STAGES) { s = 0; ph ^= 1; }
#pragma unroll
        for (int x = 8; x >= 1; x >>= 1)
#pragma unroll
          for (int u = 0; u < DEC_UNROLL; ++u) d[u] += __shfl_xor_sync(0xFFFFFFFFu, d[u], x);
        float mn = m;
#pragma unroll
        for (int u = 0; u < DEC_UNROLL; ++u) {
          if (grp + u * DEC_GROUPS >= np) d[u] = -INFINITY;
          mn = fmaxf(mn, d[u]);
        }
        const float ref = mn == -INFINITY ? 0.f : mn;   // (a half-warp that has seen no position yet)
        const float c = exp2f(m - ref);
        l *= c;
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] *= c;
#pragma unroll
        for (int u = 0; u < DEC_UNROLL; ++u) {
          const float p = exp2f(d[u] - ref);
          l += p;
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[j] = fmaf(p, vf[u][j], acc[j]);
        }
        m = mn;
      }
      {                                                 // the warp's two halves
        const float mo = __shfl_xor_sync(0xFFFFFFFFu, m, 16), lo = __shfl_xor_sync(0xFFFFFFFFu, l, 16);
        const float mn = fmaxf(m, mo), ref = mn == -INFINITY ? 0.f : mn, w = exp2f(m - ref), wo = exp2f(mo - ref);
        l = l * w + lo * wo;
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = acc[j] * w + __shfl_xor_sync(0xFFFFFFFFu, acc[j], 16) * wo;
        m = mn;
      }
      if (lane < 16) {
        *reinterpret_cast<float4*>(&part[pb][warp][l16 * 8]) = make_float4(acc[0], acc[1], acc[2], acc[3]);
        *reinterpret_cast<float4*>(&part[pb][warp][l16 * 8 + 4]) = make_float4(acc[4], acc[5], acc[6], acc[7]);
      }
      if (lane == 0) { gm[pb][warp] = m; gl[pb][warp] = l; }
      asm volatile("bar.sync 1, %0;" ::"n"(32 * DEC_WARPS) : "memory");
      if (tid < DH) {
        float o = 0.f, lt = 0.f, mt = -INFINITY;
#pragma unroll
        for (int g = 0; g < DEC_WARPS; ++g) mt = fmaxf(mt, gm[pb][g]);
        const float ref = mt == -INFINITY ? 0.f : mt;
#pragma unroll
        for (int g = 0; g < DEC_WARPS; ++g) {
          const float w = exp2f(gm[pb][g] - ref);
          lt = fmaf(w, gl[pb][g], lt);
          o = fmaf(w, part[pb][g][tid], o);
        }
        if (a.split > 1) {                              // (one unit per CTA then)
          cta_o[tid] = o;
          if (tid == 0) { cta_ml[0] = mt; cta_ml[1] = lt; }
        } else {
          const int b = unit / a.heads, h = unit - b * a.heads;
          a.o[b * a.o_sb + h * a.o_sh + tid] = __float2bfloat16_rn(o / lt);
        }
      }
    }
  }
  if (a.split > 1) {
    __syncwarp();
    ptx::cluster_sync();
    if (rank == 0 && tid < DH) {
      float pm[DEC_MAX_SPLIT], pl[DEC_MAX_SPLIT], po[DEC_MAX_SPLIT];
#pragma unroll
      for (int r = 0; r < DEC_MAX_SPLIT; ++r) {
        pm[r] = -INFINITY;
        pl[r] = po[r] = 0.f;
        if (r < a.split) {
          const uint32_t ml = ptx::mapa(ptx::smem_u32(cta_ml), (uint32_t)r);
          pm[r] = ptx::ld_cluster_f32(ml);
          pl[r] = ptx::ld_cluster_f32(ml + 4);
          po[r] = ptx::ld_cluster_f32(ptx::mapa(ptx::smem_u32(cta_o + tid), (uint32_t)r));
        }
      }
      float mt = pm[0], o = 0.f, lt = 0.f;
#pragma unroll
      for (int r = 1; r < DEC_MAX_SPLIT; ++r) mt = fmaxf(mt, pm[r]);
#pragma unroll
      for (int r = 0; r < DEC_MAX_SPLIT; ++r) {
        const float w = exp2f(pm[r] - mt);
        lt = fmaf(w, pl[r], lt);
        o = fmaf(w, po[r], o);
      }
      const int b = unit0 / a.heads, h = unit0 - b * a.heads;
      a.o[b * a.o_sb + h * a.o_sh + tid] = __float2bfloat16_rn(o / lt);
    }
    __syncwarp();
    ptx::cluster_sync();                              // no CTA leaves while its results are still being read
  }
}

int launch_decode_attention(DecodeAttnArgs a, int B, cudaStream_t st) {
  if (a.S < 1 || a.S > DEC_MAX_S || B < 1 || a.heads < 1) return SMARTMEM_ERR_UNSUPPORTED;
  if ((long long)B * a.heads >= (1ll << 28)) return SMARTMEM_ERR_UNSUPPORTED;
  const long long strides[] = {a.q_sb, a.q_sh, a.o_sb, a.o_sh};
  for (long long s : strides)
    if (s % 8) return SMARTMEM_ERR_ALIGNMENT;
  const void* ptrs[] = {a.q, a.k, a.v, a.o};
  for (const void* p : ptrs)
    if ((uintptr_t)p & 15) return SMARTMEM_ERR_ALIGNMENT;
  CUtensorMap tk, tv;
  int rc = tc_encode_2d_plain(a.k, a.pitch, a.rows, a.pitch, DH, DEC_BOX, &tk);
  if (rc == SMARTMEM_OK) rc = tc_encode_2d_plain(a.v, a.pitch, a.rows, a.pitch, DH, DEC_BOX, &tv);
  if (rc != SMARTMEM_OK) return rc;
  a.status = device_status_ptr();
  if (!a.status) return SMARTMEM_ERR_CUDA;
  // Shares per (sequence, head): whichever reads the cache fastest.  A stage takes one CTA 0.54 us by latency and 32 KB / 6.5 TB/s times the CTAs
  // at work by bandwidth, and where the two are near one another it takes their root sum of squares (with the larger of them 128 CTAs, one per
  // SM, looked as good as 256: 8 x 7386 positions of 16 heads 101 us in one share, 86 in two; 4 x 2011 29.9 in two, 26.9 in four; 3 x 849 of
  // 32 heads 41.2 in one, 36.8 in two).  A wave (of clusters) costs about 2 us and a merge across CTAs 1.  Over 120 steps of 1 to 62 sequences this
  // choice is 0.1 % from the best of all eight on average, 5 % at most.
  // (Two CTAs per SM; with 480 or 2048 sequence-heads more than one share is slower, with 16 eight are best.)
  const int units = B * a.heads;
  double best = 0.0;
  a.split = 1;
  const ClusterCtas fit = tc_cluster_ctas_all();
  for (int s = 1; s <= DEC_MAX_SPLIT; ++s) {
    const long long ctas = (long long)units * s, slots = 2ll * fit.n[s], full = ctas / slots, tail = ctas % slots;
    const double stages = ((a.S + s - 1) / s + DEC_STEP - 1) / DEC_STEP;
    auto wave = [&](long long n) { const double t = n * 0.00504; return n ? stages * sqrt(0.54 * 0.54 + t * t) + 2.0 : 0.0; };
    const double t = full * wave(slots) + wave(tail) - (s == 1 ? 0.8 * full : -1.0);
    if (s == 1 || t < best) { best = t; a.split = s; }
  }
  constexpr size_t smem = 128 + DEC_STAGES * DEC_STAGE_BYTES;
  if (ensure_max_dynamic_smem((const void*)decode_attn_kernel, (int)smem, 100) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("decode_attention", st);
  a.units = units;
  // Short contexts: CTAs walk over several units.  Beyond eight stages a unit's own length hides its start, and the hardware's
  // dealing of one unit per CTA evens out the SMs' different speeds (2048 units of 2048 positions: 308 us against 322).
  const int walk = a.split == 1 && a.S <= 8 * DEC_STEP && units > 2 * tc_sm_count();
  const dim3 grid((unsigned)(walk ? 2 * tc_sm_count() : units * a.split));
  if (launch_pdl_cluster(decode_attn_kernel, grid, dim3(DEC_THREADS), smem, st, (unsigned)a.split, tk, tv, a) != cudaSuccess)
    return SMARTMEM_ERR_CUDA;
  count_launch();
  return SMARTMEM_OK;
}

// Explicit variant: in-place rotary embedding of rows [R, 128] that all sit at position `pos`.
__global__ void rope_rows_at_kernel(__nv_bfloat16* x, long long rows, int pos, double theta, int rot) {
  pdl_wait();
  pdl_launch_dependents();
  const int half = rot / 2;                     // pairs (i, i + rot/2) of the first rot elements of a row
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= rows * half) return;
  const long long r = idx / half;
  const int i = (int)(idx - r * half);
  double sn, cs;
  sincos((double)pos * pow(theta, -(double)i / half), &sn, &cs);
  __nv_bfloat16* row = x + r * DH;
  const float a = __bfloat162float(row[i]), b = __bfloat162float(row[i + half]);
  row[i] = __float2bfloat16_rn(a * (float)cs - b * (float)sn);
  row[i + half] = __float2bfloat16_rn(b * (float)cs + a * (float)sn);
}

// Explicit variant: the Concat of the cache with the new rows, for a cache with room left: row r of
// src [R, 128] goes to dst + r * dst_row_stride (the slot of position `pos` of (sequence, head) r).
__global__ void append_rows_kernel(const __nv_bfloat16* __restrict__ src, __nv_bfloat16* dst, long long rows,
                                   long long dst_row_stride) {
  pdl_wait();
  pdl_launch_dependents();
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;   // one 16-byte vector each
  if (idx >= rows * (DH / 8)) return;
  const long long r = idx / (DH / 8);
  const int v = (int)(idx - r * (DH / 8));
  *reinterpret_cast<uint4*>(dst + r * dst_row_stride + v * 8) = *reinterpret_cast<const uint4*>(src + r * DH + v * 8);
}

int launch_rope_rows_at(void* x, long long rows, int pos, float theta, int rot, cudaStream_t st) {
  const long long n = rows * (rot / 2);
  profile_tick("rope_rows", st);
  launch_pdl(rope_rows_at_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, (__nv_bfloat16*)x, rows, pos, (double)theta, rot);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? SMARTMEM_OK : SMARTMEM_ERR_CUDA;
}

int launch_append_rows(const void* src, void* dst, long long rows, long long dst_row_stride, const char* label,
                       cudaStream_t st) {
  const long long n = rows * (DH / 8);
  profile_tick(label, st);
  launch_pdl(append_rows_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, (const __nv_bfloat16*)src,
             (__nv_bfloat16*)dst, rows, dst_row_stride);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? SMARTMEM_OK : SMARTMEM_ERR_CUDA;
}

// Head split of one token per sequence: [B, 1, 3*H*D] -> [3, B, H, 1, D].
typedef std::tuple<int, int, int> DKey;
std::mutex g_mu;
std::map<DKey, smartmem_index_map_t> g_split;

int get_split(int B, int H, int D, smartmem_index_map_t* out) {   // (a copy: clearing the cache cannot invalidate it)
  DKey key(B, H, D);
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_split.find(key);
  if (it != g_split.end()) { *out = it->second; return SMARTMEM_OK; }
  smartmem_index_map_t m;
  const int64_t b = B, h = H, d = D;
  int rc = chain_map({b, 1, 3 * h * d}, {op_reshape({b, 1, 3, h, d}), op_transpose({2, 0, 3, 1, 4})}, SMARTMEM_BF16, &m);
  if (rc != SMARTMEM_OK) return rc;
  if (g_split.size() > 64) g_split.clear();
  *out = g_split.emplace(key, m).first->second;
  return SMARTMEM_OK;
}

size_t al(size_t b) { return (b + 255) & ~(size_t)255; }

struct Layout { size_t xn, qkv, ao, split, total; };

Layout ws_layout(const smartmem_attn_params_t& p, int mode) {
  const size_t BH = al((size_t)p.B * p.hidden * 2);
  Layout L;
  memset(&L, 0, sizeof(L));
  size_t off = 0;
  auto take = [&](size_t b) { size_t o = off; off += b; return o; };
  L.xn = take(BH);
  L.qkv = take(3 * BH);        // ELIMINATE uses the first third (q only: k and v go to the caches)
  L.ao = take(BH);
  if (mode == SMARTMEM_EXPLICIT) L.split = take(3 * BH);
  L.total = off;
  return L;
}

int validate(const smartmem_attn_params_t* p, int mode) {
  if (!p) return SMARTMEM_ERR_INVALID_ARG;
  if (mode != SMARTMEM_ELIMINATE && mode != SMARTMEM_EXPLICIT) return SMARTMEM_ERR_INVALID_ARG;
  if (p->dtype != SMARTMEM_BF16) return SMARTMEM_ERR_UNSUPPORTED;
  if (p->B < 1 || p->S < 1 || p->hidden < 1 || p->heads < 1) return SMARTMEM_ERR_SHAPE;
  if (p->heads * p->head_dim != p->hidden) return SMARTMEM_ERR_SHAPE;
  if (p->head_dim != DH || p->hidden % 256) return SMARTMEM_ERR_UNSUPPORTED;
  if (p->rotary_dim != 0 && p->rotary_dim != 32 && p->rotary_dim != 64 && p->rotary_dim != 128) return SMARTMEM_ERR_UNSUPPORTED;
  return SMARTMEM_OK;
}

}  // namespace

EXPORT int smartmem_attn_decode_workspace_bytes(const smartmem_attn_params_t* p, int32_t mode, size_t* bytes) {
  int rc = validate(p, mode);
  if (rc != SMARTMEM_OK) return rc;
  if (!bytes) return SMARTMEM_ERR_INVALID_ARG;
  *bytes = ws_layout(*p, mode).total;
  return SMARTMEM_OK;
}

EXPORT int smartmem_attn_decode(const smartmem_attn_params_t* pp, int32_t pos, const void* x, void* k_cache,
                                void* v_cache, void* y, void* workspace, size_t workspace_bytes, int32_t mode,
                                void* cuda_stream) {
  int rc = validate(pp, mode);
  if (rc != SMARTMEM_OK) return rc;
  const smartmem_attn_params_t& p = *pp;
  if (pos < 0 || pos >= p.S) return SMARTMEM_ERR_SHAPE;
  // rows of the caches as the attention kernel's tensor maps count them: [B S_max] or [B heads S_max]
  if (pos + 1 > DEC_MAX_S || (long long)p.B * p.S * (mode == SMARTMEM_ELIMINATE ? 1 : p.heads) >= (1ll << 31)) return SMARTMEM_ERR_UNSUPPORTED;
  if (!x || !y || !k_cache || !v_cache || !workspace || x == y || !p.rms_g || !p.w_qkv || !p.w_o)
    return SMARTMEM_ERR_INVALID_ARG;
  const void* al16[] = {x, y, k_cache, v_cache, workspace, p.rms_g, p.w_qkv, p.w_o};
  for (const void* q : al16)
    if ((uintptr_t)q & 15) return SMARTMEM_ERR_ALIGNMENT;
  const Layout L = ws_layout(p, mode);
  if (workspace_bytes < L.total) return SMARTMEM_ERR_WORKSPACE;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) return SMARTMEM_ERR_CUDA;

  cudaStream_t st = (cudaStream_t)cuda_stream;
  const bool elim = mode == SMARTMEM_ELIMINATE;
  const long long B = p.B, Smax = p.S, H = p.heads, hid = p.hidden;
  char* w = (char*)workspace;
  auto at = [&](size_t off) { return (void*)(w + off); };
  __nv_bfloat16* kc = (__nv_bfloat16*)k_cache;
  __nv_bfloat16* vc = (__nv_bfloat16*)v_cache;

#define SM_TRY(expr) do { rc = (expr); if (rc != SMARTMEM_OK) return rc; } while (0)
  // few rows: RMSNorm rides along in the QKV GEMM, where its share of gamma fits (hidden up to 27392 at B = 49..64, more at others)
  const bool norm_in_gemm = B <= 128 && gemm_splitk_norm_fits(B, 3 * hid, hid);
  if (!norm_in_gemm) SM_TRY(launch_norm(SMARTMEM_BF16, true, x, at(L.xn), p.rms_g, nullptr, p.rms_eps, B, (int)hid, nullptr, st));
  DecodeAttnArgs a;
  memset(&a, 0, sizeof(a));
  a.heads = (int)H;
  a.S = pos + 1;
  a.scale_log2e = 1.4426950408889634f / sqrtf((float)DH);
  a.k = kc;
  a.v = vc;
  a.o = (__nv_bfloat16*)at(L.ao);
  a.o_sb = hid;                // [B, H, 1, D] and [B, 1, H*D] are the same bytes: the merge of one token is free
  a.o_sh = DH;
  {
    TcEpilogue ep;
    memset(&ep, 0, sizeof(ep));
    ep.out = at(L.qkv);
    ep.ldc = 3 * hid;
    if (elim) {
      ep.rope_cols = (int)(2 * hid);
      ep.rope_S = 1;
      ep.rope_pos0 = pos;
      ep.rope_log2_theta = log2f(p.rope_theta);
      ep.rope_dim = p.rotary_dim ? p.rotary_dim : DH;
      ep.seg_cols = (int)hid;
      ep.seg_out[0] = at(L.qkv);              ep.seg_ld[0] = hid;
      ep.seg_out[1] = kc + (long long)pos * hid;   ep.seg_ld[1] = Smax * hid;
      ep.seg_out[2] = vc + (long long)pos * hid;   ep.seg_ld[2] = Smax * hid;
    }
    ep.b_settled = norm_in_gemm ? 0 : 1;             // (with RMSNorm inside it is the call's first kernel)
    if (norm_in_gemm) { ep.rms_gamma = p.rms_g; ep.rms_eps = p.rms_eps; }
    SM_TRY(launch_gemm_tc(tc_operand_plain(norm_in_gemm ? x : at(L.xn), B, hid, hid), tc_operand_plain(p.w_qkv, 3 * hid, hid, hid), ep, 1,
                          B, 3 * hid, hid, st));
  }
  if (elim) {
    a.q = (const __nv_bfloat16*)at(L.qkv);
    a.q_sb = hid; a.q_sh = DH;
    a.pitch = (int)hid; a.rows = (int)(B * Smax); a.rows_b = (int)Smax; a.rows_h = 0; a.cols_h = DH;
  } else {
    smartmem_index_map_t split;
    SM_TRY(get_split(p.B, p.heads, DH, &split));
    SM_TRY(launch_copy_map(split, 2, at(L.qkv), at(L.split), st));
    __nv_bfloat16* sp = (__nv_bfloat16*)at(L.split);
    SM_TRY(launch_rope_rows_at(sp, 2 * B * H, pos, p.rope_theta, p.rotary_dim ? p.rotary_dim : DH, st));
    SM_TRY(launch_append_rows(sp + B * hid, kc + (long long)pos * DH, B * H, Smax * DH, "append_k", st));
    SM_TRY(launch_append_rows(sp + 2 * B * hid, vc + (long long)pos * DH, B * H, Smax * DH, "append_v", st));
    a.q = sp;
    a.q_sb = hid; a.q_sh = DH;
    a.pitch = DH; a.rows = (int)(B * H * Smax); a.rows_b = (int)(H * Smax); a.rows_h = (int)Smax; a.cols_h = 0;
  }
  SM_TRY(launch_decode_attention(a, p.B, st));
  {
    TcEpilogue ep;
    memset(&ep, 0, sizeof(ep));
    ep.out = y;
    ep.ldc = hid;
    ep.residual = p.add_residual ? x : nullptr;
    ep.b_settled = 1;
    SM_TRY(launch_gemm_tc(tc_operand_plain(at(L.ao), B, hid, hid), tc_operand_plain(p.w_o, hid, hid, hid), ep, 1, B, hid,
                          hid, st));
  }
#undef SM_TRY
  return SMARTMEM_OK;
}
