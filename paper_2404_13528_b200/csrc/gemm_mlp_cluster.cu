// Fused MLP half of a Swin block whose weights do not fit one SM: out = x + fc2(GELU(fc1(LN(x)))), C = 64 or 128, for few rows.
//
// With a few thousand rows the kernels it replaces (LayerNorm + fc1 + GELU, together or apart, and fc2 + residual) are each a launch, a
// dependency, a first load and a drain around a fraction of a microsecond of products.  Here a cluster of CTAs takes 128 rows and
// splits the hidden features: every CTA normalises the rows (redundantly), multiplies them with its slice of W1, keeps the GELU of
// its slice on chip as fc2's operand and multiplies that with its slice of W2; the fp32 partial results are exchanged as bulk
// copies between the CTAs' shared memories, each CTA adding up its share of the rows.  The weight slices are fetched before the
// dependency wait where nothing in flight can be writing them.  What it gave is beside the rule at the end.
//
// Bound by the chain of its phases (with four slices of 192 about 1.5 us rows, 0.9 first product, 1.3 GELU, 0.9 second product, 0.6
// drain, 2.2 exchange of 72 KB at the 18 bytes a cycle that shared memory takes from its peers, 1.2 sum), one tile per cluster: beyond
// one wave the second tile cannot overlap the first and the separate kernels win.  Tried and slower: the shares sent into W1's memory
// while the second product runs (12.8 us).
//
// Shared memory: the normalised rows (later the hidden slice) and both weight slices as K-major 128-byte-swizzled operands; once
// fc2 has read them the same memory holds the CTA's partial result [128][C] and what its peers send.
// Warp roles: 0-15 rows, GELU, drain and sum; 16 fetches the weights, owns the tensor memory and issues the products.
#include <cstring>

#include "gemm_tc.cuh"
#include "ln_operand.cuh"
#include "ptx.cuh"

namespace smartmem {
namespace {

constexpr int BM = 128, BK = 64;
constexpr int kWorkers = 16, kThreads = 32 * (kWorkers + 1);
constexpr int kMaxSplits = 4;
constexpr uint32_t TM_D1 = 0, TM_D2 = 256, TMEM_COLS = 512;

struct MlpClusterArgs {
  int M, hidden, hs, splits;                       // hs: hidden features of a CTA
  int w1_off, w2_off, recv_off, bar_off;           // byte offsets behind the aligned base
  float eps;
  const __nv_bfloat16 *x, *ln_g, *ln_b, *b1, *b2;
  __nv_bfloat16* out;
  int* status;
};

template <int NV, int N16>                         // C / 64, hs / 64
__global__ void __launch_bounds__(kThreads, 1)
mlp_cluster_kernel(const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ MlpClusterArgs g) {
  constexpr int C = 64 * NV;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sA = smem;                              // [NV][16 KB]: the rows; later [hs / 64][16 KB]: the hidden slice
  uint8_t* sW1 = smem + g.w1_off;                  // [NV][hs x 128 B]
  uint8_t* sW2 = smem + g.w2_off;                  // [hs / 64][C x 128 B]
  uint64_t* w1_full = reinterpret_cast<uint64_t*>(smem + g.bar_off);
  uint64_t *w2_full = w1_full + 1, *a_ready = w1_full + 2, *d1_full = w1_full + 3, *h_ready = w1_full + 4, *d2_full = w1_full + 5,
           *recv_full = w1_full + 6;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(w1_full + 7);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  __nv_bfloat16* b1_s = reinterpret_cast<__nv_bfloat16*>(tmem_slot + 2);            // [hs]
  constexpr int HS = 64 * N16;

  const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
  const int S = g.splits, rank = S > 1 ? (int)ptx::cluster_ctarank() : 0;
  const int m0 = (int)blockIdx.x / S * BM;
  const int slice_rows = BM / S;
  const uint32_t slice_bytes = (uint32_t)slice_rows * C * 4;

  if (warp == kWorkers) {
    if (ptx::elect_one()) {
      ptx::mbar_init(w1_full, 1);
      ptx::mbar_init(w2_full, 1);
      ptx::mbar_init(a_ready, kWorkers);
      ptx::mbar_init(d1_full, 1);
      ptx::mbar_init(h_ready, kWorkers);
      ptx::mbar_init(d2_full, 1);
      ptx::mbar_init(recv_full, 1);
      *abort_flag = 0;
      ptx::fence_barrier_init();
      ptx::fence_proxy_async();
      ptx::prefetch_tensormap(&tmW1);
      ptx::prefetch_tensormap(&tmW2);
      ptx::mbar_expect_tx(w1_full, (uint32_t)(g.hs * C * 2));
      ptx::mbar_expect_tx(w2_full, (uint32_t)(g.hs * C * 2));
      if (S > 1) ptx::mbar_expect_tx(recv_full, (uint32_t)(S - 1) * slice_bytes);
    }
    __syncwarp();
    // the weight slices are parameters: fetched before the dependency wait, all k-blocks of one in a copy
    if (ptx::elect_one()) ptx::tma_load_3d(sW1, &tmW1, w1_full, 0, rank * g.hs, 0);
    __syncwarp();
    if (ptx::elect_one()) ptx::tma_load_3d(sW2, &tmW2, w2_full, 0, 0, rank * (g.hs / BK));
    __syncwarp();
    ptx::tmem_alloc(tmem_slot, TMEM_COLS);
  }
  if (tid < HS / 8) reinterpret_cast<uint4*>(b1_s)[tid] = *reinterpret_cast<const uint4*>(g.b1 + rank * HS + tid * 8);
  ptx::tc_fence_before();
  __syncwarp();
  if (S > 1) ptx::cluster_sync(); else __syncthreads();    // (the peers' barriers are initialised before anything is sent to them)
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == kWorkers) {
    const uint32_t a0 = ptx::smem_u32(sA), w1 = ptx::smem_u32(sW1), w2 = ptx::smem_u32(sW2);
    bool ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(w1_full, 0, abort_flag, g.status) && ptx::mbar_wait(a_ready, 0, abort_flag, g.status) ? 1 : 0) != 0;
    if (ok) {
      ptx::tc_fence_after();
      const uint32_t idesc = ptx::make_idesc_bf16(BM, g.hs, false, false);
      if (ptx::elect_one()) {
#pragma unroll
        for (int kb = 0; kb < NV; ++kb) {
          const uint64_t ad = ptx::make_smem_desc(a0 + kb * kLnBlockBytes, 16, 1024), bd = ptx::make_smem_desc(w1 + kb * g.hs * 128, 16, 1024);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) ptx::tc_mma_bf16(tmem_base + TM_D1, ad + 2 * k, bd + 2 * k, idesc, (kb | k) ? 1u : 0u);
        }
        ptx::tc_commit(d1_full);
      }
      __syncwarp();
      ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(w2_full, 0, abort_flag, g.status) && ptx::mbar_wait(h_ready, 0, abort_flag, g.status) ? 1 : 0) != 0;
    }
    if (ok) {
      ptx::tc_fence_after();
      const uint32_t idesc = ptx::make_idesc_bf16(BM, C, false, false);
      if (ptx::elect_one()) {
        for (int kb = 0; kb < g.hs / BK; ++kb) {
          const uint64_t ad = ptx::make_smem_desc(a0 + kb * kLnBlockBytes, 16, 1024), bd = ptx::make_smem_desc(w2 + kb * C * 128, 16, 1024);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) ptx::tc_mma_bf16(tmem_base + TM_D2, ad + 2 * k, bd + 2 * k, idesc, (kb | k) ? 1u : 0u);
        }
        ptx::tc_commit(d2_full);
      }
      __syncwarp();
    }
  } else {
    // ---- rows: eight lanes per row, NV vectors each; eight rows per warp, all requested at once ---------------------------
    const int sub = lane & 7, rsub = lane >> 3;
    uint4 ga[NV], be[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      ga[k] = *reinterpret_cast<const uint4*>(g.ln_g + (sub + 8 * k) * 8);
      be[k] = *reinterpret_cast<const uint4*>(g.ln_b + (sub + 8 * k) * 8);
    }
    pdl_wait();
    pdl_launch_dependents();
    uint4 x[2][NV];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const int m = m0 + warp * 8 + j * 4 + rsub;
        x[j][k] = make_uint4(0, 0, 0, 0);
        if (m < g.M) x[j][k] = *reinterpret_cast<const uint4*>(g.x + (size_t)m * C + (sub + 8 * k) * 8);
      }
    ln_rows_to_operand<NV>(x, ga, be, g.eps, sA, warp * 8, lane);
    ptx::fence_proxy_async();
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(a_ready);

    // ---- hidden slice: a thread per row and quarter of the columns, the whole quarter in registers -------------------------
    const int q = warp & 3, grp = warp >> 2, r = q * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
    bool ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(d1_full, 0, abort_flag, g.status) ? 1 : 0) != 0;
    if (ok) {
      ptx::tc_fence_after();
      uint32_t v[N16][16];
#pragma unroll
      for (int p = 0; p < N16; ++p) ptx::tmem_ld16(tmem_base + TM_D1 + lane_addr + (grp * N16 + p) * 16, v[p]);
      ptx::tmem_ld_wait();
#pragma unroll
      for (int p = 0; p < N16; ++p) {
        const int c = (grp * N16 + p) * 16;
        const uint4 b0 = *reinterpret_cast<const uint4*>(b1_s + c), b1 = *reinterpret_cast<const uint4*>(b1_s + c + 8);
        const uint32_t bw[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        uint32_t o[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float2 f = bf16x2_to_float2(bw[e]);
          o[e] = float2_to_bf16x2(gelu_tanh(__uint_as_float(v[p][2 * e]) + f.x), gelu_tanh(__uint_as_float(v[p][2 * e + 1]) + f.y));
        }
        uint8_t* h = sA + (c >> 6) * kLnBlockBytes + r * 128;
        const int ch = (c & 63) >> 3;
        *reinterpret_cast<uint4*>(h + ((ch ^ (r & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<uint4*>(h + (((ch + 1) ^ (r & 7)) << 4)) = make_uint4(o[4], o[5], o[6], o[7]);
      }
      ptx::fence_proxy_async();
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(h_ready);
      ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(d2_full, 0, abort_flag, g.status) ? 1 : 0) != 0;
    }
    // ---- this slice's share of the result -> shared memory [128][C], 16-byte chunks swizzled by the row --------------------
    if (ok) {
      ptx::tc_fence_after();
      uint8_t* p = smem + (size_t)r * (C * 4);
      uint32_t v[NV][16];
#pragma unroll
      for (int i = 0; i < NV; ++i) ptx::tmem_ld16(tmem_base + TM_D2 + lane_addr + (grp * NV + i) * 16, v[i]);
      ptx::tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < NV; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          *reinterpret_cast<uint4*>(p + ((((grp * NV + i) * 4 + e) ^ (r & 7)) << 4)) =
              make_uint4(v[i][4 * e], v[i][4 * e + 1], v[i][4 * e + 2], v[i][4 * e + 3]);
      ptx::fence_proxy_async();                        // -> visible to the bulk copies
    }
  }
  ptx::tc_fence_before();
  __syncwarp();
  if (S > 1) ptx::cluster_sync(); else __syncthreads();    // every CTA's products are done: its memory may be written by its peers
  if (S > 1 && warp == kWorkers) {
    for (int i = 1; i < S; ++i) {                    // (every CTA starts with another peer)
      const int p = (rank + i) & (S - 1);
      if (ptx::elect_one())
        ptx::bulk_copy_cluster(ptx::mapa(ptx::smem_u32(smem + g.recv_off + (rank < p ? rank : rank - 1) * slice_bytes), (uint32_t)p),
                               smem + p * slice_bytes, slice_bytes, ptx::mapa(ptx::smem_u32(recv_full), (uint32_t)p));
      __syncwarp();
    }
  }
  if (warp < kWorkers) {
    // ---- this CTA's rows: the partial results in the order of the slices, bias, residual (requested while the shares travel) ----
    const int n = slice_rows * (C / 8);
    bool ok = true, waited = false;
    for (int i0 = tid; i0 < n; i0 += 2 * 32 * kWorkers) {
      uint4 res[2], bias[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = i0 + u * 32 * kWorkers, rl = i / (C / 8), c8 = i - rl * (C / 8), m = m0 + rank * slice_rows + rl;
        res[u] = bias[u] = make_uint4(0, 0, 0, 0);
        if (i < n && m < g.M) {
          res[u] = *reinterpret_cast<const uint4*>(g.x + (size_t)m * C + c8 * 8);
          bias[u] = *reinterpret_cast<const uint4*>(g.b2 + c8 * 8);
        }
      }
      if (S > 1 && !waited) {
        ok = ptx::mbar_wait(recv_full, 0, abort_flag, g.status);
        ptx::cluster_arrive();                       // everything sent to this CTA has come
        waited = true;
      }
      if (!ok) break;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = i0 + u * 32 * kWorkers, rl = i / (C / 8), c8 = i - rl * (C / 8), r = rank * slice_rows + rl, m = m0 + r;
        if (i >= n || m >= g.M) continue;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
#pragma unroll
        for (int s = 0; s < kMaxSplits; ++s)
          if (s < S) {
            const uint8_t* src = (s == rank ? smem + rank * slice_bytes : smem + g.recv_off + (s < rank ? s : s - 1) * slice_bytes) + (size_t)rl * (C * 4);
            const float4 w = *reinterpret_cast<const float4*>(src + (((2 * c8) ^ (r & 7)) << 4));
            const float4 z = *reinterpret_cast<const float4*>(src + (((2 * c8 + 1) ^ (r & 7)) << 4));
            a.x += w.x; a.y += w.y; a.z += w.z; a.w += w.w;
            b.x += z.x; b.y += z.y; b.z += z.z; b.w += z.w;
          }
        const float2 r0 = bf16x2_to_float2(res[u].x), r1 = bf16x2_to_float2(res[u].y), r2 = bf16x2_to_float2(res[u].z), r3 = bf16x2_to_float2(res[u].w);
        const float2 b0 = bf16x2_to_float2(bias[u].x), b1 = bf16x2_to_float2(bias[u].y), b2 = bf16x2_to_float2(bias[u].z), b3 = bf16x2_to_float2(bias[u].w);
        *reinterpret_cast<uint4*>(g.out + (size_t)m * C + c8 * 8) =
            make_uint4(float2_to_bf16x2(a.x + b0.x + r0.x, a.y + b0.y + r0.y), float2_to_bf16x2(a.z + b1.x + r1.x, a.w + b1.y + r1.y),
                       float2_to_bf16x2(b.x + b2.x + r2.x, b.y + b2.y + r2.y), float2_to_bf16x2(b.z + b3.x + r3.x, b.w + b3.y + r3.y));
      }
    }
    if (S > 1 && !waited) ptx::cluster_arrive();
  } else if (S > 1) {
    ptx::cluster_arrive();
  }
  __syncwarp();
  if (S > 1) ptx::cluster_wait(); else __syncthreads();    // no CTA leaves while its share is still being sent
  if (warp == kWorkers) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

struct Sizes {
  int w1_off, w2_off, recv_off, bar_off;
  size_t smem;
};
Sizes sizes_of(int C, int hs, int S) {
  Sizes z;
  const int rows = (C > hs ? C : hs) / BK * kLnBlockBytes;              // the rows, later the hidden slice
  z.w1_off = rows;
  z.w2_off = rows + C / BK * hs * 128;
  const int operands = z.w2_off + hs / BK * C * 128, partial = BM * C * 4, recv = (S - 1) * (BM / S) * C * 4;
  z.recv_off = partial;
  z.bar_off = operands > partial + recv ? operands : partial + recv;
  z.smem = 1024 + z.bar_off + 7 * 8 + 8 + hs * 2;
  return z;
}
// the fewest slices whose operands fit an SM (0: none)
int splits_of(long long C, long long hidden) {
  if (C != 64 && C != 128) return 0;
  for (int s = 1; s <= kMaxSplits; s *= 2)
    if (hidden % (64 * s) == 0 && hidden / s <= 256 && sizes_of((int)C, (int)(hidden / s), s).smem <= 227 * 1024) return s;
  return 0;
}

}  // namespace

bool mlp_cluster_wins(long long M, long long C, long long hidden) {
  // Whole blocks, us, separate kernels -> this one.  C = 64 (hidden 64 and 768, which the kernel with resident weights does not take): 196
  // rows 15.5 -> 10.9 and 16.8 -> 13.1, 3136 20.1 -> 13.3.  C = 128, hidden 512: 7840 rows 28.8 -> 27.5, 2352 23.4 -> 22.8, but 1568 21.0 ->
  // 21.2, 196 20.1 -> 20.6, 49 18.0 -> 19.0, hidden 256 alike; hidden 128 and 768 win at every size (196 rows 18.8 -> 18.1, 21.0 -> 20.2).
  // C = 192 lost or tied at every size once LayerNorm and fc1 were one kernel (784 rows 22.4 -> 23.3, 3920 29.2 -> 29.3) and is not covered.
  // One wave of clusters: a second one took C = 128 at 15680 rows from 18.7 to 20.8 us, the MLP half alone.
  const int s = splits_of(C, hidden);
  if (s == 0 || (M + BM - 1) / BM > tc_cluster_ctas(s) / s) return false;
  return C == 64 || M >= 2304 || hidden < 256 || hidden > 512;
}

int launch_mlp_cluster(const void* x, const void* ln_g, const void* ln_b, float eps, const void* W1, const void* b1, const void* W2,
                       const void* b2, void* out, long long M, long long C, long long hidden, bool settled, cudaStream_t st) {
  MlpClusterArgs g;
  memset(&g, 0, sizeof(g));
  g.splits = splits_of(C, hidden);
  if (g.splits == 0 || M < 1 || M >= (1ll << 31) / 4) return SMARTMEM_ERR_UNSUPPORTED;
  const void* ptrs[] = {x, ln_g, ln_b, W1, b1, W2, b2, out};
  for (const void* p : ptrs)
    if (!p || ((uintptr_t)p & 15)) return SMARTMEM_ERR_ALIGNMENT;
  g.M = (int)M; g.hidden = (int)hidden; g.hs = (int)hidden / g.splits;
  const Sizes z = sizes_of((int)C, g.hs, g.splits);
  g.w1_off = z.w1_off; g.w2_off = z.w2_off; g.recv_off = z.recv_off; g.bar_off = z.bar_off;
  g.eps = eps;
  g.x = (const __nv_bfloat16*)x; g.ln_g = (const __nv_bfloat16*)ln_g; g.ln_b = (const __nv_bfloat16*)ln_b;
  g.b1 = (const __nv_bfloat16*)b1; g.b2 = (const __nv_bfloat16*)b2; g.out = (__nv_bfloat16*)out;
  g.status = device_status_ptr();
  if (!g.status) return SMARTMEM_ERR_CUDA;
  CUtensorMap t1, t2;
  int rc = tc_encode_2d_blocks(W1, C, hidden, C / BK, g.hs, &t1);
  if (rc == SMARTMEM_OK) rc = tc_encode_2d_blocks(W2, hidden, C, g.hs / BK, C, &t2);
  if (rc != SMARTMEM_OK) return rc;
  static constexpr decltype(&mlp_cluster_kernel<1, 1>) kernels[2][4] = {
      {mlp_cluster_kernel<1, 1>, mlp_cluster_kernel<1, 2>, mlp_cluster_kernel<1, 3>, mlp_cluster_kernel<1, 4>},
      {mlp_cluster_kernel<2, 1>, mlp_cluster_kernel<2, 2>, mlp_cluster_kernel<2, 3>, mlp_cluster_kernel<2, 4>}};
  auto* fn = kernels[C / 64 - 1][g.hs / 64 - 1];
  if (ensure_max_dynamic_smem((const void*)fn, 227 * 1024) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("mlp_cluster", st);
  const unsigned grid = (unsigned)((M + BM - 1) / BM * g.splits);
  if (launch_cluster(fn, dim3(grid), dim3(kThreads), z.smem, st, (unsigned)g.splits, settled, t1, t2, g) != cudaSuccess) return SMARTMEM_ERR_CUDA;
  count_launch();
  return SMARTMEM_OK;
}

}  // namespace smartmem
