// LayerNorm o row-gather o linear (o GELU) for one wave of rows: out[m, :] = LN(X[src(m), :]) W^T + bias, rows of K = 128, 192 or 256.
//
// The kernel for K = 64 and 96 keeps all of W in shared memory and streams the rows past it; here W does not fit, and with a few
// thousand rows there is nothing to stream: a launch, a dependency and a drain cost the normalisation and the product each more
// than their work.  A CTA takes 128 rows and a slice of the output columns, normalises the rows (again in every slice: they come
// from L2) straight into the operand, and multiplies them with its slice of W, which is in L2 by then.  Bound by that
// chain (1.5 us rows, 0.9 product, 0.6 output and the dependency).  Measured, a block's attention half with norm and QKV linear as two
// kernels -> with this: 3920 x 192 19.2 -> 17.1 us (93 CTAs), 7840 x 128 20.6 -> 17.2 (124), 1568 x 256 18.2 -> 15.7 (78), 4704 x 256
// 21.9 -> 19.5 (148); whole blocks, norm + fc1 + GELU as well: 1568 x 256 32.8 -> 27.9, 3920 x 192 35.3 -> 29.2.
//
// Warp roles: 0-15 rows, then bias and output; 16 fetches W, owns the tensor memory and issues the product.
#include <cstring>

#include "gemm_tc.cuh"
#include "ln_operand.cuh"
#include "ptx.cuh"

namespace smartmem {
namespace {

constexpr int BM = 128, BK = 64;
constexpr int kWorkers = 16, kThreads = 32 * (kWorkers + 1);

struct LnWaveArgs {
  int M, N, slices, has_map, gelu, wide, w_settled;
  float eps;
  const __nv_bfloat16 *x, *ln_g, *ln_b, *bias;
  __nv_bfloat16* out;
  DevMap rowmap;
  int* status;
};

template <int NV, int NB>
constexpr int wave_smem_bytes() { return 1024 + NV * kLnBlockBytes + NV * NB * 64 * 128 + NB * 64 * 2 + 4 * 8; }

template <int NV, int NB>                          // K / 64, columns of a slice / 64
__global__ void __launch_bounds__(kThreads, 1)
ln_wave_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ LnWaveArgs g) {
  constexpr int K = 64 * NV, NS = 64 * NB;
  constexpr uint32_t TMEM_COLS = NB > 2 ? 256 : NS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sA = smem;
  uint8_t* sW = smem + NV * kLnBlockBytes;   // [NV][NS x 128 B]
  __nv_bfloat16* bias_s = reinterpret_cast<__nv_bfloat16*>(sW + NV * NS * 128);
  uint64_t* w_full = reinterpret_cast<uint64_t*>(bias_s + NS);
  uint64_t *a_ready = w_full + 1, *d_full = w_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(w_full + 3);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
  const int m0 = (int)blockIdx.x / g.slices * BM, n0 = (int)blockIdx.x % g.slices * NS;

  if (warp == kWorkers) {
    if (ptx::elect_one()) {
      ptx::mbar_init(w_full, 1);
      ptx::mbar_init(a_ready, kWorkers);
      ptx::mbar_init(d_full, 1);
      *abort_flag = 0;
      ptx::fence_barrier_init();
      ptx::fence_proxy_async();
      ptx::mbar_expect_tx(w_full, (uint32_t)(NS * K * 2));
      // W, all k-blocks in one copy: before the dependency wait where nothing in flight can be writing it, else only as far as L2
      if (g.w_settled) ptx::tma_load_3d(sW, &tmW, w_full, 0, n0, 0);
      else ptx::tma_prefetch_3d(&tmW, 0, n0, 0);
    }
    __syncwarp();
    ptx::tmem_alloc(tmem_slot, TMEM_COLS);
  } else if (warp == 0) {
    if (lane < K / 64) {
      ptx::prefetch_l2(g.ln_g + lane * 64);
      ptx::prefetch_l2(g.ln_b + lane * 64);
    } else if (g.bias && lane - K / 64 < NB) {
      ptx::prefetch_l2(g.bias + n0 + (lane - K / 64) * 64);
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == kWorkers) {
    const uint32_t a0 = ptx::smem_u32(sA), w0 = ptx::smem_u32(sW);
    if (!g.w_settled) {
      pdl_wait();
      if (ptx::elect_one()) ptx::tma_load_3d(sW, &tmW, w_full, 0, n0, 0);
      __syncwarp();
    }
    const bool ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(w_full, 0, abort_flag, g.status) && ptx::mbar_wait(a_ready, 0, abort_flag, g.status) ? 1 : 0) != 0;
    if (ok) {
      ptx::tc_fence_after();
      const uint32_t idesc = ptx::make_idesc_bf16(BM, NS, false, false);
      if (ptx::elect_one()) {
#pragma unroll
        for (int kb = 0; kb < NV; ++kb) {
          const uint64_t ad = ptx::make_smem_desc(a0 + kb * kLnBlockBytes, 16, 1024), bd = ptx::make_smem_desc(w0 + kb * NS * 128, 16, 1024);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) ptx::tc_mma_bf16(tmem_base, ad + 2 * k, bd + 2 * k, idesc, (kb | k) ? 1u : 0u);
        }
        ptx::tc_commit(d_full);
      }
      __syncwarp();
    }
  } else {
    constexpr int L = ln_lanes(NV), J = L / 4, V = 8 * NV / L;
    const int sub = lane % L, rsub = lane / L;
    // the warp's eight row offsets, one evaluation of the map per lane
    const int mrow = m0 + warp * 8 + (lane & 7);
    long long row_off = 0;
    if (mrow < g.M) row_off = g.has_map ? devmap_eval_unrolled(g.rowmap, (uint32_t)mrow) : (long long)mrow * K;
    pdl_wait();
    pdl_launch_dependents();
    uint4 x[J][V];
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int r = j * (32 / L) + rsub;
      const long long off = __shfl_sync(0xFFFFFFFFu, row_off, r);
#pragma unroll
      for (int k = 0; k < V; ++k) {
        x[j][k] = make_uint4(0, 0, 0, 0);
        if (m0 + warp * 8 + r < g.M) x[j][k] = *reinterpret_cast<const uint4*>(g.x + off + (sub + L * k) * 8);
      }
    }
    uint4 ga[V], be[V];                              // (behind the wait as well, their latency under the rows')
#pragma unroll
    for (int k = 0; k < V; ++k) {
      ga[k] = *reinterpret_cast<const uint4*>(g.ln_g + (sub + L * k) * 8);
      be[k] = *reinterpret_cast<const uint4*>(g.ln_b + (sub + L * k) * 8);
    }
    ln_rows_to_operand<NV>(x, ga, be, g.eps, sA, warp * 8, lane);
    ptx::fence_proxy_async();
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(a_ready);
    if (tid < NS / 8)
      *reinterpret_cast<uint4*>(bias_s + tid * 8) = g.bias ? *reinterpret_cast<const uint4*>(g.bias + n0 + tid * 8) : make_uint4(0, 0, 0, 0);
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kWorkers) : "memory");

    // ---- output: a thread per row and quarter of the columns, rows leave the registers as whole sectors ---------------------
    const int q = warp & 3, grp = warp >> 2, m = m0 + q * 32 + lane;
    const bool ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(d_full, 0, abort_flag, g.status) ? 1 : 0) != 0;
    if (ok) {
      ptx::tc_fence_after();
#pragma unroll
      for (int p = 0; p < NB; ++p) {
        const int c = (grp * NB + p) * 16;
        uint32_t v[16], o[8];
        ptx::tmem_ld16(tmem_base + ((uint32_t)(q * 32) << 16) + c, v);
        const uint4 b0 = *reinterpret_cast<const uint4*>(bias_s + c), b1 = *reinterpret_cast<const uint4*>(bias_s + c + 8);
        const uint32_t bw[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          float2 f = bf16x2_to_float2(bw[e]);
          f = make_float2(__uint_as_float(v[2 * e]) + f.x, __uint_as_float(v[2 * e + 1]) + f.y);
          if (g.gelu) f = make_float2(gelu_tanh(f.x), gelu_tanh(f.y));
          o[e] = float2_to_bf16x2(f.x, f.y);
        }
        if (m < g.M) ln_store16(g.out + (size_t)m * g.N + n0 + c, o, g.wide);
      }
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == kWorkers) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

template <int NV, int NB>
int launch_wave(const CUtensorMap& tw, const LnWaveArgs& g, cudaStream_t st) {
  if (ensure_max_dynamic_smem((const void*)ln_wave_kernel<NV, NB>, wave_smem_bytes<NV, NB>()) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("gemm_ln_wave", st);
  const unsigned grid = (unsigned)((g.M + BM - 1) / BM * g.slices);
  if (launch_pdl(ln_wave_kernel<NV, NB>, dim3(grid), dim3(kThreads), wave_smem_bytes<NV, NB>(), st, tw, g) != cudaSuccess) return SMARTMEM_ERR_CUDA;
  count_launch();
  return SMARTMEM_OK;
}

int launch_blocks(int nv, int nb, const CUtensorMap& tw, const LnWaveArgs& g, cudaStream_t st) {
  switch (nv * 8 + nb) {
#define SM_WAVE(NV, NB) case NV * 8 + NB: return launch_wave<NV, NB>(tw, g, st);
    SM_WAVE(2, 1) SM_WAVE(2, 2) SM_WAVE(2, 3) SM_WAVE(2, 4)
    SM_WAVE(3, 1) SM_WAVE(3, 2) SM_WAVE(3, 3) SM_WAVE(3, 4)
    SM_WAVE(4, 1) SM_WAVE(4, 2) SM_WAVE(4, 3) SM_WAVE(4, 4)
#undef SM_WAVE
  }
  return SMARTMEM_ERR_UNSUPPORTED;
}
// Columns of a slice / 64 (0: not covered, or more than one wave): the narrowest slices that fit one wave.  (Attention half:
// 1960 rows of 192 in 144 CTAs of 64 columns 14.3 us, in 48 of 192 14.8; 196 rows of 256 in 24 of 64 12.1, in 8 of 192 13.4.)  A
// second wave loses to the separate kernels (8624 rows of 192: 23.4 for 21.9 us), and so do rows of 384 and 512, whose normalisation
// in 18 and more slices takes longer than the launch it saves (588 rows of 512: 17.3 for 16.1).
int blocks_of(long long M, long long N, long long K) {
  if ((K != 128 && K != 192 && K != 256) || N % 64) return 0;
  const long long tiles = (M + BM - 1) / BM;
  for (int nb = 1; nb <= 4; ++nb)
    if ((N / 64) % nb == 0 && tiles * (N / 64 / nb) <= tc_sm_count()) return nb;
  return 0;
}

}  // namespace

bool gemm_ln_wave_wins(long long M, long long N, long long K) { return blocks_of(M, N, K) != 0; }

int launch_gemm_ln_wave(const void* X, const DevMap* rowmap, const void* gamma, const void* beta, float eps, const void* W, const void* bias,
                        int gelu, void* out, long long M, long long N, long long K, bool w_settled, cudaStream_t st) {
  const int nb = M < 1 ? 0 : blocks_of(M, N, K), ns = 64 * nb;
  if (nb == 0) return SMARTMEM_ERR_UNSUPPORTED;
  const void* ptrs[] = {X, gamma, beta, W, out};
  for (const void* p : ptrs)
    if (!p || ((uintptr_t)p & 15)) return SMARTMEM_ERR_ALIGNMENT;
  if ((uintptr_t)bias & 15) return SMARTMEM_ERR_ALIGNMENT;
  LnWaveArgs g;
  memset(&g, 0, sizeof(g));
  g.M = (int)M; g.N = (int)N; g.slices = (int)(N / ns); g.has_map = rowmap ? 1 : 0; g.gelu = gelu; g.w_settled = w_settled ? 1 : 0;
  if (rowmap) g.rowmap = *rowmap;
  g.eps = eps;
  g.x = (const __nv_bfloat16*)X; g.ln_g = (const __nv_bfloat16*)gamma; g.ln_b = (const __nv_bfloat16*)beta; g.bias = (const __nv_bfloat16*)bias; g.out = (__nv_bfloat16*)out;
  g.wide = ((uintptr_t)out & 31) == 0;
  g.status = device_status_ptr();
  if (!g.status) return SMARTMEM_ERR_CUDA;
  CUtensorMap tw;
  int rc = tc_encode_2d_blocks(W, K, N, K / BK, ns, &tw);
  return rc == SMARTMEM_OK ? launch_blocks((int)(K / 64), nb, tw, g, st) : rc;
}

}  // namespace smartmem
