// LayerNorm o gather o linear for rows of 256, 384 or 512 elements read through a map: out[m, :] = LN(X[src(m, :)]) W^T.
//
// The normalised rows of a patch merging are as large as its input: writing them and reading them back is more than half of the
// traffic, beside a launch and a dependency.  Here a pair of CTAs takes 256 rows, normalises them in registers straight into the
// operand, and multiplies them with a slice of W that stays in shared memory: only a pair has room for both (each CTA its 128
// rows and half of the slice's rows of W).  Bound by the work of one tile after the other: of about 7000 cycles for a tile of 256 x 384,
// the normalisation is 4500 (issue slots: 16 warps), the product 2000 and the output 2000, the latter two overlapped with the
// next tile's rows.  Measured against norm and linear as two kernels (us of a stream of calls, gathered rows): 25088 x 384 16.8 ->
// 14.1, 18816 x 384 14.2 -> 10.1, 37632 x 256 14.4 -> 12.1, 9408 x 512 12.3 -> 11.9; where it is taken stands at the end.
//
// Sixteen warps of rows and output (a seventeenth would leave 96 registers a thread for the 48 of rows in flight); warp 0 also
// fetches W and, in the even CTA, issues the products.  The statistics of the next tile overlap the product of this one, its
// output the product of the next (two accumulators); rows are requested four per warp ahead of the four being normalised.  Tried
// and slower: eight lanes per row (13.5 -> 15 us: twice the reads of gamma and beta), gamma and beta in registers (spills: 21), the
// map evaluated by every lane for its own vectors (1.5 us), output through shared memory (1 us).
#include <cstring>

#include "gemm_tc.cuh"
#include "ln_operand.cuh"
#include "ptx.cuh"

namespace smartmem {
namespace {

constexpr int BM = 128, BK = 64;
constexpr int kWorkers = 16, kThreads = 32 * kWorkers;

struct LnPairArgs {
  int M, N, tiles, slices, pairs, split, wide;     // tiles of 32 RW rows; pairs per slice; atoms [0, split) of the map: the row
  float eps;
  const __nv_bfloat16 *x, *ln_g, *ln_b;
  __nv_bfloat16* out;
  DevMap map;
  int* status;
};

template <int NV, int NB>
constexpr int pair_smem_bytes() {
  // rows, slice of W, gamma and beta widened and as they come, offsets of a row's vectors, barriers
  return 1024 + NV * kLnBlockBytes + NV * NB * 32 * 128 + NV * 64 * 8 + NV * 64 * 4 + NV * 8 * 4 + 5 * 8 + 8;
}

template <int NV, int NB, int RW>                  // K / 64, columns of a slice / 64, rows of a tile per warp
__global__ void __launch_bounds__(kThreads, 1)
ln_pair_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ LnPairArgs g) {
  constexpr int K = 64 * NV, NS = 64 * NB, HW = NS / 2, ROWS = kWorkers * RW;       // ROWS: of a tile per CTA
  constexpr uint32_t TM_BUF = NB == 1 ? 64 : NB == 2 ? 128 : 256, TMEM_COLS = 2 * TM_BUF;
  static_assert(pair_smem_bytes<NV, NB>() <= 227 * 1024, "operands and output of a CTA fit one SM");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sA = smem;                              // [NV][128 x 128 B]
  uint8_t* sW = sA + NV * kLnBlockBytes;           // [NV][HW x 128 B]
  // gamma and beta, widened once: floats 0-3 of every vector of eight, then floats 4-7 (16 bytes apart for neighbouring lanes)
  float* par = reinterpret_cast<float*>(sW + NV * HW * 128);
  uint4* raw = reinterpret_cast<uint4*>(par + 2 * K);                // vectors of gamma, then of beta
  int* col_s = reinterpret_cast<int*>(raw + 2 * (K / 8));            // element offset of each vector inside a row
  uint64_t* w_full = reinterpret_cast<uint64_t*>(col_s + NV * 8);
  uint64_t *a_ready = w_full + 1, *d_full = w_full + 2, *par_full = w_full + 4;      // (a_ready: the even CTA's)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(w_full + 5);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
  const int rank = (int)ptx::cluster_ctarank(), pair = (int)blockIdx.x >> 1;
  const int n0 = pair % g.slices * NS, first = pair / g.slices;

  if (warp == 0) {
    if (ptx::elect_one()) {
      ptx::mbar_init(w_full, 1);
      ptx::mbar_init(a_ready, 2 * kWorkers);
      ptx::mbar_init(&d_full[0], 1);
      ptx::mbar_init(&d_full[1], 1);
      ptx::mbar_init(par_full, K / 8);
      *abort_flag = 0;
      ptx::fence_barrier_init();
      ptx::fence_proxy_async();
      // A chain's weights are inputs like any other, perhaps still being written by the kernel before this one: before the dependency
      // wait they only come as far as L2
      ptx::tma_prefetch_3d(&tmW, 0, n0 + rank * HW, 0);
    }
    __syncwarp();
    ptx::tmem_alloc_pair(tmem_slot, TMEM_COLS);
  }
  // The map, about 700 cycles an evaluation: threads 256 and on each one vector's offset inside a row, the warps' first eight lanes
  // (below) their rows'.
  if (tid >= 256 && tid - 256 < K / 8) {
    const int v = tid - 256;
    col_s[v] = (int)devmap_part_rolled(g.map, g.split, g.map.n_atoms, (uint32_t)v).off;
    if (v < K / 64) {
      ptx::prefetch_l2(g.ln_g + v * 64);
      ptx::prefetch_l2(g.ln_b + v * 64);
    }
  }
  // the warp's eight row offsets in tile t, one evaluation of the map per lane
  auto offset_of = [&](int t) {
    const int m = t * 2 * ROWS + rank * ROWS + warp * RW + lane;
    return lane < RW && m < g.M ? g.map.base + devmap_part_rolled(g.map, 0, g.split, (uint32_t)m).off : 0ll;
  };
  long long row_off = offset_of(first);
  ptx::tc_fence_before();
  __syncwarp();
  ptx::cluster_sync();                             // both CTAs' barriers are initialised
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  {
    constexpr int L = 16, V = 8 * NV / L, J0 = 2, J1 = (RW - 4) / 2;     // four rows of a warp, then the others
    const int sub = lane % L, rsub = lane / L;
    int col[V];                                    // element offset of the lane's vectors inside a row
#pragma unroll
    for (int k = 0; k < V; ++k) col[k] = col_s[sub + L * k];
    auto request = [&](auto& x, int t, int row0, long long row_off) {      // the warp's rows from row0 of tile t
#pragma unroll
      for (int j = 0; j < (int)(sizeof(x) / sizeof(x[0])); ++j) {
        const int r = row0 + j * (32 / L) + rsub;
        const long long off = __shfl_sync(0xFFFFFFFFu, row_off, r);
        const bool in = t * 2 * ROWS + rank * ROWS + warp * RW + r < g.M;
#pragma unroll
        for (int k = 0; k < V; ++k) {
          x[j][k] = make_uint4(0, 0, 0, 0);
          if (in) x[j][k] = *reinterpret_cast<const uint4*>(g.x + off + col[k]);
        }
      }
    };
    const int q = warp & 3, grp = warp >> 2;
    const uint32_t a_ready0 = ptx::mapa(ptx::smem_u32(a_ready), 0);
    bool ok = true;
    auto product_done = [&](int it) {              // (it: the how manieth tile of the pair)
      if (ok) ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(&d_full[it & 1], (it >> 1) & 1, abort_flag, g.status) ? 1 : 0) != 0;
      if (ok) ptx::tc_fence_after();
      return ok;
    };
    auto output = [&](int it, int t) {
      int r = q * 32 + lane;
      asm volatile("" : "+r"(r));                  // (as in ln_rows_to_operand)
      const int m = t * 2 * ROWS + rank * ROWS + r;
      if (!ok || q * 32 >= ROWS) return;
#pragma unroll
      for (int p = 0; p < NB; ++p) {               // rows leave the registers as whole sectors
        uint32_t v[16], o[8];
        const int c = (grp * NB + p) * 16;
        ptx::tmem_ld16(tmem_base + (it & 1) * TM_BUF + ((uint32_t)(q * 32) << 16) + c, v);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 8; ++e) o[e] = float2_to_bf16x2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]));
        if (m < g.M && r < ROWS) ln_store16(g.out + (size_t)m * g.N + n0 + c, o, g.wide);
      }
    };
    auto affine = [&](int, int v, ptx::f32x2 (&ga)[4], ptx::f32x2 (&be)[4]) {
      const float* p = par + v * 4;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint4 a = ptx::ld_shared_v4(p + h * (K / 2)), b = ptx::ld_shared_v4(p + K + h * (K / 2));
        ga[2 * h] = ptx::pack2(__uint_as_float(a.x), __uint_as_float(a.y));
        ga[2 * h + 1] = ptx::pack2(__uint_as_float(a.z), __uint_as_float(a.w));
        be[2 * h] = ptx::pack2(__uint_as_float(b.x), __uint_as_float(b.y));
        be[2 * h + 1] = ptx::pack2(__uint_as_float(b.z), __uint_as_float(b.w));
      }
    };
    auto widen_affine = [&](int v) {
      const uint4 ga = raw[v], be = raw[K / 8 + v];
      const float2 g0 = bf16x2_to_float2(ga.x), g1 = bf16x2_to_float2(ga.y), g2 = bf16x2_to_float2(ga.z), g3 = bf16x2_to_float2(ga.w);
      const float2 b0 = bf16x2_to_float2(be.x), b1 = bf16x2_to_float2(be.y), b2 = bf16x2_to_float2(be.z), b3 = bf16x2_to_float2(be.w);
      float4* p = reinterpret_cast<float4*>(par);
      p[v] = make_float4(g0.x, g0.y, g1.x, g1.y);
      p[K / 8 + v] = make_float4(g2.x, g2.y, g3.x, g3.y);
      p[2 * (K / 8) + v] = make_float4(b0.x, b0.y, b1.x, b1.y);
      p[3 * (K / 8) + v] = make_float4(b2.x, b2.y, b3.x, b3.y);
    };
    pdl_wait();
    pdl_launch_dependents();
    auto normalise = [&](auto& x, int row0, auto&& free) {
      constexpr int J = sizeof(x) / sizeof(x[0]), JC = NV < 8 ? J : 1;   // rows of 512 two at a time: widened, four take 64 registers
      bool go = true;
#pragma unroll
      for (int j = 0; j < J; j += JC)
        go = go && ln_rows_to_operand<NV, L>(reinterpret_cast<uint4(&)[JC][V]>(x[j]), affine, g.eps, sA, warp * RW + row0 + j * (32 / L), lane,
                                             [&] { return j > 0 || free(); });
    };
    uint4 x0[J0][V], x1[J1][V];                    // rows being normalised, rows on their way
    if (warp == 0) {                               // all k-blocks of the slice in one copy
      if (ptx::elect_one()) {
        ptx::mbar_expect_tx(w_full, (uint32_t)(HW * K * 2));
        ptx::tma_load_3d(sW, &tmW, w_full, 0, n0 + rank * HW, 0);
      }
      __syncwarp();
    }
    // Gamma and beta, requested ahead of the rows; widened under the statistics of the first ones.
    const bool widens = tid >= 256 && tid - 256 < K / 8;
    if (widens) {
      ptx::cp_async16(raw + tid - 256, g.ln_g + (tid - 256) * 8);
      ptx::cp_async16(raw + K / 8 + tid - 256, g.ln_b + (tid - 256) * 8);
      ptx::cp_async_commit();
    }
    if (first < g.tiles) request(x0, first, 0, row_off);
    if (widens) {
      ptx::cp_async_wait<0>();
      widen_affine(tid - 256);
      ptx::mbar_arrive(par_full);
    }
    int it = 0;
    for (int t = first; t < g.tiles; t += g.pairs, ++it) {
      request(x1, t, 4, row_off);
      normalise(x0, 0, [&] {
        if (it > 0) return product_done(it - 1);
        return ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(par_full, 0, abort_flag, g.status) ? 1 : 0) != 0;
      });
      if (t + g.pairs < g.tiles) {
        row_off = offset_of(t + g.pairs);
        request(x0, t + g.pairs, 0, row_off);
      }
      normalise(x1, 4, [&] { return ok; });
      ptx::fence_proxy_async();
      ptx::tc_fence_before();                      // (the accumulator of the tile before last has been read)
      __syncwarp();
      // (warp 0 also answers for W, so the other CTA need not be asked)
      if (it == 0 && warp == 0) ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(w_full, 0, abort_flag, g.status) ? 1 : 0) != 0;
      if (ok && lane == 0) ptx::mbar_arrive_cluster_release(a_ready0);
      if (warp == 0 && rank == 0) {
        if (ok) ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait<true>(a_ready, it & 1, abort_flag, g.status) ? 1 : 0) != 0;
        if (ok) {
          ptx::tc_fence_after();
          const uint32_t d = tmem_base + (it & 1) * TM_BUF, a0 = ptx::smem_u32(sA), w0 = ptx::smem_u32(sW);
          constexpr uint32_t idesc = ptx::make_idesc_bf16(2 * BM, NS, false, false);
          if (ptx::elect_one()) {
#pragma unroll 1
            for (int kb = 0; kb < NV; ++kb) {      // (unrolled, the descriptors are all kept in registers across the tiles)
              const uint64_t ad = ptx::make_smem_desc(a0 + kb * kLnBlockBytes, 16, 1024), bd = ptx::make_smem_desc(w0 + kb * HW * 128, 16, 1024);
#pragma unroll
              for (int k = 0; k < BK / 16; ++k) ptx::tc_mma_bf16_pair(d, ad + 2 * k, bd + 2 * k, idesc, (kb | k) ? 1u : 0u);
            }
            ptx::tc_commit_pair(&d_full[it & 1], 3);
          }
          __syncwarp();
        }
      }
      if (it > 0) output(it - 1, t - g.pairs);
    }
    if (it > 0) {
      product_done(it - 1);
      output(it - 1, first + (it - 1) * g.pairs);
    }
  }
  ptx::tc_fence_before();
  __syncwarp();
  ptx::cluster_sync_relaxed();                     // neither CTA leaves while the other may still signal it or use its memory
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(tmem_base, TMEM_COLS);
  }
}

// Columns of a slice / 64: what fits beside the rows.
int blocks_of(long long K) { return K == 256 || K == 512 ? 2 : K == 384 ? 3 : 0; }

template <int NV, int NB, int RW>
int launch_pair(const CUtensorMap& tw, const LnPairArgs& g, cudaStream_t st) {
  if (ensure_max_dynamic_smem((const void*)ln_pair_kernel<NV, NB, RW>, pair_smem_bytes<NV, NB>()) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("gemm_ln_pair", st);
  const unsigned grid = (unsigned)(2 * g.slices * g.pairs);
  if (launch_pdl_cluster(ln_pair_kernel<NV, NB, RW>, dim3(grid), dim3(kThreads), pair_smem_bytes<NV, NB>(), st, 2u, tw, g) != cudaSuccess)
    return SMARTMEM_ERR_CUDA;
  count_launch();
  return SMARTMEM_OK;
}

}  // namespace

// The rows are normalised once per slice of the columns, so several slices win only while they all fit one round of pairs.  Norm and
// linear as two kernels -> this one, us of a stream of calls, gathered rows: 3136 x 256 in 3 slices 7.1 -> 6.5, 9408 x 256 in 2 8.7 -> 7.6,
// 9408 x 384 in 2 12.3 -> 10.0, 9408 x 512 in 2 12.3 -> 11.9; beyond a round 12544 x 256 in 2 10.0 -> 10.4, 12544 x 384 in 2 12.6 -> 13.8,
// 12544 x 512 in 2 13.8 -> 16.0, 25088 x 384 in 6 (LayerNorm into a QKV projection) 33 -> 60.  One slice wins with any number of rounds
// for rows of 256 and 384 (25088: 11.5 -> 10.7, 16.8 -> 14.1).
// Small calls are bound by the host, and what decides there is the second launch it saves: through the Python binding 10.3 -> 7.5 us.
// (On the device alone two kernels whose launches overlap are the shorter ones: 1568 x 384 in one slice 6.3 against 7.4, 784 x 512 in
// eight 7.1 against 8.4.)
bool gemm_ln_pair_wins(const smartmem_index_map_t& map, long long M, long long N, long long K) {
  const int nb = blocks_of(K);
  if (!nb || N % (64 * nb) || M < 1) return false;
  const long long tiles = (M + 2 * BM - 1) / (2 * BM);
  const long long slices = N / (64 * nb), work = tiles * slices, pairs = tc_cluster_ctas(2) / 2;
  if (work > pairs && (slices > 1 || K == 512)) return false;
  return M < (1ll << 31) / 4 && map.klass < 2 && map.vec_elems == 8 &&
         map.n_elements == M * K;
}

int launch_gemm_ln_pair(const void* X, const smartmem_index_map_t& map, const void* gamma, const void* beta, float eps, const void* W,
                        void* out, long long M, long long N, long long K, cudaStream_t st) {
  if (!gemm_ln_pair_wins(map, M, N, K)) return SMARTMEM_ERR_UNSUPPORTED;
  LnPairArgs g;
  memset(&g, 0, sizeof(g));
  if (!make_devmap(map, 0, map.n_atoms, 8, true, &g.map)) return SMARTMEM_ERR_UNSUPPORTED;
  g.split = devmap_split(g.map, K / 8);
  long long reach = 0;                                               // the largest offset inside a row
  for (int a = g.split; g.split >= 0 && a < g.map.n_atoms; ++a) reach += (long long)(g.map.ext[a].d - 1) * (g.map.stride[a] < 0 ? -g.map.stride[a] : g.map.stride[a]);
  if (g.split < 0 || g.map.n_rolls || reach >= (1ll << 31)) return SMARTMEM_ERR_UNSUPPORTED;
  const int nb = blocks_of(K), ns = 64 * nb;
  g.M = (int)M; g.N = (int)N; g.slices = (int)(N / ns);
  const int fit = tc_cluster_ctas(2) / 2 / g.slices;                 // pairs of a slice that run at once
  // Tiles of 256 rows, or of 192 where that leaves the busiest pair fewer: 25088 rows on 74 pairs are two rounds either way (15.0 us
  // with 256, 13.5 with 192).
  auto rounds = [&](int rows) { return ((M + rows - 1) / rows + fit - 1) / fit; };
  const bool narrow = rounds(192) * 192 < rounds(256) * 256;
  const int rows = narrow ? 192 : 256;
  g.tiles = (int)((M + rows - 1) / rows);
  g.pairs = g.tiles < fit ? g.tiles : fit;
  g.eps = eps;
  g.x = (const __nv_bfloat16*)X; g.ln_g = (const __nv_bfloat16*)gamma; g.ln_b = (const __nv_bfloat16*)beta; g.out = (__nv_bfloat16*)out;
  g.wide = ((uintptr_t)out & 31) == 0;
  g.status = device_status_ptr();
  if (!g.status) return SMARTMEM_ERR_CUDA;
  CUtensorMap tw;
  int rc = tc_encode_2d_blocks(W, K, N, K / BK, ns / 2, &tw);
  if (rc != SMARTMEM_OK) return rc;
  if (K == 256) return narrow ? launch_pair<4, 2, 6>(tw, g, st) : launch_pair<4, 2, 8>(tw, g, st);
  if (K == 512) return narrow ? launch_pair<8, 2, 6>(tw, g, st) : launch_pair<8, 2, 8>(tw, g, st);
  return narrow ? launch_pair<6, 3, 6>(tw, g, st) : launch_pair<6, 3, 8>(tw, g, st);
}

}  // namespace smartmem
