// Causal attention (prefill, head dimension 128) on the tcgen05 tensor cores.
//
// One CTA = 128 query positions of one head.  K and V stream through shared memory in tiles of
// 64 keys (TMA, three stages of keys and two of values a group); S = Q K^T and O += P V are tcgen05.mma with the accumulators in
// TMEM (two S buffers and one O a group: 256 columns); the four warps of a softmax group own one query row per thread (the TMEM lane),
// so row maxima and sums need no shuffles.  P goes back to the tensor core through tensor memory: it is
// written as bf16 pairs over the S buffer it was computed from and read by the second MMA as its A
// operand; V is consumed as it lies in memory ([key, d] rows) through the MN-major operand mode, so no
// transpose of V exists anywhere.  The running maximum is only
// refreshed when it grows by more than 2^8 (then O and the running sum are rescaled), which keeps
// the TMEM read-modify-write of O off the common path.
//
// A tile's softmax is a chain of about 1500 cycles for its group, in which the SM is nearly idle.  Where the query tiles fill the chip
// twice, TWO CTAs of one group share an SM (112 KB of shared memory and 256 TMEM columns each): while one is in its softmax the
// other one's MMAs run.  Where they do not, a CTA has two groups, which take the key tiles in turn with a running maximum, a sum and
// an O of their own; the shares of a row meet at the end in the threads that own its lane, so the longest rows take half as long.
//
// q, k, v are addressed as TMA boxes inside the buffer the QKV GEMM wrote ([B*S, 3*H*D], head split
// eliminated) or inside materialised [B, H, S, D] tensors (explicit variant); the output tile is
// stored at column h*D of [B*S, H*D] (head merge eliminated) or into [B, H, S, D].
#include "attn.cuh"
#include "gemm_tc.cuh"
#include "ptx.cuh"


namespace smartmem {
namespace {

constexpr int BQ = 128, BKV = 64, D = 128;
constexpr int KB = 128 * 64 * 2;                      // one 128 x 64 bf16 block (Q, P)
constexpr int KBK = BKV * 64 * 2;                     // one 64 x 64 bf16 block (K, V)
// G softmax groups: key tile j belongs to group j % G, which has two S buffers of 64 columns and an O of 128
template <int G>
struct Sizes {
  static constexpr int NS = 2 * G, KSTAGES = 3 * G, VSTAGES = 2 * G, THREADS = 64 + 128 * G;
  static constexpr uint32_t TM_S = 0, TM_O = NS * BKV, TMEM_COLS = 256 * G;
  static constexpr int N_BARS = 1 + 2 * KSTAGES + 2 * VSTAGES + 3 * NS + G + 1;
  static constexpr uint32_t SMEM = 2 * KB + 2 * (KSTAGES + VSTAGES) * KBK + N_BARS * 8 + 16 + (G > 1 ? G * BQ * 8 : 0);
};
constexpr float kRescaleThreshold = 8.0f;             // log2 units

struct TcAttnArgs {
  int S, heads, batch, n_qt;
  int q_col0, k_col0, v_col0, col_per_head;           // TMA column of (operand, head): col0 + h * col_per_head
  int plane_per_batch, plane_per_head;                // a plane of the TMA maps holds S rows: b * plane_per_batch + h * plane_per_head
  __nv_bfloat16* out;
  long long o_sn, o_sh, o_st;
  float scale_log2;
  uint32_t smem_bytes;
  int* status;
};

__device__ __forceinline__ float max3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}

template <int G>
__global__ void __launch_bounds__(Sizes<G>::THREADS, 3 - G)
causal_attn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                      const __grid_constant__ CUtensorMap tmV, const __grid_constant__ TcAttnArgs g) {
  using Z = Sizes<G>;
  constexpr int KSTAGES = Z::KSTAGES, VSTAGES = Z::VSTAGES, NS = Z::NS;
  constexpr uint32_t TM_S = Z::TM_S, TM_O = Z::TM_O, TMEM_COLS = Z::TMEM_COLS;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t pad = (1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u;
  uint8_t* smem = smem_raw + pad;
  uint8_t* sQ = smem;                                  // [2 k-blocks][16 KB]
  uint8_t* sK = sQ + 2 * KB;                           // [stages][2 k-blocks][8 KB]
  uint8_t* sV = sK + 2 * KSTAGES * KBK;                // [stages][2 d-chunks][8 KB]
  uint64_t* bars = reinterpret_cast<uint64_t*>(sV + 2 * VSTAGES * KBK);
  uint64_t *q_full = bars, *k_full = bars + 1, *k_empty = k_full + KSTAGES, *v_full = k_empty + KSTAGES, *v_empty = v_full + VSTAGES;
  uint64_t *s_full = v_empty + VSTAGES, *s_empty = s_full + NS, *p_full = s_empty + NS, *p_empty = p_full + NS, *o_done = p_empty + G;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + Z::N_BARS);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  float2* ml_s = reinterpret_cast<float2*>(tmem_slot + 4);      // (G > 1) [G][128]: a row's maximum and sum over its group's keys

  if (pad + Z::SMEM > g.smem_bytes) {
    if (threadIdx.x == 0) atomicExch(g.status, (int)SMARTMEM_ERR_UNSUPPORTED);
    return;
  }
  const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (warp: provably uniform)
  // heaviest units (last query tiles) first
  const int bh_count = g.batch * g.heads;
  const int qt = g.n_qt - 1 - (int)(blockIdx.x / bh_count);
  const int bh = (int)(blockIdx.x % bh_count);
  const int b = bh / g.heads, h = bh - b * g.heads;
  const int n_kv = min(2 * (qt + 1), (g.S + BKV - 1) / BKV);   // 64-key blocks up to and including the diagonal
  const int plane = b * g.plane_per_batch + h * g.plane_per_head;

  if (threadIdx.x == 0) {
    ptx::mbar_init(q_full, 1);
    for (int i = 0; i < KSTAGES; ++i) {
      ptx::mbar_init(&k_full[i], 1);
      ptx::mbar_init(&k_empty[i], 1);
    }
    for (int i = 0; i < VSTAGES; ++i) {
      ptx::mbar_init(&v_full[i], 1);
      ptx::mbar_init(&v_empty[i], 1);
    }
    for (int i = 0; i < NS; ++i) {
      ptx::mbar_init(&s_full[i], 1);
      ptx::mbar_init(&s_empty[i], 1);                 // P(j) lives in S buffer j % NS: freed by the commit of P V (j)
    }
    // (a barrier per S buffer: the softmax may be two tiles ahead of P V, and with one for both the issuing warp, held up for that long by a
    // slow read in its wait, found the phase that it waited for already followed by another and waited for good)
    for (int i = 0; i < NS; ++i) ptx::mbar_init(&p_full[i], 4);
    for (int i = 0; i < G; ++i) ptx::mbar_init(&p_empty[i], 1);
    ptx::mbar_init(o_done, 1);
    *abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tensormap(&tmQ);
    ptx::prefetch_tensormap(&tmK);
    ptx::prefetch_tensormap(&tmV);
  }
  if (warp == 1) ptx::tmem_alloc(tmem_slot, TMEM_COLS);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();                       // the set-up above overlapped the previous kernel's tail
  pdl_launch_dependents();

  if (warp == 0) {
    // Keys run a tile ahead of the values, one copy per tile of each, issued by an elected lane of a warp-uniform loop: with two
    // stages of both, four copies a tile issued under a branch on one lane and K(j + 1) behind the wait for V(j), a tile's keys
    // arrived 1.9 us after the products that freed their stage -- the period of a tile (S = 2048, 32 heads: 53 us).
    const int qc = (g.q_col0 + h * g.col_per_head) / 64, kc = (g.k_col0 + h * g.col_per_head) / 64, vc = (g.v_col0 + h * g.col_per_head) / 64;
    if (ptx::elect_one()) {
      ptx::mbar_expect_tx(q_full, 2 * KB);
      ptx::tma_load_4d(sQ, &tmQ, q_full, 0, qt * BQ, qc, plane);
    }
    __syncwarp();
    bool ok = true;
    uint32_t ks = 0, kph = 1;
    for (int i = -1; i < n_kv && ok; ++i) {
      if (i + 1 < n_kv) {
        ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(&k_empty[ks], kph, abort_flag, g.status) ? 1 : 0) != 0;
        if (!ok) break;
        if (ptx::elect_one()) {
          ptx::mbar_expect_tx(&k_full[ks], 2 * KBK);
          ptx::tma_load_4d(sK + ks * 2 * KBK, &tmK, &k_full[ks], 0, (i + 1) * BKV, kc, plane);
        }
        __syncwarp();
        if (++ks == KSTAGES) { ks = 0; kph ^= 1; }
      }
      if (i >= 0) {
        const int s = i % VSTAGES;
        ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(&v_empty[s], ((i / VSTAGES) & 1) ^ 1, abort_flag, g.status) ? 1 : 0) != 0;
        if (!ok) break;
        if (ptx::elect_one()) {
          ptx::mbar_expect_tx(&v_full[s], 2 * KBK);
          ptx::tma_load_4d(sV + s * 2 * KBK, &tmV, &v_full[s], 0, i * BKV, vc, plane);
        }
        __syncwarp();
      }
    }
  } else if (warp == 1) {
    // the whole warp walks the issue loop and an elected lane issues: warp-uniform control flow keeps the
    // descriptors in uniform registers
    {
      const uint32_t idesc_s = ptx::make_idesc_bf16(BQ, BKV, false, false);
      const uint32_t idesc_pv = ptx::make_idesc_bf16(BQ, D, false, true);      // V: MN-major B operand
      bool ok = __all_sync(0xFFFFFFFFu, ptx::mbar_wait(q_full, 0, abort_flag, g.status) ? 1 : 0) != 0;
      uint32_t kst = 0, kph = 0;
      auto issue_s = [&](int j) {
        const int s = j % NS;
        const uint32_t ph = (j / NS) & 1;
        ok = ok && ptx::mbar_wait(&s_empty[s], ph ^ 1, abort_flag, g.status);
        ok = ok && ptx::mbar_wait(&k_full[kst], kph, abort_flag, g.status);
        ok = __all_sync(0xFFFFFFFFu, ok ? 1 : 0) != 0;
        if (!ok) return;
        ptx::tc_fence_after();
        if (ptx::elect_one()) {
#pragma unroll
          for (int kb = 0; kb < 2; ++kb) {
            const uint64_t ad = ptx::make_smem_desc(ptx::smem_u32(sQ + kb * KB), 16, 1024);
            const uint64_t bd = ptx::make_smem_desc(ptx::smem_u32(sK + (kst * 2 + kb) * KBK), 16, 1024);
#pragma unroll
            for (int k = 0; k < 4; ++k)                 // a k16 step moves both start addresses by 32 bytes
              ptx::tc_mma_bf16(tmem_base + TM_S + s * BKV, ad + 2 * k, bd + 2 * k, idesc_s, (kb | k) ? 1u : 0u);
          }
          ptx::tc_commit(&k_empty[kst]);
          ptx::tc_commit(&s_full[s]);
        }
        __syncwarp();
        if (++kst == KSTAGES) { kst = 0; kph ^= 1; }
      };
      auto issue_pv = [&](int j) {
        static_assert(NS == VSTAGES, "one index for both");
        const int s = j % NS;
        ok = ok && ptx::mbar_wait(&p_full[s], (j / NS) & 1, abort_flag, g.status);
        ok = ok && ptx::mbar_wait(&v_full[s], (j / NS) & 1, abort_flag, g.status);
        ok = __all_sync(0xFFFFFFFFu, ok ? 1 : 0) != 0;
        if (!ok) return;
        ptx::tc_fence_after();
        const uint32_t v0 = ptx::smem_u32(sV + s * 2 * KBK);
        const uint64_t vd = ptx::make_smem_desc(v0, KBK, 1024);
        const uint32_t pa = tmem_base + TM_S + s * BKV;  // P(j): bf16 pairs over the first 32 columns of the S buffer it came from
        if (ptx::elect_one()) {
#pragma unroll
          for (int ks = 0; ks < BKV / 16; ++ks)        // 16 keys per step: P +8 packed columns, V +16 rows of 128 bytes; the two 64-wide d-chunks are KBK apart
            ptx::tc_mma_bf16_ta(tmem_base + TM_O + (j % G) * D, pa + 8 * ks, vd + (2048 >> 4) * ks, idesc_pv, (j >= G || ks) ? 1u : 0u);
          ptx::tc_commit(&v_empty[s]);
          ptx::tc_commit(&s_empty[s]);
          ptx::tc_commit(&p_empty[j % G]);
        }
        __syncwarp();
      };
      for (int j = 0; j < G && j < n_kv && ok; ++j) issue_s(j);
      for (int j = 0; j < n_kv && ok; ++j) {
        if (j + G < n_kv) issue_s(j + G);
        issue_pv(j);
      }
      if (ok && ptx::elect_one()) ptx::tc_commit(o_done);
    }
  } else {
    const int q = warp & 3;                            // TMEM lane quadrant
    const int r = q * 32 + lane;                       // query row inside the tile
    const int qi = qt * BQ + r;                        // position
    const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
    const int gi = G > 1 ? (warp - 2) >> 2 : 0;
    float m_used = -INFINITY, l = 0.f;
    bool ok = true;
    for (int j = gi, turn = 0; j < n_kv && ok; j += G, ++turn) {
      const int sb = j % NS;
      ok = ptx::mbar_wait(&s_full[sb], (j / NS) & 1, abort_flag, g.status);
      if (!ok) break;
      ptx::tc_fence_after();
      const uint32_t ts = tmem_base + TM_S + sb * BKV + lane_addr;
      const bool diag = (j >= 2 * qt);                 // the two 64-key blocks that straddle this tile's diagonal
      const int kj0 = j * BKV;
      // the whole score row of this thread: four loads in flight, one wait
      uint32_t rv[BKV];
#pragma unroll
      for (int ch = 0; ch < BKV / 32; ++ch) ptx::tmem_ld32(ts + ch * 32, rv + ch * 32);
      ptx::tmem_ld_wait();
      if (diag) {                                      // keys beyond the row's position
#pragma unroll
        for (int c = 0; c < BKV; ++c)
          if (kj0 + c > qi) rv[c] = 0xFF800000u;       // -inf
      }
      float mx4[4];                                    // row maximum, four independent chains of three-way maxima
#pragma unroll
      for (int k = 0; k < 4; ++k) mx4[k] = __uint_as_float(rv[k]);
#pragma unroll
      for (int c = 4; c < BKV; c += 2) mx4[(c >> 1) & 3] = max3(mx4[(c >> 1) & 3], __uint_as_float(rv[c]), __uint_as_float(rv[c + 1]));
      float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * g.scale_log2;   // the scale is positive
      float corr = 1.f;
      bool rescale = false;
      if (mx > m_used + kRescaleThreshold) {           // (first tile: m_used = -inf)
        corr = ptx::ex2(m_used - mx);                       // 0 on the first tile
        l *= corr;
        m_used = mx;
        rescale = turn > 0;
      }
      // (the second group's first tile can lie past the row's position as a whole: its probabilities are 2^-inf then)
      const float nm = G > 1 && m_used == -INFINITY ? 0.f : -m_used;
      // p = 2^(s - m), packed to bf16 for the second MMA
      uint32_t pk[BKV / 2];
      const ptx::f32x2 sc2 = ptx::pack2(g.scale_log2, g.scale_log2), nm2 = ptx::pack2(nm, nm);
      ptx::f32x2 l2[2] = {ptx::pack2(0.f, 0.f), ptx::pack2(0.f, 0.f)};
#pragma unroll
      for (int c = 0; c < BKV; c += 2) {
        float e0, e1;
        ptx::unpack2(ptx::fma2(ptx::pack2(__uint_as_float(rv[c]), __uint_as_float(rv[c + 1])), sc2, nm2), e0, e1);
        const float p0 = ptx::ex2(e0), p1 = ptx::ex2(e1);
        l2[(c >> 1) & 1] = ptx::add2(l2[(c >> 1) & 1], ptx::pack2(p0, p1));
        pk[c / 2] = float2_to_bf16x2(p0, p1);
      }
      {
        float l0, l1;
        ptx::unpack2(ptx::add2(l2[0], l2[1]), l0, l1);
        l += l0 + l1;
      }
      if (__any_sync(0xFFFFFFFFu, rescale)) {
        // O is rescaled in place: the previous P V, which accumulates into it, must have completed
        ok = ptx::mbar_wait(&p_empty[gi], (turn & 1) ^ 1, abort_flag, g.status);
        if (!ok) break;
        ptx::tc_fence_after();
        const uint32_t to = tmem_base + TM_O + gi * D + lane_addr;
#pragma unroll 1
        for (int ch = 0; ch < 4; ++ch) {
          uint32_t ro[32];
          ptx::tmem_ld32(to + ch * 32, ro);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 32; ++c) ro[c] = __float_as_uint(__uint_as_float(ro[c]) * (rescale ? corr : 1.f));
          ptx::tmem_st32(to + ch * 32, ro);
        }
        ptx::tmem_st_wait();
      }
      // P row r (bf16 pairs) over the first 32 columns of the S buffer this thread has just read: each
      // warp touches only its own lanes, and the buffer is not reused before P V (j) has completed
      ptx::tmem_st32(ts, pk);
      ptx::tmem_st_wait();
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&p_full[sb]);
    }
    // the groups' shares of a row meet: O = (O0 w0 + O1 w1) / (l0 w0 + l1 w1), w = 2^(m - max m), each group storing half of the columns
    float w0 = 1.f, w1 = 0.f, lsum = l;
    if constexpr (G > 1) {
      ml_s[gi * BQ + r] = make_float2(m_used, l);
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const float2 a = ml_s[r], c = ml_s[BQ + r];
      const float mt = fmaxf(a.x, c.x);
      w0 = ptx::ex2(a.x - mt);
      w1 = ptx::ex2(c.x - mt);
      lsum = a.y * w0 + c.y * w1;
    }
    if (ok) ok = ptx::mbar_wait(o_done, 0, abort_flag, g.status);
    if (ok) {
      ptx::tc_fence_after();
      const float inv = 1.f / lsum;
      const bool wide_store = (reinterpret_cast<uintptr_t>(g.out) & 31) == 0 && g.o_sn % 16 == 0 && g.o_sh % 16 == 0 && g.o_st % 16 == 0;
      __nv_bfloat16* orow = g.out + (long long)b * g.o_sn + (long long)h * g.o_sh + (long long)qi * g.o_st;
      const uint32_t to = tmem_base + TM_O + lane_addr;
#pragma unroll 1
      for (int ch = gi * (4 / G); ch < (gi + 1) * (4 / G); ++ch) {
        uint32_t rv[32];
        ptx::tmem_ld32(to + ch * 32, rv);
        if constexpr (G > 1) {
          uint32_t rw[32];
          ptx::tmem_ld32(to + D + ch * 32, rw);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 32; ++c) rv[c] = __float_as_uint(__uint_as_float(rv[c]) * w0 + __uint_as_float(rw[c]) * w1);
        }
        ptx::tmem_ld_wait();
        if (qi < g.S && wide_store) {                    // whole 32-byte sectors per store
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            uint32_t w[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
              w[e] = float2_to_bf16x2(__uint_as_float(rv[v * 16 + 2 * e]) * inv, __uint_as_float(rv[v * 16 + 2 * e + 1]) * inv);
            ptx::st_global_v8(orow + ch * 32 + v * 16, make_uint4(w[0], w[1], w[2], w[3]), make_uint4(w[4], w[5], w[6], w[7]));
          }
        } else if (qi < g.S) {
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            float o8[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) o8[e] = __uint_as_float(rv[v * 8 + e]) * inv;
            ElemIO<__nv_bfloat16>::store(orow + ch * 32 + v * 8, o8);
          }
        }
      }
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

}  // namespace

// Returns SMARTMEM_ERR_UNSUPPORTED when the operand layout is neither of the two it knows.
int launch_causal_attention_tc(const CausalAttnArgs& a, cudaStream_t st) {
  const long long S = a.S, H = a.heads, B = a.batch;
  if (S < 1 || H < 1 || B < 1) return SMARTMEM_ERR_UNSUPPORTED;
  const AttnOperand* ops[3] = {&a.q, &a.k, &a.v};
  for (auto* o : ops)
    if (o->se != 1 || ((uintptr_t)o->ptr & 15)) return SMARTMEM_ERR_UNSUPPORTED;
  if (a.o.se != 1 || a.o.st % 8 || a.o.sn % 8 || a.o.sh % 8 || ((uintptr_t)a.o.ptr & 15)) return SMARTMEM_ERR_UNSUPPORTED;
  TcAttnArgs g;
  memset(&g, 0, sizeof(g));
  CUtensorMap tq, tk, tv;
  int rc;
  const long long st_ = a.q.st;
  const bool interleaved = a.q.sh == D && a.k.sh == D && a.v.sh == D && a.k.st == st_ && a.v.st == st_ &&
                           a.q.sn == S * st_ && a.k.sn == S * st_ && a.v.sn == S * st_ && st_ % 8 == 0;
  const bool head_major = a.q.st == D && a.k.st == D && a.v.st == D && a.q.sh == S * D && a.k.sh == S * D &&
                          a.v.sh == S * D && a.q.sn == H * S * D && a.k.sn == H * S * D && a.v.sn == H * S * D;
  // Rows past a sequence's end are a plane's end, which reads as zeros: they meet probabilities of zero, and the next sequence's values, which
  // need not be finite, would make NaN of them.
  const int qbox[4] = {64, BQ, 2, 1}, kbox[4] = {64, BKV, 2, 1};
  if (interleaved) {
    // one [B*S, row pitch] matrix holds q, k and v side by side; columns are offsets from q
    const long long kcol = ((const char*)a.k.ptr - (const char*)a.q.ptr) / 2, vcol = ((const char*)a.v.ptr - (const char*)a.q.ptr) / 2;
    if (kcol < 0 || vcol < 0 || kcol + H * D > st_ || vcol + H * D > st_) return SMARTMEM_ERR_UNSUPPORTED;
    if (kcol % 64 || vcol % 64) return SMARTMEM_ERR_UNSUPPORTED;
    // [64 columns][row][chunk of 64 columns][sequence]: both chunks of a head in one copy
    const long long dims[4] = {64, S, st_ / 64, B}, strides[3] = {st_, 64, S * st_};
    if ((rc = tc_encode_nd_sw128(a.q.ptr, 4, dims, strides, qbox, &tq)) != SMARTMEM_OK) return rc;
    if ((rc = tc_encode_nd_sw128(a.q.ptr, 4, dims, strides, kbox, &tk)) != SMARTMEM_OK) return rc;   // same buffer, 64-row boxes
    tv = tk;
    g.q_col0 = 0; g.k_col0 = (int)kcol; g.v_col0 = (int)vcol; g.col_per_head = D;
    g.plane_per_batch = 1; g.plane_per_head = 0;
  } else if (head_major) {
    const long long dims[4] = {64, S, 2, B * H}, strides[3] = {D, 64, S * D};
    if ((rc = tc_encode_nd_sw128(a.q.ptr, 4, dims, strides, qbox, &tq)) != SMARTMEM_OK) return rc;
    if ((rc = tc_encode_nd_sw128(a.k.ptr, 4, dims, strides, kbox, &tk)) != SMARTMEM_OK) return rc;
    if ((rc = tc_encode_nd_sw128(a.v.ptr, 4, dims, strides, kbox, &tv)) != SMARTMEM_OK) return rc;
    g.col_per_head = 0;
    g.plane_per_batch = (int)H; g.plane_per_head = 1;
  } else {
    return SMARTMEM_ERR_UNSUPPORTED;
  }
  if (B * H * S >= (1ll << 31)) return SMARTMEM_ERR_UNSUPPORTED;
  g.S = (int)S; g.heads = (int)H; g.batch = (int)B;
  g.n_qt = (int)((S + BQ - 1) / BQ);
  g.out = (__nv_bfloat16*)a.o.ptr;
  g.o_sn = a.o.sn; g.o_sh = a.o.sh; g.o_st = a.o.st;
  g.scale_log2 = a.scale * 1.4426950408889634f;
  g.status = device_status_ptr();
  if (!g.status) return SMARTMEM_ERR_CUDA;
  const long long ctas = (long long)g.n_qt * B * H;
  if (ctas >= (1ll << 31)) return SMARTMEM_ERR_UNSUPPORTED;
  // Two softmax groups on an SM's one CTA, or two CTAs of one group each: the first where every CTA has an SM to itself, or nearly so and
  // the longest rows decide.  Us of a layer, one group -> two: 48 CTAs (2 x 333, hidden 1024) 23.9 -> 21.6, 96 (2 x 333, 2048) 37.8 -> 35.5, (1 x 1500,
  // 1024) 42.5 -> 37.4, 128 (1 x 2048, 1024) 50.9 -> 46.6, (1 x 512, 4096) 94.1 -> 90.5; 192 (1 x 1500, 2048) 75.1 -> 68.1, 256 (1 x 2048, 2048) 91.6 -> 89.5,
  // but 192 (4 x 333, 2048) 54.7 -> 55.7, 256 (4 x 512, 2048) 69.7 -> 71.5, 384 (1 x 1500, 4096) 187 -> 194, 512 (1 x 2048, 4096) 289 -> 307.
  const bool two = S > BKV && (ctas <= tc_sm_count() || (ctas <= 2 * tc_sm_count() && g.n_qt >= 10));
  // 112 KB of tiles: two CTAs per SM only fit without a spare kilobyte of alignment slack (the kernel
  // reports a misaligned base instead of overrunning)
  const size_t smem = two ? Sizes<2>::SMEM : Sizes<1>::SMEM;
  g.smem_bytes = (uint32_t)smem;
  auto* kern = two ? causal_attn_tc_kernel<2> : causal_attn_tc_kernel<1>;
  if (ensure_max_dynamic_smem((const void*)kern, (int)smem, 100) != SMARTMEM_OK) return SMARTMEM_ERR_CUDA;
  profile_tick("causal_attention_tc", st);
  launch_pdl(kern, dim3((unsigned)ctas), dim3(two ? Sizes<2>::THREADS : Sizes<1>::THREADS), smem, st, tq, tk, tv, g);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? SMARTMEM_OK : SMARTMEM_ERR_CUDA;
}

}  // namespace smartmem
