// LayerNorm of 128 rows in registers, written to shared memory as a tcgen05 operand: shared by the kernels that normalise the rows
// of one tile and multiply them where they are (gemm_ln_wave.cu, gemm_ln_pair.cu, gemm_mlp_cluster.cu, swin_attn_cluster.cu).
#pragma once
#include "common.cuh"
#include "ptx.cuh"

namespace smartmem {
namespace {

constexpr int kLnBlockBytes = 128 * 64 * 2;        // one 128 x 64 operand block: 16 KB

__device__ __forceinline__ ptx::f32x2 ln_widen(uint32_t w) { return ptx::pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u)); }
__device__ __forceinline__ float ln_hsum(ptx::f32x2 v) {
  float lo, hi;
  ptx::unpack2(v, lo, hi);
  return lo + hi;
}
__device__ __forceinline__ void ln_widen8(const uint4& u, ptx::f32x2 (&w)[4]) {
  w[0] = ln_widen(u.x); w[1] = ln_widen(u.y); w[2] = ln_widen(u.z); w[3] = ln_widen(u.w);
}

// Lanes that share a row of 64 NV elements: few (fewer reductions) while gamma and beta fit the registers beside a warp's eight rows.
constexpr int ln_lanes(int NV) { return NV <= 3 ? 8 : 16; }

// J * 32 / L rows of a warp, from tile row `row0`: x[j][k] is vector sub + L k of row row0 + (32 / L) j + lane / L, sub = lane % L.  The operand is K-major in blocks of 64 columns, 128-byte swizzled; `free` is called (by whole warps) before it is
// written and says whether it may be; `affine(k, v, gamma, beta)` gives the widened parameters of the lane's vector k, vector v of the
// row.  Issue-bound: the values are widened once and stay so.
template <int NV, int L, int J, int V, typename P, typename F>
__device__ __forceinline__ bool ln_rows_to_operand(const uint4 (&x)[J][V], P&& affine, float eps, uint8_t* sA, int row0, int lane, F&& free) {
  static_assert(V * L == 8 * NV, "a row's vectors over its lanes");
  asm volatile("" : "+r"(lane));                     // (the addresses below are not kept from one call to the next)
  const int sub = lane % L, rsub = lane / L;
  ptx::f32x2 w[J][V][4];
  float mean[J], rstd[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    ptx::f32x2 s = ptx::pack2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < V; ++k) {
      ln_widen8(x[j][k], w[j][k]);
      s = ptx::add2(s, ptx::add2(ptx::add2(w[j][k][0], w[j][k][1]), ptx::add2(w[j][k][2], w[j][k][3])));
    }
    mean[j] = ln_hsum(s);
  }
#pragma unroll
  for (int d = L / 2; d > 0; d >>= 1)
#pragma unroll
    for (int j = 0; j < J; ++j) mean[j] += __shfl_xor_sync(0xFFFFFFFFu, mean[j], d);
#pragma unroll
  for (int j = 0; j < J; ++j) {
    mean[j] *= 1.0f / (float)(64 * NV);
    const ptx::f32x2 m = ptx::pack2(-mean[j], -mean[j]);
    ptx::f32x2 s0 = ptx::pack2(0.f, 0.f), s1 = s0;
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const ptx::f32x2 a = ptx::add2(w[j][k][0], m), b = ptx::add2(w[j][k][1], m), c = ptx::add2(w[j][k][2], m), d = ptx::add2(w[j][k][3], m);
      s0 = ptx::fma2(a, a, ptx::fma2(b, b, s0));
      s1 = ptx::fma2(c, c, ptx::fma2(d, d, s1));
    }
    rstd[j] = ln_hsum(ptx::add2(s0, s1));
  }
#pragma unroll
  for (int d = L / 2; d > 0; d >>= 1)
#pragma unroll
    for (int j = 0; j < J; ++j) rstd[j] += __shfl_xor_sync(0xFFFFFFFFu, rstd[j], d);
  if (!free()) return false;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    rstd[j] = rsqrtf(rstd[j] * (1.0f / (float)(64 * NV)) + eps);
    mean[j] = -mean[j] * rstd[j];
  }
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const int v = sub + k * L;                       // chunk v % 8 of k-block v / 8
    ptx::f32x2 ga[4], be[4];
    affine(k, v, ga, be);
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int r = row0 + j * (32 / L) + rsub;
      const ptx::f32x2 r2 = ptx::pack2(rstd[j], rstd[j]), m2 = ptx::pack2(mean[j], mean[j]);
      uint32_t o[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float lo, hi;
        ptx::unpack2(ptx::fma2(ptx::fma2(w[j][k][e], r2, m2), ga[e], be[e]), lo, hi);
        o[e] = float2_to_bf16x2(lo, hi);
      }
      *reinterpret_cast<uint4*>(sA + (v >> 3) * kLnBlockBytes + r * 128 + (((v ^ r) & 7) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
  return true;
}
template <int NV, int J = ln_lanes(NV) / 4, int V = 8 * NV / ln_lanes(NV)>
__device__ __forceinline__ void ln_rows_to_operand(const uint4 (&x)[J][V], const uint4 (&ga)[V], const uint4 (&be)[V], float eps, uint8_t* sA,
                                                   int row0, int lane) {
  ln_rows_to_operand<NV, ln_lanes(NV)>(x, [&](int k, int, ptx::f32x2 (&g)[4], ptx::f32x2 (&b)[4]) { ln_widen8(ga[k], g); ln_widen8(be[k], b); }, eps, sA,
                         row0, lane, [] { return true; });
}

// Sixteen bf16 columns of an output row: one whole sector, where the output is aligned to sectors.
__device__ __forceinline__ void ln_store16(__nv_bfloat16* p, const uint32_t (&o)[8], int wide) {
  const uint4 a = make_uint4(o[0], o[1], o[2], o[3]), b = make_uint4(o[4], o[5], o[6], o[7]);
  if (wide) {
    ptx::st_global_v8(p, a, b);
  } else {
    *reinterpret_cast<uint4*>(p) = a;
    *reinterpret_cast<uint4*>(p + 8) = b;
  }
}

}  // namespace
}  // namespace smartmem
