// LayerNorm of 128 rows in registers, written to shared memory as a tcgen05 operand: shared by the kernels that normalise the rows
// of one tile and multiply them where they are (gemm_ln_wave.cu, gemm_mlp_cluster.cu).
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
// eight bf16 values: their sum, the sum of (x + nm)^2, and (x rs + ms) g + b in fp32, rounded once
__device__ __forceinline__ float ln_sum8(const uint4& u) {
  return ln_hsum(ptx::add2(ptx::add2(ln_widen(u.x), ln_widen(u.y)), ptx::add2(ln_widen(u.z), ln_widen(u.w))));
}
__device__ __forceinline__ float ln_sq8(const uint4& u, float nm) {
  const ptx::f32x2 m = ptx::pack2(nm, nm), a = ptx::add2(ln_widen(u.x), m), b = ptx::add2(ln_widen(u.y), m), c = ptx::add2(ln_widen(u.z), m),
                   d = ptx::add2(ln_widen(u.w), m);
  return ln_hsum(ptx::add2(ptx::fma2(a, a, ptx::mul2(b, b)), ptx::fma2(c, c, ptx::mul2(d, d))));
}
__device__ __forceinline__ uint32_t ln_affine2(uint32_t w, ptx::f32x2 rs, ptx::f32x2 ms, uint32_t g, uint32_t b) {
  float lo, hi;
  ptx::unpack2(ptx::fma2(ptx::fma2(ln_widen(w), rs, ms), ln_widen(g), ln_widen(b)), lo, hi);
  return float2_to_bf16x2(lo, hi);
}

// Lanes that share a row of 64 NV elements: few while gamma and beta fit the registers beside the rows (fewer reductions).
constexpr int ln_lanes(int NV) { return NV <= 3 ? 8 : 16; }

// A warp's eight rows (of 16 warps' 128): x[j][k] is vector sub + L k of row 8 warp + (32 / L) j + lane / L, sub = lane % L, L =
// ln_lanes(NV).  The operand is K-major in blocks of 64 columns, 128-byte swizzled.
template <int NV, int J = ln_lanes(NV) / 4, int V = 8 * NV / ln_lanes(NV)>
__device__ __forceinline__ void ln_rows_to_operand(const uint4 (&x)[J][V], const uint4 (&ga)[V], const uint4 (&be)[V], float eps, uint8_t* sA,
                                                   int warp, int lane) {
  constexpr int L = ln_lanes(NV);
  const int sub = lane % L, rsub = lane / L;
  float mean[J], rstd[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    mean[j] = 0.f;
#pragma unroll
    for (int k = 0; k < V; ++k) mean[j] += ln_sum8(x[j][k]);
  }
#pragma unroll
  for (int d = L / 2; d > 0; d >>= 1)
#pragma unroll
    for (int j = 0; j < J; ++j) mean[j] += __shfl_xor_sync(0xFFFFFFFFu, mean[j], d);
#pragma unroll
  for (int j = 0; j < J; ++j) {
    mean[j] *= 1.0f / (float)(64 * NV);
    rstd[j] = 0.f;
#pragma unroll
    for (int k = 0; k < V; ++k) rstd[j] += ln_sq8(x[j][k], -mean[j]);
  }
#pragma unroll
  for (int d = L / 2; d > 0; d >>= 1)
#pragma unroll
    for (int j = 0; j < J; ++j) rstd[j] += __shfl_xor_sync(0xFFFFFFFFu, rstd[j], d);
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int r = warp * 8 + j * (32 / L) + rsub;
    rstd[j] = rsqrtf(rstd[j] * (1.0f / (float)(64 * NV)) + eps);
    const float ms = -mean[j] * rstd[j];
    const ptx::f32x2 r2 = ptx::pack2(rstd[j], rstd[j]), m2 = ptx::pack2(ms, ms);
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const int v = sub + k * L;                     // chunk v % 8 of k-block v / 8
      *reinterpret_cast<uint4*>(sA + (v >> 3) * kLnBlockBytes + r * 128 + (((v ^ r) & 7) << 4)) =
          make_uint4(ln_affine2(x[j][k].x, r2, m2, ga[k].x, be[k].x), ln_affine2(x[j][k].y, r2, m2, ga[k].y, be[k].y),
                     ln_affine2(x[j][k].z, r2, m2, ga[k].z, be[k].z), ln_affine2(x[j][k].w, r2, m2, ga[k].w, be[k].w));
    }
  }
}

}  // namespace
}  // namespace smartmem
