// Pieces of the bf16 layer on row tiles of 16 R rows and mma.sync (d_model 32, 64, 128):
//   normalise_tile   LayerNorm of float rows into a tile of bf16 rows in shared memory
//   qkv_units        that tile times W_qkv^T + b_qkv, to global memory
//
// The weights take the shortest way there is: each lane loads its B fragments straight from global memory as 16-byte pieces (all
// CTAs read the same few tens of kilobytes: they stay in L1), no shared-memory staging, no barrier per weight chunk.  For that the k
// index of a product is permuted, the same way in both operands: lane t of a quad holds k = 32 i + 8 t .. + 7 of its rows, which
// serve two m16n8k16 steps.  The A operand lies in shared memory as bf16 rows in 16-byte pieces, swizzled so that the fragment reads
// (16 bytes per lane) and the writes from accumulators (4 bytes per lane) are both free of bank conflicts.
// A row's result does not depend on R, on the tile it falls into or on the layout.
#pragma once
#include "common.cuh"
#include "ptx.cuh"

namespace gsit {
namespace {

constexpr int THREADS = 256, ROW_WARPS = 8, ROWS_MAX_FF = 512;

__device__ __forceinline__ void mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Byte offset of 16-byte piece c of row r in a tile of K bf16 columns.
template <int K>
__device__ __forceinline__ uint32_t piece(int r, int c) {
  if constexpr (K == 32) return (uint32_t)(r * 64 + ((c ^ ((r >> 1) & 3)) << 4));
  else return (uint32_t)(r * (K * 2) + ((c ^ (((r & 1) << 2) | ((r >> 1) & 3))) << 4));
}
__device__ __forceinline__ uint4 lds16(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts4(uint32_t a, uint32_t v) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void sts8(uint32_t a, uint32_t v, uint32_t w) { asm volatile("st.shared.v2.b32 [%0], {%1,%2};" ::"r"(a), "r"(v), "r"(w) : "memory"); }

// Two k-steps (32 k's): rows of the slab at `lo` (row g) and `hi` (row g + 8), weights w of one n-tile.
__device__ __forceinline__ void step(float (&c)[4], const uint4& lo, const uint4& hi, const uint4& w) {
  mma(c, lo.x, hi.x, lo.y, hi.y, w.x, w.y);
  mma(c, lo.z, hi.z, lo.w, hi.w, w.z, w.w);
}
__device__ __forceinline__ uint4 ldw(const __nv_bfloat16* p) { return __ldg(reinterpret_cast<const uint4*>(p)); }

// LayerNorm of the tile's rows, eight threads per row, T / 8 rows at a time: load(r, e) gives columns e .. e + 3 of row r, real(r) says
// whether it is one (else it becomes zero).  Returns whether any row of this thread is real.
template <int D, int BM, int T = THREADS, typename Real, typename Load>
__device__ __forceinline__ bool normalise_tile(const float* gamma, const float* beta, float eps, uint32_t h, int tid, Real real_row, Load load) {
  constexpr int V = D / 32;  // float4s per thread of a row
  bool any = false;
#pragma unroll
  for (int pass = 0; pass < (BM + T / 8 - 1) / (T / 8); ++pass) {
    const int r = pass * (T / 8) + (tid >> 3);
    const bool real = r < BM && real_row(r);
    any |= real;
    float4 v[V];
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < V; ++c) v[c] = real ? load(r, 4 * ((tid & 7) + 8 * c)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int c = 0; c < V; ++c) s += (v[c].x + v[c].y) + (v[c].z + v[c].w);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float mean = s * (1.f / D);
    float q = 0.f;
#pragma unroll
    for (int c = 0; c < V; ++c) {
      v[c].x -= mean; v[c].y -= mean; v[c].z -= mean; v[c].w -= mean;
      q += fmaf(v[c].x, v[c].x, v[c].y * v[c].y) + fmaf(v[c].z, v[c].z, v[c].w * v[c].w);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    const float rstd = rsqrtf(q * (1.f / D) + eps);
    if (r < BM) {
#pragma unroll
      for (int c = 0; c < V; ++c) {
        const int e = 4 * ((tid & 7) + 8 * c);
        const float4 ga = gamma != nullptr ? make_float4(gamma[e], gamma[e + 1], gamma[e + 2], gamma[e + 3]) : make_float4(1.f, 1.f, 1.f, 1.f);
        const float4 be = beta != nullptr ? make_float4(beta[e], beta[e + 1], beta[e + 2], beta[e + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
        const uint32_t lo = ptx::pack_bf16(fmaf(v[c].x * rstd, ga.x, be.x), fmaf(v[c].y * rstd, ga.y, be.y));
        const uint32_t hi = ptx::pack_bf16(fmaf(v[c].z * rstd, ga.z, be.z), fmaf(v[c].w * rstd, ga.w, be.w));
        sts8(h + piece<D>(r, e >> 3) + (e & 4) * 2, real ? lo : 0u, real ? hi : 0u);
      }
    }
  }
  return any;
}

// qkv rows m0 + r (those the CTA owns; zeros where not real) = normalised tile h times W_qkv^T + b_qkv.  work: any real row at all?
// weights(row, k): this lane's 16-byte piece (32 k + 8 t ..) of a row of W_qkv.
template <int D, int R, int WARPS = ROW_WARPS, typename W, typename Own, typename Real>
__device__ __forceinline__ void qkv_units(W weights, const float* b_qkv, __nv_bfloat16* qkv, const int64_t m0, uint32_t h, bool work,
                                          int tid, Own own, Real real_row) {
  constexpr int GROUPS = 3 * D / 16, UNITS = GROUPS * R;
  const int warp = tid >> 5, lane = tid & 31, gr = lane >> 2, t = lane & 3;
  // units of 16 columns x one slab of 16 rows.  The two n-tiles of a unit take their columns interleaved, so that a lane ends up
  // with four consecutive ones: 8-byte stores, 32-byte sectors written whole.
#pragma unroll
  for (int u = warp; u < UNITS; u += WARPS) {
    const int grp = u % GROUPS, slab = u / GROUPS, n0 = grp * 16;
    float c[2][4] = {};
    if (work) {
      uint4 w[2][D / 32];
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int k = 0; k < D / 32; ++k) w[j][k] = weights(n0 + 4 * (gr >> 1) + (gr & 1) + 2 * j, k);
#pragma unroll
      for (int k = 0; k < D / 32; ++k) {
        const uint4 lo = lds16(h + piece<D>(slab * 16 + gr, 4 * k + t)), hi = lds16(h + piece<D>(slab * 16 + gr + 8, 4 * k + t));
        step(c[0], lo, hi, w[0][k]);
        step(c[1], lo, hi, w[1][k]);
      }
    }
    float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
    if (b_qkv != nullptr) {
      const float* p = b_qkv + n0 + 4 * t;
      b = make_float4(p[0], p[1], p[2], p[3]);
    }
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int r = slab * 16 + gr + 8 * half;
      if (!own(r)) continue;
      const bool real = work && real_row(r);
      const uint32_t lo = ptx::pack_bf16(c[0][2 * half] + b.x, c[0][2 * half + 1] + b.y), hi = ptx::pack_bf16(c[1][2 * half] + b.z, c[1][2 * half + 1] + b.w);
      *reinterpret_cast<uint2*>(qkv + (m0 + r) * (3 * D) + n0 + 4 * t) = real ? make_uint2(lo, hi) : make_uint2(0u, 0u);
    }
  }
}

}  // namespace
}  // namespace gsit
