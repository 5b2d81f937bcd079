// Linear layers and LayerNorm around the IM attention: C = act(A W^T + bias) (+ residual).
//   - bf16: cp.async-pipelined mma.sync.m16n8k16 tiles, float accumulate, fused bias / ReLU / residual /
//     padded-row zeroing epilogue, bf16 or float output.
// (float operands: linear_f32.cu)
#include "common.cuh"
#include "ptx.cuh"

namespace gsit {
namespace {

// ------------------------------------------------------------------------------------------------ bf16
constexpr int BM = 128, BK = 32, GSTAGES = 3;

__device__ __forceinline__ uint32_t swz64(uint32_t off) { return off ^ (((off >> 7) & 3) << 4); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool pred) {
  const int sz = pred ? 16 : 0;  // size 0 zero-fills the 16 destination bytes
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
}

template <int BN>
__global__ void __launch_bounds__(256) linear_bf16_kernel(const __grid_constant__ Geometry g, const __grid_constant__ LinearArgs a) {
  constexpr int WGN = (BN == 128) ? 4 : 2, WGM = 8 / WGN;
  constexpr int WTM = BM / WGM, WTN = BN / WGN;  // warp tile
  constexpr int MT = WTM / 16, NTL = WTN / 8;
  constexpr int A_BYTES = BM * BK * 2, W_BYTES = BN * BK * 2;
  __shared__ __align__(1024) uint8_t smem[GSTAGES * (A_BYTES + W_BYTES)];
  const uint32_t sA = smem_u32(smem), sW = sA + GSTAGES * A_BYTES;
  const __nv_bfloat16* A = static_cast<const __nv_bfloat16*>(a.A);
  const __nv_bfloat16* W = static_cast<const __nv_bfloat16*>(a.W);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wm = warp / WGN, wn = warp % WGN;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int KT_ = (a.K + BK - 1) / BK;
  ptx::load_params_early(g, a);
  ptx::grid_dep_wait();  // the weights, too: this kernel may be the first of a call, right behind the one that wrote them
  ptx::grid_dep_launch();

  auto load_stage = [&](int kt, int st) {
    const int k0 = kt * BK;
    for (int idx = tid; idx < BM * 4; idx += 256) {  // 4 chunks of 16 B per 32-wide row
      const int r = idx >> 2, c = idx & 3;
      const bool ok = (m0 + r < a.M) && (k0 + c * 8 < a.K);
      const __nv_bfloat16* src = ok ? A + (int64_t)(m0 + r) * a.lda + k0 + c * 8 : A;
      cp_async16(sA + st * A_BYTES + swz64(r * 64 + c * 16), src, ok);
    }
    for (int idx = tid; idx < BN * 4; idx += 256) {
      const int r = idx >> 2, c = idx & 3;
      const bool ok = (n0 + r < a.N) && (k0 + c * 8 < a.K);
      const __nv_bfloat16* src = ok ? W + (int64_t)(n0 + r) * a.K + k0 + c * 8 : W;
      cp_async16(sW + st * W_BYTES + swz64(r * 64 + c * 16), src, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  float acc[MT][NTL][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NTL; ++j) acc[i][j][0] = acc[i][j][1] = acc[i][j][2] = acc[i][j][3] = 0.f;

  for (int s = 0; s < GSTAGES - 1; ++s) {
    if (s < KT_) load_stage(s, s);
    else asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int kt = 0; kt < KT_; ++kt) {
    asm volatile("cp.async.wait_group %0;" ::"n"(GSTAGES - 2) : "memory");
    __syncthreads();
    if (kt + GSTAGES - 1 < KT_) load_stage(kt + GSTAGES - 1, (kt + GSTAGES - 1) % GSTAGES);
    else asm volatile("cp.async.commit_group;" ::: "memory");
    const int st = kt % GSTAGES;
    const uint32_t aS = sA + st * A_BYTES, wS = sW + st * W_BYTES;
#pragma unroll
    for (int ks = 0; ks < BK / 16; ++ks) {
      uint32_t af[MT][4], bf[NTL][2];
      const int mi = lane >> 3;
#pragma unroll
      for (int i = 0; i < MT; ++i) {
        const int row = wm * WTM + i * 16 + (mi & 1) * 8 + (lane & 7);
        const uint32_t ad = aS + swz64(row * 64 + (ks * 2 + (mi >> 1)) * 16);
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(af[i][0]), "=r"(af[i][1]), "=r"(af[i][2]), "=r"(af[i][3]) : "r"(ad));
      }
#pragma unroll
      for (int j = 0; j < NTL / 2; ++j) {
        const int row = wn * WTN + j * 16 + (mi >> 1) * 8 + (lane & 7);
        const uint32_t ad = wS + swz64(row * 64 + (ks * 2 + (mi & 1)) * 16);
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(bf[2 * j][0]), "=r"(bf[2 * j][1]), "=r"(bf[2 * j + 1][0]), "=r"(bf[2 * j + 1][1]) : "r"(ad));
      }
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NTL; ++j)
          asm volatile(
              "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
              : "+f"(acc[i][j][0]), "+f"(acc[i][j][1]), "+f"(acc[i][j][2]), "+f"(acc[i][j][3])
              : "r"(af[i][0]), "r"(af[i][1]), "r"(af[i][2]), "r"(af[i][3]), "r"(bf[j][0]), "r"(bf[j][1]));
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");

  // ---- epilogue: bias, ReLU, residual, padded rows -> 0 ----
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int m = m0 + wm * WTM + i * 16 + (lane >> 2) + half * 8;
      if (m >= a.M) continue;
      const bool real = !a.mask_rows || row_is_real(g, m);
#pragma unroll
      for (int j = 0; j < NTL; ++j) {
        const int n = n0 + wn * WTN + j * 8 + (lane & 3) * 2;
        if (n >= a.N) continue;  // N is even, so n + 1 < N as well
        float v0 = acc[i][j][half * 2], v1 = acc[i][j][half * 2 + 1];
        if (a.bias) { v0 += a.bias[n]; v1 += a.bias[n + 1]; }
        if (a.relu) { v0 = fmaxf(v0, 0.f); v1 = fmaxf(v1, 0.f); }
        if (a.residual) {
          const float2 r = *reinterpret_cast<const float2*>(a.residual + (int64_t)m * a.ldr + n);
          v0 += r.x; v1 += r.y;
        }
        if (!real) v0 = v1 = 0.f;
        if (a.out_f32)
          *reinterpret_cast<float2*>(static_cast<float*>(a.C) + (int64_t)m * a.ldc + n) = make_float2(v0, v1);
        else
          *reinterpret_cast<__nv_bfloat162*>(static_cast<__nv_bfloat16*>(a.C) + (int64_t)m * a.ldc + n) =
              __floats2bfloat162_rn(v0, v1);
      }
    }
}

// ------------------------------------------------------------------------------------------------ LayerNorm
// Reads 4 and writes 2 or 4 bytes per element and is bound by that traffic; a warp per row, the row in registers.
// CHUNKS > 0: d = 128 * CHUNKS and 16-byte rows: every lane has its CHUNKS 16-byte loads in flight at once, the row is read
// once, and a warp keeps gamma and beta in registers over many rows (loading them for every row costs more L1 cycles than
// the row itself: 217 us; 4-byte loads in three passes: 201 us; now 143 us at 278528 x 512).  CHUNKS = 0: any d.
template <typename OutT, int CHUNKS>
__global__ void __launch_bounds__(256) layernorm_kernel(const __grid_constant__ Geometry g, const float* __restrict__ x, const int64_t ldx,
                                                        const float* __restrict__ gamma, const float* __restrict__ beta,
                                                        const float eps, OutT* __restrict__ y, const int rows) {
  const int lane = threadIdx.x & 31, d = g.d;
  int row = (int)(blockIdx.x * 8 + (threadIdx.x >> 5));
  auto is_real = [&](int r) {
    const int b = r / g.L, p = r - b * g.L, s = segment_of(g, p);
    return p - g.off(s) < valid_rows(g, b, s);
  };
  ptx::load_params_early(g, x, ldx, gamma, beta, y);
  ptx::grid_dep_wait();
  ptx::grid_dep_launch();
  if constexpr (CHUNKS > 0) {
    float ga[4 * CHUNKS], be[4 * CHUNKS];
#pragma unroll
    for (int i = 0; i < 4 * CHUNKS; ++i) {
      const int e = 4 * (lane + 32 * (i >> 2)) + (i & 3);
      ga[i] = gamma ? gamma[e] : 1.f;
      be[i] = beta ? beta[e] : 0.f;
    }
    for (; row < rows; row += gridDim.x * 8) {
      const bool real = is_real(row);
      const float* xr = x + (int64_t)row * ldx;
      OutT* yr = y + (int64_t)row * d;
      float4 v[CHUNKS];
      float sum = 0.f;
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) v[c] = real ? __ldcs(reinterpret_cast<const float4*>(xr) + lane + 32 * c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) sum += (v[c].x + v[c].y) + (v[c].z + v[c].w);
      for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const float mean = sum / d;
      float vs = 0.f;
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) {
        v[c].x -= mean; v[c].y -= mean; v[c].z -= mean; v[c].w -= mean;
        vs += fmaf(v[c].x, v[c].x, v[c].y * v[c].y) + fmaf(v[c].z, v[c].z, v[c].w * v[c].w);
      }
      for (int o = 16; o; o >>= 1) vs += __shfl_xor_sync(0xffffffffu, vs, o);
      const float rstd = rsqrtf(vs / d + eps);
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) {
        const int e = 4 * (lane + 32 * c);
        const float t[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
        float f[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) f[j] = real ? t[j] * rstd * ga[4 * c + j] + be[4 * c + j] : 0.f;
        if constexpr (sizeof(OutT) == 2)
          *reinterpret_cast<uint2*>(yr + e) = make_uint2(ptx::pack_bf16(f[0], f[1]), ptx::pack_bf16(f[2], f[3]));
        else
          *reinterpret_cast<float4*>(yr + e) = make_float4(f[0], f[1], f[2], f[3]);
      }
    }
    return;
  }
  if (row >= rows) return;
  const bool real = is_real(row);
  const float* xr = x + (int64_t)row * ldx;
  OutT* yr = y + (int64_t)row * d;
  if (!real) {
    for (int e = lane; e < d; e += 32) yr[e] = OutT(0.f);
    return;
  }
  float sum = 0.f;
  for (int e = lane; e < d; e += 32) sum += xr[e];
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const float mean = sum / d;
  float vs = 0.f;
  for (int e = lane; e < d; e += 32) { const float t = xr[e] - mean; vs = fmaf(t, t, vs); }
  for (int o = 16; o; o >>= 1) vs += __shfl_xor_sync(0xffffffffu, vs, o);
  const float rstd = rsqrtf(vs / d + eps);
  for (int e = lane; e < d; e += 32) {
    const float v = (xr[e] - mean) * rstd * (gamma ? gamma[e] : 1.f) + (beta ? beta[e] : 0.f);
    yr[e] = OutT(v);
  }
}

template <typename OutT>
cudaError_t layernorm(const Geometry& g, const float* x, int64_t ldx, const float* gamma, const float* beta, float eps, void* y,
                      cudaStream_t st) {
  const int rows = g.batch * g.L;
  const bool vec = g.d % 128 == 0 && ldx % 4 == 0 && ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15u) == 0;
  const int chunks = vec && g.d <= 1024 ? g.d / 128 : 0;
  auto kernel = chunks == 1 ? layernorm_kernel<OutT, 1> : chunks == 2 ? layernorm_kernel<OutT, 2> : chunks == 3 ? layernorm_kernel<OutT, 3>
                : chunks == 4 ? layernorm_kernel<OutT, 4> : chunks == 6 ? layernorm_kernel<OutT, 6> : chunks == 8 ? layernorm_kernel<OutT, 8>
                : layernorm_kernel<OutT, 0>;
  int n_sm = 0;
  cudaError_t e = sm_count_and_smem_once(nullptr, 0, &n_sm);
  if (e != cudaSuccess) return e;
  const int blocks = (rows + 7) / 8;
  return launch_overlapped(kernel, dim3((unsigned)(chunks > 0 && blocks > 6 * n_sm ? 6 * n_sm : blocks)), dim3(256), 0, st, g, x, ldx, gamma, beta, eps, static_cast<OutT*>(y), rows);
}

}  // namespace

extern int g_attn_variant;  // kernel selection (attn_bf16.cu): GSIT_ATTN_LEGACY keeps every bf16 kernel on the mma.sync path

cudaError_t launch_linear_bf16(const Geometry& g, const LinearArgs& a, cudaStream_t st) {
  if (g_attn_variant != GSIT_ATTN_LEGACY && linear_tc_supported(a)) return launch_linear_tc_bf16(g, a, st);
  if (a.K % 8 != 0 || a.N % 2 != 0 || a.lda % 8 != 0) return cudaErrorNotSupported;
  const bool wide = (a.N % 128 == 0) || a.N > 256;
  const int bn = wide ? 128 : 64;
  const dim3 grid((a.N + bn - 1) / bn, (a.M + BM - 1) / BM);
  if (grid.y > 65535) return cudaErrorNotSupported;
  return launch_overlapped(wide ? linear_bf16_kernel<128> : linear_bf16_kernel<64>, grid, dim3(256), 0, st, g, a);
}

cudaError_t launch_layernorm(const Geometry& g, const float* x, int64_t ldx, const float* gamma, const float* beta,
                             float eps, void* y, int out_bf16, cudaStream_t st) {
  return out_bf16 ? layernorm<__nv_bfloat16>(g, x, ldx, gamma, beta, eps, y, st) : layernorm<float>(g, x, ldx, gamma, beta, eps, y, st);
}

}  // namespace gsit
