// Read-out of the fusion stack (paper, Eq. "All-Modal-In-One fusion": X_m = f(|| Split(a(G_intra))[-1])): the last real
// time step of each modality segment, concatenated, through the linear map f.  float accumulation; weights float or bf16.
//
// A few hundred kilobytes of work, so latency is all there is: a CTA takes 16 output features of one sample (two per
// warp), so that 64 samples x 128 features are 512 CTAs instead of 64, gathers the three rows into shared memory, and every
// lane has all its weight loads (16 bytes each) in flight at once.  One CTA per sample with 16 features per warp one after
// the other and 2-byte loads took 27 us at 64 samples, 31 us at one.
#include "common.cuh"
#include "ptx.cuh"

namespace gsit {
namespace {

constexpr int HEAD_WARPS = 8, HEAD_PER_WARP = 2;

__device__ __forceinline__ float dot_chunk(const float* z, const uint4& u, const float*) {
  return z[0] * __uint_as_float(u.x) + z[1] * __uint_as_float(u.y) + z[2] * __uint_as_float(u.z) + z[3] * __uint_as_float(u.w);
}
__device__ __forceinline__ float dot_chunk(const float* z, const uint4& u, const __nv_bfloat16*) {
  float a = 0.f;
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i)
    a = fmaf(z[2 * i], __uint_as_float(w[i] << 16), fmaf(z[2 * i + 1], __uint_as_float(w[i] & 0xffff0000u), a));
  return a;
}

// VEC: the weight rows are whole numbers of 16-byte chunks
template <typename WT, bool VEC>
__global__ void __launch_bounds__(HEAD_WARPS * 32)
stack_head_kernel(const __grid_constant__ Geometry g, const float* __restrict__ c, const int64_t ldc, const int dc, const WT* __restrict__ w,
                  const float* __restrict__ bias, float* __restrict__ out, const int n_out) {
  extern __shared__ __align__(16) float z[];  // [3 * dc]
  const int b = blockIdx.x, K = 3 * dc;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int o0 = (blockIdx.y * HEAD_WARPS + warp) * HEAD_PER_WARP;
  ptx::load_params_early(g, c, ldc, w, bias, out);
  ptx::grid_dep_wait();
  ptx::grid_dep_launch();
  for (int i = threadIdx.x; i < K; i += blockDim.x) {
    const int s = i / dc, e = i - s * dc;
    const int n = valid_rows(g, b, s);
    z[i] = (n > 0) ? c[((int64_t)b * g.L + g.off(s) + n - 1) * ldc + e] : 0.f;
  }
  __syncthreads();
  float acc[HEAD_PER_WARP] = {};
  if constexpr (VEC) {
    constexpr int E = 16 / sizeof(WT), IN_FLIGHT = 2;
    const int chunks = K / E;
    for (int c0 = lane; c0 < chunks; c0 += 32 * IN_FLIGHT) {
      uint4 u[HEAD_PER_WARP][IN_FLIGHT];
#pragma unroll
      for (int i = 0; i < HEAD_PER_WARP; ++i)
#pragma unroll
        for (int j = 0; j < IN_FLIGHT; ++j)
          u[i][j] = (o0 + i < n_out && c0 + 32 * j < chunks)
                        ? __ldg(reinterpret_cast<const uint4*>(w + (int64_t)(o0 + i) * K) + c0 + 32 * j) : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int j = 0; j < IN_FLIGHT; ++j) {
        if (c0 + 32 * j >= chunks) continue;
#pragma unroll
        for (int i = 0; i < HEAD_PER_WARP; ++i) acc[i] += dot_chunk(z + (c0 + 32 * j) * E, u[i][j], w);
      }
    }
  } else {
    for (int k = lane; k < K; k += 32)
#pragma unroll
      for (int i = 0; i < HEAD_PER_WARP; ++i)
        if (o0 + i < n_out) acc[i] = fmaf((float)w[(int64_t)(o0 + i) * K + k], z[k], acc[i]);
  }
#pragma unroll
  for (int i = 0; i < HEAD_PER_WARP; ++i) {
    for (int sft = 16; sft; sft >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], sft);
    if (lane == 0 && o0 + i < n_out) out[(int64_t)b * n_out + o0 + i] = acc[i] + (bias ? bias[o0 + i] : 0.f);
  }
}

template <typename WT>
cudaError_t launch(const Geometry& g, const float* c, int64_t ldc, int dc, const void* w, const float* bias, float* out, int n_out,
                   cudaStream_t st) {
  constexpr int PER_CTA = HEAD_WARPS * HEAD_PER_WARP;
  const size_t smem = (size_t)3 * dc * sizeof(float);
  if (smem > 48 * 1024 || (n_out + PER_CTA - 1) / PER_CTA > 65535) return cudaErrorNotSupported;
  const dim3 grid(g.batch, (n_out + PER_CTA - 1) / PER_CTA);
  const bool vec = (3 * dc * sizeof(WT)) % 16 == 0 && (reinterpret_cast<uintptr_t>(w) & 15u) == 0;
  return vec ? launch_overlapped(stack_head_kernel<WT, true>, grid, dim3(HEAD_WARPS * 32), smem, st, g, c, ldc, dc,
                                 static_cast<const WT*>(w), bias, out, n_out)
             : launch_overlapped(stack_head_kernel<WT, false>, grid, dim3(HEAD_WARPS * 32), smem, st, g, c, ldc, dc,
                                 static_cast<const WT*>(w), bias, out, n_out);
}

}  // namespace

cudaError_t launch_stack_head(const Geometry& g, int dtype, const float* c, int64_t ldc, int dc, const void* w,
                              const float* bias, float* out, int n_out, cudaStream_t st) {
  return dtype == GSIT_BF16 ? launch<__nv_bfloat16>(g, c, ldc, dc, w, bias, out, n_out, st)
                            : launch<float>(g, c, ldc, dc, w, bias, out, n_out, st);
}

}  // namespace gsit
