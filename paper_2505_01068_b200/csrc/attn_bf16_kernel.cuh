// Kernel body of the bf16 IM attention (included by attn_bf16.cu only).
#pragma once

namespace gsit {
namespace {

// What distinguishes one attention problem of a launch from the other: its tensors, its block pattern and the order in
// which its query segments are launched.
struct AttnProblem {
  CUtensorMap tmQ, tmK, tmV;
  __nv_bfloat16* out;
  float* lse;
  uint32_t allowed;
  int seg_order;
};

template <typename C>
__global__ void __launch_bounds__(NTHREADS, C::MINB)
attn_bf16_kernel(const __grid_constant__ AttnProblem prob0, const __grid_constant__ AttnProblem prob1, const __grid_constant__ Geometry g,
                 const float sl2 /* scale * log2(e) */, const int problems) {
  // One launch can serve two problems of the same geometry that differ in their tensors and block pattern (the forward
  // and the backward ring of one encoder depth); the problem index varies fastest over the grid, so both keep the
  // longest-first launch order.
  const int which = (problems == 2) ? (int)(blockIdx.x & 1u) : 0;
  const int bx = (problems == 2) ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const AttnProblem& prob = which ? prob1 : prob0;
  __nv_bfloat16* __restrict__ out = prob.out;
  float* __restrict__ lse = prob.lse;
  constexpr int CW = C::CW, G = C::G, PITCH = C::PITCH, SWZ = C::SWZ, CPR = CW / 8 /* 16-byte chunks per row */;

  extern __shared__ uint8_t smem_raw[];
  const uint32_t sQ = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int tid = threadIdx.x;
  if (tid == 0) {
    map_early(prob.tmQ);
    map_early(prob.tmK);
    map_early(prob.tmV);
  }
  init_walk<C>(sQ, tid);
  load_params_early(g, prob.out, prob.lse, prob.allowed);
  grid_dep_wait();  // q, k, v come from the kernel before this one
  grid_dep_launch();
  const int cs = blockIdx.y, xcol = cs * CW;
  const Tile t = find_tile<C::QT>(g, prob.allowed, bx, prob.seg_order);
  if (t.T > 0) {
    __syncthreads();
    attend_tile<C, NTHREADS / 32>(g, t, prob.tmQ, prob.tmK, prob.tmV, xcol, xcol, xcol, cs, sl2, lse, sQ, [] {});
  }

  // ---- coalesced 16-byte stores; padded rows are written as +0, rows of the next segment are left alone ----
  for (int idx = tid; idx < t.rows_in_tile * CPR; idx += NTHREADS) {
    const int row = idx / CPR, ch = idx % CPR;
    uint32_t v0 = 0, v1 = 0, v2 = 0, v3 = 0;
    if (row < t.q_real)
      asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];"
                   : "=r"(v0), "=r"(v1), "=r"(v2), "=r"(v3) : "r"(sQ + swz<SWZ>(row * PITCH + ch * 16)) : "memory");
    uint4* dst = reinterpret_cast<uint4*>(out + (t.grow0 + row) * g.d + xcol + ch * 8);
    *dst = make_uint4(v0, v1, v2, v3);
  }
  if (lse != nullptr) {
    const int npad = t.rows_in_tile - t.q_real;
    for (int idx = tid; idx < npad * G; idx += NTHREADS) {
      const int row = t.q_real + idx / G, head = cs * G + idx % G;
      lse[((int64_t)t.b * g.heads + head) * g.L + g.off(t.s) + t.q0 + row] = -INFINITY;
    }
  }
}

}  // namespace
}  // namespace gsit
