// A layer behind its QKV projection in one launch, on small row tiles and mma.sync (d_model 32, 64, 128):
//   attention -> out-projection + residual -> LN2 -> MLP + residual -> (the next layer's LN1 + QKV)
//
// Everything behind the attention is row-wise, so a CTA that attends with ALL heads for 16 (32, 64) query rows takes those rows through
// the rest of the layer, and through the next layer's first half, without another CTA's result: attention rows, normalised rows and
// hidden units stay in shared memory, and a layer is one launch instead of three.  What bounds small problems is the chain of dependent
// launches (each a wait for its predecessor, a round trip through L2, a tail), not what any of them computes.  The whole model on one
// sample of (50, 500, 500): 130 -> 88 us (20 launches -> 9); a layer at d 64 there 18.4 -> 14.2, at d 128 23.6 -> 20.9, on 1100 rows of
// (50, 250, 250) at d 64 14.7 -> 11.3, at d 32 12.6 -> 9.1.
// Of a launch at d 64 (16 rows per CTA, one sample; clocks): 2.1 K before the wait, 8 K the walk (4 K of it exponentials, one CTA per SM),
// 1.5 K out-projection + LN2, 1.1 K hidden units, 1.4 K the rest; all of them chains of shared-memory reads, four dependent mma and a barrier.
//
// 16 warps: as many attend as there are heads x 16-row slabs; all share the row-wise part.  Weights (W_o only at d 128, where the rest
// does not fit) and parameters come into shared memory by cp.async while the walk runs.
// The arithmetic is that of the separate kernels (attn_bf16_tile.cuh, rows_tile.cuh, fused_rows.cu), operation by operation: the same
// bits, so that which of them runs may depend on the number of problems and on the size of a batch.
#include "attn_bf16_tile.cuh"
#include "rows_tile.cuh"

namespace gsit {
namespace {

struct LayerProblem {
  CUtensorMap tmQ, tmKV;  // the fused qkv rows [rows, 3 d], boxes of QT and of KT rows
  FusedHalfArgs h;        // ln1 / qkv of it: the next layer's, or qkv null
  uint32_t allowed;
  int seg_order;
};

// A weight matrix of K columns in shared memory: rows of 2 K bytes, 64 bytes apart where those were whole 128-byte lines, so that the
// fragment reads (16 bytes per lane: two rows x 64 bytes at a time) touch every bank once.
template <int K>
struct Staged { static constexpr int PITCH = (2 * K) % 128 == 0 ? 2 * K + 64 : 2 * K; };
__device__ __forceinline__ void copy16(uint32_t dst, const void* src) { asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void copy4(uint32_t dst, const float* src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory"); }

// The 16 warps of a CTA in the row-wise part of a tile of 16 R rows: WN along the D output columns (NT groups of 8 each), WM along the
// 16-row slabs, two along the hidden units of the last product.
constexpr int TAIL_THREADS = 512, TAIL_WARPS = 16;
template <int D, int R>
struct TailTile {
  static constexpr int BM = 16 * R, KD = D / 32, WN = D / 8 < 8 ? D / 8 : 8, NT = D / 8 / WN, WK = 2, WM = TAIL_WARPS / (WN * WK), SW = R / WM;
  static constexpr int YP = D + 4;                                       // float pitch of the result rows
  static_assert(R % WM == 0, "tile");
  // parameters in shared memory, floats: b_o, ln2 gamma, beta, b_2, then the next layer's ln1 gamma, beta, b_qkv, then b_1
  static constexpr int P_BO = 0, P_G2 = D, P_E2 = 2 * D, P_B2 = 3 * D, P_G1 = 4 * D, P_E1 = 5 * D, P_BQ = 6 * D, P_B1 = 9 * D;
  // behind the walk the K and V stages hold the row-wise part's tiles: normalised rows, hidden units, result rows, shares of sums
  static constexpr int OFF_F = BM * D * 2;
  __host__ __device__ static constexpr int off_y(int d_ff) { return OFF_F + BM * d_ff * 2; }
  __host__ __device__ static constexpr int off_red(int d_ff) { return off_y(d_ff) + BM * YP * 4; }
  __host__ __device__ static constexpr int bytes(int d_ff) { return off_red(d_ff) + (WK - 1) * BM * D * 4; }
  __host__ __device__ static constexpr int param_bytes(int d_ff) { return (9 * D + d_ff) * 4; }
  // weights in shared memory, behind the parameters: all of them at D <= 64, W_o at 128 (the others do not fit)
  static constexpr bool ALL = D <= 64;
  static constexpr int PD = Staged<D>::PITCH;
  __host__ __device__ static constexpr int pf(int d_ff) { return (2 * d_ff) % 128 == 0 ? 2 * d_ff + 64 : 2 * d_ff; }
  static constexpr int W_O = 0, W_1 = D * PD;
  __host__ __device__ static constexpr int w_2(int d_ff) { return W_1 + d_ff * PD; }
  __host__ __device__ static constexpr int w_qkv(int d_ff) { return w_2(d_ff) + D * pf(d_ff); }
  __host__ __device__ static constexpr int weight_bytes(int d_ff) { return ALL ? w_qkv(d_ff) + 3 * D * PD : W_1; }
};

template <int D, typename C>
__global__ void __launch_bounds__(TAIL_THREADS, 1)
attn_mlp_rows_kernel(const __grid_constant__ LayerProblem prob0, const __grid_constant__ LayerProblem prob1, const __grid_constant__ Geometry g, const float sl2,
                     const float eps, const float next_eps, const int d_ff, const int problems, const int off_params) {
  constexpr int BM = C::QT, R = BM / 16, CPS = C::CW / 8 /* 16-byte pieces of a slice row */;
  using M = TailTile<D, R>;
  constexpr int KD = M::KD, WN = M::WN, NT = M::NT, SW = M::SW, YP = M::YP;
  static_assert(C::CW * C::SL == D && C::WARPS <= TAIL_WARPS, "all heads");
  const int which = (problems == 2) ? (int)(blockIdx.x & 1u) : 0;
  const int bx = (problems == 2) ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const LayerProblem& prob = which ? prob1 : prob0;
  const FusedHalfArgs& a = prob.h;

  extern __shared__ __align__(128) uint8_t smem_raw[];
  __shared__ float2 stat[BM][WN];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sH = base + C::OFF_K, sF = sH + M::OFF_F, sY = sH + M::off_y(d_ff), sRed = sH + M::off_red(d_ff);
  const float* par = reinterpret_cast<const float*>(smem_raw + off_params);
  const uint32_t sPar = smem_u32(smem_raw) + off_params, sW = sPar + M::param_bytes(d_ff);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gr = lane >> 2, t4 = lane & 3;
  const int wn = warp % WN, wm = warp / WN % M::WM, wk = warp / (WN * M::WM);
  const int n0 = wn * NT * 8 + 2 * t4;  // this thread's columns of a D-wide row: n0 + 8 j, n0 + 8 j + 1
  const bool next = a.qkv != nullptr;

  // ---- before the wait: what does not come from the kernel before this one.  That kernel belongs to the same call and has itself
  // waited for whatever wrote parameters and lengths ----
  if (tid == 0) {
    map_early(prob.tmQ);
    map_early(prob.tmKV);
  }
  init_walk<C>(base, tid - 32);
  const Tile t = find_tile<BM>(g, prob.allowed, bx, prob.seg_order);
  if (t.q_real_all > 0) {
    auto stage = [&](int at, const float* src, int len, float fill) {
      for (int i = tid; i < len; i += TAIL_THREADS) {
        const uint32_t dst = sPar + 4 * (at + i);
        if (src != nullptr) copy4(dst, src + i);
        else asm volatile("st.shared.f32 [%0], %1;" ::"r"(dst), "f"(fill) : "memory");
      }
    };
    stage(M::P_BO, a.b_o, D, 0.f);
    stage(M::P_G2, a.ln2_gamma, D, 1.f);
    stage(M::P_E2, a.ln2_beta, D, 0.f);
    stage(M::P_B2, a.b_2, D, 0.f);
    stage(M::P_B1, a.b_1, d_ff, 0.f);
    if (next) {
      stage(M::P_G1, a.ln1_gamma, D, 1.f);
      stage(M::P_E1, a.ln1_beta, D, 0.f);
      stage(M::P_BQ, a.b_qkv, 3 * D, 0.f);
    }
  }
  __syncthreads();
  grid_dep_wait();
  grid_dep_launch();
  if (t.q_real_all == 0) {  // padding only (or nothing at all)
    for (int i = tid; i < t.rows_in_tile * (D / 4); i += TAIL_THREADS)
      *reinterpret_cast<float4*>(a.y + (t.grow0 + i / (D / 4)) * a.ldy + 4 * (i % (D / 4))) = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  float2 x[SW][NT][2];  // the residual, requested before the walk
#pragma unroll
  for (int s = 0; s < SW; ++s)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int r = (wm * SW + s) * 16 + gr + 8 * half;
#pragma unroll
      for (int j = 0; j < NT; ++j)
        x[s][j][half] = (wk == 0 && r < t.q_real_all) ? *reinterpret_cast<const float2*>(a.x + (t.grow0 + r) * a.ldx + n0 + 8 * j) : make_float2(0.f, 0.f);
    }
  // Weights, 16 bytes at a time, behind the walk's first loads: they are wanted when it is over.
  auto stage_weights = [&]() {
    auto rows = [&](uint32_t dst, int pitch, const __nv_bfloat16* src, int n, int chunks /* 16-byte pieces of a row */) {
      for (int i = tid; i < n * chunks; i += TAIL_THREADS) copy16(dst + (i / chunks) * pitch + (i % chunks) * 16, src + (int64_t)i * 8);
    };
    rows(sW + M::W_O, M::PD, a.w_o, D, D / 8);
    if constexpr (M::ALL) {
      rows(sW + M::W_1, M::PD, a.w_1, d_ff, D / 8);
      rows(sW + M::w_2(d_ff), M::pf(d_ff), a.w_2, D, d_ff / 8);
      if (next) rows(sW + M::w_qkv(d_ff), M::PD, a.w_qkv, 3 * D, D / 8);
    }
  };
  // d 128, heads of 32, 16 rows: registers are short there, and warp-uniform control flow costs more of them than it saves (one sample of (50, 500,
  // 500), us: 21.3 with it, 21.1 without; two 23.8 / 23.6; with 32 rows 29.4 / 29.7, heads of 16 22.7 / 23.6).
  constexpr bool UNIFORM = !(D == 128 && C::HD == 32 && C::NSG == 1);
  if (t.T > 0) attend_tile<C, TAIL_WARPS, UNIFORM>(g, t, prob.tmQ, prob.tmKV, prob.tmKV, 0, D, 2 * D, 0, sl2, nullptr, base, stage_weights);
  else stage_weights();

  // ---- y1 = x + att W_o^T + b_o, in registers of the warps with wk = 0; the attention rows are where the walk left them ----
  auto w1_at = [&](int nt, int k) {
    if constexpr (M::ALL) return lds16(sW + M::W_1 + (nt * 8 + gr) * M::PD + 64 * k + 16 * t4);
    else return ldw(a.w_1 + (int64_t)(nt * 8 + gr) * D + 32 * k + 8 * t4);
  };
  uint4 w1[KD];  // the hidden units' first weights, on their way meanwhile
  if constexpr (!M::ALL)
#pragma unroll
    for (int k = 0; k < KD; ++k) w1[k] = w1_at(warp * 8 < d_ff ? warp : 0, k);
  asm volatile("cp.async.wait_all;" ::: "memory");  // this thread's parameters and weights; everybody's behind the barrier
  __syncthreads();
  float y1[SW][NT][4] = {};
  if (wk == 0) {
    uint4 wo[NT][KD];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int k = 0; k < KD; ++k) wo[j][k] = lds16(sW + M::W_O + ((wn * NT + j) * 8 + gr) * M::PD + 64 * k + 16 * t4);
#pragma unroll
    for (int s = 0; s < SW; ++s) {
      const int r0 = (wm * SW + s) * 16 + gr;
      auto att = [&](int r, int c) {  // a row without keys attends to nothing: zero
        return r < t.q_real ? lds16(base + (c / CPS) * C::Q_SLICE + swz<C::SWZ>(r * C::PITCH + (c % CPS) * 16)) : make_uint4(0, 0, 0, 0);
      };
      float c[NT][4] = {};
#pragma unroll
      for (int k = 0; k < KD; ++k) {
        const uint4 lo = att(r0, 4 * k + t4), hi = att(r0 + 8, 4 * k + t4);
#pragma unroll
        for (int j = 0; j < NT; ++j) step(c[j], lo, hi, wo[j][k]);
      }
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const float b0 = par[M::P_BO + n0 + 8 * j], b1 = par[M::P_BO + n0 + 8 * j + 1];
        y1[s][j][0] = c[j][0] + b0 + x[s][j][0].x; y1[s][j][1] = c[j][1] + b1 + x[s][j][0].y;
        y1[s][j][2] = c[j][2] + b0 + x[s][j][1].x; y1[s][j][3] = c[j][3] + b1 + x[s][j][1].y;
      }
      // statistics of this warp's 8 NT columns of the two rows
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        float sum = 0.f, q = 0.f;
#pragma unroll
        for (int j = 0; j < NT; ++j) sum += y1[s][j][2 * half] + y1[s][j][2 * half + 1];
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        sum += __shfl_xor_sync(0xffffffffu, sum, 2);
        const float mean = sum * (1.f / (8 * NT));
#pragma unroll
        for (int j = 0; j < NT; ++j) {
          const float d0 = y1[s][j][2 * half] - mean, d1 = y1[s][j][2 * half + 1] - mean;
          q += fmaf(d0, d0, d1 * d1);
        }
        q += __shfl_xor_sync(0xffffffffu, q, 1);
        q += __shfl_xor_sync(0xffffffffu, q, 2);
        if (t4 == 0) stat[r0 + 8 * half][wn] = make_float2(mean, q);
      }
    }
  }
  __syncthreads();
  if (wk == 0) {
#pragma unroll
    for (int s = 0; s < SW; ++s)
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int r = (wm * SW + s) * 16 + gr + 8 * half;
        float mean = 0.f, q = 0.f, dev = 0.f;
#pragma unroll
        for (int i = 0; i < WN; ++i) { mean += stat[r][i].x; q += stat[r][i].y; }
        mean *= 1.f / WN;
#pragma unroll
        for (int i = 0; i < WN; ++i) { const float d = stat[r][i].x - mean; dev = fmaf(d, d, dev); }
        const float rstd = rsqrtf(fmaf(dev, 8.f * NT, q) * (1.f / D) + eps);
#pragma unroll
        for (int j = 0; j < NT; ++j) {
          const float* p = par + n0 + 8 * j;
          const uint32_t v = pack_bf16(fmaf((y1[s][j][2 * half] - mean) * rstd, p[M::P_G2], p[M::P_E2]),
                                       fmaf((y1[s][j][2 * half + 1] - mean) * rstd, p[M::P_G2 + 1], p[M::P_E2 + 1]));
          sts4(sH + piece<D>(r, wn * NT + j) + 4 * t4, r < t.q_real_all ? v : 0u);
        }
      }
  }
  __syncthreads();

  // ---- hidden units: every warp takes its 8-column tiles for all slabs, with the rows' fragments in registers ----
  const int fpitch = d_ff * 2;
  auto fpiece = [&](int r, int c) { return sF + (uint32_t)(r * fpitch + ((c ^ (((r & 1) << 2) | ((r >> 1) & 3))) << 4)); };
  {
    uint4 lo[R][KD], hi[R][KD];
#pragma unroll
    for (int s = 0; s < R; ++s)
#pragma unroll
      for (int k = 0; k < KD; ++k) {
        lo[s][k] = lds16(sH + piece<D>(s * 16 + gr, 4 * k + t4));
        hi[s][k] = lds16(sH + piece<D>(s * 16 + gr + 8, 4 * k + t4));
      }
    const int tiles = d_ff / 8;
    if constexpr (M::ALL)
#pragma unroll
      for (int k = 0; k < KD; ++k) w1[k] = w1_at(warp * 8 < d_ff ? warp : 0, k);
#pragma unroll 2
    for (int nt = warp; nt < tiles; nt += TAIL_WARPS) {
      uint4 ahead[KD];
      const int nx = nt + TAIL_WARPS < tiles ? nt + TAIL_WARPS : nt;
#pragma unroll
      for (int k = 0; k < KD; ++k) ahead[k] = w1_at(nx, k);
      const float b0 = par[M::P_B1 + nt * 8 + 2 * t4], b1 = par[M::P_B1 + nt * 8 + 2 * t4 + 1];
#pragma unroll
      for (int s = 0; s < R; ++s) {
        float c[4] = {b0, b1, b0, b1};
#pragma unroll
        for (int k = 0; k < KD; ++k) step(c, lo[s][k], hi[s][k], w1[k]);
        sts4(fpiece(s * 16 + gr, nt) + 4 * t4, pack_bf16_relu(c[0], c[1]));
        sts4(fpiece(s * 16 + gr + 8, nt) + 4 * t4, pack_bf16_relu(c[2], c[3]));
      }
#pragma unroll
      for (int k = 0; k < KD; ++k) w1[k] = ahead[k];
    }
  }
  // ---- y = y1 + f W_2^T + b_2; two warps share the hidden units ----
  float acc[SW][NT][4] = {};
  const int steps = d_ff / 64;
  auto w2_at = [&](int j, int k) {
    const int row = (wn * NT + j) * 8 + gr;
    if constexpr (M::ALL) return lds16(sW + M::w_2(d_ff) + row * M::pf(d_ff) + (wk * steps + k) * 64 + 16 * t4);
    else return ldw(a.w_2 + (int64_t)row * d_ff + 8 * t4 + (wk * steps + k) * 32);
  };
  constexpr int AHEAD = M::ALL ? 2 : 4;   // weights requested this many steps ahead, the first ones before the barrier
  uint4 w[AHEAD][NT];
#pragma unroll
  for (int i = 0; i < AHEAD; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j) w[i][j] = w2_at(j, i < steps ? i : 0);
  __syncthreads();
#pragma unroll 4
  for (int k = 0; k < steps; ++k) {
    uint4 now[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      now[j] = w[0][j];
#pragma unroll
      for (int i = 0; i + 1 < AHEAD; ++i) w[i][j] = w[i + 1][j];
      w[AHEAD - 1][j] = w2_at(j, k + AHEAD < steps ? k + AHEAD : 0);
    }
#pragma unroll
    for (int s = 0; s < SW; ++s) {
      const int r = (wm * SW + s) * 16 + gr, c = 4 * (wk * steps + k) + t4;
      const uint4 lo = lds16(fpiece(r, c)), hi = lds16(fpiece(r + 8, c));
#pragma unroll
      for (int j = 0; j < NT; ++j) step(acc[s][j], lo, hi, now[j]);
    }
  }
  const uint32_t share = sRed + (uint32_t)((wm * WN + wn) * SW * NT * 512 + lane * 16);
  if (wk == 1)
#pragma unroll
    for (int s = 0; s < SW; ++s)
#pragma unroll
      for (int j = 0; j < NT; ++j)
        asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(share + (s * NT + j) * 512), "f"(acc[s][j][0]), "f"(acc[s][j][1]), "f"(acc[s][j][2]),
                     "f"(acc[s][j][3]) : "memory");
  __syncthreads();
  if (wk == 0) {
#pragma unroll
    for (int s = 0; s < SW; ++s)
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const uint4 v = lds16(share + (s * NT + j) * 512);
        const float other[4] = {__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w)};
        const int n = n0 + 8 * j;
        const float b[2] = {par[M::P_B2 + n], par[M::P_B2 + n + 1]};
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int r = (wm * SW + s) * 16 + gr + 8 * half;
          float2 o = make_float2(0.f, 0.f);
          if (r < t.q_real_all)
            o = make_float2(y1[s][j][2 * half] + (acc[s][j][2 * half] + other[2 * half] + b[0]),
                            y1[s][j][2 * half + 1] + (acc[s][j][2 * half + 1] + other[2 * half + 1] + b[1]));
          if (r < t.rows_in_tile) *reinterpret_cast<float2*>(a.y + (t.grow0 + r) * a.ldy + n) = o;
          if (next) asm volatile("st.shared.v2.f32 [%0], {%1,%2};" ::"r"(sY + (uint32_t)(r * YP + n) * 4u), "f"(o.x), "f"(o.y) : "memory");
        }
      }
  }
  if (!next) return;
  __syncthreads();
  auto is_real = [&](int r) { return r < t.q_real_all; };
  normalise_tile<D, BM, TAIL_THREADS>(par + M::P_G1, par + M::P_E1, next_eps, sH, tid, is_real, [&](int r, int e) {
    const uint4 v = lds16(sY + (uint32_t)(r * YP + e) * 4u);
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
  });
  __syncthreads();
  qkv_units<D, R, TAIL_WARPS>(
      [&](int row, int k) {
        if constexpr (M::ALL) return lds16(sW + M::w_qkv(d_ff) + row * M::PD + 64 * k + 16 * t4);
        else return ldw(a.w_qkv + (int64_t)row * D + 32 * k + 8 * t4);
      },
      par + M::P_BQ, a.qkv, t.grow0, sH, true, tid, is_real, is_real);
}

// Widest MLP whose weights fit beside the walk's memory.
constexpr int tail_max_ff(int d) { return d == 64 ? 256 : ROWS_MAX_FF; }

template <int D, typename C>
cudaError_t launch(const Geometry& g, const LayerTailArgs* args, int n, float scale, float eps, float next_eps, int d_ff, cudaStream_t st) {
  const int64_t rows = matrix_rows(g);
  alignas(64) LayerProblem pr[2];
  for (int i = 0; i < n; ++i) {
    if (!make_map(&pr[i].tmQ, args[i].qkv, rows, 3 * D, 3 * D, C::CW, C::QT) || !make_map(&pr[i].tmKV, args[i].qkv, rows, 3 * D, 3 * D, C::CW, KT))
      return cudaErrorInvalidValue;
    pr[i].h = args[i].h;
    pr[i].allowed = args[i].allowed;
    pr[i].seg_order = segment_order(g, args[i].allowed);
  }
  if (n == 1) pr[1] = pr[0];
  using M = TailTile<D, C::QT / 16>;
  // from the start of shared memory: slack, the walk's memory (or what the row-wise part puts in its place, if that is more), parameters
  const auto params_at = [](int ff) {
    const int tiles = C::OFF_K + M::bytes(ff) + 1024;
    return tiles > C::SMEM ? tiles : C::SMEM;
  };
  const auto smem = [&](int ff) { return params_at(ff) + M::param_bytes(ff) + M::weight_bytes(ff); };
  cudaError_t e = sm_count_and_smem_once(reinterpret_cast<const void*>(attn_mlp_rows_kernel<D, C>), smem(tail_max_ff(D)), nullptr);
  if (e != cudaSuccess) return e;
  int tiles = 0;
  for (int s = 0; s < 3; ++s) tiles += (g.len(s) + C::QT - 1) / C::QT;
  if ((int64_t)tiles * g.batch * n > 0x7fffffffLL) return cudaErrorNotSupported;
  return launch_overlapped(attn_mlp_rows_kernel<D, C>, dim3((unsigned)(tiles * g.batch * n)), dim3(TAIL_THREADS), smem(d_ff), st, pr[0], pr[1], g,
                           scale * 1.4426950408889634f, eps, next_eps, d_ff, n, params_at(d_ff));
}

}  // namespace

bool layer_tail_supported(const Geometry& g, int d_ff) {
  if (d_ff % 64 != 0 || d_ff > tail_max_ff(g.d)) return false;
  return ((g.d == 32 || g.d == 64) && (g.hd == 8 || g.hd == 16 || g.hd == 32)) || (g.d == 128 && (g.hd == 16 || g.hd == 32));
}

// Rows of a CTA's tile: 16 (d 32: 32) while that gives every SM at most one, else twice as many, which halve the reads of keys and weights.
// Layer at d 64 on B x (50, 250, 250), lengths half to full, us, 16 / 32 rows:  2200 rows 12.1/13.8, 3300 16.3/14.4, 6050 21.7/20.0.
namespace {
int64_t tail_ctas(const Geometry& g, int n, int rows) {
  int64_t t = 0;
  for (int s = 0; s < 3; ++s) t += (g.len(s) + rows - 1) / rows;
  return t * g.batch * n;
}
int small_tile(const Geometry& g) { return g.d == 32 ? 32 : 16; }
}  // namespace

// Time of the launch in key tiles, its CTAs handed to n_sm SMs one at a time, longest walk first (the order of the grid).  A CTA takes its walk
// and as long as eight key tiles for everything else.
namespace {
constexpr int REST_OF_CTA = 8;
struct Walks { int key_tiles; int64_t ctas; };
// ... of each segment and problem, longest first, with `thirds` thirds of every length real
int walks_of(const Geometry& g, const uint32_t* allowed, int n, int rows, int thirds, Walks (&w)[6]) {
  auto real = [&](int s) { return (int)(((int64_t)g.len(s) * thirds + 2) / 3); };
  int count = 0;
  for (int i = 0; i < n; ++i)
    for (int s = 0; s < 3; ++s) {
      Walks v = {0, (int64_t)((real(s) + rows - 1) / rows) * g.batch};
      for (int r = 0; r < 3; ++r)
        if ((allowed[i] >> (3 * s + r)) & 1u) v.key_tiles += (real(r) + KT - 1) / KT;
      if (v.ctas == 0) continue;
      int at = count++;
      for (; at > 0 && w[at - 1].key_tiles < v.key_tiles; --at) w[at] = w[at - 1];
      w[at] = v;
    }
  return count;
}
int makespan(const Walks* w, int count, int n_sm) {
  struct { int at, sms; } free_at[8] = {{0, n_sm}};  // SMs by when they are free: a set of walks that runs out splits one entry
  int groups = 1, end = 0;
  for (int i = 0; i < count; ++i)
    for (int64_t left = w[i].ctas; left > 0;) {
      int k = 0;
      for (int j = 1; j < groups; ++j)
        if (free_at[j].at < free_at[k].at) k = j;
      const int done = free_at[k].at + REST_OF_CTA + w[i].key_tiles;
      if (left >= free_at[k].sms) {
        left -= free_at[k].sms;
        free_at[k].at = done;
      } else {
        free_at[k].sms -= (int)left;
        free_at[groups++] = {done, (int)left};
        left = 0;
      }
      if (done > end) end = done;
    }
  return end;
}
}  // namespace

// One CTA fills an SM, and a second wave of long walks costs more than two launches less.  One wave always runs here; more (up to three
// waves, at d 32 two) by when the last CTA ends, in times of the longest CTA.
//
// No valid_len: every length is full, the walks are known.  The line lies at 5/3 (d 32: 7/4).  us of a layer in one launch behind the
// projection / in two; the last end:
//   d 64   6 x (50, 500, 500), intra 30.7/26.5 (2.0), both rings 41.7/40.5 (2.1);   32 x (50, 52, 52), intra 19.5/17.2 (2.0)
//          5 x (50, 500, 500), forward ring 21.0/25.8 (1.1);   4 x, both rings 26.8/27.9 (1.6)
//   d 32   54 x (50, 52, 52), intra 15.4/12.7 (2.0);   8 x (50, 500, 500), both rings 23.3/24.2 (1.6)
// Over 291 shapes beyond one wave at d 64 (segments of 8 - 1024 steps, one problem or two) this costs 0.4 % on average against the better
// of both, one launch up to the limits above 10 %; over 352 at d 32 1.3 % and 13 %.
// At d 128 the separate second half itself takes two waves above 32 rows per SM.  Below, a second wave here loses throughout (3850 rows of
// (50, 52, 52) 31.8/26.5, 4230 of (50, 116, 116) 32.4/27.2); above, two waves nearly hold their own up to eight key tiles (5250 rows of (50,
// 500, 500), intra 46.4/44.6, 4928 of (50, 52, 52) 33.8/34.1).
//
// With valid_len the lengths are unknown here, and padding cuts the second wave short -- where a segment has several tiles; a segment of
// one tile keeps its CTA however few rows are real.  So the same sum over walks of two thirds of the lengths, the line at 15/8 (among 110
// stacks at 1 - 3 waves any share from 5/8 to 3/4 does as well).  us of a stack on these lengths, the layers of this width in
// one launch / in two on packed rows:
//   d 64   42 x (21, 43, 34), depths 2 and 2   half to full 114/110, a quarter 78.5/76.4;   63 x (31, 21, 10), 4 and 3   187/165, 170/144
//          14 x (59, 16, 57), 4 and 3 (one wave)   84.1/110, 76.2/93.8
//   d 32   34 x (11, 60, 75), 2 and 1          52.3/47.1, 46.9/40.1;                            17 x (9, 152, 208), 3 and 2  85.3/86.5, 50.9/58.7
// At d 128 an encoder's other choice is packed rows, whose second half then mostly fits one wave: there two thirds of the lengths must fit
// one wave here (25 x (30, 26, 146), three layers in the stack's intra encoder, 124/111, 76.9/89.4).  A layer by itself takes up to
// three waves (32 x (50, 52, 52) half to full 33.3/35.0, few 23.4/26.7).
// Longest walk with valid_len: eight key tiles.  d 64, intra, 1.2 waves, us, one launch / two, by key tiles (lengths full, half to full,
// 0.05 - 0.4):
//   tiles     4          6          8          9          10         11         13         14
//   full  22.7/20.5  25.8/23.1  29.2/25.8  31.5/27.5  32.9/28.2  35.6/30.0  39.4/32.4  42.0/33.9
//   half  16.9/21.0  18.3/23.2  18.9/25.5  20.0/27.3  22.4/28.4  24.4/29.8  25.8/32.6  27.9/34.2
//   few   13.3/17.1  13.6/17.9  14.1/18.0  14.7/18.8  14.2/17.8  14.9/19.0  13.1/16.7  13.0/16.9
// What padding gains is a quarter from four tiles on, a fifth from ten; what a batch whose lengths are full after all loses grows from 11 % at four
// and 13 % at eight to 24 % at fourteen.  The line lies where one still clearly outweighs the other.
bool layer_tail_preferred(const Geometry& g, const uint32_t* allowed, int n, bool in_encoder) {
  int n_sm = 0;
  if (sm_count_and_smem_once(nullptr, 0, &n_sm) != cudaSuccess) return false;
  const int rows = 2 * small_tile(g);
  const int64_t ctas = tail_ctas(g, n, rows);
  if (ctas <= n_sm) return true;
  if (ctas > (g.d == 32 ? 2 : 3) * n_sm) return false;
  Walks w[6];
  int count = walks_of(g, allowed, n, rows, 3, w);
  const int longest = w[0].key_tiles;
  if (g.valid_len == nullptr) {
    const int end = 12 * makespan(w, count, n_sm), cta = REST_OF_CTA + longest;
    if (g.d == 128) return (int64_t)g.batch * g.L * n > 32LL * n_sm && (end <= 20 * cta || (end <= 24 * cta && longest <= 8));
    return end <= (g.d == 32 ? 21 : 20) * cta;
  }
  if (longest > 8) return false;
  count = walks_of(g, allowed, n, rows, 2, w);
  if (g.d == 128) {
    int64_t likely = 0;
    for (int i = 0; i < count; ++i) likely += w[i].ctas;
    return !in_encoder || likely <= n_sm;
  }
  return 8 * makespan(w, count, n_sm) <= 15 * (REST_OF_CTA + w[0].key_tiles);
}

cudaError_t launch_layer_tail(const Geometry& g, const LayerTailArgs* args, int n, float scale, float eps, float next_eps, int d_ff, cudaStream_t st) {
  if (n < 1 || n > 2) return cudaErrorInvalidValue;
  if (!layer_tail_supported(g, d_ff)) return cudaErrorNotSupported;
#define GSIT_LAUNCH(D_, HD_, CW_, KS_, SL_, NSG_, STAGES_) \
  return launch<D_, Cfg<HD_, CW_, 1, KS_, 1, SL_, NSG_, STAGES_>>(g, args, n, scale, eps, next_eps, d_ff, st)
  int n_sm = 0;
  cudaError_t e = sm_count_and_smem_once(nullptr, 0, &n_sm);
  if (e != cudaSuccess) return e;
  if (tail_ctas(g, n, small_tile(g)) <= n_sm) {
    if (g.d == 32 && g.hd == 8) GSIT_LAUNCH(32, 8, 32, 64, 1, 2, 6);
    if (g.d == 32 && g.hd == 16) GSIT_LAUNCH(32, 16, 32, 64, 1, 2, 6);
    if (g.d == 32) GSIT_LAUNCH(32, 32, 32, 32, 1, 2, 6);
    if (g.d == 64 && g.hd == 8) GSIT_LAUNCH(64, 8, 64, 64, 1, 1, 5);
    if (g.d == 64 && g.hd == 16) GSIT_LAUNCH(64, 16, 64, 64, 1, 1, 5);
    if (g.d == 64) GSIT_LAUNCH(64, 32, 64, 32, 1, 1, 5);
    if (g.hd == 16) GSIT_LAUNCH(128, 16, 64, 64, 2, 1, 4);
    GSIT_LAUNCH(128, 32, 64, 32, 2, 1, 4);
  }
  if (g.d == 32 && g.hd == 8) GSIT_LAUNCH(32, 8, 32, 64, 1, 4, 6);
  if (g.d == 32 && g.hd == 16) GSIT_LAUNCH(32, 16, 32, 64, 1, 4, 6);
  if (g.d == 32) GSIT_LAUNCH(32, 32, 32, 32, 1, 4, 6);
  if (g.d == 64 && g.hd == 8) GSIT_LAUNCH(64, 8, 64, 64, 1, 2, 5);
  if (g.d == 64 && g.hd == 16) GSIT_LAUNCH(64, 16, 64, 64, 1, 2, 5);
  if (g.d == 64) GSIT_LAUNCH(64, 32, 64, 32, 1, 2, 5);
  if (g.hd == 16) GSIT_LAUNCH(128, 16, 64, 64, 2, 2, 4);
  GSIT_LAUNCH(128, 32, 64, 32, 2, 2, 4);
#undef GSIT_LAUNCH
}

}  // namespace gsit
