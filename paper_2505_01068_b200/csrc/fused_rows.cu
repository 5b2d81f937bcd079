// The two fused halves of a bf16 layer on small row tiles and mma.sync, for d_model 32, 64 and 128:
//   ln_qkv_rows     qkv = LN1(x) W_qkv^T + b_qkv
//   proj_mlp_rows   y1 = x + att W_o^T + b_o;  y = y1 + relu(LN2(y1) W_1^T + b_1) W_2^T + b_2
//
// A CTA of eight warps takes 16 R rows through the whole half.  What bounds the halves at these widths is not arithmetic but
// latency: the chain load - LayerNorm - product - product - product - store of a tile, and how many tiles are in flight to
// cover it.  So tiles are small and many, and nothing is handed from role to role.
// Row statistics of LN2 are merged over the warps with the pairwise update of Chan, Golub and LeVeque.
// A row's result does not depend on R, on the tile it falls into or on the layout.
#include "rows_tile.cuh"

namespace gsit {
namespace {

// Rows of this CTA: m0 .. m0 + 16 R - 1, those at or past `end` are not its own.
struct Rows { int m0, end; };
template <int BM>
__device__ __forceinline__ Rows rows_of(const Geometry& g) {
  const int lo = rows_begin(g);
  return Rows{lo + (int)blockIdx.x * BM, rows_end(g)};
}
__device__ __forceinline__ bool is_real(const Geometry& g, int m, int end) {
  if (m >= end) return false;
  if (g.row_start != nullptr) return true;  // packed layout: every row is
  const int b = m / g.L, p = m - b * g.L, s = segment_of(g, p);
  return p - g.off(s) < valid_rows(g, b, s);
}

struct Pair { FusedHalfArgs a[2]; };

// ------------------------------------------------------------------------------------------------ LN1 + QKV
template <int D, int R>
__global__ void __launch_bounds__(THREADS)
ln_qkv_rows_kernel(const __grid_constant__ Geometry g, const __grid_constant__ Pair pair, const float eps, int* __restrict__ zero_word) {
  constexpr int BM = 16 * R;
  __shared__ __align__(128) uint8_t sH[BM * D * 2];
  const FusedHalfArgs& a = pair.a[blockIdx.y];
  const int tid = threadIdx.x;
  const uint32_t h = smem_u32(sH);
  ptx::load_params_early(g, a, zero_word);
  ptx::grid_dep_wait();
  ptx::grid_dep_launch();
  if (zero_word != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *zero_word = 0;
  const Rows rows = rows_of<BM>(g);
  if (rows.m0 >= rows.end) return;
  auto real = [&](int r) { return is_real(g, rows.m0 + r, rows.end); };
  const bool any = normalise_tile<D, BM>(a.ln1_gamma, a.ln1_beta, eps, h, tid, real,
                                         [&](int r, int e) { return *reinterpret_cast<const float4*>(a.x + (int64_t)(rows.m0 + r) * a.ldx + e); });
  const bool work = __syncthreads_or(any) != 0;
  qkv_units<D, R>([&](int row, int k) { return ldw(a.w_qkv + (int64_t)row * D + 32 * k + 8 * (tid & 3)); }, a.b_qkv, a.qkv, rows.m0, h, work, tid, [&](int r) { return rows.m0 + r < rows.end; }, real);
}

// ------------------------------------------------------------------------------------------------ QKV alone
// The shared projection by itself, for bf16 rows: what bounds a few thousand rows of these widths is the latency of one launch, and this
// one has no tensor memory, barriers or tensor maps to set up and fits beside its neighbours on an SM.
// It does not let its successor start early: attention CTAs placed while these still hold their SMs are spread unevenly, and where there is
// about one per SM the SM with three of them decides.  Projection and attention, d 32, us, with the early start and without:
// 8 x (520, 189, 26), every block open 23.0/19.0, 8 x (100, 300, 300) intra 11.7/10.1, 32 x (50, 50, 50) 7.1/6.9.
// Over 260 pairs of calls: 3 - 5 % on average from 100 to 300 CTAs here (up to 32 %, at most 6 % the other way), nothing below and above.
struct ProjArgs { const __nv_bfloat16* x; int64_t ldx; const __nv_bfloat16* w; const float* bias; __nv_bfloat16* qkv; };

template <int D, int R>
__global__ void __launch_bounds__(THREADS)
qkv_rows_kernel(const __grid_constant__ Geometry g, const __grid_constant__ ProjArgs a) {
  constexpr int BM = 16 * R, CPR = D / 8;
  __shared__ __align__(128) uint8_t sX[BM * D * 2];
  const int tid = threadIdx.x;
  const uint32_t h = smem_u32(sX);
  ptx::load_params_early(g, a);
  ptx::grid_dep_wait();
  const Rows rows = rows_of<BM>(g);
  if (rows.m0 >= rows.end) return;
  auto real = [&](int r) { return is_real(g, rows.m0 + r, rows.end); };
  bool any = false;
#pragma unroll
  for (int i = tid; i < BM * CPR; i += THREADS) {
    const int r = i / CPR, c = i % CPR;
    const bool ok = real(r);
    any |= ok;
    const uint4 v = ok ? *reinterpret_cast<const uint4*>(a.x + (int64_t)(rows.m0 + r) * a.ldx + 8 * c) : make_uint4(0, 0, 0, 0);
    ptx::st_shared_v4(h + piece<D>(r, c), v.x, v.y, v.z, v.w);
  }
  const bool work = __syncthreads_or(any) != 0;
  qkv_units<D, R>([&](int row, int k) { return ldw(a.w + (int64_t)row * D + 32 * k + 8 * (tid & 3)); }, a.bias, a.qkv, rows.m0, h, work, tid,
                  [&](int r) { return rows.m0 + r < rows.end; }, real);
}

// ------------------------------------------------------------------------------------------------ out-projection + LN2 + MLP
template <int D, int R>
__global__ void __launch_bounds__(THREADS, R <= 2 && D <= 64 ? (R == 1 ? 3 : 2) : 1)
proj_mlp_rows_kernel(const __grid_constant__ Geometry g, const __grid_constant__ Pair pair, const float eps, const int d_ff) {
  constexpr int BM = 16 * R, KD = D / 32;
  constexpr int WN = D / 8 < ROW_WARPS ? D / 8 : ROW_WARPS, WM = ROW_WARPS / WN;   // warps along the D output columns, along the slabs
  constexpr int NT = D / 8 / WN, SW = R / WM;                          // n-tiles and slabs of a warp in the D-wide products
  static_assert(R % WM == 0, "slabs");
  extern __shared__ __align__(128) uint8_t sm[];
  __shared__ float2 stat[BM][WN];
  const FusedHalfArgs& a = pair.a[blockIdx.y];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gr = lane >> 2, t = lane & 3;
  const int wn = warp % WN, wm = warp / WN;
  const uint32_t sH = smem_u32(sm), sF = sH + BM * D * 2;
  const int fpitch = d_ff * 2;
  auto fpiece = [&](int r, int c) { return sF + (uint32_t)(r * fpitch + ((c ^ (((r & 1) << 2) | ((r >> 1) & 3))) << 4)); };
  uint4 wo[NT][KD];
#pragma unroll
  for (int j = 0; j < NT; ++j)
#pragma unroll
    for (int k = 0; k < KD; ++k) wo[j][k] = ldw(a.w_o + (int64_t)((wn * NT + j) * 8 + gr) * D + 32 * k + 8 * t);
  ptx::load_params_early(g, a);
  ptx::grid_dep_wait();
  ptx::grid_dep_launch();
  const Rows rows = rows_of<BM>(g);
  if (rows.m0 >= rows.end) return;
  bool real[SW][2];
  bool any = false;
#pragma unroll
  for (int s = 0; s < SW; ++s)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      real[s][half] = is_real(g, rows.m0 + (wm * SW + s) * 16 + gr + 8 * half, rows.end);
      any |= real[s][half];
    }
  if (g.row_start == nullptr && !__syncthreads_or(any)) {  // padding only
    for (int i = tid; i < BM * (D / 4); i += THREADS) {
      const int m = rows.m0 + i / (D / 4);
      if (m < rows.end) *reinterpret_cast<float4*>(a.y + (int64_t)m * a.ldy + 4 * (i % (D / 4))) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    return;
  }

  // ---- y1 = x + att W_o^T + b_o, in registers; the attention rows are fragments as they lie in memory ----
  float y1[SW][NT][4];
  const uint4 zero = make_uint4(0, 0, 0, 0);
#pragma unroll
  for (int s = 0; s < SW; ++s) {
    const int64_t m = rows.m0 + (wm * SW + s) * 16 + gr;
    uint4 lo[KD], hi[KD];
    float2 x[NT][2];
#pragma unroll
    for (int k = 0; k < KD; ++k) {
      lo[k] = real[s][0] ? *reinterpret_cast<const uint4*>(a.att + m * D + 32 * k + 8 * t) : zero;
      hi[k] = real[s][1] ? *reinterpret_cast<const uint4*>(a.att + (m + 8) * D + 32 * k + 8 * t) : zero;
    }
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int half = 0; half < 2; ++half)
        x[j][half] = real[s][half] ? *reinterpret_cast<const float2*>(a.x + (m + 8 * half) * a.ldx + (wn * NT + j) * 8 + 2 * t) : make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      float c[4] = {};
#pragma unroll
      for (int k = 0; k < KD; ++k) step(c, lo[k], hi[k], wo[j][k]);
      const int n = (wn * NT + j) * 8 + 2 * t;
      const float b0 = a.b_o != nullptr ? a.b_o[n] : 0.f, b1 = a.b_o != nullptr ? a.b_o[n + 1] : 0.f;
      y1[s][j][0] = c[0] + b0 + x[j][0].x; y1[s][j][1] = c[1] + b1 + x[j][0].y;
      y1[s][j][2] = c[2] + b0 + x[j][1].x; y1[s][j][3] = c[3] + b1 + x[j][1].y;
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
      if (t == 0) stat[(wm * SW + s) * 16 + gr + 8 * half][wn] = make_float2(mean, q);
    }
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < SW; ++s)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int r = (wm * SW + s) * 16 + gr + 8 * half;
      float mean = 0.f, q = 0.f;
#pragma unroll
      for (int i = 0; i < WN; ++i) { mean += stat[r][i].x; q += stat[r][i].y; }
      mean *= 1.f / WN;
      float dev = 0.f;
#pragma unroll
      for (int i = 0; i < WN; ++i) { const float d = stat[r][i].x - mean; dev = fmaf(d, d, dev); }
      const float rstd = rsqrtf(fmaf(dev, 8.f * NT, q) * (1.f / D) + eps);
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const int n = (wn * NT + j) * 8 + 2 * t;
        const float g0 = a.ln2_gamma != nullptr ? a.ln2_gamma[n] : 1.f, g1 = a.ln2_gamma != nullptr ? a.ln2_gamma[n + 1] : 1.f;
        const float e0 = a.ln2_beta != nullptr ? a.ln2_beta[n] : 0.f, e1 = a.ln2_beta != nullptr ? a.ln2_beta[n + 1] : 0.f;
        const uint32_t v = ptx::pack_bf16(fmaf((y1[s][j][2 * half] - mean) * rstd, g0, e0), fmaf((y1[s][j][2 * half + 1] - mean) * rstd, g1, e1));
        sts4(sH + piece<D>(r, wn * NT + j) + 4 * t, real[s][half] ? v : 0u);
      }
    }
  __syncthreads();

  // ---- hidden units: every warp takes its n-tiles for all slabs, with the rows' fragments in registers ----
  {
    uint4 lo[R][KD], hi[R][KD];
#pragma unroll
    for (int s = 0; s < R; ++s)
#pragma unroll
      for (int k = 0; k < KD; ++k) {
        lo[s][k] = lds16(sH + piece<D>(s * 16 + gr, 4 * k + t));
        hi[s][k] = lds16(sH + piece<D>(s * 16 + gr + 8, 4 * k + t));
      }
    const int tiles = d_ff / 8;
    uint4 w[KD];
#pragma unroll
    for (int k = 0; k < KD; ++k) w[k] = ldw(a.w_1 + (int64_t)(warp * 8 + gr) * D + 32 * k + 8 * t);
#pragma unroll 2
    for (int nt = warp; nt < tiles; nt += ROW_WARPS) {
      uint4 next[KD];
      const int ahead = nt + ROW_WARPS < tiles ? nt + ROW_WARPS : nt;
#pragma unroll
      for (int k = 0; k < KD; ++k) next[k] = ldw(a.w_1 + (int64_t)(ahead * 8 + gr) * D + 32 * k + 8 * t);
      const int n = nt * 8 + 2 * t;
      const float b0 = a.b_1 != nullptr ? a.b_1[n] : 0.f, b1 = a.b_1 != nullptr ? a.b_1[n + 1] : 0.f;
#pragma unroll
      for (int s = 0; s < R; ++s) {
        float c[4] = {b0, b1, b0, b1};
#pragma unroll
        for (int k = 0; k < KD; ++k) step(c, lo[s][k], hi[s][k], w[k]);
        sts4(fpiece(s * 16 + gr, nt) + 4 * t, ptx::pack_bf16_relu(c[0], c[1]));
        sts4(fpiece(s * 16 + gr + 8, nt) + 4 * t, ptx::pack_bf16_relu(c[2], c[3]));
      }
#pragma unroll
      for (int k = 0; k < KD; ++k) w[k] = next[k];
    }
  }
  const __nv_bfloat16* w2[NT];
#pragma unroll
  for (int j = 0; j < NT; ++j) w2[j] = a.w_2 + (int64_t)((wn * NT + j) * 8 + gr) * d_ff + 8 * t;
  __syncthreads();

  // ---- y = y1 + f W_2^T + b_2 ----
  // The two halves of the hidden units are summed by themselves, because elsewhere two warps share them.  At d 128 they are summed side by side
  // (two independent chains per output): a layer there, its projection included, 1600 rows 19.7 -> 19.1 us, 5250 rows 32.0 -> 30.6.  At d 64 and 32
  // one after the other, where the copy in between costs less than the registers (510 rows at d 64: 10.1, side by side 10.4).
  float acc[SW][NT][4] = {}, lower[SW][NT][4];
  const int steps = d_ff / 64;
  auto add = [&](float (&sum)[SW][NT][4], int k, const uint4 (&w)[NT]) {
#pragma unroll
    for (int s = 0; s < SW; ++s) {
      const int r = (wm * SW + s) * 16 + gr;
      const uint4 lo = lds16(fpiece(r, 4 * k + t)), hi = lds16(fpiece(r + 8, 4 * k + t));
#pragma unroll
      for (int j = 0; j < NT; ++j) step(sum[s][j], lo, hi, w[j]);
    }
  };
  if constexpr (D == 128) {
#pragma unroll
    for (int i = 0; i < SW * NT * 4; ++i) (&lower[0][0][0])[i] = 0.f;
#pragma unroll 4
    for (int k = 0; k < steps; ++k) {
      uint4 w[2][NT];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int j = 0; j < NT; ++j) w[u][j] = ldw(w2[j] + 32 * (k + u * steps));
      add(lower, k, w[0]);
      add(acc, k + steps, w[1]);
    }
  } else {
#pragma unroll 4
    for (int k = 0; k < 2 * steps; ++k) {
      if (k == steps) {
#pragma unroll
        for (int s = 0; s < SW; ++s)
#pragma unroll
          for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) { lower[s][j][i] = acc[s][j][i]; acc[s][j][i] = 0.f; }
      }
      uint4 w[NT];
#pragma unroll
      for (int j = 0; j < NT; ++j) w[j] = ldw(w2[j] + 32 * k);
      add(acc, k, w);
    }
  }
#pragma unroll
  for (int s = 0; s < SW; ++s)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[s][j][i] = lower[s][j][i] + acc[s][j][i];
#pragma unroll
  for (int s = 0; s < SW; ++s)
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const int n = (wn * NT + j) * 8 + 2 * t;
      const float b0 = a.b_2 != nullptr ? a.b_2[n] : 0.f, b1 = a.b_2 != nullptr ? a.b_2[n + 1] : 0.f;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int64_t m = rows.m0 + (wm * SW + s) * 16 + gr + 8 * half;
        if (m >= rows.end) continue;
        const float v0 = y1[s][j][2 * half] + (acc[s][j][2 * half] + b0), v1 = y1[s][j][2 * half + 1] + (acc[s][j][2 * half + 1] + b1);
        *reinterpret_cast<float2*>(a.y + m * a.ldy + n) = real[s][half] ? make_float2(v0, v1) : make_float2(0.f, 0.f);
      }
    }
}

template <int D, int R>
cudaError_t launch_ln_qkv(const Geometry& g, const Pair& p, int n, float eps, int* zero_word, cudaStream_t st) {
  const int64_t tiles = (matrix_rows(g) + 16 * R - 1) / (16 * R);
  return launch_overlapped(ln_qkv_rows_kernel<D, R>, dim3((unsigned)tiles, n), dim3(THREADS), 0, st, g, p, eps, zero_word);
}
template <int D, int R>
cudaError_t launch_qkv(const Geometry& g, const ProjArgs& a, cudaStream_t st) {
  return launch_overlapped(qkv_rows_kernel<D, R>, dim3((unsigned)((matrix_rows(g) + 16 * R - 1) / (16 * R))), dim3(THREADS), 0, st, g, a);
}
template <int D, int R>
cudaError_t launch_proj_mlp(const Geometry& g, const Pair& p, int n, float eps, int d_ff, cudaStream_t st) {
  constexpr int BM = 16 * R;
  const int64_t tiles = (matrix_rows(g) + BM - 1) / BM;
  cudaError_t e = sm_count_and_smem_once(reinterpret_cast<const void*>(proj_mlp_rows_kernel<D, R>), BM * (D + ROWS_MAX_FF) * 2, nullptr);
  if (e != cudaSuccess) return e;
  return launch_overlapped(proj_mlp_rows_kernel<D, R>, dim3((unsigned)tiles, n), dim3(THREADS), BM * (D + d_ff) * 2, st, g, p, eps, d_ff);
}

}  // namespace

bool fused_rows_supported(const Geometry& g, int d_ff) {
  return (g.d == 32 || g.d == 64 || g.d == 128) && d_ff % 64 == 0 && d_ff <= ROWS_MAX_FF;
}
// Where these kernels are chosen: always at width 32 (which no tcgen05 half covers); at 64 and 128 up to 43 padded rows per SM.
// One layer without open blocks, us, these kernels / tcgen05 (148 SMs; lengths between half and full):
//   rows                2100         3150         4200         5250         6300         8400
//   d 64  padded     12.2/13.9    14.1/14.1    15.0/14.3    15.2/14.3    16.3/14.6    17.2/15.1
//   d 64  packed     10.5/14.0    11.6/14.0    12.8/14.0    13.2/14.1    14.0/14.5    15.1/15.0
//   d 64  packed, pair 13.3/14.1  14.6/14.6    15.4/15.0    15.9/15.5    16.0/15.8    21.8/17.0
//   d 128 padded     20.3/23.4    23.0/23.5    23.2/23.6    25.8/24.2    33.7/24.6    33.9/24.2
//   d 128 packed     17.6/23.4    19.5/23.4    21.1/23.6    22.3/24.2    22.4/24.4    30.6/23.8
//   d 128 packed, pair 21.2/46.6  23.2/46.6    31.0/46.9    32.3/48.2    32.6/48.6    49.7/47.5
// and at a quarter of the positions real these are the faster ones up to 8400 packed rows throughout and up to 4200 (d 64) and 5250
// (d 128) padded ones.  So the two meet anywhere between 21 and 57 rows per SM, depending on what the host does not know (the lengths)
// or must not look at: a sample gets the same bits alone, in a pair, padded, packed, and in any grouping of a batch within the limit.
// The line lies at the upper end, where that holds for batches up to six samples of 1050 rows.  What it costs there, a stack of four pairs
// at d 64 and two layers at d 128 as it runs (layers in one launch where they are chosen) / on the tcgen05 halves, us:
//   samples               half to full   three quarters full   every length full   a quarter real
//   4 (28 rows per SM)      144/168           154/172              155/166            101/138
//   5 (35)                  157/169           207/178              234/186            100/138
//   6 (43)                  217/184           239/199              260/198            135/142
constexpr int ROWS_PER_SM = 43;
static int sm_count() {
  int n = 0;
  return sm_count_and_smem_once(nullptr, 0, &n) == cudaSuccess ? n : 0;
}
bool fused_rows_preferred(const Geometry& g) { return g.d == 32 || (int64_t)g.batch * g.L <= (int64_t)ROWS_PER_SM * sm_count(); }

// Where the projection alone runs here: always at width 32; at 64 up to 2000 rows, where both kernels take the same time but the
// tcgen05 GEMM's three tensor maps are encoded on the host first (6.2 us a call there, 5.4 here); at 128 never.  us here / on the kernel
// for other widths (mma.sync at d 32, tcgen05 at 64 and 128), every position real:
//   rows      500       2000      4000      8000      16000     32000
//   d 32    2.7/4.4   2.7/4.6   2.7/4.7   3.0/4.7   3.7/5.3   5.4/7.3    (32 / 64 rows a tile: 3.7/3.9 at 16000, 5.9/5.4 at 32000)
//   d 64    3.5/3.5   3.6/3.6   3.9/3.7   5.1/5.1   8.7/5.8  11.9/6.4
//   d 128   5.0/4.0   5.2/4.1   6.2/5.6   9.5/6.2  17.4/7.2  29.3/14.6
// The rows counted are those of the matrices, packed or padded: a call on part of a packed batch takes the kernel of the whole.
bool qkv_rows_preferred(const Geometry& g) { return g.d == 32 || (g.d == 64 && matrix_rows(g) <= 2000); }
cudaError_t launch_qkv_rows(const Geometry& g, const LinearArgs& l, cudaStream_t st) {
  const ProjArgs a = {static_cast<const __nv_bfloat16*>(l.A), l.lda, static_cast<const __nv_bfloat16*>(l.W), l.bias, static_cast<__nv_bfloat16*>(l.C)};
  // 32 rows a tile up to 140 rows per SM, by the figures above
  if (g.d == 32) return matrix_rows(g) > 140 * (int64_t)sm_count() ? launch_qkv<32, 4>(g, a, st) : launch_qkv<32, 2>(g, a, st);
  if (g.d == 64) return launch_qkv<64, 1>(g, a, st);
  return cudaErrorNotSupported;
}

// n problems (1 or 2) of one geometry in one launch each.  Rows per tile: 16 (d 32: 32) for the shortest chain while a launch is about
// the latency of a tile, twice as many where the weight reads of many tiles (through L1) become what counts.  For the second half that is
// one wave of small tiles at d 64 (three CTAs per SM) and 128 (one), and three tiles per SM (two at a time) at d 32.  Limits in rows per SM; a layer without open blocks, us, small tile /
// large tile, full lengths (half to full):
//   first half,  d 32   341: 30.7/31.2    600: 49.6/49.7    900: 71.4/71.3 (63.0/62.2)    1500: 119.4/118.9 (104.4/102.8)   -> 800
//   second half, d 32    78: 12.3/12.8     92: 13.1/12.9     96: 13.2/12.9 (11.7/13.9)      99: 14.0/13.0 (13.6/13.9)       -> 96
//   second half, d 64    43: 14.7/15.2     48: 14.8/15.7   48.5: 18.6/15.8 (15.4/16.6)      50: 19.7/15.9 (15.5/16.8)       -> 48
//   second half, d 128   10: 16.4/18.1     14: 17.0/19.2     16: 16.0/19.3 (16.7/20.3)    16.5: 23.1/20.6 (18.3/20.3)       -> 16
// A row's bits do not depend on it, so the number of problems may count here.
cudaError_t launch_ln_qkv_rows(const Geometry& g, const FusedHalfArgs* h, int n, float eps, int* zero_word, cudaStream_t st) {
  Pair p;
  p.a[0] = h[0];
  p.a[1] = h[n - 1];
  const int64_t rows = (int64_t)g.batch * g.L * n, sms = sm_count();
  if (g.d == 32) return rows > 800 * sms ? launch_ln_qkv<32, 4>(g, p, n, eps, zero_word, st) : launch_ln_qkv<32, 2>(g, p, n, eps, zero_word, st);
  if (g.d == 64) return launch_ln_qkv<64, 1>(g, p, n, eps, zero_word, st);
  return launch_ln_qkv<128, 1>(g, p, n, eps, zero_word, st);
}
cudaError_t launch_proj_mlp_rows(const Geometry& g, const FusedHalfArgs* h, int n, float eps, int d_ff, cudaStream_t st) {
  Pair p;
  p.a[0] = h[0];
  p.a[1] = h[n - 1];
  const int64_t rows = (int64_t)g.batch * g.L * n, sms = sm_count();
  if (g.d == 32) return rows > 96 * sms ? launch_proj_mlp<32, 4>(g, p, n, eps, d_ff, st) : launch_proj_mlp<32, 2>(g, p, n, eps, d_ff, st);
  if (g.d == 64) return rows > 48 * sms ? launch_proj_mlp<64, 2>(g, p, n, eps, d_ff, st) : launch_proj_mlp<64, 1>(g, p, n, eps, d_ff, st);
  return rows > 16 * sms ? launch_proj_mlp<128, 2>(g, p, n, eps, d_ff, st) : launch_proj_mlp<128, 1>(g, p, n, eps, d_ff, st);
}

}  // namespace gsit
