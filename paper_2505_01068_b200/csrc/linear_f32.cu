// Linear layers and the two fused layer halves for float operands, on CUDA cores (no tensor format keeps float's 24 bits):
//   linear_f32_kernel     C = act(A W^T + bias) (+ residual), any sizes
//   ln_qkv_f32_kernel     qkv = LN1(x) W_qkv^T + b_qkv                                            (d <= 128)
//   proj_mlp_f32_kernel   y1 = x + att W_o^T + b_o;  y = y1 + relu(LN2(y1) W_1^T + b_1) W_2^T + b_2   (d <= 128)
//
// All three are the same tile: 64 rows x 64 columns per 128 threads, a thread owns 8 rows x 4 columns as packed pairs of rows
// (fma.rn.f32x2), so 64 packed multiply-adds need twelve 16-byte shared-memory reads: bound by the FMA pipe.  Rows lie k-major
// in shared memory, [k][64], with the 16-byte chunks of a row swizzled by k / 4 (the transposing writes and the reads are then
// free of bank conflicts); weights lie as they come, [64][32] with the chunks swizzled by n / 4, so that cp.async can bring
// them, in slices of 32 k's through a ring of four (a ring of two: 81 us instead of 69 for the second half below).
// The fused halves keep the normalised rows, y1's row and the hidden units of 64 rows on the SM: a float layer is three
// launches, with the seven passes over memory of the separate kernels gone.  At 32 x 925 rows, d = 64: LN + QKV 68 -> 35 us,
// out-projection .. second MLP product 189 -> 69 us (FMA pipe half busy).
#include "common.cuh"
#include "ptx.cuh"

namespace gsit {
namespace {

constexpr int FT_THREADS = 128, FT_N = 64, FT_K = 32;
constexpr int SLICE = FT_K * FT_N;  // floats of one weight slice

// A tile has BM = 16 RP rows (RP row pairs per thread).  Position of element (k, row c) of a k-major tile of BM columns:
template <int BM>
__device__ __forceinline__ int at(int k, int c) { return k * BM + ((((c >> 2) ^ ((k >> 2) & (BM / 4 - 1)))) << 2) + (c & 3); }

template <int RP>
struct Acc { float2 v[RP][4]; };  // [row pair][column]
template <int RP>
__device__ __forceinline__ void clear(Acc<RP>& a) {
#pragma unroll
  for (int i = 0; i < RP; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) a.v[i][j] = make_float2(0.f, 0.f);
}
// Writes the 2 RP values of a thread's rows at row k of a k-major tile.
template <int RP>
__device__ __forceinline__ void put_rows(float* tile, int k, int ty, const float (&h)[2 * RP]) {
  constexpr int BM = 16 * RP;
  if constexpr (RP == 1) {
    *reinterpret_cast<float2*>(tile + at<BM>(k, 2 * ty)) = make_float2(h[0], h[1]);
  } else {
#pragma unroll
    for (int i = 0; i < RP / 2; ++i)
      *reinterpret_cast<float4*>(tile + at<BM>(k, 2 * RP * ty + 4 * i)) = make_float4(h[4 * i], h[4 * i + 1], h[4 * i + 2], h[4 * i + 3]);
  }
}
template <int RP>
__device__ __forceinline__ float get(const Acc<RP>& a, int row, int col) { return (row & 1) ? a.v[row >> 1][col].y : a.v[row >> 1][col].x; }

// acc += A[k0 .. k0 + 31][rows of ty] * W[columns of tx][0 .. 31]
template <int RP>
__device__ __forceinline__ void multiply(Acc<RP>& acc, const float* A, int k0, const float* W, int ty, int tx) {
  constexpr int BM = 16 * RP, M4 = BM / 4 - 1;
#pragma unroll 2
  for (int k4 = 0; k4 < FT_K / 4; ++k4) {
    const int ka = (k0 >> 2) + k4;
    const float* ap = A + ka * 4 * BM;
    const float* wp = W + tx * 128 + ((k4 ^ (tx & 7)) << 2);
    float w[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 t = *reinterpret_cast<const float4*>(wp + j * 32);
      w[j][0] = t.x; w[j][1] = t.y; w[j][2] = t.z; w[j][3] = t.w;
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float2 ar[RP];
      if constexpr (RP == 1) {
        ar[0] = *reinterpret_cast<const float2*>(ap + kk * BM + (((ty >> 1) ^ (ka & M4)) << 2) + ((ty & 1) << 1));
      } else {
#pragma unroll
        for (int i = 0; i < RP / 2; ++i) {
          const float4 t = *reinterpret_cast<const float4*>(ap + kk * BM + (((RP / 2 * ty + i) ^ (ka & M4)) << 2));
          ar[2 * i] = make_float2(t.x, t.y);
          ar[2 * i + 1] = make_float2(t.z, t.w);
        }
      }
#pragma unroll
      for (int i = 0; i < RP; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc.v[i][j] = __ffma2_rn(ar[i], make_float2(w[j][kk], w[j][kk]), acc.v[i][j]);
    }
  }
}

// One slice of a row-major matrix: rows n0 .. n0 + 63 (or BM) (below n_end), columns k0 .. k0 + 31 (below k_end); the rest is zero.
struct Slice {
  const float* p;
  int64_t ld;
  int n0, n_end, k0, k_end;
};
template <int RP>
__device__ __forceinline__ void fetch(const Slice& s, bool vec, float4 (&r)[RP], int tid) {
  const int k = s.k0 + (tid & 7) * 4;
#pragma unroll
  for (int u = 0; u < RP; ++u) {
    const int n = s.n0 + (tid >> 3) + 16 * u;
    r[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n >= s.n_end || k >= s.k_end) continue;
    const float* p = s.p + (int64_t)n * s.ld + k;
    if (vec) {
      r[u] = *reinterpret_cast<const float4*>(p);
    } else {
      r[u].x = p[0];
      if (k + 1 < s.k_end) r[u].y = p[1];
      if (k + 2 < s.k_end) r[u].z = p[2];
      if (k + 3 < s.k_end) r[u].w = p[3];
    }
  }
}
// Stores a fetched slice transposed, as rows k0 .. k0 + 31 of the k-major tile `dst`.
template <int RP>
__device__ __forceinline__ void put(float* dst, const float4 (&r)[RP], int tid, int k0 = 0) {
  constexpr int BM = 16 * RP;
  const int k = k0 + (tid & 7) * 4;
#pragma unroll
  for (int u = 0; u < RP; ++u) {
    const int n = (tid >> 3) + 16 * u;
    dst[at<BM>(k, n)] = r[u].x;
    dst[at<BM>(k + 1, n)] = r[u].y;
    dst[at<BM>(k + 2, n)] = r[u].z;
    dst[at<BM>(k + 3, n)] = r[u].w;
  }
}

// Requests a slice as a weight tile, [n][k]; the caller commits.
__device__ __forceinline__ void request(float* dst, const Slice& s, bool vec, int tid) {
  const int c = tid & 7, k = s.k0 + c * 4;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int n = (tid >> 3) + 16 * u;
    const bool row = s.n0 + n < s.n_end;
    const float* p = s.p + (row && k < s.k_end ? (int64_t)(s.n0 + n) * s.ld + k : 0);
    const uint32_t to = smem_u32(dst + n * FT_K + ((c ^ ((n >> 2) & 7)) << 2));
    if (vec) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(p), "r"(row && k < s.k_end ? 16 : 0) : "memory");
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool ok = row && k + j < s.k_end;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(to + 4 * j), "l"(ok ? p + j : s.p), "r"(ok ? 4 : 0) : "memory");
      }
    }
  }
}
__device__ __forceinline__ void commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void wait_all_but() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ float sum16(float v) {  // over the 16 threads that share rows
#pragma unroll
  for (int off = 1; off < 16; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

__device__ __forceinline__ bool real_row(const Geometry& g, int m, int M) {  // row_is_real in 32-bit arithmetic
  if (m >= M) return false;
  const int b = m / g.L, p = m - b * g.L, s = segment_of(g, p);
  return p - g.seg_off[s] < valid_rows(g, b, s);
}

// ------------------------------------------------------------------------------------------------ any linear layer
template <int RP>
__global__ void __launch_bounds__(FT_THREADS) linear_f32_kernel(const Geometry g, const LinearArgs a, const bool vec_a, const bool vec_w,
                                                                const bool vec_c) {
  constexpr int BM = 16 * RP;
  __shared__ __align__(16) float sA[2][FT_K * BM], sW[2][SLICE];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * FT_N;
  const float* W = static_cast<const float*>(a.W);
  const int slices = (a.K + FT_K - 1) / FT_K;
  float4 ra[RP];
  ptx::grid_dep_wait();  // the weights, too: this kernel may be the first of a call, right behind the one that wrote them
  ptx::grid_dep_launch();
  request(sW[0], Slice{W, a.K, n0, a.N, 0, a.K}, vec_w, tid);
  commit();
  const Slice as{static_cast<const float*>(a.A), a.lda, m0, a.M, 0, a.K};
  fetch(as, vec_a, ra, tid);
  put(sA[0], ra, tid);
  Acc<RP> acc;
  clear(acc);
  for (int i = 0; i < slices; ++i) {
    const bool more = i + 1 < slices;
    wait_all_but<0>();
    __syncthreads();  // slice i has arrived for all; nobody reads the other buffers any more
    if (more) {
      const int k = (i + 1) * FT_K;
      request(sW[(i + 1) & 1], Slice{W, a.K, n0, a.N, k, a.K}, vec_w, tid);
      commit();
      fetch(Slice{as.p, as.ld, m0, a.M, k, a.K}, vec_a, ra, tid);
    }
    multiply(acc, sA[i & 1], 0, sW[i & 1], ty, tx);
    if (more) put(sA[(i + 1) & 1], ra, tid);
  }
  float* C = static_cast<float*>(a.C);
  const int n = n0 + 4 * tx;
  float bias[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) bias[j] = (a.bias != nullptr && n + j < a.N) ? a.bias[n + j] : 0.f;
#pragma unroll
  for (int i = 0; i < 2 * RP; ++i) {
    const int m = m0 + 2 * RP * ty + i;
    if (m >= a.M || n >= a.N) continue;
    const bool real = !a.mask_rows || real_row(g, m, a.M);
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] = get(acc, i, j) + bias[j];
      if (a.relu) v[j] = fmaxf(v[j], 0.f);
      if (a.residual != nullptr && n + j < a.N && real) v[j] += a.residual[(int64_t)m * a.ldr + n + j];
      if (!real) v[j] = 0.f;
    }
    float* c = C + (int64_t)m * a.ldc + n;
    if (vec_c && n + 3 < a.N) {
      *reinterpret_cast<float4*>(c) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (n + j < a.N) c[j] = v[j];
    }
  }
}

// ------------------------------------------------------------------------------------------------ fused halves
// Walks a sequence of weight slices through a ring in shared memory: `next(i)` names slice i, total slices in all.  The barrier
// at the start of use() also separates the caller's writes to the row tiles from the reads of multiply().
constexpr int RING = 4;  // a power of two
template <typename Next>
struct WeightStream {
  float* ring;
  Next next;
  int total, i, tid;
  __device__ __forceinline__ WeightStream(float* r, Next n, int t, int id) : ring(r), next(n), total(t), i(0), tid(id) {
#pragma unroll
    for (int j = 0; j < RING - 1; ++j) {
      if (j < total) request(ring + j * SLICE, next(j), true, tid);
      commit();
    }
  }
  template <int RP>
  __device__ __forceinline__ void use(Acc<RP>& acc, const float* A, int k0, int ty, int tx) {
    wait_all_but<RING - 2>();
    __syncthreads();  // slice i has arrived for all, and nobody reads slice i - 1 any more: its place takes slice i + 3
    if (i + RING - 1 < total) request(ring + ((i + RING - 1) & (RING - 1)) * SLICE, next(i + RING - 1), true, tid);
    commit();
    multiply(acc, A, k0, ring + (i & (RING - 1)) * SLICE, ty, tx);
    ++i;
  }
};
template <typename Next>
__device__ __forceinline__ WeightStream<Next> weight_stream(float* r, Next n, int t, int id) { return WeightStream<Next>(r, n, t, id); }

// Are any of the rows m0 .. m0 + BM - 1 real?  (Row tiles that hold padding only are answered with zeros.)
template <int BM>
__device__ __forceinline__ bool tile_has_rows(const Geometry& g, int m0, int M, int tid) {
  const int m = m0 + (tid & (BM - 1));
  return __syncthreads_or(real_row(g, m, M)) != 0;
}

// KD = slices of 32 features of the model width (d <= 32 KD).
template <int KD, int RP>
__global__ void __launch_bounds__(FT_THREADS, RP == 4 && KD <= 2 ? 4 : 1)
ln_qkv_f32_kernel(const Geometry g, const float* __restrict__ x, const int64_t ldx, const float* __restrict__ gamma,
                  const float* __restrict__ beta, const float eps, const float* __restrict__ w, const float* __restrict__ bias,
                  float* __restrict__ qkv) {
  extern __shared__ __align__(16) float sm[];
  constexpr int BM = 16 * RP;
  float* sA = sm;                  // [32 KD][BM] normalised rows
  float* sW = sm + KD * FT_K * BM;     // the weight ring
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, d = g.d, N = 3 * d, M = g.batch * g.L;
  const int m0 = blockIdx.x * BM, chunks = (N + FT_N - 1) / FT_N;
  const int my = (chunks - (int)blockIdx.y + (int)gridDim.y - 1) / (int)gridDim.y;  // column chunks of this CTA
  auto next = [&](int i) { return Slice{w, d, ((int)blockIdx.y + (i / KD) * (int)gridDim.y) * FT_N, N, (i % KD) * FT_K, d}; };
  ptx::grid_dep_wait();  // the weights, too: this kernel may be the first of a call, right behind the one that wrote them
  ptx::grid_dep_launch();
  auto stream = weight_stream(sW, next, my * KD, tid);
  const bool work = tile_has_rows<BM>(g, m0, M, tid);
  if (work) {
    // LayerNorm: eight threads per row, 16 rows at a time; a thread holds float4s 8 apart
    float ga[KD][4], be[KD][4];
#pragma unroll
    for (int c = 0; c < KD; ++c) {
      const int e = ((tid & 7) + 8 * c) * 4;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        ga[c][j] = (gamma != nullptr && e < d) ? gamma[e + j] : 1.f;
        be[c][j] = (beta != nullptr && e < d) ? beta[e + j] : 0.f;
      }
    }
#pragma unroll
    for (int u = 0; u < RP; ++u) {
      const int r = (tid >> 3) + 16 * u, m = m0 + r;
      const bool real = real_row(g, m, M);
      float4 v[KD];
      float s = 0.f;
#pragma unroll
      for (int c = 0; c < KD; ++c) {
        const int e = ((tid & 7) + 8 * c) * 4;
        v[c] = (real && e < d) ? *reinterpret_cast<const float4*>(x + (int64_t)m * ldx + e) : make_float4(0.f, 0.f, 0.f, 0.f);
        s += (v[c].x + v[c].y) + (v[c].z + v[c].w);
      }
#pragma unroll
      for (int off = 1; off < 8; off <<= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      const float mean = s / d;
      float q = 0.f;
#pragma unroll
      for (int c = 0; c < KD; ++c) {
        if (((tid & 7) + 8 * c) * 4 >= d) continue;
        v[c].x -= mean; v[c].y -= mean; v[c].z -= mean; v[c].w -= mean;
        q += fmaf(v[c].x, v[c].x, v[c].y * v[c].y) + fmaf(v[c].z, v[c].z, v[c].w * v[c].w);
      }
#pragma unroll
      for (int off = 1; off < 8; off <<= 1) q += __shfl_xor_sync(0xffffffffu, q, off);
      const float rstd = rsqrtf(q / d + eps);
#pragma unroll
      for (int c = 0; c < KD; ++c) {
        const int e = ((tid & 7) + 8 * c) * 4;
        const float t[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float n = t[j] * rstd * ga[c][j] + be[c][j];
          sA[at<BM>(e + j, r)] = (real && e < d) ? n : 0.f;
        }
      }
    }
  }
  if (!work) wait_all_but<0>();
  bool real[2 * RP];
#pragma unroll
  for (int i = 0; i < 2 * RP; ++i) real[i] = work && real_row(g, m0 + 2 * RP * ty + i, M);
  for (int c = 0; c < my; ++c) {
    const int n = ((int)blockIdx.y + c * (int)gridDim.y) * FT_N + 4 * tx;
    Acc<RP> acc;
    clear(acc);
    if (work)
#pragma unroll
      for (int kd = 0; kd < KD; ++kd) stream.use(acc, sA, kd * FT_K, ty, tx);
    if (n >= N) continue;
    const float4 b = bias != nullptr ? make_float4(bias[n], bias[n + 1], bias[n + 2], bias[n + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 2 * RP; ++i) {
      const int m = m0 + 2 * RP * ty + i;
      if (m >= M) continue;
      *reinterpret_cast<float4*>(qkv + (int64_t)m * N + n) =
          real[i] ? make_float4(get(acc, i, 0) + b.x, get(acc, i, 1) + b.y, get(acc, i, 2) + b.z, get(acc, i, 3) + b.w)
               : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
}

template <int KD, int RP>
__global__ void __launch_bounds__(FT_THREADS, RP == 4 && KD <= 2 ? 4 : 1)
proj_mlp_f32_kernel(const Geometry g, const float* __restrict__ att, const float* __restrict__ x, const int64_t ldx,
                    const float* __restrict__ w_o, const float* __restrict__ b_o, const float* __restrict__ gamma,
                    const float* __restrict__ beta, const float eps, const float* __restrict__ w_1, const float* __restrict__ b_1,
                    const float* __restrict__ w_2, const float* __restrict__ b_2, const int d_ff, float* __restrict__ y,
                    const int64_t ldy) {
  constexpr int ND = (KD + 1) / 2;  // 64-column chunks of the model width
  extern __shared__ __align__(16) float sm[];
  constexpr int BM = 16 * RP;
  float* sA = sm;                          // [32 KD][BM] attention rows, then LN2 rows
  float* sF = sm + KD * FT_K * BM;         // [64][BM] hidden units
  float* sW = sF + FT_N * BM;              // the weight ring
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, d = g.d, M = g.batch * g.L, m0 = blockIdx.x * BM;
  const int nf = (d_ff + FT_N - 1) / FT_N, per_chunk = KD + 2 * ND, first = ND * KD;
  auto next = [&](int i) {
    if (i < first) return Slice{w_o, d, (i / KD) * FT_N, d, (i % KD) * FT_K, d};
    i -= first;
    const int c = i / per_chunk, j = i - c * per_chunk;
    if (j < KD) return Slice{w_1, d, c * FT_N, d_ff, j * FT_K, d};
    return Slice{w_2, d_ff, ((j - KD) >> 1) * FT_N, d, c * FT_N + ((j - KD) & 1) * FT_K, d_ff};
  };
  auto stream = weight_stream(sW, next, first + nf * per_chunk, tid);  // before the wait: the attention before it has waited
  ptx::grid_dep_wait();
  ptx::grid_dep_launch();
  bool real[2 * RP];
#pragma unroll
  for (int i = 0; i < 2 * RP; ++i) real[i] = real_row(g, m0 + 2 * RP * ty + i, M);
  if (!tile_has_rows<BM>(g, m0, M, tid)) {
#pragma unroll
    for (int nd = 0; nd < ND; ++nd)
#pragma unroll
      for (int i = 0; i < 2 * RP; ++i)
        if (m0 + 2 * RP * ty + i < M && nd * FT_N + 4 * tx < d)
          *reinterpret_cast<float4*>(y + (int64_t)(m0 + 2 * RP * ty + i) * ldy + nd * FT_N + 4 * tx) = make_float4(0.f, 0.f, 0.f, 0.f);
    wait_all_but<0>();
    return;
  }
#pragma unroll
  for (int kd = 0; kd < KD; ++kd) {
    float4 r[RP];
    fetch(Slice{att, d, m0, M, kd * FT_K, d}, true, r, tid);
    put(sA, r, tid, kd * FT_K);
  }
  Acc<RP> acc[ND];
#pragma unroll
  for (int nd = 0; nd < ND; ++nd) {
    clear(acc[nd]);
#pragma unroll
    for (int kd = 0; kd < KD; ++kd) stream.use(acc[nd], sA, kd * FT_K, ty, tx);
  }
  // y1 = x + att W_o^T + b_o, parked in y (the same thread reads it back at the end); its LayerNorm over the 16 threads of a row
  float mean[2 * RP], rstd[2 * RP];
#pragma unroll
  for (int i = 0; i < 2 * RP; ++i) mean[i] = rstd[i] = 0.f;
#pragma unroll
  for (int nd = 0; nd < ND; ++nd) {
    const int n = nd * FT_N + 4 * tx;
    const bool in = n < d;
#pragma unroll
    for (int i = 0; i < 2 * RP; ++i) {
      const int64_t m = m0 + 2 * RP * ty + i;
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (in && real[i]) {
        const float4 xr = *reinterpret_cast<const float4*>(x + m * ldx + n);
        const float xv[4] = {xr.x, xr.y, xr.z, xr.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = get(acc[nd], i, j) + (b_o != nullptr ? b_o[n + j] : 0.f) + xv[j];
        *reinterpret_cast<float4*>(y + m * ldy + n) = make_float4(v[0], v[1], v[2], v[3]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (i & 1) acc[nd].v[i >> 1][j].y = v[j];
        else acc[nd].v[i >> 1][j].x = v[j];
      mean[i] += (v[0] + v[1]) + (v[2] + v[3]);
    }
  }
#pragma unroll
  for (int i = 0; i < 2 * RP; ++i) mean[i] = sum16(mean[i]) / d;
#pragma unroll
  for (int nd = 0; nd < ND; ++nd)
    if (nd * FT_N + 4 * tx < d)
#pragma unroll
      for (int i = 0; i < 2 * RP; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { const float t = get(acc[nd], i, j) - mean[i]; rstd[i] = fmaf(t, t, rstd[i]); }
#pragma unroll
  for (int i = 0; i < 2 * RP; ++i) rstd[i] = rsqrtf(sum16(rstd[i]) / d + eps);
#pragma unroll
  for (int nd = 0; nd < ND; ++nd)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = nd * FT_N + 4 * tx + j;
      if (n >= d) continue;
      const float ga = gamma != nullptr ? gamma[n] : 1.f, be = beta != nullptr ? beta[n] : 0.f;
      float h[2 * RP];
#pragma unroll
      for (int i = 0; i < 2 * RP; ++i) h[i] = real[i] ? (get(acc[nd], i, j) - mean[i]) * rstd[i] * ga + be : 0.f;
      put_rows<RP>(sA, n, ty, h);
    }
#pragma unroll
  for (int nd = 0; nd < ND; ++nd) clear(acc[nd]);
  for (int c = 0; c < nf; ++c) {
    Acc<RP> f;
    clear(f);
#pragma unroll
    for (int kd = 0; kd < KD; ++kd) stream.use(f, sA, kd * FT_K, ty, tx);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = c * FT_N + 4 * tx + j;
      const float b = (b_1 != nullptr && n < d_ff) ? b_1[n] : 0.f;
      float h[2 * RP];
#pragma unroll
      for (int i = 0; i < 2 * RP; ++i) h[i] = fmaxf(get(f, i, j) + b, 0.f);
      put_rows<RP>(sF, 4 * tx + j, ty, h);
    }
#pragma unroll
    for (int nd = 0; nd < ND; ++nd)
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) stream.use(acc[nd], sF, kk * FT_K, ty, tx);
  }
#pragma unroll
  for (int nd = 0; nd < ND; ++nd) {
    const int n = nd * FT_N + 4 * tx;
    if (n >= d) continue;
    const float4 b = b_2 != nullptr ? make_float4(b_2[n], b_2[n + 1], b_2[n + 2], b_2[n + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 2 * RP; ++i) {
      const int64_t m = m0 + 2 * RP * ty + i;
      if (m >= M) continue;
      float4* dst = reinterpret_cast<float4*>(y + m * ldy + n);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (real[i]) {
        const float4 r = *dst;
        v = make_float4(get(acc[nd], i, 0) + b.x + r.x, get(acc[nd], i, 1) + b.y + r.y, get(acc[nd], i, 2) + b.z + r.z,
                        get(acc[nd], i, 3) + b.w + r.w);
      }
      *dst = v;
    }
  }
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Rows per tile: 64 where that gives every SM two tiles.  Below that the chain of slices in one CTA is what takes the time, and
// it is shorter with fewer rows per thread: 32 or 16 rows (60 rows at d = 32: 22 us with one 64-row tile).
int row_pairs(int64_t rows, int n_sm) { return rows >= 128LL * n_sm ? 4 : rows >= 48LL * n_sm ? 2 : 1; }

template <int KD, int RP>
cudaError_t launch_ln_qkv(const Geometry& g, int n_sm, const float* x, int64_t ldx, const float* gamma, const float* beta, float eps,
                          const float* w, const float* bias, float* qkv, cudaStream_t st) {
  constexpr int BM = 16 * RP, smem = (KD * FT_K * BM + RING * SLICE) * 4;
  cudaError_t e = sm_count_and_smem_once(reinterpret_cast<const void*>(ln_qkv_f32_kernel<KD, RP>), smem, nullptr);
  if (e != cudaSuccess) return e;
  const int rows = (int)(((int64_t)g.batch * g.L + BM - 1) / BM), chunks = (3 * g.d + FT_N - 1) / FT_N;
  // a CTA does all column chunks of its rows (one LayerNorm) unless that leaves fewer than four CTAs per SM
  int split = 1;
  while (split < chunks && (int64_t)rows * split < 4LL * n_sm) ++split;
  return launch_overlapped(ln_qkv_f32_kernel<KD, RP>, dim3(rows, split), dim3(FT_THREADS), smem, st, g, x, ldx, gamma, beta, eps, w, bias, qkv);
}

template <int KD, int RP>
cudaError_t launch_proj_mlp(const Geometry& g, int, const float* att, const float* x, int64_t ldx, const float* w_o, const float* b_o,
                            const float* gamma, const float* beta, float eps, const float* w_1, const float* b_1, const float* w_2,
                            const float* b_2, int d_ff, float* y, int64_t ldy, cudaStream_t st) {
  constexpr int BM = 16 * RP, smem = ((KD * FT_K + FT_N) * BM + RING * SLICE) * 4;
  cudaError_t e = sm_count_and_smem_once(reinterpret_cast<const void*>(proj_mlp_f32_kernel<KD, RP>), smem, nullptr);
  if (e != cudaSuccess) return e;
  const int rows = (int)(((int64_t)g.batch * g.L + BM - 1) / BM);
  return launch_overlapped(proj_mlp_f32_kernel<KD, RP>, dim3(rows), dim3(FT_THREADS), smem, st, g, att, x, ldx, w_o, b_o, gamma, beta, eps, w_1,
                           b_1, w_2, b_2, d_ff, y, ldy);
}

}  // namespace

cudaError_t launch_linear_f32(const Geometry& g, const LinearArgs& a, cudaStream_t st) {
  int n_sm = 0;
  cudaError_t e = sm_count_and_smem_once(nullptr, 0, &n_sm);
  if (e != cudaSuccess) return e;
  const int ny = (a.N + FT_N - 1) / FT_N;
  if (ny > 65535) return cudaErrorNotSupported;
  const bool va = a.lda % 4 == 0 && a.K % 4 == 0 && aligned16(a.A), vw = a.K % 4 == 0 && aligned16(a.W), vc = a.ldc % 4 == 0 && aligned16(a.C);
  const int rp = row_pairs((int64_t)a.M * ny, n_sm), bm = 16 * rp;
  const dim3 grid((a.M + bm - 1) / bm, ny);
  auto kernel = rp == 4 ? linear_f32_kernel<4> : rp == 2 ? linear_f32_kernel<2> : linear_f32_kernel<1>;
  return launch_overlapped(kernel, grid, dim3(FT_THREADS), 0, st, g, a, va, vw, vc);
}

// 16-byte rows everywhere, and the normalised rows of a tile in shared memory: d up to 128.
bool fused_layer_f32_supported(const Geometry& g, int d_ff) { return g.d <= 128 && g.d % 4 == 0 && d_ff % 4 == 0; }

#define GSIT_BY_ROWS(KD, call, ...) \
  (rp == 4 ? call<KD, 4>(g, n_sm, __VA_ARGS__) : rp == 2 ? call<KD, 2>(g, n_sm, __VA_ARGS__) : call<KD, 1>(g, n_sm, __VA_ARGS__))
#define GSIT_BY_WIDTH(call, ...)                              \
  do {                                                        \
    int n_sm = 0;                                             \
    cudaError_t e = sm_count_and_smem_once(nullptr, 0, &n_sm); \
    if (e != cudaSuccess) return e;                           \
    const int rp = row_pairs((int64_t)g.batch * g.L, n_sm);   \
    switch ((g.d + FT_K - 1) / FT_K) {                        \
      case 1: return GSIT_BY_ROWS(1, call, __VA_ARGS__);      \
      case 2: return GSIT_BY_ROWS(2, call, __VA_ARGS__);      \
      case 3: return GSIT_BY_ROWS(3, call, __VA_ARGS__);      \
      default: return GSIT_BY_ROWS(4, call, __VA_ARGS__);     \
    }                                                         \
  } while (0)

cudaError_t launch_ln_qkv_f32(const Geometry& g, const float* x, int64_t ldx, const float* gamma, const float* beta, float eps,
                              const float* w_qkv, const float* b_qkv, float* qkv, cudaStream_t st) {
  GSIT_BY_WIDTH(launch_ln_qkv, x, ldx, gamma, beta, eps, w_qkv, b_qkv, qkv, st);
}

cudaError_t launch_proj_mlp_f32(const Geometry& g, const float* att, const float* x, int64_t ldx, const float* w_o, const float* b_o,
                                const float* gamma, const float* beta, float eps, const float* w_1, const float* b_1, const float* w_2,
                                const float* b_2, int d_ff, float* y, int64_t ldy, cudaStream_t st) {
  GSIT_BY_WIDTH(launch_proj_mlp, att, x, ldx, w_o, b_o, gamma, beta, eps, w_1, b_1, w_2, b_2, d_ff, y, ldy, st);
}

}  // namespace gsit
