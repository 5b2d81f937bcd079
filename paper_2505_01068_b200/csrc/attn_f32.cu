// fp32 IM attention on CUDA cores: flash-style, key tiles shared by all rows of a CTA, scores never leave registers.
//
// Decomposition (paper, Section "Inner Decomposition for Efficiency"): a CTA takes a tile of query rows of one segment of one
// sample and one head, and walks only the real keys of the segments the mask opens for that block row.
//
// What bounds it: 2 hd multiply-adds per (query, key) pair on the FMA pipe, 128 lanes per clock and SM -- there is no tensor
// format with float's 24 bits.  So the layout serves that pipe: a thread owns R = 2 query rows and DT features of them (the
// whole head up to 16, a slice beyond, T = hd / 16 neighbouring threads sharing a row), holds q and the accumulator of its
// slice in registers as packed pairs (fma.rn.f32x2: half the issue slots), and reads every K and V chunk from shared memory
// as a 16-byte broadcast that serves both rows.  Keys are taken eight at a time: eight independent dot products, one
// maximum and at most one rescale per group.  Scores are kept in base 2 (q is scaled by scale * log2 e once).
// K and V tiles arrive through cp.async, double-buffered; keys past the valid length are filled with zeros and masked.
// Where a launch would leave SMs idle, the warps of a CTA split the keys (2 or 4 ways) and merge at the end.
// At 32 x (50, 375, 500) x 8 heads of 8, intra: 2324 us (a warp per row, lanes over features) -> 81 us, the FMA pipe 55 % busy.
#include <float.h>

#include "common.cuh"
#include "ptx.cuh"

namespace gsit {
namespace {

constexpr int F32_WARPS = 4, F32_G = 8;  // warps per CTA, keys per step

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void* src, bool pred) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(pred ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4_zfill(uint32_t dst, const void* src, bool pred) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(pred ? 4 : 0) : "memory");
}

// DT features per thread, T threads per row, F32_R rows per thread: head widths up to DT * T (narrower ones are padded with zeros).
// key_splits (1, 2 or 4): how many ways the warps of the CTA share out the keys.  VEC: rows are 16-byte aligned and hd % 4 == 0.
template <int DT, int T, int F32_R, bool VEC, int KT /* keys per tile */>
__global__ void __launch_bounds__(F32_WARPS * 32)
attn_f32_kernel(const Geometry g, const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v,
                const int64_t row_stride, float* __restrict__ out, float* __restrict__ lse, const float sl2 /* scale * log2(e) */,
                const int key_splits) {
  constexpr int HP = DT * T;                                                // padded head width
  constexpr int TILE = KT * HP, C4 = HP / 4, NT = F32_WARPS * 32;
  extern __shared__ __align__(16) float sm[];                              // [2 buffers][K, V][KT][HP]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row_warps = F32_WARPS / key_splits, split = warp / row_warps;
  const int sub = lane % T, rpw = 32 / T * F32_R;                           // slice of the head, rows per warp
  const int rows_cta = row_warps * rpw;
  const int h = blockIdx.y, b = blockIdx.z, hd = g.hd;
  ptx::grid_dep_wait();
  ptx::grid_dep_launch();

  int tile = blockIdx.x, s = 0;                                             // query tile -> segment and first row in it
  for (; s < 2; ++s) {
    const int n = (g.seg_len[s] + rows_cta - 1) / rows_cta;
    if (tile < n) break;
    tile -= n;
  }
  const int q0 = tile * rows_cta, nq = valid_rows(g, b, s);
  const int row0 = q0 + (warp % row_warps) * rpw + lane / T;                // this thread's rows: row0, row0 + 32 / T
  const bool busy = q0 + (warp % row_warps) * rpw < nq;
  const int64_t base = (int64_t)b * g.L;
  int nk[3] = {0, 0, 0};
  int any = 0;
#pragma unroll
  for (int r = 0; r < 3; ++r)
    if (q0 < nq && ((g.allowed >> (3 * s + r)) & 1u)) any += (nk[r] = valid_rows(g, b, r));

  float2 qv[F32_R][DT / 2], o[F32_R][DT / 2];
  float m[F32_R], l[F32_R];
#pragma unroll
  for (int r = 0; r < F32_R; ++r) {
    const int row = row0 + r * (32 / T);
    const float* src = q + (base + g.seg_off[s] + row) * row_stride + (int64_t)h * hd;
#pragma unroll
    for (int i = 0; i < DT / 2; ++i) {
      const int e = sub * DT + 2 * i;
      float2 t = make_float2(0.f, 0.f);
      if (row < nq) {
        if (VEC) { if (e < hd) t = *reinterpret_cast<const float2*>(src + e); }
        else { if (e < hd) t.x = src[e]; if (e + 1 < hd) t.y = src[e + 1]; }
      }
      qv[r][i] = make_float2(t.x * sl2, t.y * sl2);
      o[r][i] = make_float2(0.f, 0.f);
    }
    m[r] = -FLT_MAX;  // not -inf: keys whose scores are all -inf (a -inf in k or q) then weigh exp2(-inf) = 0 and not NaN
    l[r] = 0.f;
  }

  if (any > 0) {
    int tiles = 0;
#pragma unroll
    for (int r = 0; r < 3; ++r) tiles += (nk[r] + KT - 1) / KT;
    // the walk over key tiles, in order of the open segments; `load` runs one tile ahead of `use`
    auto locate = [&](int j, int* seg, int* first) {
      int r = 0;
      for (; r < 2; ++r) {
        const int n = (nk[r] + KT - 1) / KT;
        if (j < n) break;
        j -= n;
      }
      *seg = r;
      *first = j * KT;
    };
    auto load = [&](int j) {
      int r, k0;
      locate(j, &r, &k0);
      const uint32_t dst = smem_u32(sm) + (uint32_t)((j & 1) * 2 * TILE * 4);
      const int n = nk[r] - k0;
      // Of a wide tile only the rounds of the CTA that hold a key are fetched or filled: nothing is read behind the last key's group.
      constexpr bool WIDE = KT > 64;
      static_assert(!WIDE || NT * 4 / HP % F32_G == 0, "a round of the CTA must hold whole groups");
      const int64_t off = (base + g.seg_off[r] + k0) * row_stride + (int64_t)h * hd;
      if (VEC) {
        for (int i = tid; i < KT * C4; i += NT) {
          if (WIDE && (i - tid) / C4 >= n) break;
          const int row = i / C4, c = i % C4;
          const bool ok = row < n && 4 * c < hd;
          const int64_t at = ok ? off + (int64_t)row * row_stride + 4 * c : 0;
          cp_async16_zfill(dst + i * 16, k + at, ok);
          cp_async16_zfill(dst + (TILE + 4 * i) * 4, v + at, ok);
        }
      } else {
        const int most = WIDE ? min(KT, (n + F32_G - 1) / F32_G * F32_G) * HP : TILE;
        for (int i = tid; i < most; i += NT) {
          const int row = i / HP, c = i % HP;
          const bool ok = row < n && c < hd;
          const int64_t at = ok ? off + (int64_t)row * row_stride + c : 0;
          cp_async4_zfill(dst + i * 4, k + at, ok);
          cp_async4_zfill(dst + (TILE + i) * 4, v + at, ok);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    load(0);
    for (int j = 0; j < tiles; ++j) {
      if (j + 1 < tiles) {
        load(j + 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncthreads();
      int r_, k0;
      locate(j, &r_, &k0);
      const int n = min(KT, nk[r_] - k0);
      const float* ks = sm + (j & 1) * 2 * TILE + sub * DT;
      const float* vs = ks + TILE;
      // a warp without a real row only helps to load
      for (int g0 = split * F32_G + (busy ? 0 : n); g0 < n; g0 += key_splits * F32_G) {
        float sc[F32_R][F32_G];
#pragma unroll
        for (int kk = 0; kk < F32_G; ++kk) {
          float2 acc[F32_R];
#pragma unroll
          for (int r = 0; r < F32_R; ++r) acc[r] = make_float2(0.f, 0.f);
#pragma unroll
          for (int i = 0; i < DT / 4; ++i) {
            const float4 kv = *reinterpret_cast<const float4*>(ks + (g0 + kk) * HP + 4 * i);
#pragma unroll
            for (int r = 0; r < F32_R; ++r) {
              acc[r] = __ffma2_rn(qv[r][2 * i], make_float2(kv.x, kv.y), acc[r]);
              acc[r] = __ffma2_rn(qv[r][2 * i + 1], make_float2(kv.z, kv.w), acc[r]);
            }
          }
#pragma unroll
          for (int r = 0; r < F32_R; ++r) sc[r][kk] = acc[r].x + acc[r].y;
        }
        if constexpr (T > 1) {
#pragma unroll
          for (int off = 1; off < T; off <<= 1)
#pragma unroll
            for (int r = 0; r < F32_R; ++r)
#pragma unroll
              for (int kk = 0; kk < F32_G; ++kk) sc[r][kk] += __shfl_xor_sync(0xffffffffu, sc[r][kk], off);
        }
        if (g0 + F32_G > n) {
#pragma unroll
          for (int r = 0; r < F32_R; ++r)
#pragma unroll
            for (int kk = 0; kk < F32_G; ++kk)
              if (g0 + kk >= n) sc[r][kk] = -INFINITY;
        }
#pragma unroll
        for (int r = 0; r < F32_R; ++r) {
          float mx = sc[r][0];
#pragma unroll
          for (int kk = 1; kk < F32_G; ++kk) mx = fmaxf(mx, sc[r][kk]);
          if (mx > m[r]) {
            const float corr = ptx::ex2(m[r] - mx);
            m[r] = mx;
            l[r] *= corr;
#pragma unroll
            for (int i = 0; i < DT / 2; ++i) o[r][i] = __fmul2_rn(o[r][i], make_float2(corr, corr));
          }
          float sum = 0.f;
#pragma unroll
          for (int kk = 0; kk < F32_G; ++kk) {
            sc[r][kk] = ptx::ex2(sc[r][kk] - m[r]);
            sum += sc[r][kk];
          }
          l[r] += sum;
        }
#pragma unroll
        for (int kk = 0; kk < F32_G; ++kk)
#pragma unroll
          for (int i = 0; i < DT / 4; ++i) {
            const float4 vv = *reinterpret_cast<const float4*>(vs + (g0 + kk) * HP + 4 * i);
#pragma unroll
            for (int r = 0; r < F32_R; ++r) {
              const float2 p = make_float2(sc[r][kk], sc[r][kk]);
              o[r][2 * i] = __ffma2_rn(p, make_float2(vv.x, vv.y), o[r][2 * i]);
              o[r][2 * i + 1] = __ffma2_rn(p, make_float2(vv.z, vv.w), o[r][2 * i + 1]);
            }
          }
      }
      __syncthreads();
    }
    if (key_splits > 1) {  // merge the splits: warps of split > 0 hand over their state through shared memory
      constexpr int ST = DT + 2;                      // floats per thread and row
      float* st = sm;                                 // [split - 1][row warp][row of the thread][ST][lane]: at most 3 * 2 * 18 * 32 floats
      for (int r = 0; r < F32_R; ++r) {
        float* mine = st + ((((split - 1) * row_warps + warp % row_warps) * F32_R + r) * ST) * 32 + lane;
        if (split > 0) {
          mine[0] = m[r];
          mine[32] = l[r];
#pragma unroll
          for (int i = 0; i < DT / 2; ++i) { mine[(2 + 2 * i) * 32] = o[r][i].x; mine[(3 + 2 * i) * 32] = o[r][i].y; }
        }
      }
      __syncthreads();
      if (split == 0) {
        for (int sp = 1; sp < key_splits; ++sp)
#pragma unroll
          for (int r = 0; r < F32_R; ++r) {
            const float* o_ = st + ((((sp - 1) * row_warps + warp) * F32_R + r) * ST) * 32 + lane;
            const float m2 = o_[0], mm = fmaxf(m[r], m2);
            const float c1 = (m[r] == mm) ? 1.f : ptx::ex2(m[r] - mm), c2 = (m2 == mm) ? 1.f : ptx::ex2(m2 - mm);
            m[r] = mm;
            l[r] = l[r] * c1 + o_[32] * c2;
#pragma unroll
            for (int i = 0; i < DT / 2; ++i) {
              o[r][i].x = o[r][i].x * c1 + o_[(2 + 2 * i) * 32] * c2;
              o[r][i].y = o[r][i].y * c1 + o_[(3 + 2 * i) * 32] * c2;
            }
          }
      }
    }
  }
  if (split > 0) return;
#pragma unroll
  for (int r = 0; r < F32_R; ++r) {
    const int row = row0 + r * (32 / T);
    if (row >= g.seg_len[s]) continue;
    const bool real = row < nq && any > 0;
    const float inv = real ? 1.f / l[r] : 0.f;
    const int64_t p = g.seg_off[s] + row;
    float* dst = out + (base + p) * g.d + (int64_t)h * hd;
#pragma unroll
    for (int i = 0; i < DT / 4; ++i) {
      const int e = sub * DT + 4 * i;
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
      if (real) t = make_float4(o[r][2 * i].x * inv, o[r][2 * i].y * inv, o[r][2 * i + 1].x * inv, o[r][2 * i + 1].y * inv);
      if (VEC) {
        if (e < hd) *reinterpret_cast<float4*>(dst + e) = t;
      } else {
        if (e < hd) dst[e] = t.x;
        if (e + 1 < hd) dst[e + 1] = t.y;
        if (e + 2 < hd) dst[e + 2] = t.z;
        if (e + 3 < hd) dst[e + 3] = t.w;
      }
    }
    if (lse != nullptr && sub == 0)
      lse[((int64_t)b * g.heads + h) * g.L + p] = real ? (m[r] + log2f(l[r])) * 0.693147180559945309f : -INFINITY;
  }
}

template <int DT, int T, int F32_R, int KT>
cudaError_t launch_tiles(const Geometry& g, const float* q, const float* k, const float* v, int64_t row_stride, float* out, float* lse,
                   float scale, cudaStream_t st) {
  constexpr int HP = DT * T;
  // tiles, double-buffered; the merge of key splits needs at most 3 * F32_R * (DT + 2) * 32 floats
  constexpr int FLOATS = 4 * KT * HP, MERGE = 3 * F32_R * (DT + 2) * 32;
  constexpr int smem = (FLOATS > MERGE ? FLOATS : MERGE) * 4;
  const bool vec = g.hd % 4 == 0 && row_stride % 4 == 0 && g.d % 4 == 0 &&
                   ((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(k) | reinterpret_cast<uintptr_t>(v) |
                     reinterpret_cast<uintptr_t>(out)) & 15u) == 0;
  auto kernel = vec ? attn_f32_kernel<DT, T, F32_R, true, KT> : attn_f32_kernel<DT, T, F32_R, false, KT>;
  int n_sm = 0;
  cudaError_t e = sm_count_and_smem_once(reinterpret_cast<const void*>(kernel), smem, &n_sm);
  if (e != cudaSuccess) return e;
  auto tiles = [&](int splits) {
    const int rows = F32_WARPS / splits * (32 / T) * F32_R;
    int64_t n = 0;
    for (int s = 0; s < 3; ++s) n += (g.seg_len[s] + rows - 1) / rows;
    return n;
  };
  // At most 128 rows per CTA, so that a segment's last tile wastes little (256: 92 us instead of 81 at the size above; 64: 88),
  // and the keys split further over the warps of a CTA while there are fewer than four CTAs (16 warps) per SM.
  int splits = T == 1 ? 2 : 1;
  while (splits < 4 && tiles(splits) * g.heads * g.batch < 4LL * n_sm) splits *= 2;
  if (tiles(splits) > 0x7fffffffLL) return cudaErrorNotSupported;
  // Heads and samples lie along y and z, which hold 65535 blocks each; more of them take further launches.  (All three folded into
  // x costs the kernel ten registers and with them a CTA per SM: 173 -> 179 us for a layer at the size above.)
  constexpr int MOST = 65535;
  for (int b0 = 0; b0 < g.batch; b0 += MOST)
    for (int h0 = 0; h0 < g.heads; h0 += MOST) {
      Geometry gs = g;
      gs.batch = g.batch - b0 < MOST ? g.batch - b0 : MOST;
      if (g.valid_len != nullptr) gs.valid_len = g.valid_len + 3 * (int64_t)b0;
      const int heads = g.heads - h0 < MOST ? g.heads - h0 : MOST;
      const int64_t in = (int64_t)b0 * g.L * row_stride + (int64_t)h0 * g.hd, to = (int64_t)b0 * g.L * g.d + (int64_t)h0 * g.hd;
      float* lse_s = lse != nullptr ? lse + ((int64_t)b0 * g.heads + h0) * g.L : nullptr;
      e = launch_overlapped(kernel, dim3((unsigned)tiles(splits), heads, gs.batch), dim3(F32_WARPS * 32), smem, st, gs, q + in, k + in, v + in,
                            row_stride, out + to, lse_s, scale * 1.4426950408889634f, splits);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

// Wide key tiles: 256 keys at head_dim 8, 128 at 16 (8 KB each of K and V, twice as many buffers: a quarter and half of the barriers of 64 keys).
// They are taken where a segment is longer than half of one; of a tile that is not full only the rounds that hold a key are filled (every place
// filled: 4 x (17, 126, 125), 16 heads of 8, a quarter real, 5.5 -> 5.95 us).  Against 64 keys throughout, us: 32 x (50, 375, 500), 8 heads of 8,
// intra 78.0 -> 75.5; 4 x (50, 300, 200) 14.0 -> 13.6; geometric means over batches of 1 - 32, all patterns and lengths, 8 and 16 heads of 8:
// (50, 500, 500) 0.96, (70, 300, 200) 0.97, (10, 256, 129) 0.97 (worst single call 1.04: 80 real keys in one tile, whose load nothing hides);
// (17, 126, 125) and (30, 120, 90) 0.995, worst 1.04: left to 64 keys.  Heads of 16: (30, 120, 90) 0.98, (17, 126, 125) 0.99, longer 0.985, worst 1.02.
template <int DT, int T, int F32_R>
cudaError_t launch(const Geometry& g, const float* q, const float* k, const float* v, int64_t row_stride, float* out, float* lse,
                   float scale, cudaStream_t st) {
  constexpr int HP = DT * T, KT = (HP <= 64) ? 64 : (HP <= 128) ? 32 : 16, WIDE = (HP <= 32) ? 2048 / HP : KT;
  if constexpr (WIDE > KT)
    if (2 * g.seg_len[0] > WIDE || 2 * g.seg_len[1] > WIDE || 2 * g.seg_len[2] > WIDE) return launch_tiles<DT, T, F32_R, WIDE>(g, q, k, v, row_stride, out, lse, scale, st);
  return launch_tiles<DT, T, F32_R, KT>(g, q, k, v, row_stride, out, lse, scale, st);
}

}  // namespace

cudaError_t launch_attn_f32(const Geometry& g, const float* q, const float* k, const float* v, int64_t row_stride,
                            float* out, float* lse, float scale, cudaStream_t st) {
  if (g.hd <= 8) return launch<8, 1, 2>(g, q, k, v, row_stride, out, lse, scale, st);
  if (g.hd <= 16) return launch<16, 1, 2>(g, q, k, v, row_stride, out, lse, scale, st);
  if (g.hd <= 32) return launch<16, 2, 2>(g, q, k, v, row_stride, out, lse, scale, st);
  if (g.hd <= 64) return launch<16, 4, 2>(g, q, k, v, row_stride, out, lse, scale, st);
  if (g.hd <= 128) return launch<16, 8, 2>(g, q, k, v, row_stride, out, lse, scale, st);
  return launch<16, 16, 2>(g, q, k, v, row_stride, out, lse, scale, st);
}

}  // namespace gsit
