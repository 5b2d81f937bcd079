// Host side of the bf16 IM attention: tensor maps and launch (included by attn_bf16.cu only).
#pragma once

namespace gsit {
namespace {

// n = 1 or 2 problems of the geometry g (g.allowed is ignored: every problem brings its own pattern).
template <typename C>
cudaError_t launch_one(const Geometry& g, const AttnOperands* ops, int n, int64_t row_stride, float scale, cudaStream_t st) {
  constexpr int CW = C::CW;
  const int64_t rows = matrix_rows(g);
  alignas(64) AttnProblem pr[2];
  for (int i = 0; i < n; ++i) {
    if (!make_map(&pr[i].tmQ, ops[i].q, rows, g.d, row_stride, CW, C::QT) || !make_map(&pr[i].tmK, ops[i].k, rows, g.d, row_stride, CW, KT) ||
        !make_map(&pr[i].tmV, ops[i].v, rows, g.d, row_stride, CW, KT))
      return cudaErrorInvalidValue;
    pr[i].out = ops[i].out;
    pr[i].lse = ops[i].lse;
    pr[i].allowed = ops[i].allowed;
    pr[i].seg_order = segment_order(g, ops[i].allowed);
  }
  if (n == 1) pr[1] = pr[0];
  {
    cudaError_t e = sm_count_and_smem_once(reinterpret_cast<const void*>(attn_bf16_kernel<C>), C::SMEM, nullptr);
    if (e != cudaSuccess) return e;
  }
  int tiles = 0;
  for (int s = 0; s < 3; ++s) tiles += (g.len(s) + C::QT - 1) / C::QT;
  if ((int64_t)tiles * g.batch * n > 0x7fffffffLL) return cudaErrorNotSupported;
  const dim3 grid((unsigned)(tiles * g.batch * n), (unsigned)(g.d / CW), 1u);
  const float sl2 = scale * 1.4426950408889634f;
  return launch_overlapped(attn_bf16_kernel<C>, grid, dim3(NTHREADS), C::SMEM, st, pr[0], pr[1], g, sl2, n);
}

}  // namespace

int g_attn_variant = 0;  // gsit_kernel_choice

// Which kernel, decided for each problem by itself, so that a launch for two problems gives the bits of two launches.
// The tensor-memory kernels take long to set up and to hand over a work item, the mma.sync kernel takes longer per score: what
// counts is the number of units (128 query rows x 64 keys of one head) that the padded lengths amount to; the real lengths are on
// the device only.  us on mma.sync / tensor memory at B x (50, 500, 500), intra, 8 heads of 16 (a call of its own, which clears
// the work counter first; then a whole layer at d 128, where the first half clears it):
//   units per SM             56           84          112          141          225
//   full lengths          33.6/33.2    48.6/45.6    58.7/51.4    72.3/62.8     114/94.5
//   half to full          28.7/29.8    36.2/36.9    43.7/42.9    53.2/51.0    83.8/75.2
//   a quarter real        12.3/18.3    13.3/19.1    16.3/21.1    19.4/23.1    30.4/33.3
//   layer, half to full   52.7/48.8    73.9/68.9    83.5/76.6    94.1/85.1     142/127
//   layer, a quarter      34.6/34.9    35.5/37.1    39.0/38.8    42.5/41.6    56.7/53.2
// -> 110: from there on the tensor-memory kernel is no slower at half-to-full lengths nor in a layer at any; a call of its own at a
// quarter real loses 3 - 5 us up to 225 units.  4 heads of 32: half to full 27.7/27.6 at 42, 32.5/30.9 at 56, 63.1/47.5 at 112; a
// quarter 10.5/16.4, 12.9/18.4, 24.1/25.4; layer, a quarter 34.4/35.8 at 56, 41.2/41.0 at 84 -> 55.
//   head_dim 64 is a dense contraction; there only a few short walks (at most two key tiles per row) are over sooner in the
//   mma.sync kernel (32 x (50, 50, 50), 2 heads: 4.4 against 5.1 us; 64 samples: 7.7 against 6.8; 128: 11.5 against 9.0).
//   head_dim 8: the tensor-memory kernel is slower throughout (55 against 44 us at 64 x (50, 500, 500)): a tcgen05 hand-over
//   per 64 keys of one head costs more than the 8192 exponentials it feeds.
bool attn_uses_tensor_memory(const Geometry& g, uint32_t allowed) {
  const int var = g_attn_variant;
  int n_sm = 0;
  if (sm_count_and_smem_once(nullptr, 0, &n_sm) != cudaSuccess) return false;
  if (var == GSIT_ATTN_LEGACY || (g.hd != 64 && !attn_tcs_supported(g))) return false;
  if (var == GSIT_ATTN_TMEM) return true;
  if (g.hd == 8) return false;
  int64_t units = 0;
  int longest = 0;  // most key tiles that a row walks
  for (int s = 0; s < 3; ++s) {
    int kt = 0;
    for (int r = 0; r < 3; ++r)
      if ((allowed >> (3 * s + r)) & 1u) kt += (g.len(r) + KT - 1) / KT;
    units += (int64_t)((g.len(s) + 127) / 128) * kt;
    if (kt > longest) longest = kt;
  }
  units *= (int64_t)g.batch * g.heads;
  if (g.hd == 64) return longest > 2 || units > 2LL * n_sm;
  return units > (g.hd == 16 ? 110LL : 55LL) * n_sm;
}

cudaError_t launch_attn_bf16_n(const Geometry& g, const AttnOperands* ops, int n, int64_t row_stride, float scale, int* next_item,
                               cudaStream_t st, bool counter_cleared) {
  if (n < 1 || n > 2) return cudaErrorInvalidValue;
  if (g.batch > 65535 || g.d % 16 != 0) return cudaErrorNotSupported;
  const int cw = (g.d % 64 == 0) ? 64 : (g.d % 32 == 0) ? 32 : 16;
  int n_sm = 0;
  cudaError_t e = sm_count_and_smem_once(nullptr, 0, &n_sm);
  if (e != cudaSuccess) return e;
  auto tiles = [&](int rows) {  // query tiles of one head of one problem
    int64_t t = 0;
    for (int s = 0; s < 3; ++s) t += (g.len(s) + rows - 1) / rows;
    return t * g.batch;
  };
  const bool tm = attn_uses_tensor_memory(g, ops[0].allowed);
  if (n == 2 && tm != attn_uses_tensor_memory(g, ops[1].allowed)) {
    for (int i = 0; i < n; ++i)
      if ((e = launch_attn_bf16_n(g, ops + i, 1, row_stride, scale, nullptr, st)) != cudaSuccess) return e;
    return cudaSuccess;
  }
  if (tm && g.hd == 64) {
    for (int i = 0; i < n; ++i) {  // one launch per problem
      Geometry gi = g;
      gi.allowed = ops[i].allowed;
      e = launch_attn_tc_hd64(gi, ops[i].q, ops[i].k, ops[i].v, row_stride, ops[i].out, ops[i].lse, scale, next_item, st, counter_cleared && i == 0);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  if (tm) return launch_attn_tcs(g, ops, n, row_stride, scale, next_item, st, counter_cleared);
  // mma.sync tiles.  Rows per warp: more of them reuse the key fragments, fewer give more CTAs and shorter walks; a row's result
  // does not depend on it (the keys per step are the same), so the number of problems may count here.
#define GSIT_LAUNCH(HD_, CW_, R_, KS_, MB_) return launch_one<Cfg<HD_, CW_, R_, KS_, MB_>>(g, ops, n, row_stride, scale, st)
  const int64_t slices = (int64_t)n * (g.d / cw);
  if (g.hd == 8 && cw == 64) {
    // Rows per CTA x CTAs per SM: 16 x 3 for few tiles, 32 x 2 (keys five tiles ahead), 32 x 3 beyond.  us at B x (50, 500, 500), 8 heads, for
    // CTAs of 64 rows per SM (which the lines count) 0.9, 1.4, 1.8, 2.3, 2.8, 3.7 (B = 8, 12, 16, 20, 24, 32):
    //   16 x 3, intra, every position real    19.4  24.9  30.0  35.9  43.0  54.1    cross, half to full  13.9  13.2  15.3  19.3  21.5  26.9
    //   32 x 2                                15.9  23.4  28.8  35.6  41.3  48.5                         14.2  15.0  15.2  16.8  20.8  24.6
    //   32 x 3                                21.8  22.2  28.5  33.2  38.8  45.0                         17.3  19.2  20.4  20.9  20.8  22.8
    //   64 x 2                                22.3  27.4  27.5  39.1  39.4  50.1                         20.0  24.1  25.2  25.9  25.8  26.0
    // 64 samples, cross, half to full: 32 x 3 40.5, 64 x 2 42.0; 32 x (50, 375, 500) 18.3 and 21.1.  64 x 2 is left for many short walks, where
    // the CTAs' own cost counts (the pattern's average below six key tiles): cross at 9.2, 11, 14.7 per SM 50.0/49.4, 58.3/57.4, 75.2/73.9, a quarter
    // real at 14.7 30.0/27.8; the ring pair of a stack of 40 and 64 samples (the same counts) 452/451, 668/663, of 32 397/402; but intra 109.7/110.7.
    const int64_t ctas = tiles(64) * slices;
    if (4 * ctas <= 5LL * n_sm) return launch_one<Cfg<8, 64, 1, 64, 3, 1, 1, 3>>(g, ops, n, row_stride, scale, st);
    if (2 * ctas <= 5LL * n_sm) GSIT_LAUNCH(8, 64, 2, 64, 2);
    int64_t walks = 0;  // key tiles of all query tiles of a sample
    for (int s = 0; s < 3; ++s)
      for (int r = 0; r < 3; ++r)
        if ((ops[0].allowed >> (3 * s + r)) & 1u) walks += (int64_t)((g.len(s) + 63) / 64) * ((g.len(r) + KT - 1) / KT);
    if (ctas > 8LL * n_sm && walks * g.batch < 6 * tiles(64)) GSIT_LAUNCH(8, 64, 4, 64, 2);
    return launch_one<Cfg<8, 64, 2, 64, 3, 1, 1, 3>>(g, ops, n, row_stride, scale, st);
  }
  if (g.hd == 8 && cw == 32) {
    // 32 rows per CTA up to four CTAs of 64 per SM, 64 rows beyond, three CTAs per SM both.  us at B x (50, 500, 500), 4 heads, 32 / 64 rows, for
    // 1.4, 2.8, 3.7, 5.5, 7.4, 14.7 of them per SM (B = 12, 24, 32, 48, 64, 128): intra, every position real 13.0/16.1, 23.1/21.8, 27.6/28.1,
    // 39.7/38.6, 49.7/45.0, 95.0/84.1; cross, half to full 10.7/14.6, 12.5/19.6, 15.4/19.6, 20.3/20.7, 26.3/24.8, 48.2/39.8.
    // (64 rows, two CTAs per SM, was taken from one per SM on: 15.3, 23.4, 28.6, 40.9, 48.1, 91.6 and 13.9, 14.7, 15.2, 20.9, 25.3, 45.3.)
    if (tiles(64) * slices <= 4LL * n_sm) GSIT_LAUNCH(8, 32, 1, 64, 3);
    return launch_one<Cfg<8, 32, 2, 64, 3, 1, 2, 4>>(g, ops, n, row_stride, scale, st);
  }
  if (g.hd == 8) GSIT_LAUNCH(8, 16, 1, 64, 2);
  if (g.hd == 16 && cw == 64) {
    // one sample of (50, 500, 500): 8 us with 16 rows per warp, 11 with 32; 8 samples: 18 and 17
    if (2 * tiles(128) * ((g.heads + 1) / 2) * n <= 3LL * n_sm) GSIT_LAUNCH(16, 64, 1, 64, 2);
    GSIT_LAUNCH(16, 64, 2, 64, 2);
  }
  if (g.hd == 16 && cw == 32) GSIT_LAUNCH(16, 32, 1, 64, 2);
  if (g.hd == 16) GSIT_LAUNCH(16, 16, 1, 64, 2);
  if (g.hd == 32 && cw == 64) GSIT_LAUNCH(32, 64, 1, 32, 2);
  if (g.hd == 32) GSIT_LAUNCH(32, 32, 1, 32, 2);
  if (g.hd == 64) GSIT_LAUNCH(64, 64, 1, 32, 2);
#undef GSIT_LAUNCH
  return cudaErrorNotSupported;
}

cudaError_t launch_attn_bf16(const Geometry& g, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                             int64_t row_stride, __nv_bfloat16* out, float* lse, float scale, int* next_item, cudaStream_t st,
                             bool counter_cleared) {
  const AttnOperands op = {q, k, v, out, lse, g.allowed};
  return launch_attn_bf16_n(g, &op, 1, row_stride, scale, next_item, st, counter_cleared);
}

}  // namespace gsit
