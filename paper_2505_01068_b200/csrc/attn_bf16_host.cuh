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
//   full lengths          30.7/28.2    44.8/41.1    54.0/45.8    66.6/56.8    103/85.5
//   half to full          25.2/24.5    32.9/31.3    40.1/37.5    48.9/44.5    74.4/64.5
//   a quarter real         9.6/12.6    14.6/16.2    15.6/16.7    19.1/19.7    28.8/26.9
//   layer, half to full   43.7/41.9    64.5/61.7    72.1/68.1    93.6/87.8     134/123
//   layer, a quarter      28.5/29.5    46.7/47.3    48.1/48.0    64.5/63.1    88.6/84.3
// -> 110: from there on the tensor-memory kernel is no slower at half-to-full lengths nor in a layer at any; a call of its own at a
// quarter real loses 1 us up to 141 units.  4 heads of 32: half to full 25.2/23.7 at 42, 30.6/26.6 at 56, 56.7/41.1 at 112; a
// quarter 11.9/14.1, 12.5/14.7, 23.2/21.6; layer, a quarter 44.6/45.8 at 56, 62.9/62.1 at 84 -> 55.
//   head_dim 64 is a dense contraction; there only a few short walks (at most two key tiles per row) are over sooner in the
//   mma.sync kernel (32 x (50, 50, 50), 2 heads: 4.3 against 4.8 us; 64 samples: 6.7 against 6.3; 128: 10.9 against 8.5).
//   head_dim 8: the tensor-memory kernel is slower throughout (44.5 against 39.5 us at 64 x (50, 500, 500)): a tcgen05 hand-over
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
  const bool full = g.valid_len == nullptr;  // every length is known here
  // CTAs of 32 rows, of all problems, that walk (three quarters of) the most key tiles.  Where lengths are given, those of segments of one tile
  // only: they keep their CTAs however few rows are real.
  auto long_walks = [&]() {
    int64_t ctas = 0;
    for (int i = 0; i < n; ++i) {
      int kt[3] = {0, 0, 0}, most = 0;
      for (int s = 0; s < 3; ++s) {
        for (int r = 0; r < 3; ++r)
          if ((ops[i].allowed >> (3 * s + r)) & 1u) kt[s] += (g.len(r) + KT - 1) / KT;
        if (kt[s] > most) most = kt[s];
      }
      for (int s = 0; s < 3; ++s)
        if (4 * kt[s] >= 3 * most && (full || g.len(s) <= 64)) ctas += (g.len(s) + 31) / 32;
    }
    return ctas * g.batch * (g.d / cw);
  };
  if (g.hd == 8 && cw == 64) {
    // Rows per CTA x CTAs per SM: 16 x 3 for few tiles, 32 x 2 (keys five tiles ahead), 32 x 3 beyond.  Times over those of the version without
    // uniform control flow (16 rows up to 1.5, 32 up to 3, 64 beyond, three key stages), geometric mean and worst over six sets of segments between
    // (60, 60, 60) and (20, 1000, 300), intra and cross, lengths full, half to full and a quarter, by CTAs of 64 rows per SM, which the lines count:
    //   per SM      1.0 - 1.25    1.25 - 1.5    1.5 - 2.5     2.5 - 3       3 - 4         4 - 5.6
    //   16 x 3       0.96 0.99     0.95 0.98     0.96 1.17     0.97 1.11     0.95 1.25     1.03 1.24
    //   32 x 2       0.99 1.22     0.99 1.19     0.94 1.00     0.93 1.01     0.88 1.15     0.93 1.11
    //   32 x 3       1.13 1.45     1.17 1.76     0.98 1.27     0.94 1.14     0.86 1.06     0.88 1.03
    //   64 x 2       1.33 1.70     1.37 1.84     1.14 1.58     1.04 1.41     0.96 0.99     0.96 0.99
    // So 16 x 3 up to 1.5, 32 x 2 up to 3; but where every length is full 32 x 3 wins from 2.5 on (32 x 2 0.94, 32 x 3 0.88), and loses to 64 x 2
    // where its long walks make one wave and up to a quarter (28 x (50, 500, 500), cross: 28.5 and 27.1).  Given lengths may do the same
    // unseen: 22 x (20, 1000, 300), intra, half to full is the 1.06 above.  Four key stages at 32 x 3 and 16 x 3, which fit too, change either
    // by less than 1 %.
    // 64 x 2 also for many short walks, where the CTAs' own cost counts (the pattern's average below six key tiles): cross at 9.2, 11, 14.7 per
    // SM 32 x 3 50.0, 64 x 2 49.4, 58.3/57.4, 75.2/73.9, a quarter real at 14.7 30.0/27.8; the ring pair of a stack of 40 and 64 samples (the
    // same counts) 452/451, 668/663, of 32 397/402; but intra 109.7/110.7.
    const int64_t ctas = tiles(64) * slices;
    if (2 * ctas <= 3LL * n_sm) return launch_one<Cfg<8, 64, 1, 64, 3, 1, 1, 3>>(g, ops, n, row_stride, scale, st);
    if (2 * ctas <= (full ? 5LL : 6LL) * n_sm) GSIT_LAUNCH(8, 64, 2, 64, 2);
    int64_t walks = 0;  // key tiles of all query tiles of a sample
    for (int s = 0; s < 3; ++s)
      for (int r = 0; r < 3; ++r)
        if ((ops[0].allowed >> (3 * s + r)) & 1u) walks += (int64_t)((g.len(s) + 63) / 64) * ((g.len(r) + KT - 1) / KT);
    const int64_t waves = full ? long_walks() : 0, wave = 3LL * n_sm;
    if ((ctas > 8LL * n_sm && walks * g.batch < 6 * tiles(64)) || (ctas > 3LL * n_sm && waves > wave && 4 * waves <= 5 * wave)) GSIT_LAUNCH(8, 64, 4, 64, 2);
    return launch_one<Cfg<8, 64, 2, 64, 3, 1, 1, 3>>(g, ops, n, row_stride, scale, st);
  }
  if (g.hd == 8 && cw == 32) {
    // 32 x 3, then 64 x 2, then 64 x 3, five key stages all.  As above, for 4 heads (32 rows up to 1, 64 x 2 beyond, three key stages, is 1):
    //   per SM      0.9 - 1.5     1.5 - 3       3 - 4.5       4.5 - 5.6     5.6 - 7.5     7.5 - 9.2
    //   32 x 3       0.84 0.99     0.87 1.20     0.89 1.15     0.93 1.01     0.94 1.10     0.97 1.08
    //   64 x 2       0.94 1.00     0.94 1.00     0.93 0.98     0.92 0.96     0.93 0.96     0.93 0.96
    //   64 x 3       0.93 1.04     1.05 1.27     0.98 1.26     0.94 1.12     0.90 1.05     0.87 0.99
    // (64 x 3 with four stages is 2 % behind.)  32 x 3 up to 4.5, then 64 x 3, which where lengths are given waits for 5.5: half to full it is 1.12 at
    // 4.6 and 0.92 at 5.3, full 0.85 at both (a quarter real is still 1.05 at 6.9).  64 x 2 between the two, and where the long walks of 32 x 3
    // make one wave and up to a third (16 x (50, 500, 500), intra, full 17.5 and 15.0 us, every block 36.3 and 30.1; 80 x (60, 60, 60), half to full,
    // 1.19 and 0.97).  Given lengths of longer segments may do the same unseen (up to 1.09; 22 x (20, 1000, 300), intra, half to full, 1.15).
    const int64_t ctas = tiles(64) * slices, waves = long_walks(), wave = 3LL * n_sm;
    if (2 * ctas <= 9LL * n_sm && !(2 * ctas > 3LL * n_sm && waves > wave && 3 * waves <= 4 * wave)) GSIT_LAUNCH(8, 32, 1, 64, 3);
    if (2 * ctas <= (full ? 9LL : 11LL) * n_sm) GSIT_LAUNCH(8, 32, 2, 64, 2);
    GSIT_LAUNCH(8, 32, 2, 64, 3);
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
