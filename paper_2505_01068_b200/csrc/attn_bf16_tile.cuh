// The key walk of one query tile of the bf16 IM attention on mma.sync: TMA-fed, online softmax in registers, the normalised
// result staged in shared memory.  Included by the kernel that stores it (attn_bf16.cu) and by the one that goes on with the
// rest of the layer (attn_mlp_rows.cu).
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "ptx.cuh"
#include "tensor_map.cuh"

namespace gsit {
namespace {

using namespace ptx;

constexpr int KT = 64;          // keys per pipeline stage
constexpr int NTHREADS = 256;   // 8 warps
constexpr int WAIT_SPINS = 1 << 20;

// HD = head_dim, CW = features per column slice, R_ = 16-row query slabs per warp, KSTEP_ = keys per softmax
// step, MINB_ = CTAs per SM the register allocation must allow, SL_ = column slices per CTA, NSG_ = warps per head,
// STAGES_ = key tiles in flight.  Three make the warps of a CTA wait for the slowest; five over three, geometric means (and worst) over (50, 500, 500)
// and (30, 120, 90), 1 - 64 samples, intra and every block, full and half to full: head_dim 8 x 2 heads 0.95 (1.01), 16 x 2 heads 0.95 (1.02), 16 x 4
// 0.96 (1.03), 32 x 1 and 32 x 4 0.96 (1.02); at 64 the walks have one or two key tiles and it is the same.  In a layer of width 32 at (50, 500, 500)
// 4 % as well, but around one wave of short walks five can lose what the next kernel's early start gains (40 x (30, 120, 90), full, 13.8 -> 14.4).
template <int HD_, int CW_, int R_, int KSTEP_, int MINB_, int SL_ = 1, int NSG_ = 8 / (CW_ / HD_ * SL_), int STAGES_ = 5>
struct Cfg {
  static constexpr int HD = HD_, CW = CW_, R = R_, KSTEP = KSTEP_, MINB = MINB_, SL = SL_, STAGES = STAGES_;
  static constexpr int G = CW / HD;                 // heads per column slice
  static constexpr int NSG = NSG_;                  // slab groups (warps per head)
  static constexpr int WARPS = G * SL * NSG;        // warps that attend; further warps of the CTA have no part in it
  static constexpr int QT = 16 * R * NSG;           // query rows per CTA
  static constexpr int PITCH = CW * 2;              // bytes per tile row
  static constexpr int SWZ = (CW == 64) ? 7 : (CW == 32) ? 3 : 1;  // swizzle mask (128B / 64B / 32B modes)
  static constexpr int NT = KSTEP / 8;              // score n-tiles per step
  static constexpr int KSQ = (HD == 8) ? 1 : HD / 16;  // k-steps of Q K^T
  static constexpr int NTO = HD / 8;                // output n-tiles
  static constexpr int Q_BYTES = QT * PITCH;
  static constexpr int KV_BYTES = KT * PITCH;
  // shared memory from a 1024-byte boundary on: Q (slice by slice), K and V stages (the slices of a stage together), barriers
  static constexpr int Q_SLICE = ((Q_BYTES + 1023) / 1024) * 1024;
  static constexpr int OFF_K = SL * Q_SLICE, OFF_V = OFF_K + STAGES * SL * KV_BYTES, OFF_BAR = OFF_V + STAGES * SL * KV_BYTES;
  static constexpr int SMEM = OFF_BAR + 1024 /*align slack*/ + 128 /*barriers*/;
  static_assert(G >= 1 && WARPS >= 1 && STAGES <= 7 && QT <= 256 && (KSTEP == 32 || KSTEP == 64), "unsupported tile configuration");
};

// TMA shared-memory swizzle: 16-byte chunk index bits [4, 4+B) are XORed with address bits [7, 7+B).
template <int SWZ>
__device__ __forceinline__ uint32_t swz(uint32_t off) { return off ^ (((off >> 7) & SWZ) << 4); }

// Bounded wait: gives up after WAIT_SPINS polls, raises GSIT_DEVFLAG_TIMEOUT and lets the CTA run on
// (its results are then invalid, but nothing hangs).
__device__ __forceinline__ void mbar_wait(const Geometry& g, uint32_t bar, uint32_t parity) {
#pragma unroll 1
  for (int it = 0; it < WAIT_SPINS; ++it) {
    if (mbar_test(bar, parity)) return;
    if (it > 64) __nanosleep(64);
  }
  raise_flag(g, GSIT_DEVFLAG_TIMEOUT);
}
// The same by a whole warp, which then knows that its lanes stay together: nothing has to be done to bring them together again.
__device__ __forceinline__ void mbar_wait_warp(const Geometry& g, uint32_t bar, uint32_t parity) {
#pragma unroll 1
  for (int it = 0; it < WAIT_SPINS; ++it) {
    if (__all_sync(0xffffffffu, mbar_test(bar, parity))) return;
    if (it > 64) __nanosleep(64);
  }
  raise_flag(g, GSIT_DEVFLAG_TIMEOUT);
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2(uint32_t addr, uint32_t& r0, uint32_t& r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma_k16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                        uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_k8(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(b0));
}

template <bool V> struct BoolTag { static constexpr bool value = V; };
template <int V> struct IntTag { static constexpr int value = V; };

// A query tile: rows q0 .. of segment s of sample b, and the keys its block row opens.
struct Tile {
  int b, s, q0;
  int q_real_all;    // real rows of the tile
  int rows_in_tile;  // rows of the tile that exist in the activation matrices: in the padded layout all that belong to the segment
                     // (padding as +0); in the packed layout only the real ones -- what follows them in memory is another segment
  int kn0, kn1, kn2, nk0, nk1;  // real keys per open key segment, key tiles of the first two
  int T;             // key tiles to walk
  int q_real;        // rows that receive a computed result
  int kbase0, kbase1, kbase2;   // first row of each key segment
  int64_t grow0;     // first row of the tile in the activation matrices
};

// `bx` = (tile in cost order) * batch + sample: the query segments with the most keys to walk come first (seg_order packs the
// three segment indices, two bits each), and CTAs that run together work on the same tile of different samples, so the last wave is
// short and made of the cheapest tiles.
template <int QT>
__device__ __forceinline__ Tile find_tile(const Geometry& g, uint32_t allowed, int bx, int seg_order) {
  Tile t;
  t.b = bx % g.batch;
  int tile = bx / g.batch, s = seg_order & 3;
#pragma unroll
  for (int rank = 0; rank < 2; ++rank) {
    const int nts = (g.len(s) + QT - 1) / QT;
    if (tile >= nts) { tile -= nts; s = (seg_order >> (2 * rank + 2)) & 3; }
  }
  t.s = s;
  t.q0 = tile * QT;
  const int in_seg = min(QT, g.len(s) - t.q0);
  t.q_real_all = max(0, min(in_seg, valid_rows(g, t.b, s) - t.q0));
  t.rows_in_tile = g.row_start != nullptr ? t.q_real_all : in_seg;
  t.kn0 = ((allowed >> (3 * s + 0)) & 1u) ? valid_rows(g, t.b, 0) : 0;
  t.kn1 = ((allowed >> (3 * s + 1)) & 1u) ? valid_rows(g, t.b, 1) : 0;
  t.kn2 = ((allowed >> (3 * s + 2)) & 1u) ? valid_rows(g, t.b, 2) : 0;
  t.nk0 = (t.kn0 + KT - 1) / KT;
  t.nk1 = (t.kn1 + KT - 1) / KT;
  t.T = t.q_real_all > 0 ? t.nk0 + t.nk1 + (t.kn2 + KT - 1) / KT : 0;
  t.q_real = t.T > 0 ? t.q_real_all : 0;
  t.grow0 = (int64_t)seg_row0(g, t.b, s) + t.q0;
  t.kbase0 = seg_row0(g, t.b, 0);
  t.kbase1 = seg_row0(g, t.b, 1);
  t.kbase2 = seg_row0(g, t.b, 2);
  return t;
}

// Barriers of a CTA's walk; before the first use a __syncthreads().
template <typename C>
__device__ __forceinline__ void init_walk(uint32_t base, int tid) {
  if (tid != 0) return;
  constexpr int STAGES = C::STAGES;
  const uint32_t bar_full = base + C::OFF_BAR, bar_empty = bar_full + 8 * STAGES;
#pragma unroll
  for (int st = 0; st < STAGES; ++st) {
    mbar_init(bar_full + 8 * st, 1);
    mbar_init(bar_empty + 8 * st, C::WARPS);
  }
  mbar_init(bar_empty + 8 * STAGES, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Walks the keys of tile t (t.T > 0), by all threads of the CTA: the heads of column slices first_slice .. + SL - 1, whose columns start at
// xq, xk, xv in the three maps.  Leaves the normalised rows as bf16 where Q was (swizzled rows of CW columns, slice by slice) and ends
// with a barrier; lse (with the heads of the whole problem) may be null.  meanwhile(): what every thread does once Q is there.
// UNIFORM: what is the same in a whole warp is made known as such (ptx.cuh), which nearly every kernel is faster for.
template <typename C, int CTA_WARPS, bool UNIFORM = true, typename F>
__device__ __forceinline__ void attend_tile(const Geometry& g, const Tile& t_, const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                                            const int xq, const int xk, const int xv, const int first_slice, const float sl2, float* __restrict__ lse,
                                            const uint32_t base, F meanwhile) {
  constexpr int HD = C::HD, CW = C::CW, G = C::G, R = C::R, PITCH = C::PITCH, SWZ = C::SWZ,
                KSTEP = C::KSTEP, NT = C::NT, KSQ = C::KSQ, NTO = C::NTO, SL = C::SL, STAGES = C::STAGES;
  auto same = [](int v) { return UNIFORM ? uniform(v) : v; };
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if constexpr (UNIFORM) mbar_wait_warp(g, bar, parity);
    else mbar_wait(g, bar, parity);
  };
  constexpr bool HOIST = (R > 1);  // several query slabs per warp reuse the K/V fragments of a step
  const int tid = threadIdx.x, warp = same(tid >> 5), lane = tid & 31;
  const int head = warp % (G * SL), sg = warp / (G * SL), slice = head / G, head_in_slice = head % G;
  // Known at compile time where every warp of the CTA attends: a walk behind a branch takes longer (14 key tiles of one 16-row slab at head_dim 8:
  // 13.75 us, 13.50 without the branch; one sample of (50, 500, 500) 8.96 and 8.80).  Not with four slabs per warp, which then spill
  // (64 samples of it 42.05 and 42.35).
  constexpr bool EVERY_WARP = C::WARPS == CTA_WARPS && R < 4;
  const bool active = EVERY_WARP || warp < C::WARPS;
  const uint32_t sQall = base, sK = base + C::OFF_K, sV = base + C::OFF_V;
  const uint32_t sQ = base + slice * C::Q_SLICE;
  const uint32_t bar_full = base + C::OFF_BAR;          // STAGES barriers of 8 bytes: TMA bytes have landed
  const uint32_t bar_empty = bar_full + 8 * STAGES;     // STAGES barriers: all attending warps are done with the stage
  const uint32_t bar_q = bar_empty + 8 * STAGES;
  const int cb = head_in_slice * (HD / 8);  // first 16-byte chunk of this warp's head inside a tile row
  const int b = t_.b, s = t_.s, q0 = t_.q0, kn0 = t_.kn0, kn1 = t_.kn1, kn2 = t_.kn2, nk0 = t_.nk0, nk1 = t_.nk1, T = same(t_.T), q_real = same(t_.q_real);
  const int kbase0 = t_.kbase0, kbase1 = t_.kbase1, kbase2 = t_.kbase2;
  const int64_t grow0 = t_.grow0;

  auto locate = [&](int i, int& krem, int& yrow) {
    int t = i, r = 0;
    if (t >= nk0) { t -= nk0; r = 1; if (t >= nk1) { t -= nk1; r = 2; } }
    const int kn = (r == 0) ? kn0 : (r == 1) ? kn1 : kn2;
    krem = kn - t * KT;
    yrow = ((r == 0) ? kbase0 : (r == 1) ? kbase1 : kbase2) + t * KT;
  };
  auto issue = [&](int i) {  // one thread: TMA loads of key tile i (of tile i - T in a second walk) into its stage
    int krem, yrow;
    locate(i >= T ? i - T : i, krem, yrow);
    const int st = i % STAGES;
    mbar_expect_tx(bar_full + 8 * st, 2 * SL * C::KV_BYTES);
#pragma unroll
    for (int sl = 0; sl < SL; ++sl) {
      tma_load_2d(sK + (st * SL + sl) * C::KV_BYTES, &tmK, xk + sl * CW, yrow, bar_full + 8 * st);
      tma_load_2d(sV + (st * SL + sl) * C::KV_BYTES, &tmV, xv + sl * CW, yrow, bar_full + 8 * st);
    }
  };

  float O[R][NTO][4];
  float m[R][2], l[R][4];  // m: reference of rows g and g + 8, in base-2 score units; l: accumulator tile of P 1 (elements 0 and
                           // 2 are the sums of those rows)
  auto reset = [&]() {
#pragma unroll
    for (int r_ = 0; r_ < R; ++r_) {
      m[r_][0] = m[r_][1] = -INFINITY;
      l[r_][0] = l[r_][1] = l[r_][2] = l[r_][3] = 0.f;
#pragma unroll
      for (int n = 0; n < NTO; ++n) O[r_][n][0] = O[r_][n][1] = O[r_][n][2] = O[r_][n][3] = 0.f;
    }
  };
  reset();

  int next_issue = 0;  // meaningful in thread 0 only: next key tile to request
  if (tid == 0) {
    mbar_expect_tx(bar_q, SL * C::Q_BYTES);
#pragma unroll
    for (int sl = 0; sl < SL; ++sl) tma_load_2d(sQall + sl * C::Q_SLICE, &tmQ, xq + sl * CW, (int)grow0, bar_q);
    for (; next_issue < STAGES && next_issue < T; ++next_issue) issue(next_issue);
  }

  // ---- query fragments, kept in registers for the whole key walk ----
  uint32_t QF[R][KSQ][4];
  if (active) {
    wait(bar_q, 0);
#pragma unroll
    for (int r_ = 0; r_ < R; ++r_) {
      const int row0 = (sg * R + r_) * 16;
      if constexpr (HD == 8) {
        const int row = row0 + (lane & 15);
        ldsm_x2(sQ + swz<SWZ>(row * PITCH + cb * 16), QF[r_][0][0], QF[r_][0][1]);
        QF[r_][0][2] = QF[r_][0][3] = 0;
      } else {
        const int mi = lane >> 3;
        const int row = row0 + (mi & 1) * 8 + (lane & 7);
#pragma unroll
        for (int ks = 0; ks < KSQ; ++ks)
          ldsm_x4(sQ + swz<SWZ>(row * PITCH + (cb + ks * 2 + (mi >> 1)) * 16), QF[r_][ks][0], QF[r_][ks][1],
                  QF[r_][ks][2], QF[r_][ks][3]);
      }
    }
  }

  meanwhile();

  // One pipeline stage (KT keys) for all query slabs of this warp.  RAGGED: the stage holds fewer than KT real keys;
  // the instantiation then covers only the first NTV score n-tiles (8 keys each, NTV even: whole 16-key groups of
  // P V), so that a tile with few real keys costs proportionally less, and only its last two n-tiles are masked
  // element by element.  Everything stays straight-line code inside an instantiation.
  //
  // Reference of the exponentials.  A softmax does not depend on what is subtracted from the scores as long as nothing
  // overflows, and float (and bf16 weights, which share its exponents) has room for 2^127: the reference of a row is the
  // maximum of its FIRST key step and stays (SAFE = false).  The weight of that maximum is 1, so the row sum cannot
  // underflow; a later score would have to exceed the reference by 2^90 to endanger it, and the end of the walk checks for
  // that: then the CTA walks its keys again with the running maximum (SAFE = true).  The running maximum cost 60 of the
  // 207 instructions per 16 x 64 scores and put its shuffles and the rescale between Q K^T and the exponentials.
  auto process = [&](auto safe_tag, auto ragged_tag, auto ntv_tag, const uint32_t sKs, const uint32_t sVs, const int krem, const bool first_tile) {
    constexpr bool SAFE = decltype(safe_tag)::value;
    constexpr bool RAGGED = decltype(ragged_tag)::value;
    constexpr int NTV = decltype(ntv_tag)::value;  // n-tiles computed (== NT for a full tile)
    static_assert(NTV % 2 == 0 && NTV >= 2 && NTV <= NT && (KT == KSTEP || !RAGGED || NTV == NT), "n-tile count");
    if constexpr (RAGGED) {
      // Rows past the valid length hold whatever follows in memory: clear this head's part of them in V so that a
      // zero weight times a NaN/Inf value cannot poison the accumulator (their scores become -inf below).  Warps
      // sharing the head write the same zeros.
      constexpr int KROWS = (KT == KSTEP) ? NTV * 8 : KT;  // key rows of the stage that the products read
      for (int idx = lane; idx < (KROWS - krem) * (HD / 8); idx += 32) {
        const int row = krem + idx / (HD / 8), ch = cb + idx % (HD / 8);
        asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(sVs + swz<SWZ>(row * PITCH + ch * 16)), "r"(0) : "memory");
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
    }
#pragma unroll
    for (int stp = 0; stp < KT / KSTEP; ++stp) {
      const int kb = stp * KSTEP;
      if (RAGGED && kb >= krem) break;
      uint32_t KF[NT][KSQ][2];
      uint32_t VF[KSTEP / 16][NTO][2];

      auto load_k_pair = [&](int p) {  // K fragments of score n-tiles 2p, 2p+1 (HD >= 16)
        const int mi = lane >> 3;
        const int key = kb + p * 16 + (mi >> 1) * 8 + (lane & 7);
#pragma unroll
        for (int ks = 0; ks < KSQ; ++ks)
          ldsm_x4(sKs + swz<SWZ>(key * PITCH + (cb + ks * 2 + (mi & 1)) * 16), KF[2 * p][ks][0], KF[2 * p][ks][1],
                  KF[2 * p + 1][ks][0], KF[2 * p + 1][ks][1]);
      };
      auto load_v_pair = [&](int kk, int np) {  // V fragments of key step kk, output n-tiles 2np, 2np+1 (HD >= 16)
        const int mi = lane >> 3;
        const int key = kb + kk * 16 + (mi & 1) * 8 + (lane & 7);
        ldsm_x4_t(sVs + swz<SWZ>(key * PITCH + (cb + np * 2 + (mi >> 1)) * 16), VF[kk][2 * np][0], VF[kk][2 * np][1],
                  VF[kk][2 * np + 1][0], VF[kk][2 * np + 1][1]);
      };
      auto load_k8 = [&](int j) {  // HD == 8: K fragments of n-tiles 4j .. 4j+3 (32 keys)
        ldsm_x4(sKs + swz<SWZ>((kb + j * 32 + lane) * PITCH + cb * 16), KF[4 * j][0][0], KF[4 * j + 1][0][0],
                KF[4 * j + 2][0][0], KF[4 * j + 3][0][0]);
      };
      auto load_v8 = [&](int j) {  // HD == 8: V fragments of key steps 2j, 2j+1 (32 keys)
        ldsm_x4_t(sVs + swz<SWZ>((kb + j * 32 + lane) * PITCH + cb * 16), VF[2 * j][0][0], VF[2 * j][0][1],
                  VF[2 * j + 1][0][0], VF[2 * j + 1][0][1]);
      };

      if constexpr (HOIST) {
        if constexpr (HD == 8) {
#pragma unroll
          for (int j = 0; j < (NTV + 3) / 4; ++j) { load_k8(j); load_v8(j); }
        } else {
#pragma unroll
          for (int p = 0; p < NTV / 2; ++p) load_k_pair(p);
#pragma unroll
          for (int kk = 0; kk < NTV / 2; ++kk)
#pragma unroll
            for (int np = 0; np < NTO / 2; ++np) load_v_pair(kk, np);
        }
      }

#pragma unroll
      for (int r_ = 0; r_ < R; ++r_) {
        const int row0 = (sg * R + r_) * 16;
        if (row0 >= q_real) continue;  // slab of padding rows only
        float S[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n) S[n][0] = S[n][1] = S[n][2] = S[n][3] = 0.f;

        // ---- S = Q K^T (raw dot products) ----
        if constexpr (HD == 8) {
#pragma unroll
          for (int j = 0; j < (NTV + 3) / 4; ++j) {
            if constexpr (!HOIST) load_k8(j);
#pragma unroll
            for (int n = 4 * j; n < 4 * j + 4; ++n)
              if (n < NTV) mma_k8(S[n], QF[r_][0][0], QF[r_][0][1], KF[n][0][0]);
          }
        } else {
#pragma unroll
          for (int p = 0; p < NTV / 2; ++p) {
            if constexpr (!HOIST) load_k_pair(p);
#pragma unroll
            for (int ks = 0; ks < KSQ; ++ks) {
              mma_k16(S[2 * p], QF[r_][ks][0], QF[r_][ks][1], QF[r_][ks][2], QF[r_][ks][3], KF[2 * p][ks][0],
                      KF[2 * p][ks][1]);
              mma_k16(S[2 * p + 1], QF[r_][ks][0], QF[r_][ks][1], QF[r_][ks][2], QF[r_][ks][3], KF[2 * p + 1][ks][0],
                      KF[2 * p + 1][ks][1]);
            }
          }
        }
        // ---- keys past the valid length get weight exactly zero ----
        if constexpr (RAGGED) {
          const int c0 = kb + (lane & 3) * 2;
#pragma unroll
          for (int n = (KT == KSTEP ? NTV - 2 : 0); n < NTV; ++n) {  // the invalid keys are a suffix of the last 16-key group
            if (c0 + n * 8 >= krem) S[n][0] = S[n][2] = -INFINITY;
            if (c0 + n * 8 + 1 >= krem) S[n][1] = S[n][3] = -INFINITY;
          }
        }
        // ---- reference of the row (base 2, scale folded into sl2); pairwise trees keep dependency chains short ----
        float al0 = 1.f, al1 = 1.f;
        if (SAFE || (first_tile && kb == 0)) {
          float t0[NTV], t1[NTV];
#pragma unroll
          for (int n = 0; n < NTV; ++n) { t0[n] = fmaxf(S[n][0], S[n][1]); t1[n] = fmaxf(S[n][2], S[n][3]); }
#pragma unroll
          for (int cnt = NTV; cnt > 1; cnt = (cnt + 1) / 2)  // pairwise tree over any count
#pragma unroll
            for (int n = 0; n < cnt / 2; ++n) {
              t0[n] = fmaxf(t0[n], t0[n + (cnt + 1) / 2]);
              t1[n] = fmaxf(t1[n], t1[n + (cnt + 1) / 2]);
            }
          float mx0 = t0[0], mx1 = t1[0];
          mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
          mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
          mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2)) * sl2;
          mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2)) * sl2;
          // every key tile that is walked holds at least one real key, so the new maximum is finite (only the old one can
          // be -inf, on the first tile, where the factor below becomes exp2(-inf) = 0)
          const float mn0 = fmaxf(m[r_][0], mx0), mn1 = fmaxf(m[r_][1], mx1);
          if constexpr (SAFE) {
            al0 = ex2(m[r_][0] - mn0);
            al1 = ex2(m[r_][1] - mn1);
          }
          m[r_][0] = mn0;
          m[r_][1] = mn1;
        }
        // One packed FMA forms s * sl2 - m * sl2 for a pair of scores; each gets its own f32 ex2 (the
        // packed bf16 form of ex2 issues two special-function operations as well, plus unpacking), and the pair is
        // rounded once into the bf16x2 layout of the A operand of P V.  The row sum is taken by the tensor core from
        // those same bf16 weights (a column of ones appended to V), so numerator and denominator of the softmax see
        // identical values.
        const float2 sl2v = make_float2(sl2, sl2), nm0 = make_float2(-m[r_][0], -m[r_][0]), nm1 = make_float2(-m[r_][1], -m[r_][1]);
        uint32_t P[NTV][2];
#pragma unroll
        for (int n = 0; n < NTV; ++n) {
          const float2 x0 = __ffma2_rn(make_float2(S[n][0], S[n][1]), sl2v, nm0);
          const float2 x1 = __ffma2_rn(make_float2(S[n][2], S[n][3]), sl2v, nm1);
          P[n][0] = __byte_perm(__float_as_uint(ex2(x0.x)), __float_as_uint(ex2(x0.y)), 0x7632);
          P[n][1] = __byte_perm(__float_as_uint(ex2(x1.x)), __float_as_uint(ex2(x1.y)), 0x7632);
        }
        if constexpr (SAFE) {
          l[r_][0] *= al0;
          l[r_][2] *= al1;
#pragma unroll
          for (int n = 0; n < NTO; ++n) {
            O[r_][n][0] *= al0; O[r_][n][1] *= al0;
            O[r_][n][2] *= al1; O[r_][n][3] *= al1;
          }
        }
        // ---- O += P V and l += P 1, the weights being the A operand ----
#pragma unroll
        for (int kk = 0; kk < NTV / 2; ++kk) {
          const uint32_t a0 = P[2 * kk][0], a1 = P[2 * kk][1], a2 = P[2 * kk + 1][0], a3 = P[2 * kk + 1][1];
          mma_k16(l[r_], a0, a1, a2, a3, 0x3F803F80u, 0x3F803F80u);  // B = ones: every column of the result is the row sum
          if constexpr (HD == 8) {
            if constexpr (!HOIST) { if ((kk & 1) == 0) load_v8(kk / 2); }
            mma_k16(O[r_][0], a0, a1, a2, a3, VF[kk][0][0], VF[kk][0][1]);
          } else {
#pragma unroll
            for (int np = 0; np < NTO / 2; ++np) {
              if constexpr (!HOIST) load_v_pair(kk, np);
              mma_k16(O[r_][2 * np], a0, a1, a2, a3, VF[kk][2 * np][0], VF[kk][2 * np][1]);
              mma_k16(O[r_][2 * np + 1], a0, a1, a2, a3, VF[kk][2 * np + 1][0], VF[kk][2 * np + 1][1]);
            }
          }
        }
      }  // slabs
    }    // steps
  };

  auto walk = [&](auto safe_tag, const int from) {  // tiles from .. from + T - 1 of the stage sequence
    const int end = from + T;
    for (int i = from; i < end; ++i) {
      const int st = i % STAGES;
      if (tid == 0) {
        // request further key tiles whose stage every warp has released; never block unless tile i itself is missing
        while (next_issue < end) {
          const uint32_t eb = bar_empty + 8 * (next_issue % STAGES);
          const uint32_t par = ((next_issue / STAGES) - 1) & 1;
          if (next_issue >= STAGES) {
            if (next_issue <= i) mbar_wait(g, eb, par);
            else if (!mbar_test(eb, par)) break;
          }
          issue(next_issue);
          ++next_issue;
        }
      }
      __syncwarp();
      wait(bar_full + 8 * st, (i / STAGES) & 1);
      int krem, yrow;
      locate(i - from, krem, yrow);
      krem = same(krem);
      const bool first = i == from;
      const uint32_t sKs = sK + (st * SL + slice) * C::KV_BYTES, sVs = sV + (st * SL + slice) * C::KV_BYTES;
      if (krem >= KT) {
        process(safe_tag, BoolTag<false>{}, IntTag<NT>{}, sKs, sVs, KT, first);
      } else if constexpr (KT == KSTEP && NT == 8) {  // as many 16-key groups as hold real keys
        if (krem <= 16) process(safe_tag, BoolTag<true>{}, IntTag<2>{}, sKs, sVs, krem, first);
        else if (krem <= 32) process(safe_tag, BoolTag<true>{}, IntTag<4>{}, sKs, sVs, krem, first);
        else if (krem <= 48) process(safe_tag, BoolTag<true>{}, IntTag<6>{}, sKs, sVs, krem, first);
        else process(safe_tag, BoolTag<true>{}, IntTag<8>{}, sKs, sVs, krem, first);
      } else {
        process(safe_tag, BoolTag<true>{}, IntTag<NT>{}, sKs, sVs, krem, first);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_empty + 8 * st);  // this warp is done with the stage
    }
  };
  if (active) walk(BoolTag<false>{}, 0);
  bool fits = true;  // did every row stay in range of its reference?
#pragma unroll
  for (int r_ = 0; r_ < R; ++r_) {
    if (!active || (sg * R + r_) * 16 >= q_real) continue;
    const int row = (sg * R + r_) * 16 + (lane >> 2);
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      if (row + 8 * half >= q_real) continue;  // rows past the last real one hold anything
      float top = 0.f;
#pragma unroll
      for (int n = 0; n < NTO; ++n) top = fmaxf(top, fmaxf(fabsf(O[r_][n][2 * half]), fabsf(O[r_][n][2 * half + 1])));
      fits = fits && top < 1.2e27f && l[r_][2 * half] < 1.2e27f;  // 2^90; a NaN sum does not fit either
    }
  }
  if (!__syncthreads_and(fits)) {
    reset();
    if (active) walk(BoolTag<true>{}, T);
  }

  // ---- normalise and stage the tile in shared memory.  A warp overwrites only the Q bytes it alone read. ----
#pragma unroll
  for (int r_ = 0; r_ < R; ++r_) {
    const int row0 = (sg * R + r_) * 16;
    if (!active || row0 >= q_real) continue;
    const float l0 = l[r_][0], l1 = l[r_][2];
    const float inv0 = l0 > 0.f ? 1.f / l0 : 0.f, inv1 = l1 > 0.f ? 1.f / l1 : 0.f;
    const int rowA = row0 + (lane >> 2), rowB = rowA + 8;
#pragma unroll
    for (int n = 0; n < NTO; ++n) {
      const int colb = (head_in_slice * HD + n * 8 + (lane & 3) * 2) * 2;  // byte column in the tile row
      const uint32_t vA = pack_bf16(O[r_][n][0] * inv0, O[r_][n][1] * inv0);
      const uint32_t vB = pack_bf16(O[r_][n][2] * inv1, O[r_][n][3] * inv1);
      asm volatile("st.shared.b32 [%0], %1;" ::"r"(sQ + swz<SWZ>(rowA * PITCH + colb)), "r"(vA) : "memory");
      asm volatile("st.shared.b32 [%0], %1;" ::"r"(sQ + swz<SWZ>(rowB * PITCH + colb)), "r"(vB) : "memory");
    }
    if (lse != nullptr && (lane & 3) == 0) {
      float* lp = lse + ((int64_t)b * g.heads + first_slice * G + head) * g.L + g.off(s) + q0;
      const float ln2 = 0.6931471805599453f;
      if (rowA < q_real) lp[rowA] = l0 > 0.f ? (m[r_][0] + log2f(l0)) * ln2 : -INFINITY;
      if (rowB < q_real) lp[rowB] = l1 > 0.f ? (m[r_][1] + log2f(l1)) * ln2 : -INFINITY;
    }
  }
  __syncthreads();
}

}  // namespace
}  // namespace gsit
