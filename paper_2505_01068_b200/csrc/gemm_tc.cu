// bf16 linear layer C = act(A W^T + bias) (+ residual) on the 5th-generation tensor cores (tcgen05), for the shared
// QKV projection at large d_model (Section "Multimodal Transformers as Graphs": one W_q, W_k, W_v for the whole
// concatenated sequence) and for every linear layer of widths that the fused layer halves do not cover.
//
// Persistent grid, one CTA per SM.  Large problems run on pairs of CTAs (clusters of two, cta_group::2): a tile is 256 rows x
// bn columns, each CTA loads its own 128 rows of A and HALF of the W rows, one tcgen05.mma of M 256 multiplies both halves
// and each CTA keeps the accumulator of its own rows.  What bounds a 128 x 256 tile per CTA is the traffic from L2: 48 KB per
// 64-wide k-block of 532 clocks on every SM is 25 TB/s; the pair needs 32 KB.  (M 278528, N 1536, K 512: 550 us one CTA per
// tile.)  Small problems keep one CTA per tile and narrower tiles, so that all SMs have one.
//
// Eleven warps:
//   warp 0      TMA producer of A and W: boxes of 64 k's (128-byte rows, 128-byte swizzle) into a ring of stages; in a pair the
//               copies of both CTAs complete on the first CTA's barrier
//   warp 1      allocates 512 TMEM columns and (in a pair: the first CTA's) issues tcgen05.mma; the accumulator is
//               double-buffered (2 x 256 columns), so the epilogue of tile i overlaps the main loop of tile i + 1
//   warps 2..9  epilogue: two groups of four warps take alternate 128-byte-wide column boxes of the tile (64 bf16 or 32 float
//               columns); thread = output row = TMEM lane: tcgen05.ld, bias / ReLU / residual / padded-row zeroing, the row's
//               piece into a shared-memory box in the 128-byte swizzle, and one TMA store per box, so that every line of C is
//               written whole (16-byte stores of 32 different rows per instruction made the float-output layers wait on
//               their stores: 687 us for N 512, K 512 with a residual)
//   warp 10     float output with a residual: loads the residual boxes by TMA ahead of the epilogue, into the very boxes the
//               sums are then stored from
// Tiles are numbered with the column tile fastest, so the CTAs that share an A tile run at the same time and W stays
// in L2.  Row tiles without a real row are not multiplied at all: their part of C is zero.
// Every wait is bounded (GSIT_DEVFLAG_TIMEOUT instead of a hang) and TMEM is always released.
#include <cuda.h>

#include "common.cuh"
#include "ptx.cuh"
#include "tensor_map.cuh"
#include "tmem_ldst.cuh"

namespace gsit {
namespace {

using namespace ptx;

constexpr int GM = 128, GK = 64;          // rows per CTA and tile, k-block width
constexpr int G_THREADS = 352;
constexpr int A_STAGE = GM * GK * 2;      // 16 KB
constexpr int BOX = GM * 128;             // one epilogue box: 128 rows of 128 bytes
constexpr int G_MAX_STAGES = 8, MAX_BOXES = 3;  // boxes per epilogue group
constexpr int G_TABLE = 512;              // tiles of a CTA whose state is looked up once
constexpr int G_BAR_BYTES = 512 + 1024 + G_TABLE;   // barriers, each epilogue group's half of the tile's bias, and that table
constexpr int G_MIN_SMEM = 120 * 1024;    // more than half an SM's shared memory: one CTA per SM, so 512 TMEM columns fit

// STORE_PACKED: bf16, rows of the packed layout: a tile whose rows are all this call's leaves by TMA like the others; in the (at
// most two) tiles that share rows with neighbouring samples every thread writes its own row, if it is one of the call's.  (Every
// tile row by row, 16 bytes of 32 rows per instruction: 461 us at 243712 real rows, N 1536, K 512; now 338.)
enum Mode { STORE_BF16 = 0, STORE_F32 = 1, STORE_PACKED = 2 };

struct GemmParams {
  int M, N, K;
  int bn;            // columns per tile (a multiple of 64, <= 256)
  int tiles_n, n_tiles;
  int stages, stage_bytes;
  int boxes;         // per epilogue group
  const float* bias;
  int has_residual;
  __nv_bfloat16* C; int64_t ldc;   // for what is not written by TMA: padding tiles, shared tiles of STORE_PACKED
  int relu, mask_rows;
  int packed;        // rows are the packed layout's: only rows_begin(g) .. rows_end(g) - 1 (read on the device) are computed
                     // and written, all of them real; everything outside that range is left untouched
};

// Does the tile of `rows` rows at m0 hold a real row?  Walks the segments it overlaps.
__device__ __forceinline__ bool tile_real(const Geometry& g, int m0, int rows, int M) {
  const int end = min(m0 + rows, M);
  for (int pos = m0; pos < end;) {
    const int b = pos / g.L, p = pos - b * g.L, s = segment_of(g, p);
    if (p - g.off(s) < valid_rows(g, b, s)) return true;
    pos = b * g.L + g.off(s) + g.len(s);
  }
  return false;
}

__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t in_first_cta(uint32_t addr) {  // the same shared-memory offset in the pair's first CTA
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// A tensor copy into this CTA's shared memory that completes on a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t cluster_bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(cluster_bar) : "memory");
}
template <bool PAIR>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if constexpr (PAIR)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
  else
    umma_ss(d, a, b, idesc, acc);
}
template <bool PAIR>
__device__ __forceinline__ void commit(uint32_t bar) {  // in a pair: the barrier of both CTAs
  if constexpr (PAIR)
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
  else
    umma_commit(bar);
}

template <bool PAIR, int MODE>
__global__ void __launch_bounds__(G_THREADS, 1)
linear_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW,
                 const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmR, const __grid_constant__ Geometry g, const __grid_constant__ GemmParams p) {
  constexpr int CTAS = PAIR ? 2 : 1, CW = (MODE == STORE_F32) ? 32 : 64;  // columns per epilogue box
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t s_box = base + p.stages * p.stage_bytes;
  const uint32_t bars = s_box + 2 * p.boxes * BOX;
  const uint32_t bar_full = bars, bar_empty = bar_full + 8 * G_MAX_STAGES, bar_accf = bar_empty + 8 * G_MAX_STAGES,
                 bar_acce = bar_accf + 16, bar_resf = bar_acce + 16, bar_rese = bar_resf + 16 * MAX_BOXES, slot = bar_rese + 16 * MAX_BOXES,
                 slot_gave_up = slot + 4, s_bias = bars + 512, s_table = s_bias + 1024;
  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  const uint32_t rank = PAIR ? cta_rank() : 0;
  const WaitCtx wc{g.status, slot_gave_up};
  const int kblocks = p.K / GK;
  const bool res = MODE == STORE_F32 && p.has_residual;

  if (tid == 0) {
    map_early(tmA);
    map_early(tmW);
    map_early(tmC);
    for (int i = 0; i < p.stages; ++i) { mbar_init(bar_full + 8 * i, 1); mbar_init(bar_empty + 8 * i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar_accf + 8 * i, 1); mbar_init(bar_acce + 8 * i, 8 * CTAS); }
    for (int i = 0; i < 2 * MAX_BOXES; ++i) { mbar_init(bar_resf + 8 * i, 1); mbar_init(bar_rese + 8 * i, 1); }
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(slot_gave_up), "r"(0u) : "memory");
    mbar_init_fence();
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(512u) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      tmem_alloc(slot, 512);
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();  // both CTAs' barriers exist before either signals the other's
  tc_fence_after();
  uint32_t tmem;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(tmem) : "r"(slot) : "memory");
  load_params_early(g, p);
  grid_dep_wait();
  grid_dep_launch();

  // The walk over the tiles, the same in every role: first row of the tile (of the pair), first column.
  const int row_lo = uniform(p.packed ? rows_begin(g) : 0), row_hi = uniform(p.packed ? rows_end(g) : p.M);
  const int t0 = PAIR ? blockIdx.x >> 1 : blockIdx.x, dt = PAIR ? gridDim.x >> 1 : gridDim.x;
  // What is done with tile t, the i-th of this CTA: multiplied, zeroed (padding only) or left alone.  Which of the first two needs the lengths and
  // divisions, the better part of a thousand clocks, and the MMA warp stood still for them at every tile (a tile's products at K 512
  // take 4256): all threads together look the first tiles up ahead.  The four products of a layer of 128 x (128, 1024, 1024), d 512, a
  // quarter of the samples at half length, one by one: 385, 250, 533, 493 -> 344, 234, 466, 467 us, the second figures with warp-uniform control
  // flow as well; the projection of 32 x (39, 55, 400) at d 128 with its attention 23.9 -> 22.3.
  enum { MULTIPLY = 0, PADDING = 1, OUTSIDE = 2 };
  auto look_up = [&](int t) -> int {
    const int m0 = (t / p.tiles_n) * GM * CTAS;
    if (m0 + GM * CTAS <= row_lo || m0 >= row_hi) return OUTSIDE;
    return p.mask_rows && !p.packed && !tile_real(g, m0, GM * CTAS, p.M) ? PADDING : MULTIPLY;
  };
  for (int i = tid; i < G_TABLE && t0 + i * (int64_t)dt < p.n_tiles; i += G_THREADS)
    asm volatile("st.shared.u8 [%0], %1;" ::"r"(s_table + i), "r"(look_up(t0 + i * dt)) : "memory");
  __syncthreads();
  auto state = [&](int t, int i) {
    if (i >= G_TABLE) return uniform(look_up(t));
    int v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(s_table + i) : "memory");
    return uniform(v);
  };

  if (warp == 0) {
    // ================================ TMA producer ================================
    const int wrows = p.bn / CTAS;
    int st = 0, use = 0;  // stage of the next k-block, times round the ring
#pragma unroll 1
    for (int t = t0, j = 0; t < p.n_tiles; t += dt, ++j) {
      if (state(t, j) != MULTIPLY) continue;
      const int m0 = (t / p.tiles_n) * GM * CTAS, n0 = (t % p.tiles_n) * p.bn;
#pragma unroll 1
      for (int kb = 0; kb < kblocks; ++kb) {
        if (use > 0) mbar_wait_warp(wc, bar_empty + 8 * st, (use - 1) & 1);
        if (elect_one()) {
          const uint32_t sA = base + st * p.stage_bytes, bytes = (uint32_t)(A_STAGE + wrows * GK * 2);
          if constexpr (PAIR) {
            if (rank == 0) mbar_expect_tx(bar_full + 8 * st, 2 * bytes);
            const uint32_t bar = in_first_cta(bar_full + 8 * st);
            tma_load_2d_pair(sA, &tmA, kb * GK, m0 + rank * GM, bar);
            tma_load_2d_pair(sA + A_STAGE, &tmW, kb * GK, n0 + rank * wrows, bar);
          } else {
            mbar_expect_tx(bar_full + 8 * st, bytes);
            tma_load_2d(sA, &tmA, kb * GK, m0, bar_full + 8 * st);
            tma_load_2d(sA + A_STAGE, &tmW, kb * GK, n0, bar_full + 8 * st);
          }
        }
        __syncwarp();
        if (++st == p.stages) { st = 0; ++use; }
      }
    }
  } else if (warp == 1) {
    // ================================ MMA issuer ================================
    if (rank == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.bn >> 3) << 17) | ((uint32_t)((GM * CTAS) >> 4) << 24);
      int st = 0, use = 0, i = 0;  // stage of the next k-block, times round the ring; tiles multiplied
#pragma unroll 1
      for (int t = t0, j = 0; t < p.n_tiles; t += dt, ++j) {
        if (state(t, j) != MULTIPLY) continue;
        const int ab = i & 1;
        if (i >= 2) mbar_wait_cluster(wc, bar_acce + 8 * ab, ((i >> 1) - 1) & 1);  // the epilogues have drained this accumulator
        tc_fence_after();
#pragma unroll 1
        for (int kb = 0; kb < kblocks; ++kb) {
          mbar_wait_warp(wc, bar_full + 8 * st, use & 1);
          tc_fence_after();
          if (elect_one()) {
            const uint32_t sA = base + st * p.stage_bytes;
#pragma unroll
            for (int k = 0; k < GK / 16; ++k)
              mma<PAIR>(tmem + ab * 256, smem_desc_sw128(sA + 32 * k), smem_desc_sw128(sA + A_STAGE + 32 * k), idesc, (kb > 0 || k > 0) ? 1u : 0u);
            commit<PAIR>(bar_empty + 8 * st);
            if (kb + 1 == kblocks) commit<PAIR>(bar_accf + 8 * ab);
          }
          __syncwarp();
          if (++st == p.stages) { st = 0; ++use; }
        }
        ++i;
      }
    }
  } else if (warp == 10) {
    // ================================ residual loader ================================
    if (res) {
      int use[2] = {0, 0};
#pragma unroll 1
      for (int t = t0, j = 0; t < p.n_tiles; t += dt, ++j) {
        if (state(t, j) != MULTIPLY) continue;
        const int m0 = (t / p.tiles_n) * GM * CTAS, n0 = (t % p.tiles_n) * p.bn;
#pragma unroll 1
        for (int c = 0; c < p.bn / CW && n0 + c * CW < p.N; ++c) {
          const int grp = c & 1, u = grp ? use[1]++ : use[0]++, box = grp * MAX_BOXES + u % p.boxes;
          if (u >= p.boxes) mbar_wait_warp(wc, bar_rese + 8 * box, (u / p.boxes - 1) & 1);
          if (elect_one()) {
            mbar_expect_tx(bar_resf + 8 * box, BOX);
            tma_load_2d(s_box + (grp * p.boxes + u % p.boxes) * BOX, &tmR, n0 + c * CW, m0 + rank * GM, bar_resf + 8 * box);
          }
          __syncwarp();
        }
      }
    }
  } else {
    // ================================ epilogue: one thread per output row ================================
    const int quarter = warp & 3, grp = (warp - 2) >> 2, r = quarter * 32 + lane;
    const bool leader = (warp == 2 || warp == 6) && lane == 0;   // issues the group's TMA stores
    const uint32_t tl = tmem + ((uint32_t)(quarter << 5) << 16);
    auto group_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory"); };
    int i = 0, u = 0;  // tiles with an accumulator, boxes of this group so far
#pragma unroll 1
    for (int t = t0, j = 0; t < p.n_tiles; t += dt, ++j) {
      const int what = state(t, j);
      if (what == OUTSIDE) continue;
      const int mp = (t / p.tiles_n) * GM * CTAS, n0 = (t % p.tiles_n) * p.bn, m0 = mp + rank * GM;
      if (what == PADDING) {  // zeros, eight threads per 128-byte line
        constexpr int ES = MODE == STORE_F32 ? 4 : 2;
        for (int c = grp; c < p.bn / CW; c += 2)
          for (int k = tid & 127; k < GM * 8; k += 128) {
            const int row = m0 + (k >> 3), col = n0 + c * CW + (k & 7) * (16 / ES);
            if (row < p.M && col < p.N)
              *reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(p.C) + ((int64_t)row * p.ldc + col) * ES) = make_uint4(0, 0, 0, 0);
          }
        continue;
      }
      const int ab = i & 1, row = m0 + r;
      const bool shared = MODE == STORE_PACKED && (m0 < row_lo || m0 + GM > row_hi);
      bool real = row >= row_lo && row < row_hi;
      if (real && p.mask_rows && !p.packed) {
        const int b = row / g.L, q = row - b * g.L, s = segment_of(g, q);
        real = q - g.off(s) < valid_rows(g, b, s);
      }
      // the bias of this group's columns, by way of shared memory: read from global memory column by column in the loop below
      // it was what bounded the bf16 layers (572 us against 368 without a bias at M 278528, N 1536, K 512)
      const uint32_t my_bias = s_bias + grp * 512;
      if (p.bias != nullptr) {
        const int j = tid & 127, col = n0 + (2 * (j / CW) + grp) * CW + j % CW;
        if (MODE == STORE_PACKED) group_sync();  // in the other modes the last box's barrier has this effect
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(my_bias + 4 * j), "f"(col < p.N ? p.bias[col] : 0.f) : "memory");
        group_sync();
      }
      mbar_wait_warp(wc, bar_accf + 8 * ab, (i >> 1) & 1);
      tc_fence_after();
#pragma unroll 1
      for (int c = grp; c < p.bn / CW && n0 + c * CW < p.N; c += 2) {
        const int col0 = n0 + c * CW, bi = u % p.boxes;
        const uint32_t box = s_box + (grp * p.boxes + bi) * BOX + r * 128;
        uint32_t v[CW];
#pragma unroll
        for (int h = 0; h < CW / 32; ++h) tmem_ld32(tl + ab * 256 + c * CW + 32 * h, *reinterpret_cast<uint32_t(*)[32]>(v + 32 * h));
        tmem_wait_ld(*reinterpret_cast<uint32_t(*)[32]>(v), *reinterpret_cast<uint32_t(*)[32]>(v + CW - 32));
        if (c + 2 >= p.bn / CW || col0 + 2 * CW >= p.N) {  // this warp has read its last column of the accumulator
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if constexpr (PAIR) arrive_remote(in_first_cta(bar_acce + 8 * ab));
            else mbar_arrive(bar_acce + 8 * ab);
          }
        }
        if (p.bias != nullptr) {
#pragma unroll
          for (int e = 0; e < CW; e += 4) {
            float4 b4;
            asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                         : "=f"(b4.x), "=f"(b4.y), "=f"(b4.z), "=f"(b4.w) : "r"(my_bias + 4 * ((c >> 1) * CW + e)) : "memory");
            v[e] = __float_as_uint(__uint_as_float(v[e]) + b4.x);
            v[e + 1] = __float_as_uint(__uint_as_float(v[e + 1]) + b4.y);
            v[e + 2] = __float_as_uint(__uint_as_float(v[e + 2]) + b4.z);
            v[e + 3] = __float_as_uint(__uint_as_float(v[e + 3]) + b4.w);
          }
        }
        if (p.relu) {
#pragma unroll
          for (int e = 0; e < CW; ++e) v[e] = __float_as_uint(fmaxf(__uint_as_float(v[e]), 0.f));
        }
        if (shared) {
          if (real) {
            __nv_bfloat16* dst = p.C + (int64_t)row * p.ldc + col0;
#pragma unroll
            for (int e = 0; e < CW; e += 8)
              if (col0 + e < p.N)
                *reinterpret_cast<uint4*>(dst + e) =
                    make_uint4(pack_bf16(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), pack_bf16(__uint_as_float(v[e + 2]), __uint_as_float(v[e + 3])),
                               pack_bf16(__uint_as_float(v[e + 4]), __uint_as_float(v[e + 5])), pack_bf16(__uint_as_float(v[e + 6]), __uint_as_float(v[e + 7])));
          }
          continue;  // no box was used: u stands
        }
        if (res) mbar_wait_warp(wc, bar_resf + 8 * (grp * MAX_BOXES + bi), (u / p.boxes) & 1);
        else group_sync();  // the leader has seen to it that this box's previous store has been read
#pragma unroll
        for (int q = 0; q < 8; ++q) {  // 16-byte pieces of the row, swizzled with the row
          const uint32_t at = box + ((q ^ (r & 7)) << 4);
          uint32_t o[4];
          if constexpr (MODE == STORE_F32) {
            float f[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) f[e] = __uint_as_float(v[4 * q + e]);
            if (res) {
              float4 x;
              asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(at) : "memory");
              f[0] += x.x; f[1] += x.y; f[2] += x.z; f[3] += x.w;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = real ? __float_as_uint(f[e]) : 0u;
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              o[e] = real ? pack_bf16(__uint_as_float(v[8 * q + 2 * e]), __uint_as_float(v[8 * q + 2 * e + 1])) : 0u;
          }
          st_shared_v4(at, o[0], o[1], o[2], o[3]);
        }
        fence_async_smem();
        group_sync();
        if (leader) {
          tma_store_2d(&tmC, s_box + (grp * p.boxes + bi) * BOX, col0, m0);
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          if (res) {  // the box before this one has been read: the loader may refill it
            asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            if (u > 0) mbar_arrive(bar_rese + 8 * (grp * MAX_BOXES + (u - 1) % p.boxes));
          } else {    // two boxes: the one before this one is the next to be written
            asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
          }
        }
        ++u;
      }
      // a group that had no box in this tile (one box of columns in all) still owes its arrivals
      if (n0 + grp * CW >= p.N || grp >= p.bn / CW) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if constexpr (PAIR) arrive_remote(in_first_cta(bar_acce + 8 * ab));
          else mbar_arrive(bar_acce + 8 * ab);
        }
      }
      ++i;
    }
    if (leader) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");  // outstanding TMA stores of this group
  }

  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();  // nobody leaves while the other CTA's instructions may still touch its memory
  if (warp == 1) {
    tc_fence_after();
    if constexpr (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
    else tmem_dealloc(tmem, 512);
  }
}

// Float tensor map: boxes of 32 columns x 128 rows, 128-byte swizzle.
bool make_map_f32(CUtensorMap* tm, const void* base, int64_t rows, int cols, int64_t row_stride) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (fn == nullptr) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows}, strides[1] = {(cuuint64_t)row_stride * 4};
  const cuuint32_t box[2] = {32, GM}, estr[2] = {1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool PAIR, int MODE>
cudaError_t launch(const CUtensorMap& tmA, const CUtensorMap& tmW, const CUtensorMap& tmC, const CUtensorMap& tmR, const Geometry& g,
                   const GemmParams& p, unsigned ctas, int smem, cudaStream_t st) {
  auto kernel = linear_tc_kernel<PAIR, MODE>;
  cudaError_t e = sm_count_and_smem_once(reinterpret_cast<const void*>(kernel), 227 * 1024, nullptr);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(G_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = PAIR ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, tmA, tmW, tmC, tmR, g, p);
}

}  // namespace

// Shapes the tensor-core path covers; everything else stays on the mma.sync kernel.
bool linear_tc_supported(const LinearArgs& a) {
  return a.K >= GK && a.K % GK == 0 && a.N >= 16 && a.N % 8 == 0 && a.lda % 8 == 0 && a.M >= 1 && (a.out_f32 || a.residual == nullptr) &&
         (a.out_f32 ? a.ldc % 4 == 0 : a.ldc % 8 == 0) && (a.residual == nullptr || a.ldr % 4 == 0) &&
         ((reinterpret_cast<uintptr_t>(a.C) | reinterpret_cast<uintptr_t>(a.residual)) & 15u) == 0;
}

cudaError_t launch_linear_tc_bf16(const Geometry& g, const LinearArgs& a, cudaStream_t st) {
  if (!linear_tc_supported(a)) return cudaErrorNotSupported;
  int n_sm = 0;
  cudaError_t e = sm_count_and_smem_once(nullptr, 0, &n_sm);
  if (e != cudaSuccess) return e;
  GemmParams p = {};
  p.M = a.M; p.N = a.N; p.K = a.K;
  p.packed = (g.row_start != nullptr) ? 1 : 0;
  if (p.packed && a.out_f32) return cudaErrorNotSupported;
  // Pairs of CTAs when every pair gets at least two tiles of 256 rows x bn columns; otherwise one CTA per tile of 128 rows, and
  // columns narrow enough (256, 128, 64) that as many SMs as possible have a tile.
  auto width = [&](int most) {  // columns per tile: equal parts of N, in whole boxes
    const int nt = (a.N + most - 1) / most;
    return (((a.N + nt - 1) / nt) + 63) & ~63;
  };
  auto tiles = [&](int rows, int bn) { return (int64_t)((a.M + rows - 1) / rows) * ((a.N + bn - 1) / bn); };
  p.bn = width(256);
  const bool pair = tiles(2 * GM, p.bn) >= n_sm;
  if (!pair)
    for (int most = 128; most >= 64 && tiles(GM, p.bn) < n_sm; most >>= 1) p.bn = width(most);
  const int ctas = pair ? 2 : 1;
  p.tiles_n = (a.N + p.bn - 1) / p.bn;
  const int64_t n_tiles = tiles(GM * ctas, p.bn);
  if (n_tiles > 0x7fffffffLL) return cudaErrorNotSupported;
  p.n_tiles = (int)n_tiles;
  p.stage_bytes = A_STAGE + p.bn / ctas * GK * 2;
  p.bias = a.bias;
  p.has_residual = a.residual != nullptr;
  p.C = static_cast<__nv_bfloat16*>(a.C); p.ldc = a.ldc;
  p.relu = a.relu; p.mask_rows = a.mask_rows;
  const int mode = p.packed ? STORE_PACKED : a.out_f32 ? STORE_F32 : STORE_BF16;
  p.boxes = p.has_residual ? 3 : 2;
  const int box_bytes = 2 * p.boxes * BOX;
  p.stages = (227 * 1024 - 1024 - G_BAR_BYTES - box_bytes) / p.stage_bytes;
  if (p.stages > G_MAX_STAGES) p.stages = G_MAX_STAGES;
  if (p.stages < 2) return cudaErrorNotSupported;
  int smem = p.stages * p.stage_bytes + box_bytes + G_BAR_BYTES + 1024;
  if (smem < G_MIN_SMEM) smem = G_MIN_SMEM;
  alignas(64) CUtensorMap tmA, tmW, tmC, tmR;
  if (!make_map(&tmA, a.A, a.M, a.K, a.lda, GK, GM) || !make_map(&tmW, a.W, a.N, a.K, a.K, GK, p.bn / ctas)) return cudaErrorInvalidValue;
  tmC = tmR = tmA;  // placeholders where the mode has no such map
  if (mode != STORE_F32 && !make_map(&tmC, a.C, a.M, a.N, a.ldc, 64, GM)) return cudaErrorInvalidValue;
  if (mode == STORE_F32 && !make_map_f32(&tmC, a.C, a.M, a.N, a.ldc)) return cudaErrorInvalidValue;
  if (p.has_residual && !make_map_f32(&tmR, a.residual, a.M, a.N, a.ldr)) return cudaErrorInvalidValue;
  const int64_t want = n_tiles * ctas;
  const unsigned grid = (unsigned)(want < n_sm ? want : pair ? n_sm & ~1 : n_sm);
  if (mode == STORE_PACKED)
    return pair ? launch<true, STORE_PACKED>(tmA, tmW, tmC, tmR, g, p, grid, smem, st) : launch<false, STORE_PACKED>(tmA, tmW, tmC, tmR, g, p, grid, smem, st);
  if (mode == STORE_F32)
    return pair ? launch<true, STORE_F32>(tmA, tmW, tmC, tmR, g, p, grid, smem, st) : launch<false, STORE_F32>(tmA, tmW, tmC, tmR, g, p, grid, smem, st);
  return pair ? launch<true, STORE_BF16>(tmA, tmW, tmC, tmR, g, p, grid, smem, st) : launch<false, STORE_BF16>(tmA, tmW, tmC, tmR, g, p, grid, smem, st);
}

}  // namespace gsit
