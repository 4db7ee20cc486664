// The networks' last hidden layer, their output and the way back through that layer in
// one kernel on the 5th-generation tensor cores (paper Eq. 2 and its derivative):
//   L3  z3 = h2 W3^T + b3,  E_row += CELU(z3) . w4,  delta3 = w4 CELU'(z3)
//   B3  delta2 = (delta3 W3) CELU'(z2)      (CELU'(z2) from h2; written over h2)
// for a 128-row tile of one species segment and one ensemble member.  As two layer GEMMs
// (mlp_tc.cu) h2 is read twice and delta3 written and read: 1.9 times the traffic.  Here
// delta3 never leaves the SM, and h2 is read once and replaced in place:
//   - h2 arrives by TMA in 64-column blocks (128-byte swizzle, both parts on the split
//     path), is L3's A operand, then B3's epilogue replaces each element by delta2 where
//     it stands, and the same tensor map stores the block.
//   - delta3 is written over z3 in tensor memory as packed BF16 pairs (high parts, then
//     low parts: the same number of columns), which is B3's A operand.
// Tensor memory (512 columns): two z3 / delta3 accumulators, so that L3 of the next tile
// runs beside this tile's epilogues, and one for delta2.
// Roles (one CTA per SM, persistent over the (member, row tile) list):
//   warps 0-15    epilogues: warp w has the rows 32 (w % 4).. and the 16-column group
//                 w / 4 of every 64-column block (16 warps: the chain of conversions of
//                 an element needs four warps per scheduler to cover it)
//   warp 16       producer of the weights: 32-wide K slices (64-byte swizzle), the high
//                 and low parts as stages of their own, through a ring.  A stage is one
//                 untiled bulk copy of an image laid out at load time
//   warp 17       MMA issuer
//   warp 18       the h2 blocks: loads, and once the epilogue has replaced a block its
//                 store and then the load of the block that takes its place
// The blocks' slots and the ring share the shared memory.  Three tiles' slots let L3 of
// the next tile go before this tile's B3 and its epilogue run beside it (BF16); with
// fewer (split operands at 192 and 160 columns: five slots of 32 KB and five stages of
// 12 KB) it goes behind, beside B3's epilogue.
// L3 and B3, two layer GEMMs -> this kernel: 100k solvated atoms, 8 networks, 41 tiles per
// SM 499 -> 357 us (h2 in two parts read and replaced, 1.23 GB: 181 us at least); 20k atoms BF16 87 -> 44 us; one tile (24
// atoms) 13 -> 10.7 us.  Bound by the chain of a tile: B3 4.3 k cycles, the last block's
// store, load and share of L3 7.1 k (beside B3's epilogue, 4.8 k), L3's epilogue 3.1 k.
// Every wait is bounded; a CTA that gives up records a timeout in the status word,
// drains what it issued, frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "../../include/nnp.h"
#include "mlp.cuh"
#include "tc_util.cuh"

namespace nnp {

namespace {

using namespace tcu;

constexpr int kHBK = 32;                       // K slice of a weight stage (64-byte swizzle)
constexpr int kHEpiWarps = kHeadParts * 4;
constexpr int kHWtWarp = kHEpiWarps, kHMmaWarp = kHEpiWarps + 1, kHIoWarp = kHEpiWarps + 2;
constexpr int kHThreads = (kHEpiWarps + 3) * 32;
constexpr int kHMaxStages = 8;
constexpr int kHMaxBlocks = 4;                 // 64-column blocks of h2
constexpr int kHMaxSlots = 3 * kHMaxBlocks;
constexpr int kHChunks3 = 3;                   // 64-column spans of z3 an epilogue warp keeps in registers
constexpr int kHPlane = 128 * 128;             // bytes of one part of a 128 x 64 block
constexpr int kHMaxDynSmem = 232448 - 2048;    // 227 KB per block minus static shared memory

struct HeadArgs {
  int h2, h3, E, S;
  int zc;                                      // tensor-memory columns of a z3 accumulator
  const float* b3; const float* w4;            // [E][S][h3]
  const uint8_t* w3; const uint8_t* w3t;       // packed weights (MlpWeights::W3_img, W3T_img)
  float* e_row; int e_row_net;                 // [parts][E][rows]
  float alpha;
  const int* seg_start;
  int* status;
  int n_blk, n_slot, ahead;                    // ahead: the next tile's L3 goes before this tile's B3
  int stages, stage_bytes;
};

// D[tmem] (+)= A[tmem] B[smem]
__device__ __forceinline__ void umma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                             uint32_t accumulate, uint32_t leader) {
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader)
      : "memory");
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2)
               : "memory");
}

// a box towards the L2 cache
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global [%0, {%1, %2, %3}];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(c0), "r"(c1), "r"(c2)
               : "memory");
}

// a pair of values as BF16 pairs: the high parts, and what they leave
template <bool SPLIT>
__device__ __forceinline__ uint32_t split_pair(float2 v, uint32_t* lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
  const uint32_t hw = *reinterpret_cast<const uint32_t*>(&h);
  if (SPLIT) {
    const float2 r = __ffma2_rn(bf2(hw), make_float2(-1.f, -1.f), v);
    const __nv_bfloat162 l = __floats2bfloat162_rn(r.x, r.y);
    *lo = *reinterpret_cast<const uint32_t*>(&l);
  }
  return hw;
}

template <bool SPLIT>
__global__ void __launch_bounds__(kHThreads, 1)
k_head_tc(const __grid_constant__ CUtensorMap mH, const __grid_constant__ CUtensorMap mHl, HeadArgs g) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kHMaxStages], empty_bar[kHMaxStages];   // weight ring
  __shared__ __align__(8) uint64_t h_full[kHMaxSlots], h_done[kHMaxSlots];          // h2 block: arrived / replaced
  __shared__ __align__(8) uint64_t z_full[2], d3_full[2], d_full, d_empty, z_read[4], done_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  constexpr int kParts = SPLIT ? 2 : 1;
  constexpr int kSlot = kParts * kHPlane;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* ring = smem + (size_t)g.n_slot * kSlot;
  volatile int* abort_flag = &abort_sh;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kHMaxStages; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], 1);
    }
    for (int i = 0; i < kHMaxSlots; ++i) {
      mbar_init(&h_full[i], 1);
      mbar_init(&h_done[i], kHEpiWarps);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&z_full[i], 1);
      mbar_init(&d3_full[i], kHEpiWarps);
    }
    for (int i = 0; i < 4; ++i) mbar_init(&z_read[i], kHeadParts);
    mbar_init(&d_full, 1);
    mbar_init(&d_empty, kHEpiWarps);
    mbar_init(&done_bar, 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base_sh)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  const uint32_t t_d = tmem + (uint32_t)(2 * g.zc);   // delta2's accumulator (z3's: at 0 and zc)
  const int row_tiles = g.seg_start[g.S] / kTileM;
  const int T = row_tiles * g.E;
  const int n_sl3 = (g.h3 + kHBK - 1) / kHBK;          // K slices of B3
  const int n_mine = blockIdx.x < T ? (T - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;   // tiles of this CTA
  auto tile = [&](int i) {
    return tile_of((int)blockIdx.x + i * (int)gridDim.x, 1, row_tiles, g.E, 0, g.seg_start, g.S);
  };
  // the order of the layers, the same for the weights, the MMAs and the epilogues: L3 of
  // a tile, with `ahead` of the next one too, and B3 of the tile.  l3(i), b3(i): false
  // ends the walk
  auto walk = [&](auto&& l3, auto&& b3) {
    int n3 = 0, nb = 0;   // tiles whose L3, B3 came
    while (nb < n_mine) {
      if (n3 < n_mine && n3 <= nb + g.ahead) {
        if (!l3(n3++)) return;
      } else {
        if (!b3(nb++)) return;
      }
    }
  };

  if (warp == kHWtWarp) {
    if (lane == 0) {
      // ---- weights
      int it = 0;   // copies issued
      Ring rg(g.stages);
      auto slices = [&](const uint8_t* img, int i, int n_sl, int N) {
        const Tile tl = tile(i);
        const unsigned bytes = (unsigned)(N * kHBK * 2);
        const uint8_t* src = img + (size_t)(tl.e * g.S + tl.s) * (size_t)(n_sl * kParts) * bytes;
        for (int k = 0; k < n_sl * kParts; ++k, ++it, rg.next()) {
          if (it >= g.stages && !mbar_wait(&empty_bar[rg.i], rg.phase ^ 1u, abort_flag)) return false;
          mbar_expect_tx(&full_bar[rg.i], bytes);
          bulk_load(ring + rg.i * g.stage_bytes, src + (size_t)k * bytes, bytes, &full_bar[rg.i]);
        }
        return true;
      };
      walk([&](int i) { return slices(g.w3, i, (g.h2 + kHBK - 1) / kHBK, g.h3); },
           [&](int i) { return slices(g.w3t, i, n_sl3, g.h2); });
      // every issued copy has landed before the CTA may exit
      if (*abort_flag)
        for (int k = max(0, it - g.stages); k < it; ++k) mbar_drain(&full_bar[k % g.stages], (k / g.stages) & 1);
    }
  } else if (warp == kHIoWarp) {
    if (lane == 0) {
      // ---- h2 blocks, numbered through the CTA's tiles; block k in slot k % n_slot
      const int n_all = n_mine * g.n_blk;
      // (a load waits for a slot; the block one tile on is sent for to the L2 cache, so
      // that its turn does not take a round trip to memory: 366 -> 357 us at 100k atoms)
      auto load = [&](int k) {
        const Tile tl = tile(k / g.n_blk);
        const int s = k % g.n_slot, b = k % g.n_blk;
        uint8_t* d = smem + (size_t)s * kSlot;
        mbar_expect_tx(&h_full[s], (unsigned)kSlot);
        tma_load_3d(d, &mH, &h_full[s], b * 64, tl.e, tl.m0);
        if (SPLIT) tma_load_3d(d + kHPlane, &mHl, &h_full[s], b * 64, tl.e, tl.m0);
        if (k + g.n_blk < n_all && k + g.n_blk >= g.n_slot) {
          const Tile nx = tile(k / g.n_blk + 1);
          tma_prefetch_3d(&mH, b * 64, nx.e, nx.m0);
          if (SPLIT) tma_prefetch_3d(&mHl, b * 64, nx.e, nx.m0);
        }
      };
      int issued = 0;
      for (; issued < min(n_all, g.n_slot); ++issued) load(issued);
      for (int k = 0; k < n_all; ++k) {
        const int s = k % g.n_slot;
        if (!mbar_wait(&h_done[s], (k / g.n_slot) & 1, abort_flag)) break;
        const Tile tl = tile(k / g.n_blk);
        const uint8_t* d = smem + (size_t)s * kSlot;
        tma_store_3d(&mH, d, (k % g.n_blk) * 64, tl.e, tl.m0);
        if (SPLIT) tma_store_3d(&mHl, d + kHPlane, (k % g.n_blk) * 64, tl.e, tl.m0);
        bulk_commit();
        if (issued < n_all) {
          bulk_wait_read<0>();
          load(issued++);
        }
      }
      bulk_wait_all();   // every store has completed
      if (*abort_flag)
        for (int k = max(0, issued - g.n_slot); k < issued; ++k) mbar_drain(&h_full[k % g.n_slot], (k / g.n_slot) & 1);
    }
  } else if (warp == kHMmaWarp) {
    {
      // ---- MMA issuer (the whole warp walks; lane 0 issues)
      const uint32_t leader = lane == 0;
      Ring rg(g.stages), hs(g.n_slot);   // weight stages; h2 blocks' slots
      auto idesc_of = [](int N) {
        return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
      };
      const uint32_t idesc3 = idesc_of(g.h3), idesc2 = idesc_of(g.h2);
      const uint32_t ring_u = smem_u32(ring), slots_u = smem_u32(smem);
      // the next weight stage, and its release once the MMAs issued so far are done
      auto stage = [&](uint32_t* addr) {
        if (!mbar_wait_warp(&full_bar[rg.i], rg.phase, abort_flag)) return false;
        tc_fence_after();
        *addr = ring_u + (uint32_t)(rg.i * g.stage_bytes);
        return true;
      };
      auto release = [&] { umma_commit_w(&empty_bar[rg.i], leader); rg.next(); };
      walk(
          [&](int i) {
            // its accumulator held delta3 of tile i - 2: that B3 is complete (the last one
            // issued; waiting for an older phase of the barrier could miss it)
            if (i >= 2 && !mbar_wait_warp(&d_full, (i - 1 - g.ahead) & 1, abort_flag)) return false;
            const uint32_t d = tmem + (uint32_t)((i & 1) * g.zc);
            for (int b = 0; b < g.n_blk; ++b, hs.next()) {
              if (!mbar_wait_warp(&h_full[hs.i], hs.phase, abort_flag)) return false;
              const uint64_t ad = sw128_desc(slots_u + (uint32_t)(hs.i * kSlot));
              const uint64_t adl = SPLIT ? sw128_desc(slots_u + (uint32_t)(hs.i * kSlot + kHPlane)) : 0;
              for (int sl = 0; sl < 2 && b * 64 + sl * kHBK < g.h2; ++sl)
#pragma unroll
                for (int part = 0; part < kParts; ++part) {
                  uint32_t w;
                  if (!stage(&w)) return false;
                  const uint64_t bd = sw64_desc(w);
#pragma unroll
                  for (int j = 0; j < kHBK / 16; ++j) {
                    const int kk = 2 * sl + j;   // 16-wide step of the block
                    if (b * 64 + kk * 16 >= g.h2) break;
                    umma_bf16_w(d, ad + (uint64_t)(kk * 2), bd + (uint64_t)(j * 2), idesc3, (part || b || kk) ? 1u : 0u, leader);
                    if (SPLIT && part == 0) umma_bf16_w(d, adl + (uint64_t)(kk * 2), bd + (uint64_t)(j * 2), idesc3, 1u, leader);
                  }
                  release();
                }
            }
            umma_commit_w(&z_full[i & 1], leader);
            return true;
          },
          [&](int i) {
            if (!mbar_wait_warp(&d3_full[i & 1], (i >> 1) & 1, abort_flag)) return false;
            if (i >= 1 && !mbar_wait_warp(&d_empty, (i - 1) & 1, abort_flag)) return false;
            tc_fence_after();
            const uint32_t a = tmem + (uint32_t)((i & 1) * g.zc), al = a + (uint32_t)(g.zc / 2);
            for (int sl = 0; sl < n_sl3; ++sl)
#pragma unroll
              for (int part = 0; part < kParts; ++part) {
                uint32_t w;
                if (!stage(&w)) return false;
                const uint64_t bd = sw64_desc(w);
#pragma unroll
                for (int j = 0; j < kHBK / 16; ++j) {
                  const int kk = 2 * sl + j;
                  if (kk * 16 >= g.h3) break;
                  umma_bf16_ta(t_d, a + (uint32_t)(kk * 8), bd + (uint64_t)(j * 2), idesc2, (part || kk) ? 1u : 0u, leader);
                  if (SPLIT && part == 0) umma_bf16_ta(t_d, al + (uint32_t)(kk * 8), bd + (uint64_t)(j * 2), idesc2, 1u, leader);
                }
                release();
              }
            umma_commit_w(&d_full, leader);
            return true;
          });
      umma_commit_w(&done_bar, leader);   // arrives when every MMA issued above has completed
      mbar_drain(&done_bar, 0);
    }
  } else {
    // ---- epilogues
    const int q = warp & 3, cg = warp >> 2;
    const int r = q * 32 + lane;
    const uint32_t lanes = (uint32_t)(q * 32) << 16;
    const float alpha = g.alpha, inv_alpha = 1.f / g.alpha;
    const float ez_scale = 1.4426950408889634f / g.alpha;   // exp(z / alpha) = 2^(z ez_scale)
    // L3: energies, delta3 over z3
    auto epi_l3 = [&](int i) {
      const Tile tl = tile(i);
      const int m = tl.m0 + r;
      const bool row_ok = NNP_IN_BOUNDS(g.status, kSiteGemmRow, m, g.seg_start[g.S]);
      const size_t es = ((size_t)tl.e * g.S + tl.s) * g.h3;
      if (!mbar_wait_warp(&z_full[i & 1], (i >> 1) & 1, abort_flag)) return false;
      tc_fence_after();
      const uint32_t tz = tmem + lanes + (uint32_t)((i & 1) * g.zc);
      uint32_t hi[kHChunks3][8], lo[SPLIT ? kHChunks3 : 1][8];
      float2 dot2 = make_float2(0.f, 0.f);   // sums over even and odd columns
#pragma unroll
      for (int ci = 0; ci < kHChunks3; ++ci) {
        const int c0 = 64 * ci + 16 * cg;
        if (c0 >= g.h3) break;
        const float4* bp = reinterpret_cast<const float4*>(g.b3 + es + c0);
        const float4* wp = reinterpret_cast<const float4*>(g.w4 + es + c0);
        float v[16];
        tmem_ld16(tz + (uint32_t)c0, v);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 b4 = __ldg(bp + k), w4 = __ldg(wp + k);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int p = 2 * k + u;
            const float2 w2 = u ? make_float2(w4.z, w4.w) : make_float2(w4.x, w4.y);
            const float2 z = __fadd2_rn(make_float2(v[2 * p], v[2 * p + 1]),
                                        u ? make_float2(b4.z, b4.w) : make_float2(b4.x, b4.y));
            float2 ez;
            dot2 = __ffma2_rn(celu2<SPLIT>(z, alpha, inv_alpha, ez_scale, ez), w2, dot2);
            float2 d3 = __fmul2_rn(w2, make_float2(z.x > 0.f ? 1.f : ez.x, z.y > 0.f ? 1.f : ez.y));
            if (!row_ok) d3 = make_float2(0.f, 0.f);   // bounds-checked build only
            hi[ci][p] = split_pair<SPLIT>(d3, &lo[SPLIT ? ci : 0][p]);
          }
        }
      }
      if (row_ok) g.e_row[(size_t)(cg * g.E + tl.e) * g.e_row_net + m] = dot2.x + dot2.y;
      // delta3 goes over columns that the other warps of these rows read: all have
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&z_read[q]);
      if (!mbar_wait_warp(&z_read[q], i & 1, abort_flag)) return false;
      tc_fence_after();
#pragma unroll
      for (int ci = 0; ci < kHChunks3; ++ci) {
        const int c0 = 64 * ci + 16 * cg;
        if (c0 >= g.h3) break;
        tmem_st8(tz + (uint32_t)(c0 / 2), hi[ci]);
        if (SPLIT) tmem_st8(tz + (uint32_t)((g.zc + c0) / 2), lo[SPLIT ? ci : 0]);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&d3_full[i & 1]);
      return true;
    };
    // B3: delta2 over h2
    Ring hs(g.n_slot);
    auto epi_b3 = [&](int i) {
      if (!mbar_wait_warp(&d_full, i & 1, abort_flag)) return false;
      tc_fence_after();
      for (int b = 0; b < g.n_blk; ++b, hs.next()) {
        const int s = hs.i;
        const int c0 = 64 * b + 16 * cg;
        if (c0 < g.h2) {
          float v[16];
          tmem_ld16(t_d + lanes + (uint32_t)c0, v);
          if (!mbar_wait_warp(&h_full[s], hs.phase, abort_flag)) return false;
          // the row's 32 bytes of each part: 16-byte pieces 2 cg and 2 cg + 1, swizzled
          uint8_t* row = smem + (size_t)s * kSlot + r * 128;
          uint4* p0 = reinterpret_cast<uint4*>(row + (((2 * cg) ^ (r & 7)) << 4));
          uint4* p1 = reinterpret_cast<uint4*>(row + (((2 * cg + 1) ^ (r & 7)) << 4));
          uint32_t w[8], wl[8];
          *reinterpret_cast<uint4*>(w) = *p0;
          *reinterpret_cast<uint4*>(w + 4) = *p1;
          if (SPLIT) {
            *reinterpret_cast<uint4*>(wl) = p0[kHPlane / 16];
            *reinterpret_cast<uint4*>(wl + 4) = p1[kHPlane / 16];
          }
#pragma unroll
          for (int p = 0; p < 8; ++p) {
            float2 a = bf2(w[p]);
            if (SPLIT) a = __fadd2_rn(a, bf2(wl[p]));
            const float2 d = __ffma2_rn(a, make_float2(inv_alpha, inv_alpha), make_float2(1.f, 1.f));
            const float2 x = __fmul2_rn(make_float2(v[2 * p], v[2 * p + 1]),
                                        make_float2(a.x > 0.f ? 1.f : d.x, a.y > 0.f ? 1.f : d.y));
            w[p] = split_pair<SPLIT>(x, &wl[p]);
          }
          *p0 = *reinterpret_cast<const uint4*>(w);
          *p1 = *reinterpret_cast<const uint4*>(w + 4);
          if (SPLIT) {
            p0[kHPlane / 16] = *reinterpret_cast<const uint4*>(wl);
            p1[kHPlane / 16] = *reinterpret_cast<const uint4*>(wl + 4);
          }
          fence_async_smem();   // for the store
        }
        if (b == g.n_blk - 1) tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (b == g.n_blk - 1) mbar_arrive(&d_empty);
          mbar_arrive(&h_done[s]);
        }
      }
      return true;
    };
    walk(epi_l3, epi_b3);
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) atomicOr(g.status, kStTimeout);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

struct HeadPlan {
  CUtensorMap mH, mHl;
  HeadArgs a;
  dim3 grid;
  size_t smem;
  bool split;
};

}  // namespace

// Tensor maps and the shared-memory split for a work arena.  Null (and the two layer
// GEMMs are used) where the widths do not fit: multiples of 16, z3 in at most three
// 64-column spans, two z3 and one delta2 accumulator in 512 columns, and one tile's h2
// beside a ring of two stages.
void* head_prepare(const MlpDims& md, const MlpWeights& mw, const MlpBufs& mb, int row_cap, bool split) {
  const int h2 = md.h2, h3 = md.h3, E = md.E, S = md.S, zc = (h3 + 31) / 32 * 32;
  if (!encode_fn() || !mw.W3_img || !mw.W3T_img || !mb.H2 || (split && !mb.H2l)) return nullptr;
  if (h2 % 16 || h3 % 16 || h2 < 16 || h3 < 16 || h2 > 64 * kHMaxBlocks || h3 > 64 * kHChunks3 || 2 * zc + h2 > 512)
    return nullptr;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return nullptr;
  const int parts = split ? 2 : 1, n_blk = (h2 + 63) / 64;
  const long long room = kHMaxDynSmem - 1024, slot = (long long)parts * kHPlane;
  const int stage = std::max(h2, h3) * kHBK * 2;
  auto stages_for = [&](int slots) {
    return room < slots * slot ? 0 : (int)std::min<long long>(kHMaxStages, (room - slots * slot) / stage);
  };
  // as many slots as leave the ring five stages
  int slots = 3 * n_blk;
  while (slots > n_blk && stages_for(slots) < 5) --slots;
  if (stages_for(slots) < 2) return nullptr;
  HeadPlan* p = new HeadPlan{};
  p->split = split;
  const uint64_t R = (uint64_t)row_cap;
  auto hmap = [&](CUtensorMap* m, const void* base) {   // dims (h2, E, rows), box (64, 1, 128)
    return make_map(m, base, h2, E, R, h2, (uint64_t)E * h2, 1, kTileM);
  };
  bool ok = hmap(&p->mH, mb.H2);
  p->mHl = p->mH;
  if (split) ok = ok && hmap(&p->mHl, mb.H2l);
  HeadArgs& a = p->a;
  a.h2 = h2; a.h3 = h3; a.E = E; a.S = S; a.zc = zc;
  a.b3 = mw.b3; a.w4 = mw.w4;
  a.e_row = mb.e_row; a.e_row_net = row_cap;
  a.w3 = static_cast<const uint8_t*>(mw.W3_img);
  a.w3t = static_cast<const uint8_t*>(mw.W3T_img);
  a.n_blk = n_blk; a.n_slot = slots; a.ahead = slots == 3 * n_blk ? 1 : 0;
  a.stages = stages_for(slots); a.stage_bytes = stage;
  // (never so small that a second CTA could share the SM: each takes all tensor memory)
  p->smem = std::max<size_t>((size_t)slots * slot + (size_t)a.stages * stage + 1024, 232448 / 2 + 1);
  const int row_tiles = (row_cap + kTileM - 1) / kTileM;
  p->grid = dim3((unsigned)std::max(1, std::min(row_tiles * E, sms)));
  const void* fn = split ? (const void*)k_head_tc<true> : (const void*)k_head_tc<false>;
  if (!ok || cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kHMaxDynSmem) != cudaSuccess) {
    cudaGetLastError();
    delete p;
    return nullptr;
  }
  return p;
}

void head_release(void* plan) { delete static_cast<HeadPlan*>(plan); }

void launch_head(void* plan, const Ws& ws, float alpha, cudaStream_t st) {
  HeadPlan* p = static_cast<HeadPlan*>(plan);
  HeadArgs a = p->a;
  a.alpha = alpha;
  a.seg_start = ws.seg_start;
  a.status = ws.status;
  if (p->split) k_head_tc<true><<<p->grid, kHThreads, p->smem, st>>>(p->mH, p->mHl, a);
  else k_head_tc<false><<<p->grid, kHThreads, p->smem, st>>>(p->mH, p->mHl, a);
}

}  // namespace nnp
