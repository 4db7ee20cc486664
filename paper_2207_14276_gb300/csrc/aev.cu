// Atomic environment vectors (paper Eqs. 3-5) and their backward to forces.
//
// One warp per centre atom.  The geometry of every neighbour of the centre is
// computed once (lane-parallel) and staged in shared memory: (R, f_c) for the
// radial list, (unit vector, R) and (f_c, f_c') for the angular sub-list.
//
// Forward
//   radial  (Eq. 4): eight lanes per neighbour of one species, four neighbours at a
//           time, a lane owns two Gaussian shells (packed FP32x2); two shuffles add
//           the four and lanes 0..15 write the block's 16 features.
//   angular (Eq. 5): lane-per-triplet.  The (j, k) pairs of one unordered
//           species pair are numbered by a quotient and a remainder; every lane
//           forms the 4 Gaussians of the averaged distance and the 8 angular
//           factors of its pair (two sections per packed FP32x2 instruction)
//           and accumulates all 32 products in registers.
//           A transpose-reduce across the warp (31 shuffles) leaves lane l with
//           feature l = 8a + z of the block: one coalesced 128-byte store.
//   The angular factor uses cos(theta - theta_z) = cos theta cos theta_z +
//   sin theta sin theta_z with sin theta from the cross product (no acos), and
//   (1 + cos(theta - theta_z))^zeta by repeated squaring (integer zeta,
//   specialised at compile time for zeta = 32).
//
// Backward (F = -dE/dr)
//   radial edges: lane-per-neighbour, 16 shells each (two per packed FP32x2
//   instruction).
//   angular: lane-per-pair (j, k) of the centre's angular neighbours, the pairs
//   taken in round-robin order (one round pairs every neighbour at most once).
//   The dE/dG of the species-pair blocks that have pairs is staged in shared
//   memory (feature order, up to 16 blocks).  Each lane contracts its block's
//   32 values to dE/dcos, dE/dRbar and dE/d(f_j f_k), forms dE/du_j and dE/du_k
//   and adds them to per-neighbour accumulators in shared memory: round r into
//   copy r mod (number of copies), so no two lanes of a pass add into the same
//   address.  Afterwards each neighbour receives one vector atomic and the
//   centre one warp-reduced atomic.  Centres with too many angular neighbours
//   or blocks go to a CTA-per-centre kernel.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "aev_device.cuh"
#include "nnp_internal.cuh"
#include "tc_util.cuh"

namespace nnp {

namespace {

constexpr int kWarps = 8;
// dE/dG blocks of a centre held in shared memory by the warp-per-centre backward
// kernel (the blocks with triplets, in block order; a centre with more goes to
// the CTA-per-centre kernel)
constexpr int kGallBlocks = kDenseBlocks;

// float4s of shared memory per warp of the backward kernel: neighbour geometry
// and cutoffs (2 cap_a), `copies` copies of the float4 accumulators (one per
// neighbour each), a region that holds first the radial dE/dG (S * 16 <= 128
// floats) and then up to kGallBlocks angular blocks' dE/dG (9 float4s per block:
// 8 in feature order and one of padding, so that lanes reading float4 i of
// different blocks hit different banks), and the bytes of the neighbours' species and of
// the species-pair -> block-slot table (64)
constexpr int kGallStride = 9;
__host__ __device__ constexpr int aev_bwd_gall_f4(int n_pairs) {
  return kGallStride * (n_pairs < kGallBlocks ? n_pairs : kGallBlocks) > 32
             ? kGallStride * (n_pairs < kGallBlocks ? n_pairs : kGallBlocks)
             : 32;
}
__host__ __device__ constexpr int aev_bwd_warp_f4(int cap_a, int n_pairs, int copies) {
  return 2 * cap_a + copies * cap_a + aev_bwd_gall_f4(n_pairs) + (cap_a + 64 + 15) / 16;
}

// Copies of the per-neighbour angular accumulators.  The triplets are taken in
// round-robin order (rr_pair below): one round pairs every neighbour at most
// once, and the lanes of one 32-triplet pass span at most `copies` consecutive
// rounds, round r adding into copy r mod copies, so no two lanes of a pass add
// into the same accumulator and plain read-add-write is race-free.  4, 2 or 1:
// the most that keep four CTAs on an SM (228 KiB of shared memory per SM, 1 KiB
// reserved per CTA, plus the static list headers).
constexpr int kBwdCtaSmem = 228 * 1024 / 4 - 1024 - kWarps * (int)sizeof(ListHdr);
int aev_bwd_copies(int cap_a, int n_pairs) {
  for (int r = 4; r > 1; r >>= 1)
    if ((size_t)kWarps * aev_bwd_warp_f4(cap_a, n_pairs, r) * sizeof(float4) <= (size_t)kBwdCtaSmem)
      return r;
  return 1;
}

// one AEV element: the FP32 row, or on the tensor-core paths (Gh != null) only
// what their first layer reads: the BF16 row, and on the split path (Gl != null)
// also the low part bf16(v - bf16(v))
__device__ __forceinline__ void put_g(float* G, uint16_t* Gh, uint16_t* Gl, int f, float v) {
  if (Gh) {
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    Gh[f] = __bfloat16_as_ushort(h);
    if (Gl) Gl[f] = __bfloat16_as_ushort(__float2bfloat16_rn(v - __bfloat162float(h)));
  } else {
    G[f] = v;
  }
}

// float4s of per-warp shared memory of the forward: angular unit vectors and R
// (cap_a), angular cutoffs (cap_a floats + 4), radial (R, f_c) pairs (cap_r)
__host__ __device__ constexpr int aev_fwd_warp_f4(int cap_a, int cap_r) {
  return cap_a + cap_a / 4 + cap_r / 2 + 2;
}

// (j, k) of triplet t of a species pair's block, cu the second species' neighbours: j = t /
// cu, k = t % cu, and for one species the pairs around a circle, (t % cu, t % cu + t / cu
// + 1).  The estimate is exact: t / cu < 512, its error below 2e-4, and (t + 0.5) / cu at
// least 0.5 / 512 from a whole number.  (With the row-major triangle, whose row takes a
// square root and two corrections, the forward of 100k solvated atoms took 299 us, 281 so;
// 313 before the radial shells and the angular Gaussians went in packed pairs, too.)
__device__ __forceinline__ void fwd_pair(int t, int same, int cu, float inv_cu, int* j, int* k) {
  const int a = (int)((t + 0.5f) * inv_cu), b = t - a * cu;
  int c = b + a + 1;
  if (c >= cu) c -= cu;
  *j = same ? b : a;
  *k = same ? c : b;
}

// whether a centre's list header makes it a dense one (the same value on every lane)
__device__ __forceinline__ bool hdr_dense(const ListHdr& H, const AevConst& ac, unsigned lane) {
  return is_dense(ac, H.off_a[ac.S], (int)lane < ac.S ? H.off_a[lane + 1] - H.off_a[lane] : 0);
}

// The AEV row of packed atom p (Eqs. 3-5) by W warps (1, or all kWarps of the CTA;
// w: this warp's number among them); out(f, v) stores feature f (each f < Dp exactly
// once, by the lane holding it).  stage: aev_fwd_warp_f4 float4s of shared memory; H:
// the list header.  The warps share the staged neighbours; warp w takes every W-th
// species' radial block and every W-th angular block.  With sparse set, only the blocks
// that touch a live slice of the row (row_slices) are stored, and *mask receives the
// row's slice mask.  With skip_dense set a dense centre is left out (returns false).
template <int ZETA, int W, class Out>
__device__ __forceinline__ bool aev_centre(const Ws& ws, const AevConst& ac, int p, float4* stage,
                                           ListHdr& H, unsigned lane, const uint8_t* pair_su,
                                           Out out, bool sparse = false, uint32_t* mask = nullptr,
                                           int w = 0, bool skip_dense = false) {
  auto sync = [] {
    if (W == 1) __syncwarp();
    else __syncthreads();
  };
  sync();   // the stage and header may still hold the previous centre
  float4* angv = stage;
  float* angf = reinterpret_cast<float*>(angv + ws.cap_a);
  float2* rad = reinterpret_cast<float2*>(angf + ws.cap_a + 4);
  const float4 xi = ws.xyzq[p];
  const SysDev& d = ws.sys[ws.pos_sys[p]];
  {   // the first lines of the neighbour lists travel while the header loads
    const int* a = nullptr;
    if (lane < 2 && (int)lane * 32 < ws.cap_r) a = ws.nb_r + (size_t)p * ws.cap_r + lane * 32;
    else if (lane == 2) a = ws.nb_a + (size_t)p * ws.cap_a;
    if (a) asm volatile("prefetch.global.L1 [%0];" ::"l"(a));
  }
  if (W == 1 || w == 0) load_hdr(ws.nb_cnt + (size_t)p * 16, ac.S, lane, &H);
  if (W > 1) __syncthreads();
  if (skip_dense && hdr_dense(H, ac, lane)) return false;
  const uint32_t m = sparse ? row_slices(H, ac, lane, pair_su) : ~0u;
  if (mask) *mask = m;
  const int* lr = ws.nb_r + (size_t)p * ws.cap_r;
  const int* la = ws.nb_a + (size_t)p * ws.cap_a;
  const float inv_rc_r = 1.f / ac.rc_r, inv_rc_a = 1.f / ac.rc_a;
  stage_list<W>(H.off_r[ac.S], lr, xi, d, ws, w * 32 + lane,
                [&](int slot, int, const Geo& g) {
                  rad[slot] = make_float2(g.r, fcut(g.r, ac.rc_r, inv_rc_r));
                });
  stage_list<W>(H.off_a[ac.S], la, xi, d, ws, w * 32 + lane,
                [&](int slot, int, const Geo& g) {
                  const float inv = rcp_approx(g.r);
                  angv[slot] = make_float4(g.dx * inv, g.dy * inv, g.dz * inv, g.r);
                  angf[slot] = fcut(g.r, ac.rc_a, inv_rc_a);
                });
  sync();
  // ---- radial, Eq. 4: eight lanes per neighbour, two shells per lane (packed FP32x2),
  // four neighbours at a time
  const float cr_ = -ac.eta_r * kLog2e;
  const float2 my_shf = make_float2(ac.shf_r[2 * (lane & 7)], ac.shf_r[2 * (lane & 7) + 1]);
  for (int s = w; s < ac.S; s += W) {
    const int o = H.off_r[s], n = H.off_r[s + 1] - o;
    if (!block_in(m, ac.rcol[s], kNR)) continue;
    float2 acc = make_float2(0.f, 0.f);
    for (int t = (int)lane >> 3; t < n; t += 4) {
      const float2 q = rad[o + t];
      const float2 x = __fadd2_rn(make_float2(q.x, q.x), make_float2(-my_shf.x, -my_shf.y));
      const float2 e = __fmul2_rn(__fmul2_rn(x, x), make_float2(cr_, cr_));
      acc = __ffma2_rn(make_float2(fast_exp2(e.x), fast_exp2(e.y)), make_float2(q.y, q.y), acc);
    }
    // sums over the four neighbour lanes; lanes 0-15 hold the shells in turn
    float v = (lane & 8) ? acc.y : acc.x;
    const float u = (lane & 8) ? acc.x : acc.y;
    v += __shfl_xor_sync(kFull, u, 8);
    v += __shfl_xor_sync(kFull, v, 16);
    if (lane < 16) out(ac.rcol[s] + 2 * (lane & 7) + (lane >> 3), v);
  }
  // ---- angular, Eq. 5: the blocks of species pairs with a pair j < k, and the
  // zero blocks of the other pairs where the row is written
  const float ca_ = -ac.eta_a * kLog2e;
  uint32_t live[2] = {0u, 0u}, zero[2] = {0u, 0u};
  for (int h = 0; h * 32 < ac.n_pairs; ++h) {
    const int q = h * 32 + (int)lane;
    bool lv = false, zr = false;
    if (q < ac.n_pairs) {
      const int sp = pair_su[q] & 15, u = pair_su[q] >> 4;
      const int cs = H.off_a[sp + 1] - H.off_a[sp], cu = H.off_a[u + 1] - H.off_a[u];
      lv = sp == u ? cs >= 2 : (cs > 0 && cu > 0);
      zr = !lv && block_in(m, ac.acol[q], 32);
    }
    live[h] = __ballot_sync(kFull, lv);
    zero[h] = __ballot_sync(kFull, zr);
  }
  if (W == 1 || w == W - 1)
    for (int h = 0; h < 2; ++h)
      for (uint32_t z = zero[h]; z; z &= z - 1)
        out(ac.acol[h * 32 + __ffs(z) - 1] + lane, 0.f);
  int turn = 0;   // live blocks in turn to the warps
  for (int h = 0; h < 2; ++h)
    for (uint32_t lv = live[h]; lv; lv &= lv - 1) {
      if (W > 1 && turn++ % W != w) continue;
      const int q = h * 32 + __ffs(lv) - 1;
      const int s = pair_su[q] & 15, u = pair_su[q] >> 4;
      const int os = H.off_a[s], cs = H.off_a[s + 1] - os;
      const int ou = H.off_a[u], cu = H.off_a[u + 1] - ou;
      const int same = (s == u);
      const int n_tri = same ? cs * (cs - 1) / 2 : cs * cu;
      const int fb = ac.acol[q];
      const float inv_cu = rcp_approx((float)cu);
      // acc2[4a + m] holds features 8a + 2m and 8a + 2m + 1 (packed FP32x2 FMAs)
      float2 acc2[16];
#pragma unroll
      for (int f = 0; f < 16; ++f) acc2[f] = make_float2(0.f, 0.f);
      for (int t0 = 0; t0 < n_tri; t0 += 32) {
        const int t = t0 + lane;
        if (t < n_tri) {
          int j, k;
          fwd_pair(t, same, cu, inv_cu, &j, &k);
          const float4 vj = angv[os + j];
          const float4 vk = angv[ou + k];
          const float fjk = ac.ang_pre * angf[os + j] * angf[ou + k];
          const float chat = vj.x * vk.x + vj.y * vk.y + vj.z * vk.z;
          const float c = ac.cos_scale * chat;
          const float sn = sin_theta(vj, vk, chat, ac.cos_scale);
          const float rb = 0.5f * (vj.w + vk.w);
          float2 A[kNA];
#pragma unroll
          for (int a = 0; a < kNA; a += 2) {
            const float2 x = __fadd2_rn(make_float2(rb, rb), make_float2(-ac.shf_a[a], -ac.shf_a[a + 1]));
            const float2 e = __fmul2_rn(__fmul2_rn(make_float2(ca_, ca_), x), x);
            const float v0 = fast_exp2(e.x) * fjk, v1 = fast_exp2(e.y) * fjk;
            A[a] = make_float2(v0, v0);
            A[a + 1] = make_float2(v1, v1);
          }
          const float2 c2 = make_float2(c, c), s2 = make_float2(sn, sn);
#pragma unroll
          for (int m = 0; m < kNZ / 2; ++m) {
            const float2 B = section_pair<ZETA>(ac, m, c2, s2);
#pragma unroll
            for (int a = 0; a < kNA; ++a) acc2[4 * a + m] = __ffma2_rn(A[a], B, acc2[4 * a + m]);
          }
        }
      }
      float acc[32];
#pragma unroll
      for (int f = 0; f < 16; ++f) {
        acc[2 * f] = acc2[f].x;
        acc[2 * f + 1] = acc2[f].y;
      }
      out(fb + lane, transpose_reduce32(acc, lane));
    }
  if (W == 1 || w == W - 1)
    for (int f = ac.D + lane; f < ac.Dp; f += 32)
      if ((m >> (f >> 6)) & 1u) out(f, 0.f);
  return true;
}

template <int ZETA>
__global__ void __launch_bounds__(kWarps * 32, 4)
k_aev_fwd(Ws ws, AevConst ac, int small) {
  extern __shared__ float4 sm4[];
  __shared__ ListHdr hdrs[kWarps];
  __shared__ uint8_t pair_su[kMaxSpecies * (kMaxSpecies + 1) / 2];
  const int w = threadIdx.x >> 5;
  const unsigned lane = threadIdx.x & 31;
  const bool sparse = ws.row_mask != nullptr;
  // grouped rows: the first row of each (species, slice) group
  __shared__ int group_row0[kMaxSpecies][32];
  if (ws.row_key && w < ac.S) {
    const int c = ws.row_hist[w * 32 + lane];
    int incl = c;
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(kFull, incl, o);
      if ((int)lane >= o) incl += u;
    }
    group_row0[w][lane] = ws.seg_start[w] + incl - c;
  }
  fill_pair_table(pair_su, ac);
  __syncthreads();
  const int n = ws.totals[0];
  // the row of packed atom p (grouped rows: from its group; lane 0 of the first warp
  // tells the later kernels)
  auto row_of = [&](int p, bool tell) {
    if (!ws.row_key) return ws.pos_slot[p];
    const uint32_t k = ws.row_key[p];
    const int slot = group_row0[__float_as_int(ws.xyzq[p].w)][k & 31] + (int)(k >> 5);
    if (tell && NNP_IN_BOUNDS(ws.status, kSiteAevRow, slot, ws.row_cap)) {
      ws.pos_slot[p] = slot;
      ws.slot_pos[slot] = p;
    }
    return slot;
  };
  auto centre = [&](auto warps, int p, int wi, float4* stage, ListHdr& H) {
    constexpr int W = decltype(warps)::value;
    const int slot = row_of(p, lane == 0 && wi == 0);   // (a dense centre's: the same twice)
    if (!NNP_IN_BOUNDS(ws.status, kSiteAevRow, slot, ws.row_cap)) return;
    const size_t row = (size_t)slot * ac.Dp;
    float* G = ws.aev + row;
    uint16_t* Gh = ws.aev_h ? ws.aev_h + row : nullptr;
    uint16_t* Gl = ws.aev_l ? ws.aev_l + row : nullptr;
    uint32_t m = 0;
    const bool done = aev_centre<ZETA, W>(ws, ac, p, stage, H, lane, pair_su,
                                          [&](int f, float v) { put_g(G, Gh, Gl, f, v); }, sparse, &m, wi,
                                          W == 1);
    if (done && sparse && lane == 0 && wi == 0) {
      ws.row_mask[slot] = m;
      atomicOr(ws.tile_mask + (slot >> 7), m);
    }
  };
  // a CTA each for the centres of a small batch and for the dense ones (a warp alone
  // works through their blocks one after the other while the chip idles)
  const bool all = n <= small;
  const int n_cta = all ? n : ws.totals[2];
  for (int h = blockIdx.x; h < n_cta; h += gridDim.x)
    centre(std::integral_constant<int, kWarps>{}, all ? h : ws.heavy[h], w, sm4, hdrs[0]);
  if (all) return;
  __syncthreads();   // the stage and header become the warps' own
  // persistent: every warp takes the next centre from a counter until none is left
  // (dense centres do not hold a CTA's other warps' slots, nor pile up in one warp)
  for (;;) {
    int p = 0;
    if (lane == 0) p = atomicAdd(ws.totals + 4, 1);
    p = __shfl_sync(kFull, p, 0);
    if (p >= n) break;
    centre(std::integral_constant<int, 1>{}, p, 0, sm4 + (size_t)w * aev_fwd_warp_f4(ws.cap_a, ws.cap_r), hdrs[w]);
  }
}

// One warp per AEV row of a species segment: zero the 64-column slices the row's
// tile reads (tile mask) that the row did not write (row mask).  Padding rows
// past a segment's atoms are left alone (their network outputs are never read).
__global__ void __launch_bounds__(256) k_aev_fill(Ws ws, AevConst ac) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5);
  const unsigned lane = threadIdx.x & 31;
  if (r >= ws.seg_start[ac.S]) return;
  int s = 0;
  while (s + 1 < ac.S && r >= ws.seg_start[s + 1]) ++s;
  if (r >= ws.seg_start[s] + ws.species_count[s]) return;
  uint32_t miss = ws.tile_mask[r >> 7] & ~ws.row_mask[r];
  const size_t row = (size_t)r * ac.Dp;
  while (miss) {
    const int k = __ffs(miss) - 1;
    miss &= miss - 1;
    const int f = k * 64 + 2 * (int)lane;      // two columns per lane
    if (f < ac.Dp) {
      if (!ws.aev_h) { *reinterpret_cast<float2*>(ws.aev + row + f) = make_float2(0.f, 0.f); continue; }
      reinterpret_cast<uint32_t*>(ws.aev_h + row + f)[0] = 0u;
      if (ws.aev_l) reinterpret_cast<uint32_t*>(ws.aev_l + row + f)[0] = 0u;
    }
  }
}

// ---- backward pieces shared by the warp-per-centre and CTA-per-centre kernels

// One radial edge (Eq. 4) of centre i: dE/dr_ij from the S*16 radial dE/dG
// values gs of neighbour j's species; the force on j goes to f_pos[j] at once,
// the centre's share (and the virial) into the caller's accumulators.
template <bool VIR>
__device__ __forceinline__ void radial_edge_bwd(const Ws& ws, const AevConst& ac, const float4& xi,
                                                const SysDev& d, int j, const float4& xj,
                                                const float* gs, float inv_rc_r, float* fi,
                                                float* vir, float4* det_slot) {
  const float cr_ = -ac.eta_r * kLog2e;
  const Geo g = pair_geo(xi, xj, d);
  float fc, dfc;
  fcut_both(g.r, ac.rc_r, inv_rc_r, &fc, &dfc);
  // dE/dR = sum_r g_r e_r (-2 eta x_r f_c + f_c') = f_c (-2 eta) sum_r g_r e_r x_r + f_c' sum_r g_r e_r
  // (shells in pairs: packed FP32x2 arithmetic, sums over the even and odd shells)
  const float2 r2 = make_float2(g.r, g.r), cr2 = make_float2(cr_, cr_);
  const float2* shf2 = reinterpret_cast<const float2*>(ac.shf_r);
  const float2* gs2 = reinterpret_cast<const float2*>(gs);   // gs: 8-byte aligned
  float2 sge2 = make_float2(0.f, 0.f), sgex2 = make_float2(0.f, 0.f);
#pragma unroll
  for (int m = 0; m < kNR / 2; ++m) {
    const float2 x = __ffma2_rn(shf2[m], make_float2(-1.f, -1.f), r2);
    const float2 q = __fmul2_rn(__fmul2_rn(x, x), cr2);
    const float2 ge = __fmul2_rn(gs2[m], make_float2(fast_exp2(q.x), fast_exp2(q.y)));
    sge2 = __fadd2_rn(sge2, ge);
    sgex2 = __ffma2_rn(ge, x, sgex2);
  }
  const float sge = sge2.x + sge2.y, sgex = sgex2.x + sgex2.y;
  const float dEdR = fmaf(fc * (-2.f * ac.eta_r), sgex, dfc * sge);
  const float sc = dEdR * rcp_approx(g.r);
  const float gx = sc * g.dx, gy = sc * g.dy, gz = sc * g.dz;
  if (det_slot) *det_slot = make_float4(-gx, -gy, -gz, 0.f);   // deterministic mode
  else atomicAdd(&ws.f_pos[j], make_float4(-gx, -gy, -gz, 0.f));
  fi[0] += gx; fi[1] += gy; fi[2] += gz;
  if (VIR) {
    vir[0] -= g.dx * gx; vir[1] -= g.dx * gy; vir[2] -= g.dx * gz;
    vir[3] -= g.dy * gx; vir[4] -= g.dy * gy; vir[5] -= g.dy * gz;
    vir[6] -= g.dz * gx; vir[7] -= g.dz * gy; vir[8] -= g.dz * gz;
  }
}

// One angular triplet (Eq. 5) of a centre: neighbours j and k (unit vector and
// R; f_c, f_c', 1/R), the 32 dE/dG values of their species-pair block in
// feature order (index 8a + z: float4 2a + h holds sections 4h .. 4h + 3 of
// radial shell a).  Returns dE/d(r_j) and dE/d(r_k) (the force terms on j and
// k; their negatives act on the centre).
template <int ZETA>
__device__ __forceinline__ void triplet_bwd(const AevConst& ac, const float4& vj, const float4& vk,
                                            const float4& fj4, const float4& fk4,
                                            const float4* gblk, float3& uj, float3& uk) {
  const float ca_ = -ac.eta_a * kLog2e;
  const float m2eta = -2.f * ac.eta_a;
  const float chat = vj.x * vk.x + vj.y * vk.y + vj.z * vk.z;
  const float c = ac.cos_scale * chat;
  const float sn = fmaxf(sin_theta(vj, vk, chat, ac.cos_scale), 1e-6f);
  const float m_c_over_s = -c * rcp_approx(sn);
  const float rb = 0.5f * (vj.w + vk.w);
  // contract the block's dE/dG over the 8 angle sections first:
  //   F_a = sum_z g[a][z] B_z,  dF_a = sum_z g[a][z] dB_z/dc,
  // dB_z/dc = zeta base^(zeta-1) (cos(theta_z) - sin(theta_z) c / s) (the factor
  // zeta is applied at the end); sections in pairs, Fp[a] holding the sums over
  // the even and the odd sections
  const float2 c2 = make_float2(c, c), s2 = make_float2(sn, sn);
  const float2 mcs2 = make_float2(m_c_over_s, m_c_over_s);
  float2 Fp[kNA], dFp[kNA];
#pragma unroll
  for (int a = 0; a < kNA; ++a) Fp[a] = dFp[a] = make_float2(0.f, 0.f);
  const float2* g2 = reinterpret_cast<const float2*>(gblk);
#pragma unroll
  for (int m = 0; m < kNZ / 2; ++m) {
    float2 B1;
    const float2 B = section_pair<ZETA>(ac, m, c2, s2, &B1);
    const float2 cz = reinterpret_cast<const float2*>(ac.cos_z)[m];
    const float2 sz = reinterpret_cast<const float2*>(ac.sin_z)[m];
    const float2 dB = __fmul2_rn(B1, __ffma2_rn(sz, mcs2, cz));
#pragma unroll
    for (int a = 0; a < kNA; ++a) {
      const float2 g = g2[4 * a + m];
      Fp[a] = __ffma2_rn(g, B, Fp[a]);
      dFp[a] = __ffma2_rn(g, dB, dFp[a]);
    }
  }
  float F[kNA], dF[kNA];
#pragma unroll
  for (int a = 0; a < kNA; ++a) {
    F[a] = Fp[a].x + Fp[a].y;
    dF[a] = dFp[a].x + dFp[a].y;
  }
  float tc = 0.f, tR = 0.f, tf = 0.f;
#pragma unroll
  for (int a = 0; a < kNA; ++a) {
    const float x = rb - ac.shf_a[a];
    const float A = fast_exp2(ca_ * x * x);
    const float AF = A * F[a];
    tf += AF;
    tR = fmaf(m2eta * x, AF, tR);
    tc = fmaf(A, dF[a], tc);
  }
  const float fjk = fj4.x * fk4.x;
  tc *= ac.ang_pre * (float)ac.zeta * fjk;  // dE/dc, c = cos_scale * cos_hat
  tR *= ac.ang_pre * fjk;                    // dE/dRbar
  tf *= ac.ang_pre;                          // dE/d(f_j f_k)
  const float dEdchat = ac.cos_scale * tc;
  const float sj = dEdchat * fj4.z, sk = dEdchat * fk4.z;
  const float rj = 0.5f * tR + tf * fj4.y * fk4.x;
  const float rk = 0.5f * tR + tf * fj4.x * fk4.y;
  uj = make_float3(sj * (vk.x - chat * vj.x) + rj * vj.x, sj * (vk.y - chat * vj.y) + rj * vj.y,
                   sj * (vk.z - chat * vj.z) + rj * vj.z);
  uk = make_float3(sk * (vj.x - chat * vk.x) + rk * vk.x, sk * (vj.y - chat * vk.y) + rk * vk.y,
                   sk * (vj.z - chat * vk.z) + rk * vk.z);
}

// A warp's virial of the system its last centres belong to, component k on lane k in
// FP64.  Added to the system's virial when the system changes and once per CTA at the
// end: nine FP64 atomics per centre on nine addresses made the backward of 9,000
// water atoms 106 us against 35 without a virial (the whole call 310 us, now 239).
struct VirialSum {
  double* dst = nullptr;
  double sum = 0.0;
  __device__ __forceinline__ void flush(unsigned lane, double* next) {
    if (dst && lane < 9) atomicAdd(dst + lane, sum);
    dst = next;
    sum = 0.0;
  }
};

// Warp per centre, for centres that are not dense (at most cap_l angular neighbours, in
// at most kGallBlocks species-pair blocks, whose dE/dG are all staged at once).
template <int ZETA, bool VIR>
__device__ __forceinline__ void bwd_centre(const Ws& ws, const AevConst& ac, int log_r, int cap_l,
                                           int p, float4* sm4, ListHdr& H, int w, unsigned lane,
                                           VirialSum& vs) {
  __syncwarp();   // the warp's previous centre is done with its shared memory
  const bool det = ws.fr_det != nullptr;   // deterministic mode
  const int n_copy = 1 << log_r;
  float4* angv = sm4 + (size_t)w * aev_bwd_warp_f4(cap_l, ac.n_pairs, n_copy);
  float4* angf = angv + cap_l;             // fc, dfc, 1/R, packed index
  float4* acc = angf + cap_l;              // dE/du per neighbour, [copy][neighbour]
  float4* uni = acc + (size_t)n_copy * cap_l;
  float* grad = reinterpret_cast<float*>(uni);   // S*16 radial dE/dG, then:
  float4* gall = uni;                            // angular dE/dG, [slot][8a + z] (+ pad)
  uint8_t* spec = reinterpret_cast<uint8_t*>(uni + aev_bwd_gall_f4(ac.n_pairs));  // [cap_l]
  uint8_t* pslot = spec + cap_l;           // [8 s + u]: block slot of species pair (s, u)

  const float4 xi = ws.xyzq[p];
  const SysDev& d = ws.sys[ws.pos_sys[p]];
  const float* g_row = ws.dEdG + (size_t)ws.pos_slot[p] * ac.Dp;
  load_hdr(ws.nb_cnt + (size_t)p * 16, ac.S, lane, &H);
  if (hdr_dense(H, ac, lane)) return;   // k_aev_bwd_cta's
  const int n_live = live_blocks((int)lane < ac.S ? H.off_a[lane + 1] - H.off_a[lane] : 0);
  const int* lr = ws.nb_r + (size_t)p * ws.cap_r;
  const int* la = ws.nb_a + (size_t)p * ws.cap_a;
  const float inv_rc_r = 1.f / ac.rc_r, inv_rc_a = 1.f / ac.rc_a;
  // the radial dE/dG (S * 16 <= 128 values) is loaded now and stored after the
  // neighbour gathers, so that the two latencies overlap
  float gr[kMaxSpecies * kNR / 32];
#pragma unroll
  for (int i = 0; i < kMaxSpecies * kNR / 32; ++i) {
    const int f = (int)lane + 32 * i;
    gr[i] = f < ac.S * kNR ? g_row[ac.rcol[f >> 4] + (f & 15)] : 0.f;
  }
  // angular neighbours: unit vector and R, (f_c, f_c', 1/R, packed index), species
  stage_list(H.off_a[ac.S], la, xi, d, ws, lane,
             [&](int slot, int j, const Geo& g) {
               const float inv = rcp_approx(g.r);
               angv[slot] = make_float4(g.dx * inv, g.dy * inv, g.dz * inv, g.r);
               float fc, dfc;
               fcut_both(g.r, ac.rc_a, inv_rc_a, &fc, &dfc);
               angf[slot] = make_float4(fc, dfc, inv, __int_as_float(j));
             });
  const int na_tot = H.off_a[ac.S];
  for (int t = lane; t < na_tot; t += 32) {
    int s = 0;
    while (s + 1 < ac.S && H.off_a[s + 1] <= t) ++s;
    spec[t] = (uint8_t)s;
  }
  for (int c = 0; c < n_copy; ++c)
    for (int t = lane; t < na_tot; t += 32) acc[c * cap_l + t] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int i = 0; i < kMaxSpecies * kNR / 32; ++i) {
    const int f = (int)lane + 32 * i;
    if (f < ac.S * kNR) grad[f] = gr[i];
  }
  __syncwarp();
  float fi[3] = {0.f, 0.f, 0.f};
  float vir[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) vir[k] = 0.f;
  // ---- radial edges, one lane per neighbour, numbered continuously over the
  // species blocks of the list (a lane finds its neighbour's species block);
  // two neighbours per lane and pass, both gathers issued before either is used
  const int nr_tot = H.off_r[ac.S];
  int sr = 0;
  for (int t0 = 0; t0 < nr_tot; t0 += 64) {
    const int ta = t0 + (int)lane, tb = ta + 32;
    int ja = ta < nr_tot ? lr[ta] : -1;
    int jb = tb < nr_tot ? lr[tb] : -1;
    if (ja >= 0 && !NNP_IN_BOUNDS(ws.status, kSiteBwdNeighbour, ja, ws.totals[0])) ja = -1;
    if (jb >= 0 && !NNP_IN_BOUNDS(ws.status, kSiteBwdNeighbour, jb, ws.totals[0])) jb = -1;
    const float4 xa = ja >= 0 ? ws.xyzq[ja] : xi;
    const float4 xb = jb >= 0 ? ws.xyzq[jb] : xi;
    if (ja >= 0) {
      while (H.off_r[sr + 1] <= ta) ++sr;
      radial_edge_bwd<VIR>(ws, ac, xi, d, ja, xa, grad + sr * kNR, inv_rc_r, fi, vir,
                           det ? ws.fr_det + (size_t)p * ws.cap_r + ta : nullptr);
    }
    if (jb >= 0) {
      while (H.off_r[sr + 1] <= tb) ++sr;
      radial_edge_bwd<VIR>(ws, ac, xi, d, jb, xb, grad + sr * kNR, inv_rc_r, fi, vir,
                           det ? ws.fr_det + (size_t)p * ws.cap_r + tb : nullptr);
    }
  }
  __syncwarp();   // the radial dE/dG's region now takes the angular blocks
  // ---- the live species-pair blocks: slot k of the k-th live pair (s <= u) in
  // the order 8 s + u, its dE/dG (32 values, index 8a + z) staged in that order
  {
    float* gf = reinterpret_cast<float*>(gall);
    unsigned m[2];
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int l = 32 * half + (int)lane, s = l >> 3, u = l & 7;
      bool live = false;
      if (s <= u && u < ac.S) {
        const int cs = H.off_a[s + 1] - H.off_a[s], cu = H.off_a[u + 1] - H.off_a[u];
        live = s == u ? cs >= 2 : (cs >= 1 && cu >= 1);
      }
      m[half] = __ballot_sync(kFull, live);
      if (live) {
        const int slot = (half ? __popc(m[0]) : 0) + __popc(m[half] & ((1u << lane) - 1u));
        pslot[8 * s + u] = (uint8_t)slot;
        pslot[8 * u + s] = (uint8_t)slot;
      }
    }
    // the blocks' loads are issued four at a time before their stores
    for (int k0 = 0; k0 < n_live; k0 += 4) {
      float gv[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        gv[k] = 0.f;
        if (k0 + k < n_live) {
          int l;
          if (m[0]) { l = __ffs(m[0]) - 1; m[0] &= m[0] - 1; }
          else { l = 32 + __ffs(m[1]) - 1; m[1] &= m[1] - 1; }
          const int s = l >> 3, u = l & 7;
          const int q = s * ac.S - s * (s - 1) / 2 + (u - s);
          gv[k] = g_row[ac.acol[q] + lane];
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k0 + k < n_live) gf[(k0 + k) * (4 * kGallStride) + lane] = gv[k];
    }
  }
  __syncwarp();
  // ---- angular triplets in round-robin order, one lane per pair: a pass takes
  // the next 32 pairs but at most n_copy rounds, round r adding into copy
  // r mod n_copy with plain read-add-write (within a round the pairs are
  // disjoint, so no two lanes of a pass touch the same accumulator); the order
  // of every addition is fixed, in the deterministic mode too
  const RoundRobin rr = make_round_robin(na_tot);
  for (int t0 = 0; t0 < rr.n_tri;) {
    const int r0 = rr_round(rr, t0);
    const int t1 = min(min(t0 + 32, (r0 + n_copy) * rr.h), rr.n_tri);
    const int t = t0 + (int)lane;
    if (t < t1) {
      int r, a, b;
      rr_pair(rr, t, &r, &a, &b);
      if (NNP_IN_BOUNDS(ws.status, kSiteBwdTriplet, a, na_tot) &&
          NNP_IN_BOUNDS(ws.status, kSiteBwdTriplet, b, na_tot)) {
        const int slot = pslot[8 * spec[a] + spec[b]];
        if (NNP_IN_BOUNDS(ws.status, kSiteBwdTriplet, slot, n_live)) {
          float3 ua, ub;
          triplet_bwd<ZETA>(ac, angv[a], angv[b], angf[a], angf[b], gall + slot * kGallStride,
                            ua, ub);
          float4* A = acc + (r & (n_copy - 1)) * cap_l;
          float4 x = A[a];
          x.x += ua.x; x.y += ua.y; x.z += ua.z;
          A[a] = x;
          float4 y = A[b];
          y.x += ub.x; y.y += ub.y; y.z += ub.z;
          A[b] = y;
        }
      }
    }
    __syncwarp();   // the next pass may add into the same accumulators
    t0 = t1;
  }
  for (int t = lane; t < na_tot; t += 32) {
    float4 a = acc[t];
    for (int c = 1; c < n_copy; ++c) {
      const float4 v = acc[c * cap_l + t];
      a.x += v.x;
      a.y += v.y;
      a.z += v.z;
    }
    const float4 v = angv[t];
    const int jt = __float_as_int(angf[t].w);
    if (det) ws.fa_det[(size_t)p * ws.cap_a + t] = make_float4(-a.x, -a.y, -a.z, 0.f);
    else if (NNP_IN_BOUNDS(ws.status, kSiteBwdNeighbour, jt, ws.totals[0]))
      atomicAdd(&ws.f_pos[jt], make_float4(-a.x, -a.y, -a.z, 0.f));
    fi[0] += a.x; fi[1] += a.y; fi[2] += a.z;
    if (VIR) {
      const float ux = v.x * v.w, uy = v.y * v.w, uz = v.z * v.w;
      vir[0] -= ux * a.x; vir[1] -= ux * a.y; vir[2] -= ux * a.z;
      vir[3] -= uy * a.x; vir[4] -= uy * a.y; vir[5] -= uy * a.z;
      vir[6] -= uz * a.x; vir[7] -= uz * a.y; vir[8] -= uz * a.z;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    fi[0] += __shfl_xor_sync(kFull, fi[0], o);
    fi[1] += __shfl_xor_sync(kFull, fi[1], o);
    fi[2] += __shfl_xor_sync(kFull, fi[2], o);
  }
  if (lane == 0) {
    if (det) ws.fs_det[p] = make_float4(fi[0], fi[1], fi[2], 0.f);
    else atomicAdd(&ws.f_pos[p], make_float4(fi[0], fi[1], fi[2], 0.f));
  }
  if (VIR && d.in.virial) {
    if (!det && vs.dst != d.in.virial) vs.flush(lane, d.in.virial);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      float v = vir[k];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
      if (det) {
        if (lane == 0) ws.v_det[(size_t)p * 9 + k] = (double)v;
      } else if ((int)lane == k) {
        vs.sum += (double)v;
      }
    }
  }
}

template <int ZETA, bool VIR>
__global__ void __launch_bounds__(kWarps * 32, 4)
k_aev_bwd(Ws ws, AevConst ac, int log_r, int cap_l, int small) {
  extern __shared__ float4 sm4[];
  __shared__ ListHdr hdrs[kWarps];
  const int w = threadIdx.x >> 5;
  const unsigned lane = threadIdx.x & 31;
  // persistent: every warp takes the next centre from a counter until none is left
  const int n = ws.totals[0];
  if (n <= small) return;   // a CTA per centre: k_aev_bwd_cta's
  VirialSum vs;
  for (;;) {
    int p = 0;
    if (lane == 0) p = atomicAdd(ws.totals + 5, 1);
    p = __shfl_sync(kFull, p, 0);
    if (p >= n) break;
    bwd_centre<ZETA, VIR>(ws, ac, log_r, cap_l, p, sm4, hdrs[w], w, lane, vs);
  }
  if (VIR) {
    // the CTA's warps that hold the same system's sum add it together
    __shared__ double vsum[kWarps][9];
    __shared__ double* vdst[kWarps];
    if (lane < 9) vsum[w][lane] = vs.sum;
    if (lane == 0) vdst[w] = vs.dst;
    __syncthreads();
    if (w == 0 && lane < 9) {
      double* dst = nullptr;
      double sum = 0.0;
      for (int k = 0; k < kWarps; ++k) {
        if (vdst[k] != dst) {
          if (dst) atomicAdd(dst + lane, sum);
          dst = vdst[k];
          sum = 0.0;
        }
        sum += vsum[k][lane];
      }
      if (dst) atomicAdd(dst + lane, sum);
    }
  }
}

// CTA per centre: for the dense centres (ws.heavy; a dense solute core can have a
// hundred neighbours, i.e. thousands of triplets), and for every centre of a small batch.  The
// CTA's eight warps share the centre's staged neighbours and dE/dG blocks and split its
// radial edges and triplets.  The triplets come in the round-robin order of k_aev_bwd
// in chunks of 32 (fewer for few neighbours: a chunk spans at most `copies` rounds of
// disjoint pairs), every eighth chunk to a warp, which adds into its own accumulator
// copies by plain read-add-write: no atomics, and the order of every addition is fixed,
// which serves the deterministic mode too.  Persistent: CTAs stride over the list.
// Dense centres of solvated100k: 44 us (65 us with shared-memory float atomics into
// lane copies and pairs numbered by species block).
constexpr int kCtaThreads = kWarps * 32;

__host__ __device__ constexpr int bwd_cta_f4(int cap_a, int n_pairs, int copies) {
  return 2 * cap_a + kWarps * copies * cap_a + kMaxSpecies * kNR / 4 + kGallStride * n_pairs + (cap_a + 64 + 15) / 16;
}
// 4 copies where three CTAs then fit an SM, else 2
int bwd_cta_copies(int cap_a, int n_pairs) {
  return bwd_cta_f4(cap_a, n_pairs, 4) * 16 <= 74 * 1024 ? 4 : 2;
}

template <int ZETA, bool VIR>
__global__ void __launch_bounds__(kCtaThreads, 3)
k_aev_bwd_cta(Ws ws, AevConst ac, int copies, int small) {
  extern __shared__ float4 smh[];
  __shared__ ListHdr H;
  __shared__ float red[kWarps][12];
  const int cap = ws.cap_a;
  const int tid = threadIdx.x, w = tid >> 5;
  const unsigned lane = tid & 31;
  float4* angv = smh;                      // unit vector and R
  float4* angf = angv + cap;               // fc, fc', 1/R, packed index
  float4* acc = angf + cap;                // [warp][copy][neighbour]
  float* grad = reinterpret_cast<float*>(acc + (size_t)kWarps * copies * cap);
  float4* gall = reinterpret_cast<float4*>(grad + kMaxSpecies * kNR);   // [block slot][8a + z] (+ pad)
  uint8_t* spec = reinterpret_cast<uint8_t*>(gall + kGallStride * ac.n_pairs);   // [cap]
  uint8_t* pslot = spec + cap;             // [8 s + u]: block slot of species pair (s, u)
  const int n = ws.totals[0];
  const bool all = n <= small;
  const int n_list = all ? n : ws.totals[2];
  const bool det = ws.fr_det != nullptr;   // deterministic mode
  const float inv_rc_r = 1.f / ac.rc_r, inv_rc_a = 1.f / ac.rc_a;
  double* vdst = nullptr;   // thread 3 + k: component k of the virial of one system
  double vsum = 0.0;
  for (int h = blockIdx.x; h < n_list; h += gridDim.x) {
    const int p = all ? h : ws.heavy[h];
    __syncthreads();   // the previous centre's shared data are no longer read
    if (w == 0) load_hdr(ws.nb_cnt + (size_t)p * 16, ac.S, lane, &H);
    const float4 xi = ws.xyzq[p];
    const SysDev& d = ws.sys[ws.pos_sys[p]];
    const float* g_row = ws.dEdG + (size_t)ws.pos_slot[p] * ac.Dp;
    const int* lr = ws.nb_r + (size_t)p * ws.cap_r;
    const int* la = ws.nb_a + (size_t)p * ws.cap_a;
    for (int f = tid; f < ac.S * kNR; f += kCtaThreads) grad[f] = g_row[ac.rcol[f >> 4] + (f & 15)];
    __syncthreads();
    const int na = H.off_a[ac.S], nr = H.off_r[ac.S];
    stage_list<kWarps>(na, la, xi, d, ws, tid, [&](int slot, int j, const Geo& g) {
      const float inv = rcp_approx(g.r);
      angv[slot] = make_float4(g.dx * inv, g.dy * inv, g.dz * inv, g.r);
      float fc, dfc;
      fcut_both(g.r, ac.rc_a, inv_rc_a, &fc, &dfc);
      angf[slot] = make_float4(fc, dfc, inv, __int_as_float(j));
    });
    for (int t = tid; t < na; t += kCtaThreads) {
      int s = 0;
      while (s + 1 < ac.S && H.off_a[s + 1] <= t) ++s;
      spec[t] = (uint8_t)s;
    }
    for (int c = w; c < kWarps * copies; c += kWarps)
      for (int t = lane; t < na; t += 32) acc[c * cap + t] = make_float4(0.f, 0.f, 0.f, 0.f);
    // the live species-pair blocks, in the order of their pairs, in turn to the warps:
    // dE/dG in feature order
    {
      float* gf = reinterpret_cast<float*>(gall);
      int slot = 0;
      for (int s = 0; s < ac.S; ++s) {
        const int cs = H.off_a[s + 1] - H.off_a[s];
        for (int u = s; u < ac.S; ++u) {
          const int cu = H.off_a[u + 1] - H.off_a[u];
          if (s == u ? cs < 2 : (cs < 1 || cu < 1)) continue;
          if (slot % kWarps == w) {
            gf[slot * (4 * kGallStride) + lane] = g_row[ac.acol[s * ac.S - s * (s - 1) / 2 + (u - s)] + lane];
            if (lane == 0) pslot[8 * s + u] = pslot[8 * u + s] = (uint8_t)slot;
          }
          ++slot;
        }
      }
    }
    float fi[3] = {0.f, 0.f, 0.f};
    float vir[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) vir[k] = 0.f;
    int sr = 0;
    for (int t = tid; t < nr; t += kCtaThreads) {
      while (H.off_r[sr + 1] <= t) ++sr;
      const int j = lr[t];
      if (!NNP_IN_BOUNDS(ws.status, kSiteBwdNeighbour, j, ws.totals[0])) continue;
      radial_edge_bwd<VIR>(ws, ac, xi, d, j, ws.xyzq[j], grad + sr * kNR, inv_rc_r, fi, vir,
                           det ? ws.fr_det + (size_t)p * ws.cap_r + t : nullptr);
    }
    __syncthreads();   // the staged neighbours, blocks and zeroed accumulators are complete
    // c consecutive pairs span at most `copies` rounds of rr.h pairs
    const RoundRobin rr = make_round_robin(na);
    const int chunk = min(32, (copies - 1) * rr.h + 1);
    for (int t0 = w * chunk; t0 < rr.n_tri; t0 += kWarps * chunk) {
      const int t = t0 + (int)lane;
      if ((int)lane < chunk && t < rr.n_tri) {
        int r, a, b;
        rr_pair(rr, t, &r, &a, &b);
        if (NNP_IN_BOUNDS(ws.status, kSiteBwdTriplet, a, na) &&
            NNP_IN_BOUNDS(ws.status, kSiteBwdTriplet, b, na)) {
          const int slot = pslot[8 * spec[a] + spec[b]];
          if (NNP_IN_BOUNDS(ws.status, kSiteBwdTriplet, slot, ac.n_pairs)) {
            float3 ua, ub;
            triplet_bwd<ZETA>(ac, angv[a], angv[b], angf[a], angf[b], gall + slot * kGallStride, ua, ub);
            float4* A = acc + (size_t)(w * copies + (r & (copies - 1))) * cap;
            float4 x = A[a];
            x.x += ua.x; x.y += ua.y; x.z += ua.z;
            A[a] = x;
            float4 y = A[b];
            y.x += ub.x; y.y += ub.y; y.z += ub.z;
            A[b] = y;
          }
        }
      }
      __syncwarp();   // the next chunk may add into the same accumulators
    }
    __syncthreads();
    // four threads per neighbour sum its copies (every fourth warp's), then combine
    const int n_copy = kWarps * copies, n4 = (na + 63) / 64 * 64;
    for (int q = tid; q < 4 * n4; q += kCtaThreads) {
      const int t = q >> 2, part = q & 3;
      float3 a = make_float3(0.f, 0.f, 0.f);
      if (t < na)
        for (int c = part; c < n_copy; c += 4) {
          const float4 x = acc[c * cap + t];
          a.x += x.x; a.y += x.y; a.z += x.z;
        }
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        a.x += __shfl_xor_sync(kFull, a.x, o);
        a.y += __shfl_xor_sync(kFull, a.y, o);
        a.z += __shfl_xor_sync(kFull, a.z, o);
      }
      if (part == 0 && t < na) {
        const float4 v = angv[t];
        const int jt = __float_as_int(angf[t].w);
        if (det) ws.fa_det[(size_t)p * ws.cap_a + t] = make_float4(-a.x, -a.y, -a.z, 0.f);
        else if (NNP_IN_BOUNDS(ws.status, kSiteBwdNeighbour, jt, ws.totals[0]))
          atomicAdd(&ws.f_pos[jt], make_float4(-a.x, -a.y, -a.z, 0.f));
        fi[0] += a.x; fi[1] += a.y; fi[2] += a.z;
        if (VIR) {
          const float ux = v.x * v.w, uy = v.y * v.w, uz = v.z * v.w;
          vir[0] -= ux * a.x; vir[1] -= ux * a.y; vir[2] -= ux * a.z;
          vir[3] -= uy * a.x; vir[4] -= uy * a.y; vir[5] -= uy * a.z;
          vir[6] -= uz * a.x; vir[7] -= uz * a.y; vir[8] -= uz * a.z;
        }
      }
    }
    // the centre's force and the virial: warp sums, then threads 0-11 over the warps
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      fi[0] += __shfl_xor_sync(kFull, fi[0], o);
      fi[1] += __shfl_xor_sync(kFull, fi[1], o);
      fi[2] += __shfl_xor_sync(kFull, fi[2], o);
#pragma unroll
      for (int k = 0; k < 9; ++k)
        if (VIR) vir[k] += __shfl_xor_sync(kFull, vir[k], o);
    }
    if (lane == 0) {
      red[w][0] = fi[0]; red[w][1] = fi[1]; red[w][2] = fi[2];
#pragma unroll
      for (int k = 0; k < 9; ++k) red[w][3 + k] = VIR ? vir[k] : 0.f;
    }
    __syncthreads();
    if (tid < 12) {
      float v = 0.f;
      for (int k = 0; k < kWarps; ++k) v += red[k][tid];
      if (tid < 3) {
        if (det) reinterpret_cast<float*>(&ws.fs_det[p])[tid] = v;
        else atomicAdd(reinterpret_cast<float*>(&ws.f_pos[p]) + tid, v);
      } else if (VIR && d.in.virial) {
        if (det) {
          ws.v_det[(size_t)p * 9 + (tid - 3)] = (double)v;
        } else {   // added up in FP64 while the CTA's centres belong to one system
          if (vdst != d.in.virial + (tid - 3)) {
            if (vdst) atomicAdd(vdst, vsum);
            vdst = d.in.virial + (tid - 3);
            vsum = 0.0;
          }
          vsum += (double)v;
        }
      }
    }
  }
  if (VIR && vdst) atomicAdd(vdst, vsum);
}

// ---------------------------------------------------------------- AEV -> first layer
// One CTA per 128-row tile of a species segment (BF16, one-network models):
// its 32 warps compute the AEV rows of the tile's atoms (four per warp, the
// same per-centre code as k_aev_fwd) straight into shared memory as BF16, in
// the 128-byte-swizzled K-major layout the tensor core reads, so the AEV never
// goes to HBM; then one thread streams the species' W1 by TMA in 64-wide K
// slices and issues tcgen05.mma (M = 128, N = h1) into tensor memory, and four
// warps apply the bias and CELU and write h1.  Rows past the segment's atom
// count are zero.
constexpr int kL1Warps = 32;
constexpr int kL1Blk = 128 * 128;          // one 64-column block of the A tile (bytes)
constexpr int kL1MaxSmem = 232448 - 16384;

struct AevL1Args {
  const float* b1;      // [S][h1]
  __nv_bfloat16* H1;    // [rows][h1]
  int h1;
  float alpha;
  int stage_bytes;      // one W1 slice: h1 x 64 BF16
};

__device__ __forceinline__ void put_tile(uint8_t* tile, int r, int f, float v) {
  const int blk = f >> 6, c = f & 63;
  uint8_t* row = tile + blk * kL1Blk + r * 128;
  const int off = ((((c >> 3) ^ (r & 7)) << 4) | ((c & 7) << 1));
  *reinterpret_cast<__nv_bfloat16*>(row + off) = __float2bfloat16_rn(v);
}

template <int ZETA>
__global__ void __launch_bounds__(kL1Warps * 32, 1)
k_aev_l1(const __grid_constant__ CUtensorMap tw1, Ws ws, AevConst ac, AevL1Args g) {
  using namespace tcu;
  extern __shared__ uint8_t smem_raw[];
  __shared__ ListHdr hdrs[kL1Warps];
  __shared__ __align__(8) uint64_t full_bar[2], empty_bar[2], done_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  __shared__ uint8_t pair_su[kMaxSpecies * (kMaxSpecies + 1) / 2];
  const int w = threadIdx.x >> 5;
  const unsigned lane = threadIdx.x & 31;
  const int S = ac.S;
  const int row_tiles = ws.seg_start[S] / kTileM;
  if ((int)blockIdx.x >= row_tiles) return;    // uniform over the CTA
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int nblk = ac.Dp / 64;
  uint8_t* tile = smem;
  uint8_t* ring = tile + nblk * kL1Blk;
  float4* stage = reinterpret_cast<float4*>(ring + 2 * g.stage_bytes) +
                  (size_t)w * aev_fwd_warp_f4(ws.cap_a, ws.cap_r);
  volatile int* abort_flag = &abort_sh;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], 1);
    }
    mbar_init(&done_bar, 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (w == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base_sh)), "r"(256u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fill_pair_table(pair_su, ac);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  const int m0 = blockIdx.x * kTileM;
  int sp = 0;
  while (sp + 1 < S && m0 >= ws.seg_start[sp + 1]) ++sp;
  const int seg_end = ws.seg_start[sp] + ws.species_count[sp];
  // ---- the tile's AEV rows into shared memory
  for (int r = w; r < kTileM; r += kL1Warps) {
    const int slot = m0 + r;
    if (slot < seg_end) {
      aev_centre<ZETA, 1>(ws, ac, ws.slot_pos[slot], stage, hdrs[w], lane, pair_su,
                          [&](int f, float v) { put_tile(tile, r, f, v); });
    } else {
      for (int f = (int)lane; f < ac.Dp; f += 32) put_tile(tile, r, f, 0.f);
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> tensor core
  __syncthreads();
  // ---- first layer: W1 of species sp by TMA, MMAs by one thread
  if (w == 0 && lane == 0) {
    const int nk = nblk;
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(g.h1 >> 3) << 17) |
                           ((uint32_t)(kTileM >> 4) << 24);
    bool ok = true;
    int issued = 0;
    for (; issued < 2 && issued < nk; ++issued) {
      mbar_expect_tx(&full_bar[issued], (unsigned)g.stage_bytes);
      tma_load_3d(ring + issued * g.stage_bytes, &tw1, &full_bar[issued], issued * 64, 0, sp);
    }
    for (int kb = 0; kb < nk && ok; ++kb) {
      const int st = kb & 1;
      if (!mbar_wait(&full_bar[st], (kb >> 1) & 1, abort_flag)) { ok = false; break; }
      tc_fence_after();
      const uint64_t ad = sw128_desc(smem_u32(tile + kb * kL1Blk));
      const uint64_t bd = sw128_desc(smem_u32(ring + st * g.stage_bytes));
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        umma_bf16(tmem, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), idesc, (kb > 0 || kk > 0) ? 1u : 0u);
      umma_commit(&empty_bar[st]);
      if (issued < nk) {
        if (!mbar_wait(&empty_bar[st], (kb >> 1) & 1, abort_flag)) { ok = false; break; }
        mbar_expect_tx(&full_bar[st], (unsigned)g.stage_bytes);
        tma_load_3d(ring + st * g.stage_bytes, &tw1, &full_bar[st], issued * 64, 0, sp);
        ++issued;
      }
    }
    umma_commit(&done_bar);   // arrives when every MMA issued above has completed
    if (!ok) {
      // every issued copy lands before the CTA may exit
      for (int k = issued - 2 < 0 ? 0 : issued - 2; k < issued; ++k)
        mbar_drain(&full_bar[k & 1], (k >> 1) & 1);
    }
  }
  // ---- epilogue: bias, CELU, h1 (TMEM lanes 32 w .. of warps 0-3)
  if (w < 4) {
    if (mbar_wait(&done_bar, 0, abort_flag)) {
      tc_fence_after();
      const int r = w * 32 + (int)lane;
      const uint32_t trow = tmem + ((uint32_t)(w * 32) << 16);
      const float* bias = g.b1 + (size_t)sp * g.h1;
      const float alpha = g.alpha, inv_alpha = 1.f / g.alpha;
      for (int c0 = 0; c0 < g.h1; c0 += 16) {
        float v[16];
        tmem_ld16(trow + (uint32_t)c0, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float z = v[i] + __ldg(bias + c0 + i);
          v[i] = z > 0.f ? z : alpha * (__expf(z * inv_alpha) - 1.f);
        }
        store_bf16x16(g.H1 + (size_t)(m0 + r) * g.h1 + c0, v);
      }
    } else {
      mbar_drain(&done_bar, 0);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) atomicOr(ws.status, kStTimeout);
  if (w == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
}

size_t aev_l1_smem(const Ws& ws, const AevConst& ac, int h1) {
  return (size_t)(ac.Dp / 64) * kL1Blk + 2 * (size_t)h1 * 64 * 2 +
         (size_t)kL1Warps * aev_fwd_warp_f4(ws.cap_a, ws.cap_r) * sizeof(float4) + 1024;
}

}  // namespace

size_t aev_fwd_smem(const Ws& ws) {
  return (size_t)kWarps * aev_fwd_warp_f4(ws.cap_a, ws.cap_r) * sizeof(float4);
}
// angular neighbours a warp of the warp-per-centre backward stages
static int light_cap(const Ws& ws) { return std::min(ws.cap_a, kDenseNeighbours); }

size_t aev_bwd_smem(const Ws& ws, int n_pairs) {
  const int cap_l = light_cap(ws);
  return (size_t)kWarps * aev_bwd_warp_f4(cap_l, n_pairs, aev_bwd_copies(cap_l, n_pairs)) *
         sizeof(float4);
}

static size_t bwd_cta_smem(const Ws& ws, int n_pairs) {
  return (size_t)bwd_cta_f4(ws.cap_a, n_pairs, bwd_cta_copies(ws.cap_a, n_pairs)) * sizeof(float4);
}

static int sm_count() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms < 1) sms = 1;
  }
  return sms;
}

// up to this many centres get a CTA each in the forward and the backward: four CTAs
// per SM, one wave.  A 50-atom region: forward 34 -> 12 us, backward 28 -> 10 us; a
// 24-atom molecule 9.1 -> 7.4 and 7.5 -> 6.0 us.
static int small_centres() { return 4 * sm_count(); }

// grid of the persistent warp-per-centre kernels: four CTAs per SM at most, fewer for
// small batches (up to `small` centres have a CTA each, and a mask may leave so few)
static int centre_grid(int n_in, int small, bool masked) {
  const int want = n_in <= small ? n_in : std::max((n_in + kWarps - 1) / kWarps, masked ? small : 1);
  return std::max(1, std::min(want, 4 * sm_count()));
}

void launch_aev_fwd(const Ws& ws, int n_in, bool masked, const AevConst& ac, cudaStream_t st) {
  if (n_in <= 0) return;
  const size_t sm = aev_fwd_smem(ws);
  const int small = small_centres(), grid = centre_grid(n_in, small, masked);
  if (ac.zeta == 32) k_aev_fwd<32><<<grid, kWarps * 32, sm, st>>>(ws, ac, small);
  else k_aev_fwd<0><<<grid, kWarps * 32, sm, st>>>(ws, ac, small);
}

void launch_aev_fill(const Ws& ws, const AevConst& ac, cudaStream_t st) {
  if (!ws.row_mask) return;
  k_aev_fill<<<(ws.row_cap + 7) / 8, 256, 0, st>>>(ws, ac);
}

void launch_aev_bwd(const Ws& ws, int n_in, bool masked, const AevConst& ac, int want_virial,
                    cudaStream_t st, const SideStream* side) {
  if (n_in <= 0) return;
  const int cap_l = light_cap(ws), small = small_centres();
  // The two kernels add to different accumulators or atomically, so with a side stream
  // they run together: the CTA-per-centre kernel first (higher priority), the other
  // beside it as room allows (6k solvated atoms: 43 us one after the other, 34 together).
  if (n_in <= small) side = nullptr;
  const cudaStream_t main_st = st;
  if (side) {
    cudaEventRecord(side->fork, st);
    cudaStreamWaitEvent(side->st, side->fork, 0);
    st = side->st;
  }
  // the CTA-per-centre kernel: where centres can exceed what a warp takes, and where
  // the batch is small (a mask may leave few centres of many atoms)
  if (n_in <= small || masked || ws.cap_a > cap_l || ac.n_pairs > kGallBlocks) {
    const size_t sm = bwd_cta_smem(ws, ac.n_pairs);
    const int copies = bwd_cta_copies(ws.cap_a, ac.n_pairs), grid = std::min(n_in, 4 * sm_count());
    if (ac.zeta == 32) {
      if (want_virial) k_aev_bwd_cta<32, true><<<grid, kCtaThreads, sm, st>>>(ws, ac, copies, small);
      else k_aev_bwd_cta<32, false><<<grid, kCtaThreads, sm, st>>>(ws, ac, copies, small);
    } else {
      if (want_virial) k_aev_bwd_cta<0, true><<<grid, kCtaThreads, sm, st>>>(ws, ac, copies, small);
      else k_aev_bwd_cta<0, false><<<grid, kCtaThreads, sm, st>>>(ws, ac, copies, small);
    }
  }
  if (n_in <= small) return;
  if (side) cudaEventRecord(side->join, st);
  st = main_st;
  const size_t sm = aev_bwd_smem(ws, ac.n_pairs);
  const int copies = aev_bwd_copies(cap_l, ac.n_pairs);
  const int log_r = copies == 4 ? 2 : copies == 2 ? 1 : 0;
  const int grid = centre_grid(n_in, small, masked);
  if (ac.zeta == 32) {
    if (want_virial) k_aev_bwd<32, true><<<grid, kWarps * 32, sm, st>>>(ws, ac, log_r, cap_l, small);
    else k_aev_bwd<32, false><<<grid, kWarps * 32, sm, st>>>(ws, ac, log_r, cap_l, small);
  } else {
    if (want_virial) k_aev_bwd<0, true><<<grid, kWarps * 32, sm, st>>>(ws, ac, log_r, cap_l, small);
    else k_aev_bwd<0, false><<<grid, kWarps * 32, sm, st>>>(ws, ac, log_r, cap_l, small);
  }
  if (side) cudaStreamWaitEvent(st, side->join, 0);
}

// raise (never lower) the dynamic shared-memory limit of the AEV kernels to what
// a launch over `ws` needs
cudaError_t aev_ensure_smem(const Ws& ws) {
  // the backward kernel's size depends on the species-pair count through the
  // number of accumulator copies: take the largest over every model size
  int need_b = 0;
  for (int np = 1; np <= kMaxSpecies * (kMaxSpecies + 1) / 2; ++np)
    need_b = std::max(need_b, (int)aev_bwd_smem(ws, np));
  const int need_f = (int)aev_fwd_smem(ws);
  int need_h = 0;
  for (int np = 1; np <= kMaxSpecies * (kMaxSpecies + 1) / 2; ++np)
    need_h = std::max(need_h, (int)bwd_cta_smem(ws, np));
  const void* fwd[2] = {(const void*)k_aev_fwd<32>, (const void*)k_aev_fwd<0>};
  const void* bwd[4] = {(const void*)k_aev_bwd<32, false>, (const void*)k_aev_bwd<32, true>,
                        (const void*)k_aev_bwd<0, false>, (const void*)k_aev_bwd<0, true>};
  const void* hvy[4] = {(const void*)k_aev_bwd_cta<32, false>,
                        (const void*)k_aev_bwd_cta<32, true>,
                        (const void*)k_aev_bwd_cta<0, false>,
                        (const void*)k_aev_bwd_cta<0, true>};
  for (int pass = 0; pass < 3; ++pass)
    for (int i = 0; i < (pass == 0 ? 2 : 4); ++i) {
      const void* fn = pass == 0 ? fwd[i] : pass == 1 ? bwd[i] : hvy[i];
      const int need = pass == 0 ? need_f : pass == 1 ? need_b : need_h;
      cudaFuncAttributes attr;
      cudaError_t e = cudaFuncGetAttributes(&attr, fn);
      if (e != cudaSuccess) return e;
      if (attr.maxDynamicSharedSizeBytes < need) {
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, need);
        if (e != cudaSuccess) return e;
      }
    }
  return cudaSuccess;
}


bool aev_l1_supported(const Ws& ws, const AevConst& ac, int E, int h1) {
  return E == 1 && ac.Dp % 64 == 0 && h1 % 16 == 0 && h1 >= 16 && h1 <= 256 && ws.slot_pos &&
         aev_l1_smem(ws, ac, h1) <= (size_t)kL1MaxSmem;
}

void launch_aev_l1(const Ws& ws, const AevConst& ac, const void* w1_bf16, const float* b1,
                   void* H1, int h1, float alpha, cudaStream_t st) {
  // W1 of every species [S][h1][Dp] BF16: dims (Dp, h1, S), box (64, h1, 1)
  CUtensorMap m;
  if (!tcu::make_map(&m, w1_bf16, ac.Dp, h1, ac.S, ac.Dp, (uint64_t)ac.Dp * h1, (uint32_t)h1, 1)) return;
  AevL1Args g{};
  g.b1 = b1;
  g.H1 = static_cast<__nv_bfloat16*>(H1);
  g.h1 = h1;
  g.alpha = alpha;
  g.stage_bytes = h1 * 64 * 2;
  const size_t sm = aev_l1_smem(ws, ac, h1);
  const int grid = (ws.row_cap + tcu::kTileM - 1) / tcu::kTileM;
  if (ac.zeta == 32) k_aev_l1<32><<<grid, kL1Warps * 32, sm, st>>>(m, ws, ac, g);
  else k_aev_l1<0><<<grid, kL1Warps * 32, sm, st>>>(m, ws, ac, g);
}

cudaError_t aev_l1_ensure_smem(const Ws& ws, const AevConst& ac, int h1) {
  const int need = (int)std::min(aev_l1_smem(ws, ac, h1), (size_t)kL1MaxSmem);
  for (const void* fn : {(const void*)k_aev_l1<32>, (const void*)k_aev_l1<0>}) {
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, fn);
    if (e != cudaSuccess) return e;
    if (attr.maxDynamicSharedSizeBytes < need) {
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, need);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

}  // namespace nnp
