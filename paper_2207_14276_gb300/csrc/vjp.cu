// Double backward of the potential: the vector-Jacobian product of the forces,
// for training by force matching (loss L(E, F), v = dL/dF, gE = dL/dE).
//
//   dL/dr      = -gE F + d/de F(r + e v)            (a Hessian-vector product)
//   dL/dtheta  = gE dE/dtheta - d/dtheta [ sum_i dE_i/dG_i . u_i ],  u_i = J_i v
//
// Kernels (FP32):
//   k_gather_v       v in packed (cell) order
//   k_aev_fwd_vjp    G_i and u_i = d/de G_i(r + e v): the forward AEV and its
//                    derivative along v from one pass over the triplets
//   (launch_gemm_dual, mlp_simt.cu: the networks' values and tangents, layer by
//                    layer, with the forward-over-reverse steps in the epilogues)
//   k_aev_bwd_dual   the AEV backward and its derivative: primal inputs (r, dE/dG)
//                    with tangents (v, q = H_e u) give F and d/de F
//   k_wgrad          weight and bias gradients of every layer, species and member
//   k_vjp_scatter    dL/dr back to the caller's atom order
#include <algorithm>

#include "aev_device.cuh"
#include "mlp.cuh"
#include "nnp_internal.cuh"
#include "vjp.cuh"

namespace nnp {

namespace {

constexpr int kWarps = 4;

// cosine cutoff (Eq. 3) and its first two derivatives
__device__ __forceinline__ void fcut3(float r, float rc, float* f, float* df, float* ddf) {
  if (r < rc) {
    const float w = kPi / rc;
    float sn, cs;
    sincospif(r / rc, &sn, &cs);
    *f = 0.5f * cs + 0.5f;
    *df = -0.5f * w * sn;
    *ddf = -0.5f * w * w * cs;
  } else {
    *f = *df = *ddf = 0.f;
  }
}

__global__ void k_gather_v(Ws ws, VjpBufs vb) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= ws.totals[0]) return;
  const int b = ws.pos_sys[p];
  const int local = ws.pos_src[p] - ws.sys[b].in.in_base;
  const float* v = ws.sys[b].in.dLdF;
  vb.v_pos[p] = make_float4(v[3 * local], v[3 * local + 1], v[3 * local + 2], 0.f);
  vb.df_pos[p] = make_float4(0.f, 0.f, 0.f, 0.f);
  vb.gE_row[ws.pos_slot[p]] = (float)ws.sys[b].in.gE;
}

// float4s of shared memory per warp of k_aev_fwd_vjp
__host__ __device__ constexpr int fwd_warp_f4(int cap_a, int cap_r) { return 3 * cap_a + cap_r; }

// G_i and u_i = d/de G_i(r + e v) (Eqs. 3-5 and their derivative along v), one warp
// per centre, lane per triplet as in k_aev_fwd.  A triplet's Gaussians, powers and
// cutoffs serve both, so the tangent costs two more packed FMAs per pair of angle
// sections; the two 32-feature blocks are transposed and reduced one after the
// other.  Latency-bound at training sizes (a few thousand centres, one wave).  1,500
// water atoms: 15 us against 15 + 34 us for the forward and a separate tangent kernel.
template <int ZETA>
__global__ void __launch_bounds__(kWarps * 32) k_aev_fwd_vjp(Ws ws, AevConst ac, VjpBufs vb) {
  extern __shared__ float4 sm4[];
  __shared__ ListHdr hdrs[kWarps];
  __shared__ uint8_t pair_su[kMaxSpecies * (kMaxSpecies + 1) / 2];
  const int w = threadIdx.x >> 5;
  const unsigned lane = threadIdx.x & 31;
  fill_pair_table(pair_su, ac);
  __syncthreads();
  const int p = blockIdx.x * kWarps + w;
  if (p >= ws.totals[0]) return;
  // per warp: angular (u, R), (fc, dfc, Rdot, 1/R), (dv, -); radial (R, fc, dfc, Rdot)
  float4* angv = sm4 + (size_t)w * fwd_warp_f4(ws.cap_a, ws.cap_r);
  float4* angf = angv + ws.cap_a;
  float4* angd = angf + ws.cap_a;
  float4* rad = angd + ws.cap_a;
  ListHdr& H = hdrs[w];
  const float4 xi = ws.xyzq[p];
  const float4 vi = vb.v_pos[p];
  const SysDev& d = ws.sys[ws.pos_sys[p]];
  const int slot = ws.pos_slot[p];
  if (!NNP_IN_BOUNDS(ws.status, kSiteAevRow, slot, ws.row_cap)) return;
  float* G = ws.aev + (size_t)slot * ac.Dp;
  float* U = vb.U + (size_t)slot * ac.Dp;
  load_hdr(ws.nb_cnt + (size_t)p * 16, ac.S, lane, &H);
  const uint32_t msk = ws.row_mask ? row_slices(H, ac, lane, pair_su) : ~0u;
  // (G to rounding, not bit by bit the rows of k_aev_fwd, which takes pairs and radial terms
  // in another order.  CELU'' jumps at z = 0, so where a pre-activation is next to zero a
  // gradient depends on the last bits of G, in any order: 40 boxes of 1,500 water atoms,
  // dL/dcoords from 64 bits 1.8e-6 of its norm in the median and 1.0e-4 on average, both with
  // this order and with the forward's own rows, and two runs, whose cells list their atoms
  // in different orders, up to 1.8e-4 from each other)
  const float inv_rc_r = 1.f / ac.rc_r, inv_rc_a = 1.f / ac.rc_a;
  stage_list(H.off_r[ac.S], ws.nb_r + (size_t)p * ws.cap_r, xi, d, ws, lane,
             [&](int t, int j, const Geo& g) {
               const float4 vj = vb.v_pos[j];
               const float rdot = (g.dx * (vj.x - vi.x) + g.dy * (vj.y - vi.y) + g.dz * (vj.z - vi.z)) / g.r;
               float f, df, ddf;
               fcut3(g.r, ac.rc_r, &f, &df, &ddf);
               rad[t] = make_float4(g.r, fcut(g.r, ac.rc_r, inv_rc_r), df, rdot);
             });
  stage_list(H.off_a[ac.S], ws.nb_a + (size_t)p * ws.cap_a, xi, d, ws, lane,
             [&](int t, int j, const Geo& g) {
               const float4 vj = vb.v_pos[j];
               const float inv = rcp_approx(g.r);
               const float dvx = vj.x - vi.x, dvy = vj.y - vi.y, dvz = vj.z - vi.z;
               float f, df, ddf;
               fcut3(g.r, ac.rc_a, &f, &df, &ddf);
               angv[t] = make_float4(g.dx * inv, g.dy * inv, g.dz * inv, g.r);
               angf[t] = make_float4(fcut(g.r, ac.rc_a, inv_rc_a), df, (g.dx * dvx + g.dy * dvy + g.dz * dvz) * inv, inv);
               angd[t] = make_float4(dvx, dvy, dvz, 0.f);
             });
  __syncwarp();
  // radial: the tangent of exp(-eta x^2) f_c(R) is exp(..) (-2 eta x f_c + f_c') Rdot
  const float cr_ = -ac.eta_r * kLog2e;
  const float my_shf = ac.shf_r[lane & 15];
  const int half = lane >> 4;
  for (int s = 0; s < ac.S; ++s) {
    float ag = 0.f, au = 0.f;
    for (int t = H.off_r[s] + half; t < H.off_r[s + 1]; t += 2) {
      const float4 q = rad[t];
      const float x = q.x - my_shf;
      const float ex = fast_exp2(cr_ * x * x);
      ag = fmaf(ex, q.y, ag);
      au = fmaf(ex * fmaf(-2.f * ac.eta_r * x, q.y, q.z), q.w, au);
    }
    ag += __shfl_xor_sync(kFull, ag, 16);
    au += __shfl_xor_sync(kFull, au, 16);
    if (lane < 16 && block_in(msk, ac.rcol[s], kNR)) {
      G[ac.rcol[s] + lane] = ag;
      U[ac.rcol[s] + lane] = au;
    }
  }
  const float ca_ = -ac.eta_a * kLog2e;
  const float m2eta = -2.f * ac.eta_a;
  for (int q = 0; q < ac.n_pairs; ++q) {
    const int s = pair_su[q] & 15, u = pair_su[q] >> 4;
    const int os = H.off_a[s], cs = H.off_a[s + 1] - os;
    const int ou = H.off_a[u], cu = H.off_a[u + 1] - ou;
    const int same = (s == u);
    const int n_tri = same ? cs * (cs - 1) / 2 : cs * cu;
    const int fb = ac.acol[q];
    if (n_tri == 0) {
      if (block_in(msk, fb, 32)) { G[fb + lane] = 0.f; U[fb + lane] = 0.f; }
      continue;
    }
    const float inv_cu = rcp_approx((float)max(cu, 1));   // decode corrects one step either way
    float2 ag[16], au[16];
#pragma unroll
    for (int f = 0; f < 16; ++f) ag[f] = au[f] = make_float2(0.f, 0.f);
    for (int t = lane; t < n_tri; t += 32) {
      int j, k;
      decode_pair(t, same, cs, cu, inv_cu, &j, &k);
      const float4 uj = angv[os + j], uk = angv[ou + k];
      const float4 fj = angf[os + j], fk = angf[ou + k];
      const float4 dj = angd[os + j], dk = angd[ou + k];
      const float chat = uj.x * uk.x + uj.y * uk.y + uj.z * uk.z;
      // tangent of cos_hat: (u_k - c u_j).dv_j / R_j + (u_j - c u_k).dv_k / R_k
      const float cdot = ((uk.x - chat * uj.x) * dj.x + (uk.y - chat * uj.y) * dj.y +
                          (uk.z - chat * uj.z) * dj.z) * fj.w +
                         ((uj.x - chat * uk.x) * dk.x + (uj.y - chat * uk.y) * dk.y +
                          (uj.z - chat * uk.z) * dk.z) * fk.w;
      const float c = ac.cos_scale * chat;
      const float sn = sin_theta(uj, uk, chat, ac.cos_scale);
      const float m_cs = -c * rcp_approx(fmaxf(sn, 1e-6f));
      const float rb = 0.5f * (uj.w + uk.w), rbdot = 0.5f * (fj.z + fk.z);
      const float fjk = ac.ang_pre * fj.x * fk.x;
      const float fjkdot = ac.ang_pre * (fj.y * fj.z * fk.x + fj.x * fk.y * fk.z);
      const float cz_ = (float)ac.zeta * ac.cos_scale * cdot;
      float2 P[kNA], Q[kNA], R[kNA];   // factors of B in G, of B in u, of dB in u
#pragma unroll
      for (int a = 0; a < kNA; ++a) {
        const float x = rb - ac.shf_a[a];
        const float A = fast_exp2(ca_ * x * x);
        const float pa = A * fjk, qa = A * fmaf(m2eta * x * rbdot, fjk, fjkdot), ra = pa * cz_;
        P[a] = make_float2(pa, pa);
        Q[a] = make_float2(qa, qa);
        R[a] = make_float2(ra, ra);
      }
      const float2 c2 = make_float2(c, c), s2 = make_float2(sn, sn), mcs2 = make_float2(m_cs, m_cs);
#pragma unroll
      for (int m = 0; m < kNZ / 2; ++m) {
        float2 B1;
        const float2 B = section_pair<ZETA>(ac, m, c2, s2, &B1);
        const float2 cz = reinterpret_cast<const float2*>(ac.cos_z)[m];
        const float2 sz = reinterpret_cast<const float2*>(ac.sin_z)[m];
        const float2 dB = __fmul2_rn(B1, __ffma2_rn(sz, mcs2, cz));
#pragma unroll
        for (int a = 0; a < kNA; ++a) {
          ag[4 * a + m] = __ffma2_rn(P[a], B, ag[4 * a + m]);
          au[4 * a + m] = __ffma2_rn(R[a], dB, __ffma2_rn(Q[a], B, au[4 * a + m]));
        }
      }
    }
    float acc[32];
#pragma unroll
    for (int f = 0; f < 16; ++f) { acc[2 * f] = ag[f].x; acc[2 * f + 1] = ag[f].y; }
    G[fb + lane] = transpose_reduce32(acc, lane);
#pragma unroll
    for (int f = 0; f < 16; ++f) { acc[2 * f] = au[f].x; acc[2 * f + 1] = au[f].y; }
    U[fb + lane] = transpose_reduce32(acc, lane);
  }
  for (int f = ac.D + lane; f < ac.Dp; f += 32)
    if ((msk >> (f >> 6)) & 1u) { G[f] = 0.f; U[f] = 0.f; }
  if (ws.row_mask && lane == 0) {
    ws.row_mask[slot] = msk;
    atomicOr(ws.tile_mask + (slot >> 7), msk);
  }
}

// sparse rows: zero the slices of G and U that a row's tile reads but the row left
// unwritten (warp per row)
__global__ void __launch_bounds__(256) k_fill_vjp(Ws ws, AevConst ac, float* U) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5);
  const unsigned lane = threadIdx.x & 31;
  if (r >= ws.seg_start[ac.S]) return;
  int s = 0;
  while (s + 1 < ac.S && r >= ws.seg_start[s + 1]) ++s;
  if (r >= ws.seg_start[s] + ws.species_count[s]) return;
  const size_t row = (size_t)r * ac.Dp;
  for (uint32_t miss = ws.tile_mask[r >> 7] & ~ws.row_mask[r]; miss; miss &= miss - 1) {
    const int f = (__ffs(miss) - 1) * 64 + 2 * (int)lane;
    if (f < ac.Dp) {
      *reinterpret_cast<float2*>(ws.aev + row + f) = make_float2(0.f, 0.f);
      *reinterpret_cast<float2*>(U + row + f) = make_float2(0.f, 0.f);
    }
  }
}

// ---------------------------------------------------------------- dual AEV backward
// float4s per warp: angular (u, R), (fc, fc', fc'', Rdot), (dv, 1/R); per neighbour
// and copy the accumulated dE/du and its tangent; the radial or (after them) the
// angular blocks' dE/dG and q; the neighbours' species and the block-slot table
constexpr int kBlkF4 = 9;   // a block's 32 values and one float4 of padding
__host__ __device__ constexpr int dual_gq_f4(int n_pairs) {
  return 2 * kBlkF4 * n_pairs > 64 ? 2 * kBlkF4 * n_pairs : 64;
}
__host__ __device__ constexpr int dual_warp_f4(int cap_a, int n_pairs, int copies) {
  return 3 * cap_a + 2 * copies * cap_a + dual_gq_f4(n_pairs) + (cap_a + 64 + 15) / 16;
}
// copies of the accumulators (rounds of disjoint pairs that a pass may span): the
// most that keep three CTAs on an SM
int dual_copies(int cap_a, int n_pairs) {
  for (int c = 4; c > 1; c >>= 1)
    if (kWarps * dual_warp_f4(cap_a, n_pairs, c) * 16 <= 74 * 1024) return c;
  return 1;
}

struct Vec3 {
  float x, y, z;
};
__device__ __forceinline__ Vec3 operator*(float s, Vec3 a) { return Vec3{s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ Vec3 operator+(Vec3 a, Vec3 b) { return Vec3{a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ Vec3 operator-(Vec3 a, Vec3 b) { return Vec3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ float dot(Vec3 a, Vec3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ Vec3 v3(const float4& a) { return Vec3{a.x, a.y, a.z}; }

// One angular triplet (Eq. 5): dE/du_j, dE/du_k (gj, gk) and their derivatives
// along (r + e v, dE/dG + e q) (gjt, gkt).  Everything angular is a function of the
// geometric angle p between u_j and u_k (c = k cos p, s = sin(acos c)); with
// base = 1 + c cos_z + s sin_z and r = d theta / d p = k sin p / s (1 for k = 1),
//   h  = dbase/dp   = r t,            t = c sin_z - s cos_z,
//   h' = d2base/dp2 = r' t - r^2 (c cos_z + s sin_z),   r' = (c/s) (1 - r^2),
//   B = base^zeta, dB = base^(zeta-1) h, ddB = (zeta-1) base^(zeta-2) h^2 + base^(zeta-1) h'
// (dB/dp and d2B/dp2 without the factor zeta), so the 32 values of dE/dG and q are
// contracted once over the angle sections (five packed sums per radial shell) and
// the rest is a handful of scalars.  The angle, not its cosine: in terms of c the
// tangent of a nearly collinear triplet is a difference of terms that grow as
// 1/sin^2 (error 1e-7 / sin^2 p), here nothing grows faster than 1/sin p.
template <int ZETA>
__device__ __forceinline__ void triplet_dual(const AevConst& ac, const float4& aj, const float4& ak,
                                             const float4& bj, const float4& bk, const float4& dj,
                                             const float4& dk, const float4* gb, const float4* qb,
                                             Vec3& gj, Vec3& gk, Vec3& gjt, Vec3& gkt) {
  const float ca_ = -ac.eta_a * kLog2e, m2eta = -2.f * ac.eta_a, zeta = (float)ac.zeta;
  const Vec3 uj = v3(aj), uk = v3(ak);
  const float ij = dj.w, ik = dk.w;          // 1 / R
  const Vec3 ujt = ij * (v3(dj) - bj.w * uj), ukt = ik * (v3(dk) - bk.w * uk);
  const float chat = dot(uj, uk), chatt = dot(ujt, uk) + dot(uj, ukt);
  const float c = ac.cos_scale * chat;
  const float sn = fmaxf(sin_theta(aj, ak, chat, ac.cos_scale), 1e-6f);
  const float sp = ac.cos_scale == 1.f ? sn : fmaxf(sin_theta(aj, ak, chat, 1.f), 1e-6f);
  const float isp = 1.f / sp;
  // the unit vectors normal to u_j and u_k in their plane (dp/dr_j = -ej / R_j) and
  // their tangents, and the tangent of p
  const Vec3 ej = isp * (uk - chat * uj), ek = isp * (uj - chat * uk);
  const Vec3 wjt = ukt - chatt * uj - chat * ujt, wkt = ujt - chatt * uk - chat * ukt;
  const float st = dot(wjt, ej);                     // tangent of sin p
  const Vec3 ejt = isp * (wjt - st * ej), ekt = isp * (wkt - dot(wkt, ek) * ek);
  const float pt = fabsf(chat) < 0.7f ? -chatt * isp : st / chat;
  const float rr = ac.cos_scale == 1.f ? 1.f : ac.cos_scale * sp / sn;
  const float rd = ac.cos_scale == 1.f ? 0.f : (c / sn) * (1.f - rr * rr);
  float2 F[kNA], dF[kNA], ddF[kNA], qF[kNA], qdF[kNA];
#pragma unroll
  for (int a = 0; a < kNA; ++a) F[a] = dF[a] = ddF[a] = qF[a] = qdF[a] = make_float2(0.f, 0.f);
  const float2 c2 = make_float2(c, c), s2 = make_float2(sn, sn), ms2 = make_float2(-sn, -sn);
  const float2 rr2 = make_float2(rr, rr), rd2 = make_float2(rd, rd), mrr = make_float2(-rr * rr, -rr * rr);
  const float2 zm1 = make_float2(zeta - 1.f, zeta - 1.f);
  const float2* g2 = reinterpret_cast<const float2*>(gb);
  const float2* q2 = reinterpret_cast<const float2*>(qb);
#pragma unroll
  for (int m = 0; m < kNZ / 2; ++m) {
    const float2 cz = reinterpret_cast<const float2*>(ac.cos_z)[m];
    const float2 sz = reinterpret_cast<const float2*>(ac.sin_z)[m];
    const float2 cs = __ffma2_rn(s2, sz, __fmul2_rn(c2, cz));   // cos(theta - theta_z)
    const float2 base = __fadd2_rn(cs, make_float2(1.f, 1.f));
    float2 B1, B2;   // base^(zeta-1), base^(zeta-2)
    if constexpr (ZETA == 32) {
      const float2 p2 = __fmul2_rn(base, base), p4 = __fmul2_rn(p2, p2), p8 = __fmul2_rn(p4, p4);
      const float2 p16 = __fmul2_rn(p8, p8);
      B2 = __fmul2_rn(__fmul2_rn(p16, p8), __fmul2_rn(p4, p2));   // ^30
      B1 = __fmul2_rn(B2, base);
    } else {
      B1 = make_float2(ipow<0>(base.x, ac.zeta - 1), ipow<0>(base.y, ac.zeta - 1));
      B2 = ac.zeta > 1 ? make_float2(ipow<0>(base.x, ac.zeta - 2), ipow<0>(base.y, ac.zeta - 2))
                       : make_float2(0.f, 0.f);
    }
    const float2 B = __fmul2_rn(B1, base);
    const float2 t = __ffma2_rn(c2, sz, __fmul2_rn(ms2, cz));
    const float2 h = __fmul2_rn(rr2, t);
    const float2 hh = __ffma2_rn(rd2, t, __fmul2_rn(mrr, cs));
    const float2 dB = __fmul2_rn(B1, h);
    const float2 ddB = __ffma2_rn(__fmul2_rn(zm1, B2), __fmul2_rn(h, h), __fmul2_rn(B1, hh));
#pragma unroll
    for (int a = 0; a < kNA; ++a) {
      const float2 g = g2[4 * a + m], q = q2[4 * a + m];
      F[a] = __ffma2_rn(g, B, F[a]);
      dF[a] = __ffma2_rn(g, dB, dF[a]);
      ddF[a] = __ffma2_rn(g, ddB, ddF[a]);
      qF[a] = __ffma2_rn(q, B, qF[a]);
      qdF[a] = __ffma2_rn(q, dB, qdF[a]);
    }
  }
  const float rb = 0.5f * (aj.w + ak.w), rbt = 0.5f * (bj.w + bk.w);
  float tc = 0.f, tR = 0.f, tf = 0.f, tct = 0.f, tRt = 0.f, tft = 0.f;
#pragma unroll
  for (int a = 0; a < kNA; ++a) {
    const float f = F[a].x + F[a].y, df = dF[a].x + dF[a].y, ddf = ddF[a].x + ddF[a].y;
    const float ft = fmaf(zeta * pt, df, qF[a].x + qF[a].y);
    const float dft = fmaf(pt, ddf, qdF[a].x + qdF[a].y);
    const float x = rb - ac.shf_a[a];
    const float A = fast_exp2(ca_ * x * x);
    const float At = m2eta * x * A * rbt;
    const float xA = m2eta * x * A, xAt = m2eta * fmaf(m2eta * x, x, 1.f) * A * rbt;
    tf = fmaf(A, f, tf);
    tR = fmaf(xA, f, tR);
    tc = fmaf(A, df, tc);
    tft = fmaf(At, f, fmaf(A, ft, tft));
    tRt = fmaf(xAt, f, fmaf(xA, ft, tRt));
    tct = fmaf(At, df, fmaf(A, dft, tct));
  }
  const float fjk = bj.x * bk.x, fjkt = bj.y * bj.w * bk.x + bj.x * bk.y * bk.w;
  const float kp = -ac.ang_pre * zeta;
  const float S = kp * tc * fjk, St = kp * (tct * fjk + tc * fjkt);          // -dE/dp
  const float TR = 0.5f * ac.ang_pre * tR * fjk, TRt = 0.5f * ac.ang_pre * (tRt * fjk + tR * fjkt);
  tf *= ac.ang_pre;
  tft *= ac.ang_pre;
  const float sj = S * ij, sk = S * ik;
  const float sjt = (St - sj * bj.w) * ij, skt = (St - sk * bk.w) * ik;
  const float rj = TR + tf * bj.y * bk.x, rk = TR + tf * bj.x * bk.y;
  const float cross = bj.y * bk.y;
  const float rjt = TRt + tft * bj.y * bk.x + tf * (bj.z * bj.w * bk.x + cross * bk.w);
  const float rkt = TRt + tft * bj.x * bk.y + tf * (cross * bj.w + bj.x * bk.z * bk.w);
  gj = sj * ej + rj * uj;
  gk = sk * ek + rk * uk;
  gjt = sjt * ej + sj * ejt + rjt * uj + rj * ujt;
  gkt = skt * ek + sk * ekt + rkt * uk + rk * ukt;
}

// The forces and their derivative along (r + e v, dE/dG + e q): one warp per
// centre, one lane per radial edge and per angular pair.  As in k_aev_bwd the pairs
// come in round-robin order and each round adds into its own accumulator copy with
// plain read-add-write; the dE/dG and q blocks of the live species pairs wait in
// shared memory.  It replaces a separate primal backward (the primal terms are
// by-products of the tangent's).  1,500 water atoms: 20 us against 17 us for the
// primal kernel and 91 us for a tangent kernel in dual-number arithmetic with six
// shared-memory float atomics per triplet.
template <int ZETA>
__global__ void __launch_bounds__(kWarps * 32, 3) k_aev_bwd_dual(Ws ws, AevConst ac, VjpBufs vb, int copies) {
  extern __shared__ float4 sm4[];
  __shared__ ListHdr hdrs[kWarps];
  const int w = threadIdx.x >> 5;
  const unsigned lane = threadIdx.x & 31;
  const int p = blockIdx.x * kWarps + w;
  if (p >= ws.totals[0]) return;
  const int cap = ws.cap_a;
  float4* angv = sm4 + (size_t)w * dual_warp_f4(cap, ac.n_pairs, copies);
  float4* angf = angv + cap;                // fc, fc', fc'', Rdot
  float4* angd = angf + cap;                // dv, 1/R
  float4* acc = angd + cap;                 // [copy][neighbour] dE/du, then its tangent
  float4* acct = acc + copies * cap;
  float4* gq = acct + copies * cap;
  uint8_t* spec = reinterpret_cast<uint8_t*>(gq + dual_gq_f4(ac.n_pairs));
  uint8_t* pslot = spec + cap;
  ListHdr& H = hdrs[w];
  const float4 xi = ws.xyzq[p];
  const float4 vi = vb.v_pos[p];
  const SysDev& d = ws.sys[ws.pos_sys[p]];
  const size_t row = (size_t)ws.pos_slot[p] * ac.Dp;
  const float* g_row = ws.dEdG + row;
  const float* q_row = vb.Q + row;
  load_hdr(ws.nb_cnt + (size_t)p * 16, ac.S, lane, &H);
  const int na = H.off_a[ac.S], nr = H.off_r[ac.S];
  const int* lr = ws.nb_r + (size_t)p * ws.cap_r;
  const int* la = ws.nb_a + (size_t)p * ws.cap_a;
  float* grad = reinterpret_cast<float*>(gq);   // radial blocks [S*16], then q
  float* gtan = grad + kMaxSpecies * kNR;
  for (int f = lane; f < ac.S * kNR; f += 32) {
    // (a block without neighbours is not read; its slice may not have been computed)
    const int c = ac.rcol[f >> 4] + (f & 15);
    const bool live = H.off_r[(f >> 4) + 1] > H.off_r[f >> 4];
    grad[f] = live ? g_row[c] : 0.f;
    gtan[f] = live ? q_row[c] : 0.f;
  }
  stage_list(na, la, xi, d, ws, lane, [&](int t, int j, const Geo& g) {
    const float4 vj = vb.v_pos[j];
    const float r = sqrtf(g.dx * g.dx + g.dy * g.dy + g.dz * g.dz);
    const float inv = 1.f / r;
    const float dvx = vj.x - vi.x, dvy = vj.y - vi.y, dvz = vj.z - vi.z;
    float f, df, ddf;
    fcut3(r, ac.rc_a, &f, &df, &ddf);
    angv[t] = make_float4(g.dx * inv, g.dy * inv, g.dz * inv, r);
    angf[t] = make_float4(f, df, ddf, (g.dx * dvx + g.dy * dvy + g.dz * dvz) * inv);
    angd[t] = make_float4(dvx, dvy, dvz, inv);
  });
  for (int t = lane; t < na; t += 32) {
    int s = 0;
    while (s + 1 < ac.S && H.off_a[s + 1] <= t) ++s;
    spec[t] = (uint8_t)s;
    for (int c = 0; c < copies; ++c)
      acc[c * cap + t] = acct[c * cap + t] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncwarp();
  Vec3 fi{0.f, 0.f, 0.f}, fit{0.f, 0.f, 0.f};
  // ---- radial edges
  const float cr_ = -ac.eta_r * kLog2e, m2r = -2.f * ac.eta_r;
  int sr = 0;
  for (int t = lane; t < nr; t += 32) {
    while (H.off_r[sr + 1] <= t) ++sr;
    const int j = lr[t];
    if (!NNP_IN_BOUNDS(ws.status, kSiteBwdNeighbour, j, ws.totals[0])) continue;
    const Geo g = pair_geo(xi, ws.xyzq[j], d);
    const float4 vj = vb.v_pos[j];
    const float r = sqrtf(g.dx * g.dx + g.dy * g.dy + g.dz * g.dz);
    const float inv = 1.f / r;
    const Vec3 u = inv * Vec3{g.dx, g.dy, g.dz};
    const Vec3 dv{vj.x - vi.x, vj.y - vi.y, vj.z - vi.z};
    const float rdot = dot(u, dv);
    float fc, dfc, ddfc;
    fcut3(r, ac.rc_r, &fc, &dfc, &ddfc);
    const float* gs = grad + sr * kNR;
    const float* qs = gtan + sr * kNR;
    // phi = e (m2 x f + f'), its derivative e (m2 x (m2 x f + f') + m2 f + m2 x f' + f'')
    float a = 0.f, at = 0.f, ad = 0.f;
#pragma unroll
    for (int k = 0; k < kNR; ++k) {
      const float x = r - ac.shf_r[k];
      const float e = fast_exp2(cr_ * x * x);
      const float mx = m2r * x;
      const float h = fmaf(mx, fc, dfc);
      const float dh = fmaf(mx, h + dfc, fmaf(m2r, fc, ddfc));
      const float ge = gs[k] * e;
      a = fmaf(ge, h, a);
      ad = fmaf(ge, dh, ad);
      at = fmaf(qs[k] * e, h, at);
    }
    at = fmaf(ad, rdot, at);
    const Vec3 f = a * u, ft = at * u + (a * inv) * (dv - rdot * u);
    atomicAdd(&ws.f_pos[j], make_float4(-f.x, -f.y, -f.z, 0.f));
    atomicAdd(&vb.df_pos[j], make_float4(-ft.x, -ft.y, -ft.z, 0.f));
    fi = fi + f;
    fit = fit + ft;
  }
  __syncwarp();   // the radial blocks' region now takes the angular ones
  // ---- the live species-pair blocks: slot k of the k-th live pair (s <= u) in the
  // order 8 s + u, its dE/dG and q (32 values each, index 8a + z)
  {
    float* gf = reinterpret_cast<float*>(gq);
    int slot = 0;
    for (int s = 0; s < ac.S; ++s) {
      const int cs = H.off_a[s + 1] - H.off_a[s];
      if (!cs) continue;
      for (int u = s; u < ac.S; ++u) {
        const int cu = H.off_a[u + 1] - H.off_a[u];
        if (s == u ? cs < 2 : cu < 1) continue;
        const int f = ac.acol[s * ac.S - s * (s - 1) / 2 + (u - s)] + (int)lane;
        gf[slot * (8 * kBlkF4) + lane] = g_row[f];
        gf[slot * (8 * kBlkF4) + 4 * kBlkF4 + lane] = q_row[f];
        if (lane == 0) pslot[8 * s + u] = pslot[8 * u + s] = (uint8_t)slot;
        ++slot;
      }
    }
  }
  __syncwarp();
  const RoundRobin rr = make_round_robin(na);
  for (int t0 = 0; t0 < rr.n_tri;) {
    const int r0 = rr_round(rr, t0);
    const int t1 = min(min(t0 + 32, (r0 + copies) * rr.h), rr.n_tri);
    const int t = t0 + (int)lane;
    if (t < t1) {
      int r, a, b;
      rr_pair(rr, t, &r, &a, &b);
      if (NNP_IN_BOUNDS(ws.status, kSiteBwdTriplet, a, na) &&
          NNP_IN_BOUNDS(ws.status, kSiteBwdTriplet, b, na)) {
        const float4* blk = gq + pslot[8 * spec[a] + spec[b]] * (2 * kBlkF4);
        Vec3 ga, gb, gat, gbt;
        triplet_dual<ZETA>(ac, angv[a], angv[b], angf[a], angf[b], angd[a], angd[b], blk, blk + kBlkF4,
                           ga, gb, gat, gbt);
        const int o = (r & (copies - 1)) * cap;
        auto add = [](float4* at, const Vec3& v) {
          float4 x = *at;
          x.x += v.x; x.y += v.y; x.z += v.z;
          *at = x;
        };
        add(acc + o + a, ga);
        add(acct + o + a, gat);
        add(acc + o + b, gb);
        add(acct + o + b, gbt);
      }
    }
    __syncwarp();   // the next pass may add into the same accumulators
    t0 = t1;
  }
  for (int t = lane; t < na; t += 32) {
    Vec3 a{0.f, 0.f, 0.f}, at{0.f, 0.f, 0.f};
    for (int c = 0; c < copies; ++c) {
      a = a + v3(acc[c * cap + t]);
      at = at + v3(acct[c * cap + t]);
    }
    const int j = la[t];
    if (NNP_IN_BOUNDS(ws.status, kSiteBwdNeighbour, j, ws.totals[0])) {
      atomicAdd(&ws.f_pos[j], make_float4(-a.x, -a.y, -a.z, 0.f));
      atomicAdd(&vb.df_pos[j], make_float4(-at.x, -at.y, -at.z, 0.f));
    }
    fi = fi + a;
    fit = fit + at;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    fi = fi + Vec3{__shfl_xor_sync(kFull, fi.x, o), __shfl_xor_sync(kFull, fi.y, o), __shfl_xor_sync(kFull, fi.z, o)};
    fit = fit + Vec3{__shfl_xor_sync(kFull, fit.x, o), __shfl_xor_sync(kFull, fit.y, o), __shfl_xor_sync(kFull, fit.z, o)};
  }
  if (lane == 0) {
    atomicAdd(&ws.f_pos[p], make_float4(fi.x, fi.y, fi.z, 0.f));
    atomicAdd(&vb.df_pos[p], make_float4(fit.x, fit.y, fit.z, 0.f));
  }
}

// ---------------------------------------------------------------- weight gradients
constexpr int kWgTile = 64, kWgRows = 8, kWgStages = 4;

__device__ __forceinline__ void cp16(float* dst, const float* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = valid ? 16 : 0;   // 0 source bytes: zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}

// Weight and bias gradients of every layer in one launch, summed over the rows of
// each species:
//   W[o][k] = scale sum_m [X1[m,o] (gE_m Y1[m,k] - Y2[m,k]) - X2[m,o] Y1[m,k]]
//   b[o]    = scale sum_m (gE_m X1[m,o] - X2[m,o])
// and for the output layer w4[k] = scale sum_m (gE_m H3[m,k] - H3'[m,k]).
// blockIdx.x: a 64 x 64 (o, k) tile of a layer (the last one: the output layer);
// y: a group of 128-row tiles; z: the ensemble member.  The row sum is what a
// training batch has most of, so it is what the CTAs split (each adds its partial
// tile to the zeroed output atomically); 8-row slices of X and Y come by cp.async
// in their row-major layout, which is the operand order of a product over rows.
// 1,500 water atoms, 4-species model: 33 us against 3 x 88 us (32 x 32 tiles, every
// CTA over all rows of its species) and 262 us for the output layer (one CTA per
// species); 2,560 atoms of molecules 56 us.
__global__ void __launch_bounds__(256) k_wgrad(WgradArgs a) {
  __shared__ __align__(16) float st[kWgStages][4][kWgRows][kWgTile];
  __shared__ float sg[kWgStages][kWgRows];
  const int total = a.seg_start[a.S] / kRowTile;
  const int rt0 = blockIdx.y * a.group, rt1 = min(rt0 + a.group, total);
  if (rt0 >= rt1) return;
  const int e = blockIdx.z, tile = blockIdx.x, tid = threadIdx.x;
  auto species = [&](int rt) {
    int s = 0;
    while (s + 1 < a.S && rt * kRowTile >= a.seg_start[s + 1]) ++s;
    return s;
  };
  if (tile >= a.tile0[3]) {   // the output layer: 256 columns per CTA and its bias
    const int k = (tile - a.tile0[3]) * 256 + tid;
    for (int rt = rt0; rt < rt1; ++rt) {
      const int s = species(rt), m0 = rt * kRowTile;
      const int rows = min(kRowTile, a.seg_start[s] + a.counts[s] - m0);
      float acc = 0.f;
      if (k < a.h3) {
        const float* h = a.H3 + ((size_t)m0 * a.E + e) * a.h3 + k;
        const float* hd = a.H3d + ((size_t)m0 * a.E + e) * a.h3 + k;
#pragma unroll 8
        for (int m = 0; m < rows; ++m)
          acc += a.gE_row[m0 + m] * h[(size_t)m * a.E * a.h3] - hd[(size_t)m * a.E * a.h3];
      } else if (k == a.h3) {
        for (int m = 0; m < rows; ++m) acc += a.gE_row[m0 + m];
      }
      if (k <= a.h3 && rows > 0) atomicAdd(a.out + ((size_t)e * a.S + s) * a.per_net + a.off4 + k, a.scale * acc);
    }
    return;
  }
  int li = 0;
  while (li < 2 && tile >= a.tile0[li + 1]) ++li;
  const WgradLayer& L = a.layer[li];
  const int nk = (L.n_in + kWgTile - 1) / kWgTile, lt = tile - a.tile0[li];
  const int o0 = lt / nk * kWgTile, k0 = lt % nk * kWgTile;
  const float* src[4] = {L.X1 + (size_t)e * L.x_net, L.X2 + (size_t)e * L.x_net,
                         L.Y1 + (size_t)e * L.y_net, L.Y2 + (size_t)e * L.y_net};
  // loader: thread (half, r, q) copies 16 bytes of row r of X1, X2 or of Y1, Y2
  const int half = tid >> 7, lr = (tid >> 4) & 7, lq = (tid & 15) * 4;
  const int c0 = (half ? k0 : o0) + lq, ld = half ? L.ldy : L.ldx;
  const bool ok_c = c0 < (half ? L.n_in : L.n_out);
  const int ty = tid >> 4, tx = tid & 15;   // outputs o0 + 4 ty + i, k0 + 4 tx + j
  float acc[4][4], accb[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    accb[i] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  }
  // slices of the group's live row tiles, in order
  auto rows_of = [&](int rt) {
    const int s = species(rt);
    return min(kRowTile, a.seg_start[s] + a.counts[s] - rt * kRowTile);
  };
  // a tile whose k slice is zero adds nothing to W; its bias still counts
  auto live = [&](int rt) {
    return !(L.masked && a.tile_mask) || k0 == 0 || ((a.tile_mask[rt] >> (k0 >> 6)) & 1u);
  };
  auto flush = [&](int s) {
    float* base = a.out + ((size_t)e * a.S + s) * a.per_net + L.off;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int o = o0 + 4 * ty + i;
      if (o < L.n_out) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int k = k0 + 4 * tx + j;
          if (k < L.n_in_real)
            atomicAdd(base + (size_t)o * L.n_in_real + (L.feat_of_col ? L.feat_of_col[k] : k), a.scale * acc[i][j]);
          acc[i][j] = 0.f;
        }
        if (k0 == 0 && tx == 0) atomicAdd(base + (size_t)L.n_out * L.n_in_real + o, a.scale * accb[i]);
        accb[i] = 0.f;
      }
    }
  };
  for (int rt = rt0; rt < rt1;) {
    const int s = species(rt);
    for (; rt < rt1 && species(rt) == s; ++rt) {
      const int m0 = rt * kRowTile, rows = rows_of(rt);
      if (rows <= 0 || !live(rt)) continue;
      const int n_sl = (rows + kWgRows - 1) / kWgRows;
      auto load = [&](int sl) {
        const int b = sl % kWgStages, r = sl * kWgRows + lr;
        const bool in = r < rows;
        const size_t m = (size_t)m0 + (in ? r : 0);
        const size_t at = m * ld + (ok_c ? c0 : 0);
        cp16(&st[b][2 * half][lr][lq], (half ? src[2] : src[0]) + at, in && ok_c);
        cp16(&st[b][2 * half + 1][lr][lq], (half ? src[3] : src[1]) + at, in && ok_c);
        if (tid < kWgRows) sg[b][tid] = sl * kWgRows + tid < rows ? a.gE_row[m0 + sl * kWgRows + tid] : 0.f;
      };
#pragma unroll
      for (int i = 0; i < kWgStages - 1; ++i) {
        if (i < n_sl) load(i);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
      }
      for (int sl = 0; sl < n_sl; ++sl) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kWgStages - 2) : "memory");
        __syncthreads();   // slice sl is visible; slice sl - 1 is done with
        if (sl + kWgStages - 1 < n_sl) load(sl + kWgStages - 1);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        const int b = sl % kWgStages;
#pragma unroll
        for (int r = 0; r < kWgRows; ++r) {
          const float4 x1 = *reinterpret_cast<const float4*>(&st[b][0][r][4 * ty]);
          const float4 x2 = *reinterpret_cast<const float4*>(&st[b][1][r][4 * ty]);
          const float4 y1 = *reinterpret_cast<const float4*>(&st[b][2][r][4 * tx]);
          const float4 y2 = *reinterpret_cast<const float4*>(&st[b][3][r][4 * tx]);
          const float g = sg[b][r];
          const float gy[4] = {fmaf(g, y1.x, -y2.x), fmaf(g, y1.y, -y2.y), fmaf(g, y1.z, -y2.z), fmaf(g, y1.w, -y2.w)};
          const float yv[4] = {y1.x, y1.y, y1.z, y1.w};
          const float xv[4] = {x1.x, x1.y, x1.z, x1.w}, xt[4] = {x2.x, x2.y, x2.z, x2.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            accb[i] += fmaf(g, xv[i], -xt[i]);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xv[i], gy[j], fmaf(-xt[i], yv[j], acc[i][j]));
          }
        }
      }
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      __syncthreads();   // the ring is refilled for the next row tile
    }
    flush(s);
  }
}

// dL/dr = d/de F - gE F, in the caller's atom order (zero outside the mask)
__global__ void k_vjp_scatter(Ws ws, VjpBufs vb) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= ws.totals[0]) return;
  const int b = ws.pos_sys[p];
  const SysDev& d = ws.sys[b];
  const int local = ws.pos_src[p] - d.in.in_base;
  const float4 df = vb.df_pos[p], f = ws.f_pos[p];
  const float g = (float)d.in.gE;
  float* out = d.in.dLdR + 3 * (size_t)local;
  out[0] = df.x - g * f.x;
  out[1] = df.y - g * f.y;
  out[2] = df.z - g * f.z;
}

size_t fwd_smem(const Ws& ws) { return (size_t)kWarps * fwd_warp_f4(ws.cap_a, ws.cap_r) * sizeof(float4); }
size_t dual_smem(const Ws& ws, int n_pairs) {
  return (size_t)kWarps * dual_warp_f4(ws.cap_a, n_pairs, dual_copies(ws.cap_a, n_pairs)) * sizeof(float4);
}

}  // namespace

// raise (never lower) the kernels' dynamic shared-memory limits: other handles
// of the process may need larger ones
cudaError_t vjp_set_smem(const Ws& ws) {
  size_t dual = 0;   // depends on the model through the number of accumulator copies
  for (int np = 1; np <= kMaxSpecies * (kMaxSpecies + 1) / 2; ++np) dual = std::max(dual, dual_smem(ws, np));
  const void* fn[4] = {(const void*)k_aev_fwd_vjp<32>, (const void*)k_aev_fwd_vjp<0>,
                       (const void*)k_aev_bwd_dual<32>, (const void*)k_aev_bwd_dual<0>};
  for (int i = 0; i < 4; ++i) {
    const int need = (int)(i < 2 ? fwd_smem(ws) : dual);
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, fn[i]);
    if (e != cudaSuccess) return e;
    if (attr.maxDynamicSharedSizeBytes < need) {
      e = cudaFuncSetAttribute(fn[i], cudaFuncAttributeMaxDynamicSharedMemorySize, need);
      if (e != cudaSuccess) return e;
    }
  }
  return gemm_fp32_ensure_smem();
}

void launch_gather_v(const Ws& ws, const VjpBufs& vb, int n_in, cudaStream_t st) {
  k_gather_v<<<(n_in + 255) / 256, 256, 0, st>>>(ws, vb);
}
void launch_aev_fwd_vjp(const Ws& ws, const AevConst& ac, const VjpBufs& vb, int n_in, cudaStream_t st) {
  const int grid = (n_in + kWarps - 1) / kWarps;
  if (ac.zeta == 32) k_aev_fwd_vjp<32><<<grid, kWarps * 32, fwd_smem(ws), st>>>(ws, ac, vb);
  else k_aev_fwd_vjp<0><<<grid, kWarps * 32, fwd_smem(ws), st>>>(ws, ac, vb);
  if (ws.row_mask) k_fill_vjp<<<(ws.row_cap + 7) / 8, 256, 0, st>>>(ws, ac, vb.U);
}
void launch_aev_bwd_dual(const Ws& ws, const AevConst& ac, const VjpBufs& vb, int n_in, cudaStream_t st) {
  const int grid = (n_in + kWarps - 1) / kWarps, copies = dual_copies(ws.cap_a, ac.n_pairs);
  const size_t sm = dual_smem(ws, ac.n_pairs);
  if (ac.zeta == 32) k_aev_bwd_dual<32><<<grid, kWarps * 32, sm, st>>>(ws, ac, vb, copies);
  else k_aev_bwd_dual<0><<<grid, kWarps * 32, sm, st>>>(ws, ac, vb, copies);
}
void launch_wgrad(WgradArgs a, int row_cap, cudaStream_t st) {
  int tiles = 0;
  for (int i = 0; i < 3; ++i) {
    a.tile0[i] = tiles;
    tiles += ((a.layer[i].n_out + kWgTile - 1) / kWgTile) * ((a.layer[i].n_in + kWgTile - 1) / kWgTile);
  }
  a.tile0[3] = tiles;
  tiles += (a.h3 + 256) / 256;
  // rows per CTA: as few tiles as leave about eight CTAs per SM (fewer atomic adds
  // for large batches, enough CTAs for small ones); y is at most 65535
  const int row_tiles = row_cap / kRowTile;
  a.group = std::max(1, (int)((long long)tiles * a.E * row_tiles / (152 * 8)));
  a.group = std::max(std::min(a.group, 32), (row_tiles + 65534) / 65535);
  k_wgrad<<<dim3(tiles, (row_tiles + a.group - 1) / a.group, a.E), 256, 0, st>>>(a);
}
void launch_vjp_scatter(const Ws& ws, const VjpBufs& vb, int n_in, cudaStream_t st) {
  k_vjp_scatter<<<(n_in + 255) / 256, 256, 0, st>>>(ws, vb);
}

}  // namespace nnp
