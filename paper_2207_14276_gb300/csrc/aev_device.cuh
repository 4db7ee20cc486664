// Device code shared by the AEV kernels (aev.cu) and their differentiated forms
// (vjp.cu): distances, cutoffs (Eq. 3), angular factors (Eq. 5), the numbering of
// a centre's pairs, and the per-warp list header.
#pragma once

#include "nnp_internal.cuh"

namespace nnp {

namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kPi = 3.14159265358979f;
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// hardware approximations (relative error of a few 1e-8): square root of the
// squared distance and the sine, reciprocals of distances and of sin(theta)
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// x^e for an integer exponent; compile-time E > 0 unrolls, E == 0 reads e
template <int E>
__device__ __forceinline__ float ipow(float x, int e) {
  if constexpr (E > 0) {
    float r = 1.f, b = x;
#pragma unroll
    for (int k = E; k; k >>= 1) {
      if (k & 1) r *= b;
      if (k > 1) b *= b;
    }
    return r;
  } else {
    float r = 1.f;
    while (e) {
      if (e & 1) r *= x;
      x *= x;
      e >>= 1;
    }
    return r;
  }
}

struct Geo {
  float dx, dy, dz, r;
};

__device__ __forceinline__ Geo pair_geo(const float4& xi, const float4& xj, const SysDev& d) {
  float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
  if (d.in.periodic) {
    float n;
    n = rintf(dx * d.in.inv_box[0]); dx = fmaf(-n, d.in.box_hi[0], dx); dx = fmaf(-n, d.in.box_lo[0], dx);
    n = rintf(dy * d.in.inv_box[1]); dy = fmaf(-n, d.in.box_hi[1], dy); dy = fmaf(-n, d.in.box_lo[1], dy);
    n = rintf(dz * d.in.inv_box[2]); dz = fmaf(-n, d.in.box_hi[2], dz); dz = fmaf(-n, d.in.box_lo[2], dz);
  }
  Geo g;
  g.dx = dx; g.dy = dy; g.dz = dz;
  g.r = sqrt_approx(dx * dx + dy * dy + dz * dz);
  return g;
}

// One lane per entry of a neighbour list: visit(slot, j, geometry) stages entry j.
// A lane takes two entries per pass and issues both gathers before either is used.
// W warps share the list (lane: the thread's number among their 32 W).
template <int W = 1, class Visit>
__device__ __forceinline__ void stage_list(int n, const int* lst, const float4& xi, const SysDev& d,
                                           const Ws& ws, unsigned lane, Visit visit) {
  const float4* xyzq = ws.xyzq;
  for (int t0 = 0; t0 < n; t0 += 64 * W) {
    const int ta = t0 + (int)lane, tb = ta + 32 * W;
    int ja = ta < n ? lst[ta] : -1;
    int jb = tb < n ? lst[tb] : -1;
    if (ja >= 0 && !NNP_IN_BOUNDS(ws.status, kSiteAevNeighbour, ja, ws.totals[0])) ja = -1;
    if (jb >= 0 && !NNP_IN_BOUNDS(ws.status, kSiteAevNeighbour, jb, ws.totals[0])) jb = -1;
    const float4 xa = ja >= 0 ? xyzq[ja] : xi;
    const float4 xb = jb >= 0 ? xyzq[jb] : xi;
    if (ja >= 0) visit(ta, ja, pair_geo(xi, xa, d));
    if (jb >= 0) visit(tb, jb, pair_geo(xi, xb, d));
  }
}

// cosine cutoff (Eq. 3) and its derivative (inv_rc = 1 / rc)
__device__ __forceinline__ float fcut(float r, float rc, float inv_rc) {
  return r < rc ? 0.5f * cospif(r * inv_rc) + 0.5f : 0.f;
}
__device__ __forceinline__ void fcut_both(float r, float rc, float inv_rc, float* f, float* df) {
  if (r < rc) {
    float sn, cs;
    sincospif(r * inv_rc, &sn, &cs);
    *f = 0.5f * cs + 0.5f;
    *df = -0.5f * kPi * inv_rc * sn;
  } else {
    *f = 0.f;
    *df = 0.f;
  }
}

// sin(theta) with theta = acos(k cos_hat): sqrt(1 - k^2 cos_hat^2) written as
// sqrt(|u_j x u_k|^2 + (1 - k^2) cos_hat^2), which keeps full relative accuracy
// for nearly collinear triplets (where 1 - cos^2 cancels)
__device__ __forceinline__ float sin_theta(const float4& a, const float4& b, float chat, float k) {
  const float cx = a.y * b.z - a.z * b.y;
  const float cy = a.z * b.x - a.x * b.z;
  const float cz = a.x * b.y - a.y * b.x;
  const float s2 = cx * cx + cy * cy + cz * cz;
  return sqrt_approx(fmaf(1.f - k * k, chat * chat, s2));
}

// The angular factors of two sections at once (the pair (z, z + 1) of one
// float2): base = 1 + c cos(theta_z) + s sin(theta_z), B = base^zeta, and
// B1 = base^(zeta - 1) where asked for.  Packed FP32x2 multiplies and FMAs (one
// instruction for both sections; each lane is an IEEE FP32 operation).
template <int ZETA>
__device__ __forceinline__ float2 section_pair(const AevConst& ac, int m, float2 c2, float2 s2,
                                               float2* B1 = nullptr) {
  const float2 cz = reinterpret_cast<const float2*>(ac.cos_z)[m];
  const float2 sz = reinterpret_cast<const float2*>(ac.sin_z)[m];
  const float2 base = __ffma2_rn(s2, sz, __ffma2_rn(c2, cz, make_float2(1.f, 1.f)));
  if constexpr (ZETA == 32) {
    const float2 p2 = __fmul2_rn(base, base), p4 = __fmul2_rn(p2, p2), p8 = __fmul2_rn(p4, p4);
    const float2 p = __fmul2_rn(p8, p8);   // ^16
    const float2 B = __fmul2_rn(p, p);
    // base^31 by products: base is 0 where a section lies opposite to a collinear pair
    // (and base^32 / base then 0 times infinity)
    if (B1) *B1 = __fmul2_rn(__fmul2_rn(p, p8), __fmul2_rn(__fmul2_rn(p4, p2), base));
    return B;
  } else {
    const float2 b1 = make_float2(ipow<0>(base.x, ac.zeta - 1), ipow<0>(base.y, ac.zeta - 1));
    if (B1) *B1 = b1;
    return __fmul2_rn(b1, base);
  }
}

// per-warp header: species offsets/counts of the radial and angular lists
struct ListHdr {
  int off_r[kMaxSpecies + 1], off_a[kMaxSpecies + 1];
  unsigned live[2];   // backward kernel: angular blocks with triplets (bit q = block q)
};

// The unordered pairs of n neighbours as rounds of disjoint pairs (the circle
// method of round-robin tournament scheduling).  n even: n - 1 rounds of
// h = n / 2 pairs, round r = (r, n - 1) and (r + i, r - i) mod (n - 1) for
// i = 1 .. h - 1; n odd: n rounds of h = (n - 1) / 2 pairs, (r + i, r - i) mod n
// for i = 1 .. h (neighbour r sits the round out).  Pair t is pair t mod h of
// round t / h; every unordered pair occurs once.
struct RoundRobin {
  int n, m, h, off, n_tri;   // m: the circle's size; off: 1 for odd n
  float inv_h;
};
__device__ __forceinline__ RoundRobin make_round_robin(int n) {
  RoundRobin rr;
  rr.n = n;
  const bool odd = n & 1;
  rr.m = odd ? n : n - 1;
  rr.h = max(odd ? (n - 1) / 2 : n / 2, 1);
  rr.off = odd ? 1 : 0;
  rr.n_tri = n * (n - 1) / 2;
  rr.inv_h = rcp_approx((float)rr.h);
  return rr;
}
// round of pair t.  Exact: t / h is below 512 (kStageCap neighbours), so the estimate is
// within 2e-4 of (t + 0.5) / h, which is at least 0.5 / 256 from a whole number.
__device__ __forceinline__ int rr_round(const RoundRobin& rr, int t) {
  int r = (int)((t + 0.5f) * rr.inv_h);
  return r;
}
__device__ __forceinline__ void rr_pair(const RoundRobin& rr, int t, int* round, int* a, int* b) {
  const int r = rr_round(rr, t);
  const int i = t - r * rr.h + rr.off;
  int x = r + i, y = r - i;
  if (x >= rr.m) x -= rr.m;
  if (y < 0) y += rr.m;
  if (i == 0) {   // even n: the fixed neighbour n - 1
    x = r;
    y = rr.n - 1;
  }
  *round = r;
  *a = x;
  *b = y;
}

__device__ __forceinline__ void load_hdr(const uint16_t* hdr, int S, unsigned lane, ListHdr* h) {
  int cr = (lane < (unsigned)S) ? hdr[lane] : 0;
  int ca = (lane < (unsigned)S) ? hdr[8 + lane] : 0;
  int ir = cr, ia = ca;
  for (int o = 1; o < 16; o <<= 1) {
    int u = __shfl_up_sync(kFull, ir, o);
    int v = __shfl_up_sync(kFull, ia, o);
    if ((int)lane >= o) { ir += u; ia += v; }
  }
  if (lane <= (unsigned)kMaxSpecies) {
    h->off_r[lane] = ir - cr;
    h->off_a[lane] = ia - ca;
  }
  __syncwarp();
}

// (j, k) of triplet t inside the block of species pair (s, u):
// same species: the t-th pair j < k of c atoms (row-major); else j = t / cu, k = t % cu
__device__ __forceinline__ void decode_pair(int t, int same, int c, int cu, float inv_cu,
                                            int* j, int* k) {
  if (same) {
    const float b = 2.f * c - 1.f;
    int jj = (int)((b - sqrt_approx(fmaxf(b * b - 8.f * t, 0.f))) * 0.5f);
    jj = max(0, min(jj, c - 2));
    if ((jj + 1) * (2 * c - jj - 2) / 2 <= t) ++jj;
    else if (jj * (2 * c - jj - 1) / 2 > t) --jj;
    *j = jj;
    *k = t - jj * (2 * c - jj - 1) / 2 + jj + 1;
  } else {
    int jj = (int)((t + 0.5f) * inv_cu);
    int kk = t - jj * cu;
    if (kk < 0) { --jj; kk += cu; }
    else if (kk >= cu) { ++jj; kk -= cu; }
    *j = jj;
    *k = kk;
  }
}

// after the call lane l holds the warp sum of v[l]
__device__ __forceinline__ float transpose_reduce32(float (&v)[32], unsigned lane) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float send = up ? v[i] : v[i + o];
      const float keep = up ? v[i + o] : v[i];
      v[i] = keep + __shfl_xor_sync(kFull, send, o);
    }
  }
  return v[0];
}

// The 64-column slices of a centre's AEV row that hold a block with any term:
// radial block s (columns 16 s ..) when the centre has neighbours of species s,
// angular block q of species pair (s, u) (columns 16 S + 32 q ..) when it has a
// pair j < k of those species; bit 0 is always set.  All other slices of the row
// are zero.  The same value on every lane.
// pair_su[q] = s | u << 4 for species pair q (s <= u, upper triangle row-major)
__device__ __forceinline__ void fill_pair_table(uint8_t* pair_su, const AevConst& ac) {
  for (int q = threadIdx.x; q < ac.n_pairs; q += blockDim.x) {
    int sp = 0, rem = q;
    while (rem >= ac.S - sp) { rem -= ac.S - sp; ++sp; }
    pair_su[q] = (uint8_t)(sp | ((sp + rem) << 4));
  }
}

__device__ __forceinline__ uint32_t row_slices(const ListHdr& H, const AevConst& ac, unsigned lane,
                                               const uint8_t* pair_su) {
  uint32_t m = 1u;
  if ((int)lane < ac.S && H.off_r[lane + 1] > H.off_r[lane]) m |= 1u << (ac.rcol[lane] >> 6);
  for (int q = (int)lane; q < ac.n_pairs; q += 32) {
    const int sp = pair_su[q] & 15, u = pair_su[q] >> 4;
    const int cs = H.off_a[sp + 1] - H.off_a[sp], cu = H.off_a[u + 1] - H.off_a[u];
    if (sp == u ? cs >= 2 : (cs > 0 && cu > 0)) {
      const int f0 = ac.acol[q];
      m |= (1u << (f0 >> 6)) | (1u << ((f0 + 31) >> 6));
    }
  }
  return __reduce_or_sync(kFull, m);
}

// whether a block of `width` columns from f0 touches a slice of mask m
__device__ __forceinline__ bool block_in(uint32_t m, int f0, int width) {
  const int a = f0 >> 6, b = (f0 + width - 1) >> 6;
  return (m >> a) & 1u || (m >> b) & 1u;
}

}  // namespace

}  // namespace nnp
