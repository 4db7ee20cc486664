// FP32 path of the per-species networks (paper Eq. 2): a tiled SIMT GEMM with
// fused epilogues, run over 128-row species segments of the AEV matrix (a
// 64-row tile never straddles two species).
//
// Forward per layer: Z = H W^T + b, H' = CELU(Z), D = CELU'(Z) (kept for the
// backward).  The last hidden layer's epilogue also forms the atomic energy
// e = H3 . w4 (the width-1 output layer as a dot product) and delta3 = w4 * D3.
// Backward to the input (dE/dG for the force kernel): delta_{l-1} =
// (delta_l W_l) * D_{l-1}, and dE/dG = delta1 W1 with the ensemble members
// concatenated along K (weights pre-transposed and pre-scaled by 1/E at create).
#include "mlp.cuh"

namespace nnp {

namespace {

constexpr int kThreads = 128;   // 4 warps
constexpr int KS = 16;          // K slice of one ring stage (K is a multiple of 16)
constexpr int NS = 4;           // ring stages (three slices in flight)
constexpr int LD = KS + 4;      // row stride of a staged slice (floats): float4 reads of
                                // consecutive rows hit different banks

__device__ __forceinline__ float celu_f(float z, float alpha, float inv_alpha) {
  return z > 0.f ? z : alpha * (__expf(z * inv_alpha) - 1.f);
}
__device__ __forceinline__ float celu_d(float z, float inv_alpha) {
  return z > 0.f ? 1.f : __expf(z * inv_alpha);
}
// CELU'' from CELU' (z <= 0: exp(z/alpha)/alpha; z > 0: 0)
__device__ __forceinline__ float celu_dd(float dz, float inv_alpha) {
  return dz < 1.f ? dz * inv_alpha : 0.f;
}

__device__ __forceinline__ void cp16(float* dst, const float* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = valid ? 16 : 0;   // 0 source bytes: zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}

__device__ __forceinline__ float comp(const float4& v, int q) {
  return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w;
}

// One output tile of BM = 4 R rows x BN = 32 C columns per CTA: a warp owns R rows,
// a lane the columns lane + 32 j.  16-wide K slices of A and B come by cp.async into
// a ring in their row-major layout (no transpose through registers), and a lane
// reads four k of a row or column as one float4.  All lanes of a warp read the same
// rows of A, so those loads are broadcasts (one shared-memory wavefront each against
// four for a column's): four k cost R + 4 C wavefronts for 4 R C FMA instructions,
// and the FMA pipes bound the kernel.  (With 8 x 4 lanes per warp and 8 x 8 outputs
// per lane the same loads took twice the wavefronts, as many cycles as the FMAs.)
// DUAL multiplies two A operands (a value and its tangent) with the same B, so that
// the force VJP reads each weight once for both and its element-wise steps between
// layers happen in the epilogue.  Sparse AEV rows skip the K slices (kmask) and the
// N tiles (nmask) that are zero or unused in the whole 128-row tile; tiles of padding
// rows only are skipped.  8 networks 1008-256-192-160-1 on 3,072 atoms: L1 383 -> 213 us,
// L2 85 -> 80, L3 68 -> 68, B3 56 -> 53, B2 86 -> 78, B1 453 -> 250 us (before: 64 x 64
// tiles, slices transposed through registers, dense rows); the FMA pipe is 53% active,
// held by the fixed latency of its instructions at 8 to 16 warps per SM.
template <int EPI, bool DUAL, int R, int C>
__global__ void __launch_bounds__(kThreads) k_gemm_fp32(GemmArgs g) {
  constexpr int BM = 4 * R, BN = 32 * C, P = DUAL ? 2 : 1;
  constexpr int kStage = (P * BM + BN) * LD;
  static_assert(BM % 32 == 0 && kRowTile % BM == 0, "loader; a tile stays inside a 128-row tile");
  extern __shared__ __align__(16) float sm[];
  // N tiles fastest: neighbouring CTAs share the rows of A
  const int n_nt = (g.N + BN - 1) / BN;
  const int m0 = (int)(blockIdx.x / n_nt) * BM, n0 = (int)(blockIdx.x % n_nt) * BN;
  const int total = g.seg_start[g.S];
  if (m0 >= total) return;
  if (g.nmask) {   // a tile that touches no live 64-column slice
    const uint32_t span = (2u << (((min(n0 + BN, g.N) - 1) >> 6) - (n0 >> 6))) - 1u;
    if (!((g.nmask[m0 >> 7] >> (n0 >> 6)) & span)) return;
  }
  int s = 0;
  while (s + 1 < g.S && m0 >= g.seg_start[s + 1]) ++s;
  if (m0 >= g.seg_start[s] + g.counts[s]) return;   // padding rows only
  const int e = blockIdx.z;
  const float* A[2] = {static_cast<const float*>(g.A) + (size_t)e * g.a_net,
                       DUAL ? static_cast<const float*>(g.A2) + (size_t)e * g.a_net : nullptr};
  const float* B = static_cast<const float*>(g.B) + e * g.b_e + s * g.b_s;
  const uint32_t km = g.kmask ? g.kmask[m0 >> 7] : ~0u;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int n_k = g.K / KS;
  auto next = [&](int k) {   // the first live slice after k (masks: 64 columns per bit)
    do ++k;
    while (k < n_k && g.kmask && !((km >> (k >> 2)) & 1u));
    return k;
  };
  auto load = [&](int k, int st) {
    float* base = sm + st * kStage + (tid & 3) * 4;
    const int r0 = tid >> 2, kc = k * KS + (tid & 3) * 4;
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int i = 0; i < BM / 32; ++i) {
        const int r = r0 + 32 * i;
        cp16(base + (p * BM + r) * LD, A[p] + (size_t)(m0 + r) * g.lda + kc, true);
      }
#pragma unroll
    for (int i = 0; i < C; ++i) {
      const int r = r0 + 32 * i;
      const bool ok = n0 + r < g.N;
      cp16(base + (P * BM + r) * LD, B + (ok ? (size_t)(n0 + r) * g.ldb + kc : 0), ok);
    }
  };
  // plain form: two partial sums per output, over even and odd k, in packed FP32x2
  // FMAs (half the instructions: the same loop of scalar FMAs lost issue slots to
  // dispatch stalls, B1 343 us against 250); dual form: one sum in the order of k
  constexpr int V = DUAL ? 1 : 2;
  float acc[P][R][C][V];
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < C; ++j)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[p][i][j][v] = 0.f;
  // every iteration commits one group (empty past the end), so "at most NS - 2
  // pending" always means that the slice in use has landed
  int k_use = next(-1), k_load = k_use;
#pragma unroll
  for (int i = 0; i < NS - 1; ++i) {
    if (k_load < n_k) { load(k_load, i); k_load = next(k_load); }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
  for (int it = 0; k_use < n_k; ++it, k_use = next(k_use)) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(NS - 2) : "memory");
    __syncthreads();   // the slice is visible to all; all are done with the one before
    if (k_load < n_k) { load(k_load, (it + NS - 1) % NS); k_load = next(k_load); }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    const float* sa = sm + (it % NS) * kStage + w * R * LD;
    const float* sb = sm + (it % NS) * kStage + (P * BM + lane) * LD;
#pragma unroll
    for (int kk = 0; kk < KS; kk += 4) {
      float4 b[C];
#pragma unroll
      for (int j = 0; j < C; ++j) b[j] = *reinterpret_cast<const float4*>(sb + 32 * j * LD + kk);
      constexpr int RG = 4;   // rows taken together: independent FMAs between dependent ones
#pragma unroll
      for (int p = 0; p < P; ++p)
#pragma unroll
        for (int i0 = 0; i0 < R; i0 += RG) {
          float4 a[RG];
#pragma unroll
          for (int i = 0; i < RG; ++i) a[i] = *reinterpret_cast<const float4*>(sa + (p * BM + i0 + i) * LD + kk);
          if constexpr (DUAL) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
              for (int i = 0; i < RG; ++i)
#pragma unroll
                for (int j = 0; j < C; ++j)
                  acc[p][i0 + i][j][0] = fmaf(comp(a[i], q), comp(b[j], q), acc[p][i0 + i][j][0]);
          } else {
#pragma unroll
            for (int q = 0; q < 4; q += 2)
#pragma unroll
              for (int i = 0; i < RG; ++i)
#pragma unroll
                for (int j = 0; j < C; ++j) {
                  float(&c)[V] = acc[p][i0 + i][j];
                  const float2 r = __ffma2_rn(make_float2(comp(a[i], q), comp(a[i], q + 1)),
                                              make_float2(comp(b[j], q), comp(b[j], q + 1)),
                                              make_float2(c[0], c[V - 1]));
                  c[0] = r.x;
                  c[V - 1] = r.y;
                }
          }
        }
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  // ---- epilogue
  const float alpha = g.alpha, inv_alpha = 1.f / g.alpha;
  float bias[C], w4[C];
  constexpr bool kBias = EPI == kEpiCelu || EPI == kEpiCeluDot;
#pragma unroll
  for (int j = 0; j < C; ++j) {
    const int n = n0 + lane + 32 * j;
    const bool ok = n < g.N;
    bias[j] = kBias && ok ? g.bias[e * g.bias_e + s * g.bias_s + n] : 0.f;
    w4[j] = EPI == kEpiCeluDot && ok ? g.w4[e * g.w4_e + s * g.w4_s + n] : 0.f;
  }
  float* const out = static_cast<float*>(g.out);
  float* const out2 = static_cast<float*>(g.out2);
  constexpr int RI = 4;   // rows whose stored values are read before any is written
#pragma unroll
  for (int i0 = 0; i0 < R; i0 += RI) {
    float ax[RI][C], ax2[RI][C];
    if (EPI == kEpiMul) {
#pragma unroll
      for (int i = 0; i < RI; ++i) {
        const size_t arow = (size_t)(m0 + w * R + i0 + i) * g.ld_aux + (size_t)e * g.aux_net;
#pragma unroll
        for (int j = 0; j < C; ++j) {
          const int n = n0 + lane + 32 * j;
          ax[i][j] = n < g.N ? static_cast<const float*>(g.aux)[arow + n] : 0.f;
          ax2[i][j] = DUAL && n < g.N ? g.aux2[arow + n] : 0.f;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < RI; ++i) {
      const int m = m0 + w * R + i0 + i;
      const size_t row = (size_t)m * g.ldo + (size_t)e * g.out_net;
      float dot = 0.f;
#pragma unroll
      for (int j = 0; j < C; ++j) {
        const int n = n0 + lane + 32 * j;
        if (n >= g.N) continue;
        const size_t o = row + n;
        float v = acc[0][i0 + i][j][0];
        if (!DUAL) v += acc[0][i0 + i][j][V - 1];
        const float vt = acc[P - 1][i0 + i][j][0];   // dual: the tangent
        if (kBias) {
          const float z = v + bias[j];
          const float h = celu_f(z, alpha, inv_alpha), d = celu_d(z, inv_alpha);
          dot = fmaf(h, w4[j], dot);
          if (!DUAL) {
            out[o] = EPI == kEpiCelu ? h : w4[j] * d;
            if (EPI == kEpiCelu) out2[o] = d;
          } else {
            out[o] = h;
            out2[o] = d * vt;
            if (EPI == kEpiCelu) {
              g.out3[o] = d;
              g.out4[o] = vt;
            } else {   // delta3 and its tangent
              g.out3[o] = w4[j] * d;
              g.out4[o] = w4[j] * celu_dd(d, inv_alpha) * vt;
            }
          }
        } else if (EPI == kEpiMul) {
          const float d = ax[i][j];
          out[o] = v * d;
          if (DUAL) out2[o] = v * celu_dd(d, inv_alpha) * ax2[i][j] + vt * d;
        } else {
          out[o] = v;
          if (DUAL) out2[o] = vt;
        }
      }
      if (EPI == kEpiCeluDot) {   // the lanes hold this tile's columns of the row
#pragma unroll
        for (int q = 1; q < 32; q <<= 1) dot += __shfl_xor_sync(0xffffffffu, dot, q);
        if (lane == 0) atomicAdd(g.e_row + (size_t)e * g.e_row_net + m, dot);
      }
    }
  }
}

template <bool DUAL, int R, int C>
constexpr int gemm_smem() {
  return NS * ((DUAL ? 2 : 1) * 4 * R + 32 * C) * LD * (int)sizeof(float);
}

template <int EPI, bool DUAL, int R, int C>
void launch_one(const GemmArgs& g, int row_cap, cudaStream_t st, int n_nets) {
  constexpr int BM = 4 * R, BN = 32 * C;
  const dim3 grid((unsigned)((row_cap + BM - 1) / BM) * ((g.N + BN - 1) / BN), 1, n_nets);
  k_gemm_fp32<EPI, DUAL, R, C><<<grid, kThreads, gemm_smem<DUAL, R, C>(), st>>>(g);
}

// 16 rows per warp (8 and their tangents in the dual form).  The width of a tile is
// the one that pads N least, the widest such for the plain form (fewest loads per
// FMA) and the narrowest for the dual one (training batches have few rows).
constexpr int kRows = 16, kRowsDual = 8;

template <int EPI>
void launch_epi(const GemmArgs& g, int row_cap, cudaStream_t st, int n_nets, bool dual) {
  int c = dual || g.nmask ? 2 : 4;   // (masked N tiles: narrow ones follow the live columns)
  auto padded = [&](int q) { return (g.N + 32 * q - 1) / (32 * q) * q; };
  for (int q = 2; q <= 4; ++q)
    if (padded(q) < padded(c)) c = q;
  if (dual) {
    if (c == 2) launch_one<EPI, true, kRowsDual, 2>(g, row_cap, st, n_nets);
    else if (c == 3) launch_one<EPI, true, kRowsDual, 3>(g, row_cap, st, n_nets);
    else launch_one<EPI, true, kRowsDual, 4>(g, row_cap, st, n_nets);
  } else {
    if (c == 2) launch_one<EPI, false, kRows, 2>(g, row_cap, st, n_nets);
    else if (c == 3) launch_one<EPI, false, kRows, 3>(g, row_cap, st, n_nets);
    else launch_one<EPI, false, kRows, 4>(g, row_cap, st, n_nets);
  }
}

template <int EPI, int C>
cudaError_t allow_smem() {
  cudaError_t e = cudaFuncSetAttribute((const void*)k_gemm_fp32<EPI, false, kRows, C>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       gemm_smem<false, kRows, C>());
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute((const void*)k_gemm_fp32<EPI, true, kRowsDual, C>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem<true, kRowsDual, C>());
}
template <int EPI>
cudaError_t allow_epi() {
  cudaError_t e = allow_smem<EPI, 2>();
  if (e == cudaSuccess) e = allow_smem<EPI, 3>();
  return e == cudaSuccess ? allow_smem<EPI, 4>() : e;
}

void launch_any(const GemmArgs& g, int row_cap, cudaStream_t st, int n_nets, bool dual) {
  switch (g.epi) {
    case kEpiCelu: launch_epi<kEpiCelu>(g, row_cap, st, n_nets, dual); break;
    case kEpiCeluDot: launch_epi<kEpiCeluDot>(g, row_cap, st, n_nets, dual); break;
    case kEpiMul: launch_epi<kEpiMul>(g, row_cap, st, n_nets, dual); break;
    default: launch_epi<kEpiStore>(g, row_cap, st, n_nets, dual); break;
  }
}

}  // namespace

cudaError_t gemm_fp32_ensure_smem() {
  cudaError_t e = allow_epi<kEpiCelu>();
  if (e == cudaSuccess) e = allow_epi<kEpiCeluDot>();
  if (e == cudaSuccess) e = allow_epi<kEpiMul>();
  return e == cudaSuccess ? allow_epi<kEpiStore>() : e;
}

void launch_gemm_fp32(const GemmArgs& g, int row_cap, cudaStream_t st, int n_nets) {
  launch_any(g, row_cap, st, n_nets, false);
}
void launch_gemm_dual(const GemmArgs& g, int row_cap, cudaStream_t st, int n_nets) {
  launch_any(g, row_cap, st, n_nets, true);
}

// The backward to the input after launch_mlp_fp32's forward (whole: every column of
// dE/dG, not only the live slices of sparse rows).  delta2 and delta1 go over H2 and H1.
void launch_mlp_fp32_bwd(const Ws& ws, const MlpDims& md, const MlpWeights& mw, const MlpBufs& mb,
                         float alpha, cudaStream_t st, StageHook* hook, bool whole) {
  const int E = md.E, S = md.S, Dp = md.Dp, h1 = md.h1, h2 = md.h2, h3 = md.h3;
  const int R = ws.row_cap;
  GemmArgs g{};
  g.alpha = alpha;
  g.seg_start = ws.seg_start;
  g.counts = ws.species_count;
  g.S = S;
  // B3: delta2 = (delta3 W3) * D2   (written over H2)
  g.A = mb.d3; g.lda = E * h3; g.a_net = h3;
  g.B = mw.W3T; g.b_s = (long long)h2 * h3; g.b_e = (long long)S * h2 * h3; g.ldb = h3;
  g.N = h2; g.K = h3;
  g.aux = mb.D2; g.ld_aux = E * h2; g.aux_net = h2;
  g.out = mb.H2; g.ldo = E * h2; g.out_net = h2;
  g.epi = kEpiMul;
  if (hook) hook->begin(6);
  launch_gemm_fp32(g, R, st, E);
  if (hook) hook->end();
  // B2: delta1 = (delta2 W2) * D1   (written over H1)
  g.A = mb.H2; g.lda = E * h2; g.a_net = h2;
  g.B = mw.W2T; g.b_s = (long long)h1 * h2; g.b_e = (long long)S * h1 * h2; g.ldb = h2;
  g.N = h1; g.K = h2;
  g.aux = mb.D1; g.ld_aux = E * h1; g.aux_net = h1;
  g.out = mb.H1; g.ldo = E * h1; g.out_net = h1;
  g.epi = kEpiMul;
  if (hook) hook->begin(7);
  launch_gemm_fp32(g, R, st, E);
  if (hook) hook->end();
  // B1: dE/dG = [delta1_e]_e [W1_e / E]_e   (K = E*h1)
  g.A = mb.H1; g.lda = E * h1; g.a_net = 0;
  g.B = mw.W1Tcat; g.b_s = (long long)Dp * E * h1; g.b_e = 0; g.ldb = E * h1;
  g.N = Dp; g.K = E * h1;
  g.out = ws.dEdG; g.ldo = Dp; g.out_net = 0;
  g.epi = kEpiStore;
  g.nmask = !whole && ws.row_mask ? ws.tile_mask : nullptr;
  if (hook) hook->begin(8);
  launch_gemm_fp32(g, R, st, 1);
  if (hook) hook->end();
}

// the six GEMMs of one forward + backward-to-input pass over every species
// (one fused kernel where the network shape has a compiled variant)
void launch_mlp_fp32(const Ws& ws, const MlpDims& md, const MlpWeights& mw, const MlpBufs& mb,
                     float alpha, cudaStream_t st, int* n_launch, StageHook* hook,
                     bool energy_only) {
  if (mlp_fused_supported(md)) {  // one kernel for the whole chain
    if (hook) hook->begin(12);
    launch_mlp_fused(ws, md, mw, mb, alpha, energy_only, st);
    if (hook) hook->end();
    if (n_launch) *n_launch += 1;
    return;
  }
  const int E = md.E, S = md.S, Dp = md.Dp, h1 = md.h1, h2 = md.h2, h3 = md.h3;
  const int R = ws.row_cap;
  GemmArgs g{};
  g.alpha = alpha;
  g.seg_start = ws.seg_start;
  g.counts = ws.species_count;
  g.S = S;
  g.e_row = mb.e_row;
  g.e_row_net = R;
  cudaMemsetAsync(mb.e_row, 0, sizeof(float) * (size_t)E * R, st);
  // L1: all ensemble members at once along N
  g.A = ws.aev; g.lda = Dp; g.a_net = 0;
  g.B = mw.W1cat; g.b_s = (long long)E * h1 * Dp; g.b_e = 0; g.ldb = Dp;
  g.bias = mw.b1cat; g.bias_s = (long long)E * h1; g.bias_e = 0;
  g.N = E * h1; g.K = Dp;
  g.out = mb.H1; g.out2 = mb.D1; g.ldo = E * h1; g.out_net = 0;
  g.epi = kEpiCelu;
  g.kmask = ws.row_mask ? ws.tile_mask : nullptr;
  if (hook) hook->begin(3);
  launch_gemm_fp32(g, R, st, 1);
  if (hook) hook->end();
  g.kmask = nullptr;
  // L2: per member
  g.A = mb.H1; g.lda = E * h1; g.a_net = h1;
  g.B = mw.W2; g.b_s = (long long)h2 * h1; g.b_e = (long long)S * h2 * h1; g.ldb = h1;
  g.bias = mw.b2; g.bias_s = h2; g.bias_e = (long long)S * h2;
  g.N = h2; g.K = h1;
  g.out = mb.H2; g.out2 = mb.D2; g.ldo = E * h2; g.out_net = h2;
  g.epi = kEpiCelu;
  if (hook) hook->begin(4);
  launch_gemm_fp32(g, R, st, E);
  if (hook) hook->end();
  // L3 + output layer as a dot product; delta3 = w4 * CELU'(Z3)
  g.A = mb.H2; g.lda = E * h2; g.a_net = h2;
  g.B = mw.W3; g.b_s = (long long)h3 * h2; g.b_e = (long long)S * h3 * h2; g.ldb = h2;
  g.bias = mw.b3; g.bias_s = h3; g.bias_e = (long long)S * h3;
  g.w4 = mw.w4; g.w4_s = h3; g.w4_e = (long long)S * h3;
  g.N = h3; g.K = h2;
  g.out = mb.d3; g.out2 = nullptr; g.ldo = E * h3; g.out_net = h3;
  g.epi = kEpiCeluDot;
  if (hook) hook->begin(5);
  launch_gemm_fp32(g, R, st, E);
  if (hook) hook->end();
  if (energy_only) {   // no forces wanted: the backward to the input is skipped
    if (n_launch) *n_launch += 4;
    return;
  }
  launch_mlp_fp32_bwd(ws, md, mw, mb, alpha, st, hook, false);
  if (n_launch) *n_launch += 7;
}

}  // namespace nnp
