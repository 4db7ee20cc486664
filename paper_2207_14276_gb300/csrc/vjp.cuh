// Buffers and launchers of the force vector-Jacobian product (double backward).
#pragma once

#include "nnp_internal.cuh"

namespace nnp {

struct VjpBufs {
  float4* v_pos;    // [n_in] dL/dF in packed order
  float4* df_pos;   // [n_in] d/de F in packed order
  float* gE_row;    // [rows] dL/dE of each row's system
  float* U;         // [rows][Dp] AEV tangent u = J v
  float* Q;         // [rows][Dp] q = H_e u
  float *H1, *D1, *Z1d, *H1d;   // [rows][E*h1]
  float *H2, *D2, *Z2d, *H2d;   // [rows][E*h2]
  float *H3, *H3d;              // [rows][E*h3]
  float *dl1, *dl1d;
  float *dl2, *dl2d;
  float *dl3, *dl3d;
  float* e_row;     // [E][rows]
};

// One layer of the weight-gradient launch: X (deltas and their tangents) against
// Y (the layer's inputs and their tangents)
struct WgradLayer {
  const float *X1, *X2;
  int ldx, x_net;
  const float *Y1, *Y2;
  int ldy, y_net;
  int n_out, n_in, n_in_real;   // n_in_real: columns of W (the rest is padding)
  long long off;                // of W within a network's flat parameters
  const int16_t* feat_of_col;   // first layer: paper index of the feature of AEV column k
  int masked;                   // Y holds sparse AEV rows: skip a tile's dead slices
};

struct WgradArgs {
  WgradLayer layer[3];
  int tile0[4];                 // first tile of each layer; [3]: the output layer's
  const float *H3, *H3d;        // output layer: [rows][E*h3]
  int h3;
  long long off4;
  int S, E;
  float scale;
  float* out;
  long long per_net;
  const int* seg_start;
  const int* counts;
  const float* gE_row;
  const uint32_t* tile_mask;    // null: dense rows
  int group;                    // 128-row tiles per CTA
};

cudaError_t vjp_set_smem(const Ws& ws);
void launch_gather_v(const Ws& ws, const VjpBufs& vb, int n_in, cudaStream_t st);
// the AEV rows (FP32) and their tangents along v
void launch_aev_fwd_vjp(const Ws& ws, const AevConst& ac, const VjpBufs& vb, int n_in, cudaStream_t st);
// forces and their tangents
void launch_aev_bwd_dual(const Ws& ws, const AevConst& ac, const VjpBufs& vb, int n_in, cudaStream_t st);
void launch_wgrad(WgradArgs a, int row_cap, cudaStream_t st);
void launch_vjp_scatter(const Ws& ws, const VjpBufs& vb, int n_in, cudaStream_t st);

}  // namespace nnp
