// Shared pieces of the adjoint's reverse-stage kernels (CUDA-core form in
// adjoint.cu, tensor-core form in adjoint_tc.cu): the launch arguments and the
// per-face-node device arithmetic of the transposed flux and of the eps
// gradient's impedance-weight terms.
#pragma once
#include "common.cuh"

namespace dgmx {

struct AdjArgs {
  const float *lr_in;  // lambda_r (read)
  float *lr_out;       // k_adj_lift: lr_scale lr + b lu (may alias lr_in, may be null); k_adj_vol: a * lr (may be
                       // null), or with the next lift fused in a * lr + b_next * lu_out (may alias lr_in)
  float lr_scale;      // k_adj_lift: the factor a of the stage reversed before, still to be applied to lr
  const float *lu_in;  // lambda_u (read; null = 0)
  float *lu_out;       // k_adj_vol: lu + dt A^T lr
  float *g;            // face data [6][K][NFF]
  float *g_next;       // k_adj_vol with the next lift fused in: that lift's face data (not g)
  float b_next;        // ... and the b of the stage it belongs to
  const float *u_s;    // stage state (eps gradient; null = no gradient)
  const float *rhs_s;  // A u_s at that stage
  double *grad;        // K, FP64 accumulation of dt <lr, dA/deps u_s>
  const float *geo;
  const float4 *fgeo;
  const int2 *fconn;
  const float *Dn;     // [3][Np][Npad] D_d[i][j]
  const float *LF;     // [Np][NFF] LIFT
  const uint8_t *fmask, *nbrtab, *nbrface;
  const float4 *fcon;  // tensor-core form: [K][4][3] per-face constants of the transposed flux (launch_adj_face_consts)
  int64_t K;
  float alpha, a, b, dt;
};

namespace adj {

// s[e] += v summed over the lanes of the warp that share e: a warp's lanes
// hold a few consecutive element indices, so for each distinct e the warp sums
// its lanes' values (shuffle tree) and one lane adds the sum to shared memory
// (instead of up to 32 lanes adding to one address). Every lane of the warp
// must call it.
__device__ __forceinline__ void add_by_element(float *s, int e, float v) {
  const int lane = threadIdx.x & 31;
  unsigned rest = 0xffffffffu;
  while (rest) {
    const int src = __ffs(rest) - 1;
    const int e0 = __shfl_sync(0xffffffffu, e, src);
    const bool mine = e == e0;
    rest &= ~__ballot_sync(0xffffffffu, mine);
    float sum = mine ? v : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == src && sum != 0.f) atomicAdd(s + e0, sum);
  }
}

__device__ __forceinline__ void cross3(const float *a, const float *b, float *c) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}

// One face node of the reverse stage: the transposed flux Jacobians of both
// sides applied to the owner's face data g and the neighbour's g2 at the
// matching node, acc = what the owner's node receives, and the eps gradient's
// contraction of both sides' face data with the flux's derivatives in the
// owner's impedances (dZ = dZ-/deps, dY = dY-/deps).
//
// With flux_E = zs n x (Z2 dH - alpha n x dE), flux_H = -ys n x (Y2 dE + alpha n x
// dH), dq = q+ - q-, zs = 1/(Z- + Z2), ys = 1/(Y- + Y2), the neighbour sees -n,
// swapped traces and the same zs, ys; (n x .)^T = -(n x .) and (n x n x .)^T =
// n x n x . leave, with D = g - g2, cE = n x D_E, nE = n x cE (cH, nH alike),
//   acc_E = alpha zs nE - n x g2_H - ys Y2 cH
//   acc_H = alpha ys nH + n x g2_E + zs Z2 cE
//   grad  = dZ zs^2 (Z2 dH.cE + alpha dE.nE) - dY ys^2 (Y2 dE.cH - alpha dH.nH):
// six cross products and four inner products where the two sides taken one
// after the other need sixteen cross products. A wall is the case g2 = (-g_E,
// g_H) with the mirrored trace q+ = (-E-, H-). (Misfit and gradients at N=4,
// 48,000 tets, 40 steps: 67.6 -> 65.8 ms.)
struct FaceNode {
  float cE[3], cH[3], nE[3], nH[3];
  __device__ __forceinline__ FaceNode(const float *n, const float *g, const float *g2, float Z2, float Y2, float zs,
                                      float ys, float alpha, float *acc) {
    float dE[3], dH[3], xE[3], xH[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      dE[c] = g[c] - g2[c];
      dH[c] = g[c + 3] - g2[c + 3];
    }
    cross3(n, dE, cE);
    cross3(n, dH, cH);
    cross3(n, cE, nE);
    cross3(n, cH, nH);
    cross3(n, g2, xE);
    cross3(n, g2 + 3, xH);
    const float az = alpha * zs, ay = alpha * ys, yw = ys * Y2, zw = zs * Z2;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc[c] = az * nE[c] - xH[c] - yw * cH[c];
      acc[c + 3] = ay * nH[c] + xE[c] + zw * cE[c];
    }
  }
  __device__ __forceinline__ float gradient(const float *qm, const float *qp, float Z2, float Y2, float zs, float ys,
                                            float alpha, float dZ, float dY) const {
    float hc = 0.f, en = 0.f, ec = 0.f, hn = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float e = qp[c] - qm[c], h = qp[c + 3] - qm[c + 3];
      hc += h * cE[c];
      en += e * nE[c];
      ec += e * cH[c];
      hn += h * nH[c];
    }
    return dZ * zs * zs * (Z2 * hc + alpha * en) - dY * ys * ys * (Y2 * ec - alpha * hn);
  }
};

} // namespace adj

// Tensor-core form of the reverse volume stage (adjoint_tc.cu, N <= 5): the
// transposed curl and lift on tcgen05 in the FP16x3 split. Returns
// cudaErrorNotSupported where it does not apply (order, device).
bool adj_tc_supported(const dg_ctx *ctx);
cudaError_t launch_adj_tc(dg_ctx *ctx, const AdjArgs &a, cudaStream_t s);
// The per-face constants the tensor-core form reads (they depend on eps
// through the impedances; computed once per adjoint call): out is [K][4][3]
// float4 {n, 1/(Z-+Z+)}, {Z+, Y+, 1/(Y-+Y+), connection kind}, {dZ-/deps,
// dY-/deps, neighbour element, 0}.
cudaError_t launch_adj_face_consts(const dg_ctx *ctx, float4 *out, cudaStream_t s);
void adj_tc_free(dg_ctx *ctx);

} // namespace dgmx
