// FP32 CUDA-core form of the fused right-hand side / LSERK stage.
//
// One block owns a tile of EB consecutive elements and runs the paper's four
// subtasks (Section 2, Fig. dg-subtasks) on it without leaving the SM, as ONE
// matrix product over the tile's (element, field) rows:
//   out[(e,c), i] = sum_k X[k, (e,c)] W[k, i],   W = [LIFT^T; D^T],
// where the curl is taken before the differentiation: for node j and direction
// d the row (e, c) of X holds the two-field combination sum_l +-(dr_d/dx_l) u_l
// whose derivative along d belongs to component c of curl H or -curl E (eq.
// dg-reference-matrices; the metric terms are constant per element), and for
// the lifting it holds the face node's flux. All products go into the same
// accumulators (24 per element and node quad, where three derivatives of six
// fields take 72), so a thread can hold two elements x two node quads and
// reads 12 X and 8 W values per 96 multiply-adds.
//
// X is built chunk by chunk in shared memory, [k][row] with rows e * 6 + c: the
// fluxes of FR face nodes, then QC node quads times three directions. W is
// staged beside it by asynchronous copies from L2 that run while X is built:
// read through L1 instead, a 16-byte load that several lanes share costs up to
// 8 data-pipe cycles (from shared memory two), and the operators crowd the
// neighbours' traces out of L1.
//
// What bounds it: at N >= 4 the FP32 pipe (53-57% of its cycles busy; packed
// FMAs with operands from shared memory reach 80-85% in isolation) and the
// latencies of the traces and of the update that the blocks of an SM do not
// cover for each other; at N <= 3 those latencies. Measured (us per stage
// before, with three derivatives per field and the operators read through L1,
// and now): N=1 162,000 tets 48.8 -> 34.0; N=2 131,712 tets 119 -> 73; N=3
// 131,712 tets 203 -> 145; N=4 82,944 tets 298 -> 206; N=5 82,944 tets 479 ->
// 395; N=6 24,576 tets 292 -> 227; N=7 24,576 tets 522 -> 422; N=8 24,576 tets
// 859 -> 685; N=9 10,368 tets 668 -> 507; 162 tets at N=3 14.8 -> 6.6, 1,296
// tets at N=5 21.1 -> 14.6. A 36-element tile at N=5 takes 110k cycles, three
// blocks sharing the SM: flux build 26k, products 44k, volume build 16k, update
// 13k, face data 5k, barriers and operator copies 7k.
//
// The shape of two elements per thread sits at its limit of 168 registers and
// spills a little in the update (bytes stored / loaded): 8-24 / 16-40, the store
// form of the gradients' forward sweeps 104-152 / 112-276, the ensemble's tiles at
// N = 4 and 7 40-60 / 60-72; the shapes of one element per thread spill nothing.
#pragma once
#include <atomic>
#include <cmath>

#include "common.cuh"
#include "flux.cuh"
#include "tiles.cuh"

namespace dgmx {

// Shape of a launch: elements per tile and products per thread, RE elements x
// CQ node quads (6 RE x 4 CQ accumulators).
//   ONE: one element x one quad and few, long chunks. A thread's chain of
//     products and a tile's chain of barriers are short, which is what counts
//     while a launch has only a few tiles per SM; at N <= 3 and N = 6 it is
//     faster than TWO at every size.
//   ONE_WIDE: the same with two or more times the elements per block (the rule is
//     at simt_shape; at N = 4 the ensembles' tuner alone has it): more elements per
//     SM in one round (N = 3: 100 instead of 96, N = 4: 56 instead of 48, N = 5: 36
//     instead of 32), one copy of the operators for all of them.
//   TWO: two elements x two quads: half the shared-memory reads per product, but
//     a tile takes as long with one element as with all of them.
enum SimtShapeKind { SHAPE_TWO = 0, SHAPE_ONE = 1, SHAPE_ONE_WIDE = 2 };
template <int N, int SHAPE>
struct SimtShape {
  using D = Dims<N>;
  static constexpr bool ONE = SHAPE != SHAPE_TWO;
  static constexpr int RE = ONE ? 1 : 2, CQ = ONE ? 1 : 2;
  static constexpr int CG = (D::NQ + CQ - 1) / CQ; // column groups: node quads cg and (CQ = 2) cg + CG
  // element groups of a block (even: neighbouring lanes hold two of them)
  static constexpr int GROUPS = SHAPE == SHAPE_TWO        ? 128 / CG / 2 * 2
                                : SHAPE == SHAPE_ONE_WIDE ? (N == 3 ? 50 : N == 4 ? 28 : N == 5 ? 18 : N == 7 ? 16 : N == 8 ? 12 : 8)
                                : N == 1 ? 64 : N <= 3 ? 32 : N == 4 ? 16 : N == 6 ? 12 : N == 8 ? 6 : N == 9 ? 4 : 8;
  static constexpr int EB = RE * GROUPS;
  // Rows of X per chunk: FR face nodes (even, a divisor of 4 Nfp) or QC node
  // quads (12 rows each).
  static constexpr int FR = ONE ? (N == 9 ? 44 : N == 8 ? 60 : N == 7 ? 72 : D::NFF)
                                  : N == 9 ? 44 : N == 8 ? 60 : N == 7 ? 72 : N == 5 ? 42 : 30;
  static constexpr int QC = ONE ? (N == 9 ? 5 : N == 8 ? 7 : N == 7 ? 6 : N == 6 || N == 5 ? 7 : D::NQ)
                                  : N == 9 ? 4 : N == 8 ? 5 : N == 7 ? 6 : N == 5 ? 4 : 2;
};

// Orders without the two-element shape, and those whose single-mesh launches have
// the wide one.
template <int N>
constexpr bool simt_one_only() {
  return N <= 3 || N == 6;
}
template <int N>
constexpr bool simt_has_wide() {
  return N == 3 || N == 5 || N >= 7;
}

template <int N, int SHAPE, int EB_ = SimtShape<N, SHAPE>::EB>
struct SimtCfg {
  using D = Dims<N>;
  using S = SimtShape<N, SHAPE>;
  static constexpr int EB = EB_;
  static_assert(EB % (2 * S::RE) == 0 && EB <= S::EB, "whole pairs of element groups");
  static constexpr int QC = S::QC, FR = S::FR, CG = S::CG;
  static_assert(D::NFF % FR == 0 && FR % 2 == 0, "whole chunks of face nodes, an even number of rows");
  static constexpr int NT = EB / S::RE * CG > 128 ? (EB / S::RE * CG + 31) / 32 * 32 : 128; // threads per block
  // Row stride of X: an odd multiple of 4 floats (16-byte loads along the rows
  // are aligned, the stores of neighbouring nodes fall into different banks)
  static constexpr int RS = (6 * EB) % 8 == 4 ? 6 * EB : 6 * EB + 4;
  static constexpr int WS = D::NPP;                      // row stride of the staged operator
  static constexpr int XR = 12 * QC > FR ? 12 * QC : FR; // rows of X
  // bytes: X and the operator rows of the chunk, face data of the tile, metric
  // terms, reference values, node tables
  static constexpr int OFF_W = XR * RS * 4;
  static constexpr int OFF_FGEO = OFF_W + XR * WS * 4; // float4 [EB * 4]
  static constexpr int OFF_FMAT = OFF_FGEO + EB * 64;  // float4 [EB * 4]
  static constexpr int OFF_FCONN = OFF_FMAT + EB * 64; // int2 [EB * 4]
  static constexpr int OFF_G = OFF_FCONN + EB * 32;    // float [EB][GS]
  static constexpr int GS = 12;                        // row stride of the metric terms
  static constexpr int OFF_REF = OFF_G + EB * GS * 4;  // float [EB][6]
  static constexpr int OFF_TAB = OFF_REF + EB * 24;
  static constexpr size_t SMEM = size_t(OFF_TAB + (100 * D::NFP + 15) / 16 * 16);
  // blocks per SM asked for: three of 168 registers per thread, or (one element per
  // thread) as many of 128 as shared memory holds
  static constexpr int FIT = int(228 * 1024 / (SMEM + 1024)) < 512 / NT ? int(228 * 1024 / (SMEM + 1024)) : 512 / NT > 0 ? 512 / NT : 1;
  static constexpr int MINB = S::ONE ? FIT : 3;
  static_assert(SMEM <= 228 * 1024 / MINB - 1024, "MINB blocks per SM");
};

// Field loads. Tile rows come from L2 past L1 (used once or twice); the face
// nodes' scattered reads hit the same lines again and go through L1, as plain
// loads (the previous stage writes these rows while this one is resident: see
// ld4). The load is written out: volatile, it stays behind griddepcontrol.wait,
// and unlike a C++ load it need not keep its place among the stores (us per stage
// as a C++ load and so: N=6 60,000 tets 550 -> 541, N=8 1,900 tets 71.1 -> 70.0). A
// persistent multi-stage launch (COHERENT) reads everything from L2: other
// blocks wrote the data in an earlier stage.
__device__ __forceinline__ float4 load_field4(const float *p) { return __ldcg(reinterpret_cast<const float4 *>(p)); }
template <bool COHERENT>
__device__ __forceinline__ float load_trace(const float *p) {
  if constexpr (COHERENT) return __ldcg(p);
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// The node tables of a block (once per launch; the first tile's barrier orders them).
template <class Cfg>
__device__ __forceinline__ void simt_setup(const StageArgs &a, float4 *smem4) {
  using D = typename Cfg::D;
  uint8_t *tab = reinterpret_cast<uint8_t *>(smem4) + Cfg::OFF_TAB;
  for (int i = threadIdx.x; i < D::NFF + kConnKinds * D::NFP; i += Cfg::NT)
    tab[i] = i < D::NFF ? a.fmask[i] : a.nbrtab[i - D::NFF];
}

template <int BYTES>
__device__ __forceinline__ void cp_async(void *dst, const void *src) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// kc contiguous operator rows into shared memory, asynchronously.
template <class Cfg>
__device__ __forceinline__ void simt_stage_operator(float *s_w, const float *__restrict__ w, int kc) {
  for (int i = threadIdx.x; i < kc * Cfg::D::NQ; i += Cfg::NT) cp_async<16>(s_w + 4 * i, w + 4 * i);
}

// acc[p][n] += (X[k][2p], X[k][2p+1]) W[k][n] over kc rows k (kc even): packed
// FP32 pairs along the rows, the operator value broadcast to both halves. The
// operands of the next row are requested before the current row's products.
template <class Cfg>
__device__ __forceinline__ void simt_product(float2 (&acc)[3 * Cfg::S::RE][4 * Cfg::S::CQ], const float *x,
                                             const float *w, int kc) {
  constexpr int RE = Cfg::S::RE, CQ = Cfg::S::CQ;
  float2 x0[3 * RE], x1[3 * RE];
  float4 w0[CQ], w1[CQ];
  auto load = [&](float2 (&xv)[3 * RE], float4 (&wv)[CQ]) {
#pragma unroll
    for (int h = 0; h < CQ; ++h) wv[h] = *reinterpret_cast<const float4 *>(w + 4 * Cfg::CG * h);
    if constexpr (RE == 2) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const float4 v = *reinterpret_cast<const float4 *>(x + 4 * i);
        xv[2 * i] = make_float2(v.x, v.y), xv[2 * i + 1] = make_float2(v.z, v.w);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 3; ++i) xv[i] = *reinterpret_cast<const float2 *>(x + 2 * i);
    }
    w += Cfg::WS;
    x += Cfg::RS;
  };
  auto product = [&](const float2 (&xv)[3 * RE], const float4 (&wv)[CQ]) {
#pragma unroll
    for (int n = 0; n < 4 * CQ; ++n) {
      const float4 q = wv[n / 4];
      const float wn = n % 4 == 0 ? q.x : n % 4 == 1 ? q.y : n % 4 == 2 ? q.z : q.w;
#pragma unroll
      for (int p = 0; p < 3 * RE; ++p) acc[p][n] = f2fma(xv[p], f2(wn), acc[p][n]);
    }
  };
  load(x0, w0);
#pragma unroll 1
  for (int k = 2; k < kc; k += 2) {
    load(x1, w1);
    product(x0, w0);
    load(x0, w0);
    product(x1, w1);
  }
  load(x1, w1);
  product(x0, w0);
  product(x1, w1);
}

// One tile of ne <= EB elements starting at k0 (all threads of the block call
// it); staged: the first chunk's operator rows are on their way already.
template <int N, int MODE, class Cfg, bool COHERENT>
__device__ __forceinline__ void simt_stage_tile(const StageArgs &a, int64_t k0, int ne, uint8_t *smem, bool staged = false) {
  using D = Dims<N>;
  constexpr int NP = D::NP, NFP = D::NFP, NPP = D::NPP, NQ = D::NQ, QC = Cfg::QC, FR = Cfg::FR, NT = Cfg::NT;
  constexpr int RS = Cfg::RS, CG = Cfg::CG, RE = Cfg::S::RE, CQ = Cfg::S::CQ;
  float *s_x = reinterpret_cast<float *>(smem), *s_w = reinterpret_cast<float *>(smem + Cfg::OFF_W); // [XR][RS], [XR][WS]
  float4 *s_fgeo = reinterpret_cast<float4 *>(smem + Cfg::OFF_FGEO);
  float4 *s_fmat = reinterpret_cast<float4 *>(smem + Cfg::OFF_FMAT);
  int2 *s_fconn = reinterpret_cast<int2 *>(smem + Cfg::OFF_FCONN);
  float *s_g = reinterpret_cast<float *>(smem + Cfg::OFF_G); // [EB][GS]
  float *s_ref = reinterpret_cast<float *>(smem + Cfg::OFF_REF); // [EB][6]
  const uint8_t *s_fm = smem + Cfg::OFF_TAB, *s_nb = s_fm + D::NFF;
  const int tid = threadIdx.x;
  const int64_t KN = a.K * NPP;
  const float *u0 = a.u + k0 * NPP;

  if (!staged) simt_stage_operator<Cfg>(s_w, a.LT, FR);
  for (int i = tid; i < ne * 4; i += NT) {
    cp_async<16>(s_fgeo + i, a.fgeo + k0 * 4 + i);
    cp_async<16>(s_fmat + i, a.fmat + k0 * 4 + i);
    cp_async<8>(s_fconn + i, a.fconn + k0 * 4 + i);
  }
  for (int i = tid; i < 3 * ne; i += NT) {
    const int e = i / 3, t = i - e * 3;
    cp_async<16>(s_g + e * Cfg::GS + 4 * t, a.geo + (k0 + e) * G_STRIDE + 4 * t);
  }
  // the tile's fields (and residual), on their way to L2
  for (int c = 0; c < 6; ++c)
    for (int i = tid * 32; i < ne * NPP; i += NT * 32) {
      asm volatile("prefetch.global.L2 [%0];" ::"l"(u0 + c * KN + i));
      if (MODE != MODE_RHS && a.rk_a != 0.f) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.res + c * KN + k0 * NPP + i));
    }
  cp_async_wait();
  __syncthreads();

  // element group and column group of this thread: neighbouring lanes share the
  // column group (a 16-byte shared-memory load takes two cycles where lanes l
  // and l ^ 1 read one address, four to six otherwise)
  const int rg = (tid >> 1) / CG * 2 + (tid & 1), cg = (tid >> 1) % CG;
  const bool worker = RE * rg < ne && RE * rg < Cfg::EB;
  const float *xr = s_x + 6 * RE * rg, *wr = s_w + 4 * cg;
  float2 acc[3 * RE][4 * CQ];
#pragma unroll
  for (int p = 0; p < 3 * RE; ++p)
#pragma unroll
    for (int n = 0; n < 4 * CQ; ++n) acc[p][n] = make_float2(0.f, 0.f);

  // Each field's mean over the element's vertices (see the volume term), or at
  // N <= 3, where four scattered loads cost 2-3% of a stage, over its first
  // four nodes. Taken after the first traces: by then the prefetched rows are
  // in L2. With one chunk of face nodes the loads go ahead of the traces.
  constexpr int RIT = (6 * Cfg::EB + NT - 1) / NT;
  auto reference_nodes = [&](int i) {
    const float *v = u0 + (i % 6) * KN + (i / 6) * NPP;
    if constexpr (N <= 3) return load_field4(v);
    else return make_float4(__ldcg(v), __ldcg(v + N), __ldcg(v + NFP - 1), __ldcg(v + NP - 1));
  };
  float4 rn[RIT];
  if constexpr (FR == D::NFF) {
#pragma unroll
    for (int t = 0; t < RIT; ++t)
      if (tid + t * NT < 6 * ne) rn[t] = reference_nodes(tid + t * NT);
  }

  // ---- flux gather and lifting, FR face nodes of every element at a time:
  // both traces from L2, the mirror state on walls; upwind flux with the
  // face's weights. The loads of B face nodes are in flight together.
#pragma unroll 1
  for (int r0 = 0; r0 < D::NFF; r0 += FR) {
    if (r0) __syncthreads(); // the previous product has read X and the operator rows
    if (r0) simt_stage_operator<Cfg>(s_w, a.LT + r0 * NPP, FR);
    const int items = ne * FR;
    constexpr int B = 2;
#pragma unroll 1
    for (int it0 = tid; it0 < items; it0 += B * NT) {
      float qm[B][6], qp[B][6];
      bool wall[B];
#pragma unroll
      for (int i = 0; i < B; ++i) {
        const int it = it0 + i * NT, e = it / FR, r = it - e * FR, fm = r0 + r, f = fm / NFP;
        wall[i] = false;
        if (it < items) {
          const int2 cn = s_fconn[e * 4 + f];
          const float *um = u0 + e * NPP + s_fm[fm], *up = um;
          wall[i] = cn.y == kBoundaryConn;
          if (!wall[i]) up = a.u + int64_t(cn.x) * NPP + s_nb[cn.y * NFP + fm - f * NFP];
#pragma unroll
          for (int c = 0; c < 6; ++c) qm[i][c] = load_trace<COHERENT>(um + c * KN);
#pragma unroll
          for (int c = 0; c < 6; ++c) qp[i][c] = load_trace<COHERENT>(up + c * KN);
        }
      }
#pragma unroll
      for (int i = 0; i < B; ++i) {
        const int it = it0 + i * NT, e = it / FR, r = it - e * FR, fm = r0 + r, f = fm / NFP;
        if (it >= items) break;
        if (wall[i]) {
#pragma unroll
          for (int c = 0; c < 3; ++c) qp[i][c] = -qm[i][c];
        }
        float fl[6];
        maxwell_flux_w(s_fgeo[e * 4 + f], qm[i], qp[i], s_fmat[e * 4 + f], a.alpha, fl);
        float2 *d = reinterpret_cast<float2 *>(s_x + r * RS + e * 6);
        d[0] = make_float2(fl[0], fl[1]);
        d[1] = make_float2(fl[2], fl[3]);
        d[2] = make_float2(fl[4], fl[5]);
      }
    }
    if (r0 == 0) {
#pragma unroll
      for (int t = 0; t < RIT; ++t) {
        const int i = tid + t * NT;
        if (i >= 6 * ne) break;
        if constexpr (FR < D::NFF) rn[t] = reference_nodes(i);
        s_ref[i] = (0.25f * rn[t].x + 0.25f * rn[t].y) + (0.25f * rn[t].z + 0.25f * rn[t].w);
      }
    }
    cp_async_wait();
    __syncthreads();
    if (worker) simt_product<Cfg>(acc, xr, wr, FR);
  }

  // ---- volume term, QC node quads at a time: the combinations of the curl
  // (d/dx_l = sum_d (dr_d/dx_l) d/dr_d) of every node and direction, then
  // their derivatives. The fields enter as differences from a mean of
  // the element's: D annihilates constants, and without the constant part
  // neither the rounded combinations nor the sums carry its rounding error
  // (right-hand side at N=5 against 64 bits: 1.5e-6 with it, 9.5e-7 with
  // differences from one node, 5.1e-7 now; 8.7e-7 with the combinations taken
  // after the differentiation; N=3: 3.7e-7, 2.5e-7 now and 3.1e-7).
#pragma unroll 1
  for (int q0 = 0; q0 < NQ; q0 += QC) {
    __syncthreads(); // the previous product has read X and the operator rows
    const int qn = NQ - q0 < QC ? NQ - q0 : QC;
    simt_stage_operator<Cfg>(s_w, a.DT + 12 * q0 * NPP, 12 * qn);
    for (int it = tid; it < ne * QC; it += NT) {
      const int e = it / QC, qq = it - e * QC;
      if (qq >= qn) continue;
      const float *up = u0 + e * NPP + 4 * (q0 + qq);
      float4 v4[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) v4[c] = load_field4(up + c * KN);
      float v[6][4];
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const float r = s_ref[e * 6 + c];
        v[c][0] = v4[c].x - r, v[c][1] = v4[c].y - r, v[c][2] = v4[c].z - r, v[c][3] = v4[c].w - r;
        if (NP % 4 != 0 && q0 + qq == NQ - 1) { // padding entries are ignored
#pragma unroll
          for (int n = NP % 4; n < 4; ++n) v[c][n] = 0.f;
        }
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float gx = s_g[e * Cfg::GS + 3 * d], gy = s_g[e * Cfg::GS + 3 * d + 1], gz = s_g[e * Cfg::GS + 3 * d + 2];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const float Ex = v[0][n], Ey = v[1][n], Ez = v[2][n], Hx = v[3][n], Hy = v[4][n], Hz = v[5][n];
          float2 *x = reinterpret_cast<float2 *>(s_x + (3 * (4 * qq + n) + d) * RS + e * 6);
          x[0] = make_float2(gy * Hz - gz * Hy, gz * Hx - gx * Hz); // curl H
          x[1] = make_float2(gx * Hy - gy * Hx, gz * Ey - gy * Ez); //         , -curl E
          x[2] = make_float2(gx * Ez - gz * Ex, gy * Ex - gx * Ey);
        }
      }
    }
    cp_async_wait();
    __syncthreads();
    if (worker) simt_product<Cfg>(acc, xr, wr, 12 * qn);
  }

  // ---- material scaling and output / operator assembly, three fields of an
  // element and node quad at a time (their loads in flight together)
  if (!worker) return;
#pragma unroll
  for (int bt = 0; bt < 2 * RE * CQ; ++bt) { // (element of the group, E or H, quad)
    const int el = bt / (2 * CQ), g = bt / CQ % 2, h = bt % CQ, e = RE * rg + el, q = cg + h * CG;
    if (e >= ne || q >= NQ) continue;
    const float *geo = a.geo + (k0 + e) * G_STRIDE;
    const float w = __ldg(geo + (g ? G_IMU : G_IEPS)), dtk = a.dt_geo ? __ldg(geo + G_DT) : a.dt;
    const int64_t off0 = 3 * g * KN + (k0 + e) * NPP + 4 * q;
    float4 rs[3], uo[3];
    if (MODE != MODE_RHS) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        // the first LSERK4 stage has a = 0: the residual it overwrites is not read
        rs[c] = a.rk_a != 0.f ? load_field4(a.res + c * KN + off0) : make_float4(0.f, 0.f, 0.f, 0.f);
        uo[c] = load_field4(a.u + c * KN + off0);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int64_t off = c * KN + off0;
      const int row = 6 * el + 3 * g + c;
      float r4[4];
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const float2 v = acc[row / 2][4 * h + n];
        r4[n] = (4 * q + n < NP) ? (row % 2 ? v.y : v.x) * w : 0.f;
      }
      if (MODE == MODE_RHS) {
        *reinterpret_cast<float4 *>(a.rhs + off) = make_float4(r4[0], r4[1], r4[2], r4[3]);
      } else {
        float rv[4] = {rs[c].x, rs[c].y, rs[c].z, rs[c].w}, uv[4] = {uo[c].x, uo[c].y, uo[c].z, uo[c].w};
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const bool pad = 4 * q + n >= NP;
          rv[n] = pad ? 0.f : fmaf(a.rk_a, rv[n], dtk * r4[n]);
          uv[n] = pad ? 0.f : fmaf(a.rk_b, rv[n], uv[n]);
        }
        *reinterpret_cast<float4 *>(a.res + off) = make_float4(rv[0], rv[1], rv[2], rv[3]);
        *reinterpret_cast<float4 *>(a.u_out + off) = make_float4(uv[0], uv[1], uv[2], uv[3]);
        // the adjoint's eps gradient reads only the E components of the stage right-hand side
        if (MODE == MODE_LSERK_STORE && g == 0)
          *reinterpret_cast<float4 *>(a.rhs + off) = make_float4(r4[0], r4[1], r4[2], r4[3]);
      }
    }
  }
}

template <int N, int MODE, int SHAPE>
__global__ void __launch_bounds__(SimtCfg<N, SHAPE>::NT, SimtCfg<N, SHAPE>::MINB) k_stage_simt(StageArgs a, TileMap<SimtCfg<N, SHAPE>::EB> tm) {
  using Cfg = SimtCfg<N, SHAPE>;
  extern __shared__ float4 smem4[];
  simt_setup<Cfg>(a, smem4);
  // (the operator is fixed: its first rows may arrive before the previous stage has ended)
  simt_stage_operator<Cfg>(reinterpret_cast<float *>(reinterpret_cast<uint8_t *>(smem4) + Cfg::OFF_W), a.LT, Cfg::FR);
  pdl_wait(); // stage after stage: fields of the previous stage from here on
  for (int t = blockIdx.x; t < tm.ntiles; t += gridDim.x) {
    if (t + int(gridDim.x) >= tm.ntiles) pdl_launch_next(); // this block's last tile
    if (t != int(blockIdx.x)) __syncthreads(); // shared memory of the previous tile is no longer read
    simt_stage_tile<N, MODE, Cfg, false>(a, tm.start(t), tm.size(t, a.K), reinterpret_cast<uint8_t *>(smem4),
                                           t == int(blockIdx.x));
  }
}

// Blocks of a launch with room for `cap`: half of them on small meshes
// (small_mesh_blocks), as far as that gains. It stops gaining at 20 elements per
// tile at N = 1 (us per stage, all blocks and half: 6,080 tets 5.15 -> 4.74, 8,360
// tets 5.33 -> 5.81), and where the larger tile's products take twice the warps: at
// N = 3 beyond 6 elements (1,368 tets 7.40 -> 7.14, 1,482 tets 7.45 -> 8.17), at
// N = 4 where the tiles of all blocks have 2, 6 or 8 elements (798 tets 9.33 ->
// 10.05, 2,622 tets 12.1 -> 13.0; but 1,026 tets 11.4 -> 10.2, 2,964 tets 14.8 ->
// 13.6). At the other orders it gains as far as half of the blocks hold the mesh
// in full tiles (N=2 3,040 tets 7.12 -> 5.88, 7,296 tets 8.76 -> 8.22, though 3,344
// tets 6.62 -> 6.96; N=5 2,432 tets 18.5 -> 15.7; N=8 912 tets 53.7 -> 35.1).
template <int N, class Cfg>
int simt_blocks(int64_t K, int cap) {
  if (N == 4 && (K + cap - 1) / cap % 4 == 2) return cap;
  return small_mesh_blocks<Cfg::EB>(K, cap, N == 1 ? 20 : N == 3 ? 6 : N == 4 ? 14 : Cfg::EB);
}

template <int N, int MODE, int SHAPE>
cudaError_t launch_simt_mode(const StageArgs &a, int dev, int sms, cudaStream_t s) {
  using Cfg = SimtCfg<N, SHAPE>;
  auto kern = k_stage_simt<N, MODE, SHAPE>;
  // the shared-memory opt-in is a per-device function attribute: set it on every launch
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(Cfg::SMEM));
  if (e != cudaSuccess) return e;
  // persistent grid: as many blocks as fit on the GPU at once (at most one per
  // tile); blocks per SM of each kernel cached per device
  constexpr int kDevCache = 64;
  static std::atomic<int> per_sm_cache[kDevCache];
  int per_sm = dev < kDevCache ? per_sm_cache[dev].load(std::memory_order_relaxed) : 0;
  if (per_sm == 0) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, Cfg::NT, Cfg::SMEM);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    if (dev < kDevCache) per_sm_cache[dev].store(per_sm, std::memory_order_relaxed);
  }
  const int cap = simt_blocks<N, Cfg>(a.K, per_sm * sms);
  const TileMap<Cfg::EB> tm = make_tiles<Cfg::EB>(a.K, cap);
  const unsigned blocks = unsigned(tm.ntiles < cap ? tm.ntiles : cap);
  return launch_pdl(kern, dim3(blocks), dim3(Cfg::NT), Cfg::SMEM, s, a, tm);
}

// The two-element shape runs in rounds of one tile per block that take the same
// time however many elements a tile has; the one-element shape's time grows with
// the element count, by simt_round_ratio times a round's time per full round of
// elements (measured, us per round and us per full round's elements in the
// one-element shape: N=4 50 / 61, N=5 63 / 85, N=7 103 / 128, N=8 134 / 181, N=9
// 168 / 228). The first is taken where its rounds cost less.
//
// The wide one-element shape is taken where the narrow one's blocks no longer hold
// the mesh in less than a round: beyond one block per SM at N >= 7, where a
// second one on the SM takes turns with the first, and beyond half of the blocks at
// N = 5, but not with six elements per narrow tile, which fill three warps (us per
// stage, narrow and wide: N=5 2,700 tets 21.4 -> 16.6, 3,300 tets 21.7 -> 23.1, 5,300
// tets 39.8 -> 26.7, 10,500 tets 66.1 -> 49.9; N=7 1,310 tets 39.7 -> 31.5; N=8 1,215
// tets 54.8 -> 43.6, 2,535 tets 111 -> 88; N=9 670 tets 72.5 -> 56.5, 2,590 tets 189 ->
// 170). At N >= 7 not where few elements are left after whole rounds: the narrow
// blocks do those beside other blocks' full tiles (N=8 1,875 tets 69.5, wide 79.2;
// 1,995 tets 92.1, wide 79.6). At N = 3 where it takes one, two or three rounds
// instead of one more (15,000 tets 22.4 -> 17.6, 45,000 tets 53.0 -> 48.5; with eight
// instead of nine 117,000 tets 128 -> 129, and 23,000 tets, two either way, 27.5 ->
// 28.1).
template <int N>
constexpr double simt_round_ratio() {
  return N == 4 ? 1.22 : N == 7 ? 1.24 : 1.35;
}
template <int N>
int simt_shape(int64_t K, int sms) {
  if constexpr (!simt_one_only<N>()) {
    const double rounds = double(K) / (double(SimtCfg<N, SHAPE_TWO>::MINB) * sms * SimtShape<N, SHAPE_TWO>::EB);
    if (std::ceil(rounds) < simt_round_ratio<N>() * rounds) return SHAPE_TWO;
  }
  if constexpr (simt_has_wide<N>()) {
    using One = SimtCfg<N, SHAPE_ONE>;
    using Wide = SimtCfg<N, SHAPE_ONE_WIDE>;
    if (N == 3) {
      const int64_t one = int64_t(One::EB) * One::MINB * sms, wide = int64_t(Wide::EB) * Wide::MINB * sms;
      return (K - 1) / wide < (K - 1) / one && K <= 3 * wide ? SHAPE_ONE_WIDE : SHAPE_ONE;
    }
    const int64_t round = int64_t(One::EB) * (N == 5 ? One::MINB / 2 : 1) * sms;
    const int64_t wide = int64_t(Wide::EB) * sms; // N >= 7: a round of the wide shape
    if (K > round) {
      if (N == 5) return (K - 1) / (int64_t(One::MINB) * sms) + 1 == 6 ? SHAPE_ONE : SHAPE_ONE_WIDE;
      const int64_t left = K % wide;
      if (left == 0 || 2 * left > sms) return SHAPE_ONE_WIDE;
    }
  }
  return SHAPE_ONE;
}

template <int N, int MODE>
cudaError_t launch_simt_shape(const StageArgs &a, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int shape = simt_shape<N>(a.K, sms);
  if constexpr (!simt_one_only<N>())
    if (shape == SHAPE_TWO) return launch_simt_mode<N, MODE, SHAPE_TWO>(a, dev, sms, s);
  if constexpr (simt_has_wide<N>())
    if (shape == SHAPE_ONE_WIDE) return launch_simt_mode<N, MODE, SHAPE_ONE_WIDE>(a, dev, sms, s);
  return launch_simt_mode<N, MODE, SHAPE_ONE>(a, dev, sms, s);
}

template <int N>
cudaError_t launch_simt_order(int mode, const StageArgs &a, cudaStream_t s) {
  if (mode == MODE_RHS) return launch_simt_shape<N, MODE_RHS>(a, s);
  if (mode == MODE_LSERK) return launch_simt_shape<N, MODE_LSERK>(a, s);
  return launch_simt_shape<N, MODE_LSERK_STORE>(a, s);
}

} // namespace dgmx
