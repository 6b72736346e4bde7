// One 128-element tile of the FP64 transport sweep on quadrilaterals with one
// local operator shared by every element (Sec. 3, eqs. transportLocalk1 and
// transportLocale), one thread per element: the thread gathers its element's
// traces at its NQ face points into registers, forms the rows Y = Gy + Hy uhat
// of the two faces it is upwind of (NQ / 2 rows; no point has beta.n = 0),
// writes the new trace there and adds w (uhat^{k+1} - uhat^k)^2 to the residual.
//
// The products run in fixed point on the integer pipe (fixed_point.cuh): the FP64
// pipe, 1.6 operations per clock and SM, bounded the double form (NQ^2 / 2 products
// per element, 200 at p = 4). What is left there is four operations per row: the
// conversion of the result, the increment, its square, the sum. Every load of a tile
// is issued before the first product, so that a small problem waits for memory twice
// (face ids, then all values).
//
// The operator is equilibrated: Hy[j][c] = 2^(s_j + t_a) Hx[j][c], t_a for the columns
// of axis a's faces, s_j for row j, both of either sign, since the columns go with
// |beta_a| / h_a and all entries with dt where that is small. The element's traces
// times 2^t_a are aligned to the largest of them with 56 bits, a row's sum and its Gy
// to the coarser of their units. (One scale for the whole operator, not below one,
// lost 2.6e-13 of a trace at 16 x 16, p = 2, dt = 1e-6, in an element fed from rest;
// the present form 5e-17, an FMA chain 8e-17.)
//
// The residual is reduced per tile (warp sums, then the warps in order) into
// partials[tile]; the tile that takes the last ticket of the sweep adds the
// partials up in a fixed order (lane l sums tiles l, l + 32, ..., then a warp
// butterfly), records r_k and decides whether the loop goes on. The result
// depends on neither the grid nor the order in which tiles run, so the
// single-problem sweep and the batched loop, which both run this code, give
// the same iterates and residuals bit for bit.
#pragma once

#include <cuda_runtime.h>

#include "ehdg_internal.h"
#include "fixed_point.cuh"
#include "sweep_common.cuh"

namespace ehdg {

constexpr int kPeTile = 128;   // elements per tile = threads per block

// Loads of data that other blocks of the same launch write (traces,
// corrections, residuals): CG = true reads through L2 only (a persistent
// launch, where an SM's L1 may hold lines other SMs have rewritten since).
template <bool CG, class T>
__device__ __forceinline__ T pe_ld(const T* p) {
  if constexpr (CG) return __ldcg(p);
  else return *p;
}

struct PeView {
  int64_t nel, nface;
  int own[2];                   // the local faces of the sweep rows: 0 or 1, 2 or 3
  const int32_t* elem_face;     // [4][nel]
  const double* face_jf;        // [nface]
  const double* fw;             // face Gauss weight of each face point
  const double* Gy;             // [slot][nel]
  float* R_out;                 // mixed precision: F(uhat) - uhat at owned points (or null)
  double* partials;             // [tiles]
  IterState* it;
  double* hist;
  int max_iter;
  double tol, res_scale;
  double* uhat;                 // [2][Nqf][nface]
  __host__ __device__ const double* uhat_slot(int s, int64_t tlen) const { return uhat + s * tlen; }
};

// The operator in limbs: the sweep rows in row order, [NQ / 2][NQ], then (t_0, t_1)
// and the NQ / 2 scales of the rows.
__host__ __device__ constexpr int pe_operator_len(int NQ) { return NQ / 2 * NQ + 1 + NQ / 4; }

// Gy + the sum of a row's products, x in units of 2^(unit - 1078) with the row's scale
template <int NQ>
__device__ __forceinline__ double pe_row(const int2* Hrow, const Limb (&x)[NQ], int unit, double gy) {
  const int4* Hr = reinterpret_cast<const int4*>(Hrow);
  Acc t(0);
#pragma unroll
  for (int c = 0; c < NQ; c += 2) {
    const int4 h = Hr[c / 2];
    t.mac(Cfx{h.x, h.y}, x[c]);
    t.mac(Cfx{h.z, h.w}, x[c + 1]);
  }
  const int L = max(unit, max(fx_exponent(gy), 1));
  return fx_value(fx_shift(t.get(), L - unit) + fx_from_double(gy, L), L - 1078);
}

// The tile's sweep; its residual sum goes to partials[tile] (thread 0). Hsh: the
// operator as above (16-byte aligned).
template <int NQ, bool CG>
__device__ __forceinline__ void pe_tile_sweep(const PeView& v, const int2* Hsh, const double* src,
                                              double* dst, int64_t tile) {
  constexpr int NQF = NQ / 4, RN = NQ / 2;
  __shared__ double red[kPeTile / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t ne = v.nel, nface = v.nface;
  const int64_t e = tile * kPeTile + tid;
  double res = 0.0;
  if (e < ne) {
    double u[NQ], gy[RN], w[NQF];
    int64_t face[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) face[f] = v.elem_face[f * ne + e];
#pragma unroll
    for (int j = 0; j < RN; ++j) gy[j] = v.Gy[j * ne + e];
    const int2 tc = Hsh[RN * NQ];
    const int* sc = reinterpret_cast<const int*>(Hsh + RN * NQ + 1);
#pragma unroll
    for (int g = 0; g < NQF; ++g) w[g] = v.fw[g];
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
      for (int g = 0; g < NQF; ++g) u[f * NQF + g] = pe_ld<CG>(src + g * nface + face[f]);
    const int64_t fo[2] = {v.own[0] ? face[1] : face[0], v.own[1] == 3 ? face[3] : face[2]};
    const double jf[2] = {v.face_jf[fo[0]], v.face_jf[fo[1]]};
    int ea[2] = {1, 1}, eg = 1;
#pragma unroll
    for (int c = 0; c < NQ; ++c) ea[c / (2 * NQF)] = max(ea[c / (2 * NQF)], fx_exponent(u[c]));
#pragma unroll
    for (int j = 0; j < RN; ++j) eg = max(eg, fx_exponent(gy[j]));
    const int em = max(ea[0] + tc.x, ea[1] + tc.y);
    double sq[2] = {0.0, 0.0};
    Limb x[NQ];
#pragma unroll
    for (int c = 0; c < NQ; ++c)
      x[c] = fx_split(fx_from_double(u[c], em - (c < 2 * NQF ? tc.x : tc.y)));
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      double acc = pe_row<NQ>(Hsh + j * NQ, x, em + sc[j], gy[j]);
      if (max(max(ea[0], ea[1]), eg) == 0x7ff)   // an input is not finite
        acc = __hiloint2double(0x7ff80000, 0);
      const int b = j / NQF, g = j - b * NQF;
      const int64_t pt = g * nface + fo[b];
      const double old = v.own[b] & 1 ? u[(2 * b + 1) * NQF + g] : u[2 * b * NQF + g];
      const double d = acc - old;
      dst[pt] = acc;
      if (v.R_out) v.R_out[pt] = (float)d;
      sq[b] = fma(w[g], d * d, sq[b]);
    }
    res = fma(jf[0], sq[0], jf[1] * sq[1]);
  }
  res = fsum_warp(res);
  if (lane == 0) red[wid] = res;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
#pragma unroll
    for (int w2 = 0; w2 < kPeTile / 32; ++w2) s += red[w2];
    v.partials[tile] = s;
  }
}

// the sum of all tiles' partials, in warp 0
__device__ __forceinline__ double pe_total(const double* partials, int64_t ntiles) {
  double s = 0.0;
  for (int64_t t = threadIdx.x & 31; t < ntiles; t += 32) s += __ldcg(partials + t);
  return fsum_warp(s);
}

// A tile with its ticket; returns true in the block that did the final reduction.
template <int NQ, bool CG = false>
__device__ __forceinline__ bool pe_tile(const PeView& v, const int2* Hsh, const double* src,
                                        double* dst, int64_t tile, int64_t ntiles, int graph_mode,
                                        cudaGraphConditionalHandle handle) {
  __shared__ bool last;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  pe_tile_sweep<NQ, CG>(v, Hsh, src, dst, tile);
  if (tid == 0) {
    __threadfence();
    last = atomicAdd(&v.it->counter, 1u) == (unsigned int)(ntiles - 1);
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  if (wid == 0) {
    const double s = pe_total(v.partials, ntiles);
    if (lane == 0) {
      IterState* it = v.it;
      const double r = v.res_scale * sqrt(s);
      const int k = it->k;
      if (k < v.max_iter) v.hist[k] = r;
      it->k = k + 1;
      it->r_last = r;
      it->counter = 0u;
      int cont = 1, status = EHDG_OK;
      if (!isfinite(r)) { cont = 0; status = EHDG_ERR_DIVERGED; }
      else if (r < v.tol) { cont = 0; status = EHDG_OK; }
      else if (k + 1 >= v.max_iter) { cont = 0; status = EHDG_ERR_NOT_CONVERGED; }
      it->cont = cont;
      it->status = status;
      __threadfence();
      if (graph_mode) cudaGraphSetConditional(handle, (unsigned int)cont);
    }
  }
  __syncthreads();
  return true;
}

// One 128-element tile of the FP32 correction sweep of mixed precision
// (delta_out = R + S Hy delta_in at the owned points), same shapes, one
// thread per element: the FP32 copy of the operator rows in Hsh32
// [n_rows][NQ], one FMA chain per row.
struct LpPeView {
  int64_t nel, nface;
  int own[2];                   // the local faces of the sweep rows
  const int32_t* elem_face;     // [4][nel]
  const float* R;               // [Nqf][nface]
  const float* in;
  float* out;
};

template <int NQ, bool CG = false>
__device__ __forceinline__ void lp_pe_tile(const LpPeView& v, const float* Hsh32, int64_t tile) {
  constexpr int NQF = NQ / 4, RN = NQ / 2;
  const int64_t ne = v.nel, nface = v.nface;
  const int64_t e = tile * kPeTile + threadIdx.x;
  if (e >= ne) return;
  int64_t face[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) face[f] = v.elem_face[f * ne + e];
  const int64_t fo[2] = {v.own[0] ? face[1] : face[0], v.own[1] == 3 ? face[3] : face[2]};
  float d[NQ], r[RN];
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int g = 0; g < NQF; ++g) d[f * NQF + g] = pe_ld<CG>(v.in + g * nface + face[f]);
#pragma unroll
  for (int j = 0; j < RN; ++j) r[j] = pe_ld<CG>(v.R + (j % NQF) * nface + fo[j / NQF]);
#pragma unroll
  for (int j = 0; j < RN; ++j) {
    const float* Hr = Hsh32 + j * NQ;
    float a = 0.f;
#pragma unroll
    for (int c = 0; c < NQ; ++c) a = fmaf(Hr[c], d[c], a);
    v.out[(j % NQF) * nface + fo[j / NQF]] = r[j] + a;
  }
}

}  // namespace ehdg
