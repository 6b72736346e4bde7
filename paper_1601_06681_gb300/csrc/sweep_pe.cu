// FP64 transport sweep on quadrilaterals with one shared local operator, one
// thread per element (the tile body in pe_tile.cuh). Small elements (2D,
// p <= 6: 8 to 28 face points, 4 to 14 sweep rows) give a thread only a few
// hundred FMAs, so the whole element stays in registers and a tile needs no
// barrier except the residual's. Its residual reduction does not depend on
// the grid, which lets a batch iterate such instances together and still
// match their single-problem runs bit for bit.
#include <cuda_runtime.h>

#include <algorithm>

#include "ehdg_internal.h"
#include "pe_tile.cuh"

namespace ehdg {

namespace {

// Blocks per SM: three from p = 4 on, four below. The spills that takes (32 to 304
// bytes from p = 3 up) cost less than another wave of blocks. Six Crank-Nicolson steps, ms at 2 / 3 / 4 / 5 blocks:
//   94 tiles:  p = 2 1.28 1.29 1.34 1.40  p = 4 1.88 2.02 2.24 2.30  p = 6 2.94 3.07 3.38 3.67
//   370 tiles: p = 2 2.70 2.40 2.45 2.51  p = 4 4.18 3.59 3.79 3.85  p = 6 6.98 5.70 5.95 6.49
//   938 tiles: p = 2 5.56 5.58 5.21 6.10  p = 4 8.70 9.27 8.65 10.7  p = 6 14.9 16.9 16.7 22.4
template <int NQ>
__global__ void __launch_bounds__(kPeTile, NQ >= 20 ? 3 : 4) k_sweep_pe(const __grid_constant__ PeView v,
                                                      const int2* Hx, int graph_mode,
                                                      cudaGraphConditionalHandle handle) {
  __shared__ __align__(16) int2 Hsh[pe_operator_len(NQ)];
  for (int i = threadIdx.x; i < pe_operator_len(NQ); i += kPeTile) Hsh[i] = Hx[i];
  __syncthreads();
  const int kk = v.it->k;                     // read before the last tile advances it
  const int64_t tlen = (int64_t)(NQ / 4) * v.nface;
  const double* src = v.uhat_slot(kk & 1, tlen);
  double* dst = const_cast<double*>(v.uhat_slot((kk + 1) & 1, tlen));
  const int64_t ntiles = (v.nel + kPeTile - 1) / kPeTile;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
    pe_tile<NQ>(v, Hsh, src, dst, tile, ntiles, graph_mode, handle);
}

template <int NQ>
cudaError_t launch_pe_t(const PeView& v, const int2* Hx, int graph_mode,
                        cudaGraphConditionalHandle handle, cudaStream_t s, int* grid_out) {
  const int bpsm = fn_blocks_per_sm((const void*)k_sweep_pe<NQ>, kPeTile, 0);
  const int64_t ntiles = (v.nel + kPeTile - 1) / kPeTile;
  int64_t grid = (int64_t)bpsm * device_sms();
  if (grid > ntiles) grid = ntiles;
  *grid_out = (int)grid;
  k_sweep_pe<NQ><<<(int)grid, kPeTile, 0, s>>>(v, Hx, graph_mode, handle);
  return cudaGetLastError();
}

// All iterations of a step in one cooperative launch: one pass over the tiles
// per iteration, the same tile code and residual sum as k_sweep_pe (so the same
// iterates and decisions bit for bit), traces read through L2. A pass ends for
// about 3 us where a launch in the conditional graph loop costs 8. Taken by
// meshes with more tiles than resident blocks; k_pe_resident has the others.
template <int NQ>
__global__ void __launch_bounds__(kPeTile, NQ >= 20 ? 3 : 4) k_pe_persist(const __grid_constant__ PeView v,
                                                        const int2* Hx) {
  __shared__ __align__(16) int2 Hsh[pe_operator_len(NQ)];
  for (int i = threadIdx.x; i < pe_operator_len(NQ); i += kPeTile) Hsh[i] = Hx[i];
  __syncthreads();
  const int64_t tlen = (int64_t)(NQ / 4) * v.nface;
  const int64_t ntiles = (v.nel + kPeTile - 1) / kPeTile;
  int k = v.it->k;
  for (unsigned int pass = 0;; ++pass, ++k) {
    const double* src = v.uhat_slot(k & 1, tlen);
    double* dst = const_cast<double*>(v.uhat_slot((k + 1) & 1, tlen));
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
      pe_tile_sweep<NQ, true>(v, Hsh, src, dst, tile);
      __syncthreads();                        // thread 0 has read the tile's warp sums
    }
    const int state = pass_end(v.it, gridDim.x, pass, v.hist, v.max_iter, v.tol, v.res_scale, [&] {
      return threadIdx.x < 32 ? pe_total(v.partials, ntiles) : 0.0;
    });
    if (state == 1) continue;
    if (state == 0 && threadIdx.x == 0) {
      v.it->status = EHDG_ERR_TIMEOUT;
      v.it->cont = 0;
    }
    return;
  }
}

// the barrier of a cluster's threads (all of them, every time), with release
// and acquire at cluster scope
__device__ __forceinline__ void pe_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// *p = x in the shared memory of block `rank` of the cluster
__device__ __forceinline__ void pe_cluster_store(double* p, int rank, double x) {
  asm volatile(
      "{\n .reg .b32 a;\n mapa.shared::cluster.u32 a, %0, %1;\n st.shared::cluster.f64 [a], %2;\n}\n" ::
          "r"((uint32_t)__cvta_generic_to_shared(p)),
      "r"(rank), "d"(x)
      : "memory");
}

// The same where every tile has a block of its own: what does not change
// between passes (face ids, Gy, weights, Jacobians) stays in registers, and so
// do the traces on the element's outflow faces, which its own thread wrote; a
// pass loads the NQ / 2 inflow values in one round through L2. The operator's
// columns are staged in the order outflow, inflow.
//
// CL: the grid is one cluster (up to kPeCluster tiles). Its hardware barrier
// ends a pass, every block holds all partial sums in shared memory and decides
// for itself: such a mesh is all latency, and the counter and the polled word
// in L2 cost more than the pass. 16 x 16, p = 2, 10 steps: 2.62 -> 1.35 ms with
// the cluster; 253 x 187, p = 4 with a block per tile 6.96 -> 5.70 (of both, 0.05 and
// 0.6 since Gy is aligned apart). The sums are those of pe_total, so iterates,
// residuals and decisions are bit for bit the same in every form.
constexpr int kPeCluster = 16;

template <int NQ, bool CL>
__global__ void __launch_bounds__(kPeTile, CL ? 1 : (NQ >= 20 ? 3 : 4))
    k_pe_resident(const __grid_constant__ PeView v, const int2* Hx) {
  constexpr int NQF = NQ / 4, RN = NQ / 2;
  __shared__ __align__(16) int2 Hsh[pe_operator_len(NQ)];
  __shared__ double red[kPeTile / 32];
  __shared__ double parts[CL ? 2 : 1][CL ? kPeCluster : 1];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int i = tid; i < RN * NQ; i += kPeTile) {
    const int j = i / NQ, c = i - j * NQ, b = c / NQF;
    const int f = b < 2 ? v.own[b] : v.own[b - 2] ^ 1;
    Hsh[i] = Hx[j * NQ + f * NQF + c - b * NQF];
  }
  for (int i = RN * NQ + tid; i < pe_operator_len(NQ); i += kPeTile) Hsh[i] = Hx[i];
  const int ntiles = (int)gridDim.x;
  const int64_t ne = v.nel, nface = v.nface, tlen = (int64_t)NQF * nface;
  const int64_t e = (int64_t)blockIdx.x * kPeTile + tid;
  const bool live = e < ne;
  int k = v.it->k;
  double uo[RN], gy[RN], w[NQF], jf[2] = {0.0, 0.0};
  int64_t fo[2] = {0, 0}, fi[2] = {0, 0};
  int eg = 1;
  const int2 tc = Hx[RN * NQ];
#pragma unroll
  for (int g = 0; g < NQF; ++g) w[g] = v.fw[g];
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    if (live) {
      fo[b] = v.elem_face[v.own[b] * ne + e];
      fi[b] = v.elem_face[(v.own[b] ^ 1) * ne + e];
      jf[b] = v.face_jf[fo[b]];
    }
#pragma unroll
    for (int g = 0; g < NQF; ++g) {
      gy[b * NQF + g] = live ? v.Gy[(b * NQF + g) * ne + e] : 0.0;
      uo[b * NQF + g] = live ? v.uhat_slot(k & 1, tlen)[g * nface + fo[b]] : 0.0;
      eg = max(eg, fx_exponent(gy[b * NQF + g]));
    }
  }
  __syncthreads();
  // (a block's shared memory is written by the others once all have started)
  if (CL) pe_cluster_sync();
  for (unsigned int pass = 0;; ++pass, ++k) {
    const double* src = v.uhat_slot(k & 1, tlen);
    double* dst = const_cast<double*>(v.uhat_slot((k + 1) & 1, tlen));
    double res = 0.0;
    if (live) {
      double ui[RN];
#pragma unroll
      for (int j = 0; j < RN; ++j) ui[j] = __ldcg(src + (j % NQF) * nface + fi[j / NQF]);
      int ea[2] = {1, 1};
#pragma unroll
      for (int j = 0; j < RN; ++j)
        ea[j / NQF] = max(ea[j / NQF], max(fx_exponent(uo[j]), fx_exponent(ui[j])));
      const int em = max(ea[0] + tc.x, ea[1] + tc.y);
      Limb x[NQ];
#pragma unroll
      for (int j = 0; j < RN; ++j) {
        const int ej = em - (j < NQF ? tc.x : tc.y);
        x[j] = fx_split(fx_from_double(uo[j], ej));
        x[RN + j] = fx_split(fx_from_double(ui[j], ej));
      }
      double sq[2] = {0.0, 0.0};
      const int* sc = reinterpret_cast<const int*>(Hsh + RN * NQ + 1);
#pragma unroll
      for (int j = 0; j < RN; ++j) {
        double acc = pe_row<NQ>(Hsh + j * NQ, x, em + sc[j], gy[j]);
        if (max(max(ea[0], ea[1]), eg) == 0x7ff) acc = __hiloint2double(0x7ff80000, 0);
        const int b = j / NQF, g = j - b * NQF;
        const double d = acc - uo[j];
        dst[g * nface + fo[b]] = acc;
        uo[j] = acc;
        sq[b] = fma(w[g], d * d, sq[b]);
      }
      res = fma(jf[0], sq[0], jf[1] * sq[1]);
    }
    res = fsum_warp(res);
    if (lane == 0) red[wid] = res;
    __syncthreads();
    if (!CL) {
      if (tid == 0) {
        double s = 0.0;
#pragma unroll
        for (int i = 0; i < kPeTile / 32; ++i) s += red[i];
        v.partials[blockIdx.x] = s;
      }
      const int state = pass_end(v.it, gridDim.x, pass, v.hist, v.max_iter, v.tol, v.res_scale,
                                 [&] { return tid < 32 ? pe_total(v.partials, ntiles) : 0.0; });
      if (state == 1) continue;
      if (state == 0 && tid == 0) {
        v.it->status = EHDG_ERR_TIMEOUT;
        v.it->cont = 0;
      }
      return;
    }
    double* mine = &parts[CL ? pass & 1 : 0][CL ? blockIdx.x : 0];
    if (tid < ntiles) {
      double s = 0.0;
#pragma unroll
      for (int i = 0; i < kPeTile / 32; ++i) s += red[i];
      pe_cluster_store(mine, tid, s);
    }
    pe_cluster_sync();
    const double r =
        v.res_scale * sqrt(fsum_warp(lane < ntiles ? parts[CL ? pass & 1 : 0][CL ? lane : 0] : 0.0));
    int cont = 1, status = EHDG_OK;
    if (!isfinite(r)) { cont = 0; status = EHDG_ERR_DIVERGED; }
    else if (r < v.tol) { cont = 0; status = EHDG_OK; }
    else if (k + 1 >= v.max_iter) { cont = 0; status = EHDG_ERR_NOT_CONVERGED; }
    if (blockIdx.x == 0 && tid == 0) {
      if (k < v.max_iter) v.hist[k] = r;
      if (!cont) {
        v.it->k = k + 1;
        v.it->r_last = r;
        v.it->status = status;
        v.it->cont = 0;
      }
    }
    if (!cont) return;
  }
}

// One cluster of all tiles, where the device takes a cluster of that size.
template <int NQ>
cudaError_t launch_pe_cluster_t(const PeView& v, const int2* Hx, int ntiles, cudaStream_t s) {
  cudaError_t e = ntiles > 8 ? cudaFuncSetAttribute((const void*)k_pe_resident<NQ, true>,
                                                    cudaFuncAttributeNonPortableClusterSizeAllowed, 1)
                             : cudaSuccess;
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned int)ntiles;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned int)ntiles);
  cfg.blockDim = dim3(kPeTile);
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int fits = 0;
  e = cudaOccupancyMaxActiveClusters(&fits, k_pe_resident<NQ, true>, &cfg);
  if (e != cudaSuccess) return e;
  if (fits < 1) return cudaErrorLaunchOutOfResources;
  return cudaLaunchKernelEx(&cfg, k_pe_resident<NQ, true>, v, Hx);
}

template <int NQ>
cudaError_t launch_pe_persist_t(const PeView& v, const int2* Hx, cudaStream_t s) {
  const int64_t ntiles = (v.nel + kPeTile - 1) / kPeTile;
  if (ntiles <= kPeCluster) {
    if (launch_pe_cluster_t<NQ>(v, Hx, (int)ntiles, s) == cudaSuccess) return cudaSuccess;
    cudaGetLastError();
  }
  void* args[] = {const_cast<PeView*>(&v), &Hx};
  const void* resident = (const void*)k_pe_resident<NQ, false>;
  if (ntiles <= (int64_t)fn_blocks_per_sm(resident, kPeTile, 0) * device_sms())
    return cudaLaunchCooperativeKernel(resident, dim3((unsigned int)ntiles), dim3(kPeTile), args, 0,
                                       s);
  const int bpsm = fn_blocks_per_sm((const void*)k_pe_persist<NQ>, kPeTile, 0);
  const int grid = (int)std::min<int64_t>((int64_t)bpsm * device_sms(), ntiles);
  return cudaLaunchCooperativeKernel((const void*)k_pe_persist<NQ>, dim3(grid), dim3(kPeTile),
                                     args, 0, s);
}

template <int NQ>
__global__ void __launch_bounds__(kPeTile) k_lp_pe(const LpPeView v, const float* Hy32) {
  constexpr int NQF = NQ / 4;
  __shared__ float Hsh[NQ / 2 * NQ];
  for (int i = threadIdx.x; i < NQ / 2 * NQ; i += kPeTile) {
    const int j = i / NQ, c = i - j * NQ;
    Hsh[i] = Hy32[(v.own[j / NQF] * NQF + j % NQF) * NQ + c];
  }
  __syncthreads();
  const int64_t ntiles = (v.nel + kPeTile - 1) / kPeTile;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) lp_pe_tile<NQ>(v, Hsh, tile);
}

template <int NQ>
cudaError_t launch_lp_pe_t(const LpPeView& v, const float* Hy32, cudaStream_t s) {
  const int bpsm = fn_blocks_per_sm((const void*)k_lp_pe<NQ>, kPeTile, 0);
  const int64_t ntiles = (v.nel + kPeTile - 1) / kPeTile;
  int64_t grid = (int64_t)bpsm * device_sms();
  if (grid > ntiles) grid = ntiles;
  k_lp_pe<NQ><<<(int)grid, kPeTile, 0, s>>>(v, Hy32);
  return cudaGetLastError();
}

}  // namespace

// The sweep rows of Hy in row order as fixed-point limbs, equilibrated (one block):
// t_a the exponent of the largest entry in the columns of axis a's faces, s_j then
// the least with row j's largest entry below 2 and its sum of magnitudes below 32,
// so that its sum with 56-bit values stays below 2^62.
static __global__ void k_pe_limbs(int NQFS, const int* rows, const double* Hy, int2* Hx) {
  __shared__ int s_t[2], s_s[kMaxQ * 2];
  const int n_rows = NQFS / 2, tid = threadIdx.x;
  if (tid < 2) s_t[tid] = kZeroGroup;
  __syncthreads();
  for (int i = tid; i < n_rows * NQFS; i += blockDim.x) {
    const double h = Hy[rows[i / NQFS] * NQFS + i % NQFS];
    if (h != 0.0) atomicMax(&s_t[(i % NQFS) / n_rows], min(1000, max(-1000, ilogb(h))));
  }
  __syncthreads();
  auto entry = [&](int j, int c) {
    const int t = s_t[c / n_rows];
    return t == kZeroGroup ? 0.0 : Hy[rows[j] * NQFS + c] * fx_pow2(-t);
  };
  if (tid < n_rows) {
    double mx = 0.0, sum = 0.0;
    for (int c = 0; c < NQFS; ++c) {
      mx = fmax(mx, fabs(entry(tid, c)));
      sum += fabs(entry(tid, c));
    }
    s_s[tid] = mx > 0.0 ? max(ilogb(mx), ilogb(sum) + 1 - 5) : 0;
  }
  __syncthreads();
  for (int i = tid; i < n_rows * NQFS; i += blockDim.x) {
    const int j = i / NQFS;
    const Limb x = fx_split(__double2ll_rn(scalbn(entry(j, i - j * NQFS), 56 - s_s[j])));
    Hx[i] = make_int2(x.h, x.l);
  }
  int* scales = reinterpret_cast<int*>(Hx + n_rows * NQFS);
  if (tid < 2) scales[tid] = s_t[tid];
  if (tid < n_rows) scales[2 + tid] = s_s[tid];
}

// FP32 correction sweep, one thread per element (quadrilaterals, shared
// operator, no beta.n = 0 point): every sweep row is an owned point.
cudaError_t launch_lp_sweep_pe(Ctx& c, const float* in, float* out) {
  LpPeView v;
  v.nel = c.nel;
  v.nface = c.nface;
  v.own[0] = c.rows_host[0] / c.Nqf;
  v.own[1] = c.rows_host[c.Nqf] / c.Nqf;
  v.elem_face = c.geo.elem_face;
  v.R = c.R32;
  v.in = in;
  v.out = out;
  switch (c.NQFS) {
    case 8: return launch_lp_pe_t<8>(v, c.Hy32, c.stream);
    case 12: return launch_lp_pe_t<12>(v, c.Hy32, c.stream);
    case 16: return launch_lp_pe_t<16>(v, c.Hy32, c.stream);
    case 20: return launch_lp_pe_t<20>(v, c.Hy32, c.stream);
    case 24: return launch_lp_pe_t<24>(v, c.Hy32, c.stream);
    default: return launch_lp_pe_t<28>(v, c.Hy32, c.stream);
  }
}

cudaError_t build_pe_operator(Ctx& c) {
  cudaError_t e = dalloc_raw(c, (void**)&c.pe_hx, sizeof(int2) * pe_operator_len(c.NQFS));
  if (e != cudaSuccess) return e;
  k_pe_limbs<<<1, 256, 0, c.stream>>>(c.NQFS, c.rows, c.Hy, reinterpret_cast<int2*>(c.pe_hx));
  return cudaGetLastError();
}

bool pe_supported(const Ctx& c) {
  return c.pde == EHDG_TRANSPORT && c.dim == 2 && c.shared_op && !c.variable_beta &&
         c.n_tan == 0 && !c.Hyt && c.NQFS >= 8 && c.NQFS <= 28 && c.n_rows == c.n_up &&
         2 * c.n_up == c.NQFS;   // the rows are the two outflow faces
}

PeView pe_view(const Ctx& c, double* fw_dev) {
  PeView v = {};
  v.nel = c.nel;
  v.nface = c.nface;
  v.own[0] = c.rows_host[0] / c.Nqf;
  v.own[1] = c.rows_host[c.Nqf] / c.Nqf;
  v.elem_face = c.geo.elem_face;
  v.face_jf = c.geo.face_jf;
  v.fw = fw_dev;
  v.Gy = c.Gy;
  v.R_out = c.mixed ? c.R32 : nullptr;
  v.partials = c.partials;
  v.it = c.it;
  v.hist = c.hist;
  v.max_iter = c.max_iter;
  v.tol = c.tol;
  v.res_scale = c.res_scale;
  v.uhat = c.uhat;
  return v;
}

cudaError_t launch_sweep_pe_persistent(Ctx& c) {
  const PeView v = pe_view(c, c.pe_fw);
  const int2* Hx = reinterpret_cast<const int2*>(c.pe_hx);
  switch (c.NQFS) {
    case 8: return launch_pe_persist_t<8>(v, Hx, c.stream);
    case 12: return launch_pe_persist_t<12>(v, Hx, c.stream);
    case 16: return launch_pe_persist_t<16>(v, Hx, c.stream);
    case 20: return launch_pe_persist_t<20>(v, Hx, c.stream);
    case 24: return launch_pe_persist_t<24>(v, Hx, c.stream);
    default: return launch_pe_persist_t<28>(v, Hx, c.stream);
  }
}

cudaError_t launch_sweep_pe(Ctx& c, int graph_mode, int* grid_out) {
  const PeView v = pe_view(c, c.pe_fw);
  const int2* Hx = reinterpret_cast<const int2*>(c.pe_hx);
  switch (c.NQFS) {
    case 8: return launch_pe_t<8>(v, Hx, graph_mode, c.handle, c.stream, grid_out);
    case 12: return launch_pe_t<12>(v, Hx, graph_mode, c.handle, c.stream, grid_out);
    case 16: return launch_pe_t<16>(v, Hx, graph_mode, c.handle, c.stream, grid_out);
    case 20: return launch_pe_t<20>(v, Hx, graph_mode, c.handle, c.stream, grid_out);
    case 24: return launch_pe_t<24>(v, Hx, graph_mode, c.handle, c.stream, grid_out);
    default: return launch_pe_t<28>(v, Hx, graph_mode, c.handle, c.stream, grid_out);
  }
}

}  // namespace ehdg
