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

// three blocks per SM from p = 4 on, four below: 253 x 187, p = 4 (370 tiles)
// then runs in one wave (6.75 ms for ten Crank-Nicolson steps; 7.74 at two
// blocks, 6.95 at four, which spill)
template <int NQ>
__global__ void __launch_bounds__(kPeTile, NQ >= 20 ? 3 : 4) k_sweep_pe(const __grid_constant__ PeView v,
                                                      const int2* Hx, int graph_mode,
                                                      cudaGraphConditionalHandle handle) {
  __shared__ __align__(16) int2 Hsh[NQ / 2 * NQ];
  for (int i = threadIdx.x; i < NQ / 2 * NQ; i += kPeTile) Hsh[i] = Hx[i];
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
// about 3 us where a launch in the conditional graph loop costs 8: 16 x 16, p = 2
// is all latency, and at 253 x 187, p = 4 it is a third of the iteration.
template <int NQ>
__global__ void __launch_bounds__(kPeTile, NQ >= 20 ? 3 : 4) k_pe_persist(const __grid_constant__ PeView v,
                                                        const int2* Hx) {
  __shared__ __align__(16) int2 Hsh[NQ / 2 * NQ];
  for (int i = threadIdx.x; i < NQ / 2 * NQ; i += kPeTile) Hsh[i] = Hx[i];
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

template <int NQ>
cudaError_t launch_pe_persist_t(const PeView& v, const int2* Hx, cudaStream_t s) {
  const int bpsm = fn_blocks_per_sm((const void*)k_pe_persist<NQ>, kPeTile, 0);
  const int64_t ntiles = (v.nel + kPeTile - 1) / kPeTile;
  const int grid = (int)std::min<int64_t>((int64_t)bpsm * device_sms(), ntiles);
  void* args[] = {const_cast<PeView*>(&v), &Hx};
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

// The sweep rows of Hy in row order as fixed-point limbs (one block): Hy =
// 2^(hs - 56) (h 2^28 + l), hs >= 0 the least with max |Hy| <= 2^(hs + 1), so
// that a coefficient is below 2 and a row's sums of at most 28 products with
// 56-bit values stay below 2^63.
static __global__ void k_pe_limbs(int n_rows, int NQFS, const int* rows, const double* Hy, int2* Hx,
                           int* hs) {
  __shared__ int s_e;
  if (threadIdx.x == 0) s_e = 0;
  __syncthreads();
  int em = 0;
  for (int i = threadIdx.x; i < n_rows * NQFS; i += blockDim.x)
    em = max(em, fx_exponent(Hy[rows[i / NQFS] * NQFS + i % NQFS]));
  atomicMax(&s_e, em);
  __syncthreads();
  const int s = max(0, s_e - 1023);            // |Hy| < 2^(s_e - 1022)
  if (threadIdx.x == 0) *hs = s;
  for (int i = threadIdx.x; i < n_rows * NQFS; i += blockDim.x) {
    const long long c = __double2ll_rn(scalbn(Hy[rows[i / NQFS] * NQFS + i % NQFS], 56 - s));
    const Limb x = fx_split(c);
    Hx[i] = make_int2(x.h, x.l);
  }
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
  cudaError_t e = dalloc_raw(c, (void**)&c.pe_hx, sizeof(int2) * c.n_rows * c.NQFS);
  if (e == cudaSuccess) e = dalloc_raw(c, (void**)&c.pe_hs, sizeof(int));
  if (e != cudaSuccess) return e;
  k_pe_limbs<<<1, 256, 0, c.stream>>>(c.n_rows, c.NQFS, c.rows, c.Hy,
                                      reinterpret_cast<int2*>(c.pe_hx), c.pe_hs);
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
  v.hs = c.pe_hs;
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
