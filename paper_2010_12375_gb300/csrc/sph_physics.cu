// Pair-interaction kernels and time-step control of the WCSPH hot path.
//
//   k_density              Eq. eqrhosum / Eq. eqrhosumnosurface (once per advection step)
//   k_viscous              Eq. eqviscous (once per advection step, fluid pairs)
//   k_dt_advection         Eq. dt-advection (one thread per instance, FP64)
//   k_dt_acoustic          Eq. dt-relax clamped to the advection step (one thread per instance)
//   (the acoustic-substep relaxation kernels live in sph_relax.cuh)
//
// Conventions: r_ij = r_i - r_j, e_ij = -r_ij/|r_ij| points from i to j, and
// grad_i W_ij = (dW/dr) r_ij/|r_ij|. Interface states of the low-dissipation
// solver: U* = (U_L+U_R)/2 + (P_L-P_R)/(2 rho_bar c0),
// P* = (P_L+P_R)/2 + rho_bar c0 beta (U_L-U_R)/2, beta = min(3 max(U_L-U_R,0)/c0, 1).
// One thread per fluid particle walks its frozen neighbour row (column-major
// ELL, so a warp's 32 index loads per row position are one 128-byte line) and
// recomputes the pair geometry from the current positions; pairs at or beyond
// 2h, or at zero distance, contribute nothing.
#include <cmath>

#include "sph_ctrl.cuh"
#include "sph_density.cuh"
#include "sph_kernels.h"

namespace sph {

namespace {

constexpr int kBlock = 256;

inline unsigned grid_for(int64_t n, int block = kBlock) {
  return (unsigned)((n + block - 1) / block);
}

__device__ __forceinline__ void raise_error(Global* g, int bit, long long idx) {
  int old = atomicOr(&g->err, bit);
  if (old == 0) g->bad_index = idx;
}

__device__ __forceinline__ int inst_index(const int* inst_of, int64_t i) {
  return inst_of ? inst_of[i] : 0;
}

// Block-wide max of |v|^2 into the instance's slot: one atomic per block when the
// whole block belongs to one instance, else one per lane.
__device__ __forceinline__ void reduce_vmax(float v2, bool valid, int k, bool uniform_block,
                                            Ctrl* ctrl) {
  __shared__ float red[kBlock / 32];
  if (!uniform_block) {
    if (valid) atomicMax(&ctrl[k].vmax2, __float_as_uint(v2));
    return;
  }
  float m = valid ? v2 : 0.0f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) atomicMax(&ctrl[k].vmax2, __float_as_uint(m));
  }
}

__device__ __forceinline__ bool block_one_instance(const int* inst_of, int64_t n, int* k_out) {
  int64_t first = (int64_t)blockIdx.x * blockDim.x;
  int64_t last = min(first + (int64_t)blockDim.x, n) - 1;
  int a = inst_index(inst_of, first), b = inst_index(inst_of, last);
  *k_out = a;
  return a == b;
}

// ---------------------------------------------------------------- import / export ----
// Quanta of a coordinate: rint((x - lo) / dq). FP64 runs at a sixty-fourth of FP32's rate on
// GB300, which bounds the import, and a division is a dozen of its operations: the quotient
// comes from the stored reciprocal, within 2^-21 of the exact one below 2^31, and only a
// coordinate within 2^-19 of a half or near the range's ends is divided (both tests on the
// doubles' high words). False outside the range or not a number.
__device__ __forceinline__ bool quanta(double x, double lo, double dq, double inv_dq, int* q) {
  const double s = (x - lo) * inv_dq;
  *q = __double2int_rn(s);
  const double off = s - (double)*q;                 // at most a half
  // high words: |s| below 2147481600, |off| below 0.5 - 2^-19
  if ((__double2hiint(s) & 0x7fffffff) < 0x41dffffe && (__double2hiint(off) & 0x7fffffff) < 0x3fdffff8) return true;
  const double lim = 2147483000.0, e = (x - lo) / dq;
  const bool in = e > -lim && e < lim;               // also catches NaN
  *q = __double2int_rn(in ? e : 0.0);
  return in;
}

// Start of a state import: |v|max cleared for it, and the clock of tank 0 (t < 0: kept).
__global__ void k_import_begin(int n_inst, Ctrl* ctrl, double t) {
  for (int k = threadIdx.x; k < n_inst; k += blockDim.x) ctrl[k].vmax2 = 0u;
  if (threadIdx.x == 0 && t >= 0.0) ctrl[0].t = t;
}

// Rows [i0, n) of the caller's arrays into the records, slot k holding caller row k until the
// next cell build, and |v|max. One pass: 314 us for 8.04M particles (568 us with divisions,
// and 54 us in passes of their own for the ids and |v|max).
template <int D>
__global__ void __launch_bounds__(kBlock)
k_import(int64_t i0, int64_t n, const double* __restrict__ pos, const double* __restrict__ vel,
         const double* __restrict__ rho, const double* __restrict__ drho,
         const int* __restrict__ inst_of, const Inst* __restrict__ inst,
         int4* __restrict__ P, float4* __restrict__ V, int* __restrict__ id, Ctrl* ctrl, Global* g) {
  const int64_t b0 = i0 + (int64_t)blockIdx.x * blockDim.x, i = b0 + threadIdx.x;
  const int ka = inst_index(inst_of, b0), kb = inst_index(inst_of, min(b0 + blockDim.x, n) - 1);
  float v2 = 0.f;
  int k = ka;
  const bool valid = i < n;
  if (valid) {
    if (ka != kb) k = inst_index(inst_of, i);
    const Inst& I = inst[k];
    int q[3] = {0, 0, 0};
    float w[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < D; ++a) {
      int qa;
      if (!quanta(pos[i * D + a], I.lo[a], I.dq_d, I.inv_dq_d, &qa)) raise_error(g, ERR_DOMAIN, i);
      if (I.period[a]) {
        qa %= I.period[a];
        if (qa < 0) qa += I.period[a];
      }
      q[a] = qa;
      w[a] = (float)vel[i * D + a];
    }
    const float dev = (float)(rho[i] - I.rho0_d);
    const float4 v = make_float4(w[0], w[1], w[2], drho ? (float)drho[i] : 0.0f);
    P[i] = make_int4(q[0], q[1], q[2], f2i(dev));
    V[i] = v;
    id[i] = (int)i;
    v2 = v.x * v.x + v.y * v.y + (D == 3 ? v.z * v.z : 0.f);
  }
  reduce_vmax(v2, valid, k, ka == kb, ctrl);
}

template <int D>
__global__ void k_import_walls(int64_t n, const double* __restrict__ pos, const double* __restrict__ nrm,
                               const double* __restrict__ vol, const int* __restrict__ inst_of,
                               const Inst* __restrict__ inst, int4* __restrict__ P,
                               float4* __restrict__ N, Global* g) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Inst& I = inst[inst_index(inst_of, i)];
  int q[3] = {0, 0, 0};
  float nv[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int a = 0; a < D; ++a) {
    int qa;
    if (!quanta(pos[i * D + a], I.lo[a], I.dq_d, I.inv_dq_d, &qa)) raise_error(g, ERR_DOMAIN, i);
    if (I.period[a]) {
      qa %= I.period[a];
      if (qa < 0) qa += I.period[a];
    }
    q[a] = qa;
    nv[a] = (float)nrm[i * D + a];
  }
  P[i] = make_int4(q[0], q[1], q[2], f2i((float)vol[i]));
  N[i] = make_float4(nv[0], nv[1], nv[2], 0.0f);
}

template <int D>
__global__ void k_export(int64_t n, const int4* __restrict__ P, const float4* __restrict__ V,
                         const int* __restrict__ id, const int* __restrict__ inst_of,
                         const Inst* __restrict__ inst, double* __restrict__ pos,
                         double* __restrict__ vel, double* __restrict__ rho,
                         double* __restrict__ drho) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Inst& I = inst[inst_index(inst_of, i)];
  int4 p = P[i];
  float4 v = V[i];
  int64_t row = id[i];
  int q[3] = {p.x, p.y, p.z};
  float vv[3] = {v.x, v.y, v.z};
#pragma unroll
  for (int a = 0; a < D; ++a) {
    if (pos) pos[row * D + a] = I.lo[a] + (double)q[a] * I.dq_d;
    if (vel) vel[row * D + a] = (double)vv[a];
  }
  if (rho) rho[row] = I.rho0_d + (double)i2f(p.w);
  if (drho) drho[row] = (double)v.w;
}

template <int D>
__global__ void k_export_acc(int64_t n, const float4* __restrict__ A, const int* __restrict__ id,
                             double* __restrict__ acc) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float4 a = A[i];
  int64_t row = id[i];
  acc[row * D + 0] = a.x;
  acc[row * D + 1] = a.y;
  if (D == 3) acc[row * D + 2] = a.z;
}

__global__ void k_export_neighbours(int64_t n, int cap, const int* __restrict__ nbr,
                                    const uint32_t* __restrict__ nbc, const int* __restrict__ id,
                                    const int* __restrict__ wid, int stride, int32_t* __restrict__ fc,
                                    int32_t* __restrict__ wc, int32_t* __restrict__ fids,
                                    int32_t* __restrict__ wids) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t c = nbc[i];
  int nf = (int)(c & 0xffffu), nw = (int)(c >> 16);
  int64_t row = id[i];
  fc[row] = nf;
  wc[row] = nw;
  for (int k = 0; k < nf; ++k) fids[row * stride + k] = id[nbr[slot_index(n, i, k)]];
  const int w0 = wall_slot0(nf);
  for (int k = 0; k < nw; ++k) wids[row * stride + k] = wid[nbr[slot_index(n, i, w0 + k)]];
}

__global__ void k_pair_count(int64_t n, const uint32_t* __restrict__ nbc, unsigned long long* out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long f = 0, w = 0;
  if (i < n) {
    f = nbc[i] & 0xffffu;
    w = nbc[i] >> 16;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    f += __shfl_xor_sync(0xffffffffu, f, o);
    w += __shfl_xor_sync(0xffffffffu, w, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&out[0], f);
    atomicAdd(&out[1], w);
  }
}

// ---------------------------------------------------------------- reductions / steps -
template <int D>
__global__ void k_vmax(int64_t n, const float4* __restrict__ V, const int* __restrict__ inst_of,
                       Ctrl* ctrl) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int k;
  bool uni = block_one_instance(inst_of, n, &k);
  float v2 = 0.f;
  bool valid = i < n;
  if (valid) {
    float4 v = V[i];
    v2 = v.x * v.x + v.y * v.y + (D == 3 ? v.z * v.z : 0.f);
    if (!uni) k = inst_index(inst_of, i);
  }
  reduce_vmax(v2, valid, k, uni, ctrl);
}

__global__ void k_reset_vmax(int n_inst, Ctrl* ctrl) {
  for (int k = threadIdx.x; k < n_inst; k += blockDim.x) ctrl[k].vmax2 = 0u;
}

// Eq. dt-advection for every tank (sph_ctrl.cuh).
__global__ void k_dt_advection(int n_inst, const Inst* __restrict__ inst, Ctrl* ctrl, Global* g) {
  for (int k = threadIdx.x; k < n_inst; k += blockDim.x) {
    dt_advection_one(inst[k], ctrl[k]);
  }
  if (threadIdx.x == 0) g->active = 1;
}

// Eq. dt-relax, clamped to the remainder of the advection step (block body in
// sph_ctrl.cuh). Sets the condition of the device-side substep loop when launched inside
// a graph.
__global__ void k_dt_acoustic(int n_inst, const Inst* __restrict__ inst, Ctrl* ctrl, Global* g,
                              cudaGraphConditionalHandle cond, int use_cond, const double* dt_cap) {
  const int any = dt_acoustic_block(n_inst, inst, ctrl, g, dt_cap);
  if (threadIdx.x == 0) {
    g->active = any;
    g->substeps += 1;
    if (use_cond) cudaGraphSetConditional(cond, any ? 1u : 0u);
  }
}

// ---------------------------------------------------------------- density -------------
template <int D, bool PER>
__global__ void __launch_bounds__(kBlock)
k_density(int64_t n, int4* P, const int* __restrict__ inst_of, const Inst* __restrict__ inst,
          const int* __restrict__ nbr, const uint32_t* __restrict__ nbc, const int4* __restrict__ WP) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Inst& I = inst[inst_index(inst_of, i)];
  const int4 pi = P[i];
  const float dev = density_dev<D, PER, 1>(I, i, 0, pi, nbc[i], n, P, reinterpret_cast<const int4*>(nbr), WP, nullptr);
  reinterpret_cast<int*>(P + i)[3] = f2i(dev);        // only .w changes; others read .xyz
}

template <int D, bool PER>
__global__ void __launch_bounds__(kBlock)
k_viscous(int64_t n, const int4* __restrict__ P, const float4* __restrict__ V,
          const float* __restrict__ mass, const int* __restrict__ inst_of,
          const Inst* __restrict__ inst, const int* __restrict__ nbr,
          const uint32_t* __restrict__ nbc, float4* __restrict__ acc_prior) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Inst& I = inst[inst_index(inst_of, i)];
  acc_prior[i] = viscous_acc<D, PER, 1>(I, i, 0, (int)(nbc[i] & 0xffffu), n, P, V, mass,
                                   reinterpret_cast<const int4*>(nbr), nullptr);
}

}  // namespace

// ---------------------------------------------------------------- launchers -----------
#define SPH_DIM_LAUNCH(b, kern, grid, block, stream, ...)                          \
  do {                                                                             \
    if ((b).dim == 2) kern<2><<<grid, block, 0, stream>>>(__VA_ARGS__);            \
    else kern<3><<<grid, block, 0, stream>>>(__VA_ARGS__);                         \
  } while (0)

void launch_import(const Buffers& b, const double* pos, const double* vel, const double* rho,
                   const double* drho, cudaStream_t s, int64_t i0, int64_t i1) {
  if (i1 < 0) i1 = b.n;
  if (i1 <= i0) return;
  SPH_DIM_LAUNCH(b, k_import, grid_for(i1 - i0), kBlock, s, i0, i1, pos, vel, rho, drho, b.inst_of, b.inst,
                 b.PS, b.VS, b.id, b.ctrl, b.glob);
}

void launch_import_begin(const Buffers& b, double t, cudaStream_t s) {
  k_import_begin<<<1, 256, 0, s>>>(b.n_inst, b.ctrl, t);
}

void launch_import_walls(const Buffers& b, const double* pos, const double* nrm, const double* vol,
                         cudaStream_t s) {
  if (b.nw == 0) return;
  SPH_DIM_LAUNCH(b, k_import_walls, grid_for(b.nw), kBlock, s, b.nw, pos, nrm, vol, b.winst_of, b.inst,
                 b.WP, b.WN, b.glob);
}

void launch_export(const Buffers& b, double* pos, double* vel, double* rho, double* drho,
                   cudaStream_t s) {
  if (b.n == 0) return;
  SPH_DIM_LAUNCH(b, k_export, grid_for(b.n), kBlock, s, b.n, b.PS, b.VS, b.id, b.inst_of, b.inst, pos,
                 vel, rho, drho);
}

void launch_export_acc(const Buffers& b, double* acc, cudaStream_t s) {
  if (b.n == 0 || !b.acc_keep) return;
  SPH_DIM_LAUNCH(b, k_export_acc, grid_for(b.n), kBlock, s, b.n, b.acc_keep, b.id, acc);
}

void launch_export_neighbours(const Buffers& b, int32_t* fc, int32_t* wc, int32_t* fids,
                              int32_t* wids, int32_t stride, cudaStream_t s) {
  if (b.n == 0) return;
  k_export_neighbours<<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.cap, b.nbr, b.nbc, b.id, b.wid, stride,
                                                        fc, wc, fids, wids);
}

void launch_pair_count(const Buffers& b, unsigned long long* out2, cudaStream_t s) {
  cudaMemsetAsync(out2, 0, 2 * sizeof(unsigned long long), s);
  if (b.n == 0) return;
  k_pair_count<<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.nbc, out2);
}

void launch_vmax(const Buffers& b, cudaStream_t s, int64_t* launches, bool reset) {
  if (reset) {
    k_reset_vmax<<<1, 256, 0, s>>>(b.n_inst, b.ctrl);
    ++*launches;
  }
  if (b.n == 0) return;
  SPH_DIM_LAUNCH(b, k_vmax, grid_for(b.n), kBlock, s, b.n, b.VS, b.inst_of, b.ctrl);
  ++*launches;
}

void launch_dt_advection(const Buffers& b, cudaStream_t s, int64_t* launches) {
  k_dt_advection<<<1, 256, 0, s>>>(b.n_inst, b.inst, b.ctrl, b.glob);
  ++*launches;
}

void launch_density(const Buffers& b, cudaStream_t s, int64_t* launches) {
  if (b.n == 0) return;
  auto kern = b.dim == 2 ? (b.any_periodic ? k_density<2, true> : k_density<2, false>)
                         : (b.any_periodic ? k_density<3, true> : k_density<3, false>);
  kern<<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.PS, b.inst_of, b.inst, b.nbr, b.nbc, b.WP);
  ++*launches;
}

void launch_viscous(const Buffers& b, cudaStream_t s, int64_t* launches) {
  if (b.n == 0 || !b.acc_prior) return;
  auto kern = b.dim == 2 ? (b.any_periodic ? k_viscous<2, true> : k_viscous<2, false>)
                         : (b.any_periodic ? k_viscous<3, true> : k_viscous<3, false>);
  kern<<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.PS, b.VS, b.mass, b.inst_of, b.inst, b.nbr, b.nbc, b.acc_prior);
  ++*launches;
}

void launch_dt_acoustic(const Buffers& b, cudaStream_t s, cudaGraphConditionalHandle cond,
                        bool use_cond, int64_t* launches) {
  k_dt_acoustic<<<1, 256, 0, s>>>(b.n_inst, b.inst, b.ctrl, b.glob, cond, use_cond ? 1 : 0, b.dt_cap);
  ++*launches;
}

}  // namespace sph
