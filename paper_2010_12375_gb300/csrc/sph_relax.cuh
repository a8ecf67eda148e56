// Acoustic-substep kernels of the position-based Verlet scheme (the hot loop).
//
//   k_pressure_relaxation  Eq. verlet-first-half (rho, r to n+1/2), Eq. eqeos,
//                          Eq. riemannsph momentum with P* of the low-dissipation
//                          solver, wall pairs by the one-sided problem of
//                          Eqs. eqriepartial / eqrienoslip / eqriepright,
//                          Eq. verlet-first-mediate (v to n+1)
//   k_density_relaxation   Eq. verlet-first-final: r to n+1 with v^{n+1}, then
//                          Eq. riemannsph continuity with U*, rho to n+1
//
// r_ij = r_i - r_j, e_ij = -r_ij/|r_ij|, grad_i W_ij = (dW/dr) r_ij/|r_ij|;
// U_L = v_i.e_ij, U_R = v_j.e_ij, U* = (U_L+U_R)/2 + (P_L-P_R)/(2 rho_bar c0),
// P* = (P_L+P_R)/2 + rho_bar c0 beta (U_L-U_R)/2, beta = min(3 max(U_L-U_R,0)/c0, 1).
//
// One thread per fluid particle walks its frozen neighbour row one quad (four
// slots, one 16-byte load, the next quad already in flight) at a time; the eight
// neighbour records of a quad are gathered together and evaluated as two packed
// pairs in the .x and .y lanes of sm_100 packed FP32 instructions (__ffma2_rn and
// friends), which halves the instruction count of the pair arithmetic. Unused
// slots of the last quad are padded with the particle itself, a pair at zero
// distance whose contribution is exactly zero. Pairs that drifted past 2h get
// t = max(1 - q/2, 0) = 0 and contribute nothing, with no branch. Each lane sums its
// pairs in plain FP32 (one fused multiply-add per term and axis) and the two lanes are
// added at the end: the accumulation error stays near 1e-7 of the sum on every parity
// state, far inside the 1e-5 per-substep bound, and compensated sums cost 8 % of the
// pressure relaxation's time on GB300.
//
// Template switches: TPP threads per particle and BLK threads per block (launch
// variants, each with its own register budget); UNI, a single-tank handle whose constant
// record arrives as the kernel argument; FG, the frozen-geometry reading, where each
// pair's vector r_i - r_j and (dW/dr)/r come from the table written at the configuration
// update instead of from the current positions; TV (pressure relaxation only), the
// transport velocity of Eq. transport, whose background-pressure term moves the mid-point
// position by dt^2/2 a_i.
//
// Launch forms: the per-particle kernels above map thread i of the grid to particle i;
// k_pressure_relaxation_rows / k_density_relaxation_rows (the row-task form, one tank)
// run the same per-particle code in one resident block an SM whose warps take 32-particle
// pieces of the search-cell rows from a queue (see the row-task section below).
#pragma once

#include "sph_kernels.h"

namespace sph {

namespace {

constexpr int kMaxBlock = 512;         // launch variants use 128, 256 or 512 threads

// Resident blocks per SM each launch variant is compiled for (its register budget):
// 896 threads per SM (72 registers) for both relaxation kernels at 128-thread blocks,
// measured fastest on the 8M 3D dam break (more warps in flight hide the neighbour
// gathers better than a larger register budget).
constexpr int pr_min_blocks(int block) { return block == 128 ? 7 : (block == 256 ? 3 : 1); }
constexpr int dr_min_blocks(int block) { return block == 128 ? 7 : (block == 256 ? 3 : 1); }
constexpr float kTinyR2 = 1e-30f;     // keeps rsqrt finite for a pair at zero distance

inline unsigned grid_for(int64_t threads, int block) {
  return (unsigned)((threads + block - 1) / block);
}

#ifndef SPH_HAVE_RAISE_ERROR
__device__ __forceinline__ void raise_error(Global* g, int bit, long long idx) {
  int old = atomicOr(&g->err, bit);
  if (old == 0) g->bad_index = idx;
}
#endif

__device__ __forceinline__ int inst_index(const int* inst_of, int64_t i) {
  return inst_of ? inst_of[i] : 0;
}

// Whether the particles [first, last] of this block (TPP threads each) share one tank.
template <int TPP>
__device__ __forceinline__ bool block_one_instance(const int* inst_of, int64_t n, int* k_out) {
  int64_t first = (int64_t)blockIdx.x * (blockDim.x / TPP);
  int64_t last = min(first + (int64_t)(blockDim.x / TPP), n) - 1;
  if (first > last) last = first;
  int a = inst_index(inst_of, min(first, n - 1)), b = inst_index(inst_of, max(last, (int64_t)0));
  *k_out = a;
  return a == b;
}

__device__ __forceinline__ void reduce_vmax(float v2, bool valid, int k, bool uniform_block, Ctrl* ctrl) {
  __shared__ float red[kMaxBlock / 32];
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

// s += a*b in both lanes (the second argument, the slot a compensated sum would keep, is
// unused: the relaxations sum plainly).
__device__ __forceinline__ void acc2(float2& s, float2&, float2 a, float2 b) { s = fma2(a, b, s); }

// Per-pair kernel factor (dW/dr)/r and |r| from the packed pair vector.
struct Geo2 {
  float2 inv_r, r, fw;
};

__device__ __forceinline__ Geo2 geometry2(float2 rx, float2 ry, float2 rz, float inv_h, float dwr) {
  Geo2 g;
  float2 r2 = fma2(rx, rx, fma2(ry, ry, fma2(rz, rz, f2(kTinyR2))));
  g.inv_r = rsqrt2(r2);
  g.r = mul2(r2, g.inv_r);
  // 1 - q/2 clamped to [0, 1] (0 beyond 2h; r >= 0 keeps it <= 1): one saturating FMA per lane
  float2 t = make_float2(__saturatef(fmaf(g.r.x, -0.5f * inv_h, 1.0f)), __saturatef(fmaf(g.r.y, -0.5f * inv_h, 1.0f)));
  g.fw = mul2(f2(dwr), mul2(mul2(t, t), t));                       // -5 alpha/h^2 (1-q/2)^3
  return g;
}

// The same factors from a stored pair vector and (dW/dr)/r (frozen-geometry reading):
// 1/|r| and |r| come out of the same operations as in geometry2.
__device__ __forceinline__ Geo2 stored_geometry2(float2 rx, float2 ry, float2 rz, float2 fw) {
  Geo2 g;
  float2 r2 = fma2(rx, rx, fma2(ry, ry, fma2(rz, rz, f2(kTinyR2))));
  g.inv_r = rsqrt2(r2);
  g.r = mul2(r2, g.inv_r);
  g.fw = fw;
  return g;
}

// Exactly converted, packed pair vector: dq (q_i - q_j) + add, lanes (a, b).
template <bool PER>
__device__ __forceinline__ float2 pair_axis(int qi, int qa, int qb, int period, float2 DQ, float2 add) {
  return fma2(add2(make_float2(biased_diff<PER>(qi, qa, period), biased_diff<PER>(qi, qb, period)),
                   f2(-kMagic)),
              DQ, add);
}

// Shared per-particle context of the pressure relaxation.
struct PrCtx {
  float hdt, dev_i, rho_i, pr_i;
  int px, py, pz;
  float2 sx, sy, sz, nx, ny, nz;      // per-lane sums (nx, ny, nz stay zero: plain sums)
  float2 bx, by, bz;                  // transport velocity: sum V_j (dW/dr)/r r_ij (plain sums)
};

// Two fluid pairs (a, b) of the pressure relaxation: returns V_j P* (dW/dr)/r and the pair
// vectors r_ij, with TV also Eq. transport's V_j (dW/dr)/r in bt.
// FG: the pair vectors and (dW/dr)/r come from the frozen table (ga, gb), else from the
// mid-point positions.
template <int D, bool PER, bool FG = false, bool TV = false>
__device__ __forceinline__ float2 pr_fluid_term2(const Inst& I, const PrCtx& C, const int4& pi, const float4& vi,
                                                 const int4& pa, const int4& pb, const float4& va, const float4& vb,
                                                 float2 mj, float2 DQ, float2& rx, float2& ry, float2& rz, float2& bt,
                                                 float4 ga = float4(), float4 gb = float4()) {
  const float2 HDT = f2(C.hdt), MHDT = f2(-C.hdt);
  // v_j - v_i; hdt (v_i - v_j) = (-hdt)(v_j - v_i) exactly, so one difference serves both
  const float2 dvx = sub2(make_float2(va.x, vb.x), f2(vi.x));
  const float2 dvy = sub2(make_float2(va.y, vb.y), f2(vi.y));
  const float2 dvz = D == 3 ? sub2(make_float2(va.z, vb.z), f2(vi.z)) : f2(0.f);
  rz = f2(0.f);
  Geo2 G;
  if (FG) {
    rx = make_float2(ga.x, gb.x);
    ry = make_float2(ga.y, gb.y);
    if (D == 3) rz = make_float2(ga.z, gb.z);
    G = stored_geometry2(rx, ry, rz, make_float2(ga.w, gb.w));
  } else {
    rx = pair_axis<PER>(pi.x, pa.x, pb.x, C.px, DQ, mul2(MHDT, dvx));
    ry = pair_axis<PER>(pi.y, pa.y, pb.y, C.py, DQ, mul2(MHDT, dvy));
    if (D == 3) rz = pair_axis<PER>(pi.z, pa.z, pb.z, C.pz, DQ, mul2(MHDT, dvz));
    G = geometry2(rx, ry, rz, I.inv_h, I.dwr_a);
  }
  const float2 dev_j = fma2(HDT, make_float2(va.w, vb.w), make_float2(i2f(pa.w), i2f(pb.w)));
  const float2 rho_j = add2(f2(I.rho0), dev_j);
  // U_L - U_R = (v_j - v_i).r_ij / |r_ij|
  const float2 dU = mul2(fma2(dvx, rx, fma2(dvy, ry, mul2(dvz, rz))), G.inv_r);
  const float2 beta = make_float2(__saturatef(I.kc * dU.x), __saturatef(I.kc * dU.y));   // min(kc max(dU, 0), 1)
  // P* = (p_i + p_j)/2 + (c0/4)(rho_i + rho_j) beta (U_L - U_R)
  const float2 pbar = mul2(f2(I.hc0sq), add2(f2(C.dev_i), dev_j));
  const float2 pstar = fma2(mul2(f2(I.qc0), add2(f2(C.rho_i), rho_j)), mul2(beta, dU), pbar);
  const float2 f = mul2(mul2(mul2(mj, rcp2(rho_j)), pstar), G.fw);       // V_j P* (dW/dr)/r
  if (TV) bt = mul2(mul2(mj, rcp2(rho_j)), G.fw);    // Eq. transport: V_j (dW/dr)/r
  return f;
}

// The terms of two pairs added to the sums.
template <int D>
__device__ __forceinline__ void pr_add2(PrCtx& C, float2 f, float2 rx, float2 ry, float2 rz) {
  acc2(C.sx, C.nx, f, rx);
  acc2(C.sy, C.ny, f, ry);
  if (D == 3) acc2(C.sz, C.nz, f, rz);
}

template <int D, bool PER, bool FG = false, bool TV = false>
__device__ __forceinline__ void pr_fluid2(const Inst& I, PrCtx& C, const int4& pi, const float4& vi, const int4& pa,
                                          const int4& pb, const float4& va, const float4& vb, float2 mj,
                                          float2 DQ, float4 ga = float4(), float4 gb = float4()) {
  float2 rx, ry, rz, b;
  const float2 f = pr_fluid_term2<D, PER, FG, TV>(I, C, pi, vi, pa, pb, va, vb, mj, DQ, rx, ry, rz, b, ga, gb);
  pr_add2<D>(C, f, rx, ry, rz);
  if (TV) {
    C.bx = fma2(b, rx, C.bx);
    C.by = fma2(b, ry, C.by);
    if (D == 3) C.bz = fma2(b, rz, C.bz);
  }
}

// Two wall pairs of the pressure relaxation (one-sided problem along the wall normal).
template <int D, bool PER, bool FG = false>
__device__ __forceinline__ float2 pr_wall_term2(const Inst& I, const PrCtx& C, const int4& pi, const float4& vi,
                                                const int4& qa, const int4& qb, const float4& na,
                                                const float4& nb, float2 Vw, float2 DQ, float2& rx, float2& ry,
                                                float2& rz, float4 ga = float4(), float4 gb = float4()) {
  rz = f2(0.f);
  Geo2 G;
  if (FG) {
    rx = make_float2(ga.x, gb.x);
    ry = make_float2(ga.y, gb.y);
    if (D == 3) rz = make_float2(ga.z, gb.z);
    G = stored_geometry2(rx, ry, rz, make_float2(ga.w, gb.w));
  } else {
    rx = pair_axis<PER>(pi.x, qa.x, qb.x, C.px, DQ, f2(C.hdt * vi.x));
    ry = pair_axis<PER>(pi.y, qa.y, qb.y, C.py, DQ, f2(C.hdt * vi.y));
    if (D == 3) rz = pair_axis<PER>(pi.z, qa.z, qb.z, C.pz, DQ, f2(C.hdt * vi.z));
    G = geometry2(rx, ry, rz, I.inv_h, I.dwr_a);
  }
  // U_L = -n.v_i, U_R = -U_L, P_R = P_L + rho_i g.(r_w - r_i), rho_R from the EoS
  const float2 UL = mul2(f2(-1.0f), fma2(make_float2(na.x, nb.x), f2(vi.x),
                                         fma2(make_float2(na.y, nb.y), f2(vi.y), mul2(make_float2(na.z, nb.z), f2(vi.z)))));
  const float2 gr = fma2(f2(I.g[0]), rx, fma2(f2(I.g[1]), ry, mul2(f2(I.g[2]), rz)));
  const float2 PR = fma2(f2(-C.rho_i), gr, f2(C.pr_i));
  const float2 rhoR = fma2(PR, f2(I.inv_c0sq), f2(I.rho0));
  const float2 dU = add2(UL, UL);
  const float2 beta = make_float2(__saturatef(I.kc * dU.x), __saturatef(I.kc * dU.y));   // min(kc max(dU, 0), 1)
  const float2 pstar = fma2(mul2(f2(I.qc0), add2(f2(C.rho_i), rhoR)), mul2(beta, dU),
                            mul2(f2(0.5f), add2(f2(C.pr_i), PR)));
  return mul2(mul2(Vw, pstar), G.fw);
}

template <int D, bool PER, bool FG = false>
__device__ __forceinline__ void pr_wall2(const Inst& I, PrCtx& C, const int4& pi, const float4& vi,
                                         const int4& qa, const int4& qb, const float4& na,
                                         const float4& nb, float2 Vw, float2 DQ,
                                         float4 ga = float4(), float4 gb = float4()) {
  float2 rx, ry, rz;
  const float2 f = pr_wall_term2<D, PER, FG>(I, C, pi, vi, qa, qb, na, nb, Vw, DQ, rx, ry, rz, ga, gb);
  pr_add2<D>(C, f, rx, ry, rz);
}


// The end of one particle's pressure relaxation from its sums: dv/dt, v to n+1, r to the mid
// point (verlet-first-half), both stored. Returns |v^{n+1}|^2.
template <int D, bool PER, bool TV>
__device__ __forceinline__ float pr_finish(const Inst& I, const PrCtx& C, int64_t i, float dt, const int4& pi,
                                           const float4& vi, float ax, float ay, float az, int4* PH, float4* VH,
                                           const float4* acc_prior, float4* acc_keep, Global* g) {
  // dv/dt = acc_prior + g - (2/rho_i) sum V_j P* grad_i W_ij
  const float sc = -2.0f / C.rho_i;
  const float4 ap = acc_prior ? acc_prior[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  const float a0 = ap.x + I.g[0] + sc * ax;
  const float a1 = ap.y + I.g[1] + sc * ay;
  const float a2 = D == 3 ? ap.z + I.g[2] + sc * az : 0.f;
  const float4 vn = make_float4(vi.x + dt * a0, vi.y + dt * a1, vi.z + dt * a2, vi.w);  // verlet-first-mediate
  const float hdt = C.hdt;
  float ux = vi.x, uy = vi.y, uz = vi.z;                   // dt/2 times this moves r to n+1/2
  if (TV) {                                                // + dt^2/2 a_i: dt/2 (v + dt a_i)
    const float tv = -2.0f * I.p_tv / C.rho_i * dt;
    ux += tv * (C.bx.x + C.bx.y);
    uy += tv * (C.by.x + C.by.y);
    uz += tv * (C.bz.x + C.bz.y);
  }
  int qx = pi.x + __float2int_rn(hdt * ux * I.inv_dq);                                // verlet-first-half
  int qy = pi.y + __float2int_rn(hdt * uy * I.inv_dq);
  int qz = D == 3 ? pi.z + __float2int_rn(hdt * uz * I.inv_dq) : 0;
  if (PER) {
    qx = wrap_coord(qx, C.px);
    qy = wrap_coord(qy, C.py);
    if (D == 3) qz = wrap_coord(qz, C.pz);
  }
  PH[i] = make_int4(qx, qy, qz, f2i(C.dev_i));
  VH[i] = vn;
  if (acc_keep) acc_keep[i] = make_float4(a0, a1, a2, 0.f);
  const float v2 = vn.x * vn.x + vn.y * vn.y + vn.z * vn.z;
  if (!isfinite(v2)) raise_error(g, ERR_NAN, i);
  return v2;
}

// ---------------------------------------------------------------- lanes of a particle --
// LPP lanes share one particle: lane `sub` evaluates quads sub, sub + LPP, ... of its row,
// and after each round of LPP quads the terms are added in row order through shared memory,
// lane a summing axis a. A particle's sums thus add the same terms in the same order as one
// lane does: the results are identical bit for bit for every LPP, while a particle's chain of
// dependent gathers is LPP times shorter. terms: this warp's [1 + D][32] float4 of shared
// memory, with the transport velocity [2 + D][32]. All lanes of a group share `valid`.
//
// Particle p of a warp's 32 / LPP has the lanes p, p + 32 / LPP, ...: neighbouring lanes hold
// neighbouring particles at the same place of their rows, whose records lie close together
// (with the lanes of a particle side by side every gather touched twice the lines).
template <int LPP>
__device__ __forceinline__ int lane_sub() { return LPP == 1 ? 0 : (int)(threadIdx.x & 31) / (32 / LPP); }
// this thread's particle among those of its block
template <int LPP>
__device__ __forceinline__ int lane_particle() {
  return LPP == 1 ? (int)threadIdx.x : (int)(threadIdx.x >> 5) * (32 / LPP) + (int)(threadIdx.x & (32 / LPP - 1));
}
template <int LPP>
__device__ __forceinline__ unsigned group_mask() {
  constexpr unsigned m = LPP == 2 ? 0x00010001u : LPP == 4 ? 0x01010101u : 0x11111111u;
  static_assert(LPP == 1 || LPP == 2 || LPP == 4 || LPP == 8, "lanes of a particle");
  return m << (threadIdx.x & (32 / LPP - 1));
}

// The start of a particle's row as one of its lanes needs it: the counts, and the lane's first
// quad (fluid quads first, wall quads right after them).
struct RowHead {
  uint32_t cnt;
  int4 quad;
  template <int LPP, typename PN, typename PC>
  __device__ __forceinline__ void load(int64_t i, int sub, int64_t n, PN nb4, PC nbc) {
    cnt = i < 0 ? 0u : nbc[i];
    const int quads = (((int)(cnt & 0xffffu) + 3) >> 2) + (((int)(cnt >> 16) + 3) >> 2);
    quad = sub < quads ? nb4[(int64_t)sub * n + i] : make_int4(0, 0, 0, 0);
  }
};

// One quad's two pair terms of this lane into the exchange.
template <int D>
__device__ __forceinline__ void put_terms(float4* terms, float2 f01, float2 x01, float2 y01, float2 z01, float2 f23,
                                          float2 x23, float2 y23, float2 z23) {
  const int lane = threadIdx.x & 31;
  terms[lane] = make_float4(f01.x, f01.y, f23.x, f23.y);
  terms[32 + lane] = make_float4(x01.x, x01.y, x23.x, x23.y);
  terms[64 + lane] = make_float4(y01.x, y01.y, y23.x, y23.y);
  if (D == 3) terms[96 + lane] = make_float4(z01.x, z01.y, z23.x, z23.y);
}

// Adds the terms of `count` lanes of the group, in order, to this lane's axis sums (axes sub,
// sub + LPP, ... below D). TV: likewise Eq. transport's terms, to t.
template <int LPP, int D, bool TV = false>
__device__ __forceinline__ void add_terms(const float4* terms, int sub, int count, float2 (&s)[2], float2 (&t)[2]) {
  const int base = threadIdx.x & (32 / LPP - 1);
  __syncwarp(group_mask<LPP>());
#pragma unroll
  for (int h = 0; h < (D + LPP - 1) / LPP; ++h) {
    const int a = sub + h * LPP;
    if (a < D) {
      for (int k = 0; k < count; ++k) {
        const float4 f = terms[base + k * (32 / LPP)], r = terms[32 * (1 + a) + base + k * (32 / LPP)];
        s[h] = fma2(make_float2(f.x, f.y), make_float2(r.x, r.y), s[h]);
        s[h] = fma2(make_float2(f.z, f.w), make_float2(r.z, r.w), s[h]);
        if (TV) {
          const float4 b = terms[32 * (1 + D) + base + k * (32 / LPP)];
          t[h] = fma2(make_float2(b.x, b.y), make_float2(r.x, r.y), t[h]);
          t[h] = fma2(make_float2(b.z, b.w), make_float2(r.z, r.w), t[h]);
        }
      }
    }
  }
  __syncwarp(group_mask<LPP>());
}

// One particle of the pressure relaxation shared by LPP lanes. Where a round takes its last
// fluid quads it takes the first wall quads too. Array types carry the caller's aliasing qualifiers. Returns
// |v^{n+1}|^2 on the lane that wrote the particle, else 0.
template <int D, bool PER, int LPP, bool TV, typename PI, typename PF, typename PM, typename PN>
__device__ __forceinline__ float pr_group(const Inst& I, int64_t i, int sub, bool valid, double dtd, int64_t n, PI PS,
                                          PF VS, int4* PH, float4* VH, PM mass, PN nb4, const RowHead& head,
                                          const int4* __restrict__ WP, const float4* __restrict__ WN,
                                          const float4* acc_prior, float4* acc_keep, Global* g, float4* terms,
                                          bool* writer_out) {
  *writer_out = valid && sub == 0;
  if (!valid) return 0.0f;
  PrCtx C;
  C.sx = C.sy = C.sz = C.nx = C.ny = C.nz = f2(0.f);
  C.bx = C.by = C.bz = f2(0.f);
  float2 sa[2] = {f2(0.f), f2(0.f)}, sb[2] = {f2(0.f), f2(0.f)};   // this lane's axis sums (LPP > 1)
  const float dt = (float)dtd;
  C.hdt = 0.5f * dt;
  C.px = PER ? I.period[0] : 0;
  C.py = PER ? I.period[1] : 0;
  C.pz = PER ? I.period[2] : 0;
  const int4 pi = PS[i];
  const float4 vi = VS[i];
  C.dev_i = i2f(pi.w) + C.hdt * vi.w;                 // Eq. verlet-first-half (density)
  C.rho_i = I.rho0 + C.dev_i;
  C.pr_i = I.c0sq * C.dev_i;                          // Eq. eqeos
  const float2 DQ = f2(I.dq);
  const uint32_t cnt = head.cnt;
  const int nf = (int)(cnt & 0xffffu), nw = (int)(cnt >> 16);
  const int nq = (nf + 3) >> 2;
  int4 cur = head.quad;
  // the quad of fluid slots s .. s + 3: the terms of its two pairs of pairs, or their sums
  auto fluid = [&](const int4& c, int s) {
    const int j0 = c.x;
    const int j1 = s + 1 < nf ? c.y : (int)i;                // self pads: zero terms
    const int j2 = s + 2 < nf ? c.z : (int)i;
    const int j3 = s + 3 < nf ? c.w : (int)i;
    const int4 p0 = PS[j0], p1 = PS[j1], p2 = PS[j2], p3 = PS[j3];
    const float4 v0 = VS[j0], v1 = VS[j1], v2 = VS[j2], v3 = VS[j3];
    float2 m01 = f2(I.mass), m23 = f2(I.mass);
    if (mass) {
      m01 = make_float2(mass[j0], mass[j1]);
      m23 = make_float2(mass[j2], mass[j3]);
    }
    if (LPP == 1) {
      pr_fluid2<D, PER, false, TV>(I, C, pi, vi, p0, p1, v0, v1, m01, DQ);
      pr_fluid2<D, PER, false, TV>(I, C, pi, vi, p2, p3, v2, v3, m23, DQ);
    } else {
      float2 x01, y01, z01, x23, y23, z23, b01 = f2(0.f), b23 = f2(0.f);
      const float2 f01 = pr_fluid_term2<D, PER, false, TV>(I, C, pi, vi, p0, p1, v0, v1, m01, DQ, x01, y01, z01, b01);
      const float2 f23 = pr_fluid_term2<D, PER, false, TV>(I, C, pi, vi, p2, p3, v2, v3, m23, DQ, x23, y23, z23, b23);
      put_terms<D>(terms, f01, x01, y01, z01, f23, x23, y23, z23);
      if (TV) terms[32 * (1 + D) + (threadIdx.x & 31)] = make_float4(b01.x, b01.y, b23.x, b23.y);
    }
  };
  auto wall = [&](const int4& c, int s) {
    const int w1 = s + 1 < nw ? c.y : c.x, w2 = s + 2 < nw ? c.z : c.x, w3 = s + 3 < nw ? c.w : c.x;
    const int4 a0 = WP[c.x], a1 = WP[w1], a2 = WP[w2], a3 = WP[w3];
    const float4 n0 = WN[c.x], n1 = WN[w1], n2 = WN[w2], n3 = WN[w3];
    const float2 V01 = make_float2(i2f(a0.w), s + 1 < nw ? i2f(a1.w) : 0.0f);   // pads carry no volume
    const float2 V23 = make_float2(s + 2 < nw ? i2f(a2.w) : 0.0f, s + 3 < nw ? i2f(a3.w) : 0.0f);
    if (LPP == 1) {
      pr_wall2<D, PER>(I, C, pi, vi, a0, a1, n0, n1, V01, DQ);
      pr_wall2<D, PER>(I, C, pi, vi, a2, a3, n2, n3, V23, DQ);
    } else {
      float2 x01, y01, z01, x23, y23, z23;
      const float2 f01 = pr_wall_term2<D, PER>(I, C, pi, vi, a0, a1, n0, n1, V01, DQ, x01, y01, z01);
      const float2 f23 = pr_wall_term2<D, PER>(I, C, pi, vi, a2, a3, n2, n3, V23, DQ, x23, y23, z23);
      put_terms<D>(terms, f01, x01, y01, z01, f23, x23, y23, z23);
      if (TV) terms[32 * (1 + D) + (threadIdx.x & 31)] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  const int nwq = (nw + 3) >> 2;
  if (LPP == 1) {
    for (int q = 0; q < nq; ++q) {
      int4 nxt = cur;
      if (q + 1 < nq + nwq) nxt = nb4[(int64_t)(q + 1) * n + i];   // next quad in flight
      fluid(cur, q << 2);
      cur = nxt;
    }
    for (int q = 0; q < nwq; ++q) {
      int4 nxt = cur;
      if (q + 1 < nwq) nxt = nb4[(int64_t)(nq + q + 1) * n + i];
      wall(cur, q << 2);
      cur = nxt;
    }
  } else {
    for (int q0 = 0; q0 < nq + nwq; q0 += LPP) {
      const int q = q0 + sub;
      int4 nxt = cur;
      if (q + LPP < nq + nwq) nxt = nb4[(int64_t)(q + LPP) * n + i];
      if (q < nq) fluid(cur, q << 2);
      else if (q < nq + nwq) wall(cur, (q - nq) << 2);
      add_terms<LPP, D, TV>(terms, sub, min(LPP, nq + nwq - q0), sa, sb);
      cur = nxt;
    }
  }
  float ax = (C.sx.x + C.nx.x) + (C.sx.y + C.nx.y);
  float ay = (C.sy.x + C.ny.x) + (C.sy.y + C.ny.y);
  float az = (C.sz.x + C.nz.x) + (C.sz.y + C.nz.y);
  if (LPP > 1) {
    const unsigned gm = group_mask<LPP>();
    const int p = threadIdx.x & (32 / LPP - 1);
    const float a = (sa[0].x + 0.0f) + (sa[0].y + 0.0f), b = (sa[1].x + 0.0f) + (sa[1].y + 0.0f);
    ax = __shfl_sync(gm, a, p);
    ay = __shfl_sync(gm, a, p + 32 / LPP);
    if (D == 3) az = LPP == 2 ? __shfl_sync(gm, b, p) : __shfl_sync(gm, a, p + 2 * (32 / LPP));
    if (TV) {                                         // the two lanes of a sum are added at the end
      const float2 t = make_float2(__shfl_sync(gm, sb[0].x, p), __shfl_sync(gm, sb[0].y, p));
      const float2 u = make_float2(__shfl_sync(gm, sb[0].x, p + 32 / LPP), __shfl_sync(gm, sb[0].y, p + 32 / LPP));
      C.bx = t;
      C.by = u;
      if (D == 3) {
        const int z = LPP == 2 ? p : p + 2 * (32 / LPP);
        const float2 w = LPP == 2 ? sb[1] : sb[0];
        C.bz = make_float2(__shfl_sync(gm, w.x, z), __shfl_sync(gm, w.y, z));
      }
    }
    if (sub != 0) return 0.0f;
  }
  return pr_finish<D, PER, TV>(I, C, i, dt, pi, vi, ax, ay, az, PH, VH, acc_prior, acc_keep, g);
}

// ---------------------------------------------------------------- pressure relaxation --
// One particle of the pressure relaxation by one thread.
// FG: pair geometry from the frozen table geo ([slot][n]) instead of the positions.
// TV: transport velocity (Eq. transport): the mid-point position written for the density
// relaxation also takes dt^2/2 a_i, a_i = -(2 p0 / rho_i) sum_j V_j grad_i W_ij over the
// fluid pairs.
// Returns |v^{n+1}|^2 when the particle was written (*writer), else 0. The array pointers
// carry the caller's aliasing qualifiers: the per-launch kernels pass __restrict__ ones, the
// persistent loop plain ones (its phases read what other blocks wrote in the previous phase).
//
// EARLY: the particle's state, counts and first quad are read (i in [0, n) also where !valid)
// without waiting for the tank's step and constants or for the counts, which put three more
// memory latencies before a row's first gather. It pays in the per-launch 2D kernel, whose
// rows have seven quads (19.1 -> 17.7 us at 180,000 particles, 35.5 -> 33.5 us at 500,000,
// 94.2 -> 90.8 us for 64 tanks of 1.07M); in 3D, twenty quads, it takes registers from the
// gathers (one 8.04M step 3 % slower as row tasks), and it gains nothing in the persistent
// loop and in the density relaxation.
template <int D, bool PER, bool FG, bool TV, bool EARLY, typename PI, typename PF>
__device__ __forceinline__ float pr_particle(const Inst& I, int64_t i, bool valid, double dtd,
                                             const float4* __restrict__ geo, int64_t n, PI PS, PF VS,
                                             int4* PH, float4* VH, const float* __restrict__ mass,
                                             const int* __restrict__ nbr, const uint32_t* __restrict__ nbc,
                                             const int4* __restrict__ WP, const float4* __restrict__ WN,
                                             const float4* __restrict__ acc_prior, float4* __restrict__ acc_keep,
                                             Global* g, bool* writer_out) {
  float v2 = 0.0f;
  static_assert(!TV || !FG, "transport velocity: recomputed geometry");
  PrCtx C;
  C.sx = C.sy = C.sz = C.nx = C.ny = C.nz = f2(0.f);
  C.bx = C.by = C.bz = f2(0.f);
  const float dt = (float)dtd;
  const int4* __restrict__ nb4 = reinterpret_cast<const int4*>(nbr);
  int4 pi = make_int4(0, 0, 0, 0), cur = pi;
  float4 vi = make_float4(0.f, 0.f, 0.f, 0.f);
  uint32_t cnt = 0;
  if (EARLY) {
    pi = PS[i];
    cnt = nbc[i];
    cur = nb4[i];                                     // not looked at without neighbours
    vi = VS[i];
  }
  if (valid) {
    C.hdt = 0.5f * dt;
    C.px = PER ? I.period[0] : 0;
    C.py = PER ? I.period[1] : 0;
    C.pz = PER ? I.period[2] : 0;
    if (!EARLY) {
      pi = PS[i];
      vi = VS[i];
      cnt = nbc[i];
    }
    C.dev_i = i2f(pi.w) + C.hdt * vi.w;               // Eq. verlet-first-half (density)
    C.rho_i = I.rho0 + C.dev_i;
    C.pr_i = I.c0sq * C.dev_i;                        // Eq. eqeos
    const float2 DQ = f2(I.dq);
    const int nf = (int)(cnt & 0xffffu), nw = (int)(cnt >> 16);
    const int nq = (nf + 3) >> 2;
    if (!EARLY && nq > 0) cur = nb4[i];
    for (int q = 0; q < nq; ++q) {
      int4 nxt = cur;
      if (q + 1 < nq) nxt = nb4[(int64_t)(q + 1) * n + i];  // next quad in flight
      const int s = q << 2;
      const int j0 = cur.x;
      const int j1 = s + 1 < nf ? cur.y : (int)i;                // self pads: zero terms
      const int j2 = s + 2 < nf ? cur.z : (int)i;
      const int j3 = s + 3 < nf ? cur.w : (int)i;
      int4 p0, p1, p2, p3;
      float4 g0 = float4(), g1 = float4(), g2 = float4(), g3 = float4();
      if (FG) {                                  // the frozen table holds the geometry: only dev_j here
        const int* __restrict__ dw = reinterpret_cast<const int*>(PS) + 3;
        p0 = make_int4(0, 0, 0, dw[4 * (int64_t)j0]);
        p1 = make_int4(0, 0, 0, dw[4 * (int64_t)j1]);
        p2 = make_int4(0, 0, 0, dw[4 * (int64_t)j2]);
        p3 = make_int4(0, 0, 0, dw[4 * (int64_t)j3]);
        const float4* __restrict__ gq = geo + (int64_t)s * n + i;
        g0 = gq[0];
        g1 = gq[n];
        g2 = gq[2 * n];
        g3 = gq[3 * n];
      } else {
        p0 = PS[j0];
        p1 = PS[j1];
        p2 = PS[j2];
        p3 = PS[j3];
      }
      const float4 v0 = VS[j0], v1 = VS[j1], v2v = VS[j2], v3 = VS[j3];
      float2 m01 = f2(I.mass), m23 = f2(I.mass);
      if (mass) {
        m01 = make_float2(mass[j0], mass[j1]);
        m23 = make_float2(mass[j2], mass[j3]);
      }
      pr_fluid2<D, PER, FG, TV>(I, C, pi, vi, p0, p1, v0, v1, m01, DQ, g0, g1);
      pr_fluid2<D, PER, FG, TV>(I, C, pi, vi, p2, p3, v2v, v3, m23, DQ, g2, g3);
      cur = nxt;
    }
    if (nw) {
      const int q0 = wall_slot0(nf) >> 2, nwq = (nw + 3) >> 2;
      for (int q = 0; q < nwq; ++q) {
        const int4 c = nb4[(int64_t)(q0 + q) * n + i];
        const int s = q << 2;
        const int w1 = s + 1 < nw ? c.y : c.x, w2 = s + 2 < nw ? c.z : c.x, w3 = s + 3 < nw ? c.w : c.x;
        const int4 a0 = WP[c.x], a1 = WP[w1], a2 = WP[w2], a3 = WP[w3];
        const float4 n0 = WN[c.x], n1 = WN[w1], n2 = WN[w2], n3 = WN[w3];
        const float2 V01 = make_float2(i2f(a0.w), s + 1 < nw ? i2f(a1.w) : 0.0f);   // pads carry no volume
        const float2 V23 = make_float2(s + 2 < nw ? i2f(a2.w) : 0.0f, s + 3 < nw ? i2f(a3.w) : 0.0f);
        float4 g0 = float4(), g1 = float4(), g2 = float4(), g3 = float4();
        if (FG) {
          const float4* __restrict__ gq = geo + (int64_t)((q0 + q) << 2) * n + i;
          g0 = gq[0];
          g1 = gq[n];
          g2 = gq[2 * n];
          g3 = gq[3 * n];
        }
        pr_wall2<D, PER, FG>(I, C, pi, vi, a0, a1, n0, n1, V01, DQ, g0, g1);
        pr_wall2<D, PER, FG>(I, C, pi, vi, a2, a3, n2, n3, V23, DQ, g2, g3);
      }
    }
  }
  float ax = (C.sx.x + C.nx.x) + (C.sx.y + C.nx.y);
  float ay = (C.sy.x + C.ny.x) + (C.sy.y + C.ny.y);
  float az = (C.sz.x + C.nz.x) + (C.sz.y + C.nz.y);
  if (valid) v2 = pr_finish<D, PER, TV>(I, C, i, dt, pi, vi, ax, ay, az, PH, VH, acc_prior, acc_keep, g);
  *writer_out = valid;
  return v2;
}

template <int D, bool PER, int TPP, int BLK, bool UNI, bool FG, bool TV = false>
__global__ void __launch_bounds__(BLK, pr_min_blocks(BLK))
k_pressure_relaxation(const Inst Ip, const float4* __restrict__ geo, int64_t n, const int4* __restrict__ PS,
                      const float4* __restrict__ VS,
                      int4* __restrict__ PH, float4* __restrict__ VH,
                      const float* __restrict__ mass, const int* __restrict__ inst_of,
                      const Inst* __restrict__ inst, Ctrl* ctrl, const int* __restrict__ nbr,
                      const uint32_t* __restrict__ nbc, const int4* __restrict__ WP,
                      const float4* __restrict__ WN, const float4* __restrict__ acc_prior,
                      float4* __restrict__ acc_keep, Global* g) {
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x / TPP) + lane_particle<TPP>();
  const int sub = lane_sub<TPP>();
  int kb;
  const bool uni = block_one_instance<TPP>(inst_of, n, &kb);
  bool valid = i < n;
  const int k = valid ? inst_index(inst_of, i) : kb;
  const double dtd = ctrl[k].dt;
  if (dtd == 0.0) valid = false;                 // tank idle for this substep
  const Inst& I = UNI ? Ip : inst[k];        // one tank: constants straight from the argument
  bool writer;
  float v2;
  if (TPP == 1) {
    v2 = pr_particle<D, PER, FG, TV, D == 2, const int4* __restrict__, const float4* __restrict__>(
        I, min(i, n - 1), valid, dtd, geo, n, PS, VS, PH, VH, mass, nbr, nbc, WP, WN, acc_prior, acc_keep, g, &writer);
  } else {
    static_assert(TPP == 1 || !FG, "frozen geometry: one thread per particle");
    __shared__ float4 terms[TPP > 1 ? BLK / 32 : 1][(1 + D + (TV ? 1 : 0)) * 32];
    RowHead head;
    head.load<TPP>(valid ? i : -1, sub, n, reinterpret_cast<const int4*>(nbr), nbc);
    v2 = pr_group<D, PER, TPP, TV>(I, i, sub, valid, dtd, n, PS, VS, PH, VH, mass,
                                   reinterpret_cast<const int4*>(nbr), head, WP, WN, acc_prior, acc_keep, g,
                                   terms[TPP > 1 ? threadIdx.x >> 5 : 0], &writer);
  }
  reduce_vmax(v2, writer, k, uni, ctrl);
}

// ---------------------------------------------------------------- density relaxation ---
struct DrCtx {
  float hdt, dev_i, rho_i;
  int px, py, pz;
  float2 s, nc;
};

// Two fluid pairs of the density relaxation: returns V_j (U* - U_L), and dW/dr in dw.
template <int D, bool PER, bool FG = false>
__device__ __forceinline__ float2 dr_fluid_term2(const Inst& I, const DrCtx& C, const int4& pi, const float4& vi,
                                                 const int4& pa, const int4& pb, const float4& va, const float4& vb,
                                                 float2 mj, float2 DQ, float2& dw, float4 ga = float4(),
                                                 float4 gb = float4()) {
  const float2 HDT = f2(C.hdt);
  float2 rx, ry, rz = f2(0.f);
  Geo2 G;
  if (FG) {
    rx = make_float2(ga.x, gb.x);
    ry = make_float2(ga.y, gb.y);
    if (D == 3) rz = make_float2(ga.z, gb.z);
    G = stored_geometry2(rx, ry, rz, make_float2(ga.w, gb.w));
  } else {
    // r_ij^{n+1} = r_ij^{n+1/2} + dt/2 (v_i - v_j)^{n+1}
    rx = pair_axis<PER>(pi.x, pa.x, pb.x, C.px, DQ, mul2(HDT, sub2(f2(vi.x), make_float2(va.x, vb.x))));
    ry = pair_axis<PER>(pi.y, pa.y, pb.y, C.py, DQ, mul2(HDT, sub2(f2(vi.y), make_float2(va.y, vb.y))));
    if (D == 3) rz = pair_axis<PER>(pi.z, pa.z, pb.z, C.pz, DQ, mul2(HDT, sub2(f2(vi.z), make_float2(va.z, vb.z))));
    G = geometry2(rx, ry, rz, I.inv_h, I.dwr_a);
  }
  const float2 dev_j = make_float2(i2f(pa.w), i2f(pb.w));
  const float2 rho_j = add2(f2(I.rho0), dev_j);
  // (U_R - U_L)/2 = (v_i - v_j).r_ij / (2 |r_ij|)
  const float2 dvx = sub2(f2(vi.x), make_float2(va.x, vb.x));
  const float2 dvy = sub2(f2(vi.y), make_float2(va.y, vb.y));
  const float2 dvz = sub2(f2(vi.z), make_float2(va.z, vb.z));
  const float2 half_dUR = mul2(fma2(dvx, rx, fma2(dvy, ry, mul2(dvz, rz))), mul2(G.inv_r, f2(0.5f)));
  // U* - U_L = (U_R - U_L)/2 + c0 (dev_i - dev_j)/(rho_i + rho_j)
  const float2 dUs = fma2(mul2(f2(I.c0), sub2(f2(C.dev_i), dev_j)), rcp2(add2(f2(C.rho_i), rho_j)), half_dUR);
  dw = mul2(G.fw, G.r);
  return mul2(mul2(mj, rcp2(rho_j)), dUs);
}

template <int D, bool PER, bool FG = false>
__device__ __forceinline__ void dr_fluid2(const Inst& I, DrCtx& C, const int4& pi, const float4& vi, const int4& pa,
                                          const int4& pb, const float4& va, const float4& vb, float2 mj,
                                          float2 DQ, float4 ga = float4(), float4 gb = float4()) {
  float2 dw;
  const float2 u = dr_fluid_term2<D, PER, FG>(I, C, pi, vi, pa, pb, va, vb, mj, DQ, dw, ga, gb);
  acc2(C.s, C.nc, u, dw);
}

template <int D, bool PER, bool FG = false>
__device__ __forceinline__ float2 dr_wall_term2(const Inst& I, const DrCtx& C, const int4& pi, const float4& vi,
                                                const int4& qa, const int4& qb, const float4& na,
                                                const float4& nb, float2 Vw, float2 DQ, float pr_i, float2& dw,
                                                float4 ga = float4(), float4 gb = float4()) {
  float2 rx, ry, rz = f2(0.f);
  Geo2 G;
  if (FG) {
    rx = make_float2(ga.x, gb.x);
    ry = make_float2(ga.y, gb.y);
    if (D == 3) rz = make_float2(ga.z, gb.z);
    G = stored_geometry2(rx, ry, rz, make_float2(ga.w, gb.w));
  } else {
    rx = pair_axis<PER>(pi.x, qa.x, qb.x, C.px, DQ, f2(C.hdt * vi.x));
    ry = pair_axis<PER>(pi.y, qa.y, qb.y, C.py, DQ, f2(C.hdt * vi.y));
    if (D == 3) rz = pair_axis<PER>(pi.z, qa.z, qb.z, C.pz, DQ, f2(C.hdt * vi.z));
    G = geometry2(rx, ry, rz, I.inv_h, I.dwr_a);
  }
  const float2 UL = mul2(f2(-1.0f), fma2(make_float2(na.x, nb.x), f2(vi.x),
                                         fma2(make_float2(na.y, nb.y), f2(vi.y), mul2(make_float2(na.z, nb.z), f2(vi.z)))));
  const float2 gr = fma2(f2(I.g[0]), rx, fma2(f2(I.g[1]), ry, mul2(f2(I.g[2]), rz)));
  const float2 PR = fma2(f2(-C.rho_i), gr, f2(pr_i));
  const float2 rhoR = fma2(PR, f2(I.inv_c0sq), f2(I.rho0));
  // U_R = -U_L: U* = (P_L - P_R)/(2 rho_bar c0) = rho_i g.r_iw / (c0 (rho_i + rho_R))
  const float2 Us = mul2(mul2(f2(C.rho_i), gr), rcp2(mul2(f2(I.c0), add2(f2(C.rho_i), rhoR))));
  dw = mul2(G.fw, G.r);
  return mul2(Vw, sub2(Us, UL));
}

template <int D, bool PER, bool FG = false>
__device__ __forceinline__ void dr_wall2(const Inst& I, DrCtx& C, const int4& pi, const float4& vi,
                                         const int4& qa, const int4& qb, const float4& na,
                                         const float4& nb, float2 Vw, float2 DQ, float pr_i,
                                         float4 ga = float4(), float4 gb = float4()) {
  float2 dw;
  const float2 u = dr_wall_term2<D, PER, FG>(I, C, pi, vi, qa, qb, na, nb, Vw, DQ, pr_i, dw, ga, gb);
  acc2(C.s, C.nc, u, dw);
}

// The end of one particle's density relaxation from its sum: rho to n+1, r to n+1
// (verlet-first-final), stored.
template <int D, bool PER>
__device__ __forceinline__ void dr_finish(const Inst& I, const DrCtx& C, int64_t i, const int4& pi, const float4& vi,
                                          float sum, int4* PS, float4* VS, Global* g) {
  const float drho = 2.0f * C.rho_i * sum;
  const float dev_n = C.dev_i + C.hdt * drho;         // Eq. verlet-first-final (density)
  const float hdt = C.hdt;
  int qx = pi.x + __float2int_rn(hdt * vi.x * I.inv_dq);
  int qy = pi.y + __float2int_rn(hdt * vi.y * I.inv_dq);
  int qz = D == 3 ? pi.z + __float2int_rn(hdt * vi.z * I.inv_dq) : 0;
  if (PER) {
    qx = wrap_coord(qx, C.px);
    qy = wrap_coord(qy, C.py);
    if (D == 3) qz = wrap_coord(qz, C.pz);
  }
  if (!isfinite(dev_n)) raise_error(g, ERR_NAN, i);
  PS[i] = make_int4(qx, qy, qz, f2i(dev_n));
  VS[i] = make_float4(vi.x, vi.y, vi.z, drho);
}

// One particle of the density relaxation shared by LPP lanes (as pr_group; terms: [2][32]).
template <int D, bool PER, int LPP, typename PI, typename PF, typename PM, typename PN>
__device__ __forceinline__ void dr_group(const Inst& I, int64_t i, int sub, double dtd, int64_t n, PI PH, PF VH,
                                         int4* PS, float4* VS, PM mass, PN nb4, const RowHead& head,
                                         const int4* __restrict__ WP,
                                         const float4* __restrict__ WN, Global* g, float4* terms) {
  DrCtx C;
  C.s = C.nc = f2(0.f);
  float2 sa[2] = {f2(0.f), f2(0.f)}, none[2];
  C.hdt = 0.5f * (float)dtd;
  C.px = PER ? I.period[0] : 0;
  C.py = PER ? I.period[1] : 0;
  C.pz = PER ? I.period[2] : 0;
  const int4 pi = PH[i];
  const float4 vi = VH[i];                            // v^{n+1}
  C.dev_i = i2f(pi.w);
  C.rho_i = I.rho0 + C.dev_i;
  const float2 DQ = f2(I.dq);
  const uint32_t cnt = head.cnt;
  const int nf = (int)(cnt & 0xffffu), nw = (int)(cnt >> 16);
  const int nq = (nf + 3) >> 2, lane = threadIdx.x & 31;
  int4 cur = head.quad;
  const float pr_i = I.c0sq * C.dev_i;
  auto fluid = [&](const int4& c, int s) {
    const int j0 = c.x;
    const int j1 = s + 1 < nf ? c.y : (int)i;
    const int j2 = s + 2 < nf ? c.z : (int)i;
    const int j3 = s + 3 < nf ? c.w : (int)i;
    const int4 p0 = PH[j0], p1 = PH[j1], p2 = PH[j2], p3 = PH[j3];
    const float4 v0 = VH[j0], v1 = VH[j1], v2 = VH[j2], v3 = VH[j3];
    float2 m01 = f2(I.mass), m23 = f2(I.mass);
    if (mass) {
      m01 = make_float2(mass[j0], mass[j1]);
      m23 = make_float2(mass[j2], mass[j3]);
    }
    if (LPP == 1) {
      dr_fluid2<D, PER>(I, C, pi, vi, p0, p1, v0, v1, m01, DQ);
      dr_fluid2<D, PER>(I, C, pi, vi, p2, p3, v2, v3, m23, DQ);
    } else {
      float2 d01, d23;
      const float2 u01 = dr_fluid_term2<D, PER>(I, C, pi, vi, p0, p1, v0, v1, m01, DQ, d01);
      const float2 u23 = dr_fluid_term2<D, PER>(I, C, pi, vi, p2, p3, v2, v3, m23, DQ, d23);
      terms[lane] = make_float4(u01.x, u01.y, u23.x, u23.y);
      terms[32 + lane] = make_float4(d01.x, d01.y, d23.x, d23.y);
    }
  };
  auto wall = [&](const int4& c, int s) {
    const int w1 = s + 1 < nw ? c.y : c.x, w2 = s + 2 < nw ? c.z : c.x, w3 = s + 3 < nw ? c.w : c.x;
    const int4 a0 = WP[c.x], a1 = WP[w1], a2 = WP[w2], a3 = WP[w3];
    const float4 n0 = WN[c.x], n1 = WN[w1], n2 = WN[w2], n3 = WN[w3];
    const float2 V01 = make_float2(i2f(a0.w), s + 1 < nw ? i2f(a1.w) : 0.0f);
    const float2 V23 = make_float2(s + 2 < nw ? i2f(a2.w) : 0.0f, s + 3 < nw ? i2f(a3.w) : 0.0f);
    if (LPP == 1) {
      dr_wall2<D, PER>(I, C, pi, vi, a0, a1, n0, n1, V01, DQ, pr_i);
      dr_wall2<D, PER>(I, C, pi, vi, a2, a3, n2, n3, V23, DQ, pr_i);
    } else {
      float2 d01, d23;
      const float2 u01 = dr_wall_term2<D, PER>(I, C, pi, vi, a0, a1, n0, n1, V01, DQ, pr_i, d01);
      const float2 u23 = dr_wall_term2<D, PER>(I, C, pi, vi, a2, a3, n2, n3, V23, DQ, pr_i, d23);
      terms[lane] = make_float4(u01.x, u01.y, u23.x, u23.y);
      terms[32 + lane] = make_float4(d01.x, d01.y, d23.x, d23.y);
    }
  };
  const int nwq = (nw + 3) >> 2;
  if (LPP == 1) {
    for (int q = 0; q < nq; ++q) {
      int4 nxt = cur;
      if (q + 1 < nq + nwq) nxt = nb4[(int64_t)(q + 1) * n + i];
      fluid(cur, q << 2);
      cur = nxt;
    }
    for (int q = 0; q < nwq; ++q) {
      int4 nxt = cur;
      if (q + 1 < nwq) nxt = nb4[(int64_t)(nq + q + 1) * n + i];
      wall(cur, q << 2);
      cur = nxt;
    }
  } else {
    for (int q0 = 0; q0 < nq + nwq; q0 += LPP) {
      const int q = q0 + sub;
      int4 nxt = cur;
      if (q + LPP < nq + nwq) nxt = nb4[(int64_t)(q + LPP) * n + i];
      if (q < nq) fluid(cur, q << 2);
      else if (q < nq + nwq) wall(cur, (q - nq) << 2);
      add_terms<LPP, 1>(terms, sub, min(LPP, nq + nwq - q0), sa, none);
      cur = nxt;
    }
  }
  float sum = (C.s.x + C.nc.x) + (C.s.y + C.nc.y);
  if (LPP > 1) {
    if (sub != 0) return;
    sum = (sa[0].x + 0.0f) + (sa[0].y + 0.0f);
  }
  dr_finish<D, PER>(I, C, i, pi, vi, sum, PS, VS, g);
}

// One particle of the density relaxation by one thread (pointer qualifiers as for
// pr_particle).
template <int D, bool PER, bool FG, typename PI, typename PF>
__device__ __forceinline__ void dr_particle(const Inst& I, int64_t i, bool valid, double dtd,
                                            const float4* __restrict__ geo, int64_t n, PI PH, PF VH,
                                            int4* PS, float4* VS, const float* __restrict__ mass,
                                            const int* __restrict__ nbr, const uint32_t* __restrict__ nbc,
                                            const int4* __restrict__ WP, const float4* __restrict__ WN, Global* g) {
  DrCtx C;
  C.s = C.nc = f2(0.f);
  int4 pi = make_int4(0, 0, 0, 0);
  float4 vi = make_float4(0.f, 0.f, 0.f, 0.f);
  C.hdt = 0.5f * (float)dtd;
  if (valid) {
    C.px = PER ? I.period[0] : 0;
    C.py = PER ? I.period[1] : 0;
    C.pz = PER ? I.period[2] : 0;
    pi = PH[i];
    vi = VH[i];                                       // v^{n+1}
    C.dev_i = i2f(pi.w);
    C.rho_i = I.rho0 + C.dev_i;
    const float2 DQ = f2(I.dq);
    const uint32_t cnt = nbc[i];
    const int nf = (int)(cnt & 0xffffu), nw = (int)(cnt >> 16);
    const int4* __restrict__ nb4 = reinterpret_cast<const int4*>(nbr);
    const int nq = (nf + 3) >> 2;
    int4 cur = nq > 0 ? nb4[i] : make_int4(0, 0, 0, 0);
    for (int q = 0; q < nq; ++q) {
      int4 nxt = cur;
      if (q + 1 < nq) nxt = nb4[(int64_t)(q + 1) * n + i];
      const int s = q << 2;
      const int j0 = cur.x;
      const int j1 = s + 1 < nf ? cur.y : (int)i;
      const int j2 = s + 2 < nf ? cur.z : (int)i;
      const int j3 = s + 3 < nf ? cur.w : (int)i;
      int4 p0, p1, p2, p3;
      float4 g0 = float4(), g1 = float4(), g2 = float4(), g3 = float4();
      if (FG) {                                  // the frozen table holds the geometry: only dev_j here
        const int* __restrict__ dw = reinterpret_cast<const int*>(PH) + 3;
        p0 = make_int4(0, 0, 0, dw[4 * (int64_t)j0]);
        p1 = make_int4(0, 0, 0, dw[4 * (int64_t)j1]);
        p2 = make_int4(0, 0, 0, dw[4 * (int64_t)j2]);
        p3 = make_int4(0, 0, 0, dw[4 * (int64_t)j3]);
        const float4* __restrict__ gq = geo + (int64_t)s * n + i;
        g0 = gq[0];
        g1 = gq[n];
        g2 = gq[2 * n];
        g3 = gq[3 * n];
      } else {
        p0 = PH[j0];
        p1 = PH[j1];
        p2 = PH[j2];
        p3 = PH[j3];
      }
      const float4 v0 = VH[j0], v1 = VH[j1], v2 = VH[j2], v3 = VH[j3];
      float2 m01 = f2(I.mass), m23 = f2(I.mass);
      if (mass) {
        m01 = make_float2(mass[j0], mass[j1]);
        m23 = make_float2(mass[j2], mass[j3]);
      }
      dr_fluid2<D, PER, FG>(I, C, pi, vi, p0, p1, v0, v1, m01, DQ, g0, g1);
      dr_fluid2<D, PER, FG>(I, C, pi, vi, p2, p3, v2, v3, m23, DQ, g2, g3);
      cur = nxt;
    }
    if (nw) {
      const float pr_i = I.c0sq * C.dev_i;
      const int q0 = wall_slot0(nf) >> 2, nwq = (nw + 3) >> 2;
      for (int q = 0; q < nwq; ++q) {
        const int4 c = nb4[(int64_t)(q0 + q) * n + i];
        const int s = q << 2;
        const int w1 = s + 1 < nw ? c.y : c.x, w2 = s + 2 < nw ? c.z : c.x, w3 = s + 3 < nw ? c.w : c.x;
        const int4 a0 = WP[c.x], a1 = WP[w1], a2 = WP[w2], a3 = WP[w3];
        const float4 n0 = WN[c.x], n1 = WN[w1], n2 = WN[w2], n3 = WN[w3];
        const float2 V01 = make_float2(i2f(a0.w), s + 1 < nw ? i2f(a1.w) : 0.0f);
        const float2 V23 = make_float2(s + 2 < nw ? i2f(a2.w) : 0.0f, s + 3 < nw ? i2f(a3.w) : 0.0f);
        float4 g0 = float4(), g1 = float4(), g2 = float4(), g3 = float4();
        if (FG) {
          const float4* __restrict__ gq = geo + (int64_t)((q0 + q) << 2) * n + i;
          g0 = gq[0];
          g1 = gq[n];
          g2 = gq[2 * n];
          g3 = gq[3 * n];
        }
        dr_wall2<D, PER, FG>(I, C, pi, vi, a0, a1, n0, n1, V01, DQ, pr_i, g0, g1);
        dr_wall2<D, PER, FG>(I, C, pi, vi, a2, a3, n2, n3, V23, DQ, pr_i, g2, g3);
      }
    }
  }
  const float sum = (C.s.x + C.nc.x) + (C.s.y + C.nc.y);
  if (!valid) return;
  dr_finish<D, PER>(I, C, i, pi, vi, sum, PS, VS, g);
}

template <int D, bool PER, int TPP, int BLK, bool UNI, bool FG>
__global__ void __launch_bounds__(BLK, dr_min_blocks(BLK))
k_density_relaxation(const Inst Ip, const float4* __restrict__ geo, int64_t n, const int4* __restrict__ PH,
                     const float4* __restrict__ VH,
                     int4* __restrict__ PS, float4* __restrict__ VS,
                     const float* __restrict__ mass, const int* __restrict__ inst_of,
                     const Inst* __restrict__ inst, const Ctrl* __restrict__ ctrl,
                     const int* __restrict__ nbr, const uint32_t* __restrict__ nbc,
                     const int4* __restrict__ WP, const float4* __restrict__ WN, Global* g) {
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x / TPP) + lane_particle<TPP>();
  const int sub = lane_sub<TPP>();
  if (TPP == 1 && i >= n) return;                     // no group shuffles to take part in
  bool valid = i < n;
  const int k = valid ? inst_index(inst_of, i) : 0;
  const double dtd = ctrl[k].dt;
  if (TPP == 1 && dtd == 0.0) return;
  if (dtd == 0.0) valid = false;
  const Inst& I = UNI ? Ip : inst[k];        // one tank: constants straight from the argument
  if (TPP == 1) {
    dr_particle<D, PER, FG, const int4* __restrict__, const float4* __restrict__>(
        I, i, valid, dtd, geo, n, PH, VH, PS, VS, mass, nbr, nbc, WP, WN, g);
  } else if (valid) {
    static_assert(TPP == 1 || !FG, "frozen geometry: one thread per particle");
    __shared__ float4 terms[TPP > 1 ? BLK / 32 : 1][2 * 32];
    RowHead head;
    head.load<TPP>(i, sub, n, reinterpret_cast<const int4*>(nbr), nbc);
    dr_group<D, PER, TPP>(I, i, sub, dtd, n, PH, VH, PS, VS, mass, reinterpret_cast<const int4*>(nbr), head, WP, WN, g,
                          terms[TPP > 1 ? threadIdx.x >> 5 : 0]);
  }
}

// ---------------------------------------------------------------- row-task form ---
// One resident block of kRowWarps warps an SM, one thread per particle. Each warp takes
// the next piece (32 consecutive particles of one search-cell row, `row_task`) from its
// block's queue: block b works through the runs of kRowWarps consecutive pieces numbered
// b, b + gridDim.x, b + 2 gridDim.x, ..., so the blocks move through the cell order side by
// side (the rows in flight share their neighbours in L1 and L2) and a warp that finishes
// early takes the next piece instead of waiting for the rest of its block. The particle
// arithmetic is that of the one-thread-per-particle kernels: results equal theirs bit for bit.
__device__ __forceinline__ bool next_row_piece(int* queue, int lane, long long pieces, long long* t_out) {
  int q = 0;
  if (lane == 0) q = atomicAdd(queue, 1);
  q = __shfl_sync(0xffffffffu, q, 0);
  const long long t = ((long long)blockIdx.x + (long long)gridDim.x * (q / kRowWarps)) * kRowWarps + q % kRowWarps;
  *t_out = t;
  return t < pieces;
}

template <int D, bool PER, bool TV>
__global__ void __launch_bounds__(kRowBlock, 1)
k_pressure_relaxation_rows(const Inst I, int64_t n, const int4* __restrict__ PS, const float4* __restrict__ VS,
                           int4* __restrict__ PH, float4* __restrict__ VH, const float* __restrict__ mass,
                           Ctrl* ctrl, const int* __restrict__ nbr, const uint32_t* __restrict__ nbc,
                           const int4* __restrict__ WP, const float4* __restrict__ WN,
                           const float4* __restrict__ acc_prior, float4* __restrict__ acc_keep, Global* g,
                           const int2* __restrict__ row_task, const uint32_t* __restrict__ row_total,
                           int64_t row_task_cap) {
  __shared__ int queue;
  __shared__ float red[kRowWarps];
  if (threadIdx.x == 0) queue = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const long long pieces = min((long long)*row_total, (long long)row_task_cap);
  const double dtd = ctrl[0].dt;
  float m = 0.0f;
  long long t;
  if (dtd != 0.0) {                              // 0: the tank is idle for this substep
    while (next_row_piece(&queue, lane, pieces, &t)) {
      const int2 piece = row_task[t];
      const bool valid = lane < piece.y;
      bool writer;
      const float v2 = pr_particle<D, PER, false, TV, false, const int4* __restrict__, const float4* __restrict__>(
          I, valid ? (int64_t)piece.x + lane : 0, valid, dtd, nullptr, n, PS, VS, PH, VH, mass, nbr, nbc,
          WP, WN, acc_prior, acc_keep, g, &writer);
      if (writer) m = fmaxf(m, v2);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = threadIdx.x < kRowWarps ? red[threadIdx.x] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) atomicMax(&ctrl[0].vmax2, __float_as_uint(m));
  }
}

template <int D, bool PER>
__global__ void __launch_bounds__(kRowBlock, 1)
k_density_relaxation_rows(const Inst I, int64_t n, const int4* __restrict__ PH, const float4* __restrict__ VH,
                          int4* __restrict__ PS, float4* __restrict__ VS, const float* __restrict__ mass,
                          const Ctrl* __restrict__ ctrl, const int* __restrict__ nbr,
                          const uint32_t* __restrict__ nbc, const int4* __restrict__ WP,
                          const float4* __restrict__ WN, Global* g, const int2* __restrict__ row_task,
                          const uint32_t* __restrict__ row_total, int64_t row_task_cap) {
  __shared__ int queue;
  if (threadIdx.x == 0) queue = 0;
  __syncthreads();
  const double dtd = ctrl[0].dt;
  if (dtd == 0.0) return;
  const int lane = threadIdx.x & 31;
  const long long pieces = min((long long)*row_total, (long long)row_task_cap);
  long long t;
  while (next_row_piece(&queue, lane, pieces, &t)) {
    const int2 piece = row_task[t];
    const bool valid = lane < piece.y;
    dr_particle<D, PER, false, const int4* __restrict__, const float4* __restrict__>(
        I, valid ? (int64_t)piece.x + lane : 0, valid, dtd, nullptr, n, PH, VH, PS, VS, mass, nbr, nbc,
        WP, WN, g);
  }
}

// Launch variants: (threads per particle, block size) per kernel, indexed by kTpp / kBlk.
template <int D, bool PER>
void launch_pr(int tpp, int block, const Buffers& b, cudaStream_t s) {
  const unsigned grid = grid_for(b.n * tpp, block);
#define SPH_PR_ARGS b.n, (const int4*)b.PS, (const float4*)b.VS, b.PH, b.VH, (const float*)b.mass, \
    b.inst_of, (const Inst*)b.inst, b.ctrl, (const int*)b.nbr, (const uint32_t*)b.nbc,                 \
    (const int4*)b.WP, (const float4*)b.WN, (const float4*)b.acc_prior, b.acc_keep, b.glob
  // one instantiation per (threads per particle, block) pair, each with its own bounds
#define SPH_PR(T, B) (b.n_inst == 1                                                                 \
      ? k_pressure_relaxation<D, PER, T, B, true, false><<<grid, B, 0, s>>>(b.inst0, nullptr, SPH_PR_ARGS) \
      : k_pressure_relaxation<D, PER, T, B, false, false><<<grid, B, 0, s>>>(b.inst0, nullptr, SPH_PR_ARGS))
  if (b.geo) {               // frozen geometry: one variant, one thread per particle
    const unsigned g1 = grid_for(b.n, 128);
    if (b.n_inst == 1) k_pressure_relaxation<D, PER, 1, 128, true, true><<<g1, 128, 0, s>>>(b.inst0, b.geo, SPH_PR_ARGS);
    else k_pressure_relaxation<D, PER, 1, 128, false, true><<<g1, 128, 0, s>>>(b.inst0, b.geo, SPH_PR_ARGS);
    return;
  }
  if (row_form(block)) {     // row-task form (one tank; the caller has built the pieces)
#define SPH_PR_ROWS(TV) k_pressure_relaxation_rows<D, PER, TV><<<b.n_sm, kRowBlock, 0, s>>>(                     \
      b.inst0, b.n, (const int4*)b.PS, (const float4*)b.VS, b.PH, b.VH, (const float*)b.mass, b.ctrl,          \
      (const int*)b.nbr, (const uint32_t*)b.nbc, (const int4*)b.WP, (const float4*)b.WN,                        \
      (const float4*)b.acc_prior, b.acc_keep, b.glob, b.row_task, b.row_off + b.n_rows, b.row_task_cap)
    if (b.any_transport) SPH_PR_ROWS(true);
    else SPH_PR_ROWS(false);
#undef SPH_PR_ROWS
    return;
  }
  if (b.any_transport) {     // transport velocity: one thread per particle, the configured block
    const unsigned g1 = grid_for(b.n, block);
#define SPH_PR_TV(B) (b.n_inst == 1                                                                \
      ? k_pressure_relaxation<D, PER, 1, B, true, false, true><<<g1, B, 0, s>>>(b.inst0, nullptr, SPH_PR_ARGS) \
      : k_pressure_relaxation<D, PER, 1, B, false, false, true><<<g1, B, 0, s>>>(b.inst0, nullptr, SPH_PR_ARGS))
    if (block == 512) SPH_PR_TV(512);
    else if (block == 256) SPH_PR_TV(256);
    else SPH_PR_TV(128);
#undef SPH_PR_TV
    return;
  }
#define SPH_PR_T(T) (block == 512 ? SPH_PR(T, 512) : block == 256 ? SPH_PR(T, 256) : SPH_PR(T, 128))
  if (tpp == 4) SPH_PR_T(4);
  else if (tpp == 2) SPH_PR_T(2);
  else SPH_PR_T(1);
#undef SPH_PR_T
#undef SPH_PR
#undef SPH_PR_ARGS
}

template <int D, bool PER>
void launch_dr(int tpp, int block, const Buffers& b, cudaStream_t s) {
  const unsigned grid = grid_for(b.n * tpp, block);
#define SPH_DR_ARGS b.n, (const int4*)b.PH, (const float4*)b.VH, b.PS, b.VS, (const float*)b.mass, \
    b.inst_of, (const Inst*)b.inst, (const Ctrl*)b.ctrl, (const int*)b.nbr, (const uint32_t*)b.nbc,   \
    (const int4*)b.WP, (const float4*)b.WN, b.glob
#define SPH_DR(T, B) (b.n_inst == 1                                                                 \
      ? k_density_relaxation<D, PER, T, B, true, false><<<grid, B, 0, s>>>(b.inst0, nullptr, SPH_DR_ARGS) \
      : k_density_relaxation<D, PER, T, B, false, false><<<grid, B, 0, s>>>(b.inst0, nullptr, SPH_DR_ARGS))
  if (b.geo) {
    const unsigned g1 = grid_for(b.n, 128);
    if (b.n_inst == 1) k_density_relaxation<D, PER, 1, 128, true, true><<<g1, 128, 0, s>>>(b.inst0, b.geo, SPH_DR_ARGS);
    else k_density_relaxation<D, PER, 1, 128, false, true><<<g1, 128, 0, s>>>(b.inst0, b.geo, SPH_DR_ARGS);
    return;
  }
  if (row_form(block)) {     // row-task form (one tank; the caller has built the pieces)
    k_density_relaxation_rows<D, PER><<<b.n_sm, kRowBlock, 0, s>>>(
        b.inst0, b.n, (const int4*)b.PH, (const float4*)b.VH, b.PS, b.VS, (const float*)b.mass,
        (const Ctrl*)b.ctrl, (const int*)b.nbr, (const uint32_t*)b.nbc, (const int4*)b.WP, (const float4*)b.WN,
        b.glob, b.row_task, b.row_off + b.n_rows, b.row_task_cap);
    return;
  }
#define SPH_DR_T(T) (block == 512 ? SPH_DR(T, 512) : block == 256 ? SPH_DR(T, 256) : SPH_DR(T, 128))
  if (tpp == 4) SPH_DR_T(4);
  else if (tpp == 2) SPH_DR_T(2);
  else SPH_DR_T(1);
#undef SPH_DR_T
#undef SPH_DR
#undef SPH_DR_ARGS
}

}  // namespace

}  // namespace sph
