// Per-particle density summation and viscous acceleration (once per advection step), shared
// by the per-launch kernels (sph_physics.cu) and the one-launch step (sph_fused_step.cuh).
//
// LPP lanes share one particle: lane `sub` evaluates quads sub, sub + LPP, ... of its row and
// the terms are added in row order through shared memory, so the sums are those of one lane
// bit for bit. Array types carry the caller's aliasing qualifiers.
#pragma once
#include "sph_kernels.h"

namespace sph {
namespace {

// the lanes p, p + 32 / LPP, ... of particle p of a warp
template <int LPP>
__device__ __forceinline__ unsigned row_lanes_mask() {
  return (LPP == 2 ? 0x00010001u : LPP == 4 ? 0x01010101u : 0x11111111u) << (threadIdx.x & (32 / LPP - 1));
}

// W of two pairs at once from their packed squared distances; lanes with mask 0 add 0.
__device__ __forceinline__ float2 kernel_W2(float2 r2, float inv_h, float w_a) {
  const float2 q = mul2(mul2(r2, rsqrt2(fma2(r2, f2(1.0f), f2(1e-30f)))), f2(inv_h));
  const float2 t = max2(fma2(q, f2(-0.5f), f2(1.0f)), 0.0f);
  const float2 t2 = mul2(t, t);
  return mul2(mul2(f2(w_a), mul2(t2, t2)), fma2(q, f2(2.0f), f2(1.0f)));
}

template <int D, bool PER>
__device__ __forceinline__ float2 pair_r2(const int4& p, const int4& a, const int4& b, const Inst& I) {
  const float2 M = f2(-kMagic), DQ = f2(I.dq);
  const float2 dx = mul2(add2(make_float2(biased_diff<PER>(p.x, a.x, I.period[0]), biased_diff<PER>(p.x, b.x, I.period[0])), M), DQ);
  const float2 dy = mul2(add2(make_float2(biased_diff<PER>(p.y, a.y, I.period[1]), biased_diff<PER>(p.y, b.y, I.period[1])), M), DQ);
  float2 r2 = fma2(dx, dx, mul2(dy, dy));
  if (D == 3) {
    const float2 dz = mul2(add2(make_float2(biased_diff<PER>(p.z, a.z, I.period[2]), biased_diff<PER>(p.z, b.z, I.period[2])), M), DQ);
    r2 = fma2(dz, dz, r2);
  }
  return r2;
}

// Eq. eqrhosum / Eq. eqrhosumnosurface: rho = rho0 sum W / sum W0 (with max(rho*, .) for a
// free surface), sum over self, fluid and wall neighbours. The Kahan sum starts from
// W(0) - sumW0 so it holds the deviation rho/rho0 - 1 with its own relative precision.
// Returns rho - rho0 (valid on lane 0 of a group); terms (LPP > 1): this warp's [32] float4.
template <int D, bool PER, int LPP, typename PP, typename PN>
__device__ __forceinline__ float density_dev(const Inst& I, int64_t i, int sub, const int4& pi, uint32_t c, int64_t n,
                                             PP P, PN nb4, const int4* __restrict__ WP, float4* terms) {
  const int nf = (int)(c & 0xffffu), nw = (int)(c >> 16);
  float2 s = make_float2(I.sig_hi, 0.0f), nc = f2(0.0f);
  kahan2(s, nc, make_float2(I.sig_lo, 0.0f), f2(1.0f));
  const int base = threadIdx.x & (32 / LPP - 1);
  auto add = [&](float4 w, int sl, int cnt) {      // the terms of one quad; slots past cnt add nothing
    kahan2(s, nc, make_float2(w.x, w.y), make_float2(1.0f, sl + 1 < cnt ? 1.0f : 0.0f));
    kahan2(s, nc, make_float2(w.z, w.w), make_float2(sl + 2 < cnt ? 1.0f : 0.0f, sl + 3 < cnt ? 1.0f : 0.0f));
  };
  auto pairs = [&](const int4& a0, const int4& a1, const int4& a2, const int4& a3) {
    const float2 w01 = kernel_W2(pair_r2<D, PER>(pi, a0, a1, I), I.inv_h, I.w_a);
    const float2 w23 = kernel_W2(pair_r2<D, PER>(pi, a2, a3, I), I.inv_h, I.w_a);
    return make_float4(w01.x, w01.y, w23.x, w23.y);
  };
  const int nq = (nf + 3) >> 2, quads = nq + ((nw + 3) >> 2);       // wall quads follow the fluid's
  int4 nxt = sub < quads ? nb4[(int64_t)sub * n + i] : make_int4(0, 0, 0, 0);
  auto quad = [&](int q, bool fluid) {              // the terms of quad q, the lane's next one in flight
    const int4 c = nxt;
    if (q + LPP < quads) nxt = nb4[(int64_t)(q + LPP) * n + i];
    const int sl = (fluid ? q : q - nq) << 2, cnt = fluid ? nf : nw;
    const int j1 = sl + 1 < cnt ? c.y : c.x, j2 = sl + 2 < cnt ? c.z : c.x, j3 = sl + 3 < cnt ? c.w : c.x;
    return fluid ? pairs(P[c.x], P[j1], P[j2], P[j3]) : pairs(WP[c.x], WP[j1], WP[j2], WP[j3]);
  };
  if (LPP == 1) {
    for (int q = 0; q < nq; ++q) add(quad(q, true), q << 2, nf);
    for (int q = nq; q < quads; ++q) add(quad(q, false), (q - nq) << 2, nw);
  } else {
    for (int q0 = 0; q0 < quads; q0 += LPP) {       // one round of quads, added in row order
      const int q = q0 + sub;
      if (q < quads) terms[threadIdx.x & 31] = quad(q, q < nq);
      __syncwarp(row_lanes_mask<LPP>());
      if (sub == 0)
        for (int k = 0; k < LPP && q0 + k < quads; ++k) {
          const bool fluid = q0 + k < nq;
          add(terms[base + k * (32 / LPP)], (fluid ? q0 + k : q0 + k - nq) << 2, fluid ? nf : nw);
        }
      __syncwarp(row_lanes_mask<LPP>());
    }
  }
  float dev = I.rho0_over_sigma0 * ((s.x + nc.x) + (s.y + nc.y));   // rho0 sumW/sumW0 - rho0
  if (I.free_surface) dev = fmaxf(i2f(pi.w), dev);
  return dev;
}

// Eq. eqviscous over the fluid pairs: (2 eta / rho_i) sum_j V_j (dW/dr)/r (v_i - v_j), pairs
// past 2h or at zero distance adding nothing. The four records of a quad are gathered
// together. terms (LPP > 1): this warp's [1 + D][32] float4; the result is valid on lane 0.
template <int D, bool PER, int LPP, typename PP, typename PV, typename PM, typename PN>
__device__ __forceinline__ float4 viscous_acc(const Inst& I, int64_t i, int sub, int nf, int64_t n, PP P, PV V, PM mass,
                                              PN nb4, float4* terms) {
  if (!(I.eta > 0.0f)) nf = 0;
  const int4 pi = P[i];
  const float4 vi = V[i];
  const float rho_i = I.rho0 + i2f(pi.w);
  float ax = 0.f, ay = 0.f, az = 0.f;
  const int nq = (nf + 3) >> 2, lane = threadIdx.x & 31, base = lane & (32 / LPP - 1);
  int4 nxt = sub < nq ? nb4[(int64_t)sub * n + i] : make_int4(0, 0, 0, 0);
  for (int q0 = 0; q0 < nq; q0 += LPP) {
    const int q = q0 + sub;
    if (LPP == 1 || q < nq) {
      const int4 cq = nxt;
      if (q + LPP < nq) nxt = nb4[(int64_t)(q + LPP) * n + i];
      const int sl = q << 2;
      const int j[4] = {cq.x, sl + 1 < nf ? cq.y : cq.x, sl + 2 < nf ? cq.z : cq.x, sl + 3 < nf ? cq.w : cq.x};
      int4 pj[4];
      float4 vj[4];
      float mj[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        pj[k] = P[j[k]];
        vj[k] = V[j[k]];
        mj[k] = mass ? mass[j[k]] : I.mass;
      }
      float f[4], ux[4], uy[4], uz[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float dx = (float)wrap_diff(pi.x - pj[k].x, PER ? I.period[0] : 0) * I.dq;
        const float dy = (float)wrap_diff(pi.y - pj[k].y, PER ? I.period[1] : 0) * I.dq;
        float r2 = dx * dx + dy * dy;
        if (D == 3) {
          const float dz = (float)wrap_diff(pi.z - pj[k].z, PER ? I.period[2] : 0) * I.dq;
          r2 += dz * dz;
        }
        const float fw = kernel_dW_over_r(sqrtf(r2), I);            // (dW/dr)/r
        const bool in = r2 < I.four_h2 && r2 != 0.0f && sl + k < nf;
        f[k] = in ? mj[k] / (I.rho0 + i2f(pj[k].w)) * fw : 0.0f;
        ux[k] = in ? vi.x - vj[k].x : 0.0f;
        uy[k] = in ? vi.y - vj[k].y : 0.0f;
        uz[k] = D == 3 && in ? vi.z - vj[k].z : 0.0f;
      }
      if (LPP == 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          ax = fmaf(f[k], ux[k], ax);
          ay = fmaf(f[k], uy[k], ay);
          if (D == 3) az = fmaf(f[k], uz[k], az);
        }
      } else {
        terms[lane] = make_float4(f[0], f[1], f[2], f[3]);
        terms[32 + lane] = make_float4(ux[0], ux[1], ux[2], ux[3]);
        terms[64 + lane] = make_float4(uy[0], uy[1], uy[2], uy[3]);
        if (D == 3) terms[96 + lane] = make_float4(uz[0], uz[1], uz[2], uz[3]);
      }
    }
    if (LPP > 1) {
      __syncwarp(row_lanes_mask<LPP>());
      if (sub == 0)
        for (int k = 0; k < LPP && q0 + k < nq; ++k) {
          const int at = base + k * (32 / LPP);
          const float4 fk = terms[at], x = terms[32 + at], y = terms[64 + at];
          ax = fmaf(fk.w, x.w, fmaf(fk.z, x.z, fmaf(fk.y, x.y, fmaf(fk.x, x.x, ax))));
          ay = fmaf(fk.w, y.w, fmaf(fk.z, y.z, fmaf(fk.y, y.y, fmaf(fk.x, y.x, ay))));
          if (D == 3) {
            const float4 z = terms[96 + at];
            az = fmaf(fk.w, z.w, fmaf(fk.z, z.z, fmaf(fk.y, z.y, fmaf(fk.x, z.x, az))));
          }
        }
      __syncwarp(row_lanes_mask<LPP>());
    }
  }
  const float s = 2.0f * I.eta / rho_i;
  return make_float4(s * ax, s * ay, s * az, 0.0f);
}

}  // namespace
}  // namespace sph
