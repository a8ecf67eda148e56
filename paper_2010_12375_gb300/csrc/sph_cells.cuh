// Device helpers of the configuration update shared by the per-launch kernels
// (sph_cells.cu) and the one-launch step (sph_fused_step.cuh).
#pragma once
#include "sph_kernels.h"

namespace sph {
namespace {

__device__ __forceinline__ void raise_error(Global* g, int bit, long long idx) {
  int old = atomicOr(&g->err, bit);
  if (old == 0) g->bad_index = idx;
}

// Search cell of a particle, half a position cell per axis (flattened x fastest, with the
// tank's first cell added); outside the grid: an error and the nearest cell.
template <int D>
__device__ __forceinline__ uint32_t hash_cell(const Inst& I, const int4& p, long long i, Global* g) {
  int q[3] = {p.x, p.y, p.z};
  long long c = 0, stride = 1;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    int ca = q[a] >> I.sbits;
    if (ca < 0 || ca >= I.scell[a]) {
      raise_error(g, ERR_DOMAIN, i);
      ca = ca < 0 ? 0 : I.scell[a] - 1;
    }
    c += (long long)ca * stride;
    stride *= I.scell[a];
  }
  return (uint32_t)(c + I.cell_base);
}

__device__ __forceinline__ int wrap_cell(int c, int n) { return c < 0 ? c + n : (c >= n ? c - n : c); }

// Distance (quanta) from a point at offset o inside its search cell (width S) to the
// slab of the cell d rows away; exact integers below 2^23, so exact in FP32.
__device__ __forceinline__ float slab_gap(int d, float o, float S) {
  return d > 0 ? (float)d * S - o : (d < 0 ? o + (float)(-d - 1) * S + 1.0f : 0.0f);
}

// Flattened search cell of a particle (clamped to its tank's grid).
template <int D>
__device__ __forceinline__ long long search_cell(const Inst& I, const int4& p) {
  const int sb = I.sbits;
  const int cx = min(max(p.x >> sb, 0), I.scell[0] - 1);
  const int cy = min(max(p.y >> sb, 0), I.scell[1] - 1);
  const int cz = D == 3 ? min(max(p.z >> sb, 0), I.scell[2] - 1) : 0;
  return I.cell_base + ((long long)cz * I.scell[1] + cy) * I.scell[0] + cx;
}

// The runs of one row of search cells (first cell `row`) that meet a chord of half length
// sqrt(rem) around x: one contiguous slot range, or two where a periodic x axis splits it.
template <bool PER, typename F>
__device__ __forceinline__ void chord_runs(const Inst& I, int x, float rem, long long row, const uint32_t* start,
                                           F&& visit) {
  const int nx = I.scell[0];
  // |dx| of a neighbour is below sqrt(rem); rsqrt-based root within 2 quanta. A coordinate in
  // the grid lies in [0, 2^31) and the root below 2^23, so the upper end fits 32 unsigned bits.
  const int xr = (int)(rem * rsqrtf(rem)) + 2;
  int xa = (x - xr) >> I.sbits, xb = (int)(((unsigned)x + (unsigned)xr) >> I.sbits);
  if (PER && I.period[0]) {
    if (xa < 0) {
      visit(start[row + xa + nx], start[row + nx]);
      xa = 0;
    }
    if (xb >= nx) {
      visit(start[row + xa], start[row + nx]);
      visit(start[row], start[row + xb - nx + 1]);
      return;
    }
  } else {
    xa = max(xa, 0);
    xb = min(xb, nx - 1);
    if (xa > xb) return;
  }
  visit(start[row + xa], start[row + xb + 1]);
}

// Visit the search-cell runs that can hold a neighbour of the particle at p: for every
// row (dy, dz) in [-2, 2]^(D-1) whose slab lies closer than 2h, the x cells that meet the
// sphere's chord in that slab. Within a row the cells of a run are one contiguous slot
// range; a periodic x axis splits a run that crosses the edge into two. The row test and
// the chord are evaluated in FP32 against R2 (1 + 2^-20), a margin above every rounding
// error of the squares, so they only ever err towards visiting more: a particle j in a
// skipped row or cell has sum (q_i - q_j)^2 >= R2 and is not a neighbour.
template <int D, bool PER, typename F>
__device__ __forceinline__ void for_neighbour_runs(const Inst& I, const int4& p,
                                                   const uint32_t* start, F&& visit) {
  const int sb = I.sbits;
  const float S = (float)(1 << sb);
  const int nx = I.scell[0], ny = I.scell[1], nz = D == 3 ? I.scell[2] : 1;
  const int cy = min(max(p.y >> sb, 0), ny - 1);
  const int cz = D == 3 ? min(max(p.z >> sb, 0), nz - 1) : 0;
  const float oy = (float)(p.y - (cy << sb));
  const float oz = D == 3 ? (float)(p.z - (cz << sb)) : 0.0f;
  const float R2m = (float)I.R2 * (1.0f + 9.5367431640625e-07f);
  const long long base = I.cell_base;
  for (int dz = (D == 3 ? -2 : 0); dz <= (D == 3 ? 2 : 0); ++dz) {
    int z = 0;
    float gz2 = 0.0f;
    if (D == 3) {
      const int zu = cz + dz;
      if (PER && I.period[2]) z = wrap_cell(zu, nz);
      else if (zu < 0 || zu >= nz) continue;
      else z = zu;
      const float gz = fmaxf(slab_gap(dz, oz, S), 0.0f);
      gz2 = gz * gz;
      if (gz2 >= R2m) continue;
    }
    for (int dy = -2; dy <= 2; ++dy) {
      const int yu = cy + dy;
      int y;
      if (PER && I.period[1]) y = wrap_cell(yu, ny);
      else if (yu < 0 || yu >= ny) continue;
      else y = yu;
      const float gy = fmaxf(slab_gap(dy, oy, S), 0.0f);
      const float rem = R2m - gz2 - gy * gy;
      if (rem <= 0.0f) continue;
      chord_runs<PER>(I, p.x, rem, base + ((long long)z * ny + y) * nx, start, visit);
    }
  }
}

// Appends neighbour indices to one particle's quad-interleaved row (slot s of particle i
// at ((s >> 2) n + i) 4 + (s & 3)) with a running pointer instead of a product per slot.
struct RowWriter {
  int* p;
  int64_t stride;   // 4n ints between consecutive quads of one particle
  int sub, count, cap;
  __device__ __forceinline__ RowWriter(int* nbr, int64_t n, int64_t i, int slot0, int cap_)
      : p(nbr + ((int64_t)(slot0 >> 2) * n + i) * 4), stride(4 * n), sub(slot0 & 3), count(0), cap(cap_ - slot0) {}
  __device__ __forceinline__ void push(int j, bool& overflow) {
    if (count < cap) {
      p[sub] = j;
      if (++sub == 4) {
        sub = 0;
        p += stride;
      }
    } else {
      overflow = true;
    }
    ++count;
  }
};

// Candidate test: the squared distance in FP32 from exactly converted integer differences
// (error < 3 ulp) less R2; only within 2^-19 R2 of the threshold is the exact integer test
// needed, so the decision is always the integer one. Two candidates at once in the lanes of
// packed FP32 instructions; a candidate is a neighbour when its key is negative (callers take
// the sign bit as it is). The exact test sits behind a warp vote: a warp takes it only when
// one of its candidates falls in the band.
template <int D, bool PER>
__device__ __forceinline__ float2 candidate_keys(const int4& p, const int4& a, const int4& b, const Inst& I, float R2f,
                                                 float band) {
  const float2 M = f2(-kMagic);
  const float2 dx = add2(make_float2(biased_diff<PER>(p.x, a.x, I.period[0]), biased_diff<PER>(p.x, b.x, I.period[0])), M);
  const float2 dy = add2(make_float2(biased_diff<PER>(p.y, a.y, I.period[1]), biased_diff<PER>(p.y, b.y, I.period[1])), M);
  float2 d2 = fma2(dx, dx, mul2(dy, dy));
  if (D == 3) {
    const float2 dz = add2(make_float2(biased_diff<PER>(p.z, a.z, I.period[2]), biased_diff<PER>(p.z, b.z, I.period[2])), M);
    d2 = fma2(dz, dz, d2);
  }
  float2 key = add2(d2, f2(-R2f));
  if (__any_sync(__activemask(), fminf(fabsf(key.x), fabsf(key.y)) < band)) {
    if (fabsf(key.x) < band) key.x = within<D>(p, a, I) ? -1.0f : 1.0f;
    if (fabsf(key.y) < band) key.y = within<D>(p, b, I) ? -1.0f : 1.0f;
  }
  return key;
}
// bits shifted up by one, with the sign bit of key below
__device__ __forceinline__ unsigned push_sign(unsigned bits, float key) {
  return __funnelshift_l(__float_as_uint(key), bits, 1);
}

// Row r of for_neighbour_runs on a grid without periodic axes, (dz, dy) = (r / 5 - 2,
// r % 5 - 2) (2D: dy = r - 2): visit(first, last) with the cells [first, last) that meet the
// sphere's chord, if there are any.
template <int D, typename F>
__device__ __forceinline__ void row_cells(const Inst& I, const int4& p, int r, F&& visit) {
  const int sb = I.sbits;
  const float S = (float)(1 << sb);
  const int nx = I.scell[0], ny = I.scell[1], nz = D == 3 ? I.scell[2] : 1;
  const int cy = min(max(p.y >> sb, 0), ny - 1);
  const int cz = D == 3 ? min(max(p.z >> sb, 0), nz - 1) : 0;
  const int dz = D == 3 ? r / 5 - 2 : 0, dy = D == 3 ? r % 5 - 2 : r - 2;
  const int z = cz + dz, y = cy + dy;
  if (z < 0 || z >= nz || y < 0 || y >= ny) return;
  const float R2m = (float)I.R2 * (1.0f + 9.5367431640625e-07f);
  const float gz = D == 3 ? fmaxf(slab_gap(dz, (float)(p.z - (cz << sb)), S), 0.0f) : 0.0f;
  const float gy = fmaxf(slab_gap(dy, (float)(p.y - (cy << sb)), S), 0.0f);
  const float gz2 = gz * gz;
  if (D == 3 && gz2 >= R2m) return;
  const float rem = R2m - gz2 - gy * gy;
  if (rem <= 0.0f) return;
  const int xr = (int)(rem * rsqrtf(rem)) + 2;                // as in chord_runs
  const int xa = max((p.x - xr) >> sb, 0), xb = min((int)(((unsigned)p.x + (unsigned)xr) >> sb), nx - 1);
  if (xa > xb) return;
  const long long row = I.cell_base + ((long long)z * ny + y) * nx;
  visit(row + xa, row + xb + 1);
}

// The rows (dz, dy) = (r / 5 - 2, r % 5 - 2) (2D: dy = r - 2), r in [r0, r1), of
// for_neighbour_runs, in its order: the share of one of the lanes that split a particle's
// search.
template <int D, bool PER, typename F>
__device__ __forceinline__ void for_neighbour_rows(const Inst& I, const int4& p, const uint32_t* start, int r0, int r1,
                                                   F&& visit) {
  const int sb = I.sbits;
  const float S = (float)(1 << sb);
  const int nx = I.scell[0], ny = I.scell[1], nz = D == 3 ? I.scell[2] : 1;
  const int cy = min(max(p.y >> sb, 0), ny - 1);
  const int cz = D == 3 ? min(max(p.z >> sb, 0), nz - 1) : 0;
  const float oy = (float)(p.y - (cy << sb));
  const float oz = D == 3 ? (float)(p.z - (cz << sb)) : 0.0f;
  const float R2m = (float)I.R2 * (1.0f + 9.5367431640625e-07f);
  for (int r = r0; r < r1; ++r) {
    const int dz = D == 3 ? r / 5 - 2 : 0, dy = D == 3 ? r % 5 - 2 : r - 2;
    int z = cz + dz, y = cy + dy;
    if (D == 3) {
      if (PER && I.period[2]) z = wrap_cell(z, nz);
      else if (z < 0 || z >= nz) continue;
    }
    if (PER && I.period[1]) y = wrap_cell(y, ny);
    else if (y < 0 || y >= ny) continue;
    const float gz = D == 3 ? fmaxf(slab_gap(dz, oz, S), 0.0f) : 0.0f;
    const float gy = fmaxf(slab_gap(dy, oy, S), 0.0f);
    const float gz2 = gz * gz;
    if (D == 3 && gz2 >= R2m) continue;
    const float rem = R2m - gz2 - gy * gy;
    if (rem <= 0.0f) continue;
    chord_runs<PER>(I, p.x, rem, I.cell_base + ((long long)z * ny + y) * nx, start, visit);
  }
}

}  // namespace
}  // namespace sph
