// Whole advection steps of one tank in one cooperative launch: the configuration update,
// Dt_ad, the density re-initialisation, the viscous acceleration and every acoustic substep,
// as phases separated by grid-wide barriers, for as many steps as the launch is asked for.
//
// A tank that fits the GPU at once is bound by latency, not by throughput: step by step it
// runs some 13 launches for the configuration update and three a substep, each a few
// microseconds of dependent memory round trips by a fraction of the SMs. Here
//  - a phase ends with one barrier (an arrival on a counter and a poll, about a microsecond)
//    instead of a kernel boundary;
//  - up to eight lanes (LPP) share a particle: they split its search
//    rows and its neighbour row, so its chain of dependent loads is LPP times shorter, and
//    exchange the terms through shared memory, which are added in row order;
//  - the search takes a lane per row of search cells (8 lanes a particle in 2D, a warp in
//    3D), which remembers its hits as bits and writes them at its place in the row;
//  - every block keeps the time-step control (Eqs. dt-advection, dt-relax: some 3,000 cycles
//    of FP64) for itself, in a warp of its own that runs it beside the neighbour search and
//    each density relaxation;
//  - where each thread has one particle a step, the counts and first quads of its row stay
//    in registers over the substeps;
//  - reordered records go to the half-step arrays, the search reads them there and writes
//    each particle's own record back, so no pass copies them;
//  - the scan of the cell counts leaves the counts zero for the next step.
// A step after the first (of a launch or, with `follow`, of a call) goes no further than its hash
// once the status holds an error: the scan and the scatter would build on counts that a launch
// whose barrier gave up has left half filled, and on barriers whose arrivals it has left counted.
// The status is read beside the hash and looked at behind its barrier, where it costs nothing (a
// test before the hash took 2 us a step). The errors of a step's own hash wait in StepCtl until
// then, so that all blocks see the same status.
// Every sum adds the terms the per-launch kernels add in their order: the state is identical
// to theirs bit for bit, whatever the launch configuration.
// A further step of the 2D dam break takes 55 us at 3,200 particles and 158 us at 100,352 (132
// and 184 us in the graph loop's launches), of the 3D one 153 us at 16,000 (275 us).
//
// Memory ordering: a phase gathers what other blocks wrote in the one before, so everything
// written here is read through plain coherent loads (sph_grid_sync.cuh has the barrier and
// its bounded wait).
#pragma once
#include <algorithm>

#include "sph_cells.cuh"
#include "sph_ctrl.cuh"
#include "sph_density.cuh"
#include "sph_grid_sync.cuh"
#define SPH_HAVE_RAISE_ERROR
#include "sph_relax.cuh"

namespace sph {
namespace {

// One block an SM: its work warps and one control warp.
template <int LPP>
constexpr int kStepThreads = LPP <= 2 ? 704 : 512;   // most work threads: 88 and 96 registers
constexpr int kStepMaxWarps = 704 / 32 + 1;

// Sum of v over the block, and the exclusive prefix of this thread.
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* warp_tot, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  __syncthreads();                               // warp_tot free
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  uint32_t before = 0, all = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    const uint32_t t = warp_tot[w];
    before += w < warp ? t : 0u;
    all += t;
  }
  *total = all;
  return before + incl - v;
}

// Elements [k, k + 4) of an array up to `end`, k a multiple of four (zeros past the end).
__device__ __forceinline__ uint4 load4(const uint32_t* a, int64_t k, int64_t end) {
  if (k + 4 <= end) return *reinterpret_cast<const uint4*>(a + k);
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (k < end) v.x = a[k];
  if (k + 1 < end) v.y = a[k + 1];
  if (k + 2 < end) v.z = a[k + 2];
  return v;
}
__device__ __forceinline__ void store4(uint32_t* a, int64_t k, int64_t end, uint4 v) {
  if (k + 4 <= end) {
    *reinterpret_cast<uint4*>(a + k) = v;
    return;
  }
  if (k < end) a[k] = v.x;
  if (k + 1 < end) a[k + 1] = v.y;
  if (k + 2 < end) a[k + 2] = v.z;
}

// LS consecutive lanes
template <int LS>
__device__ __forceinline__ unsigned search_mask() {
  return LS == 32 ? 0xffffffffu : ((1u << (LS & 31)) - 1u) << ((threadIdx.x & 31) & ~(LS - 1));
}

// Inclusive prefix of v over LS consecutive lanes, and their sum.
template <int LS>
__device__ __forceinline__ int lanes_prefix(int v, int r, int* total) {
  const unsigned gm = search_mask<LS>();
  int incl = v;
#pragma unroll
  for (int o = 1; o < LS; o <<= 1) {
    const int y = __shfl_up_sync(gm, incl, o, LS);
    if (r >= o) incl += y;
  }
  *total = __shfl_sync(gm, incl, LS - 1, LS);
  return incl;
}

// Neighbour row of particle i (records P in their new order) by a group of LS lanes, lane r
// taking search row r: the row is the one a single thread writes going through the rows in
// order. The fluid and the wall candidates of a row come together (their first four records
// each in flight at once); a lane keeps its hits as bits, and the counts' prefix over the
// group is its place in the row; a run of more than 32 candidates is tested again for the
// write. Returns nf | nw << 16 in every lane.
template <int D, int LS>
__device__ __forceinline__ uint32_t search_group(const Buffers& b, const Inst& I, int64_t i, int r, const int4& pi,
                                                 const int4* P) {
  constexpr int kRows = D == 3 ? 25 : 5;
  static_assert(LS >= kRows, "a lane per search row");
  const float R2f = (float)I.R2, band = R2f * 1.9073486328125e-06f;
  const uint32_t me = (uint32_t)i;
  uint32_t s[2] = {0u, 0u}, e[2] = {0u, 0u};      // the row's run of fluid and of wall records
  if (r < kRows)
    row_cells<D>(I, pi, r, [&](long long first, long long last) {
      s[0] = b.fstart[first];
      e[0] = b.fstart[last];
      if (b.nw) {
        s[1] = b.wstart[first];
        e[1] = b.wstart[last];
      }
    });
  // four records from j on (clamped to the run), and which of them are hits
  auto four = [&](const int4* R, uint32_t j, uint32_t end, int4 (&p)[4]) {
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) p[k] = R[min(j + k, end - 1)];
  };
  auto test = [&](const int4 (&p)[4], uint32_t j, uint32_t end, uint32_t skip) {
    const float2 k01 = candidate_keys<D, false>(pi, p[0], p[1], I, R2f, band);
    const float2 k23 = candidate_keys<D, false>(pi, p[2], p[3], I, R2f, band);
    const float key[4] = {k01.x, k01.y, k23.x, k23.y};
    unsigned h = 0;
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) h |= (unsigned)(key[k] < 0.0f && j + k < end && j + k != skip) << k;
    return h;
  };
  int4 pf[4], pw[4];
  if (s[0] < e[0]) four(P, s[0], e[0], pf);
  if (s[1] < e[1]) four(b.WP, s[1], e[1], pw);
  unsigned bits[2] = {0u, 0u};
  int mine[2] = {0, 0};
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const uint32_t skip = t == 0 ? me : 0xffffffffu;
    for (uint32_t j = s[t]; j < e[t]; j += 4) {
      if (j != s[t]) four(t == 0 ? P : (const int4*)b.WP, j, e[t], t == 0 ? pf : pw);
      const unsigned h = test(t == 0 ? pf : pw, j, e[t], skip);
      if (j - s[t] < 32) bits[t] |= h << (j - s[t]);
      mine[t] += __popc(h);
    }
  }
  bool overflow = false;
  int total[2], at[2];
#pragma unroll
  for (int t = 0; t < 2; ++t) at[t] = lanes_prefix<LS>(mine[t], r, &total[t]) - mine[t];
  const int nf = min(total[0], b.cap), nw = min(total[1], max(b.cap - wall_slot0(nf), 0));
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    RowWriter w(b.nbr, b.n, i, (t == 0 ? 0 : wall_slot0(nf)) + at[t], b.cap);
    if (e[t] - s[t] <= 32) {
      for (unsigned h = bits[t]; h; h &= h - 1) w.push((int)(s[t] + __ffs((int)h) - 1), overflow);
    } else {
      for (uint32_t j = s[t]; j < e[t]; j += 4) {
        four(t == 0 ? P : (const int4*)b.WP, j, e[t], pf);
        for (unsigned h = test(pf, j, e[t], t == 0 ? me : 0xffffffffu); h; h &= h - 1)
          w.push((int)(j + __ffs((int)h) - 1), overflow);
      }
    }
  }
  if (overflow) raise_error(b.glob, ERR_CAPACITY, i);
  return (uint32_t)nf | ((uint32_t)nw << 16);
}

// The same on a grid with a periodic axis, one list after the other: the row is the one a single thread writes going through the rows in
// order. A lane keeps its hits as bits over its candidates (in up to two runs, the second
// where a periodic x axis splits the row), and the counts' prefix over the group is its place
// in the row; a row of more than 64 candidates is tested again for the write. Returns
// nf | nw << 16 in every lane.
template <int D, bool PER, int LS>
__device__ __forceinline__ uint32_t search_group_periodic(const Buffers& b, const Inst& I, int64_t i, int r, const int4& pi,
                                                 const int4* P) {
  constexpr int kRows = D == 3 ? 25 : 5;
  static_assert(LS >= kRows, "a lane per search row");
  const float R2f = (float)I.R2, band = R2f * 1.9073486328125e-06f;
  const unsigned gm = search_mask<LS>();
  bool overflow = false;
  // all hits of one cell-linked list into the row from slot0 on; returns their number
  auto list = [&](const int4* R, const uint32_t* start, bool self, int slot0) {
    const uint32_t me = self ? (uint32_t)i : 0xffffffffu;
    unsigned long long bits = 0;
    uint32_t b0 = 0, len0 = 0, b1 = 0;
    int cand = 0, runs = 0, mine = 0;
    auto scan = [&](uint32_t s, uint32_t e, auto&& take) {
      for (uint32_t j = s; j < e; j += 4) {
        const uint32_t j1 = min(j + 1, e - 1), j2 = min(j + 2, e - 1), j3 = min(j + 3, e - 1);
        const int4 p0 = R[j], p1 = R[j1], p2 = R[j2], p3 = R[j3];
        const float2 k01 = candidate_keys<D, PER>(pi, p0, p1, I, R2f, band);
        const float2 k23 = candidate_keys<D, PER>(pi, p2, p3, I, R2f, band);
        const bool in0 = k01.x < 0.0f, in1 = k01.y < 0.0f, in2 = k23.x < 0.0f, in3 = k23.y < 0.0f;
        take(j, (unsigned)(in0 && j != me) | (unsigned)(in1 && j + 1 < e && j1 != me) << 1 |
                    (unsigned)(in2 && j + 2 < e && j2 != me) << 2 | (unsigned)(in3 && j + 3 < e && j3 != me) << 3);
      }
    };
    if (r < kRows)
      for_neighbour_rows<D, PER>(I, pi, start, r, r + 1, [&](uint32_t s, uint32_t e) {
        if (runs == 0) {
          b0 = s;
          len0 = e - s;
        } else {
          b1 = s;
        }
        ++runs;
        scan(s, e, [&](uint32_t j, unsigned h) {
          const int at = cand + (int)(j - s);
          if (at < 64) bits |= (unsigned long long)h << at;
          mine += __popc(h);
        });
        cand += (int)(e - s);
      });
    int incl = mine;
#pragma unroll
    for (int o = 1; o < LS; o <<= 1) {
      const int y = __shfl_up_sync(gm, incl, o, LS);
      if (r >= o) incl += y;
    }
    const int total = __shfl_sync(gm, incl, LS - 1, LS);
    RowWriter w(b.nbr, b.n, i, slot0 + incl - mine, b.cap);
    if (cand <= 64 && runs <= 2) {
      for (; bits; bits &= bits - 1) {
        const uint32_t at = (uint32_t)__ffsll((long long)bits) - 1u;
        w.push((int)(at < len0 ? b0 + at : b1 + (at - len0)), overflow);
      }
    } else {
      for_neighbour_rows<D, PER>(I, pi, start, r, r + 1, [&](uint32_t s, uint32_t e) {
        scan(s, e, [&](uint32_t j, unsigned h) {
          for (; h; h &= h - 1) w.push((int)(j + __ffs((int)h) - 1), overflow);
        });
      });
    }
    return total;
  };
  const int nf = min(list(P, b.fstart, true, 0), b.cap);
  int nw = 0;
  if (b.nw && b.wnear[search_cell<D>(I, pi)])            // a wall within reach
    nw = min(list(b.WP, b.wstart, false, wall_slot0(nf)), max(b.cap - wall_slot0(nf), 0));
  if (overflow) raise_error(b.glob, ERR_CAPACITY, i);
  return (uint32_t)nf | ((uint32_t)nw << 16);
}

template <int D, bool PER, int LPP, bool TV>
__global__ void __launch_bounds__(kStepThreads<LPP> + 32, 1)
k_fused_step(const __grid_constant__ Buffers b, int n_steps, int clear_counts, int follow) {
  __shared__ float4 terms_all[LPP > 1 ? kStepThreads<LPP> / 32 : 1][(1 + D + (TV ? 1 : 0)) * 32];
  __shared__ uint32_t warp_tot[kStepMaxWarps];
  __shared__ unsigned vmax_block;
  __shared__ Ctrl C;                             // the tank's control, kept alike by every block
  __shared__ int more;                           // substeps needed after the next one
  __shared__ int failed;                         // the status before a step
  constexpr int LS = D == 3 ? 32 : 8;            // lanes of a particle in the search
  const Inst& I = b.inst0;
  StepCtl* c = b.step_ctl;
  Global* g = b.glob;
  const int work = blockDim.x - 32, share = work / LPP;   // work threads; particles of a block at a time
  const bool worker = (int)threadIdx.x < work, control = (int)threadIdx.x == work;
  float4* terms = terms_all[LPP > 1 && worker ? threadIdx.x >> 5 : 0];
  const int64_t n = b.n, tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, threads = (int64_t)gridDim.x * blockDim.x;
  const int sub = lane_sub<LPP>();
  const int64_t step = (int64_t)gridDim.x * share, block0 = (int64_t)blockIdx.x * share,
                first = worker ? block0 + lane_particle<LPP>() : n;
  // this block's share of the cells
  const int64_t per = ((b.n_cells + gridDim.x - 1) / gridDim.x + 3) & ~(int64_t)3;
  const int64_t c0 = min((int64_t)blockIdx.x * per, b.n_cells), c1 = min(c0 + per, b.n_cells);
  const int4* nb4 = reinterpret_cast<const int4*>(b.nbr);
  int* id_new = reinterpret_cast<int*>(b.rank);  // free after the scatter
  unsigned target = 0;

  if (threadIdx.x == 0) C = b.ctrl[0];
  if (clear_counts) {
    for (int64_t k = tid; k < b.n_cells; k += threads) b.count[k] = 0u;
    if (!grid_barrier(&c->count, target, g)) return;
  }
  for (int st = 0; st < n_steps; ++st) {
    // ---- cells: hash, scan, sort by (cell, id)
    if (threadIdx.x == 0) failed = st > 0 || follow ? *(volatile int*)&g->err : 0;
    for (int64_t i = tid; i < n; i += threads) {
      const uint32_t cell = hash_cell<D>(I, b.PS[i], i, &c->found);
      b.cell[i] = cell;
      b.rank[i] = atomicAdd(&b.count[cell], 1u);
    }
    if (!grid_barrier(&c->count, target, g)) return;
    if (failed) {                                // an earlier step failed: every block leaves, its
      if (st == 0) return;                       // counters to the host (this barrier may not have held
      break;                                     // the blocks together, after a launch that gave up)
    }
    uint32_t sum = 0, total;
    for (int64_t k = c0 + 4 * threadIdx.x; k < c1; k += 4 * blockDim.x) {
      const uint4 v = load4(b.count, k, c1);
      sum += v.x + v.y + v.z + v.w;
    }
    block_scan(sum, warp_tot, &total);
    if (threadIdx.x == 0) c->sums[blockIdx.x] = total;
    if (!grid_barrier(&c->count, target, g)) return;
    uint32_t before = 0, run;
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += blockDim.x) before += c->sums[k];
    block_scan(before, warp_tot, &run);          // the particles of the cells before this block's
    for (int64_t k0 = c0; k0 < c1; k0 += 4 * blockDim.x) {
      const int64_t k = k0 + 4 * threadIdx.x;
      const uint4 v = load4(b.count, k, c1);
      uint4 at;
      at.x = run + block_scan(v.x + v.y + v.z + v.w, warp_tot, &total);
      at.y = at.x + v.x;
      at.z = at.y + v.y;
      at.w = at.z + v.z;
      store4(b.fstart, k, c1, at);
      store4(b.count, k, c1, make_uint4(0u, 0u, 0u, 0u));   // zero again for the next step
      run += total;
    }
    if (tid == 0) b.fstart[b.n_cells] = (uint32_t)n;
    if (!grid_barrier(&c->count, target, g)) return;
    for (int64_t i = tid; i < n; i += threads) {
      const uint32_t d = b.fstart[b.cell[i]] + b.rank[i];
      b.key[d] = b.id[i];
      b.src[d] = (int)i;
    }
    if (!grid_barrier(&c->count, target, g)) return;
    for (int64_t d = tid; d < n; d += threads) { // place in the cell: the mates with smaller ids
      const int s = b.src[d], key = b.key[d];
      const int4 p = b.PS[s];
      const float4 v = b.VS[s];
      const uint32_t cell = b.cell[s], e = b.fstart[cell + 1];
      uint32_t t = b.fstart[cell];
      for (uint32_t m = t; m < e; ++m) t += b.key[m] < key ? 1u : 0u;
      b.PH[t] = p;
      b.VH[t] = v;
      id_new[t] = key;
      if (b.mass) b.mass_tmp[t] = b.mass[s];
    }
    if (!grid_barrier(&c->count, target, g)) return;
    // ---- neighbours and density, a block's share of the particles at a time; Dt_ad and the
    // first dt beside them
    if (control) {
      const int found = blockIdx.x == 0 ? *(volatile int*)&c->found.err : 0;
      dt_advection_one(I, C);
      more = dt_acoustic_one(I, C, g, 0.0);
      if (found) {                               // the hash's errors to the status
        raise_error(g, found, *(volatile long long*)&c->found.bad_index);
        c->found.err = 0;
      }
    }
    for (int64_t i0 = block0; i0 < n; i0 += step) {
      const int count = (int)min((int64_t)share, n - i0);
      if (worker) {
        for (int p = threadIdx.x / LS; p < count; p += work / LS) {
          const int4 pi = b.PH[i0 + p];
          const int r = threadIdx.x % LS;
          const uint32_t cnt = PER ? search_group_periodic<D, PER, LS>(b, I, i0 + p, r, pi, b.PH)
                                   : search_group<D, LS>(b, I, i0 + p, r, pi, b.PH);
          if (r == 0) b.nbc[i0 + p] = cnt;
        }
      }
      __syncthreads();                           // the share's rows are written
      const int64_t i = i0 + lane_particle<LPP>();
      if (worker && i < n) {
        const int4 pi = b.PH[i];
        const float dev = density_dev<D, PER, LPP>(I, i, sub, pi, b.nbc[i], n, (const int4*)b.PH, nb4, b.WP, terms);
        if (sub == 0) {
          b.PS[i] = make_int4(pi.x, pi.y, pi.z, f2i(dev));
          b.VS[i] = b.VH[i];
          b.id[i] = id_new[i];
          if (b.mass) b.mass[i] = b.mass_tmp[i];
        }
      }
    }
    if (tid == 0) c->vm[0] = 0u;
    if (!grid_barrier(&c->count, target, g)) return;
    if (b.acc_prior) {   // read back by the lane that wrote it: no barrier
      for (int64_t i = first; i < n; i += step) {
        const float4 a = viscous_acc<D, PER, LPP>(I, i, sub, (int)(b.nbc[i] & 0xffffu), n, (const int4*)b.PS,
                                             (const float4*)b.VS, (const float*)b.mass, nb4, terms);
        if (sub == 0) b.acc_prior[i] = a;
      }
    }
    // ---- acoustic substeps
    RowHead head;
    head.load<LPP>(first < n ? first : -1, sub, n, nb4, b.nbc);
    int ran = 0;
    for (int it = 0;; it ^= 1) {
      const double dtd = C.dt;
      const int any = more;
      float v2max = 0.0f;
      if (threadIdx.x == 0) vmax_block = 0u;
      if (dtd != 0.0) {
        for (int64_t i = first; i < n; i += step) {
          bool writer;
          if (i != first || step < n) head.load<LPP>(i, sub, n, nb4, b.nbc);
          const float v2 = pr_group<D, PER, LPP, TV>(I, i, sub, true, dtd, n, (const int4*)b.PS, (const float4*)b.VS,
                                                     b.PH, b.VH, (const float*)b.mass, nb4, head, b.WP, b.WN,
                                                     (const float4*)b.acc_prior, b.acc_keep, g, terms, &writer);
          v2max = fmaxf(v2max, v2);
        }
      }
      ++ran;
      __syncthreads();                           // vmax_block is zero, C and more are read
      const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(v2max));
      if ((threadIdx.x & 31) == 0 && m) atomicMax(&vmax_block, m);
      __syncthreads();
      if (threadIdx.x == 0 && vmax_block) atomicMax(&c->vm[it], vmax_block);
      if (!grid_barrier(&c->count, target, g)) return;
      if (dtd != 0.0) {
        for (int64_t i = first; i < n; i += step) {
          if (i != first || step < n) head.load<LPP>(i, sub, n, nb4, b.nbc);
          dr_group<D, PER, LPP>(I, i, sub, dtd, n, (const int4*)b.PH, (const float4*)b.VH, b.PS, b.VS,
                                (const float*)b.mass, nb4, head, b.WP, b.WN, g, terms);
        }
      }
      if (tid == 0) c->vm[it ^ 1] = 0u;          // its last reader has passed the barrier
      if (control) {                             // the next dt
        C.vmax2 = __ldcg(&c->vm[it]);
        if (any) more = dt_acoustic_one(I, C, g, 0.0);
      }
      if (!grid_barrier(&c->count, target, g)) return;
      if (!any) break;
    }
    if (tid == 0) g->substeps += ran;
  }
  if (tid == 0) {
    b.ctrl[0] = C;
    g->active = 0;
  }
  if (threadIdx.x == 0 && atomicAdd(&c->exits, 1u) == gridDim.x - 1) {   // every block has left the barriers
    c->exits = 0u;
    c->count = 0u;
  }
}

template <int D, bool PER, int LPP, bool TV>
cudaError_t launch_t(const Buffers& b, int n_steps, int clear_counts, int follow, cudaStream_t s) {
  // the particles' lanes over all SMs, in blocks of 128 work threads or more; a few more
  // blocks where the cells would be many for them (a scan of 8192 a block)
  const int64_t lanes = b.n * LPP;
  const int work = (int)std::min<int64_t>(kStepThreads<LPP>, std::max<int64_t>(128, ((lanes + b.n_sm - 1) / b.n_sm + 31) / 32 * 32));
  const int64_t want = std::max((lanes + work - 1) / work, (b.n_cells + 8191) / 8192);
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>({want, (int64_t)b.n_sm, (int64_t)kStepMaxGrid}));
  void* args[] = {const_cast<Buffers*>(&b), &n_steps, &clear_counts, &follow};
  return cudaLaunchCooperativeKernel((const void*)k_fused_step<D, PER, LPP, TV>, dim3(grid), dim3(work + 32), args, 0, s);
}

// Lanes a particle: the most that keep a block within its work threads; two only while they
// leave half of them free. A further step of the 2D dam break took, with 8 / 4 / 2 / 1 lanes,
// 52 / 71 / 93 / 93 us at 512 particles, 85 / 79 / 102 / 110 at 9,800, 113 / 125 / 104 / 113 at
// 20,000 and 188 / 166 / 135 / 126 at 51,200; of the 3D one 106 / 150 / 278 / 348 us at 2,662
// and 183 / 153 / 253 / 319 at 16,000.
template <int D, bool PER>
cudaError_t launch_d(const Buffers& b, int n_steps, int clear, int follow, cudaStream_t s) {
  const int64_t per = (b.n + b.n_sm - 1) / b.n_sm;         // particles of an SM
  if (b.any_transport) {
    if (per * 4 <= kStepThreads<4>) return launch_t<D, PER, 4, true>(b, n_steps, clear, follow, s);
    return launch_t<D, PER, 1, true>(b, n_steps, clear, follow, s);
  }
  if (per * 8 <= kStepThreads<8>) return launch_t<D, PER, 8, false>(b, n_steps, clear, follow, s);
  if (per * 4 <= kStepThreads<4>) return launch_t<D, PER, 4, false>(b, n_steps, clear, follow, s);
  if (per * 2 <= kStepThreads<2> / 2) return launch_t<D, PER, 2, false>(b, n_steps, clear, follow, s);
  return launch_t<D, PER, 1, false>(b, n_steps, clear, follow, s);
}

}  // namespace
}  // namespace sph
