// Configuration update of the WCSPH hot path (cell-linked list, paper Sec. 6.2
// mesh_cell_linked_list, refreshed once per advection step as Sec. 2.4 fixes):
//   hash      particle -> search cell (integer: q >> (bits - 1) per axis, i.e. cells of
//             half the 2h position cell, about h; flattened x fastest)
//   sort      counting sort on the cell digit (a one-digit radix sort with radix =
//             number of cells), then each particle's rank among its cell mates by
//             caller id, which makes the order the unique (cell, id) order,
//             independent of history
//   offsets   exclusive scan of the cell counts
//   reorder   the 32-byte particle records moved to their (cell, id) slots
//   neighbours frozen set {j != i : |r_i - r_j| < 2h}, quad-interleaved ELL rows; the
//             search visits the 5^D cells around a particle clipped to its 2h sphere
//             (rows whose slab lies at >= 2h are skipped, row runs cut to the
//             sphere's chord), about 42 % of the candidates of a 3^D scan of 2h cells
#include <cstdio>

#include "sph_cells.cuh"

namespace sph {

namespace {

constexpr int kBlock = 256;
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

inline unsigned grid_for(int64_t n, int block = kBlock) {
  return (unsigned)((n + block - 1) / block);
}

// ---------------------------------------------------------------- scan ---------------
// Block-level exclusive scan of kScanTile elements; block totals to `sums`.
__global__ void k_scan_tile(const uint32_t* in, uint32_t* out,   // may alias (in-place)
                            int64_t n, uint32_t* __restrict__ sums) {
  __shared__ uint32_t warp_tot[kScanThreads / 32];
  int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  uint32_t local = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    int64_t idx = base + k;
    v[k] = idx < n ? in[idx] : 0u;
    local += v[k];
  }
  // inclusive scan of per-thread totals inside the warp
  unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (unsigned)o) incl += y;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < kScanThreads / 32 ? warp_tot[lane] : 0u;
    uint32_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= (unsigned)o) wi += y;
    }
    if (lane < kScanThreads / 32) warp_tot[lane] = wi - w;   // exclusive warp offsets
    if (lane == 31 && sums) sums[blockIdx.x] = wi;           // block total
  }
  __syncthreads();
  uint32_t run = warp_tot[warp] + incl - local;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    int64_t idx = base + k;
    if (idx < n) out[idx] = run;
    run += v[k];
  }
}

__global__ void k_scan_add(uint32_t* __restrict__ out, int64_t n, const uint32_t* __restrict__ offs) {
  int64_t idx = (int64_t)blockIdx.x * kScanTile + threadIdx.x;
  uint32_t add = offs[blockIdx.x];
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    int64_t j = idx + (int64_t)k * kScanThreads;
    if (j < n) out[j] += add;
  }
}

__global__ void k_scan_total(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int64_t n) {
  out[n] = n ? out[n - 1] + in[n - 1] : 0u;
}

}  // namespace

size_t scan_tmp_elems(int64_t n) {
  size_t total = 0;
  int64_t m = n;
  while (m > kScanTile) {
    m = (m + kScanTile - 1) / kScanTile;
    total += (size_t)m;
  }
  return total + 1;
}

static void scan_rec(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* tmp, cudaStream_t s,
                     int64_t* launches) {
  int64_t blocks = (n + kScanTile - 1) / kScanTile;
  if (blocks <= 1) {
    k_scan_tile<<<1, kScanThreads, 0, s>>>(in, out, n, nullptr);
    ++*launches;
    return;
  }
  uint32_t* sums = tmp;
  k_scan_tile<<<(unsigned)blocks, kScanThreads, 0, s>>>(in, out, n, sums);
  scan_rec(sums, sums, blocks, tmp + blocks, s, launches);
  k_scan_add<<<(unsigned)blocks, kScanThreads, 0, s>>>(out, n, sums);
  *launches += 2;
}

// Exclusive scan of in[0..n) into out[0..n], out[n] = total.
void scan_exclusive(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* tmp, cudaStream_t s,
                    int64_t* launches) {
  if (n > 0) scan_rec(in, out, n, tmp, s, launches);
  k_scan_total<<<1, 1, 0, s>>>(in, out, n);
  ++*launches;
}

namespace {

// ---------------------------------------------------------------- hash ---------------
template <int D>
__global__ void k_hash(int64_t n, const int4* __restrict__ P, const int* __restrict__ inst_of,
                       const Inst* __restrict__ inst, uint32_t* __restrict__ cell,
                       uint32_t* __restrict__ count, uint32_t* __restrict__ rank, Global* g) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Inst& I = inst[inst_of ? inst_of[i] : 0];
  const uint32_t c = hash_cell<D>(I, P[i], i, g);
  cell[i] = c;
  rank[i] = atomicAdd(&count[c], 1u);
}

__global__ void k_scatter(int64_t n, const uint32_t* __restrict__ cell, const uint32_t* __restrict__ rank,
                          const uint32_t* __restrict__ start, const int* __restrict__ id,
                          int* __restrict__ key, int* __restrict__ src) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t d = start[cell[i]] + rank[i];
  key[d] = id[i];
  src[d] = (int)i;
}

// Final slot of every particle: the counting sort left each cell's particles in arbitrary
// order; a particle's place within its cell is the number of cell mates with a smaller id,
// which makes the order the unique (cell, id) order. One thread per particle (cells hold
// a few particles), instead of one per cell.
__global__ void k_cell_rank(int64_t n, const uint32_t* __restrict__ cell, const uint32_t* __restrict__ start,
                            const int* __restrict__ key, const int* __restrict__ src, uint32_t* __restrict__ dst) {
  int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (d >= n) return;
  const uint32_t c = cell[src[d]];
  const uint32_t b = start[c], e = start[c + 1];
  const int k = key[d];
  uint32_t r = 0;
  for (uint32_t m = b; m < e; ++m) r += key[m] < k ? 1u : 0u;
  dst[d] = b + r;
}

// Records moved to their final slots (writes stay within each cell's slot range); the
// ids in the new order go to id_out.
__global__ void k_reorder(int64_t n, const int* __restrict__ src, const uint32_t* __restrict__ dst,
                          const int* __restrict__ key, const int4* __restrict__ Pin,
                          const float4* __restrict__ Vin, int4* __restrict__ Pout,
                          float4* __restrict__ Vout, const float* __restrict__ min,
                          float* __restrict__ mout, int* __restrict__ id_out) {
  int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (d >= n) return;
  const int s = src[d];
  const uint32_t t = dst[d];
  Pout[t] = Pin[s];
  Vout[t] = Vin[s];
  id_out[t] = key[d];
  if (min) mout[t] = min[s];
}

__global__ void k_copy_back(int64_t n, const int4* __restrict__ Pin, const float4* __restrict__ Vin,
                            const int* __restrict__ key, int4* __restrict__ Pout,
                            float4* __restrict__ Vout, int* __restrict__ id,
                            const float* __restrict__ min, float* __restrict__ mout) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  Pout[i] = Pin[i];
  Vout[i] = Vin[i];
  id[i] = key[i];
  if (min) mout[i] = min[i];
}

// ---------------------------------------------------------------- neighbours ---------
// All neighbours of particle i among the records R of one cell-linked list (`self`: R holds
// the particle itself) into its row from slot0 on; returns their number. The candidates of a
// run are tested first, their hits kept as bits, and written then: the stores of 32 lanes
// diverge, and inside the test loop every test paid for them. With it, the sign bits of the
// keys as hits, the tank's constants in the argument (48 registers in 3D, five blocks an SM for
// four) and 32-bit chords, the search of 1.02M particles of the 3D dam break takes 442 us (580).
template <int D, bool PER>
__device__ __forceinline__ int list_neighbours(const Inst& I, int64_t n, int64_t i, const int4& pi, const int4* R,
                                               const uint32_t* start, bool self, int slot0, int cap, int* nbr,
                                               bool& overflow) {
  const float R2f = (float)I.R2, band = R2f * 1.9073486328125e-06f;
  RowWriter w(nbr, n, i, slot0, cap);
  for_neighbour_runs<D, PER>(I, pi, start, [&](uint32_t b, uint32_t e) {
    for (; b < e; b += 32) {
      const uint32_t m = min(e - b, 32u);
      const int4* r = R + b;
      unsigned bits = 0;                             // candidate k at bit m' - 1 - k, m' = m made even
      for (uint32_t k = 0; k < m; k += 2, r += 2) {   // one past an odd run: masked out (the arrays are padded)
        const float2 key = candidate_keys<D, PER>(pi, r[0], r[1], I, R2f, band);
        bits = push_sign(push_sign(bits, key.x), key.y);
      }
      bits = __brev(bits) >> ((32u - m) & ~1u);       // candidate k at bit k
      if (m < 32u) bits &= (1u << m) - 1u;
      if (self && (uint32_t)i - b < 32u) bits &= ~(1u << ((uint32_t)i - b));
      for (; bits; bits &= bits - 1) w.push((int)(b + __ffs((int)bits) - 1), overflow);
    }
  });
  return w.count;
}

// UNI: a single tank, its constants in the kernel argument.
template <int D, bool PER, bool UNI>
__global__ void __launch_bounds__(kBlock)
k_neighbours(const Inst Ip, int64_t n, const int4* __restrict__ P, const int* __restrict__ inst_of,
             const Inst* __restrict__ inst, const uint32_t* __restrict__ fstart,
             const int4* __restrict__ WP, const uint32_t* __restrict__ wstart,
             const uint8_t* __restrict__ wnear, int cap, int* __restrict__ nbr,
             uint32_t* __restrict__ nbc, Global* g) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Inst& I = UNI ? Ip : inst[inst_of ? inst_of[i] : 0];
  const int4 pi = P[i];
  bool overflow = false;
  const int nf = min(list_neighbours<D, PER>(I, n, i, pi, P, fstart, true, 0, cap, nbr, overflow), cap);
  int nw = 0;
  if (WP && wnear[search_cell<D>(I, pi)]) {           // no wall within reach: skip the pass
    const int w0 = wall_slot0(nf);
    nw = min(list_neighbours<D, PER>(I, n, i, pi, WP, wstart, false, w0, cap, nbr, overflow), max(cap - w0, 0));
  }
  if (overflow) raise_error(g, ERR_CAPACITY, i);
  nbc[i] = (uint32_t)nf | ((uint32_t)nw << 16);
}

// ---------------------------------------------------------------- debug bounds checks --
// SPH_FLAG_DEBUG_BOUNDS: the offsets of a cell-linked list must start at 0, never decrease
// and end at the particle count; a neighbour row must fit the capacity with every fluid
// index below n and every wall index below nw. Each check reads only inside the arrays'
// own extents, whatever values they hold, and records the first violation.
__global__ void k_check_offsets(int64_t n_cells, const uint32_t* __restrict__ start, uint32_t total,
                                Global* g) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c > n_cells) return;
  bool bad = start[c] > total;
  if (c == 0) bad = bad || start[0] != 0u;
  if (c == n_cells) bad = bad || start[c] != total;
  else bad = bad || start[c] > start[c + 1];
  if (bad) raise_error(g, ERR_BOUNDS, c);
}

__global__ void k_check_table(int64_t n, int64_t nw, int cap, const int* __restrict__ nbr,
                              const uint32_t* __restrict__ nbc, Global* g) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t cnt = nbc[i];
  const int nf = (int)(cnt & 0xffffu), nwi = (int)(cnt >> 16);
  if (nf > cap || wall_slot0(nf) + nwi > cap) {
    raise_error(g, ERR_BOUNDS, i);
    return;
  }
  for (int s = 0; s < nf; ++s) {
    const int j = nbr[slot_index(n, i, s)];
    if (j < 0 || (int64_t)j >= n) {
      raise_error(g, ERR_BOUNDS, i);
      return;
    }
  }
  const int w0 = wall_slot0(nf);
  for (int s = 0; s < nwi; ++s) {
    const int w = nbr[slot_index(n, i, w0 + s)];
    if (w < 0 || (int64_t)w >= nw) {
      raise_error(g, ERR_BOUNDS, i);
      return;
    }
  }
}

// ---------------------------------------------------------------- walls ---------------
__global__ void k_wall_reorder(int64_t n, const int* __restrict__ src, const uint32_t* __restrict__ dst,
                               const int* __restrict__ key, const int4* __restrict__ Pin,
                               const float4* __restrict__ Nin, int4* __restrict__ Pout,
                               float4* __restrict__ Nout, int* __restrict__ id_out) {
  int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (d >= n) return;
  const int s = src[d];
  const uint32_t t = dst[d];
  Pout[t] = Pin[s];
  Nout[t] = Nin[s];
  id_out[t] = key[d];
}

__global__ void k_iota(int64_t n, int* __restrict__ a) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] = (int)i;
}

// Near-wall flags of the search cells: a cell is flagged when a wall particle lies within
// two search cells on every axis, i.e. in the 5^d block the neighbour search visits. The
// occupancy of the wall grid is dilated by +-2 cells one axis at a time.
__device__ __forceinline__ int cell_instance(const Inst* __restrict__ inst, int n_inst, long long c) {
  int lo = 0, hi = n_inst - 1;                 // last instance whose first cell is <= c
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (inst[mid].cell_base <= c) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__global__ void k_wall_occupied(int64_t n_cells, const uint32_t* __restrict__ wstart, uint8_t* __restrict__ out) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < n_cells) out[c] = wstart[c + 1] > wstart[c] ? 1 : 0;
}

__global__ void k_dilate_axis(int64_t n_cells, int axis, const Inst* __restrict__ inst, int n_inst,
                              const uint8_t* __restrict__ in, uint8_t* __restrict__ out) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n_cells) return;
  const Inst& I = inst[cell_instance(inst, n_inst, c)];
  long long stride = 1;
  for (int a = 0; a < axis; ++a) stride *= I.scell[a];
  const int len = I.scell[axis];
  const int pos = (int)(((c - I.cell_base) / stride) % len);
  uint8_t v = 0;
  for (int d = -2; d <= 2; ++d) {
    int p = pos + d;
    if (I.period[axis]) p = p < 0 ? p + len : (p >= len ? p - len : p);
    else if (p < 0 || p >= len) continue;
    v |= in[c + (long long)(p - pos) * stride];
  }
  out[c] = v;
}

// Row pieces of the row-task form (one tank): row r = cy + scell[1] cz holds the search
// cells (0..scell[0]-1, cy, cz), whose particles are contiguous in the cell order.
__global__ void k_row_count(const Inst I, int64_t n_rows, const uint32_t* __restrict__ fstart,
                            uint32_t* __restrict__ cnt) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_rows) return;
  const long long c0 = I.cell_base + (long long)r * I.scell[0];
  const uint32_t len = fstart[c0 + I.scell[0]] - fstart[c0];
  cnt[r] = (len + 31u) >> 5;
}

__global__ void k_row_fill(const Inst I, int64_t n_rows, const uint32_t* __restrict__ fstart,
                           const uint32_t* __restrict__ cnt, const uint32_t* __restrict__ off,
                           int2* __restrict__ task, int64_t cap) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_rows) return;
  const long long c0 = I.cell_base + (long long)r * I.scell[0];
  const int first = (int)fstart[c0];
  const int len = (int)(fstart[c0 + I.scell[0]] - fstart[c0]);
  const int k_end = (int)cnt[r];
  for (int k = 0; k < k_end; ++k) {
    const int64_t t = (int64_t)off[r] + k;
    if (t >= cap) return;            // not reached: cap >= n/32 + rows bounds the pieces
    task[t] = make_int2(first + 32 * k, min(32, len - 32 * k));
  }
}

}  // namespace

void launch_hash(const Buffers& b, cudaStream_t s, int64_t* launches) {
  cudaMemsetAsync(b.count, 0, sizeof(uint32_t) * b.n_cells, s);
  if (b.counts_zero) *b.counts_zero = false;
  if (b.n == 0) return;
  if (b.dim == 2)
    k_hash<2><<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.PS, b.inst_of, b.inst, b.cell, b.count, b.rank, b.glob);
  else
    k_hash<3><<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.PS, b.inst_of, b.inst, b.cell, b.count, b.rank, b.glob);
  ++*launches;
}

void launch_fluid_offsets(const Buffers& b, cudaStream_t s, int64_t* launches) {
  scan_exclusive(b.count, b.fstart, b.n_cells, b.scan_tmp, s, launches);
}

void launch_sort_fluid(const Buffers& b, cudaStream_t s, int64_t* launches) {
  if (b.rows_valid) *b.rows_valid = false;     // the row pieces follow the new order
  if (b.n == 0) return;
  k_scatter<<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.cell, b.rank, b.fstart, b.id, b.key, b.src);
  // final slots into rank (free after the scatter); sorted ids into cell (free after the rank)
  k_cell_rank<<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.cell, b.fstart, b.key, b.src, b.rank);
  int* ids_sorted = reinterpret_cast<int*>(b.cell);
  k_reorder<<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.src, b.rank, b.key, b.PS, b.VS, b.PH, b.VH, b.mass,
                                             b.mass_tmp, ids_sorted);
  k_copy_back<<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.PH, b.VH, ids_sorted, b.PS, b.VS, b.id, b.mass_tmp,
                                               b.mass);
  *launches += 4;
}

void launch_neighbours(const Buffers& b, cudaStream_t s, int64_t* launches) {
  if (b.n == 0) return;
  const int4* wp = b.nw ? b.WP : nullptr;
  auto kern = b.n_inst == 1
      ? (b.dim == 2 ? (b.any_periodic ? k_neighbours<2, true, true> : k_neighbours<2, false, true>)
                    : (b.any_periodic ? k_neighbours<3, true, true> : k_neighbours<3, false, true>))
      : (b.dim == 2 ? (b.any_periodic ? k_neighbours<2, true, false> : k_neighbours<2, false, false>)
                    : (b.any_periodic ? k_neighbours<3, true, false> : k_neighbours<3, false, false>));
  kern<<<grid_for(b.n), kBlock, 0, s>>>(b.inst0, b.n, b.PS, b.inst_of, b.inst, b.fstart, wp, b.wstart, b.wnear,
                                        b.cap, b.nbr, b.nbc, b.glob);
  ++*launches;
}

void launch_row_tasks(const Buffers& b, cudaStream_t s, int64_t* launches) {
  if (!b.row_task || b.n_rows == 0) return;
  const unsigned g = grid_for(b.n_rows);
  k_row_count<<<g, kBlock, 0, s>>>(b.inst0, b.n_rows, b.fstart, b.row_cnt);
  scan_exclusive(b.row_cnt, b.row_off, b.n_rows, b.row_tmp, s, launches);
  k_row_fill<<<g, kBlock, 0, s>>>(b.inst0, b.n_rows, b.fstart, b.row_cnt, b.row_off, b.row_task,
                                  b.row_task_cap);
  *launches += 2;
}

// Walls are static: sort them into cells once. Uses the fluid build scratch
// (cell/rank/count/key/src sized for max(n, nw)); wid_tmp may be b.wid.
void sort_walls(Buffers& b, int4* WP_tmp, float4* WN_tmp, int* wid_tmp, cudaStream_t s) {
  int64_t dummy = 0;
  cudaMemsetAsync(b.count, 0, sizeof(uint32_t) * b.n_cells, s);
  if (b.nw > 0) {
    if (b.dim == 2)
      k_hash<2><<<grid_for(b.nw), kBlock, 0, s>>>(b.nw, b.WP, b.winst_of, b.inst, b.cell, b.count,
                                                  b.rank, b.glob);
    else
      k_hash<3><<<grid_for(b.nw), kBlock, 0, s>>>(b.nw, b.WP, b.winst_of, b.inst, b.cell, b.count,
                                                  b.rank, b.glob);
  }
  scan_exclusive(b.count, b.wstart, b.n_cells, b.scan_tmp, s, &dummy);
  if (b.nw == 0) return;
  k_iota<<<grid_for(b.nw), kBlock, 0, s>>>(b.nw, wid_tmp);
  k_scatter<<<grid_for(b.nw), kBlock, 0, s>>>(b.nw, b.cell, b.rank, b.wstart, wid_tmp, b.key, b.src);
  k_cell_rank<<<grid_for(b.nw), kBlock, 0, s>>>(b.nw, b.cell, b.wstart, b.key, b.src, b.rank);
  int* wids_sorted = reinterpret_cast<int*>(b.cell);
  k_wall_reorder<<<grid_for(b.nw), kBlock, 0, s>>>(b.nw, b.src, b.rank, b.key, b.WP, b.WN, WP_tmp, WN_tmp,
                                                   wids_sorted);
  cudaMemcpyAsync(b.WP, WP_tmp, sizeof(int4) * b.nw, cudaMemcpyDeviceToDevice, s);
  cudaMemcpyAsync(b.WN, WN_tmp, sizeof(float4) * b.nw, cudaMemcpyDeviceToDevice, s);
  cudaMemcpyAsync(b.wid, wids_sorted, sizeof(int) * b.nw, cudaMemcpyDeviceToDevice, s);
}

void launch_check_offsets(const Buffers& b, cudaStream_t s, int64_t* launches) {
  k_check_offsets<<<grid_for(b.n_cells + 1), kBlock, 0, s>>>(b.n_cells, b.fstart, (uint32_t)b.n, b.glob);
  k_check_offsets<<<grid_for(b.n_cells + 1), kBlock, 0, s>>>(b.n_cells, b.wstart, (uint32_t)b.nw, b.glob);
  *launches += 2;
}

void launch_check_table(const Buffers& b, cudaStream_t s, int64_t* launches) {
  if (b.n == 0) return;
  k_check_table<<<grid_for(b.n), kBlock, 0, s>>>(b.n, b.nw, b.cap, b.nbr, b.nbc, b.glob);
  ++*launches;
}

// b.wnear from the sorted walls; tmp holds n_cells bytes of scratch.
void flag_near_wall_cells(const Buffers& b, uint8_t* tmp, cudaStream_t s) {
  if (b.n_cells == 0) return;
  const unsigned grid = grid_for(b.n_cells);
  uint8_t* bufs[2] = {b.wnear, tmp};
  k_wall_occupied<<<grid, kBlock, 0, s>>>(b.n_cells, b.wstart, bufs[b.dim & 1]);
  for (int a = 0; a < b.dim; ++a)       // ping-pong so the last pass writes b.wnear
    k_dilate_axis<<<grid, kBlock, 0, s>>>(b.n_cells, a, b.inst, b.n_inst, bufs[(b.dim + a) & 1],
                                          bufs[(b.dim + a + 1) & 1]);
}

}  // namespace sph
