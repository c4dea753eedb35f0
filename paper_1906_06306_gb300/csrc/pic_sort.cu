// Counting sort of particles by spatial tile: the single-GPU stand-in for the
// particle communication routines of Table 1 (arXiv:1906.06306), which move
// particles to the tile that owns them.  count -> exclusive scan -> scatter.
// Blocks work on chunks of consecutive particles, which in a nearly sorted array
// hold few bins, and reach the global counters and cursors once per bin.
#include "pic_kernels.h"

namespace pic {

// Sort bin of a cell: its tile, then the sub-tile inside it (tile-major); every
// division is an exact multiply-shift (FastDiv), and axes that are not gridded
// take none.
template <int D>
__device__ __forceinline__ int tile_key(const SortParams& P, int cell) {
  if (cell < 0 || (long long)cell >= P.g.plane) {
    atomicOr(P.status, ST_BAD_CELL);
    return 0;  // kept (in tile 0) so that no particle is lost
  }
  int x[3] = {cell, 0, 0};
  if (D >= 2) {
    x[1] = fdiv(cell, P.dn0);
    x[0] = cell - x[1] * P.g.n[0];
  }
  if (D == 3) {
    x[2] = fdiv(x[1], P.dn1);
    x[1] -= x[2] * P.g.n[1];
  }
  const FastDiv* dt[3] = {&P.dt0, &P.dt1, &P.dt2};
  const FastDiv* ds[3] = {&P.ds0, &P.ds1, &P.ds2};
  int tile = 0, sub = 0;
#pragma unroll
  for (int d = D - 1; d >= 0; --d) {
    const int t = fdiv(x[d], *dt[d]);
    tile = tile * P.t.nt[d] + t;
    x[d] -= t * P.t.T[d];
  }
  if constexpr (D > 1) {  // 1D tiles are not subdivided
#pragma unroll
    for (int d = D - 1; d >= 0; --d) sub = sub * P.t.ns[d] + fdiv(x[d], *ds[d]);
  }
  return tile * P.t.nsub + sub;
}

// Reserve `1` slot of counter[key] for every active lane; returns this lane's
// slot.  Lanes with equal keys share one atomic.
__device__ __forceinline__ int warp_reserve(int* counter, int key, unsigned active) {
  const unsigned peers = __match_any_sync(active, key);
  const int leader = __ffs(peers) - 1;
  const int lane = threadIdx.x & 31;
  int base = 0;
  if (lane == leader) base = atomicAdd(&counter[key], __popc(peers));
  base = __shfl_sync(peers, base, leader);
  return base + __popc(peers & lanemask_lt());
}

// Bins of a block's contiguous chunk of particles, counted in a shared-memory
// table before the global counters: in a sorted or nearly sorted array a
// chunk spans a few bins and their neighbours, so each of those reaches the
// global count once per block (same-address global atomics were the limit of
// a count per warp).  A table slot is claimed by compare-and-swap, looked at
// first so that a claimed slot costs a load; a bin whose slot another bin
// holds goes straight to the global count.  Lanes add 1 each: the hardware
// counts a warp's equal addresses in one go, where combining them by
// match_any first took 60 us against 43 for 16.8 M particles.
constexpr int kCountSlots = 1024;
template <int D>
__global__ void __launch_bounds__(256) k_tile_count(const SortParams P, const SortSet Q,
                                                    long long chunk) {
  grid_dependency();
  const int* __restrict__ cell = Q.sp[blockIdx.y].cell;
  int* const count = Q.sp[blockIdx.y].count;
  const long long n = Q.sp[blockIdx.y].n;
  const long long lo = (long long)blockIdx.x * chunk;
  if (lo >= n) return;  // a smaller species than another of the launch
  __shared__ int skey[kCountSlots];
  __shared__ int scnt[kCountSlots];
  for (int s = threadIdx.x; s < kCountSlots; s += blockDim.x) {
    skey[s] = -1;
    scnt[s] = 0;
  }
  __syncthreads();
  const long long hi = lo + chunk < n ? lo + chunk : n;
  constexpr int U = 4;  // rounds whose loads are issued together (4 loads in flight per thread)
  for (long long base = lo; base < hi; base += U * blockDim.x) {  // block-uniform trip count
    int c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long p = base + u * blockDim.x + threadIdx.x;
      c[u] = p < hi ? cell[p] : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (base + u * blockDim.x + threadIdx.x < hi) {
        const int key = tile_key<D>(P, c[u]);
        const int slot = (int)(((unsigned)key * 2654435761u) >> 22);  // multiplicative hash, 10 bits
        int old = *(volatile int*)&skey[slot];
        if (old == -1) old = atomicCAS(&skey[slot], -1, key);
        if (old == -1 || old == key)
          atomicAdd(&scnt[slot], 1);
        else
          atomicAdd(&count[key], 1);
      }
    }
  }
  __syncthreads();
  for (int s = threadIdx.x; s < kCountSlots; s += blockDim.x)
    if (skey[s] >= 0) atomicAdd(&count[skey[s]], scnt[s]);
}

// Exclusive scan of count[0..ntiles) into start[0..ntiles] (start[ntiles] =
// total) and cursor = start, in one block of 1024 threads per species; with
// parts, of the multi-block form's block totals instead (ntiles of them).
__global__ void __launch_bounds__(1024) k_tile_scan(const SortSet Q, int ntiles, int parts) {
  grid_dependency();
  const SortSpecies& S = Q.sp[blockIdx.x];
  const int* count = parts ? S.scratch : S.count;
  int* start = parts ? S.scratch + ntiles : S.start;
  int* cursor = parts ? S.scratch + 2 * ntiles + 1 : S.cursor;
  __shared__ int warp_sums[32];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int base = 0; base < ntiles; base += 1024) {
    const int t = base + threadIdx.x;
    const int v = t < ntiles ? count[t] : 0;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
      int s = warp_sums[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
      }
      warp_sums[lane] = s;
    }
    __syncthreads();
    const int incl = x + (wid > 0 ? warp_sums[wid - 1] : 0) + carry;
    if (t < ntiles) {
      start[t] = incl - v;
      cursor[t] = incl - v;
    }
    __syncthreads();
    if (threadIdx.x == 1023) carry = incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) start[ntiles] = carry;
}

// Multi-block form of the same exclusive scan for long count arrays (sub-tile
// sort bins): each block scans kScanChunk counts into start and leaves its
// total in part[]; one block scans part[]; every block then adds its offset
// (start[bins] = total, cursor = start).
constexpr int kScanChunk = 4096;  // counts per block: 4 per thread of 1024
__global__ void __launch_bounds__(1024) k_scan_chunks(const SortSet Q, int n) {
  grid_dependency();
  const int* __restrict__ count = Q.sp[blockIdx.y].count;
  int* start = Q.sp[blockIdx.y].start;
  int* part = Q.sp[blockIdx.y].scratch;
  __shared__ int warp_sums[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int base = blockIdx.x * kScanChunk + 4 * threadIdx.x;
  int v[4], s = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[i] = base + i < n ? count[base + i] : 0;
    s += v[i];
  }
  int x = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int w = warp_sums[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    warp_sums[lane] = w;
  }
  __syncthreads();
  int run = x - s + (wid > 0 ? warp_sums[wid - 1] : 0);  // exclusive offset in the chunk
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (base + i < n) start[base + i] = run;
    run += v[i];
  }
  if (threadIdx.x == 1023) part[blockIdx.x] = run;
}

__global__ void __launch_bounds__(1024) k_scan_add(const SortSet Q, int n) {
  grid_dependency();
  int* start = Q.sp[blockIdx.y].start;
  int* cursor = Q.sp[blockIdx.y].cursor;
  const int* part_scan = Q.sp[blockIdx.y].scratch + gridDim.x;
  const int off = part_scan[blockIdx.x];
  const int base = blockIdx.x * kScanChunk + 4 * threadIdx.x;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (base + i < n) {
      const int v = start[base + i] + off;
      start[base + i] = v;
      cursor[base + i] = v;
    }
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) start[n] = part_scan[gridDim.x];
}

#define SORT_SPECIES_ARRAYS(S)                \
  const int* __restrict__ cell = S.cell;      \
  const float* __restrict__ off = S.off;      \
  const float* __restrict__ u = S.u;          \
  const long long n = S.n, ld = S.ld;         \
  int* cursor = S.cursor;                     \
  int* __restrict__ cell_out = S.cell_out;    \
  float* __restrict__ off_out = S.off_out;    \
  float* __restrict__ u_out = S.u_out;        \
  int* __restrict__ perm = S.perm;

template <int D>
__global__ void k_tile_scatter_lanes(const SortParams P, const SortSet Q) {
  grid_dependency();
  SORT_SPECIES_ARRAYS(Q.sp[blockIdx.y])
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long base = (long long)blockIdx.x * blockDim.x; base < n; base += stride) {
    const long long p = base + threadIdx.x;
    const bool act = p < n;
    const unsigned active = __ballot_sync(0xffffffffu, act);
    if (act) {
      const int c = cell[p];
      const long long q = warp_reserve(cursor, tile_key<D>(P, c), active);
      cell_out[q] = c;
#pragma unroll
      for (int d = 0; d < D; ++d) off_out[d * ld + q] = off[d * ld + p];
#pragma unroll
      for (int a = 0; a < 3; ++a) u_out[a * ld + q] = u[a * ld + p];
      if (perm) perm[q] = (int)p;  // the slot the particle held before the sort
    }
  }
}

// Whether a warp's particles are of one bin (lanes without one count as of it;
// lane 0 has one unless none has), or of no more than two, those of its lanes 0
// and 31.  Every lane of the warp calls these.
__device__ __forceinline__ bool one_bin(int key, bool active) {
  const int first = __shfl_sync(0xffffffffu, key, 0);
  return __all_sync(0xffffffffu, !active || key == first);
}
__device__ __forceinline__ bool two_bins(int key, bool active) {
  const int first = __shfl_sync(0xffffffffu, key, 0), last = __shfl_sync(0xffffffffu, key, 31);
  return __all_sync(0xffffffffu, !active || key == first || key == last);
}

// The scatter of many particles.  A block takes U * 256 consecutive ones, puts
// them into bin order in shared memory and writes each bin's to consecutive
// slots: the array was sorted some steps ago, so a chunk holds a few bins and
// their neighbours, and a warp's stores are a few runs instead of a lane each
// wherever it falls.  16.8 M 2D particles 10 steps after a sort: 381 us (2.1
// TB/s, bound by partial sectors) -> 172 us (4.7 TB/s); 134 M 3D ones 3 steps
// after: the whole sort 3.14 -> 1.61 ms per 33.5 M.  A bin's particles of the
// block are counted in a table as in k_tile_count, each lane with its own
// shared atomic, whose result is the particle's place in its bin (combining a
// warp's equal bins first took 202 us); a particle whose table slot another
// bin holds reserves its place in the global cursor by itself.  Lanes of one
// bin take their places one after the other, which costs most in an array that
// is in order already.  A warp whose first particles of the chunk are of no more
// than two bins therefore adds 32 at once where a round's particles are of one.
// pic_sort on an array in order, two species of 16.8 M: 3D 975 -> 886 us, 2D 731
// -> 684; on one in cell order, 2D 883 -> 764; drifted arrays and sorts in a run
// within 0.3 %.  Scattered lane by lane, as few particles are below, an array in
// order takes 800 and 706, a drifted one twice as long as here.
template <int D, int U>
__global__ void __launch_bounds__(256) k_tile_scatter(const SortParams P, const SortSet Q) {
  grid_dependency();
  constexpr int kChunk = 256 * U;
  SORT_SPECIES_ARRAYS(Q.sp[blockIdx.y])
  if ((long long)blockIdx.x * kChunk >= n) return;  // a smaller species than another of the launch
  __shared__ int skey[kCountSlots];  // bin of a table slot, then the bin's reserved global slot
  __shared__ int scnt[kCountSlots];  // its particles here, then their first place in bin order
  __shared__ int sdst[kChunk];       // global slot of each place in bin order
  __shared__ int stage[2][kChunk];
  __shared__ int warp_sums[8], lone;  // lone: particles without a table slot
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  for (int i = t; i < kCountSlots; i += 256) {
    skey[i] = -1;
    scnt[i] = 0;
  }
  if (t == 0) lone = 0;
  const long long base = (long long)blockIdx.x * kChunk;
  const int here = (int)(n - base < kChunk ? n - base : kChunk);
  int c[U], slot[U], rank[U];  // slot < 0: no table slot, rank is the place among the lone ones
#pragma unroll
  for (int r = 0; r < U; ++r) c[r] = r * 256 + t < here ? cell[base + r * 256 + t] : 0;
  int lone_dst[U];
  const auto take = [&](int r, int key, int number) {  // this lane's table slot and place, for `number`
    const int s = (int)(((unsigned)key * 2654435761u) >> 22);  // multiplicative hash, 10 bits
    int old = *(volatile int*)&skey[s];
    if (old == -1) old = atomicCAS(&skey[s], -1, key);
    if (old == -1 || old == key) {
      slot[r] = s;
      rank[r] = atomicAdd(&scnt[s], number);
    } else {
      slot[r] = -1;
      rank[r] = atomicAdd(&lone, number);
      lone_dst[r] = atomicAdd(&cursor[key], number);
    }
  };
#pragma unroll
  for (int r = 0; r < U; ++r) {
    slot[r] = 0;
    rank[r] = 0;
    lone_dst[r] = 0;
  }
  __syncthreads();
  const bool in0 = t < here;
  if (two_bins(in0 ? tile_key<D>(P, c[0]) : -1, in0)) {
    unsigned together = 0;  // bit r: round r's particles of this warp are of one bin
#pragma unroll
    for (int r = 0; r < U; ++r) {
      const bool in = r * 256 + t < here;
      const int key = in ? tile_key<D>(P, c[r]) : -1;
      const bool one = one_bin(key, in);
      if (one) together |= 1u << r;
      if (in && (!one || lane == 0)) take(r, key, one ? min(32, here - (r * 256 + t)) : 1);
    }
    // after the loop, so that its atomics are in flight together
#pragma unroll
    for (int r = 0; r < U; ++r) {
      if (together >> r & 1) {
        slot[r] = __shfl_sync(0xffffffffu, slot[r], 0);
        rank[r] = __shfl_sync(0xffffffffu, rank[r], 0) + lane;
        lone_dst[r] = __shfl_sync(0xffffffffu, lone_dst[r], 0) + lane;
      }
    }
  } else {
#pragma unroll
    for (int r = 0; r < U; ++r)
      if (r * 256 + t < here) take(r, tile_key<D>(P, c[r]), 1);
  }
  __syncthreads();
  // exclusive scan of the table's counts, 4 slots to a thread; each bin's place
  // in the global order
  static_assert(kCountSlots == 4 * 256, "four table slots to a thread");
  int cnt[4], sum = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    cnt[i] = scnt[4 * t + i];
    sum += cnt[i];
  }
  int x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[wid] = x;
  __syncthreads();
  int run = x - sum;
  for (int w = 0; w < wid; ++w) run += warp_sums[w];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (cnt[i] > 0) skey[4 * t + i] = atomicAdd(&cursor[skey[4 * t + i]], cnt[i]);
    scnt[4 * t + i] = run;
    run += cnt[i];
  }
  __syncthreads();
  int place[U];  // in bin order; the lone particles follow the table's
#pragma unroll
  for (int r = 0; r < U; ++r) {
    if (r * 256 + t < here) {
      const int s = slot[r];
      place[r] = s >= 0 ? scnt[s] + rank[r] : here - lone + rank[r];
      sdst[place[r]] = s >= 0 ? skey[s] + rank[r] : lone_dst[r];
      stage[0][place[r]] = c[r];
    }
  }
  __syncthreads();
  int dst[U];
#pragma unroll
  for (int r = 0; r < U; ++r) dst[r] = r * 256 + t < here ? sdst[r * 256 + t] : -1;
  // row k of the record: cell, D offsets, 3 four-velocity components and, where
  // asked for, the slot the particle held before the sort; the next row is
  // loaded and staged while this one is written
  const int rows = 1 + D + 3 + (perm ? 1 : 0);
#pragma unroll 1
  for (int k = 0; k < rows; ++k) {
    int v[U];
    if (k + 1 < rows) {
      const int m = k + 1;
      const int* in = reinterpret_cast<const int*>(m <= D ? off + (m - 1) * ld : u + (m - 1 - D) * ld) + base;
#pragma unroll
      for (int r = 0; r < U; ++r)
        v[r] = r * 256 + t >= here ? 0 : m < 1 + D + 3 ? in[r * 256 + t] : (int)base + r * 256 + t;
    }
    int* out = k == 0 ? cell_out
               : k <= D ? reinterpret_cast<int*>(off_out + (k - 1) * ld)
               : k < 1 + D + 3 ? reinterpret_cast<int*>(u_out + (k - 1 - D) * ld)
                               : perm;
#pragma unroll
    for (int r = 0; r < U; ++r)
      if (dst[r] >= 0) out[dst[r]] = stage[k & 1][r * 256 + t];
    if (k + 1 < rows) {
#pragma unroll
      for (int r = 0; r < U; ++r)
        if (r * 256 + t < here) stage[(k + 1) & 1][place[r]] = v[r];
    }
    __syncthreads();
  }
}

SortParams make_sort_params(const GridDev& g, const TileDev& t, int* status) {
  SortParams P{};
  P.g = g;
  P.t = t;
  P.status = status;
  P.dn0 = make_fastdiv(g.n[0]);
  P.dn1 = make_fastdiv(g.n[1]);
  P.dt0 = make_fastdiv(t.T[0]);
  P.dt1 = make_fastdiv(t.T[1]);
  P.dt2 = make_fastdiv(t.T[2]);
  P.ds0 = make_fastdiv(t.S[0]);
  P.ds1 = make_fastdiv(t.S[1]);
  P.ds2 = make_fastdiv(t.S[2]);
  return P;
}

static unsigned blocks_for(long long n) {
  long long b = (n + 255) / 256;
  if (b > 152LL * 64) b = 152LL * 64;
  return (unsigned)(b < 1 ? 1 : b);
}

// The species of a sort share its launches: on small boxes a launch, not the
// work, is what a sort costs (1D box of 2 x 32,768 particles, a sort every 10
// steps, 20 steps: 188 -> 165 us; 2 x 707,560 2D ones 914 -> 886; with smaller
// chunks for the count).
static long long most_particles(const SortSet& Q) {
  long long n = 0;
  for (int s = 0; s < Q.ns; ++s) n = std::max(n, Q.sp[s].n);
  return n;
}

cudaError_t launch_tile_count(const SortParams& P, const SortSet& Q, cudaStream_t st) {
  const long long n = most_particles(Q);
  if (n == 0) return cudaSuccess;
  const int pdl = P.g.pdl;
  // contiguous chunks of 4096 particles or more (a multiple of 256), at most 16
  // blocks per SM; down to 1024 where that leaves SMs without a block
  long long nb = std::max((n + 4095) / 4096, std::min((n + 1023) / 1024, 152LL));
  if (nb > 152LL * 16) nb = 152LL * 16;
  const long long chunk = ((n + nb - 1) / nb + 255) / 256 * 256;
  const dim3 grid((unsigned)((n + chunk - 1) / chunk), Q.ns);
  switch (P.g.dim) {
    case 1: launch_kernel(pdl, k_tile_count<1>, grid, 256, 0, st, P, Q, chunk); break;
    case 2: launch_kernel(pdl, k_tile_count<2>, grid, 256, 0, st, P, Q, chunk); break;
    case 3: launch_kernel(pdl, k_tile_count<3>, grid, 256, 0, st, P, Q, chunk); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_tile_scan(const SortSet& Q, int bins, cudaStream_t st, int pdl) {
  if (bins <= kScanChunk) {
    launch_kernel(pdl, k_tile_scan, Q.ns, 1024, 0, st, Q, bins, 0);
    return cudaGetLastError();
  }
  // scratch: block totals [nb], their scan [nb + 1], the scan's cursor [nb]
  const int nb = (bins + kScanChunk - 1) / kScanChunk;
  launch_kernel(pdl, k_scan_chunks, dim3(nb, Q.ns), 1024, 0, st, Q, bins);
  launch_kernel(pdl, k_tile_scan, Q.ns, 1024, 0, st, Q, nb, 1);
  launch_kernel(pdl, k_scan_add, dim3(nb, Q.ns), 1024, 0, st, Q, bins);
  return cudaGetLastError();
}

cudaError_t launch_tile_scatter(const SortParams& P, const SortSet& Q, cudaStream_t st) {
  const long long n = most_particles(Q);
  if (n == 0) return cudaSuccess;
  const int pdl = P.g.pdl;
  const auto launch = [&](auto kernel, int chunk) {
    return launch_kernel(pdl, kernel, dim3((unsigned)((n + chunk - 1) / chunk), Q.ns), 256, 0, st,
                         P, Q);
  };
  // few particles: the lanes kernel, whose blocks of 256 spread them over more
  // of the chip (65,536 2D particles, whole sort: 70 us against 78 with 1024 to
  // a block; 262,144: 83 against 79, and 83 with 2048; 1.05 M: 133, 115, 111)
  const bool few = n < 1 << 17, some = n < 1 << 19;
  const dim3 grid(blocks_for(n), Q.ns);
#define PIC_SCATTER(D)                                                                     \
  if (few) return launch_kernel(pdl, k_tile_scatter_lanes<D>, grid, 256, 0, st, P, Q);     \
  return some ? launch(k_tile_scatter<D, 4>, 1024) : launch(k_tile_scatter<D, 8>, 2048);
  switch (P.g.dim) {
    case 1: PIC_SCATTER(1)
    case 2: PIC_SCATTER(2)
    case 3: PIC_SCATTER(3)
    default: return cudaErrorInvalidValue;
  }
#undef PIC_SCATTER
}

// Bucket starts handed in from outside: one block checks that they run from
// 0 to n without decreasing; if not, every start but the last becomes 0 (one
// bucket: the last tile's blocks take every particle, all through the stray
// path) and the status word says so.
__device__ __forceinline__ void check_buckets(int* __restrict__ t, long long nb, long long n,
                                              int* status) {
  bool bad = threadIdx.x == 0 && (t[0] != 0 || t[nb] != n);
  for (long long i = threadIdx.x; i < nb; i += blockDim.x) bad |= t[i] > t[i + 1];
  if (!__syncthreads_or(bad)) return;
  for (long long i = threadIdx.x; i < nb; i += blockDim.x) t[i] = 0;
  if (threadIdx.x == 0) {
    t[nb] = (int)n;
    atomicOr(status, ST_BAD_BUCKETS);
  }
}

__global__ void k_check_buckets(int* __restrict__ t, long long nb, long long n, int* status) {
  grid_dependency();
  check_buckets(t, nb, n, status);
}

cudaError_t launch_check_buckets(int* tstart, long long nb, long long n, int* status,
                                 cudaStream_t st, int pdl) {
  return launch_kernel(pdl, k_check_buckets, 1, 1024, 0, st, tstart, nb, n, status);
}

// Block s: species s's bucket starts, copied and checked.
__global__ void __launch_bounds__(1024) k_adopt_buckets(const BucketCopies C, long long nb,
                                                        int* dcount, int* status) {
  grid_dependency();
  const int s = blockIdx.x;
  if (threadIdx.x == 0) dcount[s] = 0;
  const int* src = C.src[s];
  int* dst = C.dst[s];
  if (!src) return;
  for (long long i = threadIdx.x; i <= nb; i += blockDim.x) dst[i] = src[i];
  __syncthreads();
  check_buckets(dst, nb, C.n[s], status);
}

cudaError_t launch_adopt_buckets(const BucketCopies& C, int nspecies, long long nb, int* dcount,
                                 int* status, cudaStream_t st, int pdl) {
  return launch_kernel(pdl, k_adopt_buckets, nspecies, 1024, 0, st, C, nb, dcount, status);
}

// Bucket starts of one slot range [lo, hi) of a species: out[i] = tstart[i]
// clamped to [lo, hi), so that bucket i of the clipped starts is bucket i's
// part inside the range (a particle launch over the clipped starts processes
// the slots of that range only).
__global__ void k_clip_starts(const int* __restrict__ t, long long nb1, int lo, int hi,
                              int* __restrict__ out) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nb1; i += stride)
    out[i] = min(max(t[i], lo), hi);
}

cudaError_t launch_clip_starts(const int* tstart, long long nb1, int lo, int hi, int* out,
                               cudaStream_t st) {
  if (nb1 <= 0) return cudaSuccess;
  const long long blocks = std::min<long long>((nb1 + 255) / 256, 4 * 152);
  k_clip_starts<<<(unsigned)blocks, 256, 0, st>>>(tstart, nb1, lo, hi, out);
  return cudaGetLastError();
}

// Adjoint of a sort's permutation: the gradient rows of the particle now in
// slot i go to the slot it held before the sort, perm[i] (out[perm[i]] =
// in[i] on each of the `rows` rows of length ld).  An entry outside [0, n)
// is skipped and reported (ST_BAD_BUCKETS): the permutation came from the
// caller.
__global__ void k_unpermute(const int* __restrict__ perm, const float* __restrict__ in,
                            float* __restrict__ out, long long n, long long ld, int rows,
                            int* status) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const long long q = perm[i];
    if (q < 0 || q >= n) {
      atomicOr(status, ST_BAD_BUCKETS);
      continue;
    }
    for (int r = 0; r < rows; ++r) out[r * ld + q] = in[r * ld + i];
  }
}

cudaError_t launch_unpermute(const int* perm, const float* in, float* out, long long n,
                             long long ld, int rows, int* status, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_unpermute<<<blocks_for(n), 256, 0, st>>>(perm, in, out, n, ld, rows, status);
  return cudaGetLastError();
}

}  // namespace pic
