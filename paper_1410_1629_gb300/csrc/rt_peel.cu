// The sorted peel-off pass of the forward launch: the walks of the peel-offs
// that the transport kernels recorded, ordered by instrument and start cell.
#include "rt_transport.cuh"

namespace rtk {

namespace {

// ---- the sorted peel-off pass
//
// The transport kernel hands each walked peel-off to this pass as a record
// (start point, weight, phase-function value) counted under its sort key
// (instrument, place of the start point's cell in an order that keeps
// neighbouring cells together).  Ordered by key, the records of a warp start in
// the same or neighbouring cells and walk parallel rays towards one
// instrument, so they cross the same cells together; in the transport kernel
// the lanes of a warp walk unrelated rays.  Each walk is the transport kernel's
// own (same arithmetic, same optical depth pair, same deposit), so only the
// order of the FP64 image additions differs from walking the peel-off in place.
//
// On trees and Voronoi grids every frame's peel-offs walk (80 % of the
// crossings): clumpy octree 52.0 -> 35.2 ms per 2e6 packets, k-d tree 70.0 ->
// 37.9 ms, Voronoi disk 52.8 -> 35.7 ms per 1.5e6 (the whole launch; the trees'
// walks kept together crossing by crossing, below); 23, 21 and 14 lanes active per
// instruction of the sorted walks against 9, 7 and 6 in place.  Bound by
// instruction issue (61-64 % of cycles), trees in the descent to the next leaf,
// Voronoi grids also by the face planes' wavefronts (74 % of the L1's).
//
// Instruments that look along the same direction (a frame and an SED of one
// view) see the same optical depth and phase-function value: one record and one
// walk serve all of them, and only the deposits differ.  Panchromatic disk
// (frame and SED; the whole calculation) 10.3 -> 8.8 ms, ragged disk 2.53 ->
// 2.44 ms.

// Resident blocks per SM that the walks' register allocation aims at (octree 3 /
// 4 / 5: 31.7 / 27.8 / 29.2 ms, k-d tree 31.5 / 30.0 / 32.7, Voronoi 29.4 / 25.6 /
// 26.2, before k_peel_together and the paired face planes; cartesian 4 / 5 / 6:
// 7.45 / 7.44 / 7.51 ms per 4e6 packets of the disk galaxy, without spills only at
// 4).
constexpr int kPeelBlocks = 4;

// Whether the walks of a warp are kept together crossing by crossing
// (k_peel_together) or only start together (k_peel_sorted): trees.  On the other
// grids the plain loop stays converged by itself and the ballot and the state
// across deposits cost more than they give (disk galaxy 7.6 against 11.6 ms per
// 4e6 packets, Voronoi disk 25.6 against 28.0 ms per 1.5e6; with ended rays
// replaced a warp's rays are no longer in the same cell: 33 ms).
template <class G>
constexpr bool kPeelTogether = false;
template <>
constexpr bool kPeelTogether<tr::OctGrid> = true;
template <>
constexpr bool kPeelTogether<tr::BinGrid> = true;

constexpr int kScanTile = 4096;  // keys per block of the scan (256 threads x 16)

// Exclusive scan of each tile of 4096 key counts in place; tile totals out.
__global__ void __launch_bounds__(256) k_peel_scan_tiles(unsigned* __restrict__ h, unsigned long long n,
                                                          unsigned* __restrict__ tile_sum) {
  __shared__ unsigned warp_tot[8];
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const unsigned long long base = (unsigned long long)blockIdx.x * kScanTile + threadIdx.x * 16ull;
  unsigned v[16];
  unsigned sum = 0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    v[j] = base + j < n ? h[base + j] : 0u;
    sum += v[j];
  }
  unsigned incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (unsigned)o) incl += t;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const unsigned w = lane < 8 ? warp_tot[lane] : 0u;
    unsigned wi = w;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= (unsigned)o) wi += t;
    }
    if (lane < 8) warp_tot[lane] = wi - w;
    if (lane == 7) tile_sum[blockIdx.x] = wi;
  }
  __syncthreads();
  unsigned run = warp_tot[warp] + incl - sum;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (base + j < n) h[base + j] = run;
    run += v[j];
  }
}

// Exclusive scan of the tile totals in place (one block).
__global__ void __launch_bounds__(1024) k_peel_scan_sums(unsigned* __restrict__ ts, unsigned long long n) {
  __shared__ unsigned warp_tot[32];
  __shared__ unsigned carry;
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0u;
  __syncthreads();
  for (unsigned long long b = 0; b < n; b += 1024) {
    const unsigned long long i = b + threadIdx.x;
    const unsigned v = i < n ? ts[i] : 0u;
    unsigned incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= (unsigned)o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const unsigned w = warp_tot[lane];
      unsigned wi = w;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, wi, o);
        if (lane >= (unsigned)o) wi += t;
      }
      warp_tot[lane] = wi - w;
    }
    __syncthreads();
    const unsigned c0 = carry;
    const unsigned ex = c0 + warp_tot[warp] + incl - v;
    if (i < n) ts[i] = ex;
    __syncthreads();
    if (threadIdx.x == 1023) carry = ex + v;
    __syncthreads();
  }
}

// The permutation that orders the records by key: a record's place is its
// tile's base, plus its key's offset in the tile, plus the records of that
// key placed before it.
__global__ void __launch_bounds__(256) k_peel_scatter(const PeelRecord* __restrict__ rec,
                                                       const unsigned long long* __restrict__ count,
                                                       unsigned long long cap, unsigned* __restrict__ h,
                                                       const unsigned* __restrict__ tile_sum,
                                                       unsigned* __restrict__ perm) {
  const unsigned long long n = min(*count, cap);
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned key = __ldg(&rec[i].key);
    const unsigned pos = tile_sum[key / kScanTile] + atomicAdd(&h[key], 1u);
    perm[pos] = (unsigned)i;
  }
}

// A lane's crossings and the peel-offs that shared another's record, kept in
// local memory: touched once per ray.
struct Counts {
  unsigned long long crossings, shared;
};

__device__ __forceinline__ void add_counts(const FwdParams& P, const Counts& sum) {
  unsigned long long crossings = sum.crossings, shared = sum.shared;
  for (int o = 16; o > 0; o >>= 1) {
    crossings += __shfl_down_sync(0xffffffffu, crossings, o);
    shared += __shfl_down_sync(0xffffffffu, shared, o);
  }
  if ((threadIdx.x & 31u) == 0) {
    if (crossings) atomicAdd(&P.counters[0], crossings);
    if (shared) atomicAdd(&P.counters[8], shared);
  }
}

// The walks of the sorted records and their deposits; one record per thread,
// consecutive threads on consecutive records of the order.
template <class G>
__global__ void __launch_bounds__(tr::kBlock, kPeelBlocks) k_peel_sorted(const __grid_constant__ FwdParams P,
                                                                            const unsigned* __restrict__ perm) {
  tr::load_grid_cache<G>(P);
  __syncthreads();
  typename G::Scratch sc = tr::lane_scratch<G>(0);
  const unsigned long long n = min(*P.peel_count, P.peel_cap);
  if (blockIdx.x == 0 && threadIdx.x == 0 && n) atomicAdd(&P.counters[8], n);
  const unsigned stride_k = (unsigned)(P.n_cells + 1);
  Counts sum{0ull, 0ull};
  asm volatile("" ::"l"(&sum) : "memory");
  for (unsigned long long j = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; j < n;
       j += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned i = perm[j];
    const float4* r = reinterpret_cast<const float4*>(&P.peel[i]);
    const float4 a = r[0], b = r[1];
    const unsigned key = __float_as_uint(a.w);
    const unsigned meta = __float_as_uint(b.w);
    const int q = (int)(key / stride_k);
    const unsigned c = key - (unsigned)q * stride_k;
    const int lam = (int)(meta & 0xffffu);
    const bool known = (meta >> 31) != 0u;
    const double L = __hiloint2double(__float_as_int(b.y), __float_as_int(b.x));
    typename G::Cell cell;
    if (known) cell = G::sorted_cell(P, c);
    tr::Ray<G> ray;
    ray.x = make_float3(a.x, a.y, a.z);
    ray.d = tr::instr_dir(P.instr[q]);
    ray.kappa = P.lam[lam].kappa;
    unsigned steps = 0;
    if (tr::ray_start<G>(P, ray, known, cell, sc)) {
      do {
        ++steps;
      } while (tr::ray_step<G>(P, ray, sc));
    }
    const ulonglong2 tag = P.peel_tag ? P.peel_tag[i] : make_ulonglong2(0ull, 0ull);
    tr::deposit_peel(P, q, lam, ray.x, L, b.z, ray.th, ray.tl, (meta >> 30) & 1u, tag.x, (int)tag.y);
    // the instruments that share the record, one crossing and one peel-off each
    sum.crossings += steps;
    for (unsigned m = P.instr[q].followers; m; m &= m - 1u) {
      tr::deposit_peel(P, __ffs(m) - 1, lam, ray.x, L, b.z, ray.th, ray.tl, (meta >> 30) & 1u, tag.x, (int)tag.y);
      sum.crossings += steps;
      sum.shared += 1ull;
    }
  }
  add_counts(P, sum);
}

// Consecutive records that one warp walks, and the ended rays for which it stops
// to deposit them and start others (12 / 16 / 24 / 32: octree 18.9 / 19.6 / 18.5 /
// 18.7 ms, k-d tree 18.2 / 18.0 / 18.2 / 19.1 ms).
constexpr int kSegment = 256, kRefill = 24;

// The walks of the sorted records and their deposits.  A warp takes kSegment
// consecutive records of the order and keeps its lanes walking: ended rays are
// deposited and replaced by the segment's next records, kRefill at a time.  The
// ballot at the loop's head brings the lanes together again after every
// crossing: in k_peel_sorted the lanes of a tree walk drift apart in the
// branches of the descent (octree 27.8 -> 18.5 ms per 2e6 packets of the clumpy
// medium, k-d tree 30.1 -> 18.2 ms).
//
// kShare: some records serve several instruments.  Their deposits are a loop, for
// which the walking lanes' rays go to local memory (left in registers, the tree
// walks spill: octree 18.7 -> 20.7 ms; saved 19.9 ms).  Without any the plain
// kernel runs.
template <class G, bool kShare>
__global__ void __launch_bounds__(tr::kBlock, kPeelBlocks) k_peel_together(const __grid_constant__ FwdParams P,
                                                                            const unsigned* __restrict__ perm) {
  tr::load_grid_cache<G>(P);
  __syncthreads();
  typename G::Scratch sc = tr::lane_scratch<G>(0);
  const unsigned long long n = min(*P.peel_count, P.peel_cap);
  if (blockIdx.x == 0 && threadIdx.x == 0 && n) atomicAdd(&P.counters[8], n);
  const unsigned stride_k = (unsigned)(P.n_cells + 1);
  const unsigned lt_mask = (1u << (threadIdx.x & 31u)) - 1u;
  const unsigned long long n_warps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
  unsigned crossings = 0;  // of the lane's segment (kShare: of its ray)
  Counts sum{0ull, 0ull};
  asm volatile("" ::"l"(&sum) : "memory");
  for (unsigned long long seg = blockIdx.x * (unsigned long long)(blockDim.x >> 5) + (threadIdx.x >> 5);
       seg * kSegment < n; seg += n_warps) {
    unsigned long long next = seg * kSegment;
    const unsigned long long end = min(n, next + kSegment);
    tr::Ray<G> ray;
    bool walking = false, held = false;
    unsigned rec = 0;  // the lane's record
    int wait = 0;
    while (true) {
      const unsigned idle = __ballot_sync(0xffffffffu, !walking);
      if (__popc(idle) >= wait) {
        tr::Ray<G> saved;
        if constexpr (kShare) {
          saved = ray;
          asm volatile("" ::"l"(&saved) : "memory");
        }
        if (held && !walking) {
          const float4* r = reinterpret_cast<const float4*>(&P.peel[rec]);
          const float4 a = r[0], b = r[1];
          const unsigned meta = __float_as_uint(b.w);
          const ulonglong2 tag = P.peel_tag ? P.peel_tag[rec] : make_ulonglong2(0ull, 0ull);
          const int q = (int)(__float_as_uint(a.w) / stride_k);
          unsigned m = kShare ? P.instr[q].followers | 1u << q : 1u << q;
          do {
            tr::deposit_peel(P, kShare ? __ffs(m) - 1 : q, (int)(meta & 0xffffu), make_float3(a.x, a.y, a.z),
                             __hiloint2double(__float_as_int(b.y), __float_as_int(b.x)), b.z, ray.th, ray.tl,
                             (meta >> 30) & 1u, tag.x, (int)tag.y);
            if constexpr (kShare) {
              sum.crossings += crossings;
              m &= m - 1u;
              if (m) sum.shared += 1ull;
            }
          } while (kShare && m);
          if constexpr (kShare) crossings = 0;
          held = false;
        }
        if constexpr (kShare) {
          asm volatile("" ::"l"(&saved) : "memory");
          ray = saved;
        }
        const unsigned long long j = next + __popc(idle & lt_mask);
        if (!walking && j < end) {
          rec = perm[j];
          const float4* r = reinterpret_cast<const float4*>(&P.peel[rec]);
          const float4 a = r[0];
          const unsigned key = __float_as_uint(a.w), meta = __float_as_uint(r[1].w);
          const unsigned q = key / stride_k;
          const bool known = (meta >> 31) != 0u;
          typename G::Cell cell;
          if (known) cell = G::sorted_cell(P, key - q * stride_k);
          ray.x = make_float3(a.x, a.y, a.z);
          ray.d = tr::instr_dir(P.instr[q]);
          ray.kappa = P.lam[meta & 0xffffu].kappa;
          walking = tr::ray_start<G>(P, ray, known, cell, sc);
          held = true;
        }
        next = min(end, next + __popc(idle));
        const int busy = __popc(__ballot_sync(0xffffffffu, held));
        if (busy == 0) break;
        // at the segment's end the remaining rays all finish first
        wait = next < end ? 32 - busy + kRefill : 32;
      }
      if (walking) {
        walking = tr::ray_step<G>(P, ray, sc);
        crossings += 1u;
      }
    }
    sum.crossings += crossings;
    crossings = 0;
  }
  add_counts(P, sum);
}

template <class G>
cudaError_t launch_walks(const FwdParams& p, const unsigned* perm, int num_sms, size_t smem, cudaStream_t stream) {
  void (*kernel)(const FwdParams, const unsigned*);
  if constexpr (kPeelTogether<G>) {
    unsigned shared = 0;
    for (int q = 0; q < p.n_instr; ++q) shared |= p.instr[q].followers;
    kernel = shared ? k_peel_together<G, true> : k_peel_together<G, false>;
  } else {
    kernel = k_peel_sorted<G>;
  }
  cudaError_t e = cudaSuccess;
  if (smem) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tr::kMaxScratch<G>);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, tr::kBlock, smem);
  if (e != cudaSuccess) return e;
  per_sm = per_sm < 1 ? 1 : per_sm;
  kernel<<<(unsigned)num_sms * (unsigned)per_sm, tr::kBlock, smem, stream>>>(p, perm);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_peel_pass(const FwdParams& p, int grid_kind, unsigned long long n_keys, unsigned* tile_sum,
                             unsigned* perm, int num_sms, cudaStream_t stream, cudaEvent_t mid) {
  const unsigned long long n_tiles = (n_keys + kScanTile - 1) / kScanTile;
  k_peel_scan_tiles<<<(unsigned)n_tiles, 256, 0, stream>>>(p.peel_hist, n_keys, tile_sum);
  k_peel_scan_sums<<<1, 1024, 0, stream>>>(tile_sum, n_tiles);
  k_peel_scatter<<<(unsigned)num_sms * 8u, 256, 0, stream>>>(p.peel, p.peel_count, p.peel_cap, p.peel_hist, tile_sum,
                                                            perm);
  if (mid) {
    const cudaError_t em = cudaEventRecord(mid, stream);
    if (em != cudaSuccess) return em;
  }
  switch (grid_kind) {
    case RT_GRID_RECTILINEAR: return launch_walks<tr::RectGrid>(p, perm, num_sms, 0, stream);
    case RT_GRID_OCTREE:
      return launch_walks<tr::OctGrid>(p, perm, num_sms, (size_t)tr::kBlock * (size_t)p.oct_levels * sizeof(int), stream);
    case RT_GRID_BINTREE: return launch_walks<tr::BinGrid>(p, perm, num_sms, 0, stream);
    case RT_GRID_VORONOI: return launch_walks<tr::VorGrid>(p, perm, num_sms, 0, stream);
    default: return launch_walks<tr::CartGrid>(p, perm, num_sms, 0, stream);
  }
}

}  // namespace rtk
