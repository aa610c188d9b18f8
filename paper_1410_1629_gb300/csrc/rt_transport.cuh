// The forward transport kernel, templated on the dust grid's cell walk:
// emission, peel-off, forced scattering with continuous absorption,
// Henyey-Greenstein scattering and termination for a stream of photon packets
// (SKIRT paper, Sect. 1 and Sect. 2.2-2.4).
//
// Execution model.  A persistent grid of warps; every warp carries more packets
// (G::kSlots, state in shared memory) than it has lanes, and a lane holds in
// registers only the walk it is on.  The expensive part of the method is the
// straight cell walk: two walks of the forced path per scattering (the first
// accumulates the optical depth to the boundary and deposits absorption, the
// second stops at the interaction) and the peel-offs that neither column sums
// (frames along a grid axis) nor the sorted pass (rt_peel.cu) take.  The main
// loop advances every walking lane by exactly one cell crossing per iteration,
// whichever walk it is in.  A lane whose walk ended gets the next packet that
// is ready to walk; the per-event work (emission, forced-scattering inversion,
// weight update, deposits, the Henyey-Greenstein draw) runs in rounds over up
// to 32 packets of the warp that all wait for the same kind of work.
//
// What bounds it: instruction issue and the latency of the dependent density
// loads.  With one packet per lane (the warp's lanes waiting for one another)
// 21 of 32 lanes walked per iteration and 40 % of the cycles went to rounds
// serving 16 lanes in five stages; with the slots 27 walk and rounds take 9-25
// % (2e6 packets of the disk galaxy, execution counters).
//
// Precision.  Geometry, the walk and the phase function are FP32.  The
// cumulative optical depth of the forced path is held as an unevaluated sum
// of two FP32 numbers updated by an error-free two-sum (about 2^-46 relative),
// bit-identical in both walks, so the interaction cell is always found; the
// inversion remainder, E = exp(-tau), tau*, packet weights and every
// accumulator are FP64.
//
// A grid policy G supplies the walk: G::Cell (the cell a position lies in),
// G::Walk (the walk state), init / exit / advance / cell / carried / clamp.
#pragma once

#include <cuda_runtime.h>

#include "rt_device.cuh"
#include "rt_internal.h"

namespace rtk {
namespace tr {

constexpr int kBlock = 256;
constexpr float kInv4PiF = 0.0795774715459476679f;
// Resident blocks per SM the register allocation aims at (4 x 256 threads,
// 64 registers: the per-event lane state lives in shared memory).
#ifndef RT_FWD_MIN_BLOCKS
#define RT_FWD_MIN_BLOCKS 4
#endif

// Rounds of per-event work: a queue of at least kRoundMin packets is served at
// once, a shorter one when kIdleMax lanes have no walk.  Between (1, 0) and
// (24, 16): 41.7 to 40.3 ms per 4e6 packets of the disk galaxy, 22.8 to 21.0
// ms per 2e6 packets of an opaque 48^3 cube; flat around the values here.
constexpr int kRoundMin = 20, kIdleMax = 12;
// A launch of few packets uses fewer blocks, down to kSpread packets per warp:
// 1e3 packets of a 32^3 cube 336 us at 4 per warp, 404 us at 16, 440 us at 32;
// 1e4 416, 444, 489 us.
constexpr int kSpread = 4;
// Packet slots per warp, by grid (see Shared): as many as leave the shared
// memory of four blocks at 164 KB on cartesian and rectilinear grids (92 KB of
// the SM's 256 remain for L1; the next step, 196 KB, costs the disk galaxy
// nothing at 52 slots of a larger layout, the last, 228 KB, 41 -> 50 ms per
// 4e6 packets) and within reach of four blocks on the others.  48 / 56 / 60 /
// 64 slots: disk galaxy 40.9 / 40.5 / 40.5 / 40.8 ms, opaque cube 21.5 / 20.2
// / 19.7 / 19.6 ms; octree 36 / 48 / 56: 30.0 / 27.0 / 30.5 ms per 1e6 packets;
// k-d tree 36 / 52 / 60: 39.4 / 36.6 / 37.1 ms.
#ifndef RT_SLOTS_INDEXED
#define RT_SLOTS_INDEXED 60
#endif
#ifndef RT_SLOTS_OCT
#define RT_SLOTS_OCT 48
#endif
#ifndef RT_SLOTS_BIN
#define RT_SLOTS_BIN 52
#endif
#ifndef RT_SLOTS_VOR
#define RT_SLOTS_VOR 52
#endif

enum Phase : int {
  kFetch = 0,      // needs a new packet
  kPeelEmit = 1,   // peel-off walk at emission (instrument q)
  kPath1 = 2,      // forced path, first walk
  kPath2 = 3,      // forced path, second walk (stops at the interaction)
  kPeelScat = 4,   // peel-off walk at a scattering (instrument q)
  kExit = 5,       // no packets left
  kPeelScan = 6,   // find the next peel-off of the event from instrument q
  kAfter = 7,      // after the scattering peel-offs
  kStart = 8       // start walk `wphase` from x along d
};

// Error-free transformation: a + b = s + e exactly (Knuth's two-sum).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  const float ap = __fsub_rn(s, bp);
  e = __fadd_rn(__fsub_rn(a, ap), __fsub_rn(b, bp));
}

__device__ __forceinline__ float inv_or_zero(float d) { return d != 0.0f ? 1.0f / d : 0.0f; }

// f 2^e in FP64 for a positive FP32 f, with integer operations (the widening
// above with the exponent moved by e); zero for results below FP64's normal
// range and for zero or non-finite f.
__device__ __forceinline__ double widen_exp(float f, int e) {
  const unsigned u = __float_as_uint(f);
  const int be = (int)((u >> 23) & 0xffu);
  if (be == 0 || be == 0xff) return be == 0 && (u & 0x7fffffu) ? ldexp((double)f, e) : 0.0;
  const int de = be - 127 + 1023 + e;  // biased FP64 exponent of the result
  if (de <= 0) return 0.0;
  const unsigned hi = ((unsigned)de << 20) | ((u & 0x7fffffu) >> 3);
  return __hiloint2double((int)hi, (int)(u << 29));
}

// A positive FP64 value v as m 2^e with m in [1/2, 1) cut to FP32 (integer
// operations); zero gives m = 0, e = 0.
__device__ __forceinline__ float split_exp(double v, int& e) {
  const long long b = __double_as_longlong(v);
  const int be = (int)((b >> 52) & 0x7ff);
  if (be == 0 || v <= 0.0) {
    e = 0;
    return 0.0f;
  }
  e = be - 1022;  // v = (1.m / 2) 2^(be - 1022)
  return __uint_as_float((126u << 23) | ((unsigned)(b >> 29) & 0x7fffffu));
}

// v as the unevaluated FP32 pair hi + lo: hi = v cut to 24 bits, lo = the
// remainder (exact in FP64) cut likewise: |v - hi - lo| < 2^-46 |v|.
__device__ __forceinline__ void split_pair(double v, float& hi, float& lo) {
  hi = cut(v);
  lo = cut(v - widen(hi));
}

// Uniform (r + 1/2) 2^-32 rounded to FP32 (= the FP64 value rounded), from
// the exact 33-bit integer 2r + 1.
__device__ __forceinline__ float u01f(uint32_t r) { return __ull2float_rn(2ull * r + 1ull) * 0x1p-33f; }

// 2u - 1 rounded to FP32, exactly: (2r + 1 - 2^32) 2^-32.
__device__ __forceinline__ float u01f_signed(uint32_t r) {
  return __ll2float_rn((long long)(2ull * r + 1ull) - (1ll << 32)) * 0x1p-32f;
}

// L2 residency: the density is read at every crossing and should stay in L2;
// absorption tallies are written once per forced-path crossing and should be
// the first lines evicted.
__device__ __forceinline__ float load_density(const float* p) {
  float v;
  asm volatile(
      "{\n\t.reg .b64 pol;\n\t"
      "createpolicy.fractional.L2::evict_last.b64 pol, 1.0;\n\t"
      "ld.global.nc.L2::cache_hint.f32 %0, [%1], pol;\n\t}"
      : "=f"(v)
      : "l"(p));
  return v;
}

// Two float4 at p (32-byte aligned) with one load.
__device__ __forceinline__ void load_pair(const float4* p, float4& a, float4& b) {
  asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
      : "l"(p));
}

__device__ __forceinline__ void add_absorption(double* p, double v) {
  asm volatile(
      "{\n\t.reg .b64 pol;\n\t"
      "createpolicy.fractional.L2::evict_first.b64 pol, 1.0;\n\t"
      "red.global.add.L2::cache_hint.f64 [%0], %1, pol;\n\t}" ::"l"(p),
      "d"(v)
      : "memory");
}

// 1 - exp(-x) for x >= 0 with a relative error below 5e-7: the alternating
// series through x^8 for x < 1/4 (truncation below 1e-10), 1 - exp(-x) above.
__device__ __forceinline__ float one_minus_exp_neg(float x) {
  if (x < 0.25f) {
    float p = fmaf(x, -1.0f / 40320.0f, 1.0f / 5040.0f);
    p = fmaf(x, p, -1.0f / 720.0f);
    p = fmaf(x, p, 1.0f / 120.0f);
    p = fmaf(x, p, -1.0f / 24.0f);
    p = fmaf(x, p, 1.0f / 6.0f);
    p = fmaf(x, p, -0.5f);
    p = fmaf(x, p, 1.0f);
    return x * p;
  }
  return 1.0f - expf(-x);
}

// Exit face of a cell: the first axis with the smallest exit parameter.
__device__ __forceinline__ float first_min(float tx, float ty, float tz, int& axis) {
  const bool by = ty < tx;
  const float txy = by ? ty : tx;
  const bool bz = tz < txy;
  axis = bz ? 2 : (by ? 1 : 0);
  return bz ? tz : txy;
}

__device__ __forceinline__ float pick(int a, float3 v) { return a == 2 ? v.z : (a == 1 ? v.y : v.x); }

// Storage stride of axis a: the launch's (FwdParams), row-major for any
// other geometry (one model of a batch).
template <class Geo>
__device__ __forceinline__ int stride_of(const Geo& P, int a) {
  return a == 0 ? 1 : (a == 1 ? P.nx : P.nx * P.ny);
}
__device__ __forceinline__ int stride_of(const FwdParams& P, int a) { return P.stride[a]; }

// ---------------------------------------------------------------- cartesian grid
struct CartGrid {
  static constexpr bool kColumns = true;  // peel-offs along grid axes may use column sums
  static constexpr bool kIndexCells = true;  // cells indexed by (ix, iy, iz) between planes
  static constexpr int kSlots = RT_SLOTS_INDEXED;
  struct Cell {
    int ix, iy, iz;
  };
  // current cell, entry parameter t of its segment, next-plane parameters
  struct Walk {
    int ix, iy, iz, cell;
    float t, tx, ty, tz;
  };
  struct Scratch {};

  // Geo: the grid geometry, nx, ny, nz, lo[3], hi[3], d[3], inv_d[3] (the
  // launch parameters, or one model of a batch).
  template <class Geo>
  __device__ static __forceinline__ float plane_t(const Geo& P, int a, int i, float xa, float ida) {
    return (fmaf((float)i, P.d[a], P.lo[a]) - xa) * ida;
  }

  // Start a walk from x along d (inverse id; id_a = 0 marks d_a = 0).  With a
  // known cell x lies in it; otherwise x is located or the entry point found.
  // False if the ray misses the grid.
  template <class Geo>
  __device__ static __forceinline__ bool init(const Geo& P, float3 x, float3 d, float3 id, bool known, const Cell& c,
                                              Walk& w, Scratch&) {
    w.t = 0.0f;
    if (known) {
      w.ix = c.ix; w.iy = c.iy; w.iz = c.iz;
    } else {
      int entry = -1;
      float3 p = x;
      if (!inside_box(P, x)) {
        const float3 ik = make_float3(id.x != 0.0f ? id.x : RT_INF, id.y != 0.0f ? id.y : RT_INF,
                                      id.z != 0.0f ? id.z : RT_INF);
        if (!ray_box_entry(P, x, d, ik, w.t, entry)) return false;
        p = make_float3(fmaf(w.t, d.x, x.x), fmaf(w.t, d.y, x.y), fmaf(w.t, d.z, x.z));
      }
      w.ix = min(max(__float2int_rd((p.x - P.lo[0]) * P.inv_d[0]), 0), P.nx - 1);
      w.iy = min(max(__float2int_rd((p.y - P.lo[1]) * P.inv_d[1]), 0), P.ny - 1);
      w.iz = min(max(__float2int_rd((p.z - P.lo[2]) * P.inv_d[2]), 0), P.nz - 1);
      if (entry == 0) w.ix = d.x > 0.0f ? 0 : P.nx - 1;
      if (entry == 1) w.iy = d.y > 0.0f ? 0 : P.ny - 1;
      if (entry == 2) w.iz = d.z > 0.0f ? 0 : P.nz - 1;
    }
    w.tx = id.x != 0.0f ? plane_t(P, 0, w.ix + (id.x > 0.0f), x.x, id.x) : RT_INF;
    w.ty = id.y != 0.0f ? plane_t(P, 1, w.iy + (id.y > 0.0f), x.y, id.y) : RT_INF;
    w.tz = id.z != 0.0f ? plane_t(P, 2, w.iz + (id.z > 0.0f), x.z, id.z) : RT_INF;
    w.cell = w.ix * stride_of(P, 0) + w.iy * stride_of(P, 1) + w.iz * stride_of(P, 2);
    return true;
  }

  // Back through face `axis`: the cell indices before the last advance (the
  // plane parameters stay; the walk ends here).
  __device__ static __forceinline__ void retreat(int axis, float3 id, Walk& w) {
    w.ix -= axis == 0 ? (id.x > 0.0f ? 1 : -1) : 0;
    w.iy -= axis == 1 ? (id.y > 0.0f ? 1 : -1) : 0;
    w.iz -= axis == 2 ? (id.z > 0.0f ? 1 : -1) : 0;
  }

  __device__ static __forceinline__ float exit(const Walk& w, float3, float3, int& axis) {
    return first_min(w.tx, w.ty, w.tz, axis);
  }

  // Move through face `axis` (w.t already at the exit); false when the ray
  // leaves the grid, in which case the walk still describes the last cell.
  // Selects rather than branches: the warp issues the advance once.
  template <class Geo>
  __device__ static __forceinline__ bool advance(const Geo& P, float3 x, float3, float3 id, int axis, Walk& w,
                                                 Scratch&) {
    const bool bz = axis == 2, by = axis == 1;
    const float ida = bz ? id.z : (by ? id.y : id.x);
    const int step = ida > 0.0f ? 1 : -1;
    const int ia = (bz ? w.iz : (by ? w.iy : w.ix)) + step;
    const int na = bz ? P.nz : (by ? P.ny : P.nx);
    if ((unsigned)ia >= (unsigned)na) return false;
    w.cell += step * (bz ? stride_of(P, 2) : (by ? stride_of(P, 1) : stride_of(P, 0)));
    const float xa = bz ? x.z : (by ? x.y : x.x);
    const float da = bz ? P.d[2] : (by ? P.d[1] : P.d[0]);
    const float loa = bz ? P.lo[2] : (by ? P.lo[1] : P.lo[0]);
    const float t_new = (fmaf((float)(ia + (step > 0)), da, loa) - xa) * ida;
    w.ix = (axis == 0) ? ia : w.ix;
    w.iy = by ? ia : w.iy;
    w.iz = bz ? ia : w.iz;
    w.tx = (axis == 0) ? t_new : w.tx;
    w.ty = by ? t_new : w.ty;
    w.tz = bz ? t_new : w.tz;
    return true;
  }

  __device__ static __forceinline__ int cell(const Walk& w) { return w.cell; }

  // The row-major cell id (records, traces, the tape).
  template <class Geo>
  __device__ static __forceinline__ int id(const Geo& P, const Walk& w) { return w.ix + P.nx * (w.iy + P.ny * w.iz); }

  // The row-major id of a carried cell.
  __device__ static __forceinline__ int cell_id(const FwdParams& P, const Cell& c) {
    return c.ix + P.nx * (c.iy + P.ny * c.iz);
  }

  // The sorted pass orders by the row-major index (by the storage index, z
  // fastest on the disk galaxy: its walks take 8.0 instead of 7.6 ms per 4e6
  // packets).
  __device__ static __forceinline__ int sort_place(const FwdParams& P, const Cell& c) { return cell_id(P, c); }
  __device__ static __forceinline__ Cell sorted_cell(const FwdParams& P, unsigned place) {
    return Cell{(int)(place % (unsigned)P.nx), (int)(place / (unsigned)P.nx % (unsigned)P.ny),
                (int)(place / ((unsigned)P.nx * (unsigned)P.ny))};
  }

  // Plane i of axis a.
  __device__ static __forceinline__ float plane(const FwdParams& P, int a, int i) {
    return fmaf((float)i, P.d[a], P.lo[a]);
  }

  // The cell of a point inside the grid.
  __device__ static __forceinline__ void locate_cell(const FwdParams& P, float3 x, Cell& c) {
    c.ix = min(max(__float2int_rd((x.x - P.lo[0]) * P.inv_d[0]), 0), P.nx - 1);
    c.iy = min(max(__float2int_rd((x.y - P.lo[1]) * P.inv_d[1]), 0), P.ny - 1);
    c.iz = min(max(__float2int_rd((x.z - P.lo[2]) * P.inv_d[2]), 0), P.nz - 1);
  }

  __device__ static __forceinline__ Cell carried(const Walk& w) { return Cell{w.ix, w.iy, w.iz}; }

  // Keep x inside cell c.
  template <class Geo>
  __device__ static __forceinline__ void clamp(const Geo& P, const Cell& c, float3& x) {
    x.x = fminf(fmaxf(x.x, fmaf((float)c.ix, P.d[0], P.lo[0])), fmaf((float)(c.ix + 1), P.d[0], P.lo[0]));
    x.y = fminf(fmaxf(x.y, fmaf((float)c.iy, P.d[1], P.lo[1])), fmaf((float)(c.iy + 1), P.d[1], P.lo[1]));
    x.z = fminf(fmaxf(x.z, fmaf((float)c.iz, P.d[2], P.lo[2])), fmaf((float)(c.iz + 1), P.d[2], P.lo[2]));
  }
};

// ---------------------------------------------------------------- rectilinear grid
// Cuboidal cells between increasing edges given per axis (Table 1(d): the
// PowCub grid places them by a power law; Sect. 2.2: logarithmic and
// power-law grids put smaller cells in the central areas).  The walk is the
// cartesian one with the plane positions read from the edge arrays (FP32
// copies of the FP64 edges); a position is located by binary search.
struct RectGrid {
  static constexpr bool kColumns = true;
  static constexpr bool kIndexCells = true;
  static constexpr int kSlots = RT_SLOTS_INDEXED;
  using Cell = CartGrid::Cell;
  using Walk = CartGrid::Walk;
  struct Scratch {};

  __device__ static __forceinline__ void retreat(int axis, float3 id, Walk& w) { CartGrid::retreat(axis, id, w); }
  __device__ static __forceinline__ float edge(const FwdParams& P, int a, int i) { return __ldg(&P.edge[a][i]); }

  // The cell along axis a that holds coordinate xa: the last i in [0, n) with
  // edge[i] <= xa (clamped into the grid).
  __device__ static __forceinline__ int locate(const FwdParams& P, int a, float xa, int n) {
    const float* e = P.edge[a];
    int lo = 0, hi = n - 1;  // answer in [lo, hi]
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(&e[mid]) <= xa) lo = mid; else hi = mid - 1;
    }
    return lo;
  }

  __device__ static __forceinline__ bool init(const FwdParams& P, float3 x, float3 d, float3 id, bool known,
                                              const Cell& c, Walk& w, Scratch&) {
    w.t = 0.0f;
    if (known) {
      w.ix = c.ix; w.iy = c.iy; w.iz = c.iz;
    } else {
      int entry = -1;
      float3 p = x;
      if (!inside_box(P, x)) {
        const float3 ik = make_float3(id.x != 0.0f ? id.x : RT_INF, id.y != 0.0f ? id.y : RT_INF,
                                      id.z != 0.0f ? id.z : RT_INF);
        if (!ray_box_entry(P, x, d, ik, w.t, entry)) return false;
        p = make_float3(fmaf(w.t, d.x, x.x), fmaf(w.t, d.y, x.y), fmaf(w.t, d.z, x.z));
      }
      w.ix = locate(P, 0, p.x, P.nx);
      w.iy = locate(P, 1, p.y, P.ny);
      w.iz = locate(P, 2, p.z, P.nz);
      if (entry == 0) w.ix = d.x > 0.0f ? 0 : P.nx - 1;
      if (entry == 1) w.iy = d.y > 0.0f ? 0 : P.ny - 1;
      if (entry == 2) w.iz = d.z > 0.0f ? 0 : P.nz - 1;
    }
    w.tx = id.x != 0.0f ? (edge(P, 0, w.ix + (id.x > 0.0f)) - x.x) * id.x : RT_INF;
    w.ty = id.y != 0.0f ? (edge(P, 1, w.iy + (id.y > 0.0f)) - x.y) * id.y : RT_INF;
    w.tz = id.z != 0.0f ? (edge(P, 2, w.iz + (id.z > 0.0f)) - x.z) * id.z : RT_INF;
    w.cell = w.ix * P.stride[0] + w.iy * P.stride[1] + w.iz * P.stride[2];
    return true;
  }

  __device__ static __forceinline__ float exit(const Walk& w, float3, float3, int& axis) {
    return first_min(w.tx, w.ty, w.tz, axis);
  }

  __device__ static __forceinline__ bool advance(const FwdParams& P, float3 x, float3, float3 id, int axis, Walk& w,
                                                 Scratch&) {
    const bool bz = axis == 2, by = axis == 1;
    const float ida = bz ? id.z : (by ? id.y : id.x);
    const int step = ida > 0.0f ? 1 : -1;
    const int ia = (bz ? w.iz : (by ? w.iy : w.ix)) + step;
    const int na = bz ? P.nz : (by ? P.ny : P.nx);
    if ((unsigned)ia >= (unsigned)na) return false;
    w.cell += step * (bz ? P.stride[2] : (by ? P.stride[1] : P.stride[0]));
    const float xa = bz ? x.z : (by ? x.y : x.x);
    const float t_new = (edge(P, axis, ia + (step > 0)) - xa) * ida;
    w.ix = (axis == 0) ? ia : w.ix;
    w.iy = by ? ia : w.iy;
    w.iz = bz ? ia : w.iz;
    w.tx = (axis == 0) ? t_new : w.tx;
    w.ty = by ? t_new : w.ty;
    w.tz = bz ? t_new : w.tz;
    return true;
  }

  __device__ static __forceinline__ int cell(const Walk& w) { return w.cell; }

  __device__ static __forceinline__ int id(const FwdParams& P, const Walk& w) {
    return w.ix + P.nx * (w.iy + P.ny * w.iz);
  }

  __device__ static __forceinline__ int cell_id(const FwdParams& P, const Cell& c) { return CartGrid::cell_id(P, c); }
  __device__ static __forceinline__ int sort_place(const FwdParams& P, const Cell& c) { return CartGrid::sort_place(P, c); }
  __device__ static __forceinline__ Cell sorted_cell(const FwdParams& P, unsigned place) {
    return CartGrid::sorted_cell(P, place);
  }

  __device__ static __forceinline__ float plane(const FwdParams& P, int a, int i) { return edge(P, a, i); }

  __device__ static __forceinline__ void locate_cell(const FwdParams& P, float3 x, Cell& c) {
    c.ix = locate(P, 0, x.x, P.nx);
    c.iy = locate(P, 1, x.y, P.ny);
    c.iz = locate(P, 2, x.z, P.nz);
  }

  __device__ static __forceinline__ Cell carried(const Walk& w) { return Cell{w.ix, w.iy, w.iz}; }

  __device__ static __forceinline__ void clamp(const FwdParams& P, const Cell& c, float3& x) {
    x.x = fminf(fmaxf(x.x, edge(P, 0, c.ix)), edge(P, 0, c.ix + 1));
    x.y = fminf(fmaxf(x.y, edge(P, 1, c.iy)), edge(P, 1, c.iy + 1));
    x.z = fminf(fmaxf(x.z, edge(P, 2, c.iz)), edge(P, 2, c.iz + 1));
  }
};

// ---------------------------------------------------------------- octree grid
// Nodes are split at box midpoints (Sect. 2.4); a point on a splitting plane
// belongs to the child the ray enters (upper if d_a >= 0, lower if d_a < 0).
constexpr int kOctStack = kMaxOctreeDepth + 1;  // path stack: depths 0..21 (3 path bits per level)
constexpr int kChildCache = 1024;                // first child[] entries kept in shared memory

__shared__ int S_CHILD[kChildCache];

struct OctGrid {
  static constexpr bool kColumns = false;
  static constexpr bool kIndexCells = false;
  static constexpr int kSlots = RT_SLOTS_OCT;
  struct Cell {
    int leaf;
    float lo[3], hi[3];
  };
  // current leaf and its box, its depth, the octants of its path (3 bits per
  // level from the root), entry parameter t; node indices of the path in the
  // lane's shared-memory stack
  struct Walk {
    int leaf, depth;
    float t;
    float lo[3], hi[3];
    unsigned long long path;
  };
  // the lane's ancestor stack: entry l at stack[l kBlock] (dynamic shared
  // memory of P.oct_levels rows; consecutive lanes on consecutive words, so
  // lanes at different levels never meet in a bank)
  struct Scratch {
    int* stack;
    __device__ __forceinline__ int& operator[](int level) const { return stack[level * kBlock]; }
  };

  __device__ static __forceinline__ int child(const FwdParams& P, int node) {
    return node < kChildCache ? S_CHILD[node] : __ldg(&P.child[node]);
  }

  __device__ static __forceinline__ int octant(float3 p, float3 d, float lo[3], float hi[3], bool descend) {
    int oct = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float mid = 0.5f * (lo[a] + hi[a]);
      const float pa = a == 0 ? p.x : (a == 1 ? p.y : p.z);
      const float da = a == 0 ? d.x : (a == 1 ? d.y : d.z);
      const bool upper = da < 0.0f ? (pa > mid) : (pa >= mid);
      if (upper) oct |= 1 << a;
      if (descend) {
        if (upper) lo[a] = mid; else hi[a] = mid;
      }
    }
    return oct;
  }

  // Descend from node stack[depth] (box w.lo/hi) to the leaf containing p.
  __device__ static __forceinline__ bool descend(const FwdParams& P, float3 p, float3 d, Walk& w, Scratch& sc) {
    int node = sc[w.depth];
    while (true) {
      const int c = child(P, node);
      if (c < 0) {
        w.leaf = -c - 1;
        return true;
      }
      if (w.depth + 1 >= P.oct_levels) {
        atomicOr(P.flags, kFlagOctreeDepth);
        w.leaf = 0;
        return false;
      }
      const int oct = octant(p, d, w.lo, w.hi, true);
      w.path |= (unsigned long long)oct << (3 * w.depth);
      node = c + oct;
      w.depth += 1;
      sc[w.depth] = node;
    }
  }

  __device__ static __forceinline__ bool locate_from_root(const FwdParams& P, float3 p, float3 d, Walk& w,
                                                          Scratch& sc) {
#pragma unroll
    for (int a = 0; a < 3; ++a) { w.lo[a] = P.lo[a]; w.hi[a] = P.hi[a]; }
    w.depth = 0;
    w.path = 0ull;
    sc[0] = 0;
    return descend(P, p, d, w, sc);
  }

  // A leaf that holds x, a point inside the grid.
  __device__ static __forceinline__ void locate_cell(const FwdParams& P, float3 x, Cell& c) {
    float lo[3] = {P.lo[0], P.lo[1], P.lo[2]}, hi[3] = {P.hi[0], P.hi[1], P.hi[2]};
    const float3 up = make_float3(1.0f, 1.0f, 1.0f);
    int v = child(P, 0);
    while (v >= 0) v = child(P, v + octant(x, up, lo, hi, true));
    c.leaf = -v - 1;
  }

  __device__ static __forceinline__ bool init(const FwdParams& P, float3 x, float3 d, float3 id, bool known,
                                              const Cell& c, Walk& w, Scratch& sc) {
    w.t = 0.0f;
    if (known) {
      // rebuild the path of the known leaf by descending to its box centre,
      // which lies strictly inside every ancestor's chosen half
      const float3 ctr = make_float3(0.5f * (c.lo[0] + c.hi[0]), 0.5f * (c.lo[1] + c.hi[1]), 0.5f * (c.lo[2] + c.hi[2]));
      if (!locate_from_root(P, ctr, d, w, sc)) return false;
      if (w.leaf != c.leaf) atomicOr(P.flags, kFlagCellRange);
      return true;
    }
    int entry = -1;
    float3 p = x;
    if (!inside_box(P, x)) {
      const float3 ik = make_float3(id.x != 0.0f ? id.x : RT_INF, id.y != 0.0f ? id.y : RT_INF,
                                    id.z != 0.0f ? id.z : RT_INF);
      if (!ray_box_entry(P, x, d, ik, w.t, entry)) return false;
      p = make_float3(fmaf(w.t, d.x, x.x), fmaf(w.t, d.y, x.y), fmaf(w.t, d.z, x.z));
      if (entry == 0) p.x = d.x > 0.0f ? P.lo[0] : P.hi[0];
      if (entry == 1) p.y = d.y > 0.0f ? P.lo[1] : P.hi[1];
      if (entry == 2) p.z = d.z > 0.0f ? P.lo[2] : P.hi[2];
    }
    return locate_from_root(P, p, d, w, sc);
  }

  __device__ static __forceinline__ float exit(const Walk& w, float3 x, float3 id, int& axis) {
    const float tx = id.x != 0.0f ? ((id.x > 0.0f ? w.hi[0] : w.lo[0]) - x.x) * id.x : RT_INF;
    const float ty = id.y != 0.0f ? ((id.y > 0.0f ? w.hi[1] : w.lo[1]) - x.y) * id.y : RT_INF;
    const float tz = id.z != 0.0f ? ((id.z > 0.0f ? w.hi[2] : w.lo[2]) - x.z) * id.z : RT_INF;
    return first_min(tx, ty, tz, axis);
  }

  // Move through face `axis` to the neighbouring leaf at the exit point.  The
  // exit point's other coordinates stay inside the current leaf, so the walk
  // never steps back across a face.  The new leaf is found by replaying the
  // current leaf's path from the root while the exit point stays on it (no
  // loads), then descending with loads below the level where it leaves it.
  __device__ static __forceinline__ bool advance(const FwdParams& P, float3 x, float3 d, float3, int axis, Walk& w,
                                                 Scratch& sc) {
    const float da = pick(axis, d);
    const float plane = da > 0.0f ? (axis == 0 ? w.hi[0] : (axis == 1 ? w.hi[1] : w.hi[2]))
                                  : (axis == 0 ? w.lo[0] : (axis == 1 ? w.lo[1] : w.lo[2]));
    const float dom_lo = axis == 0 ? P.lo[0] : (axis == 1 ? P.lo[1] : P.lo[2]);
    const float dom_hi = axis == 0 ? P.hi[0] : (axis == 1 ? P.hi[1] : P.hi[2]);
    if ((da > 0.0f && plane >= dom_hi) || (da < 0.0f && plane <= dom_lo)) return false;
    float3 p = make_float3(fminf(fmaxf(fmaf(w.t, d.x, x.x), w.lo[0]), w.hi[0]),
                           fminf(fmaxf(fmaf(w.t, d.y, x.y), w.lo[1]), w.hi[1]),
                           fminf(fmaxf(fmaf(w.t, d.z, x.z), w.lo[2]), w.hi[2]));
    if (axis == 0) p.x = plane; else if (axis == 1) p.y = plane; else p.z = plane;
    const int old_depth = w.depth;
    const unsigned long long old_path = w.path;
    float lo[3] = {P.lo[0], P.lo[1], P.lo[2]}, hi[3] = {P.hi[0], P.hi[1], P.hi[2]};
    int depth = 0;
    // When the exit point lies strictly inside the leaf's box in the two other
    // axes, the old path and the new one part at the level where the face
    // plane splits an ancestor: with i the leaf's integer coordinate along
    // `axis` at its depth D, level D - 1 - (trailing ones of i) going up,
    // D - 1 - (trailing zeros of i) going down.  With exact boxes the new path is
    // then followed from there by its bits; otherwise the ancestor's box is
    // rebuilt by halving along the old path (the same arithmetic as the
    // descent) and the exit point descends from it.  When a coordinate lies
    // on a face of the leaf (the tie rule may part the paths earlier) the
    // path is replayed from the root.
    const bool in_x = axis == 0 || (p.x > w.lo[0] && p.x < w.hi[0]);
    const bool in_y = axis == 1 || (p.y > w.lo[1] && p.y < w.hi[1]);
    const bool in_z = axis == 2 || (p.z > w.lo[2] && p.z < w.hi[2]);
    const bool inside = in_x && in_y && in_z;
    if (inside) {
      // the path's bits on `axis`, level l at bit l (Morton compaction of
      // every third bit), then moved so that the leaf's level is bit 31
      unsigned long long m = (old_path >> axis) & 0x1249249249249249ull;
      m = (m ^ (m >> 2)) & 0x10c30c30c30c30c3ull;
      m = (m ^ (m >> 4)) & 0x100f00f00f00f00full;
      m = (m ^ (m >> 8)) & 0x1f0000ff0000ffull;
      m = (m ^ (m >> 16)) & 0x1f00000000ffffull;
      m = (m ^ (m >> 32)) & 0x1fffffull;
      const unsigned top = (unsigned)m << (32 - old_depth);
      // trailing ones (up) / zeros (down) of the leaf's coordinate
      const int tb = da > 0.0f ? __clz(~top) : __clz(top);
      const int part = old_depth - 1 - tb;
      if (P.oct_exact) {
        // exact boxes: below the parting level the new path is the old one
        // with the bit of `axis` flipped (in the other axes the exit point
        // lies strictly inside the leaf, so it keeps the old octants), and it
        // is followed without position tests down to the old depth or to a
        // leaf above it.  The box: the old leaf's, moved across the face, then
        // doubled on the side away from each octant up to the level reached.
        const int flip = 1 << axis;
        int node = sc[part];
        int c = child(P, node);
        unsigned long long path = part > 0 ? (old_path & ((1ull << (3 * part)) - 1ull)) : 0ull;
        depth = part;
        while (c >= 0 && depth < old_depth) {
          const int oct = (int)((old_path >> (3 * depth)) & 7ull) ^ flip;
          path |= (unsigned long long)oct << (3 * depth);
          node = c + oct;
          depth += 1;
          sc[depth] = node;
          c = child(P, node);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          lo[a] = w.lo[a];
          hi[a] = w.hi[a];
          if (a == axis) {
            const float size = hi[a] - lo[a];
            if (da > 0.0f) { lo[a] = hi[a]; hi[a] += size; } else { hi[a] = lo[a]; lo[a] -= size; }
          }
        }
        for (int l = old_depth - 1; l >= depth; --l) {
          const int oct = (int)((old_path >> (3 * l)) & 7ull) ^ flip;
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const float size = hi[a] - lo[a];
            if ((oct >> a) & 1) lo[a] -= size; else hi[a] += size;
          }
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) { w.lo[a] = lo[a]; w.hi[a] = hi[a]; }
        w.depth = depth;
        w.path = path;
        if (c < 0) {
          w.leaf = -c - 1;
          return true;
        }
        // a finer neighbour: on by the exit point below the old depth
        return descend(P, p, d, w, sc);
      } else {
        for (; depth < part; ++depth) {
          const int oct = (int)((old_path >> (3 * depth)) & 7ull);
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const float mid = 0.5f * (lo[a] + hi[a]);
            if ((oct >> a) & 1) lo[a] = mid; else hi[a] = mid;
          }
        }
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) { w.lo[a] = lo[a]; w.hi[a] = hi[a]; }
      w.depth = depth;
      w.path = depth > 0 ? (old_path & ((1ull << (3 * depth)) - 1ull)) : 0ull;
      return descend(P, p, d, w, sc);
    }
    // replay from the root along the old path
    while (depth < old_depth) {
      float l2[3] = {lo[0], lo[1], lo[2]}, h2[3] = {hi[0], hi[1], hi[2]};
      const int oct = octant(p, d, l2, h2, true);
      if (oct != (int)((old_path >> (3 * depth)) & 7ull)) break;
#pragma unroll
      for (int a = 0; a < 3; ++a) { lo[a] = l2[a]; hi[a] = h2[a]; }
      ++depth;
    }
    if (depth == old_depth) {  // the exit point cannot lie in the leaf it leaves
      atomicOr(P.flags, kFlagWalkSteps);
      return false;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) { w.lo[a] = lo[a]; w.hi[a] = hi[a]; }
    w.depth = depth;
    w.path = depth > 0 ? (old_path & ((1ull << (3 * depth)) - 1ull)) : 0ull;
    return descend(P, p, d, w, sc);
  }

  __device__ static __forceinline__ int cell(const Walk& w) { return w.leaf; }

  __device__ static __forceinline__ int id(const FwdParams&, const Walk& w) { return w.leaf; }
  __device__ static __forceinline__ int cell_id(const FwdParams&, const Cell& c) { return c.leaf; }
  __device__ static __forceinline__ int sort_place(const FwdParams& P, const Cell& c) { return __ldg(&P.cell_rank[c.leaf]); }
  // (init only uses the middle of a known leaf's box)
  __device__ static __forceinline__ Cell sorted_cell(const FwdParams& P, unsigned place) {
    const float4 c = __ldg(&P.rank_cell[place]);
    return Cell{__float_as_int(c.w), {c.x, c.y, c.z}, {c.x, c.y, c.z}};
  }

  __device__ static __forceinline__ Cell carried(const Walk& w) {
    Cell c;
    c.leaf = w.leaf;
#pragma unroll
    for (int a = 0; a < 3; ++a) { c.lo[a] = w.lo[a]; c.hi[a] = w.hi[a]; }
    return c;
  }

  __device__ static __forceinline__ void clamp(const FwdParams&, const Cell& c, float3& x) {
    x.x = fminf(fmaxf(x.x, c.lo[0]), c.hi[0]);
    x.y = fminf(fmaxf(x.y, c.lo[1]), c.hi[1]);
    x.z = fminf(fmaxf(x.z, c.lo[2]), c.hi[2]);
  }
};

// ---------------------------------------------------------------- k-d tree grid
// A node halves its box at the midpoint of one axis (Table 1(d): BinTree).
// Device node word: (first child << 2) | split axis for an inner node (the
// lower child first, the upper one next), -(leaf + 1) for a leaf.  A point
// on a splitting plane belongs to the child the ray enters, as in octrees.
// The walk finds the next leaf at the exit point of the current one by a
// descent from the leaf's rope for the face it leaves through (the node
// across that face that covers it: the sibling of the ancestor whose split
// made the face), or from the root when the exit point lies on an edge of
// the leaf (the tie rule may then part the paths higher up).  Both give the
// leaf the root descent gives.  The first kChildCache node words sit in
// shared memory.
constexpr int kMaxBinDepth = 96;

struct BinGrid {
  static constexpr bool kColumns = false;
  static constexpr bool kIndexCells = false;
  static constexpr int kSlots = RT_SLOTS_BIN;
  using Cell = OctGrid::Cell;  // the leaf and its box
  struct Walk {
    int leaf;
    float t;
    float lo[3], hi[3];
  };
  struct Scratch {};

  __device__ static __forceinline__ int word(const FwdParams& P, int node) {
    return node < kChildCache ? S_CHILD[node] : __ldg(&P.child[node]);
  }

  // Descend from the root to the leaf holding p (direction d breaks ties).
  __device__ static __forceinline__ bool locate(const FwdParams& P, float3 p, float3 d, Walk& w) {
    return descend(P, 0, P.lo[0], P.lo[1], P.lo[2], P.hi[0], P.hi[1], P.hi[2], p, d, w);
  }

  // A leaf that holds x, a point inside the grid.
  __device__ static __forceinline__ void locate_cell(const FwdParams& P, float3 x, Cell& c) {
    Walk w;
    locate(P, x, make_float3(1.0f, 1.0f, 1.0f), w);
    c.leaf = w.leaf;
  }

  // Descend from `node` (box lo/hi) to the leaf holding p.
  __device__ static __forceinline__ bool descend(const FwdParams& P, int node, float lx, float ly, float lz, float hx,
                                                 float hy, float hz, float3 p, float3 d, Walk& w) {
    for (int depth = 0; depth <= kMaxBinDepth; ++depth) {
      const int v = word(P, node);
      if (v < 0) {
        w.leaf = -v - 1;
        w.lo[0] = lx; w.lo[1] = ly; w.lo[2] = lz;
        w.hi[0] = hx; w.hi[1] = hy; w.hi[2] = hz;
        return true;
      }
      const int a = v & 3;
      const float la = a == 0 ? lx : (a == 1 ? ly : lz), ha = a == 0 ? hx : (a == 1 ? hy : hz);
      const float pa = a == 0 ? p.x : (a == 1 ? p.y : p.z), da = a == 0 ? d.x : (a == 1 ? d.y : d.z);
      const float mid = 0.5f * (la + ha);
      const bool upper = da < 0.0f ? (pa > mid) : (pa >= mid);
      lx = (a == 0 && upper) ? mid : lx;
      ly = (a == 1 && upper) ? mid : ly;
      lz = (a == 2 && upper) ? mid : lz;
      hx = (a == 0 && !upper) ? mid : hx;
      hy = (a == 1 && !upper) ? mid : hy;
      hz = (a == 2 && !upper) ? mid : hz;
      node = (v >> 2) + (upper ? 1 : 0);
    }
    atomicOr(P.flags, kFlagOctreeDepth);
    w.leaf = 0;
    return false;
  }

  __device__ static __forceinline__ bool init(const FwdParams& P, float3 x, float3 d, float3 id, bool known,
                                              const Cell& c, Walk& w, Scratch&) {
    w.t = 0.0f;
    if (known) {
      // the known leaf: descend to its box centre, strictly inside every
      // ancestor's chosen half
      const float3 ctr = make_float3(0.5f * (c.lo[0] + c.hi[0]), 0.5f * (c.lo[1] + c.hi[1]), 0.5f * (c.lo[2] + c.hi[2]));
      if (!locate(P, ctr, d, w)) return false;
      if (w.leaf != c.leaf) atomicOr(P.flags, kFlagCellRange);
      return true;
    }
    int entry = -1;
    float3 p = x;
    if (!inside_box(P, x)) {
      const float3 ik = make_float3(id.x != 0.0f ? id.x : RT_INF, id.y != 0.0f ? id.y : RT_INF,
                                    id.z != 0.0f ? id.z : RT_INF);
      if (!ray_box_entry(P, x, d, ik, w.t, entry)) return false;
      p = make_float3(fmaf(w.t, d.x, x.x), fmaf(w.t, d.y, x.y), fmaf(w.t, d.z, x.z));
      if (entry == 0) p.x = d.x > 0.0f ? P.lo[0] : P.hi[0];
      if (entry == 1) p.y = d.y > 0.0f ? P.lo[1] : P.hi[1];
      if (entry == 2) p.z = d.z > 0.0f ? P.lo[2] : P.hi[2];
    }
    return locate(P, p, d, w);
  }

  __device__ static __forceinline__ float exit(const Walk& w, float3 x, float3 id, int& axis) {
    const float tx = id.x != 0.0f ? ((id.x > 0.0f ? w.hi[0] : w.lo[0]) - x.x) * id.x : RT_INF;
    const float ty = id.y != 0.0f ? ((id.y > 0.0f ? w.hi[1] : w.lo[1]) - x.y) * id.y : RT_INF;
    const float tz = id.z != 0.0f ? ((id.z > 0.0f ? w.hi[2] : w.lo[2]) - x.z) * id.z : RT_INF;
    return first_min(tx, ty, tz, axis);
  }

  // Into the neighbouring leaf through face `axis`: the exit point with the
  // other coordinates kept inside the current leaf (the walk never steps
  // back across a face), located from the leaf's rope for that face, or from the
  // root when it lies on an edge of the leaf.
  __device__ static __forceinline__ bool advance(const FwdParams& P, float3 x, float3 d, float3, int axis, Walk& w,
                                                 Scratch&) {
    const float da = pick(axis, d);
    const float plane = da > 0.0f ? (axis == 0 ? w.hi[0] : (axis == 1 ? w.hi[1] : w.hi[2]))
                                  : (axis == 0 ? w.lo[0] : (axis == 1 ? w.lo[1] : w.lo[2]));
    const float dom_lo = axis == 0 ? P.lo[0] : (axis == 1 ? P.lo[1] : P.lo[2]);
    const float dom_hi = axis == 0 ? P.hi[0] : (axis == 1 ? P.hi[1] : P.hi[2]);
    if ((da > 0.0f && plane >= dom_hi) || (da < 0.0f && plane <= dom_lo)) return false;
    float3 p = make_float3(fminf(fmaxf(fmaf(w.t, d.x, x.x), w.lo[0]), w.hi[0]),
                           fminf(fmaxf(fmaf(w.t, d.y, x.y), w.lo[1]), w.hi[1]),
                           fminf(fmaxf(fmaf(w.t, d.z, x.z), w.lo[2]), w.hi[2]));
    if (axis == 0) p.x = plane; else if (axis == 1) p.y = plane; else p.z = plane;
    const int old = w.leaf;
    const float t = w.t;
    const bool inside = (axis == 0 || (p.x > w.lo[0] && p.x < w.hi[0])) &&
                        (axis == 1 || (p.y > w.lo[1] && p.y < w.hi[1])) &&
                        (axis == 2 || (p.z > w.lo[2] && p.z < w.hi[2]));
    // the start of the descent (one loop for both starts: lanes of a warp
    // that start differently still descend together)
    int node = 0;
    float4 lo = make_float4(P.lo[0], P.lo[1], P.lo[2], 0.0f), hi = make_float4(P.hi[0], P.hi[1], P.hi[2], 0.0f);
    if (inside) {
      node = __ldg(&P.rope[(size_t)old * 6 + 2 * axis + (da > 0.0f ? 1 : 0)]);
      if (node < 0) return false;
      load_pair(&P.node_box[2 * (size_t)node], lo, hi);  // one load: 38.0 -> 37.4 ms per launch of the clumpy tree
    }
    if (!descend(P, node, lo.x, lo.y, lo.z, hi.x, hi.y, hi.z, p, d, w)) return false;
    w.t = t;
    if (w.leaf == old) {  // the exit point cannot lie in the leaf it leaves
      atomicOr(P.flags, kFlagWalkSteps);
      return false;
    }
    return true;
  }

  __device__ static __forceinline__ int cell(const Walk& w) { return w.leaf; }
  __device__ static __forceinline__ int id(const FwdParams&, const Walk& w) { return w.leaf; }
  __device__ static __forceinline__ int cell_id(const FwdParams&, const Cell& c) { return c.leaf; }
  __device__ static __forceinline__ int sort_place(const FwdParams& P, const Cell& c) { return __ldg(&P.cell_rank[c.leaf]); }
  // (init only uses the middle of a known leaf's box)
  __device__ static __forceinline__ Cell sorted_cell(const FwdParams& P, unsigned place) {
    const float4 c = __ldg(&P.rank_cell[place]);
    return Cell{__float_as_int(c.w), {c.x, c.y, c.z}, {c.x, c.y, c.z}};
  }

  __device__ static __forceinline__ Cell carried(const Walk& w) {
    Cell c;
    c.leaf = w.leaf;
#pragma unroll
    for (int a = 0; a < 3; ++a) { c.lo[a] = w.lo[a]; c.hi[a] = w.hi[a]; }
    return c;
  }

  __device__ static __forceinline__ void clamp(const FwdParams&, const Cell& c, float3& x) {
    x.x = fminf(fmaxf(x.x, c.lo[0]), c.hi[0]);
    x.y = fminf(fmaxf(x.y, c.lo[1]), c.hi[1]);
    x.z = fminf(fmaxf(x.z, c.lo[2]), c.hi[2]);
  }
};

// ---------------------------------------------------------------- Voronoi grid
// Cell c holds the points nearer to site c than to any other site (Table
// 1(d): VoronoiDustGrid; Sect. 2.4).  Its boundary with neighbour j is their
// bisecting plane, kept per face as the unit normal n towards s_j and the
// plane's distance h from s_c.  On entering a cell the walk finds the first
// plane ahead, t_f = (h - (x - s_c) . n) / (d . n) over the faces with
// d . n > 0, or the domain boundary if that comes first (the first minimal
// face wins ties, as in the oracle); a straight line meets each convex cell
// once, so a walk visiting more cells than the grid holds (P.max_walk) is
// stopped and flagged.  A point is located by a greedy descent from the site
// nearest to its bucket's centre: move to the nearest neighbour nearer to
// the point until none is; on a neighbour graph that holds every face inside
// the domain this ends at the nearest site.
struct VorGrid {
  static constexpr bool kColumns = false;
  static constexpr bool kIndexCells = false;
  static constexpr int kSlots = RT_SLOTS_VOR;
  using Cell = OctGrid::Cell;  // the cell id in .leaf (the box is not used)
  struct Walk {
    int leaf;   // current cell
    int next;   // the cell beyond the exit face, -1 for the domain boundary
    float t;    // entry parameter of the current segment
    float te;   // exit parameter
    float t_box;  // where the ray leaves the domain
    int steps;  // cells entered after the first
  };
  struct Scratch {};

  __device__ static __forceinline__ float dist2(float3 p, float4 s) {
    const float dx = p.x - s.x, dy = p.y - s.y, dz = p.z - s.z;
    return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
  }

  __device__ static __forceinline__ int locate(const FwdParams& P, float3 p) {
    const int bx = min(max(__float2int_rd((p.x - P.lo[0]) * P.vb_inv[0]), 0), P.vb_n[0] - 1);
    const int by = min(max(__float2int_rd((p.y - P.lo[1]) * P.vb_inv[1]), 0), P.vb_n[1] - 1);
    const int bz = min(max(__float2int_rd((p.z - P.lo[2]) * P.vb_inv[2]), 0), P.vb_n[2] - 1);
    int c = __ldg(&P.bucket_seed[bx + P.vb_n[0] * (by + P.vb_n[1] * bz)]);
    for (int it = 0; it < P.max_walk; ++it) {
      float best = dist2(p, __ldg(&P.site[c]));
      int move = -1;
      const unsigned f1 = 2u * __ldg(&P.face_off[c + 1]);
      // three neighbours at once (past the last face, and in place of a padded
      // one, the cell itself, never nearer than itself)
      for (unsigned f = 2u * __ldg(&P.face_off[c]); f < f1; f += 3) {
        int j[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) j[k] = f + k < f1 ? __ldg(&P.child[f + k]) : c;
        float4 sj[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) sj[k] = __ldg(&P.site[j[k]]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float dj = dist2(p, sj[k]);
          if (dj < best) { best = dj; move = j[k]; }
        }
      }
      if (move < 0) return c;
      c = move;
    }
    atomicOr(P.flags, kFlagWalkSteps);
    return c;
  }

  __device__ static __forceinline__ void locate_cell(const FwdParams& P, float3 x, Cell& c) { c.leaf = locate(P, x); }

  // Pairs of face planes in flight per lane.  The walk waits on the planes'
  // loads and on the L1 wavefronts they take (lanes in different cells: one per
  // lane and load), so two planes come with one 32-byte load, and two pairs at
  // once: 25.5 + 12.2 ms (sorted walks + transport, Voronoi disk, 1.5e6 packets)
  // with three 16-byte loads in flight, 29.1 + 15.3 with one pair, 23.8 + 11.3
  // with two.
  static constexpr int kPairs = 2;

  // The exit of the current cell along x + t d: parameter and next cell.
  __device__ static __forceinline__ void find_exit(const FwdParams& P, float3 x, float3 d, Walk& w) {
    const float4 s = __ldg(&P.site[w.leaf]);
    const float rx = x.x - s.x, ry = x.y - s.y, rz = x.z - s.z;
    float best = w.t_box;
    constexpr unsigned kNoFace = 0xffffffffu;
    unsigned face = kNoFace;
    const unsigned p1 = __ldg(&P.face_off[w.leaf + 1]);
    for (unsigned p = __ldg(&P.face_off[w.leaf]); p < p1; p += kPairs) {
      float4 n[2 * kPairs];
#pragma unroll
      for (int k = 0; k < kPairs; ++k) {
        if (k == 0 || p + k < p1) load_pair(&P.face[2 * (size_t)(p + k)], n[2 * k], n[2 * k + 1]);
        else n[2 * k] = n[2 * k + 1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      }
#pragma unroll
      for (int k = 0; k < 2 * kPairs; ++k) {
        const float den = fmaf(d.x, n[k].x, fmaf(d.y, n[k].y, d.z * n[k].z));
        if (den > 0.0f) {
          const float tf = (n[k].w - fmaf(rx, n[k].x, fmaf(ry, n[k].y, rz * n[k].z))) / den;
          if (tf < best) { best = tf; face = 2u * p + (unsigned)k; }
        }
      }
    }
    w.te = best;
    w.next = face != kNoFace ? __ldg(&P.child[face]) : -1;
  }

  __device__ static __forceinline__ bool init(const FwdParams& P, float3 x, float3 d, float3 id, bool known,
                                              const Cell& c, Walk& w, Scratch&) {
    w.t = 0.0f;
    w.steps = 0;
    const float tx = id.x != 0.0f ? ((id.x > 0.0f ? P.hi[0] : P.lo[0]) - x.x) * id.x : RT_INF;
    const float ty = id.y != 0.0f ? ((id.y > 0.0f ? P.hi[1] : P.lo[1]) - x.y) * id.y : RT_INF;
    const float tz = id.z != 0.0f ? ((id.z > 0.0f ? P.hi[2] : P.lo[2]) - x.z) * id.z : RT_INF;
    w.t_box = fminf(tx, fminf(ty, tz));
    if (known) {
      w.leaf = c.leaf;
    } else {
      int entry = -1;
      float3 p = x;
      if (!inside_box(P, x)) {
        const float3 ik = make_float3(id.x != 0.0f ? id.x : RT_INF, id.y != 0.0f ? id.y : RT_INF,
                                      id.z != 0.0f ? id.z : RT_INF);
        if (!ray_box_entry(P, x, d, ik, w.t, entry)) return false;
        p = make_float3(fmaf(w.t, d.x, x.x), fmaf(w.t, d.y, x.y), fmaf(w.t, d.z, x.z));
        if (entry == 0) p.x = d.x > 0.0f ? P.lo[0] : P.hi[0];
        if (entry == 1) p.y = d.y > 0.0f ? P.lo[1] : P.hi[1];
        if (entry == 2) p.z = d.z > 0.0f ? P.lo[2] : P.hi[2];
      }
      w.leaf = locate(P, p);
    }
    find_exit(P, x, d, w);
    return true;
  }

  __device__ static __forceinline__ float exit(const Walk& w, float3, float3, int& axis) {
    axis = 0;
    return w.te;
  }

  __device__ static __forceinline__ bool advance(const FwdParams& P, float3 x, float3 d, float3, int, Walk& w,
                                                 Scratch&) {
    if (w.next < 0) return false;
    if (++w.steps > P.max_walk) {
      atomicOr(P.flags, kFlagWalkSteps);
      return false;
    }
    w.leaf = w.next;
    find_exit(P, x, d, w);
    return true;
  }

  __device__ static __forceinline__ int cell(const Walk& w) { return w.leaf; }
  __device__ static __forceinline__ int id(const FwdParams&, const Walk& w) { return w.leaf; }
  __device__ static __forceinline__ int cell_id(const FwdParams&, const Cell& c) { return c.leaf; }
  __device__ static __forceinline__ int sort_place(const FwdParams& P, const Cell& c) { return __ldg(&P.cell_rank[c.leaf]); }
  // (init only uses the cell's id)
  __device__ static __forceinline__ Cell sorted_cell(const FwdParams& P, unsigned place) {
    const float4 c = __ldg(&P.rank_cell[place]);
    return Cell{__float_as_int(c.w), {c.x, c.y, c.z}, {c.x, c.y, c.z}};
  }

  __device__ static __forceinline__ Cell carried(const Walk& w) {
    Cell c;
    c.leaf = w.leaf;
    return c;
  }

  // A Voronoi cell is no box: the position is kept inside the domain only (a
  // walk from a point a rounding error outside its cell takes a zero-length
  // segment there).
  __device__ static __forceinline__ void clamp(const FwdParams& P, const Cell&, float3& x) {
    x.x = fminf(fmaxf(x.x, P.lo[0]), P.hi[0]);
    x.y = fminf(fmaxf(x.y, P.lo[1]), P.hi[1]);
    x.z = fminf(fmaxf(x.z, P.lo[2]), P.hi[2]);
  }
};

// ---------------------------------------------------------------- packet slots
// A warp carries more packets than it has lanes: G::kSlots slots of shared
// memory per warp (structure of arrays) hold the packets' state between
// walks, a lane holds in registers only the walk it is on.  A packet is either
// walked by a lane or waits in one of the warp's queues: for a lane (kQReady)
// or for per-event work of one kind (kQPath1: its first walk ended; kQEvent:
// its second walk or a peel-off walk ended; kQFetch: the slot is free and
// takes a new packet).  Lanes whose walk ended are given the next ready packet,
// so walking lanes stay near the full warp, and per-event work runs as rounds
// over up to 32 packets that all need the same work.
enum Queue : int { kQPath1 = 0, kQEvent = 1, kQFetch = 2, kQReady = 3, kQueues = 4 };
constexpr int kWarps = kBlock / 32;
constexpr int kRing = 64;  // entries of a queue's ring buffer; slots per warp are at most this

// Counts of one warp, kept by its first lane.
struct WarpTally {
  unsigned long long crossings, path_crossings, column_crossings;
  unsigned long long events, peeloffs, packets, column_peels;
};

// Luminosity tallies of one lane, in its local memory.
struct LaneTally {
  double escaped, absorbed, truncated;
};

template <class G, bool kTape>
struct Shared {
  static constexpr int kN = kWarps * G::kSlots;
  unsigned long long pid[kN];   // packet id
  double L[kN];                 // weight
  float2 hg[kN];                // the event's Henyey-Greenstein uniforms
  // what a walk starts with (path 1: the deposit weight, path 2: tau* as a
  // pair) and what it ended with (the optical depth pair; path 2: s*)
  float2 res[kN];
  float3 x[kN], k[kN];          // position, direction of travel
  typename G::Cell cell[kN];    // the cell of x (valid with the has-cell bit)
  int event[kN];                // event index
  unsigned pack[kN];            // see Pack
  float3 g[kTape ? kN : 1];     // tape: plane sums of the first walk
  WarpTally tally[kWarps];
  LaneTally lum[kWarps];        // the warps' luminosity tallies, at the end
  uint2 queues[kWarps];         // each warp's queue counts and heads (see Queues)
  unsigned char ring[kWarps][kQueues][kRing];
};

// The small fields of a slot in one word: phase (4 bits), wavelength (6),
// instrument of the next peel-off (5), has-cell (1), exponent of the deposit
// weight or the deferred peel-offs (16).
struct Pack {
  __device__ static __forceinline__ unsigned make(int phase, int lam, int q, bool has_cell, int e) {
    return (unsigned)phase | ((unsigned)lam << 4) | ((unsigned)q << 10) | (has_cell ? 1u << 15 : 0u) |
           ((unsigned)e << 16);
  }
  __device__ static __forceinline__ int phase(unsigned p) { return (int)(p & 15u); }
  __device__ static __forceinline__ int lam(unsigned p) { return (int)((p >> 4) & 63u); }
  __device__ static __forceinline__ int q(unsigned p) { return (int)((p >> 10) & 31u); }
  __device__ static __forceinline__ bool has_cell(unsigned p) { return (p >> 15) & 1u; }
  __device__ static __forceinline__ int exponent(unsigned p) { return (int)p >> 16; }
};

// the kernel's Shared (and, for octrees, the ancestor stacks behind it)
extern __shared__ __align__(16) unsigned char S_RAW[];
template <class G, bool kTape>
__device__ __forceinline__ Shared<G, kTape>& shared_state() {
  return *reinterpret_cast<Shared<G, kTape>*>(S_RAW);
}

// The walk a lane is on.
template <class G>
struct Walker {
  int slot;             // the packet's slot (index in the block's arrays), -1: none
  int phase;            // kPath1, kPath2, kPeelEmit or kPeelScat
  double* absorption;   // the tallies of this wavelength
  bool walking;
  float kappa;          // extinction per unit density at this wavelength
  float3 x;             // start of the walk
  float3 d, id;         // its direction and inverse
  typename G::Walk w;   // its current cell and exit data
  float rho;            // density of the current cell (loaded one crossing ahead)
  float th, tl;         // optical depth so far (pair sum)
  unsigned n;           // crossings so far
  // path 1: the deposit weight (1 - albedo) L as aux0 2^e: aux0 the FP32
  // weight (e = 0) while that lies in [1e-30, 1e30], with aux1 = 64, the
  // optical depth below which a deposit takes the plain FP32 product; else
  // aux0 in [1/2, 1) and e in the slot's word, aux1 = -1 (every deposit carries the
  // exponent), so that deposits keep FP64's range whatever the weight;
  // path 2: tau* as a float pair, then s*
  float aux0, aux1;
  // adjoint tape (launches that record one): plane sums of the walk, entry
  // axis of its segment, the interaction's crossing index, kappa rho and
  // remainder
  float3 g;
  int axis_in, h;
  float kr_h, rem;
};

// A packet in per-event work: its slot and the fields in registers.
template <class G, bool kTape>
struct Task {
  Shared<G, kTape>& sh;
  LaneTally& tally;
  int i;             // slot
  int phase, wphase; // kStart: the walk to start
  int lam, q, event;
  bool has_cell;
  int dep_exp;       // exponent of the deposit weight; peel-off walks: `deferred`
  unsigned deferred; // instruments whose peel-off of this event is a record of the sorted pass
  int place;         // of the position's cell in the sorted pass's order, once asked for (else -1)
  float th, tl;      // optical depth of the walk that ended (path 2: th = s*)
  unsigned n_peel, n_col, c_col;  // peel-offs, of which by column sums, and their crossings
  __device__ __forceinline__ unsigned long long& pid() const { return sh.pid[i]; }
  __device__ __forceinline__ double& L() const { return sh.L[i]; }
  __device__ __forceinline__ float3& x() const { return sh.x[i]; }
  __device__ __forceinline__ float3& k() const { return sh.k[i]; }
  __device__ __forceinline__ float2& hg() const { return sh.hg[i]; }
  __device__ __forceinline__ float2& res() const { return sh.res[i]; }
  __device__ __forceinline__ typename G::Cell& cell() const { return sh.cell[i]; }
};

template <class G, bool kTape>
__device__ __forceinline__ void trace_row(const FwdParams& P, const Task<G, kTape>& s, int event, int cell, double L,
                                          double tau_path, double tau_star) {
  if (!P.trace || s.pid() != P.trace_packet || s.lam != P.trace_lambda || event >= P.trace_cap) return;
  rt_trace_row r;
  const float3 x = s.x(), k = s.k();
  r.event = event; r.reserved = 0; r.cell = cell;
  r.x[0] = x.x; r.x[1] = x.y; r.x[2] = x.z;
  r.k[0] = k.x; r.k[1] = k.y; r.k[2] = k.z;
  r.L = L; r.tau_path = tau_path; r.tau_star = tau_star;
  P.trace[event] = r;
}

__device__ __forceinline__ float3 instr_dir(const DevInstr& I) { return make_float3(I.kobs[0], I.kobs[1], I.kobs[2]); }

// A peel-off along a frame that looks exactly along grid axis I.axis: the
// optical depth to the boundary is kappa (rho_c ds_0 + column[c]), with ds_0
// the distance to the face of the current cell that the ray leaves (the first
// segment of the walk) and column[c] the density integral of the cells beyond
// it on the same grid line.  The walk's crossings (n_cross) are counted all
// the same.  known: x lies in cell cc.  False when the position is outside the
// grid (the walk then finds the entry).
template <class G>
__device__ __forceinline__ bool column_tau(const FwdParams& P, float3 x, bool known, const CartGrid::Cell& cc,
                                           const DevInstr& I, float kappa, float& th,
                                           unsigned long long& n_cross) {
  CartGrid::Cell c;
  if (known) {
    c = cc;
  } else {
    if (!inside_box(P, x)) return false;
    G::locate_cell(P, x, c);
  }
  const int a = I.axis;
  const bool up = I.dir > 0;
  const int i = a == 0 ? c.ix : (a == 1 ? c.iy : c.iz);
  const int n = a == 0 ? P.nx : (a == 1 ? P.ny : P.nz);
  const float xa = a == 0 ? x.x : (a == 1 ? x.y : x.z);
  const float plane = G::plane(P, a, i + (up ? 1 : 0));
  const float ds0 = fmaxf(up ? plane - xa : xa - plane, 0.0f);
  const int cell = c.ix + P.nx * (c.iy + P.ny * c.iz);  // row-major: the column sums
  const int slot = c.ix * P.stride[0] + c.iy * P.stride[1] + c.iz * P.stride[2];
  th = kappa * fmaf(load_density(&P.density[slot]), ds0, __ldg(&I.column[cell]));
  n_cross = (unsigned long long)(up ? n - i : i + 1);
  return true;
}

template <class G, bool kTape>
__device__ __forceinline__ bool column_peel(const FwdParams& P, Task<G, kTape>& s, const DevInstr& I) {
  unsigned long long nc;
  if (!column_tau<G>(P, s.x(), s.has_cell, s.cell(), I, P.lam[s.lam].kappa, s.th, nc)) return false;
  s.tl = 0.0f;
  s.c_col += (unsigned)nc;
  s.n_col += 1u;
  return true;
}

// A peel-off ray of the sorted pass: the optical depth th + tl from x along d
// (FP32 pair sum, the transport kernel's walk arithmetic).
template <class G>
struct Ray {
  float3 x, d, id;
  typename G::Walk w;
  float kappa, rho, th, tl;
};

// Start the ray at x, which lies in cell cc if known; false if it misses the grid.
template <class G>
__device__ __forceinline__ bool ray_start(const FwdParams& P, Ray<G>& r, bool known, const typename G::Cell& cc,
                                          typename G::Scratch& sc) {
  r.id = make_float3(inv_or_zero(r.d.x), inv_or_zero(r.d.y), inv_or_zero(r.d.z));
  r.th = 0.0f;
  r.tl = 0.0f;
  if (!G::init(P, r.x, r.d, r.id, known, cc, r.w, sc)) return false;
  r.rho = load_density(&P.density[G::cell(r.w)]);
  return true;
}

// One cell crossing; false when the ray leaves the grid.
template <class G>
__device__ __forceinline__ bool ray_step(const FwdParams& P, Ray<G>& r, typename G::Scratch& sc) {
  int axis;
  const float te = G::exit(r.w, r.x, r.id, axis);
  const float texit = fmaxf(te, r.w.t);
  const float ds = texit - r.w.t;
  const float kr = r.kappa * r.rho;
  const float dt = kr * ds;
  float nh, e;
  two_sum(r.th, dt, nh, e);
  r.tl = r.tl + e;
  r.th = nh;
  r.w.t = texit;
  if (!G::advance(P, r.x, r.d, r.id, axis, r.w, sc)) return false;
  r.rho = load_density(&P.density[G::cell(r.w)]);
  return true;
}

// Phase-function value of a scattering peel-off towards instrument I.
__device__ __forceinline__ float peel_phase(const FwdParams& P, int lam, float3 k, const DevInstr& I) {
  return hg_phase(P.lam[lam].g, k.x * I.kobs[0] + k.y * I.kobs[1] + k.z * I.kobs[2]);
}

// Deposit a finished peel-off from x (weight L, phase-function value phase,
// optical depth th + tl) into instrument q's image(s); pid and event only
// label debug records.
__device__ __forceinline__ void deposit_peel(const FwdParams& P, int q, int lam, float3 x, double L, float phase,
                                             float th, float tl, bool scattered, unsigned long long pid, int event) {
  const DevInstr& I = P.instr[q];
  // exp(-(th + tl)) with the walk's compensated optical depth: the low word
  // enters as the first-order factor (1 - tl)
  const float tau = th;
  const double value = tau < 80.0f ? L * widen(kInv4PiF * phase * expf(-tau) * (1.0f - tl))
                                   : L * kInv4PiD * (double)phase * exp(-((double)tau + (double)tl));
  const int ch = scattered ? 2 : 1;
  if (I.sed) {
    // an SED instrument has one bin per wavelength and channel: the lanes of
    // the warp that deposit into the same bin add their values first and one of
    // them issues the atomics; consecutive lanes (nearly always the case) by
    // halving steps, 5 FP64 additions instead of up to 31
    const unsigned act = __activemask();
    const unsigned key = ((unsigned)q << 20) | ((unsigned)lam << 1) | (scattered ? 1u : 0u);
    const unsigned grp = __match_any_sync(act, key);
    const int first = __ffs(grp) - 1, last = 31 - __clz(grp), lane = (int)(threadIdx.x & 31u);
    double sum = value;
    if (__popc(grp) == last - first + 1) {
      for (int o = 16; o > 0; o >>= 1) {
        if (o > last - first) continue;  // the same for the whole group
        const double v = __shfl_sync(grp, sum, min(lane + o, last));
        if (lane + o <= last) sum += v;
      }
    } else {
      sum = 0.0;
      for (unsigned m = grp; m; m &= m - 1u) sum += __shfl_sync(grp, value, __ffs(m) - 1);
    }
    if (lane == first) {
      atomicAdd(&I.image[lam], sum);
      if (I.channels == 3) atomicAdd(&I.image[(size_t)ch * P.n_lambda + lam], sum);
    }
    if (P.records && (P.record_stride <= 1 || pid % P.record_stride == 0)) {
      const unsigned long long slot = atomicAdd(&P.counters[4], 1ull);
      if ((long long)slot < P.records_cap) {
        rt_record r;
        r.packet = pid; r.lambda = lam; r.event = scattered ? event : 0; r.instrument = q;
        r.reserved = 0; r.pixel = 0; r.value = value;
        P.records[slot] = r;
      }
    }
    return;
  }
  const float fx = (x.x * I.ex[0] + x.y * I.ex[1] + x.z * I.ex[2] + I.off_x) * I.sx;
  const float fy = (x.x * I.ey[0] + x.y * I.ey[1] + x.z * I.ey[2] + I.off_y) * I.sy;
  const size_t plane = (size_t)I.ny * I.nx;
  if (!I.bilinear) {
    const float fix = floorf(fx), fiy = floorf(fy);
    if (!(fix >= 0.0f && fiy >= 0.0f && fix < (float)I.nx && fiy < (float)I.ny)) return;
    const size_t pix = (size_t)(int)fiy * I.nx + (int)fix;
    atomicAdd(&I.image[(size_t)lam * plane + pix], value);
    if (I.channels == 3) atomicAdd(&I.image[((size_t)ch * P.n_lambda + lam) * plane + pix], value);
    if (P.records && (P.record_stride <= 1 || pid % P.record_stride == 0)) {
      const unsigned long long slot = atomicAdd(&P.counters[4], 1ull);
      if ((long long)slot < P.records_cap) {
        rt_record r;
        r.packet = pid; r.lambda = lam; r.event = scattered ? event : 0; r.instrument = q;
        r.reserved = 0; r.pixel = (int64_t)pix; r.value = value;
        P.records[slot] = r;
      }
    }
  } else {
    const float gx = fx - 0.5f, gy = fy - 0.5f;
    const float x0 = floorf(gx), y0 = floorf(gy);
    const float tx = gx - x0, ty = gy - y0;
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
#pragma unroll
      for (int dx = 0; dx < 2; ++dx) {
        const float fix = x0 + dx, fiy = y0 + dy;
        if (!(fix >= 0.0f && fiy >= 0.0f && fix < (float)I.nx && fiy < (float)I.ny)) continue;
        const double v = value * widen((dx ? tx : 1.0f - tx) * (dy ? ty : 1.0f - ty));
        const size_t pix = (size_t)(int)fiy * I.nx + (int)fix;
        atomicAdd(&I.image[(size_t)lam * plane + pix], v);
        if (I.channels == 3) atomicAdd(&I.image[((size_t)ch * P.n_lambda + lam) * plane + pix], v);
      }
    }
  }
}

template <class G, bool kTape>
__device__ __forceinline__ void peel_deposit(const FwdParams& P, const Task<G, kTape>& s, int q, bool scattered) {
  const float phase = scattered ? peel_phase(P, s.lam, s.k(), P.instr[q]) : 1.0f;
  deposit_peel(P, q, s.lam, s.x(), s.L(), phase, s.th, s.tl, scattered, s.pid(), s.event);
}

// Hand the peel-off towards instrument q from x to the sorted pass: a
// record in the next free slot (one atomic per group of lanes), counted under
// its sort key.  place: of x's cell in the sort order; known: the walk starts
// in that cell (else it locates x).  False when the buffer is full (the caller
// then walks it itself).
__device__ __forceinline__ bool defer_record(const FwdParams& P, int q, int lam, float3 x, double L, float phase,
                                             bool known, unsigned place, bool emission, unsigned long long pid,
                                             int event) {
  const unsigned m = __activemask();
  const unsigned lane = threadIdx.x & 31u;
  const int leader = __ffs(m) - 1;
  unsigned long long base = 0;
  if ((int)lane == leader) base = atomicAdd(P.peel_count, (unsigned long long)__popc(m));
  base = __shfl_sync(m, base, leader);
  const unsigned long long slot = base + __popc(m & ((1u << lane) - 1u));
  if (slot >= P.peel_cap) return false;
  const unsigned key = (unsigned)q * (unsigned)(P.n_cells + 1) + place;
  const unsigned meta = (unsigned)lam | (emission ? 0u : 1u << 30) | (known ? 1u << 31 : 0u);
  const long long Lb = __double_as_longlong(L);
  float4* r = reinterpret_cast<float4*>(&P.peel[slot]);
  r[0] = make_float4(x.x, x.y, x.z, __uint_as_float(key));
  r[1] = make_float4(__int_as_float((int)(unsigned)Lb), __int_as_float((int)(Lb >> 32)), phase, __uint_as_float(meta));
  if (P.peel_tag) P.peel_tag[slot] = make_ulonglong2(pid, (unsigned long long)event);
  atomicAdd(&P.peel_hist[key], 1u);
  return true;
}

template <class G, bool kTape>
__device__ __forceinline__ bool defer_peel(const FwdParams& P, Task<G, kTape>& s, int q, bool emission) {
  const float phase = emission ? 1.0f : peel_phase(P, s.lam, s.k(), P.instr[q]);
  if (s.place < 0) {  // once per event: the same for every instrument
    s.place = (int)P.n_cells;
    if (s.has_cell) {
      s.place = G::sort_place(P, s.cell());
    } else if (inside_box(P, s.x())) {
      typename G::Cell c;
      G::locate_cell(P, s.x(), c);
      s.place = G::sort_place(P, c);
    }
  }
  return defer_record(P, q, s.lam, s.x(), s.L(), phase, s.has_cell, (unsigned)s.place, emission, s.pid(), s.event);
}

// Emission (Sect. 3.4): source component by luminosity (FP64 comparison of
// the uniform with the cumulative fractions), position from its geometry and
// an isotropic direction (FP32).
__device__ __forceinline__ void emit(const FwdParams& P, unsigned long long pid, int lam, float3& x_out, float3& k_out) {
  const uint4 r0 = draw_block(pid, lam, 0, 0, P.seed, P.model);
  const uint4 r1 = draw_block(pid, lam, 0, 1, P.seed, P.model);
  int src = P.n_sources - 1;
  if (P.n_sources > 1) {
    const double u0 = u01(r0.x);
    for (int i = 0; i < P.n_sources; ++i) {
      if (u0 < P.src_cum[lam * P.n_sources + i]) { src = i; break; }
    }
  }
  const DevSource& S = P.src[src];
  float3 x = make_float3((float)S.center[0], (float)S.center[1], (float)S.center[2]);
  if (S.kind == RT_SOURCE_EXPDISK) {
    // R has density R exp(-R/hR): minus hR times the log of two uniforms
    const float R = -(float)S.scale_r * (logf(u01f(r0.y)) + logf(u01f(r0.z)));
    float sp, cp;
    sincospif(2.0f * u01f(r0.w), &sp, &cp);
    float z = -(float)S.scale_z * logf(u01f(r1.x));
    if (r1.y < 0x80000000u) z = -z;  // u5 < 1/2
    x.x += R * cp; x.y += R * sp; x.z += z;
  } else if (S.kind == RT_SOURCE_PLUMMER) {
    // enclosed mass fraction m = r^3 / (r^2 + a^2)^(3/2): r = a / sqrt(m^(-2/3) - 1)
    const float m = u01f(r0.y);
    const float r = (float)S.scale_r / sqrtf(expm1f(-(2.0f / 3.0f) * logf(m)));
    const float ct = u01f_signed(r0.z), st = sqrtf(fmaxf(0.0f, 1.0f - ct * ct));
    float sp, cp;
    sincospif(2.0f * u01f(r0.w), &sp, &cp);
    x.x += r * st * cp; x.y += r * st * sp; x.z += r * ct;
  }
  x_out = x;
  const float mu = u01f_signed(r1.z);
  const float st = sqrtf(fmaxf(0.0f, 1.0f - mu * mu));
  float sp, cp;
  sincospif(2.0f * u01f(r1.w), &sp, &cp);
  k_out = make_float3(st * cp, st * sp, mu);
}

// Emission by the dust (panchromatic mode): the cell with probability
// proportional to its thermal luminosity at this wavelength (the first cell
// whose running sum exceeds u times the total, FP64), a uniform position in
// it (FP32, kept inside its planes), an isotropic direction; the cell is
// known to the first walks.
template <class G>
__device__ __forceinline__ void emit_dust(const FwdParams& P, unsigned long long pid, int lam, float3& x_out,
                                          float3& k_out, typename G::Cell& cell) {
  if constexpr (G::kIndexCells) {
    const uint4 r0 = draw_block(pid, lam, 0, 0, P.seed, P.model);
    const uint4 r1 = draw_block(pid, lam, 0, 1, P.seed, P.model);
    const double* cum = P.dust_cum + (size_t)lam * P.n_cells;
    const double target = u01(r0.x) * cum[P.n_cells - 1];
    long long lo = 0, hi = P.n_cells - 1;
    while (lo < hi) {
      const long long mid = (lo + hi) >> 1;
      if (cum[mid] > target) hi = mid; else lo = mid + 1;
    }
    const int c = (int)lo;
    cell.ix = c % P.nx;
    cell.iy = (c / P.nx) % P.ny;
    cell.iz = c / (P.nx * P.ny);
    const int idx[3] = {cell.ix, cell.iy, cell.iz};
    const float u[3] = {u01f(r0.y), u01f(r0.z), u01f(r0.w)};
    float p[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float lo_a = G::plane(P, a, idx[a]), hi_a = G::plane(P, a, idx[a] + 1);
      p[a] = fminf(fmaxf(fmaf(u[a], hi_a - lo_a, lo_a), lo_a), hi_a);
    }
    x_out = make_float3(p[0], p[1], p[2]);
    const float mu = u01f_signed(r1.z);
    const float st = sqrtf(fmaxf(0.0f, 1.0f - mu * mu));
    float sp, cp;
    sincospif(2.0f * u01f(r1.w), &sp, &cp);
    k_out = make_float3(st * cp, st * sp, mu);
  }
}

// Ask for walk `phase` (towards instrument s.q for a peel-off, else along the
// direction of travel); a lane starts it when it is free.
template <class G, bool kTape>
__device__ __forceinline__ void request_walk(Task<G, kTape>& s, int phase) {
  s.wphase = phase;
  s.phase = kStart;
}

// The forced path of event s.event: its first walk carries the deposit
// weight (1 - albedo) L.
template <class G, bool kTape>
__device__ __forceinline__ void request_path(const FwdParams& P, Task<G, kTape>& s) {
  const double wdep = P.lam[s.lam].one_minus_albedo * s.L();
  // integer comparisons: positive doubles order like their bit patterns
  const bool plain = bits_of(wdep) >= bits_of(1e-30) && bits_of(wdep) <= bits_of(1e30);
  int e = 0;
  const float a = plain ? cut(wdep) : split_exp(wdep, e);
  s.res() = make_float2(a, plain ? 64.0f : -1.0f);
  s.dep_exp = e;
  request_walk(s, kPath1);
}

// ---- the stages of a control round (each for the packets in that phase)

// ---- the adjoint tape (cartesian grids; records as the adjoint's replay writes them)

// v 2^-e as FP32 (e: the unit exponent), by cutting the significand.
__device__ __forceinline__ float tape_units(double v, int e) {
  const long long b = __double_as_longlong(v);
  const int be = (int)((b >> 52) & 0x7ff);
  const int fe = be - 896 - e;
  if (be == 0x7ff || fe >= 255) return (float)ldexp(v, -e);
  if (be == 0 || fe <= 0) return 0.0f;
  const unsigned top = (unsigned)((unsigned long long)b >> 32);
  return __uint_as_float((top & 0x80000000u) | ((unsigned)fe << 23) | ((unsigned)(b >> 29) & 0x7fffffu));
}

// The unit exponent of weights: L0 = m 2^e, m in [1/2, 1).
__device__ __forceinline__ int tape_exponent(const FwdParams& P, int lam) {
  const int be = (int)((__double_as_longlong(P.L0[lam]) >> 52) & 0x7ff);
  return be == 0 ? 0 : be - 1022;
}

// The packet's records on the tape.
__device__ __forceinline__ AdjRecord* tape_records(const FwdParams& P, int lam, unsigned long long pid) {
  return P.tape + (size_t)((unsigned long long)lam * P.n_per_lambda + (pid - P.first_id)) * (size_t)P.tape_stride;
}

template <class G, bool kTape>
__device__ __forceinline__ int tape_cell(const FwdParams& P, const Task<G, kTape>& s) {
  if constexpr (G::kColumns) {
    return s.has_cell ? s.cell().ix + P.nx * (s.cell().iy + P.ny * s.cell().iz) : -1;
  } else {
    return -1;
  }
}

// The packet ends after event J: record 0 holds J and the last position.
template <class G, bool kTape>
__device__ __forceinline__ void tape_end(const FwdParams& P, const Task<G, kTape>& s, int J) {
  AdjRecord& r = tape_records(P, s.lam, s.pid())[0];
  const float3 x = s.x();
  r.h = J;
  r.x[0] = x.x; r.x[1] = x.y; r.x[2] = x.z;
  r.cell = tape_cell(P, s);
  r.L = tape_units(s.L(), tape_exponent(P, s.lam));
}

// A new packet (index w of the launch): wavelength, weight, emission.
template <class G, bool kTape>
__device__ __forceinline__ void fetch(const FwdParams& P, Task<G, kTape>& s, unsigned long long w) {
  if (w >= P.n_total) { s.phase = kExit; return; }
  int lam = min((int)(__ull2float_rz(w) * P.inv_n_per_lambda), P.n_lambda - 1);
  while (lam > 0 && (unsigned long long)lam * P.n_per_lambda > w) --lam;
  while (lam + 1 < P.n_lambda && (unsigned long long)(lam + 1) * P.n_per_lambda <= w) ++lam;
  s.lam = lam;
  const unsigned long long pid = P.first_id + (w - (unsigned long long)lam * P.n_per_lambda);
  s.pid() = pid;
  const double L0 = P.L0[lam];
  if (L0 == 0.0) {  // no emission at this wavelength (dust that emits nothing here)
    s.phase = kFetch;
    return;
  }
  s.L() = L0;
  s.event = 0;
  s.has_cell = false;
  float3 x, k;
  if constexpr (G::kIndexCells) {
    if (P.dust_cum) {
      emit_dust<G>(P, pid, lam, x, k, s.cell());
      s.has_cell = true;
    } else {
      emit(P, pid, lam, x, k);
    }
  } else {
    emit(P, pid, lam, x, k);
  }
  s.x() = x;
  s.k() = k;
  trace_row(P, s, 0, -1, L0, 0.0, 0.0);
  s.q = 0;
  s.phase = kPeelScan;
}

// Path 1 ended: escape, or the deposit bookkeeping and the forced-scattering
// inversion (FP64); then the second walk.
template <class G, bool kTape>
__device__ __forceinline__ void finish_path1(const FwdParams& P, Task<G, kTape>& s) {
  const double tau = widen(s.th) + widen(s.tl);
  if (!(tau > 0.0)) {
    trace_row(P, s, s.event, -1, s.L(), 0.0, 0.0);
    s.tally.escaped += s.L();
    if (kTape) tape_end(P, s, s.event - 1);
    s.phase = kFetch;
    return;
  }
  const double one_minus_E = one_minus_exp(tau);
  const double E = 1.0 - one_minus_E;
  const double L = s.L();
  s.tally.escaped += L * E;
  s.tally.absorbed += P.lam[s.lam].one_minus_albedo * L * one_minus_E;
  const uint4 r = draw_block(s.pid(), s.lam, s.event, 0, P.seed, P.model);
  const double tau_star = neg_log_one_minus(u01(r.x) * one_minus_E);
  s.hg() = make_float2(u01f(r.y), u01f(r.z));
  if (kTape) {
    // the record's first two sectors, whole, with 16-byte stores
    const float3 x = s.x(), k = s.k(), g = s.sh.g[s.i];
    float4* t = reinterpret_cast<float4*>(&tape_records(P, s.lam, s.pid())[s.event]);
    t[0] = make_float4(x.x, x.y, x.z, k.x);
    t[1] = make_float4(k.y, k.z, __int_as_float(tape_cell(P, s)), tape_units(L, tape_exponent(P, s.lam)));
    t[2] = make_float4((float)one_minus_E, (float)E, u01f(r.x), g.x);
    t[3] = make_float4(g.y, g.z, 0.0f, 0.0f);
  }
  s.L() = P.lam[s.lam].albedo * L * one_minus_E;  // weight after the scattering
  float2 a;
  split_pair(tau_star, a.x, a.y);
  s.res() = a;
  request_walk(s, kPath2);
}

// Path 2 ended in the interaction cell (th holds s*, the slot the cell): move
// the packet, then the scattering peel-offs.
template <class G, bool kTape>
__device__ __forceinline__ void finish_path2(const FwdParams& P, Task<G, kTape>& s) {
  const float s_star = s.th;
  const float3 x0 = s.x(), k = s.k();
  float3 x = make_float3(fmaf(s_star, k.x, x0.x), fmaf(s_star, k.y, x0.y), fmaf(s_star, k.z, x0.z));
  G::clamp(P, s.cell(), x);
  s.x() = x;
  s.has_cell = true;
  trace_row(P, s, s.event, G::cell_id(P, s.cell()), s.L(), 0.0, 0.0);
  s.q = 0;
  s.phase = kPeelScan;
}

// The peel-off of the event towards instrument q (the same for the whole warp,
// so its table is read as uniform values): along a frame that looks along a
// grid axis the optical depth comes from the column sums and is deposited at
// once; otherwise a record for the sorted pass, or (no pass, or its buffer
// full) its walk.
template <class G, bool kTape>
__device__ __forceinline__ void peel_off(const FwdParams& P, Task<G, kTape>& s, int q) {
  const DevInstr& I = P.instr[q];
  const bool emission = s.event == 0;
  s.q = q + 1;
  if constexpr (G::kColumns) {
    if (P.use_columns && I.column && column_peel(P, s, I)) {
      peel_deposit(P, s, q, !emission);
      s.n_peel += 1u;
      return;
    }
  }
  if (P.peel) {
    // walked and deposited by the sorted pass, along with another's when that is
    // a record
    if (I.leader >= 0 && (s.deferred >> I.leader & 1u)) {
      s.n_peel += 1u;
      return;
    }
    if (defer_peel(P, s, q, emission)) {
      s.deferred |= 1u << q;
      s.n_peel += 1u;
      return;
    }
  }
  s.q = q;
  s.dep_exp = (int)s.deferred;
  request_walk(s, emission ? kPeelEmit : kPeelScat);
}

// After the last instrument: the first forced path (emission) or the
// scattering (kAfter).
template <class G, bool kTape>
__device__ __forceinline__ void peels_done(const FwdParams& P, Task<G, kTape>& s) {
  if (s.event == 0) {
    s.event = 1;
    request_path(P, s);
  } else {
    s.phase = kAfter;
  }
}

// After the scattering peel-offs: new direction, then termination or the
// next forced path.
template <class G, bool kTape>
__device__ __forceinline__ void after_scattering(const FwdParams& P, Task<G, kTape>& s) {
  const float2 u = s.hg();
  const float mu = hg_sample(P.lam[s.lam].g, u.x);
  float sp, cp;
  sincospif(2.0f * u.y, &sp, &cp);
  s.k() = rotate_dir(s.k(), mu, sp, cp);
  const double L = s.L();
  if ((P.weight_cut && bits_of(L) < bits_of(P.L_cut[s.lam])) || s.event >= P.max_events) {
    s.tally.truncated += L;
    if (kTape) tape_end(P, s, s.event);
    s.phase = kFetch;
    return;
  }
  s.event += 1;
  request_path(P, s);
}

// The warp's queues: entries and heads of the four rings, one byte each (the
// same values in every lane).
struct Queues {
  unsigned count, head;
  unsigned char (*ring)[kRing];  // the warp's rings
  __device__ __forceinline__ int size(int q) const { return (int)((count >> (8 * q)) & 255u); }
  // The fullest of the queues of per-event work.
  __device__ __forceinline__ int fullest() const {
    const int a = size(kQPath1), b = size(kQEvent), c = size(kQFetch);
    return a >= b && a >= c ? kQPath1 : (b >= c ? kQEvent : kQFetch);
  }
  // Whether a round should run for n_idle lanes without a walk.
  __device__ __forceinline__ bool round_due(int n_idle) const {
    const int n = size(fullest());
    return n >= kRoundMin || (n > 0 && n_idle - size(kQReady) >= kIdleMax);
  }
  // Append `slot` of the lanes where pred holds.
  __device__ __forceinline__ int push(int q, bool pred, int slot, unsigned lt_mask) {
    const unsigned m = __ballot_sync(0xffffffffu, pred);
    if (pred) ring[q][((head >> (8 * q)) + (count >> (8 * q)) + __popc(m & lt_mask)) & (kRing - 1)] = (unsigned char)slot;
    const int n = __popc(m);
    count += (unsigned)n << (8 * q);
    return n;
  }
  // Entry r of queue q (r below its size).
  __device__ __forceinline__ int at(int q, int r) const { return ring[q][((head >> (8 * q)) + r) & (kRing - 1)]; }
  __device__ __forceinline__ void drop(int q, int n) {
    const unsigned sh = 8 * q;
    head = (head & ~(255u << sh)) | ((((head >> sh) + n) & (kRing - 1)) << sh);
    count -= (unsigned)n << sh;
  }
};

// One control round: up to 32 packets of queue `cls` (packet r of it in lane
// r) go through the per-event work they wait for, until each needs a walk, a
// new packet or nothing more; they are queued accordingly.  Returns the packets
// served.
template <class G, bool kTape>
__device__ __forceinline__ int control_round(const FwdParams& P, Queues& Q, LaneTally& tally, int cls, unsigned lane,
                                              unsigned lt_mask) {
  Shared<G, kTape>& sh = shared_state<G, kTape>();
  const unsigned warp = threadIdx.x >> 5;
  const int n = min(32, Q.size(cls));
  const bool on = (int)lane < n;
  const int local = on ? Q.at(cls, (int)lane) : 0;
  Q.drop(cls, n);
  Task<G, kTape> s{sh, tally};
  s.i = (int)warp * G::kSlots + local;
  const unsigned pk = sh.pack[s.i];
  s.phase = on ? Pack::phase(pk) : kExit;
  s.wphase = 0;
  s.lam = Pack::lam(pk);
  s.q = Pack::q(pk);
  s.has_cell = Pack::has_cell(pk);
  s.dep_exp = 0;
  s.deferred = cls == kQEvent && s.phase != kPath2 ? (unsigned)Pack::exponent(pk) & 0xffffu : 0u;
  s.place = -1;
  s.event = sh.event[s.i];
  const float2 res = sh.res[s.i];
  s.th = res.x;
  s.tl = res.y;
  s.n_peel = s.n_col = s.c_col = 0u;
  int n_events = 0, n_packets = 0;
  if (cls == kQPath1) {
    if (on) finish_path1(P, s);
  } else {
    if (cls == kQFetch) {
      // one atomic for the round
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(P.work_counter, (unsigned long long)n);
      base = __shfl_sync(0xffffffffu, base, 0);
      base += P.w_first;
      if (on) fetch(P, s, base + lane);
      n_packets = base >= P.n_total ? 0 : (int)min((unsigned long long)n, P.n_total - base);
    } else {
      const bool ended = on && s.phase == kPath2;
      n_events = __popc(__ballot_sync(0xffffffffu, ended));
      if (ended) finish_path2(P, s);
    }
    // a peel-off walk that ended, then the event's next peel-offs, instrument
    // by instrument for the packets that have reached it
    if (s.phase == kPeelEmit || s.phase == kPeelScat) {
      peel_deposit(P, s, s.q, s.phase == kPeelScat);
      s.n_peel += 1u;
      s.q += 1;
      s.phase = kPeelScan;
    }
    if (s.phase == kPeelScan && !(s.event == 0 ? P.peel_emission : P.peel_scatter)) s.q = P.n_instr;
    for (int q = 0; q < P.n_instr; ++q) {
      const bool here = s.phase == kPeelScan && s.q == q;
      if (__any_sync(0xffffffffu, here)) {
        if (here) peel_off(P, s, q);
      }
    }
    if (s.phase == kPeelScan) peels_done(P, s);
    if (s.phase == kAfter) after_scattering(P, s);
  }
  const bool start = on && s.phase == kStart, again = on && s.phase == kFetch;
  if (start) {
    sh.pack[s.i] = Pack::make(s.wphase, s.lam, s.q, s.has_cell, s.dep_exp);
    sh.event[s.i] = s.event;
  }
  Q.push(kQReady, start, local, lt_mask);
  Q.push(kQFetch, again, local, lt_mask);
  if (cls != kQPath1) {
    const unsigned np = __reduce_add_sync(0xffffffffu, s.n_peel);
    const unsigned nc = __reduce_add_sync(0xffffffffu, s.n_col);
    const unsigned cc = __reduce_add_sync(0xffffffffu, s.c_col);
    if (lane == 0) {
      WarpTally& t = sh.tally[warp];
      t.events += (unsigned long long)n_events;
      t.packets += (unsigned long long)n_packets;
      t.peeloffs += np;
      t.column_peels += nc;
      t.column_crossings += cc;
      t.crossings += cc;
    }
  }
  __syncwarp();
  return n;
}

// Start the ready packet in slot i on this lane; the first cell's density
// load is issued here.
template <class G, bool kTape>
__device__ __forceinline__ void start_walk(const FwdParams& P, Walker<G>& s, int i, typename G::Scratch& sc) {
  Shared<G, kTape>& sh = shared_state<G, kTape>();
  const unsigned pk = sh.pack[i];
  s.slot = i;
  s.phase = Pack::phase(pk);
  const int lam = Pack::lam(pk);
  s.absorption = P.absorption + (size_t)lam * P.n_cells;
  s.kappa = P.lam[lam].kappa;
  s.x = sh.x[i];
  s.d = s.phase == kPath1 || s.phase == kPath2 ? sh.k[i] : instr_dir(P.instr[Pack::q(pk)]);
  s.id = make_float3(inv_or_zero(s.d.x), inv_or_zero(s.d.y), inv_or_zero(s.d.z));
  const float2 a = sh.res[i];
  s.aux0 = a.x;
  s.aux1 = a.y;
  s.th = 0.0f;
  s.tl = 0.0f;
  s.n = 0u;
  if (kTape) {
    s.g = make_float3(0.0f, 0.0f, 0.0f);
    s.axis_in = -1;
    s.h = -1;
  }
  s.walking = G::init(P, s.x, s.d, s.id, Pack::has_cell(pk), sh.cell[i], s.w, sc);
  if (s.walking) s.rho = load_density(&P.density[G::cell(s.w)]);
}

// A lane's walk ended: its result goes to the packet's slot.
template <class G, bool kTape>
__device__ __forceinline__ void end_walk(const FwdParams& P, const Walker<G>& s) {
  Shared<G, kTape>& sh = shared_state<G, kTape>();
  const int i = s.slot;
  if (s.phase == kPath2) {
    sh.res[i] = make_float2(s.aux0, 0.0f);
    sh.cell[i] = G::carried(s.w);
    if (kTape) {
      // the record's third sector, whole
      float4* t = reinterpret_cast<float4*>(&tape_records(P, Pack::lam(sh.pack[i]), sh.pid[i])[sh.event[i]]);
      t[4] = make_float4(__int_as_float(s.h), __int_as_float(s.axis_in), __int_as_float(G::id(P, s.w)), s.kr_h);
      t[5] = make_float4(s.rem, s.g.x, s.g.y, s.g.z);
    }
  } else {
    sh.res[i] = make_float2(s.th, s.tl);
    if (kTape && s.phase == kPath1) sh.g[i] = s.g;
  }
}

// One cell crossing of the lane's walk.  Written with selects rather than
// branches where lanes in different walks (peel-off, forced path 1 or 2)
// share the step, so the warp issues it once.
//
// Between planes the step moves on and loads the next cell's density before it
// uses this cell's: a density then has a whole crossing (the deposit and the next
// step's exit) to arrive in, where half of the issue slots went to waiting
// for it (8 of 15.5 cycles per instruction).  Disk galaxy 41.8 -> 38.7 ms per
// 4e6 packets, spiral on its power-law grid 10.1 -> 8.9 ms per 1e6, tape launch
// 15.7 -> 15.0 ms.  A walk that ends in the cell steps back.  On trees and
// Voronoi grids the step to the next cell is most of the work and moves all
// of the walk's state, so it comes last there (Voronoi disk with the density
// loaded before the faces: 12.1 against 12.3 ms).
template <class G, bool kTape>
__device__ __forceinline__ void walk_step(const FwdParams& P, Walker<G>& s, typename G::Scratch& sc) {
  typename G::Walk& w = s.w;
  int axis;
  const float te = G::exit(w, s.x, s.id, axis);
  const float t_in = w.t, rho = s.rho;
  const float texit = fmaxf(te, t_in);
  const int here = G::cell(w);
  bool inside = true;
  if constexpr (G::kIndexCells) {
    w.t = texit;
    inside = G::advance(P, s.x, s.d, s.id, axis, w, sc);
    if (inside) s.rho = load_density(&P.density[G::cell(w)]);
  }
  const float ds = texit - t_in;
  const float kr = s.kappa * rho;
  const float dt = kr * ds;
  // optical depth of the walk as an exact pair sum (all walks)
  float nh, e;
  two_sum(s.th, dt, nh, e);
  const float nl = s.tl + e;
  const bool path1 = s.phase == kPath1;
  const bool path2 = s.phase == kPath2;
  if (path2 && (nh - s.aux0) + (nl - s.aux1) > 0.0f) {
    // interaction in this cell: s* = t_in + (tau* - tau_before) / (kappa rho);
    // tau* - tau_before from the two pairs (aux0 - th is exact where it matters)
    const float rem = ((s.aux0 - s.th) + s.aux1) - s.tl;
    s.aux0 = t_in + rem / kr;
    s.walking = false;
    if constexpr (G::kIndexCells) {
      if (inside) G::retreat(axis, s.id, w);
    }
    if (kTape) {
      s.kr_h = kr;
      s.rem = rem;
      s.h = (int)s.n;
    }
    return;
  }
  if (kTape && (path1 || path2)) {
    // plane sums of the path for the adjoint: +kr at the exit plane, -kr at the entry plane
    s.g.x += (axis == 0 ? kr : 0.0f) - (s.axis_in == 0 ? kr : 0.0f);
    s.g.y += (axis == 1 ? kr : 0.0f) - (s.axis_in == 1 ? kr : 0.0f);
    s.g.z += (axis == 2 ? kr : 0.0f) - (s.axis_in == 2 ? kr : 0.0f);
    s.axis_in = axis;
  }
  if (path1 && dt > 0.0f) {
    // continuous absorption: (1 - albedo) L exp(-tau_before) (1 - exp(-dtau))
    double* const a = &s.absorption[here];
    if (s.th < s.aux1) {
      add_absorption(a, widen(s.aux0 * __expf(-s.th) * one_minus_exp_neg(dt)));
    } else {
      // exp(-tau_before) = 2^-y, y = k + f with k = floor(y): the integer
      // part joins the weight's exponent, so deep deposits do not underflow
      const float y = s.th * 1.44269504f;
      const float k = floorf(y);
      add_absorption(a, widen_exp(s.aux0 * exp2f(k - y) * one_minus_exp_neg(dt),
                                  Pack::exponent(shared_state<G, kTape>().pack[s.slot]) - (int)k));
    }
  }
  s.th = nh;
  s.tl = nl;
  s.n += 1u;
  if constexpr (!G::kIndexCells) {
    w.t = texit;
    inside = G::advance(P, s.x, s.d, s.id, axis, w, sc);
    if (inside) s.rho = load_density(&P.density[G::cell(w)]);
  }
  if (!inside) {
    s.walking = false;
    if (path2) {
      // not reachable: the pair sums of both walks are identical and tau* is
      // below the path's optical depth; keep the packet at the path's end
      atomicOr(P.flags, kFlagNoInteraction);
      s.aux0 = texit;
    }
  }
}

template <class G>
__device__ __forceinline__ typename G::Scratch lane_scratch(size_t) {
  return typename G::Scratch{};
}
template <>
__device__ __forceinline__ OctGrid::Scratch lane_scratch<OctGrid>(size_t offset) {
  return OctGrid::Scratch{reinterpret_cast<int*>(S_RAW + offset) + threadIdx.x};
}

// The most dynamic shared memory of lane_scratch, over all grids of a kind.  A
// kernel's limit is set to this and not to a launch's own need: it belongs to the
// kernel, and another context's launch of a shallower tree, in another thread,
// would lower it between the setting and the launch.
template <class G>
constexpr size_t kMaxScratch = 0;
template <>
constexpr size_t kMaxScratch<OctGrid> = (size_t)kBlock * kOctStack * sizeof(int);

template <class G>
__device__ __forceinline__ void load_grid_cache(const FwdParams&) {}
template <>
__device__ __forceinline__ void load_grid_cache<BinGrid>(const FwdParams& P) {
  const int n = P.n_nodes < kChildCache ? (int)P.n_nodes : kChildCache;
  for (int i = threadIdx.x; i < n; i += kBlock) S_CHILD[i] = P.child[i];
}
template <>
__device__ __forceinline__ void load_grid_cache<OctGrid>(const FwdParams& P) {
  const int n = P.n_nodes < kChildCache ? (int)P.n_nodes : kChildCache;
  for (int i = threadIdx.x; i < n; i += kBlock) S_CHILD[i] = P.child[i];
}

// kProf: the kernel keeps the optional execution counters of P.profile (a
// separate instantiation: the counters' ballots and clock reads cost the
// plain kernel ~4 % of its time).
template <class G, bool kTape = false, bool kProf = false>
__device__ __forceinline__ void forward_body(const FwdParams& P) {
  static_assert(G::kSlots <= kRing, "a queue holds every slot of its warp");
  Shared<G, kTape>& sh = shared_state<G, kTape>();
  load_grid_cache<G>(P);
  typename G::Scratch sc = lane_scratch<G>(sizeof(Shared<G, kTape>));
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  LaneTally tally{0.0, 0.0, 0.0};
  asm volatile("" ::"l"(&tally) : "memory");  // kept in memory, not in registers
  if (lane == 0) {
    WarpTally& t = sh.tally[warp];
    t.crossings = t.path_crossings = t.column_crossings = 0ull;
    t.events = t.peeloffs = t.packets = t.column_peels = 0ull;
  }
  // the warp's slots, all free; a launch with fewer packets than the grid has
  // slots spreads them over the warps
  const unsigned n_warps = gridDim.x * (unsigned)kWarps;
  const unsigned long long share = (P.n_total - P.w_first + n_warps - 1) / n_warps;
  const int n_slots = share < (unsigned long long)G::kSlots ? (int)share : G::kSlots;
  // when all of them are resident at once nothing refills the lanes, few warps
  // share an SM and a round's latency counts: the warp then waits for all its
  // walks (1e4 packets of a 32^3 cube 611 -> 416 us, 2e5 1548 -> 1313 us; from
  // 80 packets per warp on it loses: 4e5 packets of the spiral example 5.3
  // against 7.7 ms)
  const bool lockstep = n_slots < G::kSlots;
  if (lane == 0) sh.queues[warp] = make_uint2((unsigned)n_slots << (8 * kQFetch), 0u);
  for (int i = (int)lane; i < n_slots; i += 32) sh.ring[warp][kQFetch][i] = (unsigned char)i;
  for (int i = (int)lane; i < G::kSlots; i += 32) sh.pack[(int)warp * G::kSlots + i] = 0u;
  __syncthreads();
  Walker<G> s{};
  s.slot = -1;
  s.phase = kExit;
  int wait = 0;  // ended walks the warp waits for before it serves them
  // optional execution counters (warp leader only)
  const bool prof = kProf && P.profile != nullptr && lane == 0;
  // iterations, walking lanes, rounds, lanes served, cycles in control, in
  // the walk: per warp in shared memory (no registers held across the loop)
  __shared__ unsigned long long prof_c[kProf ? kWarps : 1][6];
  unsigned long long* pc = prof_c[kProf ? warp : 0];
  if (prof)
    for (int i = 0; i < 6; ++i) pc[i] = 0ull;
  while (true) {
    const bool ended = !s.walking && s.slot >= 0;
    if (__popc(__ballot_sync(0xffffffffu, ended)) >= wait) {
      long long t0 = 0;
      if (prof) t0 = clock64();
      const uint2 qs = sh.queues[warp];
      Queues Q{qs.x, qs.y, sh.ring[warp]};
      // the ended walks' packets to their queues
      {
        const bool p1 = ended && s.phase == kPath1;
        const unsigned np = __reduce_add_sync(0xffffffffu, p1 ? s.n : 0u);
        const unsigned nq = __reduce_add_sync(0xffffffffu, ended && !p1 && s.phase != kPath2 ? s.n : 0u);
        if (ended) end_walk<G, kTape>(P, s);
        if (lane == 0) {
          sh.tally[warp].path_crossings += np;
          sh.tally[warp].crossings += (unsigned long long)np + nq;
        }
        const int local = s.slot - (int)warp * G::kSlots;
        Q.push(kQPath1, p1, local, lt_mask);
        Q.push(kQEvent, ended && !p1, local, lt_mask);
        if (ended) s.slot = -1;
        __syncwarp();
      }
      const unsigned idle = __ballot_sync(0xffffffffu, !s.walking);
      const int n_idle = __popc(idle);
      // rounds, the fullest queue first, until every idle lane has a packet; a
      // queue of few packets waits for more while few lanes are idle
      if (Q.size(kQReady) < n_idle && Q.round_due(n_idle)) {
        // the walks go to local memory for the rounds: left to itself the
        // compiler keeps part of them there for the whole loop, at 14 local
        // loads per crossing (27.2 against 18.8 ms per 2e6 packets, disk galaxy)
        Walker<G> saved = s;
        asm volatile("" ::"l"(&saved) : "memory");
        do {
          const int served = control_round<G, kTape>(P, Q, tally, Q.fullest(), lane, lt_mask);
          if (prof) { pc[2] += 1ull; pc[3] += (unsigned long long)served; }
        } while (Q.size(kQReady) < n_idle && Q.round_due(n_idle));
        asm volatile("" ::"l"(&saved) : "memory");
        s = saved;
      }
      // idle lanes take the ready packets
      const int n_start = min(n_idle, Q.size(kQReady));
      const int r = __popc(idle & lt_mask);
      if (!s.walking && r < n_start)
        start_walk<G, kTape>(P, s, (int)warp * G::kSlots + Q.at(kQReady, r), sc);
      Q.drop(kQReady, n_start);
      __syncwarp();
      if (lane == 0) sh.queues[warp] = make_uint2(Q.count, Q.head);
      __syncwarp();
      const int busy = 32 - n_idle + n_start;  // lanes with a packet
      if (busy == 0) break;                    // no packets left
      wait = lockstep ? busy : max(1, (P.control_min * busy) >> 5);
      if (prof) pc[4] += clock64() - t0;
    }
    long long t1 = 0;
    if (prof) { t1 = clock64(); pc[0] += 1ull; }
    const unsigned stepping = kProf ? __ballot_sync(0xffffffffu, s.walking) : 0u;
    if (s.walking) walk_step<G, kTape>(P, s, sc);
    if (prof) { pc[1] += __popc(stepping); pc[5] += clock64() - t1; }
  }
  if (prof) {
    for (int i = 0; i < 6; ++i) atomicAdd(&P.profile[i], pc[i]);
  }
  // the block's sums: lanes of a warp, then the warps
  double esc = tally.escaped, ab = tally.absorbed, trc = tally.truncated;
  for (int o = 16; o > 0; o >>= 1) {
    esc += __shfl_down_sync(0xffffffffu, esc, o);
    ab += __shfl_down_sync(0xffffffffu, ab, o);
    trc += __shfl_down_sync(0xffffffffu, trc, o);
  }
  if (lane == 0) sh.lum[warp] = LaneTally{esc, ab, trc};
  __syncthreads();
  {
    if (threadIdx.x == 0) {
      WarpTally a = sh.tally[0];
      for (int w = 1; w < kWarps; ++w) {
        const WarpTally& b = sh.tally[w];
        a.crossings += b.crossings; a.path_crossings += b.path_crossings; a.column_crossings += b.column_crossings;
        a.events += b.events; a.peeloffs += b.peeloffs; a.packets += b.packets; a.column_peels += b.column_peels;
        esc += sh.lum[w].escaped; ab += sh.lum[w].absorbed; trc += sh.lum[w].truncated;
      }
      if (a.packets) {  // a block that found no packets has nothing to add
        atomicAdd(&P.stats[1], esc);
        atomicAdd(&P.stats[2], ab);
        atomicAdd(&P.stats[3], trc);
        atomicAdd(&P.counters[0], a.crossings);
        atomicAdd(&P.counters[1], a.events);
        atomicAdd(&P.counters[2], a.peeloffs);
        atomicAdd(&P.counters[3], a.packets);
        atomicAdd(&P.counters[5], a.path_crossings);
        if (a.column_peels) {
          atomicAdd(&P.counters[6], a.column_peels);
          atomicAdd(&P.counters[7], a.column_crossings);
        }
      }
    }
  }
}

// Launch a forward kernel: a persistent grid of as many resident blocks per
// SM as fit (at most p.blocks_per_sm when set), fewer when the packets do not
// give every warp one.  `extra`: dynamic shared memory beyond the packet state.
template <class G, bool kTape>
cudaError_t launch_body(void (*kernel)(const FwdParams), const FwdParams& p, int num_sms, size_t extra,
                        cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(p.work_counter, 0, sizeof(unsigned long long), stream);
  if (e != cudaSuccess) return e;
  const size_t bytes = sizeof(Shared<G, kTape>) + extra;
  // static and dynamic shared memory together pass 48 KB: the launch needs
  // the dynamic part allowed explicitly
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(Shared<G, kTape>) + kMaxScratch<G>));
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBlock, bytes);
  if (e != cudaSuccess) return e;
  per_sm = per_sm < 1 ? 1 : per_sm;
  if (p.blocks_per_sm > 0 && p.blocks_per_sm < per_sm) per_sm = p.blocks_per_sm;
  unsigned long long blocks = (unsigned long long)num_sms * per_sm;
  const unsigned long long useful = (p.n_total - p.w_first + kWarps * kSpread - 1) / (kWarps * kSpread);
  if (blocks > useful) blocks = useful;
  if (blocks < 1) blocks = 1;
  kernel<<<(unsigned)blocks, kBlock, bytes, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace tr
}  // namespace rtk
