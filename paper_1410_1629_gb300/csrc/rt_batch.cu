// Many small independent models in one persistent launch: parameter
// searches run the same transport on thousands of small grids (the model
// fitting of Sect. 1), each too small to fill a GB300 alone.
//
// Every model is a cartesian grid with one wavelength, one point source and
// one single-channel frame; its packets are the forward kernel's packets with
// Philox key (seed, model index), computed with the same arithmetic, so a
// model of a batch gives the tallies of rt_launch_packets on that model
// with model_id = its index.
//
// Work list: runs of packets of one model (chunks), sorted by estimated cost,
// largest first, so that the long runs start early and the short ones fill
// the tail.  A warp takes a chunk with one atomic and hands its packets to its
// slots as they become free; the slots of a warp may hold packets of different
// models.
//
// The execution model is the transport kernels' (rt_transport.cuh): more packets
// than lanes per warp in shared-memory slots, lanes that only walk, rounds of
// per-event work over packets that wait for the same kind of work.  A lane keeps
// the geometry its walk reads in its own shared-memory words (nine: an odd
// count, so that the lanes of a warp meet no bank conflicts; at 64 bytes apart
// they met 16-way ones, half of the kernel's shared-memory cycles).  The
// luminosity tallies of a lane are flushed to the model's when it serves
// another model.
#include "rt_transport.cuh"

namespace rtk {

namespace {

using tr::CartGrid;

// Packet slots per warp (256 models: 40 / 48 / 52 / 56 / 60 / 64 slots 128 / 114 /
// 110 / 107 / 108 / 106 ms).
#ifndef RT_BATCH_SLOTS
#define RT_BATCH_SLOTS 56
#endif
constexpr int kBatchSlots = RT_BATCH_SLOTS;
constexpr int kBatchWarps = kBatchBlock / 32;
static_assert(kBatchSlots <= tr::kRing, "a queue holds every slot of its warp");

// What a walk reads of its model's grid, in the shape CartGrid reads.
struct Geo {
  int nx, ny, nz;
  float lo[3], d[3];
};

// A warp's current chunk, and its counts.
struct WarpState {
  uint2 queues;
  unsigned long long next, end;  // packet ids left of the chunk
  int model, drained;
  unsigned long long crossings, events, peeloffs, packets, column_peels, column_crossings;
};

struct BShared {
  static constexpr int kN = kBatchWarps * kBatchSlots;
  unsigned long long pid[kN];
  double L[kN];
  float2 hg[kN];     // the event's Henyey-Greenstein uniforms
  float2 res[kN];    // what a walk starts with (path 2: tau* as a pair) and ended with
  float3 x[kN], k[kN];
  CartGrid::Cell cell[kN];
  int event[kN], model[kN];
  unsigned pack[kN];  // phase, has-cell (tr::Pack)
  Geo geo[kBatchBlock];
  WarpState warp[kBatchWarps];
  unsigned char ring[kBatchWarps][tr::kQueues][tr::kRing];
};
__device__ __forceinline__ BShared& state() { return *reinterpret_cast<BShared*>(tr::S_RAW); }

// Resident blocks per SM the register allocation aims at.
#ifndef RT_BATCH_MIN_BLOCKS
#define RT_BATCH_MIN_BLOCKS 4
#endif

// Luminosity of one model gathered by one lane (in its local memory).
struct Tally {
  double escaped, absorbed, truncated;
  int model;
};

__device__ __forceinline__ void flush(const BatchParams& P, Tally& t) {
  if (t.model >= 0) {
    double* q = &P.tallies[(size_t)t.model * 4];
    if (t.escaped != 0.0) atomicAdd(&q[1], t.escaped);
    if (t.absorbed != 0.0) atomicAdd(&q[2], t.absorbed);
    if (t.truncated != 0.0) atomicAdd(&q[3], t.truncated);
  }
  t.escaped = t.absorbed = t.truncated = 0.0;
}

// The walk a lane is on.
struct BWalker {
  int slot, phase;
  bool walking;
  float kappa;
  float3 x, id;
  CartGrid::Walk w;
  float rho, th, tl;
  unsigned n;
  float aux0, aux1;   // path 2: tau* pair, then s*
  const float* dens;  // the model's densities
};

// A packet in per-event work.
struct BTask {
  Tally& tally;
  int i, phase, wphase, m, event;
  bool has_cell;
  float th, tl;
  unsigned n_peel, n_col, c_col;
};

// The forward kernel's peel-off deposit for a single-channel frame.
__device__ __forceinline__ void deposit(const DevModel& M, const BTask& s, bool scattered) {
  const DevInstr& I = M.instr;
  const float3 x = state().x[s.i], k = state().k[s.i];
  const double L = state().L[s.i];
  float phase = 1.0f;
  if (scattered) phase = hg_phase(M.g, k.x * I.kobs[0] + k.y * I.kobs[1] + k.z * I.kobs[2]);
  const float tau = s.th;
  const double value = tau < 80.0f ? L * widen(tr::kInv4PiF * phase * expf(-tau) * (1.0f - s.tl))
                                   : L * kInv4PiD * (double)phase * exp(-((double)tau + (double)s.tl));
  const float fx = (x.x * I.ex[0] + x.y * I.ex[1] + x.z * I.ex[2] + I.off_x) * I.sx;
  const float fy = (x.x * I.ey[0] + x.y * I.ey[1] + x.z * I.ey[2] + I.off_y) * I.sy;
  if (!I.bilinear) {
    const float fix = floorf(fx), fiy = floorf(fy);
    if (!(fix >= 0.0f && fiy >= 0.0f && fix < (float)I.nx && fiy < (float)I.ny)) return;
    atomicAdd(&I.image[(size_t)(int)fiy * I.nx + (int)fix], value);
    return;
  }
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
      atomicAdd(&I.image[(size_t)(int)fiy * I.nx + (int)fix], v);
    }
  }
}

// The forward kernel's column shortcut for a frame along a grid axis (see
// column_tau there); false when the position is outside the grid.
__device__ __forceinline__ bool column_peel(const BatchParams& P, const DevModel& M, BTask& s) {
  const DevInstr& I = M.instr;
  const float3 x = state().x[s.i];
  CartGrid::Cell c;
  if (s.has_cell) {
    c = state().cell[s.i];
  } else {
    if (!inside_box(M, x)) return false;
    c.ix = min(max(__float2int_rd((x.x - M.lo[0]) * M.inv_d[0]), 0), M.nx - 1);
    c.iy = min(max(__float2int_rd((x.y - M.lo[1]) * M.inv_d[1]), 0), M.ny - 1);
    c.iz = min(max(__float2int_rd((x.z - M.lo[2]) * M.inv_d[2]), 0), M.nz - 1);
  }
  const int a = I.axis;
  const bool up = I.dir > 0;
  const int i = a == 0 ? c.ix : (a == 1 ? c.iy : c.iz);
  const int n = a == 0 ? M.nx : (a == 1 ? M.ny : M.nz);
  const float xa = a == 0 ? x.x : (a == 1 ? x.y : x.z);
  const float plane = fmaf((float)(i + (up ? 1 : 0)), M.d[a], M.lo[a]);
  const float ds0 = fmaxf(up ? plane - xa : xa - plane, 0.0f);
  const int cell = c.ix + M.nx * (c.iy + M.ny * c.iz);
  s.th = M.kappa * fmaf(tr::load_density(&P.density[M.density + cell]), ds0, __ldg(&I.column[cell]));
  s.tl = 0.0f;
  s.n_col += 1u;
  s.c_col += (unsigned)(up ? n - i : i + 1);
  return true;
}

__device__ __forceinline__ void request_walk(BTask& s, int phase) {
  s.wphase = phase;
  s.phase = tr::kStart;
}

// ---- the stages of a control round (the forward kernel's, for one frame
// per model and no absorption field)

// A new packet (model m, packet id pid): emission from its point source (the
// forward kernel's event-0 draws).
__device__ __forceinline__ void begin(const BatchParams& P, BTask& s, unsigned long long pid) {
  const DevModel& M = P.models[s.m];
  state().pid[s.i] = pid;
  state().model[s.i] = s.m;
  state().L[s.i] = M.L0;
  s.event = 0;
  s.has_cell = false;
  // one point source: the position draws of block 0 are not needed
  const uint4 r1 = draw_block(pid, 0, 0, 1, P.seed, (unsigned)s.m);
  state().x[s.i] = make_float3(M.src[0], M.src[1], M.src[2]);
  const float mu = tr::u01f_signed(r1.z);
  const float st = sqrtf(fmaxf(0.0f, 1.0f - mu * mu));
  float sp, cp;
  sincospif(2.0f * tr::u01f(r1.w), &sp, &cp);
  state().k[s.i] = make_float3(st * cp, st * sp, mu);
  s.phase = tr::kPeelScan;
}

// The tally of the packet's model.
__device__ __forceinline__ Tally& tally_of(const BatchParams& P, BTask& s) {
  if (s.tally.model != s.m) {
    flush(P, s.tally);
    s.tally.model = s.m;
  }
  return s.tally;
}

__device__ __forceinline__ void finish_path1(const BatchParams& P, BTask& s) {
  const DevModel& M = P.models[s.m];
  const double tau = widen(s.th) + widen(s.tl);
  const double L = state().L[s.i];
  Tally& T = tally_of(P, s);
  if (!(tau > 0.0)) {
    T.escaped += L;
    s.phase = tr::kFetch;
    return;
  }
  const double albedo = M.albedo;
  const double one_minus_E = one_minus_exp(tau);
  const double E = 1.0 - one_minus_E;
  T.escaped += L * E;
  T.absorbed += (1.0 - albedo) * L * one_minus_E;
  const uint4 r = draw_block(state().pid[s.i], 0, s.event, 0, P.seed, (unsigned)s.m);
  const double tau_star = neg_log_one_minus(u01(r.x) * one_minus_E);
  state().hg[s.i] = make_float2(tr::u01f(r.y), tr::u01f(r.z));
  float2 a;
  tr::split_pair(tau_star, a.x, a.y);
  state().res[s.i] = a;
  state().L[s.i] = albedo * L * one_minus_E;
  request_walk(s, tr::kPath2);
}

// Path 2 ended (th holds s*, the slot the cell).
__device__ __forceinline__ void finish_path2(const BatchParams& P, BTask& s) {
  const float s_star = s.th;
  const float3 x0 = state().x[s.i], k = state().k[s.i];
  float3 x = make_float3(fmaf(s_star, k.x, x0.x), fmaf(s_star, k.y, x0.y), fmaf(s_star, k.z, x0.z));
  CartGrid::clamp(P.models[s.m], state().cell[s.i], x);
  state().x[s.i] = x;
  s.has_cell = true;
  s.phase = tr::kPeelScan;
}

__device__ __forceinline__ void after_scattering(const BatchParams& P, BTask& s) {
  const DevModel& M = P.models[s.m];
  const float2 u = state().hg[s.i];
  const float mu = hg_sample(M.g, u.x);
  float sp, cp;
  sincospif(2.0f * u.y, &sp, &cp);
  state().k[s.i] = rotate_dir(state().k[s.i], mu, sp, cp);
  const double L = state().L[s.i];
  if ((P.weight_cut && L < P.w_min * M.L0) || s.event >= P.max_events) {
    tally_of(P, s).truncated += L;
    s.phase = tr::kFetch;
    return;
  }
  s.event += 1;
  request_walk(s, tr::kPath1);
}

// Hand packets of the warp's chunk to the lanes below n, taking new chunks as
// needed: model and id of the lane's, or model -1 (no packets left).
__device__ __forceinline__ void take_packets(const BatchParams& P, WarpState& ws, int n, int lane, int& model,
                                             unsigned long long& pid) {
  unsigned long long next = ws.next, end = ws.end;
  int m = ws.model, drained = ws.drained, done = 0;
  model = -1;
  pid = 0ull;
  __syncwarp();
  while (done < n && !drained) {
    if (next >= end) {
      unsigned long long ci = 0;
      if (lane == 0) ci = atomicAdd(P.chunk_counter, 1ull);
      ci = __shfl_sync(0xffffffffu, ci, 0);
      if (ci >= (unsigned long long)P.n_chunks) {
        drained = 1;
        break;
      }
      const BatchChunk ch = P.chunks[ci];
      m = ch.model;
      next = ch.first;
      end = ch.first + ch.count;
    }
    const unsigned long long avail = end - next;
    const int take = avail < (unsigned long long)(n - done) ? (int)avail : n - done;
    if (lane >= done && lane < done + take) {
      model = m;
      pid = next + (unsigned long long)(lane - done);
    }
    next += (unsigned long long)take;
    done += take;
  }
  if (lane == 0) {
    ws.next = next;
    ws.end = end;
    ws.model = m;
    ws.drained = drained;
  }
}

// One control round (see the forward kernel's).
__device__ __forceinline__ void control_round(const BatchParams& P, tr::Queues& Q, WarpState& ws, Tally& tally, int cls,
                                              unsigned lane, unsigned lt_mask) {
  const int n = min(32, Q.size(cls));
  const bool on = (int)lane < n;
  const int local = on ? Q.at(cls, (int)lane) : 0;
  Q.drop(cls, n);
  BTask s{tally};
  s.i = (int)(threadIdx.x >> 5) * kBatchSlots + local;
  const unsigned pk = state().pack[s.i];
  s.phase = on ? tr::Pack::phase(pk) : tr::kExit;
  s.wphase = 0;
  s.has_cell = tr::Pack::has_cell(pk);
  s.m = state().model[s.i];
  s.event = state().event[s.i];
  const float2 res = state().res[s.i];
  s.th = res.x;
  s.tl = res.y;
  s.n_peel = s.n_col = s.c_col = 0u;
  int n_events = 0, n_packets = 0;
  if (cls == tr::kQPath1) {
    if (on) finish_path1(P, s);
  } else {
    if (cls == tr::kQFetch) {
      unsigned long long pid;
      take_packets(P, ws, n, (int)lane, s.m, pid);
      const bool got = on && s.m >= 0;
      n_packets = __popc(__ballot_sync(0xffffffffu, got));
      if (got) begin(P, s, pid);
      else s.phase = tr::kExit;
    } else {
      const bool ended = on && s.phase == tr::kPath2;
      n_events = __popc(__ballot_sync(0xffffffffu, ended));
      if (ended) finish_path2(P, s);
    }
    // the model's one peel-off of this event: along a grid axis by the column
    // sums, else by a walk; deposited here when it is known
    const bool walked = s.phase == tr::kPeelEmit || s.phase == tr::kPeelScat;
    if (walked || s.phase == tr::kPeelScan) {
      const DevModel& M = P.models[s.m];
      bool known = walked;
      if (!walked && (s.event == 0 ? P.peel_emission : P.peel_scatter)) {
        known = P.use_columns && M.instr.column && column_peel(P, M, s);
        if (!known) request_walk(s, s.event == 0 ? tr::kPeelEmit : tr::kPeelScat);
      }
      if (known) {
        deposit(M, s, s.event != 0);
        s.n_peel += 1u;
      }
      if (s.phase != tr::kStart) {
        if (s.event == 0) {
          s.event = 1;
          request_walk(s, tr::kPath1);
        } else {
          s.phase = tr::kAfter;
        }
      }
    }
    if (s.phase == tr::kAfter) after_scattering(P, s);
  }
  const bool start = on && s.phase == tr::kStart, again = on && s.phase == tr::kFetch;
  if (start) {
    state().pack[s.i] = tr::Pack::make(s.wphase, 0, 0, s.has_cell, 0);
    state().event[s.i] = s.event;
  }
  Q.push(tr::kQReady, start, local, lt_mask);
  Q.push(tr::kQFetch, again, local, lt_mask);
  if (cls != tr::kQPath1) {
    const unsigned np = __reduce_add_sync(0xffffffffu, s.n_peel);
    const unsigned nc = __reduce_add_sync(0xffffffffu, s.n_col);
    const unsigned cc = __reduce_add_sync(0xffffffffu, s.c_col);
    if (lane == 0) {
      ws.events += (unsigned long long)n_events;
      ws.packets += (unsigned long long)n_packets;
      ws.peeloffs += np;
      ws.column_peels += nc;
      ws.column_crossings += cc;
      ws.crossings += cc;
    }
  }
  __syncwarp();
}

// Start the ready packet in slot i on this lane.
__device__ __forceinline__ void start_walk(const BatchParams& P, BWalker& s, int i) {
  const DevModel& M = P.models[state().model[i]];
  const unsigned pk = state().pack[i];
  s.slot = i;
  s.phase = tr::Pack::phase(pk);
  s.kappa = M.kappa;
  s.dens = P.density + M.density;
  s.x = state().x[i];
  float3 d = state().k[i];
  if (s.phase == tr::kPeelEmit || s.phase == tr::kPeelScat) d = tr::instr_dir(M.instr);
  s.id = make_float3(tr::inv_or_zero(d.x), tr::inv_or_zero(d.y), tr::inv_or_zero(d.z));
  const float2 a = state().res[i];
  s.aux0 = a.x;
  s.aux1 = a.y;
  s.th = 0.0f;
  s.tl = 0.0f;
  s.n = 0u;
  Geo& G = state().geo[threadIdx.x];
  G.nx = M.nx; G.ny = M.ny; G.nz = M.nz;
#pragma unroll
  for (int c = 0; c < 3; ++c) { G.lo[c] = M.lo[c]; G.d[c] = M.d[c]; }
  CartGrid::Scratch sc;
  s.walking = CartGrid::init(M, s.x, d, s.id, tr::Pack::has_cell(pk), state().cell[i], s.w, sc);
  if (s.walking) s.rho = tr::load_density(&s.dens[s.w.cell]);
}

// One cell crossing (the forward kernel's step without the absorption field).
__device__ __forceinline__ void step(const BatchParams& P, BWalker& s) {
  const Geo& G = state().geo[threadIdx.x];
  CartGrid::Walk& w = s.w;
  int axis;
  const float te = CartGrid::exit(w, s.x, s.id, axis);
  const float texit = fmaxf(te, w.t);
  const float ds = texit - w.t;
  const float kr = s.kappa * s.rho;
  const float dt = kr * ds;
  float nh, e;
  tr::two_sum(s.th, dt, nh, e);
  const float nl = s.tl + e;
  const bool path2 = s.phase == tr::kPath2;
  if (path2 && (nh - s.aux0) + (nl - s.aux1) > 0.0f) {
    const float rem = ((s.aux0 - s.th) + s.aux1) - s.tl;
    s.aux0 = w.t + rem / kr;
    s.walking = false;
    return;
  }
  s.th = nh;
  s.tl = nl;
  s.n += 1u;
  w.t = texit;
  CartGrid::Scratch sc;
  if (CartGrid::advance(G, s.x, s.x, s.id, axis, w, sc)) {
    s.rho = tr::load_density(&s.dens[w.cell]);
  } else {
    s.walking = false;
    if (path2) {  // not reachable (see the forward kernel)
      atomicOr(P.flags, kFlagNoInteraction);
      s.aux0 = texit;
    }
  }
}

__global__ void __launch_bounds__(kBatchBlock, RT_BATCH_MIN_BLOCKS) k_batch(const BatchParams P) {
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  WarpState& ws = state().warp[warp];
  if (lane == 0) {
    ws.queues = make_uint2((unsigned)kBatchSlots << (8 * tr::kQFetch), 0u);
    ws.next = ws.end = 0ull;
    ws.model = ws.drained = 0;
    ws.crossings = ws.events = ws.peeloffs = ws.packets = ws.column_peels = ws.column_crossings = 0ull;
  }
  for (int i = (int)lane; i < kBatchSlots; i += 32) {
    state().ring[warp][tr::kQFetch][i] = (unsigned char)i;
    state().pack[(int)warp * kBatchSlots + i] = 0u;
    state().model[(int)warp * kBatchSlots + i] = 0;
  }
  __syncwarp();
  Tally tally{0.0, 0.0, 0.0, -1};
  asm volatile("" ::"l"(&tally) : "memory");  // kept in memory, not in registers
  BWalker s{};
  s.slot = -1;
  s.phase = tr::kExit;
  int wait = 0;  // ended walks the warp waits for before it serves them
  while (true) {
    const bool ended = !s.walking && s.slot >= 0;
    if (__popc(__ballot_sync(0xffffffffu, ended)) >= wait) {
      const uint2 qs = ws.queues;
      tr::Queues Q{qs.x, qs.y, state().ring[warp]};
      {
        const bool p1 = ended && s.phase == tr::kPath1;
        const unsigned nc = __reduce_add_sync(0xffffffffu, ended && s.phase != tr::kPath2 ? s.n : 0u);
        if (ended) {
          if (s.phase == tr::kPath2) {
            state().res[s.slot] = make_float2(s.aux0, 0.0f);
            state().cell[s.slot] = CartGrid::carried(s.w);
          } else {
            state().res[s.slot] = make_float2(s.th, s.tl);
          }
        }
        if (lane == 0) ws.crossings += nc;
        const int local = s.slot - (int)warp * kBatchSlots;
        Q.push(tr::kQPath1, p1, local, lt_mask);
        Q.push(tr::kQEvent, ended && !p1, local, lt_mask);
        if (ended) s.slot = -1;
        __syncwarp();
      }
      const unsigned idle = __ballot_sync(0xffffffffu, !s.walking);
      const int n_idle = __popc(idle);
      if (Q.size(tr::kQReady) < n_idle && Q.round_due(n_idle)) {
        // the walks go to local memory for the rounds (see the forward kernel)
        BWalker saved = s;
        asm volatile("" ::"l"(&saved) : "memory");
        do {
          control_round(P, Q, ws, tally, Q.fullest(), lane, lt_mask);
        } while (Q.size(tr::kQReady) < n_idle && Q.round_due(n_idle));
        asm volatile("" ::"l"(&saved) : "memory");
        s = saved;
      }
      const int n_start = min(n_idle, Q.size(tr::kQReady));
      const int r = __popc(idle & lt_mask);
      if (!s.walking && r < n_start) start_walk(P, s, (int)warp * kBatchSlots + Q.at(tr::kQReady, r));
      Q.drop(tr::kQReady, n_start);
      __syncwarp();
      if (lane == 0) ws.queues = make_uint2(Q.count, Q.head);
      __syncwarp();
      const int busy = 32 - n_idle + n_start;
      if (busy == 0) break;
      wait = max(1, (P.control_min * busy) >> 5);
    }
    if (s.walking) step(P, s);
  }
  flush(P, tally);
  if (lane == 0 && ws.packets) {
    atomicAdd(&P.counters[0], ws.crossings);
    atomicAdd(&P.counters[1], ws.events);
    atomicAdd(&P.counters[2], ws.peeloffs);
    atomicAdd(&P.counters[3], ws.packets);
    if (ws.column_peels) {
      atomicAdd(&P.counters[4], ws.column_peels);
      atomicAdd(&P.counters[5], ws.column_crossings);
    }
  }
}

// Column sums of each model whose frame looks along a grid axis: one block
// per model, one thread per grid line (the forward path's k_columns).
__global__ void k_batch_columns(const DevModel* models, int n_models, const float* density) {
  const int m = blockIdx.x;
  if (m >= n_models) return;
  const DevModel& M = models[m];
  float* out = const_cast<float*>(M.instr.column);
  if (!out) return;
  const float* dens = density + M.density;
  const int nx = M.nx, ny = M.ny, axis = M.instr.axis, dir = M.instr.dir;
  const int n = axis == 0 ? M.nx : (axis == 1 ? M.ny : M.nz);
  const long long n_lines = (long long)M.nx * M.ny * M.nz / n;
  const double d = (double)M.d[axis];
  for (long long L = threadIdx.x; L < n_lines; L += blockDim.x) {
    long long base, stride;
    if (axis == 0) {
      base = L * nx; stride = 1;
    } else if (axis == 1) {
      base = (L % nx) + (L / nx) * (long long)nx * ny; stride = nx;
    } else {
      base = L; stride = (long long)nx * ny;
    }
    double acc = 0.0;
    for (int k = 0; k < n; ++k) {
      const int j = dir > 0 ? n - 1 - k : k;
      const long long c = base + (long long)j * stride;
      out[c] = (float)acc;
      acc += (double)dens[c] * d;
    }
  }
}

// Every model emits its luminosity per launch.
__global__ void k_batch_emitted(double* tallies, const double* lum, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) tallies[(size_t)i * 4] += lum[i];
}

}  // namespace

const void* batch_kernel() { return reinterpret_cast<const void*>(&k_batch); }
const void* batch_emitted_kernel() { return reinterpret_cast<const void*>(&k_batch_emitted); }
const void* batch_columns_kernel() { return reinterpret_cast<const void*>(&k_batch_columns); }

cudaError_t launch_batch_columns(const DevModel* models, int n_models, const float* density, cudaStream_t stream) {
  k_batch_columns<<<(unsigned)n_models, 128, 0, stream>>>(models, n_models, density);
  return cudaGetLastError();
}

cudaError_t launch_batch(const BatchParams& p, unsigned blocks, cudaStream_t stream) {
  k_batch<<<blocks, kBatchBlock, batch_shared_bytes(), stream>>>(p);
  return cudaGetLastError();
}

size_t batch_shared_bytes() { return sizeof(BShared); }

cudaError_t batch_blocks_per_sm(int* blocks) {
  const cudaError_t e =
      cudaFuncSetAttribute(k_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)batch_shared_bytes());
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, k_batch, kBatchBlock, batch_shared_bytes());
}

}  // namespace rtk
